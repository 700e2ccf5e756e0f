// Complex128 fused forward / adjoint passes for sm_103a.
//
// The same plans and step programs as the complex64 passes (Secs. 3.2-3.3),
// with every amplitude, table entry and partial in float64: the
// double-precision state type the paper's library supports next to
// complex64. Generic steps apply a fused 2x2 per register bit in the forward,
// CZ signs and CNOT swaps, and un-apply one rotation at a time in the
// adjoint. Round programs apply four rotations at two FMAs per component and
// one merged diagonal per round, with pending CZ signs, so a qubit-layer of the
// hardware-efficient ansatz costs 6 FP64 instructions per amplitude pair
// forward (16 as a fused 2x2) and 17 backward (60 one rotation at a time). GB300's FP64 pipe runs at 1/61 of its FP32
// rate, so these passes are bound by FP64 instruction issue, never by memory.
//
// A CTA (256 threads) owns 4096 amplitudes per state, as in the complex64
// passes; the tile is 64 KiB per state here (16-byte amplitudes), so the
// adjoint (psi and lambda) takes 128 KiB. One CTA per SM (8 warps) keeps the
// FP64 pipe busy; the launch bound lets the 16 + 16 double2 registers of the
// adjoint step stay in registers. A launch of few tiles gets smaller CTAs, and
// a cluster of two CTAs shares a 12-qubit tile where that evens out the SMs
// (launch_pass64).
//
// Shared-memory layout: amplitude with local index i lives at
// i ^ ((i >> 4) & 7). Eight 16-byte amplitudes fill the 32 banks, and a
// 16-byte access is served eight lanes at a time. Register groups are local
// nibbles: for nibble 0 those eight lanes differ in local bits 4..6, which the
// XOR folds into the low three bits; for any other group they differ in bits
// 0..2 directly. Either way the eight lanes hit eight distinct bank quads.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "kernels.h"

namespace qf {
namespace {

__device__ __forceinline__ uint32_t swz64(uint32_t i) { return i ^ ((i >> 4) & 7u); }

// Scatter the low bits of src into the set bits of mask (ascending).
__device__ __forceinline__ uint32_t pdep(uint32_t src, uint32_t mask) {
  uint32_t r = 0;
  for (uint32_t bb = 1; mask; bb <<= 1) {
    const uint32_t low = mask & (0u - mask);
    if (src & bb) r |= low;
    mask ^= low;
  }
  return r;
}

__device__ __forceinline__ uint32_t reg_offset(uint32_t j, const uint32_t (&o)[4]) {
  return ((j & 1u) ? o[0] : 0u) ^ ((j & 2u) ? o[1] : 0u) ^ ((j & 4u) ? o[2] : 0u) ^ ((j & 8u) ? o[3] : 0u);
}

// v with its sign flipped when s = 1
__device__ __forceinline__ double flipd(double v, uint32_t s) {
  return __longlong_as_double(__double_as_longlong(v) ^ ((long long)s << 63));
}

// phase i^k times v
__device__ __forceinline__ double2 ipow(double2 v, uint32_t k) {
  switch (k & 3u) {
    case 0: return v;
    case 1: return make_double2(-v.y, v.x);
    case 2: return make_double2(-v.x, -v.y);
    default: return make_double2(v.y, -v.x);
  }
}

// (a, b) <- (u00 a + u01 b, u10 a + u11 b) on the pairs of register bit R.
template <int R>
__device__ __forceinline__ void apply_u64(double2 (&r)[16], const double2 u00, const double2 u01, const double2 u10,
                                          const double2 u11) {
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    if (j & (1 << R)) continue;
    const int j1 = j | (1 << R);
    const double2 x = r[j], y = r[j1];
    r[j].x = u00.x * x.x - u00.y * x.y + u01.x * y.x - u01.y * y.y;
    r[j].y = u00.x * x.y + u00.y * x.x + u01.x * y.y + u01.y * y.x;
    r[j1].x = u10.x * x.x - u10.y * x.y + u11.x * y.x - u11.y * y.y;
    r[j1].y = u10.x * x.y + u10.y * x.x + u11.x * y.y + u11.y * y.x;
  }
}

// Un-apply u = exp(-i phi P / 2) (P = Z, Y or X on register bit R) from psi
// and lambda; returns the thread's sum of Im<lambda|P|psi> over its pairs,
// taken before the un-apply. Re<lambda_j| du/dphi |psi_{j-1}> =
// (1/2) Im<lambda_j|P|psi_j> (Sec. 3.3); the 1/2 is applied at the flush.
template <int R, int KIND>
__device__ __forceinline__ double bwd_gate64(double2 (&p)[16], double2 (&l)[16], const double c, const double s) {
  double acc = 0.0;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    if (j & (1 << R)) continue;
    const int j1 = j | (1 << R);
    const double2 p0 = p[j], p1 = p[j1], l0 = l[j], l1 = l[j1];
    if (KIND == G_RZ) {
      acc += l0.x * p0.y - l0.y * p0.x - l1.x * p1.y + l1.y * p1.x;
      // u^dagger = diag(c + i s, c - i s)
      p[j] = make_double2(c * p0.x - s * p0.y, c * p0.y + s * p0.x);
      p[j1] = make_double2(c * p1.x + s * p1.y, c * p1.y - s * p1.x);
      l[j] = make_double2(c * l0.x - s * l0.y, c * l0.y + s * l0.x);
      l[j1] = make_double2(c * l1.x + s * l1.y, c * l1.y - s * l1.x);
    } else if (KIND == G_RY) {
      acc += l1.x * p0.x + l1.y * p0.y - l0.x * p1.x - l0.y * p1.y;
      // u^dagger = [[c, s], [-s, c]]
      p[j] = make_double2(c * p0.x + s * p1.x, c * p0.y + s * p1.y);
      p[j1] = make_double2(c * p1.x - s * p0.x, c * p1.y - s * p0.y);
      l[j] = make_double2(c * l0.x + s * l1.x, c * l0.y + s * l1.y);
      l[j1] = make_double2(c * l1.x - s * l0.x, c * l1.y - s * l0.y);
    } else {  // RX
      acc += l0.x * p1.y - l0.y * p1.x + l1.x * p0.y - l1.y * p0.x;
      // u^dagger = [[c, i s], [i s, c]]
      p[j] = make_double2(c * p0.x - s * p1.y, c * p0.y + s * p1.x);
      p[j1] = make_double2(c * p1.x - s * p0.y, c * p1.y + s * p0.x);
      l[j] = make_double2(c * l0.x - s * l1.y, c * l0.y + s * l1.x);
      l[j1] = make_double2(c * l1.x - s * l0.y, c * l1.y + s * l0.x);
    }
  }
  return acc;
}

template <int KIND>
__device__ __forceinline__ double bwd_dispatch64(uint32_t r, double2 (&p)[16], double2 (&l)[16], double c,
                                                 double s) {
  switch (r) {
    case 0: return bwd_gate64<0, KIND>(p, l, c, s);
    case 1: return bwd_gate64<1, KIND>(p, l, c, s);
    case 2: return bwd_gate64<2, KIND>(p, l, c, s);
    default: return bwd_gate64<3, KIND>(p, l, c, s);
  }
}

// CNOT with its target on register bit RT: swap the target pairs whose control
// is 1 (register bit cb when creg, else bit cb of the thread's base index gb).
// Self-inverse, so the adjoint applies the same swap to psi and lambda.
template <int RT, bool BWD>
__device__ __forceinline__ void cnot64(double2 (&r)[16], double2 (&l)[16], bool creg, uint32_t cb, uint32_t gb) {
  const uint32_t cg = (gb >> cb) & 1u;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    if (j & (1 << RT)) continue;
    const int j1 = j | (1 << RT);
    const bool on = creg ? (((uint32_t)j >> cb) & 1u) != 0 : cg != 0;
    const double2 a = r[j], b = r[j1];
    r[j] = on ? b : a;
    r[j1] = on ? a : b;
    if (BWD) {
      const double2 c = l[j], d = l[j1];
      l[j] = on ? d : c;
      l[j1] = on ? c : d;
    }
  }
}

// ---- round programs (the complex64 round programs' items in float64) -----------
// A round applies one item per register bit r (the RY, then the merged RZ
// run; the adjoint runs the exact reverse) and then the round's CZ links.
// Pending CZ signs D: the registers hold psi~ with
// psi = D psi~, D = (-1)^(c0 + sum_r A_r j_r) (bit 4: c0, bits 0..3: A);
// a gate on register bit r sees only Z_r^(A_r), folded into it; CZs between
// two register bits are signs of the round's diagonal table.

// Link q couples qubit q with q + 1 mod n: the constant (t2 & gb) and linear
// (u) parts of the links L for thread base index gb.
__device__ __forceinline__ void link_terms64(uint32_t L, uint32_t gb, int n, uint32_t& t2, uint32_t& u) {
  const uint32_t nmask = n >= 32 ? ~0u : ((1u << n) - 1u);
  const uint32_t t1 = L & gb;
  t2 = L & (((gb >> 1) | ((gb & 1u) << (n - 1))) & nmask);
  u = (((t1 << 1) | (t1 >> (n - 1))) & nmask) ^ t2;
}

__device__ __forceinline__ void chain64(uint32_t L, uint32_t gb, const uint32_t (&p)[4], int n, uint32_t& D) {
  uint32_t t2, u;
  link_terms64(L, gb, n, t2, u);
  D ^= (((u >> p[0]) & 1u) | (((u >> p[1]) & 1u) << 1) | (((u >> p[2]) & 1u) << 2) | (((u >> p[3]) & 1u) << 3)) |
       ((__popc(t2 & gb) & 1u) << 4);
}

// Multiply the registers by D (end of a step).
template <bool BWD>
__device__ __forceinline__ void pending64(uint32_t D, double2 (&r)[16], double2 (&l)[16]) {
  uint32_t S = (D & 16u) ? 0xFFFFu : 0u;
  S ^= (D & 1u) ? 0xAAAAu : 0u;
  S ^= (D & 2u) ? 0xCCCCu : 0u;
  S ^= (D & 4u) ? 0xF0F0u : 0u;
  S ^= (D & 8u) ? 0xFF00u : 0u;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const uint32_t f = (S >> j) & 1u;
    r[j] = make_double2(flipd(r[j].x, f), flipd(r[j].y, f));
    if (BWD) l[j] = make_double2(flipd(l[j].x, f), flipd(l[j].y, f));
  }
}

// One rotation on register bit R, two FMAs per real component: the rotation by
// w over cos(w/2), q = tan(w/2) (see fused.cu's rot_T). The cosines are a scale
// of the round's diagonal; |q| <= 2^54, whose products float64 holds (running
// rounds with |q| > 256 twice by half the angles took a step with every angle at
// pi, n = 12, d = 10, 256 samples, from 3,270 to 5,280 us). Against three shears, and with the diagonal's terms from
// complement differences: step of n = 12, d = 10, 256 samples 4,296 -> 3,328 us,
// as these kernels are bound by FP64 issue.
template <int R>
__device__ __forceinline__ void rot_T64(double2 (&r)[16], double q, bool rx) {
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    if (j & (1 << R)) continue;
    const int j1 = j | (1 << R);
    const double2 p0 = r[j], p1 = r[j1];
    if (rx) {  // p0 -= i q p1; p1 -= i q p0
      r[j] = make_double2(fma(q, p1.y, p0.x), fma(-q, p1.x, p0.y));
      r[j1] = make_double2(fma(q, p0.y, p1.x), fma(-q, p0.x, p1.y));
    } else {  // p0 -= q p1; p1 += q p0
      r[j] = make_double2(fma(-q, p1.x, p0.x), fma(-q, p1.y, p0.y));
      r[j1] = make_double2(fma(q, p0.x, p1.x), fma(q, p0.y, p1.y));
    }
  }
}

// A forward item (a: a pending Z_R turns w into -w). An absent rotation is skipped.
template <int R>
__device__ __forceinline__ void rot_fwd64(double2 (&r)[16], double q, uint32_t a, bool has_y, bool rx) {
  if (!has_y) return;
  if (rx) rot_T64<R>(r, a ? -q : q, true);
  else rot_T64<R>(r, a ? -q : q, false);
}

// v *= (c + i s)
__device__ __forceinline__ void cmul64(double2& v, double c, double s) {
  const double x = v.x;
  v.x = fma(c, x, -s * v.y);
  v.y = fma(s, x, c * v.y);
}

// The round's diagonal (its 4 RZ runs and the CZ links between register
// bits, merged), applied: register amplitude j times ph[j]. It commutes with
// the rotations on the other register bits and with the pending signs.
__device__ __forceinline__ void diag64(double2 (&r)[16], const double2* ph) {
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const double2 e = ph[j];
    cmul64(r[j], e.x, e.y);
  }
}

// Adjoint side of the round's diagonal: g[r] = sum_j sigma_r(j) w_j with
// w_j = Im(conj(lambda_j) psi_j), sigma_r(j) = +1 where bit r of j is clear,
// else -1 (the RZ-run terms; w_j is unchanged by the diagonal, and Z_r
// commutes with the rotations on the other bits), from the differences u_j =
// w_j - w_{15-j} as sigma_r(15 - j) = -sigma_r(j); then the un-apply.
__device__ __forceinline__ void diag_terms64(const double2 (&p)[16], const double2 (&l)[16], double (&g)[8]) {
  double u[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const double2 p0 = p[m], l0 = l[m], p1 = p[15 - m], l1 = l[15 - m];
    u[m] = fma(l1.y, p1.x, fma(-l1.x, p1.y, fma(l0.x, p0.y, -l0.y * p0.x)));
  }
  const double a0 = u[0] + u[1], a1 = u[2] + u[3], a2 = u[4] + u[5], a3 = u[6] + u[7];
  const double q0 = a0 + a1, T = q0 + (a2 + a3);
  g[0] = fma(2.0, (u[0] + u[2]) + (u[4] + u[6]), -T);
  g[1] = fma(2.0, a0 + a2, -T);
  g[2] = fma(2.0, q0, -T);
  g[3] = T;
}

// The rotation of an adjoint item on register bit R (q un-applies it), after
// the round's diagonal; gy: the thread's sum of Im<lambda|P|psi> before it. A
// pending Z_R negates q and gy. An absent rotation is skipped; its value is 0.
template <int R>
__device__ __forceinline__ void rot_bwd64(double2 (&p)[16], double2 (&l)[16], double q, uint32_t a, double& gy,
                                          bool has_y, bool rx) {
  gy = 0.0;
  if (!has_y) return;
  double g0 = 0.0, g1 = 0.0;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    if (j & (1 << R)) continue;
    const int j1 = j | (1 << R);
    const double2 p0 = p[j], p1 = p[j1], l0 = l[j], l1 = l[j1];
    if (rx) {
      g0 = fma(l0.x, p1.y, fma(l1.x, p0.y, g0));
      g1 = fma(l0.y, p1.x, fma(l1.y, p0.x, g1));
    } else {
      g0 = fma(l1.x, p0.x, fma(l1.y, p0.y, g0));
      g1 = fma(l0.x, p1.x, fma(l0.y, p1.y, g1));
    }
  }
  const double g = g0 - g1;
  gy = a ? -g : g;
  if (a) q = -q;
  if (rx) {
    rot_T64<R>(p, q, true);
    rot_T64<R>(l, q, true);
  } else {
    rot_T64<R>(p, q, false);
    rot_T64<R>(l, q, false);
  }
}

// Reduce 8 per-thread values over `lanes` lanes (8, 16 or 32; whole-warp
// call): afterwards the lanes with (lane & (lanes/8 - 1)) == 0 hold the 8
// lanes-sums, lane's being that of value *idx.
__device__ __forceinline__ double butterfly8_64(double (&v)[8], int lanes, int lane, int& idx) {
  int o = lanes >> 1;
  bool up = (lane & o) != 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const double send = up ? v[i] : v[i + 4];
    const double keep = up ? v[i + 4] : v[i];
    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
  }
  idx = up ? 4 : 0;
  o >>= 1;
  up = (lane & o) != 0;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const double send = up ? v[i] : v[i + 2];
    const double keep = up ? v[i + 2] : v[i];
    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
  }
  idx += up ? 2 : 0;
  o >>= 1;
  up = (lane & o) != 0;
  {
    const double send = up ? v[0] : v[1];
    const double keep = up ? v[1] : v[0];
    v[0] = keep + __shfl_xor_sync(0xffffffffu, send, o);
  }
  idx += up ? 1 : 0;
  for (o >>= 1; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
  return v[0];
}

struct Shared64 {
  uint32_t lg[256];                              // thread-part of the local index -> global bits
  double red[2][kThreads / 32][kMaxStepSlots];   // per-warp gradient sums of a step (double-buffered)
  int32_t slot[2][kMaxStepSlots];
  double dred[kThreads / 32];
  uint32_t gmap[16];
  uint32_t grp[4][4];
};

}  // namespace

// One complex128 pass: CTA c owns tiles c * tiles_per_cta .. (tile = sample *
// tiles_per_sample + tile within the sample); 2^(K-4) threads per tile, 16
// amplitudes per thread per step. SPLIT: a cluster of 2^a.split CTAs (a.split =
// 1) owns one tile instead; CTA `rank` holds the amplitudes whose top a.split local bits
// are its rank, and runs the columns (local indices without the group's bits)
// with those top bits. Only a step on a group that holds top bits reaches into
// the other CTAs' shared memory; every barrier is then the cluster's.
template <bool BWD, bool ROUNDS, bool RX = false, bool SPLIT = false>
__global__ void __launch_bounds__(kThreads, 1) pass64_kernel(const PassArgs64 a) {
  extern __shared__ __align__(16) double2 smem64[];
  __shared__ Shared64 sh;
  const PassDesc& pd = a.pd;
  const int K = pd.K;
  const int sp = SPLIT ? a.split : 0;
  const int KL = K - sp;                   // local bits of one CTA's part
  const int tl2 = K - kRegBits - sp;
  const int Tt = 1 << tl2;                 // threads per tile in this CTA
  const int nthr = (int)blockDim.x;
  const int tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  const int tiles_per_cta = nthr >> tl2;   // 1 when split
  const uint32_t rank = SPLIT ? blockIdx.x & ((1u << sp) - 1u) : 0u;
  const int64_t first_tile = SPLIT ? (int64_t)(blockIdx.x >> sp) : (int64_t)blockIdx.x * tiles_per_cta;
  const int tile_in_cta = tid >> tl2;
  const uint32_t tau = (uint32_t)(tid & (Tt - 1));
  const int64_t total_tiles = (int64_t)a.B << a.tps_log2;
  const int64_t tile = first_tile + tile_in_cta;
  const bool active = tile < total_tiles;
  const int64_t b = active ? (tile >> a.tps_log2) : 0;
  const uint32_t t_in = active ? (uint32_t)(tile & ((1ll << a.tps_log2) - 1)) : 0u;
  const uint32_t outer = pdep(t_in, pd.outer_mask);
  const int64_t sbase = b << a.n_eff;
  const int lam_at = nthr << kRegBits;     // lambda's part follows psi's
  double2* tp = smem64 + (tile_in_cta << KL);
  double2* tl = tp + lam_at;
  const int wpt = Tt >= 32 ? Tt / 32 : 1;  // warps per tile
  const int lanes = Tt < 32 ? Tt : 32;     // lanes per tile within a warp
  auto barrier = [&]() {
    if (SPLIT) cooperative_groups::this_cluster().sync();
    else __syncthreads();
  };
  // amplitude i of the tile (any part): psi, or lambda at offset lam_at
  auto amp = [&](uint32_t i, int off) -> double2& {
    double2* p = tp + off + swz64(i & ((1u << KL) - 1u));
    return SPLIT ? *cooperative_groups::this_cluster().map_shared_rank(p, i >> KL) : *p;
  };
  const uint32_t i_top = rank << KL;       // the part's local indices start here

  if (tid < 16) {
    sh.gmap[tid] = pd.gmap[tid];
    sh.grp[tid >> 2][tid & 3] = pd.groups[tid >> 2][tid & 3];
  }
  __syncthreads();
  for (int h = tid; h < (1 << (K - kRegBits)); h += nthr) {
    uint32_t g = 0;
    for (int j = 0; j < K - kRegBits; ++j)
      if ((h >> j) & 1) g |= 1u << sh.gmap[kRegBits + j];
    sh.lg[h] = g;
  }
  __syncthreads();

  auto gidx = [&](uint32_t i) -> uint32_t { return outer | (i & 15u) | sh.lg[i >> 4]; };
  auto state_ptr = [&](int32_t code) -> double2* {
    if (code >= 0) return a.slots + (int64_t)code * a.slot_stride + sbase;
    return a.work + sbase;
  };

  // ---- bring psi (and lambda) in: local index i = i_top | it * Tt + tau ---------
  const int32_t psrc = pd.psi_src;
  if (psrc == SRC_GENERATE && a.psi_in) {
    // given initial states [B][2^n_in]; padding qubits (n_in <= bit < n_eff) are |0>
    const int64_t din = 1ll << a.n_in;
    const double2* src = a.psi_in + b * din;
#pragma unroll 4
    for (int it = 0; it < 16; ++it) {
      const uint32_t i = (uint32_t)it * Tt + tau;
      const uint32_t g = gidx(i_top | i);
      const double2 v = (int64_t)g < din ? __ldcg(src + g) : make_double2(0.0, 0.0);
      if (active) tp[swz64(i)] = v;
    }
  } else if (psrc == SRC_GENERATE) {
    // psi_0 = (x) RY(x_q)|0>: a_x = prod_q (bit q of x ? sin(x_q/2) : cos(x_q/2))
    const double2* e = a.enc + b * a.n_eff;
#pragma unroll 1
    for (int it = 0; it < 16; ++it) {
      const uint32_t i = (uint32_t)it * Tt + tau;
      const uint32_t g = gidx(i_top | i);
      double pr = 1.0;
      for (int q = 0; q < a.n_eff; ++q) {
        const double2 f = __ldg(e + q);
        pr *= ((g >> q) & 1u) ? f.y : f.x;
      }
      if (active) tp[swz64(i)] = make_double2(pr, 0.0);
    }
  } else if (active) {
    // eight loads of each state in flight before their stores
    const bool half = (pd.flags & PF_SRC_H) != 0;
    const bool two = BWD && pd.lam_src == LAM_BUF;
    const double2* src = half ? nullptr : state_ptr(psrc);
    const float2* fsrc = half ? a.fslots + (int64_t)psrc * a.slot_stride + sbase : nullptr;
    const double2* lsrc = a.lam + sbase;
#pragma unroll
    for (int i0 = 0; i0 < 16; i0 += 8) {
      double2 vp[8], vl[8];
#pragma unroll
      for (int it = 0; it < 8; ++it) {
        const uint32_t g = gidx(i_top | ((uint32_t)(i0 + it) * Tt + tau));
        if (half) {
          const float2 h = __ldcg(fsrc + g);
          vp[it] = make_double2((double)h.x, (double)h.y);
        } else {
          vp[it] = __ldcg(src + g);
        }
        if (two) vl[it] = __ldcg(lsrc + g);
      }
#pragma unroll
      for (int it = 0; it < 8; ++it) {
        const uint32_t i = (uint32_t)(i0 + it) * Tt + tau;
        tp[swz64(i)] = vp[it];
        if (two) tl[swz64(i)] = vl[it];
      }
    }
  }
  if (BWD && pd.lam_src == LAM_BUF && psrc == SRC_GENERATE && active) {
    const double2* src = a.lam + sbase;
#pragma unroll 4
    for (int it = 0; it < 16; ++it) {
      const uint32_t i = (uint32_t)it * Tt + tau;
      tl[swz64(i)] = __ldcg(src + gidx(i_top | i));
    }
  }
  barrier();
  if (BWD && pd.lam_src == LAM_SEED) {
    // lambda_M = 2 (dL/dE_b) O psi_M (Eq. 4); (O psi)_x = i^{#Y} (-1)^{|(x^xm)&zm|} psi_{x^xm}
    double scale = 0.0;
    if (active) {
      double dl = 1.0;
      if (a.dLdE) dl = a.dLdE[b];
      else if (a.loss_kind == 1) dl = a.loss_scale * (a.e_part[b] - a.y[b]);  // one tile per sample
      scale = 2.0 * dl;
    }
#pragma unroll 1
    for (int it = 0; it < 16; ++it) {
      const uint32_t i = (uint32_t)it * Tt + tau;
      const uint32_t ip = (i_top | i) ^ pd.xm_local;
      const double2 v = ipow(amp(ip, 0), a.y_count);
      const uint32_t sg = __popc(gidx(ip) & a.z_mask) & 1u;
      tl[swz64(i)] = make_double2(flipd(v.x, sg) * scale, flipd(v.y, sg) * scale);
    }
    barrier();
  }

  // a tile's sum of its warps' values (stride words apart) in warp order, over
  // the CTAs that share it
  auto tile_sum = [&](const double* p, int stride) -> double {
    double sum = 0.0;
    for (uint32_t c = 0; c < (1u << sp); ++c) {
      const double* q = SPLIT ? cooperative_groups::this_cluster().map_shared_rank(p, c) : p;
      for (int w = 0; w < wpt; ++w) sum += q[w * stride];
    }
    return sum;
  };

  // ---- step program --------------------------------------------------------
  int buf = 0;
  int32_t pc = pd.op_begin;
  const uint2* ops = a.ops;
#pragma unroll 1
  while (pc < pd.op_end) {
    const uint2 op = __ldg(ops + pc++);
    const uint32_t code = op.x & 15u;
    if (ROUNDS && code == OP_STEP) {
      // ---- round step: rounds op.y .. op.y + nr - 1 on register group g
      const int g = (op.x >> 4) & 3;
      const int nr = (op.x >> 8) & 0xffff;
      const uint32_t lb0 = sh.grp[g][0], lb1 = sh.grp[g][1], lb2 = sh.grp[g][2], lb3 = sh.grp[g][3];
      const uint32_t gm = (1u << lb0) | (1u << lb1) | (1u << lb2) | (1u << lb3);
      // the thread's column: its bits, and the rank's above them, around the group's
      const uint32_t base = pdep((rank << tl2) | tau, ((1u << K) - 1u) & ~gm);
      const bool far = SPLIT && (gm >> KL) != 0;  // the group holds top bits
      const uint32_t pb = swz64(base & ((1u << KL) - 1u));
      const uint32_t so[4] = {swz64(1u << lb0), swz64(1u << lb1), swz64(1u << lb2), swz64(1u << lb3)};
      const uint32_t gb = gidx(base);
      const uint32_t pos[4] = {sh.gmap[lb0], sh.gmap[lb1], sh.gmap[lb2], sh.gmap[lb3]};
      double2 r[16];
      double2 l[16];
      if (far) {
        const uint32_t lo[4] = {1u << lb0, 1u << lb1, 1u << lb2, 1u << lb3};
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          r[j] = amp(base | reg_offset(j, lo), 0);
          if (BWD) l[j] = amp(base | reg_offset(j, lo), lam_at);
        }
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          r[j] = tp[pb ^ reg_offset(j, so)];
          if (BWD) l[j] = tl[pb ^ reg_offset(j, so)];
        }
      }
      uint32_t D = 0;
#pragma unroll 1
      for (int k = 0; k < nr; ++k) {
        const size_t rr = (size_t)op.y + k;
        const RoundPar64& v = a.rpar[rr];
        if (!BWD) {
          const uint4 lk = __ldg(a.rounds + rr * (kFwdRoundWords / 4) + 1);
          // the items' rotation terms (-1: absent) in words 12..15
          const uint4 ty = __ldg(a.rounds + rr * (kFwdRoundWords / 4) + 3);
          rot_fwd64<0>(r, v.q[0], D & 1u, (int)ty.x >= 0, RX && (lk.z & 1u));
          rot_fwd64<1>(r, v.q[1], (D >> 1) & 1u, (int)ty.y >= 0, RX && ((lk.z >> 1) & 1u));
          rot_fwd64<2>(r, v.q[2], (D >> 2) & 1u, (int)ty.z >= 0, RX && ((lk.z >> 2) & 1u));
          rot_fwd64<3>(r, v.q[3], (D >> 3) & 1u, (int)ty.w >= 0, RX && ((lk.z >> 3) & 1u));
          diag64(r, v.ph);
          chain64(lk.x, gb, pos, a.n_eff, D);
        } else {
          const uint4 lk = __ldg(a.rounds + rr * (kBwdRoundWords / 4) + 2);
          const uint4 ty = __ldg(a.rounds + rr * (kBwdRoundWords / 4) + 1);
          chain64(lk.x, gb, pos, a.n_eff, D);
          double gv[8];
          diag_terms64(r, l, gv);
          diag64(r, v.ph);
          diag64(l, v.ph);
          rot_bwd64<0>(r, l, v.q[0], D & 1u, gv[4], (int)ty.x >= 0, RX && (lk.z & 1u));
          rot_bwd64<1>(r, l, v.q[1], (D >> 1) & 1u, gv[5], (int)ty.y >= 0, RX && ((lk.z >> 1) & 1u));
          rot_bwd64<2>(r, l, v.q[2], (D >> 2) & 1u, gv[6], (int)ty.z >= 0, RX && ((lk.z >> 2) & 1u));
          rot_bwd64<3>(r, l, v.q[3], (D >> 3) & 1u, gv[7], (int)ty.w >= 0, RX && ((lk.z >> 3) & 1u));
          int idx;
          double sum = butterfly8_64(gv, lanes, lane, idx);
          if (idx >= 4) sum *= v.g[idx - 4];
          const bool owner = (lane & ((lanes >> 3) - 1)) == 0;
          const int32_t term = __ldg(reinterpret_cast<const int32_t*>(a.rounds + rr * (kBwdRoundWords / 4)) + idx);
          if (Tt >= 32) {
            if (owner) {
              sh.red[buf][warp][k * 8 + idx] = sum;
              if (warp == 0) sh.slot[buf][k * 8 + idx] = term;
            }
          } else if (owner && active && term >= 0) {
            a.g_part[tile * a.n_slots + term] = 0.5 * sum;
          }
        }
      }
      pending64<BWD>(D, r, l);
      if (far) {
        const uint32_t lo[4] = {1u << lb0, 1u << lb1, 1u << lb2, 1u << lb3};
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          amp(base | reg_offset(j, lo), 0) = r[j];
          if (BWD) amp(base | reg_offset(j, lo), lam_at) = l[j];
        }
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          tp[pb ^ reg_offset(j, so)] = r[j];
          if (BWD) tl[pb ^ reg_offset(j, so)] = l[j];
        }
      }
      barrier();
      if (BWD && Tt >= 32) {
        const int nk = nr * 8;
        for (int e = tid; e < (rank ? 0 : tiles_per_cta * nk); e += nthr) {
          const int tc = e / nk, kk = e - tc * nk;
          const int64_t t2 = first_tile + tc;
          const int32_t term = sh.slot[buf][kk];
          if (t2 < total_tiles && term >= 0) {
            const double sum = tile_sum(&sh.red[buf][tc * wpt][kk], kMaxStepSlots);
            a.g_part[t2 * a.n_slots + term] = 0.5 * sum;
          }
        }
        buf ^= 1;
      }
    } else if (!ROUNDS && code == OP_STEP) {
      const int g = (op.x >> 4) & 3;
      const int nops = (op.x >> 8) & 0xffff;
      const int nk = (int)op.y;
      const uint32_t lb0 = sh.grp[g][0], lb1 = sh.grp[g][1], lb2 = sh.grp[g][2], lb3 = sh.grp[g][3];
      const uint32_t gm = (1u << lb0) | (1u << lb1) | (1u << lb2) | (1u << lb3);
      // the thread's column: its bits, and the rank's above them, around the group's
      const uint32_t base = pdep((rank << tl2) | tau, ((1u << K) - 1u) & ~gm);
      const bool far = SPLIT && (gm >> KL) != 0;  // the group holds top bits
      const uint32_t pb = swz64(base & ((1u << KL) - 1u));
      const uint32_t so[4] = {swz64(1u << lb0), swz64(1u << lb1), swz64(1u << lb2), swz64(1u << lb3)};
      const uint32_t gb = gidx(base);
      const uint32_t go[4] = {1u << sh.gmap[lb0], 1u << sh.gmap[lb1], 1u << sh.gmap[lb2], 1u << sh.gmap[lb3]};
      double2 r[16];
      double2 l[16];
      if (far) {
        const uint32_t lo[4] = {1u << lb0, 1u << lb1, 1u << lb2, 1u << lb3};
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          r[j] = amp(base | reg_offset(j, lo), 0);
          if (BWD) l[j] = amp(base | reg_offset(j, lo), lam_at);
        }
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          r[j] = tp[pb ^ reg_offset(j, so)];
          if (BWD) l[j] = tl[pb ^ reg_offset(j, so)];
        }
      }
#pragma unroll 1
      for (int k = 0; k < nops; ++k) {
        const uint2 o = __ldg(ops + pc++);
        const uint32_t oc = o.x & 15u;
        if (!BWD && oc == OP_U) {
          const double2* u = a.mats + 4 * (size_t)(o.x >> 8);
          const double2 u00 = __ldg(u), u01 = __ldg(u + 1), u10 = __ldg(u + 2), u11 = __ldg(u + 3);
          switch ((o.x >> 4) & 3u) {
            case 0: apply_u64<0>(r, u00, u01, u10, u11); break;
            case 1: apply_u64<1>(r, u00, u01, u10, u11); break;
            case 2: apply_u64<2>(r, u00, u01, u10, u11); break;
            default: apply_u64<3>(r, u00, u01, u10, u11); break;
          }
        } else if (BWD && oc == OP_G) {
          const uint32_t rr = (o.x >> 4) & 3u, kind = (o.x >> 6) & 3u, ks = (o.x >> 8) & 0xffu;
          const double2 csv = __ldg(a.cs + o.y);
          double acc;
          if (kind == G_RZ) acc = bwd_dispatch64<G_RZ>(rr, r, l, csv.x, csv.y);
          else if (kind == G_RY) acc = bwd_dispatch64<G_RY>(rr, r, l, csv.x, csv.y);
          else acc = bwd_dispatch64<G_RX>(rr, r, l, csv.x, csv.y);
          for (int off = 1; off < lanes; off <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
          if (Tt >= 32) {
            if (lane == 0) sh.red[buf][warp][ks] = acc;
            if (tid == 0) sh.slot[buf][ks] = (int32_t)o.y;
          } else if (active && (lane & (Tt - 1)) == 0) {
            a.g_part[tile * a.n_slots + o.y] = 0.5 * acc;
          }
        } else if (oc == OP_CNOT) {
          const bool creg = ((o.y >> 8) & 1u) != 0;
          const uint32_t cb = o.y & 0xffu;
          switch ((o.x >> 4) & 3u) {
            case 0: cnot64<0, BWD>(r, l, creg, cb, gb); break;
            case 1: cnot64<1, BWD>(r, l, creg, cb, gb); break;
            case 2: cnot64<2, BWD>(r, l, creg, cb, gb); break;
            default: cnot64<3, BWD>(r, l, creg, cb, gb); break;
          }
        } else if (oc == OP_CHAIN || oc == OP_CZ) {
          const uint32_t links = o.y, c0 = o.y & 0xffu, c1 = (o.y >> 8) & 0xffu;
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const uint32_t x = gb | reg_offset(j, go);
            const uint32_t sg = oc == OP_CHAIN ? (__popc(x & (x >> 1) & links) & 1u) : ((x >> c0) & (x >> c1) & 1u);
            r[j].x = flipd(r[j].x, sg);
            r[j].y = flipd(r[j].y, sg);
            if (BWD) {
              l[j].x = flipd(l[j].x, sg);
              l[j].y = flipd(l[j].y, sg);
            }
          }
        }
      }
      if (far) {
        const uint32_t lo[4] = {1u << lb0, 1u << lb1, 1u << lb2, 1u << lb3};
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          amp(base | reg_offset(j, lo), 0) = r[j];
          if (BWD) amp(base | reg_offset(j, lo), lam_at) = l[j];
        }
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          tp[pb ^ reg_offset(j, so)] = r[j];
          if (BWD) tl[pb ^ reg_offset(j, so)] = l[j];
        }
      }
      barrier();
      if (BWD && Tt >= 32) {
        // per-tile sums of the step's terms in warp order (deterministic)
        for (int e = tid; e < (rank ? 0 : tiles_per_cta * nk); e += nthr) {
          const int tc = e / nk, kk = e - tc * nk;
          const int64_t t2 = first_tile + tc;
          if (t2 < total_tiles) {
            const double sum = tile_sum(&sh.red[buf][tc * wpt][kk], kMaxStepSlots);
            a.g_part[t2 * a.n_slots + sh.slot[buf][kk]] = 0.5 * sum;
          }
        }
        buf ^= 1;
      }
    } else if (code == OP_CKPT || code == OP_ANCHOR) {
      double2* sp = a.slots + (int64_t)op.y * a.slot_stride + sbase;
#pragma unroll 4
      for (int it = 0; it < 16; ++it) {
        const uint32_t i = (uint32_t)it * Tt + tau;
        if (!active) continue;
        if (code == OP_CKPT) sp[gidx(i_top | i)] = tp[swz64(i)];
        else tp[swz64(i)] = sp[gidx(i_top | i)];
      }
      barrier();
    }
  }

  // ---- write back ------------------------------------------------------------
  if (pd.psi_dst != BUF_NONE && (pd.flags & PF_DST_H)) {
    // memory-saving mode (Sec. 3.2): the stored pass output is rounded to complex64
    float2* dst = a.fslots + (int64_t)pd.psi_dst * a.slot_stride + sbase;
#pragma unroll 4
    for (int it = 0; it < 16; ++it) {
      const uint32_t i = (uint32_t)it * Tt + tau;
      const double2 v = tp[swz64(i)];
      if (active) dst[gidx(i_top | i)] = make_float2((float)v.x, (float)v.y);
    }
  } else if (pd.psi_dst != BUF_NONE) {
    double2* dst = state_ptr(pd.psi_dst);
#pragma unroll 4
    for (int it = 0; it < 16; ++it) {
      const uint32_t i = (uint32_t)it * Tt + tau;
      if (active) dst[gidx(i_top | i)] = tp[swz64(i)];
    }
  }
  if (BWD && pd.lam_dst == LAM_BUF) {
    double2* dst = a.lam + sbase;
#pragma unroll 4
    for (int it = 0; it < 16; ++it) {
      const uint32_t i = (uint32_t)it * Tt + tau;
      if (active) dst[gidx(i_top | i)] = tl[swz64(i)];
    }
  }
  if (!BWD && (pd.flags & PF_EXPECT)) {
    // <psi|O|psi> partial of this tile (Eq. 1, matrix-free as in Appendix B.2)
    double acc = 0.0;
#pragma unroll 1
    for (int it = 0; it < 16; ++it) {
      const uint32_t i = (uint32_t)it * Tt + tau;
      const uint32_t ip = (i_top | i) ^ pd.xm_local;
      const double2 v = tp[swz64(i)];
      const double2 w = ipow(amp(ip, 0), a.y_count);
      const uint32_t sg = __popc(gidx(ip) & a.z_mask) & 1u;
      acc += flipd(v.x * w.x + v.y * w.y, sg);  // Re(conj(v) w) with the Z signs
    }
    for (int off = 1; off < lanes; off <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (Tt >= 32) {
      if (lane == 0) sh.dred[warp] = acc;
      barrier();
      if (tid < tiles_per_cta && rank == 0) {
        const int64_t t2 = first_tile + tid;
        if (t2 < total_tiles) a.e_part[t2] = tile_sum(&sh.dred[tid * wpt], 1);
      }
    } else if (active && (lane & (Tt - 1)) == 0) {
      a.e_part[tile] = acc;
    }
  }
  if (SPLIT) barrier();  // no CTA leaves while another may read its shared memory
}

// ---- observables whose X/Y qubits lie outside the tile (App. B.2) -------------
// CTA (b, t) sums Re(conj(a_x) (O a)_x) over x in [t * chunk, (t + 1) * chunk)
// of sample b; one float64 partial per CTA in the [B][rows] layout of the passes.
__global__ void __launch_bounds__(kThreads) expect_full64_kernel(const double2* psi, int n_eff, int64_t rows,
                                                                 uint32_t xm, uint32_t zm, uint32_t yc,
                                                                 double* e_part) {
  __shared__ double red[kThreads / 32];
  const int64_t dim = 1ll << n_eff;
  const int64_t chunk = dim / rows;
  const int64_t b = blockIdx.x / rows, t = blockIdx.x - b * rows;
  const double2* s = psi + b * dim;
  double acc = 0.0;
  for (int64_t k = threadIdx.x; k < chunk; k += kThreads) {
    const uint32_t x = (uint32_t)(t * chunk + k), xp = x ^ xm;
    const double2 v = s[x];
    const double2 w = ipow(s[xp], yc);
    acc += flipd(v.x * w.x + v.y * w.y, __popc(xp & zm) & 1u);
  }
  for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double sum = 0.0;
    for (int w = 0; w < kThreads / 32; ++w) sum += red[w];
    e_part[blockIdx.x] = sum;
  }
}

// Adjoint seed lambda_x = 2 (dL/dE_b) (O psi_M)_x (Eq. 4) for every amplitude.
__global__ void seed_full64_kernel(const double2* psi, double2* lam, int n_eff, int64_t B, uint32_t xm,
                                   uint32_t zm, uint32_t yc, const double* dLdE) {
  const int64_t dim = 1ll << n_eff;
  const int64_t total = B * dim;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = i >> n_eff;
    const uint32_t x = (uint32_t)(i & (dim - 1)), xp = x ^ xm;
    const double scale = 2.0 * dLdE[b];
    const double2 v = ipow(psi[b * dim + xp], yc);
    const uint32_t sg = __popc(xp & zm) & 1u;
    lam[i] = make_double2(flipd(v.x, sg) * scale, flipd(v.y, sg) * scale);
  }
}

// ---- launchers -------------------------------------------------------------------
cudaError_t launch_pass64(bool bwd, const PassArgs64& a, cudaStream_t st) {
  if (a.pd.K < kRegBits || a.pd.K > kMaxTileBits) return cudaErrorInvalidValue;
  const int tl2 = a.pd.K - kRegBits;
  const int64_t total_tiles = (int64_t)a.B << a.tps_log2;
  if (total_tiles == 0) return cudaSuccess;
  const int n_sm = device_sms();
  if (n_sm == 0) return cudaErrorInvalidDevice;
  const bool rounds = a.rounds != nullptr, rx = rounds && a.rx_items;
  if (rounds && (a.rpar == nullptr || a.pd.K < 7)) return cudaErrorInvalidValue;  // 8 lanes per tile at least
  // Each of an SM's four schedulers has its own FP64 lanes and a warp keeps them
  // busy alone, so the work should sit on all schedulers: CTAs shrink to one tile
  // (one warp at least) while that leaves SMs without one, and two CTAs share a
  // 12-qubit tile. Up to one tile per two SMs both directions gain (152 SMs, n =
  // 12, d = 10, 64 samples: forward 462 -> 304 us, step 1,657 -> 981). Beyond, an
  // adjoint launch gains wherever the busiest SM's part of a tile, ceil(CTAs / SMs)
  // / 2^split, falls by it (adjoint of 160 to 228 samples 2,385 -> 1,845 us, of 500
  // 4,772 -> 4,203, of 2,048 16,718 -> 16,037; where it does not fall, 0.5 % slower).
  // A forward launch gains with one tile too many only (153 samples 891 -> 750 us);
  // its last wave's halves sit two on an SM, and everywhere else it loses 4 % (160
  // to 228 samples 892 -> 923, 500 1,756 -> 1,825, 2,048 6,083 -> 6,342): not split.
  // (Four or eight CTAs per tile gave nothing more: that leaves schedulers idle.)
  int thr = kThreads;
  while (thr > 32 && thr > (1 << tl2) && (total_tiles << tl2) < (int64_t)thr * n_sm) thr >>= 1;
  const int64_t whole = (total_tiles + n_sm - 1) / n_sm, halves = (2 * total_tiles + n_sm - 1) / n_sm;
  const bool evens = bwd ? halves < 2 * whole : 2 * total_tiles <= n_sm;
  const int split = thr == kThreads && thr == 1 << tl2 && evens ? 1 : 0;
  PassArgs64 arg = a;
  arg.split = split;
  thr >>= split;
  const int64_t grid = split ? total_tiles << split : (total_tiles + (thr >> tl2) - 1) / (thr >> tl2);
  const size_t smem = (size_t)(bwd ? 2 : 1) * thr * 16 * sizeof(double2);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)thr);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1u << split;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = split ? 1 : 0;
#define QF_RUN(...)                                                                                            \
  do {                                                                                                         \
    static OptIn once;                                                                                         \
    const cudaError_t e_ =                                                                                     \
        opt_in(reinterpret_cast<const void*>(__VA_ARGS__), 2 * (size_t)kTileAmps * sizeof(double2), once);     \
    if (e_ != cudaSuccess) return e_;                                                                          \
    return cudaLaunchKernelEx(&cfg, __VA_ARGS__, arg);                                                         \
  } while (0)
  if (split) {
    if (bwd && rx) QF_RUN(pass64_kernel<true, true, true, true>);
    if (bwd && rounds) QF_RUN(pass64_kernel<true, true, false, true>);
    if (bwd) QF_RUN(pass64_kernel<true, false, false, true>);
    if (rx) QF_RUN(pass64_kernel<false, true, true, true>);
    if (rounds) QF_RUN(pass64_kernel<false, true, false, true>);
    QF_RUN(pass64_kernel<false, false, false, true>);
  }
  if (bwd && rx) QF_RUN(pass64_kernel<true, true, true>);
  if (bwd && rounds) QF_RUN(pass64_kernel<true, true>);
  if (bwd) QF_RUN(pass64_kernel<true, false>);
  if (rx) QF_RUN(pass64_kernel<false, true, true>);
  if (rounds) QF_RUN(pass64_kernel<false, true>);
  QF_RUN(pass64_kernel<false, false>);
#undef QF_RUN
}

cudaError_t launch_expect_full64(const double2* psi, int n_eff, int64_t B, int64_t rows, uint32_t xm, uint32_t zm,
                                 uint32_t yc, double* e_part, cudaStream_t st) {
  if (B == 0) return cudaSuccess;
  expect_full64_kernel<<<(unsigned)(B * rows), kThreads, 0, st>>>(psi, n_eff, rows, xm, zm, yc, e_part);
  return cudaGetLastError();
}

cudaError_t launch_seed_full64(const double2* psi, double2* lam, int n_eff, int64_t B, uint32_t xm, uint32_t zm,
                               uint32_t yc, const double* dLdE, cudaStream_t st) {
  const int64_t total = B << n_eff;
  if (total == 0) return cudaSuccess;
  const int64_t want = (total + kThreads - 1) / kThreads;
  const unsigned grid = (unsigned)stream_grid(want);
  seed_full64_kernel<<<grid, kThreads, 0, st>>>(psi, lam, n_eff, B, xm, zm, yc, dLdE);
  return cudaGetLastError();
}

}  // namespace qf
