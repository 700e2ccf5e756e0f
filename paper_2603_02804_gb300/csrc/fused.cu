// Fused forward / adjoint pass kernels for sm_103a.
//
// One CTA (256 threads) owns 4096 amplitudes of shared memory per state:
// one tile of K = 12 tile bits, or 2^(12-K) tiles of a smaller circuit (fewer
// where a launch has few tiles, see the launch rule). A
// pass loads its tiles from HBM once (or generates psi_0 in place), runs the
// pass's step program on them in shared memory and registers, and stores them
// once: the forward and backward gate fusion of Secs. 3.2-3.3.
//
// Shared-memory layout: amplitude with local index i lives at i + (i >> 4), one
// 8-byte word of padding per 16, so that the 16 lanes of a half-warp hit 16
// distinct bank pairs for every register group (4 consecutive local bits b ..
// b + 3). The place of register j is then the thread's base plus a constant of
// (b, j): loads and stores of a step carry it as their immediate offset, one
// code copy per b. An XOR swizzle (i ^ ((i >> 4) & 15)) needed an instruction
// or two per address, about 70 a step and thread.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "kernels.h"

namespace qf {

// Sticky device error word (1: a bounded wait gave up); read and cleared by
// qf_device_status.
__device__ int g_qf_device_status = 0;

namespace {

__device__ __forceinline__ constexpr uint32_t loc(uint32_t i) { return i + (i >> 4); }
constexpr int kTilePad = kTileAmps + kTileAmps / 16;  // words of a CTA's share of one state

// Scatter the low bits of src into the set bits of mask (ascending).
__device__ __forceinline__ uint32_t pdep32(uint32_t src, uint32_t mask) {
  uint32_t r = 0;
  for (uint32_t bb = 1; mask; bb <<= 1) {
    const uint32_t low = mask & (0u - mask);
    if (src & bb) r |= low;
    mask ^= low;
  }
  return r;
}

__device__ __forceinline__ float flip(float v, uint32_t s) {
  return __int_as_float(__float_as_int(v) ^ (int)(s << 31));
}

// Pair (i, i+1), i even, to/from the padded tile (two 8-byte accesses, free of
// bank conflicts as the pairs of 16 consecutive lanes are).
__device__ __forceinline__ void st_pair(float2* sm, uint32_t p, float4 v) {
  sm[p] = make_float2(v.x, v.y);
  sm[p + 1] = make_float2(v.z, v.w);
}
__device__ __forceinline__ float4 ld_pair(const float2* sm, uint32_t p) {
  const float2 a = sm[p], b = sm[p + 1];
  return make_float4(a.x, a.y, b.x, b.y);
}

// The registers of a group on local bits B .. B + 3, at the thread's base (NR =
// 16, or 8 on bits B .. B + 2 where two threads share a column).
template <int B>
__device__ __forceinline__ constexpr int group_off(int j) {
  int o = 0;
  for (int r = 0; r < 4; ++r)
    if ((j >> r) & 1) o += (int)loc(1u << (B + r));
  return o;
}
template <int B, int NR>
__device__ __forceinline__ void ld_regs(const float2* at, float2 (&r)[NR]) {
#pragma unroll
  for (int j = 0; j < NR; ++j) r[j] = at[group_off<B>(j)];
}
template <int B, int NR>
__device__ __forceinline__ void st_regs(float2* at, const float2 (&r)[NR]) {
#pragma unroll
  for (int j = 0; j < NR; ++j) at[group_off<B>(j)] = r[j];
}
// The group's lowest local bit b is one of these in round programs (K = 7 .. 11:
// 0, 4 and K - 4; KC = 12: 0, 4, 8). at2: lambda's place (adjoint).
template <int KC, bool BWD, int NR>
__device__ __forceinline__ void ld_group(uint32_t b, const float2* at, const float2* at2, float2 (&r)[NR],
                                         float2 (&l)[NR]) {
#define QF_LD(B) { ld_regs<B>(at, r); if (BWD) ld_regs<B>(at2, l); }
  if (KC == 12) {
    if (b == 0) QF_LD(0) else if (b == 4) QF_LD(4) else QF_LD(8)
  } else {
    switch (b) {
      case 0: QF_LD(0) break;
      case 3: QF_LD(3) break;
      case 5: QF_LD(5) break;
      case 6: QF_LD(6) break;
      case 7: QF_LD(7) break;
      default: QF_LD(4) break;
    }
  }
#undef QF_LD
}
template <int KC, bool BWD, int NR>
__device__ __forceinline__ void st_group(uint32_t b, float2* at, float2* at2, const float2 (&r)[NR],
                                         const float2 (&l)[NR]) {
#define QF_ST(B) { st_regs<B>(at, r); if (BWD) st_regs<B>(at2, l); }
  if (KC == 12) {
    if (b == 0) QF_ST(0) else if (b == 4) QF_ST(4) else QF_ST(8)
  } else {
    switch (b) {
      case 0: QF_ST(0) break;
      case 3: QF_ST(3) break;
      case 5: QF_ST(5) break;
      case 6: QF_ST(6) break;
      case 7: QF_ST(7) break;
      default: QF_ST(4) break;
    }
  }
#undef QF_ST
}

// ---- forward: fused 2x2 on register bit R -----------------------------------
template <int R>
__device__ __forceinline__ void apply_u(float2 (&r)[16], const float4 m0, const float4 m1) {
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    if (j & (1 << R)) continue;
    const int j1 = j | (1 << R);
    const float2 x = r[j], y = r[j1];
    r[j].x = m0.x * x.x - m0.y * x.y + m0.z * y.x - m0.w * y.y;
    r[j].y = m0.x * x.y + m0.y * x.x + m0.z * y.y + m0.w * y.x;
    r[j1].x = m1.x * x.x - m1.y * x.y + m1.z * y.x - m1.w * y.y;
    r[j1].y = m1.x * x.y + m1.y * x.x + m1.z * y.y + m1.w * y.x;
  }
}

// ---- backward: un-apply one rotation to psi and lambda on register bit R and
// return sum over the thread's pairs of Im<lambda|P|psi> taken before the
// un-apply. With du/dt = -(i/2) P u (Sec. 3.3), Re<lambda_j|du|psi_{j-1}> =
// (1/2) Im<lambda_j|P|psi_j>; the 1/2 is applied in float64 at the flush.
template <int R, int KIND>
__device__ __forceinline__ float bwd_gate(float2 (&p)[16], float2 (&l)[16], const float c,
                                          const float s) {
  float acc = 0.f;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    if (j & (1 << R)) continue;
    const int j1 = j | (1 << R);
    const float2 p0 = p[j], p1 = p[j1], l0 = l[j], l1 = l[j1];
    if (KIND == G_RZ) {
      acc += l0.x * p0.y - l0.y * p0.x - l1.x * p1.y + l1.y * p1.x;
      // u^dagger = diag(c + i s, c - i s)
      p[j] = make_float2(c * p0.x - s * p0.y, c * p0.y + s * p0.x);
      p[j1] = make_float2(c * p1.x + s * p1.y, c * p1.y - s * p1.x);
      l[j] = make_float2(c * l0.x - s * l0.y, c * l0.y + s * l0.x);
      l[j1] = make_float2(c * l1.x + s * l1.y, c * l1.y - s * l1.x);
    } else if (KIND == G_RY) {
      acc += l1.x * p0.x + l1.y * p0.y - l0.x * p1.x - l0.y * p1.y;
      // u^dagger = [[c, s], [-s, c]]
      p[j] = make_float2(c * p0.x + s * p1.x, c * p0.y + s * p1.y);
      p[j1] = make_float2(c * p1.x - s * p0.x, c * p1.y - s * p0.y);
      l[j] = make_float2(c * l0.x + s * l1.x, c * l0.y + s * l1.y);
      l[j1] = make_float2(c * l1.x - s * l0.x, c * l1.y - s * l0.y);
    } else {  // RX
      acc += l0.x * p1.y - l0.y * p1.x + l1.x * p0.y - l1.y * p0.x;
      // u^dagger = [[c, i s], [i s, c]]
      p[j] = make_float2(c * p0.x - s * p1.y, c * p0.y + s * p1.x);
      p[j1] = make_float2(c * p1.x - s * p0.y, c * p1.y + s * p0.x);
      l[j] = make_float2(c * l0.x - s * l1.y, c * l0.y + s * l1.x);
      l[j1] = make_float2(c * l1.x - s * l0.y, c * l1.y + s * l0.x);
    }
  }
  return acc;
}

template <int KIND>
__device__ __forceinline__ float bwd_dispatch_r(uint32_t r, float2 (&p)[16], float2 (&l)[16], float c,
                                                float s) {
  switch (r) {
    case 0: return bwd_gate<0, KIND>(p, l, c, s);
    case 1: return bwd_gate<1, KIND>(p, l, c, s);
    case 2: return bwd_gate<2, KIND>(p, l, c, s);
    default: return bwd_gate<3, KIND>(p, l, c, s);
  }
}

// CNOT with its target on register bit RT: swap the target pairs whose
// control is 1 (control: register bit cb when creg, else bit cb of the
// thread's base index gb). Self-inverse, so the adjoint applies the same.
template <int RT, bool BWD>
__device__ __forceinline__ void cnot_regs(float2 (&r)[16], float2 (&l)[16], bool creg, uint32_t cb, uint32_t gb) {
  const uint32_t cg = (gb >> cb) & 1u;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    if (j & (1 << RT)) continue;
    const int j1 = j | (1 << RT);
    const bool on = creg ? (((uint32_t)j >> cb) & 1u) != 0 : cg != 0;
    const float2 a = r[j], b = r[j1];
    r[j] = on ? b : a;
    r[j1] = on ? a : b;
    if (BWD) {
      const float2 c = l[j], d = l[j1];
      l[j] = on ? d : c;
      l[j1] = on ? c : d;
    }
  }
}

__device__ __forceinline__ uint32_t reg_off(uint32_t j, const uint32_t (&o)[4]) {
  return ((j & 1u) ? o[0] : 0u) + ((j & 2u) ? o[1] : 0u) + ((j & 4u) ? o[2] : 0u) + ((j & 8u) ? o[3] : 0u);
}

// phase i^k times v
__device__ __forceinline__ float2 mul_ipow(float2 v, uint32_t k) {
  switch (k & 3u) {
    case 0: return v;
    case 1: return make_float2(-v.y, v.x);
    case 2: return make_float2(-v.x, -v.y);
    default: return make_float2(v.y, -v.x);
  }
}

// ---- round programs: pending CZ signs ------------------------------------------
// A thread's 16 registers hold psi~ with psi = D psi~, where D = (-1)^(c0 +
// sum_r A_r j_r) is the part of the CZ signs that is constant or linear in the
// register index j (bit 4 of D: c0, bits 0..3: A). D commutes with every
// diagonal gate; a gate on register bit r only sees the factor Z_r^(A_r),
// which is folded into that gate. CZs between two register bits (quadratic in
// j, the same for every thread) are signs of the round's diagonal table. A
// link that leaves the register group stays pending beyond its step, as a bit
// of `pend`: the next step starts from the D that pend gives its threads. It
// is applied only where the plan says so (a later group holds both its qubits,
// a checkpoint, the end of the pass). Applying D at every step took 80 of the
// adjoint's instructions per step and thread (n = 20, d = 24, 64 samples: step
// 26.12 -> 25.10 ms).
//
// Links L of one round, thread base index gb (register bits zero), register
// bit positions p[r]: x = gb ^ y(j) with disjoint supports, so each link q
// contributes gb_q gb_{q+1} (constant), gb_{q} y_{q+1} or y_q gb_{q+1} (linear)
// or y_q y_{q+1} (between register bits).
// Link q couples qubit q with q+1 mod n (link n-1 is a ring's CZ(n-1, 0); it
// never joins two register bits), hence the n-bit rotations.
__device__ __forceinline__ void link_terms(uint32_t L, uint32_t gb, int n, uint32_t& t2, uint32_t& u) {
  const uint32_t nmask = n >= 32 ? ~0u : ((1u << n) - 1u);
  const uint32_t t1 = L & gb;
  t2 = L & (((gb >> 1) | ((gb & 1u) << (n - 1))) & nmask);
  u = (((t1 << 1) | (t1 >> (n - 1))) & nmask) ^ t2;
}

// The pending-sign update of one round's links, from per-step constants of
// the thread (rgb = gb rotated right by one qubit, lgb = left, g12 = gb &
// rgb): as rotation distributes over &, u = rotl(L) & lgb ^ L & rgb (the
// link_terms u), and the constant part is |L & g12|. When the register bits
// sit on consecutive qubits (kContig), A is one shift of u. qubits: those of
// the register bits, a byte each.
constexpr uint32_t kContig = 0x80u;
__device__ __forceinline__ void chain_pending(uint32_t L, uint32_t rgb, uint32_t lgb, uint32_t g12, int n,
                                                uint32_t qubits, uint32_t& D) {
  // (lgb has no bits from n on, so the rotation of L needs no mask of its own)
  const uint32_t u = (((L << 1) | (L >> (n - 1))) & lgb) ^ (L & rgb);
  const uint32_t A = (qubits & kContig) ? (u >> (qubits & 31u)) & 15u
                                        : ((u >> (qubits & 31u)) & 1u) | (((u >> ((qubits >> 8) & 31u)) & 1u) << 1) |
                                              (((u >> ((qubits >> 16) & 31u)) & 1u) << 2) |
                                              (((u >> ((qubits >> 24) & 31u)) & 1u) << 3);
  D ^= A | ((__popc(L & g12) & 1u) << 4);
}

// Multiply the registers by D (end of a step).
template <bool BWD, int NR>
__device__ __forceinline__ void apply_pending(uint32_t D, float2 (&r)[NR], float2 (&l)[NR]) {
  uint32_t S = (D & 16u) ? 0xFFFFu : 0u;
  S ^= (D & 1u) ? 0xAAAAu : 0u;
  S ^= (D & 2u) ? 0xCCCCu : 0u;
  S ^= (D & 4u) ? 0xF0F0u : 0u;
  S ^= (D & 8u) ? 0xFF00u : 0u;
#pragma unroll
  for (int j = 0; j < NR; ++j) {
    const int f = (int)((S << (31 - j)) & 0x80000000u);
    r[j].x = __int_as_float(__float_as_int(r[j].x) ^ f);
    r[j].y = __int_as_float(__float_as_int(r[j].y) ^ f);
    if (BWD) {
      l[j].x = __int_as_float(__float_as_int(l[j].x) ^ f);
      l[j].y = __int_as_float(__float_as_int(l[j].y) ^ f);
    }
  }
}

// One rotation of a round on register bit R, two FMAs per real component:
//   RY: p0 -= q p1; p1 += q p0      RX: p0 -= i q p1; p1 -= i q p0
// (old values on the right), i.e. [[1, -q], [q, 1]] or [[1, -iq], [-iq, 1]]: the
// rotation by w over cos(w/2), with q = tan(w/2). The cosines of a round's four
// rotations are one scale of the state, multiplied into the 16 phases of the
// round's diagonal, which the kernel applies anyway. q is rounded before the
// scale is made from it, so that the norm is kept; a large q costs no accuracy,
// as the scaled result is rounded once. The scale of a round stays above 2^-32:
// where the four squared cosines multiply to less than kMinShrink = 2^-64 (a
// round of four angles within 0.008 of pi, or of two that are pi in float32), the
// rotations run twice, by half the angles (|q| <= 1). Their second run is a branch
// at an edge of the round's block (before it in the forward, after it in the
// adjoint): in the middle it cost every adjoint round 3 %. A step with every
// angle at pi against uniform angles: n = 12, d = 20, 256 samples 267 us against
// 211; ring of RX, RY, RZ, n = 12, d = 10, 256 samples 256 against 200 (a second run of the whole
// round, where any |tan(w/2)| > 256: 339 against 216, 330 against 200). Three shears (3 FMAs per component) need no scale and
// were slower: training step of n = 20, d = 24, 64 samples 28.35 -> 25.10 ms, of
// n = 12, d = 20, 256 samples 268 -> 237 us (with the pending links below). A
// pending Z_R turns the rotation by w into one by -w, i.e. q into -q.
template <int R, bool RX, int NR>
__device__ __forceinline__ void rot_T(float2 (&r)[NR], float q, bool rx) {
  if (RX && rx) {
#pragma unroll
    for (int j = 0; j < NR; ++j) {
      if (j & (1 << R)) continue;
      const int j1 = j | (1 << R);
      const float2 p0 = r[j], p1 = r[j1];
      r[j] = make_float2(fmaf(q, p1.y, p0.x), fmaf(-q, p1.x, p0.y));
      r[j1] = make_float2(fmaf(q, p0.y, p1.x), fmaf(-q, p0.x, p1.y));
    }
  } else {
    // RY is real: the same on re and im, one packed FFMA2 each
    const float2 q2 = make_float2(q, q), n2 = make_float2(-q, -q);
#pragma unroll
    for (int j = 0; j < NR; ++j) {
      if (j & (1 << R)) continue;
      const int j1 = j | (1 << R);
      const float2 p0 = r[j];
      r[j] = __ffma2_rn(n2, r[j1], p0);
      r[j1] = __ffma2_rn(q2, p0, r[j1]);
    }
  }
}

// q with the sign of a pending Z (a = 1).
__device__ __forceinline__ float pend_q(float q, uint32_t a) {
  return __int_as_float(__float_as_int(q) ^ (int)(a << 31));
}

// v *= (c + i s)
__device__ __forceinline__ void cmul(float2& v, float c, float s) {
  const float x = v.x;
  v.x = fmaf(c, x, -s * v.y);
  v.y = fmaf(s, x, c * v.y);
}

// The round's diagonal (its 4 RZ runs merged), applied: register amplitude j
// times the phase (cos, sin) held in ph[j / 2] (x, y for even j; z, w for odd
// j). An RZ run commutes with the rotations on the other register bits and
// with the pending signs, so the four run together, once per round, after the
// rotations (the adjoint un-applies them before its rotations, diag_bwd).
template <int NR>
__device__ __forceinline__ void apply_diag(float2 (&r)[NR], const float4* ph) {
#pragma unroll
  for (int m = 0; m < NR / 2; ++m) {
    const float4 e = ph[m];
    cmul(r[2 * m], e.x, e.y);
    cmul(r[2 * m + 1], e.z, e.w);
  }
}

// Adjoint side of the round's diagonal: its RZ-run gradient terms, then the
// un-apply. g[r] = sum_j sigma_r(j) w_j with w_j = Im(conj(lambda_j) psi_j)
// and sigma_r(j) = +1 where bit r of j is clear, else -1 (the thread's share
// of Im<lambda|Z_r|psi>). w_j is unchanged by a diagonal acting on both states
// and Z_r commutes with the rotations on the other bits, so the four terms
// are taken together at the diagonal. sigma_r(15 - j) = -sigma_r(j), so the
// differences u_j = w_j - w_{15-j} (four products in one chain, no sum of
// their own) carry all four: g[3] is their sum T, g[r] = 2 H_r - T with H_r
// the sum over the u_j with bit r clear: 14 additions instead of 42 for a
// transform of the 16 w_j.
__device__ __forceinline__ void diag_bwd(float2 (&p)[16], float2 (&l)[16], const float4* ph, float (&g)[8]) {
  float u[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const float2 p0 = p[m], l0 = l[m], p1 = p[15 - m], l1 = l[15 - m];
    u[m] = fmaf(l1.y, p1.x, fmaf(-l1.x, p1.y, fmaf(l0.x, p0.y, -l0.y * p0.x)));
  }
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const float4 e = ph[m];
    cmul(p[2 * m], e.x, e.y);
    cmul(l[2 * m], e.x, e.y);
    cmul(p[2 * m + 1], e.z, e.w);
    cmul(l[2 * m + 1], e.z, e.w);
  }
  const float a0 = u[0] + u[1], a1 = u[2] + u[3], a2 = u[4] + u[5], a3 = u[6] + u[7];
  const float q0 = a0 + a1, T = q0 + (a2 + a3);
  const float h0 = (u[0] + u[2]) + (u[4] + u[6]), h1 = a0 + a2;
  g[0] = fmaf(2.f, h0, -T);
  g[1] = fmaf(2.f, h1, -T);
  g[2] = fmaf(2.f, q0, -T);
  g[3] = T;
}

// The gradient value of an adjoint item's rotation on register bit R (RX where
// rx, uniform over the CTA, else RY): the thread's sum of Im<lambda|P|psi>, after
// the round's diagonal and before any of its rotations (they commute with P on
// the other bits). A pending Z_R (a) negates it. The round's scale multiplies it
// by a factor that is the same for every thread and sample; the owner lane of
// the reduced sum undoes it (the table's factor). All four values before the
// rotations, and psi's rotations before lambda's, need fewer registers at a time
// than rotation by rotation: adjoint of n = 20, d = 24, 64 samples 1.258 -> 1.244
// ms a launch. (A steep round takes them before its first run.)
template <int R, bool RX, int NR>
__device__ __forceinline__ float grad_T(const float2 (&p)[NR], const float2 (&l)[NR], uint32_t a, bool rx) {
  float g;
  if (RX && rx) {
    g = 0.f;
#pragma unroll
    for (int j = 0; j < NR; ++j) {
      if (j & (1 << R)) continue;
      const int j1 = j | (1 << R);
      g += l[j].x * p[j1].y - l[j].y * p[j1].x + l[j1].x * p[j].y - l[j1].y * p[j].x;
    }
  } else {
    // l1 . p0 - l0 . p1 per pair (component-wise products, two packed sums)
    float2 accp = make_float2(0.f, 0.f), accm = make_float2(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < NR; ++j) {
      if (j & (1 << R)) continue;
      const int j1 = j | (1 << R);
      accp = __ffma2_rn(l[j1], p[j], accp);
      accm = __ffma2_rn(l[j], p[j1], accm);
    }
    g = (accp.x + accp.y) - (accm.x + accm.y);
  }
  return pend_q(g, a);
}
// A round's rotations on register bits 0 .. 2 (a half column) or 0 .. 3 of one state.
template <bool RX, int NR>
__device__ __forceinline__ void rots(float2 (&z)[NR], const float4* v, uint32_t D, uint32_t rx) {
  rot_T<0, RX>(z, pend_q(v[0].x, D & 1u), rx & 1u);
  rot_T<1, RX>(z, pend_q(v[1].x, (D >> 1) & 1u), (rx >> 1) & 1u);
  rot_T<2, RX>(z, pend_q(v[2].x, (D >> 2) & 1u), (rx >> 2) & 1u);
  if constexpr (NR == 16) rot_T<3, RX>(z, pend_q(v[3].x, (D >> 3) & 1u), (rx >> 3) & 1u);
}

// The same item by item, where an item may be an RX: one branch per item takes
// its value and rotates both states (value by value, then state by state, took
// 1.28 ms a launch of 100 states of 20 qubits, this 1.25). The value then carries
// the earlier items' rotations (the table's .z).
template <int R>
__device__ __forceinline__ void item_bwd(float2 (&p)[16], float2 (&l)[16], float qt, uint32_t a, float& gy, bool rx) {
  const float q = pend_q(qt, a);
  gy = grad_T<R, true>(p, l, a, rx);
  rot_T<R, true>(p, q, rx);
  rot_T<R, true>(l, q, rx);
}

// ---- two threads per column ------------------------------------------------------
// A launch of few tiles leaves each scheduler a warp or two, and its time is a
// warp's latency through its instructions. There two neighbouring threads share
// a column (thread h holds the 8 registers with bit 3 of the index equal to h),
// each with half the instructions; the rotation on bit 3 fetches the partner's
// amplitudes by shuffles.
__device__ __forceinline__ void partner(const float2 (&r)[8], float2 (&o)[8]) {
#pragma unroll
  for (int j = 0; j < 8; ++j)
    o[j] = make_float2(__shfl_xor_sync(0xffffffffu, r[j].x, 1), __shfl_xor_sync(0xffffffffu, r[j].y, 1));
}
// rot_T on bit 3: o holds the partner's amplitudes.
template <bool RX>
__device__ __forceinline__ void rot_half(float2 (&r)[8], const float2 (&o)[8], float q, uint32_t h, bool rx) {
  if (RX && rx) {
#pragma unroll
    for (int j = 0; j < 8; ++j) r[j] = make_float2(fmaf(q, o[j].y, r[j].x), fmaf(-q, o[j].x, r[j].y));
  } else {
    const float qh = pend_q(q, h ^ 1u);  // p0 -= q p1; p1 += q p0
    const float2 q2 = make_float2(qh, qh);
#pragma unroll
    for (int j = 0; j < 8; ++j) r[j] = __ffma2_rn(q2, o[j], r[j]);
  }
}
template <bool RX>
__device__ __forceinline__ void rot_fwd_half(float2 (&r)[8], float q, uint32_t h, bool rx) {
  float2 o[8];
  partner(r, o);
  rot_half<RX>(r, o, q, h, rx);
}
// The gradient value and the rotation of an adjoint item on bit 3; gy: the
// thread's share (l_1 . p_0 in thread 1, -l_0 . p_1 in thread 0).
template <bool RX>
__device__ __forceinline__ void rot_bwd_half(float2 (&p)[8], float2 (&l)[8], float qt, uint32_t a, float& gy, uint32_t h,
                                             bool rx) {
  const float q = pend_q(qt, a);
  float2 o[8];
  partner(p, o);
  float g;
  if (RX && rx) {
    g = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) g += l[j].x * o[j].y - l[j].y * o[j].x;
  } else {
    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < 8; ++j) acc = __ffma2_rn(l[j], o[j], acc);
    g = pend_q(acc.x + acc.y, h ^ 1u);
  }
  rot_half<RX>(p, o, q, h, rx);
  partner(l, o);
  rot_half<RX>(l, o, q, h, rx);
  gy = pend_q(g, a);
}
// diag_bwd of a half column: bits 0..2 from the complements 7 - j, bit 3 from
// the whole sum, signed by the half.
__device__ __forceinline__ void diag_bwd(float2 (&p)[8], float2 (&l)[8], const float4* ph, float (&g)[8], uint32_t h) {
  float u[4], t[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const float2 p0 = p[m], l0 = l[m], p1 = p[7 - m], l1 = l[7 - m];
    const float w0 = fmaf(l0.x, p0.y, -l0.y * p0.x), w1 = fmaf(l1.x, p1.y, -l1.y * p1.x);
    u[m] = w0 - w1;
    t[m] = w0 + w1;
  }
  apply_diag(p, ph);
  apply_diag(l, ph);
  const float q0 = u[0] + u[1], T = q0 + (u[2] + u[3]);
  g[0] = fmaf(2.f, u[0] + u[2], -T);
  g[1] = fmaf(2.f, q0, -T);
  g[2] = T;
  g[3] = pend_q((t[0] + t[1]) + (t[2] + t[3]), h);
}

// Reduce 8 per-thread values over `lanes` lanes (8, 16 or 32; whole-warp
// call). Afterwards lane holds the lanes-sum of value *idx; the lanes with
// (lane & (lanes/8 - 1)) == 0 hold the 8 distinct values.
__device__ __forceinline__ float butterfly8(float (&v)[8], int lanes, int lane, int& idx) {
  int o = lanes >> 1;
  bool up = (lane & o) != 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float send = up ? v[i] : v[i + 4];
    const float keep = up ? v[i + 4] : v[i];
    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
  }
  idx = up ? 4 : 0;
  o >>= 1;
  up = (lane & o) != 0;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const float send = up ? v[i] : v[i + 2];
    const float keep = up ? v[i + 2] : v[i];
    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
  }
  idx += up ? 2 : 0;
  o >>= 1;
  up = (lane & o) != 0;
  {
    const float send = up ? v[0] : v[1];
    const float keep = up ? v[1] : v[0];
    v[0] = keep + __shfl_xor_sync(0xffffffffu, send, o);
  }
  idx += up ? 1 : 0;
  for (o >>= 1; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
  return v[0];
}

// The same through shared memory: rows of the warp's own [32 lanes][8 values].
// A lane then holds the sum over its tile's lanes of value lane & 7 (rows
// parts * k + part of its tile, so that the 32 lanes read 32 banks for whole-
// warp tiles). Two stores, eight loads and two shuffles in place of nine
// shuffles and fourteen selects (661 -> 649 instructions per warp and round of
// the adjoint): adjoint of n = 16, d = 100, 64 samples 98.9 -> 97.4 us a launch.
__device__ __forceinline__ float rows8(const float (&v)[8], int lanes, int lane, float (&rows)[32][8]) {
  float4* own = reinterpret_cast<float4*>(rows[lane]);
  __syncwarp();  // the reads of the previous round are done
  own[0] = make_float4(v[0], v[1], v[2], v[3]);
  own[1] = make_float4(v[4], v[5], v[6], v[7]);
  __syncwarp();
  const int parts = lanes >> 3;
  const int at = (lane & ~(lanes - 1)) + ((lane & (lanes - 1)) >> 3);
  float s[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) s[k] = rows[at + parts * k][lane & 7];
  float sum = ((s[0] + s[1]) + (s[2] + s[3])) + ((s[4] + s[5]) + (s[6] + s[7]));
  if (parts >= 2) sum += __shfl_xor_sync(0xffffffffu, sum, 8);
  if (parts == 4) sum += __shfl_xor_sync(0xffffffffu, sum, 16);
  return sum;
}

// Two amplitudes as bfloat16 (re, im) pairs <-> float32 (round to nearest even).
__device__ __forceinline__ float4 bf16x4_to_f4(uint2 h) {
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&h.x));
  const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&h.y));
  return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ uint2 f4_to_bf16x4(float4 v) {
  const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
  return make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
}

// 16-byte asynchronous copy global -> shared (L2 only), and its fences.
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// Parameters of one round step, staged from the round-ordered tables: per
// round kRoundPar float4 (the items' rotations, then the round's diagonal) and
// the round record.
constexpr int kMaxRoundWords = kFwdRoundWords > kBwdRoundWords ? kFwdRoundWords : kBwdRoundWords;
struct StepPar {
  float4 v[kMaxStepRounds][kRoundPar];
  uint4 rec[kMaxStepRounds * (kMaxRoundWords / 4)];
};

// ---- tensor-core block path (tcgen05) --------------------------------------------
// A forward round applies u3 (x) u2 (x) u1 (x) u0 to the 16 amplitudes of a
// register group: a 16x16 complex block, i.e. a 32x32 real matrix on the
// (re, im) vector. A warpgroup's 128 columns (one per thread) form the MMA's
// M = 128 rows: D[m][n] = sum_k A[m][k] B[n][k], A = the columns' amplitudes
// (k < 16: re of amplitude k, else im of amplitude k - 16) in tensor memory,
// B = the round's real matrix (K-major, in shared memory), D in tensor memory.
// Split precision (3xTF32): A = Ah + Al, B = Bh + Bl with TF32 parts, and
// D = Ah Bh + Ah Bl + Al Bh accumulated in float32.
constexpr int kTcCols = 256;            // tensor-memory columns per CTA
constexpr int kTcWgCols = 96;           // per warpgroup: D, A hi, A lo (32 each)
constexpr int kTcBFloats = 2 * 1024;    // one round's B: hi then lo, 32x32 each
constexpr long long kTcSpinLimit = 1ll << 26;

// idesc for kind::tf32: D f32 (bits 4-5 = 1), A and B tf32 (bits 7-9, 10-12 = 2),
// both K-major, N >> 3 at bits 17-22, M >> 4 at bits 24-28.
constexpr uint32_t kTcIdesc = (1u << 4) | (2u << 7) | (2u << 10) | ((32u >> 3) << 17) | ((128u >> 4) << 24);

// Shared-memory descriptor, K-major without swizzle: 8-row x 16-byte core
// matrices; LBO = 128 B between core matrices along K, SBO = 1024 B between
// 8-row groups; version 1 (bit 46).
__device__ __forceinline__ uint64_t tc_bdesc(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)(128u >> 4) << 16) | ((uint64_t)(1024u >> 4) << 32) |
         (1ull << 46);
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint32_t cvt_tf32(float v) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(v));
  return r;
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void tc_mma(uint32_t d, uint32_t a, uint64_t bdesc, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.u32 p, %3, 0;\n"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %4, p;\n}\n" ::"r"(d),
      "r"(a), "l"(bdesc), "r"(acc), "r"(kTcIdesc)
      : "memory");
}

__device__ __forceinline__ void tc_commit(uint64_t* mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(mbar))
               : "memory");
}

// Wait for the mbarrier phase with the given parity; false after the spin limit.
__device__ __forceinline__ bool mbar_wait(uint64_t* mbar, uint32_t parity) {
  const uint32_t addr = smem_u32(mbar);
  for (long long it = 0; it < kTcSpinLimit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(addr), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

#define QF_R8(b) "%" #b "0, %" #b "1, %" #b "2, %" #b "3, %" #b "4, %" #b "5, %" #b "6, %" #b "7"

__device__ __forceinline__ void tc_st32(uint32_t taddr, const uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
      "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
      "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]), "r"(v[18]),
      "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]),
      "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
      : "memory");
}

__device__ __forceinline__ void tc_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t u[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]), "=r"(u[8]),
        "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]), "=r"(u[15]), "=r"(u[16]),
        "=r"(u[17]), "=r"(u[18]), "=r"(u[19]), "=r"(u[20]), "=r"(u[21]), "=r"(u[22]), "=r"(u[23]), "=r"(u[24]),
        "=r"(u[25]), "=r"(u[26]), "=r"(u[27]), "=r"(u[28]), "=r"(u[29]), "=r"(u[30]), "=r"(u[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int k = 0; k < 32; ++k) v[k] = __uint_as_float(u[k]);
}

// Per-CTA state of the tensor-core path.
struct TcCtx {
  uint32_t tmem;    // tensor-memory base (lane 0, first column)
  uint64_t* mbar;   // [2] one per warpgroup, in shared memory
  float* bsm;       // B staging: [2][kMaxStepRounds][kTcBFloats]
};

// Sign mask over the 16 register indices j of the round's CZ links (x = gb ^
// y(j)): constant part, parts linear in one register bit, and links between
// two register bits (bbits).
__device__ __forceinline__ uint32_t cz_mask16(uint32_t L, uint32_t bbits, uint32_t gb, const uint32_t (&p)[4], int n) {
  uint32_t t2, u;
  link_terms(L, gb, n, t2, u);
  uint32_t S = (__popc(t2 & gb) & 1u) ? 0xFFFFu : 0u;
  S ^= ((u >> p[0]) & 1u) ? 0xAAAAu : 0u;
  S ^= ((u >> p[1]) & 1u) ? 0xCCCCu : 0u;
  S ^= ((u >> p[2]) & 1u) ? 0xF0F0u : 0u;
  S ^= ((u >> p[3]) & 1u) ? 0xFF00u : 0u;
  S ^= (bbits & 1u) ? 0x8888u : 0u;
  S ^= (bbits & 2u) ? 0xC0C0u : 0u;
  S ^= (bbits & 4u) ? 0xF000u : 0u;
  return S;
}

// The rounds of one forward step on the tensor cores. r holds the thread's 16
// amplitudes (its column) on entry and exit. Warpgroup wg issues its own MMAs
// (M = its 128 columns) and waits on its own mbarrier; ph tracks the phase.
__device__ __forceinline__ void tc_rounds(const TcCtx& tc, const StepPar& P, int nr, const float* bst, uint32_t gb,
                                          const uint32_t (&pos)[4], int n, float2 (&r)[16], uint32_t& ph, int tid) {
  const int wg = tid >> 7, wq = (tid >> 5) & 3;
  const uint32_t col0 = tc.tmem + (uint32_t)(wg * kTcWgCols);
  const uint32_t lane_off = (uint32_t)(32 * wq) << 16;
  const uint32_t d_col = col0, ah_col = col0 + 32, al_col = col0 + 64;
  float x[32];
  float n0 = 0.f;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    x[j] = r[j].x;
    x[16 + j] = r[j].y;
    n0 = fmaf(x[j], x[j], fmaf(x[16 + j], x[16 + j], n0));
  }
#pragma unroll 1
  for (int k = 0; k < nr; ++k) {
    {
      uint32_t hi[32], lo[32];
#pragma unroll
      for (int q = 0; q < 32; ++q) {
        hi[q] = cvt_tf32(x[q]);
        lo[q] = cvt_tf32(x[q] - __uint_as_float(hi[q]));
      }
      tc_st32(ah_col | lane_off, hi);
      tc_st32(al_col | lane_off, lo);
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    asm volatile("bar.sync %0, 128;" ::"r"(1 + wg) : "memory");
    if ((tid & 127) == 0) {
      tc_fence_after();
      const uint32_t bh = smem_u32(bst + (size_t)k * kTcBFloats), bl = bh + 4096u;
#pragma unroll
      for (int pr = 0; pr < 3; ++pr) {
        const uint32_t a = pr == 2 ? al_col : ah_col;
        const uint32_t b = pr == 1 ? bl : bh;
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          tc_mma(d_col, a + 8u * kk, tc_bdesc(b + 256u * kk), (pr | kk) != 0 ? 1u : 0u);
      }
      tc_commit(tc.mbar + wg);
    }
    if (!mbar_wait(tc.mbar + wg, ph)) atomicExch(&g_qf_device_status, 1);
    ph ^= 1u;
    tc_fence_after();
    tc_ld32(d_col | lane_off, x);
    // CZ links after this round's rotations
    const uint4 lk = P.rec[k * (kFwdRoundWords / 4) + 1];
    const uint32_t S = cz_mask16(lk.x, lk.y, gb, pos, n);
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const int f = (int)((S << (31 - j)) & 0x80000000u);
      x[j] = __int_as_float(__float_as_int(x[j]) ^ f);
      x[16 + j] = __int_as_float(__float_as_int(x[16 + j]) ^ f);
    }
  }
  tc_fence_before();
  // The step acts on the column by a unitary (rotations and CZ signs), so its
  // norm is invariant; the tensor cores' float32 accumulation rounds toward
  // zero and shrinks it by a few ulp per round. Restore the norm.
  float n1 = 0.f;
#pragma unroll
  for (int q = 0; q < 32; ++q) n1 = fmaf(x[q], x[q], n1);
  const float sc = n1 > 0.f ? sqrtf(n0 / n1) : 1.f;
#pragma unroll
  for (int j = 0; j < 16; ++j) r[j] = make_float2(x[j] * sc, x[16 + j] * sc);
}

}  // namespace

// ---------------------------------------------------------------------------
// Static shared memory of a pass (the tiles themselves are dynamic).
template <class Y>
__device__ void loss_block(int kind, double* E, const Y* y, int64_t B, double scale, double* loss, double* dLdE,
                           const double* e_part, int tps, int tid, int nthr);

// dL/dE of sample b (a late loss: from the sample's own E, one tile per sample).
__device__ __forceinline__ double seed_dl(const PassArgs& a, int64_t b) {
  if (a.dLdE) return a.dLdE[b];
  return a.loss_kind == 1 ? a.loss_scale * (a.e_part[b] - (double)a.y[b]) : 1.0;
}

// Round programs seed lambda with dL/dE / 2^e, e its exponent, and multiply the
// gradient partials by 2^e in float64 (exact, both): a round's scale (rot_T) takes
// up to 2^64 off the products of lambda and psi, and with a small dL/dE they left
// float32's range (1e-24 and angles 0.009 from pi: gradients 36 % off).
__device__ __forceinline__ int grad_exponent(double dl) {
  const int e = ((__double2hiint(dl) >> 20) & 0x7ff) - 1023;
  return e > -800 && e < 800 ? e : 0;  // (zero, infinities and NaN go as they are)
}
__device__ __forceinline__ double pow2(int e) { return __hiloint2double((1023 + e) << 20, 0); }
// A partial v / 2 times 2^e. A float64 product is a latency that the summing warp
// brings to the step's next barrier: small tiles, whose steps are short, add to the
// exponent's bits instead (n = 7, d = 20, 64 samples 75.6 -> 74.3 us a step; 12-qubit
// tiles are slower by it, n = 20, d = 8, 64 samples 8.40 -> 8.46 ms).
template <bool BITS>
__device__ __forceinline__ double partial(float v, int e) {
  if (!BITS) return (double)v * pow2(e - 1);
  const double d = (double)(0.5f * v);
  const int hi = __double2hiint(d);
  const bool number = (uint32_t)(hi & 0x7ff00000) - 0x00100000u < 0x7fe00000u;  // not 0, infinite or NaN
  return __hiloint2double(number ? hi + e * (1 << 20) : hi, __double2loint(d));
}

template <bool ROWS>
struct PassSharedT {
  StepPar par[2];
  float rows[ROWS ? kThreads / 32 : 1][32][8];  // round adjoints: a round's values of each lane
  int32_t gexp[kThreads >> (kRoundQubits - kRegBits)];  // round adjoints: grad_exponent per tile of the CTA
  uint32_t ticket;             // the CTA's finishing order (loss on the last CTA)
  uint32_t lg[256];
  float red[2][kThreads / 32][kMaxStepSlots];
  int32_t slot[2][kMaxStepSlots];
  double dred[kThreads / 32];
  uint32_t gmap[16];
  uint32_t gb[4];              // per register group: its lowest local bit
  uint4 gpos[4];               // its qubits
  uint32_t gqub[4];            // and the same in bytes (chain_pending)
};
using PassShared = PassSharedT<true>;

// One CTA's share of a pass: tiles first_tile .. first_tile + tiles_per_cta-1
// (tile = sample * tiles_per_sample + tile within the sample). Ends with a
// barrier, so a CTA may call it again for another pass or tile range.
// KC: the tile's qubits where they are known when compiled (12: one tile per
// CTA of 256 threads, every tile active), else 0. The constant lets the tile
// loads, the group bases and the reductions drop their index arithmetic: with
// the padded layout, 366 -> 291 instructions per warp and round forward and 786
// -> 659 adjoint; step of n = 20, d = 24, 64 samples 25.10 -> 23.00 ms, of n =
// 12, d = 20, 256 samples 237 -> 222 us.
// H: threads per column as a power of two (1: two threads of 8 registers each).
template <bool BWD, bool ROUNDS, bool TC = false, bool RX = false, int KC = 0, int H = 0, class Shared>
__device__ __forceinline__ void pass_cta(const PassArgs& a, const int64_t first_tile, float2* smem, Shared& sh,
                                         const TcCtx* tc = nullptr, float (*acc_rows)[8][32] = nullptr) {
  uint32_t (&s_lg)[256] = sh.lg;
  float (&s_red)[2][kThreads / 32][kMaxStepSlots] = sh.red;
  int32_t (&s_slot)[2][kMaxStepSlots] = sh.slot;
  double (&s_dred)[kThreads / 32] = sh.dred;
  uint32_t (&s_gmap)[16] = sh.gmap;

  const PassDesc& pd = a.pd;
  const int K = KC ? KC : pd.K;
  constexpr int NR = 16 >> H;                  // amplitudes per thread and step
  constexpr int NIT = NR / 2;                  // pairs per thread of the tile's loads and stores
  const int tl2 = K - kRegBits + H;        // log2 threads per tile
  const int Tt = 1 << tl2;
  const int tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  const int tile_in_cta = KC ? 0 : tid >> tl2;
  const uint32_t tau = KC ? (uint32_t)tid : (uint32_t)(tid & (Tt - 1));
  const int nthr = KC ? kThreads : (int)blockDim.x;
  const int tiles_per_cta = KC ? 1 : nthr >> tl2;
  const int64_t total_tiles = (int64_t)a.B << a.tps_log2;
  const int64_t tile = first_tile + tile_in_cta;
  const bool active = KC || tile < total_tiles;
  const int64_t b = active ? (tile >> a.tps_log2) : 0;
  const uint32_t t_in = active ? (uint32_t)(tile & ((1ll << a.tps_log2) - 1)) : 0u;
  const uint32_t outer = pdep32(t_in, pd.outer_mask);
  const int64_t dim = 1ll << a.n_eff;
  const int64_t sbase = b * dim;  // sample offset inside one state buffer
  float2* tp = smem + (tile_in_cta << K) + (tile_in_cta << (K - 4));  // loc(tile_in_cta << K)
  const int lam_at = KC ? kTilePad : (nthr >> H) * 17;  // words of the CTA's psi tiles: lambda's follow
  float2* tl = tp + lam_at;
  const int wpt = Tt >= 32 ? Tt / 32 : 1;  // warps per tile
  const int lanes = Tt < 32 ? Tt : 32;

  // (read here, used after the tile's loads)
  const bool seeds = BWD && (pd.lam_src == LAM_SEED || pd.lam_src == LAM_SEED_FAR);
  const double dl = active && (seeds || (BWD && ROUNDS)) ? seed_dl(a, b) : 0.0;
  // (round programs: one op per step, read a step ahead; the first one here)
  uint2 next = make_uint2(0u, 0u);
  if (ROUNDS && pd.op_begin < pd.op_end) next = __ldg(a.ops + pd.op_begin);
  if (tid < 16) {
    s_gmap[tid] = pd.gmap[tid];
    if (tid < 4) {
      sh.gb[tid] = pd.groups[tid][0];
      const uint4 q = make_uint4(pd.gmap[pd.groups[tid][0] & 15], pd.gmap[pd.groups[tid][1] & 15],
                                 pd.gmap[pd.groups[tid][2] & 15], pd.gmap[pd.groups[tid][3] & 15]);
      sh.gpos[tid] = q;
      sh.gqub[tid] = q.x | q.y << 8 | q.z << 16 | q.w << 24 |
                     (q.y == q.x + 1 && q.z == q.x + 2 && q.w == q.x + 3 ? kContig : 0u);
    }
  }
  __syncthreads();
  for (int i = tid; i < (1 << (K - kRegBits)); i += nthr) {
    uint32_t g = 0;
    for (int j = 0; j < K - kRegBits; ++j)
      if ((i >> j) & 1) g |= 1u << s_gmap[kRegBits + j];
    s_lg[i] = g;
  }
  __syncthreads();

  auto gidx = [&](uint32_t i) -> uint32_t { return outer | (i & 15u) | s_lg[i >> 4]; };
  // A thread's share of the tile is the pairs i = 2 (it Tt + tau), it < NIT: it
  // is the top local bits (K-3 .. K-1, or K-2 and K-1), so the global index
  // splits into the thread's part and `it_bits` (uniform), and for KC the place
  // in shared memory into the thread's part and it * loc(2 Tt)
  const uint32_t g_tau = gidx(2u * tau), p_tau = loc(2u * tau);
  auto it_bits = [&](int it) -> uint32_t {
    uint32_t g = 0u;
#pragma unroll
    for (int q = 0; q < 3 - H; ++q) g |= ((it >> q) & 1) ? 1u << pd.gmap[K - 3 + H + q] : 0u;
    return g;
  };
  auto g_it = [&](int it) -> uint32_t { return g_tau | it_bits(it); };
  auto p_it = [&](int it) -> uint32_t {
    return KC ? p_tau + (uint32_t)it * loc(2u * 256u) : loc(2u * ((uint32_t)it * Tt + tau));
  };
  auto state_ptr = [&](int32_t code) -> float2* {
    if (code >= 0) return a.slots + (int64_t)code * a.slot_stride + sbase;
    return a.work + sbase;
  };
  // (warp 0) the next round step at or after op q: its first round and count
  auto next_step = [&](int32_t q, uint32_t& rb, int& nr) -> bool {
    for (; q < pd.op_end; ++q) {
      const uint2 o = __ldg(a.ops + q);
      if ((o.x & 15u) == OP_STEP) {
        rb = o.y;
        nr = (int)((o.x >> 8) & 0xffffu);
        return true;
      }
    }
    return false;
  };
  // (tensor-core path, every thread) asynchronous copy of the B blocks of
  // rounds rb .. rb+nr-1 into staging buffer bb
  auto stage_b = [&](int bb, uint32_t rb, int nr) {
    const int n16 = nr * kTcBFloats / 4;
    const float* src = a.tcb + (size_t)rb * kTcBFloats;
    float* dst = tc->bsm + (size_t)bb * kMaxStepRounds * kTcBFloats;
    for (int e = tid; e < n16; e += kThreads) cp_async16(dst + 4 * e, src + 4 * e);
    cp_async_commit();
  };
  uint32_t ph = 0;  // tensor-core path: mbarrier phase of this thread's warpgroup
  // (warp 0) asynchronous copy of rounds rb .. rb+nr-1 into sh.par[pb]
  auto stage = [&](int pb, uint32_t rb, int nr) {
    constexpr int RW4 = (BWD ? kBwdRoundWords : kFwdRoundWords) / 4;
    const int nv = nr * kRoundPar, n_all = nv + nr * RW4;
    for (int e = lane; e < n_all; e += 32) {
      if (e < nv) cp_async16(&sh.par[pb].v[0][0] + e, a.rpar + (size_t)rb * kRoundPar + e);
      else cp_async16(&sh.par[pb].rec[e - nv], a.rounds + (size_t)rb * RW4 + (e - nv));
    }
    cp_async_commit();
  };

  // round programs: the first step's parameters, on their way while the tile
  // loads (after them, they were two more trips to L2 in a row: a ring of 13
  // qubits, 37 samples, adjoint 19.6 -> 18.8 us a pass and forward 10.5 -> 10.1; n
  // = 16, d = 100, 64 samples 4.88 -> 4.80 ms a step). The tile's loads go first:
  // waiting for the op word before them took n = 20 from 1.244 to 1.255 ms a pass.
  auto stage_first = [&]() {
    if (ROUNDS && warp == 0) {
      uint32_t rb;
      int nr;
      if (next_step(pd.op_begin, rb, nr)) stage(0, rb, nr);
    }
  };

  // ---- bring psi (and lambda) in -------------------------------------------
  const int32_t psrc = pd.psi_src;
  if (psrc == SRC_GENERATE || !active) stage_first();
  if (psrc == SRC_GENERATE && a.psi_in) {
    // given initial states [B][2^n_in]; padding qubits (n_in <= bit < n_eff) are |0>
    const int64_t din = 1ll << a.n_in;
    const float2* src = a.psi_in + b * din;
#pragma unroll
    for (int it = 0; it < NIT; ++it) {
      const uint32_t g = g_it(it);
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (a.n_in == a.n_eff) {
        v = __ldcg(reinterpret_cast<const float4*>(src + g));
      } else if ((int64_t)g < din) {
        const float2 u0 = src[g], u1 = (int64_t)g + 1 < din ? src[g + 1] : make_float2(0.f, 0.f);
        v = make_float4(u0.x, u0.y, u1.x, u1.y);
      }
      if (active) st_pair(tp, p_it(it), v);
    }
  } else if (psrc == SRC_GENERATE) {
    // psi_0 = (x) RY(x_q)|0>: a_x = prod_q (bit q of x ? sin(x_q/2) : cos(x_q/2));
    // the thread's pairs share every factor but those of qubit 0 and the
    // three local bits K-3 .. K-1
    const float2* e = a.enc + b * a.n_eff;
    const uint32_t vary = it_bits(NIT - 1);
    float pr = 1.f;
    for (int q = 1; q < a.n_eff; ++q) {
      if ((vary >> q) & 1u) continue;
      const float2 f = __ldg(e + q);
      pr *= ((g_tau >> q) & 1u) ? f.y : f.x;
    }
    const float2 f0 = __ldg(e);
    float2 ev[3];
#pragma unroll
    for (int q = 0; q < 3 - H; ++q) ev[q] = __ldg(e + pd.gmap[K - 3 + H + q]);
    if (active) {
#pragma unroll
      for (int it = 0; it < NIT; ++it) {
        float v = pr;
#pragma unroll
        for (int q = 0; q < 3 - H; ++q) v *= ((it >> q) & 1) ? ev[q].y : ev[q].x;
        st_pair(tp, p_it(it), make_float4(v * f0.x, 0.f, v * f0.y, 0.f));
      }
    }
  } else if (active) {
    // issue every load of the tile (psi, and lambda) before the first store
    const float2* src = state_ptr(psrc);
    const bool half = (pd.flags & PF_SRC_H) != 0;
    const __nv_bfloat162* hsrc =
        half ? reinterpret_cast<const __nv_bfloat162*>(a.hslots) + (int64_t)psrc * a.slot_stride + sbase : nullptr;
    // lambda: the buffer, or (LAM_SEED_FAR) the seed 2 (dL/dE_b) O psi_M taken
    // from psi at x ^ x_mask, which may lie in another tile. The pass does not
    // write the buffer that it reads psi from (the stored final state).
    // Seeding in a pass of its own cost a read and a write of lambda: 0.42 ms
    // of a 4.33 ms step (n = 20, 100 given states).
    const bool far = BWD && pd.lam_src == LAM_SEED_FAR;
    const bool two = BWD && (pd.lam_src == LAM_BUF || far);
    const float2* lsrc = far ? src : a.lam + sbase;
    const uint32_t lx = far ? a.x_mask & ~1u : 0u;
    float4 vp[NIT], vl[NIT];
#pragma unroll
    for (int it = 0; it < NIT; ++it) {
      const uint32_t g = g_it(it);
      if (half) vp[it] = bf16x4_to_f4(__ldcg(reinterpret_cast<const uint2*>(hsrc + g)));
      else vp[it] = __ldcg(reinterpret_cast<const float4*>(src + g));
      if (two) vl[it] = __ldcg(reinterpret_cast<const float4*>(lsrc + (g ^ lx)));
    }
    stage_first();
    if (far) {
      const float scale = (float)(2.0 * dl * (ROUNDS ? pow2(-grad_exponent(dl)) : 1.0));
#pragma unroll
      for (int it = 0; it < NIT; ++it) {
        const uint32_t xp = g_it(it) ^ a.x_mask;  // the pair's partners: xp and xp ^ 1
        const bool swap = (a.x_mask & 1u) != 0;
        const float4 v = vl[it];
        const float2 u0 = mul_ipow(swap ? make_float2(v.z, v.w) : make_float2(v.x, v.y), a.y_count);
        const float2 u1 = mul_ipow(swap ? make_float2(v.x, v.y) : make_float2(v.z, v.w), a.y_count);
        const uint32_t s0 = __popc(xp & a.z_mask) & 1u, s1 = __popc((xp ^ 1u) & a.z_mask) & 1u;
        vl[it] = make_float4(flip(u0.x, s0) * scale, flip(u0.y, s0) * scale, flip(u1.x, s1) * scale,
                             flip(u1.y, s1) * scale);
      }
    }
#pragma unroll
    for (int it = 0; it < NIT; ++it) {
      st_pair(tp, p_it(it), vp[it]);
      if (two) st_pair(tl, p_it(it), vl[it]);
    }
  }
  if (BWD && pd.lam_src == LAM_BUF && psrc == SRC_GENERATE && active) {
    const float2* src = a.lam + sbase;
#pragma unroll
    for (int it = 0; it < NIT; ++it) st_pair(tl, p_it(it), __ldcg(reinterpret_cast<const float4*>(src + g_it(it))));
  }
  if (BWD && ROUNDS && tau == 0) sh.gexp[tile_in_cta] = grad_exponent(dl);
  int sb = 0;  // round programs: the step's staging buffer
  if (ROUNDS && warp == 0) cp_async_wait_all();
  if (TC) {
    uint32_t rb;
    int nr;
    if (next_step(pd.op_begin, rb, nr)) stage_b(0, rb, nr);
    cp_async_wait_all();
    fence_proxy_async();  // B is read by the tensor cores (async proxy)
  }
  __syncthreads();
  if (BWD && pd.lam_src == LAM_SEED) {
    // lambda_M = 2 (dL/dE_b) O psi_M (Eq. 4); (O psi)_x = i^{#Y} (-1)^{|(x^xm)&zm|} psi_{x^xm}
    const float scale = (float)(2.0 * dl * (ROUNDS ? pow2(-grad_exponent(dl)) : 1.0));
#pragma unroll 1
    for (int it = 0; it < NR; ++it) {
      const uint32_t i = (uint32_t)it * Tt + tau;  // single amplitudes here
      const uint32_t ip = i ^ pd.xm_local;
      const uint32_t gp = gidx(ip);
      float2 v = tp[loc(ip)];
      v = mul_ipow(v, a.y_count);
      const uint32_t sg = __popc(gp & a.z_mask) & 1u;
      tl[loc(i)] = make_float2(flip(v.x, sg) * scale, flip(v.y, sg) * scale);
    }
    __syncthreads();
  }

  // ---- step program ------------------------------------------------------------
  int buf = 0;
  uint32_t pend = 0;  // links whose CZ signs the tile's amplitudes still lack (round programs)
  int32_t pc = pd.op_begin;
  const uint2* ops = a.ops;
#pragma unroll 1
  while (pc < pd.op_end) {
    const uint2 op = ROUNDS ? next : __ldg(ops + pc);
    ++pc;
    if (ROUNDS && pc < pd.op_end) next = __ldg(ops + pc);
    const uint32_t code = op.x & 15u;
    if (ROUNDS && code == OP_STEP) {
      // ---- round step: straight-line rounds over the 4 register bits
      const int g = (op.x >> 4) & 3;
      const int nr = (op.x >> 8) & 0xffff;
      if (warp == 0) {
        // prefetch the next step's parameters while this one runs
        uint32_t rb;
        int nr2;
        if (next_step(pc, rb, nr2)) stage(sb ^ 1, rb, nr2);
      }
      if (TC) {
        uint32_t rb;
        int nr2;
        if (next_step(pc, rb, nr2)) stage_b(sb ^ 1, rb, nr2);
      }
      const StepPar& P = sh.par[sb];
      const uint32_t lb = KC ? 4u * (uint32_t)g : sh.gb[g];
      // the column's bits around the group's (a zero in each of its four); h: the
      // thread's half of the column
      const uint32_t col = tau >> H, h = H ? tau & 1u : 0u;
      const uint32_t base = (col & ((1u << lb) - 1u)) | ((col >> lb) << (lb + 4u));
      float2* const at = tp + loc(base) + (H && h ? loc(8u << lb) : 0u);
      const uint32_t gb = gidx(base);
      const uint32_t qubits = sh.gqub[g];
      float2 r[NR];
      float2 l[NR];
      ld_group<KC, BWD>(lb, at, at + lam_at, r, l);
      const int nq = a.n_eff;
      const uint32_t nmask = nq >= 32 ? ~0u : ((1u << nq) - 1u);
      const uint32_t rgb = ((gb >> 1) | ((gb & 1u) << (nq - 1))) & nmask;
      const uint32_t lgb = ((gb << 1) | (gb >> (nq - 1))) & nmask;
      const uint32_t g12 = gb & rgb;
      uint32_t D = 0;
      if (!TC) chain_pending(pend, rgb, lgb, g12, nq, qubits, D);
      if constexpr (TC) {
        const uint4 gp = sh.gpos[g];
        const uint32_t pos[4] = {gp.x, gp.y, gp.z, gp.w};
        tc_rounds(*tc, P, nr, tc->bsm + (size_t)sb * kMaxStepRounds * kTcBFloats, gb, pos, a.n_eff, r, ph, tid);
      } else {
      // a round of steep rotations runs them twice (see rot_T)
#pragma unroll 1
      for (int k = 0; k < nr; ++k) {
        const bool steep = P.v[k][0].y < 0.f;
        if (!BWD) {
          const uint4 lk = P.rec[k * (kFwdRoundWords / 4) + 1];  // links, bbits, rx mask, leaving links
          if (steep) {
            rots<RX>(r, P.v[k], D, lk.z);
            if constexpr (H) rot_fwd_half<RX>(r, pend_q(P.v[k][3].x, (D >> 3) & 1u), h, (lk.z >> 3) & 1u);
          }
          rots<RX>(r, P.v[k], D, lk.z);
          if constexpr (H) rot_fwd_half<RX>(r, pend_q(P.v[k][3].x, (D >> 3) & 1u), h, (lk.z >> 3) & 1u);
          apply_diag(r, &P.v[k][4 + (H ? 4 * h : 0)]);
          chain_pending(lk.x, rgb, lgb, g12, nq, qubits, D);
          pend ^= lk.w;
        } else {
          const uint4 lk = P.rec[k * (kBwdRoundWords / 4) + 2];  // links, bbits, rx mask, leaving links
          chain_pending(lk.x, rgb, lgb, g12, nq, qubits, D);
          pend ^= lk.w;
          float v[8];
          if constexpr (H) diag_bwd(r, l, &P.v[k][4 + 4 * h], v, h);
          else diag_bwd(r, l, &P.v[k][4], v);
          if constexpr (RX && !H) {
            item_bwd<0>(r, l, P.v[k][0].x, D & 1u, v[4], lk.z & 1u);
            item_bwd<1>(r, l, P.v[k][1].x, (D >> 1) & 1u, v[5], (lk.z >> 1) & 1u);
            item_bwd<2>(r, l, P.v[k][2].x, (D >> 2) & 1u, v[6], (lk.z >> 2) & 1u);
            item_bwd<3>(r, l, P.v[k][3].x, (D >> 3) & 1u, v[7], (lk.z >> 3) & 1u);
            if (steep) {  // (here it spills 24 bytes, after the reduction 48)
              rots<RX>(r, P.v[k], D, lk.z);
              rots<RX>(l, P.v[k], D, lk.z);
            }
          } else {
            v[4] = grad_T<0, RX>(r, l, D & 1u, lk.z & 1u);
            v[5] = grad_T<1, RX>(r, l, (D >> 1) & 1u, (lk.z >> 1) & 1u);
            v[6] = grad_T<2, RX>(r, l, (D >> 2) & 1u, (lk.z >> 2) & 1u);
            if constexpr (H) rot_bwd_half<RX>(r, l, P.v[k][3].x, (D >> 3) & 1u, v[7], h, (lk.z >> 3) & 1u);
            else v[7] = grad_T<3, RX>(r, l, (D >> 3) & 1u, (lk.z >> 3) & 1u);
            rots<RX>(r, P.v[k], D, lk.z);
            rots<RX>(l, P.v[k], D, lk.z);
          }
          int idx;
          float sum;
          bool owner;
          if constexpr (RX && !H) {
            // shuffles here: with the rows, whose registers this instance lacks and
            // whose 8 KiB L1 then lacks, 100 states of 20 qubits took 1.27 ms a launch,
            // this 1.25
            sum = lanes == 32 ? butterfly8(v, 32, lane, idx) : butterfly8(v, lanes, lane, idx);
            owner = (lane & ((lanes >> 3) - 1)) == 0;
          } else {
            // lane holds value idx of its tile; the first 8 lanes of a tile keep theirs
            idx = lane & 7;
            sum = rows8(v, lanes, lane, sh.rows[warp]);
            owner = (lane & (lanes - 1)) < 8;
          }
          if (owner) {
            const int32_t term =
                reinterpret_cast<const int32_t*>(&P.rec[k * (kBwdRoundWords / 4)])[idx];
            if (idx >= 4) sum *= RX && !H ? P.v[k][idx - 4].z : fabsf(P.v[k][0].y);
            if (Tt >= 32) {
              s_red[buf][warp][k * 8 + idx] = sum;
              if (warp == 0) s_slot[buf][k * 8 + idx] = term;
            } else if (active && term >= 0) {
              a.g_part[tile * a.n_slots + term] = partial<KC == 0>(sum, sh.gexp[tile_in_cta]);
            }
          }
          if ((H || !RX) && steep) {
            if constexpr (H) {
              const float q3 = pend_q(P.v[k][3].x, (D >> 3) & 1u);
              rot_fwd_half<RX>(r, q3, h, (lk.z >> 3) & 1u);
              rot_fwd_half<RX>(l, q3, h, (lk.z >> 3) & 1u);
            }
            rots<RX>(r, P.v[k], D, lk.z);
            rots<RX>(l, P.v[k], D, lk.z);
          }
        }
      }
      if ((op.x >> kStepFlushBit) & 1u) {
        if (H) D = (D ^ ((D & (h << 3)) << 1)) & ~8u;  // the half's own bit 3
        apply_pending<BWD>(D, r, l);
        pend = 0;
      }
      }  // CUDA-core rounds
      st_group<KC, BWD>(lb, at, at + lam_at, r, l);
      if (TC) {
        cp_async_wait_all();
        fence_proxy_async();
      } else if (warp == 0) {
        cp_async_wait_all();
      }
      __syncthreads();
      sb ^= 1;
      if (BWD && Tt >= 32 && a.g_accum) {
        // every tile of this call belongs to one sample: one thread per term sums
        // the tiles in order and adds to row g_row (stored by the row's first
        // call); within a tile the warp sums add in float32, as the warp shuffles
        // do, then float64 across tiles
        const int nk = nr * 8;
        const bool first = a.g_first != 0;
        const double half = pow2(sh.gexp[0] - 1);
        for (int kk = nthr - 1 - tid; kk < nk; kk += nthr) {  // the last warp (warp 0 stages)
          const int32_t term = s_slot[buf][kk];
          if (term < 0) continue;
          double sum = 0.0;
          for (int tc = 0; tc < tiles_per_cta; ++tc)
            if (first_tile + tc < total_tiles) {
              float sf = 0.f;
              for (int w = 0; w < wpt; ++w) sf += s_red[buf][tc * wpt + w][kk];
              sum += (double)sf;
            }
          double* dst = a.g_part + a.g_row * a.n_slots + term;
          *dst = first ? half * sum : *dst + half * sum;
        }
        buf ^= 1;
      } else if (BWD && Tt >= 32) {
        // the tile's warp sums in float32 (one float64 value per tile and term)
        const int nk = nr * 8;
        for (int e = nthr - 1 - tid; e < tiles_per_cta * nk; e += nthr) {  // from the last warp
          const int tc = e / nk, kk = e - tc * nk;
          const int64_t t2 = first_tile + tc;
          const int32_t term = s_slot[buf][kk];
          if (t2 < total_tiles && term >= 0) {
            float sf = 0.f;
            for (int w = 0; w < wpt; ++w) sf += s_red[buf][tc * wpt + w][kk];
            a.g_part[t2 * a.n_slots + term] = partial<KC == 0>(sf, sh.gexp[KC ? 0 : tc]);
          }
        }
        buf ^= 1;
      }
    } else if (!ROUNDS && code == OP_STEP) {
      const int g = (op.x >> 4) & 3;
      const int nops = (op.x >> 8) & 0xffff;
      const int nk = (int)op.y;
      const uint32_t lb = sh.gb[g];
      const uint32_t base = (tau & ((1u << lb) - 1u)) | ((tau >> lb) << (lb + 4u));
      float2* const at = tp + loc(base);
      const uint32_t so[4] = {loc(1u << lb), loc(2u << lb), loc(4u << lb), loc(8u << lb)};
      const uint32_t gb = gidx(base);
      const uint4 gp = sh.gpos[g];
      const uint32_t go[4] = {1u << gp.x, 1u << gp.y, 1u << gp.z, 1u << gp.w};
      float2 r[16];
      float2 l[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        r[j] = at[reg_off(j, so)];
        if (BWD) l[j] = at[lam_at + reg_off(j, so)];
      }
      // ops are read two ahead and their coefficients one ahead: a step's ops
      // run one after another, and each was two dependent loads
      auto coef = [&](uint2 o, float4& m0, float4& m1) {
        if (!BWD && (o.x & 15u) == OP_U) {
          m0 = __ldg(a.mats + 2 * (o.x >> 8));
          m1 = __ldg(a.mats + 2 * (o.x >> 8) + 1);
        } else if (BWD && (o.x & 15u) == OP_G) {
          const float2 v = __ldg(a.cs + o.y);
          m0 = make_float4(v.x, v.y, 0.f, 0.f);
        }
      };
      uint2 o1 = make_uint2(0u, 0u), o2 = o1;
      float4 m0 = make_float4(0.f, 0.f, 0.f, 0.f), m1 = m0;
      if (nops > 0) o1 = __ldg(ops + pc);
      if (nops > 1) o2 = __ldg(ops + pc + 1);
      if (nops > 0) coef(o1, m0, m1);
      pc += nops;
#pragma unroll 1
      for (int k = 0; k < nops; ++k) {
        const uint2 o = o1;
        const float4 c0 = m0, c1 = m1;
        o1 = o2;
        if (k + 1 < nops) coef(o1, m0, m1);
        if (k + 2 < nops) o2 = __ldg(ops + pc - nops + k + 2);
        const uint32_t oc = o.x & 15u;
        if (!BWD && oc == OP_U) {
          switch ((o.x >> 4) & 3u) {
            case 0: apply_u<0>(r, c0, c1); break;
            case 1: apply_u<1>(r, c0, c1); break;
            case 2: apply_u<2>(r, c0, c1); break;
            default: apply_u<3>(r, c0, c1); break;
          }
        } else if (BWD && oc == OP_G) {
          const uint32_t rr = (o.x >> 4) & 3u, kind = (o.x >> 6) & 3u, ks = (o.x >> 8) & 0xffu;
          float acc;
          if (kind == G_RZ) acc = bwd_dispatch_r<G_RZ>(rr, r, l, c0.x, c0.y);
          else if (kind == G_RY) acc = bwd_dispatch_r<G_RY>(rr, r, l, c0.x, c0.y);
          else acc = bwd_dispatch_r<G_RX>(rr, r, l, c0.x, c0.y);
          if (lanes >= 8) {
            // eight terms are reduced over the tile's lanes at once (a warp's own
            // rows: no barrier; the term ids are the same in every warp): five
            // shuffles in a chain after each rotation, and the loads of its op,
            // took as long as the arithmetic (n = 10 with CNOTs, d = 6, 100
            // samples: step 163 -> 138 us)
            float (&s_acc)[8][32] = acc_rows[warp];
            s_acc[ks & 7u][lane] = acc;
            if (lane == 0) s_slot[buf][ks] = (int32_t)o.y;
            if ((ks & 7u) == 7u || (int)ks == nk - 1) {
              __syncwarp();
              float v[8];
#pragma unroll
              for (int i = 0; i < 8; ++i) v[i] = (uint32_t)i <= (ks & 7u) ? s_acc[i][lane] : 0.f;
              int idx;
              const float sum = butterfly8(v, lanes, lane, idx);
              const uint32_t kk = (ks & ~7u) + (uint32_t)idx;
              if ((lane & ((lanes >> 3) - 1)) == 0 && kk <= ks) {
                if (Tt >= 32) s_red[buf][warp][kk] = sum;
                else if (active) a.g_part[tile * a.n_slots + s_slot[buf][kk]] = (double)(0.5f * sum);
              }
              __syncwarp();
            }
          } else {
            for (int off = 1; off < lanes; off <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
            if (active && (lane & (Tt - 1)) == 0) a.g_part[tile * a.n_slots + o.y] = (double)(0.5f * acc);
          }
        } else if (oc == OP_CNOT) {
          const bool creg = ((o.y >> 8) & 1u) != 0;
          const uint32_t cb = o.y & 0xffu;
          switch ((o.x >> 4) & 3u) {
            case 0: cnot_regs<0, BWD>(r, l, creg, cb, gb); break;
            case 1: cnot_regs<1, BWD>(r, l, creg, cb, gb); break;
            case 2: cnot_regs<2, BWD>(r, l, creg, cb, gb); break;
            default: cnot_regs<3, BWD>(r, l, creg, cb, gb); break;
          }
        } else if (oc == OP_CHAIN || oc == OP_CZ) {
          const uint32_t links = o.y, c0 = o.y & 0xffu, c1 = (o.y >> 8) & 0xffu;
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const uint32_t x = gb | reg_off(j, go);
            const uint32_t sg = oc == OP_CHAIN ? (__popc(x & (x >> 1) & links) & 1u)
                                               : ((x >> c0) & (x >> c1) & 1u);
            r[j].x = flip(r[j].x, sg);
            r[j].y = flip(r[j].y, sg);
            if (BWD) {
              l[j].x = flip(l[j].x, sg);
              l[j].y = flip(l[j].y, sg);
            }
          }
        }
      }
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        at[reg_off(j, so)] = r[j];
        if (BWD) at[lam_at + reg_off(j, so)] = l[j];
      }
      __syncthreads();
      if (BWD && Tt >= 32) {
        for (int e = nthr - 1 - tid; e < tiles_per_cta * nk; e += nthr) {  // from the last warp
          const int tc = e / nk, kk = e - tc * nk;
          const int64_t t2 = first_tile + tc;
          if (t2 < total_tiles) {
            float sf = 0.f;
            for (int w = 0; w < wpt; ++w) sf += s_red[buf][tc * wpt + w][kk];
            a.g_part[t2 * a.n_slots + s_slot[buf][kk]] = (double)(0.5f * sf);
          }
        }
        buf ^= 1;
      }
    } else if (code == OP_CKPT || code == OP_ANCHOR) {
      float2* sp = a.slots + (int64_t)op.y * a.slot_stride + sbase;
#pragma unroll
      for (int it = 0; it < NIT; ++it) {
        if (!active) continue;
        if (code == OP_CKPT) *reinterpret_cast<float4*>(sp + g_it(it)) = ld_pair(tp, p_it(it));
        else st_pair(tp, p_it(it), __ldcg(reinterpret_cast<const float4*>(sp + g_it(it))));
      }
      __syncthreads();
    }
  }

  // ---- write back -----------------------------------------------------------
  if (pd.psi_dst != BUF_NONE && (pd.flags & PF_DST_H)) {
    // memory-saving mode (Sec. 3.2): the stored copy is rounded to bfloat16
    __nv_bfloat162* dst = reinterpret_cast<__nv_bfloat162*>(a.hslots) + (int64_t)pd.psi_dst * a.slot_stride + sbase;
#pragma unroll
    for (int it = 0; it < NIT; ++it) {
      if (active) *reinterpret_cast<uint2*>(dst + g_it(it)) = f4_to_bf16x4(ld_pair(tp, p_it(it)));
    }
  } else if (pd.psi_dst != BUF_NONE) {
    float2* dst = state_ptr(pd.psi_dst);
#pragma unroll
    for (int it = 0; it < NIT; ++it) {
      if (active) *reinterpret_cast<float4*>(dst + g_it(it)) = ld_pair(tp, p_it(it));
    }
  }
  if (BWD && pd.lam_dst == LAM_BUF) {
    float2* dst = a.lam + sbase;
#pragma unroll
    for (int it = 0; it < NIT; ++it) {
      if (active) *reinterpret_cast<float4*>(dst + g_it(it)) = ld_pair(tl, p_it(it));
    }
  }
  if (!BWD && (pd.flags & PF_EXPECT)) {
    // <psi|O|psi> partial of this tile (Eq. 1, matrix-free as in Appendix B.2)
    float acc = 0.f;
#pragma unroll 1
    for (int it = 0; it < NR; ++it) {
      const uint32_t i = (uint32_t)it * Tt + tau;
      const uint32_t ip = i ^ pd.xm_local;
      const float2 v = tp[loc(i)];
      float2 w = mul_ipow(tp[loc(ip)], a.y_count);
      const uint32_t sg = __popc(gidx(ip) & a.z_mask) & 1u;
      acc += flip(v.x * w.x + v.y * w.y, sg);  // Re(conj(v) w) with the Z signs
    }
    double d = (double)acc;
    for (int off = 1; off < lanes; off <<= 1) d += __shfl_xor_sync(0xffffffffu, d, off);
    if (Tt >= 32) {
      if (lane == 0) s_dred[warp] = d;
      __syncthreads();
      if (tid < tiles_per_cta) {
        const int64_t t2 = first_tile + tid;
        if (t2 < total_tiles) {
          double sum = 0.0;
          for (int w = 0; w < wpt; ++w) sum += s_dred[tid * wpt + w];
          a.e_part[t2] = sum;
        }
      }
    } else if (active && (lane & (Tt - 1)) == 0) {
      a.e_part[tile] = d;
    }
  }
  __syncthreads();
  if (!BWD && a.done && (pd.flags & PF_EXPECT)) {
    // the last CTA to finish sums E over every CTA's partials and finishes
    // the loss (the partials are fenced before the count)
    __threadfence();
    __syncthreads();
    if (tid == 0) sh.ticket = atomicAdd(a.done, 1u);
    __syncthreads();
    if (sh.ticket == gridDim.x - 1) {
      __threadfence();
      loss_block<float>(a.loss_kind, a.E, a.y, a.B, a.loss_scale, a.loss, a.dLdE_out, a.e_part, 1 << a.tps_log2,
                        tid, nthr);
    }
    __syncthreads();
  }
}

// RX: round programs holding RX items (their own instance, so that programs
// of RZ / RY items keep the plain code). MINB: CTAs per SM the registers are
// budgeted for; a forward pass (one 32 KiB state per CTA) of more tiles than
// two CTAs per SM hold runs with three per SM.
template <bool BWD, bool ROUNDS, bool RX = false, int MINB = 2, int KC = 0, int H = 0>
__global__ void __launch_bounds__(kThreads, MINB) pass_kernel(const PassArgs a) {
  extern __shared__ __align__(16) float2 smem[];
  // (the forward leaves the rows' 8 KiB to L1: n = 16, d = 20, 500 samples 2.16 -> 2.13 ms)
  __shared__ PassSharedT<BWD && ROUNDS && (H || !RX)> sh;
  const int64_t first = KC ? (int64_t)blockIdx.x : (int64_t)blockIdx.x * (blockDim.x >> (a.pd.K - kRegBits + H));
  if constexpr (BWD && !ROUNDS) {
    __shared__ float acc_rows[kThreads / 32][8][32];  // a generic step's terms waiting for their reduction
    pass_cta<BWD, ROUNDS, false, RX, KC, H>(a, first, smem, sh, nullptr, acc_rows);
  } else {
    pass_cta<BWD, ROUNDS, false, RX, KC, H>(a, first, smem, sh);
  }
}

// Forward pass with the rounds on the tensor cores: one 12-qubit tile per
// CTA (two warpgroups of 128 columns). Dynamic shared memory: the tile, then
// two B staging buffers of kMaxStepRounds rounds.
__global__ void __launch_bounds__(kThreads, 2) tc_pass_kernel(const PassArgs a) {
  extern __shared__ __align__(16) float2 smem[];
  __shared__ PassSharedT<false> sh;
  __shared__ __align__(8) uint64_t mbar[2];
  __shared__ uint32_t tmem_slot;
  const int warp = threadIdx.x >> 5;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(kTcCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 0) {
    for (int w = 0; w < 2; ++w)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar[w])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  TcCtx ctx{tmem_slot, mbar, reinterpret_cast<float*>(smem + kTilePad)};
  pass_cta<false, true, true, false, 12>(a, (int64_t)blockIdx.x, smem, sh, &ctx);
  // pass_cta ends with a barrier; every tensor-memory access is complete
  tc_fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_slot), "r"(kTcCols) : "memory");
}

// B blocks: element (n, k) of round r, n = output (re i | im i), k = input
// (re j | im j): U = u3 (x) u2 (x) u1 (x) u0 of the round's fused 2x2s,
// U[i][j] = prod_b u_b[i_b][j_b]; B[re i][re j] = Re U, B[re i][im j] = -Im U,
// B[im i][re j] = Im U, B[im i][im j] = Re U. Stored K-major (8-row x 16-byte
// core matrices, 128 B apart along K, 1024 B between row groups), TF32 hi at
// [0, 1024) and lo at [1024, 2048) of the round's block.
__global__ void tc_table_kernel(const uint4* fwd_rounds, int32_t n_rounds, const double* mats64, float* tcb) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)n_rounds * 1024) return;
  const int64_t r = e >> 10;
  const int n = (int)((e >> 5) & 31), k = (int)(e & 31);
  const int i = n & 15, j = k & 15;
  const uint4 m = fwd_rounds[r * (kFwdRoundWords / 4)];
  const uint32_t mm[4] = {m.x, m.y, m.z, m.w};
  double re = 1.0, im = 0.0;
  for (int b = 0; b < 4; ++b) {
    const double* u = mats64 + 8 * (size_t)mm[b];
    const int ib = (i >> b) & 1, jb = (j >> b) & 1;
    const double ur = u[(ib * 2 + jb) * 2], ui = u[(ib * 2 + jb) * 2 + 1];
    const double t = re * ur - im * ui;
    im = re * ui + im * ur;
    re = t;
  }
  const bool ro = n < 16, ri = k < 16;
  const double v = ro ? (ri ? re : -im) : (ri ? im : re);
  const float vf = (float)v;
  const uint32_t hi = cvt_tf32(vf);
  const uint32_t lo = cvt_tf32((float)(v - (double)__uint_as_float(hi)));
  const int off = (n >> 3) * 256 + (k >> 2) * 32 + (n & 7) * 4 + (k & 3);
  tcb[r * kTcBFloats + off] = __uint_as_float(hi);
  tcb[r * kTcBFloats + 1024 + off] = __uint_as_float(lo);
}

// ---------------------------------------------------------------------------
// Gate tables from theta in float64, rounded once to float32 (or kept in
// float64 for complex128 plans): generic programs' fused 2x2 products
// (forward) and (cos, sin) of theta/2 per term (backward); round programs'
// per-round rotations and diagonal phases (both directions); (cos, sin)
// of x/2 per sample and qubit (encoding). Element 0 also clears the forward
// pass's CTA counter when a train step finishes its loss in that pass.
__device__ void prep_one(const PrepArgs& a, int64_t i);

__global__ void prep_kernel(const PrepArgs a) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0 && a.zero_word) *a.zero_word = 0u;
  prep_one(a, i);
}

namespace {

// One out-of-line float64 sincos shared by every table of prep, so that the
// kernel's element kinds run one copy of its code (prep runs after an L2
// flush in timed steps, and each inlined copy is fetched separately).
__device__ __noinline__ void sincos_prep(double x, double* s, double* c) { sincos(x, s, c); }

// Parameter p as float64 (float32 parameters are promoted exactly).
__device__ __forceinline__ double theta_at(const PrepArgs& a, int p) {
  return a.theta64 ? a.theta64[p] : (double)a.theta[p];
}

// Fused 2x2 product of fused entry m (float64, rounded once to float32) by 4
// lanes (l: lane in the group): each takes the sincos of every fourth gate, and
// lanes 0 and 1 (2 and 3 repeat them) carry one column each through the gates.
// One thread per entry took its gates' float64 sincos and full 2x2 products one
// after another: prep of n = 4, d = 2, 8 samples 14.7 -> 5.5 us.
__device__ void fused_u(const PrepArgs& a, int64_t m, int l) {
  const int lane = threadIdx.x & 31, first = lane & ~3;
  const uint32_t group = 0xfu << first;
  const int j0 = a.fuse_off[m], j1 = a.fuse_off[m + 1], col = l & 1;
  double x0 = col == 0 ? 1.0 : 0.0, y0 = 0.0, x1 = col == 0 ? 0.0 : 1.0, y1 = 0.0;  // rows 0 and 1 of the column
  for (int j = j0; j < j1; j += 4) {
    double c = 1.0, s = 0.0;
    int kind = G_RZ;
    if (j + l < j1) {
      const FuseGate fg = a.fuse_gates[j + l];
      kind = fg.kind;
      sincos_prep(0.5 * (fg.param >= 0 ? theta_at(a, fg.param) : fg.angle), &s, &c);
    }
    const int n = min(4, j1 - j);
    for (int t = 0; t < n; ++t) {
      const double ct = __shfl_sync(group, c, first + t), st = __shfl_sync(group, s, first + t);
      const int kt = __shfl_sync(group, kind, first + t);
      const double a0 = x0, b0 = y0, a1 = x1, b1 = y1;
      // c I - i s P
      if (kt == G_RZ) {
        x0 = ct * a0 + st * b0;
        y0 = ct * b0 - st * a0;
        x1 = ct * a1 - st * b1;
        y1 = ct * b1 + st * a1;
      } else if (kt == G_RY) {
        x0 = ct * a0 - st * a1;
        y0 = ct * b0 - st * b1;
        x1 = ct * a1 + st * a0;
        y1 = ct * b1 + st * b0;
      } else {
        x0 = ct * a0 + st * b1;
        y0 = ct * b0 - st * a1;
        x1 = ct * a1 + st * b0;
        y1 = ct * b1 - st * a0;
      }
    }
  }
  if (l > 1) return;
  if (a.mats) {
    float2* u = reinterpret_cast<float2*>(a.mats + 2 * m) + col;  // u00, u01, u10, u11
    u[0] = make_float2((float)x0, (float)y0);
    u[2] = make_float2((float)x1, (float)y1);
  }
  if (a.mats64) {
    double2* u = reinterpret_cast<double2*>(a.mats64 + 8 * m) + col;
    u[0] = make_double2(x0, y0);
    u[2] = make_double2(x1, y1);
  }
}

// A term's angle is the sum of its parameters (a merged run of RZ gates).
__device__ double term_angle(const PrepArgs& a, int64_t t) {
  double phi = a.term_const ? a.term_const[t] : 0.0;
  for (int j = a.term_off[t]; j < a.term_off[t + 1]; ++j) phi += theta_at(a, a.term_params[j]);
  return phi;
}

// The angle of a resolved round term (the same summation order as
// term_angle: the constant, then the parameters).
__device__ __forceinline__ double round_term_angle(const PrepArgs& a, const RoundTerm& e) {
  if (e.p0 <= -2) return term_angle(a, -2 - e.p0);
  double phi = e.c;
  if (e.p0 >= 0) phi += theta_at(a, e.p0);
  if (e.p1 >= 0) phi += theta_at(a, e.p1);
  return phi;
}

// The multiple of 2 pi nearest to phi.
__device__ __forceinline__ double wrap_count(double phi) {
  return rint(phi * (1.0 / 6.283185307179586476925286766559));
}

// The diagonal of a round: its RZ runs (angles phi_r; 0 for a missing term)
// act on register index j as e^{-i a_j} with a_j = sum_r sigma_r(j) phi_r / 2,
// sigma_r(j) = +1 where bit r of j is clear, else -1 (RZ(phi) =
// diag(e^{-i phi/2}, e^{i phi/2})), and its CZ links between register bits r
// and r + 1 (bit r of bbits) as -1 where both bits of j are set. Gives the
// angle of the applied phase (forward: -a_j) or of the un-applied one
// (backward: +a_j) for j = m, and the CZ signs of m and its complement
// 15 - m: a_{15-m} = -a_m, so one float64 sincos of the summed angle serves both.
__device__ double diag_angle(const double (&phi)[4], uint32_t bbits, int m, bool apply, bool& f0, bool& f1) {
  double al = 0.0;
  for (int r = 0; r < 4; ++r) al += ((m >> r) & 1) ? -phi[r] : phi[r];
  const int mc = 15 - m;
  f0 = __popc(bbits & (uint32_t)m & (uint32_t)(m >> 1)) & 1;
  f1 = __popc(bbits & (uint32_t)mc & (uint32_t)(mc >> 1)) & 1;
  return al * (apply ? -0.5 : 0.5);
}

// One round's parameters by a half-warp (e: lane in it), float32 or (complex128
// plans) float64: lanes 0..3 take the 4 rotations, lanes 4..11 two phases of
// the diagonal each, one sincos per lane (see rot_T). Float64 has the exponents
// for any four tangents (at most 2^54 each), so only complex64 rounds run twice.
__device__ void round_params(const PrepArgs& a, bool on, bool fwd, int64_t r, const int32_t* rec,
                             const RoundTerm* rt, int e, int lane) {
  double ang = 0.0;
  bool odd = false, f0 = false, f1 = false;
  if (e < 4) {
    // u(phi) = (-1)^k u(w) with w = phi - 2 pi k in [-pi, pi]
    const double phi = round_term_angle(a, rt[e]), k = wrap_count(phi);
    ang = 0.5 * (phi - 6.283185307179586476925286766559 * k);
    odd = ((long long)k) & 1;
  } else if (e < 12) {
    double phi[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) phi[q] = round_term_angle(a, rt[4 + q]);
    ang = diag_angle(phi, (uint32_t)(fwd ? rec[5] : rec[9]), e - 4, fwd, f0, f1);
  }
  double c, s;
  sincos_prep(ang, &s, &c);
  const int half = lane & 16;
  const bool f64 = a.rpf64 || a.rpb64;
  // the rotations shrink the norm by the product of their cosines
  float shrink = e < 4 ? (float)(c * c) : 1.f;
  shrink *= __shfl_xor_sync(0xffffffffu, shrink, 1);
  shrink *= __shfl_xor_sync(0xffffffffu, shrink, 2);
  const bool steep = !f64 && e < 4 && shrink < kMinShrink;
  const bool twice = ((__ballot_sync(0xffffffffu, steep) >> half) & 15u) != 0;
  const uint32_t neg = __popc((__ballot_sync(0xffffffffu, odd) >> half) & 15u) & 1u;
  double q = e < 4 ? s / (twice ? 1.0 + c : c) : 0.0;  // tan(w/4) = sin(w/2) / (1 + cos(w/2))
  if (!f64) q = (double)(float)q;
  double Q[4], S = 1.0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double qk = __shfl_sync(0xffffffffu, q, half + k);
    Q[k] = 1.0 + qk * qk;
    S *= Q[k];
  }
  if (!on) return;
  float4* out = (fwd ? a.rpf : a.rpb) + r * kRoundPar;
  RoundPar64* out64 = (fwd ? a.rpf64 : a.rpb64) + r;
  if (e < 4) {
    // the factors of the rotations' gradient values: 1 / scale^2 (S: the product
    // of the Q), and, for kernels that take each after the rotations before it,
    // less those (complex128's only one)
    double g = Q[3], all = S;
#pragma unroll
    for (int k = 2; k >= 0; --k)
      if (k >= e) g *= Q[k];
    if (twice) {
      g *= S;
      all *= S;
    }
    if (!fwd) q = -q;
    if (f64) {
      out64->q[e] = q;
      out64->g[e] = g;
    } else {
      out[e] = make_float4((float)q, (float)(twice ? -all : all), (float)g, 0.f);
    }
  } else if (e < 12) {
    const double sc = (neg ? -1.0 : 1.0) * (twice ? 1.0 / S : rsqrt(S));
    const double x = c * sc, y = s * sc;
    const double2 v0 = f0 ? make_double2(-x, -y) : make_double2(x, y);
    const double2 v1 = f1 ? make_double2(-x, y) : make_double2(x, -y);
    if (f64) {
      out64->ph[e - 4] = v0;
      out64->ph[19 - e] = v1;
    } else {
      float2* ph = reinterpret_cast<float2*>(out + 4);
      ph[e - 4] = make_float2((float)v0.x, (float)v0.y);
      ph[19 - e] = make_float2((float)v1.x, (float)v1.y);
    }
  }
}

}  // namespace

// Element i of the tables: (round programs) the forward and backward round
// parameters in round order, then fused matrices, terms and encodings. A
// round's parameters are made by 16 lanes together and a fused matrix by 4;
// round_par_elems and fused_elems are multiples of 32, so that a warp is either
// wholly on one kind of the two or on neither.
__device__ void prep_one(const PrepArgs& a, int64_t i) {
  const int64_t nre = round_par_elems(a);
  if (i < nre) {
    const int64_t nr = (int64_t)a.n_rpf + a.n_rpb;
    int64_t r = i >> 4;
    const bool on = r < nr;
    if (!on) r = nr - 1;
    const int e = (int)(i & 15);
    const bool fwd = r < a.n_rpf;
    if (!fwd) r -= a.n_rpf;
    const int32_t* rec = fwd ? reinterpret_cast<const int32_t*>(a.rpf_src) + r * kFwdRoundWords
                             : reinterpret_cast<const int32_t*>(a.rpb_src) + r * kBwdRoundWords;
    const RoundTerm* rt = (fwd ? a.rpf_terms : a.rpb_terms) + r * 8;
    round_params(a, on, fwd, r, rec, rt, e, threadIdx.x & 31);
    return;
  }
  i -= nre;
  const int64_t nfe = fused_elems(a);
  if (i < nfe) {
    if (i < 4 * (int64_t)a.n_fused) fused_u(a, i >> 2, (int)(i & 3));
    return;
  }
  i -= nfe;
  if (i < a.n_terms) {
    double s, c;
    sincos_prep(0.5 * term_angle(a, i), &s, &c);
    if (a.cs64) a.cs64[i] = make_double2(c, s);
    else a.cs[i] = make_float2((float)c, (float)s);
    return;
  }
  i -= a.n_terms;
  if (i < (int64_t)a.B * a.n_eff) {
    const int64_t bb = i / a.n_eff;
    const int q = (int)(i - bb * a.n_eff);
    double s = 0.0, c = 1.0;  // a padding qubit stays |0>
    if (q < a.n) {
      // simulated bit q holds circuit qubit (q - qshift) mod n
      const int qc = a.qshift ? (q + a.n - a.qshift) % a.n : q;
      sincos_prep(0.5 * (a.x64 ? a.x64[bb * a.n + qc] : (double)a.x[bb * a.n + qc]), &s, &c);
    }
    if (a.enc64) a.enc64[i] = make_double2(c, s);
    else a.enc[i] = make_float2((float)c, (float)s);
  }
}

// E_b = sum over the tiles of sample b, in tile order (deterministic).
__global__ void e_reduce_kernel(const double* e_part, int64_t B, int tps, double* E) {
  const int64_t bb = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (bb >= B) return;
  double s = 0.0;
  for (int t = 0; t < tps; ++t) s += e_part[bb * tps + t];
  E[bb] = s;
}

// The same for many partials per sample: one block per sample, thread k sums
// partials k, k + 256, ... in order, then a fixed tree (bitwise repeatable).
__global__ void __launch_bounds__(256) e_reduce_block_kernel(const double* e_part, int tps, double* E) {
  __shared__ double red[256];
  const int64_t bb = blockIdx.x;
  double s = 0.0;
  for (int t = threadIdx.x; t < tps; t += 256) s += e_part[bb * tps + t];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) E[bb] = red[0];
}

// Stage 1 of a two-stage gradient reduction over partials [row][slot]
// (slots contiguous): block (group g, chunk c) sums rows
// g * rows_per_group + c * kGReduceChunk .. (chunk end) of each slot in row
// order; consecutive threads read consecutive slots of a row.
__global__ void g_partial_kernel(const double* g_part, int64_t rows_per_group, int64_t chunks, int64_t slot_stride,
                                 int S, double* out) {
  const int64_t gc = blockIdx.x;
  const int64_t g = gc / chunks, c = gc - g * chunks;
  const int s = blockIdx.y * blockDim.x + threadIdx.x;
  if (s >= S) return;
  const int64_t r0 = g * rows_per_group + c * kGReduceChunk;
  const int64_t r1 = g * rows_per_group + min(rows_per_group, (c + 1) * (int64_t)kGReduceChunk);
  double acc = 0.0;
#pragma unroll 8
  for (int64_t r = r0; r < r1; ++r) acc += g_part[r * slot_stride + s];
  out[gc * S + s] = acc;
}

// grad[p] (or grad[b][p]) = sum over tiles, then over the slots of p, in a
// fixed order.
__global__ void g_reduce_kernel(const GradReduceArgs a) {
  // (a.loss: the last block does the step's loss beside the gradients)
  if (a.loss && blockIdx.x == gridDim.x - 1) {
    if (a.f64)
      loss_block<double>(a.loss_kind, a.E, static_cast<const double*>(a.y), a.B, a.loss_scale, a.loss, a.dLdE, a.e_part, 1,
                         threadIdx.x, 256);
    else
      loss_block<float>(a.loss_kind, a.E, static_cast<const float*>(a.y), a.B, a.loss_scale, a.loss, a.dLdE, a.e_part, 1,
                        threadIdx.x, 256);
    return;
  }
  // one warp per output value; lane k sums rows k, k+32, ... and the warp
  // combines the 32 lane sums in a fixed butterfly (bitwise repeatable)
  const int64_t out = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const int64_t n_out = a.per_sample ? (int64_t)a.B * a.n_params : a.n_params;
  if (out >= n_out) return;  // whole warps exit together
  const int64_t bb = a.per_sample ? out / a.n_params : 0;
  const int p = (int)(a.per_sample ? out - bb * a.n_params : out);
  const int64_t rows = a.per_sample ? a.tps : (int64_t)a.B * a.tps;
  const int64_t row0 = a.per_sample ? bb * a.tps : 0;
  double s = 0.0;
  for (int k = a.param_off[p]; k < a.param_off[p + 1]; ++k) {
    const int64_t col = (int64_t)a.param_slots[k] * a.slot_step;
#pragma unroll 8
    for (int64_t t = lane; t < rows; t += 32) s += a.g_part[(row0 + t) * a.slot_stride + col];
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) a.grad[out] = s;
}

// Loss and dL/dE in one block of nthr threads (32 .. 256) with a fixed-order
// reduction (warp shuffles, then the warp sums in warp 0); labels float32, or float64
// for complex128 plans. scale = 2 / B (MSE: dL/dE_i = scale (E_i - y_i)).
// With e_part: E_i is first summed from its tps partials in tile order (as
// e_reduce_kernel does) and stored; they are read from L2, as they may come
// from other CTAs of the same launch.
template <class Y>
__device__ void loss_block(int kind, double* E, const Y* y, int64_t B, double scale, double* loss, double* dLdE,
                           const double* e_part, int tps, int tid, int nthr) {
  __shared__ double red[8];
  double s = 0.0;
#pragma unroll 4
  for (int64_t i = tid; i < B; i += nthr) {
    double Ei;
    if (e_part) {
      Ei = 0.0;
      for (int t = 0; t < tps; ++t) Ei += __ldcg(e_part + i * tps + t);
      E[i] = Ei;
    } else {
      Ei = E[i];
    }
    if (kind == 1) {
      const double d = Ei - (double)y[i];
      s += d * d;
      dLdE[i] = scale * d;
    } else {
      s += Ei;
      dLdE[i] = 1.0;
    }
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((tid & 31) == 0) red[tid >> 5] = s;
  __syncthreads();
  if (tid < 32) {
    s = tid < (nthr >> 5) ? red[tid] : 0.0;
    for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (tid == 0) loss[0] = kind == 1 ? s * (0.5 * scale) : s;
  }
}

template <class Y>
__global__ void __launch_bounds__(256) loss_kernel(int kind, double* E, const Y* y, int64_t B, double scale,
                                                   double* loss, double* dLdE, const double* e_part, int tps) {
  loss_block<Y>(kind, E, y, B, scale, loss, dLdE, e_part, tps, threadIdx.x, 256);
}

// ---- batched persistent launch -------------------------------------------------
namespace {

template <class T>
__device__ __forceinline__ T* rebase(T* p, char* base) {
  return reinterpret_cast<T*>(base + reinterpret_cast<uintptr_t>(p));
}
template <class T>
__device__ __forceinline__ const T* rebase(const T* p, char* base) {
  return reinterpret_cast<const T*>(base + reinterpret_cast<uintptr_t>(p));
}

__device__ __forceinline__ int find_circuit(const int64_t* off, int n, int64_t i) {
  int lo = 0, hi = n;  // off[lo] <= i < off[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (off[mid] <= i) lo = mid;
    else hi = mid;
  }
  return lo;
}

// Copy a circuit's pass arguments into shared memory with pass descriptor pd
// and the workspace pointers rebased.
__device__ void load_args(PassArgs& dst, const PassArgs& src, const PassDesc& pd, char* ws) {
  const uint32_t* s = reinterpret_cast<const uint32_t*>(&src);
  uint32_t* d = reinterpret_cast<uint32_t*>(&dst);
  for (int i = threadIdx.x; i < (int)(sizeof(PassArgs) / 4); i += blockDim.x) d[i] = s[i];
  __syncthreads();
  if (threadIdx.x == 0) {
    dst.pd = pd;
    dst.mats = rebase(dst.mats, ws);
    dst.rpar = rebase(dst.rpar, ws);
    dst.enc = rebase(dst.enc, ws);
    dst.work = rebase(dst.work, ws);
    dst.lam = rebase(dst.lam, ws);
    dst.slots = rebase(dst.slots, ws);
    dst.dLdE = rebase(dst.dLdE, ws);
    dst.e_part = rebase(dst.e_part, ws);
    dst.g_part = rebase(dst.g_part, ws);
  }
  __syncthreads();
}

// Shared memory of the persistent kernel: psi and lambda tiles, the arguments
// of the running pass and pass_cta's own (one dynamic block, so that the pass
// functions, which are called and not inlined, share it).
struct BatchShared {
  PassArgs args;
  PassShared pass;
};
__device__ __forceinline__ BatchShared& batch_shared() {
  extern __shared__ __align__(16) float2 smem[];
  return *reinterpret_cast<BatchShared*>(smem + 2 * kTilePad);
}
// Called, so that each instance has the registers to itself: inlined side by
// side in the persistent loop they spilled 156 bytes.
template <bool BWD, int KC>
__device__ __noinline__ void batch_pass(int64_t first_tile) {
  extern __shared__ __align__(16) float2 smem[];
  BatchShared& bs = batch_shared();
  pass_cta<BWD, true, false, false, KC>(bs.args, first_tile, smem, bs.pass);
}

// The tile groups (as many tiles as a CTA holds) rank, rank + n_ranks, ... of
// one pass over samples b0 .. b0 + ns - 1.
__device__ void run_item_pass(bool bwd, const BatchCircuit& C, const PassDesc& pd, char* ws, int64_t b0, int ns,
                              uint32_t rank, uint32_t n_ranks) {
  BatchShared& bs = batch_shared();
  load_args(bs.args, bwd ? C.ba : C.fa, pd, ws);
  const int tpc = kThreads >> (pd.K - kRegBits);
  const int64_t tps = 1ll << C.fa.tps_log2;
  const int64_t groups = (ns * tps + tpc - 1) / tpc;
  for (int64_t g = rank; g < groups; g += n_ranks) {
    if (bwd && C.ba.g_accum) {
      // rows per sample: one for each CTA that takes tiles of it
      const int64_t per = tps / tpc, gs = g & (per - 1);
      if (threadIdx.x == 0) {
        bs.args.g_row = (b0 + g / per) * C.g_ranks + (gs & (C.g_ranks - 1));
        bs.args.g_first = gs < C.g_ranks;
      }
      __syncthreads();
    }
    const int64_t first = b0 * tps + g * tpc;
    if (pd.K == kMaxTileBits) {
      if (bwd) batch_pass<true, 12>(first);
      else batch_pass<false, 12>(first);
    } else {
      if (bwd) batch_pass<true, 0>(first);
      else batch_pass<false, 0>(first);
    }
  }
}

}  // namespace

__global__ void batch_prep_kernel(const BatchArgs a, int64_t total) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total) return;
  const int c = find_circuit(a.prep_off, a.n_circ, i);
  PrepArgs p = a.circ[c].prep;
  p.theta = a.theta + a.circ[c].theta_off;
  p.x = a.x + a.circ[c].x_off;
  p.mats = rebase(p.mats, a.ws);
  p.rpf = rebase(p.rpf, a.ws);
  p.rpb = rebase(p.rpb, a.ws);
  p.enc = rebase(p.enc, a.ws);
  prep_one(p, i - a.prep_off[c]);
}

// Persistent kernel over two queues of work items (some samples of one circuit,
// longest first). Items whose samples span several tiles are run by a cluster
// of CTAs: each pass's tiles are dealt to the CTAs, with a cluster barrier
// between passes (it also orders their writes to the states). One CTA per
// sample made the longest item the length of the launch: 32 circuits of 8 to
// 16 qubits, up to 60 layers, 13.81 ms with clusters of one CTA, 6.97 with four.
// Items of single-tile circuits are then taken by the CTAs one by one. Items never wait on each other.
__device__ void run_item(const BatchArgs& a, const BatchItem item, bool wide) {
  namespace cg = cooperative_groups;
  const BatchCircuit& C = a.circ[item.c];
  const uint32_t rank = wide ? cg::this_cluster().block_rank() : 0u;
  const uint32_t n_ranks = wide ? cg::this_cluster().num_blocks() : 1u;
  const int64_t b0 = item.b0;
  const int ns = (int)min((int64_t)C.samples_per_item, C.fa.B - b0);
  auto barrier = [&]() {
    if (wide) cg::this_cluster().sync();
    else __syncthreads();
  };
  for (int p = 0; p < C.n_fwd; ++p) {
    run_item_pass(false, C, C.fwd[p], a.ws, b0, ns, rank, n_ranks);
    barrier();
  }
  // E and dL/dE of the item's samples
  if (rank == 0) {
    const int64_t tps = 1ll << C.fa.tps_log2;
    for (int i = (int)threadIdx.x; i < ns; i += kThreads) {
      const int64_t b = b0 + i;
      const double* ep = rebase(C.fa.e_part, a.ws) + b * tps;
      double e = 0.0;
      for (int64_t t = 0; t < tps; ++t) e += __ldcg(ep + t);
      const int64_t s = C.sample_off + b;
      a.E[s] = e;
      double g = 1.0, lt = e;
      if (C.loss_kind == 1) {
        const double dd = e - (double)a.y[s];
        g = 2.0 * dd * C.inv_B;
        lt = dd * dd * C.inv_B;
      }
      const_cast<double*>(rebase(C.ba.dLdE, a.ws))[b] = g;  // the item's own workspace row
      a.lterm[s] = lt;
    }
  }
  barrier();
  for (int p = 0; p < C.n_bwd; ++p) {
    run_item_pass(true, C, C.bwd[p], a.ws, b0, ns, rank, n_ranks);
    barrier();
  }
}

__global__ void __launch_bounds__(kThreads, 2) batch_kernel(const BatchArgs a) {
  namespace cg = cooperative_groups;
  __shared__ int s_item;
  for (;;) {
    if (cg::this_cluster().block_rank() == 0 && threadIdx.x == 0) s_item = atomicAdd(a.queue, 1);
    cg::this_cluster().sync();
    const int it = *cg::this_cluster().map_shared_rank(&s_item, 0);
    cg::this_cluster().sync();
    if (it >= a.n_wide) break;
    run_item(a, a.items[it], true);
  }
  for (;;) {
    if (threadIdx.x == 0) s_item = a.n_wide + atomicAdd(a.queue + 1, 1);
    __syncthreads();
    const int it = s_item;
    __syncthreads();
    if (it >= a.n_items) return;
    run_item(a, a.items[it], false);
  }
}

// grad[o], o over every circuit's parameters: one warp per value, fixed order.
__global__ void batch_g_reduce_kernel(const BatchArgs a, int64_t n_out) {
  const int64_t o = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (o >= n_out) return;
  const int c = find_circuit(a.grad_out_off, a.n_circ, o);
  const BatchCircuit& C = a.circ[c];
  const int p = (int)(o - a.grad_out_off[c]);
  const double* gp = rebase(C.ba.g_part, a.ws);
  const int64_t rows = C.ba.g_accum ? C.ba.B * C.g_ranks : (C.ba.B << C.ba.tps_log2);
  double s = 0.0;
  for (int k = C.param_off[p]; k < C.param_off[p + 1]; ++k) {
    const int term = C.param_terms[k];
    for (int64_t r = lane; r < rows; r += 32) s += gp[r * C.ba.n_slots + term];
  }
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if (lane == 0) a.grad[C.grad_off + p] = s;
}

__global__ void batch_loss_kernel(const BatchArgs a) {
  __shared__ double red[256];
  double s = 0.0;
  for (int64_t i = threadIdx.x; i < a.n_samples; i += blockDim.x) s += a.lterm[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) a.loss[0] = red[0];
}

cudaError_t opt_in(const void* fn, size_t smem, OptIn& o) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const bool tab = dev >= 0 && dev < 64;
  if (tab && o.done[dev].load(std::memory_order_acquire)) return cudaSuccess;
  e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess && tab) o.done[dev].store(true, std::memory_order_release);
  return e;
}

int device_sms() {
  static std::atomic<int> cache[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  const bool tab = dev >= 0 && dev < 64;
  if (tab) {
    const int v = cache[dev].load(std::memory_order_relaxed);
    if (v > 0) return v;
  }
  int v = 0;
  if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  if (tab) cache[dev].store(v, std::memory_order_relaxed);
  return v;
}

int64_t stream_grid(int64_t want) {
  const int64_t cap = 16ll * device_sms();
  return cap > 0 && want > cap ? cap : want;
}

namespace {
constexpr size_t kBatchSmem = 2 * (size_t)kTilePad * sizeof(float2) + sizeof(BatchShared);

cudaLaunchConfig_t batch_config(int clusters, int size, cudaStream_t st, cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(clusters * size));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kBatchSmem;
  cfg.stream = st;
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = (unsigned)size;
  attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

cudaError_t batch_opt_in() {
  static OptIn once;
  return opt_in(reinterpret_cast<const void*>(batch_kernel), kBatchSmem, once);
}
}  // namespace

// Clusters of `size` CTAs of the persistent kernel that the device runs at once
// (0 when it cannot).
int batch_clusters(int size) {
  cudaLaunchAttribute attr;
  const cudaLaunchConfig_t cfg = batch_config(1, size, nullptr, &attr);
  int n = 0;
  if (batch_opt_in() != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, reinterpret_cast<const void*>(batch_kernel), &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

cudaError_t launch_batch(const BatchArgs& a, int clusters, int cluster_size, int64_t prep_total, int64_t n_grad_out,
                         cudaStream_t st) {
  cudaError_t e = batch_opt_in();
  if (e != cudaSuccess) return e;
  if (prep_total > 0) batch_prep_kernel<<<(unsigned)((prep_total + 63) / 64), 64, 0, st>>>(a, prep_total);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(a.queue, 0, 2 * sizeof(int32_t), st)) != cudaSuccess) return e;
  if (a.n_items > 0) {
    const int narrow = (a.n_items - a.n_wide + cluster_size - 1) / cluster_size;
    const int want = a.n_wide > narrow ? a.n_wide : narrow;
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = batch_config(clusters < want ? clusters : want, cluster_size, st, &attr);
    if ((e = cudaLaunchKernelEx(&cfg, batch_kernel, a)) != cudaSuccess) return e;
  }
  if (n_grad_out > 0) batch_g_reduce_kernel<<<(unsigned)((n_grad_out * 32 + 255) / 256), 256, 0, st>>>(a, n_grad_out);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  batch_loss_kernel<<<1, 256, 0, st>>>(a);
  return cudaGetLastError();
}

// ---- launchers ----------------------------------------------------------------
cudaError_t launch_prep(const PrepArgs& a, cudaStream_t st) {
  int64_t total = prep_elems(a);
  if (total == 0 && !a.zero_word) return cudaSuccess;
  if (total == 0) total = 1;  // element 0 only clears the counter
  // float64 work per element: small blocks spread it over more SMs
  const int blk = 64;
  prep_kernel<<<(unsigned)((total + blk - 1) / blk), blk, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_pass(bool bwd, const PassArgs& a, cudaStream_t st, int fwd_ctas) {
  const int tl2 = a.pd.K - kRegBits;
  const int64_t total_tiles = (int64_t)a.B << a.tps_log2;
  if (total_tiles == 0) return cudaSuccess;
  const int n_sm = device_sms();
  if (n_sm == 0) return cudaErrorInvalidDevice;
  // CTAs of 256 threads hold several tiles of fewer than 12 qubits. While they
  // would leave SMs without one, CTAs get smaller (one tile, one warp at least):
  // n = 8, d = 20, 64 samples on 32 SMs instead of 4: step 120 -> 98 us; n = 10,
  // 256 samples 145 -> 136 us. Launches that fill the SMs keep 256 threads.
  // Rounds of launches with at most a warp per scheduler (4 per SM) run two
  // threads per column instead: n = 8, d = 20, 64 samples 96 -> 87 us a step; n =
  // 10, 256 samples 136 -> 123; n = 11, 128 samples 134 -> 124. With twice as
  // many warps it is slower (n = 10, 512 samples 155 -> 168). (12-qubit tiles
  // have two warps per scheduler as they are, and lose by it: n = 13, d = 31, 37
  // samples 375 -> 436 us.)
  const bool rounds = a.rounds != nullptr, rx = rounds && a.rx_items;
  const bool k12 = a.pd.K == kMaxTileBits;
  const bool half = rounds && !k12 && (total_tiles << tl2) <= 128ll * n_sm;
  const int tt2 = tl2 + (half ? 1 : 0);  // log2 threads per tile
  int thr = kThreads;
  while (thr > 32 && thr > (1 << tt2) && (total_tiles << tt2) < (int64_t)thr * n_sm) thr >>= 1;
  const int tiles_per_cta = thr >> tt2;
  const int64_t grid = (total_tiles + tiles_per_cta - 1) / tiles_per_cta;
  const size_t smem = (size_t)(bwd ? 2 : 1) * (thr >> (half ? 1 : 0)) * 17 * sizeof(float2);
  // 12-qubit tiles run the instances compiled for them; a single-wave forward
  // keeps the 128-register instance, more tiles than two CTAs per SM hold run
  // with three per SM (fewer registers, more warps to hide latency across waves)
  const bool three =
      rounds && !bwd && (fwd_ctas == 3 || (fwd_ctas == 0 && (total_tiles << tl2) > 2ll * kThreads * n_sm));
#define QF_RUN(...)                                                                          \
  do {                                                                                       \
    static OptIn once;                                                                       \
    const cudaError_t e_ = opt_in(reinterpret_cast<const void*>(__VA_ARGS__), 2 * kTilePad * sizeof(float2), once);   \
    if (e_ != cudaSuccess) return e_;                                                        \
    __VA_ARGS__<<<(unsigned)grid, thr, smem, st>>>(a);                                       \
    return cudaGetLastError();                                                               \
  } while (0)
  // one CTA per SM at most: the adjoint's registers need not leave room for two (150
  // instead of 109: a step of n = 12, d = 20, 64 samples 135 us against 138; a ring
  // of 13 qubits, d = 31, 37 samples 354 against 362). Rounds on smaller tiles have
  // no such launches but those of exactly 256 threads per SM: below 128 two threads
  // share a column, from there on CTAs of 128 outnumber the SMs
  const bool alone = grid <= n_sm;
  if (half && bwd) {
    if (rx) QF_RUN(pass_kernel<true, true, true, 2, 0, 1>);
    QF_RUN(pass_kernel<true, true, false, 2, 0, 1>);
  }
  if (half) {
    if (rx) QF_RUN(pass_kernel<false, true, true, 2, 0, 1>);
    QF_RUN(pass_kernel<false, true, false, 2, 0, 1>);
  }
  if (bwd) {
    if (!rounds && alone) QF_RUN(pass_kernel<true, false, false, 1>);
    if (!rounds) QF_RUN(pass_kernel<true, false>);
    if (rx && k12) QF_RUN(pass_kernel<true, true, true, 2, 12>);
    if (rx) QF_RUN(pass_kernel<true, true, true>);
    if (k12 && alone) QF_RUN(pass_kernel<true, true, false, 1, 12>);
    if (k12) QF_RUN(pass_kernel<true, true, false, 2, 12>);
    QF_RUN(pass_kernel<true, true>);
  }
  if (!rounds) QF_RUN(pass_kernel<false, false>);
  if (rx && k12 && three) QF_RUN(pass_kernel<false, true, true, 3, 12>);
  if (rx && k12) QF_RUN(pass_kernel<false, true, true, 2, 12>);
  if (rx && three) QF_RUN(pass_kernel<false, true, true, 3>);
  if (rx) QF_RUN(pass_kernel<false, true, true>);
  if (k12 && three) QF_RUN(pass_kernel<false, true, false, 3, 12>);
  if (k12) QF_RUN(pass_kernel<false, true, false, 2, 12>);
  if (three) QF_RUN(pass_kernel<false, true, false, 3>);
  QF_RUN(pass_kernel<false, true>);
#undef QF_RUN
}

// ---- observables whose X/Y qubits lie outside the tile (App. B.2) ---------------
// E partials, rows per sample (the layout of the pass kernels). O is Hermitian,
// so x and its partner x ^ xm contribute the same real part: a CTA sums
// 2 Re(conj(a_x) (O a)_x), (O a)_x = i^{#Y} (-1)^{|(x^xm)&zm|} a_{x^xm}, over its
// share of the x whose bit h (the highest of xm) is clear, two neighbouring x
// at a time. Each amplitude is read once; reading x and its partner for every
// x took 0.187 ms for 100 states of 20 qubits, this 0.146 ms.
__global__ void __launch_bounds__(kThreads) expect_full_kernel(const float2* psi, int n_eff, int64_t rows,
                                                               uint32_t xm, uint32_t zm, uint32_t yc,
                                                               double* e_part) {
  __shared__ double red[kThreads / 32];
  const int64_t dim = 1ll << n_eff;
  const int64_t pairs = dim / rows / 4;  // pairs of neighbours in a CTA's share (h >= 4, rows <= dim / 32)
  const int64_t b = blockIdx.x / rows, t = blockIdx.x - b * rows;
  const float2* s = psi + b * dim;
  const int h = 31 - __clz(xm);
  float acc = 0.f;
#pragma unroll 4
  for (int64_t k = threadIdx.x; k < pairs; k += kThreads) {
    const uint32_t q = 2u * (uint32_t)(t * pairs + k);
    const uint32_t x = (q & ((1u << h) - 1u)) | ((q >> h) << (h + 1)), xp = x ^ xm;
    const float4 v = __ldcg(reinterpret_cast<const float4*>(s + x));
    float4 w = __ldcg(reinterpret_cast<const float4*>(s + (xp & ~1u)));
    if (xm & 1u) w = make_float4(w.z, w.w, w.x, w.y);
    const float2 w0 = mul_ipow(make_float2(w.x, w.y), yc), w1 = mul_ipow(make_float2(w.z, w.w), yc);
    acc += flip(v.x * w0.x + v.y * w0.y, __popc(xp & zm) & 1u);
    acc += flip(v.z * w1.x + v.w * w1.y, __popc((xp ^ 1u) & zm) & 1u);
  }
  double d = 2.0 * (double)acc;
  for (int off = 16; off > 0; off >>= 1) d += __shfl_xor_sync(0xffffffffu, d, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = d;
  __syncthreads();
  if (threadIdx.x == 0) {
    double sum = 0.0;
    for (int w = 0; w < kThreads / 32; ++w) sum += red[w];
    e_part[blockIdx.x] = sum;
  }
}

cudaError_t launch_expect_full(const float2* psi, int n_eff, int64_t B, int64_t rows, uint32_t xm, uint32_t zm,
                               uint32_t yc, double* e_part, cudaStream_t st) {
  if (B == 0) return cudaSuccess;
  expect_full_kernel<<<(unsigned)(B * rows), kThreads, 0, st>>>(psi, n_eff, rows, xm, zm, yc, e_part);
  return cudaGetLastError();
}

cudaError_t launch_pass_tc(const PassArgs& a, cudaStream_t st) {
  if (a.pd.K != kMaxTileBits || a.rounds == nullptr || a.tcb == nullptr) return cudaErrorInvalidValue;
  const int64_t grid = (int64_t)a.B << a.tps_log2;
  if (grid == 0) return cudaSuccess;
  const size_t smem = (size_t)kTilePad * sizeof(float2) + (size_t)2 * kMaxStepRounds * kTcBFloats * sizeof(float);
  static OptIn once;
  cudaError_t e = opt_in(reinterpret_cast<const void*>(tc_pass_kernel), smem, once);
  if (e != cudaSuccess) return e;
  tc_pass_kernel<<<(unsigned)grid, kThreads, smem, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_tc_tables(const uint4* fwd_rounds, int32_t n_rounds, const double* mats64, float* tcb,
                             cudaStream_t st) {
  const int64_t total = (int64_t)n_rounds * 1024;
  if (total == 0) return cudaSuccess;
  tc_table_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(fwd_rounds, n_rounds, mats64, tcb);
  return cudaGetLastError();
}

// Failure-path check of the bounded waits: one thread waits on an mbarrier
// that nothing arrives at, gives up after `limit` polls and records the
// timeout in the device error word, exactly as the tensor-core path would.
__global__ void bounded_wait_probe_kernel(long long limit) {
  __shared__ __align__(8) uint64_t mbar;
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar)) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  const uint32_t addr = smem_u32(&mbar);
  for (long long it = 0; it < limit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(addr), "r"(0u)
        : "memory");
    if (done) return;
  }
  atomicExch(&g_qf_device_status, 1);
}

cudaError_t bounded_wait_probe(long long limit, cudaStream_t st) {
  if (limit < 1 || limit > (1ll << 20)) return cudaErrorInvalidValue;
  bounded_wait_probe_kernel<<<1, 1, 0, st>>>(limit);
  return cudaGetLastError();
}

cudaError_t device_status(int32_t* code, cudaStream_t st) {
  int32_t v = 0;
  cudaError_t e = cudaMemcpyFromSymbolAsync(&v, g_qf_device_status, sizeof(v), 0, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return e;
  *code = v;
  const int32_t zero = 0;
  e = cudaMemcpyToSymbolAsync(g_qf_device_status, &zero, sizeof(zero), 0, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  return e;
}

cudaError_t launch_e_reduce(const double* e_part, int64_t B, int tps, double* E, cudaStream_t st) {
  if (B == 0) return cudaSuccess;
  if (tps >= 256) e_reduce_block_kernel<<<(unsigned)B, 256, 0, st>>>(e_part, tps, E);
  else e_reduce_kernel<<<(unsigned)((B + 255) / 256), 256, 0, st>>>(e_part, B, tps, E);
  return cudaGetLastError();
}

cudaError_t launch_g_reduce(const GradReduceArgs& a, cudaStream_t st) {
  const int64_t n = a.per_sample ? (int64_t)a.B * a.n_params : a.n_params;
  if (n == 0) return cudaSuccess;
  GradReduceArgs r = a;
  if (g_reduce_stages(a.tps, a.slot_step) == 2) {
    // many rows per output: coalesced chunk sums first (groups: the samples
    // in per-sample mode, else all rows), then the fixed-order sum over chunks
    if (a.scratch == nullptr || a.B == 0 || a.loss) return cudaErrorInvalidValue;
    const int64_t groups = a.per_sample ? a.B : 1;
    const int64_t rows = a.per_sample ? a.tps : a.B * a.tps;
    const int64_t chunks = (rows + kGReduceChunk - 1) / kGReduceChunk;
    const int S = (int)a.slot_stride;
    const dim3 grid((unsigned)(groups * chunks), (unsigned)((S + 255) / 256));
    g_partial_kernel<<<grid, 256, 0, st>>>(a.g_part, rows, chunks, a.slot_stride, S, a.scratch);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    r.g_part = a.scratch;
    r.B = groups;
    r.tps = chunks;
    r.per_sample = a.per_sample;
  }
  const int64_t threads = n * 32;
  g_reduce_kernel<<<(unsigned)((threads + 255) / 256) + (r.loss ? 1u : 0u), 256, 0, st>>>(r);
  return cudaGetLastError();
}

cudaError_t launch_loss(int kind, const double* E, const float* y, int64_t B, double* loss, double* dLdE,
                        cudaStream_t st) {
  loss_kernel<float><<<1, 256, 0, st>>>(kind, const_cast<double*>(E), y, B, B > 0 ? 2.0 / (double)B : 0.0, loss,
                                         dLdE, nullptr, 0);
  return cudaGetLastError();
}

cudaError_t launch_loss64(int kind, const double* E, const double* y, int64_t B, double* loss, double* dLdE,
                          cudaStream_t st) {
  loss_kernel<double><<<1, 256, 0, st>>>(kind, const_cast<double*>(E), y, B, B > 0 ? 2.0 / (double)B : 0.0, loss,
                                          dLdE, nullptr, 0);
  return cudaGetLastError();
}

bool e_loss_fusable(int64_t B, int tps) { return tps < 256 && B * tps <= 65536; }

template <class Y>
static cudaError_t launch_e_loss_t(const double* e_part, int tps, int kind, double* E, const Y* y, int64_t B,
                                   double* loss, double* dLdE, cudaStream_t st) {
  loss_kernel<Y><<<1, 256, 0, st>>>(kind, E, y, B, B > 0 ? 2.0 / (double)B : 0.0, loss, dLdE, e_part, tps);
  return cudaGetLastError();
}

cudaError_t launch_e_loss(const double* e_part, int tps, int kind, double* E, const float* y, int64_t B,
                          double* loss, double* dLdE, cudaStream_t st) {
  return launch_e_loss_t<float>(e_part, tps, kind, E, y, B, loss, dLdE, st);
}

cudaError_t launch_e_loss64(const double* e_part, int tps, int kind, double* E, const double* y, int64_t B,
                            double* loss, double* dLdE, cudaStream_t st) {
  return launch_e_loss_t<double>(e_part, tps, kind, E, y, B, loss, dLdE, st);
}

}  // namespace qf
