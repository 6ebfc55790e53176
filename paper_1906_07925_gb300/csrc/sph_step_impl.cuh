// Relaxation-step kernels (the step of Algorithm 1), templated on the
// dimension D and the working precision T. Instantiated per dimension in
// sph_step_2d.cu / sph_step_3d.cu.
//
// State. Each particle is an int64 coordinate per axis (Frame). Pair vectors
// come from a per-step view: FP32 keeps the low 32 bits of X >> sv and forms
// differences modulo 2^32 (exact for nearby particles) converted without the
// conversion unit; FP64 keeps physical coordinates. Either way the rounding of
// a pair vector is relative to the pair distance, not to the domain size.
//
// Neighbour list (the neighbour search of Algorithm 1). The list of particle i holds every j
// (itself included) that can come within kappa max(h_i, h_j) before some
// particle has moved its reach (its share of the skin, k_gather_view); it is
// rebuilt, on the device, only then.
// The criterion is symmetric, so i also finds every j whose own support
// reaches i (the reverse pass gathers over such pairs).
// Passes A and B re-test the exact criteria of the current step for every
// listed pair, so the list only saves the search, never changes a result.
#pragma once

#include <algorithm>
#include <cfloat>
#include <climits>
#include <type_traits>

#include "sph_internal.h"

// resident 256-thread blocks per SM asked of the pair passes and of the list
// build (caps registers)
#ifndef SPH_PASS_MIN_BLOCKS
#define SPH_PASS_MIN_BLOCKS 4
#endif
// the pair passes are compiled for 128 and 256 threads per block
// (DevState::pass_threads picks one at launch); resident blocks per SM asked
// of them scale so that the register budget per thread is the same
// (pass B, FP32: 2D 73 against 77 us at 1,048,576 particles with 5 and 4 blocks,
// 3D 1.04 against 0.85 ms at 8,388,608: it spills at 48 registers there)
#ifndef SPH_PASSB_MIN_BLOCKS
#define SPH_PASSB_MIN_BLOCKS (D == 2 ? 5 : 4)
#endif
#ifndef SPH_PASSB_BATCH
#define SPH_PASSB_BATCH 4
#endif
#ifndef SPH_LIST_MIN_BLOCKS
#define SPH_LIST_MIN_BLOCKS 4
#endif
// the FP64 variants keep twice the registers live: at 5 blocks (48 registers)
// they spilled 600-1,000 bytes per thread; at 2 blocks (128 registers) none,
// and the 8M 3D FP64 step took 86 ms instead of 99.5 (3 blocks: 99.1)
#ifndef SPH_PASS_MIN_BLOCKS_FP64
#define SPH_PASS_MIN_BLOCKS_FP64 2
#endif
#ifndef SPH_PASSB_MIN_BLOCKS_FP64
#define SPH_PASSB_MIN_BLOCKS_FP64 2
#endif

namespace sph {

// ---------------------------------------------------------------- views ----
template <class T> struct ViewOf;
template <> struct ViewOf<float> { using type = int4; };
template <> struct ViewOf<double> { using type = V4<double>; };

// Difference of two view coordinates, in view units (finest cell edges).
// vd: the exact integer difference, rounded once to float.
// vd_coarse (the FP64 path's screen of a listed pair): the view integers are dropped to 2^-kCoarseBits c0 and their difference d (|d| < 2^22,
// certified per particle by the list build) is added to the bits of
// 1.5 * 2^(23 - kCoarseBits), whose low mantissa bit weighs 2^-kCoarseBits: the
// float is then bias + d 2^-kCoarseBits exactly, converted by one integer add
// and one float subtract instead of the conversion unit.
__device__ __forceinline__ float vd(const Frame<float>& F, int a, int b) { return (float)(a - b) * F.vscale; }
__device__ __forceinline__ double vd(const Frame<double>&, double a, double b) { return a - b; }
__device__ __forceinline__ float vd_coarse(const Frame<float>& F, int a, int b) {
  // the modular difference is exact; shift it, not the (wrapped) operands
  constexpr int s = kViewBits - kCoarseBits;
  return __int_as_float(F.mbits + ((a - b) >> s)) - F.mbias;
}
// radius H widened for a screening test on coarse vectors: each coarse component
// is the exact one floored to 2^-kCoarseBits c0, so |r_coarse - r| < sqrt(3) 2^-kCoarseBits;
// the relative term covers FP32 rounding of r^2. A pair that passes is tested
// again on the exact vectors, so the slack only admits a few extra candidates.
template <class T>
__device__ __forceinline__ T screen_radius(T H) {
  return H * T(1.0 + 1.0 / (1 << 20)) + T(1.0 / (1 << (kCoarseBits - 2)));
}
// w of a view, h in view units
__device__ __forceinline__ float view_w(const int4& v) { return __int_as_float(v.w); }
__device__ __forceinline__ double view_w(const V4<double>& v) { return v.w; }
__device__ __forceinline__ float view_h(const Frame<float>&, const int4& v) { return __int_as_float(v.w); }
__device__ __forceinline__ double view_h(const Frame<double>&, const V4<double>& v) { return v.w; }

// The build view of a particle (vbuild; FP64 path: view32 until pass B renews it):
// its position, and in w its view_w rounded up to 16 bits of mantissa with its
// reach code in the low byte. The reach, in view integers:
__device__ __forceinline__ float build_w(int4 v) { return __int_as_float(v.w & ~0xFF); }
__device__ __forceinline__ float build_reach(const Frame<float>& F, int4 v, int most = 255) {
  return (float)min(v.w & 0xFF, most) * (2.0f * F.skin_q * F.hk_int) * build_w(v);
}
// FP64 path: pass B reads the reach itself (view units) with its code in the low
// byte, where a float's mantissa leaves zeros
__device__ __forceinline__ double with_code(float reach, int code) {
  return __longlong_as_double(__double_as_longlong((double)reach) | code);
}
__device__ __forceinline__ double coded_reach(double w, int most) {
  const int code = (int)(__double_as_longlong(w) & 0xFF);
  return code > most ? w * (double)((float)most / (float)code) : w;
}

// The neighbour list of particle i has list_rows(cap) rows (list_at), split at
// its build: the entries then inside their support (r < max(kappa h_i,
// kappa h_ij)) fill rows 0, 1, ... in candidate order, the others the last row,
// the one before, ... in candidate order. A pass walks the inside part first, so the
// entries that pass its exact tests cluster at the start of every list and a
// warp skips the pair body on the later rows, where no lane's entry passes.
// lcount packs both counts (bits 0-14 and 15-29); bit 31 certifies that
// every listed pair stays within the exact range of the FP32 fast conversion
// until the next rebuild.
constexpr uint32_t kFastBit = 0x80000000u;
constexpr uint32_t kCountMask = 0x7FFFu;
constexpr int kOutShift = 15;
__device__ __forceinline__ int list_in(uint32_t lc) { return (int)(lc & kCountMask); }
__device__ __forceinline__ int list_cnt(uint32_t lc) {
  return (int)(lc & kCountMask) + (int)((lc >> kOutShift) & kCountMask);
}

struct alignas(32) LL4 {
  long long x, y, z, w;
};

// physical position (relative to lo) of an integer coordinate
template <class T>
__device__ __forceinline__ T coord_phys(const Frame<T>& F, long long X) {
  return (T)X * F.q64t;
}

// view of a particle at integer position X with smoothing length h (physical):
// FP32 integers of 2^-kViewBits c0 (rounded; the low 32 bits suffice because
// only differences of nearby particles are used), FP64 c0 units; w: view_w
template <int D>
__device__ __forceinline__ int4 make_view(const Frame<float>& F, const LL4& X, float h) {
  const long long half = 1LL << (F.sv - 1);
  return make_int4((int)((X.x + half) >> F.sv), (int)((X.y + half) >> F.sv), D == 3 ? (int)((X.z + half) >> F.sv) : 0,
                   __float_as_int(h * F.inv_qv));
}
template <int D>
__device__ __forceinline__ V4<double> make_view(const Frame<double>& F, const LL4& X, double h) {
  return V4<double>{(double)X.x * F.s2v, (double)X.y * F.s2v, D == 3 ? (double)X.z * F.s2v : 0.0, h * F.inv_qv};
}

#ifndef SPH_LIST_BATCH_X
#define SPH_LIST_BATCH_X 2  // 4 spilled at the 48 / 64-register budgets of the passes using it
#endif
// The force pairs of particle i, whose pair body also needs a record of
// the neighbour (its acceleration, an adjoint): that record, fetch(j), is
// loaded for the whole batch together with the views, so each thread keeps
// 2 x SPH_LIST_BATCH_X independent gathers in flight instead of meeting the
// record's latency inside every pair body. Words are streamed (read once), the
// next batch's loaded before this one's arithmetic.
template <class VT, class Fetch, class Fn>
__device__ __forceinline__ void for_pairs_x(const uint32_t* __restrict__ words, const VT* __restrict__ view, int i,
                                            int cnt, int cap, Fetch&& fetch, Fn&& pair) {
  using XT = decltype(fetch(0));
  constexpr int B = SPH_LIST_BATCH_X;
  const uint32_t* __restrict__ p = words + pair_at(i, 0, cap);
  int k = 0;
  uint32_t ahead[B];
  if (cnt >= B)
#pragma unroll
    for (int q = 0; q < B; ++q) ahead[q] = __ldcs(p + 32 * q);
  for (; k + B <= cnt; k += B) {
    uint32_t e[B];
    VT v[B];
    XT x[B];
#pragma unroll
    for (int q = 0; q < B; ++q) e[q] = ahead[q];
#pragma unroll
    for (int q = 0; q < B; ++q) {
      v[q] = view[e[q] >> 8];
      x[q] = fetch((int)(e[q] >> 8));
    }
    p += 32 * B;
    if (k + 2 * B <= cnt)
#pragma unroll
      for (int q = 0; q < B; ++q) ahead[q] = __ldcs(p + 32 * q);
#pragma unroll
    for (int q = 0; q < B; ++q) pair(e[q], v[q], x[q]);
  }
  for (; k < cnt; ++k, p += 32) {
    const uint32_t e = __ldcs(p);
    pair(e, view[e >> 8], fetch((int)(e >> 8)));
  }
}
// one 8- or 16-byte access, streamed: written once by pass A, read once by pass B
__device__ __forceinline__ void store_pair(PairRec<float>* p, uint32_t e, float f) {
  __stcs((uint2*)p, make_uint2(e, __float_as_uint(f)));
}
__device__ __forceinline__ void store_pair(PairRec<double>* p, uint32_t e, double f) {
  const long long b = __double_as_longlong(f);
  __stcs((uint4*)p, make_uint4((uint32_t)b, (uint32_t)(b >> 32), e, 0u));
}
__device__ __forceinline__ PairRec<float> load_pair(const PairRec<float>* p) {
  const uint2 v = __ldcs((const uint2*)p);
  return PairRec<float>{v.x, __uint_as_float(v.y)};
}
__device__ __forceinline__ PairRec<double> load_pair(const PairRec<double>* p) {
  const uint4 v = __ldcs((const uint4*)p);
  return PairRec<double>{__longlong_as_double((long long)v.x | (long long)v.y << 32), v.z, 0u};
}
// the factor that all FP32 pair records leave out: (h / tau)^(2 D) of one view unit
// (common), and the sign of their odd power of -1/H in 3D
template <int D>
__device__ __forceinline__ float pair_scale(float common) { return D == 2 ? common : -common; }
template <int D>
__device__ __forceinline__ double pair_scale(double) { return 1.0; }

// The skin list of particle i as quads of entries (split at its build, see
// kFastBit), in the order: full quads of the inside part, full quads of the
// outside part, what is left of each. quad(e, valid): four list words, and
// which of them are entries (bit q; std::true_type: all). The next full quad
// is fetched into L2 while the current one is used: its words come from DRAM,
// the neighbours' views mostly from the caches (holding the next quad in
// registers instead spilled: pass A of 8,388,608 particles 1.82 ms against 1.67).
template <class Quad>
__device__ __forceinline__ void for_quads(const uint32_t* __restrict__ list, int i, uint32_t lc, int cap, Quad&& quad) {
  const int n_in = list_in(lc), n_out = list_cnt(lc) - n_in;
  int qi = n_in >> 2, left = qi + (n_out >> 2);
  const uint4* __restrict__ at = (const uint4*)(list + list_at(i, 0, cap));
  const auto last = [&] { return (const uint4*)(list + list_at(i, list_rows(cap) - 4, cap)); };
  if (qi == 0) at = last();
  while (left > 0) {
    const uint4 w = __ldcs(at);
    at += qi > 0 ? 32 : -32;
    if (--qi == 0) at = last();
    --left;
    if (left > 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(at));
    quad(w, std::true_type{});
  }
#pragma unroll 1
  for (int part = 0; part < 2; ++part) {
    const int m = (part ? n_out : n_in) & 3;
    if (m)
      quad(__ldcs((const uint4*)(list + list_at(i, part ? list_rows(cap) - 4 - (n_out & ~3) : n_in & ~3, cap))),
           part ? (0xF0u >> m) & 0xFu : (1u << m) - 1u);
  }
}

// sum over the G lanes of a group (G a power of two), in every lane
template <int G, class V>
__device__ __forceinline__ V group_sum(V v) {
  for (int o = 1; o < G; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// the lanes of this lane's group, and those of them below it
template <int G>
__device__ __forceinline__ unsigned group_mask() {
  return G == 32 ? 0xffffffffu : ((1u << G) - 1u) << (threadIdx.x & 31 & ~(G - 1));
}
__device__ __forceinline__ unsigned lanes_below() { return (1u << (threadIdx.x & 31)) - 1u; }

// row of entry k of a list whose first n_in entries sit in rows 0.. and the
// rest in the last row, the one before, ...
__device__ __forceinline__ int list_row(int k, int n_in, int cap) {
  return k < n_in ? k : list_rows(cap) - 1 - (k - n_in);
}
// pair(e, view of e) for every entry of the skin list of particle i, what is
// left of the inside part before the outside part, four entries in flight. A
// body of FP64 arithmetic costs as much for one lane as for 32, so the lanes'
// entries have to stay in step: no loop of its own for what is left (a lane with
// 15 entries then met a lane with 16 in different loops), and not the quads'
// order with their remainders last (3 % slower).
template <class VT, class Fn>
__device__ __forceinline__ void for_skin_list(const uint32_t* __restrict__ list, const VT* __restrict__ view, int i,
                                              uint32_t lc, int cap, Fn&& pair) {
  const int cnt = list_cnt(lc), n_in = list_in(lc);
  for (int k = 0; k < cnt; k += 4) {
    uint32_t e[4];
    VT v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) e[q] = list[list_at(i, list_row(min(k + q, cnt - 1), n_in, cap), cap)];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = view[e[q] >> 8];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (k + q < cnt) pair(e[q], v[q]);
  }
}

// The FP64 path's skin list screened on its FP32 views (v32, kept current
// every step): each entry is first tested on coarse FP32 differences
// (screen), and only the entries that pass gather their FP64 view for the
// exact FP64 tests (pair). The screen is conservative, so the pairs the
// exact tests accept are the same as with an FP64 screen; the entries it
// rejects cost no FP64 arithmetic (the FP64 pipe bounds that pass).
template <class VT, class Screen, class Fn>
__device__ __forceinline__ void for_skin_list_s32(const uint32_t* __restrict__ list, const int4* __restrict__ v32,
                                                  const VT* __restrict__ view, int i, uint32_t lc, int cap,
                                                  Screen&& screen, Fn&& pair) {
  const int cnt = list_cnt(lc), n_in = list_in(lc);
  for (int k = 0; k < cnt; k += 4) {
    uint32_t e[4];
    int4 w[4];
    bool ok[4];
    VT v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) e[q] = list[list_at(i, list_row(min(k + q, cnt - 1), n_in, cap), cap)];
#pragma unroll
    for (int q = 0; q < 4; ++q) w[q] = v32[e[q] >> 8];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      ok[q] = screen(w[q]) && k + q < cnt;
      if (ok[q]) v[q] = view[e[q] >> 8];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (ok[q]) pair(e[q], v[q]);
  }
}

// Staged lists (pass A, FP32): in a block whose distinct neighbours fit in
// shared memory, entry k of particle i's list is also stored, at the same
// position of llist, as (rank << 8 | colour_j) with bit kStageSelf set for
// j = i; rank numbers j within the block's staged set (sj). The views of the
// set are gathered into shared memory once per step, so the list walk reads
// them there instead of gathering each from global memory.
constexpr uint32_t kStageSelf = 1u << 20;
__device__ __forceinline__ int stage_rank(uint32_t e) {
  const int r = (int)((e >> 8) & 0xFFFu);
  return r < kStageCap ? r : kStageCap - 1;  // in range by construction; the clamp keeps any stale word in bounds
}
// 16-byte asynchronous copy global -> shared (cp.async, L2 only), and the wait
// for every copy this thread issued
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(a), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

// a length in state units rounded to the nearest integer (ties to even): the
// FP32 value converts directly (the same integer as rounding its exact FP64
// widening, without the FP64 conversion)
__device__ __forceinline__ long long state_units(float x) { return __float2ll_rn(x); }
__device__ __forceinline__ long long state_units(double x) { return llrint(x); }

template <class T> __device__ __forceinline__ T pair_r(T r2);
template <> __device__ __forceinline__ float pair_r<float>(float r2) { return r2 * rsqrtf(r2); }
template <> __device__ __forceinline__ double pair_r<double>(double r2) { return sqrt(r2); }

// ---- two FP32 pairs per instruction -----------------------------------------
// add / mul / fma on two floats at once (one issue slot for both, each rounded
// as its scalar form)
__device__ __forceinline__ float2 both(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// a product and a sum that stay two roundings (packed ones were fused to one fma,
// also where both name their rounding; the scalar forms are not)
__device__ __forceinline__ float2 mul2_apart(float2 a, float2 b) {
  return make_float2(__fmul_rn(a.x, b.x), __fmul_rn(a.y, b.y));
}
__device__ __forceinline__ float2 add2_apart(float2 a, float2 b) {
  return make_float2(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y));
}
__device__ __forceinline__ float2 max2(float2 a, float b) { return make_float2(fmaxf(a.x, b), fmaxf(a.y, b)); }
// hardware reciprocal (1 ulp) and reciprocal square root of normal numbers
__device__ __forceinline__ float fast_rcp(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float fast_rsqrt(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float2 rcp2(float2 a) { return make_float2(fast_rcp(a.x), fast_rcp(a.y)); }
__device__ __forceinline__ float2 rsqrt2(float2 a) { return make_float2(fast_rsqrt(a.x), fast_rsqrt(a.y)); }
// the skin list of particle i two entries at a time: two(e0, r0, e1, r1, on0,
// on1) with r = load(e); a place without an entry (on = false) comes with e =
// own
template <class Load, class Two>
__device__ __forceinline__ void for_twos(const uint32_t* __restrict__ list, int i, uint32_t lc, int cap, uint32_t own,
                                         Load&& load, Two&& two) {
  for_quads(list, i, lc, cap, [&](uint4 w, auto valid) {
    if constexpr (std::is_same<decltype(valid), std::true_type>::value) {
      const auto r0 = load(w.x), r1 = load(w.y), r2 = load(w.z), r3 = load(w.w);
      two(w.x, r0, w.y, r1, valid, valid);
      two(w.z, r2, w.w, r3, valid, valid);
    } else {
      const bool o0 = valid & 1u, o1 = valid & 2u, o2 = valid & 4u, o3 = valid & 8u;
      w = make_uint4(o0 ? w.x : own, o1 ? w.y : own, o2 ? w.z : own, o3 ? w.w : own);
      const auto r0 = load(w.x), r1 = load(w.y), r2 = load(w.z), r3 = load(w.w);
      two(w.x, r0, w.y, r1, o0, o1);
      two(w.z, r2, w.w, r3, o2, o3);
    }
  });
}

template <int D, class T>
__device__ __forceinline__ void abs_pos(const Frame<T>& F, const LL4& X, T* x) {
  x[0] = F.lo[0] + coord_phys(F, X.x);
  x[1] = F.lo[1] + coord_phys(F, X.y);
  x[2] = D == 3 ? F.lo[2] + coord_phys(F, X.z) : T(0);
}

// ---------------------------------------------------------- reductions ----
__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// minimum and where it sits; ties go to the smaller index (order-independent)
__device__ __forceinline__ void argmin_merge(double& v, long long& k, double ov, long long ok) {
  if (ov < v || (ov == v && ok < k)) {
    v = ov;
    k = ok;
  }
}

// ---- FP32 path: r_c / |a| and |rho / rho_t - 1| compared without FP64 work --
// One FP64 warp instruction occupies an SM's FP64 pipe for 16 cycles: with the
// particle's quotients and the block's sums in FP64 (59 instructions per warp)
// that pipe was active 58 % of a 2D pass A and 39 % of a 3D one. So the
// reductions compare FP32 values, turn to FP64 only when those tie, and add in
// fixed point. 10 steps of 1,048,576 particles in 2D: 3.14 -> 2.29 ms; 5 steps
// of 8,388,608 in 3D: 25.2 -> 23.8 ms; positions and step sizes unchanged bit for
// bit, the sums of the statistics nearer to their exact values.
// r_c / |a| (FP32, correctly rounded: monotone in the exact quotient); is a
// before b, ties by the exact quotient (products of two floats are exact in
// FP64), then by index
__device__ __forceinline__ bool ratio_before(float rca, float ana, long long ka, float rcb, float anb, long long kb) {
  if (ka < 0 || kb < 0) return kb < 0 && ka >= 0;
  const float qa = __fdiv_rn(rca, ana), qb = __fdiv_rn(rcb, anb);
  if (qa != qb) return qa < qb;
  const double l = (double)rca * (double)anb, r = (double)rcb * (double)ana;
  return l < r || (l == r && ka < kb);
}
// |rho / rho_t - 1| to a few FP32 ulp, and as the FP64 value it stands for
__device__ __forceinline__ float err_key(float r, float t) { return t > 0.0f ? fabsf(r - t) / t : -1.0f; }
__device__ __forceinline__ double err_exact(float r, float t) { return t > 0.0f ? fabs((double)r / (double)t - 1.0) : -1.0; }
__device__ __forceinline__ bool err_above(float ra, float ta, float rb, float tb) {
  const float a = err_key(ra, ta), b = err_key(rb, tb);
  if (fabsf(a - b) > 1e-6f * fmaxf(a, b) || !(fmaxf(a, b) >= 0.0f)) return a > b;
  return err_exact(ra, ta) > err_exact(rb, tb);
}

// b into a (fixed order: a's block comes first). FP32 path: by the quotients the
// partials carry; only ties look further.
template <class T>
__device__ __forceinline__ void merge(Partial& a, const Partial& b) {
  if (sizeof(T) == 4) {
    if (b.q < a.q || (b.q == a.q && ratio_before(b.rc, b.an, b.amin, a.rc, a.an, a.amin))) {
      a.rc = b.rc;
      a.an = b.an;
      a.q = b.q;
      a.amin = b.amin;
    }
    const bool near = fabsf(a.ek - b.ek) <= 1e-6f * fmaxf(a.ek, b.ek);
    if (near ? err_above(b.er, b.et, a.er, a.et) : b.ek > a.ek) {
      a.er = b.er;
      a.et = b.et;
      a.ek = b.ek;
    }
    a.ma = fmaxf(a.ma, b.ma);
  } else {
    argmin_merge(a.min_rc_a, a.amin, b.min_rc_a, b.amin);
    a.max_a = fmax(a.max_a, b.max_a);
    a.err_max = fmax(a.err_max, b.err_max);
  }
  a.sum_rho += b.sum_rho;
  a.err_l2 += b.err_l2;
  a.ipairs += b.ipairs;
  a.fpairs += b.fpairs;
  a.lentries += b.lentries;
}
__device__ __forceinline__ Partial no_partial() {
  Partial p{};
  p.min_rc_a = DBL_MAX;
  p.amin = -1;
  p.q = __int_as_float(0x7f800000);  // infinity
  p.ek = -1.0f;
  return p;
}
// Warp reductions of whole values by the integer reduction unit: a few
// instructions where five rounds of shuffles and merges took microseconds at
// the end of every pass.
__device__ __forceinline__ long long warp_sum_u40(long long v) {  // v >= 0, the sum below 2^50
  const long long lo = __reduce_add_sync(0xffffffffu, (unsigned)(v & 0xFFFFFF));
  const long long hi = __reduce_add_sync(0xffffffffu, (unsigned)(v >> 24));
  return (hi << 24) + lo;
}
// the smallest / largest of non-negative doubles (they order as their bits)
__device__ __forceinline__ double warp_min_bits(double v) {
  const unsigned hi = (unsigned)__double2hiint(v), mh = __reduce_min_sync(0xffffffffu, hi);
  const unsigned ml = __reduce_min_sync(0xffffffffu, hi == mh ? (unsigned)__double2loint(v) : 0xffffffffu);
  return __hiloint2double((int)mh, (int)ml);
}
__device__ __forceinline__ double warp_max_bits(double v) {
  const unsigned hi = (unsigned)__double2hiint(v), mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? (unsigned)__double2loint(v) : 0u);
  return __hiloint2double((int)mh, (int)ml);
}
// the lane whose r_c / |a| = q comes first (k: its particle, < 0: none); -1: none
__device__ __forceinline__ int first_ratio(float q, float rc, float an, int k) {
  constexpr unsigned all = 0xffffffffu;
  const unsigned qb = k >= 0 ? __float_as_uint(q) : 0xffffffffu;
  const unsigned qmin = __reduce_min_sync(all, qb), who = __ballot_sync(all, qb == qmin);
  if (qmin == 0xffffffffu) return -1;
  int src = __ffs(who) - 1;
  if (who & (who - 1)) {  // FP32 quotients tie: by the exact ones, then by index
    float brc = 0, ban = 0;
    int bk = -1;
    for (unsigned m = who; m; m &= m - 1) {
      const int l = __ffs(m) - 1, ok = __shfl_sync(all, k, l);
      const float orc = __shfl_sync(all, rc, l), oan = __shfl_sync(all, an, l);
      if (ratio_before(orc, oan, ok, brc, ban, bk)) {
        brc = orc;
        ban = oan;
        bk = ok;
        src = l;
      }
    }
  }
  return src;
}
// the lane whose |rho / rho_t - 1| is largest, given it to FP32 rounding (key,
// < 0: no particle); -1: none
__device__ __forceinline__ int largest_error(float key, float rho, float rt) {
  constexpr unsigned all = 0xffffffffu;
  const float top = __uint_as_float(__reduce_max_sync(all, key >= 0.0f ? __float_as_uint(key) : 0u));
  const unsigned who = __ballot_sync(all, key >= 0.0f && key >= top * (1.0f - 1e-6f));
  int src = who ? __ffs(who) - 1 : -1;
  if (who & (who - 1)) {  // several within rounding of the largest
    float br = 0.0f, bt = 0.0f;
    for (unsigned m = who; m; m &= m - 1) {
      const int l = __ffs(m) - 1;
      const float r = __shfl_sync(all, rho, l), t = __shfl_sync(all, rt, l);
      if (err_above(r, t, br, bt)) {
        br = r;
        bt = t;
        src = l;
      }
    }
  }
  return src;
}
// the total of a warp's partials, in every lane (the sums pair up the same way
// on every run; FP64 sums commute, so both ends of a pair hold the same value)
template <class T>
__device__ __forceinline__ Partial warp_total(const Partial& p) {
  constexpr unsigned all = 0xffffffffu;
  Partial q = no_partial();
  if (sizeof(T) == 4) {
    const int l = first_ratio(p.q, p.rc, p.an, (int)p.amin), s = l < 0 ? 0 : l;
    q.rc = __shfl_sync(all, p.rc, s);
    q.an = __shfl_sync(all, p.an, s);
    q.q = __shfl_sync(all, p.q, s);
    q.amin = __shfl_sync(all, (int)p.amin, s);
    const int m = largest_error(p.ek, p.er, p.et), t = m < 0 ? 0 : m;
    q.ek = __shfl_sync(all, p.ek, t);
    q.er = __shfl_sync(all, p.er, t);
    q.et = __shfl_sync(all, p.et, t);
    q.ma = __uint_as_float(__reduce_max_sync(all, __float_as_uint(p.ma)));
  } else {
    q.min_rc_a = warp_min_bits(p.min_rc_a);
    const unsigned k = p.min_rc_a == q.min_rc_a && p.amin >= 0 ? (unsigned)p.amin : 0x7fffffffu;
    const unsigned kmin = __reduce_min_sync(all, k);
    q.amin = kmin == 0x7fffffffu ? -1 : (long long)kmin;
    q.max_a = warp_max_bits(p.max_a);
    q.err_max = warp_max_bits(p.err_max);
  }
  q.sum_rho = warp_sum(p.sum_rho);
  q.err_l2 = warp_sum(p.err_l2);
  q.ipairs = warp_sum_u40(p.ipairs);
  q.fpairs = warp_sum_u40(p.fpairs);
  q.lentries = warp_sum_u40(p.lentries);
  return q;
}

// The integer part of v (|v| < 2^22, nearest) taken off v, the rest scaled up
// by 2^22: the next 22 bits of a fixed-point number.
__device__ __forceinline__ int take_limb(float& v) {
  const float t = v + 12582912.0f;
  const int l = __float_as_int(t) - 0x4B400000;
  v = (v - (t - 12582912.0f)) * 4194304.0f;
  return l;
}
// 2^(148 - b), b the biased exponent of m >= 0: scales values up to m below 2^22
__device__ __forceinline__ int fixed_exponent(float m) { return min(275 - (__float_as_int(m) >> 23), 254); }
__device__ __forceinline__ float exponent_scale(int e) { return __int_as_float(e << 23); }

// What a warp's 32 particles contribute, reduced by integer warp reductions:
// the particles of the two extrema and the two sums as three 22-bit limbs each
// at a power-of-two scale set by the warp's largest term (66 bits: sums of
// FP32 densities come out exact where FP64 adds would round).
struct WarpSums {
  float rc, an, er, et;
  int amin;
  unsigned max_a;      // bits of the largest |a|
  int rl[3], el[3];    // limbs of sum rho, sum (rho/rho_t - 1)^2
  int re, ee;          // their scale exponents (biased)
  int ni, nf, cnt;
};

// rho/rho_t - 1 = q1 + q2 + q3, a quotient by long division in three floats (each
// remainder exact or carried with its rounding error): about 2^-68 of itself, so
// that its square keeps more than an FP64 division would give
__device__ __forceinline__ void density_error(float rho, float rt, float& q1, float& q2, float& q3) {
  const float dh = rho - rt, bb = dh - rho;
  const float dl = (rho - (dh - bb)) - (rt + bb);  // rho - rt = dh + dl
  const float ri = __frcp_rn(rt);
  q1 = dh * ri;
  q1 = fmaf(fmaf(-q1, rt, dh), ri, q1);  // to the nearest, so that the next remainder is exact
  const float r = fmaf(-q1, rt, dh), s = r + dl, sb = s - r, sl = (r - (s - sb)) + (dl - sb);
  q2 = s * ri;
  q3 = (fmaf(-q2, rt, s) + sl) * ri;
}

// every lane of the warp calls; active: this lane holds a particle. Lane 0
// writes *out.
__device__ __forceinline__ void warp_sums(bool active, int i, float rc, float an, float rho, float rt, int ni, int nf,
                                          int cnt, WarpSums* out) {
  constexpr unsigned all = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  // the smallest r_c / |a|
  const bool moves = active && an > 0.0f;
  const int first = first_ratio(moves ? __fdiv_rn(rc, an) : 0.0f, rc, an, moves ? i : -1), fl = first < 0 ? 0 : first;
  const float mrc = __shfl_sync(all, rc, fl), man = __shfl_sync(all, an, fl);
  const int mi = __shfl_sync(all, i, fl);
  // the largest |a| (NaN, which raises the error word, counts as none)
  const unsigned amax = __reduce_max_sync(all, moves ? __float_as_uint(an) : 0u);
  // the largest |rho / rho_t - 1|
  float q1 = 0.0f, q2 = 0.0f, q3 = 0.0f;
  if (active) density_error(rho, rt, q1, q2, q3);
  const int worst = largest_error(active ? fabsf(q1) : -1.0f, rho, rt), wl = worst < 0 ? 0 : worst;
  const float er = __shfl_sync(all, rho, wl), et = __shfl_sync(all, rt, wl);
  const float emax = fabsf(__shfl_sync(all, q1, wl));
  // sum rho
  const float rv = active ? rho : 0.0f;
  const int re = fixed_exponent(__uint_as_float(__reduce_max_sync(all, __float_as_uint(rv))));
  float v = rv * exponent_scale(re);
  int rl[3], el[3];
  for (int k = 0; k < 3; ++k) rl[k] = __reduce_add_sync(all, take_limb(v));
  // sum (rho/rho_t - 1)^2: q1^2 = p + pl and 2 q1 q2 = c + cl exactly, and the rest
  const float p = q1 * q1, pl = fmaf(q1, q1, -p), d1 = 2.0f * q1, c = d1 * q2;
  const float cl = fmaf(q2, q2, fmaf(d1, q3, fmaf(d1, q2, -c)));
  const int ee = fixed_exponent(emax * emax * 1.00001f);  // the largest to rounding
  const float es = exponent_scale(ee), limb = 4194304.0f;
  float a = p * es, b = pl * es * limb, bc = c * es * limb, br = cl * es * limb * limb;
  el[0] = take_limb(a);
  el[1] = take_limb(a) + take_limb(b) + take_limb(bc);
  el[2] = take_limb(a) + take_limb(b) + take_limb(bc) + take_limb(br);
  for (int k = 0; k < 3; ++k) el[k] = __reduce_add_sync(all, el[k]);
  ni = __reduce_add_sync(all, ni);
  nf = __reduce_add_sync(all, nf);
  cnt = __reduce_add_sync(all, cnt);
  if (lane == 0) {
    out->rc = mrc;
    out->an = man;
    out->amin = first >= 0 ? mi : -1;
    out->max_a = amax;
    out->er = er;
    out->et = worst >= 0 ? et : 0.0f;
    for (int k = 0; k < 3; ++k) {
      out->rl[k] = rl[k];
      out->el[k] = el[k];
    }
    out->re = re;
    out->ee = ee;
    out->ni = ni;
    out->nf = nf;
    out->cnt = cnt;
  }
}
// l0 + l1 2^-22 + l2 2^-44, over the scale 2^(e - 127)
__device__ __forceinline__ double from_limbs(const int* l, int e) {
  const double s = ((double)l[2] * 0x1p-22 + (double)l[1]) * 0x1p-22 + (double)l[0];
  return s * __longlong_as_double((long long)(1023 + 127 - e) << 52);
}
__device__ __forceinline__ Partial to_partial(const WarpSums& w) {
  Partial p = no_partial();
  p.rc = w.rc;
  p.an = w.an;
  p.amin = w.amin;
  p.ma = __uint_as_float(w.max_a);
  if (w.amin >= 0) p.q = __fdiv_rn(w.rc, w.an);
  p.er = w.er;
  p.et = w.et;
  p.ek = err_key(w.er, w.et);
  p.sum_rho = from_limbs(w.rl, w.re);
  p.err_l2 = from_limbs(w.el, w.ee);
  p.ipairs = w.ni;
  p.fpairs = w.nf;
  p.lentries = w.cnt;
  return p;
}

// L2 read of a partial another block wrote
__device__ __forceinline__ Partial load_partial(const Partial* p) {
  static_assert(sizeof(Partial) == 112, "whole 16-byte words");
  Partial q;
#pragma unroll
  for (int k = 0; k < 7; ++k) ((int4*)&q)[k] = __ldcg((const int4*)p + k);
  return q;
}
// Called by one warp of every block with the block's partial in lane 0:
// the last block of a group merges the group's partials, the last group's
// block merges the groups' (each lane a fixed stride of them, then a fixed
// tree; a grid of one group ends there). True in the warp that holds the grid's total. One block merging all
// partials took a tail of 10 us at 4,096 blocks: FP64 adds run at two lanes
// per cycle on one SM.
template <class T>
__device__ __forceinline__ bool grid_total(Partial& p, Partial* partials, unsigned* ticket) {
  const int lane = threadIdx.x & 31, nb = gridDim.x, ng = (nb + kPartialGroup - 1) / kPartialGroup;
  const int g = blockIdx.x / kPartialGroup, b0 = g * kPartialGroup, gn = min(kPartialGroup, nb - b0);
  unsigned last = 0;
  if (lane == 0) {
    partials[blockIdx.x] = p;
    __threadfence();
    last = atomicAdd(ticket + 4 + g, 1u) == (unsigned)(gn - 1);
  }
  if (!__shfl_sync(0xffffffffu, last, 0)) return false;
  __threadfence();
  Partial a = no_partial();
  for (int b = lane; b < gn; b += 32) merge<T>(a, load_partial(partials + b0 + b));
  a = warp_total<T>(a);
  if (lane == 0) ticket[4 + g] = 0u;
  if (ng == 1) {
    p = a;
    return true;
  }
  if (lane == 0) {
    partials[nb + g] = a;
    __threadfence();
    last = atomicAdd(ticket, 1u) == (unsigned)(ng - 1);
  }
  if (!__shfl_sync(0xffffffffu, last, 0)) return false;
  __threadfence();
  a = no_partial();
  for (int b = lane; b < ng; b += 32) merge<T>(a, load_partial(partials + nb + b));
  a = warp_total<T>(a);
  if (lane == 0) *ticket = 0u;
  p = a;
  return true;
}

// ------------------------------------------------------------------------
// List rebuild (runs only when ctl->rebuild). Old order: buffer 1 - buf.
// ------------------------------------------------------------------------

// Gate of the step, then the cell key of each particle in the old order (level
// from h at its position, cell coordinates X >> (cshift + level)) and its count
// per cell and per scan tile: one launch for what were four, and with the
// gather making the views, a step of seven kernels instead of twelve (FP64
// thirteen). Circle (2D, 4,289 particles) 42 -> 35 us per step, general EOS at
// 99,991 80 -> 71.
// The control block as pass B left it says whether the list is rebuilt; this
// kernel moves it on (view buffer, state buffer, flags) for the kernels that
// follow: without a rebuild at once by one thread, which touches nothing the
// other blocks read; with one by the last block to finish.
template <int D, class T>
__global__ void __launch_bounds__(256) k_rekey(int n, StepCtl* ctl, int force, unsigned* __restrict__ ticket,
                                               const LL4* __restrict__ X0, const LL4* __restrict__ X1, Frame<T> F,
                                               Grid<T> G, Geom<T> geo, uint32_t* __restrict__ key,
                                               uint32_t* __restrict__ cnt, uint32_t* __restrict__ part) {
  let_successor();
  if (!(force || *(volatile int*)&ctl->need_rebuild)) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      ctl->vp ^= 1;
      ctl->rebuild = 0;
    }
    return;
  }
  const int old = ctl->buf;  // the buffer in the old order
  for (int b0 = blockIdx.x * blockDim.x; b0 < n; b0 += gridDim.x * blockDim.x) {
    const int i = b0 + threadIdx.x;
    const unsigned mask = __ballot_sync(0xffffffffu, i < n);
    if (i >= n) continue;
    const LL4 X = (old ? X1 : X0)[i];
    T x[3];
    abs_pos<D, T>(F, X, x);
    const int l = level_of_h(G, h_of<D, T>(geo, x));
    const int sh = G.cshift + l;
    const int c[3] = {(int)min((long long)G.nx[l] - 1, X.x >> sh), (int)min((long long)G.ny[l] - 1, X.y >> sh),
                      D == 3 ? (int)min((long long)G.nz[l] - 1, X.z >> sh) : 0};
    const uint32_t k =
        G.base[l] + (uint32_t)c[0] + (uint32_t)G.nx[l] * ((uint32_t)c[1] + (uint32_t)G.ny[l] * (uint32_t)c[2]);
    key[i] = k;
    const int lane = threadIdx.x & 31;
    unsigned peers = __match_any_sync(mask, k);
    if (lane == __ffs(peers) - 1) atomicAdd(&cnt[k], (uint32_t)__popc(peers));
    peers = __match_any_sync(mask, k / kScanTile);
    if (lane == __ffs(peers) - 1) atomicAdd(&part[k / kScanTile], (uint32_t)__popc(peers));
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(ticket, 1u) == gridDim.x - 1) {  // every block has read the control block
      *ticket = 0u;
      ctl->vp ^= 1;
      ctl->buf = old ^ 1;
      ctl->rebuild = 1;
      ctl->need_rebuild = 0;
      ctl->rebuilds += 1;
      ctl->lmax = 0;
      ctl->dmax = 0;
      ctl->reach_cap = 255;
    }
  }
}

// Slot s of the scatter holds old index i; its rank among the cell's members by
// particle id gives its destination (cells ordered by key, each cell by
// particle id): the state is copied there, with the view of the new order, the
// build view with the particle's reach until the next rebuild (X.w carries its
// last move, see k_pass_b; zero: none yet), and in the FP64 path the
// FP32 view its list build and pass A's screen read. (The list only has to hold
// every pair the exact FP64 tests can accept before the next rebuild, and an
// FP32 candidate test errs by ~1e-7 of the distance, far inside the list's
// margins, while FP64 arithmetic runs at a small fraction of the FP32 rate.)
template <int D, class T>
__global__ void __launch_bounds__(256) k_gather_view(
    int n, StepCtl* __restrict__ ctl, const uint32_t* __restrict__ slots, const uint32_t* __restrict__ key,
    const uint32_t* __restrict__ cstart, LL4* __restrict__ X0, LL4* __restrict__ X1, uint32_t* __restrict__ m0,
    uint32_t* __restrict__ m1, uint32_t* __restrict__ p0, uint32_t* __restrict__ p1, Frame<T> F, Geom<T> geo,
    typename ViewOf<T>::type* __restrict__ v0, typename ViewOf<T>::type* __restrict__ v1,
    typename ViewOf<T>::type* __restrict__ vbuild, int4* __restrict__ v32, Frame<float> F32) {
  after_predecessor();
  if (!ctl->rebuild) return;
  const int nb = ctl->buf, vp = ctl->vp;  // new buffers; the old order lives in the other state buffer
  const uint32_t* __restrict__ pold = nb ? p0 : p1;
  const int first = min((int)ceilf(F.skin_u / F.skin_q), 255);  // while the speed is unknown
  int most = 0;
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x) {
    const uint32_t i = slots[s];
    const uint32_t k = key[i];
    const uint32_t id = pold[i];
    const uint32_t b = cstart[k], e = cstart[k + 1];
    uint32_t rank = 0;
    for (uint32_t t = b; t < e; ++t) rank += pold[slots[t]] < id;
    const uint32_t d = b + rank;
    const LL4 X = (nb ? X0 : X1)[i];
    (nb ? X1 : X0)[d] = X;
    (nb ? m1 : m0)[d] = (nb ? m0 : m1)[i];
    (nb ? p1 : p0)[d] = id;
    T x[3];
    abs_pos<D, T>(F, X, x);
    const auto v = make_view<D>(F, X, h_of<D, T>(geo, x));
    (vp ? v1 : v0)[d] = v;
    const float moved = __uint_as_float((uint32_t)X.w);
    const float reach = fminf(fmaf(F.skin_k, moved, F.skin_lo), F.skin_hi);
    const int code = moved > 0.0f && F.skin_k > 0.0f ? min((int)ceilf(reach / F.skin_q), 255) : first;
    most = max(most, code);
    if constexpr (std::is_same<T, double>::value) {
      const long long half = 1LL << (F32.sv - 1);
      const int w = ((__float_as_int((float)view_w(v)) + 0xFF) & ~0xFF) | code;
      const int4 u = make_int4((int)((X.x + half) >> F32.sv), (int)((X.y + half) >> F32.sv),
                               D == 3 ? (int)((X.z + half) >> F32.sv) : 0, w);
      v32[d] = u;
      vbuild[d] = V4<double>{v.x, v.y, v.z, with_code(build_reach(F32, u) * F32.vscale, code)};
    } else {
      vbuild[d] = make_int4(v.x, v.y, v.z, ((v.w + 0xFF) & ~0xFF) | code);
    }
  }
  most = __reduce_max_sync(0xffffffffu, most);
  if ((threadIdx.x & 31) == 0) atomicMax(&ctl->dmax, most);
}

// Neighbour list of each particle: every j (itself included) with
//   r < kappa max(h_i, h_j) (1 + 1e-5) + (d_i + d_j) (1 + kappa lip_h),
// d the reaches of i and j: after both moved at most their reach (and h changed
// by at most lip_h times that), any pair inside the exact
// criteria is still listed. Candidates come from rows of cells of every level
// that can hold such a j, in the order (level, z row, y row, x).
// CUT: a list that does not fit at these reaches is made again with d_i and d_j at
// most the common reach (Frame::code_u) and the change of h bounded by the longer
// of the two moves, max(d_i, d_j) kappa lip_h: no longer than a list with one skin
// of twice the common reach. From then to the next rebuild no particle may move
// further than that (ctl->reach_cap), which is less than what the other lists
// allow for, so all of them hold every pair.
// The list is built on FP32 views in both precisions. Lengths of the tests are
// view integers; with w = h (build_w, view units) and m = max(w_i, w_j), kappa m is the largest
// support of the pair and the larger of kappa h_i and kappa h_ij is kappa (w_i + m) / 2.
template <bool CUT>
struct ListTarget {
  float Rs, R2;          // search radius, view units
  float wi, di, c1, c2, u2, hk, hi, r2max;  // view integers (wi: view units)
  int l0, l1;            // levels that can hold a neighbour
  int most;              // CUT: the largest code
  __device__ __forceinline__ ListTarget(const Frame<float>& F, const Grid<float>& G, float kappa, int dmax,
                                        const int4& vi) {
    most = F.code_u;
    if (CUT) dmax = min(dmax, most);
    wi = build_w(vi);
    di = build_reach(F, vi, CUT ? most : 255);
    hk = F.hk_int;
    hi = hk * wi;
    const float hv = wi, lip = G.lip_h, dv = di * F.vscale, dm = (float)dmax * F.skin_q * kappa;
    // search radius: bound h_j by Lipschitz continuity and d_j by the largest
    // reach of this build, iterate twice
    float hhi = hv;
    c2 = 1.0f + kappa * lip;
    Rs = kappa * hv * G.rfac + (dv + dm * hv) * c2;
    for (int it = 0; it < 2; ++it) {
      hhi = hv * 1.0001f + lip * Rs;
      Rs = kappa * hhi * G.rfac + (dv + dm * hhi) * c2;
      Rs = fmaxf(Rs, kappa * hv * G.rfac);
    }
    l0 = level_of_h(G, (hv * 0.9999f - lip * Rs) * F.qv);
    l1 = level_of_h(G, hhi * F.qv);
    R2 = Rs * Rs;
    c1 = 2.0f * hk * 1.00001f;
    u2 = 2.0f * F.skin_q * hk;
    r2max = R2 / (F.vscale * F.vscale);
    if (CUT) c2 = kappa * lip;
  }
  __device__ __forceinline__ float code(const int4& v) const {
    return (float)(CUT ? min(v.w & 0xFF, most) : v.w & 0xFF);
  }
  // a pair of candidates, without a branch: listed (acc), inside its support
  // now (density or force: the front of the list)
  template <int D>
  __device__ __forceinline__ void test(const int4& vi, const int4& a, const int4& b, bool (&acc)[2],
                                       bool (&inside)[2]) const {
    const float2 dx = make_float2((float)(vi.x - a.x), (float)(vi.x - b.x));
    const float2 dy = make_float2((float)(vi.y - a.y), (float)(vi.y - b.y));
    float2 r2 = fma2(dy, dy, mul2(dx, dx));
    if (D == 3) {
      const float2 dz = make_float2((float)(vi.z - a.z), (float)(vi.z - b.z));
      r2 = fma2(dz, dz, r2);
    }
    // symmetric in i and j: j lists i whenever i lists j
    const float2 wj = make_float2(build_w(a), build_w(b)), m = make_float2(fmaxf(wi, wj.x), fmaxf(wi, wj.y));
    const float2 dj = mul2(mul2(make_float2(code(a), code(b)), both(u2)), wj), d = add2(both(di), dj);
    float2 rl = mul2(both(c1), m);
    if (CUT) rl = add2(fma2(make_float2(fmaxf(di, dj.x), fmaxf(di, dj.y)), both(c2), rl), d);
    else rl = fma2(d, both(c2), rl);
    const float2 rl2 = mul2(rl, rl), hp = fma2(m, both(hk), both(hi)), hp2 = mul2(hp, hp);
    acc[0] = r2.x < fminf(rl2.x, r2max);
    acc[1] = r2.y < fminf(rl2.y, r2max);
    inside[0] = r2.x < hp2.x;
    inside[1] = r2.y < hp2.y;
  }
  // largest axis separation (view units) a listed pair can reach before the next rebuild
  template <int D>
  __device__ __forceinline__ float reach(const Frame<float>& F, const int4& vi, const int4& vj) const {
    const int d = max(max(abs(vi.x - vj.x), abs(vi.y - vj.y)), D == 3 ? abs(vi.z - vj.z) : 0);
    return ((float)d + di + build_reach(F, vj)) * F.vscale;
  }
  // the coarse FP32 conversion is exact below 2^22 coarse integers = 2^(22 - kCoarseBits) c0
  static __device__ __forceinline__ bool fast(float reach) { return reach < 0.999f * (1 << (22 - kCoarseBits)); }
};
// the rows of level-l cells a search ball of radius Rs reaches
template <int D>
struct RowWalk {
  using T = float;
  int nx, ny, nz, cxl, cyl, czl, zlo, zhi, ylo, yhi;
  uint32_t base;
  T c, ic, fx, fy, fz;  // cell edge, position inside the own cell, view units
  __device__ __forceinline__ RowWalk(const Frame<T>& F, const Grid<T>& G, const LL4& X, T Rs, int l) {
    const int sh = G.cshift + l;
    nx = G.nx[l];
    ny = G.ny[l];
    nz = G.nz[l];
    base = G.base[l];
    cxl = (int)min((long long)nx - 1, X.x >> sh);
    cyl = (int)min((long long)ny - 1, X.y >> sh);
    czl = D == 3 ? (int)min((long long)nz - 1, X.z >> sh) : 0;
    c = G.cellv[l];
    ic = T(1) / c;
    fx = (T)((double)(X.x - ((long long)cxl << sh)) * F.s2v);
    fy = (T)((double)(X.y - ((long long)cyl << sh)) * F.s2v);
    fz = D == 3 ? (T)((double)(X.z - ((long long)czl << sh)) * F.s2v) : T(0);
    zlo = D == 3 ? (int)dfloor((fz - Rs) * ic) : 0;
    zhi = D == 3 ? (int)dfloor((fz + Rs) * ic) : 0;
    ylo = (int)dfloor((fy - Rs) * ic);
    yhi = (int)dfloor((fy + Rs) * ic);
  }
  // candidates [j, je) of row (dz, dy), trimmed to the ball; false: none
  __device__ __forceinline__ bool row(const uint32_t* __restrict__ cstart, int dz, int dy, T R2, int& j, int& je) const {
    const int czz = czl + dz, cyy = cyl + dy;
    if ((D == 3 && (czz < 0 || czz >= nz)) || cyy < 0 || cyy >= ny) return false;
    T dzp = 0;
    if (D == 3) {
      const T zrel = fz - (T)dz * c;
      dzp = zrel < T(0) ? -zrel : (zrel > c ? zrel - c : T(0));
    }
    const T yrel = fy - (T)dy * c;
    const T dyp = yrel < T(0) ? -yrel : (yrel > c ? yrel - c : T(0));
    const T dp2 = dyp * dyp + dzp * dzp;
    if (dp2 >= R2) return false;
    const T half = dsqrt(R2 - dp2);
    int x0 = cxl + (int)dfloor((fx - half) * ic), x1 = cxl + (int)dfloor((fx + half) * ic);
    x0 = x0 < 0 ? 0 : x0;
    x1 = x1 > nx - 1 ? nx - 1 : x1;
    if (x0 > x1) return false;
    const uint32_t krow = base + (uint32_t)nx * ((uint32_t)cyy + (uint32_t)ny * (uint32_t)(D == 3 ? czz : 0));
    j = (int)cstart[krow + (uint32_t)x0];
    je = (int)cstart[krow + (uint32_t)x1 + 1];
    return true;
  }
};

// What a walk over the candidates found: entries accepted (cnt), written inside
// and outside, the largest axis separation (REACH).
struct ListCount {
  int cnt, n_in, n_out;
  float reach;
};
// One thread's list. REACH: certify the coarse FP32 test (kFastBit, read by the
// FP64 path).
template <int D, bool REACH, bool CUT>
__device__ __forceinline__ ListCount walk_list(const Frame<float>& F, const Grid<float>& G, float kappa, int dmax,
                                               const LL4& X, const int4& vi, const int4* __restrict__ view,
                                               const uint32_t* __restrict__ meta,
                                               const uint32_t* __restrict__ cstart, int cap,
                                               uint32_t* __restrict__ own) {
  const ListTarget<CUT> t(F, G, kappa, dmax, vi);
  const int rows = list_rows(cap);
  ListCount c{0, 0, 0, 0.0f};
  // only the list store is conditional: most candidates fail, and a branch
  // over the tests ran for a few lanes of the warp in nearly every iteration.
  // Bound by issue slots (lanes of a warp have different rows and row lengths:
  // 11 of 32 active); two candidates per instruction, with the lengths of the
  // tests relative to w, take 31 % off a rebuild (8,388,608 particles in 3D:
  // 1.48 -> 1.03 ms per step at a rebuild every four steps).
  auto take = [&](int j, const int4& vj, bool acc, bool inside) {
    if (!acc) return;
    if (c.cnt < cap) {
      const int row = inside ? c.n_in++ : rows - 1 - c.n_out++;
      own[(size_t)(row >> 2) * 128 + (row & 3)] = ((uint32_t)j << 8) | (meta[j] & 0xFFu);
    }
    ++c.cnt;
    if (REACH) c.reach = fmaxf(c.reach, t.template reach<D>(F, vi, vj));
  };
  for (int l = t.l0; l <= t.l1; ++l) {
    const RowWalk<D> w(F, G, X, t.Rs, l);
    for (int dz = w.zlo; dz <= w.zhi; ++dz) {
      for (int dy = w.ylo; dy <= w.yhi; ++dy) {
        int j, je;
        if (!w.row(cstart, dz, dy, t.R2, j, je)) continue;
        // candidates in ascending order, two at a time (an odd last one twice)
        for (; j < je; j += 2) {
          const bool two = j + 1 < je;
          const int4 a = view[j], b = view[two ? j + 1 : j];
          bool acc[2], inside[2];
          t.template test<D>(vi, a, b, acc, inside);
          take(j, a, acc[0], inside[0]);
          take(j + 1, b, acc[1] && two, inside[1]);
        }
      }
    }
  }
  return c;
}
// The same list made by a group of G lanes: lane g walks candidate rows g,
// g + G, ... and the group's lanes test one candidate each at a time; accepted
// ones take their places in lane order. cnt, n_in, n_out: uniform over the group.
template <int D, int G, bool REACH, bool CUT>
__device__ __forceinline__ ListCount walk_list_group(const Frame<float>& F, const Grid<float>& G32, float kappa,
                                                     int dmax, const LL4& X, const int4& vi,
                                                     const int4* __restrict__ view,
                                                     const uint32_t* __restrict__ meta,
                                                     const uint32_t* __restrict__ cstart, int cap,
                                                     uint32_t* __restrict__ own) {
  const unsigned group = group_mask<G>(), below = group & lanes_below();
  const ListTarget<CUT> t(F, G32, kappa, dmax, vi);
  const int rows = list_rows(cap);
  ListCount c{0, 0, 0, 0.0f};
  for (int l = t.l0; l <= t.l1; ++l) {
    const RowWalk<D> w(F, G32, X, t.Rs, l);
    const int ny = w.yhi - w.ylo + 1, nr = ny * (w.zhi - w.zlo + 1);
    for (int r = threadIdx.x % G; __any_sync(group, r < nr); r += G) {
      int j = 0, je = 0;
      if (r < nr) w.row(cstart, w.zlo + r / ny, w.ylo + r % ny, t.R2, j, je);
      for (; __any_sync(group, j < je); j += 2) {
        bool acc[2] = {false, false}, inside[2] = {false, false};
        if (j < je) {
          const bool two = j + 1 < je;
          const int4 a = view[j], b = view[two ? j + 1 : j];
          t.template test<D>(vi, a, b, acc, inside);
          acc[1] = acc[1] && two;
          if (REACH && acc[0]) c.reach = fmaxf(c.reach, t.template reach<D>(F, vi, a));
          if (REACH && acc[1]) c.reach = fmaxf(c.reach, t.template reach<D>(F, vi, b));
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          unsigned all = __ballot_sync(group, acc[q]), in = __ballot_sync(group, acc[q] && inside[q]);
          c.cnt += __popc(all);
          if (c.cnt > cap) {  // a full list keeps the first of them
            for (int room = cap - c.n_in - c.n_out; __popc(all) > room;) all &= ~(1u << (31 - __clz(all)));
            in &= all;
          }
          if (all >> (threadIdx.x & 31) & 1u) {
            const int row = inside[q] ? c.n_in + __popc(in & below) : rows - 1 - (c.n_out + __popc(all & ~in & below));
            own[(size_t)(row >> 2) * 128 + (row & 3)] = ((uint32_t)(j + q) << 8) | (meta[j + q] & 0xFFu);
          }
          c.n_in += __popc(in);
          c.n_out += __popc(all & ~in);
        }
      }
    }
  }
  for (int o = 1; o < G; o <<= 1) c.reach = fmaxf(c.reach, __shfl_xor_sync(group, c.reach, o));
  return c;
}
__device__ __forceinline__ uint32_t list_counts(const ListCount& c, bool reach) {
  return (uint32_t)c.n_in | ((uint32_t)c.n_out << kOutShift) |
         (reach && ListTarget<false>::fast(c.reach) ? kFastBit : 0u);
}
// A list that did not fit, again at the common reach (G: lanes that make it). A
// function of its own, called last and with nothing but the kernel's parameters:
// it hardly ever runs, and neither its registers nor its arguments take any from
// the walk.
template <int D, int G, bool REACH>
__device__ __noinline__ void cut_list(StepCtl* ctl, const LL4* X0, const LL4* X1, const uint32_t* m0,
                                      const uint32_t* m1, const int4* view, const uint32_t* cstart,
                                      const Frame<float>& F, const Grid<float>& Gr, float kappa, int cap,
                                      uint32_t* list, uint32_t* lcount, int* err) {
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) / G, buf = ctl->buf;
  const uint32_t* meta = buf ? m1 : m0;
  const LL4 X = (buf ? X1 : X0)[i];
  uint32_t* own = list + list_at(i, 0, cap);
  ListCount c;
  if constexpr (G == 1) c = walk_list<D, REACH, true>(F, Gr, kappa, ctl->dmax, X, view[i], view, meta, cstart, cap, own);
  else c = walk_list_group<D, G, REACH, true>(F, Gr, kappa, ctl->dmax, X, view[i], view, meta, cstart, cap, own);
  if (threadIdx.x % G != 0) return;
  lcount[i] = list_counts(c, REACH);
  atomicMin(&ctl->reach_cap, F.code_u);
  atomicMax(&ctl->lmax, c.cnt);
  if (c.cnt > cap) atomicOr(err, kErrListOverflow);
}

// One thread per particle.
template <int D, bool REACH>
__global__ void __launch_bounds__(256, SPH_LIST_MIN_BLOCKS) k_list_build(
    int n, StepCtl* __restrict__ ctl, const LL4* __restrict__ X0, const LL4* __restrict__ X1,
    const uint32_t* __restrict__ m0, const uint32_t* __restrict__ m1, const int4* __restrict__ view,
    const uint32_t* __restrict__ cstart, const __grid_constant__ Frame<float> F,
    const __grid_constant__ Grid<float> G, float kappa, int cap, uint32_t* __restrict__ list,
    uint32_t* __restrict__ lcount, int* __restrict__ err) {
  after_predecessor();
  if (!ctl->rebuild) return;
  const int buf = ctl->buf;
  const uint32_t* __restrict__ meta = buf ? m1 : m0;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  int cnt = 0;
  if (i < n) {
    const LL4 X = (buf ? X1 : X0)[i];
    const ListCount c = walk_list<D, REACH, false>(F, G, kappa, ctl->dmax, X, view[i], view, meta, cstart, cap,
                                                   list + list_at(i, 0, cap));
    lcount[i] = list_counts(c, REACH);
    cnt = c.cnt;
  }
  // longest list of this build (one atomic per warp; every lane gets here)
  const int wmax = __reduce_max_sync(0xffffffffu, cnt <= cap ? cnt : 0);
  if ((threadIdx.x & 31) == 0 && wmax > 0) atomicMax(&ctl->lmax, wmax);
  if (cnt > cap) cut_list<D, 1, REACH>(ctl, X0, X1, m0, m1, view, cstart, F, G, kappa, cap, list, lcount, err);
}

// G lanes per particle: for particle counts that leave most of the chip idle with
// one thread per particle, where one thread's chain of row look-ups and candidate
// loads is the whole time (launch_rebuild).
template <int D, int G, bool REACH>
__global__ void __launch_bounds__(256) k_list_build_group(
    int n, StepCtl* __restrict__ ctl, const LL4* __restrict__ X0, const LL4* __restrict__ X1,
    const uint32_t* __restrict__ m0, const uint32_t* __restrict__ m1, const int4* __restrict__ view,
    const uint32_t* __restrict__ cstart, const __grid_constant__ Frame<float> F,
    const __grid_constant__ Grid<float> G32, float kappa, int cap, uint32_t* __restrict__ list,
    uint32_t* __restrict__ lcount, int* __restrict__ err) {
  __shared__ int longest;
  after_predecessor();
  if (!ctl->rebuild) return;
  if (threadIdx.x == 0) longest = 0;
  __syncthreads();
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) / G;
  int cnt = 0;
  if (i < n) {  // whole groups
    const int buf = ctl->buf;
    const uint32_t* __restrict__ meta = buf ? m1 : m0;
    const LL4 X = (buf ? X1 : X0)[i];
    const ListCount c = walk_list_group<D, G, REACH, false>(F, G32, kappa, ctl->dmax, X, view[i], view, meta, cstart,
                                                            cap, list + list_at(i, 0, cap));
    cnt = c.cnt;
    if (threadIdx.x % G == 0) {
      lcount[i] = list_counts(c, REACH);
      if (cnt <= cap) atomicMax(&longest, cnt);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 && longest > 0) atomicMax(&ctl->lmax, longest);
  if (cnt > cap) cut_list<D, G, REACH>(ctl, X0, X1, m0, m1, view, cstart, F, G32, kappa, cap, list, lcount, err);
}

// Staged pass A, set up at a list rebuild: one block per kStageBlock targets
// (the blocks of pass A). The distinct neighbours j of the block's lists go
// into a hash set in shared memory (linear probing); the occupied slots in slot
// order number them (rank), sj[block][rank] = j and scount[block] = their
// count; every list entry is written again into llist as (rank << 8 | colour),
// with kStageSelf for j = i. A block with more than kStageCap neighbours, or a
// set too crowded to probe, gets scount = -1: pass A gathers its views from
// global memory. The ranks depend on the order of the hash inserts, but pass
// A's sums follow the list order, so its results do not.
constexpr int kStageHashBits = 12;
static_assert((1 << kStageHashBits) == kStageHash, "hash set size");
constexpr int kStageProbe = 64;
__device__ __forceinline__ uint32_t stage_hash(int j) { return ((uint32_t)j * 2654435761u) >> (32 - kStageHashBits); }

template <int D>
__global__ void __launch_bounds__(kStageBlock) k_stage(int n, const StepCtl* __restrict__ ctl,
                                                      const uint32_t* __restrict__ list,
                                                      const uint32_t* __restrict__ lcount, int cap,
                                                      uint32_t* __restrict__ llist, int* __restrict__ scount,
                                                      int* __restrict__ sj) {
  after_predecessor();
  if (!ctl->rebuild) return;
  __shared__ int tab[kStageHash];
  __shared__ int rnk[kStageHash];
  __shared__ int wsum[kStageBlock / 32];
  __shared__ int bad;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  for (int q = t; q < kStageHash; q += kStageBlock) tab[q] = -1;
  if (t == 0) bad = 0;
  __syncthreads();
  const int i = blockIdx.x * kStageBlock + t;
  const uint32_t lc = i < n ? lcount[i] : 0u;
  const int cnt = list_cnt(lc), n_in = list_in(lc);
  for (int k = 0; k < cnt; ++k) {
    const int j = (int)(list[list_at(i, list_row(k, n_in, cap), cap)] >> 8);
    uint32_t q = stage_hash(j);
    int p = 0;
    for (; p < kStageProbe; ++p) {
      const int old = atomicCAS(&tab[q], -1, j);
      if (old == -1 || old == j) break;
      q = (q + 1) & (kStageHash - 1);
    }
    if (p == kStageProbe) bad = 1;
  }
  __syncthreads();
  const bool crowded = bad != 0;
  // ranks: thread t owns slots [per t, per (t + 1)); exclusive scan of the counts
  constexpr int per = kStageHash / kStageBlock;
  int c = 0;
  for (int q = 0; q < per; ++q) c += tab[t * per + q] >= 0;
  int x = c;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[w] = x;
  __syncthreads();
  int r = x - c, m = 0;
  for (int q = 0; q < kStageBlock / 32; ++q) {
    r += q < w ? wsum[q] : 0;
    m += wsum[q];
  }
  if (crowded || m > kStageCap) {
    if (t == 0) scount[blockIdx.x] = -1;
    return;
  }
  int* __restrict__ sjb = sj + (size_t)blockIdx.x * kStageCap;
  for (int q = 0; q < per; ++q) {
    const int slot = t * per + q;
    const int j = tab[slot];
    if (j >= 0) {
      rnk[slot] = r;
      sjb[r] = j;
      ++r;
    }
  }
  __syncthreads();
  for (int k = 0; k < cnt; ++k) {
    const size_t pos = list_at(i, list_row(k, n_in, cap), cap);
    const uint32_t e = list[pos];
    const int j = (int)(e >> 8);
    uint32_t q = stage_hash(j);
    for (int p = 0; p < kStageProbe && tab[q] != j; ++p) q = (q + 1) & (kStageHash - 1);
    llist[pos] = ((uint32_t)rnk[q] << 8) | (e & 0xFFu) | (j == i ? kStageSelf : 0u);
  }
  if (t == 0) scount[blockIdx.x] = m;
}

// --------------------------------------------------------------------------
// Density pass (general gamma): rho_i (Eq. density_sum) and p_i / rho_i^2 with
// p = P0 (rho/rho_t)^gamma (Eq. EOS_current), needed by the neighbours' forces.
// --------------------------------------------------------------------------
template <int D, class T>
__global__ void __launch_bounds__(256) k_density(int n, const StepCtl* __restrict__ ctl,
                                                 const typename ViewOf<T>::type* __restrict__ v0,
                                                 const typename ViewOf<T>::type* __restrict__ v1,
                                                 const uint32_t* __restrict__ list,
                                                 const uint32_t* __restrict__ lcount, int cap, Frame<T> F,
                                                 Phys<T> P, T* __restrict__ rho_out, T* __restrict__ pc_out) {
  using VT = typename ViewOf<T>::type;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const VT* __restrict__ view = ctl->vp ? v1 : v0;
  const VT vi = view[i];
  const T hv = view_h(F, vi);
  const T Hd = P.kappa * hv, Hd2 = Hd * Hd, invHd = T(1) / Hd;
  const uint32_t lc = lcount[i];
  T acc = 0;
  if constexpr (std::is_same<T, float>::value) {  // two entries at a time, as pass A
    const float2 id2 = both(-0.5f / (F.hk_int * view_w(vi))), one2 = both(1.0f);
    float2 ds2 = both(0.0f), dq2 = both(0.0f);
    auto two = [&](uint32_t, const VT& a, uint32_t, const VT& b, auto on0, auto on1) {
      const float2 dx = make_float2((float)(vi.x - a.x), (float)(vi.x - b.x));
      const float2 dy = make_float2((float)(vi.y - a.y), (float)(vi.y - b.y));
      float2 r2 = fma2(dy, dy, mul2(dx, dx));
      if (D == 3) {
        const float2 dz = make_float2((float)(vi.z - a.z), (float)(vi.z - b.z));
        r2 = fma2(dz, dz, r2);
      }
      r2 = make_float2(fmaxf(r2.x, 1.0f), fmaxf(r2.y, 1.0f));
      if (!on0) r2.x = 1e30f;
      if (!on1) r2.y = 1e30f;
      const float2 r = mul2(r2, rsqrt2(r2)), q = mul2(r, id2), u = max2(add2(q, one2), 0.0f), u2 = mul2(u, u), u4 = mul2(u2, u2);
      ds2 = add2(ds2, u4);
      dq2 = fma2(u4, q, dq2);
    };
    auto load = [&](uint32_t e) -> VT { return view[e >> 8]; };
    for_twos(list, i, lc, cap, (uint32_t)i << 8, load, two);
    acc = (ds2.x + ds2.y) - 4.0f * (dq2.x + dq2.y);
  } else {
    for_skin_list(list, view, i, lc, cap, [&](uint32_t, const VT& vj) {
      const T dx = vd(F, vi.x, vj.x), dy = vd(F, vi.y, vj.y);
      const T dz = D == 3 ? vd(F, vi.z, vj.z) : T(0);
      const T r2 = dx * dx + dy * dy + dz * dz;
      if (!(r2 < Hd2)) return;
      const T q = r2 > T(0) ? pair_r<T>(r2) * invHd : T(0);
      const T u = T(1) - q, u2 = u * u;
      acc += u2 * u2 * (T(1) + T(4) * q);
    });
  }
  const T Hphys = Hd * F.qv;
  const T rho = acc * P.alpha / (D == 2 ? Hphys * Hphys : Hphys * Hphys * Hphys);
  const T irt2 = inv_rho_t2<D, T>(hv * F.qv, P.inv_tau);
  const T rt = T(1) / dsqrt(irt2);
  rho_out[i] = rho;
  pc_out[i] = P.P0 * (T)pow((double)(rho / rt), (double)P.gamma) / (rho * rho);
}

// The end of pass A, called by warp 0 of every block with the block's partial in
// lane 0: the grid's total, the step sizes, the statistics, the schedule. A
// function of its own: inlined, its registers spilled into the pair loop.
template <class T>
__device__ __noinline__ void finish_step(Partial part, Partial* partials, unsigned* ticket, StepCtl* ctl,
                                         Scalars* scal, int advance, const double* __restrict__ dt_fix,
                                         double* __restrict__ dt_rec) {
  if (!grid_total<T>(part, partials, ticket)) return;
  if ((threadIdx.x & 31) == 0) {
    const Partial& acc = part;
    const StepCtl cc = *ctl;  
    const long long step = cc.step;
    // Eq. time_step_size with v_n = 0 (the velocity reset of Algorithm 1): the
    // first time step keeps only the body-force term, dt1 = min_i 0.25
    // sqrt(r_c,i/|a_i|). With v~_i = a_i dt1/2 and nu_i = 0.1 r_c,i |v~_i|, the
    // second time step's terms are
    // r_c/(40|v~|) = m/(20 dt1) and 0.125 r_c^2/nu = 2.5 m/dt1, m = min r_c/|a|
    // (all three are monotone in r_c,i/|a_i|, so their minima share the argmin).
    constexpr bool f32 = std::is_same<T, float>::value;
    const double m = !f32 ? acc.min_rc_a : acc.amin >= 0 ? (double)acc.rc / (double)acc.an : DBL_MAX;
    double dt1 = 0.0, dt2 = 0.0;
    if (m < DBL_MAX) {
      dt1 = 0.25 * sqrt(m);
      dt2 = fmin(dt1, fmin(m / (20.0 * dt1), 2.5 * m / dt1));
    }
    if (dt_fix) {  // prescribed step sizes
      dt1 = dt_fix[0];
      dt2 = dt_fix[1];
    }
    if (dt_rec) {
      dt_rec[0] = dt1;
      dt_rec[1] = dt2;
    }
    // the step-size history of a reverse-pass run: replay or record
    const long long hk = step - cc.dt_base;
    if (cc.dt_mode && cc.dt_hist && hk >= 0 && hk < cc.dt_len) {
      if (cc.dt_mode == 2) {
        dt1 = cc.dt_hist[2 * hk];
        dt2 = cc.dt_hist[2 * hk + 1];
      } else {
        cc.dt_hist[2 * hk] = dt1;
        cc.dt_hist[2 * hk + 1] = dt2;
      }
    }
    scal->dt1 = dt1;
    scal->dt2 = dt2;
    scal->min_rc_a = m;
    scal->argmin = acc.amin;
    scal->max_a = f32 ? (double)acc.ma : acc.max_a;
    scal->sum_rho = acc.sum_rho;
    scal->err_l2 = acc.err_l2;
    scal->err_max = f32 ? fmax(err_exact(acc.er, acc.et), 0.0) : acc.err_max;
    scal->sigma = (double)(T)sigma_of(cc, step);
    scal->ipairs = acc.ipairs / 2;
    scal->fpairs = acc.fpairs / 2;
    scal->lentries = acc.lentries;
    scal->wall_moved = 0;
    scal->step_of_stats = step;
    if (advance && cc.auto_on && !cc.auto_done) {
      // convergence of the partition (Sec. 3.3): the interface-pair count stays
      // within auto_tol of the count that opened the run for auto_window steps;
      // then the ramp of Eq. sph_st_sigma starts: t0 = this step, t1 = (1 + theta) t0
      const long long ip = acc.ipairs / 2;
      long long ref = cc.auto_ref;
      int stable = cc.auto_stable;
      if (ref >= 0 && fabs((double)(ip - ref)) <= cc.auto_tol * (double)ref) {
        ++stable;
      } else {
        ref = ip;
        stable = 0;
      }
      ctl->auto_ref = ref;
      ctl->auto_stable = stable;
      if (stable >= cc.auto_window) {
        ctl->t0 = (double)step;
        ctl->t1 = (1.0 + cc.auto_theta) * (double)step;
        ctl->auto_done = 1;
      }
    }
    if (advance) ctl->step = step + 1;
  }
}

// --------------------------------------------------------------------------
// Pass A (Algorithm 1: velocity reset, forces, first time step): per target i,
// over its listed j
//   rho_i = sum_j W(r_ij, h_i)                                 (Eq. density_sum)
//   a_i   = -sum_j [(P_i + P_j) + beta_ij P0 (1/rho_t,i^2 + 1/rho_t,j^2)]
//                  dW(r_ij, h_ij)/dr e_ij                      (Eqs. sph_pressure_force_2,
//                                                                   sph_st_force, sph_st_beta)
// with P = P0/rho_t^2 at gamma = 2 (Eq. EOS_2) or p/rho^2 otherwise;
// e_ij = (r_i - r_j)/r_ij, h_ij = (h_i + h_j)/2, and for the Wendland C2 kernel
// of support H: dW/dr e_ij = -20 alpha (1 - q)^3 (r_i - r_j) / H^(D+2).
// Writes a_i and g_i = 0.05 rho_t,i r_c,i |a_i| (eta_i = dt1 g_i, Eq.
// viscosity_coefficient with v~ = a dt1 / 2), the force pairs for pass B, and
// block partials (FP32: fixed-point sums and the particles of the extrema,
// WarpSums; FP64: values) of min r_c/|a|, max |a|, sum rho, sum (rho/rho_t - 1)^2,
// max |rho/rho_t - 1|, pair counts; the last block reduces them in fixed order and
// sets dt1, dt2 (Eq. time_step_size, see finish_step).
// --------------------------------------------------------------------------
template <int D, class T, bool GENERAL, bool DBG, bool SURF, int NT, bool STG = false, int G = 1>
__global__ void __launch_bounds__(NT, (sizeof(T) == 8 ? SPH_PASS_MIN_BLOCKS_FP64 : SPH_PASS_MIN_BLOCKS) * 256 / NT) k_pass_a(int n, StepCtl* ctl,
                                                const typename ViewOf<T>::type* __restrict__ v0,
                                                const typename ViewOf<T>::type* __restrict__ v1,
                                                const uint32_t* __restrict__ m0, const uint32_t* __restrict__ m1,
                                                const uint32_t* __restrict__ p0, const uint32_t* __restrict__ p1,
                                                const uint32_t* __restrict__ list,
                                                const uint32_t* __restrict__ lcount, int cap, Frame<T> F,
                                                Phys<T> P, const T* __restrict__ pc, V4<T>* __restrict__ acc_out,
                                                T* __restrict__ rho_out, Partial* __restrict__ partials,
                                                Scalars* __restrict__ scal, unsigned* __restrict__ ticket,
                                                int* __restrict__ err, int advance, int* __restrict__ dbg_count,
                                                long long* __restrict__ dbg_sum, PairRec<T>* __restrict__ plist,
                                                uint32_t* __restrict__ pcount, const double* __restrict__ dt_fix,
                                                double* __restrict__ dt_rec, const LL4* __restrict__ X0,
                                                const LL4* __restrict__ X1, Geom<T> geo,
                                                const uint32_t* __restrict__ llist, const int* __restrict__ scount,
                                                const int* __restrict__ sj, const int4* __restrict__ v32,
                                                Frame<float> F32) {
  using VT = typename ViewOf<T>::type;
  static_assert(!STG || (std::is_same<T, float>::value && !GENERAL && !DBG && !SURF && NT == kStageBlock),
                "staged pass A: FP32, gamma = 2, 256-target blocks");
  constexpr bool PACKED = std::is_same<T, float>::value && !DBG && !SURF;
  static_assert(G == 1 || (sizeof(T) == 8 && !DBG && !SURF && NT == 32 * G),
                "several lanes per particle: FP64, 32 particles per block");
  extern __shared__ __align__(16) unsigned char stage_smem[];
  // G lanes per particle (pass_a_shape): all of a warp's lanes stay together in
  // the loop, those past the end with an empty list; warp 0 holds the block's 32
  // particles afterwards
  const int slot = (blockIdx.x * NT + threadIdx.x) / G;
  int i = G == 1 ? slot : min(slot, n - 1);
  bool lead = slot < n;
  const int buf = ctl->buf;
  const VT* __restrict__ view = ctl->vp ? v1 : v0;
  const T sigma = (T)sigma_of(*ctl, ctl->step);
  Partial part = no_partial();
  float own_rc = 0, own_an = 0, own_rho = 0, own_rt = 0;  // FP32 path: this particle's share of the reductions
  int own_ni = 0, own_nf = 0, own_cnt = 0;
  // staged block: this step's views of its neighbour set into shared memory
  bool staged = false;
  const int* __restrict__ sjb = nullptr;
  VT* sview = reinterpret_cast<VT*>(stage_smem);
  if constexpr (STG) {
    const int m = min(scount[blockIdx.x], kStageCap);
    staged = m >= 0;
    if (staged) {
      sjb = sj + (size_t)blockIdx.x * kStageCap;
      for (int k = threadIdx.x; k < m; k += NT) cp_async16(sview + k, view + min(__ldg(sjb + k), n - 1));
      cp_async_wait_all();
    }
    __syncthreads();
  }
  if (G > 1 || i < n) {
    const uint32_t* __restrict__ pid = buf ? p1 : p0;
    const VT vi = view[i];
    const uint32_t* __restrict__ meta = buf ? m1 : m0;
    const uint32_t mi = meta[i];
    const uint32_t ci = mi & 0xFFu;
    // a feature-surface particle (Sec. 3.5) takes forces from surface particles
    // only (SURF: the variant launched when the handle has any)
    const bool surf = SURF && (mi & kSurfaceBit) != 0;
    T hv = view_h(F, vi);
    const T qv = F.qv;
    T Hd = P.kappa * hv;
    const T Hd2 = Hd * Hd, invHd = T(1) / Hd;
    const T inv_tau_v = P.inv_tau * qv;     // h in view units -> (h/tau)
    T qi = inv_rho_t2<D, T>(hv, inv_tau_v);  // 1/rho_t,i^2
    const T Pi = GENERAL ? pc[i] : P.P0 * qi;
    const T sP0 = sigma * P.P0;
    [[maybe_unused]] const T half_kappa = T(0.5) * P.kappa;
    T dsum = 0, ax = 0, ay = 0, az = 0;
    int nf = 0, ni = 0, nd = 0;
    long long sd = 0, sf = 0;
    const uint32_t lc = lead ? lcount[i] : 0u;
    int cnt = list_cnt(lc);
    PairRec<T>* __restrict__ pw = plist + pair_at(i, 0, cap);  // this step's force pairs, for pass B
    // FP32: the listed entries two at a time, every FP32 operation on both at
    // once, on exact differences throughout (a coarse screen first saved the
    // conversions but evaluated the passing two thirds twice). The kernel's
    // factors 1 - r/H are clamped at zero, so a pair outside a support adds
    // nothing and needs no test; only an iteration in which neither entry is
    // inside is skipped. What bounds it: the latency of the view gathers (issue
    // slots 51 % busy, L1 data pipe 56 %). With the reductions above, at
    // 1,048,576 particles: 304 -> 231 us in 3D (249 -> 144 million warp
    // instructions), 216 -> 114 us in 2D; 8,388,608 in 3D 1.50 ms. 64 registers
    // (four 256-thread blocks per SM): an earlier form at 48 spilled (2.30 ms
    // against 1.59), at 80 too few warps hid the gathers (1.84 ms).
    if constexpr (PACKED) {
      // distances and supports H = kappa (h_i + h_j) / 2 in view integers, powers of
      // h and of H in view units; what all pairs have in common (pair_scale, P0)
      // comes in once, after the sum. A pair's terms round alike for both its ends,
      // so that the forces of a pair cancel exactly: with powers relative to the
      // target's h they did not, and after 8 steps of 20,011 particles in 2D the
      // gradients by positions were off by 6.3e-7 instead of 5.7e-7, that by sigma0 by
      // 2.7e-7 instead of 1.7e-7 (means over 80 starts; in 3D 5.3e-7 and 2.3e-7).
      const float wi = F.hk_int * view_w(vi);  // kappa h_i / 2
      const float2 h2 = both(view_w(vi)), id2 = both(-0.5f / wi), one2 = both(1.0f), unit2 = both((float)(1 << kViewBits));
      const auto power = [](float2 h) {  // h^(2 D), rounded before it enters a sum
        const float2 t2 = mul2(h, h), t4 = mul2_apart(t2, t2);
        return D == 2 ? t4 : mul2_apart(t4, t2);
      };
      const float2 qi2 = power(h2);
      const float hd2 = 4.0f * wi * wi;  // (kappa h_i)^2
      const float common = inv_rho_t2<D, float>(1.0f, inv_tau_v);  // (h / tau)^(2 D) from h in view units
      const float sq = GENERAL ? sP0 * common : 1.0f + sigma;
      const uint32_t own = ((uint32_t)i << 8) | ci;
      uint32_t counts = 0;  // force pairs, of them other colours << 16
      float dq = 0.0f;
      float2 ax2 = both(0.0f), ay2 = both(0.0f), az2 = both(0.0f);
      auto sums = [&](auto stagedc) {
        constexpr bool ST = decltype(stagedc)::value;  // e = (rank << 8 | colour), view from shared memory
        auto load = [&](uint32_t e) -> VT { return ST ? sview[stage_rank(e)] : view[e >> 8]; };
        auto two = [&](uint32_t e0, const VT& v0, uint32_t e1, const VT& v1, auto on0, auto on1) {
          const float2 dx = make_float2((float)(vi.x - v0.x), (float)(vi.x - v1.x));
          const float2 dy = make_float2((float)(vi.y - v0.y), (float)(vi.y - v1.y));
          float2 r2 = fma2(dy, dy, mul2(dx, dx)), dz = both(0.0f);
          if (D == 3) {
            dz = make_float2((float)(vi.z - v0.z), (float)(vi.z - v1.z));
            r2 = fma2(dz, dz, r2);
          }
          r2 = make_float2(fmaxf(r2.x, 1.0f), fmaxf(r2.y, 1.0f));  // 1 for the particle itself: r = 2^-24 c0, dx = 0
          if (!on0) r2.x = 1e30f;
          if (!on1) r2.y = 1e30f;
          const float2 hj = make_float2(view_w(v0), view_w(v1));
          const float2 S = add2(h2, hj), H = make_float2(F.hk_int * S.x, F.hk_int * S.y), H2 = mul2(H, H);
          const bool f0 = r2.x < H2.x, f1 = r2.y < H2.y;
          if (!(f0 || f1 || (!GENERAL && (r2.x < hd2 || r2.y < hd2)))) return;
          const float2 r = mul2(r2, rsqrt2(r2));
          if (!GENERAL) {  // W ~ (1 - q)^4 (1 + 4 q); q = 1 - u where u > 0
            const float2 u = max2(fma2(r, id2, one2), 0.0f), u2 = mul2(u, u), u4 = mul2(u2, u2);
            const float2 m = mul2(u4, mul2(r, id2));
            dsum += u4.x + u4.y;
            dq += m.x + m.y;
          }
          const float2 nH = rcp2(make_float2(-H.x, -H.y));
          const float2 u = max2(fma2(r, nH, one2), 0.0f), g = mul2(nH, unit2), g2 = mul2(g, g), g4 = mul2(g2, g2);
          const float2 w = mul2(mul2(mul2(u, u), u), D == 2 ? g4 : mul2(g4, g));  // 3D: negative (g < 0)
          const float2 ts = add2_apart(qi2, power(hj));  // 1 / rho_t,i^2 + 1 / rho_t,j^2 over `common`
          const bool o0 = ((e0 ^ own) & 0xFFu) != 0, o1 = ((e1 ^ own) & 0xFFu) != 0;
          const float2 tw = mul2(ts, w);
          float2 s;
          if (GENERAL) {
            const float2 pp = make_float2(pc[e0 >> 8], pc[e1 >> 8]);
            s = mul2(fma2(make_float2(o0 ? sq : 0.0f, o1 ? sq : 0.0f), ts, add2(both(Pi), pp)), w);
          } else {
            s = mul2(tw, make_float2(o0 ? sq : 1.0f, o1 ? sq : 1.0f));
          }
          ax2 = fma2(s, dx, ax2);
          ay2 = fma2(s, dy, ay2);
          if (D == 3) az2 = fma2(s, dz, az2);
          auto push = [&](uint32_t e, bool inside, bool other, float f) {
            if (inside && !(ST ? (e & kStageSelf) != 0 : e == own)) {
              store_pair(pw, ST ? ((uint32_t)__ldg(sjb + stage_rank(e)) << 8) | (e & 0xFFu) : e, f);
              pw += 32;
              counts += other ? 0x10001u : 1u;  // at most 2^15 - 1 pairs
            }
          };
          push(e0, f0, o0, tw.x);
          push(e1, f1, o1, tw.y);
        };
        for_twos(ST ? llist : list, i, lc, cap, ST ? ci | kStageSelf : own, load, two);
      };
      if (STG && staged) sums(std::integral_constant<bool, STG>{});
      else sums(std::false_type{});
      dsum -= 4.0f * dq;  // dq holds the terms in -q
      nf = counts & 0xFFFFu;
      ni = counts >> 16;
      const float back = F.vscale * pair_scale<D>(GENERAL ? 1.0f : P.P0 * common);
      ax = (ax2.x + ax2.y) * back;
      ay = (ay2.x + ay2.y) * back;
      az = (az2.x + az2.y) * back;
    } else {
    // FP64, feature surfaces, diagnostics: one entry at a time, the exact
    // criteria on every entry (FP64 path with current FP32 views: on those that
    // pass a screen in FP32, for_skin_list_s32)
    constexpr bool S32_OK = std::is_same<T, double>::value && !GENERAL && !DBG && !SURF;
    // G > 1: the pairs of the group's lanes one after another, in lane order
    auto push_all = [&](bool have, uint32_t e, bool other, T f) {
      const unsigned m = __ballot_sync(0xffffffffu, have) & group_mask<G>();
      if (have) {
        store_pair(pw + 32 * __popc(m & lanes_below()), e, f);
        ni += other;
      }
      pw += 32 * __popc(m);
      nf += __popc(m);
    };
    const T iscale = T(1) / pair_scale<D>(inv_rho_t2<D, T>(T(1), inv_tau_v));
    bool have = false, have_other = false;  // G > 1: what the lane's entry adds to the group's pairs
    T have_f = 0;
    auto pair = [&](uint32_t e, const VT& vj) {
      const int j = (int)(e >> 8);
      const T dx = vd(F, vi.x, vj.x), dy = vd(F, vi.y, vj.y);
      const T dz = D == 3 ? vd(F, vi.z, vj.z) : T(0);
      const T hj = view_h(F, vj);
      T r2, Hf;
      bool inD, inF;
      if constexpr (std::is_same<T, float>::value) {
        // the tests of the packed path, rounding for rounding (there in view
        // integers: a power of two apart), so that diagnostics name its pairs
        const float w = F.half_kappa * hv, H = F.half_kappa * (hv + hj);
        r2 = fmaf(dy, dy, __fmul_rn(dx, dx));
        if (D == 3) r2 = fmaf(dz, dz, r2);
        Hf = H;
        inD = r2 < __fmul_rn(4.0f * w, w);
        inF = r2 < __fmul_rn(H, H);
      } else {
        r2 = dx * dx + dy * dy + dz * dz;
        Hf = half_kappa * (hv + hj);
        inD = r2 < Hd2;
        inF = r2 < Hf * Hf;
      }
      inD = inD && !GENERAL;
      inF = inF && j != i && (!surf || (meta[j] & kSurfaceBit));
      if (!(inD || inF)) return;
      const T r = r2 > T(0) ? pair_r<T>(r2) : T(0);
      if (inD) {
        const T q = r * invHd;
        const T u = T(1) - q, u2 = u * u;
        dsum += u2 * u2 * (T(1) + T(4) * q);
        if (DBG) {
          ++nd;
          sd += pid[j];
        }
      }
      if (inF) {
        const T invH = drcp<T>(Hf);
        const T q = r * invH;
        const T u = T(1) - q;
        const T invH2 = invH * invH;
        const T w = u * u * u * (D == 2 ? invH2 * invH2 : invH2 * invH2 * invH);
        const T qj = inv_rho_t2<D, T>(hj, inv_tau_v);
        const T Pj = GENERAL ? pc[j] : P.P0 * qj;
        const bool other = (e & 0xFFu) != ci;
        const T coef = (Pi + Pj) + (other ? sP0 * (qi + qj) : T(0));
        const T s = coef * w;
        ax += s * dx;
        ay += s * dy;
        az += s * dz;
        if (G == 1) {
          store_pair(pw, e, (qi + qj) * w * iscale);
          pw += 32;
          ++nf;
          ni += other;
        } else {
          have = true;
          have_other = other;
          have_f = (qi + qj) * w * iscale;
        }
        if (DBG) sf += pid[j];
      }
    };
    if constexpr (G > 1) {
      // lane g of the group takes entries g, g + G, ...
      const int n_in = list_in(lc);
      for (int k = threadIdx.x % G; __any_sync(0xffffffffu, k < cnt); k += G) {
        have = false;
        uint32_t e = 0;
        if (k < cnt) {
          e = list[list_at(i, list_row(k, n_in, cap), cap)];
          pair(e, view[e >> 8]);
        }
        push_all(have, e, have_other, have_f);
      }
      dsum = group_sum<G>(dsum);
      ax = group_sum<G>(ax);
      ay = group_sum<G>(ay);
      az = group_sum<G>(az);
    } else if (S32_OK && v32 && (lc & kFastBit)) {
      const int4 wi = v32[i];
      const float ws = F32.half_kappa, wi32 = ws * view_w(wi), Hd32 = 2.0f * wi32;  // view units
      auto screen = [&](const int4& w) {
        const float cx = vd_coarse(F32, wi.x, w.x), cy = vd_coarse(F32, wi.y, w.y);
        const float cz = D == 3 ? vd_coarse(F32, wi.z, w.z) : 0.0f;
        const float Hf32 = fmaf(ws, view_w(w), wi32);
        const float Hm = screen_radius<float>(Hf32 > Hd32 ? Hf32 : Hd32);
        return cx * cx + cy * cy + cz * cz < Hm * Hm;
      };
      for_skin_list_s32(list, v32, view, i, lc, cap, screen, pair);
    } else {
      for_skin_list(list, view, i, lc, cap, pair);
    }
    }
    if constexpr (G > 1) {
      // the 32 particles of the block to the lanes of warp 0: what follows
      // costs a warp as much for one particle as for 32
      __shared__ T sums[4][32];
      __shared__ int counted[3][32];
      ni = group_sum<G>(ni);
      const int t = threadIdx.x / G;
      if (threadIdx.x % G == 0) {
        sums[0][t] = dsum;
        sums[1][t] = ax;
        sums[2][t] = ay;
        sums[3][t] = az;
        counted[0][t] = nf;
        counted[1][t] = ni;
        counted[2][t] = cnt;
      }
      __syncthreads();
      if (threadIdx.x >= 32) return;
      dsum = sums[0][threadIdx.x];
      ax = sums[1][threadIdx.x];
      ay = sums[2][threadIdx.x];
      az = sums[3][threadIdx.x];
      nf = counted[0][threadIdx.x];
      ni = counted[1][threadIdx.x];
      cnt = counted[2][threadIdx.x];
      i = blockIdx.x * 32 + threadIdx.x;
      lead = i < n;
      i = min(i, n - 1);
    }
    // the target's lengths again (of another target where G > 1): kept over the
    // loop they cost registers that spill
    hv = view_h(F, view[i]);
    Hd = P.kappa * hv;
    qi = inv_rho_t2<D, T>(hv, P.inv_tau * qv);
    if (G == 1) cnt = list_cnt(lcount[i]);
    if (lead) pcount[i] = (uint32_t)nf;
    // back to physical units: rho ~ 1/H^D, a ~ (view length)^-(D+1)
    const T Hphys = Hd * qv;
    const T rho = GENERAL ? rho_out[i] : dsum * P.alpha / (D == 2 ? Hphys * Hphys : Hphys * Hphys * Hphys);
    const T iq = F.inv_qv;
    const T k20 = T(20) * P.alpha * (D == 2 ? iq * iq * iq : iq * iq * iq * iq);
    ax *= k20;
    ay *= k20;
    az *= k20;
    if (surf) {  // Eq. force_surface: the normal component is dropped
      T xa[3], N[3];
      abs_pos<D, T>(F, (buf ? X1 : X0)[i], xa);
      surface_normal(geo, xa, D, N);
      const T dn = ax * N[0] + ay * N[1] + az * N[2];
      ax -= dn * N[0];
      ay -= dn * N[1];
      az -= dn * N[2];
    }
    const T an = dsqrt(ax * ax + ay * ay + az * az);
    const T rt = T(1) / dsqrt(qi);
    const T rc = Hphys;
    const T g = T(0.05) * rt * rc * an;
    if (lead) acc_out[i] = V4<T>{ax, ay, az, g};
    if (!GENERAL && rho_out && lead) rho_out[i] = rho;
    if constexpr (std::is_same<T, float>::value) {
      own_rc = rc;
      own_an = an;
      own_rho = rho;
      own_rt = rt;
      own_ni = lead ? ni : 0;
      own_nf = lead ? nf : 0;
      own_cnt = lead ? cnt : 0;
    } else {
      const double e = (double)rho / (double)rt - 1.0;
      if (lead) {
        part.min_rc_a = an > T(0) ? (double)rc / (double)an : DBL_MAX;
        part.amin = an > T(0) ? (long long)i : -1;
        part.max_a = (double)an;
        part.sum_rho = (double)rho;
        part.err_l2 = e * e;
        part.err_max = fabs(e);
        part.ipairs = ni;
        part.fpairs = nf;
        part.lentries = cnt;
      }
    }
    if (lead && !(isfinite(an) && isfinite(rho))) atomicOr(err, kErrNonfinite);
    if (DBG) {
      const uint32_t id = pid[i];
      dbg_count[2 * id] = nd;
      dbg_count[2 * id + 1] = nf;
      dbg_sum[2 * id] = sd;
      dbg_sum[2 * id + 1] = sf;
    }
  }
  // the block's partial in warp 0 (the other warps are done), then the grid's
  constexpr int NW = G > 1 ? 1 : NT / 32;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if constexpr (std::is_same<T, float>::value) {
    __shared__ WarpSums ws[NW];
    warp_sums(lead, i, own_rc, own_an, own_rho, own_rt, own_ni, own_nf, own_cnt, ws + warp);
    if (NW > 1) {
      __syncthreads();
      if (warp != 0) return;
    } else {
      __syncwarp();
    }
    part = lane < NW ? to_partial(ws[lane]) : no_partial();
    if (NW > 1) part = warp_total<T>(part);
  } else {
    part = warp_total<T>(part);
    if constexpr (NW > 1) {
      __shared__ Partial sm[NW];
      if (lane == 0) sm[warp] = part;
      __syncthreads();
      if (warp != 0) return;
      part = warp_total<T>(lane < NW ? sm[lane] : no_partial());
    }
  }
  finish_step<T>(part, partials, ticket, ctl, scal, advance, dt_fix, dt_rec);
}

// --------------------------------------------------------------------------
// Pass B (Algorithm 1: viscous force, kicks, drift, projection): viscous force (Eq. sph_viscous_force with
// rho := rho_t, Eq. sph_viscous_force_2), the kicks and the drift
// (Eqs. time_int_01..03) and the level-set projection (Eq. displacement_surface).
// With v~ = a dt1/2 and eta = dt1 g:
//   a~_i = (dt1^2 / 2) B_i,
//   B_i  = sum_j HM(g_i, g_j) (1/rho_t,i^2 + 1/rho_t,j^2) (dW/dr / r)(a_i - a_j),
//   v_i  = dt1 a_i / 2 + dt2 a~_i / 2,   r_i += v_i dt2.
// The new view goes to the other view buffer; a particle that moved its
// reach since the list was built raises need_rebuild.
// Bound by the gather of the neighbour's acceleration, one per force pair: the
// pair's geometry factor comes from pass A's record (8,388,608 particles in 3D,
// FP32: 1.40 -> 0.74 ms with 128-thread blocks; 300,007 in FP64: 1.40 -> 0.43).
// TAPE: a step of the reverse pass's tape also keeps the pairs' list words (a
// kernel of its own that took them out of the records added 13 us to a step of
// 262,144 particles in 2D).
// --------------------------------------------------------------------------
template <int D, class T, int NT, int G = 1, bool TAPE = false>
__global__ void __launch_bounds__(NT, (sizeof(T) == 8 ? SPH_PASSB_MIN_BLOCKS_FP64 : SPH_PASSB_MIN_BLOCKS) * 256 / NT) k_pass_b(int n, StepCtl* __restrict__ ctl,
                                                const typename ViewOf<T>::type* __restrict__ v0,
                                                const typename ViewOf<T>::type* __restrict__ v1,
                                                typename ViewOf<T>::type* __restrict__ w0,
                                                typename ViewOf<T>::type* __restrict__ w1,
                                                const typename ViewOf<T>::type* __restrict__ vbuild,
                                                LL4* __restrict__ X0, LL4* __restrict__ X1,
                                                const PairRec<T>* __restrict__ plist,
                                                const uint32_t* __restrict__ pcount, int cap,
                                                const V4<T>* __restrict__ acc, Frame<T> F, Phys<T> P, Geom<T> geo,
                                                const Scalars* __restrict__ scal, V4<T>* __restrict__ visc_out,
                                                int* __restrict__ err, unsigned long long* __restrict__ wall_moved,
                                                int move, const uint32_t* __restrict__ m0,
                                                const uint32_t* __restrict__ m1, int4* __restrict__ v32out,
                                                int sv32, uint32_t* __restrict__ words) {
  using VT = typename ViewOf<T>::type;
  __shared__ int moved_sm[NT / 32];
  // G lanes per particle, as pass A
  static_assert(G == 1 || NT == 32 * G, "several lanes per particle: 32 particles per block");
  const int slot = (blockIdx.x * NT + threadIdx.x) / G;
  int i = G == 1 ? slot : min(slot, n - 1);
  bool lead = slot < n;
  const int vp = ctl->vp, buf = ctl->buf;
  int moved = 0, far = 0;
  if (G > 1 || i < n) {
    const VT* __restrict__ view = vp ? v1 : v0;
    V4<T> ai = acc[i];
    T bx = 0, by = 0, bz = 0;
    // this step's pairs as pass A left them: the geometry in a factor per pair,
    // so only the neighbour's acceleration is gathered and no distance, root or
    // kernel value is computed again. FP32, 8,388,608 particles in 3D: 1.40 ->
    // 0.74 ms, and pass A, which writes the factor, 0.06 ms longer; FP64, where the
    // FP64 pipe bounds both passes, 300,007 in 3D: 1.40 -> 0.43 ms.
    const int cnt = lead ? (int)pcount[i] : 0;
    const PairRec<T>* __restrict__ p = plist + pair_at(i, 0, cap);
    // TAPE: after the gathers of the same pairs are on their way, so that it waits
    // for nothing of its own
    const auto keep = [&](const PairRec<T>* q, const PairRec<T>& r) {
      if (TAPE) __stcs(words + (q - plist), r.e);
    };
    if constexpr (std::is_same<T, float>::value) {
      // two pairs per instruction; sums of (a_j - a_i), factor gi gj / (gi + gj)
      const float2 g2 = both(ai.w), nx2 = both(-ai.x), ny2 = both(-ai.y), nz2 = both(-ai.z);
      float2 bx2 = both(0.0f), by2 = both(0.0f), bz2 = both(0.0f);
      auto two = [&](const PairRec<T>& r0, const V4<T>& a0, const PairRec<T>& r1, const V4<T>& a1) {
        const float2 gj = make_float2(a0.w, a1.w);
        float2 gs = add2(g2, gj);
        gs = make_float2(fmaxf(gs.x, 1e-37f), fmaxf(gs.y, 1e-37f));  // both zero: 0 / 1e-37
        const float2 s = mul2(mul2(mul2(g2, rcp2(gs)), gj), make_float2(r0.f, r1.f));
        bx2 = fma2(s, add2(make_float2(a0.x, a1.x), nx2), bx2);
        by2 = fma2(s, add2(make_float2(a0.y, a1.y), ny2), by2);
        if (D == 3) bz2 = fma2(s, add2(make_float2(a0.z, a1.z), nz2), bz2);
      };
      constexpr int B = SPH_PASSB_BATCH;
      int k = 0;
      if constexpr (G > 1) {
        for (k = 2 * (threadIdx.x % G), p += 32 * k; k < cnt; k += 2 * G, p += 64 * G) {
          const PairRec<T> r0 = load_pair(p);
          PairRec<T> r1{r0.e, 0.0f};
          if (k + 1 < cnt) r1 = load_pair(p + 32);
          const V4<T> a0 = acc[r0.e >> 8], a1 = acc[r1.e >> 8];
          keep(p, r0);
          if (k + 1 < cnt) keep(p + 32, r1);
          two(r0, a0, r1, a1);
        }
        __syncwarp();
      } else {
      PairRec<T> ahead[B];
      if (cnt >= B)
#pragma unroll
        for (int q = 0; q < B; ++q) ahead[q] = load_pair(p + 32 * q);
      for (; k + B <= cnt; k += B) {
        PairRec<T> r[B];
        V4<T> a[B];
#pragma unroll
        for (int q = 0; q < B; ++q) r[q] = ahead[q];
#pragma unroll
        for (int q = 0; q < B; ++q) a[q] = acc[r[q].e >> 8];
        p += 32 * B;
        if (k + 2 * B <= cnt)
#pragma unroll
          for (int q = 0; q < B; ++q) ahead[q] = load_pair(p + 32 * q);
        if (TAPE)
#pragma unroll
          for (int q = 0; q < B; ++q) keep(p + 32 * q - 32 * B, r[q]);
#pragma unroll
        for (int q = 0; q < B; q += 2) two(r[q], a[q], r[q + 1], a[q + 1]);
      }
#pragma unroll 1
      for (; k < cnt; k += 2, p += 64) {
        const PairRec<T> r0 = load_pair(p);
        PairRec<T> r1{r0.e, 0.0f};  // no second pair: a zero factor
        if (k + 1 < cnt) r1 = load_pair(p + 32);
        const V4<T> a0 = acc[r0.e >> 8], a1 = acc[r1.e >> 8];
        keep(p, r0);
        if (k + 1 < cnt) keep(p + 32, r1);
        two(r0, a0, r1, a1);
      }
      }
      bx = -2.0f * (bx2.x + bx2.y);
      by = -2.0f * (by2.x + by2.y);
      bz = -2.0f * (bz2.x + bz2.y);
    } else {
      auto pair = [&](const PairRec<T>& r, const V4<T>& aj) {
        const T gs = ai.w + aj.w;
        const T s = gs > T(0) ? T(2) * ai.w * aj.w * drcp<T>(gs) * r.f : T(0);
        bx += s * (ai.x - aj.x);
        by += s * (ai.y - aj.y);
        bz += s * (ai.z - aj.z);
      };
      int k = 0;
      if constexpr (G > 1) {
        for (k = threadIdx.x % G, p += 32 * k; k < cnt; k += G, p += 32 * G) {
          const PairRec<T> r0 = load_pair(p);
          const V4<T> a0 = acc[r0.e >> 8];
          keep(p, r0);
          pair(r0, a0);
        }
        __syncwarp();
      }
      for (; k < cnt; k += 2, p += 64) {  // a zero factor where there is no second pair
        const PairRec<T> r0 = load_pair(p);
        PairRec<T> r1{T(0), r0.e, 0u};
        if (k + 1 < cnt) r1 = load_pair(p + 32);
        const V4<T> a0 = acc[r0.e >> 8], a1 = acc[r1.e >> 8];
        keep(p, r0);
        if (k + 1 < cnt) keep(p + 32, r1);
        pair(r0, a0);
        if (k + 1 < cnt) pair(r1, a1);
      }
    }
    if constexpr (G > 1) {  // the block's 32 particles to warp 0
      __shared__ T sums[3][32];
      bx = group_sum<G>(bx);
      by = group_sum<G>(by);
      bz = group_sum<G>(bz);
      if (threadIdx.x % G == 0) {
        sums[0][threadIdx.x / G] = bx;
        sums[1][threadIdx.x / G] = by;
        sums[2][threadIdx.x / G] = bz;
      }
      __syncthreads();
      i = blockIdx.x * 32 + threadIdx.x;
      lead = threadIdx.x < 32 && i < n;
      i = min(i, n - 1);
      bx = sums[0][threadIdx.x & 31];
      by = sums[1][threadIdx.x & 31];
      bz = sums[2][threadIdx.x & 31];
      ai = acc[i];
    }
    if (G == 1 || threadIdx.x < 32) {
    const VT vi = view[i];
    const T hv = view_h(F, vi);
    // dW/dr / r = -20 alpha (1-q)^3 / H^(D+2); view lengths -> physical
    const T iq = F.inv_qv;
    const T km = T(-20) * P.alpha * (D == 2 ? iq * iq * iq * iq : iq * iq * iq * iq * iq) *
                 pair_scale<D>(inv_rho_t2<D, T>(T(1), P.inv_tau * F.qv));
    bx *= km;
    by *= km;
    bz *= km;
    const bool surf = ((buf ? m1 : m0)[i] & kSurfaceBit) != 0;
    if (surf) {  // Eq. force_surface for the viscous force too
      T xs[3], N[3];
      abs_pos<D, T>(F, (buf ? X1 : X0)[i], xs);
      surface_normal(geo, xs, D, N);
      const T dn = bx * N[0] + by * N[1] + bz * N[2];
      bx -= dn * N[0];
      by -= dn * N[1];
      bz -= dn * N[2];
    }
    const T dt1 = (T)scal->dt1, dt2 = (T)scal->dt2;
    const T kv = T(0.5) * dt1 * dt1;  // a~ = kv B
    // a~ for the caller when asked (a run-time test: one compiled kernel, so
    // recording cannot change the arithmetic of the step)
    if (visc_out && lead) visc_out[i] = V4<T>{kv * bx, kv * by, kv * bz, T(0)};
    if (move && lead) {
    T d[3];
    d[0] = (T(0.5) * dt1 * ai.x + T(0.5) * dt2 * kv * bx) * dt2;
    d[1] = (T(0.5) * dt1 * ai.y + T(0.5) * dt2 * kv * by) * dt2;
    d[2] = D == 3 ? (T(0.5) * dt1 * ai.z + T(0.5) * dt2 * kv * bz) * dt2 : T(0);
    LL4* __restrict__ Xs = buf ? X1 : X0;
    LL4 X = Xs[i];
    const bool finite = isfinite(d[0]) && isfinite(d[1]) && isfinite(d[2]);
    if (!finite) atomicOr(err, kErrNonfinite);
    if (finite) {
      long long* Xc[3] = {&X.x, &X.y, &X.z};
      for (int k = 0; k < D; ++k) {
        long long v = *Xc[k] + state_units(d[k] * F.inv_q64t);
        // bounding box (first constraint): clamp, the closest point
        if (v < 0) { v = 0; moved |= !surf; }
        if (v > F.xmax[k]) { v = F.xmax[k]; moved |= !surf; }
        *Xc[k] = v;
      }
      // shape constraints, in order, at the absolute position; a feature-surface
      // particle goes onto the surface it belongs to instead (Eq. displacement_surface)
      T xa[3];
      abs_pos<D, T>(F, X, xa);
      int mv = 0;
      if (surf) {
        project_to_surface(geo, xa, D);
        mv = 1;
      } else {
        for (int s = 0; s < geo.n_shapes; ++s) mv |= project_shape(geo, s, xa, D);
        moved |= mv;
      }
      if (mv) {
        for (int k = 0; k < D; ++k) {
          long long v = state_units((xa[k] - F.lo[k]) * F.inv_q64t);
          v = v < 0 ? 0 : (v > F.xmax[k] ? F.xmax[k] : v);
          *Xc[k] = v;
        }
        abs_pos<D, T>(F, X, xa);
      }
      // the move in units of kappa h, for the next list's reach (never zero: that
      // would mean none yet)
      const float mx = (float)d[0], my = (float)d[1], mz = (float)d[2];
      X.w = (long long)__float_as_uint(
          fmaxf(sqrtf(mx * mx + my * my + mz * mz) / (float)(P.kappa * hv * F.qv), 1e-30f));
      Xs[i] = X;
      // smoothing length at the new position (the target field of the next step)
      const T hn = h_of<D, T>(geo, xa);
      const VT vn = make_view<D>(F, X, hn);
      (vp ? w0 : w1)[i] = vn;
      if (v32out) {  // FP64 path: its FP32 view of the next step (as k_gather_view makes it)
        const long long half = 1LL << (sv32 - 1);
        v32out[i] = make_int4((int)((X.x + half) >> sv32), (int)((X.y + half) >> sv32),
                              D == 3 ? (int)((X.z + half) >> sv32) : 0, __float_as_int((float)view_w(vn)));
      }
      // skin test against the view at list build
      const VT vb = vbuild[i];
      const T ex = vd(F, vn.x, vb.x), ey = vd(F, vn.y, vb.y);
      const T ez = D == 3 ? vd(F, vn.z, vb.z) : T(0);
      T lim;  // the reach, view units
      const int most = ctl->reach_cap;
      if constexpr (std::is_same<T, float>::value) lim = build_reach(F, vb, most) * F.vscale;
      else lim = coded_reach(vb.w, most);
      far = (ex * ex + ey * ey + ez * ez) >= lim * lim;
    } else {
      (vp ? w0 : w1)[i] = vi;
    }
    }  // move
    }
  }
  if (__syncthreads_or(far) && threadIdx.x == 0) ctl->need_rebuild = 1;
  int v = moved;
  for (int s = 16; s > 0; s >>= 1) v += __shfl_xor_sync(0xffffffffu, v, s);
  if ((threadIdx.x & 31) == 0) moved_sm[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += moved_sm[w];
    if (t) atomicAdd(wall_moved, (unsigned long long)t);
  }
}

// --------------------------------------------------------------------------
// State in / out
// --------------------------------------------------------------------------
template <int D, class T>
__global__ void __launch_bounds__(256) k_set_state(int n, const double* __restrict__ xyz,
                                                   const uint8_t* __restrict__ col, Frame<T> F,
                                                   LL4* __restrict__ X0, uint32_t* __restrict__ meta0,
                                                   uint32_t* __restrict__ pid0, int* __restrict__ err) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  long long v[3] = {0, 0, 0};
  for (int k = 0; k < D; ++k) {
    const double x = xyz[(size_t)i * D + k];
    if (!isfinite(x)) {
      atomicOr(err, kErrNonfinite);
      continue;
    }
    const double u = (x - F.lod[k]) * F.inv_q64;
    if (u < 0.0 || u > (double)F.xmax[k] + 0.5) atomicOr(err, kErrOutOfDomain);
    long long w = (long long)llrint(u < 0.0 ? 0.0 : (u > (double)F.xmax[k] ? (double)F.xmax[k] : u));
    v[k] = w;
  }
  X0[i] = LL4{v[0], v[1], v[2], 0};
  meta0[i] = (uint32_t)col[i];
  pid0[i] = (uint32_t)i;
}

template <int D, class T>
__global__ void __launch_bounds__(256) k_get_positions(int n, const StepCtl* __restrict__ ctl,
                                                       const LL4* __restrict__ X0, const LL4* __restrict__ X1,
                                                       const uint32_t* __restrict__ p0,
                                                       const uint32_t* __restrict__ p1, Frame<T> F,
                                                       double* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int buf = ctl->buf;
  const LL4 X = (buf ? X1 : X0)[i];
  const uint32_t id = (buf ? p1 : p0)[i];
  out[(size_t)id * D + 0] = F.lod[0] + (double)X.x * F.q64;
  out[(size_t)id * D + 1] = F.lod[1] + (double)X.y * F.q64;
  if (D == 3) out[(size_t)id * D + 2] = F.lod[2] + (double)X.z * F.q64;
}

// which: 0 rho (n), 1 acc (n x D), 2 visc (n x D); source arrays in the current order
template <int D, class T>
__global__ void __launch_bounds__(256) k_get_fields(int n, int which, const StepCtl* __restrict__ ctl,
                                                    const uint32_t* __restrict__ p0,
                                                    const uint32_t* __restrict__ p1, const T* __restrict__ rho,
                                                    const V4<T>* __restrict__ acc, const V4<T>* __restrict__ visc,
                                                    double* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint32_t id = (ctl->buf ? p1 : p0)[i];
  if (which == 0) {
    out[id] = (double)rho[i];
    return;
  }
  const V4<T> v = which == 1 ? acc[i] : visc[i];
  out[(size_t)id * D + 0] = (double)v.x;
  out[(size_t)id * D + 1] = (double)v.y;
  if (D == 3) out[(size_t)id * D + 2] = (double)v.z;
}

// --------------------------------------------------------------------------
// Launchers
// --------------------------------------------------------------------------
inline int grid_for(int n, int tb) { return (n + tb - 1) / tb; }

template <int D, class T>
cudaError_t launch_rebuild(const DevState& S, int force, const Grid<T>& G, const Frame<T>& F, const Geom<T>& g,
                           T kappa, cudaStream_t st, const Grid<float>* G32, const Frame<float>* F32) {
  using VT = typename ViewOf<T>::type;
  // the cheap per-particle kernels on a capped grid (an idle launch costs a
  // few us); the list build on one block per 256 targets: a grid capped at
  // 16 or 32 blocks per SM made its rebuilds of the 8M 3D workload slower
  // (cells 2.01 / 1.93 vs 1.86 ms per step), its blocks no longer finishing
  // and refilling the SMs independently
  const int tb = 256, gb = rebuild_grid(S.n, tb, 8);
  const LL4* X0 = (const LL4*)S.X[0];
  const LL4* X1 = (const LL4*)S.X[1];
  k_rekey<D, T><<<gb, tb, 0, st>>>(S.n, S.ctl, force, S.tickets + 1, X0, X1, F, G, g, S.key, S.cnt, S.scan_part);
  cudaError_t e = build_cells(S, st);
  if (e != cudaSuccess) return e;
  // the FP64 path lists its pairs through an FP32 view (same frame origin, same
  // cells, same list format)
  if (std::is_same<T, double>::value && (!S.view32 || !F32 || !G32)) return cudaErrorInvalidValue;
  launch_after(k_gather_view<D, T>, gb, tb, 0, st, S.n, S.ctl, S.tmp, S.key, S.cstart, (LL4*)S.X[0], (LL4*)S.X[1], S.meta[0],
                                         S.meta[1], S.pid[0], S.pid[1], F, g, (VT*)S.view[0], (VT*)S.view[1],
                                         (VT*)S.vbuild, (int4*)S.view32, F32 ? *F32 : Frame<float>{});
  constexpr bool f64 = std::is_same<T, double>::value;
  const Frame<float>* Fl = F32;
  const Grid<float>* Gl = G32;
  const int4* view = (const int4*)(f64 ? S.view32 : S.vbuild);
  if constexpr (!f64) {
    Fl = &F;
    Gl = &G;
  }
  const bool group = S.n <= kListGroupMax;
  auto build = [&](auto* kernel, int blocks) {
    launch_after(kernel, blocks, tb, 0, st, S.n, S.ctl, X0, X1, S.meta[0], S.meta[1], view, S.cstart, *Fl, *Gl,
                 (float)kappa, S.cap, S.list, S.lcount, S.err);
  };
  if (group) build(k_list_build_group<D, kListLanes, f64>, grid_for(S.n * kListLanes, tb));
  else build(k_list_build<D, f64>, grid_for(S.n, tb));
  if constexpr (!f64) {
    if (S.stage && S.llist)
      launch_after(k_stage<D>, grid_for(S.n, kStageBlock), kStageBlock, 0, st, S.n, S.ctl, S.list, S.lcount, S.cap, S.llist,
                                                                  S.scount, S.sj);
  }
  return cudaGetLastError();
}

template <int D, class T>
cudaError_t launch_pass_a(const DevState& S, const Frame<T>& F, const Phys<T>& P, PassFlags f, cudaStream_t st) {
  using VT = typename ViewOf<T>::type;
  Geom<T> geo{};
  if (f.geo) geo = *(const Geom<T>*)f.geo;
  T* rho = (T*)S.rho;
  T* pc = (T*)S.pc;
  // the FP64 path screens on its FP32 views when the caller passes their frame
  const bool s32 = std::is_same<T, double>::value && S.view32 && f.f32;
  const int4* v32 = s32 ? (const int4*)S.view32 : nullptr;
  const Frame<float> f32 = s32 ? *f.f32 : Frame<float>{};
  auto run = [&](auto* kernel, int threads, int lanes, size_t smem) {
    kernel<<<grid_for(S.n * lanes, threads), threads, smem, st>>>(
        S.n, S.ctl, (const VT*)S.view[0], (const VT*)S.view[1], S.meta[0], S.meta[1], S.pid[0], S.pid[1], S.list, S.lcount, S.cap, F, P, pc, (V4<T>*)S.acc4, rho, S.partials, S.scal, S.tickets, S.err, f.advance, S.dbg_count,
        S.dbg_sum, (PairRec<T>*)S.plist, S.pcount, f.dt_fix, f.dt_rec, (const LL4*)S.X[0], (const LL4*)S.X[1], geo,
        S.llist, S.scount, S.sj, v32, f32);
    return cudaGetLastError();
  };
  const auto density = [&](auto* kernel, int threads) {
    kernel<<<grid_for(S.n, threads), threads, 0, st>>>(S.n, S.ctl, (const VT*)S.view[0], (const VT*)S.view[1], S.list,
                                                       S.lcount, S.cap, F, P, rho, pc);
  };
  // one of the compiled variants at one block size (the diagnostics at one only)
  auto pick = [&](auto nt) -> cudaError_t {
    constexpr int NT = decltype(nt)::value;
    if (f.general_eos)
      return run(f.surface ? k_pass_a<D, T, true, false, true, NT> : k_pass_a<D, T, true, false, false, NT>, NT, 1, 0);
    return run(f.surface ? k_pass_a<D, T, false, false, true, NT> : k_pass_a<D, T, false, false, false, NT>, NT, 1, 0);
  };
  auto diagnose = [&](auto nt) -> cudaError_t {
    constexpr int NT = decltype(nt)::value;
    if (f.general_eos)
      return run(f.surface ? k_pass_a<D, T, true, true, true, NT> : k_pass_a<D, T, true, true, false, NT>, NT, 1, 0);
    return run(f.surface ? k_pass_a<D, T, false, true, true, NT> : k_pass_a<D, T, false, true, false, NT>, NT, 1, 0);
  };
  constexpr bool f64 = std::is_same<T, double>::value;
  if (f.general_eos) density(k_density<D, T>, f64 ? fp64_threads(S.n) : 256);
  if (f.nbr_debug) return diagnose(std::integral_constant<int, f64 ? 64 : 256>{});
  const PassShape shape = pass_a_shape(S, !f.surface);
  if constexpr (f64) {
    if (shape.lanes > 1)
      return f.general_eos ? run(k_pass_a<D, T, true, false, false, 32 * kLanes64, false, kLanes64>, shape.threads, kLanes64, 0)
                           : run(k_pass_a<D, T, false, false, false, 32 * kLanes64, false, kLanes64>, shape.threads, kLanes64, 0);
    if (shape.threads == 32) return pick(std::integral_constant<int, 32>{});
    if (shape.threads == 64) return pick(std::integral_constant<int, 64>{});
  } else if (staged_pass(S, f)) {
    return run(k_pass_a<D, T, false, false, false, kStageBlock, true>, kStageBlock, 1, kStageCap * sizeof(int4));
  }
  if (shape.threads == 128) return pick(std::integral_constant<int, 128>{});
  return pick(std::integral_constant<int, 256>{});
}

template <int D>
cudaError_t prepare_staged_pass() {
  static cudaError_t e = cudaFuncSetAttribute(k_pass_a<D, float, false, false, false, kStageBlock, true>,
                                              cudaFuncAttributePreferredSharedMemoryCarveout,
                                              (int)cudaSharedmemCarveoutMaxShared);
  return e;
}

template <int D, class T>
cudaError_t launch_pass_b(const DevState& S, const Frame<T>& F, const Phys<T>& P, const Geom<T>& g, PassFlags f,
                          cudaStream_t st) {
  using VT = typename ViewOf<T>::type;
  unsigned long long* wm = (unsigned long long*)&S.scal->wall_moved;
  auto run = [&](auto* kernel, int threads, int lanes) {
    kernel<<<grid_for(S.n * lanes, threads), threads, 0, st>>>(
        S.n, S.ctl, (const VT*)S.view[0], (const VT*)S.view[1], (VT*)S.view[0], (VT*)S.view[1], (const VT*)S.vbuild,
        (LL4*)S.X[0], (LL4*)S.X[1], (const PairRec<T>*)S.plist, S.pcount, S.cap, (const V4<T>*)S.acc4, F, P, g, S.scal,
        f.record ? (V4<T>*)S.visc : nullptr, S.err, wm, f.move, S.meta[0], S.meta[1],
        (std::is_same<T, double>::value && S.view32 && f.f32) ? (int4*)S.view32 : nullptr, f.f32 ? f.f32->sv : 0,
        f.words);
    return cudaGetLastError();
  };
  // threads per block and lanes per particle, taped or not
  auto pick = [&](auto nt, auto lanes) {
    constexpr int NT = decltype(nt)::value, G = decltype(lanes)::value;
    return f.words ? run(k_pass_b<D, T, NT, G, true>, NT, G) : run(k_pass_b<D, T, NT, G>, NT, G);
  };
  using one = std::integral_constant<int, 1>;
  const PassShape shape = pass_b_shape(S);
  if constexpr (std::is_same<T, float>::value) {
    if (shape.lanes > 1)
      return pick(std::integral_constant<int, 32 * kPassLanes>{}, std::integral_constant<int, kPassLanes>{});
  } else {
    if (shape.lanes > 1) return pick(std::integral_constant<int, 32 * kLanes64>{}, std::integral_constant<int, kLanes64>{});
    if (shape.threads == 32) return pick(std::integral_constant<int, 32>{}, one{});
    if (shape.threads == 64) return pick(std::integral_constant<int, 64>{}, one{});
  }
  if (shape.threads == 128) return pick(std::integral_constant<int, 128>{}, one{});
  return pick(std::integral_constant<int, 256>{}, one{});
}

template <int D, class T>
cudaError_t launch_set_state(const DevState& S, const Frame<T>& F, const double* xyz, const uint8_t* col,
                             cudaStream_t st) {
  const int tb = 256, gb = grid_for(S.n, tb);
  if (S.n > 0)
    k_set_state<D, T><<<gb, tb, 0, st>>>(S.n, xyz, col, F, (LL4*)S.X[0], S.meta[0], S.pid[0], S.err);
  return cudaGetLastError();
}

template <int D, class T>
cudaError_t launch_get_positions(const DevState& S, const Frame<T>& F, double* out, cudaStream_t st) {
  const int tb = 256, gb = grid_for(S.n, tb);
  if (S.n > 0)
    k_get_positions<D, T><<<gb, tb, 0, st>>>(S.n, S.ctl, (const LL4*)S.X[0], (const LL4*)S.X[1], S.pid[0],
                                             S.pid[1], F, out);
  return cudaGetLastError();
}

template <int D, class T>
cudaError_t launch_get_fields(const DevState& S, int which, double* out, cudaStream_t st) {
  const int tb = 256, gb = grid_for(S.n, tb);
  if (S.n > 0)
    k_get_fields<D, T><<<gb, tb, 0, st>>>(S.n, which, S.ctl, S.pid[0], S.pid[1], (const T*)S.rho,
                                          (const V4<T>*)S.acc4, (const V4<T>*)S.visc, out);
  return cudaGetLastError();
}

#define SPH_INSTANTIATE_STEP(D, T)                                                                             \
  template cudaError_t launch_rebuild<D, T>(const DevState&, int, const Grid<T>&, const Frame<T>&,            \
                                            const Geom<T>&, T, cudaStream_t, const Grid<float>*,              \
                                            const Frame<float>*);                                             \
  template cudaError_t launch_pass_a<D, T>(const DevState&, const Frame<T>&, const Phys<T>&, PassFlags,       \
                                           cudaStream_t);                                                     \
  template cudaError_t launch_pass_b<D, T>(const DevState&, const Frame<T>&, const Phys<T>&, const Geom<T>&,  \
                                           PassFlags, cudaStream_t);                                          \
  template cudaError_t launch_set_state<D, T>(const DevState&, const Frame<T>&, const double*, const uint8_t*, \
                                              cudaStream_t);                                                  \
  template cudaError_t launch_get_positions<D, T>(const DevState&, const Frame<T>&, double*, cudaStream_t);   \
  template cudaError_t launch_get_fields<D, T>(const DevState&, int, double*, cudaStream_t);

}  // namespace sph
