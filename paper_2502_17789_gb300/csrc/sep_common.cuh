// Shared device code of the separable-phasor gridder and degridder
// (gridder_sep_kernels.cuh, degridder_sep_kernels.cuh).
//
// The phase of Eq. 7 over a subgrid, phi_k(i,j) = a_k i' + b_k j' + w_k n'(i,j)
// (turns; i' = i - L/2, j' = j - L/2), is separable but for the w term, and
// that term nearly so.  With w_ref the middle of the subgrid's w range,
// delta_k = w_k - w_ref, |delta_k| <= x, and the fit n'(i,j) = A_i + B_j + p_i q_j
// + r_ij (sep_fit, SepTables),
//   e^{2 pi i phi_k} = P(i,j) E_k(i) F_k(j) (1 + 2 pi i delta_k p_i q_j) + O(x r, (x p q)^2)
//   P(i,j) = e^{2 pi i w_ref n'(i,j)} (1 - (2 pi x p_i q_j)^2 / 4),
//   E_k(i) = e^{2 pi i (a_k i' + delta_k A_i)},  F_k(j) = e^{2 pi i (b_k j' + delta_k B_j)}.
// P is the same for every visibility of the subgrid and is applied once per
// pixel (sep_pixel); its real factor halves the second-order term at either
// end of the w range.  The sums over visibilities (gridder) or pixels
// (degridder) become real matrix products of an E side and an F side, so a
// visibility needs 2 L sines and cosines instead of L^2 and the
// multiply-accumulate runs on the tensor cores at full tile sizes.  The plan
// keeps the neglected terms below kSepTolerance for a source anywhere in the
// usable part of the field (sep_fit), with subgrids of a wide w range worked on
// in parts (sep_parts), and takes the general kernels where that takes too many.
//
// Products: tcgen05.mma kind::f16 with FP32 accumulation in tensor memory.
// Every FP32 operand is split into two halves hi + lo (22 bits), and the
// product taken as hi hi + lo hi + hi lo; the first-order term is about 1e-3
// of the sum and takes one more product of rounded halves.
#pragma once

#include <cuda_fp16.h>

#include "kernels_common.cuh"

namespace idg {

constexpr int kSepThreads = 512;
constexpr int kSepK = 16;                       // contraction length of one chunk (one MMA step)
constexpr float kTurnsToRad = 1.4629180792671596e-9f;  // 2 pi / 2^32

// ---------------------------------------------------------------- tcgen05

// Shared-memory matrix descriptor, K-major without swizzle: 8-row x 16-byte
// core matrices, `k_stride` bytes between core matrices along K and 128
// bytes between those along M or N (consecutive rows 16 bytes apart).
__device__ __forceinline__ uint64_t sep_desc(uint32_t addr, uint32_t k_stride) {
  return uint64_t((addr >> 4) & 0x3fff) | (uint64_t(k_stride >> 4) << 16) | (uint64_t(128 >> 4) << 32) |
         (uint64_t(1) << 46);
}
// kind::f16 instruction descriptor: FP32 accumulator, f16 A and B, both K-major, M = 128; negate: D -= A B
__host__ __device__ constexpr uint32_t sep_idesc(int n, bool negate = false) {
  return (1u << 4) | (uint32_t(negate) << 13) | (uint32_t(n >> 3) << 17) | (uint32_t(128 >> 4) << 24);
}
// D (+)= A B with A in tensor memory (row = lane, two halves per column) and B in shared memory
__device__ __forceinline__ void sep_mma(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d),
      "r"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}
// The tensor core adds each MMA to the FP32 accumulator with truncation: measured against 64 bits, sums shrink by
// 1.7e-8 per MMA (1.4 .. 2.1e-8 over chains of 16 to 120 MMAs and all subgrid sizes).  Results are scaled back by the
// mean, and chains are kept short (kSepMaxChain chunks of 8 MMAs in the gridder, L / 16 in the degridder): the grid's
// error against 64 bits at L = 96 falls from 9.7e-7 to 5e-7, and does not grow with the length of a segment.
constexpr int kSepMaxChain = 8;
__device__ __forceinline__ float sep_unbias(float chunks) { return fmaf(1.7e-8f * 8.f, chunks, 1.f); }

// arrive on `bar` when every MMA issued so far by this thread has completed
__device__ __forceinline__ void sep_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t* dst, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)), "r"(cols)
               : "memory");
}
__device__ __forceinline__ void tmem_free(uint32_t addr, uint32_t cols) {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld16(float (&v)[16], uint32_t addr) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(addr));
#pragma unroll
  for (int k = 0; k < 16; ++k) v[k] = __uint_as_float(r[k]);
}
__device__ __forceinline__ void tmem_st4(uint32_t addr, const uint32_t (&v)[4]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(v[0]), "r"(v[1]),
               "r"(v[2]), "r"(v[3])
               : "memory");
}
__device__ __forceinline__ void tmem_st2(uint32_t addr, uint32_t a, uint32_t b) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1,%2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// ---------------------------------------------------------------- roles

// The block's first 256 threads (producers) write operands and issue MMAs, the
// others (consumers) read the accumulators; each half has its own barrier.
constexpr int kSepHalf = 256;
constexpr int kSepProducerBar = 1, kSepConsumerBar = 2;
__device__ __forceinline__ void half_sync(int bar) {
  asm volatile("bar.sync %0, 256;" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// the 65536 registers of the launch (512 threads x 128) split between the halves: REGS + 256 - REGS
template <int REGS>
__device__ __forceinline__ void regs_take() {
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS));
}
template <int REGS>
__device__ __forceinline__ void regs_give() {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS));
}

// host: whether the kernel was built with the registers per thread that its roles divide among them (a block whose
// roles ask for more than it was launched with would wait for them forever)
template <typename K>
cudaError_t sep_check_regs(K kernel, int regs) {
  cudaFuncAttributes at;
  const cudaError_t e = cudaFuncGetAttributes(&at, kernel);
  return e != cudaSuccess ? e : at.numRegs == regs ? cudaSuccess : cudaErrorInvalidConfiguration;
}

// one lane of the (converged) warp: code under it may use the uniform datapath that MMA operands come from
__device__ __forceinline__ bool elect_one() {
  uint32_t ok;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok));
  return ok != 0;
}
// whether a wait of the block has given up
__device__ __forceinline__ bool sep_failed(const int* fail) { return *reinterpret_cast<const volatile int*>(fail) != 0; }

// bounded wait (a.wait_ns) that reports a timeout once and then lets every later wait of the block pass; from then on
// the barriers say nothing about the data behind them, so nothing whose addresses come from such data may be started
// (sep_failed).  It sleeps between polls, SLEEP ns where the wait is expected to be long: polling takes issue slots from the working
// warps (with 40 ns throughout, a quarter of the degridder's instructions were polls).
template <int SLEEP = 32, typename Args>
__device__ __forceinline__ void sep_wait(uint64_t* bar, uint32_t parity, int* fail, const Args& a) {
  if (mbar_try_wait(bar, parity)) return;
  if (sep_failed(fail)) return;
  if (a.wait_ns) {  // 0: no wait at all
    const uint64_t t0 = global_ns();
    do {
#pragma unroll 1
      for (int k = 0; k < 64; ++k) {
        __nanosleep(SLEEP);
        if (mbar_try_wait(bar, parity)) return;
      }
    } while (global_ns() - t0 <= a.wait_ns);
  }
  atomicOr(a.status, kStatusTimeout);
  *reinterpret_cast<volatile int*>(fail) = 1;
}

// The block's end, after every role's last wait: where a wait gave up, MMAs may still run.  The lane that issued them
// (elect.sync picks the same lane of a full warp each time; a commit tracks the MMAs of its own thread) waits for them,
// bounded, on a barrier that nothing else uses, before the tensor memory goes.
__device__ __forceinline__ void sep_drain(const int* fail, bool issuer_warp, uint64_t* drain) {
  tc_fence_before();
  __syncthreads();
  if (sep_failed(fail)) {  // the same for the whole block: no wait is left that could set it
    if (issuer_warp) {
      if (elect_one()) {
        sep_commit(drain);
        mbar_wait_bounded(drain, 0);
      }
      __syncwarp();
    }
    __syncthreads();
  }
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// all but the newest N groups of this thread have landed
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// the thread's warp as a value the compiler knows to be the same for the whole warp, so that a role taken by one
// warp is a branch for the others and not predicated through
__device__ __forceinline__ int uniform_warp() { return __shfl_sync(0xffffffffu, int(threadIdx.x) >> 5, 0); }

// The items of a block: runs of `run` neighbouring items of the longest-first list, every `stride`-th run.  A run
// re-reads the subgrid it belongs to from L2 at its own time (with single items as many SMs as a subgrid has items
// read the same lines at once: 5.5 instead of 4.9 ms in the degridder of the uneven array), and the stride gives every
// block an even share of long and short items.
struct SepShare {
  int first, last, stride, run;
  __device__ __forceinline__ int next(int idx) const { return (idx + 1) % run ? idx + 1 : idx + 1 + (stride - 1) * run; }
};

// ---------------------------------------------------------------- operands

// phase (radians) of slope `fix` (turns per pixel in units of 2^-32, so the
// product wraps exactly to [-pi, pi]) at pixel offset `off`, plus the w part
// `delta_k` x `fit` (fit carries 2 pi), at most kSepPhase more in the usable
// part of the field and about twice that at its edges
__device__ __forceinline__ float sep_phase(int fix, int off, float delta, float fit) {
  return fmaf(float(int(unsigned(fix) * unsigned(off))), kTurnsToRad, delta * fit);
}

// the same phase's sine and cosine to a unit in the last place (half turns, sincospif): __sincosf's absolute error of 2^-21
// is the largest of the factored form, which takes three of them where one phasor per visibility and pixel takes one
__device__ __forceinline__ void sep_sincos_exact(int fix, int off, float delta, float fit, float* s, float* c) {
  sincospif(fmaf(float(int(unsigned(fix) * unsigned(off))), 4.656612873077393e-10f, delta * fit * 0.3183098861837907f), s, c);
}

// slope in turns per pixel as a multiple of 2^-32 (whole turns wrap away)
__device__ __forceinline__ int sep_fix(double turns) { return int(unsigned(__double2ll_rn(turns * 4294967296.0))); }

// power of two that brings `m` into [8192, 16384); 1 for 0, infinity and NaN.  A complex product of values whose
// components are bounded by `m` stays below 2^1.5 m = 46341 of a half's 65504, so that hi + lo halves keep 22 bits of
// values down to 2^-13 of the largest, and an absolute 2^-38 of it below.
__device__ __forceinline__ float sep_scale(float m) {
  if (!(m > 0.f) || isinf(m)) return 1.f;
  const int e = 13 - ilogbf(m);
  return ldexpf(1.f, e > 126 ? 126 : e);
}

__device__ __forceinline__ uint32_t h2_bits(__half2 h) { return *reinterpret_cast<uint32_t*>(&h); }

// (hi, lo) halves of a pair: hi = x rounded to half, lo = (x - hi) rounded to half; returns hi
__device__ __forceinline__ __half2 sep_split(float2 x, uint32_t& hi, uint32_t& lo) {
  const __half2 h = __floats2half2_rn(x.x, x.y);
  hi = h2_bits(h);
  const float2 f = __half22float2(h);
  lo = h2_bits(__floats2half2_rn(x.x - f.x, x.y - f.y));
  return h;
}
// e^{i phase} of two contraction indices: slopes in units of 2^-32 turns, deltas
__device__ __forceinline__ void sep_phasor2(int fix0, int fix1, int off, float2 delta, float fit, float2& c,
                                            float2& s) {
  __sincosf(sep_phase(fix0, off, delta.x, fit), &s.x, &c.x);
  __sincosf(sep_phase(fix1, off, delta.y, fit), &s.y, &c.y);
}
__device__ __forceinline__ float2 pair_of(const float4& v, int h) {
  return h ? make_float2(v.z, v.w) : make_float2(v.x, v.y);
}
__device__ __forceinline__ void sts128(uint32_t addr, const uint32_t (&v)[4]) {
  asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3])
               : "memory");
}

// the F side of one column index for 8 consecutive contraction indices: Re and Im rows at dst and dst + block,
// the levels (hi, lo, first order) `level` bytes apart
struct SepF {
  uint32_t r_hi[4], i_hi[4], r_lo[4], i_lo[4], r_c[4], i_c[4];
};
__device__ __forceinline__ void sep_store_f(const SepF& f, uint32_t dst, uint32_t block, uint32_t level) {
  sts128(dst, f.r_hi);
  sts128(dst + block, f.i_hi);
  sts128(dst + level, f.r_lo);
  sts128(dst + level + block, f.i_lo);
  sts128(dst + 2 * level, f.r_c);
  sts128(dst + 2 * level + block, f.i_c);
}
// D (+)= E F for one contraction step of 16: the E side in tensor memory at column `e` as (Re hi, Im hi, Re lo, Im lo,
// Re first order, Im first order) of 8 columns each, the F side in shared memory (sep_store_f, k groups `group`
// bytes apart), D = re at column d and im at d + n, n columns each.  Products lo hi, hi lo, first order, hi hi; all
// MMAs on one accumulator have the same shape, so they run in the order of issue.
// CORR: columns from d to an accumulator of its own for all but hi hi, or 0: the truncations then happen at the
// corrections' magnitude, and 2 of 8 MMAs a chunk truncate the sum itself.
template <uint32_t CORR = 0>
__device__ __forceinline__ void sep_product(uint32_t d, uint32_t e, uint32_t f, int n, uint32_t block, uint32_t group,
                                            uint32_t level, bool first) {
  const uint32_t add = sep_idesc(n), sub = sep_idesc(n, true);
  const uint32_t el[4] = {1, 0, 2, 0}, fl[4] = {0, 1, 2, 0};
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const uint32_t ea = e + el[t] * 16, fa = f + fl[t] * level;
    const uint32_t acc = first && (t == 0 || (t == 3 && CORR)) ? 0u : 1u, dt = t < 3 ? d + CORR : d;
    const uint64_t fr = sep_desc(fa, group), fi = sep_desc(fa + block, group);
    sep_mma(dt, ea, fr, add, acc);           // re += Re E Re F
    sep_mma(dt + n, ea, fi, add, acc);       // im += Re E Im F
    sep_mma(dt, ea + 8, fi, sub, 1u);        // re -= Im E Im F
    sep_mma(dt + n, ea + 8, fr, add, 1u);    // im += Im E Re F
  }
}

// P of a pixel: w = (w_ref, x^2 / 4), the two-float n' (exact range reduction), 2 pi p_i q_j; exact: sine and cosine to
// a unit in the last place (sep_sincos_exact)
__device__ __forceinline__ float2 sep_pixel(float2 w, float2 n1, float pq, bool exact = false) {
  const float t = w.x * n1.x;
  const float lo = fmaf(w.x, n1.y, fmaf(w.x, n1.x, -t));
  const float turns = (t - rintf(t)) + lo;
  const float k = fmaf(-w.y * pq, pq, 1.f);
  float s, c;
  if (exact)
    sincospif(2.f * turns, &s, &c);
  else
    __sincosf(turns * kTwoPiF, &s, &c);
  return make_float2(k * c, k * s);
}

}  // namespace idg
