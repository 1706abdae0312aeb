// Subgrid Fourier transforms and the master-grid adder / splitter.
//
// Section 2.5 imaging steps 2b-2c (Eq. 8, Eq. 6) and prediction steps
// 3a-3b.  The centred transform
//   Vhat(x,y) = sum_{ij} X(i,j) e^{-2 pi i [(x-L/2)(i-L/2) + (y-L/2)(j-L/2)]/L}
// equals (-1)^(x+y) FFT[(-1)^(i+j) X](x,y) for even L.  The gridder already
// applied (-1)^(i+j); the adder applies (-1)^(x+y) while it adds into the
// FP64 master grid.  The splitter applies (-1)^(x+y) on the way in and the
// degridder's prologue (-1)^(i+j) after the inverse transform.
//
// One block transforms one polarisation plane of one subgrid (L x L complex
// FP32; 4 correlation planes, or the one Stokes-I plane) in shared memory,
// columns then rows.  A line of L = R1 R2 points takes two steps in registers: R2
// transforms of R1 points at stride R2, twiddles, then R1 transforms of R2
// points, each step writing where it read, so a step needs no second barrier
// and leaves logical index k1 + R1 k2 at place k1 R2 + k2 (fft_place), which
// the output undoes.  The first step reads global memory directly.
//
// What bounds it: shared memory (8 passes over the plane; a sequence of radix
// 4, 2 and 3 stages with loads and stores apart took 18) and, in the adder,
// the FP64 atomics: two neighbouring lanes add the parts of one cell, so a
// warp's addition covers whole 32-byte sectors.  Measured on GB300, MWA-like
// workload (12600 subgrids of 96 x 96, 4 planes, per call): transform and adder 1.9 ms
// against 3.7, splitter and transform 2.1 against 4.1.
#include "sep_common.cuh"

namespace idg {

// L = kR1 kR2; lines are processed at a pitch of L + 1, so lanes along rows hit distinct banks.  kBlocks: blocks per SM
// the registers are budgeted for (what shared memory allows)
template <int L>
struct FftShape;
template <>
struct FftShape<32> {
  static constexpr int kR1 = 4, kR2 = 8, kThreads = 128, kBlocks = 12;
};
template <>
struct FftShape<64> {
  static constexpr int kR1 = 8, kR2 = 8, kThreads = 256, kBlocks = 6;
};
template <>
struct FftShape<96> {
  static constexpr int kR1 = 8, kR2 = 12, kThreads = 384, kBlocks = 3;
};
template <>
struct FftShape<128> {
  static constexpr int kR1 = 8, kR2 = 16, kThreads = 512, kBlocks = 1;
};

__device__ __forceinline__ float2 c2mul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// e^{DIR 2 pi i k / R}
template <int R, int DIR>
__device__ __forceinline__ float2 cis(int k) {
  constexpr float c16[16] = {1.f, 0.92387953251128674f, 0.70710678118654752f, 0.38268343236508977f, 0.f, -0.38268343236508977f,
                             -0.70710678118654752f, -0.92387953251128674f, -1.f, -0.92387953251128674f,
                             -0.70710678118654752f, -0.38268343236508977f, 0.f, 0.38268343236508977f,
                             0.70710678118654752f, 0.92387953251128674f};
  constexpr float c12[12] = {1.f, 0.86602540378443865f, 0.5f, 0.f, -0.5f, -0.86602540378443865f,
                             -1.f, -0.86602540378443865f, -0.5f, 0.f, 0.5f, 0.86602540378443865f};
  if constexpr (R == 12) return make_float2(c12[k], DIR * c12[(k + 9) % 12]);
  constexpr int q = 16 / (R == 12 ? 16 : R);
  return make_float2(c16[k * q], DIR * c16[(k * q + 12) % 16]);
}

// R-point transform in registers, natural order in and out
template <int R, int DIR>
__device__ __forceinline__ void dft(float2 (&v)[R]) {
  if constexpr (R == 2) {
    const float2 a = v[0], b = v[1];
    v[0] = make_float2(a.x + b.x, a.y + b.y);
    v[1] = make_float2(a.x - b.x, a.y - b.y);
  } else if constexpr (R == 3) {
    const float s = DIR * 0.86602540378443865f;
    const float2 t = make_float2(v[1].x + v[2].x, v[1].y + v[2].y);
    const float2 m = make_float2(fmaf(-0.5f, t.x, v[0].x), fmaf(-0.5f, t.y, v[0].y));
    const float2 d = make_float2(-s * (v[1].y - v[2].y), s * (v[1].x - v[2].x));
    v[0] = make_float2(v[0].x + t.x, v[0].y + t.y);
    v[1] = make_float2(m.x + d.x, m.y + d.y);
    v[2] = make_float2(m.x - d.x, m.y - d.y);
  } else if constexpr (R == 4) {
    const float2 a0 = make_float2(v[0].x + v[2].x, v[0].y + v[2].y), a1 = make_float2(v[0].x - v[2].x, v[0].y - v[2].y);
    const float2 a2 = make_float2(v[1].x + v[3].x, v[1].y + v[3].y), d = make_float2(v[1].x - v[3].x, v[1].y - v[3].y);
    const float2 a3 = DIR < 0 ? make_float2(d.y, -d.x) : make_float2(-d.y, d.x);
    v[0] = make_float2(a0.x + a2.x, a0.y + a2.y);
    v[1] = make_float2(a1.x + a3.x, a1.y + a3.y);
    v[2] = make_float2(a0.x - a2.x, a0.y - a2.y);
    v[3] = make_float2(a1.x - a3.x, a1.y - a3.y);
  } else {
    constexpr int B = R / 4;  // R = 4 B: B transforms of 4 points, then 4 of B points
    float2 u[B][4];
#pragma unroll
    for (int b = 0; b < B; ++b) {
#pragma unroll
      for (int q = 0; q < 4; ++q) u[b][q] = v[b + B * q];
      dft<4, DIR>(u[b]);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float2 w[B];
#pragma unroll
      for (int b = 0; b < B; ++b) w[b] = (b == 0 || k == 0) ? u[b][k] : c2mul(u[b][k], cis<R, DIR>(b * k));
      dft<B, DIR>(w);
#pragma unroll
      for (int q = 0; q < B; ++q) v[k + 4 * q] = w[q];
    }
  }
}

// place of logical index k after the two steps of a line
template <int L>
__device__ __forceinline__ int fft_place(int k) {
  return (k % FftShape<L>::kR1) * FftShape<L>::kR2 + k / FftShape<L>::kR1;
}

template <int R, int DIR>
__device__ __forceinline__ void twiddle(float2 (&v)[R], const float2* tw, int n) {
#pragma unroll
  for (int k = 1; k < R; ++k) {
    float2 w = tw[n * k];
    if (DIR > 0) w.y = -w.y;
    v[k] = c2mul(v[k], w);
  }
}

// both dimensions of an L x L plane: load(j, i) gives the input, buf (pitch L + 1) receives the transform at
// buf[fft_place(y) * (L + 1) + fft_place(x)]; tw: e^{-2 pi i m / L}, visible to the block
template <int L, int DIR, typename Load>
__device__ __forceinline__ void fft2d(float2* buf, const float2* tw, Load load) {
  using F = FftShape<L>;
  constexpr int R1 = F::kR1, R2 = F::kR2, P = L + 1;
  for (int t = threadIdx.x; t < L * R2; t += F::kThreads) {  // lanes along columns i
    const int n = t / L, i = t - n * L;
    float2 v[R1];
#pragma unroll
    for (int q = 0; q < R1; ++q) v[q] = load(n + R2 * q, i);
    dft<R1, DIR>(v);
    twiddle<R1, DIR>(v, tw, n);
#pragma unroll
    for (int k = 0; k < R1; ++k) buf[(n + R2 * k) * P + i] = v[k];
  }
  __syncthreads();
  for (int t = threadIdx.x; t < L * R1; t += F::kThreads) {
    const int k1 = t / L, i = t - k1 * L;
    float2* at = buf + k1 * R2 * P + i;
    float2 v[R2];
#pragma unroll
    for (int q = 0; q < R2; ++q) v[q] = at[q * P];
    dft<R2, DIR>(v);
#pragma unroll
    for (int q = 0; q < R2; ++q) at[q * P] = v[q];
  }
  __syncthreads();
  for (int t = threadIdx.x; t < L * R2; t += F::kThreads) {  // lanes along rows
    const int n = t / L, r = t - n * L;
    float2* at = buf + r * P + n;
    float2 v[R1];
#pragma unroll
    for (int q = 0; q < R1; ++q) v[q] = at[R2 * q];
    dft<R1, DIR>(v);
    twiddle<R1, DIR>(v, tw, n);
#pragma unroll
    for (int k = 0; k < R1; ++k) at[R2 * k] = v[k];
  }
  __syncthreads();
  for (int t = threadIdx.x; t < L * R1; t += F::kThreads) {
    const int k1 = t / L, r = t - k1 * L;
    float2* at = buf + r * P + k1 * R2;
    float2 v[R2];
#pragma unroll
    for (int q = 0; q < R2; ++q) v[q] = at[q];
    dft<R2, DIR>(v);
#pragma unroll
    for (int q = 0; q < R2; ++q) at[q] = v[q];
  }
  __syncthreads();
}

// grid-direction: transform the gridder's subgrid image and add it into the
// FP64 master grid (mode 0) or leave the transform in scratch (mode 1)
template <int L, int MODE>
__global__ void __launch_bounds__(FftShape<L>::kThreads, FftShape<L>::kBlocks) fft_adder_kernel(const FftArgs a) {
  constexpr int T = FftShape<L>::kThreads, P = L + 1;
  extern __shared__ float2 sbuf[];
  float2* buf = sbuf;
  float2* tw = sbuf + L * P;
  const int sgi = blockIdx.x / a.npol, pol = blockIdx.x % a.npol;
  const SubgridDesc sd = a.sg[sgi];
  float2* plane = a.scratch + (size_t(sgi) * 4 + pol) * L * L;
  for (int e = threadIdx.x; e < L; e += T) tw[e] = a.twiddle[e];
  __syncthreads();
  fft2d<L, -1>(buf, tw, [&](int j, int i) { return plane[j * L + i]; });
  if (MODE == 0) {
    // plane set of the subgrid's w layer, then the polarisation plane
    double* g = reinterpret_cast<double*>(a.grid) +
                ((size_t(sd.layer) * a.npol + pol) * a.N * a.N + size_t(sd.y0) * a.N + sd.x0) * 2;
    const float* val = reinterpret_cast<const float*>(buf);
    for (int e = threadIdx.x; e < 2 * L * L; e += T) {  // even lanes the real parts, odd lanes the imaginary parts
      const int y = e / (2 * L), c = e - y * (2 * L), x = c >> 1;
      const float v = val[(fft_place<L>(y) * P + fft_place<L>(x)) * 2 + (c & 1)];
      atomicAdd(g + size_t(y) * a.N * 2 + c, double(((x + y) & 1) ? -v : v));
    }
  } else {
    for (int e = threadIdx.x; e < L * L; e += T) {
      const int y = e / L, x = e - y * L;
      plane[e] = buf[fft_place<L>(y) * P + fft_place<L>(x)];
    }
  }
}

// degrid-direction: copy the subgrid's footprint out of the master grid
// (FP64 -> FP32, times (-1)^(x+y)) and inverse-transform it into scratch; EXACT: FftArgs.exact (as a branch it costs
// the others 2 % of a small call)
template <int L, bool EXACT>
__global__ void __launch_bounds__(FftShape<L>::kThreads, FftShape<L>::kBlocks) splitter_ifft_kernel(const FftArgs a) {
  constexpr int T = FftShape<L>::kThreads, P = L + 1;
  extern __shared__ float2 sbuf[];
  float2* buf = sbuf;
  float2* tw = sbuf + L * P;
  const int sgi = blockIdx.x / a.npol, pol = blockIdx.x % a.npol;
  const SubgridDesc sd = a.sg[sgi];
  for (int e = threadIdx.x; e < L; e += T) tw[e] = a.twiddle[e];
  __syncthreads();
  const double2* g = a.grid + (size_t(sd.layer) * a.npol + pol) * a.N * a.N + size_t(sd.y0) * a.N + sd.x0;
  fft2d<L, +1>(buf, tw, [&](int y, int x) {
    const double2 v = g[size_t(y) * a.N + x];
    const float sgn = ((x + y) & 1) ? -1.f : 1.f;
    return make_float2(sgn * float(v.x), sgn * float(v.y));
  });
  if (!a.ymax) {
    float2* dst = a.scratch + (size_t(sgi) * 4 + pol) * L * L;
    for (int e = threadIdx.x; e < L * L; e += T) {
      const int j = e / L, i = e - j * L;
      dst[e] = buf[fft_place<L>(j) * P + fft_place<L>(i)];
    }
    return;
  }
  // what every visibility of the subgrid shares (sep_common.cuh), once per pixel here instead of once per segment;
  // written as the degridder reads it, [32 columns][row pair][re, im][column] of the values at both rows
  const float2 w_ref = a.w_ref[sgi];
  float2* pairs = a.scratch + (size_t(sgi) * 4 + pol) * L * L;
  float m = 0.f;
  for (int e = threadIdx.x; e < L * L / 2; e += T) {
    const int jp = e / L, i = e - jp * L;
    const int ip = fft_place<L>(i);
    const float2 v0 = buf[fft_place<L>(2 * jp) * P + ip], v1 = buf[fft_place<L>(2 * jp + 1) * P + ip];
    const float ti = a.taper[i] * ((i & 1) ? -1.f : 1.f), t0 = ti * a.taper[2 * jp], t1 = -ti * a.taper[2 * jp + 1];
    const float fit_p = __ldg(a.sep.p + i);
    const float2 p0 = sep_pixel(w_ref, __ldg(a.sep.n1 + 2 * jp * L + i), fit_p * __ldg(a.sep.q + 2 * jp), EXACT);
    const float2 p1 = sep_pixel(w_ref, __ldg(a.sep.n1 + (2 * jp + 1) * L + i), fit_p * __ldg(a.sep.q + 2 * jp + 1), EXACT);
    const float2 re = make_float2(t0 * (v0.x * p0.x + v0.y * p0.y), t1 * (v1.x * p1.x + v1.y * p1.y));
    const float2 im = make_float2(t0 * (v0.y * p0.x - v0.x * p0.y), t1 * (v1.y * p1.x - v1.x * p1.y));
    m = fmaxf(fmaxf(fmaxf(m, fabsf(re.x)), fabsf(re.y)), fmaxf(fabsf(im.x), fabsf(im.y)));
    float2* dst = pairs + (size_t(i >> 5) * (L / 2) + jp) * 64 + (i & 31);
    dst[0] = re;
    dst[32] = im;
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  float* part = reinterpret_cast<float*>(tw);  // the twiddles are done with
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < T / 32; ++w) m = fmaxf(m, part[w]);
    a.ymax[sgi * 4 + pol] = m;
  }
}

// plan-order export of subgrid images for inspection, undoing (-1)^(x+y); parts of a subgrid add up (out starts at 0)
template <int L>
__global__ void export_kernel(const SubgridDesc* sg, const float2* scratch, float2* out, int npol) {
  const int sgi = blockIdx.x / npol, pol = blockIdx.x % npol;
  const int dst_sg = sg[sgi].plan_index;
  const bool part = (sg[sgi].flags & kSubgridPart) != 0;
  const float2* src = scratch + (size_t(sgi) * 4 + pol) * L * L;
  float2* dst = out + (size_t(dst_sg) * npol + pol) * L * L;
  for (int e = threadIdx.x; e < L * L; e += blockDim.x) {
    const int y = e / L, x = e - y * L;
    const float sgn = ((x + y) & 1) ? -1.f : 1.f;
    const float2 v = src[e];
    if (part) {
      atomicAdd(&dst[e].x, sgn * v.x);
      atomicAdd(&dst[e].y, sgn * v.y);
    } else {
      dst[e] = make_float2(sgn * v.x, sgn * v.y);
    }
  }
}

template <int L>
static size_t fft_smem() {
  return sizeof(float2) * (L * (L + 1) + L);
}

template <int L>
static int configure_t() {
  const int smem = int(fft_smem<L>());
  cudaError_t e = cudaFuncSetAttribute(fft_adder_kernel<L, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fft_adder_kernel<L, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(splitter_ifft_kernel<L, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(splitter_ifft_kernel<L, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  // shared memory is what bounds these kernels' occupancy: ask for the largest carveout
  const void* fns[4] = {reinterpret_cast<const void*>(fft_adder_kernel<L, 0>),
                        reinterpret_cast<const void*>(fft_adder_kernel<L, 1>),
                        reinterpret_cast<const void*>(splitter_ifft_kernel<L, false>),
                        reinterpret_cast<const void*>(splitter_ifft_kernel<L, true>)};
  for (const void* fn : fns)
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, int(cudaSharedmemCarveoutMaxShared));
  return int(e);
}

int configure_kernels(int L) {
  switch (L) {
    case 32: return configure_t<32>();
    case 64: return configure_t<64>();
    case 96: return configure_t<96>();
    case 128: return configure_t<128>();
    default: return int(cudaErrorInvalidValue);
  }
}

template <int L>
static int fft_adder_t(const FftArgs& a, int n, int mode, void* stream) {
  if (n <= 0) return 0;
  if (mode == 0)
    fft_adder_kernel<L, 0><<<n * a.npol, FftShape<L>::kThreads, fft_smem<L>(), cudaStream_t(stream)>>>(a);
  else
    fft_adder_kernel<L, 1><<<n * a.npol, FftShape<L>::kThreads, fft_smem<L>(), cudaStream_t(stream)>>>(a);
  return int(cudaGetLastError());
}

template <int L>
static int splitter_t(const FftArgs& a, int n, void* stream) {
  if (n <= 0) return 0;
  if (a.exact)
    splitter_ifft_kernel<L, true><<<n * a.npol, FftShape<L>::kThreads, fft_smem<L>(), cudaStream_t(stream)>>>(a);
  else
    splitter_ifft_kernel<L, false><<<n * a.npol, FftShape<L>::kThreads, fft_smem<L>(), cudaStream_t(stream)>>>(a);
  return int(cudaGetLastError());
}

template <int L>
static int export_t(const SubgridDesc* sg, const float2* scratch, float2* out, int n, int npol, void* stream) {
  if (n <= 0) return 0;
  export_kernel<L><<<n * npol, 256, 0, cudaStream_t(stream)>>>(sg, scratch, out, npol);
  return int(cudaGetLastError());
}

int launch_fft_adder(int L, const FftArgs& a, int n, int mode, void* stream) {
  switch (L) {
    case 32: return fft_adder_t<32>(a, n, mode, stream);
    case 64: return fft_adder_t<64>(a, n, mode, stream);
    case 96: return fft_adder_t<96>(a, n, mode, stream);
    case 128: return fft_adder_t<128>(a, n, mode, stream);
    default: return int(cudaErrorInvalidValue);
  }
}

int launch_splitter_ifft(int L, const FftArgs& a, int n, void* stream) {
  switch (L) {
    case 32: return splitter_t<32>(a, n, stream);
    case 64: return splitter_t<64>(a, n, stream);
    case 96: return splitter_t<96>(a, n, stream);
    case 128: return splitter_t<128>(a, n, stream);
    default: return int(cudaErrorInvalidValue);
  }
}

int launch_export_subgrids(int L, const SubgridDesc* sg, const float2* scratch, float2* out, int n, int npol,
                           void* stream) {
  switch (L) {
    case 32: return export_t<32>(sg, scratch, out, n, npol, stream);
    case 64: return export_t<64>(sg, scratch, out, n, npol, stream);
    case 96: return export_t<96>(sg, scratch, out, n, npol, stream);
    case 128: return export_t<128>(sg, scratch, out, n, npol, stream);
    default: return int(cudaErrorInvalidValue);
  }
}

}  // namespace idg
