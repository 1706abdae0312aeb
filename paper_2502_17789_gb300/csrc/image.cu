// Image-domain wrapper (Section 2.5 imaging step 3, Eq. 11, and prediction
// step 2, Eq. 12): the element-wise pass beside each master-grid transform.
// The centred transform of even length N is
//   sum_X f(X) e^{-+2 pi i (X - N/2)(p - N/2)/N}
//     = (-1)^p sum_X (-1)^X f(X) e^{-+2 pi i X p/N}   (per axis, up to e^{-+i pi N/2}, 1 over both axes),
// and the sign on the grid's side of a plain FFT is a shift by N/2 on the
// image's: one pass on the image's side does both, and the grid is transformed
// as it lies.  Each w layer's image is multiplied by e^{+2 pi i w0 n'(l,m)}
// (w-stacking); the taper correction divides by L^2 T(l_p) T(m_q); with the
// A-term power normalisation of Section 3.3 a last pass divides by the
// averaged weights.
#include "kernels_common.cuh"

namespace idg {

// For every pixel (x, y) of the N x N image and each of the npol planes, with
//   f(x, y) = c * w[x] w[y] * (-1)^(x+y) * e^{i 2 pi w0 n'(x,y)},
//   kToImage:  out(x, y) = in(x + N/2, y + N/2) f(x, y)    (added to out with accumulate),
//   otherwise: out(x + N/2, y + N/2) = in(x, y) f(x, y),
// positions modulo N; n' = sqrt(1 - l^2 - m^2) - 1 at l = (x - N/2) FOV/N, m
// likewise (the phase only for kPhase; sincospi keeps it accurate for large
// w0 n').  in == out is allowed: a pixel and the one N/2 away are read and
// written by the same thread.
//
// What bounds it is the chip's FP64 rate, not memory (32 bytes an element): a
// phase takes some 70 double operations and a complex product 4.  The phase
// depends on |x - N/2| and |y - N/2| only, so one thread takes the four
// mirrored pixels of (a, b) with their four partners N/2 away: two phases for
// eight pixels, with the same bits as one per pixel; without a phase the factor
// is real and an element takes two products.  Four 2048 x 2048 planes with a
// phase: 290 us, where a phase per pixel took 620 us and the grid side's signs
// another 143 us in a pass of their own.
template <bool kPhase, bool kToImage>
__global__ void __launch_bounds__(256) image_pass_kernel(int npol, const double2* in, double2* out, const double* w,
                                                         double c, double w0, double fov, int N, bool accumulate) {
  const int H = N / 2, nb = H / 2 + 1;
  const int64_t npix = int64_t(N) * N, total = int64_t(H + 1) * nb;
  const int64_t stride = int64_t(gridDim.x) * blockDim.x;
  auto phase = [&](int dx, int dy, double* s, double* co) {
    const double l = double(dx) * fov / double(N), m = double(dy) * fov / double(N);
    const double n1 = sqrt(1.0 - l * l - m * m) - 1.0;
    sincospi(2.0 * w0 * n1, s, co);
  };
  for (int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; e < total; e += stride) {
    const int b = int(e / (H + 1)), a = int(e - int64_t(b) * (H + 1));
    // (a, b) and (H - a, H - b) are the same eight pixels; b <= H/2 leaves the row b = H/2 twice
    if (2 * b == H && 2 * a > H) continue;
    double sp = 0.0, cp = 1.0, sq = 0.0, cq = 1.0;
    if (kPhase) {
      phase(H - a, H - b, &sp, &cp);
      phase(a, b, &sq, &cq);
    }
    // mirror images that fall on the pixel itself, and a class that is its own partner
    const bool one_x = a == 0 || a == H || (2 * a == H && 2 * b == H), one_y = b == 0 || b == H;
#pragma unroll
    for (int my = 0; my < 2; ++my) {
      if (my && one_y) continue;
      const int y = my ? N - b : b, y2 = y < H ? y + H : y - H;
#pragma unroll
      for (int mx = 0; mx < 2; ++mx) {
        if (mx && one_x) continue;
        const int x = mx ? N - a : a, x2 = x < H ? x + H : x - H;
        const int64_t ip = int64_t(y) * N + x, iq = int64_t(y2) * N + x2;
        // N/2 apart on both axes: the same sign
        const double c1 = (x + y) & 1 ? -c : c;
        const double fp = c1 * w[x] * w[y], fq = c1 * w[x2] * w[y2];
        // the factor belongs to the image's side: the pixel read, or the one written
        const double f_in_p = kToImage ? fq : fp, f_in_q = kToImage ? fp : fq;
        const double rp = f_in_p * (kToImage ? cq : cp), jp = f_in_p * (kToImage ? sq : sp);
        const double rq = f_in_q * (kToImage ? cp : cq), jq = f_in_q * (kToImage ? sp : sq);
#pragma unroll 4
        for (int k = 0; k < npol; ++k) {
          const double2* src = in + int64_t(k) * npix;
          double2* dst = out + int64_t(k) * npix;
          const double2 vp = src[ip], vq = src[iq];
          double2 tp, tq;  // what the pixels read at p and q become: written at q and p
          if (kPhase) {
            tp = make_double2(vp.x * rp - vp.y * jp, vp.x * jp + vp.y * rp);
            tq = make_double2(vq.x * rq - vq.y * jq, vq.x * jq + vq.y * rq);
          } else {
            tp = make_double2(vp.x * f_in_p, vp.y * f_in_p);
            tq = make_double2(vq.x * f_in_q, vq.y * f_in_q);
          }
          if (kToImage && accumulate) {
            const double2 oq = dst[iq], op = dst[ip];
            tp.x += oq.x;
            tp.y += oq.y;
            tq.x += op.x;
            tq.y += op.y;
          }
          dst[iq] = tp;
          dst[ip] = tq;
        }
      }
    }
  }
}

int launch_image_pass(int npol, const double2* in, double2* out, const double* w, double c, double w0, double fov,
                      int N, int flags, void* stream) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return int(e);
  const int64_t want = (int64_t(N / 2 + 1) * (N / 4 + 1) + 255) / 256;
  const int blocks = int(want < int64_t(sms) * 8 ? want : int64_t(sms) * 8);
  const bool to_image = flags & kPassToImage, acc = flags & kPassAccumulate;
  auto kernel = w0 != 0.0 ? (to_image ? image_pass_kernel<true, true> : image_pass_kernel<true, false>)
                          : (to_image ? image_pass_kernel<false, true> : image_pass_kernel<false, false>);
  kernel<<<blocks, 256, 0, cudaStream_t(stream)>>>(npol, in, out, w, c, w0, fov, N, acc);
  return int(cudaGetLastError());
}

// A-term power correction (Section 3.3): divide every image pixel by the
// visibility-weighted average of the normalisation factor, W = aw[j L + i] /
// aw[L L] on the subgrid lattice (l_i = (i - L/2) FOV/L), interpolated
// bilinearly at the fractional lattice index (p - N/2) L/N + L/2 (flat beyond
// the last lattice point).  A zero W (no visibilities) leaves the pixel.
__global__ void __launch_bounds__(256) weight_correction_kernel(int npol, double2* img, const double* aw, int N,
                                                                int L) {
  const int64_t npix = int64_t(N) * N;
  const int64_t stride = int64_t(gridDim.x) * blockDim.x;
  const double total = aw[int64_t(L) * L];
  for (int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; e < npix; e += stride) {
    const int x = int(e % N), y = int(e / N);
    auto lattice = [&](int p, int* i0, double* fr) {
      const double f = double(p - N / 2) * (double(L) / double(N)) + double(L / 2);
      int i = int(floor(f));
      i = i < 0 ? 0 : (i > L - 2 ? L - 2 : i);
      double r = f - double(i);
      *i0 = i;
      *fr = r < 0.0 ? 0.0 : (r > 1.0 ? 1.0 : r);
    };
    int i0, j0;
    double fx, fy;
    lattice(x, &i0, &fx);
    lattice(y, &j0, &fy);
    const double* r0 = aw + int64_t(j0) * L + i0;
    const double* r1 = r0 + L;
    const double wv = ((1.0 - fx) * r0[0] + fx * r0[1]) * (1.0 - fy) + ((1.0 - fx) * r1[0] + fx * r1[1]) * fy;
    if (!(wv > 0.0) || !(total > 0.0)) continue;
    const double c = total / wv;
#pragma unroll 4
    for (int k = 0; k < npol; ++k) {
      double2 v = img[int64_t(k) * npix + e];
      v.x *= c;
      v.y *= c;
      img[int64_t(k) * npix + e] = v;
    }
  }
}

int launch_weight_correction(int npol, double2* image, const double* aweights, int N, int L, void* stream) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return int(e);
  const int64_t want = (int64_t(N) * N + 255) / 256;
  const int blocks = int(want < int64_t(sms) * 8 ? want : int64_t(sms) * 8);
  if (blocks <= 0) return 0;
  weight_correction_kernel<<<blocks, 256, 0, cudaStream_t(stream)>>>(npol, image, aweights, N, L);
  return int(cudaGetLastError());
}

}  // namespace idg
