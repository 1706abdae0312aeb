// Gridder with separable phasors (templates), included by the per-subgrid-size
// translation units gridder_sep_lNN.cu.  See sep_common.cuh for the split of
// the phase.
//
// Eq. 10's sum of one A-term segment over a tile of 32 pixel columns i and
// all L rows j is a complex matrix product over the segment's visibilities,
//   X_p(i,j) = sum_k [V_{k,p} E_k(i)] F_k(j) (1 + 2 pi i delta_k p_i q_j):
// rows (p, i), 4 x 32 = 128, the height of one tcgen05 tile at every L;
// columns (re | im, j), N = 2 L.  The E side is stored as its real and
// imaginary parts, the F side as rows (-Im | Re | Im), so that
//   D += Re(E) [Re F | Im F] + Im(E) [-Im F | Re F]
// takes two MMAs per 16 visibilities and per product of the split (hi hi,
// lo hi, hi lo, first order).
//
// One block of 512 threads per bundle of items (subgrid, 32 columns), split
// into two halves that run side by side.  Producers: per chunk of 16 visibilities every
// thread writes one row (p, i) x 8 visibilities of the E side and, of the F
// side, one row j x 8 visibilities, into a ring of 2-4 chunk buffers; one of
// them issues the chunk's 8 MMAs, whose commit frees the buffer.  Consumers:
// the accumulator alternates between two column ranges of tensor memory from
// segment to segment; while one fills, they take the other through a shared
// memory transpose, apply A_p^H X A_q and add to their pixels in registers (two
// neighbouring rows per thread, packed f32x2).  w_ref, taper and centring
// sign are applied once, when the item's pixels are written.  The pixel sums
// need 8 L / 8 registers of a consumer, so the halves split the block's
// registers unevenly.
//
// Measured (GB300, MWA-like workload, 96 x 96 subgrids, segments of about 60
// visibilities, per grid call): @@ ms, against 29.0 ms with all threads
// producing and then consuming in turn, and 81.7 ms of the kernel with one
// phasor per visibility and pixel (gridder_tc_kernels.cuh); grid error 9e-7
// against 2.2e-6.
#pragma once

#include "sep_common.cuh"

namespace idg {

template <int L>
struct Gsep {
  static constexpr int kN = 2 * L;                               // accumulator columns (re | im)
  static constexpr int kColStride = L <= 32 ? 64 : L <= 64 ? 128 : 256;  // between the two accumulators
  static constexpr uint32_t kTmemCols = 2 * kColStride;
  static constexpr uint32_t kABytes = 6 * 4096;                  // (hi, lo, first order) x (re, im), 128 x 16 halves
  static constexpr uint32_t kFBlock = L * 16;                    // one (k group, block) of the F side
  static constexpr uint32_t kFGroup = 3 * kFBlock;               // one k group
  static constexpr uint32_t kFLevel = 2 * kFGroup;               // one level
  static constexpr uint32_t kBufBytes = kABytes + 3 * kFLevel;
  static constexpr int kSteps = L / 16;                          // epilogue steps of 16 rows j
  static constexpr int kConsumerRegs = L == 128 ? 184 : 168;     // the producers keep 256 less
};

// per-block state after the chunk ring: two transpose buffers, the chunk records, barriers
struct GsepTail {
  float2 x[2][4 * 2 * 256];  // [buffer][pol][re, im][row pair of 8][column of 32]
  float4 rec[2][kGsepChunkFloat4];
  uint64_t empty[4];         // chunk buffer read by its MMAs
  uint64_t full[2];          // accumulator complete
  uint64_t drained[2];       // accumulator read by the 8 consumer warps
  uint32_t tmem;
  int fail;
};

template <int L>
size_t gsep_smem(int nbuf, int nodes) {
  return size_t(nbuf) * Gsep<L>::kBufBytes + sizeof(GsepTail) + size_t(nodes) * 4 * 32 * sizeof(float4);
}

template <int L>
int gsep_buffers(int nodes) {
  for (int nb = 4; nb > 2; --nb)
    if (gsep_smem<L>(nb, nodes) <= kSepSmemLimit) return nb;
  return 2;
}

// E side row (p, i) and F side row j of one chunk (producer thread)
template <int L>
__device__ __forceinline__ void gsep_produce(uint32_t buf, const float4* rec, int i_off, float fit_a, float fit_p,
                                             int j_off, float fit_b, float fit_q) {
  using C = Gsep<L>;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  {
    const int p = warp & 3, g = warp >> 2;
    const float2* val = reinterpret_cast<const float2*>(rec + kSepK) + p;
    uint32_t re_hi[4], re_lo[4], re_c[4], im_hi[4], im_lo[4], im_c[4];
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      float xr[2], xi[2], dp[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int k = 8 * g + 2 * h + e;
        const float4 prm = rec[k];
        const float2 v = val[4 * k];
        float s, c;
        __sincosf(sep_phase(__float_as_int(prm.x), i_off, prm.z, fit_a), &s, &c);
        xr[e] = v.x * c - v.y * s;
        xi[e] = v.x * s + v.y * c;
        dp[e] = prm.z * fit_p;
      }
      const __half2 d = __floats2half2_rn(dp[0], dp[1]);
      re_c[h] = h2_bits(__hmul2(sep_split(xr[0], xr[1], re_hi[h], re_lo[h]), d));
      im_c[h] = h2_bits(__hmul2(sep_split(xi[0], xi[1], im_hi[h], im_lo[h]), d));
    }
    const uint32_t dst = buf + g * 2048 + (p * 32 + lane) * 16;
    sts128(dst, re_hi);
    sts128(dst + 4096, im_hi);
    sts128(dst + 2 * 4096, re_lo);
    sts128(dst + 3 * 4096, im_lo);
    sts128(dst + 4 * 4096, re_c);
    sts128(dst + 5 * 4096, im_c);
  }
  if (tid < 2 * L) {
    const int g = tid / L, j = tid - g * L;
    const __half2 q2 = __float2half2_rn(fit_q), mq2 = __float2half2_rn(-fit_q);
    SepF f;
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      float c[2], s[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float4 prm = rec[8 * g + 2 * h + e];
        __sincosf(sep_phase(__float_as_int(prm.y), j_off, prm.z, fit_b), &s[e], &c[e]);
      }
      const __half2 hc = sep_split(c[0], c[1], f.r_hi[h], f.r_lo[h]);
      const __half2 hs = sep_split(s[0], s[1], f.i_hi[h], f.i_lo[h]);
      f.r_c[h] = h2_bits(__hmul2(hs, mq2));  // i q F
      f.i_c[h] = h2_bits(__hmul2(hc, q2));
    }
    sep_store_f(f, buf + C::kABytes + g * C::kFGroup + j * 16, C::kFBlock, C::kFLevel);
  }
}

// the chunk's MMAs (one thread), first: the segment's first chunk
template <int L>
__device__ __forceinline__ void gsep_issue(uint32_t buf, uint32_t d, bool first) {
  using C = Gsep<L>;
  constexpr uint32_t idesc = sep_idesc(C::kN);
  const uint32_t f = buf + C::kABytes;
  // (E level, F level): lo hi, hi lo, first order, hi hi
  const uint32_t el[4] = {1, 0, 2, 0}, fl[4] = {0, 1, 2, 0};
#pragma unroll
  for (int n = 0; n < 4; ++n) {
    const uint32_t ea = buf + el[n] * 8192, fa = f + fl[n] * C::kFLevel;
    sep_mma(d, sep_desc(ea, 2048), sep_desc(fa + C::kFBlock, C::kFGroup), idesc, (first && n == 0) ? 0u : 1u);
    sep_mma(d, sep_desc(ea + 4096, 2048), sep_desc(fa, C::kFGroup), idesc, 1u);
  }
}

__device__ __forceinline__ int gsep_chunks(const SegmentDesc& d) { return (d.k_end - d.k_begin + kSepK - 1) / kSepK; }

// items first, first + stride, ... below last, producers' side
template <int L>
__device__ __forceinline__ void gsep_producer(const GridArgs& a, int first, int last, int stride, int nbuf,
                                              unsigned char* ring, GsepTail& S) {
  using C = Gsep<L>;
  const int tid = threadIdx.x, lane = tid & 31;
  const int j = tid < 2 * L ? tid % L : 0;
  const float fit_b = a.sep.b[j], fit_q = a.sep.q[j];
  const uint32_t ring0 = smem_u32(ring);
  uint32_t cg = 0, sc = 0;  // chunks and segments of this block so far
  int slot = 0;             // cg % nbuf
  uint32_t turn = 0;        // cg / nbuf
  for (int idx = first; idx < last; idx += stride) {
    const GridItem item = a.items[idx];
    const SubgridDesc sd = a.sg[item.sg];
    const int i = item.tile * kGsepColumns + lane;
    const float fit_a = a.sep.a[i], fit_p = a.sep.p[i];
    const float4* recs = a.records + size_t(sd.rec_offset) * kRecordFloat4;
    int total = 0;
    for (int s = 0; s < sd.seg_count; ++s) total += gsep_chunks(a.seg[sd.seg_begin + s]);
    int s = 0, c_in = 0, n_in = gsep_chunks(a.seg[sd.seg_begin]);
    if (tid < kGsepChunkFloat4) S.rec[cg & 1][tid] = __ldg(recs + tid);
    half_sync(kSepProducerBar);
    for (int c = 0; c < total; ++c) {
      float4 nxt;
      const bool more = c + 1 < total && tid < kGsepChunkFloat4;
      if (more) nxt = __ldg(recs + size_t(c + 1) * kGsepChunkFloat4 + tid);
      if (turn > 0) sep_wait(&S.empty[slot], (turn - 1) & 1, &S.fail, a.status);
      const uint32_t buf = ring0 + slot * C::kBufBytes;
      gsep_produce<L>(buf, S.rec[cg & 1], i - L / 2, fit_a, fit_p, j - L / 2, fit_b, fit_q);
      if (more) S.rec[(cg + 1) & 1][tid] = nxt;
      fence_proxy_async();
      half_sync(kSepProducerBar);
      const bool last_c = c_in + 1 == n_in;
      if (tid == 0) {
        // the accumulator's previous segment (two back) has been read
        if (c_in == 0 && sc >= 2) sep_wait(&S.drained[sc & 1], ((sc >> 1) - 1) & 1, &S.fail, a.status);
        tc_fence_after();
        gsep_issue<L>(buf, S.tmem + (sc & 1) * C::kColStride, c_in == 0);
        sep_commit(&S.empty[slot]);
        if (last_c) sep_commit(&S.full[sc & 1]);
      }
      ++cg;
      if (++slot == nbuf) {
        slot = 0;
        ++turn;
      }
      ++c_in;
      if (last_c) {
        ++sc;
        ++s;
        c_in = 0;
        if (c + 1 < total) n_in = gsep_chunks(a.seg[sd.seg_begin + s]);
      }
    }
  }
}

// consumers' side: thread = column i of the tile x one row pair of every 16 rows
template <int L>
__device__ __forceinline__ void gsep_consumer(const GridArgs& a, int first, int last, int stride, GsepTail& S,
                                              float4* R) {
  using C = Gsep<L>;
  const int warp = (threadIdx.x >> 5) - kSepHalf / 32, lane = threadIdx.x & 31;
  const int nodes = a.g.nodes, nA = nodes * nodes * 4;
  const int pol = warp & 3, cgp = warp >> 2;
  const uint32_t d0 = S.tmem + (uint32_t(pol * 32) << 16) + 8 * cgp;
  uint32_t sc = 0;  // segments of this block so far
  for (int idx = first; idx < last; idx += stride) {
    const GridItem item = a.items[idx];
    const SubgridDesc sd = a.sg[item.sg];
    const int i = item.tile * kGsepColumns + lane;
    const NodeWeight wx = node_weight(i, nodes, L);
    const float4* rec = a.records + size_t(sd.rec_offset) * kRecordFloat4;  // first chunk of the segment
    c2 acc[C::kSteps][4];
#pragma unroll
    for (int st = 0; st < C::kSteps; ++st)
#pragma unroll
      for (int p = 0; p < 4; ++p) acc[st][p] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};

    for (int s = 0; s < sd.seg_count; ++s, ++sc) {
      const SegmentDesc seg = a.seg[sd.seg_begin + s];
      const int sp = seg.interval * a.g.n_st + sd.p, sq = seg.interval * a.g.n_st + sd.q;
      const bool diag = a.adiag[sp] && a.adiag[sq];
      const float inv = __ldg(&rec[0].w);  // 1 / scale of the segment's values, undone on the p side
      rec += size_t(gsep_chunks(seg)) * kGsepChunkFloat4;
      half_sync(kSepConsumerBar);  // A-term rows and transpose buffers free
      // A-terms interpolated along i at every node row: [row][p (2 float4), q (2 float4)][32]
      for (int e = warp; e < 2 * nodes; e += kSepHalf / 32) {
        const int r = e >> 1, st = e & 1;
        const float4* n0 = reinterpret_cast<const float4*>(a.aterms + size_t(st ? sq : sp) * nA +
                                                           (size_t(r) * nodes + wx.a) * 4);
        const float k1 = st ? wx.f : wx.f * inv, k0 = st ? 1.f - wx.f : (1.f - wx.f) * inv;
        float4 v[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float4 x = __ldg(n0 + h), y = __ldg(n0 + 2 + h);
          v[h] = make_float4(k0 * x.x + k1 * y.x, k0 * x.y + k1 * y.y, k0 * x.z + k1 * y.z, k0 * x.w + k1 * y.w);
        }
        float4* dst = R + (r * 4 + 2 * st) * 32 + lane;
        dst[0] = diag ? make_float4(v[0].x, v[0].y, v[1].z, v[1].w) : v[0];
        if (!diag) dst[32] = v[1];
      }
      sep_wait(&S.full[sc & 1], (sc >> 1) & 1, &S.fail, a.status);
      tc_fence_after();
      const uint32_t d = d0 + (sc & 1) * C::kColStride;
#pragma unroll
      for (int st = 0; st < C::kSteps; ++st) {
        float re[8], im[8];
        tmem_ld8(re, d + 16 * st);
        tmem_ld8(im, d + L + 16 * st);
        tmem_wait_ld();
        if (st + 1 == C::kSteps) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&S.drained[sc & 1]);
        }
        float2* xw = S.x[st & 1] + pol * 512 + 4 * cgp * 32 + lane;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          xw[e * 32] = make_float2(re[2 * e], re[2 * e + 1]);
          xw[256 + e * 32] = make_float2(im[2 * e], im[2 * e + 1]);
        }
        half_sync(kSepConsumerBar);
        const int j = 16 * st + 2 * warp;
        const float2* xr = S.x[st & 1] + warp * 32 + lane;
        c2 X[4];
#pragma unroll
        for (int p = 0; p < 4; ++p) X[p] = {xr[p * 512], xr[p * 512 + 256]};
        const NodeWeight w0 = node_weight(j, nodes, L), w1 = node_weight(j + 1, nodes, L);
        // entries (2h, 2h+1) of matrix m at both rows; n: minus the imaginary part
        c2 e[2];
        float2 n[2];
        auto lerp = [&](int w) {
          const float4* r0 = R + (w0.a * 4 + w) * 32 + lane;
          float4 u = r0[0], v = r0[128];
          float4 dl = make_float4(v.x - u.x, v.y - u.y, v.z - u.z, v.w - u.w);
          e[0].re.x = fmaf(w0.f, dl.x, u.x);
          e[0].im.x = fmaf(w0.f, dl.y, u.y);
          n[0].x = fmaf(-w0.f, dl.y, -u.y);
          e[1].re.x = fmaf(w0.f, dl.z, u.z);
          e[1].im.x = fmaf(w0.f, dl.w, u.w);
          n[1].x = fmaf(-w0.f, dl.w, -u.w);
          if (w1.a != w0.a) {  // the pair straddles a node row (the same for the whole warp)
            u = v;
            v = r0[256];
            dl = make_float4(v.x - u.x, v.y - u.y, v.z - u.z, v.w - u.w);
          }
          e[0].re.y = fmaf(w1.f, dl.x, u.x);
          e[0].im.y = fmaf(w1.f, dl.y, u.y);
          n[0].y = fmaf(-w1.f, dl.y, -u.y);
          e[1].re.y = fmaf(w1.f, dl.z, u.z);
          e[1].im.y = fmaf(w1.f, dl.w, u.w);
          n[1].y = fmaf(-w1.f, dl.w, -u.w);
        };
        // t = conj(x) y [+ t], nx = -Im x;  t += x y
        auto conj_mul = [](const c2& x, float2 nx, const c2& y) {
          return c2{ffma2(x.im, y.im, fmul2(x.re, y.re)), ffma2(nx, y.re, fmul2(x.re, y.im))};
        };
        auto mul_add = [](const c2& x, float2 nx, const c2& y, c2& t) {
          t.re = ffma2(nx, y.im, ffma2(x.re, y.re, t.re));
          t.im = ffma2(x.im, y.re, ffma2(x.re, y.im, t.im));
        };
        if (diag) {  // conj(p_a) X_ab q_b
          c2 t[4];
          lerp(0);
#pragma unroll
          for (int b = 0; b < 2; ++b) {
            t[b] = conj_mul(e[0], n[0], X[b]);
            t[2 + b] = conj_mul(e[1], n[1], X[2 + b]);
          }
          lerp(2);
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            mul_add(e[0], n[0], t[2 * r], acc[st][2 * r]);
            mul_add(e[1], n[1], t[2 * r + 1], acc[st][2 * r + 1]);
          }
        } else {  // A_p^H (X A_q): rows 0 and 1 of A_q, then of A_p
          c2 m[4];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            lerp(2 + h);
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
              for (int b = 0; b < 2; ++b) {
                c2& t = m[2 * r + b];
                if (h == 0) t = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                mul_add(e[b], n[b], X[2 * r + h], t);
              }
          }
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            lerp(h);
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
              for (int b = 0; b < 2; ++b) {
                c2& t = acc[st][2 * r + b];
                const c2& y = m[2 * h + b];
                t.re = ffma2(e[r].im, y.im, ffma2(e[r].re, y.re, t.re));
                t.im = ffma2(n[r], y.re, ffma2(e[r].re, y.im, t.im));
              }
          }
        }
      }
    }

    // ---- pixels of the item: w_ref, taper, centring sign; [sg][pol][j][i]; Stokes I: plane 0, (XX + YY) / 2
    const float w_ref = a.w_ref[item.sg];
    const float ti = a.taper[i];
#pragma unroll
    for (int st = 0; st < C::kSteps; ++st) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int j = 16 * st + 2 * warp + h;
        const float2 ph = sep_w_phasor(w_ref, __ldg(a.sep.n1 + j * L + i));
        const float wgt = ti * a.taper[j] * (((i + j) & 1) ? -1.f : 1.f);
        const cf rot = {wgt * ph.x, wgt * ph.y};
        float2* dst = a.scratch + size_t(item.sg) * 4 * L * L + j * L + i;
        cf v[4];
#pragma unroll
        for (int p = 0; p < 4; ++p)
          v[p] = h ? cf{acc[st][p].re.y, acc[st][p].im.y} : cf{acc[st][p].re.x, acc[st][p].im.x};
        if (a.g.npol == 1) {
          const cf x = cmul(rot, cf{0.5f * (v[0].re + v[3].re), 0.5f * (v[0].im + v[3].im)});
          dst[0] = make_float2(x.re, x.im);
        } else {
#pragma unroll
          for (int p = 0; p < 4; ++p) {
            const cf x = cmul(rot, v[p]);
            dst[size_t(p) * L * L] = make_float2(x.re, x.im);
          }
        }
      }
    }
  }
}

template <int L>
__device__ __forceinline__ void gridder_sep_block(const GridArgs& a, int first, int last, int stride, int nbuf,
                                                  unsigned char* smem) {
  using C = Gsep<L>;
  GsepTail& S = *reinterpret_cast<GsepTail*>(smem + size_t(nbuf) * C::kBufBytes);
  float4* R = reinterpret_cast<float4*>(&S + 1);
  if (threadIdx.x == 0) {
    for (int k = 0; k < nbuf; ++k) mbar_init(&S.empty[k], 1);
    for (int k = 0; k < 2; ++k) {
      mbar_init(&S.full[k], 1);
      mbar_init(&S.drained[k], kSepHalf / 32);
    }
    fence_mbar_init();
    S.fail = 0;
  }
  if (threadIdx.x < 32) tmem_alloc(&S.tmem, C::kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (threadIdx.x < kSepHalf) {
    regs_give<256 - C::kConsumerRegs>();
    gsep_producer<L>(a, first, last, stride, nbuf, smem, S);
  } else {
    regs_take<C::kConsumerRegs>();
    gsep_consumer<L>(a, first, last, stride, S, R);
  }
  // after a wait that gave up: one more bounded wait for MMAs that may still run before their memory goes
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x < 32) {
    if (*reinterpret_cast<volatile int*>(&S.fail) && threadIdx.x == 0) {
      sep_commit(&S.full[0]);
      mbar_wait_bounded(&S.full[0], 0);
    }
    __syncwarp();
    tc_fence_after();
    tmem_free(S.tmem, C::kTmemCols);
  }
}

template <int L>
__global__ void __launch_bounds__(kSepThreads, 1) gridder_sep_kernel(const GridArgs a, int nbuf, int bundle) {
  extern __shared__ __align__(128) unsigned char sep_smem[];
  const int b = blockIdx.x;
  if (bundle > 0)  // neighbouring items (tiles of one subgrid)
    gridder_sep_block<L>(a, b * bundle, imin((b + 1) * bundle, a.n_items), 1, nbuf, sep_smem);
  else             // persistent: every gridDim-th item of the longest-first list
    gridder_sep_block<L>(a, b, a.n_items, gridDim.x, nbuf, sep_smem);
}

// One launch over the items of several plans (items = (plan slot, item index))
template <int L>
__global__ void __launch_bounds__(kSepThreads, 1) gridder_sep_multi_kernel(const GridArgs* args, const int2* items,
                                                                          int nbuf) {
  extern __shared__ __align__(128) unsigned char sep_smem[];
  __shared__ __align__(16) unsigned char s_args_raw[sizeof(GridArgs)];
  const int2 it = items[blockIdx.x];
  if (threadIdx.x == 0) memcpy(s_args_raw, args + it.x, sizeof(GridArgs));
  __syncthreads();
  gridder_sep_block<L>(*reinterpret_cast<const GridArgs*>(s_args_raw), it.y, it.y + 1, 1, nbuf, sep_smem);
}

template <int L>
int configure_gridder_sep_l(int* persistent_blocks) {
  cudaError_t e = cudaFuncSetAttribute(gridder_sep_kernel<L>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kSepSmemLimit);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(gridder_sep_multi_kernel<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSepSmemLimit);
  int dev = 0, sms = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  *persistent_blocks = sms;  // 512 threads of up to 128 registers: one block per SM
  return int(e);
}

template <int L>
int launch_gridder_sep_l(const GridArgs& a, int n_items, int persistent_blocks, int bundle, void* stream) {
  if (n_items <= 0) return 0;
  const int nb = gsep_buffers<L>(a.g.nodes);
  const int blocks = persistent_blocks > 0 ? (persistent_blocks < n_items ? persistent_blocks : n_items)
                                           : (n_items + bundle - 1) / bundle;
  gridder_sep_kernel<L><<<blocks, kSepThreads, gsep_smem<L>(nb, a.g.nodes), cudaStream_t(stream)>>>(
      a, nb, persistent_blocks > 0 ? 0 : bundle);
  return int(cudaGetLastError());
}

template <int L>
int launch_gridder_sep_multi_l(const GridArgs* args, const int2* items, int n_items, int max_nodes, void* stream) {
  if (n_items <= 0) return 0;
  const int nb = gsep_buffers<L>(max_nodes);
  gridder_sep_multi_kernel<L><<<n_items, kSepThreads, gsep_smem<L>(nb, max_nodes), cudaStream_t(stream)>>>(args, items,
                                                                                                        nb);
  return int(cudaGetLastError());
}

}  // namespace idg
