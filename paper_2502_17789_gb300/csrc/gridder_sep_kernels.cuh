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
// One block of 512 threads per item (subgrid, 32 columns).  Chunks of 16
// visibilities: threads 0-255 write the E side (thread = row (p, i) x 8
// visibilities), the others the F side (thread = row j x 8 visibilities), into
// a ring of 2-4 chunk buffers; one thread issues the chunk's 8 MMAs, whose
// commit frees the buffer.  The accumulator alternates between two column
// ranges of tensor memory from segment to segment, so the epilogue of a
// segment (tensor memory -> shared memory transpose -> A_p^H X A_q, added to
// the thread's pixels in registers) overlaps the MMAs of the next one.  w_ref,
// taper and centring sign are applied once, when the item's pixels are
// written.
//
// Measured (GB300, MWA-like workload, 96 x 96 subgrids, segments of about 60
// visibilities, per grid call): 29.0 ms, against 81.7 ms of the kernel with
// one phasor per visibility and pixel (gridder_tc_kernels.cuh); grid error
// 9e-7 against 2.2e-6.
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
};

// per-block state after the chunk ring: two transpose buffers, the chunk records, the interpolated A-terms
struct GsepTail {
  float2 x[2][4 * 512];     // [buffer][pol][row of 16][column of 32]
  float4 rec[2][kGsepChunkFloat4];
  uint64_t bar[4];          // one per chunk buffer
  uint32_t tmem;
  int fail;
  int item;
  float inv_scale[2];       // by segment parity
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

template <int L>
struct GsepItem {
  using C = Gsep<L>;
  const GridArgs& a;
  unsigned char* ring;     // chunk buffers
  GsepTail& S;
  float4* R;               // [node row][p 0/1, q 0/1][32] x-interpolated A-terms of the segment
  const int nbuf;
  uint32_t cg;             // chunks of this block so far (ring position and parity)

  // wait until the chunk `c` (counted over the block's life) has left its buffer / reached tensor memory
  __device__ __forceinline__ void wait_chunk(uint32_t c) {
    if (*reinterpret_cast<volatile int*>(&S.fail)) return;
    if (!mbar_wait_bounded(&S.bar[c % nbuf], (c / nbuf) & 1)) {
      atomicOr(a.status, kStatusTimeout);
      *reinterpret_cast<volatile int*>(&S.fail) = 1;
    }
  }

  // E side rows (p, i) and F side rows j of one chunk
  __device__ __forceinline__ void produce(uint32_t buf, const float4* rec, int i_off, float fit_a, float fit_p,
                                          int j_off, float fit_b, float fit_q) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid < 256) {
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
    } else if (tid - 256 < 2 * L) {
      const int g = (tid - 256) / L, j = (tid - 256) - g * L;
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
  __device__ __forceinline__ void issue(uint32_t buf, uint32_t d, bool first, uint64_t* bar) {
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
    sep_commit(bar);
  }

  __device__ __forceinline__ bool run(int item_idx) {
    const GridItem item = a.items[item_idx];
    const SubgridDesc sd = a.sg[item.sg];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nodes = a.g.nodes, nA = nodes * nodes * 4;
    const int i = item.tile * 32 + lane;     // this thread's pixel column (E side and epilogue)
    const int jf = (tid - 256) % L;          // this thread's row of the F side (tid >= 256)
    const bool fside = tid >= 256;
    const float fit_a = a.sep.a[i], fit_p = a.sep.p[i];
    const float fit_b = fside ? a.sep.b[jf] : 0.f, fit_q = fside ? a.sep.q[jf] : 0.f;
    const float4* recs = a.records + size_t(sd.rec_offset) * kRecordFloat4;
    const uint32_t ring0 = smem_u32(ring);
    const NodeWeight wx = node_weight(i, nodes, L);

    int total = 0;
    for (int s = 0; s < sd.seg_count; ++s) {
      const SegmentDesc d = a.seg[sd.seg_begin + s];
      total += (d.k_end - d.k_begin + kSepK - 1) / kSepK;
    }

    cf acc[C::kSteps][4];
#pragma unroll
    for (int s = 0; s < C::kSteps; ++s)
#pragma unroll
      for (int p = 0; p < 4; ++p) acc[s][p] = {0.f, 0.f};

    // A_p^H X A_q of segment `s` (its last chunk is `last`) added to acc
    auto epilogue = [&](int s, uint32_t last) {
      const SegmentDesc seg = a.seg[sd.seg_begin + s];
      const float2* Ap = a.aterms + (size_t(seg.interval) * a.g.n_st + sd.p) * nA;
      const float2* Aq = a.aterms + (size_t(seg.interval) * a.g.n_st + sd.q) * nA;
      const bool diag = a.adiag[seg.interval * a.g.n_st + sd.p] && a.adiag[seg.interval * a.g.n_st + sd.q];
      // A-terms interpolated along i at every node row (the scale of the values undone on the p side)
      const float inv = S.inv_scale[s & 1];
      for (int r = warp; r < nodes; r += kSepThreads / 32) {
#pragma unroll
        for (int st = 0; st < 2; ++st) {
          const float4* n0 = reinterpret_cast<const float4*>((st ? Aq : Ap) + (size_t(r) * nodes + wx.a) * 4);
          const float k1 = st ? wx.f : wx.f * inv, k0 = st ? 1.f - wx.f : (1.f - wx.f) * inv;
          float4 e[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const float4 u = __ldg(n0 + h), v = __ldg(n0 + 2 + h);
            e[h] = make_float4(k0 * u.x + k1 * v.x, k0 * u.y + k1 * v.y, k0 * u.z + k1 * v.z, k0 * u.w + k1 * v.w);
          }
          if (diag) {
            R[(r * 4 + 2 * st) * 32 + lane] = make_float4(e[0].x, e[0].y, e[1].z, e[1].w);
          } else {
            R[(r * 4 + 2 * st) * 32 + lane] = e[0];
            R[(r * 4 + 2 * st + 1) * 32 + lane] = e[1];
          }
        }
      }
      wait_chunk(last);
      tc_fence_after();
      const int pol = warp & 3, cgp = warp >> 2;
      const uint32_t d = S.tmem + (uint32_t(pol * 32) << 16) + (s & 1) * C::kColStride + 4 * cgp;
#pragma unroll
      for (int st = 0; st < C::kSteps; ++st) {
        float re[4], im[4];
        tmem_ld4(re, d + 16 * st);
        tmem_ld4(im, d + L + 16 * st);
        tmem_wait_ld();
        float2* xw = S.x[st & 1] + pol * 512 + 4 * cgp * 32 + lane;
#pragma unroll
        for (int e = 0; e < 4; ++e) xw[e * 32] = make_float2(re[e], im[e]);
        __syncthreads();
        const int j = 16 * st + warp;
        const float2* xr = S.x[st & 1] + warp * 32 + lane;
        Jones X;
#pragma unroll
        for (int p = 0; p < 4; ++p) X.m[p] = {xr[p * 512].x, xr[p * 512].y};
        const NodeWeight wy = node_weight(j, nodes, L);
        const float4* r0 = R + wy.a * 128 + lane;
        auto lerp = [&](int w) {
          const float4 u = r0[w * 32], v = r0[128 + w * 32];
          return make_float4(fmaf(wy.f, v.x - u.x, u.x), fmaf(wy.f, v.y - u.y, u.y), fmaf(wy.f, v.z - u.z, u.z),
                             fmaf(wy.f, v.w - u.w, u.w));
        };
        Jones E;
        if (diag) {
          const float4 p4 = lerp(0), q4 = lerp(2);
          E = jdiag_ah_x_b(JonesDiag{{p4.x, p4.y}, {p4.z, p4.w}}, X, JonesDiag{{q4.x, q4.y}, {q4.z, q4.w}});
        } else {
          const float4 pa = lerp(0), pb = lerp(1), qa = lerp(2), qb = lerp(3);
          const Jones P = {{{pa.x, pa.y}, {pa.z, pa.w}, {pb.x, pb.y}, {pb.z, pb.w}}};
          const Jones Q = {{{qa.x, qa.y}, {qa.z, qa.w}, {qb.x, qb.y}, {qb.z, qb.w}}};
          E = jmul_ah(P, jmul(X, Q));
        }
#pragma unroll
        for (int p = 0; p < 4; ++p) acc[st][p] = cadd(acc[st][p], E.m[p]);
      }
      tc_fence_before();  // the accumulator is free once every thread has passed the next barrier
    };

    // records of the first chunk
    if (tid < kGsepChunkFloat4) S.rec[cg & 1][tid] = __ldg(recs + tid);
    __syncthreads();

    int s = 0, c_in = 0;  // segment of the current chunk, its index there
    int n_in = 0;         // chunks of segment s
    {
      const SegmentDesc d = a.seg[sd.seg_begin];
      n_in = (d.k_end - d.k_begin + kSepK - 1) / kSepK;
    }
    for (int c = 0; c < total; ++c) {
      const uint32_t cc = cg + uint32_t(c);
      float4 nxt;
      const bool more = c + 1 < total && tid < kGsepChunkFloat4;
      if (more) nxt = __ldg(recs + size_t(c + 1) * kGsepChunkFloat4 + tid);
      if (cc >= uint32_t(nbuf)) wait_chunk(cc - nbuf);
      const uint32_t buf = ring0 + (cc % nbuf) * C::kBufBytes;
      produce(buf, S.rec[cc & 1], i - L / 2, fit_a, fit_p, jf - L / 2, fit_b, fit_q);
      if (c_in == 0 && tid == 0) S.inv_scale[s & 1] = S.rec[cc & 1][0].w;
      if (more) S.rec[(cc + 1) & 1][tid] = nxt;
      fence_proxy_async();
      __syncthreads();
      if (tid == 0) {
        tc_fence_after();
        issue(buf, S.tmem + (s & 1) * C::kColStride, c_in == 0, &S.bar[cc % nbuf]);
      }
      // the previous segment's epilogue, behind as many chunks of this one as fit the ring beside its last chunk
      if (s > 0 && c_in == (n_in < nbuf - 1 ? n_in : nbuf - 1) - 1) epilogue(s - 1, cc - uint32_t(c_in) - 1);
      if (++c_in == n_in && c + 1 < total) {
        ++s;
        c_in = 0;
        const SegmentDesc d = a.seg[sd.seg_begin + s];
        n_in = (d.k_end - d.k_begin + kSepK - 1) / kSepK;
      }
    }
    __syncthreads();  // S.inv_scale of the last segment, S.x of an epilogue just before
    epilogue(s, cg + uint32_t(total) - 1);
    cg += uint32_t(total);

    // ---- pixels of the item: w_ref, taper, centring sign; [sg][pol][j][i]; Stokes I: plane 0, (XX + YY) / 2
    const float w_ref = a.w_ref[item.sg];
    const float ti = a.taper[i];
#pragma unroll
    for (int st = 0; st < C::kSteps; ++st) {
      const int j = 16 * st + warp;
      const float2 ph = sep_w_phasor(w_ref, __ldg(a.sep.n1 + j * L + i));
      const float wgt = ti * a.taper[j] * (((i + j) & 1) ? -1.f : 1.f);
      const cf rot = {wgt * ph.x, wgt * ph.y};
      float2* dst = a.scratch + size_t(item.sg) * 4 * L * L + j * L + i;
      if (a.g.npol == 1) {
        const cf v = cmul(rot, cf{0.5f * (acc[st][0].re + acc[st][3].re), 0.5f * (acc[st][0].im + acc[st][3].im)});
        dst[0] = make_float2(v.re, v.im);
      } else {
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          const cf v = cmul(rot, acc[st][p]);
          dst[size_t(p) * L * L] = make_float2(v.re, v.im);
        }
      }
    }
    return !*reinterpret_cast<volatile int*>(&S.fail);
  }
};

// block set-up: barriers and tensor memory; items either one per block or drained from a queue
template <int L, bool PERSIST>
__device__ __forceinline__ void gridder_sep_block(const GridArgs& a, int first_item, int nbuf, unsigned char* smem) {
  using C = Gsep<L>;
  GsepTail& S = *reinterpret_cast<GsepTail*>(smem + size_t(nbuf) * C::kBufBytes);
  float4* R = reinterpret_cast<float4*>(&S + 1);
  if (threadIdx.x == 0) {
    for (int k = 0; k < nbuf; ++k) mbar_init(&S.bar[k], 1);
    fence_mbar_init();
    S.fail = 0;
  }
  if (threadIdx.x < 32) tmem_alloc(&S.tmem, C::kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  GsepItem<L> it{a, smem, S, R, nbuf, 0};
  if constexpr (!PERSIST) {
    it.run(first_item);
  } else {
    for (;;) {
      if (threadIdx.x == 0) S.item = atomicAdd(a.queue, 1);
      __syncthreads();
      const int idx = S.item;
      if (idx >= a.n_items || !it.run(idx)) break;
      __syncthreads();  // S.item and the transpose buffers free for the next item
    }
  }
  // a wait that gave up: give the MMAs in flight one more bounded wait before their memory goes
  if (*reinterpret_cast<volatile int*>(&S.fail) && it.cg > 0)
    mbar_wait_bounded(&S.bar[(it.cg - 1) % nbuf], ((it.cg - 1) / nbuf) & 1);
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x < 32) {
    tc_fence_after();
    tmem_free(S.tmem, C::kTmemCols);
  }
}

template <int L, bool PERSIST>
__global__ void __launch_bounds__(kSepThreads, 1) gridder_sep_kernel(const GridArgs a, int nbuf) {
  extern __shared__ __align__(128) unsigned char sep_smem[];
  gridder_sep_block<L, PERSIST>(a, blockIdx.x, nbuf, sep_smem);
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
  gridder_sep_block<L, false>(*reinterpret_cast<const GridArgs*>(s_args_raw), it.y, nbuf, sep_smem);
}

template <int L>
int configure_gridder_sep_l(int* persistent_blocks) {
  cudaError_t e = cudaFuncSetAttribute(gridder_sep_kernel<L, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kSepSmemLimit);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(gridder_sep_kernel<L, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSepSmemLimit);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(gridder_sep_multi_kernel<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSepSmemLimit);
  int dev = 0, sms = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  *persistent_blocks = sms;  // 512 threads of up to 128 registers: one block per SM
  return int(e);
}

template <int L>
int launch_gridder_sep_l(const GridArgs& a, int n_items, int persistent_blocks, void* stream) {
  if (n_items <= 0) return 0;
  const int nb = gsep_buffers<L>(a.g.nodes);
  const size_t smem = gsep_smem<L>(nb, a.g.nodes);
  if (persistent_blocks > 0)
    gridder_sep_kernel<L, true><<<persistent_blocks < n_items ? persistent_blocks : n_items, kSepThreads, smem,
                                  cudaStream_t(stream)>>>(a, nb);
  else
    gridder_sep_kernel<L, false><<<n_items, kSepThreads, smem, cudaStream_t(stream)>>>(a, nb);
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
