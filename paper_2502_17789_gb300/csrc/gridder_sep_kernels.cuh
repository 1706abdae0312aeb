// Gridder with separable phasors (templates), included by the per-subgrid-size
// translation units gridder_sep_lNN.cu.  See sep_common.cuh for the split of
// the phase.
//
// Eq. 10's sum of one A-term segment over a tile of 32 pixel columns i and
// J rows j (J = L, 64 for L = 128) is a complex matrix product over the
// segment's visibilities,
//   X_p(i,j) = sum_k [V_{k,p} E_k(i)] F_k(j) (1 + 2 pi i delta_k p_i q_j):
// rows (p, i), 4 x 32 = 128, the height of one tcgen05 tile at every L;
// columns j, real and imaginary sums as two accumulators of J columns.
//
// A block of 512 threads works through a share of the items (subgrid, tile),
// split into two halves that run side by side.  Producers: per chunk of 16 visibilities
// every thread writes one row (p, i) x 8 visibilities of the E side to tensor
// memory and, of the F side, one row j x 8 visibilities to shared memory, in
// a ring of 2-4 chunks; one of them issues the chunk's 16 MMAs, whose commit
// frees the chunk.  Consumers: the accumulator alternates between two column
// ranges of tensor memory from segment to segment; while one fills, they take
// the other through a shared memory transpose (thread = row (p, i) to thread =
// column i x J / 8 neighbouring rows, all correlations), apply A_p^H X A_q with
// two rows at a time in packed f32x2 and add to their pixels in registers.
// w_ref, taper and centring sign are applied once, when the item's pixels are
// written.  The pixel sums need J registers of a consumer, so the halves
// split the block's registers unevenly.
//
// What bounds it: the latency of a chunk's chain (phasors, splits, the stores to
// tensor memory, a barrier) at 4 warps a scheduler, which the pixel sums'
// registers allow: 61 % of the issue slots, tensor pipe 38 % and shared-memory
// loads and stores 46 % busy (profiles/gridder_sep_mwa_like_90st.md).  With the E side in shared memory too, operands, their reads by the MMAs
// and a transpose per 16 rows kept shared memory 80 % busy (21.2 ms where that took
// 17.6); the E side in tensor memory costs none.  E's phasors computed once for the
// 4 correlations and passed through shared memory lengthen the chain (16.0 ms).
// Measured (GB300, MWA-like workload, 96 x 96 subgrids, segments of about 60
// visibilities, per grid call): 15.3 ms, against 81.7 ms of the kernel with one
// phasor per visibility and pixel (gridder_tc_kernels.cuh); grid error 5e-7
// against 2.2e-6.
#pragma once

#include <type_traits>

#include "sep_common.cuh"

namespace idg {

template <int L>
struct Gsep {
  static constexpr int kRows = gsep_rows(L);                     // J
  static constexpr int kColStride = 2 * kRows;                   // between the two accumulators (re, im)
  static constexpr int kECol = 2 * kColStride;                   // first column of the E side ring
  static constexpr int kRing = kRows > 64 ? 2 : 4;               // chunks: what tensor memory leaves beside the sums
  static constexpr uint32_t kTmemCols = 512;
  static constexpr uint32_t kFBlock = kRows * 16;                // Re or Im of one k group
  static constexpr uint32_t kFGroup = 2 * kFBlock;
  static constexpr uint32_t kFLevel = 2 * kFGroup;
  static constexpr uint32_t kBufBytes = 3 * kFLevel;
  static constexpr int kSpan = kRows / 8;                        // rows of a consumer thread
  static constexpr int kPairs = kSpan / 2;
  static constexpr int kConsumerRegs = kRows > 64 ? 184 : 160;   // the producers keep 256 less
  // How a producer gets the next chunk's record: with 72 registers by cp.async (a register held for it is spilled at
  // once, and the spill waits for the load: 16.0 -> 15.2 ms at L = 96), with 96 through registers (3.9 -> 3.8 ms at 64)
  static constexpr bool kAsyncRecord = kRows > 64;
  static_assert(kECol + kRing * 48 <= int(kTmemCols), "tensor memory");
};

// shared memory: F side ring, this, node samples of two segments
template <int L>
struct GsepShared {
  unsigned char ring[Gsep<L>::kRing * Gsep<L>::kBufBytes];
  float2 x[4][2][Gsep<L>::kRows / 2][32];  // [pol][re, im][row pair][column] of a segment's sums
  float4 rec[2][kGsepChunkFloat4];
  int part[2];               // [chunk parity] its place in its part: 1 first, 2 last
  uint64_t empty[4];         // chunk read by its MMAs
  uint64_t full[2];          // accumulator complete
  uint64_t drained[2];       // accumulator read by the 8 consumer warps
  uint64_t drain;            // every MMA complete, after a wait that gave up
  uint32_t tmem;
  int fail;
};
template <int L>
size_t gsep_smem(int nodes) {
  return sizeof(GsepShared<L>) + size_t(4) * nodes * nodes * 4 * sizeof(float2);
}
static_assert(sizeof(GsepShared<96>) + 4 * kMaxAtermNodes * kMaxAtermNodes * 32 <= size_t(kSepSmemLimit), "shared memory");

// E side row (p, i) and F side row j of one chunk (producer thread)
template <int L>
__device__ __forceinline__ void gsep_produce(uint32_t e_col, uint32_t buf, const float4* rec, int i_off, float fit_a,
                                             float fit_p, int j_off, float fit_b, float fit_q) {
  using C = Gsep<L>;
  const int tid = threadIdx.x, warp = tid >> 5;
  {
    const int p = warp & 3, g = warp >> 2;
    const float4* val = rec + 16 + 8 * p + 2 * g;
    uint32_t re_hi[4], re_lo[4], re_c[4], im_hi[4], im_lo[4], im_c[4];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const float4 fx = rec[2 * g + u], dl = rec[8 + 2 * g + u], vr = val[u], vi = val[4 + u];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int h = 2 * u + e;
        const float2 f = pair_of(fx, e), d = pair_of(dl, e);
        float2 c, s;
        sep_phasor2(__float_as_int(f.x), __float_as_int(f.y), i_off, d, fit_a, c, s);
        const __half2 d2 = __floats2half2_rn(d.x * fit_p, d.y * fit_p);
        const float2 r = pair_of(vr, e), m = pair_of(vi, e);
        re_c[h] = h2_bits(__hmul2(sep_split(make_float2(r.x * c.x - m.x * s.x, r.y * c.y - m.y * s.y), re_hi[h], re_lo[h]), d2));
        im_c[h] = h2_bits(__hmul2(sep_split(make_float2(r.x * s.x + m.x * c.x, r.y * s.y + m.y * c.y), im_hi[h], im_lo[h]), d2));
      }
    }
    const uint32_t dst = e_col + (uint32_t(p * 32) << 16) + 4 * g;
    tmem_st4(dst, re_hi);
    tmem_st4(dst + 8, im_hi);
    tmem_st4(dst + 16, re_lo);
    tmem_st4(dst + 24, im_lo);
    tmem_st4(dst + 32, re_c);
    tmem_st4(dst + 40, im_c);
  }
  if (tid < 2 * C::kRows) {
    const int g = tid / C::kRows, j = tid - g * C::kRows;
    const __half2 q2 = __float2half2_rn(fit_q), mq2 = __float2half2_rn(-fit_q);
    SepF f;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const float4 fx = rec[4 + 2 * g + u], dl = rec[8 + 2 * g + u];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int h = 2 * u + e;
        const float2 x = pair_of(fx, e);
        float2 c, s;
        sep_phasor2(__float_as_int(x.x), __float_as_int(x.y), j_off, pair_of(dl, e), fit_b, c, s);
        const __half2 hc = sep_split(c, f.r_hi[h], f.r_lo[h]);
        const __half2 hs = sep_split(s, f.i_hi[h], f.i_lo[h]);
        f.r_c[h] = h2_bits(__hmul2(hs, mq2));  // i q F
        f.i_c[h] = h2_bits(__hmul2(hc, q2));
      }
    }
    sep_store_f(f, buf + g * C::kFGroup + j * 16, C::kFBlock, C::kFLevel);
  }
}

__device__ __forceinline__ int gsep_chunks(const SegmentDesc& d) { return (d.k_end - d.k_begin + kSepK - 1) / kSepK; }
// A segment is summed in parts of up to kSepMaxChain chunks, each with its own accumulation and correction: chunks of
// the next part when `left` remain
__device__ __forceinline__ int gsep_part(int left) {
  const int parts = (left + kSepMaxChain - 1) / kSepMaxChain;
  return parts <= 1 ? left : (left + parts - 1) / parts;
}

// first column and row of an item's tile
template <int L>
__device__ __forceinline__ int2 gsep_origin(const GridItem& item) {
  constexpr int n = L / Gsep<L>::kRows;
  return make_int2(item.tile / n * kGsepColumns, item.tile % n * Gsep<L>::kRows);
}

// Producers' side.  What stands between two chunks is kept off their path: of the two warps without a part of F one
// issues the MMAs, the other keeps the segments (whose lengths come from global memory) and waits for the next
// chunk's place in the ring, which the barrier passes on to the others (per chunk at L = 96 some 150 and 100 of 2350
// clocks when every warp did both; 16.8 -> 16.0 ms, at L = 64 4.3 -> 3.8).
template <int L>
__device__ __forceinline__ void gsep_producer(const GridArgs& a, SepShare share, GsepShared<L>& S) {
  using C = Gsep<L>;
  const int tid = threadIdx.x, lane = tid & 31;
  // the producer warps with the least to write: one issues, one waits for places of the ring
  const bool issuer = uniform_warp() == kSepHalf / 32 - 1, waiter = uniform_warp() == kSepHalf / 32 - 2;
  const uint32_t ring0 = smem_u32(S.ring), tm = S.tmem;
  uint32_t cg = 0, sc = 0;  // chunks and segment parts of this block so far
  for (int idx = share.first; idx < share.last; idx = share.next(idx)) {
    const GridItem item = a.items[idx];
    const SubgridDesc sd = a.sg[item.sg];
    const int2 org = gsep_origin<L>(item);
    const int i = org.x + lane, j = org.y + tid % C::kRows;
    const float fit_a = a.sep.a[i], fit_p = a.sep.p[i], fit_b = a.sep.b[j], fit_q = a.sep.q[j];
    const float4* recs = a.records + size_t(sd.rec_offset) * kRecordFloat4;
    int total = 0;
    for (int s = 0; s < sd.seg_count; ++s) total += gsep_chunks(a.seg[sd.seg_begin + s]);
    int s = 0, left = gsep_chunks(a.seg[sd.seg_begin]);  // segment, its chunks not yet in a finished part
    int c_in = 0, n_in = gsep_part(left);                 // chunk of the part, its length
    if (tid < kGsepChunkFloat4) S.rec[cg & 1][tid] = __ldg(recs + tid);
    half_sync(kSepProducerBar);
    for (int c = 0; c < total; ++c) {
      // the next chunk's record
      float4 nxt;
      const bool more = c + 1 < total && tid < kGsepChunkFloat4;
      if (more) {
        const float4* src = recs + size_t(c + 1) * kGsepChunkFloat4 + tid;
        if (C::kAsyncRecord)
          cp_async16(&S.rec[(cg + 1) & 1][tid], src);
        else
          nxt = __ldg(src);
      }
      if (C::kAsyncRecord) cp_async_commit();
      const uint32_t slot = cg % C::kRing, turn = cg / C::kRing;
      if (turn > 0) tc_fence_after();
      const uint32_t buf = ring0 + slot * C::kBufBytes, e_col = tm + C::kECol + slot * 48;
      gsep_produce<L>(e_col, buf, S.rec[cg & 1], i - L / 2, fit_a, fit_p, j - L / 2, fit_b, fit_q);
      if (!C::kAsyncRecord && more) S.rec[(cg + 1) & 1][tid] = nxt;
      if (waiter) {
        const bool last_c = c_in + 1 == n_in;
        if (lane == 0) S.part[cg & 1] = int(c_in == 0) | int(last_c) << 1;
        ++c_in;
        if (last_c) {
          left -= n_in;
          c_in = 0;
          if (left == 0 && c + 1 < total) left = gsep_chunks(a.seg[sd.seg_begin + ++s]);
          n_in = gsep_part(left);
        }
        if (cg + 1 >= uint32_t(C::kRing))
          sep_wait(&S.empty[(cg + 1) % C::kRing], ((cg + 1) / C::kRing - 1) & 1, &S.fail, a);
      }
      if (C::kAsyncRecord) cp_async_wait<0>();
      tmem_wait_st();
      tc_fence_before();
      fence_proxy_async();
      half_sync(kSepProducerBar);
      if (issuer) {
        const int part = S.part[cg & 1];
        if (elect_one()) {
          // the accumulator's previous segment (two back) has been read
          if ((part & 1) && sc >= 2) sep_wait(&S.drained[sc & 1], ((sc >> 1) - 1) & 1, &S.fail, a);
          tc_fence_after();
          // also after a wait that gave up (the sums are lost then, but operands and accumulator are the block's own, and
          // sep_drain waits): a look at S.fail here costs 2 % at L = 64
          sep_product(tm + (sc & 1) * C::kColStride, e_col, buf, C::kRows, C::kFBlock, C::kFGroup, C::kFLevel, part & 1);
          sep_commit(&S.empty[slot]);
          if (part & 2) sep_commit(&S.full[sc & 1]);
        }
        sc += part >> 1;
      }
      ++cg;
    }
  }
}

// consumers' side: thread = column i of the tile x kSpan neighbouring rows
template <int L>
__device__ __forceinline__ void gsep_consumer(const GridArgs& a, SepShare share, GsepShared<L>& S, float4* raw) {
  using C = Gsep<L>;
  const int warp = (threadIdx.x >> 5) - kSepHalf / 32, lane = threadIdx.x & 31;
  const int nodes = a.g.nodes, n4 = nodes * nodes * 2;  // float4s of one station's samples
  const bool poller = uniform_warp() == kSepHalf / 32;
  // rows of a thread within one node cell: every cell starts at a multiple of kSpan rows
  const bool one_cell = L % (nodes - 1) == 0 && L / (nodes - 1) % C::kSpan == 0;
  uint32_t sc = 0;  // segment parts of this block so far
  for (int idx = share.first; idx < share.last; idx = share.next(idx)) {
    const GridItem item = a.items[idx];
    const SubgridDesc sd = a.sg[item.sg];
    const int2 org = gsep_origin<L>(item);
    const int i = org.x + lane, j0 = org.y + warp * C::kSpan;
    const NodeWeight wx = node_weight(i, nodes, L);
    // 1 / scale of the next segment's first chunk, for the correlation that the warp takes from tensor memory
    const float* rec = reinterpret_cast<const float*>(a.records + size_t(sd.rec_offset) * kRecordFloat4) + 48 + (warp & 3);
    cf acc[C::kSpan][4];
#pragma unroll
    for (int r = 0; r < C::kSpan; ++r)
#pragma unroll
      for (int p = 0; p < 4; ++p) acc[r][p] = {0.f, 0.f};

    // A-term samples of the item's next part (the block's part number c), on their way while another is worked on
    int diag_next = 0;
    float inv_next = 0.f;
    int s = 0, left = 0;                    // segments fetched, chunks of the last one not yet in a part
    SegmentDesc seg = a.seg[sd.seg_begin];  // of the part fetched next
    auto fetch = [&](uint32_t c) {
      const int sp = seg.interval * a.g.n_st + sd.p, sq = seg.interval * a.g.n_st + sd.q;
      float4* dst = raw + (c & 1) * 2 * n4;
      const float4* pp = reinterpret_cast<const float4*>(a.aterms) + size_t(sp) * n4;
      const float4* qq = reinterpret_cast<const float4*>(a.aterms) + size_t(sq) * n4;
      for (int e = threadIdx.x - kSepHalf; e < n4; e += kSepHalf) {
        cp_async16(dst + e, pp + e);
        cp_async16(dst + n4 + e, qq + e);
      }
      cp_async_commit();
      if (left == 0) left = gsep_chunks(seg);
      const int n = gsep_part(left);
      diag_next = a.adiag[sp] & a.adiag[sq];
      // the scale of the segment's values and the accumulation's bias, undone on the way to S.x
      inv_next = __ldg(rec) * sep_unbias(float(n));
      rec += size_t(n) * kGsepChunkFloat4 * 4;
      left -= n;
      if (left == 0 && ++s < sd.seg_count) seg = a.seg[sd.seg_begin + s];
    };
    half_sync(kSepConsumerBar);  // every thread is done with the previous item's samples
    fetch(sc);
    for (bool more = true; more; ++sc) {
      const bool diag = diag_next != 0;
      const float inv = inv_next;
      if (poller) sep_wait<100>(&S.full[sc & 1], (sc >> 1) & 1, &S.fail, a);
      half_sync(kSepConsumerBar);  // the segment's sums complete; S.x and the other samples free
      tc_fence_after();
      more = s < sd.seg_count;
      if (more) fetch(sc + 1);
      // sums of the part: tensor memory -> S.x; warp = correlation, half of the rows
      {
        const int pol = warp & 3, r0 = (warp >> 2) * (C::kRows / 2);
        const uint32_t d = S.tmem + (uint32_t(pol * 32) << 16) + (sc & 1) * C::kColStride + r0;
#pragma unroll
        for (int b = 0; b < C::kRows / 2; b += 16) {
          float re[16], im[16];
          tmem_ld16(re, d + b);
          tmem_ld16(im, d + C::kRows + b);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            S.x[pol][0][(r0 + b) / 2 + e][lane] = make_float2(re[2 * e] * inv, re[2 * e + 1] * inv);
            S.x[pol][1][(r0 + b) / 2 + e][lane] = make_float2(im[2 * e] * inv, im[2 * e + 1] * inv);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&S.drained[sc & 1]);
      }
      if (more)
        cp_async_wait<1>();
      else
        cp_async_wait<0>();
      half_sync(kSepConsumerBar);  // S.x and the samples of this segment visible

      // vector w of node row r interpolated along i: entries (0, 1), (2, 3) of p, then of q; of diagonal matrices
      // (0, 3) of p, then of q
      const float4* smp = raw + (sc & 1) * 2 * n4 + 2 * wx.a;
      auto row = [&](int r, int w, auto dtag) {
        constexpr bool DIAG = decltype(dtag)::value;
        const int st = DIAG ? w : w >> 1;
        const float4* n0 = smp + st * n4 + r * nodes * 2;
        const float k1 = wx.f, k0 = 1.f - wx.f;
        if constexpr (DIAG) {
          const float4 x0 = n0[0], x1 = n0[1], y0 = n0[2], y1 = n0[3];
          return make_float4(k0 * x0.x + k1 * y0.x, k0 * x0.y + k1 * y0.y, k0 * x1.z + k1 * y1.z, k0 * x1.w + k1 * y1.w);
        } else {
          const float4 x = n0[w & 1], y = n0[2 + (w & 1)];
          return make_float4(k0 * x.x + k1 * y.x, k0 * x.y + k1 * y.y, k0 * x.z + k1 * y.z, k0 * x.w + k1 * y.w);
        }
      };
      auto diff = [](const float4& v, const float4& u) {
        return make_float4(v.x - u.x, v.y - u.y, v.z - u.z, v.w - u.w);
      };
      // one_cell: the thread's rows lie in one node cell, so its rows are read once; otherwise the cell is followed
      // from row to row
      auto pixels = [&](auto dtag, auto one_cell) {
        constexpr int NV = decltype(dtag)::value ? 2 : 4;
        constexpr bool ONE = decltype(one_cell)::value;
        float4 u[4], dl[4];  // the node row below the pixel row and the step to the next
        auto load_cell = [&](int node) {
#pragma unroll
          for (int w = 0; w < NV; ++w) {
            u[w] = row(node, w, dtag);
            dl[w] = diff(row(node + 1, w, dtag), u[w]);
          }
        };
        // node cell and position of the next row; kept opaque so that the rows' values are not all held over the
        // segments (registers)
        const int step = nodes - 1;
        int jn = step * j0;
        asm volatile("" : "+r"(jn));
        int at = jn / L, rem = jn - at * L, node = -1;
        if (ONE) load_cell(at);
        auto next_row = [&]() {
          const NodeWeight w = {at, float(rem) * (1.f / float(L))};
          rem += step;
          if (!ONE && rem >= L) {
            rem -= L;
            ++at;
          }
          return w;
        };
#pragma unroll
        for (int st = 0; st < C::kPairs; ++st) {
          const NodeWeight w0 = next_row(), w1 = next_row();
          if (!ONE && w0.a != node) {  // the same for the whole warp
            node = w0.a;
            load_cell(node);
          }
          float2 xr[4], xi[4];
#pragma unroll
          for (int p = 0; p < 4; ++p) {
            xr[p] = S.x[p][0][warp * C::kPairs + st][lane];
            xi[p] = S.x[p][1][warp * C::kPairs + st][lane];
          }
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const NodeWeight wn = h ? w1 : w0;
            cf X[4];
#pragma unroll
            for (int p = 0; p < 4; ++p) X[p] = h ? cf{xr[p].y, xi[p].y} : cf{xr[p].x, xi[p].x};
            cf e[2];  // the two entries of vector w
            auto lerp = [&](int w) {
              float4 v = u[w], d = dl[w];
              if (!ONE && h == 1 && w1.a != w0.a) {  // a node row between the two
                v = row(w1.a, w, dtag);
                d = diff(row(w1.a + 1, w, dtag), v);
              }
              e[0] = {fmaf(wn.f, d.x, v.x), fmaf(wn.f, d.y, v.y)};
              e[1] = {fmaf(wn.f, d.z, v.z), fmaf(wn.f, d.w, v.w)};
            };
            auto mul_add = [](cf x, cf y, cf& t) {  // t += x y
              t.re = fmaf(-x.im, y.im, fmaf(x.re, y.re, t.re));
              t.im = fmaf(x.im, y.re, fmaf(x.re, y.im, t.im));
            };
            auto conj_mul_add = [](cf x, cf y, cf& t) {  // t += conj(x) y
              t.re = fmaf(x.im, y.im, fmaf(x.re, y.re, t.re));
              t.im = fmaf(-x.im, y.re, fmaf(x.re, y.im, t.im));
            };
            cf* o = acc[2 * st + h];
            if constexpr (decltype(dtag)::value) {  // conj(p_a) X_ab q_b
              cf t[4];
              lerp(0);
#pragma unroll
              for (int k = 0; k < 4; ++k) t[k] = cmulc(e[k >> 1], X[k]);
              lerp(1);
#pragma unroll
              for (int k = 0; k < 4; ++k) mul_add(t[k], e[k & 1], o[k]);
            } else {  // A_p^H (X A_q): by the rows of A_q, then of A_p
              cf m[4];
              lerp(2);
#pragma unroll
              for (int k = 0; k < 4; ++k) m[k] = cmul(X[k & 2], e[k & 1]);
              lerp(3);
#pragma unroll
              for (int k = 0; k < 4; ++k) mul_add(X[(k & 2) + 1], e[k & 1], m[k]);
#pragma unroll
              for (int r = 0; r < 2; ++r) {
                lerp(r);
#pragma unroll
                for (int k = 0; k < 4; ++k) conj_mul_add(e[k >> 1], m[2 * r + (k & 1)], o[k]);
              }
            }
          }
        }
      };
      if (one_cell) {
        if (diag)
          pixels(std::true_type{}, std::true_type{});
        else
          pixels(std::false_type{}, std::true_type{});
      } else if (diag) {
        pixels(std::true_type{}, std::false_type{});
      } else {
        pixels(std::false_type{}, std::false_type{});
      }
    }

    // ---- pixels of the item: w_ref, taper, centring sign; [sg][pol][j][i]; Stokes I: plane 0, (XX + YY) / 2
    const float2 w_ref = a.w_ref[item.sg];
    const float fit_p = a.sep.p[i];
    const float ti = a.taper[i];
#pragma unroll
    for (int r = 0; r < C::kSpan; ++r) {
      const int j = j0 + r;
      const float2 ph = sep_pixel(w_ref, __ldg(a.sep.n1 + j * L + i), fit_p * a.sep.q[j]);
      const float wgt = ti * a.taper[j] * (((i + j) & 1) ? -1.f : 1.f);
      const cf rot = {wgt * ph.x, wgt * ph.y};
      float2* dst = a.scratch + size_t(item.sg) * 4 * L * L + j * L + i;
      if (a.g.npol == 1) {
        const cf x = cmul(rot, cf{0.5f * (acc[r][0].re + acc[r][3].re), 0.5f * (acc[r][0].im + acc[r][3].im)});
        dst[0] = make_float2(x.re, x.im);
      } else {
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          const cf x = cmul(rot, acc[r][p]);
          dst[size_t(p) * L * L] = make_float2(x.re, x.im);
        }
      }
    }
  }
}

template <int L>
__device__ __forceinline__ void gridder_sep_block(const GridArgs& a, SepShare share, unsigned char* smem) {
  using C = Gsep<L>;
  GsepShared<L>& S = *reinterpret_cast<GsepShared<L>*>(smem);
  if (threadIdx.x == 0) {
    for (int k = 0; k < C::kRing; ++k) mbar_init(&S.empty[k], 1);
    mbar_init(&S.drain, 1);
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
    gsep_producer<L>(a, share, S);
  } else {
    regs_take<C::kConsumerRegs>();
    gsep_consumer<L>(a, share, S, reinterpret_cast<float4*>(&S + 1));
  }
  sep_drain(&S.fail, uniform_warp() == kSepHalf / 32 - 1, &S.drain);
  if (threadIdx.x < 32) {
    tc_fence_after();
    tmem_free(S.tmem, C::kTmemCols);
  }
}

template <int L>
__global__ void __launch_bounds__(kSepThreads, 1) gridder_sep_kernel(const GridArgs a) {
  extern __shared__ __align__(128) unsigned char sep_smem[];
  gridder_sep_block<L>(a, SepShare{int(blockIdx.x) * a.run, a.n_items, int(gridDim.x), a.run}, sep_smem);
}

// One launch over the items of several plans: blocks = (plan slot, first run), each taking every `stride`-th run of its
// plan from there
template <int L>
__global__ void __launch_bounds__(kSepThreads, 1) gridder_sep_multi_kernel(const GridArgs* args, const int2* blocks) {
  extern __shared__ __align__(128) unsigned char sep_smem[];
  __shared__ __align__(16) unsigned char s_args_raw[sizeof(GridArgs)];
  const int2 it = blocks[blockIdx.x];
  if (threadIdx.x == 0) memcpy(s_args_raw, args + it.x, sizeof(GridArgs));
  __syncthreads();
  const GridArgs& a = *reinterpret_cast<const GridArgs*>(s_args_raw);
  gridder_sep_block<L>(a, SepShare{it.y * a.run, a.n_items, a.stride, a.run}, sep_smem);
}

template <int L>
int configure_gridder_sep_l(int* persistent_blocks) {
  // the halves' register split is of the registers the block is launched with
  cudaError_t e = sep_check_regs(gridder_sep_kernel<L>, 128);
  if (e == cudaSuccess) e = sep_check_regs(gridder_sep_multi_kernel<L>, 128);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(gridder_sep_kernel<L>, cudaFuncAttributeMaxDynamicSharedMemorySize,
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
int launch_gridder_sep_l(const GridArgs& args, int n_items, int blocks, void* stream) {
  if (n_items <= 0) return 0;
  GridArgs a = args;
  a.n_items = n_items;
  gridder_sep_kernel<L><<<blocks, kSepThreads, gsep_smem<L>(a.g.nodes), cudaStream_t(stream)>>>(a);
  return int(cudaGetLastError());
}

template <int L>
int launch_gridder_sep_multi_l(const GridArgs* args, const int2* blocks, int n_blocks, int max_nodes, void* stream) {
  if (n_blocks <= 0) return 0;
  gridder_sep_multi_kernel<L><<<n_blocks, kSepThreads, gsep_smem<L>(max_nodes), cudaStream_t(stream)>>>(args, blocks);
  return int(cudaGetLastError());
}

}  // namespace idg
