// Degridder with separable phasors (templates), included by the per-subgrid-size
// translation units degridder_sep_lNN.cu.  See sep_common.cuh for the split
// of the phase; this is the adjoint of gridder_sep_kernels.cuh.
//
// For one A-term segment, Z = A_p Y A_q^H with Y the subgrid image times
// taper, centring sign and e^{-2 pi i w_ref n'} (applied by the splitter):
//   V_k = sum_i conj(E_k(i)) D_k(i),
//   D_k(i) = sum_j Z(i,j) conj(F_k(j)) (1 - 2 pi i delta_k p_i q_j).
// D is a complex matrix product on the tensor cores: rows (p, i) for 4
// correlations x 32 pixel columns, contraction over the L rows j, columns
// (re | im, k) for the item's visibilities k, so a short segment makes a
// narrow product instead of an empty one.  The remaining sum over i takes one
// complex multiply-add per (visibility, column), 1/L of the direct sum.
//
// One block of 512 threads per bundle of items (an item is up to kv
// visibilities of one segment).  The F side of all L rows stays in shared
// memory for the item; the Z side streams through a ring of two buffers of
// 32 columns x 32 rows: thread = row (p, i) x 8 rows j, from Y in global
// memory and the A-terms interpolated along i in shared memory.  One thread issues
// the MMAs; the accumulator alternates between two ranges of tensor memory
// from column block to column block, so the sum over i of one block overlaps
// the MMAs of the next.  At the end of the item each warp adds its 32 columns
// with a transposing butterfly.
#pragma once

#include "sep_common.cuh"

namespace idg {

template <int L>
struct Dsep {
  static constexpr int kBlocks = L / 32;                  // column blocks, and 32-row pieces of the contraction
  static constexpr int kMaxVis = L <= 64 ? 128 : 64;      // visibilities per item at most
  static constexpr int kVisBlocks = kMaxVis / 64;         // 16-visibility blocks per warp
  static constexpr int kColStride = 2 * kMaxVis;          // between the two accumulators
  static constexpr uint32_t kTmemCols = 2 * kColStride;
  static constexpr uint32_t kChunk = 6 * 4096;            // Z side of 16 rows: (hi, lo, first order) x (re, im)
  static constexpr uint32_t kRing = 2 * 2 * kChunk;       // two buffers of 32 rows
};

struct DsepTail {
  uint64_t bar[2];
  uint32_t tmem;
  int fail;
  int item;
  float inv_scale;
};

// shared memory: ring, F side, visibility parameters, A-term rows, tail
template <int L>
__host__ __device__ inline size_t dsep_smem(int kv, int nodes) {
  return size_t(Dsep<L>::kRing) + size_t(kv) * (L * 18 + 16) + size_t(nodes) * 8 * 32 * sizeof(float2) +
         sizeof(DsepTail);
}

// visibilities per item for A-terms of `nodes` samples per axis: what fits beside the ring, a multiple of 8
template <int L>
int dsep_vis(int nodes) {
  int kv = Dsep<L>::kMaxVis;
  while (kv > 8 && dsep_smem<L>(kv, nodes) > size_t(kSepSmemLimit)) kv -= 8;
  return kv;
}

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

// a + f (b - a)
__device__ __forceinline__ cf cf_lerp(cf a, cf d, float f) { return {fmaf(f, d.re, a.re), fmaf(f, d.im, a.im)}; }
__device__ __forceinline__ cf cf_sub(cf a, cf b) { return {a.re - b.re, a.im - b.im}; }
// a * conj(b)
__device__ __forceinline__ cf cmul_conj(cf a, cf b) {
  return {a.re * b.re + a.im * b.im, a.im * b.re - a.re * b.im};
}

template <int L>
struct DsepItem {
  using C = Dsep<L>;
  const DegridArgs& a;
  unsigned char* ring;
  unsigned char* fside;
  float4* prm;             // [kv] (a fix, b fix, delta, 0)
  float2* R;               // [node row][p 00 01 10 11, q 00 01 10 11][32]
  DsepTail& S;
  uint32_t cg;             // 32-row pieces of this block so far (ring position and parity)

  __device__ __forceinline__ void wait_piece(uint32_t c) {
    if (*reinterpret_cast<volatile int*>(&S.fail)) return;
    if (!mbar_wait_bounded(&S.bar[c & 1], (c >> 1) & 1)) {
      atomicOr(a.status, kStatusTimeout);
      *reinterpret_cast<volatile int*>(&S.fail) = 1;
    }
  }

  // A-terms of the segment interpolated along i at every node row for column block ib; p times `scale`
  __device__ __forceinline__ void rows(const float2* Ap, const float2* Aq, int ib, float scale) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nodes = a.g.nodes;
    const NodeWeight wx = node_weight(ib * 32 + lane, nodes, L);
    for (int e = warp; e < 2 * nodes; e += kSepThreads / 32) {
      const int r = e >> 1, st = e & 1;
      const float4* n0 = reinterpret_cast<const float4*>((st ? Aq : Ap) + (size_t(r) * nodes + wx.a) * 4);
      const float k1 = st ? wx.f : wx.f * scale, k0 = st ? 1.f - wx.f : (1.f - wx.f) * scale;
      float2* dst = R + (r * 8 + 4 * st) * 32 + lane;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float4 u = __ldg(n0 + h), v = __ldg(n0 + 2 + h);
        dst[2 * h * 32] = make_float2(k0 * u.x + k1 * v.x, k0 * u.y + k1 * v.y);
        dst[(2 * h + 1) * 32] = make_float2(k0 * u.z + k1 * v.z, k0 * u.w + k1 * v.w);
      }
    }
  }

  // conj(F) of the item's visibilities (n_pad rows) at all L rows j
  __device__ __forceinline__ void produce_f(int n_pad) {
    const uint32_t block = uint32_t(n_pad) * 16, group = 3 * block, chunk = 2 * group, level = (L / 16) * chunk;
    const uint32_t base = smem_u32(fside);
    for (int idx = threadIdx.x; idx < n_pad * (L / 8); idx += kSepThreads) {
      const int o = idx / n_pad, n = idx - o * n_pad;
      const float4 v = prm[n];
      const int fix = __float_as_int(v.y);
      const float4* tb = reinterpret_cast<const float4*>(a.sep.b + 8 * o);
      const float4* tq = reinterpret_cast<const float4*>(a.sep.q + 8 * o);
      SepF f;
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const float4 b4 = __ldg(tb + u), q4 = __ldg(tq + u);
        const float fb[4] = {b4.x, b4.y, b4.z, b4.w}, fq[4] = {q4.x, q4.y, q4.z, q4.w};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float c[2], s[2];
#pragma unroll
          for (int e = 0; e < 2; ++e)
            __sincosf(sep_phase(fix, 8 * o + 4 * u + 2 * h + e - L / 2, v.z, fb[2 * h + e]), &s[e], &c[e]);
          const __half2 d = __floats2half2_rn(-v.z * fq[2 * h], -v.z * fq[2 * h + 1]);
          const int w = 2 * u + h;
          const __half2 hc = sep_split(c[0], c[1], f.r_hi[w], f.r_lo[w]);
          const __half2 hs = sep_split(-s[0], -s[1], f.i_hi[w], f.i_lo[w]);
          // -i delta q conj(F): re = delta q Im, im = -delta q Re
          f.r_c[w] = h2_bits(__hneg2(__hmul2(hs, d)));
          f.i_c[w] = h2_bits(__hmul2(hc, d));
        }
      }
      sep_store_f(f, base + (o >> 1) * chunk + (o & 1) * group + n * 16, block, level);
    }
  }

  // Z of rows 32 sc .. 32 sc + 31 for column block ib: thread = (p, i) x 8 rows j
  template <bool DIAG>
  __device__ __forceinline__ void produce_z(uint32_t buf, const float2* Y, int ib, int sc, __half2 fit_p) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int p = warp & 3, g = (warp >> 2) & 1, h = warp >> 3;
    const int pa = p >> 1, pb = p & 1;
    const int j0 = 32 * sc + 16 * h + 8 * g;
    const float2* y0 = Y + size_t(j0) * L + ib * 32 + lane;
    const int step = a.g.nodes - 1;
    int node = step * j0 / L, rem = step * j0 - node * L;
    constexpr int NE = DIAG ? 2 : 4;
    const bool stokes = a.g.npol == 1;
    // entries this row needs: diagonal p_aa, q_bb; full p_a0, p_a1, q_b0, q_b1
    int off[NE];
    if constexpr (DIAG) {
      off[0] = (3 * pa) * 32 + lane;
      off[1] = (4 + 3 * pb) * 32 + lane;
    } else {
      off[0] = (2 * pa) * 32 + lane;
      off[1] = (2 * pa + 1) * 32 + lane;
      off[2] = (4 + 2 * pb) * 32 + lane;
      off[3] = (4 + 2 * pb + 1) * 32 + lane;
    }
    cf u[NE], d[NE];
    auto load_rows = [&](int r) {
#pragma unroll
      for (int e = 0; e < NE; ++e) {
        const float2 x = R[r * 256 + off[e]], y = R[(r + 1) * 256 + off[e]];
        u[e] = {x.x, x.y};
        d[e] = {y.x - x.x, y.y - x.y};
      }
    };
    load_rows(node);
    uint32_t re_hi[4], re_lo[4], re_c[4], im_hi[4], im_lo[4], im_c[4];
    // Y of this row's correlations: diagonal A-terms read one, full ones all four (Stokes I: one plane, on the
    // diagonal of the brightness matrix)
    float2 yv[8];
    if (DIAG || stokes) {
#pragma unroll
      for (int q = 0; q < 8; ++q) yv[q] = y0[(stokes ? 0 : size_t(p) * L * L) + q * L];
    }
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      float zr[2], zi[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int q = 2 * w + e;
        const float f = float(rem) * (1.f / float(L));
        cf z;
        if constexpr (DIAG) {
          z = cmul_conj(cmul(cf_lerp(u[0], d[0], f), cf{yv[q].x, yv[q].y}), cf_lerp(u[1], d[1], f));
          if (stokes && pa != pb) z = {0.f, 0.f};
        } else {
          const cf p0 = cf_lerp(u[0], d[0], f), p1 = cf_lerp(u[1], d[1], f);
          const cf q0 = cf_lerp(u[2], d[2], f), q1 = cf_lerp(u[3], d[3], f);
          if (stokes) {
            z = cmul(cadd(cmul_conj(p0, q0), cmul_conj(p1, q1)), cf{yv[q].x, yv[q].y});
          } else {
            cf y[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const float2 v = y0[size_t(k) * L * L + q * L];
              y[k] = {v.x, v.y};
            }
            z = cadd(cmul_conj(cadd(cmul(p0, y[0]), cmul(p1, y[2])), q0),
                     cmul_conj(cadd(cmul(p0, y[1]), cmul(p1, y[3])), q1));
          }
        }
        zr[e] = z.re;
        zi[e] = z.im;
        rem += step;
        if (rem >= L) {  // the next row lies in the next node cell (the same for the whole warp)
          rem -= L;
          ++node;
          if (q < 7) load_rows(node);
        }
      }
      re_c[w] = h2_bits(__hmul2(sep_split(zr[0], zr[1], re_hi[w], re_lo[w]), fit_p));
      im_c[w] = h2_bits(__hmul2(sep_split(zi[0], zi[1], im_hi[w], im_lo[w]), fit_p));
    }
    const uint32_t dst = buf + h * C::kChunk + g * 2048 + (p * 32 + lane) * 16;
    sts128(dst, re_hi);
    sts128(dst + 4096, im_hi);
    sts128(dst + 2 * 4096, re_lo);
    sts128(dst + 3 * 4096, im_lo);
    sts128(dst + 4 * 4096, re_c);
    sts128(dst + 5 * 4096, im_c);
  }

  // MMAs of one 32-row piece (one thread)
  __device__ __forceinline__ void issue(uint32_t buf, uint32_t d, int sc, int n_pad, bool first, uint64_t* bar) {
    const uint32_t block = uint32_t(n_pad) * 16, group = 3 * block, chunk = 2 * group, level = (L / 16) * chunk;
    const uint32_t idesc = sep_idesc(2 * n_pad);
    const uint32_t zl[4] = {1, 0, 2, 0}, fl[4] = {0, 1, 2, 0};
    const uint32_t f0 = smem_u32(fside);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint32_t f = f0 + (2 * sc + h) * chunk, z = buf + h * C::kChunk;
#pragma unroll
      for (int n = 0; n < 4; ++n) {
        const uint32_t za = z + zl[n] * 8192, fa = f + fl[n] * level;
        sep_mma(d, sep_desc(za, 2048), sep_desc(fa + block, group), idesc, (first && h == 0 && n == 0) ? 0u : 1u);
        sep_mma(d, sep_desc(za + 4096, 2048), sep_desc(fa, group), idesc, 1u);
      }
    }
    sep_commit(bar);
  }

  __device__ __forceinline__ bool run(int item_idx) {
    const DegridItem item = a.items[item_idx];
    const SubgridDesc sd = a.sg[item.sg];
    const SegmentDesc seg = a.seg[item.segment];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nodes = a.g.nodes, nA = nodes * nodes * 4, nc = sd.c1 - sd.c0;
    const int nv = item.k_end - item.k_begin, n_pad = (nv + 7) & ~7;
    const int sp = seg.interval * a.g.n_st + sd.p, sq = seg.interval * a.g.n_st + sd.q;
    const float2 *Ap = a.aterms + size_t(sp) * nA, *Aq = a.aterms + size_t(sq) * nA;
    const bool diag = a.adiag[sp] && a.adiag[sq];
    const float2* Y = a.scratch + size_t(item.sg) * 4 * L * L;
    // power-of-two scale of Z from the largest components of Y and of the A-terms' nodes
    float ym = 0.f;
    for (int k = 0; k < a.g.npol; ++k) ym = fmaxf(ym, a.ymax[item.sg * 4 + k]);
    const float scale = sep_scale(ym * a.amax[sp] * a.amax[sq]);
    const uint32_t ring0 = smem_u32(ring);

    if (tid < n_pad) {
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (tid < nv) {
        const int k = item.k_begin + tid, row = k / nc, ch = sd.c0 + (k - row * nc);
        const double* r = a.uvw + (size_t(sd.b) * a.g.n_t + sd.t0 + row) * 3;
        const double fs = subgrid_sign(sd) * a.fscale[ch], inv_l = 1.0 / double(L);
        v.x = __int_as_float(sep_fix(((r[0] * fs) * a.g.fov - double(sd.x0 + L / 2 - a.g.N / 2)) * inv_l));
        v.y = __int_as_float(sep_fix(((r[1] * fs) * a.g.fov - double(sd.y0 + L / 2 - a.g.N / 2)) * inv_l));
        v.z = float(r[2] * fs - (double(a.w_ref[item.sg]) + subgrid_w0(a.g, sd)));
      }
      prm[tid] = v;
    }
    rows(Ap, Aq, 0, scale);
    __syncthreads();
    produce_f(n_pad);

    float acc[C::kVisBlocks][32];  // [16 visibilities][re, im]
#pragma unroll
    for (int b = 0; b < C::kVisBlocks; ++b)
#pragma unroll
      for (int k = 0; k < 32; ++k) acc[b][k] = 0.f;

    // conj(E) D of column block ib (its last piece is `last`) added to acc: thread = row (p, i), 16-visibility
    // blocks warp / 4, warp / 4 + 4
    auto sum_columns = [&](int ib, uint32_t last) {
      const int i = ib * 32 + lane;
      const float fit_a = __ldg(a.sep.a + i);
      wait_piece(last);
      tc_fence_after();
      const uint32_t d = S.tmem + (uint32_t((warp & 3) * 32) << 16) + (ib & 1) * C::kColStride;
#pragma unroll
      for (int b = 0; b < C::kVisBlocks; ++b) {
        const int k0 = 16 * ((warp >> 2) + 4 * b);
        if (k0 < n_pad) {
          float re[16], im[16];
          tmem_ld16(re, d + k0);
          tmem_ld16(im, d + n_pad + k0);
          tmem_wait_ld();
#pragma unroll
          for (int k = 0; k < 16; ++k) {
            const float4 v = prm[imin(k0 + k, n_pad - 1)];
            float s, c;
            __sincosf(sep_phase(__float_as_int(v.x), i - L / 2, v.z, fit_a), &s, &c);
            acc[b][2 * k] = fmaf(re[k], c, fmaf(im[k], s, acc[b][2 * k]));
            acc[b][2 * k + 1] = fmaf(im[k], c, fmaf(-re[k], s, acc[b][2 * k + 1]));
          }
        }
      }
      tc_fence_before();
    };

    constexpr int NB = C::kBlocks;
#pragma unroll 1
    for (int ib = 0; ib < NB; ++ib) {
      const __half2 fit_p = __float2half2_rn(__ldg(a.sep.p + ib * 32 + lane));
      if (ib > 0) {
        rows(Ap, Aq, ib, scale);
        __syncthreads();
      }
#pragma unroll 1
      for (int sc = 0; sc < NB; ++sc) {
        const uint32_t cc = cg + uint32_t(ib * NB + sc);
        if (cc >= 2) wait_piece(cc - 2);
        const uint32_t buf = ring0 + (cc & 1) * (2 * C::kChunk);
        if (diag)
          produce_z<true>(buf, Y, ib, sc, fit_p);
        else
          produce_z<false>(buf, Y, ib, sc, fit_p);
        fence_proxy_async();
        __syncthreads();
        if (tid == 0) {
          tc_fence_after();
          issue(buf, S.tmem + (ib & 1) * C::kColStride, sc, n_pad, sc == 0, &S.bar[cc & 1]);
        }
        if (sc == 0 && ib > 0) sum_columns(ib - 1, cc - 1);
      }
    }
    sum_columns(NB - 1, cg + uint32_t(NB * NB) - 1);
    cg += uint32_t(NB * NB);

    // sums over the 32 columns of the warp: lane l ends with component l & 1 of visibility l / 2 of the block
    float* out = reinterpret_cast<float*>(ring);  // [n_pad][8]; every MMA has read its operands
    const float inv = 1.f / scale;
#pragma unroll
    for (int b = 0; b < C::kVisBlocks; ++b) {
#pragma unroll
      for (int w = 16; w; w >>= 1) {
        const bool up = lane & w;
#pragma unroll
        for (int k = 0; k < w; ++k) {
          const float keep = up ? acc[b][k + w] : acc[b][k], give = up ? acc[b][k] : acc[b][k + w];
          acc[b][k] = keep + __shfl_xor_sync(0xffffffffu, give, w);
        }
      }
      const int k = 16 * ((warp >> 2) + 4 * b) + (lane >> 1);
      if (k < n_pad) out[k * 8 + 2 * (warp & 3) + (lane & 1)] = inv * acc[b][0];
    }
    __syncthreads();
    if (tid < nv) {
      const int k = item.k_begin + tid, row = k / nc;
      const size_t vrow = (size_t(sd.b) * a.g.n_t + sd.t0 + row) * a.g.n_ch + sd.c0 + (k - row * nc);
      const float4* o = reinterpret_cast<const float4*>(out + tid * 8);
      float4 v0 = o[0], v1 = o[1];
      if (sd.flags & kSubgridMirrored) mirror_values(v0, v1);
      a.vis[2 * vrow] = v0;
      a.vis[2 * vrow + 1] = v1;
    }
    __syncthreads();  // ring, parameters and A-term rows free for the next item
    return !*reinterpret_cast<volatile int*>(&S.fail);
  }
};

// items [first, last) of the block, or bundles of `bundle` items drained from the queue
template <int L, bool PERSIST>
__device__ __forceinline__ void degridder_sep_block(const DegridArgs& a, int first, int last, int bundle,
                                                    unsigned char* smem) {
  using C = Dsep<L>;
  unsigned char* fside = smem + C::kRing;
  float4* prm = reinterpret_cast<float4*>(fside + size_t(a.kv) * L * 18);
  float2* R = reinterpret_cast<float2*>(prm + a.kv);
  DsepTail& S = *reinterpret_cast<DsepTail*>(R + size_t(a.g.nodes) * 8 * 32);
  if (threadIdx.x == 0) {
    mbar_init(&S.bar[0], 1);
    mbar_init(&S.bar[1], 1);
    fence_mbar_init();
    S.fail = 0;
  }
  if (threadIdx.x < 32) tmem_alloc(&S.tmem, C::kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  DsepItem<L> it{a, smem, fside, prm, R, S, 0};
  bool ok = true;
  if constexpr (!PERSIST) {
    for (int k = first; k < last && ok; ++k) ok = it.run(k);
  } else {
    while (ok) {
      if (threadIdx.x == 0) S.item = atomicAdd(a.queue, bundle);
      __syncthreads();
      const int k0 = S.item;
      __syncthreads();
      if (k0 >= a.n_items) break;
      for (int k = k0; k < imin(k0 + bundle, a.n_items) && ok; ++k) ok = it.run(k);
    }
  }
  // a wait that gave up: give the MMAs in flight one more bounded wait before their memory goes
  if (!ok && it.cg > 0) mbar_wait_bounded(&S.bar[(it.cg - 1) & 1], ((it.cg - 1) >> 1) & 1);
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x < 32) {
    tc_fence_after();
    tmem_free(S.tmem, C::kTmemCols);
  }
}

template <int L, bool PERSIST>
__global__ void __launch_bounds__(kSepThreads, 1) degridder_sep_kernel(const DegridArgs a, int bundle) {
  extern __shared__ __align__(128) unsigned char sep_smem[];
  degridder_sep_block<L, PERSIST>(a, blockIdx.x * bundle, imin((blockIdx.x + 1) * bundle, a.n_items), bundle, sep_smem);
}

// One launch over the items of several plans (items = (plan slot, item index))
template <int L>
__global__ void __launch_bounds__(kSepThreads, 1) degridder_sep_multi_kernel(const DegridArgs* args,
                                                                            const int2* items) {
  extern __shared__ __align__(128) unsigned char sep_smem[];
  __shared__ __align__(16) unsigned char s_args_raw[sizeof(DegridArgs)];
  const int2 it = items[blockIdx.x];
  if (threadIdx.x == 0) memcpy(s_args_raw, args + it.x, sizeof(DegridArgs));
  __syncthreads();
  degridder_sep_block<L, false>(*reinterpret_cast<const DegridArgs*>(s_args_raw), it.y, it.y + 1, 1, sep_smem);
}

template <int L>
int configure_degridder_sep_l(int* persistent_blocks) {
  cudaError_t e = cudaFuncSetAttribute(degridder_sep_kernel<L, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kSepSmemLimit);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(degridder_sep_kernel<L, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSepSmemLimit);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(degridder_sep_multi_kernel<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSepSmemLimit);
  int dev = 0, sms = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  *persistent_blocks = sms;  // 512 threads of up to 128 registers: one block per SM
  return int(e);
}

template <int L>
int degridder_sep_vis_l(int nodes) {
  return dsep_vis<L>(nodes);
}

template <int L>
int launch_degridder_sep_l(const DegridArgs& a, int n_items, int persistent_blocks, int bundle, void* stream) {
  if (n_items <= 0) return 0;
  const size_t smem = dsep_smem<L>(a.kv, a.g.nodes);
  const int n = (n_items + bundle - 1) / bundle;
  if (persistent_blocks > 0)
    degridder_sep_kernel<L, true><<<persistent_blocks < n ? persistent_blocks : n, kSepThreads, smem,
                                    cudaStream_t(stream)>>>(a, bundle);
  else
    degridder_sep_kernel<L, false><<<n, kSepThreads, smem, cudaStream_t(stream)>>>(a, bundle);
  return int(cudaGetLastError());
}

template <int L>
int launch_degridder_sep_multi_l(const DegridArgs* args, const int2* items, int n_items, int max_nodes,
                                 void* stream) {
  if (n_items <= 0) return 0;
  size_t smem = 0;  // the largest layout of any plan of up to max_nodes (items of a plan are cut to its own)
  for (int n = 2; n <= max_nodes; ++n) {
    const size_t s = dsep_smem<L>(dsep_vis<L>(n), n);
    smem = s > smem ? s : smem;
  }
  degridder_sep_multi_kernel<L><<<n_items, kSepThreads, smem, cudaStream_t(stream)>>>(args, items);
  return int(cudaGetLastError());
}

}  // namespace idg
