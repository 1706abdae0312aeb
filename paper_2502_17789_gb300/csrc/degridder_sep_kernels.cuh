// Degridder with separable phasors (templates), included by the per-subgrid-size
// translation units degridder_sep_lNN.cu.  See sep_common.cuh for the split
// of the phase; this is the adjoint of gridder_sep_kernels.cuh.
//
// For one A-term segment, Z = A_p Y A_q^H with Y the subgrid image times
// taper, centring sign and e^{-2 pi i w_ref n'} (applied by the splitter):
//   V_k = sum_i conj(E_k(i)) D_k(i),
//   D_k(i) = sum_j Z(i,j) conj(F_k(j)) (1 - 2 pi i delta_k p_i q_j).
// D is a complex matrix product on the tensor cores: rows (p, i) for 4
// correlations x 32 pixel columns, contraction over the L rows j, columns the
// item's visibilities k (real and imaginary sums as two accumulators), so a
// short segment makes a narrow product instead of an empty one.  The remaining
// sum over i takes one complex multiply-add per (visibility, column), 1/L of
// the direct sum.
//
// One block of 512 threads per bundle of items (an item is up to kv
// visibilities of one segment), split into two halves that run side by side.
// Producers: per piece of 16 rows j of a block of 32 columns, thread = row
// (p, i) x 8 rows j writes Z to tensor memory (two rows at a time in packed f32x2),
// from Y pieces copied to shared memory two pieces ahead; one of them issues the
// piece's 16 MMAs, whose commit frees it.  Consumers: while an item runs they
// prepare the next one (phase slopes, the F side of all L rows, A-term samples;
// double buffers), and take the accumulators, which alternate between two
// column ranges of tensor memory from column block to column block, through
// the sum over i; a transposing butterfly per item adds the 32 columns of a
// warp.
//
// Measured (GB300, MWA-like workload, 96 x 96 subgrids, segments of about 60
// visibilities, per degrid call): 38.4 ms, against 46.8 ms with all threads
// doing each step in turn and Z in shared memory, and 78.4 ms of the kernel
// with one phasor per visibility and pixel (degridder_tc_kernels.cuh).
#pragma once

#include "sep_common.cuh"

namespace idg {

constexpr int kDsepMaxVis = 64;   // visibilities per item at most
constexpr int kDsepRing = 4;      // Z pieces in tensor memory
constexpr int kDsepYRing = 3;     // Y pieces in shared memory
constexpr int kDsepColStride = 2 * kDsepMaxVis;       // between the two accumulators (re, im)
constexpr int kDsepZCol = 2 * kDsepColStride;         // first column of the Z ring
constexpr uint32_t kDsepTmemCols = 512;
static_assert(kDsepZCol + kDsepRing * 48 <= int(kDsepTmemCols), "tensor memory");

struct alignas(128) DsepShared {
  float2 y[kDsepYRing][4][8][2][32];  // [piece][pol][row pair][re, im][column]
  float fix_a[2][kDsepMaxVis], fix_b[2][kDsepMaxVis], delta[2][kDsepMaxVis];  // [item parity][visibility]
  float out[kDsepMaxVis][8];
  // the producers' part of an item, by item parity
  struct Info {
    float scale;   // of Z, a power of two
    int sg, n_pad, diag;
  } info[2];
  uint64_t ready[2];        // item prepared (8 consumer warps)
  uint64_t empty[kDsepRing];  // Z piece read by its MMAs
  uint64_t full[2];         // accumulator complete
  uint64_t drained[2];      // accumulator read (8 consumer warps)
  uint32_t tmem;
  int fail;
};

// shared memory: DsepShared, F sides of two items, A-term samples of two items
template <int L>
__host__ __device__ inline size_t dsep_smem(int kv, int nodes) {
  return sizeof(DsepShared) + size_t(2) * kv * L * 12 + size_t(2) * 2 * nodes * nodes * 4 * sizeof(float2);
}

// visibilities per item for A-terms of `nodes` samples per axis: what fits, a multiple of 16
template <int L>
int dsep_vis(int nodes) {
  int kv = kDsepMaxVis;
  while (kv > 16 && dsep_smem<L>(kv, nodes) > size_t(kSepSmemLimit)) kv -= 16;
  return kv;
}

template <int L>
struct Dsep {
  const DegridArgs& a;
  DsepShared& S;
  unsigned char* fside;   // [item parity][level][16 rows][k group][Re, Im][visibility] rows of 16 bytes
  float4* raw;            // [item parity][station][nodes][nodes][2]
  const int first, last, stride;

  static constexpr int kBlocks = L / 32, kPieces = L / 16;

  __device__ __forceinline__ void wait(uint64_t* bar, uint32_t parity) { sep_wait(bar, parity, &S.fail, a.status); }

  // ---------------------------------------------------------------- producers

  // Y rows 16 jc .. of column block ib of batch subgrid sg, on their way to buffer y
  __device__ __forceinline__ void fetch_y(int buf, int sg, int ib, int jc) {
    const int pol = threadIdx.x >> 6, u = threadIdx.x & 63;  // 64 threads per correlation
    if (pol < a.g.npol) {
      // [pol][row pair][re, im][column]: 16 runs of 256 bytes
      const float2* src = a.scratch + size_t(sg) * 4 * L * L + (size_t(pol) * (L / 2) + 8 * jc) * 2 * L + 32 * ib;
      float2* dst = &S.y[buf][pol][0][0][0];
#pragma unroll
      for (int e = u; e < 256; e += 64) cp_async16(dst + 2 * e, src + (e >> 4) * L + 2 * (e & 15));
    }
    cp_async_commit();
  }

  // Z of rows 16 jc .. for column block ib: thread = (p, i) x 8 rows j.  QUAD: node cells start at multiples of four
  // rows, so the cell can change only half way and not at every row.
  template <bool DIAG, bool QUAD>
  __device__ __forceinline__ void produce(uint32_t e_col, const float2* yb, const float4* samples, float scale,
                                          NodeWeight wx, int jc, __half2 fit_p) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int p = warp & 3, g = warp >> 2, pa = p >> 1, pb = p & 1;
    const int nodes = a.g.nodes, step = nodes - 1;
    const bool stokes = a.g.npol == 1;
    constexpr int NE = DIAG ? 1 : 2;  // entries of each station's matrix that this correlation needs
    // an off-diagonal correlation of a Stokes-I model with diagonal matrices is zero
    const float kp = (DIAG && stokes && pa != pb) ? 0.f : scale;
    const float k1[2] = {wx.f * kp, wx.f}, k0[2] = {(1.f - wx.f) * kp, 1.f - wx.f};
    const float2* smp[2];
#pragma unroll
    for (int st = 0; st < 2; ++st)
      smp[st] = reinterpret_cast<const float2*>(samples + st * nodes * nodes * 2) + wx.a * 4 +
                (DIAG ? 3 * (st ? pb : pa) : 2 * (st ? pb : pa));
    // node row r interpolated along i, p_aa, q_bb (diagonal) or p_a0, p_a1, q_b0, q_b1, and the step to the next
    cf u[2][NE], d[2][NE];
    auto load_cell = [&](int r) {
#pragma unroll
      for (int st = 0; st < 2; ++st)
#pragma unroll
        for (int e = 0; e < NE; ++e) {
          const float2* n0 = smp[st] + r * nodes * 4 + e;
          const float2 x0 = n0[0], y0 = n0[4], x1 = n0[nodes * 4], y1 = n0[nodes * 4 + 4];
          u[st][e] = {k0[st] * x0.x + k1[st] * y0.x, k0[st] * x0.y + k1[st] * y0.y};
          d[st][e] = {fmaf(k0[st], x1.x, fmaf(k1[st], y1.x, -u[st][e].re)),
                      fmaf(k0[st], x1.y, fmaf(k1[st], y1.y, -u[st][e].im))};
        }
    };
    // row q of the octet lies at (rem + step q) / L of the cell that starts at node row `at`
    int at = step * (16 * jc + 8 * g) / L, rem = step * (16 * jc + 8 * g) - at * L;
    load_cell(at);
    float f0 = float(rem) * (1.f / float(L));
    const float df = float(step) * (1.f / float(L));
    const float2* y0 = yb + (4 * g) * 64 + lane;  // [pol][row pair][re, im][column]
    uint32_t re_hi[4], re_lo[4], re_c[4], im_hi[4], im_lo[4], im_c[4];
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      float2 yr[DIAG ? 1 : 4], yi[DIAG ? 1 : 4];  // Y at both rows of the pair
#pragma unroll
      for (int k = 0; k < (DIAG ? 1 : 4); ++k) {
        const float2* y = y0 + (stokes ? 0 : DIAG ? p : k) * 512 + w * 64;
        yr[k] = y[0];
        yi[k] = y[32];
      }
      float2 zr, zi;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int q = 2 * w + h;
        if (QUAD ? q == 4 : q > 0) {
          if (rem + step * q >= L) {  // the same for the whole warp
            rem -= L;
            f0 -= 1.f;
            load_cell(++at);
          }
        }
        const float f = fmaf(float(q), df, f0);
        cf m[2][NE];  // the entries at this row
#pragma unroll
        for (int st = 0; st < 2; ++st)
#pragma unroll
          for (int e = 0; e < NE; ++e) m[st][e] = {fmaf(f, d[st][e].re, u[st][e].re), fmaf(f, d[st][e].im, u[st][e].im)};
        cf y[DIAG ? 1 : 4];
#pragma unroll
        for (int k = 0; k < (DIAG ? 1 : 4); ++k) y[k] = h ? cf{yr[k].y, yi[k].y} : cf{yr[k].x, yi[k].x};
        cf z;
        if constexpr (DIAG) {
          z = cmulc(m[1][0], cmul(m[0][0], y[0]));
        } else if (stokes) {
          z = cadd(cmulc(m[1][0], cmul(m[0][0], y[0])), cmulc(m[1][1], cmul(m[0][1], y[0])));
        } else {
          z = cadd(cmulc(m[1][0], cadd(cmul(m[0][0], y[0]), cmul(m[0][1], y[2]))),
                   cmulc(m[1][1], cadd(cmul(m[0][0], y[1]), cmul(m[0][1], y[3]))));
        }
        if (h) {
          zr.y = z.re;
          zi.y = z.im;
        } else {
          zr.x = z.re;
          zi.x = z.im;
        }
      }
      re_c[w] = h2_bits(__hmul2(sep_split(zr, re_hi[w], re_lo[w]), fit_p));
      im_c[w] = h2_bits(__hmul2(sep_split(zi, im_hi[w], im_lo[w]), fit_p));
    }
    const uint32_t dst = e_col + (uint32_t(p * 32) << 16) + 4 * g;
    tmem_st4(dst, re_hi);
    tmem_st4(dst + 8, im_hi);
    tmem_st4(dst + 16, re_lo);
    tmem_st4(dst + 24, im_lo);
    tmem_st4(dst + 32, re_c);
    tmem_st4(dst + 40, im_c);
  }

  __device__ __forceinline__ void producer() {
    const int lane = threadIdx.x & 31, nodes = a.g.nodes;
    const bool issuer = uniform_warp() == 0;
    const bool quad = L % (nodes - 1) == 0 && L / (nodes - 1) % 4 == 0;
    const uint32_t tm = S.tmem;
    uint32_t pg = 0, dg = 0, n = 0;  // pieces, accumulators and items of this block so far
    int yb = 0;                      // pg % kDsepYRing
    if (first >= last) return;
    wait(&S.ready[0], 0);
    int y_sg = S.info[0].sg, y_ib = 0, y_jc = 0;  // the piece of Y to fetch next
    auto fetch_next = [&](int buf) {
      fetch_y(buf, y_sg, y_ib, y_jc);
      if (++y_jc == kPieces) {
        y_jc = 0;
        ++y_ib;
      }
    };
    fetch_next(0);
    fetch_next(1);
    cp_async_wait<1>();
    half_sync(kSepProducerBar);
    for (int idx = first; idx < last; idx += stride, ++n) {
      const DsepShared::Info info = S.info[n & 1];
      const bool more = idx + stride < last;
      const float4* samples = raw + (n & 1) * 4 * nodes * nodes;
      const uint32_t block = uint32_t(info.n_pad) * 16, group = 2 * block, chunk = 2 * group, level = kPieces * chunk;
      const uint32_t f0 = smem_u32(fside) + (n & 1) * uint32_t(a.kv) * L * 12;
#pragma unroll 1
      for (int ib = 0; ib < kBlocks; ++ib, ++dg) {
        const int i = ib * 32 + lane;
        const NodeWeight wx = node_weight(i, nodes, L);
        const __half2 fit_p = __float2half2_rn(__ldg(a.sep.p + i));
#pragma unroll 1
        for (int jc = 0; jc < kPieces; ++jc, ++pg) {
          // two pieces ahead, in the next item past this one's end
          if (y_ib == kBlocks && more) {
            wait(&S.ready[(n + 1) & 1], ((n + 1) >> 1) & 1);
            y_sg = S.info[(n + 1) & 1].sg;
            y_ib = 0;
          }
          const int buf = yb;
          if (++yb == kDsepYRing) yb = 0;
          if (y_ib < kBlocks)
            fetch_next(buf == 0 ? 2 : buf - 1);
          else
            cp_async_commit();  // keeps the count of groups
          const uint32_t slot = pg % kDsepRing, turn = pg / kDsepRing;
          if (turn > 0) {
            wait(&S.empty[slot], (turn - 1) & 1);
            tc_fence_after();
          }
          const uint32_t e_col = tm + kDsepZCol + slot * 48;
          const float2* y = &S.y[buf][0][0][0][0];
          if (quad) {
            if (info.diag)
              produce<true, true>(e_col, y, samples, info.scale, wx, jc, fit_p);
            else
              produce<false, true>(e_col, y, samples, info.scale, wx, jc, fit_p);
          } else if (info.diag) {
            produce<true, false>(e_col, y, samples, info.scale, wx, jc, fit_p);
          } else {
            produce<false, false>(e_col, y, samples, info.scale, wx, jc, fit_p);
          }
          cp_async_wait<1>();
          tmem_wait_st();
          tc_fence_before();
          half_sync(kSepProducerBar);
          if (issuer && elect_one()) {
            // the accumulator's previous column block (two back) has been read
            if (jc == 0 && dg >= 2) wait(&S.drained[dg & 1], ((dg >> 1) - 1) & 1);
            tc_fence_after();
            sep_product(tm + (dg & 1) * kDsepColStride, e_col, f0 + jc * chunk, info.n_pad, block, group, level, jc == 0);
            sep_commit(&S.empty[slot]);
            if (jc + 1 == kPieces) sep_commit(&S.full[dg & 1]);
          }
        }
      }
    }
    cp_async_wait<0>();
  }

  // ---------------------------------------------------------------- consumers

  // item idx, number n of the block: phase slopes, A-term samples, conj(F) at all rows, the producers' part
  __device__ __forceinline__ void prepare(int idx, uint32_t n) {
    const int tid = threadIdx.x - kSepHalf, lane = tid & 31;
    const DegridItem item = a.items[idx];
    const SubgridDesc sd = a.sg[item.sg];
    const SegmentDesc seg = a.seg[item.segment];
    const int nv = item.k_end - item.k_begin, n_pad = (nv + 15) & ~15, b = n & 1;
    const int nodes = a.g.nodes, n4 = nodes * nodes * 2;
    const int sp = seg.interval * a.g.n_st + sd.p, sq = seg.interval * a.g.n_st + sd.q;
    {
      const float4* src = reinterpret_cast<const float4*>(a.aterms);
      float4* dst = raw + size_t(b) * 2 * n4;
      for (int e = tid; e < 2 * n4; e += kSepHalf)
        cp_async16(dst + e, src + (e < n4 ? size_t(sp) * n4 + e : size_t(sq) * n4 + e - n4));
      cp_async_commit();
    }
    if (tid < n_pad) {
      int fa = 0, fb = 0;
      float dl = 0.f;
      if (tid < nv) {
        const int nc = sd.c1 - sd.c0, k = item.k_begin + tid, row = k / nc, ch = sd.c0 + (k - row * nc);
        const double* r = a.uvw + (size_t(sd.b) * a.g.n_t + sd.t0 + row) * 3;
        const double fs = subgrid_sign(sd) * a.fscale[ch], inv_l = 1.0 / double(L);
        fa = sep_fix(((r[0] * fs) * a.g.fov - double(sd.x0 + L / 2 - a.g.N / 2)) * inv_l);
        fb = sep_fix(((r[1] * fs) * a.g.fov - double(sd.y0 + L / 2 - a.g.N / 2)) * inv_l);
        dl = float(r[2] * fs - (double(a.w_ref[item.sg]) + subgrid_w0(a.g, sd)));
      }
      S.fix_a[b][tid] = __int_as_float(fa);
      S.fix_b[b][tid] = __int_as_float(fb);
      S.delta[b][tid] = dl;
    }
    if (tid == 0) {
      // scale of Z from the largest components of Y and of the A-terms' nodes
      float ym = 0.f;
      for (int k = 0; k < a.g.npol; ++k) ym = fmaxf(ym, a.ymax[item.sg * 4 + k]);
      S.info[b] = {sep_scale(ym * a.amax[sp] * a.amax[sq]), item.sg, n_pad, a.adiag[sp] && a.adiag[sq]};
    }
    half_sync(kSepConsumerBar);
    const uint32_t block = uint32_t(n_pad) * 16, group = 2 * block, chunk = 2 * group, level = kPieces * chunk;
    const uint32_t base = smem_u32(fside) + b * uint32_t(a.kv) * L * 12;
    for (int e = tid; e < n_pad * (L / 8); e += kSepHalf) {
      const int o = e / n_pad, k = e - o * n_pad;
      const int fix = __float_as_int(S.fix_b[b][k]);
      const float dl = S.delta[b][k];
      const float4* tb = reinterpret_cast<const float4*>(a.sep.b + 8 * o);
      const float4* tq = reinterpret_cast<const float4*>(a.sep.q + 8 * o);
      SepF f;
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const float4 b4 = __ldg(tb + u), q4 = __ldg(tq + u);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int w = 2 * u + h, off = 8 * o + 2 * w - L / 2;
          const float2 fb = pair_of(b4, h), fq = pair_of(q4, h);
          float2 c, s;
          __sincosf(sep_phase(fix, off, dl, fb.x), &s.x, &c.x);
          __sincosf(sep_phase(fix, off + 1, dl, fb.y), &s.y, &c.y);
          const __half2 d2 = __floats2half2_rn(-dl * fq.x, -dl * fq.y);
          const __half2 hc = sep_split(c, f.r_hi[w], f.r_lo[w]);
          const __half2 hs = sep_split(s, f.i_hi[w], f.i_lo[w]);
          // conj(F) = (c, -s); -i delta q conj(F) = (-delta q s, -delta q c)
          f.i_hi[w] ^= 0x80008000u;
          f.i_lo[w] ^= 0x80008000u;
          f.r_c[w] = h2_bits(__hmul2(hs, d2));
          f.i_c[w] = h2_bits(__hmul2(hc, d2));
        }
      }
      sep_store_f(f, base + (o >> 1) * chunk + (o & 1) * group + k * 16, block, level);
    }
    cp_async_wait<0>();
    fence_proxy_async();
    __syncwarp();
    if (lane == 0) mbar_arrive(&S.ready[b]);
  }

  __device__ __forceinline__ void consumer() {
    const int tid = threadIdx.x - kSepHalf, warp = tid >> 5, lane = tid & 31;
    const bool poller = uniform_warp() == kSepHalf / 32;
    uint32_t dg = 0, n = 0;  // accumulators and items of this block so far
    if (first >= last) return;
    prepare(first, 0);
    for (int idx = first; idx < last; idx += stride, ++n) {
      if (idx + stride < last) prepare(idx + stride, n + 1);
      const DegridItem item = a.items[idx];
      const int nv = item.k_end - item.k_begin, n_pad = (nv + 15) & ~15, b = n & 1;
      const float inv = 1.f / S.info[b].scale;
      // thread = row (p, i), 16-visibility blocks warp / 4 and warp / 4 + 2
      float2 re[2][8], im[2][8];  // visibility pairs
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int k = 0; k < 8; ++k) re[h][k] = im[h][k] = make_float2(0.f, 0.f);
#pragma unroll 1
      for (int ib = 0; ib < kBlocks; ++ib, ++dg) {
        const int i = ib * 32 + lane;
        const float fit_a = __ldg(a.sep.a + i);
        if (poller) wait(&S.full[dg & 1], (dg >> 1) & 1);
        half_sync(kSepConsumerBar);
        tc_fence_after();
        const uint32_t d = S.tmem + (uint32_t((warp & 3) * 32) << 16) + (dg & 1) * kDsepColStride;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int k0 = 16 * ((warp >> 2) + 2 * h);
          if (k0 < n_pad) {
            float dr[16], di[16];
            tmem_ld16(dr, d + k0);
            tmem_ld16(di, d + n_pad + k0);
            tmem_wait_ld();
            const float4* fx = reinterpret_cast<const float4*>(&S.fix_a[b][k0]);
            const float4* dl = reinterpret_cast<const float4*>(&S.delta[b][k0]);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              const float2 f = pair_of(fx[k >> 1], k & 1);
              float2 c, s;
              sep_phasor2(__float_as_int(f.x), __float_as_int(f.y), i - L / 2, pair_of(dl[k >> 1], k & 1), fit_a, c, s);
              const float2 r = make_float2(dr[2 * k], dr[2 * k + 1]), m = make_float2(di[2 * k], di[2 * k + 1]);
              re[h][k].x = fmaf(r.x, c.x, fmaf(m.x, s.x, re[h][k].x));
              re[h][k].y = fmaf(r.y, c.y, fmaf(m.y, s.y, re[h][k].y));
              im[h][k].x = fmaf(m.x, c.x, fmaf(-r.x, s.x, im[h][k].x));
              im[h][k].y = fmaf(m.y, c.y, fmaf(-r.y, s.y, im[h][k].y));
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&S.drained[dg & 1]);
      }
      // sums over the 32 columns of the warp: lane l ends with component l & 1 of visibility l / 2 of the block
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int k0 = 16 * ((warp >> 2) + 2 * h);
        if (k0 < n_pad) {
          float v[32];
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            v[4 * k] = re[h][k].x;
            v[4 * k + 1] = im[h][k].x;
            v[4 * k + 2] = re[h][k].y;
            v[4 * k + 3] = im[h][k].y;
          }
#pragma unroll
          for (int w = 16; w; w >>= 1) {
            const bool up = lane & w;
#pragma unroll
            for (int k = 0; k < w; ++k) {
              const float keep = up ? v[k + w] : v[k], give = up ? v[k] : v[k + w];
              v[k] = keep + __shfl_xor_sync(0xffffffffu, give, w);
            }
          }
          S.out[k0 + (lane >> 1)][2 * (warp & 3) + (lane & 1)] = inv * v[0];
        }
      }
      half_sync(kSepConsumerBar);
      if (tid < nv) {
        const SubgridDesc sd = a.sg[item.sg];
        const int nc = sd.c1 - sd.c0, k = item.k_begin + tid, row = k / nc;
        const size_t vrow = (size_t(sd.b) * a.g.n_t + sd.t0 + row) * a.g.n_ch + sd.c0 + (k - row * nc);
        const float4* o = reinterpret_cast<const float4*>(S.out[tid]);
        float4 v0 = o[0], v1 = o[1];
        if (sd.flags & kSubgridMirrored) mirror_values(v0, v1);
        a.vis[2 * vrow] = v0;
        a.vis[2 * vrow + 1] = v1;
      }
      half_sync(kSepConsumerBar);  // S.out free
    }
  }
};

// items first, first + stride, ... below last
template <int L>
__device__ __forceinline__ void degridder_sep_block(const DegridArgs& a, int first, int last, int stride,
                                                    unsigned char* smem) {
  DsepShared& S = *reinterpret_cast<DsepShared*>(smem);
  unsigned char* fside = reinterpret_cast<unsigned char*>(&S + 1);
  if (threadIdx.x == 0) {
    for (int k = 0; k < kDsepRing; ++k) mbar_init(&S.empty[k], 1);
    for (int k = 0; k < 2; ++k) {
      mbar_init(&S.full[k], 1);
      mbar_init(&S.drained[k], kSepHalf / 32);
      mbar_init(&S.ready[k], kSepHalf / 32);
    }
    fence_mbar_init();
    S.fail = 0;
  }
  if (threadIdx.x < 32) tmem_alloc(&S.tmem, kDsepTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  Dsep<L> it{a, S, fside, reinterpret_cast<float4*>(fside + size_t(2) * a.kv * L * 12), first, last, stride};
  if (threadIdx.x < kSepHalf)
    it.producer();
  else
    it.consumer();
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
    tmem_free(S.tmem, kDsepTmemCols);
  }
}

template <int L>
__global__ void __launch_bounds__(kSepThreads, 1) degridder_sep_kernel(const DegridArgs a, int bundle) {
  extern __shared__ __align__(128) unsigned char sep_smem[];
  const int b = blockIdx.x;
  if (bundle > 0)  // neighbouring items (segments of one subgrid)
    degridder_sep_block<L>(a, b * bundle, imin((b + 1) * bundle, a.n_items), 1, sep_smem);
  else             // persistent: every gridDim-th item of the longest-first list
    degridder_sep_block<L>(a, b, a.n_items, gridDim.x, sep_smem);
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
  degridder_sep_block<L>(*reinterpret_cast<const DegridArgs*>(s_args_raw), it.y, it.y + 1, 1, sep_smem);
}

template <int L>
int configure_degridder_sep_l(int* persistent_blocks) {
  cudaError_t e = cudaFuncSetAttribute(degridder_sep_kernel<L>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kSepSmemLimit);
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
  const int blocks = persistent_blocks > 0 ? (persistent_blocks < n_items ? persistent_blocks : n_items)
                                           : (n_items + bundle - 1) / bundle;
  degridder_sep_kernel<L><<<blocks, kSepThreads, dsep_smem<L>(a.kv, a.g.nodes), cudaStream_t(stream)>>>(
      a, persistent_blocks > 0 ? 0 : bundle);
  return int(cudaGetLastError());
}

template <int L>
int launch_degridder_sep_multi_l(const DegridArgs* args, const int2* items, int n_items, int max_nodes,
                                 void* stream) {
  if (n_items <= 0) return 0;
  size_t smem = 0;  // the largest layout of any plan of up to max_nodes (a plan's items are cut to its own)
  for (int n = 2; n <= max_nodes; ++n) {
    const size_t s = dsep_smem<L>(dsep_vis<L>(n), n);
    smem = s > smem ? s : smem;
  }
  degridder_sep_multi_kernel<L><<<n_items, kSepThreads, smem, cudaStream_t(stream)>>>(args, items);
  return int(cudaGetLastError());
}

}  // namespace idg
