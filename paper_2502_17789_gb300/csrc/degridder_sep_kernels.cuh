// Degridder with separable phasors (templates), included by the per-subgrid-size
// translation units degridder_sep_lNN.cu.  See sep_common.cuh for the split
// of the phase; this is the adjoint of gridder_sep_kernels.cuh.
//
// For one A-term segment, Z = A_p Y A_q^H with Y the subgrid image times
// taper, centring sign and e^{-2 pi i w_ref n'} (sep_pixel; applied by the splitter):
//   V_k = sum_i conj(E_k(i)) D_k(i),
//   D_k(i) = sum_j Z(i,j) conj(F_k(j)) (1 - 2 pi i delta_k p_i q_j).
// D is a complex matrix product on the tensor cores: rows (p, i) for 4
// correlations x 32 pixel columns, contraction over the L rows j, columns the
// item's visibilities k (real and imaginary sums as two accumulators), so a
// short segment makes a narrow product instead of an empty one.  The remaining
// sum over i takes one complex multiply-add per (visibility, column), 1/L of
// the direct sum.
//
// A block of 20 warps works through a share of the items (an item is up to kv
// visibilities of one segment); its warps have roles that run side by side.
// Producers (three groups of 4 warps, pieces in turn): per piece of 16 rows j of a block of 32 columns, thread = row
// (p, i) x 16 rows j writes Z to tensor memory, from Y pieces that a loading warp
// copies to shared memory up to four pieces ahead; an issuing warp starts the piece's
// 16 MMAs, whose commit frees it.  Consumers take the accumulators, which alternate
// between two column ranges of tensor memory from column block to column
// block, through the sum over i: a transposing butterfly adds the 32 columns of a
// warp.  Preparing warps write the next item's phase slopes, F side of all L
// rows and A-term samples (double buffers) while one runs.
//
// What bounds it: the producers' issue slots and instruction supply (81 % of the slots, tensor pipe 31 %;
// profiles/degridder_sep_mwa_like_90st.md).  With all threads
// doing each step in turn and Z in shared memory it took 46.8 ms (MWA-like workload, 96 x
// 96 subgrids, segments of about 60 visibilities, per degrid call on GB300), with a half
// of producers in step and a half of consumers 31.4 ms, with roles and a thread's 8 rows
// of a piece written out 19.7 ms; 16 rows per thread pay a piece's waits and set-up for
// twice the rows, and four rows at a time in a loop keep the code small (18.2 ms; full
// Jones matrices, 64 stations: 1.43 -> 1.16; written out 16 times 20.6 and 1.65).  The
// kernel with one phasor per visibility and pixel (degridder_tc_kernels.cuh) takes 78.4 ms.  With subgrids of a wide w range
// in parts it is 18.8 ms.
#pragma once

#include "sep_common.cuh"

namespace idg {

constexpr int kDsepMaxVis = 64;   // visibilities per item at most
constexpr int kDsepRing = 4;      // Y pieces in shared memory, Z pieces in tensor memory
// roles: three producer groups of 4 warps, 4 consumer warps, the issuing warp, the loading warp, 2 preparing warps
constexpr int kDsepGroups = 3;
// Arrivals of Y pieces have a barrier per (slot, group) pair in turn: a wait on a barrier's parity is only sound for a
// warp that has waited for every phase before it, and a slot's pieces go to the groups in rotation, so with one barrier
// per slot a group could take the phase of a piece that is still on its way to another group for its own.
constexpr int kDsepLoaded = 12;
static_assert(kDsepLoaded % kDsepGroups == 0 && kDsepLoaded % kDsepRing == 0,
              "a barrier's pieces belong to one group and slot");
constexpr int kDsepThreads = 640, kDsepConsumer = 384, kDsepIssuer = 512, kDsepLoader = 544, kDsepPreparer = 576;
constexpr int kDsepPreparers = 64;
static_assert(kDsepMaxVis <= kDsepPreparers, "a visibility per preparing thread");
constexpr int kDsepPreparerBar = 4;
// registers per thread: 96 at launch, then by role
constexpr int kDsepLaunchRegs = 96, kDsepProducerRegs = 88, kDsepConsumerRegs = 136, kDsepOtherRegs = 80;
static_assert(kDsepConsumer * kDsepProducerRegs + 128 * (kDsepConsumerRegs + kDsepOtherRegs) <= kDsepThreads * kDsepLaunchRegs,
              "registers");
constexpr int kDsepColStride = 2 * kDsepMaxVis;       // between the two accumulators (re, im)
constexpr int kDsepZCol = 2 * kDsepColStride;         // first column of the Z ring
// Items of few visibilities have a kernel of their own (idg_plan_create says which), which keeps the accuracy of the FP32
// kernels that take them elsewhere (errors of single-channel plans at L = 32 .. 128: 3.2 .. 5.0e-7 without it, 2.4 ..
// 3.0e-7 with it, 2.3 .. 3.7e-7 on FP32): the corrections have accumulators of their own (sep_product) in the columns
// that the visibilities leave, and the F side exact sines and cosines.  As branches of the one kernel they cost its
// regular items 8 % (22.8 ms on the MWA-like workload).
constexpr int kDsepFewCorr = kDsepMaxVis;   // columns from the sums to the corrections
static_assert(kDsepFewVis % 16 == 0 && 2 * kDsepFewVis <= kDsepFewCorr, "corrections beside the sums");
constexpr uint32_t kDsepTmemCols = 512;
static_assert(kDsepZCol + kDsepRing * 48 <= int(kDsepTmemCols), "tensor memory");

struct alignas(128) DsepShared {
  float2 y[kDsepRing][4][8][2][32];  // [piece][pol][row pair][re, im][column]
  float fix_a[2][kDsepMaxVis], fix_b[2][kDsepMaxVis], delta[2][kDsepMaxVis];  // [item parity][visibility]
  float out[kDsepMaxVis][8];
  // the producers' part of an item, by item parity
  struct Info {
    float scale[4];  // of each correlation's Z, a power of two
    int sg, diag;
  } info[2];
  uint64_t ready[2];        // item prepared (2 preparing warps)
  uint64_t loaded[kDsepLoaded];  // Y piece copied, by piece modulo kDsepLoaded
  uint64_t done[2];         // item's visibilities written, its operands read (4 consumer warps)
  uint64_t filled[kDsepRing]; // Z piece written (4 producer warps)
  uint64_t empty[kDsepRing];  // Z piece read by its MMAs
  uint64_t full[2];         // accumulator complete
  uint64_t drained[2];      // accumulator read (4 consumer warps)
  uint64_t drain;           // every MMA complete, after a wait that gave up
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

template <int L, bool FEW>
struct Dsep {
  const DegridArgs& a;
  DsepShared& S;
  unsigned char* fside;   // [item parity][level][16 rows][k group][Re, Im][visibility] rows of 16 bytes
  float4* raw;            // [item parity][station][nodes][nodes][2]
  const SepShare share;

  static constexpr int kBlocks = L / 32, kPieces = L / 16;
  static constexpr int kGroups16 = (FEW ? kDsepFewVis : kDsepMaxVis) / 16;

  template <int SLEEP = 32>
  __device__ __forceinline__ void wait(uint64_t* bar, uint32_t parity) {
    sep_wait<SLEEP>(bar, parity, &S.fail, a);
  }

  // ---------------------------------------------------------------- producers

  // Z of rows 16 jc .. for column block ib: thread = (p, i) x 16 rows j.  QUAD: node cells start at multiples of four
  // rows, so the cell can change only there and not at every row.
  template <bool DIAG, bool QUAD>
  __device__ __forceinline__ void produce(uint32_t e_col, const float2* yb, const float4* samples, float scale,
                                          NodeWeight wx, int jc, __half2 fit_p) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int p = warp & 3, pa = p >> 1, pb = p & 1;
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
    // row r of the piece lies at (rem + step r) / L of the cell that starts at node row `at`; four rows at a time, in
    // a loop that stays small: with the rows written out 16 times the warps wait for instructions
    int at = step * 16 * jc / L, rem = step * 16 * jc - at * L;
    load_cell(at);
    const float df = float(step) * (1.f / float(L));
    const float2* y0 = yb + lane;  // [pol][row pair][re, im][column]
    uint32_t dst = e_col + (uint32_t(p * 32) << 16);
#pragma unroll 1
    for (int r = 0; r < 4; ++r, dst += 2, y0 += 128, rem += 4 * step) {
      uint32_t re_hi[2], re_lo[2], re_c[2], im_hi[2], im_lo[2], im_c[2];
      float f0 = float(rem) * (1.f / float(L));
#pragma unroll
      for (int w = 0; w < 2; ++w) {
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
          if (!QUAD || q == 0) {
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
      tmem_st2(dst, re_hi[0], re_hi[1]);
      tmem_st2(dst + 8, im_hi[0], im_hi[1]);
      tmem_st2(dst + 16, re_lo[0], re_lo[1]);
      tmem_st2(dst + 24, im_lo[0], im_lo[1]);
      tmem_st2(dst + 32, re_c[0], re_c[1]);
      tmem_st2(dst + 40, im_c[0], im_c[1]);
    }
  }

  // the groups take the block's pieces in turn; the warps of a group go their own way between the rings' barriers
  __device__ __forceinline__ void producer() {
    constexpr uint32_t kItemPieces = kBlocks * kPieces;
    const int lane = threadIdx.x & 31, nodes = a.g.nodes;
    const bool quad = L % (nodes - 1) == 0 && L / (nodes - 1) % 4 == 0;
    const uint32_t tm = S.tmem;
    const float inv_p = 1.f / a.sep.p_scale;
    uint32_t n = 0, pg = uniform_warp() >> 2, base = 0;  // items so far, the group's next piece, the item's first
    for (int idx = share.first; idx < share.last; idx = share.next(idx), ++n, base += kItemPieces) {
      // an item without a piece of this group is passed over: its barriers may be phases ahead
      if (pg >= base + kItemPieces) continue;
      wait(&S.ready[n & 1], (n >> 1) & 1);
      const float scale = S.info[n & 1].scale[(threadIdx.x >> 5) & 3];
      const bool diag = S.info[n & 1].diag != 0;
      const float4* samples = raw + (n & 1) * 4 * nodes * nodes;
#pragma unroll 1
      for (; pg < base + kItemPieces; pg += kDsepGroups) {
        const int t = pg - base, ib = t / kPieces, jc = t - ib * kPieces, i = ib * 32 + lane;
        const NodeWeight wx = node_weight(i, nodes, L);
        const __half2 fit_p = __float2half2_rn(__ldg(a.sep.p + i) * inv_p);
        const uint32_t slot = pg % kDsepRing;
        wait(&S.loaded[pg % kDsepLoaded], (pg / kDsepLoaded) & 1);
        if (pg >= uint32_t(kDsepRing)) tc_fence_after();  // the loader has seen the slot's last MMAs complete
        const uint32_t e_col = tm + kDsepZCol + slot * 48;
        const float2* y = &S.y[slot][0][0][0][0];
        if (quad) {
          if (diag)
            produce<true, true>(e_col, y, samples, scale, wx, jc, fit_p);
          else
            produce<false, true>(e_col, y, samples, scale, wx, jc, fit_p);
        } else if (diag) {
          produce<true, false>(e_col, y, samples, scale, wx, jc, fit_p);
        } else {
          produce<false, false>(e_col, y, samples, scale, wx, jc, fit_p);
        }
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&S.filled[slot]);
      }
    }
  }

  // ---------------------------------------------------------------- loader (one warp)

  // Y in scratch: [pol][column block][row pair][re, im][32 columns], so a piece is one run of 4 KB per plane
  __device__ __forceinline__ void loader() {
    uint32_t n = 0, pg = 0;  // items and pieces of this block so far
    uint32_t issued = 0;     // pieces the elected lane has started to copy
    for (int idx = share.first; idx < share.last; idx = share.next(idx), ++n) {
      wait<64>(&S.ready[n & 1], (n >> 1) & 1);
      const float2* Y = a.scratch + size_t(S.info[n & 1].sg) * 4 * L * L;
#pragma unroll 1
      for (int t = 0; t < kBlocks * kPieces; ++t, ++pg) {
        const uint32_t slot = pg % kDsepRing, turn = pg / kDsepRing;
        // the slot's previous piece of Y has been read and its Z multiplied: one wait less for every producer
        if (turn > 0) wait(&S.empty[slot], (turn - 1) & 1);
        __syncwarp();
        // none after a wait that gave up: the subgrid, and the barrier's phase, may then be anything
        if (elect_one() && !sep_failed(&S.fail)) {
          mbar_arrive_expect_tx(&S.loaded[pg % kDsepLoaded], 4096 * a.g.npol);
          for (int pol = 0; pol < a.g.npol; ++pol)
            bulk_copy_g2s(&S.y[slot][pol][0][0][0], Y + size_t(pol) * L * L + t * 512, 4096, &S.loaded[pg % kDsepLoaded]);
          ++issued;
        }
        __syncwarp();
      }
    }
    // the producers wait for every piece, but not once a wait of theirs has given up
    if (elect_one())
      for (uint32_t k = issued > kDsepLoaded ? issued - kDsepLoaded : 0; k < issued; ++k)
        mbar_wait_bounded(&S.loaded[k % kDsepLoaded], (k / kDsepLoaded) & 1);
  }

  // ---------------------------------------------------------------- issuer (one warp)

  __device__ __forceinline__ void issuer() {
    const uint32_t tm = S.tmem;
    uint32_t n = 0, pg = 0, dg = 0;  // items, pieces and accumulators of this block so far
    // columns of an item: from the item itself, a step ahead, so that the MMAs' shapes and operands are the block's own
    // also after a wait that gave up (their sums are lost then, and sep_drain waits for them)
    const auto columns = [&](int idx) {
      return idx < share.last ? (a.items[idx].k_end - a.items[idx].k_begin + 15) & ~15 : 16;
    };
    int n_next = columns(share.first);
    for (int idx = share.first; idx < share.last; idx = share.next(idx), ++n) {
      const int n_pad = n_next;
      n_next = columns(share.next(idx));
      wait(&S.ready[n & 1], (n >> 1) & 1);
      const uint32_t block = uint32_t(n_pad) * 16, group = 2 * block, chunk = 2 * group, level = kPieces * chunk;
      const uint32_t f0 = smem_u32(fside) + (n & 1) * uint32_t(a.kv) * L * 12;
#pragma unroll 1
      for (int ib = 0; ib < kBlocks; ++ib, ++dg) {
        // the accumulator's previous column block (two back) has been read
        if (dg >= 2) wait(&S.drained[dg & 1], ((dg >> 1) - 1) & 1);
#pragma unroll 1
        for (int jc = 0; jc < kPieces; ++jc, ++pg) {
          const uint32_t slot = pg % kDsepRing;
          wait(&S.filled[slot], (pg / kDsepRing) & 1);
          tc_fence_after();
          __syncwarp();
          if (elect_one()) {
            sep_product<FEW ? kDsepFewCorr : 0>(tm + (dg & 1) * kDsepColStride, tm + kDsepZCol + slot * 48,
                                                f0 + jc * chunk, n_pad, block, group, level, jc == 0);
            sep_commit(&S.empty[slot]);
            if (jc + 1 == kPieces) sep_commit(&S.full[dg & 1]);
          }
          __syncwarp();
        }
      }
    }
  }

  // ---------------------------------------------------------------- preparers

  // item idx, number n of the block: phase slopes, A-term samples, conj(F) at all rows, the producers' part
  __device__ __forceinline__ void prepare(int idx, uint32_t n) {
    const int tid = threadIdx.x - kDsepPreparer, lane = tid & 31;
    const DegridItem item = a.items[idx];
    const SubgridDesc sd = a.sg[item.sg];
    const SegmentDesc seg = a.seg[item.segment];
    const int nv = item.k_end - item.k_begin, n_pad = (nv + 15) & ~15, b = n & 1;
    const int nodes = a.g.nodes, n4 = nodes * nodes * 2;
    const int sp = seg.interval * a.g.n_st + sd.p, sq = seg.interval * a.g.n_st + sd.q;
    // what comes from global memory, before the buffers are free
    int fa = 0, fb = 0;
    float dl = 0.f;
    if (tid < nv) {
      const int nc = sd.c1 - sd.c0, k = item.k_begin + tid, row = k / nc, ch = sd.c0 + (k - row * nc);
      const double* r = a.uvw + (size_t(sd.b) * a.g.n_t + sd.t0 + row) * 3;
      const double fs = subgrid_sign(sd) * a.fscale[ch], inv_l = 1.0 / double(L);
      fa = sep_fix(((r[0] * fs) * a.g.fov - double(sd.x0 + L / 2 - a.g.N / 2)) * inv_l);
      fb = sep_fix(((r[1] * fs) * a.g.fov - double(sd.y0 + L / 2 - a.g.N / 2)) * inv_l);
      dl = float(r[2] * fs - (double(a.w_ref[item.sg].x) + subgrid_w0(a.g, sd)));
    }
    // scale of each correlation's Z = A_p Y A_q^H (thread = correlation (r, c)) from the largest components of Y and of
    // the A-terms' nodes: a faint correlation keeps its bits beside a bright one
    const int diag = a.adiag[sp] & a.adiag[sq];
    float bound;
    {
      const float4 am = a.amax[sp], bm = a.amax[sq], y = *reinterpret_cast<const float4*>(a.ymax + item.sg * 4);
      const int r = (tid >> 1) & 1, c = tid & 1;
      const float p0 = r ? am.z : am.x, p1 = r ? am.w : am.y, q0 = c ? bm.z : bm.x, q1 = c ? bm.w : bm.y;
      if (a.g.npol == 1)
        bound = diag ? (r == c ? (r ? p1 * q1 : p0 * q0) * y.x : 0.f) : (p0 * q0 + p1 * q1) * y.x;
      else if (diag)
        bound = (r ? p1 : p0) * (r ? (c ? y.w : y.z) : (c ? y.y : y.x)) * (c ? q1 : q0);
      else
        bound = p0 * (y.x * q0 + y.y * q1) + p1 * (y.z * q0 + y.w * q1);
    }
    if (n >= 2) wait<100>(&S.done[b], ((n >> 1) - 1) & 1);  // the buffers' previous item (two back) is done
    {
      const float4* src = reinterpret_cast<const float4*>(a.aterms);
      float4* dst = raw + size_t(b) * 2 * n4;
      for (int e = tid; e < 2 * n4; e += kDsepPreparers)
        cp_async16(dst + e, src + (e < n4 ? size_t(sp) * n4 + e : size_t(sq) * n4 + e - n4));
      cp_async_commit();
    }
    if (tid < n_pad) {
      S.fix_a[b][tid] = __int_as_float(fa);
      S.fix_b[b][tid] = __int_as_float(fb);
      S.delta[b][tid] = dl;
    }
    if (tid < 4) S.info[b].scale[tid] = sep_scale(bound);
    if (tid == 0) {
      S.info[b].sg = item.sg;
      S.info[b].diag = diag;
    }
    asm volatile("bar.sync %0, %1;" ::"n"(kDsepPreparerBar), "n"(kDsepPreparers) : "memory");
    const uint32_t block = uint32_t(n_pad) * 16, group = 2 * block, chunk = 2 * group, level = kPieces * chunk;
    const uint32_t base = smem_u32(fside) + b * uint32_t(a.kv) * L * 12;
    for (int e = tid; e < n_pad * (L / 8); e += kDsepPreparers) {
      const int o = e / n_pad, k = e - o * n_pad;
      const int fix = __float_as_int(S.fix_b[b][k]);
      const float dl = S.delta[b][k], dp = dl * a.sep.p_scale;
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
          if (FEW) {
            sep_sincos_exact(fix, off, dl, fb.x, &s.x, &c.x);
            sep_sincos_exact(fix, off + 1, dl, fb.y, &s.y, &c.y);
          } else {
            __sincosf(sep_phase(fix, off, dl, fb.x), &s.x, &c.x);
            __sincosf(sep_phase(fix, off + 1, dl, fb.y), &s.y, &c.y);
          }
          const __half2 d2 = __floats2half2_rn(-dp * fq.x, -dp * fq.y);
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

  __device__ __forceinline__ void preparer() {
    uint32_t n = 0;
    for (int idx = share.first; idx < share.last; idx = share.next(idx), ++n) prepare(idx, n);
  }

  // ---------------------------------------------------------------- consumers

  // thread = row (p, i) of the column block
  __device__ __forceinline__ void consumer() {
    const int tid = threadIdx.x - kDsepConsumer, pol = tid >> 5, lane = tid & 31;
    uint32_t dg = 0, n = 0;  // accumulators and items of this block so far
    for (int idx = share.first; idx < share.last; idx = share.next(idx), ++n) {
      const DegridItem item = a.items[idx];
      const int nv = item.k_end - item.k_begin, n_pad = (nv + 15) & ~15, b = n & 1;
      wait(&S.ready[b], (n >> 1) & 1);
      const float inv = sep_unbias(FEW ? 0.25f * kPieces : float(kPieces)) / S.info[b].scale[pol];
      float sum[kGroups16];  // component lane & 1 of visibility 16 h + lane / 2
#pragma unroll
      for (int h = 0; h < kGroups16; ++h) sum[h] = 0.f;
#pragma unroll 1
      for (int ib = 0; ib < kBlocks; ++ib, ++dg) {
        const int i = ib * 32 + lane;
        const float fit_a = __ldg(a.sep.a + i);
        wait<250>(&S.full[dg & 1], (dg >> 1) & 1);
        tc_fence_after();
        const uint32_t d = S.tmem + (uint32_t(pol * 32) << 16) + (dg & 1) * kDsepColStride;
#pragma unroll
        for (int h = 0; h < kGroups16; ++h) {
          const int k0 = 16 * h;
          if (k0 < n_pad) {
            float v[32];  // (re, im) of 16 visibilities
            {
              float dr[16], di[16];
              tmem_ld16(dr, d + k0);
              tmem_ld16(di, d + n_pad + k0);
              tmem_wait_ld();
              if (FEW) {
                float cr[16], ci[16];
                tmem_ld16(cr, d + kDsepFewCorr + k0);
                tmem_ld16(ci, d + kDsepFewCorr + n_pad + k0);
                tmem_wait_ld();
#pragma unroll
                for (int k = 0; k < 16; ++k) {
                  dr[k] += cr[k];
                  di[k] += ci[k];
                }
              }
              const float4* fx = reinterpret_cast<const float4*>(&S.fix_a[b][k0]);
              const float4* dl = reinterpret_cast<const float4*>(&S.delta[b][k0]);
#pragma unroll
              for (int k = 0; k < 16; ++k) {
                const float4 f4 = fx[k >> 2], d4 = dl[k >> 2];
                const float f = (k & 3) == 0 ? f4.x : (k & 3) == 1 ? f4.y : (k & 3) == 2 ? f4.z : f4.w;
                const float dk = (k & 3) == 0 ? d4.x : (k & 3) == 1 ? d4.y : (k & 3) == 2 ? d4.z : d4.w;
                float c, s;
                __sincosf(sep_phase(__float_as_int(f), i - L / 2, dk, fit_a), &s, &c);
                v[2 * k] = fmaf(dr[k], c, di[k] * s);
                v[2 * k + 1] = fmaf(di[k], c, -dr[k] * s);
              }
            }
            // sum over the 32 columns of the warp, lane l ending with value l
#pragma unroll
            for (int w = 16; w; w >>= 1) {
              const bool up = lane & w;
#pragma unroll
              for (int k = 0; k < w; ++k) {
                const float keep = up ? v[k + w] : v[k], give = up ? v[k] : v[k + w];
                v[k] = keep + __shfl_xor_sync(0xffffffffu, give, w);
              }
            }
            sum[h] += v[0];
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&S.drained[dg & 1]);
      }
#pragma unroll
      for (int h = 0; h < kGroups16; ++h)
        if (16 * h < n_pad) S.out[16 * h + (lane >> 1)][2 * pol + (lane & 1)] = inv * sum[h];
      asm volatile("bar.sync %0, 128;" ::"n"(kSepConsumerBar) : "memory");
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
      if (lane == 0) mbar_arrive(&S.done[b]);
      asm volatile("bar.sync %0, 128;" ::"n"(kSepConsumerBar) : "memory");  // S.out free
    }
  }
};

template <int L, bool FEW = false>
__device__ __forceinline__ void degridder_sep_block(const DegridArgs& a, SepShare share, unsigned char* smem) {
  DsepShared& S = *reinterpret_cast<DsepShared*>(smem);
  unsigned char* fside = reinterpret_cast<unsigned char*>(&S + 1);
  if (threadIdx.x == 0) {
    for (int k = 0; k < kDsepRing; ++k) {
      mbar_init(&S.empty[k], 1);
      mbar_init(&S.filled[k], 4);
    }
    for (int k = 0; k < kDsepLoaded; ++k) mbar_init(&S.loaded[k], 1);
    mbar_init(&S.drain, 1);
    for (int k = 0; k < 2; ++k) {
      mbar_init(&S.full[k], 1);
      mbar_init(&S.drained[k], 4);
      mbar_init(&S.ready[k], kDsepPreparers / 32);
      mbar_init(&S.done[k], 4);
    }
    fence_mbar_init();
    S.fail = 0;
  }
  if (threadIdx.x < 32) tmem_alloc(&S.tmem, kDsepTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  Dsep<L, FEW> it{a, S, fside, reinterpret_cast<float4*>(fside + size_t(2) * a.kv * L * 12), share};
  if (threadIdx.x < kDsepConsumer) {
    regs_give<kDsepProducerRegs>();
    it.producer();
  } else if (threadIdx.x < kDsepIssuer) {
    regs_take<kDsepConsumerRegs>();
    it.consumer();
  } else {
    regs_give<kDsepOtherRegs>();
    if (threadIdx.x < kDsepLoader)
      it.issuer();
    else if (threadIdx.x < kDsepPreparer)
      it.loader();
    else
      it.preparer();
  }
  sep_drain(&S.fail, uniform_warp() == kDsepIssuer / 32, &S.drain);
  if (threadIdx.x < 32) {
    tc_fence_after();
    tmem_free(S.tmem, kDsepTmemCols);
  }
}

template <int L>
__global__ void __launch_bounds__(kDsepThreads, 1) degridder_sep_kernel(const DegridArgs a) {
  extern __shared__ __align__(128) unsigned char sep_smem[];
  degridder_sep_block<L>(a, SepShare{int(blockIdx.x) * a.run, a.n_items, int(gridDim.x), a.run}, sep_smem);
}

// One launch over the items of several plans: blocks = (plan slot, first run), each taking every `stride`-th run of its
// plan from there
template <int L>
__global__ void __launch_bounds__(kDsepThreads, 1) degridder_sep_multi_kernel(const DegridArgs* args,
                                                                            const int2* blocks) {
  extern __shared__ __align__(128) unsigned char sep_smem[];
  __shared__ __align__(16) unsigned char s_args_raw[sizeof(DegridArgs)];
  const int2 it = blocks[blockIdx.x];
  if (threadIdx.x == 0) memcpy(s_args_raw, args + it.x, sizeof(DegridArgs));
  __syncthreads();
  const DegridArgs& a = *reinterpret_cast<const DegridArgs*>(s_args_raw);
  degridder_sep_block<L>(a, SepShare{it.y * a.run, a.n_items, a.stride, a.run}, sep_smem);
}

// The same two for items of at most kDsepFewVis visibilities
template <int L>
__global__ void __launch_bounds__(kDsepThreads, 1) degridder_sep_few_kernel(const DegridArgs a) {
  extern __shared__ __align__(128) unsigned char sep_smem[];
  degridder_sep_block<L, true>(a, SepShare{int(blockIdx.x) * a.run, a.n_items, int(gridDim.x), a.run}, sep_smem);
}

template <int L>
__global__ void __launch_bounds__(kDsepThreads, 1) degridder_sep_few_multi_kernel(const DegridArgs* args,
                                                                                const int2* blocks) {
  extern __shared__ __align__(128) unsigned char sep_smem[];
  __shared__ __align__(16) unsigned char s_args_raw[sizeof(DegridArgs)];
  const int2 it = blocks[blockIdx.x];
  if (threadIdx.x == 0) memcpy(s_args_raw, args + it.x, sizeof(DegridArgs));
  __syncthreads();
  const DegridArgs& a = *reinterpret_cast<const DegridArgs*>(s_args_raw);
  degridder_sep_block<L, true>(a, SepShare{it.y * a.run, a.n_items, a.stride, a.run}, sep_smem);
}

template <int L>
int configure_degridder_sep_l(int* persistent_blocks) {
  // the roles' register split is of the registers the block is launched with
  cudaError_t e = cudaSuccess;
  const auto configure = [&e](auto kernel) {
    if (e == cudaSuccess) e = sep_check_regs(kernel, kDsepLaunchRegs);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSepSmemLimit);
  };
  configure(degridder_sep_kernel<L>);
  configure(degridder_sep_multi_kernel<L>);
  configure(degridder_sep_few_kernel<L>);
  configure(degridder_sep_few_multi_kernel<L>);
  int dev = 0, sms = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  *persistent_blocks = sms;  // one block per SM (registers, tensor memory)
  return int(e);
}

template <int L>
int degridder_sep_vis_l(int nodes) {
  return dsep_vis<L>(nodes);
}

template <int L>
int launch_degridder_sep_l(const DegridArgs& args, int n_items, int blocks, bool few, void* stream) {
  if (n_items <= 0) return 0;
  DegridArgs a = args;
  a.n_items = n_items;
  const size_t smem = dsep_smem<L>(a.kv, a.g.nodes);
  if (few)
    degridder_sep_few_kernel<L><<<blocks, kDsepThreads, smem, cudaStream_t(stream)>>>(a);
  else
    degridder_sep_kernel<L><<<blocks, kDsepThreads, smem, cudaStream_t(stream)>>>(a);
  return int(cudaGetLastError());
}

template <int L>
int launch_degridder_sep_multi_l(const DegridArgs* args, const int2* blocks, int n_blocks, int max_nodes, bool few,
                                 void* stream) {
  if (n_blocks <= 0) return 0;
  size_t smem = 0;  // the largest layout of any plan of up to max_nodes (a plan's items are cut to its own)
  for (int n = 2; n <= max_nodes; ++n) {
    const size_t s = dsep_smem<L>(dsep_vis<L>(n), n);
    smem = s > smem ? s : smem;
  }
  if (few)
    degridder_sep_few_multi_kernel<L><<<n_blocks, kDsepThreads, smem, cudaStream_t(stream)>>>(args, blocks);
  else
    degridder_sep_multi_kernel<L><<<n_blocks, kDsepThreads, smem, cudaStream_t(stream)>>>(args, blocks);
  return int(cudaGetLastError());
}

}  // namespace idg
