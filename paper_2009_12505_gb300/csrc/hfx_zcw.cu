// HFX_OZAKI: the D_FG and D_FB pieces for jobs with a block or an atom A of
// more than 16 AOs (hfx_zc.cu has the products, the job plan and the kernel for
// smaller blocks).
//
// The first product, Z = sum_F C_AF D, is the one of k_zc.  Its contraction with
// Y costs nao(B) or nao(G) multiply-adds per Z element, in double-float twelve
// operations a pair, and at 27 AOs that was three quarters of the time; here it
// is a second tensor-core product, on the mma.sync path because its operands
// are registers:
//  * a row tile of A holds whole al (ZcRows), so row r of every tile is the same
//    a, and the sums over al are sums over tiles and slots in place;
//  * tcgen05.ld 16x256b gives a warp a 16 x 16 piece of Z in the fragment layout
//    of mma.sync's A operand; each epilogue warp takes one such piece (its rows
//    and column group) and no data moves between warps until the job ends;
//  * Z and Y become six digits of 8 bits (exact in bf16), Z with an exponent per
//    row of the fragment, Y with one per (al, output); D's column exponents, which
//    Z's columns are in units of, are multiplied into Y.  Digit products of one
//    order are exact in f32; the orders, scaled by both exponents, join the
//    double-float sum of their (row, output).
// Precision: the digits drop what is 2^-48 below the largest Z of the row times the
// largest Y of that al and output (over at most 16 columns, each in units of its
// D column).  The first product has already rounded every Z to 2^-42 of its C row
// times its D column, so each element of Sigma, small or large, has the error of
// the first product alone.  (One exponent per al and a scale per job, relative to
// the largest product of all, left outputs 2^-24 below the largest with 24 bits.)
//
// Roles (one CTA per SM, persistent): warps 0-15 as above; warp 16 streams A and
// B tiles into a ring of shared stages, warp 17 issues the tcgen05 MMAs into one
// of two TMEM accumulators, warp 18 copies each tile's Y rows and row
// exponents.  Every wait is bounded; on expiry the kernel records
// HFX_DEV_ERR_TIMEOUT, drains its copies and MMAs, frees TMEM and returns.
//
// What bounds it: the epilogue, beside up to 22 operand stages a tile.  8-atom
// two-element cell (13/60 and 27/90, C, D to 9 bohr): 178.7 ms for its wide jobs
// with a double-float contraction from global memory, 127 ms with that contraction
// halved and Y staged, 109.7 ms with this product and two warps that looked for
// one exponent per al before a tile could be read, 97.8 ms with the exponents taken
// from each fragment's own loads (35 ms of bf16 products at the sustained peak).
#include "zc_common.cuh"

namespace split {

// Epilogue: 16 warps, one per TMEM lane quarter, group of 16 columns and 16-row
// fragment, so that each scheduler has four of them to hide latencies; with the
// other roles a scheduler has five warps, which leaves 96 registers a thread, too
// few for the digits, order groups and sums at once: ptxas spills 572 bytes a
// thread (952 of loads).
constexpr int ZC_EPI = 16;
constexpr int ZC_NQ = 2;                         // column groups
constexpr int ZC_CW = ZC_COLS / ZC_NQ;           // Z columns per epilogue warp
constexpr int ZC_ET = ZC_EPI * 32;               // epilogue threads
constexpr int ZC_THREADS = (ZC_EPI + 3) * 32;    // + A/B loader, MMA issuer, Y loader
// Staged Y rows of one al end with a pad of ZC_YPAD pairs, which moves the rows
// of the next al to other banks.
constexpr int ZC_YPAD = 2;
constexpr int ZC_PASS = 8;   // outputs of a block per pass through the reduction buffer
constexpr int ZC_DIG = 6;    // digits of the second product's operands (8 bits each)

struct ZcwSmem {
  uint64_t full[8], empty[8], tfull[2], tempty[2], yfull, yempty, drain;
  unsigned long long t_start;  // globaltimer at the start of the roles
  uint32_t tslot;
  int abort_f;
  __align__(16) int16_t erow[128];  // row exponents of the tile that Y is staged for
  // column exponents of the pair's jobs: the largest of each column group, and
  // each column's 2^(exponent - largest) (column group q at q * CW)
  int emax[2][ZC_NQ];
  __align__(8) float cw[2][ZC_COLS];
  ZcEpiJob ej[2][2];     // [pair parity][job of the pair]
};

// 2^e as f32: zero below the normal range, 2^127 above it (both are far outside
// what Sigma's words hold, |x| from 2^-64 to 2^31).
__device__ __forceinline__ float zc_exp2(int e) {
  return e < -126 ? 0.f : __int_as_float((min(e, 127) + 127) << 23);
}

// From the largest magnitude's bit pattern: e with |x| < 2^e, and 2^-e (NaN from
// 2^126 on, infinities and NaN included: the sums carry it to the range check).
__device__ __forceinline__ int zc_exp_of(uint32_t m, float &sc) {
  const int f = (int)(m >> 23);
  sc = f > 252 ? __int_as_float(0x7FC00000) : __int_as_float((253 - f) << 23);
  return f - 126;
}

__device__ __forceinline__ uint32_t zc_max_abs(uint64_t v) {
  const float2 x = f2_un(v);
  return max(__float_as_uint(fabsf(x.x)), __float_as_uint(fabsf(x.y)));
}

__device__ __forceinline__ void zc_mma(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                       uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// The next digit of two elements (f32x2 lanes) given as pairs, |h| <= 1 at
// first.  ZC_DIG digits of 8 bits: digit i is a multiple of 2^-(7 + 8 i),
// exact in bf16, and the digits' sum is within 2^-48 of the element.  Adding
// and taking away 1.5 2^(16 - 8 i) rounds h to that multiple; the rest stays
// in h, exactly, and the low words l join it once it is below them.
__device__ __forceinline__ uint32_t zc_digit(int i, uint64_t &h, uint64_t l) {
  const float m = __int_as_float(((16 - 8 * i + 127) << 23) | 0x400000);
  const uint64_t M = f2_pk(m, m);
  const uint64_t t = f2_sub(f2_add(h, M), M);
  h = f2_sub(h, t);
  if (i == 2) h = f2_add(h, l);
  const float2 v = f2_un(t);
  uint32_t d;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(v.y), "f"(v.x));
  return d;
}

// This lane's part of the 16 x 8 fragment of Y (contracted index k .. = kc +
// {0, 1, 8, 9}, one output): pairs y[k] (P1) or y[16 k], times the column weights
// cw, as f32x2 of the high and of the low words.  nk: valid k; live: it is an
// output.
template <bool P1>
__device__ __forceinline__ void zc_y_frag(const float2 *__restrict__ y, int k, int nk, bool live,
                                          const float *cw, uint64_t (&h)[2], uint64_t (&l)[2]) {
  float2 v[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int ku = k + (u & 1) + 8 * (u >> 1);
    v[u] = live && ku < nk ? y[ku * (P1 ? 1 : 16)] : make_float2(0.f, 0.f);
  }
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const float2 w = *reinterpret_cast<const float2 *>(cw + k + 8 * u);
    const uint64_t w2 = f2_pk(w.x, w.y);
    h[u] = f2_mul(f2_pk(v[2 * u].x, v[2 * u + 1].x), w2);
    l[u] = f2_mul(f2_pk(v[2 * u].y, v[2 * u + 1].y), w2);
  }
}

// Exchange v with this warp's 2 N spare TMEM columns at ta (the sums of the
// pair's other job); load == false: store v and take zeros.
template <int N>
__device__ __forceinline__ void zc_exchange(uint32_t ta, uint64_t (&v)[N], bool load) {
  uint32_t r[N / 8][16];
  umma::tmem_wait_st();  // of the exchange before
#pragma unroll
  for (int c = 0; c < N / 8; ++c) umma::tmem_ld16_nowait(ta + 16 * c, r[c]);
  umma::tmem_wait_ld();
#pragma unroll
  for (int c = 0; c < N / 8; ++c) {
    uint32_t o[16];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      o[2 * i] = (uint32_t)v[8 * c + i];
      o[2 * i + 1] = (uint32_t)(v[8 * c + i] >> 32);
      v[8 * c + i] = load ? ((uint64_t)r[c][2 * i + 1] << 32) | r[c][2 * i] : 0;
    }
    umma::tmem_st16(ta + 16 * c, o);
  }
}

// Y loader's view of a job: its Y pairs, sizes, and each column block's G size
// and first 16-column block of Y.
struct ZcYJob {
  const float2 *Y2;
  int64_t czrow0;
  int pA, nb, mtz, q, ng0, ng1, cb0, cb1;
};

__device__ __forceinline__ void zc_y_job(const SplitShared &S, const SplitWave &W, int jbeg,
                                         int r, ZcYJob &Y) {
  const ZcJob jb = zc_job(W, jbeg, r);
  const WorkItem it = S.items[jb.w];
  Y.Y2 = reinterpret_cast<const float2 *>(W.scratch + W.y2_off[(int)(jb.w - W.w0)]);
  Y.pA = S.nabf[it.a];
  Y.nb = S.nao[it.b];
  Y.mtz = zc_tiles(Y.pA, S.nao[it.a]);
  Y.q = zc_rows_of(S.nao[it.a]).q;
  Y.czrow0 = S.czw_rowpre[it.a];
  Y.ng0 = Y.ng1 = Y.cb0 = Y.cb1 = 0;
  if (jb.nblk > 0) {
    Y.ng0 = S.nao[S.nbr[it.gbase + jb.g[0]].other];
    Y.cb0 = S.kofs[it.gbase + jb.g[0]] / 16;
  }
  if (jb.nblk > 1) {
    Y.ng1 = S.nao[S.nbr[it.gbase + jb.g[1]].other];
    Y.cb1 = S.kofs[it.gbase + jb.g[1]] / 16;
  }
}

// NST operand stages; YST: Y is staged (else the epilogue reads it from global
// memory).
template <int KS, int NST, bool YST>
__global__ void __launch_bounds__(ZC_THREADS, 1) k_zcw(SplitShared S, SplitWave W, ZcCfg cfg) {
  constexpr int NTM = 4;               // groups of 8 outputs
  constexpr int NV = NTM * 2 * 2;      // f32x2 accumulators of a thread
  constexpr int YPAD = ZC_YPAD;
  constexpr int A_BYTES = KS * 128 * 16 * 2;
  constexpr int B_BYTES = KS * ZC_COLS * 16 * 2;
  constexpr int STG = A_BYTES + B_BYTES;
  constexpr int SH = 7 * (KS + 1);
  extern __shared__ __align__(1024) uint8_t smem[];
  uint8_t *ybuf = smem + NST * STG;                                  // [ybytes]
  float2 *red = reinterpret_cast<float2 *>(ybuf + cfg.ybytes);       // [ZC_NQ][ZC_PASS][128]
  ZcwSmem *ctl = reinterpret_cast<ZcwSmem *>(red + ZC_NQ * ZC_PASS * 128);
  volatile int *abort_f = &ctl->abort_f;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int njobs = cfg.jend - cfg.jbeg;
  // this CTA's jobs and pairs
  const int ncj = zc_cta_jobs(njobs, blockIdx.x, gridDim.x);
  const int npair = (ncj + 1) / 2;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; ++s) {
      umma::mbar_init(&ctl->full[s], 1);
      umma::mbar_init(&ctl->empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      umma::mbar_init(&ctl->tfull[b], 1);
      umma::mbar_init(&ctl->tempty[b], ZC_EPI);
    }
    umma::mbar_init(&ctl->yfull, 1);
    umma::mbar_init(&ctl->yempty, ZC_EPI);
    umma::mbar_init(&ctl->drain, 1);
    ctl->abort_f = 0;
    umma::fence_barrier_init();
  }
  if (warp == 0) {
    umma::tmem_alloc(&ctl->tslot, 512);
    umma::tmem_relinquish();
  }
  umma::fence_before_sync();
  __syncthreads();
  umma::fence_after_sync();
  const uint32_t tbase = ctl->tslot;
  if (threadIdx.x == 0) {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    ctl->t_start = t;  // in shared memory: no register held across the roles
  }

  if (warp == ZC_EPI) {
    // ------------------------------------------------------------ A / B loader
    zc_loader<KS, NST, true, true>(S, W, cfg.jbeg, ncj, npair, smem, ctl->full, ctl->empty, abort_f,
                                   lane);
  } else if (warp == ZC_EPI + 2) {
    // ------------------------------------------------------------ Y loader
    // each tile's Y rows and row exponents (with Y in global memory only these)
    long long hand = 0;
    bool ok = true;
    for (int p = 0; p < npair && ok; ++p) {
      if (__shfl_sync(0xffffffffu, lane == 0 ? *abort_f : 0, 0)) break;
      ZcPair<true> pr;
      pr.begin(p, ncj);
      ZcYJob Y, Yo;
      zc_y_job(S, W, cfg.jbeg, pr.r0, Y);
      pr.m0 = Y.mtz;
      if (pr.two) {
        zc_y_job(S, W, cfg.jbeg, pr.r1, Yo);
        pr.m1 = Yo.mtz;
      }
      int cur = 0, x, mt;
      while (pr.next(x, mt)) {
        if (x != cur) {
          zc_swap(Y, Yo);
          cur = x;
        }
        bool w = true;
        if (lane == 0) {  // the buffer is free
          if (hand >= 1)
            w = umma::mbar_wait(&ctl->yempty, (uint32_t)((hand - 1) & 1), S.err, ZC_WAIT);
          w = w && !*abort_f;
        }
        if (!__shfl_sync(0xffffffffu, (int)w, 0)) {
          if (lane == 0) *abort_f = 1;
          ok = false;
          break;
        }
        ++hand;
        if constexpr (YST) {
          const int al0 = mt * Y.q, nal = min(Y.q, Y.pA - al0);
          const int ystr = Y.nb * 16 + YPAD;             // staged pairs per al
          const uint32_t run = (uint32_t)(Y.nb * 16 * 8);  // one al's [b][16] pairs
          const int n0 = (Y.ng0 + 15) / 16 * nal, ncopy = n0 + (Y.ng1 + 15) / 16 * nal;
          if (lane == 0) {
            umma::mbar_arrive_expect_tx(&ctl->yfull, (uint32_t)ncopy * run + 256);
            umma::bulk_g2s(ctl->erow, S.cz_e + Y.czrow0 + mt * 128, 256, &ctl->yfull);
          }
          __syncwarp();
          for (int q = lane; q < ncopy; q += 32) {
            const int b = q < n0 ? 0 : 1;
            const int r = q - (b ? n0 : 0), k = r / nal, al = al0 + r - k * nal;
            umma::bulk_g2s(ybuf + (int64_t)q * ystr * 8,
                           zc_y_global(Y.Y2, (b ? Y.cb1 : Y.cb0) + k, Y.pA, Y.nb, al), run,
                           &ctl->yfull);
          }
        } else {
          for (int r = lane; r < 128; r += 32) ctl->erow[r] = S.cz_e[Y.czrow0 + mt * 128 + r];
          __syncwarp();
          if (lane == 0) umma::mbar_arrive(&ctl->yfull);
        }
      }
    }
    // copies of a tile that nobody waits for any more after a failure elsewhere
    if (YST && lane == 0 && hand > 0)
      umma::mbar_wait(&ctl->yfull, (uint32_t)((hand - 1) & 1), S.err, ZC_WAIT);
  } else if (warp == ZC_EPI + 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0)
      zc_issuer<KS, NST, true, true>(S, W, cfg.jbeg, ncj, npair, smem, tbase, ctl->full, ctl->empty,
                                     ctl->tfull, ctl->tempty, &ctl->drain, abort_f);
  } else {
    // ------------------------------------------------------------ epilogue
    // TMEM lane quarter, column group, fragment of 16 rows
    const int q4 = warp & 3, hf = (warp >> 2) & 1, r0 = q4 * 32 + 16 * (warp >> 3);
    const int et = threadIdx.x;  // 0 .. ZC_ET - 1
    // this lane's rows r0 + 8 h + lr and columns kc + {0, 1, 8, 9}
    const int lr = lane >> 2, kc = 2 * (lane & 3);
    const uint32_t tfrag = tbase + ((uint32_t)r0 << 16);
    const uint32_t tpark = tbase + ((uint32_t)(q4 * 32) << 16) +
                           (uint32_t)((hf ? 448 : 192) + 32 * (warp >> 3));
    long long hand = 0;
    bool aborted = false;
    for (int p = 0; p < npair && !aborted; ++p) {
      const int pp = p & 1;
      ZcPair<true> pr;
      pr.begin(p, ncj);
      // the pair's epilogue data: warps 0 and 1 the jobs' scalars and Sigma
      // offsets, warps 2 + x + 4 hf the column exponents of job x's column
      // group hf.  The previous pair's reads of the column exponents are
      // behind its jobs' last barriers, and its data sit in the other parity.
      if (warp < 2) {
        if (warp == 0 || pr.two)
          zc_epi_job<true>(S, W, cfg.jbeg, warp ? pr.r1 : pr.r0, lane, ctl->ej[pp][warp]);
      } else if (warp < 8 && q4 >= 2 && (q4 == 2 || pr.two)) {
        const int e = zc_col_exp<ZC_CW>(S, W, cfg.jbeg, q4 == 3 ? pr.r1 : pr.r0, hf, lane);
        const int m = __reduce_max_sync(0xffffffffu, e);
        if (lane < ZC_CW) ctl->cw[q4 - 2][hf * ZC_CW + lane] = zc_exp2(e - m);
        if (lane == 0) ctl->emax[q4 - 2][hf] = m;
      }
      asm volatile("bar.sync 1, %0;" ::"r"(ZC_ET) : "memory");
      pr.m0 = ctl->ej[pp][0].mtz;
      if (pr.two) pr.m1 = ctl->ej[pp][1].mtz;
      // sums of the current tile's job over its tiles, one per (row, output) of
      // this warp, as f32 pairs: [output group][row half], high words then low
      // words; the pair's other job keeps its own in spare TMEM columns
      uint64_t acc[NV];
#pragma unroll
      for (int k = 0; k < NV; ++k) acc[k] = 0;
      bool parked = false, bad = false;
      int cur = 0, x, mt;
      while (pr.next(x, mt)) {
        if (x != cur) {
          zc_exchange<NV>(tpark, acc, parked);
          parked = true;
          cur = x;
        }
        const ZcEpiJob &ej = ctl->ej[pp][x];
        const int tb = (int)(hand & 1);
        const uint32_t ypar = (uint32_t)(hand & 1);
        // this warp's column group: block hb, its first column c0
        int c0 = 0;
        const int hb = zc_group_block<ZC_CW>(ej.nblk, ej.R0b, hf, c0);
        // a wait that fails ends the build: this warp then only walks to the
        // job's end, where all epilogue warps take the same decision
        auto wait = [&](uint64_t *bar, uint32_t parity) {
          if (!bad && (*abort_f || !umma::mbar_wait(bar, parity, S.err, ZC_WAIT))) {
            *abort_f = 1;
            bad = true;
          }
          bad = __any_sync(0xffffffffu, bad);
        };
        wait(&ctl->tfull[tb], (uint32_t)((hand >> 1) & 1));
        ++hand;
        // Z of the fragment: order groups (exact f32 integers) summed in
        // double-float, four column pairs [column half][row half]
        uint64_t zh[4], zl[4];
        if (!bad) {
          umma::fence_after_sync();
#pragma unroll
          for (int j = 0; j < 4; ++j) zh[j] = zl[j] = 0;
          if (hb >= 0) {
            // block hb's order g occupies TMEM columns hb 16 KS + g R .. + R
            const int Rh = hb > 0 ? 16 : ej.R0b;
            const uint32_t ta = tfrag + (uint32_t)(tb * 256 + hb * 16 * KS + c0);
#pragma unroll
            for (int g0 = 0; g0 < KS; g0 += 3) {
              uint32_t r[3][8];
#pragma unroll
              for (int v = 0; v < 3; ++v)
                if (g0 + v < KS) umma::tmem_ld_frag_nowait(ta + (uint32_t)((g0 + v) * Rh), r[v]);
              umma::tmem_wait_ld();
#pragma unroll
              for (int v = 0; v < 3; ++v) {
                if (g0 + v >= KS) break;
                const float cg = __int_as_float((7 * (KS - 1 - g0 - v) + 127) << 23);
                const uint64_t c2 = f2_pk(cg, cg);
#pragma unroll
                for (int j = 0; j < 4; ++j)
                  df_acc2(zh[j], zl[j],
                          f2_mul(f2_pk(__uint_as_float(r[v][2 * j]),
                                       __uint_as_float(r[v][2 * j + 1])), c2));
              }
            }
          }
          umma::fence_before_sync();
          __syncwarp();
          if (lane == 0) umma::mbar_arrive(&ctl->tempty[tb]);
        }
        wait(&ctl->yfull, ypar);
        const int nal = min(ej.q, ej.pA - mt * ej.q);
        // the al [alf, ale) whose rows this fragment holds, and those of this
        // lane's two rows (-1: none)
        const int rr = r0 & (ej.u - 1), alb = (r0 >> ej.ush) * ej.slots;
        const int alf = alb + ((rr * ej.inv) >> 16);
        const int ale = min(nal, alb + min(ej.slots, (((rr + 15) * ej.inv) >> 16) + 1));
        if (!bad && hb >= 0 && alf < ale) {
          const int hq = hb > 0 ? 1 : 0, nb = ej.nb;
          const int no = ej.nout[hq], cend = min(ZC_CW, ej.ncv[hq] - c0);
          const bool p1 = ej.pc[hq] == 1;
          // Y of al in 16-column block k of this warp's block ([b][16] pairs)
          auto yrow = [&](int k, int al) -> const float2 * {
            if constexpr (YST)
              return reinterpret_cast<const float2 *>(ybuf) +
                     (((hq ? ej.ncb0 : 0) + k) * nal + al) * (nb * 16 + YPAD);
            else
              return zc_y_global(reinterpret_cast<const float2 *>(W.scratch + ej.y2off),
                                 ej.gcb[hq] + k, ej.pA, nb, mt * ej.q + al);
          };
          // Z = raw 2^(row exponent - SH + column exponent), raw as f32 pairs; raw is
          // zero past the block's columns and in rows that hold no al, as the
          // operands are.  Its digits, with an exponent per row (over this warp's
          // columns), and each row's al (-1: none) and exponent in all
          const float *cw = ctl->cw[x] + hf * ZC_CW;
          int alr[2], er[2];
          uint32_t zm[2] = {0, 0};
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const uint64_t r = zl[j];
            zl[j] = 0;
            df_acc2(zh[j], zl[j], r);
            zm[j & 1] = max(zm[j & 1], zc_max_abs(zh[j]));
          }
          float zs[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int sl = ((rr + 8 * h + lr) * ej.inv) >> 16;
            alr[h] = sl < ej.slots && alb + sl < nal ? alb + sl : -1;
            zm[h] = max(zm[h], __shfl_xor_sync(0xffffffffu, zm[h], 1));
            zm[h] = max(zm[h], __shfl_xor_sync(0xffffffffu, zm[h], 2));
            er[h] = zc_exp_of(zm[h], zs[h]) + ctl->erow[r0 + 8 * h + lr] - SH +
                    ctl->emax[x][hf];
          }
          if (__any_sync(0xffffffffu, (zm[0] | zm[1]) != 0)) {  // else nothing but zeros
            uint32_t A[4][ZC_DIG];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const uint64_t s2 = f2_pk(zs[j & 1], zs[j & 1]), l = f2_mul(zl[j], s2);
              uint64_t h = f2_mul(zh[j], s2);
#pragma unroll
              for (int i = 0; i < ZC_DIG; ++i) A[j][i] = zc_digit(i, h, l);
            }
#pragma unroll
            for (int nt = 0; nt < NTM; ++nt) {
              if (nt * 8 >= no) break;
              float cg[ZC_DIG][4];
#pragma unroll
              for (int g = 0; g < ZC_DIG; ++g)
#pragma unroll
                for (int k = 0; k < 4; ++k) cg[g][k] = 0.f;
              const int o = nt * 8 + lr;
              // exponents of Y for this lane's sums: rows h, outputs 2 (lane % 4) + {0, 1}
              int ey[2][2] = {{0, 0}, {0, 0}};
              for (int al = alf; al < ale; ++al) {
                uint64_t bh[2], bl[2];
                if (p1)  // out b = o: Y[al][b][G, g = c0 + k]
                  zc_y_frag<true>(yrow(c0 >> 4, al) + o * 16, kc, cend, o < no, cw, bh, bl);
                else  // out g = o: Y[al][b = c0 + k][G, g]
                  zc_y_frag<false>(yrow(nt >> 1, al) + c0 * 16 + (o & 15), kc, cend, o < no, cw,
                                   bh, bl);
                uint32_t m = max(zc_max_abs(bh[0]), zc_max_abs(bh[1]));
                m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
                m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
                float ys;
                const int e = zc_exp_of(m, ys);
                const int e0 = __shfl_sync(0xffffffffu, e, 8 * (lane & 3));
                const int e1 = __shfl_sync(0xffffffffu, e, 8 * (lane & 3) + 4);
                const uint64_t s2 = f2_pk(ys, ys);
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                  bh[u] = f2_mul(bh[u], s2);
                  bl[u] = f2_mul(bl[u], s2);
                }
                uint32_t kp[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                  kp[h] = alr[h] == al ? ~0u : 0u;
                  if (alr[h] == al) {
                    ey[h][0] = e0;
                    ey[h][1] = e1;
                  }
                }
#pragma unroll
                for (int jd = 0; jd < ZC_DIG; ++jd) {
                  const uint32_t b0 = zc_digit(jd, bh[0], bl[0]), b1 = zc_digit(jd, bh[1], bl[1]);
#pragma unroll
                  for (int i = 0; i < ZC_DIG - jd; ++i)
                    zc_mma(cg[i + jd], A[0][i] & kp[0], A[1][i] & kp[1], A[2][i] & kp[0],
                           A[3][i] & kp[1], b0, b1);
                }
              }
              // order groups into the sums: the first three exactly (TwoSum), the
              // others are below the low words' resolution
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                const int k = nt * 2 + h;
                const uint64_t sc = f2_pk(zc_exp2(er[h] + ey[h][0]), zc_exp2(er[h] + ey[h][1]));
                uint64_t t[ZC_DIG];
#pragma unroll
                for (int g = 0; g < ZC_DIG; ++g) t[g] = f2_pk(cg[g][2 * h], cg[g][2 * h + 1]);
                uint64_t lo =
                    f2_fma(f2_add(t[3], f2_add(t[4], t[5])), sc, acc[NV / 2 + k]);
#pragma unroll
                for (int g = 2; g >= 0; --g) df_acc2(acc[k], lo, f2_mul(t[g], sc));
                acc[NV / 2 + k] = lo;
              }
            }
          }
        }
        __syncwarp();
        if (!bad && lane == 0) umma::mbar_arrive(&ctl->yempty);
        if (mt + 1 < ej.mtz) continue;
        // the job's last tile: sum its rows (slots and column groups) in a fixed
        // order and add the finished blocks to Sigma (and mirrors); a sum
        // outside the fixed-point range is not added and fails the build
        if (umma::bar_any(bad || *abort_f, ZC_ET)) {
          *abort_f = 1;
          aborted = true;
          break;
        }
        const int nout0 = ej.nout[0], nout1 = ej.nout[1];
        const int na = ej.na, npass = (max(nout0, nout1) + ZC_PASS - 1) / ZC_PASS;
        const int own0 = na * nout0, nown = own0 + na * nout1;
        unsigned qm[2] = {0, 0};  // column groups feeding block 0 and block 1 (bit q)
#pragma unroll
        for (int q = 0; q < ZC_NQ; ++q) {
          int cq;
          const int bq = zc_group_block<ZC_CW>(ej.nblk, ej.R0b, q, cq);
          qm[0] |= (bq == 0 ? 1u : 0u) << q;
          qm[1] |= (bq == 1 ? 1u : 0u) << q;
        }
        bool inrange = true;
#pragma unroll
        for (int pass = 0; pass < NTM; ++pass) {
          if (pass >= npass) break;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int k = pass * 2 + h;
            const float2 vh = f2_un(acc[k]), vl = f2_un(acc[NV / 2 + k]);
            float2 *o = red + (hf * ZC_PASS + kc) * 128 + r0 + 8 * h + lr;
            o[0] = make_float2(vh.x, vl.x);
            o[128] = make_float2(vh.y, vl.y);
          }
          asm volatile("bar.sync 1, %0;" ::"r"(ZC_ET) : "memory");
          for (int idx = et; idx < nown; idx += ZC_ET) {
            const int b1 = idx >= own0 ? 1 : 0;
            const int nob = ej.nout[b1], rem = idx - (b1 ? own0 : 0);
            const int o = (rem * ej.inv) >> 16, a = rem - o * na;  // consecutive: consecutive a
            if (o / ZC_PASS != pass) continue;
            float h = 0.f, l = 0.f;
#pragma unroll
            for (int q = 0; q < ZC_NQ; ++q) {
              if (!((qm[b1] >> q) & 1u)) continue;
              const float2 *rq = red + ((int64_t)q * ZC_PASS + (o & (ZC_PASS - 1))) * 128 + a;
              for (int r = 0; r < 128; r += ej.u)
                for (int sl = 0; sl < ej.slots; ++sl) df_add(h, l, rq[r + sl * na]);
            }
            if (!fx_df_in_range(h)) {
              inrange = false;
              continue;
            }
            const int64_t t0 = ej.sg[b1][0], t1 = ej.sg[b1][1];
            if (t0 < 0) continue;  // missing key: recorded when the pair started
            const float2 v = make_float2(h, l);
            fx_add_df(S.acc + 2 * (t0 + (int64_t)a * nob + o), v, true);
            if (t1 >= 0) fx_add_df(S.acc + 2 * (t1 + (int64_t)o * na + a), v, true);
          }
          asm volatile("bar.sync 1, %0;" ::"r"(ZC_ET) : "memory");
        }
        if (!inrange) atomicOr(S.err, HFX_DEV_ERR_BOUNDS);
#pragma unroll
        for (int k = 0; k < NV; ++k) acc[k] = 0;
      }
    }
  }
  umma::fence_before_sync();
  __syncthreads();
  if (warp == 0) umma::tmem_dealloc(tbase, 512);
  if (threadIdx.x == 0) {
    unsigned long long t_end;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t_end));
    W.cta_ns[cfg.cta0 + blockIdx.x] = (long long)(t_end - ctl->t_start);
  }
}

// Variants by what fits 227 KB next to the reduction buffer (16 KB) and the
// operand stages (30 KB each with 6 digits).  One Y buffer: a second one was slower
// even where it fits beside four stages (6 digits, 27/90 alone: 10.1 against
// 9.4 ms; 20/70 alone: 15.7 against 14.0).  Four stages and five take about the
// same time (two-element cell, 13/60 and 27/90: 97.8 and 100.3 ms with 6 digits,
// 82.1 and 83.5 with 4), so does the fallback of three (99.0, 84.6).  Y is read
// from global memory (115.7 ms there) only beside atoms of very few AOs, whose row
// tiles hold many al.
template <int KS>
cudaError_t zcw_run_t(const SplitShared &S, const SplitWave &W, int ybytes, int nsm, int jbeg,
                      int jend, int cta0, cudaStream_t st) {
  const int blocks = (int)std::min<int64_t>(jend - jbeg, nsm);
  if (blocks <= 0) return cudaSuccess;
  auto launch = [&](auto kern, int nst, int yb, bool probe) -> cudaError_t {
    const size_t smem = (size_t)nst * KS * (128 + ZC_COLS) * 16 * 2 + (size_t)yb +
                        (size_t)ZC_NQ * ZC_PASS * 128 * sizeof(float2) + sizeof(ZcwSmem) + 64;
    if (probe && smem > 227 * 1024) return cudaErrorMemoryAllocation;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<blocks, ZC_THREADS, smem, st>>>(S, W, ZcCfg{yb, jbeg, jend, cta0});
    return cudaGetLastError();
  };
  cudaError_t e = launch(k_zcw<KS, 4, true>, 4, ybytes, true);
  if (e == cudaErrorMemoryAllocation) e = launch(k_zcw<KS, 3, true>, 3, ybytes, true);
  if (e == cudaErrorMemoryAllocation) e = launch(k_zcw<KS, 5, false>, 5, 0, false);
  return e;
}

// Shared bytes of one staged Y buffer (both blocks of a tile) over the AO
// counts that occur (bit n of present: some atom has n AOs): the al of a row
// tile of atom A, all b, the 16-column blocks of the Gs (two blocks share a job
// when both have at most 16 Z columns), plus the pads.
int zcw_ybytes(uint64_t present) {
  int cbs = 1, cmin = 2, bytes = 0;
  for (int n = 1; n <= 32; ++n)
    if ((present >> n) & 1) {
      cbs = n <= 16 ? 1 : 2;
      cmin = std::min(cmin, cbs);
    }
  for (int na = 1; na <= 32; ++na)
    for (int nb = 1; nb <= 32; ++nb) {
      if (!((present >> na) & 1) || !((present >> nb) & 1)) continue;
      const int ncb = nb <= 16 ? 2 * cbs : std::max(cbs, cmin == 1 ? 2 : 1);
      bytes = std::max(bytes, zc_rows_of(na).q * (nb * 16 + ZC_YPAD) * 8 * ncb);
    }
  return bytes;
}

}  // namespace split

cudaError_t split_zcw_run(const SplitShared &S, const SplitWave &W, int ks, int ybytes, int nsm,
                          int jbeg, int jend, int cta0, cudaStream_t st) {
  switch (ks) {
    case 2: return split::zcw_run_t<2>(S, W, ybytes, nsm, jbeg, jend, cta0, st);
    case 4: return split::zcw_run_t<4>(S, W, ybytes, nsm, jbeg, jend, cta0, st);
    case 5: return split::zcw_run_t<5>(S, W, ybytes, nsm, jbeg, jend, cta0, st);
    case 6: return split::zcw_run_t<6>(S, W, ybytes, nsm, jbeg, jend, cta0, st);
    default: return cudaErrorInvalidValue;
  }
}

int split_zcw_ybytes(uint64_t present) { return split::zcw_ybytes(present); }
