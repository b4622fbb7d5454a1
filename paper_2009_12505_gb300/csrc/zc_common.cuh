// Device code shared by the two kernels of the D_FG / D_FB products: k_zc for
// blocks of at most 16 AOs (hfx_zc.cu) and k_zcw for wider ones (hfx_zcw.cu).
#pragma once

#include <cuda_bf16.h>

#include <algorithm>

#include "hfx_split.h"
#include "split_common.cuh"
#include "stage_ring.h"

namespace split {

constexpr int ZC_COLS = 32;                      // Z columns per job
constexpr long long ZC_WAIT = 2000000000ll;      // cycles per bounded wait

// Job handed to CTA b in round r of the persistent loop: rounds alternate
// direction (snake order), so over a longest-first list every CTA gets a
// similar mix of long and short jobs.  The last round is partial.
__device__ __forceinline__ int zc_job_of(int r, int b, int G) {
  return r * G + ((r & 1) ? G - 1 - b : b);
}

// Epilogue data of one job, written to shared memory by a few lanes when its
// pair starts and read by every epilogue thread on each of the job's tiles.
struct ZcEpiJob {
  int64_t y2off;     // the work item's Y pairs in the wave scratch
  int64_t sg[2][2];  // block q: Sigma offset of its outputs, of their mirror (-1: none)
  int pA, na, nb, mtz, nblk, R0b;
  int nout[2], ncv[2], pc[2], gcb[2];
  int64_t czrow0;        // first row of atom A's C exponents
  int u, ush, slots, q;  // the A operand's rows (ZcRows, wide operand), u = 2^ush
  int inv;          // x / na = x inv >> 16 for x < 2048
  int ncb0;  // 16-column blocks of Y of block 0 (block 1's follow them in a staged buffer)
};

// Number of jobs CTA b receives from zc_job_of over a list of njobs.
__device__ __forceinline__ int zc_cta_jobs(int njobs, int b, int G) {
  const int full = njobs / G, rem = njobs - full * G;
  return full + (((full & 1) ? G - 1 - b : b) < rem ? 1 : 0);
}

// Tile order of a CTA.  Its jobs r = 0 .. n - 1 run heaviest first (operand
// stages x row tiles); pair p is job n - 1 - p (light) and job p (heavy), and
// their row tiles alternate while both have some: the MMAs of a long tile then
// run beside the epilogue of a short one, where one job after the other leaves
// the epilogue idle through the long tiles and the tensor pipe idle through
// the short ones.  Without PAIR, pair p is job p alone.  Every role walks the
// same order.
template <bool PAIR>
struct ZcPair {
  int r0, r1, m0, m1, t0, t1, last;
  bool two;
  __device__ __forceinline__ void begin(int p, int n) {
    r0 = PAIR ? n - 1 - p : p;
    r1 = PAIR ? p : -1;
    two = PAIR && r1 < r0;
    m0 = m1 = t0 = t1 = 0;
    last = 1;
  }
  // next tile: job x of the pair (0: r0, 1: r1) and its row tile mt
  __device__ __forceinline__ bool next(int &x, int &mt) {
    const bool a = t0 < m0, b = t1 < m1;
    if (!a && !b) return false;
    x = (a && (!b || last == 1)) ? 0 : 1;
    last = x;
    mt = x ? t1++ : t0++;
    return true;
  }
};

template <class T>
__device__ __forceinline__ void zc_swap(T &a, T &b) {
  const T t = a;
  a = b;
  b = t;
}

__device__ __forceinline__ ZcJob zc_job(const SplitWave &W, int jbeg, int r) {
  return W.zc_jobs[jbeg + zc_job_of(r, blockIdx.x, gridDim.x)];
}

// rows of a job's lone column block (16, in wide jobs also 32); two blocks have
// 16 each
template <bool WIDE>
__device__ __forceinline__ int zc_rows(const SplitShared &S, const ZcJob &jb, const WorkItem &it) {
  if (!WIDE || jb.nblk != 1) return 16;
  const int ncb = jb.piece[0] == 1 ? S.nao[S.nbr[it.gbase + jb.g[0]].other] : S.nao[it.b];
  return ncb <= 16 ? 16 : 32;
}

// row tiles of atom a's A operand
template <bool WIDE>
__device__ __forceinline__ int zc_row_tiles(const SplitShared &S, int a) {
  return WIDE ? zc_tiles(S.nabf[a], S.nao[a]) : (S.nabf[a] * S.nao[a] + 127) / 128;
}

// block and first column cq of column group q of width CW: two 16-column
// blocks take half the groups each; one block takes the groups below its R
template <int CW>
__device__ __forceinline__ int zc_group_block(int nblk, int R0b, int q, int &cq) {
  const int jc = q * CW;
  if (nblk == 2) { cq = jc & 15; return jc >> 4; }
  cq = jc;
  return jc < R0b ? 0 : -1;
}

// Epilogue data of job r, by one whole warp: lanes 0 .. 3 look up the Sigma
// offsets of block lane / 2 (odd lanes: the mirror), lane 4 the scalars.  A
// missing Sigma key fails the build, and the block is not added.
template <bool WIDE>
__device__ __forceinline__ void zc_epi_job(const SplitShared &S, const SplitWave &W, int jbeg,
                                           int r, int lane, ZcEpiJob &e) {
  const ZcJob jb = zc_job(W, jbeg, r);
  const WorkItem it = S.items[jb.w];
  const int q = (lane >> 1) & 1, m = lane & 1;
  int64_t t = -1;
  bool miss = false;
  if (lane < 4 && q < jb.nblk) {
    const int pcb = q ? jb.piece[1] : jb.piece[0];
    const bool mir = S.sym && (pcb == 2 || it.role == 1);
    if (m == 0 || mir) {
      if (pcb == 1) {
        t = m == 0 ? dh_find(S.shash, hk_pack(it.a, it.b, it.n[0], it.n[1], it.n[2]))
                   : dh_find(S.shash, hk_pack(it.b, it.a, -it.n[0], -it.n[1], -it.n[2]));
      } else {
        const NbrEntry eg = S.nbr[it.gbase + (q ? jb.g[1] : jb.g[0])];
        const int n0 = it.n[0] + eg.n[0], n1 = it.n[1] + eg.n[1], n2 = it.n[2] + eg.n[2];
        t = m == 0 ? dh_find(S.shash, hk_pack(it.a, eg.other, n0, n1, n2))
                   : dh_find(S.shash, hk_pack(eg.other, it.a, -n0, -n1, -n2));
      }
      miss = t < 0;
      if (miss) atomicOr(S.err, HFX_DEV_ERR_MISSING);
    }
  }
  const bool bad = __shfl_sync(0xffffffffu, (int)miss, lane & ~1) |
                   __shfl_sync(0xffffffffu, (int)miss, lane | 1);
  if (lane < 4) e.sg[q][m] = bad ? -1 : t;
  if (lane == 4) {
    const int pA = S.nabf[it.a], na = S.nao[it.a], nb = S.nao[it.b];
    e.y2off = W.y2_off[(int)(jb.w - W.w0)];
    e.pA = pA;
    e.na = na;
    e.nb = nb;
    const ZcRows R = zc_rows_of(na);
    e.u = R.u;
    e.ush = __ffs(R.u) - 1;
    e.slots = R.slots;
    e.q = R.q;
    e.inv = (65536 + na - 1) / na;
    e.mtz = zc_row_tiles<WIDE>(S, it.a);
    e.czrow0 = (WIDE ? S.czw_rowpre : S.cz_rowpre)[it.a];
    e.nblk = jb.nblk;
    e.R0b = 16;
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      e.nout[b] = e.ncv[b] = e.pc[b] = e.gcb[b] = 0;
      if (b < jb.nblk) {
        const int ng = S.nao[S.nbr[it.gbase + jb.g[b]].other];
        e.pc[b] = jb.piece[b];
        e.gcb[b] = S.kofs[it.gbase + jb.g[b]] / 16;
        e.ncv[b] = jb.piece[b] == 1 ? ng : nb;
        e.nout[b] = jb.piece[b] == 1 ? nb : ng;
      }
    }
    if (jb.nblk > 0) e.R0b = e.ncv[0] <= 16 ? 16 : 32;
    e.ncb0 = jb.nblk > 0 ? (S.nao[S.nbr[it.gbase + jb.g[0]].other] + 15) / 16 : 0;
  }
}

// Exponent of column `lane` of job r's column group hf (CW columns; -1000: none).
template <int CW>
__device__ __forceinline__ int zc_col_exp(const SplitShared &S, const SplitWave &W, int jbeg,
                                          int r, int hf, int lane) {
  const ZcJob jb = zc_job(W, jbeg, r);
  const WorkItem it = S.items[jb.w];
  int ncv0 = 0, R0b = 16;
  if (jb.nblk > 0) {
    ncv0 = jb.piece[0] == 1 ? S.nao[S.nbr[it.gbase + jb.g[0]].other] : S.nao[it.b];
    R0b = ncv0 <= 16 ? 16 : 32;
  }
  int c0 = 0;
  const int hb = zc_group_block<CW>(jb.nblk, R0b, hf, c0);
  if (hb < 0 || lane >= CW) return -1000;
  const int pc = hb ? jb.piece[1] : jb.piece[0], g = hb ? jb.g[1] : jb.g[0];
  const int at = pc == 1 ? S.nbr[it.gbase + g].other : it.b;
  // piece 1: nao(G) columns; piece 2: nao(B)
  return c0 + lane < S.nao[at] ? row_exponent((long long)S.de[S.aoff[at] + c0 + lane]) : -1000;
}

// A launch's shared bytes of one staged Y buffer and its range of the job list.
struct ZcCfg {
  int ybytes;
  int jbeg, jend;
  int cta0;  // first slot of its CTAs' busy times
};

// Y rows al in [al0, al0 + nal) of the 16-column block cb: [al][b][16] pairs.
__device__ __forceinline__ const float2 *zc_y_global(const float2 *Y2, int cb, int pA, int nb,
                                                     int al) {
  return Y2 + (((int64_t)cb * pA + al) * nb) * 16;
}

// One operand stage's MMAs (K = 16): for each block b, A digit i times the
// block's B digits 0 .. KS - 1 - i stacked along N (N = R (KS - i)) into TMEM
// columns b 16 KS + i R ..  Descriptors are the stage's two base descriptors
// plus constant offsets (the 14-bit start field cannot carry: shared
// addresses stay below 2^18).
template <int KS>
__device__ __forceinline__ void zc_stage_mmas(uint32_t a0, uint32_t b0, uint32_t dcol, int nblk,
                                              int R, const uint32_t (&id16)[KS],
                                              const uint32_t (&id32)[KS], bool first) {
  const uint64_t adesc = umma::smem_desc(a0, 128, 256);
  const uint64_t bdesc = umma::smem_desc(b0, 128, 256);
  for (int b = 0; b < nblk; ++b) {
    const uint64_t bd = bdesc + (uint64_t)((b * (KS * 16 * 16 * 2)) >> 4);
#pragma unroll
    for (int i = 0; i < KS; ++i) {
      const uint64_t ad = adesc + (uint64_t)((i * (128 * 16 * 2)) >> 4);
      umma::mma_bf16(dcol + (uint32_t)(b * 16 * KS + i * R), ad, bd, R == 16 ? id16[i] : id32[i],
                     (!first || i) ? 1u : 0u);
    }
  }
}

// Loader-warp view of a job: operand bases, its entries (lane l holds entry
// held + l) and the B rows per block.
struct ZcLd {
  const __nv_bfloat16 *A;
  int64_t ktot, ent;
  int nent, nblk, Rl, mtz, held;
  ZcEnt mine;
};

template <bool WIDE>
__device__ __forceinline__ void zc_ld_job(const SplitShared &S, const SplitWave &W, int jbeg,
                                          int r, ZcLd &L) {
  const ZcJob jb = zc_job(W, jbeg, r);
  const WorkItem it = S.items[jb.w];
  L.A = S.cz + (WIDE ? S.czw_base : S.cz_base)[it.a];
  L.ktot = S.ktotZ[it.a];
  L.ent = jb.ent;
  L.nent = jb.nent;
  L.nblk = jb.nblk;
  L.Rl = zc_rows<WIDE>(S, jb, it);
  L.mtz = zc_row_tiles<WIDE>(S, it.a);
  L.held = -1;
  L.mine = ZcEnt{0, {-1, -1}};
}

// The A / B loader of both kernels, by one whole warp: the jobs' operand stages
// into the ring of NST stages at smem.  Lane l holds entry q0 + l of the job
// (fetched 32 at a time, off the per-stage path) and waits for its stage, arms
// it and issues its copies itself; the lanes take turns, as the ring's parities
// need the stages in order, and one vote a stage ends the walk in all of them.
template <int KS, int NST, bool WIDE, bool PAIR>
__device__ __forceinline__ void zc_loader(const SplitShared &S, const SplitWave &W, int jbeg,
                                          int ncj, int npair, uint8_t *smem, uint64_t *full,
                                          uint64_t *empty, volatile int *abort_f, int lane) {
  constexpr int A_BYTES = KS * 128 * 16 * 2;
  constexpr int STG = A_BYTES + KS * ZC_COLS * 16 * 2;
  StageRing<NST> ring;
  bool ok = true;
  for (int p = 0; p < npair && ok; ++p) {
    // one decision for the whole warp
    if (__shfl_sync(0xffffffffu, lane == 0 ? *abort_f : 0, 0)) break;
    ZcPair<PAIR> pr;
    pr.begin(p, ncj);
    ZcLd L, Lo;  // L: the job of the current tile, Lo: the pair's other job
    zc_ld_job<WIDE>(S, W, jbeg, pr.r0, L);
    pr.m0 = L.mtz;
    if (pr.two) {
      zc_ld_job<WIDE>(S, W, jbeg, pr.r1, Lo);
      pr.m1 = Lo.mtz;
    }
    int cur = 0, x, mt;
    while (ok && pr.next(x, mt)) {
      if (x != cur) {
        zc_swap(L, Lo);
        cur = x;
      }
      const uint32_t bb = (uint32_t)(KS * 16 * 2) * (uint32_t)L.Rl;  // bytes of a B block
      for (int q0 = 0; q0 < L.nent && ok; q0 += 32) {
        if (L.held != q0) {
          if (q0 + lane < L.nent) L.mine = W.zc_ents[L.ent + q0 + lane];
          L.held = q0;
        }
        const __nv_bfloat16 *a = L.A + ((int64_t)mt * L.ktot + L.mine.kofs) * KS * 128;
        const __nv_bfloat16 *b0 = L.mine.dz[0] >= 0 ? S.dz + L.mine.dz[0] : S.dzero;
        const __nv_bfloat16 *b1 = L.mine.dz[1] >= 0 ? S.dz + L.mine.dz[1] : S.dzero;
        ok = ring_stages(
            ring, min(32, L.nent - q0),
            [&](int q) {
              if (lane != q) return true;
              if (!ring.fresh() && !umma::mbar_try_wait(&empty[ring.s], ring.ph) &&
                  (*abort_f || !umma::mbar_wait(&empty[ring.s], ring.ph, S.err, ZC_WAIT))) {
                *abort_f = 1;
                return false;
              }
              uint8_t *st = smem + ring.s * STG;
              uint64_t *bar = &full[ring.s];
              umma::mbar_arrive_expect_tx(bar, A_BYTES + bb * (uint32_t)L.nblk);
              umma::bulk_g2s(st, a, A_BYTES, bar);
              // B stage block-major: block b's KS digits of Rl rows x 16 K at b KS 16 16
              umma::bulk_g2s(st + A_BYTES, b0, bb, bar);
              if (L.nblk > 1) umma::bulk_g2s(st + A_BYTES + KS * 16 * 16 * 2, b1, bb, bar);
              return true;
            },
            [](bool c) { return __all_sync(0xffffffffu, c) != 0; });
      }
    }
  }
  // the last stages armed must have landed before the CTA exits
  if (lane == 0)
    for (int t = ring.pending(); t < ring.step; ++t)
      umma::mbar_wait(&full[t % NST], (uint32_t)((t / NST) & 1), S.err, ZC_WAIT);
}

// The MMA issuer of both kernels, by one thread: every stage of the jobs' tiles
// into the TMEM accumulators (two, 256 columns each) in turn.
template <int KS, int NST, bool WIDE, bool PAIR>
__device__ __forceinline__ void zc_issuer(const SplitShared &S, const SplitWave &W, int jbeg,
                                          int ncj, int npair, uint8_t *smem, uint32_t tbase,
                                          uint64_t *full, uint64_t *empty, uint64_t *tfull,
                                          uint64_t *tempty, uint64_t *drain,
                                          volatile int *abort_f) {
  constexpr int A_BYTES = KS * 128 * 16 * 2;
  constexpr int STG = A_BYTES + KS * ZC_COLS * 16 * 2;
  long long hand = 0;
  int s = 0;  // operand slot and its parity
  uint32_t ph = 0;
  // N = R (KS - i) for a block of R rows (16, in wide jobs also 32), at most 192
  uint32_t idesc16[KS], idesc32[KS];
#pragma unroll
  for (int i = 0; i < KS; ++i) {
    idesc16[i] = umma::idesc_bf16_f32(128, 16 * (KS - i));
    idesc32[i] = umma::idesc_bf16_f32(128, 32 * (KS - i));
  }
  const uint32_t sbase = umma::smem_u32(smem);
  bool ok = true;
  for (int p = 0; p < npair && ok && !*abort_f; ++p) {
    ZcPair<PAIR> pr;
    pr.begin(p, ncj);
    // entries, blocks and rows per block of the pair's two jobs
    int ne[2] = {0, 0}, nk[2] = {0, 0}, R[2] = {16, 16}, mtz[2] = {0, 0};
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      if (j == 1 && !pr.two) break;
      const ZcJob jb = zc_job(W, jbeg, j ? pr.r1 : pr.r0);
      const WorkItem it = S.items[jb.w];
      ne[j] = jb.nent;
      nk[j] = jb.nblk;
      R[j] = zc_rows<WIDE>(S, jb, it);
      mtz[j] = zc_row_tiles<WIDE>(S, it.a);
    }
    pr.m0 = mtz[0];
    pr.m1 = mtz[1];
    int x, mt;
    while (ok && !*abort_f && pr.next(x, mt)) {
      const int nent = x ? ne[1] : ne[0], nblk = x ? nk[1] : nk[0], Rx = x ? R[1] : R[0];
      const int tb = (int)(hand & 1);
      const long long use = hand >> 1;
      if (use >= 1 && !umma::mbar_wait(&tempty[tb], (uint32_t)((use - 1) & 1), S.err, ZC_WAIT)) {
        ok = false;
        break;
      }
      umma::fence_after_sync();
      const uint32_t dcol = tbase + (uint32_t)(tb * 256);
      for (int q = 0; q < nent; ++q) {
        if (!umma::mbar_wait(&full[s], ph, S.err, ZC_WAIT)) {
          ok = false;
          break;
        }
        umma::fence_after_sync();
        const uint32_t a0 = sbase + (uint32_t)(s * STG);
        zc_stage_mmas<KS>(a0, a0 + A_BYTES, dcol, nblk, Rx, idesc16, idesc32, q == 0);
        umma::mma_commit(&empty[s]);
        if (++s == NST) {
          s = 0;
          ph ^= 1;
        }
      }
      if (!ok) break;
      umma::mma_commit(&tfull[tb]);
      ++hand;
    }
  }
  if (!ok) *abort_f = 1;
  umma::mma_commit(drain);
  umma::mbar_wait(drain, 0, S.err, ZC_WAIT);
}

}  // namespace split
