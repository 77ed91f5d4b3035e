// qpm_objectives.cu -- the other objectives of the paper's designs.
//
// SHG field (Sec. 2.1, the single integral before the cascade):
//   E2 prop. to int_0^L d(z) e^{-i dk z} dz = phi(kappa) sum_j d_j e^{-i kappa j},
// used by the multi-wavelength SHG designs of Sec. 5.  A plain complex sum per
// row: one CTA per SM takes an equal run of rows, its warps segments of domains.
//
// Multi-wavelength objective (Sec. 5): f = sum_k |G0 - G_k| + beta (G_max - G_min)
// with G_k = |d_eff(kappa1_k, kappa2_k)|, to be minimised.  The K cascaded scans
// share one read of the genes: the row sweep of qpm_eval (qpm_rows.cuh) with the
// K sign-block tables streamed side by side, every block of 4 domains appended to K
// running monoids.  For K = 1 this is qpm_eval's arithmetic, operation for operation.
#include <math.h>

#include <algorithm>
#include <vector>

#include "qpm_common.cuh"
#include "qpm_internal.h"
#include "qpm_rows.cuh"

namespace qpm {

// ------------------------------------------------------------------ SHG field
// Bound by HBM (4 bytes a domain, 2 FMA), so all that counts is bytes in flight and an even
// share per SM.  One CTA per SM takes an equal run of rows.  Its work items are (segment of
// 256 domains, block of 4 rows), dealt to the 16 warps as equal runs in segment-major order,
// so a warp holds the segment's phasors in registers from item to item, issues the 8 16-byte
// loads of an item at once with the next item's already in flight (up to 8 KB a warp, 128 KB an
// SM) and reduces the item's 4 row sums by halving exchanges (9 shuffles for the 8 components).
// Each warp adds its items into its own row sums in shared memory, the CTA the warps' in warp
// order at the end, both compensated.
// 5000 rows of N = 3000 (60 MB, 8.9 us at the copy rate), per call: 30.7 us for the form before
// it, a CTA per 8 rows (625 CTAs on 608 slots, a second wave for 17 of them, and loads under
// conditions that were issued one at a time); 14.3 us now (14.1 with plain sums).
static constexpr int SHG_WARPS = 16;
static constexpr int SHG_Q = 2;                 // 128-domain pieces per segment
static constexpr int SHG_SEG = 128 * SHG_Q;
static constexpr int SHG_RB = 4;                // rows per item; 1 where a CTA has one row
static constexpr int SHG_RMAX = 64;             // rows whose sums are kept at a time

// VEC: rows of 16-byte aligned groups, lane l takes domains 4 l .. 4 l + 3 of a piece with one
// load; else lane l takes domains l, l + 32, l + 64, l + 96, so that every load of a warp is 128
// contiguous bytes whatever the rows' alignment.
// RB: rows per item.  A CTA with one row (up to as many rows as SMs) takes items of one: repeating
// that row four times cost the loads and sums of four, and since each of its items is another
// segment, the phasors come with the genes an item ahead (a row of 1e5 domains: 51 us with items of
// four rows, 32 for the form before them, 30 now; 15 unaligned).  The order of the sums is the same.
template <bool VEC, int RB>
static __global__ void __launch_bounds__(SHG_WARPS * 32, 1)
    k_shg(const float *__restrict__ genes, int64_t ld, int NP, int N, int rows_per_cta,
          const float4 *__restrict__ table, const float2 *__restrict__ konst,
          float2 *__restrict__ eout, float *__restrict__ fout) {
  __shared__ float sums[SHG_WARPS][2 * SHG_RMAX], comp[SHG_WARPS][2 * SHG_RMAX];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // a programmatic dependent of whatever ran before, which may have written genes or the table
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int rend = (int)min((int64_t)NP, (int64_t)(blockIdx.x + 1) * rows_per_cta);
  const int nseg = (N + SHG_SEG - 1) / SHG_SEG;
  const int glast = 4 * (N >> 2) - 4;  // the row's last whole group (VEC: N >= 4)
  for (int64_t rs = (int64_t)blockIdx.x * rows_per_cta; rs < rend; rs += SHG_RMAX) {
    const int r0 = (int)rs, rn = min(SHG_RMAX, rend - r0), nrb = (rn + RB - 1) / RB;
    for (int e = threadIdx.x; e < SHG_WARPS * 2 * SHG_RMAX; e += SHG_WARPS * 32)
      (&sums[0][0])[e] = (&comp[0][0])[e] = 0.f;
    __syncthreads();
    const int64_t items = (int64_t)nseg * nrb;
    const int64_t i0 = items * warp / SHG_WARPS, i1 = items * (warp + 1) / SHG_WARPS;
    int seg = (int)(i0 / nrb), rb = (int)(i0 - (int64_t)seg * nrb);
    int nseg_x = seg, nrb_x = rb;  // the item whose loads are issued next
    // the lane's domain q of piece k of segment sg
    auto dom = [&](int sg, int k, int q) {
      return sg * SHG_SEG + 128 * k + (VEC ? 4 * lane + q : lane + 32 * q);
    };
    float4 x[RB][SHG_Q], y[RB][SHG_Q];  // this item's genes, the next one's in flight
    float2 pn[SHG_Q * 4];               // RB 1: the next item's phasors
    auto fetch = [&]() {
      if (RB == 1) {
#pragma unroll
        for (int k = 0; k < SHG_Q; ++k)
#pragma unroll
          for (int q = 0; q < 4; ++q) pn[4 * k + q] = __ldg((const float2 *)(table + min(dom(nseg_x, k, q), N - 1)));
      }
#pragma unroll
      for (int r = 0; r < RB; ++r) {
        const int row = min(r0 + nrb_x * RB + r, rend - 1);  // a repeated row's sums are dropped
        const float *g = genes + (int64_t)row * ld;
#pragma unroll
        for (int k = 0; k < SHG_Q; ++k) {
          // no load under a condition, so that all of an item's are in flight together: past
          // the row they repeat its last domains, whose phasors below are zero
          if (VEC) {
            y[r][k] = __ldg((const float4 *)(g + min(dom(nseg_x, k, 0), glast)));
          } else {
            y[r][k] = make_float4(
                __ldg(g + min(dom(nseg_x, k, 0), N - 1)), __ldg(g + min(dom(nseg_x, k, 1), N - 1)),
                __ldg(g + min(dom(nseg_x, k, 2), N - 1)), __ldg(g + min(dom(nseg_x, k, 3), N - 1)));
          }
        }
      }
      if (++nrb_x == nrb) {
        nrb_x = 0;
        ++nseg_x;
      }
    };
    if (i0 < i1) fetch();
    float2 p[SHG_Q * 4];  // e^{-i kappa m} of the lane's domains of the segment
    bool fresh = true;
    for (int64_t it = i0; it < i1; ++it) {
#pragma unroll
      for (int r = 0; r < RB; ++r)
#pragma unroll
        for (int k = 0; k < SHG_Q; ++k) x[r][k] = y[r][k];
      if (RB == 1) {
#pragma unroll
        for (int k = 0; k < SHG_Q; ++k)
#pragma unroll
          for (int q = 0; q < 4; ++q) p[4 * k + q] = dom(seg, k, q) < N ? pn[4 * k + q] : make_float2(0.f, 0.f);
      }
      if (it + 1 < i1) fetch();
      if (VEC && (N & 3) != 0 && (seg + 1) * SHG_SEG > N) {  // the row's last, partial group
#pragma unroll
        for (int k = 0; k < SHG_Q; ++k) {
          if (dom(seg, k, 0) == glast + 4) {
#pragma unroll
            for (int r = 0; r < RB; ++r) {
              const float *g = genes + (int64_t)min(r0 + rb * RB + r, rend - 1) * ld;
              x[r][k] = make_float4(__ldg(g + dom(seg, k, 0)), __ldg(g + min(dom(seg, k, 1), N - 1)),
                                    __ldg(g + min(dom(seg, k, 2), N - 1)), 0.f);
            }
          }
        }
      }
      if (RB > 1 && fresh) {
#pragma unroll
        for (int k = 0; k < SHG_Q; ++k)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const float4 e = __ldg(table + min(dom(seg, k, q), N - 1));
            p[4 * k + q] = dom(seg, k, q) < N ? make_float2(e.x, e.y) : make_float2(0.f, 0.f);
          }
        fresh = false;
      }
      float v[2 * RB];  // (re, im) of the rows' partial sums
#pragma unroll
      for (int r = 0; r < RB; ++r) {
        float sx = 0.f, sy = 0.f;
#pragma unroll
        for (int k = 0; k < SHG_Q; ++k) {
          const float g4[4] = {x[r][k].x, x[r][k].y, x[r][k].z, x[r][k].w};
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const float d = g4[q] < 0.f ? -1.f : 1.f;
            sx = fmaf(d, p[4 * k + q].x, sx);
            sy = fmaf(d, p[4 * k + q].y, sy);
          }
        }
        v[2 * r] = sx;
        v[2 * r + 1] = sy;
      }
      // 8 values over 32 lanes: three halving exchanges leave lane l the value l / 4 summed
      // over 8 lanes, two more steps sum the rest (2 values: one exchange, four steps)
      constexpr int G = 16 / RB;  // lanes per value
#pragma unroll
      for (int w = RB, o = 16; w >= 1; w >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int e = 0; e < w; ++e) {
          const float keep = up ? v[w + e] : v[e], give = up ? v[e] : v[w + e];
          v[e] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
      }
      float t = v[0];
#pragma unroll
      for (int o = G / 2; o >= 1; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (lane % G == 0 && rb * RB + lane / (2 * G) < rn) {
        const int e = 2 * RB * rb + lane / G;
        kahan_add(sums[warp][e], comp[warp][e], t);
      }
      if (++rb == nrb) {
        rb = 0;
        ++seg;
        fresh = true;
      }
    }
    __syncthreads();
    const int r = threadIdx.x;
    if (r < rn) {
      float2 t = make_float2(0.f, 0.f), c = t;
#pragma unroll
      for (int w = 0; w < SHG_WARPS; ++w) {
        kahan_add(t.x, c.x, __fsub_rn(sums[w][2 * r], comp[w][2 * r]));
        kahan_add(t.y, c.y, __fsub_rn(sums[w][2 * r + 1], comp[w][2 * r + 1]));
      }
      const float2 ph = konst[3];  // phi(kappa)
      const float2 E = make_float2(ph.x * t.x - ph.y * t.y, ph.x * t.y + ph.y * t.x);
      eout[r0 + r] = E;
      if (fout) fout[r0 + r] = fit_of(E);
    }
    __syncthreads();  // the sums are zeroed again
  }
}

// ------------------------------------------------- multi-wavelength objective
static constexpr int MW_KMAX = 4;

template <int K>
struct MultiOut {
  const float2 *konst[K];
  float G0, beta;
  float2 *deff;
  float *obj;
};
// the objective of one row from its K combined scans
template <int K>
__device__ __forceinline__ void multi_close(const MultiOut<K> &o, int row, const Mono *m) {
  float f = 0.f, gmax = -1.f, gmin = 3.0e38f;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const float2 D = deff_from(m[k], o.konst[k][0], o.konst[k][1]);
    if (o.deff) o.deff[(size_t)row * K + k] = D;
    const float G = sqrtf(fit_of(D));
    f += fabsf(o.G0 - G);
    gmax = fmaxf(gmax, G);
    gmin = fminf(gmin, G);
  }
  o.obj[row] = f + o.beta * (gmax - gmin);
}

// The qpm_eval sweep with K sign-block tables: for K = 1 the same split and order, so it
// reproduces qpm_eval's plain scan bit for bit.
template <int K, int W, int MODE>
static __global__ void __launch_bounds__(W * 32, rs_ctas(K, W))
    k_multi_genes(const __grid_constant__ GeneMaps maps, const float *__restrict__ src, int64_t ld,
                  RowPlan pl, RowTables<K> tabs, float2 *part, unsigned *ctr, MultiOut<K> out) {
  rows_sweep<K, W, MODE, false>(maps, src, ld, pl, tabs, part, ctr,
                                [&](int row, const Mono *m) { multi_close<K>(out, row, m); });
}

// the K combined scans (as in qpm_eval), then the objective; a programmatic dependent
template <int K>
static __global__ void __launch_bounds__(RC_THREADS)
    k_multi_combine(RowPlan pl, int runs, const float2 *__restrict__ part, MultiOut<K> out) {
  __shared__ Mono sh[K][RC_THREADS];
  const int rows = RC_THREADS / runs, run = threadIdx.x / rows;
  const int row = blockIdx.x * rows + threadIdx.x - run * rows;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  Mono acc[K];
  combine_pieces<K>(pl, part, runs, row, run, sh, acc);
  if (run == 0 && row < pl.NP) multi_close<K>(out, row, acc);
}

template <int K, int W, int MODE>
static qpm_status launch_multi_genes(const GeneMaps &gm, const float *g, int64_t ld, const RowPlan &pl,
                                     const RowTables<K> &tabs, float2 *part, unsigned *ctr,
                                     const MultiOut<K> &out, cudaStream_t s) {
  static SmemAttr attr;
  const void *fn = (const void *)k_multi_genes<K, W, MODE>;
  const qpm_status st = attr.set(fn, rs_smem(K, W));
  if (st != QPM_OK) return st;
  void *args[] = {(void *)&gm, (void *)&g, (void *)&ld, (void *)&pl, (void *)&tabs, (void *)&part,
                  (void *)&ctr, (void *)&out};
  return launch_dependent(fn, dim3(pl.C), dim3(W * 32), args, rs_smem(K, W), s);
}

template <int K>
static qpm_status launch_multi(const float2 *const *blk, const float2 *const *konst, const float *g,
                               int64_t ld, const RowPlan &pl, float G0, float beta, void *scratch,
                               float2 *deff, float *obj, TableLease &lease, cudaStream_t s) {
  constexpr int MANY = K == 1 ? 4 : 8, FEW = K == 1 ? 1 : 2;  // genes_plan's warps per CTA
  GeneMaps gm;
  int mode;
  qpm_status st = make_gene_maps(&gm, &mode, g, pl.NP, pl.N, ld);
  if (st != QPM_OK) return st;
  float2 *part = (float2 *)scratch;
  unsigned *ctr = nullptr;
  if (row_fuse(pl, lease)) {
    void *counters = nullptr;
    if ((st = lease.scratch(FUSE_BYTES, &counters)) != QPM_OK) return st;
    ctr = (unsigned *)counters;
  }
  RowTables<K> tabs;
  MultiOut<K> out{{}, G0, beta, deff, obj};
  for (int k = 0; k < K; ++k) {
    tabs.blk[k] = blk[k];
    out.konst[k] = konst[k];
  }
#define QPM_MG(W, M) st = launch_multi_genes<K, W, M>(gm, g, ld, pl, tabs, part, ctr, out, s)
  if (pl.W == MANY) {
    if (mode == ROWS_TMA) QPM_MG(MANY, ROWS_TMA);
    else QPM_MG(MANY, ROWS_TMA4);
  } else {
    if (mode == ROWS_TMA) QPM_MG(FEW, ROWS_TMA);
    else QPM_MG(FEW, ROWS_TMA4);
  }
#undef QPM_MG
  if (st != QPM_OK || ctr) return st;
  int runs = rc_runs(pl);
  const int rows = RC_THREADS / runs;
  void *args[] = {(void *)&pl, &runs, &part, &out};
  return launch_dependent((const void *)k_multi_combine<K>, dim3((pl.NP + rows - 1) / rows),
                          dim3(RC_THREADS), args, 0, s);
}

}  // namespace qpm

using namespace qpm;

extern "C" qpm_status qpm_eval_shg(const qpm_problem *prob, const float *genes, int64_t ld,
                                   int32_t NP, float *e_shg, float *fit, qpm_stream_t stream) {
  if (!prob || !genes || !e_shg) return fail(QPM_ERR_ARG, "qpm_eval_shg: NULL pointer");
  if (prob->N < 1 || NP < 1) return fail(QPM_ERR_ARG, "qpm_eval_shg: need N >= 1 and NP >= 1");
  if (ld < prob->N) return fail(QPM_ERR_ARG, "qpm_eval_shg: leading dimension smaller than the row");
  cudaStream_t s = (cudaStream_t)stream;
  TableLease lease(prob, 1, s);  // held until the launch below is enqueued
  const float4 *table;
  const float2 *konst;
  qpm_status st = lease.table(prob, &table, &konst);
  if (st != QPM_OK) return st;
  const bool vec = (ld % 4 == 0) && (((uintptr_t)genes & 15) == 0) && prob->N >= 4;
  const int sms = sm_count(), rpc = (NP + sms - 1) / sms, grid = (NP + rpc - 1) / rpc;
  float2 *e = (float2 *)e_shg;
  void *args[] = {(void *)&genes, &ld, &NP, (void *)&prob->N, (void *)&rpc, (void *)&table, (void *)&konst, &e, &fit};
  const void *fn = rpc == 1 ? (vec ? (const void *)k_shg<true, 1> : (const void *)k_shg<false, 1>)
                            : (vec ? (const void *)k_shg<true, SHG_RB> : (const void *)k_shg<false, SHG_RB>);
  return launch_dependent(fn, dim3(grid), dim3(SHG_WARPS * 32), args, 0, s);
}

extern "C" qpm_status qpm_eval_multi(const qpm_problem *probs, int32_t K, const float *genes,
                                     int64_t ld, int32_t NP, float G0, float beta, float *d_eff,
                                     float *objective, void *scratch, size_t scratch_bytes,
                                     qpm_stream_t stream) {
  if (!probs || !genes || !objective) return fail(QPM_ERR_ARG, "qpm_eval_multi: NULL pointer");
  if (K < 1 || K > MW_KMAX) return fail(QPM_ERR_ARG, "qpm_eval_multi: need 1 <= K <= 4");
  const int N = probs[0].N;
  for (int k = 1; k < K; ++k)
    if (probs[k].N != N) return fail(QPM_ERR_ARG, "qpm_eval_multi: all problems need the same N");
  if (N < 1 || NP < 1) return fail(QPM_ERR_ARG, "qpm_eval_multi: need N >= 1 and NP >= 1");
  if (ld < N) return fail(QPM_ERR_ARG, "qpm_eval_multi: leading dimension smaller than the row");
  cudaStream_t s = (cudaStream_t)stream;
  const float2 *blk[MW_KMAX], *konst[MW_KMAX];
  if (NP > EVAL_MAX_ROWS) return fail(QPM_ERR_UNSUPPORTED, "qpm_eval_multi: too many rows");
  // one lease for all K lookups and the launches: room for the K tables is made
  // before the first lookup, so no lookup can evict a table returned before it
  TableLease lease(probs, K, s);
  for (int k = 0; k < K; ++k) {
    qpm_status st = lease.block_table(&probs[k], &blk[k], &konst[k]);
    if (st != QPM_OK) return st;
  }
  const RowPlan pl = genes_plan(K, NP, N, rows_aligned(genes, NP, ld));
  if (!scratch || scratch_bytes < plan_bytes(pl, K))
    return fail(QPM_ERR_ARG, "qpm_eval_multi: scratch smaller than qpm_eval_multi_scratch_bytes()");
#define QPM_MW(KK) \
  launch_multi<KK>(blk, konst, genes, ld, pl, G0, beta, scratch, (float2 *)d_eff, objective, lease, s)
  return K == 1 ? QPM_MW(1) : K == 2 ? QPM_MW(2) : K == 3 ? QPM_MW(3) : QPM_MW(4);
#undef QPM_MW
}

extern "C" size_t qpm_eval_multi_scratch_bytes(int32_t K, int32_t N, int32_t NP) {
  if (K < 1 || N < 1 || NP < 1) return 0;
  const size_t bytes = plan_bytes(genes_plan(std::min(K, (int32_t)MW_KMAX), NP, N, false), K);
  return K > 1 ? bytes : std::max(bytes, plan_bytes(genes_plan(1, NP, N, true), 1));  // only K = 1 looks at it
}
