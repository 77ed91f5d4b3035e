// qpm_hwsda.cu -- the HWSDA generation step (Sec. 3.2, Steps 1-7) on sm_103a.
//
// One CTA is the team for one individual at a time: its T threads split the
// N domains into contiguous chunks of c domains (c a multiple of 4), every thread
// builds its chunk of the new vector (DE trial or GWO candidate) straight from
// the generator and the parent rows, scans it into a monoid partial, and the CTA
// combines the partials in index order to d_eff.  The population is stored in
// the matching permuted order, so that every warp-wide float4 access to a row
// (target, donors, leaders, new vector, phasor table) is one contiguous 512 B
// segment.
//
// Every individual owns two row slots; the new vector is always written to the
// slot that is not current and survives by flipping a per-individual slot
// selector, so no row is ever copied.  DE reads selectors of generation parity
// p and writes those of parity p^1; GWO works in place on parity p^1 (it only
// moves omega wolves and only reads the leaders).
//
// Per generation: k_de (all NP trials + greedy selection + leader choice by the
// last CTA) and k_gwo (omega wolves + greedy selection + generation counter by
// the last CTA); or one cooperative persistent kernel that runs both phases for
// many generations with bounded grid barriers in between; or, for many
// instances, one launch of k_batch in which thread-block clusters take whole
// instances from a queue.
#include <math.h>

#include <string.h>

#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "qpm_common.cuh"
#include "qpm_internal.h"
#include "qpm_sync.cuh"

namespace qpm {

struct InstDev {
  int32_t N, Npad, NP, T, c, G;
  int32_t combine, compensated;
  float F, CR;
  uint32_t crthr;  // cr_threshold(CR)
  uint32_t inst;
  uint2 key;
  double kappa1, kappa2;
  float *pop;            // [NP][2][Npad], permuted rows
  int32_t *sel0, *sel1;  // slot selectors, parity 0 / 1
  float *fit;            // [NP]
  float2 *dval;          // [NP]
  float4 *table;         // [Npad], permuted
  double2 *tpart;        // table reduction scratch
  float2 *konst;         // phi1 phi2, cdiag
  double2 *konst64;      // phi1 phi2, cdiag, psi, phi1 (FP64)
  int32_t *lead;         // [3] (four for the discrete GWO)
  unsigned long long *topk;  // [2][NP * 3] partial leader keys (by generation parity)
  unsigned *ctr;         // [4] CTA-completion counters
  int32_t *gen;          // [1] completed generations
  double2 *rpart;        // [3 ceil(N / 128)] FP64 partials of the best design (get_best)
  float *trace;          // optional fitness trace
  float *Fsched;         // [G + 1] F of every generation, or NULL for constant F; the
                         // adaptive F (f_schedule 2) writes entry g + 1 during generation g
  const float *Fbase;    // [G + 1] adaptive F only: the schedule of its intermediate state
  int32_t adaptive;      // f_schedule == 2
  // the objective (qpm_objective): kind, problems of the multi-wavelength kinds (the
  // first one's table and constants are table / konst), G0, beta; minimised for the
  // multi-wavelength kinds
  int32_t obj, K, minimize;
  int32_t wide;          // launches form: the kernels of 112 registers a thread, not 80 (occupancy)
  const uint32_t *dthr;  // [G][7] discrete GWO (combine 2): social, flip, plus[0..4] thresholds
  float G0, beta;
  const float4 *mtab[8];   // [Npad] permuted phasor tables of the K problems
  const float2 *mkonst[8];  // their FP32 constants
  unsigned long long *dekey;  // [NP] persistent form: DE survivor keys (lead_key) for Step 3
};

template <bool NC>
__device__ __forceinline__ float4 ld4(const float *p) {
  if (NC) return __ldg((const float4 *)p);
  return *(const float4 *)p;
}
// phasor table entry: from shared memory (TS) or through the read-only path
template <bool TS>
__device__ __forceinline__ float4 ldt(const float4 *p) {
  if (TS) return *p;
  return __ldg(p);
}

// Running monoid of a thread's chunk.  Plain: FP32 sums.  Compensated: the
// domains are summed plainly in blocks of 8 and every block is Kahan-folded into
// the running triple (blocked Kahan summation: error of order 8 eps instead of c eps).
template <bool COMP>
struct Acc {
  MonoQ m;  // plain sums / current block
  MonoK k;  // compensated running triple
  __device__ __forceinline__ void zero() {
    m.zero();
    if (COMP) k = monok_zero();
  }
  __device__ __forceinline__ void push(f2x dd, const float4 &p) { mono_push(m, dd, p); }
  // end of a block of domains
  __device__ __forceinline__ void fold() {
    if (COMP) {
      monok_fold_in(k, m.mono());
      m.zero();
    }
  }
  __device__ __forceinline__ Mono get() {
    if (COMP) {
      fold();
      return monok_fold(k);
    }
    return m.mono();
  }
};

__device__ __forceinline__ float sgn(float x) { return x < 0.f ? -1.f : 1.f; }

// ----------------------------------------------------------------- objectives
// The fitness the optimiser works on (qpm_objective.kind): the cascaded d_eff of Sec. 2.1
// (|d_eff|^2, maximised; the default), the SHG field of Sec. 2.1's first step (|E|^2,
// maximised), or the multi-wavelength objective of Sec. 5, sum_k |G0 - G_k| + beta
// (G_max - G_min) over K problems, G_k the cascaded or the SHG field magnitude
// (minimised).  The two single kinds share the one scan (the SHG field is
// phi(kappa1) sum_j d_j e^{-i kappa1 j}, the scan's B); the multi-wavelength kinds run K
// scans of the same vector in their own kernel variants (MK).
constexpr int OBJ_THG = 0, OBJ_SHG = 1, OBJ_MULTI_THG = 2, OBJ_MULTI_SHG = 3;

// the field of a single kind from its reduced scan
__device__ __forceinline__ float2 field_of(const InstDev &I, const Mono &m) {
  if (I.obj == OBJ_SHG) {
    const float2 ph = I.konst[3];  // phi(kappa1)
    return make_float2(ph.x * m.B.x - ph.y * m.B.y, ph.x * m.B.y + ph.y * m.B.x);
  }
  return deff_from(m, I.konst[0], I.konst[1]);
}

// selection key of fitness f of individual i: a larger key is a better individual,
// ties to the lower index (an objective to minimise is >= 0, so ~bits orders it)
__device__ __forceinline__ unsigned long long sel_key(bool minimize, float f, int i) {
  const uint32_t b = __float_as_uint(f);
  return ((unsigned long long)(minimize ? ~b : b) << 32) | (0xFFFFFFFFu - (uint32_t)i);
}

// a phasor-table entry of a multi-wavelength kind: read-only path, kept in L1 ahead of
// other lines (every team on the SM sweeps the same K tables for every individual)
__device__ __forceinline__ float4 ld_table_keep(const float4 *p) {
  float4 v;
  asm("ld.global.nc.L1::evict_last.v4.f32 {%0, %1, %2, %3}, [%4];"
      : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
      : "l"(p));
  return v;
}

// MK != 0: the K scans of a multi-wavelength kind, plain FP32 sums, phasors from the
// problems' tables in global memory (cached in L1 and L2)
// smt (optional): the K tables copied into shared memory by the CTA, [K][Npad] in the
// same permuted order, float4 (p1, p2) entries for the cascaded kind and float2 (p1)
// entries for the SHG kind, which needs p1 only
template <int MK>
struct MultiAcc {
  static constexpr int KMAX = MK == OBJ_MULTI_THG ? 4 : (MK == OBJ_MULTI_SHG ? 8 : 1);
  MonoQ m[KMAX];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int k = 0; k < KMAX; ++k) m[k].zero();
  }
  // one domain of problem k with sign d (dd = (d, d)) and its phasors p (p.zw unused for SHG)
  __device__ __forceinline__ void push1(int k, f2x dd, const float4 &p) {
    if (MK == OBJ_MULTI_THG) mono_push(m[k], dd, p);
    else m[k].B = f2_fma(dd, f2_pack(p.x, p.y), m[k].B);  // the SHG field's sum of d p1
  }
  // group k4 of this thread's chunk (4 domains of signs u); one uniform branch picks
  // the tables' place for the whole group
  __device__ __forceinline__ void push4(const InstDev &I, int k4, int t, float4 u,
                                        const void *smt = nullptr) {
    const Signs4 sg = signs4(u);
    const f2x *d = sg.d;
    if (smt) {
      const int e0 = k4 * 4 * I.T + t;
#pragma unroll
      for (int k = 0; k < KMAX; ++k) {
        if (k < I.K) {
          const int ek = k * I.Npad + e0;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            float4 p;
            if (MK == OBJ_MULTI_SHG) {
              const float2 p1 = ((const float2 *)smt)[ek + q * I.T];
              p = make_float4(p1.x, p1.y, 0.f, 0.f);
            } else {
              p = ((const float4 *)smt)[ek + q * I.T];
            }
            push1(k, d[q], p);
          }
        }
      }
      return;
    }
#pragma unroll
    for (int k = 0; k < KMAX; ++k) {
      if (k < I.K) {
        const float4 *tb = I.mtab[k] + ((uint32_t)k4 * 4u * (uint32_t)I.T + (uint32_t)t);
#pragma unroll
        for (int q = 0; q < 4; ++q) push1(k, d[q], ld_table_keep(tb + (size_t)q * I.T));
      }
    }
  }
};

// Several teams per CTA (the multi-wavelength kinds with shared-memory tables): a team
// is the T consecutive threads [team T, team T + T); team_sync is the team's own
// named barrier (1 + team), a warp barrier for one-warp teams, or the CTA barrier
// when the CTA is one team.
__device__ __forceinline__ int team_thread(const InstDev &I) { return (int)threadIdx.x & (I.T - 1); }
__device__ __forceinline__ void team_sync(const InstDev &I) {
  if ((int)blockDim.x == I.T) {
    __syncthreads();
  } else if (I.T == 32) {
    __syncwarp();
  } else {
    const int team = (int)threadIdx.x / I.T;
    asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "r"(I.T) : "memory");
  }
}

// One step of the K-fold ordered reduction: `n` problems a lane go to n / 2.  Of a pair of lanes
// s apart the lower keeps the first half of the problems and the upper the second half, each
// gets the other's partial of what it keeps, and both combine them lower lanes first.
template <int n, bool SHG, int KM>
__device__ __forceinline__ void multi_halve(Mono (&m)[KM], int s) {
  const bool up = (threadIdx.x & s) != 0;
#pragma unroll
  for (int e = 0; e < n / 2; ++e) {
    const Mono keep = up ? m[n / 2 + e] : m[e], give = up ? m[e] : m[n / 2 + e];
    Mono got;
    got.B.x = __shfl_xor_sync(0xffffffffu, give.B.x, s);
    got.B.y = __shfl_xor_sync(0xffffffffu, give.B.y, s);
    if (SHG) {
      m[e].B = make_float2(keep.B.x + got.B.x, keep.B.y + got.B.y);
    } else {
      got.A.x = __shfl_xor_sync(0xffffffffu, give.A.x, s);
      got.A.y = __shfl_xor_sync(0xffffffffu, give.A.y, s);
      got.C.x = __shfl_xor_sync(0xffffffffu, give.C.x, s);
      got.C.y = __shfl_xor_sync(0xffffffffu, give.C.y, s);
      // mono_combine of (lower, upper): its sums commute, its product does not
      Mono L = keep, R = got;
      if (up) {
        L.B = got.B;
        R.A = keep.A;
        L.A = got.A;
        R.B = keep.B;
      }
      m[e] = mono_combine(L, R);
    }
  }
}

// Reduce the K scans of a team (WT: a warp team) and form the objective: f and the first
// problem's field D0 are valid in the team's first thread; every thread returns.
// The K ordered warp reductions run as one: the first steps halve the number of problems a
// lane carries (multi_halve), after which each of KM lanes finishes one problem's.  The same
// tree of the same additions per problem as K separate reductions, in about a third of the
// shuffles (K = 3: 6 monoids exchanged instead of 15).  A CTA team then passes the warps'
// partials through shared memory (sh holds KM x warps monoids); lane k of its first warp adds
// problem k's in warp order and forms G_k, and the first thread sums the objective in order.
template <int MK, bool WT>
__device__ void multi_finish(const InstDev &I, MultiAcc<MK> &acc, Mono *sh, float &f, float2 &D0) {
  constexpr int KM = MultiAcc<MK>::KMAX;  // 4 or 8
  constexpr bool SHG = MK == OBJ_MULTI_SHG;
  const int t = WT ? (int)(threadIdx.x & 31) : team_thread(I), lane = threadIdx.x & 31;
  Mono m[KM];
#pragma unroll
  for (int k = 0; k < KM; ++k) m[k] = acc.m[k].mono();  // zero past K
  if (KM == 8) {
    multi_halve<8, SHG>(m, 1);
    multi_halve<4, SHG>(m, 2);
    multi_halve<2, SHG>(m, 4);
  } else {
    multi_halve<4, SHG>(m, 1);
    multi_halve<2, SHG>(m, 2);
  }
  // lane l < KM now carries problem k(l): the bits of l in reverse
  const int prob = KM == 8 ? ((lane & 1) << 2) | (lane & 2) | ((lane >> 2) & 1)
                           : ((lane & 1) << 1) | ((lane >> 1) & 1);
  Mono r = m[0];
#pragma unroll
  for (int s = KM; s < 32; s <<= 1) {
    if (SHG) {
      r.B.x += __shfl_down_sync(0xffffffffu, r.B.x, s);
      r.B.y += __shfl_down_sync(0xffffffffu, r.B.y, s);
    } else {
      r = mono_combine(r, mono_shfl_down(r, s));
    }
  }
  if (!WT) {
    // the team's warps and its share of the scratch
    const int warp = t >> 5, nw = I.T >> 5;
    sh += (size_t)((int)threadIdx.x / I.T) * KM * nw;
    if (nw > 1) {
      if (lane < KM) {
        if (SHG) sh[prob * nw + warp].B = r.B;
        else sh[prob * nw + warp] = r;
      }
      team_sync(I);
      if (t < KM) {
        for (int w = 1; w < nw; ++w) {
          const Mono &q = sh[prob * nw + w];
          if (SHG) r.B = make_float2(r.B.x + q.B.x, r.B.y + q.B.y);
          else r = mono_combine(r, q);
        }
      }
    }
  }
  if (t >= 32) return;  // whole warps: the objective is the first warp's
  float2 Dk = make_float2(0.f, 0.f);
  float G = 0.f;
  if (lane < KM && prob < I.K) {
    if (MK == OBJ_MULTI_THG) {
      Dk = deff_from(r, I.mkonst[prob][0], I.mkonst[prob][1]);
    } else {
      const float2 ph = I.mkonst[prob][3];
      Dk = make_float2(ph.x * r.B.x - ph.y * r.B.y, ph.x * r.B.y + ph.y * r.B.x);
    }
    G = sqrtf(fit_of(Dk));
  }
  float obj = 0.f, gmax = -1.f, gmin = 3.0e38f;
#pragma unroll
  for (int k = 0; k < KM; ++k) {
    if (k < I.K) {
      const int src = KM == 8 ? ((k & 1) << 2) | (k & 2) | ((k >> 2) & 1)
                              : ((k & 1) << 1) | ((k >> 1) & 1);
      const float Gk = __shfl_sync(0xffffffffu, G, src);
      obj += fabsf(I.G0 - Gk);
      gmax = fmaxf(gmax, Gk);
      gmin = fminf(gmin, Gk);
    }
  }
  D0 = Dk;  // lane 0 carries problem 0
  f = obj + I.beta * (gmax - gmin);
}

// push the 4 domains of group k4 of this thread's chunk
template <bool COMP, bool TS>
__device__ __forceinline__ void push4(Acc<COMP> &acc, const float4 *tbl, int T, int k4, int t,
                                      float4 u) {
  const float4 *tb = tbl + ((uint32_t)k4 * 4u * (uint32_t)T + (uint32_t)t);
  const Signs4 sg = signs4(u);
  acc.push(sg.d[0], ldt<TS>(tb));
  acc.push(sg.d[1], ldt<TS>(tb + T));
  acc.push(sg.d[2], ldt<TS>(tb + 2 * T));
  acc.push(sg.d[3], ldt<TS>(tb + 3 * T));
}

// Groups of 4 domains thread t of a CTA team works on: none when its whole warp lies past the row
// (t c >= N: the widest teams round N up to 4 T, 24 % at N = 3300 and T = 256).  Such a warp's
// monoid is zero either way, since padding domains carry zero phasors, and the padding genes are
// never read for anything else.
__device__ __forceinline__ int team_groups(const InstDev &I, int t) {
  return (t & ~31) * I.c < I.N ? I.c >> 2 : 0;
}

__device__ __forceinline__ float *row_ptr(const InstDev &I, int i, int slot) {
  return I.pop + ((size_t)2 * i + slot) * I.Npad;
}

// float4 group `off` of individual i's current row.  DUAL: both slots are read
// together with the selector, which takes the selector load off the critical path.
template <bool NC, bool DUAL>
__device__ __forceinline__ float4 ld_cur(const InstDev &I, int i, int slot, uint32_t off) {
  if (DUAL) {
    const float *r0 = I.pop + (size_t)2 * i * I.Npad + off;
    const float4 v0 = ld4<NC>(r0), v1 = ld4<NC>(r0 + I.Npad);
    return slot ? v1 : v0;
  }
  return ld4<NC>(row_ptr(I, i, slot) + off);
}

// ---------------------------------------------------- Step 1: initialisation
// WT: the team is one warp (t = lane, warp reduction) instead of the whole CTA
template <bool COMP, int MK = 0, bool WT = false>
__device__ void init_individual(const InstDev &I, int i, Mono *sh) {
  const int t = WT ? (int)(threadIdx.x & 31) : (int)threadIdx.x;
  const PhiloxKey K = philox_schedule(I.key);
  float *row = row_ptr(I, i, 0);
  Acc<COMP> acc;
  acc.zero();
  MultiAcc<MK> macc;
  if (MK) macc.zero();
  for (int k4 = 0; k4 < I.c / 4; ++k4) {
    const int j0 = t * I.c + 4 * k4;
    const uint4 w = rng4(K, I.inst, TAG_INIT, GEN_INIT, (uint32_t)i, (uint32_t)(j0 >> 2));
    float4 x;
    x.x = __fsub_rn(__fmul_rn(2.0f, u24(w.x)), 1.0f);
    x.y = __fsub_rn(__fmul_rn(2.0f, u24(w.y)), 1.0f);
    x.z = __fsub_rn(__fmul_rn(2.0f, u24(w.z)), 1.0f);
    x.w = __fsub_rn(__fmul_rn(2.0f, u24(w.w)), 1.0f);
    *(float4 *)(row + ((size_t)k4 * I.T + t) * 4) = x;
    if (MK) {
      macc.push4(I, k4, t, x);
    } else {
      push4<COMP, false>(acc, I.table, I.T, k4, t, x);
      if (k4 & 1) acc.fold();
    }
  }
  float2 D = make_float2(0.f, 0.f);
  float f = 0.f;
  if constexpr (MK != 0) {
    multi_finish<MK, WT>(I, macc, sh, f, D);
  } else {
    const Mono m = WT ? warp_reduce(acc.get()) : block_reduce(acc.get(), sh);
    if (t == 0) {
      D = field_of(I, m);
      f = fit_of(D);
    }
  }
  if (t == 0) {
    I.fit[i] = f;
    I.dval[i] = D;
    I.sel0[i] = 0;
    I.sel1[i] = 0;
    if (I.trace) I.trace[i] = f;
  }
}

template <bool COMP, int MK = 0>
static __global__ void k_init(InstDev I) {
  extern __shared__ Mono sh[];
  for (int i = blockIdx.x; i < I.NP; i += gridDim.x) {
    if (i != (int)blockIdx.x) __syncthreads();  // the reduction scratch is reused
    init_individual<COMP, MK>(I, i, sh);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *I.gen = 0;
    for (int k = 0; k < 4; ++k) I.ctr[k] = 0u;
  }
}

// All instances of a state in one launch (blockIdx.y the instance, largest first; one-warp
// teams, 8 per CTA).  One launch per instance kept 64 to 512 one-warp CTAs on the GPU, each
// bound by the latency of its own chain: 27-52 us an instance.  512 instances of 64 individuals,
// tables included: 28.9 ms -> 0.52 ms.
constexpr int INIT_WARPS = 8;
static __global__ void __launch_bounds__(INIT_WARPS * 32)
    k_init_many(const InstDev *__restrict__ insts, const int32_t *__restrict__ order, int n) {
  const int w0 = blockIdx.x * INIT_WARPS + (threadIdx.x >> 5), stride = gridDim.x * INIT_WARPS;
  for (int k = blockIdx.y; k < n; k += gridDim.y) {
    const InstDev I = insts[order[k]];
    for (int i = w0; i < I.NP; i += stride) {
      if (I.compensated) init_individual<true, 0, true>(I, i, nullptr);
      else init_individual<false, 0, true>(I, i, nullptr);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      *I.gen = 0;
      for (int c = 0; c < 4; ++c) I.ctr[c] = 0u;
    }
  }
}

// ------------------------------------------------------------- row staging
// Row staging (STG): the four rows an update reads (own + three donors or leaders)
// and, when the phasor table is not in shared memory (!TS), the group's four table
// entries are copied ahead into shared memory with cp.async, so the next group's
// loads are in flight during this group's arithmetic without holding registers.
// Two stages (one group ahead): a third stage, measured where the table comes from
// global memory, sped the memory-bound DE phase up by 2 % and slowed the GWO phase
// down by 7 %.  Each thread owns its slots
// stg[(stage * SPS + k) * blockDim.x + threadIdx.x] (SPS = 4 rows, + 4 table
// entries when !TS) and reads back only what it copied itself, so no barrier is
// needed.
constexpr int BATCH_WARPS = 16;  // warps per CTA of the batched form
__host__ __device__ constexpr int stg_stages(bool) { return 2; }
__host__ __device__ constexpr int stg_f4_per_thread(bool ts) {
  return stg_stages(ts) * (ts ? 4 : 8);
}
// The pipeline of one individual's groups: the row and table pointers of the next group to copy
// move on by one group (64-bit adds on the ALU pipe; an index times a stride is a wide multiply
// on the FMA-heavy pipe, which the generator already fills: 512 instances 3.45 -> 3.24 ms per
// generation).  WT: one-warp teams of the batched form, whose T = 32 and CTA width are constants.
template <bool TS, bool WT>
struct RowStage {
  static constexpr int SPS = stg_f4_per_thread(TS) / stg_stages(TS);
  const float4 *r[4], *tb;
  float4 *s;       // this thread's slots of stage 0
  int left, cur;   // groups not yet copied; stage of the next copy
  __device__ __forceinline__ int nt() const { return WT ? BATCH_WARPS * 32 : (int)blockDim.x; }
  // t: the thread's place in the team; the first group's copies are issued
  __device__ __forceinline__ void begin(float4 *stg, int n4, int T, int t, const float *r0,
                                        const float *r1, const float *r2, const float *r3,
                                        const float4 *tbl) {
    r[0] = (const float4 *)r0 + t;
    r[1] = (const float4 *)r1 + t;
    r[2] = (const float4 *)r2 + t;
    r[3] = (const float4 *)r3 + t;
    tb = tbl + t;
    s = stg + threadIdx.x;
    left = n4;
    cur = 0;
    copy(T);
  }
  __device__ __forceinline__ void copy(int T) {
    if (left > 0) {
      float4 *d = s + (cur ? SPS * nt() : 0);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        cp_async16(d + k * nt(), r[k]);
        r[k] += T;
      }
      if (!TS) {
#pragma unroll
        for (int q = 0; q < 4; ++q) cp_async16(d + (4 + q) * nt(), tb + q * T);
        tb += 4 * T;
      }
      --left;
    }
    cp_async_commit();  // possibly empty: one group of copies per iteration
    cur ^= 1;
  }
  // the next group has landed; its slots: rows at [0, 4 nt), table entries at [4 nt, 8 nt) if !TS
  __device__ __forceinline__ const float4 *next(int T) {
    copy(T);
    cp_async_wait<1>();
    return s + (cur ? SPS * nt() : 0);
  }
};
// the push of one staged group: table entries from the stage when !TS
template <bool COMP, bool TS, bool WT>
__device__ __forceinline__ void push4_staged(Acc<COMP> &acc, const float4 *tbl, int T, int k4,
                                             int t, const float4 *st, float4 u) {
  if (TS) push4<COMP, true>(acc, tbl, T, k4, t, u);
  else push4<COMP, true>(acc, st + 4 * (WT ? BATCH_WARPS * 32 : (int)blockDim.x),
                         WT ? BATCH_WARPS * 32 : (int)blockDim.x, 0, 0, u);
}

// The DE donors of the individuals first, first + stride, ...: lane l of a warp draws those of the
// l-th next one, 32 at a time, and each is handed out by shuffles.  (Every thread of the team
// drawing the same four numbers per individual was a tenth of the DE phase at N = 3300; 5000
// rows of it 157.2 -> 152.5 us per generation.  k_de and the batched form, where it made no
// difference beyond 2 % either way, draw per individual.)
struct Donors {
  int4 mine;
  int k;
  __device__ __forceinline__ Donors() : k(0) {}
  __device__ __forceinline__ int4 next(const InstDev &I, const PhiloxKey &K, int g, int i, int stride) {
    if ((k & 31) == 0) {
      const int64_t e = (int64_t)i + (int64_t)(threadIdx.x & 31) * stride;
      mine = de_indices(K, I.inst, (uint32_t)g, e < I.NP ? (int)e : i, I.NP, I.N);
    }
    const int s = k & 31;
    ++k;
    return make_int4(__shfl_sync(0xffffffffu, mine.x, s), __shfl_sync(0xffffffffu, mine.y, s),
                     __shfl_sync(0xffffffffu, mine.z, s), __shfl_sync(0xffffffffu, mine.w, s));
  }
};

// ---------------------------------------------------- the updates of 4 genes
// DE rand/1/bin of 4 neighbouring genes: v = fl(x_r1 + fl(F fl(x_r2 - x_r3))) (no FMA), clamped;
// u = v if U <= CR (integer form, w) or j == jrand, else x.  jm: jrand - (the first gene's index).
// Packed pairs: every operation keeps its own rounding.
__device__ __forceinline__ float4 de_update4(const float4 &x, const float4 &b, const float4 &p,
                                             const float4 &q, uint4 w, float F, uint32_t crthr,
                                             uint32_t jm) {
  const f2x nF = f2_pack(-F, -F);  // b - fl(-F d): the product must round by itself
  const float2 v0 = f2_unpack(
      f2_sub(f2_pack(b.x, b.y), f2_mul(nF, f2_sub(f2_pack(p.x, p.y), f2_pack(q.x, q.y)))));
  const float2 v1 = f2_unpack(
      f2_sub(f2_pack(b.z, b.w), f2_mul(nF, f2_sub(f2_pack(p.z, p.w), f2_pack(q.z, q.w)))));
  if (jm < 4u) {  // one thread of the team, once per individual
    if (jm == 0u) w.x = 0u;
    if (jm == 1u) w.y = 0u;
    if (jm == 2u) w.z = 0u;
    if (jm == 3u) w.w = 0u;
  }
  float4 u;
  u.x = w.x <= crthr ? clamp1(v0.x) : x.x;
  u.y = w.y <= crthr ? clamp1(v0.y) : x.y;
  u.z = w.z <= crthr ? clamp1(v1.x) : x.z;
  u.w = w.w <= crthr ? clamp1(v1.y) : x.w;
  return u;
}

// one leader's pull on two genes: A = fl(fl(2a r1) - a), C = 2 r2, D = |fl(fl(C Xp) - x)|,
// Y = fl(Xp - fl(A D)), in this order, no FMA
__device__ __forceinline__ f2x gwo_pull2(f2x Xp, f2x x, uint32_t w0, uint32_t w1, f2x two_a, f2x a) {
  const float2 A = f2_unpack(f2_sub(f2_mul(two_a, u16hi2(w0, w1)), a));
  const float2 d = f2_unpack(f2_sub(f2_mul(twice_u16lo2(w0, w1), Xp), x));
  return f2_sub(Xp, f2_pack(__fmul_rn(A.x, fabsf(d.x)), __fmul_rn(A.y, fabsf(d.y))));
}
// the three pulls on two genes and their combination: the mean, or |Y_k|-weighted (WEIGHTED)
template <bool WEIGHTED>
__device__ __forceinline__ float2 gwo_update2(f2x x, f2x L0, f2x L1, f2x L2, uint32_t a0, uint32_t a1,
                                              uint32_t b0, uint32_t b1, uint32_t c0, uint32_t c1,
                                              f2x two_a, f2x a) {
  const f2x Y0 = gwo_pull2(L0, x, a0, a1, two_a, a), Y1 = gwo_pull2(L1, x, b0, b1, two_a, a);
  const f2x Y2 = gwo_pull2(L2, x, c0, c1, two_a, a);
  float2 v;
  if (!WEIGHTED) {
    v = div3_rn2(f2_add(f2_add(Y0, Y1), Y2));
  } else {
    const float2 y0 = f2_unpack(Y0), y1 = f2_unpack(Y1), y2 = f2_unpack(Y2);
    auto mean = [](float p, float q, float r) {
      const float m0 = fabsf(p), m1 = fabsf(q), m2 = fabsf(r);
      const float s = __fadd_rn(__fadd_rn(m0, m1), m2);
      const float num = __fadd_rn(__fadd_rn(__fmul_rn(m0, p), __fmul_rn(m1, q)), __fmul_rn(m2, r));
      return (s == 0.0f) ? 0.0f : __fdiv_rn(num, __fmul_rn(3.0f, s));
    };
    v = make_float2(mean(y0.x, y1.x, y2.x), mean(y0.y, y1.y, y2.y));
  }
  return make_float2(clamp1(v.x), clamp1(v.y));
}
template <bool WEIGHTED>
__device__ __forceinline__ float4 gwo_update4(const float4 &x, const float4 &L0, const float4 &L1,
                                              const float4 &L2, const uint4 w[3], float two_a,
                                              float a) {
  const f2x t2 = f2_pack(two_a, two_a), a2 = f2_pack(a, a);
  const float2 lo = gwo_update2<WEIGHTED>(f2_pack(x.x, x.y), f2_pack(L0.x, L0.y), f2_pack(L1.x, L1.y),
                                          f2_pack(L2.x, L2.y), w[0].x, w[0].y, w[1].x, w[1].y,
                                          w[2].x, w[2].y, t2, a2);
  const float2 hi = gwo_update2<WEIGHTED>(f2_pack(x.z, x.w), f2_pack(L0.z, L0.w), f2_pack(L1.z, L1.w),
                                          f2_pack(L2.z, L2.w), w[0].z, w[0].w, w[1].z, w[1].w,
                                          w[2].z, w[2].w, t2, a2);
  return make_float4(lo.x, lo.y, hi.x, hi.y);
}

// The CTA reductions of consecutive individuals take turns on two scratch buffers, so that the
// other warps start on the next individual while thread 0 still folds the warps' totals and
// selects: the barrier inside the next reduction is what frees this one's buffer.  (With one
// buffer and a barrier per individual, 5000 rows of N = 3300 took 164 us per generation; 157 with two.)
__device__ __forceinline__ Mono *red_next(Mono *sh, int &turn) {
  turn ^= 1;
  return sh + (turn ? 0 : (int)(blockDim.x >> 5));
}

// ------------------------------------------ Step 2: DE rand/1/bin + selection
// returns (in thread 0) the key of the survivor for the leader choice
// WT: the team is one warp (t = lane, warp reduction) instead of the whole CTA
// r = (r1, r2, r3, jrand) from de_indices
// STG: rows staged through stg (known slots only, so not with DUAL)
// has_wcr: wcr is the crossover word of the thread's first group of 4 domains, drawn
// earlier (while waiting at the grid barrier)
template <bool COMP, bool NC, bool TS, bool DUAL, bool WT = false, bool STG = false, int MK = 0>
__device__ unsigned long long de_individual(const InstDev &I, const PhiloxKey &K,
                                            const float4 *tbl, int g, int i, const int4 r,
                                            const int32_t *sel_in, int32_t *sel_out, Mono *sh,
                                            int *slot_out = nullptr, float4 *stg = nullptr,
                                            bool has_wcr = false,
                                            uint4 wcr = make_uint4(0u, 0u, 0u, 0u),
                                            int own_slot = -1, int *impr_out = nullptr,
                                            const void *smt = nullptr) {
  static_assert(!(STG && DUAL), "staged rows need known slots");
  // only the multi-wavelength kinds put several teams in a CTA
  const int t = WT ? (int)(threadIdx.x & 31) : (MK ? team_thread(I) : (int)threadIdx.x);
  const float fx = (t == 0) ? I.fit[i] : 0.f;  // issued early, used after the scan
  // own_slot >= 0: the individual's current slot, known to the caller
  const int si = own_slot >= 0 ? own_slot : sel_in[i];
  const int s1 = sel_in[r.x], s2 = sel_in[r.y], s3 = sel_in[r.z];
  float4 *out = (float4 *)row_ptr(I, i, si ^ 1) + t;
  const float F = I.Fsched ? I.Fsched[g] : I.F;
  const uint32_t crthr = I.crthr;
  const int n4 = WT ? I.c / 4 : team_groups(I, t);
  const float *ra = row_ptr(I, i, si), *rb = row_ptr(I, r.x, s1);
  const float *rp = row_ptr(I, r.y, s2), *rq = row_ptr(I, r.z, s3);
  const int T = WT ? 32 : I.T;
  RowStage<TS, WT> rows;
  if (STG) rows.begin(stg, n4, T, t, ra, rb, rp, rq, tbl);
  Acc<COMP> acc;
  acc.zero();
  MultiAcc<MK> macc;
  if (MK) macc.zero();
  for (int k4 = 0; k4 < n4; ++k4) {
    const uint32_t off = ((uint32_t)k4 * (uint32_t)T + (uint32_t)t) * 4u;
    float4 a, b, p, q;
    const float4 *st = nullptr;
    if (STG) {
      st = rows.next(T);
      const int nt = rows.nt();
      a = st[0];
      b = st[nt];
      p = st[2 * nt];
      q = st[3 * nt];
    } else {
      // a known own slot needs one row read, not both
      a = own_slot >= 0 ? ld_cur<NC, false>(I, i, si, off) : ld_cur<NC, DUAL>(I, i, si, off);
      b = ld_cur<NC, DUAL>(I, r.x, s1, off);
      p = ld_cur<NC, DUAL>(I, r.y, s2, off);
      q = ld_cur<NC, DUAL>(I, r.z, s3, off);
    }
    const int j0 = t * I.c + 4 * k4;
    const uint4 w = (has_wcr && k4 == 0)
                        ? wcr
                        : rng4(K, I.inst, TAG_CR, (uint32_t)g, (uint32_t)i, (uint32_t)(j0 >> 2));
    const float4 u = de_update4(a, b, p, q, w, F, crthr, (uint32_t)(r.w - j0));
    *out = u;
    out += T;
    if (MK) {
      macc.push4(I, k4, t, u, smt);
    } else {
      if (STG) push4_staged<COMP, TS, WT>(acc, tbl, T, k4, t, st, u);
      else push4<COMP, TS>(acc, tbl, T, k4, t, u);
      if (k4 & 1) acc.fold();
    }
  }
  float2 D = make_float2(0.f, 0.f);
  float f = 0.f;
  if constexpr (MK != 0) {
    multi_finish<MK, WT>(I, macc, sh, f, D);
  } else {
    // a single group of 4 domains per thread needs no compensation (its plain sums are
    // what the fold would return, up to the sign of a zero), and skipping the fold
    // takes a dependent chain off the phase's critical path
    const Mono mine = (COMP && !WT && n4 <= 1) ? acc.m.mono() : acc.get();
    const Mono m = WT ? warp_reduce(mine) : block_reduce(mine, sh);
    if (t == 0) {
      D = field_of(I, m);
      f = fit_of(D);
    }
  }
  unsigned long long key = 0ull;
  if (t == 0) {
    // greedy one-to-one selection: maximising, or minimising the multi-wavelength kinds
    const bool accept = MK ? (f <= fx) : (f >= fx);
    sel_out[i] = accept ? (si ^ 1) : si;
    if (accept) {
      I.fit[i] = f;
      I.dval[i] = D;
    }
    if (I.trace) I.trace[(size_t)I.NP * (1 + 2 * (size_t)g) + i] = f;
    key = sel_key(MK != 0, accept ? f : fx, i);
    if (slot_out) *slot_out = accept ? (si ^ 1) : si;  // the survivor's slot
    if (impr_out) *impr_out = MK ? (f < fx) : (f > fx);  // a strict improvement (adaptive F)
  }
  return key;
}

// a_g = 2 (G - g) / G
__device__ __forceinline__ float a_of(const InstDev &I, int g) {
  return __fdiv_rn((float)(2 * (I.G - g)), (float)I.G);
}

// ------------------------------------------------ Step 4-5: GWO + selection
// a = a_of(I, g), computed once per phase
// PRE: the three GWO random words of the thread's first group of 4 domains were
// drawn earlier (while waiting at the grid barrier) and are passed in wpre.
// One word per leader and gene gives that leader's (r1, r2) as its 16-bit halves.
template <bool COMP, bool NC, bool TS, bool DUAL, bool WT = false, bool PRE = false,
          bool STG = false, int MK = 0>
__device__ void gwo_individual(const InstDev &I, const PhiloxKey &K, const float4 *tbl, int g,
                               float a, int i, int32_t *sel, int la, int lb, int ld, Mono *sh,
                               const uint4 *wpre = nullptr,
                               float4 own0 = make_float4(0.f, 0.f, 0.f, 0.f),
                               float4 own1 = make_float4(0.f, 0.f, 0.f, 0.f),
                               const int32_t *lslot = nullptr, float4 *stg = nullptr,
                               int own_slot = -1, int *slot_out = nullptr,
                               const void *smt = nullptr) {
  static_assert(!(STG && (DUAL || PRE)), "staged rows need known slots and no prefetched row");
  // only the multi-wavelength kinds put several teams in a CTA
  const int t = WT ? (int)(threadIdx.x & 31) : (MK ? team_thread(I) : (int)threadIdx.x);
  const float fx = (t == 0) ? I.fit[i] : 0.f;
  // lslot: the leaders' current slots, when the leader search delivered them;
  // own_slot >= 0: the individual's current slot, known to the caller
  const int si = own_slot >= 0 ? own_slot : sel[i];
  const int sa = lslot ? lslot[0] : sel[la], sb = lslot ? lslot[1] : sel[lb];
  const int sd = lslot ? lslot[2] : sel[ld];
  float4 *out = (float4 *)row_ptr(I, i, si ^ 1) + t;
  const float two_a = __fmul_rn(2.0f, a);
  const int n4 = WT ? I.c / 4 : team_groups(I, t);
  const float *rx = row_ptr(I, i, si), *r0 = row_ptr(I, la, sa), *r1 = row_ptr(I, lb, sb);
  const float *r2 = row_ptr(I, ld, sd);
  const int T = WT ? 32 : I.T;
  RowStage<TS, WT> rows;
  if (STG) rows.begin(stg, n4, T, t, rx, r0, r1, r2, tbl);
  Acc<COMP> acc;
  acc.zero();
  MultiAcc<MK> macc;
  if (MK) macc.zero();
  for (int k4 = 0; k4 < n4; ++k4) {
    const uint32_t off = ((uint32_t)k4 * (uint32_t)T + (uint32_t)t) * 4u;
    float4 x, L0, L1, L2;
    const float4 *st = nullptr;
    if (STG) {
      st = rows.next(T);
      const int nt = rows.nt();
      x = st[0];
      L0 = st[nt];
      L1 = st[2 * nt];
      L2 = st[3 * nt];
    } else {
      x = (PRE && k4 == 0) ? (si ? own1 : own0) : ld_cur<NC, DUAL>(I, i, si, off);
      // a known slot needs one row read, not both
      L0 = lslot ? ld_cur<NC, false>(I, la, sa, off) : ld_cur<NC, DUAL>(I, la, sa, off);
      L1 = lslot ? ld_cur<NC, false>(I, lb, sb, off) : ld_cur<NC, DUAL>(I, lb, sb, off);
      L2 = lslot ? ld_cur<NC, false>(I, ld, sd, off) : ld_cur<NC, DUAL>(I, ld, sd, off);
    }
    const uint32_t jg = (uint32_t)((t * I.c + 4 * k4) >> 2);
    uint4 w[3];
    if (PRE && k4 == 0) {
#pragma unroll
      for (int k = 0; k < 3; ++k) w[k] = wpre[k];
    } else {
#pragma unroll
      for (int k = 0; k < 3; ++k) w[k] = rng4(K, I.inst, TAG_GWO + k, (uint32_t)g, (uint32_t)i, jg);
    }
    const float4 y = I.combine == 0 ? gwo_update4<false>(x, L0, L1, L2, w, two_a, a)
                                    : gwo_update4<true>(x, L0, L1, L2, w, two_a, a);
    *out = y;
    out += T;
    if (MK) {
      macc.push4(I, k4, t, y, smt);
    } else {
      if (STG) push4_staged<COMP, TS, WT>(acc, tbl, T, k4, t, st, y);
      else push4<COMP, TS>(acc, tbl, T, k4, t, y);
      if (k4 & 1) acc.fold();
    }
  }
  float2 D = make_float2(0.f, 0.f);
  float f = 0.f;
  if constexpr (MK != 0) {
    multi_finish<MK, WT>(I, macc, sh, f, D);
  } else {
    // a single group of 4 domains per thread needs no compensation (its plain sums are
    // what the fold would return, up to the sign of a zero), and skipping the fold
    // takes a dependent chain off the phase's critical path
    const Mono mine = (COMP && !WT && n4 <= 1) ? acc.m.mono() : acc.get();
    const Mono m = WT ? warp_reduce(mine) : block_reduce(mine, sh);
    if (t == 0) {
      D = field_of(I, m);
      f = fit_of(D);
    }
  }
  if (t == 0) {
    const bool accept = MK ? (f <= fx) : (f >= fx);
    if (accept) {
      sel[i] = si ^ 1;
      I.fit[i] = f;
      I.dval[i] = D;
    }
    if (I.trace) I.trace[(size_t)I.NP * (2 + 2 * (size_t)g) + i] = f;
    if (slot_out) *slot_out = accept ? (si ^ 1) : si;  // the survivor's slot
  }
}

// The keys carry the survivor's slot and whether its trial strictly improved on the
// target: fitness bits << 32 | (0x3FFFFFFF - i) << 2 | improved << 1 | slot, which
// orders like lead_key (the two low bits never separate two individuals).
__device__ __forceinline__ unsigned long long slot_key(unsigned long long key, int i, int slot,
                                                       int improved = 0) {
  return (key & 0xFFFFFFFF00000000ull) |
         (unsigned long long)(((0x3FFFFFFFu - (uint32_t)i) << 2) | ((uint32_t)improved << 1) |
                              (uint32_t)slot);
}
__device__ __forceinline__ int slot_key_index(unsigned long long k) {
  return (int)(0x3FFFFFFFu - ((uint32_t)k >> 2));
}

// ------------------------------------------------------------- adaptive F
// Sec. 3.1.1's adaptive F (f_schedule 2).  The paper keeps F in [0.01, 0.1], raises it
// when the population's diversity is low (standard deviation below a threshold, or a
// convergence rate below 0.1), lowers it when diversity is too high or the fitness
// range small (deviation above a threshold, or range below 10^3), and otherwise lets
// it follow the cosine-times-quadratic decay.  Readings (the paper gives neither the
// thresholds nor the steps): after the DE phase of generation g, over the DE survivors,
// cv = the fitness' standard deviation over its mean, the convergence rate = the
// fraction of trials that strictly improved on their target; cv < 0.05 or a rate below
// 0.1 raises F to min(0.1, 1.25 F); cv > 0.5 or max f - min f < 10^3 lowers it to
// max(0.01, 0.8 F); otherwise F = Fbase[g + 1] = 0.1 (cos(pi (g+1) / 2G) + 1) / 2
// (1 - 0.2 ((g+1)/G)^2).  The decision uses exact integer statistics, so that it does
// not depend on a summation order: with E such that 2^(E-1) <= max f < 2^E, every
// fitness is quantised to n = floor(f 2^(20 - E)) by shifting its significand, and
// S1 = sum n, S2 = sum n^2 are 64-bit integers (NP <= 2^23); cv^2 < t^2 is tested as
// NP S2 - S1^2 < t^2 S1^2 with every FP64 operation rounded once.
constexpr float AF_FMIN = 0.01f, AF_FMAX = 0.1f, AF_UP = 1.25f, AF_DOWN = 0.8f;

// n = floor(f 2^(20 - E)) for the fitness bits fb (f >= 0) and the exponent field emax
// (>= 1) of the largest fitness: f = m 2^(e - 150), m the 24-bit significand
__device__ __forceinline__ uint32_t af_quantise(uint32_t fb, uint32_t emax) {
  uint32_t e = (fb >> 23) & 0xFFu, m = fb & 0x7FFFFFu;
  if (e == 0) e = 1;
  else m |= 0x800000u;
  const uint32_t sh = 4u + emax - e;
  return sh >= 24u ? 0u : m >> sh;
}

// F of generation g + 1 from the survivor keys of generation g (slot_key layout), by
// every thread of one CTA; thread 0 writes it to I.Fsched[g + 1].  Every thread returns
// after a CTA barrier.
__device__ void adaptive_F_block(const InstDev &I, const unsigned long long *keys, int g) {
  __shared__ uint32_t red_u[3][32];
  __shared__ unsigned long long red_s[2][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  uint32_t mx = 0u, mn = 0xFFFFFFFFu, cnt = 0u;
  for (int i = threadIdx.x; i < I.NP; i += blockDim.x) {
    const unsigned long long k = keys[i];
    const uint32_t fb = I.minimize ? ~(uint32_t)(k >> 32) : (uint32_t)(k >> 32);  // f's bits
    mx = max(mx, fb);
    mn = min(mn, fb);
    cnt += ((uint32_t)k >> 1) & 1u;
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  mn = __reduce_min_sync(0xffffffffu, mn);
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  if (lane == 0) {
    red_u[0][warp] = mx;
    red_u[1][warp] = mn;
    red_u[2][warp] = cnt;
  }
  __syncthreads();
  mx = 0u;
  mn = 0xFFFFFFFFu;
  cnt = 0u;
  for (int w = 0; w < nw; ++w) {
    mx = max(mx, red_u[0][w]);
    mn = min(mn, red_u[1][w]);
    cnt += red_u[2][w];
  }
  uint32_t emax = (mx >> 23) & 0xFFu;
  if (emax == 0) emax = 1;
  unsigned long long s1 = 0ull, s2 = 0ull;
  for (int i = threadIdx.x; i < I.NP; i += blockDim.x) {
    const uint32_t hi = (uint32_t)(keys[i] >> 32);
    const uint32_t n = af_quantise(I.minimize ? ~hi : hi, emax);
    s1 += n;
    s2 += (unsigned long long)n * n;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s1 += __shfl_xor_sync(0xffffffffu, s1, o);
    s2 += __shfl_xor_sync(0xffffffffu, s2, o);
  }
  if (lane == 0) {
    red_s[0][warp] = s1;
    red_s[1][warp] = s2;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    s1 = s2 = 0ull;
    for (int w = 0; w < nw; ++w) {
      s1 += red_s[0][w];
      s2 += red_s[1][w];
    }
    const double a = __dmul_rn((double)I.NP, (double)s2);
    const double b = __dmul_rn((double)s1, (double)s1);
    const double num = __dsub_rn(a, b);
    const float range = __fsub_rn(__uint_as_float(mx), __uint_as_float(mn));
    const bool low = (s1 == 0ull) || (num < __dmul_rn(0.0025, b)) ||
                     (10ull * cnt < (unsigned long long)I.NP);
    const bool high = !low && ((num > __dmul_rn(0.25, b)) || (range < 1000.0f));
    const float Fg = I.Fsched[g];
    I.Fsched[g + 1] = low ? fminf(AF_FMAX, __fmul_rn(Fg, AF_UP))
                          : (high ? fmaxf(AF_FMIN, __fmul_rn(Fg, AF_DOWN)) : I.Fbase[g + 1]);
  }
  __syncthreads();
}

// ------------------------------------------- four-leader discrete GWO (Sec. 3.1.2)
// The paper describes it only qualitatively (continuous positions mapped to +-1; state
// transitions from the four leaders' state distribution with a dispersion parameter;
// much disturbance early, the dominant state and rare flips late; a falling social-
// learning rate that copies a random leader).  Reading, per omega wolf and gene, with
// n the number of the four leaders whose gene is +1 and tau = g / G: with probability
// sigma = 0.3 (1 - tau) take leader kl's state (kl uniform in 0..3), else +1 with
// probability P_n = (1 - delta) q_n + delta / 2, delta = 0.5 (1 - tau),
// q_n = (1 - tau) n / 4 + tau [n > 2, or 1/2 for n = 2]; then flip with probability
// mu = 0.1 (1 - tau) + 0.01 tau.  The probabilities are 16-bit thresholds per
// generation (computed on the host in FP64, I.dthr), tested against the 16-bit halves
// of two words per gene (tag GWO: social high, transition low; tag GWO + 1: flip high,
// kl the low two bits).  The new genes are +-1.
__device__ __forceinline__ void top4_insert(unsigned long long &k0, unsigned long long &k1,
                                            unsigned long long &k2, unsigned long long &k3,
                                            unsigned long long x) {
  if (x > k0) { k3 = k2; k2 = k1; k1 = k0; k0 = x; }
  else if (x > k1) { k3 = k2; k2 = k1; k1 = x; }
  else if (x > k2) { k3 = k2; k2 = x; }
  else if (x > k3) { k3 = x; }
}

// the generation's thresholds: social, flip, and P(+1) for 0 .. 4 leaders at +1
struct DiscThr {
  uint32_t soc, flip, p0, p1, p2, p3, p4;
};

// the new state of one gene from the four leaders' genes and the two random words
__device__ __forceinline__ float disc_gene(float a, float b, float c, float d, uint32_t w1,
                                           uint32_t w2, const DiscThr &th) {
  const float s0 = sgn(a), s1 = sgn(b), s2 = sgn(c), s3 = sgn(d);
  const int n = (s0 > 0.f) + (s1 > 0.f) + (s2 > 0.f) + (s3 > 0.f);
  const uint32_t kl = w2 & 3u;
  float v;
  if ((w1 >> 16) < th.soc) {  // social learning: a random leader's state
    v = kl == 0u ? s0 : (kl == 1u ? s1 : (kl == 2u ? s2 : s3));
  } else {  // transition from the leaders' state distribution
    const uint32_t tp = n == 0 ? th.p0 : (n == 1 ? th.p1 : (n == 2 ? th.p2 : (n == 3 ? th.p3 : th.p4)));
    v = (w1 & 0xFFFFu) < tp ? 1.f : -1.f;
  }
  return (w2 >> 16) < th.flip ? -v : v;  // disturbance
}

// one candidate of the discrete GWO for omega wolf i and its greedy selection, by the
// CTA (team T); L: the four leaders' current rows
template <bool COMP>
__device__ void gwo_discrete_individual(const InstDev &I, const PhiloxKey &K, int g, int i,
                                        int32_t *sel, const float *L0, const float *L1,
                                        const float *L2, const float *L3, Mono *sh) {
  const int t = threadIdx.x;
  const float fx = (t == 0) ? I.fit[i] : 0.f;
  const int si = sel[i];
  float *out = row_ptr(I, i, si ^ 1);
  const uint32_t *tg = I.dthr + (size_t)7 * g;
  const DiscThr th{tg[0], tg[1], tg[2], tg[3], tg[4], tg[5], tg[6]};
  Acc<COMP> acc;
  acc.zero();
  const int n4 = team_groups(I, t);
  for (int k4 = 0; k4 < n4; ++k4) {
    const uint32_t off = ((uint32_t)k4 * (uint32_t)I.T + (uint32_t)t) * 4u;
    const float4 l0 = __ldg((const float4 *)(L0 + off)), l1 = __ldg((const float4 *)(L1 + off));
    const float4 l2 = __ldg((const float4 *)(L2 + off)), l3 = __ldg((const float4 *)(L3 + off));
    const uint32_t jg = (uint32_t)((t * I.c + 4 * k4) >> 2);
    const uint4 w1 = rng4(K, I.inst, TAG_GWO, (uint32_t)g, (uint32_t)i, jg);
    const uint4 w2 = rng4(K, I.inst, TAG_GWO + 1, (uint32_t)g, (uint32_t)i, jg);
    float4 y;
    y.x = disc_gene(l0.x, l1.x, l2.x, l3.x, w1.x, w2.x, th);
    y.y = disc_gene(l0.y, l1.y, l2.y, l3.y, w1.y, w2.y, th);
    y.z = disc_gene(l0.z, l1.z, l2.z, l3.z, w1.z, w2.z, th);
    y.w = disc_gene(l0.w, l1.w, l2.w, l3.w, w1.w, w2.w, th);
    *(float4 *)(out + off) = y;
    push4<COMP, false>(acc, I.table, I.T, k4, t, y);
    if (k4 & 1) acc.fold();
  }
  const Mono m = block_reduce(acc.get(), sh);
  if (t == 0) {
    const float2 D = field_of(I, m);
    const float f = fit_of(D);
    const bool accept = f >= fx;
    if (accept) {
      sel[i] = si ^ 1;
      I.fit[i] = f;
      I.dval[i] = D;
    }
    if (I.trace) I.trace[(size_t)I.NP * (2 + 2 * (size_t)g) + i] = f;
  }
}

// top-3 merge over the CTA: every thread passes its sorted triple, thread 0 gets the result
__device__ void block_top3(unsigned long long &k0, unsigned long long &k1, unsigned long long &k2,
                           unsigned long long *sh) {
  for (int s = 16; s > 0; s >>= 1) {
    const unsigned long long p0 = __shfl_xor_sync(0xffffffffu, k0, s);
    const unsigned long long p1 = __shfl_xor_sync(0xffffffffu, k1, s);
    const unsigned long long p2 = __shfl_xor_sync(0xffffffffu, k2, s);
    top3_insert(k0, k1, k2, p0);
    top3_insert(k0, k1, k2, p1);
    top3_insert(k0, k1, k2, p2);
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  __syncthreads();
  if (lane == 0) {
    sh[3 * warp] = k0;
    sh[3 * warp + 1] = k1;
    sh[3 * warp + 2] = k2;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < nw; ++w) {
      top3_insert(k0, k1, k2, sh[3 * w]);
      top3_insert(k0, k1, k2, sh[3 * w + 1]);
      top3_insert(k0, k1, k2, sh[3 * w + 2]);
    }
  }
  __syncthreads();
}

// merge all per-CTA partial triples in topk[0 .. 3*nparts) into the leaders; warp 0
// does the work, every thread returns after the CTA barrier (thread 0 writes lead)
__device__ void merge_leaders(const unsigned long long *topk, int nparts, int32_t *lead,
                              int32_t *lead_sh) {
  if (threadIdx.x < 32) {
    unsigned long long k0 = 0, k1 = 0, k2 = 0;
    for (int e = threadIdx.x; e < 3 * nparts; e += 32) top3_insert(k0, k1, k2, topk[e]);
    for (int s = 16; s > 0; s >>= 1) {
      const unsigned long long p0 = __shfl_xor_sync(0xffffffffu, k0, s);
      const unsigned long long p1 = __shfl_xor_sync(0xffffffffu, k1, s);
      const unsigned long long p2 = __shfl_xor_sync(0xffffffffu, k2, s);
      top3_insert(k0, k1, k2, p0);
      top3_insert(k0, k1, k2, p1);
      top3_insert(k0, k1, k2, p2);
    }
    if (threadIdx.x == 0) {
      const int l0 = key_index(k0), l1 = key_index(k1), l2 = key_index(k2);
      if (lead) { lead[0] = l0; lead[1] = l1; lead[2] = l2; }
      if (lead_sh) { lead_sh[0] = l0; lead_sh[1] = l1; lead_sh[2] = l2; }
    }
  }
  __syncthreads();
}

// the same for four leaders (the discrete GWO): topk holds 4 keys per part
__device__ void merge_leaders4(const unsigned long long *topk, int nparts, int32_t *lead) {
  if (threadIdx.x < 32) {
    unsigned long long k0 = 0, k1 = 0, k2 = 0, k3 = 0;
    for (int e = threadIdx.x; e < 4 * nparts; e += 32) top4_insert(k0, k1, k2, k3, topk[e]);
    for (int s = 16; s > 0; s >>= 1) {
      const unsigned long long p0 = __shfl_xor_sync(0xffffffffu, k0, s);
      const unsigned long long p1 = __shfl_xor_sync(0xffffffffu, k1, s);
      const unsigned long long p2 = __shfl_xor_sync(0xffffffffu, k2, s);
      const unsigned long long p3 = __shfl_xor_sync(0xffffffffu, k3, s);
      top4_insert(k0, k1, k2, k3, p0);
      top4_insert(k0, k1, k2, k3, p1);
      top4_insert(k0, k1, k2, k3, p2);
      top4_insert(k0, k1, k2, k3, p3);
    }
    if (threadIdx.x == 0) {
      lead[0] = key_index(k0);
      lead[1] = key_index(k1);
      lead[2] = key_index(k2);
      lead[3] = key_index(k3);
    }
  }
  __syncthreads();
}

// true in every thread of the last CTA to finish (classic fence + counter pattern)
__device__ bool last_cta(unsigned *ctr) {
  __shared__ bool is_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned prev = atomicAdd(ctr, 1u);
    is_last = (prev == gridDim.x - 1);
  }
  __syncthreads();
  if (is_last) __threadfence();
  return is_last;
}

// dynamic shared memory of k_de and k_gwo: [row + table staging (long rows)][reduction]
// The multi-wavelength kinds (MK) stage the rows only: their K phasor tables are read
// through L1, which keeps them (the rows bypass it).
//
// WIDE: 112 registers a thread instead of 80; `occupancy` picks the form.  Two 256-thread CTAs an SM
// instead of three, but no spills and more loads in flight.  Long rows are faster so (us per
// generation, graph form, 112 against 80: N = 12000, NP = 1000 123 / 131, compensated 124 / 133; 3300 x
// 1000 in teams of 128 60 / 68, compensated 62 / 70; 4000 x 500 35.4 / 37.7; 1e5 x 1024 782 / 801); the
// short rows of DUAL and the discrete GWO where it costs them no round of individuals (1320 x 5000,
// 17 rounds for 11: 102 / 92, discrete 120 / 101; discrete 1000 x 1000 in teams of 128, 2 rounds each:
// 29.6 / 34.0).  72 and 64 registers are slower throughout.  The K scans of MK take 128 (96: 3 % slower
// at K = 4 cascaded problems, 10-35 % at K = 8 SHG ones).
template <bool COMP, bool DUAL, int MK = 0, bool WIDE = true>
static __global__ void __maxnreg__(MK ? 128 : WIDE ? 112 : 80) k_de(InstDev I) {
  constexpr bool STG = !DUAL, TSS = MK != 0;
  extern __shared__ float4 dyn[];
  float4 *stg = dyn;
  Mono *sh = (Mono *)(dyn + (STG ? stg_f4_per_thread(TSS) * blockDim.x : 0));
  const int g = *I.gen;
  const PhiloxKey K = philox_schedule(I.key);
  const int32_t *sel_in = (g & 1) ? I.sel1 : I.sel0;
  int32_t *sel_out = (g & 1) ? I.sel0 : I.sel1;
  const bool four = I.combine == 2;  // the discrete GWO's four leaders
  unsigned long long k0 = 0, k1 = 0, k2 = 0, k3 = 0;
  int turn = 0;
  for (int i = blockIdx.x; i < I.NP; i += gridDim.x) {
    if (MK && i != (int)blockIdx.x) __syncthreads();  // their one reduction scratch is reused
    int slot = 0, impr = 0;
    const unsigned long long key =
        de_individual<COMP, true, TSS, DUAL, false, STG, MK>(
            I, K, I.table, g, i, de_indices(K, I.inst, (uint32_t)g, i, I.NP, I.N), sel_in, sel_out,
            MK ? sh : red_next(sh, turn), &slot, stg, false, make_uint4(0u, 0u, 0u, 0u), -1, &impr);
    if (threadIdx.x == 0) {
      if (four) top4_insert(k0, k1, k2, k3, key);
      else top3_insert(k0, k1, k2, key);
      if (I.adaptive) I.dekey[i] = slot_key(key, i, slot, impr);
    }
  }
  if (threadIdx.x == 0) {
    if (four) {
      I.topk[4 * blockIdx.x] = k0;
      I.topk[4 * blockIdx.x + 1] = k1;
      I.topk[4 * blockIdx.x + 2] = k2;
      I.topk[4 * blockIdx.x + 3] = k3;
    } else {
      I.topk[3 * blockIdx.x] = k0;
      I.topk[3 * blockIdx.x + 1] = k1;
      I.topk[3 * blockIdx.x + 2] = k2;
    }
  }
  if (last_cta(&I.ctr[0])) {
    if (four) merge_leaders4(I.topk, gridDim.x, I.lead);  // Step 3
    else merge_leaders(I.topk, gridDim.x, I.lead, nullptr);
    if (I.adaptive) adaptive_F_block(I, I.dekey, g);     // Step 6: the next F
    if (threadIdx.x == 0) I.ctr[0] = 0u;
  }
}

template <bool COMP, bool DUAL, int MK = 0, bool WIDE = true>
static __global__ void __maxnreg__(MK ? 128 : WIDE ? 112 : 80) k_gwo(InstDev I) {
  constexpr bool STG = !DUAL, TSS = MK != 0;
  extern __shared__ float4 dyn[];
  float4 *stg = dyn;
  Mono *sh = (Mono *)(dyn + (STG ? stg_f4_per_thread(TSS) * blockDim.x : 0));
  const int g = *I.gen;
  const PhiloxKey K = philox_schedule(I.key);
  int32_t *sel = (g & 1) ? I.sel0 : I.sel1;
  const int la = I.lead[0], lb = I.lead[1], ld = I.lead[2];
  const float a = a_of(I, g);
  int turn = 0;
  for (int i = blockIdx.x; i < I.NP; i += gridDim.x) {
    if (i == la || i == lb || i == ld) continue;  // the leaders do not move
    if (MK) __syncthreads();  // their one reduction scratch is reused
    gwo_individual<COMP, true, TSS, DUAL, false, false, STG, MK>(
        I, K, I.table, g, a, i, sel, la, lb, ld, MK ? sh : red_next(sh, turn), nullptr, make_float4(0.f, 0.f, 0.f, 0.f),
        make_float4(0.f, 0.f, 0.f, 0.f), nullptr, stg);
  }
  if (I.trace && blockIdx.x == 0 && threadIdx.x < 3) {
    const int l = threadIdx.x == 0 ? la : (threadIdx.x == 1 ? lb : ld);
    I.trace[(size_t)I.NP * (2 + 2 * (size_t)g) + l] = __int_as_float(0x7fc00000);
  }
  if (last_cta(&I.ctr[1])) {
    if (threadIdx.x == 0) {
      *I.gen = g + 1;  // Step 6/7: next generation (a is derived from g)
      I.ctr[1] = 0u;
    }
  }
}

// ------------------------------- the multi-wavelength kinds, tables in shared memory
// When their K tables fit, the multi-wavelength kinds run several teams of T threads
// per CTA (threads [team T, team T + T) are the team of one individual, with its own
// named barrier, or none for one-warp teams) so that one copy of the K tables in
// shared memory serves every team
// on the SM: read through L1, the tables of three N = 3000 problems (147 KB) did not
// stay there.  The cascaded kind keeps (p1, p2) per domain, the SHG kind p1 only.
// Dynamic shared memory: [K tables][row staging][reduction scratch of every team].
// Teams take individuals from a counter (ctr[2] in DE, ctr[3] in GWO, reset by the
// phase's last CTA), so that every SM ends within about one individual of the others
// (a fixed deal of 5000 individuals to 152 x 8 teams leaves the fifth round 11 % full).
// Which team evaluates an individual does not change any result.
__device__ __forceinline__ int mt_next(const InstDev &I, unsigned *ctr, int &cur) {
  __shared__ int next_sh[16];
  const int team = (int)threadIdx.x / I.T;
  if (team_thread(I) == 0) next_sh[team] = cur;
  team_sync(I);  // also: the previous individual's reduction scratch is free again
  const int i = next_sh[team];
  // the one after, requested while this one is evaluated
  if (i < I.NP && team_thread(I) == 0) cur = (int)atomicAdd(ctr, 1u);
  return i;
}

template <int MK>
__host__ __device__ constexpr size_t mt_entry_bytes() {
  return MK == OBJ_MULTI_SHG ? sizeof(float2) : sizeof(float4);
}
template <int MK>
__device__ void mt_load_tables(const InstDev &I, void *smt) {
#pragma unroll
  for (int k = 0; k < MultiAcc<MK>::KMAX; ++k) {
    if (k < I.K) {
      const float4 *src = I.mtab[k];
      for (int j = threadIdx.x; j < I.Npad; j += blockDim.x) {
        const float4 p = __ldg(src + j);
        const size_t e = (size_t)k * I.Npad + j;
        if (MK == OBJ_MULTI_SHG) ((float2 *)smt)[e] = make_float2(p.x, p.y);
        else ((float4 *)smt)[e] = p;
      }
    }
  }
  __syncthreads();
}
template <int MK>
__device__ __forceinline__ void mt_layout(const InstDev &I, void *&smt, float4 *&stg, Mono *&sh) {
  extern __shared__ float4 dyn[];
  smt = dyn;
  stg = (float4 *)((char *)dyn + (size_t)I.K * I.Npad * mt_entry_bytes<MK>());
  sh = (Mono *)(stg + stg_f4_per_thread(true) * blockDim.x);
}

template <int MK>
static __global__ void __launch_bounds__(512, 1) k_de_mt(InstDev I) {
  // launched as a programmatic dependent of the phase before: the next phase's CTAs may
  // start as this grid's retire, and every CTA loads its tables (fixed per problem)
  // before it waits for the phase before to complete and its writes to be visible
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  void *smt;
  float4 *stg;
  Mono *sh;
  mt_layout<MK>(I, smt, stg, sh);
  mt_load_tables<MK>(I, smt);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int g = *I.gen;
  const PhiloxKey K = philox_schedule(I.key);
  const int32_t *sel_in = (g & 1) ? I.sel1 : I.sel0;
  int32_t *sel_out = (g & 1) ? I.sel0 : I.sel1;
  const int nteams = (int)blockDim.x / I.T, team = (int)threadIdx.x / I.T, t = team_thread(I);
  unsigned long long k0 = 0, k1 = 0, k2 = 0;
  int cur = t == 0 ? (int)atomicAdd(&I.ctr[2], 1u) : 0;
  for (;;) {
    const int i = mt_next(I, &I.ctr[2], cur);
    if (i >= I.NP) break;
    int slot = 0, impr = 0;
    const unsigned long long key = de_individual<false, true, true, false, false, true, MK>(
        I, K, I.table, g, i, de_indices(K, I.inst, (uint32_t)g, i, I.NP, I.N), sel_in, sel_out,
        sh, &slot, stg, false, make_uint4(0u, 0u, 0u, 0u), -1, &impr, smt);
    if (t == 0) {
      top3_insert(k0, k1, k2, key);
      if (I.adaptive) I.dekey[i] = slot_key(key, i, slot, impr);
    }
  }
  // the teams' top three, merged by thread 0 (team 0's first thread)
  __shared__ unsigned long long tk[3 * 16];
  if (t == 0) {
    tk[3 * team] = k0;
    tk[3 * team + 1] = k1;
    tk[3 * team + 2] = k2;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int m = 1; m < nteams; ++m)
      for (int e = 0; e < 3; ++e) top3_insert(k0, k1, k2, tk[3 * m + e]);
    I.topk[3 * blockIdx.x] = k0;
    I.topk[3 * blockIdx.x + 1] = k1;
    I.topk[3 * blockIdx.x + 2] = k2;
  }
  if (last_cta(&I.ctr[0])) {
    merge_leaders(I.topk, gridDim.x, I.lead, nullptr);  // Step 3
    if (I.adaptive) adaptive_F_block(I, I.dekey, g);     // Step 6: the next F
    if (threadIdx.x == 0) {
      I.ctr[0] = 0u;
      I.ctr[2] = 0u;
    }
  }
}

template <int MK>
static __global__ void __launch_bounds__(512, 1) k_gwo_mt(InstDev I) {
  // launched as a programmatic dependent of the phase before: the next phase's CTAs may
  // start as this grid's retire, and every CTA loads its tables (fixed per problem)
  // before it waits for the phase before to complete and its writes to be visible
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  void *smt;
  float4 *stg;
  Mono *sh;
  mt_layout<MK>(I, smt, stg, sh);
  mt_load_tables<MK>(I, smt);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int g = *I.gen;
  const PhiloxKey K = philox_schedule(I.key);
  int32_t *sel = (g & 1) ? I.sel0 : I.sel1;
  const int la = I.lead[0], lb = I.lead[1], ld = I.lead[2];
  const float a = a_of(I, g);
  int cur = team_thread(I) == 0 ? (int)atomicAdd(&I.ctr[3], 1u) : 0;
  for (;;) {
    const int i = mt_next(I, &I.ctr[3], cur);
    if (i >= I.NP) break;
    if (i == la || i == lb || i == ld) continue;  // the leaders do not move
    gwo_individual<false, true, true, false, false, false, true, MK>(
        I, K, I.table, g, a, i, sel, la, lb, ld, sh, nullptr, make_float4(0.f, 0.f, 0.f, 0.f),
        make_float4(0.f, 0.f, 0.f, 0.f), nullptr, stg, -1, nullptr, smt);
  }
  if (I.trace && blockIdx.x == 0 && threadIdx.x < 3) {
    const int l = threadIdx.x == 0 ? la : (threadIdx.x == 1 ? lb : ld);
    I.trace[(size_t)I.NP * (2 + 2 * (size_t)g) + l] = __int_as_float(0x7fc00000);
  }
  if (last_cta(&I.ctr[1])) {
    if (threadIdx.x == 0) {
      *I.gen = g + 1;  // Step 6/7: next generation (a is derived from g)
      I.ctr[1] = 0u;
      I.ctr[3] = 0u;
    }
  }
}

// Steps 4-5 with the four-leader discrete GWO (launches form)
template <bool COMP, bool WIDE>
static __global__ void __maxnreg__(WIDE ? 112 : 80) k_gwo_disc(InstDev I) {
  extern __shared__ float4 dyn[];
  Mono *sh = (Mono *)dyn;
  const int g = *I.gen;
  const PhiloxKey K = philox_schedule(I.key);
  int32_t *sel = (g & 1) ? I.sel0 : I.sel1;
  // the leaders do not move in this phase
  const int la = I.lead[0], lb = I.lead[1], lc = I.lead[2], ld = I.lead[3];
  const float *L0 = row_ptr(I, la, sel[la]), *L1 = row_ptr(I, lb, sel[lb]);
  const float *L2 = row_ptr(I, lc, sel[lc]), *L3 = row_ptr(I, ld, sel[ld]);
  int turn = 0;
  for (int i = blockIdx.x; i < I.NP; i += gridDim.x) {
    if (i == la || i == lb || i == lc || i == ld) continue;
    gwo_discrete_individual<COMP>(I, K, g, i, sel, L0, L1, L2, L3, red_next(sh, turn));
  }
  if (I.trace && blockIdx.x == 0 && threadIdx.x < 4)
    I.trace[(size_t)I.NP * (2 + 2 * (size_t)g) + I.lead[threadIdx.x]] = __int_as_float(0x7fc00000);
  if (last_cta(&I.ctr[1])) {
    if (threadIdx.x == 0) {
      *I.gen = g + 1;
      I.ctr[1] = 0u;
    }
  }
}

// ------------------------------------------------------ persistent kernel
// Step 3 of the persistent form, after the grid barrier that follows DE: the top
// three of the DE survivor keys of all individuals; every thread returns after the
// CTA barrier with lead_sh and the leaders' current slots (slot_sh) set.  Every thread reads its
// share of the keys, every warp takes its top three with redux.sync and warp 0 those of the warps.
// (Warp 0 reading all keys and merging lane triples by shuffles: 7.89 against 7.31 us per
// generation at N = 1000, NP = 256; at N = 2500 9.8 / 9.1 with 152 individuals, 26.3 / 25.1 with 900, 126
// / 122 with 5000; at N = 1e5 and 1024 individuals 677 / 675.)  Teams of one or two warps on long rows
// (NARROW) take that form: many of them search at once on an SM, and it has fewer instructions (N =
// 3300, NP = 1000 58.8 / 64.4 in teams of 32, 43.8 / 45.9 of 64, 38.0 / 37.4 of 128; NP = 5000 249 / 286 in
// teams of 32, 172 / 186 of 64).  The keys are
// written in the DE phase only, so a CTA that is still choosing leaders never sees a fitness
// already changed by another CTA's GWO selection.
template <bool NARROW>
__device__ void leaders_from_keys(const unsigned long long *keys, int NP, int32_t *lead,
                                  int32_t *lead_sh, int32_t *slot_sh) {
  if (NARROW && blockDim.x <= 64) {
    if (threadIdx.x < 32) {
      unsigned long long k0 = 0, k1 = 0, k2 = 0;
      for (int i = threadIdx.x; i < NP; i += 32) top3_insert(k0, k1, k2, keys[i]);
      for (int s = 16; s > 0; s >>= 1) {
        const unsigned long long p0 = __shfl_xor_sync(0xffffffffu, k0, s);
        const unsigned long long p1 = __shfl_xor_sync(0xffffffffu, k1, s);
        const unsigned long long p2 = __shfl_xor_sync(0xffffffffu, k2, s);
        top3_insert(k0, k1, k2, p0);
        top3_insert(k0, k1, k2, p1);
        top3_insert(k0, k1, k2, p2);
      }
      if (threadIdx.x == 0) {
        lead_sh[0] = slot_key_index(k0);
        lead_sh[1] = slot_key_index(k1);
        lead_sh[2] = slot_key_index(k2);
        slot_sh[0] = (int32_t)(k0 & 1u);
        slot_sh[1] = (int32_t)(k1 & 1u);
        slot_sh[2] = (int32_t)(k2 & 1u);
        if (lead) { lead[0] = lead_sh[0]; lead[1] = lead_sh[1]; lead[2] = lead_sh[2]; }
      }
    }
    __syncthreads();
    return;
  }
  __shared__ unsigned long long wtop[3 * 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  unsigned long long k0 = 0, k1 = 0, k2 = 0;
#pragma unroll 4
  for (int i = threadIdx.x; i < NP; i += blockDim.x) top3_insert(k0, k1, k2, keys[i]);
  warp_top3(k0, k1, k2);
  if (lane == 0) {
    wtop[3 * warp] = k0;
    wtop[3 * warp + 1] = k1;
    wtop[3 * warp + 2] = k2;
  }
  __syncthreads();
  if (warp == 0) {
    k0 = k1 = k2 = 0ull;
    if (lane < nw) {
      k0 = wtop[3 * lane];
      k1 = wtop[3 * lane + 1];
      k2 = wtop[3 * lane + 2];
    }
    warp_top3(k0, k1, k2);
    if (lane == 0) {
      lead_sh[0] = slot_key_index(k0);
      lead_sh[1] = slot_key_index(k1);
      lead_sh[2] = slot_key_index(k2);
      slot_sh[0] = (int32_t)(k0 & 1u);
      slot_sh[1] = (int32_t)(k1 & 1u);
      slot_sh[2] = (int32_t)(k2 & 1u);
      if (lead) { lead[0] = lead_sh[0]; lead[1] = lead_sh[1]; lead[2] = lead_sh[2]; }
    }
  }
  __syncthreads();
}

// All generations [*gen, g_end) in one cooperative launch; every CTA keeps the
// same individuals (i = blockIdx.x + k gridDim.x), the phasor table sits in
// shared memory when it fits (TS).  Two grid barriers per generation: after DE
// (the leaders need every DE survivor) and after GWO (the next donors are any
// individuals).  With one individual per CTA and 4 domains per thread, the GWO
// random words are drawn between the arrival at the first barrier and the wait.
// MAXT: the largest team the variant runs (256: two CTAs per SM; 512: one)
template <bool COMP, bool TS, bool DUAL, int MAXT = 256>
static __global__ void __launch_bounds__(MAXT, MAXT > 256 ? 1 : 2)
    k_persist(InstDev I, int g_end, Barrier bar) {
  // dynamic shared memory: [row staging (long rows)][phasor table (TS)][reduction]
  constexpr bool STG = !DUAL;
  extern __shared__ float4 dyn[];
  __shared__ int32_t lead_sh[3], lslot_sh[3], own_slot_sh;
  float4 *stg = dyn;
  float4 *tab = dyn + (STG ? stg_f4_per_thread(TS) * blockDim.x : 0);
  Mono *sh = (Mono *)(tab + (TS ? I.Npad : 0));
  if (TS) {
    for (int e = threadIdx.x; e < I.Npad; e += blockDim.x) tab[e] = __ldg(I.table + e);
    __syncthreads();
  }
  const float4 *tbl = TS ? (const float4 *)tab : I.table;
  const PhiloxKey K = philox_schedule(I.key);
  const bool pre = DUAL && (I.c == 4) && (gridDim.x == (unsigned)I.NP);
  unsigned target = 0;
  int turn = 0;  // see red_next
  int g = *I.gen;
  // pre (one individual per CTA, one group of 4 domains per thread): the DE donors
  // and the crossover word of a generation depend on (g, i) only and are drawn
  // while the previous generation's last barrier completes
  const uint32_t jg0 = (uint32_t)((threadIdx.x * I.c) >> 2);
  // pre: own_slot_sh carries the individual's current slot from one phase to the next
  // (set by thread 0 after its selection), so its selector is not read back; the first
  // DE phase of a launch reads it
  bool own_known = false;
  int4 r_pre = make_int4(0, 0, 0, 0);
  uint4 wcr_pre = make_uint4(0u, 0u, 0u, 0u);
  if (pre && g < g_end) {
    r_pre = de_indices(K, I.inst, (uint32_t)g, blockIdx.x, I.NP, I.N);
    wcr_pre = rng4(K, I.inst, TAG_CR, (uint32_t)g, (uint32_t)blockIdx.x, jg0);
  }
  for (; g < g_end; ++g) {
    const int32_t *sel_in = (g & 1) ? I.sel1 : I.sel0;
    int32_t *sel_out = (g & 1) ? I.sel0 : I.sel1;
    Donors donors;
    for (int i = blockIdx.x; i < I.NP; i += gridDim.x) {
      const int4 r = pre ? r_pre : donors.next(I, K, g, i, gridDim.x);
      int slot = 0, impr = 0;
      const unsigned long long key =
          de_individual<COMP, false, TS, DUAL, false, STG>(I, K, tbl, g, i, r, sel_in, sel_out,
                                                            red_next(sh, turn), &slot, stg, pre, wcr_pre,
                                                            own_known ? own_slot_sh : -1, &impr);
      // ordered before the barrier's release
      if (threadIdx.x == 0) {
        I.dekey[i] = slot_key(key, i, slot, impr);
        own_slot_sh = slot;  // read after the barrier's CTA synchronisation
      }
    }
    grid_arrive(bar, target);
    const float a = a_of(I, g);
    uint4 wpre[3];
    if (pre) {
      const uint32_t jg = (uint32_t)((threadIdx.x * I.c) >> 2);
#pragma unroll
      for (int k = 0; k < 3; ++k)
        wpre[k] = rng4(K, I.inst, TAG_GWO + k, (uint32_t)g, (uint32_t)blockIdx.x, jg);
    }
    if (!grid_wait(bar, target)) return;
    // the own row (its current slot, known from this CTA's own selection) is
    // requested before the leaders are known, so that its latency overlaps the
    // leader search
    float4 own0 = make_float4(0.f, 0.f, 0.f, 0.f), own1 = own0;
    if (pre) {
      const float *r0 = I.pop + ((size_t)2 * blockIdx.x + own_slot_sh) * I.Npad +
                        (size_t)threadIdx.x * 4;
      own0 = *(const float4 *)r0;
      own1 = own0;
    }
    // every CTA finds the leaders itself (Sec. 3.2 Step 3) from the DE keys
    leaders_from_keys<!DUAL>(I.dekey, I.NP, blockIdx.x == 0 ? I.lead : nullptr, lead_sh, lslot_sh);
    const int la = lead_sh[0], lb = lead_sh[1], ld = lead_sh[2];
    // Step 6, the adaptive F of the next generation: by the CTA of the alpha leader (which
    // moves no wolf) when every CTA holds one individual, else by the last CTA, before its
    // own wolves (it holds one individual fewer than the first ones unless the deal is even).
    // The survivor keys stay unchanged until the next DE phase, which the barrier below
    // keeps after this.
    if (I.adaptive &&
        (int)blockIdx.x == (gridDim.x == (unsigned)I.NP ? la : (int)gridDim.x - 1))
      adaptive_F_block(I, I.dekey, g);
    for (int i = blockIdx.x; i < I.NP; i += gridDim.x) {
      if (i == la || i == lb || i == ld) continue;
      if (pre) {
        int gslot = 0;
        gwo_individual<COMP, false, TS, DUAL, false, true>(I, K, tbl, g, a, i, sel_out, la, lb, ld,
                                                           red_next(sh, turn), wpre, own0, own1, lslot_sh,
                                                           nullptr, own_slot_sh, &gslot);
        // read by every thread after the next barrier's CTA synchronisation
        if (threadIdx.x == 0) own_slot_sh = gslot;
      }
      else
        gwo_individual<COMP, false, TS, DUAL, false, false, STG>(
            I, K, tbl, g, a, i, sel_out, la, lb, ld, red_next(sh, turn), nullptr,
            make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f), lslot_sh, stg);
    }
    if (I.trace && blockIdx.x == 0 && threadIdx.x < 3) {
      const int l = threadIdx.x == 0 ? la : (threadIdx.x == 1 ? lb : ld);
      I.trace[(size_t)I.NP * (2 + 2 * (size_t)g) + l] = __int_as_float(0x7fc00000);
    }
    // the next DE phase reads any individual: every CTA must have finished GWO
    grid_arrive(bar, target);
    own_known = pre;
    if (pre && g + 1 < g_end) {
      r_pre = de_indices(K, I.inst, (uint32_t)(g + 1), blockIdx.x, I.NP, I.N);
      wcr_pre = rng4(K, I.inst, TAG_CR, (uint32_t)(g + 1), (uint32_t)blockIdx.x, jg0);
    }
    if (!grid_wait(bar, target)) return;
  }
  // every CTA read the start generation before its first barrier; later kernels
  // see the new value after this launch completes
  if (blockIdx.x == 0 && threadIdx.x == 0) *I.gen = g_end;
}

// ------------------------------------------------------------ batched form
// Many independent instances in one launch.  Each thread-block cluster (1, 2, 4
// or 8 CTAs on as many SMs) takes whole instances from a queue (largest first)
// and runs them for the requested generations: every warp is the team of one
// individual (instances use T = 32), the individuals of an instance are dealt to
// the warps of all CTAs of the cluster, and the two dependencies of a generation
// are cluster barriers (release/acquire at cluster scope, which also orders the
// population writes in global memory).  Each CTA's leader candidates are read by
// the others through distributed shared memory.  No cluster waits for another,
// so no co-residency beyond the cluster's own is needed.  Splitting an instance
// over a cluster keeps the largest instance from setting the batch's makespan.
__device__ __forceinline__ unsigned cluster_rank() {
  return cooperative_groups::this_cluster().block_rank();
}
__device__ __forceinline__ unsigned cluster_size() {
  return cooperative_groups::this_cluster().num_blocks();
}
// every thread of every CTA of the cluster (CL) or of the CTA; writes before it
// (shared and global) are visible to every thread of the cluster after it
template <bool CL>
__device__ __forceinline__ void cluster_sync_all() {
  if (CL) cooperative_groups::this_cluster().sync();
  else __syncthreads();
}
// the word at `p` in the shared memory of CTA `rank` of this cluster
__device__ __forceinline__ unsigned long long ld_dsmem_u64(unsigned long long *p, unsigned rank) {
  return *cooperative_groups::this_cluster().map_shared_rank(p, rank);
}

// one instance, generations [*gen, min(*gen + gens, G)), by the whole CTA
// CL: the instance is shared by the CTAs of a cluster (more than one)
template <bool COMP, bool TS, bool CL>
__device__ void batch_instance(const InstDev &I, const PhiloxKey &K, int gens, float4 *dyn, unsigned long long *wk,
                               unsigned long long *ck, int32_t *lead_sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const unsigned crank = CL ? cluster_rank() : 0u, csize = CL ? cluster_size() : 1u;
  const int gw = (int)crank * nw + warp, gstride = (int)csize * nw;  // warp in the cluster
  // dynamic shared memory: [row staging][phasor table (TS)]
  float4 *stg = dyn, *tab = dyn + stg_f4_per_thread(TS) * blockDim.x;
  if (TS) {
    for (int e = threadIdx.x; e < I.Npad; e += blockDim.x) tab[e] = __ldg(I.table + e);
  }
  const float4 *tbl = TS ? (const float4 *)tab : I.table;
  int g = *I.gen;
  const int g_end = min(g + gens, I.G);
  __syncthreads();
  for (; g < g_end; ++g) {
    const int32_t *sel_in = (g & 1) ? I.sel1 : I.sel0;
    int32_t *sel_out = (g & 1) ? I.sel0 : I.sel1;
    // each warp's running top three lives in shared memory (lane 0), which keeps
    // six registers free across the DE loop
    if (lane == 0) wk[3 * warp] = wk[3 * warp + 1] = wk[3 * warp + 2] = 0ull;
    for (int i = gw; i < I.NP; i += gstride) {
      int impr = 0;
      const unsigned long long key =
          de_individual<COMP, false, TS, false, true, true>(
              I, K, tbl, g, i, de_indices(K, I.inst, (uint32_t)g, i, I.NP, I.N), sel_in, sel_out,
              nullptr, nullptr, stg, false, make_uint4(0u, 0u, 0u, 0u), -1, &impr);
      if (lane == 0 && I.adaptive) I.dekey[i] = slot_key(key, i, 0, impr);
      if (lane == 0) {
        unsigned long long a = wk[3 * warp], b = wk[3 * warp + 1], c = wk[3 * warp + 2];
        top3_insert(a, b, c, key);
        wk[3 * warp] = a;
        wk[3 * warp + 1] = b;
        wk[3 * warp + 2] = c;
      }
    }
    __syncthreads();
    unsigned long long k0 = wk[0], k1 = wk[1], k2 = wk[2];
    if (threadIdx.x == 0) {  // this CTA's candidates
      for (int w = 1; w < nw; ++w) {
        top3_insert(k0, k1, k2, wk[3 * w]);
        top3_insert(k0, k1, k2, wk[3 * w + 1]);
        top3_insert(k0, k1, k2, wk[3 * w + 2]);
      }
      ck[0] = k0;
      ck[1] = k1;
      ck[2] = k2;
    }
    // every DE survivor of the instance and every CTA's candidates are now visible
    cluster_sync_all<CL>();
    if (threadIdx.x == 0) {  // Step 3: leaders of this instance (the same in every CTA)
      for (unsigned r = 0; CL && r < csize; ++r) {
        if (r == crank) continue;
        top3_insert(k0, k1, k2, ld_dsmem_u64(ck, r));
        top3_insert(k0, k1, k2, ld_dsmem_u64(ck + 1, r));
        top3_insert(k0, k1, k2, ld_dsmem_u64(ck + 2, r));
      }
      lead_sh[0] = key_index(k0);
      lead_sh[1] = key_index(k1);
      lead_sh[2] = key_index(k2);
      if (crank == 0) {
        I.lead[0] = lead_sh[0];
        I.lead[1] = lead_sh[1];
        I.lead[2] = lead_sh[2];
      }
    }
    __syncthreads();
    // Step 6: the adaptive F of the next generation, by the cluster's first CTA; the
    // cluster barrier after the GWO phase orders it before the next DE phase
    if (I.adaptive && crank == 0) adaptive_F_block(I, I.dekey, g);
    const int la = lead_sh[0], lb = lead_sh[1], ld = lead_sh[2];
    const float a = a_of(I, g);
    for (int i = gw; i < I.NP; i += gstride) {
      if (i == la || i == lb || i == ld) continue;
      gwo_individual<COMP, false, TS, false, true, false, true>(
          I, K, tbl, g, a, i, sel_out, la, lb, ld, nullptr, nullptr, make_float4(0.f, 0.f, 0.f, 0.f),
          make_float4(0.f, 0.f, 0.f, 0.f), nullptr, stg);
    }
    if (I.trace && crank == 0 && threadIdx.x < 3) {
      const int l = threadIdx.x == 0 ? la : (threadIdx.x == 1 ? lb : ld);
      I.trace[(size_t)I.NP * (2 + 2 * (size_t)g) + l] = __int_as_float(0x7fc00000);
    }
    // the next DE reads any individual, and ck is rewritten only after every CTA read it
    cluster_sync_all<CL>();
  }
  if (crank == 0 && threadIdx.x == 0) *I.gen = g_end;
}

// SAME: every instance has the round keys `key`, which as a kernel parameter are constant
// operands of the rounds' xors and take no registers (the FMA-heavy pipe and the registers bound
// this kernel: 512 instances 3.14 -> 3.04 ms per generation); else each instance's own.  The
// single-instance kernels build them from the parameter's seed, which measured faster there
// (N = 3300, NP = 5000: 168.8 us per generation against 170.8 with constant operands).
template <bool TS, bool CL, bool SAME>
static __global__ void __launch_bounds__(BATCH_WARPS * 32, 1)
    k_batch(const InstDev *__restrict__ insts, const int32_t *__restrict__ order, int n_inst,
            unsigned *queue, int gens, const __grid_constant__ PhiloxKey key) {
  extern __shared__ float4 dyn[];
  __shared__ unsigned long long wk[3 * BATCH_WARPS];
  __shared__ unsigned long long ck[3];  // this CTA's leader candidates, read by the cluster
  __shared__ int32_t lead_sh[3];
  __shared__ unsigned long long job_sh;
  for (;;) {
    int job;
    {
      const unsigned crank = CL ? cluster_rank() : 0u;
      if (crank == 0 && threadIdx.x == 0) job_sh = (unsigned long long)atomicAdd(queue, 1u);
      cluster_sync_all<CL>();
      job = (int)(crank == 0 ? job_sh : ld_dsmem_u64(&job_sh, 0));
      cluster_sync_all<CL>();  // every CTA has the job before rank 0 takes the next one
    }
    if (job >= n_inst) break;
    const InstDev I = insts[order[job]];
    const PhiloxKey own = philox_schedule(I.key);  // unused, and so not computed, if SAME
    const PhiloxKey &K = SAME ? key : own;
    if (I.compensated) batch_instance<true, TS, CL>(I, K, gens, dyn, wk, ck, lead_sh);
    else batch_instance<false, TS, CL>(I, K, gens, dyn, wk, ck, lead_sh);
  }
}

// ------------------------------------------------ outputs: best, FP64, layout
__device__ __forceinline__ size_t perm_pos(const InstDev &I, int j) {
  const int t = j / I.c, e = j - t * I.c;
  return ((size_t)(e >> 2) * I.T + t) * 4 + (e & 3);
}

struct Mono64 {
  double2 A, B, C;
};
__device__ __forceinline__ Mono64 m64_combine(const Mono64 &L, const Mono64 &R) {
  Mono64 o;
  o.A = make_double2(L.A.x + R.A.x, L.A.y + R.A.y);
  o.B = make_double2(L.B.x + R.B.x, L.B.y + R.B.y);
  o.C = make_double2(L.C.x + R.C.x + (R.A.x * L.B.x - R.A.y * L.B.y),
                     L.C.y + R.C.y + (R.A.x * L.B.y + R.A.y * L.B.x));
  return o;
}
__device__ __forceinline__ double2 shfl_down2(double2 v, int s) {
  return make_double2(__shfl_down_sync(0xffffffffu, v.x, s), __shfl_down_sync(0xffffffffu, v.y, s));
}
// ordered reduction over the 32 lanes of a warp, valid in lane 0
__device__ __forceinline__ Mono64 m64_warp_reduce(Mono64 m) {
#pragma unroll
  for (int s = 1; s < 32; s <<= 1) {
    Mono64 r;
    r.A = shfl_down2(m.A, s);
    r.B = shfl_down2(m.B, s);
    r.C = shfl_down2(m.C, s);
    m = m64_combine(m, r);  // lanes that are no multiple of 2s hold values nobody reads
  }
  return m;
}
__device__ __forceinline__ double2 cmul64(const double2 &a, const double2 &b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// e^{-i kappa q}, q = 1, 2, 3, of both mismatches (host)
struct BestRot {
  double2 r1[3], r2[3];
};

// The best individual (A11): its index, fitness and genes, and the partial sums of its FP64
// re-evaluation (closed form, FP64 phasors).  Bound by the FP64 unit, which retires about two
// lanes a cycle and SM on this GPU: one CTA doing all of it with two sincos a domain took
// 109 us at N = 1000 and 2.08 ms at N = 1e5.  So the domains are spread over the whole GPU, a
// warp per 128 domains in a CTA of its own, every CTA finding the best individual itself (a
// few KB of fitness from L2, no grid-wide wait), and a lane takes 4 neighbouring domains with
// one sincos per mismatch, the other three phasors by rotation: 118 -> 15 us a call at N = 1000
// and NP = 256, 171 -> 17 at 3300 and 5000, 2.16 ms -> 25 us at 1e5 and 1024.
constexpr int BEST_THREADS = 128, BEST_DOMAINS = 128;
static __global__ void __launch_bounds__(BEST_THREADS)
    k_best(InstDev I, BestRot rot, float *genes_out, float *fit_out, int32_t *index_out, int scan) {
  __shared__ unsigned long long shk[BEST_THREADS / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long key = 0;
#pragma unroll 8
  for (int i = threadIdx.x; i < I.NP; i += BEST_THREADS) {
    const unsigned long long k = sel_key(I.minimize != 0, I.fit[i], i);
    key = k > key ? k : key;
  }
  const uint32_t hi = (uint32_t)(key >> 32), mhi = __reduce_max_sync(0xffffffffu, hi);
  const uint32_t mlo = __reduce_max_sync(0xffffffffu, hi == mhi ? (uint32_t)key : 0u);
  if (lane == 0) shk[warp] = ((unsigned long long)mhi << 32) | mlo;
  __syncthreads();
  key = shk[0];
#pragma unroll
  for (int w = 1; w < BEST_THREADS / 32; ++w) key = shk[w] > key ? shk[w] : key;
  const int i = key_index(key);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (index_out) *index_out = i;
    if (fit_out) *fit_out = I.fit[i];
  }
  const int32_t *sel = (*I.gen & 1) ? I.sel1 : I.sel0;
  const float *row = row_ptr(I, i, sel[i]);
  const int b0 = blockIdx.x * BEST_DOMAINS;
  if (genes_out && b0 + (int)threadIdx.x < I.N)
    genes_out[b0 + threadIdx.x] = row[perm_pos(I, b0 + threadIdx.x)];
  if (!scan || warp != 0) return;
  Mono64 m;
  m.A = m.B = m.C = make_double2(0.0, 0.0);
  const int m0 = b0 + 4 * lane;
  if (m0 < I.N) {
    const float4 x = *(const float4 *)(row + perm_pos(I, m0));  // a group of 4 is contiguous
    const float xs[4] = {x.x, x.y, x.z, x.w};
    double sn, cs;
    sincos(reduce_2pi((double)m0 * I.kappa1), &sn, &cs);
    const double2 p1 = make_double2(cs, -sn);
    sincos(reduce_2pi((double)m0 * I.kappa2), &sn, &cs);
    const double2 p2 = make_double2(cs, -sn);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (m0 + q < I.N) {
        const double d = xs[q] < 0.f ? -1.0 : 1.0;
        const double2 c1 = q ? cmul64(p1, rot.r1[q ? q - 1 : 0]) : p1;
        const double2 c2 = q ? cmul64(p2, rot.r2[q ? q - 1 : 0]) : p2;
        const double2 a = make_double2(d * c2.x, d * c2.y);
        m.C.x += a.x * m.B.x - a.y * m.B.y;
        m.C.y += a.x * m.B.y + a.y * m.B.x;
        m.A.x += a.x;
        m.A.y += a.y;
        m.B.x += d * c1.x;
        m.B.y += d * c1.y;
      }
    }
  }
  m = m64_warp_reduce(m);
  if (lane == 0) {
    I.rpart[3 * blockIdx.x] = m.A;
    I.rpart[3 * blockIdx.x + 1] = m.B;
    I.rpart[3 * blockIdx.x + 2] = m.C;
  }
}

// the partials in index order, and the field: one CTA, a programmatic dependent of k_best
static __global__ void __launch_bounds__(BEST_THREADS)
    k_best_close(InstDev I, int nparts, double *d64_out) {
  __shared__ Mono64 sh[BEST_THREADS / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int per = (nparts + BEST_THREADS - 1) / BEST_THREADS;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  Mono64 m;
  m.A = m.B = m.C = make_double2(0.0, 0.0);
  if (warp * 32 * per < nparts) {  // the warp has partials
    const int s0 = min(nparts, (int)threadIdx.x * per), s1 = min(nparts, s0 + per);
    for (int s = s0; s < s1; ++s) {
      Mono64 r;
      r.A = I.rpart[3 * s];
      r.B = I.rpart[3 * s + 1];
      r.C = I.rpart[3 * s + 2];
      m = m64_combine(m, r);
    }
    m = m64_warp_reduce(m);
  }
  if (lane == 0) sh[warp] = m;
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int w = 1; w < BEST_THREADS / 32 && w * 32 * per < nparts; ++w) m = m64_combine(m, sh[w]);
  double re, im;
  if (I.obj == OBJ_SHG || I.obj == OBJ_MULTI_SHG) {  // SHG field: phi(kappa1) sum d p1
    const double2 ph = I.konst64[3];
    re = ph.x * m.B.x - ph.y * m.B.y;
    im = ph.x * m.B.y + ph.y * m.B.x;
  } else {  // cascaded d_eff
    const double2 p12 = I.konst64[0], cd = I.konst64[1];
    re = p12.x * m.C.x - p12.y * m.C.y + cd.x;
    im = p12.x * m.C.y + p12.y * m.C.x + cd.y;
  }
  d64_out[0] = re;
  d64_out[1] = im;
}

// Rows back to natural order.  A row is a [c / 4][T] matrix of float4 groups and its natural
// order the transposed one, so a warp takes a tile of 32 threads' groups x 8, reads it by 512 B
// along T, and writes runs of up to 128 B along c / 4 through shared memory (16 bytes a lane
// where the output rows allow it).  A gene at a time, with a division and reads 16 bytes apart,
// ran at 2.7-4.3 TB/s of read + write (66 MB of N = 3300 rows in 50 us; a call 54 -> 31
// us, of N = 1e5 and NP = 1024 182 -> 135).  The fitness and field outputs are copied by the same
// launch.
constexpr int POP_THREADS = 256, POP_KB = 8;
static __global__ void __launch_bounds__(POP_THREADS)
    k_population(InstDev I, float *__restrict__ out, int64_t ld, float *__restrict__ fit_out,
                 float2 *__restrict__ d_out) {
  __shared__ float4 tile[POP_THREADS / 32][POP_KB * 33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i = blockIdx.x * POP_THREADS + threadIdx.x; i < I.NP; i += gridDim.x * POP_THREADS) {
    if (fit_out) fit_out[i] = I.fit[i];
    if (d_out) d_out[i] = I.dval[i];
  }
  if (!out) return;
  const int32_t *sel = (*I.gen & 1) ? I.sel1 : I.sel0;
  const int n4 = I.c >> 2, nk = (n4 + POP_KB - 1) / POP_KB;
  const uint32_t tiles = (uint32_t)(I.T >> 5) * nk, total = tiles * (uint32_t)I.NP;
  const bool vec = (((uintptr_t)out & 15) == 0) && (ld & 3) == 0;
  float4 *S = tile[warp];
  for (uint32_t w = blockIdx.x * (POP_THREADS / 32) + warp; w < total;
       w += gridDim.x * (POP_THREADS / 32)) {
    const int i = (int)(w / tiles), r = (int)(w - (uint32_t)i * tiles);
    const int t0 = r / nk * 32, k0 = r % nk * POP_KB, kb = min(POP_KB, n4 - k0);
    const float4 *row = (const float4 *)row_ptr(I, i, sel[i]) + (size_t)k0 * I.T + t0 + lane;
    float4 v[POP_KB];
#pragma unroll
    for (int k = 0; k < POP_KB; ++k)
      if (k < kb) v[k] = row[(size_t)k * I.T];
    __syncwarp();  // the previous tile has been read
#pragma unroll
    for (int k = 0; k < POP_KB; ++k)
      if (k < kb) S[k * 33 + lane] = v[k];
    __syncwarp();
    float *o = out + (int64_t)i * ld;
    const int sft = kb > 4 ? 3 : (kb > 2 ? 2 : kb - 1);  // 2^sft >= kb groups of a run
    if (vec) {
      for (int it = 0; it < (1 << sft); ++it) {
        const int e = it * 32 + lane, tt = e >> sft, k = e & ((1 << sft) - 1);
        const int j = (t0 + tt) * I.c + 4 * (k0 + k);
        if (k >= kb || j >= I.N) continue;
        const float4 x = S[k * 33 + tt];
        if (j + 4 <= I.N) {
          *(float4 *)(o + j) = x;
        } else {
          o[j] = x.x;
          if (j + 1 < I.N) o[j + 1] = x.y;
          if (j + 2 < I.N) o[j + 2] = x.z;
        }
      }
    } else {
      for (int it = 0; it < (4 << sft); ++it) {
        const int e = it * 32 + lane, tt = e >> (sft + 2), q = e & ((4 << sft) - 1);
        const int j = (t0 + tt) * I.c + 4 * k0 + q;
        if (q < 4 * kb && j < I.N) o[j] = ((const float *)S)[((q >> 2) * 33 + tt) * 4 + (q & 3)];
      }
    }
  }
}

// ------------------------------------------------------------ leader polish
// The three best individuals are polished on the relaxed fitness: theta = tau x,
// `steps` ascent steps theta += lr g / max|g| (g = df/dtheta from the adjoint
// kernels), then x' = clamp(theta / tau, -1, 1) is re-mapped to +-1 and kept
// only if its +-1 fitness is at least the current one (the same greedy rule as
// Sec. 2.2.1 step 4).
static __global__ void k_polish_pick(InstDev I, int32_t *lead_out) {
  __shared__ unsigned long long shk[3 * 32];
  unsigned long long k0 = 0, k1 = 0, k2 = 0;
  for (int i = threadIdx.x; i < I.NP; i += blockDim.x)
    top3_insert(k0, k1, k2, sel_key(I.minimize != 0, I.fit[i], i));
  block_top3(k0, k1, k2, shk);
  if (threadIdx.x == 0) {
    lead_out[0] = key_index(k0);
    lead_out[1] = key_index(k1);
    lead_out[2] = key_index(k2);
  }
}

static __global__ void k_polish_theta(InstDev I, const int32_t *lead, float tau, float *theta) {
  const int k = blockIdx.x, i = lead[k];
  const int32_t *sel = (*I.gen & 1) ? I.sel1 : I.sel0;
  const float *row = row_ptr(I, i, sel[i]);
  for (int j = threadIdx.x; j < I.N; j += blockDim.x)
    theta[(size_t)k * I.Npad + j] = __fmul_rn(tau, row[perm_pos(I, j)]);
}

static __global__ void k_polish_step(int N, int64_t ld, float lr, float *theta, const float *grad) {
  __shared__ float red[32];
  const float *g = grad + (size_t)blockIdx.x * ld;
  float *th = theta + (size_t)blockIdx.x * ld;
  float m = 0.f;
  for (int j = threadIdx.x; j < N; j += blockDim.x) m = fmaxf(m, fabsf(g[j]));
  for (int s = 16; s > 0; s >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, s));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = fmaxf(m, red[w]);
    red[0] = m;
  }
  __syncthreads();
  m = red[0];
  if (m > 0.f && isfinite(m)) {
    const float s = lr / m;
    for (int j = threadIdx.x; j < N; j += blockDim.x) th[j] = fmaf(s, g[j], th[j]);
  }
}

// one CTA (team of T threads) per leader
template <bool COMP>
static __global__ void k_polish_accept(InstDev I, const int32_t *lead, float tau,
                                       const float *theta, int32_t *accepted) {
  extern __shared__ Mono sh[];
  const int k = blockIdx.x, i = lead[k], t = threadIdx.x;
  int32_t *sel = (*I.gen & 1) ? I.sel1 : I.sel0;
  const int si = sel[i];
  float *out = row_ptr(I, i, si ^ 1);
  const float *th = theta + (size_t)k * I.Npad;
  Acc<COMP> acc;
  acc.zero();
  for (int k4 = 0; k4 < I.c / 4; ++k4) {
    const int j0 = t * I.c + 4 * k4;
    float4 x;
    x.x = j0 < I.N ? clamp1(__fdiv_rn(th[j0], tau)) : 0.f;
    x.y = j0 + 1 < I.N ? clamp1(__fdiv_rn(th[j0 + 1], tau)) : 0.f;
    x.z = j0 + 2 < I.N ? clamp1(__fdiv_rn(th[j0 + 2], tau)) : 0.f;
    x.w = j0 + 3 < I.N ? clamp1(__fdiv_rn(th[j0 + 3], tau)) : 0.f;
    *(float4 *)(out + ((size_t)k4 * I.T + t) * 4) = x;
    push4<COMP, false>(acc, I.table, I.T, k4, t, x);
    if (k4 & 1) acc.fold();
  }
  const Mono m = block_reduce(acc.get(), sh);
  if (t == 0) {
    const float2 D = deff_from(m, I.konst[0], I.konst[1]);
    const float f = fit_of(D);
    const bool accept = f >= I.fit[i];
    if (accept) {
      sel[i] = si ^ 1;
      I.fit[i] = f;
      I.dval[i] = D;
    }
    if (accepted) accepted[k] = accept ? 1 : 0;
  }
}

// ------------------------------------------------------ checkpoint / resume
// Natural-order genes [NP][ld] -> slot 0 of every row (permuted), both selectors
// 0, fitness recomputed with the same scan as every other evaluation (so it is
// bit-identical to the value the run had), generation counter set.
template <bool COMP, int MK = 0>
static __global__ void k_load_population(InstDev I, const float *__restrict__ genes, int64_t ld,
                                         int generation) {
  extern __shared__ Mono sh[];
  const int t = threadIdx.x;
  for (int i = blockIdx.x; i < I.NP; i += gridDim.x) {
    if (i != (int)blockIdx.x) __syncthreads();  // the reduction scratch is reused
    float *row = row_ptr(I, i, 0);
    const float *src = genes + (int64_t)i * ld;
    Acc<COMP> acc;
    acc.zero();
    MultiAcc<MK> macc;
    if (MK) macc.zero();
    for (int k4 = 0; k4 < I.c / 4; ++k4) {
      const int j0 = t * I.c + 4 * k4;
      float4 x;
      x.x = j0 < I.N ? src[j0] : 0.f;
      x.y = j0 + 1 < I.N ? src[j0 + 1] : 0.f;
      x.z = j0 + 2 < I.N ? src[j0 + 2] : 0.f;
      x.w = j0 + 3 < I.N ? src[j0 + 3] : 0.f;
      *(float4 *)(row + ((size_t)k4 * I.T + t) * 4) = x;
      if (MK) {
        macc.push4(I, k4, t, x);
      } else {
        push4<COMP, false>(acc, I.table, I.T, k4, t, x);
        if (k4 & 1) acc.fold();
      }
    }
    float2 D = make_float2(0.f, 0.f);
    float f = 0.f;
    if constexpr (MK != 0) {
      multi_finish<MK, false>(I, macc, sh, f, D);
    } else {
      const Mono m = block_reduce(acc.get(), sh);
      if (t == 0) {
        D = field_of(I, m);
        f = fit_of(D);
      }
    }
    if (t == 0) {
      I.fit[i] = f;
      I.dval[i] = D;
      I.sel0[i] = 0;
      I.sel1[i] = 0;
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *I.gen = generation;
    for (int k = 0; k < 4; ++k) I.ctr[k] = 0u;
  }
}

}  // namespace qpm

// =========================================================== host: the state
using qpm::InstDev;

struct qpm_state {
  int dev = 0;
  int n = 0;
  std::vector<InstDev> h;
  std::vector<qpm_problem> probs;
  std::vector<qpm_params> params;
  std::vector<int> grid_plain, grid_persist;
  std::vector<int> grid_init, grid_load;  // k_init and k_load_population of the single kinds
  std::vector<int> grid_mt;  // CTAs of the multi-team kernels of the multi-wavelength kinds
  void *arena = nullptr;
  int g = 0;
  int G_min = 0;
  bool inited = false;
  cudaStream_t cap_stream = nullptr;
  cudaGraphExec_t gexec = nullptr;
  int graph_n = -1;
  unsigned *bar = nullptr;  // [0] count, [1] unused, [2] err, [3] batch queue
  unsigned long long timeout_ns = 5000000000ull;
  InstDev *d_insts = nullptr;  // device copy of the descriptors (batched form)
  qpm::TableJob *d_jobs = nullptr;  // the instances' tables (qpm_init of many instances)
  int max_npad = 0, max_np = 0;
  int32_t *d_order = nullptr;  // instances by decreasing work
  size_t batch_smem = 0;       // dynamic shared memory of the batched kernel
  bool batch_same = false;     // all instances have one seed, whose round keys are
  qpm::PhiloxKey batch_key;    // this
  bool batch_ts = false;       // phasor tables in shared memory (else read from global)
  int grid_batch = 0;
  int batch_cluster = 1;       // CTAs per thread-block cluster in the batched form
  cudaGraphExec_t gexec_b = nullptr;
  int graph_b_n = -1;
  void *polish = nullptr;  // leader-polish scratch (allocated on first use)
  size_t polish_bytes = 0;
  std::vector<qpm_objective> objs;  // per instance (kind 0 unless qpm_set_objective)
  std::vector<void *> objmem;       // tables of a multi-wavelength kind's problems 2 .. K
};

namespace qpm {

// threads per individual: the smallest power of two in [32, 256] giving at most
// 4 domains per thread; beyond 1024 domains the 256 threads take more each
static int choose_team(int N) {
  int T = 32;
  while (T < 256 && N > 4 * T) T *= 2;
  return T;
}

static size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// (two buffers, see red_next)
static size_t smem_bytes(int T) { return sizeof(Mono) * 2 * (size_t)(T / 32); }
// the reduction scratch of the multi-wavelength kinds: one monoid per problem and warp
static size_t smem_bytes_multi(int T) { return sizeof(Mono) * (size_t)(8 * (T / 32) + 1); }

// kernel variants of one instance
struct Variant {
  const void *de, *gwo, *persist;
  size_t smem, persist_smem;
  int block = 0;  // threads per CTA of de / gwo (0: the team width)
};

static constexpr int TS_MAX_NPAD = 4096;  // phasor table in shared memory up to 64 KB
static constexpr size_t BATCH_TS_MAX_BYTES = 160 * 1024;  // batched form: table in smem up to 160 KB

// rows short enough to be read from both of an individual's slots before its slot is known (DUAL)
static bool short_rows(const InstDev &I) { return I.c <= 8; }

template <bool COMP, bool DUAL, bool WIDE>
static Variant variant3(const InstDev &I) {
  Variant v;
  v.de = (const void *)k_de<COMP, DUAL, 0, WIDE>;
  v.gwo = I.combine == 2 ? (const void *)k_gwo_disc<COMP, WIDE>  // the discrete GWO: its own kernel
                         : (const void *)k_gwo<COMP, DUAL, 0, WIDE || !DUAL>;
  // k_de / k_gwo read the table from global memory: long rows stage rows and table
  v.smem = (DUAL ? 0 : sizeof(float4) * stg_f4_per_thread(false) * (size_t)I.T) + smem_bytes(I.T);
  const bool wide = I.T > 256;
  // row staging of the long-row variants (DUAL false)
  const bool ts = I.Npad <= TS_MAX_NPAD;
  const size_t stg = DUAL ? 0 : sizeof(float4) * stg_f4_per_thread(ts) * (size_t)I.T;
  if (ts) {
    v.persist = wide ? (const void *)k_persist<COMP, true, DUAL, 512>
                     : (const void *)k_persist<COMP, true, DUAL>;
    v.persist_smem = stg + sizeof(float4) * (size_t)I.Npad + smem_bytes(I.T);
  } else {
    v.persist = wide ? (const void *)k_persist<COMP, false, DUAL, 512>
                     : (const void *)k_persist<COMP, false, DUAL>;
    v.persist_smem = stg + smem_bytes(I.T);
  }
  return v;
}

template <bool COMP>
static Variant variant2(const InstDev &I) {
  if (short_rows(I)) return I.wide ? variant3<COMP, true, true>(I) : variant3<COMP, true, false>(I);
  return I.wide ? variant3<COMP, false, true>(I) : variant3<COMP, false, false>(I);
}

// the multi-wavelength kinds: launches form only, rows staged; their K tables in shared
// memory shared by the teams of a CTA of up to 512 threads (at most 8 teams with their
// named barriers, 16 one-warp teams) where they fit, else through L1
static size_t optin_smem() {
  int dev = 0, v = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
    return 0;
  return (size_t)v;
}
// the dynamic shared memory the multi-team kernels may take: the opt-in limit less their
// own static shared memory (their attribute is set to it, so states of any size can
// take turns on the same kernels)
template <int MK>
static size_t mt_smem_cap() {
  static const size_t cap = [] {
    cudaFuncAttributes a{}, b{};
    const size_t optin = optin_smem();
    if (cudaFuncGetAttributes(&a, (const void *)k_de_mt<MK>) != cudaSuccess ||
        cudaFuncGetAttributes(&b, (const void *)k_gwo_mt<MK>) != cudaSuccess)
      return (size_t)0;
    const size_t st = std::max(a.sharedSizeBytes, b.sharedSizeBytes);
    return optin > st ? optin - st : (size_t)0;
  }();
  return cap;
}
template <int MK>
static Variant variant_multi(const InstDev &I) {
  Variant v;
  // at most 8 named barriers (1 .. 8); one-warp teams need none (16 per CTA)
  const int nteams = std::max(1, std::min(I.T == 32 ? 16 : 8, 512 / I.T));
  const int block = nteams * I.T;
  const size_t mt = (size_t)I.K * I.Npad * mt_entry_bytes<MK>() +
                    sizeof(float4) * stg_f4_per_thread(true) * (size_t)block +
                    sizeof(Mono) * (size_t)MultiAcc<MK>::KMAX * (I.T / 32) * nteams;
  if (mt <= mt_smem_cap<MK>()) {
    v.de = (const void *)k_de_mt<MK>;
    v.gwo = (const void *)k_gwo_mt<MK>;
    v.smem = mt;
    v.block = block;
    v.persist = nullptr;
    v.persist_smem = 0;
    return v;
  }
  v.de = (const void *)k_de<false, false, MK>;
  v.gwo = (const void *)k_gwo<false, false, MK>;
  v.smem = sizeof(float4) * stg_f4_per_thread(true) * (size_t)I.T + smem_bytes_multi(I.T);
  v.persist = nullptr;
  v.persist_smem = 0;
  return v;
}

static Variant variant_of(const InstDev &I) {
  if (I.obj == OBJ_MULTI_THG) return variant_multi<OBJ_MULTI_THG>(I);
  if (I.obj == OBJ_MULTI_SHG) return variant_multi<OBJ_MULTI_SHG>(I);
  return I.compensated ? variant2<true>(I) : variant2<false>(I);
}

// the shared-memory attribute of a persistent variant is the same for every
// instance (the largest any instance can need), so occupancy figures computed
// for one instance stay valid after another instance is set up
static size_t persist_smem_cap(bool ts) {
  return sizeof(float4) * stg_f4_per_thread(ts) * 512 + smem_bytes(512) +
         (ts ? sizeof(float4) * (size_t)TS_MAX_NPAD : 0);
}

template <bool SAME>
static const void *batch_kernel(bool ts, bool cl) {
  if (ts) return cl ? (const void *)k_batch<true, true, SAME> : (const void *)k_batch<true, false, SAME>;
  return cl ? (const void *)k_batch<false, true, SAME> : (const void *)k_batch<false, false, SAME>;
}
static const void *batch_kernel(const qpm_state *st, int cs) {
  return st->batch_same ? batch_kernel<true>(st->batch_ts, cs > 1)
                        : batch_kernel<false>(st->batch_ts, cs > 1);
}

// co-resident CTAs of the batched kernel for clusters of `cs` CTAs (a multiple of cs)
static qpm_status batch_grid(const qpm_state *st, int cs, int *grid) {
  const void *kb = batch_kernel(st, cs);
  // the largest any state of this kernel variant can need, so that a state with smaller
  // tables cannot fail the captured launch of another
  const size_t cap = sizeof(float4) * stg_f4_per_thread(st->batch_ts) * BATCH_WARPS * 32 +
                     (st->batch_ts ? BATCH_TS_MAX_BYTES : 0);
  QPM_CUDA(cudaFuncSetAttribute(kb, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cap));
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)(cs * sm_count()));
  cfg.blockDim = dim3(BATCH_WARPS * 32);
  cfg.dynamicSmemBytes = st->batch_smem;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int clusters = 0;
  QPM_CUDA(cudaOccupancyMaxActiveClusters(&clusters, kb, &cfg));
  if (clusters < 1) return fail(QPM_ERR_UNSUPPORTED, "batched form: clusters of this size do not fit");
  *grid = clusters * cs;
  return QPM_OK;
}

static qpm_status plain_occupancy(const InstDev &I, int *plain) {
  const Variant v = variant_of(I);
  int a = 0, b = 0;
  // the largest dynamic shared memory any instance's k_de / k_gwo can need
  const int plain_cap = (int)(sizeof(float4) * stg_f4_per_thread(false) * 512 + smem_bytes(512));
  QPM_CUDA(cudaFuncSetAttribute(v.de, cudaFuncAttributeMaxDynamicSharedMemorySize, plain_cap));
  QPM_CUDA(cudaFuncSetAttribute(v.gwo, cudaFuncAttributeMaxDynamicSharedMemorySize, plain_cap));
  QPM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, v.de, I.T, v.smem));
  QPM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, v.gwo, I.T, v.smem));
  *plain = std::max(1, std::min(a, b));
  return QPM_OK;
}

// resident CTAs per SM of the plain and the persistent kernels; sets I.wide
static qpm_status occupancy(InstDev &I, int *plain, int *persist) {
  int wide = 0, narrow = 0;
  I.wide = 1;
  qpm_status r = plain_occupancy(I, &wide);
  if (r != QPM_OK) return r;
  *plain = wide;
  if (short_rows(I) || I.combine == 2) {  // 112 registers where that is no more rounds of individuals
    I.wide = 0;
    if ((r = plain_occupancy(I, &narrow)) != QPM_OK) return r;
    auto rounds = [&](int occ) { return (I.NP + occ * sm_count() - 1) / (occ * sm_count()); };
    I.wide = rounds(wide) <= rounds(narrow);
    *plain = I.wide ? wide : narrow;
  }
  const Variant v = variant_of(I);
  int b = 0;
  QPM_CUDA(cudaFuncSetAttribute(v.persist, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)persist_smem_cap(I.Npad <= TS_MAX_NPAD)));
  QPM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, v.persist, I.T, v.persist_smem));
  *persist = std::max(1, b);
  return QPM_OK;
}

static qpm_status enqueue_step(qpm_state *st, cudaStream_t s) {
  for (int k = 0; k < st->n; ++k) {
    InstDev I = st->h[k];
    const Variant v = variant_of(I);
    void *args[] = {&I};
    const bool mt = v.block != 0;  // several teams per CTA
    const dim3 grid(mt ? st->grid_mt[k] : st->grid_plain[k]), block(mt ? v.block : I.T);
    if (mt) {  // each phase a programmatic dependent of the one before
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[0].val.programmaticStreamSerializationAllowed = 1;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = grid;
      cfg.blockDim = block;
      cfg.dynamicSmemBytes = v.smem;
      cfg.stream = s;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      QPM_CUDA(cudaLaunchKernelExC(&cfg, v.de, args));
      QPM_CUDA(cudaLaunchKernelExC(&cfg, v.gwo, args));
      continue;
    }
    QPM_CUDA(cudaLaunchKernel(v.de, grid, block, args, v.smem, s));
    QPM_CUDA(cudaLaunchKernel(v.gwo, grid, block, args, v.smem, s));
  }
  return QPM_OK;
}

static int best_parts(int N) { return (N + BEST_DOMAINS - 1) / BEST_DOMAINS; }

static TableJob table_job(const InstDev &I) {
  return TableJob{{I.N, I.Npad, I.T, I.c, I.kappa1, I.kappa2}, I.table, I.tpart, I.konst, I.konst64};
}

// A copy from pageable memory may return before its last bytes are on the device, and the streams
// that read the descriptors next (qpm_init of many instances, the batched form) need not wait for
// the legacy stream it ran on.
static cudaError_t descriptors_landed() { return cudaStreamSynchronize(nullptr); }

static qpm_status check_state(qpm_state *st, int gens) {
  if (!st) return fail(QPM_ERR_ARG, "NULL state");
  if (!st->inited) return fail(QPM_ERR_STATE, "qpm_init has not been called");
  if (gens < 0) return fail(QPM_ERR_ARG, "negative generation count");
  if (st->g + gens > st->G_min)
    return fail(QPM_ERR_ARG, "running past the last generation G of an instance");
  int dev = -1;
  QPM_CUDA(cudaGetDevice(&dev));
  if (dev != st->dev) return fail(QPM_ERR_STATE, "state belongs to another device");
  return QPM_OK;
}

}  // namespace qpm

using namespace qpm;

extern "C" qpm_status qpm_create(const qpm_problem *probs, const qpm_params *params,
                                 int32_t n_inst, qpm_state **out) {
  if (!probs || !params || !out) return fail(QPM_ERR_ARG, "qpm_create: NULL pointer");
  if (n_inst < 1) return fail(QPM_ERR_ARG, "qpm_create: n_inst < 1");
  *out = nullptr;
  for (int k = 0; k < n_inst; ++k) {
    const qpm_problem &p = probs[k];
    const qpm_params &q = params[k];
    if (p.N < 1) return fail(QPM_ERR_ARG, "qpm_create: N < 1");
    if (p.N > (1 << 26)) return fail(QPM_ERR_UNSUPPORTED, "qpm_create: N too large");
    if (q.NP < 4) return fail(QPM_ERR_ARG, "qpm_create: NP < 4 (rand/1 needs three donors)");
    if (q.NP > (1 << 28)) return fail(QPM_ERR_UNSUPPORTED, "qpm_create: NP above 2^28");
    if (q.G < 1) return fail(QPM_ERR_ARG, "qpm_create: G < 1");
    if (!(q.F >= 0.f && q.F <= 2.f)) return fail(QPM_ERR_ARG, "qpm_create: F outside [0, 2]");
    if (!(q.CR >= 0.f && q.CR <= 1.f)) return fail(QPM_ERR_ARG, "qpm_create: CR outside [0, 1]");
    if (q.gwo_combine < 0 || q.gwo_combine > 2)
      return fail(QPM_ERR_ARG, "qpm_create: gwo_combine must be 0, 1 or 2");
    if (q.team != 0 && q.team != 32 && q.team != 64 && q.team != 128 && q.team != 256 &&
        q.team != 512)
      return fail(QPM_ERR_ARG, "qpm_create: team must be 0, 32, 64, 128, 256 or 512");
    if (q.f_schedule < 0 || q.f_schedule > 2)
      return fail(QPM_ERR_ARG, "qpm_create: f_schedule must be 0, 1 or 2");
    if (q.f_schedule == 2 && q.NP > (1 << 23))
      return fail(QPM_ERR_UNSUPPORTED, "qpm_create: the adaptive F needs NP <= 2^23");
    if (!std::isfinite(p.kappa1) || !std::isfinite(p.kappa2))
      return fail(QPM_ERR_ARG, "qpm_create: kappa must be finite");
  }
  qpm_state *st = new qpm_state();
  cudaError_t e = cudaGetDevice(&st->dev);
  if (e != cudaSuccess) { delete st; return cuda_fail(e, "cudaGetDevice"); }
  st->n = n_inst;
  st->probs.assign(probs, probs + n_inst);
  st->params.assign(params, params + n_inst);
  st->h.resize(n_inst);
  st->grid_plain.resize(n_inst);
  st->grid_init.resize(n_inst);
  st->grid_load.resize(n_inst);
  st->grid_mt.assign(n_inst, 0);
  st->grid_persist.resize(n_inst);
  st->objs.assign(n_inst, qpm_objective{});
  st->objmem.assign(n_inst, nullptr);
  st->G_min = params[0].G;
  const int nsm = sm_count();
  size_t total = 0;
  std::vector<size_t> base(n_inst);
  for (int k = 0; k < n_inst; ++k) {
    const qpm_problem &p = probs[k];
    const qpm_params &q = params[k];
    InstDev &I = st->h[k];
    memset(&I, 0, sizeof(I));
    I.N = p.N;
    I.T = q.team ? q.team : (n_inst > 1 ? 32 : choose_team(p.N));
    I.Npad = (int32_t)align_up((size_t)p.N, 4 * (size_t)I.T);
    I.c = I.Npad / I.T;
    I.NP = q.NP;
    I.G = q.G;
    I.combine = q.gwo_combine;
    I.compensated = q.compensated ? 1 : 0;
    I.F = q.F;
    I.CR = q.CR;
    I.crthr = cr_threshold(q.CR);
    I.inst = (uint32_t)k;
    I.key = make_uint2((uint32_t)q.seed, (uint32_t)(q.seed >> 32));
    I.kappa1 = p.kappa1;
    I.kappa2 = p.kappa2;
    st->G_min = std::min(st->G_min, q.G);
    int occ_plain = 1, occ_persist = 1;
    qpm_status s2 = occupancy(I, &occ_plain, &occ_persist);
    if (s2 != QPM_OK) { delete st; return s2; }
    if (q.team == 0 && n_inst == 1 && I.T == 256 && I.c >= 16) {
      // long rows: 512 threads per individual (one CTA per SM) when that leaves fewer
      // CTA slots idle in the last round of individuals of a phase
      InstDev W = I;
      W.T = 512;
      W.Npad = (int32_t)align_up((size_t)p.N, 4 * (size_t)W.T);
      W.c = W.Npad / W.T;
      int wp = 1, wq = 1;
      s2 = occupancy(W, &wp, &wq);
      if (s2 != QPM_OK) { delete st; return s2; }
      auto fill = [&](int slots) {
        const int rounds = (I.NP + slots - 1) / slots;
        return (double)I.NP / ((double)rounds * slots);
      };
      if (fill(wq * nsm) > fill(occ_persist * nsm) + 0.05) {
        I.T = W.T;
        I.Npad = W.Npad;
        I.c = W.c;
        I.wide = W.wide;
        occ_plain = wp;
        occ_persist = wq;
      }
    }
    st->grid_plain[k] = std::min(I.NP, occ_plain * nsm);
    int occ_init = 1;  // of its own: it needs fewer registers than the phases
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &occ_init, I.compensated ? (const void *)k_init<true> : (const void *)k_init<false>, I.T, smem_bytes(I.T));
    if (e != cudaSuccess) { delete st; return cuda_fail(e, "occupancy of k_init"); }
    st->grid_init[k] = std::min(I.NP, std::max(1, occ_init) * nsm);
    // 768 threads an SM: more of them read the caller's rows more slowly (5000 x 13200 191 us for 170, 5000 x
    // 1320 29 for 25)
    st->grid_load[k] = std::min(I.NP, std::max(1, std::min(occ_init, 768 / I.T)) * nsm);
    st->grid_persist[k] = std::min(I.NP, occ_persist * nsm);
    base[k] = total;
    const size_t NP = (size_t)I.NP, Np = (size_t)I.Npad;
    total += align_up(2 * NP * Np * sizeof(float), 256);
    total += 2 * align_up(NP * sizeof(int32_t), 256);
    total += align_up(NP * sizeof(float), 256) + align_up(NP * sizeof(float2), 256);
    total += align_up(Np * sizeof(float4), 256);
    total += align_up((size_t)table_part_count(I.Npad) * sizeof(double2), 256);
    total += 256 + 256 + 256;  // konst, konst64, lead
    total += align_up(6 * NP * sizeof(unsigned long long), 256);
    total += align_up(NP * sizeof(unsigned long long), 256);  // DE survivor keys
    total += 2 * align_up((size_t)(q.G + 1) * sizeof(float), 256);  // F history, F base
    total += align_up((size_t)q.G * 7 * sizeof(uint32_t), 256);     // discrete GWO thresholds
    total += 256 + 256;  // ctr, gen
    total += align_up(3 * (size_t)best_parts(p.N) * sizeof(double2), 256);
  }
  const size_t desc_off = total;
  total += align_up(sizeof(InstDev) * (size_t)n_inst, 256);
  const size_t jobs_off = total;
  total += align_up(sizeof(TableJob) * (size_t)n_inst, 256);
  const size_t order_off = total;
  total += align_up(sizeof(int32_t) * (size_t)n_inst, 256);
  total += 256;  // barrier words
  e = cudaMalloc(&st->arena, total);
  if (e != cudaSuccess) { delete st; return cuda_fail(e, "cudaMalloc(state arena)"); }
  e = cudaMemset(st->arena, 0, total);
  if (e != cudaSuccess) { cudaFree(st->arena); delete st; return cuda_fail(e, "cudaMemset"); }
  for (int k = 0; k < n_inst; ++k) {
    InstDev &I = st->h[k];
    char *p = (char *)st->arena + base[k];
    auto take = [&](size_t bytes) { char *r = p; p += align_up(bytes, 256); return (void *)r; };
    const size_t NP = (size_t)I.NP, Np = (size_t)I.Npad;
    I.pop = (float *)take(2 * NP * Np * sizeof(float));
    I.sel0 = (int32_t *)take(NP * sizeof(int32_t));
    I.sel1 = (int32_t *)take(NP * sizeof(int32_t));
    I.fit = (float *)take(NP * sizeof(float));
    I.dval = (float2 *)take(NP * sizeof(float2));
    I.table = (float4 *)take(Np * sizeof(float4));
    I.tpart = (double2 *)take((size_t)table_part_count(I.Npad) * sizeof(double2));
    I.konst = (float2 *)take(4 * sizeof(float2));
    I.K = 1;  // the cascaded d_eff of the problem until qpm_set_objective
    I.mtab[0] = I.table;
    I.mkonst[0] = I.konst;
    I.konst64 = (double2 *)take(4 * sizeof(double2));
    I.lead = (int32_t *)take(4 * sizeof(int32_t));  // four for the discrete GWO
    I.topk = (unsigned long long *)take(6 * NP * sizeof(unsigned long long));
    I.dekey = (unsigned long long *)take(NP * sizeof(unsigned long long));
    {
      float *fs = (float *)take((size_t)(I.G + 1) * sizeof(float));
      float *fb = (float *)take((size_t)(I.G + 1) * sizeof(float));
      I.Fsched = st->params[k].f_schedule ? fs : nullptr;
      I.Fbase = st->params[k].f_schedule == 2 ? fb : nullptr;
      I.adaptive = st->params[k].f_schedule == 2 ? 1 : 0;
    }
    {
      uint32_t *th = (uint32_t *)take((size_t)I.G * 7 * sizeof(uint32_t));
      I.dthr = I.combine == 2 ? th : nullptr;
    }
    I.ctr = (unsigned *)take(4 * sizeof(unsigned));
    I.gen = (int32_t *)take(sizeof(int32_t));
    I.rpart = (double2 *)take(3 * (size_t)best_parts(I.N) * sizeof(double2));
  }
  st->bar = (unsigned *)((char *)st->arena + total - 256);
  st->d_insts = (InstDev *)((char *)st->arena + desc_off);
  st->d_order = (int32_t *)((char *)st->arena + order_off);
  st->d_jobs = (TableJob *)((char *)st->arena + jobs_off);
  {
    // largest instances first (longest-processing-time order for the batch queue)
    std::vector<int32_t> order(n_inst);
    for (int k = 0; k < n_inst; ++k) order[k] = k;
    std::stable_sort(order.begin(), order.end(), [&](int32_t a, int32_t b) {
      return (long long)st->h[a].NP * st->h[a].Npad > (long long)st->h[b].NP * st->h[b].Npad;
    });
    // F schedules (Sec. 3.1.1): cosine decay times a quadratic factor 1.0 -> 0.8, for
    // generations 0 .. G; from F (f_schedule 1), or from the top 0.1 of the adaptive
    // F's interval (f_schedule 2: its intermediate state's values in Fbase, and its
    // first generation's F in the history)
    // thresholds of the discrete GWO (Sec. 3.1.2): per generation g (tau = g / G) the
    // social rate, the disturbance and P(+1) for 0 .. 4 leaders at +1, as 16-bit
    // thresholds floor(65536 p), evaluated in FP64
    for (int k = 0; k < n_inst && e == cudaSuccess; ++k) {
      if (!st->h[k].dthr) continue;
      const int G = st->h[k].G;
      std::vector<uint32_t> th((size_t)G * 7);
      for (int g = 0; g < G; ++g) {
        const double tau = (double)g / (double)G;
        const double delta = 0.5 * (1.0 - tau), sigma = 0.3 * (1.0 - tau);
        const double mu = 0.1 * (1.0 - tau) + 0.01 * tau;
        th[7 * (size_t)g] = (uint32_t)std::floor(65536.0 * sigma);
        th[7 * (size_t)g + 1] = (uint32_t)std::floor(65536.0 * mu);
        for (int n = 0; n <= 4; ++n) {
          const double m = n > 2 ? 1.0 : (n < 2 ? 0.0 : 0.5);
          const double qn = (1.0 - tau) * ((double)n / 4.0) + tau * m;
          th[7 * (size_t)g + 2 + n] = (uint32_t)std::floor(65536.0 * ((1.0 - delta) * qn + 0.5 * delta));
        }
      }
      e = cudaMemcpy((void *)st->h[k].dthr, th.data(), sizeof(uint32_t) * th.size(),
                     cudaMemcpyHostToDevice);
    }
    for (int k = 0; k < n_inst && e == cudaSuccess; ++k) {
      if (!st->h[k].Fsched) continue;
      const int G = st->h[k].G;
      const bool adaptive = st->h[k].adaptive != 0;
      const double top = adaptive ? 0.1 : (double)st->params[k].F;
      std::vector<float> F(G + 1);
      for (int g = 0; g <= G; ++g) {
        const double x = (double)g / (double)G;
        const double c = 0.5 * (std::cos(M_PI * (double)g / (2.0 * (double)G)) + 1.0);
        const double qd = 1.0 - 0.2 * x * x;
        F[g] = (float)(top * c * qd);
      }
      e = cudaMemcpy(st->h[k].Fsched, F.data(), sizeof(float) * (G + 1), cudaMemcpyHostToDevice);
      if (e == cudaSuccess && adaptive)
        e = cudaMemcpy((void *)st->h[k].Fbase, F.data(), sizeof(float) * (G + 1),
                       cudaMemcpyHostToDevice);
    }
    if (e == cudaSuccess)
      e = cudaMemcpy(st->d_order, order.data(), sizeof(int32_t) * n_inst, cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
      e = cudaMemcpy(st->d_insts, st->h.data(), sizeof(InstDev) * n_inst, cudaMemcpyHostToDevice);
    std::vector<TableJob> jobs(n_inst);
    for (int k = 0; k < n_inst; ++k) jobs[k] = table_job(st->h[k]);
    if (e == cudaSuccess)
      e = cudaMemcpy(st->d_jobs, jobs.data(), sizeof(TableJob) * n_inst, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = descriptors_landed();
    if (e != cudaSuccess) { cudaFree(st->arena); delete st; return cuda_fail(e, "cudaMemcpy"); }
    int maxpad = 0;
    for (int k = 0; k < n_inst; ++k) {
      maxpad = std::max(maxpad, st->h[k].Npad);
      st->max_np = std::max(st->max_np, st->h[k].NP);
    }
    st->max_npad = maxpad;
    st->batch_same = true;
    st->batch_key = philox_schedule(st->h[0].key);
    for (int k = 1; k < n_inst; ++k) st->batch_same &= params[k].seed == params[0].seed;
    st->batch_ts = (size_t)maxpad * sizeof(float4) <= BATCH_TS_MAX_BYTES;
    st->batch_smem = sizeof(float4) * stg_f4_per_thread(st->batch_ts) * BATCH_WARPS * 32 +
                     (st->batch_ts ? (size_t)maxpad * sizeof(float4) : 0);
    st->grid_batch = 0;  // set on the first batched run (or by qpm_set_batch_cluster)
  }
  e = cudaStreamCreateWithFlags(&st->cap_stream, cudaStreamNonBlocking);
  if (e != cudaSuccess) { cudaFree(st->arena); delete st; return cuda_fail(e, "cudaStreamCreate"); }
  *out = st;
  return QPM_OK;
}

extern "C" qpm_status qpm_set_trace(qpm_state *st, int32_t inst, float *trace) {
  if (!st || inst < 0 || inst >= st->n) return fail(QPM_ERR_ARG, "qpm_set_trace: bad instance");
  st->h[inst].trace = trace;
  if (st->gexec) {
    cudaGraphExecDestroy(st->gexec);
    st->gexec = nullptr;
    st->graph_n = -1;
  }
  cudaError_t e = cudaMemcpy(st->d_insts + inst, &st->h[inst], sizeof(InstDev), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = descriptors_landed();
  if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpy(descriptor)");
  return QPM_OK;
}

extern "C" qpm_status qpm_init(qpm_state *st, qpm_stream_t stream) {
  if (!st) return fail(QPM_ERR_ARG, "NULL state");
  cudaStream_t s = (cudaStream_t)stream;
  // many instances of one-warp teams and single kinds: three launches for all of them
  bool many = st->n > 1;
  for (int k = 0; many && k < st->n; ++k) many = st->h[k].T == 32 && st->h[k].obj < OBJ_MULTI_THG;
  if (many) {
    qpm_status r = launch_tables(st->d_jobs, st->n, st->max_npad, s);
    if (r != QPM_OK) return r;
    const dim3 grid(std::min(64, (st->max_np + INIT_WARPS - 1) / INIT_WARPS), std::min(st->n, 65535));
    k_init_many<<<grid, INIT_WARPS * 32, 0, s>>>(st->d_insts, st->d_order, st->n);
    QPM_CUDA(cudaGetLastError());
  }
  for (int k = 0; !many && k < st->n; ++k) {
    const InstDev &I = st->h[k];
    TableSpec ts{I.N, I.Npad, I.T, I.c, I.kappa1, I.kappa2};
    qpm_status r = launch_table(ts, I.table, I.tpart, I.konst, I.konst64, s);
    if (r != QPM_OK) return r;
    // the other problems of a multi-wavelength kind (one after the other: they share
    // the reduction scratch on this stream)
    for (int q = 1; q < (I.obj >= OBJ_MULTI_THG ? I.K : 1); ++q) {
      TableSpec tq{I.N, I.Npad, I.T, I.c, st->objs[k].kappa1[q], st->objs[k].kappa2[q]};
      r = launch_table(tq, (float4 *)I.mtab[q], I.tpart, (float2 *)I.mkonst[q], nullptr, s);
      if (r != QPM_OK) return r;
    }
    const size_t sm = smem_bytes(I.T), smm = smem_bytes_multi(I.T);
    if (I.obj == OBJ_MULTI_THG) k_init<false, OBJ_MULTI_THG><<<st->grid_plain[k], I.T, smm, s>>>(I);
    else if (I.obj == OBJ_MULTI_SHG) k_init<false, OBJ_MULTI_SHG><<<st->grid_plain[k], I.T, smm, s>>>(I);
    else if (I.compensated) k_init<true><<<st->grid_init[k], I.T, sm, s>>>(I);
    else k_init<false><<<st->grid_init[k], I.T, sm, s>>>(I);
    QPM_CUDA(cudaGetLastError());
  }
  st->g = 0;
  st->inited = true;
  return QPM_OK;
}

extern "C" qpm_status qpm_step(qpm_state *st, qpm_stream_t stream) {
  qpm_status r = check_state(st, 1);
  if (r != QPM_OK) return r;
  r = enqueue_step(st, (cudaStream_t)stream);
  if (r == QPM_OK) st->g += 1;
  return r;
}

extern "C" qpm_status qpm_run(qpm_state *st, int32_t generations, int32_t mode,
                              qpm_stream_t stream) {
  qpm_status r = check_state(st, generations);
  if (r != QPM_OK) return r;
  cudaStream_t s = (cudaStream_t)stream;
  if (generations == 0) return QPM_OK;
  if (mode == QPM_RUN_LAUNCHES) {
    for (int g = 0; g < generations; ++g) {
      r = enqueue_step(st, s);
      if (r != QPM_OK) return r;
    }
  } else if (mode == QPM_RUN_GRAPH) {
    if (st->graph_n != generations || !st->gexec) {
      if (st->gexec) {
        cudaGraphExecDestroy(st->gexec);
        st->gexec = nullptr;
      }
      QPM_CUDA(cudaStreamBeginCapture(st->cap_stream, cudaStreamCaptureModeThreadLocal));
      for (int g = 0; g < generations; ++g) {
        r = enqueue_step(st, st->cap_stream);
        if (r != QPM_OK) {
          cudaGraph_t junk;
          cudaStreamEndCapture(st->cap_stream, &junk);
          if (junk) cudaGraphDestroy(junk);
          return r;
        }
      }
      cudaGraph_t graph;
      QPM_CUDA(cudaStreamEndCapture(st->cap_stream, &graph));
      cudaError_t e = cudaGraphInstantiate(&st->gexec, graph, 0);
      cudaGraphDestroy(graph);
      if (e != cudaSuccess) return cuda_fail(e, "cudaGraphInstantiate");
      st->graph_n = generations;
    }
    QPM_CUDA(cudaGraphLaunch(st->gexec, s));
  } else if (mode == QPM_RUN_PERSISTENT) {
    for (int k = 0; k < st->n; ++k)
      if (st->h[k].obj >= OBJ_MULTI_THG || st->h[k].combine == 2)
        return fail(QPM_ERR_UNSUPPORTED, "the multi-wavelength objectives and the discrete GWO "
                                         "run in the launches and graph forms");
    QPM_CUDA(cudaMemsetAsync(st->bar, 0, 3 * sizeof(unsigned), s));
    for (int k = 0; k < st->n; ++k) {
      InstDev I = st->h[k];
      const Variant v = variant_of(I);
      int g_end = st->g + generations;
      // each instance gets a fresh arrival counter; the error word is shared
      QPM_CUDA(cudaMemsetAsync(st->bar, 0, sizeof(unsigned), s));
      Barrier b{st->bar, (int32_t *)(st->bar + 2), st->timeout_ns};
      void *args[] = {&I, &g_end, &b};
      QPM_CUDA(cudaLaunchCooperativeKernel(v.persist, st->grid_persist[k], I.T, args,
                                           v.persist_smem, s));
    }
    int32_t err = 0;
    QPM_CUDA(cudaMemcpyAsync(&err, st->bar + 2, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    QPM_CUDA(cudaStreamSynchronize(s));
    if (err != 0) {
      st->g += generations;
      return fail(QPM_ERR_TIMEOUT, "persistent kernel: a bounded grid-barrier wait gave up");
    }
  } else if (mode == QPM_RUN_BATCHED) {
    for (int k = 0; k < st->n; ++k)
      if (st->h[k].obj >= OBJ_MULTI_THG || st->h[k].combine == 2)
        return fail(QPM_ERR_UNSUPPORTED, "the multi-wavelength objectives and the discrete GWO "
                                         "run in the launches and graph forms");
    for (int k = 0; k < st->n; ++k)
      if (st->h[k].T != 32)
        return fail(QPM_ERR_UNSUPPORTED, "batched form needs 32 threads per individual (team 32)");
    if (st->grid_batch == 0) {
      qpm_status r = batch_grid(st, st->batch_cluster, &st->grid_batch);
      if (r != QPM_OK) return r;
    }
    if (st->graph_b_n != generations || !st->gexec_b) {
      if (st->gexec_b) {
        cudaGraphExecDestroy(st->gexec_b);
        st->gexec_b = nullptr;
      }
      QPM_CUDA(cudaStreamBeginCapture(st->cap_stream, cudaStreamCaptureModeThreadLocal));
      cudaError_t e = cudaMemsetAsync(st->bar + 3, 0, sizeof(unsigned), st->cap_stream);
      if (e == cudaSuccess) {
        int n = st->n, gens = generations;
        unsigned *queue = st->bar + 3;
        void *args[] = {&st->d_insts, &st->d_order, &n, &queue, &gens, &st->batch_key};
        const void *kb = batch_kernel(st, st->batch_cluster);
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)st->batch_cluster;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3((unsigned)st->grid_batch);
        cfg.blockDim = dim3(BATCH_WARPS * 32);
        cfg.dynamicSmemBytes = st->batch_smem;
        cfg.stream = st->cap_stream;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        e = cudaLaunchKernelExC(&cfg, kb, args);
      }
      cudaGraph_t graph = nullptr;
      cudaError_t e2 = cudaStreamEndCapture(st->cap_stream, &graph);
      if (e != cudaSuccess || e2 != cudaSuccess) {
        if (graph) cudaGraphDestroy(graph);
        return cuda_fail(e != cudaSuccess ? e : e2, "capturing the batched launch");
      }
      e = cudaGraphInstantiate(&st->gexec_b, graph, 0);
      cudaGraphDestroy(graph);
      if (e != cudaSuccess) return cuda_fail(e, "cudaGraphInstantiate");
      st->graph_b_n = generations;
    }
    QPM_CUDA(cudaGraphLaunch(st->gexec_b, s));
  } else {
    return fail(QPM_ERR_ARG, "qpm_run: unknown mode");
  }
  st->g += generations;
  return QPM_OK;
}

extern "C" qpm_status qpm_set_batch_cluster(qpm_state *st, int32_t ctas) {
  if (!st) return fail(QPM_ERR_ARG, "qpm_set_batch_cluster: NULL state");
  if (ctas != 1 && ctas != 2 && ctas != 4 && ctas != 8)
    return fail(QPM_ERR_ARG, "qpm_set_batch_cluster: ctas must be 1, 2, 4 or 8");
  int dev = -1;
  QPM_CUDA(cudaGetDevice(&dev));
  if (dev != st->dev) return fail(QPM_ERR_STATE, "state belongs to another device");
  int grid = 0;
  qpm_status r = batch_grid(st, ctas, &grid);
  if (r != QPM_OK) return r;
  if (st->gexec_b) {  // the captured launch has the old shape
    QPM_CUDA(cudaDeviceSynchronize());
    cudaGraphExecDestroy(st->gexec_b);
    st->gexec_b = nullptr;
    st->graph_b_n = -1;
  }
  st->batch_cluster = ctas;
  st->grid_batch = grid;
  return QPM_OK;
}

extern "C" qpm_status qpm_set_objective(qpm_state *st, int32_t inst, const qpm_objective *o) {
  if (!st || inst < 0 || inst >= st->n || !o) return fail(QPM_ERR_ARG, "qpm_set_objective: bad arguments");
  if (st->inited) return fail(QPM_ERR_STATE, "qpm_set_objective: call it before qpm_init");
  if (o->kind < OBJ_THG || o->kind > OBJ_MULTI_SHG)
    return fail(QPM_ERR_ARG, "qpm_set_objective: kind must be one of QPM_OBJ_*");
  const bool multi = o->kind >= OBJ_MULTI_THG;
  const int kmax = o->kind == OBJ_MULTI_THG ? 4 : 8;
  if (multi && (o->K < 1 || o->K > kmax))
    return fail(QPM_ERR_ARG, "qpm_set_objective: need 1 <= K <= 4 (THG) or 8 (SHG)");
  for (int k = 0; multi && k < o->K; ++k)
    if (!std::isfinite(o->kappa1[k]) || !std::isfinite(o->kappa2[k]))
      return fail(QPM_ERR_ARG, "qpm_set_objective: kappa must be finite");
  if (multi && (!std::isfinite(o->G0) || !(o->beta >= 0.f) || !std::isfinite(o->beta)))
    return fail(QPM_ERR_ARG, "qpm_set_objective: need finite G0 and beta >= 0");
  int dev = -1;
  QPM_CUDA(cudaGetDevice(&dev));
  if (dev != st->dev) return fail(QPM_ERR_STATE, "state belongs to another device");
  InstDev &I = st->h[inst];
  if (multi && I.combine == 2)
    return fail(QPM_ERR_UNSUPPORTED, "qpm_set_objective: the discrete GWO optimises the single kinds");
  if (st->objmem[inst]) {
    QPM_CUDA(cudaFree(st->objmem[inst]));
    st->objmem[inst] = nullptr;
  }
  I.obj = o->kind;
  I.minimize = multi ? 1 : 0;
  I.K = multi ? o->K : 1;
  I.G0 = multi ? o->G0 : 0.f;
  I.beta = multi ? o->beta : 0.f;
  for (int k = 0; k < 8; ++k) {
    I.mtab[k] = nullptr;
    I.mkonst[k] = nullptr;
  }
  I.mtab[0] = I.table;
  I.mkonst[0] = I.konst;
  if (multi) {
    // the first problem is the instance's own: its table, constants and FP64 re-check
    I.kappa1 = o->kappa1[0];
    I.kappa2 = o->kappa2[0];
    st->probs[inst].kappa1 = o->kappa1[0];
    st->probs[inst].kappa2 = o->kappa2[0];
    if (o->K > 1) {
      const size_t tb = align_up(sizeof(float4) * (size_t)I.Npad, 256);
      void *mem = nullptr;
      QPM_CUDA(cudaMalloc(&mem, (size_t)(o->K - 1) * (tb + 256)));
      st->objmem[inst] = mem;
      for (int k = 1; k < o->K; ++k) {
        char *p = (char *)mem + (size_t)(k - 1) * (tb + 256);
        I.mtab[k] = (const float4 *)p;
        I.mkonst[k] = (const float2 *)(p + tb);
      }
    }
  }
  st->objs[inst] = *o;
  // the kernel variants of the kind and their occupancy
  int occ_plain = 1, occ_persist = 1;
  if (multi && variant_of(I).block != 0) {
    // several teams per CTA sharing the K tables in shared memory
    const Variant v = variant_of(I);
    int a = 0, b = 0;
    // the largest any state can need: a smaller value would fail another state's launch
    const int cap = (int)(I.obj == OBJ_MULTI_THG ? mt_smem_cap<OBJ_MULTI_THG>()
                                                 : mt_smem_cap<OBJ_MULTI_SHG>());
    for (const void *fn : {v.de, v.gwo})
      QPM_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
    QPM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, v.de, v.block, v.smem));
    QPM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, v.gwo, v.block, v.smem));
    if (std::min(a, b) < 1) return fail(QPM_ERR_UNSUPPORTED, "qpm_set_objective: kernels do not fit");
    const int nteams = v.block / I.T;
    st->grid_mt[inst] = std::min((I.NP + nteams - 1) / nteams, std::min(a, b) * sm_count());
    // k_init and k_load_population keep one team per CTA
    int c = 0;
    QPM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &c, I.obj == OBJ_MULTI_THG ? (const void *)k_init<false, OBJ_MULTI_THG>
                                   : (const void *)k_init<false, OBJ_MULTI_SHG>,
        I.T, smem_bytes_multi(I.T)));
    st->grid_plain[inst] = std::min(I.NP, std::max(1, c) * sm_count());
  } else if (multi) {
    const Variant v = variant_of(I);
    // the largest dynamic shared memory a team of up to 512 threads needs
    const int cap = (int)(sizeof(float4) * stg_f4_per_thread(true) * 512 + smem_bytes_multi(512));
    int a = 0, b = 0;
    for (const void *fn : {v.de, v.gwo}) {
      QPM_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
      QPM_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout,
                                    (int)cudaSharedmemCarveoutDefault));
    }
    QPM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, v.de, I.T, v.smem));
    QPM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, v.gwo, I.T, v.smem));
    occ_plain = std::max(1, std::min(a, b));
    // ask for no more shared memory than the resident CTAs use, so that the rest of
    // the SM's L1 holds the K phasor tables; kept only if the occupancy stays
    int dev = 0, smem_sm = 0;
    QPM_CUDA(cudaGetDevice(&dev));
    QPM_CUDA(cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev));
    const int pct = (int)std::min<size_t>(
        100, (100 * (size_t)occ_plain * (v.smem + 1024) + (size_t)smem_sm - 1) / (size_t)smem_sm);
    for (const void *fn : {v.de, v.gwo})
      QPM_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, pct));
    int a2 = 0, b2 = 0;
    QPM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a2, v.de, I.T, v.smem));
    QPM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b2, v.gwo, I.T, v.smem));
    if (std::min(a2, b2) < occ_plain)
      for (const void *fn : {v.de, v.gwo})
        QPM_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout,
                                      (int)cudaSharedmemCarveoutDefault));
    st->grid_plain[inst] = std::min(I.NP, occ_plain * sm_count());
  } else {
    qpm_status r = occupancy(I, &occ_plain, &occ_persist);
    if (r != QPM_OK) return r;
    st->grid_plain[inst] = std::min(I.NP, occ_plain * sm_count());
    st->grid_persist[inst] = std::min(I.NP, occ_persist * sm_count());
  }
  if (st->gexec) {
    cudaGraphExecDestroy(st->gexec);
    st->gexec = nullptr;
    st->graph_n = -1;
  }
  QPM_CUDA(cudaMemcpy(st->d_insts + inst, &I, sizeof(InstDev), cudaMemcpyHostToDevice));
  const TableJob job = table_job(I);
  QPM_CUDA(cudaMemcpy(st->d_jobs + inst, &job, sizeof(TableJob), cudaMemcpyHostToDevice));
  QPM_CUDA(descriptors_landed());
  return QPM_OK;
}

extern "C" qpm_status qpm_team_of(const qpm_state *st, int32_t inst, int32_t *team_out) {
  if (!st || !team_out || inst < 0 || inst >= st->n) return fail(QPM_ERR_ARG, "bad arguments");
  *team_out = st->h[inst].T;
  return QPM_OK;
}

extern "C" qpm_status qpm_instance_shape(const qpm_state *st, int32_t inst, int32_t *N_out,
                                         int32_t *NP_out, int32_t *G_out) {
  if (!st || inst < 0 || inst >= st->n) return fail(QPM_ERR_ARG, "bad state or instance");
  if (N_out) *N_out = st->h[inst].N;
  if (NP_out) *NP_out = st->h[inst].NP;
  if (G_out) *G_out = st->h[inst].G;
  return QPM_OK;
}

static __global__ void k_copy_F(InstDev I, float *out) {
  for (int g = threadIdx.x + blockIdx.x * blockDim.x; g <= I.G; g += blockDim.x * gridDim.x)
    out[g] = I.Fsched ? I.Fsched[g] : I.F;
}

extern "C" qpm_status qpm_get_F(qpm_state *st, int32_t inst, float *F_out, qpm_stream_t stream) {
  if (!st || inst < 0 || inst >= st->n || !F_out) return fail(QPM_ERR_ARG, "bad arguments");
  if (!st->inited) return fail(QPM_ERR_STATE, "qpm_init has not been called");
  const InstDev &I = st->h[inst];
  k_copy_F<<<(I.G + 256) / 256, 256, 0, (cudaStream_t)stream>>>(I, F_out);
  QPM_CUDA(cudaGetLastError());
  return QPM_OK;
}

extern "C" qpm_status qpm_set_F(qpm_state *st, int32_t inst, const float *F_in, qpm_stream_t stream) {
  if (!st || inst < 0 || inst >= st->n || !F_in) return fail(QPM_ERR_ARG, "bad arguments");
  const InstDev &I = st->h[inst];
  if (!I.Fsched) return fail(QPM_ERR_ARG, "qpm_set_F: constant F (f_schedule 0) has no history");
  QPM_CUDA(cudaMemcpyAsync(I.Fsched, F_in, sizeof(float) * (size_t)(I.G + 1),
                           cudaMemcpyDeviceToDevice, (cudaStream_t)stream));
  return QPM_OK;
}

extern "C" qpm_status qpm_generation(const qpm_state *st, int32_t *g_out) {
  if (!st || !g_out) return fail(QPM_ERR_ARG, "NULL pointer");
  *g_out = st->g;
  return QPM_OK;
}

extern "C" qpm_status qpm_set_population(qpm_state *st, int32_t inst, const float *genes,
                                         int64_t ld, int32_t generation, qpm_stream_t stream) {
  if (!st || inst < 0 || inst >= st->n || !genes) return fail(QPM_ERR_ARG, "bad arguments");
  const InstDev &I = st->h[inst];
  if (ld < I.N) return fail(QPM_ERR_ARG, "ld < N");
  if (generation < 0 || generation > I.G) return fail(QPM_ERR_ARG, "generation outside [0, G]");
  if (!st->inited) return fail(QPM_ERR_STATE, "qpm_init has not been called");
  for (int k = 0; k < st->n; ++k)
    if (k != inst && generation != st->g)
      return fail(QPM_ERR_UNSUPPORTED, "all instances of a state share one generation count");
  cudaStream_t s = (cudaStream_t)stream;
  const size_t sm = smem_bytes(I.T), smm = smem_bytes_multi(I.T);
  if (I.obj == OBJ_MULTI_THG)
    k_load_population<false, OBJ_MULTI_THG><<<st->grid_plain[inst], I.T, smm, s>>>(I, genes, ld, generation);
  else if (I.obj == OBJ_MULTI_SHG)
    k_load_population<false, OBJ_MULTI_SHG><<<st->grid_plain[inst], I.T, smm, s>>>(I, genes, ld, generation);
  else if (I.compensated)
    k_load_population<true><<<st->grid_load[inst], I.T, sm, s>>>(I, genes, ld, generation);
  else
    k_load_population<false><<<st->grid_load[inst], I.T, sm, s>>>(I, genes, ld, generation);
  QPM_CUDA(cudaGetLastError());
  st->g = generation;
  return QPM_OK;
}

extern "C" qpm_status qpm_get_population(qpm_state *st, int32_t inst, float *genes_out, int64_t ld,
                                         float *fit_out, float *d_eff_out, qpm_stream_t stream) {
  if (!st || inst < 0 || inst >= st->n) return fail(QPM_ERR_ARG, "bad state or instance");
  if (!st->inited) return fail(QPM_ERR_STATE, "qpm_init has not been called");
  const InstDev &I = st->h[inst];
  if (genes_out && ld < I.N) return fail(QPM_ERR_ARG, "ld < N");
  cudaStream_t s = (cudaStream_t)stream;
  // a warp per tile of 32 x 8 groups, at most 8 CTAs per SM; no genes: a thread per individual
  const int64_t warps = (int64_t)I.NP * (I.T / 32) * ((I.c / 4 + POP_KB - 1) / POP_KB);
  const int64_t ctas = genes_out ? (warps * 32 + POP_THREADS - 1) / POP_THREADS
                                 : (I.NP + POP_THREADS - 1) / POP_THREADS;
  if (genes_out || fit_out || d_eff_out)
    k_population<<<(int)std::min<int64_t>(ctas, 8 * sm_count()), POP_THREADS, 0, s>>>(
        I, genes_out, ld, fit_out, (float2 *)d_eff_out);
  QPM_CUDA(cudaGetLastError());
  return QPM_OK;
}

extern "C" qpm_status qpm_get_best(qpm_state *st, int32_t inst, float *genes_out,
                                   double *d_eff64_out, float *fit_out, int32_t *index_out,
                                   qpm_stream_t stream) {
  if (!st || inst < 0 || inst >= st->n) return fail(QPM_ERR_ARG, "bad state or instance");
  if (!st->inited) return fail(QPM_ERR_STATE, "qpm_init has not been called");
  const InstDev &I = st->h[inst];
  cudaStream_t s = (cudaStream_t)stream;
  BestRot rot;
  for (int q = 1; q <= 3; ++q) {
    rot.r1[q - 1] = make_double2(std::cos(q * I.kappa1), -std::sin(q * I.kappa1));
    rot.r2[q - 1] = make_double2(std::cos(q * I.kappa2), -std::sin(q * I.kappa2));
  }
  const int parts = best_parts(I.N);
  k_best<<<genes_out || d_eff64_out ? parts : 1, BEST_THREADS, 0, s>>>(I, rot, genes_out, fit_out,
                                                                       index_out, d_eff64_out != nullptr);
  QPM_CUDA(cudaGetLastError());
  if (!d_eff64_out) return QPM_OK;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3(1);
  cfg.blockDim = dim3(BEST_THREADS);
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  QPM_CUDA(cudaLaunchKernelEx(&cfg, k_best_close, I, parts, d_eff64_out));
  return QPM_OK;
}

extern "C" qpm_status qpm_destroy(qpm_state *st) {
  if (!st) return QPM_OK;
  cudaDeviceSynchronize();
  if (st->gexec) cudaGraphExecDestroy(st->gexec);
  if (st->gexec_b) cudaGraphExecDestroy(st->gexec_b);
  if (st->polish) cudaFree(st->polish);
  for (void *p : st->objmem)
    if (p) cudaFree(p);
  if (st->cap_stream) cudaStreamDestroy(st->cap_stream);
  cudaFree(st->arena);
  delete st;
  return QPM_OK;
}

extern "C" qpm_status qpm_set_wait_timeout_ns(qpm_state *st, uint64_t ns) {
  if (!st) return fail(QPM_ERR_ARG, "NULL state");
  st->timeout_ns = ns;
  return QPM_OK;
}

extern "C" qpm_status qpm_polish_leaders(qpm_state *st, int32_t inst, int32_t steps, float lr,
                                         float tau, int32_t *accepted_out, qpm_stream_t stream) {
  if (!st || inst < 0 || inst >= st->n) return fail(QPM_ERR_ARG, "bad state or instance");
  if (!st->inited) return fail(QPM_ERR_STATE, "qpm_init has not been called");
  if (steps < 0 || !(lr >= 0.f) || !(tau > 0.f))
    return fail(QPM_ERR_ARG, "qpm_polish_leaders: need steps >= 0, lr >= 0, tau > 0");
  const InstDev &I = st->h[inst];
  if (I.obj != OBJ_THG)
    return fail(QPM_ERR_UNSUPPORTED, "qpm_polish_leaders: the cascaded |d_eff|^2 objective only");
  cudaStream_t s = (cudaStream_t)stream;
  const size_t Np = (size_t)I.Npad;
  const size_t saved_bytes = align_up(3 * (size_t)qpm_relaxed_saved_floats(I.N) * sizeof(float), 256);
  const size_t need = 256 + align_up(3 * Np * sizeof(float), 256) * 2 + 256 + saved_bytes;
  if (st->polish_bytes < need) {
    if (st->polish) {
      QPM_CUDA(cudaDeviceSynchronize());
      QPM_CUDA(cudaFree(st->polish));
      st->polish = nullptr;
      st->polish_bytes = 0;
    }
    QPM_CUDA(cudaMalloc(&st->polish, need));
    st->polish_bytes = need;
  }
  char *p = (char *)st->polish;
  int32_t *lead = (int32_t *)p;
  float *theta = (float *)(p + 256);
  float *grad = (float *)(p + 256 + align_up(3 * Np * sizeof(float), 256));
  float *D = (float *)(p + 256 + 2 * align_up(3 * Np * sizeof(float), 256));
  float *saved = D + 256 / sizeof(float);
  k_polish_pick<<<1, 256, 0, s>>>(I, lead);
  k_polish_theta<<<3, 256, 0, s>>>(I, lead, tau, theta);
  QPM_CUDA(cudaGetLastError());
  const qpm_problem prob = st->probs[inst];
  for (int k = 0; k < steps; ++k) {
    qpm_status r = qpm_deff_relaxed_fwd(&prob, theta, (int64_t)Np, 3, D, nullptr, saved, stream);
    if (r != QPM_OK) return r;
    r = qpm_deff_relaxed_bwd(&prob, theta, (int64_t)Np, 3, D, saved, nullptr, grad, (int64_t)Np,
                             stream);
    if (r != QPM_OK) return r;
    k_polish_step<<<3, 256, 0, s>>>(I.N, (int64_t)Np, lr, theta, grad);
  }
  if (I.compensated)
    k_polish_accept<true><<<3, I.T, smem_bytes(I.T), s>>>(I, lead, tau, theta, accepted_out);
  else
    k_polish_accept<false><<<3, I.T, smem_bytes(I.T), s>>>(I, lead, tau, theta, accepted_out);
  QPM_CUDA(cudaGetLastError());
  return QPM_OK;
}

extern "C" qpm_status qpm_solve(const qpm_problem *prob, const qpm_params *params, int32_t mode,
                                float *best_genes_host, double *best_deff64_host,
                                float *best_fit_host) {
  if (!prob || !params) return fail(QPM_ERR_ARG, "qpm_solve: NULL pointer");
  qpm_state *st = nullptr;
  qpm_status r = qpm_create(prob, params, 1, &st);
  if (r != QPM_OK) return r;
  cudaStream_t s = st->cap_stream;
  float *dgenes = nullptr;
  double *dd = nullptr;
  float *df = nullptr;
  cudaError_t e = cudaMalloc(&dgenes, sizeof(float) * (size_t)prob->N + 64);
  if (e == cudaSuccess) e = cudaMalloc(&dd, 2 * sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc(&df, sizeof(float));
  if (e != cudaSuccess) r = cuda_fail(e, "cudaMalloc");
  if (r == QPM_OK && mode == QPM_RUN_GRAPH) mode = QPM_RUN_LAUNCHES;  // one pass: nothing to reuse
  if (r == QPM_OK) r = qpm_init(st, (qpm_stream_t)s);
  if (r == QPM_OK) r = qpm_run(st, params->G, mode, (qpm_stream_t)s);
  if (r == QPM_OK) r = qpm_get_best(st, 0, dgenes, dd, df, nullptr, (qpm_stream_t)s);
  if (r == QPM_OK && best_genes_host) {
    e = cudaMemcpyAsync(best_genes_host, dgenes, sizeof(float) * (size_t)prob->N,
                        cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) r = cuda_fail(e, "cudaMemcpyAsync");
  }
  if (r == QPM_OK && best_deff64_host) {
    e = cudaMemcpyAsync(best_deff64_host, dd, 2 * sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) r = cuda_fail(e, "cudaMemcpyAsync");
  }
  if (r == QPM_OK && best_fit_host) {
    e = cudaMemcpyAsync(best_fit_host, df, sizeof(float), cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) r = cuda_fail(e, "cudaMemcpyAsync");
  }
  if (r == QPM_OK) {
    e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) r = cuda_fail(e, "cudaStreamSynchronize");
  }
  cudaFree(dgenes);
  cudaFree(dd);
  cudaFree(df);
  qpm_destroy(st);
  return r;
}
