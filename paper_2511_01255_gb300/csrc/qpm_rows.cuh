// qpm_rows.cuh -- the row sweep shared by the fitness kernels of qpm_eval, qpm_eval_packed
// and the multi-wavelength objective.
//
// A warp takes 32 rows (lane = row) and walks a run of domains in index order, one block of
// 4 domains at a time: a block of +-1 domains takes one of 16 sign patterns and its monoid
// triple depends on the pattern only, so the sweep appends one table entry per block.  The
// global sign-block table (launch_block_table) holds the 8 patterns with d_0 = +1; staging a
// step of 128 domains in shared memory expands them to all 16 (the complement negates A and B),
// which costs a CTA a few stores per step and takes the fold of the pattern and the four sign
// flips out of every lane's block: 12 instructions a block and problem instead of 22-27.  The
// 16 entries of a block are 24 bytes apart and fall in distinct bank pairs, so a lookup is
// three conflict-free LDS.64.  The complex sums are packed FP32 pairs (add.rn.f32x2).
//
// Split of the work (RowPlan): the rows are taken in blocks of W groups of 32 (the W warps of
// a CTA, sharing one staged table), and the row blocks' sub-steps of 32 domains laid end to end
// are dealt to the CTAs as equal contiguous runs, a multiple of the resident CTAs, so that
// every SM ends at the same time whatever NP and N are.  A run that crosses the end of a row
// block becomes a piece of each.  The pieces of a row are combined in index order by the CTA that
// completes its row block, where they are few, else by a second kernel.
//
// What bounds it and what it measured (ncu, cold and serialised, against the form before it:
// 8-pattern table through cp.async, segments rounded to 128 domains, unaligned rows by 4-byte
// register loads):
//   5000 x 6601 unaligned rows   HBM (5.7 TB/s while the SMs are active): 35.6 -> 28.0 us
//   1024 x 1e5 packed signs      the shared-memory data path (70 % of its cycles): 31.6 -> 28.3 us
//                                (25.8 per call with the combining kernel, 36.9 before)
//   5000 x 3000, 3 problems      shared memory and HBM together: 28.2 -> 18.8 us
//   1024 x 1e5 aligned rows      HBM: 62.8 -> 65 us, and 4 us less for the combination
#pragma once
#include "qpm_common.cuh"
#include "qpm_internal.h"
#include "qpm_tma.cuh"

namespace qpm {

constexpr int RS_RING = 3;              // gene tiles per warp
constexpr int RS_ENTRY = 24;            // bytes of an entry (A, B, C as float2)
constexpr int RS_BLOCK = 16 * RS_ENTRY; // the 16 entries of a block of 4 domains
constexpr int RS_TAB = 32 * RS_BLOCK;   // a step of 128 domains, one problem: 12 KB
constexpr int RS_MAXSUB = 60;           // longest run in sub-steps (1920 domains: no plain FP32
                                        // partial sum of C exceeds about 1920^2 / 2 < 2^24)

// ------------------------------------------------------------------- the split
// first sub-step (of all row blocks laid end to end) of CTA x
__host__ __device__ __forceinline__ int64_t rp_start(const RowPlan &p, int64_t x) {
  return (int64_t)p.RB * p.nunit * x / p.C * p.gran;
}
// the CTA holding the first unit of row block b, and the number of pieces of row block b
__host__ __device__ __forceinline__ int rp_first(const RowPlan &p, int64_t unit) {
  return (int)(((unit + 1) * p.C - 1) / ((int64_t)p.RB * p.nunit));
}
__host__ __device__ __forceinline__ int rp_pieces(const RowPlan &p, int b) {
  return rp_first(p, (int64_t)(b + 1) * p.nunit - 1) - rp_first(p, (int64_t)b * p.nunit) + 1;
}

struct MonoP {
  f2x A, B, C;
};
// m (+) the entry at `e`: mono_combine's operations in its order
__device__ __forceinline__ void rs_push(MonoP &m, const unsigned char *e) {
  const f2x a = *(const f2x *)e, b = *(const f2x *)(e + 8);
  const float2 av = f2_unpack(a), B = f2_unpack(m.B);
  float2 c = f2_unpack(f2_add(m.C, *(const f2x *)(e + 16)));
  c.x = fmaf(av.x, B.x, c.x);
  c.x = fmaf(-av.y, B.y, c.x);
  c.y = fmaf(av.x, B.y, c.y);
  c.y = fmaf(av.y, B.x, c.y);
  m.C = f2_pack(c.x, c.y);
  m.A = f2_add(m.A, a);
  m.B = f2_add(m.B, b);
}

// Running monoid of a lane's row.  Plain: FP32 sums over a step of 128 domains, each step's
// then added to the run's (two short sums instead of one long one: 10 operations per 32 blocks
// for about the error of the shorter).  COMP: plain sums over 16 domains (4 sign blocks)
// Kahan-folded into a compensated triple.
template <bool COMP>
struct RowAcc {
  MonoP m;
  Mono o;
  MonoK k;
  __device__ __forceinline__ void zero() {
    m.A = m.B = m.C = 0ull;
    if (COMP) k = monok_zero();
    else o = mono_zero();
  }
  __device__ __forceinline__ Mono plain() const {
    Mono r;
    r.A = f2_unpack(m.A);
    r.B = f2_unpack(m.B);
    r.C = f2_unpack(m.C);
    return r;
  }
  __device__ __forceinline__ void fold() {  // every 4 blocks
    if (COMP) {
      monok_fold_in(k, plain());
      m.A = m.B = m.C = 0ull;
    }
  }
  __device__ __forceinline__ void step() {  // every 128 domains
    if (!COMP) {
      o = mono_combine(o, plain());
      m.A = m.B = m.C = 0ull;
    }
  }
  __device__ __forceinline__ Mono get() {  // after the last step()
    if (COMP) {
      fold();
      return monok_fold(k);
    }
    return o;
  }
};

// ------------------------------------------------------------- staged table steps
// The global entries of one step of one problem in the registers of a CTA of W warps: thread i
// holds entries i + j 32 W (entry = 8 * block + stored pattern), fetched a step ahead.
template <int W>
struct StepRegs {
  static constexpr int N = 256 / (32 * W);
  f2x a[N], b[N], c[N];
  // blocks from b0 on; zero past the problem's nb blocks
  __device__ __forceinline__ void load(const float2 *__restrict__ blk, int b0, int nb) {
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const int e = threadIdx.x + j * 32 * W, g = b0 + (e >> 3);
      a[j] = b[j] = c[j] = 0ull;
      if (g < nb) {
        const f2x *s = (const f2x *)(blk + (size_t)8 * 3 * b0) + 3 * e;
        a[j] = __ldg(s);
        b[j] = __ldg(s + 1);
        c[j] = __ldg(s + 2);
      }
    }
  }
  // stored pattern e is pattern 2 e; its complement 15 - 2 e has A and B negated
  __device__ __forceinline__ void store(unsigned char *tab) const {
    const f2x neg = 0x8000000080000000ull;
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const int e = threadIdx.x + j * 32 * W;
      unsigned char *t = tab + (e >> 3) * RS_BLOCK;
      f2x *p = (f2x *)(t + 2 * (e & 7) * RS_ENTRY);
      f2x *n = (f2x *)(t + (15 - 2 * (e & 7)) * RS_ENTRY);
      p[0] = a[j];
      p[1] = b[j];
      p[2] = c[j];
      n[0] = a[j] ^ neg;
      n[1] = b[j] ^ neg;
      n[2] = c[j];
    }
  }
};

// ------------------------------------------------------------------- gene tiles
// per-warp tile: 32 rows x 32 domains as float4 [row][c4], the column xor-swizzled by the row
// so that both the staging stores (8 columns of a row per quarter-warp) and the row walks (8
// rows of a column) are free of bank conflicts: the layout of a TMA copy's 128-byte swizzle
__device__ __forceinline__ int er_tix(int row, int c4) { return row * 8 + (c4 ^ (row & 7)); }

// sign pattern of 4 genes: bit j set iff gene j < 0 (d_j = -1; -0.0 and NaN count as +1)
__device__ __forceinline__ uint32_t er_pattern(const float4 &x) {
  return (x.x < 0.f ? 1u : 0u) | (x.y < 0.f ? 2u : 0u) | (x.z < 0.f ? 4u : 0u) |
         (x.w < 0.f ? 8u : 0u);
}
// byte offset of the pattern's entry within its block
__device__ __forceinline__ uint32_t er_offset(const float4 &x) {
  uint32_t o = x.x < 0.f ? 1u * RS_ENTRY : 0u;
  if (x.y < 0.f) o += 2u * RS_ENTRY;
  if (x.z < 0.f) o += 4u * RS_ENTRY;
  if (x.w < 0.f) o += 8u * RS_ENTRY;
  return o;
}

// How the genes reach the tiles.
//   ROWS_TMA    rows of 16-byte aligned pitch and base: one 32 x 32 TMA copy per sub-step
//   ROWS_TMA4   any other rows: rows r with the same r % 4 start at the same offset from a
//               16-byte boundary, so the four classes are four matrices of pitch 4 ld, each
//               mapped from the boundary below its first row (shift[c] = 0..3 floats before
//               it) and copied as four 8 x 32 boxes per sub-step.  Lane l walks the row 4 (l %
//               8) + l / 8 of its group, and a block's pattern is taken across two neighbouring
//               16-byte pieces.
enum { ROWS_TMA = 0, ROWS_TMA4 = 1 };
struct GeneMaps {
  CUtensorMap m[4];
  int shift[4];
};
// fills the maps of NP x N genes and the mode (host)
qpm_status make_gene_maps(GeneMaps *gm, int *mode, const float *genes, int NP, int N, int64_t ld);
template <int MODE>
__device__ __forceinline__ int rs_row_of_lane(int lane) {
  return MODE == ROWS_TMA4 ? 4 * (lane & 7) + (lane >> 3) : lane;
}

template <int K>
struct RowTables {
  const float2 *blk[K];  // sign-block tables (launch_block_table)
};

// dynamic shared memory: [gene tiles, 1024-byte aligned][2 steps of K tables][mbarriers]
__host__ __device__ constexpr size_t rs_smem(int K, int W) {
  return 1024 + (size_t)W * RS_RING * 4096 + 2 * (size_t)K * RS_TAB + (size_t)W * RS_RING * 8;
}
// resident CTAs per SM (shared memory; 227 KB less 1 KB reserved per CTA)
__host__ __device__ constexpr int rs_ctas(int K, int W) {
  const int n = (int)(232448 / (rs_smem(K, W) + 1024));
  return n < 1 ? 1 : n;
}

// ------------------------------------------------------ combination by the last CTA
// Most pieces of a row that the sweep combines itself: the combining kernel costs a call 4-6 us
// after the sweep (256 x 1000: 17.9 -> 7.4 us per call without it, together with the shorter host
// path), but one CTA's threads have the loads of about 16 pieces (6 registers each) in flight at a
// time, and rows cut finer than that are few and long, where the kernel spreads them over the GPU.
constexpr int RC_FUSE = 16;
// True in every thread of the CTA that is the last of the n to arrive at *ctr, which it leaves at 0 (the
// counter wraps), and then the others' partials are visible to it.  The counters are 0 between calls:
// they belong to one stream, whose calls follow one another, and captured calls use none.  (Words
// that need no state, tagged by each call, cost a call the look at them or the tag's write before
// the piece: 946 x 1106 11.1 us instead of 10.5, compensated 5000 x 1000 8.0 instead of 7.7; a flag
// per piece and a look at all of them 8.4; the arrival by compare-and-swap 11.1.)
__device__ __forceinline__ bool rows_last(unsigned *ctr, int n) {
  __shared__ unsigned last_sh;
  __syncthreads();
  if (n == 1) return true;
  if (threadIdx.x == 0) {
    __threadfence();
    last_sh = atomicInc(ctr, (unsigned)n - 1u) == (unsigned)n - 1u;
    __threadfence();
  }
  __syncthreads();
  return last_sh != 0u;
}
// thread = row of the row block: its P pieces (RC_FUSE at most), all loads of a problem in flight
// together, combined pairwise in index order (as accurate as a compensated chain at these
// lengths, and a fifth of its latency)
template <int K, class Close>
__device__ __forceinline__ void fused_combine(const RowPlan &pl, const float2 *part, int P, int row,
                                              Close &&close) {
  if (row >= pl.NP) return;
  const size_t NPp = pl.NPpad;
  Mono m[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    Mono r[RC_FUSE];
#pragma unroll
    for (int p = 0; p < RC_FUSE; ++p) {
      r[p] = mono_zero();
      if (p < P) {
        const float2 *q = part + ((size_t)K * p + k) * 3 * NPp + row;
        r[p].A = __ldcg(q);
        r[p].B = __ldcg(q + NPp);
        r[p].C = __ldcg(q + 2 * NPp);
      }
    }
#pragma unroll
    for (int s = 1; s < RC_FUSE; s <<= 1)
#pragma unroll
      for (int p = 0; p < RC_FUSE; p += 2 * s) r[p] = mono_combine(r[p], r[p + s]);
    m[k] = r[0];
  }
  close(row, m);
}

// Sweep of float genes.  Sub-step u's tile is issued RS_RING - 1 sub-steps ahead into the slot
// its predecessor has left, on the slot's mbarrier; the tables' steps come a step ahead through
// registers behind one CTA barrier per step.  A wait on an mbarrier is bounded (%globaltimer);
// one that runs out makes the rows' results NaN and stops the warp's copies.
// Partials: part[((piece K + k) 3 + {A, B, C}) NPpad + row].
// ctr (with a plan of at most RC_FUSE pieces a row): the CTA that completes a row block, found by
// the block's counter (rows_last), combines it and calls close(row, the K monoids).  (As a form of
// its own the sweep without it has 126 registers instead of 156 with one table, which gave 1024 x 1e5
// 0.3 us of 67.9 and cost 64 x 1e5 1.1 us of 10.8.)
template <int K, int W, int MODE, bool COMP, class Close>
__device__ __forceinline__ void rows_sweep(const GeneMaps &maps, const float *__restrict__ src,
                                           int64_t ld, const RowPlan &pl, const RowTables<K> &tabs,
                                           float2 *part, unsigned *ctr, Close &&close) {
  extern __shared__ unsigned char rs_raw[];
  unsigned char *base = rs_raw + ((1024 - (smem_u32(rs_raw) & 1023)) & 1023);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float4 *ring = (float4 *)base + warp * (RS_RING * 256);
  unsigned char *tab = base + (size_t)W * RS_RING * 4096;
  const unsigned bar0 = smem_u32(tab + 2 * (size_t)K * RS_TAB) + warp * RS_RING * 8;
  const int nb = (pl.N + 3) >> 2;
  const int my = rs_row_of_lane<MODE>(lane);
  const int sft = MODE == ROWS_TMA4 ? maps.shift[lane >> 3] : 0;
  // the next phase may be scheduled as this grid's CTAs retire
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (lane == 0) {
    for (int k = 0; k < RS_RING; ++k) mbar_init(bar0 + 8 * k, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
  }
  // the kernel before (which may still be reading the partials, or writing genes or tables)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  bool ok = true;
  int done = 0;    // tiles consumed by this warp so far (all pieces): slot done % RS_RING
  int issued = 0;  // tiles issued so far
  int failed = 0;  // done when a wait ran out
  auto issue = [&](int n, int m, int r0) {  // tile n of this warp: domains m .. m + 31
    const unsigned bar = bar0 + 8 * (n % RS_RING);
    float4 *dst = ring + (n % RS_RING) * 256;
    if (lane == 0) {
      fence_async_smem();
      mbar_expect_tx(bar, 4096);
      if constexpr (MODE == ROWS_TMA) {
        tma_load_tile(dst, &maps.m[0], m, r0, bar);
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) tma_load_tile(dst + 64 * c, &maps.m[c], m, r0 >> 2, bar);
      }
    }
    ++issued;
  };
  auto arrived = [&](int n) {
    const bool a = ok && mbar_wait(bar0 + 8 * (n % RS_RING), (n / RS_RING) & 1);
    if (ok) failed = n;
    ok = __all_sync(0xffffffffu, a);
  };
  const int64_t f1 = min(rp_start(pl, (int64_t)blockIdx.x + 1), (int64_t)pl.RB * pl.nunit * pl.gran);
  const int64_t per = (int64_t)pl.nunit * pl.gran;  // sub-steps of a row block (the last may be empty)
  for (int64_t f = rp_start(pl, blockIdx.x); f < f1;) {
    const int b = (int)(f / per), u0 = (int)(f - b * per);
    const int u1 = (int)min(per, (int64_t)u0 + (f1 - f));
    f += u1 - u0;
    const int m0 = 32 * u0, nsub = min(u1, pl.nsub) - u0;
    const int nsteps = (nsub + 3) >> 2;
    const int r0 = (b * W + warp) * 32;
    const bool live = r0 < pl.NP;
    const int row = r0 + my;
    StepRegs<W> R[K];
#pragma unroll
    for (int p = 0; p < K; ++p) R[p].load(tabs.blk[p], m0 >> 2, nb);
    uint32_t tail = 0;  // ROWS_TMA4: pattern of the row's first domains past the last tile
    if (live) {
#pragma unroll
      for (int u = 0; u < RS_RING - 1; ++u)
        if (ok && u < nsub) issue(done + u, m0 + 32 * u, r0);
      if constexpr (MODE == ROWS_TMA4) {
        // the row's last sft columns lie past the last tile: its domains d0 .. d0 + sft - 1
        const int64_t d0 = 32 * (int64_t)(u0 + nsub) - sft;
#pragma unroll
        for (int q = 0; q < 3; ++q)
          if (q < sft && row < pl.NP && d0 + q < pl.N && src[(int64_t)row * ld + d0 + q] < 0.f)
            tail |= 1u << q;
      }
    }
    __syncthreads();  // the table buffers of the piece before are free
#pragma unroll
    for (int p = 0; p < K; ++p) {
      R[p].store(tab + p * RS_TAB);
      if (nsteps > 1) R[p].load(tabs.blk[p], (m0 >> 2) + 32, nb);
    }
    RowAcc<COMP> acc[K];
#pragma unroll
    for (int p = 0; p < K; ++p) acc[p].zero();
    uint32_t pat = 0;  // ROWS_TMA4: pattern of the next 16-byte piece
    for (int k = 0; k < nsteps; ++k) {
      __syncthreads();  // step k is staged; everyone is done with step k - 1
      if (live && ok && 4 * k + RS_RING - 1 < nsub)
        issue(done + RS_RING - 1, m0 + 32 * (4 * k + RS_RING - 1), r0);
      if (k + 1 < nsteps) {
#pragma unroll
        for (int p = 0; p < K; ++p) {
          R[p].store(tab + (((k + 1) & 1) * K + p) * RS_TAB);
          if (k + 2 < nsteps) R[p].load(tabs.blk[p], (m0 >> 2) + 32 * (k + 2), nb);
        }
      }
      if (!live) continue;
      const unsigned char *bp = tab + (size_t)(k & 1) * K * RS_TAB;
#pragma unroll 1
      for (int q = 0; q < 4; ++q) {  // 4 sub-steps of 32 domains
        const int u = 4 * k + q;
        if (u >= nsub) break;
        const float4 *T = ring + (done % RS_RING) * 256;
        __syncwarp();  // the warp's lanes are done with the tile before
        if (q > 0 && ok && u + RS_RING - 1 < nsub)
          issue(done + RS_RING - 1, m0 + 32 * (u + RS_RING - 1), r0);
        if (MODE == ROWS_TMA || u == 0) arrived(done);
        const unsigned char *E = bp + q * (8 * RS_BLOCK);
        if constexpr (MODE == ROWS_TMA4) {
          if (u == 0) pat = er_pattern(T[er_tix(lane, 0)]);
          uint32_t last = tail;  // the pattern after this tile's 8 pieces
          if (u + 1 < nsub) {
            arrived(done + 1);
            last = er_pattern((ring + ((done + 1) % RS_RING) * 256)[er_tix(lane, 0)]);
          }
#pragma unroll
          for (int c4 = 0; c4 < 8; ++c4) {
            const uint32_t nxt = c4 < 7 ? er_pattern(T[er_tix(lane, c4 < 7 ? c4 + 1 : 7)]) : last;
            const uint32_t e = (((nxt << 4) | pat) >> sft) & 15u;
            pat = nxt;
#pragma unroll
            for (int p = 0; p < K; ++p) {
              rs_push(acc[p].m, E + p * RS_TAB + c4 * RS_BLOCK + e * RS_ENTRY);
              if ((c4 & 3) == 3) acc[p].fold();
            }
          }
        } else {
#pragma unroll
          for (int c4 = 0; c4 < 8; ++c4) {
            const uint32_t o = er_offset(T[er_tix(lane, c4)]);
#pragma unroll
            for (int p = 0; p < K; ++p) {
              rs_push(acc[p].m, E + p * RS_TAB + c4 * RS_BLOCK + o);
              if ((c4 & 3) == 3) acc[p].fold();
            }
          }
        }
        ++done;
      }
#pragma unroll
      for (int p = 0; p < K; ++p) acc[p].step();
    }
    const int piece = (int)blockIdx.x - rp_first(pl, (int64_t)b * pl.nunit);
    if (live && row < pl.NP) {
#pragma unroll
      for (int p = 0; p < K; ++p) {
        Mono m = acc[p].get();
        if (!ok) m.A.x = m.A.y = m.B.x = m.B.y = m.C.x = m.C.y = __int_as_float(0x7fc00000);
        float2 *o = part + ((size_t)piece * K + p) * 3 * pl.NPpad + row;
        o[0] = m.A;
        o[pl.NPpad] = m.B;
        o[2 * (size_t)pl.NPpad] = m.C;
      }
    }
    if (ctr) {
      const int P = rp_pieces(pl, b);
      if (rows_last(ctr + b, P)) fused_combine<K>(pl, part, P, b * W * 32 + (int)threadIdx.x, close);
    }
  }
  if (!ok && lane == 0) {  // copies of a failed warp may still be in flight
    for (int n = failed; n < issued; ++n) mbar_wait(bar0 + 8 * (n % RS_RING), (n / RS_RING) & 1);
  }
}

// ------------------------------------------------------------------- combination
// The pieces of every row, combined in index order: a CTA of 256 threads takes 256 / runs rows,
// `runs` threads a row, each a contiguous run of pieces, then a pairwise tree over the runs.  A
// run is combined pairwise in groups whose loads are in flight together; where it has several
// groups they are summed compensated.  (Compensated from piece to piece, 1024 x 1e5 packed signs
// took 26.4 us per call instead of 25.8, for the same error against 64 bits.)  Up to RC_FUSE pieces
// it is fused_combine's tree, so a row has the same bits either way.
// Latency-bound (a few L2 round trips), so runs
// grows with the pieces: 2 to 4 pieces a thread, 8 rows a CTA at the most pieces.
constexpr int RC_THREADS = 256;
inline int rc_runs(const RowPlan &p) {
  int r = 4;
  while (r < 32 && 2 * r < p.P) r *= 2;
  return r;
}
// K monoids of row `row` (valid in run 0); sh: K x 256 monoids
template <int K>
__device__ __forceinline__ void combine_pieces(const RowPlan &pl, const float2 *__restrict__ part,
                                               int runs, int row, int run, Mono (*sh)[RC_THREADS],
                                               Mono out[K]) {
  const int P = rp_pieces(pl, min(row, pl.NP - 1) / (pl.W * 32));
  const int c = (P + runs - 1) / runs;
  const int p0 = run * c, p1 = min(P, p0 + c);
  const size_t NPp = pl.NPpad;
  MonoK acc[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    acc[k] = monok_zero();
    out[k] = mono_zero();
  }
  constexpr int U = K == 1 ? 4 : 2;  // pieces whose loads are in flight together
  for (int p = p0; p < p1; p += U) {
    Mono r[U][K];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const float2 *q = part + (size_t)3 * K * NPp * min(p + u, P - 1) + min(row, pl.NP - 1);
#pragma unroll
      for (int k = 0; k < K; ++k) {
        r[u][k].A = __ldcg(q + 3 * k * NPp);
        r[u][k].B = __ldcg(q + (3 * k + 1) * NPp);
        r[u][k].C = __ldcg(q + (3 * k + 2) * NPp);
      }
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
#pragma unroll
      for (int u = 1; u < U; ++u)
        if (p + u >= p1) r[u][k] = mono_zero();
#pragma unroll
      for (int s = 1; s < U; s <<= 1)
#pragma unroll
        for (int u = 0; u < U; u += 2 * s) r[u][k] = mono_combine(r[u][k], r[u + s][k]);
      if (c <= U) out[k] = r[0][k];
      else monok_fold_in(acc[k], r[0][k]);
    }
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    if (c > U) out[k] = monok_fold(acc[k]);
    sh[k][threadIdx.x] = out[k];
  }
  const int rows = RC_THREADS / runs;  // thread = run * rows + row of the CTA
  for (int s = 1; s < runs; s <<= 1) {
    __syncthreads();
    if ((run & (2 * s - 1)) == 0) {
#pragma unroll
      for (int k = 0; k < K; ++k) {
        out[k] = mono_combine(out[k], sh[k][threadIdx.x + s * rows]);
        sh[k][threadIdx.x] = out[k];
      }
    }
  }
}

}  // namespace qpm
