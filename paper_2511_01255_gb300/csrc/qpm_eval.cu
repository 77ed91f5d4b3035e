// qpm_eval.cu -- fitness of caller-supplied sign sequences (Sec. 2.1).
//
// The row sweep of qpm_rows.cuh with one sign-block table: a warp takes 32 rows (lane = row) and
// appends one table entry per block of 4 domains.  Float genes arrive as 32 x 32 tiles by TMA
// (rows of any alignment, see GeneMaps) and are transposed through the tile; packed sign words
// (32 domains each) are read four at a time straight into the lane of their row.  A second kernel
// combines the pieces of every row in index order and closes d_eff = phi1 phi2 C + cdiag.
#include <math.h>

#include <algorithm>
#include <atomic>
#include <map>
#include <mutex>
#include <new>
#include <string.h>

#include <string>
#include <tuple>

#include "qpm_common.cuh"
#include "qpm_internal.h"
#include "qpm_rows.cuh"

namespace qpm {

// Resident CTAs of the packed sweep per SM: 3 of 8 warps, whose 80 registers hold the lookups of
// several blocks in flight (1024 x 1e5, per call: 26.4 us with the combination of then; 4 of them
// at 64 registers 30.0, 2 at 115 registers 28.0; 4-warp CTAs 28.8-37.1), or 8 of 2 warps (up to
// 64 rows).
constexpr int ep_ctas(int W) { return W == 8 ? 3 : 8; }

// float genes: see rows_sweep; ctr not NULL: the sweep combines the rows itself
template <int W, int MODE, bool COMP>
static __global__ void __launch_bounds__(W * 32, rs_ctas(1, W))
    k_eval_genes(const __grid_constant__ GeneMaps maps, const float *__restrict__ src, int64_t ld,
                 RowPlan pl, RowTables<1> tabs, float2 *part, unsigned *ctr,
                 const float2 *__restrict__ konst, float2 *__restrict__ deff,
                 float *__restrict__ fit) {
  rows_sweep<1, W, MODE, COMP>(maps, src, ld, pl, tabs, part, ctr, [&](int row, const Mono *m) {
    const float2 D = deff_from(m[0], konst[0], konst[1]);
    deff[row] = D;
    if (fit) fit[row] = fit_of(D);
  });
}

// Packed sign words.  Bound by the shared-memory data path (a lookup returns 24 bytes a lane: 6
// cycles of the SM's 128 bytes per block of 4 domains and warp), so the rest is kept below it:
// the 8 nibbles of a word cost one byte permute and one multiply each, and the 16-pattern table
// needs no sign flips.  Units of 128 domains (a word quadruple, 16-byte loads when VECW).
template <int W, bool VECW, bool COMP>
static __global__ void __launch_bounds__(W * 32, ep_ctas(W))
    k_eval_packed(const uint32_t *__restrict__ src, int64_t ld, RowPlan pl, RowTables<1> tabs,
                  float2 *__restrict__ part) {
  __shared__ __align__(16) unsigned char tab[2 * RS_TAB];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nb = (pl.N + 3) >> 2, nw = (pl.N + 31) >> 5;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");  // genes, tables, the partials' last readers
  const int64_t per = (int64_t)pl.nunit * pl.gran;
  const int64_t f1 = rp_start(pl, (int64_t)blockIdx.x + 1);
  for (int64_t f = rp_start(pl, blockIdx.x); f < f1;) {
    const int b = (int)(f / per), u0 = (int)(f - b * per);
    const int u1 = (int)min(per, (int64_t)u0 + (f1 - f));
    f += u1 - u0;
    const int row = (b * W + warp) * 32 + lane, rr = min(row, pl.NP - 1);
    const bool live = (b * W + warp) * 32 < pl.NP;
    const int w0 = u0, nsteps = (min(u1, pl.nsub) - u0 + 3) >> 2;  // u0 is a multiple of 4
    const uint32_t *rp = src + (int64_t)rr * ld;
    // words past the row's last are never read; their blocks have zero entries
    auto words = [&](int w) {
      if (VECW && w + 4 <= nw) return __ldg((const uint4 *)(rp + w));
      return make_uint4(__ldg(rp + min(w, nw - 1)), __ldg(rp + min(w + 1, nw - 1)),
                        __ldg(rp + min(w + 2, nw - 1)), __ldg(rp + min(w + 3, nw - 1)));
    };
    StepRegs<W> R;
    R.load(tabs.blk[0], 8 * w0, nb);
    uint4 nxt = words(w0);
    __syncthreads();  // the table buffers of the piece before are free
    R.store(tab);
    if (nsteps > 1) R.load(tabs.blk[0], 8 * w0 + 32, nb);
    RowAcc<COMP> acc;
    acc.zero();
    for (int k = 0; k < nsteps; ++k) {
      __syncthreads();  // step k is staged; everyone is done with step k - 1
      if (k + 1 < nsteps) {
        R.store(tab + ((k + 1) & 1) * RS_TAB);
        if (k + 2 < nsteps) R.load(tabs.blk[0], 8 * w0 + 32 * (k + 2), nb);
      }
      if (!live) continue;
      const uint32_t ws[4] = {nxt.x, nxt.y, nxt.z, nxt.w};
      if (k + 1 < nsteps) nxt = words(w0 + 4 * (k + 1));
      const unsigned char *E = tab + (k & 1) * RS_TAB;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t lo = ws[q] & 0x0F0F0F0Fu, hi = (ws[q] >> 4) & 0x0F0F0F0Fu;
#pragma unroll
        for (int j = 0; j < 8; ++j) {  // the word's 8 blocks of 4 domains
          const uint32_t e = __byte_perm((j & 1) ? hi : lo, 0u, 0x4440u + (j >> 1));
          rs_push(acc.m, E + (8 * q + j) * RS_BLOCK + e * RS_ENTRY);
          if ((j & 3) == 3) acc.fold();
        }
      }
      acc.step();
    }
    if (row < pl.NP) {
      const int piece = (int)blockIdx.x - rp_first(pl, (int64_t)b * pl.nunit);
      const Mono m = acc.get();
      float2 *o = part + (size_t)piece * 3 * pl.NPpad + row;
      o[0] = m.A;
      o[pl.NPpad] = m.B;
      o[2 * (size_t)pl.NPpad] = m.C;
    }
  }
}

// d_eff = phi1 phi2 C + cdiag of the combined pieces; a programmatic dependent of the sweep
static __global__ void __launch_bounds__(RC_THREADS)
    k_eval_combine(RowPlan pl, int runs, const float2 *__restrict__ part,
                   const float2 *__restrict__ konst, float2 *__restrict__ deff,
                   float *__restrict__ fit) {
  __shared__ Mono sh[1][RC_THREADS];
  const int rows = RC_THREADS / runs, run = threadIdx.x / rows;
  const int row = blockIdx.x * rows + threadIdx.x - run * rows;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  Mono acc[1];
  combine_pieces<1>(pl, part, runs, row, run, sh, acc);
  if (run == 0 && row < pl.NP) {
    const float2 D = deff_from(acc[0], konst[0], konst[1]);
    deff[row] = D;
    if (fit) fit[row] = fit_of(D);
  }
}

// ------------------------------------------------------------- caches (host)
namespace {
// Device memory of the library that graphs may hold too: a captured call's nodes have its address
// for as long as the graph or an executable instance of it lives, so a user object of the graph
// counts it in `graphs`, and memory that is held is retired instead of freed.
struct DevMem {
  int dev = 0;
  void *p[4] = {nullptr, nullptr, nullptr, nullptr};  // a table: phasors, partials, constants, sign blocks
  size_t bytes = 0;                                   // scratch: of p[0]
  unsigned long long capture = 0;                     // the last capture that took hold of it
  cudaStream_t stream = nullptr;                      // scratch: the stream captured
  std::atomic<int> graphs{0};
  DevMem *next = nullptr;  // in g_kept
};
struct TableEntry {
  DevMem *mem = nullptr;
  cudaEvent_t ready = nullptr;
  bool built = false;  // `ready` was seen complete: no stream needs to wait for it any more
  cudaEvent_t blk_ready = nullptr;  // of the sign-block table, built on the first call that needs it
  bool blk_built = false;
};
struct ScratchEntry {
  void *ptr = nullptr;  // FUSE_BLOCKS counters, then partial sums
  size_t bytes = 0;
};
std::mutex g_mu;
std::map<std::tuple<int, int32_t, double, double>, TableEntry> g_tables;
// per (device, stream, thread's stream): the handle cudaStreamPerThread names another stream in each
// thread, which its id tells apart (0 for the others: a destroyed stream's handle does not come back
// before its work is done)
std::map<std::tuple<int, cudaStream_t, unsigned long long>, ScratchEntry> g_scratch;
constexpr size_t MAX_THREADS = 64;  // threads whose scratch is kept per device
DevMem *g_kept = nullptr;  // captured calls' scratch, and tables no longer cached that graphs held
constexpr size_t MAX_TABLES = 64;  // captured calls, which evict nothing, may add as many again

// This thread's calls that are not allowed beside a capture in the global or thread-local mode
// (allocations, event queries; a forbidden one would end that capture) are made in the relaxed one.
struct RelaxedMode {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  RelaxedMode() { cudaThreadExchangeStreamCaptureMode(&mode); }
  ~RelaxedMode() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

void free_mem(DevMem *m) {
  for (void *q : m->p)
    if (q) cudaFree(q);
  delete m;
}

void keep(DevMem *m) {
  m->next = g_kept;
  g_kept = m;
}

// the kept memory of `dev` whose graphs are all gone
void free_unheld(int dev) {
  for (DevMem **q = &g_kept; *q;) {
    DevMem *m = *q;
    if (m->dev == dev && m->graphs.load(std::memory_order_acquire) == 0) {
      *q = m->next;
      free_mem(m);
    } else {
      q = &m->next;
    }
  }
}

void CUDART_CB drop_hold(void *m) {  // on a thread of CUDA's: no CUDA call
  static_cast<DevMem *>(m)->graphs.fetch_sub(1, std::memory_order_release);
}

// the capture's graph holds m from here on
qpm_status hold(DevMem *m, const Capture &cap) {
  if (m->capture == cap.id && m->graphs.load(std::memory_order_relaxed) > 0) return QPM_OK;
  cudaUserObject_t obj;
  QPM_CUDA(cudaUserObjectCreate(&obj, m, drop_hold, 1, cudaUserObjectNoDestructorSync));
  m->graphs.fetch_add(1, std::memory_order_relaxed);
  const cudaError_t e = cudaGraphRetainUserObject(cap.graph, obj, 1, cudaGraphUserObjectMove);
  if (e != cudaSuccess) {
    cudaUserObjectRelease(obj, 1);
    return cuda_fail(e, "cudaGraphRetainUserObject");
  }
  m->capture = cap.id;
  return QPM_OK;
}

void drop_entry(TableEntry &e) {
  if (e.ready) cudaEventDestroy(e.ready);
  if (e.blk_ready) cudaEventDestroy(e.blk_ready);
  if (e.mem && e.mem->graphs.load(std::memory_order_acquire) > 0) keep(e.mem);
  else if (e.mem) free_mem(e.mem);
}

// frees the scratch of `dev`, of its per-thread streams only if so asked (the device is idle)
void drop_scratch(int dev, bool threads_only) {
  for (auto it = g_scratch.begin(); it != g_scratch.end();) {
    if (std::get<0>(it->first) == dev && (!threads_only || std::get<2>(it->first) != 0)) {
      cudaFree(it->second.ptr);
      it = g_scratch.erase(it);
    } else {
      ++it;
    }
  }
}

qpm_status release_device_caches(int dev) {
  QPM_CUDA(cudaDeviceSynchronize());
  for (auto it = g_tables.begin(); it != g_tables.end();) {
    if (std::get<0>(it->first) == dev) {
      drop_entry(it->second);
      it = g_tables.erase(it);
    } else {
      ++it;
    }
  }
  drop_scratch(dev, false);
  free_unheld(dev);
  return QPM_OK;
}

size_t device_table_count(int dev) {
  size_t n = 0;
  for (const auto &kv : g_tables) n += (std::get<0>(kv.first) == dev);
  return n;
}

// `stream` waits for `ev`, unless it was seen complete (a wait costs every call about 0.4 us of host
// time); a captured call, which cannot wait for an event from outside its graph, waits here.
qpm_status wait_built(cudaStream_t stream, const Capture &cap, cudaEvent_t ev, bool &built) {
  if (built) return QPM_OK;
  {
    RelaxedMode relaxed;
    cudaError_t e = cudaEventQuery(ev);
    if (e == cudaErrorNotReady && cap.graph) e = cudaEventSynchronize(ev);
    built = e == cudaSuccess;
  }
  if (built) return QPM_OK;
  cudaGetLastError();  // not ready
  QPM_CUDA(cudaStreamWaitEvent(stream, ev, 0));
  return QPM_OK;
}

// Runs build(stream) and records its end: on the caller's stream, `ready` behind it; in a captured
// call on a stream outside the capture, complete on return (built; no event).
template <class F>
qpm_status build_table(cudaStream_t stream, const Capture &cap, cudaEvent_t *ready, bool *built, F &&build) {
  cudaError_t e;
  qpm_status st;
  if (cap.graph) {
    cudaStream_t side = nullptr;
    QPM_CUDA(cudaStreamCreateWithFlags(&side, cudaStreamNonBlocking));
    st = build(side);
    e = cudaStreamSynchronize(side);
    cudaStreamDestroy(side);
    if (st == QPM_OK && e != cudaSuccess) st = cuda_fail(e, "building a phasor table");
    *built = st == QPM_OK;
    return st;
  }
  QPM_CUDA(cudaEventCreateWithFlags(ready, cudaEventDisableTiming));
  st = build(stream);
  if (st == QPM_OK && (e = cudaEventRecord(*ready, stream)) != cudaSuccess) st = cuda_fail(e, "cudaEventRecord");
  return st;
}

// phasor table in natural order for (device, problem); built on a miss.
// blk (if non-NULL) receives the sign-block table, built the first time it is asked for.
// Never evicts: TableLease makes room before its first lookup.  A captured call's graph holds
// what it is given; where the cache is full its tables are the graph's alone.
// Caller holds g_mu.
qpm_status get_table(int dev, const qpm_problem *p, cudaStream_t stream, const Capture &cap,
                     const float4 **table, const float2 **konst, const float2 **blk = nullptr) {
  auto key = std::make_tuple(dev, p->N, p->kappa1, p->kappa2);
  auto it = g_tables.find(key);
  TableEntry own;
  const bool hit = it != g_tables.end(), cached = hit || !cap.graph || device_table_count(dev) < 2 * MAX_TABLES;
  TableEntry &e = hit ? it->second : own;
  if (!hit) {
    RelaxedMode relaxed;
    const int32_t Npad = (p->N + 3) & ~3;
    e.mem = new (std::nothrow) DevMem;
    if (!e.mem) return fail(QPM_ERR_CUDA, "out of host memory");
    e.mem->dev = dev;
    cudaError_t ce = cudaMalloc(&e.mem->p[0], sizeof(float4) * (size_t)Npad);
    if (ce == cudaSuccess) ce = cudaMalloc(&e.mem->p[1], sizeof(double2) * (size_t)table_part_count(Npad));
    if (ce == cudaSuccess) ce = cudaMalloc(&e.mem->p[2], sizeof(float2) * 4);
    qpm_status st = ce == cudaSuccess ? QPM_OK : cuda_fail(ce, "allocating a phasor table");
    if (st == QPM_OK)
      st = build_table(stream, cap, &e.ready, &e.built, [&](cudaStream_t s) {
        TableSpec ts{p->N, Npad, 1, Npad, p->kappa1, p->kappa2};
        return launch_table(ts, (float4 *)e.mem->p[0], (double2 *)e.mem->p[1], (float2 *)e.mem->p[2],
                            nullptr, s);
      });
    if (st != QPM_OK) {  // the cache keeps no half-built entry
      drop_entry(e);
      return st;
    }
  } else {
    const qpm_status st = wait_built(stream, cap, e.ready, e.built);
    if (st != QPM_OK) return st;
  }
  qpm_status st = QPM_OK;
  if (blk && !e.mem->p[3]) {
    RelaxedMode relaxed;
    void *b = nullptr;
    const cudaError_t ce = cudaMalloc(&b, sizeof(float2) * BLK_F2 * ((size_t)(p->N + 3) / 4));
    st = ce == cudaSuccess ? build_table(stream, cap, &e.blk_ready, &e.blk_built,
                                         [&](cudaStream_t s) {
                                           return launch_block_table(p->N, p->kappa1, p->kappa2,
                                                                     (float2 *)b, s);
                                         })
                           : cuda_fail(ce, "allocating a sign-block table");
    if (st == QPM_OK) {
      e.mem->p[3] = b;
    } else {  // the entry keeps no half-built table
      if (b) cudaFree(b);
      if (e.blk_ready) cudaEventDestroy(e.blk_ready);
      e.blk_ready = nullptr;
    }
  } else if (blk) {
    st = wait_built(stream, cap, e.blk_ready, e.blk_built);
  }
  if (st == QPM_OK && cap.graph) st = hold(e.mem, cap);
  DevMem *const m = e.mem;
  if (!hit && cached) g_tables.emplace(key, e);
  else if (!hit && st == QPM_OK) keep(m);
  else if (!hit) drop_entry(e);
  if (st != QPM_OK) return st;
  *table = (const float4 *)m->p[0];
  *konst = (const float2 *)m->p[2];
  if (blk) *blk = (const float2 *)m->p[3];
  return QPM_OK;
}

// Scratch of a stream that is not being captured, so that clearing the counters runs here and now.
qpm_status get_scratch(int dev, cudaStream_t stream, size_t bytes, void **ptr) {
  unsigned long long id = 0;
  if (stream == cudaStreamPerThread) {
    QPM_CUDA(cudaStreamGetId(stream, &id));
    size_t n = 0;
    for (const auto &kv : g_scratch) n += std::get<0>(kv.first) == dev && std::get<2>(kv.first) != 0;
    if (n >= MAX_THREADS && !g_scratch.count(std::make_tuple(dev, stream, id))) {
      QPM_CUDA(cudaDeviceSynchronize());
      drop_scratch(dev, true);
    }
  }
  ScratchEntry &e = g_scratch[std::make_tuple(dev, stream, id)];
  if (e.bytes < bytes) {
    if (e.ptr) {
      QPM_CUDA(cudaStreamSynchronize(stream));
      QPM_CUDA(cudaFree(e.ptr));
      e.ptr = nullptr;
      e.bytes = 0;
    }
    free_unheld(dev);
    QPM_CUDA(cudaMalloc(&e.ptr, bytes));
    const cudaError_t ce = cudaMemsetAsync(e.ptr, 0, FUSE_BYTES, stream);
    if (ce != cudaSuccess) {  // no scratch without its counters
      cudaFree(e.ptr);
      e.ptr = nullptr;
      return cuda_fail(ce, "clearing the scratch counters");
    }
    e.bytes = bytes;
  }
  *ptr = e.ptr;
  return QPM_OK;
}

// Scratch of a captured call: never the stream's own, which later calls use and may replace.  The
// calls captured on one stream in one capture run one after the other and share a block; other
// captures get another, new or of graphs that are gone.
qpm_status graph_scratch(int dev, cudaStream_t stream, const Capture &cap, size_t bytes, void **ptr) {
  DevMem *best = nullptr;
  for (DevMem *m = g_kept; m; m = m->next) {
    if (m->dev != dev || m->bytes < bytes) continue;
    const bool held = m->graphs.load(std::memory_order_acquire) > 0;
    if (held && m->capture == cap.id && m->stream == stream) {
      *ptr = m->p[0];
      return QPM_OK;
    }
    if (!held && (!best || m->bytes < best->bytes)) best = m;
  }
  if (!best) {
    RelaxedMode relaxed;
    free_unheld(dev);
    best = new (std::nothrow) DevMem;
    if (!best) return fail(QPM_ERR_CUDA, "out of host memory");
    best->dev = dev;
    const cudaError_t e = cudaMalloc(&best->p[0], bytes);
    if (e != cudaSuccess) {
      delete best;
      return cuda_fail(e, "allocating the scratch of a captured call");
    }
    best->bytes = bytes;
    keep(best);
  }
  best->stream = stream;
  const qpm_status st = hold(best, cap);
  if (st == QPM_OK) *ptr = best->p[0];
  return st;
}
}  // namespace

// a row block of nunit units touches at most this many runs of floor(units / C) or more units
static int row_pieces(const RowPlan &p) {
  const int64_t q = std::max<int64_t>(1, (int64_t)p.RB * p.nunit / p.C);
  return (int)std::min<int64_t>(std::min<int64_t>(p.nunit, p.C), (p.nunit + q - 1) / q + 1);
}

RowPlan row_plan(int NP, int N, int W, int64_t full, int gran, int maxsub, int min_units) {
  RowPlan p;
  p.NP = NP;
  p.N = N;
  const int groups = (NP + 31) / 32;
  p.NPpad = groups * 32;
  p.W = W;
  p.RB = (groups + W - 1) / W;
  p.nsub = (N + 31) / 32;
  p.gran = gran;
  p.nunit = (p.nsub + gran - 1) / gran;
  const int64_t tot = (int64_t)p.RB * p.nunit;
  // whole rounds of the resident CTAs, as few as keep every run within maxsub
  const int64_t rounds = (tot * gran + full * maxsub - 1) / (full * maxsub);
  int64_t C = std::max<int64_t>(1, rounds) * full;
  C = std::min(C, std::max<int64_t>(1, tot / min_units));
  p.C = (int)C;
  p.P = row_pieces(p);
  return p;
}

// Warps per CTA.  One table: 4 (12 warps an SM in 3 CTAs); a single group of rows: 1 (5 warps an
// SM, where 4 would keep 3 alive).  K tables: 8 warps share the staged steps (8 warps an SM),
// or 2 where that keeps more warps alive (few row groups).
static int genes_warps(int K, int NP) {
  const int g = (NP + 31) / 32, few = K == 1 ? 1 : 2, many = K == 1 ? 4 : 8;
  auto alive = [&](int W) {  // live warps per SM
    return (double)W * rs_ctas(K, W) * g / ((g + W - 1) / W * W);
  };
  return alive(few) > alive(many) ? few : many;
}
RowPlan genes_plan(int K, int NP, int N, bool aligned, bool whole) {
  const int W = genes_warps(K, NP);
  if (!whole) {
    const int full = rs_ctas(K, W) * sm_count();
    RowPlan p = row_plan(NP, N, W, full, 1, RS_MAXSUB, 4);
    // Whole rounds of CTAs, all in step, lose to runs of the full length where a few row blocks of
    // very long aligned rows need three rounds or more (one table): 256 x 1e6 215 us against 194,
    // 512 x 600000 232 / 208, 128 x 2e6 220 / 196, 64 x 3e6 179 / 165, 512 x 1e6 363 / 372.  Not with
    // rows of odd pitch (256 x 1e6 185 / 212), more row blocks (1024 x 250000 168 / 184) or two rounds
    // (1024 x 131072 89 / 110).
    if (K == 1 && aligned && p.RB <= 4 && p.C > 2 * full) {
      p.C = p.RB * ((p.nunit + RS_MAXSUB - 1) / RS_MAXSUB);
      p.P = row_pieces(p);
    }
    return p;
  }
  // runs of whole rows, cut only where a row is longer than a run may be
  const int nsub = (N + 31) / 32, runs = (nsub + RS_MAXSUB - 1) / RS_MAXSUB;
  RowPlan p = row_plan(NP, N, W, 1, (nsub + runs - 1) / runs, nsub, 1);
  p.C = p.RB * p.nunit;
  p.P = p.nunit;
  return p;
}
static RowPlan packed_plan(int NP, int N, int W) {
  return row_plan(NP, N, W, ep_ctas(W) * sm_count(), 4, 128, 1);
}

qpm_status make_gene_maps(GeneMaps *gm, int *mode, const float *genes, int NP, int N, int64_t ld) {
  memset(gm, 0, sizeof(*gm));
  const int64_t row = ((int64_t)N + 3) & ~(int64_t)3;  // the pitch of a matrix of one row
  *mode = ROWS_TMA;
  if (make_tile_map(&gm->m[0], genes, NP, N, NP == 1 ? row : ld, 32)) return QPM_OK;
  *mode = ROWS_TMA4;
  for (int c = 0; c < 4; ++c) {
    const float *first = genes + (int64_t)std::min(c, NP - 1) * ld;  // a class without rows maps row NP - 1
    const int s = (int)(((uintptr_t)first & 15) / 4);
    gm->shift[c] = s;
    const int rows = c < NP ? (NP - c + 3) / 4 : 1;
    if (!make_tile_map(&gm->m[c], first - s, rows, (int64_t)N + s, rows == 1 ? row + 4 : 4 * ld, 8))
      return fail(QPM_ERR_CUDA, "cuTensorMapEncodeTiled refused the genes' tensor map");
  }
  return QPM_OK;
}

// what closes a call: the counters of the fused combination (NULL: the combining kernel), the constants and
// the outputs
struct EvalOut {
  unsigned *ctr;
  const float2 *konst;
  float2 *deff;
  float *fit;
};

template <int W, int MODE, bool COMP>
static qpm_status launch_genes(const GeneMaps &gm, const float *g, int64_t ld, const RowPlan &pl,
                               const RowTables<1> &tabs, float2 *part, const EvalOut &out,
                               cudaStream_t stream) {
  static SmemAttr attr;
  const void *fn = (const void *)k_eval_genes<W, MODE, COMP>;
  const qpm_status st = attr.set(fn, rs_smem(1, W));
  if (st != QPM_OK) return st;
  void *args[] = {(void *)&gm, (void *)&g, (void *)&ld, (void *)&pl, (void *)&tabs, (void *)&part,
                  (void *)&out.ctr, (void *)&out.konst, (void *)&out.deff, (void *)&out.fit};
  return launch_dependent(fn, dim3(pl.C), dim3(W * 32), args, rs_smem(1, W), stream);
}

static qpm_status launch_combine(const RowPlan &pl, const float2 *part, const EvalOut &out,
                                 cudaStream_t stream) {
  int runs = rc_runs(pl);
  const int rows = RC_THREADS / runs;
  void *args[] = {(void *)&pl, &runs, (void *)&part, (void *)&out.konst, (void *)&out.deff,
                  (void *)&out.fit};
  return launch_dependent((const void *)k_eval_combine, dim3((pl.NP + rows - 1) / rows),
                          dim3(RC_THREADS), args, 0, stream);
}

// the sweep of float genes and, unless it combines its rows itself, the combining kernel
static qpm_status launch_eval_rows(bool comp, const float *g, int64_t ld, const RowPlan &pl,
                                   const float2 *blk, float2 *part, const EvalOut &out,
                                   cudaStream_t stream) {
  GeneMaps gm;
  int mode;
  qpm_status st = make_gene_maps(&gm, &mode, g, pl.NP, pl.N, ld);
  if (st != QPM_OK) return st;
  const RowTables<1> tabs{{blk}};
#define QPM_EG(WW, M)                                                       \
  st = comp ? launch_genes<WW, M, true>(gm, g, ld, pl, tabs, part, out, stream) \
            : launch_genes<WW, M, false>(gm, g, ld, pl, tabs, part, out, stream)
  if (pl.W == 4) {
    if (mode == ROWS_TMA) QPM_EG(4, ROWS_TMA);
    else QPM_EG(4, ROWS_TMA4);
  } else {
    if (mode == ROWS_TMA) QPM_EG(1, ROWS_TMA);
    else QPM_EG(1, ROWS_TMA4);
  }
#undef QPM_EG
  if (st != QPM_OK || out.ctr) return st;
  return launch_combine(pl, part, out, stream);
}

template <int W>
static qpm_status launch_packed(bool vecw, bool comp, const uint32_t *src, int64_t ld,
                                const RowPlan &pl, const RowTables<1> &tabs, float2 *part,
                                cudaStream_t stream) {
  const void *fn = vecw ? (comp ? (const void *)k_eval_packed<W, true, true>
                                : (const void *)k_eval_packed<W, true, false>)
                        : (comp ? (const void *)k_eval_packed<W, false, true>
                                : (const void *)k_eval_packed<W, false, false>);
  void *args[] = {(void *)&src, (void *)&ld, (void *)&pl, (void *)&tabs, (void *)&part};
  return launch_dependent(fn, dim3(pl.C), dim3(W * 32), args, 0, stream);
}

bool row_fuse(const RowPlan &pl, const TableLease &lease) {
  return pl.P <= RC_FUSE && pl.RB <= FUSE_BLOCKS && !lease.captured();
}

static qpm_status eval_common(const qpm_problem *prob, const void *src, int64_t ld, int32_t NP,
                              int kind, float *d_eff, float *fit, int32_t comp,
                              cudaStream_t stream) {
  if (!prob || !src || !d_eff) return fail(QPM_ERR_ARG, "qpm_eval: NULL pointer");
  if (prob->N < 1 || NP < 1) return fail(QPM_ERR_ARG, "qpm_eval: need N >= 1 and NP >= 1");
  if (prob->N > (1 << 28)) return fail(QPM_ERR_UNSUPPORTED, "qpm_eval: N too large");
  if (kind == 2 ? (ld < (prob->N + 31) / 32) : (ld < prob->N))
    return fail(QPM_ERR_ARG, "qpm_eval: leading dimension smaller than the row");
  TableLease lease(prob, 1, stream);  // held until the launches below are enqueued
  const float2 *konst, *blk = nullptr;
  qpm_status st = lease.block_table(prob, &blk, &konst);
  if (st != QPM_OK) return st;
  if (NP > EVAL_MAX_ROWS) return fail(QPM_ERR_UNSUPPORTED, "qpm_eval: too many rows");
  const int W = kind == 2 ? (NP <= 64 ? 2 : 8) : 0;
  const RowPlan pl = kind == 2 ? packed_plan(NP, prob->N, W)
                               : genes_plan(1, NP, prob->N, rows_aligned((const float *)src, NP, ld));
  void *scratch;
  st = lease.scratch(FUSE_BYTES + plan_bytes(pl, 1), &scratch);
  if (st != QPM_OK) return st;
  float2 *part = (float2 *)((char *)scratch + FUSE_BYTES);
  EvalOut out{nullptr, konst, (float2 *)d_eff, fit};
  if (kind == 2) {
    const bool vecw = (ld % 4 == 0) && (((uintptr_t)src & 15) == 0);
    const RowTables<1> tabs{{blk}};
    st = W == 8 ? launch_packed<8>(vecw, comp != 0, (const uint32_t *)src, ld, pl, tabs, part, stream)
                : launch_packed<2>(vecw, comp != 0, (const uint32_t *)src, ld, pl, tabs, part, stream);
    return st != QPM_OK ? st : launch_combine(pl, part, out, stream);
  }
  if (row_fuse(pl, lease)) out.ctr = (unsigned *)scratch;
  return launch_eval_rows(comp != 0, (const float *)src, ld, pl, blk, part, out, stream);
}


// ---------------------------------------------------------------------------
// Allocation-free variant of qpm_eval.  For callers that must not allocate device
// memory: host callbacks and other code that may not call into the allocator,
// processes whose device memory is all owned by an external allocator, and real-time
// paths where the implicit device synchronisation of cudaMalloc/cudaFree is not
// acceptable.  Its scratch (sign-block table, the constants' reduction, segment
// partials) lives in one file-scope device array of fixed size that every GPU
// loading this library holds until the process exits.
// ---------------------------------------------------------------------------
static constexpr size_t NOALLOC_SCRATCH_BYTES = (size_t)16 << 20;  // 16 MiB
static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_SCRATCH_BYTES];

namespace {
std::mutex g_noalloc_mu;
void *g_noalloc_ptr[128] = {nullptr};  // device address of g_noalloc_scratch, per device

// One-time set-up per device (with that device current): the host name
// g_noalloc_scratch is only a host-side stand-in, so its device address is
// looked up once and cached.
qpm_status noalloc_base(void **out) {
  int dev = 0;
  QPM_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 128) return fail(QPM_ERR_UNSUPPORTED, "device ordinal out of range");
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    void *p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_noalloc_scratch)");
    g_noalloc_ptr[dev] = p;
  }
  *out = g_noalloc_ptr[dev];
  return QPM_OK;
}

size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

// bytes of the fixed array one call uses: the sign-block table (192 bytes per block of
// 4 domains), the reduction partials of the constants, the constants, and the pieces'
// partials of the scan (3 float2 per piece and padded row)
size_t noalloc_bytes(int32_t N, const RowPlan &pl) {
  const int32_t Npad = (N + 3) & ~3;
  return up256(sizeof(float2) * BLK_F2 * (size_t)(Npad / 4)) +
         up256(sizeof(double2) * (size_t)table_part_count(Npad)) + 256 +
         up256(plan_bytes(pl, 1));
}
}  // namespace

}  // namespace qpm

extern "C" qpm_status qpm_eval_noalloc(const qpm_problem *prob, const float *genes, int64_t ld,
                                       int32_t NP, float *d_eff, float *fit, int32_t compensated,
                                       qpm_stream_t stream) {
  using namespace qpm;
  if (!prob || !genes || !d_eff) return fail(QPM_ERR_ARG, "qpm_eval_noalloc: NULL pointer");
  if (prob->N < 1 || NP < 1) return fail(QPM_ERR_ARG, "qpm_eval_noalloc: need N >= 1 and NP >= 1");
  if (ld < prob->N) return fail(QPM_ERR_ARG, "qpm_eval_noalloc: leading dimension smaller than the row");
  if (prob->N > (1 << 28) || NP > (1 << 26))
    return fail(QPM_ERR_ARG, "qpm_eval_noalloc: N above 2^28 or NP above 2^26");
  if (NP > EVAL_MAX_ROWS) return fail(QPM_ERR_UNSUPPORTED, "qpm_eval_noalloc: too many rows");
  const int32_t Npad = (prob->N + 3) & ~3;
  const bool aligned = rows_aligned(genes, NP, ld);
  RowPlan pl = genes_plan(1, NP, prob->N, aligned);
  size_t need = noalloc_bytes(prob->N, pl);
  if (need > NOALLOC_SCRATCH_BYTES) {  // rows split no further than the longest run needs
    pl = genes_plan(1, NP, prob->N, aligned, true);
    need = noalloc_bytes(prob->N, pl);
  }
  if (need > NOALLOC_SCRATCH_BYTES)
    return fail(QPM_ERR_ARG, "qpm_eval_noalloc: N and NP need " + std::to_string(need) +
                                 " bytes of scratch, more than the fixed 16 MiB (16777216)");
  void *base = nullptr;
  qpm_status st = noalloc_base(&base);
  if (st != QPM_OK) return st;
  cudaStream_t s = (cudaStream_t)stream;
  char *p = (char *)base;
  const size_t b_blk = up256(sizeof(float2) * BLK_F2 * (size_t)(Npad / 4));
  const size_t b_tpart = up256(sizeof(double2) * (size_t)table_part_count(Npad));
  float2 *blk = (float2 *)p;
  double2 *tpart = (double2 *)(p + b_blk);
  float2 *konst = (float2 *)(p + b_blk + b_tpart);
  float2 *part = (float2 *)(p + b_blk + b_tpart + 256);
  // every word read below is written first in this call (the sign-block table, the
  // constants and their partial sums, every piece of every row), so
  // nothing needs zeroing; the constants come from k_table without a phasor table
  TableSpec ts{prob->N, Npad, 1, Npad, prob->kappa1, prob->kappa2};
  st = launch_table(ts, nullptr, tpart, konst, nullptr, s);
  if (st != QPM_OK) return st;
  st = launch_block_table(prob->N, prob->kappa1, prob->kappa2, blk, s);
  if (st != QPM_OK) return st;
  // always the combining kernel: the call may be captured and replayed
  return launch_eval_rows(compensated != 0, genes, ld, pl, blk, part,
                          EvalOut{nullptr, konst, (float2 *)d_eff, fit}, s);
}

qpm::TableLease::TableLease(const qpm_problem *problems, int count, cudaStream_t stream) : stream_(stream) {
  g_mu.lock();
  cudaError_t e = cudaGetDevice(&dev_);
  if (e != cudaSuccess) {
    st_ = cuda_fail(e, "cudaGetDevice");
    return;
  }
  const int dev = dev_;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  // The query also makes the device's context current in a thread that has made no CUDA call yet:
  // a call that finds its tables and scratch makes no other before it encodes tensor maps, which
  // needs one.  (It refuses the legacy stream beside another's capture: the launches will say so.)
  if (cudaStreamIsCapturing(stream, &cap) != cudaSuccess) cudaGetLastError();
  else if (cap != cudaStreamCaptureStatusNone)
    e = cudaStreamGetCaptureInfo(stream, &cap, &cap_.id, &cap_.graph, nullptr, nullptr, nullptr);
  if (e != cudaSuccess || cap == cudaStreamCaptureStatusInvalidated) {
    st_ = e != cudaSuccess ? cuda_fail(e, "cudaStreamGetCaptureInfo")
                           : fail(QPM_ERR_CUDA, "the stream's capture has been invalidated");
    return;
  }
  if (cap_.graph) return;  // a captured call evicts nothing: it must not wait for the device
  size_t misses = 0;
  for (int k = 0; k < count; ++k) {
    const qpm_problem &p = problems[k];
    bool seen = g_tables.count(std::make_tuple(dev, p.N, p.kappa1, p.kappa2)) != 0;
    for (int m = 0; m < k && !seen; ++m)
      seen = problems[m].N == p.N && problems[m].kappa1 == p.kappa1 &&
             problems[m].kappa2 == p.kappa2;
    misses += !seen;
  }
  if (misses > 0 && device_table_count(dev) + misses > MAX_TABLES)
    st_ = release_device_caches(dev);
}

qpm::TableLease::~TableLease() { g_mu.unlock(); }

qpm_status qpm::TableLease::table(const qpm_problem *p, const float4 **table, const float2 **konst) {
  if (st_ != QPM_OK) return st_;
  return get_table(dev_, p, stream_, cap_, table, konst);
}

qpm_status qpm::TableLease::block_table(const qpm_problem *p, const float2 **blk, const float2 **konst) {
  if (st_ != QPM_OK) return st_;
  const float4 *table;
  return get_table(dev_, p, stream_, cap_, &table, konst, blk);
}

qpm_status qpm::TableLease::scratch(size_t bytes, void **ptr) {
  if (st_ != QPM_OK) return st_;
  return cap_.graph ? graph_scratch(dev_, stream_, cap_, bytes, ptr)
                    : get_scratch(dev_, stream_, bytes, ptr);
}

extern "C" qpm_status qpm_eval(const qpm_problem *prob, const float *genes, int64_t ld,
                               int32_t NP, float *d_eff, float *fit, int32_t compensated,
                               qpm_stream_t stream) {
  return qpm::eval_common(prob, genes, ld, NP, 1, d_eff, fit, compensated,
                          (cudaStream_t)stream);
}

extern "C" qpm_status qpm_eval_packed(const qpm_problem *prob, const uint32_t *signs,
                                      int64_t ld_words, int32_t NP, float *d_eff, float *fit,
                                      int32_t compensated, qpm_stream_t stream) {
  return qpm::eval_common(prob, signs, ld_words, NP, 2, d_eff, fit, compensated,
                          (cudaStream_t)stream);
}

extern "C" qpm_status qpm_release_caches(void) {
  std::lock_guard<std::mutex> lock(qpm::g_mu);
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return qpm::cuda_fail(e, "cudaGetDevice");
  return qpm::release_device_caches(dev);
}
