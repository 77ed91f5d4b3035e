// qpm_internal.h -- host-side declarations shared by the library's translation units.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <string>

#include "qpm.h"

namespace qpm {

void set_error(const std::string &msg);
qpm_status fail(qpm_status s, const std::string &msg);
qpm_status cuda_fail(cudaError_t e, const char *what);

#define QPM_CUDA(call)                                  \
  do {                                                  \
    cudaError_t e_ = (call);                            \
    if (e_ != cudaSuccess) return ::qpm::cuda_fail(e_, #call); \
  } while (0)

// Phasor table layout: dimension m of a row split over T threads of c dims each
// (c a multiple of 4) lives at float4 index ((k4 * 4 + q) * T + t) with t = m / c,
// k4 = (m % c) / 4, q = m % 4.  T = 1, c = Npad is the natural order.
struct TableSpec {
  int32_t N, Npad, T, c;
  double kappa1, kappa2;
};

// float2 konst[4] = {phi1*phi2, cdiag, psi, phi1}; double2 konst64[4] = {phi1*phi2, cdiag, psi, phi1}
// part: scratch of table_part_count(Npad) double2; table may be NULL (constants only)
int table_part_count(int32_t Npad);
qpm_status launch_table(const TableSpec &s, float4 *table, double2 *part, float2 *konst,
                        double2 *konst64, cudaStream_t stream);

// the tables and constants of n problems in two launches (d_jobs: device array)
struct TableJob {
  TableSpec s;
  float4 *table;
  double2 *part;
  float2 *konst;
  double2 *konst64;
};
qpm_status launch_tables(const TableJob *d_jobs, int n, int32_t max_npad, cudaStream_t stream);

// sign-block table of the row sweeps: 8 patterns x (A, B, C) as float2 for every
// block of 4 domains, float2 blk[(8 b + e) * 3 + k], ceil(N / 4) blocks (24 float2
// = 192 bytes each); built in FP64, rounded to FP32
qpm_status launch_block_table(int32_t N, double kappa1, double kappa2, float2 *blk,
                              cudaStream_t stream);
constexpr int BLK_F2 = 24;  // float2 per block of 4 domains

// Access to the per-(device, N, kappa1, kappa2) cache of phasor tables, FP32
// constants and sign-block tables.  A lease holds the cache's lock from its
// construction to its destruction: the caller keeps it alive from the first lookup
// until the last launch that uses the returned pointers has been enqueued, so no
// other host thread can evict those tables in between.  The cache holds at most
// MAX_TABLES problems per device; a lease that will look up `problems` distinct
// problems makes room for all of them when it is created (freeing every table of
// the device once, after a device synchronisation), never between two lookups.
// Where the stream is being captured, what the lease gives out stays valid for as long as the
// capture's graph, or an executable instance of it, lives.
struct Capture {
  cudaGraph_t graph = nullptr;  // NULL: the stream is not being captured
  unsigned long long id = 0;
};
class TableLease {
 public:
  TableLease(const qpm_problem *problems, int count, cudaStream_t stream);
  ~TableLease();
  TableLease(const TableLease &) = delete;
  TableLease &operator=(const TableLease &) = delete;
  // status of the set-up (a failed eviction is reported by the first lookup)
  qpm_status status() const { return st_; }
  bool captured() const { return cap_.graph != nullptr; }
  // natural-order phasor table and FP32 constants; built on a miss
  qpm_status table(const qpm_problem *p, const float4 **table, const float2 **konst);
  // the same entry's sign-block table (built the first time) and constants
  qpm_status block_table(const qpm_problem *p, const float2 **blk, const float2 **konst);
  // scratch for one call's launches: the stream's, which starts with FUSE_BLOCKS counters that are 0
  // between calls, or the captured graph's own
  qpm_status scratch(size_t bytes, void **ptr);

 private:
  int dev_ = 0;
  cudaStream_t stream_;
  Capture cap_;
  qpm_status st_ = QPM_OK;
};

// split of the row sweeps (qpm_rows.cuh): row blocks of W groups of 32 rows, each nunit units
// of gran sub-steps of 32 domains, laid end to end and dealt to C CTAs as equal runs
struct RowPlan {
  int NP, N;
  int NPpad;  // NP rounded up to 32
  int W;      // warps (row groups) per CTA
  int RB;     // row blocks
  int nsub;   // sub-steps of a row, ceil(N / 32)
  int gran, nunit;  // sub-steps per unit, units of a row
  int C;      // CTAs
  int P;      // pieces of a row at most
};
// full: resident CTAs of the GPU; gran: sub-steps per unit; maxsub: longest run; min_units: no run
// shorter than this while CTAs are left idle
RowPlan row_plan(int NP, int N, int W, int64_t full, int gran, int maxsub, int min_units);
// the plan of the float-gene sweep with K sign-block tables; aligned: see rows_aligned; whole: no
// row is split unless it is longer than a run may be (fewest pieces)
RowPlan genes_plan(int K, int NP, int N, bool aligned, bool whole = false);
// all rows start on 16-byte boundaries
inline bool rows_aligned(const float *genes, int NP, int64_t ld) {
  return ((uintptr_t)genes & 15) == 0 && (NP == 1 || ld % 4 == 0);
}
// whether the sweep combines the rows itself, with the counters of the stream's scratch: where a row
// has few pieces and the call is not captured, whose replays may run beside the stream's calls
constexpr int FUSE_BLOCKS = 4096;  // row blocks of such a plan at most
constexpr size_t FUSE_BYTES = sizeof(unsigned) * FUSE_BLOCKS;
bool row_fuse(const RowPlan &pl, const TableLease &lease);
constexpr int EVAL_MAX_ROWS = 128 * 65535;  // rows a call of the row sweeps takes
// bytes of the plan's partial monoids for K problems
inline size_t plan_bytes(const RowPlan &p, int K) {
  return sizeof(float2) * 3 * (size_t)K * (size_t)p.P * (size_t)p.NPpad;
}

// launch as a programmatic dependent of the stream's last kernel: the kernel's CTAs may be
// scheduled as that one's retire, and the kernel itself waits (griddepcontrol.wait) for it
qpm_status launch_dependent(const void *fn, dim3 grid, dim3 block, void **args, size_t smem,
                            cudaStream_t stream);
// dynamic shared memory of a kernel, set once per device (always to the same value)
struct SmemAttr {
  unsigned char done[128] = {0};
  qpm_status set(const void *fn, size_t bytes);
};

// current device's SM count (cached per device)
int sm_count();

}  // namespace qpm
