// api_internal.h -- host-side helpers shared by the C-ABI translation units.
#pragma once

#include <cuda_runtime.h>

#include <cstdarg>
#include <cstdint>
#include <memory>
#include <vector>

#include "dpgpu.h"
#include "mcm_kernels.cuh"
#include "sdp_kernels.cuh"

namespace dph {

// Records a thread-local error message and returns `code`.
dp_status fail(dp_status code, const char* fmt, ...);
dp_status fail_cuda(cudaError_t e, const char* what);

struct DevState {
  int device = -1;
  int sms = 0;
  int occ[2] = {0, 0};        // MCM blocks per SM, int32 / int64 costs
  int32_t* status = nullptr;  // library-owned status word
  cudaStream_t aux = nullptr; // plan building (waited for before a plan is used)
};

// Per-device state for the current device (created on first use).
dp_status current_dev(DevState** out);

// Stream-ordered workspace of an S-DP path that has another way without it
// (dp_test_refuse_scratch makes it report that there is no memory).
cudaError_t scratch_alloc(void** p, size_t bytes, cudaStream_t st);

cudaError_t traceback_configure();  // kernel attributes of the current device (traceback.cu)

long long spin_limit();     // bounded-wait budget in clock cycles

// Kernel timing (dp_profile_begin / dp_profile_end): when enabled, the
// launchers bracket each solver kernel with events on its stream.
bool profiling();
void profile_mark(int which, cudaStream_t st, bool after);  // which: 0 = MCM, 1 = S-DP

// ---------------------------------------------------------------------------
// MCM plans
// ---------------------------------------------------------------------------
struct McmStatic {
  bool i64 = false;
  int device = -1;
  std::vector<int32_t> ns;
  std::vector<dpk::McmInstDev> insts;   // static fields only
  std::vector<int32_t> cursors;         // first place of each queue bin, then 0 (McmQueueArgs)
  int64_t ntasks = 0, ntiles = 0, nslots = 0, pp_total = 0, pk_total = 0;
  int32_t levels_per_part = 0;
  double split_evals = 0;
  int32_t max_nt = 1;                    // tiles per side of the longest chain
  // device copies (immutable after creation)
  dpk::McmTask* d_tasks = nullptr;
  int32_t* d_accslot = nullptr;
  dpk::McmInstDev* d_insts = nullptr;
  bool owns_device = true;               // false: device pointers borrowed from a workspace
  ~McmStatic();
};

struct McmLayout {
  size_t af = 0, bf = 0, flags = 0, counters = 0, queue = 0, acc = 0, pp = 0, pk = 0, insts = 0;
  size_t zero_begin = 0, zero_bytes = 0, total = 0;
};

// Lays a plan out (host arithmetic, no queue); with upload=true the queue, the
// slot table and the chain records are built in fresh device memory owned by
// the result.  levels_per_part: external levels per bulk task (0 = the default).
dp_status mcm_build_static(const std::vector<int32_t>& ns, bool i64, std::shared_ptr<McmStatic>* out,
                           bool upload = true, int levels_per_part = 0);
// Enqueues the building of sp's queue from its records and cursors on the device.
dp_status mcm_build_queue(const McmStatic& sp, int32_t* d_cursors, cudaStream_t st);
// The queue on the host, in the order a single chain's has on the device.
std::vector<dpk::McmTask> mcm_host_queue(const McmStatic& sp);
McmLayout mcm_layout(const McmStatic& sp);
// Resident blocks per SM for a queue of ntasks tasks over max_nt tile-diagonals.
int mcm_blocks_per_sm(int64_t ntasks, int max_nt, bool i64, int sms, int occ);
// Enqueues memsets + prologue + main kernel for a static plan on `ws`.
// w_all != nullptr: the interval DP with per-cell weights laid out like m_all
// (a weight pass is enqueued before the prologue).
dp_status mcm_enqueue(const McmStatic& sp, const McmLayout& L, void* ws, const int32_t* p_all,
                      const int64_t* p_off, const int64_t* tab_off, void* m_all, int16_t* s_all,
                      int32_t* status, cudaStream_t st, long long limit_override = 0,
                      int32_t drop_task = -1, int blocks_per_sm = 0, const void* w_all = nullptr);

// ---------------------------------------------------------------------------
// S-DP
// ---------------------------------------------------------------------------
dp_status sdp_validate(int64_t n, const int32_t* a, int32_t k, int op);
// Approximate device time of the step kernel for `cells` cells, microseconds.
double sdp_plain_us(int64_t cells, int32_t ak, int32_t k);
struct SdpSteps {  // the same for several lengths
  SdpSteps(int32_t ak, int32_t k);
  double us(int64_t cells) const { return cells <= 0 ? 0.0 : (double)((cells + W - 1) / W) * step_us; }
  int64_t W;
  double step_us;
};
void sdp_shape(int32_t a1, int32_t ak, int* threads, int* ring_log2);
// (x) = min: the first cell from which the table repeats its last g cells, g
// the gcd of the offsets (host arithmetic on the offsets only; see
// sdp_kernels.cuh).  0: not below n, or not found within a bounded search, of
// about budget_us of host time where given; the budget of a single solve, and
// the word operations that a search may take.
int64_t sdp_min_tail(int64_t n, const int32_t* a, int32_t k, int32_t* g, double budget_us = 1e9);
double sdp_min_tail_budget_us(int64_t n, const int32_t* a, int32_t k);
int64_t sdp_min_tail_ops(int64_t n, const int32_t* a, int32_t k, double budget_us);
// How one table is solved: in `chunks` >= 2 chunks from jumped windows, or by
// the step kernel, with tail_from > 0 up to there and the rest filled (known
// with chunks too, for when their workspace cannot be had).
struct SdpRoute {
  int chunks = 0;
  int64_t tail_from = 0;
  int32_t g = 0;
  double us = 0.0;  // (x) = + in chunks: the model's time
};
SdpRoute sdp_route(int64_t n, const int32_t* a, int32_t k, int op, int sms);
// Solves a table whose route is in chunks; without memory for the workspace
// it enqueues nothing and turns the route into the step kernel's.
dp_status sdp_in_chunks(uint32_t* ST, int64_t n, const int32_t* a, int32_t k, int op, SdpRoute* route,
                        int32_t* status, cudaStream_t st);
// Fills the arguments of the step kernel's launch for one table (not for chunks >= 2).
void sdp_single_args(dpk::SdpLaunchArgs* args, uint32_t* ST, int64_t n, const int32_t* a, int32_t k, int op,
                     const SdpRoute& route, int sms, int32_t* status);
// (x) = + on one instance, by chunks that start from jumped windows
// (sdp_jump.cu): the number of chunks the cost model picks (0: solve step by
// step; otherwise *us is the model's time), and the solve with a given number
// of chunks.
int sdp_jump_chunks(int64_t n, const int32_t* a, int32_t k, int sms, double* us = nullptr);
// The plan behind it (host arithmetic only): P, L, L0, squarings, reach of
// the impulse response, chunks per major window, major windows, chunks asked.
int sdp_jump_plan(int64_t n, const int32_t* a, int32_t k, int sms, int64_t out[8]);
// Without memory for its workspace it sets *no_scratch, where given, and enqueues
// nothing: the table is then to be solved step by step.
dp_status sdp_add_jump(uint32_t* ST, int64_t n, const int32_t* a, int32_t k, int chunks, int32_t* status,
                       cudaStream_t st, bool* no_scratch = nullptr);
// (x) = min on one instance, by chunks whose windows come from Boolean
// products modulo the characteristic polynomial (sdp_minjump.cu): whether the
// path applies (a_k >= 32, a_1 <= 8192, a long enough table, the window on
// chip), the number of chunks the cost model picks (0: solve step by step, up
// to tail_from when that is not 0), and the solve with a given number of chunks.
bool sdp_min_jump_eligible(int64_t n, const int32_t* a, int32_t k);
int sdp_min_jump_chunks(int64_t n, const int32_t* a, int32_t k, int sms, int64_t tail_from);
// The plan behind it (host arithmetic only): P, L, L0, squarings, chunks asked.
int sdp_min_jump_plan(int64_t n, const int32_t* a, int32_t k, int sms, int64_t out[5]);
// no_scratch as for sdp_add_jump.
dp_status sdp_min_jump(uint32_t* ST, int64_t n, const int32_t* a, int32_t k, int chunks, int32_t* status,
                       cudaStream_t st, bool* no_scratch = nullptr);

}  // namespace dph
