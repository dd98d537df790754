// Launch wrappers of the device kernels (host-callable).
#pragma once
#include <cuda_runtime.h>

#include "device.h"

namespace ajf {

cudaError_t set_kernel_smem_limits();

// Launches of a program's chain of dependent kernels. Every kernel of the chain is launched with
// programmatic stream serialization and waits (griddepcontrol.wait) before its first access to what
// other kernels read or write, so its launch latency, descriptor loads and offset tables overlap the
// end of the kernel before it. Such a kernel is resident while others still write the tensors that it is
// going to read, and while others read what lay at their addresses before. So no pointer to data that another
// kernel writes is __restrict__ here: that would promise memory that does not change while the kernel lives,
// and allow non-coherent loads and loads moved above the wait. (Descriptors, uploaded before the chain
// starts, may be.) `early`: the kernel lets its successor start as soon as it has itself waited; set for
// short kernels only (chain_early), because a successor that waits for long holds shared memory and warps
// that other streams could use. Not before its own wait: a run of early kernels would then all be resident
// at once, while the trigger behind the wait lets a kernel start only when everything but its predecessor is
// complete, and is no slower (in turn on one GPU, before / behind, us: twelve uneven circuits 1,264 / 1,247,
// 4 x 5 grid F64 782 / 775, n = 16 bf16x6 1,524 / 1,513, tiny 78 / 77).
template <typename... KArgs, typename... Args>
cudaError_t launch_chained(void (*kernel)(KArgs...), dim3 grid, unsigned threads, size_t smem, cudaStream_t s,
                           Args... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// Fixed device arena (static_arena.cu) for evaluations that allocate nothing: its size, and its
// device address on `device`, which must be the current device (cudaErrorInvalidDevice otherwise).
constexpr size_t kStaticArenaBytes = size_t(64) << 20;
cudaError_t static_arena_address(int device, void** ptr);
size_t step_table_bytes(const StepDev& st);
size_t perm_table_bytes(const PermDev& p);

cudaError_t launch_leaves(const LeafDev* d_leaves, int n, const double* d_in, void* arena, cudaStream_t s);
cudaError_t launch_small(const StepDev* d_steps, int nsteps, int total_blocks, size_t smem, void* arena, cudaStream_t s,
                         bool early = false);
cudaError_t launch_splitk(const StepDev* d_steps, int nsteps, int total_blocks, size_t smem, void* arena,
                          double2* partial, double2* scalars, cudaStream_t s);
// op_f64: the operands are FP64 (staged in FP64); otherwise every format is staged in FP32.
cudaError_t launch_perm(const PermDev* d_perms, int nperm, int grid_x, size_t smem, const void* arena, void* base,
                        bool op_f64, cudaStream_t s, bool early = false);
// Tiled FP64 full contraction (k_dot) of steps with a scalar result, then the partial-sum pass.
// The tiled dot's staged form (FP32 operands, FP32 products): the step qualifies on the host side;
// the kernel also checks the operands' bit positions and alignment and otherwise falls back.
bool dot_staged(const StepDev& st, bool f32_products);
size_t dot_smem_bytes(const StepDev& st, bool f32_products);
// f32_products: FP32 products summed in FP32 per tile, tile sums in FP64 (reduced-precision modes).
cudaError_t launch_dot(const StepDev* d_steps, int nsteps, int total_blocks, size_t smem, const void* arena,
                       double2* partial, double2* scalars, bool f32_products, cudaStream_t s);
cudaError_t launch_gemm_simt(const void* A, const void* B, void* C, int64_t M, int64_t N, int64_t K, bool f64,
                             cudaStream_t s);
cudaError_t launch_final(const FinalDev* d_fd, int open_bits_nchunks, int nblocks, const void* arena,
                         const double2* scalars, double* traces, double* partial, double* result, cudaStream_t s);
// Persistent kernel: one thread block per network runs that network's whole program (leaves,
// all steps level by level, the FP64 trace and F) -- n_jobs networks in one launch. `smem`:
// dynamic shared memory per block (the largest work region among the jobs with job.smem = 1).
cudaError_t launch_persistent(const InterpJob* d_jobs, int n_jobs, const InterpOp* d_ops, size_t smem, int threads,
                              cudaStream_t s);
constexpr size_t kPersistentSmemMax = 96 * 1024;

// GEMMs of the FP64 and FP32 modes on the fp16 tensor cores (dg_gemm.cu, digits.cuh): bytes of a
// digit operand (rows x kcols real columns), supported shapes and K splits.
size_t dg_operand_bytes(int64_t rows, int64_t kcols, int mode);
bool dg_gemm_supported(int64_t M, int64_t N, int64_t K);
int dg_gemm_splits(int64_t M, int64_t N, int64_t K);
// Row exponents of the operands whose K spans several gather tiles (PermDev::strips > 0), then the
// gather itself; `mode` is the (common) digit mode of the perms.
cudaError_t launch_row_exp(const PermDev* d_perms, int nperm, int grid_x, size_t smem, const void* arena, void* base,
                           cudaStream_t s);
cudaError_t launch_digits(const PermDev* d_perms, int nperm, int grid_x, size_t smem, const void* arena, void* base,
                          int mode, cudaStream_t s, bool early = false);
struct DgGemm {
  const void* x = nullptr;   // X digits (M rows: embedded complex rows), Y digits (N rows)
  const void* y = nullptr;
  const int* ex = nullptr;   // row exponent fields: M / 2 and N values
  const int* ey = nullptr;
  void* C = nullptr;         // M x N, FP64 (OPM_DIG6) or FP32 (OPM_DIG4)
  double* ws = nullptr;      // ksplit > 1: ksplit * M * N FP64 partials
  int* status = nullptr;
  int64_t M = 0, N = 0, K = 0;
  int ksplit = 1, mode = OPM_DIG6;
  bool early = false;        // see launch_chained
  unsigned long long wait_ns = 0;  // bound of every device-side wait
};
cudaError_t launch_dg_gemm(const DgGemm& g, cudaStream_t s);
cudaError_t set_dg_smem_limits();

// Tensor-core GEMM (tcgen05, tc_gemm.cu): C[M][N] (FP32, row-major) =
// sum_{i + j < terms} A_i[M][K] . B_j[N][K]^T for the split terms A_t, B_t (byte offsets from
// `base`), FP32 accumulation promoted per K block. kind 0: tf32, 1: bf16, 2: scaled fp16.
// Returns cudaErrorNotSupported when the shape is not tile-aligned.
bool tc_gemm_supported(int64_t M, int64_t N, int64_t K, int kind);
// K splits for an M x N x K GEMM: GEMMs with fewer 128 x BN tiles than SMs divide K over several
// CTAs, each writing an FP32 partial tile to a workspace of ksplit * M * N floats that a
// deterministic pass then sums into C. 1 = no split (no workspace).
int tc_gemm_splits(int64_t M, int64_t N, int64_t K, int kind);
// A tensor-core GEMM launch prepared on the host (tensor maps, tiling, kernel parameters), so that
// enqueueing it later costs one kernel launch (two with a K split) and no host set-up.
struct TcPrepared {
  alignas(64) unsigned char params[1024];  // the kernel's parameter block
  cudaError_t (*run)(const void* params, unsigned grid, size_t smem, cudaStream_t s, bool early) = nullptr;
  unsigned grid = 0;
  size_t smem = 0;
  int ksplit = 1;
  float* ws = nullptr;
  float* C = nullptr;
  int64_t n = 0;  // M * N
  bool ready = false;
};
cudaError_t tc_gemm_prepare(TcPrepared* t, char* base, const int64_t* a_off, const int64_t* b_off, int terms,
                            float* C, int64_t M, int64_t N, int64_t K, int kind, float* ws, int ksplit,
                            int* d_status, unsigned long long wait_ns, int stall_loads);
cudaError_t tc_gemm_run(const TcPrepared& t, cudaStream_t s, bool early = false);
// Bound of every device-side wait in the GEMM and the step interpreter (nanoseconds).
constexpr unsigned long long kTcWaitNs = 2000000000ull;
// Persistent step interpreter (queue.cu): one launch of `blocks` blocks (at most one per SM) runs
// the tasks of the phases (device tables; see device.h). d_counters: kQPhase0 + nphases ints,
// zeroed by the launch. A dependency wait that expires sets *d_status (code 21) and the error
// counter; a GEMM wait sets its own code, as in the standalone kernel.
size_t queue_smem_bytes();
// d_prof (optional, 3 * kQKinds counters, accumulated): per kind of task, its busy nanoseconds,
// the nanoseconds its block waited for the previous phase, and its task count.
constexpr int kQKinds = 10;
cudaError_t launch_queue(const QPhase* d_phases, int nphases, const QTask* d_tasks, int ntasks, int* d_counters,
                         int* d_status, int blocks, cudaStream_t s, unsigned long long wait_ns = kTcWaitNs,
                         unsigned long long* d_prof = nullptr);
// A prepared tensor-core GEMM's parameter block for the interpreter (its fixed pipeline geometry),
// written to `out` (queue_gemm_params_bytes() bytes, 64-byte aligned in device memory when used);
// its tile width, operand kind and work-item count.
size_t queue_gemm_params_bytes();
cudaError_t queue_gemm_params(const TcPrepared& t, void* out, int* bn, int* bf16, int* nwork);
cudaError_t launch_gemm_tc(char* base, const int64_t* a_off, const int64_t* b_off, int terms, float* C, int64_t M,
                           int64_t N, int64_t K, int kind, float* ws, int ksplit, int* d_status, cudaStream_t s);
// Same with an explicit bound on every device-side wait and a test hook: stall_loads = 1 makes the
// producer issue no loads, so the MMA and epilogue waits expire and the kernel reports a status
// code and returns.
cudaError_t launch_gemm_tc_ex(char* base, const int64_t* a_off, const int64_t* b_off, int terms, float* C, int64_t M,
                              int64_t N, int64_t K, int kind, float* ws, int ksplit, int* d_status, cudaStream_t s,
                              unsigned long long wait_ns, int stall_loads);

}  // namespace ajf
