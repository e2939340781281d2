// Internal launch interface between the host state machine and the sm_100a kernels.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

namespace psk {

constexpr int P = 813258;
constexpr int P_PAD = 813312;          // floats per stored parameter / gradient vector
constexpr int P_VEC4 = P_PAD / 4;      // 203,328 float4 columns
constexpr int MAX_WORKERS = 256;
constexpr int MAX_RING = 16;
constexpr int MAX_GROUPS = 16;
constexpr int MAX_CHAIN = 8;           // servers in a replication chain, the frontend included

constexpr int OFF_C1W = 0, OFF_C1B = 144, OFF_C2W = 160, OFF_C2B = 4768;
constexpr int OFF_F1W = 4800, OFF_F1B = 807616, OFF_F2W = 808128, OFF_F2B = 813248;

constexpr int IMG = 28, C1 = 16, H1 = 14, C2 = 32, H2 = 7;
constexpr int P1_ELEMS = C1 * H1 * H1;   // 3136
constexpr int P1_PLANE_ELEMS = 2 * 256 * 4;   // 32-bit words of one sample's p1 in the tensor-core plane layout (8 KB of BF16)
constexpr int FLAT = C2 * H2 * H2;       // 1568
constexpr int HID = 512, NCLS = 10;
constexpr int CONV_SPB = 4;              // samples per partial-sum slot of the convolutions' filter gradients
constexpr int MIN_RANGE = CONV_SPB;       // shortest range of rows of a filter-gradient block (tensor-core path)
constexpr int C2_GRAD = 4608 + 32, C1_GRAD = 144 + 16;
constexpr int FC_PART = NCLS * HID + HID + NCLS + 2;   // fc2.w, fc1.b, fc2.b gradients, loss sum, padding
// Blocks per worker in the output layer's kernel, each with its own partial sums: at least eight samples to a block, about
// two blocks per SM in all (W * fc2_split(W, b) <= max(W, FC2_BLOCKS)).
constexpr int FC2_BLOCKS = 296, FC2_MAX_SPLIT = 8;
__host__ __device__ inline int fc2_split(int W, int b) {
  int s = FC2_BLOCKS / W;
  s = s < 1 ? 1 : (s > FC2_MAX_SPLIT ? FC2_MAX_SPLIT : s);
  const int most = (b + 7) / 8;
  return s < most ? s : most;
}

// The second convolution's filters as tensor-core operands, per weight group: BANK2_BLOCKS blocks of 32 rows of the forward
// kernel (two planes of eight input channels), and the input gradient's 12 x 48 rows; a row is eight BF16 values.
constexpr int BANK2_BLOCKS = 40, BANK2_FWD_ROWS = 32 * BANK2_BLOCKS, BANK2_FWD_BYTES = 2 * BANK2_FWD_ROWS * 16;
constexpr int BANK2_DX_ROWS = 12 * 48, BANK2_DX_BYTES = BANK2_DX_ROWS * 16, BANK2_BYTES = BANK2_FWD_BYTES + BANK2_DX_BYTES;
constexpr uint8_t BANK2_ZERO_BLOCK = 255;
struct Bank2Taps { uint8_t tap[BANK2_BLOCKS]; };      // filter tap ky * 3 + kx of a block's 32 filters; BANK2_ZERO_BLOCK: zeros

// FP32 path: the same filters as BF16 pieces (bf16x3.cuh) for its own kernels, [piece][octet][row] forward and
// [filter row][octet][piece][column] for the input gradient; and the first convolution's output, [image row of the bordered
// map][piece][octet of channels][slot (X & 1) * 8 + X / 2][8 channels] BF16.
constexpr int BANK3_BLOCKS = 36, BANK3_FWD_ROWS = 32 * BANK3_BLOCKS, BANK3_FWD_BYTES = 3 * 2 * BANK3_FWD_ROWS * 16;
constexpr int BANK3_DX_BYTES = 12 * 3 * 48 * 16, BANK3_BYTES = BANK3_FWD_BYTES + BANK3_DX_BYTES;
struct Bank3Taps { uint8_t tap[BANK3_BLOCKS]; };      // filter tap ky * 3 + kx of a block's 32 filters
constexpr int P1X_ROW = 3 * 2 * 16 * 16, P1X_BYTES = 16 * P1X_ROW;

constexpr uint32_t STATUS_BAD_LABEL = 1u;
constexpr uint32_t STATUS_WAIT_TIMEOUT = 2u;   // a bounded barrier wait in a tensor-core kernel gave up

// Optional per-kernel timing: when switched on, every launch is bracketed by two CUDA events on
// the launching stream; totals per kernel are read back after a synchronisation.
enum KernelId {
  K_CONV1_FWD = 0, K_CONV2_FWD, K_FC1_FWD, K_FC2_FWD_BWD, K_FC1_DW, K_FC1_DX, K_CONV2_BWD, K_CONV1_BWD,
  K_CONV_GRAD_REDUCE, K_SUM_APPLY_DIRECT, K_SUM_PARTIAL, K_SUM_FINISH, K_ASYNC_APPLY, K_COPY_ROWS,
  K_DROPOUT_MASK, K_CONV2_DW, K_PREP_W1, K_SQ_NORM, K_COEF_FINISH, K_EVAL_FINISH, K_CLIP_SUM, K_COUNT
};
const char* kernel_name(int id);

struct Profiler {
  bool on = false;
  struct Rec { int id; cudaEvent_t a, b; };
  std::vector<Rec> recs;
  std::vector<cudaEvent_t> free_events;
  cudaEvent_t get() {
    if (!free_events.empty()) { cudaEvent_t e = free_events.back(); free_events.pop_back(); return e; }
    cudaEvent_t e = nullptr;
    cudaEventCreate(&e);
    return e;
  }
  void begin(int id, cudaStream_t st) {
    if (!on) return;
    Rec r{id, get(), get()};
    cudaEventRecord(r.a, st);
    recs.push_back(r);
  }
  void end(cudaStream_t st) {
    if (!on) return;
    cudaEventRecord(recs.back().b, st);
  }
  // Caller has synchronised the stream.  Adds elapsed times into ms[K_COUNT] / n[K_COUNT] and recycles events.
  void collect(double* ms, int64_t* n) {
    for (auto& r : recs) {
      float t = 0.f;
      if (cudaEventElapsedTime(&t, r.a, r.b) == cudaSuccess) { ms[r.id] += t; n[r.id] += 1; }
      free_events.push_back(r.a);
      free_events.push_back(r.b);
    }
    recs.clear();
  }
  ~Profiler() {
    for (auto& r : recs) { cudaEventDestroy(r.a); cudaEventDestroy(r.b); }
    for (auto e : free_events) cudaEventDestroy(e);
  }
};

// Per-call tables passed by value as kernel parameters.
// Workers are processed in "sorted" order: workers sharing a weight snapshot are adjacent, so
// that a group's samples form one contiguous block of activation rows.
struct WorkerTable {
  float* grad[MAX_WORKERS];     // destination gradient vector (P_PAD floats) of sorted worker s
  int32_t wid[MAX_WORKERS];     // logical worker id (dropout key)
  int32_t src[MAX_WORKERS];     // index of the worker in the caller's arrays (x, y, loss, argmax)
  int16_t group[MAX_WORKERS];   // group of sorted worker s
};

struct GroupTable {
  const float* theta[MAX_GROUPS];  // weight snapshot of the group
  int32_t first[MAX_GROUPS + 1];   // first sorted worker of the group; first[n_groups] = W
  int32_t n_groups;
};

// Activation workspace carved from the arena (rows = sorted worker * b + sample).
struct Workspace {
  float* p1;       // conv1 -> ReLU -> pool: [rows][2 planes][256][8] BF16 (tensor-core path)
  uint8_t* p1x;    // the same in BF16 pieces: [rows][P1X_BYTES] (FP32 path)
  uint8_t* code1;  // [rows][3136]        pool-1 decisions. [4 channel quads][196][4]; FP32 path: argmax 0..3, 4 = no gradient (max <= 0); tensor-core path:
                   //                     the byte 1 << argmax, 0 = no gradient
  float* p2;       // [rows][1568]        conv2 -> ReLU -> pool, channel-major flatten (tensor-core path)
  uint8_t* code2;  // [rows][1568]        [8 channel quads][49][4], argmax 0..3, 4 = no gradient
  float* d;        // [rows][512]         fc1 -> ReLU -> dropout (scaled)
  float* da1;      // [rows][512]         gradient w.r.t. fc1 pre-activation (tensor-core path)
  float* dp2;      // [rows][1568]        gradient w.r.t. p2 (tensor-core path: BF16 in the first half of each row)
  float* dp1;      // [rows][3136]        gradient w.r.t. p1, [4 channel quads][196][4]: fp32 (FP32 path) or BF16 in the first half of the row (tensor-core path)
  float* part2;    // [W][chunks][4640]   per-block partial conv2 weight/bias gradients
  float* part1;    // [W][chunks][160]    per-block partial conv1 weight/bias gradients
  float* partf;    // [W][fc2_split][FC_PART] per-block partial output-layer gradients and loss sums
  float* w1r;      // [groups][512][1568] TF32-rounded fc1 weights of each weight group of the call
  float* w1tr;     // [groups][1568][512] and their transpose
  uint16_t *p2x, *da1x;   // FP32 path: p2 and da1 as BF16 pieces, [3][rows of the call][1568] and [3][rows of the call][512]
  uint16_t* w1x;   // FP32 path: [groups][3][512][1568] W1 as BF16 pieces
  uint8_t* bank2;  // [groups][BANK2_BYTES] (FP32 path: BANK3_BYTES) conv2's filters as its kernels' operands (forward, then input gradient)
  uint32_t* status;
};

struct GradStepArgs {
  int W, b;
  const float* x;      // [W][b][784] caller order
  const int32_t* y;    // [W][b]
  float* loss;         // [W]
  int32_t* argmax;     // [W][b]
  uint64_t seed, step;
  float drop_p;
  uint32_t drop_thresh;   // keep iff word >= thresh
  int precision;          // 0 = FP32 (second convolution and dense layer on the tensor cores, operands in BF16 pieces); otherwise tensor cores (BF16 convolution products, TF32 dense layer)
  int skip_prep_w1;       // the rounded copies of the dense-layer weights of these very snapshots are still valid
  int after_wait = 0;     // the caller has just made the stream wait for another one
};

// Side streams (and the events that fork from / join into the caller's stream) for the independent
// branches of the backward pass; null streams mean "run everything on the caller's stream".
struct SideStreams {
  cudaStream_t s1 = nullptr, s2 = nullptr;
  cudaEvent_t fork1 = nullptr, join1 = nullptr, fork2 = nullptr, join2 = nullptr;
};

// The summed step (all workers on one snapshot, only the sum of their gradients wanted): where it goes and the scratch
// for the partial sums of the 512-unit layer's weight gradient.
struct SummedStep {
  float* grad_sum;      // [P_PAD] the sum over workers
  float* super_part;    // [n_super][P_PAD] scratch
  int n_super;          // groups of W / n_super workers (a divisor of W, at most 16)
};

// Lets a kernel use `bytes` of dynamic shared memory.  Asked for by every ps_create, so what is already in force is left
// alone: setting it again for the library's twenty kernels made a new server's first pass 0.1 ms longer.
inline cudaError_t allow_smem(const void* kernel, int bytes) {
  cudaFuncAttributes at;
  const cudaError_t e = cudaFuncGetAttributes(&at, kernel);
  if (e != cudaSuccess || at.maxDynamicSharedSizeBytes >= bytes) return e;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

// Part A. Returns the number of kernels launched, or -1 on a launch error.  sum == nullptr: one gradient per worker.
int launch_grad_step(const GradStepArgs& a, const WorkerTable& wt, const GroupTable& gt, const Workspace& ws,
                     cudaStream_t st, const SideStreams& side, Profiler* prof, const SummedStep* sum = nullptr);
int launch_dropout_mask(uint64_t seed, uint32_t worker, uint64_t step, int b, uint32_t thresh,
                        uint8_t* keep, cudaStream_t st, Profiler* prof);
int configure_x3_conv2_kernels();
const Bank3Taps& conv2_fwd_x3_taps();
void launch_conv2_fwd_x3(const GradStepArgs& a, const GroupTable& gt, const Workspace& ws, cudaStream_t st, Profiler* prof);
void launch_conv2_dx_x3(const GradStepArgs& a, const GroupTable& gt, const Workspace& ws, cudaStream_t st, Profiler* prof);
int launch_conv2_dw_x3(const GradStepArgs& a, const Workspace& ws, cudaStream_t st, Profiler* prof, int* seg_len);
int configure_x3_gemm_kernels();
void launch_prep_w1_x3(const GroupTable& gt, const Workspace& ws, cudaStream_t st, Profiler* prof);
int launch_fc1_fwd_x3(const GradStepArgs& a, const WorkerTable& wt, const GroupTable& gt, const Workspace& ws, cudaStream_t st, Profiler* prof, bool after_join);
int launch_fc1_dx_x3(const GradStepArgs& a, const WorkerTable& wt, const GroupTable& gt, const Workspace& ws, cudaStream_t st, Profiler* prof);
int launch_fc1_dw_x3(const GradStepArgs& a, const WorkerTable& wt, const GroupTable& gt, const Workspace& ws, cudaStream_t st, Profiler* prof);
extern int g_sm_count;   // SMs of the current device, set by configure_tc5_kernels
int configure_tc5_kernels();
int configure_conv5_kernels();
int configure_conv1_kernels();
int configure_dw5_kernels();
int configure_c1d5_kernels();
void launch_output_layer(bool eval, const GradStepArgs& a, const WorkerTable& wt, const GroupTable& gt, const Workspace& ws, cudaStream_t st, Profiler* prof);
int launch_conv1_dw_tc5(const GradStepArgs& a, const WorkerTable& wt, const Workspace& ws, cudaStream_t st, Profiler* prof,
                        int* seg_len);
int launch_conv2_dw_tc5(const GradStepArgs& a, const WorkerTable& wt, const Workspace& ws, cudaStream_t st, Profiler* prof,
                        int* seg_len, bool in_line);
int launch_conv1_fwd_planes(bool eval, const GradStepArgs& a, const WorkerTable& wt, const GroupTable& gt, const Workspace& ws,
                            cudaStream_t st, Profiler* prof);
const Bank2Taps& conv2_fwd_taps();
void launch_conv2_fwd_tc5(bool eval, const GradStepArgs& a, const WorkerTable& wt, const GroupTable& gt, const Workspace& ws,
                          cudaStream_t st, Profiler* prof);
void launch_conv2_dx_tc5(const GradStepArgs& a, const WorkerTable& wt, const GroupTable& gt, const Workspace& ws,
                         cudaStream_t st, Profiler* prof);
int launch_prep_w1(const GroupTable& gt, const Workspace& ws, cudaStream_t st, Profiler* prof);
int launch_fc1_fwd_tc5(const GradStepArgs& a, const WorkerTable& wt, const GroupTable& gt, const Workspace& ws,
                       cudaStream_t st, Profiler* prof, bool after_join = false);
int launch_fc1_dx_tc5(const GradStepArgs& a, const WorkerTable& wt, const GroupTable& gt, const Workspace& ws,
                      cudaStream_t st, Profiler* prof);
int launch_fc1_dw_tc5(const GradStepArgs& a, const WorkerTable& wt, const GroupTable& gt, const Workspace& ws,
                      cudaStream_t st, Profiler* prof);

// Part B.
struct SumApplyArgs {
  const float* queue;       // slot 0 of the gradient queue; slot k at queue + k*P_PAD
  int64_t K;                // gradients to sum (slots 0..K-1)
  const float* theta_in;    // current head
  float* theta_out;         // new head (may equal theta_in)
  float* replica;           // mirror target or nullptr
  float coef;               // lr*scale/divisor
  float* partial;           // [max_split][P_PAD] scratch
  int max_split;
  const float* coef_k;      // per-gradient factors [K] that replace coef (the stale-gradient treatments), or nullptr
};
int launch_sum_apply(const SumApplyArgs& a, cudaStream_t st, Profiler* prof);

constexpr int ASYNC_SEG = 256;   // gradients per ordered-apply launch
struct AsyncOrder { int32_t slot[ASYNC_SEG]; };
struct AsyncApplyArgs {
  const float* queue;
  int K;                    // 1..ASYNC_SEG gradients in this segment
  const float* theta_in;    // version v0
  float* ring[MAX_RING];    // ring slot buffers
  int ring_depth;
  uint64_t v0;              // version of theta_in; version v0+k+1 is stored in ring[(v0+k+1) % depth]
  int first_stored;         // only k >= first_stored are stored (the last ring_depth versions)
  int n_mirror;             // chain-replication stores of this segment (at most one per server behind the frontend)
  int mirror_k[MAX_CHAIN];  // k whose result is also written to replica[m]
  float* replica[MAX_CHAIN];
  float coef;               // lr*scale
  const float* coef_k;      // per-gradient factors indexed by queue slot that replace coef, or nullptr
};
int launch_async_apply(const AsyncApplyArgs& a, const AsyncOrder& ord, cudaStream_t st, Profiler* prof);

int launch_copy_rows(float* dst, const float* src, int64_t rows, cudaStream_t st, Profiler* prof);

// Clipping by global norm: coef_k[k] *= min(1, clip / ||queue[k]||_2) for k < K.  norm_part: [K][NORM_CHUNKS] scratch.
constexpr int NORM_CHUNKS = 8;
// Clipping, summing and applying in one pass (sync and replay steps).  words: CLIP_EXCHANGE_BYTES of scratch, where the
// CTAs exchange their partial sums of squares.  Returns 0, with nothing launched, where the kernel does not fit: on a device
// with too few SMs (clip_sum_fits), or in a stream confined to a part of it.
constexpr int NORM_WORDS = 160, CS_RING = 64, CS_COPIES = 8;      // words per copy (one per CTA, at most), gradients, copies
constexpr int CLIP_EXCHANGE_BYTES = NORM_WORDS * CS_RING * CS_COPIES * 8;
int configure_apply_kernels();
bool clip_sum_fits(int sms);
int launch_clip_sum_apply(const SumApplyArgs& a, float clip, uint64_t* words, uint32_t* status, cudaStream_t st, Profiler* prof);
int launch_clip_factors(const float* queue, int64_t K, float clip, float* coef_k, float* norm_part, cudaStream_t st, Profiler* prof);

// Evaluation pass: forward only, no dropout; loss [W] mean cross-entropy, argmax [W][b], correct [W] = samples whose
// argmax equals the label.  Returns the number of kernels launched or -1.
int launch_eval(const GradStepArgs& a, const WorkerTable& wt, const GroupTable& gt, const Workspace& ws, int32_t* correct,
                cudaStream_t st, Profiler* prof);

// One warp of four waits on a barrier nobody arrives at, for at most limit_cycles; all four then stop, and STATUS_WAIT_TIMEOUT
// is set in *status.
int launch_wait_timeout_probe(uint32_t* status, long long limit_cycles, cudaStream_t st);

}  // namespace psk
