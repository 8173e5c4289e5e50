// Internal launch interface between the C-ABI layer (seer_api.cu) and the
// kernel translation units.  Not part of the public ABI.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace seer {

// Epilogue variants of the GEMM kernels.
enum GemmMode : int {
  kGemmStore = 0,     // C = A B^T
  kGemmResidual = 1,  // C = A B^T + R
  kGemmSwiglu = 2,    // act = SiLU(A Bg^T) * (A Bu^T), optional near-zero counts
  kGemmCount = 3,     // counts only (detector): A rows gathered per sequence window
  kGemmRope = 4,      // C = A B^T, then columns < rope_cols rotated per head (rotary embedding)
  kGemmKv = 5,        // C = A B^T, columns >= split stored at mapped rows of a second matrix (K/V cache)
};

// Rows of segments that live at other places in another matrix: row r of segment
// b (cu[b] <= r < cu[b+1]) is row start[b] (+ add[b]) + r - cu[b] there.
struct RowMap {
  const int* cu;          // [B+1], or null: no mapping
  const int* start;       // [B]
  const int* add;         // [B], or null
  int B;
  int rows;               // rows of the other matrix
};

struct GemmParams {
  int M_cap;              // rows available in A / C
  const int* M_dev;       // optional device row count (<= M_cap)
  int N;                  // output columns (Swiglu/Count: F)
  int K;
  void* C;                // output [M, ldc]
  int ldc;
  const void* R;          // residual [M, ldr]
  int ldr;
  int* counts;            // [B * Nw] near-zero counts (Swiglu hook / Count)
  float act_eps;
  const int* cu;          // segment offsets [B+1] for the Swiglu count hook
  int B;
  const int* resp_start;  // first response row per sequence
  int Nw;                 // response window
  int* err;               // device error word
  uint32_t idesc;         // tcgen05 instruction descriptor (operand type f16 or bf16)
  int out_type;           // ElemType of C (kBF16 / kF16; kF32 on the CUDA-core path)
  int res_type;           // ElemType of R
  int bn;                 // accumulator columns per tile (multiple of 32)
  int stages;             // operand ring: stages
  int few_m;              // with at most this many row tiles (of cg * 128 rows), and bit (row tiles - 1) ...
  uint64_t few_mask;      // ... of this set (counts above 64: always), instead of bn ...
  int few_bn;             // ... this many columns per tile (single-weight modes; mB1 has its boxes) ...
  int few_stages;         // ... and stages
  int group_m;            // raster: row tiles per group (see tc_gemm.cu)
  const float2* rope_tab; // Rope: (cos, sin) of each row's 64 pairs
  int rope_cols;          // Rope: leading output columns that are rotated (the q|k columns)
  void* C2;               // Kv: matrix of the mapped columns [map.rows, ldc2]
  int ldc2;
  int split;              // Kv: first mapped column (multiple of 32)
  RowMap map;             // Kv: where its rows go
};

struct AttnParams {
  const int* cu;          // [B+1] query segment offsets (rows of the q source)
  const int* kv_len;      // [B] keys per segment, or null (= the K/V segment length)
  const int* cu_kv;       // [B+1] K/V segment offsets, or null (= cu: q, k, v share rows)
  const void* kv;         // K/V rows (fp32 path), or null (= the qkv buffer)
  int ld_kv;              // elements per K/V row
  int xk0, xv0;           // column of head 0's K and V inside a K/V row
  int B;
  int T_cap;
  int n_heads;
  int head_dim;
  void* out;              // [T, H*dh]
  int ldo;                // elements
  const int4* work;       // schedule: (b, h, first q-tile, q-tiles), or null: made in the kernel
  const int* work_count;  // units in `work`
  int* work_next;         // next unit to hand out (zeroed by the schedule kernel)
  int kv_rows;            // rows of the K/V source (capacity)
  bool keys_together;     // a unit's keys are not shared among CTAs
  int parts;              // CTAs sharing a unit's keys (set by launch_tc_attn)
  int* err;
};

// tcgen05 / TMA kernels (16-bit operands).  Tensor maps are encoded on the host.
// How one GEMM call is tiled: a tile is cg * 128 rows by bn accumulator columns,
// computed by cg SMs together.
struct GemmPlan {
  int cg;        // SMs per tile: 1, or 2 (paired tensor-core tiles)
  int bn;        // accumulator columns per tile (Swiglu / Count: bn / 2 of F)
  int stages;    // operand ring: stages
  int group_m;   // raster: row tiles per group
  int depth;     // 64-deep k-blocks per stage: 1 or 2
  int few_m;     // tile choice of a call whose device row count leaves at most few_m row
  int few_bn;    // tiles: few_bn columns (few_m = 0: no second choice), but for counts of
  uint64_t few_mask;   // up to 64 row tiles only those whose bit (row tiles - 1) is set
};
// m_tiles: 128-row tiles; n_cols: accumulator columns (N; Swiglu / Count: 2 F);
// K: depth; device_rows: the row count is read on the device (m_tiles is a bound);
// num_sms: SMs of the device.
GemmPlan tc_gemm_plan(int mode, long m_tiles, long n_cols, int K, bool device_rows, int num_sms);
// mC: the 16-bit output C (Store, Residual, Rope) or act (Swiglu) with 32 x 32
// boxes and no swizzle, for the epilogue's TMA stores (unused by Count).  mA
// has boxes of 128 rows, mB0 and mB1 boxes of bn / 2 rows (mB1 of few_bn / 2 where
// the plan has a second choice); mC2 is C2 in boxes
// like mC's (Kv only).
cudaError_t launch_tc_gemm(int mode, const GemmPlan& plan, const CUtensorMap& mA, const CUtensorMap& mB0,
                           const CUtensorMap& mB1, const CUtensorMap& mC, const CUtensorMap& mC2, const GemmParams& p,
                           int num_sms, cudaStream_t st);
int tc_attn_smem_bytes();
// persistent CTAs (at most one per SM) that take the units of the schedule from
// p.work_next until *p.work_count are done, or, where units are few and keys many,
// a cluster of CTAs per unit
cudaError_t launch_tc_attn(const CUtensorMap& mQ, const CUtensorMap& mKV, AttnParams p, bool f16, int num_sms,
                           cudaStream_t st);
// Whether the kernel makes the schedule of such a call itself (AttnParams::work null).
bool attn_schedules_itself(int B, int n_heads, int T_cap, int num_sms);
// Bytes of schedule workspace the 16-bit attention kernels need for a launch
// sized for T_cap rows, B segments and H heads: H * (ceil(T_cap/128) + B) work
// units of 16 bytes, rounded up to 256 bytes, plus 256 bytes for the unit
// count and the persistent kernel's unit counter.
size_t attn_sched_bytes(int T_cap, int B, int H);
// Arguments of the attention schedule: the units go to work (at most max_units),
// their number to work_count[0], and work_count[1] (the attention kernel's unit
// counter) is zeroed.
struct ScheduleArgs {
  const int* cu;
  const int* cu_kv;       // or null
  const int* kv_len;      // or null
  int B, n_heads, T_cap;
  int4* work;             // null: no schedule
  int* work_count;
  int max_units;
};
cudaError_t launch_attn_schedule(const ScheduleArgs& a, int* err, cudaStream_t st);

// cos and sin of the rotary angles of each row: tab[row * 64 + i] for pair i of a
// 128-wide head, rows of the segments cu[0 .. B].
struct RopeTable {
  float2* tab;            // [T_cap, 64], or null
  const int* cu;
  int B, T_cap;
  float theta;
};
cudaError_t launch_rope_table(const RopeTable& t, int* err, int num_sms, cudaStream_t st);

// What a layer's first norm can do beside its rows, in blocks of its own.
struct Prelude {
  ScheduleArgs sched;
  RopeTable rope;
};
// Whether launch_rmsnorm takes a prelude for these rows and segments.
bool norm_takes_prelude(int in_type, int out_type, int d, int B);

// CUDA-core kernels (fp32 storage; small shapes).
cudaError_t launch_simt_gemm(int mode, const float* A, const float* B0, const float* B1, const GemmParams& p,
                             int num_sms, cudaStream_t st);
cudaError_t launch_simt_attn(const float* qkv, const AttnParams& p, int num_sms, cudaStream_t st);

// Element-wise / scan kernels (both storage types).
// map.cu set: row r of y is the norm of the row of x that the map names (rows
// of segments outside x become zero and are recorded).  pre: also done, or null.
cudaError_t launch_rmsnorm(const void* x, int in_type, const void* g, void* y, int out_type, int M_cap,
                           const int* M_dev, int d, float eps, const RowMap& map, const Prelude* pre, int* err,
                           int num_sms, cudaStream_t st);
cudaError_t launch_rope(void* qkv, int type, const int* cu, int B, int T_cap, int n_heads, int head_dim, float theta,
                        int* err, int num_sms, cudaStream_t st);
// Per-segment row copies (see aux_kernels.cu): rows of segment b go from src
// rows src_start[b] (+ src_add[b]) to dst rows dst_start[b] (+ dst_add[b]);
// n = (len ? len[b] : src_start[b+1] - src_start[b]) (- len_sub[b]).
// Offsets and sizes in bytes; max_rows bounds any segment's n (grid size).
cudaError_t launch_rows_copy(const void* src, long src_ld, int src_c0, void* dst, long dst_ld, int dst_c0, int row_bytes,
                             const int* src_start, const int* src_add, const int* len, const int* len_sub,
                             const int* dst_start, const int* dst_add, int B, int src_rows, int dst_rows, int max_rows,
                             int* err, cudaStream_t st);
// cu_ctx = exclusive sums of ctx; cu_resp[b] = cu[b] - cu_ctx[b] (either output may be null).
cudaError_t launch_resp_layout(const int* cu, const int* ctx, int B, int* cu_resp, int* cu_ctx, int* err,
                               cudaStream_t st);
cudaError_t launch_zero(int* p, size_t n, int num_sms, cudaStream_t st);
// A bounded wait on a barrier that never completes (records kErrTimeout).
cudaError_t launch_wait_selftest(uint64_t limit_ns, int* err, cudaStream_t st);
cudaError_t launch_convert(const void* src, int in_type, void* dst, int out_type, size_t n, int* err, cudaStream_t st);
cudaError_t launch_snr_scan(const int* counts, int B, int N, int F, double tau_jump, double gamma, int window,
                            int* L_star, int* i_star, cudaStream_t st);
cudaError_t launch_pack_route(const void* x_full, int elem_bytes, const int* cu_full, const int* ctx_len,
                              const int* L_star, int B, int d, int N, int T_cap, double tau_pad,
                              int eager_max_bucket, int bucket_min, void* x_packed, int* cu_out, int* kv_out,
                              int* meta_out,
                              int* host_ctrl_dev, int epoch, int* err, int num_sms, cudaStream_t st);

// Sets the message returned by seer_last_error() on this thread.
void set_last_error(const char* msg);

constexpr int kCtrlMaxGroups = 32;
constexpr int kCtrlWords = 8 + 4 * kCtrlMaxGroups;

}  // namespace seer
