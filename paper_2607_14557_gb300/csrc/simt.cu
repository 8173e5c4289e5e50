// CUDA-core kernels for fp32 storage (the small fp32 workload).  The tensor
// cores have no fp32-input mode, so fp32 layers run here with fp32 FMAs.
// Same epilogues and count hooks as the tcgen05 GEMM (tc_gemm.cu), and the
// same attention definition as tc_attn.cu (Sec. 3.6 Eqs. 6-7, 9-10).
#include <math.h>

#include "common.cuh"
#include "kernels.h"

namespace seer {
namespace {

__device__ __forceinline__ float silu_f(float g) { return g / (1.0f + __expf(-g)); }

// Asynchronous copy of VEC floats (16 or 4 bytes) to shared memory; the rest of a
// copy past `valid` is filled with zeros (nothing is read when !valid).
template <int VEC>
__device__ __forceinline__ void cp_async(float* dst, const float* src, bool valid) {
  if (VEC == 4)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(valid ? 16 : 0)
                 : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(valid ? 4 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Floats per staged row of TK: an odd number of 16-byte words, so 16-byte reads
// of 8 rows meet no bank twice.
__host__ __device__ constexpr int staged_ld(int tk) { return tk + 4; }

// acc.x += a0 * b0, acc.y += a1 * b1 (packed fp32 multiply-add, sm_100+).
__device__ __forceinline__ void ffma2(float2& acc, float a0, float a1, float b0, float b1) {
  asm("{\n\t.reg .b64 ra, rb, rc;\n\t"
      "mov.b64 ra, {%2, %3};\n\t"
      "mov.b64 rb, {%4, %5};\n\t"
      "mov.b64 rc, {%0, %1};\n\t"
      "fma.rn.f32x2 rc, ra, rb, rc;\n\t"
      "mov.b64 {%0, %1}, rc;\n\t}"
      : "+f"(acc.x), "+f"(acc.y) : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}

// C tile BM x BN per block, TM x TN outputs per thread (rows ty + i * TY, columns
// tx + j * TX).  Both operands stay row-major in shared memory (k contiguous) and
// a thread reads four k of a row with one 16-byte load, so four k cost TM + TN
// loads for 4 TM TN multiply-adds; STAGES k-steps are in flight by cp.async.  The
// multiply-adds are packed pairs: an output is the sum of its even-k and its odd-k
// chain; the detector's (Count) is one chain over ascending k.
// For Swiglu / Count the block holds BN / 2 gate columns and the matching up
// columns, and a thread's first TN / 2 columns are gates.
// Lanes: neighbours (lane ^ 1) differ in their row, lanes two apart in their column.
// A 16-byte shared-memory read takes four passes, or two where every lane shares its
// address with lane ^ 1 or with lane ^ 2; so both operands' reads take two.  With 16
// consecutive lanes along a row the columns' reads took four: 208 x 768 x 256 8.7 us
// (now 7.1 at the 16 x 32 tile), 208 x 512 x 1536 29.3 (24.8), 2624 x 512 x 1536 at the
// 32 x 64 tile 142.6 (136.2), 64 x 64 tiles -1%.
// Bound by the packed multiply-adds' register reads (44 TFLOP/s of 80 at the largest
// shape; a loop of them over an 8 x 4 tile in registers alone 46, scalar ones 66, but
// twice the instructions: scalar 42 here) and, for few rows, by the latency of the
// k-steps.
template <int MODE, int BM, int BN, int TM, int TN, int TK, int STAGES, int MIN_BLOCKS, int VEC>
__global__ void __launch_bounds__((BM / TM) * (BN / TN), MIN_BLOCKS)
    simt_gemm_kernel(const float* __restrict__ A, const float* __restrict__ B0, const float* __restrict__ B1,
                     const GemmParams p) {
  pdl_enter();
  constexpr int TX = BN / TN, TY = BM / TM, NTHR = TX * TY, LDT = staged_ld(TK);
  constexpr bool PAIR = MODE != kGemmCount;
  constexpr bool TWO = (MODE == kGemmSwiglu || MODE == kGemmCount);
  constexpr int COLS = TWO ? BN / 2 : BN;            // columns of p.N per block
  extern __shared__ float4 simt_smem[];
  float* sm = reinterpret_cast<float*>(simt_smem);   // [STAGES][BM + BN][LDT]

  int M = p.M_cap;
  int tiles_per_seq = 1;
  if (MODE == kGemmCount) {
    tiles_per_seq = (p.Nw + BM - 1) / BM;
  } else if (p.M_dev != nullptr) {
    const int md = *p.M_dev;
    if (md < 0 || md > p.M_cap) {
      if (threadIdx.x == 0 && blockIdx.x == 0 && blockIdx.y == 0) record_error(p.err, kErrRows);
      M = md < 0 ? 0 : p.M_cap;
    } else {
      M = md;
    }
  }
  const int mt = blockIdx.y, nt = blockIdx.x;
  int row_base, rows_here, seq = 0;
  if (MODE == kGemmCount) {
    seq = mt / tiles_per_seq;
    if (seq >= p.B) return;
    const int j = mt - seq * tiles_per_seq;
    const int rs = p.resp_start[seq];
    if (rs < 0 || rs + p.Nw > p.M_cap) {
      if (threadIdx.x == 0) record_error(p.err, kErrLayout);
      return;
    }
    row_base = rs + j * BM;
    rows_here = min(BM, p.Nw - j * BM);
  } else {
    row_base = mt * BM;
    if (row_base >= M) return;
    rows_here = min(BM, M - row_base);
  }
  const int col_base = nt * COLS;
  const int lane = threadIdx.x & 31;
  const int tx = (lane >> 1) % TX, ty = (threadIdx.x >> 5) * (32 / TX) + (lane & 1) + 2 * ((lane >> 1) / TX);

  // stage k0 .. k0 + TK - 1 of both operands (zeros past the rows, columns and K)
  auto load = [&](int stage, int k0) {
    float* dst = sm + stage * (BM + BN) * LDT;
    constexpr int PER_ROW = TK / VEC;
#pragma unroll 4
    for (int i = threadIdx.x; i < (BM + BN) * PER_ROW; i += NTHR) {
      const int r = i / PER_ROW, kk = (i % PER_ROW) * VEC;
      const bool kin = k0 + kk < p.K;                // K % VEC == 0
      const float* src = A;
      bool valid = false;
      if (r < BM) {
        valid = kin && r < rows_here;
        if (valid) src = A + static_cast<size_t>(row_base + r) * p.K + k0 + kk;
      } else {
        const int c = r - BM;
        const int col = col_base + (TWO && c >= COLS ? c - COLS : c);
        valid = kin && col < p.N;
        const float* w = TWO && c >= COLS ? B1 : B0;
        if (valid) src = w + static_cast<size_t>(col) * p.K + k0 + kk;
      }
      cp_async<VEC>(dst + r * LDT + kk, src, valid);
    }
    cp_async_commit();
  };

  float2 acc[TM][TN] = {};
  const int steps = (p.K + TK - 1) / TK;
#pragma unroll
  for (int s = 0; s < STAGES - 1; ++s) {
    if (s < steps) load(s, s * TK);
    else cp_async_commit();
  }
  for (int s = 0; s < steps; ++s) {
    cp_async_wait<STAGES - 2>();
    __syncthreads();                                 // step s landed; the stage filled next is read out
    if (s + STAGES - 1 < steps) load((s + STAGES - 1) % STAGES, (s + STAGES - 1) * TK);
    else cp_async_commit();
    const float* As = sm + (s % STAGES) * (BM + BN) * LDT;
    const float* Bs = As + BM * LDT;
#pragma unroll
    for (int k = 0; k < TK; k += 4) {
      float4 b[TN];
#pragma unroll
      for (int j = 0; j < TN; ++j) b[j] = *reinterpret_cast<const float4*>(Bs + (tx + j * TX) * LDT + k);
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const float4 a = *reinterpret_cast<const float4*>(As + (ty + i * TY) * LDT + k);
#pragma unroll
        for (int j = 0; j < TN; ++j) {
          if (PAIR) {
            ffma2(acc[i][j], a.x, a.y, b[j].x, b[j].y);
            ffma2(acc[i][j], a.z, a.w, b[j].z, b[j].w);
          } else {
            acc[i][j].x = fmaf(a.x, b[j].x, acc[i][j].x);
            acc[i][j].x = fmaf(a.y, b[j].y, acc[i][j].x);
            acc[i][j].x = fmaf(a.z, b[j].z, acc[i][j].x);
            acc[i][j].x = fmaf(a.w, b[j].w, acc[i][j].x);
          }
        }
      }
    }
  }

  float* C = reinterpret_cast<float*>(p.C);
  const float* R = reinterpret_cast<const float*>(p.R);
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int lr = ty + i * TY;
    const bool in = lr < rows_here;
    const int row = row_base + lr;
    int cnt = 0;
    if (in) {
#pragma unroll
      for (int j = 0; j < (TWO ? TN / 2 : TN); ++j) {
        const int col = col_base + tx + j * TX;
        if (col >= p.N) continue;
        const float v0 = PAIR ? acc[i][j].x + acc[i][j].y : acc[i][j].x;
        if (MODE == kGemmStore) {
          C[static_cast<size_t>(row) * p.ldc + col] = v0;
        } else if (MODE == kGemmResidual) {
          C[static_cast<size_t>(row) * p.ldc + col] = v0 + R[static_cast<size_t>(row) * p.ldr + col];
        } else {
          const float2 u = acc[i][TWO ? j + TN / 2 : j];
          const float v = silu_f(v0) * (PAIR ? u.x + u.y : u.x);
          cnt += fabsf(v) < p.act_eps ? 1 : 0;
          if (MODE == kGemmSwiglu) C[static_cast<size_t>(row) * p.ldc + col] = v;
        }
      }
    }
    if (TWO && p.counts != nullptr) {
      // a row's TX threads are every other lane: one atomic per row and block
#pragma unroll
      for (int off = TX; off > 1; off >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, off);
      if (in && tx == 0 && cnt > 0) {
        int idx = -1;
        if (MODE == kGemmCount) {
          idx = seq * p.Nw + (mt - seq * tiles_per_seq) * BM + lr;
        } else {
          int lo = 0, hi = p.B;
          while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (p.cu[mid] <= row) lo = mid; else hi = mid;
          }
          const int tl = row - p.resp_start[lo];
          if (tl >= 0 && tl < p.Nw && row < p.cu[lo + 1]) idx = lo * p.Nw + tl;
        }
        if (idx >= 0) atomicAdd(&p.counts[idx], cnt);
      }
    }
  }
}

// Attention of BQ query rows of one segment and head per block (16 x TY threads),
// keys in tiles of 64 with an online softmax (fp32, expf).
// Scores: a thread holds BQ / TY rows (ty + TY i) x 4 keys (tx + 16 j), Q and K
// row-major in shared memory and read four dims at a time; a row's 16 threads are
// every other lane of a warp, so its max and sum are shuffles; the probabilities go
// through shared memory and a thread accumulates its rows x the output columns
// 4 tx .. 4 tx + 3 (and + 64).  The next K tile is copied by cp.async while the
// current tile's softmax and PV run, the next V tile while the next scores do.
// Bound by shared-memory reads (two passes each, see the GEMM's lanes) beside as many
// FMA cycles.  A warp per (row, head) that reads every key itself took 1190 us for an
// 8-segment batch of 58 .. 790 rows, 8 heads of 64; this kernel 132.
// Blocks per SM are what its shared memory allows, so the registers are bounded to it:
// five blocks at 16 rows and 128 threads (without the bound 114 registers let four in,
// one segment of 1500 rows 216 -> 308 us); heads wider than 64 (HALVES = 2: a second
// float4 of output columns per thread) fit two blocks, and bounded as the others they
// spilled (four of 1000 rows, 4 heads of 128: 395 -> 441).
constexpr int AKV = 64;                      // keys per tile
constexpr int APS = AKV + 16;                // floats per row of probabilities (two rows meet no bank twice)

__host__ __device__ constexpr int attn_ld(int dh) { return 4 * ((dh / 4) | 1); }   // an odd number of 16-byte words

template <int BQ, int TY, int VEC, int HALVES>
__global__ void __launch_bounds__(16 * TY, HALVES == 2 ? 2 : (BQ == 32 ? 4 : (TY == 8 ? 5 : 3)))
    simt_attn_kernel(const float* __restrict__ qkv, const AttnParams p) {
  pdl_enter();
  constexpr int TM = BQ / TY;
  const int H = p.n_heads, dh = p.head_dim, D = H * dh;
  const int total = p.cu[p.B];
  if (total < 0 || total > p.T_cap) {
    if (blockIdx.x == 0 && threadIdx.x == 0) record_error(p.err, kErrRows);
    return;
  }
  // segments that no block's slot leads to are checked by the last block, whose own
  // slot is past every segment's tiles unless all of them end in a partial tile
  if (blockIdx.x == gridDim.x - 1)
    for (int b = threadIdx.x; b < p.B; b += blockDim.x)
      if (p.cu[b] < 0 || p.cu[b + 1] < p.cu[b] || p.cu[b + 1] > p.T_cap) record_error(p.err, kErrLayout);
  // slot -> (segment, query tile): the slots of segment b start at cu[b] / BQ + b,
  // at least as far apart as its tiles
  const int slot = blockIdx.x / H, h = blockIdx.x % H;
  int lo = 0, hi = p.B;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (p.cu[mid] / BQ + mid <= slot) lo = mid; else hi = mid;
  }
  const int seq0 = p.cu[lo], L = p.cu[lo + 1] - seq0;
  const int q0 = (slot - (seq0 / BQ + lo)) * BQ;
  if (q0 < 0 || q0 >= L) return;
  const int kv0 = p.cu_kv ? p.cu_kv[lo] : seq0;
  const int Lkv = p.cu_kv ? p.cu_kv[lo + 1] - kv0 : L;
  const int kvL = p.kv_len ? p.kv_len[lo] : Lkv;
  // rows outside either buffer are neither read nor written: the offsets come from the
  // device, and a segment's tiles reach all of cu[lo] .. cu[lo + 1] - 1
  if (seq0 < 0 || L > p.T_cap - seq0 || kvL <= 0 || kvL > Lkv || kv0 < 0 || kvL > p.kv_rows - kv0) {
    if (threadIdx.x == 0) record_error(p.err, kErrLayout);
    return;
  }
  const int rows = min(BQ, L - q0);
  const int ld = attn_ld(dh);
  extern __shared__ float4 simt_smem[];
  float* Qs = reinterpret_cast<float*>(simt_smem);   // [BQ][ld]
  float* Ks = Qs + BQ * ld;                           // [AKV][ld]
  float* Vs = Ks + AKV * ld;                          // [AKV][ld]
  float* Ps = Vs + AKV * ld;                          // [BQ][APS]
  const int tx = (threadIdx.x & 31) >> 1, ty = (threadIdx.x >> 5) * 2 + (threadIdx.x & 1);   // lanes as in the GEMM
  const int per_row = dh / VEC;

  for (int i = threadIdx.x; i < BQ * per_row; i += 16 * TY) {
    const int r = i / per_row, c = (i - r * per_row) * VEC;
    const bool valid = r < rows;
    cp_async<VEC>(Qs + r * ld + c, qkv + static_cast<size_t>(seq0 + q0 + (valid ? r : 0)) * 3 * D + h * dh + c, valid);
  }
  const float* kvsrc = p.kv ? static_cast<const float*>(p.kv) : qkv;
  auto load_keys = [&](float* dst, int column, int k0) {   // one K or V tile, zeros past the valid keys
    for (int i = threadIdx.x; i < AKV * per_row; i += 16 * TY) {
      const int r = i / per_row, c = (i - r * per_row) * VEC;
      const bool valid = k0 + r < kvL;
      cp_async<VEC>(dst + r * ld + c, kvsrc + static_cast<size_t>(kv0 + (valid ? k0 + r : 0)) * p.ld_kv + column + h * dh + c,
                    valid);
    }
    cp_async_commit();
  };
  load_keys(Ks, p.xk0, 0);                            // Q is part of this group
  load_keys(Vs, p.xv0, 0);

  const float scale = 1.0f / sqrtf(static_cast<float>(dh));
  float m[TM], l[TM], o[TM][4 * HALVES];
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    m[i] = -INFINITY;
    l[i] = 0.f;
#pragma unroll
    for (int c = 0; c < 4 * HALVES; ++c) o[i][c] = 0.f;
  }
  const int c0 = 4 * tx;                              // output columns of this thread: c0 .. c0 + 3 (and + 64)
  const int tiles = (kvL + AKV - 1) / AKV;
  for (int t = 0; t < tiles; ++t) {
    cp_async_wait<1>();                               // K of tile t (its V is the group after)
    __syncthreads();
    // A score is summed in blocks of 16 dims, each two packed chains of 8, and the blocks
    // in two chains: about the roundings of a tree over a warp's lanes.  One chain over the
    // head's dims was up to 2.5 times further from 64 bits (q and k of size 3, 2 heads of
    // 128, 1000 rows: 1.76e-6; so 5.7e-7, a warp per row 7.0e-7; of size 1 7.0e-7, 5.9e-7
    // and 7.5e-7) and no faster at heads of 64 (132 and 136 us above; of 128 2-4% faster).
    float sc[TM][4] = {}, odd[TM][4] = {};
    for (int k0 = 0; k0 < dh; k0 += 16) {
      float2 part[TM][4] = {};
#pragma unroll 1
      for (int k = k0; k < min(k0 + 16, dh); k += 4) {
        float4 kk[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) kk[j] = *reinterpret_cast<const float4*>(Ks + (tx + 16 * j) * ld + k);
#pragma unroll
        for (int i = 0; i < TM; ++i) {
          const float4 q = *reinterpret_cast<const float4*>(Qs + (ty + TY * i) * ld + k);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            ffma2(part[i][j], q.x, q.y, kk[j].x, kk[j].y);
            ffma2(part[i][j], q.z, q.w, kk[j].z, kk[j].w);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float v = part[i][j].x + part[i][j].y;
          if (k0 & 16) odd[i][j] += v;
          else sc[i][j] += v;
        }
    }
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) sc[i][j] += odd[i][j];
    __syncthreads();                                  // every warp is done with K
    if (t + 1 < tiles) load_keys(Ks, p.xk0, (t + 1) * AKV);
    else cp_async_commit();
    const int valid = kvL - t * AKV;                  // keys of this tile, >= 1
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      float mx = m[i];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        sc[i][j] = tx + 16 * j < valid ? sc[i][j] * scale : -INFINITY;
        mx = fmaxf(mx, sc[i][j]);
      }
#pragma unroll
      for (int off = 16; off > 1; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
      const float alpha = expf(m[i] - mx);
      m[i] = mx;
      float sum = 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float e = expf(sc[i][j] - mx);
        sum += e;
        Ps[(ty + TY * i) * APS + tx + 16 * j] = e;
      }
      l[i] = l[i] * alpha + sum;                      // this thread's share; summed over the row at the end
#pragma unroll
      for (int c = 0; c < 4 * HALVES; ++c) o[i][c] *= alpha;
    }
    cp_async_wait<1>();                               // V of tile t
    __syncthreads();
    const int keys = min(AKV, (valid + 3) & ~3);      // past the valid keys P is 0 and V is zero-filled
    for (int k = 0; k < keys; k += 4) {
      float4 pr[TM];
#pragma unroll
      for (int i = 0; i < TM; ++i) pr[i] = *reinterpret_cast<const float4*>(Ps + (ty + TY * i) * APS + k);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float* vrow = Vs + (k + e) * ld;
#pragma unroll
        for (int h2 = 0; h2 < HALVES; ++h2) {
          if (c0 + 64 * h2 >= dh) continue;
          const float4 v = *reinterpret_cast<const float4*>(vrow + c0 + 64 * h2);
#pragma unroll
          for (int i = 0; i < TM; ++i) {
            const float w = e == 0 ? pr[i].x : (e == 1 ? pr[i].y : (e == 2 ? pr[i].z : pr[i].w));
            o[i][4 * h2 + 0] = fmaf(w, v.x, o[i][4 * h2 + 0]);
            o[i][4 * h2 + 1] = fmaf(w, v.y, o[i][4 * h2 + 1]);
            o[i][4 * h2 + 2] = fmaf(w, v.z, o[i][4 * h2 + 2]);
            o[i][4 * h2 + 3] = fmaf(w, v.w, o[i][4 * h2 + 3]);
          }
        }
      }
    }
    __syncthreads();                                  // every warp is done with V
    if (t + 1 < tiles) load_keys(Vs, p.xv0, (t + 1) * AKV);
    else cp_async_commit();
  }
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    float sum = l[i];
#pragma unroll
    for (int off = 16; off > 1; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
    const int r = ty + TY * i;
    if (r >= rows) continue;
    float* out = reinterpret_cast<float*>(p.out) + static_cast<size_t>(seq0 + q0 + r) * p.ldo + h * dh;
#pragma unroll
    for (int h2 = 0; h2 < HALVES; ++h2) {
      if (c0 + 64 * h2 >= dh) continue;
#pragma unroll
      for (int c = 0; c < 4; ++c) out[c0 + 64 * h2 + c] = o[i][4 * h2 + c] / sum;
    }
  }
}

}  // namespace

namespace {

template <int MODE, int BM, int BN, int TM, int TN, int TK, int STAGES, int MIN_BLOCKS, int VEC>
cudaError_t launch_vec(dim3 grid, const float* A, const float* B0, const float* B1, const GemmParams& p, cudaStream_t st) {
  constexpr int smem = static_cast<int>(sizeof(float)) * STAGES * (BM + BN) * staged_ld(TK);
  if (smem > 48 * 1024) {
    static bool attr_set[64] = {};
    cudaError_t e = set_smem_limit_once(simt_gemm_kernel<MODE, BM, BN, TM, TN, TK, STAGES, MIN_BLOCKS, VEC>, smem, attr_set);
    if (e != cudaSuccess) return e;
  }
  return launch_kernel(simt_gemm_kernel<MODE, BM, BN, TM, TN, TK, STAGES, MIN_BLOCKS, VEC>, grid, dim3((BM / TM) * (BN / TN)), smem, st,
                       A, B0, B1, p);
}

template <int MODE, int BM, int BN, int TM, int TN, int TK, int STAGES, int MIN_BLOCKS>
cudaError_t launch_tile(const float* A, const float* B0, const float* B1, const GemmParams& p, bool vec,
                        cudaStream_t st) {
  constexpr int COLS = (MODE == kGemmSwiglu || MODE == kGemmCount) ? BN / 2 : BN;
  const long mtiles = MODE == kGemmCount ? static_cast<long>(p.B) * ((p.Nw + BM - 1) / BM) : (p.M_cap + BM - 1l) / BM;
  const long ntiles = (p.N + COLS - 1l) / COLS;
  if (mtiles <= 0 || ntiles <= 0) return cudaSuccess;
  if (mtiles > 65535) return cudaErrorInvalidValue;
  const dim3 grid(static_cast<unsigned>(ntiles), static_cast<unsigned>(mtiles));
  return vec ? launch_vec<MODE, BM, BN, TM, TN, TK, STAGES, MIN_BLOCKS, 4>(grid, A, B0, B1, p, st)
             : launch_vec<MODE, BM, BN, TM, TN, TK, STAGES, MIN_BLOCKS, 1>(grid, A, B0, B1, p, st);
}

// The tile that is expected to finish first.  A k-step costs a block's share of its
// SM, `share`, for each of the n = tiles / SMs blocks of an SM (and half of one more:
// the last blocks do not spread evenly), but at least one, plus `latency`, what the
// blocks in flight do not hide.  Both in us per 32 k, fitted to 100 shapes of 64 ..
// 8192 rows (rms 6-7%; the choice is 1% from the best of the four tiles on average).
// The rule before (the largest tile that leaves every SM several blocks) was 5% from
// it, at worst a third: 208 x 3072 x 1024 69 -> 52 us, 1300 x 512 x 1536 109 -> 82, 2624 x
// 256 x 768 55 -> 42, 208 x 768 x 256 8.7 -> 7.1; none more than 1% slower.  At 64 x 64 / 32 x 64 / 32 x 32 / 16 x 32 tiles, us: 2624 x 1536 x 512 108 /
// 111 / 125 / 168 (a transposing 64 x 64 kernel 147); 2624 x 512 x 1536 148 / 136 / 134 /
// 171 (191); 208 x 256 x 768 40 / 25 / 16 / 11.4 (44); 8192 x 4096 x 1024 44 TFLOP/s at
// 64 x 64.
template <int MODE>
cudaError_t launch_mode(const float* A, const float* B0, const float* B1, const GemmParams& p, int num_sms,
                        cudaStream_t st) {
  const auto aligned = [](const float* q) { return (reinterpret_cast<uintptr_t>(q) & 15u) == 0; };
  const bool vec = p.K % 4 == 0 && aligned(A) && aligned(B0) && (B1 == nullptr || aligned(B1));
  constexpr bool TWO = MODE == kGemmSwiglu || MODE == kGemmCount;
  const auto m_tiles = [&](int bm) {
    return MODE == kGemmCount ? static_cast<long>(p.B) * ((p.Nw + bm - 1) / bm) : (p.M_cap + bm - 1l) / bm;
  };
  const auto tiles = [&](int bm, int bn) { return m_tiles(bm) * ((p.N + (TWO ? bn / 2 : bn) - 1l) / (TWO ? bn / 2 : bn)); };
  const auto cost = [&](int bm, int bn, float latency, float share) {
    if (bm < 64 && m_tiles(bm) > 65535) return INFINITY;   // more row tiles than a grid takes
    return latency + share * fmaxf(1.0f, static_cast<float>(tiles(bm, bn)) / static_cast<float>(num_sms) + 0.5f);
  };
  const float t0 = cost(64, 64, 0.62f, 0.89f), t1 = cost(32, 64, 0.42f, 0.49f), t2 = cost(32, 32, 0.22f, 0.29f);
  const float t3 = cost(16, 32, 0.08f, 0.205f), best = fminf(fminf(t0, t1), fminf(t2, t3));
  if (t0 == best) return launch_tile<MODE, 64, 64, 8, 4, 32, 3, 3>(A, B0, B1, p, vec, st);
  if (t1 == best) return launch_tile<MODE, 32, 64, 4, 4, 32, 4, 4>(A, B0, B1, p, vec, st);
  if (t2 == best) return launch_tile<MODE, 32, 32, 4, 2, 32, 5, 1>(A, B0, B1, p, vec, st);
  return launch_tile<MODE, 16, 32, 2, 2, 32, 6, 1>(A, B0, B1, p, vec, st);
}

template <int BQ, int TY, int VEC, int HALVES>
cudaError_t launch_attn_halves(const float* qkv, const AttnParams& p, cudaStream_t st) {
  const long blocks = ((static_cast<long>(p.T_cap) + BQ - 1) / BQ + p.B) * p.n_heads;
  if (blocks > 0x7fffffffL) return cudaErrorInvalidValue;
  constexpr auto bytes = [](int dh) { return static_cast<int>(sizeof(float)) * ((BQ + 2 * AKV) * attn_ld(dh) + BQ * APS); };
  static bool attr_set[64] = {};
  cudaError_t e = set_smem_limit_once(simt_attn_kernel<BQ, TY, VEC, HALVES>, bytes(64 * HALVES), attr_set);
  if (e != cudaSuccess) return e;
  return launch_kernel(simt_attn_kernel<BQ, TY, VEC, HALVES>, dim3(static_cast<unsigned>(blocks)), dim3(16 * TY),
                       bytes(p.head_dim), st, qkv, p);
}

template <int BQ, int TY, int VEC>
cudaError_t launch_attn(const float* qkv, const AttnParams& p, cudaStream_t st) {
  return p.head_dim <= 64 ? launch_attn_halves<BQ, TY, VEC, 1>(qkv, p, st) : launch_attn_halves<BQ, TY, VEC, 2>(qkv, p, st);
}

}  // namespace

cudaError_t launch_simt_gemm(int mode, const float* A, const float* B0, const float* B1, const GemmParams& p,
                             int num_sms, cudaStream_t st) {
  switch (mode) {
    case kGemmStore: return launch_mode<kGemmStore>(A, B0, B1, p, num_sms, st);
    case kGemmResidual: return launch_mode<kGemmResidual>(A, B0, B1, p, num_sms, st);
    case kGemmSwiglu: return launch_mode<kGemmSwiglu>(A, B0, B1, p, num_sms, st);
    case kGemmCount: return launch_mode<kGemmCount>(A, B0, B1, p, num_sms, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_simt_attn(const float* qkv, const AttnParams& p, int num_sms, cudaStream_t st) {
  if (p.T_cap <= 0) return cudaSuccess;
  const auto aligned = [](const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15u) == 0; };
  // rows of the separate K/V source start 16-byte aligned when its width and columns do
  const bool vec = aligned(qkv) && (p.kv == nullptr || (aligned(p.kv) && p.ld_kv % 4 == 0)) && p.xk0 % 4 == 0 && p.xv0 % 4 == 0;
  // 32-row tiles once their blocks fill the SMs three times (unless most segments are
  // far shorter); else 16-row tiles, with twice the threads unless heads of at most 64
  // let five blocks share an SM and the blocks fill the SMs four times.  Measured at 32
  // rows / 16 rows / 16 rows with 256 threads, us: segments of 58 .. 790 rows, 8 heads of
  // 64 (4.7 times) 132 / 148 / 151; four of 500 (3.5) 92 / 109 / 115; four of 800, 4 heads
  // of 128 (2.7) 281 / 348 / 273; one of 1500, 8 heads of 64 (2.5; 16 rows 4.9) 262 / 216 /
  // 241; one of 700 (1.2; 2.3) 85 / 90 / 69; sixteen of 60, 8 heads of 32 (2.4; 4.0) 13.0 /
  // 10.8 / 10.8; one of 121, 4 heads 15.4 / 11.5 / 8.1.  Of 28 shapes it misses the best by
  // more than 5% at four: six of 300, 8 heads of 128 126 / 138 / 109; one of 1000 199 / 287 /
  // 225; eight of 300, 8 heads of 32 71 / 64 / 64; eight of 40, 8 heads of 64 9.7 / 7.8 / 8.5.
  const auto blocks = [&](long bq) { return (p.T_cap / bq + p.B) * p.n_heads; };
  if (blocks(32) >= 3l * num_sms && p.T_cap / p.B >= 16)
    return vec ? launch_attn<32, 8, 4>(qkv, p, st) : launch_attn<32, 8, 1>(qkv, p, st);
  if (p.head_dim <= 64 && blocks(16) > 4l * num_sms)
    return vec ? launch_attn<16, 8, 4>(qkv, p, st) : launch_attn<16, 8, 1>(qkv, p, st);
  return vec ? launch_attn<16, 16, 4>(qkv, p, st) : launch_attn<16, 16, 1>(qkv, p, st);
}

}  // namespace seer
