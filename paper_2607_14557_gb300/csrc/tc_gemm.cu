// Persistent tcgen05 GEMM for sm_103a: C[M, N] = A[M, K] * B[N, K]^T with
// 16-bit operands (both f16 or both bf16, chosen by the instruction
// descriptor) and fp32 accumulation in tensor memory (TMEM); C and the
// residual R are f16 or bf16 independently.
//
// A tile is 256 rows x bn columns computed by a pair of SMs (cta_group::2: each
// CTA of a 2-CTA cluster stages its own 128 rows of A and half of B's rows, one
// thread of the first CTA issues the MMAs for both, and each CTA's tensor memory
// receives its own rows), or 128 x bn by one SM when there is a single row tile.
// The pair reads a third less operand data per product than one-SM tiles of 128
// x 256 (64 instead of 96 bytes per clock and SM at the tensor rate), which
// leaves room for six stages instead of four; bn is chosen per call so that the
// last wave of tiles is nearly full (tc_gemm_plan, with the measured times).
//
// One CTA per SM, 192 threads, warp-specialised, persistent over the tiles:
//   warp 0      TMA producer: A and B tiles 64 deep (128-byte swizzle) into a
//               192 KB ring; in a pair every byte is counted on the first
//               CTA's barrier and a stage is released by a commit to both;
//   warp 1      TMEM allocator + MMA issuer: 4 x tcgen05.mma (K = 16) per stage
//               into one of two 256-column fp32 accumulators (double
//               buffered, 512 columns);
//               producer and issuer are whole warps in lockstep, one elected
//               lane issuing;
//   warps 2-5   epilogue: tcgen05.ld of the accumulator (each warp owns one
//               32-lane quarter of TMEM = 32 output rows), fused epilogue,
//               32 x 32 output chunks staged in shared memory and written by
//               TMA stores marked L2 evict-first (a tile whose rows run past
//               the device row count stores its valid rows lane by lane).
// The epilogue of tile t overlaps the main loop of tile t+1.  Every CTA sets up
// its barriers and tensor memory, then waits for the previous kernel of the
// stream (griddepcontrol.wait), and lets the next kernel launch once its last
// MMAs are issued.
//
// Epilogues (Sec. 3.1 Eq. 2 projections; Sec. 3.2 sparsity hook):
//   Store     C = A B^T                                    (QKV projection)
//   Residual  C = A B^T + R                                (O / down projection)
//   Swiglu    B = [Wg tile ; Wu tile] -> act = SiLU(g) * u  (gate/up), plus the
//             per-row count of |act| < eps on response rows (step-0 hook)
//   Count     detector: A rows gathered per sequence window, counts only
//   Rope      Store, then the q|k columns rotated per 128-wide head by the
//             rotary embedding at each row's position in its sequence
//   Kv        Store, with the columns past a split going to mapped rows of a second
//             matrix: the K | V projections straight into a K/V cache
// Every stored 16-bit value passes a range guard: an infinite or NaN result
// (an f16 intermediate that overflowed +-65504) records kErrRange in the
// device error word, which seer_check_device reports.
#include <math.h>

#include "common.cuh"
#include "kernels.h"

namespace seer {
namespace {

constexpr int BM = 128;                              // rows per CTA of a tile
constexpr int BK = 64;
constexpr int A_TILE_BYTES = BM * BK * 2;            // 16 KB
constexpr int MAX_STAGES = 12;
constexpr int THREADS = 192;
constexpr int ACC_COLS = 256;                        // one of the two accumulators
constexpr int TMEM_COLS = 512;
constexpr int BAR_BYTES = 256;
constexpr int ROPE_HEAD = 128;                       // head width of the Rope epilogue
constexpr int EPI_CHUNK = 32 * 32 * 2;              // a warp's 32 rows x 32 columns, 16-bit
constexpr int EPI_BYTES = 4 * 2 * EPI_CHUNK;         // 4 epilogue warps x 2 staging buffers
constexpr int FIXED_BYTES = BAR_BYTES + EPI_BYTES + 1024;
constexpr int RING_BYTES = 196608;                   // operand ring: six stages of a 256-column pair tile
static_assert(8 * (2 * MAX_STAGES + 4) + 8 <= BAR_BYTES, "barrier block");
static_assert(RING_BYTES + FIXED_BYTES <= 232448, "shared memory per CTA");

// Operand bytes one CTA stages per 64-deep k-block.
__host__ __device__ constexpr int stage_bytes(int cg, int bn) { return A_TILE_BYTES + bn / cg * BK * 2; }

// Raster: groups of `group_m` row tiles; inside a group m varies fastest and
// the group sweeps every n-tile.  group_m = 1 keeps the whole B operand hot in
// L2 while A streams once; a larger group_m keeps a slab of A hot while B
// streams once per group (chosen in tc_gemm_plan).
__device__ __forceinline__ void tile_coords(int t, int num_m, int num_n, int group_m, int& m, int& n) {
  const int per_group = group_m * num_n;
  const int g = t / per_group;
  const int r = t - g * per_group;
  const int m0 = g * group_m;
  const int gm = min(group_m, num_m - m0);
  m = m0 + r % gm;
  n = r / gm;
}

__device__ __forceinline__ float silu_f(float g) { return g / (1.0f + __expf(-g)); }
// The same with the approximate quotient (2 ulp, and 0 where 1 + exp(-g) passes
// 2^126): no branch, so the 32 activations of a chunk run side by side.  The IEEE
// division's slow-path branch made each thread compute them one after the other,
// ~15 us per 128 x 128 tile, exposed at the end of every call (one 8B layer with
// its detector at 842 rows: 440 -> 416 us, the cached layer at 848 rows 434 -> 418).
// Its values are stored in 16 bits, and the error of those against 64 bits is the same
// to four digits (300 x 2048 x 1024: f16 2.077e-4, bf16 1.654e-3); counts are decided on
// the IEEE value (count_near_zero).  Where g < -87.3 the quotient's 0 is what f16 operands
// and results give as well; with bf16 ones on either side the IEEE value may be stored
// (at least 1e-38, or u beyond 1e30), so a chunk with such a g is computed again.
__device__ __forceinline__ float silu_fast(float g) { return __fdividef(g, 1.0f + __expf(-g)); }

// Number of |SiLU(g) * u| < eps over a chunk, as the IEEE division decides it; a
// holds the fast values.  Those differ from the IEEE ones by at most 4 ulp, or
// where g < -87 the fast quotient may be 0, so only a chunk with a value within
// 2^-18 of eps, or such a g, is computed again.
__device__ __forceinline__ int count_near_zero(const float (&a)[32], const uint32_t (&g)[32], const uint32_t (&u)[32],
                                               float eps) {
  const float band = eps * 0x1p-18f;
  int cnt = 0;
  bool near = false;
  float g_min = 0.f;
#pragma unroll
  for (int i = 0; i < 32; ++i) {
    const float v = fabsf(a[i]);
    cnt += v < eps ? 1 : 0;
    near = near || fabsf(v - eps) < band;
    g_min = fminf(g_min, __uint_as_float(g[i]));
  }
  if (near || g_min < -87.f) {
    cnt = 0;
#pragma unroll
    for (int i = 0; i < 32; ++i)
      cnt += fabsf(silu_f(__uint_as_float(g[i])) * __uint_as_float(u[i])) < eps ? 1 : 0;
  }
  return cnt;
}

template <int MODE, int CG, int DEPTH>
__global__ void __launch_bounds__(THREADS, 1)
    tc_gemm_kernel(const __grid_constant__ CUtensorMap mA, const __grid_constant__ CUtensorMap mB0,
                   const __grid_constant__ CUtensorMap mB1, const __grid_constant__ CUtensorMap mC,
                   const __grid_constant__ CUtensorMap mC2, const GemmParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* fixed = smem + RING_BYTES;
  uint64_t* full = reinterpret_cast<uint64_t*>(fixed);
  uint64_t* empty = full + MAX_STAGES;
  uint64_t* acc_full = empty + MAX_STAGES;
  uint64_t* acc_empty = acc_full + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  uint8_t* epi_stage = fixed + BAR_BYTES;                // [4 warps][2][EPI_CHUNK]

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = CG == 2 ? cluster_ctarank() : 0u;   // CTA of the pair; rank 0 issues the MMAs

  if (threadIdx.x == 0) {
    for (int s = 0; s < MAX_STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&acc_full[a], 1);
      mbar_init(&acc_empty[a], 4 * CG);                     // every epilogue warp of the tile's CTAs
    }
    *abort_flag = 0;
    fence_barrier_init();
    tma_prefetch_desc(&mA);
    tma_prefetch_desc(&mB0);
    tma_prefetch_desc(&mB1);
  }
  if (warp == 1) tmem_alloc<CG>(tmem_slot, TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  if (CG == 2) cluster_sync();                              // the peer's barriers are initialised
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  // barriers, tensor memory and descriptors are set up while the previous kernel
  // drains; nothing before this reads or writes global memory
  pdl_wait();

  // ---- problem size (device row counts are clamped, never trusted blindly)
  int M = p.M_cap;
  int num_mt, tiles_per_seq = 1;                            // 128-row tiles, one per CTA of a tile
  if (MODE == kGemmCount) {
    tiles_per_seq = (p.Nw + BM - 1) / BM;
    num_mt = p.B * tiles_per_seq;
  } else {
    if (p.M_dev != nullptr) {
      const int md = *p.M_dev;
      if (md < 0 || md > p.M_cap) {
        if (threadIdx.x == 0 && blockIdx.x == 0) record_error(p.err, kErrRows);
        M = md < 0 ? 0 : p.M_cap;
      } else {
        M = md;
      }
    }
    num_mt = (M + BM - 1) / BM;
  }
  constexpr bool halfN = (MODE == kGemmSwiglu || MODE == kGemmCount);
  // the tile choice for the rows there are: a call sized for more may be better off
  // with other tiles (tc_gemm_plan)
  const int num_m = (num_mt + CG - 1) / CG;
  const bool few = !halfN && MODE != kGemmRope && num_m > 0 && num_m <= p.few_m &&
                   (num_m > 64 || ((p.few_mask >> (num_m - 1)) & 1) != 0);
  const int BN = few ? p.few_bn : p.bn;
  const int stages = few ? p.few_stages : p.stages;         // of DEPTH k-blocks
  const int bbytes = stage_bytes(CG, BN);                   // operand bytes of a k-block
  const int sbytes = DEPTH * bbytes;
  const int tile_n = halfN ? BN / 2 : BN;                   // columns of p.N covered by a tile
  const int num_n = (p.N + tile_n - 1) / tile_n;
  const int num_tiles = num_m * num_n;
  const int KB = p.K / BK;
  const int group_m = p.group_m > 0 ? p.group_m : 1;
  const int t_first = blockIdx.x / CG, t_step = gridDim.x / CG;

  if (warp == 0) {
    // ------------------------------------------------ TMA producer
    // Producer and issuer run as whole warps in lockstep (every wait by all
    // lanes, with a warp-uniform outcome); the elected lane issues the copies
    // and MMAs.  A lone lane in a divergent branch loses issue slots to the
    // FMA-heavy epilogue warp on its SM sub-partition.
    // In a pair each CTA loads its own 128 rows of A and its half of B's rows
    // and counts the bytes on rank 0's barrier, which expects both CTAs' bytes;
    // each waits on its own `empty`, signalled in both by the MMAs' commit (by
    // then rank 0's barrier has completed the stage's phase, so a peer's bytes
    // can only reach the phase they belong to).
    const bool leader = elect_one();
    const uint32_t full0 = CG == 2 ? cluster_addr(full, 0) : 0u;
    const int half_b = BN / 2 * BK * 2;                     // bytes of one half of B's rows
    // both halves come from one matrix unless they are gate and up rows
    const CUtensorMap* mapB0 = few ? &mB1 : &mB0;
    const CUtensorMap* mapB1 = halfN ? &mB1 : mapB0;
    int s = 0;
    uint32_t ph = 0;
    long issued = 0;
    for (int t = t_first; t < num_tiles && !__any_sync(0xffffffffu, *abort_flag != 0); t += t_step) {
      int m, n;
      tile_coords(t, num_m, num_n, group_m, m, n);
      const int mt = m * CG + static_cast<int>(rank);
      int a_row;
      if (MODE == kGemmCount) {
        const int mv = min(mt, num_mt - 1);                 // a pair's second tile may not exist: any rows
        const int b = mv / tiles_per_seq;
        const int j = mv - b * tiles_per_seq;
        const int rs = p.resp_start[b];
        if (leader && (rs < 0 || rs + p.Nw > p.M_cap)) record_error(p.err, kErrLayout);
        a_row = rs + j * BM;
      } else {
        a_row = mt * BM;
      }
      const int b_row0 = n * tile_n;
      const int b_row1 = halfN ? n * tile_n : n * tile_n + BN / 2;
      bool ok = true;
      for (int kb = 0; kb < KB; kb += DEPTH) {
        if (!warp_wait(&empty[s], ph ^ 1u, abort_flag, p.err)) { ok = false; break; }
        if (leader) {
          const int here = DEPTH == 1 ? 1 : min(DEPTH, KB - kb);   // k-blocks of this stage
          uint8_t* sa = smem + s * sbytes;
          const uint32_t bar = full0 + static_cast<uint32_t>(s * sizeof(uint64_t));
          if (CG == 1) mbar_arrive_expect_tx(&full[s], here * bbytes);
          else if (rank == 0) mbar_arrive_expect_tx(&full[s], 2 * here * bbytes);
#pragma unroll
          for (int u = 0; u < DEPTH; ++u, sa += bbytes) {
            if (u > 0 && u >= here) break;
            const int x = (kb + u) * BK;
            if (CG == 1) {
              tma_load_2d(sa, &mA, &full[s], x, a_row);
              tma_load_2d(sa + A_TILE_BYTES, mapB0, &full[s], x, b_row0);
              tma_load_2d(sa + A_TILE_BYTES + half_b, mapB1, &full[s], x, b_row1);
            } else {
              tma_load_2d_pair(sa, &mA, bar, x, a_row);
              if (rank == 0) tma_load_2d_pair(sa + A_TILE_BYTES, mapB0, bar, x, b_row0);
              else tma_load_2d_pair(sa + A_TILE_BYTES, mapB1, bar, x, b_row1);
            }
          }
        }
        __syncwarp();
        ++issued;
        if (++s == stages) { s = 0; ph ^= 1u; }
      }
      if (!ok) break;
    }
    if (CG == 2) {
      // wait until the MMAs have released every stage (their commits arrive here too)
      for (int i = 0; i < stages && warp_wait(&empty[s], ph ^ 1u, abort_flag, p.err); ++i)
        if (++s == stages) { s = 0; ph ^= 1u; }
    }
    if (*abort_flag && leader && rank == 0) {
      // let copies still in flight land before the shared memory is released
      // (a pair's second CTA leaves only after this one, see the final barrier)
      const long first = issued > stages ? issued - stages : 0;
      for (long i = first; i < issued; ++i)
        mbar_wait_drain(&full[i % stages], static_cast<uint32_t>((i / stages) & 1), 200000000ull);
    }
    if (CG == 2 && rank != 0 && leader) pdl_trigger();      // rank 0 triggers after its last MMAs
  } else if (warp == 1) {
    // ------------------------------------------------ MMA issuer
    // Every lane waits for a stage and the lanes vote once per stage, between the elected
    // one's MMAs and its commit: the commit lets the stage be filled again, and a lane
    // still waiting for the old filling would then find the barrier's parity flipped
    // back and wait for nothing until the time limit.  The vote there delays no MMA (us
    // at 127 rows, QKV / O / down: 22.0 / 13.1 / 35.0; before the MMAs 22.1 / 13.6 / 35.3,
    // the elected lane waiting alone 22.7 / 13.8 / 37.0).
    const bool leader = elect_one();
    const uint32_t idesc = (p.idesc & ~(0x3Fu << 17)) | (static_cast<uint32_t>(BN >> 3) << 17);   // N of the tile
    int s = 0;
    uint32_t ph = 0;
    int acc = 0;
    uint32_t acc_ph = 0;
    for (int t = t_first; t < num_tiles && rank == 0; t += t_step) {
      if (!warp_wait(&acc_empty[acc], acc_ph ^ 1u, abort_flag, p.err)) break;
      tc_fence_after();
      const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(acc * ACC_COLS);
      bool ok = true;
      for (int kb = 0; kb < KB; kb += DEPTH) {
        const bool here = mbar_wait(&full[s], ph, abort_flag, p.err);
        tc_fence_after();
        if (leader && here) {
          const uint32_t sa = smem_u32(smem + s * sbytes);
          const uint64_t adesc = make_sdesc_sw128(sa, 16, 1024);
          const uint64_t bdesc = make_sdesc_sw128(sa + A_TILE_BYTES, 16, 1024);
#pragma unroll
          for (int u = 0; u < DEPTH; ++u) {
            if (u > 0 && kb + u >= KB) break;
            const uint64_t off = static_cast<uint64_t>((u * bbytes) >> 4);
#pragma unroll
            for (int k = 0; k < BK / 16; ++k) {
              // +32 bytes along K inside the 128-byte swizzle atom = +2 in the address field
              const uint32_t add = u > 0 || k > 0 || kb > 0 ? 1u : 0u;
              if (CG == 1) tc_mma_f16(d_tmem, adesc + off + 2 * k, bdesc + off + 2 * k, idesc, add);
              else tc_mma_f16_pair(d_tmem, adesc + off + 2 * k, bdesc + off + 2 * k, idesc, add);
            }
          }
        }
        if (!__all_sync(0xffffffffu, here)) { ok = false; break; }
        if (leader) {
          if (CG == 1) tc_commit(&empty[s]);
          else tc_commit_pair(&empty[s]);
        }
        if (++s == stages) { s = 0; ph ^= 1u; }
      }
      if (!ok) break;
      if (leader) {
        if (CG == 1) tc_commit(&acc_full[acc]);
        else tc_commit_pair(&acc_full[acc]);
      }
      __syncwarp();
      if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
    }
    if (leader && rank == 0) pdl_trigger();      // last MMAs issued: the next kernel may launch
  } else {
    // -------------------------------------------------- epilogue warps 2..5
    const int q = warp & 3;                    // TMEM lane quarter owned by this warp
    const int row_in_tile = q * 32 + lane;
    const uint32_t lane_off = static_cast<uint32_t>(q * 32) << 16;
    uint8_t* my_stage = epi_stage + q * 2 * EPI_CHUNK;
    // outputs stream through L2 marked evict-first, so they do not push the
    // operand slabs the raster keeps resident out of the cache
    const uint64_t out_policy = l2_policy_evict_first();
    int n_chunks = 0;                            // bulk stores issued by this warp (staging buffer = n & 1)
    // one staged 32 x 32 chunk of this warp's rows -> a TMA store at (x, y); the
    // buffer used two chunks ago is reused only once its store has read it
    auto store_chunk = [&](const CUtensorMap& map, const uint32_t (&w)[16], int x, int y) {
      uint8_t* buf = my_stage + (n_chunks & 1) * EPI_CHUNK;
      if (lane == 0 && n_chunks >= 2) bulk_wait_read_1();
      __syncwarp();
      uint4* d = reinterpret_cast<uint4*>(buf + lane * 64);
#pragma unroll
      for (int i = 0; i < 4; ++i) d[i] = make_uint4(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]);
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) {
        tma_store_2d_hint(&map, buf, x, y, out_policy);
        bulk_commit();
      }
      ++n_chunks;
    };
    int acc = 0;
    uint32_t acc_ph = 0;
    uint32_t nonfinite = 0;                      // range guard over this thread's stores
    const uint32_t acc_empty0 = CG == 2 ? cluster_addr(acc_empty, 0) : 0u;
    for (int t = t_first; t < num_tiles; t += t_step) {
      int m, n;
      tile_coords(t, num_m, num_n, group_m, m, n);
      const int mt = m * CG + static_cast<int>(rank);          // this CTA's 128-row tile
      // columns of this tile inside the matrix (the last tile may be narrower)
      const int cols = min(tile_n, p.N - n * tile_n);
      const bool slab_full = mt * BM + q * 32 + 32 <= M;       // this warp's 32 rows all valid: TMA store
      const bool of16 = p.out_type == kF16, rf16 = p.res_type == kF16;
      const int row = mt * BM + row_in_tile;
      const bool valid = row < M;
      // the tile's residual row is loaded while the MMAs run: fetched chunk by chunk
      // after them, its latency was most of the epilogue (O projection of 842 rows
      // 26.9 -> 25.0 us)
      uint4 res[MODE == kGemmResidual ? ACC_COLS / 8 : 1];
      if (MODE == kGemmResidual) {
        const uint4* rp = reinterpret_cast<const uint4*>(reinterpret_cast<const uint16_t*>(p.R) +
                                                         static_cast<size_t>(valid ? row : 0) * p.ldr + n * BN);
#pragma unroll
        for (int i = 0; i < ACC_COLS / 8; ++i) res[i] = valid && i * 8 < cols ? rp[i] : make_uint4(0, 0, 0, 0);
      }
      // Kv: where this row's columns past the split go, and whether the warp's 32
      // rows go to 32 consecutive ones (then a TMA store takes them together)
      int row2 = -1, row2_0 = -1;
      bool slab2 = false;
      if (MODE == kGemmKv) {
        row2 = valid ? mapped_row(p.map, row, p.M_cap, p.err) : -1;
        row2_0 = __shfl_sync(0xffffffffu, row2, 0);
        slab2 = __all_sync(0xffffffffu, row2 >= 0 && row2 == row2_0 + lane);
      }
      // warp-uniform outcome: the TMEM loads below are warp-collective, and
      // after an abort the lanes of a warp could otherwise decide differently
      if (!__all_sync(0xffffffffu, mbar_wait(&acc_full[acc], acc_ph, abort_flag, p.err))) break;
      tc_fence_after();
      const uint32_t tacc = tmem_base + lane_off + static_cast<uint32_t>(acc * ACC_COLS);
      if (MODE == kGemmRope) {
        // the tile holds whole heads; pair (c, c + 64) of a head rotates by pos * f_c,
        // its cos and sin read from the row's table (64 sincosf per row here lengthened
        // every call's last epilogue by several us)
        const bool rotate = n * BN < p.rope_cols;       // tile-uniform (rope_cols % 256 == 0, BN 128 or 256)
        const int heads = cols / ROPE_HEAD;
        uint16_t* crow = reinterpret_cast<uint16_t*>(p.C) + static_cast<size_t>(valid ? row : 0) * p.ldc + n * BN;
        const float4* trow = reinterpret_cast<const float4*>(p.rope_tab + static_cast<size_t>(valid ? row : 0) * (ROPE_HEAD / 2));
#pragma unroll 1
        for (int c = 0; c < ROPE_HEAD / 64; ++c) {
          float cs[32], sn[32];
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            const float4 t2 = rotate && valid ? trow[c * 16 + e] : make_float4(1.f, 0.f, 1.f, 0.f);
            cs[2 * e] = t2.x;
            sn[2 * e] = t2.y;
            cs[2 * e + 1] = t2.z;
            sn[2 * e + 1] = t2.w;
          }
#pragma unroll 1
          for (int hh = 0; hh < heads; ++hh) {
            const int c0 = hh * ROPE_HEAD + c * 32, c1 = c0 + ROPE_HEAD / 2;
            uint32_t r0[32], r1[32];
            tmem_ld32(tacc + c0, r0);
            tmem_ld32(tacc + c1, r1);
            tmem_ld_wait();
            if (slab_full || valid) {
              uint32_t q0[16], q1[16];
#pragma unroll
              for (int e = 0; e < 32; e += 2) {
                const float x0 = __uint_as_float(r0[e]), x1 = __uint_as_float(r1[e]);
                const float y0 = __uint_as_float(r0[e + 1]), y1 = __uint_as_float(r1[e + 1]);
                q0[e / 2] = pack2(fmaf(x0, cs[e], -x1 * sn[e]), fmaf(y0, cs[e + 1], -y1 * sn[e + 1]), of16);
                q1[e / 2] = pack2(fmaf(x1, cs[e], x0 * sn[e]), fmaf(y1, cs[e + 1], y0 * sn[e + 1]), of16);
                nonfinite |= nonfinite_term(q0[e / 2], of16) | nonfinite_term(q1[e / 2], of16);
              }
              if (slab_full) {
                store_chunk(mC, q0, n * BN + c0, mt * BM + q * 32);
                store_chunk(mC, q1, n * BN + c1, mt * BM + q * 32);
              } else {
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                  st_global_32(crow + c0 + 16 * i, q0[8 * i], q0[8 * i + 1], q0[8 * i + 2], q0[8 * i + 3], q0[8 * i + 4],
                               q0[8 * i + 5], q0[8 * i + 6], q0[8 * i + 7]);
                  st_global_32(crow + c1 + 16 * i, q1[8 * i], q1[8 * i + 1], q1[8 * i + 2], q1[8 * i + 3], q1[8 * i + 4],
                               q1[8 * i + 5], q1[8 * i + 6], q1[8 * i + 7]);
                }
              }
            }
          }
        }
      } else if (MODE == kGemmStore || MODE == kGemmResidual || MODE == kGemmKv) {
        // two chunks of 32 columns per step, their accumulator loads in flight together
#pragma unroll
        for (int c = 0; c < ACC_COLS / 32; c += 2) {
          if (c * 32 >= cols) break;
          uint32_t acc32[2][32];
          tmem_ld32(tacc + c * 32, acc32[0]);
          tmem_ld32(tacc + c * 32 + 32, acc32[1]);        // past bn: stale columns, not stored
          tmem_ld_wait();
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int col = n * BN + (c + h) * 32;
            const bool second = MODE == kGemmKv && col >= p.split;   // a chunk lies on one side of the split
            const bool slab = second ? slab2 : slab_full;
            if ((c + h) * 32 < cols && (slab || (second ? row2 >= 0 : valid))) {
              float v[32];
#pragma unroll
              for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(acc32[h][i]);
              if (MODE == kGemmResidual) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                  const uint4 rv = res[(c + h) * 4 + i];
                  v[8 * i + 0] += lo16(rv.x, rf16); v[8 * i + 1] += hi16(rv.x, rf16);
                  v[8 * i + 2] += lo16(rv.y, rf16); v[8 * i + 3] += hi16(rv.y, rf16);
                  v[8 * i + 4] += lo16(rv.z, rf16); v[8 * i + 5] += hi16(rv.z, rf16);
                  v[8 * i + 6] += lo16(rv.w, rf16); v[8 * i + 7] += hi16(rv.w, rf16);
                }
              }
              uint32_t w[16];
#pragma unroll
              for (int i = 0; i < 16; ++i) {
                w[i] = pack2(v[2 * i], v[2 * i + 1], of16);
                nonfinite |= nonfinite_term(w[i], of16);
              }
              if (slab) {
                store_chunk(second ? mC2 : mC, w, second ? col - p.split : col, second ? row2_0 : mt * BM + q * 32);
              } else {
                // a lane owns one row: 64 contiguous bytes
                uint16_t* crow = second ? reinterpret_cast<uint16_t*>(p.C2) + static_cast<size_t>(row2) * p.ldc2 + col - p.split
                                        : reinterpret_cast<uint16_t*>(p.C) + static_cast<size_t>(row) * p.ldc + col;
                st_global_32(crow, w[0], w[1], w[2], w[3], w[4], w[5], w[6], w[7]);
                st_global_32(crow + 16, w[8], w[9], w[10], w[11], w[12], w[13], w[14], w[15]);
              }
            }
          }
        }
      } else {
        // gate columns 0 .. BN/2 - 1, up columns BN/2 .. BN - 1 of the accumulator
        int cnt_idx = -1;
        bool store = false;
        if (MODE == kGemmCount) {
          const int b = mt / tiles_per_seq;
          const int tl = (mt - b * tiles_per_seq) * BM + row_in_tile;
          if (mt < num_mt && tl < p.Nw) cnt_idx = b * p.Nw + tl;
        } else {
          store = valid;
          if (store && p.counts != nullptr) {
            // segment of this row (binary search in cu), then its window offset
            int lo = 0, hi = p.B;
            while (hi - lo > 1) {
              const int mid = (lo + hi) >> 1;
              if (p.cu[mid] <= row) lo = mid; else hi = mid;
            }
            const int tl = row - p.resp_start[lo];
            if (tl >= 0 && tl < p.Nw && row < p.cu[lo + 1]) cnt_idx = lo * p.Nw + tl;
          }
        }
        int cnt = 0;
        const bool wide_range = !of16 || ((p.idesc >> 7) & 7u) != 0;   // bf16 operands or results
        uint16_t* arow =
            MODE == kGemmSwiglu ? reinterpret_cast<uint16_t*>(p.C) + static_cast<size_t>(store ? row : 0) * p.ldc + n * tile_n
                                : nullptr;
#pragma unroll 1
        for (int c = 0; c < cols / 32; ++c) {
          uint32_t g[32], u[32];
          tmem_ld32(tacc + c * 32, g);
          tmem_ld32(tacc + BN / 2 + c * 32, u);
          tmem_ld_wait();
          float a[32];
#pragma unroll
          for (int i = 0; i < 32; ++i) a[i] = silu_fast(__uint_as_float(g[i])) * __uint_as_float(u[i]);
          if (MODE == kGemmSwiglu && wide_range) {
            float g_min = 0.f;
#pragma unroll
            for (int i = 0; i < 32; ++i) g_min = fminf(g_min, __uint_as_float(g[i]));
            if (g_min < -87.f) {
#pragma unroll
              for (int i = 0; i < 32; ++i) a[i] = silu_f(__uint_as_float(g[i])) * __uint_as_float(u[i]);
            }
          }
          if (cnt_idx >= 0) cnt += count_near_zero(a, g, u, p.act_eps);
          if (MODE == kGemmSwiglu) {
            if (slab_full || store) {
              uint32_t w[16];
#pragma unroll
              for (int i = 0; i < 16; ++i) {
                w[i] = pack2(a[2 * i], a[2 * i + 1], of16);
                nonfinite |= nonfinite_term(w[i], of16);
              }
              if (slab_full) {
                store_chunk(mC, w, n * tile_n + c * 32, mt * BM + q * 32);
              } else {
                st_global_32(arow + c * 32, w[0], w[1], w[2], w[3], w[4], w[5], w[6], w[7]);
                st_global_32(arow + c * 32 + 16, w[8], w[9], w[10], w[11], w[12], w[13], w[14], w[15]);
              }
            }
          }
        }
        if (cnt_idx >= 0) atomicAdd(&p.counts[cnt_idx], cnt);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (CG == 1) mbar_arrive(&acc_empty[acc]);
        else mbar_arrive_cluster(acc_empty0 + static_cast<uint32_t>(acc * sizeof(uint64_t)));
      }
      if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
    }
    report_range(nonfinite, p.err);              // a stored value overflowed the 16-bit type (or was NaN)
    if (lane == 0) bulk_wait_all();              // outputs written before the CTA exits
    __syncwarp();
  }

  tc_fence_before();
  __syncthreads();
  // a pair leaves together: neither CTA's shared memory goes while the other's
  // MMAs, copies or arrivals may still reach it
  if (CG == 2) cluster_sync();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc<CG>(tmem_base, TMEM_COLS);
  }
}

int plan_stages(int cg, int bn, int depth) {
  const int fit = RING_BYTES / (depth * stage_bytes(cg, bn));
  return fit < MAX_STAGES ? fit : MAX_STAGES;
}

template <int MODE, int CG, int DEPTH>
cudaError_t launch_mode(const GemmPlan& plan, const CUtensorMap& mA, const CUtensorMap& mB0, const CUtensorMap& mB1,
                        const CUtensorMap& mC, const CUtensorMap& mC2, GemmParams p, int num_sms, cudaStream_t st) {
  static bool attr_set[64] = {};
  cudaError_t e = set_smem_limit_once(tc_gemm_kernel<MODE, CG, DEPTH>, RING_BYTES + FIXED_BYTES, attr_set);
  if (e != cudaSuccess) return e;
  long num_mt;
  if (MODE == kGemmCount) num_mt = static_cast<long>(p.B) * ((p.Nw + BM - 1) / BM);
  else num_mt = (p.M_cap + BM - 1) / BM;
  const auto tiles_of = [&](long m, int bn) {
    const int tile_n = (MODE == kGemmSwiglu || MODE == kGemmCount) ? bn / 2 : bn;
    return m * ((p.N + tile_n - 1) / tile_n);
  };
  const long num_m = (num_mt + CG - 1) / CG;
  long tiles = tiles_of(num_m, plan.bn);
  if (tiles <= 0) return cudaSuccess;
  if (plan.few_m > 0) {
    const long few = tiles_of(plan.few_m < num_m ? plan.few_m : num_m, plan.few_bn);
    if (few > tiles) tiles = few;
  }
  p.bn = plan.bn;
  p.few_m = plan.few_m;
  p.few_mask = plan.few_mask;
  p.few_bn = plan.few_bn;
  p.few_stages = plan.few_m > 0 ? plan_stages(CG, plan.few_bn, DEPTH) : 0;
  p.stages = plan.stages;
  p.group_m = plan.group_m;
  const int units = num_sms / CG;
  const int grid = static_cast<int>(tiles < units ? tiles : units);
  // long calls gain little from the overlap but lose nothing (one layer of 35k rows:
  // 11.9 ms either way); one of 842 rows 391 us without any, 383 with calls of up to
  // five tiles per SM overlapped, 379 with all
  return launch_kernel_overlap(launch_overlap_enabled(), CG, tc_gemm_kernel<MODE, CG, DEPTH>, dim3(grid * CG), dim3(THREADS),
                               RING_BYTES + FIXED_BYTES, st, mA, mB0, mB1, mC, mC2, p);
}

template <int MODE>
cudaError_t launch_cg(const GemmPlan& plan, const CUtensorMap& mA, const CUtensorMap& mB0, const CUtensorMap& mB1,
                      const CUtensorMap& mC, const CUtensorMap& mC2, const GemmParams& p, int num_sms, cudaStream_t st) {
  if (plan.cg == 2)
    return plan.depth == 2 ? launch_mode<MODE, 2, 2>(plan, mA, mB0, mB1, mC, mC2, p, num_sms, st)
                           : launch_mode<MODE, 2, 1>(plan, mA, mB0, mB1, mC, mC2, p, num_sms, st);
  return plan.depth == 2 ? launch_mode<MODE, 1, 2>(plan, mA, mB0, mB1, mC, mC2, p, num_sms, st)
                         : launch_mode<MODE, 1, 1>(plan, mA, mB0, mB1, mC, mC2, p, num_sms, st);
}

}  // namespace

// Tile choice: the tile with the smallest modelled time, waves of tiles x
// k-blocks x time of a k-block + the fixed part of a call (launch, first
// operands, last epilogue).  The constants (us) are fits to GB300 timings of the
// 8B layer's shapes at 127, 300, 842 and 2976 rows: per 64-deep k-block with all
// SMs busy a pair takes 0.281 at 256 columns (the tensor rate), 0.254 at 224, 0.22
// at 192, 0.19 at 160, 0.165 at 128 and 0.14 at 64; one SM, which stages a third
// more operand bytes per product, 0.366 / 0.35 / 0.29 / 0.2 at 256 / 224 / 192 / 128
// columns (the SMs together read ~15 TB/s from L2) and 0.15 at 32.  So pairs are
// the rule; one-SM tiles remain where a pair's second SM would idle (an odd,
// small number of row tiles), and narrower tiles where they fill the last wave.
// Examples (us, one-SM 256-column tiles -> chosen): 848 rows QKV 76.0 -> 59.5
// (224 columns, 2.9 waves of pairs instead of 2.2 of SMs), O 27.7 -> 25.0 and
// down 74.6 -> 59.6 (224: 76 tiles on 76 pairs); 127 rows QKV 31.5 -> 22.1, O 27.8 ->
// 13.2, down 71.7 -> 35.0; 2976 rows O 71.3 -> 59.4, down 215 -> 173; 35194 rows
// QKV 1990 -> 1927, down 2323 -> 2154.
// Narrow tiles stage two k-blocks at a time: the issuer's wait, vote, commit and loop
// per stage (~100 cycles) exceed what the MMAs of a narrow tile hide (127 rows, one
// k-block / two: O 15.4 / 13.2, down 37.2 / 35.0; 300 rows, pairs of 128 columns, O 17.4 /
// 17.8, down 39.7 / 40.3; at 224 columns 842 rows down 61.0 / 63.2).
// A row count read on the device may leave fewer row tiles than the call is sized
// for (a packed batch in buffers for its full windows): single-weight modes then get
// a second width for four fifths of the tiles, used at the counts of up to that many
// where the model has it ahead; and among choices within 8% of the best at full size the
// one that is best over both is taken.  With / without the second width, us at fills of
// 0.4, 0.8 and 1 of the rows a call is sized for: 640 rows QKV 26.2 / 28.4, 39 / 45, 46 / 46;
// 1049 rows O 19.9 / 28.5, 26 / 29, 31.6 / 30.2, down 44.8 / 70, 63 / 72, 80 / 75; 1500 rows down
// 53 / 53, 83 / 93, 97 / 97; 3000 rows O 36 / 40, 54 / 58, 62 / 62.  At every count below four fifths
// instead, 1500 rows down took 76 at 0.4 and 3000 rows 141 for 120 at 0.6.
GemmPlan tc_gemm_plan(int mode, long m_tiles, long n_cols, int K, bool device_rows, int num_sms) {
  const bool half_n = mode == kGemmSwiglu || mode == kGemmCount;
  // whole 32-column chunks of the output, and whole heads for Rope
  const int step = mode == kGemmRope ? 128 : (half_n ? 64 : 32);
  const auto cost = [&](int cg, int bn, long mt) {
    const long tiles = ((mt + cg - 1) / cg) * ((n_cols + bn - 1) / bn);
    const long units = num_sms / cg;
    const bool narrow = bn / cg <= 64;
    const double block = cg == 2 ? (narrow ? 0.115 + 0.0004 * bn : 0.03 + 0.001 * bn)
                                 : (narrow ? 0.143 + 0.0003 * bn : fmax(0.19, 0.08 + 0.00112 * bn));
    const double fixed = cg == 2 ? 6.0 + 0.015 * bn : 4.2 + 0.0125 * bn;
    return fixed + static_cast<double>((tiles + units - 1) / units) * (K / BK) * block;
  };
  // cheapest width for mt row tiles; narrower than 256 only where clearly faster
  const auto width = [&](int cg, long mt, int depth) {
    int best = 0;
    for (int bn = 256; bn >= step; bn -= step)
      if ((depth == 0 || depth == (bn / cg <= 64 ? 2 : 1)) && (best == 0 || cost(cg, bn, mt) < 0.98 * cost(cg, best, mt)))
        best = bn;
    return best;
  };
  const auto depth_of = [](int cg, int bn) { return bn / cg <= 64 ? 2 : 1; };
  const long few = device_rows && m_tiles > 2 ? (4 * m_tiles + 4) / 5 : m_tiles;
  const bool second = !half_n && mode != kGemmRope;

  GemmPlan g{2, width(2, m_tiles, 0), 0, 1, 1, 0, 0, 0};
  int one = width(1, m_tiles, 0);                      // the one-SM choice
  const double pair_full = cost(2, g.bn, m_tiles), one_full = cost(1, one, m_tiles);
  bool use_one = one_full < 0.98 * pair_full;
  if (few < m_tiles) {
    const int pair_bn = second ? width(2, few, depth_of(2, g.bn)) : g.bn;
    const int one_bn = second ? width(1, few, depth_of(1, one)) : one;
    const double pair_few = cost(2, pair_bn > 0 ? pair_bn : g.bn, few), one_few = cost(1, one_bn > 0 ? one_bn : one, few);
    if (fmax(pair_full, one_full) <= 1.08 * fmin(pair_full, one_full)) use_one = one_full + one_few < pair_full + pair_few;
    const int other = use_one ? one_bn : pair_bn, cg = use_one ? 1 : 2;
    if (second && other > 0 && other != (use_one ? one : g.bn)) {
      g.few_bn = other;
      g.few_m = static_cast<int>((few + cg - 1) / cg);
      const int full_bn = use_one ? one : g.bn;
      for (int m = 1; m <= (g.few_m < 64 ? g.few_m : 64); ++m)
        if (cost(cg, other, static_cast<long>(m) * cg) < cost(cg, full_bn, static_cast<long>(m) * cg))
          g.few_mask |= uint64_t{1} << (m - 1);
    }
  }
  if (use_one) {
    g.cg = 1;
    g.bn = one;
  }
  g.depth = depth_of(g.cg, g.bn);
  g.stages = plan_stages(g.cg, g.bn, g.depth);
  // L2 raster: the 76 pair tiles in flight form a block of about 16 x 5, so each
  // operand slab is shared by many SMs at once: 16 columns of tiles swept per row
  // tile where the matrix has no more, else groups of 16 row tiles.  Swept on GB300
  // (35194 rows, us): QKV 2137 / 1980 / 1934 / 1950 / 2134 at groups 1 / 8 / 16 / 24 /
  // 48, gate/up 4487 / 3991 / 3822 / 3821 / 4180, O (16 columns of tiles) 661 / 675 /
  // 674 / 682 / 743, down 2005 / 2039 / 2038 / 2073 / 2219.
  // Under the power cap the order is the same (gate/up 5250 / 4340 / 4255 / 4285 / 4790).
  g.group_m = (n_cols + g.bn - 1) / g.bn <= 16 ? 1 : 16;
  return g;
}

cudaError_t launch_tc_gemm(int mode, const GemmPlan& plan, const CUtensorMap& mA, const CUtensorMap& mB0,
                           const CUtensorMap& mB1, const CUtensorMap& mC, const CUtensorMap& mC2, const GemmParams& p,
                           int num_sms, cudaStream_t st) {
  switch (mode) {
    case kGemmStore: return launch_cg<kGemmStore>(plan, mA, mB0, mB1, mC, mC2, p, num_sms, st);
    case kGemmResidual: return launch_cg<kGemmResidual>(plan, mA, mB0, mB1, mC, mC2, p, num_sms, st);
    case kGemmSwiglu: return launch_cg<kGemmSwiglu>(plan, mA, mB0, mB1, mC, mC2, p, num_sms, st);
    case kGemmCount: return launch_cg<kGemmCount>(plan, mA, mB0, mB1, mC, mC2, p, num_sms, st);
    case kGemmKv: return launch_cg<kGemmKv>(plan, mA, mB0, mB1, mC, mC2, p, num_sms, st);
    case kGemmRope: return launch_cg<kGemmRope>(plan, mA, mB0, mB1, mC, mC2, p, num_sms, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace seer
