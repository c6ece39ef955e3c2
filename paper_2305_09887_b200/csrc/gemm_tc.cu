// The dense products of a GraphSAGE-mean layer on the 5th-generation tensor cores
// (tcgen05.mma, accumulators in tensor memory, operands staged by bulk-tensor loads).
//
// Activations live in memory as split bf16 planes (hi, lo); the weights are repacked into the
// same form once per step.  Each product is three bf16 MMAs accumulated in fp32:
// hi*hi + lo*hi + hi*lo (relative error per product about 2^-16).  Nothing is converted
// inside the main loop: bulk-tensor loads feed the tensor core directly.
//
//   rows kernel   D[128 rows x BN] = [A0 | A1] * B^T   -- forward ([H | Abar H] times [Ws; Wn],
//                 bias + ReLU epilogue, written back as planes, or as fp32 logits for the last
//                 layer) and dgrad ([dZ | Abar^T dZ] times [Ws^T; Wn^T], gated by the sign of H
//                 and written as planes over H).  A tiles are K-major straight from the planes,
//                 B from the repacked weights.
//   wgrad kernel  D[128 x 64 n] = dZ^T * [H | Abar H] over a chunk of rows.  Both
//                 operands are MN-major straight from the planes.  Rows between parts are
//                 zero in every plane, so chunks need no masking.  The bias gradient (column
//                 sums of dZ) is added up from the staged dZ tiles by the otherwise idle
//                 epilogue warps.
//
// The rows kernel also runs on pairs of blocks (a cluster of two, one MMA of 256 rows: rows_use_pairs).
//
// Warp roles: warp 0 = loader (one lane), warp 1 = TMEM owner and MMA issuer (one lane), the
// remaining warps = epilogue (each warp reads its quarter of the 128 TMEM lanes).  Every
// mbarrier wait is bounded; a wait that runs out raises the context's device error word and
// the block winds down.
#include <algorithm>
#include <cstdlib>

#include "tc_common.cuh"
#include "train.cuh"

namespace {

constexpr int TC_THREADS = 192;
constexpr int TC_BM = 128;
constexpr int TC_BK = 64;                     // bf16 per 128-byte swizzle row
constexpr int PLANE_TILE_BYTES = TC_BM * 128;  // one plane of an A tile: 16 KB
constexpr int MAX_STAGES = 4;
constexpr int SMEM_BUDGET = 200 * 1024;

struct PipeBarriers {
    uint64_t full[MAX_STAGES];   // loads landed
    uint64_t empty[MAX_STAGES];  // MMA finished reading the stage
    uint64_t accum;              // all MMAs of the tile finished
    uint32_t tmem_base;
    int abort;
};

__device__ __forceinline__ bool wait_or_abort(uint64_t* bar, uint32_t parity, PipeBarriers* pb, int* error_word) {
    for (uint32_t i = 0; i < tc::WAIT_POLLS; ++i) {
        if (tc::mbar_try_wait(bar, parity)) return true;
        if ((i & 1023u) == 1023u && *reinterpret_cast<volatile int*>(&pb->abort)) break;
    }
    *reinterpret_cast<volatile int*>(&pb->abort) = 1;
    atomicExch(error_word, 1);
    return false;
}

__device__ __forceinline__ uint8_t* align_1024(uint8_t* p) {
    return reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(p) + 1023) & ~uintptr_t(1023));
}

// ------------------------------------------------------------------------------------
// weight repack: for every part of the group, B operands of the rows kernel
//   forward  Bf[n][kk], n < Npad_f, kk < Kf = 2 * 64 * ceil(d_in / 64):
//            kk <  Kf/2 : Ws[kk][n]          (zero beyond d_in / d_out)
//            kk >= Kf/2 : Wn[kk - Kf/2][n]
//   dgrad    Bd[j][kk], j < Npad_d (d_in valid), kk < Kd = 2 * 64 * ceil(d_out / 64):
//            kk <  Kd/2 : Ws[j][kk]          (zero beyond d_in / d_out)
//            kk >= Kd/2 : Wn[j][kk - Kd/2]
// each written as a hi and a lo bf16 matrix.
// Head form (head_cp > 0; the last layer when its aggregate is taken after the product,
// Abar (H Wn) instead of (Abar H) Wn): the weight matrices side by side along n,
//   forward  Bf[n][kk], kk < Kf = 64 * ceil(d_in / 64):
//            n <  head_cp : Ws[kk][n]           (zero beyond d_out)
//            n >= head_cp : Wn[kk][n - head_cp] (one-matrix layers have the first block only)
// ------------------------------------------------------------------------------------
struct PrepArgs {
    LayerShape ls;
    int head_cp;
    int Npad_f, Kf, Npad_d, Kd;
    __nv_bfloat16 *Bf_hi, *Bf_lo, *Bd_hi, *Bd_lo;  // [group slot][Npad][K]
};

constexpr int PREP_MAX_JOBS = 2 * RTMA_MAX_LAYERS;  // encoder and decoder layers of one step
struct PrepBatch {
    PrepArgs job[PREP_MAX_JOBS];
};

// blockIdx.z = layer (all layers of a step are repacked by one launch), blockIdx.y = part, blockIdx.x = tile of 32 rows
// (n or j) x 64 of K.  The forward operand is the transpose: its tile goes through shared memory, so that both the
// weights and the planes move in whole lines (read down their columns, one 32-byte sector per value, the weights took
// 17 us a step for 8 parts of 128-256-256-47).
constexpr int PREP_ROWS = 32, PREP_K = 64;
__host__ __device__ inline int prep_tiles(int npad, int k) { return (npad + PREP_ROWS - 1) / PREP_ROWS * (k / PREP_K); }

__global__ void __launch_bounds__(256)
tc_weight_prep_kernel(const __grid_constant__ GroupDesc g, const __grid_constant__ PrepBatch batch,
                      const float* __restrict__ params) {
    wait_for_kernel_before();
    __shared__ float tile[PREP_K][PREP_ROWS + 1];
    const PrepArgs& a = batch.job[blockIdx.z];
    const int k = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float* W = params + (int64_t)g.part[k] * a.ls.P + a.ls.param_offset;
    const int d_in = a.ls.d_in, d_out = a.ls.d_out, nsrc = a.ls.nsrc;
    const int fwd_tiles = prep_tiles(a.Npad_f, a.Kf);
    int at = blockIdx.x;
    if (at < fwd_tiles) {
        const int kt = a.Kf / PREP_K, n0 = at / kt * PREP_ROWS, kk0 = at % kt * PREP_K;
        const int n = n0 + lane;
        // head form: which weight matrix, which of its columns (at most two matrices); else one block of K per matrix
        const int blk = a.head_cp > 0 && n >= a.head_cp ? 1 : 0, c = n - blk * a.head_cp;
        const int half = a.head_cp > 0 || nsrc == 1 ? a.Kf : a.Kf / 2;
        const bool n_ok = blk < nsrc && c < d_out;
        float x[PREP_K / 8];
#pragma unroll
        for (int j = 0; j < PREP_K / 8; ++j) {
            const int kk = kk0 + warp + 8 * j;
            const int second = kk >= half ? 1 : 0, src = kk - second * half;
            x[j] = n_ok && src < d_in ? __ldg(W + (int64_t)((blk + second) * d_in + src) * d_out + c) : 0.f;
        }
#pragma unroll
        for (int j = 0; j < PREP_K / 8; ++j) tile[warp + 8 * j][lane] = x[j];
        __syncthreads();
#pragma unroll
        for (int j = 0; j < PREP_ROWS / 8; ++j) {
            const int r = warp + 8 * j;
            if (n0 + r >= a.Npad_f) break;
            uint32_t h, l;
            split_pair(tile[2 * lane][r], tile[2 * lane + 1][r], h, l);
            const int64_t o = ((int64_t)k * a.Npad_f + n0 + r) * a.Kf + kk0 + 2 * lane;
            *reinterpret_cast<uint32_t*>(a.Bf_hi + o) = h;
            *reinterpret_cast<uint32_t*>(a.Bf_lo + o) = l;
        }
        return;
    }
    at -= fwd_tiles;
    if (!a.Bd_hi || at >= prep_tiles(a.Npad_d, a.Kd)) return;
    const int kt = a.Kd / PREP_K, j0 = at / kt * PREP_ROWS, kk = at % kt * PREP_K + 2 * lane;
    const int half = nsrc == 1 ? a.Kd : a.Kd / 2;  // a multiple of 64: both of the lane's values lie in one block
    const int m = kk >= half ? 1 : 0, c = kk - m * half;
    float x[PREP_ROWS / 8][2];
#pragma unroll
    for (int j = 0; j < PREP_ROWS / 8; ++j) {
        const int row = j0 + warp + 8 * j;
        const float* w = W + (int64_t)(m * d_in + row) * d_out + c;
        x[j][0] = row < d_in && c < d_out ? __ldg(w) : 0.f;
        x[j][1] = row < d_in && c + 1 < d_out ? __ldg(w + 1) : 0.f;
    }
#pragma unroll
    for (int j = 0; j < PREP_ROWS / 8; ++j) {
        const int row = j0 + warp + 8 * j;
        if (row >= a.Npad_d) break;
        uint32_t h, l;
        split_pair(x[j][0], x[j][1], h, l);
        const int64_t o = ((int64_t)k * a.Npad_d + row) * a.Kd + kk;
        *reinterpret_cast<uint32_t*>(a.Bd_hi + o) = h;
        *reinterpret_cast<uint32_t*>(a.Bd_lo + o) = l;
    }
}

// ------------------------------------------------------------------------------------
// rows kernel
// ------------------------------------------------------------------------------------
struct RowsArgs {
    GroupDesc g;
    CUtensorMap mapA0h, mapA0l, mapA1h, mapA1l, mapBh, mapBl;
    CUtensorMap mapOh, mapOl;    // plane output: boxes of 64 columns x 32 rows
    CUtensorMap mapOh32, mapOl32;  // and of 32 x 32, for the last columns of a tile whose width is an odd multiple of 32
    int kb0, kb1;          // 64-wide k blocks taken from source 0 / source 1
    int BN, Npad, N;       // column tile, B rows per part, valid output columns
    int tmem_cols, stages; // columns of one accumulator buffer (two are allocated); pipeline depth
    int64_t row_tiles;     // 128-row tiles over all parts
    Planes out_planes;     // hi != NULL: write split planes
    float* out;            // else: fp32
    int64_t ld_out;
    const float* params;   // bias = params + part * P + bias_offset (bias_offset < 0: none)
    int64_t P, bias_offset;
    int relu;
    int single;            // 1: operands rounded to bf16 (hi planes only, one MMA per product)
    const __nv_bfloat16* gate_hi;  // plane output only: entries whose gate value (same row and column,
                                   // leading dimension of out_planes) is <= 0 become 0; NULL: none
    int* error_word;
};

// A role's walk over a block's tiles, which come in ascending order: the part reached and its first row tile are kept (looking
// a tile's place up anew, with a 64-bit division by the column tiles, cost every role 0.2 to 0.4 us of the 7 us of a tile).
template <int TILE_ROWS>
struct RowsWalk {
    int k = 0;
    uint32_t base = 0;
    // part, first row in it and first column of `tile`; false past the last part
    __device__ __forceinline__ bool at(const RowsArgs& a, uint32_t tile, uint32_t n_tiles, int* r0, int* n0) {
        const uint32_t row_tile = n_tiles == 1 ? tile : tile / n_tiles;
        while (k < a.g.num) {
            const uint32_t here = (uint32_t)(a.g.rows[k] + TILE_ROWS - 1) / TILE_ROWS;
            if (row_tile < base + here) break;
            base += here;
            ++k;
        }
        *r0 = (int)(row_tile - base) * TILE_ROWS;
        *n0 = n_tiles == 1 ? 0 : (int)(tile - row_tile * n_tiles) * a.BN;
        return k < a.g.num;
    }
};

// Persistent: a block walks tiles blockIdx.x, blockIdx.x + gridDim.x, ... (tile = row tile x
// column tile, column tiles of one row tile adjacent).  Two accumulator buffers in tensor
// memory let the epilogue of one tile overlap the main loop of the next; the shared-memory
// ring keeps running across tiles.  Warps: 0 = loader, 1 = MMA issuer / TMEM owner,
// 2..5 = epilogue (a warp per TMEM lane quarter, 64 columns at a time).
constexpr int ROWS_THREADS = 192;
constexpr int ROWS_EPI_WARPS = 4;
constexpr int ROWS_MAX_STAGES = 6;
enum RowsOut { OUT_F32, OUT_PLANES, OUT_GATED };  // fp32; split planes; split planes gated by the sign of `gate_hi`
constexpr int ROWS_SLAB_BYTES = 2 * 32 * 128;     // per epilogue warp: 32 rows x 64 columns of both planes
constexpr int ROWS_RING_BUDGET = 192 * 1024;      // shared memory for the operand ring
constexpr int ROWS_SMEM_MAX = ROWS_RING_BUDGET + 1024 + ROWS_EPI_WARPS * ROWS_SLAB_BYTES;

struct RowsBarriers {
    uint64_t full[ROWS_MAX_STAGES];
    uint64_t empty[ROWS_MAX_STAGES];
    uint64_t acc_full[2];   // all MMAs of the tile in this buffer finished
    uint64_t acc_empty[2];  // the epilogue has drained this buffer
    uint32_t tmem_base;
    int abort;
};

// PAIR: the barrier may be signalled from the pair's other block
template <bool PAIR>
__device__ __forceinline__ bool rows_wait(uint64_t* bar, uint32_t parity, RowsBarriers* pb, int* error_word) {
    for (uint32_t i = 0; i < tc::WAIT_POLLS; ++i) {
        if (PAIR ? tc::mbar_try_wait_cluster(bar, parity) : tc::mbar_try_wait(bar, parity)) return true;
        if ((i & 1023u) == 1023u && *reinterpret_cast<volatile int*>(&pb->abort)) break;
    }
    *reinterpret_cast<volatile int*>(&pb->abort) = 1;
    atomicExch(error_word, 1);
    return false;
}

// PAIR = false: a block works on tiles of 128 rows by itself.  PAIR = true: two blocks of a cluster work on tiles of
// 256 rows; `rank` 0 issues the MMAs of both (see tc_common.cuh).  HALF: the last 64 columns of a tile are 32 at most, which
// the epilogue finishes by themselves (compiled apart: the test costs gated tiles of 64 columns a twentieth).
template <int OUT, bool PAIR, bool HALF>
__device__ __forceinline__ void rows_body(const RowsArgs& a) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ RowsBarriers pb;
    __shared__ __align__(16) float bias_slab[ROWS_EPI_WARPS][64];
    uint8_t* smem = align_1024(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int TILE_ROWS = PAIR ? 2 * TC_BM : TC_BM;
    const int rank = PAIR ? (int)tc::cluster_rank() : 0;
    const uint32_t first_tile = PAIR ? blockIdx.x >> 1 : blockIdx.x, tile_step = PAIR ? gridDim.x >> 1 : gridDim.x;
    const int BN = a.BN, stages = a.stages, KB = a.kb0 + a.kb1;
    const int b_rows = PAIR ? BN / 2 : BN;  // rows of the right operand this block stages
    const uint32_t n_tiles = (uint32_t)(a.Npad / BN), total_tiles = (uint32_t)a.row_tiles * n_tiles;  // the launch has checked that it fits
    const uint32_t b_tile_bytes = (uint32_t)b_rows * 128u;
    const bool single = a.single != 0;
    const uint32_t np = single ? 1u : 2u;  // planes staged per operand
    const uint32_t stage_bytes = np * (PLANE_TILE_BYTES + b_tile_bytes);
    auto a_hi = [&](int s) { return smem + (size_t)s * stage_bytes; };
    auto a_lo = [&](int s) { return smem + (size_t)s * stage_bytes + PLANE_TILE_BYTES; };
    auto b_hi = [&](int s) { return smem + (size_t)s * stage_bytes + np * PLANE_TILE_BYTES; };
    auto b_lo = [&](int s) { return smem + (size_t)s * stage_bytes + np * PLANE_TILE_BYTES + b_tile_bytes; };

    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            tc::mbar_init(&pb.full[s], 1);
            tc::mbar_init(&pb.empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(&pb.acc_full[b], 1);
            tc::mbar_init(&pb.acc_empty[b], (PAIR ? 2 : 1) * ROWS_EPI_WARPS);  // the first block's counts the warps of both
        }
        pb.abort = 0;
        tc::fence_barrier_init();
        tc::prefetch_tensormap(&a.mapA0h);
        tc::prefetch_tensormap(&a.mapA0l);
        tc::prefetch_tensormap(&a.mapA1h);
        tc::prefetch_tensormap(&a.mapA1l);
        tc::prefetch_tensormap(&a.mapBh);
        tc::prefetch_tensormap(&a.mapBl);
    }
    if (warp == 1) {
        if constexpr (PAIR) {
            tc::tmem_alloc_pair(&pb.tmem_base, 2u * (uint32_t)a.tmem_cols);
            tc::tmem_relinquish_pair();
        } else {
            tc::tmem_alloc(&pb.tmem_base, 2u * (uint32_t)a.tmem_cols);
            tc::tmem_relinquish();
        }
    }
    tc::tc_fence_before_sync();
    __syncthreads();
    if constexpr (PAIR) tc::cluster_sync();  // both blocks' barriers and tensor memory exist before either is signalled
    tc::tc_fence_after_sync();
    wait_for_kernel_before();
    const uint32_t tmem_base = pb.tmem_base;

    if (warp == 0) {
        if (lane == 0) {
            int s = 0;
            uint32_t phase = 0;   // of the stage about to be filled: flips when the ring wraps
            int64_t filled = 0;
            bool ok = true;
            RowsWalk<TILE_ROWS> walk;
            for (uint32_t tile = first_tile; tile < total_tiles && ok; tile += tile_step) {
                int r0, n0;
                if (!walk.at(a, tile, n_tiles, &r0, &n0)) break;
                const int k = walk.k;
                const int arow = (int)(a.g.row_ws[k] + r0) + rank * TC_BM;
                const int brow = k * a.Npad + n0 + rank * b_rows;
                for (int kb = 0; kb < KB; ++kb) {
                    ok = rows_wait<PAIR>(&pb.empty[s], phase ^ 1u, &pb, a.error_word);
                    if (!ok) break;
                    const CUtensorMap* mh = kb < a.kb0 ? &a.mapA0h : &a.mapA1h;
                    const CUtensorMap* ml = kb < a.kb0 ? &a.mapA0l : &a.mapA1l;
                    const int ax = (kb < a.kb0 ? kb : kb - a.kb0) * TC_BK;
                    if constexpr (PAIR) {
                        // both blocks' bytes are counted on the first block's barrier, whose loader announces them; the
                        // other's bytes may land before that (the phase still lacks the announcing arrival)
                        if (rank == 0) tc::mbar_arrive_expect_tx(&pb.full[s], 2u * stage_bytes);
                        const uint32_t bar = tc::leader_addr(&pb.full[s]);
                        tc::tma_load_2d_pair(a_hi(s), mh, bar, ax, arow);
                        tc::tma_load_2d_pair(b_hi(s), &a.mapBh, bar, kb * TC_BK, brow);
                        if (!single) {
                            tc::tma_load_2d_pair(a_lo(s), ml, bar, ax, arow);
                            tc::tma_load_2d_pair(b_lo(s), &a.mapBl, bar, kb * TC_BK, brow);
                        }
                    } else {
                        tc::mbar_arrive_expect_tx(&pb.full[s], stage_bytes);
                        tc::tma_load_2d(a_hi(s), mh, &pb.full[s], ax, arow);
                        if (!single) tc::tma_load_2d(a_lo(s), ml, &pb.full[s], ax, arow);
                        tc::tma_load_2d(b_hi(s), &a.mapBh, &pb.full[s], kb * TC_BK, brow);
                        if (!single) tc::tma_load_2d(b_lo(s), &a.mapBl, &pb.full[s], kb * TC_BK, brow);
                    }
                    ++filled;
                    if (++s == stages) {
                        s = 0;
                        phase ^= 1u;
                    }
                }
            }
            if constexpr (PAIR) {
                // Leave no signal under way: every stage filled is waited for until it has been released (both blocks
                // get that signal) or, after a give-up, until its loads have landed (the first block, for both).
                const int64_t tail = filled < stages ? filled : stages;
                for (int64_t n = filled - tail; n < filled; ++n) {
                    const int ts = (int)(n % stages);
                    const uint32_t tp = (uint32_t)((n / stages) & 1);
                    if (!ok || !rows_wait<PAIR>(&pb.empty[ts], tp, &pb, a.error_word)) {
                        ok = false;
                        if (rank == 0)
                            for (uint32_t i = 0; i < (1u << 14) && !tc::mbar_try_wait_cluster(&pb.full[ts], tp); ++i) {}
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0 && rank == 0) {
            const uint32_t idesc = tc::idesc_bf16(TILE_ROWS, BN, false, false);
            auto mma = [&](uint32_t d, uint64_t da, uint64_t db, uint32_t acc) {
                if constexpr (PAIR) tc::mma_bf16_pair(d, da, db, idesc, acc);
                else tc::mma_bf16(d, da, db, idesc, acc);
            };
            auto commit = [&](uint64_t* bar) {
                if constexpr (PAIR) tc::mma_commit_pair(bar);
                else tc::mma_commit(bar);
            };
            int s = 0;
            uint32_t phase = 0;
            uint32_t t = 0;  // tiles started
            bool ok = true;
            // descriptors are a constant plus an address in units of 16 bytes
            const uint64_t desc = tc::smem_desc_sw128(0, 16, 1024);
            for (uint32_t tile = first_tile; tile < total_tiles && ok; tile += tile_step, ++t) {
                const int buf = (int)(t & 1);
                ok = rows_wait<PAIR>(&pb.acc_empty[buf], (t >> 1 & 1u) ^ 1u, &pb, a.error_word);
                if (!ok) break;
                tc::tc_fence_after_sync();
                const uint32_t d_tmem = tmem_base + (uint32_t)(buf * a.tmem_cols);
                for (int kb = 0; kb < KB; ++kb) {
                    ok = rows_wait<PAIR>(&pb.full[s], phase, &pb, a.error_word);
                    if (!ok) break;
                    tc::tc_fence_after_sync();
                    const uint64_t dah0 = desc + (tc::smem_u32(a_hi(s)) >> 4), dal0 = desc + (tc::smem_u32(a_lo(s)) >> 4);
                    const uint64_t dbh0 = desc + (tc::smem_u32(b_hi(s)) >> 4), dbl0 = desc + (tc::smem_u32(b_lo(s)) >> 4);
#pragma unroll
                    for (int ks = 0; ks < TC_BK / 16; ++ks) {
                        const uint64_t dah = dah0 + 2 * ks, dbh = dbh0 + 2 * ks;  // 16 bf16 = 32 bytes along K inside the swizzle row
                        if (single) {
                            mma(d_tmem, dah, dbh, (kb | ks) ? 1u : 0u);
                        } else {
                            mma(d_tmem, dal0 + 2 * ks, dbh, (kb | ks) ? 1u : 0u);
                            mma(d_tmem, dah, dbl0 + 2 * ks, 1u);
                            mma(d_tmem, dah, dbh, 1u);
                        }
                    }
                    commit(&pb.empty[s]);
                    if (++s == stages) {
                        s = 0;
                        phase ^= 1u;
                    }
                }
                if (ok) commit(&pb.acc_full[buf]);
            }
        }
    } else {
        const int q = warp & 3;           // the TMEM lane quarter this warp may read: rows 32 q .. 32 q + 31 of the tile
        uint8_t* slab_hi = smem + (size_t)stages * stage_bytes + (size_t)q * ROWS_SLAB_BYTES;  // [32 rows][64 columns] of either plane
        uint8_t* slab_lo = slab_hi + ROWS_SLAB_BYTES / 2;
        uint32_t t = 0;
        bool ok = true;
        RowsWalk<TILE_ROWS> walk;
        for (uint32_t tile = first_tile; tile < total_tiles && ok; tile += tile_step, ++t) {
            int r0, n0;
            if (!walk.at(a, tile, n_tiles, &r0, &n0)) break;
            const int k = walk.k;
            r0 += rank * TC_BM + q * 32;  // the warp's first row (of a pair's tile: in this block's half)
            const int buf = (int)(t & 1);
            const int rows_here = min(32, a.g.rows[k] - r0);  // live rows of the warp; not positive past the part's end
            const bool live = lane < rows_here;
            const int64_t orow0 = a.g.row_ws[k] + r0;
            // a chunk's bias (lane l: columns l and l + 32) and the lane's row of its gate, requested a chunk ahead
            const float* bias = a.bias_offset >= 0 ? a.params + (int64_t)a.g.part[k] * a.P + a.bias_offset : nullptr;
            const int gate_end = min((int)a.out_planes.ld, n0 + BN);
            float nb0 = 0.f, nb1 = 0.f;
            uint4 gw[8];
            auto request = [&](int c0) {
                const int n = n0 + c0;
                if (bias) {
                    nb0 = n + lane < a.N ? __ldg(bias + n + lane) : 0.f;
                    nb1 = n + 32 + lane < a.N ? __ldg(bias + n + 32 + lane) : 0.f;
                }
                if constexpr (OUT == OUT_GATED) {
                    const uint4* gp = reinterpret_cast<const uint4*>(a.gate_hi + (orow0 + lane) * a.out_planes.ld + n);
#pragma unroll
                    for (int j = 0; j < 8; ++j) gw[j] = live && n + 8 * j < gate_end ? gp[j] : make_uint4(0u, 0u, 0u, 0u);
                }
            };
            request(0);
            ok = rows_wait<PAIR>(&pb.acc_full[buf], (t >> 1 & 1u), &pb, a.error_word);
            if (!ok) break;
            tc::tc_fence_after_sync();
            const uint32_t acc = tmem_base + (uint32_t)(buf * a.tmem_cols) + ((uint32_t)(q * 32) << 16);
            // Longest chain of the products with K <= 256, and bound by what its stores can move (8 warps with half the work
            // each took as long).  Stores of 64-byte pieces by the warps, or of own rows 32 bytes at a time, were slower
            // (gated 99 and 126 us against 90); unrolled chunks did not fit the instruction cache (11 us a tile against 7).
#pragma unroll 1
            for (int c0 = 0; c0 < BN && rows_here > 0; c0 += 64) {
                const bool half = HALF && c0 + 32 >= BN;  // 32 columns or fewer are left
                uint32_t raw[2][32];
                tc::tmem_load_issue(acc + (uint32_t)c0, raw[0]);
                if (!half) tc::tmem_load_issue(acc + (uint32_t)(c0 + 32), raw[1]);
                if (bias) {
                    __syncwarp();
                    bias_slab[q][lane] = nb0;
                    bias_slab[q][32 + lane] = nb1;
                    __syncwarp();
                }
                uint32_t mask[32];  // 0xFFFF in the halves that the gate lets pass
                if constexpr (OUT == OUT_GATED) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        mask[4 * j] = positive_halves(gw[j].x);
                        mask[4 * j + 1] = positive_halves(gw[j].y);
                        mask[4 * j + 2] = positive_halves(gw[j].z);
                        mask[4 * j + 3] = positive_halves(gw[j].w);
                    }
                }
                if (c0 + 64 < BN) request(c0 + 64);
                tc::tmem_load_wait(raw[0]);
                tc::tmem_load_wait(raw[1]);
                const int nbase = n0 + c0;
                if constexpr (OUT == OUT_F32) {
                    // fp32 output (logits): every lane stores its own row
                    float* o = a.out + (orow0 + lane) * a.ld_out;
                    if (live) {
#pragma unroll
                        for (int j = 0; j < 64; j += 4) {
                            if (j >= 32 && half) break;
                            const int n = nbase + j;
                            float x[4];
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                x[e] = __uint_as_float(raw[j >> 5][(j & 31) + e]);
                                if (bias) x[e] += bias_slab[q][j + e];
                                if (a.relu) x[e] = fmaxf(x[e], 0.f);
                            }
                            if (n + 3 < a.N) {
                                *reinterpret_cast<float4*>(o + n) = make_float4(x[0], x[1], x[2], x[3]);
                            } else {
#pragma unroll
                                for (int e = 0; e < 4; ++e)
                                    if (n + e < a.N) o[n + e] = x[e];
                            }
                        }
                    }
                    __syncwarp();
                } else {
                    // Columns past the layer's width need no masking: the repacked weights are zero there and so is the
                    // bias, hence the accumulator, the sum and its ReLU are zero and the padding columns stay zero.
                    // (What lies past the accumulator's BN columns is past the planes' too and is not stored.)
                    uint32_t h[32], l[32];
#pragma unroll
                    for (int q0 = 0; q0 < 32; q0 += 16) {
                        if (q0 > 0 && half) break;
#pragma unroll
                        for (int j = q0; j < q0 + 16; j += 2) {
                            float x[4];
#pragma unroll
                            for (int e = 0; e < 4; ++e) x[e] = __uint_as_float(raw[j >> 4][2 * (j & 15) + e]);
                            if (bias) {
                                const float4 b4 = *reinterpret_cast<const float4*>(&bias_slab[q][2 * j]);
                                add_pair(x[0], x[1], b4.x, b4.y);
                                add_pair(x[2], x[3], b4.z, b4.w);
                            }
                            if (a.relu) {
#pragma unroll
                                for (int e = 0; e < 4; ++e) x[e] = fmaxf(x[e], 0.f);
                            }
                            split_pair(x[0], x[1], h[j], l[j]);
                            split_pair(x[2], x[3], h[j + 1], l[j + 1]);
                            if constexpr (OUT == OUT_GATED) {
                                h[j] &= mask[j];
                                l[j] &= mask[j];
                                h[j + 1] &= mask[j + 1];
                                l[j + 1] &= mask[j + 1];
                            }
                        }
                    }
                    // Out through shared memory, one bulk-tensor store per plane: row r's 16-byte piece j at piece j ^ (r % 8), of
                    // rows of 32 columns at piece j ^ (r / 2 % 4), as the maps' swizzles have it.
                    const uint32_t pitch = half ? 64u : 128u;
                    auto swizzle = [&](uint32_t row) { return half ? row >> 1 & 3u : row & 7u; };
                    const uint32_t own = (uint32_t)lane * pitch, swz = swizzle(lane);
                    if (lane == 0) tc::tma_store_wait_read();  // the chunk before has left the slab
                    __syncwarp();
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        if (j >= 4 && half) break;
                        const uint32_t at = own + (((uint32_t)j ^ swz) << 4);
                        *reinterpret_cast<uint4*>(slab_hi + at) = make_uint4(h[4 * j], h[4 * j + 1], h[4 * j + 2], h[4 * j + 3]);
                        *reinterpret_cast<uint4*>(slab_lo + at) = make_uint4(l[4 * j], l[4 * j + 1], l[4 * j + 2], l[4 * j + 3]);
                    }
                    if (rows_here == 32) {
                        tc::fence_proxy_async_smem();
                        __syncwarp();
                        if (lane == 0 && nbase < a.out_planes.ld) {
                            tc::tma_store_2d(half ? &a.mapOh32 : &a.mapOh, slab_hi, nbase, (int)orow0);
                            tc::tma_store_2d(half ? &a.mapOl32 : &a.mapOl, slab_lo, nbase, (int)orow0);
                            tc::tma_store_commit();
                        }
                    } else {  // the part's last rows: the rows behind them are not this part's
                        __syncwarp();
                        const int n = nbase + 8 * (lane & 7);
                        for (int row = lane >> 3; row < rows_here; row += 4) {
                            if (n < a.out_planes.ld && !(half && (lane & 7) >= 4)) {
                                const uint32_t at = (uint32_t)row * pitch + ((((uint32_t)lane & 7u) ^ swizzle(row)) << 4);
                                const int64_t o = (orow0 + row) * a.out_planes.ld + n;
                                *reinterpret_cast<uint4*>(a.out_planes.hi + o) = *reinterpret_cast<const uint4*>(slab_hi + at);
                                *reinterpret_cast<uint4*>(a.out_planes.lo + o) = *reinterpret_cast<const uint4*>(slab_lo + at);
                            }
                        }
                        __syncwarp();
                    }
                }
            }
            tc::tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) {  // every epilogue warp (of both blocks) arrives: the buffer may be overwritten
                if constexpr (PAIR) tc::mbar_arrive_cluster(tc::leader_addr(&pb.acc_empty[buf]));
                else tc::mbar_arrive(&pb.acc_empty[buf]);
            }
        }
        if (OUT != OUT_F32 && lane == 0) tc::tma_store_wait_all();
    }
    tc::tc_fence_before_sync();
    __syncthreads();
    if constexpr (PAIR) {
        tc::cluster_sync();  // neither block leaves while the other may still signal it or read its operands
        if (warp == 1) tc::tmem_dealloc_pair(tmem_base, 2u * (uint32_t)a.tmem_cols);
    } else {
        if (warp == 1) tc::tmem_dealloc(tmem_base, 2u * (uint32_t)a.tmem_cols);
    }
}

template <int OUT, bool HALF>
__global__ void __launch_bounds__(ROWS_THREADS, 1) tc_rows_kernel(const __grid_constant__ RowsArgs a) {
    rows_body<OUT, false, HALF>(a);
}
template <int OUT, bool HALF>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(ROWS_THREADS, 1) tc_rows_pair_kernel(const __grid_constant__ RowsArgs a) {
    rows_body<OUT, true, HALF>(a);
}

// ------------------------------------------------------------------------------------
// wgrad kernel
// ------------------------------------------------------------------------------------
struct WgradArgs {
    GroupDesc g;
    SplitPlan sp;
    CUtensorMap mapHh, mapHl, mapNh, mapNl, mapZh, mapZl;
    int d_in, d_out;
    int src_atoms;    // 64-wide atoms over d_in, per source
    int total_atoms;  // of all sources
    int col_atoms;    // of them a block takes (the last block of a chunk may have fewer)
    int z_tiles;      // 128-wide tiles over d_out that a block takes: 1 or 2
    int tmem_cols, stages;
    int bk;           // rows (k) per pipeline stage: 64 or 32
    int single;       // 1: operands rounded to bf16 (hi planes only)
    CUtensorMap mapP; // partial as rows of d_out values, boxes of 32 x 32; used where its rows start at multiples of 16 bytes
    float* partial;   // [slot][(nsrc d_in + 1)] rows, ld_partial apart
    int64_t ld_partial;
    int* error_word;
};

// The product is taken transposed: the gradient dZ is the operand whose columns are the accumulator's rows (one or two
// tiles of 128 of them), the sources' columns, H's and behind them N's, are the accumulator's columns, as many atoms of 64
// as the tensor memory and the stages have room for (wgrad_shape).  A few classes then cost one MMA with 256 columns where
// they cost two with 64 or 128.  The partial sums leave through shared memory, 32 x 32 of them by a bulk-tensor store, in rows
// padded to 16 bytes where the scratch holds that (stored by the threads, 16 bytes of 32 rows at a time, they took 4 us of an 18 us launch;
// stored down their columns, a line per warp, 8 us more than that: so they are where it does not, in chunks of thousands of rows).  The thread that issues the MMAs is as easily the longest chain as the loads are, with one
// plane per operand above all: its loop keeps descriptors as a constant plus an address and no division by the number of
// stages (500,000 rows, 1,024 x 512 in bf16: 658 us, with this form and divisions 975, now 574).
// us a launch before and after: the head of 47 classes on 200 k rows of 256 62 / 55, on 2 M 615 / 495, of two classes on 5 M
// 1,390 / 1,152; 512 -> 256 on 200 k rows 145 / 130, on 2 M 1,400 / 1,272; 256 -> 256 on 5 M 1,910 / 1,840 (5.6 TB/s; 1,634
// without the MMAs); 180 -> 90 on three parts of 10 k rows 18 / 13.
__global__ void __launch_bounds__(TC_THREADS, 1) tc_wgrad_kernel(const __grid_constant__ WgradArgs a) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ PipeBarriers pb;
    const int slot = blockIdx.y;
    int k = 0;
    while (k + 1 < a.g.num && a.sp.split_begin[k + 1] <= slot) ++k;
    const int chunk = slot - a.sp.split_begin[k];
    const int n_p = a.g.rows[k];
    const int v0 = min(n_p, chunk * a.sp.rows_per_split[k]);
    const int v1 = min(n_p, v0 + a.sp.rows_per_split[k]);
    const int BK = a.bk;
    const int KB = (v1 - v0 + BK - 1) / BK;
    const int d_in = a.d_in, d_out = a.d_out;
    const int first_atom = (int)blockIdx.x * a.col_atoms;             // of the sources' columns
    const int NA = min(a.col_atoms, a.total_atoms - first_atom);      // atoms of this block
    const int cbase = (int)blockIdx.z * a.z_tiles * TC_BM;            // first output column
    const int ccount = min(a.z_tiles * TC_BM, d_out - cbase);         // output columns of this block
    const int ZA = (ccount + 63) / 64, z_tiles = (ccount + TC_BM - 1) / TC_BM;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t bias_row = (int64_t)a.total_atoms / a.src_atoms * d_in;  // behind the sources' columns
    const int64_t slot_row = (int64_t)slot * (bias_row + 1);
    float* P = a.partial + slot_row * a.ld_partial + cbase;

    const bool bias_tile = blockIdx.x == 0;  // these blocks also produce the bias gradient of their columns

    if (KB == 0) {  // empty chunk: the gradient contribution is zero
        wait_for_kernel_before();
        for (int idx = threadIdx.x; idx < 64 * NA * ccount; idx += TC_THREADS) {
            const int at = first_atom + idx / ccount / 64, j = at % a.src_atoms * 64 + idx / ccount % 64;
            if (j < d_in) P[((int64_t)(at / a.src_atoms) * d_in + j) * a.ld_partial + idx % ccount] = 0.f;
        }
        if (bias_tile)
            for (int c = threadIdx.x; c < ccount; c += TC_THREADS) P[bias_row * a.ld_partial + c] = 0.f;
        return;
    }

    uint8_t* smem = align_1024(smem_raw);
    const int stages = a.stages;
    const uint32_t ATOM_BYTES = (uint32_t)BK * 128u;  // one 64-wide column of BK k-rows
    const bool single = a.single != 0;
    const uint32_t np = single ? 1u : 2u;  // planes staged per operand
    const uint32_t z_bytes = (uint32_t)ZA * ATOM_BYTES, s_bytes = (uint32_t)NA * ATOM_BYTES;
    const uint32_t stage_bytes = np * (z_bytes + s_bytes);  // no more than the launch counted on
    // A stage: dZ, then the sources, hi before lo.  Where the last tile of dZ has one atom, the MMA reads whatever lies behind it
    // as the other: that only reaches accumulator rows that are not stored.
    auto z_hi = [&](int s) { return smem + (size_t)s * stage_bytes; };
    auto z_lo = [&](int s) { return smem + (size_t)s * stage_bytes + z_bytes; };
    auto s_hi = [&](int s) { return smem + (size_t)s * stage_bytes + np * z_bytes; };
    auto s_lo = [&](int s) { return smem + (size_t)s * stage_bytes + np * z_bytes + s_bytes; };

    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            tc::mbar_init(&pb.full[s], 1);
            tc::mbar_init(&pb.empty[s], bias_tile ? 1 + 128 : 1);  // MMA commit (+ the column-sum readers)
        }
        tc::mbar_init(&pb.accum, 1);
        pb.abort = 0;
        tc::fence_barrier_init();
        tc::prefetch_tensormap(&a.mapHh);
        tc::prefetch_tensormap(&a.mapNh);
        tc::prefetch_tensormap(&a.mapZh);
        tc::prefetch_tensormap(&a.mapZl);
    }
    if (warp == 1) {
        tc::tmem_alloc(&pb.tmem_base, (uint32_t)a.tmem_cols);
        tc::tmem_relinquish();
    }
    tc::tc_fence_before_sync();
    __syncthreads();
    tc::tc_fence_after_sync();
    wait_for_kernel_before();
    const uint32_t tmem_base = pb.tmem_base;
    const uint32_t acc_cols = 64u * (uint32_t)NA;  // accumulator columns of one tile of dZ

    if (warp == 0) {
        if (lane == 0) {
            const int row = (int)(a.g.row_ws[k] + v0);
            tc::RingAt at;
            for (int kb = 0; kb < KB; ++kb, at.advance(stages)) {
                const int s = at.s;
                if (!wait_or_abort(&pb.empty[s], at.phase ^ 1u, &pb, a.error_word)) break;
                tc::mbar_arrive_expect_tx(&pb.full[s], stage_bytes);
                for (int t = 0; t < ZA; ++t) {
                    tc::tma_load_2d(z_hi(s) + t * ATOM_BYTES, &a.mapZh, &pb.full[s], cbase + 64 * t, row + kb * BK);
                    if (!single) tc::tma_load_2d(z_lo(s) + t * ATOM_BYTES, &a.mapZl, &pb.full[s], cbase + 64 * t, row + kb * BK);
                }
                for (int t = 0; t < NA; ++t) {
                    const bool second = first_atom + t >= a.src_atoms;
                    const int x = 64 * (first_atom + t - (second ? a.src_atoms : 0));
                    tc::tma_load_2d(s_hi(s) + t * ATOM_BYTES, second ? &a.mapNh : &a.mapHh, &pb.full[s], x, row + kb * BK);
                    if (!single) tc::tma_load_2d(s_lo(s) + t * ATOM_BYTES, second ? &a.mapNl : &a.mapHl, &pb.full[s], x, row + kb * BK);
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // up to 256 columns per MMA.  One thread feeds the tensor core: descriptors are a constant plus an address.
            const uint32_t idesc0 = tc::idesc_bf16(TC_BM, 64 * min(NA, 4), true, true), idesc1 = tc::idesc_bf16(TC_BM, 64 * max(NA - 4, 1), true, true);
            const uint64_t desc = tc::smem_desc_sw128(0, ATOM_BYTES, 1024);
            const uint32_t atom = ATOM_BYTES >> 4;  // addresses of descriptors are in units of 16 bytes
            // the products of one 128-wide tile of dZ with one group of the sources' atoms
            auto product = [&](uint32_t d_tmem, uint32_t zh, uint32_t zl, uint32_t sh, uint32_t sl, uint32_t idesc, uint32_t accumulate) {
                if (single) {
                    tc::mma_bf16(d_tmem, desc + zh, desc + sh, idesc, accumulate);
                } else {
                    tc::mma_bf16(d_tmem, desc + zh, desc + sl, idesc, accumulate);
                    tc::mma_bf16(d_tmem, desc + zl, desc + sh, idesc, 1u);
                    tc::mma_bf16(d_tmem, desc + zh, desc + sh, idesc, 1u);
                }
            };
            tc::RingAt at;
            for (int kb = 0; kb < KB; ++kb, at.advance(stages)) {
                const int s = at.s;
                if (!wait_or_abort(&pb.full[s], at.phase, &pb, a.error_word)) break;
                tc::tc_fence_after_sync();
                uint32_t zh = tc::smem_u32(z_hi(s)) >> 4, zl = tc::smem_u32(z_lo(s)) >> 4, sh = tc::smem_u32(s_hi(s)) >> 4, sl = tc::smem_u32(s_lo(s)) >> 4;
#pragma unroll 2
                for (int ks = 0; ks < BK / 16; ++ks) {
                    const uint32_t accumulate = (kb | ks) ? 1u : 0u;
                    product(tmem_base, zh, zl, sh, sl, idesc0, accumulate);
                    if (z_tiles > 1) product(tmem_base + acc_cols, zh + 2 * atom, zl + 2 * atom, sh, sl, idesc0, accumulate);
                    else if (NA > 4) product(tmem_base + 256u, zh, zl, sh + 4 * atom, sl + 4 * atom, idesc1, accumulate);
                    zh += 128; zl += 128; sh += 128; sl += 128;  // 16 k-rows of 128 bytes
                }
                tc::mma_commit(&pb.empty[s]);
            }
            tc::mma_commit(&pb.accum);
        }
    } else {
        const int tw = threadIdx.x - 64;  // 0..127
        // Bias gradient = column sums of dZ.  While the MMAs run, the epilogue warps of the bias
        // blocks add up the dZ tiles sitting in shared memory.  In an atom a 16-byte chunk id
        // is (k-row r = id / 8, stored chunk s = id % 8) and holds logical chunk s ^ (r % 8).
        // Thread tw takes ids tw, tw + 128, ...: rows tw / 8 + 16 i, which agree
        // mod 8, so it always sums the same 8 columns of every atom.
        float colsum[4][8];
#pragma unroll
        for (int t = 0; t < 4; ++t)
#pragma unroll
            for (int e = 0; e < 8; ++e) colsum[t][e] = 0.f;
        bool ok = true;
        if (bias_tile) {
            tc::RingAt at;
            for (int kb = 0; kb < KB && ok; ++kb, at.advance(stages)) {
                const int s = at.s;
                ok = wait_or_abort(&pb.full[s], at.phase, &pb, a.error_word);
                if (!ok) break;
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    if (t < ZA) {
                        const uint4* bh = reinterpret_cast<const uint4*>(z_hi(s) + t * ATOM_BYTES);
                        const uint4* bl = reinterpret_cast<const uint4*>(z_lo(s) + t * ATOM_BYTES);
                        for (int i = 0; i < BK / 16; ++i) {
                            Pack8 p;
                            p.zero();
                            p.add_planes(bh[tw + 128 * i], single ? make_uint4(0u, 0u, 0u, 0u) : bl[tw + 128 * i]);
#pragma unroll
                            for (int e = 0; e < 8; ++e) colsum[t][e] += p.v[e];
                        }
                    }
                }
                tc::mbar_arrive(&pb.empty[s]);
            }
        }
        if (ok) ok = wait_or_abort(&pb.accum, 0, &pb, a.error_word);
        asm volatile("bar.sync 1, 128;" ::: "memory");  // the four epilogue warps agree on the outcome
        ok = *reinterpret_cast<volatile int*>(&pb.abort) == 0;
        tc::tc_fence_after_sync();
        if (ok && bias_tile) {
            // every load has landed and every MMA has finished: the ring is free to hold the sums
            float* red = reinterpret_cast<float*>(smem);  // [128 threads][32]
#pragma unroll
            for (int t = 0; t < 4; ++t)
#pragma unroll
                for (int e = 0; e < 8; ++e) red[tw * 32 + t * 8 + e] = colsum[t][e];
            asm volatile("bar.sync 1, 128;" ::: "memory");
            for (int c = tw; c < ccount; c += 128) {
                const int t = c >> 6, lc = (c & 63) >> 3, e = c & 7;
                float sum = 0.f;
                for (int h = 0; h < 16; ++h) sum += red[(h * 8 + (lc ^ (h & 7))) * 32 + t * 8 + e];  // fixed order
                P[bias_row * a.ld_partial + c] = sum;
            }
        }
        if (ok) {
            // A lane holds output column c of 32 source columns j: through a 32 x 32 slab (row j, 16-byte piece c / 4 at piece
            // c / 4 ^ j % 8, as the map's swizzle has it; the ring is free, behind the column sums' 16 KB) and out as a box.
            const int q = warp & 3;
            const bool boxes = a.ld_partial % 4 == 0;
            uint8_t* slab[2] = {smem + 16384 + q * 8192, smem + 16384 + q * 8192 + 4096};
            int n_out = 0;
            for (int t = 0; t < z_tiles; ++t) {
                const int c0 = t * TC_BM + q * 32;                 // the warp's first output column
                if (c0 >= ccount) break;
                const uint32_t acc = tmem_base + (uint32_t)t * acc_cols + ((uint32_t)(q * 32) << 16);
#pragma unroll 1
                for (int n = 0; n < 2 * NA; ++n) {
                    const bool second = first_atom + n / 2 >= a.src_atoms;
                    const int j0 = 64 * (first_atom + n / 2 - (second ? a.src_atoms : 0)) + 32 * (n & 1);  // first source column of the 32
                    if (j0 >= d_in) continue;
                    uint32_t raw[32];
                    tc::tmem_load_issue(acc + 32u * (uint32_t)n, raw);
                    tc::tmem_load_wait(raw);
                    const int64_t row = slot_row + (second ? d_in : 0) + j0;
                    if (boxes && j0 + 32 <= d_in) {
                        uint8_t* out = slab[n_out++ & 1];
                        if (lane == 0) tc::tma_store_wait_read_but_one();  // the box before the last has left the slab
                        __syncwarp();
#pragma unroll
                        for (int e = 0; e < 32; ++e)
                            *reinterpret_cast<uint32_t*>(out + e * 128 + (((lane >> 2) ^ (e & 7)) << 4) + (lane & 3) * 4) = raw[e];
                        tc::fence_proxy_async_smem();
                        __syncwarp();
                        if (lane == 0) {
                            tc::tma_store_2d(&a.mapP, out, cbase + c0, (int)row);
                            tc::tma_store_commit();
                        }
                    } else if (c0 + lane < ccount) {  // the source's last columns (the rows behind them are not its), or rows at any address
                        float* o = a.partial + row * a.ld_partial + cbase + c0 + lane;
#pragma unroll
                        for (int e = 0; e < 32; ++e)
                            if (j0 + e < d_in) o[(int64_t)e * a.ld_partial] = __uint_as_float(raw[e]);
                    }
                    __syncwarp();
                }
            }
            if (lane == 0) tc::tma_store_wait_all();
        }
    }
    tc::tc_fence_before_sync();
    __syncthreads();
    if (warp == 1) tc::tmem_dealloc(tmem_base, (uint32_t)a.tmem_cols);
}

// ------------------------------------------------------------------------------------
// self-test of the bounded wait: a barrier nothing ever arrives at
// ------------------------------------------------------------------------------------
__global__ void wait_selftest_kernel(int* error_word, int polls) {
    wait_for_kernel_before();
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        tc::mbar_init(&bar, 1);
        tc::fence_barrier_init();
        bool done = false;
        for (int i = 0; i < polls && !done; ++i) done = tc::mbar_try_wait(&bar, 0);
        if (!done) atomicExch(error_word, 2);  // gave up, as the pipeline kernels do
    }
}

}  // namespace

extern "C" int32_t rtma_selftest_wait_timeout(rtma_ctx* ctx, void* stream) {
    if (!ctx) return RTMA_ERR_INVALID_ARG;
    RTMA_CUDA(ctx, cudaSetDevice(ctx->device));
    launch_kernel(wait_selftest_kernel, 1, 32, 0, static_cast<cudaStream_t>(stream), ctx->error_word, 1 << 10);
    RTMA_LAUNCH_CHECK(ctx);
    return RTMA_OK;
}

namespace {

// ------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled() {
    static EncodeTiledFn fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
        cudaGetLastError();
    }
    return fn;
}

uint32_t tmem_columns_for(int n) {
    uint32_t c = 32;
    while ((int)c < n) c <<= 1;
    return c;
}

int stages_for(size_t stage_bytes, int kblocks) {
    int s = (int)(SMEM_BUDGET / stage_bytes);
    if (s > MAX_STAGES) s = MAX_STAGES;
    if (s > kblocks) s = kblocks < 1 ? 1 : kblocks;
    return s;
}

int32_t set_smem_limit(rtma_ctx* ctx, const void* kernel) {
    RTMA_CUDA(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BUDGET + 2048));
    return RTMA_OK;
}

bool plane_maps(CUtensorMap* hi, CUtensorMap* lo, Planes p, uint64_t rows, uint64_t cols, uint32_t box_cols,
                uint32_t box_rows) {
    return make_tensor_map_bf16(hi, p.hi, rows, cols, p.ld, box_cols, box_rows) &&
           make_tensor_map_bf16(lo, p.lo, rows, cols, p.ld, box_cols, box_rows);
}

}  // namespace

bool make_tensor_map_bf16(CUtensorMap* out, const void* base, uint64_t rows, uint64_t cols, uint64_t ld,
                          uint32_t box_cols, uint32_t box_rows) {
    EncodeTiledFn fn = encode_tiled();
    if (!fn || rows == 0 || cols == 0) return false;
    const cuuint64_t gdim[2] = {cols, rows};
    const cuuint64_t gstride[1] = {ld * sizeof(__nv_bfloat16)};
    const cuuint32_t box[2] = {box_cols, box_rows};
    const cuuint32_t estride[2] = {1, 1};
    return fn(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), gdim, gstride, box, estride,
              CU_TENSOR_MAP_INTERLEAVE_NONE, box_cols <= 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// fp32 rows in boxes of 32 x 32, 128-byte swizzle
static bool make_tensor_map_f32(CUtensorMap* out, const float* base, uint64_t rows, uint64_t cols, uint64_t ld) {
    EncodeTiledFn fn = encode_tiled();
    if (!fn || rows == 0 || cols == 0) return false;
    const cuuint64_t gdim[2] = {cols, rows};
    const cuuint64_t gstride[1] = {ld * sizeof(float)};
    const cuuint32_t box[2] = {32, 32};
    const cuuint32_t estride[2] = {1, 1};
    return fn(out, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(base), gdim, gstride, box, estride, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Column tile of the rows kernel for `d` columns: at most 256 wide, equal tiles, a multiple of 16; from 64 columns on a
// multiple of 32, the step of an MMA of a pair of blocks.  Not coarser: with tiles in multiples of 64, what the epilogue stores
// at a time, 300 columns paid for 384 instead of 320 (a step of 200 k rows, 128 -> 300 -> 300: forward 395 / 386 us, input
// gradients 352 / 334; one plane 244 / 231 and 256 / 250); in multiples of 16 it gains nothing.
static int column_tile(int d) {
    const int tiles = (int)ceil_div(d, 256), step = d >= 64 ? 32 : 16;
    return (int)ceil_div(ceil_div(d, tiles), step) * step;
}

TcLayerPlan tc_plan_layer(LayerShape ls) {
    TcLayerPlan p{};
    p.Kf = ls.nsrc * TC_BK * (int)ceil_div(ls.d_in, TC_BK);
    p.BN_f = column_tile(ls.d_out);
    p.Npad_f = p.BN_f * (int)ceil_div(ls.d_out, 256);
    p.Kd = ls.nsrc * TC_BK * (int)ceil_div(ls.d_out, TC_BK);
    p.BN_d = column_tile(ls.d_in);
    p.Npad_d = p.BN_d * (int)ceil_div(ls.d_in, 256);
    return p;
}

TcLayerPlan tc_plan_head(LayerShape ls, int head_cp) {
    TcLayerPlan p = tc_plan_layer(ls);  // the dgrad operand is the usual one
    p.Kf = TC_BK * (int)ceil_div(ls.d_in, TC_BK);
    p.BN_f = p.Npad_f = column_tile(ls.nsrc * head_cp);  // at most 128 columns
    return p;
}

size_t tc_prep_elems(const TcLayerPlan& p, bool with_dgrad) {
    return 2 * ((size_t)p.Npad_f * p.Kf + (with_dgrad ? (size_t)p.Npad_d * p.Kd : 0));
}

bool tc_available() { return encode_tiled() != nullptr; }

int32_t launch_tc_weight_prep(rtma_ctx* ctx, const GroupDesc& g, const TcPrepJob* jobs, int njobs, const float* params,
                              cudaStream_t s) {
    if (g.num == 0 || njobs == 0) return RTMA_OK;
    if (njobs > PREP_MAX_JOBS) return rtma_fail(ctx, RTMA_ERR_INVALID_ARG, "internal: %d weight repack jobs", njobs);
    PrepBatch b{};
    int most = 0;
    for (int j = 0; j < njobs; ++j) {
        const TcLayerPlan& p = jobs[j].plan;
        b.job[j] = PrepArgs{jobs[j].ls, jobs[j].head_cp, p.Npad_f, p.Kf, p.Npad_d, p.Kd, jobs[j].Bf_hi, jobs[j].Bf_lo, jobs[j].Bd_hi, jobs[j].Bd_lo};
        most = std::max(most, prep_tiles(p.Npad_f, p.Kf) + (jobs[j].Bd_hi ? prep_tiles(p.Npad_d, p.Kd) : 0));
    }
    dim3 grid((unsigned)most, (unsigned)g.num, (unsigned)njobs);
    { KernelScope ks(ctx, KC_WEIGHT_PREP, s); launch_kernel(tc_weight_prep_kernel, grid, 256, 0, s, g, b, params); }
    RTMA_LAUNCH_CHECK(ctx);
    return RTMA_OK;
}

// Do a product's tiles go to pairs of blocks (256 rows, each block staging half of the weight tile)?  A block by itself
// moves 96 KB through shared memory per 64 of K, two planes and 128 x 256 outputs, a third of it activations, next to what
// the MMAs read there; a pair 64 KB each.  That pays where this main loop is the longest chain, hence from a depth K times
// planes on.  Where the output is the longer chain the pair's blocks only wait for each other.  us alone / in pairs:
//   two planes, 200 k rows: K = 512, 256 columns 145 / 115, gated 150 / 127; all products of a step with K = 384, 160 columns
//   205 / 194, gated 162 / 155; but K = 256 84 / 90, gated 90 / 95;
//   one plane (operands rounded to bf16): K = 512, 256 columns and the layers around it 167 / 179, gated 185 / 192; K = 768, 384
//   columns 273 / 264; K = 1024, 512 columns 359 / 335.  Gated it starts to pay later, the gate words are read with one plane
//   as with two: K = 768 294 / 306, K = 896 367 / 380, K = 1024 394 / 390.
// And only where a launch has tiles for every SM: 10 k rows a part, 3 parts 12.5 / 13.2.
static bool rows_use_pairs(const rtma_ctx* ctx, const GroupDesc& g, int K, int BN, bool single, bool gated) {
    const int deep = single ? (gated ? 1024 : 768) : 384;
    return BN % 32 == 0 && BN >= 128 && K >= deep && group_tiles(g, TC_BM) >= ctx->sm_count;
}

using RowsKernel = void (*)(RowsArgs);
static const RowsKernel rows_kernels[2][2][3] = {  // [pairs][last 64 columns of a tile are 32 at most][output]
    {{tc_rows_kernel<OUT_F32, false>, tc_rows_kernel<OUT_PLANES, false>, tc_rows_kernel<OUT_GATED, false>},
     {tc_rows_kernel<OUT_F32, true>, tc_rows_kernel<OUT_PLANES, true>, tc_rows_kernel<OUT_GATED, true>}},
    {{tc_rows_pair_kernel<OUT_F32, false>, tc_rows_pair_kernel<OUT_PLANES, false>, tc_rows_pair_kernel<OUT_GATED, false>},
     {tc_rows_pair_kernel<OUT_F32, true>, tc_rows_pair_kernel<OUT_PLANES, true>, tc_rows_pair_kernel<OUT_GATED, true>}}};

static int32_t launch_rows(rtma_ctx* ctx, RowsArgs& a, int64_t rows_total, bool pairs, int kclass, cudaStream_t s) {
    if (!ctx->rows_configured) {  // per device: the context is bound to one
        for (const auto& by_width : rows_kernels)
            for (const auto& by_output : by_width)
                for (const RowsKernel kernel : by_output)
                    RTMA_CUDA(ctx, cudaFuncSetAttribute(reinterpret_cast<const void*>(kernel), cudaFuncAttributeMaxDynamicSharedMemorySize, ROWS_SMEM_MAX));
        ctx->rows_configured = true;
    }
    const size_t stage_bytes = (a.single ? 1 : 2) * ((size_t)PLANE_TILE_BYTES + (size_t)(pairs ? a.BN / 2 : a.BN) * 128);
    a.stages = std::max(1, std::min<int>(ROWS_MAX_STAGES, (int)(ROWS_RING_BUDGET / stage_bytes)));
    a.tmem_cols = (int)tmem_columns_for(a.BN);
    a.error_word = ctx->error_word;
    a.row_tiles = group_tiles(a.g, pairs ? 2 * TC_BM : TC_BM);
    if (a.row_tiles == 0) return RTMA_OK;
    const int64_t total_tiles = a.row_tiles * (a.Npad / a.BN);
    if (total_tiles >= (int64_t(1) << 31)) return rtma_fail(ctx, RTMA_ERR_OVERFLOW, "too many tiles");
    const unsigned grid = pairs ? 2u * (unsigned)std::min<int64_t>(total_tiles, ctx->sm_count / 2)
                                : (unsigned)std::min<int64_t>(total_tiles, ctx->sm_count);
    const bool half = a.BN % 64 != 0 && a.BN % 64 <= 32;
    if (a.out_planes.hi && (!plane_maps(&a.mapOh, &a.mapOl, a.out_planes, rows_total, (uint64_t)a.out_planes.ld, 64, 32) ||
                            (half && !plane_maps(&a.mapOh32, &a.mapOl32, a.out_planes, rows_total, (uint64_t)a.out_planes.ld, 32, 32))))
        return rtma_fail(ctx, RTMA_ERR_CUDA, "cuTensorMapEncodeTiled refused the output planes");
    // the epilogue's slabs are only allocated for plane output: shared memory comes out of L1
    const size_t ring = a.stages * stage_bytes + 1024;
    const size_t smem = a.out_planes.hi ? ring + ROWS_EPI_WARPS * ROWS_SLAB_BYTES : ring;
    {
        KernelScope ks(ctx, kclass, s);
        const int out = !a.out_planes.hi ? OUT_F32 : a.gate_hi ? OUT_GATED : OUT_PLANES;
        launch_kernel(rows_kernels[pairs ? 1 : 0][half ? 1 : 0][out], grid, ROWS_THREADS, smem, s, a);
    }
    RTMA_LAUNCH_CHECK(ctx);
    return RTMA_OK;
}

int32_t launch_tc_forward(rtma_ctx* ctx, const GroupDesc& g, LayerShape ls, const TcLayerPlan& p, int64_t rows_total,
                          const float* params, Planes H, Planes N, const __nv_bfloat16* Bf_hi,
                          const __nv_bfloat16* Bf_lo, Planes out_planes, Mat out_f32, bool relu, bool single,
                          cudaStream_t s) {
    RowsArgs a{};
    a.g = g;
    a.single = single ? 1 : 0;
    const bool pairs = rows_use_pairs(ctx, g, p.Kf, p.BN_f, single, false);
    const uint32_t b_rows = (uint32_t)(pairs ? p.BN_f / 2 : p.BN_f);
    if (!plane_maps(&a.mapA0h, &a.mapA0l, H, rows_total, ls.d_in, TC_BK, TC_BM) ||
        !plane_maps(&a.mapA1h, &a.mapA1l, N, rows_total, ls.d_in, TC_BK, TC_BM) ||
        !make_tensor_map_bf16(&a.mapBh, Bf_hi, (uint64_t)g.num * p.Npad_f, p.Kf, p.Kf, TC_BK, b_rows) ||
        !make_tensor_map_bf16(&a.mapBl, Bf_lo, (uint64_t)g.num * p.Npad_f, p.Kf, p.Kf, TC_BK, b_rows))
        return rtma_fail(ctx, RTMA_ERR_CUDA, "cuTensorMapEncodeTiled refused the forward operands");
    if (ls.nsrc == 2) {
        a.kb0 = a.kb1 = p.Kf / (2 * TC_BK);
    } else {  // one weight matrix: the aggregate is the only operand
        a.mapA0h = a.mapA1h;
        a.mapA0l = a.mapA1l;
        a.kb0 = p.Kf / TC_BK;
        a.kb1 = 0;
    }
    a.BN = p.BN_f;
    a.Npad = p.Npad_f;
    a.N = ls.d_out;
    a.out_planes = out_planes;
    a.out = out_f32.ptr;
    a.ld_out = out_f32.ld;
    a.params = params;
    a.P = ls.P;
    a.bias_offset = ls.has_bias ? ls.param_offset + (int64_t)ls.nsrc * ls.d_in * ls.d_out : -1;
    a.relu = relu ? 1 : 0;
    a.gate_hi = nullptr;
    return launch_rows(ctx, a, rows_total, pairs, KC_GEMM_FWD, s);
}

int32_t launch_tc_dgrad(rtma_ctx* ctx, const GroupDesc& g, LayerShape ls, const TcLayerPlan& p, int64_t rows_total,
                        Planes dZ, Planes Q, const __nv_bfloat16* Bd_hi, const __nv_bfloat16* Bd_lo, Planes H, bool gate,
                        bool single, cudaStream_t s) {
    RowsArgs a{};
    a.g = g;
    a.single = single ? 1 : 0;
    const bool pairs = rows_use_pairs(ctx, g, p.Kd, p.BN_d, single, gate);
    const uint32_t b_rows = (uint32_t)(pairs ? p.BN_d / 2 : p.BN_d);
    if (!plane_maps(&a.mapA0h, &a.mapA0l, dZ, rows_total, ls.d_out, TC_BK, TC_BM) ||
        !plane_maps(&a.mapA1h, &a.mapA1l, Q, rows_total, ls.d_out, TC_BK, TC_BM) ||
        !make_tensor_map_bf16(&a.mapBh, Bd_hi, (uint64_t)g.num * p.Npad_d, p.Kd, p.Kd, TC_BK, b_rows) ||
        !make_tensor_map_bf16(&a.mapBl, Bd_lo, (uint64_t)g.num * p.Npad_d, p.Kd, p.Kd, TC_BK, b_rows))
        return rtma_fail(ctx, RTMA_ERR_CUDA, "cuTensorMapEncodeTiled refused the dgrad operands");
    if (ls.nsrc == 2) {
        a.kb0 = a.kb1 = p.Kd / (2 * TC_BK);
    } else {
        a.mapA0h = a.mapA1h;
        a.mapA0l = a.mapA1l;
        a.kb0 = p.Kd / TC_BK;
        a.kb1 = 0;
    }
    a.BN = p.BN_d;
    a.Npad = p.Npad_d;
    a.N = ls.d_in;
    a.out_planes = H;  // every tile reads the gate of exactly the block it then overwrites
    a.out = nullptr;
    a.ld_out = 0;
    a.params = nullptr;
    a.P = 0;
    a.bias_offset = -1;
    a.relu = 0;
    a.gate_hi = gate ? H.hi : nullptr;
    return launch_rows(ctx, a, rows_total, pairs, KC_GEMM_DGRAD, s);
}

// How a chunk of a layer's weight gradient is cut into blocks.  Two tiles of dZ leave tensor memory for four atoms of the sources,
// one for eight; and three stages of 32 rows are to fit (16 atoms of one plane, 8 of two).
struct WgradShape {
    int z_tiles, z_atoms;        // of dZ, per block
    int col_atoms, total_atoms;  // of the sources: per block, of all
    int blocks_x, blocks_z;
};
static WgradShape wgrad_shape(const LayerShape& ls, bool single) {
    WgradShape w;
    const int all_z = (int)ceil_div(ls.d_out, 64);
    w.z_tiles = all_z > 2 ? 2 : 1;
    w.z_atoms = std::min(all_z, 2 * w.z_tiles);
    w.total_atoms = ls.nsrc * (int)ceil_div(ls.d_in, 64);
    const int most = std::min(8 / w.z_tiles, (single ? 16 : 8) - w.z_atoms);
    w.blocks_x = (int)ceil_div(w.total_atoms, most);
    w.col_atoms = (int)ceil_div(w.total_atoms, w.blocks_x);
    w.blocks_z = (int)ceil_div(all_z, 2 * w.z_tiles);
    return w;
}

WgradCost tc_wgrad_cost(const LayerShape& ls, bool single) {
    const WgradShape w = wgrad_shape(ls, single);
    WgradCost c;
    c.blocks_per_slot = (int64_t)w.blocks_x * w.blocks_z;
    c.plain_blocks_per_slot = ceil_div(ls.nsrc * ceil_div(ls.d_in, 128), 2) * ceil_div(ls.d_out, 256);
    c.bytes_per_row = (single ? 1 : 2) * 128 * (w.z_atoms + w.col_atoms);
    c.params = (int64_t)(ls.nsrc * ls.d_in + 1) * ls.d_out;
    return c;
}

int32_t launch_tc_wgrad(rtma_ctx* ctx, const GroupDesc& g, const SplitPlan& sp, LayerShape ls, int64_t rows_total,
                        Planes H, Planes N, Planes dZ, float* partial, int64_t ld_partial, bool single, cudaStream_t s) {
    if (!ctx->wgrad_configured) {
        RTMA_TRY(set_smem_limit(ctx, reinterpret_cast<const void*>(tc_wgrad_kernel)));
        ctx->wgrad_configured = true;
    }
    const int slots = sp.split_begin[g.num];
    if (slots == 0) return RTMA_OK;
    if (slots > 65535) return rtma_fail(ctx, RTMA_ERR_UNSUPPORTED, "too many weight-gradient chunks (%d)", slots);
    const WgradShape w = wgrad_shape(ls, single);
    WgradArgs a{};
    a.g = g;
    a.sp = sp;
    a.d_in = ls.d_in;
    a.d_out = ls.d_out;
    a.src_atoms = w.total_atoms / ls.nsrc;
    a.total_atoms = w.total_atoms;
    a.col_atoms = w.col_atoms;
    a.z_tiles = w.z_tiles;
    a.tmem_cols = (int)tmem_columns_for(w.z_tiles * 64 * w.col_atoms);
    a.single = single ? 1 : 0;
    // 32-row stages where 64-row ones would leave fewer than three of them
    const size_t stage64 = (single ? 1 : 2) * (size_t)(w.z_atoms + w.col_atoms) * 64 * 128;
    a.bk = SMEM_BUDGET / stage64 >= 3 ? 64 : 32;
    const size_t stage_bytes = stage64 * a.bk / 64;
    a.stages = stages_for(stage_bytes, MAX_STAGES);
    a.partial = partial;
    a.ld_partial = ld_partial;
    if (ld_partial % 4 == 0 && !make_tensor_map_f32(&a.mapP, partial, (uint64_t)slots * (ls.nsrc * ls.d_in + 1), ls.d_out, a.ld_partial))
        return rtma_fail(ctx, RTMA_ERR_CUDA, "cuTensorMapEncodeTiled refused the partial sums");
    a.error_word = ctx->error_word;
    // boxes of 64 columns x BK rows: one atom of a stage
    if (!plane_maps(&a.mapHh, &a.mapHl, H, rows_total, ls.d_in, 64, (uint32_t)a.bk) ||
        !plane_maps(&a.mapNh, &a.mapNl, N, rows_total, ls.d_in, 64, (uint32_t)a.bk) ||
        !plane_maps(&a.mapZh, &a.mapZl, dZ, rows_total, ls.d_out, 64, (uint32_t)a.bk))
        return rtma_fail(ctx, RTMA_ERR_CUDA, "cuTensorMapEncodeTiled refused the wgrad operands");
    if (ls.nsrc == 1) {  // the aggregate is the only source
        a.mapHh = a.mapNh;
        a.mapHl = a.mapNl;
    }
    const dim3 grid((unsigned)w.blocks_x, (unsigned)slots, (unsigned)w.blocks_z);
    { KernelScope ks(ctx, KC_GEMM_WGRAD, s); launch_kernel(tc_wgrad_kernel, grid, TC_THREADS, a.stages * stage_bytes + 1024, s, a); }
    RTMA_LAUNCH_CHECK(ctx);
    return RTMA_OK;
}
