// Mean aggregation (the row-normalised adjacency Abar of Theorem 2, and its transpose) on the tensor
// cores, for parts whose rows are stored so that most neighbours of a row are rows nearby (the nodes
// of a super-node kept together, Sec. 3.2).
//
// For a tile of 128 consecutive rows of a part, the entries whose column lies in the window of
// DENSE_WINDOW rows around the tile form a small dense matrix A [128 x DENSE_WINDOW]: its entry
// (v, u) is 1 where u occurs in row v (forward; the result is scaled by 1/deg v afterwards) or
// 1/deg u there (transposed pass).  Once per call every row's window is recorded as a bit mask
// (dense_lists_kernel); per launch the kernel expands the masks into A in shared memory, in the layout
// the tensor core reads, 64 window rows at a time, and multiplies A with the window's source rows, which
// bulk-tensor loads bring in straight from the split planes:
//     out[tile] = A * src[window]       accumulated in fp32 in tensor memory.
// Ones are exact in bf16, so the forward pass is two MMAs per step (A * hi + A * lo) and sums exactly
// the values the gather kernel sums; the transposed pass carries its weights as a split pair and takes
// three (A_hi * hi + A_lo * hi + A_hi * lo).  The few entries outside the window are listed by the same
// once-per-call kernel (up to DT_LCAP per row; a row with more is marked and its entries are looked up
// again).  Per launch spmm_outside_kernel first writes their sum to the output row, and the epilogue of
// the tile adds the tile's product to it before it writes the row.  Which parts go this way is decided per part
// (dense_decide_kernel, from a sample of the part's rows; a part in which some row repeats an entry inside
// its window is taken back, a bit cannot count), so that the arithmetic a part sees does not depend on
// which other parts share its launch.
//
// Warps: 0 = MMA issuer and owner of the tensor memory (one lane), 1..4 = builders of A (a thread per tile
// row; the first of them also issues the stage's bulk-tensor loads, which wait for the same barrier),
// 5..12 = epilogue.  Two accumulators let the epilogue of one tile run
// beside the main loop of the next.  Every wait is bounded; one that runs out raises the context's
// device error word and the block winds down.
#include <algorithm>

#include "tc_common.cuh"
#include "train.cuh"

RTMA_BOUNDS_TU()

namespace {

constexpr int DT_THREADS = 416;
constexpr int DT_BUILDERS = 128;
constexpr int DT_EPI_THREADS = 256;
constexpr int DT_BM = DENSE_TILE_ROWS;           // rows of a tile
constexpr int DT_BK = 64;                        // window rows per pipeline stage
constexpr int DT_HALO = DENSE_HALO;              // window rows before the tile, and after it
constexpr int DT_KB = DENSE_WINDOW / DT_BK;
static_assert(DT_KB <= 8 && GROUP_ROW_ALIGN % 32 == 0, "a byte holds the blocks of a window, 32 rows lie in one part");
constexpr int DT_A_BYTES = DT_BM * 128;          // one plane of A for one stage: 16 KB
constexpr int DT_ATOM_BYTES = DT_BK * 128;       // 64 source rows x 64 columns of one plane: 8 KB
constexpr int DT_STAGING_BYTES = 4096;           // per epilogue warp
constexpr int DT_MAX_STAGES = 6;
constexpr int DT_TILE_ATOMS = 4;                 // 64-column atoms of a column tile
constexpr int DT_LCAP = DENSE_LEFT_CAP;          // listed entries outside the window, per row
constexpr unsigned char DT_OVERFLOW = 255;       // left_cnt of a row with more than that
constexpr unsigned char DT_HUB_MARK = 254;       // and of one with more than DT_HUB
constexpr int DT_HUB = 64;                       // entries outside the window up to which a row is not shared by a block
constexpr int DT_HUBS_PER_BLOCK = 24;            // rows of more that a block takes one after another; more of them: a warp each
constexpr int DT_SMEM_MAX = 225 * 1024;           // with the static part (under 2 KB) within the 227 KB a block may have
static_assert(DT_BM == 128 && DENSE_WINDOW % DT_BK == 0 && DT_HALO % DT_BK == 0, "tile shape of the MMA and whole stages");

// byte of a window mask -> the four 32-bit words of the 16-byte chunk it stands for, sixteen ones per set bit
struct MaskLut {
    uint32_t w[256][4];
    constexpr MaskLut() : w{} {
        for (int b = 0; b < 256; ++b)
            for (int p = 0; p < 4; ++p)
                w[b][p] = (((b >> (2 * p)) & 1) ? 0x0000FFFFu : 0u) | (((b >> (2 * p + 1)) & 1) ? 0xFFFF0000u : 0u);
    }
};
__device__ const MaskLut mask_lut{};

struct DenseArgs {
    GroupDesc g;
    const float* inv_deg;
    const int* dense;              // per trainer: 1 = this part is aggregated here
    const unsigned long long* win_bits;  // [scratch row][DT_KB]: bit c of word b = the row has window column 64 b + c
    const unsigned char* block_mask;  // per 32 scratch rows: the window blocks in which one of them has an entry
    const unsigned char* left_cnt; // per scratch row: entries outside the window (DT_OVERFLOW: more than DT_LCAP);
                                   // where it is not 0 the output row holds their sum when the kernel starts
    CUtensorMap mapSh, mapSl;      // source planes, boxes of 64 columns x DT_BK rows
    Planes out;
    int width;                     // columns of the planes that hold data (a multiple of 8)
    int n_atoms;                   // 64-column atoms over the width
    int col_tiles;                 // column tiles of at most DT_TILE_ATOMS atoms
    int tmem_cols, stages;
    int64_t row_tiles;
    int* error_word;
};

struct DenseBarriers {
    uint64_t full[DT_MAX_STAGES];   // source rows landed and A written
    uint64_t empty[DT_MAX_STAGES];  // the MMAs have read the stage
    uint64_t acc_full[2];
    uint64_t acc_empty[2];
    uint64_t builders;              // meeting point of the builder threads (transposed pass)
    uint32_t tmem_base;
    int abort;
};

__device__ __forceinline__ bool dense_wait(uint64_t* bar, uint32_t parity, DenseBarriers* pb, int* error_word) {
    for (uint32_t i = 0; i < tc::WAIT_POLLS; ++i) {
        if (tc::mbar_try_wait(bar, parity)) return true;
        if ((i & 1023u) == 1023u && *reinterpret_cast<volatile int*>(&pb->abort)) break;
    }
    *reinterpret_cast<volatile int*>(&pb->abort) = 1;
    atomicExch(error_word, 1);
    return false;
}

// Adds to the bytes the barrier's current phase waits for, without arriving.
__device__ __forceinline__ void expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(tc::smem_u32(bar)), "r"(bytes) : "memory");
}

// 32 lanes x 16 consecutive 32-bit columns of tensor memory: thread i of the warp receives lane (base lane + i).
__device__ __forceinline__ void tmem_load_32x16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// A tile of a block's walk.  What a role needs of it first is requested when the walk comes to it, a tile ahead of its use: every
// role goes through the same loads tile after tile, and waited for them each time.
struct TileAt {
    bool valid;
    int k, r0, ct, n_p;    // slot of its part in the group, first row in the part, column tile, rows of the part
    int64_t ws;            // first scratch row of the part
    uint32_t mask[DT_BM / 32];
    // The stages of the tile: bit b = some row of the tile has an entry in window block b (of 100-member super-nodes kept
    // together, 4.7 of 6 on average; the blocks left out cost 64 source rows through shared memory and an MMA of zeros each).
    // A tile without any takes the block of its own first rows, so that its accumulator is written.
    __device__ __forceinline__ uint32_t blocks() const {
        uint32_t m = 0;
#pragma unroll
        for (int j = 0; j < DT_BM / 32; ++j) m |= mask[j];
        return m ? m : 1u << (DT_HALO / DT_BK);
    }
};
// A block's tiles blockIdx.x, blockIdx.x + gridDim.x, ..., without those of parts that are not aggregated here
struct TileWalk {
    uint32_t tile, total;
    int k;           // the part reached, and its first row tile
    uint32_t base;
    __device__ __forceinline__ TileWalk(const DenseArgs& a) : tile(blockIdx.x), total((uint32_t)(a.row_tiles * a.col_tiles)), k(0), base(0) {}
    __device__ __forceinline__ TileAt next(const DenseArgs& a) {
        TileAt t{};
        for (; tile < total; tile += gridDim.x) {
            const uint32_t row_tile = a.col_tiles == 1 ? tile : tile / (uint32_t)a.col_tiles;
            uint32_t here;
            while (row_tile >= base + (here = (uint32_t)(a.g.rows[k] + DT_BM - 1) / DT_BM)) {
                base += here;
                ++k;
            }
            if (!a.dense[a.g.part[k]]) continue;
            t.valid = true;
            t.k = k;
            t.r0 = (int)(row_tile - base) * DT_BM;
            t.ct = a.col_tiles == 1 ? 0 : (int)(tile - row_tile * (uint32_t)a.col_tiles);
            t.n_p = a.g.rows[k];
            t.ws = a.g.row_ws[k];
#pragma unroll
            for (int j = 0; j < DT_BM / 32; ++j) t.mask[j] = t.r0 + 32 * j < t.n_p ? __ldg(a.block_mask + (t.ws + t.r0) / 32 + j) : 0u;
            tile += gridDim.x;
            break;
        }
        return t;
    }
};

// TRANSPOSED = false: A counts, out = (1 / deg v) * A src;  true: A = counts x 1 / deg u, out = A src
// AHEAD: the rows' windows and weights are requested a tile ahead
template <bool TRANSPOSED, bool AHEAD>
__global__ void __launch_bounds__(DT_THREADS, 1) spmm_dense_kernel(const __grid_constant__ DenseArgs a) {
    wait_for_kernel_before();
    extern __shared__ uint8_t smem_raw[];
    __shared__ DenseBarriers pb;
    {   // nothing to do unless a part of this launch is aggregated here: leave before any set-up
        bool any = false;
        for (int k = 0; k < a.g.num; ++k) any = any || a.dense[a.g.part[k]] != 0;
        if (!any) return;
    }
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int stages = a.stages;
    constexpr uint32_t NPA = TRANSPOSED ? 2u : 1u;  // planes of A
    // a stage: the plane(s) of A, then the tile's atoms of the hi plane of the source rows and, right behind
    // them, those of the lo plane: one N-major operand of twice the tile's width
    const uint32_t stage_bytes = NPA * DT_A_BYTES + 2u * (uint32_t)min(DT_TILE_ATOMS, a.n_atoms) * DT_ATOM_BYTES;
    auto a_hi = [&](int s) { return smem + (size_t)s * stage_bytes; };
    auto a_lo = [&](int s) { return smem + (size_t)s * stage_bytes + DT_A_BYTES; };
    auto b_hi = [&](int s) { return smem + (size_t)s * stage_bytes + NPA * DT_A_BYTES; };

    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            tc::mbar_init(&pb.full[s], DT_BUILDERS);
            tc::mbar_init(&pb.empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(&pb.acc_full[b], 1);
            tc::mbar_init(&pb.acc_empty[b], DT_EPI_THREADS);
        }
        tc::mbar_init(&pb.builders, DT_BUILDERS);
        pb.abort = 0;
        tc::fence_barrier_init();
        tc::prefetch_tensormap(&a.mapSh);
        tc::prefetch_tensormap(&a.mapSl);
    }
    if (warp == 0) {
        tc::tmem_alloc(&pb.tmem_base, 2u * (uint32_t)a.tmem_cols);
        tc::tmem_relinquish();
    }
    tc::tc_fence_before_sync();
    __syncthreads();
    tc::tc_fence_after_sync();
    const uint32_t tmem_base = pb.tmem_base;

    // Every role walks the same tiles in the same order and skips the same ones: `at` follows the stages and `t` counts the
    // tiles a block has worked on, and both must agree between the roles.
    if (warp == 0) {
        if (lane == 0) {
            // One thread feeds the tensor core: descriptors are a constant plus an address in units of 16 bytes.
            // A is K-major (a 128-byte row holds the 64 window rows of the stage): 16 of them = 32 bytes;
            // the source rows are N-major (a 128-byte row per window row): 16 of them = 2048 bytes.
            const uint64_t desc_a = tc::smem_desc_sw128(0, 16, 1024), desc_b = tc::smem_desc_sw128(0, DT_ATOM_BYTES, 1024);
            tc::RingAt at;
            uint32_t t = 0;
            bool ok = true;
            TileWalk walk(a);
            TileAt tile = walk.next(a);
            while (tile.valid && ok) {
                const int NA = min(DT_TILE_ATOMS, a.n_atoms - DT_TILE_ATOMS * tile.ct);
                const int n_stages = __popc(tile.blocks());
                tile = walk.next(a);
                // A tile of at most two atoms multiplies A with [hi | lo] (the lo atoms lie right behind the hi atoms)
                // in ONE MMA of twice the tile's width: columns [0, 64 NA) of the accumulator take the product with the
                // hi plane, [64 NA, 128 NA) that with the lo plane, and the epilogue adds the halves.  An MMA that
                // narrow costs its issue, not its arithmetic.  Wider tiles take one MMA per plane into the same columns.
                const bool joined = NA <= 2;
                const uint32_t idesc_hi = tc::idesc_bf16(DT_BM, 64 * NA, false, true);
                const uint32_t idesc_first = joined ? tc::idesc_bf16(DT_BM, 128 * NA, false, true) : idesc_hi;
                const uint32_t lo_off = (uint32_t)NA * (DT_ATOM_BYTES >> 4);
                const int buf = (int)(t & 1);
                ok = dense_wait(&pb.acc_empty[buf], ((t >> 1) & 1u) ^ 1u, &pb, a.error_word);
                if (!ok) break;
                tc::tc_fence_after_sync();
                const uint32_t d_tmem = tmem_base + (uint32_t)(buf * a.tmem_cols);
                for (int stage = 0; stage < n_stages; ++stage, at.advance(stages)) {
                    const int s = at.s;
                    ok = dense_wait(&pb.full[s], at.phase, &pb, a.error_word);
                    if (!ok) break;
                    tc::tc_fence_after_sync();
                    const uint32_t ah = tc::smem_u32(a_hi(s)) >> 4, al = tc::smem_u32(a_lo(s)) >> 4, bh = tc::smem_u32(b_hi(s)) >> 4;
#pragma unroll
                    for (int ks = 0; ks < DT_BK / 16; ++ks) {
                        const uint64_t dah = desc_a + (ah + 2 * ks), db = desc_b + (bh + 128 * ks);
                        tc::mma_bf16(d_tmem, dah, joined ? db : db + lo_off, idesc_first, stage > 0 || ks > 0 ? 1u : 0u);
                        if (!joined) tc::mma_bf16(d_tmem, dah, db, idesc_hi, 1u);
                        if (TRANSPOSED) tc::mma_bf16(d_tmem, desc_a + (al + 2 * ks), db, idesc_hi, 1u);  // + A_lo * hi (into the first half)
                    }
                    tc::mma_commit(&pb.empty[s]);
                }
                if (ok) tc::mma_commit(&pb.acc_full[buf]);
                ++t;
            }
        }
    } else if (warp < 1 + DT_BUILDERS / 32) {
        const int r = threadIdx.x - 32;  // the tile row this thread writes
        const uint32_t swz = (uint32_t)(r & 7);
        // transposed pass: the split weights 1 / deg of the tile's window rows, stage by stage as the 32 words
        // of a row of A with every bit set; written once per tile between two barriers of the builder warps
        __shared__ __align__(16) uint32_t wpair[DT_KB][2][DT_BK / 2];
        tc::RingAt at;
        uint32_t meetings = 0;
        // all builder threads meet (a bounded wait like every other: a thread that has given up is not waited for)
        auto meet = [&]() {
            tc::mbar_arrive(&pb.builders);
            return dense_wait(&pb.builders, meetings++ & 1u, &pb, a.error_word);
        };
        // the window of the thread's row and (transposed pass) the weights of the tile's window rows r, r + 128, ...
        constexpr int PER_THREAD = DENSE_WINDOW / DT_BUILDERS;
        unsigned long long next_bits[DT_KB];
        float next_w[PER_THREAD];
        auto request = [&](const TileAt& t) {
#pragma unroll
            for (int q = 0; q < DT_KB; ++q) next_bits[q] = 0ULL;
            if (t.valid && t.r0 + r < t.n_p) {
                const ulonglong2* wb = reinterpret_cast<const ulonglong2*>(a.win_bits + (t.ws + t.r0 + r) * DT_KB);
#pragma unroll
                for (int q = 0; q < DT_KB / 2; ++q) {
                    const ulonglong2 v2 = __ldg(wb + q);
                    next_bits[2 * q] = v2.x;
                    next_bits[2 * q + 1] = v2.y;
                }
            }
            if (TRANSPOSED) {
#pragma unroll
                for (int q = 0; q < PER_THREAD; ++q) {
                    const int u = t.r0 - DT_HALO + q * DT_BUILDERS + r;
                    next_w[q] = t.valid && u >= 0 && u < t.n_p ? __ldg(a.inv_deg + t.ws + u) : 0.f;
                }
            }
        };
        bool ok = true;
        TileWalk walk(a);
        TileAt tile = walk.next(a);
        if (AHEAD) request(tile);
        while (tile.valid && ok) {
            if (!AHEAD) request(tile);
            const uint32_t blocks = tile.blocks();
            const int NA = min(DT_TILE_ATOMS, a.n_atoms - DT_TILE_ATOMS * tile.ct);
            const int ct = tile.ct, y0 = (int)(tile.ws + tile.r0 - DT_HALO);  // the window's first scratch row; may be negative: reads zeros
            unsigned long long bits[DT_KB];
#pragma unroll
            for (int q = 0; q < DT_KB; ++q) bits[q] = next_bits[q];
            if (TRANSPOSED) {
                ok = meet();  // every thread has written the previous tile's last stage
                if (!ok) break;
#pragma unroll
                for (int q = 0; q < PER_THREAD; ++q) {
                    const int wr = q * DT_BUILDERS + r;  // window row
                    uint32_t h, l;
                    split_bits(next_w[q], h, l);
                    reinterpret_cast<unsigned short*>(wpair[wr / DT_BK][0])[wr % DT_BK] = (unsigned short)h;
                    reinterpret_cast<unsigned short*>(wpair[wr / DT_BK][1])[wr % DT_BK] = (unsigned short)l;
                }
                ok = meet();
                if (!ok) break;
            }
            if (AHEAD) {
                tile = walk.next(a);
                request(tile);
            }
            for (uint32_t rest = blocks; rest; rest &= rest - 1, at.advance(stages)) {
                const int kb = __ffs(rest) - 1;
                const int s = at.s;
                ok = dense_wait(&pb.empty[s], at.phase ^ 1u, &pb, a.error_word);
                if (!ok) break;
                if (r == 0) {
                    // the stage's source rows, requested before this thread writes its row of A: window rows
                    // 64 kb .. 64 kb + 63, all column atoms of the tile
                    expect_tx(&pb.full[s], 2u * (uint32_t)NA * DT_ATOM_BYTES);
                    const int y = y0 + kb * DT_BK;
                    for (int t = 0; t < NA; ++t) {
                        tc::tma_load_2d(b_hi(s) + t * DT_ATOM_BYTES, &a.mapSh, &pb.full[s], (DT_TILE_ATOMS * ct + t) * 64, y);
                        tc::tma_load_2d(b_hi(s) + (NA + t) * DT_ATOM_BYTES, &a.mapSl, &pb.full[s], (DT_TILE_ATOMS * ct + t) * 64, y);
                    }
                }
                unsigned long long m = bits[0];
#pragma unroll
                for (int q = 1; q < DT_KB; ++q) m = kb == q ? bits[q] : m;
                // row r of the stage's A: 128 bytes, 16-byte chunk c (8 window rows) stored at chunk c ^ (r % 8)
                uint8_t* row_hi = a_hi(s) + r * 128;
                uint8_t* row_lo = a_lo(s) + r * 128;
#pragma unroll
                for (uint32_t c4 = 0; c4 < 8; c4 += 4) {  // four chunks at a time: all their loads, then all their stores
                    uint4 mk[4];  // sixteen ones for every set bit
#pragma unroll
                    for (uint32_t c = 0; c < 4; ++c)
                        mk[c] = __ldg(reinterpret_cast<const uint4*>(mask_lut.w[(uint32_t)(m >> (8 * (c4 + c))) & 0xFFu]));
                    if (TRANSPOSED) {
                        uint4 wh[4], wl[4];
#pragma unroll
                        for (uint32_t c = 0; c < 4; ++c) {
                            wh[c] = *reinterpret_cast<const uint4*>(&wpair[kb][0][4 * (c4 + c)]);
                            wl[c] = *reinterpret_cast<const uint4*>(&wpair[kb][1][4 * (c4 + c)]);
                        }
#pragma unroll
                        for (uint32_t c = 0; c < 4; ++c) {
                            *reinterpret_cast<uint4*>(row_hi + (((c4 + c) ^ swz) << 4)) =
                                make_uint4(mk[c].x & wh[c].x, mk[c].y & wh[c].y, mk[c].z & wh[c].z, mk[c].w & wh[c].w);
                            *reinterpret_cast<uint4*>(row_lo + (((c4 + c) ^ swz) << 4)) =
                                make_uint4(mk[c].x & wl[c].x, mk[c].y & wl[c].y, mk[c].z & wl[c].z, mk[c].w & wl[c].w);
                        }
                    } else {
                        constexpr uint32_t ONES = 0x3F803F80u;  // 1.0 | 1.0
#pragma unroll
                        for (uint32_t c = 0; c < 4; ++c)
                            *reinterpret_cast<uint4*>(row_hi + (((c4 + c) ^ swz) << 4)) =
                                make_uint4(mk[c].x & ONES, mk[c].y & ONES, mk[c].z & ONES, mk[c].w & ONES);
                    }
                }
                tc::fence_proxy_async_smem();  // the tensor core reads what this thread has just written
                tc::mbar_arrive(&pb.full[s]);
            }
            if (!AHEAD) tile = walk.next(a);
        }
    } else {
        const int ew = warp - (1 + DT_BUILDERS / 32);  // 0..7
        const int q = warp & 3;                        // the quarter of the tensor memory's lanes this warp may read
        const int col_phase = ew >> 2;                 // which of the quarter's two warps: even or odd 32-column chunks
        uint8_t* stg = smem + (size_t)stages * stage_bytes + (size_t)ew * DT_STAGING_BYTES;
        float4* st = reinterpret_cast<float4*>(stg);
        const int p = lane & 3;
        const uint32_t out_row_bytes = (uint32_t)a.out.ld * 2u;
        TileWalk walk(a);
        TileAt tile = walk.next(a);
        uint32_t t = 0;
        bool ok = true;
        while (tile.valid && ok) {
            const int k = tile.k, r0 = tile.r0, ct = tile.ct;
            const int BN = 64 * min(DT_TILE_ATOMS, a.n_atoms - DT_TILE_ATOMS * ct);
            const int n0 = ct * 64 * DT_TILE_ATOMS;
            const int rows_here = min(32, a.g.rows[k] - (r0 + q * 32));
            const int64_t orow0 = a.g.row_ws[k] + r0 + q * 32;
            // of the thread's four rows: the scale, and whether the output row already holds a sum to add to.  (Not a tile ahead: 13 warps leave
            // a thread 128 registers, the loop below needs them, and spilled forward it took 1,290 us instead of 1,100 for 256 columns of 2 M
            // rows, 560 instead of 484 for 64; 1,170 and 550 with two divisions a stage and nothing ahead but this.)
            float scale[4];
            bool has_left[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int row = j * 8 + (lane >> 2);
                scale[j] = 1.f;
                has_left[j] = false;
                if (row < rows_here) {
                    if (!TRANSPOSED) scale[j] = __ldg(a.inv_deg + orow0 + row);
                    has_left[j] = a.left_cnt[orow0 + row] != 0;
                }
            }
            // every chunk's existing rows are requested before the chunk before them is finished: the epilogue is the longest chain of the
            // kernel, and these loads its latency
            uint4 gh[4], gl[4];
            auto request = [&](int c0) {  // what the rows already hold (written by the launch before this one)
                const int n = n0 + c0 + 8 * p;
                if (c0 >= BN || n >= a.width) return;
                const char* oh = reinterpret_cast<const char*>(a.out.hi + (orow0 + (lane >> 2)) * a.out.ld + n);
                const char* ol = reinterpret_cast<const char*>(a.out.lo + (orow0 + (lane >> 2)) * a.out.ld + n);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (has_left[j]) {
                        gh[j] = __ldcg(reinterpret_cast<const uint4*>(oh + (size_t)(j * 8) * out_row_bytes));
                        gl[j] = __ldcg(reinterpret_cast<const uint4*>(ol + (size_t)(j * 8) * out_row_bytes));
                    }
                }
            };
            request(col_phase * 32);
            const int buf = (int)(t & 1);
            ok = dense_wait(&pb.acc_full[buf], (t >> 1) & 1u, &pb, a.error_word);
            if (!ok) break;
            tc::tc_fence_after_sync();
            const uint32_t d_tmem = tmem_base + (uint32_t)(buf * a.tmem_cols);
            for (int c0 = col_phase * 32; c0 < BN && rows_here > 0; c0 += 64) {
                // Of a tile of at most two atoms the accumulator holds the product with the hi plane and, BN columns
                // further, that with the lo plane.  The sum goes through the warp's staging slab (16-byte chunk j of row r at chunk
                // j ^ (r % 8)), so that a thread then owns 8 consecutive columns and a store writes whole 64-byte
                // pieces of rows.
                __syncwarp();
#pragma unroll
                for (int half = 0; half < 2; ++half) {  // 16 accumulator columns at a time: few registers
                    float v[16];
                    tmem_load_32x16(d_tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(c0 + 16 * half), v);
                    if (BN <= 128) {  // the tile's planes were multiplied side by side
                        float v2[16];
                        tmem_load_32x16(d_tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(BN + c0 + 16 * half), v2);
#pragma unroll
                        for (int e = 0; e < 16; ++e) v[e] += v2[e];
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int jj = 4 * half + j;
                        st[lane * 8 + (jj ^ (lane & 7))] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
                    }
                }
                __syncwarp();
                const int n = n0 + c0 + 8 * p;
                const bool col_ok = n < a.width;
                char* oh = reinterpret_cast<char*>(a.out.hi + (orow0 + (lane >> 2)) * a.out.ld + n);
                char* ol = reinterpret_cast<char*>(a.out.lo + (orow0 + (lane >> 2)) * a.out.ld + n);
                Pack8 x[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int row = j * 8 + (lane >> 2);
                    const float4 x0 = st[row * 8 + ((2 * p) ^ (row & 7))];
                    const float4 x1 = st[row * 8 + ((2 * p + 1) ^ (row & 7))];
                    x[j].v[0] = x0.x; x[j].v[1] = x0.y; x[j].v[2] = x0.z; x[j].v[3] = x0.w;
                    x[j].v[4] = x1.x; x[j].v[5] = x1.y; x[j].v[6] = x1.z; x[j].v[7] = x1.w;
                    if (has_left[j] && col_ok) x[j].add_planes_mixed(gh[j], gl[j]);
                }
                request(c0 + 64);  // the registers are free again
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int row = j * 8 + (lane >> 2);
                    if (row < rows_here && col_ok) {
                        if (!TRANSPOSED) {
#pragma unroll
                            for (int e = 0; e < 8; ++e) x[j].v[e] *= scale[j];
                        }
                        uint4 h, l;
                        x[j].to_planes_lean(h, l);
                        *reinterpret_cast<uint4*>(oh + (size_t)(j * 8) * out_row_bytes) = h;
                        *reinterpret_cast<uint4*>(ol + (size_t)(j * 8) * out_row_bytes) = l;
                    }
                }
            }
            tc::tc_fence_before_sync();
            tc::mbar_arrive(&pb.acc_empty[buf]);
            ++t;
            tile = walk.next(a);
        }
    }
    tc::tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem_base, 2u * (uint32_t)a.tmem_cols);
}

// The n-th set bit of m (n from 0), or 32: halving by popcounts.  (__fns walks the bits.)
__device__ __forceinline__ unsigned nth_bit(unsigned m, int n) {
    unsigned pos = 0;
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) {
        const int c = __popc((m >> pos) & ((1u << w) - 1u));
        if (n >= c) {
            n -= c;
            pos += w;
        }
    }
    return n == 0 && (m >> pos & 1u) ? pos : 32u;
}

// The entries outside the window of their row's tile, before the tiles run: for every row that has any,
// out[row] = their sum (transposed pass: weighted by 1 / deg of the column), unscaled; the tile's epilogue adds
// its product and the scale.  Bound by the latency of chains of loads, so the rows are told apart, and rows that take long
// begin first.  Blocks 0 .. hub_blocks - 1 take the rows of more than DT_HUB such entries, a block each: its warps take every eighth piece of
// 32 of the row's entries in the part's CSR, and the sums are added in a fixed order.  The next many_blocks take the other rows of more than
// DT_LCAP, a warp each.  The rest: a warp takes 32 consecutive rows with up to DT_LCAP, their counts and listed columns with one load
// each; then the rows that have entries, several at a time, two source rows of each requested together (most
// rows have one or two).  LPR lanes own a row (pieces of 8 values per lane): 32 for rows wider than 64 values,
// two rows at a time per warp; 8 for narrower rows, eight at a time, two per quarter of the warp.
// In one kernel with the long rows looked up by the warp that met them: 610 us for 2 M rows of 256 values of which 27 % have such
// entries (1.2 M entries; now 335), of 48 values 285 (now 180), 40,000 rows with hubs of 280 entries 105 (now 23).
// MANY: all blocks but those of the hubs take long rows (the last ones behind them their listed rows), and the hubs if no block takes them, a
// warp each, with the sums in the same order; and where the scratch had no room to list the long rows, 32 rows at a time are looked
// through for their marks.  launch_spmm_dense says when.
template <bool TRANSPOSED, int LPR, bool MANY>
__global__ void __launch_bounds__(256, 3)
spmm_outside_kernel(const __grid_constant__ GroupDesc g, const int64_t* __restrict__ rowptr_out,
                    const int32_t* __restrict__ col_out, const float* __restrict__ inv_deg,
                    const int* __restrict__ dense, const unsigned char* __restrict__ left_cnt,
                    const int32_t* __restrict__ left_col, const LongRows long_rows, const unsigned hub_blocks, const unsigned many_blocks,
                    const Planes src, const Planes out, const int width, const int64_t total_groups) {
    wait_for_kernel_before();
    constexpr int S = 32 / LPR;            // rows side by side in a warp
    constexpr int NR = 2;                  // rows a lane works on at a time
    constexpr int EL = 2;                  // listed entries of each of them requested together (most rows have one or two)
    const int lane = threadIdx.x & 31;
    const int sub = lane / LPR, sl = lane % LPR;
    const int warp = threadIdx.x >> 5;
    if (MANY || blockIdx.x < hub_blocks + many_blocks) {
        // ---- the rows whose entries are looked up again ----
        // A hub block takes hubs; the warps of the other blocks take the other long rows, and the hubs if there are no hub blocks
        const bool hub_block = blockIdx.x < hub_blocks, hub_by_warp = MANY && hub_blocks == 0;
        const int mine_hub = hub_block || hub_by_warp ? long_rows.hubs : 0, mine_many = hub_block ? 0 : long_rows.many;
        __shared__ __align__(16) float piece[8][LPR * 8];
        // the sum of one row by this warp (a hub in a hub block: of this warp's share, the block's first warp then adds the shares and
        // stores; a hub elsewhere: share by share)
        auto do_row = [&](const int row, const bool marked_hub) {
            const bool hub = MANY ? marked_hub : hub_block;
            int k = 0;
            while (k < g.num && !(row >= g.row_ws[k] && row < g.row_ws[k] + g.rows[k])) ++k;
            if (k == g.num || !dense[g.part[k]]) return;  // past a part's end, of a part that has finished its steps or was taken back
            const int i = (int)(row - g.row_ws[k]), n_p = g.rows[k];
            const int64_t ws = g.row_ws[k];
            const int64_t* rp = rowptr_out + g.row_abs[k] + g.part[k];
            const int32_t* cols = col_out + g.edge_abs[k];
            const int w_begin = i / DT_BM * DT_BM - DT_HALO, w_end = w_begin + DENSE_WINDOW;
            const int64_t e0 = rp[i], e1 = rp[i + 1];
            for (int cb = 0; cb < width; cb += LPR * 8) {  // the same trip count for every lane: the shuffles below need the whole warp
                const int c0 = cb + sl * 8;
                const bool live = c0 < width;
                const __nv_bfloat16* sh = src.hi + ws * src.ld + (live ? c0 : 0);  // lanes past the width read column 0 and store nothing
                const __nv_bfloat16* sl_ = src.lo + ws * src.ld + (live ? c0 : 0);
                Pack8 acc;
                for (int share = 0; share < (MANY && hub && !hub_block ? 8 : 1); ++share) {
                    const int64_t eb0 = e0 + (hub ? (hub_block ? warp : share) * 32 : 0);
                    if (share > 0 && eb0 >= e1) break;  // acc holds the sum of the shares before
                    acc.zero();
                    for (int64_t eb = eb0; eb < e1; eb += hub ? 8 * 32 : 32) {
                        const int64_t e = eb + lane;
                        bool outside = false;
                        int c = 0;
                        if (e < e1) {
                            c = __ldg(cols + e);
                            outside = rtma_index_ok(c, n_p, 5) && (c < w_begin || c >= w_end);
                        }
                        unsigned votes = __ballot_sync(0xffffffffu, outside);
                        while (votes) {
                            int u[4];
                            uint4 yh[4], yl[4];
                            float wy[4];
#pragma unroll
                            for (int b = 0; b < 4; ++b) {
                                // quarter `sub` takes the entries sub, sub + S, ... of those still to do
                                const unsigned from = nth_bit(votes, b * S + sub);
                                u[b] = __shfl_sync(0xffffffffu, c, from < 32u ? (int)from : 0);
                                if (from >= 32u) u[b] = -1;
                            }
#pragma unroll
                            for (int b = 0; b < 4 * S; ++b) votes &= votes - 1;
#pragma unroll
                            for (int b = 0; b < 4; ++b) {
                                if (u[b] >= 0) {
                                    yh[b] = __ldg(reinterpret_cast<const uint4*>(sh + (int64_t)u[b] * src.ld));
                                    yl[b] = __ldg(reinterpret_cast<const uint4*>(sl_ + (int64_t)u[b] * src.ld));
                                    if (TRANSPOSED) wy[b] = __ldg(inv_deg + ws + u[b]);
                                }
                            }
#pragma unroll
                            for (int b = 0; b < 4; ++b) {
                                if (u[b] >= 0) {
                                    if (TRANSPOSED) acc.fma_planes_mixed(wy[b], yh[b], yl[b]);
                                    else acc.add_planes_mixed(yh[b], yl[b]);
                                }
                            }
                        }
                    }
                    // the quarters' sums, added in a fixed order
#pragma unroll
                    for (int step_ = S / 2; step_ > 0; step_ >>= 1)
#pragma unroll
                        for (int e = 0; e < 8; ++e) acc.v[e] += __shfl_down_sync(0xffffffffu, acc.v[e], step_ * LPR);
                    if (MANY && hub && !hub_block && sub == 0) {  // the shares' sums, added as a block adds them
                        for (int e = 0; e < 8; ++e) {
                            float& sum = piece[warp][sl * 8 + e];
                            sum = acc.v[e] = share == 0 ? acc.v[e] : sum + acc.v[e];
                        }
                    }
                }
                if (hub_block) {  // and the warps'
                    __syncthreads();
                    if (sub == 0)
#pragma unroll
                        for (int e = 0; e < 8; ++e) piece[warp][sl * 8 + e] = acc.v[e];
                    __syncthreads();
                    if (warp == 0 && sub == 0) {
                        for (int w = 1; w < 8; ++w)
#pragma unroll
                            for (int e = 0; e < 8; ++e) acc.v[e] += piece[w][sl * 8 + e];
                    }
                }
                if (live && sub == 0 && (!hub_block || warp == 0)) {
                    uint4 h, l;
                    acc.to_planes_lean(h, l);
                    *reinterpret_cast<uint4*>(out.hi + (int64_t)row * out.ld + c0) = h;
                    *reinterpret_cast<uint4*>(out.lo + (int64_t)row * out.ld + c0) = l;
                }
            }
        };
        // scratch rows from the list's front (hubs) or back, or 32 rows and their marks
        const bool listed = !MANY || long_rows.listed;
        const int takers = (int)(MANY ? gridDim.x - hub_blocks : many_blocks);  // blocks whose warps take rows
        const int items = listed ? mine_hub + mine_many : (int)total_groups, step = hub_block ? (int)hub_blocks : takers * 8;
#pragma unroll 1
        for (int item = hub_block ? (int)blockIdx.x : (int)(blockIdx.x - hub_blocks) * 8 + warp; item < items; item += step) {
            int first;
            unsigned rest = 1u, hubs;
            if (listed) {
                hubs = item < mine_hub ? 1u : 0u;
                first = long_rows.list[hubs ? (int64_t)item : long_rows.room - 1 - (item - mine_hub)];
            } else {
                int k, i0;
                if (!locate_tile(g, 32, item, &k, &i0)) break;
                first = (int)g.row_ws[k] + i0;
                const int mark = dense[g.part[k]] && i0 + lane < g.rows[k] ? (int)left_cnt[first + lane] : 0;
                hubs = __ballot_sync(0xffffffffu, mark == DT_HUB_MARK && mine_hub > 0);
                rest = __ballot_sync(0xffffffffu, mark == DT_OVERFLOW && mine_many > 0) | hubs;
            }
#pragma unroll 1
            for (; rest; rest &= rest - 1) {
                const int at = __ffs(rest) - 1;
                do_row(first + at, hubs >> at & 1u);
            }
        }
        if (blockIdx.x < hub_blocks + many_blocks) return;
    }
    const int64_t warps = (int64_t)(gridDim.x - hub_blocks - many_blocks) * 8;
    for (int64_t grp = (int64_t)(blockIdx.x - hub_blocks - many_blocks) * 8 + warp; grp < total_groups; grp += warps) {
        int k, i0;
        if (!locate_tile(g, 32, grp, &k, &i0)) break;
        if (!dense[g.part[k]]) continue;
        const int n_p = g.rows[k];
        const int64_t ws = g.row_ws[k];
        const int my_cnt = i0 + lane < n_p ? (int)left_cnt[ws + i0 + lane] : 0;
        int4 my_cols = make_int4(0, 0, 0, 0);
        if (my_cnt > 0 && my_cnt <= DT_LCAP) my_cols = *reinterpret_cast<const int4*>(left_col + (ws + i0 + lane) * DT_LCAP);
        const unsigned listed = __ballot_sync(0xffffffffu, my_cnt > 0 && my_cnt <= DT_LCAP);
        if (!listed) continue;
        const __nv_bfloat16* sh = src.hi + ws * src.ld;
        const __nv_bfloat16* sl_ = src.lo + ws * src.ld;
        for (int cb = 0; cb < width; cb += LPR * 8) {  // the same trip count for every lane: the shuffles below need the whole warp
            const int c0 = cb + sl * 8;
            const bool live = c0 < width;
            const int cx = live ? c0 : 0;  // lanes past the width read column 0 and store nothing
            for (unsigned rest = listed; rest;) {
                int row[NR], cnt[NR];
                int4 cols[NR];
#pragma unroll
                for (int t = 0; t < NR; ++t) {
                    // the (t * S + sub)-th row still to do
                    const unsigned owner = S == 1 ? (unsigned)(__ffs(rest) - 1) : nth_bit(rest, t * S + sub);
                    const bool have = owner < 32u;
                    const int from = have ? (int)owner : 0;
                    row[t] = i0 + from;
                    cnt[t] = __shfl_sync(0xffffffffu, my_cnt, from);
                    cols[t].x = __shfl_sync(0xffffffffu, my_cols.x, from);
                    cols[t].y = __shfl_sync(0xffffffffu, my_cols.y, from);
                    cols[t].z = __shfl_sync(0xffffffffu, my_cols.z, from);
                    cols[t].w = __shfl_sync(0xffffffffu, my_cols.w, from);
                    if (!have) cnt[t] = 0;
                    if (S == 1) rest &= rest - 1;
                }
                if (S > 1) {
#pragma unroll
                    for (int t = 0; t < S * NR; ++t) rest &= rest - 1;
                }
                Pack8 acc[NR];
#pragma unroll
                for (int t = 0; t < NR; ++t) acc[t].zero();
                bool more = true;
#pragma unroll
                for (int l0 = 0; l0 < DT_LCAP; l0 += EL) {
                    if (l0 > 0) {  // a further round only where some row of the warp has that many entries
                        bool mine = false;
#pragma unroll
                        for (int t = 0; t < NR; ++t) mine = mine || cnt[t] > l0;
                        more = __any_sync(0xffffffffu, mine);
                    }
                    if (!more) break;
                    uint4 xh[NR][EL], xl[NR][EL];
                    float wt[NR][EL];
#pragma unroll
                    for (int t = 0; t < NR; ++t) {
                        const int us[DT_LCAP] = {cols[t].x, cols[t].y, cols[t].z, cols[t].w};
#pragma unroll
                        for (int l = 0; l < EL; ++l) {
                            if (l0 + l < cnt[t]) {
                                xh[t][l] = __ldg(reinterpret_cast<const uint4*>(sh + (int64_t)us[l0 + l] * src.ld + cx));
                                xl[t][l] = __ldg(reinterpret_cast<const uint4*>(sl_ + (int64_t)us[l0 + l] * src.ld + cx));
                                if (TRANSPOSED) wt[t][l] = __ldg(inv_deg + ws + us[l0 + l]);
                            }
                        }
                    }
#pragma unroll
                    for (int t = 0; t < NR; ++t) {
#pragma unroll
                        for (int l = 0; l < EL; ++l) {
                            if (l0 + l < cnt[t]) {
                                if (TRANSPOSED) acc[t].fma_planes_mixed(wt[t][l], xh[t][l], xl[t][l]);
                                else acc[t].add_planes_mixed(xh[t][l], xl[t][l]);
                            }
                        }
                    }
                }
#pragma unroll
                for (int t = 0; t < NR; ++t) {
                    if (cnt[t] > 0 && live) {
                        uint4 h, l;
                        acc[t].to_planes_lean(h, l);
                        *reinterpret_cast<uint4*>(out.hi + (ws + row[t]) * out.ld + c0) = h;
                        *reinterpret_cast<uint4*>(out.lo + (ws + row[t]) * out.ld + c0) = l;
                    }
                }
            }
        }
    }
}

// Once per call, for every row of a part that takes the tiles: its window as DT_KB 64-bit masks, and the
// entries outside the window in row order: up to DT_LCAP columns and their number, or DT_OVERFLOW or DT_HUB_MARK when there
// are more; and such rows in long_rows, hubs from its front (long_count[0] of them), others from its back ([1]), as far as its long_room
// words reach: the list is complete if the two numbers together are no larger.  A row that repeats an entry inside its window takes its
// part back to the gather kernels (dense[trainer] = 0): a bit cannot count.
__global__ void __launch_bounds__(256)
dense_lists_kernel(const __grid_constant__ GroupDesc g, const int64_t* __restrict__ rowptr_out,
                   const int32_t* __restrict__ col_out, int* __restrict__ dense,
                   unsigned long long* __restrict__ win_bits, unsigned char* __restrict__ block_mask,
                   unsigned char* __restrict__ left_cnt, int32_t* __restrict__ left_col, int* __restrict__ long_count, int32_t* __restrict__ long_rows,
                   const int64_t long_room) {
    wait_for_kernel_before();
    int k, r0;
    if (!locate_tile(g, 256, blockIdx.x, &k, &r0)) return;
    const int i = r0 + threadIdx.x;
    if (!__any_sync(0xffffffffu, i < g.rows[k] && *reinterpret_cast<volatile int*>(dense + g.part[k]))) return;
    const bool live = i < g.rows[k];
    const int64_t* rp = rowptr_out + g.row_abs[k] + g.part[k];
    const int32_t* cols = col_out + g.edge_abs[k];
    const int64_t row = g.row_ws[k] + i;
    const int w_begin = i / DT_BM * DT_BM - DT_HALO, w_end = w_begin + DENSE_WINDOW;
    unsigned long long bits[DT_KB];
#pragma unroll
    for (int q = 0; q < DT_KB; ++q) bits[q] = 0ULL;
    bool repeated = false;
    int cnt = 0;
    const int64_t e_end = live ? rp[i + 1] : 0;
    for (int64_t e = live ? rp[i] : 0; e < e_end; ++e) {
        const int c = cols[e];
        if (!rtma_index_ok(c, g.rows[k], 5)) continue;
        if (c >= w_begin && c < w_end) {
            const int rel = c - w_begin;
            const unsigned long long bit = 1ULL << (rel & 63);
#pragma unroll
            for (int q = 0; q < DT_KB; ++q) {
                if ((rel >> 6) == q) {
                    repeated = repeated || (bits[q] & bit) != 0ULL;
                    bits[q] |= bit;
                }
            }
        } else {
            if (cnt < DT_LCAP) left_col[row * DT_LCAP + cnt] = c;
            ++cnt;
        }
    }
    __syncwarp();
    uint32_t blocks = 0;
#pragma unroll
    for (int q = 0; q < DT_KB; ++q) blocks |= bits[q] ? 1u << q : 0u;
    blocks = __reduce_or_sync(0xffffffffu, blocks);
    if (!live) return;
    if ((threadIdx.x & 31) == 0) block_mask[row / 32] = (unsigned char)blocks;  // parts start at multiples of 64 scratch rows
    if (cnt > DT_LCAP) {  // the order in the list does not matter
        const bool hub = cnt > DT_HUB;
        const int64_t at = atomicAdd(long_count + (hub ? 0 : 1), 1);
        if (at < long_room) long_rows[hub ? at : long_room - 1 - at] = (int32_t)row;
    }
#pragma unroll
    for (int q = 0; q < DT_KB; ++q) win_bits[row * DT_KB + q] = bits[q];
    left_cnt[row] = cnt <= DT_LCAP ? (unsigned char)cnt : cnt <= DT_HUB ? DT_OVERFLOW : DT_HUB_MARK;
    if (repeated) dense[g.part[k]] = 0;
}

// Sample of a part's rows: the first row of every 64 (a function of the part alone, whatever shares its
// launch).  counts[3 p + 0 .. 2] += entries inside the window of the row's tile, entries, rows.
__global__ void __launch_bounds__(256)
dense_probe_kernel(const __grid_constant__ GroupDesc g, const int64_t* __restrict__ rowptr_out,
                   const int32_t* __restrict__ col_out, const int64_t tiles, unsigned long long* __restrict__ counts) {
    wait_for_kernel_before();
    for (int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x; t < tiles; t += (int64_t)gridDim.x * 256) {
        int k, i;
        if (!locate_tile(g, 64, t, &k, &i)) break;
        const int64_t* rp = rowptr_out + g.row_abs[k] + g.part[k];
        const int32_t* cols = col_out + g.edge_abs[k];
        const int w_begin = i / DT_BM * DT_BM - DT_HALO, w_end = w_begin + DENSE_WINDOW;
        unsigned long long inside = 0;
        const int64_t b = rp[i], e = rp[i + 1];
        for (int64_t x = b; x < e; ++x) {
            const int c = cols[x];
            inside += (c >= w_begin && c < w_end) ? 1u : 0u;
        }
        // integer sums: their order does not matter.  Lanes whose rows lie in the same part add up first.
        unsigned long long entries = (unsigned long long)(e - b), rows = 1ULL;
        const unsigned peers = __match_any_sync(__activemask(), k);
        const int leader = __ffs(peers) - 1;
        for (unsigned rest = peers & ~(1u << leader); rest; rest &= rest - 1) {
            const int src_lane = __ffs(rest) - 1;
            const unsigned long long a0 = __shfl_sync(peers, inside, src_lane), a1 = __shfl_sync(peers, entries, src_lane);
            if ((int)(threadIdx.x & 31) == leader) {
                inside += a0;
                entries += a1;
                rows += 1ULL;
            }
        }
        if ((int)(threadIdx.x & 31) == leader) {
            unsigned long long* cnt = counts + 3 * g.part[k];
            atomicAdd(cnt, inside);
            atomicAdd(cnt + 1, entries);
            atomicAdd(cnt + 2, rows);
        }
    }
}

// dense[trainer] = 1 where at least half of the sampled entries of the part fall into their row's window
// and the sampled rows have at least 4 entries on average (below that, gathering is cheaper than a tile).
__global__ void dense_decide_kernel(const __grid_constant__ GroupDesc g, const unsigned long long* __restrict__ counts,
                                    const int mode, int* __restrict__ dense) {
    wait_for_kernel_before();
    const int k = threadIdx.x;
    if (k >= g.num) return;
    const int p = g.part[k];
    const unsigned long long in_window = counts[3 * p], entries = counts[3 * p + 1], rows = counts[3 * p + 2];
    dense[p] = (mode == 2 || (entries > 0 && 2 * in_window >= entries && entries >= 4 * rows)) ? 1 : 0;
}

}  // namespace

int32_t launch_dense_probe(rtma_ctx* ctx, const GroupDesc& g, const int64_t* rowptr_out, const int32_t* col_out,
                           int mode, unsigned long long* counts, int* dense, cudaStream_t s) {
    const int64_t tiles = group_tiles(g, 64);
    if (tiles == 0) return RTMA_OK;
    const unsigned grid = (unsigned)std::min<int64_t>(ceil_div(tiles, 256), 148 * 4);
    { KernelScope ks(ctx, KC_INV_DEGREE, s); launch_kernel(dense_probe_kernel, grid, 256, 0, s, g, rowptr_out, col_out, tiles, counts); }
    RTMA_LAUNCH_CHECK(ctx);
    { KernelScope ks(ctx, KC_INV_DEGREE, s); launch_kernel(dense_decide_kernel, 1, RTMA_MAX_PARTS, 0, s, g, counts, mode, dense); }
    RTMA_LAUNCH_CHECK(ctx);
    return RTMA_OK;
}

int32_t launch_dense_lists(rtma_ctx* ctx, const GroupDesc& g, const int64_t* rowptr_out, const int32_t* col_out,
                           int* dense, unsigned long long* win_bits, unsigned char* block_mask, unsigned char* left_cnt,
                           int32_t* left_col, int* long_count, int32_t* long_rows, int64_t long_room, cudaStream_t s) {
    const int64_t tiles = group_tiles(g, 256);
    if (tiles == 0) return RTMA_OK;
    { KernelScope ks(ctx, KC_INV_DEGREE, s); launch_kernel(dense_lists_kernel, (unsigned)tiles, 256, 0, s, g, rowptr_out, col_out, dense, win_bits, block_mask, left_cnt, left_col, long_count, long_rows, long_room); }
    RTMA_LAUNCH_CHECK(ctx);
    return RTMA_OK;
}

bool spmm_dense_applies(int d) { return d >= 16 && d <= 1024; }

int32_t launch_spmm_dense(rtma_ctx* ctx, int kclass, const GroupDesc& g, const int64_t* rowptr_out, const int32_t* col_out,
                          const float* inv_deg, const SpmmOrder& order, Planes src, Planes out, int d, bool transposed,
                          cudaStream_t s) {
    const int* dense = order.dense;
    const int64_t rows_total = order.rows_total;
    const int64_t row_tiles = group_tiles(g, DT_BM);
    if (row_tiles == 0) return RTMA_OK;
    if (!ctx->dense_configured) {
        for (const void* kernel : {reinterpret_cast<const void*>(spmm_dense_kernel<false, true>), reinterpret_cast<const void*>(spmm_dense_kernel<true, true>),
                                   reinterpret_cast<const void*>(spmm_dense_kernel<true, false>)})
            RTMA_CUDA(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, DT_SMEM_MAX));
        ctx->dense_configured = true;
    }
    DenseArgs a{};
    a.g = g;
    a.inv_deg = inv_deg;
    a.dense = dense;
    a.win_bits = order.win_bits;
    a.block_mask = order.block_mask;
    a.left_cnt = order.left_cnt;
    a.out = out;
    a.width = (int)planes_ld(d);
    a.n_atoms = (int)ceil_div(a.width, 64);
    a.col_tiles = (int)ceil_div(a.n_atoms, DT_TILE_ATOMS);
    const int tile_atoms = std::min(DT_TILE_ATOMS, a.n_atoms);
    uint32_t tmem = 32;  // columns of one accumulator: twice the tile's width where the two planes' products lie side by side
    while ((int)tmem < (tile_atoms <= 2 ? 128 : 64) * tile_atoms) tmem <<= 1;
    a.tmem_cols = (int)tmem;
    const size_t stage_bytes = (transposed ? 2 : 1) * (size_t)DT_A_BYTES + 2 * (size_t)tile_atoms * DT_ATOM_BYTES;
    const size_t fixed = 1024 + 8 * (size_t)DT_STAGING_BYTES;
    a.stages = (int)std::min<size_t>(DT_MAX_STAGES, (DT_SMEM_MAX - fixed) / stage_bytes);
    if (a.stages < 2) return rtma_fail(ctx, RTMA_ERR_UNSUPPORTED, "internal: aggregation tile does not fit shared memory");
    a.row_tiles = row_tiles;
    if (row_tiles * a.col_tiles >= (int64_t(1) << 31)) return rtma_fail(ctx, RTMA_ERR_OVERFLOW, "too many aggregation tiles");
    a.error_word = ctx->error_word;
    // the planes as [rows_total x width] matrices: rows before the first and past the last scratch row, and
    // columns past the width, read as zero
    if (!make_tensor_map_bf16(&a.mapSh, src.hi, (uint64_t)rows_total, (uint64_t)a.width, (uint64_t)src.ld, 64, DT_BK) ||
        !make_tensor_map_bf16(&a.mapSl, src.lo, (uint64_t)rows_total, (uint64_t)a.width, (uint64_t)src.ld, 64, DT_BK))
        return rtma_fail(ctx, RTMA_ERR_CUDA, "cuTensorMapEncodeTiled refused the aggregation operands");
    // A block per SM for the hubs, two for the other long rows.  100,000 rows, us a forward pass of 48 / 256 columns.  Hubs by warps from 24 a
    // block on: 2,000 hubs of 280 entries by blocks 82 / 126, by warps 91 / 141; 4,000 102 / 194 and 109 / 185; 8,300 185 / 362 and 155 / 277; 100,000
    // of 70 entries 830 / 1,440 and 229 / 366.  All blocks for the other long rows where these are most of the rows and give the warps of
    // many_blocks more than 28 each: 98,000 of 10 entries 79 / 110 by many_blocks, 74 / 103 by all; 56,000 of 100,000 52 / 69 and 53 / 71 (740,000 of 2 M:
    // 3 to 5 % slower by all); 36,000 of 40,000 with 100 hubs 35 / 46 and 40 / 53.
    const int64_t groups = group_tiles(g, 32);
    const LongRows& lr = order.long_rows;
    const unsigned sms = (unsigned)ctx->sm_count;
    const bool hubs_by_warp = lr.hubs > DT_HUBS_PER_BLOCK * (int)sms, many = !lr.listed || hubs_by_warp || (lr.hubs <= 4 * (int)sms && 2 * (int64_t)lr.many > rows_total && lr.many > 28 * 16 * (int)sms);
    const unsigned hub_blocks = hubs_by_warp || lr.hubs == 0 ? 0u : sms, many_blocks = lr.many > 0 || hubs_by_warp ? 2u * sms : 0u;
    const unsigned lgrid = hub_blocks + many_blocks + (unsigned)std::min<int64_t>(ceil_div(groups, 8), (int64_t)sms * 12);
    {
        KernelScope ks(ctx, kclass, s);
#define RTMA_OUTSIDE(T, L, MANY)                                                                                              \
    launch_kernel(spmm_outside_kernel<T, L, MANY>, lgrid, 256, 0, s, g, rowptr_out, col_out, inv_deg, dense, order.left_cnt, order.left_col, \
                  lr, hub_blocks, many_blocks, src, out, a.width, groups)
#define RTMA_OUTSIDE_BY_WIDTH(T, MANY)                  \
    do {                                                \
        if (a.width <= 64) RTMA_OUTSIDE(T, 8, MANY);    \
        else RTMA_OUTSIDE(T, 32, MANY);                 \
    } while (0)
        if (transposed && many) RTMA_OUTSIDE_BY_WIDTH(true, true);
        else if (transposed) RTMA_OUTSIDE_BY_WIDTH(true, false);
        else if (many) RTMA_OUTSIDE_BY_WIDTH(false, true);
        else RTMA_OUTSIDE_BY_WIDTH(false, false);
#undef RTMA_OUTSIDE_BY_WIDTH
#undef RTMA_OUTSIDE
    }
    RTMA_LAUNCH_CHECK(ctx);
    const unsigned grid = (unsigned)std::min<int64_t>(row_tiles * a.col_tiles, ctx->sm_count);
    const size_t smem = a.stages * stage_bytes + fixed;
    {
        KernelScope ks(ctx, kclass, s);
        // transposed with several column tiles: 2 M rows of 512 values 3,460 us with the windows a tile ahead, 3,330 without; of 64 and 128
        // values on 300,000 rows 97 / 136 and 102 / 139
        if (!transposed) launch_kernel(spmm_dense_kernel<false, true>, grid, DT_THREADS, smem, s, a);
        else if (a.col_tiles == 1) launch_kernel(spmm_dense_kernel<true, true>, grid, DT_THREADS, smem, s, a);
        else launch_kernel(spmm_dense_kernel<true, false>, grid, DT_THREADS, smem, s, a);
    }
    RTMA_LAUNCH_CHECK(ctx);
    return RTMA_OK;
}
