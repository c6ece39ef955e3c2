// One hop of the GraphSAGE neighbour sampler that shrinks the message-flow graph of a mini-batch
// (Sec. 4.1 "Mini-batch and Negative Sampling"), on one part's induced subgraph.
//
// A frontier node with at most `fanout` entries keeps them all; otherwise it keeps the `fanout`
// entries with the smallest 64-bit keys, key = S(S(seed ^ ((hop + 1) << 48)) ^ ((v << 32) | pos)),
// S = one SplitMix64 step (equal keys: the smaller position first): a uniform sample without
// replacement that depends on nothing but (seed, hop, node, position), hence the same on any machine.
//
//   1. count      one thread per frontier node: min(degree, fanout); marks the node in the member flags
//   2. scan       block_rowptr = exclusive scan of the counts
//   3. select     half a warp per frontier node: candidates below a bound that the fanout-th smallest key does not
//                 exceed, the kept ones by their rank among the candidates, in row order; their end points
//                 are written to block_col and marked as members
//   4. scan       positions of the members = exclusive scan of the flags; next_size = its total
//   5. emit       next_frontier[position] = node;  block_col[e] = position of its node
// No atomics on data, no waits: the result is unique.
#include <algorithm>
#include <cmath>

#include "common.cuh"

RTMA_BOUNDS_TU()

namespace {

__device__ __forceinline__ uint64_t mix_step(uint64_t x) {  // one step of the SplitMix64 generator
    uint64_t z = x + 0x9E3779B97F4A7C15ULL;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

__global__ void __launch_bounds__(256)
sample_count_kernel(const int64_t* __restrict__ rowptr, int64_t n, int64_t frontier_size, const int32_t* __restrict__ frontier,
                    int32_t fanout, int32_t* __restrict__ counts, int32_t* __restrict__ member) {
    wait_for_kernel_before();
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= frontier_size) return;
    const int32_t v = frontier[i];
    if (!rtma_index_ok(v, n, 7)) {
        counts[i] = 0;
        return;
    }
    const int64_t deg = rowptr[v + 1] - rowptr[v];
    counts[i] = (int32_t)(deg < fanout ? deg : fanout);
    member[v] = 1;
}

constexpr int SEL_LANES = 16;   // lanes that work on one frontier node
constexpr int SEL_NODES = 256 / SEL_LANES;  // nodes of a block
constexpr int SEL_CAND = 128;   // candidates a node may have

// The kept entries of one node by the whole warp, whatever its degree and the fan-out: the fanout-th smallest key bit by
// bit (rounds of counting the keys that share the prefix found so far and have a 0 in the next bit), then a pass that
// writes the entries below the prefix and the first few that share it, in row order.  OFTEN: the rounds end as soon as no
// more keys share the prefix than are still to be kept, after about log2 of the degree of them; where one row in a million comes
// here the count is left out, it costs the kernel four registers and 2 % of the time of small fan-outs.
template <bool OFTEN>
__device__ void select_bit_by_bit(const int32_t* __restrict__ col, int64_t n, int64_t begin, int64_t deg, uint64_t vkey, int32_t fanout,
                                  uint64_t base, int64_t out, int32_t* __restrict__ block_col, int32_t* __restrict__ member) {
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    uint64_t prefix = 0;
    int64_t want = fanout, left = deg;  // keys to be kept among those that share the prefix, and how many share it
    int bit = 63;
    for (; bit >= 0 && (!OFTEN || left > want); --bit) {
        const uint64_t above = bit == 63 ? 0ULL : ~0ULL << (bit + 1);
        int64_t zeros = 0;
        for (int64_t q = lane; q < deg; q += 32) {
            const uint64_t key = mix_step(base ^ (vkey | (uint64_t)q));
            zeros += ((key & above) == prefix && !((key >> bit) & 1ULL)) ? 1 : 0;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) zeros += __shfl_xor_sync(0xffffffffu, zeros, o);
        if (want > zeros) {  // the key has a 1 here; the `zeros` keys with a 0 are all smaller
            want -= zeros;
            left -= zeros;
            prefix |= 1ULL << bit;
        } else {
            left = zeros;
        }
    }
    const uint64_t mask = OFTEN && bit >= 0 ? ~0ULL << (bit + 1) : ~0ULL;  // the bits that were found (at least one: left > want at first)
    int64_t ties_seen = 0;  // entries that share the prefix: the first `want` in row order are kept (all, or those with equal keys)
    for (int64_t q0 = 0; q0 < deg; q0 += 32) {
        const int64_t q = q0 + lane;
        const uint64_t key = mix_step(base ^ (vkey | (uint64_t)q)) & mask;
        const bool tie = q < deg && key == prefix;
        bool keep = q < deg && key < prefix;
        const unsigned tie_votes = __ballot_sync(0xffffffffu, tie);
        if (tie && ties_seen + __popc(tie_votes & below) < want) keep = true;
        ties_seen += __popc(tie_votes);
        const int32_t u = keep ? col[begin + q] : 0;
        if (keep && !rtma_index_ok(u, n, 5)) keep = false;
        const unsigned votes = __ballot_sync(0xffffffffu, keep);
        if (keep) {
            block_col[out + __popc(votes & below)] = u;
            member[u] = 1;
        }
        out += __popc(votes);
    }
}

// Half a warp per frontier node (two nodes of 30 entries fill a warp's lanes).  The keys are uniform 64-bit numbers, so the
// fanout-th smallest of deg lies near fanout / deg of their range: one pass over the row hashes every entry once and collects
// those below a bound at which `tight` of them are expected, in row order, in shared memory; a candidate is kept when
// fewer than `fanout` candidates are smaller.  Only kept entries' columns are read.  Bound by instruction issue (the hash,
// 25 instructions per entry, and the ranking, candidates squared), hence few candidates: tight = fanout + 2.7 sqrt(fanout) + 1,
// which leaves one row in a hundred short; its half warp goes through the row once more with a bound for wide = fanout +
// 6 sqrt(fanout) + 16.  Neither expects more than half way between the fan-out and the candidates' room: too few or too
// many candidates at the wide bound come once in 10^6 rows up to a fan-out of 35, in 20,000 at 50, in 1,000 at 64, in 60 at 80
// and in 8 at SEL_FANOUT; such rows, and all that are cut to larger fan-outs, are done bit by bit.
// Bound and ranking look at the upper 32 bits of the keys; where these do not single out `fanout` candidates (equal ones at
// the cut) the row is done bit by bit too.
// Three hops (fan-outs 15, 10, 5) from 8,192 of 800,000 nodes, the whole call: with the wide bound alone and whole keys ranked
// 848 us, with two waits for sizes a hop instead of one; now 584.
constexpr int SEL_FANOUT = 96;  // largest fan-out for which candidates are collected
constexpr int SEL_RARE = 35;    // largest fan-out at which a row without the right number of them is one in a million
template <bool OFTEN>
__global__ void __launch_bounds__(256)
sample_select_kernel(const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col, int64_t n, int64_t frontier_size,
                     const int32_t* __restrict__ frontier, int32_t fanout, float tight, float wide, uint64_t base,
                     const int64_t* __restrict__ block_rowptr, int32_t* __restrict__ block_col, int32_t* __restrict__ member) {
    wait_for_kernel_before();
    __shared__ __align__(16) uint32_t cand_key[SEL_NODES][SEL_CAND];
    __shared__ int32_t cand_pos[SEL_NODES][SEL_CAND];
    const int lane = threadIdx.x & 31, sub = threadIdx.x / SEL_LANES, sl = threadIdx.x % SEL_LANES;
    const int shift = lane & 16;                       // first lane of this node's half
    const unsigned below = (1u << sl) - 1u;
    const int64_t i = (int64_t)blockIdx.x * SEL_NODES + sub;
    int32_t v = i < frontier_size ? frontier[i] : -1;
    if (v >= 0 && !rtma_index_ok(v, n, 7)) v = -1;
    const int64_t begin = v >= 0 ? rowptr[v] : 0, deg = v >= 0 ? rowptr[v + 1] - begin : 0;
    const int64_t out = v >= 0 ? block_rowptr[i] : 0;
    const uint64_t vkey = (uint64_t)(uint32_t)v << 32;
    const bool sel = deg > fanout;

    // short rows: everything is kept
    if (!sel) {
        for (int64_t q = sl; q < deg; q += SEL_LANES) {
            const int32_t u = col[begin + q];
            const bool good = rtma_index_ok(u, n, 5);
            block_col[out + q] = good ? u : 0;  // node id for now; its position in the next frontier later
            if (good) member[u] = 1;            // every writer stores the same value
        }
    }
    // the others: candidates (both halves of the warp go through the longer row's rounds)
    const bool collect = sel && fanout <= SEL_FANOUT && deg < (int64_t(1) << 31);  // positions are 32-bit
    int64_t count = 0;
    for (int attempt = 0; attempt < 2; ++attempt) {
        const bool mine = collect && (attempt == 0 || count < fanout);
        if (attempt == 1 && (!__any_sync(0xffffffffu, mine) || wide <= tight)) break;
        __syncwarp();  // the second attempt overwrites what other lanes wrote in the first
        const float share = (attempt == 0 ? tight : wide) / (float)deg;
        const uint32_t bound = share >= 0.999f ? 0xFFFFFFFFu : (uint32_t)(share * 4294967296.f);
        const int rounds = mine ? (int)((deg + SEL_LANES - 1) / SEL_LANES) : 0;
        const int most = max(rounds, __shfl_xor_sync(0xffffffffu, rounds, 16));
        if (mine) count = 0;
        for (int t = 0; t < most; ++t) {
            const uint32_t q = (uint32_t)t * SEL_LANES + sl;
            const uint32_t key = (uint32_t)(mix_step(base ^ (vkey | (uint64_t)q)) >> 32);
            const bool cand = mine && q < (uint32_t)deg && key <= bound;
            const unsigned votes = (__ballot_sync(0xffffffffu, cand) >> shift) & 0xFFFFu;
            const int64_t at = count + __popc(votes & below);
            if (cand && at < SEL_CAND) {
                cand_key[sub][at] = key;
                cand_pos[sub][at] = (int32_t)q;
            }
            count += __popc(votes);
        }
    }
    bool ok = collect && count >= fanout && count <= SEL_CAND;
    const int m = ok ? (int)count : 0;
    if (sl < 3 && m + sl < (m + 3) / 4 * 4) cand_key[sub][m + sl] = 0xFFFFFFFFu;  // up to whole vectors: never smaller than a key
    __syncwarp();
    unsigned keep_mask = 0;  // bit t: the lane's candidate 16 t + sl is kept
    int kept = 0;
    for (int c0 = 0; c0 < m; c0 += SEL_LANES) {  // nothing crosses the halves
        const int c = c0 + sl;
        const uint32_t key = c < m ? cand_key[sub][c] : 0xFFFFFFFFu;
        int rank = 0;  // candidates with a smaller key
        for (int j = 0; j < m; j += 4) {
            const uint4 other = *reinterpret_cast<const uint4*>(&cand_key[sub][j]);
            rank += (other.x < key) + (other.y < key) + (other.z < key) + (other.w < key);
        }
        const bool keep = c < m && rank < fanout;
        keep_mask |= keep ? 1u << (c0 / SEL_LANES) : 0u;
        kept += __popc(__ballot_sync(0xFFFFu << shift, keep));
    }
    __syncwarp();
    ok = ok && kept == fanout;  // more of them: candidates that share the upper half of the last kept key
    const int m_write = ok ? m : 0, m_most = max(m_write, __shfl_xor_sync(0xffffffffu, m_write, 16));
    int64_t at = out;
    for (int c0 = 0; c0 < m_most; c0 += SEL_LANES) {
        bool keep = c0 < m_write && (keep_mask >> (c0 / SEL_LANES) & 1u);
        const int32_t u = keep ? col[begin + cand_pos[sub][c0 + sl]] : 0;
        if (keep && !rtma_index_ok(u, n, 5)) keep = false;
        const unsigned votes = (__ballot_sync(0xffffffffu, keep) >> shift) & 0xFFFFu;
        if (keep) {
            block_col[at + __popc(votes & below)] = u;
            member[u] = 1;
        }
        at += __popc(votes);
    }
    // fan-outs past the candidates' room, and the rare row whose candidates were too few or too many
    for (unsigned rest = __ballot_sync(0xffffffffu, sel && !ok && sl == 0); rest; rest &= rest - 1) {
        const int from = __ffs(rest) - 1;
        const int64_t b = __shfl_sync(0xffffffffu, begin, from), d = __shfl_sync(0xffffffffu, deg, from), o = __shfl_sync(0xffffffffu, out, from);
        select_bit_by_bit<OFTEN>(col, n, b, d, __shfl_sync(0xffffffffu, vkey, from), fanout, base, o, block_col, member);
    }
}

__global__ void __launch_bounds__(256)
sample_emit_frontier_kernel(int64_t n, const int32_t* __restrict__ member, const int64_t* __restrict__ position,
                            int32_t* __restrict__ next_frontier, int64_t* __restrict__ next_size) {
    wait_for_kernel_before();
    const int64_t v = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (v < n && member[v]) next_frontier[position[v]] = (int32_t)v;
    if (v == 0) *next_size = position[n];
}

__global__ void __launch_bounds__(256)
sample_relabel_kernel(const int64_t* __restrict__ block_rowptr, int64_t frontier_size, const int64_t* __restrict__ position,
                      int32_t* __restrict__ block_col) {
    wait_for_kernel_before();
    const int64_t entries = block_rowptr[frontier_size];
    for (int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x; e < entries; e += (int64_t)gridDim.x * 256)
        block_col[e] = (int32_t)position[block_col[e]];
}

}  // namespace

extern "C" int32_t rtma_sample_hop(rtma_ctx* ctx, int64_t n, const int64_t* rowptr, const int32_t* col, int64_t frontier_size,
                                   const int32_t* frontier, int32_t fanout, uint64_t seed, int32_t hop,
                                   int64_t* block_rowptr, int32_t* block_col, int32_t* next_frontier, int64_t* next_size,
                                   void* stream_) {
    if (!ctx) return RTMA_ERR_INVALID_ARG;
    if (n < 0 || n >= (int64_t(1) << 31) || frontier_size < 0 || frontier_size > n)
        return rtma_fail(ctx, RTMA_ERR_INVALID_ARG, "rtma_sample_hop: n=%lld, frontier_size=%lld", (long long)n, (long long)frontier_size);
    if (fanout < 1 || hop < 0 || hop >= 65535) return rtma_fail(ctx, RTMA_ERR_INVALID_ARG, "rtma_sample_hop: fanout=%d hop=%d", fanout, hop);
    if (!block_rowptr || !next_size || (n > 0 && (!rowptr || !next_frontier)) || (frontier_size > 0 && (!frontier || !block_col)))
        return rtma_fail(ctx, RTMA_ERR_INVALID_ARG, "rtma_sample_hop: null pointer");
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    RTMA_CUDA(ctx, cudaSetDevice(ctx->device));
    RTMA_TRY(order_after_training(ctx, stream));
    const int64_t scan_n = n > frontier_size ? n : frontier_size;
    const size_t need = ArenaCursor::granule(sizeof(int32_t) * (frontier_size + 1)) + ArenaCursor::granule(sizeof(int32_t) * (n + 1)) +
                        ArenaCursor::granule(sizeof(int64_t) * (n + 2)) + ArenaCursor::granule(sizeof(int64_t) * scan_scratch_elems(scan_n));
    RTMA_TRY(rtma_reserve(ctx, need));
    ArenaCursor cur(ctx->arena);
    int32_t* counts = cur.take<int32_t>(frontier_size + 1);
    int32_t* member = cur.take<int32_t>(n + 1);
    int64_t* position = cur.take<int64_t>(n + 2);
    int64_t* scratch = cur.take<int64_t>(scan_scratch_elems(scan_n));
    RTMA_CUDA(ctx, cudaMemsetAsync(member, 0, sizeof(int32_t) * (n + 1), stream));
    if (frontier_size > 0) {
        KernelScope ks(ctx, KC_LINK, stream);
        launch_kernel(sample_count_kernel, (unsigned)ceil_div(frontier_size, 256), 256, 0, stream, rowptr, n, frontier_size, frontier, fanout, counts, member);
    }
    RTMA_LAUNCH_CHECK(ctx);
    RTMA_TRY(exclusive_scan_i32_to_i64(ctx, counts, frontier_size, block_rowptr, scratch, stream));
    if (frontier_size > 0) {
        const uint64_t base_in = seed ^ ((uint64_t)(hop + 1) << 48);
        // the hop's key stream: one SplitMix64 step of the seed and the hop, on the host (same arithmetic)
        uint64_t z = base_in + 0x9E3779B97F4A7C15ULL;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
        const uint64_t base = z ^ (z >> 31);
        KernelScope ks(ctx, KC_LINK, stream);
        // candidates per row (see the kernel)
        const double root = std::sqrt((double)fanout), half_way = 0.5 * ((double)fanout + SEL_CAND);
        const float tight = (float)std::min(fanout + 2.7 * root + 1.0, half_way), wide = (float)std::min(fanout + 6.0 * root + 16.0, half_way);
        launch_kernel(fanout > SEL_RARE ? sample_select_kernel<true> : sample_select_kernel<false>, (unsigned)ceil_div(frontier_size, SEL_NODES), 256, 0, stream,
            rowptr, col, n, frontier_size, frontier, fanout, tight, wide, base, block_rowptr, block_col, member);
    }
    RTMA_LAUNCH_CHECK(ctx);
    RTMA_TRY(exclusive_scan_i32_to_i64(ctx, member, n, position, scratch, stream));
    {
        KernelScope ks(ctx, KC_LINK, stream);
        launch_kernel(sample_emit_frontier_kernel, (unsigned)ceil_div(n > 0 ? n : 1, 256), 256, 0, stream, n, member, position, next_frontier, next_size);
    }
    RTMA_LAUNCH_CHECK(ctx);
    if (frontier_size > 0) {
        const int64_t bound = frontier_size * (int64_t)(fanout < 4096 ? fanout : 4096);  // kept entries, roughly: sizes the grid only
        KernelScope ks(ctx, KC_LINK, stream);
        launch_kernel(sample_relabel_kernel, (unsigned)std::min<int64_t>(ceil_div(bound, 256), 148 * 32), 256, 0, stream, block_rowptr, frontier_size,
                                                                                                        position, block_col);
    }
    RTMA_LAUNCH_CHECK(ctx);
    return RTMA_OK;
}
