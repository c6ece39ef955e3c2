// The input gradient of a last layer with very few classes, on the plain ALUs:
//   dH[r][j] = sum_c dZ[r][c] Ws[j][c] + Q[r][c] Wn[j][c],   Q = Abar^T dZ,
// gated by the sign of the layer's input H (the ReLU of the layer below) and written over it as
// split planes.  With two classes that is four multiply-adds per output: the tensor cores would
// spend their time on zero padding (K = 2 x 2 padded to 2 x 64), while this kernel only streams
// the gate in and the gradient out.  It was bound by instructions and by the loads that a warp had in flight:
// with the coefficients two to a word (instead of a 16-byte piece per plane, eight values for two), up to eight rows
// in flight instead of four, multiply-adds two at a time and the gate as a mask on the packed planes, 5 M rows of 256
// columns and two classes take 1,285 us instead of 1,560 (6.2 TB/s), three 1,372 instead of 1,500, four 1,929 instead of 2,530.
#include "train.cuh"

namespace {

constexpr int DN_THREADS = 256;
constexpr int DN_TILE_ROWS = 512;  // rows of one part handled by a block: 64 per warp
// Rows a warp has in flight: as many as the weights (eight registers a product) leave room for at two blocks per SM.  5 M rows of 256
// columns, us: six products with 4 rows 1,458, 5 rows 1,372, 8 rows 2,315 (they spill; alone on an SM 1,637); eight products with 3
// rows 1,929, 4 rows 1,909 (they spill), 8 rows 3,320.  With one load per plane for the two words of a row: before, 4 rows 1,513.
template <int PRODUCTS>
constexpr int DN_ROWS = PRODUCTS <= 4 ? 8 : PRODUCTS <= 6 ? 5 : 3;

// The c-th of the values whose planes lie two to a word
template <int N>
__device__ __forceinline__ float half_of(const uint32_t (&hi)[N], const uint32_t (&lo)[N], const int c) {
    return c & 1 ? __uint_as_float(hi[c / 2] & 0xFFFF0000u) + __uint_as_float(lo[c / 2] & 0xFFFF0000u)
                 : __uint_as_float(hi[c / 2] << 16) + __uint_as_float(lo[c / 2] << 16);
}

// A row's first values, two to a word, with one load
__device__ __forceinline__ void load_words(const __nv_bfloat16* p, uint32_t (&w)[1]) { w[0] = *reinterpret_cast<const uint32_t*>(p); }
__device__ __forceinline__ void load_words(const __nv_bfloat16* p, uint32_t (&w)[2]) {
    const uint2 v = *reinterpret_cast<const uint2*>(p);
    w[0] = v.x;
    w[1] = v.y;
}

// NSRC weight matrices (2: Ws and Wn; 1: W alone, multiplying Q), C classes: NSRC * C products per output
template <int NSRC, int C>
__global__ void __launch_bounds__(DN_THREADS, 2)
dgrad_narrow_kernel(const __grid_constant__ GroupDesc g, const LayerShape ls, const float* __restrict__ params,
                    const Planes dZ, const Planes Q, const Planes H, const int gate) {
    wait_for_kernel_before();
    constexpr int BATCH = DN_ROWS<NSRC * C>;
    int k, r0;
    if (!locate_tile(g, DN_TILE_ROWS, blockIdx.x, &k, &r0)) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int d_in = ls.d_in;
    const float* W = params + (int64_t)g.part[k] * ls.P + ls.param_offset;  // Ws [d_in][C], then Wn [d_in][C]
    const int rows_here = min(DN_TILE_ROWS, g.rows[k] - r0);
    constexpr int RPW = DN_TILE_ROWS / (DN_THREADS / 32);
    const int q_begin = warp * RPW, q_end = min(rows_here, q_begin + RPW);
    for (int c0 = lane * 8; c0 < (int)H.ld; c0 += 256) {
        // the lane's eight columns j = c0 .. c0+7: their weights for every product
        float w[NSRC * C][8];
#pragma unroll
        for (int e = 0; e < 8; ++e)
#pragma unroll
            for (int m = 0; m < NSRC; ++m)
#pragma unroll
                for (int c = 0; c < C; ++c)
                    w[m * C + c][e] = c0 + e < d_in ? __ldg(W + (int64_t)(m * d_in + c0 + e) * C + c) : 0.f;
        for (int q0 = q_begin; q0 < q_end; q0 += BATCH) {
            // the rows' coefficients: dZ for the first weight matrix, Q for the second (or only) one; two to a word
            constexpr int CW = (C + 1) / 2;
            uint32_t zh[BATCH][CW], zl[BATCH][CW], qh[BATCH][CW], ql[BATCH][CW];
            uint4 gw[BATCH];
#pragma unroll
            for (int b = 0; b < BATCH; ++b) {
                const int64_t r = g.row_ws[k] + r0 + min(q0 + b, q_end - 1);
                if (NSRC == 2) {
                    load_words(dZ.hi + r * dZ.ld, zh[b]);
                    load_words(dZ.lo + r * dZ.ld, zl[b]);
                }
                load_words(Q.hi + r * Q.ld, qh[b]);
                load_words(Q.lo + r * Q.ld, ql[b]);
                gw[b] = gate ? *reinterpret_cast<const uint4*>(H.hi + r * H.ld + c0) : make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll
            for (int b = 0; b < BATCH; ++b) {
                if (q0 + b >= q_end) break;
                const int64_t r = g.row_ws[k] + r0 + q0 + b;
                Pack8 x;
                x.zero();
#pragma unroll
                for (int e = 0; e < 8; e += 2) {
#pragma unroll
                    for (int c = 0; c < C; ++c) {
                        if (NSRC == 2) fma_pair(x.v[e], x.v[e + 1], half_of(zh[b], zl[b], c), w[c][e], w[c][e + 1]);
                        fma_pair(x.v[e], x.v[e + 1], half_of(qh[b], ql[b], c), w[(NSRC - 1) * C + c][e], w[(NSRC - 1) * C + c][e + 1]);
                    }
                }
                uint32_t hw[4], lw[4];
                const uint32_t g4[4] = {gw[b].x, gw[b].y, gw[b].z, gw[b].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    split_pair(x.v[2 * e], x.v[2 * e + 1], hw[e], lw[e]);
                    if (gate) {
                        const uint32_t pass = positive_halves(g4[e]);
                        hw[e] &= pass;
                        lw[e] &= pass;
                    }
                }
                const uint4 h = make_uint4(hw[0], hw[1], hw[2], hw[3]), l = make_uint4(lw[0], lw[1], lw[2], lw[3]);
                *reinterpret_cast<uint4*>(H.hi + r * H.ld + c0) = h;
                *reinterpret_cast<uint4*>(H.lo + r * H.ld + c0) = l;
            }
        }
    }
}

}  // namespace

bool dgrad_narrow_applies(const LayerShape& ls) { return ls.d_out <= 4; }

int32_t launch_dgrad_narrow(rtma_ctx* ctx, const GroupDesc& g, LayerShape ls, const float* params, Planes dZ, Planes Q,
                            Planes H, bool gate, cudaStream_t s) {
    const int64_t tiles = group_tiles(g, DN_TILE_ROWS);
    if (tiles == 0) return RTMA_OK;
    const int gt = gate ? 1 : 0;
    {
        KernelScope ks(ctx, KC_GEMM_DGRAD, s);
#define RTMA_DN(NS, CC) launch_kernel(dgrad_narrow_kernel<NS, CC>, (unsigned)tiles, DN_THREADS, 0, s, g, ls, params, dZ, Q, H, gt)
        const int key = ls.nsrc * 10 + ls.d_out;
        switch (key) {
            case 11: RTMA_DN(1, 1); break;
            case 12: RTMA_DN(1, 2); break;
            case 13: RTMA_DN(1, 3); break;
            case 14: RTMA_DN(1, 4); break;
            case 21: RTMA_DN(2, 1); break;
            case 22: RTMA_DN(2, 2); break;
            case 23: RTMA_DN(2, 3); break;
            case 24: RTMA_DN(2, 4); break;
            default: return rtma_fail(ctx, RTMA_ERR_UNSUPPORTED, "internal: narrow dgrad with %d classes", ls.d_out);
        }
#undef RTMA_DN
    }
    RTMA_LAUNCH_CHECK(ctx);
    return RTMA_OK;
}
