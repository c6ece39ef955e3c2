// Layer Normalization before the activation and PReLU (the paper's encoders, Sec. 4.1 "GNN
// Encoders"), forward and backward, on split bf16 planes:
//   U = gamma * (Z - mean) / sqrt(var + eps) + beta over the row's features (biased variance,
//       eps = 1e-5), or U = Z without normalisation;
//   H = U if U > 0 else a * U, one learnable slope a per layer (a = 0: ReLU).
// One warp per row, the row held in registers (8 values per 16-byte piece, up to four pieces per
// lane); 64-row tiles.  The backward pass recomputes U from Z and the saved (mean, 1/std),
// writes dZ over Z, and leaves per-tile sums for d gamma, d beta and d a, which a second kernel
// adds up in a fixed order and applies (W <- W - lr * grad, Algorithm 2).
#include "train.cuh"

namespace {

constexpr int POST_THREADS = 128;
constexpr int POST_WARPS = POST_THREADS / 32;
constexpr int POST_TILE_ROWS = 64;
constexpr int POST_ROWS_PER_WARP = POST_TILE_ROWS / POST_WARPS;
constexpr int POST_MAX_WIDTH = 1024;
constexpr float LN_EPS = 1e-5f;

struct PostArgs {
    LayerShape ls;          // the layer whose output is normalised / activated (width = ls.d_out)
    const float* params;    // all replicas
    Planes Z, H;            // forward: Z in, H out.  backward: H = dH in, Z in and dZ out
    float2* stats;          // [scratch row] (mean, 1/std); unused without normalisation
    float* partial;         // backward: [tile][2 * d + 1]
};

// Both kernels are bound by instruction issue, not by the bytes they stream: two values per instruction (f32x2) wherever
// the arithmetic allows, and two rows side by side so that one row's shuffles overlap the other's arithmetic.
// 200,000 rows of 256 values (8 parts): forward 93 -> 80 us, backward 188 -> 109 us (614 MB, 86 % of the copy rate).
typedef unsigned long long f2;  // two fp32 numbers, the lower half first
__device__ __forceinline__ f2 pack2(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(f2 x, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x)); }
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}
__device__ __forceinline__ float halves_sum(f2 x) {
    float a, b;
    unpack2(x, a, b);
    return a + b;
}

// the lane's eight values of piece c of row r (zeros past the width)
__device__ __forceinline__ void load_piece(const Planes m, int64_t r, int col, int d, uint4& h, uint4& l) {
    h = l = make_uint4(0u, 0u, 0u, 0u);
    if (col < d) {
        h = *reinterpret_cast<const uint4*>(m.hi + r * m.ld + col);
        l = *reinterpret_cast<const uint4*>(m.lo + r * m.ld + col);
    }
}
__device__ __forceinline__ void join_piece(const uint4 h, const uint4 l, f2 (&x)[4]) {
    const uint32_t hw[4] = {h.x, h.y, h.z, h.w}, lw[4] = {l.x, l.y, l.z, l.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
        x[i] = pack2(add_f32_bf16(__uint_as_float(hw[i] << 16), (unsigned short)(lw[i] & 0xFFFFu)),
                     add_f32_bf16(__uint_as_float(hw[i] & 0xFFFF0000u), (unsigned short)(lw[i] >> 16)));
}
// keep: all ones in the halves of the 32-bit words that lie inside the width
__device__ __forceinline__ void store_piece(const Planes m, int64_t r, int col, int d, const f2 (&x)[4], const uint32_t (&keep)[4]) {
    if (col >= d) return;
    uint32_t h[4], l[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float x0, x1;
        unpack2(x[i], x0, x1);
        split_pair(x0, x1, h[i], l[i]);
        h[i] &= keep[i];
        l[i] &= keep[i];
    }
    *reinterpret_cast<uint4*>(m.hi + r * m.ld + col) = make_uint4(h[0], h[1], h[2], h[3]);
    *reinterpret_cast<uint4*>(m.lo + r * m.ld + col) = make_uint4(l[0], l[1], l[2], l[3]);
}
__device__ __forceinline__ void width_mask(int col, int d, uint32_t (&keep)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
        keep[i] = (col + 2 * i < d ? 0x0000FFFFu : 0u) | (col + 2 * i + 1 < d ? 0xFFFF0000u : 0u);
}

// RB rows at a time per warp
template <int NP, bool NORM>
__global__ void __launch_bounds__(POST_THREADS)
post_forward_kernel(const __grid_constant__ GroupDesc g, const PostArgs a) {
    wait_for_kernel_before();
    constexpr int RB = NP == 1 ? 2 : 1;
    int k, r0;
    if (!locate_tile(g, POST_TILE_ROWS, blockIdx.x, &k, &r0)) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int d = a.ls.d_out;
    const float* P = a.params + (int64_t)g.part[k] * a.ls.P;
    const float slope = a.ls.slope_offset >= 0 ? P[a.ls.slope_offset] : 0.f;
    const f2 slope2 = pack2(slope, slope);
    f2 gam[NP][4], bet[NP][4];
    uint32_t keep[NP][4];
#pragma unroll
    for (int c = 0; c < NP; ++c) {
        const int col = (c * 32 + lane) * 8;
        width_mask(col, d, keep[c]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int j = col + 2 * i;
            gam[c][i] = NORM ? pack2(j < d ? P[a.ls.gamma_offset + j] : 1.f, j + 1 < d ? P[a.ls.gamma_offset + j + 1] : 1.f) : 0ull;
            bet[c][i] = NORM ? pack2(j < d ? P[a.ls.beta_offset + j] : 0.f, j + 1 < d ? P[a.ls.beta_offset + j + 1] : 0.f) : 0ull;
        }
    }
    const int n_p = g.rows[k];
    const int i_end = min(n_p, r0 + (warp + 1) * POST_ROWS_PER_WARP);
    for (int i0 = r0 + warp * POST_ROWS_PER_WARP; i0 < i_end; i0 += RB) {
        f2 x[RB][NP][4];
#pragma unroll
        for (int b = 0; b < RB; ++b) {
            const int64_t r = g.row_ws[k] + min(i0 + b, i_end - 1);
#pragma unroll
            for (int c = 0; c < NP; ++c) {
                uint4 h, l;
                load_piece(a.Z, r, (c * 32 + lane) * 8, d, h, l);
                join_piece(h, l, x[b][c]);
            }
        }
        float mean[RB], rstd[RB];
        if (NORM) {
            float s[RB], v[RB];
#pragma unroll
            for (int b = 0; b < RB; ++b) {
                f2 s2 = 0ull;
#pragma unroll
                for (int c = 0; c < NP; ++c)
#pragma unroll
                    for (int i = 0; i < 4; ++i) s2 = add2(s2, x[b][c][i]);  // padding columns hold zeros
                s[b] = halves_sum(s2);
            }
#pragma unroll
            for (int b = 0; b < RB; ++b) mean[b] = warp_sum(s[b]) / (float)d;
#pragma unroll
            for (int b = 0; b < RB; ++b) {
                const f2 minus = pack2(-mean[b], -mean[b]);
                f2 v2 = 0ull;
#pragma unroll
                for (int c = 0; c < NP; ++c)
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        x[b][c][i] = add2(x[b][c][i], minus);
                        f2 t = x[b][c][i];
                        if (keep[c][i] != 0xFFFFFFFFu) {  // columns past the width do not count
                            float t0, t1;
                            unpack2(t, t0, t1);
                            t = pack2(keep[c][i] & 0xFFFFu ? t0 : 0.f, keep[c][i] >> 16 ? t1 : 0.f);
                        }
                        v2 = fma2(t, t, v2);
                    }
                v[b] = halves_sum(v2);
            }
#pragma unroll
            for (int b = 0; b < RB; ++b) {
                rstd[b] = rsqrtf(warp_sum(v[b]) / (float)d + LN_EPS);
                if (lane == 0 && i0 + b < i_end) a.stats[g.row_ws[k] + i0 + b] = make_float2(mean[b], rstd[b]);
            }
        }
#pragma unroll
        for (int b = 0; b < RB; ++b) {
            if (i0 + b >= i_end) break;
            const f2 rstd2 = NORM ? pack2(rstd[b], rstd[b]) : 0ull;
#pragma unroll
            for (int c = 0; c < NP; ++c) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    f2 u = x[b][c][i];
                    if (NORM) u = fma2(gam[c][i], mul2(u, rstd2), bet[c][i]);
                    float u0, u1, n0, n1;
                    unpack2(u, u0, u1);
                    unpack2(mul2(u, slope2), n0, n1);
                    x[b][c][i] = pack2(u0 > 0.f ? u0 : n0, u1 > 0.f ? u1 : n1);
                }
                store_piece(a.H, g.row_ws[k] + i0 + b, (c * 32 + lane) * 8, d, x[b][c], keep[c]);
            }
        }
    }
}

template <int NP, bool NORM>
__global__ void __launch_bounds__(POST_THREADS)
post_backward_kernel(const __grid_constant__ GroupDesc g, const PostArgs a) {
    wait_for_kernel_before();
    constexpr int RB = NP == 1 ? 2 : 1;
    __shared__ float red[POST_WARPS][2 * NP * 256 + 1];
    int k, r0;
    if (!locate_tile(g, POST_TILE_ROWS, blockIdx.x, &k, &r0)) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int d = a.ls.d_out;
    const float* P = a.params + (int64_t)g.part[k] * a.ls.P;
    const float slope = a.ls.slope_offset >= 0 ? P[a.ls.slope_offset] : 0.f;
    const f2 slope2 = pack2(slope, slope);
    f2 gam[NP][4], bet[NP][4], dgam[NP][4], dbet[NP][4], dslope = 0ull;
    uint32_t keep[NP][4];
#pragma unroll
    for (int c = 0; c < NP; ++c) {
        const int col = (c * 32 + lane) * 8;
        width_mask(col, d, keep[c]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int j = col + 2 * i;
            gam[c][i] = NORM ? pack2(j < d ? P[a.ls.gamma_offset + j] : 1.f, j + 1 < d ? P[a.ls.gamma_offset + j + 1] : 1.f) : 0ull;
            bet[c][i] = NORM ? pack2(j < d ? P[a.ls.beta_offset + j] : 0.f, j + 1 < d ? P[a.ls.beta_offset + j + 1] : 0.f) : 0ull;
            dgam[c][i] = dbet[c][i] = 0ull;
        }
    }
    const int n_p = g.rows[k];
    const int i_end = min(n_p, r0 + (warp + 1) * POST_ROWS_PER_WARP);
    for (int i0 = r0 + warp * POST_ROWS_PER_WARP; i0 < i_end; i0 += RB) {
        uint4 zh[RB][NP], zl[RB][NP], hh[RB][NP], hl[RB][NP];
        float2 st[RB];
#pragma unroll
        for (int b = 0; b < RB; ++b) {
            const bool row_ok = i0 + b < i_end;  // past the warp's rows: zeros, which add nothing
            const int64_t r = g.row_ws[k] + i0 + b;
#pragma unroll
            for (int c = 0; c < NP; ++c) {
                load_piece(a.Z, r, (c * 32 + lane) * 8, row_ok ? d : 0, zh[b][c], zl[b][c]);
                load_piece(a.H, r, (c * 32 + lane) * 8, row_ok ? d : 0, hh[b][c], hl[b][c]);
            }
            st[b] = NORM && row_ok ? a.stats[r] : make_float2(0.f, 1.f);
        }
        f2 xh[RB][NP][4], dx[RB][NP][4];
        float m1[RB], m2[RB];
#pragma unroll
        for (int b = 0; b < RB; ++b) {
            const f2 minus = pack2(-st[b].x, -st[b].x), rstd2 = pack2(st[b].y, st[b].y);
            f2 s1 = 0ull, s2 = 0ull;
#pragma unroll
            for (int c = 0; c < NP; ++c) {
                f2 gr[4];
                join_piece(zh[b][c], zl[b][c], xh[b][c]);
                join_piece(hh[b][c], hl[b][c], gr);  // the padding columns of dH hold zeros
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (NORM) xh[b][c][i] = mul2(add2(xh[b][c][i], minus), rstd2);
                    const f2 u = NORM ? fma2(gam[c][i], xh[b][c][i], bet[c][i]) : xh[b][c][i];
                    float u0, u1, g0, g1, n0, n1, t0, t1;
                    unpack2(u, u0, u1);
                    unpack2(gr[i], g0, g1);
                    unpack2(mul2(slope2, gr[i]), n0, n1);
                    unpack2(mul2(gr[i], u), t0, t1);
                    const f2 du = pack2(u0 > 0.f ? g0 : n0, u1 > 0.f ? g1 : n1);
                    dslope = add2(dslope, pack2(u0 > 0.f ? 0.f : t0, u1 > 0.f ? 0.f : t1));
                    if (NORM) {
                        dgam[c][i] = fma2(du, xh[b][c][i], dgam[c][i]);
                        dbet[c][i] = add2(dbet[c][i], du);
                        dx[b][c][i] = mul2(du, gam[c][i]);
                        s1 = add2(s1, dx[b][c][i]);
                        s2 = fma2(dx[b][c][i], xh[b][c][i], s2);
                    } else {
                        dx[b][c][i] = du;
                    }
                }
            }
            m1[b] = halves_sum(s1);
            m2[b] = halves_sum(s2);
        }
        if (NORM) {
#pragma unroll
            for (int b = 0; b < RB; ++b) {
                m1[b] = warp_sum(m1[b]) / (float)d;
                m2[b] = warp_sum(m2[b]) / (float)d;
            }
        }
#pragma unroll
        for (int b = 0; b < RB; ++b) {
            if (i0 + b >= i_end) break;
            if (NORM) {
                const f2 minus1 = pack2(-m1[b], -m1[b]), minus2 = pack2(-m2[b], -m2[b]), rstd2 = pack2(st[b].y, st[b].y);
#pragma unroll
                for (int c = 0; c < NP; ++c)
#pragma unroll
                    for (int i = 0; i < 4; ++i) dx[b][c][i] = mul2(rstd2, fma2(xh[b][c][i], minus2, add2(dx[b][c][i], minus1)));
            }
#pragma unroll
            for (int c = 0; c < NP; ++c) store_piece(a.Z, g.row_ws[k] + i0 + b, (c * 32 + lane) * 8, d, dx[b][c], keep[c]);
        }
    }
    // per-tile sums, warps added in a fixed order
    const float dslope_sum = warp_sum(halves_sum(dslope));
#pragma unroll
    for (int c = 0; c < NP; ++c)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int j = (c * 32 + lane) * 8 + 2 * i;
            unpack2(dgam[c][i], red[warp][j], red[warp][j + 1]);
            unpack2(dbet[c][i], red[warp][NP * 256 + j], red[warp][NP * 256 + j + 1]);
        }
    if (lane == 0) red[warp][2 * NP * 256] = dslope_sum;
    __syncthreads();
    float* out = a.partial + (int64_t)blockIdx.x * (2 * d + 1);
    for (int j = threadIdx.x; j < 2 * d + 1; j += POST_THREADS) {
        const int at = j < d ? j : (j < 2 * d ? NP * 256 + (j - d) : 2 * NP * 256);
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < POST_WARPS; ++w) s += red[w][at];
        out[j] = s;
    }
}

// 32 parameters per block; eight threads per parameter each add every eighth tile in order, and
// the eight partial sums are added in a fixed order: the result does not change from run to run.
__global__ void __launch_bounds__(256)
post_reduce_sgd_kernel(const __grid_constant__ GroupDesc g, const LayerShape ls, const float* __restrict__ partial,
                       const float lr, float* __restrict__ params, float* __restrict__ grads_record) {
    wait_for_kernel_before();
    __shared__ float red[8][33];
    const int k = blockIdx.y;
    const int d = ls.d_out;
    const int col = threadIdx.x & 31, lane_t = threadIdx.x >> 5;
    const int j = blockIdx.x * 32 + col;
    int64_t first = 0;
    for (int q = 0; q < k; ++q) first += (g.rows[q] + POST_TILE_ROWS - 1) / POST_TILE_ROWS;
    const int64_t count = (g.rows[k] + POST_TILE_ROWS - 1) / POST_TILE_ROWS;
    float s = 0.f;
    if (j < 2 * d + 1)
#pragma unroll 8
        for (int64_t t = lane_t; t < count; t += 8) s += __ldcs(partial + (first + t) * (2 * d + 1) + j);  // eight loads in flight
    red[lane_t][col] = s;
    __syncthreads();
    if (lane_t != 0 || j >= 2 * d + 1) return;
    int64_t at;
    if (j < d) at = ls.gamma_offset < 0 ? -1 : ls.gamma_offset + j;
    else if (j < 2 * d) at = ls.beta_offset < 0 ? -1 : ls.beta_offset + (j - d);
    else at = ls.slope_offset;
    if (at < 0) return;
    float sum = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) sum += red[w][col];
    at += (int64_t)g.part[k] * ls.P;
    if (grads_record) grads_record[at] = sum;
    params[at] -= lr * sum;
}

}  // namespace

int64_t post_tiles(const GroupDesc& g) { return group_tiles(g, POST_TILE_ROWS); }

#define RTMA_POST_DISPATCH(KERNEL, ls, ...)                                                                   \
    do {                                                                                                      \
        const bool norm = (ls).gamma_offset >= 0;                                                             \
        if ((ls).d_out <= 256) {                                                                              \
            if (norm) launch_kernel(KERNEL<1, true>, (unsigned)tiles, POST_THREADS, 0, s, __VA_ARGS__);                  \
            else launch_kernel(KERNEL<1, false>, (unsigned)tiles, POST_THREADS, 0, s, __VA_ARGS__);                      \
        } else if ((ls).d_out <= 512) {                                                                       \
            if (norm) launch_kernel(KERNEL<2, true>, (unsigned)tiles, POST_THREADS, 0, s, __VA_ARGS__);                  \
            else launch_kernel(KERNEL<2, false>, (unsigned)tiles, POST_THREADS, 0, s, __VA_ARGS__);                      \
        } else {                                                                                              \
            if (norm) launch_kernel(KERNEL<4, true>, (unsigned)tiles, POST_THREADS, 0, s, __VA_ARGS__);                  \
            else launch_kernel(KERNEL<4, false>, (unsigned)tiles, POST_THREADS, 0, s, __VA_ARGS__);                      \
        }                                                                                                     \
    } while (0)

int32_t launch_post_forward(rtma_ctx* ctx, const GroupDesc& g, LayerShape ls, const float* params, Planes Z, Planes H,
                            float2* stats, cudaStream_t s) {
    const int64_t tiles = post_tiles(g);
    if (tiles == 0) return RTMA_OK;
    if (ls.d_out > POST_MAX_WIDTH) return rtma_fail(ctx, RTMA_ERR_UNSUPPORTED, "normalised width %d > %d", ls.d_out, POST_MAX_WIDTH);
    PostArgs a{ls, params, Z, H, stats, nullptr};
    { KernelScope ks(ctx, KC_POST, s); RTMA_POST_DISPATCH(post_forward_kernel, ls, g, a); }
    RTMA_LAUNCH_CHECK(ctx);
    return RTMA_OK;
}

int32_t launch_post_backward(rtma_ctx* ctx, const GroupDesc& g, LayerShape ls, float* params, Planes Z, Planes dH,
                             float2* stats, float* partial, float lr, float* grads_record, cudaStream_t s) {
    const int64_t tiles = post_tiles(g);
    if (tiles == 0) return RTMA_OK;
    if (ls.d_out > POST_MAX_WIDTH) return rtma_fail(ctx, RTMA_ERR_UNSUPPORTED, "normalised width %d > %d", ls.d_out, POST_MAX_WIDTH);
    PostArgs a{ls, params, Z, dH, stats, partial};
    { KernelScope ks(ctx, KC_POST, s); RTMA_POST_DISPATCH(post_backward_kernel, ls, g, a); }
    RTMA_LAUNCH_CHECK(ctx);
    if (ls.gamma_offset >= 0 || ls.slope_offset >= 0) {
        dim3 grid((unsigned)ceil_div(2 * ls.d_out + 1, 32), (unsigned)g.num);
        { KernelScope ks(ctx, KC_POST, s); launch_kernel(post_reduce_sgd_kernel, grid, 256, 0, s, g, ls, partial, lr, params, grads_record); }
        RTMA_LAUNCH_CHECK(ctx);
    }
    return RTMA_OK;
}
