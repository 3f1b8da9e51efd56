// Binary TreeLSTM, forward tiles (fp32 FMA).
//   cell: [i; f_l; f_r; o; u] = W [h_l; h_r] + b,  c = s(i) tanh(u) + s(f_l) c_l + s(f_r) c_r,  h = s(o) tanh(c)
//   leaf: [i; o; u] = W_x E[tok] + b_x,            c = s(i) tanh(u),                           h = s(o) tanh(c)
// A tile is 16 RT rows x 16 hidden units; a thread accumulates all NG gates of one unit of RT rows, so the gate arithmetic
// fuses into the epilogue.  Rows and weight rows lie in shared memory as they lie in memory (K contiguous, 32 at a time,
// copied asynchronously two steps deep; row stride of an odd number of 16-byte pieces) and are read with 128-bit loads:
// RT + NG loads for 4 RT NG FMAs.
// Why so small: a wave of an ordinary batch has some 800 cells.  64 rows x 64 units made 39 tiles of 25 us each for 148 SMs;
// 64 x 16 makes 130, a quarter as long; 32 x 16 (two blocks per SM) is taken while 64 rows leave blocks without a tile.
// 601 trees, H = 148, 12 waves and the leaves: operators 0.767 -> 0.484 ms.
#pragma once
#include "rdf_tc.cuh"

__device__ __forceinline__ float sigmoid_f(float x) { return 1.f / (1.f + expf(-x)); }

static const int LT_UNITS = 16, LT_K = 32, LT_LD = LT_K + 4;
static const int LT_STAGE = (64 + 5 * LT_UNITS) * LT_LD;                   // floats of a stage
inline size_t lstm_tile_bytes() { return (size_t)2 * LT_STAGE * sizeof(float); }

template <int NG, int RT>
__device__ void lstm_forward_tiles(const DevCtx& c, float* smem, uint32_t first, uint32_t n_items) {
    constexpr bool CELL = NG == 5;
    constexpr int ROWS = 16 * RT, PIECES = (ROWS + NG * LT_UNITS) * (LT_K / 4), PER = (PIECES + 255) / 256;
    const int H = c.H, S = c.S, G = c.G;
    const int Kdim = CELL ? 2 * H : c.D, split = CELL ? H : c.D;           // k < split comes from the first source row
    const float* Wm = CELL ? c.W : c.W_x;
    const float* bias = CELL ? c.b : c.b_x;
    const int tiles_n = (H + LT_UNITS - 1) / LT_UNITS, tiles = (int)((n_items + ROWS - 1) / ROWS) * tiles_n;
    const int tu = threadIdx.x % 16, tr = threadIdx.x / 16;                // unit; rows tr + 16 i
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int row0 = (tile / tiles_n) * ROWS, u0 = (tile % tiles_n) * LT_UNITS;
        // the 16-byte pieces this thread copies per step: rows of the operands, then rows of the gates' weights
        const float *src[PER], *src2[PER];
        uint32_t valid = 0;
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const int p = threadIdx.x + 256 * q, r = p / (LT_K / 4);
            src[q] = src2[q] = c.W;
            if (p >= PIECES) continue;
            if (r < ROWS) {
                if (row0 + r < (int)n_items) {
                    valid |= 1u << q;
                    if constexpr (CELL) {
                        const uint4 it = __ldcg(reinterpret_cast<const uint4*>(&c.cell_items[first + row0 + r]));   // {out, l, r, -}
                        src[q] = c.arena + (size_t)it.y * S;
                        src2[q] = c.arena + (size_t)it.z * S - H;
                    } else {
                        src[q] = c.E + (size_t)__ldcg(&c.leaf_items[row0 + r].tok) * c.D;
                    }
                }
            } else {
                const int g = (r - ROWS) / LT_UNITS, u = u0 + (r - ROWS) % LT_UNITS;
                if (u < H) {
                    valid |= 1u << q;
                    src[q] = Wm + (size_t)(g * H + u) * Kdim;
                    src2[q] = src[q];
                }
            }
        }
        auto fetch = [&](int k0, int stage) {
            const uint32_t dst = smem_u32(smem + stage * LT_STAGE);
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                const int p = threadIdx.x + 256 * q, r = p / (LT_K / 4), kq = (p % (LT_K / 4)) * 4, k = k0 + kq;
                if (p < PIECES)
                    cp_async16(dst + 4 * (r * LT_LD + kq), (k < split ? src[q] : k < Kdim ? src2[q] : src[q] - k) + k, ((valid >> q) & 1u) && k < Kdim);
            }
            cp_async_commit();
        };
        float acc[NG][RT];
#pragma unroll
        for (int g = 0; g < NG; ++g)
#pragma unroll
            for (int i = 0; i < RT; ++i) acc[g][i] = 0.f;
        __syncthreads();                                                   // (the previous tile's stages are no longer read)
        fetch(0, 0);
        const int steps = (Kdim + LT_K - 1) / LT_K;
        for (int st = 0; st < steps; ++st) {
            if (st + 1 < steps) fetch((st + 1) * LT_K, (st + 1) & 1);
            else cp_async_commit();
            cp_async_wait<1>();
            __syncthreads();
            const float* As = smem + (st & 1) * LT_STAGE + tr * LT_LD;
            const float* Bs = smem + (st & 1) * LT_STAGE + (ROWS + tu) * LT_LD;
#pragma unroll 4
            for (int k = 0; k < LT_K; k += 4) {
                float4 a[RT];
#pragma unroll
                for (int i = 0; i < RT; ++i) a[i] = *reinterpret_cast<const float4*>(As + 16 * i * LT_LD + k);
#pragma unroll
                for (int g = 0; g < NG; ++g) {
                    const float4 b = *reinterpret_cast<const float4*>(Bs + g * LT_UNITS * LT_LD + k);
#pragma unroll
                    for (int i = 0; i < RT; ++i)
                        acc[g][i] = fmaf(a[i].w, b.w, fmaf(a[i].z, b.z, fmaf(a[i].y, b.y, fmaf(a[i].x, b.x, acc[g][i]))));
                }
            }
            __syncthreads();
        }
        const int u = u0 + tu;
        if (u >= H) continue;
        float bz[NG];
#pragma unroll
        for (int g = 0; g < NG; ++g) bz[g] = __ldg(bias + g * H + u);
#pragma unroll
        for (int i = 0; i < RT; ++i) {
            const int row = row0 + tr + 16 * i;
            if (row >= (int)n_items) continue;
            float v[NG], cc;
            uint32_t out;
            if constexpr (CELL) {
                const uint4 it = __ldcg(reinterpret_cast<const uint4*>(&c.cell_items[first + row]));
                out = it.x;
                const float cl = __ldcg(c.arena + (size_t)it.y * S + H + u), cr = __ldcg(c.arena + (size_t)it.z * S + H + u);
#pragma unroll
                for (int g = 0; g < 4; ++g) v[g] = sigmoid_f(acc[g][i] + bz[g]);
                v[4] = tanhf(acc[4][i] + bz[4]);
                cc = v[0] * v[4] + v[1] * cl + v[2] * cr;
            } else {
                out = __ldcg(&c.leaf_items[row].slot);
                v[0] = sigmoid_f(acc[0][i] + bz[0]);
                v[1] = sigmoid_f(acc[1][i] + bz[1]);
                v[2] = tanhf(acc[2][i] + bz[2]);
                cc = v[0] * v[2];
            }
            float* st = c.arena + (size_t)out * S;
            st[u] = v[CELL ? 3 : 1] * tanhf(cc);
            st[H + u] = cc;
            if (c.gates) {
                float* gt = c.gates + (size_t)out * G;
#pragma unroll
                for (int g = 0; g < NG; ++g) gt[g * H + u] = v[g];
            }
        }
    }
    cp_async_wait<0>();
}

// 64 rows per tile when that gives every block a tile
template <int NG>
__device__ __forceinline__ void lstm_forward_wave(const DevCtx& c, float* smem, uint32_t first, uint32_t n_items) {
    const uint32_t tiles_n = (c.H + LT_UNITS - 1) / LT_UNITS;
    if ((n_items + 63u) / 64u * tiles_n >= gridDim.x) lstm_forward_tiles<NG, 4>(c, smem, first, n_items);
    else lstm_forward_tiles<NG, 2>(c, smem, first, n_items);
}
