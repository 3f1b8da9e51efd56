// Binary TreeLSTM, forward tiles (fp32 FMA).
//   cell: [i; f_l; f_r; o; u] = W [h_l; h_r] + b,  c = s(i) tanh(u) + s(f_l) c_l + s(f_r) c_r,  h = s(o) tanh(c)
//   leaf: [i; o; u] = W_x E[tok] + b_x,            c = s(i) tanh(u),                           h = s(o) tanh(c)
// A tile is 64, 32 or 16 rows x 16 hidden units.  The threads form KS groups that split the contraction; a thread accumulates
// all NG gates of one unit of RT rows over its group's k, the groups' sums meet in shared memory, and each group finishes (gate
// arithmetic) its share of the rows.  Rows and weight rows lie in shared memory as they lie in memory (K contiguous, 32 at a
// time, copied asynchronously two steps ahead; row stride of an odd number of 16-byte pieces) and are read with 128-bit loads:
// RT + NG loads for 4 RT NG FMAs.
// Why so small: a wave of an ordinary batch has some 800 cells.  64 rows x 64 units made 39 tiles of 25 us each for 148 SMs;
// with 16 units two blocks per SM find work, and splitting the contraction keeps RT at 4 to 8 for the smaller tiles, too.
// 601 trees, H = 148, 12 waves and the leaves: operators 0.767 -> 0.484 (no split, one step ahead) -> 0.416 ms.
#pragma once
#include "rdf_tc.cuh"

__device__ __forceinline__ float sigmoid_f(float x) { return 1.f / (1.f + expf(-x)); }

static const int LT_UNITS = 16, LT_K = 32, LT_LD = LT_K + 4;
static const int LT_STAGE = (64 + 5 * LT_UNITS) * LT_LD;                   // floats of a stage
static const int LT_STAGES = 3;
inline size_t lstm_tile_bytes() { return (size_t)LT_STAGES * LT_STAGE * sizeof(float); }

template <int NG, int RT, int KS>
__device__ void lstm_forward_tiles(const DevCtx& c, float* smem, uint32_t first, uint32_t n_items) {
    constexpr bool CELL = NG == 5;
    constexpr int TG = 256 / KS, RSTEP = TG / 16;                          // threads of a group; rows between two of a thread
    constexpr int ROWS = RSTEP * RT, PIECES = (ROWS + NG * LT_UNITS) * (LT_K / 4), PER = (PIECES + 255) / 256;
    const int H = c.H, S = c.S, G = c.G;
    const int Kdim = CELL ? 2 * H : c.D, split = CELL ? H : c.D;           // k < split comes from the first source row
    const float* Wm = CELL ? c.W : c.W_x;
    const float* bias = CELL ? c.b : c.b_x;
    const int tiles_n = (H + LT_UNITS - 1) / LT_UNITS, tiles = (int)((n_items + ROWS - 1) / ROWS) * tiles_n;
    const int group = threadIdx.x / TG, tid = threadIdx.x % TG, tu = tid % 16, tr = tid / 16;      // unit; rows tr + RSTEP i
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
        const int steps = (Kdim + LT_K - 1) / LT_K;
        fetch(0, 0);
        fetch(LT_K, 1);                                                    // (beyond the last step: zeros)
        for (int st = 0; st < steps; ++st) {
            cp_async_wait<1>();
            __syncthreads();                                               // step st is there; step st - 1 is no longer read
            if (st + 2 < steps) fetch((st + 2) * LT_K, (st + 2) % LT_STAGES);
            else cp_async_commit();
            const float* As = smem + (st % LT_STAGES) * LT_STAGE + tr * LT_LD;
            const float* Bs = smem + (st % LT_STAGES) * LT_STAGE + (ROWS + tu) * LT_LD;
#pragma unroll 4
            for (int k = group * (LT_K / KS); k < (group + 1) * (LT_K / KS); k += 4) {
                float4 a[RT];
#pragma unroll
                for (int i = 0; i < RT; ++i) a[i] = *reinterpret_cast<const float4*>(As + RSTEP * i * LT_LD + k);
#pragma unroll
                for (int g = 0; g < NG; ++g) {
                    const float4 b = *reinterpret_cast<const float4*>(Bs + g * LT_UNITS * LT_LD + k);
#pragma unroll
                    for (int i = 0; i < RT; ++i)
                        acc[g][i] = fmaf(a[i].w, b.w, fmaf(a[i].z, b.z, fmaf(a[i].y, b.y, fmaf(a[i].x, b.x, acc[g][i]))));
                }
            }
        }
        cp_async_wait<0>();
        __syncthreads();
        // the groups' partial sums meet in shared memory (the stages are done with); each group finishes its share of the rows
        static_assert(256 * RT * 5 <= 2 * LT_STAGE && RT % KS == 0, "the sums fit the stages");
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
            for (int g = 0; g < NG; ++g) smem[((group * RT + i) * NG + g) * TG + tid] = acc[g][i];
        __syncthreads();
        const int u = u0 + tu;
        if (u >= H) continue;
        float bz[NG];
#pragma unroll
        for (int g = 0; g < NG; ++g) bz[g] = __ldg(bias + g * H + u);
#pragma unroll
        for (int ii = 0; ii < RT / KS; ++ii) {
            const int i = group * (RT / KS) + ii, row = row0 + tr + RSTEP * i;
            if (row >= (int)n_items) continue;
            float z[NG], v[NG], cc;
#pragma unroll
            for (int g = 0; g < NG; ++g) {
                z[g] = bz[g];
#pragma unroll
                for (int q = 0; q < KS; ++q) z[g] += smem[((q * RT + i) * NG + g) * TG + tid];
            }
            uint32_t out;
            if constexpr (CELL) {
                const uint4 it = __ldcg(reinterpret_cast<const uint4*>(&c.cell_items[first + row]));
                out = it.x;
                const float cl = __ldcg(c.arena + (size_t)it.y * S + H + u), cr = __ldcg(c.arena + (size_t)it.z * S + H + u);
#pragma unroll
                for (int g = 0; g < 4; ++g) v[g] = sigmoid_f(z[g]);
                v[4] = tanhf(z[4]);
                cc = v[0] * v[4] + v[1] * cl + v[2] * cr;
            } else {
                out = __ldcg(&c.leaf_items[row].slot);
                v[0] = sigmoid_f(z[0]);
                v[1] = sigmoid_f(z[1]);
                v[2] = tanhf(z[2]);
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

// The largest tile that gives every block one; 16 rows where 32 would leave half of the blocks without (0.431 -> 0.423 ms).
template <int NG>
__device__ __forceinline__ void lstm_forward_wave(const DevCtx& c, float* smem, uint32_t first, uint32_t n_items) {
    const uint32_t tiles_n = (c.H + LT_UNITS - 1) / LT_UNITS;
    if ((n_items + 63u) / 64u * tiles_n >= gridDim.x) lstm_forward_tiles<NG, 8, 2>(c, smem, first, n_items);
    else if ((n_items + 31u) / 32u * tiles_n >= gridDim.x / 2) lstm_forward_tiles<NG, 4, 2>(c, smem, first, n_items);
    else lstm_forward_tiles<NG, 4, 4>(c, smem, first, n_items);
}
