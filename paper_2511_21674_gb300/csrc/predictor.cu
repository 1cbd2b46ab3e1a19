// Learned learning-signal predictor: BF16 MLP with FP32 accumulation on the
// tensor cores, trained by Adam, all on the GPU (forward, backward and
// update kernels below).  Semantics and layouts: include/eprop_predictor.h.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "eprop_predictor.h"
#include "predictor_internal.h"

using bf16 = __nv_bfloat16;

struct eprop_predictor {
    int n_in = 0, hidden = 0, n_out = 0, max_rows = 0;
    long long n_params = 0;
    long long off_W[3] = {0, 0, 0}, off_b[3] = {0, 0, 0};
    cudaStream_t st = nullptr;
    int own_stream = 0;
    float *params = nullptr, *grads = nullptr, *m = nullptr, *v = nullptr;
    // BF16 arrays have rows padded to multiples of 8 values (16-byte pieces)
    int ldX = 0, ldH = 0, ldK = 0;
    bf16 *Wh[3] = {nullptr, nullptr, nullptr};
    bf16 *Xh = nullptr, *H1h = nullptr, *H2h = nullptr, *dYh = nullptr, *dA2h = nullptr, *dA1h = nullptr;
    float *A1 = nullptr, *A2 = nullptr, *Y = nullptr;
    float *bpart = nullptr;          // [row tiles][2 hidden + n_out] bias gradients of row tiles
    float *lpart = nullptr;          // [row tiles] squared errors
    int sm_count = 1;
    float *xin = nullptr, *ein = nullptr, *yout = nullptr, *loss = nullptr;
    float *stage = nullptr;          // FP32 widening of BF16 buffers for eprop_predictor_read
    float *in_scale = nullptr;       // [n_in] input scale (part of the model; default 1)
    long long adam_t = 0;
    int rows = 0;
    std::string err;
    std::vector<void *> allocs;
};

namespace pred {

// ------------------------------------------------------------------ kernels

__device__ __forceinline__ float gelu(float x) { return 0.5f * x * erfcf(-x * 0.70710678118654752f); }
__device__ __forceinline__ float gelu_grad(float x) {
    return 0.5f * erfcf(-x * 0.70710678118654752f) + x * expf(-0.5f * x * x) * 0.39894228040143268f;
}

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
// 16-byte asynchronous copy; zeros when !in
__device__ __forceinline__ void cp16(void *dst, const void *src, bool in) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(dst)), "l"(src), "r"(in ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void ldm4(uint32_t (&r)[4], const void *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_addr(p)) : "memory");
}
__device__ __forceinline__ void ldm4t(uint32_t (&r)[4], const void *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_addr(p)) : "memory");
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The whole MLP of a tile of 16 MT rows in one block: inputs scaled and
// rounded, three layers, and in training the output delta, the loss and both
// hidden deltas.  The tile's activations stay in shared memory; the weights
// (174 KB at 74-256-256-10) stream from L2 in chunks of 64 x 256 through a ring
// of asynchronous copies that runs on across the layers.  Each of the 8 warps
// owns 32 columns of a 256-column block and all rows of the tile.  What bounds
// a call is latency (launches, the chunks' round trips), not the tensor cores:
// at 256 rows the products are 45 MFLOP.  One GEMM launch per product with
// element-wise staging took 33 us each (a 16-deep K-step per barrier); the
// products keep its K order, so the forward pass has the same bits.
// Measured (74-256-256-10, host arrays in and out): inference of 256 rows 108
// -> 54 us, training step of 4096 rows 2.08 -> 0.17 ms.
// Fragment layouts of m16n8k16 (row.col), lane = 4 g + t: A (g, 2t..2t+1),
// (g+8, ..), (g, 2t+8..), (g+8, 2t+8..); B (2t..2t+1, g), (2t+8.., g); C (g,
// 2t..2t+1), (g+8, 2t..2t+1).
constexpr int kChunkK = 64, kChunkN = 256;
constexpr int kMlpThreads = 256, kNarrowThreads = 64;

struct Mlp {
    int rows, I, H, K, ldX, ldH, ldK, stages;
    const float *x, *scale, *e, *b1, *b2, *b3;
    const bf16 *W1, *W2, *W3;
    bf16 *Xh, *H1h, *H2h, *dYh, *dA2h, *dA1h;
    float *A1, *A2, *Y, *bpart, *lpart;
    float inv;
};

__host__ __device__ inline int pad16(int x) { return (x + 15) & ~15; }
// A ring stage holds 64 rows of a layer's columns or, backward, as many rows of
// 64 columns; narrow networks need few columns (and many blocks then share an SM).
__host__ __device__ inline int mlp_cols(int H, int K) {
    const int c = ((H > K ? H : K) + 31) & ~31;
    return c < kChunkN ? c : kChunkN;
}
__host__ __device__ inline int mlp_stage(int H, int K) {
    const int c = mlp_cols(H, K), fwd = kChunkK * (c + 8), bwd = c * (kChunkK + 8);
    return fwd > bwd ? fwd : bwd;
}
// The inputs' tile is dead once the first layer is done: the second layer's
// output takes its place.  (Not where its rows have padding columns, which have
// to stay zero.)
__host__ __device__ inline bool mlp_alias(int H) { return H % 16 == 0; }
static size_t mlp_smem(const Mlp &a, int MT, bool train) {
    const size_t x = (size_t)(pad16(a.I) + 8), h = (size_t)(pad16(a.H) + 8);
    const size_t row = (mlp_alias(a.H) ? std::max(x, h) : x + h) + h + (train ? pad16(a.K) + 8 : 0);
    return (row * 16 * MT + (size_t)a.stages * mlp_stage(a.H, a.K)) * sizeof(bf16);
}

template <int MT, bool TRAIN, int NT = kMlpThreads>
__global__ void __launch_bounds__(NT) mlp_kernel(Mlp a) {
    extern __shared__ __align__(16) unsigned char pred_sm[];
    __shared__ float red[NT / 32];
    const int SX = pad16(a.I) + 8, SH = pad16(a.H) + 8, SK = pad16(a.K) + 8;
    constexpr int R = 16 * MT;
    bf16 *ring = reinterpret_cast<bf16 *>(pred_sm);
    const int stage_n = mlp_stage(a.H, a.K), ldS = mlp_cols(a.H, a.K) + 8;
    bf16 *Xs = ring + (size_t)a.stages * stage_n;
    const bool alias = mlp_alias(a.H);
    bf16 *P1 = Xs + R * (alias ? max(SX, SH) : SX), *P2 = alias ? Xs : P1 + R * SH;
    bf16 *dYs = alias ? P1 + R * SH : P2 + R * SH;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int r0 = blockIdx.x * R;
    // phases: 0..2 the layers, 3 dA2 = dY W3^T, 4 dA1 = dA2 W2^T
    constexpr int kPhases = TRAIN ? 5 : 3;
    auto kdim = [&](int ph) { return ph == 0 ? a.I : ph == 3 ? a.K : a.H; };
    auto ndim = [&](int ph) { return ph == 2 ? a.K : a.H; };
    struct Pos {
        int ph, n0, k0;
    };
    auto advance = [&](Pos &p) {
        p.k0 += kChunkK;
        if (p.k0 < kdim(p.ph)) return;
        p.k0 = 0;
        p.n0 += kChunkN;
        if (p.n0 < ndim(p.ph)) return;
        p.n0 = 0;
        ++p.ph;
    };
    // chunk of the phase's weights: layers [k][n] rows, backward [n][k] rows
    auto load = [&](const Pos &p, bf16 *st) {
        if (p.ph < kPhases) {
            const int N = ndim(p.ph), Kd = kdim(p.ph);
            if (p.ph < 3) {
                const bf16 *W = p.ph == 0 ? a.W1 : p.ph == 1 ? a.W2 : a.W3;
                const int ld = p.ph == 2 ? a.ldK : a.ldH;
                const int pieces = (min(kChunkN, N - p.n0) + 31) / 32 * 4;      // of 8 columns
                auto piece = [&](int k, int c) {
                    const bool in = p.k0 + k < Kd && p.n0 + c < ld;
                    cp16(st + k * ldS + c, in ? W + (size_t)(p.k0 + k) * ld + p.n0 + c : W, in);
                };
                // a full chunk without divisions: with two per copy, 1024-1024-1024
                // took 395 us for one row (192 chunks), now 263
                if (pieces == kChunkN / 8) {
#pragma unroll
                    for (int i = 0; i < kChunkK * kChunkN / 8 / NT; ++i)
                        piece((tid >> 5) + i * (NT / 32), (tid & 31) * 8);
                } else {
                    for (int q = tid; q < kChunkK * pieces; q += NT) piece(q / pieces, q % pieces * 8);
                }
            } else {
                const bf16 *W = p.ph == 3 ? a.W3 : a.W2;
                const int ld = p.ph == 3 ? a.ldK : a.ldH;
                const int pieces = min(kChunkK, pad16(Kd) - p.k0) / 8;
                const int rows = (min(kChunkN, N - p.n0) + 31) & ~31;
                auto piece = [&](int nn, int c) {
                    const bool in = p.n0 + nn < N && p.k0 + c < ld;
                    cp16(st + nn * (kChunkK + 8) + c, in ? W + (size_t)(p.n0 + nn) * ld + p.k0 + c : W, in);
                };
                if (pieces == kChunkK / 8) {
#pragma unroll 8
                    for (int nn = tid >> 3; nn < rows; nn += NT / 8) piece(nn, (tid & 7) * 8);
                } else {
                    for (int q = tid; q < rows * pieces; q += NT) piece(q / pieces, q % pieces * 8);
                }
            }
        }
        cp_commit();
    };
    Pos lp{0, 0, 0};
    for (int q = 0; q < a.stages - 1; ++q) {
        load(lp, ring + (size_t)q * stage_n);
        if (lp.ph < kPhases) advance(lp);
    }
    // activation tiles: padding columns and rows past the end stay zero
    const int tiles_n = R * ((alias ? SH : 2 * SH) + (TRAIN ? SK : 0)) / 2;
    for (int q = tid; q < tiles_n; q += NT) reinterpret_cast<uint32_t *>(P1)[q] = 0u;
#pragma unroll 4
    for (int m = warp; m < R; m += NT / 32) {
        const bool row = r0 + m < a.rows;
        const float *x = a.x + (size_t)(row ? r0 + m : 0) * a.I;
        bf16 *xh = a.Xh + (size_t)(row ? r0 + m : 0) * a.ldX;
        for (int c = lane; c < SX; c += 32) {
            const bf16 h = __float2bfloat16_rn(row && c < a.I ? x[c] * a.scale[c] : 0.f);
            Xs[m * SX + c] = h;
            if (row && c < a.ldX) xh[c] = h;
        }
    }
    float sq = 0.f;
    float acc[MT][4][4];
    Pos p{0, 0, 0};
    for (int c = 0; p.ph < kPhases; ++c) {
        if (a.stages == 4) cp_wait<2>();
        else if (a.stages == 3) cp_wait<1>();
        else cp_wait<0>();
        __syncthreads();                 // chunk c is there, chunk c - 1 and its tiles are done
        {
            const int q = c + a.stages - 1;
            load(lp, ring + (size_t)(q % a.stages) * stage_n);
            if (lp.ph < kPhases) advance(lp);
        }
        const bf16 *st = ring + (size_t)(c % a.stages) * stage_n;
        const int N = ndim(p.ph), Kd = kdim(p.ph);
        const int nb = p.n0 + warp * 32;
        const bool last = p.k0 + kChunkK >= Kd;
        if (nb < N) {
            if (p.k0 == 0) {
#pragma unroll
                for (int m = 0; m < MT; ++m)
#pragma unroll
                    for (int j = 0; j < 4; ++j)
#pragma unroll
                        for (int e = 0; e < 4; ++e) acc[m][j][e] = 0.f;
            }
            const bf16 *As = p.ph == 0 ? Xs : p.ph == 1 ? P1 : p.ph == 3 ? dYs : P2;
            const int lda = p.ph == 0 ? SX : p.ph == 3 ? SK : SH;
            const int steps = min(kChunkK, pad16(Kd) - p.k0) / 16;
            for (int ks = 0; ks < steps; ++ks) {
                uint32_t af[MT][4], bfr[2][4];
#pragma unroll
                for (int m = 0; m < MT; ++m)
                    ldm4(af[m], As + (m * 16 + (lane & 15)) * lda + p.k0 + ks * 16 + (lane >> 4) * 8);
                const int mt = lane >> 3, lr = lane & 7;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int nl = warp * 32 + h * 16 + (mt >> 1) * 8;
                    const int kl = ks * 16 + (mt & 1) * 8;
                    if (p.ph < 3) ldm4t(bfr[h], st + (kl + lr) * ldS + nl);
                    else ldm4(bfr[h], st + (nl + lr) * (kChunkK + 8) + kl);
                }
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int m = 0; m < MT; ++m) mma_bf16(acc[m][j], af[m], bfr[j >> 1][(j & 1) * 2], bfr[j >> 1][(j & 1) * 2 + 1]);
            }
            if (last) {
                const float *bias = p.ph == 0 ? a.b1 : p.ph == 1 ? a.b2 : a.b3;
                float *pre = (p.ph == 0 || p.ph == 4) ? a.A1 : a.A2;
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int f = 0; f < 2; ++f) {
                        const int nn = nb + j * 8 + 2 * t + f;
                        float col = 0.f;             // the column's share of a bias gradient
#pragma unroll
                        for (int mh = 0; mh < 2 * MT; ++mh) {
                            const int m = (mh >> 1) * 16 + (mh & 1) * 8 + g, r = r0 + m;
                            if (r >= a.rows || nn >= N) continue;
                            float v = acc[mh >> 1][j][(mh & 1) * 2 + f];
                            if (p.ph < 2) {
                                v += bias[nn];
                                pre[(size_t)r * a.H + nn] = v;
                                const bf16 h = __float2bfloat16_rn(gelu(v));
                                (p.ph == 0 ? P1 : P2)[m * SH + nn] = h;
                                (p.ph == 0 ? a.H1h : a.H2h)[(size_t)r * a.ldH + nn] = h;
                            } else if (p.ph == 2) {
                                v += bias[nn];
                                a.Y[(size_t)r * a.K + nn] = v;
                                if (TRAIN) {
                                    const float d = v - a.e[(size_t)r * a.K + nn];
                                    sq = fmaf(d, d, sq);
                                    const float dy = d * a.inv;
                                    col += dy;
                                    const bf16 h = __float2bfloat16_rn(dy);
                                    dYs[m * SK + nn] = h;
                                    a.dYh[(size_t)r * a.ldK + nn] = h;
                                }
                            } else {
                                v *= gelu_grad(pre[(size_t)r * a.H + nn]);   // this thread's own value
                                col += v;
                                const bf16 h = __float2bfloat16_rn(v);
                                if (p.ph == 3) P2[m * SH + nn] = h;          // dA2 takes H2's place
                                (p.ph == 3 ? a.dA2h : a.dA1h)[(size_t)r * a.ldH + nn] = h;
                            }
                        }
                        if (TRAIN && p.ph >= 2) {
                            for (int o = 4; o < 32; o <<= 1) col += __shfl_xor_sync(0xffffffffu, col, o);
                            const int off = p.ph == 4 ? 0 : p.ph == 3 ? a.H : 2 * a.H;
                            if (g == 0 && nn < N) a.bpart[(size_t)blockIdx.x * (2 * a.H + a.K) + off + nn] = col;
                        }
                    }
            }
        }
        advance(p);
    }
    cp_wait<0>();
    if (TRAIN) {
        for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
        if (lane == 0) red[warp] = sq;
        __syncthreads();
        if (tid == 0) {
            float s = 0.f;
            for (int w = 0; w < NT / 32; ++w) s += red[w];
            a.lpart[blockIdx.x] = s;
        }
    }
}

// Weight gradients dW[m][n] = sum_r A[r][m] D[r][n] of the three layers in one
// launch, one block per 32 x 32 tile over all rows.  The rows are not split: one
// accumulator per element, 16 rows per step in row order, keeps the sums' bits
// (Adam divides small gradients by their own size, so a changed last bit of a
// gradient near zero would move its weight), and with eight chunks of 64 rows
// in flight the walk is bound by L2, not by its length.  64 x 32 tiles with
// element-wise staging took 678 us per layer at 4096 rows; this launch 21 us
// for all three.
constexpr int kDwThreads = 128, kDwTile = 32, kDwRows = 64, kDwStages = 8, kDwLd = kDwTile + 8;
struct Dw {
    int rows, tiles[3];
    const bf16 *A[3], *D[3];
    int ldA[3], ldD[3], M[3], N[3];
    float *out[3];
};

__global__ void __launch_bounds__(kDwThreads) dw_kernel(Dw a) {
    extern __shared__ __align__(16) unsigned char pred_sm[];
    bf16 *ring = reinterpret_cast<bf16 *>(pred_sm);
    constexpr int kStage = 2 * kDwRows * kDwLd;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    int l = 0, tile = blockIdx.x;
    while (l < 2 && tile >= a.tiles[l]) tile -= a.tiles[l++];
    const int M = a.M[l], N = a.N[l], nt = (N + kDwTile - 1) / kDwTile;
    const int m0 = tile / nt * kDwTile, n0 = tile % nt * kDwTile;
    const int chunks = (a.rows + kDwRows - 1) / kDwRows;
    auto load = [&](int c) {
        if (c < chunks) {
            bf16 *st = ring + (c % kDwStages) * kStage;
#pragma unroll
            for (int q = tid; q < 2 * kDwRows * (kDwTile / 8); q += kDwThreads) {
                const int which = q / (kDwRows * (kDwTile / 8)), k = (q / (kDwTile / 8)) % kDwRows;
                const int cc = (q % (kDwTile / 8)) * 8;
                const bf16 *src = which ? a.D[l] : a.A[l];
                const int ld = which ? a.ldD[l] : a.ldA[l], c0 = (which ? n0 : m0) + cc, r = c * kDwRows + k;
                const bool in = r < a.rows && c0 < ld;
                cp16(st + which * kDwRows * kDwLd + k * kDwLd + cc, in ? src + (size_t)r * ld + c0 : src, in);
            }
        }
        cp_commit();
    };
    for (int c = 0; c < kDwStages - 1; ++c) load(c);
    float acc[2][4];
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[j][e] = 0.f;
    const int wm = (warp >> 1) * 16, wn = (warp & 1) * 16, mt = lane >> 3, lr = lane & 7;
    for (int c = 0; c < chunks; ++c) {
        cp_wait<kDwStages - 2>();
        __syncthreads();
        load(c + kDwStages - 1);
        const bf16 *As = ring + (c % kDwStages) * kStage, *Ds = As + kDwRows * kDwLd;
#pragma unroll
        for (int ks = 0; ks < kDwRows / 16; ++ks) {
            uint32_t af[4], bfr[4];
            ldm4t(af, As + (ks * 16 + (mt >> 1) * 8 + lr) * kDwLd + wm + (mt & 1) * 8);
            ldm4t(bfr, Ds + (ks * 16 + (mt & 1) * 8 + lr) * kDwLd + wn + (mt >> 1) * 8);
            mma_bf16(acc[0], af, bfr[0], bfr[1]);
            mma_bf16(acc[1], af, bfr[2], bfr[3]);
        }
    }
    cp_wait<0>();
    float *out = a.out[l];
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int mm = m0 + wm + g + (e >= 2 ? 8 : 0), nn = n0 + wn + j * 8 + 2 * t + (e & 1);
            if (mm < M && nn < N) out[(size_t)mm * N + nn] = acc[j][e];
        }
}

// layout of the packed parameters: layer l holds W [I_l][O_l] then b [O_l]
struct Layout {
    int I[3], O[3], ld[3];
    long long offW[3], offb[3];
    bf16 *Wh[3];
};
__device__ __forceinline__ void locate(const Layout &L, long long q, int &l, long long &i, bool &bias) {
    l = q >= L.offW[2] ? 2 : q >= L.offW[1] ? 1 : 0;
    bias = q >= L.offb[l];
    i = q - (bias ? L.offb[l] : L.offW[l]);
}
__device__ __forceinline__ void put_weight(const Layout &L, int l, long long i, float w) {
    const long long r = i / L.O[l];
    L.Wh[l][r * L.ld[l] + (i - r * L.O[l])] = __float2bfloat16_rn(w);
}
__global__ void refresh_kernel(Layout L, const float *w, long long n) {
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < n;
         q += (long long)gridDim.x * blockDim.x) {
        int l;
        long long i;
        bool bias;
        locate(L, q, l, i, bias);
        if (!bias) put_weight(L, l, i, w[q]);
    }
}

// Adam (Eq. adam1, Eq. adam2, Eq. adam) on the FP32 masters: sums the bias
// gradients of the row tiles in order, steps, and refreshes the BF16 weights;
// block 0 also sums the loss.
__global__ void adam_kernel(Layout L, float *w, float *grad, float *m, float *v, long long n, const float *bpart,
                            const float *lpart, int tiles, float half_inv, float *loss, float lr, float c1, float c2) {
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < n;
         q += (long long)gridDim.x * blockDim.x) {
        int l;
        long long i;
        bool bias;
        locate(L, q, l, i, bias);
        float gq;
        if (bias) {
            gq = 0.f;
            const long long nb = L.O[0] + L.O[1] + L.O[2];
            const float *bp = bpart + (l == 0 ? 0 : l == 1 ? L.O[0] : L.O[0] + L.O[1]) + i;
#pragma unroll 8
            for (int s = 0; s < tiles; ++s) gq += bp[s * nb];
            grad[q] = gq;
        } else {
            gq = grad[q];
        }
        const float mq = 0.9f * m[q] + 0.1f * gq;
        const float vq = 0.999f * v[q] + 0.001f * gq * gq;
        m[q] = mq;
        v[q] = vq;
        const float wq = w[q] - lr * (mq / c1) / (sqrtf(vq / c2) + 1e-8f);
        w[q] = wq;
        if (!bias) put_weight(L, l, i, wq);
    }
    if (blockIdx.x == 0 && threadIdx.x < 32) {
        float s = 0.f;
        for (int q = threadIdx.x; q < tiles; q += 32) s += lpart[q];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) *loss = half_inv * s;
    }
}

// rows of `cols` BF16 values with leading dimension ld, widened
__global__ void bf16_to_float_kernel(const bf16 *src, int ld, int cols, float *dst, long long n) {
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < n;
         q += (long long)gridDim.x * blockDim.x)
        dst[q] = __bfloat162float(src[q / cols * ld + q % cols]);
}

// ------------------------------------------------------------------ host

constexpr int kMlpSmemMax = 220 * 1024;
constexpr int kDwSmem = kDwStages * 2 * kDwRows * kDwLd * (int)sizeof(bf16);

static unsigned blocks_for(long long n) {
    long long b = (n + 255) / 256;
    return (unsigned)(b < 1 ? 1 : (b > 4096 ? 4096 : b));
}

static uint64_t splitmix(uint64_t x) {
    x += 0x9E3779B97F4A7C15ULL;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ULL;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBULL;
    return x ^ (x >> 31);
}

}  // namespace pred

using namespace pred;

static eprop_status pfail(eprop_predictor *p, eprop_status s, const char *msg) {
    if (p) p->err = msg;
    return s;
}

static eprop_status pcuda(eprop_predictor *p, cudaError_t e, const char *what) {
    if (p) p->err = std::string(what) + ": " + cudaGetErrorString(e);
    return e == cudaErrorMemoryAllocation ? EPROP_ENOMEM : EPROP_ECUDA;
}

#define PCK(p, call)                                          \
    do {                                                      \
        cudaError_t _e = (call);                              \
        if (_e != cudaSuccess) return pcuda((p), _e, #call);  \
    } while (0)

template <typename T>
static cudaError_t palloc(eprop_predictor *p, T **ptr, long long count) {
    void *q = nullptr;
    cudaError_t e = cudaMalloc(&q, (size_t)(count > 0 ? count : 1) * sizeof(T));
    if (e != cudaSuccess) return e;
    p->allocs.push_back(q);
    *ptr = static_cast<T *>(q);
    return cudaMemset(q, 0, (size_t)(count > 0 ? count : 1) * sizeof(T));
}

static thread_local std::string g_pred_create_err;

extern "C" eprop_status eprop_predictor_create(int32_t n_in, int32_t hidden, int32_t n_out, int32_t max_rows,
                                               const float *params, uint64_t seed, void *stream,
                                               eprop_predictor **out) {
    if (!out) return EPROP_EINVAL;
    *out = nullptr;
    if (n_in < 1 || n_in > 1024 || n_out < 1 || n_out > 1024 || hidden < 16 || hidden > 1024 || max_rows < 1 ||
        max_rows > 65536) {
        g_pred_create_err = "predictor sizes out of range";
        return EPROP_EINVAL;
    }
    eprop_predictor *p = new eprop_predictor();
    p->n_in = n_in;
    p->hidden = hidden;
    p->n_out = n_out;
    p->max_rows = max_rows;
    const int fan_in[3] = {n_in, hidden, hidden}, fan_out[3] = {hidden, hidden, n_out};
    long long o = 0;
    for (int l = 0; l < 3; ++l) {
        p->off_W[l] = o;
        o += (long long)fan_in[l] * fan_out[l];
        p->off_b[l] = o;
        o += fan_out[l];
    }
    p->n_params = o;
    eprop_status s = EPROP_OK;
    cudaError_t e = cudaSuccess;
    if (stream) {
        p->st = static_cast<cudaStream_t>(stream);
    } else {
        e = cudaStreamCreateWithFlags(&p->st, cudaStreamNonBlocking);
        p->own_stream = 1;
    }
    const long long R = max_rows, H = hidden;
    auto pad8 = [](int x) { return (x + 7) & ~7; };
    p->ldX = pad8(n_in);
    p->ldH = pad8(hidden);
    p->ldK = pad8(n_out);
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&p->sm_count, cudaDevAttrMultiProcessorCount, dev);
    const long long tiles = (R + 15) / 16;
    if (e == cudaSuccess) e = palloc(p, &p->params, o);
    if (e == cudaSuccess) e = palloc(p, &p->grads, o);
    if (e == cudaSuccess) e = palloc(p, &p->m, o);
    if (e == cudaSuccess) e = palloc(p, &p->v, o);
    for (int l = 0; l < 3 && e == cudaSuccess; ++l)
        e = palloc(p, &p->Wh[l], (long long)fan_in[l] * (l == 2 ? p->ldK : p->ldH));
    if (e == cudaSuccess) e = palloc(p, &p->Xh, R * p->ldX);
    if (e == cudaSuccess) e = palloc(p, &p->H1h, R * p->ldH);
    if (e == cudaSuccess) e = palloc(p, &p->H2h, R * p->ldH);
    if (e == cudaSuccess) e = palloc(p, &p->dYh, R * p->ldK);
    if (e == cudaSuccess) e = palloc(p, &p->dA2h, R * p->ldH);
    if (e == cudaSuccess) e = palloc(p, &p->dA1h, R * p->ldH);
    if (e == cudaSuccess) e = palloc(p, &p->bpart, tiles * (2 * H + n_out));
    if (e == cudaSuccess) e = palloc(p, &p->lpart, tiles);
    if (e == cudaSuccess) e = palloc(p, &p->A1, R * H);
    if (e == cudaSuccess) e = palloc(p, &p->A2, R * H);
    if (e == cudaSuccess) e = palloc(p, &p->Y, R * n_out);
    if (e == cudaSuccess) e = palloc(p, &p->xin, R * n_in);
    if (e == cudaSuccess) e = palloc(p, &p->ein, R * n_out);
    if (e == cudaSuccess) e = palloc(p, &p->yout, R * n_out);
    if (e == cudaSuccess) e = palloc(p, &p->loss, 1);
    if (e == cudaSuccess) e = palloc(p, &p->stage, R * (H > n_in ? (H > n_out ? H : n_out) : (n_in > n_out ? n_in : n_out)));
    if (e == cudaSuccess) e = palloc(p, &p->in_scale, n_in);
    if (e == cudaSuccess) {
        std::vector<float> ones((size_t)n_in, 1.0f);
        e = cudaMemcpy(p->in_scale, ones.data(), (size_t)n_in * 4, cudaMemcpyHostToDevice);
    }
    if (e != cudaSuccess) {
        g_pred_create_err = std::string("predictor allocation: ") + cudaGetErrorString(e);
        eprop_predictor_destroy(p);
        return e == cudaErrorMemoryAllocation ? EPROP_ENOMEM : EPROP_ECUDA;
    }
    cudaFuncSetAttribute(mlp_kernel<1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMlpSmemMax);
    cudaFuncSetAttribute(mlp_kernel<2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMlpSmemMax);
    cudaFuncSetAttribute(mlp_kernel<1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMlpSmemMax);
    cudaFuncSetAttribute(mlp_kernel<2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMlpSmemMax);
    cudaFuncSetAttribute(dw_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kDwSmem);
    std::vector<float> init;
    if (!params) {
        init.assign((size_t)o, 0.f);
        for (int l = 0; l < 3; ++l) {
            const double sd = 1.0 / std::sqrt((double)fan_in[l]);
            const long long cnt = (long long)fan_in[l] * fan_out[l];
            for (long long q = 0; q < cnt; ++q) {
                const uint64_t h1 = splitmix(seed ^ splitmix((uint64_t)(p->off_W[l] + q) * 2 + 0));
                const uint64_t h2 = splitmix(seed ^ splitmix((uint64_t)(p->off_W[l] + q) * 2 + 1));
                const double u1 = ((double)(h1 >> 11) + 1.0) * (1.0 / 9007199254740992.0);
                const double u2 = (double)(h2 >> 11) * (1.0 / 9007199254740992.0);
                init[(size_t)(p->off_W[l] + q)] =
                    (float)(sd * std::sqrt(-2.0 * std::log(u1)) * std::cos(6.283185307179586 * u2));
            }
        }
        params = init.data();
    }
    s = eprop_predictor_set_params(p, params);
    if (s != EPROP_OK) {
        g_pred_create_err = p->err;
        eprop_predictor_destroy(p);
        return s;
    }
    *out = p;
    return EPROP_OK;
}

extern "C" int64_t eprop_predictor_num_params(const eprop_predictor *p) { return p ? p->n_params : 0; }

static Layout layout_of(eprop_predictor *p) {
    Layout L{};
    const int I[3] = {p->n_in, p->hidden, p->hidden}, O[3] = {p->hidden, p->hidden, p->n_out};
    for (int l = 0; l < 3; ++l) {
        L.I[l] = I[l];
        L.O[l] = O[l];
        L.ld[l] = l == 2 ? p->ldK : p->ldH;
        L.offW[l] = p->off_W[l];
        L.offb[l] = p->off_b[l];
        L.Wh[l] = p->Wh[l];
    }
    return L;
}

static void refresh_weights(eprop_predictor *p) {
    refresh_kernel<<<blocks_for(p->n_params), 256, 0, p->st>>>(layout_of(p), p->params, p->n_params);
}

extern "C" eprop_status eprop_predictor_set_params(eprop_predictor *p, const float *params) {
    if (!p || !params) return EPROP_EINVAL;
    PCK(p, cudaMemcpyAsync(p->params, params, (size_t)p->n_params * 4, cudaMemcpyHostToDevice, p->st));
    PCK(p, cudaMemsetAsync(p->m, 0, (size_t)p->n_params * 4, p->st));
    PCK(p, cudaMemsetAsync(p->v, 0, (size_t)p->n_params * 4, p->st));
    p->adam_t = 0;
    refresh_weights(p);
    PCK(p, cudaGetLastError());
    PCK(p, cudaStreamSynchronize(p->st));
    return EPROP_OK;
}

// forward (and in training the deltas, the loss and the bias gradients) on x
// already on the device; leaves Y in p->Y and returns the number of row tiles
static int issue_mlp(eprop_predictor *p, const float *x, const float *e, int rows, cudaStream_t st) {
    Mlp a{};
    a.rows = rows; a.I = p->n_in; a.H = p->hidden; a.K = p->n_out;
    a.ldX = p->ldX; a.ldH = p->ldH; a.ldK = p->ldK;
    a.x = x; a.scale = p->in_scale; a.e = e;
    a.b1 = p->params + p->off_b[0]; a.b2 = p->params + p->off_b[1]; a.b3 = p->params + p->off_b[2];
    a.W1 = p->Wh[0]; a.W2 = p->Wh[1]; a.W3 = p->Wh[2];
    a.Xh = p->Xh; a.H1h = p->H1h; a.H2h = p->H2h; a.dYh = p->dYh; a.dA2h = p->dA2h; a.dA1h = p->dA1h;
    a.A1 = p->A1; a.A2 = p->A2; a.Y = p->Y; a.bpart = p->bpart; a.lpart = p->lpart;
    a.inv = 1.0f / (float)rows;
    const bool train = e != nullptr;
    // 32-row tiles once 16-row tiles fill the SMs; four ring stages where they
    // fit; of several waves of tiles two blocks share an SM where two stages
    // allow it (65,536 rows of 74-256-10: inference 619 -> 448 us).  Narrow
    // layers keep one or two of the eight warps busy: many rows of them run in
    // blocks of two warps, many to an SM (65,536 rows of 74-64-10: 415 -> 266 us)
    a.stages = 4;
    const int cols = mlp_cols(a.H, a.K);
    const bool narrow = cols <= kNarrowThreads && rows > 32 * p->sm_count;
    int mt = rows > 16 * p->sm_count && cols > 128 ? 2 : 1;
    if (mlp_smem(a, mt, train) > (size_t)kMlpSmemMax) mt = 1;
    const int tiles = (rows + 16 * mt - 1) / (16 * mt);
    while (a.stages > 2 && mlp_smem(a, mt, train) > (size_t)kMlpSmemMax) --a.stages;
    Mlp two = a;
    two.stages = 2;
    if (narrow) a.stages = 2;
    else if (tiles > p->sm_count && mlp_smem(two, mt, train) <= (size_t)kMlpSmemMax / 2)
        while (mlp_smem(a, mt, train) > (size_t)kMlpSmemMax / 2) --a.stages;
    const size_t sm = mlp_smem(a, mt, train);
    if (narrow) {
        if (train) mlp_kernel<1, true, kNarrowThreads><<<tiles, kNarrowThreads, sm, st>>>(a);
        else mlp_kernel<1, false, kNarrowThreads><<<tiles, kNarrowThreads, sm, st>>>(a);
    } else if (train) {
        if (mt == 2) mlp_kernel<2, true><<<tiles, kMlpThreads, sm, st>>>(a);
        else mlp_kernel<1, true><<<tiles, kMlpThreads, sm, st>>>(a);
    } else {
        if (mt == 2) mlp_kernel<2, false><<<tiles, kMlpThreads, sm, st>>>(a);
        else mlp_kernel<1, false><<<tiles, kMlpThreads, sm, st>>>(a);
    }
    p->rows = rows;
    return tiles;
}

static void issue_forward(eprop_predictor *p, const float *x, int rows, cudaStream_t st) {
    issue_mlp(p, x, nullptr, rows, st);
}

const float *predictor_issue_forward(eprop_predictor *p, const float *x_dev, int rows, cudaStream_t st) {
    issue_forward(p, x_dev, rows, st);
    return p->Y;
}

void predictor_dims(const eprop_predictor *p, int *n_in, int *n_out, int *max_rows) {
    *n_in = p->n_in;
    *n_out = p->n_out;
    *max_rows = p->max_rows;
}

extern "C" eprop_status eprop_predictor_forward(eprop_predictor *p, const float *x, int32_t rows, float *y,
                                                int32_t is_device) {
    if (!p || !x || !y) return EPROP_EINVAL;
    if (rows < 1 || rows > p->max_rows) return pfail(p, EPROP_EINVAL, "rows out of range");
    const float *xd = x;
    if (!is_device) {
        PCK(p, cudaMemcpyAsync(p->xin, x, (size_t)rows * p->n_in * 4, cudaMemcpyHostToDevice, p->st));
        xd = p->xin;
    }
    issue_forward(p, xd, rows, p->st);
    PCK(p, cudaGetLastError());
    PCK(p, cudaMemcpyAsync(y, p->Y, (size_t)rows * p->n_out * 4,
                           is_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, p->st));
    if (!is_device) PCK(p, cudaStreamSynchronize(p->st));
    return EPROP_OK;
}

extern "C" eprop_status eprop_predictor_train_step(eprop_predictor *p, const float *x, const float *e,
                                                   int32_t rows, float lr, float *loss_out, int32_t is_device) {
    if (!p || !x || !e) return EPROP_EINVAL;
    if (rows < 1 || rows > p->max_rows) return pfail(p, EPROP_EINVAL, "rows out of range");
    const int H = p->hidden, K = p->n_out, I = p->n_in;
    const float *xd = x, *ed = e;
    if (!is_device) {
        PCK(p, cudaMemcpyAsync(p->xin, x, (size_t)rows * I * 4, cudaMemcpyHostToDevice, p->st));
        PCK(p, cudaMemcpyAsync(p->ein, e, (size_t)rows * K * 4, cudaMemcpyHostToDevice, p->st));
        xd = p->xin;
        ed = p->ein;
    }
    const int tiles = issue_mlp(p, xd, ed, rows, p->st);
    Dw d{};
    d.rows = rows;
    const bf16 *A[3] = {p->Xh, p->H1h, p->H2h}, *D[3] = {p->dA1h, p->dA2h, p->dYh};
    const int ldA[3] = {p->ldX, p->ldH, p->ldH}, ldD[3] = {p->ldH, p->ldH, p->ldK};
    const int M[3] = {I, H, H}, N[3] = {H, H, K};
    int blocks = 0;
    for (int l = 0; l < 3; ++l) {
        d.A[l] = A[l]; d.D[l] = D[l]; d.ldA[l] = ldA[l]; d.ldD[l] = ldD[l]; d.M[l] = M[l]; d.N[l] = N[l];
        d.out[l] = p->grads + p->off_W[l];
        d.tiles[l] = ((M[l] + kDwTile - 1) / kDwTile) * ((N[l] + kDwTile - 1) / kDwTile);
        blocks += d.tiles[l];
    }
    dw_kernel<<<blocks, kDwThreads, kDwSmem, p->st>>>(d);
    // Adam step
    p->adam_t += 1;
    const float c1 = (float)(1.0 - std::pow(0.9, (double)p->adam_t));
    const float c2 = (float)(1.0 - std::pow(0.999, (double)p->adam_t));
    adam_kernel<<<blocks_for(p->n_params), 256, 0, p->st>>>(layout_of(p), p->params, p->grads, p->m, p->v, p->n_params,
                                                             p->bpart, p->lpart, tiles,
                                                             0.5f / (float)rows, p->loss, lr, c1, c2);
    PCK(p, cudaGetLastError());
    if (loss_out) {
        PCK(p, cudaMemcpyAsync(loss_out, p->loss, 4, cudaMemcpyDeviceToHost, p->st));
        PCK(p, cudaStreamSynchronize(p->st));
    }
    return EPROP_OK;
}

extern "C" eprop_status eprop_predictor_read(eprop_predictor *p, int32_t which, float *dst, int64_t count) {
    if (!p || !dst) return EPROP_EINVAL;
    const long long R = p->rows, H = p->hidden, K = p->n_out;
    const float *srcF = nullptr;
    const bf16 *srcH = nullptr;
    int ld = p->ldH, cols = p->hidden;
    long long n = 0;
    switch (which) {
        case 0: srcF = p->params; n = p->n_params; break;
        case 1: srcF = p->grads; n = p->n_params; break;
        case 2: srcF = p->A1; n = R * H; break;
        case 3: srcH = p->H1h; n = R * H; break;
        case 4: srcF = p->A2; n = R * H; break;
        case 5: srcH = p->H2h; n = R * H; break;
        case 6: srcF = p->Y; n = R * K; break;
        case 7: srcH = p->dYh; n = R * K; ld = p->ldK; cols = p->n_out; break;
        case 8: srcH = p->dA2h; n = R * H; break;
        case 9: srcH = p->dA1h; n = R * H; break;
        case 10: srcF = p->m; n = p->n_params; break;
        case 11: srcF = p->v; n = p->n_params; break;
        case 12: srcH = p->Xh; n = R * p->n_in; ld = p->ldX; cols = p->n_in; break;
        default: return pfail(p, EPROP_EINVAL, "unknown buffer");
    }
    if (count < n) return pfail(p, EPROP_EINVAL, "destination too small");
    if (srcH) {
        bf16_to_float_kernel<<<blocks_for(n), 256, 0, p->st>>>(srcH, ld, cols, p->stage, n);
        PCK(p, cudaGetLastError());
        PCK(p, cudaMemcpyAsync(dst, p->stage, (size_t)n * 4, cudaMemcpyDeviceToHost, p->st));
    } else {
        PCK(p, cudaMemcpyAsync(dst, srcF, (size_t)n * 4, cudaMemcpyDeviceToHost, p->st));
    }
    PCK(p, cudaStreamSynchronize(p->st));
    return EPROP_OK;
}

extern "C" eprop_status eprop_predictor_set_input_scale(eprop_predictor *p, const float *scale) {
    if (!p || !scale) return EPROP_EINVAL;
    PCK(p, cudaStreamSynchronize(p->st));
    PCK(p, cudaMemcpy(p->in_scale, scale, (size_t)p->n_in * 4, cudaMemcpyHostToDevice));
    return EPROP_OK;
}

extern "C" eprop_status eprop_predictor_sync(eprop_predictor *p) {
    if (!p) return EPROP_EINVAL;
    PCK(p, cudaStreamSynchronize(p->st));
    PCK(p, cudaGetLastError());
    return EPROP_OK;
}

extern "C" void eprop_predictor_destroy(eprop_predictor *p) {
    if (!p) return;
    if (p->st) cudaStreamSynchronize(p->st);
    for (void *q : p->allocs) cudaFree(q);
    if (p->own_stream && p->st) cudaStreamDestroy(p->st);
    delete p;
}

extern "C" const char *eprop_predictor_last_error(const eprop_predictor *p) {
    return p ? p->err.c_str() : g_pred_create_err.c_str();
}
