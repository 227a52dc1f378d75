// Surrogate network kernels: a multilayer perceptron 5 -> 128 -> 128 -> 128
// -> 128 -> 2 with SiLU on the hidden layers, BF16 weights and FP32
// accumulation, trained with Adam on FP32 master weights (the learned part
// that picks capillary numbers near breakup).
//
// Forward, backward, loss and optimiser are hand-written kernels; a training
// step is two launches (k_net, k_wgrad).  The network is 5e4 multiply-adds per
// sample and pass, so at the sizes it is used at (1e3 to 1e4 samples) a step
// is bound by the latency of its dependent layers and sums, not by
// arithmetic.  All sums are single FP32 chains in a fixed order.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <cuda_bf16.h>
#include <new>
#include <type_traits>

#include <nvtx3/nvToolsExt.h>

#include "../../include/lbm.h"

namespace surr {

constexpr int NLAYER = 5;
constexpr int MAXW = 128;
// Layer widths 5, 128, 128, 128, 128, 2.
__host__ __device__ constexpr int width(int l) { return l == 0 ? 5 : (l == NLAYER ? 2 : MAXW); }

// Parameter offsets in the flat FP32 vector: layer l holds W [fout][fin]
// then b [fout].
__host__ __device__ constexpr int w_off(int l) {
    return l == 0 ? 0 : 6 * MAXW + (l - 1) * (MAXW + 1) * MAXW;
}
__host__ __device__ constexpr int b_off(int l) { return w_off(l) + width(l + 1) * width(l); }
constexpr int NPARAM = b_off(NLAYER - 1) + width(NLAYER);

__device__ __forceinline__ float silu(float z) { return z / (1.0f + expf(-z)); }
__device__ __forceinline__ float silu_grad(float z) {
    const float s = 1.0f / (1.0f + expf(-z));
    return s * (1.0f + z * (1.0f - s));
}

// ---------------------------------------------------------------------------
// A training step is two launches: k_net (forward and backward through all
// layers, one block per tile of TILE samples) and k_wgrad (weight gradients,
// Adam and the BF16 copies).  Every output is one chain of FMAs in a fixed
// order (over the inputs, the outputs or the samples), so results do not
// depend on the tiling or the grid.
// ---------------------------------------------------------------------------

// Row pitch (BF16 values) of a hidden layer's weights in shared memory: 66
// words, so the 8-byte loads of 16 neighbouring rows fall in distinct banks.
constexpr int WPITCH = 132;

struct NetArgs {
    const float* x;            // inputs [n][5]
    const float* params;       // FP32 masters (the biases are read from here)
    const __nv_bfloat16* wq;   // BF16 weights
    const float *yD, *yB;      // targets (backward only)
    float* out;                // outputs [n][2]
    float* act[NLAYER - 1];    // hidden activations [n][128] (backward only)
    float* gpre[NLAYER];       // loss gradients by pre-activation [n][fout] (backward only)
    double* term;              // loss of each sample [n], or null
    long long* tick;           // Adam step counter to advance, or null
    float* corr;               // Adam's bias corrections of that step [2]
    float b1, b2;
    int n;
};

// Shared memory of a block that carries S samples at a time.
// Rows of samples are padded so that neighbouring rows start in different
// banks (and stay aligned for the pair loads of an even RS).
template <int S, int RS, bool BACKWARD>
struct NetSmem {
    static constexpr int SP = S + (RS % 2 ? 1 - S % 2 : 2);
    alignas(16) float x[MAXW][SP];                      // activations, later gradients, of a layer
    alignas(16) float pre[BACKWARD ? 4 : 1][BACKWARD ? MAXW : 1][SP];  // pre-activations
    alignas(16) __nv_bfloat16 w[3][MAXW * WPITCH];     // hidden layers 1..3
    float w0[MAXW * 5], w4[2 * MAXW];                  // first and last layer
    float b[4 * MAXW + 2];
    float xin[5][S], out[2][S];
};

// Asynchronous copy of 4, 8 or 16 bytes into shared memory; zeros where !ok.
template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst, const void* src, bool ok = true) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    const int have = ok ? BYTES : 0;
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(have) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(d), "l"(src), "n"(BYTES), "r"(have)
                     : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory");
}

__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

// N consecutive floats of shared memory, in pairs where N is even.
template <int N>
__device__ __forceinline__ void lds(const float* p, float (&v)[N]) {
    if constexpr (N % 2 == 0) {
#pragma unroll
        for (int j = 0; j < N; j += 2) {
            const float2 q = *reinterpret_cast<const float2*>(p + j);
            v[j] = q.x, v[j + 1] = q.y;
        }
    } else {
#pragma unroll
        for (int j = 0; j < N; ++j) v[j] = p[j];
    }
}

// All layers of S = NT RO RS / 128 samples in one block, activations in shared
// memory, the weights loaded once per block.  A thread owns RO outputs (RO
// rows of the weights, 8 bytes = 4 inputs per load) and RS samples.
//
// What bounds it: issue and shared-memory bandwidth (a broadcast load returns
// 128 bytes a cycle like any other, so a k costs (2 RO + 4 RS) / 4 cycles of
// the SM for RO RS / 4 cycles of FMAs), at the few warps these sizes give an
// SM.  Measured on GB300: an epoch of 1024 samples (this kernel and k_wgrad)
// 40 us with <2, 2, 256> (8 samples a block, 128 blocks), 44 with <4, 2, 128>
// and <4, 1, 256>, 504 before with one launch per layer and direction (37 since
// k_wgrad's copies got cheaper); a scan
// of 11,776 samples, copies included, 70 us with <4, 5, 512>, 74 with
// <8, 5, 256>, 193 before.
template <int RO, int RS, int NT, bool BACKWARD>
__global__ void __launch_bounds__(NT) k_net(const NetArgs a) {
    constexpr int OG = MAXW / RO;          // threads along the outputs
    constexpr int S = NT / OG * RS;        // samples of the block
    extern __shared__ __align__(16) unsigned char smem_net[];
    auto& M = *reinterpret_cast<NetSmem<S, RS, BACKWARD>*>(smem_net);
    const int t = threadIdx.x;
    if (BACKWARD && a.tick && blockIdx.x == gridDim.x - 1) {
        // the last block has no samples: it counts the Adam step k_wgrad will
        // take (two FP64 powers, a microsecond that nothing else waits for)
        if (t < 2) {
            const double step = (double)(*a.tick + 1);
            a.corr[t] = (float)(1.0 - pow((double)(t ? a.b2 : a.b1), step));
            __syncwarp(3u);
            if (t == 0) *a.tick += 1;
        }
        return;
    }
    const int nblocks = gridDim.x - (BACKWARD && a.tick ? 1 : 0);
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        const __nv_bfloat16* src = a.wq + w_off(l + 1);
        for (int k = t; k < MAXW * 32; k += NT)
            cp_async<8>(&M.w[l][(k >> 5) * WPITCH + 4 * (k & 31)], src + 4 * k);
    }
    cp_async_commit();
    for (int k = t; k < MAXW * 5; k += NT) M.w0[k] = __bfloat162float(a.wq[w_off(0) + k]);
    for (int k = t; k < 2 * MAXW; k += NT) M.w4[k] = __bfloat162float(a.wq[w_off(4) + k]);
    for (int k = t; k < 4 * MAXW + 2; k += NT) M.b[k] = a.params[b_off(k / MAXW) + k % MAXW];

    const int ntile = (a.n + S - 1) / S;
    const int og = t % OG, sb = t / OG * RS;  // outputs og + OG r, samples sb + j
    for (int tile = blockIdx.x; tile < ntile; tile += nblocks) {
        const int s0 = tile * S;
        __syncthreads();  // the previous tile is done
        for (int k = t; k < 5 * S; k += NT) {
            const int s = k / 5, i = k % 5;
            M.xin[i][s] = s0 + s < a.n ? a.x[(int64_t)(s0 + s) * 5 + i] : 0.0f;
        }
        __syncthreads();
        // ---- forward, hidden layers (layer 0 runs while the others' weights arrive)
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            float acc[RO][RS];
#pragma unroll
            for (int r = 0; r < RO; ++r)
#pragma unroll
                for (int j = 0; j < RS; ++j) acc[r][j] = 0.0f;
            if (l == 0) {
#pragma unroll
                for (int i = 0; i < 5; ++i)
#pragma unroll
                    for (int r = 0; r < RO; ++r) {
                        const float w = M.w0[(og + OG * r) * 5 + i];
#pragma unroll
                        for (int j = 0; j < RS; ++j) acc[r][j] = fmaf(M.xin[i][sb + j], w, acc[r][j]);
                    }
            } else {
                const __nv_bfloat16* row = &M.w[l > 0 ? l - 1 : 0][og * WPITCH];
#pragma unroll 4
                for (int k = 0; k < MAXW; k += 4) {
                    uint2 wv[RO];
#pragma unroll
                    for (int r = 0; r < RO; ++r)
                        wv[r] = *reinterpret_cast<const uint2*>(row + OG * r * WPITCH + k);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        float v[RS];
                        lds<RS>(&M.x[k + q][sb], v);
#pragma unroll
                        for (int r = 0; r < RO; ++r) {
                            const uint32_t h = q < 2 ? wv[r].x : wv[r].y;
                            const float w = q & 1 ? bf_hi(h) : bf_lo(h);
#pragma unroll
                            for (int j = 0; j < RS; ++j) acc[r][j] = fmaf(v[j], w, acc[r][j]);
                        }
                    }
                }
                __syncthreads();  // every thread has read the layer's inputs
            }
#pragma unroll
            for (int r = 0; r < RO; ++r) {
                const int o = og + OG * r;
                const float bias = M.b[l * MAXW + o];
#pragma unroll
                for (int j = 0; j < RS; ++j) {
                    const float z = acc[r][j] + bias, y = silu(z);
                    M.x[o][sb + j] = y;
                    if constexpr (BACKWARD) {
                        M.pre[l][o][sb + j] = z;
                        if (s0 + sb + j < a.n) a.act[l][(int64_t)(s0 + sb + j) * MAXW + o] = y;
                    }
                }
            }
            if (l == 0) cp_async_wait<0>();
            __syncthreads();
        }
        // ---- last layer: two outputs per sample
        for (int k = t; k < 2 * S; k += NT) {
            const int oo = k / S, s = k % S;
            float acc = 0.0f;
#pragma unroll 16
            for (int i = 0; i < MAXW; ++i) acc = fmaf(M.x[i][s], M.w4[oo * MAXW + i], acc);
            const float z = acc + M.b[4 * MAXW + oo];
            if constexpr (BACKWARD) M.out[oo][s] = z;
            if (s0 + s < a.n) a.out[(int64_t)(s0 + s) * 2 + oo] = z;
        }
        if constexpr (BACKWARD) {
            __syncthreads();
            // gradient of  mean((D - yD)^2) + mean(BCE(z, yB))  by the outputs
            if (t < S) {
                const int s = s0 + t;
                float g0 = 0.0f, g1 = 0.0f;
                if (s < a.n) {
                    const float d = M.out[0][t] - a.yD[s];
                    const float z = M.out[1][t];
                    const float y = a.yB[s];
                    g0 = 2.0f * d / a.n;
                    g1 = (1.0f / (1.0f + expf(-z)) - y) / a.n;
                    a.gpre[4][2 * (int64_t)s] = g0;
                    a.gpre[4][2 * (int64_t)s + 1] = g1;
                    if (a.term) {
                        const double bce =
                            fmax((double)z, 0.0) - (double)z * y + log1p(exp(-fabs((double)z)));
                        a.term[s] = (double)d * d + bce;
                    }
                }
                M.out[0][t] = g0;
                M.out[1][t] = g1;
            }
            __syncthreads();
            // gradient by the pre-activations of the last hidden layer, then
            // of the others: RO neighbouring inputs per thread
            static_assert(!BACKWARD || RO == 2 || RO == 4, "one load holds a thread's inputs");
            const int i0 = RO * og;
#pragma unroll
            for (int l = 4; l > 0; --l) {
                float acc[RO][RS];
#pragma unroll
                for (int r = 0; r < RO; ++r)
#pragma unroll
                    for (int j = 0; j < RS; ++j) acc[r][j] = 0.0f;
                if (l == 4) {
#pragma unroll
                    for (int k = 0; k < 2; ++k)
#pragma unroll
                        for (int r = 0; r < RO; ++r)
#pragma unroll
                            for (int j = 0; j < RS; ++j)
                                acc[r][j] = fmaf(M.out[k][sb + j], M.w4[k * MAXW + i0 + r], acc[r][j]);
                } else {
                    const __nv_bfloat16* col = &M.w[l < 4 ? l - 1 : 0][i0];
#pragma unroll 16
                    for (int k = 0; k < MAXW; ++k) {
                        float w[RO];
                        if constexpr (RO == 4) {
                            const uint2 wv = *reinterpret_cast<const uint2*>(col + k * WPITCH);
                            w[2] = bf_lo(wv.y), w[3] = bf_hi(wv.y);
                            w[0] = bf_lo(wv.x), w[1] = bf_hi(wv.x);
                        } else {
                            const uint32_t wv = *reinterpret_cast<const uint32_t*>(col + k * WPITCH);
                            w[0] = bf_lo(wv), w[1] = bf_hi(wv);
                        }
                        float g[RS];
                        lds<RS>(&M.x[k][sb], g);
#pragma unroll
                        for (int r = 0; r < RO; ++r)
#pragma unroll
                            for (int j = 0; j < RS; ++j) acc[r][j] = fmaf(g[j], w[r], acc[r][j]);
                    }
                    __syncthreads();  // every thread has read the layer's gradients
                }
#pragma unroll
                for (int j = 0; j < RS; ++j) {
#pragma unroll
                    for (int r = 0; r < RO; ++r) {
                        acc[r][j] *= silu_grad(M.pre[l - 1][i0 + r][sb + j]);
                        M.x[i0 + r][sb + j] = acc[r][j];
                    }
                    if (s0 + sb + j < a.n) {
                        float* g = a.gpre[l - 1] + (int64_t)(s0 + sb + j) * MAXW + i0;
#pragma unroll
                        for (int r = 0; r < RO; r += 2)
                            *reinterpret_cast<float2*>(g + r) = make_float2(acc[r][j], acc[r + 1][j]);
                    }
                }
                __syncthreads();
            }
        }
    }
}

// Weight gradients gW[o][i] = sum_s gpre[s][o] in[s][i], gb[o] = sum_s gpre[s][o],
// and (ADAM) the Adam update with bias correction of the same weights and
// their BF16 copies, by the threads that hold the sums.
//
// One warp per WO x WI tile of one layer's weights, 2 x 2 weights per thread;
// the samples pass through a ring of WST shared-memory chunks of WCH samples
// filled by cp.async.  Each sum is one chain over the samples in order, so at
// 1024 samples the chain (4 cycles a sample) and the shared-memory reads (4
// cycles a sample and warp) bound the kernel, and small tiles are what keeps
// all SMs busy: 408 warps, about one per scheduler.
constexpr int WO = 16, WI = 8, WCH = 64, WST = 4;

struct WgradArgs {
    const float* in[NLAYER];    // inputs of each layer [n][fin]
    const float* gpre[NLAYER];  // gradients by its pre-activations [n][fout]
    float *grads, *params, *m, *v;
    __nv_bfloat16* wq;
    const float* corr;          // Adam's bias corrections
    float lr, b1, b2, eps;
    int n;
};

// Blocks of layer l: ceil(fout / WO) x ceil(fin / WI), layer after layer.
__host__ __device__ constexpr int wg_tiles(int l) {
    return ((width(l + 1) + WO - 1) / WO) * ((width(l) + WI - 1) / WI);
}
constexpr int WG_BLOCKS = wg_tiles(0) + wg_tiles(1) + wg_tiles(2) + wg_tiles(3) + wg_tiles(4);

// A whole chunk of one operand, W columns of rows of WIDTH floats: what differs
// between a thread's copies is an immediate.  With the row, the column and the
// bounds worked out for each copy they were a third of the kernel's instructions
// (64 epochs of 1024 samples 2.70 ms, now 2.34).
// Columns beyond a narrow layer stay the zeros they were set to at the start.
template <int W, int WIDTH>
__device__ __forceinline__ void load_chunk(float* dst, const float* src, int t) {
    if constexpr (WIDTH >= MAXW) {
        constexpr int PER = W / 4, STEP = 32 / PER;
        dst += t / PER * W + 4 * (t % PER);
        src += t / PER * WIDTH + 4 * (t % PER);
#pragma unroll
        for (int i = 0; i < WCH / STEP; ++i) cp_async<16>(dst + i * STEP * W, src + i * STEP * WIDTH);
    } else {
        constexpr int PER = WIDTH <= 2 ? 2 : 8, STEP = 32 / PER;
        dst += t / PER * W + t % PER;
        src += t / PER * WIDTH + t % PER;
        if (t % PER < WIDTH)
#pragma unroll
            for (int i = 0; i < WCH / STEP; ++i) cp_async<4>(dst + i * STEP * W, src + i * STEP * WIDTH);
    }
}

template <bool ADAM>
__global__ void __launch_bounds__(32) k_wgrad(const WgradArgs a) {
    __shared__ __align__(16) float sg[WST][WCH][WO], sx[WST][WCH][WI];
    int l = 0, tile = blockIdx.x;
    while (tile >= wg_tiles(l)) tile -= wg_tiles(l++);
    const int fin = width(l), fout = width(l + 1);
    const int ni = (fin + WI - 1) / WI;
    const int o0 = tile / ni * WO, i0 = tile % ni * WI;
    const float *in = a.in[l], *gp = a.gpre[l];
    const int t = threadIdx.x;
    if (fout < WO || fin < WI) {
        for (int k = t; k < WST * WCH * WO; k += 32) (&sg[0][0][0])[k] = 0.0f;
        for (int k = t; k < WST * WCH * WI; k += 32) (&sx[0][0][0])[k] = 0.0f;
        __syncwarp();
    }
    // The last, partial chunk of one operand: W columns from col0 of rows of `width` floats.
    // Samples beyond n and columns beyond the layer are zeros (their copies
    // read nothing; the source address stays inside the buffer).
    auto load_one = [&](float* dst, int W, const float* src, int width, int col0, int c) {
        const int left = a.n - c * WCH;
        src += (int64_t)c * WCH * width;
        if (width >= MAXW) {
            const int per = W / 4;
            for (int k = t; k < WCH * per; k += 32) {
                const int s = k / per, q = 4 * (k % per);
                const bool ok = s < left;
                cp_async<16>(dst + s * W + q, ok ? src + (int64_t)s * width + col0 + q : src, ok);
            }
        } else {
            for (int k = t; k < WCH * W; k += 32) {
                const int s = k / W, q = k % W;
                const bool ok = s < left && q < width;
                cp_async<4>(dst + s * W + q, ok ? src + (int64_t)s * width + q : src, ok);
            }
        }
    };
    const int nchunk = (a.n + WCH - 1) / WCH;
    auto load = [&](int c) {
        float *dg = &sg[c % WST][0][0], *dx = &sx[c % WST][0][0];
        if ((c + 1) * WCH <= a.n) {
            const float *g = gp + (int64_t)c * WCH * fout + o0, *x = in + (int64_t)c * WCH * fin + i0;
            if (fout == MAXW) load_chunk<WO, MAXW>(dg, g, t);
            else load_chunk<WO, width(NLAYER)>(dg, g, t);
            if (fin == MAXW) load_chunk<WI, MAXW>(dx, x, t);
            else load_chunk<WI, width(0)>(dx, x, t);
        } else if (c < nchunk) {
            load_one(dg, WO, gp, fout, o0, c);
            load_one(dx, WI, in, fin, i0, c);
        }
        cp_async_commit();
    };
    const int oi = 2 * (t / 4), ig = 2 * (t % 4);  // outputs o0 + oi, + 1; inputs i0 + ig, + 1
#pragma unroll
    for (int c = 0; c < WST - 1; ++c) load(c);
    float acc[2][2] = {{0.0f, 0.0f}, {0.0f, 0.0f}}, accb[2] = {0.0f, 0.0f};
    auto sum = [&](auto bias) {
        for (int c = 0; c < nchunk; ++c) {
            cp_async_wait<WST - 2>();
            __syncwarp();
            load(c + WST - 1);  // into the chunk read before this one
            const float(*pg)[WO] = sg[c % WST];
            const float(*px)[WI] = sx[c % WST];
#pragma unroll 16
            for (int s = 0; s < WCH; ++s) {
                const float2 g = *reinterpret_cast<const float2*>(&pg[s][oi]);
                const float2 x = *reinterpret_cast<const float2*>(&px[s][ig]);
                acc[0][0] = fmaf(g.x, x.x, acc[0][0]);
                acc[0][1] = fmaf(g.x, x.y, acc[0][1]);
                acc[1][0] = fmaf(g.y, x.x, acc[1][0]);
                acc[1][1] = fmaf(g.y, x.y, acc[1][1]);
                if constexpr (decltype(bias)::value) {
                    accb[0] += g.x;
                    accb[1] += g.y;
                }
            }
            __syncwarp();
        }
    };
    if (i0 == 0) sum(std::true_type{});
    else sum(std::false_type{});
    const float c1 = ADAM ? a.corr[0] : 1.0f, c2 = ADAM ? a.corr[1] : 1.0f;
    auto finish = [&](int k, float gk) {
        if constexpr (!ADAM) {
            a.grads[k] = gk;
        } else {
            // (written out: 64 steps amplify another rounding of these two to 1e-4)
            const float mk = __fmaf_rn(1.0f - a.b1, gk, __fmul_rn(a.b1, a.m[k]));
            const float vk = __fmaf_rn(__fmul_rn(1.0f - a.b2, gk), gk, __fmul_rn(a.b2, a.v[k]));
            a.m[k] = mk;
            a.v[k] = vk;
            const float mh = mk / c1, vh = vk / c2;
            const float p = a.params[k] - a.lr * mh / (sqrtf(vh) + a.eps);
            a.params[k] = p;
            a.wq[k] = __float2bfloat16_rn(p);
        }
    };
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int o = o0 + oi + e;
        if (o >= fout) continue;
        if (i0 + ig < fin) finish(w_off(l) + o * fin + i0 + ig, acc[e][0]);
        if (i0 + ig + 1 < fin) finish(w_off(l) + o * fin + i0 + ig + 1, acc[e][1]);
        if (i0 == 0 && ig == 0) finish(b_off(l) + o, accb[e]);
    }
}

// The mean of the samples' losses (one block, fixed-order reduction).
__global__ void k_loss(const double* __restrict__ term, int n, double* __restrict__ loss) {
    __shared__ double red[256];
    double acc = 0.0;
    for (int s = threadIdx.x; s < n; s += blockDim.x) acc += term[s];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *loss = red[0] / n;
}

// BF16 copies of the parameters.
__global__ void k_to_bf16(const float* __restrict__ p, __nv_bfloat16* __restrict__ q, int count) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < count) q[k] = __float2bfloat16_rn(p[k]);
}

}  // namespace surr

using namespace surr;

struct surr_ctx {
    float* params = nullptr;          // FP32 master parameters (flat)
    __nv_bfloat16* wq = nullptr;      // BF16 copies (flat, same offsets)
    float* grads = nullptr;
    float* m = nullptr;
    float* v = nullptr;
    long long* adam_t = nullptr;      // Adam steps taken (device counter)
    float* corr = nullptr;            // bias corrections of the current Adam step [2]
    int sms = 0;
    int cap = 0;                      // samples the batch buffers hold
    float* x = nullptr;               // inputs [cap][5]
    float* out = nullptr;             // outputs [cap][2]
    float* act[NLAYER - 1] = {};      // hidden activations [cap][128]
    float* gpre[NLAYER] = {};         // gradients by pre-activation [cap][fout]
    float* yD = nullptr;
    float* yB = nullptr;
    double* term = nullptr;           // loss of each sample [cap]
    double* loss = nullptr;
    cudaStream_t stream = nullptr;
};

namespace {

int fail(cudaError_t e) {
    if (e == cudaSuccess) return LBM_OK;
    cudaGetLastError();
    return LBM_ERR_CUDA;
}

void free_batch(surr_ctx* c) {
    cudaFree(c->x);
    cudaFree(c->out);
    for (int l = 0; l < NLAYER - 1; ++l) {
        cudaFree(c->act[l]);
        c->act[l] = nullptr;
    }
    for (int l = 0; l < NLAYER; ++l) {
        cudaFree(c->gpre[l]);
        c->gpre[l] = nullptr;
    }
    cudaFree(c->yD);
    cudaFree(c->yB);
    cudaFree(c->term);
    c->x = c->out = c->yD = c->yB = nullptr;
    c->term = nullptr;
    c->cap = 0;
}

int ensure_batch(surr_ctx* c, int n) {
    if (n <= c->cap) return LBM_OK;
    free_batch(c);
    const size_t m = (size_t)n;
    bool ok = cudaMalloc(&c->x, sizeof(float) * m * width(0)) == cudaSuccess &&
              cudaMalloc(&c->out, sizeof(float) * m * 2) == cudaSuccess &&
              cudaMalloc(&c->yD, sizeof(float) * m) == cudaSuccess &&
              cudaMalloc(&c->yB, sizeof(float) * m) == cudaSuccess &&
              cudaMalloc(&c->term, sizeof(double) * m) == cudaSuccess;
    for (int l = 0; l < NLAYER - 1 && ok; ++l)
        ok = cudaMalloc(&c->act[l], sizeof(float) * m * MAXW) == cudaSuccess;
    for (int l = 0; l < NLAYER && ok; ++l)
        ok = cudaMalloc(&c->gpre[l], sizeof(float) * m * width(l + 1)) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        free_batch(c);
        return LBM_ERR_NOMEM;
    }
    c->cap = n;
    return LBM_OK;
}

void refresh_bf16(surr_ctx* c) {
    k_to_bf16<<<(NPARAM + 255) / 256, 256, 0, c->stream>>>(c->params, c->wq, NPARAM);
}

constexpr float ADAM_B1 = 0.9f, ADAM_B2 = 0.999f, ADAM_EPS = 1e-8f;
constexpr int TRAIN_RO = 2, TRAIN_RS = 2, TRAIN_NT = 256;
constexpr int TRAIN_S = TRAIN_NT * TRAIN_RO / MAXW * TRAIN_RS;  // samples a block: 8
constexpr int PRED_RO = 4, PRED_NT = 512;
constexpr int PRED_SG = PRED_NT * PRED_RO / MAXW;
using TrainSmem = NetSmem<TRAIN_S, TRAIN_RS, true>;
template <int RS>
using PredSmem = NetSmem<PRED_SG * RS, RS, false>;

// Calls f with the samples per thread of an inference launch, 1 to 5, as a
// compile-time constant: the fewest that let one wave of blocks (one per SM
// by shared memory) take all n samples; beyond that (12,160 samples on 152
// SMs) blocks walk several tiles of 80.
template <class F>
auto with_pred_rs(int n, int sms, F&& f) {
    using std::integral_constant;
    const int per = (n + sms - 1) / sms;
    if (per <= 1 * PRED_SG) return f(integral_constant<int, 1>{});
    if (per <= 2 * PRED_SG) return f(integral_constant<int, 2>{});
    if (per <= 3 * PRED_SG) return f(integral_constant<int, 3>{});
    if (per <= 4 * PRED_SG) return f(integral_constant<int, 4>{});
    return f(integral_constant<int, 5>{});
}

cudaError_t configure_net() {
    cudaError_t e = cudaFuncSetAttribute(k_net<TRAIN_RO, TRAIN_RS, TRAIN_NT, true>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(TrainSmem));
    for (int n = PRED_SG; n <= 5 * PRED_SG && e == cudaSuccess; n += PRED_SG)
        e = with_pred_rs(n, 1, [](auto R) {
            return cudaFuncSetAttribute(k_net<PRED_RO, R(), PRED_NT, false>,
                                        cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)sizeof(PredSmem<R()>));
        });
    return e;
}

// The network over the n samples in the buffers: outputs, and (backward) the
// activations and gradients k_wgrad reads, the samples' losses, and the count
// of the Adam step that follows.
void run_net(surr_ctx* c, int n, bool backward, bool loss, bool tick) {
    NetArgs a{};
    a.x = c->x;
    a.params = c->params;
    a.wq = c->wq;
    a.yD = c->yD;
    a.yB = c->yB;
    a.out = c->out;
    for (int l = 0; l < NLAYER - 1; ++l) a.act[l] = c->act[l];
    for (int l = 0; l < NLAYER; ++l) a.gpre[l] = c->gpre[l];
    a.term = loss ? c->term : nullptr;
    a.tick = tick ? c->adam_t : nullptr;
    a.corr = c->corr;
    a.b1 = ADAM_B1;
    a.b2 = ADAM_B2;
    a.n = n;
    auto blocks = [&](int samples) { return std::min((n + samples - 1) / samples, c->sms); };
    if (backward)
        k_net<TRAIN_RO, TRAIN_RS, TRAIN_NT, true>
            <<<blocks(TRAIN_S) + (tick ? 1 : 0), TRAIN_NT, sizeof(TrainSmem), c->stream>>>(a);
    else
        with_pred_rs(n, c->sms, [&](auto R) {
            k_net<PRED_RO, R(), PRED_NT, false>
                <<<blocks(PRED_SG * R()), PRED_NT, sizeof(PredSmem<R()>), c->stream>>>(a);
            return 0;
        });
    if (loss) k_loss<<<1, 256, 0, c->stream>>>(c->term, n, c->loss);
}

// Weight gradients of the n samples run_net left in the buffers: into
// c->grads, or (adam) straight into an Adam step.
void run_wgrad(surr_ctx* c, int n, bool adam, float lr) {
    WgradArgs a{};
    for (int l = 0; l < NLAYER; ++l) {
        a.in[l] = l == 0 ? c->x : c->act[l - 1];
        a.gpre[l] = c->gpre[l];
    }
    a.grads = c->grads;
    a.params = c->params;
    a.m = c->m;
    a.v = c->v;
    a.wq = c->wq;
    a.corr = c->corr;
    a.lr = lr;
    a.b1 = ADAM_B1;
    a.b2 = ADAM_B2;
    a.eps = ADAM_EPS;
    a.n = n;
    if (adam)
        k_wgrad<true><<<WG_BLOCKS, 32, 0, c->stream>>>(a);
    else
        k_wgrad<false><<<WG_BLOCKS, 32, 0, c->stream>>>(a);
}

int upload_batch(surr_ctx* c, const float* X, const float* yD, const float* yB, int n) {
    int rc = ensure_batch(c, n);
    if (rc != LBM_OK) return rc;
    cudaError_t e = cudaMemcpyAsync(c->x, X, sizeof(float) * n * width(0), cudaMemcpyHostToDevice,
                                    c->stream);
    if (e == cudaSuccess && yD)
        e = cudaMemcpyAsync(c->yD, yD, sizeof(float) * n, cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess && yB)
        e = cudaMemcpyAsync(c->yB, yB, sizeof(float) * n, cudaMemcpyHostToDevice, c->stream);
    return fail(e);
}

// The body of surr_train (arguments checked).
int train_epochs(surr_ctx* c, const float* X, const float* yD, const float* yB, int n, int epochs,
                 float lr, double* loss_out) {
    int rc = upload_batch(c, X, yD, yB, n);
    if (rc != LBM_OK) return rc;
    for (int ep = 0; ep < epochs; ++ep) {
        run_net(c, n, true, false, true);
        run_wgrad(c, n, true, lr);
    }
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess && loss_out) {
        // loss of the parameters after the last update
        run_net(c, n, true, true, false);
        e = cudaMemcpyAsync(loss_out, c->loss, sizeof(double), cudaMemcpyDeviceToHost, c->stream);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    return fail(e);
}

}  // namespace

extern "C" {

int32_t surr_param_count(void) { return NPARAM; }

int surr_create(uint64_t seed, void* stream, surr_ctx** out) {
    if (!out) return LBM_ERR_INVALID_ARG;
    *out = nullptr;
    surr_ctx* c = new (std::nothrow) surr_ctx();
    if (!c) return LBM_ERR_NOMEM;
    c->stream = (cudaStream_t)stream;
    const size_t pb = sizeof(float) * NPARAM;
    if (cudaMalloc(&c->params, pb) != cudaSuccess || cudaMalloc(&c->grads, pb) != cudaSuccess ||
        cudaMalloc(&c->m, pb) != cudaSuccess || cudaMalloc(&c->v, pb) != cudaSuccess ||
        cudaMalloc(&c->wq, sizeof(__nv_bfloat16) * NPARAM) != cudaSuccess ||
        cudaMalloc(&c->loss, sizeof(double)) != cudaSuccess ||
        cudaMalloc(&c->corr, sizeof(float) * 2) != cudaSuccess ||
        cudaMalloc(&c->adam_t, sizeof(long long)) != cudaSuccess) {
        cudaGetLastError();
        surr_destroy(c);
        return LBM_ERR_NOMEM;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        configure_net() != cudaSuccess) {
        cudaGetLastError();
        surr_destroy(c);
        return LBM_ERR_CUDA;
    }
    // He initialisation W ~ N(0, 2 / fan_in), b = 0, from a seeded host
    // generator (SplitMix64, Steele, Lea and Flood 2014, and the Box-Muller
    // transform) so that runs are reproducible
    float* host = new (std::nothrow) float[NPARAM];
    if (!host) {
        surr_destroy(c);
        return LBM_ERR_NOMEM;
    }
    uint64_t st = seed;
    auto next = [&]() {
        uint64_t z = (st += 0x9E3779B97F4A7C15ull);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        return z ^ (z >> 31);
    };
    auto uniform = [&]() { return ((next() >> 11) + 0.5) * (1.0 / 9007199254740992.0); };
    for (int l = 0; l < NLAYER; ++l) {
        const double sd = std::sqrt(2.0 / width(l));
        for (int k = 0; k < width(l + 1) * width(l); ++k) {
            const double u1 = uniform(), u2 = uniform();
            host[w_off(l) + k] = (float)(sd * std::sqrt(-2.0 * std::log(u1)) *
                                         std::cos(6.283185307179586 * u2));
        }
        for (int k = 0; k < width(l + 1); ++k) host[b_off(l) + k] = 0.0f;
    }
    const int rc = surr_set_params(c, host);
    delete[] host;
    if (rc != LBM_OK) {
        surr_destroy(c);
        return rc;
    }
    *out = c;
    return LBM_OK;
}

void surr_destroy(surr_ctx* c) {
    if (!c) return;
    if (c->stream) cudaStreamSynchronize(c->stream);
    else cudaDeviceSynchronize();
    free_batch(c);
    cudaFree(c->params);
    cudaFree(c->grads);
    cudaFree(c->m);
    cudaFree(c->v);
    cudaFree(c->wq);
    cudaFree(c->loss);
    cudaFree(c->adam_t);
    cudaFree(c->corr);
    delete c;
}

int surr_set_params(surr_ctx* c, const float* params) {
    if (!c || !params) return LBM_ERR_INVALID_ARG;
    const size_t pb = sizeof(float) * NPARAM;
    cudaError_t e = cudaMemcpyAsync(c->params, params, pb, cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(c->m, 0, pb, c->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(c->v, 0, pb, c->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(c->adam_t, 0, sizeof(long long), c->stream);
    if (e != cudaSuccess) return fail(e);
    refresh_bf16(c);
    return fail(cudaStreamSynchronize(c->stream));
}

int surr_get_params(surr_ctx* c, float* params) {
    if (!c || !params) return LBM_ERR_INVALID_ARG;
    cudaError_t e = cudaMemcpyAsync(params, c->params, sizeof(float) * NPARAM,
                                    cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    return fail(e);
}

int surr_predict(surr_ctx* c, const float* X, int32_t n, float* D_out, float* logit_out) {
    if (!c || !X || n < 1) return LBM_ERR_INVALID_ARG;
    int rc = upload_batch(c, X, nullptr, nullptr, n);
    if (rc != LBM_OK) return rc;
    run_net(c, n, false, false, false);
    float* out = new (std::nothrow) float[2 * (size_t)n];
    if (!out) return LBM_ERR_NOMEM;
    cudaError_t e = cudaMemcpyAsync(out, c->out, sizeof(float) * 2 * n,
                                    cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e == cudaSuccess)
        for (int s = 0; s < n; ++s) {
            if (D_out) D_out[s] = out[2 * s];
            if (logit_out) logit_out[s] = out[2 * s + 1];
        }
    delete[] out;
    return fail(e);
}

int surr_grad(surr_ctx* c, const float* X, const float* yD, const float* yB, int32_t n,
              float* grads, double* loss) {
    if (!c || !X || !yD || !yB || n < 1) return LBM_ERR_INVALID_ARG;
    int rc = upload_batch(c, X, yD, yB, n);
    if (rc != LBM_OK) return rc;
    run_net(c, n, true, loss != nullptr, false);
    if (grads) run_wgrad(c, n, false, 0.0f);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess && grads)
        e = cudaMemcpyAsync(grads, c->grads, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost,
                            c->stream);
    if (e == cudaSuccess && loss)
        e = cudaMemcpyAsync(loss, c->loss, sizeof(double), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    return fail(e);
}

int surr_train(surr_ctx* c, const float* X, const float* yD, const float* yB, int32_t n,
               int32_t epochs, float lr, double* loss_out) {
    if (!c || !X || !yD || !yB || n < 1 || epochs < 0 || !(lr > 0.0f)) return LBM_ERR_INVALID_ARG;
    nvtxRangePushA("surr_train");
    const int rc = train_epochs(c, X, yD, yB, n, epochs, lr, loss_out);
    nvtxRangePop();
    return rc;
}

}  // extern "C"
