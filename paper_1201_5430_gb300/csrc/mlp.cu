// Selector network of the learned form: forward pass, loss gradient and Adam
// update, FP32 arithmetic on bfloat16 weights.
//
// The paper fixes one truncation number for the whole tree (Sec. 5 names
// "variable truncation number" among the optimisations it left out); the
// learned form picks one per level.  Network (weights W_k (out x in), row-major,
// stored as bfloat16; biases FP32):
//   h1 = relu(W1 x + b1) 12 -> 64,  h2 = relu(W2 h1 + b2) 64 -> 64,
//   h3 = relu(W3 h2 + b3) 64 -> 64, z = W4 h3 + b4 64 -> 21
// z[0:17] score p = 4 .. 20, z[17:21] score the leaf caps 16, 32, 64, 128.
// Loss: mean cross-entropy of the labelled p rows plus mean cross-entropy of the
// labelled leaf rows; gradients by the chain rule through the same layers.
// The network is tiny (10,304 weights): blocks of 256 threads over tiles of 8 or 32
// rows, weights and activations in shared memory, FP32 atomics to combine blocks.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "lhv_internal.cuh"

namespace lhv {

namespace {

constexpr int IN = LHV_MLP_IN, HID = LHV_MLP_HIDDEN, OUT = LHV_MLP_OUT, NP = LHV_MLP_NP;
constexpr int THREADS = 256;
// per layer k = 0..3: input / output widths, offsets of W_k and b_k, and the
// (odd, bank-conflict-free) row stride of W_k in shared memory
__host__ __device__ constexpr int din(int k) { return k == 0 ? IN : HID; }
__host__ __device__ constexpr int dout(int k) { return k == 3 ? OUT : HID; }
__host__ __device__ constexpr int w_off(int k) { return k == 0 ? 0 : HID * IN + (k - 1) * HID * HID; }
__host__ __device__ constexpr int b_off(int k) { return k * HID; }
__host__ __device__ constexpr int ldw(int k) { return din(k) + 1; }
__host__ __device__ constexpr int sw_off(int k) { return k == 0 ? 0 : HID * (IN + 1) + (k - 1) * HID * (HID + 1); }
constexpr int SW_TOTAL = HID * (IN + 1) + 2 * HID * (HID + 1) + OUT * (HID + 1);
constexpr int LDA = HID + 4;    // activation rows: 16-byte aligned for the four-wide broadcast reads
constexpr int SPLIT_R = THREADS / HID;  // threads with the same output and different rows

// A tile of R rows.  R = 8 spreads a training batch of a few hundred rows over the chip (one
// row per warp in the loss); R = 32 shares the staged weights and the barriers among more rows.
template <int R>
struct Smem {
    float act[4][R][LDA];  // act[0]: input, act[k]: relu of the output of layer k
    float d[2][R][LDA];    // the gradient flowing back, two layers at a time
    float w[SW_TOTAL];
    float b[LHV_MLP_NB];
    float z[R][OUT + 1];
    float loss;
};

template <int R>
__device__ void stage_weights(Smem<R>& s, const __nv_bfloat16* __restrict__ W, const float* __restrict__ b) {
#pragma unroll
    for (int k = 0; k < 4; ++k)
        for (int e = threadIdx.x; e < dout(k) * din(k); e += THREADS) {
            const int o = e / din(k), i = e - o * din(k);
            s.w[sw_off(k) + o * ldw(k) + i] = __bfloat162float(W[w_off(k) + e]);
        }
    for (int e = threadIdx.x; e < LHV_MLP_NB; e += THREADS) s.b[e] = b[e];
}

// rows r0 .. r0 + nr - 1 (absent rows of the tile read as zero): act[0] <- X, act[1..3] <- relu
// of the layers, z <- logits.  Thread t holds output t % 64 of R / 4 rows: the weight row is
// read once for all of them, the activations come as four-wide broadcasts.
template <int R>
__device__ void forward_rows(Smem<R>& s, const float* __restrict__ X, int64_t r0, int nr) {
    constexpr int RT = R / SPLIT_R;
    for (int e = threadIdx.x; e < R * IN; e += THREADS) {
        const int r = e / IN, i = e - r * IN;
        s.act[0][r][i] = r < nr ? X[(r0 + r) * IN + i] : 0.0f;
    }
    __syncthreads();
    const int o = threadIdx.x % HID, rb = threadIdx.x / HID * RT;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (o < dout(k)) {
            const float* w = s.w + sw_off(k) + o * ldw(k);
            float acc[RT];
#pragma unroll
            for (int r = 0; r < RT; ++r) acc[r] = s.b[b_off(k) + o];
#pragma unroll 4
            for (int i = 0; i < din(k); i += 4) {
                const float w0 = w[i], w1 = w[i + 1], w2 = w[i + 2], w3 = w[i + 3];
#pragma unroll
                for (int r = 0; r < RT; ++r) {
                    const float4 a = *reinterpret_cast<const float4*>(&s.act[k][rb + r][i]);
                    acc[r] = fmaf(w3, a.w, fmaf(w2, a.z, fmaf(w1, a.y, fmaf(w0, a.x, acc[r]))));
                }
            }
#pragma unroll
            for (int r = 0; r < RT; ++r) {
                if (k < 3) s.act[k < 3 ? k + 1 : 0][rb + r][o] = fmaxf(acc[r], 0.0f);
                else s.z[rb + r][o] = acc[r];
            }
        }
        __syncthreads();
    }
}

template <int R>
__global__ void __launch_bounds__(THREADS) k_mlp_forward(int rows, const float* __restrict__ X,
                                                         const __nv_bfloat16* __restrict__ W,
                                                         const float* __restrict__ b, float* __restrict__ Z) {
    extern __shared__ __align__(16) unsigned char raw[];
    Smem<R>& s = *reinterpret_cast<Smem<R>*>(raw);
    stage_weights(s, W, b);
    __syncthreads();
    for (int64_t r0 = (int64_t)blockIdx.x * R; r0 < rows; r0 += (int64_t)gridDim.x * R) {
        const int nr = (int)(rows - r0 < R ? rows - r0 : R);
        forward_rows(s, X, r0, nr);
        for (int e = threadIdx.x; e < nr * OUT; e += THREADS) {
            const int r = e / OUT, o = e - r * OUT;
            Z[(r0 + r) * OUT + o] = s.z[r][o];
        }
        __syncthreads();
    }
}

// Zeroes the outputs of the gradient and counts the labelled rows: every block clears a part,
// block 0 counts (its 1024 threads read the labels of one launch's COUNT_ROWS rows at most in
// COUNT_ROWS / 1024 steps; larger batches are counted by k_mlp_count).
constexpr int COUNT_ROWS = 1 << 15;
__device__ __forceinline__ void warp_sum2(int& a, int& c) {
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        c += __shfl_down_sync(0xffffffffu, c, o);
    }
}

__global__ void __launch_bounds__(1024) k_mlp_begin(int rows, const int* __restrict__ yp, const int* __restrict__ yl,
                                                    float* __restrict__ gW, float* __restrict__ gb,
                                                    float* __restrict__ loss, int* __restrict__ cnt) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < LHV_MLP_NW) gW[i] = 0.0f;
    if (i < LHV_MLP_NB) gb[i] = 0.0f;
    if (blockIdx.x > 0) return;
    __shared__ int sa[32], sc[32];
    int a = 0, c = 0;
    if (rows <= COUNT_ROWS)
        for (int r = threadIdx.x; r < rows; r += blockDim.x) {
            a += yp[r] >= 0;
            c += yl[r] >= 0;
        }
    warp_sum2(a, c);
    if ((threadIdx.x & 31) == 0) {
        sa[threadIdx.x >> 5] = a;
        sc[threadIdx.x >> 5] = c;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        a = sa[threadIdx.x];
        c = sc[threadIdx.x];
        warp_sum2(a, c);
        if (threadIdx.x == 0) {
            cnt[0] = a;
            cnt[1] = c;
            *loss = 0.0f;
        }
    }
}

__global__ void k_mlp_count(int rows, const int* __restrict__ yp, const int* __restrict__ yl, int* __restrict__ cnt) {
    int a = 0, c = 0;
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < rows; r += gridDim.x * blockDim.x) {
        a += yp[r] >= 0;
        c += yl[r] >= 0;
    }
    warp_sum2(a, c);
    if ((threadIdx.x & 31) == 0) {
        if (a) atomicAdd(cnt, a);
        if (c) atomicAdd(cnt + 1, c);
    }
}

// Softmax cross-entropy of one row by one warp: lanes [0, NP) hold the p scores, [NP, OUT) the
// leaf scores; y < 0 leaves that head out.  Writes dz = (softmax - onehot) * scale of every
// score and returns the row's loss (the same value in every lane).
__device__ float xent_row(const float* z, float* dz, int yp, int yl, float sp, float sl) {
    const int lane = threadIdx.x & 31;
    const bool leaf = lane >= NP, live = lane < OUT;
    const float v = live ? z[lane] : -INFINITY;
    float mp = leaf ? -INFINITY : v, ml = leaf ? v : -INFINITY;
    for (int o = 16; o > 0; o >>= 1) {
        mp = fmaxf(mp, __shfl_xor_sync(0xffffffffu, mp, o));
        ml = fmaxf(ml, __shfl_xor_sync(0xffffffffu, ml, o));
    }
    const float e = live ? expf(v - (leaf ? ml : mp)) : 0.0f;
    float ep = leaf ? 0.0f : e, el = leaf ? e : 0.0f;
    for (int o = 16; o > 0; o >>= 1) {
        ep += __shfl_xor_sync(0xffffffffu, ep, o);
        el += __shfl_xor_sync(0xffffffffu, el, o);
    }
    const int y = leaf ? yl : yp;
    if (live)
        dz[lane] = y >= 0 ? (e / (leaf ? el : ep) - ((leaf ? lane - NP : lane) == y ? 1.0f : 0.0f)) * (leaf ? sl : sp)
                          : 0.0f;
    float part = 0.0f;
    if (yp >= 0) part += (logf(ep) + mp - z[yp]) * sp;
    if (yl >= 0) part += (logf(el) + ml - z[NP + yl]) * sl;
    return part;
}

// One block per tile of R rows (persistent over tiles): forward, loss, backward, the weight
// gradients of all its tiles in registers (41 per thread: entry t + 256 j of each layer) and
// one atomic add per weight at the end.  Bound by latency: 800 rows are 49 Mflop.  The earlier
// form (64 rows and 64 threads a block, everything serial over its rows, 13 blocks at 800 rows)
// took 297 us for loss, gradient and Adam where this one takes 44 us.
template <int R>
__global__ void __launch_bounds__(THREADS) k_mlp_grad(int rows, const float* __restrict__ X, const int* __restrict__ yp,
                                                      const int* __restrict__ yl, const __nv_bfloat16* __restrict__ W,
                                                      const float* __restrict__ b, const int* __restrict__ cnt,
                                                      float* __restrict__ gW, float* __restrict__ gb,
                                                      float* __restrict__ loss) {
    extern __shared__ __align__(16) unsigned char raw[];
    Smem<R>& s = *reinterpret_cast<Smem<R>*>(raw);
    constexpr int RT = R / SPLIT_R;
    constexpr int NJ[4] = {3, 16, 16, 6};  // entries of W_k per thread
    const int t = threadIdx.x, col = t % HID, sub = t / HID;
    stage_weights(s, W, b);
    if (t == 0) s.loss = 0.0f;
    const float sp = cnt[0] > 0 ? 1.0f / cnt[0] : 0.0f, sl = cnt[1] > 0 ? 1.0f / cnt[1] : 0.0f;
    float g0[NJ[0]] = {}, g1[NJ[1]] = {}, g2[NJ[2]] = {}, g3[NJ[3]] = {}, gbias = 0.0f;
    float part = 0.0f;
    __syncthreads();
    for (int64_t r0 = (int64_t)blockIdx.x * R; r0 < rows; r0 += (int64_t)gridDim.x * R) {
        const int nr = (int)(rows - r0 < R ? rows - r0 : R);
        forward_rows(s, X, r0, nr);
        for (int r = t >> 5; r < R; r += THREADS / 32) {  // one warp per row; absent rows carry no gradient
            const int a = r < nr ? yp[r0 + r] : -1, c = r < nr ? yl[r0 + r] : -1;
            part += xent_row(s.z[r], s.d[0][r], a, c, sp, sl);
        }
        __syncthreads();
        // gW_k[o][i] += d[r][o] in_k[r][i]; thread t holds the columns i = t % 64, rows o = t / 64 + 4 j
        auto weights = [&](auto& g, int k, const float(*d)[LDA]) {
#pragma unroll 2
            for (int r = 0; r < R; ++r) {
                const float a = s.act[k][r][col];
#pragma unroll
                for (int j = 0; j < (int)(sizeof(g) / sizeof(g[0])); ++j) {
                    const int o = sub + SPLIT_R * j;
                    if (o < dout(k)) g[j] = fmaf(d[r][o], a, g[j]);
                }
            }
        };
        // d_{k-1}[r][i] = (sum_o d[r][o] W_k[o][i]) [layer k's input > 0]
        auto back = [&](int k, const float(*d)[LDA], float(*dn)[LDA]) {
            const float* w = s.w + sw_off(k) + col;
            float acc[RT] = {};
#pragma unroll 4
            for (int o = 0; o < dout(k); ++o) {
                const float wo = w[o * ldw(k)];
#pragma unroll
                for (int r = 0; r < RT; ++r) acc[r] = fmaf(d[sub * RT + r][o], wo, acc[r]);
            }
#pragma unroll
            for (int r = 0; r < RT; ++r)
                dn[sub * RT + r][col] = s.act[k][sub * RT + r][col] > 0.0f ? acc[r] : 0.0f;
        };
        // the bias gradient of layer k belongs to the 64 threads sub == k
        auto bias = [&](int k, const float(*d)[LDA]) {
            if (sub == k && col < dout(k))
                for (int r = 0; r < R; ++r) gbias += d[r][col];
        };
        weights(g3, 3, s.d[0]);
        bias(3, s.d[0]);
        back(3, s.d[0], s.d[1]);
        __syncthreads();
        weights(g2, 2, s.d[1]);
        bias(2, s.d[1]);
        back(2, s.d[1], s.d[0]);
        __syncthreads();
        weights(g1, 1, s.d[0]);
        bias(1, s.d[0]);
        back(1, s.d[0], s.d[1]);
        __syncthreads();
        bias(0, s.d[1]);
#pragma unroll
        for (int j = 0; j < NJ[0]; ++j) {
            const int e = t + THREADS * j, o = e / IN, i = e - o * IN;
            for (int r = 0; r < R; ++r) g0[j] = fmaf(s.d[1][r][o], s.act[0][r][i], g0[j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < NJ[0]; ++j) atomicAdd(gW + t + THREADS * j, g0[j]);
#pragma unroll
    for (int j = 0; j < NJ[1]; ++j) {
        atomicAdd(gW + w_off(1) + t + THREADS * j, g1[j]);
        atomicAdd(gW + w_off(2) + t + THREADS * j, g2[j]);
    }
#pragma unroll
    for (int j = 0; j < NJ[3]; ++j)
        if (sub + SPLIT_R * j < OUT) atomicAdd(gW + w_off(3) + t + THREADS * j, g3[j]);
    if (col < dout(sub)) atomicAdd(gb + b_off(sub) + col, gbias);
    if ((t & 31) == 0 && part != 0.0f) atomicAdd(&s.loss, part);
    __syncthreads();
    if (t == 0 && s.loss != 0.0f) atomicAdd(loss, s.loss);
}

// Adam (Kingma & Ba 2015) on the FP32 master weights, then their bfloat16 copy.
__global__ void k_mlp_adam(float* __restrict__ W32, __nv_bfloat16* __restrict__ W, const float* __restrict__ gW,
                           float* __restrict__ mW, float* __restrict__ vW, float* __restrict__ b,
                           const float* __restrict__ gb, float* __restrict__ mb, float* __restrict__ vb, float c1,
                           float c2, float lr) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    if (i < LHV_MLP_NW) {
        const float g = gW[i];
        const float m = b1 * mW[i] + (1.0f - b1) * g;
        const float v = b2 * vW[i] + (1.0f - b2) * g * g;
        mW[i] = m;
        vW[i] = v;
        const float w = W32[i] - lr * (m / c1) / (sqrtf(v / c2) + eps);
        W32[i] = w;
        W[i] = __float2bfloat16_rn(w);
    } else if (i < LHV_MLP_NW + LHV_MLP_NB) {
        const int j = i - LHV_MLP_NW;
        const float g = gb[j];
        const float m = b1 * mb[j] + (1.0f - b1) * g;
        const float v = b2 * vb[j] + (1.0f - b2) * g * g;
        mb[j] = m;
        vb[j] = v;
        b[j] -= lr * (m / c1) / (sqrtf(v / c2) + eps);
    }
}

// 32-row tiles once they fill the chip, else 8-row tiles (800 rows: 100 blocks against 25)
bool big_tiles(int rows) { return rows >= 152 * 32; }
int blocks_for(int rows, int R) { return std::max(1, std::min((rows + R - 1) / R, 152)); }

template <int R>
cudaError_t forward(cudaStream_t s, int rows, const float* X, const __nv_bfloat16* W, const float* b, float* Z) {
    cudaError_t e = cudaFuncSetAttribute(k_mlp_forward<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(Smem<R>));
    if (e != cudaSuccess) return e;
    k_mlp_forward<R><<<blocks_for(rows, R), THREADS, sizeof(Smem<R>), s>>>(rows, X, W, b, Z);
    return cudaGetLastError();
}

template <int R>
cudaError_t grad(cudaStream_t s, int rows, const float* X, const int* yp, const int* yl, const __nv_bfloat16* W,
                 const float* b, const int* cnt, float* gW, float* gb, float* loss) {
    cudaError_t e = cudaFuncSetAttribute(k_mlp_grad<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(Smem<R>));
    if (e != cudaSuccess) return e;
    k_mlp_grad<R><<<blocks_for(rows, R), THREADS, sizeof(Smem<R>), s>>>(rows, X, yp, yl, W, b, cnt, gW, gb, loss);
    return cudaGetLastError();
}

}  // namespace

cudaError_t mlp_forward(cudaStream_t s, int rows, const float* X, const uint16_t* W, const float* b, float* Z) {
    const __nv_bfloat16* Wb = reinterpret_cast<const __nv_bfloat16*>(W);
    return big_tiles(rows) ? forward<32>(s, rows, X, Wb, b, Z) : forward<8>(s, rows, X, Wb, b, Z);
}

cudaError_t mlp_grad(cudaStream_t s, int rows, const float* X, const int* yp, const int* yl, const uint16_t* W,
                     const float* b, float* gW, float* gb, float* loss, int* cnt) {
    const __nv_bfloat16* Wb = reinterpret_cast<const __nv_bfloat16*>(W);
    k_mlp_begin<<<(LHV_MLP_NW + 1023) / 1024, 1024, 0, s>>>(rows, yp, yl, gW, gb, loss, cnt);
    if (rows > COUNT_ROWS) k_mlp_count<<<152, 256, 0, s>>>(rows, yp, yl, cnt);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return big_tiles(rows) ? grad<32>(s, rows, X, yp, yl, Wb, b, cnt, gW, gb, loss)
                           : grad<8>(s, rows, X, yp, yl, Wb, b, cnt, gW, gb, loss);
}

cudaError_t mlp_adam(cudaStream_t s, float* W32, uint16_t* W, const float* gW, float* mW, float* vW, float* b,
                     const float* gb, float* mb, float* vb, int t, float lr) {
    const float c1 = 1.0f - powf(0.9f, (float)t), c2 = 1.0f - powf(0.999f, (float)t);
    const int n = LHV_MLP_NW + LHV_MLP_NB;
    k_mlp_adam<<<(n + 255) / 256, 256, 0, s>>>(W32, reinterpret_cast<__nv_bfloat16*>(W), gW, mW, vW, b, gb, mb, vb,
                                               c1, c2, lr);
    return cudaGetLastError();
}

}  // namespace lhv
