// Learned warm start: a small 1-D convolutional neural operator that maps the data
// of eq. (1.1) -- u0, f(., t_n) for n = 0..s, alpha, d+, d- -- to a space-time
// initial guess u_1..u_s of the GMRES solve.  It works with sine-series
// coefficients c_j (v(x_i) = sum_j c_j sin(j pi x_i), j = 1..K): the convolution runs
// along the mode index (length K) over channels [c_j(u0), c_j(f(., t_n)) for
// n = 0..s, (alpha-1.5)/0.4, (mean d+ - 1.25)/0.75, (mean d- - 1.25)/0.75, j/K], and
// its s output channels are the coefficients of u_1..u_s, synthesised back to the
// grid.  The paper has no learned component; the solve is still judged by
// its true FP64 residual, and pgmres_solve falls back to the zero guess when the
// predicted guess is worse than zero.
//
// Network: L convolution layers (kernel K, zero padding, same length), ReLU after
// all but the last; parameters flat per layer: W (C_out, C_in, K) then b (C_out).
// Kernels: tiled forward convolution (FP32, or FP16 storage with FP32 accumulation
// for inference), backward-data as the forward kernel on the flipped / transposed
// weights with the ReLU mask fused, backward-weight reduction split over the
// batch, MSE loss gradient and Adam.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "fde_internal.h"
#include "nop_tile.cuh"

namespace fde {

constexpr int CV_KMAX = 7;
constexpr int CV_TP = 16;        // output channels per CTA
constexpr int CV_WARPS = 8;      // warps per CTA, which share the input channels of a chunk
constexpr int CV_LDW = CV_TP + 1;

__device__ __forceinline__ float ldf(const float* p) { return *p; }
__device__ __forceinline__ float ldf(const __half* p) { return __half2float(*p); }
__device__ __forceinline__ void stf(float* p, float v) { *p = v; }
__device__ __forceinline__ void stf(__half* p, float v) { *p = __float2half_rn(v); }

// stage nq channels of a batch of Q (nmax - nq zero rows behind them) from x, their first one in the
// tile's first sample: one warp a channel, lanes along the slots (whose sources do not depend on
// the channel)
template <typename TI>
__device__ __forceinline__ void cv_stage(const TI* __restrict__ x, size_t sample, int nq, int nmax, int x0, int m,
                                         int h, int len, float* s, int ld) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int t = lane; t < len; t += 32) {
        const CvPoint p = cv_slot(x0, m, h, t);
        const TI* src = x + cv_offset(p, sample);
#pragma unroll 4
        for (int c = warp; c < nmax; c += CV_WARPS)
            s[c * ld + t] = p.x >= 0 && c < nq ? ldf(src + (size_t)c * m) : 0.f;
    }
}

// positions of a CTA's tile and input channels of a chunk (conv_kernel)
constexpr int cv_positions(int NL, bool pos) { return 4 * NL * (pos ? CV_WARPS : 1); }
constexpr int cv_channels(int NL, bool pos) { return pos ? 16 : NL == 4 ? 8 * CV_WARPS : 4 * CV_WARPS; }

// y[b][p][x] = bias[p] + sum_q sum_k Wacc(p,q,k) x[b][q][x + k - K/2]
//   TRANS = false: Wacc(p,q,k) = W[p][q][k]            (W: P x Q x K)
//   TRANS = true : Wacc(p,q,k) = W[q][p][K-1-k]        (W: Q x P x K; gradient w.r.t. the input)
// relu: apply max(., 0); mask: multiply by (mask[b][p][x] > 0) (backward through a ReLU).
//
// The layers are small (64 channels, 16 modes, 32 samples: 21 MFLOP), so a launch is bound by
// latency and by how many SMs it reaches.  A CTA takes 16 channels x 4 NL positions of the
// flattened batch; its eight warps split the input channels of a chunk and their partial sums
// are added in a fixed order.  Per layer at that size 9 us forward and 13 backward against 51
// and 45 for a tile of 128 positions of one sample, seven eighths of which were padding.
// KT: the kernel size, or 0 to take it from K (a known size makes the weights' indices cheap).
// POS: the warps take positions of their own instead (32 NL a CTA), for layers of few input channels,
// whose sums are shorter than the addition of eight partial ones.
template <typename TI, typename TW, typename TO, bool TRANS, int NL, int KT, bool POS>
__global__ void __launch_bounds__(32 * CV_WARPS)
conv_kernel(const TI* __restrict__ x, int Q, const TW* __restrict__ W, const float* __restrict__ bias, int P, int Kr,
            int m, long N, int relu, const float* __restrict__ mask, TO* __restrict__ y, int ld) {
    const int K = KT ? KT : Kr;
    constexpr int TN = cv_positions(NL, POS), QC = cv_channels(NL, POS);
    constexpr int CW = POS ? 1 : CV_WARPS;  // warps that share a position's channels
    extern __shared__ float cv_smem[];
    float* s_in = cv_smem;            // [QC][ld]
    float* s_w = cv_smem + QC * ld;   // [QC][K][CV_LDW]
    const long n0 = (long)blockIdx.x * TN;
    const CvTile tile = cv_tile(n0, m);
    const int p0 = blockIdx.y * CV_TP, count = (int)min((long)TN, N - n0);
    const int h = K / 2, len = cv_length(count, tile.x0, m, h);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, pl = lane >> 2;
    const int cw = POS ? 0 : warp, nl = (lane & 3) + (POS ? 4 * NL * warp : 0);  // the warp's channels and positions
    float acc[2][NL];
    int at[NL];
#pragma unroll
    for (int j = 0; j < NL; ++j) {
        acc[0][j] = acc[1][j] = 0.f;
        at[j] = cv_place(min(nl + 4 * j, count - 1), tile.x0, m, h);
    }
    for (int q0 = 0; q0 < Q; q0 += QC) {
        const int nq = min(QC, Q - q0);
        cv_stage(x + ((size_t)tile.b0 * Q + q0) * m, (size_t)Q * m, nq, nq, tile.x0, m, h, len, s_in, ld);
        // 16 threads a row of weights: channel o's (TRANS = false) or input channel c's
        const int row = tid >> 4;
        if (TRANS) {
#pragma unroll 2
            for (int c = row; c < nq; c += 2 * CV_WARPS)
                for (int r = tid & 15; r < CV_TP * K; r += 16) {
                    const int o = r / K, k = r - o * K;
                    s_w[(c * K + K - 1 - k) * CV_LDW + o] =
                        p0 + o < P ? ldf(W + ((size_t)(q0 + c) * P + p0) * K + r) : 0.f;
                }
        } else {
            const TW* wr = W + ((size_t)(p0 + row) * Q + q0) * K;
#pragma unroll 8
            for (int r = tid & 15; r < nq * K; r += 16) s_w[r * CV_LDW + row] = p0 + row < P ? ldf(wr + r) : 0.f;
        }
        __syncthreads();
        for (int c = cw; c < nq; c += CW) {
            const float* in = s_in + c * ld;
            const float* w = s_w + c * K * CV_LDW + 2 * pl;
#pragma unroll
            for (int k = 0; k < (KT ? KT : CV_KMAX); ++k) {
                if (!KT && k >= K) break;
                const float w0 = w[k * CV_LDW], w1 = w[k * CV_LDW + 1];
#pragma unroll
                for (int j = 0; j < NL; ++j) {
                    const float v = in[at[j] + k];
                    acc[0][j] += w0 * v;
                    acc[1][j] += w1 * v;
                }
            }
        }
        __syncthreads();
    }
    // add the warps' partial sums: red[warp][channel][position]
    float* red = cv_smem;
#pragma unroll
    for (int j = 0; j < NL; ++j) {
        red[(cw * CV_TP + 2 * pl) * TN + nl + 4 * j] = acc[0][j];
        red[(cw * CV_TP + 2 * pl + 1) * TN + nl + 4 * j] = acc[1][j];
    }
    __syncthreads();
    for (int e = tid; e < CV_TP * TN; e += 32 * CV_WARPS) {
        const int p = p0 + e / TN, n = e % TN;
        if (p >= P || n >= count) continue;
        float v = 0.f;
#pragma unroll
        for (int w = 0; w < CW; ++w) v += red[w * CV_TP * TN + e];
        if (bias) v += bias[p];
        if (relu) v = fmaxf(v, 0.f);
        const size_t idx = ((size_t)tile.b0 * P + p) * m + cv_offset(cv_position(tile.x0, m, n), (size_t)P * m);
        if (mask && !(mask[idx] > 0.f)) v = 0.f;
        stf(y + idx, v);
    }
}

// db[o] = sum g of one channel, by a CTA of its own: its terms are added in fours in FP32, the rest in
// FP64 and in a fixed order, so db repeats to the bit and its rounding does not grow with the batch.
__device__ __forceinline__ void bias_sum(const float* __restrict__ g, int O, int m, int B, int o,
                                         float* __restrict__ db) {
    __shared__ double red[8];
    const long N = (long)B * m;
    const size_t sample = (size_t)O * m;
    g += (size_t)o * m;
    double v = 0.0;
    for (long n = threadIdx.x; n < N; n += 8 * 256) {
        float s[2] = {0.f, 0.f};
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const long q = n + 256 * j;
            if (q < N) {
                const CvTile at = cv_tile(q, m);
                s[j / 4] += g[at.b0 * sample + at.x0];
            }
        }
        v += (double)s[0];
        v += (double)s[1];
    }
    for (int off = 16; off; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) v += red[w];
        db[o] = (float)v;
    }
}

// dW[o][c][k] += sum_{b in group} sum_x g[b][o][x] a[b][c][x + k - K/2]; one thread per (o, c)
// of a 16 x 16 tile, the flattened positions of the batch split over `groups` of `per` (atomic
// accumulation).  The CTAs behind the groups form the bias gradients db, a channel each (before them
// they cost a large gradient 10 %: fewer of the others start together; with several channels a CTA they
// are the last to finish: 2390 us a gradient at 16 x 2047 positions, 16 channels, with a warp a channel, 640 so).
// 10 us a layer at 64 channels, 16 modes, 32 samples, against 22 (64-position tiles of single
// samples) and 10 for the bias sums in a launch of their own.
constexpr int WG_N = 64;  // positions staged at once
__global__ void __launch_bounds__(256)
conv_wgrad_kernel(const float* __restrict__ g, int O, const float* __restrict__ a, int C, int K, int m, int B,
                  int groups, long per, float* __restrict__ dW, float* __restrict__ db, int ld) {
    extern __shared__ float wg_smem[];
    float* s_g = wg_smem;                  // [16][WG_N + 1]
    float* s_a = wg_smem + 16 * (WG_N + 1);  // [16][ld]
    const int o0 = blockIdx.y * 16, c0 = blockIdx.x * 16;
    if ((int)blockIdx.z >= groups) {
        const int q = (blockIdx.z - groups) * gridDim.x + blockIdx.x;
        if (q < 16 && o0 + q < O) bias_sum(g, O, m, B, o0 + q, db);
        return;
    }
    const int ol = threadIdx.x / 16, cl = threadIdx.x % 16;
    const int h = K / 2;
    float acc[CV_KMAX];
#pragma unroll
    for (int k = 0; k < CV_KMAX; ++k) acc[k] = 0.f;
    const long lo = blockIdx.z * per, total = min((long)B * m, lo + per) - lo;
    CvTile tile = cv_tile(lo, m);
    const size_t sample_g = (size_t)O * m, sample_a = (size_t)C * m;
    g += tile.b0 * sample_g + (size_t)o0 * m;  // the tile's first sample, the CTA's channels
    a += tile.b0 * sample_a + (size_t)c0 * m;
    for (long n0 = 0; n0 < total; n0 += WG_N) {
        const int count = (int)min((long)WG_N, total - n0), len = cv_length(count, tile.x0, m, h);
        {
            const int t = threadIdx.x % WG_N;
            const float* gr = g + cv_offset(cv_position(tile.x0, m, t), sample_g);
#pragma unroll
            for (int r = threadIdx.x / WG_N; r < 16; r += 256 / WG_N)
                s_g[r * (WG_N + 1) + t] = o0 + r < O && t < count ? gr[(size_t)r * m] : 0.f;
        }
        cv_stage(a, sample_a, min(16, C - c0), 16, tile.x0, m, h, len, s_a, ld);
        __syncthreads();
        int x = tile.x0;
        const float* ap = s_a + cl * ld;
        for (int t = 0; t < count; ++t) {
            const float gv = s_g[ol * (WG_N + 1) + t];
#pragma unroll
            for (int k = 0; k < CV_KMAX; ++k)
                if (k < K) acc[k] += gv * ap[k];
            ++ap;
            if (++x == m) {  // the next sample's piece
                x = 0;
                ap += 2 * h;
            }
        }
        const CvPoint next = cv_position(tile.x0, m, WG_N);
        tile.x0 = next.x;
        g += next.d * sample_g;
        a += next.d * sample_a;
        __syncthreads();
    }
    if (o0 + ol < O && c0 + cl < C)
        for (int k = 0; k < K; ++k) atomicAdd(dW + ((size_t)(o0 + ol) * C + c0 + cl) * K + k, acc[k]);
}

// g = 2 (y - t) / N, loss += sum (y - t)^2 / N
__global__ void mse_kernel(const float* __restrict__ y, const float* __restrict__ t, long n, float* __restrict__ g,
                           double* __restrict__ loss) {
    double s = 0.0;
    const double inv = 1.0 / (double)n;
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
        const float d = y[i] - t[i];
        g[i] = (float)(2.0 * d * inv);
        s += (double)d * d;
    }
    for (int off = 16; off; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    __shared__ double part[8];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {  // one atomic a CTA (256 threads)
        for (int w = 1; w < 8; ++w) s += part[w];
        atomicAdd(loss, s * inv);
    }
}

__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m1,
                            float* __restrict__ m2, long n, float lr, float b1, float b2, float eps, float c1,
                            float c2) {
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float a = b1 * m1[i] + (1.f - b1) * gi;
        const float v = b2 * m2[i] + (1.f - b2) * gi * gi;
        m1[i] = a;
        m2[i] = v;
        p[i] -= lr * (a / c1) / (sqrtf(v / c2) + eps);
    }
}

// splitmix64 (Steele, Lea & Flood 2014) on (seed, index) -> uniform in [-1, 1)
__device__ __forceinline__ float splitmix_uniform(unsigned long long seed, unsigned long long i) {
    unsigned long long z = seed + (i + 1) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z = z ^ (z >> 31);
    return (float)((double)(z >> 11) * (1.0 / 9007199254740992.0)) * 2.f - 1.f;
}

__global__ void init_kernel(float* __restrict__ p, long off, long n, float scale, unsigned long long seed) {
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
        p[off + i] = scale * splitmix_uniform(seed, (unsigned long long)(off + i));
}

__global__ void to_half_kernel(const float* __restrict__ a, __half* __restrict__ b, long n) {
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
        b[i] = __float2half_rn(a[i]);
}

// Sine-series coefficients c[r][j] = 2/(m+1) sum_i v_r[i] sin(j pi (i+1)/(m+1)) of
// `rows` grid vectors v_r (stride m), so that v_r[i] = sum_j c[r][j] sin(j pi (i+1)/(m+1))
// on the first modes: one warp per (row, mode).
__global__ void sine_analysis_kernel(const double* __restrict__ v, int rows, int m, int K, float* __restrict__ out,
                                     int out_stride, int out_off) {
    const int lane = threadIdx.x & 31;
    const long w = ((long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (w >= (long)rows * K) return;
    const int r = (int)(w / K), j = (int)(w % K);
    const double* vr = v + (size_t)r * m;
    double c = 0.0;
    for (int i = lane; i < m; i += 32) c += vr[i] * sinpi((double)(j + 1) * (i + 1) / (double)(m + 1));
    for (int off = 16; off; off >>= 1) c += __shfl_xor_sync(0xffffffffu, c, off);
    if (lane == 0) out[(size_t)(out_off + r) * out_stride + j] = (float)(c * (2.0 / (double)(m + 1)));
}

// Scalar channels of the spectral input: (alpha-1.5)/0.4, mean d+, mean d- (normalised), j/K.
__global__ void scalar_channels_kernel(int m, int K, int c0, double alpha, const double* __restrict__ dp,
                                       const double* __restrict__ dm, float* __restrict__ in) {
    __shared__ double sp[256], sm[256];
    double a = 0.0, b = 0.0;
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        a += dp[i];
        b += dm[i];
    }
    sp[threadIdx.x] = a;
    sm[threadIdx.x] = b;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            sp[threadIdx.x] += sp[threadIdx.x + w];
            sm[threadIdx.x] += sm[threadIdx.x + w];
        }
        __syncthreads();
    }
    for (int j = threadIdx.x; j < K; j += blockDim.x) {
        in[(size_t)(c0 + 0) * K + j] = (float)((alpha - 1.5) / 0.4);
        in[(size_t)(c0 + 1) * K + j] = (float)((sp[0] / m - 1.25) / 0.75);
        in[(size_t)(c0 + 2) * K + j] = (float)((sm[0] / m - 1.25) / 0.75);
        in[(size_t)(c0 + 3) * K + j] = (float)(j + 1) / (float)K;
    }
}

// x0[t][i] = sum_j c[t][j] sin(j pi (i+1)/(m+1)): one CTA per time level.
__global__ void sine_synthesis_kernel(const float* __restrict__ c, int m, int K, double* __restrict__ x0) {
    extern __shared__ double coef[];
    const int t = blockIdx.x;
    for (int j = threadIdx.x; j < K; j += blockDim.x) coef[j] = (double)c[(size_t)t * K + j];
    __syncthreads();
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        double v = 0.0;
        for (int j = 0; j < K; ++j) v += coef[j] * sinpi((double)(j + 1) * (i + 1) / (double)(m + 1));
        x0[(size_t)t * m + i] = v;
    }
}

static int grid1(long n) {
    long g = (n + 255) / 256;
    return (int)(g > 1216 ? 1216 : (g < 1 ? 1 : g));
}

}  // namespace fde

using namespace fde;

struct fde_nop {
    int m = 0, s = 0, cin = 0, cout = 0, width = 0, layers = 0, K = 0;
    int modes = 0;                   // length of the convolution axis (sine modes)
    cudaStream_t stream = nullptr;
    std::vector<int> din, dout;      // per layer
    std::vector<long> woff, boff;    // offsets in the flat parameter vector
    long nparam = 0;
    float *p = nullptr, *g = nullptr, *m1 = nullptr, *m2 = nullptr;
    __half* p16 = nullptr;
    bool p16_valid = false;
    int t = 0;
    int bcap = 0;
    std::vector<float*> act;         // act[1..L], float, bcap x C_l x m
    float *ga = nullptr, *gb = nullptr;  // gradient ping-pong, bcap x max C x m
    __half *h_a = nullptr, *h_b = nullptr;  // FP16 inference activations (batch 1)
    float* feat = nullptr;           // features of one problem (cin x m)
    float* out1 = nullptr;           // output of one inference (s x m)
    double* d_loss = nullptr;
    double* h_loss = nullptr;        // pinned
};

namespace {

// Longest staged row of any tile of `tile` positions.
int staged_length(int tile, long N, int m, int K) {
    const int n = (int)std::min<long>(tile, N);
    const int pieces = (int)((n + (long)m - 2) / m) + 1;  // samples a tile can touch
    return n + pieces * 2 * (K / 2);
}

template <typename TI, typename TW, typename TO, bool TRANS, int NL, int KT, bool POS = false>
int conv_tiles(const TI* x, int Q, const TW* W, const float* bias, int P, int K, int m, long N, int relu,
               const float* mask, TO* y, cudaStream_t st) {
    constexpr int TN = cv_positions(NL, POS), QC = cv_channels(NL, POS);
    const int ld = staged_length(TN, N, m, K) | 1;
    const size_t stage = (size_t)QC * (ld + K * CV_LDW), red = (size_t)(POS ? 1 : CV_WARPS) * CV_TP * TN;
    const size_t smem = (stage > red ? stage : red) * sizeof(float);
    auto kern = conv_kernel<TI, TW, TO, TRANS, NL, KT, POS>;
    FDE_TRY(allow_smem((const void*)kern, 227 * 1024));
    const dim3 grid((unsigned)((N + TN - 1) / TN), (P + CV_TP - 1) / CV_TP);
    kern<<<grid, 32 * CV_WARPS, smem, st>>>(x, Q, W, bias, P, K, m, N, relu, mask, y, ld);
    FDE_LAUNCH_CHECK("conv_kernel");
    return FDE_OK;
}

// 16 positions a CTA while that leaves the launch within a few waves of the 152 SMs; beyond
// it 64, which reads the weights a quarter as often.  With at most 16 input channels and 128 positions
// for every SM, 128 of them in warps of their own: three layers of 16 channels on 16 x 2047 positions, forward,
// 48 to 59 us; 62 to 72 in tiles of 64 whose warps share the channels.
template <typename TI, typename TW, typename TO, bool TRANS>
int conv(const TI* x, int Q, const TW* W, const float* bias, int P, int K, int m, int B, int relu, const float* mask,
         TO* y, cudaStream_t st) {
    const long N = (long)B * m, pt = (P + CV_TP - 1) / CV_TP;
    const auto go = [&](auto NL, auto KT, auto POS) {
        return conv_tiles<TI, TW, TO, TRANS, NL.value, KT.value, POS.value>(x, Q, W, bias, P, K, m, N, relu, mask, y, st);
    };
    using std::false_type;
    using std::true_type;
    using N4 = std::integral_constant<int, 4>;
    using Any = std::integral_constant<int, 0>;
    if (Q <= 16 && (N + 127) / 128 * pt >= 152) {
        if (K == 3) return go(N4(), std::integral_constant<int, 3>(), true_type());
        if (K == 5) return go(N4(), std::integral_constant<int, 5>(), true_type());
        if (K == 7) return go(N4(), std::integral_constant<int, 7>(), true_type());
        return go(N4(), Any(), true_type());
    }
    if ((N + 15) / 16 * pt > 8 * 152) return go(std::integral_constant<int, 16>(), Any(), false_type());
    if (K == 3) return go(N4(), std::integral_constant<int, 3>(), false_type());
    if (K == 5) return go(N4(), std::integral_constant<int, 5>(), false_type());
    if (K == 7) return go(N4(), std::integral_constant<int, 7>(), false_type());
    return go(N4(), Any(), false_type());
}

int ensure_batch(fde_nop* n, int B) {
    if (B <= n->bcap) return FDE_OK;
    for (size_t l = 1; l < n->act.size(); ++l)
        if (n->act[l]) cudaFree(n->act[l]);
    if (n->ga) cudaFree(n->ga);
    if (n->gb) cudaFree(n->gb);
    n->act.assign(n->layers + 1, nullptr);
    int cmax = n->cin;
    for (int l = 0; l < n->layers; ++l) {
        FDE_CUDA_TRY(cudaMalloc(&n->act[l + 1], (size_t)B * n->dout[l] * n->modes * sizeof(float)));
        cmax = std::max(cmax, n->dout[l]);
    }
    FDE_CUDA_TRY(cudaMalloc(&n->ga, (size_t)B * cmax * n->modes * sizeof(float)));
    FDE_CUDA_TRY(cudaMalloc(&n->gb, (size_t)B * cmax * n->modes * sizeof(float)));
    n->bcap = B;
    return FDE_OK;
}

int forward32(fde_nop* n, const float* in, int B) {
    int rc = ensure_batch(n, B);
    if (rc) return rc;
    const float* x = in;
    for (int l = 0; l < n->layers; ++l) {
        rc = conv<float, float, float, false>(x, n->din[l], n->p + n->woff[l], n->p + n->boff[l], n->dout[l], n->K,
                                              n->modes, B, l < n->layers - 1, nullptr, n->act[l + 1], n->stream);
        if (rc) return rc;
        x = n->act[l + 1];
    }
    return FDE_OK;
}

}  // namespace

extern "C" {

void fde_nop_destroy(fde_nop* n) {
    if (!n) return;
    cudaStreamSynchronize(n->stream);
    for (size_t l = 1; l < n->act.size(); ++l)
        if (n->act[l]) cudaFree(n->act[l]);
    void* bufs[] = {n->p, n->g, n->m1, n->m2, n->p16, n->ga, n->gb, n->h_a, n->h_b, n->feat, n->out1, n->d_loss};
    for (void* b : bufs)
        if (b) cudaFree(b);
    if (n->h_loss) cudaFreeHost(n->h_loss);
    delete n;
}

int fde_nop_create(int m, int s, int modes, int width, int layers, int ksize, unsigned long long seed, void* stream,
                   fde_nop** out) {
    if (!out || m < 1 || s < 1 || modes < 1 || modes > m || width < 1 || layers < 1 || ksize < 1 ||
        ksize > CV_KMAX || ksize % 2 == 0)
        return set_error(FDE_ERR_ARG, "need m, s, width, layers >= 1, 1 <= modes <= m, odd kernel size <= 7");
    *out = nullptr;
    fde_nop* n = new (std::nothrow) fde_nop();
    if (!n) return set_error(FDE_ERR_ALLOC, "host allocation failed");
    n->m = m; n->s = s; n->modes = modes; n->cin = s + 6; n->cout = s; n->width = width; n->layers = layers;
    n->K = ksize;
    n->stream = (cudaStream_t)stream;
    for (int l = 0; l < layers; ++l) {
        n->din.push_back(l == 0 ? n->cin : width);
        n->dout.push_back(l == layers - 1 ? n->cout : width);
        n->woff.push_back(n->nparam);
        n->nparam += (long)n->dout[l] * n->din[l] * ksize;
        n->boff.push_back(n->nparam);
        n->nparam += n->dout[l];
    }
    const size_t pb = (size_t)n->nparam * sizeof(float);
    bool ok = cudaMalloc(&n->p, pb) == cudaSuccess && cudaMalloc(&n->g, pb) == cudaSuccess &&
              cudaMalloc(&n->m1, pb) == cudaSuccess && cudaMalloc(&n->m2, pb) == cudaSuccess &&
              cudaMalloc(&n->p16, (size_t)n->nparam * sizeof(__half)) == cudaSuccess &&
              cudaMalloc(&n->h_a, (size_t)std::max(n->cin, width) * modes * sizeof(__half)) == cudaSuccess &&
              cudaMalloc(&n->h_b, (size_t)std::max(n->cin, width) * modes * sizeof(__half)) == cudaSuccess &&
              cudaMalloc(&n->feat, (size_t)n->cin * modes * sizeof(float)) == cudaSuccess &&
              cudaMalloc(&n->out1, (size_t)s * modes * sizeof(float)) == cudaSuccess &&
              cudaMalloc(&n->d_loss, sizeof(double)) == cudaSuccess &&
              cudaMallocHost(&n->h_loss, sizeof(double)) == cudaSuccess;
    if (!ok) {
        fde_nop_destroy(n);
        return set_error(FDE_ERR_ALLOC, "device allocation failed");
    }
    // He-uniform weights (last layer scaled down), zero biases, zero Adam moments
    cudaMemsetAsync(n->p, 0, pb, n->stream);
    cudaMemsetAsync(n->m1, 0, pb, n->stream);
    cudaMemsetAsync(n->m2, 0, pb, n->stream);
    for (int l = 0; l < layers; ++l) {
        const long nw = (long)n->dout[l] * n->din[l] * ksize;
        float a = std::sqrt(6.0f / (float)(n->din[l] * ksize));
        if (l == layers - 1) a *= 0.1f;
        init_kernel<<<grid1(nw), 256, 0, n->stream>>>(n->p, n->woff[l], nw, a, seed);
        note_launch();
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        fde_nop_destroy(n);
        return cuda_error(e, "fde_nop_create");
    }
    *out = n;
    return FDE_OK;
}

long long fde_nop_num_params(const fde_nop* n) { return n ? n->nparam : 0; }
int fde_nop_in_channels(const fde_nop* n) { return n ? n->cin : 0; }

int fde_nop_set_params(fde_nop* n, const float* params) {
    if (!n || !params) return set_error(FDE_ERR_ARG, "NULL argument");
    FDE_CUDA_TRY(cudaMemcpyAsync(n->p, params, n->nparam * sizeof(float), cudaMemcpyHostToDevice, n->stream));
    FDE_CUDA_TRY(cudaStreamSynchronize(n->stream));
    n->p16_valid = false;
    return FDE_OK;
}

int fde_nop_get_params(fde_nop* n, float* params) {
    if (!n || !params) return set_error(FDE_ERR_ARG, "NULL argument");
    FDE_CUDA_TRY(cudaMemcpyAsync(params, n->p, n->nparam * sizeof(float), cudaMemcpyDeviceToHost, n->stream));
    FDE_CUDA_TRY(cudaStreamSynchronize(n->stream));
    return FDE_OK;
}

int fde_nop_forward(fde_nop* n, const float* in, float* out, int batch) {
    if (!n || !in || !out || batch < 1) return set_error(FDE_ERR_ARG, "bad argument");
    int rc = forward32(n, in, batch);
    if (rc) return rc;
    FDE_CUDA_TRY(cudaMemcpyAsync(out, n->act[n->layers], (size_t)batch * n->cout * n->modes * sizeof(float),
                                 cudaMemcpyDeviceToDevice, n->stream));
    return FDE_OK;
}

int fde_nop_loss_grad(fde_nop* n, const float* in, const float* target, int batch, double* loss, float* grad_host) {
    if (!n || !in || !target || batch < 1) return set_error(FDE_ERR_ARG, "bad argument");
    int rc = forward32(n, in, batch);
    if (rc) return rc;
    const int L = n->layers, m = n->modes, B = batch;
    const long ny = (long)B * n->cout * m;
    FDE_CUDA_TRY(cudaMemsetAsync(n->d_loss, 0, sizeof(double), n->stream));
    FDE_CUDA_TRY(cudaMemsetAsync(n->g, 0, n->nparam * sizeof(float), n->stream));
    mse_kernel<<<grid1(ny), 256, 0, n->stream>>>(n->act[L], target, ny, n->ga, n->d_loss);
    FDE_LAUNCH_CHECK("mse_kernel");
    float* g = n->ga;      // gradient w.r.t. the output of layer l (after its ReLU mask)
    float* gnext = n->gb;
    for (int l = L - 1; l >= 0; --l) {
        const float* a = l == 0 ? in : n->act[l];
        const int O = n->dout[l], C = n->din[l];
        const int groups = (int)std::min<long>(((long)B * m + 15) / 16, 16), cx = (C + 15) / 16, cy = (O + 15) / 16;
        const long per = ((long)B * m + groups - 1) / groups;
        const dim3 wg(cx, cy, groups + (16 + cx - 1) / cx);
        const int ld = staged_length(WG_N, (long)B * m, m, n->K) | 1;
        const size_t smem = (size_t)16 * (WG_N + 1 + ld) * sizeof(float);
        FDE_TRY(allow_smem((const void*)conv_wgrad_kernel, smem));
        conv_wgrad_kernel<<<wg, 256, smem, n->stream>>>(g, O, a, C, n->K, m, B, groups, per, n->g + n->woff[l],
                                                        n->g + n->boff[l], ld);
        FDE_LAUNCH_CHECK("conv_wgrad_kernel");
        if (l > 0) {
            // gradient w.r.t. the layer input, through the ReLU of layer l-1 (mask = its output)
            rc = conv<float, float, float, true>(g, O, n->p + n->woff[l], nullptr, C, n->K, m, B, 0, n->act[l], gnext,
                                                 n->stream);
            if (rc) return rc;
            std::swap(g, gnext);
        }
    }
    FDE_CUDA_TRY(cudaMemcpyAsync(n->h_loss, n->d_loss, sizeof(double), cudaMemcpyDeviceToHost, n->stream));
    if (grad_host)
        FDE_CUDA_TRY(cudaMemcpyAsync(grad_host, n->g, n->nparam * sizeof(float), cudaMemcpyDeviceToHost, n->stream));
    FDE_CUDA_TRY(cudaStreamSynchronize(n->stream));
    if (loss) *loss = *n->h_loss;
    return FDE_OK;
}

int fde_nop_adam_step(fde_nop* n, float lr) {
    if (!n) return set_error(FDE_ERR_ARG, "NULL network");
    ++n->t;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - std::pow(b1, (float)n->t), c2 = 1.f - std::pow(b2, (float)n->t);
    adam_kernel<<<grid1(n->nparam), 256, 0, n->stream>>>(n->p, n->g, n->m1, n->m2, n->nparam, lr, b1, b2, 1e-8f, c1,
                                                         c2);
    FDE_LAUNCH_CHECK("adam_kernel");
    n->p16_valid = false;
    return FDE_OK;
}

int fde_nop_features(fde_nop* n, fde_problem* h, float* in) {
    if (!n || !h || !in) return set_error(FDE_ERR_ARG, "NULL argument");
    Problem& P = *problem_of(h);
    if (P.m != n->m || P.s != n->s) return set_error(FDE_ERR_ARG, "problem size differs from the network's");
    const int K = n->modes;
    const long w0 = (long)1 * K * 32, w1 = (long)(P.s + 1) * K * 32;
    sine_analysis_kernel<<<(int)((w0 + 255) / 256), 256, 0, n->stream>>>(P.d_u0, 1, P.m, K, in, K, 0);
    FDE_LAUNCH_CHECK("sine_analysis_kernel(u0)");
    sine_analysis_kernel<<<(int)((w1 + 255) / 256), 256, 0, n->stream>>>(P.d_f, P.s + 1, P.m, K, in, K, 1);
    FDE_LAUNCH_CHECK("sine_analysis_kernel(f)");
    scalar_channels_kernel<<<1, 256, 0, n->stream>>>(P.m, K, P.s + 2, P.alpha, P.d_dplus, P.d_dminus, in);
    FDE_LAUNCH_CHECK("scalar_channels_kernel");
    return FDE_OK;
}

int fde_nop_coefficients(fde_nop* n, const double* x, float* coef) {
    if (!n || !x || !coef) return set_error(FDE_ERR_ARG, "NULL argument");
    const long w = (long)n->s * n->modes * 32;
    sine_analysis_kernel<<<(int)((w + 255) / 256), 256, 0, n->stream>>>(x, n->s, n->m, n->modes, coef, n->modes, 0);
    FDE_LAUNCH_CHECK("sine_analysis_kernel(x)");
    return FDE_OK;
}

int fde_nop_warm_start(fde_nop* n, fde_problem* h, double* x0) {
    if (!n || !h || !x0) return set_error(FDE_ERR_ARG, "NULL argument");
    int rc = fde_nop_features(n, h, n->feat);
    if (rc) return rc;
    if (!n->p16_valid) {
        to_half_kernel<<<grid1(n->nparam), 256, 0, n->stream>>>(n->p, n->p16, n->nparam);
        FDE_LAUNCH_CHECK("to_half_kernel");
        n->p16_valid = true;
    }
    // FP16 storage of weights and activations, FP32 accumulation and biases
    const int L = n->layers, m = n->modes;
    const __half* xh = nullptr;
    for (int l = 0; l < L; ++l) {
        __half* dst = (l % 2 == 0) ? n->h_a : n->h_b;
        const float* bias = n->p + n->boff[l];
        if (l == L - 1) {
            if (l == 0)
                rc = conv<float, __half, float, false>(n->feat, n->din[l], n->p16 + n->woff[l], bias, n->dout[l], n->K,
                                                       m, 1, 0, nullptr, n->out1, n->stream);
            else
                rc = conv<__half, __half, float, false>(xh, n->din[l], n->p16 + n->woff[l], bias, n->dout[l], n->K, m,
                                                        1, 0, nullptr, n->out1, n->stream);
        } else if (l == 0) {
            rc = conv<float, __half, __half, false>(n->feat, n->din[l], n->p16 + n->woff[l], bias, n->dout[l], n->K,
                                                    m, 1, 1, nullptr, dst, n->stream);
        } else {
            rc = conv<__half, __half, __half, false>(xh, n->din[l], n->p16 + n->woff[l], bias, n->dout[l], n->K, m, 1,
                                                     1, nullptr, dst, n->stream);
        }
        if (rc) return rc;
        xh = dst;
    }
    sine_synthesis_kernel<<<n->s, 256, n->modes * sizeof(double), n->stream>>>(n->out1, n->m, n->modes, x0);
    FDE_LAUNCH_CHECK("sine_synthesis_kernel");
    return FDE_OK;
}

int fde_nop_synthesize(fde_nop* n, const float* coef, double* x) {
    if (!n || !coef || !x) return set_error(FDE_ERR_ARG, "NULL argument");
    sine_synthesis_kernel<<<n->s, 256, n->modes * sizeof(double), n->stream>>>(coef, n->m, n->modes, x);
    FDE_LAUNCH_CHECK("sine_synthesis_kernel");
    return FDE_OK;
}

}  // extern "C"
