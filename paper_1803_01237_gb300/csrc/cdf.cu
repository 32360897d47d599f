// cdf.cu -- the learned splitter proposal: a 1-32-32-1 CDF network of the
// keys, trained on the device from (key, rank) pairs and inverted to propose
// the splitters of the next job before round 1 of the histogram rounds.
//
// The paper proposes no learned model; its rounds (Sec. 4.2.2) accept any
// candidate cuts, and this network is one source of them.  Everything is
// float32 on the CUDA cores: the network has 1153 parameters and a training
// batch holds a few thousand points, far too small a contraction for tensor
// cores to matter.  Under HSS_CDF_W_BF16 every evaluation uses the parameters
// rounded to bfloat16 (the float32 master copy takes the Adam updates).
//
//   feature   x = clip((raw(u) - lo) / (hi - lo), 0, 1), raw(u) = u or
//             log2(1 + u), u = order-preserving key bits (double precision)
//   network   y = w3 . relu(W2 relu(w1 x + b1) + b2) + b3
//   loss      L = (1/n) sum_b (y_b - rank_b / N)^2
//   update    Adam (Kingma and Ba, 2015), bias-corrected
#include "hss_internal.cuh"

#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>

namespace hss {
namespace {

constexpr int kH = HSS_CDF_HIDDEN;
constexpr int kP = HSS_CDF_NPARAM;
constexpr int kOffB1 = kH, kOffW2 = 2 * kH, kOffB2 = 2 * kH + kH * kH, kOffW3 = kOffB2 + kH, kOffB3 = kOffW3 + kH;
constexpr int kGradThreads = 128;   // a point each; four warps, one per scheduler
constexpr int kMaxGradBlocks = 32;  // training shares the GPU with the sorts it serves: a few SMs
constexpr int kPartStride = kP + 3;  // gradient, loss partial, padding (a multiple of four floats)
constexpr int kStage = kH + 4;       // row of a staged activation vector: 16-byte aligned, rows start four banks apart
constexpr int kRowGroups = kGradThreads / 64;  // 64 threads hold the 4 x 4 tiles of dW2, each group sums a share of the rows
constexpr uint32_t kInitTag = 0x43444621u;
constexpr float kBeta1 = 0.9f, kBeta2 = 0.999f, kAdamEps = 1e-8f;

__device__ __forceinline__ float feature_of(uint64_t bits, const hss_cdf_model* M, uint64_t flip) {
    const double u = (double)(bits ^ flip);
    const double raw = M->feature == HSS_CDF_LOG ? log2(1.0 + u) : u;
    double x = (raw - M->lo) / (M->hi - M->lo);
    x = x < 0.0 ? 0.0 : (x > 1.0 ? 1.0 : x);
    return (float)x;
}

// Parameter k as the network uses it: float32, or rounded to bfloat16
// (nearest, ties to even) under HSS_CDF_W_BF16.
__device__ __forceinline__ float weight_of(const hss_cdf_model* M, int k) {
    const float w = M->theta[k];
    return M->weights == HSS_CDF_W_BF16 ? __bfloat162float(__float2bfloat16_rn(w)) : w;
}

// Hidden layers of one point with the parameters in shared memory (every
// thread reads the same weights at the same time: broadcasts, four at once).
// Four rows of W2 advance together, so four chains of multiply-adds hide each
// other's latency.  Returns y(x).
__device__ __forceinline__ float layers(const float* th, float x, float (&h1)[kH], float (&h2)[kH]) {
#pragma unroll
    for (int i = 0; i < kH; ++i) h1[i] = fmaxf(fmaf(th[i], x, th[kOffB1 + i]), 0.f);
    float y = th[kOffB3];
#pragma unroll
    for (int i = 0; i < kH; i += 4) {
        float a[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) a[r] = th[kOffB2 + i + r];
#pragma unroll
        for (int j = 0; j < kH; j += 4) {
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const float4 w = *(const float4*)(th + kOffW2 + (i + r) * kH + j);
                a[r] = fmaf(w.x, h1[j], a[r]);
                a[r] = fmaf(w.y, h1[j + 1], a[r]);
                a[r] = fmaf(w.z, h1[j + 2], a[r]);
                a[r] = fmaf(w.w, h1[j + 3], a[r]);
            }
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            h2[i + r] = fmaxf(a[r], 0.f);
            y = fmaf(th[kOffW3 + i + r], h2[i + r], y);
        }
    }
    return y;
}
// y(x) alone, the same operations in the same order, a few rows unrolled: a
// loop around it (the bisection) would have the compiler keep every weight of
// `layers` in registers, and spill them.
__device__ __forceinline__ float net(const float* th, float x) {
    float h1[kH];
#pragma unroll
    for (int i = 0; i < kH; ++i) h1[i] = fmaxf(fmaf(th[i], x, th[kOffB1 + i]), 0.f);
    float y = th[kOffB3];
#pragma unroll 4
    for (int i = 0; i < kH; ++i) {
        float a = th[kOffB2 + i];
#pragma unroll
        for (int j = 0; j < kH; ++j) a = fmaf(th[kOffW2 + i * kH + j], h1[j], a);
        y = fmaf(th[kOffW3 + i], fmaxf(a, 0.f), y);
    }
    return y;
}

__global__ void k_cdf_init(hss_cdf_model* M, uint64_t seed, int feature, int key_type, double lo, double hi) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k == 0) {
        M->step = 0; M->feature = feature; M->key_type = key_type; M->weights = HSS_CDF_W_FP32; M->lo = lo; M->hi = hi;
    }
    if (k >= kP) return;
    const Philox4 r = philox4x32_10((uint32_t)k, 0u, 0u, kInitTag, (uint32_t)seed, (uint32_t)(seed >> 32));
    const float u = (float)(r.v[0] >> 8) * (1.0f / 16777216.0f);
    const float scale = 0.4330127018922193f;  // sqrt(6 / 32)
    float w;
    if (k < kOffB1) {
        w = ((k & 1) ? -1.f : 1.f) * (1.f + u) * 4.f;
    } else if (k < kOffW2) {  // knot of hidden-1 unit i at (i + 0.5) / 32
        const int i = k - kOffB1;
        const Philox4 r1 = philox4x32_10((uint32_t)i, 0u, 0u, kInitTag, (uint32_t)seed, (uint32_t)(seed >> 32));
        const float u1 = (float)(r1.v[0] >> 8) * (1.0f / 16777216.0f);
        const float w1 = ((i & 1) ? -1.f : 1.f) * (1.f + u1) * 4.f;
        w = -w1 * ((float)i + 0.5f) / (float)kH;
    } else if (k < kOffB2) {
        w = (2.f * u - 1.f) * scale;
    } else if (k < kOffW3) {
        w = 0.1f;
    } else if (k < kOffB3) {
        w = (2.f * u - 1.f) * scale;
    } else {
        w = 0.5f;
    }
    M->theta[k] = w;
    M->m[k] = 0.f;
    M->v[k] = 0.f;
}

// Feature and target of a training point.
__device__ __forceinline__ float2 point_of(const hss_cdf_model* M, const uint64_t* __restrict__ keys,
                                           const uint64_t* __restrict__ ranks, uint64_t b, double invN) {
    const uint64_t flip = M->key_type == HSS_KEY_I64 ? kSignBit : 0ull;
    return make_float2(feature_of(keys[b], M, flip), (float)((double)ranks[b] * invN));
}

// Features and targets of the training points, once per call: the feature map
// is double precision (log2), which the steps would otherwise repeat.
__global__ __launch_bounds__(kGradThreads) void k_cdf_points(const hss_cdf_model* __restrict__ M,
                                                             const uint64_t* __restrict__ keys,
                                                             const uint64_t* __restrict__ ranks, uint32_t n, double invN,
                                                             float2* __restrict__ pts, uint32_t* __restrict__ arrived) {
    const uint32_t b = blockIdx.x * kGradThreads + threadIdx.x;
    if (b == 0) *arrived = 0u;
    if (b >= n) return;
    pts[b] = point_of(M, keys, ranks, b, invN);
}

// One step: the gradient of the mean squared error, and Adam.  Each CTA takes
// a grid-stride share of the points, a thread running the forward and backward
// pass of one; the activations and their gradients are staged in shared memory,
// where dW2 = DZ2^T H1 is summed as 4 x 4 tiles (two 16-byte reads per 16
// multiply-adds) and the other entries column by column, and the CTA writes
// one partial.  The last CTA to arrive sums the partials in block order
// (deterministic) and applies the update: one launch per step.
// Bound by the latency of its dependent chains (four warps on an SM, a few
// SMs).  4096 points: 78 us per step as two kernels that walked the 256 staged
// rows one load at a time, here 19 us.
// PTS: the points come from pts.  Without (a scratch buffer that has no room
// for them, see Work) every step computes them from the keys and ranks.
template <bool PTS>
__global__ __launch_bounds__(kGradThreads) void k_cdf_step(hss_cdf_model* M, const float2* __restrict__ pts,
                                                           const uint64_t* __restrict__ keys,
                                                           const uint64_t* __restrict__ ranks, double invN, uint32_t n,
                                                           float inv_n, float* __restrict__ part,
                                                           uint32_t* __restrict__ arrived, float lr, int apply,
                                                           float* __restrict__ grad_out, float* __restrict__ loss_out) {
    extern __shared__ __align__(16) float sm[];
    float* th = sm;                                 // kP (+3)
    float* H1s = th + kP + 3;                       // rows of kStage
    float* H2s = H1s + kGradThreads * kStage;
    float* DZ2s = H2s + kGradThreads * kStage;
    float* DZ1s = DZ2s + kGradThreads * kStage;
    float* Xs = DZ1s + kGradThreads * kStage;       // kGradThreads
    float* Ds = Xs + kGradThreads;                  // kGradThreads
    __shared__ float s_sum[2 * kGradThreads / 32];
    __shared__ uint32_t s_last;
    __shared__ float s_c[2];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    {
        const bool half = M->weights == HSS_CDF_W_BF16;
#pragma unroll
        for (int u = 0; u < (kP + kGradThreads - 1) / kGradThreads; ++u) {
            const int k = tid + u * kGradThreads;
            if (k < kP) {
                const float x = M->theta[k];
                th[k] = half ? __bfloat162float(__float2bfloat16_rn(x)) : x;
            }
        }
    }
    __syncthreads();

    const int tile = tid & 63, i0 = (tile >> 3) * 4, j0 = (tile & 7) * 4, grp = tid >> 6;
    float acc[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = 0.f;
    float accS = 0.f;              // warp 0: dw1, 1: db1, 2: db2, 3: dw3, a column per lane
    float accD = 0.f, accL = 0.f;  // db3 and the squared errors of this thread's points
    for (uint64_t base = (uint64_t)blockIdx.x * kGradThreads; base < n; base += (uint64_t)gridDim.x * kGradThreads) {
        const uint64_t b = base + tid;
        float x = 0.f, d = 0.f;
        float h1[kH], h2[kH], dz1[kH];
        if (b < n) {
            const float2 pt = PTS ? pts[b] : point_of(M, keys, ranks, b, invN);
            x = pt.x;
            const float e = layers(th, x, h1, h2) - pt.y;
            d = 2.f * e * inv_n;
            accL = fmaf(e, e, accL);
        } else {
#pragma unroll
            for (int i = 0; i < kH; ++i) { h1[i] = 0.f; h2[i] = 0.f; }
        }
        accD += d;
#pragma unroll
        for (int j = 0; j < kH; ++j) dz1[j] = 0.f;
#pragma unroll
        for (int i = 0; i < kH; ++i) {
            const float dz2 = h2[i] > 0.f ? d * th[kOffW3 + i] : 0.f;
            DZ2s[tid * kStage + i] = dz2;
#pragma unroll
            for (int j = 0; j < kH; j += 4) {
                const float4 wv = *(const float4*)(th + kOffW2 + i * kH + j);
                dz1[j] = fmaf(wv.x, dz2, dz1[j]);
                dz1[j + 1] = fmaf(wv.y, dz2, dz1[j + 1]);
                dz1[j + 2] = fmaf(wv.z, dz2, dz1[j + 2]);
                dz1[j + 3] = fmaf(wv.w, dz2, dz1[j + 3]);
            }
        }
#pragma unroll
        for (int j = 0; j < kH; ++j) {
            H1s[tid * kStage + j] = h1[j];
            H2s[tid * kStage + j] = h2[j];
            DZ1s[tid * kStage + j] = h1[j] > 0.f ? dz1[j] : 0.f;
        }
        Xs[tid] = x;
        Ds[tid] = d;
        __syncthreads();
        // dW2[i][j] = sum_b dz2[b][i] h1[b][j]
        constexpr int kRows = kGradThreads / kRowGroups;
#pragma unroll 8
        for (int r = grp * kRows; r < (grp + 1) * kRows; ++r) {
            const float4 a = *(const float4*)(DZ2s + r * kStage + i0), h = *(const float4*)(H1s + r * kStage + j0);
            const float av[4] = {a.x, a.y, a.z, a.w}, hv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[p][q] = fmaf(av[p], hv[q], acc[p][q]);
        }
        // dw1[j] = sum_b dz1[b][j] x_b, db1, db2, dw3[i] = sum_b d_b h2[b][i]
        {
            const float* col = (w < 2 ? DZ1s : (w == 2 ? DZ2s : H2s)) + lane;
            const float* f = w == 0 ? Xs : Ds;
            const bool plain = w == 1 || w == 2;
            float t[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
            for (int r = 0; r < kGradThreads; r += 4)
#pragma unroll
                for (int u = 0; u < 4; ++u) t[u] = fmaf(col[(r + u) * kStage], plain ? 1.f : f[r + u], t[u]);
            accS += (t[0] + t[1]) + (t[2] + t[3]);
        }
        __syncthreads();
    }
    // the row groups of dW2 together, through the staging area
    if (grp > 0) {
#pragma unroll
        for (int p = 0; p < 4; ++p)
            *(float4*)(H1s + (grp - 1) * 1024 + (i0 + p) * kH + j0) = make_float4(acc[p][0], acc[p][1], acc[p][2], acc[p][3]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        accD += __shfl_xor_sync(0xffffffffu, accD, o);
        accL += __shfl_xor_sync(0xffffffffu, accL, o);
    }
    if (lane == 0) { s_sum[w] = accD; s_sum[kGradThreads / 32 + w] = accL; }
    __syncthreads();
    float* out = part + (uint64_t)blockIdx.x * kPartStride;
    const bool vec = PTS || ((uintptr_t)part & 15u) == 0;  // the partials lie on 16 bytes
    if (grp == 0) {
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            float4 v = make_float4(acc[p][0], acc[p][1], acc[p][2], acc[p][3]);
#pragma unroll
            for (int g = 1; g < kRowGroups; ++g) {
                const float4 o = *(const float4*)(H1s + (g - 1) * 1024 + (i0 + p) * kH + j0);
                v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w;
            }
            float* o = out + kOffW2 + (i0 + p) * kH + j0;
            if (vec) {
                *(float4*)o = v;
            } else {
                o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
            }
        }
    }
    out[(w == 0 ? 0 : (w == 1 ? kOffB1 : (w == 2 ? kOffB2 : kOffW3))) + lane] = accS;
    if (tid == 0) {
        float sd = 0.f, sl = 0.f;
        for (int i = 0; i < kGradThreads / 32; ++i) { sd += s_sum[i]; sl += s_sum[kGradThreads / 32 + i]; }
        out[kOffB3] = sd;
        out[kP] = sl;
    }
    // the last CTA sums the partials
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicInc(arrived, gridDim.x - 1) == gridDim.x - 1 ? 1u : 0u;  // back to 0 for the next step
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const uint32_t t = M->step + 1;
    if (apply && tid < 2) {  // 1 - beta^t by squaring (pow takes microseconds in double precision)
        double f = (double)(tid ? kBeta2 : kBeta1), q = 1.0;
        for (uint32_t e = t; e > 0; e >>= 1) {
            if (e & 1u) q *= f;
            f *= f;
        }
        s_c[tid] = (float)(1.0 - q);
    }
    const int G = (int)gridDim.x;
    for (int k = tid; !vec && k < kPartStride; k += kGradThreads) {
        float g = 0.f;
        for (int c = 0; c < G; ++c) g += __ldcg(part + (uint64_t)c * kPartStride + k);
        H1s[k] = g;
    }
    for (int k4 = tid; vec && k4 < kPartStride / 4; k4 += kGradThreads) {
        float4 g4 = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 16
        for (int c = 0; c < G; ++c) {
            const float4 v = __ldcg((const float4*)(part + (uint64_t)c * kPartStride) + k4);
            g4.x += v.x; g4.y += v.y; g4.z += v.z; g4.w += v.w;
        }
        ((float4*)H1s)[k4] = g4;
    }
    __syncthreads();
    if (tid == 0 && loss_out) *loss_out = H1s[kP] * inv_n;
    constexpr int kPer = (kP + kGradThreads - 1) / kGradThreads;
    if (grad_out) {
        for (int k = tid; k < kP; k += kGradThreads) grad_out[k] = H1s[k];
    }
    if (apply) {  // all loads first: the stores go to the same struct
        float m[kPer], v[kPer], x[kPer];
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const int k = tid + u * kGradThreads;
            if (k < kP) { m[u] = M->m[k]; v[u] = M->v[k]; x[u] = M->theta[k]; }
        }
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const int k = tid + u * kGradThreads;
            if (k >= kP) continue;
            const float g = H1s[k];
            m[u] = kBeta1 * m[u] + (1.f - kBeta1) * g;
            v[u] = kBeta2 * v[u] + (1.f - kBeta2) * g * g;
            M->m[k] = m[u];
            M->v[k] = v[u];
            M->theta[k] = x[u] - lr * (m[u] / s_c[0]) / (sqrtf(v[u] / s_c[1]) + kAdamEps);
        }
    }
    __syncthreads();
    if (apply && tid == 0) M->step = t;
}

__global__ void k_cdf_set_weights(hss_cdf_model* M, int weights) { M->weights = weights; }

__global__ void k_cdf_eval(const hss_cdf_model* __restrict__ M, const uint64_t* __restrict__ keys, uint32_t n,
                           float* __restrict__ y) {
    __shared__ __align__(16) float th[kP + 3];
    for (int k = threadIdx.x; k < kP; k += blockDim.x) th[k] = weight_of(M, k);
    __syncthreads();
    const uint64_t b = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= n) return;
    const uint64_t flip = M->key_type == HSS_KEY_I64 ? kSignBit : 0ull;
    float h1[kH], h2[kH];
    y[b] = layers(th, feature_of(keys[b], M, flip), h1, h2);
}

// Cut q = (i-1) per + k of splitter i (1..p-1): target tau = i/p + delta
// (2k/(per-1) - 1) clipped to [0, 1] (i/p when per = 1); bisection for the
// smallest x in [0, 1] with y(x) >= tau, then the inverse feature map,
// clamped to the key range.
__global__ void k_cdf_propose(const hss_cdf_model* __restrict__ M, uint32_t p, uint32_t per, double delta, int iters,
                              uint64_t* __restrict__ out) {
    __shared__ __align__(16) float th[kP + 3];
    for (int k = threadIdx.x; k < kP; k += blockDim.x) th[k] = weight_of(M, k);
    __syncthreads();
    const uint64_t q = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= (uint64_t)(p - 1) * per) return;
    const uint32_t i = (uint32_t)(q / per) + 1, k = (uint32_t)(q % per);
    double tau_d = (double)i / (double)p;
    if (per > 1) tau_d += delta * (2.0 * (double)k / (double)(per - 1) - 1.0);
    tau_d = tau_d < 0.0 ? 0.0 : (tau_d > 1.0 ? 1.0 : tau_d);
    const float tau = (float)tau_d;
    float a = 0.f, b = 1.f;
    for (int it = 0; it < iters; ++it) {
        const float mid = 0.5f * (a + b);
        if (net(th, mid) < tau) a = mid; else b = mid;
    }
    const double r = M->lo + (double)b * (M->hi - M->lo);
    const double u = M->feature == HSS_CDF_LOG ? exp2(r) - 1.0 : r;
    uint64_t bits;
    if (!(u > 0.0)) bits = 0ull;
    else if (u >= 18446744073709551615.0) bits = ~0ull;
    else bits = (uint64_t)u;
    const uint64_t flip = M->key_type == HSS_KEY_I64 ? kSignBit : 0ull;
    out[q] = bits ^ flip;
}

size_t grad_smem() { return (size_t)(kP + 3 + 4 * kGradThreads * kStage + 2 * kGradThreads) * sizeof(float); }

uint32_t grad_blocks(uint32_t n, int points) {  // CTAs for n points, `points` to a CTA
    return (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(kMaxGradBlocks, ((uint64_t)n + points - 1) / points));
}

// Scratch of a call: the CTAs' partials, the arrival counter, the points.  A
// buffer too small for that, but of the least size (a partial for every 256
// points, 32 at most: independent of n from 8192 points on), holds that many
// partials, the counter in the first one's padding, and no points.
struct Work {
    uint32_t blocks;
    float* part;
    uint32_t* arrived;
    float2* pts;  // null: none kept
    static size_t parts(uint32_t blocks) { return (size_t)blocks * kPartStride * sizeof(float); }  // a multiple of 16
    static size_t least(uint32_t n) { return parts(grad_blocks(n, 256)); }
    static size_t bytes(uint32_t n) { return 16 + parts(grad_blocks(n, kGradThreads)) + 16 + (size_t)n * sizeof(float2); }
    Work(void* base, size_t size, uint32_t n) {
        if (size >= bytes(n)) {
            blocks = grad_blocks(n, kGradThreads);
            char* q = (char*)(((uintptr_t)base + 15) & ~(uintptr_t)15);
            part = (float*)q;
            arrived = (uint32_t*)(q + parts(blocks));
            pts = (float2*)(q + parts(blocks) + 16);
        } else {
            blocks = grad_blocks(n, 256);
            part = (float*)base;
            arrived = (uint32_t*)(part + kP + 1);
            pts = nullptr;
        }
    }
};

// One call's steps: the points (or the counter alone), then a kernel per step.
int run_steps(hss_cdf_model* M, const uint64_t* keys, const uint64_t* ranks, uint32_t n, uint64_t N, const Work& wk,
              uint32_t steps, float lr, int apply, float* grad, float* loss, cudaStream_t st) {
    const double invN = 1.0 / (double)N;
    const float inv_n = (float)(1.0 / (double)n);
    const void* fn = wk.pts ? (const void*)k_cdf_step<true> : (const void*)k_cdf_step<false>;
    if (ensure_func_attrs(fn, (int)grad_smem()) != cudaSuccess) return HSS_ERR_CUDA;
    if (wk.pts)
        HSS_LAUNCH(k_cdf_points, (unsigned)(((uint64_t)n + kGradThreads - 1) / kGradThreads), kGradThreads, 0, st, M, keys,
                   ranks, n, invN, wk.pts, wk.arrived);
    else if (cudaMemsetAsync(wk.arrived, 0, sizeof(uint32_t), st) != cudaSuccess)
        return HSS_ERR_CUDA;
    for (uint32_t s = 0; s < steps; ++s) {
        float* l = s + 1 == steps ? loss : nullptr;
        if (wk.pts)
            HSS_LAUNCH(k_cdf_step<true>, wk.blocks, kGradThreads, grad_smem(), st, M, wk.pts, nullptr, nullptr, invN, n, inv_n,
                       wk.part, wk.arrived, lr, apply, grad, l);
        else
            HSS_LAUNCH(k_cdf_step<false>, wk.blocks, kGradThreads, grad_smem(), st, M, nullptr, keys, ranks, invN, n, inv_n,
                       wk.part, wk.arrived, lr, apply, grad, l);
    }
    return cudaGetLastError() == cudaSuccess ? HSS_OK : HSS_ERR_CUDA;
}

bool raw_bound(uint64_t key, int feature, int key_type, double* out) {
    const uint64_t u = key ^ (key_type == HSS_KEY_I64 ? kSignBit : 0ull);
    *out = feature == HSS_CDF_LOG ? std::log2(1.0 + (double)u) : (double)u;
    return std::isfinite(*out);
}

}  // namespace
}  // namespace hss

using namespace hss;

extern "C" {

size_t hss_cdf_model_bytes(void) { return sizeof(hss_cdf_model); }

int hss_cdf_set_weights(hss_cdf_model* d_model, int weights, void* stream) {
    if (!d_model || (weights != HSS_CDF_W_FP32 && weights != HSS_CDF_W_BF16)) return HSS_ERR_INVALID;
    HSS_LAUNCH(k_cdf_set_weights, 1, 1, 0, (cudaStream_t)stream, d_model, weights);
    return cudaGetLastError() == cudaSuccess ? HSS_OK : HSS_ERR_CUDA;
}

size_t hss_cdf_work_bytes(uint32_t n) { return Work::bytes(n); }

int hss_cdf_init(hss_cdf_model* d_model, uint64_t seed, int feature, int key_type, uint64_t lo_key, uint64_t hi_key,
                 void* stream) {
    if (!d_model || (feature != HSS_CDF_LINEAR && feature != HSS_CDF_LOG)) return HSS_ERR_INVALID;
    if (key_type != HSS_KEY_U64 && key_type != HSS_KEY_I64) return HSS_ERR_INVALID;
    double lo, hi;
    if (!raw_bound(lo_key, feature, key_type, &lo) || !raw_bound(hi_key, feature, key_type, &hi) || !(hi > lo))
        return HSS_ERR_INVALID;
    HSS_LAUNCH(k_cdf_init, (kP + 255) / 256, 256, 0, (cudaStream_t)stream, d_model, seed, feature, key_type, lo, hi);
    return cudaGetLastError() == cudaSuccess ? HSS_OK : HSS_ERR_CUDA;
}

int hss_cdf_grad(const hss_cdf_model* d_model, const void* d_keys, const uint64_t* d_ranks, uint32_t n, uint64_t N,
                 float* d_grad, float* d_loss, void* d_work, size_t work_bytes, void* stream) {
    if (!d_model || n == 0 || N == 0 || !d_keys || !d_ranks || !d_work) return HSS_ERR_INVALID;
    if (work_bytes < Work::least(n)) return HSS_ERR_WORKSPACE;
    cudaStream_t st = (cudaStream_t)stream;
    return run_steps(const_cast<hss_cdf_model*>(d_model), (const uint64_t*)d_keys, d_ranks, n, N, Work(d_work, work_bytes, n), 1,
                     0.f, 0, d_grad, d_loss, st);
}

int hss_cdf_train(hss_cdf_model* d_model, const void* d_keys, const uint64_t* d_ranks, uint32_t n, uint64_t N,
                  uint32_t steps, float lr, float* d_loss, void* d_work, size_t work_bytes, void* stream) {
    if (!d_model || n == 0 || N == 0 || !d_keys || !d_ranks || !d_work || !(lr > 0.f)) return HSS_ERR_INVALID;
    if (work_bytes < Work::least(n)) return HSS_ERR_WORKSPACE;
    cudaStream_t st = (cudaStream_t)stream;
    if (steps == 0) return HSS_OK;
    return run_steps(d_model, (const uint64_t*)d_keys, d_ranks, n, N, Work(d_work, work_bytes, n), steps, lr, 1, nullptr, d_loss, st);
}

int hss_cdf_eval(const hss_cdf_model* d_model, const void* d_keys, uint32_t n, float* d_y, void* stream) {
    if (!d_model || (n > 0 && (!d_keys || !d_y))) return HSS_ERR_INVALID;
    if (n == 0) return HSS_OK;
    HSS_LAUNCH(k_cdf_eval, (n + 255) / 256, 256, 0, (cudaStream_t)stream, d_model, (const uint64_t*)d_keys, n, d_y);
    return cudaGetLastError() == cudaSuccess ? HSS_OK : HSS_ERR_CUDA;
}

int hss_cdf_propose(const hss_cdf_model* d_model, uint32_t p, uint32_t per_splitter, double delta, void* d_out_keys,
                    void* stream) {
    if (!d_model || p == 0 || per_splitter == 0 || !(delta >= 0.0) || (p > 1 && !d_out_keys)) return HSS_ERR_INVALID;
    if (p == 1) return HSS_OK;
    const uint64_t n = (uint64_t)(p - 1) * per_splitter;
    if (n > 0xffffffffull) return HSS_ERR_INVALID;
    HSS_LAUNCH(k_cdf_propose, (unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream, d_model, p, per_splitter, delta,
               40, (uint64_t*)d_out_keys);
    return cudaGetLastError() == cudaSuccess ? HSS_OK : HSS_ERR_CUDA;
}

}  // extern "C"
