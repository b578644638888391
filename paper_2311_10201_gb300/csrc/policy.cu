// The schedule policy network: parameters on the device (fbpt_policy) and its
// training kernels.  The network is used by the level scheduler (engine.cu,
// policy_forward) to pick how the coming level expands; it never changes a bit
// of the output.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>
#include <vector>

#include "internal.cuh"

using namespace fbpt;

extern "C" int fbpt_policy_param_count(void) { return 2 * kPolicyIn + kPolicyParams; }

extern "C" int fbpt_policy_create(const float* params, uint64_t count, fbpt_policy** out) {
    if (!out) return fail(FBPT_EINVAL, "fbpt_policy_create: out is NULL");
    *out = nullptr;
    const uint64_t want = 2 * kPolicyIn + kPolicyParams;
    if (!params || count != want)
        return fail(FBPT_EINVAL, "fbpt_policy_create: needs " + std::to_string(want) + " parameters");
    for (int i = 0; i < kPolicyIn; ++i)
        if (!(params[kPolicyIn + i] > 0.f)) return fail(FBPT_EINVAL, "fbpt_policy_create: input scales must be > 0");
    fbpt_policy* p = new fbpt_policy();
    std::memcpy(p->h_params, params, sizeof(float) * want);
    if (device_malloc(&p->d_params, sizeof(float) * want) != cudaSuccess ||
        cudaMemcpy(p->d_params, params, sizeof(float) * want, cudaMemcpyHostToDevice) != cudaSuccess) {
        cudaFree(p->d_params);
        delete p;
        cudaGetLastError();
        return fail(FBPT_ENOMEM, "fbpt_policy_create: device copy failed");
    }
    *out = p;
    return FBPT_OK;
}

extern "C" int fbpt_policy_destroy(fbpt_policy* p) {
    if (!p) return FBPT_OK;
    cudaFree(p->d_params);
    delete p;
    return FBPT_OK;
}

extern "C" int fbpt_policy_get(const fbpt_policy* p, float* params, uint64_t count) {
    const uint64_t want = 2 * kPolicyIn + kPolicyParams;
    if (!p || !params || count != want) return fail(FBPT_EINVAL, "fbpt_policy_get: bad arguments");
    std::memcpy(params, p->h_params, sizeof(float) * want);
    return FBPT_OK;
}

extern "C" int fbpt_policy_save(const fbpt_policy* p, const char* path) {
    if (!p || !path) return fail(FBPT_EINVAL, "fbpt_policy_save: null argument");
    FILE* f = std::fopen(path, "w");
    if (!f) return fail(FBPT_EINVAL, std::string("fbpt_policy_save: cannot write ") + path);
    const uint64_t want = 2 * kPolicyIn + kPolicyParams;
    bool ok = true;
    for (uint64_t i = 0; i < want && ok; ++i) ok = std::fprintf(f, "%.9g\n", (double)p->h_params[i]) > 0;
    ok = (std::fclose(f) == 0) && ok;
    return ok ? FBPT_OK : fail(FBPT_EINVAL, std::string("fbpt_policy_save: write failed on ") + path);
}

extern "C" int fbpt_policy_load(const char* path, fbpt_policy** out) {
    if (!path || !out) return fail(FBPT_EINVAL, "fbpt_policy_load: null argument");
    *out = nullptr;
    FILE* f = std::fopen(path, "r");
    if (!f) return fail(FBPT_EINVAL, std::string("fbpt_policy_load: cannot read ") + path);
    const uint64_t want = 2 * kPolicyIn + kPolicyParams;
    std::vector<float> v;
    char tok[64];
    bool bad = false;
    while (std::fscanf(f, "%63s", tok) == 1) {
        char* end = nullptr;
        const float x = std::strtof(tok, &end);
        if (end == tok || *end != '\0') {
            bad = true;
            break;
        }
        v.push_back(x);
        if (v.size() > want) break;
    }
    std::fclose(f);
    if (bad) return fail(FBPT_EINVAL, std::string("fbpt_policy_load: not a number in ") + path);
    if (v.size() != want)
        return fail(FBPT_EINVAL, "fbpt_policy_load: expected " + std::to_string(want) + " numbers in " + path);
    return fbpt_policy_create(v.data(), want, out);
}

// ---- training ----------------------------------------------------------------------
//
// Rows are levels from traces: six features, the action the level ran with and
// its log2 device time.  Loss: mean over rows of (out[action] - target)^2; only
// the taken action's output gets a gradient.  Full-batch Adam (Kingma and Ba,
// ICLR 2015) on the weights and biases; the input mean and scale stay fixed.

namespace fbpt {
namespace {

constexpr int kNP = 2 * kPolicyIn + kPolicyParams;  // 1,556 floats
constexpr int kOffW1 = 2 * kPolicyIn;
constexpr int kOffB1 = kOffW1 + kPolicyIn * kPolicyHidden;
constexpr int kOffW2 = kOffB1 + kPolicyHidden;
constexpr int kOffB2 = kOffW2 + kPolicyHidden * kPolicyHidden;
constexpr int kOffW3 = kOffB2 + kPolicyHidden;
constexpr int kOffB3 = kOffW3 + kPolicyHidden * kPolicyOut;

// Loss and gradient, and with an Adam step (adam_t > 0) the update too.
//
// What bounds it: FP32 multiply-adds, ~3,500 a row (forward 1,248, backward
// 2,272).  A warp takes 32 rows at a time and keeps their activations and errors
// unit-major in shared memory ([unit][row], rows padded to 36 floats), so that
// every contraction (layer 2 forward, its error, the gradient of W2) is a 32 x 32
// x 32 product in which a lane owns a 4 x 8 block: 32 independent accumulators,
// 16-byte shared loads without bank conflicts, short loops.  The gradients stay in
// registers over all of the warp's rows; the CTA's warps are summed in shared
// memory and the CTAs in FP64.  What is left is the latency of a tile's ~7,100
// instructions: 16 warps an SM (128 registers) take 65,536 rows in one round.
// Measured at 65,536 rows, one pass with its update: float atomics on a shared
// gradient, every lane of a warp at one address, 810 us; 12 warps an SM and two
// rounds 45 us; this form 39 us.
// The last CTA to add its share applies the Adam step and clears the gradient
// and the loss for the next one: one launch a step instead of two and two fills.
constexpr int kTrainThreads = 256;
constexpr int kTrainCtasPerSm = 2;
constexpr int kTileStride = 36;  // floats per unit's 32 rows

struct TrainWarp {
    // e: layer 2's activations, then its errors, then layer 1's errors
    alignas(16) float h1[kPolicyHidden][kTileStride], e[kPolicyHidden][kTileStride];
    float x[kPolicyIn][kTileStride], d[kTileStride];
    uint32_t a[kTileStride];
};

struct TrainSmem {
    TrainWarp warp[kTrainThreads / 32];
    alignas(16) float w1[kPolicyHidden][8];              // rows padded to 16-byte loads
    alignas(16) float w2[kPolicyHidden][kPolicyHidden];  // [unit][input]
    alignas(16) float w2t[kPolicyHidden][kPolicyHidden]; // [input][unit]
    float b1[kPolicyHidden], b2[kPolicyHidden];
    float w3[kPolicyOut][kPolicyHidden + 1];  // lanes read different rows: stride 33
    float b3[kPolicyOut], mu[8], sd[8];
    double loss;  // a CTA's sum of squares may be beyond FP32 where the mean is not
    uint32_t last;
};

// One Adam step (Kingma and Ba, ICLR 2015, Algorithm 1: beta1 = 0.9, beta2 =
// 0.999, eps = 1e-8) of a weight or bias with gradient gi: moments updated, the
// amount to subtract returned (the input mean and scale are not trained).
// The decay factors and their complements are each the float nearest to the
// decimal constant (1 - 0.999f would be 1.3e-5 away from 0.001), and the bias
// corrections 1 - beta^t are formed as -expm1(t log1p(-(1 - beta))), which
// keeps their relative error at a few float ulps for every t.
__device__ __forceinline__ float adam_step(float gi, float& m, float& v, float c1, float c2, float lr) {
    const float b1 = 0.9f, b2 = 0.999f, omb1 = 0.1f, omb2 = 0.001f, eps = 1e-8f;
    m = b1 * m + omb1 * gi;
    v = b2 * v + omb2 * gi * gi;
    return lr * (m / c1) / (sqrtf(v / c2) + eps);
}
__device__ __forceinline__ void adam_corrections(int t, float& c1, float& c2) {
    c1 = -expm1f((float)t * log1pf(-0.1f));
    c2 = -expm1f((float)t * log1pf(-0.001f));
}

// acc += a * b.  kGuard (a warp with a non-finite value among its rows): a
// factor that is zero adds nothing, whatever the other factor is.
template <bool kGuard>
__device__ __forceinline__ void grad_add(float& acc, float a, float b) {
    if (!kGuard || (a != 0.f && b != 0.f)) acc += a * b;
}

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }

// acc[i][c] += sum over k of A[k][4 x + i] * B[k][8 y + c] (a lane's 4 x 8 block of
// a 32 x 32 product; x = lane / 4, y = lane % 4).
template <int strideA>
__device__ __forceinline__ void block_product(const float (*A)[strideA], const float (*B)[kTileStride], uint32_t lane,
                                              float (&acc)[4][8]) {
    const uint32_t x = (lane >> 2) * 4, y = (lane & 3) * 8;
#pragma unroll 4
    for (int k = 0; k < kPolicyHidden; ++k) {
        const float4 a = ld4(&A[k][x]), p = ld4(&B[k][y]), q = ld4(&B[k][y + 4]);
        const float av[4] = {a.x, a.y, a.z, a.w}, bv[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[i][c] += av[i] * bv[c];
    }
}

// Gradient of W2: g[i][c] += sum over the rows r of e[lane / 4 + 8 i][r] * h1[lane % 4 + 4 c][r],
// and of b2 (unit `lane`).
template <bool kGuard>
__device__ __forceinline__ void grad_w2(const TrainWarp& w, uint32_t lane, float (&g)[4][8], float& gb2) {
    const uint32_t x = lane >> 2, y = lane & 3;
#pragma unroll 1
    for (int r = 0; r < 32; r += 4) {
        float4 e[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) e[i] = ld4(&w.e[x + 8 * i][r]);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const float4 h = ld4(&w.h1[y + 4 * c][r]);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                grad_add<kGuard>(g[i][c], e[i].x, h.x);
                grad_add<kGuard>(g[i][c], e[i].y, h.y);
                grad_add<kGuard>(g[i][c], e[i].z, h.z);
                grad_add<kGuard>(g[i][c], e[i].w, h.w);
            }
        }
        const float4 b = ld4(&w.e[lane][r]);
        gb2 += b.x; gb2 += b.y; gb2 += b.z; gb2 += b.w;
    }
}

// Gradients of row `lane` of W1 and of b1, from the first layer's errors (in w.e).
template <bool kGuard>
__device__ __forceinline__ void grad_w1(const TrainWarp& w, uint32_t lane, float (&g1)[kPolicyIn], float& gb1) {
#pragma unroll 1
    for (int r = 0; r < 32; r += 4) {
        const float4 e = ld4(&w.e[lane][r]);
#pragma unroll
        for (int q = 0; q < kPolicyIn; ++q) {
            const float4 x = ld4(&w.x[q][r]);
            if (!kGuard || e.x != 0.f) g1[q] += e.x * x.x;
            if (!kGuard || e.y != 0.f) g1[q] += e.y * x.y;
            if (!kGuard || e.z != 0.f) g1[q] += e.z * x.z;
            if (!kGuard || e.w != 0.f) g1[q] += e.w * x.w;
        }
        gb1 += e.x; gb1 += e.y; gb1 += e.z; gb1 += e.w;
    }
}

__global__ void __launch_bounds__(kTrainThreads, kTrainCtasPerSm)
    k_mlp_grad(float* __restrict__ P, const float* __restrict__ X, const uint32_t* __restrict__ act,
               const float* __restrict__ Y, uint64_t rows, double* grad, double* loss, unsigned* done, float* m,
               float* v, int adam_t, float lr) {
    extern __shared__ float4 train_smem[];
    TrainSmem& s = *reinterpret_cast<TrainSmem*>(train_smem);
    const uint32_t t = threadIdx.x, lane = lane_id(), warp = t >> 5;
    constexpr int kPer = (kNP + kTrainThreads - 1) / kTrainThreads;  // parameters a thread loads, and updates
    float pv[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) pv[k] = t + k * kTrainThreads < kNP ? __ldcg(&P[t + k * kTrainThreads]) : 0.f;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int i = t + k * kTrainThreads;
        const float p = pv[k];
        if (i < kPolicyIn) s.mu[i] = p;
        else if (i < kOffW1) s.sd[i - kPolicyIn] = p;
        else if (i < kOffB1) s.w1[(i - kOffW1) / kPolicyIn][(i - kOffW1) % kPolicyIn] = p;
        else if (i < kOffW2) s.b1[i - kOffB1] = p;
        else if (i < kOffB2) {
            const int j = (i - kOffW2) / kPolicyHidden, q = (i - kOffW2) % kPolicyHidden;
            s.w2[j][q] = p;
            s.w2t[q][j] = p;
        } else if (i < kOffW3) s.b2[i - kOffB2] = p;
        else if (i < kOffB3) s.w3[(i - kOffW3) / kPolicyHidden][(i - kOffW3) % kPolicyHidden] = p;
        else if (i < kNP) s.b3[i - kOffB3] = p;
    }
    if (t == 0) s.loss = 0.0;
    __syncthreads();
    const float inv = 2.0f / (float)rows;
    float lsum = 0.f;
    float g2[4][8] = {}, g1[kPolicyIn] = {}, g3[kPolicyOut] = {}, gb1 = 0.f, gb2 = 0.f, gb3 = 0.f;
    TrainWarp& w = s.warp[warp];
    const uint32_t bx = (lane >> 2) * 4, by = (lane & 3) * 8;
    const uint64_t nwarp = (uint64_t)gridDim.x * (kTrainThreads / 32);
    for (uint64_t base = ((uint64_t)blockIdx.x * (kTrainThreads / 32) + warp) * 32; base < rows; base += nwarp * 32) {
        // a lane is a row: features, layer 1
        const uint64_t r = base + lane;
        const bool in = r < rows;
        float xn[kPolicyIn];
        float fin = 0.f;  // finite unless a value of the row is not
#pragma unroll
        for (int k = 0; k < kPolicyIn; ++k) {
            xn[k] = in ? (__ldg(&X[r * kPolicyIn + k]) - s.mu[k]) / s.sd[k] : 0.f;
            w.x[k][lane] = xn[k];
            fin += fabsf(xn[k]);
        }
        const uint32_t act_r = in ? __ldg(&act[r]) : 0u;
        const uint32_t a = act_r < (uint32_t)kPolicyOut ? act_r : 0u;
        const float y = in ? __ldg(&Y[r]) : 0.f;
#pragma unroll 4
        for (int j = 0; j < kPolicyHidden; ++j) {
            const float4 wa = ld4(&s.w1[j][0]);
            const float2 wb = *reinterpret_cast<const float2*>(&s.w1[j][4]);
            float z = s.b1[j];
            z += wa.x * xn[0]; z += wa.y * xn[1]; z += wa.z * xn[2]; z += wa.w * xn[3];
            z += wb.x * xn[4]; z += wb.y * xn[5];
            z = in && z > 0.f ? z : 0.f;
            w.h1[j][lane] = z;
            fin += z;
        }
        __syncwarp();
        // layer 2: units bx .. bx + 3 of rows by .. by + 7
        float acc[4][8];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[i][c] = s.b2[bx + i];
        block_product<kPolicyHidden>(s.w2t, w.h1, lane, acc);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[i][c] = base + by + c < rows && acc[i][c] > 0.f ? acc[i][c] : 0.f;
            *reinterpret_cast<float4*>(&w.e[bx + i][by]) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
            *reinterpret_cast<float4*>(&w.e[bx + i][by + 4]) = make_float4(acc[i][4], acc[i][5], acc[i][6], acc[i][7]);
        }
        __syncwarp();
        // a lane is a row: the taken output and its error
        float o = s.b3[a];
#pragma unroll 8
        for (int j = 0; j < kPolicyHidden; ++j) o += s.w3[a][j] * w.e[j][lane];
        const float res = in ? o - y : 0.f;
        lsum += res * res;
        const float d = in ? inv * res : 0.f;
        w.d[lane] = d;
        w.a[lane] = a;
        __syncwarp();
        // gradients of column `lane` of W3, and of b3 in lanes 0 .. 7
#pragma unroll 1
        for (int q = 0; q < 32; q += 4) {
            const float4 h = ld4(&w.e[lane][q]), dd = ld4(&w.d[q]);
            const uint4 aa = *reinterpret_cast<const uint4*>(&w.a[q]);
            const float hv[4] = {h.x, h.y, h.z, h.w}, dv[4] = {dd.x, dd.y, dd.z, dd.w};
            const uint32_t av[4] = {aa.x, aa.y, aa.z, aa.w};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
#pragma unroll
                for (int k = 0; k < kPolicyOut; ++k)
                    if (av[c] == (uint32_t)k) g3[k] += dv[c] * hv[c];
                if (av[c] == lane) gb3 += dv[c];
            }
        }
        __syncwarp();
        // errors of layer 2, in its activations' place
#pragma unroll 8
        for (int j = 0; j < kPolicyHidden; ++j) {
            const float e = w.e[j][lane] > 0.f ? d * s.w3[a][j] : 0.f;
            w.e[j][lane] = e;
            fin += fabsf(e);
        }
        const bool guard = __any_sync(0xffffffffu, !(fin < __int_as_float(0x7f800000)));
        __syncwarp();
        if (guard) grad_w2<true>(w, lane, g2, gb2);
        else grad_w2<false>(w, lane, g2, gb2);
        // errors of layer 1: W2^T e where the unit is on
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[i][c] = 0.f;
        block_product<kPolicyHidden>(s.w2, w.e, lane, acc);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[i][c] = w.h1[bx + i][by + c] > 0.f ? acc[i][c] : 0.f;
            *reinterpret_cast<float4*>(&w.e[bx + i][by]) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
            *reinterpret_cast<float4*>(&w.e[bx + i][by + 4]) = make_float4(acc[i][4], acc[i][5], acc[i][6], acc[i][7]);
        }
        __syncwarp();
        if (guard) grad_w1<true>(w, lane, g1, gb1);
        else grad_w1<false>(w, lane, g1, gb1);
        __syncwarp();
    }
    lsum = warp_sum(lsum);
    // the CTA's warps into one gradient (in the tiles' place), one warp after another
    __syncthreads();
    float* g = reinterpret_cast<float*>(s.warp);
    static_assert(sizeof(s.warp) >= sizeof(float) * kNP, "the CTA's gradient fits the tiles");
    for (int i = t; i < kNP; i += kTrainThreads) g[i] = 0.f;
    __syncthreads();
    for (uint32_t k = 0; k < kTrainThreads / 32; ++k) {
        if (warp == k) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    g[kOffW2 + ((lane >> 2) + 8 * i) * kPolicyHidden + (lane & 3) + 4 * c] += g2[i][c];
#pragma unroll
            for (int q = 0; q < kPolicyIn; ++q) g[kOffW1 + lane * kPolicyIn + q] += g1[q];
#pragma unroll
            for (int q = 0; q < kPolicyOut; ++q) g[kOffW3 + q * kPolicyHidden + lane] += g3[q];
            if (lane < kPolicyOut) g[kOffB3 + lane] += gb3;
            g[kOffB1 + lane] += gb1;
            g[kOffB2 + lane] += gb2;
            if (lane == 0) s.loss += (double)lsum;
        }
        __syncthreads();
    }
    for (int i = kOffW1 + t; i < kNP; i += kTrainThreads)
        if (g[i] != 0.f) atomicAdd(&grad[i], (double)g[i]);
    if (t == 0 && s.loss != 0.0) atomicAdd(loss, s.loss / (double)rows);
    if (adam_t <= 0) return;
    __threadfence();
    __syncthreads();
    if (t == 0) s.last = atomicAdd(done, 1u) + 1u == gridDim.x;
    __syncthreads();
    if (!s.last) return;
    __threadfence();
    float c1, c2;
    adam_corrections(adam_t, c1, c2);
    // all loads of a thread's weights go out before any is updated
    double gv[kPer];
    float mv[kPer], vv[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int i = t + k * kTrainThreads;
        const bool in = i >= kOffW1 && i < kNP;
        gv[k] = in ? __ldcg(&grad[i]) : 0.0;
        pv[k] = in ? __ldcg(&P[i]) : 0.f;
        mv[k] = in ? __ldcg(&m[i]) : 0.f;
        vv[k] = in ? __ldcg(&v[i]) : 0.f;
    }
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int i = t + k * kTrainThreads;
        if (i < kOffW1 || i >= kNP) continue;
        P[i] = pv[k] - adam_step((float)gv[k], mv[k], vv[k], c1, c2, lr);
        m[i] = mv[k];
        v[i] = vv[k];
        grad[i] = 0.0;
    }
    if (t == 0) {
        *loss = 0.0;
        *done = 0u;
    }
}

__global__ void k_adam(float* P, const double* grad, float* m, float* v, int t, float lr) {
    float c1, c2;
    adam_corrections(t, c1, c2);
    for (int i = kOffW1 + blockIdx.x * blockDim.x + threadIdx.x; i < kNP; i += gridDim.x * blockDim.x)
        P[i] -= adam_step((float)grad[i], m[i], v[i], c1, c2, lr);
}

// Device buffers of one training call, allocated and freed on its stream.
struct TrainBufs {
    cudaStream_t st = nullptr;
    float *P = nullptr, *m = nullptr, *v = nullptr, *X = nullptr, *Y = nullptr;
    uint32_t* A = nullptr;
    double *grad = nullptr, *loss = nullptr;  // the CTAs' FP32 sums are added up in FP64
    unsigned* done = nullptr;  // CTAs of the running step that have added their gradient
    explicit TrainBufs(cudaStream_t s) : st(s) {}
    ~TrainBufs() {
        for (void* p : {(void*)P, (void*)grad, (void*)m, (void*)v, (void*)loss, (void*)X, (void*)Y, (void*)A, (void*)done})
            if (p) cudaFreeAsync(p, st);
        cudaStreamSynchronize(st);
    }
};

// Parameters (and, with rows > 0, the trace rows) to the device; Adam moments zeroed.
int upload(TrainBufs& b, const float* params, const float* X, const uint32_t* A, const float* Y, uint64_t rows) {
    const cudaStream_t st = b.st;
    FBPT_CUDA_TRY(pool_malloc(nullptr, &b.P, sizeof(float) * kNP, st));
    FBPT_CUDA_TRY(pool_malloc(nullptr, &b.grad, sizeof(double) * kNP, st));
    FBPT_CUDA_TRY(pool_malloc(nullptr, &b.m, sizeof(float) * kNP, st));
    FBPT_CUDA_TRY(pool_malloc(nullptr, &b.v, sizeof(float) * kNP, st));
    FBPT_CUDA_TRY(pool_malloc(nullptr, &b.loss, sizeof(double), st));
    FBPT_CUDA_TRY(cudaMemcpyAsync(b.P, params, sizeof(float) * kNP, cudaMemcpyHostToDevice, st));
    FBPT_CUDA_TRY(cudaMemsetAsync(b.m, 0, sizeof(float) * kNP, st));
    FBPT_CUDA_TRY(cudaMemsetAsync(b.v, 0, sizeof(float) * kNP, st));
    FBPT_CUDA_TRY(cudaMemsetAsync(b.grad, 0, sizeof(double) * kNP, st));
    FBPT_CUDA_TRY(cudaMemsetAsync(b.loss, 0, sizeof(double), st));
    if (rows) {
        FBPT_CUDA_TRY(pool_malloc(nullptr, &b.done, sizeof(unsigned), st));
        FBPT_CUDA_TRY(cudaMemsetAsync(b.done, 0, sizeof(unsigned), st));
        FBPT_CUDA_TRY(pool_malloc(nullptr, &b.X, sizeof(float) * kPolicyIn * rows, st));
        FBPT_CUDA_TRY(pool_malloc(nullptr, &b.Y, sizeof(float) * rows, st));
        FBPT_CUDA_TRY(pool_malloc(nullptr, &b.A, sizeof(uint32_t) * rows, st));
        FBPT_CUDA_TRY(cudaMemcpyAsync(b.X, X, sizeof(float) * kPolicyIn * rows, cudaMemcpyHostToDevice, st));
        FBPT_CUDA_TRY(cudaMemcpyAsync(b.Y, Y, sizeof(float) * rows, cudaMemcpyHostToDevice, st));
        FBPT_CUDA_TRY(cudaMemcpyAsync(b.A, A, sizeof(uint32_t) * rows, cudaMemcpyHostToDevice, st));
    }
    return FBPT_OK;
}

// Adds the rows' loss and gradient to b.loss and b.grad (zero before); with
// adam_t > 0 applies Adam step adam_t and leaves both zero again.
int grad_pass(TrainBufs& b, uint64_t rows, int adam_t = 0, float lr = 0.f) {
    // a warp takes 32 rows at a time; up to kTrainCtasPerSm CTAs an SM
    FBPT_CUDA_TRY(cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmem)));
    // and no more CTAs than the rounds that takes need (each adds 1,544 atomics)
    const uint64_t warps = kTrainThreads / 32, tiles = (rows + 31) / 32;
    const uint64_t most = (uint64_t)device_sm_count() * kTrainCtasPerSm * warps;
    const uint64_t rounds = (tiles + most - 1) / most;
    const int blocks = (int)((tiles + rounds * warps - 1) / (rounds * warps));
    k_mlp_grad<<<blocks, kTrainThreads, sizeof(TrainSmem), b.st>>>(b.P, b.X, b.A, b.Y, rows, b.grad, b.loss, b.done, b.m,
                                                                    b.v, adam_t, lr);
    FBPT_CUDA_TRY(cudaGetLastError());
    return FBPT_OK;
}

// Deterministic initial weights: He-scaled normals from SplitMix64 + Box-Muller.
uint64_t splitmix(uint64_t& s) {
    uint64_t z = (s += 0x9E3779B97F4A7C15ULL);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

double normal01(uint64_t& s) {
    const double u1 = ((splitmix(s) >> 11) + 0.5) / 9007199254740992.0;
    const double u2 = ((splitmix(s) >> 11) + 0.5) / 9007199254740992.0;
    return std::sqrt(-2.0 * std::log(u1)) * std::cos(6.283185307179586 * u2);
}

}  // namespace
}  // namespace fbpt

extern "C" int fbpt_policy_loss_grad(const float* params, const float* features, const uint32_t* actions,
                                     const float* targets, uint64_t rows, float* loss, float* grad, void* stream) {
    if (!params || !features || !actions || !targets || rows == 0 || !loss || !grad)
        return fail(FBPT_EINVAL, "fbpt_policy_loss_grad: bad arguments");
    TrainBufs b((cudaStream_t)stream);
    FBPT_TRY(upload(b, params, features, actions, targets, rows));
    FBPT_TRY(grad_pass(b, rows));
    double g[kNP], l = 0.0;
    FBPT_CUDA_TRY(cudaMemcpyAsync(g, b.grad, sizeof(g), cudaMemcpyDeviceToHost, b.st));
    FBPT_CUDA_TRY(cudaMemcpyAsync(&l, b.loss, sizeof(double), cudaMemcpyDeviceToHost, b.st));
    FBPT_CUDA_TRY(cudaStreamSynchronize(b.st));
    *loss = (float)l;
    for (int i = 0; i < kNP; ++i) grad[i] = i < kOffW1 ? 0.f : (float)g[i];
    return FBPT_OK;
}

extern "C" int fbpt_policy_adam_step(float* params, const float* grad, float* m, float* v, uint32_t t, float lr,
                                     void* stream) {
    if (!params || !grad || !m || !v || t == 0 || !(lr > 0.f))
        return fail(FBPT_EINVAL, "fbpt_policy_adam_step: bad arguments");
    TrainBufs b((cudaStream_t)stream);
    FBPT_TRY(upload(b, params, nullptr, nullptr, nullptr, 0));
    double g[kNP];
    for (int i = 0; i < kNP; ++i) g[i] = grad[i];
    FBPT_CUDA_TRY(cudaMemcpyAsync(b.grad, g, sizeof(g), cudaMemcpyHostToDevice, b.st));
    FBPT_CUDA_TRY(cudaMemcpyAsync(b.m, m, sizeof(float) * kNP, cudaMemcpyHostToDevice, b.st));
    FBPT_CUDA_TRY(cudaMemcpyAsync(b.v, v, sizeof(float) * kNP, cudaMemcpyHostToDevice, b.st));
    k_adam<<<8, 256, 0, b.st>>>(b.P, b.grad, b.m, b.v, (int)t, lr);
    FBPT_CUDA_TRY(cudaGetLastError());
    FBPT_CUDA_TRY(cudaMemcpyAsync(params, b.P, sizeof(float) * kNP, cudaMemcpyDeviceToHost, b.st));
    FBPT_CUDA_TRY(cudaMemcpyAsync(m, b.m, sizeof(float) * kNP, cudaMemcpyDeviceToHost, b.st));
    FBPT_CUDA_TRY(cudaMemcpyAsync(v, b.v, sizeof(float) * kNP, cudaMemcpyDeviceToHost, b.st));
    FBPT_CUDA_TRY(cudaStreamSynchronize(b.st));
    return FBPT_OK;
}

extern "C" int fbpt_policy_train(const float* features, const uint32_t* actions, const float* targets, uint64_t rows,
                                 const fbpt_train_opts* opts, const float* init_params, fbpt_policy** out,
                                 float* final_loss) {
    if (!features || !actions || !targets || rows == 0 || !out) return fail(FBPT_EINVAL, "fbpt_policy_train: bad arguments");
    fbpt_train_opts o = {};
    if (opts) o = *opts;
    const uint32_t steps = o.steps ? o.steps : 2000;
    const float lr = o.lr > 0.f ? o.lr : 3e-3f;
    float P[kNP];
    if (init_params) {
        std::memcpy(P, init_params, sizeof(P));
    } else {
        for (int k = 0; k < kPolicyIn; ++k) {  // input mean and scale from the data
            double s = 0, s2 = 0;
            for (uint64_t r = 0; r < rows; ++r) {
                const double x = features[r * kPolicyIn + k];
                s += x;
                s2 += x * x;
            }
            const double mu = s / rows, var = s2 / rows - mu * mu;
            P[k] = (float)mu;
            P[kPolicyIn + k] = (float)(var > 1e-6 ? std::sqrt(var) : 1.0);
        }
        uint64_t st = o.seed ^ 0x5EEDull;
        auto fill = [&](int off, int count, int fan_in) {
            const double sc = std::sqrt(2.0 / fan_in);
            for (int i = 0; i < count; ++i) P[off + i] = (float)(sc * normal01(st));
        };
        fill(kOffW1, kPolicyIn * kPolicyHidden, kPolicyIn);
        fill(kOffW2, kPolicyHidden * kPolicyHidden, kPolicyHidden);
        fill(kOffW3, kPolicyHidden * kPolicyOut, kPolicyHidden);
        for (int i = 0; i < kPolicyHidden; ++i) P[kOffB1 + i] = P[kOffB2 + i] = 0.f;
        double ym = 0;  // start the outputs at the mean target
        for (uint64_t r = 0; r < rows; ++r) ym += targets[r];
        for (int i = 0; i < kPolicyOut; ++i) P[kOffB3 + i] = (float)(ym / rows);
    }
    TrainBufs b((cudaStream_t)o.stream);
    FBPT_TRY(upload(b, P, features, actions, targets, rows));
    for (uint32_t t = 1; t <= steps; ++t) FBPT_TRY(grad_pass(b, rows, (int)t, lr));
    FBPT_TRY(grad_pass(b, rows));
    FBPT_CUDA_TRY(cudaMemcpyAsync(P, b.P, sizeof(P), cudaMemcpyDeviceToHost, b.st));
    double fl = 0.0;
    FBPT_CUDA_TRY(cudaMemcpyAsync(&fl, b.loss, sizeof(double), cudaMemcpyDeviceToHost, b.st));
    FBPT_CUDA_TRY(cudaStreamSynchronize(b.st));
    if (final_loss) *final_loss = (float)fl;
    return fbpt_policy_create(P, kNP, out);
}
