// policy.cu -- learned push/pull direction policy: FP32 MLP 10 -> 32 -> 32 -> 3
// (ReLU) with its forward, backward (softmax cross-entropy on labels, or
// least-squares regression of the outputs on per-row targets) and Adam update
// in this library's own kernels.  The paper has no learned policy; it stands in
// for the Beamer direction switch the paper cites (Section 5).
#include "common.cuh"
#include "policy_dev.cuh"

#include <cmath>
#include <vector>

struct bfs_policy {
    float* w = nullptr;   // device [NWEIGHTS]
    float* m1 = nullptr;  // Adam first moment [NPARAM]
    float* m2 = nullptr;  // Adam second moment [NPARAM]
    float* grad = nullptr;
    float* loss = nullptr;
    float* part = nullptr;  // the training CTAs' partial gradients [part_ctas][NPARAM + 1], made on first use
    int part_ctas = 0;
    std::vector<float> host;  // host mirror of w
};

namespace bfsgb {

const float* policy_device_weights(const bfs_policy* p) { return p ? p->w : nullptr; }

namespace {

// ------------------------------------------------------------ one row a lane
// A warp works on 32 rows, one per lane; activations stay in registers and
// the weights come from shared memory in broadcast 16-byte loads.  Sums run in
// the order bias, k = 0, 1, ... with one FMA a term.  The unit of work is
// FP32 arithmetic (the three layers and their gradients are 1.6 GFLOP at
// 200,000 rows; the inputs are 10 MB), so two sums at a time go through the
// packed fma.rn.f32x2, which is two ordinary FP32 FMAs in one issue slot.

// Weights in shared memory: both orders of the layers that are multiplied
// along their rows in the forward pass and along their columns in the backward
// pass, so that neighbouring sums are neighbours in memory.
struct alignas(16) MlpSmem {
    float w1t[MLP_IN][MLP_H];  // [k][j]
    float w2t[MLP_H][MLP_H];   // [k][j]
    float w2[MLP_H][MLP_H];    // [j][k]
    float w3[MLP_OUT][MLP_H];
    float b1[MLP_H], b2[MLP_H], b3[4];
    float mean[MLP_IN], istd[MLP_IN];
};

__device__ __forceinline__ void load_weights(MlpSmem& s, const float* __restrict__ w) {
    for (int i = threadIdx.x; i < MLP_H * MLP_IN; i += blockDim.x) s.w1t[i % MLP_IN][i / MLP_IN] = w[OFF_W1 + i];
    for (int i = threadIdx.x; i < MLP_H * MLP_H; i += blockDim.x) {
        const float x = w[OFF_W2 + i];
        s.w2[i / MLP_H][i % MLP_H] = x;
        s.w2t[i % MLP_H][i / MLP_H] = x;
    }
    for (int i = threadIdx.x; i < MLP_OUT * MLP_H; i += blockDim.x) s.w3[i / MLP_H][i % MLP_H] = w[OFF_W3 + i];
    for (int i = threadIdx.x; i < MLP_H; i += blockDim.x) {
        s.b1[i] = w[OFF_B1 + i];
        s.b2[i] = w[OFF_B2 + i];
    }
    for (int i = threadIdx.x; i < MLP_IN; i += blockDim.x) {
        s.mean[i] = w[OFF_MEAN + i];
        s.istd[i] = w[OFF_ISTD + i];
    }
    if (threadIdx.x < MLP_OUT) s.b3[threadIdx.x] = w[OFF_B3 + threadIdx.x];
    __syncthreads();
}

// {a.x * b.x + c.x, a.y * b.y + c.y}, each rounded once
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    unsigned long long r, x, y, z;
    asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(y) : "f"(b.x), "f"(b.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(z) : "f"(c.x), "f"(c.y));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(x), "l"(y), "l"(z));
    float2 d;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(r));
    return d;
}

// acc[j] += row[j] * x over a 16-byte aligned shared-memory row of 32
__device__ __forceinline__ void axpy32(float (&acc)[MLP_H], const float* row, float x) {
    const float2 xx = make_float2(x, x);
#pragma unroll
    for (int q = 0; q < MLP_H / 4; ++q) {
        const float4 w = *reinterpret_cast<const float4*>(row + 4 * q);
        const float2 lo = fma2(make_float2(w.x, w.y), xx, make_float2(acc[4 * q], acc[4 * q + 1]));
        const float2 hi = fma2(make_float2(w.z, w.w), xx, make_float2(acc[4 * q + 2], acc[4 * q + 3]));
        acc[4 * q] = lo.x;
        acc[4 * q + 1] = lo.y;
        acc[4 * q + 2] = hi.x;
        acc[4 * q + 3] = hi.y;
    }
}

__device__ __forceinline__ void forward_row(const MlpSmem& s, const float (&xn)[MLP_IN], float (&h1)[MLP_H],
                                            float (&h2)[MLP_H], float (&z)[MLP_OUT]) {
#pragma unroll
    for (int j = 0; j < MLP_H; ++j) h1[j] = s.b1[j];
#pragma unroll
    for (int k = 0; k < MLP_IN; ++k) axpy32(h1, s.w1t[k], xn[k]);
#pragma unroll
    for (int j = 0; j < MLP_H; ++j) {
        h1[j] = fmaxf(h1[j], 0.0f);
        h2[j] = s.b2[j];
    }
#pragma unroll
    for (int k = 0; k < MLP_H; ++k) axpy32(h2, s.w2t[k], h1[k]);
#pragma unroll
    for (int j = 0; j < MLP_H; ++j) h2[j] = fmaxf(h2[j], 0.0f);
#pragma unroll
    for (int c = 0; c < MLP_OUT; ++c) {
        float a = s.b3[c];
#pragma unroll
        for (int k = 0; k < MLP_H; ++k) a = fmaf(s.w3[c][k], h2[k], a);
        z[c] = a;
    }
}

__global__ void __launch_bounds__(128) mlp_forward_kernel(const float* __restrict__ w, const float* __restrict__ X,
                                                          int64_t rows, float* __restrict__ logits) {
    __shared__ MlpSmem s;
    load_weights(s, w);
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < rows; r += (int64_t)gridDim.x * blockDim.x) {
        asm volatile("" ::: "memory");  // the weights are read again for each row, not kept (spilled) across rows
        float xn[MLP_IN], h1[MLP_H], h2[MLP_H], z[MLP_OUT];
#pragma unroll
        for (int k = 0; k < MLP_IN; ++k) xn[k] = (X[r * MLP_IN + k] - s.mean[k]) * s.istd[k];
        forward_row(s, xn, h1, h2, z);
#pragma unroll
        for (int c = 0; c < MLP_OUT; ++c) logits[r * MLP_OUT + c] = z[c];
    }
}

// ------------------------------------------------------------ training
constexpr int TR_T = 128;         // threads of a training CTA
constexpr int TR_W = TR_T / 32;
constexpr int TR_PER_SM = 2;      // resident CTAs (244 registers a thread, 255 with the softmax)
constexpr int TR_LD = 36;         // row pitch of the staged activations: 16-byte stores of 8 lanes then hit 8 bank groups
constexpr int NPART = NPARAM + 1; // a CTA's partial gradient, then its share of the loss

// A warp's 32 rows of two activation arrays, staged for the outer products.
struct alignas(16) MlpStage {
    float a[32][TR_LD];
    float b[32][TR_LD];
    float x[32][12];
    float z[32][4];
};

struct alignas(16) MlpTrainSmem {
    MlpSmem w;
    union {
        MlpStage st[TR_W];
        float part[TR_W][NPART + 1];
    };
};

__device__ __forceinline__ void stage32(float (*dst)[TR_LD], const float (&v)[MLP_H]) {
    float* d = dst[lane_id()];
#pragma unroll
    for (int q = 0; q < MLP_H / 4; ++q)
        *reinterpret_cast<float4*>(d + 4 * q) = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
}

// Forward, loss, backward and this CTA's share of the gradient.
// REGRESS = false: mean softmax cross-entropy on the labels y.  REGRESS =
// true: mean of sum_c (z_c - t_c)^2 / 2 on the row's targets t (3 floats),
// dL/dz = z - t.
//
// A parameter's gradient is a sum over rows of products of two activations:
//   dW1[j][k] = sum da1_j xn_k, db1 = sum da1, dW2[j][k] = sum da2_j h1_k,
//   db2 = sum da2, dW3[c][k] = sum dz_c h2_k, db3 = sum dz.
// Each warp stages its 32 rows' activations in shared memory and adds their
// outer products to its own register tile (dW2: 4 x 8 entries a lane, three
// 16-byte loads for 32 FMAs), over all the rows it is dealt; the warps' tiles
// are added once at the end, and a CTA writes one partial gradient, so no
// activation goes to memory and no sum goes through an atomic.  Writing every
// row's 121 activations out (97 MB at 200,000 rows) and re-reading them by
// 1,507 reduction threads a chunk took 444 us a step.
template <bool REGRESS>
__global__ void __launch_bounds__(TR_T, TR_PER_SM)
    mlp_train_kernel(const float* __restrict__ w, const float* __restrict__ X, const int32_t* __restrict__ y,
                     const float* __restrict__ t, int64_t rows, float* __restrict__ part) {
    extern __shared__ __align__(16) unsigned char mlp_train_dyn[];
    MlpTrainSmem& sm = *reinterpret_cast<MlpTrainSmem*>(mlp_train_dyn);
    load_weights(sm.w, w);
    const int lane = (int)lane_id(), warp = (int)(threadIdx.x >> 5);
    MlpStage& st = sm.st[warp];
    const float inv_rows = 1.0f / (float)rows;
    const int j0 = (lane >> 2) * 4, k0 = (lane & 3) * 8;  // this lane's tile of dW2
    float g2[4][8], g1[MLP_IN], g3[MLP_OUT], gb1 = 0.0f, gb2 = 0.0f, gb3 = 0.0f, lsum = 0.0f;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int k = 0; k < 8; ++k) g2[i][k] = 0.0f;
#pragma unroll
    for (int k = 0; k < MLP_IN; ++k) g1[k] = 0.0f;
#pragma unroll
    for (int c = 0; c < MLP_OUT; ++c) g3[c] = 0.0f;

    for (int64_t r0 = ((int64_t)blockIdx.x * TR_W + warp) * 32; r0 < rows; r0 += (int64_t)gridDim.x * TR_W * 32) {
        const int64_t r = r0 + lane;
        const bool valid = r < rows;
        // the tile's inputs in one contiguous run of loads, rows apart in shared memory
        const int64_t x0 = r0 * MLP_IN, xe = rows * MLP_IN;
#pragma unroll
        for (int k = 0; k < MLP_IN; ++k) {
            const int i = k * 32 + lane;
            st.x[i / MLP_IN][i % MLP_IN] = x0 + i < xe ? X[x0 + i] : 0.0f;
        }
        __syncwarp();
        float xn[MLP_IN], h1[MLP_H], h2[MLP_H], z[MLP_OUT], dz[MLP_OUT];
#pragma unroll
        for (int k = 0; k < MLP_IN; ++k) xn[k] = (st.x[lane][k] - sm.w.mean[k]) * sm.w.istd[k];
        forward_row(sm.w, xn, h1, h2, z);
        if (REGRESS) {
#pragma unroll
            for (int c = 0; c < MLP_OUT; ++c) {
                const float e = valid ? z[c] - t[r * MLP_OUT + c] : 0.0f;
                lsum = fmaf(0.5f * e, e, lsum);
                dz[c] = e * inv_rows;
            }
        } else {
            const float zmax = fmaxf(z[0], fmaxf(z[1], z[2]));
            float se = 0.0f;
#pragma unroll
            for (int c = 0; c < MLP_OUT; ++c) se += expf(z[c] - zmax);
            const float lse = zmax + logf(se);
            const int yr = valid ? y[r] : 0;
            if (valid) lsum += lse - (yr == 0 ? z[0] : yr == 1 ? z[1] : z[2]);
#pragma unroll
            for (int c = 0; c < MLP_OUT; ++c)
                dz[c] = valid ? (expf(z[c] - lse) - (c == yr ? 1.0f : 0.0f)) * inv_rows : 0.0f;
        }
        if (!valid) {  // rows past the end add 0 * 0, whatever the weights hold
#pragma unroll
            for (int j = 0; j < MLP_H; ++j) h1[j] = h2[j] = 0.0f;
#pragma unroll
            for (int k = 0; k < MLP_IN; ++k) xn[k] = 0.0f;
        }
        float da2[MLP_H], da1[MLP_H];
#pragma unroll
        for (int j = 0; j < MLP_H; ++j) {
            float d = 0.0f;
#pragma unroll
            for (int c = 0; c < MLP_OUT; ++c) d = fmaf(sm.w.w3[c][j], dz[c], d);
            da2[j] = h2[j] > 0.0f ? d : 0.0f;
            da1[j] = 0.0f;
        }
        stage32(st.a, da2);
        stage32(st.b, h1);
#pragma unroll
        for (int k = 0; k < MLP_IN; ++k) st.x[lane][k] = xn[k];
        *reinterpret_cast<float4*>(st.z[lane]) = make_float4(dz[0], dz[1], dz[2], 0.0f);
#pragma unroll
        for (int j = 0; j < MLP_H; ++j) axpy32(da1, sm.w.w2[j], da2[j]);
#pragma unroll
        for (int k = 0; k < MLP_H; ++k) da1[k] = h1[k] > 0.0f ? da1[k] : 0.0f;
        __syncwarp();
#pragma unroll 4
        for (int q = 0; q < 32; ++q) {
            const float4 da = *reinterpret_cast<const float4*>(&st.a[q][j0]);
            const float4 p0 = *reinterpret_cast<const float4*>(&st.b[q][k0]);
            const float4 p1 = *reinterpret_cast<const float4*>(&st.b[q][k0 + 4]);
            const float dv[4] = {da.x, da.y, da.z, da.w};
            const float hv[8] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int k = 0; k < 8; k += 2) {
                    const float2 o = fma2(make_float2(hv[k], hv[k + 1]), make_float2(dv[i], dv[i]),
                                          make_float2(g2[i][k], g2[i][k + 1]));
                    g2[i][k] = o.x;
                    g2[i][k + 1] = o.y;
                }
            gb2 += st.a[q][lane];
        }
        __syncwarp();
        stage32(st.a, da1);
        stage32(st.b, h2);
        __syncwarp();
#pragma unroll 4
        for (int q = 0; q < 32; ++q) {
            const float d1 = st.a[q][lane], v2 = st.b[q][lane];
            const float4 dq = *reinterpret_cast<const float4*>(st.z[q]);
            gb1 += d1;
#pragma unroll
            for (int k = 0; k < MLP_IN; ++k) g1[k] = fmaf(d1, st.x[q][k], g1[k]);
            g3[0] = fmaf(dq.x, v2, g3[0]);
            g3[1] = fmaf(dq.y, v2, g3[1]);
            g3[2] = fmaf(dq.z, v2, g3[2]);
            gb3 += lane == 0 ? dq.x : lane == 1 ? dq.y : dq.z;
        }
        __syncwarp();
    }
    lsum = warp_sum(lsum);
    __syncthreads();  // every warp is done with its staged rows: the partials take their place
    float* o = sm.part[warp];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int k = 0; k < 8; ++k) o[OFF_W2 + (j0 + i) * MLP_H + k0 + k] = g2[i][k];
#pragma unroll
    for (int k = 0; k < MLP_IN; ++k) o[OFF_W1 + lane * MLP_IN + k] = g1[k];
#pragma unroll
    for (int c = 0; c < MLP_OUT; ++c) o[OFF_W3 + c * MLP_H + lane] = g3[c];
    o[OFF_B1 + lane] = gb1;
    o[OFF_B2 + lane] = gb2;
    if (lane < MLP_OUT) o[OFF_B3 + lane] = gb3;
    if (lane == 0) o[NPARAM] = lsum;
    __syncthreads();
    for (int q = threadIdx.x; q < NPART; q += TR_T) {
        float a = sm.part[0][q];
#pragma unroll
        for (int i = 1; i < TR_W; ++i) a += sm.part[i][q];
        part[(int64_t)blockIdx.x * NPART + q] = a;
    }
}

// Gradient = sum of the CTAs' partials (32 sums a parameter side by side,
// always in the same order), then the Adam update of the parameter.  Only
// load latency counts here: eight sums of 38 partials each took 9.9 us.
constexpr int AD_P = 32, AD_G = 32;
__global__ void __launch_bounds__(AD_P* AD_G)
    mlp_update_kernel(float* __restrict__ w, float* __restrict__ m1, float* __restrict__ m2, float* __restrict__ grad,
                      float* __restrict__ loss, const float* __restrict__ part, int nparts, float inv_rows, float lr,
                      float b1, float b2, float eps, float c1, float c2) {
    __shared__ float s[AD_G][AD_P];
    const int pl = threadIdx.x % AD_P, gl = threadIdx.x / AD_P;
    const int q = blockIdx.x * AD_P + pl;
    float a = 0.0f;
    if (q < NPART) {
#pragma unroll 10
        for (int i = gl; i < nparts; i += AD_G) a += part[(int64_t)i * NPART + q];
    }
    s[gl][pl] = a;
    __syncthreads();
    if (gl != 0 || q >= NPART) return;
    float g = s[0][pl];
#pragma unroll
    for (int i = 1; i < AD_G; ++i) g += s[i][pl];
    if (q == NPARAM) {
        *loss = g * inv_rows;
        return;
    }
    grad[q] = g;
    const float a1 = b1 * m1[q] + (1.0f - b1) * g;
    const float a2 = b2 * m2[q] + (1.0f - b2) * g * g;
    m1[q] = a1;
    m2[q] = a2;
    w[q] -= lr * (a1 / c1) / (sqrtf(a2 / c2) + eps);
}

}  // namespace
}  // namespace bfsgb

using namespace bfsgb;

extern "C" bfs_status bfs_policy_load(const float* weights, int32_t nw, bfs_policy** out) {
    if (!out) return fail(BFS_EINVAL, "out is NULL");
    *out = nullptr;
    if (!weights) return fail(BFS_EINVAL, "weights is NULL");
    if (nw != NWEIGHTS && nw != NPARAM)
        return fail(BFS_EINVAL, "expected %d (or %d) floats, got %d", NWEIGHTS, NPARAM, nw);
    bfs_policy* p = new (std::nothrow) bfs_policy();
    if (!p) return fail(BFS_ENOMEM, "host allocation");
    p->host.assign(NWEIGHTS, 0.0f);
    for (int i = 0; i < nw; ++i) p->host[i] = weights[i];
    if (nw == NPARAM)
        for (int k = 0; k < MLP_IN; ++k) p->host[OFF_ISTD + k] = 1.0f;
    bool ok = cudaMalloc(&p->w, NWEIGHTS * 4) == cudaSuccess && cudaMalloc(&p->m1, NPARAM * 4) == cudaSuccess &&
              cudaMalloc(&p->m2, NPARAM * 4) == cudaSuccess && cudaMalloc(&p->grad, NPARAM * 4) == cudaSuccess &&
              cudaMalloc(&p->loss, 4) == cudaSuccess;
    if (ok) ok = cudaMemcpy(p->w, p->host.data(), NWEIGHTS * 4, cudaMemcpyHostToDevice) == cudaSuccess &&
                 cudaMemset(p->m1, 0, NPARAM * 4) == cudaSuccess && cudaMemset(p->m2, 0, NPARAM * 4) == cudaSuccess &&
                 cudaStreamSynchronize(nullptr) == cudaSuccess;  // zero for a step on any stream
    if (!ok) {
        cudaGetLastError();
        bfs_policy_free(p);
        return fail(BFS_ENOMEM, "policy device memory");
    }
    *out = p;
    return BFS_OK;
}

extern "C" bfs_status bfs_policy_weights(const bfs_policy* p, float* out, int32_t nw) {
    if (!p || !out) return fail(BFS_EINVAL, "null argument");
    if (nw < NWEIGHTS) return fail(BFS_EINVAL, "need %d floats", NWEIGHTS);
    BFS_CUDA(cudaMemcpy(out, p->w, NWEIGHTS * 4, cudaMemcpyDeviceToHost));
    return BFS_OK;
}

extern "C" bfs_status bfs_policy_set_norm(bfs_policy* p, const float* mean_inv_std) {
    if (!p || !mean_inv_std) return fail(BFS_EINVAL, "null argument");
    BFS_CUDA(cudaMemcpy(p->w + OFF_MEAN, mean_inv_std, 2 * MLP_IN * 4, cudaMemcpyHostToDevice));
    return BFS_OK;
}

extern "C" void bfs_policy_free(bfs_policy* p) {
    if (!p) return;
    cudaFree(p->w);
    cudaFree(p->m1);
    cudaFree(p->m2);
    cudaFree(p->grad);
    cudaFree(p->loss);
    cudaFree(p->part);
    delete p;
}

extern "C" bfs_status bfs_policy_forward(const bfs_policy* p, const float* X, int64_t rows, float* logits, void* cuda_stream) {
    if (!p || (rows > 0 && (!X || !logits))) return fail(BFS_EINVAL, "null argument");
    if (rows < 0) return fail(BFS_EINVAL, "rows < 0");
    if (rows == 0) return BFS_OK;
    if (!is_device_ptr(X) || !is_device_ptr(logits)) return fail(BFS_EINVAL, "X and logits must be device memory");
    int blocks = (int)std::min<int64_t>(div_up(rows, 128), (int64_t)num_sms() * 8);
    mlp_forward_kernel<<<blocks, 128, 0, (cudaStream_t)cuda_stream>>>(p->w, X, rows, logits);
    BFS_CUDA(cudaGetLastError());
    return BFS_OK;
}

namespace {

// One training step on either objective: gradient into p->grad (optionally
// copied out), Adam update of the parameters, mean loss optionally read back.
bfs_status train_step(bfs_policy* p, const float* X, const int32_t* y, const float* t, int64_t rows, float lr,
                      int32_t step, float* loss_out, float* grad_out, cudaStream_t st) {
    if (rows <= 0 || step < 1) return fail(BFS_EINVAL, "rows must be > 0 and step >= 1");
    if (rows > (int64_t)512 * 65535) return fail(BFS_ERANGE, "at most %lld rows per step", (long long)512 * 65535);
    const int most = num_sms() * TR_PER_SM;
    if (p->part_ctas < most) {
        BFS_CUDA(cudaStreamSynchronize(st));
        cudaFree(p->part);
        p->part = nullptr;
        p->part_ctas = 0;
        if (cudaMalloc(&p->part, (size_t)most * NPART * sizeof(float)) != cudaSuccess) {
            cudaGetLastError();
            return fail(BFS_ENOMEM, "training scratch for %lld rows", (long long)rows);
        }
        p->part_ctas = most;
    }
    const int blocks = (int)std::min<int64_t>(div_up(rows, TR_T), most);
    auto kernel = t ? mlp_train_kernel<true> : mlp_train_kernel<false>;
    BFS_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(MlpTrainSmem)));
    kernel<<<blocks, TR_T, sizeof(MlpTrainSmem), st>>>(p->w, X, y, t, rows, p->part);
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    float c1 = (float)(1.0 - std::pow(0.9, (double)step)), c2 = (float)(1.0 - std::pow(0.999, (double)step));
    mlp_update_kernel<<<(NPART + AD_P - 1) / AD_P, AD_P * AD_G, 0, st>>>(p->w, p->m1, p->m2, p->grad, p->loss, p->part,
                                                                        blocks, 1.0f / (float)rows, lr, b1, b2, eps, c1,
                                                                        c2);
    if (grad_out) BFS_CUDA(cudaMemcpyAsync(grad_out, p->grad, NPARAM * 4, cudaMemcpyDeviceToDevice, st));
    BFS_CUDA(cudaGetLastError());
    if (loss_out) {
        BFS_CUDA(cudaMemcpyAsync(loss_out, p->loss, 4, cudaMemcpyDeviceToHost, st));
        BFS_CUDA(cudaStreamSynchronize(st));
    }
    return BFS_OK;
}

}  // namespace

extern "C" bfs_status bfs_policy_train_step(bfs_policy* p, const float* X, const int32_t* y, int64_t rows, float lr,
                                            int32_t step, float* loss_out, float* grad_out, void* cuda_stream) {
    if (!p || !X || !y) return fail(BFS_EINVAL, "null argument");
    if (!is_device_ptr(X) || !is_device_ptr(y)) return fail(BFS_EINVAL, "X and y must be device memory");
    return train_step(p, X, y, nullptr, rows, lr, step, loss_out, grad_out, (cudaStream_t)cuda_stream);
}

extern "C" bfs_status bfs_policy_train_step_regress(bfs_policy* p, const float* X, const float* target, int64_t rows,
                                                    float lr, int32_t step, float* loss_out, float* grad_out,
                                                    void* cuda_stream) {
    if (!p || !X || !target) return fail(BFS_EINVAL, "null argument");
    if (!is_device_ptr(X) || !is_device_ptr(target)) return fail(BFS_EINVAL, "X and target must be device memory");
    return train_step(p, X, nullptr, target, rows, lr, step, loss_out, grad_out, (cudaStream_t)cuda_stream);
}

extern "C" bfs_status bfs_policy_features(const bfs_graph* g, int32_t level, int64_t f, int64_t e_f, int64_t m_u,
                                          int64_t f_prev, int32_t prev_dir, float* out10) {
    if (!g || !out10) return fail(BFS_EINVAL, "null argument");
    float x[MLP_IN];
    policy_features(x, f, e_f, m_u, f_prev, level, prev_dir, g->n, g->m, g->deg_max);
    if (is_device_ptr(out10)) {
        BFS_CUDA(cudaMemcpy(out10, x, sizeof(x), cudaMemcpyHostToDevice));
    } else {
        for (int k = 0; k < MLP_IN; ++k) out10[k] = x[k];
    }
    return BFS_OK;
}
