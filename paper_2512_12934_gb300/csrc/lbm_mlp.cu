// Surrogate MLP ensemble (4 -> 128 -> 128 -> 128 -> 2, GELU), FP32, with
// fused forward, backward and Adam kernels, and an inference kernel that
// runs the two hidden layers on the tcgen05 tensor cores (FP32-accurate
// split products; the default inference path).
//
// Training runs whole epochs inside thread-block clusters, one or more per
// member (mlp_train_kernel): the chain rule and Adam stay on chip and in L2,
// every sum has a fixed order (deterministic).
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "lbm.h"
#include "lbm_internal.h"

namespace {

constexpr int I = 4, H = 128, O = 2;
constexpr int oW1 = 0, ob1 = oW1 + H * I, oW2 = ob1 + H, ob2 = oW2 + H * H, oW3 = ob2 + H, ob3 = oW3 + H * H;
constexpr int oW4 = ob3 + H, ob4 = oW4 + O * H, P = ob4 + O;
// Device stride of one member's parameters: P rounded up to 32 floats so that
// every member (and every weight matrix in it) starts 128-byte aligned.
constexpr int PS = (P + 31) & ~31;

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
// GELU and its derivative of one pre-activation.
__device__ __forceinline__ void gelu_both(float z, float& a, float& d) {
    const float t = 1.0f + erff(z * 0.70710678118654752f);
    a = 0.5f * z * t;
    d = 0.5f * t + z * 0.3989422804014327f * expf(-0.5f * z * z);
}

// One Adam update (c1, c2: 1 - beta^t).
__device__ __forceinline__ void adam_update(float& w, float& m, float& v, float g, float lr, float b1, float b2,
                                            float c1, float c2, float eps) {
    m = b1 * m + (1.0f - b1) * g;
    v = b2 * v + (1.0f - b2) * g * g;
    w -= lr * (m / c1) / (sqrtf(v / c2) + eps);
}

// ---- training: forward, backward and Adam inside thread-block clusters ----
// One cluster of CL CTAs trains one member; a launch runs many steps.  Every
// CTA holds the member's whole parameter set in shared memory (136 KB) and
// takes its share of each minibatch through forward and backward in chunks of
// TS samples; the two 128x128 weight gradients accumulate in registers (64 per
// thread).  At the end of a step each CTA writes its partial gradient (L2
// resident), CTA r sums slice r of all partials in rank order (deterministic),
// applies Adam to it, and every CTA reloads the parameters: two cluster
// barriers a step, no launches.
// What bounds it: a minibatch of 64 is 4 samples per CTA, so a step is a chain
// of eleven short phases (6 us) and the exchange of 140 KB per CTA (6 us); a
// full batch is bound by shared-memory reads of the weights (16 us per chunk
// of 16 samples).  Exchanging over distributed shared memory instead of L2
// took 11 us (8 CTAs) and 15 us (16 CTAs).  The form before this, one CTA per
// 32 samples and three launches per step, left all but 10 SMs idle at a
// minibatch of 64 and staged transposed weights with uncoalesced reads.
// Step of 5 members, that form / this one: minibatch 64 109 / 15 us, 256 111 /
// 28, 1024 161 / 68, 4096 449 / 206.
constexpr int TT = 512;                        // threads per CTA
constexpr int WS = H + 4;                      // padded weight row: 16-byte accesses of 8 rows or of one row
constexpr int iW2 = 0, iW3 = iW2 + H * WS;     // shared parameter image (floats)
constexpr int iW1 = iW3 + H * WS, ib1 = iW1 + H * I, ib2 = ib1 + H, ib3 = ib2 + H, iW4 = ib3 + H, ib4 = iW4 + O * H;
constexpr int IMG = (ib4 + O + 3) & ~3;
static_assert(oW1 % 4 == 0 && oW2 % 4 == 0 && oW3 % 4 == 0 && oW4 % 4 == 0 && ob4 % 4 == 0 && PS >= ob4 + 4,
              "a group of four image floats must be a group of four parameters");

// Parameter offset of image group q (four floats from 4 q), -1 for row padding.
__device__ __forceinline__ int img_param(int q) {
    const int i = 4 * q;
    if (i < iW1) {
        const int l = i >= iW3, t = i - l * iW3, r = t / WS, c = t % WS;
        return c < H ? (l ? oW3 : oW2) + r * H + c : -1;
    }
    if (i < ib2) return i - iW1 + oW1;  // W1, b1
    if (i < ib3) return i - ib2 + ob2;
    return i - ib3 + ob3;  // b3, W4, b4
}

// The parameter image from global memory (other SMs write it during a launch:
// read through L2).
__device__ __forceinline__ void load_image(float* img, const float* p) {
    // both weight matrices: rows of 32 groups, one row per warp and pass
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int r = 0; r < 2 * H; r += TT / 32) {
        const int row = r + w, l = row / H, j = row % H;
        *reinterpret_cast<float4*>(img + l * iW3 + j * WS + 4 * lane) =
            __ldcg(reinterpret_cast<const float4*>(p + (l ? oW3 : oW2) + j * H) + lane);
    }
    for (int q = iW1 / 4 + (int)threadIdx.x; q < IMG / 4; q += TT)
        reinterpret_cast<float4*>(img)[q] = __ldcg(reinterpret_cast<const float4*>(p + img_param(q)));
}

struct TrainArgs {
    float *params, *m, *v;    // [E][PS]
    const float *X, *T;       // data rows
    const int* idx;           // row order (NULL: rows 0, 1, ...)
    const float2* coef;       // per step: 1 - beta1^t, 1 - beta2^t
    float* part;              // [E][clusters][CL][IMG] partial gradients
    float* out;               // gradient sums [E][clusters][P] instead of Adam (NULL: Adam)
    int B, nsteps;            // minibatch rows, steps of this launch
    int n, spe;               // rows of one epoch in idx, steps per epoch
    float lr, b1, b2, eps;
};

// Samples of a chunk (TS = 4, 8 or 16): the chunk runs through the network
// together.  Wider chunks reuse each weight read more; 4 is what a CTA gets of
// a minibatch of 64.
template <int TS>
struct TrainSmem {
    static constexpr int ACT = TS * H;
    static constexpr int PART = 16 * 4 * H;  // partial sums of the split contractions
    static constexpr size_t BYTES = (size_t)(IMG + 6 * ACT + PART + 2 * TS * (I + O) + TS * O) * 4;
};

__device__ __forceinline__ float dot4(float4 a, float4 b, float c) {
    return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, c))));
}

// part[g][s][j] = sum over contraction group g of a[s][k] W[j][k]: a warp owns
// four samples and 8 SG of the 128 terms, a lane the outputs j = lane + 32 r.
template <int TS>
__device__ __forceinline__ void train_gemm_nt(const float* W, const float* a, float* part) {
    constexpr int SG = TS / 4;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, sg = w % SG, g = w / SG;
    float acc[4][4] = {};
#pragma unroll
    for (int k = g * 8 * SG; k < (g + 1) * 8 * SG; k += 4) {
        float4 av[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) av[s] = *reinterpret_cast<const float4*>(a + (4 * sg + s) * H + k);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const float4 wv = *reinterpret_cast<const float4*>(W + (lane + 32 * r) * WS + k);
#pragma unroll
            for (int s = 0; s < 4; ++s) acc[r][s] = dot4(av[s], wv, acc[r][s]);
        }
    }
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int r = 0; r < 4; ++r) part[(g * TS + 4 * sg + s) * H + lane + 32 * r] = acc[r][s];
}

// part[g][s][k] = sum over contraction group g of z[s][j] W[j][k]; a lane owns
// the outputs k = 4 lane .. 4 lane + 3.
template <int TS>
__device__ __forceinline__ void train_gemm_nn(const float* W, const float* z, float* part) {
    constexpr int SG = TS / 4;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, sg = w % SG, g = w / SG;
    float4 acc[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) acc[s] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int j = g * 8 * SG; j < (g + 1) * 8 * SG; j += 4) {
        float4 zv[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) zv[s] = *reinterpret_cast<const float4*>(z + (4 * sg + s) * H + j);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 wv = *reinterpret_cast<const float4*>(W + (j + q) * WS + 4 * lane);
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const float t = q == 0 ? zv[s].x : (q == 1 ? zv[s].y : (q == 2 ? zv[s].z : zv[s].w));
                acc[s].x = fmaf(t, wv.x, acc[s].x);
                acc[s].y = fmaf(t, wv.y, acc[s].y);
                acc[s].z = fmaf(t, wv.z, acc[s].z);
                acc[s].w = fmaf(t, wv.w, acc[s].w);
            }
        }
    }
#pragma unroll
    for (int s = 0; s < 4; ++s) *reinterpret_cast<float4*>(part + (g * TS + 4 * sg + s) * H + 4 * lane) = acc[s];
}

// Sum of the contraction groups of output o = s * H + j, in group order.
template <int TS>
__device__ __forceinline__ float train_fold(const float* part, int o) {
    float z = part[o];
#pragma unroll
    for (int g = 1; g < 64 / TS; ++g) z += part[g * TS * H + o];
    return z;
}

// dw[a][c] += sum_s z[s][8 warp + a] x[s][4 lane + c]
template <int TS>
__device__ __forceinline__ void train_outer(const float* z, const float* x, float (&dw)[8][4]) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll 2
    for (int s = 0; s < TS; ++s) {
        const float4 z0 = *reinterpret_cast<const float4*>(z + s * H + 8 * w);
        const float4 z1 = *reinterpret_cast<const float4*>(z + s * H + 8 * w + 4);
        const float4 xv = *reinterpret_cast<const float4*>(x + s * H + 4 * lane);
        const float zz[8] = {z0.x, z0.y, z0.z, z0.w, z1.x, z1.y, z1.z, z1.w};
#pragma unroll
        for (int a = 0; a < 8; ++a) {
            dw[a][0] = fmaf(zz[a], xv.x, dw[a][0]);
            dw[a][1] = fmaf(zz[a], xv.y, dw[a][1]);
            dw[a][2] = fmaf(zz[a], xv.z, dw[a][2]);
            dw[a][3] = fmaf(zz[a], xv.w, dw[a][3]);
        }
    }
}

template <int TS>
__device__ __forceinline__ float train_column_sum(const float* z, int j) {
    float t = 0.f;
#pragma unroll
    for (int s = 0; s < TS; ++s) t += z[s * H + j];
    return t;
}

template <int TS, int CL>
__global__ void __launch_bounds__(TT, 1) mlp_train_kernel(const TrainArgs a) {
    extern __shared__ __align__(16) float smem[];
    using SM = TrainSmem<TS>;
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    float* img = smem;
    float *A1 = img + IMG, *A2 = A1 + SM::ACT, *A3 = A2 + SM::ACT;     // activations
    float *D1 = A3 + SM::ACT, *D2 = D1 + SM::ACT, *D3 = D2 + SM::ACT;  // GELU', then dZ
    float* part = D3 + SM::ACT;
    float* xs = part + SM::PART;      // [2][TS][I]
    float* ts = xs + 2 * TS * I;      // [2][TS][O]
    float* dY = ts + 2 * TS * O;      // [TS][O]
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int e = blockIdx.z, rank = (int)cluster.block_rank();
    const float* p = a.params + (size_t)e * PS;
    load_image(img, p);
    // rows of this cluster and of this CTA in every minibatch
    const int c0 = (int)((long long)a.B * blockIdx.y / gridDim.y);
    const int c1 = (int)((long long)a.B * (blockIdx.y + 1) / gridDim.y);
    const int r0 = c0 + (int)((long long)(c1 - c0) * rank / CL), r1 = c0 + (int)((long long)(c1 - c0) * (rank + 1) / CL);
    const int nch = (r1 - r0 + TS - 1) / TS;
    const float scale = 2.0f / ((float)a.B * (float)O);
    // Rows travel two chunks ahead of their use: threads [0, TS) look up the data
    // row of the chunk after next and load the inputs of the next one, so
    // neither of the two dependent reads is waited for.  Chunk position (ps,
    // pc); a negative row stands for a sample past the end (zeros).
    int ps = 0, pc = 0;
    auto lookup = [&]() -> int {
        int row = r0 + pc * TS + tid;
        if (ps >= a.nsteps || row >= r1) row = -1;
        else if (a.idx) row = a.idx[(long long)(ps / a.spe) * a.n + (long long)(ps % a.spe) * a.B + row];
        if (++pc >= nch) {
            pc = 0;
            ++ps;
        }
        return row;
    };
    auto fetch = [&](int row, float4& x, float2& t) {
        x = make_float4(0.f, 0.f, 0.f, 0.f);
        t = make_float2(0.f, 0.f);
        if (row >= 0) {
            x = *reinterpret_cast<const float4*>(a.X + (size_t)row * I);
            t = *reinterpret_cast<const float2*>(a.T + (size_t)row * O);
        }
    };
    auto put = [&](int buf, const float4& x, const float2& t) {
        *reinterpret_cast<float4*>(xs + (buf * TS + tid) * I) = x;
        *reinterpret_cast<float2*>(ts + (buf * TS + tid) * O) = t;
    };
    int buf = 0, row_next = -1;
    if (tid < TS) {
        float4 x;
        float2 t;
        fetch(lookup(), x, t);
        put(0, x, t);
        row_next = lookup();
    }
    __syncthreads();
#pragma unroll 1
    for (int step = 0; step < a.nsteps; ++step) {
        float dw2[8][4] = {}, dw3[8][4] = {};
        float dw1 = 0.f, dw4 = 0.f, db1v = 0.f, db2v = 0.f, db3v = 0.f, db4v = 0.f;
#pragma unroll 1
        for (int ch = 0; ch < nch; ++ch) {
            const float* x = xs + buf * TS * I;
            float4 nx_;
            float2 nt;
            if (tid < TS) {
                fetch(row_next, nx_, nt);
                row_next = lookup();
            }
            const int live = r1 - (r0 + ch * TS);  // samples of this chunk that exist
#pragma unroll
            for (int o = tid; o < TS * H; o += TT) {
                const int s = o / H, j = o % H;
                const float z = dot4(*reinterpret_cast<const float4*>(x + s * I),
                                     *reinterpret_cast<const float4*>(img + iW1 + j * I), img[ib1 + j]);
                gelu_both(z, A1[o], D1[o]);
            }
            __syncthreads();
            train_gemm_nt<TS>(img + iW2, A1, part);
            __syncthreads();
#pragma unroll
            for (int o = tid; o < TS * H; o += TT) gelu_both(train_fold<TS>(part, o) + img[ib2 + o % H], A2[o], D2[o]);
            __syncthreads();
            train_gemm_nt<TS>(img + iW3, A2, part);
            __syncthreads();
#pragma unroll
            for (int o = tid; o < TS * H; o += TT) gelu_both(train_fold<TS>(part, o) + img[ib3 + o % H], A3[o], D3[o]);
            __syncthreads();
            // output layer and dZ3: one warp per sample
            if (w < TS) {
                const float4 av = *reinterpret_cast<const float4*>(A3 + w * H + 4 * lane);
                const float4 u0 = *reinterpret_cast<const float4*>(img + iW4 + 4 * lane);
                const float4 u1 = *reinterpret_cast<const float4*>(img + iW4 + H + 4 * lane);
                float y0 = dot4(av, u0, 0.f), y1 = dot4(av, u1, 0.f);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    y0 += __shfl_xor_sync(0xffffffffu, y0, o);
                    y1 += __shfl_xor_sync(0xffffffffu, y1, o);
                }
                const float* t = ts + (buf * TS + w) * O;
                const bool in = w < live;
                const float d0 = in ? scale * (y0 + img[ib4] - t[0]) : 0.f;
                const float d1 = in ? scale * (y1 + img[ib4 + 1] - t[1]) : 0.f;
                if (lane == 0) {
                    dY[w * O] = d0;
                    dY[w * O + 1] = d1;
                }
                float4* dz = reinterpret_cast<float4*>(D3 + w * H + 4 * lane);
                const float4 gv = *dz;
                *dz = in ? make_float4((d0 * u0.x + d1 * u1.x) * gv.x, (d0 * u0.y + d1 * u1.y) * gv.y,
                                       (d0 * u0.z + d1 * u1.z) * gv.z, (d0 * u0.w + d1 * u1.w) * gv.w)
                         : make_float4(0.f, 0.f, 0.f, 0.f);
            }
            __syncthreads();
            train_gemm_nn<TS>(img + iW3, D3, part);
            train_outer<TS>(D3, A2, dw3);
            if (tid < O * H) {
#pragma unroll
                for (int s = 0; s < TS; ++s) dw4 = fmaf(dY[s * O + tid / H], A3[s * H + tid % H], dw4);
            } else if (tid < O * H + H) {
                db3v += train_column_sum<TS>(D3, tid - O * H);
            } else if (tid < O * H + H + O) {
#pragma unroll
                for (int s = 0; s < TS; ++s) db4v += dY[s * O + tid - O * H - H];
            }
            __syncthreads();
#pragma unroll
            for (int o = tid; o < TS * H; o += TT) D2[o] = o / H < live ? train_fold<TS>(part, o) * D2[o] : 0.f;
            __syncthreads();
            train_gemm_nn<TS>(img + iW2, D2, part);
            train_outer<TS>(D2, A1, dw2);
            if (tid < H) db2v += train_column_sum<TS>(D2, tid);
            __syncthreads();
#pragma unroll
            for (int o = tid; o < TS * H; o += TT) D1[o] = o / H < live ? train_fold<TS>(part, o) * D1[o] : 0.f;
            __syncthreads();
            {
                const int j = tid / I, i = tid % I;
#pragma unroll
                for (int s = 0; s < TS; ++s) dw1 = fmaf(D1[s * H + j], x[s * I + i], dw1);
            }
            if (tid < H) db1v += train_column_sum<TS>(D1, tid);
            buf ^= 1;
            if (tid < TS) put(buf, nx_, nt);
            __syncthreads();
        }
        // this CTA's partial gradient, in the order of the parameter image
        float* gp = a.part + (size_t)((e * gridDim.y + blockIdx.y) * CL + rank) * IMG;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            __stcg(reinterpret_cast<float4*>(gp + iW2 + (8 * w + r) * WS + 4 * lane),
                   make_float4(dw2[r][0], dw2[r][1], dw2[r][2], dw2[r][3]));
            __stcg(reinterpret_cast<float4*>(gp + iW3 + (8 * w + r) * WS + 4 * lane),
                   make_float4(dw3[r][0], dw3[r][1], dw3[r][2], dw3[r][3]));
        }
        gp[iW1 + tid] = dw1;
        if (tid < O * H) gp[iW4 + tid] = dw4;
        else if (tid < O * H + H) gp[ib3 + tid - O * H] = db3v;
        else if (tid < O * H + H + O) gp[ib4 + tid - O * H - H] = db4v;
        if (tid < H) {
            gp[ib1 + tid] = db1v;
            gp[ib2 + tid] = db2v;
        }
        cluster.sync();
        // slice of this rank: partials summed in rank order, Adam
        constexpr int PER = (IMG / 4 + CL - 1) / CL;
        const float* g0 = a.part + (size_t)((e * gridDim.y + blockIdx.y) * CL) * IMG;
        const float2 cf = a.out ? make_float2(1.f, 1.f) : a.coef[step];
#pragma unroll 1
        for (int i = tid; i < PER; i += TT) {
            const int q = rank * PER + i, o = q < IMG / 4 ? img_param(q) : -1;
            if (o < 0) continue;
            const size_t n = (size_t)e * PS + o;
            float4 t[CL], wv, mv, vv;
#pragma unroll
            for (int c = 0; c < CL; ++c) t[c] = __ldcg(reinterpret_cast<const float4*>(g0 + (size_t)c * IMG) + q);
            if (!a.out) {
                wv = *reinterpret_cast<const float4*>(a.params + n);
                mv = *reinterpret_cast<const float4*>(a.m + n);
                vv = *reinterpret_cast<const float4*>(a.v + n);
            }
            float4 g = t[0];
#pragma unroll
            for (int c = 1; c < CL; ++c) {
                g.x += t[c].x;
                g.y += t[c].y;
                g.z += t[c].z;
                g.w += t[c].w;
            }
            if (a.out) {
                float* go = a.out + ((size_t)e * gridDim.y + blockIdx.y) * P + o;
                const float gv[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (o + k < P) go[k] = gv[k];
                continue;
            }
            adam_update(wv.x, mv.x, vv.x, g.x, a.lr, a.b1, a.b2, cf.x, cf.y, a.eps);
            adam_update(wv.y, mv.y, vv.y, g.y, a.lr, a.b1, a.b2, cf.x, cf.y, a.eps);
            adam_update(wv.z, mv.z, vv.z, g.z, a.lr, a.b1, a.b2, cf.x, cf.y, a.eps);
            adam_update(wv.w, mv.w, vv.w, g.w, a.lr, a.b1, a.b2, cf.x, cf.y, a.eps);
            __stcg(reinterpret_cast<float4*>(a.params + n), wv);
            *reinterpret_cast<float4*>(a.m + n) = mv;
            *reinterpret_cast<float4*>(a.v + n) = vv;
        }
        if (step + 1 == a.nsteps) break;
        cluster.sync();
        load_image(img, p);
        __syncthreads();
    }
}

// Sum of the clusters' gradient partials gp [E][np][P] in cluster order ->
// gradient (grad_out) or an Adam update.
__global__ void __launch_bounds__(256) mlp_adam_kernel(float* __restrict__ params, float* __restrict__ m,
                                                       float* __restrict__ v, const float* __restrict__ gp, int np,
                                                       float lr, float b1, float b2, float c1, float c2, float eps,
                                                       float* __restrict__ grad_out) {
    const int e = blockIdx.y;
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= P) return;
    float g = 0.0f;
    for (int t = 0; t < np; ++t) g += gp[((size_t)e * np + t) * P + q];
    if (grad_out) {
        grad_out[(size_t)e * P + q] = g;
        return;
    }
    const size_t n = (size_t)e * PS + q;
    adam_update(params[n], m[n], v[n], g, lr, b1, b2, c1, c2, eps);
}

// ---- inference kernel: 128 samples per CTA, 8x8 register tiles -----------
// Activations live feature-major in shared memory (act[k][s]); the hidden
// weights are staged from a k-major copy (Wt[k][j]) with 16-byte loads, so a
// thread's inner step reads two float4 of weights and two float4 of inputs
// for 64 FMAs.
constexpr int TB = 128;   // samples per CTA
constexpr int NTB = 256;  // threads: 16 neuron groups x 16 sample groups of 8
constexpr size_t SMEM_BIG = (size_t)(H * H + 2 * H * TB) * sizeof(float);

// Wt[e][l][k][j] = W_{l+2}[j][k] for the two hidden 128x128 layers.
__global__ void mlp_transpose_kernel(const float* __restrict__ params, float* __restrict__ wt) {
    const int e = blockIdx.y;
    const int q = blockIdx.x * blockDim.x + threadIdx.x;  // over 2 * H * H
    if (q >= 2 * H * H) return;
    const int l = q / (H * H), r = q % (H * H), k = r / H, j = r % H;
    wt[(size_t)e * 2 * H * H + q] = params[(size_t)e * PS + (l ? oW3 : oW2) + j * H + k];
}

__global__ void __launch_bounds__(NTB) mlp_infer_kernel(const float* __restrict__ params,
                                                         const float* __restrict__ wt, const float* __restrict__ X,
                                                         int B, float* __restrict__ Y) {
    extern __shared__ __align__(16) float smem[];
    float* Wt = smem;              // [H][H]
    float* actA = smem + H * H;    // [H][TB]
    float* actB = actA + H * TB;   // [H][TB]
    const int e = blockIdx.y, s0 = blockIdx.x * TB;
    const float* p = params + (size_t)e * PS;
    // layer 1 (K = 4): consecutive threads take consecutive samples
    for (int q = threadIdx.x; q < TB * H; q += NTB) {
        const int j = q / TB, sl = q % TB, b = s0 + sl;
        float z = __ldg(p + ob1 + j);
        if (b < B) {
#pragma unroll
            for (int k = 0; k < I; ++k) z = fmaf(__ldg(p + oW1 + j * I + k), __ldg(X + (size_t)b * I + k), z);
        }
        actA[j * TB + sl] = gelu(z);
    }
    const int ng = threadIdx.x % 16, sg = threadIdx.x / 16;
    float* in = actA;
    float* out = actB;
#pragma unroll 1
    for (int l = 0; l < 2; ++l) {
        __syncthreads();  // the previous layer's outputs and reads of Wt are complete
        const float4* src = reinterpret_cast<const float4*>(wt + ((size_t)e * 2 + l) * H * H);
        for (int q = threadIdx.x; q < H * H / 4; q += NTB) reinterpret_cast<float4*>(Wt)[q] = __ldg(src + q);
        __syncthreads();
        const float* bias = p + (l ? ob3 : ob2);
        // acc[r][c2] holds outputs (8 ng + 2 c2, 8 ng + 2 c2 + 1) of sample
        // 8 sg + r: one packed FP32x2 FMA updates both (each lane rounds as
        // fmaf does)
        float2 acc[8][4];
#pragma unroll
        for (int c2 = 0; c2 < 4; ++c2) {
            const float2 bc = make_float2(__ldg(bias + 8 * ng + 2 * c2), __ldg(bias + 8 * ng + 2 * c2 + 1));
#pragma unroll
            for (int r = 0; r < 8; ++r) acc[r][c2] = bc;
        }
#pragma unroll 2
        for (int k = 0; k < H; ++k) {
            const float4 w0 = reinterpret_cast<const float4*>(Wt + k * H + 8 * ng)[0];
            const float4 w1 = reinterpret_cast<const float4*>(Wt + k * H + 8 * ng)[1];
            const float4 a0 = reinterpret_cast<const float4*>(in + k * TB + 8 * sg)[0];
            const float4 a1 = reinterpret_cast<const float4*>(in + k * TB + 8 * sg)[1];
            const float2 w[4] = {make_float2(w0.x, w0.y), make_float2(w0.z, w0.w), make_float2(w1.x, w1.y),
                                 make_float2(w1.z, w1.w)};
            const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const float2 ar = make_float2(a[r], a[r]);
#pragma unroll
                for (int c2 = 0; c2 < 4; ++c2) acc[r][c2] = __ffma2_rn(ar, w[c2], acc[r][c2]);
            }
        }
#pragma unroll
        for (int c2 = 0; c2 < 4; ++c2) {
            float4* o0 = reinterpret_cast<float4*>(out + (8 * ng + 2 * c2) * TB + 8 * sg);
            float4* o1 = reinterpret_cast<float4*>(out + (8 * ng + 2 * c2 + 1) * TB + 8 * sg);
            o0[0] = make_float4(gelu(acc[0][c2].x), gelu(acc[1][c2].x), gelu(acc[2][c2].x), gelu(acc[3][c2].x));
            o0[1] = make_float4(gelu(acc[4][c2].x), gelu(acc[5][c2].x), gelu(acc[6][c2].x), gelu(acc[7][c2].x));
            o1[0] = make_float4(gelu(acc[0][c2].y), gelu(acc[1][c2].y), gelu(acc[2][c2].y), gelu(acc[3][c2].y));
            o1[1] = make_float4(gelu(acc[4][c2].y), gelu(acc[5][c2].y), gelu(acc[6][c2].y), gelu(acc[7][c2].y));
        }
        float* t = in;
        in = out;
        out = t;
    }
    __syncthreads();
    // layer 4: one thread per (sample, output)
    {
        const int sl = threadIdx.x % TB, o = threadIdx.x / TB, b = s0 + sl;
        const float* w4 = p + oW4 + o * H;
        float y = __ldg(p + ob4 + o);
#pragma unroll 8
        for (int k = 0; k < H; ++k) y = fmaf(in[k * TB + sl], __ldg(w4 + k), y);
        if (b < B) Y[((size_t)e * B + b) * O + o] = y;
    }
}

// ---- inference on the tensor cores (tcgen05) ------------------------------
// The two hidden layers are D = A . W^T on 128-sample tiles (M = 128 samples,
// N = 128 neurons, K = 128), with A the previous layer's activations and W
// the layer's weight matrix [neuron][input].  FP32 accuracy from three
// products accumulated into one FP32 D in tensor memory:
//   A . W^T  ~  Ah . Wh^T + Al . Wh^T + Ab . Wl^T
// with Ah = tf32(A), Al = A - Ah, Wh = tf32(W) (the first two on kind::tf32,
// where Al is truncated to TF32 by the unit), Wl = bf16(W - Wh) and
// Ab = bf16(A) (kind::f16 with bf16 operands).  The dropped Al . Wl term and
// the roundings of the third product are below 2^-20 of |A||W|.
// Activations go to tensor memory (tcgen05.st, the MMA's A operand); the
// weights of both layers of the CTA's member sit in shared memory in the
// no-swizzle K-major layout (8-row x 16-byte core matrices, the next core
// matrix along K 128 bytes on, the next 8 rows (K * bytes / 16) * 128 bytes
// on), copied in by one bulk copy of the member's prepared image.  Layers 1
// (K = 4) and 4 (N = 2), the biases and GELU run on the FP32 pipes in the
// epilogues; thread (w, l) owns sample 32 (w % 4) + l (its TMEM lane) and
// neurons 32 c + 8 (w / 4) .. + 7 of each chunk c of 32.
constexpr int TCT = 512;
constexpr int TC_WH = H * H * 4, TC_WL = H * H * 2, TC_LAYER = TC_WH + TC_WL, TC_IMG = 2 * TC_LAYER;
constexpr size_t TC_SMEM = (size_t)TC_IMG + 128;
constexpr unsigned MLP_TC_TIMEOUT = 1u;

__host__ __device__ inline int tc_canon(int r, int k, int esize) {
    const int E = 16 / esize;
    return (r / 8) * ((H / E) * 128) + (k / E) * 128 + (r % 8) * 16 + (k % E) * esize;
}

__device__ __forceinline__ float tf32_rna(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return __uint_as_float(r);
}

// img[e][l] = { Wh (TF32 values in FP32 containers), Wl (bf16) } of hidden
// layer l + 2, both in the shared-memory layout above.
__global__ void mlp_tc_prep_kernel(const float* __restrict__ params, unsigned char* __restrict__ img) {
    const int e = blockIdx.y;
    const int q = blockIdx.x * blockDim.x + threadIdx.x;  // over 2 * H * H
    if (q >= 2 * H * H) return;
    const int l = q / (H * H), r = q % (H * H), j = r / H, k = r % H;
    const float w = params[(size_t)e * PS + (l ? oW3 : oW2) + j * H + k];
    const float wh = tf32_rna(w);
    unsigned char* base = img + (size_t)e * TC_IMG + (size_t)l * TC_LAYER;
    *reinterpret_cast<float*>(base + tc_canon(j, k, 4)) = wh;
    *reinterpret_cast<__nv_bfloat16*>(base + TC_WH + tc_canon(j, k, 2)) = __float2bfloat16_rn(w - wh);
}

__device__ __forceinline__ uint32_t tc_smem(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t tc_desc(uint32_t addr, uint32_t sbo) {
    // start >> 4, leading byte offset 128 >> 4, stride byte offset >> 4,
    // descriptor version 1 (bit 46), no swizzle
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(128u >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) |
           (1ull << 46);
}

// instruction descriptor of kind::tf32 (fmt 2) / kind::f16 with bf16 (fmt 1):
// FP32 D, K-major A and B, N = 128, M = 128
__host__ __device__ constexpr uint32_t tc_idesc(uint32_t fmt) {
    return (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(H >> 3) << 17) | ((uint32_t)(TB >> 4) << 24);
}

__device__ __forceinline__ void tc_mma(bool tf32, uint32_t d, uint32_t a, uint64_t b, uint32_t id, int acc) {
    if (tf32)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                     "tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n\t}"
                     :: "r"(d), "r"(a), "l"(b), "r"(id), "r"(acc) : "memory");
    else
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                     "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
                     :: "r"(d), "r"(a), "l"(b), "r"(id), "r"(acc) : "memory");
}

__device__ __forceinline__ void tc_st8(uint32_t t, const uint32_t (&v)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 :: "r"(t), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
}
__device__ __forceinline__ void tc_st4(uint32_t t, const uint32_t (&v)[4]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};"
                 :: "r"(t), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]) : "memory");
}
// Eight columns of this thread's lane (the caller waits for its loads).
__device__ __forceinline__ void tc_ld8(uint32_t t, float* v) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                 : "r"(t) : "memory");
}

// The loads above have landed; ties the values to the wait.
__device__ __forceinline__ void tc_ld_wait(float (&v)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7]),
                   "+f"(v[8]), "+f"(v[9]), "+f"(v[10]), "+f"(v[11])
                 :: "memory");
    asm volatile("" : "+f"(v[12]), "+f"(v[13]), "+f"(v[14]), "+f"(v[15]), "+f"(v[16]), "+f"(v[17]), "+f"(v[18]),
                      "+f"(v[19]), "+f"(v[20]), "+f"(v[21]));
    asm volatile("" : "+f"(v[22]), "+f"(v[23]), "+f"(v[24]), "+f"(v[25]), "+f"(v[26]), "+f"(v[27]), "+f"(v[28]),
                      "+f"(v[29]), "+f"(v[30]), "+f"(v[31]));
}

// Bounded wait on phase `parity` of an mbarrier; false (and the status bit)
// if it did not complete within `limit` SM clock cycles.
constexpr long long TC_WAIT_LIMIT = 2000000000LL;  // about a second at 2 GHz
__device__ __forceinline__ bool tc_wait(uint64_t* bar, uint32_t parity, unsigned* status, long long limit) {
    const long long t0 = clock64();
    for (;;) {
        // test_wait does not suspend: the limit counts from the first probe
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done) : "r"(tc_smem(bar)), "r"(parity) : "memory");
        if (done) return true;
        if (clock64() - t0 > limit) {
            atomicOr(status, MLP_TC_TIMEOUT);
            return false;
        }
        __nanosleep(20);
    }
}

__device__ __forceinline__ void tc_sync() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// GELU of two values in packed FP32x2 operations: z Phi(z) = (z + |z|)/2 - t h(t),
// t = |z|, h(t) = erfc(t/sqrt 2)/2 = exp(-t^2/2) P(1/(1 + 0.38 t)), the form of
// Hastings' approximations (Abramowitz and Stegun 7.1.25-28) with a degree-6 P
// fitted here by weighted minimax: the error of t h(t) is below 3.3e-9, so FP32
// rounding dominates (rms 4.2e-8 over |z| < 6, erff's form 5.3e-8).  Both
// branches of erff and its divergence go: 21 instructions per pair instead of
// about 46.  The clamp keeps t exp(..) finite; infinities and NaN pass through
// the first term, which is halved before it is added so that it stays finite for
// every finite z.
__device__ __forceinline__ float2 gelu2(float2 z) {
    const float2 t = make_float2(fminf(fabsf(z.x), 1e4f), fminf(fabsf(z.y), 1e4f));
    const float2 d = __ffma2_rn(t, make_float2(0.38f, 0.38f), make_float2(1.f, 1.f));
    const float2 x = __fmul2_rn(__fmul2_rn(t, make_float2(-0.72134752f, -0.72134752f)), t);  // -t^2/2 log2 e
    float2 u, e;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(u.x) : "f"(d.x));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(u.y) : "f"(d.y));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.x) : "f"(x.x));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.y) : "f"(x.y));
    constexpr float c[7] = {-0.0014650963712483644f, -0.13392633199691772f, -0.2417038530111313f,
                            0.1196700930595398f,     -0.4798668920993805f,  0.2958149015903473f,
                            -0.05852290615439415f};  // -P
    float2 q = make_float2(c[6], c[6]);
#pragma unroll
    for (int k = 5; k >= 0; --k) q = __ffma2_rn(q, u, make_float2(c[k], c[k]));
    const float2 s = __fmul2_rn(z, make_float2(0.5f, 0.5f));
    return __ffma2_rn(t, __fmul2_rn(e, q), make_float2(s.x + fabsf(s.x), s.y + fabsf(s.y)));
}

// The activations a[8] of neurons j0..j0+7 (j0 even) of this thread's sample as
// the next MMA's A operand: Ah, Al (one column each) and Ab (two per column,
// the even neuron in the low half).
__device__ __forceinline__ void tc_put_act(uint32_t tAh, uint32_t tAl, uint32_t tAb, int j0, const float (&a)[8]) {
    uint32_t h[8], lo[8], b2[4];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float ah = tf32_rna(a[i]);
        h[i] = __float_as_uint(ah);
        lo[i] = __float_as_uint(a[i] - ah);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __nv_bfloat162 pr = __floats2bfloat162_rn(a[2 * i], a[2 * i + 1]);  // .x = low half
        b2[i] = *reinterpret_cast<const uint32_t*>(&pr);
    }
    tc_st8(tAh + j0, h);
    tc_st8(tAl + j0, lo);
    tc_st4(tAb + j0 / 2, b2);
}

// The chunk's A columns are written: hand it to warp 0, whose first thread
// issues the chunk's 10 MMAs (K = 32: four TF32 steps of Ah and of Al, two BF16
// steps of Ab; a K step moves the descriptor's start address by 256 bytes, +16
// in its field).  The other warps go on to the next chunk at once.
__device__ __forceinline__ void tc_issue_chunk(int c, uint32_t tmem, uint32_t wh) {
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    if (threadIdx.x >= 32) {
        asm volatile("bar.arrive %0, %1;" ::"r"(c + 1), "n"(TCT) : "memory");
        return;
    }
    asm volatile("bar.sync %0, %1;" ::"r"(c + 1), "n"(TCT) : "memory");
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (threadIdx.x == 0) {
        const uint32_t it = tc_idesc(2), ib = tc_idesc(1);
        const uint32_t d = tmem, ah = tmem + 128, al = tmem + 256, ab = tmem + 384;
        const uint64_t dh = tc_desc(wh, (H / 4) * 128), dl = tc_desc(wh + TC_WH, (H / 8) * 128);
#pragma unroll
        for (int q = 0; q < 4; ++q) tc_mma(true, d, ah + 8 * (4 * c + q), dh + 16 * (4 * c + q), it, c > 0 || q > 0);
#pragma unroll
        for (int q = 0; q < 4; ++q) tc_mma(true, d, al + 8 * (4 * c + q), dh + 16 * (4 * c + q), it, 1);
#pragma unroll
        for (int q = 0; q < 2; ++q) tc_mma(false, d, ab + 8 * (2 * c + q), dl + 16 * (2 * c + q), ib, 1);
    }
    __syncwarp();
}

// Persistent per member: CTA (x, e) loads member e's weights once and runs
// tiles x, x + gridDim.x, ... of that member.  The FP32 work between the layers
// (GELU, operand splitting) bounds it, so the MMAs run under it: a layer's input
// is produced in four chunks of 32 neurons (8 per warp quarter) and each chunk's
// MMAs are issued while the next chunk is computed: 140 us for 65,536 points x 5
// members (222 with erff and the whole layer written before one barrier, 40 MMAs
// and a wait, the tensor pipe idle 78 % of the time).
__global__ void __launch_bounds__(TCT, 1) mlp_infer_tc_kernel(const float* __restrict__ params,
                                                              const unsigned char* __restrict__ img,
                                                              const float* __restrict__ X, int B,
                                                              float* __restrict__ Y, unsigned* status,
                                                              long long limit) {
    extern __shared__ __align__(128) unsigned char tc_raw[];
    unsigned char* sw = tc_raw + ((128u - (tc_smem(tc_raw) & 127u)) & 127u);
    __shared__ uint32_t s_tmem;
    __shared__ __align__(8) uint64_t s_bar[2];  // [0] weights landed, [1] MMAs of a layer done
    __shared__ __align__(16) float s_w1[I][H], s_b[3][H], s_w4[O][H];
    __shared__ float s_b4[O];
    __shared__ float s_part[4][O][TB];
    __shared__ int s_ok;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = warp & 3, qc = warp >> 2;
    const int row = 32 * g + lane;
    const int e = blockIdx.y, ntiles = (B + TB - 1) / TB;
    const float* p = params + (size_t)e * PS;
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(tc_smem(&s_bar[0])) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(tc_smem(&s_bar[1])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_ok = 1;
    }
    __syncthreads();
    bool weights = false;  // thread 0: the weight image has landed
    int pending = -1;      // thread 0: layer whose MMAs are committed and not waited for
    if (tid == 0) {
        // the member's weight image: four bulk copies onto one transaction count
        const unsigned char* src = img + (size_t)e * TC_IMG;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(tc_smem(&s_bar[0])), "r"(TC_IMG) : "memory");
#pragma unroll
        for (int c = 0; c < 4; ++c)
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         :: "r"(tc_smem(sw + c * (TC_IMG / 4))), "l"(src + c * (TC_IMG / 4)), "r"(TC_IMG / 4),
                            "r"(tc_smem(&s_bar[0])) : "memory");
        // the other threads stage the small parameters meanwhile
        weights = tc_wait(&s_bar[0], 0, status, limit);
        if (!weights) s_ok = 0;
    }
    for (int i = tid; i < H * I; i += TCT) s_w1[i % I][i / I] = p[oW1 + i];
    for (int i = tid; i < H; i += TCT) {
        s_b[0][i] = p[ob1 + i];
        s_b[1][i] = p[ob2 + i];
        s_b[2][i] = p[ob3 + i];
    }
    for (int i = tid; i < O * H; i += TCT) s_w4[i / H][i % H] = p[oW4 + i];
    if (tid < O) s_b4[tid] = p[ob4 + tid];
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(tc_smem(&s_tmem)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_sync();
    const uint32_t tmem = s_tmem, lane_off = (uint32_t)(32 * g) << 16;
    const uint32_t tD = tmem + lane_off, tAh = tD + 128, tAl = tD + 256, tAb = tD + 384;
    bool ok = s_ok != 0;  // the same in every thread
    float x[I];
    auto load_x = [&](int t) {
        const int b = t * TB + row;
#pragma unroll
        for (int k = 0; k < I; ++k) x[k] = t < ntiles && b < B ? __ldg(X + (size_t)b * I + k) : 0.0f;
    };
    // every thread waits for the layer's MMAs; one decision for the whole CTA
    auto layer_done = [&](int l) {
        if (tid == 0) {
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                         :: "r"(tc_smem(&s_bar[1])) : "memory");
            pending = l;
        }
        // two commits per tile: phase parity = layer
        ok = __syncthreads_and(tc_wait(&s_bar[1], (uint32_t)l, status, limit)) != 0;
        if (ok) pending = -1;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    };
    if (ok) load_x(blockIdx.x);
#pragma unroll 1
    for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
        // ---- layer 1 (K = 4) on the FP32 pipes, GELU, A of layer 2 ----
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int j0 = 32 * c + 8 * qc;
            float a[8];
#pragma unroll
            for (int i = 0; i < 8; i += 4) {
                const float4 b4 = *reinterpret_cast<const float4*>(&s_b[0][j0 + i]);
                float2 z0 = make_float2(b4.x, b4.y), z1 = make_float2(b4.z, b4.w);
#pragma unroll
                for (int k = 0; k < I; ++k) {
                    const float4 w4 = *reinterpret_cast<const float4*>(&s_w1[k][j0 + i]);
                    z0 = __ffma2_rn(make_float2(w4.x, w4.y), make_float2(x[k], x[k]), z0);
                    z1 = __ffma2_rn(make_float2(w4.z, w4.w), make_float2(x[k], x[k]), z1);
                }
                z0 = gelu2(z0);
                z1 = gelu2(z1);
                a[i] = z0.x;
                a[i + 1] = z0.y;
                a[i + 2] = z1.x;
                a[i + 3] = z1.y;
            }
            tc_put_act(tAh, tAl, tAb, j0, a);
            tc_issue_chunk(c, tmem, tc_smem(sw));
        }
        load_x(t + gridDim.x);  // arrives while the hidden layers run
        layer_done(0);
        if (!ok) break;
        float v[32];
#pragma unroll
        for (int c = 0; c < 4; ++c) tc_ld8(tD + 32 * c + 8 * qc, v + 8 * c);
        tc_ld_wait(v);
        // ---- epilogue of layer 2: bias, GELU, A of layer 3.  The first chunk's
        // barrier also says that every warp has read its part of D, which that
        // chunk's MMAs overwrite ----
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int j0 = 32 * c + 8 * qc;
            float a[8];
#pragma unroll
            for (int i = 0; i < 8; i += 2) {
                const float2 b2 = *reinterpret_cast<const float2*>(&s_b[1][j0 + i]);
                const float2 z = gelu2(__fadd2_rn(make_float2(v[8 * c + i], v[8 * c + i + 1]), b2));
                a[i] = z.x;
                a[i + 1] = z.y;
            }
            tc_put_act(tAh, tAl, tAb, j0, a);
            tc_issue_chunk(c, tmem, tc_smem(sw + TC_LAYER));
        }
        layer_done(1);
        if (!ok) break;
#pragma unroll
        for (int c = 0; c < 4; ++c) tc_ld8(tD + 32 * c + 8 * qc, v + 8 * c);
        tc_ld_wait(v);
        // ---- epilogue of layer 3 and layer 4 (N = 2): partial sums over this thread's neurons ----
        float2 y0 = make_float2(0.f, 0.f), y1 = y0;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int j0 = 32 * c + 8 * qc;
#pragma unroll
            for (int i = 0; i < 8; i += 2) {
                const float2 b2 = *reinterpret_cast<const float2*>(&s_b[2][j0 + i]);
                const float2 z = gelu2(__fadd2_rn(make_float2(v[8 * c + i], v[8 * c + i + 1]), b2));
                y0 = __ffma2_rn(z, *reinterpret_cast<const float2*>(&s_w4[0][j0 + i]), y0);
                y1 = __ffma2_rn(z, *reinterpret_cast<const float2*>(&s_w4[1][j0 + i]), y1);
            }
        }
        s_part[qc][0][row] = y0.x + y0.y;
        s_part[qc][1][row] = y1.x + y1.y;
        tc_sync();
        if (tid < O * TB) {
            const int r = tid % TB, o = tid / TB, bb = t * TB + r;
            const float y = s_b4[o] + ((s_part[0][o][r] + s_part[1][o][r]) + (s_part[2][o][r] + s_part[3][o][r]));
            if (bb < B) Y[((size_t)e * B + bb) * O + o] = y;
        }
    }
    // a weight copy or MMAs still in flight (their wait ran out) complete
    // before the CTA frees its tensor memory and leaves
    tc_sync();
    if (tid == 0) {
        if (!weights) tc_wait(&s_bar[0], 0, status, TC_WAIT_LIMIT);
        if (pending >= 0) tc_wait(&s_bar[1], (uint32_t)pending, status, TC_WAIT_LIMIT);
    }
    tc_sync();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(512) : "memory");
}

// Ensemble mean and relative spread (max over outputs of the population std
// over members / |mean|), two passes over the members.
// mean, spread and status_out may be mapped host memory: the inference status
// word goes out with the results, so a call needs no copy after it.
__global__ void mlp_reduce_kernel(const float* __restrict__ Y, int E, int B, float* __restrict__ mean,
                                  float* __restrict__ spread, const unsigned* __restrict__ status,
                                  unsigned* __restrict__ status_out) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b == 0) *status_out = *status;
    if (b >= B) return;
    float sp = 0.0f;
#pragma unroll
    for (int o = 0; o < O; ++o) {
        float s = 0.0f;
        for (int e = 0; e < E; ++e) s += Y[((size_t)e * B + b) * O + o];
        const float mu = s / (float)E;
        float s2 = 0.0f;
        for (int e = 0; e < E; ++e) {
            const float d = Y[((size_t)e * B + b) * O + o] - mu;
            s2 = fmaf(d, d, s2);
        }
        mean[(size_t)b * O + o] = mu;
        sp = fmaxf(sp, sqrtf(s2 / (float)E) / fmaxf(fabsf(mu), 1e-30f));
    }
    spread[b] = sp;
}

// splitmix64: deterministic host generator for initial weights and shuffles.
uint64_t splitmix64(uint64_t& s) {
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
double uniform01(uint64_t& s) { return (double)(splitmix64(s) >> 11) * (1.0 / 9007199254740992.0); }

}  // namespace

struct lbm_mlp {
    int E = 0;
    cudaStream_t stream = nullptr;
    float* params = nullptr;  // [E][P]
    float* m = nullptr;
    float* v = nullptr;
    int64_t t = 0;            // Adam steps taken
    uint64_t seed = 0;
    float* wt = nullptr;      // [E][2][H][H] k-major copy of the hidden weights (inference)
    unsigned char* tcimg = nullptr;  // [E][TC_IMG] tensor-core images of the hidden weights
    unsigned* status = nullptr;      // device status word of the tensor-core inference
    int infer_path = LBM_MLP_INFER_TENSOR;
    int sms = 1;  // SMs of the device (persistent tensor-core grid)
    int clusters8 = 0, clusters16 = 0;  // training clusters of 8 / 16 CTAs that fit on the device at once
    long long wait_limit = TC_WAIT_LIMIT;  // SM cycles a tensor-core wait may take
    void* ws = nullptr;       // grow-only device workspace of the per-call buffers
    size_t ws_bytes = 0;
    unsigned* hstatus = nullptr;  // pinned: status word of the last prediction
    float* hio = nullptr;         // pinned: X, mean and spread of a small host prediction
    std::string err;
};

namespace {

// Host predictions of up to this many points run on mapped pinned memory: the
// kernels read X and write the results over the host link themselves, two
// launches and one synchronisation instead of those plus four copies (221
// points: 63 -> 31 us a call; beyond a few thousand points the copy engine moves the
// bytes faster than every member reading X over the link).  The pinned block costs
// 110 us at creation and 160 when it is freed in a process that holds no other
// pinned memory, 2 us otherwise.
constexpr int kMappedPoints = 4096;

lbm_status mfail(lbm_mlp* m, lbm_status st, const std::string& msg) {
    if (m) m->err = msg;
    else lbm::set_thread_error(msg.c_str());
    return st;
}

#define MCK(call)                                                                                          \
    do {                                                                                                   \
        cudaError_t e_ = (call);                                                                           \
        if (e_ != cudaSuccess) return mfail(mm, LBM_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

template <int TS, int CL>
cudaError_t train_attr() {
    cudaError_t e = cudaFuncSetAttribute(mlp_train_kernel<TS, CL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)TrainSmem<TS>::BYTES);
    if (e == cudaSuccess && CL > 8)
        e = cudaFuncSetAttribute(mlp_train_kernel<TS, CL>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

std::once_flag g_attr_once;
cudaError_t g_attr_err = cudaSuccess;

cudaError_t set_smem_attrs() {
    std::call_once(g_attr_once, [] {
        for (cudaError_t e : {train_attr<4, 8>(), train_attr<8, 8>(), train_attr<16, 8>(), train_attr<4, 16>(),
                              train_attr<8, 16>(), train_attr<16, 16>()})
            if (g_attr_err == cudaSuccess) g_attr_err = e;
        if (g_attr_err == cudaSuccess)
            g_attr_err = cudaFuncSetAttribute(mlp_infer_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)SMEM_BIG);
        if (g_attr_err == cudaSuccess)
            g_attr_err = cudaFuncSetAttribute(mlp_infer_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)TC_SMEM);
    });
    return g_attr_err;
}

// Per-call device buffers, carved out of the ensemble's workspace (grown, never
// shrunk; reallocated only after the stream has drained).
struct Scratch {
    float *X = nullptr, *T = nullptr, *Y = nullptr, *gp = nullptr, *grad = nullptr;
    float2* coef = nullptr;
    int* idx = nullptr;
};

// Element counts of X, T, Y, gp, grad (floats), coef (pairs) and idx (ints).
lbm_status carve(lbm_mlp* mm, Scratch& s, size_t nX, size_t nT, size_t nY, size_t ngp, size_t ngrad, size_t ncoef,
                 size_t nidx) {
    const size_t cnt[7] = {nX, nT, nY, ngp, ngrad, 2 * ncoef, nidx};
    size_t off[7], total = 0;
    for (int k = 0; k < 7; ++k) {
        off[k] = total;
        total += (cnt[k] * 4 + 255) / 256 * 256;
    }
    if (total > mm->ws_bytes) {
        MCK(cudaStreamSynchronize(mm->stream));
        if (mm->ws) cudaFree(mm->ws);
        mm->ws = nullptr;
        mm->ws_bytes = 0;
        const size_t want = total + total / 4;
        cudaError_t e = cudaMalloc(&mm->ws, want);
        if (e != cudaSuccess) {
            mm->ws = nullptr;
            return mfail(mm, e == cudaErrorMemoryAllocation ? LBM_ERR_OOM : LBM_ERR_CUDA,
                         std::string("mlp workspace: ") + cudaGetErrorString(e));
        }
        mm->ws_bytes = want;
    }
    char* b = static_cast<char*>(mm->ws);
    float** fp[5] = {&s.X, &s.T, &s.Y, &s.gp, &s.grad};
    for (int k = 0; k < 5; ++k) *fp[k] = cnt[k] ? reinterpret_cast<float*>(b + off[k]) : nullptr;
    s.coef = cnt[5] ? reinterpret_cast<float2*>(b + off[5]) : nullptr;
    s.idx = cnt[6] ? reinterpret_cast<int*>(b + off[6]) : nullptr;
    return LBM_OK;
}

#define CARVE(...)                                   \
    do {                                             \
        lbm_status cs_ = carve(mm, s, __VA_ARGS__);  \
        if (cs_ != LBM_OK) return cs_;               \
    } while (0)

// How a minibatch of B rows is trained: clusters of `cl` CTAs, `nc` of them per
// member, chunks of `ts` samples.
struct TrainPlan {
    int cl, nc, ts;
};

// The plan with the smallest estimated step: waves of clusters times (a fixed
// 11 us for the exchange and barriers, plus the chunks: 4 us for up to four
// rows per CTA, 7.5 us for up to eight, 16 us for each sixteen), plus 10 us for
// the second launch when several clusters share a member.  Measured on GB300
// for 1 to 8 members and minibatches of 16 to 4096: the choice is within a few
// percent of the best plan tried (e.g. 5 members: minibatch 64 16x1 15 us, 8x1
// 19 us; 4096 8x3 206 us, 16x1 277 us, 8x1 516 us; 8 members, minibatch 64: 8x1
// 19 us, 16x1, of which 7 clusters fit, 31 us).
TrainPlan train_plan(const lbm_mlp* mm, int B) {
    TrainPlan best{8, 1, 16};
    double best_us = 1e300;
    for (int cl : {8, 16}) {
        const int fit = cl == 16 ? mm->clusters16 : mm->clusters8;
        if (cl == 16 && fit < 1) continue;
        for (int nc = 1; nc == 1 || nc * mm->E <= fit; ++nc) {
            const int rows = (B + cl * nc - 1) / (cl * nc), waves = (mm->E * nc + std::max(1, fit) - 1) / std::max(1, fit);
            const double chunks = rows <= 4 ? 4.0 : (rows <= 8 ? 7.5 : 16.0 * ((rows + 15) / 16));
            const double us = waves * (11.0 + chunks) + (nc > 1 ? 10.0 : 0.0);
            if (us < best_us) {
                best_us = us;
                best = {cl, nc, rows <= 4 ? 4 : (rows <= 8 ? 8 : 16)};
            }
        }
    }
    return best;
}

template <int TS, int CL>
cudaError_t launch_train(const TrainArgs& a, int nc, int E, cudaStream_t st, int* max_clusters = nullptr) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)CL, (unsigned)nc, (unsigned)E);
    cfg.blockDim = dim3(TT);
    cfg.dynamicSmemBytes = TrainSmem<TS>::BYTES;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim = {(unsigned)CL, 1, 1};
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (max_clusters) return cudaOccupancyMaxActiveClusters(max_clusters, mlp_train_kernel<TS, CL>, &cfg);
    return cudaLaunchKernelEx(&cfg, mlp_train_kernel<TS, CL>, a);
}

template <int CL>
cudaError_t launch_train_cl(const TrainArgs& a, const TrainPlan& p, int E, cudaStream_t st) {
    return p.ts == 4   ? launch_train<4, CL>(a, p.nc, E, st)
           : p.ts == 8 ? launch_train<8, CL>(a, p.nc, E, st)
                       : launch_train<16, CL>(a, p.nc, E, st);
}

cudaError_t run_train(const TrainArgs& a, const TrainPlan& p, int E, cudaStream_t st) {
    return p.cl == 16 ? launch_train_cl<16>(a, p, E, st) : launch_train_cl<8>(a, p, E, st);
}

// Gradient exchange of a plan: the CTAs' partials, then (several clusters per
// member) the clusters' sums.
size_t part_floats(const lbm_mlp* mm, const TrainPlan& p) {
    return (size_t)mm->E * p.nc * p.cl * IMG + (p.nc > 1 ? (size_t)mm->E * p.nc * P : 0);
}
float* cluster_sums(const lbm_mlp* mm, const TrainPlan& p, float* gp) { return gp + (size_t)mm->E * p.nc * p.cl * IMG; }

constexpr float kBeta1 = 0.9f, kBeta2 = 0.999f, kEps = 1e-8f;

float2 adam_coef(int64_t t) {
    return make_float2((float)(1.0 - std::pow(0.9, (double)t)), (float)(1.0 - std::pow(0.999, (double)t)));
}

// Refresh the k-major copy of the hidden weights after any parameter change.
lbm_status refresh_wt(lbm_mlp* mm) {
    mlp_transpose_kernel<<<dim3((2 * H * H + 255) / 256, mm->E), 256, 0, mm->stream>>>(mm->params, mm->wt);
    MCK(cudaGetLastError());
    mlp_tc_prep_kernel<<<dim3((2 * H * H + 255) / 256, mm->E), 256, 0, mm->stream>>>(mm->params, mm->tcimg);
    MCK(cudaGetLastError());
    return LBM_OK;
}

lbm_status launch_infer(lbm_mlp* mm, const float* dX, int n, float* dY) {
    if (mm->infer_path == LBM_MLP_INFER_TENSOR) {
        // persistent per member: about one CTA per SM over all members
        const int ntiles = (n + TB - 1) / TB;
        const int per = std::max(1, std::min(ntiles, mm->sms / mm->E));
        mlp_infer_tc_kernel<<<dim3(per, mm->E), TCT, TC_SMEM, mm->stream>>>(mm->params, mm->tcimg, dX, n, dY,
                                                                             mm->status, mm->wait_limit);
    } else {
        mlp_infer_kernel<<<dim3((n + TB - 1) / TB, mm->E), NTB, SMEM_BIG, mm->stream>>>(mm->params, mm->wt, dX, n,
                                                                                          dY);
    }
    MCK(cudaGetLastError());
    return LBM_OK;
}

// After the stream has drained: a tensor-core wait that ran out is an error
// (the outputs of that call are undefined); the word is cleared for the next.
lbm_status infer_result(lbm_mlp* mm, unsigned st) {
    if (st) {
        MCK(cudaMemset(mm->status, 0, sizeof(unsigned)));
        return mfail(mm, LBM_ERR_TIMEOUT, "a tensor-core wait of the inference kernel ran out; outputs undefined");
    }
    return LBM_OK;
}

lbm_status check_infer(lbm_mlp* mm) {
    unsigned st = 0;
    MCK(cudaMemcpy(&st, mm->status, sizeof(unsigned), cudaMemcpyDeviceToHost));
    return infer_result(mm, st);
}

}  // namespace

extern "C" {

int64_t lbm_mlp_num_params(void) { return P; }

lbm_status lbm_mlp_create(int members, uint64_t seed, void* cuda_stream, lbm_mlp** out) {
    if (!out) return mfail(nullptr, LBM_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    if (members < 1 || members > 64) return mfail(nullptr, LBM_ERR_INVALID_ARG, "members must be in [1, 64]");
    lbm_mlp* mm = new (std::nothrow) lbm_mlp();
    if (!mm) return mfail(nullptr, LBM_ERR_OOM, "host allocation failed");
    mm->E = members;
    mm->stream = static_cast<cudaStream_t>(cuda_stream);
    mm->seed = seed;
    cudaError_t e = set_smem_attrs();
    int dev = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&mm->sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = launch_train<16, 8>(TrainArgs{}, 1, members, mm->stream, &mm->clusters8);
    if (e == cudaSuccess) {
        // 16 CTAs exceed the portable cluster size: a device may refuse them
        if (launch_train<16, 16>(TrainArgs{}, 1, members, mm->stream, &mm->clusters16) != cudaSuccess) {
            cudaGetLastError();
            mm->clusters16 = 0;
        }
    }
    const size_t bytes = (size_t)members * PS * sizeof(float);
    if (e == cudaSuccess) e = cudaMalloc((void**)&mm->params, bytes);
    if (e == cudaSuccess) e = cudaMalloc((void**)&mm->m, bytes);
    if (e == cudaSuccess) e = cudaMalloc((void**)&mm->v, bytes);
    if (e == cudaSuccess) e = cudaMemset(mm->m, 0, bytes);
    if (e == cudaSuccess) e = cudaMemset(mm->v, 0, bytes);
    if (e == cudaSuccess) e = cudaMalloc((void**)&mm->wt, (size_t)members * 2 * H * H * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc((void**)&mm->tcimg, (size_t)members * TC_IMG);
    if (e == cudaSuccess) e = cudaMalloc((void**)&mm->status, sizeof(unsigned));
    if (e == cudaSuccess) e = cudaMemset(mm->status, 0, sizeof(unsigned));
    if (e == cudaSuccess) e = cudaMallocHost((void**)&mm->hstatus, sizeof(unsigned));
    if (e == cudaSuccess) e = cudaMallocHost((void**)&mm->hio, (size_t)kMappedPoints * (I + O + 1) * sizeof(float));
    if (e != cudaSuccess) {
        const std::string msg = std::string("mlp allocation: ") + cudaGetErrorString(e);
        lbm_mlp_destroy(mm);
        return mfail(nullptr, e == cudaErrorMemoryAllocation ? LBM_ERR_OOM : LBM_ERR_CUDA, msg);
    }
    // uniform(-1/sqrt(fan_in), 1/sqrt(fan_in)) weights, zero biases; member e
    // draws from seed + e
    std::vector<float> h((size_t)members * P, 0.0f);
    for (int m = 0; m < members; ++m) {
        uint64_t st = seed + (uint64_t)m * 0x632BE59BD9B4E019ull;
        float* p = h.data() + (size_t)m * P;
        auto fill = [&](int off, int n, int fan_in) {
            const double bound = 1.0 / std::sqrt((double)fan_in);
            for (int i = 0; i < n; ++i) p[off + i] = (float)((2.0 * uniform01(st) - 1.0) * bound);
        };
        fill(oW1, H * I, I);
        fill(oW2, H * H, H);
        fill(oW3, H * H, H);
        fill(oW4, O * H, H);
    }
    e = cudaMemcpy2D(mm->params, PS * sizeof(float), h.data(), P * sizeof(float), P * sizeof(float), members,
                     cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        const std::string msg = std::string("mlp upload: ") + cudaGetErrorString(e);
        lbm_mlp_destroy(mm);
        return mfail(nullptr, LBM_ERR_CUDA, msg);
    }
    if (refresh_wt(mm) != LBM_OK) {
        const std::string msg = mm->err;
        lbm_mlp_destroy(mm);
        return mfail(nullptr, LBM_ERR_CUDA, msg);
    }
    *out = mm;
    return LBM_OK;
}

lbm_status lbm_mlp_set_params(lbm_mlp* mm, const float* params) {
    if (!mm || !params) return mfail(mm, LBM_ERR_INVALID_ARG, "NULL argument");
    MCK(cudaStreamSynchronize(mm->stream));
    MCK(cudaMemcpy2D(mm->params, PS * sizeof(float), params, P * sizeof(float), P * sizeof(float), mm->E,
                     cudaMemcpyHostToDevice));
    MCK(cudaMemset(mm->m, 0, (size_t)mm->E * PS * sizeof(float)));
    MCK(cudaMemset(mm->v, 0, (size_t)mm->E * PS * sizeof(float)));
    mm->t = 0;
    return refresh_wt(mm);
}

lbm_status lbm_mlp_get_params(lbm_mlp* mm, float* params) {
    if (!mm || !params) return mfail(mm, LBM_ERR_INVALID_ARG, "NULL argument");
    MCK(cudaStreamSynchronize(mm->stream));
    MCK(cudaMemcpy2D(params, P * sizeof(float), mm->params, PS * sizeof(float), P * sizeof(float), mm->E,
                     cudaMemcpyDeviceToHost));
    return LBM_OK;
}

lbm_status lbm_mlp_forward(lbm_mlp* mm, const float* X, int n, float* Y) {
    if (!mm || !X || !Y || n < 1) return mfail(mm, LBM_ERR_INVALID_ARG, "bad forward request");
    Scratch s;
    CARVE((size_t)n * I, 0, (size_t)mm->E * n * O, 0, 0, 0, 0);
    MCK(cudaMemcpyAsync(s.X, X, (size_t)n * I * sizeof(float), cudaMemcpyHostToDevice, mm->stream));
    lbm_status st = launch_infer(mm, s.X, n, s.Y);
    if (st != LBM_OK) return st;
    MCK(cudaMemcpyAsync(Y, s.Y, (size_t)mm->E * n * O * sizeof(float), cudaMemcpyDeviceToHost, mm->stream));
    MCK(cudaStreamSynchronize(mm->stream));
    return check_infer(mm);
}

lbm_status lbm_mlp_gradient(lbm_mlp* mm, const float* X, const float* T, int n, float* grad) {
    if (!mm || !X || !T || !grad || n < 1) return mfail(mm, LBM_ERR_INVALID_ARG, "bad gradient request");
    const TrainPlan p = train_plan(mm, n);
    Scratch s;
    CARVE((size_t)n * I, (size_t)n * O, 0, part_floats(mm, p), (size_t)mm->E * P, 0, 0);
    MCK(cudaMemcpyAsync(s.X, X, (size_t)n * I * sizeof(float), cudaMemcpyHostToDevice, mm->stream));
    MCK(cudaMemcpyAsync(s.T, T, (size_t)n * O * sizeof(float), cudaMemcpyHostToDevice, mm->stream));
    TrainArgs a{mm->params, mm->m, mm->v, s.X, s.T, nullptr, nullptr, s.gp, p.nc > 1 ? cluster_sums(mm, p, s.gp) : s.grad,
                n, 1, n, 1, 0.f, kBeta1, kBeta2, kEps};
    MCK(run_train(a, p, mm->E, mm->stream));
    if (p.nc > 1) {
        mlp_adam_kernel<<<dim3((P + 255) / 256, mm->E), 256, 0, mm->stream>>>(
            mm->params, mm->m, mm->v, a.out, p.nc, 0.f, kBeta1, kBeta2, 1.f, 1.f, kEps, s.grad);
        MCK(cudaGetLastError());
    }
    MCK(cudaMemcpyAsync(grad, s.grad, (size_t)mm->E * P * sizeof(float), cudaMemcpyDeviceToHost, mm->stream));
    MCK(cudaStreamSynchronize(mm->stream));
    return LBM_OK;
}

lbm_status lbm_mlp_train(lbm_mlp* mm, const float* X, const float* T, int n, int epochs, int batch, double lr,
                         uint64_t shuffle_seed) {
    if (!mm || !X || !T || n < 1 || epochs < 0 || batch < 1 || !(lr > 0.0))
        return mfail(mm, LBM_ERR_INVALID_ARG, "bad training request");
    batch = std::min(batch, n);
    const TrainPlan p = train_plan(mm, batch);
    const int spe = n / batch;  // steps per epoch (a ragged tail is dropped)
    // epochs per launch: as many as about a megabyte of row order holds
    const int group = (int)std::max<int64_t>(1, std::min<int64_t>(epochs, (1 << 18) / n));
    Scratch s;
    CARVE((size_t)n * I, (size_t)n * O, 0, part_floats(mm, p), 0, (size_t)group * spe, (size_t)group * n);
    MCK(cudaMemcpyAsync(s.X, X, (size_t)n * I * sizeof(float), cudaMemcpyHostToDevice, mm->stream));
    MCK(cudaMemcpyAsync(s.T, T, (size_t)n * O * sizeof(float), cudaMemcpyHostToDevice, mm->stream));
    // two host buffers: a group is drawn while the previous one's upload and
    // training may still be running
    std::vector<int> order[2];
    std::vector<float2> coefs[2];
    for (int b = 0; b < (group < epochs ? 2 : 1); ++b) {
        order[b].resize((size_t)group * n);
        coefs[b].resize((size_t)group * spe);
    }
    uint64_t rs = shuffle_seed;
    for (int ep = 0; ep < epochs; ep += group) {
        std::vector<int>& perm = order[(ep / group) & 1];
        std::vector<float2>& coef = coefs[(ep / group) & 1];
        const int ne = std::min(group, epochs - ep);
        for (int g = 0; g < ne; ++g) {
            int* q = perm.data() + (size_t)g * n;
            for (int i = 0; i < n; ++i) q[i] = i;
            for (int i = n - 1; i > 0; --i) {  // Fisher-Yates with splitmix64
                const int j = (int)(splitmix64(rs) % (uint64_t)(i + 1));
                std::swap(q[i], q[j]);
            }
        }
        const int steps = ne * spe;
        for (int i = 0; i < steps; ++i) coef[i] = adam_coef(mm->t + 1 + i);
        MCK(cudaStreamSynchronize(mm->stream));  // the previous group reads s.idx and s.coef
        MCK(cudaMemcpyAsync(s.idx, perm.data(), (size_t)ne * n * sizeof(int), cudaMemcpyHostToDevice, mm->stream));
        MCK(cudaMemcpyAsync(s.coef, coef.data(), (size_t)steps * sizeof(float2), cudaMemcpyHostToDevice, mm->stream));
        TrainArgs a{mm->params, mm->m, mm->v, s.X, s.T, s.idx, s.coef, s.gp, nullptr,
                    batch, steps, n, spe, (float)lr, kBeta1, kBeta2, kEps};
        if (p.nc == 1) {
            MCK(run_train(a, p, mm->E, mm->stream));
        } else {
            a.out = cluster_sums(mm, p, s.gp);
            a.nsteps = 1;
            for (int i = 0; i < steps; ++i) {
                a.idx = s.idx + (size_t)(i / spe) * n + (size_t)(i % spe) * batch;
                MCK(run_train(a, p, mm->E, mm->stream));
                mlp_adam_kernel<<<dim3((P + 255) / 256, mm->E), 256, 0, mm->stream>>>(
                    mm->params, mm->m, mm->v, a.out, p.nc, (float)lr, kBeta1, kBeta2, coef[i].x, coef[i].y, kEps,
                    nullptr);
                MCK(cudaGetLastError());
            }
        }
        mm->t += steps;
    }
    lbm_status st = refresh_wt(mm);
    if (st != LBM_OK) return st;
    MCK(cudaStreamSynchronize(mm->stream));
    return LBM_OK;
}

lbm_status lbm_mlp_predict(lbm_mlp* mm, const float* X, int n, float* mean, float* spread, int dst_is_device) {
    if (!mm || !X || !mean || !spread || n < 1) return mfail(mm, LBM_ERR_INVALID_ARG, "bad predict request");
    Scratch s;
    const bool mapped = !dst_is_device && n <= kMappedPoints;
    const size_t hn = dst_is_device || mapped ? 0 : (size_t)n;
    CARVE(hn * I, hn * O, (size_t)mm->E * n * O, 0, hn, 0, 0);
    const float* dX = X;
    float *dm = mean, *ds = spread;
    if (mapped) {
        float* h = mm->hio;
        std::memcpy(h, X, (size_t)n * I * sizeof(float));
        dX = h;
        dm = h + (size_t)kMappedPoints * I;
        ds = dm + (size_t)kMappedPoints * O;
    } else if (!dst_is_device) {
        MCK(cudaMemcpyAsync(s.X, X, (size_t)n * I * sizeof(float), cudaMemcpyHostToDevice, mm->stream));
        dX = s.X;
        dm = s.T;
        ds = s.grad;
    }
    lbm_status st = launch_infer(mm, dX, n, s.Y);
    if (st != LBM_OK) return st;
    mlp_reduce_kernel<<<(n + 255) / 256, 256, 0, mm->stream>>>(s.Y, mm->E, n, dm, ds, mm->status, mm->hstatus);
    MCK(cudaGetLastError());
    if (!dst_is_device && !mapped) {
        MCK(cudaMemcpyAsync(mean, dm, (size_t)n * O * sizeof(float), cudaMemcpyDeviceToHost, mm->stream));
        MCK(cudaMemcpyAsync(spread, ds, (size_t)n * sizeof(float), cudaMemcpyDeviceToHost, mm->stream));
    }
    MCK(cudaStreamSynchronize(mm->stream));
    if (mapped) {
        std::memcpy(mean, dm, (size_t)n * O * sizeof(float));
        std::memcpy(spread, ds, (size_t)n * sizeof(float));
    }
    return infer_result(mm, *static_cast<volatile unsigned*>(mm->hstatus));
}

lbm_status lbm_mlp_set_wait_limit(lbm_mlp* mm, long long cycles) {
    if (!mm) return mfail(nullptr, LBM_ERR_INVALID_ARG, "mlp is NULL");
    if (cycles < 0) return mfail(mm, LBM_ERR_INVALID_ARG, "cycles must be >= 0");
    MCK(cudaStreamSynchronize(mm->stream));
    mm->wait_limit = cycles ? cycles : TC_WAIT_LIMIT;
    return LBM_OK;
}

lbm_status lbm_mlp_set_infer_path(lbm_mlp* mm, int path) {
    if (!mm) return mfail(nullptr, LBM_ERR_INVALID_ARG, "mlp is NULL");
    if (path != LBM_MLP_INFER_TENSOR && path != LBM_MLP_INFER_SIMT)
        return mfail(mm, LBM_ERR_INVALID_ARG, "unknown inference path");
    MCK(cudaStreamSynchronize(mm->stream));
    mm->infer_path = path;
    return LBM_OK;
}

void lbm_mlp_destroy(lbm_mlp* mm) {
    if (!mm) return;
    if (mm->stream) cudaStreamSynchronize(mm->stream);
    void* p[] = {mm->params, mm->m, mm->v, mm->wt, mm->tcimg, mm->status, mm->ws};
    for (void* q : p)
        if (q) cudaFree(q);
    if (mm->hstatus) cudaFreeHost(mm->hstatus);
    if (mm->hio) cudaFreeHost(mm->hio);
    delete mm;
}

const char* lbm_mlp_last_error(const lbm_mlp* mm) { return mm ? mm->err.c_str() : lbm_last_error(nullptr); }

}  // extern "C"
