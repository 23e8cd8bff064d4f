// mlp.cu -- the learned surrogate: a 3 -> 64 -> 64 -> 4 GELU perceptron in
// FP32 with hand-written training (forward, backward, Adam) and inference
// kernels, and a batched bisection that inverts sigma(kappa).
//
// Every kernel works on passes of kS = 8 samples per CTA of 256 threads:
// parameters and activations of the pass in shared memory, the 64 x 64 layer
// as register tiles of 4 samples x 4 units with the 64 terms split over
// eight lanes (forward and backward), and a 4 x 4 tile of its weight gradient
// per thread.  (A load of 16 bytes per lane costs shared memory four clocks,
// so the tile's reuse sets the pace of these phases; the split keeps all
// threads busy with 8 samples.)  The matrices are 64 wide and the data set a
// few thousand samples,
// so plain FP32 FMAs are used (FP32 accumulation is required; tensor cores
// would round the operands), and what bounds a minibatch is the chain of its
// phases and its exchange of gradients, not its 1.7 M multiply-adds.
// One pass costs about 4000 clocks, the exchange with its two barriers 4000.
//
// Training: one thread-block cluster of kC = 16 CTAs runs whole epochs in one
// launch (k_train).  Each CTA takes a sixteenth of a minibatch, sends its
// gradient sums to their owners through distributed shared memory (CTA r owns
// hidden units 4r .. 4r + 3 of every layer), and after a cluster barrier the
// owners add the sixteen contributions in a fixed order, apply Adam with their
// moments in registers and send the new parameters to every CTA; a second
// barrier starts the next minibatch.  Every CTA runs the same number of
// barriers and none leaves early.  Batches of more than kClusterMax samples
// instead spread their passes over the whole device (k_grad) and add the
// CTAs' rows of partial gradients in a second launch.  The sums' order depends
// on the sizes alone: results are deterministic.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "lbm_internal.cuh"

namespace {

constexpr int NI = LBM_MLP_IN, NH = LBM_MLP_HIDDEN, NO = LBM_MLP_OUT;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + NH * NI, OFF_W2 = OFF_B1 + NH, OFF_B2 = OFF_W2 + NH * NH,
              OFF_W3 = OFF_B2 + NH, OFF_B3 = OFF_W3 + NO * NH, NP = OFF_B3 + NO;
static_assert(NP == LBM_MLP_NPARAMS, "parameter count");
constexpr int kT = 256;             // threads per CTA
constexpr int kS = 8;               // samples per pass
constexpr int kLd3 = NH + 16;       // padded row of W3: rows 16 banks apart
constexpr int kLd = NH + 4;         // padded row of 64: 16-byte aligned, eight rows on 32 banks
constexpr int kC = 16;              // CTAs of the training cluster (more than 8: not portable, asked for)
constexpr int kOwn = NH / kC;       // hidden units whose parameters a CTA of the cluster owns
constexpr int NPL = NP + 1;         // partial-gradient row: parameters + loss
// a gradient slice: W2 rows, W1 rows, b1, b2, W3 columns of the owned units; b3 and the loss (owner 0)
constexpr int SL_W2 = 0, SL_W1 = SL_W2 + kOwn * NH, SL_B1 = SL_W1 + kOwn * NI, SL_B2 = SL_B1 + kOwn,
              SL_W3 = SL_B2 + kOwn, SL_B3 = SL_W3 + NO * kOwn, SL_LOSS = SL_B3 + NO, kSlice = 300;
static_assert(SL_LOSS < kSlice && kSlice % 4 == 0 && SL_LOSS == SL_B3 + NO && kOwn * NH == kT && kOwn == 4, "slice size");
constexpr int kSmall = SL_B3 - SL_W1;   // owned parameters outside W2

struct Norm {
    float in_mean[NI], in_std[NI], out_mean[NO], out_std[NO];
};

// ---- shared memory ---------------------------------------------------------
struct Net {
    float W2[NH * kLd];
    float W3[NO * kLd3];
    float W1[NH * NI], b1[NH], b2[NH], b3[NO];
};
// Activations of a pass.  G1, G2 hold the GELU derivatives, which the
// backward pass turns into dL/dz in place.
struct Pass {
    float H1[kS * kLd], G1[kS * kLd], H2[kS * kLd], G2[kS * kLd];
    float X[2][kS * 4], Y[2][kS * NO];   // inputs and targets, of this pass and the next
    float DY[kS * NO], L[kS];
    float one[kS * 4], zero[kS];         // a column of ones, of zeros
};

// Parameter p of the flat array in the shared-memory copy.
__device__ __forceinline__ float& net_at(Net& N, int p) {
    if (p < OFF_B1) return N.W1[p - OFF_W1];
    if (p < OFF_W2) return N.b1[p - OFF_B1];
    if (p < OFF_B2) return N.W2[((p - OFF_W2) / NH) * kLd + (p - OFF_W2) % NH];
    if (p < OFF_W3) return N.b2[p - OFF_B2];
    if (p < OFF_B3) return N.W3[((p - OFF_W3) / NH) * kLd3 + (p - OFF_W3) % NH];
    return N.b3[p - OFF_B3];
}
__device__ __forceinline__ void load_net(Net& N, const float* __restrict__ P) {
    for (int p = threadIdx.x; p < NP; p += kT) net_at(N, p) = P[p];
}

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float dot4(float4 a, float4 b, float c) {
    return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, c))));
}

// GELU and, for training, its derivative.
template <bool TRAIN> __device__ __forceinline__ float gelu(float z, float* d) {
    const float e = erff(z * 0.70710678118654752f);
    if (TRAIN) *d = 0.5f * (1.0f + e) + z * 0.39894228040143268f * expf(-0.5f * z * z);
    return 0.5f * z * (1.0f + e);
}

// Sums of a 4 x 4 tile over the eight lanes that hold its parts: each
// exchange halves the values a lane carries; lane l of the eight ends with
// entries (tile_row(l), tile_col(l)) and the one after it.
__device__ __forceinline__ int tile_row(int lane) { return (lane >> 1) & 3; }
__device__ __forceinline__ int tile_col(int lane) { return (lane & 1) * 2; }
__device__ __forceinline__ void tile_sums(const float (&v)[4][4], float (&out)[2]) {
    const int lane = threadIdx.x & 31;
    float a[2][4], b[4];
    const bool u4 = lane & 4, u2 = lane & 2, u1 = lane & 1;
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c)
            a[r][c] = (u4 ? v[r + 2][c] : v[r][c]) + __shfl_xor_sync(0xffffffffu, u4 ? v[r][c] : v[r + 2][c], 4);
#pragma unroll
    for (int c = 0; c < 4; ++c) b[c] = (u2 ? a[1][c] : a[0][c]) + __shfl_xor_sync(0xffffffffu, u2 ? a[0][c] : a[1][c], 2);
#pragma unroll
    for (int c = 0; c < 2; ++c) out[c] = (u1 ? b[c + 2] : b[c]) + __shfl_xor_sync(0xffffffffu, u1 ? b[c] : b[c + 2], 1);
}

// Both hidden layers of the pass whose inputs are in A.X[buf].  Ends with
// every H2 (and G1, G2) written, before a barrier.
template <bool TRAIN> __device__ __forceinline__ void hidden(const Net& N, Pass& A, int buf) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    {
        const int j = t & (NH - 1);
        const float w0 = N.W1[j * NI], w1 = N.W1[j * NI + 1], w2 = N.W1[j * NI + 2], b = N.b1[j];
#pragma unroll
        for (int s = t / NH; s < kS; s += kT / NH) {
            const float4 x = ld4(A.X[buf] + s * 4);
            A.H1[s * kLd + j] = gelu<TRAIN>(fmaf(w2, x.z, fmaf(w1, x.y, fmaf(w0, x.x, b))), &A.G1[s * kLd + j]);
        }
    }
    __syncthreads();
    {
        // tile of samples 4 sq .. and units 4 jq .., quads 4 (8 q + part) of its sums
        const int part = lane & 7, tile = warp * 4 + (lane >> 3), sq = tile & 1, jq = tile >> 1;
        const float *w = N.W2 + jq * 4 * kLd + part * 4, *h = A.H1 + sq * 4 * kLd + part * 4;
        float acc[4][4];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            float4 wv[4], hv[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) wv[c] = ld4(w + c * kLd + q * 32);
#pragma unroll
            for (int r = 0; r < 4; ++r) hv[r] = ld4(h + r * kLd + q * 32);
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[r][c] = dot4(wv[c], hv[r], q ? acc[r][c] : 0.0f);
        }
        float z[2];
        tile_sums(acc, z);
        const int s = sq * 4 + tile_row(lane), j = jq * 4 + tile_col(lane), o = s * kLd + j;
#pragma unroll
        for (int c = 0; c < 2; ++c) A.H2[o + c] = gelu<TRAIN>(z[c] + N.b2[j + c], &A.G2[o + c]);
    }
}

// Output k of sample s, (s, k) = divmod(t / 8, 4), in all eight threads of the group.
__device__ __forceinline__ float output(const Net& N, const Pass& A) {
    const int t = threadIdx.x, o = t >> 3, s = o >> 2, k = o & 3, part = (t & 7) * 4;
    float y = 0.0f;
#pragma unroll
    for (int i = 0; i < NH; i += 32) y = dot4(ld4(N.W3 + k * kLd3 + part + i), ld4(A.H2 + s * kLd + part + i), y);
    y += __shfl_xor_sync(0xffffffffu, y, 1);
    y += __shfl_xor_sync(0xffffffffu, y, 2);
    y += __shfl_xor_sync(0xffffffffu, y, 4);
    return y + N.b3[k];
}

// This thread's gradient sums: a 4 x 4 tile of W2, one entry each of W3, of
// W1 or b1 (threads from 192 on), and of b2, b3 or the loss.
struct Sums {
    float w2[4][4] = {}, w3 = 0.0f, w1 = 0.0f, b = 0.0f;
};

// Forward and backward pass of the nloc samples in A.X[buf], A.Y[buf] (the
// rest of the kS rows contribute nothing), added to G.  Ends before a barrier.
__device__ __forceinline__ void backward(const Net& N, Pass& A, int buf, int nloc, float inv_norm, Sums& G) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    hidden<true>(N, A, buf);
    __syncthreads();
    {
        const float y = output(N, A);
        const int s = t >> 5, k = (t >> 3) & 3;
        const float e = s < nloc ? y - A.Y[buf][s * NO + k] : 0.0f;
        float l = e * e;
        l += __shfl_xor_sync(0xffffffffu, l, 8);
        l += __shfl_xor_sync(0xffffffffu, l, 16);
        if ((t & 7) == 0) A.DY[s * NO + k] = 2.0f * e * inv_norm;
        if (lane == 0) A.L[s] = l * inv_norm;
    }
    __syncthreads();
    {   // dZ2 = (W3^T dY) * gelu'(z2)
        const int j = t & (NH - 1);
        const float w0 = N.W3[j], w1 = N.W3[kLd3 + j], w2 = N.W3[2 * kLd3 + j], w3 = N.W3[3 * kLd3 + j];
#pragma unroll
        for (int s = t / NH; s < kS; s += kT / NH) {
            const float4 d = ld4(A.DY + s * NO);
            A.G2[s * kLd + j] *= fmaf(w3, d.w, fmaf(w2, d.z, fmaf(w1, d.y, w0 * d.x)));
        }
    }
    __syncthreads();
    {   // dZ1 = (W2^T dZ2) * gelu'(z1): tile of samples 4 sq .. and units 4 iq .., terms 8 q + part of its sums
        const int part = lane & 7, tile = warp * 4 + (lane >> 3), sq = tile & 1, iq = tile >> 1;
        const float *w = N.W2 + part * kLd + iq * 4, *d = A.G2 + sq * 4 * kLd + part;
        float acc[4][4] = {};
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float4 wv = ld4(w + q * 8 * kLd);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const float dv = d[r * kLd + q * 8];
                acc[r][0] = fmaf(dv, wv.x, acc[r][0]);
                acc[r][1] = fmaf(dv, wv.y, acc[r][1]);
                acc[r][2] = fmaf(dv, wv.z, acc[r][2]);
                acc[r][3] = fmaf(dv, wv.w, acc[r][3]);
            }
        }
        float z[2];
        tile_sums(acc, z);
        float* const g = A.G1 + (sq * 4 + tile_row(lane)) * kLd + iq * 4 + tile_col(lane);
        g[0] *= z[0];
        g[1] *= z[1];
    }
    __syncthreads();
    // this pass's share of the gradient, summed over its samples; entries
    // that a thread does not have read a column of ones or zeros
    const int jq = (t >> 4) * 4, iq = (t & 15) * 4;
    const float *dy = A.DY + (t >> 6), *h2 = A.H2 + (t & (NH - 1));
    const float *g1 = A.G1 + (t < NH * NI ? t / NI : t - NH * NI), *x1 = t < NH * NI ? A.X[buf] + t % NI : A.one;
    const float* pb = t < NH ? A.G2 + t : (t < NH + NO ? A.DY + t - NH : (t == NH + NO ? A.L : A.zero));
    const int ldb = t < NH ? kLd : (t < NH + NO ? NO : 1);
#pragma unroll
    for (int s = 0; s < kS; ++s) {
        const float4 d = ld4(A.G2 + s * kLd + jq), h = ld4(A.H1 + s * kLd + iq);
        const float dv[4] = {d.x, d.y, d.z, d.w}, hv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) G.w2[r][c] = fmaf(dv[r], hv[c], G.w2[r][c]);
        G.w3 = fmaf(dy[s * NO], h2[s * kLd], G.w3);
        G.w1 = fmaf(g1[s * kLd], x1[s * 4], G.w1);
        G.b += pb[s * ldb];
    }
}

// The columns of ones and zeros (before the first pass).
__device__ __forceinline__ void fill_constants(Pass& A) {
    if (threadIdx.x < kS * 4) A.one[threadIdx.x] = 1.0f;
    if (threadIdx.x < kS) A.zero[threadIdx.x] = 0.0f;
}

// The sample a thread fetches for a pass, and its part of it: thread
// (s, c), c < 7, brings column c of sample s (three inputs, four targets).
__device__ __forceinline__ float fetch(const float* __restrict__ X, const float* __restrict__ Y, int g, int c) {
    return c < NI ? __ldg(X + static_cast<long long>(g) * NI + c) : __ldg(Y + static_cast<long long>(g) * NO + c - NI);
}
__device__ __forceinline__ void put(Pass& A, int buf, int s, int c, float v) {
    if (c < NI) A.X[buf][s * 4 + c] = v;
    else A.Y[buf][s * NO + c - NI] = v;
}

// ---- training: whole epochs in one cluster ---------------------------------
struct TrainArgs {
    float *P, *M, *V;
    const float *X, *Y;      // n x 3 standardised inputs, n x 4 standardised targets
    const int* order;        // sample order of every epoch, n each
    const float2* corr;      // Adam's bias corrections 1 - b1^t, 1 - b2^t, per minibatch
    float* losses;           // per minibatch
    int n, batch, epochs;
    float lr, b1, b2, eps;
};

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_barrier() {
    asm volatile(
        "barrier.cluster.arrive.release.aligned;\n\t"
        "barrier.cluster.wait.acquire.aligned;" ::
            : "memory");
}
__device__ __forceinline__ uint32_t cluster_map(const void* p, unsigned rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(lbm::smem_u32(p)), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_cluster(uint32_t a, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void st_cluster4(uint32_t a, float4 v) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}
__device__ __forceinline__ void st_cluster4(uint32_t a, const float (&v)[4]) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v[0]), "f"(v[1]), "f"(v[2]),
                 "f"(v[3])
                 : "memory");
}

struct TrainSmem {
    Net N;
    Pass A;
    float R[kC][kSlice];   // the gradient slice this CTA owns, from every CTA of the cluster
};

// Flat parameter index of entry e (< kSmall) of the owned parameters outside W2.
__device__ __forceinline__ int small_param(int e, int unit0) {
    if (e < SL_B1 - SL_W1) return OFF_W1 + unit0 * NI + e;
    e -= SL_B1 - SL_W1;
    if (e < kOwn) return OFF_B1 + unit0 + e;
    e -= kOwn;
    if (e < kOwn) return OFF_B2 + unit0 + e;
    e -= kOwn;
    return OFF_W3 + (e / kOwn) * NH + unit0 + e % kOwn;
}

// A minibatch of 128 is one pass per CTA and takes 5.2 us (68 us as one
// thread per sample on two CTAs and a second launch for the sums and Adam):
// 600 epochs of 2000 samples in minibatches of 128 take 0.05 s, not 0.65.
// The index of a sample is fetched two passes ahead (from the host's memory)
// and the sample one, Adam's corrections at the start of the minibatch, so
// that no load from outside the SM is waited for.
__global__ void __launch_bounds__(kT, 1) k_train(const TrainArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TrainSmem& S = *reinterpret_cast<TrainSmem*>(smem_raw);
    const int t = threadIdx.x;
    const int rank = static_cast<int>(cluster_rank());
    const int unit0 = rank * kOwn;
    load_net(S.N, a.P);
    fill_constants(S.A);
    // the owned parameters of this thread: one of W2, and for the first ones
    // one outside it (b3 on CTA 0), with their moments; thread kSmall + NO of
    // CTA 0 has the loss
    const int wrow = t / NH, wcol = t % NH, pw = OFF_W2 + (unit0 + wrow) * NH + wcol;
    int ps = -1;
    if (t < kSmall) ps = small_param(t, unit0);
    else if (rank == 0 && t < kSmall + NO) ps = OFF_B3 + t - kSmall;
    const bool has_loss = rank == 0 && t == kSmall + NO, small = ps >= 0 || has_loss;
    const int es = has_loss ? SL_LOSS : (t < kSmall ? SL_W1 + t : (small ? SL_B3 + t - kSmall : 0));
    float mw = a.M[pw], vw = a.V[pw], ms = ps >= 0 ? a.M[ps] : 0.0f, vs = ps >= 0 ? a.V[ps] : 0.0f;
    float* const w = &S.N.W2[(unit0 + wrow) * kLd + wcol];
    float* const u = &net_at(S.N, ps >= 0 ? ps : 0);
    // what this thread sends: quad t % 64 of the owned W2 rows, and quad
    // t / kC (three of W1, b1, b2, four of W3, b3 from CTA 0) to CTA t % kC
    const float* const quad = &S.N.W2[(unit0 + ((t >> 4) & 3)) * kLd + (t & 15) * 4];
    const float* squad = nullptr;
    const int sq = t / kC;
    if (sq < 3) squad = S.N.W1 + unit0 * NI + sq * 4;
    else if (sq == 3) squad = S.N.b1 + unit0;
    else if (sq == 4) squad = S.N.b2 + unit0;
    else if (sq < 9) squad = S.N.W3 + (sq - 5) * kLd3 + unit0;
    else if (sq == 9 && rank == 0) squad = S.N.b3;

    const int nb = (a.n + a.batch - 1) / a.batch, total = nb * a.epochs;
    // minibatch k of an epoch: this CTA's samples are order[base .. base + cnt) of the epoch
    struct Mb { int count, per, base, cnt; };
    auto minibatch = [&](int k) {
        Mb b;
        b.count = min(a.batch, a.n - k * a.batch);
        b.per = (b.count + kC - 1) / kC;
        b.base = k * a.batch + rank * b.per;
        b.cnt = max(0, min(b.per, b.count - rank * b.per));
        return b;
    };
    const int fs = t / 7, fc = t - fs * 7;
    const bool fetches = fs < kS;
    int fmb = 0, fk = 0, fq = 0;   // the pass whose index is fetched next
    const int* forder = a.order;   // of its epoch
    auto fetch_index = [&]() -> int {
        int g = -1;
        if (fmb < total) {
            const Mb b = minibatch(fk);
            if (fetches && fq * kS + fs < b.cnt) g = __ldg(forder + b.base + fq * kS + fs);
            if (++fq * kS >= b.per) {
                fq = 0;
                ++fmb;
                if (++fk == nb) {
                    fk = 0;
                    forder += a.n;
                }
            }
        }
        return g;
    };
    int g_next = fetch_index();
    if (fetches) put(S.A, 0, fs, fc, g_next >= 0 ? fetch(a.X, a.Y, g_next, fc) : 0.0f);
    g_next = fetch_index();
    cluster_barrier();   // every CTA has started, and this one's shared memory is filled

    int buf = 0;
#pragma unroll 1
    for (int mb = 0, k = 0; mb < total; ++mb, k = k + 1 == nb ? 0 : k + 1) {
        const Mb b = minibatch(k);
        const float inv_norm = 1.0f / (static_cast<float>(b.count) * NO);
        const float2 corr = __ldg(a.corr + mb);
        Sums G;
#pragma unroll 1
        for (int q = 0; q * kS < b.per; ++q) {
            const float v = fetches && g_next >= 0 ? fetch(a.X, a.Y, g_next, fc) : 0.0f;
            g_next = fetch_index();
            backward(S.N, S.A, buf, b.cnt - q * kS, inv_norm, G);
            buf ^= 1;
            if (fetches) put(S.A, buf, fs, fc, v);   // read two passes ago
            if ((q + 1) * kS < b.per) __syncthreads();
        }
        // the sums to their owners
        {
            const int jq = (t >> 4) * 4, iq = (t & 15) * 4;
            const uint32_t to = cluster_map(&S.R[rank][SL_W2 + iq], jq / kOwn);
#pragma unroll
            for (int r = 0; r < kOwn; ++r) st_cluster4(to + r * NH * 4, G.w2[r]);
            const int k3 = t >> 6, j3 = t & (NH - 1);
            st_cluster(cluster_map(&S.R[rank][SL_W3 + k3 * kOwn + j3 % kOwn], j3 / kOwn), G.w3);
            const int j1 = t < NH * NI ? t / NI : t - NH * NI;
            const int e1 = t < NH * NI ? SL_W1 + (j1 % kOwn) * NI + t % NI : SL_B1 + j1 % kOwn;
            st_cluster(cluster_map(&S.R[rank][e1], j1 / kOwn), G.w1);
            if (t < NH) st_cluster(cluster_map(&S.R[rank][SL_B2 + t % kOwn], t / kOwn), G.b);
            else if (t <= NH + NO) st_cluster(cluster_map(&S.R[rank][SL_B3 + t - NH], 0), G.b);
        }
        cluster_barrier();
        // the owners: the contributions in rank order, Adam, new parameters to every CTA
        float g = 0.0f, gs = 0.0f;
#pragma unroll
        for (int r = 0; r < kC; ++r) {
            g += S.R[r][SL_W2 + t];
            gs += S.R[r][es];
        }
        if (has_loss) a.losses[mb] = gs;
        auto adam = [&](float p, float grad, float& m, float& v) {
            m = a.b1 * m + (1.0f - a.b1) * grad;
            v = a.b2 * v + (1.0f - a.b2) * grad * grad;
            return p - a.lr * (m / corr.x) / (sqrtf(v / corr.y) + a.eps);
        };
        // (every thread runs both updates side by side; those without a
        // parameter outside W2 drop the second)
        float md = ms, vd = vs;
        const float wn = adam(*w, g, mw, vw), un = adam(*u, gs, md, vd);
        *w = wn;
        if (ps >= 0) {
            *u = un;
            ms = md;
            vs = vd;
        }
        __syncthreads();
        // 16 bytes per store: the owned W2 rows to four CTAs per thread, and
        // the quads outside W2
#pragma unroll
        for (int r = 0; r < 4; ++r) st_cluster4(cluster_map(quad, (t >> 6) * 4 + r), ld4(quad));
        if (squad) st_cluster4(cluster_map(squad, t % kC), ld4(squad));
        cluster_barrier();
    }
    a.P[pw] = *w;
    a.M[pw] = mw;
    a.V[pw] = vw;
    if (ps >= 0) {
        a.P[ps] = *u;
        a.M[ps] = ms;
        a.V[ps] = vs;
    }
}

// ---- large batches: passes over the whole device ---------------------------
// Samples order[first .. first + count) (order NULL: as they are), each CTA
// every gridDim-th pass; one row of partial gradients per CTA.
struct GradSmem {
    Net N;
    Pass A;
};
__global__ void __launch_bounds__(kT, 2) k_grad(const float* __restrict__ P, const float* __restrict__ X,
                                             const float* __restrict__ Y, const int* __restrict__ order, int first,
                                             int count, float inv_norm, float* __restrict__ partials) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    GradSmem& S = *reinterpret_cast<GradSmem*>(smem_raw);
    const int t = threadIdx.x, fs = t / 7, fc = t - fs * 7;
    load_net(S.N, P);
    fill_constants(S.A);
    Sums G;
    for (int c0 = blockIdx.x * kS; c0 < count; c0 += gridDim.x * kS) {
        if (fs < kS) {
            const int k = c0 + fs;
            put(S.A, 0, fs, fc, k < count ? fetch(X, Y, order ? order[first + k] : first + k, fc) : 0.0f);
        }
        __syncthreads();
        backward(S.N, S.A, 0, count - c0, inv_norm, G);
        __syncthreads();
    }
    float* const out = partials + static_cast<long long>(blockIdx.x) * NPL;
    const int jq = (t >> 4) * 4, iq = (t & 15) * 4;
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) out[OFF_W2 + (jq + r) * NH + iq + c] = G.w2[r][c];
    out[OFF_W3 + t] = G.w3;
    out[t < NH * NI ? OFF_W1 + t : OFF_B1 + t - NH * NI] = G.w1;
    if (t < NH) out[OFF_B2 + t] = G.b;
    else if (t < NH + NO) out[OFF_B3 + t - NH] = G.b;
    else if (t == NH + NO) out[NP] = G.b;
}

// Sum the partial-gradient rows in a fixed order; optionally apply Adam.
__global__ void k_reduce_adam(const float* __restrict__ partials, int nparts, float* __restrict__ P,
                              float* __restrict__ M, float* __restrict__ V, float* __restrict__ grad_out,
                              float* __restrict__ loss_out, int do_update, float lr, float b1, float b2, float eps,
                              float c1, float c2) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p > NP) return;
    float g = 0.0f;
    for (int r = 0; r < nparts; ++r) g += partials[static_cast<long long>(r) * NPL + p];
    if (p == NP) {
        if (loss_out) *loss_out = g;
        return;
    }
    if (grad_out) grad_out[p] = g;
    if (do_update) {
        const float m = b1 * M[p] + (1.0f - b1) * g;
        const float v = b2 * V[p] + (1.0f - b2) * g * g;
        M[p] = m;
        V[p] = v;
        P[p] -= lr * (m / c1) / (sqrtf(v / c2) + eps);
    }
}

// Raw samples to standardised ones, by IEEE division (in place or not).  Bound
// by the pinned memory's latency, one sample value a thread; with the sample
// orders read in place it replaces five copies a call (2000 samples, 4
// epochs of minibatches of 128: 466 -> 453 us).
__global__ void k_standardise(const float* x, const float* y, int n, Norm nm, float* X, float* Y) {
    const long long nx = static_cast<long long>(n) * NI, all = static_cast<long long>(n) * (NI + NO);
    for (long long i = blockIdx.x * static_cast<long long>(kT) + threadIdx.x; i < all;
         i += static_cast<long long>(gridDim.x) * kT) {
        if (i < nx) {
            const int c = static_cast<int>(i % NI);
            X[i] = (x[i] - nm.in_mean[c]) / nm.in_std[c];
        } else {
            const long long j = i - nx;
            const int k = static_cast<int>(j % NO);
            Y[j] = (y[j] - nm.out_mean[k]) / nm.out_std[k];
        }
    }
}

// New parameters, moments at zero.
__global__ void k_set_params(const float* __restrict__ from, float* __restrict__ P, float* __restrict__ M,
                             float* __restrict__ V) {
    const int p = blockIdx.x * kT + threadIdx.x;
    if (p >= NP) return;
    P[p] = from[p];
    M[p] = V[p] = 0.0f;
}

// ---- inference ---------------------------------------------------------------
// Inference on raw inputs: standardise, forward, de-standardise; CTAs
// striding over the passes.
__global__ void __launch_bounds__(kT, 2) k_predict(const float* __restrict__ P, Norm nm, const float* __restrict__ X,
                                                int n, float* __restrict__ Y) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    GradSmem& S = *reinterpret_cast<GradSmem*>(smem_raw);
    const int t = threadIdx.x;
    load_net(S.N, P);
    for (int c0 = blockIdx.x * kS; c0 < n; c0 += gridDim.x * kS) {
        if (t < kS * NI) {
            const int s = t / NI, c = t - s * NI;
            S.A.X[0][s * 4 + c] =
                c0 + s < n ? (X[static_cast<long long>(c0) * NI + t] - nm.in_mean[c]) / nm.in_std[c] : 0.0f;
        }
        __syncthreads();
        hidden<false>(S.N, S.A, 0);
        __syncthreads();
        const float y = output(S.N, S.A);
        const int s = t >> 5, k = (t >> 3) & 3;
        if ((t & 7) == 0 && c0 + s < n) Y[static_cast<long long>(c0 + s) * NO + k] = y * nm.out_std[k] + nm.out_mean[k];
        __syncthreads();
    }
}

// Bisection on kappa for each target: predicted sigma (output 0) decreases in
// kappa.  A bisection is a chain of 2 + kHalvings evaluations; here one pass
// evaluates the midpoints of the next LEVELS halvings at once (a binary tree
// of 2^LEVELS - 1 of them per target, 8 / 2^LEVELS targets per CTA), then
// walks down the tree: the same midpoints, formed by the same arithmetic, and
// the same choices as one halving after another, in kHalvings / LEVELS
// passes.  LEVELS = 1 takes 8 targets per CTA, one halving per pass.
constexpr int kHalvings = 40;
template <int LEVELS>
__global__ void __launch_bounds__(kT, 2) k_invert(const float* __restrict__ P, Norm nm, const float* __restrict__ tr,
                                               const float* __restrict__ A, const float* __restrict__ sig, int m,
                                               float lo, float hi, float* __restrict__ kappa) {
    constexpr int kSlots = LEVELS == 1 ? 1 : 1 << LEVELS;   // rows of a pass per target
    constexpr int kTargets = kS / kSlots;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    GradSmem& S = *reinterpret_cast<GradSmem*>(smem_raw);
    __shared__ float s_sigma[kS];
    const int t = threadIdx.x;
    load_net(S.N, P);
    const int row = t % kS, target = blockIdx.x * kTargets + row / kSlots, slot = row % kSlots, base = row - slot;
    if (t < kS) {
        S.A.X[0][t * 4] = target < m ? (tr[target] - nm.in_mean[0]) / nm.in_std[0] : 0.0f;
        S.A.X[0][t * 4 + 1] = target < m ? (A[target] - nm.in_mean[1]) / nm.in_std[1] : 0.0f;
    }
    // sigma of the kS rows' kappas (in the first kS threads)
    auto evaluate = [&](float k) {
        if (t < kS) S.A.X[0][t * 4 + 2] = (k - nm.in_mean[2]) / nm.in_std[2];
        __syncthreads();
        hidden<false>(S.N, S.A, 0);
        __syncthreads();
        const float y = output(S.N, S.A);
        if ((t & 31) == 0) s_sigma[t >> 5] = y * nm.out_std[0] + nm.out_mean[0];
        __syncthreads();
    };
    const float want = target < m ? sig[target] : 0.0f;
    float a = lo, b = hi;
    bool inside;
    if (kSlots == 1) {
        evaluate(a);
        const float fa = s_sigma[row] - want;
        __syncthreads();
        evaluate(b);
        inside = fa >= 0.0f && s_sigma[row] - want <= 0.0f;
    } else {
        evaluate(slot == 0 ? a : b);
        inside = s_sigma[base] - want >= 0.0f && s_sigma[base + 1] - want <= 0.0f;
    }
    __syncthreads();
    for (int it = 0; it < kHalvings; it += LEVELS) {
        // node `slot` of the tree (1: the root; children 2k, taken when b moves, and 2k + 1, when a does)
        float x = a, y = b, mid = 0.5f * (x + y);
        if (kSlots > 1 && slot > 0) {
            for (int bit = 30 - __clz(slot); bit >= 0; --bit) {
                if ((slot >> bit) & 1) x = mid; else y = mid;
                mid = 0.5f * (x + y);
            }
        }
        evaluate(mid);
        int node = 1;
        for (int l = 0; l < LEVELS && it + l < kHalvings; ++l) {
            const float md = 0.5f * (a + b);
            const bool up = s_sigma[kSlots == 1 ? row : base + node] - want >= 0.0f;
            if (up) a = md; else b = md;
            node = 2 * node + (up ? 1 : 0);
        }
        __syncthreads();
    }
    if (t < kS && slot == 0 && target < m) kappa[target] = inside ? 0.5f * (a + b) : nanf("");
}

uint64_t splitmix(uint64_t& s) {
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

double uniform01(uint64_t& s) { return (splitmix(s) >> 11) * (1.0 / 9007199254740992.0); }

}  // namespace

struct lbm_mlp {
    int max_n = 0;
    void* dev = nullptr;     // the device memory that the buffers are in
    cudaStream_t st = nullptr;
    Norm norm{};
    float *P = nullptr, *M = nullptr, *V = nullptr, *X = nullptr, *Y = nullptr, *partials = nullptr,
          *grad = nullptr, *sum = nullptr, *io = nullptr;   // sum: the loss of a single gradient
    // training (from the first call of it on): the sample orders, bias
    // corrections and losses of a launch's epochs, twice, so that the host
    // prepares a launch while another runs; in pinned memory, where the
    // kernels fetch them minibatches ahead of their use
    int* order[2] = {};
    float2* corr[2] = {};
    float* loss[2] = {};
    void* stage = nullptr;   // the memory these are in
    cudaEvent_t done[2] = {};
    lbm::Pinned pinned;
    float* h_io = nullptr;   // in it (pinned and mapped): NI + NO floats of up to io_n samples (or the parameters), for the kernels
    int io_n = 0;
    int cap = 0;             // samples (and minibatches) each of them holds
    int adam_t = 0;
    bool cluster = false;    // the device holds the training cluster (else every batch goes over the whole device)
};

namespace {

constexpr int kRows = 304;            // CTAs of k_grad: two per SM
constexpr int kOrderMin = 1 << 14;    // samples of the order buffers at least
constexpr int kIoMax = 1 << 16;       // samples of the pinned buffer at most
// Batches up to this size are trained in the cluster, larger ones over the
// whole device (per minibatch of 128 / 512 / 768 / 1024 / 4096 samples: 5.4 / 12.4 /
// 16.7 / 21.7 / 77 us in the cluster, 14.6 / 17.3 / 17.9 / 18.6 / 39 us as two launches).
constexpr int kClusterMax = 768;

bool valid(lbm_mlp* m) { return m && m->P; }
// the samples, or the parameters
size_t io_bytes(const lbm_mlp* m) {
    return sizeof(float) * std::max<size_t>((NI + NO) * static_cast<size_t>(m->io_n), NP);
}

// A block of memory cut into buffers, each a multiple of 16 bytes so that all
// are aligned alike (with at == NULL: their sizes only).
struct Cut {
    char* at;
    size_t used;
    void* take(size_t bytes) {
        void* p = at ? at + used : nullptr;
        used += (bytes + 15) / 16 * 16;
        return p;
    }
};

// The buffers of training, made by its first call and kept.
int ensure_stage(lbm_mlp* m) {
    if (m->cap) return LBM_OK;
    const size_t cap = std::max(m->max_n, kOrderMin);
    auto cut = [&](Cut c) {
        for (int k = 0; k < 2; ++k) {
            m->corr[k] = static_cast<float2*>(c.take(cap * sizeof(float2)));
            m->order[k] = static_cast<int*>(c.take(cap * sizeof(int)));
            m->loss[k] = static_cast<float*>(c.take(cap * sizeof(float)));
        }
        return c.used;
    };
    const size_t bytes = cut({nullptr, 0});
    bool ok = m->stage || cudaHostAlloc(&m->stage, bytes, cudaHostAllocMapped) == cudaSuccess;
    for (auto& e : m->done) ok = ok && (e || cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess);
    if (!ok) {
        cudaGetLastError();
        return LBM_ENOMEM;
    }
    cut({static_cast<char*>(m->stage), 0});
    m->cap = static_cast<int>(cap);
    return LBM_OK;
}

// Standardised samples to m->X, m->Y, enqueued: from pinned memory, which
// every call has done with before it returns, or in place from copies.
int standardise_upload(lbm_mlp* m, const float* X, const float* Y, int n) {
    const size_t bytes = static_cast<size_t>(n) * sizeof(float);
    const float *x = m->X, *y = m->Y;
    if (n <= m->io_n) {
        std::memcpy(m->h_io, X, NI * bytes);
        std::memcpy(m->h_io + static_cast<size_t>(n) * NI, Y, NO * bytes);
        x = m->h_io;
        y = m->h_io + static_cast<size_t>(n) * NI;
    } else if (cudaMemcpyAsync(m->X, X, NI * bytes, cudaMemcpyHostToDevice, m->st) != cudaSuccess ||
               cudaMemcpyAsync(m->Y, Y, NO * bytes, cudaMemcpyHostToDevice, m->st) != cudaSuccess ||
               cudaStreamSynchronize(m->st) != cudaSuccess) {
        return LBM_ECUDA;
    }
    const int blocks = std::min(n / 32 + 1, 8 * kRows);
    k_standardise<<<blocks, kT, 0, m->st>>>(x, y, n, m->norm, m->X, m->Y);
    return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_ECUDA;
}

float2 next_corr(lbm_mlp* m, float b1, float b2) {
    ++m->adam_t;
    return make_float2(1.0f - std::pow(b1, static_cast<float>(m->adam_t)),
                       1.0f - std::pow(b2, static_cast<float>(m->adam_t)));
}

// The launch of the training cluster.
void train_config(cudaStream_t st, cudaLaunchConfig_t& cfg, cudaLaunchAttribute& attr) {
    cfg = {};
    cfg.gridDim = dim3(kC);
    cfg.blockDim = dim3(kT);
    cfg.dynamicSmemBytes = sizeof(TrainSmem);
    cfg.stream = st;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = kC;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
}

// The kernels' attributes on the current device, set by the first network
// made on it, and whether it can hold the training cluster.
bool prepare_kernels(bool* cluster) {
    constexpr int kDevices = 64;
    static std::mutex mu;
    static int known[kDevices];   // 1: attributes set, no cluster; 2: cluster too
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    std::lock_guard<std::mutex> lock(mu);
    int k = dev >= 0 && dev < kDevices ? known[dev] : 0;
    if (!k) {
        auto room = [](auto fn, size_t bytes) {
            return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes)) ==
                   cudaSuccess;
        };
        if (!room(k_train, sizeof(TrainSmem)) || !room(k_grad, sizeof(GradSmem)) || !room(k_predict, sizeof(GradSmem)) ||
            !room(k_invert<1>, sizeof(GradSmem)) || !room(k_invert<2>, sizeof(GradSmem)) ||
            !room(k_invert<3>, sizeof(GradSmem)) ||
            cudaFuncSetAttribute(k_train, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
            return false;
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr;
        int n = 0;
        train_config(nullptr, cfg, attr);
        k = cudaOccupancyMaxActiveClusters(&n, &k_train, &cfg) == cudaSuccess && n > 0 ? 2 : 1;
        if (k == 1) cudaGetLastError();
        if (dev >= 0 && dev < kDevices) known[dev] = k;
    }
    *cluster = k == 2;
    return true;
}

// Epochs in the cluster, enqueued.
cudaError_t launch_train(lbm_mlp* m, const TrainArgs& a) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr;
    train_config(m->st, cfg, attr);
    return cudaLaunchKernelEx(&cfg, &k_train, a);
}

// Gradient (and optional Adam update) over samples order[first .. first +
// count) (order NULL: samples first ..) on the whole device, enqueued.
cudaError_t grad_pass(lbm_mlp* m, const int* order, int first, int count, bool update, float lr, float b1, float b2,
                      float eps, float2 corr, float* loss_slot) {
    const int chunks = (count + kS - 1) / kS, rows = std::min(chunks, kRows);
    k_grad<<<rows, kT, sizeof(GradSmem), m->st>>>(m->P, m->X, m->Y, order, first, count,
                                                  1.0f / (static_cast<float>(count) * NO), m->partials);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_reduce_adam<<<(NP + 1 + 127) / 128, 128, 0, m->st>>>(m->partials, rows, m->P, m->M, m->V, m->grad, loss_slot,
                                                           update ? 1 : 0, lr, b1, b2, eps, corr.x, corr.y);
    return cudaGetLastError();
}

}  // namespace

extern "C" {

int lbm_mlp_create(lbm_mlp** out, int max_samples, unsigned long long seed, void* stream) {
    if (!out || max_samples < 1) return LBM_EINVAL;
    *out = nullptr;
    lbm_mlp* m = new lbm_mlp();
    m->max_n = max_samples;
    m->st = static_cast<cudaStream_t>(stream);
    const size_t max_rows = std::min((max_samples + kS - 1) / kS, kRows), rows = static_cast<size_t>(max_samples);
    m->io_n = std::min(max_samples, kIoMax);
    auto cut = [&](Cut c) {
        auto floats = [&](size_t n) { return static_cast<float*>(c.take(n * sizeof(float))); };
        m->P = floats(NP);
        m->M = floats(NP);
        m->V = floats(NP);
        m->grad = floats(NP);
        m->sum = floats(1);
        m->X = floats(NI * rows);
        m->Y = floats(NO * rows);
        m->io = floats(NO * rows);
        m->partials = floats(NPL * max_rows);
        return c.used;
    };
    const bool ok = cudaMalloc(&m->dev, cut({nullptr, 0})) == cudaSuccess &&
                    (m->pinned = lbm::pinned_get(io_bytes(m))).p != nullptr;
    m->h_io = static_cast<float*>(m->pinned.p);
    cut({ok ? static_cast<char*>(m->dev) : nullptr, 0});
    if (!ok) {
        cudaGetLastError();
        lbm_mlp_destroy(m);
        return LBM_ENOMEM;
    }
    if (!prepare_kernels(&m->cluster)) {
        lbm_mlp_destroy(m);
        return LBM_ECUDA;
    }
    // Glorot-uniform weights from a seeded splitmix64 stream, zero biases
    std::vector<float> p(NP, 0.0f);
    uint64_t s = seed;
    auto fill = [&](int off, int rows, int cols) {
        const double a = std::sqrt(6.0 / (rows + cols));
        for (int i = 0; i < rows * cols; ++i) p[off + i] = static_cast<float>((2.0 * uniform01(s) - 1.0) * a);
    };
    fill(OFF_W1, NH, NI);
    fill(OFF_W2, NH, NH);
    fill(OFF_W3, NO, NH);
    for (int c = 0; c < NI; ++c) { m->norm.in_mean[c] = 0.0f; m->norm.in_std[c] = 1.0f; }
    for (int k = 0; k < NO; ++k) { m->norm.out_mean[k] = 0.0f; m->norm.out_std[k] = 1.0f; }
    int rc = lbm_mlp_set_params(m, p.data());
    if (rc) {
        lbm_mlp_destroy(m);
        return rc;
    }
    *out = m;
    return LBM_OK;
}

void lbm_mlp_destroy(lbm_mlp* m) {
    if (!m) return;
    if (m->P) cudaStreamSynchronize(m->st);   // also: nothing uses the pinned memory any more
    if (m->dev) cudaFree(m->dev);
    if (m->stage) cudaFreeHost(m->stage);
    lbm::pinned_put(m->pinned);
    for (cudaEvent_t e : m->done)
        if (e) cudaEventDestroy(e);
    delete m;
}

int lbm_mlp_set_normalization(lbm_mlp* m, const float in_mean[3], const float in_std[3], const float out_mean[4],
                              const float out_std[4]) {
    if (!valid(m) || !in_mean || !in_std || !out_mean || !out_std) return LBM_EINVAL;
    for (int c = 0; c < NI; ++c)
        if (!(in_std[c] > 0.0f) || !std::isfinite(in_mean[c])) return LBM_EINVAL;
    for (int k = 0; k < NO; ++k)
        if (!(out_std[k] > 0.0f) || !std::isfinite(out_mean[k])) return LBM_EINVAL;
    std::memcpy(m->norm.in_mean, in_mean, sizeof m->norm.in_mean);
    std::memcpy(m->norm.in_std, in_std, sizeof m->norm.in_std);
    std::memcpy(m->norm.out_mean, out_mean, sizeof m->norm.out_mean);
    std::memcpy(m->norm.out_std, out_std, sizeof m->norm.out_std);
    return LBM_OK;
}

int lbm_mlp_set_params(lbm_mlp* m, const float* params) {
    if (!valid(m) || !params) return LBM_EINVAL;
    std::memcpy(m->h_io, params, NP * sizeof(float));
    k_set_params<<<(NP + kT - 1) / kT, kT, 0, m->st>>>(m->h_io, m->P, m->M, m->V);
    if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(m->st) != cudaSuccess) return LBM_ECUDA;
    m->adam_t = 0;
    return LBM_OK;
}

int lbm_mlp_get_params(lbm_mlp* m, float* params) {
    if (!valid(m) || !params) return LBM_EINVAL;
    if (cudaMemcpyAsync(params, m->P, NP * sizeof(float), cudaMemcpyDeviceToHost, m->st) != cudaSuccess ||
        cudaStreamSynchronize(m->st) != cudaSuccess)
        return LBM_ECUDA;
    return LBM_OK;
}

int lbm_mlp_loss_grad(lbm_mlp* m, const float* X, const float* Y, int n, float* loss, float* grad) {
    if (!valid(m) || !X || !Y || n < 1 || n > m->max_n) return LBM_EINVAL;
    int rc = standardise_upload(m, X, Y, n);
    if (rc) return rc;
    if (grad_pass(m, nullptr, 0, n, false, 0, 0, 0, 0, make_float2(1, 1), m->sum) != cudaSuccess) return LBM_ECUDA;
    if (loss && cudaMemcpyAsync(loss, m->sum, sizeof(float), cudaMemcpyDeviceToHost, m->st) != cudaSuccess)
        return LBM_ECUDA;
    if (grad && cudaMemcpyAsync(grad, m->grad, NP * sizeof(float), cudaMemcpyDeviceToHost, m->st) != cudaSuccess)
        return LBM_ECUDA;
    return cudaStreamSynchronize(m->st) == cudaSuccess ? LBM_OK : LBM_ECUDA;
}

int lbm_mlp_adam_step(lbm_mlp* m, const float* X, const float* Y, int n, float lr, float beta1, float beta2,
                      float eps) {
    if (!valid(m) || !X || !Y || n < 1 || n > m->max_n || !(lr > 0)) return LBM_EINVAL;
    int rc = standardise_upload(m, X, Y, n);
    if (rc) return rc;
    if (grad_pass(m, nullptr, 0, n, true, lr, beta1, beta2, eps, next_corr(m, beta1, beta2), m->sum) != cudaSuccess)
        return LBM_ECUDA;
    return cudaStreamSynchronize(m->st) == cudaSuccess ? LBM_OK : LBM_ECUDA;
}

int lbm_mlp_train(lbm_mlp* m, const float* X, const float* Y, int n, int epochs, int batch, float lr,
                  unsigned long long seed, float* loss_per_epoch) {
    if (!valid(m) || !X || !Y || n < 1 || n > m->max_n || epochs < 1 || batch < 1 || !(lr > 0)) return LBM_EINVAL;
    int rc = ensure_stage(m);
    if (!rc) rc = standardise_upload(m, X, Y, n);
    if (rc) return rc;
    std::vector<int> order(n);
    for (int i = 0; i < n; ++i) order[i] = i;
    uint64_t s = seed;
    batch = std::min(batch, n);   // a larger batch is the whole set
    const int nb = (n + batch - 1) / batch, most = m->cap / n;   // epochs the buffers hold
    constexpr float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    // launches of one epoch, then two, four, ... : the host shuffles the
    // next launch's epochs while the one before runs, and only the first
    // epoch's shuffle is waited for
    int pending[2] = {0, 0}, at[2] = {0, 0};   // epochs in flight in each set of buffers, and the first of them
    auto collect = [&](int k) -> int {
        if (!pending[k]) return LBM_OK;
        if (cudaEventSynchronize(m->done[k]) != cudaSuccess) return LBM_ECUDA;
        for (int e = 0; e < pending[k] && loss_per_epoch; ++e) {
            double acc = 0;
            for (int b = 0; b < nb; ++b) acc += m->loss[k][e * nb + b];
            loss_per_epoch[at[k] + e] = static_cast<float>(acc / nb);
        }
        pending[k] = 0;
        return LBM_OK;
    };
    auto run = [&]() -> int {
        for (int e0 = 0, k = 0, len = 1; e0 < epochs; e0 += len, k ^= 1, len = std::min(2 * len, most)) {
            len = std::min(len, epochs - e0);
            int r = collect(k);
            if (r) return r;
            for (int e = 0; e < len; ++e) {
                for (int i = n - 1; i > 0; --i) {   // Fisher-Yates with splitmix64
                    const int j = static_cast<int>(splitmix(s) % static_cast<uint64_t>(i + 1));
                    std::swap(order[i], order[j]);
                }
                std::memcpy(m->order[k] + static_cast<size_t>(e) * n, order.data(), n * sizeof(int));
                for (int b = 0; b < nb; ++b) m->corr[k][e * nb + b] = next_corr(m, b1, b2);
            }
            if (m->cluster && batch <= kClusterMax) {
                const TrainArgs a = {m->P, m->M, m->V, m->X, m->Y, m->order[k], m->corr[k], m->loss[k], n,
                                     batch, len, lr, b1, b2, eps};
                if (launch_train(m, a) != cudaSuccess) return LBM_ECUDA;
            } else {
                for (int q = 0; q < len * nb; ++q) {
                    const int first = (q % nb) * batch;
                    if (grad_pass(m, m->order[k] + static_cast<size_t>(q / nb) * n, first, std::min(batch, n - first),
                                  true, lr, b1, b2, eps, m->corr[k][q], m->loss[k] + q) != cudaSuccess)
                        return LBM_ECUDA;
                }
            }
            if (cudaEventRecord(m->done[k], m->st) != cudaSuccess) return LBM_ECUDA;
            pending[k] = len;
            at[k] = e0;
        }
        const int r = collect(0);
        return r ? r : collect(1);
    };
    rc = run();
    if (cudaStreamSynchronize(m->st) != cudaSuccess && !rc) rc = LBM_ECUDA;
    return rc;
}

int lbm_mlp_predict(lbm_mlp* m, const float* X, int n, float* Y) {
    if (!valid(m) || !X || !Y || n < 1 || n > m->max_n) return LBM_EINVAL;
    // the kernel reads and writes pinned host memory where the samples fit it:
    // two copies fewer to enqueue and to wait for
    const bool near = n <= m->io_n;
    const size_t in = static_cast<size_t>(n) * NI, out = static_cast<size_t>(n) * NO;
    float *x = near ? m->h_io : m->X, *y = near ? m->h_io + in : m->io;
    if (near) std::memcpy(x, X, in * sizeof(float));
    else if (cudaMemcpyAsync(x, X, in * sizeof(float), cudaMemcpyHostToDevice, m->st) != cudaSuccess) return LBM_ECUDA;
    k_predict<<<std::min((n + kS - 1) / kS, 2 * kRows), kT, sizeof(GradSmem), m->st>>>(m->P, m->norm, x, n, y);
    if (cudaGetLastError() != cudaSuccess) return LBM_ECUDA;
    if (!near && cudaMemcpyAsync(Y, y, out * sizeof(float), cudaMemcpyDeviceToHost, m->st) != cudaSuccess)
        return LBM_ECUDA;
    if (cudaStreamSynchronize(m->st) != cudaSuccess) return LBM_ECUDA;
    if (near) std::memcpy(Y, y, out * sizeof(float));
    return LBM_OK;
}

int lbm_mlp_invert_kappa(lbm_mlp* m, const float* t_over_tc, const float* A, const float* sigma, int count,
                         float kappa_lo, float kappa_hi, float* kappa_out) {
    if (!valid(m) || !t_over_tc || !A || !sigma || !kappa_out || count < 1 || count > m->max_n ||
        !(kappa_lo < kappa_hi))
        return LBM_EINVAL;
    // inputs as three columns t, A, sigma, kappas behind them (as in lbm_mlp_predict)
    const bool near = count <= m->io_n;
    const size_t bytes = static_cast<size_t>(count) * sizeof(float);
    float *x = near ? m->h_io : m->X, *y = near ? m->h_io + static_cast<size_t>(count) * 3 : m->io;
    const float* const cols[3] = {t_over_tc, A, sigma};
    for (int c = 0; c < 3; ++c) {
        float* const to = x + static_cast<size_t>(c) * count;
        if (near) std::memcpy(to, cols[c], bytes);
        else if (cudaMemcpyAsync(to, cols[c], bytes, cudaMemcpyHostToDevice, m->st) != cudaSuccess) return LBM_ECUDA;
    }
    // as many halvings per pass as keep every target on a CTA that is
    // resident (16 targets: 31 us, 767 as one thread per target; 304 / 608 /
    // 1216 / 8192 targets: 38 / 44 / 54 / 233 us)
    auto invert = [&](auto fn, int targets) {
        fn<<<(count + targets - 1) / targets, kT, sizeof(GradSmem), m->st>>>(
            m->P, m->norm, x, x + count, x + 2 * static_cast<size_t>(count), count, kappa_lo, kappa_hi, y);
    };
    if (count <= kRows) invert(k_invert<3>, 1);
    else if (count <= 2 * kRows) invert(k_invert<2>, 2);
    else invert(k_invert<1>, 8);
    if (cudaGetLastError() != cudaSuccess) return LBM_ECUDA;
    if (!near && cudaMemcpyAsync(kappa_out, y, bytes, cudaMemcpyDeviceToHost, m->st) != cudaSuccess) return LBM_ECUDA;
    if (cudaStreamSynchronize(m->st) != cudaSuccess) return LBM_ECUDA;
    if (near) std::memcpy(kappa_out, y, bytes);
    return LBM_OK;
}

}  // extern "C"
