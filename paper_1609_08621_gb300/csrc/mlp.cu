// Learned opening criterion: training (FP32), inference (BF16 tensor cores) and the audit that
// produces training labels from the plain method's own force errors.  Not in the paper, whose
// criterion is the fixed-theta test of Sec. 3.1; see mlp.cuh for the network.
#include <math.h>

#include <algorithm>

#include "expansions.cuh"
#include "fmm_internal.cuh"
#include "mlp.cuh"

// ---------------------------------------------------------------- packing for inference

__global__ void k_mlp_pack(const float* __restrict__ p, unsigned char* __restrict__ out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    __nv_bfloat16* w1 = reinterpret_cast<__nv_bfloat16*>(out + MLPP_W1);
    __nv_bfloat16* w2 = reinterpret_cast<__nv_bfloat16*>(out + MLPP_W2);
    __nv_bfloat16* w3 = reinterpret_cast<__nv_bfloat16*>(out + MLPP_W3);
    __nv_bfloat16* w4 = reinterpret_cast<__nv_bfloat16*>(out + MLPP_W4);
    if (i < 64 * 24) {
        const int r = i / 24, c = i % 24;
        w1[i] = __float2bfloat16_rn(c < MLP_F ? p[MLP_W1 + r * MLP_F + c] : 0.0f);
    }
    if (i < 64 * 72) {
        const int r = i / 72, c = i % 72;
        w2[i] = __float2bfloat16_rn(c < MLP_H ? p[MLP_W2 + r * MLP_H + c] : 0.0f);
        w3[i] = __float2bfloat16_rn(c < MLP_H ? p[MLP_W3 + r * MLP_H + c] : 0.0f);
    }
    if (i < 8 * 72) {
        const int r = i / 72, c = i % 72;
        w4[i] = __float2bfloat16_rn(r == 0 && c < MLP_H ? p[MLP_W4 + c] : 0.0f);
    }
    if (i < MLP_H) {
        reinterpret_cast<float*>(out + MLPP_B1)[i] = p[MLP_B1 + i];
        reinterpret_cast<float*>(out + MLPP_B2)[i] = p[MLP_B2 + i];
        reinterpret_cast<float*>(out + MLPP_B3)[i] = p[MLP_B3 + i];
    }
    if (i < 4) reinterpret_cast<float*>(out + MLPP_B4)[i] = i == 0 ? p[MLP_B4] : 0.0f;
    if (i < MLP_F) {
        reinterpret_cast<float*>(out + MLPP_MEAN)[i] = p[MLP_MEAN + i];
        reinterpret_cast<float*>(out + MLPP_ISTD)[i] = p[MLP_ISTD + i];
    }
    if (i < MLP_NSUR) reinterpret_cast<float*>(out + MLPP_SUR)[i] = p[MLP_SUR + i];
}

cudaError_t fmm_mlp_pack(const float* params, unsigned char* packed, cudaStream_t s)
{
    k_mlp_pack<<<(64 * 72 + 255) / 256, 256, 0, s>>>(params, packed);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- training (FP32)

// Gradient of 0.5 * mean((y - label)^2) over a minibatch.  A block takes tiles of 64 rows and keeps its
// weight gradients in registers over them; its sums go to a slot of its own, and k_mlp_step adds the
// slots in order, so the weights of a training run are a function of its inputs (atomics gave each run another
// order of arrival from three blocks on, and training turns a rounding into 1e-5 to 6e-3 of the weights).  (The loss is summed row by row
// with atomics.)
//
// The six products of a tile (two hidden layers forward, their deltas, their weight gradients) are
// 64 wide and run from shared memory: 2 rows x 4 units per thread forward and for the deltas, 2 x 4
// weights per thread for the gradients, operands as float4 (6 loads for 32 multiply-adds, 2 for 8).
// Both hidden matrices lie there twice, as stored and transposed, so that either product reads along
// its output.  FP32 throughout, every sum in the order of its index.  Bound by its shared-memory loads
// and the chain of layers: a minibatch of 4096 rows is 64 blocks of one tile.  One thread per hidden
// unit, two warps a block, with the weights read from global memory and the gradients added with
// atomics took 252 us for it.
#define GR_ROWS 64
#define GR_THREADS 512
#define GR_PAD 68  // row stride of the activations and weights in shared memory
struct GradSmem {
    float W2t[MLP_H * GR_PAD], W3t[MLP_H * GR_PAD];  // [k][j], forward
    float W2[MLP_H * GR_PAD], W3[MLP_H * GR_PAD];    // [i][j], deltas
    float W1t[MLP_F * GR_PAD];
    float H1[GR_ROWS * GR_PAD], H2[GR_ROWS * GR_PAD], H3[GR_ROWS * GR_PAD];
    float Da[GR_ROWS * GR_PAD], Db[GR_ROWS * GR_PAD];
    float X[GR_ROWS * MLP_F];
    float b1[MLP_H], b2[MLP_H], b3[MLP_H], zero[MLP_H], w4[MLP_H];
    float dy[GR_ROWS];
};

// out[s][j] = f(b[j] + sum_k in[s][k] Wt[k][j]), f the ReLU, or (MASK) zero where mask[s][j] is not > 0
template <int K, int KSTRIDE, bool MASK>
__device__ __forceinline__ void grad_layer(const float* __restrict__ in, const float* __restrict__ Wt,
                                           const float* __restrict__ b, const float* __restrict__ mask,
                                           float* __restrict__ out, int tid)
{
    const int r0 = (tid >> 4) * 2, j0 = (tid & 15) * 4;
    const float4 bv = *reinterpret_cast<const float4*>(b + j0);
    float4 z0 = bv, z1 = bv;
#pragma unroll 4
    for (int k = 0; k < K; k += 4) {
        const float4 h0 = *reinterpret_cast<const float4*>(in + r0 * KSTRIDE + k);
        const float4 h1 = *reinterpret_cast<const float4*>(in + (r0 + 1) * KSTRIDE + k);
        const float a0[4] = {h0.x, h0.y, h0.z, h0.w}, a1[4] = {h1.x, h1.y, h1.z, h1.w};
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const float4 w = *reinterpret_cast<const float4*>(Wt + (k + q) * GR_PAD + j0);
            z0.x = fmaf(w.x, a0[q], z0.x);
            z0.y = fmaf(w.y, a0[q], z0.y);
            z0.z = fmaf(w.z, a0[q], z0.z);
            z0.w = fmaf(w.w, a0[q], z0.w);
            z1.x = fmaf(w.x, a1[q], z1.x);
            z1.y = fmaf(w.y, a1[q], z1.y);
            z1.z = fmaf(w.z, a1[q], z1.z);
            z1.w = fmaf(w.w, a1[q], z1.w);
        }
    }
#pragma unroll
    for (int h = 0; h < 2; h++) {
        float4 z = h ? z1 : z0;
        float* const o = out + (r0 + h) * GR_PAD + j0;
        if (MASK) {
            const float4 m = *reinterpret_cast<const float4*>(mask + (r0 + h) * GR_PAD + j0);
            z = make_float4(m.x > 0.0f ? z.x : 0.0f, m.y > 0.0f ? z.y : 0.0f, m.z > 0.0f ? z.z : 0.0f,
                            m.w > 0.0f ? z.w : 0.0f);
        } else {
            z = make_float4(fmaxf(z.x, 0.0f), fmaxf(z.y, 0.0f), fmaxf(z.z, 0.0f), fmaxf(z.w, 0.0f));
        }
        *reinterpret_cast<float4*>(o) = z;
    }
}

// g[a][c] += sum_s D[s][j0 + a] H[s][k0 + c]
__device__ __forceinline__ void grad_weights(const float* __restrict__ D, const float* __restrict__ H, float g[2][4],
                                             int tid)
{
    const int j0 = (tid >> 4) * 2, k0 = (tid & 15) * 4;
#pragma unroll 4
    for (int s = 0; s < GR_ROWS; s++) {
        const float2 d = *reinterpret_cast<const float2*>(D + s * GR_PAD + j0);
        const float4 h = *reinterpret_cast<const float4*>(H + s * GR_PAD + k0);
        const float dv[2] = {d.x, d.y};
#pragma unroll
        for (int a = 0; a < 2; a++) {
            g[a][0] = fmaf(dv[a], h.x, g[a][0]);
            g[a][1] = fmaf(dv[a], h.y, g[a][1]);
            g[a][2] = fmaf(dv[a], h.z, g[a][2]);
            g[a][3] = fmaf(dv[a], h.w, g[a][3]);
        }
    }
}

__global__ void __launch_bounds__(GR_THREADS) k_mlp_grad(const float* __restrict__ p, const float* __restrict__ feats,
                                                         const float* __restrict__ labels,
                                                         const unsigned int* __restrict__ idx, long long nrows,
                                                         float inv_b, float loss_scale, float* __restrict__ part,
                                                         float* __restrict__ loss)
{
    extern __shared__ __align__(16) unsigned char gsm[];
    GradSmem& S = *reinterpret_cast<GradSmem*>(gsm);
    const int tid = threadIdx.x;
    for (int i = tid; i < MLP_H * MLP_H; i += GR_THREADS) {
        const int j = i >> 6, k = i & 63;
        const float w2 = p[MLP_W2 + i], w3 = p[MLP_W3 + i];
        S.W2[j * GR_PAD + k] = w2;
        S.W2t[k * GR_PAD + j] = w2;
        S.W3[j * GR_PAD + k] = w3;
        S.W3t[k * GR_PAD + j] = w3;
    }
    for (int i = tid; i < MLP_H * MLP_F; i += GR_THREADS) S.W1t[(i & 7) * GR_PAD + (i >> 3)] = p[MLP_W1 + i];
    if (tid < MLP_H) {
        S.b1[tid] = p[MLP_B1 + tid];
        S.b2[tid] = p[MLP_B2 + tid];
        S.b3[tid] = p[MLP_B3 + tid];
        S.w4[tid] = p[MLP_W4 + tid];
        S.zero[tid] = 0.0f;
    }
    // this thread's gradients: 2 x 4 of each hidden matrix, one of the first, one of the four vectors
    float g2[2][4] = {}, g3[2][4] = {}, g1 = 0.0f, gv = 0.0f, gb4 = 0.0f;
    const int vj = tid & 63, vq = tid >> 6;  // vector gradient: b1, b2, b3, w4 of unit vj
    const long long tiles = fmm_ceil_div(nrows, GR_ROWS);
    for (long long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const long long r0 = tile * GR_ROWS;
        const int nr = (int)min((long long)GR_ROWS, nrows - r0);
        __syncthreads();
        {
            const int s = tid >> 3, k = tid & 7;  // one feature per thread
            float x = 0.0f;
            if (s < nr) {
                const unsigned int r = idx ? idx[r0 + s] : (unsigned int)(r0 + s);
                x = (feats[(long long)r * MLP_F + k] - p[MLP_MEAN + k]) * p[MLP_ISTD + k];
                if (k == 0) S.dy[s] = labels[r];
            }
            S.X[s * MLP_F + k] = x;
        }
        __syncthreads();
        grad_layer<MLP_F, MLP_F, false>(S.X, S.W1t, S.b1, nullptr, S.H1, tid);
        __syncthreads();
        grad_layer<MLP_H, GR_PAD, false>(S.H1, S.W2t, S.b2, nullptr, S.H2, tid);
        __syncthreads();
        grad_layer<MLP_H, GR_PAD, false>(S.H2, S.W3t, S.b3, nullptr, S.H3, tid);
        __syncthreads();
        if (tid < GR_ROWS) {
            // output and its error, a row per lane, summed in the order of the units
            float y = p[MLP_B4];
#pragma unroll 8
            for (int k = 0; k < MLP_H; k += 4) {
                const float4 w = *reinterpret_cast<const float4*>(S.w4 + k);
                const float4 h = *reinterpret_cast<const float4*>(S.H3 + tid * GR_PAD + k);
                y = fmaf(w.w, h.w, fmaf(w.z, h.z, fmaf(w.y, h.y, fmaf(w.x, h.x, y))));
            }
            const float r = tid < nr ? y - S.dy[tid] : 0.0f;
            if (tid < nr) atomicAdd(loss, 0.5f * r * r * loss_scale);
            S.dy[tid] = r * inv_b;
        }
        __syncthreads();
        // delta of layer 3
        for (int i = tid; i < GR_ROWS * MLP_H; i += GR_THREADS) {
            const int s = i >> 6, j = i & 63;
            S.Da[s * GR_PAD + j] = S.H3[s * GR_PAD + j] > 0.0f ? S.dy[s] * S.w4[j] : 0.0f;
        }
        __syncthreads();
        if (vq == 3) {
            for (int s = 0; s < GR_ROWS; s++) gv = fmaf(S.H3[s * GR_PAD + vj], S.dy[s], gv);
            if (vj == 0)
                for (int s = 0; s < GR_ROWS; s++) gb4 += S.dy[s];
        } else if (vq == 2) {
            for (int s = 0; s < GR_ROWS; s++) gv += S.Da[s * GR_PAD + vj];
        }
        grad_weights(S.Da, S.H2, g3, tid);
        grad_layer<MLP_H, GR_PAD, true>(S.Da, S.W3, S.zero, S.H2, S.Db, tid);
        __syncthreads();
        if (vq == 1)
            for (int s = 0; s < GR_ROWS; s++) gv += S.Db[s * GR_PAD + vj];
        grad_weights(S.Db, S.H1, g2, tid);
        grad_layer<MLP_H, GR_PAD, true>(S.Db, S.W2, S.zero, S.H1, S.Da, tid);
        __syncthreads();
        if (vq == 0)
            for (int s = 0; s < GR_ROWS; s++) gv += S.Da[s * GR_PAD + vj];
        {
            const int j = tid >> 3, k = tid & 7;
            for (int s = 0; s < GR_ROWS; s++) g1 = fmaf(S.Da[s * GR_PAD + j], S.X[s * MLP_F + k], g1);
        }
    }
    // the block's sums in its slot, in the order of the parameters, then its loss
    float* const out = part + (long long)blockIdx.x * MLP_PART;
    {
        const int j0 = (tid >> 4) * 2, k0 = (tid & 15) * 4;
#pragma unroll
        for (int a = 0; a < 2; a++)
#pragma unroll
            for (int c = 0; c < 4; c++) {
                out[MLP_W2 + (j0 + a) * MLP_H + k0 + c] = g2[a][c];
                out[MLP_W3 + (j0 + a) * MLP_H + k0 + c] = g3[a][c];
            }
        out[MLP_W1 + tid] = g1;
        if (vq < 4) out[(vq == 0 ? MLP_B1 : vq == 1 ? MLP_B2 : vq == 2 ? MLP_B3 : MLP_W4) + vj] = gv;
        if (tid == 3 * 64) out[MLP_B4] = gb4;
    }
}

// Adds the blocks' sums in order, each addition rounded to FP32: the gradient, written to grad, or taken at once by an
// Adam step on the trainable weights (bias-corrected moments).
struct AdamArgs {
    float *p, *m, *v;
    float lr, b1, b2, eps, c1, c2;
};
template <bool ADAM>
__global__ void __launch_bounds__(64) k_mlp_step(const float* __restrict__ part, int nb, float* __restrict__ grad,
                                                 AdamArgs a)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= MLP_NW) return;
    float gi = 0.0f;
#pragma unroll 16
    for (int b = 0; b < nb; b++) gi += part[(long long)b * MLP_PART + i];
    if (!ADAM) {
        grad[i] = gi;
        return;
    }
    const float mi = a.b1 * a.m[i] + (1.0f - a.b1) * gi;
    const float vi = a.b2 * a.v[i] + (1.0f - a.b2) * gi * gi;
    a.m[i] = mi;
    a.v[i] = vi;
    a.p[i] -= a.lr * (mi / a.c1) / (sqrtf(vi / a.c2) + a.eps);
}

static cudaError_t launch_grad(const float* params, const float* feats, const float* labels, const unsigned int* idx,
                               long long nrows, float inv_b, float loss_scale, float* part, float* loss, int* nb,
                               cudaStream_t s)
{
    static std::atomic<unsigned long long> attr{0};
    cudaError_t e = fmm_smem_attr_once(k_mlp_grad, (int)sizeof(GradSmem), attr);
    if (e != cudaSuccess) return e;
    *nb = (int)std::min<long long>(fmm_ceil_div(nrows, GR_ROWS), MLP_GRAD_BLOCKS);
    k_mlp_grad<<<*nb, GR_THREADS, sizeof(GradSmem), s>>>(params, feats, labels, idx, nrows, inv_b, loss_scale, part,
                                                              loss);
    return cudaGetLastError();
}

// grad (MLP_NW values) of the rows, and their loss added to *loss; part: MLP_GRAD_BLOCKS * MLP_PART floats
cudaError_t fmm_mlp_grad(const float* params, const float* feats, const float* labels, const unsigned int* idx,
                         long long nrows, float inv_b, float loss_scale, float* part, float* grad, float* loss,
                         cudaStream_t s)
{
    int nb = 0;
    cudaError_t e = launch_grad(params, feats, labels, idx, nrows, inv_b, loss_scale, part, loss, &nb, s);
    if (e != cudaSuccess) return e;
    k_mlp_step<false><<<(MLP_NW + 63) / 64, 64, 0, s>>>(part, nb, grad, AdamArgs{});
    return cudaGetLastError();
}

// one Adam step on the rows' gradient; their loss is added to *loss
cudaError_t fmm_mlp_adam(float* p, const float* feats, const float* labels, const unsigned int* idx, long long nrows,
                         float inv_b, float loss_scale, float* part, float* m, float* v, float lr, int step, float* loss,
                         cudaStream_t s)
{
    int nb = 0;
    cudaError_t e = launch_grad(p, feats, labels, idx, nrows, inv_b, loss_scale, part, loss, &nb, s);
    if (e != cudaSuccess) return e;
    AdamArgs a;
    a.p = p;
    a.m = m;
    a.v = v;
    a.lr = lr;
    a.b1 = 0.9f;
    a.b2 = 0.999f;
    a.eps = 1e-8f;
    a.c1 = 1.0f - powf(a.b1, (float)step);
    a.c2 = 1.0f - powf(a.b2, (float)step);
    k_mlp_step<true><<<(MLP_NW + 63) / 64, 64, 0, s>>>(part, nb, nullptr, a);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- inference (tensor cores)

__global__ void __launch_bounds__(128) k_mlp_predict(const unsigned char* __restrict__ packed,
                                                     const float* __restrict__ feats, long long n,
                                                     float* __restrict__ out)
{
    extern __shared__ __align__(16) unsigned char msm[];
    unsigned char* W = msm;
    unsigned char* scratch = msm + MLPP_SIZE + (threadIdx.x >> 5) * MLP_WARP_SCRATCH;
    mlp_load_smem(packed, W);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long base = gw * 32; base < n; base += nw * 32) {
        const long long r = base + lane;
        float f[MLP_F];
#pragma unroll
        for (int k = 0; k < MLP_F; k++) f[k] = r < n ? feats[r * MLP_F + k] : 0.0f;
        const float y = mlp_predict_warp(W, scratch, f, lane, __ballot_sync(FMM_FULL_MASK, r < n));
        if (r < n) out[r] = y;
    }
}

size_t fmm_mlp_predict_smem(int warps) { return MLPP_SIZE + (size_t)warps * MLP_WARP_SCRATCH; }

cudaError_t fmm_mlp_predict(const unsigned char* packed, const float* feats, long long n, float* out, cudaStream_t s)
{
    static std::atomic<unsigned long long> attr{0};
    cudaError_t e = fmm_smem_attr_once(k_mlp_predict, (int)fmm_mlp_predict_smem(4), attr);
    if (e != cudaSuccess) return e;
    long long blocks = fmm_ceil_div(n, 128);
    if (blocks > 152LL * 16) blocks = 152LL * 16;
    if (blocks < 1) blocks = 1;
    k_mlp_predict<<<(unsigned)blocks, 128, fmm_mlp_predict_smem(4), s>>>(packed, feats, n, out);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- audit labels

// For every recorded (sink k, source s) pair: the 8 features and the label log10 of the largest
// relative force error, over up to 32 sink particles i of k, of accepting s for k as a
// cell-cell interaction (M2L about k's centre, then L2P at i) instead of summing s's particles
// directly: |a_expansion - a_direct| / |a_ref_i|, a_ref the particle's total acceleration from a
// reference solve.  One warp per pair, one sampled sink particle per lane.
__global__ void __launch_bounds__(128) k_audit_labels(
    const int2* __restrict__ pairs, long long npairs, const int* __restrict__ cfirst, const int* __restrict__ ccount,
    const Com4* __restrict__ com, const float* __restrict__ rec, const float4* __restrict__ mnorm,
    const float* __restrict__ amin,
    const WalkNode* __restrict__ node, const int* __restrict__ bucket_of, const int* __restrict__ bucket_cell,
    const float4* __restrict__ off, const unsigned int* __restrict__ perm, const float* __restrict__ acc_ref,
    long long n, float eps, float* __restrict__ feats, float* __restrict__ labels)
{
    const int lane = threadIdx.x & 31;
    const long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    const float eps2 = eps * eps;
    for (long long q = gw; q < npairs; q += nw) {
        const int k = pairs[q].x, s = pairs[q].y;
        const Com4 ck = com[k], cs = com[s];
        const int fk = cfirst[k], nk = ccount[k], fs = cfirst[s], ns = ccount[s];
        // local expansion of s about k's centre
        float L[FMM_NL];
#pragma unroll
        for (int i = 0; i < FMM_NL; i++) L[i] = 0.0f;
        {
            float M[FMM_NMOM];
            const float4* r4 = reinterpret_cast<const float4*>(rec + (long long)s * FMM_NREC);
#pragma unroll
            for (int i = 0; i < FMM_NMOM / 4; i++) {
                const float4 v = r4[i];
                M[4 * i] = v.x;
                M[4 * i + 1] = v.y;
                M[4 * i + 2] = v.z;
                M[4 * i + 3] = v.w;
            }
            fmm_m2l_acc(M, __double2float_rn(ck.x - cs.x), __double2float_rn(ck.y - cs.y),
                        __double2float_rn(ck.z - cs.z), eps2, L);
        }
        float err = 0.0f;
        const int ns_sample = nk < 32 ? nk : 32;
        if (lane < ns_sample) {
            const int i = fk + (int)(((long long)lane * nk) / ns_sample);
            const Com4 cb = com[bucket_cell[bucket_of[i]]];
            const float4 oi = off[i];
            const float ux = __double2float_rn(cb.x - ck.x) + oi.x, uy = __double2float_rn(cb.y - ck.y) + oi.y,
                        uz = __double2float_rn(cb.z - ck.z) + oi.z;
            float ax = 0.f, ay = 0.f, az = 0.f, ph = 0.f;
            fmm_l2p_acc(L, ux, uy, uz, ax, ay, az, ph);
            float ex = 0.f, ey = 0.f, ez = 0.f;
            int b = -1;
            float bx = 0.f, by = 0.f, bz = 0.f;
            for (int j = fs; j < fs + ns; j++) {
                const int bj = bucket_of[j];
                if (bj != b) {
                    b = bj;
                    const Com4 cj = com[bucket_cell[bj]];
                    bx = __double2float_rn(cj.x - ck.x);
                    by = __double2float_rn(cj.y - ck.y);
                    bz = __double2float_rn(cj.z - ck.z);
                }
                const float4 o = off[j];
                const float dx = bx + o.x - ux, dy = by + o.y - uy, dz = bz + o.z - uz;
                const float ir = rsqrtf(fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, eps2))));
                const float w = o.w * ir * ir * ir;
                ex = fmaf(w, dx, ex);
                ey = fmaf(w, dy, ey);
                ez = fmaf(w, dz, ez);
            }
            const unsigned int pi = perm[i];
            const float rx = acc_ref[pi], ry = acc_ref[n + pi], rz = acc_ref[2 * n + pi];
            const float ref = sqrtf(rx * rx + ry * ry + rz * rz);
            const float dxe = ax - ex, dye = ay - ey, dze = az - ez;
            err = sqrtf(dxe * dxe + dye * dye + dze * dze) / fmaxf(ref, 1e-30f);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) err = fmaxf(err, __shfl_xor_sync(FMM_FULL_MASK, err, o));
        if (lane == 0) {
            labels[q] = log10f(err + 1e-12f);
            mlp_pair_features(node[k], node[s], mnorm[s], mlp_log_accel(amin[k]), eps, feats + q * MLP_F);
        }
    }
}

cudaError_t fmm_launch_audit_labels(DevTree& t, const int2* pairs, long long npairs, const float* acc_ref,
                                    long long n, float eps, float* feats, float* labels, cudaStream_t s)
{
    long long blocks = fmm_ceil_div(npairs, 4);
    if (blocks > 152LL * 32) blocks = 152LL * 32;
    if (blocks < 1) blocks = 1;
    k_audit_labels<<<(unsigned)blocks, 128, 0, s>>>(pairs, npairs, t.cfirst, t.ccount, t.com, t.rec, t.mnorm, t.amin, t.node,
                                                     t.bucket_of, t.bucket_cell, t.off, t.idx, acc_ref, n, eps, feats,
                                                     labels);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- sink acceleration scale

// Per cell, the smallest |a| of its particles from an acceleration estimate acc (3 x n SoA in
// input order, e.g. the previous step's forces): bucket cells scan their particles, and the
// second child to arrive at a parent takes the smaller of the two (arrive[] zeroed first).
__global__ void __launch_bounds__(128) k_cell_amin(const unsigned int* __restrict__ nbucket,
                                                   const int* __restrict__ bucket_cell,
                                                   const int* __restrict__ cfirst, const int* __restrict__ ccount,
                                                   const int* __restrict__ cparent, const int* __restrict__ cchild,
                                                   const unsigned int* __restrict__ perm,
                                                   const float* __restrict__ acc, long long n, float* amin,
                                                   unsigned int* arrive)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= (int)*nbucket) return;
    const int c = bucket_cell[b];
    float a = INFINITY;
    for (int j = cfirst[c], e = cfirst[c] + ccount[c]; j < e; j++) {
        const unsigned int p = perm[j];
        const float x = acc[p], y = acc[n + p], z = acc[2 * n + p];
        a = fminf(a, sqrtf(x * x + y * y + z * z));
    }
    amin[c] = a;
    int p = cparent[c];
    while (p >= 0) {
        __threadfence();
        if (atomicAdd(&arrive[p], 1u) == 0u) return;
        __threadfence();
        amin[p] = fminf(__ldcg(&amin[cchild[2 * p]]), __ldcg(&amin[cchild[2 * p + 1]]));
        p = cparent[p];
    }
}

cudaError_t fmm_launch_cell_amin(DevTree& t, const float* acc, long long n, cudaStream_t s)
{
    const long long nb = t.cap_grid ? t.cap_cells : t.n_buckets, nc = t.cap_grid ? t.cap_cells : t.n_cells;
    cudaError_t e = cudaMemsetAsync(t.arrive, 0, sizeof(unsigned int) * (size_t)nc, s);
    if (e != cudaSuccess) return e;
    k_cell_amin<<<(unsigned)fmm_ceil_div(nb, 128), 128, 0, s>>>(t.dcount + 1, t.bucket_cell, t.cfirst, t.ccount,
                                                                 t.cparent, t.cchild, t.idx, acc, n, t.amin, t.arrive);
    return cudaGetLastError();
}
