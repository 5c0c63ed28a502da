// Batched K-cycle (Sec. 2.3, "Summary"; Table kcycle): nrhs right-hand sides
// that share one hierarchy (one gauge field) are solved together.
//
// Every vector of the one-vector solver becomes a block of nrhs vectors stored
// back to back, and every Krylov scalar an array over the right-hand sides.
// Each launch covers all right-hand sides (grid.y, or grid.z where grid.y is
// the basis index); a right-hand side whose flag is set is skipped by every
// block of its row, so one fixed launch sequence serves any set of
// still-active systems and the coarse cycle stays a single CUDA graph.  The
// coarse operator on the nrhs * Ls_c columns is the tensor-core contraction
// (mg_coarse_tc.cu).  With one right-hand side it is the one-vector stencil:
// that is the path mg_solve takes with the GCR coarse solver on 2-d and 4-d
// lattices (4-d hierarchies take one right-hand side per call).  Per
// right-hand side the iteration is exactly the
// one-vector solver's: FP64 reliable updates of the true residual around
// FGCR(gcr_restart) in FP32, the wall restriction, coarse GCR to coarse_tol,
// prolongation and post_smooth GCR steps.
//
// Reductions: one row of partial sums and completion counters per right-hand
// side (and per basis vector for the Gram-Schmidt dots of vectors that fit in
// L2; larger vectors take all basis vectors in one pass over w), so the rows
// finish independently and each result is summed in a fixed order.
#include <algorithm>
#include <chrono>
#include <mutex>
#include <string.h>
#include <string>
#include <thread>
#include <vector>

#include "mg.cuh"

namespace dwf {
namespace {

constexpr int BK_MAX = 32;            // bound on the restart lengths
constexpr int BMDOT_BLOCKS = 608;     // partial slots per (right-hand side, basis vector) of a Gram-Schmidt dot
constexpr int BMDOT_ROW_BLOCKS = 152; // blocks per row of the per-row form
constexpr long long BMDOT_FUSE_N = 8LL << 20;   // complex values from which the fused form is used
constexpr int CROW = (RED_GROUPS + 1) * RED_CSTRIDE;   // unsigneds of completion counters per row
constexpr int PROW = RED_MAX * RED_BLOCKS;             // doubles of partial sums per row

// Krylov scalars of one right-hand side.  The GCR iterations keep only the
// orthogonalised images w_k = A p'_k and the residual up to date; the search
// directions are p'_k = p_k - sum_{j<k} C[k][j] p'_j of the stored raw
// directions p_k, so the solution update sum_k A[k] p'_k is assembled once per
// cycle as sum_j y_j p_j with (I + C)^T y = A (back substitution): every step
// then reads and writes the raw basis only once.
struct BGcr {
    double coef[BK_MAX][2];          // projection coefficients of the current pass
    double nrm[BK_MAX];              // |w_k|^2
    double alpha[2];                 // alpha of the current step
    double rr2;                      // |r|^2 after the current step
    double pad;
    double C[BK_MAX][BK_MAX][2];     // C[k][j], j < k: summed over the Gram-Schmidt passes of step k
    double A[BK_MAX][2];             // alpha of step k
};

__device__ __forceinline__ RedScratch row_scratch(RedScratch base, int r) {
    return RedScratch{base.partials + (size_t)r * PROW, base.counter + (size_t)r * CROW};
}

__device__ __forceinline__ void cdot4(const float4 a, const float4 b, float& re, float& im) {
    re += a.x * b.x + a.y * b.y + a.z * b.z + a.w * b.w;
    im += a.x * b.y - a.y * b.x + a.z * b.w - a.w * b.z;
}

__device__ __forceinline__ void csub4(float4& x, const float4 a, const float2 c) {
    x.x -= c.x * a.x - c.y * a.y; x.y -= c.x * a.y + c.y * a.x;
    x.z -= c.x * a.z - c.y * a.w; x.w -= c.x * a.w + c.y * a.z;
}

__device__ __forceinline__ void cadd4(float4& x, const float4 a, const float2 c) {
    x.x += c.x * a.x - c.y * a.y; x.y += c.x * a.y + c.y * a.x;
    x.z += c.x * a.z - c.y * a.w; x.w += c.x * a.w + c.y * a.z;
}

static dim3 row_grid(long long n2, int nrhs, int cap = 1216);

#define ROW_LOOP(i, n2) for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < (n2); i += (long long)gridDim.x * blockDim.x)

// ---- element-wise kernels; n = complex values per right-hand side (even) ----
__global__ void k_bcopy(float2* __restrict__ out, const float2* __restrict__ in, long long n, const int* skip) {
    const int r = blockIdx.y;
    if (skip && skip[r]) return;
    const float4* a = reinterpret_cast<const float4*>(in + r * n);
    float4* o = reinterpret_cast<float4*>(out + r * n);
    ROW_LOOP(i, n >> 1) o[i] = a[i];
}

__global__ void k_bsub32(float2* __restrict__ out, const float2* __restrict__ a, const float2* __restrict__ b,
                         long long n, const int* skip) {
    const int r = blockIdx.y;
    if (skip && skip[r]) return;
    const float4* x = reinterpret_cast<const float4*>(a + r * n);
    const float4* y = reinterpret_cast<const float4*>(b + r * n);
    float4* o = reinterpret_cast<float4*>(out + r * n);
    ROW_LOOP(i, n >> 1) {
        const float4 u = x[i], v = y[i];
        o[i] = make_float4(u.x - v.x, u.y - v.y, u.z - v.z, u.w - v.w);
    }
}

__global__ void k_bsub64(double2* __restrict__ out, const double2* __restrict__ a, const double2* __restrict__ b,
                         long long n, const int* skip) {
    const int r = blockIdx.y;
    if (skip && skip[r]) return;
    a += r * n; b += r * n; out += r * n;
    ROW_LOOP(i, n) { const double2 u = a[i], v = b[i]; out[i] = make_double2(u.x - v.x, u.y - v.y); }
}

// out (FP32) = a (FP64) * scale[r]
__global__ void k_bd2f_scale(float2* __restrict__ out, const double2* __restrict__ a, const double* scale, long long n,
                             const int* skip) {
    const int r = blockIdx.y;
    if (skip && skip[r]) return;
    const double s = scale[r];
    a += r * n; out += r * n;
    ROW_LOOP(i, n) { const double2 u = a[i]; out[i] = make_float2((float)(u.x * s), (float)(u.y * s)); }
}

// Slice-paired packed FP32 fine vectors (4-d, one right-hand side): packed float4 i holds
// element d of site x on slices 2j and 2j+1; pk_canon gives the canonical complex index of the
// slice-2j value (the slice-2j+1 value is V dof further).
struct PackIdx {
    long long V, NB;
    int dof;
};
__device__ __forceinline__ long long pk_canon(const PackIdx& q, long long i) {
    const int lane = (int)(i & 31);
    const long long t = i >> 5;
    const int d = (int)(t % q.dof);
    const long long t2 = t / q.dof;
    const long long x = (t2 % q.NB) * 32 + lane;
    const long long j = t2 / q.NB;
    return ((2 * j) * q.V + x) * q.dof + d;
}

// out (packed FP32) = scale * a (canonical FP64)
__global__ void k_bd2f_scale_pk(float2* __restrict__ out, const double2* __restrict__ a, const double* scale,
                                long long n, const int* skip, PackIdx q) {
    if (skip && skip[0]) return;
    const double s = scale[0];
    float4* o = reinterpret_cast<float4*>(out);
    const long long sv = q.V * q.dof;
    ROW_LOOP(i, n >> 1) {
        const long long c = pk_canon(q, i);
        const double2 u = a[c], w = a[c + sv];
        o[i] = make_float4((float)(u.x * s), (float)(u.y * s), (float)(w.x * s), (float)(w.y * s));
    }
}

// out[r] = |x_r|^2.  FP64 data: every product in FP64; FP32 data: per-thread
// FP32 partials over a few elements, FP64 across threads.
__global__ void __launch_bounds__(RED_THREADS) k_bnorm2_64(const double2* __restrict__ x, long long n, RedScratch rs,
                                                           double* out, const int* skip) {
    const int r = blockIdx.y;
    if (skip && skip[r]) return;
    x += r * n;
    double v[1] = {0.0};
    ROW_LOOP(i, n) { const double2 a = x[i]; v[0] += a.x * a.x + a.y * a.y; }
    grid_reduce<1>(v, row_scratch(rs, r), [=] __device__(double* t) { out[r] = t[0]; });
}

__global__ void __launch_bounds__(RED_THREADS) k_bnorm2_32(const float2* __restrict__ x, long long n, RedScratch rs,
                                                           double* out, const int* skip) {
    const int r = blockIdx.y;
    if (skip && skip[r]) return;
    const float4* a = reinterpret_cast<const float4*>(x + r * n);
    float acc = 0.f;
    ROW_LOOP(i, n >> 1) { const float4 u = a[i]; acc += u.x * u.x + u.y * u.y + u.z * u.z + u.w * u.w; }
    const float v[1] = {acc};
    grid_reduce_f<1>(v, row_scratch(rs, r), [=] __device__(double* t) { out[r] = t[0]; });
}

// rout = rin - alpha w, rr2 = |rout|^2 per right-hand side (rout may be rin).
// With `done`: iters[r] += 1 and done[r] = 1 once rr2 <= tol2 * ref2[r] or
// iters[r] >= maxit.  `skip` and `done` may be the same array: every block of a
// row reads the flag before the row's last block (the only writer) runs its
// finaliser.
__global__ void __launch_bounds__(RED_THREADS) k_bres_update(const float2* rin, float2* rout,
                                                             const float2* __restrict__ w, BGcr* g, long long n,
                                                             RedScratch rs, const int* skip, int* done,
                                                             const double* ref2, double tol2, int* iters, int maxit) {
    const int r = blockIdx.y;
    if (skip && skip[r]) return;
    const float ar = (float)g[r].alpha[0], ai = (float)g[r].alpha[1];
    const float4* a4 = reinterpret_cast<const float4*>(rin + r * n);
    float4* o4 = reinterpret_cast<float4*>(rout + r * n);
    const float4* w4 = reinterpret_cast<const float4*>(w + r * n);
    float acc = 0.f;
    ROW_LOOP(i, n >> 1) {
        const float4 wi = w4[i];
        float4 ri = a4[i];
        ri.x -= ar * wi.x - ai * wi.y; ri.y -= ar * wi.y + ai * wi.x;
        ri.z -= ar * wi.z - ai * wi.w; ri.w -= ar * wi.w + ai * wi.z;
        o4[i] = ri;
        acc += ri.x * ri.x + ri.y * ri.y + ri.z * ri.z + ri.w * ri.w;
    }
    const float v[1] = {acc};
    grid_reduce_f<1>(v, row_scratch(rs, r), [=] __device__(double* t) {
        g[r].rr2 = t[0];
        if (done) {
            iters[r] += 1;
            if (t[0] <= tol2 * ref2[r] || iters[r] >= maxit) done[r] = 1;
        }
    });
}

// Classical Gram-Schmidt dots: coef[j] = <W_j, w> / nrm[j] for j < k (k =
// gridDim.y), per right-hand side, also summed into C[k][j] (set on the first
// pass).  Grid (B, k, nrhs); W: device array of basis block pointers.
__global__ void __launch_bounds__(RED_THREADS) k_bmdot_rows(float2* const* __restrict__ W, const float2* __restrict__ w,
                                                       long long n, double* __restrict__ part, unsigned* counters,
                                                       BGcr* g, int first, const int* skip) {
    const int r = blockIdx.z, j = blockIdx.y;
    if (skip && skip[r]) return;
    const float4* Wj = reinterpret_cast<const float4*>(W[j] + r * n);
    const float4* w4 = reinterpret_cast<const float4*>(w + r * n);
    const long long n2 = n >> 1;
    float re = 0.f, im = 0.f;
    const long long stride = (long long)gridDim.x * blockDim.x;
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    for (; i + 3 * stride < n2; i += 4 * stride) {
        const float4 a0 = Wj[i], a1 = Wj[i + stride], a2 = Wj[i + 2 * stride], a3 = Wj[i + 3 * stride];
        const float4 b0 = w4[i], b1 = w4[i + stride], b2 = w4[i + 2 * stride], b3 = w4[i + 3 * stride];
        cdot4(a0, b0, re, im); cdot4(a1, b1, re, im); cdot4(a2, b2, re, im); cdot4(a3, b3, re, im);
    }
    for (; i < n2; i += stride) cdot4(Wj[i], w4[i], re, im);
    const float vf[2] = {re, im};
    double v[2];
    block_sum_f<2>(vf, v);
    const size_t rowi = (size_t)r * BK_MAX + j;
    double* pr = part + rowi * 2 * BMDOT_BLOCKS;
    if (threadIdx.x == 0) {
        pr[blockIdx.x] = v[0];
        pr[BMDOT_BLOCKS + blockIdx.x] = v[1];
    }
    if (!grid_last_block(counters + rowi * CROW)) return;
    __threadfence();
    double w2[2];
    grid_final_sum<2>(pr, BMDOT_BLOCKS, w2);
    if (threadIdx.x == 0) {
        const double nn = g[r].nrm[j];
        const double cr = nn > 0 ? w2[0] / nn : 0.0, ci = nn > 0 ? w2[1] / nn : 0.0;
        const int k = gridDim.y;
        g[r].coef[j][0] = cr;
        g[r].coef[j][1] = ci;
        g[r].C[k][j][0] = first ? cr : g[r].C[k][j][0] + cr;
        g[r].C[k][j][1] = first ? ci : g[r].C[k][j][1] + ci;
    }
}

// The same dots for vectors larger than L2: coef[j] = <W_j, w> / nrm[j] for j < k, per
// right-hand side, also summed into C[k][j] (set on the first pass).  Grid
// (B, nrhs): each thread reads its elements of w once and of every W_j once
// (k + 1 vectors per pass instead of 2 k), keeping the k partial dots in
// registers (KM >= k, unrolled with guards).  The last block of a row sums the
// per-block partials of every j in a fixed order.  W: device array of basis
// block pointers.
template <int KM>
__global__ void __launch_bounds__(RED_THREADS) k_bmdot(float2* const* __restrict__ W, const float2* __restrict__ w,
                                                       long long n, int k, double* __restrict__ part,
                                                       unsigned* counters, BGcr* g, int first, const int* skip) {
    const int r = blockIdx.y;
    if (skip && skip[r]) return;
    __shared__ const float4* Wp[KM];
    for (int j = threadIdx.x; j < k; j += blockDim.x) Wp[j] = reinterpret_cast<const float4*>(W[j] + r * n);
    __syncthreads();
    const float4* w4 = reinterpret_cast<const float4*>(w + r * n);
    float re[KM], im[KM];
#pragma unroll
    for (int j = 0; j < KM; ++j) { re[j] = 0.f; im[j] = 0.f; }
    ROW_LOOP(i, n >> 1) {
        const float4 wi = w4[i];
#pragma unroll
        for (int j = 0; j < KM; ++j)
            if (j < k) cdot4(Wp[j][i], wi, re[j], im[j]);
    }
    double* pr = part + (size_t)r * BK_MAX * 2 * BMDOT_BLOCKS;     // [j][re / im][block]
#pragma unroll
    for (int j0 = 0; j0 < KM; j0 += 4) {
        if (j0 >= k) break;                                       // block-uniform
        float vf[8];
#pragma unroll
        for (int q = 0; q < 4; ++q) { vf[2 * q] = re[j0 + q]; vf[2 * q + 1] = im[j0 + q]; }
        double v[8];
        block_sum_f<8>(vf, v);
        if (threadIdx.x == 0)
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (j0 + q < k) {
                    pr[(size_t)(j0 + q) * 2 * BMDOT_BLOCKS + blockIdx.x] = v[2 * q];
                    pr[(size_t)(j0 + q) * 2 * BMDOT_BLOCKS + BMDOT_BLOCKS + blockIdx.x] = v[2 * q + 1];
                }
    }
    if (!grid_last_block(counters + (size_t)r * BK_MAX * CROW)) return;
    __threadfence();
    // quantity q = 2 j + (0: Re, 1: Im) of block b at pr[q * BMDOT_BLOCKS + b]; warp w sums q = w, w + 8, ...
    __shared__ double tot[2 * KM];
    {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        for (int q = warp; q < 2 * k; q += RED_THREADS / 32) {
            double sq = 0.0;
            for (unsigned bb = lane; bb < gridDim.x; bb += 32) sq += __ldcg(pr + (size_t)q * BMDOT_BLOCKS + bb);
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) sq += __shfl_down_sync(0xffffffffu, sq, off);
            if (lane == 0) tot[q] = sq;
        }
    }
    __syncthreads();
    for (int j = 0; j < k; ++j) {
        if (threadIdx.x == 0) {
            const double nn = g[r].nrm[j];
            const double cr = nn > 0 ? tot[2 * j] / nn : 0.0, ci = nn > 0 ? tot[2 * j + 1] / nn : 0.0;
            g[r].coef[j][0] = cr;
            g[r].coef[j][1] = ci;
            g[r].C[k][j][0] = first ? cr : g[r].C[k][j][0] + cr;
            g[r].C[k][j][1] = first ? ci : g[r].C[k][j][1] + ci;
        }
    }
}

static void launch_bmdot(dim3 grid, float2* const* W, const float2* w, long long n, int k, double* part,
                         unsigned* counters, BGcr* g, int first, const int* skip, cudaStream_t st) {
    if (k <= 4)       k_bmdot<4><<<grid, RED_THREADS, 0, st>>>(W, w, n, k, part, counters, g, first, skip);
    else if (k <= 8)  k_bmdot<8><<<grid, RED_THREADS, 0, st>>>(W, w, n, k, part, counters, g, first, skip);
    else if (k <= 16) k_bmdot<16><<<grid, RED_THREADS, 0, st>>>(W, w, n, k, part, counters, g, first, skip);
    else              k_bmdot<32><<<grid, RED_THREADS, 0, st>>>(W, w, n, k, part, counters, g, first, skip);
}

// w -= sum_{j<k} coef_j W_j per right-hand side.  FINAL: also nrm[k] = |w|^2,
// alpha = A[k] = <w, res> / |w|^2, and steps[r] = k + 1 (steps may be null).
template <bool FINAL>
__global__ void __launch_bounds__(RED_THREADS) k_bmaxpy(float2* __restrict__ w, float2* const* __restrict__ W, BGcr* g,
                                                        int k, const float2* __restrict__ res, long long n,
                                                        RedScratch rs, int* steps, const int* skip) {
    const int r = blockIdx.y;
    if (skip && skip[r]) return;
    __shared__ float2 c[BK_MAX];
    __shared__ const float4* Wp[BK_MAX];
    for (int j = threadIdx.x; j < k; j += blockDim.x) {
        c[j] = make_float2((float)g[r].coef[j][0], (float)g[r].coef[j][1]);
        Wp[j] = reinterpret_cast<const float4*>(W[j] + r * n);
    }
    __syncthreads();
    float4* w4 = reinterpret_cast<float4*>(w + r * n);
    const float4* r4 = reinterpret_cast<const float4*>(res + r * n);
    float f0 = 0.f, f1 = 0.f, f2 = 0.f;
    ROW_LOOP(i, n >> 1) {
        float4 wi = w4[i];
        int j = 0;
        for (; j + 3 < k; j += 4) {
            const float4 a0 = Wp[j][i], a1 = Wp[j + 1][i], a2 = Wp[j + 2][i], a3 = Wp[j + 3][i];
            csub4(wi, a0, c[j]); csub4(wi, a1, c[j + 1]); csub4(wi, a2, c[j + 2]); csub4(wi, a3, c[j + 3]);
        }
        for (; j < k; ++j) csub4(wi, Wp[j][i], c[j]);
        if (k > 0) w4[i] = wi;
        if (FINAL) {
            f0 += wi.x * wi.x + wi.y * wi.y + wi.z * wi.z + wi.w * wi.w;
            cdot4(wi, r4[i], f1, f2);
        }
    }
    if (FINAL) {
        const float v[3] = {f0, f1, f2};
        grid_reduce_f<3>(v, row_scratch(rs, r), [=] __device__(double* t) {
            const double ar = t[0] > 0 ? t[1] / t[0] : 0.0, ai = t[0] > 0 ? t[2] / t[0] : 0.0;
            g[r].nrm[k] = t[0];
            g[r].alpha[0] = ar; g[r].alpha[1] = ai;
            g[r].A[k][0] = ar; g[r].A[k][1] = ai;
            if (steps) steps[r] = k + 1;
        });
    }
}

// ---------------------------------------------------------------------------
// GCR in blocks of up to SB steps (cgs_passes = 1): the directions of a block are
// p_0 = r, p_1 = A p_0, .., p_{m-1} = A p_{m-2}, which span the same Krylov space
// as m single steps, so the block ends at the residual that m single steps end
// at (the minimum over that space).  Its images w_i = A p_i are orthogonalised
// together: one reduction pass reads every vector of the basis once for all of
// the block and one element-wise pass writes the block's orthogonal images and the new
// residual, where single steps pass over the basis twice per step.  8 steps
// take 45 passes over a vector instead of 128, 16 steps 123 instead of 420.
//
// With W_j the orthogonal images so far (r is orthogonal to them), the reduction
// sums d_ij = <W_j, w_i>, G_ab = <w_a, w_b>, <w_i, r> and |r|^2, and the rest is
// algebra on scalars in FP64:
//   c_ij = d_ij / |W_j|^2,   G'_ab = G_ab - sum_j conj(d_aj) d_bj / |W_j|^2,
//   G' = L D L^H by elimination: w'_i = w_i - sum_j c_ij W_j - sum_{l<i} L_il w'_l,
//   |w'_i|^2 = D_i,  <w'_i, r> = <w_i, r> - sum_{l<i} conj(L_il) <w'_l, r>,
//   alpha_i = <w'_i, r> / D_i,   |r'|^2 = |r|^2 - sum_i |<w'_i, r>|^2 / D_i.
// |r|^2 is summed afresh in every block; only the prediction for its end
// decides convergence.  A direction with D_i below BSTEP_BREAK |w_i|^2 is not
// resolved by FP32 sums: it and the rest of its block are dropped (alpha = 0),
// and a block that loses its first direction ends that row's coarse solve.
// SB = 4: the powers of A in a block have a Gram matrix of condition 4e4 on the
// 2-d and 4-d operators (FP32 sums resolve it; 8 powers reach 4e10 and do not).
// Against single steps: 256^2 x 16 gradient step (two solves to 1e-12) 1017 -> 630 ms,
// 12^3 x 24 x 16 solve 1011 -> 614 ms, 14 sources on 64^2, 128^2, 256^2 1282 -> 764 ms, with the
// same iteration counts.
// ---------------------------------------------------------------------------
constexpr int SB = 4;
constexpr double BSTEP_BREAK = 1e-5;
constexpr int BLK_Q0 = 25;            // Gram 4 + 2 * 6, <w_i, r> 2 * 4, |r|^2
constexpr int BLK_KM = 12;            // basis vectors one thread takes together; more go SB to a group (grid.z)
constexpr int BLK_GROUP = 10;         // blocks of a row whose partial sums meet first
constexpr int BLK_GROUPS_MAX = 31;    // 304 blocks in groups of 10
// quantity of d_ij: BLK_Q0 + 2 (SB j + i) (+ 1: Im)

// The sums over a warp of N quantities per lane (N a multiple of 32): afterwards v[q] of lane l,
// q < N / 32, is the sum of quantity l N / 32 + q.  Every exchange halves the quantities a lane
// still carries: N - N / 32 shuffles, where a tree per quantity takes 5 N.
template <int N>
__device__ __forceinline__ void warp_sums(float (&v)[N]) {
    const int lane = threadIdx.x & 31;
    int half = N / 2;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1, half >>= 1) {
        const bool up = lane & off;
#pragma unroll
        for (int i = 0; i < N / 2; ++i)
            if (i < half) {
                const float send = up ? v[i] : v[i + half];
                const float keep = up ? v[i + half] : v[i];
                v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
            }
    }
}

// The scalars of a block from the totals of its reduction (shared memory), by one warp: rows
// k .. k + m - 1 of C, nrm and A, then |r'|^2 and, with `done`, the convergence test.  An FP64
// instruction holds the SM's FP64 unit 16 clocks whether one lane or 32 take part, so the
// elimination runs over the lanes: lane 8 a + b holds M_ab = G'_ab for b < SB and
// M_a,SB = <w_a, r>, and step l subtracts conj(L_al) M_lb everywhere at once (one thread alone
// took about 6 us).
__device__ __forceinline__ void blk_scalars(const double* tot, int k, int m, BGcr& G, int* steps, int* done, double ref2,
                                            double tol2, int* iters, int maxit) {
    __shared__ double inv[BK_MAX];
    __shared__ double2 cc[BK_MAX][SB];
    const int lane = threadIdx.x & 31;
    const int a = lane >> 3, b = lane & 7;
    const int it0 = done ? *iters : 0;
    if (lane < k) {                                              // k < BK_MAX = 32
        const double nn = G.nrm[lane];
        inv[lane] = nn > 0 ? 1.0 / nn : 0.0;
    }
    __syncwarp();
    for (int e = lane; e < SB * k; e += 32) {
        const int i = e % SB, j = e / SB;
        const double2 c = make_double2(tot[BLK_Q0 + 2 * e] * inv[j], tot[BLK_Q0 + 2 * e + 1] * inv[j]);
        cc[j][i] = c;
        if (i < m) { G.C[k + i][j][0] = c.x; G.C[k + i][j][1] = c.y; }
    }
    __syncwarp();
    double2 M = make_double2(0.0, 0.0);
    if (b < SB) {
        const int lo = a < b ? a : b, hi = a < b ? b : a;
        if (a == b) M.x = tot[a];
        else {
            M.x = tot[4 + hi * (hi - 1) + 2 * lo];
            M.y = (a < b ? 1.0 : -1.0) * tot[5 + hi * (hi - 1) + 2 * lo];
        }
        for (int j = 0; j < k; ++j) {
            const double2 c = cc[j][a];
            const double dx = tot[BLK_Q0 + 2 * (SB * j + b)], dy = tot[BLK_Q0 + 2 * (SB * j + b) + 1];
            M.x -= c.x * dx; M.x -= c.y * dy;
            M.y -= c.x * dy; M.y += c.y * dx;
        }
    } else if (b == SB) {
        M = make_double2(tot[16 + 2 * a], tot[17 + 2 * a]);
    }
    const int left = done ? (maxit > it0 ? maxit - it0 : 1) : m;   // steps the iteration cap leaves
    const int take = left < m ? left : m;
    bool ok = true, first = true;
    double fall = 0.0;                                           // of |r|^2: this lane's share
#pragma unroll
    for (int l = 0; l < SB; ++l) {
        if (l >= m) break;
        const double d = __shfl_sync(0xffffffffu, M.x, 9 * l);
        if (!(d > BSTEP_BREAK * tot[l])) { ok = false; if (l == 0) first = false; }
        const bool use = ok && l < take;
        const double id = use ? 1.0 / d : 0.0;
        const double2 row = make_double2(__shfl_sync(0xffffffffu, M.x, 8 * l + b), __shfl_sync(0xffffffffu, M.y, 8 * l + b));
        const double2 la = make_double2(__shfl_sync(0xffffffffu, M.x, 8 * l + a), __shfl_sync(0xffffffffu, M.y, 8 * l + a));
        if (a == l) {                                            // this lane's M is M_lb
            const double2 q = make_double2(M.x * id, M.y * id);
            if (b < m && b > l) { G.C[k + b][k + l][0] = q.x; G.C[k + b][k + l][1] = q.y; }
            if (b == SB) {
                G.A[k + l][0] = q.x; G.A[k + l][1] = q.y;
                fall = M.x * q.x + M.y * q.y;
            }
            if (b == l) G.nrm[k + l] = use ? d : 0.0;
        } else if (a > l) {
            const double lx = la.x * id, ly = la.y * id;         // L_al
            M.x -= lx * row.x; M.x -= ly * row.y;
            M.y -= lx * row.y; M.y += ly * row.x;
        }
    }
    double rr = tot[24];
#pragma unroll
    for (int l = 0; l < SB; ++l) rr -= __shfl_sync(0xffffffffu, fall, 8 * l + SB);
    if (lane != 0) return;
    G.rr2 = rr;
    if (steps) *steps = k + m;
    if (done) {
        *iters = it0 + take;
        if (!first || rr <= tol2 * ref2 || it0 + take >= maxit) *done = 1;
    }
}

// The images of a block before orthogonalisation: w_i
struct BlkVecs {
    const float2* w[SB];
};

// Grid (B, nrhs, groups of KM basis vectors), k = KM * groups: no guards in the loop, so that all
// KM + 5 16-byte loads of an iteration are in flight before the first product (with a guard per
// basis vector the loads went one by one: 687 us, now 248, for 12 basis vectors at 12^3 x 24 x 16).  Memory-bound at
// fine sizes, at coarse sizes launch and tail.  The partial sums go to part as [block][quantity],
// so that they are added up in contiguous runs.  done == nullptr: no convergence test (the smoother).
template <int KM>
__global__ void __launch_bounds__(RED_THREADS)
k_blk_dots(float2* const* __restrict__ W, BlkVecs bv, const float2* __restrict__ res, long long n, int k, int m,
           double* __restrict__ part, unsigned* counters, BGcr* g, const int* skip, int* steps, int* done,
           const double* ref2, double tol2, int* iters, int maxit) {
    constexpr int NQ = BLK_Q0 + 2 * SB * KM;
    constexpr int NV = (NQ + 31) / 32 * 32;
    const int r = blockIdx.y, j0 = blockIdx.z * KM;
    if (skip && skip[r]) return;
    __shared__ double sh[NV][RED_THREADS / 32 + 1];
    const float4* Wp[KM + 1];
#pragma unroll
    for (int j = 0; j < KM; ++j) Wp[j] = reinterpret_cast<const float4*>(W[j0 + j] + r * n);
    const float4* r4 = reinterpret_cast<const float4*>(res + r * n);
    const float4* w4[SB];
#pragma unroll
    for (int i = 0; i < SB; ++i) w4[i] = i < m ? reinterpret_cast<const float4*>(bv.w[i] + r * n) : nullptr;
    float v[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = 0.f;
    const bool gram = blockIdx.z == 0;
    ROW_LOOP(x, n >> 1) {
        float4 a[SB], b[KM + 1];
#pragma unroll
        for (int i = 0; i < SB; ++i) a[i] = i < m ? w4[i][x] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int j = 0; j < KM; ++j) b[j] = Wp[j][x];
        if (gram) {
            const float4 c = r4[x];
#pragma unroll
            for (int i = 0; i < SB; ++i) {
                v[i] += a[i].x * a[i].x + a[i].y * a[i].y + a[i].z * a[i].z + a[i].w * a[i].w;
                cdot4(a[i], c, v[16 + 2 * i], v[17 + 2 * i]);
#pragma unroll
                for (int l = 0; l < i; ++l) cdot4(a[l], a[i], v[4 + i * (i - 1) + 2 * l], v[5 + i * (i - 1) + 2 * l]);
            }
            v[24] += c.x * c.x + c.y * c.y + c.z * c.z + c.w * c.w;
        }
#pragma unroll
        for (int j = 0; j < KM; ++j)
#pragma unroll
            for (int i = 0; i < SB; ++i)
                cdot4(b[j], a[i], v[BLK_Q0 + 2 * (SB * j + i)], v[BLK_Q0 + 2 * (SB * j + i) + 1]);
    }
    // the tree over each warp in FP32, every sum across warps and blocks in FP64
    warp_sums<NV>(v);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < NV / 32; ++q) sh[lane * (NV / 32) + q][warp] = (double)v[q];
    __syncthreads();
    const int nq = BLK_Q0 + 2 * SB * k;                          // quantities of the whole row
    const int B = gridDim.x;
    double* pr = part + (size_t)r * BK_MAX * 2 * BMDOT_BLOCKS;   // [block][quantity]
    for (int q = threadIdx.x; q < NQ; q += blockDim.x) {
        if (q < BLK_Q0 && !gram) continue;
        double t = 0.0;
#pragma unroll
        for (int u = 0; u < RED_THREADS / 32; ++u) t += sh[q][u];
        pr[(size_t)blockIdx.x * nq + (q < BLK_Q0 ? q : q + 2 * SB * j0)] = t;
        __threadfence();
    }
    __syncthreads();
    // Blocks meet twice: the last of each group of BLK_GROUP adds the group's partials up (in order), and the last
    // group's last block adds the groups: one SM alone would spend 2 us and more on the FP64 sums of 128 blocks.
    const unsigned ngroups = (B + BLK_GROUP - 1) / BLK_GROUP, grp = blockIdx.x / BLK_GROUP;
    const int rows = min(BLK_GROUP, B - (int)grp * BLK_GROUP);
    unsigned* cnt = counters + (size_t)r * BK_MAX * CROW;         // [ngroups] then the top one, 128 bytes apart
    __shared__ bool last;
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(cnt + grp * RED_CSTRIDE, 1u) == (unsigned)rows * gridDim.z - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    constexpr int NT = BLK_Q0 + 2 * SB * BK_MAX;
    __shared__ double tot[NT];
    double* gr = pr + (size_t)grp * BLK_GROUP * nq;              // the group's sums replace its first row
    for (int q = threadIdx.x; q < nq; q += blockDim.x) {
        double t = 0.0;
#pragma unroll
        for (int u = 0; u < BLK_GROUP; ++u) t += u < rows ? __ldcg(gr + (size_t)u * nq + q) : 0.0;
        if (ngroups == 1) tot[q] = t;
        else gr[q] = t;
        __threadfence();
    }
    __syncthreads();
    if (ngroups > 1) {
        if (threadIdx.x == 0) {
            cnt[grp * RED_CSTRIDE] = 0u;
            __threadfence();
            last = atomicAdd(cnt + BLK_GROUPS_MAX * RED_CSTRIDE, 1u) == ngroups - 1;
            if (last) cnt[BLK_GROUPS_MAX * RED_CSTRIDE] = 0u;
        }
        __syncthreads();
        if (!last) return;
        __threadfence();
        for (int q = threadIdx.x; q < nq; q += blockDim.x) {
            double t = 0.0;
#pragma unroll 8
            for (unsigned u = 0; u < ngroups; ++u) t += __ldcg(pr + (size_t)u * BLK_GROUP * nq + q);
            tot[q] = t;
        }
        __syncthreads();
    } else if (threadIdx.x == 0) {
        cnt[grp * RED_CSTRIDE] = 0u;
    }
    if (warp == 0)
        blk_scalars(tot, k, m, g[r], steps ? steps + r : nullptr, done ? done + r : nullptr, ref2 ? ref2[r] : 0.0, tol2,
                    iters ? iters + r : nullptr, maxit);
}

static void launch_blk_dots(float2* const* W, const BlkVecs& bv, const float2* res, long long n, int nrhs, int k, int m,
                            double* part, unsigned* counters, BGcr* g, const int* skip, int* steps, int* done,
                            const double* ref2, double tol2, int* iters, int maxit, cudaStream_t st) {
    // about 4 float4 per thread, at most two blocks per SM (one where the sums leave registers for no more), and no
    // more than the row's partial sums have room for
    const int nq = BLK_Q0 + 2 * SB * k, km = k <= BLK_KM ? k : SB;
    long long B = ((n >> 1) + 4 * RED_THREADS - 1) / (4 * RED_THREADS);
    const long long cap = km <= 4 ? 304 : 152, room = (long long)BK_MAX * 2 * BMDOT_BLOCKS / nq;
    if (B > cap) B = cap;
    if (B > room) B = room;
    if (B < 1) B = 1;
    const dim3 grid((unsigned)B, (unsigned)nrhs, (unsigned)(km > 0 ? k / km : 1));
#define DWF_BLK(KM) k_blk_dots<KM><<<grid, RED_THREADS, 0, st>>>(W, bv, res, n, k, m, part, counters, g, skip, steps, \
                                                                 done, ref2, tol2, iters, maxit)
    if (km == 0)      DWF_BLK(0);
    else if (km == 4) DWF_BLK(4);
    else if (km == 8) DWF_BLK(8);
    else              DWF_BLK(12);
#undef DWF_BLK
}

// The element-wise pass of a block: w'_i into Wout[i] (STORE: a later block needs them) and
// r' = r - sum_i alpha_i w'_i, or with rsub the difference rsub - r' (the image of the smoother's
// whole correction), into rout.  w'_i may overwrite w_i.
struct BlkOut {
    float2* w[SB];
};
template <bool STORE>
__global__ void __launch_bounds__(RED_THREADS)
k_blk_update(float2* const* __restrict__ W, BlkVecs bv, BlkOut bo, const BGcr* g, int k, int m,
             const float2* __restrict__ rin, const float2* __restrict__ rsub, float2* __restrict__ rout, long long n,
             const int* skip) {
    const int r = blockIdx.y;
    if (skip && skip[r]) return;
    __shared__ float2 c[SB][BK_MAX];                             // c_ij (j < k) and L_il (j = k + l)
    __shared__ float2 al[SB];
    __shared__ const float4* Wp[BK_MAX];
    const BGcr& G = g[r];
    for (int e = threadIdx.x; e < SB * (k + SB); e += blockDim.x) {
        const int i = e % SB, j = e / SB;
        if (i < m && j < k + i) c[i][j] = make_float2((float)G.C[k + i][j][0], (float)G.C[k + i][j][1]);
    }
    if (threadIdx.x < m) al[threadIdx.x] = make_float2((float)G.A[k + threadIdx.x][0], (float)G.A[k + threadIdx.x][1]);
    for (int j = threadIdx.x; j < k; j += blockDim.x) Wp[j] = reinterpret_cast<const float4*>(W[j] + r * n);
    __syncthreads();
    const float4* r4 = reinterpret_cast<const float4*>(rin + r * n);
    const float4* s4 = rsub ? reinterpret_cast<const float4*>(rsub + r * n) : nullptr;
    float4* o4 = reinterpret_cast<float4*>(rout + r * n);
    const float4* w4[SB];
    float4* q4[SB];
#pragma unroll
    for (int i = 0; i < SB; ++i) {
        w4[i] = i < m ? reinterpret_cast<const float4*>(bv.w[i] + r * n) : nullptr;
        q4[i] = STORE && i < m ? reinterpret_cast<float4*>(bo.w[i] + r * n) : nullptr;
    }
    ROW_LOOP(x, n >> 1) {
        float4 a[SB];
#pragma unroll
        for (int i = 0; i < SB; ++i) a[i] = i < m ? w4[i][x] : make_float4(0.f, 0.f, 0.f, 0.f);
        float4 rr = r4[x];
        float4 ss = make_float4(0.f, 0.f, 0.f, 0.f);
        if (s4) ss = s4[x];
        for (int j = 0; j < k; j += 4) {                         // k is a multiple of SB = 4
            const float4 b0 = Wp[j][x], b1 = Wp[j + 1][x], b2 = Wp[j + 2][x], b3 = Wp[j + 3][x];
#pragma unroll
            for (int i = 0; i < SB; ++i)
                if (i < m) {
                    csub4(a[i], b0, c[i][j]); csub4(a[i], b1, c[i][j + 1]);
                    csub4(a[i], b2, c[i][j + 2]); csub4(a[i], b3, c[i][j + 3]);
                }
        }
#pragma unroll
        for (int i = 0; i < SB; ++i)
            if (i < m) {
#pragma unroll
                for (int l = 0; l < i; ++l) csub4(a[i], a[l], c[i][k + l]);
                if (STORE) q4[i][x] = a[i];
                csub4(rr, a[i], al[i]);
            }
        if (s4) rr = make_float4(ss.x - rr.x, ss.y - rr.y, ss.z - rr.z, ss.w - rr.w);
        o4[x] = rr;
    }
}

// One block of GCR steps k .. k + m - 1: the raw images are in P[k + 1] .. P[k + m - 1] and
// Q[k + m - 1], the residual in P[k]; Q[k] .. Q[k + m - 1] receive the orthogonal images (when
// `store`) and rout the new residual (with rsub: rsub minus it).
static dwf_status bblock(BGcr* g, float2* const* P, float2* const* Q, float2* const* dQ, int k, int m, bool store,
                         const float2* rsub, float2* rout, long long n, int nrhs, double* part, unsigned* counters,
                         const int* skip, int* steps, int* done, const double* ref2, double tol2, int* iters,
                         int maxit, cudaStream_t st) {
    BlkVecs bv{};
    BlkOut bo{};
    for (int i = 0; i < m; ++i) {
        bv.w[i] = i + 1 < m ? P[k + i + 1] : Q[k + m - 1];
        bo.w[i] = Q[k + i];
    }
    launch_blk_dots(dQ, bv, P[k], n, nrhs, k, m, part, counters, g, skip, steps, done, ref2, tol2, iters, maxit, st);
    const dim3 eg = row_grid(n >> 1, nrhs);
    if (store) k_blk_update<true><<<eg, RED_THREADS, 0, st>>>(dQ, bv, bo, g, k, m, P[k], rsub, rout, n, skip);
    else       k_blk_update<false><<<eg, RED_THREADS, 0, st>>>(dQ, bv, bo, g, k, m, P[k], rsub, rout, n, skip);
    DWF_CHECK_LAUNCH();
    return DWF_OK;
}

// y of the deferred solution update for the first m <= 32 steps: (I + C)^T y = A,
// y_j = A_j - sum_{k>j} C[k][j] y_k, by one warp in FP64 (lane j holds y_j; one thread alone
// took 7 us for 16 steps, at the start of every block of the combination)
__device__ __forceinline__ void back_substitute(const BGcr& g, int m, float2* y) {
    const int j = threadIdx.x;
    if (j >= 32) return;
    double a = 0.0, b = 0.0;
    if (j < m) { a = g.A[j][0]; b = g.A[j][1]; }
    for (int k = m - 1; k > 0; --k) {
        const double yr = __shfl_sync(0xffffffffu, a, k), yi = __shfl_sync(0xffffffffu, b, k);
        if (j < k) {
            const double cr = g.C[k][j][0], ci = g.C[k][j][1];
            a -= cr * yr - ci * yi;
            b -= cr * yi + ci * yr;
        }
    }
    if (j < m) y[j] = make_float2((float)a, (float)b);
}

// out += sum_{j<m} y_j P_j (FP32), m = nsteps[r] or m_fixed when nsteps is
// null; rows with m == 0 are left alone.  With wout: also wout = ra - rb.
__global__ void __launch_bounds__(RED_THREADS) k_bcombine32(float2* __restrict__ out, float2* const* __restrict__ P,
                                                            const BGcr* g, const int* nsteps, int m_fixed, long long n,
                                                            const float2* __restrict__ ra, const float2* __restrict__ rb,
                                                            float2* __restrict__ wout, const int* skip) {
    const int r = blockIdx.y;
    if (skip && skip[r]) return;
    const int m = nsteps ? nsteps[r] : m_fixed;
    __shared__ float2 y[BK_MAX];
    __shared__ const float4* Pp[BK_MAX];
    if (m > 0) back_substitute(g[r], m, y);
    for (int j = threadIdx.x; j < m; j += blockDim.x) Pp[j] = reinterpret_cast<const float4*>(P[j] + r * n);
    __syncthreads();
    float4* o4 = reinterpret_cast<float4*>(out + r * n);
    const float4* a4 = wout ? reinterpret_cast<const float4*>(ra + r * n) : nullptr;
    const float4* b4 = wout ? reinterpret_cast<const float4*>(rb + r * n) : nullptr;
    float4* w4 = wout ? reinterpret_cast<float4*>(wout + r * n) : nullptr;
    ROW_LOOP(i, n >> 1) {
        if (m > 0) {
            float4 x = o4[i];
            int j = 0;
            for (; j + 3 < m; j += 4) {
                const float4 b0 = Pp[j][i], b1 = Pp[j + 1][i], b2 = Pp[j + 2][i], b3 = Pp[j + 3][i];
                cadd4(x, b0, y[j]); cadd4(x, b1, y[j + 1]); cadd4(x, b2, y[j + 2]); cadd4(x, b3, y[j + 3]);
            }
            for (; j < m; ++j) cadd4(x, Pp[j][i], y[j]);
            o4[i] = x;
        }
        if (wout) {
            const float4 u = a4[i], v = b4[i];
            w4[i] = make_float4(u.x - v.x, u.y - v.y, u.z - v.z, u.w - v.w);
        }
    }
}

// X (FP64) += s[r] * sum_{j<m} y_j Z_j, m = nsteps[r]; rows with m == 0 are left alone
__global__ void __launch_bounds__(RED_THREADS) k_bcombine64(double2* __restrict__ X, float2* const* __restrict__ Z,
                                                            const BGcr* g, const int* nsteps, const double* s,
                                                            long long n) {
    const int r = blockIdx.y;
    const int m = nsteps[r];
    if (m <= 0) return;
    __shared__ float2 y[BK_MAX];
    __shared__ const float4* Zp[BK_MAX];
    back_substitute(g[r], m, y);
    for (int j = threadIdx.x; j < m; j += blockDim.x) Zp[j] = reinterpret_cast<const float4*>(Z[j] + r * n);
    __syncthreads();
    const double sc = s[r];
    double2* x2 = X + r * n;
    ROW_LOOP(i, n >> 1) {
        float4 e = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int j = 0; j < m; ++j) cadd4(e, Zp[j][i], y[j]);
        double2 a = x2[2 * i], b = x2[2 * i + 1];
        a.x += sc * e.x; a.y += sc * e.y; b.x += sc * e.z; b.y += sc * e.w;
        x2[2 * i] = a; x2[2 * i + 1] = b;
    }
}

// k_bcombine64 with the basis in the packed layout and X canonical (one right-hand side)
__global__ void __launch_bounds__(RED_THREADS) k_bcombine64_pk(double2* __restrict__ X, float2* const* __restrict__ Z,
                                                               const BGcr* g, const int* nsteps, const double* s,
                                                               long long n, PackIdx q) {
    const int m = nsteps[0];
    if (m <= 0) return;
    __shared__ float2 y[BK_MAX];
    __shared__ const float4* Zp[BK_MAX];
    back_substitute(g[0], m, y);
    for (int j = threadIdx.x; j < m; j += blockDim.x) Zp[j] = reinterpret_cast<const float4*>(Z[j]);
    __syncthreads();
    const double sc = s[0];
    const long long sv = q.V * q.dof;
    ROW_LOOP(i, n >> 1) {
        float4 e = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int j = 0; j < m; ++j) cadd4(e, Zp[j][i], y[j]);
        const long long c = pk_canon(q, i);
        double2 a = X[c], b = X[c + sv];
        a.x += sc * e.x; a.y += sc * e.y; b.x += sc * e.z; b.y += sc * e.w;
        X[c] = a; X[c + sv] = b;
    }
}

// --------------------------------------------------------------------------
// workspace: one arena per handle, sized for `cap` right-hand sides
// --------------------------------------------------------------------------
struct BView {
    int nrhs;
    long long nf, nc;
    float2 *rA, *r, *tmp, *rs_, *ps;
    float2 *Z[BK_MAX], *W[BK_MAX], *Ps[BK_MAX], *Qs[BK_MAX];
    float2 *rc, *ec, *crr, *ct;
    float2 *Zc[BK_MAX], *Wc[BK_MAX];
    double2 *r64, *t64;
    float2** dptr;            // device pointer arrays: Z, W, Ps, Qs, Zc, Wc (BK_MAX each)
    double* mpart;            // Gram-Schmidt partials [nrhs][BK_MAX][2][BMDOT_BLOCKS]
    unsigned* mcount;         // Gram-Schmidt counters [nrhs][BK_MAX][CROW]
    RedScratch red;           // reductions: [nrhs][PROW] partials, [nrhs][CROW] counters
    BGcr *outer, *smooth, *cgcr;
    double *bn2, *rn2, *rA2, *ref2, *cref2, *scale, *rn;
    int *odone, *idone, *cdone, *iters, *citers, *csteps;
    double* pg_part;          // persistent coarse GCR (one right-hand side): partial sums
    unsigned* pg_bar;         // its grid barrier state (count, gen, error, pad)
    int* pg_iters;            // its step counter
    double* pg_rr2;
};

struct Carver {
    char* base;
    size_t off = 0;
    template <class T> T* take(size_t count) {
        off = (off + 255) & ~(size_t)255;
        T* p = reinterpret_cast<T*>(base ? base + off : nullptr);
        off += count * sizeof(T);
        return p;
    }
};

static void carve(const dwf_mg* h, int nrhs, char* base, BView& v, size_t* total, size_t* zero_begin,
                  size_t* zero_end) {
    Carver c{base};
    const int K = h->prm.gcr_restart, S = h->prm.post_smooth, KC = h->prm.coarse_restart;
    v.nrhs = nrhs;
    v.nf = fine_len(h);
    v.nc = coarse_len(h);
    const size_t F = (size_t)nrhs * v.nf, C = (size_t)nrhs * v.nc;
    v.rA = c.take<float2>(F); v.r = c.take<float2>(F);
    v.tmp = c.take<float2>(F); v.ps = c.take<float2>(F);
    v.rs_ = h->prm.cgs_passes == 2 ? c.take<float2>(F) : nullptr;
    for (int k = 0; k < BK_MAX; ++k) {
        v.Z[k] = k < K ? c.take<float2>(F) : nullptr;
        v.W[k] = k < K ? c.take<float2>(F) : nullptr;
        v.Ps[k] = k < S ? c.take<float2>(F) : nullptr;
        v.Qs[k] = k < S ? c.take<float2>(F) : nullptr;
    }
    v.r64 = c.take<double2>(F); v.t64 = c.take<double2>(F);
    v.rc = c.take<float2>(C); v.ec = c.take<float2>(C); v.crr = c.take<float2>(C); v.ct = c.take<float2>(C);
    for (int k = 0; k < BK_MAX; ++k) {
        v.Zc[k] = k < KC ? c.take<float2>(C) : nullptr;
        v.Wc[k] = k < KC ? c.take<float2>(C) : nullptr;
    }
    v.dptr = c.take<float2*>(6 * BK_MAX);
    v.mpart = c.take<double>((size_t)nrhs * BK_MAX * 2 * BMDOT_BLOCKS);
    v.red.partials = c.take<double>((size_t)nrhs * PROW);
    v.outer = c.take<BGcr>(nrhs); v.smooth = c.take<BGcr>(nrhs); v.cgcr = c.take<BGcr>(nrhs);
    v.bn2 = c.take<double>(nrhs); v.rn2 = c.take<double>(nrhs); v.rA2 = c.take<double>(nrhs);
    v.ref2 = c.take<double>(nrhs); v.cref2 = c.take<double>(nrhs); v.scale = c.take<double>(nrhs);
    v.rn = c.take<double>(nrhs);
    v.pg_part = c.take<double>(64 * 1024);
    v.pg_rr2 = c.take<double>(1);
    // from here on the arena is zeroed once at allocation (counters must start at 0)
    c.off = (c.off + 255) & ~(size_t)255;
    *zero_begin = c.off;
    v.mcount = c.take<unsigned>((size_t)nrhs * BK_MAX * CROW);
    v.red.counter = c.take<unsigned>((size_t)nrhs * CROW);
    v.odone = c.take<int>(nrhs); v.idone = c.take<int>(nrhs); v.cdone = c.take<int>(nrhs);
    v.iters = c.take<int>(nrhs); v.citers = c.take<int>(nrhs); v.csteps = c.take<int>(nrhs);
    v.pg_bar = c.take<unsigned>(4);
    v.pg_iters = c.take<int>(1);
    *zero_end = c.off;
    *total = c.off;
}

struct BatchedState {
    void* arena = nullptr;
    int cap = 0;
    BView v{};
    int* hflags = nullptr;            // pinned: odone, idone, cdone, iters, citers [5][cap], + 2 spare
    double* hvals = nullptr;          // pinned: bn2, rn2, rA2, ref2, scale, rn [6][cap]
    cudaGraphExec_t gfirst = nullptr, gcycle = nullptr;
    int gnrhs = 0;                    // right-hand sides the graphs were captured for
    int cycles = 1;                   // restart cycles the last coarse solve took (launched ahead of the first check)
    ~BatchedState() {
        if (gfirst) cudaGraphExecDestroy(gfirst);
        if (gcycle) cudaGraphExecDestroy(gcycle);
        if (arena) cudaFree(arena);
        if (hflags) cudaFreeHost(hflags);
        if (hvals) cudaFreeHost(hvals);
    }
};

static dwf_status ensure_batched(dwf_mg* h, int nrhs) {
    BatchedState*& bs = reinterpret_cast<BatchedState*&>(h->batched);
    if (bs && bs->cap >= nrhs) {
        if (bs->v.nrhs != nrhs) {
            size_t total, z0, z1;
            carve(h, nrhs, (char*)bs->arena, bs->v, &total, &z0, &z1);
            // a different row count moves the carved regions: zero the counters and flags again
            DWF_CHECK_CUDA(cudaStreamSynchronize(h->st));
            DWF_CHECK_CUDA(cudaMemset((char*)bs->arena + z0, 0, z1 - z0));
        }
    } else {
        if (bs) {
            cudaStreamSynchronize(h->st);
            delete bs;
            bs = nullptr;
        }
        BatchedState* n = new (std::nothrow) BatchedState();
        if (!n) { set_error("host allocation failed"); return DWF_ERR_OOM; }
        size_t total, z0, z1;
        carve(h, nrhs, nullptr, n->v, &total, &z0, &z1);
        cudaError_t e = cudaMalloc(&n->arena, total);
        if (e != cudaSuccess) {
            delete n;
            set_error("batched solver workspace of %zu bytes: %s", total, cudaGetErrorString(e));
            return DWF_ERR_OOM;
        }
        carve(h, nrhs, (char*)n->arena, n->v, &total, &z0, &z1);
        if (cudaMemset((char*)n->arena + z0, 0, z1 - z0) != cudaSuccess ||
            cudaMallocHost((void**)&n->hflags, (5 * nrhs + 2) * sizeof(int)) != cudaSuccess ||
            cudaMallocHost((void**)&n->hvals, 6 * sizeof(double) * nrhs) != cudaSuccess) {
            delete n;
            set_error("batched solver workspace setup failed");
            return DWF_ERR_OOM;
        }
        n->cap = nrhs;
        bs = n;
    }
    BView& v = bs->v;
    float2* hp[6 * BK_MAX];
    for (int k = 0; k < BK_MAX; ++k) {
        hp[0 * BK_MAX + k] = v.Z[k]; hp[1 * BK_MAX + k] = v.W[k];
        hp[2 * BK_MAX + k] = v.Ps[k]; hp[3 * BK_MAX + k] = v.Qs[k];
        hp[4 * BK_MAX + k] = v.Zc[k]; hp[5 * BK_MAX + k] = v.Wc[k];
    }
    DWF_CHECK_CUDA(cudaMemcpy(v.dptr, hp, sizeof(hp), cudaMemcpyHostToDevice));
    if (bs->gnrhs != nrhs) {
        if (bs->gfirst) cudaGraphExecDestroy(bs->gfirst);
        if (bs->gcycle) cudaGraphExecDestroy(bs->gcycle);
        bs->gfirst = bs->gcycle = nullptr;
        bs->gnrhs = 0;
    }
    return DWF_OK;
}

// --------------------------------------------------------------------------
// solver
// --------------------------------------------------------------------------
struct BSolver {
    dwf_mg* h;
    BatchedState* bs;
    BView* v;
    cudaStream_t st;
    int nrhs;
    bool pk = false;             // FP32 fine vectors in the slice-paired layout (4-d, one right-hand side)
    long long l3_iters = 0;      // coarsest iterations of a three-level hierarchy
    long long l3_solves = 0;     // and coarsest solves
};

static dim3 row_grid(long long n2, int nrhs, int cap) {
    long long b = (n2 + 255) / 256;
    if (b < 1) b = 1;
    if (b > cap) b = cap;
    return dim3((unsigned)b, (unsigned)nrhs);
}

static dwf_status bapply_A(BSolver& s, const float2* in, float2* out, const int* skip) {
    dwf_mg* h = s.h;
    if (s.pk) {
        DWF_TRY(fine_apply_4d_paired(h->G, h->Upk, in, s.v->tmp, h->M5, h->mf, false, h->prm.fine_prec, s.st, skip));
        return fine_apply_4d_paired(h->G, h->Upk, s.v->tmp, out, h->M5, 1.0, true, h->prm.fine_prec, s.st, skip);
    }
    DWF_TRY(fine_apply_rhs(h->G, h->Ulo, in, s.v->tmp, h->M5, h->mf, false, h->prm.fine_prec, s.nrhs, skip, s.st));
    DWF_TRY(fine_apply_rhs(h->G, h->Ulo, s.v->tmp, out, h->M5, 1.0, true, h->prm.fine_prec, s.nrhs, skip, s.st));
    return DWF_OK;
}

// Orthogonalise Wb[k] against Wb[0..k-1] (classical Gram-Schmidt, cgs_passes
// passes), then nrm[k], alpha = A[k] = <w, res> / |w|^2; steps[r] = k + 1.
static dwf_status borthogonalise(BSolver& s, BGcr* g, float2* const* Wb, int k, const float2* res, long long n,
                                 float2* const* dW, int* steps, const int* skip) {
    BView& v = *s.v;
    const int rg = red_grid4(n);
    const dim3 rgrid((unsigned)rg, (unsigned)s.nrhs);
    if (k > 0) {
        const bool fused = n >= BMDOT_FUSE_N;
        const int nb = fused ? BMDOT_BLOCKS : BMDOT_ROW_BLOCKS;
        const dim3 mgrid((unsigned)(rg < nb ? rg : nb), fused ? (unsigned)s.nrhs : (unsigned)k,
                         fused ? 1u : (unsigned)s.nrhs);
        const dim3 egrid = row_grid(n >> 1, s.nrhs, 152 * 16);
        const int passes = s.h->prm.cgs_passes;
        for (int pass = 0; pass < passes; ++pass) {
            if (fused) launch_bmdot(mgrid, dW, Wb[k], n, k, v.mpart, v.mcount, g, pass == 0, skip, s.st);
            else k_bmdot_rows<<<mgrid, RED_THREADS, 0, s.st>>>(dW, Wb[k], n, v.mpart, v.mcount, g, pass == 0, skip);
            if (pass + 1 < passes)
                k_bmaxpy<false><<<egrid, RED_THREADS, 0, s.st>>>(Wb[k], dW, g, k, res, n, v.red, steps, skip);
            else
                k_bmaxpy<true><<<rgrid, RED_THREADS, 0, s.st>>>(Wb[k], dW, g, k, res, n, v.red, steps, skip);
        }
    } else {
        k_bmaxpy<true><<<rgrid, RED_THREADS, 0, s.st>>>(Wb[0], dW, g, 0, res, n, v.red, steps, skip);
    }
    DWF_CHECK_LAUNCH();
    return DWF_OK;
}

// Coarse GCR on every right-hand side with idone == 0 (cdone starts as a copy
// of idone).  The residual at the start of a restart cycle is crr; step k
// keeps its residual in Zc[k] (the raw direction of step k) and writes the
// next one to Zc[k + 1], or to crr after the last step; the cycle ends with
// ec += sum_j y_j Zc[j] over the csteps[r] steps that right-hand side took.
static dwf_status bcoarse_prologue(BSolver& s) {
    BView& v = *s.v;
    const long long n = v.nc;
    DWF_CHECK_CUDA(cudaMemsetAsync(v.ec, 0, (size_t)s.nrhs * n * sizeof(float2), s.st));
    DWF_CHECK_CUDA(cudaMemcpyAsync(v.crr, v.rc, (size_t)s.nrhs * n * sizeof(float2), cudaMemcpyDeviceToDevice, s.st));
    DWF_CHECK_CUDA(cudaMemcpyAsync(v.cdone, v.idone, s.nrhs * sizeof(int), cudaMemcpyDeviceToDevice, s.st));
    DWF_CHECK_CUDA(cudaMemsetAsync(v.citers, 0, s.nrhs * sizeof(int), s.st));
    k_bnorm2_32<<<dim3((unsigned)red_grid4(n), (unsigned)s.nrhs), RED_THREADS, 0, s.st>>>(v.rc, n, v.red, v.cref2,
                                                                                           v.idone);
    DWF_CHECK_LAUNCH();
    return DWF_OK;
}

static dwf_status bcoarse_cycle(BSolver& s) {
    dwf_mg* h = s.h;
    BView& v = *s.v;
    const long long n = v.nc;
    const int KC = h->prm.coarse_restart;
    const double tol2 = h->prm.coarse_tol * h->prm.coarse_tol;
    const dim3 eg = row_grid(n >> 1, s.nrhs);
    const dim3 rg((unsigned)red_grid4(n), (unsigned)s.nrhs);
    DWF_CHECK_CUDA(cudaMemsetAsync(v.csteps, 0, s.nrhs * sizeof(int), s.st));
    k_bcopy<<<eg, 256, 0, s.st>>>(v.Zc[0], v.crr, n, v.cdone);
    DWF_CHECK_LAUNCH();
    const bool blocks = h->prm.cgs_passes == 1;
    for (int k = 0; k < KC;) {
        const int m = !blocks ? 1 : KC - k < SB ? KC - k : SB;
        for (int i = 0; i < m; ++i) {
            float2* out = i + 1 < m ? v.Zc[k + i + 1] : v.Wc[k + m - 1];
            if (s.nrhs == 1) {
                // one column: the one-vector stencil has the shorter latency
                DWF_TRY(coarse_dwf_apply(h, v.Zc[k + i], v.ct, h->mf, false, v.cdone, s.st));
                DWF_TRY(coarse_dwf_apply(h, v.ct, out, 1.0, true, v.cdone, s.st));
            } else {
                DWF_TRY(coarse_apply_multi_tc(h, s.nrhs, v.Zc[k + i], v.ct, h->mf, false, v.cdone, s.st));
                DWF_TRY(coarse_apply_multi_tc(h, s.nrhs, v.ct, out, 1.0, true, v.cdone, s.st));
            }
        }
        float2* rnext = k + m < KC ? v.Zc[k + m] : v.crr;
        if (blocks) {
            DWF_TRY(bblock(v.cgcr, v.Zc, v.Wc, v.dptr + 5 * BK_MAX, k, m, k + m < KC, nullptr, rnext, n, s.nrhs, v.mpart,
                           v.mcount, v.cdone, v.csteps, v.cdone, v.cref2, tol2, v.citers, h->prm.coarse_maxiter,
                           s.st));
        } else {
            DWF_TRY(borthogonalise(s, v.cgcr, v.Wc, k, v.Zc[k], n, v.dptr + 5 * BK_MAX, v.csteps, v.cdone));
            k_bres_update<<<rg, RED_THREADS, 0, s.st>>>(v.Zc[k], rnext, v.Wc[k], v.cgcr, n, v.red, v.cdone, v.cdone,
                                                        v.cref2, tol2, v.citers, h->prm.coarse_maxiter);
        }
        DWF_CHECK_LAUNCH();
        k += m;
    }
    k_bcombine32<<<eg, RED_THREADS, 0, s.st>>>(v.ec, v.dptr + 4 * BK_MAX, v.cgcr, v.csteps, 0, n, nullptr, nullptr,
                                               nullptr, nullptr);
    DWF_CHECK_LAUNCH();
    return DWF_OK;
}

static dwf_status bcapture(BSolver& s, bool with_prologue, cudaGraphExec_t* out) {
    cudaGraph_t graph = nullptr;
    if (!s.h->cap_stream) DWF_CHECK_CUDA(cudaStreamCreateWithFlags(&s.h->cap_stream, cudaStreamNonBlocking));
    const cudaStream_t user = s.st;
    s.st = s.h->cap_stream;
    DWF_CHECK_CUDA(cudaStreamBeginCapture(s.st, cudaStreamCaptureModeThreadLocal));
    dwf_status st = DWF_OK;
    if (with_prologue) st = bcoarse_prologue(s);
    if (st == DWF_OK) st = bcoarse_cycle(s);
    cudaError_t e = cudaStreamEndCapture(s.st, &graph);
    s.st = user;
    if (st != DWF_OK) { if (graph) cudaGraphDestroy(graph); return st; }
    if (e != cudaSuccess) { set_error("graph capture: %s", cudaGetErrorString(e)); return DWF_ERR_CUDA; }
    e = cudaGraphInstantiate(out, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) { set_error("graph instantiation: %s", cudaGetErrorString(e)); return DWF_ERR_CUDA; }
    return DWF_OK;
}

// runs the coarse GCR until every active right-hand side is done; citers_out[r]
// receives the iterations of right-hand side r
static dwf_status bcoarse_solve(BSolver& s, int* citers_out) {
    dwf_mg* h = s.h;
    BatchedState* bs = s.bs;
    BView& v = *s.v;
    if (s.nrhs == 1 && h->prm.coarse_persistent == 2 && coarse_gcr_persistent_ok(h)) {
        // one right-hand side: the whole coarse GCR in one cooperative launch
        const int KC = h->prm.coarse_restart;
        float2* S[BK_MAX + 1];
        for (int k = 0; k < KC; ++k) S[k] = v.Zc[k];
        S[KC] = v.crr;
        DWF_CHECK_CUDA(cudaMemsetAsync(v.pg_iters, 0, sizeof(int), s.st));
        DWF_TRY(coarse_gcr_persistent(h, v.rc, v.ec, S, v.Wc, v.ct, v.pg_part, v.pg_bar, v.pg_iters, v.pg_rr2,
                                      s.st));
        unsigned* hb = reinterpret_cast<unsigned*>(bs->hflags + 5 * bs->cap);   // spare slot
        DWF_CHECK_CUDA(cudaMemcpyAsync(citers_out, v.pg_iters, sizeof(int), cudaMemcpyDeviceToHost, s.st));
        DWF_CHECK_CUDA(cudaMemcpyAsync(hb, v.pg_bar + 2, sizeof(unsigned), cudaMemcpyDeviceToHost, s.st));
        DWF_CHECK_CUDA(cudaStreamSynchronize(s.st));
        if (*hb != 0u) { set_error("persistent coarse GCR: a grid barrier or bulk copy timed out"); return DWF_ERR_TIMEOUT; }
        return DWF_OK;
    }
    if (!bs->gfirst) {
        // the contraction's form is chosen by timing, before it is frozen into the graphs
        if (s.nrhs > 1 && h->prm.coarse_tc == 0) DWF_TRY(coarse_tc_tune(h, s.nrhs, v.Zc[0], v.ct, s.st));
        DWF_TRY(bcapture(s, true, &bs->gfirst));
        DWF_TRY(bcapture(s, false, &bs->gcycle));
        bs->gnrhs = s.nrhs;
    }
    // As many restart cycles as the last solve took are launched before the host looks: a check costs about 25 us
    // (the copy, the wait and the next launch), and a cycle past the end about as much (every kernel of it
    // returns at once), while consecutive solves take 3 or 4 cycles each: 256^2 x 16 gradient step 522 -> 494 ms.
    int* hcd = bs->hflags + 2 * bs->cap;
    int launched = 0;
    for (;;) {
        const int n = launched == 0 ? bs->cycles : 1;
        for (int i = 0; i < n && (launched == 0 || launched < h->prm.coarse_maxiter); ++i) {
            DWF_CHECK_CUDA(cudaGraphLaunch(launched == 0 ? bs->gfirst : bs->gcycle, s.st));
            launched += h->prm.coarse_restart;
        }
        DWF_CHECK_CUDA(cudaMemcpyAsync(hcd, v.cdone, s.nrhs * sizeof(int), cudaMemcpyDeviceToHost, s.st));
        DWF_CHECK_CUDA(cudaMemcpyAsync(citers_out, v.citers, s.nrhs * sizeof(int), cudaMemcpyDeviceToHost, s.st));
        DWF_CHECK_CUDA(cudaStreamSynchronize(s.st));
        bool all = true;
        for (int r = 0; r < s.nrhs; ++r) all = all && hcd[r];
        if (all || launched >= h->prm.coarse_maxiter) break;
    }
    int most = 1;
    for (int r = 0; r < s.nrhs; ++r) most = std::max(most, citers_out[r]);
    bs->cycles = (most + h->prm.coarse_restart - 1) / h->prm.coarse_restart;
    return DWF_OK;
}

// z = M(r) and w = A z for every right-hand side with idone == 0.  With two
// Gram-Schmidt passes the smoother's step j keeps its residual in Ps[j] and writes the next one to
// Ps[j + 1] (rs_ after the last step); z += sum_j y_j Ps[j] and w = r - rs_
// come out of one final pass.
static dwf_status bprecondition(BSolver& s, const float2* res, float2* zout, float2* wout, int* citers_out) {
    dwf_mg* h = s.h;
    BView& v = *s.v;
    const long long n = v.nf;
    const dim3 eg = row_grid(n >> 1, s.nrhs);
    DWF_TRY(restrict_wall(h, res, v.rc, v.idone, s.st, s.nrhs, s.pk));
    if (h->lvl3) {
        // three levels: flexible GCR on the intermediate level, preconditioned by the coarsest solve
        int l2 = 0, l3 = 0;
        DWF_TRY(level2_solve(h, v.rc, v.ec, &l2, &l3, s.st));
        citers_out[0] = l2;
        s.l3_iters += l3;
        s.l3_solves += l2;
    } else {
        DWF_TRY(bcoarse_solve(s, citers_out));
    }
    DWF_TRY(prolong_wall(h, v.ec, zout, v.idone, s.st, s.nrhs, s.pk));
    const int S = h->prm.post_smooth;
    if (S == 0) return bapply_A(s, zout, wout, v.idone);
    DWF_TRY(bapply_A(s, zout, v.ps, v.idone));
    k_bsub32<<<eg, 256, 0, s.st>>>(v.Ps[0], res, v.ps, n, v.idone);
    DWF_CHECK_LAUNCH();
    if (h->prm.cgs_passes == 1) {
        // blocks of steps; the last one leaves w = r - rs_ in place of the residual rs_
        for (int j = 0; j < S;) {
            const int m = S - j < SB ? S - j : SB;
            for (int i = 0; i < m; ++i)
                DWF_TRY(bapply_A(s, v.Ps[j + i], i + 1 < m ? v.Ps[j + i + 1] : v.Qs[j + m - 1], v.idone));
            const bool last = j + m == S;
            DWF_TRY(bblock(v.smooth, v.Ps, v.Qs, v.dptr + 3 * BK_MAX, j, m, !last, last ? res : nullptr,
                           last ? wout : v.Ps[j + m], n, s.nrhs, v.mpart, v.mcount, v.idone, nullptr, nullptr, nullptr,
                           0.0, nullptr, 0, s.st));
            j += m;
        }
        k_bcombine32<<<eg, RED_THREADS, 0, s.st>>>(zout, v.dptr + 2 * BK_MAX, v.smooth, nullptr, S, n, nullptr, nullptr,
                                                   nullptr, v.idone);
        DWF_CHECK_LAUNCH();
        return DWF_OK;
    }
    const dim3 rg((unsigned)red_grid4(n), (unsigned)s.nrhs);
    for (int j = 0; j < S; ++j) {
        DWF_TRY(bapply_A(s, v.Ps[j], v.Qs[j], v.idone));
        DWF_TRY(borthogonalise(s, v.smooth, v.Qs, j, v.Ps[j], n, v.dptr + 3 * BK_MAX, nullptr, v.idone));
        k_bres_update<<<rg, RED_THREADS, 0, s.st>>>(v.Ps[j], j + 1 < S ? v.Ps[j + 1] : v.rs_, v.Qs[j], v.smooth, n,
                                                    v.red, v.idone, nullptr, nullptr, 0.0, nullptr, 0);
        DWF_CHECK_LAUNCH();
    }
    k_bcombine32<<<eg, RED_THREADS, 0, s.st>>>(zout, v.dptr + 2 * BK_MAX, v.smooth, nullptr, S, n, res, v.rs_, wout,
                                               v.idone);
    DWF_CHECK_LAUNCH();
    return DWF_OK;
}

}  // namespace

void batched_state_free(dwf_mg* h) {
    if (h && h->batched) {
        delete reinterpret_cast<BatchedState*>(h->batched);
        h->batched = nullptr;
    }
}

dwf_status mg_solve_batched_impl(dwf_mg* h, int nrhs, const double2* B, double2* X, double tol, int maxiter,
                                 dwf_solve_stats* stats) {
    auto t0 = std::chrono::steady_clock::now();
    if (stats) memset(stats, 0, sizeof(*stats) * (size_t)(nrhs > 0 ? nrhs : 0));
    if (!h || !B || !X) { set_error("NULL argument"); return DWF_ERR_ARG; }
    if (nrhs < 1 || nrhs > 65535) { set_error("nrhs must be in [1, 65535]"); return DWF_ERR_ARG; }
    if (!(tol > 0.0)) { set_error("tol must be > 0"); return DWF_ERR_ARG; }
    if (nrhs > 1 && h->lvl3) {
        set_error("a three-level hierarchy solves one right-hand side per call");
        return DWF_ERR_UNSUPPORTED;
    }
    if (nrhs > 1 && (h->mg.nd != 2 || h->mg.ncd != 16)) {
        set_error("more than one right-hand side per hierarchy needs a 2-d lattice with nvec = 8");
        return DWF_ERR_UNSUPPORTED;
    }
    if (h->prm.gcr_restart < 1 || h->prm.gcr_restart > BK_MAX || h->prm.post_smooth > BK_MAX ||
        h->prm.coarse_restart < 1 || h->prm.coarse_restart > BK_MAX) {
        set_error("gcr_restart, post_smooth and coarse_restart must be in [1, %d]", BK_MAX); return DWF_ERR_ARG;
    }
    DWF_TRY(ensure_batched(h, nrhs));
    BSolver s;
    s.h = h;
    s.bs = reinterpret_cast<BatchedState*>(h->batched);
    s.v = &s.bs->v;
    s.st = h->st;
    s.nrhs = nrhs;
    s.pk = h->pk != 0 && nrhs == 1;
    const PackIdx pq{h->G.V, (h->G.V + 31) / 32, (int)site_dof(h->G)};
    BView& v = *s.v;
    BatchedState& bs = *s.bs;
    const long long n = v.nf;
    const int cap = bs.cap;
    int* hod = bs.hflags;             // odone
    int* hid = bs.hflags + cap;       // idone
    int* hit = bs.hflags + 3 * cap;   // iters
    int* hci = bs.hflags + 4 * cap;   // coarse iterations of the last coarse solve
    double* hbn2 = bs.hvals;
    double* hrn2 = bs.hvals + cap;
    double* hrA2 = bs.hvals + 2 * cap;
    double* href2 = bs.hvals + 3 * cap;
    double* hscale = bs.hvals + 4 * cap;
    double* hrn = bs.hvals + 5 * cap;
    const dim3 eg64 = row_grid(n, nrhs);
    const dim3 eg32 = row_grid(n >> 1, nrhs);
    const dim3 rg64((unsigned)red_grid(n), (unsigned)nrhs);
    const dim3 rg32((unsigned)red_grid4(n), (unsigned)nrhs);

    DWF_CHECK_CUDA(cudaMemsetAsync(X, 0, (size_t)nrhs * n * sizeof(double2), s.st));
    k_bnorm2_64<<<rg64, RED_THREADS, 0, s.st>>>(B, n, v.red, v.bn2, nullptr);
    DWF_CHECK_LAUNCH();
    DWF_CHECK_CUDA(cudaMemcpyAsync(hbn2, v.bn2, nrhs * sizeof(double), cudaMemcpyDeviceToHost, s.st));
    DWF_CHECK_CUDA(cudaStreamSynchronize(s.st));

    std::vector<int> outer(nrhs, 0), restarts(nrhs, 0), conv(nrhs, 0);
    std::vector<long long> fine(nrhs, 0), coarse_it(nrhs, 0), coarse_solves(nrhs, 0);
    std::vector<double> res(nrhs, 1.0);
    for (int r = 0; r < nrhs; ++r) {
        hod[r] = 0;
        if (hbn2[r] == 0.0) { hod[r] = 1; conv[r] = 1; res[r] = 0.0; }
    }
    const int K = h->prm.gcr_restart, S = h->prm.post_smooth;
    bool first = true;
    for (;;) {
        if (first) {
            DWF_CHECK_CUDA(cudaMemcpyAsync(v.r64, B, (size_t)nrhs * n * sizeof(double2), cudaMemcpyDeviceToDevice,
                                           s.st));
            for (int r = 0; r < nrhs; ++r) hrn2[r] = hbn2[r];
            first = false;
        } else {
            DWF_CHECK_CUDA(cudaMemcpyAsync(v.odone, hod, nrhs * sizeof(int), cudaMemcpyHostToDevice, s.st));
            DWF_TRY(fine_apply_rhs(h->G, h->U64, X, v.t64, h->M5, h->mf, false, DWF_F64, nrhs, v.odone, s.st));
            k_bsub64<<<eg64, 256, 0, s.st>>>(v.r64, B, v.t64, n, v.odone);
            k_bnorm2_64<<<rg64, RED_THREADS, 0, s.st>>>(v.r64, n, v.red, v.rn2, v.odone);
            DWF_CHECK_LAUNCH();
            DWF_CHECK_CUDA(cudaMemcpyAsync(hrn2, v.rn2, nrhs * sizeof(double), cudaMemcpyDeviceToHost, s.st));
            DWF_CHECK_CUDA(cudaStreamSynchronize(s.st));
            for (int r = 0; r < nrhs; ++r) if (!hod[r]) fine[r] += 1;
        }
        bool any = false;
        for (int r = 0; r < nrhs; ++r) {
            if (hod[r]) continue;
            res[r] = sqrt(hrn2[r] / hbn2[r]);
            if (res[r] <= tol) { hod[r] = 1; conv[r] = 1; continue; }
            if (outer[r] >= maxiter || restarts[r] > h->prm.max_restarts) { hod[r] = 1; continue; }
            any = true;
        }
        if (!any) break;
        for (int r = 0; r < nrhs; ++r) {
            hid[r] = hod[r];
            hrn[r] = hod[r] ? 0.0 : sqrt(hrn2[r]);
            hscale[r] = hod[r] ? 0.0 : 1.0 / hrn[r];
            if (!hod[r]) { restarts[r] += 1; fine[r] += 1; }
        }
        DWF_CHECK_CUDA(cudaMemcpyAsync(v.odone, hod, nrhs * sizeof(int), cudaMemcpyHostToDevice, s.st));
        DWF_CHECK_CUDA(cudaMemcpyAsync(v.idone, hid, nrhs * sizeof(int), cudaMemcpyHostToDevice, s.st));
        DWF_CHECK_CUDA(cudaMemcpyAsync(v.scale, hscale, nrhs * sizeof(double), cudaMemcpyHostToDevice, s.st));
        DWF_CHECK_CUDA(cudaMemcpyAsync(v.rn, hrn, nrhs * sizeof(double), cudaMemcpyHostToDevice, s.st));
        // correction system in FP32: A e = D_PV^dag r / |r|
        if (s.pk) {
            k_bd2f_scale_pk<<<eg32, 256, 0, s.st>>>(v.ps, v.r64, v.scale, n, v.idone, pq);
            DWF_CHECK_LAUNCH();
            DWF_TRY(fine_apply_4d_paired(h->G, h->Upk, v.ps, v.rA, h->M5, 1.0, true, h->prm.fine_prec, s.st, v.idone));
        } else {
            k_bd2f_scale<<<eg64, 256, 0, s.st>>>(v.ps, v.r64, v.scale, n, v.idone);
            DWF_CHECK_LAUNCH();
            DWF_TRY(fine_apply_rhs(h->G, h->Ulo, v.ps, v.rA, h->M5, 1.0, true, h->prm.fine_prec, nrhs, v.idone, s.st));
        }
        k_bcopy<<<eg32, 256, 0, s.st>>>(v.r, v.rA, n, v.idone);
        k_bnorm2_32<<<rg32, RED_THREADS, 0, s.st>>>(v.rA, n, v.red, v.rA2, v.idone);
        DWF_CHECK_LAUNCH();
        DWF_CHECK_CUDA(cudaMemcpyAsync(hrA2, v.rA2, nrhs * sizeof(double), cudaMemcpyDeviceToHost, s.st));
        DWF_CHECK_CUDA(cudaStreamSynchronize(s.st));
        for (int r = 0; r < nrhs; ++r) {
            if (hid[r]) { href2[r] = 0.0; continue; }
            double delta = h->prm.inner_tol;
            const double need = 0.5 * tol * sqrt(hbn2[r]) / hrn[r];
            if (need > delta) delta = need;
            href2[r] = delta * delta * hrA2[r];
        }
        DWF_CHECK_CUDA(cudaMemcpyAsync(v.ref2, href2, nrhs * sizeof(double), cudaMemcpyHostToDevice, s.st));
        DWF_CHECK_CUDA(cudaMemsetAsync(v.iters, 0, nrhs * sizeof(int), s.st));
        const dim3 rg((unsigned)red_grid4(n), (unsigned)nrhs);
        for (int k = 0; k < K; ++k) {
            bool active = false;
            for (int r = 0; r < nrhs; ++r) active = active || !hid[r];
            if (!active) break;
            DWF_TRY(bprecondition(s, v.r, v.Z[k], v.W[k], hci));
            for (int r = 0; r < nrhs; ++r)
                if (!hid[r]) { coarse_it[r] += hci[r]; coarse_solves[r] += 1; fine[r] += 2 + 2 * S; outer[r] += 1; }
            DWF_TRY(borthogonalise(s, v.outer, v.W, k, v.r, n, v.dptr + 1 * BK_MAX, nullptr, v.idone));
            k_bres_update<<<rg, RED_THREADS, 0, s.st>>>(v.r, v.r, v.W[k], v.outer, n, v.red, v.idone, v.idone,
                                                        v.ref2, 1.0, v.iters, K);
            DWF_CHECK_LAUNCH();
            DWF_CHECK_CUDA(cudaMemcpyAsync(hid, v.idone, nrhs * sizeof(int), cudaMemcpyDeviceToHost, s.st));
            DWF_CHECK_CUDA(cudaStreamSynchronize(s.st));
            for (int r = 0; r < nrhs; ++r)
                if (!hod[r] && outer[r] >= maxiter) hid[r] = 1;    // iteration cap: leave the cycle
            DWF_CHECK_CUDA(cudaMemcpyAsync(v.idone, hid, nrhs * sizeof(int), cudaMemcpyHostToDevice, s.st));
        }
        // x += |r| sum_k y_k Z_k over the iters[r] steps of this cycle
        if (s.pk)
            k_bcombine64_pk<<<row_grid(n >> 1, 1), RED_THREADS, 0, s.st>>>(X, v.dptr + 0 * BK_MAX, v.outer, v.iters,
                                                                            v.rn, n, pq);
        else
            k_bcombine64<<<row_grid(n >> 1, nrhs), RED_THREADS, 0, s.st>>>(X, v.dptr + 0 * BK_MAX, v.outer, v.iters,
                                                                            v.rn, n);
        DWF_CHECK_LAUNCH();
    }
    (void)hit;
    DWF_TRY(coarse_wait_status(h, s.st));
    int nconv = 0;
    for (int r = 0; r < nrhs; ++r) nconv += conv[r];
    const double secs = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    if (stats)
        for (int r = 0; r < nrhs; ++r) {
            stats[r].iterations = outer[r];
            stats[r].restarts = restarts[r];
            stats[r].fine_applies = fine[r];
            stats[r].coarse_applies = 2 * coarse_it[r];
            stats[r].coarse_avg_iters = coarse_solves[r] ? (double)coarse_it[r] / coarse_solves[r] : 0.0;
            stats[r].coarsest_avg_iters = s.l3_solves ? (double)s.l3_iters / s.l3_solves : 0.0;
            stats[r].true_residual = res[r];
            stats[r].seconds = secs;
        }
    if (nconv < nrhs) {
        double worst = 0.0;
        for (int r = 0; r < nrhs; ++r) if (!conv[r] && res[r] > worst) worst = res[r];
        set_error("mg_solve_batched: %d of %d right-hand sides stopped above tol %.3e (worst %.3e)", nrhs - nconv,
                  nrhs, tol, worst);
        return DWF_ERR_NOCONV;
    }
    return DWF_OK;
}

}  // namespace dwf

using namespace dwf;

extern "C" dwf_status mg_solve_batched(dwf_mg* h, int nrhs, const void* b, void* x, double tol, int maxiter,
                                       dwf_solve_stats* stats, void* stream) {
    clear_error();
    if (h && stream) h->st = as_stream(stream);
    return mg_solve_batched_impl(h, nrhs, (const double2*)b, (double2*)x, tol, maxiter, stats);
}

extern "C" dwf_status mg_solve_groups(int ngroups, dwf_mg* const* handles, const int* nrhs, const void* const* b,
                                      void* const* x, double tol, int maxiter, dwf_solve_stats* const* stats) {
    clear_error();
    if (ngroups < 1 || !handles || !nrhs || !b || !x) { set_error("NULL argument or ngroups < 1"); return DWF_ERR_ARG; }
    for (int i = 0; i < ngroups; ++i) {
        if (!handles[i]) { set_error("handle %d is NULL", i); return DWF_ERR_ARG; }
        for (int j = 0; j < i; ++j)
            if (handles[j] == handles[i]) { set_error("handles %d and %d are the same hierarchy", j, i); return DWF_ERR_ARG; }
    }
    // each hierarchy gets its own non-blocking stream and host thread, so the
    // groups' launches overlap on the device
    std::vector<cudaStream_t> streams(ngroups, nullptr);
    std::vector<cudaStream_t> saved(ngroups, nullptr);
    for (int i = 0; i < ngroups; ++i) {
        if (cudaStreamCreateWithFlags(&streams[i], cudaStreamNonBlocking) != cudaSuccess) {
            for (int j = 0; j < i; ++j) cudaStreamDestroy(streams[j]);
            set_error("stream creation failed");
            return DWF_ERR_CUDA;
        }
        saved[i] = handles[i]->st;
    }
    // the caller's prior work on the handles' streams must be complete
    for (int i = 0; i < ngroups; ++i) cudaStreamSynchronize(saved[i]);
    std::vector<dwf_status> st(ngroups, DWF_OK);
    std::vector<std::string> msg(ngroups);
    int dev = 0;
    cudaGetDevice(&dev);
    std::vector<std::thread> th;
    for (int i = 0; i < ngroups; ++i) {
        th.emplace_back([&, i]() {
            cudaSetDevice(dev);
            handles[i]->st = streams[i];
            st[i] = mg_solve_batched_impl(handles[i], nrhs[i], (const double2*)b[i], (double2*)x[i], tol, maxiter,
                                          stats ? stats[i] : nullptr);
            if (st[i] != DWF_OK) msg[i] = dwf_last_error();
            cudaStreamSynchronize(streams[i]);
        });
    }
    for (auto& t : th) t.join();
    dwf_status out = DWF_OK;
    for (int i = 0; i < ngroups; ++i) {
        handles[i]->st = saved[i];
        cudaStreamDestroy(streams[i]);
        if (st[i] != DWF_OK && out == DWF_OK) {
            out = st[i];
            set_error("group %d: %s", i, msg[i].c_str());
        }
    }
    return out;
}
