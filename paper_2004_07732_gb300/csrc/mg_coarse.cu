// Coarse-level operators of the multigrid (Sec. 2.3):
//   * the coarse Shamir operator Dhat_DW(m) of Eq. coarsenDW: on every coarse
//     slice the Galerkin kernel Dhat_W (self block + one block per hop
//     direction) plus 1, the Phat_pm = (1 pm sigma_3)/2 s-hops and the -m wall
//     terms; the adjoint uses the transposed neighbour blocks, so it is the
//     exact adjoint of the stored operator;
//   * truncated wall restriction / prolongation (Eq. TruncProjectInterpolate).
// Coarse vectors are [s][coarse site][chirality][vec], complex64.
#include <algorithm>
#include <mutex>

#include "mg.cuh"
#include "async_copy.cuh"
#include "mma_f16.cuh"

namespace dwf {

__device__ __forceinline__ long long coarse_neighbour(const CoarseParams& p, long long xc, int dir) {
    if (dir == 0) return xc;
    const int mu = (dir - 1) >> 1;
    const int step = ((dir - 1) & 1) ? -1 : 1;
    // extent and stride of direction mu without indexing the parameter arrays dynamically
    const long long L0 = p.Lc[0], L1 = p.Lc[1], L2 = p.Lc[2], L3 = p.Lc[3];
    const long long Lm = mu == 0 ? L0 : mu == 1 ? L1 : mu == 2 ? L2 : L3;
    const long long stride = mu == 0 ? 1 : mu == 1 ? L0 : mu == 2 ? L0 * L1 : L0 * L1 * L2;
    const long long c = (xc / stride) % Lm;
    long long cn = c + step;
    if (cn < 0) cn += Lm;
    if (cn >= Lm) cn -= Lm;
    return xc + (cn - c) * stride;
}

__device__ __forceinline__ float2 cfma(float2 a, float2 b, float2 acc) {
    acc.x = fmaf(a.x, b.x, fmaf(-a.y, b.y, acc.x));
    acc.y = fmaf(a.x, b.y, fmaf(a.y, b.x, acc.y));
    return acc;
}
__device__ __forceinline__ float2 cfma_conj(float2 a, float2 b, float2 acc) {   // conj(a) * b
    acc.x = fmaf(a.x, b.x, fmaf(a.y, b.y, acc.x));
    acc.y = fmaf(a.x, b.y, fmaf(-a.y, b.x, acc.y));
    return acc;
}

// One warp per coarse site.  B holds (2 nvec)^2 blocks column-major per
// [coarse site][dir]: the Galerkin blocks of Dhat_W for the operator, or the
// pre-transposed blocks of Dhat_W^dag (block (x, dir) = Y(x + dir, -dir)^dag)
// for the adjoint, so both read B coalesced.  Lane l owns rows
// i = (l & 15) + 16 k and slices s = 8 g + (l >> 4) + 2 k' (g = 0, 1, .. for Ls_c > 8); the j loop is unrolled so
// every block and input load of a direction is in flight together.  CG = true
// reads the input through L2 (other blocks of a persistent launch wrote it).
// Returns the lane's share of |out|^2.
template <int NCD, bool CG>
__device__ __forceinline__ double warp_site_apply(const float2* __restrict__ B, const float2* __restrict__ in,
                                                  float2* __restrict__ out, const CoarseParams& p, long long xc,
                                                  float mf, bool dag, int lane) {
    const int ncd = NCD > 0 ? NCD : p.ncd;
    const long long slice = p.Vc * ncd;
    const long long bsz = (long long)ncd * ncd;
    const int sg = lane >> 4;
    double nrm = 0.0;
    // slices in groups of 8 (the blocks of a later group come from L1/L2)
    for (int s0 = 0; s0 < p.Ls_c; s0 += 8)
    for (int i = lane & 15; i < ncd; i += 16) {
        float2 acc[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int s = s0 + sg + 2 * k;
            acc[k] = make_float2(0.f, 0.f);
            if (s < p.Ls_c) acc[k] = CG ? __ldcg(in + s * slice + xc * ncd + i) : __ldg(in + s * slice + xc * ncd + i);
        }
        for (int dir = 0; dir < p.ndir; ++dir) {
            const long long nb = coarse_neighbour(p, xc, dir);
            const float2* Bb = B + (xc * p.ndir + dir) * bsz + i;
            const float2* v = in + nb * ncd;
#pragma unroll
            for (int j = 0; j < ncd; ++j) {
                const float2 y = __ldg(Bb + (long long)j * ncd);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int s = s0 + sg + 2 * k;
                    if (s < p.Ls_c) acc[k] = cfma(y, CG ? __ldcg(v + s * slice + j) : __ldg(v + s * slice + j), acc[k]);
                }
            }
        }
        const int c = i / p.nvec;
        const bool from_below = dag ? (c == 1) : (c == 0);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int s = s0 + sg + 2 * k;
            if (s >= p.Ls_c) break;
            long long hi;
            float sc = 1.f;
            if (from_below) { if (s > 0) hi = (s - 1) * slice; else { hi = (p.Ls_c - 1) * slice; sc = -mf; } }
            else            { if (s < p.Ls_c - 1) hi = (s + 1) * slice; else { hi = 0; sc = -mf; } }
            const float2 h = CG ? __ldcg(in + hi + xc * ncd + i) : __ldg(in + hi + xc * ncd + i);
            acc[k].x += sc * h.x;
            acc[k].y += sc * h.y;
            out[s * slice + xc * ncd + i] = acc[k];
            nrm += (double)acc[k].x * acc[k].x + (double)acc[k].y * acc[k].y;
        }
    }
    return nrm;
}

// Specialisation for 2 nvec = 16 coarse dof and Ls_c <= 4: lane i = l & 15,
// slices sg = l >> 4 and sg + 2.  For each direction all 16 block columns and
// both 16-value input rows are loaded into registers before any arithmetic
// (the inputs as 128-bit broadcast loads), so a warp keeps 32 loads in flight.
template <bool CG>
__device__ __forceinline__ float4 ld4(const float2* p) {
    return CG ? __ldcg(reinterpret_cast<const float4*>(p)) : __ldg(reinterpret_cast<const float4*>(p));
}

template <bool CG>
__device__ __forceinline__ double warp_site16(const float2* __restrict__ B, const float2* __restrict__ in,
                                              float2* __restrict__ out, const CoarseParams& p, long long xc, float mf,
                                              bool dag, int lane) {
    const long long slice = p.Vc * 16;
    const int i = lane & 15, sg = lane >> 4;
    const bool h0 = sg < p.Ls_c, h1 = sg + 2 < p.Ls_c;
    const int s0 = h0 ? sg : 0, s1 = h1 ? sg + 2 : 0;
    float2 acc0 = CG ? __ldcg(in + s0 * slice + xc * 16 + i) : __ldg(in + s0 * slice + xc * 16 + i);
    float2 acc1 = CG ? __ldcg(in + s1 * slice + xc * 16 + i) : __ldg(in + s1 * slice + xc * 16 + i);
    for (int dir = 0; dir < p.ndir; ++dir) {
        const long long nb = coarse_neighbour(p, xc, dir);
        const float2* Bb = B + (xc * p.ndir + dir) * 256 + i;
        const float2* va = in + s0 * slice + nb * 16;
        const float2* vb = in + s1 * slice + nb * 16;
        float2 y[16];
        float4 a[8], b[8];
#pragma unroll
        for (int j = 0; j < 16; ++j) y[j] = __ldg(Bb + j * 16);
#pragma unroll
        for (int m = 0; m < 8; ++m) a[m] = ld4<CG>(va + 2 * m);
#pragma unroll
        for (int m = 0; m < 8; ++m) b[m] = ld4<CG>(vb + 2 * m);
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            acc0 = cfma(y[2 * m], make_float2(a[m].x, a[m].y), acc0);
            acc0 = cfma(y[2 * m + 1], make_float2(a[m].z, a[m].w), acc0);
            acc1 = cfma(y[2 * m], make_float2(b[m].x, b[m].y), acc1);
            acc1 = cfma(y[2 * m + 1], make_float2(b[m].z, b[m].w), acc1);
        }
    }
    const int c = i / p.nvec;
    const bool from_below = dag ? (c == 1) : (c == 0);
    double nrm = 0.0;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const bool has = k == 0 ? h0 : h1;
        if (!has) continue;
        const int s = k == 0 ? s0 : s1;
        float2 acc = k == 0 ? acc0 : acc1;
        long long hi;
        float sc = 1.f;
        if (from_below) { if (s > 0) hi = (s - 1) * slice; else { hi = (p.Ls_c - 1) * slice; sc = -mf; } }
        else            { if (s < p.Ls_c - 1) hi = (s + 1) * slice; else { hi = 0; sc = -mf; } }
        const float2 hv = CG ? __ldcg(in + hi + xc * 16 + i) : __ldg(in + hi + xc * 16 + i);
        acc.x += sc * hv.x;
        acc.y += sc * hv.y;
        out[s * slice + xc * 16 + i] = acc;
        nrm += (double)acc.x * acc.x + (double)acc.y * acc.y;
    }
    return nrm;
}

// ---------------------------------------------------------------------------
// 2-d tiles of the persistent coarse solvers (16 coarse dof, Ls_c <= 4; a single apply is the faster
// from global memory, k_coarse_w16).  A block of 8 warps applies the
// operator on a 4 x 2 tile of coarse sites, one warp per site:
//   * the five 16 x 16 blocks of every site of the tile (10 KB contiguous per
//     site) are copied into shared memory by one cp.async.bulk per site,
//     completing on an mbarrier (asynchronous: no registers, all in flight);
//   * meanwhile the threads stage the tile's inputs and their one-site halo
//     (6 x 4 sites x Ls_c slices x 16 values) into shared memory;
//   * the warp then multiplies from shared memory only.
// The mbarrier wait is bounded (%globaltimer); on expiry the block records
// an error in *status, waits once more (bounded) for its copies and returns.
// ---------------------------------------------------------------------------
constexpr int TILE_X = 4, TILE_Y = 2, TILE_HX = TILE_X + 2, TILE_HY = TILE_Y + 2;
constexpr int TILE_SITES = TILE_X * TILE_Y;
constexpr int TILE_THREADS = 32 * TILE_SITES;
// BT: storage of the Galerkin blocks, float2 (FP32) or __half2 (FP16)
template <class BT>
struct TileSmemT {
    BT Y[TILE_SITES][5][256];              // column-major blocks per direction
    float2 v[4][TILE_HY][TILE_HX][16];     // staged inputs with halo
    unsigned long long mbar;
};
template <class BT> __host__ __device__ constexpr unsigned site_block_bytes() { return 5u * 256u * (unsigned)sizeof(BT); }

__device__ __forceinline__ float2 to_f2(float2 a) { return a; }
__device__ __forceinline__ float2 to_f2(__half2 a) { return __half22float2(a); }

template <class BT>
__device__ __forceinline__ void tile_stage(TileSmemT<BT>& sm, const float2* __restrict__ in, const CoarseParams& p,
                                           int x0, int y0) {
    const int L0 = p.Lc[0], L1 = p.Lc[1];
    const long long slice = p.Vc * 16;
    const int total = p.Ls_c * TILE_HY * TILE_HX * 16;
    for (int e = threadIdx.x; e < total; e += blockDim.x) {
        const int j = e & 15;
        const int h = (e >> 4) % (TILE_HY * TILE_HX);
        const int s = (e >> 4) / (TILE_HY * TILE_HX);
        const int hx = h % TILE_HX, hy = h / TILE_HX;
        int gx = x0 + hx - 1, gy = y0 + hy - 1;
        gx = (gx % L0 + L0) % L0;
        gy = (gy % L1 + L1) % L1;
        const long long site = (long long)gy * L0 + gx;
        sm.v[s][hy][hx][j] = __ldcg(in + s * slice + site * 16 + j);   // written by other blocks of this launch
    }
}

// Thread 0 starts the bulk copies of the tile's blocks (phase completes when
// all bytes have landed).  Returns the number of bytes expected.
template <class BT>
__device__ __forceinline__ void tile_issue_blocks(TileSmemT<BT>& sm, const BT* __restrict__ B, const CoarseParams& p,
                                                  int x0, int y0) {
    if (threadIdx.x != 0) return;
    constexpr unsigned SITE_BLOCK_BYTES = site_block_bytes<BT>();
    unsigned bytes = 0;
    for (int w = 0; w < TILE_SITES; ++w) {
        const int gx = x0 + w % TILE_X, gy = y0 + w / TILE_X;
        if (gx < p.Lc[0] && gy < p.Lc[1]) bytes += SITE_BLOCK_BYTES;
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    mbar_expect_tx(&sm.mbar, bytes);
    for (int w = 0; w < TILE_SITES; ++w) {
        const int gx = x0 + w % TILE_X, gy = y0 + w / TILE_X;
        if (gx < p.Lc[0] && gy < p.Lc[1]) {
            const long long xc = (long long)gy * p.Lc[0] + gx;
            bulk_g2s(&sm.Y[w][0][0], B + xc * 5 * 256, SITE_BLOCK_BYTES, &sm.mbar);
        }
    }
}

// Multiply for this warp's site from shared memory; returns the lane's |out|^2.
// The adjoint uses gamma_5-hermiticity of the Galerkin kernel: the chirality-
// preserving prolongator gives Dhat_W^dag = sigma_3 Dhat_W sigma_3 (P^dag gamma_5
// D_W gamma_5 P), so the same blocks serve with sign flips on the chirality -
// components of input and output (2 nvec = 16: components 8..15).
// optional epilogue of tile_site: called with (index, value) of every output written
struct NoEpilogue {
    __device__ __forceinline__ void operator()(long long, float2) const {}
};

template <class BT, class Epi = NoEpilogue>
__device__ __forceinline__ double tile_site(const TileSmemT<BT>& sm, float2* __restrict__ out, const CoarseParams& p,
                                            int x0, int y0, float mf, bool dag, Epi epi = Epi()) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tx = warp % TILE_X, ty = warp / TILE_X;
    const int gx = x0 + tx, gy = y0 + ty;
    if (gx >= p.Lc[0] || gy >= p.Lc[1]) return 0.0;
    const long long xc = (long long)gy * p.Lc[0] + gx;
    const long long slice = p.Vc * 16;
    const int i = lane & 15, sg = lane >> 4;
    const bool h0 = sg < p.Ls_c, h1 = sg + 2 < p.Ls_c;
    const int s0 = h0 ? sg : 0, s1 = h1 ? sg + 2 : 0;
    const int hx = tx + 1, hy = ty + 1;
    float2 acc0 = make_float2(0.f, 0.f), acc1 = make_float2(0.f, 0.f);   // hopping sums for the up / down halves
    float2 acm0 = make_float2(0.f, 0.f), acm1 = make_float2(0.f, 0.f);   // contributions of chirality - inputs
#pragma unroll
    for (int dir = 0; dir < 5; ++dir) {
        const int nx = hx + (dir == 1 ? 1 : dir == 2 ? -1 : 0);
        const int ny = hy + (dir == 3 ? 1 : dir == 4 ? -1 : 0);
        const BT* Yd = &sm.Y[warp][dir][i];
        const float4* va = reinterpret_cast<const float4*>(&sm.v[s0][ny][nx][0]);
        const float4* vb = reinterpret_cast<const float4*>(&sm.v[s1][ny][nx][0]);
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            const float4 a = va[m], b = vb[m];
            const float2 y0v = to_f2(Yd[(2 * m) * 16]), y1v = to_f2(Yd[(2 * m + 1) * 16]);
            if (m < 4) {
                acc0 = cfma(y0v, make_float2(a.x, a.y), acc0);
                acc0 = cfma(y1v, make_float2(a.z, a.w), acc0);
                acc1 = cfma(y0v, make_float2(b.x, b.y), acc1);
                acc1 = cfma(y1v, make_float2(b.z, b.w), acc1);
            } else {
                acm0 = cfma(y0v, make_float2(a.x, a.y), acm0);
                acm0 = cfma(y1v, make_float2(a.z, a.w), acm0);
                acm1 = cfma(y0v, make_float2(b.x, b.y), acm1);
                acm1 = cfma(y1v, make_float2(b.z, b.w), acm1);
            }
        }
    }
    // hop sum: Dhat_W v (operator) or sigma_3 Dhat_W sigma_3 v (adjoint)
    const float si = (dag && i >= 8) ? -1.f : 1.f;
    const float sm_ = dag ? -1.f : 1.f;
    const float2 hop0 = make_float2(si * (acc0.x + sm_ * acm0.x), si * (acc0.y + sm_ * acm0.y));
    const float2 hop1 = make_float2(si * (acc1.x + sm_ * acm1.x), si * (acc1.y + sm_ * acm1.y));
    const int c = i / p.nvec;
    const bool from_below = dag ? (c == 1) : (c == 0);
    double nrm = 0.0;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const bool has = k == 0 ? h0 : h1;
        if (!has) continue;
        const int s = k == 0 ? s0 : s1;
        const float2 hop = k == 0 ? hop0 : hop1;
        const float2 self = sm.v[s][hy][hx][i];                 // the "+1" of Dhat_W + 1
        int sh;
        float sc = 1.f;
        if (from_below) { if (s > 0) sh = s - 1; else { sh = p.Ls_c - 1; sc = -mf; } }
        else            { if (s < p.Ls_c - 1) sh = s + 1; else { sh = 0; sc = -mf; } }
        const float2 hv = sm.v[sh][hy][hx][i];
        float2 acc;
        acc.x = hop.x + self.x + sc * hv.x;
        acc.y = hop.y + self.y + sc * hv.y;
        out[s * slice + xc * 16 + i] = acc;
        epi(s * slice + xc * 16 + i, acc);
        nrm += (double)acc.x * acc.x + (double)acc.y * acc.y;
    }
    return nrm;
}

constexpr unsigned long long TILE_WAIT_NS = 2000000000ULL;   // 2 s

__device__ __forceinline__ float2 not_a_number2() {
    const float q = __int_as_float(0x7fffffff);
    return make_float2(q, q);
}

// A bulk-copy wait that nothing will end, which records its expiry as the stencils do
__global__ void k_coarse_wait_expires(unsigned long long budget_ns, int* status) {
    __shared__ unsigned long long bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        mbar_expect_tx(&bar, 16);
    }
    __syncthreads();
    if (!mbar_wait_bounded(&bar, 0, budget_ns) && threadIdx.x == 0) atomicExch(status, 2);
}

// DWF_ERR_TIMEOUT if a coarse stencil on this handle gave up waiting for a copy since the last call of this
// function, which forgets it: the end of every call that synchronises anyway.
dwf_status coarse_wait_status(const dwf_mg* h, cudaStream_t st) {
    int hs = 0;
    DWF_CHECK_CUDA(cudaMemcpyAsync(&hs, h->status + 1, sizeof(int), cudaMemcpyDeviceToHost, st));
    DWF_CHECK_CUDA(cudaStreamSynchronize(st));
    if (hs == 0) return DWF_OK;
    DWF_CHECK_CUDA(cudaMemsetAsync(h->status + 1, 0, sizeof(int), st));
    DWF_CHECK_CUDA(cudaStreamSynchronize(st));
    set_error("coarse stencil: a bulk copy wait timed out");
    return DWF_ERR_TIMEOUT;
}

static bool tile_ok(const CoarseParams& p) { return p.nd == 2 && p.ncd == 16 && p.Ls_c <= 4; }

static dwf_status site_init_attributes();

static dwf_status mma_init_attributes();

dwf_status coarse_init_attributes() {
    DWF_TRY(mma_init_attributes());
    return site_init_attributes();
}

template <int NCD>
__global__ void __launch_bounds__(256) k_coarse_dwf(const float2* __restrict__ B, const float2* __restrict__ in,
                                                    float2* __restrict__ out, CoarseParams p, bool dag, const int* skip) {
    if (skip && *skip) return;
    const long long xc = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (xc >= p.Vc) return;
    // (a caller's vector may start on an 8-byte boundary; warp_site16 reads its input 16 bytes at a time)
    if (NCD == 16 && p.Ls_c <= 4 && (reinterpret_cast<uintptr_t>(in) & 15) == 0) warp_site16<false>(B, in, out, p, xc, p.mf, dag, threadIdx.x & 31);
    else warp_site_apply<NCD, false>(B, in, out, p, xc, p.mf, dag, threadIdx.x & 31);
}

// ---------------------------------------------------------------------------
// One vector, 2-d, 16 coarse dof, Ls_c <= 4: one warp per coarse site, everything straight from
// global memory.  Lane 4 g + q holds the columns 2 g, 2 g + 1 and the rows 4 q .. 4 q + 3 of a
// block, so a block arrives as two 16-byte loads per lane (FP16 storage) and its inputs as one
// per slice (broadcast over q), nothing is staged or waited for, and every FP32 multiply-add of the block is done
// once: 640 per lane and site.  The 4 rows x 4 slices of partial sums then fold over the 8
// lanes g in three exchanges that each halve what a lane carries, which leaves slice lane / 8 and
// two adjacent rows in a lane: one 16-byte store.  The adjoint uses sigma_3 (Dhat_W^dag =
// sigma_3 Dhat_W sigma_3): the sign of the chirality - columns goes onto a lane's sums.
// Bound by FP32 issue and the L2 round trips of five directions (the 21 MB of blocks of a
// 64^2 lattice stay in L2).  Staging blocks and inputs in shared memory (8 sites per thread block,
// bulk copies, every block element converted twice) took 12.5 us at 64^2 x 4; 256^2 x 16
// gradient step 630 -> 522 ms.
// ---------------------------------------------------------------------------
constexpr int W16_WARPS = 4;

// rows 4 q .. 4 q + 3 of one block column
__device__ __forceinline__ void ld_rows4(const __half2* p, float2 (&y)[4]) {
    const uint4 u = __ldg(reinterpret_cast<const uint4*>(p));
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int r = 0; r < 4; ++r) y[r] = __half22float2(*reinterpret_cast<const __half2*>(&w[r]));
}
__device__ __forceinline__ void ld_rows4(const float2* p, float2 (&y)[4]) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(p)), b = __ldg(reinterpret_cast<const float4*>(p) + 1);
    y[0] = make_float2(a.x, a.y); y[1] = make_float2(a.z, a.w);
    y[2] = make_float2(b.x, b.y); y[3] = make_float2(b.z, b.w);
}
// two adjacent complex values; V4: 16-byte aligned
template <bool V4>
__device__ __forceinline__ float4 ld_pair(const float2* p) {
    if (V4) return __ldg(reinterpret_cast<const float4*>(p));
    const float2 a = __ldg(p), b = __ldg(p + 1);
    return make_float4(a.x, a.y, b.x, b.y);
}

template <class BT, bool V4>
__global__ void __launch_bounds__(W16_WARPS * 32, 5)
k_coarse_w16(const BT* __restrict__ B, const float2* __restrict__ in, float2* __restrict__ out, CoarseParams p,
             bool dag, const int* skip) {
    if (skip && *skip) return;
    const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
    const int xc = blockIdx.x * W16_WARPS + (threadIdx.x >> 5);
    if (xc >= p.Vc) return;                              // whole warps; no block-wide barrier below
    const int L0 = p.Lc[0], L1 = p.Lc[1], y0 = xc / L0, x0 = xc - y0 * L0;
    const int nb[5] = {xc, x0 + 1 == L0 ? xc - x0 : xc + 1, x0 == 0 ? xc + L0 - 1 : xc - 1,
                       y0 + 1 == L1 ? x0 : xc + L0, y0 == 0 ? xc + (L1 - 1) * L0 : xc - L0};
    const long long slice = p.Vc * 16;
    const BT* Bl = B + (long long)xc * (5 * 256) + 2 * g * 16 + 4 * q;
    float2 acc[4][4];                                    // [slice][row]
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[s][r] = make_float2(0.f, 0.f);
#pragma unroll
    for (int dir = 0; dir < 5; ++dir) {
        const float2* v = in + (long long)nb[dir] * 16 + 2 * g;
        float4 a[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) a[s] = s < p.Ls_c ? ld_pair<V4>(v + s * slice) : make_float4(0.f, 0.f, 0.f, 0.f);
        float2 ya[4], yb[4];
        ld_rows4(Bl + dir * 256, ya);
        ld_rows4(Bl + dir * 256 + 16, yb);
#pragma unroll
        for (int s = 0; s < 4; ++s)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                acc[s][r] = cfma(ya[r], make_float2(a[s].x, a[s].y), acc[s][r]);
                acc[s][r] = cfma(yb[r], make_float2(a[s].z, a[s].w), acc[s][r]);
            }
    }
    // fold over g: bit 4 of the lane keeps slices 0, 1 or 2, 3, bit 3 one of the two, bit 2 rows 0, 1 or 2, 3
    const float sg = dag && g >= 4 ? -1.f : 1.f;
    const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
    float2 h2[2][4], h1[4], h0[2];
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const float2 keep = b4 ? acc[s + 2][r] : acc[s][r], send = b4 ? acc[s][r] : acc[s + 2][r];
            // the partner's columns have the other chirality: each side signs its own sums
            h2[s][r].x = sg * keep.x + __shfl_xor_sync(0xffffffffu, sg * send.x, 16);
            h2[s][r].y = sg * keep.y + __shfl_xor_sync(0xffffffffu, sg * send.y, 16);
        }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const float2 keep = b3 ? h2[1][r] : h2[0][r], send = b3 ? h2[0][r] : h2[1][r];
        h1[r].x = keep.x + __shfl_xor_sync(0xffffffffu, send.x, 8);
        h1[r].y = keep.y + __shfl_xor_sync(0xffffffffu, send.y, 8);
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const float2 keep = b2 ? h1[r + 2] : h1[r], send = b2 ? h1[r] : h1[r + 2];
        h0[r].x = keep.x + __shfl_xor_sync(0xffffffffu, send.x, 4);
        h0[r].y = keep.y + __shfl_xor_sync(0xffffffffu, send.y, 4);
    }
    const int s = lane >> 3, row = 4 * q + (b2 ? 2 : 0);
    if (s >= p.Ls_c) return;
    const int c = row / p.nvec;                          // nvec = 8: both rows have one chirality
    const float si = dag && c == 1 ? -1.f : 1.f;
    const bool from_below = dag ? (c == 1) : (c == 0);
    const int sh = from_below ? (s > 0 ? s - 1 : p.Ls_c - 1) : (s < p.Ls_c - 1 ? s + 1 : 0);
    const float sc = from_below ? (s > 0 ? 1.f : -p.mf) : (s < p.Ls_c - 1 ? 1.f : -p.mf);
    const float2* me = in + (long long)xc * 16 + row;
    const float4 self = ld_pair<V4>(me + s * slice), hv = ld_pair<V4>(me + sh * slice);
    const float4 o = make_float4(si * h0[0].x + self.x + sc * hv.x, si * h0[0].y + self.y + sc * hv.y,
                                 si * h0[1].x + self.z + sc * hv.z, si * h0[1].y + self.w + sc * hv.w);
    float2* op = out + s * slice + (long long)xc * 16 + row;
    if (V4) *reinterpret_cast<float4*>(op) = o;
    else { op[0] = make_float2(o.x, o.y); op[1] = make_float2(o.z, o.w); }
}

template <class BT>
static void launch_w16(const void* B, const float2* in, float2* out, const CoarseParams& p, bool dag, const int* skip,
                       cudaStream_t st) {
    const unsigned grid = (unsigned)((p.Vc + W16_WARPS - 1) / W16_WARPS);
    if (aligned16(in) && aligned16(out))
        k_coarse_w16<BT, true><<<grid, W16_WARPS * 32, 0, st>>>((const BT*)B, in, out, p, dag, skip);
    else
        k_coarse_w16<BT, false><<<grid, W16_WARPS * 32, 0, st>>>((const BT*)B, in, out, p, dag, skip);
}

// ---------------------------------------------------------------------------
// Per-site kernel for wide coarse blocks (4-d: 9 directions, 2 nvec = 48 dof).
// One block per coarse site: the site's ndir blocks (contiguous, 83 KB in FP16
// at 48 dof) arrive in shared memory by one cp.async.bulk on an mbarrier while
// the threads stage the neighbours' inputs; thread (i, s) then forms output row
// i of slice s from shared memory only.  At one right-hand side the blocks are
// read once per apply, so the kernel is bound by their HBM traffic.  The
// adjoint uses sigma_3 (Dhat_W^dag = sigma_3 Dhat_W sigma_3), so the same blocks
// serve both.
// ---------------------------------------------------------------------------
// neighbour of coarse site xc in direction dir (0 self, 1 + 2 mu forward, 2 + 2 mu
// backward) with 32-bit index arithmetic (coarse lattices have < 2^31 sites)
__device__ __forceinline__ int coarse_nb32(const CoarseParams& p, int xc, int dir) {
    if (dir == 0) return xc;
    const int mu = (dir - 1) >> 1;
    const int L0 = p.Lc[0], L1 = p.Lc[1], L2 = p.Lc[2], L3 = p.Lc[3];
    const int Lm = mu == 0 ? L0 : mu == 1 ? L1 : mu == 2 ? L2 : L3;
    const int stride = mu == 0 ? 1 : mu == 1 ? L0 : mu == 2 ? L0 * L1 : L0 * L1 * L2;
    const int c = (xc / stride) % Lm;
    const int cn = ((dir - 1) & 1) ? (c == 0 ? Lm - 1 : c - 1) : (c == Lm - 1 ? 0 : c + 1);
    return xc + (cn - c) * stride;
}

template <class BT>
__host__ __device__ constexpr size_t site_smem_bytes(int ndir, int ncd, int Ls_c) {
    return ((size_t)ndir * ncd * ncd * sizeof(BT) + 15) / 16 * 16 + (size_t)ndir * Ls_c * ncd * sizeof(float2) + 16;
}

template <class BT>
__global__ void __launch_bounds__(512) k_coarse_site(const BT* __restrict__ B, const float2* __restrict__ in,
                                                     float2* __restrict__ out, CoarseParams p, bool dag,
                                                     const int* skip, int* status) {
    if (skip && *skip) return;
    extern __shared__ __align__(128) unsigned char site_raw[];
    const int ncd = p.ncd, ndir = p.ndir, Ls_c = p.Ls_c;
    const size_t yb_bytes = ((size_t)ndir * ncd * ncd * sizeof(BT) + 15) / 16 * 16;
    BT* yb = reinterpret_cast<BT*>(site_raw);
    float2* vs = reinterpret_cast<float2*>(site_raw + yb_bytes);                 // [dir][s][j]
    unsigned long long* mbar = reinterpret_cast<unsigned long long*>(site_raw + yb_bytes +
                                                                     (size_t)ndir * Ls_c * ncd * sizeof(float2));
    const long long xc = blockIdx.x;
    const long long slice = p.Vc * ncd;
    const unsigned bytes = (unsigned)((size_t)ndir * ncd * ncd * sizeof(BT));
    if (threadIdx.x == 0) {
        mbar_init(mbar, 1);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect_tx(mbar, bytes);
        bulk_g2s(yb, B + xc * (long long)ndir * ncd * ncd, bytes, mbar);
    }
    __shared__ int nbs[MG_MAX_DIRS];
    if (threadIdx.x < ndir) nbs[threadIdx.x] = coarse_nb32(p, (int)xc, threadIdx.x);
    __syncthreads();
    const int nv = ndir * Ls_c * ncd;
    for (int e = threadIdx.x; e < nv; e += blockDim.x) {
        const int j = e % ncd, s = (e / ncd) % Ls_c, dir = e / (ncd * Ls_c);
        vs[e] = __ldg(in + s * slice + (long long)nbs[dir] * ncd + j);
    }
    __syncthreads();
    if (!mbar_wait_bounded(mbar, 0, TILE_WAIT_NS)) {
        atomicExch(status, 2);
        mbar_wait_bounded(mbar, 0, TILE_WAIT_NS);          // let the copy land before the block exits
        const int e = threadIdx.x;
        if (e < ncd * Ls_c) out[e / ncd * slice + xc * ncd + e % ncd] = not_a_number2();
        return;
    }
    const int i = threadIdx.x % ncd, s = threadIdx.x / ncd;
    if (s >= Ls_c) return;
    const int nvec = p.nvec;
    // inputs j < nvec / j >= nvec, each summed in four independent chains (j mod 4)
    float2 a_lo[4], a_hi[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) { a_lo[u] = make_float2(0.f, 0.f); a_hi[u] = a_lo[u]; }
    for (int dir = 0; dir < ndir; ++dir) {
        const BT* yd = yb + (size_t)dir * ncd * ncd + i;
        const float2* v = vs + (dir * Ls_c + s) * ncd;
        int j = 0;
        for (; j + 4 <= nvec; j += 4) {
#pragma unroll
            for (int u = 0; u < 4; ++u) a_lo[u] = cfma(to_f2(yd[(j + u) * ncd]), v[j + u], a_lo[u]);
        }
        for (; j < nvec; ++j) a_lo[0] = cfma(to_f2(yd[j * ncd]), v[j], a_lo[0]);
        for (; j + 4 <= ncd; j += 4) {
#pragma unroll
            for (int u = 0; u < 4; ++u) a_hi[u] = cfma(to_f2(yd[(j + u) * ncd]), v[j + u], a_hi[u]);
        }
        for (; j < ncd; ++j) a_hi[0] = cfma(to_f2(yd[j * ncd]), v[j], a_hi[0]);
    }
    const float2 lo = make_float2((a_lo[0].x + a_lo[1].x) + (a_lo[2].x + a_lo[3].x),
                                  (a_lo[0].y + a_lo[1].y) + (a_lo[2].y + a_lo[3].y));
    const float2 hi = make_float2((a_hi[0].x + a_hi[1].x) + (a_hi[2].x + a_hi[3].x),
                                  (a_hi[0].y + a_hi[1].y) + (a_hi[2].y + a_hi[3].y));
    const float sj = dag ? -1.f : 1.f;                   // sigma_3 on the inputs
    const float si = (dag && i >= nvec) ? -1.f : 1.f;    // sigma_3 on the output
    float2 acc = make_float2(si * (lo.x + sj * hi.x), si * (lo.y + sj * hi.y));
    const float2* v0 = vs;                               // dir 0 = the site itself
    const float2 self = v0[s * ncd + i];
    const int c = i / nvec;
    const bool from_below = dag ? (c == 1) : (c == 0);
    int sh;
    float sc = 1.f;
    if (from_below) { if (s > 0) sh = s - 1; else { sh = Ls_c - 1; sc = -p.mf; } }
    else            { if (s < Ls_c - 1) sh = s + 1; else { sh = 0; sc = -p.mf; } }
    const float2 hv = v0[sh * ncd + i];
    acc.x += self.x + sc * hv.x;
    acc.y += self.y + sc * hv.y;
    out[s * slice + xc * ncd + i] = acc;
}

// ---------------------------------------------------------------------------
// Tensor-core form of the 48-dof stencil (4-d, FP16 blocks, Ls_c <= 4).  One
// warp per coarse site.  Per direction the complex product Y v over the Ls_c
// slices is the real product of A = [Re Y; Im Y] (96 x 48, FP16 as stored)
// with B (48 x 8), column 2 s the real and 2 s + 1 the imaginary part of
// slice s: C = A B holds Re Y Re v, Re Y Im v (rows < 48) and Im Y Re v, Im Y Im v
// (rows >= 48) of one slice in one lane, so
// Re(Y v) = C[i][Re] - C[48 + i][Im] and Im(Y v) = C[48 + i][Re] + C[i][Im]
// are sums of its own accumulators.
//
// Inputs: the 24 values of a slice and chirality are scaled by a power of two
// and split into two FP16 parts (mma_f16.cuh: 22 bits, as a TF32 pair keeps), so
// that mma.m16n8k16 takes the blocks as they are stored: half the products of
// the TF32 form and no conversion of a block.  The chiralities are scaled apart
// because on the slices near a wall they differ by orders of magnitude; the column
// tiles of 16 that hold both are multiplied as two of 8.  The products of a
// direction with the parts of a chirality accumulate in FP32, four sums that are
// added up with their scales taken back, as the directions are.
//
// Only the self block and the four forward blocks of a site are stored: the
// kernel is gamma_5-hermitian, so the backward block of x is
// sigma_3 Y_+mu(x - mu)^dag sigma_3 of its neighbour's forward block, which that
// neighbour's warp reads too: once from HBM, then from L2 (the farthest
// neighbour, one coarse t-slice away, is 23 MB of blocks behind at 8^3 x 16).
// A block lies in memory as 8 x 8 tiles, and ldmatrix reads it from shared
// memory as it is or transposed; sigma_3 and the conjugate are signs of the
// inputs and of the sums.
//
// Each warp brings the block of direction d + 1 into the other half of its
// shared-memory ring by one bulk copy while it multiplies that of direction
// d: 9.2 KB per warp, 12 warps per SM.  Bound by the block bytes (L2 to SM:
// 83 KB per site; HBM: 46 KB): 34 us at 6^3 x 12 sites x 4 slices and 82 us at 8^3 x 16
// (8.3 TB/s of block bytes), where nine stored blocks and TF32 products took 44 and 114 us.
// (One scale per slice, with both parts and chiralities in one sum: 33 and 81 us.  The
// inputs of direction d + 1 are split behind the products of d: before them, 37 and 89 us.)
// ---------------------------------------------------------------------------
constexpr int CM_WARPS = 4;
constexpr int CM_BLOCKS = 5;                             // stored blocks per site: self, +mu
constexpr unsigned CM_BLOCK_BYTES = 96 * 48 * sizeof(__half);
struct CmSmem {
    unsigned char ring[2][CM_BLOCK_BYTES];               // [row tile 12][column tile 6][8][8] halves
    unsigned long long bar[2];
    unsigned long long pad[14];                          // the next warp's ring on a 128-byte line
};

// This lane's inputs of one direction: column g = 2 s + part, dof 8 j + 2 t and 8 j + 2 t + 1 (j < 6)
template <bool V4>
__device__ __forceinline__ void cm_load(float (&v)[6][2], const float2* vin, bool colv, int part) {
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const float4 u = colv ? ld_pair<V4>(vin + 8 * j) : make_float4(0.f, 0.f, 0.f, 0.f);
        v[j][0] = part ? u.y : u.x;
        v[j][1] = part ? u.w : u.z;
    }
}
// B fragments: hi[j] and lo[j] hold dof 8 j + 2 t, + 1; chirality - dof (j >= 3) change sign with
// `neg`.  back[c] undoes the scale of chirality c of this lane's slice.
__device__ __forceinline__ void cm_split(uint32_t (&hi)[6], uint32_t (&lo)[6], const float (&v)[6][2], bool neg,
                                         float (&back)[2]) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        float m = 0.f;
#pragma unroll
        for (int j = 3 * c; j < 3 * c + 3; ++j) m = fmaxf(m, fmaxf(fabsf(v[j][0]), fabsf(v[j][1])));
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));    // the chirality's values: lanes t, and part
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 4));
        float scale;
        f16_scale(m, scale, back[c]);
        if (neg && c == 1) scale = -scale;
#pragma unroll
        for (int j = 3 * c; j < 3 * c + 3; ++j) {
            __half2 h, l;
            f16_split(v[j][0] * scale, v[j][1] * scale, h, l);
            hi[j] = *reinterpret_cast<const uint32_t*>(&h);
            lo[j] = *reinterpret_cast<const uint32_t*>(&l);
        }
    }
}
// One row tile: C[0], C[1] the products with the high parts of chirality +, -, C[2], C[3] with the low
// ones; a[kt] holds the columns 16 kt .., of which those from 24 on have chirality -
__device__ __forceinline__ void cm_products(float (&C)[4][4], const uint32_t (&a)[3][4], const uint32_t (&hi)[6],
                                            const uint32_t (&lo)[6]) {
    mma_f16_zero(C[0], a[0][0], a[0][1], a[0][2], a[0][3], hi[0], hi[1]);
    mma_f16_zero(C[1], a[2][0], a[2][1], a[2][2], a[2][3], hi[4], hi[5]);
    mma_f16_zero(C[2], a[0][0], a[0][1], a[0][2], a[0][3], lo[0], lo[1]);
    mma_f16_zero(C[3], a[2][0], a[2][1], a[2][2], a[2][3], lo[4], lo[5]);
    mma_f16_k8(C[0], a[1][0], a[1][1], hi[2]);
    mma_f16_k8(C[1], a[1][2], a[1][3], hi[3]);
    mma_f16_k8(C[2], a[1][0], a[1][1], lo[2]);
    mma_f16_k8(C[3], a[1][2], a[1][3], lo[3]);
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int q = 0; q < 4; ++q) C[c][q] = fmaf(F16_LOW, C[2 + c][q], C[c][q]);
}

template <bool V4>
__global__ void __launch_bounds__(CM_WARPS * 32, 3) k_coarse_mma(const unsigned char* __restrict__ Ym,
                                                                 const float2* __restrict__ in,
                                                                 float2* __restrict__ out, CoarseParams p, bool dag,
                                                                 const int* skip, int* status) {
    if (skip && *skip) return;
    extern __shared__ __align__(128) unsigned char cm_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    CmSmem& sm = reinterpret_cast<CmSmem*>(cm_raw)[warp];
    const int xc = blockIdx.x * CM_WARPS + warp;
    if (xc >= p.Vc) return;                              // whole warps; no block-wide barrier below
    const int Ls_c = p.Ls_c;
    const long long slice = p.Vc * 48;
    const int part = g & 1, sB = g >> 1;                 // B column g
    const bool colv = sB < Ls_c;
    const float2* vb = in + (colv ? sB : 0) * slice + 2 * t;
    // steps: the self block, the four forward hops, the four backward hops (the neighbour's forward block)
    constexpr int STEPS = 2 * CM_BLOCKS - 1;
    // (lane d finds the neighbour of step d: its index divisions are done once per site)
    const int mine = coarse_nb32(p, xc, lane == 0 || lane >= STEPS ? 0 : lane < CM_BLOCKS ? 2 * lane - 1 : 2 * (lane - CM_BLOCKS) + 2);
    auto neighbour = [&](int d) { return __shfl_sync(0xffffffffu, mine, d); };
    auto issue = [&](int d, int nb) {
        if (lane != 0) return;
        const long long blk = d < CM_BLOCKS ? (long long)xc * CM_BLOCKS + d : (long long)nb * CM_BLOCKS + d - CM_BLOCKS + 1;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect_tx(&sm.bar[d & 1], CM_BLOCK_BYTES);
        bulk_g2s(sm.ring[d & 1], Ym + blk * CM_BLOCK_BYTES, CM_BLOCK_BYTES, &sm.bar[d & 1]);
    };
    if (lane == 0) { mbar_init(&sm.bar[0], 1); mbar_init(&sm.bar[1], 1); }
    __syncwarp();
    issue(0, xc);
    issue(1, xc);
    float acc[3][4];                                     // rows 16 m + g (re, im), 16 m + g + 8 (re, im) of slice t
#pragma unroll
    for (int m = 0; m < 3; ++m)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[m][q] = 0.f;
    const int r8 = lane & 7, i8 = (lane >> 3) & 1, i16 = lane >> 4;
    float v[6][2];
    cm_load<V4>(v, vb + (long long)xc * 48, colv, part);
    uint32_t hi[6], lo[6];
    float back[2];
    cm_split(hi, lo, v, dag, back);                      // sigma_3 on the inputs: of the adjoint operator
#pragma unroll
    for (int c = 0; c < 2; ++c) back[c] = __shfl_sync(0xffffffffu, back[c], 8 * t);
    cm_load<V4>(v, vb + (long long)neighbour(1) * 48, colv, part);
#pragma unroll 1
    for (int d = 0; d < STEPS; ++d) {
        const bool fwd = d < CM_BLOCKS;
        if (!__all_sync(0xffffffffu, mbar_wait_bounded(&sm.bar[d & 1], (d >> 1) & 1, TILE_WAIT_NS))) {
            if (lane == 0) atomicExch(status, 2);
            // let the copies land before the warp exits
            mbar_wait_bounded(&sm.bar[d & 1], (d >> 1) & 1, TILE_WAIT_NS);
            if (d + 1 < STEPS) mbar_wait_bounded(&sm.bar[(d + 1) & 1], ((d + 1) >> 1) & 1, TILE_WAIT_NS);
            for (int e = lane; e < 48 * Ls_c; e += 32) out[e / 48 * slice + (long long)xc * 48 + e % 48] = not_a_number2();
            return;
        }
        const uint32_t ring = smem_u32(sm.ring[d & 1]);
        if (fwd) {
            // tiles (row 2 m, 2 m + 1) x (column 2 kt, 2 kt + 1)
            const uint32_t base = ring + (i8 * 6 + i16) * 128 + r8 * 16;
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                uint32_t a[2][3][4];                     // Re Y, Im Y
                float C[2][4][4];
#pragma unroll
                for (int ri = 0; ri < 2; ++ri)
#pragma unroll
                    for (int kt = 0; kt < 3; ++kt) ldmatrix4<false>(a[ri][kt], base + (12 * (m + 3 * ri) + 2 * kt) * 128);
                cm_products(C[0], a[0], hi, lo);
                cm_products(C[1], a[1], hi, lo);
#pragma unroll
                for (int c = 0; c < 2; ++c)
#pragma unroll
                    for (int q = 0; q < 4; q += 2) {
                        acc[m][q] = fmaf(back[c], C[0][c][q] - C[1][c][q + 1], acc[m][q]);
                        acc[m][q + 1] = fmaf(back[c], C[0][c][q + 1] + C[1][c][q], acc[m][q + 1]);
                    }
            }
        } else {
            // outputs 16 m .. are columns (tiles 2 m, 2 m + 1), inputs 16 kt .. rows (tiles 2 kt, 2 kt + 1) of Re Y and Im Y
            const uint32_t base = ring + (i16 * 6 + i8) * 128 + r8 * 16;
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                uint32_t a[2][3][4];
                float C[2][4][4];
#pragma unroll
                for (int ri = 0; ri < 2; ++ri)
#pragma unroll
                    for (int kt = 0; kt < 3; ++kt) ldmatrix4<true>(a[ri][kt], base + (12 * (kt + 3 * ri) + 2 * m) * 128);
                cm_products(C[0], a[0], hi, lo);
                cm_products(C[1], a[1], hi, lo);
#pragma unroll
                for (int c = 0; c < 2; ++c)
#pragma unroll
                    for (int q = 0; q < 4; q += 2) {
                        // conj(Y): Re + Im parts; sigma_3 on outputs 8 (2 m + q / 2) and up
                        const float sb = 2 * m + q / 2 >= 3 ? -back[c] : back[c];
                        acc[m][q] = fmaf(sb, C[0][c][q] + C[1][c][q + 1], acc[m][q]);
                        acc[m][q + 1] = fmaf(sb, C[0][c][q + 1] - C[1][c][q], acc[m][q + 1]);
                    }
            }
        }
        if (d + 1 < STEPS) {
            // the next direction's inputs; sigma_3 of the adjoint operator and of a backward block
            cm_split(hi, lo, v, dag != (d + 1 >= CM_BLOCKS), back);
#pragma unroll
            for (int c = 0; c < 2; ++c) back[c] = __shfl_sync(0xffffffffu, back[c], 8 * t);
            if (d + 2 < STEPS) cm_load<V4>(v, vb + (long long)neighbour(d + 2) * 48, colv, part);
        }
        __syncwarp();                                    // every lane has read this half of the ring
        if (d + 2 < STEPS) issue(d + 2, neighbour(d + 2));
    }
    const int s = t;
    if (s >= Ls_c) return;
#pragma unroll
    for (int m = 0; m < 3; ++m)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = 16 * m + 8 * h + g;
            const int c = r >= 24;
            const float si = dag && c ? -1.f : 1.f;      // sigma_3 on the output
            const bool from_below = dag ? (c == 1) : (c == 0);
            const int sh = from_below ? (s > 0 ? s - 1 : Ls_c - 1) : (s < Ls_c - 1 ? s + 1 : 0);
            const float sc = from_below ? (s > 0 ? 1.f : -p.mf) : (s < Ls_c - 1 ? 1.f : -p.mf);
            const float2* me = in + (long long)xc * 48 + r;
            const float2 self = __ldg(me + s * slice), hv = __ldg(me + sh * slice);
            out[s * slice + (long long)xc * 48 + r] = make_float2(si * acc[m][2 * h] + self.x + sc * hv.x,
                                                                  si * acc[m][2 * h + 1] + self.y + sc * hv.y);
        }
}

static dwf_status mma_init_attributes() {
    const int sh = (int)(CM_WARPS * sizeof(CmSmem));
    DWF_CHECK_CUDA(cudaFuncSetAttribute(k_coarse_mma<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, sh));
    DWF_CHECK_CUDA(cudaFuncSetAttribute(k_coarse_mma<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, sh));
    return DWF_OK;
}

constexpr size_t SITE_SMEM_MAX = 200 * 1024;
static dwf_status site_init_attributes() {
    DWF_CHECK_CUDA(cudaFuncSetAttribute(k_coarse_site<float2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)SITE_SMEM_MAX));
    DWF_CHECK_CUDA(cudaFuncSetAttribute(k_coarse_site<__half2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)SITE_SMEM_MAX));
    return DWF_OK;
}

// the per-site kernel: 4-d blocks (or wide 2-d ones) whose shared-memory copy fits in a block
static bool site_ok(const CoarseParams& p, int half) {
    if (p.ncd < 24 || p.ncd * p.Ls_c > 512) return false;
    const size_t b = half ? site_smem_bytes<__half2>(p.ndir, p.ncd, p.Ls_c) : site_smem_bytes<float2>(p.ndir, p.ncd, p.Ls_c);
    return b <= SITE_SMEM_MAX;
}

static CoarseParams coarse_params(const dwf_mg* h, double mf) {
    CoarseParams p;
    p.Vc = h->mg.Vc;
    p.nd = h->mg.nd;
    for (int mu = 0; mu < 4; ++mu) p.Lc[mu] = h->mg.Lc[mu];
    p.Ls_c = h->mg.Ls_c;
    p.ncd = h->mg.ncd;
    p.nvec = h->mg.nvec;
    p.ndir = h->mg.ndir;
    p.mf = (float)mf;
    return p;
}

dwf_status coarse_dwf_apply(const dwf_mg* h, const float2* in, float2* out, double mf, bool dagger, const int* skip,
                            cudaStream_t st) {
    CoarseParams p = coarse_params(h, mf);
    const int thr = 256;
    const unsigned grid = (unsigned)((p.Vc * 32 + thr - 1) / thr);
    const float2* B = dagger ? h->Yd32 : h->Y32;
    if (tile_ok(p)) {
        if (h->ytile_half) launch_w16<__half2>(h->Ytile, in, out, p, dagger, skip, st);
        else               launch_w16<float2>(h->Ytile, in, out, p, dagger, skip, st);
    } else if (h->Ymma && p.ncd == 48 && p.ndir == 9 && p.Ls_c <= 4) {
        const unsigned grid1 = (unsigned)((p.Vc + CM_WARPS - 1) / CM_WARPS);
        constexpr size_t sh = CM_WARPS * sizeof(CmSmem);
        if (aligned16(in))
            k_coarse_mma<true><<<grid1, CM_WARPS * 32, sh, st>>>((const unsigned char*)h->Ymma, in, out, p, dagger, skip, h->status + 1);
        else
            k_coarse_mma<false><<<grid1, CM_WARPS * 32, sh, st>>>((const unsigned char*)h->Ymma, in, out, p, dagger, skip, h->status + 1);
    } else if (site_ok(p, h->ytile_half)) {
        const int threads = p.ncd * p.Ls_c;
        if (h->ytile_half)
            k_coarse_site<__half2><<<(unsigned)p.Vc, threads, site_smem_bytes<__half2>(p.ndir, p.ncd, p.Ls_c), st>>>(
                (const __half2*)h->Ytile, in, out, p, dagger, skip, h->status + 1);
        else
            k_coarse_site<float2><<<(unsigned)p.Vc, threads, site_smem_bytes<float2>(p.ndir, p.ncd, p.Ls_c), st>>>(
                (const float2*)h->Ytile, in, out, p, dagger, skip, h->status + 1);
    } else if (p.ncd == 16) k_coarse_dwf<16><<<grid, thr, 0, st>>>(B, in, out, p, dagger, skip);
    else             k_coarse_dwf<0><<<grid, thr, 0, st>>>(B, in, out, p, dagger, skip);
    DWF_CHECK_LAUNCH();
    return DWF_OK;
}

dwf_status coarse_site_apply(const CoarseParams& p, const __half2* B, const float2* in, float2* out, bool dagger,
                             const int* skip, int* status, cudaStream_t st) {
    if (!site_ok(p, 1)) { set_error("the per-site coarse stencil does not take %d dof on %d slices", p.ncd, p.Ls_c);
                          return DWF_ERR_UNSUPPORTED; }
    k_coarse_site<__half2><<<(unsigned)p.Vc, p.ncd * p.Ls_c, site_smem_bytes<__half2>(p.ndir, p.ncd, p.Ls_c), st>>>(
        B, in, out, p, dagger, skip, status);
    DWF_CHECK_LAUNCH();
    return DWF_OK;
}

dwf_status coarse_site_apply(const CoarseParams& p, const float2* B, const float2* in, float2* out, bool dagger,
                             const int* skip, int* status, cudaStream_t st) {
    if (!site_ok(p, 0)) { set_error("the per-site coarse stencil does not take %d dof on %d slices", p.ncd, p.Ls_c);
                          return DWF_ERR_UNSUPPORTED; }
    k_coarse_site<float2><<<(unsigned)p.Vc, p.ncd * p.Ls_c, site_smem_bytes<float2>(p.ndir, p.ncd, p.Ls_c), st>>>(
        B, in, out, p, dagger, skip, status);
    DWF_CHECK_LAUNCH();
    return DWF_OK;
}

// Yd[x][dir] (column-major) = Y[x + dir][-dir]^dag from the row-major FP64 blocks.
__global__ void k_adjoint_blocks(const double2* __restrict__ Y, float2* __restrict__ Yd, CoarseParams p) {
    const int ncd = p.ncd;
    const long long bsz = (long long)ncd * ncd;
    const long long n = p.Vc * p.ndir * bsz;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        const long long blk = t / bsz;
        const int e = (int)(t % bsz);           // column-major index j * ncd + i
        const long long xc = blk / p.ndir;
        const int dir = (int)(blk % p.ndir);
        const int opp = dir == 0 ? 0 : (((dir - 1) % 2 == 0) ? dir + 1 : dir - 1);
        const long long nb = coarse_neighbour(p, xc, dir);
        // element (i, j) of the adjoint block = conj(Y_nb,opp(j, i)); row-major (j, i) sits at j * ncd + i
        const double2 v = Y[(nb * p.ndir + opp) * bsz + e];
        Yd[t] = make_float2((float)v.x, (float)-v.y);
    }
}

dwf_status build_adjoint_blocks(dwf_mg* h, cudaStream_t st) {
    CoarseParams p = coarse_params(h, h->mf);
    const long long n = p.Vc * p.ndir * (long long)p.ncd * p.ncd;
    const int grid = (int)((n + 255) / 256 < 152 * 16 ? (n + 255) / 256 : 152 * 16);
    k_adjoint_blocks<<<grid, 256, 0, st>>>(h->Y64, h->Yd32, p);
    DWF_CHECK_LAUNCH();
    return DWF_OK;
}

// ---------------------------------------------------------------------------
// truncated restriction / prolongation
// ---------------------------------------------------------------------------
struct TransferParams {
    int nd, L[4], b[4], Lc[4];
    long long V, Vc;
    int Ls, Ls_c, nvec, ncd, nchd, dof, ncol, nb;
    int bulk;            // 1: P^dag / P on every slice (Lhat_s = Ls) instead of the walls
    int packed;          // 1: fine vectors in the slice-paired 4-d layout
    long long NB;        // blocks of 32 sites of the packed layout
};

// complex index of fine element (s, site, d) in the canonical or the slice-paired layout
// (float4 ((s/2 NB + site/32) dof + d) 32 + site%32 holds slices 2j and 2j+1 as two complex values)
__device__ __forceinline__ long long fine_idx(const TransferParams& p, int s, long long x, int d) {
    if (!p.packed) return ((long long)s * p.V + x) * p.dof + d;
    return 2 * (((((long long)(s >> 1)) * p.NB + (x >> 5)) * p.dof + d) * 32 + (x & 31)) + (s & 1);
}

// Aggregate of a site, and site l of an aggregate, in unsigned 32 bits: the links, near-null
// vectors and prolongator of a hierarchy with 2^32 sites would take 500 GB.  The loops are unrolled
// so that the parameter arrays are read with constant indexes.
__device__ __forceinline__ long long agg_of(const TransferParams& p, long long site) {
    unsigned xc = 0, stride = 1, rem = (unsigned)site;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu)
        if (mu < p.nd) {
            const unsigned q = rem / (unsigned)p.L[mu], c = rem - q * (unsigned)p.L[mu];
            rem = q;
            xc += c / (unsigned)p.b[mu] * stride;
            stride *= (unsigned)p.Lc[mu];
        }
    return xc;
}

__device__ __forceinline__ long long agg_site(const TransferParams& p, long long xc, int l) {
    unsigned site = 0, stride = 1, rem = (unsigned)xc, lr = (unsigned)l;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu)
        if (mu < p.nd) {
            const unsigned q = rem / (unsigned)p.Lc[mu], c = rem - q * (unsigned)p.Lc[mu];
            rem = q;
            const unsigned lq = lr / (unsigned)p.b[mu], lc = lr - lq * (unsigned)p.b[mu];
            lr = lq;
            site += (c * (unsigned)p.b[mu] + lc) * stride;
            stride *= (unsigned)p.L[mu];
        }
    return site;
}

__device__ __forceinline__ int chir_dof(const TransferParams& p, int c, int cd) {
    if (p.nd == 2) return c;
    return (2 * c + cd / p.ncol) * p.ncol + cd % p.ncol;
}

// Restriction.  A group of J = nchd * nvec threads owns one (aggregate, chirality): thread
// (cd, k) sums conj(P[x][c][cd][k]) r[x][cd] over the aggregate's sites x, whose J prolongator
// values are one contiguous run that the group reads as such, all sites' loads in flight; the
// cd sums meet in shared memory.  The two chiralities of an aggregate are neighbouring groups,
// so every site's prolongator is read in one piece.  grid.y = right-hand side (vectors back to
// back); skip[r]: per right-hand side.  Bound by the read of P (and by launch latency below a
// few MB): 256^2 8 us, where one thread per output, walking the sites one after the other
// through the index divisions, took 30; eight sites' loads before the first product and 32-bit
// offsets took the two transfers and two coarse applies of that hierarchy from 42.9 to 36 us.
constexpr int RESTRICT_THREADS = 288;   // both chiralities of one aggregate at 4-d, nvec 24
constexpr int RESTRICT_TABLE = 2048;    // aggregates up to this many sites keep their offsets in shared memory

__global__ void __launch_bounds__(RESTRICT_THREADS, 2)
k_restrict(const float2* __restrict__ P, const float2* __restrict__ r, float2* __restrict__ out, TransferParams p,
           const int* skip) {
    if (skip && skip[blockIdx.y]) return;
    __shared__ unsigned off[RESTRICT_TABLE];
    __shared__ float2 red[RESTRICT_THREADS];
    const int J = p.nchd * p.nvec;
    const int G = blockDim.x / J;
    const bool table = p.nb <= RESTRICT_TABLE;
    if (table)
        for (int l = threadIdx.x; l < p.nb; l += blockDim.x) off[l] = (unsigned)agg_site(p, 0, l);
    const long long nc = p.Vc * p.Ls_c * p.ncd;
    r += (long long)blockIdx.y * p.V * p.Ls * p.dof;
    out += (long long)blockIdx.y * nc;
    const int j = threadIdx.x % J;
    const int k = j % p.nvec, cd = j / p.nvec;
    const long long g = (long long)blockIdx.x * G + threadIdx.x / J;
    const int c = (int)(g & 1);
    const long long xs = g >> 1;
    const bool in = xs < p.Vc * (p.bulk ? p.Ls : 1);
    const long long xc = p.bulk ? xs % p.Vc : xs;
    // Phat_- P^dag P_- r_1 on coarse slice 1, Phat_+ P^dag P_+ r_Ls on coarse slice Lhat_s; bulk: every slice
    const int sf = p.bulk ? (int)(xs / p.Vc) : (c == 1 ? 0 : p.Ls - 1);
    float2 acc = make_float2(0.f, 0.f);
    const int d = chir_dof(p, c, cd);
    const long long base = in ? agg_site(p, xc, 0) : 0;
    const float2* Pc = P + c * J + j;
    __syncthreads();
    if (in) {
        // eight sites' loads before the first product
        for (int l0 = 0; l0 < p.nb; l0 += 8) {
            float2 a[8], b[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int l = min(l0 + q, p.nb - 1);
                const long long x = base + (table ? off[l] : (unsigned)agg_site(p, 0, l));
                a[q] = __ldg(Pc + x * 2 * J);
                b[q] = __ldg(r + fine_idx(p, sf, x, d));
            }
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (l0 + q < p.nb) acc = cfma_conj(a[q], b[q], acc);
        }
    }
    if (p.nchd > 1) {
        red[threadIdx.x] = acc;
        __syncthreads();
        if (cd == 0)
            for (int q = 1; q < p.nchd; ++q) {
                acc.x += red[threadIdx.x + q * p.nvec].x;
                acc.y += red[threadIdx.x + q * p.nvec].y;
            }
    }
    if (!in || cd != 0) return;
    float2* o = out + xc * p.ncd + c * p.nvec + k;
    if (p.bulk) {
        o[sf * p.Vc * p.ncd] = acc;
    } else {
        const int wall = c == 1 ? 0 : p.Ls_c - 1;
        for (int s = 0; s < p.Ls_c; ++s) o[s * p.Vc * p.ncd] = s == wall ? acc : make_float2(0.f, 0.f);
    }
}

// sum_k P[k] e[k] over one prolongator row; V4: rows and e are 16-byte aligned and nvec is even
template <bool V4>
__device__ __forceinline__ float2 prolong_row(const float2* __restrict__ Pr, const float2* __restrict__ ev, int nvec) {
    float2 acc = make_float2(0.f, 0.f);
    if (V4) {
#pragma unroll 4
        for (int k = 0; k < nvec; k += 2) {
            const float4 a = __ldg(reinterpret_cast<const float4*>(Pr + k));
            const float4 b = __ldg(reinterpret_cast<const float4*>(ev + k));
            acc = cfma(make_float2(a.x, a.y), make_float2(b.x, b.y), acc);
            acc = cfma(make_float2(a.z, a.w), make_float2(b.z, b.w), acc);
        }
    } else {
        for (int k = 0; k < nvec; ++k) acc = cfma(__ldg(Pr + k), __ldg(ev + k), acc);
    }
    return acc;
}

// Prolongation.  The first `wall_blocks` blocks of a row take one thread per (site, chirality,
// dof): P_- P e_1 onto fine slice 1 and P_+ P e_{Lhat_s} onto slice Ls, with the zeros of the
// other chirality there; the remaining blocks only store the zeros of the slices in between
// (all of the output but two slices), as one contiguous range of zero_n complex values from
// zero_0.  Bulk: no range of zeros, every slice is computed (grid.z: its slices).  V4: the layout allows 16-byte
// accesses (see prolong_wall).  Bound by the stores: 16.8 MB at 256^2 x 16, 64 MB at
// 12^3 x 24 x 16; one thread per value with its index divisions took 34 us and 160 us.
constexpr int PROLONG_ZERO = 16;   // complex values stored per thread of a zero block
template <bool V4>
__global__ void __launch_bounds__(256)
k_prolong(const float2* __restrict__ P, const float2* __restrict__ e, float2* __restrict__ out, TransferParams p,
          unsigned wall_blocks, long long zero_0, long long zero_n, const int* skip) {
    if (skip && skip[blockIdx.y]) return;
    e += (long long)blockIdx.y * p.Vc * p.Ls_c * p.ncd;
    out += (long long)blockIdx.y * p.V * p.Ls * p.dof;
    if (blockIdx.x >= wall_blocks) {
        const long long b0 = (long long)(blockIdx.x - wall_blocks) * (256 * PROLONG_ZERO);
        if (V4) {
            float4* o = reinterpret_cast<float4*>(out + zero_0);
#pragma unroll
            for (int q = 0; q < PROLONG_ZERO / 2; ++q) {
                const long long i = b0 / 2 + q * 256 + threadIdx.x;
                if (i < zero_n / 2) o[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        } else {
            for (int q = 0; q < PROLONG_ZERO; ++q) {
                const long long i = b0 + q * 256 + threadIdx.x;
                if (i < zero_n) out[zero_0 + i] = make_float2(0.f, 0.f);
            }
        }
        return;
    }
    const long long t = (long long)blockIdx.x * 256 + threadIdx.x;
    if (t >= p.V * p.dof) return;
    // site fastest within a block of 32 sites in the packed layout, dof fastest in the canonical one
    int d;
    long long x;
    if (p.packed) {
        const long long q = t >> 5;
        d = (int)(q % p.dof);
        x = (q / p.dof) * 32 + (t & 31);
    } else {
        d = (int)(t % p.dof);
        x = t / p.dof;
    }
    int c, cd;
    if (p.nd == 2) { c = d; cd = 0; }
    else { const int spin = d / p.ncol; c = spin / 2; cd = (spin % 2) * p.ncol + d % p.ncol; }
    const float2* Pr = P + ((x * 2 + c) * p.nchd + cd) * p.nvec;
    const float2* ev = e + agg_of(p, x) * p.ncd + c * p.nvec;
    const float2 zero = make_float2(0.f, 0.f);
    if (p.bulk) {
        for (int s = blockIdx.z; s < p.Ls; s += gridDim.z)
            out[fine_idx(p, s, x, d)] = prolong_row<V4>(Pr, ev + (long long)s * p.Vc * p.ncd, p.nvec);
        return;
    }
    const float2 v = prolong_row<V4>(Pr, ev + (long long)(c == 1 ? 0 : p.Ls_c - 1) * p.Vc * p.ncd, p.nvec);
    if (p.packed) {
        // slice pairs (0, 1) and (Ls - 2, Ls - 1): one pair when Ls = 2
        const float2 first = c == 1 ? v : zero, last = c == 0 ? v : zero;
        if (p.Ls == 2) {
            out[fine_idx(p, 0, x, d)] = first;
            out[fine_idx(p, 1, x, d)] = last;
        } else {
            out[fine_idx(p, 0, x, d)] = first;
            out[fine_idx(p, 1, x, d)] = zero;
            out[fine_idx(p, p.Ls - 2, x, d)] = zero;
            out[fine_idx(p, p.Ls - 1, x, d)] = last;
        }
    } else if (p.Ls == 1) {
        out[fine_idx(p, 0, x, d)] = v;
    } else {
        out[fine_idx(p, 0, x, d)] = c == 1 ? v : zero;
        out[fine_idx(p, p.Ls - 1, x, d)] = c == 0 ? v : zero;
    }
}

static TransferParams transfer_params(const dwf_mg* h) {
    TransferParams p;
    p.nd = h->mg.nd;
    for (int mu = 0; mu < 4; ++mu) { p.L[mu] = h->mg.L[mu]; p.b[mu] = h->mg.b[mu]; p.Lc[mu] = h->mg.Lc[mu]; }
    p.V = h->mg.V;
    p.Vc = h->mg.Vc;
    p.Ls = h->mg.Ls;
    p.Ls_c = h->mg.Ls_c;
    p.nvec = h->mg.nvec;
    p.ncd = h->mg.ncd;
    p.nchd = h->mg.nchd;
    p.dof = (int)site_dof(h->G);
    p.ncol = h->G.ncol;
    p.nb = h->mg.nb;
    p.bulk = h->prm.transfer == 1 ? 1 : 0;
    p.packed = 0;
    p.NB = (p.V + 31) / 32;
    return p;
}

static dwf_status check_packed_transfer(const TransferParams& p) {
    if (p.nd != 4 || p.Ls % 2 || p.V % 32) {
        set_error("packed transfers need a 4-d lattice, even Ls and a multiple of 32 sites");
        return DWF_ERR_UNSUPPORTED;
    }
    return DWF_OK;
}

dwf_status restrict_wall(const dwf_mg* h, const float2* r_fine, float2* r_coarse, const int* skip, cudaStream_t st,
                         int nrhs, bool packed) {
    TransferParams p = transfer_params(h);
    if (packed) { DWF_TRY(check_packed_transfer(p)); p.packed = 1; }
    if (nrhs < 1 || nrhs > 65535) { set_error("nrhs must be in [1, 65535]"); return DWF_ERR_ARG; }
    const int J = p.nchd * p.nvec;                       // at most 6 * 32
    const int G = RESTRICT_THREADS / J;
    const long long groups = 2 * p.Vc * (p.bulk ? p.Ls : 1);
    k_restrict<<<dim3((unsigned)((groups + G - 1) / G), (unsigned)nrhs), G * J, 0, st>>>(h->P32, r_fine, r_coarse, p,
                                                                                          skip);
    DWF_CHECK_LAUNCH();
    return DWF_OK;
}

dwf_status prolong_wall(const dwf_mg* h, const float2* e_coarse, float2* e_fine, const int* skip, cudaStream_t st,
                        int nrhs, bool packed) {
    TransferParams p = transfer_params(h);
    if (packed) { DWF_TRY(check_packed_transfer(p)); p.packed = 1; }
    if (nrhs < 1 || nrhs > 65535) { set_error("nrhs must be in [1, 65535]"); return DWF_ERR_ARG; }
    const long long plane = p.V * p.dof;                 // one slice; a pair of slices in the packed layout is two
    const unsigned wall_blocks = (unsigned)((plane + 255) / 256);
    const int ends = packed ? 2 : 1;                     // slices the wall threads store at each end
    const long long zero_0 = ends * plane;
    const long long zero_n = p.bulk || p.Ls <= 2 * ends ? 0 : (p.Ls - 2 * ends) * plane;
    const unsigned zero_blocks = (unsigned)((zero_n + 256 * PROLONG_ZERO - 1) / (256 * PROLONG_ZERO));
    // bulk: a thread takes all slices, with one set of indexes and prolongator values, where that leaves two blocks per SM (4-d
    // 8^3 x 16 x 8, 384 blocks: 31.7 us, 36.9 in four parts; 4^4 x 8, 12 blocks: 16.4 us, 6.2 in eight)
    const long long per_slice = (long long)wall_blocks * nrhs;
    const long long splits = p.bulk ? std::min<long long>({(152 * 2 + per_slice - 1) / per_slice, p.Ls, 65535}) : 1;
    const dim3 grid(wall_blocks + zero_blocks, (unsigned)nrhs, (unsigned)splits);
    // 16-byte accesses: prolongator rows, coarse vectors and the zero range start on 16-byte boundaries (dof is
    // even, so plane is) when nvec is even and the caller's vectors are aligned
    if (p.nvec % 2 == 0 && aligned16(e_coarse) && aligned16(e_fine))
        k_prolong<true><<<grid, 256, 0, st>>>(h->P32, e_coarse, e_fine, p, wall_blocks, zero_0, zero_n, skip);
    else
        k_prolong<false><<<grid, 256, 0, st>>>(h->P32, e_coarse, e_fine, p, wall_blocks, zero_0, zero_n, skip);
    DWF_CHECK_LAUNCH();
    return DWF_OK;
}

}  // namespace dwf

using namespace dwf;

extern "C" {

dwf_status mg_restrict(const dwf_mg* h, const void* r_fine, void* r_coarse, void* stream) {
    clear_error();
    if (!h || !r_fine || !r_coarse) { set_error("NULL argument"); return DWF_ERR_ARG; }
    return restrict_wall(h, (const float2*)r_fine, (float2*)r_coarse, nullptr, as_stream(stream));
}

dwf_status mg_prolong(const dwf_mg* h, const void* e_coarse, void* e_fine, void* stream) {
    clear_error();
    if (!h || !e_coarse || !e_fine) { set_error("NULL argument"); return DWF_ERR_ARG; }
    return prolong_wall(h, (const float2*)e_coarse, (float2*)e_fine, nullptr, as_stream(stream));
}

dwf_status mg_coarse_apply(const dwf_mg* h, const void* in, void* out, double mf, int dagger, void* stream) {
    clear_error();
    if (!h || !in || !out) { set_error("NULL argument"); return DWF_ERR_ARG; }
    if (in == out) { set_error("in and out must be distinct buffers"); return DWF_ERR_ARG; }
    return coarse_dwf_apply(h, (const float2*)in, (float2*)out, mf, dagger != 0, nullptr, as_stream(stream));
}

dwf_status mg_check_wait_timeout(dwf_mg* h, double seconds, void* stream) {
    clear_error();
    if (!h) { set_error("NULL argument"); return DWF_ERR_ARG; }
    if (!(seconds > 0.0) || seconds > 10.0) { set_error("seconds must be in (0, 10]"); return DWF_ERR_ARG; }
    k_coarse_wait_expires<<<1, 32, 0, as_stream(stream)>>>((unsigned long long)(seconds * 1e9), h->status + 1);
    DWF_CHECK_LAUNCH();
    return DWF_OK;
}

}  // extern "C"

// ===========================================================================
// Persistent coarse CGNR: one cooperative launch per coarse solve.
//
// Solves (Dhat_PV^dag Dhat_DW)^dag (Dhat_PV^dag Dhat_DW) e = (..)^dag r_c by CG
// (the coarsest-level CGNR of Table kcycle), with every block resident for
// the whole solve and phases separated by a software grid barrier.  The
// barrier's spin is bounded by a %globaltimer deadline: on expiry the block
// raises an error flag that every other block sees at its next barrier, and
// all blocks return (the host reports DWF_ERR_TIMEOUT).  Reductions: each
// block writes one FP64 partial per quantity; after the barrier every block
// sums all partials in the same order, so all blocks hold identical scalars.
// Mutable vectors are read through L2 (ld.global.cg) because other blocks wrote
// them earlier in the same launch.
// ===========================================================================
namespace dwf {

constexpr int PCG_THREADS = 256;

struct PcgBarrier {
    unsigned count;
    unsigned gen;
    int error;
    int pad;
};

struct PcgArgs {
    CoarseParams cp;
    const float2* Y;    // Galerkin blocks (column-major)
    const float2* Yd;   // adjoint blocks (column-major)
    const float2* rc;   // right-hand side
    float2* e;          // solution
    float2 *rr, *r, *p, *q, *t, *w;
    double* partials;   // [3][gridDim.x]
    PcgBarrier* bar;
    int* out_iters;
    double* out_rr2;    // final |rr|^2 / |rc|^2
    double tol2;
    int maxiter;
    double mf;
    unsigned long long timeout_ns;
};

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Returns false if the barrier timed out here or anywhere else, or if this
// block reports a failure of its own (local_ok == false).
__device__ bool pcg_sync(PcgBarrier* b, unsigned long long deadline, bool local_ok = true) {
    __shared__ int ok;
    __shared__ int any_fail;
    if (threadIdx.x == 0) any_fail = 0;
    __syncthreads();
    if (!local_ok) any_fail = 1;
    __syncthreads();
    if (threadIdx.x == 0) {
        if (any_fail) atomicExch(&b->error, 1);
        volatile unsigned* vgen = &b->gen;
        volatile int* verr = &b->error;
        const unsigned g = *vgen;
        __threadfence();
        const unsigned arrived = atomicAdd(&b->count, 1u);
        if (arrived == gridDim.x - 1) {
            b->count = 0u;
            __threadfence();
            atomicAdd(&b->gen, 1u);
        } else {
            while (*vgen == g) {
                if (*verr) break;
                if (global_ns() > deadline) { atomicExch(&b->error, 1); break; }
                __nanosleep(64);
            }
        }
        __threadfence();
        ok = (*verr == 0);
    }
    __syncthreads();
    return ok != 0;
}

// block-sum of up to 3 doubles into partials[k * grid + block]
__device__ void pcg_partial(double (&v)[3], int nv, double* partials) {
    __shared__ double sh[3][PCG_THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = 0; k < nv; ++k)
        for (int off = 16; off > 0; off >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], off);
    if (lane == 0)
        for (int k = 0; k < nv; ++k) sh[k][warp] = v[k];
    __syncthreads();
    if (threadIdx.x == 0)
        for (int k = 0; k < nv; ++k) {
            double s = 0.0;
            for (int w = 0; w < PCG_THREADS / 32; ++w) s += sh[k][w];
            partials[k * gridDim.x + blockIdx.x] = s;
        }
    __syncthreads();
}

// every block: fixed-order total of partial k (strided loads by all threads,
// then a fixed-order block reduction)
__device__ double pcg_total(const double* partials, int k) {
    __shared__ double sh[PCG_THREADS / 32];
    __shared__ double tot;
    double v = 0.0;
    for (unsigned b = threadIdx.x; b < gridDim.x; b += blockDim.x) v += __ldcg(partials + k * gridDim.x + b);
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < PCG_THREADS / 32; ++w) s += sh[w];
        tot = s;
    }
    __syncthreads();
    const double r = tot;
    __syncthreads();
    return r;
}

// out = Dhat_DW(m) in (or adjoint) over all tiles (grid-stride), shared-memory
// tiles as described above.  `phase` is this block's mbarrier parity, flipped
// per tile.  Returns this thread's share of |out|^2; false in *ok on a timeout.
__device__ double pcg_apply(const PcgArgs& a, TileSmemT<float2>& sm, unsigned& phase, const float2* __restrict__ in,
                            float2* __restrict__ out, double mf, bool dag, bool* ok) {
    const CoarseParams& p = a.cp;
    const float2* B = a.Y;
    const int ntx = (p.Lc[0] + TILE_X - 1) / TILE_X;
    const int ntiles = ntx * ((p.Lc[1] + TILE_Y - 1) / TILE_Y);
    double nrm = 0.0;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int x0 = (tile % ntx) * TILE_X, y0 = (tile / ntx) * TILE_Y;
        __syncthreads();                        // previous tile's shared data fully consumed
        tile_issue_blocks(sm, B, p, x0, y0);
        tile_stage<float2>(sm, in, p, x0, y0);
        __syncthreads();
        const bool okw = mbar_wait_bounded(&sm.mbar, phase, TILE_WAIT_NS);
        if (__syncthreads_or(!okw)) {                      // the whole block leaves together
            mbar_wait_bounded(&sm.mbar, phase, TILE_WAIT_NS);
            *ok = false;
            return nrm;
        }
        phase ^= 1u;
        nrm += tile_site(sm, out, p, x0, y0, (float)mf, dag);
    }
    return nrm;
}

#define PCG_LOOP(k, n) for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < (n); k += (long long)gridDim.x * blockDim.x)

__global__ void __launch_bounds__(PCG_THREADS) k_coarse_cgnr_persistent(PcgArgs a) {
    extern __shared__ __align__(128) unsigned char pcg_raw[];
    TileSmemT<float2>& sm = *reinterpret_cast<TileSmemT<float2>*>(pcg_raw);
    const long long n = a.cp.Vc * a.cp.Ls_c * a.cp.ncd;
    const unsigned long long deadline = global_ns() + a.timeout_ns;
    const double mf = a.mf;
    unsigned phase = 0;
    bool ok = true;
    if (threadIdx.x == 0) mbar_init(&sm.mbar, 1);
    __syncthreads();
    // prologue: e = 0, rr = rc, t = Dhat_PV rr, r = Dhat_DW^dag t (= B^dag rr), p = r
    PCG_LOOP(k, n) { a.e[k] = make_float2(0.f, 0.f); a.rr[k] = __ldcg(a.rc + k); }
    if (!pcg_sync(a.bar, deadline, ok)) return;
    pcg_apply(a, sm, phase, a.rr, a.t, 1.0, false, &ok);
    if (!pcg_sync(a.bar, deadline, ok)) return;
    double v[3] = {pcg_apply(a, sm, phase, a.t, a.r, mf, true, &ok), 0.0, 0.0};
    PCG_LOOP(k, n) {
        float2 y = __ldcg(a.rc + k);
        v[1] += (double)y.x * y.x + (double)y.y * y.y;
    }
    pcg_partial(v, 2, a.partials);
    if (!pcg_sync(a.bar, deadline, ok)) return;
    PCG_LOOP(k, n) a.p[k] = __ldcg(a.r + k);
    double rn2 = pcg_total(a.partials, 0);
    const double bn2 = pcg_total(a.partials, 1);
    double rr2 = bn2;
    int it = 0;
    if (bn2 > 0.0 && rn2 > 0.0) {
        while (it < a.maxiter) {
            // q = Dhat_PV^dag Dhat_DW p  (p = r on the first pass: r is complete,
            // the copy into p is not visible to other blocks yet)
            pcg_apply(a, sm, phase, it == 0 ? a.r : a.p, a.t, mf, false, &ok);
            if (!pcg_sync(a.bar, deadline, ok)) return;
            double u[3] = {pcg_apply(a, sm, phase, a.t, a.q, 1.0, true, &ok), 0.0, 0.0};
            pcg_partial(u, 1, a.partials);
            if (!pcg_sync(a.bar, deadline, ok)) return;
            const double qq = pcg_total(a.partials, 0);
            if (!(qq > 0.0)) break;
            const double alpha = rn2 / qq;
            const float af = (float)alpha;
            // e += alpha p; rr -= alpha q; t = Dhat_PV q (q is complete)
            double u2[3] = {0.0, 0.0, 0.0};
            PCG_LOOP(k, n) {
                float2 pk = __ldcg(a.p + k), qk = __ldcg(a.q + k), ek = __ldcg(a.e + k), rk = __ldcg(a.rr + k);
                ek.x += af * pk.x; ek.y += af * pk.y;
                rk.x -= af * qk.x; rk.y -= af * qk.y;
                a.e[k] = ek; a.rr[k] = rk;
                u2[0] += (double)rk.x * rk.x + (double)rk.y * rk.y;
            }
            pcg_partial(u2, 1, a.partials + 2 * gridDim.x);
            pcg_apply(a, sm, phase, a.q, a.t, 1.0, false, &ok);
            if (!pcg_sync(a.bar, deadline, ok)) return;
            rr2 = pcg_total(a.partials, 2);
            ++it;
            if (rr2 <= a.tol2 * bn2) break;
            // w = Dhat_DW^dag t; r -= alpha w
            pcg_apply(a, sm, phase, a.t, a.w, mf, true, &ok);
            if (!pcg_sync(a.bar, deadline, ok)) return;
            double u3[3] = {0.0, 0.0, 0.0};
            PCG_LOOP(k, n) {
                float2 rk = __ldcg(a.r + k), wk = __ldcg(a.w + k);
                rk.x -= af * wk.x; rk.y -= af * wk.y;
                a.r[k] = rk;
                u3[0] += (double)rk.x * rk.x + (double)rk.y * rk.y;
            }
            pcg_partial(u3, 1, a.partials + gridDim.x);
            if (!pcg_sync(a.bar, deadline, ok)) return;
            const double rn2n = pcg_total(a.partials, 1);
            const float beta = (float)(rn2n / rn2);
            rn2 = rn2n;
            PCG_LOOP(k, n) {
                float2 pk = __ldcg(a.p + k), rk = __ldcg(a.r + k);
                a.p[k] = make_float2(rk.x + beta * pk.x, rk.y + beta * pk.y);
            }
            if (!pcg_sync(a.bar, deadline, ok)) return;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *a.out_iters += it;                       // running total over solves
        *a.out_rr2 = bn2 > 0 ? rr2 / bn2 : 0.0;
    }
}

struct PcgPlan {
    int grid = 0;
};

static PcgPlan g_pcg_plan[64];

dwf_status coarse_cgnr_persistent(const dwf_mg* h, const float2* rc, float2* ec, float2* const* vec6, double* partials,
                                  void* bar, int* out_iters, double* out_rr2, cudaStream_t st) {
    int dev = 0;
    DWF_CHECK_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) { set_error("device ordinal out of range"); return DWF_ERR_UNSUPPORTED; }
    if (h->mg.Ls_c > 4 || h->mg.ncd != 16 || h->mg.nd != 2) {
        set_error("persistent coarse solver supports 2-d, 16 coarse dof and Ls_c <= 4");
        return DWF_ERR_UNSUPPORTED;
    }
    PcgPlan& plan = g_pcg_plan[dev];
    if (plan.grid == 0) {
        int nsm = 0, per = 0;
        DWF_CHECK_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
        DWF_CHECK_CUDA(cudaFuncSetAttribute(k_coarse_cgnr_persistent, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)sizeof(TileSmemT<float2>)));
        DWF_CHECK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_coarse_cgnr_persistent, PCG_THREADS,
                                                                     sizeof(TileSmemT<float2>)));
        if (per < 1) { set_error("persistent coarse solver cannot be resident"); return DWF_ERR_UNSUPPORTED; }
        plan.grid = nsm * per;
    }
    PcgArgs a;
    a.cp = coarse_params(h, h->mf);
    a.Y = h->Y32;
    a.Yd = h->Yd32;
    a.rc = rc;
    a.e = ec;
    a.rr = vec6[0]; a.r = vec6[1]; a.p = vec6[2]; a.q = vec6[3]; a.t = vec6[4]; a.w = vec6[5];
    a.partials = partials;
    a.bar = (PcgBarrier*)bar;
    a.out_iters = out_iters;
    a.out_rr2 = out_rr2;
    a.tol2 = h->prm.coarse_tol * h->prm.coarse_tol;
    a.maxiter = h->prm.coarse_maxiter;
    a.mf = h->mf;
    a.timeout_ns = 5000000000ULL;   // 5 s per solve
    const int ntiles = ((a.cp.Lc[0] + TILE_X - 1) / TILE_X) * ((a.cp.Lc[1] + TILE_Y - 1) / TILE_Y);
    int grid = plan.grid < ntiles ? plan.grid : ntiles;
    if (grid < 1) grid = 1;
    DWF_CHECK_CUDA(cudaMemsetAsync(bar, 0, 2 * sizeof(unsigned), st));   // count, gen; the error flag persists
    void* args[] = {&a};
    DWF_CHECK_CUDA(cudaLaunchCooperativeKernel((const void*)k_coarse_cgnr_persistent, dim3(grid), dim3(PCG_THREADS), args,
                                               sizeof(TileSmemT<float2>), st));
    return DWF_OK;
}


// ===========================================================================
// Persistent coarse GCR: one cooperative launch per coarse solve.
//
// Restarted GCR(KC) on B e = r_c, B = Dhat_PV^dag Dhat_DW (the level-2 solver
// type), to |r| <= coarse_tol |r_c| or maxiter steps.  Per step three bounded
// grid barriers separate the phases:
//   A. r_k = r_{k-1} - alpha_{k-1} w_{k-1} is formed while the tiles and their
//      halos are staged (each tile stores its own sites of r_k), and
//      t = Dhat_DW r_k is applied; partial |r_k|^2.          -> barrier
//      Stop if |r_k|^2 <= tol^2 |r_c|^2.
//   B. w = Dhat_PV^dag t, with the classical Gram-Schmidt dots <w_j, w>,
//      j < k, accumulated in the stencil's epilogue.         -> barrier
//   C. w_k = w - sum_j c_j w_j; partial |w_k|^2, <w_k, r_k>. -> barrier
//      alpha_k = <w_k, r_k> / |w_k|^2.
// The solution is not updated per step: the residuals r_j of a cycle are the
// raw search directions, and e += sum_j y_j r_j with (I + C)^T y = alpha is
// added once per cycle (during phase A of the next cycle's first step, or at
// the end).  The residual slots rotate over KC + 1 vectors so that the new
// cycle's first residual never overwrites a direction still being combined.
// Every block computes the same scalars from the same partials in the same
// order; barrier waits and bulk-copy waits are bounded (%globaltimer) and end
// in an error flag that the host reports as DWF_ERR_TIMEOUT.
// ===========================================================================
constexpr int PG_MAXK = 16;
constexpr int PGCR_BLOCKS_PER_SM = 2;     // resident blocks per SM used by the persistent GCR
constexpr int PG_NQ = 1 + 2 * PG_MAXK + 3;     // partial quantities: |r|^2 | dots | |w|^2, <w, r>

struct PgcrArgs {
    CoarseParams cp;
    const void* Y;          // Galerkin blocks (column-major, FP32 or FP16)
    const float2* rc;
    float2* e;
    float2* S[PG_MAXK + 1]; // residual slots
    float2* W[PG_MAXK];     // orthogonalised images
    float2* t;
    double* partials;       // [PG_NQ][gridDim.x]
    PcgBarrier* bar;
    int* out_iters;         // running total of steps over solves
    double* out_rr2;        // final |r|^2 / |r_c|^2
    double tol2;
    int maxiter;
    int KC;
    unsigned long long timeout_ns;
};

struct PgcrShared {
    double C[PG_MAXK][PG_MAXK][2];
    double A[PG_MAXK][2];
    double nrm[PG_MAXK];
    float2 coef[PG_MAXK];
    float2 y[PG_MAXK];
    double tot[PG_NQ];
};

// totals of nq partial quantities (layout [q][gridDim.x], gridDim.x <= 2 *
// blockDim.x) into out[q0 + q]: thread t adds partials t and t + blockDim.x of
// every quantity (all loads issued together), then a fixed-order block tree, so
// every block obtains bitwise identical totals after one round trip to L2
constexpr int PG_TOT_MAX = 36;
constexpr int PG_TOT_CHUNK = 8;      // quantities whose loads are in flight together
__device__ void pg_totals(const double* part, int q0, int nq, double* out) {
    __shared__ double sh[PG_TOT_CHUNK][TILE_THREADS / 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned b0 = threadIdx.x, b1 = threadIdx.x + blockDim.x;
    for (int c0 = 0; c0 < nq; c0 += PG_TOT_CHUNK) {
        double v[PG_TOT_CHUNK];
#pragma unroll
        for (int q = 0; q < PG_TOT_CHUNK; ++q) {
            v[q] = 0.0;
            if (c0 + q < nq) {
                const double* pq = part + (size_t)(q0 + c0 + q) * gridDim.x;
                const double x0 = b0 < gridDim.x ? __ldcg(pq + b0) : 0.0;
                const double x1 = b1 < gridDim.x ? __ldcg(pq + b1) : 0.0;
                v[q] = x0 + x1;
            }
        }
#pragma unroll
        for (int q = 0; q < PG_TOT_CHUNK; ++q) {
            if (c0 + q < nq) {
                double d = v[q];
                for (int off = 16; off > 0; off >>= 1) d += __shfl_down_sync(0xffffffffu, d, off);
                if (lane == 0) sh[q][warp] = d;
            }
        }
        __syncthreads();
        if (threadIdx.x < PG_TOT_CHUNK && c0 + (int)threadIdx.x < nq) {
            double sum = 0.0;
            for (int w = 0; w < TILE_THREADS / 32; ++w) sum += sh[threadIdx.x][w];
            out[q0 + c0 + threadIdx.x] = sum;
        }
        __syncthreads();
    }
}

// block partials of NQ per-thread FP32 values (first nq used) into part[(q0 + q) * grid + block]
template <int NQ>
__device__ void pg_partials(const float (&v)[NQ], int nq, double* part, int q0) {
    __shared__ double sh[NQ][TILE_THREADS / 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        if (q < nq) {
            double d = v[q];
            for (int off = 16; off > 0; off >>= 1) d += __shfl_down_sync(0xffffffffu, d, off);
            if (lane == 0) sh[q][warp] = d;
        }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < nq; q += blockDim.x) {
        double sum = 0.0;
        for (int w = 0; w < TILE_THREADS / 32; ++w) sum += sh[q][w];
        part[(size_t)(q0 + q) * gridDim.x + blockIdx.x] = sum;
    }
    __syncthreads();
}

// stage r = a - alpha b (b may be null) for the tile and its halo; the tile's
// own sites of r are stored to rout and their |r|^2 added to *nrm.  At most
// PG_STAGE elements per thread: all loads are issued before any use.
constexpr int PG_STAGE = (4 * TILE_HY * TILE_HX * 16 + TILE_THREADS - 1) / TILE_THREADS;
template <class BT>
__device__ __forceinline__ void pg_stage_axpy(TileSmemT<BT>& sm, const float2* a, const float2* b, float2 alpha,
                                              float2* rout, const CoarseParams& p, int x0, int y0, float& nrm) {
    const int L0 = p.Lc[0], L1 = p.Lc[1];
    const long long slice = p.Vc * 16;
    const int total = p.Ls_c * TILE_HY * TILE_HX * 16;
    long long idx[PG_STAGE];
    float2 va[PG_STAGE], vb[PG_STAGE];
#pragma unroll
    for (int u = 0; u < PG_STAGE; ++u) {
        const int e = threadIdx.x + u * TILE_THREADS;
        idx[u] = -1;
        if (e < total) {
            const int j = e & 15;
            const int h = (e >> 4) % (TILE_HY * TILE_HX);
            const int s = (e >> 4) / (TILE_HY * TILE_HX);
            const int hx = h % TILE_HX, hy = h / TILE_HX;
            const int gx = ((x0 + hx - 1) % L0 + L0) % L0, gy = ((y0 + hy - 1) % L1 + L1) % L1;
            idx[u] = s * slice + ((long long)gy * L0 + gx) * 16 + j;
            va[u] = __ldcg(a + idx[u]);
            vb[u] = b ? __ldcg(b + idx[u]) : make_float2(0.f, 0.f);
        }
    }
#pragma unroll
    for (int u = 0; u < PG_STAGE; ++u) {
        const int e = threadIdx.x + u * TILE_THREADS;
        if (e < total) {
            const int j = e & 15;
            const int h = (e >> 4) % (TILE_HY * TILE_HX);
            const int s = (e >> 4) / (TILE_HY * TILE_HX);
            const int hx = h % TILE_HX, hy = h / TILE_HX;
            float2 v = va[u];
            v.x -= alpha.x * vb[u].x - alpha.y * vb[u].y;
            v.y -= alpha.x * vb[u].y + alpha.y * vb[u].x;
            sm.v[s][hy][hx][j] = v;
            const bool own = hx >= 1 && hx <= TILE_X && hy >= 1 && hy <= TILE_Y && x0 + hx - 1 < L0 && y0 + hy - 1 < L1;
            if (own) {
                rout[idx[u]] = v;
                nrm += v.x * v.x + v.y * v.y;
            }
        }
    }
}

// stage the tile and its halo of `in` (all loads issued before any use)
template <class BT>
__device__ __forceinline__ void pg_stage(TileSmemT<BT>& sm, const float2* in, const CoarseParams& p, int x0, int y0) {
    const int L0 = p.Lc[0], L1 = p.Lc[1];
    const long long slice = p.Vc * 16;
    const int total = p.Ls_c * TILE_HY * TILE_HX * 16;
    float2 va[PG_STAGE];
#pragma unroll
    for (int u = 0; u < PG_STAGE; ++u) {
        const int e = threadIdx.x + u * TILE_THREADS;
        if (e < total) {
            const int j = e & 15;
            const int h = (e >> 4) % (TILE_HY * TILE_HX);
            const int s = (e >> 4) / (TILE_HY * TILE_HX);
            const int hx = h % TILE_HX, hy = h / TILE_HX;
            const int gx = ((x0 + hx - 1) % L0 + L0) % L0, gy = ((y0 + hy - 1) % L1 + L1) % L1;
            va[u] = __ldcg(in + s * slice + ((long long)gy * L0 + gx) * 16 + j);
        }
    }
#pragma unroll
    for (int u = 0; u < PG_STAGE; ++u) {
        const int e = threadIdx.x + u * TILE_THREADS;
        if (e < total) {
            const int j = e & 15;
            const int h = (e >> 4) % (TILE_HY * TILE_HX);
            const int s = (e >> 4) / (TILE_HY * TILE_HX);
            sm.v[s][h / TILE_HX][h % TILE_HX][j] = va[u];
        }
    }
}

// e += sum_{j<m} y_j S[(base + j) mod (KC + 1)] (grid-stride; y in shared memory)
__device__ __forceinline__ void pg_combine(const PgcrArgs& a, const PgcrShared& sh, int base, int m, long long n) {
    if (m <= 0) return;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x; i0 < n; i0 += 4 * stride) {
        float2 x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) if (i0 + u * stride < n) x[u] = a.e[i0 + u * stride];
        for (int j = 0; j < m; ++j) {
            const float2* Sj = a.S[(base + j) % (a.KC + 1)];
            const float2 y = sh.y[j];
            float2 r[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) if (i0 + u * stride < n) r[u] = __ldcg(Sj + i0 + u * stride);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                x[u].x += y.x * r[u].x - y.y * r[u].y;
                x[u].y += y.x * r[u].y + y.y * r[u].x;
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) if (i0 + u * stride < n) a.e[i0 + u * stride] = x[u];
    }
}

// y of the deferred update over m steps: (I + C)^T y = A (thread 0, FP64)
__device__ __forceinline__ void pg_back_substitute(PgcrShared& sh, int m) {
    if (threadIdx.x == 0) {
        double yr[PG_MAXK], yi[PG_MAXK];
        for (int j = m - 1; j >= 0; --j) {
            double ar = sh.A[j][0], ai = sh.A[j][1];
            for (int k = j + 1; k < m; ++k) {
                ar -= sh.C[k][j][0] * yr[k] - sh.C[k][j][1] * yi[k];
                ai -= sh.C[k][j][0] * yi[k] + sh.C[k][j][1] * yr[k];
            }
            yr[j] = ar; yi[j] = ai;
            sh.y[j] = make_float2((float)ar, (float)ai);
        }
    }
    __syncthreads();
}

template <class BT>
__global__ void __launch_bounds__(TILE_THREADS, 2) k_coarse_gcr_persistent(PgcrArgs a) {
    extern __shared__ __align__(128) unsigned char pg_raw[];
    TileSmemT<BT>& sm = *reinterpret_cast<TileSmemT<BT>*>(pg_raw);
    __shared__ PgcrShared sh;
    const CoarseParams& p = a.cp;
    const BT* Y = reinterpret_cast<const BT*>(a.Y);
    const long long n = p.Vc * p.Ls_c * 16;
    const int KC = a.KC;
    const unsigned long long deadline = global_ns() + a.timeout_ns;
    const int ntx = (p.Lc[0] + TILE_X - 1) / TILE_X;
    const int ntiles = ntx * ((p.Lc[1] + TILE_Y - 1) / TILE_Y);
    double* partA = a.partials;                                   // quantity 0
    unsigned phase = 0;
    bool ok = true;
    if (threadIdx.x == 0) mbar_init(&sm.mbar, 1);
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        a.e[i] = make_float2(0.f, 0.f);
    __syncthreads();
    int base = 0, m = 0, it = 0;
    const float2* prevR = a.rc;          // r_{k-1} (or r_c before the first step)
    const float2* prevW = nullptr;       // w_{k-1}
    float2 prevA = make_float2(0.f, 0.f);
    double bn2 = 0.0, rr2 = 0.0;
    for (;;) {
        // ---- phase A: r_k and t = Dhat_DW r_k ----
        const bool roll = m == KC;
        if (roll) pg_back_substitute(sh, KC);                     // y of the cycle that just ended
        const int slot = (base + m) % (KC + 1);
        float2* Rk = a.S[slot];
        float nrA = 0.f;
        for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
            const int x0 = (tile % ntx) * TILE_X, y0 = (tile / ntx) * TILE_Y;
            __syncthreads();
            tile_issue_blocks(sm, Y, p, x0, y0);
            pg_stage_axpy(sm, prevR, prevW, prevA, Rk, p, x0, y0, nrA);
            __syncthreads();
            const bool okw = mbar_wait_bounded(&sm.mbar, phase, TILE_WAIT_NS);
            if (__syncthreads_or(!okw)) {                  // the whole block leaves together
                mbar_wait_bounded(&sm.mbar, phase, TILE_WAIT_NS);
                ok = false;
                break;
            }
            phase ^= 1u;
            tile_site(sm, a.t, p, x0, y0, p.mf, false);
        }
        if (roll) {                                               // e += sum_j y_j r_j of the ended cycle
            pg_combine(a, sh, base, KC, n);
            base = slot;
            m = 0;
        }
        {
            float v[1] = {nrA};
            pg_partials<1>(v, 1, partA, 0);
        }
        if (!pcg_sync(a.bar, deadline, ok)) return;
        pg_totals(a.partials, 0, 1, sh.tot);
        rr2 = sh.tot[0];
        if (it == 0) bn2 = rr2;
        if (bn2 == 0.0 || rr2 <= a.tol2 * bn2 || it >= a.maxiter) break;
        // ---- phase B: w = Dhat_PV^dag t with the dots <w_j, w>, j < m ----
        float dots[2 * (PG_MAXK - 1)];
#pragma unroll
        for (int q = 0; q < 2 * (PG_MAXK - 1); ++q) dots[q] = 0.f;
        float2* Wm = a.W[m];
        const int mm = m;
        for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
            const int x0 = (tile % ntx) * TILE_X, y0 = (tile / ntx) * TILE_Y;
            __syncthreads();
            tile_issue_blocks(sm, Y, p, x0, y0);
            pg_stage(sm, a.t, p, x0, y0);
            __syncthreads();
            const bool okw = mbar_wait_bounded(&sm.mbar, phase, TILE_WAIT_NS);
            if (__syncthreads_or(!okw)) {                  // the whole block leaves together
                mbar_wait_bounded(&sm.mbar, phase, TILE_WAIT_NS);
                ok = false;
                break;
            }
            phase ^= 1u;
            tile_site(sm, Wm, p, x0, y0, 1.0f, true, [&](long long idx, float2 w) {
#pragma unroll
                for (int j = 0; j < PG_MAXK - 1; ++j) {
                    if (j < mm) {
                        const float2 u = __ldcg(a.W[j] + idx);
                        dots[2 * j] += u.x * w.x + u.y * w.y;
                        dots[2 * j + 1] += u.x * w.y - u.y * w.x;
                    }
                }
            });
        }
        pg_partials<2 * (PG_MAXK - 1)>(dots, 2 * m, a.partials, 1);
        if (!pcg_sync(a.bar, deadline, ok)) return;
        if (m > 0) pg_totals(a.partials, 1, 2 * m, sh.tot);
        if (threadIdx.x < m) {
            const int j = threadIdx.x;
            const double nn = sh.nrm[j];
            const double cr = nn > 0 ? sh.tot[1 + 2 * j] / nn : 0.0, ci = nn > 0 ? sh.tot[2 + 2 * j] / nn : 0.0;
            sh.C[m][j][0] = cr;
            sh.C[m][j][1] = ci;
            sh.coef[j] = make_float2((float)cr, (float)ci);
        }
        __syncthreads();
        // ---- phase C: w_m = w - sum_j c_j w_j; |w_m|^2, <w_m, r_m> ----
        float vc[3] = {0.f, 0.f, 0.f};
        {
            const long long stride = (long long)gridDim.x * blockDim.x;
            for (long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x; i0 < n; i0 += 4 * stride) {
                float2 w[4], r[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const long long i = i0 + u * stride;
                    if (i < n) { w[u] = __ldcg(Wm + i); r[u] = __ldcg(Rk + i); }
                }
                for (int j = 0; j < m; ++j) {
                    const float2 c = sh.coef[j];
                    float2 q[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const long long i = i0 + u * stride;
                        if (i < n) q[u] = __ldcg(a.W[j] + i);
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        w[u].x -= c.x * q[u].x - c.y * q[u].y;
                        w[u].y -= c.x * q[u].y + c.y * q[u].x;
                    }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const long long i = i0 + u * stride;
                    if (i < n) {
                        if (m > 0) Wm[i] = w[u];
                        vc[0] += w[u].x * w[u].x + w[u].y * w[u].y;
                        vc[1] += w[u].x * r[u].x + w[u].y * r[u].y;
                        vc[2] += w[u].x * r[u].y - w[u].y * r[u].x;
                    }
                }
            }
        }
        pg_partials<3>(vc, 3, a.partials, 1 + 2 * PG_MAXK);
        if (!pcg_sync(a.bar, deadline, ok)) return;
        pg_totals(a.partials, 1 + 2 * PG_MAXK, 3, sh.tot);
        {
            const double ww = sh.tot[1 + 2 * PG_MAXK];
            const double ar = ww > 0 ? sh.tot[2 + 2 * PG_MAXK] / ww : 0.0;
            const double ai = ww > 0 ? sh.tot[3 + 2 * PG_MAXK] / ww : 0.0;
            if (threadIdx.x == 0) {
                sh.nrm[m] = ww;
                sh.A[m][0] = ar;
                sh.A[m][1] = ai;
            }
            prevA = make_float2((float)ar, (float)ai);
        }
        __syncthreads();
        prevR = Rk;
        prevW = Wm;
        ++m;
        ++it;
    }
    // final update with the steps of the current cycle
    pg_back_substitute(sh, m);
    pg_combine(a, sh, base, m, n);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *a.out_iters += it;
        *a.out_rr2 = bn2 > 0 ? rr2 / bn2 : 0.0;
    }
}

// resident blocks per SM of the persistent coarse GCR, set up once per (device, block storage)
// under a mutex (the kernel's shared-memory limit is a per-device attribute)
template <class BT>
static dwf_status pgcr_blocks_per_sm(int* out) {
    static std::mutex mu;
    static int per_sm[64] = {0};
    int dev = 0;
    DWF_CHECK_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) { set_error("device ordinal %d out of range", dev); return DWF_ERR_UNSUPPORTED; }
    std::lock_guard<std::mutex> lock(mu);
    if (per_sm[dev] == 0) {
        const size_t smem = sizeof(TileSmemT<BT>);
        int per = 0;
        DWF_CHECK_CUDA(cudaFuncSetAttribute(k_coarse_gcr_persistent<BT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)smem));
        DWF_CHECK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_coarse_gcr_persistent<BT>, TILE_THREADS,
                                                                     smem));
        if (per < 1) { set_error("persistent coarse GCR cannot be resident"); return DWF_ERR_UNSUPPORTED; }
        per_sm[dev] = per < PGCR_BLOCKS_PER_SM ? per : PGCR_BLOCKS_PER_SM;
    }
    *out = per_sm[dev];
    return DWF_OK;
}

template <class BT>
static dwf_status launch_pgcr(PgcrArgs& a, int nsm, cudaStream_t st) {
    const size_t smem = sizeof(TileSmemT<BT>);
    int per = 0;
    DWF_TRY(pgcr_blocks_per_sm<BT>(&per));
    const int ntiles = ((a.cp.Lc[0] + TILE_X - 1) / TILE_X) * ((a.cp.Lc[1] + TILE_Y - 1) / TILE_Y);
    int grid = nsm * per;
    if (grid > ntiles) grid = ntiles;
    if (grid < 1) grid = 1;
    void* args[] = {&a};
    DWF_CHECK_CUDA(cudaLaunchCooperativeKernel((const void*)k_coarse_gcr_persistent<BT>, dim3(grid), dim3(TILE_THREADS),
                                               args, smem, st));
    return DWF_OK;
}

bool coarse_gcr_persistent_ok(const dwf_mg* h) {
    return h->mg.nd == 2 && h->mg.ncd == 16 && h->mg.Ls_c <= 4 && h->prm.coarse_restart <= PG_MAXK &&
           h->prm.coarse_restart >= 1;
}

dwf_status coarse_gcr_persistent(const dwf_mg* h, const float2* rc, float2* ec, float2* const* S, float2* const* W,
                                 float2* t, double* partials, void* bar, int* out_iters, double* out_rr2,
                                 cudaStream_t st) {
    if (!coarse_gcr_persistent_ok(h)) {
        set_error("persistent coarse GCR supports 2-d, 16 coarse dof, Ls_c <= 4 and coarse_restart <= %d", PG_MAXK);
        return DWF_ERR_UNSUPPORTED;
    }
    int dev = 0, nsm = 0;
    DWF_CHECK_CUDA(cudaGetDevice(&dev));
    DWF_CHECK_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    PgcrArgs a;
    a.cp = coarse_params(h, h->mf);
    a.rc = rc;
    a.e = ec;
    const int KC = h->prm.coarse_restart;
    for (int k = 0; k <= PG_MAXK; ++k) a.S[k] = k <= KC ? S[k] : nullptr;
    for (int k = 0; k < PG_MAXK; ++k) a.W[k] = k < KC ? W[k] : nullptr;
    a.t = t;
    a.partials = partials;
    a.bar = (PcgBarrier*)bar;
    a.out_iters = out_iters;
    a.out_rr2 = out_rr2;
    a.tol2 = h->prm.coarse_tol * h->prm.coarse_tol;
    a.maxiter = h->prm.coarse_maxiter;
    a.KC = KC;
    a.timeout_ns = 5000000000ULL;   // 5 s per solve
    DWF_CHECK_CUDA(cudaMemsetAsync(bar, 0, 2 * sizeof(unsigned), st));   // count, gen; the error flag persists
    if (h->ytile_half) {
        a.Y = h->Ytile;
        return launch_pgcr<__half2>(a, nsm, st);
    }
    a.Y = h->Y32;
    return launch_pgcr<float2>(a, nsm, st);
}

}  // namespace dwf
