// Fine-level Shamir domain-wall operator D_DW(m) (Eq. DWoperator, Sec. 2) and
// its Pauli-Villars / dagger variants, 2-d U(1) and 4-d SU(3).
//
// One thread owns one d-dim site and walks a chunk of s slices with a sliding
// window: psi_{s+1}(x) is loaded once and reused for slice s+1, so every
// spinor is read from HBM once per apply; the Wilson neighbours psi_s(x +- mu)
// of the same slice are shared between threads through L1/L2.  The links of
// the site are loaded once per s-chunk and reused on every slice (they do not
// depend on s).  The s-hops P_+ psi_{s-1} and P_- psi_{s+1} are a component
// select in the chiral basis (gamma_5 diagonal), fused into the same pass.
#include <algorithm>

#include "common.cuh"
#include "fine_kernels.cuh"

namespace dwf {

// ----------------------------------------------------------------------------
// 2-d U(1): spinor = 2 complex components (chirality +, -)
// ----------------------------------------------------------------------------
template <class R> struct Sp2 { typename cplx<R>::T c0, c1; };

__device__ __forceinline__ Sp2<float> ld_sp(const Sp2<float>* p, long long i) {
    float4 v = __ldg(reinterpret_cast<const float4*>(p) + i);
    Sp2<float> s; s.c0 = make_float2(v.x, v.y); s.c1 = make_float2(v.z, v.w); return s;
}
__device__ __forceinline__ Sp2<double> ld_sp(const Sp2<double>* p, long long i) {
    const double2* q = reinterpret_cast<const double2*>(p) + 2 * i;
    Sp2<double> s; s.c0 = __ldg(q); s.c1 = __ldg(q + 1); return s;
}
__device__ __forceinline__ void st_sp(Sp2<float>* p, long long i, const Sp2<float>& s) {
    reinterpret_cast<float4*>(p)[i] = make_float4(s.c0.x, s.c0.y, s.c1.x, s.c1.y);
}
__device__ __forceinline__ void st_sp(Sp2<double>* p, long long i, const Sp2<double>& s) {
    double2* q = reinterpret_cast<double2*>(p) + 2 * i;
    q[0] = s.c0; q[1] = s.c1;
}
// one chirality component of a spinor: comp 0 = P_+, comp 1 = P_-
template <class R>
__device__ __forceinline__ typename cplx<R>::T ld_comp(const Sp2<R>* p, long long i, int comp) {
    const typename cplx<R>::T* q = reinterpret_cast<const typename cplx<R>::T*>(p) + 2 * i + comp;
    return __ldg(q);
}

// Wilson hopping term -1/2 sum_mu [ (1 -+ gamma_mu) U psi(x+mu) + (1 +- gamma_mu) U^dag psi(x-mu) ]
// (upper signs: D_W; lower: D_W^dag = gamma_5 D_W gamma_5), for links that come with the -1/2 in
// them (exact).
template <class R, bool DAG>
__device__ __forceinline__ Sp2<R> hop2d(const Sp2<R>& xf, const Sp2<R>& xb, const Sp2<R>& yf, const Sp2<R>& yb,
                                        typename cplx<R>::T u0f, typename cplx<R>::T u0b,
                                        typename cplx<R>::T u1f, typename cplx<R>::T u1b) {
    using C = typename cplx<R>::T;
    C s0, s1;
    if (!DAG) {
        C t0f = cmul(u0f, xf.c0 - xf.c1);               // (1 - g1): (h, -h)
        C t0b = cmulc(u0b, xb.c0 + xb.c1);              // (1 + g1): (h,  h)
        C t1f = cmul(u1f, yf.c0 + times_i(yf.c1));     // (1 - g2): (h, -i h)
        C t1b = cmulc(u1b, yb.c0 - times_i(yb.c1));     // (1 + g2): (h,  i h)
        s0 = t0f + t0b + t1f + t1b;
        s1 = (t0b - t0f) + times_i(t1b - t1f);
    } else {
        C t0f = cmul(u0f, xf.c0 + xf.c1);               // (1 + g1): (h,  h)
        C t0b = cmulc(u0b, xb.c0 - xb.c1);              // (1 - g1): (h, -h)
        C t1f = cmul(u1f, yf.c0 - times_i(yf.c1));      // (1 + g2): (h,  i h)
        C t1b = cmulc(u1b, yb.c0 + times_i(yb.c1));     // (1 - g2): (h, -i h)
        s0 = t0f + t0b + t1f + t1b;
        s1 = (t0f - t0b) + times_i(t1f - t1b);
    }
    Sp2<R> o;
    o.c0 = s0;
    o.c1 = s1;
    return o;
}

// The same in FP64.  With t_f, t_b the transported half spinors of a direction, the two components
// take p = t_f + t_b and t_b - t_f (times 1 or i): p grows in t_f by fused multiply-adds, and the
// difference is p - 2 t_f.  The FP64 kernel is bound by FP64 issue (ncu: 86% of the pipe), and this
// takes 40 instructions per site and slice with the diagonal and the s-hops, where separate
// products, sums and scaling take 48: D_PV^dag D_DW at 250 x 333 x 13 180 us against 219 (with longer
// walks too), at the same error (9.6e-17 of one application at 64 x 48 x 12).  For that the sums stay
// trees and the largest term, the diagonal one, comes last, after the s-hop (before it: 9.8e-17).
// The adjoint's c1 comes with the opposite sign, which rides on the sum with the s-hop.
template <bool DAG>
__device__ __forceinline__ Sp2<double> hop2d_fused(const Sp2<double>& xf, const Sp2<double>& xb, const Sp2<double>& yf,
                                                   const Sp2<double>& yb, double2 u0f, double2 u0b, double2 u1f,
                                                   double2 u1b) {
    using C = double2;
    // (1 - g1): (h, -h), (1 + g1): (h, h); (1 - g2): (h, -i h), (1 + g2): (h, i h)
    const C t0 = cmul(u0f, DAG ? xf.c0 + xf.c1 : xf.c0 - xf.c1);
    const C t1 = cmul(u1f, DAG ? yf.c0 - times_i(yf.c1) : yf.c0 + times_i(yf.c1));
    const C p0 = cmacc(t0, u0b, DAG ? xb.c0 - xb.c1 : xb.c0 + xb.c1);
    const C p1 = cmacc(t1, u1b, DAG ? yb.c0 + times_i(yb.c1) : yb.c0 - times_i(yb.c1));
    const C m0 = mk<C>(fma(-2.0, t0.x, p0.x), fma(-2.0, t0.y, p0.y));   // t_b - t_f
    const C m1 = mk<C>(fma(-2.0, t1.x, p1.x), fma(-2.0, t1.y, p1.y));
    Sp2<double> o;
    o.c0 = p0 + p1;
    o.c1 = m0 + times_i(m1);
    return o;
}

// Any component infinite or NaN (integer instructions: the FP64 pipe is what the kernel is bound by)
__device__ __forceinline__ bool not_finite(const Sp2<double>& s) {
    const int a = max(__double2hiint(s.c0.x) & 0x7fffffff, __double2hiint(s.c0.y) & 0x7fffffff);
    const int b = max(__double2hiint(s.c1.x) & 0x7fffffff, __double2hiint(s.c1.y) & 0x7fffffff);
    return max(a, b) >= 0x7ff00000;
}

// streaming (evict-first) store of an output spinor: the output is not read
// again by this kernel, so it should not displace input planes from L2
__device__ __forceinline__ void st_sp_cs(Sp2<float>* p, long long i, const Sp2<float>& s) {
    __stcs(reinterpret_cast<float4*>(p) + i, make_float4(s.c0.x, s.c0.y, s.c1.x, s.c1.y));
}
__device__ __forceinline__ void st_sp_cs(Sp2<double>* p, long long i, const Sp2<double>& s) {
    double2* q = reinterpret_cast<double2*>(p) + 2 * i;
    __stcs(q, s.c0);
    __stcs(q + 1, s.c1);
}

// One site, slices [s0, s1): the body shared by the single-lattice kernel and
// the batched (many right-hand sides, mixed lattices) kernel.  While slice s is computed, the load
// of psi_{s+2} at this site is in flight and psi_{s+4} on its way to L2.  Every stream has a
// pointer of its own that moves by a plane: addresses formed from slice and site kept the FP32
// kernel at 72% issue.  Bound by HBM: 1024^2 x 16, FP16 links, 96.6 us (5.6 TB/s) against 98.3 with
// such addresses; without the L2 prefetch 112, one plane nearer or two farther 102 and 101.  UNROLL 2
// saves the window's moves; the batched kernel is the faster without (151 against 158 us).
template <class LT, class R, bool DAG, int UNROLL>
__device__ __forceinline__ void dwf2d_site(const typename LT::store* __restrict__ U, const Sp2<R>* __restrict__ psi,
                                           Sp2<R>* __restrict__ out, const Fine2dParams& p, long long site, int s0,
                                           int s1) {
    using C = typename cplx<R>::T;
    const long long V = p.V;
    const int Lx = p.L0;
    const int x = V <= 0xffffffffLL ? (int)((unsigned)site % (unsigned)Lx) : (int)(site % Lx);
    const int Ls = p.Ls;

    // neighbour sites with periodic wrap, relative to this one
    const bool xe = x == Lx - 1, xs = x == 0, ye = site + Lx >= V, ys = site - Lx < 0;
    const long long dxf = xe ? 1 - Lx : 1, dxb = xs ? Lx - 1 : -1;
    const long long dyf = ye ? Lx - V : Lx, dyb = ys ? V - Lx : -Lx;

    // links, loaded once for all s, with the hops' -1/2 (antiperiodic boundaries flip the hop sign)
    const C u0f = scale(load_link(U, site), p.anti0 && xe ? R(0.5) : R(-0.5));
    const C u1f = scale(load_link(U, V + site), p.anti1 && ye ? R(0.5) : R(-0.5));
    const C u0b = scale(load_link(U, site + dxb), p.anti0 && xs ? R(0.5) : R(-0.5));
    const C u1b = scale(load_link(U, V + site + dyb), p.anti1 && ys ? R(0.5) : R(-0.5));
    const R diag = param_cast<R>(p.diag, p.diag_f);
    const R mf = param_cast<R>(p.mf, p.mf_f);
    // component fed from below (s-1) and from above (s+1):
    //   D:     out.c0 += psi_{s-1}.c0, out.c1 += psi_{s+1}.c1
    //   D^dag: out.c0 += psi_{s+1}.c0, out.c1 += psi_{s-1}.c1
    const int cb = DAG ? 1 : 0;   // component taken from s-1
    const int ca = DAG ? 0 : 1;   // component taken from s+1
    const int slast = s1 < Ls ? s1 : Ls - 1;   // last plane the window needs
    const bool lead = (threadIdx.x & (128 / sizeof(Sp2<R>) - 1)) == 0;   // one lane per 128-byte line

    const Sp2<R>* pc = psi + ((long long)s0 * V + site);
    Sp2<R> cur = ld_sp(pc, 0), next = cur;
    if (s0 + 1 <= slast) next = ld_sp(pc + V, 0);
    C below = (s0 > 0) ? ld_comp(pc - V, 0, cb) : scale(ld_comp(psi, (long long)(Ls - 1) * V + site, cb), -mf);
    const C wall0 = (s0 == 0) ? (ca == 0 ? cur.c0 : cur.c1) : C();
    const Sp2<R>*pxf = pc + dxf, *pxb = pc + dxb, *pyf = pc + dyf, *pyb = pc + dyb, *pn = pc + 2 * V;
    Sp2<R>* po = out + ((long long)s0 * V + site);

#pragma unroll UNROLL
    for (int s = s0; s < s1; ++s) {
        const Sp2<R> nb_xf = ld_sp(pxf, 0), nb_xb = ld_sp(pxb, 0), nb_yf = ld_sp(pyf, 0), nb_yb = ld_sp(pyb, 0);
        C above;
        if (s + 1 < Ls) {
            above = (ca == 0) ? next.c0 : next.c1;
        } else {
            const C w = (s0 == 0) ? wall0 : ld_comp(psi, site, ca);
            above = scale(w, -mf);
        }
        Sp2<R> over = next;
        if (s + 2 <= slast) over = ld_sp(pn, 0);
        if (lead && s + 4 <= slast) asm volatile("prefetch.global.L2 [%0];" ::"l"(pn + 2 * V));
        Sp2<R> o;
        if constexpr (sizeof(R) == 8) {
            o = hop2d_fused<DAG>(nb_xf, nb_xb, nb_yf, nb_yb, u0f, u0b, u1f, u1b);
            // p - 2 t_f turns an infinite t_f into NaN: take the differences themselves (the empty
            // statement keeps this a branch: D_PV^dag D_DW at 250 x 333 x 13 180 us, as without the check; with
            // both forms computed and one selected 266)
            if (__builtin_expect(not_finite(o), 0)) {
                asm volatile("" ::: "memory");
                o = hop2d<double, DAG>(ld_sp(pxf, 0), ld_sp(pxb, 0), ld_sp(pyf, 0), ld_sp(pyb, 0), u0f, u0b, u1f, u1b);
                if (DAG) o.c1 = scale(o.c1, -1.0);
            }
            const C in0 = cb == 0 ? below : above, in1 = cb == 0 ? above : below;
            o.c0.x = fma(diag, cur.c0.x, o.c0.x + in0.x); o.c0.y = fma(diag, cur.c0.y, o.c0.y + in0.y);
            o.c1.x = fma(diag, cur.c1.x, DAG ? in1.x - o.c1.x : o.c1.x + in1.x);
            o.c1.y = fma(diag, cur.c1.y, DAG ? in1.y - o.c1.y : o.c1.y + in1.y);
        } else {
            o = hop2d<R, DAG>(nb_xf, nb_xb, nb_yf, nb_yb, u0f, u0b, u1f, u1b);
            o.c0 = o.c0 + scale(cur.c0, diag);
            o.c1 = o.c1 + scale(cur.c1, diag);
            if (cb == 0) { o.c0 = o.c0 + below; o.c1 = o.c1 + above; }
            else         { o.c1 = o.c1 + below; o.c0 = o.c0 + above; }
        }
        st_sp_cs(po, 0, o);
        below = (cb == 0) ? cur.c0 : cur.c1;
        cur = next;
        next = over;
        pxf += V; pxb += V; pyf += V; pyb += V; pn += V; po += V;
    }
}

constexpr int BLOCK_MAX = 128;             // threads per block of k_dwf2d and k_dwf2d_multi (block_threads)
template <class LT, class R, bool DAG>
__global__ void __launch_bounds__(BLOCK_MAX, sizeof(R) == 8 ? 4 : 8)
k_dwf2d(const typename LT::store* __restrict__ U, const Sp2<R>* __restrict__ psi, Sp2<R>* __restrict__ out,
        Fine2dParams p) {
    const long long site = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (site >= p.V) return;
    const int s0 = p.s_base + blockIdx.y * p.s_chunk;
    if (s0 >= p.s_end) return;
    dwf2d_site<LT, R, DAG, 2>(U, psi, out, p, site, s0, min(s0 + p.s_chunk, p.s_end));
}

// nrhs right-hand sides on the same lattice and links, stored back to back
// (stride V * Ls spinors): grid.z walks the right-hand sides; skip[r] != 0
// (device flags, may be null) leaves right-hand side r untouched.
template <class LT, class R, bool DAG>
__global__ void __launch_bounds__(BLOCK_MAX, sizeof(R) == 8 ? 4 : 8)
k_dwf2d_multi(const typename LT::store* __restrict__ U, const Sp2<R>* __restrict__ psi, Sp2<R>* __restrict__ out,
              Fine2dParams p, const int* __restrict__ skip) {
    const int r = blockIdx.z;
    if (skip && skip[r]) return;
    const long long site = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (site >= p.V) return;
    const int s0 = blockIdx.y * p.s_chunk;
    if (s0 >= p.Ls) return;
    const long long off = (long long)r * p.V * p.Ls;
    dwf2d_site<LT, R, DAG, 2>(U, psi + off, out + off, p, site, s0, min(s0 + p.s_chunk, p.Ls));
}

// Threads per block.  Fewer threads than 256 for each of the 152 SMs are spread over more SMs in blocks
// of 64: in FP64 one block of 256 keeps its SM's FP64 unit busy for 3 us per slice while others
// idle (32^2 x 8 in FP64: 7.9 -> 5.4 us a call).  Otherwise blocks of 128, which end more evenly
// than ones of 256 (512 x 256 x 16: 17.0 against 18.6 us).
static int block_threads(long long threads) { return threads < 152LL * 256 ? 64 : BLOCK_MAX; }

template <class LT, class R>
static void launch2d_multi(const void* U, const void* psi, void* out, const Fine2dParams& p, int nrhs,
                           const int* skip, bool dagger, cudaStream_t st) {
    const unsigned chunks = (unsigned)((p.Ls + p.s_chunk - 1) / p.s_chunk);
    const int threads = block_threads(p.V * chunks * nrhs);
    dim3 grid((unsigned)((p.V + threads - 1) / threads), chunks, (unsigned)nrhs);
    auto Ut = reinterpret_cast<const typename LT::store*>(U);
    auto pi = reinterpret_cast<const Sp2<R>*>(psi);
    auto po = reinterpret_cast<Sp2<R>*>(out);
    if (dagger) k_dwf2d_multi<LT, R, true><<<grid, threads, 0, st>>>(Ut, pi, po, p, skip);
    else        k_dwf2d_multi<LT, R, false><<<grid, threads, 0, st>>>(Ut, pi, po, p, skip);
}

// Many right-hand sides on possibly different lattices in one launch: virtual
// block vb of the concatenated block ranges maps to (right-hand side r, block
// within r) through the descriptors' block offsets (binary search).
template <class LT, class R, bool DAG>
__global__ void __launch_bounds__(256, sizeof(R) == 8 ? 2 : 4)
k_dwf2d_batched(const __grid_constant__ BatchArgs2d a) {
    for (long long vb = blockIdx.x; vb < a.total_blocks; vb += gridDim.x) {
        int lo = 0, hi = a.nrhs - 1;                              // last r with block0 <= vb
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (a.d[mid].block0 <= vb) lo = mid; else hi = mid - 1;
        }
        const BatchDesc2d& q = a.d[lo];
        const long long site = (vb - q.block0) * blockDim.x + threadIdx.x;
        if (site < q.p.V)
            dwf2d_site<LT, R, DAG, 1>(reinterpret_cast<const typename LT::store*>(q.U),
                                      reinterpret_cast<const Sp2<R>*>(q.psi), reinterpret_cast<Sp2<R>*>(q.out), q.p,
                                      site, 0, q.p.Ls);
    }
}

template <class LT, class R>
static void launch2d_batched(const BatchArgs2d& a, int grid, bool dagger, cudaStream_t st) {
    if (dagger) k_dwf2d_batched<LT, R, true><<<grid, 256, 0, st>>>(a);
    else        k_dwf2d_batched<LT, R, false><<<grid, 256, 0, st>>>(a);
}

dwf_status fine_apply_2d_batched(const BatchArgs2d& a, bool dagger, int prec, cudaStream_t st) {
    // one block per 256-site range of every right-hand side, all in one launch:
    // like the single-lattice apply, many short blocks hide the s-walk latency
    // better than a few persistent ones (measured: 608 persistent blocks reached
    // 24% of HBM on the 64-source batch)
    long long g = a.total_blocks < (1LL << 31) - 1 ? a.total_blocks : (1LL << 31) - 1;
    const int grid = (int)(g < 1 ? 1 : g);
    switch (prec) {
        case DWF_F64:       launch2d_batched<LinkF64, double>(a, grid, dagger, st); break;
        case DWF_F32:       launch2d_batched<LinkF32, float>(a, grid, dagger, st); break;
        case DWF_F32_L16:   launch2d_batched<LinkH16, float>(a, grid, dagger, st); break;
        case DWF_F32_LBF16: launch2d_batched<LinkBF16, float>(a, grid, dagger, st); break;
        default: set_error("bad precision %d", prec); return DWF_ERR_ARG;
    }
    DWF_CHECK_LAUNCH();
    return DWF_OK;
}

dwf_status fine_apply_2d_range(const Geom& g, const void* U, const void* psi, void* out, double M5, double mf,
                               bool dagger, int prec, int s_lo, int s_hi, cudaStream_t st, int s_chunk);

template <class LT, class R>
static void launch2d(const void* U, const void* psi, void* out, const Fine2dParams& p, bool dagger,
                     cudaStream_t st) {
    const unsigned chunks = (unsigned)((p.s_end - p.s_base + p.s_chunk - 1) / p.s_chunk);
    const int threads = block_threads(p.V * chunks);
    dim3 grid((unsigned)((p.V + threads - 1) / threads), chunks);
    auto Ut = reinterpret_cast<const typename LT::store*>(U);
    auto pi = reinterpret_cast<const Sp2<R>*>(psi);
    auto po = reinterpret_cast<Sp2<R>*>(out);
    if (dagger) k_dwf2d<LT, R, true><<<grid, threads, 0, st>>>(Ut, pi, po, p);
    else        k_dwf2d<LT, R, false><<<grid, threads, 0, st>>>(Ut, pi, po, p);
}

// Slices per thread.  A longer walk re-reads fewer boundary planes and loads the links less often, a
// shorter one gives the SMs more threads: the walk is split until there are 512 threads per SM
// in FP32 (256^2 x 16, FP16 links: 8.6 us with 8 slices, 11.4 with 2; 400^2 x 16: 18.5 with 16, 19.1
// with 4) and 2048 in FP64, which is bound by issue and wants its SMs evenly loaded (D_PV^dag
// D_DW at 250 x 333 x 13: 181 us with 4 slices, 193 with 2, 210 with 1).  A walk of more than 16
// slices is as long as the whole call where its blocks come in one round or in a few and a bit more
// (400^2 x 32: 1250 blocks of which 1216 are resident): it is kept where 768 threads per SM come in one
// round (256^2 x 64: 26.7 us with 32 slices, 27.6 with 16) or from four rounds on (1024^2 x 32: 181
// with 32, 189 with 16), else 16 slices are the most (400^2 x 32: 37.1 against 43.0, 280^2 x 128: 60.7
// against 70.0, 700^2 x 32: 96.6 against 98.5).
constexpr int WALK_MAX = 16;
static int choose_s_chunk(long long V, int Ls, bool f64) {
    auto slices = [&](long long threads) {
        const long long n = std::min({std::max((threads + V - 1) / V, 1LL), (long long)Ls, 65535LL});   // grid.y
        return (int)((Ls + n - 1) / n);
    };
    const int chunk = slices(152LL * (f64 ? 2048 : 512));
    if (f64 || chunk <= WALK_MAX) return chunk;
    const int walk = slices(152LL * 768);
    const long long blocks = (V + BLOCK_MAX - 1) / BLOCK_MAX * ((Ls + walk - 1) / walk), resident = 152LL * 8;
    if (blocks <= resident || blocks >= 4 * resident) return walk;
    return std::max(WALK_MAX, (Ls + 65534) / 65535);
}

dwf_status fine_apply_2d(const Geom& g, const void* U, const void* psi, void* out, double M5, double mf,
                         bool dagger, int prec, int s_chunk, cudaStream_t st) {
    return fine_apply_2d_range(g, U, psi, out, M5, mf, dagger, prec, 0, g.Ls, st, s_chunk);
}

dwf_status fine_apply_2d_range(const Geom& g, const void* U, const void* psi, void* out, double M5, double mf,
                               bool dagger, int prec, int s_lo, int s_hi, cudaStream_t st) {
    return fine_apply_2d_range(g, U, psi, out, M5, mf, dagger, prec, s_lo, s_hi, st, 0);
}

dwf_status fine_apply_2d_range(const Geom& g, const void* U, const void* psi, void* out, double M5, double mf,
                               bool dagger, int prec, int s_lo, int s_hi, cudaStream_t st, int s_chunk) {
    if (s_lo < 0 || s_hi > g.Ls || s_lo >= s_hi) { set_error("bad slice range [%d, %d)", s_lo, s_hi); return DWF_ERR_ARG; }
    Fine2dParams p;
    p.s_base = s_lo;
    p.s_end = s_hi;
    p.V = g.V;
    p.L0 = g.L[0];
    p.L1 = g.L[1];
    p.Ls = g.Ls;
    p.anti0 = g.anti[0];
    p.anti1 = g.anti[1];
    p.diag = (double)g.nd - M5 + 1.0;
    p.mf = mf;
    p.diag_f = (float)p.diag;
    p.mf_f = (float)p.mf;
    p.s_chunk = s_chunk > 0 ? s_chunk : choose_s_chunk(g.V, s_hi - s_lo, prec == DWF_F64);
    switch (prec) {
        case DWF_F64:      launch2d<LinkF64, double>(U, psi, out, p, dagger, st); break;
        case DWF_F32:      launch2d<LinkF32, float>(U, psi, out, p, dagger, st); break;
        case DWF_F32_L16:  launch2d<LinkH16, float>(U, psi, out, p, dagger, st); break;
        case DWF_F32_LBF16: launch2d<LinkBF16, float>(U, psi, out, p, dagger, st); break;
        default: set_error("bad precision %d", prec); return DWF_ERR_ARG;
    }
    DWF_CHECK_LAUNCH();
    return DWF_OK;
}

dwf_status fine_apply_2d_multi(const Geom& g, const void* U, const void* psi, void* out, double M5, double mf,
                               bool dagger, int prec, int nrhs, const int* skip, cudaStream_t st) {
    if (g.nd != 2) { set_error("multi-right-hand-side fine apply: 2-d lattices only"); return DWF_ERR_UNSUPPORTED; }
    if (nrhs < 1 || nrhs > 65535) { set_error("nrhs must be in [1, 65535]"); return DWF_ERR_ARG; }
    Fine2dParams p;
    p.V = g.V;
    p.L0 = g.L[0];
    p.L1 = g.L[1];
    p.Ls = g.Ls;
    p.anti0 = g.anti[0];
    p.anti1 = g.anti[1];
    p.diag = (double)g.nd - M5 + 1.0;
    p.mf = mf;
    p.diag_f = (float)p.diag;
    p.mf_f = (float)p.mf;
    p.s_chunk = choose_s_chunk(g.V * nrhs, g.Ls, prec == DWF_F64);
    p.s_base = 0;
    p.s_end = g.Ls;
    switch (prec) {
        case DWF_F64:       launch2d_multi<LinkF64, double>(U, psi, out, p, nrhs, skip, dagger, st); break;
        case DWF_F32:       launch2d_multi<LinkF32, float>(U, psi, out, p, nrhs, skip, dagger, st); break;
        case DWF_F32_L16:   launch2d_multi<LinkH16, float>(U, psi, out, p, nrhs, skip, dagger, st); break;
        case DWF_F32_LBF16: launch2d_multi<LinkBF16, float>(U, psi, out, p, nrhs, skip, dagger, st); break;
        default: set_error("bad precision %d", prec); return DWF_ERR_ARG;
    }
    DWF_CHECK_LAUNCH();
    return DWF_OK;
}

}  // namespace dwf
