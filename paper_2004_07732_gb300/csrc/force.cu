// Differentiation of x = D_DW^-1 b with respect to the links: U(1) link
// angles (2-d), and for any group the complex link gradient and (SU(3)) the
// force projected onto the algebra.
//
// For a real loss L(x) with upstream gradient g = dL/dRe x + i dL/dIm x, the
// adjoint solution lambda = D_DW^-dag g gives dL/db = lambda and
//   dL/dtheta_mu(y) = -Re( lambda^dag (dD_DW / dtheta_mu(y)) x ).
// Only the Wilson hops of D_W (Sec. 2) depend on U_mu(y) = exp(i theta_mu(y)),
// on every s slice: the forward hop -1/2 (1 - gamma_mu) U_mu(y) (row y, column
// y + mu) differentiates to -1/2 (1 - gamma_mu) i U_mu(y), the backward hop
// -1/2 (1 + gamma_mu) U_mu(y)^* (row y + mu, column y) to
// -1/2 (1 + gamma_mu) (-i) U_mu(y)^*.
//
// The adjoint solve uses Gamma_5 = gamma_5 R (Sec. 2.1): D^dag = Gamma_5 D Gamma_5,
// so D^-dag g = Gamma_5 D^-1 Gamma_5 g and any forward solver serves.
#include "common.cuh"
#include "fine_kernels.cuh"

namespace dwf {

__global__ void k_links_from_angles(const double* __restrict__ th, double2* __restrict__ U, long long n) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        double sn, cs;
        sincos(th[i], &sn, &cs);
        U[i] = make_double2(cs, sn);
    }
}

// out_s = gamma_5 in_{Ls-1-s}; chirality - components change sign.
template <class C>
__global__ void k_gamma5_reflect(const C* __restrict__ in, C* __restrict__ out, long long V, int Ls, int dof,
                                 int half) {
    const long long n = V * Ls * dof;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        const int d = (int)(t % dof);
        const long long rest = t / dof;
        const long long x = rest % V;
        const int s = (int)(rest / V);
        C v = in[((long long)(Ls - 1 - s) * V + x) * dof + d];
        if (d >= half) { v.x = -v.x; v.y = -v.y; }
        out[t] = v;
    }
}

// ---------------------------------------------------------------------------
// Link derivatives.  Both kernels run at the FP64 rate of the chip (two FMAs per
// clock and SM), far above their memory time, so they are written for the fewest
// FP64 instructions: 1 -+ gamma_mu has half the rank of the spin space, and
//   sum_a lam_a ((1 -+ gamma_mu) x)_a^dag = sum_{a < rank} h(lam)_a h(x)_a^dag
// with the same half spinors h on both sides, since the lower spins of
// (1 -+ gamma_mu) x are unitary images of the upper ones.
//
// A block is (LINK_THREADS / SP) links x SP groups of slices: group g sums the slices g,
// g + SP, ..; the groups' sums meet in shared memory in group order.  SP
// (link_slice_groups) splits a small lattice until its threads fill the SMs,
// and a large one no further than leaves several blocks per SM to even out
// the last wave.
// ---------------------------------------------------------------------------
constexpr int LINK_THREADS = 128;

// 152 SMs hold 16 warps each at the 128 registers of the SU(3) kernel: the slices are split until
// two such waves are there.  SU(3) force at 12^3 x 24 x 12 (2.1 waves unsplit) with 1, 2, 4, 8
// groups: 756, 767, 760, 884 us.
// U(1), with 36 warps per SM and as many adds per group as two slices take: two thirds of a wave (128^2 x 8 with 4
// and 8 groups: 12.8 and 16.0 us; 256^2 x 4 with 1 and 2: 20.5 and 22.7).
static int link_slice_groups(bool su3, long long threads, int Ls) {
    const long long target = 152LL * (su3 ? 1024 : 768);
    int sp = 1;
    while (sp < 8 && 2 * sp <= Ls && threads * sp < target) sp *= 2;
    return sp;
}

// v[k] of group 0 += v[k] of groups 1 .. SP - 1, in order; sh holds (SP - 1) * N * TX doubles
template <int N>
__device__ __forceinline__ void sum_slice_groups(double (&v)[N], double* sh) {
    const int TX = blockDim.x, tx = threadIdx.x, ty = threadIdx.y;
    if (blockDim.y == 1) return;
    if (ty > 0)
#pragma unroll
        for (int k = 0; k < N; ++k) sh[((ty - 1) * N + k) * TX + tx] = v[k];
    __syncthreads();
    if (ty == 0)
        for (int g = 0; g + 1 < (int)blockDim.y; ++g)
#pragma unroll
            for (int k = 0; k < N; ++k) v[k] += sh[(g * N + k) * TX + tx];
}

// 2-d U(1).  Per link, summed over s, with t1 = lam(y)^dag (1 - gamma_mu) x(y + mu) and
// t2 = lam(y + mu)^dag (1 + gamma_mu) x(y):  R = Re(t1 + t2), I = Im(t2 - t1).
//   gradient: Re(lam^dag dD x) = Re(conj(G) dU) for any change dU (the backward hop reads
//     conj(U)): G = -1/2 ph (R + i I);
//   FORCE: the derivative along theta (dU = i U dtheta): -1/2 ph (U.x I - U.y R).
// 16 FP64 instructions per (link, slice): each of the four products of R and of I has a sum of its
// own, since one chain of all of them rounds every product at the size of the whole sum (error 1.9e-16 at
// 300 x 400 x 12).  512^2 x 16: 252 us; 254 with the one chain, 295 with each slice's products summed first.
// grid.y = mu, as for SU(3): a thread with the sums of both needs 78 registers instead of 56, and the 1024 blocks of
// a 128^2 lattice then come in a round and a bit (128^2 x 8: 17 us against 12.8).
template <int MU>
__device__ __forceinline__ void link_sum_u1(const double2* __restrict__ lam, const double2* __restrict__ x, long long V,
                                            int Ls, long long site, long long nb, double (&v)[2]) {
    double re[4] = {0.0, 0.0, 0.0, 0.0}, im[4] = {0.0, 0.0, 0.0, 0.0};
    for (int s = threadIdx.y; s < Ls; s += blockDim.y) {
        const long long b = (long long)s * V;
        const double2 l0 = __ldg(lam + 2 * (b + site)), l1 = __ldg(lam + 2 * (b + site) + 1);
        const double2 x0 = __ldg(x + 2 * (b + site)), x1 = __ldg(x + 2 * (b + site) + 1);
        const double2 m0 = __ldg(lam + 2 * (b + nb)), m1 = __ldg(lam + 2 * (b + nb) + 1);
        const double2 y0 = __ldg(x + 2 * (b + nb)), y1 = __ldg(x + 2 * (b + nb) + 1);
        // h = c0 -+ (c1 or -i c1): gamma_1 pairs c0 with c1, gamma_2 with -i c1
        const double2 p = MU == 0 ? l0 - l1 : l0 + times_i(l1), q = MU == 0 ? y0 - y1 : y0 + times_i(y1);
        const double2 r = MU == 0 ? m0 + m1 : m0 - times_i(m1), t = MU == 0 ? x0 + x1 : x0 - times_i(x1);
        re[0] = fma(p.x, q.x, re[0]); re[1] = fma(p.y, q.y, re[1]);
        re[2] = fma(r.x, t.x, re[2]); re[3] = fma(r.y, t.y, re[3]);
        im[0] = fma(p.y, q.x, im[0]); im[1] = fma(-p.x, q.y, im[1]);
        im[2] = fma(r.x, t.y, im[2]); im[3] = fma(-r.y, t.x, im[3]);
    }
    v[0] = (re[0] + re[1]) + (re[2] + re[3]);
    v[1] = (im[0] + im[1]) + (im[2] + im[3]);
}

template <bool FORCE>
__global__ void __launch_bounds__(LINK_THREADS)
k_linkgrad_u1_2d(const double2* __restrict__ U, const double2* __restrict__ lam, const double2* __restrict__ x,
                 double* __restrict__ out, int L0, long long V, int Ls, int anti0, int anti1) {
    extern __shared__ double link_sh[];
    const long long site = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool in = site < V;
    const int mu = blockIdx.y;
    const bool cross = mu == 0 ? (int)(site % L0) == L0 - 1 : site + L0 >= V;
    const long long nb = mu == 0 ? (cross ? site - (L0 - 1) : site + 1) : (cross ? site + L0 - V : site + L0);
    double v[2] = {0.0, 0.0};                     // R, I
    if (in) {
        if (mu == 0) link_sum_u1<0>(lam, x, V, Ls, site, nb, v);
        else         link_sum_u1<1>(lam, x, V, Ls, site, nb, v);
    }
    sum_slice_groups<2>(v, link_sh);
    if (!in || threadIdx.y != 0) return;
    const double ph = (cross && (mu == 0 ? anti0 : anti1)) ? 0.5 : -0.5;
    const long long t = mu * V + site;
    if (FORCE) {
        const double2 u = __ldg(U + t);
        out[t] = ph * (u.x * v[1] - u.y * v[0]);
    } else {
        reinterpret_cast<double2*>(out)[t] = make_double2(ph * v[0], ph * v[1]);
    }
}

// the half spinor h of (1 + SGN gamma_MU) v in the chiral basis gamma_mu = [[0, A], [A^dag, 0]],
// A = -i sigma_1, -i sigma_2, -i sigma_3, 1: h = v_up + SGN A v_low
template <int MU, int SGN>
__device__ __forceinline__ void half_spinor(const double2* __restrict__ v, double2 (&h)[6]) {
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double2 up = __ldg(v + a * 3 + c);
            const double2 low = __ldg(v + (2 + (MU < 2 ? 1 - a : a)) * 3 + c);
            double2 w;                                         // A v_low
            if (MU == 0) w = make_double2(low.y, -low.x);      // -i
            if (MU == 1) w = a == 0 ? make_double2(-low.x, -low.y) : low;
            if (MU == 2) w = a == 0 ? make_double2(low.y, -low.x) : make_double2(-low.y, low.x);
            if (MU == 3) w = low;
            h[a * 3 + c] = SGN > 0 ? up + w : up - w;
        }
}

// G += sum_a a_a b_a^dag (colour outer products over the two half spins)
__device__ __forceinline__ void outer_half(const double2 (&a)[6], const double2 (&b)[6], double (&G)[18]) {
#pragma unroll
    for (int sp = 0; sp < 2; ++sp)
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const double2 u = a[sp * 3 + i], w = b[sp * 3 + j];
                double& re = G[2 * (i * 3 + j)];
                double& im = G[2 * (i * 3 + j) + 1];
                re = fma(u.x, w.x, re); re = fma(u.y, w.y, re);
                im = fma(u.y, w.x, im); im = fma(-u.x, w.y, im);
            }
}

// The thread's slices: 8 products per slice and real number of G.  Runs of LINK_RUN slices are
// summed by themselves before they are added to the total: one chain of multiply-adds over all slices, whose
// every product is rounded at the size of the whole sum, has an error of 3.4e-16 at Ls = 12, runs of
// four slices 2.2e-16 and of two 1.8e-16 (sums of four products and no half spinors: 2.6e-16).  A run costs 18 more
// FP64 instructions, but the first (SU(3) force at 12^3 x 24 x 12: one run 757 us, four slices 771, two about 795); the totals live in shared memory,
// since the registers hold one set of 18.
constexpr int LINK_RUN = 4;
template <int MU>
__device__ __forceinline__ void link_sum_su3(const double2* __restrict__ lam, const double2* __restrict__ x,
                                             long long V, int Ls, long long site, long long nb, double* total) {
    const int step = blockDim.y, run = LINK_RUN * step;
    for (int s0 = threadIdx.y; s0 < Ls; s0 += run) {
        double G[18];
#pragma unroll
        for (int e = 0; e < 18; ++e) G[e] = 0.0;
#pragma unroll 1
        for (int s = s0; s < min(Ls, s0 + run); s += step) {
            const long long b = (long long)s * V;
            double2 h[6], k[6];
            half_spinor<MU, -1>(lam + 12 * (b + site), h);
            half_spinor<MU, -1>(x + 12 * (b + nb), k);
            outer_half(h, k, G);
            half_spinor<MU, 1>(x + 12 * (b + site), h);
            half_spinor<MU, 1>(lam + 12 * (b + nb), k);
            outer_half(h, k, G);
        }
        if (s0 != (int)threadIdx.y) {                    // not the first run
#pragma unroll
            for (int e = 0; e < 18; ++e) G[e] += total[e * LINK_THREADS];
        }
#pragma unroll
        for (int e = 0; e < 18; ++e) total[e * LINK_THREADS] = G[e];
    }
}

// 4-d SU(3) link gradient G_mu(y) (3 x 3): Re(lam^dag dD x) = Re sum_ij conj(G_ij) dU_ij for any change
// dU of U_mu(y): G = -1/2 ph [ sum_a lam_a(y) y_a^dag + sum_a z_a lam_a(y + mu)^dag ], summed over s,
// with y = (1 - gamma_mu) x(y + mu), z = (1 + gamma_mu) x(y) (colour outer products over the spins a).
// FORCE: the su(3) projection F = Pi(i U G^dag) (traceless Hermitian part), for which
// Re(lam^dag dD x) = tr(H F) under U -> exp(i eps H) U.
// grid.y = mu, a compile-time constant of each branch, so that gamma_mu is a choice of
// components and signs: 192 FP64 instructions per (link, slice), 0.66 ms of the FP64 rate at
// 12^3 x 24 x 12 (the memory floor is 35 us); measured 0.77 ms.  With gamma_mu looked up at run
// time and all four spins multiplied out the kernel ran 3.20 ms.
template <bool FORCE>
__global__ void __launch_bounds__(LINK_THREADS, 4)
k_linkgrad_su3(const double2* __restrict__ U, const double2* __restrict__ lam, const double2* __restrict__ x,
               double2* __restrict__ out, int4 L, long long V, int Ls, int4 anti) {
    extern __shared__ double link_sh[];
    const long long site = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool in = site < V;
    const int mu = blockIdx.y;
    const int Lm = mu == 0 ? L.x : mu == 1 ? L.y : mu == 2 ? L.z : L.w;
    const long long stride = mu == 0 ? 1 : mu == 1 ? (long long)L.x : mu == 2 ? (long long)L.x * L.y
                                                                              : (long long)L.x * L.y * L.z;
    const int c = (int)((site / stride) % Lm);
    const bool cross = c == Lm - 1;
    const long long nb = cross ? site - (long long)(Lm - 1) * stride : site + stride;
    const int am = mu == 0 ? anti.x : mu == 1 ? anti.y : mu == 2 ? anti.z : anti.w;
    const double ph = (cross && am) ? 0.5 : -0.5;
    if (in) {
        double* total = link_sh + threadIdx.y * blockDim.x + threadIdx.x;
        switch (mu) {
            case 0: link_sum_su3<0>(lam, x, V, Ls, site, nb, total); break;
            case 1: link_sum_su3<1>(lam, x, V, Ls, site, nb, total); break;
            case 2: link_sum_su3<2>(lam, x, V, Ls, site, nb, total); break;
            default: link_sum_su3<3>(lam, x, V, Ls, site, nb, total); break;
        }
    }
    __syncthreads();
    if (!in || threadIdx.y != 0) return;
    // the groups' sums in order (every group has a slice: link_slice_groups)
    double G[18];
#pragma unroll
    for (int e = 0; e < 18; ++e) {
        double t = link_sh[e * LINK_THREADS + threadIdx.x];
        for (int g = 1; g < (int)blockDim.y; ++g) t += link_sh[e * LINK_THREADS + g * blockDim.x + threadIdx.x];
        G[e] = ph * t;
    }
    const long long t = mu * V + site;
    double2* o = out + 9 * t;
    if (!FORCE) {
#pragma unroll
        for (int e = 0; e < 9; ++e) o[e] = make_double2(G[2 * e], G[2 * e + 1]);
        return;
    }
    // A = i U G^dag; F = (A + A^dag) / 2 - tr / 3
    const double2* u = U + 9 * t;
    double2 A[9];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            double re = 0.0, im = 0.0;       // sum_k U_ik conj(G_jk)
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const double2 a = u[i * 3 + k];
                const double gx = G[2 * (j * 3 + k)], gy = G[2 * (j * 3 + k) + 1];
                re += a.x * gx + a.y * gy;
                im += a.y * gx - a.x * gy;
            }
            A[i * 3 + j] = make_double2(-im, re);    // times i
        }
    const double tr = (A[0].x + A[4].x + A[8].x) / 3.0;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const double2 a = A[i * 3 + j], b = A[j * 3 + i];
            double2 f = make_double2(0.5 * (a.x + b.x), 0.5 * (a.y - b.y));
            if (i == j) f.x -= tr;
            o[i * 3 + j] = f;
        }
}

template <bool FORCE>
static dwf_status launch_link(const Geom& G, const void* U, const void* lam, const void* x, void* out,
                              cudaStream_t st) {
    const bool su3 = G.nd == 4;
    const int sp = link_slice_groups(su3, (su3 ? 4 : 2) * G.V, G.Ls);
    const dim3 block(LINK_THREADS / sp, sp);
    const dim3 grid((unsigned)((G.V + block.x - 1) / block.x), su3 ? 4u : 2u);
    // SU(3): the 18 totals of every thread; U(1): the sums of groups 1 .. sp - 1
    const size_t sh = (su3 ? 18 * LINK_THREADS : (size_t)(sp - 1) * 2 * block.x) * sizeof(double);
    if (su3)
        k_linkgrad_su3<FORCE><<<grid, block, sh, st>>>((const double2*)U, (const double2*)lam, (const double2*)x,
                                                       (double2*)out, make_int4(G.L[0], G.L[1], G.L[2], G.L[3]), G.V,
                                                       G.Ls, make_int4(G.anti[0], G.anti[1], G.anti[2], G.anti[3]));
    else
        k_linkgrad_u1_2d<FORCE><<<grid, block, sh, st>>>((const double2*)U, (const double2*)lam, (const double2*)x,
                                                         (double*)out, G.L[0], G.V, G.Ls, G.anti[0], G.anti[1]);
    DWF_CHECK_LAUNCH();
    return DWF_OK;
}

}  // namespace dwf

using namespace dwf;

extern "C" {

dwf_status dwf_links_from_angles(const dwf_geom* g, const double* theta, void* U_out, void* stream) {
    clear_error();
    Geom G;
    DWF_TRY(check_geom(g, &G));
    if (G.group != DWF_U1) { set_error("link angles apply to U(1) only"); return DWF_ERR_ARG; }
    const long long n = link_len(G);
    if (n == 0) return DWF_OK;
    if (!theta || !U_out) { set_error("NULL device pointer"); return DWF_ERR_ARG; }
    const int grid = (int)((n + 255) / 256 < 152 * 16 ? (n + 255) / 256 : 152 * 16);
    k_links_from_angles<<<grid, 256, 0, as_stream(stream)>>>(theta, (double2*)U_out, n);
    DWF_CHECK_LAUNCH();
    return DWF_OK;
}

dwf_status dwf_gamma5_reflect(const dwf_geom* g, const void* in, void* out, int prec, void* stream) {
    clear_error();
    Geom G;
    DWF_TRY(check_geom(g, &G));
    if (!valid_prec(prec)) { set_error("bad precision %d", prec); return DWF_ERR_ARG; }
    const long long n = spinor_len(G);
    if (n == 0) return DWF_OK;
    if (!in || !out) { set_error("NULL device pointer"); return DWF_ERR_ARG; }
    if (in == out) { set_error("in and out must be distinct buffers"); return DWF_ERR_ARG; }
    const int dof = (int)site_dof(G);
    const int half = dof / 2;
    const int grid = (int)((n + 255) / 256 < 152 * 16 ? (n + 255) / 256 : 152 * 16);
    cudaStream_t st = as_stream(stream);
    if (prec == DWF_F64) k_gamma5_reflect<double2><<<grid, 256, 0, st>>>((const double2*)in, (double2*)out, G.V, G.Ls, dof, half);
    else                 k_gamma5_reflect<float2><<<grid, 256, 0, st>>>((const float2*)in, (float2*)out, G.V, G.Ls, dof, half);
    DWF_CHECK_LAUNCH();
    return DWF_OK;
}

dwf_status dwf_link_force(const dwf_geom* g, const void* U, const void* lam, const void* x, double* force,
                          void* stream) {
    clear_error();
    Geom G;
    DWF_TRY(check_geom(g, &G));
    if (G.V == 0) return DWF_OK;
    if (!U || !lam || !x || !force) { set_error("NULL device pointer"); return DWF_ERR_ARG; }
    if (!(G.nd == 2 && G.group == DWF_U1) && !(G.nd == 4 && G.group == DWF_SU3)) {
        set_error("the link force is built for 2-d U(1) and 4-d SU(3)");
        return DWF_ERR_UNSUPPORTED;
    }
    return launch_link<true>(G, U, lam, x, force, as_stream(stream));
}

dwf_status dwf_link_grad(const dwf_geom* g, const void* lam, const void* x, void* grad, void* stream) {
    clear_error();
    Geom G;
    DWF_TRY(check_geom(g, &G));
    if (G.V == 0) return DWF_OK;
    if (!lam || !x || !grad) { set_error("NULL device pointer"); return DWF_ERR_ARG; }
    if (!(G.nd == 2 && G.group == DWF_U1) && !(G.nd == 4 && G.group == DWF_SU3)) {
        set_error("the link gradient is built for 2-d U(1) and 4-d SU(3)");
        return DWF_ERR_UNSUPPORTED;
    }
    return launch_link<false>(G, nullptr, lam, x, grad, as_stream(stream));
}

}  // extern "C"
