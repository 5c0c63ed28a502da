// 4-d SU(3) Shamir operator: Eq. DWoperator with the 4-d Wilson kernel on
// 4 spins x 3 colours, chiral basis gamma_5 = diag(1, 1, -1, -1).
//
// One thread per 5-d site; a block is 32 consecutive sites x 8 slices, so the
// eight threads of a site that differ in s read its links through L1.  In the
// chiral basis gamma_mu = [[0, A_mu], [A_mu^dag, 0]] (A = -i sigma_k, or 1 for
// mu = 3); (1 -+ gamma_mu) psi = (h, -+ A^dag h) with the half spinor
// h = psi_up -+ A psi_low, so each hop multiplies two colour vectors by the
// link (the spin projection of the Wilson operator).  P_+ / P_- are the upper /
// lower spin pairs, so the s-hops add half spinors of psi_{s-1} and psi_{s+1}.
//
// Layout: canonical, psi[s][site][spin][colour] and U[mu][site][3][3], as the
// C ABI defines them.  The packed layout (dwf_pack_spinor / dwf_apply_packed) has
// its own kernel in dwf_fine4d_pair.cu; this file keeps the packed links'
// conversion and the packed entry points.
#include <algorithm>

#include "common.cuh"
#include "fine_kernels.cuh"

namespace dwf {

// Canonical layout: a site's 12 complex values are one record of 96 (FP32) or 192 (FP64) bytes.
// With W32 (records on 32-byte boundaries) they move in 32-byte pieces: a warp's load touches every
// one of its lines once per piece, and L1 handles a line per touch, so pieces of 16 bytes cost twice
// the L1 time.  Sites are 32-bit (a 4-d lattice has at most 2^28 of them); slice offsets 64-bit.
__device__ __forceinline__ void ld32(const float2* p, float2 (&v)[4]) {
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(v[0].x), "=f"(v[0].y), "=f"(v[1].x), "=f"(v[1].y), "=f"(v[2].x), "=f"(v[2].y), "=f"(v[3].x), "=f"(v[3].y)
        : "l"(p));
}
__device__ __forceinline__ void ld32(const double2* p, double2 (&v)[2]) {
    asm("ld.global.nc.v4.f64 {%0, %1, %2, %3}, [%4];"
        : "=d"(v[0].x), "=d"(v[0].y), "=d"(v[1].x), "=d"(v[1].y) : "l"(p));
}
__device__ __forceinline__ void ld16(const float2* p, float2 (&v)[2]) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(p));
    v[0] = make_float2(a.x, a.y); v[1] = make_float2(a.z, a.w);
}
__device__ __forceinline__ void ld16(const double2* p, double2 (&v)[1]) { v[0] = __ldg(p); }

// N values from p into v[0 .. N - 1]: 16-byte pieces up to the first 32-byte boundary (HEAD values) and at the end
template <bool W32, int N, int HEAD, class C>
__device__ __forceinline__ void ld_values(const C* p, C* v) {
    constexpr int P16 = 16 / sizeof(C), P32 = 32 / sizeof(C);
    constexpr int n32 = W32 ? (N - HEAD) / P32 : 0, first = W32 ? HEAD : 0;
#pragma unroll
    for (int i = 0; i < n32; ++i) {
        C t[P32];
        ld32(p + first + i * P32, t);
#pragma unroll
        for (int j = 0; j < P32; ++j) v[first + i * P32 + j] = t[j];
    }
#pragma unroll
    for (int e = 0; e < N; e += P16) {
        if (e >= first && e < first + n32 * P32) continue;
        C t[P16];
        ld16(p + e, t);
#pragma unroll
        for (int j = 0; j < P16; ++j) v[e + j] = t[j];
    }
}
template <bool W32, class C>
__device__ __forceinline__ void ld_spin4(const C* p, C (&v)[4][3]) { ld_values<W32, 12, 0>(p, &v[0][0]); }
// spins 2 hi, 2 hi + 1 (hi = 0: upper pair, 1: lower pair)
template <bool W32, int HI, class C>
__device__ __forceinline__ void ld_half(const C* p, C (&h)[2][3]) {
    ld_values<W32, 6, HI && sizeof(C) == 8 ? 2 : 0>(p + 6 * HI, &h[0][0]);
}
__device__ __forceinline__ void st_piece(float2* p, const float2* v, bool w32) {
    if (w32)
        asm volatile("st.global.cs.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(v[0].x), "f"(v[0].y),
                     "f"(v[1].x), "f"(v[1].y), "f"(v[2].x), "f"(v[2].y), "f"(v[3].x), "f"(v[3].y) : "memory");
    else
#pragma unroll
        for (int j = 0; j < 4; j += 2)
            __stcs(reinterpret_cast<float4*>(p + j), make_float4(v[j].x, v[j].y, v[j + 1].x, v[j + 1].y));
}
__device__ __forceinline__ void st_piece(double2* p, const double2* v, bool w32) {
    if (w32)
        asm volatile("st.global.cs.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(v[0].x), "d"(v[0].y), "d"(v[1].x),
                     "d"(v[1].y) : "memory");
    else {
        __stcs(p, v[0]);
        __stcs(p + 1, v[1]);
    }
}
template <bool W32, class C>
__device__ __forceinline__ void st_spin4(C* p, const C (&v)[4][3]) {
    constexpr int P32 = 32 / sizeof(C);
#pragma unroll
    for (int e = 0; e < 12; e += P32) st_piece(p + e, &v[0][0] + e, W32);
}

// A psi_low for direction mu (A = -i sigma_1, -i sigma_2, -i sigma_3, 1)
template <class C>
__device__ __forceinline__ void apply_A(int mu, const C (&l)[2][3], C (&o)[2][3]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        if (mu == 0) { o[0][c] = mk<C>(l[1][c].y, -l[1][c].x); o[1][c] = mk<C>(l[0][c].y, -l[0][c].x); }      // -i l1, -i l0
        else if (mu == 1) { o[0][c] = mk<C>(-l[1][c].x, -l[1][c].y); o[1][c] = l[0][c]; }                      // -l1, l0
        else if (mu == 2) { o[0][c] = mk<C>(l[0][c].y, -l[0][c].x); o[1][c] = mk<C>(-l[1][c].y, l[1][c].x); }  // -i l0, i l1
        else { o[0][c] = l[0][c]; o[1][c] = l[1][c]; }
    }
}
// A^dag h
template <class C>
__device__ __forceinline__ void apply_Adag(int mu, const C (&h)[2][3], C (&o)[2][3]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        if (mu == 0) { o[0][c] = mk<C>(-h[1][c].y, h[1][c].x); o[1][c] = mk<C>(-h[0][c].y, h[0][c].x); }      // i h1, i h0
        else if (mu == 1) { o[0][c] = h[1][c]; o[1][c] = mk<C>(-h[0][c].x, -h[0][c].y); }                      // h1, -h0
        else if (mu == 2) { o[0][c] = mk<C>(-h[0][c].y, h[0][c].x); o[1][c] = mk<C>(h[1][c].y, -h[1][c].x); }  // i h0, -i h1
        else { o[0][c] = h[0][c]; o[1][c] = h[1][c]; }
    }
}

// Block: 32 consecutive sites x 8 slices (fewer where there are fewer).  Blocks are numbered slice group
// fastest, so the slice groups of one set of sites run together and share its
// links and boundary slices in L2.  Bound by L1 (a spinor piece touches 24 lines per warp) and FP32
// issue; FP64 by the FP64 pipe.  16^3 x 32 x 16, FP16 links: 160 us against 222 us with 16-byte
// pieces and products and sums apart; 12^3 x 24 x 12 in FP64, at the 128 registers its values need,
// 799 against 1159 us.  (One table of neighbours per block in shared memory: 173 us, its barrier
// costs more than the divisions; the block's links in shared memory too: 191 us, and 226 us for
// the adjoint, whose registers then spill.)
template <class LT, class R, bool DAG, bool W32>
__global__ void __launch_bounds__(256, sizeof(R) == 8 ? 2 : 3) k_dwf4d(const typename LT::store* __restrict__ U,
                                               const typename cplx<R>::T* __restrict__ psi,
                                               typename cplx<R>::T* __restrict__ out, Fine4dParams p,
                                               int ngroups, const int* skip) {
    if (skip && *skip) return;
    using C = typename cplx<R>::T;
    const int V = (int)p.V;
    const int base = (int)(blockIdx.x / ngroups) * 32;
    const int site = base + threadIdx.x;
    const int s = (int)(blockIdx.x % ngroups) * 8 + threadIdx.y;
    if (site >= V || s >= p.Ls) return;
    int stride[4];
    int coord[4];
    {
        int st = 1, rem = site;
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) {
            const int q = rem / p.L[mu];
            stride[mu] = st;
            coord[mu] = rem - q * p.L[mu];
            rem = q;
            st *= p.L[mu];
        }
    }
    // s-hops.  D: up += psi_{s-1}.up (or -m psi_{Ls-1}.up), lo += psi_{s+1}.lo (or -m psi_0.lo)
    //          D^dag: up from s+1 / wall psi_0, lo from s-1 / wall psi_{Ls-1}
    const R mf = param_cast<R>(p.mf, p.mf_f);
    const int s_up = DAG ? (s + 1 < p.Ls ? s + 1 : 0) : (s > 0 ? s - 1 : p.Ls - 1);
    const int s_lo = DAG ? (s > 0 ? s - 1 : p.Ls - 1) : (s + 1 < p.Ls ? s + 1 : 0);
    const R f_up = DAG ? (s + 1 < p.Ls ? R(1) : -mf) : (s > 0 ? R(1) : -mf);
    const R f_lo = DAG ? (s > 0 ? R(1) : -mf) : (s + 1 < p.Ls ? R(1) : -mf);
    C up[2][3], lo[2][3];     // upper / lower spin pairs
    // In FP64 the sums start with the s-hops (at the end, all their inputs beside the sums made 100 registers
    // spill: 12^3 x 24 x 12 837 us against 798); in FP32 they end with them
    constexpr bool FIRST = sizeof(R) == 8;
    auto s_hops = [&] {
        C hu[2][3], hl[2][3];
        ld_half<W32, 0>(psi + ((long long)s_up * V + site) * 12, hu);
        ld_half<W32, 1>(psi + ((long long)s_lo * V + site) * 12, hl);
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                up[a][c] = FIRST ? scale(hu[a][c], f_up) : up[a][c] + scale(hu[a][c], f_up);
                lo[a][c] = FIRST ? scale(hl[a][c], f_lo) : lo[a][c] + scale(hl[a][c], f_lo);
            }
    };
    if (FIRST) s_hops();
    else
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int c = 0; c < 3; ++c) { up[a][c] = mk<C>(R(0), R(0)); lo[a][c] = mk<C>(R(0), R(0)); }
    const C* plane = psi + (long long)s * V * 12;

#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        // forward: y = x + mu, link U_mu(x); backward: y = x - mu, link U_mu(y)^dag
#pragma unroll
        for (int dirn = 0; dirn < 2; ++dirn) {
            const bool fwd = dirn == 0;
            const int L = p.L[mu];
            const bool cross = fwd ? (coord[mu] == L - 1) : (coord[mu] == 0);
            const int nb = fwd ? (cross ? site - (L - 1) * stride[mu] : site + stride[mu])
                               : (cross ? site + (L - 1) * stride[mu] : site - stride[mu]);
            const R ph = (cross && p.anti[mu]) ? R(0.5) : R(-0.5);
            // projector sign: D uses (1 - gamma) forward, (1 + gamma) backward; D^dag the opposite
            const bool minus = (fwd != DAG);
            C v[4][3];
            ld_spin4<W32>(plane + (long long)nb * 12, v);
            C lw[2][3] = {{v[2][0], v[2][1], v[2][2]}, {v[3][0], v[3][1], v[3][2]}};
            C Al[2][3];
            apply_A(mu, lw, Al);
            C h[2][3];
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
                for (int c = 0; c < 3; ++c) h[a][c] = minus ? (v[a][c] - Al[a][c]) : (v[a][c] + Al[a][c]);
            C u[3][3];
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int b = 0; b < 3; ++b) u[a][b] = load_link(U, ((long long)mu * V + (fwd ? site : nb)) * 9 + a * 3 + b);
            C uh[2][3];
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    // forward: U h; backward: U^dag h
                    C acc = fwd ? cmul(u[c][0], h[a][0]) : cmulc(u[0][c], h[a][0]);
#pragma unroll
                    for (int b = 1; b < 3; ++b) acc = fwd ? cmac(acc, u[c][b], h[a][b]) : cmacc(acc, u[b][c], h[a][b]);
                    uh[a][c] = acc;
                }
            C Ad[2][3];
            apply_Adag(mu, uh, Ad);
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    // the -1/2 and the boundary phase ride on the accumulating multiply-adds
                    up[a][c] = up[a][c] + scale(uh[a][c], ph);
                    lo[a][c] = lo[a][c] + scale(Ad[a][c], minus ? -ph : ph);
                }
        }
    }
    if (!FIRST) s_hops();
    // The diagonal term is the largest and comes last: error against 64 bits 5.0e-8 in FP32, 5.4e-8 with the s-hop after it
    const R diag = param_cast<R>(p.diag, p.diag_f);
    C self[4][3], o[4][3];
    ld_spin4<W32>(plane + (long long)site * 12, self);
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            o[a][c] = up[a][c] + scale(self[a][c], diag);
            o[a + 2][c] = lo[a][c] + scale(self[a + 2][c], diag);
        }
    st_spin4<W32>(out + ((long long)s * V + site) * 12, o);
}

static dwf_status grid4d(const Fine4dParams& p, unsigned* blocks, int* ngroups) {
    if (p.V > (1LL << 28)) { set_error("4-d lattices are limited to 2^28 sites"); return DWF_ERR_UNSUPPORTED; }
    const long long nb = (p.V + 31) / 32, ng = (p.Ls + 7) / 8;
    if (nb * ng > 0x7fffffffLL) { set_error("4-d lattice too large for one launch"); return DWF_ERR_ARG; }
    *blocks = (unsigned)(nb * ng);
    *ngroups = (int)ng;
    return DWF_OK;
}

template <class LT, class R>
static dwf_status launch4d(const void* U, const void* psi, void* out, const Fine4dParams& p, bool dagger,
                           cudaStream_t st, const int* skip = nullptr) {
    unsigned blocks;
    int ng;
    DWF_TRY(grid4d(p, &blocks, &ng));
    // fewer than 8 slices: no warps that end at once and hold their block's registers (12^3 x 24 x 1 in FP64 83 us
    // against 165, x 4 in FP32 19 against 25)
    const dim3 block(32, (unsigned)std::min(p.Ls, 8));
    using C = typename cplx<R>::T;
    auto Ut = reinterpret_cast<const typename LT::store*>(U);
    auto pi = reinterpret_cast<const C*>(psi);
    auto po = reinterpret_cast<C*>(out);
    // the ABI promises 16-byte alignment; records (96 or 192 bytes) keep a 32-byte aligned base's alignment
    const bool w32 = ((reinterpret_cast<uintptr_t>(psi) | reinterpret_cast<uintptr_t>(out)) & 31u) == 0;
    if (w32) {
        if (dagger) k_dwf4d<LT, R, true, true><<<blocks, block, 0, st>>>(Ut, pi, po, p, ng, skip);
        else        k_dwf4d<LT, R, false, true><<<blocks, block, 0, st>>>(Ut, pi, po, p, ng, skip);
    } else {
        if (dagger) k_dwf4d<LT, R, true, false><<<blocks, block, 0, st>>>(Ut, pi, po, p, ng, skip);
        else        k_dwf4d<LT, R, false, false><<<blocks, block, 0, st>>>(Ut, pi, po, p, ng, skip);
    }
    return DWF_OK;
}

static Fine4dParams params4d(const Geom& g, double M5, double mf) {
    Fine4dParams p;
    p.V = g.V;
    for (int mu = 0; mu < 4; ++mu) { p.L[mu] = g.L[mu]; p.anti[mu] = g.anti[mu]; }
    p.Ls = g.Ls;
    p.diag = (double)g.nd - M5 + 1.0;
    p.mf = mf;
    p.diag_f = (float)p.diag;
    p.mf_f = (float)mf;
    p.s_chunk = 0;
    return p;
}

dwf_status fine_apply_4d(const Geom& g, const void* U, const void* psi, void* out, double M5, double mf,
                         bool dagger, int prec, int s_chunk, cudaStream_t st, const int* skip) {
    (void)s_chunk;
    const Fine4dParams p = params4d(g, M5, mf);
    switch (prec) {
        case DWF_F64:       DWF_TRY((launch4d<LinkF64, double>(U, psi, out, p, dagger, st, skip))); break;
        case DWF_F32:       DWF_TRY((launch4d<LinkF32, float>(U, psi, out, p, dagger, st, skip))); break;
        case DWF_F32_L16:   DWF_TRY((launch4d<LinkH16, float>(U, psi, out, p, dagger, st, skip))); break;
        case DWF_F32_LBF16: DWF_TRY((launch4d<LinkBF16, float>(U, psi, out, p, dagger, st, skip))); break;
        default: set_error("bad precision %d", prec); return DWF_ERR_ARG;
    }
    DWF_CHECK_LAUNCH();
    return DWF_OK;
}

template <class T> __device__ __forceinline__ T cvt_link_p(double2 v);
template <> __device__ __forceinline__ float2 cvt_link_p<float2>(double2 v) {
    return make_float2(__double2float_rn(v.x), __double2float_rn(v.y));
}
template <> __device__ __forceinline__ __half2 cvt_link_p<__half2>(double2 v) {
    return __halves2half2(__double2half(v.x), __double2half(v.y));
}
template <> __device__ __forceinline__ __nv_bfloat162 cvt_link_p<__nv_bfloat162>(double2 v) {
    return __halves2bfloat162(__double2bfloat16(v.x), __double2bfloat16(v.y));
}
// one thread per packed link entry (mu, block, j, slot); entries of sites past V are zero
template <class T>
__global__ void k_pack_links(const double2* __restrict__ in, T* __restrict__ out, long long V, long long NB, long long n) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const long long slot = i & 31, j = (i >> 5) % 9, blk = (i >> 5) / 9;
        const long long mu = blk / NB, site = (blk % NB) * 32 + slot;
        out[i] = site < V ? cvt_link_p<T>(in[(mu * V + site) * 9 + j]) : cvt_link_p<T>(make_double2(0.0, 0.0));
    }
}

static dwf_status check_packed(const dwf_geom* g, Geom* G) {
    DWF_TRY(check_geom(g, G));
    if (G->nd != 4) { set_error("the packed layout is defined for 4-d SU(3) lattices"); return DWF_ERR_UNSUPPORTED; }
    return DWF_OK;
}
static int grid_for(long long n) { return (int)std::min<long long>((n + 255) / 256, 152LL * 16); }

}  // namespace dwf

using namespace dwf;

extern "C" {

size_t dwf_packed_spinor_size(const dwf_geom* g) {
    Geom G;
    if (check_geom(g, &G) != DWF_OK || G.nd != 4 || G.Ls % 2) return 0;
    return (size_t)(G.Ls * ((G.V + 31) / 32) * 32 * 12);
}

size_t dwf_packed_link_size(const dwf_geom* g) {
    Geom G;
    if (check_geom(g, &G) != DWF_OK || G.nd != 4) return 0;
    return (size_t)(4 * ((G.V + 31) / 32) * 32 * 9);
}

dwf_status dwf_pack_links(const dwf_geom* g, const void* U64, void* U_packed, int prec, void* stream) {
    clear_error();
    Geom G;
    DWF_TRY(check_packed(g, &G));
    if (prec != DWF_F32 && prec != DWF_F32_L16 && prec != DWF_F32_LBF16) {
        set_error("packed links take precision F32, F32_L16 or F32_LBF16 (got %d)", prec);
        return DWF_ERR_ARG;
    }
    const long long NB = (G.V + 31) / 32, n = 4 * NB * 32 * 9;
    if (!U64 || !U_packed) { set_error("NULL link pointer"); return DWF_ERR_ARG; }
    cudaStream_t st = as_stream(stream);
    auto in = reinterpret_cast<const double2*>(U64);
    const int blocks = grid_for(n);
    if (prec == DWF_F32) k_pack_links<float2><<<blocks, 256, 0, st>>>(in, (float2*)U_packed, G.V, NB, n);
    else if (prec == DWF_F32_L16) k_pack_links<__half2><<<blocks, 256, 0, st>>>(in, (__half2*)U_packed, G.V, NB, n);
    else k_pack_links<__nv_bfloat162><<<blocks, 256, 0, st>>>(in, (__nv_bfloat162*)U_packed, G.V, NB, n);
    DWF_CHECK_LAUNCH();
    return DWF_OK;
}

dwf_status dwf_pack_spinor(const dwf_geom* g, const void* psi, void* packed, void* stream) {
    clear_error();
    Geom G;
    DWF_TRY(check_packed(g, &G));
    if (!psi || !packed) { set_error("NULL device pointer"); return DWF_ERR_ARG; }
    if (!aligned16(psi) || !aligned16(packed)) { set_error("spinor buffers must be 16-byte aligned"); return DWF_ERR_ARG; }
    if (psi == packed) { set_error("psi and packed must be distinct buffers"); return DWF_ERR_ARG; }
    return pack_spinor_paired(G, psi, packed, as_stream(stream));
}

dwf_status dwf_unpack_spinor(const dwf_geom* g, const void* packed, void* psi, void* stream) {
    clear_error();
    Geom G;
    DWF_TRY(check_packed(g, &G));
    if (!psi || !packed) { set_error("NULL device pointer"); return DWF_ERR_ARG; }
    if (!aligned16(psi) || !aligned16(packed)) { set_error("spinor buffers must be 16-byte aligned"); return DWF_ERR_ARG; }
    if (psi == packed) { set_error("psi and packed must be distinct buffers"); return DWF_ERR_ARG; }
    return unpack_spinor_paired(G, packed, psi, as_stream(stream));
}

dwf_status dwf_apply_packed(const dwf_geom* g, const void* U_packed, const void* psi, void* out, double M5,
                            double mf, int dagger, int prec, void* stream) {
    clear_error();
    Geom G;
    DWF_TRY(check_packed(g, &G));
    if (!U_packed || !psi || !out) { set_error("NULL device pointer"); return DWF_ERR_ARG; }
    if (!aligned16(psi) || !aligned16(out)) { set_error("spinor buffers must be 16-byte aligned"); return DWF_ERR_ARG; }
    if (psi == out) { set_error("psi and out must be distinct buffers"); return DWF_ERR_ARG; }
    return fine_apply_4d_paired(G, U_packed, psi, out, M5, mf, dagger != 0, prec, as_stream(stream));
}

}  // extern "C"
