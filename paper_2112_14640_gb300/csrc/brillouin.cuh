// brillouin.cuh -- multi-RHS Brillouin Dirac operator, Eq. (app_bril) with
// Eqs. (def_ider, def_blap) at r = 1, c_SW = 0:
//   (D_B psi)(n) = (m0 - lambda_0/2) psi(n)
//       + sum_{s in {-1,0,1}^4, s != 0} [sgn rho_k sum_mu s_mu gamma_mu - lambda_k/2] (x) W_s(n) psi(n+s)
// rho = (64,16,4,1)/432, lambda = (-240,8,4,2,1)/64, k = |s|_1, W_s from
// Tab. off-axis, built once per gauge field (links.cu) and stored in the
// order q, with the scale rho_k s_lead and the per-site layout of bril_dirs.h.  The derivative
// carries every axis the offset moves along (sum_mu s_mu gamma_mu), the
// reading of Eq. (def_ider).  sgn = +1 gives D_B, sgn = -1 gives
// D_B^dag = gamma5 D_B gamma5 (the derivative part flips sign).  A clover
// term, when the operator carries one, is added site by site at the end
// (clover.cuh; Eq. def_bril).
//
// With the stored W~ = rho_k s_lead W_s every offset contributes
//   sgn * W~ [ sum_{mu in M} e_mu gamma_mu psi(n+s) + d psi(n+s) ],
//   e_mu = s_lead s_mu,  d = -sgn c_k s_lead,
// and the common factor sgn is applied once to the accumulated sum.  The
// offsets are visited row by row (bril_dirs.h), every support M a compile-time
// mask, so the gamma matrices of the axes outside M cost nothing: in the
// chiral basis of App. A each gamma_mu is a signed permutation of the spin
// components, and the spin combination costs 8k real FMAs per colour and RHS
// instead of 40.  The sign patterns of the y, z, t axes run in a loop; the
// three offsets of a row read neighbours that share cache lines.
//
// What bounds it: the FP32 pipe (209 multiply-adds per offset and RHS, 0.65 ms
// at 16^3x32, N_v = 12, N_c = 3, FP32) and, beside it, the L1 pipe.  With W~
// loaded by each thread, an element of W~ was a warp-wide load touching one
// cache line per site, half of the L1 work, and issue slots ran out first
// (69% busy): 1.256 ms.  W~ staged in shared memory for the block
// (wstage.cuh), rows in x order and packed products (common.cuh: one issue
// slot for two multiply-adds; 778 M instead of 1074 M warp instructions):
// 1.067 ms, the FP32 pipe 65% busy.  Packed products alone gave 1.128 ms.
#pragma once
#include "bril_dirs.h"
#include "clover.cuh"
#include "internal.h"
#include "wstage.cuh"

namespace dgb {
namespace bril {

// phase * p[pi] of gamma_mu acting on spin S (chiral basis of App. A):
//   t: pi = (2,3,0,1), phases ( 1,  1, 1,  1)    z: pi = (2,3,0,1), phases (-i, i, i, -i)
//   y: pi = (3,2,1,0), phases (-1,  1, 1, -1)    x: pi = (3,2,1,0), phases (-i, -i, i, i)
template <int MU, int S, typename A>
__device__ __forceinline__ cx<A> gamma_term(const cx<A> (&p)[4]) {
    constexpr int PI = MU >= 2 ? (S ^ 2) : (3 - S);
    // 0: +1, 1: -1, 2: +i, 3: -i
    constexpr int PH = MU == 3 ? 0
                     : MU == 2 ? ((S == 0 || S == 3) ? 3 : 2)
                     : MU == 1 ? ((S == 0 || S == 3) ? 1 : 0)
                               : (S <= 1 ? 3 : 2);
    const cx<A> v = p[PI];
    if constexpr (PH == 0) return v;
    else if constexpr (PH == 1) return cx<A>{-v.re, -v.im};
    else if constexpr (PH == 2) return cx<A>{-v.im, v.re};
    else return cx<A>{v.im, -v.re};
}

// f += e_mu * (gamma_mu p)_S for the axes MU.. of M other than the lead
template <int M, int S, int MU, typename A>
__device__ __forceinline__ void add_axes(cx<A> &f, const cx<A> (&p)[4], const A (&e)[4]) {
    if constexpr (MU < 4) {
        if constexpr (((M >> MU) & 1) && MU != lead_axis(M)) {
            const cx<A> t = gamma_term<MU, S>(p);
            f.re = fma(e[MU], t.re, f.re);
            f.im = fma(e[MU], t.im, f.im);
        }
        add_axes<M, S, MU + 1>(f, p, e);
    }
}

// spin component S of  sum_{mu in M} e_mu gamma_mu p + d p
template <int M, int S, typename A>
__device__ __forceinline__ cx<A> spin_mix(const cx<A> (&p)[4], const A (&e)[4], A d) {
    cx<A> f = gamma_term<lead_axis(M), S>(p);
    add_axes<M, S, 0>(f, p, e);
    f.re = fma(d, p[S].re, f.re);
    f.im = fma(d, p[S].im, f.im);
    return f;
}

// Packed FP32 forms of the same: gamma_t and gamma_y only permute and negate
// whole components (one packed multiply-add), gamma_z and gamma_x also swap
// real and imaginary parts (two scalar ones).
template <int MU, int S>
constexpr int gamma_perm() { return MU >= 2 ? (S ^ 2) : (3 - S); }
// y: -1 on spins 0 and 3
template <int MU, int S>
constexpr bool gamma_neg() { return MU == 1 && (S == 0 || S == 3); }

template <int M, int S, int MU>
__device__ __forceinline__ void add_axes(pk2 &f, const pk2 (&p)[4], const float (&e)[4]) {
    if constexpr (MU < 4) {
        if constexpr (((M >> MU) & 1) && MU != lead_axis(M)) {
            constexpr int PI = gamma_perm<MU, S>();
            if constexpr (MU == 3 || MU == 1) {
                f = fma2(bcast2(gamma_neg<MU, S>() ? -e[MU] : e[MU]), p[PI], f);
            } else {
                const cx<float> q[4] = {unpack2(p[0]), unpack2(p[1]), unpack2(p[2]), unpack2(p[3])};
                const cx<float> t = gamma_term<MU, S>(q), g = unpack2(f);
                f = pack2(fma(e[MU], t.re, g.re), fma(e[MU], t.im, g.im));
            }
        }
        add_axes<M, S, MU + 1>(f, p, e);
    }
}

template <int M, int S>
__device__ __forceinline__ pk2 spin_mix(const pk2 (&p)[4], const float (&e)[4], float d) {
    constexpr int LM = lead_axis(M), PI = gamma_perm<LM, S>();
    pk2 f;
    if constexpr (LM == 3 || (LM == 1 && !gamma_neg<LM, S>())) {
        f = fma2(bcast2(d), p[S], p[PI]);
    } else if constexpr (LM == 1) {
        f = fma2(bcast2(-1.f), p[PI], mul2(bcast2(d), p[S]));
    } else {
        const cx<float> q[4] = {unpack2(p[0]), unpack2(p[1]), unpack2(p[2]), unpack2(p[3])};
        const cx<float> t = gamma_term<LM, S>(q);
        f = pack2(fma(d, q[S].re, t.re), fma(d, q[S].im, t.im));
    }
    add_axes<M, S, 0>(f, p, e);
    return f;
}

// spin component S of  sum_mu e_mu gamma_mu p + d p  for all four axes
// (e_mu = 0 off the support; the run-time-mask path of large N_c)
template <int S, typename A>
__device__ __forceinline__ cx<A> spin_mix_rt(const cx<A> (&p)[4], const A (&e)[4], A d) {
    cx<A> f = {d * p[S].re, d * p[S].im};
    const cx<A> t[4] = {gamma_term<0, S>(p), gamma_term<1, S>(p), gamma_term<2, S>(p), gamma_term<3, S>(p)};
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        f.re = fma(e[mu], t[mu].re, f.re);
        f.im = fma(e[mu], t[mu].im, f.im);
    }
    return f;
}

template <int NC, int VR, typename E, typename EL, int LAYOUT>
struct Ctx {
    using A = typename Acc<E>::T;
    const EL *wp;          // this site's W~ (offset 0, element 0), [q][a][b]
    const E *in;
    int n;                 // output site (volumes are below 2^31 sites)
    long long vbase;       // offset of this thread's RHS inside a site (complex numbers)
    int dp[4], dm[4];      // site-index offsets of n + mu and n - mu (periodic)
    Lat g;
    A sgn;
};

// One offset of support M with the signs sig, applied to the neighbour m with W~ in W.
template <typename P, int M, int NC, int VR, typename E, typename EL, int LAYOUT, typename A>
__device__ __forceinline__ void offset(const Ctx<NC, VR, E, EL, LAYOUT> &C, int m, const A (&sig)[4],
                                       const cx<A> (&W)[NC][NC], typename P::Acc (&acc)[NC][4][VR]) {
    using L = Layout<LAYOUT>;
    using V = typename P::Vec;
    constexpr int K = popc4(M);
    const A ck = (A)c_lambda(K);
    const long long cs = L::cs_stride(C.g);
    const A sl = sig[lead_axis(M)];
    A e[4];
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) e[mu] = sig[mu] * sl;
    const A d = -C.sgn * ck * sl;
    const E *pm = C.in + 2 * (L::vec(C.g, (long long)m, NC * 4, 0) + C.vbase);
#pragma unroll
    for (int kc = 0; kc < NC; ++kc) {
        cx<A> p[4][VR];
#pragma unroll
        for (int s = 0; s < 4; ++s) load_cx<E, VR, A>(pm + 2 * (kc * 4 + s) * cs, p[s]);
        typename P::Mul w[NC];
#pragma unroll
        for (int a = 0; a < NC; ++a) w[a] = P::mul(W[a][kc]);
#pragma unroll
        for (int v = 0; v < VR; ++v) {
            const V pv[4] = {P::vec(p[0][v]), P::vec(p[1][v]), P::vec(p[2][v]), P::vec(p[3][v])};
            const V f0 = spin_mix<M, 0>(pv, e, d);
            const V f1 = spin_mix<M, 1>(pv, e, d);
            const V f2 = spin_mix<M, 2>(pv, e, d);
            const V f3 = spin_mix<M, 3>(pv, e, d);
#pragma unroll
            for (int a = 0; a < NC; ++a) {
                acc[a][0][v].mac(w[a], f0);
                acc[a][1][v].mac(w[a], f1);
                acc[a][2][v].mac(w[a], f2);
                acc[a][3][v].mac(w[a], f3);
            }
        }
    }
}

// The W~ of a run of offsets: read from the block's staged copy ...
template <int NC, typename EL, typename A>
struct StagedW {
    wst::Ring<NC, EL> ring;
    const EL *w = nullptr;
    __device__ __forceinline__ void enter(int stage) { w = ring.enter(stage); }
    // matrix i of the stage (compile-time i)
    __device__ __forceinline__ void get(int i, cx<A> (&W)[NC][NC]) { wst::load_mat_shared<NC, EL, A>(w + i * (2 * NC * NC), W); }
    __device__ __forceinline__ void skip(int n) { w += n * (2 * NC * NC); }
};

// Large N_c: one offset (its signs sig run-time values, 0 off the support) with
// the W~ read one row at a time instead of a register double buffer of N_c^2
// elements; the spin-mixed neighbour spinor of every colour is formed first.
// With e_mu = s_mu s_lead on the axes of M and 0 elsewhere, the spin factor
// is sum_mu e_mu gamma_mu + d (as in `offset`, without compile-time masks).
template <int NC, int VR, typename E, typename EL, int LAYOUT, typename A>
__device__ __forceinline__ void offset_rows(const Ctx<NC, VR, E, EL, LAYOUT> &C, int q, const A (&sig)[4],
                                            cx<A> (&acc)[NC][4][VR]) {
    using L = Layout<LAYOUT>;
    const int K = (sig[0] != 0) + (sig[1] != 0) + (sig[2] != 0) + (sig[3] != 0);
    const A ck = (A)(27.0 / 128.0) * (A)(1 << K);   // c_k = 27/64 2^(k-1)
    const long long cs = L::cs_stride(C.g);
    int m = C.n;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) m += sig[mu] > 0 ? C.dp[mu] : sig[mu] < 0 ? C.dm[mu] : 0;
    // the sign of the highest axis s moves along
    const A sl = sig[3] != 0 ? sig[3] : sig[2] != 0 ? sig[2] : sig[1] != 0 ? sig[1] : sig[0];
    A e[4];
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) e[mu] = sig[mu] * sl;
    const A d = -C.sgn * ck * sl;
    const E *pm = C.in + 2 * (L::vec(C.g, (long long)m, NC * 4, 0) + C.vbase);
    cx<A> f[NC][4][VR];
#pragma unroll
    for (int kc = 0; kc < NC; ++kc) {
        cx<A> p[4][VR];
#pragma unroll
        for (int s = 0; s < 4; ++s) load_cx<E, VR, A>(pm + 2 * (kc * 4 + s) * cs, p[s]);
#pragma unroll
        for (int v = 0; v < VR; ++v) {
            const cx<A> pv[4] = {p[0][v], p[1][v], p[2][v], p[3][v]};
            f[kc][0][v] = spin_mix_rt<0>(pv, e, d);
            f[kc][1][v] = spin_mix_rt<1>(pv, e, d);
            f[kc][2][v] = spin_mix_rt<2>(pv, e, d);
            f[kc][3][v] = spin_mix_rt<3>(pv, e, d);
        }
    }
    const EL *wq = C.wp + q * (2 * NC * NC);
#pragma unroll 1
    for (int a = 0; a < NC; ++a) {
        cx<A> wr[NC];
#pragma unroll
        for (int kc = 0; kc < NC; ++kc) wr[kc] = ld1<EL, A>(wq + 2 * (a * NC + kc));
        cx<A> o[4][VR];
#pragma unroll
        for (int s = 0; s < 4; ++s)
#pragma unroll
            for (int v = 0; v < VR; ++v) o[s][v] = cx<A>{0, 0};
#pragma unroll
        for (int kc = 0; kc < NC; ++kc)
#pragma unroll
            for (int s = 0; s < 4; ++s)
#pragma unroll
                for (int v = 0; v < VR; ++v) cmac(o[s][v], wr[kc], f[kc][s][v]);
        // run-time row index: add through a compile-time switch over rows
#pragma unroll
        for (int r = 0; r < NC; ++r)
            if (r == a)
#pragma unroll
                for (int s = 0; s < 4; ++s)
#pragma unroll
                    for (int v = 0; v < VR; ++v) acc[r][s][v] = acc[r][s][v] + o[s][v];
    }
}

// ... or by each thread from global memory, the next matrix requested while the
// current one is applied (few threads per site).
template <int NC, typename EL, typename A>
struct DirectW {
    const EL *p;            // the matrix held in nxt
    const EL *last;
    cx<A> nxt[NC][NC];
    __device__ __forceinline__ void start(const EL *w) {
        p = w;
        last = w + 79 * (2 * NC * NC);
        load_mat<NC, EL, A>(p, nxt);
    }
    __device__ __forceinline__ void enter(int) {}
    __device__ __forceinline__ void get(int, cx<A> (&W)[NC][NC]) {
#pragma unroll
        for (int a = 0; a < NC; ++a)
#pragma unroll
            for (int b = 0; b < NC; ++b) W[a][b] = nxt[a][b];
        if (p != last) load_mat<NC, EL, A>(p += 2 * NC * NC, nxt);
    }
    __device__ __forceinline__ void skip(int) {}
};

// Signs of the y, z, t axes of support R (sign pattern b) and the row's site.
template <int R, int NC, int VR, typename E, typename EL, int LAYOUT, typename A>
__device__ __forceinline__ int row_signs(const Ctx<NC, VR, E, EL, LAYOUT> &C, int b, A (&sig)[4]) {
    int m = C.n, j = 0;
    sig[0] = 1;
#pragma unroll
    for (int mu = 1; mu < 4; ++mu) {
        sig[mu] = 1;
        if ((R >> (mu - 1)) & 1) {
            const bool neg = (b >> j++) & 1;
            sig[mu] = neg ? (A)-1 : (A)1;
            m += neg ? C.dm[mu] : C.dp[mu];
        }
    }
    return m;
}

// The rows of support R and up, two rows (six offsets) per stage of W~.
// Everything that depends on the support alone is fixed at compile time; the
// signs run in a loop.  The neighbours of a row, s_x = 0, +1, -1, share cache
// lines.
template <typename P, int R, int NC, int VR, typename E, typename EL, int LAYOUT, typename A, typename WSRC>
__device__ __forceinline__ void rows_from(const Ctx<NC, VR, E, EL, LAYOUT> &C, WSRC &w, int &stage,
                                          typename P::Acc (&acc)[NC][4][VR]) {
    if constexpr (R <= 7) {
        cx<A> W[NC][NC];
        A sig[4];
        if constexpr (R == 0) {
            w.enter(stage++);
            row_signs<0>(C, 0, sig);
            w.get(0, W);
            offset<P, 1>(C, C.n + C.dp[0], sig, W, acc);
            sig[0] = -1;
            w.get(1, W);
            offset<P, 1>(C, C.n + C.dm[0], sig, W, acc);
        } else {
#pragma unroll 1
            for (int b = 0; b < (1 << popc4(R)); b += 2) {
                w.enter(stage++);
#pragma unroll 1
                for (int r = 0; r < 2; ++r) {
                    const int m = row_signs<R>(C, b + r, sig);
                    w.get(0, W);
                    offset<P, R << 1>(C, m, sig, W, acc);
                    w.get(1, W);
                    offset<P, (R << 1) | 1>(C, m + C.dp[0], sig, W, acc);
                    sig[0] = -1;
                    w.get(2, W);
                    offset<P, (R << 1) | 1>(C, m + C.dm[0], sig, W, acc);
                    w.skip(3);
                }
            }
        }
        rows_from<P, R + 1, NC, VR, E, EL, LAYOUT, A>(C, w, stage, acc);
    }
}

}  // namespace bril

// STAGED: W~ through shared memory, one ring per block (wstage.cuh); else each
// thread reads its own.
template <int NC, int VR, typename E, int MINB, int LAYOUT, typename EL, bool STAGED>
__global__ void __launch_bounds__(stencil_max_threads(MINB), (MINB > 1 ? 1 : 0))
    brillouin_kernel(const EL *__restrict__ W, const E *__restrict__ in, E *__restrict__ out, Lat g,
                     typename Acc<E>::T centre, typename Acc<E>::T sgn, const EL *__restrict__ clov) {
    using A = typename Acc<E>::T;
    using L = Layout<LAYOUT>;
    const int nchunk = g.nv / VR;
    const long long total = g.nsites * nchunk, tid0 = (long long)blockIdx.x * blockDim.x;
    long long tid = tid0 + threadIdx.x;
    // a staged block's threads all copy and wait; those past the end repeat the last one's work
    const bool live = tid < total;
    if (!live) {
        if constexpr (!STAGED) return;
        tid = total - 1;
    }
    long long i;
    int j;
    split_tid(tid, nchunk, i, j);
    const long long n = g.n0 + i;
    const Coord c = site_coords(g, n);

    bril::Ctx<NC, VR, E, EL, LAYOUT> C;
    C.g = g;
    C.in = in;
    C.n = (int)n;
    C.sgn = sgn;
    C.vbase = (long long)j * VR;
    // W~ of one site contiguous in visiting order for either vector layout
    C.wp = W + 2LL * n * 80 * NC * NC;
    {
        const int co[4] = {c.x, c.y, c.z, c.t};
        const int ext[4] = {g.nx, g.ny, g.nz, g.nt};
        int stride = 1;
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) {
            C.dp[mu] = (co[mu] == ext[mu] - 1 ? -(ext[mu] - 1) : 1) * stride;
            C.dm[mu] = (co[mu] == 0 ? ext[mu] - 1 : -1) * stride;
            stride *= ext[mu];
        }
    }

    cx<A> acc[NC][4][VR];
    if constexpr (NC <= kMaxNcSmall) {
        using P = StencilProd<NC, 4, VR, MINB, A>;
        typename P::Acc sum[NC][4][VR];
        int stage = 0;
        if constexpr (STAGED) {
            extern __shared__ __align__(16) unsigned char w_ring[];
            const long long s0 = tid0 / nchunk, end = tid0 + blockDim.x < total ? tid0 + blockDim.x : total;
            bril::StagedW<NC, EL, A> w;
            w.ring.src = reinterpret_cast<const unsigned char *>(W + 2LL * (g.n0 + s0) * 80 * NC * NC);
            w.ring.smem = w_ring;
            w.ring.nsites = (int)((end - 1) / nchunk - s0 + 1);
            w.ring.slots = wst::block_sites(blockDim.x, nchunk);
            w.ring.mine = (int)(i - s0);
            w.ring.start();
            bril::rows_from<P, 0, NC, VR, E, EL, LAYOUT, A>(C, w, stage, sum);
            if (!live) return;
        } else {
            bril::DirectW<NC, EL, A> w;
            w.start(C.wp);
            bril::rows_from<P, 0, NC, VR, E, EL, LAYOUT, A>(C, w, stage, sum);
        }
#pragma unroll
        for (int a = 0; a < NC; ++a)
#pragma unroll
            for (int s = 0; s < 4; ++s)
#pragma unroll
                for (int v = 0; v < VR; ++v) acc[a][s][v] = sum[a][s][v].value();
    } else {
#pragma unroll
        for (int a = 0; a < NC; ++a)
#pragma unroll
            for (int s = 0; s < 4; ++s)
#pragma unroll
                for (int v = 0; v < VR; ++v) acc[a][s][v] = cx<A>{0, 0};
        // the offsets in storage order: rows R = 0..7, sign patterns b, s_x = 0, +1, -1
        int q = 0;
#pragma unroll 1
        for (int r = 0; r < 8; ++r)
#pragma unroll 1
            for (int b = 0; b < (1 << bril::popc4(r)); ++b)
#pragma unroll 1
                for (int x = r ? 0 : 1; x < 3; ++x) {
                    A sig[4] = {x == 0 ? (A)0 : x == 1 ? (A)1 : (A)-1, 0, 0, 0};
                    int jbit = 0;
#pragma unroll
                    for (int mu = 1; mu < 4; ++mu)
                        if ((r >> (mu - 1)) & 1) sig[mu] = (b >> jbit++) & 1 ? (A)-1 : (A)1;
                    bril::offset_rows(C, q++, sig, acc);
                }
    }

    const long long base = 2 * (L::vec(g, n, NC * 4, 0) + (long long)j * VR);
    write_site<-1, NC, VR, LAYOUT, E, A, EL>(in, out, clov, g, n, base, centre, sgn, acc);
}

template <typename E, int LAYOUT, typename EL>
int launch_brillouin_v(const dirac_op *op, const void *in, void *out, double m0, int sgn, cudaStream_t s) {
    int vr, minb, block;
    launch_variant(op, vr, minb, block);
    vr = aligned_vr(vr, op->prec, in, out);
    using A = typename Acc<E>::T;
    return dispatch_nc<big_nc_ok<E>()>(op->nc, [&](auto ncc) {
        constexpr int NC = decltype(ncc)::value;
        return dispatch_vr(vr, [&](auto vrc) {
            constexpr int VR = decltype(vrc)::value;
            if constexpr (!vr_compiled<NC>(VR)) return (int)DIRAC_ERR_INVALID_ARG;
            else {
                const int nchunk = op->nv / VR;
                const long long threads = op->lat.nsites * nchunk;
                // m0 - lambda_0 / 2 = m0 + 240/128
                auto go = [&](auto kernel, int T, size_t smem) {
                    kernel<<<grid_for(threads, T), T, smem, s>>>((const EL *)op->w, (const E *)in, (E *)out, op->lat,
                                                                (A)(m0 + 240.0 / 128.0), (A)sgn, (const EL *)op->clover);
                    return launch_check("brillouin_kernel");
                };
                const size_t smem = NC <= kMaxNcSmall ? wst::smem_bytes<NC, EL>(block, nchunk) : 0;
                if (NC > kMaxNcSmall || nchunk < wst::kMinChunks<EL> || smem > wst::kMaxSmem) {
                    // W~ read by each thread: compiled for two register classes only
                    if constexpr (NC == 3 && VR == 1) {
                        if (minb > 1) return go(brillouin_kernel<NC, VR, E, 4, LAYOUT, EL, false>, block <= 512 ? block : 512, 0);
                    }
                    return go(brillouin_kernel<NC, VR, E, 1, LAYOUT, EL, false>, block <= kStencilBlock ? block : kStencilBlock, 0);
                }
                if constexpr (NC <= kMaxNcSmall) {
                    return dispatch_minb<NC>(minb, [&](auto mbc) {
                        constexpr int MINB = decltype(mbc)::value;
                        if (smem > 48 * 1024) {
                            const int rc = cuda_check(
                                cudaFuncSetAttribute(brillouin_kernel<NC, VR, E, MINB, LAYOUT, EL, true>,
                                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)wst::kMaxSmem),
                                "brillouin_kernel shared memory");
                            if (rc) return rc;
                        }
                        return go(brillouin_kernel<NC, VR, E, MINB, LAYOUT, EL, true>, block, smem);
                    });
                }
                return (int)DIRAC_ERR_INVALID_ARG;
            }
        });
    });
}

}  // namespace dgb
