// force.cu -- link derivative of the pseudofermion action
//   S = sum_v Re phi_v^dag (D_W^dag D_W)^-1 phi_v       (the paper has no force; derived)
// Given psi = (D^dag D)^-1 phi and chi = D psi, the two hops of D_W through
// U_mu(n) give, with spin and RHS summed,
//   B_mu(n) = sum psi(n+mu) [(1 - gamma_mu) chi(n)]^dag,
//   C_mu(n) = sum psi(n) [(1 + gamma_mu) chi(n+mu)]^dag,
//   dS = Re sum tr[dU_mu(n) (B_mu(n) + C_mu(n)^dag)].
// mode TA:   F_mu(n) = P_TA(U B - C U^dag), so that dS/deps = Re sum tr[X F] for
//            U -> exp(eps X) U, X in su(Nc);
// mode GRAD: G_mu(n) = bc * (B^dag + C), so that dS = Re sum conj(G) dU for the
//            caller's (unphased) links.
// One thread per (site, mu).  1 + a gamma_mu is half its own square and its
// lower two spins are the upper two times a phase and a permutation, so
//   sum over four spins of psi [(1 + a gamma) chi]^dag
//     = sum over the upper two of [(1 + a gamma) psi] [(1 + a gamma) chi]^dag,
// half the products.  The permutation and phase of mu are selects, so the four
// directions of a site, neighbours in a warp, run the same instructions and
// read the same lines.  What bounds it is the L1 tag rate (up to 32 lines per
// load, the sites being a spinor apart), so a load takes as many right-hand
// sides as N_v and the alignment allow, up to 32 bytes.
// One right-hand side per load and four spins, and now, us (site-outer, N_c = 3;
// 26 is the traffic floor of D_W at N_v = 4): 16^3x32, FP32, D_W N_v = 4: 243 and
// 106, N_v = 8: 447 and 178; D_S N_v = 8: 104 and 70; 12^3x16, FP64, N_v = 4: D_W
// 401 and 228.
//
// The staggered operator (Eq. def_stag) gives the same final form with
//   B_mu(n) = -eta_mu(n) sum psi(n+mu) chi(n)^dag,  C_mu(n) = eta_mu(n) sum psi(n) chi(n+mu)^dag
// (colour vectors, RHS summed; eta_mu(n+mu) = eta_mu(n) because eta_mu only
// depends on the coordinates before mu).
#include "internal.h"

namespace dgb {

// Component S (0 or 1) of (1 + a gamma_mu) p, a = -1 where `minus`, in the chiral
// basis of App. A, for NC colours and VR right-hand sides of one site:
//   mu = 1: p0 - a i p3, p1 - a i p2    mu = 2: p0 - a p3, p1 + a p2
//   mu = 3: p0 - a i p2, p1 + a i p3    mu = 4: p0 + a p2, p1 + a p3
template <int NC, int VR, int S, typename E, typename A>
__device__ __forceinline__ void load_half(const E *__restrict__ p, long long cs, int mu, bool minus,
                                          cx<A> (&h)[NC][VR]) {
    const int partner = mu < 2 ? 3 - S : 2 + S;
    const bool im = !(mu & 1);
    const A f = minus != (S == 0 ? mu != 3 : mu == 0) ? (A)-1 : (A)1;
#pragma unroll
    for (int a = 0; a < NC; ++a) {
        cx<A> y[VR];
        load_cx<E, VR, A>(p + 2 * (a * 4 + S) * cs, h[a]);
        load_cx<E, VR, A>(p + 2 * (a * 4 + partner) * cs, y);
#pragma unroll
        for (int v = 0; v < VR; ++v)
            h[a][v] = cx<A>{fma(f, im ? -y[v].im : y[v].re, h[a][v].re), fma(f, im ? y[v].re : y[v].im, h[a][v].im)};
    }
}

// M += sum over the VR right-hand sides of x y^dag
template <int NC, int VR, typename A>
__device__ __forceinline__ void add_outer(cx<A> (&M)[NC][NC], const cx<A> (&x)[NC][VR], const cx<A> (&y)[NC][VR]) {
#pragma unroll
    for (int v = 0; v < VR; ++v)
#pragma unroll
        for (int a = 0; a < NC; ++a)
#pragma unroll
            for (int b = 0; b < NC; ++b) cmac(M[a][b], x[a][v], conj(y[b][v]));
}

// F = P_TA(U B - C U^dag) (mode 0) or G = bc (B^dag + C) (mode 1) for link (n, mu)
template <int NC, typename E, int LAYOUT>
__device__ __forceinline__ void force_out(const E *__restrict__ U, E *__restrict__ out, const Lat &g, long long tid,
                                          long long n, int mu, const Coord &c, const cx<typename Acc<E>::T> (&B)[NC][NC],
                                          const cx<typename Acc<E>::T> (&C)[NC][NC], int bc0, int bc1, int bc2, int bc3,
                                          int mode) {
    using L = Layout<LAYOUT>;
    using A = typename Acc<E>::T;
    E *o = out + 2 * (tid * NC * NC);
    if (mode == 1) {   // G = bc (B^dag + C)
        const int coord = mu == 0 ? c.x : mu == 1 ? c.y : mu == 2 ? c.z : c.t;
        const int ext = mu == 0 ? g.nx : mu == 1 ? g.ny : mu == 2 ? g.nz : g.nt;
        const int bcm = mu == 0 ? bc0 : mu == 1 ? bc1 : mu == 2 ? bc2 : bc3;
        const A ph = (coord == ext - 1) ? (A)bcm : (A)1;
        for (int a = 0; a < NC; ++a)
            for (int b = 0; b < NC; ++b) {
                cx<A> gv = conj(B[b][a]) + C[a][b];
                o[2 * (a * NC + b)] = from_acc<E, A>(ph * gv.re);
                o[2 * (a * NC + b) + 1] = from_acc<E, A>(ph * gv.im);
            }
        return;
    }
    // M = U B - C U^dag, U = phased link
    cx<A> Lk[NC][NC], M[NC][NC];
    load_mat_s<NC, E, A>(U + 2 * L::template mat<NC>(g, n, 4, mu), L::template mat_stride<NC>(g), Lk);
    for (int a = 0; a < NC; ++a)
        for (int b = 0; b < NC; ++b) {
            cx<A> acc = {0, 0};
            for (int k = 0; k < NC; ++k) {
                cmac(acc, Lk[a][k], B[k][b]);
                cmac(acc, C[a][k], cx<A>{-Lk[b][k].re, Lk[b][k].im});   // - C U^dag
            }
            M[a][b] = acc;
        }
    // P_TA(M) = (M - M^dag)/2 - tr(M - M^dag)/(2 Nc)
    A trim = 0;
    for (int a = 0; a < NC; ++a) trim += M[a][a].im;
    trim /= (A)NC;
    for (int a = 0; a < NC; ++a)
        for (int b = 0; b < NC; ++b) {
            cx<A> f = {(A)0.5 * (M[a][b].re - M[b][a].re), (A)0.5 * (M[a][b].im + M[b][a].im)};
            if (a == b) f.im -= trim;
            o[2 * (a * NC + b)] = from_acc<E, A>(f.re);
            o[2 * (a * NC + b) + 1] = from_acc<E, A>(f.im);
        }
}

template <int NC, int VR, typename E, int LAYOUT>
__global__ void __launch_bounds__(128, (NC == 3 && VR < 4 && sizeof(E) == 4 ? VR + 2 : 1)) force_kernel(const E *__restrict__ U, const E *__restrict__ psi,
                                                    const E *__restrict__ chi, E *__restrict__ out, Lat g, int bc0,
                                                    int bc1, int bc2, int bc3, int mode) {
    using L = Layout<LAYOUT>;
    using A = typename Acc<E>::T;
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (tid >= g.V * 4) return;
    const long long n = tid / 4;
    const int mu = (int)(tid % 4);
    const Coord c = site_coords(g, n);
    const long long m = neighbour(g, n, c, mu, +1);
    const long long csd = L::cs_stride(g);
    const long long on = 2 * L::vec(g, n, NC * 4, 0), om = 2 * L::vec(g, m, NC * 4, 0);
    cx<A> B[NC][NC], C[NC][NC];
    for (int a = 0; a < NC; ++a)
        for (int b = 0; b < NC; ++b) B[a][b] = C[a][b] = cx<A>{0, 0};
#pragma unroll 1
    for (int v = 0; v < g.nv; v += VR) {
        cx<A> x[NC][VR], y[NC][VR];
        // B: (1 - gamma) psi(n+mu), (1 - gamma) chi(n); C: (1 + gamma) psi(n), (1 + gamma) chi(n+mu)
        load_half<NC, VR, 0, E, A>(psi + om + 2 * v, csd, mu, true, x);
        load_half<NC, VR, 0, E, A>(chi + on + 2 * v, csd, mu, true, y);
        add_outer<NC, VR, A>(B, x, y);
        load_half<NC, VR, 1, E, A>(psi + om + 2 * v, csd, mu, true, x);
        load_half<NC, VR, 1, E, A>(chi + on + 2 * v, csd, mu, true, y);
        add_outer<NC, VR, A>(B, x, y);
        load_half<NC, VR, 0, E, A>(psi + on + 2 * v, csd, mu, false, x);
        load_half<NC, VR, 0, E, A>(chi + om + 2 * v, csd, mu, false, y);
        add_outer<NC, VR, A>(C, x, y);
        load_half<NC, VR, 1, E, A>(psi + on + 2 * v, csd, mu, false, x);
        load_half<NC, VR, 1, E, A>(chi + om + 2 * v, csd, mu, false, y);
        add_outer<NC, VR, A>(C, x, y);
    }
    force_out<NC, E, LAYOUT>(U, out, g, tid, n, mu, c, B, C, bc0, bc1, bc2, bc3, mode);
}

// D_W above N_c = 4, one thread per row a of a link's matrices: B and C of a
// whole link do not fit a thread's registers, and accumulators left to local
// memory are what the results must not hang on (with N_c^2 of them indexed in
// rolled loops the first 16 bytes of B were not zero at N_c = 7 and 8).  A row
// of both is 4 N_c reals and every index here is a compile-time one.  A thread
// loads its own colour of psi and chi; the colours of chi meet in shared
// memory, and so do the rows at the end: of B (for U B and B^dag), of U (for
// C U^dag), of M = U B - C U^dag.  Neighbouring threads take the colours of a site-outer
// vector, consecutive links of a site-inner one.  A thread per link before and
// now, us, 12^3x16, FP32, N_v = 4, site-inner: N_c = 5 78 and 66, 6 165 and 91, 7
// 325 and 112, 8 413 and 154 (every colour's chi read by every row: 135 at
// N_c = 5); 8^3x16, FP64, N_v = 2: 220 and 133, 345 and 197, 431 and 292, 592 and 401.
constexpr int kRowLinks = 32;   // links per block
template <int NC, int VR, typename E, int LAYOUT>
__global__ void __launch_bounds__(kRowLinks * NC, sizeof(E) == 4 ? 2 : 1)
    force_rows_kernel(const E *__restrict__ U, const E *__restrict__ psi, const E *__restrict__ chi,
                      E *__restrict__ out, Lat g, int bc0, int bc1, int bc2, int bc3, int mode) {
    using L = Layout<LAYOUT>;
    using A = typename Acc<E>::T;
    using Chi = cx<A>[4][NC][VR][kRowLinks + 1];   // the four projected components, [colour][RHS][link]
    using Rows = cx<A>[NC][NC][kRowLinks + 1];
    __shared__ __align__(16) unsigned char buf[2 * sizeof(Chi) > sizeof(Rows) ? 2 * sizeof(Chi) : sizeof(Rows)];
    Chi *ys = reinterpret_cast<Chi *>(buf);        // two, used in turn
    auto &rows = *reinterpret_cast<Rows *>(buf);   // a matrix per link
    const int l = LAYOUT == 0 ? threadIdx.x / NC : threadIdx.x % kRowLinks;
    const int a = LAYOUT == 0 ? threadIdx.x % NC : threadIdx.x / kRowLinks;
    const long long own = (long long)blockIdx.x * kRowLinks + l;
    const bool live = own < g.V * 4;
    const long long tid = live ? own : g.V * 4 - 1;
    const long long n = tid / 4;
    const int mu = (int)(tid % 4);
    const Coord c = site_coords(g, n);
    const long long m = neighbour(g, n, c, mu, +1);
    const long long csd = L::cs_stride(g);
    const long long oa = 2 * (a * 4) * csd;
    const long long on = 2 * L::vec(g, n, NC * 4, 0) + oa, om = 2 * L::vec(g, m, NC * 4, 0) + oa;
    cx<A> B[NC], C[NC];
#pragma unroll
    for (int b = 0; b < NC; ++b) B[b] = C[b] = cx<A>{0, 0};
#pragma unroll 1
    for (int v = 0, half = 0; v < g.nv; v += VR, half ^= 1) {
        // B: (1 - gamma) psi(n+mu), (1 - gamma) chi(n); C: (1 + gamma) psi(n), (1 + gamma) chi(n+mu)
        cx<A> x[4][1][VR], y[4][1][VR];
        load_half<1, VR, 0, E, A>(psi + om + 2 * v, csd, mu, true, x[0]);
        load_half<1, VR, 1, E, A>(psi + om + 2 * v, csd, mu, true, x[1]);
        load_half<1, VR, 0, E, A>(psi + on + 2 * v, csd, mu, false, x[2]);
        load_half<1, VR, 1, E, A>(psi + on + 2 * v, csd, mu, false, x[3]);
        load_half<1, VR, 0, E, A>(chi + on + 2 * v, csd, mu, true, y[0]);
        load_half<1, VR, 1, E, A>(chi + on + 2 * v, csd, mu, true, y[1]);
        load_half<1, VR, 0, E, A>(chi + om + 2 * v, csd, mu, false, y[2]);
        load_half<1, VR, 1, E, A>(chi + om + 2 * v, csd, mu, false, y[3]);
        Chi &yv = ys[half];
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int i = 0; i < VR; ++i) yv[k][a][i][l] = y[k][0][i];
        __syncthreads();   // also ends the reads of the other half, before the next trip writes to it
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int b = 0; b < NC; ++b)
#pragma unroll
                for (int i = 0; i < VR; ++i) cmac(k < 2 ? B[b] : C[b], x[k][0][i], conj(yv[k][b][i][l]));
    }
    auto exchange = [&](const cx<A> (&row)[NC]) {
        __syncthreads();   // what was there has been read
#pragma unroll
        for (int b = 0; b < NC; ++b) rows[a][b][l] = row[b];
        __syncthreads();
    };
    exchange(B);
    E *o = out + 2 * ((tid * NC + a) * NC);
    auto put = [&](int b, cx<A> f) {
        if (live) store_cx<E, 1, A>(o + 2 * b, &f);
    };
    if (mode == 1) {   // G = bc (B^dag + C)
        const int coord = mu == 0 ? c.x : mu == 1 ? c.y : mu == 2 ? c.z : c.t;
        const int ext = mu == 0 ? g.nx : mu == 1 ? g.ny : mu == 2 ? g.nz : g.nt;
        const int bcm = mu == 0 ? bc0 : mu == 1 ? bc1 : mu == 2 ? bc2 : bc3;
        const A ph = (coord == ext - 1) ? (A)bcm : (A)1;
#pragma unroll
        for (int b = 0; b < NC; ++b) put(b, ph * (conj(rows[b][a][l]) + C[b]));
        return;
    }
    // M = U B - C U^dag, row a; U the phased link
    const E *link = U + 2 * L::template mat<NC>(g, n, 4, mu) + 2 * L::template mat_stride<NC>(g) * (a * NC);
    cx<A> M[NC], u[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        u[k] = ld1<E, A>(link + 2 * L::template mat_stride<NC>(g) * k);
        M[k] = cx<A>{0, 0};
    }
#pragma unroll
    for (int k = 0; k < NC; ++k)
#pragma unroll
        for (int b = 0; b < NC; ++b) cmac(M[b], u[k], rows[k][b][l]);
    exchange(u);
#pragma unroll
    for (int k = 0; k < NC; ++k)
#pragma unroll
        for (int b = 0; b < NC; ++b) {
            const cx<A> w = rows[b][k][l];
            cmac(M[b], C[k], cx<A>{-w.re, w.im});
        }
    exchange(M);
    // P_TA(M) = (M - M^dag)/2 - tr(M - M^dag)/(2 Nc)
    A trim = 0;
#pragma unroll
    for (int b = 0; b < NC; ++b) trim += rows[b][b][l].im;
    trim /= (A)NC;
#pragma unroll
    for (int b = 0; b < NC; ++b) {
        const cx<A> t = rows[b][a][l];
        put(b, cx<A>{(A)0.5 * (M[b].re - t.re), (A)0.5 * (M[b].im + t.im) - (a == b ? trim : (A)0)});
    }
}

template <int NC, int VR, typename E, int LAYOUT>
__global__ void __launch_bounds__(128, (NC == 3 && sizeof(E) == 4 ? 3 : 1)) force_stag_kernel(const E *__restrict__ U, const E *__restrict__ psi,
                                                         const E *__restrict__ chi, E *__restrict__ out, Lat g,
                                                         int bc0, int bc1, int bc2, int bc3, int mode) {
    using L = Layout<LAYOUT>;
    using A = typename Acc<E>::T;
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (tid >= g.V * 4) return;
    const long long n = tid / 4;
    const int mu = (int)(tid % 4);
    const Coord c = site_coords(g, n);
    const long long m = neighbour(g, n, c, mu, +1);
    const long long csd = L::cs_stride(g);
    const long long on = 2 * L::vec(g, n, NC, 0), om = 2 * L::vec(g, m, NC, 0);
    // eta_mu(n) = (-1)^(sum_{nu<mu} (x_nu + 1)), the paper's 1-based convention
    const int e[4] = {0, c.x + 1, c.x + c.y + 2, c.x + c.y + c.z + 3};
    const A eta = (e[mu] & 1) ? (A)-1 : (A)1;
    cx<A> B[NC][NC], C[NC][NC];
    for (int a = 0; a < NC; ++a)
        for (int b = 0; b < NC; ++b) B[a][b] = C[a][b] = cx<A>{0, 0};
    if constexpr (NC <= kMaxNcSmall) {
        auto load = [&](const E *p, cx<A> (&x)[NC][VR]) {
#pragma unroll
            for (int a = 0; a < NC; ++a) load_cx<E, VR, A>(p + 2 * a * csd, x[a]);
        };
#pragma unroll 1
        for (int v = 0; v < g.nv; v += VR) {
            cx<A> x[NC][VR], y[NC][VR];
            load(psi + om + 2 * v, x);
            load(chi + on + 2 * v, y);
            add_outer<NC, VR, A>(B, x, y);
            load(psi + on + 2 * v, x);
            load(chi + om + 2 * v, y);
            add_outer<NC, VR, A>(C, x, y);
        }
    } else {
        for (int v = 0; v < g.nv; ++v) {
            cx<A> pn[NC], pm[NC], cn[NC], cm[NC];
            for (int a = 0; a < NC; ++a) {
                const long long on = 2 * (L::vec(g, n, NC, 0) + (long long)a * csd + v);
                const long long om = 2 * (L::vec(g, m, NC, 0) + (long long)a * csd + v);
                pn[a] = ld1<E, A>(psi + on);
                pm[a] = ld1<E, A>(psi + om);
                cn[a] = ld1<E, A>(chi + on);
                cm[a] = ld1<E, A>(chi + om);
            }
            for (int a = 0; a < NC; ++a)
                for (int b = 0; b < NC; ++b) {
                    cmac(B[a][b], pm[a], conj(cn[b]));
                    cmac(C[a][b], pn[a], conj(cm[b]));
                }
        }
    }
    for (int a = 0; a < NC; ++a)
        for (int b = 0; b < NC; ++b) {
            B[a][b] = (-eta) * B[a][b];
            C[a][b] = eta * C[a][b];
        }
    force_out<NC, E, LAYOUT>(U, out, g, tid, n, mu, c, B, C, bc0, bc1, bc2, bc3, mode);
}

template <int NC, int VR, typename E>
static int run_force(const dirac_op *op, const void *psi, const void *chi, void *force_out, int mode, cudaStream_t s) {
    return dispatch_layout(op->geom.layout, [&](auto lyc) {
        constexpr int LAYOUT = decltype(lyc)::value;
        const unsigned blocks = grid_for(op->V * 4, 128);
        const int *bc = op->geom.bc;
        const E *U = (const E *)op->links, *p = (const E *)psi, *c = (const E *)chi;
        if (op->kind == DIRAC_STAGGERED) {
            if constexpr (NC <= kMaxNcSmall || VR == 1)
                force_stag_kernel<NC, VR, E, LAYOUT>
                    <<<blocks, 128, 0, s>>>(U, p, c, (E *)force_out, op->lat, bc[0], bc[1], bc[2], bc[3], mode);
        } else if constexpr (NC <= kMaxNcSmall)
            force_kernel<NC, VR, E, LAYOUT>
                <<<blocks, 128, 0, s>>>(U, p, c, (E *)force_out, op->lat, bc[0], bc[1], bc[2], bc[3], mode);
        else
            force_rows_kernel<NC, VR, E, LAYOUT><<<grid_for(op->V * 4, kRowLinks), kRowLinks * NC, 0, s>>>(
                U, p, c, (E *)force_out, op->lat, bc[0], bc[1], bc[2], bc[3], mode);
        return launch_check(op->kind == DIRAC_STAGGERED ? "force_stag_kernel" : "force_kernel");
    });
}

}  // namespace dgb

using namespace dgb;

extern "C" int dirac_force(const dirac_op *op, const void *psi, const void *chi, void *force_out, int mode,
                           void *stream) {
    if (!op || !psi || !chi || !force_out) return DIRAC_ERR_INVALID_ARG;
    if ((op->kind != DIRAC_WILSON && op->kind != DIRAC_STAGGERED && op->kind != DIRAC_BRILLOUIN) ||
        (mode != 0 && mode != 1))
        return DIRAC_ERR_INVALID_ARG;
    if (op->clover) return DIRAC_ERR_INVALID_ARG;   // derived without the clover term
    if (((uintptr_t)psi & 15) || ((uintptr_t)chi & 15)) return DIRAC_ERR_ALIGNMENT;
    if (op->prec != DIRAC_F64 && op->prec != DIRAC_F32) return DIRAC_ERR_UNSUPPORTED_PREC;
    cudaStream_t s = (cudaStream_t)stream;
    // the handle owns the Brillouin force's scratch (allocated on first use)
    if (op->kind == DIRAC_BRILLOUIN) return launch_bril_force(const_cast<dirac_op *>(op), psi, chi, force_out, mode, s);
    // right-hand sides per load: 32 bytes where N_v and the vectors allow.  D_S
    // with fewer than eight: two trips of half the width overlap better (16^3x32,
    // N_v = 4, site-inner, N_c = 3: 48 us, one trip 54; N_c = 2: 22.7 and 20.6, so
    // not there).  D_W on site-inner vectors at N_c = 1, 2, where the loads of a
    // warp are whole lines anyway: one each up to N_v = 4 (25 and 57 us, four: 29
    // and 62; N_v = 8: 88 and 178, four: 52 and 99).
    const bool narrow = op->kind == DIRAC_WILSON && op->geom.layout == DIRAC_LAYOUT_SITE_INNER && op->nc <= 2 &&
                        op->nv <= 4 && op->prec == DIRAC_F32;
    int vr = narrow ? 1 : op->prec == DIRAC_F32 && (op->kind == DIRAC_WILSON || op->nv >= 8 || op->nc <= 2) ? 4 : 2;
    while (op->nv % vr) vr /= 2;
    vr = aligned_vr(vr, op->prec, psi, chi);
    if (op->nc > kMaxNcSmall) vr = op->kind == DIRAC_WILSON && op->prec == DIRAC_F32 && op->nv % 2 == 0 ? 2 : 1;
    return dispatch_prec(op->prec, [&](auto tag) {
        using E = std::remove_pointer_t<decltype(tag)>;
        if constexpr (sizeof(E) == 2) {
            return (int)DIRAC_ERR_UNSUPPORTED_PREC;
        } else {
            return dispatch_nc(op->nc, [&](auto ncc) {
                constexpr int NC = decltype(ncc)::value;
                if constexpr (NC <= kMaxNcSmall) {
                    if constexpr (sizeof(E) == 4)
                        if (vr == 4) return run_force<NC, 4, E>(op, psi, chi, force_out, mode, s);
                    if (vr == 2) return run_force<NC, 2, E>(op, psi, chi, force_out, mode, s);
                } else if constexpr (sizeof(E) == 4) {
                    if (vr == 2) return run_force<NC, 2, E>(op, psi, chi, force_out, mode, s);
                }
                return run_force<NC, 1, E>(op, psi, chi, force_out, mode, s);
            });
        }
    });
}

extern "C" int dirac_force_wilson(const dirac_op *op, const void *psi, const void *chi, void *force_out, int mode,
                                  void *stream) {
    if (op && op->kind != DIRAC_WILSON) return DIRAC_ERR_INVALID_ARG;
    return dirac_force(op, psi, chi, force_out, mode, stream);
}
