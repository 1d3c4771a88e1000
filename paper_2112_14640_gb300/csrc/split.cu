// split.cu -- FP64 applies on small lattices: the hops of one site and
// right-hand side spread over eight lanes.
//
// The FP64 pipe of this GPU takes about 64 cycles per warp instruction on each
// of its 608 quarter-SMs, so a stencil with fewer warps than that (thread <->
// site and RHS, 888 FP64 instructions for D_W at N_c = 3) takes the time of one
// warp however small the lattice.  Here eight lanes share the work of a thread:
// each applies one hop (80/8 offsets for the Brillouin kinds) with its
// direction's permutations and signs as selects on the integer pipe, the same
// instructions in every lane, and the sums are exchanged so that each lane ends
// with an eighth of the output components.  A sum is eight short ones.
// Plain and split, N_c = 3, us (back-to-back launches; about 9 of these are the
// launch): 4^4, N_v = 1: D_W 36 and 10, D_S 16 and 9, D_B 552 and 98, blap 429
// and 66; 6144 sites: D_W 36 and 17, D_S 17 and 11, D_B 553 and 273, blap 429
// and 179.
#include "bril_dirs.h"
#include "internal.h"

namespace dgb {

// Sites times RHS below which the lanes are split: half a warp of the plain
// kernel per quarter-SM.  At 12288 the two are even at N_c = 3 (D_W 37 and 27 us,
// D_S 17 and 17, D_B 558 and 538, bsuv 127 and 101) and N_c = 1 loses (D_B 107
// and 138); at 18432 D_S and D_B lose at N_c = 3 as well (17 and 23, 558 and 715).
constexpr long long kSplitItems = 608 * 16;

namespace split {

enum { WILSON = 0, STAGGERED = 1, LAP = 2, BRILLOUIN = 3, BLAP = 4 };

struct Offsets {
    signed char s[80][4];
};
__host__ __device__ constexpr Offsets make_offsets() {
    Offsets t{};
    for (int d = 0; d < 81; ++d) {
        const int s[4] = {d % 3 - 1, (d / 3) % 3 - 1, (d / 9) % 3 - 1, d / 27 - 1};
        if (d == 40) continue;
        double scale = 0;
        const int q = bril::store_index(s, &scale);
        for (int mu = 0; mu < 4; ++mu) t.s[q][mu] = (signed char)s[mu];
    }
    return t;
}
static __constant__ Offsets kOffsets = make_offsets();

__device__ __forceinline__ cx<double> sel(bool c, cx<double> a, cx<double> b) {
    return cx<double>{c ? a.re : b.re, c ? a.im : b.im};
}
// i a where c, else a
__device__ __forceinline__ cx<double> mul_i(bool c, cx<double> a) {
    return cx<double>{c ? flip(a.im, true) : a.re, c ? a.re : a.im};
}

// gamma_mu p, spin S, as in the chiral basis of App. A (mu a compile-time axis)
template <int S>
__device__ __forceinline__ void add_gammas(cx<double> &f, const cx<double> (&p)[4], const double (&e)[4]) {
    // gamma_1 p = (-i p3, -i p2, i p1, i p0); gamma_2 p = (-p3, p2, p1, -p0);
    // gamma_3 p = (-i p2, i p3, i p0, -i p1); gamma_4 p = (p2, p3, p0, p1)
    const cx<double> x = p[3 - S], z = p[S ^ 2];
    const double s1 = S <= 1 ? -e[0] : e[0], s2 = (S == 0 || S == 3) ? -e[1] : e[1], s3 = (S == 0 || S == 3) ? -e[2] : e[2];
    f.re = fma(-s1, x.im, f.re);
    f.im = fma(s1, x.re, f.im);
    f.re = fma(s2, x.re, f.re);
    f.im = fma(s2, x.im, f.im);
    f.re = fma(-s3, z.im, f.re);
    f.im = fma(s3, z.re, f.im);
    f.re = fma(e[3], z.re, f.re);
    f.im = fma(e[3], z.im, f.im);
}

// out = centre in + coef (the sum of the hops); M: the phased links, or W~
template <int KIND, int NC, int NS, int LAYOUT>
__global__ void __launch_bounds__(128) split_kernel(const double *__restrict__ M, const double *__restrict__ in,
                                                    double *__restrict__ out, Lat g, double centre, double coef,
                                                    int sgn) {
    using L = Layout<LAYOUT>;
    const long long items = g.nsites * g.nv;
    const long long item0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / 8;
    const int h = threadIdx.x % 8;
    const bool live = item0 < items;   // whole groups of eight lanes; they still exchange
    long long i;
    int v;
    split_tid(live ? item0 : items - 1, g.nv, i, v);
    const long long n = g.n0 + i;
    const Coord c = site_coords(g, n);
    const long long cs = L::cs_stride(g);
    cx<double> acc[NC][NS];
#pragma unroll
    for (int a = 0; a < NC; ++a)
#pragma unroll
        for (int s = 0; s < NS; ++s) acc[a][s] = cx<double>{0, 0};

    if constexpr (KIND <= LAP) {
        // lane h: direction h / 2, forward (even) or backward
        const int mu = h >> 1;
        const bool back = h & 1;
        const long long m = neighbour(g, n, c, mu, back ? -1 : +1);
        const double *link = M + 2 * link_index(back ? m : n, 4, NC * NC, mu, 0);
        constexpr long long ls = 2 * link_stride(NC * NC);
        const double *p = in + 2 * (L::vec(g, m, NC * NS, 0) + v);
        cx<double> Lk[NC][NC];   // the link, or its adjoint
#pragma unroll
        for (int a = 0; a < NC; ++a)
#pragma unroll
            for (int b = 0; b < NC; ++b) {
                const cx<double> u = ld1<double, double>(link + ls * (back ? b * NC + a : a * NC + b));
                Lk[a][b] = cx<double>{u.re, flip(u.im, back)};
            }
        if constexpr (KIND == WILSON) {
            // forward (1 - sgn gamma), backward (1 + sgn gamma)
            const bool minus = (sgn < 0) == back;   // a = -1
            const bool xy = mu < 2, im = !(mu & 1);
#pragma unroll
            for (int b = 0; b < NC; ++b) {
                cx<double> q[4];
#pragma unroll
                for (int s = 0; s < 4; ++s) q[s] = ld1<double, double>(p + 2 * (b * 4 + s) * cs);
                // h0 = p0 -+ a (i) p3 or p2, h1 = p1 -+ a (i) p2 or p3 (wilson.cuh, project)
                const cx<double> h0 = q[0] + flip(mul_i(im, sel(xy, q[3], q[2])), minus != (mu != 3));
                const cx<double> h1 = q[1] + flip(mul_i(im, sel(xy, q[2], q[3])), minus != (mu == 0));
#pragma unroll
                for (int a = 0; a < NC; ++a) {
                    cmac(acc[a][0], Lk[a][b], h0);
                    cmac(acc[a][1], Lk[a][b], h1);
                }
            }
            // the lower two spins from the upper two (wilson.cuh, reconstruct)
#pragma unroll
            for (int a = 0; a < NC; ++a) {
                acc[a][2] = flip(mul_i(im, sel(xy, acc[a][1], acc[a][0])), minus);
                acc[a][3] = flip(mul_i(im, sel(xy, acc[a][0], acc[a][1])), minus != (mu == 1 || mu == 2));
            }
        } else {
            bool neg = false;
            if constexpr (KIND == STAGGERED) {
                // eta_mu (forward), -eta_mu (backward)
                const int e = mu == 0 ? 0 : mu == 1 ? c.x + 1 : mu == 2 ? c.x + c.y + 2 : c.x + c.y + c.z + 3;
                neg = ((e & 1) != 0) != back;
            }
#pragma unroll
            for (int b = 0; b < NC; ++b)
#pragma unroll
                for (int s = 0; s < NS; ++s) {
                    const cx<double> q = flip(ld1<double, double>(p + 2 * (b * NS + s) * cs), neg);
#pragma unroll
                    for (int a = 0; a < NC; ++a) cmac(acc[a][s], Lk[a][b], q);
                }
        }
    } else {
        // lane h: offsets h, h + 8, ... of the site's 80
        const int co[4] = {c.x, c.y, c.z, c.t};
        const int ext[4] = {g.nx, g.ny, g.nz, g.nt};
        int dp[4], dm[4], stride = 1;
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) {
            dp[mu] = (co[mu] == ext[mu] - 1 ? -(ext[mu] - 1) : 1) * stride;
            dm[mu] = (co[mu] == 0 ? ext[mu] - 1 : -1) * stride;
            stride *= ext[mu];
        }
        const double *W = M + 2 * bril::w_index(0, 0, n, NC);
#pragma unroll 1
        for (int q = h; q < 80; q += 8) {
            double e[4];
            int m = (int)n, k = 0;
            double sl = 1;   // the sign of the highest axis
#pragma unroll
            for (int mu = 0; mu < 4; ++mu) {
                const int s = kOffsets.s[q][mu];
                m += s > 0 ? dp[mu] : s < 0 ? dm[mu] : 0;
                k += s != 0;
                e[mu] = s;
                if (s != 0) sl = s;
            }
            const double ck = (27.0 / 128.0) * (double)(1 << k);   // c_k = 27/64 2^(k-1)
            const double d = KIND == BLAP ? -ck * sl : -sgn * ck * sl;
#pragma unroll
            for (int mu = 0; mu < 4; ++mu) e[mu] = sl < 0 ? flip(e[mu], e[mu] != 0) : e[mu];
            const double *p = in + 2 * (L::vec(g, (long long)m, NC * NS, 0) + v);
#pragma unroll
            for (int b = 0; b < NC; ++b) {
                cx<double> f[NS];
                if constexpr (KIND == BLAP) {
#pragma unroll
                    for (int s = 0; s < NS; ++s) f[s] = d * ld1<double, double>(p + 2 * (b * NS + s) * cs);
                } else {
                    cx<double> r[4];
#pragma unroll
                    for (int s = 0; s < 4; ++s) r[s] = ld1<double, double>(p + 2 * (b * 4 + s) * cs);
                    f[0] = d * r[0];
                    f[1] = d * r[1];
                    f[2] = d * r[2];
                    f[3] = d * r[3];
                    add_gammas<0>(f[0], r, e);
                    add_gammas<1>(f[1], r, e);
                    add_gammas<2>(f[2], r, e);
                    add_gammas<3>(f[3], r, e);
                }
#pragma unroll
                for (int a = 0; a < NC; ++a) {
                    const cx<double> w = ld1<double, double>(W + 2 * ((q * NC + a) * NC + b));
#pragma unroll
                    for (int s = 0; s < NS; ++s) cmac(acc[a][s], w, f[s]);
                }
            }
        }
    }

    // Sum over the eight lanes.  The 2 NS N_c real numbers are halved between
    // partners while they divide, so each lane adds only what it keeps.
    double r[2 * NC * NS];
#pragma unroll
    for (int a = 0; a < NC; ++a)
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            r[2 * (a * NS + s)] = acc[a][s].re;
            r[2 * (a * NS + s) + 1] = acc[a][s].im;
        }
    constexpr int N0 = 2 * NC * NS;
    constexpr bool kHalve3 = N0 % 8 == 0;   // four spins; else only the first exchange halves
    int first = 0;
    auto halve = [&](auto lenc, int bit) {
        constexpr int H = decltype(lenc)::value;
        const bool up = h & bit;
#pragma unroll
        for (int k = 0; k < H; ++k) {
            const double give = up ? r[k] : r[k + H], keep = up ? r[k + H] : r[k];
            r[k] = keep + __shfl_xor_sync(~0u, give, bit);
        }
        first += up ? H : 0;
    };
    halve(std::integral_constant<int, N0 / 2>{}, 4);
    constexpr int LEN = kHalve3 ? N0 / 8 : N0 / 2;
    if constexpr (kHalve3) {
        halve(std::integral_constant<int, N0 / 4>{}, 2);
        halve(std::integral_constant<int, N0 / 8>{}, 1);
    } else {
#pragma unroll
        for (int bit = 2; bit > 0; bit /= 2)
#pragma unroll
            for (int k = 0; k < LEN; ++k) r[k] += __shfl_xor_sync(~0u, r[k], bit);
    }
    if (!live || (!kHalve3 && (h & 3))) return;
    const long long base = 2 * (L::vec(g, n, NC * NS, 0) + v);
#pragma unroll
    for (int k = 0; k < LEN; ++k) {
        const int e = first + k;   // real number e = 2 component + (re, im)
        const long long o = base + 2 * (long long)(e >> 1) * cs + (e & 1);
        out[o] = fma(coef, r[k], centre * __ldg(in + o));
    }
}

template <int KIND, int NC, int NS>
static int run(const dirac_op *op, const void *M, const void *in, void *out, double centre, double coef, int sgn,
               cudaStream_t s) {
    const long long threads = op->lat.nsites * op->nv * 8;
    return dispatch_layout(op->geom.layout, [&](auto lyc) {
        split_kernel<KIND, NC, NS, decltype(lyc)::value><<<grid_for(threads, 64), 64, 0, s>>>(
            (const double *)M, (const double *)in, (double *)out, op->lat, centre, coef, sgn);
        return launch_check("split_kernel");
    });
}

}  // namespace split

bool split_applies(const dirac_op *op) {
    // by the whole lattice, so that a part of it gives the same bits; a launch
    // variant chosen by the caller is one of the plain kernel
    return !op->vr && op->prec == DIRAC_F64 && op->nc <= kMaxNcSmall && !op->clover && op->V * op->nv < kSplitItems;
}

int launch_split(const dirac_op *op, const void *in, void *out, double m0, int sgn, cudaStream_t s) {
    using namespace split;
    return dispatch_nc<false>(op->nc, [&](auto ncc) {
        constexpr int NC = decltype(ncc)::value;
        switch (op->kind) {
        case DIRAC_WILSON: return run<WILSON, NC, 4>(op, op->links, in, out, 4.0 + m0, -0.5, sgn, s);
        case DIRAC_STAGGERED: return run<STAGGERED, NC, 1>(op, op->links, in, out, m0, 0.5 * sgn, sgn, s);
        case DIRAC_WLAP: return run<LAP, NC, 4>(op, op->links, in, out, 4.0 + 0.5 * m0 * m0, -0.5, sgn, s);
        case DIRAC_WSUV: return run<LAP, NC, 1>(op, op->links, in, out, 4.0 + 0.5 * m0 * m0, -0.5, sgn, s);
        case DIRAC_BRILLOUIN: return run<BRILLOUIN, NC, 4>(op, op->w, in, out, m0 + 240.0 / 128.0, sgn, sgn, s);
        case DIRAC_BLAP: return run<BLAP, NC, 4>(op, op->w, in, out, 0.5 * m0 * m0 + 240.0 / 128.0, 1.0, sgn, s);
        case DIRAC_BSUV: return run<BLAP, NC, 1>(op, op->w, in, out, 0.5 * m0 * m0 + 240.0 / 128.0, 1.0, sgn, s);
        }
        return (int)DIRAC_ERR_INVALID_ARG;
    });
}

}  // namespace dgb
