// links.cu -- gauge-field preparation done once per field:
//  * phase_links: the operator's own copy of U in its storage precision with
//    the boundary phase bc[mu] folded into U_mu(n) where n_mu = N_mu - 1;
//  * build_w: the 80 off-centre Brillouin links of Tab. off-axis,
//      W_s(n) = (1/k!) sum over the k! minimal paths n -> n+s of the ordered
//               products of signed links V_{+mu}(m) = U_mu(m), V_{-mu}(m) = U_mu(m-mu)^dag.
//    Grouping the paths by their last hop sigma gives the recursion
//      W_s(n) = (1/k) sum_{mu: s_mu != 0} W_{s - s_mu mu}(n) V_{s_mu mu}(n + s - s_mu mu),
//    evaluated level by level (k = 1..4) in shared memory, one thread block
//    per tile of sites, in FP64 for FP64 operators and FP32 otherwise; the
//    result is stored in the link precision;
//  * build_clover: the clover term of Eq. (def_clov) in the block form of
//    clover.cuh, from the clover-leaf field strength
//      F_mu,nu(n) = (Q_mu,nu(n) - Q_mu,nu(n)^dag) / (8i),
//    Q the sum of the four plaquettes of the (mu,nu) plane with a corner at
//    n, all traversed the same way (mu-step first, then nu-step);
//  * stout_smear: the fat links V the paper builds its operators and F
//    from (Sec. 2, App. F), steps of Morningstar-Peardon stout smearing.
#include "bril_dirs.h"
#include "hypercube.cuh"
#include "internal.h"
#include "linkalg.cuh"

namespace dgb {

struct Phases {
    int bc[4];
};


template <typename UE, typename E>
__global__ void phase_links_kernel(const UE *__restrict__ U, E *__restrict__ out, Lat g, Phases ph, int nc,
                                   int layout) {
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;   // (site, mu)
    if (tid >= g.V * 4) return;
    const long long n = tid / 4;
    const int mu = (int)(tid % 4);
    const Coord c = site_coords(g, n);
    const int coord = mu == 0 ? c.x : mu == 1 ? c.y : mu == 2 ? c.z : c.t;
    const int ext = mu == 0 ? g.nx : mu == 1 ? g.ny : mu == 2 ? g.nz : g.nt;
    const double f = (coord == ext - 1) ? (double)ph.bc[mu] : 1.0;
    const int per = nc * nc;
    for (int e = 0; e < per; ++e) {
        cx<double> u = ld_u(U, tid * per + e);
        // blocks of 32 sites, [mu][a][b][site % 32] within (common.cuh, link_index)
        const long long o = link_index(n, 4, per, mu, e);
        out[2 * o] = from_acc<E, double>(f * u.re);
        out[2 * o + 1] = from_acc<E, double>(f * u.im);
    }
}

// signed link V_{sign mu}(m) with boundary phase, in the arithmetic type AB
template <int NC, typename UE, typename AB>
__device__ __forceinline__ void signed_link(const UE *__restrict__ U, const Lat &g, const Phases &ph,
                                            const int x[4], int mu, int sign, cx<AB> (&L)[NC][NC]) {
    const int ext[4] = {g.nx, g.ny, g.nz, g.nt};
    int y[4] = {x[0], x[1], x[2], x[3]};
    if (sign < 0) y[mu] = (y[mu] == 0) ? ext[mu] - 1 : y[mu] - 1;
    const long long site = (((long long)y[3] * g.nz + y[2]) * g.ny + y[1]) * g.nx + y[0];
    const double f = (y[mu] == ext[mu] - 1) ? (double)ph.bc[mu] : 1.0;
    const long long base = (site * 4 + mu) * NC * NC;
#pragma unroll
    for (int a = 0; a < NC; ++a)
#pragma unroll
        for (int b = 0; b < NC; ++b) {
            cx<double> u = ld_u(U, base + (sign > 0 ? a * NC + b : b * NC + a));
            L[a][b] = sign > 0 ? cx<AB>{(AB)(f * u.re), (AB)(f * u.im)} : cx<AB>{(AB)(f * u.re), (AB)(-f * u.im)};
        }
}

// The caller's links [site][mu][a][b] with the boundary phase, in the
// arithmetic type AB: the source of W for 16-bit link storage, whose own
// links are already rounded (hyper::NativeLinks reads those of FP64 and FP32).
template <int NC, typename UE, typename AB>
struct CallerLinks {
    const UE *U;
    Lat g;
    Phases ph;
    __device__ __forceinline__ AB phase(long long site, int mu) const {
        const Coord c = site_coords(g, site);
        const int co = mu == 0 ? c.x : mu == 1 ? c.y : mu == 2 ? c.z : c.t;
        const int ext = mu == 0 ? g.nx : mu == 1 ? g.ny : mu == 2 ? g.nz : g.nt;
        const int bc = mu == 0 ? ph.bc[0] : mu == 1 ? ph.bc[1] : mu == 2 ? ph.bc[2] : ph.bc[3];
        return co == ext - 1 ? (AB)bc : (AB)1;
    }
    __device__ __forceinline__ cx<AB> at(long long site, int mu, bool dag, int a, int b) const {
        const cx<double> u = ld_u(U, (site * 4 + mu) * NC * NC + (dag ? b * NC + a : a * NC + b));
        const AB f = phase(site, mu);   // +-1: exact after the conversion
        return cx<AB>{f * (AB)u.re, f * (AB)(dag ? -u.im : u.im)};
    }
    __device__ __forceinline__ void load(long long site, int mu, bool dag, cx<AB> (&L)[NC][NC]) const {
        const AB f = phase(site, mu);
#pragma unroll
        for (int a = 0; a < NC; ++a)
#pragma unroll
            for (int b = 0; b < NC; ++b) {
                const cx<double> u = ld_u(U, (site * 4 + mu) * NC * NC + (dag ? b * NC + a : a * NC + b));
                L[a][b] = cx<AB>{f * (AB)u.re, f * (AB)(dag ? -u.im : u.im)};
            }
    }
};

// W in FP64 for FP64 links, in FP32 otherwise (FP32 links carry 24 bits; the
// four levels add a few FP32 roundings, and FP64 arithmetic is slow here).
template <typename E>
using WArith = std::conditional_t<sizeof(E) == 8, double, float>;

// The scale rho_k s_lead on a value of the builder's arithmetic type.  FP32:
// the scale as a sum of two floats, so that the product carries one rounding
// only, as it would from FP64, without the (slow) FP64 multiply.
struct WScale {
    float hi, lo;
};
__host__ __device__ constexpr WScale w_scale(double v) {
    const float hi = (float)v;
    return WScale{hi, (float)(v - (double)hi)};
}
__device__ __forceinline__ float scaled(float w, WScale s) { return __fmaf_rn(s.hi, w, __fmul_rn(s.lo, w)); }

// store two consecutive complex numbers
template <typename E, typename AB>
__device__ __forceinline__ void store_pair(E *p, cx<AB> a, cx<AB> b) {
    const cx<AB> v[2] = {a, b};
    if constexpr (sizeof(E) <= 4) {
        store_cx<E, 2, AB>(p, v);
    } else {
        store_cx<E, 1, AB>(p, v);
        store_cx<E, 1, AB>(p + 2, v + 1);
    }
}

// Level recursion W_s(n) = (1/k) sum_mu W_{s - s_mu mu}(n) V_{s_mu mu}(n + s - s_mu mu)
// on a tile of S sites per block (hypercube.cuh).  Bound by the L1 / shared
// memory pipe (216 products per site, each one link and one W operand) and by
// writing W.  With one block per site and one thread per offset, every link
// load touched as many cache lines as the warp has lanes and the FP64 phase
// multiply and conversion of each element ran on the slow FP64 pipe: 4.96 ms
// at 16^3x32, N_c = 3, FP32 from FP64 links, against 0.37 ms now (writing the
// 755 MB of W takes 0.11 ms).  Lanes over consecutive sites make the link
// loads contiguous, and the operator's own phased links need no conversion.
template <int NC, typename E>
struct WTile {
    using AB = WArith<E>;
    static constexpr int S = hyper::tile_sites(80, NC, sizeof(cx<AB>), true);
    static constexpr int PAD = hyper::tile_pad(S);   // the transposed read of the output phase is conflict-free
    static constexpr int R = 80 * NC * NC;           // rows of the tile: element e of W_q at q N_c^2 + e
    static constexpr size_t smem = (size_t)R * PAD * sizeof(cx<AB>);
};

template <int NC, typename E, typename SRC>
__global__ void __launch_bounds__(hyper::kThreads, 2) build_w_kernel(SRC src, E *__restrict__ W, Lat g) {
    using AB = WArith<E>;
    using T = WTile<NC, E>;
    extern __shared__ __align__(16) unsigned char w_smem[];
    __shared__ WScale scale[80];
    __shared__ double scale_d[sizeof(AB) == 8 ? 80 : 1];
    cx<AB> *Ws = reinterpret_cast<cx<AB> *>(w_smem);
    const long long n0 = (long long)blockIdx.x * T::S;
    const int lane = threadIdx.x % T::S, worker = threadIdx.x / T::S;
    // lanes past the last site repeat it; they store nothing below
    const long long n = n0 + lane < g.V ? n0 + lane : g.V - 1;
    const hyper::Steps st = hyper::steps_at(g, n);
    if (threadIdx.x < 80) {
        const hyper::Offset &o = hyper::kTable.o[threadIdx.x];
        const double v = bril::rho(o.k) * (double)o.s[o.mu[o.k - 1]];   // the lead axis is the highest
        scale[o.q] = w_scale(v);
        if constexpr (sizeof(AB) == 8) scale_d[o.q] = v;
    }
    constexpr int NW = hyper::kThreads / T::S;
    auto row = [](int pos) { return (int)hyper::kTable.o[pos].q; };
    hyper::w_level<1, NC, T::PAD, NW>(Ws, src, n, st, lane, worker, row);
    hyper::w_level<2, NC, T::PAD, NW>(Ws, src, n, st, lane, worker, row);
    hyper::w_level<3, NC, T::PAD, NW>(Ws, src, n, st, lane, worker, row);
    hyper::w_level<4, NC, T::PAD, NW>(Ws, src, n, st, lane, worker, row);
    // stored as rho_k s_lead W_s, [site][q][a][b] (bril_dirs.h): a site's rows
    // are contiguous, two complex numbers per store (80 N_c^2 is even)
    constexpr int H = T::R / 2;
    for (int p = threadIdx.x; p < T::S * H; p += hyper::kThreads) {
        const int site = p / H, r = 2 * (p - site * H);
        if (n0 + site >= g.V) break;
        cx<AB> v[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const cx<AB> w = Ws[(r + i) * T::PAD + site];
            const int q = (r + i) / (NC * NC);
            if constexpr (sizeof(AB) == 8) v[i] = scale_d[q] * w;
            else v[i] = cx<AB>{scaled(w.re, scale[q]), scaled(w.im, scale[q])};
        }
        store_pair<E, AB>(W + 2 * ((n0 + site) * T::R + r), v[0], v[1]);
    }
}

// The stored W~ back to W_s in the public order d = (st+1)*27 + (sz+1)*9 +
// (sy+1)*3 + (sx+1), centre left out, in the operator's layout and link precision.
template <typename E>
__global__ void unpack_w_kernel(const E *__restrict__ Wst, E *__restrict__ out, Lat g, int nc, int layout) {
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;   // (site, dirp)
    if (tid >= g.V * 80) return;
    const long long n = tid / 80;
    const int dirp = (int)(tid % 80);
    const int dir = dirp < 40 ? dirp : dirp + 1;
    const int s[4] = {dir % 3 - 1, (dir / 3) % 3 - 1, (dir / 9) % 3 - 1, dir / 27 - 1};
    double scale;
    const int q = bril::store_index(s, &scale);
    const int per = nc * nc;
    for (int e = 0; e < per; ++e) {
        const long long i = bril::w_index(q, e, n, nc);
        const long long o = layout == 0 ? (n * 80 + dirp) * per + e : ((long long)dirp * per + e) * g.V + n;
        using A = typename Acc<E>::T;
        out[2 * o] = from_acc<E, double>((double)to_acc<E>(Wst[2 * i]) / scale);
        out[2 * o + 1] = from_acc<E, double>((double)to_acc<E>(Wst[2 * i + 1]) / scale);
    }
}

int launch_unpack_w(const dirac_op *op, void *out, cudaStream_t s) {
    return dispatch_prec(link_prec(op), [&](auto tag) {
        using E = std::remove_pointer_t<decltype(tag)>;
        const long long threads = op->V * 80;
        unpack_w_kernel<E><<<grid_for(threads, 128), 128, 0, s>>>((const E *)op->w, (E *)out, op->lat, op->nc,
                                                                  op->geom.layout);
        return launch_check("unpack_w_kernel");
    });
}


static Phases phases_of(const dirac_op *op) {
    Phases ph;
    for (int m = 0; m < 4; ++m) ph.bc[m] = op->geom.bc[m];
    return ph;
}

int launch_phase_links(dirac_op *op, const void *U, dirac_prec u_prec, cudaStream_t s) {
    return dispatch_uprec(u_prec, [&](auto utag) {
        using UE = std::remove_pointer_t<decltype(utag)>;
        return dispatch_prec(link_prec(op), [&](auto tag) {
            using E = std::remove_pointer_t<decltype(tag)>;
            const long long threads = op->V * 4;
            phase_links_kernel<UE, E><<<grid_for(threads, 128), 128, 0, s>>>((const UE *)U, (E *)op->links,
                                                                            op->lat, phases_of(op), op->nc,
                                                                            op->geom.layout);
            return launch_check("phase_links_kernel");
        });
    });
}

template <int NC, typename E, typename SRC>
static int run_build_w(const dirac_op *op, const SRC &src, cudaStream_t s) {
    using T = WTile<NC, E>;
    if constexpr (T::smem > 48 * 1024) {
        const int rc = cuda_check(cudaFuncSetAttribute(build_w_kernel<NC, E, SRC>,
                                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)T::smem),
                                  "build_w_kernel shared memory");
        if (rc) return rc;
    }
    build_w_kernel<NC, E, SRC><<<grid_for(op->V, T::S), hyper::kThreads, T::smem, s>>>(src, (E *)op->w, op->lat);
    return launch_check("build_w_kernel");
}

// W from the operator's phased links (already written by launch_phase_links on
// the same stream) for FP64 and FP32 links, from the caller's field for 16-bit ones.
int launch_build_w(dirac_op *op, const void *U, dirac_prec u_prec, cudaStream_t s) {
    return dispatch_prec(link_prec(op), [&](auto tag) {
        using E = std::remove_pointer_t<decltype(tag)>;
        return dispatch_nc<big_nc_ok<E>()>(op->nc, [&](auto ncc) {
            constexpr int NC = decltype(ncc)::value;
            if constexpr (sizeof(E) >= 4) {
                return run_build_w<NC, E>(op, hyper::NativeLinks<NC, E, WArith<E>>{(const E *)op->links}, s);
            } else {
                return dispatch_uprec(u_prec, [&](auto utag) {
                    using UE = std::remove_pointer_t<decltype(utag)>;
                    return run_build_w<NC, E>(
                        op, CallerLinks<NC, UE, WArith<E>>{(const UE *)U, op->lat, phases_of(op)}, s);
                });
            }
        });
    });
}

// ------------------------------------------------------------ clover term


// F_mu,nu at site x0 from the four leaves (+mu,+nu), (+nu,-mu), (-mu,-nu),
// (-nu,+mu); the leaf (a, b) is V_a(n) V_b(n+a) V_-a(n+a+b) V_-b(n+b).
template <int NC, typename UE, typename AB>
__device__ void field_strength(const UE *__restrict__ U, const Lat &g, const Phases &ph, const int x0[4], int mu,
                               int nu, cx<AB> (&F)[NC][NC]) {
    const int ext[4] = {g.nx, g.ny, g.nz, g.nt};
    const int st[4][4] = {{mu, 1, nu, 1}, {nu, 1, mu, -1}, {mu, -1, nu, -1}, {nu, -1, mu, 1}};
    cx<AB> Q[NC][NC];
#pragma unroll
    for (int a = 0; a < NC; ++a)
#pragma unroll
        for (int b = 0; b < NC; ++b) Q[a][b] = cx<AB>{0, 0};
    for (int l = 0; l < 4; ++l) {
        const int am = st[l][0], as = st[l][1], bm = st[l][2], bs = st[l][3];
        int xa[4] = {x0[0], x0[1], x0[2], x0[3]};
        step(xa, ext, am, as);
        int xab[4] = {xa[0], xa[1], xa[2], xa[3]};
        step(xab, ext, bm, bs);
        int xb[4] = {x0[0], x0[1], x0[2], x0[3]};
        step(xb, ext, bm, bs);
        cx<AB> P[NC][NC], L[NC][NC], T[NC][NC];
        signed_link<NC, UE, AB>(U, g, ph, x0, am, as, P);
        signed_link<NC, UE, AB>(U, g, ph, xa, bm, bs, L);
        mat_mul<NC, AB>(P, L, T);
        signed_link<NC, UE, AB>(U, g, ph, xab, am, -as, L);
        mat_mul<NC, AB>(T, L, P);
        signed_link<NC, UE, AB>(U, g, ph, xb, bm, -bs, L);
        mat_mul<NC, AB>(P, L, T);
#pragma unroll
        for (int a = 0; a < NC; ++a)
#pragma unroll
            for (int b = 0; b < NC; ++b) Q[a][b] = Q[a][b] + T[a][b];
    }
    // (Q - Q^dag) / (8i) = -i (Q - Q^dag) / 8
#pragma unroll
    for (int a = 0; a < NC; ++a)
#pragma unroll
        for (int b = 0; b < NC; ++b) {
            const cx<AB> d = {Q[a][b].re - Q[b][a].re, Q[a][b].im + Q[b][a].im};
            F[a][b] = cx<AB>{d.im / (AB)8, -d.re / (AB)8};
        }
}

// One thread per (site, block k = 2 chi + w): block A (w = 0) of chirality chi
// needs the planes (1,2), (3,4); block B (w = 1) the planes (1,4), (2,3),
// (1,3), (2,4) (clover.cuh).  FP64 arithmetic for FP64 storage, FP32 otherwise.
template <int NC, typename UE, typename E>
__global__ void __launch_bounds__(128) build_clover_kernel(const UE *__restrict__ U, E *__restrict__ out, Lat g,
                                                           Phases ph, double csw, int layout) {
    using AB = std::conditional_t<sizeof(E) == 8, double, float>;
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (tid >= g.V * 4) return;
    const long long n = tid / 4;
    const int k = (int)(tid % 4), chi = k >> 1, w = k & 1;
    const AB e = chi == 0 ? (AB)1 : (AB)-1;
    const Coord c = site_coords(g, n);
    const int x0[4] = {c.x, c.y, c.z, c.t};
    // (plane, complex coefficient) pairs of the block, planes as (mu, nu) 0-based
    int planes[4][2];
    cx<AB> coef[4];
    int np;
    if (w == 0) {   // -F_12 + e F_34
        np = 2;
        planes[0][0] = 0, planes[0][1] = 1, coef[0] = cx<AB>{-1, 0};
        planes[1][0] = 2, planes[1][1] = 3, coef[1] = cx<AB>{e, 0};
    } else {        // e F_14 - F_23 - i F_13 - i e F_24
        np = 4;
        planes[0][0] = 0, planes[0][1] = 3, coef[0] = cx<AB>{e, 0};
        planes[1][0] = 1, planes[1][1] = 2, coef[1] = cx<AB>{-1, 0};
        planes[2][0] = 0, planes[2][1] = 2, coef[2] = cx<AB>{0, -1};
        planes[3][0] = 1, planes[3][1] = 3, coef[3] = cx<AB>{0, -e};
    }
    cx<AB> acc[NC][NC];
#pragma unroll
    for (int a = 0; a < NC; ++a)
#pragma unroll
        for (int b = 0; b < NC; ++b) acc[a][b] = cx<AB>{0, 0};
    for (int i = 0; i < np; ++i) {
        cx<AB> F[NC][NC];
        field_strength<NC, UE, AB>(U, g, ph, x0, planes[i][0], planes[i][1], F);
#pragma unroll
        for (int a = 0; a < NC; ++a)
#pragma unroll
            for (int b = 0; b < NC; ++b) cmac(acc[a][b], coef[i], F[a][b]);
    }
    const double f = -0.5 * csw;
    const int per = NC * NC;
#pragma unroll
    for (int a = 0; a < NC; ++a)
#pragma unroll
        for (int b = 0; b < NC; ++b) {
            const int el = a * NC + b;
            // the links' layout (common.cuh, link_index)
            const long long o = link_index(n, 4, per, k, el);
            out[2 * o] = from_acc<E, double>(f * (double)acc[a][b].re);
            out[2 * o + 1] = from_acc<E, double>(f * (double)acc[a][b].im);
        }
}

int launch_build_clover(dirac_op *op, const void *V, dirac_prec v_prec, cudaStream_t s) {
    return dispatch_uprec(v_prec, [&](auto utag) {
        using UE = std::remove_pointer_t<decltype(utag)>;
        return dispatch_prec(link_prec(op), [&](auto tag) {
            using E = std::remove_pointer_t<decltype(tag)>;
            return dispatch_nc<big_nc_ok<E>()>(op->nc, [&](auto ncc) {
                constexpr int NC = decltype(ncc)::value;
                const long long threads = op->V * 4;
                // closed loops do not see the boundary phases: leave them out
                Phases none;
                for (int m = 0; m < 4; ++m) none.bc[m] = 1;
                build_clover_kernel<NC, UE, E><<<grid_for(threads, 128), 128, 0, s>>>(
                    (const UE *)V, (E *)op->clover, op->lat, none, op->csw, op->geom.layout);
                return launch_check("build_clover_kernel");
            });
        });
    });
}

template <typename S, typename D>
__global__ void convert_scalars_kernel(const S *__restrict__ src, D *__restrict__ dst, long long count) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) dst[i] = from_acc<D, typename Acc<S>::T>(to_acc<S>(src[i]));
}

static int convert_array(const void *src, dirac_prec sp, void *dst, dirac_prec dp, long long count, cudaStream_t s) {
    return dispatch_prec(sp, [&](auto stag) {
        using S = std::remove_pointer_t<decltype(stag)>;
        return dispatch_prec(dp, [&](auto dtag) {
            using D = std::remove_pointer_t<decltype(dtag)>;
            convert_scalars_kernel<S, D><<<grid_for(count, 256), 256, 0, s>>>((const S *)src, (D *)dst, count);
            return launch_check("convert_scalars_kernel");
        });
    });
}

int launch_convert_links(const dirac_op *src, dirac_op *dst, cudaStream_t s) {
    long long n = link_sites(src->V) * 4 * src->nc * src->nc * 2;
    int rc = convert_array(src->links, link_prec(src), dst->links, link_prec(dst), n, s);
    if (rc) return rc;
    if (src->w) {
        // same order, scale and layout, element by element
        n = src->V * 80 * src->nc * src->nc * 2;
        rc = convert_array(src->w, link_prec(src), dst->w, link_prec(dst), n, s);
    }
    if (!rc && src->clover) {
        n = link_sites(src->V) * 4 * src->nc * src->nc * 2;
        rc = convert_array(src->clover, link_prec(src), dst->clover, link_prec(dst), n, s);
    }
    return rc;
}

}  // namespace dgb
