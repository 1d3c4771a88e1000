// force_bril.cu -- link derivative of the pseudofermion action for the
// Brillouin operator (the paper has no force; derived here):
//   S = sum_v Re phi_v^dag (D_B^dag D_B)^-1 phi_v,  psi = (D^dag D)^-1 phi,  chi = D_B psi.
// From Eq. (app_bril), dS = -2 Re <chi, dD psi> and
//   dD psi(n) = sum_s S_s (x) dW_s(n) psi(n+s),  S_s = rho_k sum_mu s_mu gamma_mu - lambda_k/2,
// so dS = Re sum_{n,s} tr[dW_s(n) G_s(n)] with G_s = -2 M_s,
//   M_s(n) = sum_{v, spin} (S_s psi(n+s)) chi(n)^dag        (an N_c x N_c matrix).
// W_s is the average of the k! hop orderings of Tab. off-axis; built level by
// level it obeys W_s(n) = (1/k) sum_{mu in supp s} W_{s - s_mu mu}(n) V_{s_mu mu}(n + s - s_mu mu)
// (grouping the orderings by their last hop), and the adjoint of that
// recursion carries G down the levels:
//   G_{s - s_mu mu} += (1/k) V G_s          (at the same site n),
//   link term  tr[dV X],  X = (1/k) G_s W_{s - s_mu mu},
// where V = U_mu(m) receives K_mu(m) += X and V = U_mu(m - mu)^dag receives
// K_mu(m - mu) += X^dag (m = n + s - s_mu mu), with dS = Re sum tr[dU K].
//
// N_c <= 4 (launch_tiled): the sites of a tile lie on neighbouring lanes
// (hypercube.cuh) and the scratch is stored tile by tile, [tile][slot][e][site]:
//   1. psi and chi are copied to [component][RHS][site] order within each tile;
//   2. M_s for the three offsets of one (y, z, t) row at a time, one lane per
//      site, the spin mix done once on chi(n) and shared by the row;
//   3. W by the level recursion, then G level by level from k = 4 down to 1,
//      each level gathering from the level above (no atomics: deterministic);
//      every (s, mu) link term X goes to a scratch slot;
//   4. K_mu(m) gathers the 54 slots that land on the link -- 27 offsets enter
//      it forward, 27 backward -- and writes F = P_TA(U K) or G = bc K^dag
//      (force_out of force.cu with C = 0).
// 16^3x32, N_c = 3, N_v = 4, FP32: 1.84 ms, against 6.86 ms for one block per
// site.  There every psi, chi and link load of a warp touched one cache line
// per lane and chi was spin-mixed anew for every offset; what remains is the
// FP32 work of steps 2 and 3 (about 140 k multiply-adds per site) and writing
// and reading the 216 link terms (2 GB each way).
// Larger N_c (bril_force_site_kernel, bril_force_link_kernel): one block per
// site and one thread per offset for steps 2 and 3, whose N_c x N_c matrices
// do not fit a tile's registers and shared memory.
// Arithmetic in FP64 for FP64 operators and FP32 otherwise, like the W builder.
#include "bril_dirs.h"
#include "hypercube.cuh"
#include "internal.h"
#include "linkalg.cuh"

namespace dgb {

namespace bforce {

__host__ __device__ constexpr int kk(int d) {
    return (d % 3 != 1) + ((d / 3) % 3 != 1) + ((d / 9) % 3 != 1) + (d / 27 != 1);
}
__host__ __device__ constexpr int comp(int d, int mu) {   // s_mu of offset index d
    return mu == 0 ? d % 3 - 1 : mu == 1 ? (d / 3) % 3 - 1 : mu == 2 ? (d / 9) % 3 - 1 : d / 27 - 1;
}
// first scratch slot of offset d: the slots of (d, mu) for mu in supp(s_d), increasing mu
__host__ __device__ constexpr int slot_base(int d) {
    int o = 0;
    for (int j = 0; j < d; ++j) o += kk(j);
    return o;
}
constexpr int kSlots = 216;   // sum over offsets of their hop count
// slot of the link term (d, mu), -1 where offset d does not move along mu:
// a table in constant memory, built at compile time (computing it per call
// took an O(d) loop of integer divisions, which made both force kernels
// integer-bound)
struct SlotTable {
    short slot[81][4];
};
__host__ __device__ constexpr SlotTable make_slot_table() {
    SlotTable t{};
    for (int d = 0; d < 81; ++d) {
        int o = slot_base(d);
        for (int mu = 0; mu < 4; ++mu) t.slot[d][mu] = comp(d, mu) != 0 ? (short)o++ : (short)-1;
    }
    return t;
}
static __constant__ SlotTable kSlotTable = make_slot_table();
__device__ __forceinline__ int slot_of(int d, int mu) { return kSlotTable.slot[d][mu]; }
// x + off on a periodic axis of extent ext, off in {-1, 0, 1}
__device__ __forceinline__ int wrap(int x, int ext) { return x < 0 ? x + ext : (x >= ext ? x - ext : x); }
constexpr int pow3(int mu) { return mu == 0 ? 1 : mu == 1 ? 3 : mu == 2 ? 9 : 27; }

template <int NC, typename E>
using Arith = std::conditional_t<sizeof(E) == 8, double, float>;
template <int NC, typename E>
constexpr size_t site_smem() { return 2 * sizeof(cx<Arith<NC, E>>) * 81 * NC * NC; }

// V_{sign mu}(x) from the operator's phased links: U_mu(x) or U_mu(x - mu)^dag
template <int NC, typename E, typename AB>
__device__ __forceinline__ void hop_link(const E *__restrict__ U, const Lat &g, const int x[4], int mu, int sign,
                                         cx<AB> (&L)[NC][NC]) {
    int y[4] = {x[0], x[1], x[2], x[3]};
    const int ext[4] = {g.nx, g.ny, g.nz, g.nt};
    if (sign < 0) y[mu] = (y[mu] == 0) ? ext[mu] - 1 : y[mu] - 1;
    const long long site = (((long long)y[3] * g.nz + y[2]) * g.ny + y[1]) * g.nx + y[0];
    const E *p = U + 2 * Layout<0>::template mat<NC>(g, site, 4, mu);
    const long long ls = Layout<0>::template mat_stride<NC>(g);
#pragma unroll
    for (int a = 0; a < NC; ++a)
#pragma unroll
        for (int b = 0; b < NC; ++b) {
            const cx<AB> u = ld1<E, AB>(p + 2 * ls * (sign > 0 ? a * NC + b : b * NC + a));
            L[a][b] = sign > 0 ? u : cx<AB>{u.re, -u.im};
        }
}

// (S_s psi)_sigma for one colour and RHS: rho_k sum_mu s_mu (gamma_mu p)_sigma - lambda_k/2 p_sigma,
// gammas of App. A in the chiral basis (the same signed permutations as the stencil)
template <typename A>
__device__ __forceinline__ cx<A> gamma_comp(int mu, int sg, const cx<A> p[4]) {
    // gamma_1 psi = (-i p3, -i p2, i p1, i p0); gamma_2 psi = (-p3, p2, p1, -p0);
    // gamma_3 psi = (-i p2, i p3, i p0, -i p1); gamma_4 psi = (p2, p3, p0, p1)
    switch (mu) {
    case 0: {
        const cx<A> v = p[3 - sg];
        return sg <= 1 ? cx<A>{v.im, -v.re} : cx<A>{-v.im, v.re};
    }
    case 1: {
        const cx<A> v = p[3 - sg];
        return (sg == 0 || sg == 3) ? cx<A>{-v.re, -v.im} : v;
    }
    case 2: {
        const cx<A> v = p[sg ^ 2];
        return (sg == 0 || sg == 3) ? cx<A>{v.im, -v.re} : cx<A>{-v.im, v.re};
    }
    default:
        return p[sg ^ 2];
    }
}

}  // namespace bforce

// F = P_TA(U K) (mode 0, U the phased link) or G = bc K^dag (mode 1, for the
// caller's unphased links) of link (m, mu).
template <int NC, typename E, typename A>
__device__ __forceinline__ void link_output(const E *__restrict__ U, E *__restrict__ o, const Lat &g, long long m,
                                            int mu, const Coord &c, const cx<A> (&K)[NC][NC], int bc0, int bc1, int bc2,
                                            int bc3, int mode) {
    if (mode == 1) {
        const int coord = mu == 0 ? c.x : mu == 1 ? c.y : mu == 2 ? c.z : c.t;
        const int ext = mu == 0 ? g.nx : mu == 1 ? g.ny : mu == 2 ? g.nz : g.nt;
        const int bcm = mu == 0 ? bc0 : mu == 1 ? bc1 : mu == 2 ? bc2 : bc3;
        const A ph = (coord == ext - 1) ? (A)bcm : (A)1;
#pragma unroll
        for (int a = 0; a < NC; ++a)
#pragma unroll
            for (int b = 0; b < NC; ++b) {
                o[2 * (a * NC + b)] = from_acc<E, A>(ph * K[b][a].re);
                o[2 * (a * NC + b) + 1] = from_acc<E, A>(-ph * K[b][a].im);
            }
        return;
    }
    cx<A> Lk[NC][NC], M[NC][NC];
    load_mat_s<NC, E, A>(U + 2 * Layout<0>::template mat<NC>(g, m, 4, mu), Layout<0>::template mat_stride<NC>(g), Lk);
#pragma unroll
    for (int a = 0; a < NC; ++a)
#pragma unroll
        for (int b = 0; b < NC; ++b) {
            cx<A> acc = {0, 0};
#pragma unroll
            for (int q = 0; q < NC; ++q) cmac(acc, Lk[a][q], K[q][b]);
            M[a][b] = acc;
        }
    A trim = 0;
#pragma unroll
    for (int a = 0; a < NC; ++a) trim += M[a][a].im;
    trim /= (A)NC;
#pragma unroll
    for (int a = 0; a < NC; ++a)
#pragma unroll
        for (int b = 0; b < NC; ++b) {
            cx<A> f = {(A)0.5 * (M[a][b].re - M[b][a].re), (A)0.5 * (M[a][b].im + M[b][a].im)};
            if (a == b) f.im -= trim;
            o[2 * (a * NC + b)] = from_acc<E, A>(f.re);
            o[2 * (a * NC + b) + 1] = from_acc<E, A>(f.im);
        }
}

// N_c > 4.  Kernel 1: per site n, the 216 link terms X_(s, mu)(n) into scratch[n][slot][NC^2].
template <int NC, typename E, int LAYOUT>
__global__ void __launch_bounds__(96) bril_force_site_kernel(const E *__restrict__ U, const E *__restrict__ psi,
                                                             const E *__restrict__ chi, E *__restrict__ X, Lat g) {
    using AB = bforce::Arith<NC, E>;
    using L = Layout<LAYOUT>;
    extern __shared__ __align__(16) unsigned char bf_smem[];
    auto Ws = reinterpret_cast<cx<AB>(*)[NC * NC]>(bf_smem);
    auto Gs = Ws + 81;
    const long long n = blockIdx.x;
    const int d = threadIdx.x < 81 ? kLevelOrder.d[threadIdx.x] : 81;   // offsets of a level share warps
    const Coord c = site_coords(g, n);
    const int x0[4] = {c.x, c.y, c.z, c.t};
    const int ext[4] = {g.nx, g.ny, g.nz, g.nt};
    int s[4] = {0, 0, 0, 0}, k = -1;
    if (d < 81) {
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) s[mu] = bforce::comp(d, mu);
        k = bforce::kk(d);
    }
    // ---- forward: W_s(n) level by level (W_0 = 1)
    if (k == 0)
        for (int e = 0; e < NC * NC; ++e) Ws[40][e] = cx<AB>{(AB)((e / NC) == (e % NC) ? 1 : 0), (AB)0};
    __syncthreads();
    for (int level = 1; level <= 4; ++level) {
        if (k == level) {
            cx<AB> acc[NC][NC];
            for (int a = 0; a < NC; ++a)
                for (int b = 0; b < NC; ++b) acc[a][b] = cx<AB>{0, 0};
            for (int mu = 0; mu < 4; ++mu) {
                if (s[mu] == 0) continue;
                const int prev = d - s[mu] * bforce::pow3(mu);
                int m[4];
                for (int nu = 0; nu < 4; ++nu) m[nu] = bforce::wrap(x0[nu] + (nu == mu ? 0 : s[nu]), ext[nu]);
                cx<AB> V[NC][NC];
                bforce::hop_link<NC, E, AB>(U, g, m, mu, s[mu], V);
                for (int a = 0; a < NC; ++a)
                    for (int b = 0; b < NC; ++b)
                        for (int q = 0; q < NC; ++q) cmac(acc[a][b], Ws[prev][a * NC + q], V[q][b]);
            }
            const AB inv = (AB)1 / (AB)level;
            for (int a = 0; a < NC; ++a)
                for (int b = 0; b < NC; ++b) Ws[d][a * NC + b] = inv * acc[a][b];
        }
        __syncthreads();
    }
    // ---- G_s = -2 M_s(n),  M_s = sum_{v, spin} (S_s psi(n+s)) chi(n)^dag
    if (k >= 1) {
        const AB rho = (AB)bril::rho(k);
        const AB lam_half = (AB)(0.5 * (double)(1 << (4 - k)) / 64.0);   // lambda_k / 2, lambda = (8,4,2,1)/64
        int m[4];
        for (int nu = 0; nu < 4; ++nu) m[nu] = bforce::wrap(x0[nu] + s[nu], ext[nu]);
        const long long ns = (((long long)m[3] * g.nz + m[2]) * g.ny + m[1]) * g.nx + m[0];
        const long long csd = L::cs_stride(g);
        const long long pb = L::vec(g, ns, NC * 4, 0), cb = L::vec(g, n, NC * 4, 0);
        cx<AB> M[NC][NC];
        for (int a = 0; a < NC; ++a)
            for (int b = 0; b < NC; ++b) M[a][b] = cx<AB>{0, 0};
        for (int v = 0; v < g.nv; ++v) {
            cx<AB> sp[NC][4], ch[NC][4];
#pragma unroll
            for (int a = 0; a < NC; ++a) {
                cx<AB> p[4];
#pragma unroll
                for (int sg = 0; sg < 4; ++sg) {
                    p[sg] = ld1<E, AB>(psi + 2 * (pb + (long long)(a * 4 + sg) * csd + v));
                    ch[a][sg] = ld1<E, AB>(chi + 2 * (cb + (long long)(a * 4 + sg) * csd + v));
                }
#pragma unroll
                for (int sg = 0; sg < 4; ++sg) {
                    cx<AB> f = {-lam_half * p[sg].re, -lam_half * p[sg].im};
#pragma unroll
                    for (int mu = 0; mu < 4; ++mu) {
                        if (s[mu] == 0) continue;
                        const cx<AB> t = bforce::gamma_comp<AB>(mu, sg, p);
                        const AB w = rho * (AB)s[mu];
                        f.re += w * t.re;
                        f.im += w * t.im;
                    }
                    sp[a][sg] = f;
                }
            }
#pragma unroll
            for (int a = 0; a < NC; ++a)
#pragma unroll
                for (int b = 0; b < NC; ++b)
#pragma unroll
                    for (int sg = 0; sg < 4; ++sg) cmac(M[a][b], sp[a][sg], conj(ch[b][sg]));
        }
        for (int a = 0; a < NC; ++a)
            for (int b = 0; b < NC; ++b) Gs[d][a * NC + b] = (AB)-2 * M[a][b];
    }
    __syncthreads();
    // ---- backward, level 4 down to 1
    for (int level = 4; level >= 1; --level) {
        if (k == level) {
            // link terms X = (1/k) G_s W_{s - s_mu mu} of this offset
            const AB inv = (AB)1 / (AB)level;
            for (int mu = 0; mu < 4; ++mu) {
                if (s[mu] == 0) continue;
                const int prev = d - s[mu] * bforce::pow3(mu);
                E *o = X + 2 * (((long long)n * bforce::kSlots + bforce::slot_of(d, mu)) * NC * NC);
                for (int a = 0; a < NC; ++a)
                    for (int b = 0; b < NC; ++b) {
                        cx<AB> t = {0, 0};
                        for (int q = 0; q < NC; ++q) cmac(t, Gs[d][a * NC + q], Ws[prev][q * NC + b]);
                        o[2 * (a * NC + b)] = from_acc<E, AB>(inv * t.re);
                        o[2 * (a * NC + b) + 1] = from_acc<E, AB>(inv * t.im);
                    }
            }
        }
        __syncthreads();
        if (level > 1 && k == level - 1) {
            // G_p += (1/level) V_{sign mu}(n + p) G_{p + sign mu}  over the parents of p
            const AB inv = (AB)1 / (AB)level;
            int m[4];
            for (int nu = 0; nu < 4; ++nu) m[nu] = bforce::wrap(x0[nu] + s[nu], ext[nu]);
            cx<AB> acc[NC][NC];
            for (int a = 0; a < NC; ++a)
                for (int b = 0; b < NC; ++b) acc[a][b] = Gs[d][a * NC + b];
            for (int mu = 0; mu < 4; ++mu) {
                if (s[mu] != 0) continue;
                for (int sign = -1; sign <= 1; sign += 2) {
                    const int child = d + sign * bforce::pow3(mu);
                    cx<AB> V[NC][NC];
                    bforce::hop_link<NC, E, AB>(U, g, m, mu, sign, V);
                    for (int a = 0; a < NC; ++a)
                        for (int b = 0; b < NC; ++b) {
                            cx<AB> t = {0, 0};
                            for (int q = 0; q < NC; ++q) cmac(t, V[a][q], Gs[child][q * NC + b]);
                            acc[a][b] = acc[a][b] + inv * t;
                        }
                }
            }
            for (int a = 0; a < NC; ++a)
                for (int b = 0; b < NC; ++b) Gs[d][a * NC + b] = acc[a][b];
        }
        __syncthreads();
    }
}

// Kernel 2: K_mu(m) from the 54 slots landing on link (m, mu), then F or G.
template <int NC, typename E, int LAYOUT>
__global__ void bril_force_link_kernel(const E *__restrict__ U, const E *__restrict__ X, E *__restrict__ out, Lat g,
                                       int bc0, int bc1, int bc2, int bc3, int mode) {
    using A = typename Acc<E>::T;
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (tid >= g.V * 4) return;
    const long long m = tid / 4;
    const int mu = (int)(tid % 4);
    const Coord c = site_coords(g, m);
    const int xm[4] = {c.x, c.y, c.z, c.t};
    const int ext[4] = {g.nx, g.ny, g.nz, g.nt};
    cx<A> K[NC][NC];
    for (int a = 0; a < NC; ++a)
        for (int b = 0; b < NC; ++b) K[a][b] = cx<A>{0, 0};
    for (int d = 0; d < 81; ++d) {
        const int smu = bforce::comp(d, mu);
        if (smu == 0) continue;
        // forward hop (s_mu = +1): n = m + mu - s;  backward hop (s_mu = -1): n = m - s
        int nn[4];
#pragma unroll
        for (int nu = 0; nu < 4; ++nu) {
            const int sn = bforce::comp(d, nu);
            const int off = (smu > 0 && nu == mu) ? 1 - sn : -sn;
            nn[nu] = bforce::wrap(xm[nu] + off, ext[nu]);
        }
        const long long n = (((long long)nn[3] * g.nz + nn[2]) * g.ny + nn[1]) * g.nx + nn[0];
        const E *x = X + 2 * ((n * bforce::kSlots + bforce::slot_of(d, mu)) * NC * NC);
        for (int a = 0; a < NC; ++a)
            for (int b = 0; b < NC; ++b) {
                const cx<A> v = ld1<E, A>(x + 2 * (smu > 0 ? a * NC + b : b * NC + a));
                K[a][b] = K[a][b] + (smu > 0 ? v : conj(v));
            }
    }
    link_output<NC, E>(U, out + 2 * (tid * NC * NC), g, m, mu, c, K, bc0, bc1, bc2, bc3, mode);
}

// ------------------------------------------------------------ tiled (N_c <= 4)
namespace bforce {

// Scratch of one tile: 216 slots of N_c x N_c matrices for the tile's S sites,
// [slot][e][site].  The link terms X of level k (k of them per offset) fill
// the slots from xbase(k) on, level 4 first.  Before a level's link terms are
// written its slots hold M_s (one per offset); the slots between hold the
// tile's psi and chi in [component][RHS][site] order for at most kChunk(N_c)
// right-hand sides at a time.
__host__ __device__ constexpr int xbase(int k) { return k == 4 ? 0 : k == 3 ? 64 : k == 2 ? 160 : 208; }
__host__ __device__ constexpr int mslot(int pos, int k) { return xbase(k) + pos - hyper::level_begin(k); }
__host__ __device__ constexpr int xslot(int pos, int k, int j) { return xbase(k) + (pos - hyper::level_begin(k)) * k + j; }
constexpr int kPsiSlot = 16, kChiSlot = 96;   // 48 and 64 slots long
__host__ __device__ constexpr int chunk(int nc) { return 12 * nc; }   // 4 N_c chunk <= 48 N_c^2

template <int NC, typename E>
struct FTile {
    using AB = Arith<NC, E>;
    static constexpr int NN = NC * NC;
    static constexpr int kMats = 88;   // W of levels 1, 2; W then G of level 3; G of level 4, then of level 2
    static constexpr int S = hyper::tile_sites(kMats, NC, sizeof(cx<AB>), false);
    static constexpr size_t smem = (size_t)kMats * NN * S * sizeof(cx<AB>);
    static constexpr long long tile = (long long)kSlots * NN * S;   // complex numbers of scratch per tile
    // element 0 of a slot for one site
    static __device__ __forceinline__ long long at(long long site, int slot) {
        return (site / S) * tile + (long long)slot * NN * S + site % S;
    }
};

// One tile-ordered copy of RHS v0 .. v0 + cnt - 1 of a vector: component c
// (colour, spin) and RHS v of a site at slot0 + (c cnt + v) lanes apart by S.
template <int NC, typename E, int LAYOUT>
__global__ void __launch_bounds__(256) bril_force_stage_kernel(const E *__restrict__ psi, const E *__restrict__ chi,
                                                               E *__restrict__ X, Lat g, int v0, int cnt) {
    using T = FTile<NC, E>;
    using A = typename Acc<E>::T;
    using L = Layout<LAYOUT>;
    __shared__ cx<A> tile[32][33];
    const int M = NC * 4 * cnt, c0 = blockIdx.y * 32;
    const long long n0 = (long long)blockIdx.x * 32;
    const E *in = blockIdx.z ? chi : psi;
    const int slot = blockIdx.z ? kChiSlot : kPsiSlot;
    const long long csd = L::cs_stride(g);
    const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
    // read with lanes over (component, RHS), write with lanes over sites
    for (int r = ty; r < 32; r += 8) {
        const long long n = n0 + r;
        const int c = c0 + tx;
        if (n < g.V && c < M)
            tile[r][tx] = ld1<E, A>(in + 2 * (L::vec(g, n, NC * 4, 0) + (c / cnt) * csd + v0 + c % cnt));
    }
    __syncthreads();
    for (int r = ty; r < 32; r += 8) {
        const long long n = n0 + tx;
        const int c = c0 + r;
        if (n < g.V && c < M) store_cx<E, 1, A>(X + 2 * (T::at(n, slot) + (long long)c * T::S), &tile[tx][r]);
    }
}

// f += sign gamma_MU p for the four spins of one colour
template <int MU, typename A>
__device__ __forceinline__ void add_gamma(cx<A> (&f)[4], const cx<A> (&p)[4], A sign) {
#pragma unroll
    for (int sg = 0; sg < 4; ++sg) {
        const cx<A> t = gamma_comp<A>(MU, sg, p);
        f[sg].re = fma(sign, t.re, f[sg].re);
        f[sg].im = fma(sign, t.im, f[sg].im);
    }
}

// Step 2: G_s = -2 M_s(n) for the offsets of one warp's rows.  Lane = site;
// warp w of a block takes the nine rows with s_t = w - 1, and of each row the
// three s_x at once (FP32, N_c <= 3) or one by one.  With
// S_s = rho_k (sum_mu s_mu gamma_mu - c_k) hermitian,
//   M_s = rho_k sum_{v, spin} psi(n+s) [(sum_mu s_mu gamma_mu - c_k) chi(n)]^dag,
// and the gamma terms of y, z, t on chi(n) are formed once per row and RHS.
// Bound by the FP32 pipe: about 210 multiply-adds per offset and RHS.
template <int NC, typename E>
__global__ void __launch_bounds__(96, sizeof(E) == 4 && NC <= 3 ? 4 : 2) bril_force_outer_kernel(E *__restrict__ X, Lat g, int cnt, int first) {
    using T = FTile<NC, E>;
    using A = Arith<NC, E>;
    const long long n_own = (long long)blockIdx.x * 32 + threadIdx.x % 32;
    const bool live = n_own < g.V;
    const long long n = live ? n_own : g.V - 1;
    const hyper::Steps st = hyper::steps_at(g, n);
    const int s_t = (int)(threadIdx.x / 32) - 1;
    const E *chi = X + 2 * T::at(n, kChiSlot);
    constexpr int G = sizeof(A) == 4 && NC <= 3 ? 3 : 1;   // s_x values per pass
    auto axis = [](const hyper::Steps &q, int mu, int sgn) { return sgn > 0 ? q.p[mu] : (sgn < 0 ? q.m[mu] : 0); };
#pragma unroll 1
    for (int row = 0; row < 9; ++row) {
        const int s_z = row / 3 - 1, s_y = row % 3 - 1;
        const int krow = (s_t != 0) + (s_z != 0) + (s_y != 0);
        const long long nrow = n + axis(st, 3, s_t) + axis(st, 2, s_z) + axis(st, 1, s_y);
#pragma unroll 1
        for (int x0 = -1; x0 <= 1; x0 += G) {
            cx<A> M[G][NC][NC];
#pragma unroll
            for (int i = 0; i < G; ++i)
#pragma unroll
                for (int a = 0; a < NC; ++a)
#pragma unroll
                    for (int b = 0; b < NC; ++b) M[i][a][b] = cx<A>{0, 0};
            const E *psi[G];
#pragma unroll
            for (int i = 0; i < G; ++i) psi[i] = X + 2 * T::at(nrow + axis(st, 0, x0 + i), kPsiSlot);
#pragma unroll 1
            for (int v = 0; v < cnt; ++v) {
                cx<A> ch[NC][4], f[NC][4];
#pragma unroll
                for (int b = 0; b < NC; ++b) {
#pragma unroll
                    for (int sg = 0; sg < 4; ++sg) {
                        ch[b][sg] = ld1<E, A>(chi + 2LL * ((b * 4 + sg) * cnt + v) * T::S);
                        f[b][sg] = cx<A>{0, 0};
                    }
                    if (s_y != 0) add_gamma<1>(f[b], ch[b], (A)s_y);
                    if (s_z != 0) add_gamma<2>(f[b], ch[b], (A)s_z);
                    if (s_t != 0) add_gamma<3>(f[b], ch[b], (A)s_t);
                }
#pragma unroll
                for (int i = 0; i < G; ++i) {
                    const int s_x = x0 + i, k = krow + (s_x != 0);
                    if (k == 0) continue;
                    const A ck = (A)(27.0 / 128.0) * (A)(1 << k);   // c_k = 27/64 2^(k-1)
                    cx<A> h[NC][4];
#pragma unroll
                    for (int b = 0; b < NC; ++b) {
#pragma unroll
                        for (int sg = 0; sg < 4; ++sg)
                            h[b][sg] = cx<A>{fma(-ck, ch[b][sg].re, f[b][sg].re), fma(-ck, ch[b][sg].im, f[b][sg].im)};
                        if (s_x != 0) add_gamma<0>(h[b], ch[b], (A)s_x);
                    }
#pragma unroll
                    for (int a = 0; a < NC; ++a) {
                        cx<A> p[4];
#pragma unroll
                        for (int sg = 0; sg < 4; ++sg)
                            p[sg] = ld1<E, A>(psi[i] + 2LL * ((a * 4 + sg) * cnt + v) * T::S);
#pragma unroll
                        for (int b = 0; b < NC; ++b)
#pragma unroll
                            for (int sg = 0; sg < 4; ++sg) cmac_conj(M[i][a][b], h[b][sg], p[sg]);
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < G; ++i) {
                const int s_x = x0 + i, k = krow + (s_x != 0);
                if (k == 0 || !live) continue;
                const A w = (A)-2 * (A)bril::rho(k);
                const int pos = hyper::kTable.pos[(s_t + 1) * 27 + (s_z + 1) * 9 + (s_y + 1) * 3 + s_x + 1];
                E *o = X + 2 * T::at(n, xbase(k) + pos - hyper::level_begin(k));
#pragma unroll
                for (int a = 0; a < NC; ++a)
#pragma unroll
                    for (int b = 0; b < NC; ++b) {
                        cx<A> m = w * M[i][a][b];
                        E *oe = o + 2LL * (a * NC + b) * T::S;
                        if (!first) m = m + ld1<E, A>(oe);
                        store_cx<E, 1, A>(oe, &m);
                    }
            }
        }
    }
}

// Step 3, G of level K into shared memory: G_s = -2 M_s + (1/(K+1)) sum over
// the offsets one hop further of V G, read from the level above.  `mat` maps
// a position in the offset table to its matrix in shared memory.
template <int K, int NC, typename E, typename SRC, typename MAT>
__device__ __forceinline__ void force_g(cx<Arith<NC, E>> (&acc)[NC][NC], const cx<Arith<NC, E>> *mats,
                                        const E *__restrict__ X, const SRC &src, long long n, const hyper::Steps &st,
                                        int lane, int pos, MAT mat) {
    using T = FTile<NC, E>;
    using A = Arith<NC, E>;
    const E *m = X + 2 * T::at(n, mslot(pos, K));
#pragma unroll
    for (int a = 0; a < NC; ++a)
#pragma unroll
        for (int b = 0; b < NC; ++b) acc[a][b] = ld1<E, A>(m + 2LL * (a * NC + b) * T::S);
    if constexpr (K < 4) {
        const hyper::Offset &o = hyper::kTable.o[pos];
        const long long site = n + hyper::step_of(st, o.s);
        const A inv = (A)1 / (A)(K + 1);
#pragma unroll 2
        for (int c = 0; c < 2 * (4 - K); ++c) {
            const int mu = o.cmu[c];
            const bool back = o.csign[c] < 0;
            cx<A> V[NC][NC];
            src.load(site + (back ? hyper::pick(st.m, mu) : 0), mu, back, V);
            const cx<A> *P = mats + mat(o.child[c]) * T::NN * T::S + lane;
            cx<A> t[NC][NC];
#pragma unroll
            for (int a = 0; a < NC; ++a)
#pragma unroll
                for (int b = 0; b < NC; ++b) t[a][b] = cx<A>{0, 0};
#pragma unroll
            for (int q = 0; q < NC; ++q)
#pragma unroll
                for (int b = 0; b < NC; ++b) {
                    const cx<A> gq = P[(q * NC + b) * T::S];
#pragma unroll
                    for (int a = 0; a < NC; ++a) cmac(t[a][b], V[a][q], gq);
                }
#pragma unroll
            for (int a = 0; a < NC; ++a)
#pragma unroll
                for (int b = 0; b < NC; ++b) acc[a][b] = acc[a][b] + inv * t[a][b];
        }
    }
}

// Step 3, link terms X = (1/K) G_s W_{s - s_mu mu} of one offset of level K >= 2
template <int K, int NC, typename E, typename MAT>
__device__ __forceinline__ void force_x(const cx<Arith<NC, E>> *mats, E *__restrict__ X, long long n, bool live,
                                        int lane, int pos, MAT mat) {
    using T = FTile<NC, E>;
    using A = Arith<NC, E>;
    const hyper::Offset &o = hyper::kTable.o[pos];
    cx<A> g[NC][NC];
    const cx<A> *Gs = mats + mat(pos) * T::NN * T::S + lane;
#pragma unroll
    for (int a = 0; a < NC; ++a)
#pragma unroll
        for (int b = 0; b < NC; ++b) g[a][b] = Gs[(a * NC + b) * T::S];
    const A inv = (A)1 / (A)K;
#pragma unroll 1
    for (int j = 0; j < K; ++j) {
        const cx<A> *P = mats + o.prev[j] * T::NN * T::S + lane;
        cx<A> t[NC][NC];
#pragma unroll
        for (int a = 0; a < NC; ++a)
#pragma unroll
            for (int b = 0; b < NC; ++b) t[a][b] = cx<A>{0, 0};
#pragma unroll
        for (int q = 0; q < NC; ++q)
#pragma unroll
            for (int b = 0; b < NC; ++b) {
                const cx<A> w = P[(q * NC + b) * T::S];
#pragma unroll
                for (int a = 0; a < NC; ++a) cmac(t[a][b], g[a][q], w);
            }
        if (!live) continue;
        E *x = X + 2 * T::at(n, xslot(pos, K, j));
#pragma unroll
        for (int a = 0; a < NC; ++a)
#pragma unroll
            for (int b = 0; b < NC; ++b) {
                const cx<A> v = inv * t[a][b];
                store_cx<E, 1, A>(x + 2LL * (a * NC + b) * T::S, &v);
            }
    }
}

// Step 3: one block per tile.  Shared memory (88 matrices per site): W of
// levels 1 to 3 at their positions 0..63, the slots of level 3 taken over by
// its G once the link terms of level 4 are done; G of level 4 at 64..79, its
// slots taken over by G of level 2 (positions 8..31).  A barrier stands
// between the reads of a level's M_s and the link terms that replace them.
template <int NC, typename E>
__global__ void __launch_bounds__(hyper::kThreads, 2) bril_force_tile_kernel(const E *__restrict__ U,
                                                                             E *__restrict__ X, Lat g) {
    using T = FTile<NC, E>;
    using A = Arith<NC, E>;
    constexpr int NW = hyper::kThreads / T::S;
    extern __shared__ __align__(16) unsigned char bt_smem[];
    cx<A> *mats = reinterpret_cast<cx<A> *>(bt_smem);
    const int lane = threadIdx.x % T::S, worker = threadIdx.x / T::S;
    const long long n_own = (long long)blockIdx.x * T::S + lane;
    const bool live = n_own < g.V;
    const long long n = live ? n_own : g.V - 1;
    const hyper::Steps st = hyper::steps_at(g, n);
    const hyper::NativeLinks<NC, E, A> src{U};
    auto ident = [](int pos) { return pos; };
    auto q24 = [](int pos) { return pos >= 64 ? pos : 64 + pos - 8; };   // G of level 4, and of level 2
    hyper::w_level<1, NC, T::S, NW>(mats, src, n, st, lane, worker, ident);
    hyper::w_level<2, NC, T::S, NW>(mats, src, n, st, lane, worker, ident);
    hyper::w_level<3, NC, T::S, NW>(mats, src, n, st, lane, worker, ident);
    auto put = [&](int m, const cx<A> (&v)[NC][NC]) {
#pragma unroll
        for (int a = 0; a < NC; ++a)
#pragma unroll
            for (int b = 0; b < NC; ++b) mats[(m * T::NN + a * NC + b) * T::S + lane] = v[a][b];
    };
    cx<A> acc[NC][NC];
    for (int pos = 64 + worker; pos < 80; pos += NW) {
        force_g<4, NC, E>(acc, mats, X, src, n, st, lane, pos, q24);
        put(pos, acc);
    }
    __syncthreads();
    for (int pos = 64 + worker; pos < 80; pos += NW) force_x<4, NC, E>(mats, X, n, live, lane, pos, ident);
    __syncthreads();
    for (int pos = 32 + worker; pos < 64; pos += NW) {
        force_g<3, NC, E>(acc, mats, X, src, n, st, lane, pos, q24);
        put(pos, acc);
    }
    __syncthreads();
    for (int pos = 32 + worker; pos < 64; pos += NW) force_x<3, NC, E>(mats, X, n, live, lane, pos, ident);
    for (int pos = 8 + worker; pos < 32; pos += NW) {
        force_g<2, NC, E>(acc, mats, X, src, n, st, lane, pos, ident);
        put(q24(pos), acc);
    }
    __syncthreads();
    for (int pos = 8 + worker; pos < 32; pos += NW) force_x<2, NC, E>(mats, X, n, live, lane, pos, q24);
    // level 1: X = G_s (W of the centre is 1); at most one offset per worker
    static_assert(NW >= 8, "one level-1 offset per worker");
    if (worker < 8) force_g<1, NC, E>(acc, mats, X, src, n, st, lane, worker, q24);
    __syncthreads();
    if (worker < 8 && live) {
        E *x = X + 2 * T::at(n, xslot(worker, 1, 0));
#pragma unroll
        for (int a = 0; a < NC; ++a)
#pragma unroll
            for (int b = 0; b < NC; ++b) store_cx<E, 1, A>(x + 2LL * (a * NC + b) * T::S, &acc[a][b]);
    }
}

// The 54 link terms that land on a link (m, mu): slot, the step from m to the
// site that holds the term, and whether the hop runs forward along the link.
struct LinkTerm {
    short slot;
    signed char sh[4];
    signed char fwd;
};
struct LinkTerms {
    LinkTerm t[4][54];
};
__host__ __device__ constexpr LinkTerms make_link_terms() {
    LinkTerms r{};
    const hyper::Table tb = hyper::make_table();
    for (int mu = 0; mu < 4; ++mu) {
        int c = 0;
        for (int pos = 0; pos < 80; ++pos) {
            const hyper::Offset &o = tb.o[pos];
            if (o.s[mu] == 0) continue;
            int j = 0;
            while (o.mu[j] != mu) ++j;
            LinkTerm &t = r.t[mu][c++];
            t.slot = (short)xslot(pos, o.k, j);
            t.fwd = o.s[mu] > 0;
            // forward hop (s_mu = +1): n = m + mu - s;  backward hop (s_mu = -1): n = m - s
            for (int nu = 0; nu < 4; ++nu) t.sh[nu] = (signed char)(-o.s[nu] + (nu == mu && o.s[mu] > 0 ? 1 : 0));
        }
    }
    return r;
}
static __constant__ LinkTerms kLinkTerms = make_link_terms();

// Step 4: one thread per link, lanes over sites, blockIdx.y = mu.
template <int NC, typename E>
__global__ void __launch_bounds__(128) bril_force_gather_kernel(const E *__restrict__ U, const E *__restrict__ X,
                                                                E *__restrict__ out, Lat g, int bc0, int bc1, int bc2,
                                                                int bc3, int mode) {
    using T = FTile<NC, E>;
    using A = typename Acc<E>::T;
    const long long m = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= g.V) return;
    const int mu = blockIdx.y;
    const hyper::Steps st = hyper::steps_at(g, m);
    cx<A> K[NC][NC];
#pragma unroll
    for (int a = 0; a < NC; ++a)
#pragma unroll
        for (int b = 0; b < NC; ++b) K[a][b] = cx<A>{0, 0};
#pragma unroll 2
    for (int i = 0; i < 54; ++i) {
        const LinkTerm &t = kLinkTerms.t[mu][i];   // uniform over the block
        const E *x = X + 2 * T::at(m + hyper::step_of(st, t.sh), t.slot);
        const bool fwd = t.fwd;
#pragma unroll
        for (int a = 0; a < NC; ++a)
#pragma unroll
            for (int b = 0; b < NC; ++b) {
                const cx<A> v = ld1<E, A>(x + 2LL * (fwd ? a * NC + b : b * NC + a) * T::S);
                K[a][b] = K[a][b] + cx<A>{v.re, fwd ? v.im : -v.im};
            }
    }
    E *o = out + 2 * ((m * 4 + mu) * T::NN);
    const Coord c = site_coords(g, m);
    link_output<NC, E>(U, o, g, m, mu, c, K, bc0, bc1, bc2, bc3, mode);
}

template <int NC, typename E, int LAYOUT>
int launch_tiled(const dirac_op *op, const void *psi, const void *chi, void *out, int mode, cudaStream_t s) {
    using T = FTile<NC, E>;
    E *X = (E *)op->force_ws;
    const Lat &g = op->lat;
    const int step = chunk(NC);
    for (int v0 = 0; v0 < op->nv; v0 += step) {
        const int cnt = op->nv - v0 < step ? op->nv - v0 : step;
        const dim3 grid(grid_for(op->V, 32), (unsigned)((NC * 4 * cnt + 31) / 32), 2);
        bril_force_stage_kernel<NC, E, LAYOUT><<<grid, 256, 0, s>>>((const E *)psi, (const E *)chi, X, g, v0, cnt);
        int rc = launch_check("bril_force_stage_kernel");
        if (rc) return rc;
        bril_force_outer_kernel<NC, E><<<grid_for(op->V, 32), 96, 0, s>>>(X, g, cnt, v0 == 0);
        rc = launch_check("bril_force_outer_kernel");
        if (rc) return rc;
    }
    if constexpr (T::smem > 48 * 1024) {
        const int rc = cuda_check(cudaFuncSetAttribute(bril_force_tile_kernel<NC, E>,
                                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)T::smem),
                                  "bril_force_tile_kernel shared memory");
        if (rc) return rc;
    }
    bril_force_tile_kernel<NC, E><<<grid_for(op->V, T::S), hyper::kThreads, T::smem, s>>>((const E *)op->links, X, g);
    const int rc = launch_check("bril_force_tile_kernel");
    if (rc) return rc;
    const int *bc = op->geom.bc;
    bril_force_gather_kernel<NC, E><<<dim3(grid_for(op->V, 128), 4), 128, 0, s>>>(
        (const E *)op->links, X, (E *)out, g, bc[0], bc[1], bc[2], bc[3], mode);
    return launch_check("bril_force_gather_kernel");
}

}  // namespace bforce

// Brillouin force: scratch of 216 link terms per site, owned by the operator
// (allocated on first use, freed with it).
int launch_bril_force(dirac_op *op, const void *psi, const void *chi, void *out, int mode, cudaStream_t s) {
    // whole tiles of at most 32 sites
    const size_t sites = (size_t)(op->V + 31) / 32 * 32;
    const size_t need = sites * bforce::kSlots * op->nc * op->nc * 2 * elem_bytes(op->prec);
    if (op->force_ws_bytes < need) {
        cudaFree(op->force_ws);
        op->force_ws = nullptr;
        op->force_ws_bytes = 0;
        if (cudaMalloc(&op->force_ws, need) != cudaSuccess) {
            cudaGetLastError();
            op->force_ws = nullptr;
            return DIRAC_ERR_OOM;
        }
        op->force_ws_bytes = need;
    }
    return dispatch_prec(op->prec, [&](auto tag) {
        using E = std::remove_pointer_t<decltype(tag)>;
        if constexpr (sizeof(E) == 2) {
            return (int)DIRAC_ERR_UNSUPPORTED_PREC;
        } else {
            return dispatch_nc(op->nc, [&](auto ncc) {
                constexpr int NC = decltype(ncc)::value;
                return dispatch_layout(op->geom.layout, [&](auto lyc) {
                    constexpr int LAYOUT = decltype(lyc)::value;
                    if constexpr (NC <= kMaxNcSmall) {
                        return bforce::launch_tiled<NC, E, LAYOUT>(op, psi, chi, out, mode, s);
                    } else {
                    constexpr size_t smem = bforce::site_smem<NC, E>();
                    if constexpr (smem > 48 * 1024) {
                        const int rc = cuda_check(cudaFuncSetAttribute(bril_force_site_kernel<NC, E, LAYOUT>,
                                                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                                       (int)smem),
                                                  "bril_force_site_kernel shared memory");
                        if (rc) return rc;
                    }
                    bril_force_site_kernel<NC, E, LAYOUT><<<(unsigned)op->V, 96, smem, s>>>(
                        (const E *)op->links, (const E *)psi, (const E *)chi, (E *)op->force_ws, op->lat);
                    int rc = launch_check("bril_force_site_kernel");
                    if (rc) return rc;
                    const int *bc = op->geom.bc;
                    bril_force_link_kernel<NC, E, LAYOUT><<<grid_for(op->V * 4, 128), 128, 0, s>>>(
                        (const E *)op->links, (const E *)op->force_ws, (E *)out, op->lat, bc[0], bc[1], bc[2], bc[3],
                        mode);
                    return launch_check("bril_force_link_kernel");
                    }
                });
            });
        }
    });
}

}  // namespace dgb
