// laplace.cuh -- multi-RHS Laplace operators A = -1/2 Lap + m^2/2 (Secs. 6
// and 7; the paper's wlap, blap, wsuv, bsuv routines of App. F):
//   Eq. (app_wlap): (A psi)(n) = (4 + m^2/2) psi(n)
//        - 1/2 sum_mu [ U_mu(n) psi(n+mu) + U_mu(n-mu)^dag psi(n-mu) ]
//   Eq. (app_blap): (A psi)(n) = (m^2/2 - lambda_0/2) psi(n) - 1/2 sum_{s != 0} lambda_k W_s(n) psi(n+s)
// acting trivially on NS spin components per colour (NS = 4: Wilson-type
// vectors, NS = 1: colour-only vectors).  A is hermitian: no dagger variant.
//
// Same thread mapping as the Dirac stencils (thread <-> site, VR consecutive
// right-hand sides; write-once register accumulator).  The Brillouin
// Laplacian reads the operator's stored W~_q = rho_k s_lead W_s (bril_dirs.h),
// per site in visiting order, and weighs each with -c_k s_lead, which is
// -lambda_k/2 on W_s; offsets and weights come from a table in constant
// memory (one broadcast read per offset, uniform over the warp).  In FP32 W~ is
// staged in shared memory for the block (wstage.cuh) and its products are packed
// (common.cuh): blap 0.991 -> 0.920 ms, bsuv 0.490 -> 0.293 ms at 16^3x32,
// N_v = 12, N_c = 3.
#pragma once
#include "bril_dirs.h"
#include "internal.h"
#include "wstage.cuh"

namespace dgb {
namespace bril {

// The offsets in storage order with the weight of the Brillouin Laplacian on
// the stored W~: -lambda_k/2 W_s = -c_k s_lead W~_q (Eq. app_blap).
struct OffsetTable {
    signed char s[80][4];
    double lap[80];
};
__host__ __device__ constexpr OffsetTable make_offset_table() {
    OffsetTable t{};
    for (int d = 0; d < 81; ++d) {
        const int s[4] = {d % 3 - 1, (d / 3) % 3 - 1, (d / 9) % 3 - 1, d / 27 - 1};
        const int k = (s[0] != 0) + (s[1] != 0) + (s[2] != 0) + (s[3] != 0);
        if (k == 0) continue;
        double scale = 0;
        const int q = store_index(s, &scale);
        for (int mu = 0; mu < 4; ++mu) t.s[q][mu] = (signed char)s[mu];
        t.lap[q] = -c_lambda(k) * (scale < 0 ? -1.0 : 1.0);
    }
    return t;
}

}  // namespace bril

static __constant__ bril::OffsetTable kLapOffsets = bril::make_offset_table();

// Whether a hop multiplies its weight into the N_c x N_c matrix (N_c^2 complex
// scalings) and its products into the running sum, or sums its own N_c
// products first and adds that sum with the weight (one real multiply-add per
// complex component).  Without many components per matrix the second costs no
// more and its sums are short, so its error is the smaller.
template <int NC, int NS, int VR>
constexpr bool fold_weight() { return NS * VR > NC; }

// The running sum of a component: of products P where they go into it
// directly, a plain number where a hop's own sum is added.
template <typename P, int NC, int NS, int VR, typename A>
using LapAcc = std::conditional_t<fold_weight<NC, NS, VR>(), typename P::Acc, typename Prod<A, false>::Acc>;

// acc[c][s] += f L psi(m) (or f L^dag psi(m)) for every spin component s
template <typename P, int NC, int NS, int VR, bool DAG, typename E, typename A>
__device__ __forceinline__ void lap_hop(LapAcc<P, NC, NS, VR, A> (&acc)[NC][NS][VR], const cx<A> (&L)[NC][NC],
                                        const E *__restrict__ psi, long long cs_stride, A f) {
    if constexpr (fold_weight<NC, NS, VR>()) {
        // one colour component of the neighbour at a time: column k of the matrix
        // and NS VR vector components in registers
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            typename P::Mul w[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) w[c] = P::mul(f * (DAG ? conj(L[k][c]) : L[c][k]));
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                cx<A> p[VR];
                load_cx<E, VR, A>(psi + 2 * (k * NS + s) * cs_stride, p);
#pragma unroll
                for (int v = 0; v < VR; ++v) {
                    const typename P::Vec pv = P::vec(p[v]);
#pragma unroll
                    for (int c = 0; c < NC; ++c) acc[c][s][v].mac(w[c], pv);
                }
            }
        }
    } else {
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            cx<A> p[NC][VR];
#pragma unroll
            for (int k = 0; k < NC; ++k) load_cx<E, VR, A>(psi + 2 * (k * NS + s) * cs_stride, p[k]);
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                typename P::Acc t[VR];
#pragma unroll
                for (int k = 0; k < NC; ++k) {
                    const typename P::Mul w = P::mul(DAG ? conj(L[k][c]) : L[c][k]);
#pragma unroll
                    for (int v = 0; v < VR; ++v) t[v].mac(w, P::vec(p[k][v]));
                }
#pragma unroll
                for (int v = 0; v < VR; ++v) rmac(acc[c][s][v].s, f, t[v].value());
            }
        }
    }
}

template <typename P, int NC, int NS, int VR, int LAYOUT, typename E, typename A>
__device__ __forceinline__ void lap_write(const E *__restrict__ in, E *__restrict__ out, const Lat &g, long long n,
                                          int j, A centre, const LapAcc<P, NC, NS, VR, A> (&acc)[NC][NS][VR]) {
    using L = Layout<LAYOUT>;
    const long long cs = L::cs_stride(g);
    const long long base = 2 * (L::vec(g, n, NC * NS, 0) + (long long)j * VR);
#pragma unroll
    for (int a = 0; a < NC; ++a)
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            cx<A> p[VR], o[VR];
            const long long off = base + 2LL * (a * NS + s) * cs;
            load_cx<E, VR, A>(in + off, p);
#pragma unroll
            for (int v = 0; v < VR; ++v) o[v] = centre * p[v] + acc[a][s][v].value();
            store_cx<E, VR, A>(out + off, o);
        }
}

// Eq. (app_wlap): centre = 4 + m^2/2, each hop weighted -1/2
template <int NC, int NS, int VR, typename E, int MINB, int LAYOUT>
__global__ void __launch_bounds__(stencil_max_threads(MINB),
                                  (stencil_min_blocks<NC, NS, VR, MINB, typename Acc<E>::T>(NC <= 2, NC * NS + NC * NC)))
    wlap_kernel(const E *__restrict__ U, const E *__restrict__ in, E *__restrict__ out, Lat g,
                typename Acc<E>::T centre) {
    using A = typename Acc<E>::T;
    using L = Layout<LAYOUT>;
    const int nchunk = g.nv / VR;
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (tid >= g.nsites * nchunk) return;
    long long i;
    int j;
    split_tid(tid, nchunk, i, j);
    const long long n = g.n0 + i;
    const Coord c = site_coords(g, n);
    const long long cs = L::cs_stride(g), ls = L::template mat_stride<NC>(g);

    using P = Prod<A, false>;   // packed products measured slower here (0.121 vs 0.115 ms): the second
                                // accumulator costs warps, and the loads bound this kernel
    LapAcc<P, NC, NS, VR, A> acc[NC][NS][VR];
    const A mhalf = (A)-0.5;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        const long long fw = neighbour(g, n, c, mu, +1);
        const long long bw = neighbour(g, n, c, mu, -1);
        cx<A> Lm[NC][NC];
        load_mat_s<NC, E, A>(U + 2 * L::template mat<NC>(g, n, 4, mu), ls, Lm);
        lap_hop<P, NC, NS, VR, false, E, A>(acc, Lm, in + 2 * (L::vec(g, fw, NC * NS, 0) + (long long)j * VR), cs, mhalf);
        load_mat_s<NC, E, A>(U + 2 * L::template mat<NC>(g, bw, 4, mu), ls, Lm);
        lap_hop<P, NC, NS, VR, true, E, A>(acc, Lm, in + 2 * (L::vec(g, bw, NC * NS, 0) + (long long)j * VR), cs, mhalf);
    }
    lap_write<P, NC, NS, VR, LAYOUT, E, A>(in, out, g, n, j, centre, acc);
}

// Eq. (app_blap): centre = m^2/2 - lambda_0/2, offset q weighted kLapOffsets.lap[q] on W~_q
// STAGED: W~ through shared memory, one ring per block (wstage.cuh); else each
// thread reads its own.
template <int NC, int NS, int VR, typename E, int MINB, int LAYOUT, bool STAGED>
__global__ void __launch_bounds__(stencil_max_threads(MINB),
                                  (stencil_min_blocks<NC, NS, VR, MINB, typename Acc<E>::T>(NS == 4 ? NC == 4 || NC == 5 : NC == 4 || NC >= 6, NC * NS * VR + NC * NC)))
    blap_kernel(const E *__restrict__ W, const E *__restrict__ in, E *__restrict__ out, Lat g,
                typename Acc<E>::T centre) {
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
    const long long cs = L::cs_stride(g);
    // site-index steps of +1 / -1 along each axis, with the periodic wrap
    // (32-bit: volumes are below 2^31 sites)
    int dp[4], dm[4];
    {
        const int co[4] = {c.x, c.y, c.z, c.t};
        const int ext[4] = {g.nx, g.ny, g.nz, g.nt};
        int stride = 1;
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) {
            dp[mu] = (co[mu] == ext[mu] - 1 ? -(ext[mu] - 1) : 1) * stride;
            dm[mu] = (co[mu] == 0 ? ext[mu] - 1 : -1) * stride;
            stride *= ext[mu];
        }
    }
    using P = StencilProd<NC, NS, VR, MINB, A>;
    LapAcc<P, NC, NS, VR, A> acc[NC][NS][VR];
    // W~ of one site contiguous in visiting order (either vector layout)
    const E *inj = in + 2LL * j * VR;
    auto hop = [&](int q, const cx<A>(&Wm)[NC][NC]) {
        int m = (int)n;
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) {
            const int sm = kLapOffsets.s[q][mu];
            m += sm > 0 ? dp[mu] : (sm < 0 ? dm[mu] : 0);
        }
        lap_hop<P, NC, NS, VR, false, E, A>(acc, Wm, inj + 2 * L::vec(g, (long long)m, NC * NS, 0), cs,
                                         (A)kLapOffsets.lap[q]);
    };
    if constexpr (STAGED) {
        extern __shared__ __align__(16) unsigned char w_ring[];
        const long long s0 = tid0 / nchunk, end = tid0 + blockDim.x < total ? tid0 + blockDim.x : total;
        wst::Ring<NC, E> ring;
        ring.src = reinterpret_cast<const unsigned char *>(W + 2LL * (g.n0 + s0) * 80 * NC * NC);
        ring.smem = w_ring;
        ring.nsites = (int)((end - 1) / nchunk - s0 + 1);
        ring.slots = wst::block_sites(blockDim.x, nchunk);
        ring.mine = (int)(i - s0);
        ring.start();
        int q = 0;
#pragma unroll 1
        for (int stage = 0; stage < wst::kStages; ++stage) {
            const E *w = ring.enter(stage);
            const int end_q = 2 + 6 * stage;
#pragma unroll 1
            for (; q < end_q; q += 2, w += 4 * NC * NC) {
                cx<A> Wm[NC][NC];
                wst::load_mat_shared<NC, E, A>(w, Wm);
                hop(q, Wm);
                wst::load_mat_shared<NC, E, A>(w + 2 * NC * NC, Wm);
                hop(q + 1, Wm);
            }
        }
        if (!live) return;
    } else if constexpr (NC <= kMaxNcSmall) {
        const E *wp = W + 2LL * n * 80 * NC * NC;
        // two offsets per trip: the W~ of the next offset is loaded while the
        // current one is applied, the two buffers swapping roles (80 is even)
        cx<A> Wa[NC][NC], Wb[NC][NC];
        load_mat<NC, E, A>(wp, Wa);
#pragma unroll 1
        for (int q = 0; q < 80; q += 2) {
            load_mat<NC, E, A>(wp + 2 * (q + 1) * NC * NC, Wb);
            hop(q, Wa);
            if (q + 2 < 80) load_mat<NC, E, A>(wp + 2 * (q + 2) * NC * NC, Wa);
            hop(q + 1, Wb);
        }
    } else {
        const E *wp = W + 2LL * n * 80 * NC * NC;
        // large N_c: one N_c x N_c buffer (the register file holds no second one)
#pragma unroll 1
        for (int q = 0; q < 80; ++q) {
            cx<A> Wm[NC][NC];
            load_mat<NC, E, A>(wp + 2 * q * NC * NC, Wm);
            hop(q, Wm);
        }
    }
    lap_write<P, NC, NS, VR, LAYOUT, E, A>(in, out, g, n, j, centre, acc);
}

template <typename E, int LAYOUT>
int launch_laplace_v(const dirac_op *op, const void *in, void *out, double m, cudaStream_t s) {
    int vr, minb, block;
    launch_variant(op, vr, minb, block);
    vr = aligned_vr(vr, op->prec, in, out);
    using A = typename Acc<E>::T;
    const bool bril = uses_w(op->kind);
    const double centre = bril ? 0.5 * m * m + 240.0 / 128.0 : 4.0 + 0.5 * m * m;
    return dispatch_nc<big_nc_ok<E>()>(op->nc, [&](auto ncc) {
        constexpr int NC = decltype(ncc)::value;
        return dispatch_vr(vr, [&](auto vrc) {
            constexpr int VR = decltype(vrc)::value;
            if constexpr (!vr_compiled<NC>(VR)) return (int)DIRAC_ERR_INVALID_ARG;
            else {
                const int nchunk = op->nv / VR;
                const long long threads = op->lat.nsites * nchunk;
                auto on_spins = [&](auto &&go) {
                    return spins_of(op->kind) == 4 ? go(std::integral_constant<int, 4>{})
                                                   : go(std::integral_constant<int, 1>{});
                };
                auto run_w = [&](auto kernel, int T, size_t smem) {
                    if (smem > 48 * 1024) {
                        const int rc = cuda_check(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                                       (int)wst::kMaxSmem),
                                                  "blap_kernel shared memory");
                        if (rc) return rc;
                    }
                    kernel<<<grid_for(threads, T), T, smem, s>>>((const E *)op->w, (const E *)in, (E *)out, op->lat,
                                                                (A)centre);
                    return launch_check("blap_kernel");
                };
                if (!bril)
                    return dispatch_minb<NC>(minb, [&](auto mbc) {
                        constexpr int MINB = decltype(mbc)::value;
                        return on_spins([&](auto nsc) {
                            constexpr int NS = decltype(nsc)::value;
                            wlap_kernel<NC, NS, VR, E, MINB, LAYOUT><<<grid_for(threads, block), block, 0, s>>>(
                                (const E *)op->links, (const E *)in, (E *)out, op->lat, (A)centre);
                            return launch_check("wlap_kernel");
                        });
                    });
                // read by each thread: FP64, bound by its own pipe (bsuv, 16^4,
                // N_c = 3, N_v = 4: 1.53 ms, staged 1.58; blap 5.77 and 5.92); and
                // N_c = 1 on site-inner vectors once four threads share the 8 bytes
                // of a matrix (blap, 16^4, N_v = 8: 72 and 75 us, 12: 115 and 124, 24:
                // 210 and 228; N_v = 4: 51 and 47; site-outer, N_v = 12: 152 and 140)
                const bool direct = sizeof(E) == 8 || (NC == 1 && LAYOUT == DIRAC_LAYOUT_SITE_INNER && VR == 2 &&
                                                       nchunk >= 4 && spins_of(op->kind) == 4);
                const size_t smem = NC <= kMaxNcSmall ? wst::smem_bytes<NC, E>(block, nchunk) : 0;
                if (NC > kMaxNcSmall || direct || nchunk < wst::kMinChunks<E> || smem > wst::kMaxSmem)
                    return on_spins([&](auto nsc) {
                        constexpr int NS = decltype(nsc)::value;
                        return run_w(blap_kernel<NC, NS, VR, E, 1, LAYOUT, false>,
                                     block <= kStencilBlock ? block : kStencilBlock, 0);
                    });
                if constexpr (NC <= kMaxNcSmall) {
                    return dispatch_minb<NC>(minb, [&](auto mbc) {
                        constexpr int MINB = decltype(mbc)::value;
                        return on_spins([&](auto nsc) {
                            constexpr int NS = decltype(nsc)::value;
                            return run_w(blap_kernel<NC, NS, VR, E, MINB, LAYOUT, true>, block, smem);
                        });
                    });
                }
                return (int)DIRAC_ERR_INVALID_ARG;
            }
        });
    });
}

}  // namespace dgb
