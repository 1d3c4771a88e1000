// hypercube.cuh -- the 80 offsets s in {-1,0,1}^4 \ {0} as a table for the
// kernels that walk the 3^4 hypercube around a site level by level (the W
// builder in links.cu and the Brillouin force in force_bril.cu), and the tile
// of sites such a kernel works on.
//
// Both kernels put consecutive sites on consecutive lanes: a block owns S
// sites, thread t works on site t % S, and t / S picks one offset of the
// level.  Every link and every stored matrix is then read and written by
// neighbouring lanes at neighbouring addresses ([..][element][site], as the
// links are stored), and the matrices of the recursion sit in shared memory
// as [matrix][element][site], free of bank conflicts.
#pragma once
#include "bril_dirs.h"
#include "internal.h"

namespace dgb {
namespace hyper {

// Offsets sorted by level k = |s|_1 (8, 24, 32, 16 of them).
__host__ __device__ constexpr int level_begin(int k) { return k <= 1 ? 0 : k == 2 ? 8 : k == 3 ? 32 : k == 4 ? 64 : 80; }

struct Offset {
    signed char s[4];
    unsigned char k;
    unsigned char q;         // storage index of W~ (bril_dirs.h)
    unsigned char mu[4];     // the axes s moves along, ascending; k of them
    unsigned char prev[4];   // position in this table of s - s_mu mu (0 when that is the centre)
    // the offsets s +- mu one level up, for the 4 - k axes s does not move
    // along: axis, sign and position in this table
    unsigned char cmu[6], child[6];
    signed char csign[6];
};
struct Table {
    Offset o[80];
    int pos[81];             // position of the offset d = (st+1)*27 + (sz+1)*9 + (sy+1)*3 + (sx+1); -1: centre
};

__host__ __device__ constexpr int dir_index(const signed char *s) {
    return (s[3] + 1) * 27 + (s[2] + 1) * 9 + (s[1] + 1) * 3 + (s[0] + 1);
}

__host__ __device__ constexpr Table make_table() {
    Table t{};
    const int pow3[4] = {1, 3, 9, 27};
    int i = 0;
    t.pos[40] = -1;
    for (int k = 1; k <= 4; ++k)
        for (int d = 0; d < 81; ++d) {
            const int s[4] = {d % 3 - 1, (d / 3) % 3 - 1, (d / 9) % 3 - 1, d / 27 - 1};
            if ((s[0] != 0) + (s[1] != 0) + (s[2] != 0) + (s[3] != 0) != k) continue;
            Offset &o = t.o[i];
            int j = 0;
            for (int mu = 0; mu < 4; ++mu) {
                o.s[mu] = (signed char)s[mu];
                if (s[mu]) o.mu[j++] = (unsigned char)mu;
            }
            double scale = 0;
            o.k = (unsigned char)k;
            o.q = (unsigned char)bril::store_index(s, &scale);
            t.pos[d] = i++;
        }
    for (i = 0; i < 80; ++i) {
        Offset &o = t.o[i];
        const int d = dir_index(o.s);
        for (int j = 0; j < o.k; ++j) {
            const int p = t.pos[d - o.s[o.mu[j]] * pow3[o.mu[j]]];
            o.prev[j] = (unsigned char)(p < 0 ? 0 : p);
        }
        int c = 0;
        for (int mu = 0; mu < 4; ++mu)
            for (int sg = -1; sg <= 1 && o.s[mu] == 0; sg += 2) {
                o.cmu[c] = (unsigned char)mu;
                o.csign[c] = (signed char)sg;
                o.child[c++] = (unsigned char)t.pos[d + sg * pow3[mu]];
            }
    }
    return t;
}
static __constant__ Table kTable = make_table();

// Sites per block: the largest power of two whose `mats` matrices per site
// leave room for two blocks in an SM's 227 KB of shared memory.
__host__ __device__ constexpr int tile_pad(int S) { return S >= 8 ? S + 1 : S; }
__host__ __device__ constexpr int tile_sites(int mats, int nc, int cx_bytes, bool padded) {
    for (int S = 32; S > 1; S /= 2)
        if ((long long)mats * nc * nc * (padded ? tile_pad(S) : S) * cx_bytes <= 112 * 1024) return S;
    return 1;
}
constexpr int kThreads = 256;

// Index steps of +1 and -1 along each axis from one site (periodic).
struct Steps {
    int p[4], m[4];
};
__device__ __forceinline__ Steps steps_at(const Lat &g, long long n) {
    const Coord c = site_coords(g, n);
    const int co[4] = {c.x, c.y, c.z, c.t};
    const int ext[4] = {g.nx, g.ny, g.nz, g.nt};
    Steps st;
    int stride = 1;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        st.p[mu] = (co[mu] == ext[mu] - 1 ? -(ext[mu] - 1) : 1) * stride;
        st.m[mu] = (co[mu] == 0 ? ext[mu] - 1 : -1) * stride;
        stride *= ext[mu];
    }
    return st;
}
// index step of the whole offset s, and of one axis picked at run time
__device__ __forceinline__ int step_of(const Steps &st, const signed char *s) {
    int d = 0;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) d += s[mu] > 0 ? st.p[mu] : (s[mu] < 0 ? st.m[mu] : 0);
    return d;
}
__device__ __forceinline__ int pick(const int (&v)[4], int mu) {
    return mu == 0 ? v[0] : mu == 1 ? v[1] : mu == 2 ? v[2] : v[3];
}

// The operator's own phased links (storage of common.cuh), in the arithmetic
// type AB; dag: the adjoint.
template <int NC, typename E, typename AB>
struct NativeLinks {
    const E *U;
    __device__ __forceinline__ void load(long long site, int mu, bool dag, cx<AB> (&L)[NC][NC]) const {
        const E *p = U + 2 * link_index(site, 4, NC * NC, mu, 0);
        constexpr long long st = 2 * link_stride(NC * NC);
#pragma unroll
        for (int a = 0; a < NC; ++a)
#pragma unroll
            for (int b = 0; b < NC; ++b) {
                // the adjoint as selects on one set of loads (dag differs between the lanes of a warp)
                const cx<AB> u = ld1<E, AB>(p + st * (dag ? b * NC + a : a * NC + b));
                L[a][b] = cx<AB>{u.re, dag ? -u.im : u.im};
            }
    }
    __device__ __forceinline__ cx<AB> at(long long site, int mu, bool dag, int a, int b) const {
        const cx<AB> u = ld1<E, AB>(U + 2 * (link_index(site, 4, NC * NC, mu, 0) +
                                             (long long)link_stride(NC * NC) * (dag ? b * NC + a : a * NC + b)));
        return cx<AB>{u.re, dag ? -u.im : u.im};
    }
};

// One level of the recursion W_s(n) = (1/K) sum_mu W_{s - s_mu mu}(n) V_{s_mu mu}(n + s - s_mu mu)
// for the sites of a tile: mats[row(o) N_c^2 + e][lane], rows STRIDE lanes
// long, row(o) the caller's numbering of the offsets.  Ends with a barrier.
template <int K, int NC, int STRIDE, int NW, typename AB, typename SRC, typename ROW>
__device__ __forceinline__ void w_level(cx<AB> *mats, const SRC &src, long long n, const Steps &st, int lane,
                                        int worker, ROW row) {
    constexpr int NN = NC * NC, B0 = level_begin(K), CNT = level_begin(K + 1) - B0;
    const AB inv = (AB)1 / (AB)K;
    // site of the link of the term along axis j: n + s, one step back where s_mu > 0
    auto link_site = [&](const Offset &o, int full, int j, int &mu, bool &dag) {
        mu = o.mu[j];
        dag = o.s[mu] < 0;
        return n + full - (dag ? 0 : pick(st.p, mu));
    };
    if constexpr (NC <= kMaxNcSmall) {
        for (int i = worker; i < CNT; i += NW) {
            const Offset &o = kTable.o[B0 + i];
            const int full = step_of(st, o.s);
            cx<AB> acc[NC][NC];
            // FP32: all K links requested before the first product
            constexpr int AHEAD = sizeof(AB) == 4 ? K : 1;
            cx<AB> L[AHEAD][NC][NC];
            int mu;
            bool dag;
#pragma unroll
            for (int j = 0; j < AHEAD; ++j) {
                const long long site = link_site(o, full, j, mu, dag);
                src.load(site, mu, dag, L[j]);
            }
            if constexpr (K == 1) {
#pragma unroll
                for (int a = 0; a < NC; ++a)
#pragma unroll
                    for (int b = 0; b < NC; ++b) acc[a][b] = L[0][a][b];
            } else {
#pragma unroll
                for (int a = 0; a < NC; ++a)
#pragma unroll
                    for (int b = 0; b < NC; ++b) acc[a][b] = cx<AB>{0, 0};
#pragma unroll
                for (int j = 0; j < K; ++j) {
                    if (AHEAD == 1 && j > 0) {
                        const long long site = link_site(o, full, j, mu, dag);
                        src.load(site, mu, dag, L[0]);
                    }
                    const cx<AB>(&Lj)[NC][NC] = L[AHEAD == 1 ? 0 : j];
                    const cx<AB> *P = mats + (row(o.prev[j]) * NN) * STRIDE + lane;
#pragma unroll
                    for (int a = 0; a < NC; ++a)
#pragma unroll
                        for (int c = 0; c < NC; ++c) {
                            const cx<AB> w = P[(a * NC + c) * STRIDE];
#pragma unroll
                            for (int b = 0; b < NC; ++b) cmac(acc[a][b], w, Lj[c][b]);
                        }
                }
            }
            cx<AB> *O = mats + (row(B0 + i) * NN) * STRIDE + lane;
#pragma unroll
            for (int a = 0; a < NC; ++a)
#pragma unroll
                for (int b = 0; b < NC; ++b) O[(a * NC + b) * STRIDE] = K == 1 ? acc[a][b] : inv * acc[a][b];
        }
    } else {
        // large N_c: one row of W_s per task, the link read element by element
        for (int i = worker; i < CNT * NC; i += NW) {
            const Offset &o = kTable.o[B0 + i / NC];
            const int a = i % NC, full = step_of(st, o.s);
            cx<AB> acc[NC];
#pragma unroll
            for (int b = 0; b < NC; ++b) acc[b] = cx<AB>{0, 0};
            for (int j = 0; j < K; ++j) {
                int mu;
                bool dag;
                const long long site = link_site(o, full, j, mu, dag);
                const cx<AB> *P = mats + (row(o.prev[j]) * NN + a * NC) * STRIDE + lane;
#pragma unroll 1
                for (int c = 0; c < NC; ++c) {
                    const cx<AB> w = K == 1 ? cx<AB>{(AB)(a == c), (AB)0} : P[c * STRIDE];
#pragma unroll
                    for (int b = 0; b < NC; ++b) cmac(acc[b], w, src.at(site, mu, dag, c, b));
                }
            }
            cx<AB> *O = mats + (row(B0 + i / NC) * NN + a * NC) * STRIDE + lane;
#pragma unroll
            for (int b = 0; b < NC; ++b) O[b * STRIDE] = inv * acc[b];
        }
    }
    __syncthreads();
}

}  // namespace hyper
}  // namespace dgb
