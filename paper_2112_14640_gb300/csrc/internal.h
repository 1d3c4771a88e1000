// internal.h -- operator handle and launcher prototypes shared by the
// translation units of libdirac.so (not part of the public ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdio.h>

#include <type_traits>
#include <utility>

#include "../../include/dirac.h"
#include "common.cuh"

struct dirac_op {
    dirac_kind kind;
    dirac_geom geom;
    dgb::Lat lat;
    int nc, nv;
    dirac_prec prec;
    long long V;
    long long rows;        // complex rows per RHS column: V*nc*4 (Wilson-type) or V*nc
    size_t vec_bytes;      // bytes of one multi-RHS vector
    size_t link_bytes;     // bytes of the phased link copy
    size_t w_bytes;        // bytes of the 80 W links per site (Brillouin)
    void *links;           // [V][4][nc][nc], boundary phases folded in
    void *w;               // [V][80][nc][nc] (Brillouin only)
    void *clover;          // clover term (clover.cuh), links' shape and layout; null when c_SW = 0
    double csw;            // c_SW folded into `clover`
    void *scratch;         // one vector: intermediate of D^dag D
    void *stage_in;        // host-apply staging buffers (lazy)
    void *stage_out;
    struct dirac_host_pipe *pipe;   // host-apply copy streams and events (lazy)
    double *red_partial;   // reduction partials [red_blocks][nv][2]
    int red_blocks;
    void *solver_ws;       // solver workspace (lazy), solver_ws_bytes long
    size_t solver_ws_bytes;
    double *solver_host;   // pinned copy of a run of CG iterations' scalars (lazy)
    void *force_ws;        // Brillouin force: 216 link terms per site (lazy), force_ws_bytes long
    size_t force_ws_bytes;
    dirac_op *inner[4][2]; // lower-precision twins for mixed solves (lazy), by [prec][link storage]
    int vr, minb, block;   // stencil launch variant (RHS per thread, register class, threads per block);
                           // 0 = default
    bool variant_set;      // the variant is the caller's own (dirac_op_set_launch), not a tuned one
};

namespace dgb {

inline int cuda_check(cudaError_t e, const char *what) {
    if (e != cudaSuccess) {
        fprintf(stderr, "libdirac: %s: %s\n", what, cudaGetErrorString(e));
        cudaGetLastError();   // clear a non-sticky error so it is not blamed on a later call
        return DIRAC_ERR_CUDA;
    }
    return DIRAC_OK;
}
inline int launch_check(const char *what) { return cuda_check(cudaGetLastError(), what); }

inline size_t elem_bytes(dirac_prec p) { return p == DIRAC_F64 ? 8 : p == DIRAC_F32 ? 4 : 2; }

// precision the links and W links are stored in
inline dirac_prec link_prec(const dirac_op *op) {
    return (op->geom.link_storage == DIRAC_LINKS_F32 && (op->prec == DIRAC_BF16 || op->prec == DIRAC_F16))
               ? DIRAC_F32 : op->prec;
}

// dispatch the link element type EL for vectors of element type E
template <typename E, typename F>
int dispatch_link_elem(const dirac_op *op, F &&f) {
    if constexpr (sizeof(E) == 2) {
        if (link_prec(op) == DIRAC_F32) return f((float *)nullptr);
    }
    return f((E *)nullptr);
}

// Largest RHS-vector width (complex numbers per thread) that divides nv and
// gives at most 16-byte loads.
inline int pick_vr(dirac_prec p, int nv) {
    int vr = (int)(16 / (2 * elem_bytes(p)));
    while (vr > 1 && nv % vr) vr /= 2;
    return vr;
}

template <typename F>
int dispatch_prec(dirac_prec p, F &&f) {
    switch (p) {
    case DIRAC_F64: return f((double *)nullptr);
    case DIRAC_F32: return f((float *)nullptr);
    case DIRAC_BF16: return f((__nv_bfloat16 *)nullptr);
    case DIRAC_F16: return f((__half *)nullptr);
    }
    return DIRAC_ERR_UNSUPPORTED_PREC;
}

// Colour counts compiled: 1..8 (the paper's N_c sweep reaches 8 within this
// range).  N_c 5..8 are compiled for FP64 and FP32 storage only (BIG = false
// restricts a dispatch to 1..4, as the 16-bit stencils use it), with one RHS
// per thread and the compiler's own register choice (kMaxNcSmall below).
constexpr int kMaxNc = 8;
constexpr int kMaxNcSmall = 4;
constexpr int kTunedNc = 3;
// Products of a stencil over the Brillouin offsets: packed FP32 pairs
// (common.cuh) where the two accumulators of each of the NC NS VR components
// leave the register class (the cap of MINB, below) about 60
// registers for the rest; plain ones where they would spill, and above N_c = 4.
template <int NC, int NS, int VR, int MINB>
constexpr bool packed_fits() {
    return NC <= kMaxNcSmall && 4 * NC * NS * VR + 60 <= (MINB > 1 ? 65536 / (128 * MINB) : 208);
}
template <int NC, int NS, int VR, int MINB, typename A>
using StencilProd = Prod<A, sizeof(A) == 4 && packed_fits<NC, NS, VR, MINB>()>;
template <bool BIG = true, typename F>
int dispatch_nc(int nc, F &&f) {
    switch (nc) {
    case 1: return f(std::integral_constant<int, 1>{});
    case 2: return f(std::integral_constant<int, 2>{});
    case 3: return f(std::integral_constant<int, 3>{});
    case 4: return f(std::integral_constant<int, 4>{});
    }
    if constexpr (BIG) {
        switch (nc) {
        case 5: return f(std::integral_constant<int, 5>{});
        case 6: return f(std::integral_constant<int, 6>{});
        case 7: return f(std::integral_constant<int, 7>{});
        case 8: return f(std::integral_constant<int, 8>{});
        }
    }
    return DIRAC_ERR_UNSUPPORTED_NC;
}
// N_c compiled for a vector element type (16-bit storage: 1..4)
template <typename E>
constexpr bool big_nc_ok() { return sizeof(E) >= 4; }
inline bool nc_supported(int nc, dirac_prec p) {
    return nc >= 1 && nc <= (p == DIRAC_F64 || p == DIRAC_F32 ? kMaxNc : kMaxNcSmall);
}

// VR values compiled for NC colours: 1, 2, 4 for N_c <= 4; 1 above
template <int NC>
constexpr bool vr_compiled(int vr) { return NC <= kMaxNcSmall || vr == 1; }

template <typename F>
int dispatch_vr(int vr, F &&f) {
    switch (vr) {
    case 1: return f(std::integral_constant<int, 1>{});
    case 2: return f(std::integral_constant<int, 2>{});
    case 4: return f(std::integral_constant<int, 4>{});
    }
    return DIRAC_ERR_INVALID_ARG;
}

// Stencil launch variants: VR right-hand sides per thread and a register
// class MINB: the register cap of MINB resident 128-thread blocks per SM
// (65536 / (128 MINB) registers), compiled as __launch_bounds__(128 MINB, 1)
// so that blocks of up to 128 MINB threads can be launched with it; MINB = 1
// compiles with the plain __launch_bounds__(128) (the compiler's own register
// heuristic, which differs from an explicit minimum of one block).  Every
// (VR, MINB) pair below is compiled for N_c = 3; other N_c have MINB = 1 only.
// Larger blocks cover more consecutive x-rows, so more of the y-neighbours a
// block reads are already in its SM's L1.
constexpr int kStencilBlock = 128;
__host__ __device__ constexpr int stencil_max_threads(int minb) { return minb > 1 ? 128 * minb : 128; }
inline bool variant_compiled(int nc, int vr, int minb) {
    if (vr != 1 && vr != 2 && vr != 4) return false;
    if (nc > kMaxNcSmall) return vr == 1 && minb == 1;
    if (minb == 1) return true;
    return nc == 3 && (minb >= 3 && minb <= 6);
}
inline bool variant_ok(const dirac_op *op, int vr, int minb) {
    return variant_compiled(op->nc, vr, minb) && op->nv % vr == 0;
}

// Second launch bound of a stencil.  N_c = 3 has its register classes (MINB);
// the other N_c are compiled once, and there the compiler left to itself often
// holds few loads in flight (D_W at N_c = 4, VR = 1: 86 registers, 0.525 ms at
// 16^3x32, N_v = 24; 128 registers: 0.328 ms).  Where it measured faster
// (`bound`) they get the registers for what a thread keeps: NC NS VR
// accumulators, `extra` further complex numbers (neighbour components, the
// link), and about 40 for addresses.  16^4, N_v = 12, FP32, without and with:
// D_W N_c = 2: 39 and 35 us, 4: 103 and 85 (N_c = 1: 14.9 and 16.0, N_c = 6,
// N_v = 5: 109 and 117, left alone); D_S N_c = 2: 14 and 12, 4: 35 and 29, 6:
// 119 and 111 (N_c = 1: 9.7 and 12.3); the Laplacian wlap N_c = 2: 39 and 36
// (N_c = 4, VR = 1: 102 and 113); blap N_c = 4: 125 and 118 on 8^3x16, and on
// 12^3x16 N_c = 5, N_v = 6: 550 and 371 (N_c = 6: 565 and 661, left alone; N_c = 2:
// 47 and 49); bsuv N_c = 6, N_v = 8: 370 and 310, N_v = 3: 369 and 431, 7: 552 and
// 412 (N_c = 5, N_v = 8: 294 and 226, but N_v = 3: 261 and 313, 4: 217 and 237, 6:
// 268 and 345, left alone).
template <int NC, int NS, int VR, int MINB, typename A>
constexpr int stencil_min_blocks(bool bound, int extra) {
    if (MINB > 1) return 1;
    if (NC == kTunedNc || !bound) return 0;
    const int need = 2 * (NC * NS * VR + extra) * (int)(sizeof(A) / 4) + 40;
    const int b = 65536 / (128 * need);
    return b < 1 ? 1 : b > 8 ? 8 : b;
}

template <typename F>
int dispatch_layout(int layout, F &&f) {
    switch (layout) {
    case DIRAC_LAYOUT_SITE_OUTER: return f(std::integral_constant<int, 0>{});
    case DIRAC_LAYOUT_SITE_INNER: return f(std::integral_constant<int, 1>{});
    }
    return DIRAC_ERR_INVALID_ARG;
}

template <int NC, typename F>
int dispatch_minb(int minb, F &&f) {
    if constexpr (NC != 3) {
        return minb == 1 ? f(std::integral_constant<int, 1>{}) : DIRAC_ERR_INVALID_ARG;
    } else {
        switch (minb) {
        case 1: return f(std::integral_constant<int, 1>{});
        case 3: return f(std::integral_constant<int, 3>{});
        case 4: return f(std::integral_constant<int, 4>{});
        case 5: return f(std::integral_constant<int, 5>{});
        case 6: return f(std::integral_constant<int, 6>{});
        }
        return DIRAC_ERR_INVALID_ARG;
    }
}

// kind properties: the Laplace operators -1/2 Lap + m^2/2 (hermitian), the
// number of spin components per colour of the kind's vectors, and whether the
// kind stencils with the 80 Brillouin W links
inline bool is_laplace(dirac_kind k) { return k >= DIRAC_WLAP && k <= DIRAC_BSUV; }
inline int spins_of(dirac_kind k) { return (k == DIRAC_STAGGERED || k == DIRAC_WSUV || k == DIRAC_BSUV) ? 1 : 4; }
inline bool uses_w(dirac_kind k) { return k == DIRAC_BRILLOUIN || k == DIRAC_BLAP || k == DIRAC_BSUV; }

// (vr, minb, block) an operator launches with: its tuned choice or the default.
inline void launch_variant(const dirac_op *op, int &vr, int &minb, int &block) {
    if (op->vr) {
        vr = op->vr;
        minb = op->minb ? op->minb : 1;
        block = op->block ? op->block : kStencilBlock;
        return;
    }
    // untuned: the widest 16-byte RHS group and, for N_c = 3, the register
    // class and block size the autotuner picks for FP32 on 16^3x32 lattices
    vr = op->nc > kMaxNcSmall ? 1 : pick_vr(op->prec, op->nv);
    minb = 1;
    block = kStencilBlock;
    // D_S reads 24 N_v bytes a site beside 72 of links per hop: the widest
    // group of one 32-byte access spreads a link over the most RHS (16^3x32,
    // N_v = 12, FP32: 36 us, two RHS per thread 41 us; 16^4, N_v = 8: 12.4 and
    // 14.3), while that leaves two warps per quarter-SM (D^dag D on 14x8x26x8,
    // N_v = 4: 15.1 us, two RHS 12.6)
    if (op->kind == DIRAC_STAGGERED && op->prec == DIRAC_F32 && op->nc <= kMaxNcSmall && op->nv % 4 == 0 &&
        op->V * op->nv / 4 >= 2 * 608 * 32)
        vr = 4;
    // D_S classes: 16^3x32, N_v = 8, BF16 23.1 us with FP32 links in class 3 (24.8 in
    // 5), 24.9 with BF16 links in class 5 (26.9 in 3); FP64 takes the same time in
    // 6 as in 3 (16^4, N_v = 1 to 12)
    if (op->nc == 3) {
        if (op->kind == DIRAC_WILSON) minb = vr == 4 ? 3 : 4;
        else if (op->kind == DIRAC_STAGGERED) minb = vr == 4 ? (link_prec(op) != op->prec ? 3 : 5) : 6;
    }
    // 81-point stencils on 4 spins in FP32 arithmetic: two accumulators per
    // component (common.cuh), so one RHS per thread from N_c = 3 on (16^3x32,
    // N_v = 12, D_B: 1.07 ms, two RHS 1.06 ms at 8 warps per SM; the Brillouin
    // Laplacian 0.94 against 1.13 ms).  16-bit vectors too: their loads shrink to
    // 4 bytes, but four RHS per thread, as before, took longer everywhere (16^4,
    // FP16, N_v = 4: 250 and 534 us, 12: 705 and 970; with FP32 links 623 and 1344).
    // FP64 keeps one RHS per thread in the compiler's own registers (in 384-thread
    // blocks of class 3, as before, 16^4, N_c = 3, N_v = 1: 3.17 ms, now 2.13; 4: 7.91
    // and 7.43; 12: 22.1 and 21.6; N_c = 4 had this form before and loses 3% below
    // N_v = 12 by the row order: 12^3x16, N_v = 4: 5.18 and 5.35)
    if (uses_w(op->kind) && spins_of(op->kind) == 4 && op->prec != DIRAC_F64 && op->nc <= kMaxNcSmall) {
        vr = op->nc >= 3 || vr == 1 ? 1 : 2;
        if (op->nc == 3) minb = 4;
    }
    // bsuv with few threads per site: with the compiler's own choice of registers
    // a block holds fewer warps than its ring allows (18x10x14x14, N_v = 3: 88 us,
    // with a class 66; 13x9x5x4, N_v = 5: 32 and 19; but 22x13x25x4, N_v = 23: 171
    // and 207)
    if (op->kind == DIRAC_BSUV && op->prec == DIRAC_F32 && op->nc == 3 && op->nv / vr < 8) minb = 4;
}

// VR complex numbers of an element are one access of up to 32 bytes, which
// needs that alignment; vectors are only required to be 16-byte aligned, so a
// launch on less aligned ones takes the widest group of 16 bytes instead.
inline int aligned_vr(int vr, dirac_prec p, const void *in, const void *out) {
    const int most = (int)(16 / (2 * elem_bytes(p)));
    return vr > most && (((uintptr_t)in | (uintptr_t)out) & 31) ? most : vr;
}

inline unsigned grid_for(long long threads, int block) {
    return (unsigned)((threads + block - 1) / block);
}

// stencils (sgn = +1: D, -1: D^dag)
int launch_wilson(const dirac_op *op, const void *in, void *out, double m0, int sgn, cudaStream_t s);
int launch_staggered(const dirac_op *op, const void *in, void *out, double m0, int sgn, cudaStream_t s);
int launch_brillouin(const dirac_op *op, const void *in, void *out, double m0, int sgn, cudaStream_t s);
// A = -1/2 Lap + m^2/2 for the Laplace kinds (laplace.cuh); m is the mass of A
int launch_laplace(const dirac_op *op, const void *in, void *out, double m, cudaStream_t s);

// FP64 applies on small lattices with the hops of a site spread over lanes (split.cu)
bool split_applies(const dirac_op *op);
int launch_split(const dirac_op *op, const void *in, void *out, double m0, int sgn, cudaStream_t s);

// link preparation
int launch_phase_links(dirac_op *op, const void *U, dirac_prec u_prec, cudaStream_t s);
int launch_build_w(dirac_op *op, const void *U, dirac_prec u_prec, cudaStream_t s);
// one stout-smearing step of a periodic field [site][mu][a][b] (F64 or F32)
int launch_stout_step(const void *U, void *out, const Lat &g, int nc, dirac_prec prec, double rho, cudaStream_t s);
// chain rule through nsteps stout steps (links.cu): G_V -> G_U, GRAD convention; synchronises s
int launch_stout_backward(const void *U, const void *G_V, void *G_U, const Lat &g, int nc, dirac_prec prec, double rho,
                          int nsteps, cudaStream_t s);
// clover term of c_SW = op->csw from gauge field V into op->clover (allocated)
int launch_build_clover(dirac_op *op, const void *V, dirac_prec v_prec, cudaStream_t s);
// the stored W~ (order and scale of bril_dirs.h) back to W_s in the public order
int launch_unpack_w(const dirac_op *op, void *out, cudaStream_t s);
int launch_convert_links(const dirac_op *src, dirac_op *dst, cudaStream_t s);
// Brillouin fermion force (force_bril.cu): F = P_TA(U K) (mode 0) or G = bc K^dag (mode 1)
int launch_bril_force(dirac_op *op, const void *psi, const void *chi, void *out, int mode, cudaStream_t s);

// BLAS-1 (vectors in precision p with op's shape)
int blas_norm2(const dirac_op *op, dirac_prec p, const void *v, double *out, cudaStream_t s);
int blas_dot(const dirac_op *op, dirac_prec p, const void *u, const void *v, double *out, cudaStream_t s);
int blas_norm2_range(const dirac_op *op, dirac_prec p, const void *v, long long site0, long long nsites, double *out,
                     cudaStream_t s);
int blas_dot_range(const dirac_op *op, dirac_prec p, const void *u, const void *v, long long site0, long long nsites,
                   double *out, cudaStream_t s);
int blas_axpy(const dirac_op *op, dirac_prec p, const double *alpha, const void *x, void *y, cudaStream_t s);
// z = a x + b y per RHS; a = as * a_coef[v] (complex pairs) or as when a_coef is null (same for b);
// x or y may be null; z may alias x or y; norm_out (device, nv doubles) receives |z|^2 if non-null.
int blas_axpby(const dirac_op *op, dirac_prec p, void *z, const void *x, const double *a_coef, double as,
               const void *y, const double *b_coef, double bs, double *norm_out, cudaStream_t s);
// Device scalars of a CG recurrence, nv doubles each unless noted, and the
// rule by which the device ends a run of iterations that the host enqueued
// ahead (blas.cu).
struct CgScalars {
    double *rr, *rr_prev, *pq, *alpha, *beta;   // alpha, beta: (re, im) pairs, im = 0
    const double *act;                          // 0: frozen RHS
    enum Rule { kNone, kPlain, kReliable } rule;
    bool positive;                              // steps only where <p, A p> and |r|^2 are > 0 (not just nonzero)
    // kPlain: stop once every active |r| < tol |b|; kReliable: once one falls
    // below delta rmax or tol |b| sig, or has not improved for `stall`
    // iterations; both: on a NaN or infinity
    double tol, delta;
    int stall;
    const double *nb, *sig;
    double *best, *rmax, *since;
    // [0] stopped, [1] iterations done since both were cleared, [2] an update
    // of x and p is due (alpha and beta of the last iteration not yet used)
    int *ctl;
    double *hist;         // per iteration: <p, A p>, old |r|^2, new |r|^2 (3 nv)
    double *partial;      // per block a row of nv sums (16 bytes each, 16-byte aligned)
    unsigned *counter;    // zero between launches
};
// pq = Re <p, q> and alpha = rr / pq
int blas_cg_dot(const dirac_op *op, dirac_prec prec, const void *p, const void *q, const CgScalars &c, cudaStream_t s);
// iterations of history `hist` holds, and the blocks `partial` has rows for
constexpr int kCgHistory = 20, kCgBlocks = 608;
// r -= alpha q; rr_prev = rr, rr = |r|^2, beta = rr / rr_prev, history and stop rule
int blas_cg_residual(const dirac_op *op, dirac_prec prec, void *r, const void *q, const CgScalars &c, cudaStream_t s);
// x += alpha p, p = r + beta p, if due and not stopped (always where c.ctl is null)
int blas_cg_update(const dirac_op *op, dirac_prec prec, void *x, void *p, const void *r, const CgScalars &c,
                   cudaStream_t s);
int blas_gamma5(const dirac_op *op, dirac_prec p, void *v, cudaStream_t s);
int blas_fill_hash(const dirac_op *op, dirac_prec p, void *v, unsigned seed, cudaStream_t s);
int blas_convert(const dirac_op *op, const void *src, dirac_prec sp, void *dst, dirac_prec dp, cudaStream_t s);

// the same between layouts (DIRAC_LAYOUT_*)
int blas_convert_layout(const dirac_op *op, const void *src, dirac_prec sp, int src_layout, void *dst, dirac_prec dp,
                        int dst_layout, cudaStream_t s);

// CG scalars of the operator's solver workspace (solver.cu), no stop rule set
int solver_cg(const dirac_op *op, void **vecs, int nvecs, CgScalars *c, cudaStream_t s);
// q = A p and alpha = rr / <p, q>
int solver_cg_step(const dirac_op *op, const void *p, void *q, double m0, const CgScalars &c, cudaStream_t s);
// beta = rr_new / rr_prev and rr = rr_new, after rr_new was recomputed
int solver_cg_beta(const dirac_op *op, const double *rr_new, const CgScalars &c, cudaStream_t s);

// operator handle helpers (capi.cu)
int op_apply(const dirac_op *op, const void *in, void *out, double m0, int sgn, cudaStream_t s);
int op_apply_normal(const dirac_op *op, const void *in, void *out, double m0, cudaStream_t s);
// the operator CG iterates with: D^dag D, or A itself for the (hermitian) Laplace kinds
int op_apply_cg(const dirac_op *op, const void *in, void *out, double m0, cudaStream_t s);
int op_alloc(dirac_kind kind, const dirac_geom *g, dirac_op **out);
int op_inner(const dirac_op *op, dirac_prec p, int link_storage, dirac_op **out, cudaStream_t s);
// The same operator on site-inner vectors, the order the solvers iterate in: a
// view that shares op's links and buffers and must not outlive the call.
dirac_op op_site_inner(const dirac_op *op);
void op_destroy(dirac_op *op);

}  // namespace dgb
