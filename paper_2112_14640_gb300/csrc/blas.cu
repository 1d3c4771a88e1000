// blas.cu -- multi-RHS linear algebra of Sec. 3 on the RHS-innermost layout:
// a vector is a [rows][nv] array of complex numbers (rows = sites x internal
// dofs), and every operation acts column by column with its own coefficient.
//
// Reductions (norm^2, dot) carry at least FP64-like precision whatever the
// storage precision (Sec. 3 accumulates sp norms in dp) and are
// deterministic: a fixed grid of blocks, thread (r, v) of a block owns column
// v, the threads' sums are combined in a fixed tree inside the block, and the
// blocks' rows in a fixed order by a second kernel with a block per column (in
// the CG passes by the last block to finish).  FP64 vectors accumulate in
// FP64.  FP32 and 16-bit vectors accumulate per thread in FP32 with error-free
// transformations (Dekker's product, Knuth's two-sum): every product is split
// exactly into a rounded part and its error, and the rounded parts are summed
// with their rounding errors collected in a pair (sum, error).  That keeps the
// thread loops on the FP32 pipe: FP64 arithmetic on this GPU runs at a small
// fraction of the FP32 rate and would limit the reductions far below HBM
// bandwidth.
//
// Across threads the sums are added as FP64 would or better.  FP64 additions of
// every thread's sum cost as much as a small reduction (8^4, N_v = 3: 2.3 us
// more per CG pass), so while it stays in FP32's range a column is added up as
// three floats (72 bits); a column that leaves it is added up once more, from
// the threads' own sums, in FP64.  Only a single thread's share of the rows is
// bound to the range of FP32.
//
// Every thread handles four rows per loop trip so that four independent
// 16-byte loads per operand are in flight.
#include <atomic>

#include "internal.h"

namespace dgb {

constexpr int kRedThreads = 256;

// Complex numbers per thread and per access: one 16-byte load when N_v allows.
inline int blas_group(dirac_prec p, int nv) { return pick_vr(p, nv); }

// Threads per block: a multiple of the number of column groups nv/G.
inline int red_block(int ngroups) { return ngroups * (kRedThreads / ngroups); }

// Accumulator of a real sum.  FP64 data: a plain double.  FP32 data: the
// exact value s + c (+ e) of everything added so far up to the errors of the
// error-free steps (Knuth's two-sum and Dekker's product via FMA); the explicit
// __f*_rn intrinsics keep the compiler from contracting or reassociating them.
// A thread's own sum is the pair (s, c); joining two accumulators also keeps
// the rounding errors of c, in e, so that it adds nothing to the error of an
// FP64 number.  Once s has left FP32's range it is infinite or NaN and stays so.
template <typename A>
struct RedAcc;
template <>
struct RedAcc<double> {
    double s = 0.0;
    __device__ __forceinline__ void mac(double x, double y) { s = fma(x, y, s); }
    __device__ __forceinline__ void join(const RedAcc &o) { s += o.s; }
    __device__ __forceinline__ RedAcc down(int lanes) const { return RedAcc{__shfl_down_sync(~0u, s, lanes)}; }
    __device__ __forceinline__ bool in_range() const { return true; }
    __device__ __forceinline__ double value() const { return s; }
};
template <>
struct RedAcc<float> {
    float s = 0.f, c = 0.f, e = 0.f;
    // a + b = sum + err exactly
    static __device__ __forceinline__ void two_sum(float a, float b, float &sum, float &err) {
        const float t = __fadd_rn(a, b);
        const float bp = __fsub_rn(t, a);
        err = __fadd_rn(__fsub_rn(a, __fsub_rn(t, bp)), __fsub_rn(b, bp));
        sum = t;
    }
    __device__ __forceinline__ void mac(float x, float y) {
        const float p = __fmul_rn(x, y);
        float err;
        two_sum(s, p, s, err);
        c = __fadd_rn(c, err);
        c = __fadd_rn(c, __fmaf_rn(x, y, -p));
    }
    __device__ __forceinline__ void join(const RedAcc &o) {
        float e1, e2, e3;
        two_sum(s, o.s, s, e1);
        two_sum(c, o.c, c, e2);
        two_sum(c, e1, c, e3);
        e = __fadd_rn(__fadd_rn(e, o.e), __fadd_rn(e2, e3));
    }
    __device__ __forceinline__ RedAcc down(int lanes) const {
        return RedAcc{__shfl_down_sync(~0u, s, lanes), __shfl_down_sync(~0u, c, lanes), __shfl_down_sync(~0u, e, lanes)};
    }
    __device__ __forceinline__ bool in_range() const { return fabsf(s) <= 3.4028234e38f; }
    __device__ __forceinline__ double value() const { return (double)s + ((double)c + (double)e); }
};

// A block's sum of a column as it goes to the last block of a CG pass: an
// accumulator, or an FP64 number where the accumulator has no range for it.
template <typename A>
struct RedRow;
template <>
struct RedRow<double> {
    double v;
    static __device__ __forceinline__ RedRow wide(double v) { return RedRow{v}; }
    static __device__ __forceinline__ RedRow of(const RedAcc<double> &a) { return RedRow{a.s}; }
    static __device__ __forceinline__ RedRow load(const RedRow *p) { return RedRow{__ldcg(&p->v)}; }
    __device__ __forceinline__ bool is_wide() const { return false; }
    __device__ __forceinline__ RedAcc<double> acc() const { return RedAcc<double>{v}; }
    __device__ __forceinline__ double value() const { return v; }
};
template <>
struct RedRow<float> {
    float4 v;   // s, c, e, 0; or the two words of a double, unused, 1
    static __device__ __forceinline__ RedRow wide(double d) {
        return RedRow{make_float4(__int_as_float(__double2loint(d)), __int_as_float(__double2hiint(d)), 0.f, 1.f)};
    }
    static __device__ __forceinline__ RedRow of(const RedAcc<float> &a) { return RedRow{make_float4(a.s, a.c, a.e, 0.f)}; }
    static __device__ __forceinline__ RedRow load(const RedRow *p) { return RedRow{__ldcg(&p->v)}; }
    __device__ __forceinline__ bool is_wide() const { return v.w != 0.f; }
    __device__ __forceinline__ RedAcc<float> acc() const { return RedAcc<float>{v.x, v.y, v.z}; }
    __device__ __forceinline__ double value() const {
        return is_wide() ? __hiloint2double(__float_as_int(v.y), __float_as_int(v.x)) : acc().value();
    }
};

// Rows of a column in shared memory: [column][row], an odd pitch.
__host__ __device__ constexpr int red_pitch(int rows) { return rows | 1; }

// Sum of get(0 .. rows - 1) in FP64 by one warp, in lane 0: lanes take rows
// lane, lane + 32, ..., then a fixed tree.
template <typename GET>
__device__ __forceinline__ double warp_sum(int rows, GET get) {
    double acc = 0.0;
    for (int r = threadIdx.x & 31; r < rows; r += 32) acc += get(r);
    for (int off = 16; off > 0; off /= 2) acc += __shfl_down_sync(~0u, acc, off);
    return acc;
}

// Join the `rows` sums of every column, one warp per column at a time, in the
// order of warp_sum; put(column, row) runs in lane 0.  Whole warps only
// (blocks need not be a multiple of 32 threads).
template <typename A, typename PUT>
__device__ __forceinline__ void join_columns(const RedAcc<A> *sh, int cols, int rows, PUT put) {
    const int nwarps = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp >= nwarps) return;
    for (int c = warp; c < cols; c += nwarps) {
        const RedAcc<A> *col = sh + c * red_pitch(rows);
        RedAcc<A> acc;
        for (int r = lane; r < rows; r += 32) acc.join(col[r]);
        for (int off = 16; off > 0; off /= 2) acc.join(acc.down(off));
        RedRow<A> row = RedRow<A>::of(acc);
        if (__any_sync(~0u, lane == 0 && !acc.in_range()))
            row = RedRow<A>::wide(warp_sum(rows, [&](int r) { return col[r].value(); }));
        if (lane == 0) put(c, row);
    }
}

// The sums vals[G][NOUT] of the R row-threads of a block, joined per column;
// put(v NOUT + q, row) for each.
template <int G, int NOUT, typename A, typename PUT>
__device__ __forceinline__ void block_reduce(const RedAcc<A> (&vals)[G][NOUT], RedAcc<A> *sh, int r, int vg, int R,
                                             int ng, PUT put) {
    if (r < R)
#pragma unroll
        for (int i = 0; i < G; ++i)
#pragma unroll
            for (int q = 0; q < NOUT; ++q) sh[((vg * G + i) * NOUT + q) * red_pitch(R) + r] = vals[i][q];
    __syncthreads();
    join_columns(sh, ng * G * NOUT, R, put);
}

// Second pass of a reduction: partial[b][col] (col = v*NOUT + q) -> out[col],
// one block per column, so that the columns' FP64 additions run side by side.
// The order is fixed by the number of blocks.
constexpr int kFinThreads = 256;
__global__ void __launch_bounds__(kFinThreads) finalize_kernel(const double *__restrict__ partial, int nblocks,
                                                               double *__restrict__ out) {
    __shared__ double sh[kFinThreads / 32];
    const int cols = gridDim.x, c = blockIdx.x, warp = threadIdx.x / 32;
    // warp w adds up the rows 32 w .. 32 w + 31 of every 256
    double acc = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += kFinThreads) acc += partial[(long long)b * cols + c];
    const double sum = warp_sum(32, [&](int) { return acc; });
    if (threadIdx.x % 32 == 0) sh[warp] = sum;
    __syncthreads();
    if (warp == 0) {
        const double all = warp_sum(kFinThreads / 32, [&](int w) { return sh[w]; });
        if (threadIdx.x == 0) out[c] = all;
    }
}

// thread (r, vg) of a block walks the rows r0 = block*R + r, stride grid*R and
// owns columns vg*G .. vg*G+G-1
#define BLAS_THREAD_SETUP                                   \
    const int ng = nv / G;                                  \
    const int R = blockDim.x / ng;                          \
    const int r = threadIdx.x / ng, vg = threadIdx.x % ng;  \
    const bool live = r < R;                                \
    const long long stride = (long long)gridDim.x * R;

// Rows of a reduction over part of a vector: `rows` logical rows in segments
// of seg_len, segment k starting at row k * seg_stride + seg_off (the sites
// [site0, site0 + nsites) of every component of a site-inner vector).
struct RowMap {
    long long seg_len = 0, seg_stride = 0, seg_off = 0;   // seg_len = 0: identity
    __device__ __forceinline__ long long operator()(long long row) const {
        return seg_len ? (row / seg_len) * seg_stride + seg_off + row % seg_len : row;
    }
};

template <typename E, int G>
__global__ void norm2_kernel(const E *__restrict__ x, long long rows, int nv,
                             double *__restrict__ partial, RowMap rm = RowMap{}) {
    extern __shared__ __align__(8) unsigned char red_smem[];
    using A = typename Acc<E>::T;
    RedAcc<A> *sh = reinterpret_cast<RedAcc<A> *>(red_smem);
    BLAS_THREAD_SETUP
    RedAcc<A> acc[G][1];
    auto add = [&](const cx<A> (&a)[G]) {
#pragma unroll
        for (int i = 0; i < G; ++i) {
            acc[i][0].mac(a[i].re, a[i].re);
            acc[i][0].mac(a[i].im, a[i].im);
        }
    };
    if (live) {
        long long row = (long long)blockIdx.x * R + r;
        for (; row + 3 * stride < rows; row += 4 * stride) {
            cx<A> a[4][G];
#pragma unroll
            for (int u = 0; u < 4; ++u) load_cx<E, G, A>(x + 2 * (rm(row + u * stride) * nv + vg * G), a[u]);
#pragma unroll
            for (int u = 0; u < 4; ++u) add(a[u]);
        }
        for (; row < rows; row += stride) {
            cx<A> a[1][G];
            load_cx<E, G, A>(x + 2 * (rm(row) * nv + vg * G), a[0]);
            add(a[0]);
        }
    }
    block_reduce(acc, sh, r, vg, R, ng,
                 [&](int c, const RedRow<A> &v) { partial[(long long)blockIdx.x * nv + c] = v.value(); });
}

template <typename E, int G>
__global__ void dot_kernel(const E *__restrict__ x, const E *__restrict__ y, long long rows, int nv,
                           double *__restrict__ partial, RowMap rm = RowMap{}) {
    extern __shared__ __align__(8) unsigned char red_smem[];
    using A = typename Acc<E>::T;
    RedAcc<A> *sh = reinterpret_cast<RedAcc<A> *>(red_smem);
    BLAS_THREAD_SETUP
    RedAcc<A> acc[G][2];
    auto add = [&](const cx<A> (&a)[G], const cx<A> (&b)[G]) {
#pragma unroll
        for (int i = 0; i < G; ++i) {   // conj(x) * y
            acc[i][0].mac(a[i].re, b[i].re);
            acc[i][0].mac(a[i].im, b[i].im);
            acc[i][1].mac(a[i].re, b[i].im);
            acc[i][1].mac(-a[i].im, b[i].re);
        }
    };
    if (live) {
        long long row = (long long)blockIdx.x * R + r;
        for (; row + 3 * stride < rows; row += 4 * stride) {
            cx<A> a[4][G], b[4][G];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const long long e = 2 * (rm(row + u * stride) * nv + vg * G);
                load_cx<E, G, A>(x + e, a[u]);
                load_cx<E, G, A>(y + e, b[u]);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) add(a[u], b[u]);
        }
        for (; row < rows; row += stride) {
            cx<A> a[1][G], b[1][G];
            const long long e = 2 * (rm(row) * nv + vg * G);
            load_cx<E, G, A>(x + e, a[0]);
            load_cx<E, G, A>(y + e, b[0]);
            add(a[0], b[0]);
        }
    }
    block_reduce(acc, sh, r, vg, R, ng,
                 [&](int c, const RedRow<A> &v) { partial[2LL * blockIdx.x * nv + c] = v.value(); });
}

template <typename A>
__device__ __forceinline__ cx<A> coef(const double *c, double scale, int v) {
    return c ? cx<A>{(A)(scale * c[2 * v]), (A)(scale * c[2 * v + 1])} : cx<A>{(A)scale, (A)0};
}

// z = a x + b y per column; a, b = scale * coef[v] (complex pairs) or scale
// alone when coef is null; x or y may be null (term dropped); z may alias x
// or y.  With partial != null also reduces |z|^2 per column.
template <typename E, int G>
__global__ void axpby_kernel(E *z, const E *x, const E *y, const double *__restrict__ ac, double as,
                             const double *__restrict__ bc, double bs, long long rows, int nv,
                             double *partial) {
    extern __shared__ __align__(8) unsigned char red_smem[];
    using A = typename Acc<E>::T;
    RedAcc<A> *sh = reinterpret_cast<RedAcc<A> *>(red_smem);
    BLAS_THREAD_SETUP
    cx<A> a[G], b[G];
#pragma unroll
    for (int i = 0; i < G; ++i) {
        a[i] = coef<A>(ac, as, vg * G + i);
        b[i] = coef<A>(bc, bs, vg * G + i);
    }
    RedAcc<A> acc[G][1];
    // one row: combine, store, and (optionally) add |z|^2 of the value as
    // stored: the registers rounded through the storage type (z may alias x
    // or y, so it is not re-read)
    auto finish = [&](long long e, const cx<A> (&tx)[G], const cx<A> (&ty)[G]) {
        cx<A> out[G];
#pragma unroll
        for (int i = 0; i < G; ++i) {
            out[i] = cx<A>{0, 0};
            if (x) cmac(out[i], a[i], tx[i]);
            if (y) cmac(out[i], b[i], ty[i]);
        }
        store_cx<E, G, A>(z + e, out);
        if (partial) {
#pragma unroll
            for (int i = 0; i < G; ++i) {
                const A re = (A)to_acc<E>(from_acc<E, A>(out[i].re));
                const A im = (A)to_acc<E>(from_acc<E, A>(out[i].im));
                acc[i][0].mac(re, re);
                acc[i][0].mac(im, im);
            }
        }
    };
    if (live) {
        long long row = (long long)blockIdx.x * R + r;
        for (; row + 3 * stride < rows; row += 4 * stride) {
            cx<A> tx[4][G], ty[4][G];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const long long e = 2 * ((row + u * stride) * nv + vg * G);
                if (x) load_cx<E, G, A>(x + e, tx[u]);
                if (y) load_cx<E, G, A>(y + e, ty[u]);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) finish(2 * ((row + u * stride) * nv + vg * G), tx[u], ty[u]);
        }
        for (; row < rows; row += stride) {
            const long long e = 2 * (row * nv + vg * G);
            cx<A> tx[1][G], ty[1][G];
            if (x) load_cx<E, G, A>(x + e, tx[0]);
            if (y) load_cx<E, G, A>(y + e, ty[0]);
            finish(e, tx[0], ty[0]);
        }
    }
    if (partial)
        block_reduce(acc, sh, r, vg, R, ng,
                     [&](int c, const RedRow<A> &v) { partial[(long long)blockIdx.x * nv + c] = v.value(); });
}

// ------------------------------------------------------------ CG kernels
// The three vector passes of a CG iteration with the scalar work between them
// done by the last block of the pass that produces its input: one launch each
// where a pass, its reduction's second stage and a coefficient kernel were
// three, and no value the host has to see before the next launch.  The
// iterations that the host enqueues ahead of the stop rule do nothing once it
// has been met (ctl[0]).  Memory-bound on large lattices (16^3x32, D_W,
// N_v = 4, FP32, from cold caches: dot 23, residual 27, update 37 us; the update
// moves 250 MB at 6.8 TB/s), bound by the chain load - reduce - last block on
// small ones (8^4, N_v = 3: 8, 10 and 4 us).

// Join the blocks' rows (nv sums each) in the last block to arrive; the N_v
// values there, null in every other block.  Fixed order, so reproducible.
// This block's row was written before the call.
template <typename A>
__device__ __forceinline__ const double *last_block_sum(const RedRow<A> *partial, unsigned *counter, int nv,
                                                        RedAcc<A> *sh) {
    __shared__ bool last;
    __shared__ double sums[64];
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicInc(counter, gridDim.x - 1) == gridDim.x - 1;
    __syncthreads();
    if (!last) return nullptr;
    __threadfence();
    const int T = blockDim.x / nv, t = threadIdx.x / nv, c = threadIdx.x - t * nv;
    bool wide = false;
    if (t < T) {
        RedAcc<A> acc;
        constexpr int U = 8;   // rows in flight per thread
        for (int b0 = t; b0 < (int)gridDim.x; b0 += U * T) {
            RedRow<A> in[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                in[u] = b0 + u * T < (int)gridDim.x ? RedRow<A>::load(partial + (long long)(b0 + u * T) * nv + c)
                                                    : RedRow<A>::of(RedAcc<A>{});   // zero past the last row
#pragma unroll
            for (int u = 0; u < U; ++u) {
                wide |= in[u].is_wide();
                acc.join(in[u].acc());
            }
        }
        wide |= !acc.in_range();
        sh[c * red_pitch(T) + t] = acc;
    }
    if (__syncthreads_or(wide)) {
        const int nwarps = blockDim.x >> 5, warp = threadIdx.x >> 5;
        for (int v = warp; v < nv && warp < nwarps; v += nwarps) {
            const double sum = warp_sum(gridDim.x, [&](int b) {
                return RedRow<A>::load(partial + (long long)b * nv + v).value();
            });
            if ((threadIdx.x & 31) == 0) sums[v] = sum;
        }
    } else {
        join_columns(sh, nv, T, [&](int col, const RedRow<A> &v) { sums[col] = v.value(); });
    }
    __syncthreads();
    return sums;
}

// The rows row, row + stride, ... of a thread, four at a time: batch(count,
// whole, row) takes `count` of them and skips those past the end unless
// `whole`.  Four complex numbers per access (16-bit storage) unpack to twice the
// registers that two FP32 ones take: with the skips the four rows are held at
// once (update 154 registers, one block per SM), so there whole batches are
// followed by single rows (48 registers; 32^3x16, N_v = 12, FP16: update 419 and
// 228 us, a memory rate of 6.6 TB/s).  Elsewhere the single rows at the end cost
// more (8^4, N_v = 3: 3.90 and 3.98 ms a solve).
template <int G, typename BATCH>
__device__ __forceinline__ void rows_by_four(long long row, long long stride, long long rows, BATCH batch) {
    using Four = std::integral_constant<int, 4>;
    if constexpr (G == 4) {
        for (; row + 3 * stride < rows; row += 4 * stride) batch(Four{}, std::true_type{}, row);
        for (; row < rows; row += stride) batch(std::integral_constant<int, 1>{}, std::true_type{}, row);
    } else {
        for (; row < rows; row += 4 * stride) batch(Four{}, std::false_type{}, row);
    }
}

__device__ __forceinline__ bool cg_stopped(const CgScalars &k) { return k.ctl && *(volatile int *)k.ctl; }

template <typename E, int G>
__global__ void cg_dot_kernel(const E *__restrict__ x, const E *__restrict__ y, long long rows, int nv, CgScalars k) {
    extern __shared__ __align__(8) unsigned char red_smem[];
    using A = typename Acc<E>::T;
    RedAcc<A> *sh = reinterpret_cast<RedAcc<A> *>(red_smem);
    if (cg_stopped(k)) return;
    BLAS_THREAD_SETUP
    RedAcc<A> acc[G][1];
    auto add = [&](const cx<A> (&a)[G], const cx<A> (&b)[G]) {
#pragma unroll
        for (int i = 0; i < G; ++i) {
            acc[i][0].mac(a[i].re, b[i].re);
            acc[i][0].mac(a[i].im, b[i].im);
        }
    };
    if (live)
        rows_by_four<G>((long long)blockIdx.x * R + r, stride, rows, [&](auto count, auto whole, long long row) {
            constexpr int N = decltype(count)::value;
            cx<A> a[N][G], b[N][G];
#pragma unroll
            for (int u = 0; u < N; ++u) {
                const long long e = 2 * ((row + u * stride) * nv + vg * G);
                if (whole || row + u * stride < rows) {
                    load_cx<E, G, A>(x + e, a[u]);
                    load_cx<E, G, A>(y + e, b[u]);
                }
            }
#pragma unroll
            for (int u = 0; u < N; ++u)
                if (whole || row + u * stride < rows) add(a[u], b[u]);
        });
    RedRow<A> *partial = reinterpret_cast<RedRow<A> *>(k.partial);
    block_reduce(acc, sh, r, vg, R, ng,
                 [&](int c, const RedRow<A> &v) { partial[(long long)blockIdx.x * nv + c] = v; });
    const double *sums = last_block_sum(partial, k.counter, nv, sh);
    if (!sums) return;
    const int v = threadIdx.x;
    if (v >= nv) return;
    const double pq = sums[v];
    const bool go = k.act[v] != 0.0 && (k.positive ? pq > 0.0 : pq != 0.0);
    k.pq[v] = pq;
    k.alpha[2 * v] = go ? k.rr[v] / pq : 0.0;
    k.alpha[2 * v + 1] = 0.0;
}

template <typename E, int G>
__global__ void cg_residual_kernel(E *rv, const E *__restrict__ q, long long rows, int nv, CgScalars k) {
    extern __shared__ __align__(8) unsigned char red_smem[];
    using A = typename Acc<E>::T;
    RedAcc<A> *sh = reinterpret_cast<RedAcc<A> *>(red_smem);
    if (cg_stopped(k)) return;
    BLAS_THREAD_SETUP
    A a[G];
#pragma unroll
    for (int i = 0; i < G; ++i) a[i] = live ? (A)(-k.alpha[2 * (vg * G + i)]) : (A)0;
    RedAcc<A> acc[G][1];
    // |r|^2 of the value as stored (rounded through the storage type)
    auto finish = [&](long long e, const cx<A> (&tr)[G], const cx<A> (&tq)[G]) {
        cx<A> o[G];
#pragma unroll
        for (int i = 0; i < G; ++i) {
            o[i] = cx<A>{fma(a[i], tq[i].re, tr[i].re), fma(a[i], tq[i].im, tr[i].im)};
            const A re = (A)to_acc<E>(from_acc<E, A>(o[i].re));
            const A im = (A)to_acc<E>(from_acc<E, A>(o[i].im));
            acc[i][0].mac(re, re);
            acc[i][0].mac(im, im);
        }
        store_cx<E, G, A>(rv + e, o);
    };
    if (live)
        rows_by_four<G>((long long)blockIdx.x * R + r, stride, rows, [&](auto count, auto whole, long long row) {
            constexpr int N = decltype(count)::value;
            cx<A> tr[N][G], tq[N][G];
#pragma unroll
            for (int u = 0; u < N; ++u) {
                const long long e = 2 * ((row + u * stride) * nv + vg * G);
                if (whole || row + u * stride < rows) {
                    load_cx<E, G, A>(rv + e, tr[u]);
                    load_cx<E, G, A>(q + e, tq[u]);
                }
            }
#pragma unroll
            for (int u = 0; u < N; ++u)
                if (whole || row + u * stride < rows)
                    finish(2 * ((row + u * stride) * nv + vg * G), tr[u], tq[u]);
        });
    RedRow<A> *partial = reinterpret_cast<RedRow<A> *>(k.partial);
    block_reduce(acc, sh, r, vg, R, ng,
                 [&](int c, const RedRow<A> &v) { partial[(long long)blockIdx.x * nv + c] = v; });
    const double *sums = last_block_sum(partial, k.counter, nv, sh);
    if (!sums) return;
    const int v = threadIdx.x;
    bool bad = false, pass = true, trip = false;
    if (v < nv) {
        const double rn = sums[v], ro = k.rr[v];
        const bool on = k.act[v] != 0.0;
        k.rr_prev[v] = ro;
        k.rr[v] = rn;
        k.beta[2 * v] = on && (k.positive ? ro > 0.0 : ro != 0.0) ? rn / ro : 0.0;
        k.beta[2 * v + 1] = 0.0;
        if (k.rule != CgScalars::kNone) {
            double *h = k.hist + (long long)k.ctl[1] * 3 * nv;
            h[v] = k.pq[v];
            h[nv + v] = ro;
            h[2 * nv + v] = rn;
            bad = !isfinite(rn);
            const double rnorm = sqrt(rn), goal = k.tol * sqrt(k.nb[v]);
            if (k.rule == CgScalars::kPlain) {
                pass = !on || rnorm < goal;
            } else {
                if (on) {
                    if (rnorm < k.best[v]) {
                        k.best[v] = rnorm;
                        k.since[v] = 0.0;
                    } else {
                        k.since[v] += 1.0;
                        trip = k.since[v] >= k.stall;
                    }
                    trip = trip || rnorm < k.delta * k.rmax[v] || rnorm < goal * k.sig[v];
                }
                k.rmax[v] = fmax(k.rmax[v], rnorm);
            }
        }
    }
    if (k.rule == CgScalars::kNone) return;
    const bool any_bad = __syncthreads_or(bad), any_trip = __syncthreads_or(trip);
    const bool all_pass = __syncthreads_and(pass);
    if (threadIdx.x == 0) {
        k.ctl[1] += 1;
        k.ctl[2] = 1;
        k.ctl[0] = any_bad || (k.rule == CgScalars::kPlain ? all_pass : any_trip);
    }
}

// x += alpha p, then p = r + beta p (real coefficients)
template <typename E, int G>
__global__ void cg_update_kernel(E *x, E *p, const E *__restrict__ r_, long long rows, int nv, CgScalars k) {
    using A = typename Acc<E>::T;
    if (cg_stopped(k) || (k.ctl && k.ctl[2] == 0)) return;
    BLAS_THREAD_SETUP
    if (!live) return;
    A a[G], b[G];
#pragma unroll
    for (int i = 0; i < G; ++i) {
        a[i] = (A)k.alpha[2 * (vg * G + i)];
        b[i] = (A)k.beta[2 * (vg * G + i)];
    }
    auto finish = [&](long long e, cx<A> (&xv)[G], cx<A> (&pv)[G], const cx<A> (&rv)[G]) {
#pragma unroll
        for (int i = 0; i < G; ++i) {
            rmac(xv[i], a[i], pv[i]);
            pv[i] = cx<A>{fma(b[i], pv[i].re, rv[i].re), fma(b[i], pv[i].im, rv[i].im)};
        }
        store_cx<E, G, A>(x + e, xv);
        store_cx<E, G, A>(p + e, pv);
    };
    rows_by_four<G>((long long)blockIdx.x * R + r, stride, rows, [&](auto count, auto whole, long long row) {
        constexpr int N = decltype(count)::value;
        cx<A> xv[N][G], pv[N][G], rv[N][G];
#pragma unroll
        for (int u = 0; u < N; ++u) {
            const long long e = 2 * ((row + u * stride) * nv + vg * G);
            if (whole || row + u * stride < rows) {
                load_cx<E, G, A>(x + e, xv[u]);
                load_cx<E, G, A>(p + e, pv[u]);
                load_cx<E, G, A>(r_ + e, rv[u]);
            }
        }
#pragma unroll
        for (int u = 0; u < N; ++u)
            if (whole || row + u * stride < rows)
                finish(2 * ((row + u * stride) * nv + vg * G), xv[u], pv[u], rv[u]);
    });
}

#undef BLAS_THREAD_SETUP

template <typename F>
static int dispatch_group(int g, F &&f) {
    switch (g) {
    case 1: return f(std::integral_constant<int, 1>{});
    case 2: return f(std::integral_constant<int, 2>{});
    case 4: return f(std::integral_constant<int, 4>{});
    }
    return DIRAC_ERR_INVALID_ARG;
}

// launch geometry shared by the reduction kernels: threads per block, shared bytes
struct RedLaunch {
    int G, tb;
    size_t sh;
};
static RedLaunch red_launch(dirac_prec p, int nv, int nout) {
    RedLaunch L;
    L.G = blas_group(p, nv);
    const int ng = nv / L.G;
    L.tb = red_block(ng);
    // one extra row of slots absorbs the threads beyond R (tb is a multiple of ng)
    L.sh = (size_t)(L.tb + ng) * L.G * nout * (p == DIRAC_F64 ? sizeof(RedAcc<double>) : sizeof(RedAcc<float>));
    return L;
}

template <typename E>
__global__ void gamma5_kernel(E *__restrict__ v, Lat g, int nc, int staggered, int layout) {
    const long long rows = staggered ? g.V * nc : g.V * nc * 4;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= rows * g.nv) return;
    const long long row = i / g.nv;   // (site, cs) site-outer or (cs, site) site-inner
    bool neg;
    if (staggered) {
        const Coord c = site_coords(g, layout == 0 ? row / nc : row % g.V);
        neg = (c.x + c.y + c.z + c.t) & 1;        // epsilon(n) = (-1)^(x+y+z+t)
    } else {
        const long long spin = layout == 0 ? row % 4 : (row / g.V) % 4;
        neg = spin >= 2;                          // gamma5 = diag(1, 1, -1, -1)
    }
    if (neg) {
        using A = typename Acc<E>::T;
        v[2 * i] = from_acc<E, A>(-to_acc<E>(v[2 * i]));
        v[2 * i + 1] = from_acc<E, A>(-to_acc<E>(v[2 * i + 1]));
    }
}

template <typename S, typename D>
__global__ void convert_kernel(const S *__restrict__ src, D *__restrict__ dst, long long count) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) dst[i] = from_acc<D, typename Acc<S>::T>(to_acc<S>(src[i]));
}

// A vector in the other layout (and precision): one thread per complex number
// in the order of dst.  inner: dst is [cs][site][v], src [site][cs][v]; else
// the reverse.
template <typename S, typename D>
__global__ void __launch_bounds__(256) relayout_kernel(const S *__restrict__ src, D *__restrict__ dst, long long V,
                                                       int ncs, int nv, int inner) {
    using A = typename Acc<S>::T;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= V * ncs * nv) return;
    long long row;   // the pair (site, cs) in dst's order
    int v;
    split_tid(i, nv, row, v);
    long long o;
    if (inner) {
        const long long cs = row / V;
        o = (row - cs * V) * ncs + cs;
    } else {
        long long site;
        int cs;
        split_tid(row, ncs, site, cs);
        o = cs * V + site;
    }
    const cx<A> z = ld1<S, A>(src + 2 * (o * nv + v));
    const D e[2] = {from_acc<D, A>(z.re), from_acc<D, A>(z.im)};
    if constexpr (sizeof(D) == 8) {
        *reinterpret_cast<double2 *>(dst + 2 * i) = double2{e[0], e[1]};
    } else {
        typename Raw<2 * (int)sizeof(D)>::T raw;
        __builtin_memcpy(&raw, e, sizeof(raw));
        *reinterpret_cast<decltype(raw) *>(dst + 2 * i) = raw;
    }
}

// Deterministic pseudo-random fill in [-1, 1) (a 32-bit integer hash of the
// element index), used to give timing runs realistic, non-zero operands.
template <typename E>
__global__ void fill_hash_kernel(E *__restrict__ v, long long count, unsigned seed) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    unsigned h = (unsigned)i * 2654435761u ^ seed;
    h ^= h >> 16;
    h *= 2246822519u;
    h ^= h >> 13;
    h *= 3266489917u;
    h ^= h >> 16;
    const float f = (float)(h >> 8) * (1.0f / 8388608.0f) - 1.0f;
    v[i] = from_acc<E, typename Acc<E>::T>((typename Acc<E>::T)f);
}

int blas_fill_hash(const dirac_op *op, dirac_prec p, void *v, unsigned seed, cudaStream_t s) {
    return dispatch_prec(p, [&](auto tag) {
        using E = std::remove_pointer_t<decltype(tag)>;
        const long long n = op->rows * op->nv * 2;
        fill_hash_kernel<E><<<grid_for(n, 256), 256, 0, s>>>((E *)v, n, seed);
        return launch_check("fill_hash_kernel");
    });
}

static inline int red_grid(const dirac_op *op) { return op->red_blocks; }

template <typename E>
static int launch_norm2(const E *v, long long rows, int nv, dirac_prec p, double *buf, int blocks, double *out,
                        cudaStream_t s) {
    const RedLaunch L = red_launch(p, nv, 1);
    return dispatch_group(L.G, [&](auto gc) {
        constexpr int G = decltype(gc)::value;
        norm2_kernel<E, G><<<blocks, L.tb, L.sh, s>>>(v, rows, nv, buf);
        finalize_kernel<<<nv, kFinThreads, 0, s>>>(buf, blocks, out);
        return launch_check("norm2_kernel");
    });
}

int blas_norm2(const dirac_op *op, dirac_prec p, const void *v, double *out, cudaStream_t s) {
    return dispatch_prec(p, [&](auto tag) {
        using E = std::remove_pointer_t<decltype(tag)>;
        return launch_norm2<E>((const E *)v, op->rows, op->nv, p, op->red_partial, red_grid(op), out, s);
    });
}

int blas_dot(const dirac_op *op, dirac_prec p, const void *u, const void *v, double *out, cudaStream_t s) {
    return dispatch_prec(p, [&](auto tag) {
        using E = std::remove_pointer_t<decltype(tag)>;
        const RedLaunch L = red_launch(p, op->nv, 2);
        return dispatch_group(L.G, [&](auto gc) {
            constexpr int G = decltype(gc)::value;
            dot_kernel<E, G><<<red_grid(op), L.tb, L.sh, s>>>((const E *)u, (const E *)v, op->rows, op->nv,
                                                              op->red_partial);
            finalize_kernel<<<2 * op->nv, kFinThreads, 0, s>>>(op->red_partial, red_grid(op), out);
            return launch_check("dot_kernel");
        });
    });
}

// The rows of sites [site0, site0 + nsites): one run for site-outer vectors,
// one run per internal component for site-inner ones.
static void site_rows(const dirac_op *op, long long site0, long long nsites, long long &first, long long &rows,
                      RowMap &rm) {
    const long long ncs = op->rows / op->V;
    rows = nsites * ncs;
    if (op->geom.layout == DIRAC_LAYOUT_SITE_OUTER) {
        first = site0 * ncs;
        rm = RowMap{};
    } else {
        first = 0;
        rm = RowMap{nsites, op->V, site0};
    }
}

int blas_norm2_range(const dirac_op *op, dirac_prec p, const void *v, long long site0, long long nsites, double *out,
                     cudaStream_t s) {
    long long first, rows;
    RowMap rm;
    site_rows(op, site0, nsites, first, rows, rm);
    return dispatch_prec(p, [&](auto tag) {
        using E = std::remove_pointer_t<decltype(tag)>;
        const RedLaunch L = red_launch(p, op->nv, 1);
        return dispatch_group(L.G, [&](auto gc) {
            constexpr int G = decltype(gc)::value;
            norm2_kernel<E, G><<<red_grid(op), L.tb, L.sh, s>>>((const E *)v + 2 * first * op->nv, rows, op->nv,
                                                                op->red_partial, rm);
            finalize_kernel<<<op->nv, kFinThreads, 0, s>>>(op->red_partial, red_grid(op), out);
            return launch_check("norm2_kernel");
        });
    });
}

int blas_dot_range(const dirac_op *op, dirac_prec p, const void *u, const void *v, long long site0, long long nsites,
                   double *out, cudaStream_t s) {
    long long first, rows;
    RowMap rm;
    site_rows(op, site0, nsites, first, rows, rm);
    return dispatch_prec(p, [&](auto tag) {
        using E = std::remove_pointer_t<decltype(tag)>;
        const RedLaunch L = red_launch(p, op->nv, 2);
        return dispatch_group(L.G, [&](auto gc) {
            constexpr int G = decltype(gc)::value;
            dot_kernel<E, G><<<red_grid(op), L.tb, L.sh, s>>>((const E *)u + 2 * first * op->nv,
                                                              (const E *)v + 2 * first * op->nv, rows, op->nv,
                                                              op->red_partial, rm);
            finalize_kernel<<<2 * op->nv, kFinThreads, 0, s>>>(op->red_partial, red_grid(op), out);
            return launch_check("dot_kernel");
        });
    });
}

int blas_axpby(const dirac_op *op, dirac_prec p, void *z, const void *x, const double *a, double as, const void *y,
               const double *b, double bs, double *norm_out, cudaStream_t s) {
    return dispatch_prec(p, [&](auto tag) {
        using E = std::remove_pointer_t<decltype(tag)>;
        const RedLaunch L = red_launch(p, op->nv, 1);
        return dispatch_group(L.G, [&](auto gc) {
            constexpr int G = decltype(gc)::value;
            axpby_kernel<E, G><<<red_grid(op), L.tb, L.sh, s>>>((E *)z, (const E *)x, (const E *)y, a, as, b, bs,
                                                                op->rows, op->nv,
                                                                norm_out ? op->red_partial : nullptr);
            if (norm_out) finalize_kernel<<<op->nv, kFinThreads, 0, s>>>(op->red_partial, red_grid(op), norm_out);
            return launch_check("axpby_kernel");
        });
    });
}

int blas_axpy(const dirac_op *op, dirac_prec p, const double *alpha, const void *x, void *y, cudaStream_t s) {
    return blas_axpby(op, p, y, x, alpha, 1.0, y, nullptr, 1.0, nullptr, s);
}

// Blocks of the CG passes: one row per thread on small lattices, at most
// kCgBlocks (four per SM: enough loads in flight for the memory rate, and the
// last block has few partial rows to read).
static inline int cg_grid(const dirac_op *op, const RedLaunch &L) {
    const long long want = (op->rows + L.tb / (op->nv / L.G) - 1) / (L.tb / (op->nv / L.G));
    return (int)(want < kCgBlocks ? want : kCgBlocks);
}

template <typename F>
static int dispatch_cg(const dirac_op *op, dirac_prec prec, F &&f) {
    return dispatch_prec(prec, [&](auto tag) {
        using E = std::remove_pointer_t<decltype(tag)>;
        const RedLaunch L = red_launch(prec, op->nv, 1);
        return dispatch_group(L.G, [&](auto gc) { return f((E *)nullptr, gc, L); });
    });
}

int blas_cg_dot(const dirac_op *op, dirac_prec prec, const void *p, const void *q, const CgScalars &c,
                cudaStream_t s) {
    return dispatch_cg(op, prec, [&](auto tag, auto gc, const RedLaunch &L) {
        using E = std::remove_pointer_t<decltype(tag)>;
        cg_dot_kernel<E, decltype(gc)::value><<<cg_grid(op, L), L.tb, L.sh, s>>>((const E *)p, (const E *)q, op->rows,
                                                                             op->nv, c);
        return launch_check("cg_dot_kernel");
    });
}

int blas_cg_residual(const dirac_op *op, dirac_prec prec, void *r, const void *q, const CgScalars &c,
                     cudaStream_t s) {
    return dispatch_cg(op, prec, [&](auto tag, auto gc, const RedLaunch &L) {
        using E = std::remove_pointer_t<decltype(tag)>;
        cg_residual_kernel<E, decltype(gc)::value><<<cg_grid(op, L), L.tb, L.sh, s>>>((E *)r, (const E *)q, op->rows,
                                                                                  op->nv, c);
        return launch_check("cg_residual_kernel");
    });
}

int blas_cg_update(const dirac_op *op, dirac_prec prec, void *x, void *p, const void *r, const CgScalars &c,
                   cudaStream_t s) {
    return dispatch_cg(op, prec, [&](auto tag, auto gc, const RedLaunch &L) {
        using E = std::remove_pointer_t<decltype(tag)>;
        cg_update_kernel<E, decltype(gc)::value><<<2 * cg_grid(op, L), L.tb, 0, s>>>((E *)x, (E *)p, (const E *)r, op->rows,
                                                                              op->nv, c);
        return launch_check("cg_update_kernel");
    });
}

int blas_gamma5(const dirac_op *op, dirac_prec p, void *v, cudaStream_t s) {
    return dispatch_prec(p, [&](auto tag) {
        using E = std::remove_pointer_t<decltype(tag)>;
        const long long n = op->rows * op->nv;
        gamma5_kernel<E><<<grid_for(n, 256), 256, 0, s>>>((E *)v, op->lat, op->nc, spins_of(op->kind) == 1,
                                                          op->geom.layout);
        return launch_check("gamma5_kernel");
    });
}

int blas_convert(const dirac_op *op, const void *src, dirac_prec sp, void *dst, dirac_prec dp, cudaStream_t s) {
    return dispatch_prec(sp, [&](auto stag) {
        using S = std::remove_pointer_t<decltype(stag)>;
        return dispatch_prec(dp, [&](auto dtag) {
            using D = std::remove_pointer_t<decltype(dtag)>;
            const long long n = op->rows * op->nv * 2;
            convert_kernel<S, D><<<grid_for(n, 256), 256, 0, s>>>((const S *)src, (D *)dst, n);
            return launch_check("convert_kernel");
        });
    });
}

int blas_convert_layout(const dirac_op *op, const void *src, dirac_prec sp, int src_layout, void *dst, dirac_prec dp,
                        int dst_layout, cudaStream_t s) {
    if (src_layout == dst_layout) return blas_convert(op, src, sp, dst, dp, s);
    return dispatch_prec(sp, [&](auto stag) {
        using S = std::remove_pointer_t<decltype(stag)>;
        return dispatch_prec(dp, [&](auto dtag) {
            using D = std::remove_pointer_t<decltype(dtag)>;
            relayout_kernel<S, D><<<grid_for(op->rows * op->nv, 256), 256, 0, s>>>(
                (const S *)src, (D *)dst, op->V, (int)(op->rows / op->V), op->nv,
                dst_layout == DIRAC_LAYOUT_SITE_INNER);
            return launch_check("relayout_kernel");
        });
    });
}

// ------------------------------------------------------------------------
// Allocation-free variant of the norm^2 reduction (dirac_vec_norm2_noalloc):
// the per-block partial sums go to a file-scope device array instead of the
// operator's buffer.  Host code must not pass the symbol itself to a kernel
// (in host code it names a host-side shadow, not device memory): its device
// address is looked up once per device with cudaGetSymbolAddress.
static __device__ __align__(256) double g_noalloc_partial[DIRAC_NOALLOC_MAX_BLOCKS * 64];

static double *noalloc_partial_ptr(int *rc) {
    // one cached device address per device; host threads may race on the
    // first lookup, so the slots are atomics (every racer stores the same value)
    static std::atomic<double *> addr[128];
    int dev = 0;
    *rc = cuda_check(cudaGetDevice(&dev), "cudaGetDevice");
    if (*rc) return nullptr;
    if (dev < 0 || dev >= 128) {
        *rc = DIRAC_ERR_CAPACITY;
        return nullptr;
    }
    double *p = addr[dev].load(std::memory_order_acquire);
    if (!p) {
        *rc = cuda_check(cudaGetSymbolAddress((void **)&p, g_noalloc_partial), "cudaGetSymbolAddress");
        if (*rc) return nullptr;
        addr[dev].store(p, std::memory_order_release);
    }
    return p;
}

}  // namespace dgb

extern "C" int dirac_vec_norm2_noalloc(const void *v, dirac_prec prec, long long rows, int nv, double *out_dev,
                                       void *stream) {
    using namespace dgb;
    if (!v || !out_dev || rows < 1) return DIRAC_ERR_INVALID_ARG;
    if ((uintptr_t)v & 15) return DIRAC_ERR_ALIGNMENT;
    if (prec < DIRAC_F64 || prec > DIRAC_F16) return DIRAC_ERR_UNSUPPORTED_PREC;
    if (nv < 1) return DIRAC_ERR_INVALID_ARG;
    if (nv > 64) {
        fprintf(stderr, "libdirac: dirac_vec_norm2_noalloc: nv = %d exceeds the static capacity of 64\n", nv);
        return DIRAC_ERR_CAPACITY;
    }
    int rc = DIRAC_OK;
    double *partial = noalloc_partial_ptr(&rc);
    if (rc) return rc;
    const RedLaunch L = red_launch(prec, nv, 1);
    const int R = L.tb / (nv / L.G);
    long long want = (rows + R - 1) / R;
    const int blocks = (int)(want < DIRAC_NOALLOC_MAX_BLOCKS ? want : DIRAC_NOALLOC_MAX_BLOCKS);
    cudaStream_t s = (cudaStream_t)stream;
    return dispatch_prec(prec, [&](auto tag) {
        using E = std::remove_pointer_t<decltype(tag)>;
        return launch_norm2<E>((const E *)v, rows, nv, prec, partial, blocks, out_dev, s);
    });
}
