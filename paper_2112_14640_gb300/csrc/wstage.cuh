// wstage.cuh -- the W~ of a block's sites in shared memory, for the stencils
// over the 80 Brillouin offsets (brillouin.cuh, laplace.cuh).
//
// The N_v / VR threads of a site all need the same N_c x N_c matrices.  Read
// from global memory by each of them, one element of W~ is a warp-wide load
// that touches as many cache lines as the warp covers sites, and these loads
// and the neighbour spinors together keep the L1 pipe as busy as the FP32
// pipe; they also push the spinors out of L1.  Here the block copies W~ once
// with cp.async (L1 bypassed), a few offsets per stage, three stages in the
// ring: one in use, one arriving, one being requested.  The matrices of one
// site are contiguous in visiting order (bril_dirs.h), so a stage is one
// contiguous run per site.  Stage 0 is the two offsets of R = 0, the other 13
// stages are two rows (six offsets) each.
#pragma once
#include "bril_dirs.h"
#include "internal.h"

namespace dgb {
namespace wst {

constexpr int kStages = 14, kRing = 3;

template <int NC, typename EL>
struct Shape {
    static constexpr int mat = NC * NC * 2 * (int)sizeof(EL);   // bytes of one matrix
    static constexpr int bytes = 6 * mat, first = 2 * mat;      // of a stage, of stage 0
    // widest copy that divides every run and every run's start
    static constexpr int chunk = (bytes % 16 == 0 && first % 16 == 0) ? 16 : 8;
    static_assert(bytes % chunk == 0 && first % chunk == 0 && (80 * mat) % chunk == 0, "W~ stage runs");
    // distance of two sites in a stage: an odd multiple of 16 bytes, so that
    // the sites of a warp fall on different banks
    static constexpr int pitch = bytes + ((bytes % 32 == 0) ? 16 : 0);
};

// sites a block of T threads can touch at nchunk threads per site
__host__ __device__ inline int block_sites(int T, int nchunk) { return (T - 1) / nchunk + 2; }
template <int NC, typename EL>
inline size_t smem_bytes(int T, int nchunk) {
    return (size_t)kRing * block_sites(T, nchunk) * Shape<NC, EL>::pitch;
}
// Staging pays wherever a block's ring leaves room for two blocks per SM, also
// with few threads per site: FP32, N_c = 3, 18x10x14x14, read by each thread
// and staged: D_B N_v = 3: 168 and 113 us, N_v = 2: 124 and 96, blap N_v = 3: 168
// and 109, bsuv N_v = 3: 120 and 88; N_c = 2, N_v = 2, 31x14x15x18: 224 and 150.
// (N_c = 3, N_v = 1 does not fit.)  FP64 is bound by its own pipe and D_B gains
// little: there only where four threads share a site, as the ring of fewer is
// too large at N_c = 3 (ms, read by each thread and staged: 16^4, N_c = 3, N_v = 4:
// 7.37 and 7.43, 12: 21.54 and 21.64; 12^3x16, N_v = 12, N_c = 2: 4.92 and 4.88, 4: 15.91
// and 15.42); the Laplacians in FP64 never (laplace.cuh).
template <typename EL>
constexpr int kMinChunks = sizeof(EL) == 8 ? 4 : 1;
constexpr size_t kMaxSmem = 100 * 1024;

template <int BYTES>
__device__ __forceinline__ void cp_async(unsigned dst, const void *src) {
    if constexpr (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}

// The ring of one block: sites s0 .. s0 + nsites - 1.
template <int NC, typename EL>
struct Ring {
    using S = Shape<NC, EL>;
    const unsigned char *src;   // W~ of site s0
    unsigned char *smem;
    int nsites, slots;          // sites copied, sites a stage has room for
    int mine;                   // this thread's site, counted from s0

    template <int LEN>
    __device__ __forceinline__ void copy(unsigned dst, const unsigned char *g) {
        for (int i = threadIdx.x; i < nsites * LEN; i += blockDim.x) {
            const int site = i / LEN, c = i - site * LEN;
            cp_async<S::chunk>(dst + site * S::pitch + c * S::chunk, g + (long long)site * (80 * S::mat) + c * S::chunk);
        }
    }
    __device__ __forceinline__ void request(int stage) {
        if (stage < kStages) {
            const unsigned dst = (unsigned)__cvta_generic_to_shared(smem + (stage % kRing) * slots * S::pitch);
            if (stage == 0) copy<S::first / S::chunk>(dst, src);
            else copy<S::bytes / S::chunk>(dst, src + S::first + (stage - 1) * S::bytes);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    __device__ __forceinline__ void start() {
        request(0);
        request(1);
    }
    // Make `stage` readable by the whole block and request the one after the next.
    __device__ __forceinline__ const EL *enter(int stage) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();   // every thread's copies of this stage have landed; slot (stage + 2) % 3 is free
        request(stage + 2);
        return reinterpret_cast<const EL *>(smem + ((stage % kRing) * slots + mine) * S::pitch);
    }
};

// one matrix of the current stage
template <int NC, typename EL, typename A>
__device__ __forceinline__ void load_mat_shared(const EL *p, cx<A> (&M)[NC][NC]) {
#pragma unroll
    for (int a = 0; a < NC; ++a)
#pragma unroll
        for (int b = 0; b < NC; ++b) {
            const EL *q = p + 2 * (a * NC + b);
            if constexpr (sizeof(EL) == 8) {
                const double2 d = *reinterpret_cast<const double2 *>(q);
                M[a][b] = cx<A>{(A)d.x, (A)d.y};
            } else if constexpr (sizeof(EL) == 4) {
                const float2 f = *reinterpret_cast<const float2 *>(q);
                M[a][b] = cx<A>{(A)f.x, (A)f.y};
            } else {
                const unsigned raw = *reinterpret_cast<const unsigned *>(q);
                EL e[2];
                __builtin_memcpy(e, &raw, 4);
                M[a][b] = cx<A>{(A)to_acc<EL>(e[0]), (A)to_acc<EL>(e[1])};
            }
        }
}

}  // namespace wst
}  // namespace dgb
