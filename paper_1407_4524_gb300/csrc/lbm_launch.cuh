// lbm_launch.cuh -- typed launchers of the step kernels; included by the
// precision translation units (lbm_fp64.cu, lbm_fp32.cu).
#pragma once

#include <algorithm>

#include "lbm_internal.h"
#include "lbm_pair.cuh"
#include "lbm_stage.cuh"
#include "lbm_tma.cuh"

namespace lbm {

// Threads of a row's blocks.  Rows of up to BULK_THREADS nodes: the warps the
// row has (a block holds the registers of idle warps until it ends: the 93x61x57
// duct's step 16.5 -> 15.2 us with 96 threads instead of 128).  Longer rows: in
// FP64 mode, with 16 warps an SM, the size that leaves the fewest idle warps,
// the larger of two that leave as many (135x1073 disc 75 -> 69 us with 96); in
// the reduced modes BULK_THREADS (151x97x84: 66.2 us, 67.5 with 96).
inline dim3 bulk_block(const Params &p) {
    if (p.nx <= BULK_THREADS) return dim3((p.nx + 31) / 32 * 32, 1, 1);
    if (!p.exact) return dim3(BULK_THREADS, 1, 1);
    int best = BULK_THREADS, least = 0;
    for (int bx = BULK_THREADS; bx >= 64; bx -= 32) {
        const int threads = (p.nx + bx - 1) / bx * bx;
        if (least == 0 || threads < least) {
            best = bx;
            least = threads;
        }
    }
    return dim3(best, 1, 1);
}

inline dim3 bulk_grid(const Params &p) {
    dim3 b = bulk_block(p);
    return dim3((p.nx + b.x - 1) / b.x, p.ny, p.zc ? p.zc : p.nz);
}

template <class L, class P>
cudaError_t init_t(const Params &p, void *dst, void *mac, const uint8_t *flags, const double u0[3], cudaStream_t s) {
    k_init<L, P><<<bulk_grid(p), bulk_block(p), 0, s>>>(p, (typename P::S *)dst, (typename P::C *)mac, flags, u0[0],
                                                         u0[1], u0[2]);
    return cudaGetLastError();
}

template <class L, class P>
cudaError_t load_t(const Params &p, const double *stage, long long c0, long long n, void *dst, void *mac,
                   const uint8_t *flags, cudaStream_t s) {
    const unsigned grid = (unsigned)((n + BULK_THREADS - 1) / BULK_THREADS);
    k_load<L, P><<<grid, BULK_THREADS, 0, s>>>(p, stage, c0, n, (typename P::S *)dst, (typename P::C *)mac, flags);
    return cudaGetLastError();
}

template <class L, class P>
cudaError_t macros_t(const Params &p, const void *src, const uint16_t *owner, long long c0, long long n, double *out,
                     cudaStream_t s) {
    const unsigned grid = (unsigned)((n + BULK_THREADS - 1) / BULK_THREADS);
    k_macros<L, P><<<grid, BULK_THREADS, 0, s>>>(p, (const typename P::S *)src, owner, c0, n, out);
    return cudaGetLastError();
}

template <class L, class P> cudaError_t links_t(const Params &p, const StepBufs &sb, int grid, cudaStream_t s) {
    if (p.nb == 0 || grid <= 0) return cudaSuccess;
    if (P::exact) k_links<L, P><<<grid * (LINK_THREADS / 32), 32, 0, s>>>(p, sb);
    else k_links<L, P><<<grid, LINK_THREADS, 0, s>>>(p, sb);
    return cudaGetLastError();
}

// reduced precision with 16-byte aligned rows: rows staged by bulk copies
template <class L, class P> void staged_launch(const Params &p, const StepBufs &sb, cudaStream_t s) {
    using S = typename P::S;
    const int seg = std::min(STAGE_SEG, p.nx);
    const long long nseg = (long long)((p.nx + seg - 1) / seg) * p.ny * p.nz;
    const int grid = (int)std::min<long long>(nseg, (long long)std::max(1, p.nsm) * STAGE_BLOCKS_PER_SM);
    k_bulk_staged<L, P><<<grid, seg, stage_smem<L, S>(seg), s>>>(p, (const S *)sb.src, (S *)sb.dst, sb.flags,
                                                                  sb.counters, (float *)sb.mac_t1);
}

// one kernel per face mode: the fewer faces, the less code in the loop
template <class L, class P> cudaError_t bulk_t(const Params &p, const StepBufs &sb, cudaStream_t s) {
    if constexpr (!P::exact) {
        if (p.staged && staged_ok<L, P>(p)) {
            staged_launch<L, P>(p, sb, s);
            return cudaGetLastError();
        }
    }
    const int fm = face_mode(p);
    const typename P::S *src = (const typename P::S *)sb.src;
    typename P::S *dst = (typename P::S *)sb.dst;
    const typename P::C *mt = (const typename P::C *)sb.mac_t;
    typename P::C *mt1 = (typename P::C *)sb.mac_t1;
    bool pair = false, tma = false;
    if constexpr (!P::exact) pair = p.pair && pair_ok(p, fm);
    if constexpr (std::is_same<typename P::S, __half>::value) tma = sb.counters && tma_ok<L, P>(p, src);
    if (tma) {
        if constexpr (std::is_same<typename P::S, __half>::value) {
            const bool room = sb.n_moving > 0, xf = fm == FM_XFACES;
            const auto run = xf ? (room ? tma_launch<L, P, FM_XFACES, true> : tma_launch<L, P, FM_XFACES, false>)
                                : (room ? tma_launch<L, P, FM_PERIODIC, true> : tma_launch<L, P, FM_PERIODIC, false>);
            const cudaError_t e = run(p, src, dst, sb.flags, sb.counters, mt1, s);
            if (e != cudaSuccess) return e;
        }
    } else if (pair) {
        if constexpr (!P::exact) k_bulk_pair<L, P><<<pair_grid(p), pair_block(p), 0, s>>>(p, src, dst, sb.flags, mt1);
    } else if (fm == FM_PERIODIC)
        k_bulk<L, P, FM_PERIODIC><<<bulk_grid(p), bulk_block(p), 0, s>>>(p, src, dst, sb.flags, mt, mt1);
    else if (fm == FM_XFACES)
        k_bulk<L, P, FM_XFACES><<<bulk_grid(p), bulk_block(p), 0, s>>>(p, src, dst, sb.flags, mt, mt1);
    else
        k_bulk<L, P, FM_GENERAL><<<bulk_grid(p), bulk_block(p), 0, s>>>(p, src, dst, sb.flags, mt, mt1);
    return cudaGetLastError();
}

// the Zou-He face nodes, which the bulk kernel skips
template <class L, class P> cudaError_t zouhe_t(const Params &p, const StepBufs &sb, cudaStream_t s) {
    if (!p.zouhe) return cudaSuccess;
    long long plane = 0;
    const long long n[3] = {p.nx, p.ny, p.nz};
    for (int a = 0; a < 3; ++a) plane = std::max(plane, n[(a + 1) % 3] * n[(a + 2) % 3]);
    const dim3 grid((unsigned)((plane + ZOUHE_THREADS - 1) / ZOUHE_THREADS), 1, 6);
    k_zouhe<L, P><<<grid, ZOUHE_THREADS, 0, s>>>(p, (const typename P::S *)sb.src, (typename P::S *)sb.dst, sb.flags,
                                                 (const typename P::C *)sb.mac_t, (typename P::C *)sb.mac_t1);
    return cudaGetLastError();
}

template <class L, class P> cudaError_t finish_t(const Params &p, const StepBufs &sb, cudaStream_t s) {
    const int grid = p.nb + sb.n_moving;
    if (grid == 0) return cudaSuccess;
    k_finish<L, P><<<grid, IMP_THREADS, 0, s>>>(p, sb);
    return cudaGetLastError();
}

} // namespace lbm
