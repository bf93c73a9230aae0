// lbm_tma.cuh -- two-node stream-collide with the source rows of a tile of
// whole rows brought to shared memory by bulk asynchronous copies.
//
// What bounds the direct two-node kernel with FP16 storage is not the memory
// but its loads: 19 four-byte loads a thread, held in registers until the
// moments need them, at eight blocks of 128 threads an SM (45 % of the warps):
// 0.78 of the measured copy rate on the 512x256x256 swarm, 0.59 on the
// 256x128x128 channel, whose x faces the direct kernels step one node a thread.
// This one: 0.93 (403 us in the step, bound by DRAM) and 0.80 (59 us, 5 of them
// filling and draining the ring); instructions a node 275 -> 241.
// Here a block takes a tile of TY whole rows of one plane z.  Whole rows are
// contiguous, so the sources of direction i -- rows y - c_iy of plane z - c_iz
// of population i -- are one copy of TY * nx values (two where the tile meets
// the periodic y seam), and the x shift and its periodic wrap are an index into
// the row.  Up to TMA_STAGES tiles of 19 copies are in flight per SM (nothing
// of that in registers), issued by a producer warp.  Each other warp waits for
// a tile, takes two nodes a lane, releases the stage and goes on with
// moments_pair / collide_pair: the operations of the direct kernels, so the
// same values.
//
// Channels along x (FM_XFACES: inlet or wall at x-lo, outlet at x-hi): the
// first node of a row takes its bounced populations from global memory (loaded
// a tile ahead), the last one the row's last column, as pull_core.
//
// Every wait on an mbarrier is bounded (mbar_wait_bounded); a wait that gives
// up sets LBM_TIMEOUT_FLAG in counters[6] and its warp leaves the loop; the
// block then drains its own copies (bounded) before it returns.
#pragma once

#include "lbm_pair.cuh"
#include "lbm_stage.cuh"

namespace lbm {

constexpr int TMA_SLOT = 2048; // bytes of one direction of a tile
constexpr int TMA_STAGES = 3;  // 19 * 2 KB * 3 = 117 KB of shared memory; 2, 4 and 5 stages measured the same or slower

template <class S> __host__ __device__ constexpr int tma_tile() { return TMA_SLOT / (int)sizeof(S); } // nodes of a tile
template <class S> __host__ __device__ constexpr int tma_threads() { return tma_tile<S>() / 2 + 32; } // a pair a thread, and the producer warp
// threads the register allocation is made for: with ROOM (moving bodies) 80
// registers, so that an SM sub-partition's five warps leave space for the two
// warps of a geometry block (48 registers) and the side stream runs beside the
// pass; the 96 registers the kernel takes otherwise keep it out until the end
// (512x256x256 swarm: step 0.488 ms against 0.437), and are 4 % faster where
// there is no geometry (256x128x128 channel)
template <class S, bool ROOM> __host__ __device__ constexpr int tma_reg_threads() { return ROOM ? 768 : tma_threads<S>(); }

__device__ __forceinline__ void mbar_arrive(unsigned long long *bar) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(smem_u32(bar)) : "memory");
}

// one shared-memory pair (two neighbouring nodes of a row) and single values
template <class S> struct Shr;
template <> struct Shr<__half> {
    using T = unsigned;
    static __device__ __forceinline__ T pair(const __half *p) { return *reinterpret_cast<const unsigned *>(p); }
    static __device__ __forceinline__ T left(const __half *e, T own) { // (*e, own 0)
        return __byte_perm((unsigned)*reinterpret_cast<const unsigned short *>(e), own, 0x5410);
    }
    static __device__ __forceinline__ T right(T own, const __half *e) { // (own 1, *e)
        return __byte_perm(own, (unsigned)*reinterpret_cast<const unsigned short *>(e), 0x5432);
    }
    static __device__ __forceinline__ T first(T own, __half v) { return __byte_perm((unsigned)__half_as_ushort(v), own, 0x7610); }
};
// rows of a tile and tiles of a plane
template <class S> __host__ __device__ inline int tma_rows(int nx, int ny) {
    const int r = tma_tile<S>() / nx;
    return r < ny ? r : ny;
}

template <class L, class P, int FM, bool ROOM>
__global__ void __launch_bounds__(tma_reg_threads<typename P::S, ROOM>(), 1)
    k_bulk_tma(Params p, const typename P::S *__restrict__ src, typename P::S *__restrict__ dst,
               const uint8_t *__restrict__ flags, unsigned long long *counters, typename P::C *__restrict__ mac_t1) {
    using S = typename P::S;
    using PT = Pair<S>;
    using SH = Shr<S>;
    using T = typename SH::T;
    constexpr int TILE = tma_tile<S>(), CONS = TILE / 2;
    constexpr int STAGE = L::Q * TILE; // values of a stage
    extern __shared__ __align__(128) unsigned char smem[];
    unsigned long long *full = (unsigned long long *)smem, *empty = full + TMA_STAGES;
    S *stages = (S *)(smem + 128);
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    const int TY = tma_rows<S>(nx, ny);
    const int tpp = (ny + TY - 1) / TY; // tiles of a plane
    const int ntiles = tpp * nz;
    const unsigned N32 = (unsigned)p.N;
    if (threadIdx.x == 0) {
        for (int s = 0; s < TMA_STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], CONS / 32);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    // lane i: the copies of direction i of the k-th tile of this block
    auto issue = [&](int k) {
        const int tile = blockIdx.x + k * gridDim.x, st = k % TMA_STAGES;
        const int z = tile / tpp, y0 = (tile - z * tpp) * TY;
        const int rows = min(TY, ny - y0);
        const unsigned row_bytes = (unsigned)(nx * (int)sizeof(S));
        if (lane == 0) mbar_arrive_expect_tx(&full[st], (unsigned)L::Q * (unsigned)rows * row_bytes);
        __syncwarp();
        if (p.stage_expire_test) return; // test hook: no copies, so the waits expire
        if (lane < L::Q) {
            const int cy = L::cy(lane), cz = L::cz(lane);
            int sz = z - cz;
            sz = sz < 0 ? nz - 1 : (sz >= nz ? 0 : sz);
            const S *plane = src + (size_t)N32 * (unsigned)lane + (size_t)((unsigned)sz * (unsigned)ny) * (unsigned)nx;
            S *slot = stages + (size_t)st * STAGE + (size_t)lane * TILE;
            const int ys = y0 - cy;
            if (ys < 0) { // row ny - 1, then rows 0 ..
                bulk_g2s(slot, plane + (size_t)(ny - 1) * nx, row_bytes, &full[st]);
                if (rows > 1) bulk_g2s(slot + nx, plane, (unsigned)(rows - 1) * row_bytes, &full[st]);
            } else if (ys + rows > ny) { // .. row ny - 1, then row 0
                if (rows > 1) bulk_g2s(slot, plane + (size_t)ys * nx, (unsigned)(rows - 1) * row_bytes, &full[st]);
                bulk_g2s(slot + (size_t)(rows - 1) * nx, plane, row_bytes, &full[st]);
            } else {
                bulk_g2s(slot, plane + (size_t)ys * nx, (unsigned)rows * row_bytes, &full[st]);
            }
        }
        __syncwarp();
    };
    const int mine = (ntiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x; // tiles of this block
    if (threadIdx.x >= CONS) { // producer warp
        int k = 0;
        for (; k < mine; ++k) {
            // the stage's last tile has been read by every warp
            const int r = k - TMA_STAGES;
            if (r >= 0 && !__all_sync(0xffffffffu, mbar_wait_bounded(&empty[r % TMA_STAGES], (unsigned)((r / TMA_STAGES) & 1)))) {
                if (lane == 0) atomicOr(&counters[6], LBM_TIMEOUT_FLAG);
                break;
            }
            issue(k);
        }
        // every copy has landed before the block's shared memory goes away
        for (int j = max(0, k - TMA_STAGES); j < k; ++j)
            mbar_wait_bounded(&full[j % TMA_STAGES], (unsigned)((j / TMA_STAGES) & 1));
        return;
    }
    const int t = threadIdx.x, half = nx >> 1;
    const int row = t / half, x0 = 2 * (t - row * half);
    const bool own_row = row < TY;
    // x neighbours of the pair inside the row (wrapped), as indices into a slot
    const int base = 2 * t;
    const int il = x0 == 0 ? base + nx - 1 : base - 1, ir = x0 + 2 >= nx ? base + 2 - nx : base + 2;
    const int li = own_row ? il : 0, ri = own_row ? ir : 0;
    bool lo_b = false, hi_out = false;
    if constexpr (FM == FM_XFACES) {
        lo_b = own_row && x0 == 0;
        hi_out = own_row && x0 + 2 >= nx;
    }
    const uint8_t skip = FL_SOLID | (p.linkmode ? 0 : FL_BND);
    // what a tile reads past the ring, one tile ahead: the flags of the pair
    // and the bounced populations of the row's first node (opposite
    // direction, own cell)
    unsigned cell0 = 0u, fl2 = 0u;
    bool valid = false;
    int y = 0;
    S bl[L::Q];
    auto ahead = [&](int tile) {
        const int z = tile / tpp;
        y = (tile - z * tpp) * TY + row;
        valid = own_row && y < ny && tile < ntiles;
        cell0 = valid ? ((unsigned)z * (unsigned)ny + (unsigned)y) * (unsigned)nx + (unsigned)x0 : 0u;
        fl2 = __ldg(reinterpret_cast<const unsigned short *>(flags + cell0));
        if constexpr (FM == FM_XFACES) {
            if (lo_b) {
#pragma unroll
                for (int i = 0; i < L::Q; ++i)
                    if (L::cx(i) == 1) bl[i] = __ldg(src + (size_t)N32 * (unsigned)L::opp(i) + cell0);
            }
        }
    };
    ahead(blockIdx.x);
    for (int k = 0; k < mine; ++k) {
        const int s = k % TMA_STAGES;
        if (!__all_sync(0xffffffffu, mbar_wait_bounded(&full[s], (unsigned)((k / TMA_STAGES) & 1)))) {
            if (lane == 0) atomicOr(&counters[6], LBM_TIMEOUT_FLAG);
            break;
        }
        const S *st = stages + (size_t)s * STAGE;
        F2 f[L::Q];
#pragma unroll
        for (int i = 0; i < L::Q; ++i) {
            const S *slot = st + i * TILE;
            const T own = SH::pair(slot + base);
            T v = own;
            if (L::cx(i) == 1) {
                v = SH::left(slot + li, own);
                if constexpr (FM == FM_XFACES) {
                    if (lo_b) v = SH::first(v, bl[i]);
                }
            } else if (L::cx(i) == -1) {
                v = SH::right(own, slot + (FM == FM_XFACES && hi_out ? base + 1 : ri));
            }
            f[i] = PT::cvt(v);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[s]);
        const unsigned here = cell0;
        const unsigned fl0 = fl2 & 0xffu, fl1 = fl2 >> 8;
        const bool act0 = valid && !(fl0 & skip), act1 = valid && !(fl1 & skip);
        if constexpr (FM == FM_XFACES) { // momentum terms of the wall / inlet links (face_terms, quasi-incompressible)
            if (lo_b) {
#pragma unroll
                for (int i = 0; i < L::Q; ++i) {
                    if (L::cx(i) != 1) continue;
                    const float uB = p.edge[0] != 2 ? 0.0f : (p.inlet_parabolic ? (float)inlet_u(p, y, L::cy(i)) : p.u_inf);
                    const float2 v = unf2(f[i]);
                    f[i] = f2(fmaf(6.0f * L::template w<float>(i) * p.rho0f, uB, v.x), v.y);
                }
            }
        }
        ahead(blockIdx.x + (k + 1) * gridDim.x);
        F2 drho, u[3];
        moments_pair<L>(p, f, drho, u);
        if (p.linkmode && ((act0 && (fl0 & FL_MAC)) || (act1 && (fl1 & FL_MAC)))) {
            const float2 d = unf2(drho), u0 = unf2(u[0]), u1 = unf2(u[1]), u2 = unf2(u[2]);
            if (act0 && (fl0 & FL_MAC)) {
                const float uu[3] = {u0.x, u1.x, u2.x};
                store_mac((float *)mac_t1, here, d.x, uu);
            }
            if (act1 && (fl1 & FL_MAC)) {
                const float uu[3] = {u0.y, u1.y, u2.y};
                store_mac((float *)mac_t1, here + 1, d.y, uu);
            }
        }
        collide_pair<L>(p, f, drho, u);
        if (act0 && act1) {
#pragma unroll
            for (int i = 0; i < L::Q; ++i)
                PT::st(reinterpret_cast<S *>(reinterpret_cast<char *>(dst) + (unsigned)(N32 * (unsigned)sizeof(S) * (unsigned)i + here * (unsigned)sizeof(S))), f[i]);
        } else if (act0 || act1) { // one node of the pair is solid (or a boundary node): store the other
            const unsigned c = act0 ? here : here + 1;
#pragma unroll
            for (int i = 0; i < L::Q; ++i) {
                const float2 e = unf2(f[i]);
                stS(dst + (size_t)N32 * (unsigned)i + c, act0 ? e.x : e.y);
            }
        }
    }
}

template <class L> __host__ __device__ constexpr size_t tma_smem() { return 128 + (size_t)TMA_STAGES * L::Q * TMA_SLOT; }

// D3Q19 with FP16 storage (with FP32 the direct kernels are at the memory's
// rate: the 256x128x128 channel's pass takes 102 us there, 113 us here; a D2Q9
// tile is too little work: 1024x2048 takes 19.0 us a step there, 20.5 us here);
// whole rows that fit a slot and start on 16 bytes; the face forms above;
// 32-bit byte offsets.  Filling and draining the ring costs some 5 us, so a
// domain needs tiles enough an SM (step, direct -> here): x faces (the direct
// kernel takes one node a thread there) 64^3 12.4 -> 12.4 us, 128x64x64 16.3 ->
// 16.1, 192x96x96 42.4 -> 33.8, 256x128x128 82.6 -> 60.9; periodic 96x80x72
// (4 tiles an SM) 15.3 -> 16.2, 192x96x96 (13) 39.1 -> 33.5, 256x128x128 69.4 ->
// 59.7 us.
template <class L, class P> inline bool tma_ok(const Params &p, const void *src) {
    using S = typename P::S;
    const int fm = face_mode(p);
    if (L::D != 3 || !p.pair || p.has_force || p.zouhe || fm == FM_GENERAL) return false;
    if (fm == FM_XFACES && (p.eq != 0 || p.edge[1] != 3)) return false;
    if (((size_t)p.nx * sizeof(S)) % 16 != 0 || p.nx > tma_tile<S>() || ((uintptr_t)src) % 16 != 0) return false;
    if ((unsigned long long)p.N * L::Q * sizeof(S) >= (1ull << 32)) return false;
    const int ty = tma_rows<S>(p.nx, p.ny);
    return (long long)((p.ny + ty - 1) / ty) * p.nz >= (fm == FM_XFACES ? 4ll : 8ll) * p.nsm;
}

template <class L, class P, int FM, bool ROOM>
cudaError_t tma_launch(const Params &p, const typename P::S *src, typename P::S *dst, const uint8_t *flags,
                       unsigned long long *counters, typename P::C *mac_t1, cudaStream_t s) {
    using S = typename P::S;
    constexpr size_t smem = tma_smem<L>();
    cudaError_t e = cudaFuncSetAttribute(k_bulk_tma<L, P, FM, ROOM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int ty = tma_rows<S>(p.nx, p.ny);
    const int ntiles = (p.ny + ty - 1) / ty * p.nz;
    cudaLaunchAttribute prio;
    prio.id = cudaLaunchAttributePriority;
    int lo = 0, hi = 0;
    cudaDeviceGetStreamPriorityRange(&lo, &hi);
    prio.val.priority = hi;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)std::min(ntiles, p.nsm), 1, 1);
    cfg.blockDim = dim3(tma_threads<S>(), 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &prio;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_bulk_tma<L, P, FM, ROOM>, p, src, dst, flags, counters, mac_t1);
}

} // namespace lbm
