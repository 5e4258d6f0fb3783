// Rows of a tile computed from shared memory.  The smallest-first layout keeps most columns of a
// tile of consecutive pi_0 rows inside the tile (128 rows: 90 % of a random-geometric graph's
// entries, 63 % of a 3D grid's), and the others repeat (a tile reads 0.46 and 1.77 distinct
// outside rows of X per row of its own).  So a producer warp copies what a tile needs into
// one of a few shared-memory stages ahead of the compute warps -- the tile's descriptors, 16-bit
// local columns and values and its own rows of X by bulk copy, the outside rows ("halo") by
// 16-byte cp.async -- and the compute warps gather from shared memory alone.  Against
// gathering every entry through L1 this keeps no registers for loads in flight, reads 2-byte
// instead of 4-byte columns, and moves each distinct row of X once per tile.
#pragma once

#include "device_common.cuh"

namespace arrow {

constexpr int kStWarps = 8;                       // compute warps; one more warp copies
constexpr int kStThreads = 32 * (kStWarps + 1);
constexpr int kStMaxStages = 4;
constexpr int kStMaxEnt = 2048;                   // entries of a staged tile at most
constexpr int kStMaxT = 8;                        // lanes per row slice: 128 bytes of X

struct StPipe {
    uint64_t full[kStMaxStages];    // 1 arrival with the bulk copies' bytes + 32 of the cp.async lanes
    uint64_t empty[kStMaxStages];   // one arrival per compute warp
    int hdr[kStMaxStages][8];
    int issued[kStMaxStages];
    int failed;
};
constexpr int kStPipeBytes = 384;
static_assert(sizeof(StPipe) <= kStPipeBytes, "pipeline state must fit");

// Shared-memory layout of one stage and the launch shape (staged_plan).
struct StLayout {
    int desc, col, val, x;   // byte offsets of the regions inside a stage
    int stage_bytes, stages;
};

// What the producer needs of one matrix.
struct StMat {
    const int4* tile;          // [n_tiles+1] first row, first entry, first halo row of each tile
    const uint32_t* desc;      // [n] row descriptors (row_desc_pack) of the staged tiles
    const uint16_t* col;       // [nnz] row of the staged X: own rows first, then the halo
    const void* val;
    const int32_t* halo;       // pi_0 positions of the halo rows
    const int32_t* rowptr;
};

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Arrives on the barrier when the thread's cp.async copies so far have landed (counted among the
// barrier's expected arrivals).
__device__ __forceinline__ void cp_async_arrive(uint64_t* bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Copy rows idx[0..cnt) of X (slices of 16 << lt bytes at X, row stride ld bytes) to the staged
// rows at dst: a lane per 16 bytes, eight rows' copies issued per lane and round, the next round's
// indices loaded before this round's copies.  CONTIG: idx is null and row i is i.
template <bool OWN>
__device__ __forceinline__ void st_copy_rows(const int32_t* __restrict__ idx, int cnt, const char* X, int64_t ld,
                                             uint32_t dst, int lt, int lane) {
    const int rpw = 32 >> lt, lr = lane >> lt, lq = (lane & ((1 << lt) - 1)) * 16;
    const char* src = X + lq;
    dst += uint32_t(lq);
    constexpr int U = 8;
    int32_t c[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int i = u * rpw + lr;
        c[u] = OWN ? i : (i < cnt ? __ldg(idx + i) : 0);
    }
    for (int i0 = 0; i0 < cnt; i0 += U * rpw) {
        int32_t nx[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + (U + u) * rpw + lr;
            nx[u] = OWN ? i : (i < cnt ? __ldg(idx + i) : 0);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + u * rpw + lr;
            if (i < cnt) cp_async16(dst + (uint32_t(i) << (lt + 4)), src + int64_t(c[u]) * ld);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) c[u] = nx[u];
    }
}

// R entries of a staged row: columns, values and X from shared memory, accumulated in order.
template <int R, typename TX, typename TV, int T>
__device__ __forceinline__ void st_round(const uint16_t* scol, const TV* sval, int base, const char* sx, float* acc) {
    uint4 x[R];
#pragma unroll
    for (int u = 0; u < R; ++u) x[u] = *reinterpret_cast<const uint4*>(sx + uint32_t(scol[base + u]) * uint32_t(16 * T));
#pragma unroll
    for (int u = 0; u < R; ++u) axpy_vec<TX, TV>(sval[base + u], x[u], acc);
}
template <typename TX, typename TV, int T>
__device__ __forceinline__ void st_row(const uint16_t* scol, const TV* sval, int s, int e, const char* sx, float* acc) {
    int base = s;
    for (; base + 8 <= e; base += 8) st_round<8, TX, TV, T>(scol, sval, base, sx, acc);
    switch (e - base) {
        case 7: st_round<7, TX, TV, T>(scol, sval, base, sx, acc); break;
        case 6: st_round<6, TX, TV, T>(scol, sval, base, sx, acc); break;
        case 5: st_round<5, TX, TV, T>(scol, sval, base, sx, acc); break;
        case 4: st_round<4, TX, TV, T>(scol, sval, base, sx, acc); break;
        case 3: st_round<3, TX, TV, T>(scol, sval, base, sx, acc); break;
        case 2: st_round<2, TX, TV, T>(scol, sval, base, sx, acc); break;
        case 1: st_round<1, TX, TV, T>(scol, sval, base, sx, acc); break;
        default: break;
    }
}

__device__ __forceinline__ void st_init(StPipe* ps, int stages) {
    if (threadIdx.x == 0) {
        for (int b = 0; b < stages; ++b) {
            mbar_init(&ps->full[b], 1 + 32);
            mbar_init(&ps->empty[b], kStWarps);
            ps->issued[b] = 0;
        }
        ps->failed = 0;
        fence_mbar_init();
    }
    __syncthreads();
}

// Producer warp: stage tile t of matrix m into stage b (its previous use released, waited for by the
// caller).  X, ld: the column slice's first row and the row stride in bytes; lt = log2(lanes
// per slice); contig: rows of the slice are adjacent, so the tile's own rows are one bulk copy.
template <typename TV>
__device__ __forceinline__ void st_fill(StPipe* ps, unsigned char* stage, const StLayout& L, int b, const StMat& m,
                                        const int4& t0, const int4& t1, const char* X, int64_t ld, int lt, bool contig,
                                        int lane) {
    constexpr int VE = 16 / int(sizeof(TV));
    const int r0 = t0.x, nrows = t1.x - t0.x, nh = t1.z - t0.z;
    fence_proxy_async_smem();
    if (lane == 0) {
        const int ra = r0 & ~3, rb = (t1.x + 3) & ~3;
        const int ca = t0.y & ~7, cb = (t1.y + 7) & ~7;
        const int va = t0.y & ~(VE - 1), vb = (t1.y + VE - 1) & ~(VE - 1);
        const uint32_t bd = uint32_t(rb - ra) * 4u, bc = uint32_t(cb - ca) * 2u, bv = uint32_t(vb - va) * uint32_t(sizeof(TV));
        const uint32_t bx = contig ? uint32_t(nrows) << (lt + 4) : 0u;
        ps->issued[b]++;
        mbar_arrive_expect_tx(&ps->full[b], bd + bc + bv + bx);
        bulk_g2s(stage + L.desc, m.desc + ra, bd, &ps->full[b]);
        if (bc) bulk_g2s(stage + L.col, m.col + ca, bc, &ps->full[b]);
        if (bv) bulk_g2s(stage + L.val, static_cast<const TV*>(m.val) + va, bv, &ps->full[b]);
        if (bx) bulk_g2s(stage + L.x, X + int64_t(r0) * ld, bx, &ps->full[b]);
    }
    const uint32_t dx = smem_u32(stage + L.x);
    if (!contig) st_copy_rows<true>(nullptr, nrows, X + int64_t(r0) * ld, ld, dx, lt, lane);
    st_copy_rows<false>(m.halo + t0.z, nh, X, ld, dx + (uint32_t(nrows) << (lt + 4)), lt, lane);
    cp_async_arrive(&ps->full[b]);
}

// After the loops, all threads: the producer's copies have landed; after a failed wait, bounded
// waits for the latest use of every stage.
__device__ __forceinline__ bool st_finish(StPipe* ps, int stages) {
    cp_async_wait_all();
    __syncthreads();
    if (!ps->failed) return true;
    if (threadIdx.x == 0)
        for (int b = 0; b < stages; ++b)
            if (ps->issued[b] > 0) mbar_wait_bounded(&ps->full[b], uint32_t((ps->issued[b] - 1) & 1), kWaitLimitNs);
    return false;
}

}  // namespace arrow
