// Multi-matrix kernels shared by the batched path (arrow_batch.cu) and the serving runtime
// (arrow_server.cu).  Work units of all matrices of a launch live in one index space: unit w
// belongs to matrix m with base[m] <= w < base[m+1]; every matrix carries its own feature
// width and ping-pong state, so a matrix computes the same bits whatever else shares the launch.
#pragma once

#include "device_common.cuh"

namespace arrow {

struct MatDesc {
    const int32_t* rowptr;
    const uint32_t* row_desc;
    const int32_t* col;
    const void* val;
    const int32_t* tile_row;
    const int32_t* tile_ent;
    const int32_t* lcol;
    const void* lval;
    const int32_t* seg_begin;
    const int32_t* seg_end;
    const int32_t* long_rows;
    const int32_t* long_segptr;
    const int32_t* perm0;
    const int32_t* iperm0;
    const void* x_user;   // caller's X (vertex order)
    void* y_user;         // caller's Y (vertex order)
    void* xa;             // pi_0-ordered ping-pong buffers
    void* xb;
    float* partials;      // [n_seg][k]
    int64_t n;
    int64_t k;
    int32_t T;            // lanes per row = k / V
    int32_t flip;         // xor-ed into the launch parity (per-request ping-pong state)
    int32_t out;          // 1: this launch's iteration is the last, its rows go to y_user
    int32_t pad;
};

struct BatchArgs {
    const MatDesc* d;
    const int64_t* base;   // [n_mats+1] prefix of this kernel class's work units
    int32_t n_mats;
    int64_t total;
    int32_t parity;        // 0: xa -> xb, 1: xb -> xa
    int32_t dir;           // gather: 0 permute-in, 1 permute-out
    int32_t out;           // rows, combine: the last iteration of every matrix (MatDesc::out)
    int32_t* status;
    int32_t rp_bytes, col_bytes, buf_bytes;   // staged-tile layout (rows kernel)
    int32_t parts;         // rows kernel: CTAs that share a tile's rows (row_parts); unit w is tile w / parts
};

__device__ __forceinline__ int find_mat(const int64_t* base, int n, int64_t w) {
    int lo = 0, hi = n - 1;   // largest m with base[m] <= w
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(base + mid) <= w) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// The last iteration of a matrix stores its rows straight at their vertices in the caller's Y
// (row p at pi_0^{-1}(p)), without a permute-out pass; rows narrower than a 32-byte sector keep the pass
// (fold_permute_out, arrow_spmm.cu, has the reason and the figures).
__host__ __device__ inline bool folds_out(int64_t k, int sx) { return k * sx >= 32; }

inline int batch_smem_bytes(const TileLayout& L) { return 128 + kStages * L.buf; }

// Rows of every matrix's tiles (the fused arrow-row kernel of arrow_spmm with a per-tile
// matrix descriptor and a run-time team width); same tile pipeline without block barriers.
// Resident CTAs per SM that the register use of the batched rows kernel allows (64 registers).
// A tile's rows come in order of length (row_desc), so the exact-size remainder rounds of
// gather_row hardly diverge: 24 random-geometric matrices (FP16, k 8..64) 2277 -> 1988 us per
// 10-iteration call against rows in position order with predicated rounds of 8.
#ifndef ARROW_BATCH_MIN_BLOCKS
#define ARROW_BATCH_MIN_BLOCKS 4
#endif
constexpr int kBatchMinBlocks = ARROW_BATCH_MIN_BLOCKS;

// NARROW: every matrix of the launch has rows of one vector (T = 1), so a warp takes 32 rows: in row
// order, from the row pointers, their gathers share lines and their stores are contiguous, and
// predicated rounds keep the lanes together.  24 random-geometric matrices and an R-MAT, 10 iterations in one graph,
// k = 8 BF16: 344 us before the rows came by length, 396 by length, 318 in this form; k = 4 FP32 359 / 396 / 311.
template <typename TX, typename TV, bool NARROW>
__global__ void __launch_bounds__(256, kBatchMinBlocks) arrow_batch_rows_kernel(BatchArgs a) {
    using P = Pack<TX>;
    constexpr int V = P::V;
    constexpr int VE = 16 / int(sizeof(TV));
    constexpr int NW = 8;
    extern __shared__ __align__(128) unsigned char smem[];
    PipeSmem* ps = reinterpret_cast<PipeSmem*>(smem);
    unsigned char* bufs = smem + 128;
    const int lane = threadIdx.x & 31;
    const int64_t G = gridDim.x;
    const int parts = NARROW ? 1 : a.parts;   // (256 teams: a tile's rows are few for one CTA)
    const int64_t U = a.total * parts;
    auto issue = [&](int64_t u, int b) {
        const int64_t w = parts == 1 ? u : int64_t(uint32_t(u) / uint32_t(parts));   // parts > 1: U < 2^31
        const int m = find_mat(a.base, a.n_mats, w);
        const MatDesc& d = a.d[m];
        const int t = int(w - a.base[m]);
        const int r0 = d.tile_row[t], r1 = d.tile_row[t + 1], e0 = d.tile_ent[t], e1 = d.tile_ent[t + 1];
        ps->hdr[b][0] = m; ps->hdr[b][1] = r0; ps->hdr[b][2] = r1; ps->hdr[b][3] = e0;
        stage_tile<TV>(NARROW ? reinterpret_cast<const uint32_t*>(d.rowptr) : d.row_desc, d.col, static_cast<const TV*>(d.val),
                       r0, r1, e0, e1, bufs + b * a.buf_bytes, &ps->full[b], a.rp_bytes, a.col_bytes);
        ps->issued[b]++;
    };
    if (threadIdx.x == 0) {
        for (int b = 0; b < kStages; ++b) {
            mbar_init(&ps->full[b], 1);
            ps->done[b] = 0;
            ps->issued[b] = 0;
        }
        ps->failed = 0;
        fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (int b = 0; b < kStages; ++b)
            if (int64_t(blockIdx.x) + b * G < U) issue(blockIdx.x + b * G, b);
    pdl_wait();
    // The next kernel comes in early where every CTA of this one has at most one unit, or many.  With a few,
    // some CTAs hold their places much longer than others, and a next rows kernel that came in beside
    // them was placed as unevenly: 3 random-geometric matrices (k = 8, 16, 32 BF16), 10 iterations in one graph 136
    // us with an early trigger, 113 without (131 before launches overlapped).  25 small ones 146 / 148;
    // 24 of up to 1 M rows (21 units a CTA) 1985 / 1996; 25 of up to 200,000 (6 units) 585 / 583.
    if (U <= G || U >= 8 * G) pdl_launch();
    int i = 0;
    for (int64_t w = blockIdx.x; w < U; w += G, ++i) {
        const int b = i % kStages;
        unsigned char* buf = bufs + b * a.buf_bytes;
        const bool ok = mbar_wait_bounded(&ps->full[b], (i / kStages) & 1, kWaitLimitNs);
        if (__any_sync(0xffffffffu, !ok)) {
            if (lane == 0) { ps->failed = 1; atomicExch(a.status, kStatusTimeout); }
            break;
        }
        const int m = ps->hdr[b][0], r0 = ps->hdr[b][1], r1 = ps->hdr[b][2], e0 = ps->hdr[b][3];
        const MatDesc& d = a.d[m];
        const int T = NARROW ? 1 : d.T;
        const int teams = 256 / T;
        const int team = threadIdx.x / T, tl = threadIdx.x & (T - 1);
        const int64_t ldx = NARROW ? V : d.k;
        const int par = a.parity ^ d.flip;
        const TX* __restrict__ X = static_cast<const TX*>(par ? d.xb : d.xa) + tl * V;
        const bool fin = !NARROW && (a.out | d.out) && folds_out(ldx, int(sizeof(TX)));
        const int32_t* oidx = fin ? d.iperm0 + r0 : nullptr;
        TX* __restrict__ Y = static_cast<TX*>(fin ? d.y_user : par ? d.xa : d.xb) + tl * V;
        const uint32_t* sdesc = reinterpret_cast<const uint32_t*>(buf) + (r0 & 3);
        const int32_t* scol = reinterpret_cast<const int32_t*>(buf + a.rp_bytes) + (e0 & 3);
        const TV* sval = reinterpret_cast<const TV*>(buf + a.rp_bytes + a.col_bytes) + (e0 & (VE - 1));
        const int nrows = r1 - r0;
        const int part = parts == 1 ? 0 : int(uint32_t(w) % uint32_t(parts));
        for (int q = team + part * teams; q < nrows; q += teams * parts) {
            const RowDesc rd = NARROW ? RowDesc{int(sdesc[q]) - e0, q, int(sdesc[q + 1] - sdesc[q])}
                                      : row_desc_unpack(sdesc[q], d.rowptr, r0);
            const int64_t yr = oidx ? __ldg(oidx + rd.row) : r0 + rd.row;
            float acc[V];
#pragma unroll
            for (int v = 0; v < V; ++v) acc[v] = 0.f;
            if constexpr (NARROW) gather_row_pred<TX, TV>(scol, sval, rd.start, rd.start + rd.len, X, ldx, acc);
            else gather_row<TX, TV>(scol, sval, rd.start, rd.start + rd.len, X, ldx, acc);
            *reinterpret_cast<uint4*>(Y + yr * ldx) = P::from_float(acc);
        }
        __syncwarp();
        if (lane == 0)
            release_buffer(ps, b, NW, [&](int bb) {
                const int64_t wn = w + kStages * G;
                if (wn < U) issue(wn, bb);
            });
    }
    if (NARROW) pdl_launch();   // (short rows: 73 us against 81 without, 3 matrices at k = 4 FP32)
    __syncthreads();
    if (ps->failed && threadIdx.x == 0) drain_pipeline(ps);
}

// One warp per split-row segment of any matrix (first stage of the head-row reduction): the
// same arithmetic as arrow_segments_kernel, dispatched on the matrix's team width.
template <typename TX, typename TV, int T, bool AHEAD>
__device__ __forceinline__ void batch_segment(const MatDesc& d, int64_t g, int par, int lane) {
    using P = Pack<TX>;
    constexpr int V = P::V;
    const int tl = lane & (T - 1), tw = lane / T;
    const TX* __restrict__ X = static_cast<const TX*>(par ? d.xb : d.xa) + tl * V;
    const int32_t s = __ldg(d.seg_begin + g), e = __ldg(d.seg_end + g);
    float acc[V];
    if constexpr (AHEAD) segment_partial_ahead<TX, TV, T>(d.lcol, static_cast<const TV*>(d.lval), X, d.k, s, e, lane, acc);
    else segment_partial<TX, TV, T>(d.lcol, static_cast<const TV*>(d.lval), X, d.k, s, e, lane, acc);
#pragma unroll
    for (int off = T; off < 32; off <<= 1)
#pragma unroll
        for (int v = 0; v < V; ++v) acc[v] += __shfl_xor_sync(0xffffffffu, acc[v], off);
    if (tw == 0) {
        float4* p = reinterpret_cast<float4*>(d.partials + g * d.k + tl * V);
#pragma unroll
        for (int q = 0; q < V / 4; ++q) p[q] = make_float4(acc[4 * q], acc[4 * q + 1], acc[4 * q + 2], acc[4 * q + 3]);
    }
}

template <typename TX, typename TV, bool AHEAD>
__global__ void __launch_bounds__(256, AHEAD ? 1 : ARROW_SEG_MIN_BLOCKS) arrow_batch_segments_kernel(BatchArgs a) {
    const int lane = threadIdx.x & 31;
    const int64_t warp0 = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
    pdl_wait();
    for (int64_t w = warp0; w < a.total; w += nwarps) {
        const int m = find_mat(a.base, a.n_mats, w);
        const MatDesc& d = a.d[m];
        const int64_t g = w - a.base[m];
        const int par = a.parity ^ d.flip;
        switch (d.T) {
            case 1: batch_segment<TX, TV, 1, AHEAD>(d, g, par, lane); break;
            case 2: batch_segment<TX, TV, 2, AHEAD>(d, g, par, lane); break;
            case 4: batch_segment<TX, TV, 4, AHEAD>(d, g, par, lane); break;
            case 8: batch_segment<TX, TV, 8, AHEAD>(d, g, par, lane); break;
            case 16: batch_segment<TX, TV, 16, AHEAD>(d, g, par, lane); break;
            default: batch_segment<TX, TV, 32, AHEAD>(d, g, par, lane); break;
        }
    }
}

// One warp per split row of any matrix: its segment partials in segment order (second stage).
template <typename TX>
__global__ void __launch_bounds__(256) arrow_batch_combine_kernel(BatchArgs a) {
    using P = Pack<TX>;
    constexpr int V = P::V;
    const int lane = threadIdx.x & 31;
    const int64_t warp0 = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
    pdl_wait();
    for (int64_t w = warp0; w < a.total; w += nwarps) {
        const int m = find_mat(a.base, a.n_mats, w);
        const MatDesc& d = a.d[m];
        const int64_t li = w - a.base[m];
        if (lane >= d.T) continue;
        float acc[V];
#pragma unroll
        for (int v = 0; v < V; ++v) acc[v] = 0.f;
        const int g0 = __ldg(d.long_segptr + li), g1 = __ldg(d.long_segptr + li + 1);
        for (int g = g0; g < g1; ++g) {
            const float4* p = reinterpret_cast<const float4*>(d.partials + int64_t(g) * d.k + lane * V);
#pragma unroll
            for (int q = 0; q < V / 4; ++q) {
                const float4 f = p[q];
                acc[4 * q + 0] += f.x; acc[4 * q + 1] += f.y; acc[4 * q + 2] += f.z; acc[4 * q + 3] += f.w;
            }
        }
        const bool fin = (a.out | d.out) && folds_out(d.k, int(sizeof(TX)));
        TX* Y = static_cast<TX*>(fin ? d.y_user : (a.parity ^ d.flip) ? d.xa : d.xb);
        const int32_t r = __ldg(d.long_rows + li);
        *reinterpret_cast<uint4*>(Y + int64_t(fin ? __ldg(d.iperm0 + r) : r) * d.k + lane * V) = P::from_float(acc);
    }
}

// Permute-in (dir 0: xa[p] = X[pi_0^{-1}(p)]) or permute-out (dir 1: Y[v] = buf[pi_0(v)], buf =
// xa or xb by parity) of every matrix; a warp per chunk of 32 rows.
template <typename TX>
__global__ void __launch_bounds__(256) arrow_batch_gather_kernel(BatchArgs a) {
    using P = Pack<TX>;
    constexpr int V = P::V;
    const int lane = threadIdx.x & 31;
    const int64_t warp0 = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
    pdl_wait();
    for (int64_t w = warp0; w < a.total; w += nwarps) {
        const int m = find_mat(a.base, a.n_mats, w);
        const MatDesc& d = a.d[m];
        const int64_t c = w - a.base[m];
        const int nv = d.T, rpw = 32 / nv, lr = lane / nv, lq = lane - lr * nv;
        const TX* src;
        TX* dst;
        const int32_t* idx;
        if (a.dir == 0) {
            src = static_cast<const TX*>(d.x_user); dst = static_cast<TX*>(d.xa); idx = d.iperm0;
        } else {
            src = static_cast<const TX*>((a.parity ^ d.flip) ? d.xb : d.xa); dst = static_cast<TX*>(d.y_user);
            idx = d.perm0;
        }
        const int64_t r_end = min(d.n, (c + 1) * 32);
        for (int64_t r = c * 32 + lr; r < r_end; r += rpw) {
            const int64_t s = __ldg(idx + r);
            *reinterpret_cast<uint4*>(dst + r * d.k + lq * V) = ld_x(src + s * d.k + lq * V);
        }
    }
}

}  // namespace arrow
