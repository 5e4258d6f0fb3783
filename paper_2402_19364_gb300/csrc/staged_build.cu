// Builds the staged form of a handle's short rows (staged_rows.cuh) on the device when the handle
// is uploaded: a tile table of its own, the distinct outside rows of X of every tile, the
// entries' 16-bit columns into the staged rows, and the row descriptors.  It does not depend on
// the feature width or the launch tuning.
#include <algorithm>
#include <string>
#include <vector>

#include "arrow_internal.h"
#include "staged_rows.cuh"

namespace arrow {

int cuda_fail(cudaError_t e, const char* what);

namespace {

#define BCK(call)                                          \
    do {                                                   \
        cudaError_t e_ = (call);                           \
        if (e_ != cudaSuccess) return cuda_fail(e_, #call); \
    } while (0)

// One CTA per tile: its entries' outside columns sorted and made distinct in shared memory.
// !WRITE: their number.  WRITE: the halo list, every entry's local column, and the tile's row
// descriptors (a row's place is the number of rows that are longer, or as long and before it).
template <bool WRITE>
__global__ void __launch_bounds__(256) arrow_halo_kernel(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                                                         const int4* __restrict__ tile, int n_tiles,
                                                         int32_t* __restrict__ count, int32_t* __restrict__ halo,
                                                         uint16_t* __restrict__ lcol, uint32_t* __restrict__ desc) {
    __shared__ uint32_t key[kStMaxEnt];
    __shared__ uint32_t uniq[kStMaxEnt];
    __shared__ int fill, wsum[8], len[256];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int t = blockIdx.x; t < n_tiles; t += gridDim.x) {
        const int4 t0 = tile[t], t1 = tile[t + 1];
        const int r0 = t0.x, nrows = t1.x - t0.x, e0 = t0.y, ne = t1.y - t0.y;
        if (tid == 0) fill = 0;
        __syncthreads();
        for (int j = tid; j < ne; j += 256) {
            const int c = col[e0 + j];
            if (c < r0 || c >= r0 + nrows) key[atomicAdd(&fill, 1)] = uint32_t(c);
        }
        __syncthreads();
        const int m = fill;
        int p2 = 1;
        while (p2 < m) p2 <<= 1;
        for (int j = m + tid; j < p2; j += 256) key[j] = 0xffffffffu;
        for (int k = 2; k <= p2; k <<= 1)
            for (int s = k >> 1; s > 0; s >>= 1) {
                __syncthreads();
                for (int i = tid; i < p2; i += 256) {
                    const int o = i ^ s;
                    if (o > i) {
                        const uint32_t a = key[i], b = key[o];
                        if ((a > b) == ((i & k) == 0)) { key[i] = b; key[o] = a; }
                    }
                }
            }
        __syncthreads();
        // distinct keys, in order: a thread takes a run of consecutive keys
        const int run = (m + 255) / 256;
        int mine = 0;
        for (int i = tid * run; i < min(m, tid * run + run); ++i) mine += i == 0 || key[i] != key[i - 1];
        int incl = mine;
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        int before = 0, total = 0;
        for (int w = 0; w < 8; ++w) {
            if (w < warp) before += wsum[w];
            total += wsum[w];
        }
        if (!WRITE) {
            if (tid == 0) count[t] = total;
        } else {
            int at = before + incl - mine;
            for (int i = tid * run; i < min(m, tid * run + run); ++i)
                if (i == 0 || key[i] != key[i - 1]) {
                    uniq[at] = key[i];
                    halo[t0.z + at] = int32_t(key[i]);
                    ++at;
                }
            for (int j = tid; j < nrows; j += 256) len[j] = rowptr[r0 + j + 1] - rowptr[r0 + j];
            __syncthreads();
            for (int j = tid; j < ne; j += 256) {
                const int c = col[e0 + j];
                int loc = c - r0;
                if (c < r0 || c >= r0 + nrows) {
                    int lo = 0, hi = total - 1;
                    while (lo < hi) {
                        const int mid = (lo + hi) >> 1;
                        if (uniq[mid] < uint32_t(c)) lo = mid + 1; else hi = mid;
                    }
                    loc = nrows + lo;
                }
                lcol[e0 + j] = uint16_t(loc);
            }
            for (int j = tid; j < nrows; j += 256) {
                const int l = len[j];
                int place = 0;
                for (int i = 0; i < nrows; ++i) place += len[i] > l || (len[i] == l && i < j);
                desc[r0 + place] = row_desc_pack(uint32_t(rowptr[r0 + j] - e0), uint32_t(j), uint32_t(l));
            }
        }
        __syncthreads();
    }
}

// Distinct columns outside [r0, r1) of the rows [r0, r1).
int host_halo(const arrow_handle_s* h, int r0, int r1, std::vector<int32_t>& tmp) {
    tmp.clear();
    for (int j = h->f_rowptr[r0]; j < h->f_rowptr[r1]; ++j)
        if (h->f_col[j] < r0 || h->f_col[j] >= r1) tmp.push_back(h->f_col[j]);
    std::sort(tmp.begin(), tmp.end());
    return int(std::unique(tmp.begin(), tmp.end()) - tmp.begin());
}

// [r0, r1) cut in halves until rows + halo fit cap; false if a single row does not.
bool split_tile(const arrow_handle_s* h, int r0, int r1, int cap, std::vector<int4>& out, std::vector<int32_t>& tmp) {
    if (r1 - r0 + host_halo(h, r0, r1, tmp) <= cap) {
        out.push_back(make_int4(r0, h->f_rowptr[r0], 0, 0));
        return true;
    }
    if (r1 - r0 == 1) return false;
    const int mid = r0 + (r1 - r0) / 2;
    return split_tile(h, r0, mid, cap, out, tmp) && split_tile(h, mid, r1, cap, out, tmp);
}

}  // namespace

// Leaves d.st_tiles = 0 (no staged form; the rows kernel gathers from global memory) where the
// tiles read too many distinct outside rows (power-law graphs: 3.7 per row), or n is 0.
int build_staged(arrow_handle_s* h) {
    DeviceData& d = h->dev;
    const int64_t n = h->n, nnz = int64_t(h->f_col.size());
    if (n == 0 || nnz == 0) return ARROW_OK;
    // rows per tile: 128, fewer where that would leave SMs without a tile
    const int W = n >= int64_t(d.sm_count) * 256 ? 128 : n >= int64_t(d.sm_count) * 128 ? 64 : 32;
    std::vector<int4> tiles;
    const int32_t* rp = h->f_rowptr.data();
    for (int64_t r = 0; r < n;) {
        int64_t e = std::min<int64_t>(n, r + W);
        if (rp[e] - rp[r] > kStMaxEnt) e = std::upper_bound(rp + r, rp + e + 1, rp[r] + kStMaxEnt) - rp - 1;
        if (e <= r) return ARROW_OK;   // a row longer than a tile holds
        tiles.push_back(make_int4(int(r), rp[r], 0, 0));
        r = e;
    }
    const int4 last = make_int4(int(n), int(nnz), 0, 0);
    int4* dt = nullptr;
    int32_t* dc = nullptr;
    std::vector<int32_t> cnt;
    cudaError_t e = cudaSuccess;
    auto count = [&]() {
        tiles.push_back(last);
        if (dt) cudaFree(dt);
        if (dc) cudaFree(dc);
        dt = nullptr;
        dc = nullptr;
        const int nt = int(tiles.size()) - 1;
        cnt.assign(nt, 0);
        e = cudaMalloc(&dt, tiles.size() * sizeof(int4));
        if (e == cudaSuccess) e = cudaMalloc(&dc, size_t(nt) * sizeof(int32_t));
        if (e == cudaSuccess) e = cudaMemcpy(dt, tiles.data(), tiles.size() * sizeof(int4), cudaMemcpyHostToDevice);
        if (e == cudaSuccess) {
            arrow_halo_kernel<false><<<std::min(nt, d.sm_count * 8), 256>>>(d.rowptr, d.col, dt, nt, dc, nullptr, nullptr, nullptr);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaMemcpy(cnt.data(), dc, size_t(nt) * sizeof(int32_t), cudaMemcpyDeviceToHost);
        tiles.pop_back();
    };
    auto release = [&](int rc) {
        if (dt) cudaFree(dt);
        if (dc) cudaFree(dc);
        return rc;
    };
    count();
    if (e != cudaSuccess) return release(cuda_fail(e, "arrow_upload: staged rows"));
    int64_t total = 0;
    for (int32_t c : cnt) total += c;
    if (total > 5 * n / 2) return release(ARROW_OK);
    // rows a stage holds: what all but one tile in a hundred (or in a thousand, if that takes little
    // more) need; the others (the head's tiles) are cut into smaller ones
    std::vector<int32_t> need(cnt.size());
    for (size_t t = 0; t < cnt.size(); ++t) need[t] = cnt[t] + (t + 1 < tiles.size() ? tiles[t + 1].x : int(n)) - tiles[t].x;
    std::vector<int32_t> srt = need;
    std::sort(srt.begin(), srt.end());
    const int p99 = srt[srt.size() * 99 / 100], p999 = srt[srt.size() * 999 / 1000], top = srt.back();
    const int cap = top <= p99 + p99 / 4 ? top : p999 <= p99 + p99 / 4 ? p999 : p99;
    if (top > cap) {
        std::vector<int4> cut;
        std::vector<int32_t> tmp;
        for (size_t t = 0; t < tiles.size(); ++t) {
            if (need[t] <= cap) cut.push_back(tiles[t]);
            else if (!split_tile(h, tiles[t].x, t + 1 < tiles.size() ? tiles[t + 1].x : int(n), cap, cut, tmp)) return release(ARROW_OK);
        }
        tiles.swap(cut);
        count();
        if (e != cudaSuccess) return release(cuda_fail(e, "arrow_upload: staged rows"));
    }
    const int nt = int(tiles.size());
    tiles.push_back(last);
    int64_t at = 0;
    int max_ent = 0, max_rows = 0;
    for (int t = 0; t < nt; ++t) {
        tiles[t].z = int(at);
        at += cnt[t];
        max_ent = std::max(max_ent, tiles[t + 1].y - tiles[t].y);
        max_rows = std::max(max_rows, tiles[t + 1].x - tiles[t].x);
    }
    tiles[nt].z = int(at);
    if (at > INT32_MAX) return release(ARROW_OK);
    constexpr size_t pad = 64;
    e = cudaMemcpy(dt, tiles.data(), tiles.size() * sizeof(int4), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMalloc(&d.st_halo, size_t(at) * 4 + pad);
    if (e == cudaSuccess) e = cudaMalloc(&d.st_col, size_t(nnz) * 2 + pad);
    if (e == cudaSuccess) e = cudaMalloc(&d.st_desc, size_t(n) * 4 + pad);
    if (e == cudaSuccess) e = cudaMemset(reinterpret_cast<char*>(d.st_col) + size_t(nnz) * 2, 0, pad);
    if (e == cudaSuccess) e = cudaMemset(reinterpret_cast<char*>(d.st_desc) + size_t(n) * 4, 0, pad);
    if (e == cudaSuccess) {
        arrow_halo_kernel<true><<<std::min(nt, d.sm_count * 8), 256>>>(d.rowptr, d.col, dt, nt, nullptr, d.st_halo, d.st_col,
                                                                       d.st_desc);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaDeviceSynchronize();
    }
    if (e != cudaSuccess) return release(cuda_fail(e, "arrow_upload: staged rows"));
    d.st_tile = dt;
    dt = nullptr;
    d.st_tiles = nt;
    d.st_cap = std::max(cap, max_rows);
    d.st_rows = max_rows;
    d.st_ent = max_ent;
    d.bytes += tiles.size() * sizeof(int4) + size_t(at) * 4 + size_t(nnz) * 2 + size_t(n) * 4 + 3 * pad;
    return release(ARROW_OK);
}

}  // namespace arrow
