// Level analysis (Eq. 2), the level-ordering map m (Eq. 3) and input validation.
//
// Levels are computed by one sync-free kernel: rows are visited in the order of the lower
// problem (i for L, n-1-i for the reversed U of Sec. 2.2) and each row waits, point to point,
// for the levels of its dependencies, which are always earlier in that order.  Work is handed
// out statically, chunk c to warp c mod W, under a cooperative launch that guarantees all warps
// are resident, so the warp holding the earliest unfinished chunk can always proceed.
//
// The map is a stable counting sort of rows by level (least-significant-digit radix passes
// over the level), which keeps the rows of each level in ascending order of the lower
// problem's index as Eq. 3 requires; it is exact integer work and bit-identical to the plain
// serial construction.
#include <algorithm>
#include <vector>

#include "internal.cuh"
#include "sync.cuh"

namespace hec {
namespace {

// ---- validation -----------------------------------------------------------------------------
// code: UNSORTED (row not strictly ascending, column out of range, bad rowptr),
// NOT_TRIANGULAR, MISSING_DIAG.  uplo: 0 lower, 1 upper, -1 general (only sortedness).
__global__ void k_validate(int n, const int* __restrict__ rp, const int* __restrict__ col, int uplo, int* code) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int a = rp[i], b = rp[i + 1];
    if (b < a || a < 0) { atomicCAS(code, 0, HEC_ERR_UNSORTED); return; }
    int prev = -1;
    bool diag = false;
    for (int p = a; p < b; ++p) {
        int j = col[p];
        if (j < 0 || j >= n || j <= prev) { atomicCAS(code, 0, HEC_ERR_UNSORTED); return; }
        prev = j;
        if (j == i) diag = true;
        if ((uplo == 0 && j > i) || (uplo == 1 && j < i)) { atomicCAS(code, 0, HEC_ERR_NOT_TRIANGULAR); return; }
    }
    if (uplo >= 0 && !diag) atomicCAS(code, 0, HEC_ERR_MISSING_DIAG);
}

// ---- levels ---------------------------------------------------------------------------------
// lower_only: treat only j < i (uplo 0) / j > i (uplo 1) as dependencies and ignore the rest
// (used for the lower pattern of a general matrix by the factorization).
//
// A warp takes a chunk of 32 consecutive rows of the lower problem, one a lane; chunk c goes to
// warp c mod W.  What bounds the kernel is the latency of the dependency chain (a poll of a level
// another warp publishes is an L2 round trip), so a lane's level is published as soon as it is
// final and not when the chunk is: rows that continue a grid line depend on the chunk before, and
// a chunk that publishes only as a whole would chain every chunk to its predecessor.
//  - Dependencies on earlier chunks are polled kLevBatch entries of the row at a time.
//  - Dependencies inside the chunk: with runs, maximal stretches of lanes each depending on the
//    lane before it, the levels of a run are l_i = max over j <= i of (e_j + i - j) (e: from the
//    earlier chunks), one segmented maximum scan of five shuffles; lane i is final when every lane
//    of its run up to i has all of its e.  Other dependencies on lanes of the same run add nothing
//    (the run already orders them).  Only a chunk with a dependency on a lane outside the run (a
//    grid line shorter than a chunk, an entry dropped from a factor) takes the general pass: 32
//    shuffles in lane order.  Either is done when a lane has just read its last outside level.
//  - The more warps are resident the more rows are in flight, but the polls of the warps that are
//    still far from the wavefront delay everyone's: with 64 warps an SM polling continuously one
//    analysis takes 10 to 300 ms.  So a warp that has not read a single level yet sleeps between
//    its polls; one that has read some polls continuously.
// Whole analysis (validation and sort included) of ILU(0) factors, publishing whole chunks / this:
// 7-point 128^3 (lines of whole chunks) 0.75 / 0.61 ms; 576 Schwarz boxes of 128^3 (lines of 34 rows)
// 59 / 0.80 ms; ILUT of the 27-point stencil on 100^3 about 80 / 1.4 ms.  One microsecond of sleep:
// with none 9.7, 160 and 56 ms for 128^3, 127^3 and that ILUT factor, with 1 us 0.61, 1.59 and 1.39, with
// 2 us 0.87, 1.44 and 1.11; with 32 warps an SM and no sleep 0.96, 1.37 and 1.11.
constexpr int kLevBatch = 4;
constexpr int kLevFarNs = 1000;

__global__ void __launch_bounds__(256, 8) k_levels(int n, const int* __restrict__ rp, const int* __restrict__ col, int uplo,
                                                int* level, int* nlev, int* status, long long budget) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    const int chunks = (n + 31) >> 5;
    const unsigned below = (2u << lane) - 1u;  // this lane and those before it
    int mymax = 0;
    for (int c = gw; c < chunks; c += nw) {
        const int base = c << 5, t = base + lane;
        const int i = uplo ? n - 1 - t : t;
        int lev = 0, p = 0, b = 0, cc[kLevBatch];
        unsigned intra = 0, pend = 0;  // lanes of this chunk this row depends on; slots of cc still to be read
        auto load_batch = [&]() {
#pragma unroll
            for (int q = 0; q < kLevBatch; ++q) cc[q] = p + q < b ? __ldg(col + p + q) : -1;
#pragma unroll
            for (int q = 0; q < kLevBatch; ++q) {
                const int j = cc[q];
                if (j < 0 || j >= n || !(uplo ? j > i : j < i)) continue;
                const int tj = uplo ? n - 1 - j : j;  // its position in the lower problem, < t
                if (tj >= base) intra |= 1u << (tj - base);
                else pend |= 1u << q;
            }
        };
        if (t < n) {
            p = __ldg(rp + i);
            b = __ldg(rp + i + 1);
            load_batch();
        }
        unsigned ready = 0u, out = 0u;  // lanes whose outside levels are all read; lanes published
        bool first = true;
        const long long t0 = clock64();
        unsigned failed = 0u;
        for (unsigned it = 1;; ++it) {
            if (it > 1u && !__any_sync(full, lev > 0)) __nanosleep(kLevFarNs);  // nothing has arrived: far ahead
            int v[kLevBatch];
#pragma unroll
            for (int q = 0; q < kLevBatch; ++q)
                if ((pend >> q) & 1u) v[q] = (int)ld_relaxed_u32(level + cc[q]);
#pragma unroll
            for (int q = 0; q < kLevBatch; ++q)
                if (((pend >> q) & 1u) && v[q] != kSentI) {
                    lev = max(lev, v[q] + 1);
                    pend &= ~(1u << q);
                }
            if (pend == 0u && p + kLevBatch < b) {
                p += kLevBatch;
                load_batch();
            }
            const unsigned now = __ballot_sync(full, pend == 0u && p + kLevBatch >= b);
            if (now != ready || first) {
                ready = now;
                first = false;
                const unsigned starts = __ballot_sync(full, lane == 0 || !((intra >> (lane - 1)) & 1u));
                const int rs = 31 - __clz((int)(starts & below));
                const unsigned mine = below & ~((1u << rs) - 1u);  // the run up to this lane
                int l;
                bool fin;
                if (!__any_sync(full, ((ready >> lane) & 1u) && (intra & ~mine))) {
                    l = lev - lane;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int u = __shfl_up_sync(full, l, o);
                        if (lane - o >= rs) l = max(l, u);
                    }
                    l += lane;
                    fin = (ready & mine) == mine;
                } else {
                    l = lev | (((ready >> lane) & 1u) ? 0 : (int)0x80000000);  // sign: not final
#pragma unroll
                    for (int d = 0; d < 32; ++d) {
                        const int u = __shfl_sync(full, l, d);
                        if ((intra >> d) & 1u) l = u < 0 ? (int)0x80000000 : l < 0 ? l : max(l, u + 1);
                    }
                    fin = l >= 0;
                }
                if (fin && !((out >> lane) & 1u) && t < n) {
                    publish_i32(level + i, l);
                    mymax = max(mymax, l + 1);
                }
                out = __ballot_sync(full, fin);
                if (out == full) break;
            } else if ((it & 63u) == 0u) {
                const bool give_up = clock64() - t0 > budget || failed != 0u;
                if (__any_sync(full, give_up)) {  // every wait of the kernel ends: the levels are void
                    record(status, HEC_ERR_TIMEOUT);
                    pend = 0u;
                    p = b;
                }
                failed = ld_relaxed_u32(status);
            }
        }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) mymax = max(mymax, __shfl_xor_sync(full, mymax, o));
    if (lane == 0 && mymax) atomicMax(nlev, mymax);
}

// ---- stable counting sort by level ------------------------------------------------------------
// Least-significant-digit passes of at most kRadixBits bits, as few and as even as the largest key
// allows: up to 1024 levels are one pass.  A tile of kTileItems keys is one warp's; what a pass
// costs besides the keys is its table of (digits x tiles) counts and their scan.
constexpr int kRadixBits = 10;
constexpr int kTileItems = 32 * 32;  // keys per warp tile
constexpr int kSortWarps = 4;        // warps per block (4 x 1024 counters: 16 KB of shared memory)

// key and value at position t: from the arrays, or, in the first pass of the level sort, the level of
// the row at position t of the lower problem and that original row
struct SortIn {
    const int* key;
    const int* val;
    const int* level;  // not NULL: the first pass of the level sort
    int uplo;
    __device__ __forceinline__ int row(int n, long t) const { return uplo ? n - 1 - (int)t : (int)t; }
    __device__ __forceinline__ int k(int n, long t) const { return level ? level[row(n, t)] : key[t]; }
    __device__ __forceinline__ int v(int n, long t) const { return level ? row(n, t) : val[t]; }
};

__global__ void k_digit_count(int n, SortIn in, int shift, int bits, int ntiles, int* counts) {
    extern __shared__ int sort_smem[];
    const int digits = 1 << bits;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int* cnt = sort_smem + warp * digits;
    const int tile = blockIdx.x * kSortWarps + warp;
    for (int d = lane; d < digits; d += 32) cnt[d] = 0;
    __syncwarp();
    if (tile < ntiles) {
        const long base = (long)tile * kTileItems;
#pragma unroll 8
        for (int k = lane; k < kTileItems; k += 32) {
            const long t = base + k;
            if (t < n) atomicAdd(cnt + ((in.k(n, t) >> shift) & (digits - 1)), 1);
        }
        __syncwarp();
        for (int d = lane; d < digits; d += 32) counts[(long)d * ntiles + tile] = cnt[d];
    }
}

// okey / oval: the sorted pairs (okey may be NULL); inv (may be NULL): inv[value] = its position
__global__ void k_digit_scatter(int n, SortIn in, int shift, int bits, int ntiles, const int* __restrict__ offs, int* okey,
                                int* oval, int* inv) {
    extern __shared__ int sort_smem[];
    const int digits = 1 << bits;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int* base = sort_smem + warp * digits;
    const int tile = blockIdx.x * kSortWarps + warp;
    if (tile >= ntiles) return;  // whole warp leaves together
    for (int d = lane; d < digits; d += 32) base[d] = offs[(long)d * ntiles + tile];
    __syncwarp();
    const unsigned lt = (1u << lane) - 1u;
    const long t0 = (long)tile * kTileItems;
    long t = t0 + lane;
    int kn = t < n ? in.k(n, t) : 0, vn = t < n ? in.v(n, t) : 0;  // one step ahead: the loads overlap the ranking
    for (int r = 0; r < kTileItems && t0 + r < n; r += 32, t += 32) {
        const bool ok = t < n;
        const int k = kn, v = vn;
        if (t + 32 < n) {
            kn = in.k(n, t + 32);
            vn = in.v(n, t + 32);
        }
        const int d = ok ? ((k >> shift) & (digits - 1)) : digits + lane;  // invalid lanes get unique digits
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const int rank = __popc(peers & lt);
        const int pos = ok ? base[d] + rank : 0;
        __syncwarp();
        if (ok && rank == 0) base[d] += __popc(peers);
        __syncwarp();
        if (ok) {
            if (okey) okey[pos] = k;
            oval[pos] = v;
            if (inv) inv[v] = pos;
        }
    }
}

// level_ptr from the scanned counts of a single pass (the first position of each digit), or from the
// sorted keys (every level has a row)
__global__ void k_level_ptr_offs(int nlev, int n, int ntiles, const int* __restrict__ offs, int* level_ptr) {
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l < nlev) level_ptr[l] = offs[(long)l * ntiles];
    if (l == nlev) level_ptr[l] = n;
}
__global__ void k_level_ptr_keys(int nlev, int n, const int* __restrict__ key, int* level_ptr) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < n && (p == 0 || key[p] != key[p - 1])) level_ptr[key[p]] = p;
    if (p == 0) level_ptr[nlev] = n;
}

// One sort by keys in [0, max_key]: passes and bits a pass
struct SortShape {
    int passes, bits, ntiles, blocks;
    size_t smem;
    SortShape(int n, long long max_key) {
        int b = 0;
        while ((1LL << b) <= max_key) b++;
        passes = std::max(1, (b + kRadixBits - 1) / kRadixBits);
        bits = std::max(1, (b + passes - 1) / passes);
        ntiles = (n + kTileItems - 1) / kTileItems;
        blocks = (ntiles + kSortWarps - 1) / kSortWarps;
        smem = sizeof(int) * ((size_t)kSortWarps << bits);
    }
    size_t counts() const { return ((size_t)ntiles << bits) + 1; }
};

}  // namespace

hec_status validate_csr(int n, const int* rp, const int* col, int uplo, cudaStream_t s) {
    if (n == 0) return HEC_OK;
    int* code = nullptr;
    HEC_CHECK(dalloc(&code, 1));
    cudaMemsetAsync(code, 0, sizeof(int), s);
    k_validate<<<(n + 255) / 256, 256, 0, s>>>(n, rp, col, uplo, code);
    count_launch();
    int h = 0;
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, code, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    dfree(code);
    if (e != cudaSuccess) return cuda_error(e, "validate");
    switch (h) {
        case 0: return HEC_OK;
        case HEC_ERR_UNSORTED: return set_error(HEC_ERR_UNSORTED, "CSR row not strictly ascending, column out of range or bad rowptr");
        case HEC_ERR_NOT_TRIANGULAR: return set_error(HEC_ERR_NOT_TRIANGULAR, "entry on the wrong side of the diagonal");
        case HEC_ERR_MISSING_DIAG: return set_error(HEC_ERR_MISSING_DIAG, "row without its diagonal entry");
        default: return set_error((hec_status)h, "invalid CSR");
    }
}

// Levels + map for a validated pattern.  dep_side: 0 = j < i, 1 = j > i.  Fills lv (device
// arrays allocated here).  Synchronizes.
hec_status compute_levels(int n, const int* rp, const int* col, int dep_side, hec_levels* lv, cudaStream_t s) {
    lv->n = n;
    lv->uplo = dep_side;
    HEC_CHECK(dalloc(&lv->level, (size_t)n));
    HEC_CHECK(dalloc(&lv->perm, (size_t)n));
    HEC_CHECK(dalloc(&lv->iperm, (size_t)n));
    int* dnlev = nullptr;
    int* status = nullptr;
    HEC_CHECK(dalloc(&dnlev, 2));
    status = dnlev + 1;
    HEC_CUDA(cudaMemsetAsync(dnlev, 0, 2 * sizeof(int), s));
    if (n > 0) {
        HEC_CUDA(cudaMemsetAsync(lv->level, 0xFF, sizeof(int) * (size_t)n, s));
        const int threads = 256;
        int per_sm = max_coop_blocks((const void*)k_levels, threads, 0);
        if (per_sm <= 0) { dfree(dnlev); return set_error(HEC_ERR_CUDA, "level kernel cannot be resident"); }
        int chunks = (n + 31) / 32;
        int blocks = std::min(per_sm * num_sms(), (chunks + threads / 32 - 1) / (threads / 32));
        blocks = std::max(blocks, 1);
        long long budget = 4000000000LL;
        int nn = n, up = dep_side;
        void* args[] = {&nn, (void*)&rp, (void*)&col, &up, &lv->level, &dnlev, &status, &budget};
        HEC_CUDA(cudaLaunchCooperativeKernel((const void*)k_levels, dim3(blocks), dim3(threads), args, 0, s));
        count_launch();
    }
    int h[2] = {0, 0};
    HEC_CUDA(cudaMemcpyAsync(h, dnlev, 2 * sizeof(int), cudaMemcpyDeviceToHost, s));
    HEC_CUDA(cudaStreamSynchronize(s));
    dfree(dnlev);
    if (h[1] != 0) return set_error((hec_status)h[1], "level analysis: dependency wait timed out");
    lv->nlev = h[0];
    HEC_CHECK(dalloc(&lv->level_ptr, (size_t)lv->nlev + 1));
    if (n == 0) {
        HEC_CUDA(cudaMemsetAsync(lv->level_ptr, 0, sizeof(int), s));
        HEC_CUDA(cudaStreamSynchronize(s));
        return HEC_OK;
    }
    // stable LSD radix sort of (level, row): the last pass writes the map and its inverse
    const SortShape sh(n, lv->nlev - 1);
    int *k0 = nullptr, *v0 = nullptr, *k1 = nullptr, *v1 = nullptr, *counts = nullptr;
    hec_status st = HEC_OK;
    if ((st = dalloc(&counts, sh.counts())) ||
        (sh.passes > 1 && ((st = dalloc(&k0, (size_t)n)) || (st = dalloc(&v0, (size_t)n)) || (st = dalloc(&k1, (size_t)n)) ||
                           (st = dalloc(&v1, (size_t)n))))) {
        dfree(k0); dfree(v0); dfree(k1); dfree(v1); dfree(counts);
        return st;
    }
    for (int ps = 0; ps < sh.passes && st == HEC_OK; ++ps) {
        const SortIn in{k0, v0, ps == 0 ? lv->level : nullptr, dep_side};
        const bool last = ps == sh.passes - 1;
        k_digit_count<<<sh.blocks, 32 * kSortWarps, sh.smem, s>>>(n, in, ps * sh.bits, sh.bits, sh.ntiles, counts);
        count_launch();
        st = exclusive_scan_i32(counts, counts, (int)(sh.counts() - 1), false, s);
        if (st != HEC_OK) break;
        k_digit_scatter<<<sh.blocks, 32 * kSortWarps, sh.smem, s>>>(n, in, ps * sh.bits, sh.bits, sh.ntiles, counts, k1,
                                                                    last ? lv->iperm : v1, last ? lv->perm : nullptr);
        count_launch();
        std::swap(k0, k1);
        std::swap(v0, v1);
    }
    if (st == HEC_OK) {
        if (sh.passes == 1)
            k_level_ptr_offs<<<lv->nlev / 256 + 1, 256, 0, s>>>(lv->nlev, n, sh.ntiles, counts, lv->level_ptr);
        else
            k_level_ptr_keys<<<(n + 255) / 256, 256, 0, s>>>(lv->nlev, n, k0, lv->level_ptr);
        count_launch();
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) st = cuda_error(e, "level sort");
    }
    dfree(k0); dfree(v0); dfree(k1); dfree(v1); dfree(counts);
    return st;
}

// Stable sort of (key, val) pairs by key, 0 <= key <= max_key, in place (LSD radix).  Synchronizes.
hec_status sort_pairs_i32(int* keys, int* vals, int n, int max_key, cudaStream_t s) {
    if (n <= 1) return HEC_OK;
    int *k1 = nullptr, *v1 = nullptr, *counts = nullptr;
    const SortShape sh(n, max_key);
    hec_status st = HEC_OK;
    if ((st = dalloc(&k1, (size_t)n)) || (st = dalloc(&v1, (size_t)n)) || (st = dalloc(&counts, sh.counts()))) {
        dfree(k1); dfree(v1); dfree(counts);
        return st;
    }
    int *ka = keys, *va = vals, *kb = k1, *vb = v1;
    for (int ps = 0; ps < sh.passes && st == HEC_OK; ++ps) {
        const SortIn in{ka, va, nullptr, 0};
        k_digit_count<<<sh.blocks, 32 * kSortWarps, sh.smem, s>>>(n, in, ps * sh.bits, sh.bits, sh.ntiles, counts);
        count_launch();
        st = exclusive_scan_i32(counts, counts, (int)(sh.counts() - 1), false, s);
        if (st != HEC_OK) break;
        k_digit_scatter<<<sh.blocks, 32 * kSortWarps, sh.smem, s>>>(n, in, ps * sh.bits, sh.bits, sh.ntiles, counts, kb, vb,
                                                                    nullptr);
        count_launch();
        std::swap(ka, kb);
        std::swap(va, vb);
    }
    if (st == HEC_OK && ka != keys) {
        cudaMemcpyAsync(keys, ka, sizeof(int) * (size_t)n, cudaMemcpyDeviceToDevice, s);
        cudaMemcpyAsync(vals, va, sizeof(int) * (size_t)n, cudaMemcpyDeviceToDevice, s);
    }
    cudaError_t e = cudaStreamSynchronize(s);
    if (st == HEC_OK && e != cudaSuccess) st = cuda_error(e, "sort");
    dfree(k1); dfree(v1); dfree(counts);
    return st;
}

void free_levels(hec_levels* lv) {
    if (!lv) return;
    dfree(lv->level);
    dfree(lv->perm);
    dfree(lv->iperm);
    dfree(lv->level_ptr);
    delete lv;
}

}  // namespace hec

using namespace hec;

HEC_API hec_status sptrsv_analyze(int n, const int* rowptr, const int* col, int uplo, hec_levels** out, void* stream) {
    clear_error();
    if (!out || n < 0 || (uplo != 0 && uplo != 1) || (n > 0 && (!rowptr || !col)))
        return set_error(HEC_ERR_INVALID_ARG, "sptrsv_analyze: bad argument");
    *out = nullptr;
    cudaStream_t s = S(stream);
    HEC_CHECK(validate_csr(n, rowptr, col, uplo, s));
    hec_levels* lv = new hec_levels();
    hec_status st = compute_levels(n, rowptr, col, uplo, lv, s);
    if (st != HEC_OK) { free_levels(lv); return st; }
    *out = lv;
    return HEC_OK;
}

HEC_API hec_status hec_levels_get(const hec_levels* lv, int* n, int* nlev, int* uplo, const int** level, const int** perm,
                                  const int** iperm, const int** level_ptr) {
    if (!lv) return set_error(HEC_ERR_INVALID_ARG, "hec_levels_get: NULL handle");
    if (n) *n = lv->n;
    if (nlev) *nlev = lv->nlev;
    if (uplo) *uplo = lv->uplo;
    if (level) *level = lv->level;
    if (perm) *perm = lv->perm;
    if (iperm) *iperm = lv->iperm;
    if (level_ptr) *level_ptr = lv->level_ptr;
    return HEC_OK;
}

HEC_API hec_status hec_levels_destroy(hec_levels* lv) {
    free_levels(lv);
    return HEC_OK;
}
