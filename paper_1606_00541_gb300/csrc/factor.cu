// Incomplete LU factorization on the GPU: ILU(0), ILU(1) and ILU(k) (Sec. 3); the ILU(k) pattern for
// k >= 2 comes from iluk.cu.
//
// Row i of the factors needs the finished U rows of every q < i in its lower pattern, which is
// the same dependency structure as the triangular solve with L.  The numeric kernel therefore
// runs rows in the level order of the lower pattern with the same persistent, point-to-point
// scheme as the sweeps: a row waits (acquire) for the completion flag of each pivot row it
// uses, eliminates, and publishes its own flag (release) after its values are written.
//
// ILU(1)'s pattern adds to A the entries (i, j) reachable as i -> q -> j through an original
// entry a_iq (q < i) and an original entry a_qj (j > q): fill of level 1.  Each row's pattern is
// the sorted union of its own columns and the upper parts of its pivot rows, built by a k-way
// merge of those sorted lists (no dependency between rows, so this step is fully parallel).
#include <algorithm>

#include "internal.cuh"
#include "quotient.cuh"
#include "sync.cuh"

namespace hec {
hec_status validate_csr(int n, const int* rp, const int* col, int uplo, cudaStream_t s);
hec_status iluk_pattern(int n, const int* rp, const int* ci, int k, int** prp, int** pci, long long* nnz,
                        cudaStream_t s);
hec_status compute_levels(int n, const int* rp, const int* col, int dep_side, hec_levels* lv, cudaStream_t s);
void free_levels(hec_levels* lv);

namespace {

// diagonal positions; code[2] and code[3] receive the longest row and the most pivots in a row
__global__ void k_find_diag(int n, const int* __restrict__ rp, const int* __restrict__ col, int* dg, int* code) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int len = 0, npiv = 0;
    if (i < n) {
        const int a = rp[i], e = rp[i + 1];
        int d = -1;
        for (int p = a; p < e; ++p)
            if (col[p] == i) d = p;
        dg[i] = d;
        if (d < 0) atomicCAS(code, 0, HEC_ERR_MISSING_DIAG);
        len = e - a;
        npiv = d - a;
    }
    len = __reduce_max_sync(0xffffffffu, len);
    npiv = __reduce_max_sync(0xffffffffu, npiv);
    if ((threadIdx.x & 31) == 0) {
        if (len > code[2]) atomicMax(code + 2, len);
        if (npiv > code[3]) atomicMax(code + 3, npiv);
    }
}

// lu holds A's values on the pattern; on return the factors in place.  done[] zeroed.
// One warp per row, rows taken in the level order of the lower pattern (order[t]); the row's
// columns and values sit in shared memory (rows longer than kIluCap are worked in place in
// global memory).  For each pivot k < i in ascending order: every lane acquires row k's
// completion flag, l_ik = a_ik / u_kk, and the lanes split row k's upper entries, each finding
// its column in row i by binary search and applying a_ij <- fma(-l_ik, u_kj, a_ij).  Every entry
// receives the same operations in the same order as in a serial IKJ elimination.  The division is the
// corrected product with the pivot's reciprocal, kept with its row (div_by): the FP64 unit spends 16
// SM-cycles on a warp instruction, and with the compiler's division 13 pivots a row of the 27-point
// stencil on 100^3 are 8 ms of it.  ILU(0) of that matrix / of its 48^3 / ILU(1) of the 7-point 100^3, division /
// this: 11.0 / 9.5, 2.83 / 2.70, 7.0 / 6.6 ms.
constexpr int kIluCap = 256;
constexpr int kIluWarps = 8;

__device__ __forceinline__ int lower_bound_i(const int* c, int lo, int hi, int v) {
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (c[mid] < v) lo = mid + 1; else hi = mid;
    }
    return lo;
}

__global__ void __launch_bounds__(kIluWarps * 32) k_ilu_numeric(int n, const int* __restrict__ rp,
                                                                const int* __restrict__ col, const int* __restrict__ dg,
                                                                const int* __restrict__ order, double* lu, double* rcp, int* done,
                                                                int* status, long long budget) {
    __shared__ int s_col[kIluWarps][kIluCap];
    __shared__ double s_val[kIluWarps][kIluCap];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    const int W = gridDim.x * kIluWarps;
    for (int t = blockIdx.x * kIluWarps + wl; t < n; t += W) {
        const int i = __ldg(order + t);
        const int a = __ldg(rp + i), di = __ldg(dg + i), e = __ldg(rp + i + 1);
        const int len = e - a, dpos = di - a;
        const bool sm = len <= kIluCap;
        const int* rc = sm ? s_col[wl] : col + a;
        double* rv = sm ? s_val[wl] : lu + a;
        if (sm) {
            for (int q = lane; q < len; q += 32) {
                s_col[wl][q] = __ldg(col + a + q);
                s_val[wl][q] = lu[a + q];
            }
        }
        __syncwarp();
        bool bad = false;
        for (int p = 0; p < dpos; ++p) {
            const int k = rc[p];
            // Everything of row k but its values is known before it is finished: its range, the column of
            // this lane's first entry and that column's place in row i.  After the flag one load of values
            // remains, the pivot and the lane's entry together.
            const int dk = __ldg(dg + k), ek = __ldg(rp + k + 1);
            int q = dk + 1 + lane;
            int pos = len;
            auto place = [&]() {
                pos = len;
                if (q < ek) {
                    const int j = __ldg(col + q);
                    const int at = lower_bound_i(rc, p + 1, len, j);
                    if (at < len && rc[at] == j) pos = at;
                }
            };
            place();
            // every lane acquires row k (bounded), so its reads of row k are ordered after the release
            bool ready = ld_acquire_i32(done + k) != 0;
            if (!__all_sync(full, ready)) {
                const long long t0 = clock64();
                for (unsigned it = 1; !__all_sync(full, ready); ++it) {
                    ready = ld_acquire_i32(done + k) != 0;
                    if ((it & 63u) == 0u && __any_sync(full, clock64() - t0 > budget || ld_relaxed_u32(status) != 0u)) {
                        if (lane == 0) record(status, HEC_ERR_TIMEOUT);
                        bad = true;
                        break;
                    }
                }
            }
            if (bad) break;
            const double piv = lu[dk], y = rcp[k];
            double u = pos < len ? lu[q] : 0.0;
            if (piv == 0.0) {
                if (lane == 0) record(status, HEC_ERR_ZERO_PIVOT);
                continue;
            }
            const double lik = div_by(rv[p], piv, y);
            __syncwarp();
            if (lane == 0) rv[p] = lik;
            for (int qb = dk + 1; qb < ek; qb += 32) {
                if (qb > dk + 1) {
                    q = qb + lane;
                    place();
                    u = pos < len ? lu[q] : 0.0;
                }
                if (pos < len) rv[pos] = fma(-lik, u, rv[pos]);
            }
            __syncwarp();
        }
        if (sm)
            for (int q = lane; q < len; q += 32) lu[a + q] = s_val[wl][q];
        __syncwarp();
        if (lane == 0) {
            if (rv[dpos] == 0.0) record(status, HEC_ERR_ZERO_PIVOT);
            rcp[i] = __drcp_rn(rv[dpos]);
            __threadfence();
            st_release_i32(done + i, 1);
        }
        __syncwarp();
    }
}

// The elimination for short rows (at most kShortLen entries, kShortPiv of them pivots: the 5- and
// 7-point patterns): one thread per row, rows in the level order of the lower pattern, U's values
// their own flags.
//   What bounds it is the latency of a level: the values of the rows before must be seen and the
// row's own published.  One warp per row with a completion flag pays an acquire, a dependent load
// of the pivot row for each pivot, a fence and a release: 11 us a level.  Here the U values are
// words that start as the sentinel (sync.cuh) and are published one by one with relaxed stores, so a
// row needs no fence and reads all of its words together: each pivot row's diagonal and its first
// entry in this row's pattern (further matches, rare, one by one).  Which entries meet the pattern
// is found before the first wait, and entries that no pivot changes are published then, so that
// usually only the diagonals are waited for.
//   The rows of a warp lie scattered in memory: every word polled is a sector of its own, and more
// than one block an SM (two or three levels of 128^3 in flight) only adds polls.  A warp's rows of
// one level go together, since an FP64 division costs the same for one lane as for 32; a warp that
// holds the end of a level and the start of the next takes them in turn.
//   ilu_factor of the 7-point 128^3 matrix as a whole, warp per row / this: 5.77 / 2.33 ms (3.1 ms with the
// words of a warp's rows waited for lane by lane, 2.65 ms with every U value published at the end).
// The operations and their order are those of the kernel above.
constexpr int kShortLen = 8, kShortPiv = 4;
constexpr int kShortThreads = 256, kShortBlocks = 1;

// spin on one word (bounded); 0 when the wait gave up
__device__ __noinline__ double spin_u(const double* p, int* status, long long budget) {
    return wait_f64(p, status, budget);
}

__global__ void __launch_bounds__(kShortThreads) k_ilu_short(int n, const int* __restrict__ rp, const int* __restrict__ col,
                                                             const double* __restrict__ a, const int* __restrict__ dg,
                                                             const int* __restrict__ order, const int* __restrict__ level,
                                                             const int* __restrict__ lrp,
                                                             const int* __restrict__ urp, const int* __restrict__ uci,
                                                             double* lv, double* uv, int* status, long long budget) {
    __shared__ double s_val[kShortLen][kShortThreads];
    __shared__ int s_col[kShortLen][kShortThreads];
    const unsigned full = 0xffffffffu;
    const int tid = threadIdx.x;
    const int stride = gridDim.x * kShortThreads;
    for (int tb = blockIdx.x * kShortThreads + (tid & ~31); tb < n; tb += stride) {
        const int t = tb + (tid & 31);
        const bool act = t < n;
        int i = 0, len = 0, npiv = 0, lev = 0, l0 = 0, u0 = 0;
        int du[kShortPiv], mu[kShortPiv];         // U word of the pivot's diagonal, of its first match (-1: none)
        unsigned match[kShortPiv];                // per entry of the pivot row right of its diagonal: 4 bits, the
                                                  // position of its column in this row (15: not in the pattern)
        unsigned hit = 0;                         // positions of this row that some pivot changes
        unsigned pend = 0;                        // words still to be read: bit p the diagonal, bit 4 + p the match
        double piv[kShortPiv], mv[kShortPiv];
#pragma unroll
        for (int p = 0; p < kShortPiv; ++p) {
            du[p] = 0;
            mu[p] = -1;
            match[p] = 0xffffffffu;
            piv[p] = mv[p] = 0.0;
        }
        if (act) {
            i = __ldg(order + t);
            const int r0 = __ldg(rp + i);
            len = __ldg(rp + i + 1) - r0;
            npiv = __ldg(dg + i) - r0;
            lev = __ldg(level + i);
            l0 = __ldg(lrp + i);
            u0 = __ldg(urp + i);
#pragma unroll
            for (int e = 0; e < kShortLen; ++e)
                if (e < len) {
                    s_col[e][tid] = __ldg(col + r0 + e);
                    s_val[e][tid] = __ldg(a + r0 + e);
                }
#pragma unroll
            for (int p = 0; p < kShortPiv; ++p)
                if (p < npiv) {
                    const int k = s_col[p][tid];
                    const int b = __ldg(urp + k), ul = __ldg(urp + k + 1) - b;
                    du[p] = b;
                    pend |= 1u << p;
                    int pos = p + 1;
#pragma unroll 1
                    for (int q = 1; q < ul; ++q) {
                        const int j = __ldg(uci + b + q);
                        while (pos < len && s_col[pos][tid] < j) ++pos;
                        if (pos < len && s_col[pos][tid] == j) {
                            hit |= 1u << pos;
                            match[p] = (match[p] & ~(15u << (4 * (q - 1)))) | ((unsigned)pos << (4 * (q - 1)));
                            if (mu[p] < 0) {
                                mu[p] = b + q;
                                pend |= 16u << p;
                            }
                        }
                    }
                }
        }
        // U entries that no pivot changes are final: published before the first wait
        for (int e = npiv + 1; e < len; ++e)
            if (!((hit >> e) & 1u)) publish_f64(uv + u0 + e - npiv, s_val[e][tid]);
        // no entry left of the diagonal is changed by an earlier pivot: the quotients are independent
        const bool indep = (hit & ((1u << npiv) - 1u)) == 0u;
        bool todo = act;
        const long long t0 = clock64();
        // the warp's rows of its lowest level, then those of the next one
        while (__any_sync(full, todo)) {
            const int lowest = __reduce_min_sync(full, todo ? lev : 0x7fffffff);
            const bool now = todo && lev == lowest;
            for (unsigned it = 1; __any_sync(full, now && pend != 0u); ++it) {
                if (now) {
                    unsigned long long w[2 * kShortPiv];
#pragma unroll
                    for (int p = 0; p < kShortPiv; ++p) {
                        if ((pend >> p) & 1u) w[p] = ld_relaxed_u64(uv + du[p]);
                        if ((pend >> (4 + p)) & 1u) w[kShortPiv + p] = ld_relaxed_u64(uv + mu[p]);
                    }
#pragma unroll
                    for (int p = 0; p < kShortPiv; ++p) {
                        if (((pend >> p) & 1u) && w[p] != kSent64) {
                            piv[p] = __longlong_as_double((long long)w[p]);
                            pend &= ~(1u << p);
                        }
                        if (((pend >> (4 + p)) & 1u) && w[kShortPiv + p] != kSent64) {
                            mv[p] = __longlong_as_double((long long)w[kShortPiv + p]);
                            pend &= ~(16u << p);
                        }
                    }
                }
                if ((it & 63u) == 0u && (clock64() - t0 > budget || ld_relaxed_u32(status) != 0u)) {
                    record(status, HEC_ERR_TIMEOUT);  // every wait of the kernel ends: the factors are void
                    pend = 0u;
                }
            }
            if (now) {
                double lik[kShortPiv];
#pragma unroll
                for (int p = 0; p < kShortPiv; ++p) lik[p] = indep && p < npiv ? s_val[p][tid] / piv[p] : 0.0;
#pragma unroll
                for (int p = 0; p < kShortPiv; ++p)
                    if (p < npiv) {
                        if (piv[p] == 0.0) {
                            record(status, HEC_ERR_ZERO_PIVOT);
                            continue;
                        }
                        if (!indep) lik[p] = s_val[p][tid] / piv[p];
                        s_val[p][tid] = lik[p];
                        if (mu[p] < 0) continue;
                        int q = mu[p] - du[p];  // its first match, then the others
                        double u = mv[p];
                        for (unsigned rest = match[p] >> (4 * (q - 1));;) {
                            const int pos = (int)(rest & 15u);
                            s_val[pos][tid] = fma(-lik[p], u, s_val[pos][tid]);
                            do {
                                rest = (rest >> 4) | 0xf0000000u;
                                ++q;
                            } while ((rest & 15u) == 15u && q < kShortLen);
                            if (q >= kShortLen) break;
                            u = spin_u(uv + du[p] + q, status, budget);
                        }
                    }
                const double d = s_val[npiv][tid];
                if (d == 0.0) record(status, HEC_ERR_ZERO_PIVOT);
                for (int e = npiv + 1; e < len; ++e)
                    if ((hit >> e) & 1u) publish_f64(uv + u0 + e - npiv, s_val[e][tid]);
                publish_f64(uv + u0, d);
                for (int e = 0; e < npiv; ++e) lv[l0 + e] = s_val[e][tid];
                lv[l0 + npiv] = 1.0;
                todo = false;
            }
        }
    }
}

__global__ void k_split_len(int n, const int* __restrict__ rp, const int* __restrict__ dg, int* llen, int* ulen) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    llen[i] = dg[i] - rp[i] + 1;
    ulen[i] = rp[i + 1] - dg[i];
}

// L and U from the pattern and the factors in place; without `lu` only the columns, and U's values
// set to the sentinel (k_ilu_short writes the values)
__global__ void k_split(int n, const int* __restrict__ rp, const int* __restrict__ col, const int* __restrict__ dg,
                        const double* __restrict__ lu, const int* __restrict__ lrp, int* lci, double* lv,
                        const int* __restrict__ urp, int* uci, double* uv) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int ql = lrp[i];
    for (int p = rp[i]; p < dg[i]; ++p, ++ql) {
        lci[ql] = col[p];
        if (lu) lv[ql] = lu[p];
    }
    lci[ql] = i;
    if (lu) lv[ql] = 1.0;
    int qu = urp[i];
    for (int p = dg[i]; p < rp[i + 1]; ++p, ++qu) {
        uci[qu] = col[p];
        uv[qu] = lu ? lu[p] : __longlong_as_double((long long)kSent64);
    }
}

// ILU(1) pattern: the sorted union of row i's columns and, for each q < i in row i, the columns
// j > q of row q.  k-way merge over at most kMaxLists sorted lists.
constexpr int kMaxLists = 64;

template <bool kFill>
__global__ void k_ilu1_pattern(int n, const int* __restrict__ rp, const int* __restrict__ col,
                               const int* __restrict__ prp, int* pci, int* plen, int* code) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int head[kMaxLists], end[kMaxLists];
    int nl = 0;
    head[nl] = rp[i];
    end[nl] = rp[i + 1];
    nl++;
    for (int p = rp[i]; p < rp[i + 1]; ++p) {
        int q = col[p];
        if (q >= i) break;
        if (nl >= kMaxLists) {
            atomicCAS(code, 0, HEC_ERR_INVALID_ARG);
            return;
        }
        int a = rp[q], b = rp[q + 1];
        while (a < b && col[a] <= q) ++a;  // upper part of row q
        head[nl] = a;
        end[nl] = b;
        nl++;
    }
    int cnt = 0, last = -1;
    int out = kFill ? prp[i] : 0;
    while (true) {
        int best = 0x7fffffff;
        for (int l = 0; l < nl; ++l)
            if (head[l] < end[l]) best = min(best, col[head[l]]);
        if (best == 0x7fffffff) break;
        for (int l = 0; l < nl; ++l)
            if (head[l] < end[l] && col[head[l]] == best) head[l]++;
        if (best != last) {
            if (kFill) pci[out + cnt] = best;
            cnt++;
            last = best;
        }
    }
    if (!kFill) plen[i] = cnt;
}

// scatter A's values into the (sorted, superset) pattern; fill entries start at 0
__global__ void k_scatter_vals(int n, const int* __restrict__ rp, const int* __restrict__ col,
                               const double* __restrict__ val, const int* __restrict__ prp,
                               const int* __restrict__ pci, double* pv) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int q = prp[i];
    const int e = prp[i + 1];
    for (int p = prp[i]; p < e; ++p) pv[p] = 0.0;
    for (int p = rp[i]; p < rp[i + 1]; ++p) {
        while (q < e && pci[q] < col[p]) ++q;
        pv[q] = val[p];
    }
}

hec_status read_code(int* dcode, cudaStream_t s, int* h) {
    HEC_CUDA(cudaMemcpyAsync(h, dcode, sizeof(int), cudaMemcpyDeviceToHost, s));
    HEC_CUDA(cudaStreamSynchronize(s));
    return HEC_OK;
}

}  // namespace

void free_csr(hec_csr* M) {
    if (!M) return;
    dfree(M->rowptr);
    dfree(M->col);
    dfree(M->val);
    delete M;
}

}  // namespace hec

using namespace hec;

HEC_API hec_status hec_csr_get(const hec_csr* M, int* n, long long* nnz, const int** rowptr, const int** col,
                               const double** val) {
    if (!M) return set_error(HEC_ERR_INVALID_ARG, "hec_csr_get: NULL");
    if (n) *n = M->n;
    if (nnz) *nnz = M->nnz;
    if (rowptr) *rowptr = M->rowptr;
    if (col) *col = M->col;
    if (val) *val = M->val;
    return HEC_OK;
}

namespace hec {
namespace {
// keep (i, j) when j <= i (uplo 0) or j >= i (uplo 1), the diagonal excluded when strict
__device__ __forceinline__ bool keep_entry(int i, int j, int uplo, int strict) {
    return uplo == 0 ? (strict ? j < i : j <= i) : (strict ? j > i : j >= i);
}
__global__ void k_tri_count(int n, const int* __restrict__ rp, const int* __restrict__ col, int uplo, int strict,
                            int* __restrict__ len) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int c = 0;
    for (int p = rp[i]; p < rp[i + 1]; ++p) c += keep_entry(i, col[p], uplo, strict);
    len[i] = c;
}
__global__ void k_tri_fill(int n, const int* __restrict__ rp, const int* __restrict__ col, const double* __restrict__ val,
                           int uplo, int strict, const int* __restrict__ orp, int* __restrict__ ocol,
                           double* __restrict__ oval) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int o = orp[i];
    for (int p = rp[i]; p < rp[i + 1]; ++p)
        if (keep_entry(i, col[p], uplo, strict)) {
            ocol[o] = col[p];
            oval[o] = val[p];
            ++o;
        }
}
}  // namespace
}  // namespace hec

HEC_API hec_status csr_triangle(int n, const int* rowptr, const int* col, const double* val, int uplo, int strict,
                                hec_csr** out, void* stream) {
    clear_error();
    if (!out || n < 0 || (uplo != 0 && uplo != 1) || (n > 0 && (!rowptr || !col || !val)))
        return set_error(HEC_ERR_INVALID_ARG, "csr_triangle: bad argument");
    *out = nullptr;
    cudaStream_t s = S(stream);
    HEC_CHECK(validate_csr(n, rowptr, col, -1, s));
    hec_csr* T = new hec_csr();
    T->n = n;
    int* len = nullptr;
    hec_status st = HEC_OK;
    auto fail = [&](hec_status e) {
        dfree(len);
        free_csr(T);
        return e;
    };
    if ((st = dalloc(&len, (size_t)n + 1)) || (st = dalloc(&T->rowptr, (size_t)n + 1))) return fail(st);
    const int g = std::max(1, (n + 255) / 256);
    if (n > 0) k_tri_count<<<g, 256, 0, s>>>(n, rowptr, col, uplo, strict, len);
    count_launch();
    if ((st = exclusive_scan_i32(len, T->rowptr, n, true, s))) return fail(st);
    int nnz = 0;
    HEC_CUDA(cudaMemcpyAsync(&nnz, T->rowptr + n, sizeof(int), cudaMemcpyDeviceToHost, s));
    HEC_CUDA(cudaStreamSynchronize(s));
    T->nnz = nnz;
    if ((st = dalloc(&T->col, (size_t)std::max(nnz, 1))) || (st = dalloc(&T->val, (size_t)std::max(nnz, 1))))
        return fail(st);
    if (n > 0) k_tri_fill<<<g, 256, 0, s>>>(n, rowptr, col, val, uplo, strict, T->rowptr, T->col, T->val);
    count_launch();
    HEC_CUDA(cudaGetLastError());
    dfree(len);
    *out = T;
    return HEC_OK;
}

HEC_API hec_status hec_csr_destroy(hec_csr* M) {
    free_csr(M);
    return HEC_OK;
}

HEC_API hec_status ilu_factor(int n, const int* rowptr, const int* col, const double* val, int k, hec_csr** Lout,
                              hec_csr** Uout, void* stream) {
    clear_error();
    if (!Lout || !Uout || n < 0 || k < 0 || (n > 0 && (!rowptr || !col || !val)))
        return set_error(HEC_ERR_INVALID_ARG, "ilu_factor: bad argument (k must be >= 0)");
    *Lout = *Uout = nullptr;
    cudaStream_t s = S(stream);
    HEC_CHECK(validate_csr(n, rowptr, col, -1, s));
    int *dg = nullptr, *code = nullptr, *done = nullptr, *prp = nullptr, *pci = nullptr, *plen = nullptr;
    double *lu = nullptr, *rcp = nullptr;
    hec_levels* lv = nullptr;
    hec_csr *L = new hec_csr(), *U = new hec_csr();
    hec_status st = HEC_OK;
    auto cleanup = [&]() {
        dfree(dg); dfree(code); dfree(done); dfree(plen); dfree(lu); dfree(rcp);
        if (prp != rowptr) dfree(prp);
        if (pci != col) dfree(pci);
        free_levels(lv);
    };
    auto fail = [&](hec_status e) {
        cleanup();
        free_csr(L);
        free_csr(U);
        return e;
    };
    const int g = (n + 255) / 256;
    // [0] errors of the pattern, [1] of the elimination, [2] longest row, [3] most pivots in a row
    if ((st = dalloc(&code, 4))) return fail(st);
    HEC_CUDA(cudaMemsetAsync(code, 0, 4 * sizeof(int), s));
    int hcode = 0;
    long long pnnz = 0;
    // ---- pattern ----
    if (k == 0) {
        prp = const_cast<int*>(rowptr);
        pci = const_cast<int*>(col);
        int h = 0;
        if (n > 0) HEC_CUDA(cudaMemcpy(&h, rowptr + n, sizeof(int), cudaMemcpyDeviceToHost));
        pnnz = h;
    } else if (k >= 2) {
        if (n > 0) {
            if ((st = iluk_pattern(n, rowptr, col, k, &prp, &pci, &pnnz, s))) return fail(st);
            if ((st = dalloc(&lu, (size_t)pnnz))) return fail(st);
            k_scatter_vals<<<g, 256, 0, s>>>(n, rowptr, col, val, prp, pci, lu);
            count_launch();
        }
    } else {
        if ((st = dalloc(&plen, (size_t)n + 1)) || (st = dalloc(&prp, (size_t)n + 1))) return fail(st);
        if (n > 0) {
            k_ilu1_pattern<false><<<g, 256, 0, s>>>(n, rowptr, col, nullptr, nullptr, plen, code);
            count_launch();
        }
        if ((st = read_code(code, s, &hcode))) return fail(st);
        if (hcode) return fail(set_error(HEC_ERR_INVALID_ARG, "ilu_factor: a row has more than 63 pivots (ILU(1) limit)"));
        if ((st = exclusive_scan_i32(plen, prp, n, true, s))) return fail(st);
        int h = 0;
        HEC_CUDA(cudaMemcpy(&h, prp + n, sizeof(int), cudaMemcpyDeviceToHost));
        pnnz = h;
        if ((st = dalloc(&pci, (size_t)pnnz)) || (st = dalloc(&lu, (size_t)pnnz))) return fail(st);
        if (n > 0) {
            k_ilu1_pattern<true><<<g, 256, 0, s>>>(n, rowptr, col, prp, pci, nullptr, code);
            k_scatter_vals<<<g, 256, 0, s>>>(n, rowptr, col, val, prp, pci, lu);
            count_launch(2);
        }
    }
    if (n == 0) {
        if ((st = dalloc(&L->rowptr, 1)) || (st = dalloc(&U->rowptr, 1))) return fail(st);
        cudaMemset(L->rowptr, 0, sizeof(int));
        cudaMemset(U->rowptr, 0, sizeof(int));
        cleanup();
        *Lout = L;
        *Uout = U;
        return HEC_OK;
    }
    // ---- diagonal positions, levels of the lower pattern ----
    if ((st = dalloc(&dg, (size_t)n))) return fail(st);
    k_find_diag<<<g, 256, 0, s>>>(n, prp, pci, dg, code);
    count_launch();
    int hc[4] = {0, 0, 0, 0};
    HEC_CUDA(cudaMemcpyAsync(hc, code, sizeof(hc), cudaMemcpyDeviceToHost, s));
    HEC_CUDA(cudaStreamSynchronize(s));
    if (hc[0]) return fail(set_error(HEC_ERR_MISSING_DIAG, "ilu_factor: a row has no diagonal entry"));
    lv = new hec_levels();
    if ((st = compute_levels(n, prp, pci, 0, lv, s))) return fail(st);
    // ---- L (unit lower, diagonal stored) and U: row pointers and storage ----
    int *llen = nullptr, *ulen = nullptr;
    if ((st = dalloc(&llen, (size_t)n + 1)) || (st = dalloc(&ulen, (size_t)n + 1))) {
        dfree(llen);
        return fail(st);
    }
    k_split_len<<<g, 256, 0, s>>>(n, prp, dg, llen, ulen);
    count_launch();
    L->n = U->n = n;
    if ((st = dalloc(&L->rowptr, (size_t)n + 1)) || (st = dalloc(&U->rowptr, (size_t)n + 1)) ||
        (st = exclusive_scan_i32(llen, L->rowptr, n, true, s)) || (st = exclusive_scan_i32(ulen, U->rowptr, n, true, s))) {
        dfree(llen); dfree(ulen);
        return fail(st);
    }
    dfree(llen);
    dfree(ulen);
    int ln = 0, un = 0;
    HEC_CUDA(cudaMemcpyAsync(&ln, L->rowptr + n, sizeof(int), cudaMemcpyDeviceToHost, s));
    HEC_CUDA(cudaMemcpyAsync(&un, U->rowptr + n, sizeof(int), cudaMemcpyDeviceToHost, s));
    HEC_CUDA(cudaStreamSynchronize(s));
    L->nnz = ln;
    U->nnz = un;
    if ((st = dalloc(&L->col, (size_t)ln)) || (st = dalloc(&L->val, (size_t)ln)) || (st = dalloc(&U->col, (size_t)un)) ||
        (st = dalloc(&U->val, (size_t)un)))
        return fail(st);
    // ---- numeric elimination in level order ----
    // short rows: thread per row, straight into L and U; longer ones: warp per row, in place, then split
    const bool shortrows = hc[2] <= kShortLen && hc[3] <= kShortPiv;
    long long budget = 4000000000LL;
    int nn = n;
    int* status = code + 1;
    if (shortrows) {
        k_split<<<g, 256, 0, s>>>(n, prp, pci, dg, nullptr, L->rowptr, L->col, L->val, U->rowptr, U->col, U->val);
        count_launch();
        const int per_sm = std::min(kShortBlocks, max_coop_blocks((const void*)k_ilu_short, kShortThreads, 0));
        if (per_sm <= 0) return fail(set_error(HEC_ERR_CUDA, "factor kernel cannot be resident"));
        const int blocks = std::max(1, std::min(per_sm * num_sms(), (n + kShortThreads - 1) / kShortThreads));
        const double* av = k == 0 ? val : lu;
        void* args[] = {&nn, &prp, &pci, &av, &dg, &lv->iperm, &lv->level, &L->rowptr, &U->rowptr, &U->col, &L->val, &U->val, &status,
                        &budget};
        HEC_CUDA(cudaLaunchCooperativeKernel((const void*)k_ilu_short, dim3(blocks), dim3(kShortThreads), args, 0, s));
        count_launch();
    } else {
        if (k == 0) {
            if ((st = dalloc(&lu, (size_t)pnnz))) return fail(st);
            HEC_CUDA(cudaMemcpyAsync(lu, val, sizeof(double) * (size_t)pnnz, cudaMemcpyDeviceToDevice, s));
        }
        if ((st = dalloc(&done, (size_t)n)) || (st = dalloc(&rcp, (size_t)n))) return fail(st);
        HEC_CUDA(cudaMemsetAsync(done, 0, sizeof(int) * (size_t)n, s));
        const int threads = kIluWarps * 32;
        int per_sm = max_coop_blocks((const void*)k_ilu_numeric, threads, 0);
        if (per_sm <= 0) return fail(set_error(HEC_ERR_CUDA, "factor kernel cannot be resident"));
        int blocks = std::max(1, std::min(per_sm * num_sms(), (n + kIluWarps - 1) / kIluWarps));
        void* args[] = {&nn, &prp, &pci, &dg, &lv->iperm, &lu, &rcp, &done, &status, &budget};
        HEC_CUDA(cudaLaunchCooperativeKernel((const void*)k_ilu_numeric, dim3(blocks), dim3(threads), args, 0, s));
        count_launch();
    }
    int hs[2] = {0, 0};
    HEC_CUDA(cudaMemcpyAsync(hs, code, 2 * sizeof(int), cudaMemcpyDeviceToHost, s));
    HEC_CUDA(cudaStreamSynchronize(s));
    if (hs[1] == HEC_ERR_ZERO_PIVOT) return fail(set_error(HEC_ERR_ZERO_PIVOT, "ilu_factor: zero pivot"));
    if (hs[1]) return fail(set_error((hec_status)hs[1], "ilu_factor: dependency wait timed out"));
    if (!shortrows) {
        k_split<<<g, 256, 0, s>>>(n, prp, pci, dg, lu, L->rowptr, L->col, L->val, U->rowptr, U->col, U->val);
        count_launch();
    }
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return fail(cuda_error(e, "ilu_factor: split"));
    cleanup();
    *Lout = L;
    *Uout = U;
    return HEC_OK;
}
