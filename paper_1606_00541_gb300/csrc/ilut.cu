// ILUT(p, tol) on the GPU (Sec. 3 names ILUT; the dual-threshold rule is Saad's): for row i,
// tau_i = tol * ||a_i||_2; the row's entries k < i are eliminated in ascending column order,
// w_k <- w_k / u_kk, a multiplier with |w_k| < tau_i is dropped, otherwise w_j <- w_j - w_k u_kj
// for the entries j > k of U row k (creating fill); then entries below tau_i are dropped and
// the p largest magnitudes are kept in the strict lower and in the strict upper part (ties to
// the smaller column), the diagonal always.  L is unit lower with its 1.0 diagonal stored.
//
// GB300 design: one cooperative persistent launch.  The rows are cut into runs, stretches of
// consecutive rows each with an entry in the column before its own (a grid line, for a stencil).
// A run belongs to a group of warps, dealt out in turn (run r to group r mod G), and its rows to the
// group's warps in turn; every warp takes its rows in increasing order, so the smallest unfinished
// row can always proceed.  A row is tens of microseconds of work for one warp (a few for each
// pivot), so the time is (rows / rows that can work at once): dealt one by one over all warps, only
// W consecutive rows are in flight, half a plane of a 100^3 grid, whose wavefront keeps a few dozen of
// the 4,864 warps busy.  Groups put a dozen planes in flight, and a run held by a group holds back no row
// (each waits for the row before it anyway), while its warps work on the earlier pivots of the rows
// ahead.  With enough rows at work the FP64 unit counts (16 SM-cycles a warp instruction): per row
// about 25 divisions and 40 ranked candidates (268 FP64 warp instructions are left: the unit is busy 43 % of the time
// on 64^3 and, by that count, 62 % on 100^3; the rest is a pivot's flag and the loads behind it, one pivot after the other),
// so the ranking compares magnitudes as integers and the division takes five FP64 instructions (div_by).  27-point 100^3 / 7-point 100^3: 45.2 / 37.7 ms with
// FP64 compares and __ddiv_rn, 28.5 / 26.6 with integer compares, 22.0 / 23.2 with both.
//   The groups, before that.  ILUT(10, 1e-3) of the 27-point stencil on 100^3 / 64^3 and of the 7-point matrix on 100^3:
// row by row 167.6 / 45.1 / 189.0 ms, groups of 8 warps 45.2 / 17.2 / 37.7 (1 warp 100 / 39.7 / 110,
// 4 warps 61.4 / 22.2 / 56.2, 16 warps 54.4 / 20.0 / 43.0, 32 warps 147 / 41.5 / 153).  Where there
// are too few runs to give every group one, the groups grow (31 x 33 x 29: 4.9 / 5.2 ms); a group is never larger than a
// run of average length, since only as many of its warps have a row of a run (eight colours of the 27-point 64^3,
// runs of one row: groups of 8 warps 36.8 ms, of one 8.3; red-black 7-point 100^3 201 / 33.1).
//   A warp keeps its row as a sorted (column, value) list in shared memory; merging U row k is a
// warp-parallel binary search plus a ballot-ranked insertion of the fill.  A finished row is
// written into fixed slots (p strictly lower, 1 + p upper entries) and published with a release
// store of its U length; a row that needs U row k waits for that flag (acquire, bounded).  The
// arithmetic is the definition's, operation by operation and without fused multiply-adds
// (w_j - (w_k * u_kj), the norm summed in row order), so the drop decisions match any IEEE
// FP64 implementation that performs the same operations in the same order.
#include <algorithm>

#include "internal.cuh"
#include "quotient.cuh"
#include "sync.cuh"

namespace hec {
void free_csr(hec_csr* M);
hec_status validate_csr(int n, const int* rp, const int* col, int uplo, cudaStream_t s);

namespace {

constexpr unsigned kAll = 0xffffffffu;
// working-list capacity per warp and warps per block, tried in this order when a row's fill
// outgrows the list (24 bytes per entry and warp: two column and two value buffers)
constexpr int kCaps[4] = {120, 240, 1984, 9000};
constexpr int kWarpsFor[4] = {8, 8, 4, 1};

struct IlutParams {
    int n, p;
    double tol;
    const int* __restrict__ rp;
    const int* __restrict__ ci;
    const double* __restrict__ v;
    int* lcol;     // [n * p]
    double* lval;
    int* llen;     // [n]
    int* ucol;     // [n * (p + 1)], diagonal first
    double* uval;
    double* urcp;  // [n] reciprocals of the pivots
    int* ulen;     // [n], 0 until the row is published
    int* status;
    long long budget;
    int cap;       // entries of a row's working list
    const int* __restrict__ runs;  // [nruns + 1] first row of each run
    int nruns;
    int g;         // warps that share a run
    int* made;     // [kMade * 8] rows published, counted in kMade words of 32 bytes each
};
constexpr int kMade = 64;

__device__ __forceinline__ int ld_acquire_flag(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int ldcg_i(const int* p) { return __ldcg(p); }
__device__ __forceinline__ double ldcg_d(const double* p) { return __ldcg(p); }

// position of the first entry with column >= c in cols[lo, hi)
__device__ __forceinline__ int lower_bound(const int* cols, int lo, int hi, int c) {
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (cols[mid] < c) lo = mid + 1; else hi = mid;
    }
    return lo;
}

}  // namespace
}  // namespace hec

namespace hec {
namespace {

// publish U row i: its length is the flag later rows wait on (release after the warp's stores)
__device__ __forceinline__ void ilut_publish(const IlutParams& P, int i, int lane, int nu1) {
    __syncwarp();
    if (lane == 0) {
        atomicAdd(P.made + 8 * (blockIdx.x % kMade), 1);
        __threadfence();
        st_release_i32(P.ulen + i, nu1);
    }
    __syncwarp();
}

// U row k's length, waited for; -1 when the wait gave up.  A wait can span every row of the runs in flight (half of
// the matrix for one long chain), so its budget is for the time without any row published by anyone: when it
// has run out, the wait goes on if the count of rows has moved since it last ran out.
__device__ __forceinline__ int ilut_wait(const IlutParams& P, int k) {
    int ul = ld_acquire_flag(P.ulen + k);
    if (ul != 0) return ul;
    long long t0 = clock64();
    unsigned seen = 0u;  // rows published when the budget last ran out
    for (unsigned it = 1; (ul = ld_acquire_flag(P.ulen + k)) == 0; ++it) {
        if ((it & 63u) != 0u) continue;
        if (ld_relaxed_u32(P.status) != 0u) return -1;
        if (clock64() - t0 > P.budget) {
            unsigned made = 0u;
            for (int w = 0; w < kMade; ++w) made += ld_relaxed_u32(P.made + 8 * w);
            if (made == seen) return -1;
            seen = made;
            t0 = clock64();
        }
    }
    return ul;
}

// magnitude of a value as a word that compares like it (a NaN above everything)
__device__ __forceinline__ unsigned long long mag(double v) {
    return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
}

// One strict part of a finished row, list positions [b0, b1): the entries with w != 0 and
// |w| >= tau (least, as a word) are the candidates; the p largest magnitudes are kept (ties to the smaller column)
// and written to out_col / out_val in column order.  The candidates are first compacted, in
// column order, into the warp's spare buffer; up to 64 of them are ranked with shuffles (two per
// lane), more by a scan of the compacted list.  Returns the number kept.  Magnitudes are compared
// as integers: an FP64 compare occupies the SM's FP64 unit for 16 cycles, and four for each
// candidate were half of the kernel's FP64 instructions.
__device__ __forceinline__ int ilut_select(const int* col, const double* val, int b0, int b1, unsigned long long least, int p,
                                           int lane, int* scol, double* sval, int* out_col, double* out_val) {
    const unsigned lt = (1u << lane) - 1u;
    int m = 0;
    for (int bb = b0; bb < b1; bb += 32) {
        const int b = bb + lane;
        bool c = false;
        if (b < b1) {
            const unsigned long long v = mag(val[b]);
            c = v != 0ull && v >= least;
        }
        const unsigned cm = __ballot_sync(kAll, c);
        if (c) {
            scol[m + __popc(cm & lt)] = col[b];
            sval[m + __popc(cm & lt)] = val[b];
        }
        m += __popc(cm);
    }
    __syncwarp();
    if (m == 0 || p == 0) return 0;
    int kept = 0;
    if (m <= 64) {
        const bool h0 = lane < m, h1 = lane + 32 < m;
        const unsigned long long a0 = h0 ? mag(sval[lane]) : 0ull, a1 = h1 ? mag(sval[lane + 32]) : 0ull;
        int r0 = 0, r1 = 0;  // candidates ahead of this lane's two (larger, or equal with a smaller column)
        if (m > p) {
            for (int t = 0; t < m; ++t) {
                const unsigned long long at = __shfl_sync(kAll, t < 32 ? a0 : a1, t & 31);
                r0 += (t < lane ? at >= a0 : at > a0) ? 1 : 0;
                r1 += (t < lane + 32 ? at >= a1 : at > a1) ? 1 : 0;
            }
        }
        const bool k0 = h0 && r0 < p, k1 = h1 && r1 < p;
        const unsigned m0 = __ballot_sync(kAll, k0), m1 = __ballot_sync(kAll, k1);
        if (k0) { out_col[__popc(m0 & lt)] = scol[lane]; out_val[__popc(m0 & lt)] = sval[lane]; }
        if (k1) {
            out_col[__popc(m0) + __popc(m1 & lt)] = scol[lane + 32];
            out_val[__popc(m0) + __popc(m1 & lt)] = sval[lane + 32];
        }
        kept = __popc(m0) + __popc(m1);
    } else {
        for (int eb = 0; eb < m; eb += 32) {
            const int e = eb + lane;
            bool k = false;
            if (e < m) {
                const unsigned long long ae = mag(sval[e]);
                int rank = 0;
                for (int t = 0; t < m && rank < p; ++t) {
                    const unsigned long long at = mag(sval[t]);
                    rank += (t < e ? at >= ae : at > ae) ? 1 : 0;
                }
                k = rank < p;
            }
            const unsigned km = __ballot_sync(kAll, k);
            if (k) { out_col[kept + __popc(km & lt)] = scol[e]; out_val[kept + __popc(km & lt)] = sval[e]; }
            kept += __popc(km);
        }
    }
    __syncwarp();
    return kept;
}

// a row that cannot be factored (error recorded): diagonal 1.0 only, so later rows still finish
__device__ __forceinline__ void ilut_fail(const IlutParams& P, int i, int lane, int code) {
    if (lane == 0) {
        record(P.status, code);
        P.ucol[(long)i * (P.p + 1)] = i;
        P.uval[(long)i * (P.p + 1)] = 1.0;
        P.urcp[i] = 1.0;
        P.llen[i] = 0;
    }
    ilut_publish(P, i, lane, 1);
}

__global__ void __launch_bounds__(256) k_ilut(IlutParams P) {
    // per warp: values [2][cap] (8-byte aligned first), columns [2][cap], the merge's new columns [32]
    extern __shared__ __align__(16) unsigned char ilut_smem[];
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5, nwb = blockDim.x >> 5;
    const int cap = P.cap;
    double* wv = (double*)(ilut_smem + (size_t)wl * (24 * (size_t)cap + 128));
    int* wc = (int*)(wv + 2 * cap);
    int* s_newp = wc + 2 * cap;
    const int W = gridDim.x * nwb;
    const int up = P.p + 1;
    // the group of P.g warps this warp is in, its place there, the current run's next row of it and its end
    const int gid = blockIdx.x * nwb + wl;
    int run = gid / P.g, i = 0, rend = 0;
    const int place = gid % P.g, groups = W / P.g;
    if (run >= groups) return;  // the last warps do not fill a group
    for (;;) {
        i += P.g;
        if (i >= rend) {
            do {  // runs shorter than this warp's place have no row for it
                if (run >= P.nruns) return;
                i = __ldg(P.runs + run) + place;
                rend = __ldg(P.runs + run + 1);
                run += groups;
            } while (i >= rend);
        }
        int cur = 0;
        int* col = wc;
        double* val = wv;
        const int a0 = __ldg(P.rp + i);
        int len = __ldg(P.rp + i + 1) - a0;
        if (len + 1 > cap) { ilut_fail(P, i, lane, HEC_ERR_OUT_OF_BOUNDS); continue; }
        for (int e = lane; e < len; e += 32) {
            col[e] = __ldg(P.ci + a0 + e);
            val[e] = __ldg(P.v + a0 + e);
        }
        __syncwarp();
        // tau = tol * ||a_i||_2, the squares summed in row order
        double nrm = 0.0;
        for (int eb = 0; eb < len; eb += 32) {  // 32 squares with one instruction, then the sum in order
            const double v = eb + lane < len ? val[eb + lane] : 0.0;
            const double sq = __dmul_rn(v, v);
            const int m = min(32, len - eb);
            for (int e = 0; e < m; ++e) nrm = __dadd_rn(nrm, __shfl_sync(kAll, sq, e));
        }
        const double tau = __dmul_rn(P.tol, __dsqrt_rn(nrm));
        const unsigned long long least = isnan(tau) ? 0ull : mag(tau);  // a NaN tau drops nothing
        // a structural diagonal slot when the row has none
        {
            const int dpos = lower_bound(col, 0, len, i);
            if (dpos == len || col[dpos] != i) {
                int* ncol = (wc + (cur ^ 1) * cap);
                double* nval = (wv + (cur ^ 1) * cap);
                for (int e = lane; e < len; e += 32) {
                    ncol[e + (e >= dpos)] = col[e];
                    nval[e + (e >= dpos)] = val[e];
                }
                if (lane == 0) { ncol[dpos] = i; nval[dpos] = 0.0; }
                __syncwarp();
                cur ^= 1; col = ncol; val = nval; ++len;
            }
        }
        int failed = 0;  // the error code of a row that cannot be finished
        for (int pos = 0; pos < len && col[pos] < i; ++pos) {
            const int k = col[pos];
            int ul = 0;
            if (lane == 0) ul = ilut_wait(P, k);
            ul = __shfl_sync(kAll, ul, 0);
            if (ul < 0) { failed = HEC_ERR_TIMEOUT; break; }
            // U row k's first 32 entries in one batch of loads; u_kk is its first entry
            int j0 = 0;
            double u0 = 0.0;
            const double y = ldcg_d(P.urcp + k);
            if (lane < ul) {
                j0 = ldcg_i(P.ucol + (long)k * up + lane);
                u0 = ldcg_d(P.uval + (long)k * up + lane);
            }
            const double wk = div_by(val[pos], __shfl_sync(kAll, u0, 0), y);
            __syncwarp();
            if (mag(wk) < least) {  // dropped multiplier
                if (lane == 0) val[pos] = 0.0;
                __syncwarp();
                continue;
            }
            if (lane == 0) val[pos] = wk;
            __syncwarp();
            // w_j -= w_k * u_kj for the entries j > k of U row k (q >= 1), 32 at a time
            for (int qb = 0; qb < ul; qb += 32) {
                const int q = qb + lane;
                const bool has = q >= 1 && q < ul;
                int j = j0;
                double u = u0;
                if (qb > 0 && has) {
                    j = ldcg_i(P.ucol + (long)k * up + q);
                    u = ldcg_d(P.uval + (long)k * up + q);
                }
                const int at = has ? lower_bound(col, pos + 1, len, j) : len;
                const bool found = has && at < len && col[at] == j;
                const double prod = __dmul_rn(wk, u);
                if (found) val[at] = __dsub_rn(val[at], prod);
                const unsigned newm = __ballot_sync(kAll, has && !found);
                const int nnew = __popc(newm);
                __syncwarp();
                if (nnew == 0) continue;
                if (len + nnew > cap) { failed = HEC_ERR_OUT_OF_BOUNDS; break; }
                const int rk = __popc(newm & ((1u << lane) - 1u));
                if (has && !found) s_newp[rk] = j;
                __syncwarp();
                int* ncol = (wc + (cur ^ 1) * cap);
                double* nval = (wv + (cur ^ 1) * cap);
                for (int e = lane; e < len; e += 32) {
                    const int c = col[e];
                    int sh = 0;
                    for (int t = 0; t < nnew; ++t) sh += s_newp[t] < c;
                    ncol[e + sh] = c;
                    nval[e + sh] = val[e];
                }
                if (has && !found) {  // a fill entry: 0 - w_k u_kj
                    ncol[at + rk] = j;
                    nval[at + rk] = __dsub_rn(0.0, prod);
                }
                __syncwarp();
                cur ^= 1; col = ncol; val = nval; len += nnew;
            }
            if (failed) break;
        }
        if (failed) {
            ilut_fail(P, i, lane, failed);
            continue;
        }
        // drop below tau, keep the p largest of each strict part (ties to the smaller column); the
        // upper part first, so the rows waiting for U row i are released before the lower part
        const int dp = lower_bound(col, 0, len, i);
        const double wd = val[dp];
        if (wd == 0.0) { ilut_fail(P, i, lane, HEC_ERR_ZERO_PIVOT); continue; }
        int* scol = wc + (cur ^ 1) * cap;
        double* sval = wv + (cur ^ 1) * cap;
        const int nu = ilut_select(col, val, dp + 1, len, least, P.p, lane, scol, sval, P.ucol + (long)i * up + 1,
                                   P.uval + (long)i * up + 1);
        if (lane == 0) {
            P.ucol[(long)i * up] = i;
            P.uval[(long)i * up] = wd;
            P.urcp[i] = __drcp_rn(wd);
        }
        ilut_publish(P, i, lane, nu + 1);
        const int nl = ilut_select(col, val, 0, dp, least, P.p, lane, scol, sval, P.lcol + (long)i * P.p,
                                   P.lval + (long)i * P.p);
        if (lane == 0) P.llen[i] = nl;
    }
}

// run starts: rows without an entry in the column before their own, and every kRunRows-th row (a
// longer stretch is a chain however it is cut); kRunWarps is the least size of a group
constexpr int kRunRows = 4096;
constexpr int kRunWarps = 8;
__global__ void k_run_flags(int n, const int* __restrict__ rp, const int* __restrict__ ci, int* flag) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int a = rp[i], b = rp[i + 1];
    const int at = lower_bound(ci, a, b, i - 1);
    flag[i] = i % kRunRows == 0 || at == b || ci[at] != i - 1;
}
__global__ void k_run_starts(int n, const int* __restrict__ flag, const int* __restrict__ pos, int* runs) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n && flag[i]) runs[pos[i]] = i;
    if (i == 0) runs[pos[n]] = n;
}

// CSR of L (kept strict entries, then the unit diagonal) and U (diagonal first) from the slots
__global__ void k_ilut_rowlen(int n, const int* __restrict__ llen, const int* __restrict__ ulen, int* lrl, int* url) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        lrl[i] = llen[i] + 1;
        url[i] = ulen[i];
    }
}

__global__ void k_ilut_pack(int n, int p, const int* __restrict__ lrp, const int* __restrict__ llen,
                            const int* __restrict__ lcol, const double* __restrict__ lval, int* Lc, double* Lv,
                            const int* __restrict__ urp, const int* __restrict__ ucol, const double* __restrict__ uval,
                            int* Uc, double* Uv) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int l0 = lrp[i], nl = llen[i];
    for (int a = 0; a < nl; ++a) {
        Lc[l0 + a] = lcol[(long)i * p + a];
        Lv[l0 + a] = lval[(long)i * p + a];
    }
    Lc[l0 + nl] = i;
    Lv[l0 + nl] = 1.0;
    const int u0 = urp[i], nu = urp[i + 1] - u0;
    for (int a = 0; a < nu; ++a) {
        Uc[u0 + a] = ucol[(long)i * (p + 1) + a];
        Uv[u0 + a] = uval[(long)i * (p + 1) + a];
    }
}

}  // namespace
}  // namespace hec

using namespace hec;

HEC_API hec_status ilut_factor(int n, const int* rowptr, const int* col, const double* val, int p, double tol,
                               hec_csr** Lout, hec_csr** Uout, void* stream) {
    clear_error();
    if (!Lout || !Uout || n < 0 || p < 0 || !(tol >= 0.0) || (n > 0 && (!rowptr || !col || !val)))
        return set_error(HEC_ERR_INVALID_ARG, "ilut_factor: bad argument (need p >= 0, tol >= 0)");
    *Lout = *Uout = nullptr;
    cudaStream_t s = S(stream);
    HEC_CHECK(validate_csr(n, rowptr, col, -1, s));
    hec_csr *L = new hec_csr(), *U = new hec_csr();
    int *lcol = nullptr, *llen = nullptr, *ucol = nullptr, *ulen = nullptr, *status = nullptr, *lrl = nullptr,
        *url = nullptr, *runs = nullptr;
    double *lval = nullptr, *uval = nullptr, *urcp = nullptr;
    auto cleanup = [&]() {
        dfree(lcol); dfree(llen); dfree(ucol); dfree(ulen); dfree(status); dfree(lrl);
        dfree(url); dfree(runs); dfree(lval); dfree(uval); dfree(urcp);
    };
    auto fail = [&](hec_status e) {
        cleanup();
        free_csr(L);
        free_csr(U);
        return e;
    };
    hec_status st = HEC_OK;
    const size_t ln = (size_t)n * p + 1, un = (size_t)n * (p + 1) + 1;
    if ((st = dalloc(&lcol, ln)) || (st = dalloc(&lval, ln)) || (st = dalloc(&llen, (size_t)n + 1)) ||
        (st = dalloc(&ucol, un)) || (st = dalloc(&uval, un)) || (st = dalloc(&urcp, (size_t)n)) || (st = dalloc(&ulen, (size_t)n + 1)) ||
        (st = dalloc(&status, 8 + 8 * kMade)) || (st = dalloc(&lrl, (size_t)n + 1)) || (st = dalloc(&url, (size_t)n + 1)) ||
        (st = dalloc(&L->rowptr, (size_t)n + 1)) || (st = dalloc(&U->rowptr, (size_t)n + 1)))
        return fail(st);
    if (cudaMemsetAsync(ulen, 0, sizeof(int) * ((size_t)n + 1), s) != cudaSuccess ||
        cudaMemsetAsync(status, 0, sizeof(int) * (8 + 8 * kMade), s) != cudaSuccess)
        return fail(cuda_error(cudaGetLastError(), "ilut_factor: memset"));
    L->n = U->n = n;
    if (n > 0) {
        IlutParams P;
        P.n = n; P.p = p; P.tol = tol; P.rp = rowptr; P.ci = col; P.v = val;
        P.lcol = lcol; P.lval = lval; P.llen = llen; P.ucol = ucol; P.uval = uval; P.urcp = urcp; P.ulen = ulen;
        P.status = status;
        // the runs (lrl and url hold the flags and their prefix until the row lengths take them)
        const int gr = (n + 255) / 256;
        k_run_flags<<<gr, 256, 0, s>>>(n, rowptr, col, lrl);
        count_launch();
        if ((st = exclusive_scan_i32(lrl, url, n, true, s))) return fail(st);
        int nruns = 0;
        if (cudaMemcpyAsync(&nruns, url + n, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess)
            return fail(cuda_error(cudaGetLastError(), "ilut_factor: runs"));
        if ((st = dalloc(&runs, (size_t)nruns + 1))) return fail(st);
        k_run_starts<<<gr, 256, 0, s>>>(n, lrl, url, runs);
        count_launch();
        P.runs = runs;
        P.nruns = nruns;
        P.budget = 4000000000LL;  // about two seconds of SM cycles without a row published
        P.made = status + 8;
        const void* k = (const void*)k_ilut;
        int h = 0, cap = 0;
        // a larger working list (fewer warps per block) only when a row's fill outgrew the last one
        for (int t = 0; t < 4; ++t) {
            cap = kCaps[t];
            const int warps = kWarpsFor[t];
            const size_t smem = (size_t)warps * (24 * (size_t)cap + 128);
            if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
                return fail(cuda_error(cudaGetLastError(), "ilut_factor: shared memory"));
            const int per_sm = max_coop_blocks(k, warps * 32, smem);
            if (per_sm <= 0) return fail(set_error(HEC_ERR_CUDA, "ilut_factor: kernel cannot be resident"));
            const int blocks = (int)std::max(1L, std::min((long)per_sm * num_sms(), ((long)n + warps - 1) / warps));
            if (t > 0 && (cudaMemsetAsync(ulen, 0, sizeof(int) * ((size_t)n + 1), s) != cudaSuccess ||
                          cudaMemsetAsync(status, 0, sizeof(int), s) != cudaSuccess))
                return fail(cuda_error(cudaGetLastError(), "ilut_factor: memset"));
            P.cap = cap;
            P.g = std::max(kRunWarps, 2 * blocks * warps / std::max(1, nruns));
            P.g = std::max(1, std::min({P.g, blocks * warps, n / std::max(1, nruns)}));
            void* args[] = {&P};
            if (cudaLaunchCooperativeKernel(k, dim3(blocks), dim3(warps * 32), args, smem, s) != cudaSuccess)
                return fail(cuda_error(cudaGetLastError(), "ilut_factor: launch"));
            count_launch();
            if (cudaMemcpyAsync(&h, status, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
                cudaStreamSynchronize(s) != cudaSuccess)
                return fail(cuda_error(cudaGetLastError(), "ilut_factor"));
            if (h != HEC_ERR_OUT_OF_BOUNDS) break;
        }
        if (h == HEC_ERR_ZERO_PIVOT) return fail(set_error(HEC_ERR_ZERO_PIVOT, "ilut_factor: zero pivot"));
        if (h == HEC_ERR_OUT_OF_BOUNDS)
            return fail(set_error(HEC_ERR_OUT_OF_BOUNDS, "ilut_factor: a row's working fill exceeds " +
                                                             std::to_string(cap) + " entries"));
        if (h) return fail(set_error((hec_status)h, "ilut_factor: a dependency wait timed out"));
        const int g = (n + 255) / 256;
        k_ilut_rowlen<<<g, 256, 0, s>>>(n, llen, ulen, lrl, url);
        count_launch();
    }
    if ((st = exclusive_scan_i32(lrl, L->rowptr, n, true, s)) || (st = exclusive_scan_i32(url, U->rowptr, n, true, s)))
        return fail(st);
    int hl = 0, hu = 0;
    if (cudaMemcpy(&hl, L->rowptr + n, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(&hu, U->rowptr + n, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
        return fail(cuda_error(cudaGetLastError(), "ilut_factor: nnz"));
    L->nnz = hl;
    U->nnz = hu;
    if ((st = dalloc(&L->col, (size_t)hl)) || (st = dalloc(&L->val, (size_t)hl)) || (st = dalloc(&U->col, (size_t)hu)) ||
        (st = dalloc(&U->val, (size_t)hu)))
        return fail(st);
    if (n > 0) {
        k_ilut_pack<<<(n + 255) / 256, 256, 0, s>>>(n, p, L->rowptr, llen, lcol, lval, L->col, L->val, U->rowptr, ucol,
                                                   uval, U->col, U->val);
        count_launch();
    }
    if (cudaStreamSynchronize(s) != cudaSuccess) return fail(cuda_error(cudaGetLastError(), "ilut_factor: pack"));
    cleanup();
    *Lout = L;
    *Uout = U;
    return HEC_OK;
}
