// AIRG setup on the GPU (Sec. 2 of arXiv 2508.17517), level by level:
//   truncation test (Sec. 2.4) -> strength + S+S^T -> PMISR -> DDC (Sec. 2.1)
//   -> block extraction (Eq. 3) -> GMRES polynomial coefficients (Eq. 7)
//   -> fixed-sparsity inverse (Eq. 8) -> Z = -A_cf Ahat^-1 with R drop
//   -> one-point W -> A_coarse = R A P with drop + lumping
// and finally the coarse-grid Newton polynomial (Sec. 2.3).
//
// Reproducibility: every value that feeds a discrete decision (strength,
// DDC bins, drops, one-point choice, truncation) is computed with a fixed
// operation order: row sums run left to right in column order from +0.0
// with explicitly rounded products (__dmul_rn/__dadd_rn, no FMA), sparse
// products accumulate each entry in ascending inner index, and dot products
// are correctly rounded (exact_dot.cuh).  The results are therefore the
// bits of the sequential definitions, whatever the launch shape.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdlib>
#include <cstring>

#include "dev_util.cuh"
#include "exact_dot.cuh"
#include "handle.h"
#include "hostmath.h"
#include "setup_index.h"

namespace airg {

namespace {

constexpr int TB = 256;
enum { PURPOSE_COEF = 1, PURPOSE_PMISR = 2, PURPOSE_COARSE = 3, PURPOSE_TRUNC = 4, PURPOSE_COEF_C = 5 };

// ------------------------------------------------------------- prefix sum --
constexpr int SCAN_B = 1024;

__global__ void k_scan_block(const int* in, int* out, int* sums, int n)
{
    __shared__ int wsum[32];
    int i = blockIdx.x * SCAN_B + threadIdx.x;
    int v = i < n ? in[i] : 0;
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[w] = x;
    __syncthreads();
    if (w == 0) {
        int s = wsum[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        wsum[lane] = s;
    }
    __syncthreads();
    int incl = x + (w > 0 ? wsum[w - 1] : 0);
    if (i < n) out[i] = incl - v;
    if (threadIdx.x == SCAN_B - 1) sums[blockIdx.x] = incl;
}

// single block: exclusive scan of the block sums, in chunks, in 64-bit;
// *total = -1 if any prefix exceeds the int32 index space
__global__ void k_scan_sums(int* sums, int nb, int* total)
{
    __shared__ long long wsum[32];
    __shared__ long long carry;
    __shared__ int overflow;
    if (threadIdx.x == 0) { carry = 0; overflow = 0; }
    __syncthreads();
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int base = 0; base < nb; base += SCAN_B) {
        int i = base + threadIdx.x;
        long long v = i < nb ? sums[i] : 0;
        long long x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            long long y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[w] = x;
        __syncthreads();
        if (w == 0) {
            long long s = wsum[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                long long y = __shfl_up_sync(0xffffffffu, s, o);
                if (lane >= o) s += y;
            }
            wsum[lane] = s;
        }
        __syncthreads();
        long long incl = x + (w > 0 ? wsum[w - 1] : 0);
        long long c = carry;
        long long ex = c + incl - v;
        if (i < nb) {
            if (ex > 0x7fffffffLL) overflow = 1;
            sums[i] = int(ex);
        }
        __syncthreads();
        if (threadIdx.x == SCAN_B - 1) carry = c + incl;
        __syncthreads();
    }
    if (threadIdx.x == 0) *total = (overflow || carry > 0x7fffffffLL) ? -1 : int(carry);
}

__global__ void k_scan_add(int* out, const int* sums, int n, const int* total)
{
    int i = blockIdx.x * SCAN_B + threadIdx.x;
    if (i < n) out[i] += sums[blockIdx.x];
    if (blockIdx.x == 0 && threadIdx.x == 0) out[n] = *total;
}

}  // namespace

void exclusive_scan_async(const int* in, int* out, int n, cudaStream_t st)
{
    int nb = std::max(1, (n + SCAN_B - 1) / SCAN_B);
    DBuf<int> sums(size_t(nb) + 1);
    k_scan_block<<<nb, SCAN_B, 0, st>>>(in, out, sums.p, n);
    k_scan_sums<<<1, SCAN_B, 0, st>>>(sums.p, nb, sums.p + nb);
    k_scan_add<<<nb, SCAN_B, 0, st>>>(out, sums.p, n, sums.p + nb);
    CK_LAUNCH();
    CK(cudaStreamSynchronize(st));   // sums is released on return
}

int exclusive_scan(const int* in, int* out, int n, cudaStream_t st)
{
    exclusive_scan_async(in, out, n, st);
    int total = read1(out + n, st);
    if (total < 0) fail(AIRG_ERR_OOM, "index space of a setup product exceeds 2^31 entries");
    return total;
}

namespace {

// ---------------------------------------------------------- random streams --
__device__ __forceinline__ unsigned long long sm64_mix(unsigned long long z)
{
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
    return z ^ (z >> 31);
}
constexpr unsigned long long SM64_GAMMA = 0x9e3779b97f4a7c15ULL;

inline unsigned long long host_mix(unsigned long long z)
{
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
    return z ^ (z >> 31);
}
inline unsigned long long stream_key(unsigned long long seed, long long level, long long purpose)
{
    unsigned long long tag = ((unsigned long long)level << 8) | (unsigned long long)purpose;
    return host_mix(seed + SM64_GAMMA * (tag + 1ULL));
}

__global__ void k_rng_uniform(unsigned long long key, long long n, double* out)
{
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    unsigned long long z = sm64_mix(key + SM64_GAMMA * (unsigned long long)(i + 1));
    out[i] = (double)(z >> 11) * 0x1.0p-53;
}

__global__ void k_rng_u32(unsigned long long key, long long n, unsigned* out)
{
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    unsigned long long z = sm64_mix(key + SM64_GAMMA * (unsigned long long)(i + 1));
    out[i] = (unsigned)(z >> 32);
}

// ------------------------------------------------------------- validation --
// Row i of a caller's CSR.  The row pointers are checked first (0 = rp[0] <=
// rp[i] <= rp[i+1] <= rp[n] = nnz); only a row whose bounds pass has its
// entries read.  flags: [0] columns out of range or not strictly
// ascending, [1] no stored diagonal, [2] bad row pointers, [3] a value that
// is not finite.
__global__ void k_validate(int n_rows, int n_cols, int nnz, const int* rp, const int* ci, const double* v,
                           int square, int* flags)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_rows) return;
    const int a = rp[i], b = rp[i + 1];
    if (a < 0 || b < a || b > nnz || (i == 0 && a != 0) || (i == n_rows - 1 && b != nnz)) {
        flags[2] = 1;
        return;
    }
    int prev = -1;
    bool diag = false;
    for (int k = a; k < b; ++k) {
        int j = ci[k];
        if (j <= prev || j < 0 || j >= n_cols) flags[0] = 1;
        if (!isfinite(v[k])) flags[3] = 1;
        prev = j;
        if (j == i) diag = true;
    }
    if (square && !diag) flags[1] = 1;
}

// ------------------------------------------------------- strength / graph --
__global__ void k_strength(int n, const int* rp, const int* ci, const double* v, double theta,
                           int8_t* s)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double m = 0.0;
    for (int k = rp[i]; k < rp[i + 1]; ++k)
        if (ci[k] != i && fabs(v[k]) > m) m = fabs(v[k]);
    double thr = __dmul_rn(theta, m);
    for (int k = rp[i]; k < rp[i + 1]; ++k)
        s[k] = (int8_t)(ci[k] != i && m > 0.0 && fabs(v[k]) >= thr);
}

__global__ void k_count_strong_t(int n, const int* rp, const int* ci, const int8_t* s, int* cnt)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int k = rp[i]; k < rp[i + 1]; ++k)
        if (s[k]) atomicAdd(cnt + ci[k], 1);
}

__global__ void k_fill_strong_t(int n, const int* rp, const int* ci, const int8_t* s,
                                const int* rpt, int* cursor, int* ct)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int k = rp[i]; k < rp[i + 1]; ++k)
        if (s[k]) {
            int j = ci[k];
            ct[rpt[j] + atomicAdd(cursor + j, 1)] = i;
        }
}

// insertion sort of each row's column list (rows are short)
__global__ void k_sort_rows(int n, const int* rp, int* c)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int a = rp[i] + 1; a < rp[i + 1]; ++a) {
        int key = c[a], b = a - 1;
        while (b >= rp[i] && c[b] > key) { c[b + 1] = c[b]; --b; }
        c[b + 1] = key;
    }
}

// sort each row's (col, val) pairs by column
__global__ void k_sort_rows_kv(int n, const int* rp, int* c, double* v)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int a = rp[i] + 1; a < rp[i + 1]; ++a) {
        int key = c[a];
        double val = v[a];
        int b = a - 1;
        while (b >= rp[i] && c[b] > key) { c[b + 1] = c[b]; v[b + 1] = v[b]; --b; }
        c[b + 1] = key;
        v[b + 1] = val;
    }
}

// row i of S + S^T: merge of the strong columns of row i and the sorted
// row i of S^T, without duplicates
__global__ void k_union(int n, const int* rp, const int* ci, const int8_t* s, const int* rpt,
                        const int* ct, const int* rpg, int* cg, int* cnt)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int a = rp[i], ae = rp[i + 1], b = rpt[i], be = rpt[i + 1];
    int c = 0, o = rpg ? rpg[i] : 0;
    while (true) {
        while (a < ae && !s[a]) ++a;
        if (a >= ae && b >= be) break;
        int ja = a < ae ? ci[a] : 0x7fffffff;
        int jb = b < be ? ct[b] : 0x7fffffff;
        int j = ja < jb ? ja : jb;
        if (ja == j) ++a;
        if (jb == j) ++b;
        if (cg) cg[o + c] = j;
        ++c;
    }
    if (cnt) cnt[i] = c;
}

// ------------------------------------------------------------------ PMISR --
__device__ __forceinline__ bool key_beats(int dj, unsigned wj, int j, int di, unsigned wi, int i)
{
    if (dj != di) return dj > di;
    if (wj != wi) return wj > wi;
    return j > i;
}

__global__ void k_pmisr_select(int n, const int* rpg, const int* cg, const unsigned* w,
                               const int8_t* state, int8_t* newf)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (state[i] != 0) { newf[i] = 0; return; }
    int di = rpg[i + 1] - rpg[i];
    int8_t sel = 1;
    for (int k = rpg[i]; k < rpg[i + 1]; ++k) {
        int j = cg[k];
        if (state[j] == 0 && key_beats(rpg[j + 1] - rpg[j], w[j], j, di, w[i], i)) { sel = 0; break; }
    }
    newf[i] = sel;
}

__global__ void k_pmisr_update(int n, const int* rpg, const int* cg, int8_t* state,
                               const int8_t* newf, int* undecided)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || state[i] != 0) return;
    if (newf[i]) { state[i] = 1; return; }
    for (int k = rpg[i]; k < rpg[i + 1]; ++k)
        if (newf[cg[k]]) { state[i] = 2; return; }
    atomicAdd(undecided, 1);
}

__global__ void k_state_to_f(int n, const int8_t* state, int8_t* is_f)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) is_f[i] = state[i] == 1;
}

// -------------------------------------------------------------------- DDC --
__global__ void k_ddc_ratio(int n, const int* rp, const int* ci, const double* v,
                            const int8_t* is_f, double* ratio, unsigned long long* rmax_bits)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long m = 0ULL;
    if (i < n && !is_f[i]) ratio[i] = -1.0;
    else if (i < n) {
        double s = 0.0, d = 0.0;
        for (int k = rp[i]; k < rp[i + 1]; ++k) {
            int j = ci[k];
            if (j == i) d = fabs(v[k]);
            else if (is_f[j]) s = __dadd_rn(s, fabs(v[k]));
        }
        const double r = d > 0.0 ? __ddiv_rn(s, d) : __longlong_as_double(0x7ff0000000000000LL);
        ratio[i] = r;
        m = (unsigned long long)__double_as_longlong(r);   // r >= 0: its bits order like its value
    }
    // one atomic for a warp's rows, and only where it raises the maximum: an
    // atomic per row on one address serialises the grid (1.2 ms a call on
    // average over the levels of 4096^2)
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long u = __shfl_xor_sync(0xffffffffu, m, o);
        m = u > m ? u : m;
    }
    if ((threadIdx.x & 31) == 0 && m > *(volatile unsigned long long*)rmax_bits) atomicMax(rmax_bits, m);
}

__global__ void k_ddc_bin(int n, const int8_t* is_f, const double* ratio, double rmax, int nbins,
                          int* bins, int* hist)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || !is_f[i]) return;
    double t = __dmul_rn(__ddiv_rn(ratio[i], rmax), (double)nbins);
    int b = (int)floor(t);
    if (b > nbins - 1) b = nbins - 1;
    bins[i] = b;
    atomicAdd(hist + b, 1);
}

__global__ void k_ddc_convert(int n, int8_t* is_f, const int* bins, int B)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n && is_f[i] && bins[i] >= B) is_f[i] = 0;
}

// ----------------------------------------------------------- local indices --
__global__ void k_flag_eq(int n, const int8_t* is_f, int want, int* flag)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) flag[i] = (is_f[i] == want);
}

__global__ void k_local_index(int n, const int8_t* is_f, int want, const int* excl, int* idx,
                              int* ids)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (is_f[i] == want) { idx[i] = excl[i]; ids[excl[i]] = i; }
    else idx[i] = -1;
}

// --------------------------------------------------------------- extract --
// rows: list of source rows (nullptr = identity); colmap: new column of each
// source column or -1 to drop (nullptr = keep all, same index)
__global__ void k_sub_count(int nr, const int* rows, const int* rp, const int* ci,
                            const int* colmap, int* cnt)
{
    int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= nr) return;
    int i = rows ? rows[r] : r;
    int c = 0;
    for (int k = rp[i]; k < rp[i + 1]; ++k)
        if (!colmap || colmap[ci[k]] >= 0) ++c;
    cnt[r] = c;
}

__global__ void k_sub_fill(int nr, const int* rows, const int* rp, const int* ci, const double* v,
                           const int* colmap, const int* orp, int* oci, double* ov)
{
    int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= nr) return;
    int i = rows ? rows[r] : r;
    int o = orp[r];
    for (int k = rp[i]; k < rp[i + 1]; ++k) {
        int j = colmap ? colmap[ci[k]] : ci[k];
        if (j >= 0) { oci[o] = j; ov[o] = v[k]; ++o; }
    }
}

// -------------------------------------------------------- Arnoldi pieces --
__global__ void k_spmv_det(int n, const int* rp, const int* ci, const double* v,
                           const double* x, double* y)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double s = 0.0;
    for (int k = rp[i]; k < rp[i + 1]; ++k) s = __dadd_rn(s, __dmul_rn(v[k], x[ci[k]]));
    y[i] = s;
}

__global__ void k_div_dev(long long n, double* out, const double* w, const double* h)
{
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = __ddiv_rn(w[i], *h);
}

__global__ void k_sub(long long n, const double* a, const double* b, double* out)
{
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = __dsub_rn(a[i], b[i]);
}

__global__ void k_newton_real_x(long long n, double* x, const double* r, double a)
{
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) x[i] = __dadd_rn(x[i], __ddiv_rn(r[i], a));
}

__global__ void k_newton_r(long long n, double* r, const double* w, double a)
{
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) r[i] = __dsub_rn(r[i], __ddiv_rn(w[i], a));
}

__global__ void k_newton_pair(long long n, double* x, const double* r, const double* w,
                              double* t, double a2, double mod2)
{
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double tt = __dsub_rn(__dmul_rn(a2, r[i]), w[i]);
    t[i] = tt;
    x[i] = __dadd_rn(x[i], __ddiv_rn(tt, mod2));
}

// --------------------------------------------------- fixed-sparsity powers --
__global__ void k_fsp_init(int n, const int* rp, const int* ci, double a0, double* acc)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int k = rp[i]; k < rp[i + 1]; ++k) acc[k] = ci[k] == i ? a0 : 0.0;
}

__device__ __forceinline__ int find_col(const int* ci, int lo, int hi, int j)
{
    while (lo < hi) {
        int mid = lo + ((hi - lo) >> 1);
        if (ci[mid] < j) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// Rows of at least FSP_WARP_ROW entries are computed by k_fsp_power_warp.
constexpr int FSP_WARP_ROW = 16;

__global__ void k_fsp_power(int n, const int* rp, const int* ci, const double* a,
                            const double* tprev, double* tout)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (rp[i + 1] - rp[i] >= FSP_WARP_ROW) return;
    for (int q = rp[i]; q < rp[i + 1]; ++q) {
        int j = ci[q];
        double s = 0.0;
        for (int p = rp[i]; p < rp[i + 1]; ++p) {
            int l = ci[p];
            int r = find_col(ci, rp[l], rp[l + 1], j);
            if (r < rp[l + 1] && ci[r] == j) s = __dadd_rn(s, __dmul_rn(a[p], tprev[r]));
        }
        tout[q] = s;
    }
}

// The long rows of k_fsp_power, one warp each: lane t computes the entries
// q = rp[i] + t, t + 32, ... of the row, each summed over the row's entries
// p in column order exactly as the one-thread kernel does.
__global__ void k_fsp_power_warp(int n, const int* rp, const int* ci, const double* a,
                                 const double* tprev, double* tout)
{
    const int lane = threadIdx.x & 31;
    const long long i = warp_index(blockIdx.x, blockDim.x, threadIdx.x);
    if (i >= n) return;
    const int r0 = rp[i], r1 = rp[i + 1];
    if (r1 - r0 < FSP_WARP_ROW) return;
    for (int q = r0 + lane; q < r1; q += 32) {
        const int j = ci[q];
        double s = 0.0;
        for (int p = r0; p < r1; ++p) {
            const int l = ci[p];
            const int r = find_col(ci, rp[l], rp[l + 1], j);
            if (r < rp[l + 1] && ci[r] == j) s = __dadd_rn(s, __dmul_rn(a[p], tprev[r]));
        }
        tout[q] = s;
    }
}

__global__ void k_fsp_acc(int nnz, double* acc, const double* T, double ak)
{
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < nnz) acc[k] = __dadd_rn(acc[k], __dmul_rn(ak, T[k]));
}

__global__ void k_scale(int nnz, double* v, double s)
{
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < nnz) v[k] = v[k] * s;
}

// -------------------------------------------------------------- SpGEMM ----
// C = A B.  An entry of C is the left-to-right sum of its products in
// ascending inner index (A's column), starting from +0.0.  The products of a
// row are numbered in that order (A's entries in turn, each with its row of
// B), and every path below adds products with the same column in that order.
// Rows are handled by the number of their products:
//   at most 8 / 32: a group of 8 / 32 lanes sorts them by column in
//     registers;
//   more: a warp adds them into a hash table in shared memory and ranks the
//     columns with a bitmap over their range.
//   rows with more distinct columns than GEMM_CAP: tables in global memory,
//     sorted by column in shared memory.
// The sorted rows go to a scratch piece and from there, packed, into C.
// Bound: latency of the loads of B's rows and of the shared-memory table, at
// 12-16 warps per SM.  Tables in global memory for every row, sized at twice
// the products, cleared and scanned as a whole and sorted with bitonic
// networks, took 1.20 s of the 4096^2 setup (restrictor and RAP together);
// this takes 0.35 s.
constexpr int GEMM_TINY = 8, GEMM_SMALL = 32;   // products per lane group
constexpr int GEMM_SLOTS = 1024, GEMM_SLOTS_LOW = 512;   // shared-memory table of a warp
constexpr int GEMM_CAP = GEMM_SLOTS / 4 * 3;    // distinct columns a table takes
constexpr int GEMM_LOW = GEMM_SLOTS_LOW / 4 * 3;   // products of a row of the smaller table
constexpr int GEMM_WORDS = 1024;                // bitmap words: columns within 32,768 of each other
constexpr int GEMM_WARPS = 4;                   // rows per block

__device__ __forceinline__ unsigned hash_col(int j) { return (unsigned)j * 2654435761u; }

// Products of each row (saturated at 2^30 - 1), and its scratch entries: never
// more than its products or GEMM_CAP.
__global__ void k_gemm_bound(int m, const int* arp, const int* aci, const int* brp, int* prod, int* room)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    long long b = 0;
    for (int p = arp[i]; p < arp[i + 1]; ++p) b += brp[aci[p] + 1] - brp[aci[p]];
    const int n = int(b < 0x3fffffffLL ? b : 0x3fffffffLL);
    prod[i] = n;
    room[i] = n < GEMM_CAP ? n : GEMM_CAP;
}

__device__ __forceinline__ int gemm_class(int b)
{
    return b <= 0 ? -1 : (b <= GEMM_TINY ? 0 : (b <= GEMM_SMALL ? 1 : (b <= GEMM_LOW ? 2 : 3)));
}

// Class lists of the rows of a piece (one aggregated atomic per warp and
// class; the order of a list does not matter), and zero counts for the rows
// without products.  lists: four of m entries each, counts: their lengths.
__global__ void k_gemm_lists(int m, const int* prod, int* lists, int* counts, int* cnt)
{
    const int li = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    const int cl = li < m ? gemm_class(prod[li]) : -1;
    if (li < m && cl < 0) cnt[li] = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const unsigned b = __ballot_sync(0xffffffffu, cl == c);
        if (!b) continue;
        int at = 0;
        if (lane == 0) at = atomicAdd(counts + c, __popc(b));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (cl == c) lists[(long long)c * m + at + __popc(b & ((1u << lane) - 1u))] = li;
    }
}

// Product f of the entries held by a group of G lanes: lane k holds an
// entry of A (value a, its row of B at bs) and `inc`, the number of products
// up to and including it.  Sets the product's column and value.
template <int G>
__device__ __forceinline__ void gemm_product(int f, int inc, int len, double a, int bs, const int* __restrict__ bci,
                                             const double* __restrict__ bv, bool valid, int& j, double& pr)
{
    const unsigned full = 0xffffffffu;
    int k = 0;
#pragma unroll
    for (int s = G / 2; s > 0; s >>= 1)
        if (__shfl_sync(full, inc, k + s - 1, G) <= f) k += s;
    const int before = __shfl_sync(full, inc - len, k, G), b0 = __shfl_sync(full, bs, k, G);
    const double ak = __shfl_sync(full, a, k, G);
    j = 0x7fffffff;
    pr = 0.0;
    if (valid) {
        const int q = b0 + (f - before);
        j = __ldg(bci + q);
        pr = __dmul_rn(ak, __ldg(bv + q));
    }
}

// Rows of at most G products (G = 8 or 32): one product per lane, sorted by
// (column, order) with a bitonic network; the first lane of each column adds
// the others in order.
template <int G>
__global__ void k_gemm_lanes(int nlist, const int* __restrict__ list, int row0, const int* __restrict__ arp,
                             const int* __restrict__ aci, const double* __restrict__ av,
                             const int* __restrict__ brp, const int* __restrict__ bci,
                             const double* __restrict__ bv, const int* __restrict__ toff, int* __restrict__ tci,
                             double* __restrict__ tv, int* __restrict__ cnt)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, g = lane & (G - 1);
    const long long at = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / G;
    const bool row = at < nlist;                  // uniform over the group
    if (!__any_sync(full, row)) return;
    const int li = row ? list[at] : 0, i = row0 + li;
    const int a0 = row ? arp[i] : 0, alen = row ? arp[i + 1] - a0 : 0;
    // A's entries with an empty row of B may exceed the lanes: only entries
    // with products are kept
    int have = 0, inc = 0, len = 0, bs = 0;
    double a = 0.0;
    const int most = __reduce_max_sync(full, alen);
    for (int p0 = 0; p0 < most; p0 += G) {
        const int p = p0 + g;
        int l = 0, n = 0, s = 0;
        if (p < alen) {
            l = aci[a0 + p];
            s = brp[l];
            n = brp[l + 1] - s;
        }
        const unsigned mask = __ballot_sync(full, n > 0) >> (lane & ~(G - 1)) & (G == 32 ? full : ((1u << (G & 31)) - 1u));
        // the t-th kept entry of this step goes to lane have + t
        const int t = g - have;
        const int src = t >= 0 && t < __popc(mask) ? int(__fns(mask, 0, t + 1)) : -1;
        const int sn = __shfl_sync(full, n, src < 0 ? 0 : src, G), ss = __shfl_sync(full, s, src < 0 ? 0 : src, G);
        if (src >= 0) {
            len = sn;
            bs = ss;
            a = av[a0 + p0 + src];
        }
        have += __popc(mask);
    }
    inc = len;
#pragma unroll
    for (int o = 1; o < G; o <<= 1) {
        const int u = __shfl_up_sync(full, inc, o, G);
        if (g >= o) inc += u;
    }
    const int total = __shfl_sync(full, inc, G - 1, G);
    int j;
    double v;
    gemm_product<G>(g, inc, len, a, bs, bci, bv, row && g < total, j, v);
    unsigned long long key = ((unsigned long long)(unsigned)j << 8) | (unsigned)g;
#pragma unroll
    for (int size = 2; size <= G; size <<= 1)
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            const unsigned long long ok = __shfl_xor_sync(full, key, stride, G);
            const double ov = __shfl_xor_sync(full, v, stride, G);
            const bool lower = (g & stride) == 0, up = (g & size) == 0;
            if (lower == up ? ok < key : ok > key) {
                key = ok;
                v = ov;
            }
        }
    j = int(key >> 8);
    const int prev = __shfl_up_sync(full, j, 1, G);
    const bool valid = row && g < total, head = valid && (g == 0 || prev != j);
    double s = __dadd_rn(0.0, v);
    bool more = head;
    for (int t = 1; t < G; ++t) {
        const int nj = __shfl_down_sync(full, j, t, G);
        const double nv = __shfl_down_sync(full, v, t, G);
        more = more && g + t < total && nj == j;
        if (!__any_sync(full, more)) break;
        if (more) s = __dadd_rn(s, nv);
    }
    const unsigned heads = __ballot_sync(full, head) >> (lane & ~(G - 1)) & (G == 32 ? full : ((1u << (G & 31)) - 1u));
    if (head) {
        const int o = toff[li] + __popc(heads & ((1u << g) - 1u));
        tci[o] = j;
        tv[o] = s;
    }
    if (row && g == 0) cnt[li] = __popc(heads);
}

// Adds the products of row i of A B, in order, into the warp's table: 32 at
// a time, lane by lane where several have the same column.  Returns the
// number of columns (their range in cmin, cmax), or -1 where they exceed
// three quarters of a full-size table.
template <int SLOTS>
__device__ __forceinline__ int gemm_accumulate(int i, const int* __restrict__ arp, const int* __restrict__ aci,
                                               const double* __restrict__ av, const int* __restrict__ brp,
                                               const int* __restrict__ bci, const double* __restrict__ bv,
                                               int* keys, double* vals, int size, int& cmin, int& cmax)
{
    const unsigned full = 0xffffffffu, lane = threadIdx.x & 31, below = (1u << lane) - 1u;
    const unsigned mask = unsigned(size) - 1u;
    int c = 0;
    const int a0 = arp[i], a1 = arp[i + 1];
    for (int p0 = a0; p0 < a1; p0 += 32) {
        const int p = p0 + int(lane);
        int len = 0, bs = 0;
        double a = 0.0;
        if (p < a1) {
            const int l = aci[p];
            a = av[p];
            bs = brp[l];
            len = brp[l + 1] - bs;
        }
        int inc = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(full, inc, o);
            if (lane >= o) inc += u;
        }
        const int total = __shfl_sync(full, inc, 31);
        int j, nj;
        double pr, npr;
        gemm_product<32>(int(lane), inc, len, a, bs, bci, bv, int(lane) < total, j, pr);
        for (int f0 = 0; f0 < total; f0 += 32, j = nj, pr = npr) {
            // the next 32 products load while these are added
            gemm_product<32>(f0 + 32 + int(lane), inc, len, a, bs, bci, bv, f0 + 32 + int(lane) < total, nj, npr);
            const bool take = f0 + int(lane) < total;
            unsigned h = hash_col(j) & mask;
            bool claimed = false;
            if (take) {
                cmin = min(cmin, j);
                cmax = max(cmax, j);
                while (true) {
                    int key = *(volatile int*)(keys + h);
                    if (key == -1) {
                        key = atomicCAS(keys + h, -1, j);
                        if (key == -1) {
                            vals[h] = 0.0;
                            claimed = true;
                            break;
                        }
                    }
                    if (key == j) break;
                    h = (h + 1u) & mask;
                }
            }
            __syncwarp();
            c += __popc(__ballot_sync(full, claimed));
            const unsigned same = __match_any_sync(full, take ? j : -1 - int(lane));
            const int rank = __popc(same & below), rounds = __reduce_max_sync(full, rank);
            for (int t = 0; t <= rounds; ++t) {
                if (take && rank == t) vals[h] = __dadd_rn(vals[h], pr);
                __syncwarp();
            }
            if (size == SLOTS && c > SLOTS / 4 * 3) return -1;   // at least a quarter stays free
        }
    }
    return c;
}

// The rows of a class list, one warp each: accumulate, rank the columns,
// write the row in column order to the scratch piece.  A row that does not
// fit gets count -1 and a place on the overflow list.
template <int SLOTS>
__global__ void __launch_bounds__(GEMM_WARPS * 32)
k_gemm_hash(int nlist, const int* __restrict__ list, int row0, const int* __restrict__ arp,
            const int* __restrict__ aci, const double* __restrict__ av, const int* __restrict__ brp,
            const int* __restrict__ bci, const double* __restrict__ bv, const int* __restrict__ prod,
            const int* __restrict__ toff, int* __restrict__ tci, double* __restrict__ tv, int* __restrict__ cnt,
            int* __restrict__ over, int* nover)
{
    extern __shared__ __align__(16) unsigned char gemm_raw[];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    double* vals = reinterpret_cast<double*>(gemm_raw) + w * SLOTS;
    int* keys = reinterpret_cast<int*>(reinterpret_cast<double*>(gemm_raw) + GEMM_WARPS * SLOTS) + w * SLOTS;
    unsigned* bits = reinterpret_cast<unsigned*>(reinterpret_cast<double*>(gemm_raw) + GEMM_WARPS * SLOTS) +
                     GEMM_WARPS * SLOTS + w * GEMM_WORDS;
    unsigned short* pre = reinterpret_cast<unsigned short*>(
                              reinterpret_cast<unsigned*>(reinterpret_cast<double*>(gemm_raw) + GEMM_WARPS * SLOTS) +
                              GEMM_WARPS * SLOTS + GEMM_WARPS * GEMM_WORDS) + w * GEMM_WORDS;
    const int at = blockIdx.x * GEMM_WARPS + w;
    if (at >= nlist) return;                      // uniform over the warp
    const int li = list[at], i = row0 + li;
    int size = 64;
    while (size < SLOTS && size < 2 * prod[li]) size <<= 1;
    for (int t = lane; t < size; t += 32) keys[t] = -1;
    __syncwarp();
    int cmin = 0x7fffffff, cmax = -1;
    const int c = gemm_accumulate<SLOTS>(i, arp, aci, av, brp, bci, bv, keys, vals, size, cmin, cmax);
    if (c < 0) {
        if (lane == 0) {
            cnt[li] = -1;
            over[atomicAdd(nover, 1)] = li;
        }
        return;
    }
    cmin = __reduce_min_sync(full, cmin);
    cmax = __reduce_max_sync(full, cmax);
    const int o = toff[li];
    const long long range = (long long)cmax - cmin + 1;
    if (range <= 32LL * GEMM_WORDS) {
        const int nw = int((range + 31) >> 5);
        for (int t = lane; t < nw; t += 32) bits[t] = 0u;
        __syncwarp();
        for (int t = lane; t < size; t += 32) {
            const int d = keys[t] - cmin;
            if (keys[t] >= 0) atomicOr(bits + (d >> 5), 1u << (d & 31));
        }
        __syncwarp();
        int carry = 0;
        for (int w0 = 0; w0 < nw; w0 += 32) {
            const int n = w0 + lane < nw ? __popc(bits[w0 + lane]) : 0;
            int inc = n;
#pragma unroll
            for (int q = 1; q < 32; q <<= 1) {
                const int u = __shfl_up_sync(full, inc, q);
                if (lane >= q) inc += u;
            }
            if (w0 + lane < nw) pre[w0 + lane] = (unsigned short)(carry + inc - n);
            carry += __shfl_sync(full, inc, 31);
        }
        __syncwarp();
        for (int t = lane; t < size; t += 32) {
            const int key = keys[t];
            if (key < 0) continue;
            const int d = key - cmin;
            const int r = int(pre[d >> 5]) + __popc(bits[d >> 5] & ((1u << (d & 31)) - 1u));
            tci[o + r] = key;
            tv[o + r] = vals[t];
        }
    } else {
        // columns too far apart for the bitmap: an entry's rank is the
        // number of smaller columns
        int* seen = reinterpret_cast<int*>(bits);
        int n = 0;
        for (int t0 = 0; t0 < size; t0 += 32) {
            const int key = keys[t0 + lane];
            const unsigned b = __ballot_sync(full, key >= 0);
            if (key >= 0) seen[n + __popc(b & ((1u << lane) - 1u))] = key;
            n += __popc(b);
        }
        __syncwarp();
        for (int t = lane; t < size; t += 32) {
            const int key = keys[t];
            if (key < 0) continue;
            int r = 0;
            for (int q = 0; q < n; ++q) r += seen[q] < key;
            tci[o + r] = key;
            tv[o + r] = vals[t];
        }
    }
    if (lane == 0) cnt[li] = c;
}
inline size_t gemm_smem(int slots) { return size_t(GEMM_WARPS) * (size_t(slots) * 12 + GEMM_WORDS * 6); }

// Rows of the scratch piece to their packed place, a warp for 32 rows.
__global__ void k_gemm_pack(int m, const int* __restrict__ toff, const int* __restrict__ crp,
                            const int* __restrict__ cnt, const int* __restrict__ tci,
                            const double* __restrict__ tv, int* __restrict__ cci, double* __restrict__ cv)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int r0 = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32;
    if (r0 >= m) return;
    const int r = r0 + lane;
    const int n = r < m ? max(cnt[r], 0) : 0, s = r < m ? toff[r] : 0, d = r < m ? crp[r] : 0;
    // lanes over the entries of the 32 rows together
    int inc = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(full, inc, o);
        if (lane >= o) inc += u;
    }
    const int total = __shfl_sync(full, inc, 31);
    for (int f0 = 0; f0 < total; f0 += 32) {
        const int f = f0 + lane;
        int k = 0;
#pragma unroll
        for (int q = 16; q > 0; q >>= 1)
            if (__shfl_sync(full, inc, k + q - 1) <= f) k += q;
        const int before = __shfl_sync(full, inc - n, k), ss = __shfl_sync(full, s, k), dd = __shfl_sync(full, d, k);
        if (f < total) {
            cci[dd + f - before] = tci[ss + f - before];
            cv[dd + f - before] = tv[ss + f - before];
        }
    }
}

// Rows of the overflow list: tables in global memory, one warp each.  The
// entries of A's row are taken one at a time, in column order, by the whole
// warp; the lanes share that entry's row of B, whose columns are distinct.
// tsize: slots of each row's table, -1 for more than 32-bit offsets reach.
__global__ void k_gemm_table_size(int nlist, const int* list, const int* prod, int n_cols, int* tsize)
{
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nlist) return;
    const long long size = gemm_table_slots(prod[list[t]], n_cols);
    tsize[t] = size <= GEMM_MAX_SLOTS ? int(size) : -1;
}

__global__ void k_gemm_hash_global(int nlist, const int* list, int row0, const int* arp, const int* aci,
                                   const double* av, const int* brp, const int* bci, const double* bv,
                                   const int* toff, int* keys, double* vals, int* cnt, int* run_cnt)
{
    const int lane = threadIdx.x & 31;
    const int at = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (at >= nlist) return;                   // uniform over the warp
    const int i = row0 + list[at];
    const int base = toff[at], size = toff[at + 1] - base;
    const unsigned mask = (unsigned)size - 1u;
    int c = 0;
    for (int p = arp[i]; p < arp[i + 1]; ++p) {
        const int l = aci[p];
        const double a = av[p];
        for (int q = brp[l] + lane; q < brp[l + 1]; q += 32) {
            const int j = bci[q];
            const double prod = __dmul_rn(a, bv[q]);
            unsigned h = hash_col(j) & mask;
            while (true) {
                int key = *(volatile int*)(keys + base + h);
                if (key == -1) {
                    key = atomicCAS(keys + base + h, -1, j);
                    if (key == -1) {
                        vals[base + h] = __dadd_rn(0.0, prod);
                        ++c;
                        break;
                    }
                }
                if (key == j) {
                    vals[base + h] = __dadd_rn(vals[base + h], prod);
                    break;
                }
                h = (h + 1u) & mask;
            }
        }
        __syncwarp();
    }
    for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
    if (lane == 0) cnt[list[at]] = run_cnt[at] = c;
}

// Their entries in column order, packed, one block per row: the table's
// occupied slots go to the row's place, are sorted by column EMIT_CHUNK at a
// time in shared memory, and in rows of several chunks each entry's rank is
// its position in its own chunk plus its lower bounds in the others (the
// columns of a row are distinct).  The sorted chunks wait in the table, which
// has at least twice as many slots as the row has entries and is not needed
// any more.  Bound: latency of the scan of the table, which is read once.
// Ranking every entry against all slots, of a table sized by the products,
// took entries x slots reads: setup of 3,142 rows of 61 entries (coarse rows
// of 2,048) 1160 -> 18.8 ms, of 6,354 rows 4067 -> 46.4 ms.
constexpr int EMIT_CHUNK = 2048;

__global__ void __launch_bounds__(TB)
k_gemm_emit_global(const int* toff, int* keys, double* vals, const int* crp, int* cci, double* cv)
{
    __shared__ int k[EMIT_CHUNK];
    __shared__ double v[EMIT_CHUNK];
    __shared__ int filled;
    const int lane = threadIdx.x & 31;
    const int o = crp[blockIdx.x], n = crp[blockIdx.x + 1] - o, t0 = toff[blockIdx.x], t1 = toff[blockIdx.x + 1];
    if (threadIdx.x == 0) filled = 0;
    __syncthreads();
    for (int tb = t0; tb < t1; tb += TB) {
        const int t = tb + threadIdx.x;
        const int key = t < t1 ? keys[t] : -1;
        const unsigned b = __ballot_sync(0xffffffffu, key >= 0);
        int at = 0;
        if (lane == 0 && b) at = atomicAdd(&filled, __popc(b));
        at = o + __shfl_sync(0xffffffffu, at, 0) + __popc(b & ((1u << lane) - 1u));
        if (key >= 0) {
            cci[at] = key;
            cv[at] = vals[t];
        }
    }
    __syncthreads();
    for (int c0 = 0; c0 < n; c0 += EMIT_CHUNK) {
        const int m = min(EMIT_CHUNK, n - c0);
        int size = 1;
        while (size < m) size <<= 1;
        for (int t = threadIdx.x; t < size; t += TB) {
            k[t] = t < m ? cci[o + c0 + t] : 0x7fffffff;
            v[t] = t < m ? cv[o + c0 + t] : 0.0;
        }
        __syncthreads();
        for (int run = 2; run <= size; run <<= 1)
            for (int stride = run >> 1; stride > 0; stride >>= 1) {
                for (int p = threadIdx.x; p < size / 2; p += TB) {
                    const int t = 2 * p - (p & (stride - 1)), u = t + stride;
                    const int a = k[t], b = k[u];
                    if ((a > b) == ((t & run) == 0) && a != b) {
                        k[t] = b;
                        k[u] = a;
                        const double x = v[t];
                        v[t] = v[u];
                        v[u] = x;
                    }
                }
                __syncthreads();
            }
        for (int t = threadIdx.x; t < m; t += TB) {
            if (n <= EMIT_CHUNK) {
                cci[o + t] = k[t];
                cv[o + t] = v[t];
            } else {
                keys[t0 + c0 + t] = k[t];
                vals[t0 + c0 + t] = v[t];
            }
        }
        __syncthreads();
    }
    if (n <= EMIT_CHUNK) return;
    for (int e = threadIdx.x; e < n; e += TB) {
        const int key = keys[t0 + e], own = e / EMIT_CHUNK;
        int r = e - own * EMIT_CHUNK;
        for (int c = 0; c * EMIT_CHUNK < n; ++c) {
            if (c == own) continue;
            const int* q = keys + t0 + c * EMIT_CHUNK;
            int lo = 0, hi = min(EMIT_CHUNK, n - c * EMIT_CHUNK);
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (q[mid] < key) lo = mid + 1;
                else hi = mid;
            }
            r += lo;
        }
        cci[o + r] = key;
        cv[o + r] = vals[t0 + e];
    }
}

// Packed rows src of a list to their places in C, one warp each.
__global__ void k_gemm_pack_list(int nlist, const int* list, const int* srp, const int* crp, const int* sci,
                                 const double* sv, int* cci, double* cv)
{
    const int lane = threadIdx.x & 31, at = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (at >= nlist) return;
    const int o = crp[list[at]] - srp[at];
    for (int t = srp[at] + lane; t < srp[at + 1]; t += 32) {
        cci[o + t] = sci[t];
        cv[o + t] = sv[t];
    }
}

// overflow rows: empty in the scratch piece
__global__ void k_gemm_mark(int nlist, const int* list, int* cnt)
{
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < nlist) cnt[list[t]] = 0;
}

__global__ void k_sum_int(int n, const int* __restrict__ x, unsigned long long* out)
{
    unsigned long long s = 0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        s += (unsigned long long)x[i];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0 && s) atomicAdd(out, s);
}

__global__ void k_shift_rowptr(int m, const int* prp, int off, int* crp)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < m) crp[i] = prp[i] + off;
}

// ------------------------------------------------------------ drop rules --
__global__ void k_drop_rows(int n, const int* rp, const double* v, double tol, int8_t* keep,
                            int* cnt)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double m = 0.0;
    for (int k = rp[i]; k < rp[i + 1]; ++k)
        if (fabs(v[k]) > m) m = fabs(v[k]);
    double thr = __dmul_rn(tol, m);
    int c = 0;
    for (int k = rp[i]; k < rp[i + 1]; ++k) {
        int8_t kp = (int8_t)(v[k] != 0.0 && fabs(v[k]) >= thr);
        keep[k] = kp;
        c += kp;
    }
    cnt[i] = c;
}

__global__ void k_drop_lump(int n, const int* rp, const int* ci, const double* v, double tol,
                            int lump, int8_t* keep, double* vout, int* cnt, int* bad)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double m = 0.0;
    int dpos = -1;
    for (int k = rp[i]; k < rp[i + 1]; ++k) {
        if (ci[k] == i) dpos = k;
        else if (fabs(v[k]) > m) m = fabs(v[k]);
    }
    if (dpos < 0) { *bad = 1; cnt[i] = 0; return; }
    double thr = __dmul_rn(tol, m);
    double d = v[dpos];
    int c = 0;
    for (int k = rp[i]; k < rp[i + 1]; ++k) {
        vout[k] = v[k];
        if (k == dpos) { keep[k] = 1; ++c; continue; }
        if (v[k] == 0.0 || fabs(v[k]) < thr) {
            keep[k] = 0;
            if (lump) d = __dadd_rn(d, v[k]);
        } else {
            keep[k] = 1;
            ++c;
        }
    }
    vout[dpos] = d;
    cnt[i] = c;
}

// The three row kernels above and below for rows of more than a few entries:
// one warp per row, adjacent lanes on adjacent entries, with the same
// decisions and the same order of the sums.
__global__ void k_drop_rows_warp(int n, const int* __restrict__ rp, const double* __restrict__ v, double tol,
                                 int8_t* __restrict__ keep, int* __restrict__ cnt)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const long long i = warp_index(blockIdx.x, blockDim.x, threadIdx.x);
    if (i >= n) return;
    const int b = rp[i], e = rp[i + 1];
    double m = 0.0;
    for (int k = b + lane; k < e; k += 32)
        if (fabs(v[k]) > m) m = fabs(v[k]);
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(full, m, o));
    const double thr = __dmul_rn(tol, m);
    int c = 0;
    for (int k0 = b; k0 < e; k0 += 32) {
        const int k = k0 + lane;
        const double x = k < e ? v[k] : 0.0;
        const bool kp = x != 0.0 && fabs(x) >= thr;
        if (k < e) keep[k] = (int8_t)kp;
        c += __popc(__ballot_sync(full, kp));
    }
    if (lane == 0) cnt[i] = c;
}

__global__ void k_drop_lump_warp(int n, const int* __restrict__ rp, const int* __restrict__ ci,
                                 const double* __restrict__ v, double tol, int lump, int8_t* __restrict__ keep,
                                 double* __restrict__ vout, int* __restrict__ cnt, int* bad)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const long long i = warp_index(blockIdx.x, blockDim.x, threadIdx.x);
    if (i >= n) return;
    const int b = rp[i], e = rp[i + 1];
    double m = 0.0;
    int dpos = -1;
    for (int k = b + lane; k < e; k += 32) {
        if (ci[k] == i) dpos = k;
        else if (fabs(v[k]) > m) m = fabs(v[k]);
    }
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(full, m, o));
    dpos = __reduce_max_sync(full, dpos);
    if (dpos < 0) {
        if (lane == 0) {
            *bad = 1;
            cnt[i] = 0;
        }
        return;
    }
    const double thr = __dmul_rn(tol, m);
    double d = v[dpos];
    int c = 0;
    for (int k0 = b; k0 < e; k0 += 32) {
        const int k = k0 + lane;
        const bool in = k < e;
        const double x = in ? v[k] : 0.0;
        const bool drop = in && k != dpos && (x == 0.0 || fabs(x) < thr);
        if (in) {
            keep[k] = (int8_t)!drop;
            if (k != dpos) vout[k] = x;
        }
        c += __popc(__ballot_sync(full, in && !drop));
        if (lump)
            for (unsigned left = __ballot_sync(full, drop); left; left &= left - 1u)
                d = __dadd_rn(d, __shfl_sync(full, x, __ffs(left) - 1));
    }
    if (lane == 0) {
        vout[dpos] = d;
        cnt[i] = c;
    }
}

__global__ void k_compact_warp(int n, const int* __restrict__ rp, const int* __restrict__ ci,
                               const double* __restrict__ v, const int8_t* __restrict__ keep,
                               const int* __restrict__ nrp, int* __restrict__ nci, double* __restrict__ nv)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const long long i = warp_index(blockIdx.x, blockDim.x, threadIdx.x);
    if (i >= n) return;
    const int b = rp[i], e = rp[i + 1];
    int o = nrp[i];
    for (int k0 = b; k0 < e; k0 += 32) {
        const int k = k0 + lane;
        const bool kp = k < e && keep[k];
        const unsigned on = __ballot_sync(full, kp);
        if (kp) {
            const int at = o + __popc(on & ((1u << lane) - 1u));
            nci[at] = ci[k];
            nv[at] = v[k];
        }
        o += __popc(on);
    }
}

__global__ void k_compact(int n, const int* rp, const int* ci, const double* v,
                          const int8_t* keep, const int* nrp, int* nci, double* nv)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int o = nrp[i];
    for (int k = rp[i]; k < rp[i + 1]; ++k)
        if (keep[k]) { nci[o] = ci[k]; nv[o] = v[k]; ++o; }
}

// --------------------------------------------------------- one-point W ----
__global__ void k_one_point(int n, const int* rp, const int* ci, const double* v,
                            const int8_t* strong, const int8_t* is_f, const int* c_index,
                            const int* f_index, int* W)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || !is_f[i]) return;
    int best = -1;
    for (int pass = 0; pass < 2 && best < 0; ++pass) {
        double bestv = -1.0;
        for (int k = rp[i]; k < rp[i + 1]; ++k) {
            int j = ci[k];
            if (j == i || is_f[j]) continue;
            if (pass == 0 && !strong[k]) continue;
            double a = fabs(v[k]);
            if (a > bestv) { bestv = a; best = j; }
        }
    }
    W[f_index[i]] = best >= 0 ? c_index[best] : -1;
}

// P = [W; I] in the fine numbering: one entry (weight 1) per row
__global__ void k_p_count(int n, const int8_t* is_f, const int* f_index, const int* W, int* cnt)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) cnt[i] = is_f[i] ? (W[f_index[i]] >= 0) : 1;
}

__global__ void k_p_fill(int n, const int8_t* is_f, const int* f_index, const int* c_index,
                         const int* W, const int* prp, int* pci, double* pv)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || prp[i + 1] == prp[i]) return;
    pci[prp[i]] = is_f[i] ? W[f_index[i]] : c_index[i];
    pv[prp[i]] = 1.0;
}

// R = [Z I] in the fine numbering: row c holds Z's row (F columns mapped to
// their fine index) and a 1 at the C point itself, columns ascending
__global__ void k_r_rowptr(int nc, const int* zrp, int* rrp)
{
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c <= nc) rrp[c] = zrp[c] + c;
}

__global__ void k_r_fill(int nc, const int* zrp, const int* zci, const double* zv,
                         const int* f_ids, const int* c_ids, const int* rrp, int* rci, double* rv)
{
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= nc) return;
    int o = rrp[c], self = c_ids[c];
    bool done = false;
    for (int k = zrp[c]; k < zrp[c + 1]; ++k) {
        int col = f_ids[zci[k]];
        if (!done && self < col) { rci[o] = self; rv[o] = 1.0; ++o; done = true; }
        rci[o] = col;
        rv[o] = zv[k];
        ++o;
    }
    if (!done) { rci[o] = self; rv[o] = 1.0; }
}

// ------------------------------------------------------------- transpose --
__global__ void k_count_cols(int n, const int* rp, const int* ci, int* cnt)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int k = rp[i]; k < rp[i + 1]; ++k) atomicAdd(cnt + ci[k], 1);
}

__global__ void k_fill_transpose(int n, const int* rp, const int* ci, const double* v,
                                 const int* trp, int* cursor, int* tci, double* tv)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int k = rp[i]; k < rp[i + 1]; ++k) {
        int j = ci[k];
        int pos = trp[j] + atomicAdd(cursor + j, 1);
        tci[pos] = i;
        tv[pos] = v[k];
    }
}

// =========================================================================
// host-side building blocks
// =========================================================================
struct Ctx {
    cudaStream_t st;
    DBuf<unsigned long long> xacc;   // exact-dot accumulator
    DBuf<int> xbad;
    DBuf<unsigned> xticket;          // last-block ticket of k_xdot
    long long ndots = 0;             // exact dot products launched
    HBuf<double> hcol;               // one Hessenberg column on the host
    // grid state of k_mgs_column: accumulators, barrier arrivals, and what
    // earlier launches left there
    DBuf<unsigned long long> cdig;
    DBuf<unsigned> cbar;
    unsigned cbase = 0;
    int cphase = 0;
    bool columns = true;             // false once a launch of it gave up waiting
    long long spin_limit = XC_SPIN_LIMIT;
    explicit Ctx(cudaStream_t s) : st(s)
    {
        xacc.alloc(XD_DIGITS);
        xbad.alloc(1);
        xticket.alloc(1);
        CK(cudaMemsetAsync(xacc.p, 0, xacc.bytes(), st));
        CK(cudaMemsetAsync(xbad.p, 0, xbad.bytes(), st));
        CK(cudaMemsetAsync(xticket.p, 0, xticket.bytes(), st));
        cdig.alloc(3 * XD_DIGITS);
        cbar.alloc(1);
        CK(cudaMemsetAsync(cdig.p, 0, cdig.bytes(), st));
        CK(cudaMemsetAsync(cbar.p, 0, cbar.bytes(), st));
        if (const char* e = getenv("AIRG_COLUMN_SPINS")) spin_limit = std::max(0LL, atoll(e));
    }
};

int num_sms()
{
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        CK(cudaGetDevice(&dev));
        CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    }
    return sms;
}

void xdot(Ctx& c, long long n, const double* x, const double* y, double* out, double* out_sqrt)
{
    const int grid = xd_grid(n, num_sms());
    k_xdot<<<grid, XD_THREADS, 0, c.st>>>(n, x, y, c.xacc.p, c.xbad.p, c.xticket.p, out, out_sqrt);
    CK_LAUNCH();
    ++c.ndots;
}

// MGS step w -= (*hprev) vprev (skipped when vprev is null) fused with the
// correctly rounded <w, y> (y null: <w, w>) into out / out_sqrt.
void mgs_xdot(Ctx& c, long long n, double* w, const double* vprev, const double* hprev, const double* y,
              double* out, double* out_sqrt)
{
    const int grid = xd_grid(n, num_sms());
    k_mgs_xdot<<<grid, XD_THREADS, 0, c.st>>>(n, w, vprev, hprev, y, c.xacc.p, c.xbad.p, c.xticket.p, out,
                                               out_sqrt);
    CK_LAUNCH();
    ++c.ndots;
}

// Column j of the Gram-Schmidt process of w (length n) against v_0 .. v_j,
// one launch; false where a row's worth of registers per SM does not hold w,
// where the blocks cannot be resident together (a GPU shared out by SMs), or
// after a launch that gave up waiting.  *err is set by one that does.
// Few elements a thread as long as blocks are left: a block's share of the
// integer work is ~0.25 us per element and thread, another block adds little
// to the barrier; up to 2048 elements one block has no barrier at all.
bool mgs_column(Ctx& c, long long n, const double* V, int j, const double* w, double* vnext, double* hcol,
                int* err)
{
    const long long per = XC_THREADS, sms = num_sms();
    int E = 1;
    long long grid = 1;
    if (n <= 4 * per) E = 4;
    else {
        while (E < XC_MAX_E && (n + per * E - 1) / (per * E) > sms) E *= 2;
        grid = (n + per * E - 1) / (per * E);
    }
    if (!c.columns || grid > sms || grid < 1) return false;
    auto launch = [&](auto kernel) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(unsigned(grid));
        cfg.blockDim = dim3(XC_THREADS);
        cfg.stream = c.st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = grid > 1 ? 1 : 0;
        return cudaLaunchKernelEx(&cfg, kernel, int(n), V, j, w, vnext, hcol, c.cdig.p, c.cphase, c.cbar.p, c.cbase,
                                  c.xbad.p, err, c.spin_limit);
    };
    const cudaError_t e = E == 1   ? launch(k_mgs_column<1>)
                          : E == 2 ? launch(k_mgs_column<2>)
                          : E == 4 ? launch(k_mgs_column<4>)
                                   : launch(k_mgs_column<8>);
    if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) {
        (void)cudaGetLastError();
        c.columns = false;
        return false;
    }
    CK(e);
    c.ndots += j + 2;
    if (grid > 1) {
        c.cbase += unsigned(grid) * unsigned(j + 2);
        c.cphase = (c.cphase + j + 2) % 3;
    }
    return true;
}

// Wall time of one setup phase, added to *acc: the stream is synchronised
// when the phase starts and when it ends, so the time covers the phase's
// kernels and its host work and nothing else.
struct PhaseTimer {
    cudaStream_t st;
    double* acc;
    std::chrono::steady_clock::time_point t0;
    PhaseTimer(cudaStream_t s, double* a) : st(s), acc(a)
    {
        CK(cudaStreamSynchronize(st));
        t0 = std::chrono::steady_clock::now();
    }
    ~PhaseTimer()
    {
        cudaStreamSynchronize(st);   // errors surface at the next checked call
        *acc += std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    }
};

// Builds CSR from per-row counts already in rp[0..n-1]; returns nnz.
int counts_to_rowptr(DBuf<int>& rp, int n, cudaStream_t st) { return exclusive_scan(rp.p, rp.p, n, st); }

void submatrix(const DevCSR& A, const int* rows, int nr, const int* colmap, int ncols, DevCSR& out,
               cudaStream_t st)
{
    out.n_rows = nr;
    out.n_cols = ncols;
    out.rp.alloc(size_t(nr) + 1);
    if (nr) k_sub_count<<<grid_for(nr, TB), TB, 0, st>>>(nr, rows, A.rp.p, A.ci.p, colmap, out.rp.p);
    CK_LAUNCH();
    out.nnz = counts_to_rowptr(out.rp, nr, st);
    out.ci.alloc(out.nnz);
    out.v.alloc(out.nnz);
    if (nr) k_sub_fill<<<grid_for(nr, TB), TB, 0, st>>>(nr, rows, A.rp.p, A.ci.p, A.v.p, colmap,
                                                          out.rp.p, out.ci.p, out.v.p);
    CK_LAUNCH();
}

// Rows [r0, r1) of C = A B as a piece of its own (packed).  prod, room: the
// rows' products and scratch entries.
struct GemmPiece {
    int r0 = 0, r1 = 0, nnz = 0;
    DBuf<int> rp, ci;
    DBuf<double> v;
};

void gemm_piece(const DevCSR& A, const DevCSR& B, const int* prod, const int* room, long long limit, GemmPiece& P,
                cudaStream_t st)
{
    const int mc = P.r1 - P.r0;
    DBuf<int> toff(size_t(mc) + 1);
    const int nroom = mc ? exclusive_scan(room, toff.p, mc, st) : 0;
    DBuf<int> tci(size_t(std::max(nroom, 1)));
    DBuf<double> tv(size_t(std::max(nroom, 1)));
    DBuf<int> lists(4 * size_t(std::max(mc, 1))), over(size_t(std::max(mc, 1))), counts(8), cnt(size_t(mc) + 1);
    CK(cudaMemsetAsync(counts.p, 0, counts.bytes(), st));
    if (mc) k_gemm_lists<<<grid_for(mc, TB), TB, 0, st>>>(mc, prod, lists.p, counts.p, cnt.p);
    CK_LAUNCH();
    int nc[4];
    d2h(nc, counts.p, 4, st);
    auto list = [&](int c) { return lists.p + size_t(c) * size_t(mc); };
    if (nc[0])
        k_gemm_lanes<GEMM_TINY><<<grid_for(nc[0], TB / GEMM_TINY), TB, 0, st>>>(
            nc[0], list(0), P.r0, A.rp.p, A.ci.p, A.v.p, B.rp.p, B.ci.p, B.v.p, toff.p, tci.p, tv.p, cnt.p);
    if (nc[1])
        k_gemm_lanes<GEMM_SMALL><<<grid_for(nc[1], TB / GEMM_SMALL), TB, 0, st>>>(
            nc[1], list(1), P.r0, A.rp.p, A.ci.p, A.v.p, B.rp.p, B.ci.p, B.v.p, toff.p, tci.p, tv.p, cnt.p);
    auto hash = [&](auto kernel, int slots, int c) {
        if (!nc[c]) return;
        CK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(gemm_smem(slots))));
        kernel<<<grid_for(nc[c], GEMM_WARPS), GEMM_WARPS * 32, gemm_smem(slots), st>>>(
            nc[c], list(c), P.r0, A.rp.p, A.ci.p, A.v.p, B.rp.p, B.ci.p, B.v.p, prod, toff.p, tci.p, tv.p, cnt.p,
            over.p, counts.p + 4);
    };
    hash(k_gemm_hash<GEMM_SLOTS_LOW>, GEMM_SLOTS_LOW, 2);
    hash(k_gemm_hash<GEMM_SLOTS>, GEMM_SLOTS, 3);
    CK_LAUNCH();
    // rows beyond the shared-memory tables, in runs whose tables hold at most
    // `limit` slots together (a row's own table may be larger); each run's
    // sorted rows wait in a piece of their own until the row pointers stand
    struct Run {
        int first = 0, n = 0;
        DBuf<int> rp, ci;
        DBuf<double> v;
    };
    std::vector<Run> runs;
    const int nover = nc[3] ? read1(counts.p + 4, st) : 0;
    if (nover) {
        DBuf<int> tsize(static_cast<size_t>(nover));
        k_gemm_table_size<<<grid_for(nover, TB), TB, 0, st>>>(nover, over.p, prod, B.n_cols, tsize.p);
        CK_LAUNCH();
        std::vector<int> ts(static_cast<size_t>(nover));
        d2h(ts.data(), tsize.p, size_t(nover), st);
        for (int t : ts)
            if (t < 0) fail(AIRG_ERR_OOM, "a row of a sparse product may have more than 2^29 columns");
        for (int t0 = 0; t0 < nover;) {
            Run R;
            R.first = t0;
            long long slots = 0;
            while (t0 < nover && (t0 == R.first || slots + ts[t0] <= limit)) slots += ts[t0++];
            R.n = t0 - R.first;
            const int* rows = over.p + R.first;
            DBuf<int> gtoff(size_t(R.n) + 1), keys;
            DBuf<double> vals;
            CK(cudaMemcpyAsync(gtoff.p, tsize.p + R.first, size_t(R.n) * sizeof(int), cudaMemcpyDeviceToDevice, st));
            const int total = exclusive_scan(gtoff.p, gtoff.p, R.n, st);
            keys.alloc(size_t(total));
            vals.alloc(size_t(total));
            CK(cudaMemsetAsync(keys.p, 0xff, keys.bytes(), st));
            R.rp.alloc(size_t(R.n) + 1);
            k_gemm_hash_global<<<grid_for(R.n, TB / 32), TB, 0, st>>>(R.n, rows, P.r0, A.rp.p, A.ci.p, A.v.p, B.rp.p,
                                                                     B.ci.p, B.v.p, gtoff.p, keys.p, vals.p, cnt.p,
                                                                     R.rp.p);
            CK_LAUNCH();
            const int n = exclusive_scan(R.rp.p, R.rp.p, R.n, st);
            R.ci.alloc(size_t(std::max(n, 1)));
            R.v.alloc(size_t(std::max(n, 1)));
            k_gemm_emit_global<<<R.n, TB, 0, st>>>(gtoff.p, keys.p, vals.p, R.rp.p, R.ci.p, R.v.p);
            CK_LAUNCH();
            CK(cudaStreamSynchronize(st));   // the tables are released
            runs.push_back(std::move(R));
        }
    }
    P.rp.alloc(size_t(mc) + 1);
    P.nnz = exclusive_scan(cnt.p, P.rp.p, mc, st);
    if (nover) {   // nothing of theirs is in the scratch piece
        k_gemm_mark<<<grid_for(nover, TB), TB, 0, st>>>(nover, over.p, cnt.p);
        CK_LAUNCH();
    }
    P.ci.alloc(std::max(P.nnz, 1));
    P.v.alloc(std::max(P.nnz, 1));
    if (mc)
        k_gemm_pack<<<grid_for(mc, TB), TB, 0, st>>>(mc, toff.p, P.rp.p, cnt.p, tci.p, tv.p, P.ci.p, P.v.p);
    for (const Run& R : runs)
        k_gemm_pack_list<<<grid_for(R.n, TB / 32), TB, 0, st>>>(R.n, over.p + R.first, R.rp.p, P.rp.p, R.ci.p, R.v.p,
                                                               P.ci.p, P.v.p);
    CK_LAUNCH();
    CK(cudaStreamSynchronize(st));   // the scratch is released on return
}

// C = A B.  Rows are processed in pieces whose scratch rows hold at most
// 2^28 entries (3 GiB) together, so large fill-heavy levels neither overflow
// the int32 offsets nor exhaust memory; the pieces are then joined.
void spgemm(const DevCSR& A, const DevCSR& B, DevCSR& C, cudaStream_t st)
{
    int m = A.n_rows;
    C.n_rows = m;
    C.n_cols = B.n_cols;
    static long long kLimit = 0;
    if (!kLimit) {
        const char* e = getenv("AIRG_SPGEMM_SLOTS");   // tuning / testing override
        kLimit = gemm_piece_limit(e ? atoll(e) : (1LL << 28));
    }
    DBuf<int> prod(size_t(std::max(m, 1))), room(size_t(std::max(m, 1)));
    DBuf<unsigned long long> sum(1);
    CK(cudaMemsetAsync(sum.p, 0, sizeof(unsigned long long), st));
    if (m) {
        k_gemm_bound<<<grid_for(m, TB), TB, 0, st>>>(m, A.rp.p, A.ci.p, B.rp.p, prod.p, room.p);
        k_sum_int<<<std::min(grid_for(m, TB), 1024), TB, 0, st>>>(m, room.p, sum.p);
    }
    CK_LAUNCH();
    std::vector<int> cut{0};
    if ((long long)read1(sum.p, st) > kLimit) {
        std::vector<int> rm(static_cast<size_t>(m));
        d2h(rm.data(), room.p, size_t(m), st);
        long long acc = 0;
        for (int i = 0; i < m; ++i) {
            if (acc + rm[i] > kLimit && i > cut.back()) { cut.push_back(i); acc = 0; }
            acc += rm[i];
        }
    }
    cut.push_back(m);
    std::vector<GemmPiece> pieces;
    long long total = 0;
    for (size_t c = 0; c + 1 < cut.size(); ++c) {
        GemmPiece P;
        P.r0 = cut[c];
        P.r1 = cut[c + 1];
        gemm_piece(A, B, prod.p + P.r0, room.p + P.r0, kLimit, P, st);
        total += P.nnz;
        pieces.push_back(std::move(P));
    }
    if (total > 0x7fffffffLL) fail(AIRG_ERR_OOM, "sparse product exceeds 2^31 entries");
    C.nnz = int(total);
    if (pieces.size() == 1) {
        C.rp = std::move(pieces[0].rp);
        C.ci = std::move(pieces[0].ci);
        C.v = std::move(pieces[0].v);
        return;
    }
    C.rp.alloc(size_t(m) + 1);
    C.ci.alloc(std::max(C.nnz, 1));
    C.v.alloc(std::max(C.nnz, 1));
    int off = 0;
    for (GemmPiece& P : pieces) {
        int mc = P.r1 - P.r0;
        if (mc) k_shift_rowptr<<<grid_for(mc, TB), TB, 0, st>>>(mc, P.rp.p, off, C.rp.p + P.r0);
        CK_LAUNCH();
        if (P.nnz) {
            CK(cudaMemcpyAsync(C.ci.p + off, P.ci.p, size_t(P.nnz) * sizeof(int), cudaMemcpyDeviceToDevice, st));
            CK(cudaMemcpyAsync(C.v.p + off, P.v.p, size_t(P.nnz) * sizeof(double), cudaMemcpyDeviceToDevice, st));
        }
        off += P.nnz;
    }
    CK(cudaMemcpyAsync(C.rp.p + m, &C.nnz, sizeof(int), cudaMemcpyHostToDevice, st));
    CK(cudaStreamSynchronize(st));
}

// Rows of more than 8 entries on average take the row kernels with a warp per
// row: with one thread per row the 32 rows of a warp are that far apart in
// memory.  Drop and lumping of the 4096^2 setup with its compaction: 55 ->
// 30 ms.
bool long_rows(const DevCSR& A) { return A.n_rows > 0 && A.nnz > 8LL * A.n_rows; }

void compact(const DevCSR& A, const int8_t* keep, DBuf<int>& cnt, DevCSR& out, cudaStream_t st)
{
    int n = A.n_rows;
    out.n_rows = n;
    out.n_cols = A.n_cols;
    out.rp = std::move(cnt);
    out.nnz = counts_to_rowptr(out.rp, n, st);
    out.ci.alloc(out.nnz);
    out.v.alloc(out.nnz);
    if (long_rows(A))
        k_compact_warp<<<grid_for(n, TB / 32), TB, 0, st>>>(n, A.rp.p, A.ci.p, A.v.p, keep, out.rp.p, out.ci.p,
                                                            out.v.p);
    else if (n)
        k_compact<<<grid_for(n, TB), TB, 0, st>>>(n, A.rp.p, A.ci.p, A.v.p, keep, out.rp.p, out.ci.p, out.v.p);
    CK_LAUNCH();
}

// Local indices of the rows with is_f == want: idx (n), ids (count); returns count
int local_index(const DBuf<int8_t>& is_f, int n, int want, DBuf<int>& idx, DBuf<int>& ids,
                cudaStream_t st)
{
    DBuf<int> ex(size_t(n) + 1);
    if (n) k_flag_eq<<<grid_for(n, TB), TB, 0, st>>>(n, is_f.p, want, ex.p);
    CK_LAUNCH();
    int cnt = exclusive_scan(ex.p, ex.p, n, st);
    idx.alloc(n);
    ids.alloc(std::max(cnt, 1));
    if (n) k_local_index<<<grid_for(n, TB), TB, 0, st>>>(n, is_f.p, want, ex.p, idx.p, ids.p);
    CK_LAUNCH();
    return cnt;
}

// ---------------------------------------------------------------- Arnoldi --
struct ArnoldiOut {
    std::vector<double> H;   // (k+1) x k row-major
    int k = 0;
    bool broke = false;
    double beta = 0.0;
};

// m steps of MGS Arnoldi from b (device, length n); dots correctly rounded.
ArnoldiOut arnoldi(Ctx& c, const DevCSR& A, const double* b, int m, double tol, double exact_tol)
{
    cudaStream_t st = c.st;
    long long n = A.n_rows;
    // H on the device by columns, each behind the word that its launch sets
    // when it gives up, so that one copy brings both to the host
    const size_t ld = size_t(m) + 2;
    DBuf<double> V(size_t(m + 1) * n), w(n), Hd(ld * m + 1);
    CK(cudaMemsetAsync(Hd.p, 0, Hd.bytes(), st));
    double* beta_d = Hd.p + ld * m;
    xdot(c, n, b, b, nullptr, beta_d);
    int g = grid_for(n, TB);
    k_div_dev<<<g, TB, 0, st>>>(n, V.p, b, beta_d);
    CK_LAUNCH();
    std::vector<double> Hh(size_t(m + 1) * m, 0.0);
    const double beta_h = read1(beta_d, st);
    ArnoldiOut out;
    out.k = m;
    c.hcol.alloc(ld);
    const double* col = c.hcol.p + 1;
    for (int j = 0; j < m; ++j) {
        k_spmv_det<<<grid_for(n, TB), TB, 0, st>>>(int(n), A.rp.p, A.ci.p, A.v.p, V.p + size_t(j) * n, w.p);
        CK_LAUNCH();
        // h_ij = <w, v_i> then w -= h_ij v_i, for i = 0..j (modified
        // Gram-Schmidt), and v_{j+1} = w / ||w||: in one launch where w fits
        // in registers, else, or where that launch gave up, one per dot (each
        // update fused with the next)
        double* hj = Hd.p + ld * j + 1;
        double* hn = hj + j + 1;
        auto dots = [&] {
            for (int i = 0; i <= j; ++i)
                mgs_xdot(c, n, w.p, i ? V.p + size_t(i - 1) * n : nullptr, i ? hj + i - 1 : nullptr,
                         V.p + size_t(i) * n, hj + i, nullptr);
            mgs_xdot(c, n, w.p, V.p + size_t(j) * n, hj + j, nullptr, nullptr, hn);
        };
        bool column = mgs_column(c, n, V.p, j, w.p, V.p + size_t(j + 1) * n, hj, reinterpret_cast<int*>(hj - 1));
        if (!column) dots();
        d2h(c.hcol.p, hj - 1, size_t(j) + 3, st);
        if (*reinterpret_cast<const int*>(c.hcol.p)) {
            c.columns = column = false;
            dots();
            d2h(c.hcol.p + 1, hj, size_t(j) + 2, st);
        }
        for (int i = 0; i <= j + 1; ++i) Hh[size_t(i) * m + j] = col[i];
        double s = 0.0;
        for (int i = 0; i <= j + 1; ++i) s = s + col[i] * col[i];
        if (col[j + 1] <= tol * std::sqrt(s)) {
            out.k = j + 1;
            out.broke = true;
            break;
        }
        {
            // GMRES residual of the (j+2) x (j+1) least-squares problem
            int kk = j + 1;
            std::vector<double> Hs(size_t(kk + 1) * kk);
            for (int i = 0; i <= kk; ++i)
                for (int q = 0; q < kk; ++q) Hs[size_t(i) * kk + q] = Hh[size_t(i) * m + q];
            if (givens_residual(Hs, kk, beta_h) <= exact_tol * beta_h) {
                out.k = kk;
                break;
            }
        }
        if (j + 1 < m && !column) {
            k_div_dev<<<g, TB, 0, st>>>(n, V.p + size_t(j + 1) * n, w.p, hn);
            CK_LAUNCH();
        }
    }
    out.beta = beta_h;
    int k = out.k;
    out.H.assign(size_t(k + 1) * k, 0.0);
    for (int i = 0; i <= k; ++i)
        for (int j = 0; j < k; ++j) out.H[size_t(i) * k + j] = Hh[size_t(i) * m + j];
    return out;
}

std::vector<double> gmres_poly_coeffs(Ctx& c, const DevCSR& Aff, const airg_options& o, int level,
                                      int& kout, int purpose = PURPOSE_COEF)
{
    int p = o.poly_order;
    long long n = Aff.n_rows;
    DBuf<double> b(n);
    k_rng_uniform<<<grid_for(n, TB), TB, 0, c.st>>>(stream_key(o.seed, level, purpose), n, b.p);
    CK_LAUNCH();
    ArnoldiOut ar = arnoldi(c, Aff, b.p, p + 1, o.breakdown_tol, o.exact_tol);
    std::vector<double> y = givens_lsq(ar.H, ar.k, ar.beta);
    std::vector<double> alpha = power_coefficients(ar.H, ar.k, ar.beta, y);
    alpha.resize(size_t(p) + 1, 0.0);
    kout = ar.k;
    return alpha;
}

// max_i |a_ii| as the bit pattern of a non-negative double (such patterns
// order like the values), so the atomic maximum is exact and order-free
__global__ void k_diag_absmax(int n, const int* rp, const int* ci, const double* v, unsigned long long* out)
{
    int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    for (int k = rp[r]; k < rp[r + 1]; ++k)
        if (ci[k] == r) {
            atomicMax(out, (unsigned long long)__double_as_longlong(fabs(v[k])));
            break;
        }
}

// nAIR (Sec. 3.3.1): power-basis coefficients of w sum_{k<=p} (I - w A)^k,
// w = 1 / max |a_ii|, i.e. alpha_j = w (-w)^j C(p+1, j+1), with (-w)^j formed
// by repeated products
std::vector<double> neumann_coeffs(const DevCSR& A, const airg_options& o, cudaStream_t st)
{
    const int p = o.poly_order;
    double dmax = 1.0;
    if (A.n_rows) {
        DBuf<unsigned long long> m(1);
        CK(cudaMemsetAsync(m.p, 0, sizeof(unsigned long long), st));
        k_diag_absmax<<<grid_for(A.n_rows, TB), TB, 0, st>>>(A.n_rows, A.rp.p, A.ci.p, A.v.p, m.p);
        CK_LAUNCH();
        unsigned long long bits = 0;
        d2h(&bits, m.p, 1, st);
        std::memcpy(&dmax, &bits, sizeof dmax);
        if (!(dmax > 0.0)) fail(AIRG_ERR_BREAKDOWN, "block without a nonzero diagonal (Neumann polynomial)");
    }
    const double w = 1.0 / dmax;
    // binomial C(p+1, j+1) from Pascal's triangle (exact in 64 bits for p <= 30)
    std::vector<unsigned long long> row(size_t(p) + 2, 0);
    row[0] = 1;
    for (int i = 1; i <= p + 1; ++i)
        for (int j = i; j >= 1; --j) row[j] += row[j - 1];
    std::vector<double> alpha(size_t(p) + 1);
    double pw = 1.0;
    for (int j = 0; j <= p; ++j) {
        alpha[j] = (w * pw) * (double)row[j + 1];
        pw = pw * -w;
    }
    return alpha;
}

std::vector<double> smoother_coeffs(Ctx& c, const DevCSR& A, const airg_options& o, int level, int& kout,
                                    int purpose)
{
    if (o.inverse_type == AIRG_INVERSE_NEUMANN) {
        kout = o.poly_order + 1;
        return neumann_coeffs(A, o, c.st);
    }
    return gmres_poly_coeffs(c, A, o, level, kout, purpose);
}

void fixed_sparsity_inverse(const DevCSR& Aff, const std::vector<double>& alpha, DevCSR& out,
                            cudaStream_t st)
{
    int n = Aff.n_rows, nnz = Aff.nnz;
    out.alloc(n, n, nnz);
    CK(cudaMemcpyAsync(out.rp.p, Aff.rp.p, (n + 1) * sizeof(int), cudaMemcpyDeviceToDevice, st));
    CK(cudaMemcpyAsync(out.ci.p, Aff.ci.p, nnz * sizeof(int), cudaMemcpyDeviceToDevice, st));
    if (!n) return;
    k_fsp_init<<<grid_for(n, TB), TB, 0, st>>>(n, Aff.rp.p, Aff.ci.p, alpha[0], out.v.p);
    DBuf<double> T(nnz), Tn(nnz);
    CK(cudaMemcpyAsync(T.p, Aff.v.p, nnz * sizeof(double), cudaMemcpyDeviceToDevice, st));
    for (size_t k = 1; k < alpha.size(); ++k) {
        if (k >= 2) {
            k_fsp_power<<<grid_for(n, TB), TB, 0, st>>>(n, Aff.rp.p, Aff.ci.p, Aff.v.p, T.p, Tn.p);
            k_fsp_power_warp<<<grid_for(n, TB / 32), TB, 0, st>>>(n, Aff.rp.p, Aff.ci.p, Aff.v.p, T.p, Tn.p);
            std::swap(T.p, Tn.p);
        }
        k_fsp_acc<<<grid_for(nnz, TB), TB, 0, st>>>(nnz, out.v.p, T.p, alpha[k]);
        CK_LAUNCH();
    }
    CK(cudaStreamSynchronize(st));
}

// Newton application x = q(A) b (Sec. 2.3), deterministic kernels.
void newton_apply(Ctx& c, const DevCSR& A, const std::vector<Root>& roots, const double* b,
                  double* x)
{
    cudaStream_t st = c.st;
    long long n = A.n_rows;
    DBuf<double> r(n), w(n), t(n);
    CK(cudaMemsetAsync(x, 0, n * sizeof(double), st));
    CK(cudaMemcpyAsync(r.p, b, n * sizeof(double), cudaMemcpyDeviceToDevice, st));
    int g = grid_for(n, TB);
    for (size_t idx = 0; idx < roots.size(); ++idx) {
        bool last = idx + 1 == roots.size();
        double a = roots[idx].re, bi = roots[idx].im;
        if (bi == 0.0) {
            k_newton_real_x<<<g, TB, 0, st>>>(n, x, r.p, a);
            if (!last) {
                k_spmv_det<<<g, TB, 0, st>>>(int(n), A.rp.p, A.ci.p, A.v.p, r.p, w.p);
                k_newton_r<<<g, TB, 0, st>>>(n, r.p, w.p, a);
            }
        } else {
            double mod2 = a * a + bi * bi;
            k_spmv_det<<<g, TB, 0, st>>>(int(n), A.rp.p, A.ci.p, A.v.p, r.p, w.p);
            k_newton_pair<<<g, TB, 0, st>>>(n, x, r.p, w.p, t.p, 2.0 * a, mod2);
            if (!last) {
                k_spmv_det<<<g, TB, 0, st>>>(int(n), A.rp.p, A.ci.p, A.v.p, t.p, w.p);
                k_newton_r<<<g, TB, 0, st>>>(n, r.p, w.p, mod2);
            }
        }
        CK_LAUNCH();
    }
    CK(cudaStreamSynchronize(st));
}

std::vector<Root> coarse_polynomial(Ctx& c, const DevCSR& A, const airg_options& o, int level,
                                    int m, int& kout)
{
    long long n = A.n_rows;
    DBuf<double> b(n);
    k_rng_uniform<<<grid_for(n, TB), TB, 0, c.st>>>(stream_key(o.seed, level, PURPOSE_COARSE), n, b.p);
    CK_LAUNCH();
    ArnoldiOut ar = arnoldi(c, A, b.p, m, o.breakdown_tol, o.exact_tol);
    std::vector<double> wr, wi;
    if (!harmonic_ritz(ar.H, ar.k, ar.broke, wr, wi))
        fail(AIRG_ERR_BREAKDOWN, "harmonic Ritz eigenvalue iteration did not converge");
    kout = ar.k;
    return order_roots(wr, wi, o.addroot_log10, o.addroot_per);
}

double truncation_residual(Ctx& c, const DevCSR& A, const std::vector<Root>& roots,
                           const airg_options& o, int level)
{
    cudaStream_t st = c.st;
    long long n = A.n_rows;
    DBuf<double> b2(n), x(n), y(n), r(n), nrm(2);
    k_rng_uniform<<<grid_for(n, TB), TB, 0, st>>>(stream_key(o.seed, level, PURPOSE_TRUNC), n, b2.p);
    CK_LAUNCH();
    newton_apply(c, A, roots, b2.p, x.p);
    k_spmv_det<<<grid_for(n, TB), TB, 0, st>>>(int(n), A.rp.p, A.ci.p, A.v.p, x.p, y.p);
    k_sub<<<grid_for(n, TB), TB, 0, st>>>(n, b2.p, y.p, r.p);
    CK_LAUNCH();
    xdot(c, n, r.p, r.p, nullptr, nrm.p);
    xdot(c, n, b2.p, b2.p, nullptr, nrm.p + 1);
    double h[2];
    d2h(h, nrm.p, 2, st);
    return h[0] / h[1];
}

// ------------------------------------------------------------- CF split --
void cf_split(Ctx& c, SetupLevel& L, const airg_options& o, int level)
{
    cudaStream_t st = c.st;
    const DevCSR& A = L.A;
    int n = A.n_rows;
    int g = grid_for(n, TB);
    L.strong.alloc(std::max(A.nnz, 1));
    k_strength<<<g, TB, 0, st>>>(n, A.rp.p, A.ci.p, A.v.p, o.strong_threshold, L.strong.p);
    // S^T
    DBuf<int> rpt(size_t(n) + 1), cursor(n);
    CK(cudaMemsetAsync(rpt.p, 0, rpt.bytes(), st));
    CK(cudaMemsetAsync(cursor.p, 0, cursor.bytes(), st));
    k_count_strong_t<<<g, TB, 0, st>>>(n, A.rp.p, A.ci.p, L.strong.p, rpt.p);
    CK_LAUNCH();
    int nst = exclusive_scan(rpt.p, rpt.p, n, st);
    DBuf<int> ct(std::max(nst, 1));
    k_fill_strong_t<<<g, TB, 0, st>>>(n, A.rp.p, A.ci.p, L.strong.p, rpt.p, cursor.p, ct.p);
    k_sort_rows<<<g, TB, 0, st>>>(n, rpt.p, ct.p);
    CK_LAUNCH();
    // G = S + S^T
    DBuf<int> rpg(size_t(n) + 1);
    k_union<<<g, TB, 0, st>>>(n, A.rp.p, A.ci.p, L.strong.p, rpt.p, ct.p, nullptr, nullptr, rpg.p);
    CK_LAUNCH();
    int ng = exclusive_scan(rpg.p, rpg.p, n, st);
    DBuf<int> cg(std::max(ng, 1));
    k_union<<<g, TB, 0, st>>>(n, A.rp.p, A.ci.p, L.strong.p, rpt.p, ct.p, rpg.p, cg.p, nullptr);
    CK_LAUNCH();
    // PMISR rounds
    DBuf<unsigned> w(n);
    DBuf<int8_t> state(n), newf(n);
    DBuf<int> und(1);
    k_rng_u32<<<g, TB, 0, st>>>(stream_key(o.seed, level, PURPOSE_PMISR), n, w.p);
    CK(cudaMemsetAsync(state.p, 0, state.bytes(), st));
    int rounds = 0;
    while (true) {
        ++rounds;
        CK(cudaMemsetAsync(und.p, 0, sizeof(int), st));
        k_pmisr_select<<<g, TB, 0, st>>>(n, rpg.p, cg.p, w.p, state.p, newf.p);
        k_pmisr_update<<<g, TB, 0, st>>>(n, rpg.p, cg.p, state.p, newf.p, und.p);
        CK_LAUNCH();
        if (read1(und.p, st) == 0) break;
        if (rounds > n + 1) fail(AIRG_ERR_STATE, "PMISR made no progress");
    }
    L.pmisr_rounds = rounds;
    L.is_f.alloc(n);
    k_state_to_f<<<g, TB, 0, st>>>(n, state.p, L.is_f.p);
    CK_LAUNCH();
    // DDC passes (Sec. 2.1): 1000 equal bins over [0, max ratio]
    const int nbins = 1000;
    DBuf<double> ratio(n);
    DBuf<int> bins(n), hist(nbins), cnt(size_t(n) + 1);
    DBuf<unsigned long long> rmax(1);
    L.ddc_converted.clear();
    for (int it = 0; it < o.ddc_its; ++it) {
        k_flag_eq<<<g, TB, 0, st>>>(n, L.is_f.p, 1, cnt.p);
        CK_LAUNCH();
        int n_f = exclusive_scan(cnt.p, cnt.p, n, st);
        if (n_f == 0) { L.ddc_converted.push_back(0); continue; }
        CK(cudaMemsetAsync(rmax.p, 0, sizeof(unsigned long long), st));
        k_ddc_ratio<<<g, TB, 0, st>>>(n, A.rp.p, A.ci.p, A.v.p, L.is_f.p, ratio.p, rmax.p);
        CK_LAUNCH();
        unsigned long long rb = read1(rmax.p, st);
        double rm;
        std::memcpy(&rm, &rb, sizeof rm);
        if (!(rm > 0.0)) { L.ddc_converted.push_back(0); continue; }
        if (std::isinf(rm)) fail(AIRG_ERR_BREAKDOWN, "zero diagonal in an F row");
        long long k = (long long)std::ceil(o.ddc_fraction * double(n_f));
        CK(cudaMemsetAsync(hist.p, 0, hist.bytes(), st));
        k_ddc_bin<<<g, TB, 0, st>>>(n, L.is_f.p, ratio.p, rm, nbins, bins.p, hist.p);
        CK_LAUNCH();
        std::vector<int> hh(nbins);
        d2h(hh.data(), hist.p, nbins, st);
        // boundary B whose count at or above it is closest to k (ties: higher B)
        long long above = 0;
        int best_b = nbins;
        long long best_d = k;   // |0 - k|
        std::vector<long long> ab(nbins + 1, 0);
        for (int b = nbins - 1; b >= 0; --b) { above += hh[b]; ab[b] = above; }
        for (int b = nbins - 1; b >= 0; --b) {
            long long d = std::llabs(ab[b] - k);
            if (d < best_d) { best_d = d; best_b = b; }
        }
        L.ddc_converted.push_back(int(best_b < nbins ? ab[best_b] : 0));
        if (best_b < nbins) {
            k_ddc_convert<<<g, TB, 0, st>>>(n, L.is_f.p, bins.p, best_b);
            CK_LAUNCH();
        }
    }
}

}  // namespace

// ===========================================================================
// Runs the bounded wait of k_mgs_column for an arrival that never comes;
// true if it gave up, as designed.
bool column_timeout_check(long long limit, cudaStream_t st)
{
    DBuf<unsigned> state(2);
    CK(cudaMemsetAsync(state.p, 0, state.bytes(), st));
    k_column_timeout_check<<<1, 32, 0, st>>>(state.p, limit);
    CK_LAUNCH();
    return read1(state.p + 1, st) != 0;
}

void dot_exact_device(long long n, const double* x, const double* y, double* out,
                      double* out_sqrt, cudaStream_t st)
{
    Ctx c(st);
    xdot(c, n, x, y, out, out_sqrt);
    CK(cudaStreamSynchronize(st));
}

void rng_uniform_device(uint64_t seed, long long level, long long purpose, long long n,
                        double* out, cudaStream_t st)
{
    if (n <= 0) return;
    k_rng_uniform<<<grid_for(n, TB), TB, 0, st>>>(stream_key(seed, level, purpose), n, out);
    CK_LAUNCH();
    CK(cudaStreamSynchronize(st));
}

void validate_csr(const DevCSR& A, bool square, cudaStream_t st)
{
    DBuf<int> flags(4);
    CK(cudaMemsetAsync(flags.p, 0, flags.bytes(), st));
    if (A.n_rows)
        k_validate<<<grid_for(A.n_rows, TB), TB, 0, st>>>(A.n_rows, A.n_cols, A.nnz, A.rp.p, A.ci.p, A.v.p,
                                                            square ? 1 : 0, flags.p);
    CK_LAUNCH();
    int f[4];
    d2h(f, flags.p, 4, st);
    if (f[2]) fail(AIRG_ERR_ARG, "row pointers not monotone within [0, nnz] with rowptr[0] = 0, rowptr[n] = nnz");
    if (f[0]) fail(AIRG_ERR_ARG, "CSR columns out of range or not strictly ascending");
    if (f[1]) fail(AIRG_ERR_ARG, "a row has no stored diagonal");
    if (f[3]) fail(AIRG_ERR_ARG, "a matrix value is not finite");
}

void csr_transpose(const DevCSR& A, DevCSR& T, cudaStream_t st)
{
    int n = A.n_rows, m = A.n_cols;
    T.n_rows = m;
    T.n_cols = n;
    T.nnz = A.nnz;
    T.rp.alloc(size_t(m) + 1);
    DBuf<int> cursor(std::max(m, 1));
    CK(cudaMemsetAsync(T.rp.p, 0, T.rp.bytes(), st));
    CK(cudaMemsetAsync(cursor.p, 0, cursor.bytes(), st));
    if (n) k_count_cols<<<grid_for(n, TB), TB, 0, st>>>(n, A.rp.p, A.ci.p, T.rp.p);
    CK_LAUNCH();
    exclusive_scan(T.rp.p, T.rp.p, m, st);
    T.ci.alloc(A.nnz);
    T.v.alloc(A.nnz);
    if (n) k_fill_transpose<<<grid_for(n, TB), TB, 0, st>>>(n, A.rp.p, A.ci.p, A.v.p, T.rp.p,
                                                              cursor.p, T.ci.p, T.v.p);
    if (m) k_sort_rows_kv<<<grid_for(m, TB), TB, 0, st>>>(m, T.rp.p, T.ci.p, T.v.p);
    CK_LAUNCH();
    CK(cudaStreamSynchronize(st));
}

std::unique_ptr<Hierarchy> build_hierarchy(DevCSR&& A0, const airg_options& o, cudaStream_t st)
{
    auto t0 = std::chrono::steady_clock::now();
    auto H = std::make_unique<Hierarchy>();
    H->opt = o;
    Ctx c(st);
    DevCSR A = std::move(A0);
    int level = 0;
    while (true) {
        int n = A.n_rows;
        bool last = level >= o.max_levels - 1 || n <= o.coarse_min_rows;
        int m_c = std::min(o.coarse_poly_order, n);
        double trunc_rel = NAN;
        const double trunc_before = H->phase_ms[AIRG_PHASE_TRUNCATION];
        if (!last && o.trunc_rtol > 0.0 && level >= o.trunc_start_level) {
            int k = 0;
            std::vector<Root> roots;
            {
                PhaseTimer pt(st, &H->phase_ms[AIRG_PHASE_TRUNCATION]);
                roots = coarse_polynomial(c, A, o, level, m_c, k);
                trunc_rel = truncation_residual(c, A, roots, o, level);
            }
            if (trunc_rel <= o.trunc_rtol) {
                // the test's polynomial becomes the coarse solver
                H->phase_ms[AIRG_PHASE_COARSE_POLY] += H->phase_ms[AIRG_PHASE_TRUNCATION] - trunc_before;
                H->phase_ms[AIRG_PHASE_TRUNCATION] = trunc_before;
                H->coarse.A = std::move(A);
                H->coarse.roots = std::move(roots);
                H->coarse.k = k;
                H->coarse.trunc_rel = trunc_rel;
                H->coarse.truncated = true;
                break;
            }
        }
        auto L = std::make_unique<SetupLevel>();
        L->n = n;
        L->A = std::move(A);
        if (!last) {
            PhaseTimer pt(st, &H->phase_ms[AIRG_PHASE_CF_SPLIT]);
            cf_split(c, *L, o, level);
            L->n_f = local_index(L->is_f, n, 1, L->f_index, L->f_ids, st);
            L->n_c = n - L->n_f;
            if (L->n_f == 0 || L->n_f == n) last = true;
        }
        if (last) {
            PhaseTimer pt(st, &H->phase_ms[AIRG_PHASE_COARSE_POLY]);
            int k = 0;
            H->coarse.roots = coarse_polynomial(c, L->A, o, level, m_c, k);
            H->coarse.k = k;
            H->coarse.trunc_rel = trunc_rel;
            H->coarse.A = std::move(L->A);
            break;
        }
        L->trunc_rel = trunc_rel;
        const DevCSR& Al = L->A;
        DevCSR A_cf;
        {
            PhaseTimer pt(st, &H->phase_ms[AIRG_PHASE_EXTRACT]);
            local_index(L->is_f, n, 0, L->c_index, L->c_ids, st);
            // blocks of Eq. 3
            submatrix(Al, L->f_ids.p, L->n_f, L->f_index.p, L->n_f, L->A_ff, st);
            submatrix(Al, L->f_ids.p, L->n_f, L->c_index.p, L->n_c, L->A_fc, st);
            submatrix(Al, L->c_ids.p, L->n_c, L->f_index.p, L->n_f, A_cf, st);
        }
        // GMRES polynomial (Eq. 7) and fixed-sparsity inverse (Eq. 8)
        {
            PhaseTimer pt(st, &H->phase_ms[AIRG_PHASE_SMOOTHER_POLY]);
            L->alpha = smoother_coeffs(c, L->A_ff, o, level, L->alpha_k, PURPOSE_COEF);
        }
        DevCSR Ainv;
        {
            PhaseTimer pt(st, &H->phase_ms[AIRG_PHASE_FIXED_SPARSITY]);
            fixed_sparsity_inverse(L->A_ff, L->alpha, Ainv, st);
        }
        // Z = -A_cf Ahat^-1, then the relative drop on R
        DevCSR Zfull;
        {
            PhaseTimer pt(st, &H->phase_ms[AIRG_PHASE_RESTRICTOR]);
            spgemm(A_cf, Ainv, Zfull, st);
        }
        if (o.smoother == AIRG_SMOOTH_ASSEMBLED) L->Ainv = std::move(Ainv);
        if (o.smooth_type != AIRG_SMOOTH_F) {
            // C-point smoothing (Sec. 2): the GMRES polynomial of A_cc from
            // its own random stream, and the row blocks its residuals use
            {
                PhaseTimer pt(st, &H->phase_ms[AIRG_PHASE_EXTRACT]);
                submatrix(Al, L->c_ids.p, L->n_c, L->c_index.p, L->n_c, L->A_cc, st);
                submatrix(Al, L->c_ids.p, L->n_c, nullptr, n, L->Crows, st);
                if (o.smooth_type == AIRG_SMOOTH_FCF) submatrix(Al, L->f_ids.p, L->n_f, nullptr, n, L->Frows, st);
            }
            {
                PhaseTimer pt(st, &H->phase_ms[AIRG_PHASE_SMOOTHER_POLY]);
                L->alpha_c = smoother_coeffs(c, L->A_cc, o, level, L->alpha_c_k, PURPOSE_COEF_C);
            }
            PhaseTimer pt(st, &H->phase_ms[AIRG_PHASE_FIXED_SPARSITY]);
            if (o.smoother == AIRG_SMOOTH_ASSEMBLED) fixed_sparsity_inverse(L->A_cc, L->alpha_c, L->Ainv_cc, st);
        }
        {
            PhaseTimer pt(st, &H->phase_ms[AIRG_PHASE_RESTRICTOR]);
            if (Zfull.nnz) k_scale<<<grid_for(Zfull.nnz, TB), TB, 0, st>>>(Zfull.nnz, Zfull.v.p, -1.0);
            DBuf<int8_t> keep(std::max(Zfull.nnz, 1));
            DBuf<int> cnt(size_t(L->n_c) + 1);
            if (long_rows(Zfull))
                k_drop_rows_warp<<<grid_for(L->n_c, TB / 32), TB, 0, st>>>(L->n_c, Zfull.rp.p, Zfull.v.p, o.r_drop,
                                                                           keep.p, cnt.p);
            else if (L->n_c)
                k_drop_rows<<<grid_for(L->n_c, TB), TB, 0, st>>>(L->n_c, Zfull.rp.p, Zfull.v.p, o.r_drop, keep.p,
                                                                 cnt.p);
            CK_LAUNCH();
            compact(Zfull, keep.p, cnt, L->Z, st);
        }
        // one-point prolongator
        std::unique_ptr<PhaseTimer> pt_p = std::make_unique<PhaseTimer>(st, &H->phase_ms[AIRG_PHASE_PROLONGATOR]);
        L->W.alloc(std::max(L->n_f, 1));
        k_one_point<<<grid_for(n, TB), TB, 0, st>>>(n, Al.rp.p, Al.ci.p, Al.v.p, L->strong.p,
                                                    L->is_f.p, L->c_index.p, L->f_index.p, L->W.p);
        CK_LAUNCH();
        // P = [W; I] and R = [Z I] in the fine numbering
        DevCSR P, R, AP, Ac;
        P.n_rows = n;
        P.n_cols = L->n_c;
        P.rp.alloc(size_t(n) + 1);
        k_p_count<<<grid_for(n, TB), TB, 0, st>>>(n, L->is_f.p, L->f_index.p, L->W.p, P.rp.p);
        CK_LAUNCH();
        P.nnz = counts_to_rowptr(P.rp, n, st);
        P.ci.alloc(P.nnz);
        P.v.alloc(P.nnz);
        k_p_fill<<<grid_for(n, TB), TB, 0, st>>>(n, L->is_f.p, L->f_index.p, L->c_index.p, L->W.p,
                                                 P.rp.p, P.ci.p, P.v.p);
        CK_LAUNCH();
        R.n_rows = L->n_c;
        R.n_cols = n;
        R.nnz = L->Z.nnz + L->n_c;
        R.rp.alloc(size_t(L->n_c) + 1);
        R.ci.alloc(R.nnz);
        R.v.alloc(R.nnz);
        k_r_rowptr<<<grid_for(L->n_c + 1, TB), TB, 0, st>>>(L->n_c, L->Z.rp.p, R.rp.p);
        k_r_fill<<<grid_for(L->n_c, TB), TB, 0, st>>>(L->n_c, L->Z.rp.p, L->Z.ci.p, L->Z.v.p,
                                                      L->f_ids.p, L->c_ids.p, R.rp.p, R.ci.p, R.v.p);
        CK_LAUNCH();
        pt_p.reset();
        // A_coarse = R (A P), then drop + lump
        {
            PhaseTimer pt(st, &H->phase_ms[AIRG_PHASE_RAP]);
            spgemm(Al, P, AP, st);
            spgemm(R, AP, Ac, st);
            // rows of AP at the F points: A_fc + A_ff W (the solve's residual operator)
            submatrix(AP, L->f_ids.p, L->n_f, nullptr, L->n_c, L->M, st);
        }
        {
            PhaseTimer pt(st, &H->phase_ms[AIRG_PHASE_DROP_LUMP]);
            int nc = Ac.n_rows;
            DBuf<int8_t> keep(std::max(Ac.nnz, 1));
            DBuf<double> vout(std::max(Ac.nnz, 1));
            DBuf<int> cnt(size_t(nc) + 1), bad(1);
            CK(cudaMemsetAsync(bad.p, 0, sizeof(int), st));
            if (long_rows(Ac))
                k_drop_lump_warp<<<grid_for(nc, TB / 32), TB, 0, st>>>(nc, Ac.rp.p, Ac.ci.p, Ac.v.p, o.a_drop, o.a_lump,
                                                                       keep.p, vout.p, cnt.p, bad.p);
            else if (nc)
                k_drop_lump<<<grid_for(nc, TB), TB, 0, st>>>(nc, Ac.rp.p, Ac.ci.p, Ac.v.p, o.a_drop, o.a_lump, keep.p,
                                                             vout.p, cnt.p, bad.p);
            CK_LAUNCH();
            if (read1(bad.p, st)) fail(AIRG_ERR_BREAKDOWN, "coarse row without a diagonal");
            std::swap(Ac.v.p, vout.p);
            DevCSR Acd;
            compact(Ac, keep.p, cnt, Acd, st);
            A = std::move(Acd);
        }
        CK(cudaStreamSynchronize(st));
        H->levels.push_back(std::move(L));
        ++level;
    }
    {
        PhaseTimer pt(st, &H->phase_ms[AIRG_PHASE_SOLVE_LAYOUT]);
        build_solve_data(*H, st);
    }
    H->exact_dots = c.ndots;
    CK(cudaStreamSynchronize(st));
    H->setup_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    return H;
}

}  // namespace airg
