// Correctly rounded dot product on the GPU.
//
// <x, y> is defined as the exact sum of the exact products x_i * y_i,
// rounded once to the nearest double (ties to even).  That value does not
// depend on the order of summation, so it is the same however the grid is
// shaped and equals any other correct implementation bit for bit; the setup
// uses it for every Arnoldi inner product and norm (Sec. 2.2-2.4) so that
// the polynomial coefficients, and from them every sparsity decision of the
// hierarchy, are reproducible.
//
// A finite double is m * 2^e with an integer m < 2^53 and e >= -1074, so the
// product of two is an integer below 2^106 (a 128-bit integer product) times
// 2^(ex+ey), ex+ey >= -2148.  The accumulator is a signed fixed-point integer
// with least significant bit 2^-2148 stored as 140 digits of 32 bits, each
// digit held in a 64-bit word so that many deposits can wait for one carry
// pass.  Threads add their products into a 192-bit register window, warps
// reduce the windows into their shared-memory accumulators, blocks add
// theirs into a global accumulator (two's-complement wrap-around makes signed
// addition exact), and the last block propagates carries and rounds.
//
// What bounds it: at 16.8M elements the integer work per product (split,
// 53 x 53 bits, shift, 192-bit add: ~60 instructions) beside 16-24 bytes of
// memory traffic; at a few thousand elements the serial tail (launch, block
// reduction, rounding).  Against the form it replaces (one element in flight
// per thread, a shared-memory atomic per lane and digit at the end, a
// single-thread walk over all 140 digits): the 2,100 dots of a 97 x 80 setup
// with their SpMVs and host reads 64 -> 23 ms, the truncation tests of the
// 4096^2 setup 789 -> 469 ms.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "exact_dot_limits.h"

namespace airg {

constexpr int XD_DIGITS = 140;   // 140 * 32 = 4480 bits >= 2148 + 2046 + 2
constexpr int XD_BIAS = 2148;    // digit-bit position of 2^0
constexpr int XD_WARPS = 8;      // warps (shared accumulators) per block
constexpr int XD_UNROLL = 4;     // elements whose loads a thread has in flight at once
constexpr int XD_THREADS = XD_WARPS * 32;

__device__ __forceinline__ bool xd_split(double x, unsigned long long& m, int& e, int& neg)
{
    unsigned long long b = (unsigned long long)__double_as_longlong(x);
    neg = int(b >> 63);
    int ex = int((b >> 52) & 0x7ffULL);
    unsigned long long fr = b & ((1ULL << 52) - 1ULL);
    if (ex == 0) { m = fr; e = -1074; }
    else { m = fr | (1ULL << 52); e = ex - 1075; }
    return m != 0ULL;
}

// A thread's register window: a 192-bit two's-complement sum whose least
// significant word stands at digit d0 of the accumulator.  A product at bit
// position pos covers the five words from digit d = pos >> 5 on; products of
// similar magnitude share d, so most of them are added here with one carry
// chain and only a move of the window (or the end of the thread's loop)
// deposits it.  The sums are exact integer sums, so the result does not
// depend on when they are deposited.  Headroom: a product at digit d0 + 1 is
// below 2^169, so 2^20 products fit between deposits; a thread of any launch
// here takes fewer than 2^15 (n < 2^31 over at least 2^16 threads, or a
// small n).
struct XdWin {
    unsigned w[6];
    int d0;
};

__device__ __forceinline__ void xd_win_init(XdWin& a)
{
#pragma unroll
    for (int k = 0; k < 6; ++k) a.w[k] = 0u;
    a.d0 = -8;
}

// Deposit of one thread's window from inside the loop (rare, divergent):
// words unsigned, the sign as -1 at digit d0 + 6.
__device__ __forceinline__ void xd_win_deposit(unsigned long long* acc, const XdWin& a)
{
    if (a.d0 < 0) return;
#pragma unroll
    for (int k = 0; k < 6; ++k)
        if (a.w[k]) atomicAdd(acc + a.d0 + k, (unsigned long long)a.w[k]);
    if (a.w[5] >> 31) atomicAdd(acc + a.d0 + 6, ~0ULL);
}

// Deposit of a whole warp's windows into its own accumulator at the end of
// the loop.  Lanes whose windows stand at the same digit are added with
// 32-lane integer reductions (16-bit halves, so a sum of 32 fits a word) and
// one lane per digit writes the sum: a 64-bit shared-memory atomic add per
// lane and digit is a compare-and-swap loop that serialises the warp.
__device__ __forceinline__ void xd_warp_deposit(unsigned long long* acc, const XdWin& a)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    __syncwarp();
    unsigned todo = __ballot_sync(full, a.d0 >= 0);
    while (todo) {
        const int d = __shfl_sync(full, a.d0, __ffs(todo) - 1);
        const bool mine = a.d0 == d;
        todo &= ~__ballot_sync(full, mine);
        unsigned long long s = 0ULL;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const unsigned v = mine ? a.w[k] : 0u;
            const unsigned lo = __reduce_add_sync(full, v & 0xffffu), hi = __reduce_add_sync(full, v >> 16);
            if (lane == k) s = (unsigned long long)lo + ((unsigned long long)hi << 16);
        }
        const unsigned neg = __popc(__ballot_sync(full, mine && (a.w[5] >> 31)));
        if (lane == 6) s = 0ULL - neg;
        if (lane < 7 && s) acc[d + lane] += s;
        __syncwarp();
    }
}

__device__ __forceinline__ void xd_win_add(unsigned long long* acc, XdWin& a, double x, double y, int* bad)
{
    unsigned long long mx, my;
    int ex, ey, nx, ny;
    bool zx = !xd_split(x, mx, ex, nx);
    bool zy = !xd_split(y, my, ey, ny);
    if (ex == 972 || ey == 972) { *bad = 1; return; }   // exponent field 2047: inf or nan
    if (zx || zy) return;
    const unsigned __int128 p = (unsigned __int128)mx * my;
    const unsigned p0 = unsigned(p), p1 = unsigned(p >> 32), p2 = unsigned(p >> 64), p3 = unsigned(p >> 96);
    const int pos = ex + ey + XD_BIAS;
    const int d = pos >> 5;
    if (d != a.d0 && d != a.d0 + 1) {
        // the window moves so that it holds this digit and the neighbour
        // that the product is nearer to: products within 16 bits of this one
        // need no further move (each is seven shared-memory atomics)
        xd_win_deposit(acc, a);
        const int d0 = (pos & 31) < 16 && d > 0 ? d - 1 : d;
        xd_win_init(a);
        a.d0 = d0;
    }
    const unsigned m = (nx ^ ny) ? 0xffffffffu : 0u;   // -p = ~p + 1
    const unsigned q0 = __funnelshift_l(0u, p0, pos) ^ m;
    const unsigned q1 = __funnelshift_l(p0, p1, pos) ^ m;
    const unsigned q2 = __funnelshift_l(p1, p2, pos) ^ m;
    const unsigned q3 = __funnelshift_l(p2, p3, pos) ^ m;
    const unsigned q4 = __funnelshift_l(p3, 0u, pos) ^ m;
    const bool up = d != a.d0;                          // product one digit above the window's base
    const unsigned r0 = up ? m : q0, r1 = up ? q0 : q1, r2 = up ? q1 : q2, r3 = up ? q2 : q3, r4 = up ? q3 : q4,
                   r5 = up ? q4 : m;
    asm("{\n\t"
        ".reg .u32 t;\n\t"
        "add.cc.u32 t, %12, %12;\n\t"                   // carry in = 1 for a negative product
        "addc.cc.u32 %0, %0, %6;\n\t"
        "addc.cc.u32 %1, %1, %7;\n\t"
        "addc.cc.u32 %2, %2, %8;\n\t"
        "addc.cc.u32 %3, %3, %9;\n\t"
        "addc.cc.u32 %4, %4, %10;\n\t"
        "addc.u32 %5, %5, %11;\n\t"
        "}"
        : "+r"(a.w[0]), "+r"(a.w[1]), "+r"(a.w[2]), "+r"(a.w[3]), "+r"(a.w[4]), "+r"(a.w[5])
        : "r"(r0), "r"(r1), "r"(r2), "r"(r3), "r"(r4), "r"(r5), "r"(m));
}

// Digits lo .. hi of an accumulator, spread too far for the lanes of a warp:
// one thread walks them.  The accumulator is left altered.
static __device__ inline double xd_round_serial(unsigned long long* g, int lo, int hi)
{
    double r = 0.0;
    long long* d = reinterpret_cast<long long*>(g);
    const long long MASK = 0xffffffffLL;
    long long carry = 0;
    int top = hi;
    for (int i = lo; i <= hi; ++i) {
        const long long v = d[i] + carry;
        d[i] = v & MASK;
        carry = v >> 32;                       // floor((v - low) / 2^32)
    }
    while (carry != 0 && carry != -1 && top < XD_DIGITS - 1) {
        d[++top] = carry & MASK;
        carry >>= 32;
    }
    const bool neg = carry < 0;
    if (neg) {                                 // magnitude: two's complement of the digits
        long long c = 1;
        for (int i = lo; i <= top; ++i) {
            const long long v = (~d[i] & MASK) + c;
            d[i] = v & MASK;
            c = v >> 32;
        }
        if (c && top < XD_DIGITS - 1) d[++top] = c;
    }
    const int last = top;
    while (top >= lo && d[top] == 0) --top;
    if (top >= lo) {
        const int hb = 63 - __clzll(d[top]);
        const int P = top * 32 + hb;           // most significant bit
        int lsb = P - 52;                      // last bit kept
        if (lsb < XD_BIAS - 1074) lsb = XD_BIAS - 1074;
        auto dig = [&](int i) -> unsigned long long {
            return i >= lo && i <= last ? (unsigned long long)d[i] : 0ULL;
        };
        const int q = lsb >> 5, s = lsb & 31;  // lsb >= XD_BIAS - 1074 > 0
        unsigned long long M = (dig(q) | (dig(q + 1) << 32)) >> s;
        if (s) M |= dig(q + 2) << (64 - s);
        const int rp = lsb - 1;                // rounding bit; the bits below it are sticky
        const int rb = int((dig(rp >> 5) >> (rp & 31)) & 1ULL);
        bool sticky = (dig(rp >> 5) & ((1ULL << (rp & 31)) - 1ULL)) != 0ULL;
        for (int i = lo; i < (rp >> 5) && i <= last && !sticky; ++i) sticky = d[i] != 0;
        if (rb && (sticky || (M & 1ULL))) M += 1ULL;
        r = scalbn((double)M, lsb - XD_BIAS);
        if (neg) r = -r;
    }
    return r;
}

// One warp: carry propagation and round-to-nearest-even of an accumulator in
// shared memory.  The products of one dot product touch a few digits of the
// 140; with at most 28 between the lowest and the highest nonzero one, lane
// i takes digit lo + i and the whole number, a two's complement of 32 digits,
// is resolved at once: two local carry steps leave each digit within one unit
// of its range, and the remaining chains of carries and borrows are a mask
// addition each (a run of all-ones digits passes a carry on as a run of ones
// does in an integer).  A thread that walked the digits took about as long as
// the rest of a small dot product.  Every lane gets the result.
static __device__ inline double xd_round(unsigned long long* g)
{
    const unsigned full = 0xffffffffu, M = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    int lo = XD_DIGITS, hi = -1;
#pragma unroll
    for (int k = 0; k < (XD_DIGITS + 31) / 32; ++k) {
        const int i = k * 32 + lane;
        const unsigned b = __ballot_sync(full, i < XD_DIGITS && g[i] != 0ULL);
        if (b) {
            lo = min(lo, k * 32 + __ffs(b) - 1);
            hi = k * 32 + 31 - __clz(b);
        }
    }
    if (hi < 0) return 0.0;
    if (hi - lo > 27) {
        const double r = lane == 0 ? xd_round_serial(g, lo, hi) : 0.0;
        return __shfl_sync(full, r, 0);
    }
    // v = l + 2^32 h; each digit passes its h up, twice: t in [-1, 2^32]
    long long v = lo + lane <= hi ? (long long)g[lo + lane] : 0LL;
#pragma unroll
    for (int step = 0; step < 2; ++step) {
        long long up = __shfl_up_sync(full, v >> 32, 1);
        if (lane == 0) up = 0;
        v = (v & 0xffffffffLL) + up;
    }
    // digits u = 2^32 generate a carry, all-ones digits pass one on
    const bool minus = v < 0;                       // -1: a digit 0 that owes one
    unsigned u = minus ? 0u : unsigned(v);
    unsigned gen = __ballot_sync(full, v > 0xffffffffLL), pass = __ballot_sync(full, v == 0xffffffffLL);
    u += (((pass + (gen << 1)) ^ pass) >> lane) & 1u;
    // then the owed units: digits 0 that owe generate a borrow, digits that
    // come out 0 pass one on
    gen = __ballot_sync(full, minus && u == 0u);
    const unsigned w = u - (minus ? 1u : 0u);
    pass = __ballot_sync(full, w == 0u);
    u = w - ((((pass + (gen << 1)) ^ pass) >> lane) & 1u);
    // magnitude of a negative number (at least four digits above hi hold its sign)
    const bool neg = __shfl_sync(full, u, 31) >> 31;
    if (neg) {
        u = ~u;
        pass = __ballot_sync(full, u == M);
        u += (((pass + 1u) ^ pass) >> lane) & 1u;
    }
    const unsigned nz = __ballot_sync(full, u != 0u);
    if (!nz) return 0.0;
    const int top = 31 - __clz(nz);
    const int P = (lo + top) * 32 + 31 - __clz(__shfl_sync(full, u, top));   // most significant bit
    int lsb = P - 52;                               // last bit kept
    if (lsb < XD_BIAS - 1074) lsb = XD_BIAS - 1074;
    auto dig = [&](int i) -> unsigned long long {
        const unsigned x = __shfl_sync(full, u, (i - lo) & 31);
        return i >= lo && i < lo + 32 ? x : 0u;
    };
    const int q = lsb >> 5, s = lsb & 31;           // lsb >= XD_BIAS - 1074 > 0
    const unsigned long long d0 = dig(q), d1 = dig(q + 1), d2 = dig(q + 2);
    unsigned long long m = (d0 | (d1 << 32)) >> s;
    if (s) m |= d2 << (64 - s);
    const int rp = lsb - 1;                         // rounding bit; the bits below it are sticky
    const unsigned long long dr = dig(rp >> 5);
    const bool sticky = (dr & ((1ULL << (rp & 31)) - 1ULL)) != 0ULL ||
                        __ballot_sync(full, u != 0u && lo + lane < (rp >> 5)) != 0u;
    if (((dr >> (rp & 31)) & 1ULL) && (sticky || (m & 1ULL))) m += 1ULL;
    const double r = scalbn((double)m, lsb - XD_BIAS);
    return neg ? -r : r;
}

// The products of one block: load(i) reads the operands of element i,
// XD_UNROLL elements in flight per thread, and ops(i, raw) gives its two
// factors (and may store).  The block's digits are in sacc[0] afterwards.
template <class Load, class Ops>
__device__ __forceinline__ void xd_block(long long n, unsigned long long (*sacc)[XD_DIGITS], int* bad,
                                         const Load& load, const Ops& ops)
{
    using Raw = decltype(load(0LL));
    for (int t = threadIdx.x; t < XD_WARPS * XD_DIGITS; t += XD_THREADS) (&sacc[0][0])[t] = 0ULL;
    __syncthreads();
    unsigned long long* mine = sacc[threadIdx.x >> 5];
    XdWin win;
    xd_win_init(win);
    const long long stride = (long long)gridDim.x * XD_THREADS;
    for (long long i = (long long)blockIdx.x * XD_THREADS + threadIdx.x; i < n; i += XD_UNROLL * stride) {
        Raw v[XD_UNROLL];
#pragma unroll
        for (int u = 0; u < XD_UNROLL; ++u)
            if (i + u * stride < n) v[u] = load(i + u * stride);
#pragma unroll
        for (int u = 0; u < XD_UNROLL; ++u)
            if (i + u * stride < n) {
                const double2 f = ops(i + u * stride, v[u]);
                xd_win_add(mine, win, f.x, f.y, bad);
            }
    }
    xd_warp_deposit(mine, win);
    __syncthreads();
    for (int t = threadIdx.x; t < XD_DIGITS; t += XD_THREADS) {
        unsigned long long s = 0ULL;
#pragma unroll
        for (int w = 0; w < XD_WARPS; ++w) s += sacc[w][t];
        sacc[0][t] = s;
    }
}

// Adds the block's digits into the global accumulator; true in the last
// block to arrive (atomic ticket, reset for the next call), which then holds
// the global digits in sacc[0] and has cleared them.  A launch of one block
// keeps its digits where they are.
__device__ __forceinline__ bool xd_grid_sum(unsigned long long (*sacc)[XD_DIGITS], unsigned long long* gacc,
                                            unsigned* ticket)
{
    __shared__ bool last;
    if (gridDim.x == 1) {
        __syncthreads();
        return true;
    }
    for (int t = threadIdx.x; t < XD_DIGITS; t += XD_THREADS)
        if (sacc[0][t]) atomicAdd(gacc + t, sacc[0][t]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return false;
    __threadfence();
    for (int t = threadIdx.x; t < XD_DIGITS; t += XD_THREADS) sacc[0][t] = atomicExch(gacc + t, 0ULL);
    if (threadIdx.x == 0) *ticket = 0u;
    __syncthreads();
    return true;
}

// First warp of a block: rounds and writes the double and its square root
__device__ __forceinline__ void xd_write(unsigned long long* g, const int* bad, double* out, double* out_sqrt)
{
    if (threadIdx.x >= 32) return;
    double r = xd_round(g);
    if (threadIdx.x != 0) return;
    if (*(volatile const int*)bad) r = __longlong_as_double(0x7ff8000000000000LL);
    if (out) *out = r;
    if (out_sqrt) *out_sqrt = __dsqrt_rn(r);
}

// Blocks of a dot product of length n: at least XD_UNROLL elements per
// thread before another block is worth its share of the final sum, at most
// four resident blocks (32 warps) per SM.  Up to 2048 elements one block
// takes all (at most 8 elements a thread) and the global sum falls away.
inline int xd_grid(long long n, int sms)
{
    if (n <= 2048) return 1;
    const long long b = (n + XD_THREADS * XD_UNROLL - 1) / (XD_THREADS * XD_UNROLL);
    return int(b < 4LL * sms ? b : 4LL * sms);
}

// Block: XD_THREADS threads.  gacc: XD_DIGITS words, zero on entry of the
// first block (cleared by the caller).  bad: set when an input is inf/nan.
static __global__ void __launch_bounds__(XD_THREADS, 4)
k_xdot_accumulate(long long n, const double* __restrict__ x, const double* __restrict__ y,
                  unsigned long long* __restrict__ gacc, int* bad)
{
    __shared__ unsigned long long sacc[XD_WARPS][XD_DIGITS];
    xd_block(n, sacc, bad, [&](long long i) { return make_double2(x[i], y[i]); },
             [](long long, double2 v) { return v; });
    for (int t = threadIdx.x; t < XD_DIGITS; t += XD_THREADS)
        if (sacc[0][t]) atomicAdd(gacc + t, sacc[0][t]);
}

// One warp: takes the global digits into shared memory (reading and
// clearing each word in one atomic exchange) and rounds.
static __global__ void k_xdot_finalize(unsigned long long* gacc, const int* bad, double* out,
                                       double* out_sqrt)
{
    __shared__ unsigned long long d[XD_DIGITS];
    if (blockIdx.x != 0 || threadIdx.x >= 32) return;
    for (int t = threadIdx.x; t < XD_DIGITS; t += 32) d[t] = atomicExch(gacc + t, 0ULL);
    __syncwarp();
    xd_write(d, bad, out, out_sqrt);
}

// Accumulation and rounding in one launch: the last block to finish takes
// the global digits, clearing them, and rounds.
static __global__ void __launch_bounds__(XD_THREADS, 4)
k_xdot(long long n, const double* __restrict__ x, const double* __restrict__ y,
       unsigned long long* __restrict__ gacc, int* bad, unsigned* ticket, double* out, double* out_sqrt)
{
    __shared__ unsigned long long sacc[XD_WARPS][XD_DIGITS];
    xd_block(n, sacc, bad, [&](long long i) { return make_double2(x[i], y[i]); },
             [](long long, double2 v) { return v; });
    if (xd_grid_sum(sacc, gacc, ticket)) xd_write(sacc[0], bad, out, out_sqrt);
}

// One modified Gram-Schmidt step fused with the next correctly rounded dot
// product, in one pass: when vprev is given, w_i <- w_i - (h * vprev_i)
// with h = *hprev (product rounded, then the difference: the same two
// roundings as a separate update kernel); then <w, y> (y = w itself when
// null) accumulated exactly and rounded by the last block, as k_xdot.
static __global__ void __launch_bounds__(XD_THREADS, 4)
k_mgs_xdot(long long n, double* __restrict__ w, const double* __restrict__ vprev, const double* hprev,
           const double* __restrict__ y, unsigned long long* __restrict__ gacc, int* bad, unsigned* ticket,
           double* out, double* out_sqrt)
{
    __shared__ unsigned long long sacc[XD_WARPS][XD_DIGITS];
    const double h = vprev ? *hprev : 0.0;
    xd_block(n, sacc, bad,
             [&](long long i) { return make_double3(w[i], vprev ? vprev[i] : 0.0, y ? y[i] : 0.0); },
             [&](long long i, double3 v) {
                 double wi = v.x;
                 if (vprev) {
                     wi = __dsub_rn(wi, __dmul_rn(h, v.y));
                     w[i] = wi;
                 }
                 return make_double2(wi, y ? v.z : wi);
             });
    if (xd_grid_sum(sacc, gacc, ticket)) xd_write(sacc[0], bad, out, out_sqrt);
}

constexpr int XC_WARPS = 16, XC_THREADS = XC_WARPS * 32, XC_MAX_E = 8;
constexpr long long XC_SPIN_LIMIT = 2000000;   // ~1 s of polls

// One thread: waits until *arrivals has reached target; false, with *err
// set, after `limit` polls without it or once *err is set.
__device__ __forceinline__ bool xc_wait(unsigned* arrivals, unsigned target, int* err, long long limit)
{
    for (long long spins = 0;; ++spins) {
        unsigned seen;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(arrivals) : "memory");
        if (int(seen - target) >= 0) return true;
        if (spins >= limit) {
            atomicExch(err, 1);
            return false;
        }
        if ((spins & 1023) == 1023 && *(volatile int*)err) return false;
    }
}

// Failure-detection check: one block waits for a second one's arrival, which
// never comes, and must give up after `limit` polls.
// state: [arrivals, err], zero.
static __global__ void k_column_timeout_check(unsigned* state, long long limit)
{
    if (threadIdx.x != 0) return;
    atomicAdd(state, 1u);
    xc_wait(state, 2u, reinterpret_cast<int*>(state + 1), limit);
}

// One column of a modified Gram-Schmidt process in one launch: for i = 0..j
// h_i = <w, v_i> (correctly rounded), w <- w - (h_i v_i) (product rounded,
// then the difference), then h_{j+1} = ||w|| and v_{j+1} = w / h_{j+1}.  The
// dots are a serial chain; a launch for each costs its start, its last
// block's global sums and their round trips, ~14 us at a few thousand
// elements.  Here w stays in registers (E elements a thread), the next basis
// vector loads while the dot is summed, the blocks add their digits into one
// of three rotating accumulators, meet at a grid barrier, and every block
// rounds the sum for itself.  Measured against one k_mgs_xdot per dot: the
// 2,100 dots of a 97 x 80 setup with their SpMVs and host reads 23 -> 15 ms,
// the coarse polynomial of 106k rows (100 steps, 5,150 dots) 103 -> 67 ms;
// bound by the chain of one dot (~5 us: digits, barrier, rounding).
//   gdig: 3 x XD_DIGITS words, zero before the first launch; `phase`: dots
// summed there by earlier launches, mod 3; the accumulator two places ahead
// is cleared behind each barrier, before the next one.
//   arrivals: counter of barrier arrivals, `base` of them by earlier
// launches.  One block needs none of these.
//   The wait for the other blocks is bounded.  A block that gives up (`limit`
// polls, or another block's word that it did) sets *err and ends there, so
// nothing is ever computed from an incomplete sum: w and the earlier columns
// are as they were, hcol, vnext and the accumulators are not to be used, and
// the caller takes the column from w again, one launch per dot.
template <int E>
static __global__ void __launch_bounds__(XC_THREADS, 1)
k_mgs_column(int n, const double* __restrict__ V, int j, const double* __restrict__ w,
             double* __restrict__ vnext, double* __restrict__ hcol, unsigned long long* gdig, int phase,
             unsigned* arrivals, unsigned base, int* bad, int* err, long long limit)
{
    __shared__ unsigned long long sacc[XC_WARPS][XD_DIGITS];
    __shared__ unsigned long long tot[XD_DIGITS];
    __shared__ double hs;
    __shared__ bool gave_up;
    if (threadIdx.x == 0) gave_up = false;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int t = threadIdx.x; t < XC_WARPS * XD_DIGITS; t += XC_THREADS) (&sacc[0][0])[t] = 0ULL;
    const int i0 = blockIdx.x * (XC_THREADS * E) + threadIdx.x;
    double we[E], y[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int r = i0 + e * XC_THREADS;
        we[e] = r < n ? w[r] : 0.0;
        y[e] = r < n ? V[r] : 0.0;
    }
    __syncthreads();
    for (int i = 0;; ++i) {
        XdWin win;
        xd_win_init(win);
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (i0 + e * XC_THREADS < n) xd_win_add(sacc[warp], win, we[e], i <= j ? y[e] : we[e], bad);
        double yn[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int r = i0 + e * XC_THREADS;
            yn[e] = i < j && r < n ? V[(long long)(i + 1) * n + r] : 0.0;
        }
        xd_warp_deposit(sacc[warp], win);
        __syncthreads();
        unsigned long long* g = gdig + ((phase + i) % 3) * XD_DIGITS;
        if (threadIdx.x < XD_DIGITS) {
            const int t = threadIdx.x;
            unsigned long long s = 0ULL;
#pragma unroll
            for (int q = 0; q < XC_WARPS; ++q) {
                s += sacc[q][t];
                sacc[q][t] = 0ULL;
            }
            if (gridDim.x == 1) tot[t] = s;
            else if (s) atomicAdd(g + t, s);
        }
        __syncthreads();
        if (warp == 0) {
            if (gridDim.x > 1) {
                if (lane == 0) {
                    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(arrivals) : "memory");
                    gave_up = !xc_wait(arrivals, base + gridDim.x * unsigned(i + 1), err, limit);
                }
                __syncwarp();
                for (int t = lane; t < XD_DIGITS; t += 32) tot[t] = __ldcg(g + t);
                __syncwarp();
            }
            double r = xd_round(tot);
            if (lane == 0) {
                if (*(volatile int*)bad) r = __longlong_as_double(0x7ff8000000000000LL);
                if (i > j) r = __dsqrt_rn(r);
                hs = r;
                if (blockIdx.x == 0) hcol[i] = r;
            }
            if (gridDim.x > 1 && blockIdx.x == 0) {
                unsigned long long* z = gdig + ((phase + i + 2) % 3) * XD_DIGITS;
                for (int t = lane; t < XD_DIGITS; t += 32) z[t] = 0ULL;
            }
        }
        __syncthreads();
        if (gave_up) return;
        const double h = hs;
        if (i > j) {
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (i0 + e * XC_THREADS < n) vnext[i0 + e * XC_THREADS] = __ddiv_rn(we[e], h);
            return;
        }
#pragma unroll
        for (int e = 0; e < E; ++e) {
            we[e] = __dsub_rn(we[e], __dmul_rn(h, y[e]));
            y[e] = yn[e];
        }
    }
}

}  // namespace airg
