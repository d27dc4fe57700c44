// Many right-hand sides on one hierarchy: the V-cycle of Eq. 6 applied to k
// vectors at once (an SpMM-style V-cycle) inside k independent FGMRES
// iterations advanced in lockstep.
//
// Layout: a batch of k vectors of length n is stored row-major, [row][rhs],
// in the nested F/C order of the single solve.  Every operator kernel gives
// a row to a group of lanes, each with adjacent right-hand sides (Lanes
// below): each stored entry of the row is read once per group (broadcast) and
// reused for all k right-hand sides, and the gathers of x read k consecutive
// values of one row -- contiguous, coalesced.  The operator bytes of a
// V-cycle are thus paid once per k right-hand sides.
//
// A right-hand side whose FGMRES residual reaches its tolerance is frozen:
// its next basis vector is zero and its least-squares solution uses only
// the columns built while it was active.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>

#include "dev_util.cuh"
#include "handle.h"
#include "solve_internal.cuh"

namespace airg {

namespace {

constexpr int BT = 256;          // threads per block (8 rows of the batch)
constexpr int MAXB = 16;         // restart length of the batched FGMRES
constexpr int MAXK = 128;        // right-hand sides per batch (KW <= 4)


// How the lanes of a warp share the k right-hand sides of a row: each lane
// holds VEC adjacent ones (one 16-byte load where k allows it, else one), a
// group of 2^lg lanes covers a row, and the warp's other groups take the
// next rows.  A lane then keeps the loads of 32 >> lg rows' worth of work in
// flight per warp instruction, and a narrow batch leaves no lane idle: with
// one warp per row, 7 right-hand sides used 7 of 32 lanes of every FP64
// instruction, and a row of 2-3 entries was a warp's whole work.  Wider
// batches than a warp covers take KW steps of it.  The sums of a (row,
// right-hand side) are the same in every shape.
// Bound: FP64 issue and gather latency on the long rows, memory on the short
// ones.  Measured before and after, per launch: coarse step of 7 right-hand
// sides (10k rows of 71 entries, FP64) 55.6 -> 20.2 us; of 32 (41k rows of
// 199 entries, FP32) 197 -> 81 us; first smoother term of 32 (1.8M rows of
// 1.4 entries) 335 -> 174 us (4.3 TB/s); FP64 top-level product of 32 (4.2M
// rows of 3 entries) 1.64 -> 1.15 ms.
template <class T, int VEC, int KW>
struct Lanes {
    int ql, lg, k;
    __device__ __forceinline__ int q(int j) const { return (ql + (j << lg)) * VEC; }
    // KW = 2 and 4 hold more than 32 and 64 packs
    __device__ __forceinline__ bool ok(int j) const { return j < KW / 2 || q(j) < k; }
};
template <class T, int VEC>
struct alignas(sizeof(T) * VEC) Pack {
    T v[VEC];
};
// this lane's values of one row
template <class T, int VEC, int KW>
struct Vals {
    Pack<T, VEC> p[KW];
};

template <class T, int VEC, int KW>
__device__ __forceinline__ Vals<T, VEC, KW> bload(const Lanes<T, VEC, KW>& L, const T* __restrict__ a, long long r)
{
    Vals<T, VEC, KW> o;
#pragma unroll
    for (int j = 0; j < KW; ++j) {
        if (a && r >= 0 && L.ok(j)) o.p[j] = *reinterpret_cast<const Pack<T, VEC>*>(a + size_t(r) * L.k + L.q(j));
        else
#pragma unroll
            for (int u = 0; u < VEC; ++u) o.p[j].v[u] = T(0);
    }
    return o;
}
template <class T, int VEC, int KW>
__device__ __forceinline__ void bstore(const Lanes<T, VEC, KW>& L, T* a, long long r, const Vals<T, VEC, KW>& o)
{
#pragma unroll
    for (int j = 0; j < KW; ++j)
        if (L.ok(j)) *reinterpret_cast<Pack<T, VEC>*>(a + size_t(r) * L.k + L.q(j)) = o.p[j];
}
// a[r] = f(values of the operands), element by element.  With four steps of
// the warp the values are formed under the store's condition, so that a step
// past the last right-hand side costs no FP64 work (96 right-hand sides, FP64,
// 1024^2: 244.9 -> 241.6 ms); with fewer, all steps but the last are full and
// that condition costs registers (31: 78.5 -> 80.0 ms).
template <class T, int VEC, int KW, class F, class... A>
__device__ __forceinline__ void bstore(const Lanes<T, VEC, KW>& L, T* a, long long r, const F& f,
                                       const Vals<T, VEC, KW>& x, const A&... more)
{
    Vals<T, VEC, KW> o;
#pragma unroll
    for (int j = 0; j < KW; ++j) {
        if (KW == 4 && !L.ok(j)) continue;
#pragma unroll
        for (int u = 0; u < VEC; ++u) o.p[j].v[u] = f(x.p[j].v[u], more.p[j].v[u]...);
        if (KW == 4) *reinterpret_cast<Pack<T, VEC>*>(a + size_t(r) * L.k + L.q(j)) = o.p[j];
    }
    if (KW < 4) bstore(L, a, r, o);
}

// Rows of operator S times the k right-hand sides x ([row][rhs]): row r is
// handled by one lane group (above) of PW warps of a block.  Warp `part` of
// a row adds the row's stored entries e = part, part + PW, ... in order
// (after the dense diagonal term, part 0); with PW > 1 the partial rows meet
// in shared memory and are added in part order.  PW is fixed per operator
// from its row lengths (1 for short rows, 4 for long ones), so results do
// not depend on timing.  pre(r, L) loads the row's other operands before the
// product, so those loads overlap the gathers; entries are taken four at a
// time with all their loads issued before their FMAs, which run in entry
// order, and up to three that are left together too.  Rows of several steps
// of a warp (KW > 1) take those one by one, know their row's warp at compile
// time and add zeros for lanes without a right-hand side: each of these saves
// registers, and with them a third of the warps in flight (FP64, 1024^2: 33
// right-hand sides 137 -> 122 ms, 65 300 -> 237, 127 327 -> 253; FP32: 63 59
// -> 55, 65 94 -> 69, 127 114 -> 88).  Then epi(r, L, sums, pre) runs once per
// row.  `dot` = false skips the product (sums 0).  Every thread of the block
// reaches the barrier.
// X: the type x is stored in (FP32 under an FP64 operator: widened exactly).
template <class T, int VEC, int KW, int PW, class V, class X, class Pre, class Epi>
__device__ __forceinline__ void bfor_rows(const SellView<T, V>& S, const X* __restrict__ x, int k, int lg,
                                          bool dot, const Pre& pre, const Epi& epi, int rev = 0)
{
    using LN = Lanes<T, VEC, KW>;
    using PK = Pack<X, VEC>;
    using PV = decltype(pre(0, LN{}));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int part = warp % PW;
    if constexpr (KW > 1) lg = 5;   // a whole warp a row
    const LN L{lane & ((1 << lg) - 1), lg, k};
    // rev != 0: blocks take the rows in reverse order (serpentine chains)
    const int bx = rev ? int(gridDim.x) - 1 - int(blockIdx.x) : int(blockIdx.x);
    long long rr = (long long)bx * (BT / 32 / PW) + warp / PW;
    if constexpr (KW == 1) rr = rr * (32 >> lg) + (lane >> lg);
    const bool valid = rr < S.n_rows;
    const int r = valid ? int(rr) : 0;
    const bool lead = valid && part == 0;
    const PV pv = lead ? pre(r, L) : PV{};
    Vals<T, VEC, KW> acc;
#pragma unroll
    for (int j = 0; j < KW; ++j)
#pragma unroll
        for (int u = 0; u < VEC; ++u) acc.p[j].v[u] = T(0);
    if (valid && dot) {
        if (part == 0 && S.diag) {
            const T dg = __ldg(S.diag + r);
#pragma unroll
            for (int j = 0; j < KW; ++j)
                if (L.ok(j)) {
                    const PK d = *reinterpret_cast<const PK*>(x + size_t(r) * k + L.q(j));
#pragma unroll
                    for (int u = 0; u < VEC; ++u) acc.p[j].v[u] = dg * wide<T>(d.v[u]);
                }
        }
        const int s = r >> 5;
        const int b = S.sptr[s] + (r & 31), w = (S.sptr[s + 1] - S.sptr[s]) >> 5;
        int e = part;
        for (; e + 3 * PW < w; e += 4 * PW) {
            T v[4];
            const X* xr[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int idx = b + 32 * (e + u * PW);
                v[u] = ldval<T>(S.val + idx);
                xr[u] = x + size_t(__ldg(S.col + idx)) * k;
            }
            PK xv[4][KW];
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int j = 0; j < KW; ++j)
                    if (L.ok(j)) xv[u][j] = *reinterpret_cast<const PK*>(xr[u] + L.q(j));
                    else if constexpr (VEC == 1)
#pragma unroll
                        for (int i = 0; i < VEC; ++i) xv[u][j].v[i] = X(0);
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int j = 0; j < KW; ++j)
                    if (VEC == 1 || L.ok(j))
#pragma unroll
                        for (int i = 0; i < VEC; ++i) acc.p[j].v[i] = fma(v[u], wide<T>(xv[u][j].v[i]), acc.p[j].v[i]);
        }
        if constexpr (KW > 1) {
            for (; e < w; e += PW) {
                const int idx = b + 32 * e;
                const T v = ldval<T>(S.val + idx);
                const X* xr = x + size_t(__ldg(S.col + idx)) * k;
#pragma unroll
                for (int j = 0; j < KW; ++j)
                    if (L.ok(j)) {
                        const PK xv = *reinterpret_cast<const PK*>(xr + L.q(j));
#pragma unroll
                        for (int i = 0; i < VEC; ++i) acc.p[j].v[i] = fma(v, wide<T>(xv.v[i]), acc.p[j].v[i]);
                    }
            }
        } else if (e < w) {   // up to three entries left, their loads together too
            T v[3];
            const X* xr[3];
            PK xv[3][KW];
#pragma unroll
            for (int u = 0; u < 3; ++u)
                if (e + u * PW < w) {
                    const int idx = b + 32 * (e + u * PW);
                    v[u] = ldval<T>(S.val + idx);
                    xr[u] = x + size_t(__ldg(S.col + idx)) * k;
                }
#pragma unroll
            for (int u = 0; u < 3; ++u)
#pragma unroll
                for (int j = 0; j < KW; ++j)
                    if (e + u * PW < w && L.ok(j)) xv[u][j] = *reinterpret_cast<const PK*>(xr[u] + L.q(j));
#pragma unroll
            for (int u = 0; u < 3; ++u)
#pragma unroll
                for (int j = 0; j < KW; ++j)
                    if (e + u * PW < w && L.ok(j))
#pragma unroll
                        for (int i = 0; i < VEC; ++i) acc.p[j].v[i] = fma(v[u], wide<T>(xv[u][j].v[i]), acc.p[j].v[i]);
        }
    }
    if constexpr (PW > 1) {
        __shared__ T red[BT / 32][KW * VEC][32];
#pragma unroll
        for (int j = 0; j < KW; ++j)
#pragma unroll
            for (int u = 0; u < VEC; ++u) red[warp][j * VEC + u][lane] = acc.p[j].v[u];
        __syncthreads();
        if (part == 0) {
#pragma unroll
            for (int p = 1; p < PW; ++p)
#pragma unroll
                for (int j = 0; j < KW; ++j)
#pragma unroll
                    for (int u = 0; u < VEC; ++u) acc.p[j].v[u] += red[warp + p][j * VEC + u][lane];
        }
    }
    if (lead) epi(r, L, acc, pv);
}

// blocks for n rows at PW warps per lane group of 2^lg lanes
inline int grid_rows(long long n, int pw, int lg)
{
    const int per = (BT / 32 / pw) * (32 >> lg);
    return grid_for(n, per);
}

template <class T, int VEC, int KW>
struct Vals2 {
    Vals<T, VEC, KW> a, b;
};

template <class T, int VEC, int KW, int PW, class X>
__global__ void kb_spmv(SellView<T> S, const X* __restrict__ x, T* __restrict__ y, int k, int lg)
{
    using LN = Lanes<T, VEC, KW>;
    using VL = Vals<T, VEC, KW>;
    bfor_rows<T, VEC, KW, PW>(S, x, k, lg, true, [](int, const LN&) { return 0; },
                              [&](int r, const LN& L, const VL& d, int) { bstore(L, y, r, d); });
}

template <class T, int VEC, int KW, int PW, class V = T>
__global__ void kb_restrict(SellView<T, V> Z, const T* __restrict__ sf, const T* __restrict__ sc,
                            T* __restrict__ dc, int k, int lg)
{
    using LN = Lanes<T, VEC, KW>;
    using VL = Vals<T, VEC, KW>;
    bfor_rows<T, VEC, KW, PW>(Z, sf, k, lg, true, [&](int r, const LN& L) { return bload(L, sc, r); },
                              [&](int r, const LN& L, const VL& d, const VL& c) {
                                  bstore(L, dc, r, [](T a, T b) { return a + b; }, c, d);
                              });
}

template <class T, int VEC, int KW, int PW>
__global__ void kb_fresid(SellView<T> M, const T* __restrict__ rf, const T* __restrict__ ec,
                          T* __restrict__ t, T* __restrict__ w, T ap, int k, int lg)
{
    using LN = Lanes<T, VEC, KW>;
    using VL = Vals<T, VEC, KW>;
    bfor_rows<T, VEC, KW, PW>(M, ec, k, lg, true, [&](int r, const LN& L) { return bload(L, rf, r); },
                              [&](int r, const LN& L, const VL& d, const VL& f) {
                                  bstore(L, t, r, [](T a, T b) { return a - b; }, f, d);
                                  bstore(L, w, r, [&](T a, T b) { return ap * (a - b); }, f, d);
                              });
}

template <class T, int VEC, int KW, int PW>
__global__ void kb_horner(SellView<T> A, const T* __restrict__ t, const T* __restrict__ win,
                          T* __restrict__ wout, T ak, int k, int lg, int rev)
{
    using LN = Lanes<T, VEC, KW>;
    using VL = Vals<T, VEC, KW>;
    bfor_rows<T, VEC, KW, PW>(A, win, k, lg, true, [&](int r, const LN& L) { return bload(L, t, r); },
                              [&](int r, const LN& L, const VL& d, const VL& tv) {
                                  bstore(L, wout, r, [&](T a, T b) { return fma(ak, a, b); }, tv, d);
                              }, rev);
}

template <class T, int VEC, int KW, int PW>
__global__ void kb_horner_last(SellView<T> A, const T* __restrict__ t, const T* __restrict__ win,
                               const T* __restrict__ ec, const int* __restrict__ W,
                               T* __restrict__ ef, T a0, int k, int lg, int rev)
{
    using LN = Lanes<T, VEC, KW>;
    using VL = Vals<T, VEC, KW>;
    using V2 = Vals2<T, VEC, KW>;
    bfor_rows<T, VEC, KW, PW>(A, win, k, lg, true,
                              [&](int r, const LN& L) { return V2{bload(L, t, r), bload(L, ec, W[r])}; },
                              [&](int r, const LN& L, const VL& d, const V2& q) {
                                  bstore(L, ef, r, [&](T e, T a, T b) { return e + fma(a0, a, b); }, q.b, q.a, d);
                              }, rev);
}

// last Horner term of an in-place smoother: e += a_0 t + A win (C-point
// smooth, second F-point smooth of FCF; with win = t and a_0 = 0 it applies
// an assembled inverse)
template <class T, int VEC, int KW, int PW>
__global__ void kb_horner_acc(SellView<T> A, const T* __restrict__ t, const T* __restrict__ win, T* e, T a0,
                              int k, int lg, int rev)
{
    using LN = Lanes<T, VEC, KW>;
    using VL = Vals<T, VEC, KW>;
    using V2 = Vals2<T, VEC, KW>;
    bfor_rows<T, VEC, KW, PW>(A, win, k, lg, true,
                              [&](int r, const LN& L) { return V2{bload(L, t, r), bload(L, (const T*)e, r)}; },
                              [&](int r, const LN& L, const VL& d, const V2& q) {
                                  bstore(L, e, r, [&](T ee, T a, T b) { return ee + fma(a0, a, b); }, q.b, q.a, d);
                              }, rev);
}

// degree-0 in-place correction e += a_0 t, and a copy, over m values
template <class T>
__global__ void kb_acc0(long long m, const T* __restrict__ t, T* __restrict__ e, T a0)
{
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < m) e[i] = e[i] + a0 * t[i];
}
template <class T>
__global__ void kb_copy(long long m, const T* __restrict__ a, T* __restrict__ b)
{
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < m) b[i] = a[i];
}

template <class T>
__global__ void kb_smooth0(long long n, const T* __restrict__ t, const T* __restrict__ ec,
                           const int* __restrict__ W, T* __restrict__ ef, T a0, int k)
{
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * k) return;
    long long r = i / k;
    int q = int(i % k);
    int wc = W[r];
    ef[i] = (wc >= 0 ? ec[size_t(wc) * k + q] : T(0)) + a0 * t[i];
}

// Newton steps of the coarse polynomial (Sec. 2.3) for k right-hand sides
template <class T, int VEC, int KW, int PW>
__global__ void kb_newton_real(SellView<T> A, const T* __restrict__ rin, T* __restrict__ rout,
                               T* __restrict__ x, T inv, int first, int last, int k, int lg, int rev)
{
    using LN = Lanes<T, VEC, KW>;
    using VL = Vals<T, VEC, KW>;
    using V2 = Vals2<T, VEC, KW>;
    bfor_rows<T, VEC, KW, PW>(A, rin, k, lg, !last,
                              [&](int r, const LN& L) {
                                  return V2{bload(L, rin, r), bload(L, first ? (const T*)nullptr : (const T*)x, r)};
                              },
                              [&](int r, const LN& L, const VL& d, const V2& q) {
                                  bstore(L, x, r, [&](T a, T b) { return fma(a, inv, b); }, q.a, q.b);
                                  if (!last)
                                      bstore(L, rout, r, [&](T a, T b) { return a - b * inv; }, q.a, d);
                              }, rev);
}

template <class T, int VEC, int KW, int PW>
__global__ void kb_newton_pair1(SellView<T> A, const T* __restrict__ rin, T* __restrict__ t,
                                T* __restrict__ x, T two_a, T inv2, int first, int k, int lg, int rev)
{
    using LN = Lanes<T, VEC, KW>;
    using VL = Vals<T, VEC, KW>;
    using V2 = Vals2<T, VEC, KW>;
    bfor_rows<T, VEC, KW, PW>(A, rin, k, lg, true,
                              [&](int r, const LN& L) {
                                  return V2{bload(L, rin, r), bload(L, first ? (const T*)nullptr : (const T*)x, r)};
                              },
                              [&](int r, const LN& L, const VL& d, const V2& q) {
                                  bstore(L, t, r, [&](T a, T b) { return two_a * a - b; }, q.a, d);
                                  bstore(L, x, r, [&](T a, T b, T c) { return fma(two_a * a - b, inv2, c); }, q.a, d, q.b);
                              }, rev);
}

template <class T, int VEC, int KW, int PW>
__global__ void kb_newton_pair2(SellView<T> A, const T* __restrict__ rin, const T* __restrict__ t,
                                T* __restrict__ rout, T inv2, int k, int lg, int rev)
{
    using LN = Lanes<T, VEC, KW>;
    using VL = Vals<T, VEC, KW>;
    bfor_rows<T, VEC, KW, PW>(A, t, k, lg, true, [&](int r, const LN& L) { return bload(L, rin, r); },
                              [&](int r, const LN& L, const VL& d, const VL& ri) {
                                  bstore(L, rout, r, [&](T a, T b) { return a - b * inv2; }, ri, d);
                              }, rev);
}

__global__ void kb_d2f(long long m, const double* a, float* b)
{
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < m) b[i] = (float)a[i];
}
// [q][i] (caller: right-hand sides one after the other, natural order) <->
// [pos(i)][q] (batch: rows in nested order, right-hand sides adjacent), a
// transpose with a row permutation.  A block moves a tile of 32 rows x 32
// right-hand sides through shared memory so that both the reads and the
// writes are runs of 32 consecutive doubles.  Block: 32 x 8 threads; grid:
// (ceil(n/32), ceil(k/32)).
constexpr int TT = 32;
__global__ void __launch_bounds__(256)
kb_to_nested(long long n, int k, const int* pos, const double* a, double* b)
{
    __shared__ double tile[TT][TT + 1];
    const long long i0 = (long long)blockIdx.x * TT;
    const int q0 = blockIdx.y * TT;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int qq = ty; qq < TT; qq += 8) {              // read: consecutive i
        const long long i = i0 + tx;
        const int q = q0 + qq;
        if (i < n && q < k) tile[qq][tx] = a[size_t(q) * n + i];
    }
    __syncthreads();
    for (int ii = ty; ii < TT; ii += 8) {              // write: consecutive q
        const long long i = i0 + ii;
        const int q = q0 + tx;
        if (i < n && q < k) b[size_t(pos[i]) * k + q] = tile[tx][ii];
    }
}
__global__ void __launch_bounds__(256)
kb_from_nested(long long n, int k, const int* pos, const double* a, double* b)
{
    __shared__ double tile[TT][TT + 1];
    const long long i0 = (long long)blockIdx.x * TT;
    const int q0 = blockIdx.y * TT;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int ii = ty; ii < TT; ii += 8) {              // read: consecutive q
        const long long i = i0 + ii;
        const int q = q0 + tx;
        if (i < n && q < k) tile[tx][ii] = a[size_t(pos[i]) * k + q];
    }
    __syncthreads();
    for (int qq = ty; qq < TT; qq += 8) {              // write: consecutive i
        const long long i = i0 + tx;
        const int q = q0 + qq;
        if (i < n && q < k) b[size_t(q) * n + i] = tile[qq][tx];
    }
}

inline dim3 grid_tiles(long long n, int k) { return dim3(unsigned((n + TT - 1) / TT), unsigned((k + TT - 1) / TT)); }

// ----------------------------------------------------- batched Krylov work --
constexpr int RG = 608;   // reduction blocks

// out[i*k + q] = sum_r V_i[r][q] * w[r][q] for i < M, and out[M*k + q] =
// <w_q, w_q> when selfdot, compiled for the exact M; blocks write partial
// sums, the last block adds them in a fixed order.
template <int M>
__global__ void __launch_bounds__(BT)
kb_multidot(long long n, int k, const double* __restrict__ V, long long ldv, const double* __restrict__ w,
            double* __restrict__ part, double* __restrict__ out, unsigned* ticket, int selfdot)
{
    const int m = M + (selfdot ? 1 : 0);
    __shared__ double red[BT];
    __shared__ bool last_block;
    const int ng = BT / k;                 // row groups per block
    const int q = threadIdx.x % k, grp = threadIdx.x / k;
    double acc[M + 1];
#pragma unroll
    for (int i = 0; i < M + 1; ++i) acc[i] = 0.0;
    if (grp < ng) {
        for (long long r = (long long)blockIdx.x * ng + grp; r < n; r += (long long)gridDim.x * ng) {
            const long long t = r * k + q;
            const double wv = __ldg(w + t);
#pragma unroll
            for (int i = 0; i < M; ++i) acc[i] = fma(__ldg(V + i * ldv + t), wv, acc[i]);
            acc[M] = fma(wv, wv, acc[M]);
        }
    }
#pragma unroll
    for (int i = 0; i < M + 1; ++i) {
        if (i < m) {
            red[threadIdx.x] = grp < ng ? acc[i] : 0.0;
            __syncthreads();
            if (threadIdx.x < k) {
                double s = 0.0;
                for (int g = 0; g < ng; ++g) s += red[g * k + threadIdx.x];
                part[((long long)blockIdx.x * m + i) * k + threadIdx.x] = s;
            }
            __syncthreads();
        }
    }
    __threadfence();
    if (threadIdx.x == 0) last_block = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last_block) return;
    __threadfence();
    for (int o = threadIdx.x; o < m * k; o += blockDim.x) {
        double s = 0.0;
        for (int b = 0; b < (int)gridDim.x; ++b) s += part[(long long)b * m * k + o];
        out[o] = s;
    }
    if (threadIdx.x == 0) *ticket = 0u;
}

// w[r][q] -= sum_i h[i*k+q] V_i[r][q] (terms in the order i = 0, 1, ...),
// and out[q] = ||w_q||^2 of the result
template <int M>
__global__ void __launch_bounds__(BT)
kb_multiaxpy_norm(long long n, int k, const double* __restrict__ V, long long ldv, const double* __restrict__ h,
                  double* __restrict__ w, double* __restrict__ part, double* __restrict__ out, unsigned* ticket)
{
    __shared__ double red[BT];
    __shared__ bool last_block;
    const int ng = BT / k;
    const int q = threadIdx.x % k, grp = threadIdx.x / k;
    double c[M];
#pragma unroll
    for (int i = 0; i < M; ++i) c[i] = -h[i * k + q];
    double ss = 0.0;
    if (grp < ng) {
        for (long long r = (long long)blockIdx.x * ng + grp; r < n; r += (long long)gridDim.x * ng) {
            const long long t = r * k + q;
            double v[M];
#pragma unroll
            for (int i = 0; i < M; ++i) v[i] = __ldg(V + i * ldv + t);
            double s = w[t];
#pragma unroll
            for (int i = 0; i < M; ++i) s = fma(c[i], v[i], s);
            w[t] = s;
            ss = fma(s, s, ss);
        }
    }
    red[threadIdx.x] = grp < ng ? ss : 0.0;
    __syncthreads();
    if (threadIdx.x < k) {
        double s = 0.0;
        for (int g = 0; g < ng; ++g) s += red[g * k + threadIdx.x];
        part[(long long)blockIdx.x * k + threadIdx.x] = s;
    }
    __threadfence();
    if (threadIdx.x == 0) last_block = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last_block) return;
    __threadfence();
    for (int o = threadIdx.x; o < k; o += blockDim.x) {
        double s = 0.0;
        for (int b = 0; b < (int)gridDim.x; ++b) s += part[(long long)b * k + o];
        out[o] = s;
    }
    if (threadIdx.x == 0) *ticket = 0u;
}

// x[r][q] += sum_i y[i*k+q] Z_i[r][q] (terms in the order i = 0, 1, ...)
template <int M, class Z>
__global__ void kb_update(long long n, int k, const Z* __restrict__ Zs, long long ldz,
                          const double* __restrict__ y, double* __restrict__ x)
{
    long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * k) return;
    int q = int(t % k);
    double v[M];
#pragma unroll
    for (int i = 0; i < M; ++i) v[i] = wide<double>(__ldg(Zs + i * ldz + t));
    double s = x[t];
#pragma unroll
    for (int i = 0; i < M; ++i) s = fma(y[i * k + q], v[i], s);
    x[t] = s;
}

// v = w * inv, in FP32 as well where v32 is given (the V-cycle's input)
__global__ void kb_scale(long long n, int k, const double* __restrict__ w, const double* __restrict__ inv,
                         double* __restrict__ v, float* __restrict__ v32)
{
    long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * k) return;
    const double q = w[t] * inv[t % k];
    v[t] = q;
    if (v32) v32[t] = float(q);
}

__global__ void kb_sub(long long m, const double* b, const double* y, double* r)
{
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < m) r[i] = b[i] - y[i];
}

// Shape of a batch of k vectors of type T (Lanes): 16-byte packs where every
// row of k values starts on a 16-byte boundary, the smallest power of two of
// lanes that covers the packs, and KW steps of a whole warp beyond 32.
// `packs` false: FP64 batches of more than 32 take none.  There the lanes are
// all used without, and the registers of the packs' loads in flight (56 a
// thread against 32) cost warps: 64 right-hand sides on 2048^2 602 -> 535 ms,
// 32 as packs 306.  The top-level product of an FP32 V-cycle's vectors, which
// reads half the bytes, is faster with them (64 on 2048^2: 18.1 against 25.4
// ms a solve).
struct BShape {
    int vec, lg, kw;
};
template <class T>
BShape bshape(int k, bool packs)
{
    const int full = 16 / int(sizeof(T));
    BShape s{k % full == 0 && (packs || sizeof(T) == 4 || k <= 32) ? full : 1, 0, 1};
    const int n = k / s.vec;
    while (s.lg < 5 && (1 << s.lg) < n) ++s.lg;
    s.kw = n <= 32 ? 1 : (n <= 64 ? 2 : 4);
    return s;
}

// Runs the statement with VEC, KW and lg of a batch of k vectors of type T,
// and PW (warps per row: 1 for operators with short rows, 4 for long rows)
// of operator S.  PKW: the most steps that packs take (16-byte packs: at most
// 128 / 4 FP32 or, without `packs`, 32 / 2 FP64 lanes, one step).
#define WITH_SHAPE(T, PKW, bs, ...)                                                  \
    do {                                                                             \
        if ((bs).vec == 1) {                                                         \
            constexpr int VEC = 1;                                                   \
            if ((bs).kw == 1) { constexpr int KW = 1; __VA_ARGS__; }                 \
            else if ((bs).kw == 2) { constexpr int KW = 2; __VA_ARGS__; }            \
            else { constexpr int KW = 4; __VA_ARGS__; }                              \
        } else {                                                                     \
            constexpr int VEC = 16 / int(sizeof(T));                                 \
            if ((bs).kw == 1) { constexpr int KW = 1; __VA_ARGS__; }                 \
            else { constexpr int KW = PKW; __VA_ARGS__; }                            \
        }                                                                            \
    } while (0)
#define WITH_BATCH_SHAPE(T, PKW, bs, S, ...)                                         \
    do {                                                                             \
        const BShape bs_ = (bs);                                                     \
        const int lg = bs_.lg;                                                       \
        if ((S).pw == 1) { constexpr int PW = 1; WITH_SHAPE(T, PKW, bs_, __VA_ARGS__); } \
        else { constexpr int PW = 4; WITH_SHAPE(T, PKW, bs_, __VA_ARGS__); }         \
    } while (0)
#define WITH_BATCH(T, k, S, ...) WITH_BATCH_SHAPE(T, 1, bshape<T>(k, false), S, __VA_ARGS__)

}  // namespace

// Work space of one batch width k.
struct BatchData {
    int k = 0, m = 0;
    long long nk = 0;
    DBuf<double> V, Zs, w, bp, xp, r, part, hdev, inv;   // Zs: FP64 V-cycle
    DBuf<float> Zs32;                                    // FP32 V-cycle
    DBuf<double> rwork, t, wa, wb, cr0, cr1, ct, rcs;          // FP64 V-cycle
    DBuf<float> rwork32, vin32, t32, wa32, wb32, cr032, cr132, ct32, rcs32;  // FP32 V-cycle
    DBuf<unsigned> ticket;
    HBuf<double> hh;
    struct GEntry { const void* v; void* z; cudaGraphExec_t exec; long long kernels; };
    std::vector<GEntry> graphs;
    ~BatchData()
    {
        for (GEntry& g : graphs) cudaGraphExecDestroy(g.exec);
    }
};

namespace {

template <class T>
struct BWork {
    T* rwork; T* t; T* wa; T* wb; T* cr0; T* cr1; T* ct;
    T* rcs;    // saved C residuals, one slot per level l >= 1 (C-point smoothing)
};

template <class T>
const SolveLevelT<T>& bops(const SolveLevel& L);
template <>
const SolveLevelT<double>& bops<double>(const SolveLevel& L) { return L.d; }
template <>
const SolveLevelT<float>& bops<float>(const SolveLevel& L) { return L.f; }

template <class T>
const Sell<T>& bcoarse(const SolveData& S);
template <>
const Sell<double>& bcoarse<double>(const SolveData& S) { return S.Ac; }
template <>
const Sell<float>& bcoarse<float>(const SolveData& S) { return S.Ac32; }

// Prolongation and F-point smooth of level l for k right-hand sides (Eq. 6)
template <class T>
void bf_smooth(SolveData& S, int l, int k, const T* v, T* e, const BWork<T>& wk, cudaStream_t st)
{
    constexpr long long VB = sizeof(T);
    const long long kk = k;
    const SolveLevel& lv = *S.lv[l];
    const T* src = l == 0 ? v : wk.rwork;
    const SolveLevelT<T>& o = bops<T>(lv);
    const T* rf = src + size_t(lv.off) * k;
    const T* ec = e + size_t(lv.off + lv.n_f) * k;
    T* ef = e + size_t(lv.off) * k;
    const int nf = lv.n_f;
    const int p = int(lv.alpha.size()) - 1;
    const long long fB = (long long)nf * VB * kk;
    S.cur_level = l;
    LAUNCH_F(S, PK_FRESID, mat_bytes32(o.M) + (long long)lv.n_c * VB * kk + 3 * fB, (2 * o.M.nnz + 2LL * nf) * kk,
           WITH_BATCH(T, k, o.M, kb_fresid<T, VEC, KW, PW><<<grid_rows(nf, PW, lg), BT, 0, st>>>(view(o.M), rf, ec, wk.t, wk.wa,
                                                                    T(lv.alpha[p]), k, lg)));
    if (o.Ainv.n_rows) {
        // assembled smoother: e_f = W e_c + Ahat^-1 t (last Horner kernel, a0 = 0)
        LAUNCH_F(S, PK_HORNER, mat_bytes32(o.Ainv) + 4 * fB + 4LL * nf, (2 * o.Ainv.nnz + 3LL * nf) * kk,
                 WITH_BATCH(T, k, o.Ainv, kb_horner_last<T, VEC, KW, PW><<<grid_rows(nf, PW, lg), BT, 0, st>>>(view(o.Ainv), wk.t, wk.t, ec,
                                                                               lv.W.p, ef, T(0), k, lg, 0)));
        return;
    }
    if (p == 0) {
        LAUNCH_F(S, PK_HORNER, 3 * fB + 4LL * nf, 3LL * nf * kk,
               kb_smooth0<T><<<grid_for((long long)nf * k, BT), BT, 0, st>>>(nf, wk.t, ec, lv.W.p, ef,
                                                                            T(lv.alpha[0]), k));
        return;
    }
    const long long hB = mat_bytes32(o.Aff) + 3 * fB;
    T* win = wk.wa;
    T* wout = wk.wb;
    for (int kq = p - 1; kq >= 1; --kq) {
        LAUNCH_F(S, PK_HORNER, hB, (2 * o.Aff.nnz + 2LL * nf) * kk,
               WITH_BATCH(T, k, o.Aff, kb_horner<T, VEC, KW, PW><<<grid_rows(nf, PW, lg), BT, 0, st>>>(view(o.Aff), wk.t, win, wout,
                                                                        T(lv.alpha[kq]), k, lg, serpentine(p - 1 - kq))));
        std::swap(win, wout);
    }
    LAUNCH_F(S, PK_HORNER, hB + fB + 4LL * nf, (2 * o.Aff.nnz + 3LL * nf) * kk,
           WITH_BATCH(T, k, o.Aff, kb_horner_last<T, VEC, KW, PW><<<grid_rows(nf, PW, lg), BT, 0, st>>>(view(o.Aff), wk.t, win, ec,
                                                                         lv.W.p, ef, T(lv.alpha[0]), k, lg, serpentine(p - 1))));
}

// e += q(A) t by Horner for k right-hand sides, w = a_p t already in wk.wa
template <class T>
void bhorner_into(SolveData& S, const Sell<T>& A, const std::vector<double>& al, const BWork<T>& wk, T* e,
                  int n, int k, cudaStream_t st)
{
    constexpr long long VB = sizeof(T);
    const long long kk = k, fB = (long long)n * VB * kk;
    const int p = int(al.size()) - 1;
    if (p == 0) {
        LAUNCH_F(S, PK_HORNER, 3 * fB, 2LL * n * kk,
                 kb_acc0<T><<<grid_for((long long)n * k, BT), BT, 0, st>>>((long long)n * k, wk.t, e, T(al[0])));
        return;
    }
    const long long hB = mat_bytes32(A) + 3 * fB;
    T* win = wk.wa;
    T* wout = wk.wb;
    for (int kq = p - 1; kq >= 1; --kq) {
        LAUNCH_F(S, PK_HORNER, hB, (2 * A.nnz + 2LL * n) * kk,
                 WITH_BATCH(T, k, A, kb_horner<T, VEC, KW, PW><<<grid_rows(n, PW, lg), BT, 0, st>>>(view(A), wk.t, win, wout,
                                                                                      T(al[kq]), k, lg, serpentine(p - 1 - kq))));
        std::swap(win, wout);
    }
    LAUNCH_F(S, PK_HORNER, hB + fB, (2 * A.nnz + 3LL * n) * kk,
             WITH_BATCH(T, k, A, kb_horner_acc<T, VEC, KW, PW><<<grid_rows(n, PW, lg), BT, 0, st>>>(view(A), wk.t, win, e,
                                                                                      T(al[0]), k, lg, serpentine(p - 1))));
}

// C-point smooth of level l for k right-hand sides (Sec. 2):
// t_c = r_c - [A_cf A_cc] e_l, e_c += q_c(A_cc) t_c (or Ahat_cc^-1 t_c)
template <class T>
void bc_smooth(SolveData& S, int l, int k, const T* v, T* e, const BWork<T>& wk, cudaStream_t st)
{
    constexpr long long VB = sizeof(T);
    const long long kk = k;
    const SolveLevel& lv = *S.lv[l];
    const SolveLevelT<T>& o = bops<T>(lv);
    const int nc = lv.n_c;
    if (!nc) return;
    const T* rc = l == 0 ? v + size_t(lv.off + lv.n_f) * k : wk.rcs + size_t(lv.rc_off) * k;
    T* el = e + size_t(lv.off) * k;
    T* ec = el + size_t(lv.n_f) * k;
    const int p = int(lv.alpha_c.size()) - 1;
    const long long cB = (long long)nc * VB * kk;
    LAUNCH_F(S, PK_FRESID, mat_bytes32(o.Mc) + (long long)(lv.n_f + nc) * VB * kk + 3 * cB,
             (2 * o.Mc.nnz + 2LL * nc) * kk,
             WITH_BATCH(T, k, o.Mc, kb_fresid<T, VEC, KW, PW><<<grid_rows(nc, PW, lg), BT, 0, st>>>(view(o.Mc), rc, el, wk.t, wk.wa,
                                                                                   T(lv.alpha_c[p]), k, lg)));
    if (o.Ainvc.n_rows) {
        LAUNCH_F(S, PK_HORNER, mat_bytes32(o.Ainvc) + 4 * cB, (2 * o.Ainvc.nnz + 2LL * nc) * kk,
                 WITH_BATCH(T, k, o.Ainvc, kb_horner_acc<T, VEC, KW, PW><<<grid_rows(nc, PW, lg), BT, 0, st>>>(
                                           view(o.Ainvc), wk.t, wk.t, ec, T(0), k, lg, 0)));
        return;
    }
    bhorner_into<T>(S, o.Acc, lv.alpha_c, wk, ec, nc, k, st);
}

// second F-point smooth of FCF for k right-hand sides
template <class T>
void bf_smooth_again(SolveData& S, int l, int k, const T* v, T* e, const BWork<T>& wk, cudaStream_t st)
{
    constexpr long long VB = sizeof(T);
    const long long kk = k;
    const SolveLevel& lv = *S.lv[l];
    const SolveLevelT<T>& o = bops<T>(lv);
    const int nf = lv.n_f;
    if (!nf) return;
    const T* rf = (l == 0 ? v : wk.rwork) + size_t(lv.off) * k;
    T* el = e + size_t(lv.off) * k;
    const int p = int(lv.alpha.size()) - 1;
    const long long fB = (long long)nf * VB * kk;
    LAUNCH_F(S, PK_FRESID, mat_bytes32(o.Mf) + (long long)(nf + lv.n_c) * VB * kk + 3 * fB,
             (2 * o.Mf.nnz + 2LL * nf) * kk,
             WITH_BATCH(T, k, o.Mf, kb_fresid<T, VEC, KW, PW><<<grid_rows(nf, PW, lg), BT, 0, st>>>(view(o.Mf), rf, el, wk.t, wk.wa,
                                                                                   T(lv.alpha[p]), k, lg)));
    if (o.Ainv.n_rows) {
        LAUNCH_F(S, PK_HORNER, mat_bytes32(o.Ainv) + 4 * fB, (2 * o.Ainv.nnz + 2LL * nf) * kk,
                 WITH_BATCH(T, k, o.Ainv, kb_horner_acc<T, VEC, KW, PW><<<grid_rows(nf, PW, lg), BT, 0, st>>>(
                                          view(o.Ainv), wk.t, wk.t, el, T(0), k, lg, 0)));
        return;
    }
    bhorner_into<T>(S, o.Aff, lv.alpha, wk, el, nf, k, st);
}

// e = M^-1 v for k right-hand sides (nested order, [row][rhs])
template <class T>
void bvcycle(SolveData& S, int k, const T* v, T* e, const BWork<T>& wk, cudaStream_t st)
{
    const int L = S.nlev;
    constexpr long long VB = sizeof(T);
    const long long kk = k;
    for (int l = 0; l < L; ++l) {
        const SolveLevel& lv = *S.lv[l];
        const T* src = l == 0 ? v : wk.rwork;
        const Sell<T>& Z = bops<T>(lv).Z;
        const Sell<T, bf16s>& Zb = bops<T>(lv).Zb;
        S.cur_level = l;
        if (l > 0 && lv.n_c && S.smooth_type != AIRG_SMOOTH_F)   // restriction overwrites r_c in place
            LAUNCH_F(S, PK_RESTRICT, 2LL * lv.n_c * VB * kk, 0,
                     kb_copy<T><<<grid_for((long long)lv.n_c * k, BT), BT, 0, st>>>(
                         (long long)lv.n_c * k, src + size_t(lv.off + lv.n_f) * k, wk.rcs + size_t(lv.rc_off) * k));
        if (lv.n_c && Zb.val.n)
            LAUNCH_F(S, PK_RESTRICT, mat_bytes32(Zb) + (2LL * lv.n_c + lv.n_f + lv.n_c) * VB * kk,
                     (2 * Zb.nnz + lv.n_c) * kk,
                     WITH_BATCH(T, k, Zb, kb_restrict<T, VEC, KW, PW, bf16s><<<grid_rows(lv.n_c, PW, lg), BT, 0, st>>>(
                                    view(Zb), src + size_t(lv.off) * k, src + size_t(lv.off + lv.n_f) * k,
                                    wk.rwork + size_t(lv.off + lv.n_f) * k, k, lg)));
        else if (lv.n_c)
            LAUNCH_F(S, PK_RESTRICT, mat_bytes32(Z) + (2LL * lv.n_c + lv.n_f + lv.n_c) * VB * kk,
                     (2 * Z.nnz + lv.n_c) * kk,
                   WITH_BATCH(T, k, Z, kb_restrict<T, VEC, KW, PW><<<grid_rows(lv.n_c, PW, lg), BT, 0, st>>>(
                                  view(Z), src + size_t(lv.off) * k, src + size_t(lv.off + lv.n_f) * k,
                                  wk.rwork + size_t(lv.off + lv.n_f) * k, k, lg)));
    }
    {
        const T* rc = (L == 0 ? v : wk.rwork) + size_t(S.off_c) * k;
        T* x = e + size_t(S.off_c) * k;
        const Sell<T>& A = bcoarse<T>(S);
        SellView<T> Av = view(A);
        const int nco = S.n_coarse;
        const long long nB = (long long)nco * VB * kk, mB = mat_bytes32(A);
        S.cur_level = L;
        const T* rin = rc;
        T* bufs[2] = {wk.cr0, wk.cr1};
        int nb = 0;
        size_t nr = S.roots.size();
        int nsp = 0;   // SpMVs with the coarse operator so far (their direction alternates)
        for (size_t i = 0; i < nr; ++i) {
            bool last = i + 1 == nr;
            const Root& q = S.roots[i];
            T* rout = bufs[nb];
            if (q.im == 0.0) {
                LAUNCH_F(S, PK_NEWTON, (last ? 0 : mB + 2 * nB) + (i == 0 ? 2 : 3) * nB,
                         (last ? 2LL * nco : 2 * A.nnz + 4LL * nco) * kk,
                       WITH_BATCH(T, k, A, kb_newton_real<T, VEC, KW, PW><<<grid_rows(nco, PW, lg), BT, 0, st>>>(
                                      Av, rin, rout, x, T(1.0 / q.re), i == 0, last, k, lg, serpentine(nsp))));
                nsp += 1;
            } else {
                double mod2 = q.re * q.re + q.im * q.im;
                LAUNCH_F(S, PK_NEWTON, mB + (i == 0 ? 3 : 4) * nB, (2 * A.nnz + 4LL * nco) * kk,
                       WITH_BATCH(T, k, A, kb_newton_pair1<T, VEC, KW, PW><<<grid_rows(nco, PW, lg), BT, 0, st>>>(
                                      Av, rin, wk.ct, x, T(2.0 * q.re), T(1.0 / mod2), i == 0, k, lg, serpentine(nsp))));
                if (!last)
                    LAUNCH_F(S, PK_NEWTON, mB + 3 * nB, (2 * A.nnz + 2LL * nco) * kk,
                           WITH_BATCH(T, k, A, kb_newton_pair2<T, VEC, KW, PW><<<grid_rows(nco, PW, lg), BT, 0, st>>>(
                                          Av, rin, wk.ct, rout, T(1.0 / mod2), k, lg, serpentine(nsp + 1))));
                nsp += 2;
            }
            if (!last) { rin = rout; nb ^= 1; }
        }
        if (nr == 0) CK(cudaMemsetAsync(x, 0, sizeof(T) * size_t(nco) * k, st));
    }
    for (int l = L - 1; l >= 0; --l) {
        S.cur_level = l;
        bf_smooth<T>(S, l, k, v, e, wk, st);
        if (S.smooth_type != AIRG_SMOOTH_F) {
            bc_smooth<T>(S, l, k, v, e, wk, st);
            if (S.smooth_type == AIRG_SMOOTH_FCF) bf_smooth_again<T>(S, l, k, v, e, wk, st);
        }
    }
    S.close_run(st);
    S.cur_level = 0;
    CK_LAUNCH();
}

// z = M^-1 v: the FP64 V-cycle, or (z an FP32 vector) the FP32 one from
// vin32, which the kernel that formed the FP64 vector has filled
void bprecond_launch(Hierarchy& H, BatchData& B, const double* v, double* z, cudaStream_t st)
{
    BWork<double> wk{B.rwork.p, B.t.p, B.wa.p, B.wb.p, B.cr0.p, B.cr1.p, B.ct.p, B.rcs.p};
    bvcycle<double>(*H.solve, B.k, v, z, wk, st);
}
void bprecond_launch(Hierarchy& H, BatchData& B, const float* v, float* z, cudaStream_t st)
{
    BWork<float> wk{B.rwork32.p, B.t32.p, B.wa32.p, B.wb32.p, B.cr032.p, B.cr132.p, B.ct32.p, B.rcs32.p};
    bvcycle<float>(*H.solve, B.k, v, z, wk, st);
}

template <class T>
void bprecond(Hierarchy& H, BatchData& B, const T* v, T* z, cudaStream_t st)
{
    SolveData& S = *H.solve;
    if (S.prof || !S.use_graphs) {
        bprecond_launch(H, B, v, z, st);
        return;
    }
    BatchData::GEntry* ge = nullptr;
    for (auto& g : B.graphs)
        if (g.v == v && g.z == z) { ge = &g; break; }
    if (ge) {
        CK(cudaGraphLaunch(ge->exec, st));
        S.launches += ge->kernels;
        return;
    }
    // first use: launched directly, and captured while the kernels run
    bprecond_launch(H, B, v, z, st);
    const long long before = S.launches;
    CK(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal));
    try {
        bprecond_launch(H, B, v, z, st);
    } catch (...) {
        cudaGraph_t g0;
        cudaStreamEndCapture(st, &g0);
        if (g0) cudaGraphDestroy(g0);
        throw;
    }
    cudaGraph_t graph;
    CK(cudaStreamEndCapture(st, &graph));
    cudaGraphExec_t exec;
    cudaError_t e = cudaGraphInstantiate(&exec, graph, 0);
    cudaGraphDestroy(graph);
    CK(e);
    B.graphs.push_back(BatchData::GEntry{v, z, exec, S.launches - before});
    S.launches = before;
}

void ensure_batch(Hierarchy& H, int k)
{
    SolveData& S = *H.solve;
    if (S.batch && S.batch->k == k) return;
    S.batch.reset();
    auto B = std::make_shared<BatchData>();
    B->k = k;
    B->m = std::min(std::max(1, H.opt.gmres_restart), MAXB);
    long long n = S.n0;
    B->nk = n * k;
    size_t nk = size_t(B->nk);
    int m = B->m;
    B->V.alloc(size_t(m + 1) * nk);
    if (mixed_precision(H.opt)) B->Zs32.alloc(size_t(m) * nk);
    else B->Zs.alloc(size_t(m) * nk);
    B->w.alloc(nk); B->bp.alloc(nk); B->xp.alloc(nk); B->r.alloc(nk);
    B->part.alloc(size_t(RG) * (MAXB + 1) * k);
    B->hdev.alloc(size_t(3 * (MAXB + 2)) * k);
    B->inv.alloc(size_t(k));
    B->hh.alloc(size_t(3 * (MAXB + 2)) * k);
    B->ticket.alloc(1);
    CK(cudaMemset(B->ticket.p, 0, sizeof(unsigned)));
    size_t nf = size_t(std::max({S.max_nf, S.max_nc, 1})) * k, nc = size_t(std::max(S.n_coarse, 1)) * k;
    const size_t nrc = S.smooth_type != AIRG_SMOOTH_F ? size_t(std::max<long long>(S.rc_total, 1)) * k : 0;
    if (mixed_precision(H.opt)) {
        B->rwork32.alloc(nk); B->vin32.alloc(nk);
        B->t32.alloc(nf); B->wa32.alloc(nf); B->wb32.alloc(nf);
        B->cr032.alloc(nc); B->cr132.alloc(nc); B->ct32.alloc(nc);
        if (nrc) B->rcs32.alloc(nrc);
    } else {
        B->rwork.alloc(nk);
        B->t.alloc(nf); B->wa.alloc(nf); B->wb.alloc(nf);
        B->cr0.alloc(nc); B->cr1.alloc(nc); B->ct.alloc(nc);
        if (nrc) B->rcs.alloc(nrc);
    }
    S.batch = B;
}

// per-RHS 2-norms of a batch
void bnorms(SolveData& S, BatchData& B, const double* x, std::vector<double>& out, cudaStream_t st)
{
    long long n = S.n0;
    int k = B.k;
    LAUNCH_F(S, PK_KRYLOV, 8 * B.nk, 2 * B.nk,
           kb_multidot<1><<<RG, BT, 0, st>>>(n, k, x, B.nk, x, B.part.p, B.hdev.p, B.ticket.p, 0));
    out.resize(k);
    d2h(out.data(), B.hdev.p, size_t(k), st);
    for (double& v : out) v = std::sqrt(std::max(v, 0.0));
}

}  // namespace

// Lockstep FGMRES(m) for k right-hand sides (device b, x in the caller's
// layout: k vectors of length n one after the other).
void solve_batched(Hierarchy& H, int k, const double* b, double* x, double rtol, double atol,
                   int maxit, airg_solve_info& info, cudaStream_t st)
{
    SolveData& S = *H.solve;
    ensure_batch(H, k);
    BatchData& B = *S.batch;
    const long long n = S.n0, nk = B.nk;
    const int m = B.m;
    const int g = grid_for(nk, BT);
    SellView<double> A = view(S.Atop);
    const long long topB = mat_bytes32(S.Atop) + 16 * nk;
    const bool mixed = mixed_precision(H.opt);
    float* v32 = mixed ? B.vin32.p : nullptr;
    const long long scaleB = (mixed ? 20 : 16) * nk;
    LAUNCH(S, PK_LAYOUT, 20 * nk, kb_to_nested<<<grid_tiles(n, k), 256, 0, st>>>(n, k, S.pos0.p, b, B.bp.p));
    LAUNCH(S, PK_LAYOUT, 20 * nk, kb_to_nested<<<grid_tiles(n, k), 256, 0, st>>>(n, k, S.pos0.p, x, B.xp.p));
    std::vector<double> bn, rn, tol(k);
    bnorms(S, B, B.bp.p, bn, st);
    for (int q = 0; q < k; ++q) tol[q] = std::max(rtol * bn[q], atol);
    auto residual = [&]() {
        LAUNCH_F(S, PK_TOPSPMV, topB, 2 * S.Atop.nnz * k,
               WITH_BATCH(double, k, S.Atop, kb_spmv<double, VEC, KW, PW, double><<<grid_rows(n, PW, lg), BT, 0, st>>>(A, B.xp.p, B.w.p, k, lg)));
        LAUNCH_F(S, PK_KRYLOV, 24 * nk, nk, kb_sub<<<g, BT, 0, st>>>(nk, B.bp.p, B.w.p, B.r.p));
        bnorms(S, B, B.r.p, rn, st);
    };
    residual();
    int its = 0;
    if (H.opt.outer == AIRG_OUTER_RICHARDSON) {
        // lockstep Richardson: x_q += M^-1 r_q for every unconverged q
        std::vector<double> yq(k);
        while (its < maxit) {
            int nact = 0;
            for (int q = 0; q < k; ++q) {
                yq[q] = rn[q] > tol[q] ? 1.0 : 0.0;
                nact += rn[q] > tol[q];
            }
            if (!nact) break;
            h2d(B.hdev.p, yq.data(), size_t(k), st);
            if (mixed) {
                LAUNCH(S, PK_LAYOUT, 12 * nk, kb_d2f<<<g, BT, 0, st>>>(nk, B.r.p, B.vin32.p));
                bprecond(H, B, (const float*)B.vin32.p, B.Zs32.p, st);
                LAUNCH_F(S, PK_KRYLOV, 20 * nk, 2 * nk, kb_update<1, float><<<g, BT, 0, st>>>(n, k, B.Zs32.p, nk, B.hdev.p, B.xp.p));
            } else {
                bprecond(H, B, (const double*)B.r.p, B.Zs.p, st);
                LAUNCH_F(S, PK_KRYLOV, 24 * nk, 2 * nk, kb_update<1, double><<<g, BT, 0, st>>>(n, k, B.Zs.p, nk, B.hdev.p, B.xp.p));
            }
            residual();
            ++its;
        }
    }
    std::vector<double> Hm(size_t(m + 1) * m * k), cs(size_t(m) * k), sn(size_t(m) * k),
        gv(size_t(m + 1) * k), Y(size_t(m) * k), inv(k);
    std::vector<int> active(k), jdone(k);
    auto hq = [&](int i, int j, int q) -> double& { return Hm[(size_t(i) * m + j) * k + q]; };
    double* hh = B.hh.p;
    while (H.opt.outer == AIRG_OUTER_FGMRES && its < maxit) {
        int nact = 0;
        for (int q = 0; q < k; ++q) {
            active[q] = rn[q] > tol[q];
            nact += active[q];
            jdone[q] = 0;
            inv[q] = active[q] ? 1.0 / rn[q] : 0.0;
        }
        if (!nact) break;
        std::fill(gv.begin(), gv.end(), 0.0);
        for (int q = 0; q < k; ++q) gv[q] = rn[q];
        h2d(B.inv.p, inv.data(), size_t(k), st);
        LAUNCH_F(S, PK_KRYLOV, scaleB, nk, kb_scale<<<g, BT, 0, st>>>(n, k, B.r.p, B.inv.p, B.V.p, v32));
        for (int j = 0; j < m; ++j) {
            double* vj = B.V.p + size_t(j) * nk;
            if (mixed) {
                float* zj = B.Zs32.p + size_t(j) * nk;
                bprecond(H, B, (const float*)B.vin32.p, zj, st);
                LAUNCH_F(S, PK_TOPSPMV, topB - 4 * nk, 2 * S.Atop.nnz * k,
                       WITH_BATCH_SHAPE(double, 2, bshape<double>(k, true), S.Atop, kb_spmv<double, VEC, KW, PW, float><<<grid_rows(n, PW, lg), BT, 0, st>>>(A, zj, B.w.p, k, lg)));
            } else {
                double* zj = B.Zs.p + size_t(j) * nk;
                bprecond(H, B, (const double*)vj, zj, st);
                LAUNCH_F(S, PK_TOPSPMV, topB, 2 * S.Atop.nnz * k,
                       WITH_BATCH(double, k, S.Atop, kb_spmv<double, VEC, KW, PW, double><<<grid_rows(n, PW, lg), BT, 0, st>>>(A, zj, B.w.p, k, lg)));
            }
            // CGS with a second pass only if the first cancelled, for some
            // active right-hand side, more than reorth_ratio() allows
            double* h1 = B.hdev.p;
            double* h2 = B.hdev.p + size_t(MAXB + 2) * k;
            double* hnp = B.hdev.p + size_t(2) * (MAXB + 2) * k;
            LAUNCH_F(S, PK_KRYLOV, 8LL * nk * (j + 2), 2LL * nk * (j + 2),
                   WITH_M(j + 1, kb_multidot<MM><<<RG, BT, 0, st>>>(n, k, B.V.p, nk, B.w.p, B.part.p, h1,
                                                                     B.ticket.p, 1)));
            LAUNCH_F(S, PK_KRYLOV, 8LL * nk * (j + 3), 2LL * nk * (j + 2),
                   WITH_M(j + 1, kb_multiaxpy_norm<MM><<<RG, BT, 0, st>>>(n, k, B.V.p, nk, h1, B.w.p, B.part.p,
                                                                           hnp, B.ticket.p)));
            CK(cudaMemcpyAsync(hh, B.hdev.p, sizeof(double) * 3 * (MAXB + 2) * k, cudaMemcpyDeviceToHost, st));
            CK(cudaStreamSynchronize(st));
            bool again = false;
            const double ro = reorth_ratio();
            for (int q = 0; q < k; ++q)
                if (active[q] && hh[size_t(2) * (MAXB + 2) * k + q] < ro * hh[size_t(j + 1) * k + q]) again = true;
            for (int q = 0; q < k; ++q)
                for (int i = 0; i <= j; ++i) hq(i, j, q) = hh[size_t(i) * k + q];
            if (again) {
                LAUNCH_F(S, PK_KRYLOV, 8LL * nk * (j + 2), 2LL * nk * (j + 1),
                       WITH_M(j + 1, kb_multidot<MM><<<RG, BT, 0, st>>>(n, k, B.V.p, nk, B.w.p, B.part.p, h2,
                                                                         B.ticket.p, 0)));
                LAUNCH_F(S, PK_KRYLOV, 8LL * nk * (j + 3), 2LL * nk * (j + 2),
                       WITH_M(j + 1, kb_multiaxpy_norm<MM><<<RG, BT, 0, st>>>(n, k, B.V.p, nk, h2, B.w.p, B.part.p,
                                                                               hnp, B.ticket.p)));
                CK(cudaMemcpyAsync(hh, B.hdev.p, sizeof(double) * 3 * (MAXB + 2) * k, cudaMemcpyDeviceToHost, st));
                CK(cudaStreamSynchronize(st));
                for (int q = 0; q < k; ++q)
                    for (int i = 0; i <= j; ++i) hq(i, j, q) += hh[(size_t(MAXB + 2) + i) * k + q];
            }
            ++its;
            int still = 0;
            for (int q = 0; q < k; ++q) {
                inv[q] = 0.0;
                if (!active[q]) continue;
                double hn = std::sqrt(std::max(hh[size_t(2) * (MAXB + 2) * k + q], 0.0));
                hq(j + 1, j, q) = hn;
                for (int i = 0; i < j; ++i) {
                    double a = hq(i, j, q), c = hq(i + 1, j, q);
                    hq(i, j, q) = cs[size_t(i) * k + q] * a + sn[size_t(i) * k + q] * c;
                    hq(i + 1, j, q) = -sn[size_t(i) * k + q] * a + cs[size_t(i) * k + q] * c;
                }
                double a = hq(j, j, q), c = hq(j + 1, j, q);
                double den = std::hypot(a, c);
                cs[size_t(j) * k + q] = den > 0 ? a / den : 1.0;
                sn[size_t(j) * k + q] = den > 0 ? c / den : 0.0;
                hq(j, j, q) = den;
                hq(j + 1, j, q) = 0.0;
                gv[size_t(j + 1) * k + q] = -sn[size_t(j) * k + q] * gv[size_t(j) * k + q];
                gv[size_t(j) * k + q] = cs[size_t(j) * k + q] * gv[size_t(j) * k + q];
                jdone[q] = j + 1;
                if (std::fabs(gv[size_t(j + 1) * k + q]) <= tol[q] || den == 0.0 || hn == 0.0) {
                    active[q] = 0;
                } else {
                    inv[q] = 1.0 / hn;
                    ++still;
                }
            }
            if (!still || its >= maxit || j + 1 == m) break;
            h2d(B.inv.p, inv.data(), size_t(k), st);
            LAUNCH_F(S, PK_KRYLOV, scaleB, nk,
                   kb_scale<<<g, BT, 0, st>>>(n, k, B.w.p, B.inv.p, B.V.p + size_t(j + 1) * nk, v32));
        }
        // least squares per right-hand side, zero-padded to the common width
        int jmax = 0;
        std::fill(Y.begin(), Y.end(), 0.0);
        for (int q = 0; q < k; ++q) {
            int jd = jdone[q];
            jmax = std::max(jmax, jd);
            for (int j = jd - 1; j >= 0; --j) {
                double s = gv[size_t(j) * k + q];
                for (int i = j + 1; i < jd; ++i) s -= hq(j, i, q) * Y[size_t(i) * k + q];
                Y[size_t(j) * k + q] = s / hq(j, j, q);
            }
        }
        if (jmax) {
            h2d(B.hdev.p, Y.data(), size_t(jmax) * k, st);
            if (mixed)
                LAUNCH_F(S, PK_KRYLOV, 4LL * nk * (jmax + 4), 2LL * nk * jmax,
                       WITH_M(jmax, kb_update<MM, float><<<g, BT, 0, st>>>(n, k, B.Zs32.p, nk, B.hdev.p, B.xp.p)));
            else
                LAUNCH_F(S, PK_KRYLOV, 8LL * nk * (jmax + 2), 2LL * nk * jmax,
                       WITH_M(jmax, kb_update<MM, double><<<g, BT, 0, st>>>(n, k, B.Zs.p, nk, B.hdev.p, B.xp.p)));
        }
        residual();
    }
    int conv = 1;
    double worst = 0.0;
    for (int q = 0; q < k; ++q) {
        double rel = bn[q] > 0 ? rn[q] / bn[q] : 0.0;
        worst = std::max(worst, rel);
        if (rn[q] > tol[q]) conv = 0;
    }
    LAUNCH(S, PK_LAYOUT, 20 * nk, kb_from_nested<<<grid_tiles(n, k), 256, 0, st>>>(n, k, S.pos0.p, B.xp.p, x));
    CK_LAUNCH();
    info.iterations = std::max(info.iterations, its);
    info.rel_residual = std::max(info.rel_residual, worst);
    info.converged = info.converged && conv;
}

int batch_max_width() { return MAXK; }

}  // namespace airg
