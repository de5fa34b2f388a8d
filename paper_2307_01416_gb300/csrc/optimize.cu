// Robust spot-weight optimisation over the scenarios' influence matrices
// (Sec. 2.E: robust optimisation over 13 scenarios against the target
// constraints of Table 3).  The paper's optimiser is an in-house
// trial-and-error procedure; the objective here is a worst case over the
// scenarios of quadratic target under- and overdose and ring-overdose
// penalties, minimised by Adam with non-negative weights.
//
// Only target and ring voxels enter the objective and its gradient, so one
// setup pass per call copies those rows of every scenario into a compact CSR
// (16-bit spot indices, rows padded to 8 entries: one 16-byte load of
// columns and two of values per lane and step).  Each iteration then runs,
// with no host synchronisation:
//   k_fwd         d_s = A_s x on the compact rows of every scenario (a warp
//                 per row, eight lanes for short rows), the scenario's
//                 objective f_s (compensated sums per block, FP64 over the
//                 blocks) and max_i |f'(d_i)|;
//   k_bwd_fixed   s* = first s with the largest f_s (every block), recorded;
//                 g = A_s*^T f'(d_s*) over the compact rows (a warp per row)
//                 as 64-bit fixed-point sums: shared-memory atomics per
//                 block, one global atomic per spot and block;
//   k_adam_fixed  g_j back to floating point, then the Adam step on x_j,
//                 clamped at zero.
// Integer sums do not depend on the order of the adds, so repeated calls
// give the same bits.  The iteration is HBM-bound.  Full-matrix products
// (dose of the weights, target indices over all voxels) use k_spmv: a
// sub-warp per row of the caller's CSR.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "vpmc_internal.cuh"

namespace vpmc {
namespace {

constexpr unsigned kFullMask = 0xffffffffu;
constexpr int kLanesPerRow = 8;                 // full-matrix products: 4 rows per warp
constexpr int kSpmvBlocks = 16;                 // full-matrix products: blocks per SM and matrix

struct Csr {
    const long long* row_ptr;
    const int* col;
    const float* val;
};

struct ObjParams {
    float dp, w_u, w_o, w_r, over, ring;       // prescription and weights
    float inv_nt, inv_nr;                       // 1 / |T|, 1 / |R|
};

__device__ __forceinline__ float obj_term(float d, unsigned char c, const ObjParams& q)
{
    if (c == 1) {
        const float u = fmaxf(q.dp - d, 0.0f), o = fmaxf(d - q.over * q.dp, 0.0f);
        return q.inv_nt * (q.w_u * u * u + q.w_o * o * o);
    }
    if (c == 2) {
        const float r = fmaxf(d - q.ring * q.dp, 0.0f);
        return q.inv_nr * q.w_r * r * r;
    }
    return 0.0f;
}

__device__ __forceinline__ float obj_grad(float d, unsigned char c, const ObjParams& q)
{
    if (c == 1) {
        const float u = fmaxf(q.dp - d, 0.0f), o = fmaxf(d - q.over * q.dp, 0.0f);
        return 2.0f * q.inv_nt * (q.w_o * o - q.w_u * u);
    }
    if (c == 2) return 2.0f * q.inv_nr * q.w_r * fmaxf(d - q.ring * q.dp, 0.0f);
    return 0.0f;
}

struct CsrSet {
    Csr m[kMaxScen];
};

// Per scenario: [count(d >= D_p in T), count(T), count(d >= D_p)], and as FP32
// bit patterns of non-negative doses (which order as integers) max_T d and
// kMaxBits - min_T d, so that all five start at zero.
constexpr int kMaxBits = 0x7f7fffff;
struct IndexSums {
    unsigned long long hit, target, high;
    int neg_min, max;
};

// d = A x of one matrix (kIndices false) or the target indices of every
// scenario's dose (grid.y) without storing the doses.  A sub-warp of
// kLanesPerRow lanes per row, each summing every kLanesPerRow-th entry in
// order.  HBM-bound (8 bytes an entry): kBatch loads of columns and values are
// in flight per lane, and the next row's pointers are read before this row's
// entries are used, since most rows are shorter than one batch of the
// sub-warp and the chain pointers -> entries -> weights would be their time.
// 13 matrices of 6.4e7 entries: 3.1 ms with one entry per lane in flight,
// 1.63 ms with eight and an even number of warps, 1.36 ms with an odd one (one
// matrix 172 -> 140 us).  Batches of 4, 6, 12, 16: 1.88, 1.74, 1.48, 1.71 ms;
// the weights staged in shared memory (two blocks of 512 threads per SM) 1.69;
// a warp on each row of more than 32 entries 2.6.
constexpr int kBatch = 8;
template <bool kIndices>
__global__ void __launch_bounds__(256) k_spmv(const __grid_constant__ CsrSet mats, long long n_rows, int n_cols,
                                              const float* __restrict__ x, const unsigned char* __restrict__ cls,
                                              float dp, float* __restrict__ dose, IndexSums* __restrict__ sums)
{
    const Csr A = mats.m[blockIdx.y];
    const int lane = threadIdx.x & 31, sub = lane & (kLanesPerRow - 1);
    constexpr int kRowsPerWarp = 32 / kLanesPerRow;
    // an odd number of warps: rows of one phase of a grid whose width is a power
    // of two times 4 are all inside the field or all empty
    const long long wstride = (((long long)gridDim.x * (blockDim.x >> 5) - 1) | 1) * kRowsPerWarp;
    unsigned hit = 0, target = 0, high = 0;
    int mn = kMaxBits, mx = 0;
    // warp-uniform loop over groups of kRowsPerWarp rows (the shuffles below
    // need every lane of the warp in every iteration)
    long long base = ((long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * kRowsPerWarp;
    long long b = 0, e = 0;
    auto row_bounds = [&](long long row) {
        b = e = 0;
        if (row < n_rows) {
            b = __ldg(A.row_ptr + row);
            e = __ldg(A.row_ptr + row + 1);
        }
    };
    if (base >= wstride) base = n_rows;                // (the warp too many)
    row_bounds(base + lane / kLanesPerRow);
    for (; base < n_rows; base += wstride) {
        const long long row = base + lane / kLanesPerRow;
        long long k = b + sub;
        const long long end = e;
        row_bounds(row + wstride);
        const unsigned char c = kIndices && row < n_rows ? __ldg(cls + row) : 0;
        float acc = 0.0f;
        for (; k < end; k += kBatch * kLanesPerRow) {
            int j[kBatch];
            float v[kBatch], xj[kBatch];
#pragma unroll
            for (int u = 0; u < kBatch; ++u) {
                const bool in = k + u * kLanesPerRow < end;
                j[u] = in ? __ldcs(A.col + k + u * kLanesPerRow) : -1;
                v[u] = in ? __ldcs(A.val + k + u * kLanesPerRow) : 0.0f;
            }
#pragma unroll
            for (int u = 0; u < kBatch; ++u) xj[u] = (unsigned)j[u] < (unsigned)n_cols ? __ldg(x + j[u]) : 0.0f;
#pragma unroll
            for (int u = 0; u < kBatch; ++u)
                if ((unsigned)j[u] < (unsigned)n_cols) acc = fmaf(v[u], xj[u], acc);
        }
#pragma unroll
        for (int o = kLanesPerRow / 2; o >= 1; o >>= 1) acc += __shfl_xor_sync(kFullMask, acc, o);
        if (sub == 0 && row < n_rows) {
            if (kIndices) {
                const float d = fmaxf(acc, 0.0f);
                const bool t = c == 1, hi = d >= dp;
                hit += (t && hi) ? 1u : 0u;
                target += t ? 1u : 0u;
                high += hi ? 1u : 0u;
                if (t) {
                    mn = min(mn, __float_as_int(d));
                    mx = max(mx, __float_as_int(d));
                }
            } else {
                dose[row] = acc;
            }
        }
    }
    if (kIndices) {
        hit = __reduce_add_sync(kFullMask, hit);
        target = __reduce_add_sync(kFullMask, target);
        high = __reduce_add_sync(kFullMask, high);
        mn = __reduce_min_sync(kFullMask, mn);
        mx = __reduce_max_sync(kFullMask, mx);
        if (lane == 0) {
            IndexSums& r = sums[blockIdx.y];
            if (hit) atomicAdd(&r.hit, (unsigned long long)hit);
            if (target) atomicAdd(&r.target, (unsigned long long)target);
            if (high) atomicAdd(&r.high, (unsigned long long)high);
            if (mn < kMaxBits) atomicMax(&r.neg_min, kMaxBits - mn);
            if (mx > 0) atomicMax(&r.max, mx);
        }
    }
}

constexpr int kPadRow = 8;                      // compact CSR row padding (entries)
constexpr size_t kBwdSmemMax = 227 * 1024;      // shared memory of one gradient block

// ---- target and ring rows, in voxel order ----
constexpr int kClsThreads = 256, kClsPer = 16;  // voxels of one block: 4096

struct ClassTotals {
    unsigned long long target, ring;
};

__device__ __forceinline__ int class_voxels(const unsigned char* __restrict__ cls, long long n_rows, long long v0,
                                            unsigned char (&c)[kClsPer])
{
    int n = 0;
#pragma unroll
    for (int i = 0; i < kClsPer; ++i) {
        c[i] = v0 + i < n_rows ? __ldg(cls + v0 + i) : 0;
        n += c[i] == 1 || c[i] == 2;
    }
    return n;
}

// Target and ring voxels per block of 4096, and both totals.
__global__ void __launch_bounds__(kClsThreads) k_cls_count(const unsigned char* __restrict__ cls, long long n_rows,
                                                           long long* __restrict__ counts, ClassTotals* __restrict__ totals)
{
    __shared__ unsigned s_n, s_t;
    if (threadIdx.x == 0) s_n = s_t = 0u;
    __syncthreads();
    unsigned char c[kClsPer];
    const unsigned n = (unsigned)class_voxels(cls, n_rows, ((long long)blockIdx.x * kClsThreads + threadIdx.x) * kClsPer, c);
    unsigned t = 0;
#pragma unroll
    for (int i = 0; i < kClsPer; ++i) t += c[i] == 1;
    const unsigned wn = __reduce_add_sync(kFullMask, n), wt = __reduce_add_sync(kFullMask, t);
    if ((threadIdx.x & 31) == 0 && wn) {
        atomicAdd(&s_n, wn);
        atomicAdd(&s_t, wt);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        counts[blockIdx.x] = s_n;
        if (s_t) atomicAdd(&totals->target, (unsigned long long)s_t);
        if (s_n > s_t) atomicAdd(&totals->ring, (unsigned long long)(s_n - s_t));
    }
}

// Their voxel numbers and classes, at the blocks' offsets.
__global__ void __launch_bounds__(kClsThreads) k_cls_rows(const unsigned char* __restrict__ cls, long long n_rows,
                                                          const long long* __restrict__ offset, int* __restrict__ tr_rows,
                                                          unsigned char* __restrict__ tr_cls)
{
    __shared__ int s_w[kClsThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long v0 = ((long long)blockIdx.x * kClsThreads + threadIdx.x) * kClsPer;
    unsigned char c[kClsPer];
    const int n = class_voxels(cls, n_rows, v0, c);
    int inc = n;
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(kFullMask, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) s_w[warp] = inc;
    __syncthreads();
    long long pos = offset[blockIdx.x] + inc - n;
    for (int w = 0; w < warp; ++w) pos += s_w[w];
#pragma unroll
    for (int i = 0; i < kClsPer; ++i)
        if (c[i] == 1 || c[i] == 2) {
            tr_rows[pos] = (int)(v0 + i);
            tr_cls[pos] = c[i];
            ++pos;
        }
}

// plen[s (n_tr + 1) + i] = padded entries of target/ring row i in scenario s
// (0 at i = n_tr); nnz[s] its entries, longest the longest padded row.
__global__ void k_tr_len(const __grid_constant__ CsrSet mats, const int* __restrict__ tr_rows, int n_tr,
                         long long* __restrict__ plen, unsigned long long* __restrict__ nnz,
                         unsigned long long* __restrict__ longest)
{
    const int s = blockIdx.y;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    long long l = 0;
    if (i < n_tr) {
        const long long* rp = mats.m[s].row_ptr;
        const int r = __ldg(tr_rows + i);
        l = __ldg(rp + r + 1) - __ldg(rp + r);
    }
    const long long p = (l + kPadRow - 1) / kPadRow * kPadRow;
    if (i <= n_tr) plen[(long long)s * (n_tr + 1) + i] = p;
    long long sum = l, mx = p;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        sum += __shfl_xor_sync(kFullMask, sum, o);
        mx = max(mx, __shfl_xor_sync(kFullMask, mx, o));
    }
    if ((threadIdx.x & 31) == 0 && sum > 0) {
        atomicAdd(nnz + s, (unsigned long long)sum);
        atomicMax(longest, (unsigned long long)mx);
    }
}

// Copies the target/ring rows into the compact CSR: a warp per row and
// scenario; pads and entries with an out-of-range spot become (0, 0.0).
// Sets *unordered if a row's spot indices are not strictly increasing (a
// row may then repeat a spot).  HBM-bound (14 bytes an entry): four loads of
// columns and values in flight per lane, a lane's predecessor from its
// neighbour.
__global__ void __launch_bounds__(256) k_tr_gather(const __grid_constant__ CsrSet mats, const int* __restrict__ tr_rows,
                                                   int n_tr, int n_cols, const long long* __restrict__ crp,
                                                   unsigned short* __restrict__ ccol, float* __restrict__ cval,
                                                   int* __restrict__ unordered, unsigned* __restrict__ max_abs)
{
    constexpr int kU = 4;
    const int s = blockIdx.y, lane = threadIdx.x & 31;
    const int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (i >= n_tr) return;                            // warp-uniform
    const Csr A = mats.m[s];
    const int row = __ldg(tr_rows + i);
    const long long b = __ldg(A.row_ptr + row), len = __ldg(A.row_ptr + row + 1) - b;
    const long long dst = crp[(long long)s * (n_tr + 1) + i];
    const long long plen = crp[(long long)s * (n_tr + 1) + i + 1] - dst;
    unsigned amax = 0u;                               // |a| as bits: non-negative floats order as integers
    int before = -1;                                  // the column before this pass's first
    bool bad = false;
    for (long long k0 = 0; k0 < plen; k0 += 32 * kU) {
        int j[kU];
        float v[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const long long k = k0 + 32 * u + lane;
            j[u] = k < len ? __ldcs(A.col + b + k) : 0x7fffffff;
            v[u] = k < len ? __ldcs(A.val + b + k) : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const long long k = k0 + 32 * u + lane;
            int prev = __shfl_up_sync(kFullMask, j[u], 1);
            if (lane == 0) prev = before;
            before = __shfl_sync(kFullMask, j[u], 31);
            bad |= k > 0 && k < len && j[u] <= prev;
            if ((unsigned)j[u] >= (unsigned)n_cols) {
                j[u] = 0;
                v[u] = 0.0f;
            }
            if (k < plen) {
                ccol[dst + k] = (unsigned short)j[u];
                cval[dst + k] = v[u];
            }
            amax = max(amax, __float_as_uint(fabsf(v[u])));
        }
    }
    if (bad) *unordered = 1;
    amax = __reduce_max_sync(kFullMask, amax);
    if (lane == 0 && amax) atomicMax(max_abs + s, amax);
}

// Entries of one spot over the compact rows, at most: the row count, or the
// entry count when a row may repeat a spot.
__global__ void k_count_bound(const int* __restrict__ unordered, const unsigned long long* __restrict__ nnz, int n_tr,
                              int n_scen, float* __restrict__ bound)
{
    const int s = threadIdx.x;
    if (s < n_scen) bound[s] = *unordered ? (float)max(nnz[s], 1ull) : (float)n_tr;
}

// Iteration kernels are launched with programmatic serialisation: a kernel
// starts while its predecessor drains and waits here for its results.  What
// an iteration changes is read after the wait and by ordinary loads (its
// pointers carry no __restrict__: a load through the read-only path may only
// read what no kernel running beside it writes).
__device__ __forceinline__ void wait_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_successor_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// A sum hi + lo of FP32 terms: lo collects the roundings of hi (the exact error
// of an addition is a binary32, Knuth).  A block's objective is summed this way
// and rounded once, so that its accuracy does not depend on the rows per block
// (the largest sum picks the worst scenario); the blocks' FP32 sums then add up
// exactly in FP64 while they lie within 29 binary places of each other,
// whatever their order.  In FP64 from the terms on
// the same sums take 7 % of an iteration on a plan of 300 spots (2.00 against
// 1.87 ms for 60 iterations): the FP64 pipe is narrow.
struct Sum2 {
    float hi, lo;
};
__device__ __forceinline__ Sum2 add(Sum2 a, Sum2 b)
{
    const float s = __fadd_rn(a.hi, b.hi), t = __fsub_rn(s, a.hi);
    const float err = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, t)), __fsub_rn(b.hi, t));
    return Sum2{s, err + (a.lo + b.lo)};
}

// d_s on the compact rows, f_s and max_i |f'(d_i)| (as float bits); grid
// (row blocks, scenarios), 256 threads, kL lanes per row.  HBM-bound on large
// plans (a warp per row: 6 bytes an entry at 6.1 TB/s); on small ones, whose
// rows of some 80 entries a warp leaves two thirds idle, 8 lanes per row.
template <int kL>
__global__ void __launch_bounds__(256) k_fwd(const long long* __restrict__ crp, const unsigned short* __restrict__ ccol,
                                             const float* __restrict__ cval, int n_tr, const float* x,
                                             const unsigned char* __restrict__ tr_cls, ObjParams q, float* dose_tr,
                                             double* fsum, unsigned* max_r)
{
    constexpr int kRowsPerBlock = 8 * (32 / kL);
    const int s = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane & (kL - 1);
    const long long* rp = crp + (long long)s * (n_tr + 1);
    const int i = blockIdx.x * kRowsPerBlock + warp * (32 / kL) + lane / kL;
    long long k = 0, e = 0;
    unsigned char c = 0;
    if (i < n_tr) {
        k = __ldg(rp + i) + sub * kPadRow;
        e = __ldg(rp + i + 1);
        c = __ldg(tr_cls + i);
    }
    wait_predecessor();                               // x; the rows do not change between iterations
    let_successor_start();
    float acc = 0.0f;
#pragma unroll 2
    for (; k < e; k += kL * kPadRow) {
        const uint4 cc = __ldcs(reinterpret_cast<const uint4*>(ccol + k));
        const float4 v0 = __ldcs(reinterpret_cast<const float4*>(cval + k));
        const float4 v1 = __ldcs(reinterpret_cast<const float4*>(cval + k + 4));
        acc = fmaf(v0.x, x[cc.x & 0xffffu], acc);
        acc = fmaf(v0.y, x[cc.x >> 16], acc);
        acc = fmaf(v0.z, x[cc.y & 0xffffu], acc);
        acc = fmaf(v0.w, x[cc.y >> 16], acc);
        acc = fmaf(v1.x, x[cc.z & 0xffffu], acc);
        acc = fmaf(v1.y, x[cc.z >> 16], acc);
        acc = fmaf(v1.z, x[cc.w & 0xffffu], acc);
        acc = fmaf(v1.w, x[cc.w >> 16], acc);
    }
#pragma unroll
    for (int o = kL / 2; o >= 1; o >>= 1) acc += __shfl_xor_sync(kFullMask, acc, o);
    Sum2 f{0.0f, 0.0f};
    float rabs = 0.0f;
    if (sub == 0 && i < n_tr) {
        dose_tr[(long long)s * n_tr + i] = acc;
        f.hi = obj_term(acc, c, q);
        rabs = fabsf(obj_grad(acc, c, q));
    }
#pragma unroll
    for (int o = 16; o >= kL; o >>= 1) {
        f = add(f, Sum2{__shfl_xor_sync(kFullMask, f.hi, o), __shfl_xor_sync(kFullMask, f.lo, o)});
        rabs = fmaxf(rabs, __shfl_xor_sync(kFullMask, rabs, o));
    }
    __shared__ Sum2 part[8];
    __shared__ float pmax[8];
    if (lane == 0) {
        part[warp] = f;
        pmax[warp] = rabs;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        Sum2 t = part[0];
        float mx = pmax[0];
#pragma unroll
        for (int w = 1; w < 8; ++w) {
            t = add(t, part[w]);
            mx = fmaxf(mx, pmax[w]);
        }
        const float sum = isfinite(t.lo) ? t.hi + t.lo : t.hi;      // (an infinite term: no rest)
        if (sum != 0.0f) atomicAdd(fsum + s, (double)sum);
        if (mx > 0.0f) atomicMax(max_r + s, __float_as_uint(mx));
    }
}

// p 2^k as a 64-bit integer, truncated toward zero (p a binary32 with
// |p| 2^k < 2^63; zero and subnormal p give 0).  Integer operations only.
__device__ __forceinline__ long long to_fixed_pow2(float p, int k)
{
    const unsigned bits = __float_as_uint(p);
    const int ex = (int)((bits >> 23) & 0xffu);
    if (ex == 0) return 0;
    const long long mant = (long long)((bits & 0x7fffffu) | 0x800000u);
    const int sh = ex - 150 + k;                      // p 2^k = mant 2^sh
    long long v;
    if (sh >= 0)
        v = mant << sh;
    else
        v = sh > -24 ? (mant >> -sh) : 0;
    return (bits >> 31) ? -v : v;
}

// Rows are cut into pieces of at most kRowChunk entries so that the
// gradient's warps get work of similar length: piece c of the worst
// scenario is row c / per_row, entries [k kRowChunk, (k + 1) kRowChunk) of it
// with k = c % per_row (empty when the row is shorter).
constexpr int kRowChunk = 1024;

// Worst scenario and the gradient in 64-bit fixed point.  The scale 2^k,
// k = 62 - ceil(log2 B) with B = max_i |f'(d_i)| x (compact rows) x max |a|
// of the worst scenario, bounds every partial sum by 2^62 (the row count is
// replaced by the scenario's entry count when a row may repeat a spot).
// Each warp takes row pieces (consecutive pieces go to different blocks;
// rows with f'(d_i) = 0 add nothing and are skipped) and adds a f'(d_i) 2^k to a
// shared-memory copy of g per block, held as two 32-bit words per spot: the
// low word by a native 32-bit atomic whose returned old value gives the
// carry, the high word by a second one (exact, whatever the order).  The
// block adds its copy to g with one 64-bit atomic per spot.  Grid: number of
// SMs, 1024 threads, n_cols x 8 bytes of shared memory.
__global__ void __launch_bounds__(1024) k_bwd_fixed(const long long* __restrict__ crp, int per_row,
                                                    const unsigned short* __restrict__ ccol,
                                                    const float* __restrict__ cval, int n_tr, int n_cols,
                                                    const float* dose_tr, const unsigned char* __restrict__ tr_cls,
                                                    ObjParams q, const double* fsum_cur, const unsigned* max_r_cur,
                                                    double* fsum_next, unsigned* max_r_next,
                                                    const unsigned* __restrict__ max_abs,
                                                    const float* __restrict__ count_bound, int n_scen, float* hist,
                                                    int it, unsigned long long* g, int* g_shift)
{
    extern __shared__ unsigned gsw[];
    unsigned* lo = gsw;
    unsigned* hi = gsw + n_cols;
    __shared__ double s_f[kMaxScen];
    __shared__ int s_star, s_k;
    for (int j = threadIdx.x; j < 2 * n_cols; j += blockDim.x) gsw[j] = 0u;
    wait_predecessor();
    let_successor_start();
    if (threadIdx.x < n_scen) s_f[threadIdx.x] = fsum_cur[threadIdx.x];
    __syncthreads();
    if (threadIdx.x == 0) {
        int w = 0;
        for (int k = 1; k < n_scen; ++k)
            if (s_f[k] > s_f[w]) w = k;
        const float bound = __uint_as_float(max_r_cur[w]) * count_bound[w] * __uint_as_float(max_abs[w]);
        int e = 129;                                  // an overflowed bound: above any binary32
        if (bound <= 3.4028235e38f) frexpf(bound, &e);  // bound < 2^e
        s_star = w;
        s_k = bound > 0.0f ? 62 - e : 0;
        if (blockIdx.x == 0) {
            if (hist) hist[it] = (float)s_f[w];
            *g_shift = s_k;
        }
    }
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x < n_scen) {
        fsum_next[threadIdx.x] = 0.0;
        max_r_next[threadIdx.x] = 0u;
    }
    const int s = s_star, kq = s_k, lane = threadIdx.x & 31;
    const float* d = dose_tr + (long long)s * n_tr;
    const int warps = blockDim.x >> 5;
    const long long* rp = crp + (long long)s * (n_tr + 1);
    const long long nc = (long long)n_tr * per_row;
    for (long long ci = blockIdx.x + (long long)gridDim.x * (threadIdx.x >> 5); ci < nc;
         ci += (long long)gridDim.x * warps) {
        const int i = (int)(ci / per_row);
        const long long rb = __ldg(rp + i), re = __ldg(rp + i + 1);
        const long long b = rb + (ci - (long long)i * per_row) * kRowChunk;
        if (b >= re) continue;                        // warp-uniform: the row is shorter
        const float ri = obj_grad(d[i], __ldg(tr_cls + i), q);
        if (ri == 0.0f) continue;                     // warp-uniform
        const long long e = min(b + kRowChunk, re);
#pragma unroll 2
        for (long long k = b + lane * kPadRow; k < e; k += 32 * kPadRow) {
            const uint4 c = __ldcs(reinterpret_cast<const uint4*>(ccol + k));
            const float4 v0 = __ldcs(reinterpret_cast<const float4*>(cval + k));
            const float4 v1 = __ldcs(reinterpret_cast<const float4*>(cval + k + 4));
            const unsigned js[8] = {c.x & 0xffffu, c.x >> 16, c.y & 0xffffu, c.y >> 16,
                                    c.z & 0xffffu, c.z >> 16, c.w & 0xffffu, c.w >> 16};
            const float as[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
            unsigned l[8], h[8], old[8];
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const unsigned long long fx = (unsigned long long)to_fixed_pow2(as[t] * ri, kq);
                l[t] = (unsigned)fx;
                h[t] = (unsigned)(fx >> 32);
            }
            // the eight low adds are in flight together; their old values give
            // the carries of the high ones (adding 0 changes nothing)
#pragma unroll
            for (int t = 0; t < 8; ++t) old[t] = l[t] ? atomicAdd(lo + js[t], l[t]) : 0u;
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const unsigned hi_add = h[t] + (old[t] + l[t] < old[t] ? 1u : 0u);
                if (hi_add) atomicAdd(hi + js[t], hi_add);
            }
        }
    }
    __syncthreads();
    for (int j = threadIdx.x; j < n_cols; j += blockDim.x) {
        const unsigned long long t = ((unsigned long long)hi[j] << 32) | lo[j];
        if (t != 0ull) atomicAdd(g + j, t);
    }
}

// g_j = (fixed-point sum) 2^-k, reset for the next iteration, then Adam
// (Kingma & Ba 2015) on x_j, clamped at zero.
__global__ void k_adam_fixed(unsigned long long* g, const int* g_shift, int n_cols, float* x, float* m, float* v, float step,
                             float c1, float c2, float eps)
{
    wait_predecessor();
    let_successor_start();
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n_cols) return;
    const long long gi = (long long)g[j];
    g[j] = 0ull;
    const float gj = (float)ldexp((double)gi, -*g_shift);
    const float mj = fmaf(0.9f, m[j], 0.1f * gj), vj = fmaf(0.999f, v[j], 0.001f * gj * gj);
    m[j] = mj;
    v[j] = vj;
    x[j] = fmaxf(x[j] - step * (mj * c1) / (sqrtf(vj * c2) + eps), 0.0f);
}

}  // namespace

// ---------------------------------------------------------------------------
// Host side (called from api.cu).
// ---------------------------------------------------------------------------
// One device allocation cut into aligned parts.
struct Arena {
    unsigned char* base = nullptr;
    size_t used = 0;
    ~Arena() { cudaFree(base); }
    // offsets first, then one allocation
    template <class T>
    size_t add(size_t n)
    {
        const size_t at = used;
        used += (std::max<size_t>(n, 1) * sizeof(T) + 255) / 256 * 256;
        return at;
    }
    cudaError_t allocate() { return cudaMalloc(reinterpret_cast<void**>(&base), used); }
    template <class T>
    T* at(size_t offset) const { return reinterpret_cast<T*>(base + offset); }
};

// Counts the target and ring voxels (classes 1 and 2); *ws keeps the device
// arrays for run_robust_optimize and is freed by free_class_rows.
struct ClassRows {
    Arena a;
    size_t offset = 0;
    long long blocks = 0;
};

cudaError_t count_class_rows(const unsigned char* cls, long long n_rows, cudaStream_t st, ClassRows** ws, long long* n_target,
                             long long* n_ring)
{
    ClassRows* w = new ClassRows;
    *ws = w;
    w->blocks = (n_rows + kClsThreads * kClsPer - 1) / (kClsThreads * kClsPer);
    const size_t o_cnt = w->a.add<long long>((size_t)w->blocks);
    w->offset = w->a.add<long long>((size_t)w->blocks);
    const size_t o_tmp = w->a.add<long long>(scan_tmp_elems(w->blocks)), o_tot = w->a.add<ClassTotals>(1);
    ClassTotals h{};
    cudaError_t e = w->a.allocate();
    if (e == cudaSuccess) e = cudaMemsetAsync(w->a.at<ClassTotals>(o_tot), 0, sizeof h, st);
    if (e != cudaSuccess) return e;
    k_cls_count<<<(unsigned)w->blocks, kClsThreads, 0, st>>>(cls, n_rows, w->a.at<long long>(o_cnt),
                                                             w->a.at<ClassTotals>(o_tot));
    e = cudaGetLastError();
    if (e == cudaSuccess)
        e = launch_exclusive_scan(w->a.at<long long>(o_cnt), w->a.at<long long>(w->offset), w->blocks,
                                  w->a.at<long long>(o_tmp), st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, w->a.at<ClassTotals>(o_tot), sizeof h, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    *n_target = (long long)h.target;
    *n_ring = (long long)h.ring;
    return e;
}

void free_class_rows(ClassRows* w) { delete w; }

cudaError_t run_robust_optimize(const long long* const* rp, const int* const* col, const float* const* val, int n_scen,
                                long long n_rows, int n_cols, const unsigned char* cls, const ClassRows& rows,
                                const OptSpec& spec, float* x, float* hist_host, cudaStream_t st, float* ms_out,
                                OptSetupInfo* info)
{
    cudaError_t e;
#define OPT_TRY(expr) do { if ((e = (expr)) != cudaSuccess) return e; } while (0)
    if ((size_t)n_cols * sizeof(unsigned long long) > kBwdSmemMax) return cudaErrorInvalidValue;
    const int n_tr = (int)(spec.n_target + spec.n_ring);
    const int S = n_scen;
    CsrSet set;
    for (int s = 0; s < S; ++s) set.m[s] = Csr{rp[s], col[s], val[s]};
    cudaEvent_t ev[3] = {nullptr, nullptr, nullptr};
    struct EvFree {
        cudaEvent_t* e;
        ~EvFree() { for (int k = 0; k < 3; ++k) if (e[k]) cudaEventDestroy(e[k]); }
    } evfree{ev};
    for (auto& q : ev) OPT_TRY(cudaEventCreate(&q));
    OPT_TRY(cudaEventRecord(ev[0], st));
    // working arrays in one allocation; the first part starts at zero
    Arena a;
    const size_t o_g = a.add<unsigned long long>((size_t)n_cols), o_m = a.add<float>((size_t)n_cols),
                 o_v = a.add<float>((size_t)n_cols), o_fsum = a.add<double>((size_t)2 * S),
                 o_maxr = a.add<unsigned>((size_t)2 * S), o_maxabs = a.add<unsigned>(S), o_unord = a.add<int>(1),
                 o_nnz = a.add<unsigned long long>((size_t)S + 1), zeroed = a.used;      // entries per scenario, longest row
    const size_t o_shift = a.add<int>(1), o_bound = a.add<float>(S), o_hist = a.add<float>(std::max(spec.iterations, 1)),
                 o_rows = a.add<int>(n_tr), o_cls = a.add<unsigned char>(n_tr),
                 o_dose = a.add<float>((size_t)S * n_tr);
    const size_t n_ptr = (size_t)S * (n_tr + 1);
    const size_t o_plen = a.add<long long>(n_ptr), o_crp = a.add<long long>(n_ptr),
                 o_tmp = a.add<long long>(scan_tmp_elems((long long)n_ptr));
    OPT_TRY(a.allocate());
    OPT_TRY(cudaMemsetAsync(a.base, 0, zeroed, st));
    int* tr_rows = a.at<int>(o_rows);
    unsigned char* tr_cls = a.at<unsigned char>(o_cls);
    long long* crp = a.at<long long>(o_crp);
    unsigned long long* nnz = a.at<unsigned long long>(o_nnz);
    // compact row layout
    k_cls_rows<<<(unsigned)rows.blocks, kClsThreads, 0, st>>>(cls, n_rows, rows.a.at<long long>(rows.offset), tr_rows, tr_cls);
    OPT_TRY(cudaGetLastError());
    k_tr_len<<<dim3((unsigned)((n_tr + 256) / 256), (unsigned)S), 256, 0, st>>>(set, tr_rows, n_tr,
                                                                                a.at<long long>(o_plen), nnz, nnz + S);
    OPT_TRY(cudaGetLastError());
    OPT_TRY(launch_exclusive_scan(a.at<long long>(o_plen), crp, (long long)n_ptr, a.at<long long>(o_tmp), st));
    long long total_c = 0;
    std::vector<unsigned long long> h_nnz((size_t)S + 1);
    OPT_TRY(cudaMemcpyAsync(&total_c, crp + n_ptr - 1, sizeof total_c, cudaMemcpyDeviceToHost, st));
    OPT_TRY(cudaMemcpyAsync(h_nnz.data(), nnz, sizeof(unsigned long long) * h_nnz.size(), cudaMemcpyDeviceToHost, st));
    OPT_TRY(cudaStreamSynchronize(st));
    const long long longest = (long long)h_nnz[S];
    const int per_row = (int)std::max<long long>(1, (longest + kRowChunk - 1) / kRowChunk);
    Arena compact;
    const size_t o_ccol = compact.add<unsigned short>((size_t)total_c), o_cval = compact.add<float>((size_t)total_c);
    OPT_TRY(compact.allocate());
    unsigned short* ccol = compact.at<unsigned short>(o_ccol);
    float* cval = compact.at<float>(o_cval);
    k_tr_gather<<<dim3((unsigned)((n_tr + 7) / 8), (unsigned)S), 256, 0, st>>>(
        set, tr_rows, n_tr, n_cols, crp, ccol, cval, a.at<int>(o_unord), a.at<unsigned>(o_maxabs));
    OPT_TRY(cudaGetLastError());
    k_count_bound<<<1, kMaxScen, 0, st>>>(a.at<int>(o_unord), nnz, n_tr, S, a.at<float>(o_bound));
    OPT_TRY(cudaGetLastError());
    const int smem = (int)(sizeof(unsigned long long) * n_cols);
    OPT_TRY(cudaFuncSetAttribute(k_bwd_fixed, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    int dev = 0, nsm = 0;
    OPT_TRY(cudaGetDevice(&dev));
    OPT_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    OPT_TRY(cudaEventRecord(ev[1], st));
    const ObjParams q{spec.dp, spec.w_u, spec.w_o, spec.w_r, spec.over, spec.ring,
                      1.0f / (float)std::max<long long>(spec.n_target, 1),
                      1.0f / (float)std::max<long long>(spec.n_ring, 1)};
    // 8 lanes serve a row of up to 128 entries in two passes
    const bool short_rows = total_c <= 128ll * S * n_tr;
    const auto fwd = short_rows ? k_fwd<8> : k_fwd<32>;
    const int rows_per_block = short_rows ? 32 : 8;
    const dim3 gf((unsigned)std::max((n_tr + rows_per_block - 1) / rows_per_block, 1), (unsigned)S);
    double* fsum = a.at<double>(o_fsum);
    unsigned* max_r = a.at<unsigned>(o_maxr);
    float* dose = a.at<float>(o_dose);
    float* hist = a.at<float>(o_hist);
    unsigned long long* g = a.at<unsigned long long>(o_g);
    int* g_shift = a.at<int>(o_shift);
    for (int it = 0; it < spec.iterations; ++it) {
        const int cu = it & 1, nx = (it + 1) & 1;
        OPT_TRY(launch_after(fwd, gf, 256, 0, st, crp, ccol, cval, n_tr, x, tr_cls, q, dose, fsum + cu * S, max_r + cu * S));
        OPT_TRY(launch_after(k_bwd_fixed, dim3((unsigned)nsm), 1024, (size_t)smem, st, crp, per_row, ccol, cval, n_tr, n_cols,
                             dose, tr_cls, q, fsum + cu * S, max_r + cu * S, fsum + nx * S, max_r + nx * S,
                             a.at<unsigned>(o_maxabs), a.at<float>(o_bound), S, hist, it, g, g_shift));
        const double t = it + 1;
        OPT_TRY(launch_after(k_adam_fixed, dim3((unsigned)((n_cols + 255) / 256)), 256, 0, st, g, g_shift, n_cols, x,
                             a.at<float>(o_m), a.at<float>(o_v), spec.step, (float)(1.0 / (1.0 - std::pow(0.9, t))),
                             (float)(1.0 / (1.0 - std::pow(0.999, t))), spec.eps));
    }
    OPT_TRY(cudaEventRecord(ev[2], st));
    if (hist_host && spec.iterations > 0)
        OPT_TRY(cudaMemcpyAsync(hist_host, hist, sizeof(float) * spec.iterations, cudaMemcpyDeviceToHost, st));
    OPT_TRY(cudaStreamSynchronize(st));
    float setup = 0.0f, iters = 0.0f;
    cudaEventElapsedTime(&setup, ev[0], ev[1]);
    cudaEventElapsedTime(&iters, ev[1], ev[2]);
    if (ms_out) {
        ms_out[0] = iters;
        ms_out[1] = setup;
    }
    if (info) {
        info->n_tr = n_tr;
        info->nnz_tr = 0;
        for (int s = 0; s < S; ++s) info->nnz_tr += (long long)h_nnz[s];
        info->compact_entries = total_c;
    }
#undef OPT_TRY
    return cudaSuccess;
}

cudaError_t run_weights_dose(const long long* rp, const int* col, const float* val, long long n_rows, int n_cols,
                             const float* x, float* dose, cudaStream_t st, int num_sms)
{
    CsrSet set;
    set.m[0] = Csr{rp, col, val};
    k_spmv<false><<<dim3((unsigned)(num_sms * kSpmvBlocks), 1), 256, 0, st>>>(set, n_rows, n_cols, x, nullptr, 0.0f, dose,
                                                                             nullptr);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? cudaStreamSynchronize(st) : e;
}

cudaError_t run_target_indices(const long long* const* rp, const int* const* col, const float* const* val, int n_scen,
                               long long n_rows, int n_cols, const unsigned char* cls, float dp, const float* x,
                               double* out, cudaStream_t st, int num_sms)
{
    CsrSet set;
    for (int s = 0; s < n_scen; ++s) set.m[s] = Csr{rp[s], col[s], val[s]};
    IndexSums* sums = nullptr;
    std::vector<IndexSums> h(n_scen);
    const size_t bytes = sizeof(IndexSums) * n_scen;
    cudaError_t e = cudaMalloc(&sums, bytes);
    if (e == cudaSuccess) e = cudaMemsetAsync(sums, 0, bytes, st);
    if (e == cudaSuccess) {
        k_spmv<true><<<dim3((unsigned)(num_sms * kSpmvBlocks), (unsigned)n_scen), 256, 0, st>>>(set, n_rows, n_cols, x, cls, dp,
                                                                                             nullptr, sums);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(h.data(), sums, bytes, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(sums);
    if (e != cudaSuccess) return e;
    for (int s = 0; s < n_scen; ++s) {
        const IndexSums& r = h[s];
        const double nt = (double)std::max<unsigned long long>(r.target, 1);
        const int mn_bits = kMaxBits - r.neg_min;
        float mn, mx;
        std::memcpy(&mn, &mn_bits, 4);
        std::memcpy(&mx, &r.max, 4);
        out[4 * s + 0] = (double)r.hit / nt;
        out[4 * s + 1] = r.target ? mn / dp : 0.0;
        out[4 * s + 2] = (double)r.high / nt;
        out[4 * s + 3] = r.target ? mx / dp : 0.0;
    }
    return cudaSuccess;
}

}  // namespace vpmc
