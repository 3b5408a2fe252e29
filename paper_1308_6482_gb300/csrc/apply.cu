// K3: per-particle force and torque from the pair results (Sec. III B):
//   f_i += F_i,  t_i += T_i + (y*_i - r_i) x F_i,
//   f_j -= F_i,  t_j -= T_i + (y*_j - r_j) x F_i   (Eq. lub:resistance).
// Two variants:
//   atomic         one thread per pair, atomic adds (fast, order-dependent
//                  rounding); lanes of a warp that share particle i (pairs
//                  come sorted by i) are combined first with a segmented
//                  warp reduction, so i-side atomics drop to one per run.
//   deterministic  incidence lists (counting sort by particle, entries
//                  sorted by pair index and side), eight lanes or one lane
//                  per particle summing in that fixed order: bitwise
//                  reproducible.
#include "pair_force.cuh"

namespace {

// v, or -v where side is 1, off the FP64 pipe
__device__ __forceinline__ float side_sign(float v, int side) { return side ? -v : v; }
__device__ __forceinline__ double side_sign(double v, int side)
{
    return __hiloint2double(__double2hiint(v) ^ (side << 31), __double2loint(v));
}

// (six multiply-adds in all: in FP64 mode the FP64 pipe bounds the sums)
template <typename T>
__device__ __forceinline__ void pair_contrib(const T *__restrict__ FT, const T *__restrict__ lever, size_t C,
                                             int k, int side, T out[6])
{
    const V3<T> F = mk<T>(FT[k], FT[C + k], FT[2 * C + k]);
    const V3<T> Tq = mk<T>(FT[3 * C + k], FT[4 * C + k], FT[5 * C + k]);
    const V3<T> l = side ? mk<T>(lever[3 * C + k], lever[4 * C + k], lever[5 * C + k])
                         : mk<T>(lever[k], lever[C + k], lever[2 * C + k]);
    out[0] = side_sign(F.x, side);
    out[1] = side_sign(F.y, side);
    out[2] = side_sign(F.z, side);
    out[3] = side_sign(fma(l.y, F.z, fma(-l.z, F.y, Tq.x)), side);
    out[4] = side_sign(fma(l.z, F.x, fma(-l.x, F.z, Tq.y)), side);
    out[5] = side_sign(fma(l.x, F.y, fma(-l.y, F.x, Tq.z)), side);
}

template <typename T>
__global__ void __launch_bounds__(256) k_apply_atomic(const int32_t *__restrict__ pi, const int32_t *__restrict__ pj,
                                                      const int32_t *__restrict__ d_count, int32_t cap,
                                                      const T *__restrict__ FT, const T *__restrict__ lever, int n,
                                                      T *__restrict__ force, T *__restrict__ torque)
{
    pdl_wait();
    pdl_trigger();
    const int count = pair_count(d_count, cap);
    const size_t C = (size_t)cap;
    const size_t N = (size_t)n;
    // the loop bound is warp-uniform so the whole warp takes part in the shuffles
    for (int base = blockIdx.x * blockDim.x; base < count; base += gridDim.x * blockDim.x) {
        const int k = base + threadIdx.x;
        const bool active = k < count;
        int i = active ? pi[k] : -1;
        int j = active ? pj[k] : -1;
        if (i < 0 || i >= n) i = -1;
        T ci[6] = {0, 0, 0, 0, 0, 0}, cj[6] = {0, 0, 0, 0, 0, 0};
        if (i >= 0) {
            pair_contrib<T>(FT, lever, C, k, 0, ci);
            if (j >= 0 && j < n) pair_contrib<T>(FT, lever, C, k, 1, cj);
        }
        scatter_warp<T>(i, (j >= 0 && j < n) ? j : -1, N, ci, cj, force, torque);
    }
}

// deterministic variant ------------------------------------------------------
// Each pair side's place among its particle's entries, taken where the entries
// are counted (the fill then needs no second round of atomics).
__global__ void k_inc_count(const int32_t *__restrict__ pi, const int32_t *__restrict__ pj,
                            const int32_t *__restrict__ d_count, int32_t cap, int n, int32_t *__restrict__ cnt,
                            int2 *__restrict__ place)
{
    pdl_wait();
    pdl_trigger();
    const int count = pair_count(d_count, cap);
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < count; k += gridDim.x * blockDim.x) {
        const int i = pi[k], j = pj[k];
        if (i < 0 || i >= n) continue;
        int2 pl = make_int2(atomicAdd(cnt + i, 1), 0);
        if (j >= 0 && j < n) pl.y = atomicAdd(cnt + j, 1);
        place[k] = pl;
    }
}

__global__ void k_inc_fill(const int32_t *__restrict__ pi, const int32_t *__restrict__ pj,
                           const int32_t *__restrict__ d_count, int32_t cap, int n,
                           const int32_t *__restrict__ start, const int2 *__restrict__ place,
                           int32_t *__restrict__ inc)
{
    pdl_wait();
    pdl_trigger();
    const int count = pair_count(d_count, cap);
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < count; k += gridDim.x * blockDim.x) {
        const int i = pi[k], j = pj[k];
        if (i < 0 || i >= n) continue;
        // the slots stay inside the 2 cap entries even if the scan's offsets were wrong (a timed-out wait)
        const int2 pl = place[k];
        const int si = start[i] + pl.x;
        if (si >= 0 && si < 2 * cap) inc[si] = 2 * k;
        if (j >= 0 && j < n) {
            const int sj = start[j] + pl.y;
            if (sj >= 0 && sj < 2 * cap) inc[sj] = 2 * k + 1;
        }
    }
}

// The sums, eight lanes per particle: the lanes sort the particle's entries
// (pair index, side) by rank, fetch the contributions of eight entries at a
// time (nine scattered loads each, the bound: one lane per particle had
// them one entry after the other, 37 us at 100,003 particles and 340k pairs
// against 13) and six lanes add one component each in the sorted order, as a
// single lane would.  A particle of more than kRankMax entries is sorted in
// place by one lane.
constexpr int kGroup = 8, kRankMax = 32;

// One lane per particle, sorting in place, is the better form where there are
// enough particles to fill the GPU and too few entries for eight lanes: below
// 1.5 a particle from kLaneFrom particles on, below 3.5 from kLaneMore on.  The
// number of entries is known on the device only, so the kernel has both forms.
// Whole call in mixed precision, eight lanes and one: 200,000 particles with
// 0.8 entries each 24.5 and 18.8 us, with 2.4 each 30.9 and 33.3; 262,144 with
// 1.6 each 33.9 and 30.1, with 4.8 each 57.5 and 67.5; 400,000 with 2.2 each
// 50.9 and 48.4, with 3.2 each 61.7 and 63.7, but 81.6 and 63.4 in arrays of 16
// pairs a particle (random order, components 26 MB apart).
constexpr int kLaneFrom = 131072, kLaneMore = 250000;
__device__ __forceinline__ bool one_lane(int n, int entries)
{
    return n >= kLaneFrom && 2 * (int64_t)entries < (n >= kLaneMore ? 7 : 3) * (int64_t)n;
}

// a particle's entries [b, e), sorted in place by the calling lane
__device__ __forceinline__ void sort_entries(int32_t *inc, int b, int e)
{
    for (int a = b + 1; a < e; ++a) {
        const int v = inc[a];
        int c = a - 1;
        while (c >= b && inc[c] > v) {
            inc[c + 1] = inc[c];
            --c;
        }
        inc[c + 1] = v;
    }
}

// a component of a particle's sum
template <typename T>
__device__ __forceinline__ void store_sum(T *force, T *torque, size_t N, int p, int comp, T v, int accumulate)
{
    T *const dst = comp < 3 ? force + comp * N + p : torque + (comp - 3) * N + p;
    *dst = accumulate ? *dst + v : v;
}

// the sums by one lane per particle
template <typename T>
__device__ __forceinline__ void sum_by_lane(const int32_t *__restrict__ start, int entries, int32_t *__restrict__ inc,
                                            int n, const T *__restrict__ FT, const T *__restrict__ lever, int32_t cap,
                                            T *__restrict__ force, T *__restrict__ torque, int accumulate,
                                            int blocks)
{
    const size_t C = (size_t)cap, N = (size_t)n;
    if ((int)blockIdx.x >= blocks) return;
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += blocks * blockDim.x) {
        const int b = max(0, min(start[p], 2 * cap));
        const int e = max(b, min((p + 1 < n) ? start[p + 1] : entries, 2 * cap));
        sort_entries(inc, b, e);
        T acc[6] = {0, 0, 0, 0, 0, 0};
        for (int a = b; a < e; ++a) {
            const int v = inc[a];
            if (v < 0 || (v >> 1) >= cap) continue;  // never filled (after a timed-out scan)
            T c6[6];
            pair_contrib<T>(FT, lever, C, v >> 1, v & 1, c6);
#pragma unroll
            for (int q = 0; q < 6; ++q) acc[q] += c6[q];
        }
#pragma unroll
        for (int q = 0; q < 6; ++q) store_sum(force, torque, N, p, q, acc[q], accumulate);
    }
}

// resident blocks of 256 threads per SM: the registers' limit
template <typename T>
constexpr int sum_blocks() { return sizeof(T) == 4 ? 8 : 5; }

template <typename T>
__global__ void __launch_bounds__(256, sum_blocks<T>()) k_inc_sum(const int32_t *__restrict__ start, const int32_t *__restrict__ total,
                                                 int32_t *__restrict__ inc, int n, const T *__restrict__ FT,
                                                 const T *__restrict__ lever, int32_t cap, T *__restrict__ force,
                                                 T *__restrict__ torque, int accumulate, int wave)
{
    pdl_wait();
    pdl_trigger();
    constexpr int NGRP = 256 / kGroup;
    __shared__ int key_s[NGRP][kRankMax + 1], sorted_s[NGRP][kRankMax + 1];
    __shared__ T c_s[NGRP][kGroup * 6 + 1];
    const size_t C = (size_t)cap, N = (size_t)n;
    if (one_lane(n, *total)) {  // (the same for every block)
        sum_by_lane<T>(start, *total, inc, n, FT, lever, cap, force, torque, accumulate,
                       min((int)gridDim.x, wave));
        return;
    }
    const int sub = threadIdx.x % kGroup, g = threadIdx.x / kGroup;
    int *const key = key_s[g], *const sorted = sorted_s[g];
    T *const cs = c_s[g];
    // the same trip count for every lane of a warp
    for (int p0 = blockIdx.x * NGRP; p0 < n; p0 += gridDim.x * NGRP) {
        const int p = p0 + g;
        int b = 0, e = 0;
        if (p < n) {
            b = max(0, min(start[p], 2 * cap));
            e = max(b, min((p + 1 < n) ? start[p + 1] : *total, 2 * cap));
        }
        const int m = e - b;
        const bool many = m > kRankMax;
        if (!many)
            for (int q = sub; q < m; q += kGroup) key[q] = inc[b + q];
        else if (sub == 0)
            sort_entries(inc, b, e);
        __syncwarp();
        if (!many)
            for (int q = sub; q < m; q += kGroup) {
                const int v = key[q];
                int r = 0;
                for (int t = 0; t < m; ++t) r += key[t] < v;
                sorted[r] = v;
            }
        __syncwarp();
        const int mw = (int)__reduce_max_sync(0xffffffffu, (unsigned)m);
        T acc = 0;
        for (int q0 = 0; q0 < mw; q0 += kGroup) {
            const int q = q0 + sub;
            if (q < m) {
                const int v = many ? inc[b + q] : sorted[q];
                T c6[6] = {0, 0, 0, 0, 0, 0};
                // (an entry never filled, after a timed-out scan, is skipped)
                if (v >= 0 && (v >> 1) < cap) pair_contrib<T>(FT, lever, C, v >> 1, v & 1, c6);
#pragma unroll
                for (int a = 0; a < 6; ++a) cs[sub * 6 + a] = c6[a];
            }
            __syncwarp();
            if (sub < 6)
                for (int t = 0; t < kGroup && q0 + t < m; ++t) acc += cs[t * 6 + sub];
            __syncwarp();
        }
        if (p < n && sub < 6) store_sum(force, torque, N, p, sub, acc, accumulate);
    }
}

template <typename T>
void launch_sum(int num_sms, cudaStream_t st, const int32_t *start, const int32_t *total, int32_t *inc, int n,
                const T *FT, const T *lever, int32_t cap, T *force, T *torque, int accumulate)
{
    constexpr int block = 256;
    const int grid = grid_for((int64_t)n * kGroup, block, num_sms, n >= kLaneFrom ? 16 : 32);
    const int wave = sum_blocks<T>() * num_sms;
    // A grid of less than one wave, but more than two blocks an SM, and the form
    // by one lane take a plain launch: with a programmatic one the blocks fill
    // those SMs first that the kernel before leaves first, eight to an SM, while
    // others stay empty (20,000 particles with 8 entries each: 22.4 us for the
    // call against 17.4, in FP64 27.2 and 21.0)
    if (n >= kLaneFrom || (grid > 2 * num_sms && grid < wave))
        k_inc_sum<T><<<grid, block, 0, st>>>(start, total, inc, n, FT, lever, cap, force, torque, accumulate, wave);
    else
        (void)launch_pdl(k_inc_sum<T>, grid, block, 0, st, start, total, inc, n, FT, lever, cap, force, torque,
                         accumulate, wave);
}

inline size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

}  // namespace

int launch_apply(lub_ctx *ctx, const int32_t *pi, const int32_t *pj, const int32_t *d_count, int32_t cap,
                 const void *FT, const void *lever, int32_t n, void *force, void *torque, int precision,
                 int accumulate, int deterministic, cudaStream_t st)
{
    const size_t esz = precision == LUB_MIXED ? sizeof(float) : sizeof(double);
    if (n == 0) return LUB_OK;
    if (!deterministic) {
        if (!accumulate) {
            const int rc = zero_force_torque(ctx, force, torque, 3 * (size_t)n * esz, st);
            if (rc) return rc;
        }
        if (cap == 0) return LUB_OK;
        const Shape2 sh = tuned_shape(ctx, LUB_TUNE_APPLY, cap);
        const int grid = sh.grid, block = sh.block;
        lub_trace_mark(ctx, LUB_TRACE_APPLY, st);
        if (precision == LUB_MIXED)
            (void)launch_pdl(k_apply_atomic<float>, grid, block, 0, st, pi, pj, d_count, cap, (const float *)FT,
                                                          (const float *)lever, n, (float *)force, (float *)torque);
        else
            (void)launch_pdl(k_apply_atomic<double>, grid, block, 0, st, pi, pj, d_count, cap, (const double *)FT,
                                                           (const double *)lever, n, (double *)force,
                                                           (double *)torque);
        lub_trace_mark(ctx, LUB_TRACE_APPLY, st);
        return lub_check_cuda(ctx, cudaGetLastError(), "k_apply_atomic launch");
    }
    // scratch: cnt/start [n] and the scan's state (cleared together), total [1],
    // inc [2 cap], place [cap]
    const size_t b_cnt = align256((size_t)n * 4), b_tmp = align256(scan_tmp_bytes(n)), b_tot = 256,
                 b_inc = align256(2 * (size_t)cap * 4 + 4), b_place = align256((size_t)cap * sizeof(int2));
    int rc = lub_ensure_scratch(ctx, b_cnt + b_tmp + b_tot + b_inc + b_place);
    if (rc) return rc;
    char *s = (char *)ctx->scratch;
    int32_t *cnt = (int32_t *)s;
    void *tmp = s + b_cnt;
    int32_t *tot = (int32_t *)(s + b_cnt + b_tmp);
    int32_t *inc = (int32_t *)(s + b_cnt + b_tmp + b_tot);
    int2 *place = (int2 *)(s + b_cnt + b_tmp + b_tot + b_inc);
    rc = zero_async(ctx, ctx->num_sms, cnt, b_cnt + b_tmp, st);
    if (rc) return rc;
    const int block = 256;
    const int gp = grid_for(cap > 0 ? cap : 1, block, ctx->num_sms, 8);
    (void)launch_pdl(k_inc_count, gp, block, 0, st, pi, pj, d_count, cap, n, cnt, place);
    rc = scan_exclusive(ctx, cnt, n, tot, tmp, b_tmp, st, ctx->d_flags + 1, true);
    if (rc) return rc;
    (void)launch_pdl(k_inc_fill, gp, block, 0, st, pi, pj, d_count, cap, n, (const int32_t *)cnt, (const int2 *)place,
                     inc);
    if (precision == LUB_MIXED)
        launch_sum<float>(ctx->num_sms, st, cnt, tot, inc, n, (const float *)FT, (const float *)lever, cap,
                          (float *)force, (float *)torque, accumulate);
    else
        launch_sum<double>(ctx->num_sms, st, cnt, tot, inc, n, (const double *)FT, (const double *)lever, cap,
                           (double *)force, (double *)torque, accumulate);
    return lub_check_cuda(ctx, cudaGetLastError(), "deterministic apply launch");
}
