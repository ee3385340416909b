// Radially averaged three-dimensional correlation C(r) and structure factor S(k) of one
// lattice (Methods, "Calculating the correlation function": the spin-spin sum for every
// lag vector from FFTs, Eq. (3), then a radial average; Results: S(k,t) is the Fourier
// transform of C).
//
//   1. k_unpack_real: packed spins -> +-1 reals in cuFFT's padded in-place R2C layout
//      (rows of 2(L/2+1) reals).
//   2. cuFFT R2C (library FFT).
//   3. k_power: P(q) = |F(q)|^2 per mode of the half spectrum, summed per radial bin for S
//      (modes with 0 < qx < L/2 stand for their Hermitian partner too), and written back
//      as (P, 0) for the inverse.
//   4. cuFFT C2R: g(k) = sum_q P(q) e^{iqk} = N G(k), G(k) = sum_i s_i s_(i+k).
//   5. k_radial_corr: G(k) = g/N rounded to the nearest integer and summed per radial bin in
//      int64.  G(k) is an integer; when the FFT error stays below 1/2 (always in double
//      precision, at small L in single) the rounding recovers it exactly and C is exact.  A
//      lag whose g/N lies more than 1/4 from an integer is counted as inexact.
//   6. k_radial_finish: bin means, C(b) = sum_G / (N n_b), S(b) = sum_P / (N n_b), and the
//      length l at which C first crosses c for r <= L/2.
//
// Binning: reflecting any component leaves a vector's bin.  So one thread takes the values at
// (x, +-dy, +-dz) together (and (L - x, +-dy, +-dz) for lags): one bin computation for up to eight.  The
// integers of a lag pass are summed over a walk of the thread along dy or dz while the bin stays, then
// added to the CTA's bins in shared memory.  The modes' |F|^2 are summed in their precision over runs
// of equal bins of 32 consecutive x (a warp scan per row), then in double over the four rows and the
// bins.  (With a bin, a scan and a 64-bit atomic per value and row these passes took 0.80 and 0.94 ms
// at L = 512 for 1.07 and 0.54 GB, the count 0.69; now 0.43, 0.27 and 0.06.)
// The number of vectors per bin does not depend on the state and is counted once per context.
// The transform buffer and cuFFT's work area stay allocated in the context between calls.
//
// Bins: components as minimal images, squared length D, bin round(sqrt(D)) computed exactly
// as (isqrt(4D) + 1) / 2.
#include <cufft.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace ising {

namespace {

__host__ __device__ __forceinline__ int isqrt_exact(int v)
{
    int s = (int)sqrtf((float)v);  // within one or two of the answer; corrected exactly below
    while (s > 0 && s * s > v) --s;
    while ((s + 1) * (s + 1) <= v) ++s;
    return s;
}

// round(sqrt(D)): the b with b^2 - b < D <= b^2 + b (D < 2^24, so the estimate is off by at most one).
__device__ __forceinline__ int bin_of(int D)
{
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"((float)D));
    int b = __float2int_rn(r);
    b += D > b * b + b;
    b -= (b > 0) & (D <= b * b - b);
    return b;
}

template <typename T>
struct Cx;
template <>
struct Cx<float> {
    using type = cufftComplex;
};
template <>
struct Cx<double> {
    using type = cufftDoubleComplex;
};

template <typename T>
struct Pair;
template <>
struct Pair<float> {
    using type = float2;
};
template <>
struct Pair<double> {
    using type = double2;
};

constexpr int RAD_THREADS = 256;
constexpr int RAD_FOLD_THREADS = 544;  // 0 .. L/2 of L = 1024 in one pass, of L = 2048 in two

}  // namespace

int64_t radial_nbins(int L) { return (int64_t)((isqrt_exact(3 * L * L) + 1) >> 1) + 1; }

// 1. A warp takes a row, a lane four consecutive sites, two of each sublattice (rows are aligned
// to a pair only, so two stores of a pair each).
template <typename T>
__global__ void __launch_bounds__(RAD_THREADS) k_unpack_real(const uint32_t *lat_r, T *buf, Geom g, int64_t P)
{
    const int L = g.L, Q = L / 4;  // L is a multiple of 4
    const int lane = threadIdx.x & 31, nwarp = gridDim.x * (RAD_THREADS / 32);
    for (int row = blockIdx.x * (RAD_THREADS / 32) + (threadIdx.x >> 5); row < L * L; row += nwarp) {
        const int z = row / L, y = row - z * L;
        const int64_t q0 = (y + z) & 1;  // sublattice of even x
        const uint32_t *r0 = lat_r + q0 * g.nw + (int64_t)row * g.W, *r1 = lat_r + (1 - q0) * g.nw + (int64_t)row * g.W;
        typename Pair<T>::type *dst = reinterpret_cast<typename Pair<T>::type *>(buf + (int64_t)row * P);
#pragma unroll 4
        for (int k = lane; k < Q; k += 32) {
            const int bit = 2 * (k & 15);  // compressed index 2 k
            const uint32_t w0 = __ldg(r0 + (k >> 4)) >> bit, w1 = __ldg(r1 + (k >> 4)) >> bit;
            typename Pair<T>::type a, b;
            a.x = (w0 & 1u) ? T(1) : T(-1);
            a.y = (w1 & 1u) ? T(1) : T(-1);
            b.x = (w0 & 2u) ? T(1) : T(-1);
            b.y = (w1 & 2u) ? T(1) : T(-1);
            dst[2 * k] = a;
            dst[2 * k + 1] = b;
        }
    }
}

template <typename V>
__device__ __forceinline__ void zero_bins(V *h, int nb)
{
    for (int i = threadIdx.x; i < nb; i += blockDim.x) h[i] = V(0);
    __syncthreads();
}

template <typename V>
__device__ __forceinline__ void flush_bins(const V *h, V *global, int nb)
{
    __syncthreads();
    for (int i = threadIdx.x; i < nb; i += blockDim.x)
        if (h[i] != V(0)) atomicAdd(&global[i], h[i]);
}

// v added to a bin in shared memory.  A 64-bit integer bin is two 32-bit words and the carry is taken
// from the first word's old value: native 32-bit atomics, where a 64-bit one is a compare-and-swap loop.
__device__ __forceinline__ void bin_add(unsigned long long *bin, unsigned long long v)
{
    uint32_t *w = reinterpret_cast<uint32_t *>(bin);
    const uint32_t lo = (uint32_t)v, old = atomicAdd(w, lo);
    const uint32_t hi = (uint32_t)(v >> 32) + (uint32_t)(old + lo < old);
    if (hi) atomicAdd(w + 1, hi);
}

template <typename V>
struct BinRun {
    V *hist;
    V sum = V(0);
    int bin = -1;
    __device__ __forceinline__ void add(int b, V v)
    {
        if (b != bin) {
            if (bin >= 0) bin_add(&hist[bin], sum);
            bin = b;
            sum = v;
        } else {
            sum += v;
        }
    }
    __device__ __forceinline__ void flush()
    {
        if (bin >= 0) bin_add(&hist[bin], sum);
        bin = -1;
    }
};

// Rows (+-dy, +-dz) of one fold: n of them, row indices y + L z.
struct FoldRows {
    int n;
    int row[4];
};
__device__ __forceinline__ FoldRows fold_rows(int L, int dy, int dz)
{
    const int yb = (dy == 0 || 2 * dy == L) ? -1 : L - dy, zb = (dz == 0 || 2 * dz == L) ? -1 : L - dz;
    FoldRows f;
    f.n = (yb < 0 ? 1 : 2) * (zb < 0 ? 1 : 2);
    f.row[0] = dy + L * dz;
    f.row[1] = yb >= 0 ? yb + L * dz : dy + L * zb;
    f.row[2] = dy + L * zb;
    f.row[3] = yb + L * zb;
    return f;
}

// Calls fn(rows, x, D) for every fold of the CTA's share, x = thread (0 .. L/2, and past it up to a whole
// warp), and end() after each run of folds.  A work item is `chunk` folds: for SHORT along the smaller
// of dy and dz (fewer changes of bin), else along dy, which keeps rows that are also written next to
// each other (k_power is slower by a fifth along the smaller one).
template <bool SHORT, class Fn, class End>
__device__ __forceinline__ void fold_walk(int L, int chunk, Fn fn, End end)
{
    const int H = L / 2, nc = H / chunk + 1, per = SHORT ? 2 * nc : nc;
    for (int item = blockIdx.x; item < (H + 1) * per; item += gridDim.x) {
        const int M = item / per, rest = item - M * per;
        const bool ymajor = SHORT && rest >= nc;  // y the larger (strictly), else z
        const int m0 = (rest - (ymajor ? nc : 0)) * chunk;
        const int m1 = min(!SHORT ? H + 1 : (ymajor ? M : M + 1), m0 + chunk);
        if (m0 >= m1) continue;
        for (int x = threadIdx.x; (x & ~31) <= H; x += blockDim.x) {
#pragma unroll 2
            for (int m = m0; m < m1; ++m)
                fn(ymajor ? fold_rows(L, M, m) : fold_rows(L, m, M), x, x * x + m * m + M * M);
            end();
        }
    }
}

// Sum of four run sums in double.
template <typename T>
__device__ __forceinline__ double sum4(const T (&v)[4])
{
    return ((double)v[0] + (double)v[1]) + ((double)v[2] + (double)v[3]);
}

// 3. |F|^2 per mode of the half spectrum; S sums per bin; (P, 0) written back.
template <typename T>
__global__ void __launch_bounds__(RAD_FOLD_THREADS) k_power(typename Cx<T>::type *F, int L, int chunk, int nb,
                                                             double *sumS)
{
    extern __shared__ double hs[];
    zero_bins(hs, nb);
    const int H = L / 2, H1 = H + 1;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    fold_walk<false>(
        L, chunk,
        [&](const FoldRows &r, int x, int D) {
            const bool in = x <= H;
            T v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                v[i] = T(0);
                if (i < r.n && in) {
                    typename Cx<T>::type *p = F + (int64_t)r.row[i] * H1 + x;
                    const typename Cx<T>::type f = *p;
                    const T q = f.x * f.x + f.y * f.y;
                    v[i] = (x == 0 || x == H) ? q : T(2) * q;  // 0 < x < L/2: also the partner -q
                    typename Cx<T>::type o;
                    o.x = q;
                    o.y = T(0);
                    *p = o;
                }
            }
            // runs of equal bins among the 32 lanes; single precision stays in fp32 up to a run's sum
            const int b = in ? bin_of(D) : -1;
            const int bp = __shfl_up_sync(FULL, b, 1);
            const unsigned heads = __ballot_sync(FULL, lane == 0 || bp != b);
            const int start = 31 - __clz(heads & (FULL >> (31 - lane)));  // first lane of this lane's run
#pragma unroll
            for (int d = 1; d < 32; d <<= 1)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const T w = __shfl_up_sync(FULL, v[i], d);
                    if (lane - d >= start) v[i] += w;
                }
            const bool last = lane == 31 || ((heads >> (lane + 1)) & 1u);
            if (last && in) atomicAdd(&hs[b], sum4(v));
        },
        [] {});
    flush_bins(hs, sumS, nb);
}

// 5. G(k) = rint(g/N) per lag, summed per bin in int64.  SMALL: N <= 2^27, so eight values' sum stays
// within 32 bits.
template <typename T, bool SMALL>
__global__ void __launch_bounds__(RAD_FOLD_THREADS) k_radial_corr(const T *g, int L, int chunk, int64_t P, int nb,
                                                                   double invN, unsigned long long *sumG,
                                                                   unsigned long long *inexact)
{
    extern __shared__ unsigned long long hg[];
    zero_bins(hg, nb);
    const int H = L / 2;
    unsigned long long bad = 0ull;
    BinRun<unsigned long long> run{hg};
    fold_walk<true>(
        L, chunk,
        [&](const FoldRows &r, int x, int D) {
            if (x > H) return;
            const int xr = (x == 0 || x == H) ? -1 : L - x;
            T f[8];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (i < r.n) f[i] = g[(int64_t)r.row[i] * P + x];
                if (i < r.n && xr >= 0) f[4 + i] = g[(int64_t)r.row[i] * P + xr];
            }
            unsigned long long G = 0ull;
            int G32 = 0;
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if ((i & 3) < r.n && (i < 4 || xr >= 0)) {
                    const T v = f[i] * (T)invN;
                    const T q = rint(v);
                    if (fabs(v - q) > T(0.25)) ++bad;
                    // two's complement: the unsigned sums wrap to the signed result
                    if (SMALL) G32 += (int)q;
                    else G += (fabs(q) < T(2147483520)) ? (unsigned long long)(long long)(int)q
                                                   : (unsigned long long)(long long)q;
                }
            run.add(bin_of(D), SMALL ? (unsigned long long)(long long)G32 : G);
        },
        [&]() { run.flush(); });
    flush_bins(hg, sumG, nb);
    if (bad) atomicAdd(inexact, bad);
}

// Vectors per bin (independent of the state; once per context).
__global__ void __launch_bounds__(RAD_FOLD_THREADS) k_radial_count(int L, int chunk, int nb, unsigned long long *count)
{
    extern __shared__ unsigned long long hc[];
    zero_bins(hc, nb);
    const int H = L / 2;
    BinRun<unsigned long long> run{hc};
    fold_walk<true>(
        L, chunk,
        [&](const FoldRows &r, int x, int D) {
            if (x <= H) run.add(bin_of(D), (unsigned long long)(r.n * ((x == 0 || x == H) ? 1 : 2)));
        },
        [&]() { run.flush(); });
    flush_bins(hc, count, nb);
}

// 6. out = [C(0..nb-1), S(0..nb-1), l]; cnt = [n_b (nb), inexact lags].
__global__ void k_radial_finish(int L, int nb, double c, const unsigned long long *sumG, const double *sumS,
                                const unsigned long long *count, const unsigned long long *inexact, double *out,
                                int64_t *cnt)
{
    const double N = (double)L * (double)L * (double)L;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
        const double denom = __dmul_rn(N, (double)count[b]);
        out[b] = count[b] ? __ddiv_rn((double)(long long)sumG[b], denom) : 0.0;
        out[nb + b] = count[b] ? __ddiv_rn(sumS[b], denom) : 0.0;
        cnt[b] = (int64_t)count[b];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double ell = __longlong_as_double(0x7ff8000000000000ll);  // NaN: no crossing
        for (int r = 0; r < L / 2; ++r) {
            const double c0 = out[r], c1 = out[r + 1];
            if (c0 >= c && c > c1) {
                ell = __dadd_rn((double)r, __ddiv_rn(__dsub_rn(c0, c), __dsub_rn(c0, c1)));
                break;
            }
        }
        out[2 * nb] = ell;
        cnt[nb] = (int64_t)*inexact;
    }
}

// ---------------------------------------------------------------------------------
struct RadialPlans {
    int L = 0;
    bool made[2] = {false, false};
    cufftHandle fwd[2] = {0, 0}, inv[2] = {0, 0};
    size_t work[2] = {0, 0};
    char *buf = nullptr;  // transform buffer (grown to the largest precision used)
    size_t buf_bytes = 0;
    char *wk = nullptr;   // cuFFT work area
    size_t wk_bytes = 0;
    unsigned long long *count = nullptr;  // vectors per bin (counted at the first call)
    char *acc = nullptr;                  // per-call sums: sumG, sumS, inexact
};

RadialPlans *radial_plans_create() { return new (std::nothrow) RadialPlans(); }

void radial_release(RadialPlans *p, cudaStream_t s)
{
    if (!p) return;
    if (p->buf) cudaFreeAsync(p->buf, s);
    if (p->wk) cudaFreeAsync(p->wk, s);
    p->buf = p->wk = nullptr;
    p->buf_bytes = p->wk_bytes = 0;
}

void radial_plans_destroy(RadialPlans *p, cudaStream_t s)
{
    if (!p) return;
    radial_release(p, s);
    if (p->count) cudaFreeAsync(p->count, s);
    if (p->acc) cudaFreeAsync(p->acc, s);
    for (int i = 0; i < 2; ++i)
        if (p->made[i]) {
            cufftDestroy(p->fwd[i]);
            cufftDestroy(p->inv[i]);
        }
    delete p;
}

static int make_plans(RadialPlans *p, int L, int prec)
{
    if (p->made[prec]) return CUFFT_SUCCESS;
    long long n[3] = {L, L, L};
    size_t w1 = 0, w2 = 0;
    cufftResult r;
    if ((r = cufftCreate(&p->fwd[prec])) != CUFFT_SUCCESS) return r;
    if ((r = cufftCreate(&p->inv[prec])) != CUFFT_SUCCESS) {
        cufftDestroy(p->fwd[prec]);
        return r;
    }
    cufftSetAutoAllocation(p->fwd[prec], 0);
    cufftSetAutoAllocation(p->inv[prec], 0);
    r = cufftMakePlanMany64(p->fwd[prec], 3, n, nullptr, 1, 0, nullptr, 1, 0, prec ? CUFFT_D2Z : CUFFT_R2C, 1, &w1);
    if (r == CUFFT_SUCCESS)
        r = cufftMakePlanMany64(p->inv[prec], 3, n, nullptr, 1, 0, nullptr, 1, 0, prec ? CUFFT_Z2D : CUFFT_C2R, 1,
                                &w2);
    if (r != CUFFT_SUCCESS) {
        cufftDestroy(p->fwd[prec]);
        cufftDestroy(p->inv[prec]);
        return r;
    }
    p->L = L;
    p->work[prec] = std::max(w1, w2);
    p->made[prec] = true;
    return CUFFT_SUCCESS;
}

size_t radial_scratch_bytes(int L, int prec)
{
    const size_t elem = prec ? sizeof(double) : sizeof(float);
    return (size_t)L * (size_t)L * (size_t)(L / 2 + 1) * 2 * elem;
}

// Grow a cached device allocation to at least `bytes` (stream-ordered).
static cudaError_t ensure(char **ptr, size_t *have, size_t bytes, cudaStream_t s)
{
    if (*have >= bytes && (*ptr || bytes == 0)) return cudaSuccess;
    if (*ptr) cudaFreeAsync(*ptr, s);
    *ptr = nullptr;
    *have = 0;
    if (bytes == 0) return cudaSuccess;
    cudaError_t e = cudaMallocAsync((void **)ptr, bytes, s);
    if (e != cudaSuccess) {
        *ptr = nullptr;
        return e;
    }
    *have = bytes;
    return cudaSuccess;
}

template <typename T>
static cudaError_t run_radial(RadialPlans *p, const uint32_t *lat_r, int L, double c, double *out, int64_t *cnt,
                              cudaStream_t s, int64_t *launches, int *cufft_status)
{
    constexpr int prec = sizeof(T) == 8 ? 1 : 0;
    const Geom g = make_geom(L);
    const int nb = (int)radial_nbins(L);
    const int64_t P = 2 * (int64_t)(L / 2 + 1);
    int cs = make_plans(p, L, prec);
    if (cs != CUFFT_SUCCESS) {
        *cufft_status = cs;
        return cudaErrorUnknown;
    }
    cudaError_t e;
    if ((e = ensure(&p->buf, &p->buf_bytes, radial_scratch_bytes(L, prec), s)) != cudaSuccess) return e;
    if ((e = ensure(&p->wk, &p->wk_bytes, p->work[prec], s)) != cudaSuccess) return e;
    const size_t acc_bytes = (size_t)nb * 2 * sizeof(double) + 64;
    if (!p->acc && (e = cudaMallocAsync((void **)&p->acc, acc_bytes, s)) != cudaSuccess) {
        p->acc = nullptr;
        return e;
    }
    unsigned long long *sumG = reinterpret_cast<unsigned long long *>(p->acc);
    double *sumS = reinterpret_cast<double *>(p->acc) + nb;
    unsigned long long *inexact = reinterpret_cast<unsigned long long *>(p->acc) + 2 * nb;
    if ((e = cudaMemsetAsync(p->acc, 0, acc_bytes, s)) != cudaSuccess) return e;
    int dev = 0, sms = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    // threads for x = 0 .. L/2 in as few passes as 544 allow; folds per work item so that there are a
    // few items per resident CTA
    const int nx = L / 2 + 1, passes = (nx + RAD_FOLD_THREADS - 1) / RAD_FOLD_THREADS;
    const int fold_threads = ((nx + passes - 1) / passes + 31) / 32 * 32;
    const unsigned grid = (unsigned)(sms * std::max(1, 2048 / fold_threads));
    const int chunk = std::max(1, std::min(16, nx * nx / (4 * (int)grid)));
    const size_t smem = (size_t)nb * sizeof(double);  // 28 KB at L = 4096: within the default limit
    if (!p->count) {
        if ((e = cudaMallocAsync((void **)&p->count, sizeof(unsigned long long) * nb, s)) != cudaSuccess) {
            p->count = nullptr;
            return e;
        }
        if ((e = cudaMemsetAsync(p->count, 0, sizeof(unsigned long long) * nb, s)) != cudaSuccess) return e;
        k_radial_count<<<grid, fold_threads, smem, s>>>(L, chunk, nb, p->count);
        if (launches) *launches += 1;
    }

    k_unpack_real<T><<<(unsigned)(sms * 16), RAD_THREADS, 0, s>>>(lat_r, reinterpret_cast<T *>(p->buf), g, P);
    cufftHandle f = p->fwd[prec], iv = p->inv[prec];
    if ((cs = cufftSetStream(f, s)) != CUFFT_SUCCESS || (cs = cufftSetStream(iv, s)) != CUFFT_SUCCESS ||
        (cs = cufftSetWorkArea(f, p->wk)) != CUFFT_SUCCESS || (cs = cufftSetWorkArea(iv, p->wk)) != CUFFT_SUCCESS) {
        *cufft_status = cs;
        return cudaErrorUnknown;
    }
    using C = typename Cx<T>::type;
    if (prec)
        cs = cufftExecD2Z(f, reinterpret_cast<cufftDoubleReal *>(p->buf), reinterpret_cast<cufftDoubleComplex *>(p->buf));
    else
        cs = cufftExecR2C(f, reinterpret_cast<cufftReal *>(p->buf), reinterpret_cast<cufftComplex *>(p->buf));
    if (cs != CUFFT_SUCCESS) {
        *cufft_status = cs;
        return cudaErrorUnknown;
    }
    k_power<T><<<grid, fold_threads, smem, s>>>(reinterpret_cast<C *>(p->buf), L, chunk, nb, sumS);
    if (prec)
        cs = cufftExecZ2D(iv, reinterpret_cast<cufftDoubleComplex *>(p->buf), reinterpret_cast<cufftDoubleReal *>(p->buf));
    else
        cs = cufftExecC2R(iv, reinterpret_cast<cufftComplex *>(p->buf), reinterpret_cast<cufftReal *>(p->buf));
    if (cs != CUFFT_SUCCESS) {
        *cufft_status = cs;
        return cudaErrorUnknown;
    }
    const double invN = 1.0 / ((double)L * (double)L * (double)L);  // exact where L is a power of two
    auto corr = (int64_t)L * L * L <= (1 << 27) ? k_radial_corr<T, true> : k_radial_corr<T, false>;
    corr<<<grid, fold_threads, smem, s>>>(reinterpret_cast<const T *>(p->buf), L, chunk, P, nb, invN, sumG, inexact);
    k_radial_finish<<<1, 256, 0, s>>>(L, nb, c, sumG, sumS, p->count, inexact, out, cnt);
    if (launches) *launches += 4;  // own kernels; the two cuFFT executions are library launches
    return cudaGetLastError();
}

cudaError_t launch_radial(RadialPlans *p, const uint32_t *lat_r, int L, int precision, double c, double *out,
                          int64_t *cnt, cudaStream_t s, int64_t *launches, int *cufft_status)
{
    *cufft_status = CUFFT_SUCCESS;
    if (precision)
        return run_radial<double>(p, lat_r, L, c, out, cnt, s, launches, cufft_status);
    return run_radial<float>(p, lat_r, L, c, out, cnt, s, launches, cufft_status);
}

}  // namespace ising
