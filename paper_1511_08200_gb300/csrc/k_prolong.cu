// k_prolong.cu -- the cell-centred trilinear prolongation of a coarse grid's correction on larger
// grids, as tiles: v += P (vc - v0c), weights (3/4, 1/4) per axis as 3 x + y and one 1/64 at the end.
//
// A CTA takes TI x 8 x 32 coarse cells.  It forms the differences e = vc - v0c of these cells and their
// halo once, in shared memory; each thread then marches its coarse column over the TI planes, forms the
// k- and j-stages of a plane once (nine shared loads) and keeps them for the three planes that use them.
//
// FP64: the correction travels as integers.  GB300 runs FP64 at 2 lanes a clock per SM, and the gather
// kernel's 9 FP64 operations a fine cell, or 4.4 of a march along i, set their time (40 us for 64^3 ->
// 128^3, 185 for 128^3 -> 256^3).  Here the largest |e| of the tile gives a common exponent, each e becomes
// a multiple of 2^-56 of it (the e below keep what lies above that), the stages are exact 64-bit integer
// multiply-adds, and only the difference and the final sum with v are FP64: 1.2 operations a fine cell.  The
// correction is off by at most 1.3e-16 of the tile's largest difference (seven FP64 multiply-adds round
// by as much where the differences are of a size; a cell whose own are far smaller loses more than FP64
// would, 2^-56 of the largest), and a correction is itself corrected by the next cycle.  A tile whose largest
// |e| is not finite, zero or below 2^-900 takes the FP64 operations of the gather kernel.
// Now 11.0 us (64^3 -> 128^3), 19 (72^3 -> 144^3, was 57) and 70 (128^3 -> 256^3).  In FP32 120^3 -> 240^3
// 53 -> 23 us, 256^3 -> 512^3 258 -> 188.  Four planes a CTA below 96^3 coarse cells, where eight would
// leave SMs without one.
//
// FP32: the operations of the gather kernel in the same order, equal to it to the bit.
#include "mg5_kernels.cuh"

namespace mg5 {

namespace {

constexpr int PT_J = 8, PT_K = 32;               // coarse tile (j, k)
constexpr int PT_THREADS = PT_J * PT_K;          // a coarse column a thread
constexpr int PT_RJ = PT_J + 2, PT_RK = PT_K + 2;
constexpr int PT_PL = PT_RJ * PT_RK;             // cells of a plane with its halo

template <typename T>
struct Elem;
template <>
struct Elem<float> {
    using E = float;        // a difference in shared memory
    using V = float2;       // two fine cells
};
template <>
struct Elem<double> {
    using E = long long;
    using V = double2;
};

__device__ __forceinline__ float three(float x, float y) { return fmaf(3.0f, x, y); }
__device__ __forceinline__ double three(double x, double y) { return fma(3.0, x, y); }
__device__ __forceinline__ long long three(long long x, long long y) { return 3 * x + y; }

// a double as a multiple of 2^(E - 1078), E >= its exponent field (truncated)
__device__ __forceinline__ long long to_fixed(double x, int E)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int d = E - (int)((b >> 52) & 0x7ff);
    const unsigned long long m = ((b & 0xfffffffffffffull) | 0x10000000000000ull) << 3;
    const long long t = d < 60 ? (long long)(m >> d) : 0ll;
    return (long long)b < 0 ? -t : t;
}

// o 2^(E - 1084) as a double, |o| < 2^62, E in [124, 2046]: truncated to 53 bits
__device__ __forceinline__ double from_fixed(long long o, int E)
{
    const unsigned long long a = (unsigned long long)(o < 0 ? -o : o);
    if (a == 0)
        return 0.0;
    const int lz = __clzll((long long)a);
    const unsigned long long m = (a << lz) >> 11;   // bit 52 set
    // 2^(63 - lz) 2^(E - 1084): the exponent field E + 2 - lz, of which bit 52 of m adds one
    const unsigned long long r = m + ((unsigned long long)(E + 1 - lz) << 52);
    return __longlong_as_double((long long)(r | ((unsigned long long)o & 0x8000000000000000ull)));
}

// the k- and j-stages of a plane at (row j, column k) of the tile with its halo
template <typename A, typename L>
__device__ __forceinline__ void stages(const L &at, A y[2][2])
{
    A Z[3][2];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        const A e0 = at(b, 0), e1 = at(b, 1), e2 = at(b, 2);
        Z[b][0] = three(e1, e0);
        Z[b][1] = three(e1, e2);
    }
#pragma unroll
    for (int cj = 0; cj < 2; ++cj)
#pragma unroll
        for (int ck = 0; ck < 2; ++ck)
            y[cj][ck] = three(Z[1][ck], Z[cj ? 2 : 0][ck]);
}

__device__ __forceinline__ float add_part(float v, float o, int) { return fmaf(o, 1.0f / 64.0f, v); }
__device__ __forceinline__ double add_part(double v, double o, int) { return fma(o, 1.0 / 64.0, v); }
__device__ __forceinline__ double add_part(double v, long long o, int E) { return v + from_fixed(o, E); }

// planes I0 .. I0 + TI - 1 of the thread's coarse column: AT(plane of the tile, j, k) -> A
template <typename T, typename A, int TI, typename L>
__device__ __forceinline__ void march(const L &at, T *__restrict__ vf, int I0, int J, int K, int nc, int E)
{
    using V = typename Elem<T>::V;
    const int n = 2 * nc;
    A ym[2][2], y0[2][2], yp[2][2];
    stages([&](int b, int c) { return at(0, b, c); }, ym);
    stages([&](int b, int c) { return at(1, b, c); }, y0);
#pragma unroll
    for (int p = 0; p < TI; ++p) {
        if (I0 + p >= nc)
            break;
        V v[2][2];
        V *at_f[2][2];
#pragma unroll
        for (int ci = 0; ci < 2; ++ci)
#pragma unroll
            for (int cj = 0; cj < 2; ++cj) {
                at_f[ci][cj] = &MG5_AT(
                    reinterpret_cast<V *>(vf + ((long long)(2 * (I0 + p) + ci) * n + (2 * J + cj)) * n + 2 * K), 0);
                v[ci][cj] = *at_f[ci][cj];
            }
        stages([&](int b, int c) { return at(p + 2, b, c); }, yp);
#pragma unroll
        for (int ci = 0; ci < 2; ++ci)
#pragma unroll
            for (int cj = 0; cj < 2; ++cj) {
                v[ci][cj].x = add_part(v[ci][cj].x, three(y0[cj][0], ci ? yp[cj][0] : ym[cj][0]), E);
                v[ci][cj].y = add_part(v[ci][cj].y, three(y0[cj][1], ci ? yp[cj][1] : ym[cj][1]), E);
                *at_f[ci][cj] = v[ci][cj];
            }
#pragma unroll
        for (int cj = 0; cj < 2; ++cj)
#pragma unroll
            for (int ck = 0; ck < 2; ++ck) {
                ym[cj][ck] = y0[cj][ck];
                y0[cj][ck] = yp[cj][ck];
            }
    }
}

template <typename T, int TI>
__global__ void __launch_bounds__(PT_THREADS)
    k_prolong_tile(const T *__restrict__ vc, const T *__restrict__ v0c, int nc, T *__restrict__ vf,
                   double *c_fine, const double *c_coarse)
{
    using E = typename Elem<T>::E;
    constexpr int CELLS = (TI + 2) * PT_PL, PER = (CELLS + PT_THREADS - 1) / PT_THREADS;
    __shared__ E S[CELLS];
    __shared__ unsigned top_s[PT_THREADS / 32];
    const int tid = threadIdx.x;
    const int K0 = blockIdx.x * PT_K, J0 = blockIdx.y * PT_J, I0 = blockIdx.z * TI;
    if (blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && tid == 0 && c_fine && c_coarse)
        MG5_AT(c_fine, 0) += MG5_AT(c_coarse, 0);
    // the differences (periodic; 2 nc > PT_K, so an index is at most one period out)
    T e[PER];
    unsigned top = 0;   // largest high word of |e|
#pragma unroll
    for (int m = 0; m < PER; ++m) {
        const int q = tid + m * PT_THREADS;
        e[m] = (T)0;
        if (q < CELLS) {
            const int pl = q / PT_PL, r = q - pl * PT_PL, j = r / PT_RK, k = r - j * PT_RK;
            const auto wrap = [&](int x) { return x < 0 ? x + nc : (x >= nc ? x - nc : x); };
            const long long o = ((long long)wrap(I0 + pl - 1) * nc + wrap(J0 + j - 1)) * nc + wrap(K0 + k - 1);
            e[m] = v0c ? MG5_AT(vc, o) - MG5_AT(v0c, o) : MG5_AT(vc, o);
        }
    }
    int ex = 0;
    bool fixed = false;
    if constexpr (sizeof(T) == 8) {
#pragma unroll
        for (int m = 0; m < PER; ++m)
            top = max(top, (unsigned)__double2hiint(e[m]) & 0x7fffffffu);
        top = __reduce_max_sync(0xffffffffu, top);
        if ((tid & 31) == 0)
            top_s[tid >> 5] = top;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < PT_THREADS / 32; ++w)
            top = max(top, top_s[w]);
        ex = (int)(top >> 20);
        fixed = ex >= 124 && ex < 0x7ff;
#pragma unroll
        for (int m = 0; m < PER; ++m)
            if (tid + m * PT_THREADS < CELLS)
                MG5_AT(S, tid + m * PT_THREADS) = fixed ? to_fixed(e[m], ex) : __double_as_longlong(e[m]);
    } else {
#pragma unroll
        for (int m = 0; m < PER; ++m)
            if (tid + m * PT_THREADS < CELLS)
                MG5_AT(S, tid + m * PT_THREADS) = e[m];
    }
    __syncthreads();
    const int j = tid / PT_K, k = tid - j * PT_K, J = J0 + j, K = K0 + k;
    if (J >= nc || K >= nc)
        return;
    const E *base = S + j * PT_RK + k;
    const auto at = [&](int pl, int b, int c) { return MG5_AT(base, pl * PT_PL + b * PT_RK + c); };
    if constexpr (sizeof(T) == 8) {
        if (!fixed) {
            march<T, double, TI>([&](int pl, int b, int c) { return __longlong_as_double(at(pl, b, c)); }, vf, I0, J, K,
                                 nc, 0);
            return;
        }
    }
    march<T, E, TI>(at, vf, I0, J, K, nc, ex);
}

}  // namespace

template <typename T>
cudaError_t launch_prolong_tile(const T *vc, const T *v0c, int nc, T *vf, double *c_fine,
                                const double *c_coarse, cudaStream_t st)
{
    if (2 * nc <= PT_K)
        return cudaErrorInvalidValue;
    const int gk = (nc + PT_K - 1) / PT_K, gj = (nc + PT_J - 1) / PT_J;
    if (nc >= 96)
        k_prolong_tile<T, 8><<<dim3(gk, gj, (nc + 7) / 8), PT_THREADS, 0, st>>>(vc, v0c, nc, vf, c_fine, c_coarse);
    else
        k_prolong_tile<T, 4><<<dim3(gk, gj, (nc + 3) / 4), PT_THREADS, 0, st>>>(vc, v0c, nc, vf, c_fine, c_coarse);
    count_launch(1);
    return cudaGetLastError();
}

template cudaError_t launch_prolong_tile<double>(const double *, const double *, int, double *, double *,
                                                 const double *, cudaStream_t);
template cudaError_t launch_prolong_tile<float>(const float *, const float *, int, float *, double *,
                                                const double *, cudaStream_t);

}  // namespace mg5
