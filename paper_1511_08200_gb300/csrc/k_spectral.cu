// k_spectral.cu -- coarsest-grid solve for periodic coarsest grids of more than 6^3 cells.
//
// A grid side N = 2^a m with m odd stops halving at 2m (the 8-child restriction needs
// even sides), so N = 144, 176, 208, 240 end on coarsest grids of 18^3 .. 30^3 where
// Gauss-Seidel alone needs hundreds of sweeps to reduce the residual 1e-3 (the coarsest
// solve of Sec. 3.1's multigrid).  Here each iteration computes the residual
// r = f + c - op(v) (c = minus its mean, the compatibility constant), solves L d = r for
// the periodic 7-point Laplacian exactly -- separable discrete Fourier transforms, d_hat =
// r_hat / lambda(k), the mean mode dropped -- adds d to v, and smooths with two red-black
// sweeps.  L is the linear part of the operator, so the correction removes the smooth
// error the sweeps cannot, and the sweeps the local nonlinear part.  A fixed number of
// iterations keeps the launch sequence fixed (the same in captured graphs).  Multi-CTA
// kernels: the grid is at most 32^3.
#include "mg5_fin.cuh"

namespace mg5 {

template <typename T>
struct Cplx;
template <>
struct Cplx<double> {
    using type = double2;
};
template <>
struct Cplx<float> {
    using type = float2;
};

__device__ __forceinline__ void sincos_pi(double x, double *s, double *c) { sincospi(x, s, c); }
__device__ __forceinline__ void sincos_pi(float x, float *s, float *c) { sincospif(x, s, c); }

// r = f + c - op(v) into the real parts (imaginary parts 0); block partial sums of (r, r^2);
// each call counts the two sweeps of its iteration.
template <typename T, bool BASE>
__global__ void k_spec_residual(const T *__restrict__ v, const T *__restrict__ f,
                                const double *__restrict__ cptr, int n, CoefT<T> cf,
                                const T *__restrict__ B, typename Cplx<T>::type *__restrict__ out,
                                Moments *__restrict__ partials, int *sweeps, Fin fin)
{
    const int n3 = n * n * n;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    MomAcc<T> acc;
    if (t < n3) {
        const int k = t % n, j = (t / n) % n, i = t / (n * n);
        const Rows r = periodic_rows(n, i, j);
        const int kp = (k == n - 1) ? 0 : k + 1, km = (k == 0) ? n - 1 : k - 1;
        St<T> s, sb;
        gather(v, v, r, k, kp, km, s);
        if constexpr (BASE)
            gather(B, B, r, k, kp, km, sb);
        const T res = resid_of<T, BASE>(s, sb, MG5_AT(f, t) + (T)(MG5_AT(cptr, 0)), cf);
        MG5_AT(out, t).x = res;
        MG5_AT(out, t).y = (T)0;
        acc.add(res);
    }
    const Moments m = block_moments(acc);
    if (threadIdx.x == 0) {
        MG5_AT(partials, blockIdx.x) = m;
        if (blockIdx.x == 0 && sweeps)
            atomicAdd(&MG5_AT(sweeps, 0), 2);
    }
    finalize_if_last(reinterpret_cast<double2 *>(partials), fin);   // c -= mean r
}

// cos and sin of 2 pi q / n, q = 0 .. n - 1, once per block: an FP64 sincospi is ~50 FP64
// instructions (2 lanes a clock per SM), and one a term made an 18^3 transform along one axis take
// 68 us; with the table, and blocks small enough that its warps reach every SM, 9.2 us (FP32, 30^3:
// 11.4 -> 4.5 us).  What is left is the chain of 2 x 18 FP64 multiply-adds of each output.
constexpr int kDftMax = 32;   // largest coarsest side
template <typename T>
__device__ __forceinline__ void dft_table(int n, T *cs, T *sn)
{
    for (int q = threadIdx.x; q < n; q += blockDim.x)
        sincos_pi((T)(2 * q) / (T)n, &MG5_AT(sn, q), &MG5_AT(cs, q));
    __syncthreads();
}

// One-dimensional DFT along `axis` (0: i, 1: j, 2: k) of every line:
// out[m'] = sum_m in[m] exp(-+ 2 pi i m m' / n) (sign: forward -, inverse +).  With `addto`,
// the real part times `scale` is added to it instead of writing `out`.
// DIVIDE (the last forward axis): the result is divided by the eigenvalue of the periodic 7-point
// Laplacian, lambda = (2 cos 2 pi kx/n + 2 cos 2 pi ky/n + 2 cos 2 pi kz/n - 6) / h^2; the mean mode
// becomes zero.
template <typename T, bool DIVIDE>
__global__ void k_dft_axis(const typename Cplx<T>::type *__restrict__ in,
                           typename Cplx<T>::type *__restrict__ out, int n, int axis, int inverse,
                           T *__restrict__ addto, T scale, T h2)
{
    __shared__ T cs[kDftMax], sn[kDftMax];
    dft_table<T>(n, cs, sn);
    const int n3 = n * n * n;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n3)
        return;
    const int k = t % n, j = (t / n) % n, i = t / (n * n);
    const int mo = axis == 0 ? i : (axis == 1 ? j : k);
    const int stride = axis == 0 ? n * n : (axis == 1 ? n : 1);
    const int base = t - mo * stride;
    const T sgn = inverse ? (T)1 : (T)-1;
    T re = 0, im = 0;
    for (int m = 0, q = 0; m < n; ++m) {   // q = m mo mod n
        const T s = MG5_AT(sn, q) * sgn, c = MG5_AT(cs, q);
        const typename Cplx<T>::type a = MG5_AT(in, base + m * stride);
        re += a.x * c - a.y * s;
        im += a.x * s + a.y * c;
        q += mo;
        q = q >= n ? q - n : q;
    }
    if constexpr (DIVIDE) {
        const T inv = t == 0 ? (T)0 : h2 / ((T)2 * (MG5_AT(cs, i) + MG5_AT(cs, j) + MG5_AT(cs, k)) - (T)6);
        re *= inv;
        im *= inv;
    }
    if (addto) {
        MG5_AT(addto, t) += re * scale;
    } else {
        MG5_AT(out, t).x = re;
        MG5_AT(out, t).y = im;
    }
}

template <typename T>
cudaError_t launch_coarsest_spectral(T *v, T *tmp, const T *f, int n, CoefT<T> cf, LevelScal *ls,
                                     int iters, unsigned long long *clamp, int *sweeps,
                                     double2 *partials, void *w0v, void *w1v, cudaStream_t st,
                                     const T *B)
{
    using C = typename Cplx<T>::type;
    C *w0 = static_cast<C *>(w0v), *w1 = static_cast<C *>(w1v);
    const int n3 = n * n * n;
    const int bs = block_spread(n3), g = grid_spread(n3);   // warps over all SMs
    if (g > kMomentBlocks || n > kDftMax)
        return cudaErrorInvalidValue;
    Moments *mp = reinterpret_cast<Moments *>(partials);
    const T inv_n3 = (T)1 / (T)n3;
    for (int it = 0; it < iters; ++it) {
        const Fin fin{ls, FIN_RESID, (double)n3};
        if (B)
            k_spec_residual<T, true><<<g, bs, 0, st>>>(v, f, &ls->c, n, cf, B, w0, mp, sweeps, fin);
        else
            k_spec_residual<T, false><<<g, bs, 0, st>>>(v, f, &ls->c, n, cf, B, w0, mp, sweeps, fin);
        count_launch(1);
        cudaError_t e;
        k_dft_axis<T, false><<<g, bs, 0, st>>>(w0, w1, n, 2, 0, nullptr, (T)0, (T)0);
        k_dft_axis<T, false><<<g, bs, 0, st>>>(w1, w0, n, 1, 0, nullptr, (T)0, (T)0);
        k_dft_axis<T, true><<<g, bs, 0, st>>>(w0, w1, n, 0, 0, nullptr, (T)0, cf.h2);
        k_dft_axis<T, false><<<g, bs, 0, st>>>(w1, w0, n, 0, 1, nullptr, (T)0, (T)0);
        k_dft_axis<T, false><<<g, bs, 0, st>>>(w0, w1, n, 1, 1, nullptr, (T)0, (T)0);
        k_dft_axis<T, false><<<g, bs, 0, st>>>(w1, w0, n, 2, 1, v, inv_n3, (T)0);   // v += Re(d)
        count_launch(6);
        if ((e = cudaGetLastError()) != cudaSuccess)
            return e;
        e = launch_sweep<T>(v, tmp, f, &ls->c, n, cf, clamp, st, B);
        if (e == cudaSuccess)
            e = launch_sweep<T>(tmp, v, f, &ls->c, n, cf, clamp, st, B);
        if (e != cudaSuccess)
            return e;
    }
    return cudaSuccess;
}

template cudaError_t launch_coarsest_spectral<double>(double *, double *, const double *, int,
                                                      CoefT<double>, LevelScal *, int,
                                                      unsigned long long *, int *, double2 *, void *,
                                                      void *, cudaStream_t, const double *);
template cudaError_t launch_coarsest_spectral<float>(float *, float *, const float *, int,
                                                     CoefT<float>, LevelScal *, int,
                                                     unsigned long long *, int *, double2 *, void *,
                                                     void *, cudaStream_t, const float *);

}  // namespace mg5
