// k_split.cu -- the FP64 half-sweep, residual and right-hand side of the larger grids in the
// split arithmetic of mg5_split.cuh: the FP64 solves' smoother, residual + restriction and FAS
// right-hand side (periodic grids and the finest grid of a refinement patch).
//
// What bounds them: the plain FP64 kernels sit at 84% of the FP64 pipe (2 lanes a clock per SM).
// In the split arithmetic a cell costs FP32 and integer instructions instead (~495 a cell updated at 256^3,
// ~370 a residual, half of them packed), and the bound becomes instruction issue (70% and 57% busy) with
// the shared-memory (50%) and FMA (50%) pipes near behind.  Measured on GB300, plain FP64 -> split:
// half-sweep 11.3 -> 5.5 us at 64^3, 64.4 -> 22.0 at 128^3, 500 -> 148 at 256^3; residual 26.6 ->
// 12.3, 132 -> 41.5 and 994 -> 257 us.
//
// A CTA takes a tile of 2 SUB x 8 x 32 cells as two half-tiles of SUB planes whose cells are
// computed as packed pairs; the exponent of the pieces is the tile's own.  It reads the tile and
// one cell around each half (10 rows of 34 values a plane, mostly L2 hits), finds the largest
// exponent, cuts every value into its pieces in shared memory once, and computes the cells from
// there.  The half-sweep keeps the two colours in separate arrays, so that the 16 active cells of
// a row are contiguous.  Half-tiles of 4 planes leave room for 3 or 4 CTAs an SM, whose loads and
// barriers overlap: with 8 planes and 2 CTAs a 256^3 half-sweep took 190 us, with the column's
// plane sums kept in registers a 128^3 residual 46 us.  The statistics stay in FP32 pairs until the
// thread's last tile: in FP64 per tile they took half of the FP64 pipe (333 -> 268 us at 256^3).
#include "mg5_fin.cuh"
#include "mg5_split.cuh"

namespace mg5 {

using namespace split;

namespace {

constexpr int TJ = 8, TK = 32;           // tile sides along j and k (k: a warp's row)
constexpr int NJ = TJ + 2, NK = TK + 2;  // with one cell on each side
constexpr int THREADS = 256, WARPS = THREADS / 32;

__device__ __forceinline__ int wrap1(int x, int n) { return x < 0 ? x + n : (x >= n ? x - n : x); }

// Offset of (i, j, 0), each from -1 to its side, in the stored array: the periodic grid (indices
// wrapped) or the box with its ghost shell.
template <bool BOX>
__device__ __forceinline__ long long row_at(int i, int j, int n0, int n1, int n2)
{
    if constexpr (BOX)
        return ((long long)(i + 1) * (n1 + 2) + (j + 1)) * (n2 + 2) + 1;
    else
        return ((long long)wrap1(i, n0) * n1 + wrap1(j, n1)) * n2;
}
// A cell's 19 values from global memory: faces from F, edges and the centre from E.
template <bool BOX>
__device__ __forceinline__ void gather_at(const double *F, const double *E, int i, int j, int k, int n0,
                                          int n1, int n2, St<double> &s)
{
    if constexpr (BOX)
        gather3(F, E, E, box_rows(n1 + 2, n2 + 2, i + 1, j + 1), k + 1, k + 2, k, s);
    else
        gather3(F, E, E, periodic_rows(n0, i, j), k, k == n2 - 1 ? 0 : k + 1, k == 0 ? n2 - 1 : k - 1, s);
}

__device__ __forceinline__ int exponent(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// The tile's common exponent from every thread's largest one, and whether the split arithmetic takes
// the tile, which it does not where all are 0 (every thread of the CTA must call it).
__device__ __forceinline__ bool tile_exponent(int mine, const Coef &cs, int *sm, int &eb, Kap &kap)
{
    mine = __reduce_max_sync(0xffffffffu, mine);
    if ((threadIdx.x & 31) == 0)
        sm[threadIdx.x >> 5] = mine;
    __syncthreads();
    eb = sm[0];
#pragma unroll
    for (int w = 1; w < WARPS; ++w)
        eb = max(eb, sm[w]);
    const bool in_range = eb >= kMinExp && eb <= kMaxExp;
    const float u = __int_as_float((in_range ? eb - kUnitBias + 127 : 127) << 23);
    kap = Kap{cs.k3h * u, cs.k3l * u, cs.kh * u, cs.kl * u};
    return cs.ok && in_range && kap.k3h <= kMaxKappa;
}

__device__ __forceinline__ P3 split_two(double a, double b, int eb)
{
    return split2((unsigned)__double2hiint(a), (unsigned)__double2loint(a), (unsigned)__double2hiint(b),
                  (unsigned)__double2loint(b), eb);
}
__device__ __forceinline__ Pair pair_two(double a, double b)
{
    Pair p;
    pair_words((unsigned)__double2hiint(a), (unsigned)__double2loint(a), p.h.x, p.l.x);
    pair_words((unsigned)__double2hiint(b), (unsigned)__double2loint(b), p.h.y, p.l.y);
    return p;
}
// x u as a double
__device__ __forceinline__ double unit_f64(float x, int eb)
{
    unsigned hi, lo;
    unit_words(x, eb, hi, lo);
    return __hiloint2double((int)hi, (int)lo);
}
__device__ __forceinline__ double pow2(int e) { return __hiloint2double((e + 1023) << 20, 0); }

// A tile's values in registers, the two half-tiles' side by side.  Of the ten rows of a plane warp w
// takes row w (a lane a cell, kk = 1 .. 32) on every plane, so that a plane's address is uniform;
// then the last two rows of all planes are dealt to the warps, and the rows' two ends to the threads.
template <int SUB>
struct TileRegs {
    static constexpr int PLANES = SUB + 2, EXTRA = (2 * PLANES + WARPS - 1) / WARPS;
    static constexpr int ENDS = (2 * NJ * PLANES + THREADS - 1) / THREADS;
    double a[PLANES + EXTRA + ENDS], b[PLANES + EXTRA + ENDS];

    // Position m: plane ii, row jj, column kk (false: none).
    static __device__ __forceinline__ bool at(int m, int &ii, int &jj, int &kk)
    {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        if (m < PLANES) {
            ii = m;
            jj = warp;
            kk = lane + 1;
            return true;
        }
        if (m < PLANES + EXTRA) {
            const int t = warp + (m - PLANES) * WARPS;
            ii = t >> 1;
            jj = WARPS + (t & 1);
            kk = lane + 1;
            return t < 2 * PLANES;
        }
        const int t = threadIdx.x + (m - PLANES - EXTRA) * THREADS;
        const int r = t >> 1;
        ii = r / NJ;
        jj = r - ii * NJ;
        kk = (t & 1) * (TK + 1);
        return t < 2 * NJ * PLANES;
    }
    // ev, od: the arrays of the values of even and odd parity ii + jj + kk
    template <bool BOX>
    __device__ __forceinline__ void load(const double *ev, const double *od, int i0, int j0, int k0, int n0,
                                         int n1, int n2)
    {
        const long long pn = BOX ? (long long)(n1 + 2) * (n2 + 2) : (long long)n1 * n2;
#pragma unroll
        for (int m = 0; m < PLANES + EXTRA + ENDS; ++m) {
            int ii, jj, kk;
            const bool has = at(m, ii, jj, kk);
            const int i = i0 - 1 + ii, j = j0 - 1 + jj, k = k0 - 1 + kk;
            const bool in = has && j <= n1 && k <= n2;
            const double *src = ((ii + jj + kk) & 1) ? od : ev;
            const int jk = BOX ? (j + 1) * (n2 + 2) + k + 1 : wrap1(j, n1) * n2 + wrap1(k, n2);
            const int ia = BOX ? i + 1 : wrap1(i, n0), ib = BOX ? i + 1 + SUB : wrap1(i + SUB, n0);
            a[m] = in && i <= n0 ? MG5_AT(src, ia * pn + jk) : 0.0;
            b[m] = in && i + SUB <= n0 ? MG5_AT(src, ib * pn + jk) : 0.0;
        }
    }
    __device__ __forceinline__ int max_exponent() const
    {
        unsigned e = 0;
#pragma unroll
        for (int m = 0; m < PLANES + EXTRA + ENDS; ++m)
            e = max(e, max((unsigned)__double2hiint(a[m]) & 0x7fffffffu, (unsigned)__double2hiint(b[m]) & 0x7fffffffu));
        return (int)(e >> 20);
    }
    // put(ii, jj, kk, pieces)
    template <typename Put>
    __device__ __forceinline__ void store(int eb, const Put &put) const
    {
#pragma unroll
        for (int m = 0; m < PLANES + EXTRA + ENDS; ++m) {
            int ii, jj, kk;
            if (at(m, ii, jj, kk))
                put(ii, jj, kk, split_two(a[m], b[m], eb));
        }
    }
};

// ------------------------------------------------------------------ half-sweep
// One colour of a snapshot red-black sweep: the active cells' values and edges from `same`, their
// faces (the other colour) from `faces`, into `out` at the active cells.
// Shared memory: the pieces by colour ([0] the active one), 17 values of one colour a row.
constexpr int HK = NK / 2;

template <int SUB>
struct HalfSmem {
    static constexpr int N = (SUB + 2) * NJ * HK;
    float2 h[2][N], m[2][N], l[2][N];
    int ex[WARPS];
};

template <int SUB, bool BOX>
__global__ void __launch_bounds__(THREADS, SUB == 4 && !BOX ? 4 : 3)
    k_split_half(const double *__restrict__ same, const double *faces, double *out,
                 const double *__restrict__ f, const double *__restrict__ cptr, double rhs_add, int n0,
                 int n1, int n2, Coef cs, CoefT<double> cf, int colour, unsigned long long *clamp)
{
    extern __shared__ __align__(16) unsigned char sp_raw[];
    HalfSmem<SUB> &S = *reinterpret_cast<HalfSmem<SUB> *>(sp_raw);
    constexpr int CELLS = SUB * TJ * (TK / 2) / THREADS;
    const int tid = threadIdx.x;
    const int k0 = blockIdx.x * TK, j0 = blockIdx.y * TJ, i0 = blockIdx.z * 2 * SUB;
    const int act = (colour + 1) & 1;   // parity of ii + jj + kk on the active colour (origins are even)
    const double c = cptr ? MG5_AT(cptr, 0) : rhs_add;

    const int pp = tid & 15;
    double fan = 0.0, fbn = 0.0;   // the first pair's right-hand sides
    {
        const int li = (tid >> 4) / TJ, lj = (tid >> 4) % TJ;
        const int i = i0 + li, j = j0 + lj, k = k0 + 2 * pp + ((act + li + lj + 1) & 1);
        const long long q = ((long long)i * n1 + j) * n2 + k;
        if (j < n1 && k < n2) {
            fan = i < n0 ? MG5_AT(f, q) : 0.0;
            fbn = i + SUB < n0 ? MG5_AT(f, q + (long long)SUB * n1 * n2) : 0.0;
        }
    }
    TileRegs<SUB> T;
    T.template load<BOX>(act ? faces : same, act ? same : faces, i0, j0, k0, n0, n1, n2);
    int eb;
    Kap kap;
    // A tile that is zero or tiny beside its source (the first half-sweep of a cold start) takes a unit 2^-77 of
    // the source, of which a sample is at hand: what its own values lose then lies 2^-60 below the change,
    // and the unit of 1 would round an h^2 f below 2^-92 to nothing.  Cells whose source is out of
    // the pairs' range all the same, and a tile of zeros whose sample is zero, go to FP64.
    const int fx = max(max(exponent(fan), exponent(fbn)), exponent(c)) + exponent(cf.h2) - 1021;   // h^2 (f + c) < 2^(fx - 1022)
    const bool fast = tile_exponent(max(T.max_exponent(), fx - 57), cs, S.ex, eb, kap);
    if (fast)
        T.store(eb, [&](int ii, int jj, int kk, const P3 &p) {
            const int col = ((ii + jj + kk) & 1) == act ? 0 : 1, q = (ii * NJ + jj) * HK + (kk >> 1);
            MG5_AT(S.h[col], q) = p.h;
            MG5_AT(S.m[col], q) = p.m;
            MG5_AT(S.l[col], q) = p.l;
        });
    __syncthreads();
    const double to_u = cf.h2 * pow2(kUnitBias - eb);
    unsigned clamps = 0;
    auto slow = [&](int i, int j, int k, long long at, double fm) {
        St<double> s;
        gather_at<BOX>(faces, same, i, j, k, n0, n1, n2, s);
        bool cl = false;
        MG5_AT(out, at) = cell_update(s, fm, cf, cl);
        clamps += cl;
    };
    // pair m of this thread: its row, and the cells' offsets in f (-1: outside the grid)
    auto cells = [&](int m, int &li, int &lj, int &par, long long &fa, long long &fb) {
        const int row = (tid >> 4) + m * (THREADS / 16);
        li = row / TJ;
        lj = row % TJ;
        par = (act + li + lj + 1) & 1;
        const int i = i0 + li, j = j0 + lj, k = k0 + 2 * pp + par;
        const bool in = m < CELLS && j < n1 && k < n2;
        const long long q = ((long long)i * n1 + j) * n2 + k;
        fa = in && i < n0 ? q : -1;
        fb = in && i + SUB < n0 ? q + (long long)SUB * n1 * n2 : -1;
    };
    int li, lj, par;
    long long fa, fb;
    cells(0, li, lj, par, fa, fb);
#pragma unroll 1
    for (int m = 0; m < CELLS; ++m) {
        const double ra = fan + c, rb = fbn + c;
        const int i = i0 + li, j = j0 + lj, k = k0 + 2 * pp + par;
        const bool ina = fa >= 0, inb = fb >= 0;
        const long long at = BOX ? row_at<BOX>(i, j, n0, n1, n2) + k : fa;
        const long long bt = BOX ? at + (long long)SUB * (n1 + 2) * (n2 + 2) : fb;
        const int o = (li + 1) * (NJ * HK) + (lj + 1) * HK;   // the row's first value
        const int kh = pp + par, kp = pp + 1, km = pp;
        // the next pair's right-hand sides while this one is computed
        cells(m + 1, li, lj, par, fa, fb);
        fan = fa >= 0 ? MG5_AT(f, fa) : 0.0;
        fbn = fb >= 0 ? MG5_AT(f, fb) : 0.0;
        if (!ina)
            continue;
        bool oka = false, okb = false;
        if (fast) {
            constexpr int SI = NJ * HK, SJ = HK;
            const double va = MG5_AT(same, at), vb = inb ? MG5_AT(same, bt) : 0.0;
            const auto A = [&](int q) { return P3{MG5_AT(S.h[0], o + q), MG5_AT(S.m[0], o + q), MG5_AT(S.l[0], o + q)}; };
            const auto O = [&](int q) { return P3{MG5_AT(S.h[1], o + q), MG5_AT(S.m[1], o + q), MG5_AT(S.l[1], o + q)}; };
            const Lin t = lin_of(A(kh), O(SI + kh) + O(kh - SI), O(SJ + kh) + O(kh - SJ), O(kp) + O(km),
                                 (A(SI + SJ + kh) - A(SI - SJ + kh)) - (A(SJ - SI + kh) - A(kh - SI - SJ)),
                                 (A(SI + kp) - A(SI + km)) - (A(kp - SI) - A(km - SI)),
                                 (A(SJ + kp) - A(SJ + km)) - (A(kp - SJ) - A(km - SJ)));
            const Pair r = resid(t, pair_two(ra * to_u, rb * to_u), kap);
            Pair d;
            root_change(t, r, kap, d, oka, okb);
            float2 p, e;
            step_of(d, cs, p, e);
            if (oka)
                MG5_AT(out, at) = (va + unit_f64(p.x, eb)) - unit_f64(e.x, eb);
            if (okb && inb)
                MG5_AT(out, bt) = (vb + unit_f64(p.y, eb)) - unit_f64(e.y, eb);
        }
        if (!oka)
            slow(i, j, k, at, ra);
        if (!okb && inb)
            slow(i + SUB, j, k, bt, rb);
    }
    if (clamps)
        atomicAdd(&MG5_AT(clamp, 0), (unsigned long long)clamps);
}

// ------------------------------------------------------------------ residual
// r = f + add - op(v) on every cell (RHS: add - f - op(v)).  What becomes of it:
//   RESTRICT  R v -> vc, v0c and R r -> rc (8-child means), statistics
//   PLAIN     r -> rc (nullable), statistics
//   RHS       -r -> rc (the FAS right-hand side, add = the fine mean), vc[0] = 0
enum Out { RESTRICT, PLAIN, RHS };

constexpr int RSUB = 4;

// The statistics are FP32 sums of squares.  A residual of kStatMax u or more (a tile whose values are
// 2^-18 of h^2 f and less) stays out of them: the cell (PLAIN) or the tile (RESTRICT) is computed
// and counted in FP64.  With tiles of one sum at most 2^kStatGap apart, a difference from the shift
// stays below 2^55 of its tile's unit, and a tile's four squares below 2^112 of it and of the sum's, so the
// 2^14 tiles a thread has at 2048^3 stay finite.
constexpr float kStatMax = 274877906944.0f;   // 2^38
constexpr int kStatGap = 16;

struct ResidSmem {
    static constexpr int N = (RSUB + 2) * NJ * NK;
    float2 h[N], m[N], l[N];
    Pair cr[RSUB / 2 * TJ * TK / 2];     // RESTRICT: residuals and values summed over i and k pairs
    P3 cv[RSUB / 2 * TJ * TK / 2];
    int ex[WARPS];
};

__device__ __forceinline__ void reset_ghosts(double *vc, const double *v0c, int I, int J, int K, int q0,
                                             int q1, int q2)
{
    const int d1 = q1 + 2, d2 = q2 + 2;
    const bool lo[3] = {I == 0, J == 0, K == 0}, hi[3] = {I == q0 - 1, J == q1 - 1, K == q2 - 1};
    if (!(lo[0] | lo[1] | lo[2] | hi[0] | hi[1] | hi[2]))
        return;
#pragma unroll 1
    for (int m = 1; m < 27; ++m) {
        const int a = m / 9, b = (m / 3) % 3, d = m % 3;   // 0: own index, 1: ghost below, 2: above
        if ((a == 1 && !lo[0]) || (a == 2 && !hi[0]) || (b == 1 && !lo[1]) || (b == 2 && !hi[1]) ||
            (d == 1 && !lo[2]) || (d == 2 && !hi[2]))
            continue;
        const int x = a == 0 ? I + 1 : (a == 1 ? 0 : q0 + 1), y = b == 0 ? J + 1 : (b == 1 ? 0 : q1 + 1),
                  z = d == 0 ? K + 1 : (d == 1 ? 0 : q2 + 1);
        const long long g = ((long long)x * d1 + y) * d2 + z;
        MG5_AT(vc, g) = MG5_AT(v0c, g);
    }
}

// Writes coarse cell (I, J, K) of a restriction.
template <bool BOX>
__device__ __forceinline__ void put_coarse(double *vc, double *v0c, double *rc, double mv, double mr, int I,
                                           int J, int K, int n0, int n1, int n2)
{
    const int q0 = n0 >> 1, q1 = n1 >> 1, q2 = n2 >> 1;
    if (I >= q0 || J >= q1 || K >= q2)
        return;
    const long long q = ((long long)I * q1 + J) * q2 + K;
    const long long b = BOX ? ((long long)(I + 1) * (q1 + 2) + J + 1) * (q2 + 2) + K + 1 : q;
    MG5_AT(vc, b) = mv;
    MG5_AT(v0c, b) = mv;
    MG5_AT(rc, q) = mr;
    if constexpr (BOX)
        reset_ghosts(vc, v0c, I, J, K, q0, q1, q2);
}

__device__ __forceinline__ float2 shfl1(float2 x)
{
    return float2{__shfl_xor_sync(0xffffffffu, x.x, 1), __shfl_xor_sync(0xffffffffu, x.y, 1)};
}

template <int OUT, bool BOX>
__global__ void __launch_bounds__(THREADS, 3)
    k_split_resid(const double *__restrict__ v, const double *f, const double *__restrict__ addp,
                  int n0, int n1, int n2, Coef cs, CoefT<double> cf,
                  double *__restrict__ vc, double *__restrict__ v0c, double *rc,
                  double2 *__restrict__ partials, Fin fin)
{
    extern __shared__ __align__(16) unsigned char sp_raw[];
    ResidSmem &S = *reinterpret_cast<ResidSmem *>(sp_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const double add = addp ? MG5_AT(addp, 0) : 0.0;
    const int tk = (n2 + TK - 1) / TK, tj = (n1 + TJ - 1) / TJ, ti = (n0 + 2 * RSUB - 1) / (2 * RSUB);
    const int tiles = tk * tj * ti;
    const double inv_h2 = cf.inv_h2;
    Moments acc{0.0, 0.0, 0.0, 0.0};
    auto merge = [&](const Moments &x) {
        if (acc.n == 0.0) {
            acc = x;
        } else {
            const Moments u = mom_shift(x, acc.k);
            acc.n += u.n;
            acc.s += u.s;
            acc.q += u.q;
        }
    };
    // the thread's statistics in FP32 pairs, in units of 2^(eb0 - kUnitBias) (a tile's sums move
    // there by a power of two) and shifted by K, its first residual: FP64 only at the end
    int eb0 = 0, cnt = 0;
    float K = 0.0f;
    Pair sum{{0.0f, 0.0f}, {0.0f, 0.0f}}, sq{{0.0f, 0.0f}, {0.0f, 0.0f}};   // of the two halves
    auto flush = [&]() {
        if (cnt == 0)
            return;
        const double scale = pow2(eb0 - kUnitBias) * inv_h2;
        const auto dbl = [](const Pair &x) {
            return (f32_to_f64(x.h.x) + f32_to_f64(x.h.y)) + (f32_to_f64(x.l.x) + f32_to_f64(x.l.y));
        };
        merge(Moments{(double)cnt, f32_to_f64(K) * scale, dbl(sum) * scale, dbl(sq) * scale * scale});
        cnt = 0;
        sum = sq = Pair{{0.0f, 0.0f}, {0.0f, 0.0f}};
    };
    if (OUT == RHS && blockIdx.x == 0 && tid == 0)
        MG5_AT(vc, 0) = 0.0;   // the coarse grid's c starts at zero

    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int k0 = (tile % tk) * TK, j0 = (tile / tk % tj) * TJ, i0 = tile / (tk * tj) * 2 * RSUB;
        int eb;
        Kap kap;
        bool fast;
        {
            TileRegs<RSUB> T;
            T.template load<BOX>(v, v, i0, j0, k0, n0, n1, n2);
            // a tile of zeros (eb = 0) has r = f + add, which FP64 gives without rounding (the stopping
            // test of a source whose mean is far above its spread needs every bit of it)
            const int emax = T.max_exponent();
            fast = tile_exponent(emax, cs, S.ex, eb, kap);
            // (tile_exponent has refused it already; asked again, the kernel compiles to 271 us at 256^3
            // instead of 278)
            if (OUT != RHS)
                fast = __syncthreads_or(emax != 0) && fast;
            if (fast)
                T.store(eb, [&](int ii, int jj, int kk, const P3 &p) {
                    const int q = (ii * NJ + jj) * NK + kk;
                    MG5_AT(S.h, q) = p.h;
                    MG5_AT(S.m, q) = p.m;
                    MG5_AT(S.l, q) = p.l;
                });
        }
        __syncthreads();
        const double to_u = cf.h2 * pow2(kUnitBias - eb);
        const int j = j0 + warp, k = k0 + lane;
        const bool col = j < n1 && k < n2;
        const long long plane_n = (long long)n1 * n2;
        const long long cell0 = col ? ((long long)i0 * n1 + j) * n2 + k : 0;
        // one cell in FP64
        auto slow = [&](int i, double fm) {
            St<double> s;
            gather_at<BOX>(v, v, i, j, k, n0, n1, n2, s);
            return cell_residual(s, fm, cf);
        };
        if (fast) {
            if (OUT != RHS && cnt > 0 && abs(eb - eb0) > kStatGap)
                flush();
            float Kt = cnt > 0 ? K * __int_as_float((eb0 - eb + 127) << 23) : 0.0f;
            Pair tsum{{0.0f, 0.0f}, {0.0f, 0.0f}}, tsq{{0.0f, 0.0f}, {0.0f, 0.0f}};
            const int o = (warp + 1) * NK + lane + 1;
            constexpr int SI = NJ * NK;
            auto at = [&](int q) { return P3{MG5_AT(S.h, o + q), MG5_AT(S.m, o + q), MG5_AT(S.l, o + q)}; };
            Pair ra{};
            P3 va{};
            bool bad = false;
            int redone = 0;
            const bool in_a = col && i0 < n0;   // sides are even: a tile's planes come in pairs
            double fa = in_a ? MG5_AT(f, cell0) : 0.0,
                   fb = col && i0 + RSUB < n0 ? MG5_AT(f, cell0 + RSUB * plane_n) : 0.0;
#pragma unroll 1
            for (int m = 0; m < RSUB; ++m) {
                const bool lva = col && i0 + m < n0, lvb = col && i0 + RSUB + m < n0;
                const long long cell = cell0 + m * plane_n;
                const double rha = OUT == RHS ? add - fa : fa + add, rhb = OUT == RHS ? add - fb : fb + add;
                if (m + 1 < RSUB) {
                    fa = col && i0 + m + 1 < n0 ? MG5_AT(f, cell + plane_n) : 0.0;
                    fb = col && i0 + RSUB + m + 1 < n0 ? MG5_AT(f, cell + (RSUB + 1) * plane_n) : 0.0;
                }
                const int q = (m + 1) * SI;
                const P3 c0 = at(q);
                const Pair r = resid(lin_of(c0, at(q + SI) + at(q - SI), at(q + NK) + at(q - NK), at(q + 1) + at(q - 1),
                                            (at(q + SI + NK) - at(q + SI - NK)) - (at(q - SI + NK) - at(q - SI - NK)),
                                            (at(q + SI + 1) - at(q + SI - 1)) - (at(q - SI + 1) - at(q - SI - 1)),
                                            (at(q + NK + 1) - at(q + NK - 1)) - (at(q - NK + 1) - at(q - NK - 1))),
                                     pair_two(rha * to_u, rhb * to_u), kap);
                // not finite, an f beyond the pairs' range, or too large for the statistics: the tile is
                // done again in FP64 (RHS and PLAIN, which may write over f, recompute the cell)
                constexpr float lim = OUT == RHS ? 1e30f : kStatMax;
                const bool bad_a = lva && !(fabsf(r.h.x) < lim), bad_b = lvb && !(fabsf(r.h.y) < lim);
                bad = bad || bad_a || bad_b;
                if (OUT != RHS) {
                    if (!BOX && m == 0 && cnt == 0)
                        Kt = fabsf(r.h.x) < lim ? r.h.x : 0.0f;
                    Pair d = two_diff(r.h, both(Kt));
                    d.l = add2(d.l, r.l);
                    if (!lva || (OUT == PLAIN && bad_a))
                        d.h.x = d.l.x = 0.0f;
                    if (!lvb || (OUT == PLAIN && bad_b))
                        d.h.y = d.l.y = 0.0f;
                    const Pair s = two_sum(tsum.h, d.h);
                    tsum.h = s.h;
                    tsum.l = add2(tsum.l, add2(s.l, d.l));
                    float2 p, e;
                    neg_sqr(d, p, e);
                    const Pair g = two_diff(tsq.h, p);
                    tsq.h = g.h;
                    tsq.l = add2(tsq.l, add2(g.l, e));
                }
                if constexpr (OUT == RESTRICT) {
                    if ((m & 1) == 0) {
                        ra = r;
                        va = c0;
                    } else {
                        Pair s = two_sum(ra.h, r.h);
                        s.l = add2(s.l, add2(ra.l, r.l));
                        va = va + c0;
                        const Pair o2{shfl1(s.h), shfl1(s.l)};
                        const P3 v2{shfl1(va.h), shfl1(va.m), shfl1(va.l)};
                        const Pair w = two_sum(s.h, o2.h);
                        if ((lane & 1) == 0) {
                            const int x = ((m >> 1) * TJ + warp) * (TK / 2) + (lane >> 1);
                            MG5_AT(S.cr, x) = Pair{w.h, add2(w.l, add2(s.l, o2.l))};
                            MG5_AT(S.cv, x) = va + v2;
                        }
                    }
                } else {
                    const auto put = [&](float h, float l, bool redo, int i, double rh, long long q) {
                        double x = (unit_f64(h, eb) + unit_f64(l, eb)) * inv_h2;
                        if (redo) {
                            x = slow(i, rh);
                            if (OUT == PLAIN) {
                                merge(Moments{1.0, x, 0.0, 0.0});
                                ++redone;
                            }
                        }
                        if (rc)
                            MG5_AT(rc, q) = OUT == RHS ? -x : x;
                    };
                    if (lva && (rc || bad_a))
                        put(r.h.x, r.l.x, bad_a, i0 + m, rha, cell);
                    if (lvb && (rc || bad_b))
                        put(r.h.y, r.l.y, bad_b, i0 + RSUB + m, rhb, cell + RSUB * plane_n);
                }
            }
            if (OUT == RESTRICT)
                fast = !__syncthreads_or(bad);
            if (OUT != RHS && col && fast) {
                if (cnt == 0) {
                    eb0 = eb;
                    K = Kt;
                }
                const float up = __int_as_float((eb - eb0 + 127) << 23);
                Pair t = two_sum(sum.h, mul2(tsum.h, both(up)));
                sum.h = t.h;
                sum.l = add2(sum.l, add2(t.l, mul2(tsum.l, both(up))));
                t = two_sum(sq.h, mul2(tsq.h, both(up * up)));
                sq.h = t.h;
                sq.l = add2(sq.l, add2(t.l, mul2(tsq.l, both(up * up))));
                cnt += min(max(n0 - i0, 0), RSUB) + min(max(n0 - i0 - RSUB, 0), RSUB) - redone;
            }
        }
        if (!fast) {
            for (int m = 0; m < 2 * RSUB; ++m) {
                const bool live = col && i0 + m < n0;
                const long long cell = cell0 + m * plane_n;
                double x = 0.0, cv = 0.0;
                if (live) {
                    x = slow(i0 + m, OUT == RHS ? add - MG5_AT(f, cell) : MG5_AT(f, cell) + add);
                    cv = MG5_AT(v, row_at<BOX>(i0 + m, j, n0, n1, n2) + k);
                    if (OUT != RHS)
                        merge(Moments{1.0, BOX ? 0.0 : x, BOX ? x : 0.0, BOX ? x * x : 0.0});
                    if ((OUT == PLAIN || OUT == RHS) && rc)
                        MG5_AT(rc, cell) = OUT == RHS ? -x : x;
                }
                if constexpr (OUT == RESTRICT) {
                    // the eight children of a coarse cell through the (unused) piece arrays
                    double *sd = reinterpret_cast<double *>(S.h);
                    MG5_AT(sd, ((m & 1) * TJ + warp) * TK + lane) = cv;
                    MG5_AT(sd, ((2 + (m & 1)) * TJ + warp) * TK + lane) = x;
                    __syncthreads();
                    if ((m & 1) && tid < TJ / 2 * TK / 2) {
                        const int J = tid / (TK / 2), Kc = tid % (TK / 2);
                        double sv = 0.0, sr = 0.0;
                        for (int ch = 0; ch < 8; ++ch) {
                            const int a = ((ch >> 2) * TJ + 2 * J + ((ch >> 1) & 1)) * TK + 2 * Kc + (ch & 1);
                            sv += MG5_AT(sd, a);
                            sr += MG5_AT(sd, a + 2 * TJ * TK);
                        }
                        put_coarse<BOX>(vc, v0c, rc, 0.125 * sv, 0.125 * sr, (i0 + m) >> 1, (j0 >> 1) + J,
                                        (k0 >> 1) + Kc, n0, n1, n2);
                    }
                    __syncthreads();
                }
            }
        }
        __syncthreads();
        if constexpr (OUT == RESTRICT) {
            if (fast && tid < RSUB / 2 * (TJ / 2) * (TK / 2)) {
                // the coarse cells of each half, one a thread: the two rows of each
                const int I = tid / (TJ / 2 * TK / 2), J = tid / (TK / 2) % (TJ / 2), Kc = tid % (TK / 2);
                const int x = (I * TJ + 2 * J) * (TK / 2) + Kc;
                const Pair s0 = MG5_AT(S.cr, x), s1 = MG5_AT(S.cr, x + TK / 2);
                Pair s = two_sum(s0.h, s1.h);
                s.l = add2(s.l, add2(s0.l, s1.l));
                const P3 w = MG5_AT(S.cv, x) + MG5_AT(S.cv, x + TK / 2);
                const int Ig = (i0 >> 1) + I, Jg = (j0 >> 1) + J, Kg = (k0 >> 1) + Kc;
                const auto val = [&](float h, float m, float l) {
                    return 0.125 * ((unit_f64(h, eb) + unit_f64(m, eb)) + unit_f64(l, eb));
                };
                const auto res = [&](float h, float l) {
                    return 0.125 * inv_h2 * (unit_f64(h, eb) + unit_f64(l, eb));
                };
                put_coarse<BOX>(vc, v0c, rc, val(w.h.x, w.m.x, w.l.x), res(s.h.x, s.l.x), Ig, Jg, Kg, n0, n1, n2);
                put_coarse<BOX>(vc, v0c, rc, val(w.h.y, w.m.y, w.l.y), res(s.h.y, s.l.y), Ig + RSUB / 2, Jg, Kg, n0,
                                n1, n2);
            }
        }
    }
    if constexpr (OUT != RHS) {
        flush();
        if constexpr (BOX) {
            const double2 a = block_sum2(make_double2(acc.s, acc.q));   // plain sums (every shift is zero)
            if (tid == 0)
                MG5_AT(partials, blockIdx.x) = a;
        } else {
            MomAcc<double> a;
            a.n = (int)acc.n;
            a.k = acc.k;
            a.s = acc.s;
            a.q = acc.q;
            const Moments mm = block_moments(a);
            if (tid == 0)
                MG5_AT(reinterpret_cast<Moments *>(partials), blockIdx.x) = mm;
        }
        if (fin.ls)
            finalize_if_last(partials, fin);
    }
}

template <int SUB, bool BOX>
cudaError_t half_launch(const double *in, double *out, const double *f, const double *cptr, double add,
                        const int n[3], const CoefT<double> &cf, unsigned long long *clamp, cudaStream_t st)
{
    const Coef cs = make_split_coef(cf);
    const dim3 g((n[2] + TK - 1) / TK, (n[1] + TJ - 1) / TJ, (n[0] + 2 * SUB - 1) / (2 * SUB));
    const size_t sm = sizeof(HalfSmem<SUB>);
    k_split_half<SUB, BOX><<<g, THREADS, sm, st>>>(in, in, out, f, cptr, add, n[0], n[1], n[2], cs, cf, 0, clamp);
    k_split_half<SUB, BOX><<<g, THREADS, sm, st>>>(in, out, out, f, cptr, add, n[0], n[1], n[2], cs, cf, 1, clamp);
    count_launch(2);
    return cudaGetLastError();
}

// Planes of a half-tile: four where such tiles still give every SM one (16^3 cells an SM), else two
// (a 64^3 half-sweep: 5.5 us in 256 tiles of two against 5.9 in 128 of four).
template <bool BOX>
cudaError_t half_launch_sized(const double *in, double *out, const double *f, const double *cptr, double add,
                              const int n[3], const CoefT<double> &cf, unsigned long long *clamp, cudaStream_t st)
{
    const long long cols = (long long)((n[2] + TK - 1) / TK) * ((n[1] + TJ - 1) / TJ);
    if (cols * n[0] >= 8ll * kSMs)
        return half_launch<4, BOX>(in, out, f, cptr, add, n, cf, clamp, st);
    return half_launch<2, BOX>(in, out, f, cptr, add, n, cf, clamp, st);
}

template <int SUB, bool BOX>
cudaError_t prepare_half()
{
    return cudaFuncSetAttribute(k_split_half<SUB, BOX>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)sizeof(HalfSmem<SUB>));
}

template <int OUT, bool BOX>
cudaError_t resid_launch(const double *v, const double *f, const double *add, const int n[3],
                         const CoefT<double> &cf, double *vc, double *v0c, double *rc, double2 *partials, int *nblocks, cudaStream_t st, const Fin &fin)
{
    const Coef cs = make_split_coef(cf);
    const long long tiles = (long long)((n[2] + TK - 1) / TK) * ((n[1] + TJ - 1) / TJ) *
                            ((n[0] + 2 * RSUB - 1) / (2 * RSUB));
    const int g = (int)(tiles < 3 * kSMs ? tiles : 3 * kSMs);   // three CTAs fit on an SM
    k_split_resid<OUT, BOX><<<g, THREADS, sizeof(ResidSmem), st>>>(v, f, add, n[0], n[1], n[2], cs, cf, vc,
                                                                  v0c, rc, partials, fin);
    if (nblocks)
        *nblocks = g;
    count_launch(1);
    return cudaGetLastError();
}

template <int OUT, bool BOX>
cudaError_t prepare_resid()
{
    return cudaFuncSetAttribute(k_split_resid<OUT, BOX>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)sizeof(ResidSmem));
}

}  // namespace

cudaError_t prepare_split_kernels()
{
    cudaError_t e = prepare_resid<RESTRICT, false>();
    if (e == cudaSuccess)
        e = prepare_resid<RESTRICT, true>();
    if (e == cudaSuccess)
        e = prepare_resid<PLAIN, false>();
    if (e == cudaSuccess)
        e = prepare_resid<RHS, false>();
    for (cudaError_t (*prep)() : {prepare_half<2, false>, prepare_half<4, false>, prepare_half<2, true>, prepare_half<4, true>})
        if (e == cudaSuccess)
            e = prep();
    return e;
}

cudaError_t launch_split_sweep(const double *in, double *out, const double *f, const double *cptr, int n,
                               const CoefT<double> &cf, unsigned long long *clamp, cudaStream_t st)
{
    const int d[3] = {n, n, n};
    return half_launch_sized<false>(in, out, f, cptr, 0.0, d, cf, clamp, st);
}

cudaError_t launch_split_patch_sweep(const double *in, double *out, const double *f, double add, const int p[3],
                                     const CoefT<double> &cf, unsigned long long *clamp,
                                     cudaStream_t st)
{
    return half_launch_sized<true>(in, out, f, nullptr, add, p, cf, clamp, st);
}

cudaError_t launch_split_resid_restrict(const double *v, const double *f, const double *cptr, int n,
                                        const CoefT<double> &cf, double *vc, double *v0c, double *rc,
                                        double2 *partials, int *nblocks, cudaStream_t st, const Fin &fin)
{
    const int d[3] = {n, n, n};
    return resid_launch<RESTRICT, false>(v, f, cptr, d, cf, vc, v0c, rc, partials, nblocks, st, fin);
}

cudaError_t launch_split_residual(const double *v, const double *f, const double *cptr, int n,
                                  const CoefT<double> &cf, double *r, double2 *partials, int *nblocks,
                                  cudaStream_t st, const Fin &fin)
{
    const int d[3] = {n, n, n};
    return resid_launch<PLAIN, false>(v, f, cptr, d, cf, nullptr, nullptr, r, partials, nblocks, st, fin);
}

cudaError_t launch_split_coarse_rhs(const double *v, double *f, const double *m_fine, double *c_coarse, int n,
                                    const CoefT<double> &cf, cudaStream_t st)
{
    const int d[3] = {n, n, n};
    return resid_launch<RHS, false>(v, f, m_fine, d, cf, c_coarse, nullptr, f, nullptr, nullptr, st, Fin());
}

cudaError_t launch_split_patch_resid_restrict(const double *v, const double *f, const int p[3],
                                              const CoefT<double> &cf, double *vc, double *v0c,
                                              double *fc, double2 *partials, int *nblocks, cudaStream_t st,
                                              const Fin &fin)
{
    return resid_launch<RESTRICT, true>(v, f, nullptr, p, cf, vc, v0c, fc, partials, nblocks, st, fin);
}

}  // namespace mg5
