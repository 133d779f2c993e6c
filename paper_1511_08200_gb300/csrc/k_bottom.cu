// k_bottom.cu -- the bottom of an FP32 V-cycle in one CTA: the visit of the grids from 16^3 (or 12^3)
// down to the coarsest one (4^3 or 6^3) as one launch, with the same steps, in the same order and with
// the same cell arithmetic as the level-by-level launches (Sec. 3.1: FAS coarse right-hand side, nu1
// snapshot red-black sweeps, residual with its mean subtracted from the compatibility constant,
// 8-child restriction, the coarsest-grid iteration, trilinear prolongation of the correction, nu2
// sweeps).  On these grids every launch costs more than its cells.  The FP64 solves have k_visit.cu.
//
// On entry the finest of these grids holds v = R v (the restricted iterate of the grid above) and
// f = R r; on exit v is the corrected iterate and the level scalars its constant c and residual mean m.
// Periodic grids, correction form with the restricted bases B.
//
// Everything lives in shared memory (207 KB for 16^3 and below).  The cells of a grid are kept by
// colour (red: i + j + k even), each colour's rows of n / 2 cells one after the other: the lanes of a
// half-sweep read 19 values at consecutive addresses whatever their k's parity, only the threads of
// one colour run, and a sweep goes from one array to the other without copying the resting colour (a
// red cell reads old values only, a black one new red faces and old black edges).  The sums and
// differences of B, which no sweep changes, are formed once a visit: a cell update then reads 19
// values of e, two 16-byte words of B's parts and f.
//
// The coarsest grid is iterated by two to eight warps, a cell a thread.  In FP64 its two sums (for the
// mean and the stopping norm) and the norm's square root took most of an iteration (an FP64
// instruction of a warp takes 16 clocks of the SM's pipe).  The sum of r is now formed in FP32 pairs
// (48 bits: the residuals' 24-bit values add up exactly unless one is 2^-24 of the sum), the mean from
// it in a pair rounded once, and the stopping test norm <= rtol norm_0 in FP32 wherever it is not
// close: else it is formed in FP64.
//
// From 12^3 the results are those of the launches to the bit; from 16^3 and 8^3 the mean residual of 8^3 is
// summed in pairs instead, which may round the constant c otherwise (fields within 2^-17 in the tests).
//
// A visit from 16^3 takes 47 us (launch by launch ~77, of it 29 for 8^3 and 4^3 in one CTA that
// gathered through offset tables), from 12^3 40-46 (its 6^3 grid alone took 70).  Bound by shared-memory
// bandwidth and latency on the one SM: a half-sweep of 16^3 is 1.9 kclk of shared loads.
#include "mg5_fin.cuh"

namespace mg5 {

namespace {

constexpr int kBotThreads = 512;
constexpr int kBotLevels = 3;

struct BotLevel {
    CoefT<float> cf;
    const float *B;
    LevelScal *ls;
};

struct BotArgs {
    BotLevel lv[kBotLevels];
    float *v;
    const float *f;
    const LevelScal *ls_up;
    int nu1, nu2, nu_coarse;
    double rtol;
    unsigned long long *clamp;
    int *sweeps;
};

// One grid's arrays in shared memory, x[colour * HC + (i N + j) H + (k >> 1)].  The sides are template
// arguments: with sides at run time the divisions of a cell's index and its neighbours' addresses cost
// more than its arithmetic (a visit from 16^3 took 71 us, from 12^3 40).
template <int N>
struct BotGrid {
    static constexpr int H = N / 2, HC = N * N * H, CELLS = N * N * N;
    static constexpr int FLOATS = 12 * CELLS;
    // planes that the threads of a half-sweep cover at once: an even divisor of N
    static constexpr int S = N == 16 ? 4 : N == 12 ? 6 : N;
    static_assert(S % 2 == 0 && N % S == 0 && S * N * H <= kBotThreads, "threads of a half-sweep");
    float4 *bs, *bd;         // B's parts: (S, a, b, c) and (dxy, dxz, dyz, centre)
    float *v, *w, *f, *v0;
    __device__ __forceinline__ explicit BotGrid(float *at)
    {
        bs = reinterpret_cast<float4 *>(at);
        bd = bs + CELLS;
        v = at + 8 * CELLS;
        w = v + CELLS;
        f = w + CELLS;
        v0 = f + CELLS;
    }
    __device__ __forceinline__ void turn(int sweeps)   // v and w change places at every sweep
    {
        float *a = v, *b = w;
        v = (sweeps & 1) ? b : a;
        w = (sweeps & 1) ? a : b;
    }
    static __device__ __forceinline__ int idx(int i, int j, int k)
    {
        return ((i + j + k) & 1) * HC + (i * N + j) * H + (k >> 1);
    }
};

// offsets of a cell's 19 points: rows (i + a, j + b), places of k, k - 1, k + 1 in a row
struct BotNbr {
    int r00, rp0, rm0, r0p, r0m, rpp, rpm, rmp, rmm, k0, km, kp;
};

template <int N>
__device__ __forceinline__ BotNbr bot_nbr(int i, int j, int k)
{
    constexpr int H = N / 2;
    const int ip = i + 1 == N ? 0 : i + 1, im = i == 0 ? N - 1 : i - 1;
    const int jp = j + 1 == N ? 0 : j + 1, jm = j == 0 ? N - 1 : j - 1;
    const auto row = [](int a, int b) { return (a * N + b) * H; };
    const int kk = k >> 1;
    return BotNbr{row(i, j),   row(ip, j),  row(im, j),  row(i, jp),  row(i, jm), row(ip, jp),
                  row(ip, jm), row(im, jp), row(im, jm), kk,
                  (k & 1) ? kk : (kk == 0 ? H - 1 : kk - 1),
                  (k & 1) ? (kk + 1 == H ? 0 : kk + 1) : kk};
}

// the place q of a cell in the arrays -> its colour and neighbours
template <int N>
__device__ __forceinline__ BotNbr bot_at(int q, int &colour)
{
    using G = BotGrid<N>;
    colour = q >= G::HC ? 1 : 0;
    const int r = q - colour * G::HC, row = r / G::H, i = row / N, j = row - i * N;
    return bot_nbr<N>(i, j, 2 * (r - row * G::H) + ((i + j + colour) & 1));
}

// own: the cell's colour (centre and edges), oth: the other one (faces)
__device__ __forceinline__ void bot_gather(const float *own, const float *oth, const BotNbr &b, St<float> &s)
{
    s.c = MG5_AT(own, b.r00 + b.k0);
    s.xp = MG5_AT(oth, b.rp0 + b.k0);
    s.xm = MG5_AT(oth, b.rm0 + b.k0);
    s.yp = MG5_AT(oth, b.r0p + b.k0);
    s.ym = MG5_AT(oth, b.r0m + b.k0);
    s.zp = MG5_AT(oth, b.r00 + b.kp);
    s.zm = MG5_AT(oth, b.r00 + b.km);
    s.xpyp = MG5_AT(own, b.rpp + b.k0);
    s.xpym = MG5_AT(own, b.rpm + b.k0);
    s.xmyp = MG5_AT(own, b.rmp + b.k0);
    s.xmym = MG5_AT(own, b.rmm + b.k0);
    s.xpzp = MG5_AT(own, b.rp0 + b.kp);
    s.xpzm = MG5_AT(own, b.rp0 + b.km);
    s.xmzp = MG5_AT(own, b.rm0 + b.kp);
    s.xmzm = MG5_AT(own, b.rm0 + b.km);
    s.ypzp = MG5_AT(own, b.r0p + b.kp);
    s.ypzm = MG5_AT(own, b.r0p + b.km);
    s.ymzp = MG5_AT(own, b.r0m + b.kp);
    s.ymzm = MG5_AT(own, b.r0m + b.km);
}

// (S, a, b, c) and (dxy, dxz, dyz, centre) of a cell, the operations of parts2_of in scalar form
__device__ __forceinline__ void bot_parts(const St<float> &s, float4 &p, float4 &d)
{
    const float sx = __fadd_rn(s.xp, s.xm), sy = __fadd_rn(s.yp, s.ym), sz = __fadd_rn(s.zp, s.zm);
    p = make_float4(__fadd_rn(__fadd_rn(sx, sy), sz), __fsub_rn(sx, sy), __fsub_rn(sx, sz), __fsub_rn(sy, sz));
    d = make_float4(__fsub_rn(__fsub_rn(s.xpyp, s.xpym), __fsub_rn(s.xmyp, s.xmym)),
                    __fsub_rn(__fsub_rn(s.xpzp, s.xpzm), __fsub_rn(s.xmzp, s.xmzm)),
                    __fsub_rn(__fsub_rn(s.ypzp, s.ypzm), __fsub_rn(s.ymzp, s.ymzm)), s.c);
}

__device__ __forceinline__ Parts2 bot_pair(const float4 &p, const float4 &d, const float4 &bs, const float4 &bd)
{
    Parts2 q;
    q.S = make_float2(p.x, bs.x);
    q.a = make_float2(p.y, bs.y);
    q.b = make_float2(p.z, bs.z);
    q.c = make_float2(p.w, bs.w);
    q.dxy = make_float2(d.x, bd.x);
    q.dxz = make_float2(d.y, bd.y);
    q.dyz = make_float2(d.z, bd.z);
    return q;
}

// op(B + e) - op(B) at a cell
__device__ __forceinline__ float bot_op(const float *own, const float *oth, const BotNbr &nb,
                                        const float4 &bs, const float4 &bd, const CoefT<float> &cf)
{
    St<float> s;
    bot_gather(own, oth, nb, s);
    float4 p, d;
    bot_parts(s, p, d);
    return cell_op_corr_parts(bot_pair(p, d, bs, bd), bd.w, d.w, cf);
}

__device__ __forceinline__ float bot_update(const float *own, const float *oth, const BotNbr &nb,
                                            const float4 &bs, const float4 &bd, float rhs,
                                            const CoefT<float> &cf, bool &clamped)
{
    St<float> s;
    bot_gather(own, oth, nb, s);
    float4 p, d;
    bot_parts(s, p, d);
    return cell_update_corr_parts(bot_pair(p, d, bs, bd), bd.w, d.w, rhs, cf, clamped);
}

// `count` sweeps of a grid (the caller turns its arrays).  A thread's cells are one (j, k) on the planes
// i0, i0 + S, ...; S is even, so they are of one colour.
template <int N>
__device__ __noinline__ void bot_sweeps(BotGrid<N> g, int count, float c, const CoefT<float> &cf_in,
                                        unsigned &clamps)
{
    using G = BotGrid<N>;
    const CoefT<float> cf = cf_in;
    constexpr int per = N * G::H;
    const int i0 = threadIdx.x / per, rest = threadIdx.x - i0 * per;
    const int j = rest / G::H, kk = rest - j * G::H;
    const bool mine = i0 < G::S;
    for (int it = 0; it < count; ++it) {
#pragma unroll 1
        for (int colour = 0; colour < 2; ++colour) {
            const float *own = g.v + colour * G::HC, *oth = colour == 0 ? g.v + G::HC : g.w;
            const float *f = g.f + colour * G::HC;
            const float4 *bs = g.bs + colour * G::HC, *bd = g.bd + colour * G::HC;
            float *out = g.w + colour * G::HC;
            if (mine) {
#pragma unroll
                for (int m = 0; m < N / G::S; ++m) {
                    const BotNbr nb = bot_nbr<N>(i0 + m * G::S, j, 2 * kk + ((i0 + j + colour) & 1));
                    const int q = nb.r00 + kk;
                    bool cl = false;
                    MG5_AT(out, q) = bot_update(own, oth, nb, MG5_AT(bs, q), MG5_AT(bd, q), MG5_AT(f, q) + c, cf, cl);
                    clamps += cl ? 1u : 0u;
                }
            }
            __syncthreads();
        }
        g.turn(1);
    }
}

__device__ __forceinline__ float2 two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    return make_float2(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t)));
}
__device__ __forceinline__ float2 pair_sum(float2 a, float2 b)
{
    const float2 s = two_sum(a.x, b.x);
    const float l = __fadd_rn(s.y, __fadd_rn(a.y, b.y));
    const float h = __fadd_rn(s.x, l);
    return make_float2(h, __fsub_rn(l, __fsub_rn(h, s.x)));
}
__device__ __forceinline__ float2 pair_xor(float2 a, int o)
{
    return make_float2(__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o));
}

__device__ __forceinline__ void bot_bar(int threads) { asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory"); }

struct BotShared {
    double c[kBotLevels], m;         // constants of the grids, residual mean of the one above
    float cf, mf;                    // c of the grid at work and m, in FP32
    int iters;                       // sweeps of the coarsest grid
    Moments mom[kBotThreads / 32];
    float2 sum[kBotThreads / 32];
    float sq[8], sq2[8];
    double2 sum64[8];
};

// Sums over the WARPS values in `sm`.  Every lane of every warp gets the same bits (each lane starts
// from one of the values and the additions commute): barriers are taken by what the sums decide.
template <int WARPS>
__device__ __forceinline__ float warps_sum(const float *sm)
{
    static_assert(WARPS <= 32 && (WARPS & (WARPS - 1)) == 0, "a power of two");
    float y = sm[threadIdx.x & (WARPS - 1)];
#pragma unroll
    for (int o = WARPS / 2; o > 0; o >>= 1)
        y = __fadd_rn(y, __shfl_xor_sync(0xffffffffu, y, o));
    return y;
}
template <int WARPS>
__device__ __forceinline__ float2 warps_pair_sum(const float2 *sm)
{
    static_assert(WARPS <= 32 && (WARPS & (WARPS - 1)) == 0, "a power of two");
    float2 y = sm[threadIdx.x & (WARPS - 1)];
#pragma unroll
    for (int o = WARPS / 2; o > 0; o >>= 1)
        y = pair_sum(y, pair_xor(y, o));
    return y;
}

// The coarsest grid (at most 216 cells): before each sweep c = -mean r; until the norm of r - mean is
// rtol times the first one.
template <int N>
__device__ __forceinline__ void bot_coarsest(BotGrid<N> g, const CoefT<float> &cf_in, const BotArgs &A,
                                             BotShared &sh, double *c_out, unsigned &clamps)
{
    using G = BotGrid<N>;
    constexpr int cpt = (G::HC + 31) & ~31, threads = 2 * cpt, warps = threads >> 5;   // cpt threads a colour
    static_assert(warps <= 8, "warps of the coarsest grid");
    const int p = threadIdx.x;
    if (p >= threads)
        return;
    const int colour = p >= cpt ? 1 : 0, q = p - colour * cpt;
    const bool mine = q < G::HC;
    BotNbr nb{};
    float4 bs{}, bd{};
    float f = 0.0f;
    if (mine) {
        int col;
        nb = bot_at<N>(colour * G::HC + q, col);
        bs = MG5_AT(g.bs, colour * G::HC + q);
        bd = MG5_AT(g.bd, colour * G::HC + q);
        f = MG5_AT(g.f, colour * G::HC + q);
    }
    const CoefT<float> cf = cf_in;
    constexpr double n3 = (double)G::CELLS, inv = 1.0 / n3;
    constexpr float inv_h = (float)inv, inv_l = (float)(inv - (double)inv_h);
    const float rtol2 = (float)(A.rtol * A.rtol);
    double r0 = -1.0;
    float q0 = 0.0f;   // norm_0^2
    float2 tot = make_float2(0.0f, 0.0f);
    int it = 0;
    for (; it < A.nu_coarse; ++it) {
        float res = 0.0f;
        if (mine)
            res = __fsub_rn(f, bot_op(g.v + colour * G::HC, g.v + (1 - colour) * G::HC, nb, bs, bd, cf));
        float2 s = make_float2(res, 0.0f);
        float y = __fmul_rn(res, res);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            s = pair_sum(s, pair_xor(s, o));
            y = __fadd_rn(y, __shfl_xor_sync(0xffffffffu, y, o));
        }
        if ((p & 31) == 0) {
            sh.sum[p >> 5] = s;
            sh.sq[p >> 5] = y;
        }
        bot_bar(threads);
        tot = warps_pair_sum<warps>(sh.sum);
        y = warps_sum<warps>(sh.sq);
        // mean = tot / n3 in a pair, rounded once
        const float mh = __fmul_rn(tot.x, inv_h);
        const float ml = __fmaf_rn(tot.x, inv_h, -mh);
        const float m = __fadd_rn(mh, __fadd_rn(ml, __fmaf_rn(tot.x, inv_l, __fmul_rn(tot.y, inv_h))));
        float q2 = __fmaf_rn(-(float)n3 * m, m, y);
        bool decided = y > 1e-30f && y < 1e30f;
        if (decided && q2 <= 0.05f * y) {   // mostly the mean's: the sum about it
            float z = mine ? __fsub_rn(res, m) : 0.0f;
            z = __fmul_rn(z, z);
            for (int o = 16; o > 0; o >>= 1)
                z = __fadd_rn(z, __shfl_xor_sync(0xffffffffu, z, o));
            if ((p & 31) == 0)
                sh.sq2[p >> 5] = z;
            bot_bar(threads);
            q2 = warps_sum<warps>(sh.sq2);
            decided = q2 > 1e-7f * y && q2 > 1e-30f;   // (r - m carries m's 2^-24)
        }
        const float tol2 = rtol2 * q0;
        if (decided && it == 0) {
            q0 = q2;
        } else if (decided && q0 > 0.0f && fabsf(q2 - tol2) > 1e-5f * tol2) {
            if (q2 < tol2)
                break;
        } else {   // the norm in FP64
            double2 a = make_double2((double)res, (double)res * (double)res);
            for (int o = 16; o > 0; o >>= 1) {
                a.x += __shfl_xor_sync(0xffffffffu, a.x, o);
                a.y += __shfl_xor_sync(0xffffffffu, a.y, o);
            }
            if ((p & 31) == 0)
                sh.sum64[p >> 5] = a;
            bot_bar(threads);
            a = make_double2(0.0, 0.0);
            for (int w = 0; w < warps; ++w) {
                a.x += sh.sum64[w].x;
                a.y += sh.sum64[w].y;
            }
            const double md = a.x * inv, qd = a.y - n3 * md * md;
            const double rn = sqrt(qd > 0.0 ? qd : 0.0);
            if (r0 < 0.0)
                r0 = q0 > 0.0f ? sqrt((double)q0) : rn;
            if (rn <= A.rtol * r0)
                break;
        }
        const float rhs = __fadd_rn(f, -m);
        bool cl = false;
        if (mine && colour == 0)
            MG5_AT(g.w, q) = bot_update(g.v, g.v + G::HC, nb, bs, bd, rhs, cf, cl);
        bot_bar(threads);
        if (mine && colour == 1)
            MG5_AT(g.w, G::HC + q) = bot_update(g.v + G::HC, g.w, nb, bs, bd, rhs, cf, cl);
        clamps += cl ? 1u : 0u;
        bot_bar(threads);
        g.turn(1);
    }
    if (p == 0) {
        *c_out = A.nu_coarse > 0 ? -(((double)tot.x + (double)tot.y) * inv) : 0.0;
        sh.iters = it;
    }
}

// B of a grid, in its v0, to B's parts
template <int N>
__device__ __forceinline__ void bot_base(const BotGrid<N> &g)
{
    for (int q = threadIdx.x; q < BotGrid<N>::CELLS; q += kBotThreads) {
        int colour;
        const BotNbr nb = bot_at<N>(q, colour);
        St<float> s;
        bot_gather(g.v0 + colour * BotGrid<N>::HC, g.v0 + (1 - colour) * BotGrid<N>::HC, nb, s);
        bot_parts(s, MG5_AT(g.bs, q), MG5_AT(g.bd, q));
    }
}

// one of the grids' arrays <-> global memory (row-major); the trip count is known, so the loads of all
// a thread's cells are in flight at once
template <int N>
__device__ __forceinline__ void bot_load(float *dst, const float *src)
{
#pragma unroll
    for (int m = 0; m < (BotGrid<N>::CELLS + kBotThreads - 1) / kBotThreads; ++m) {
        const int q = m * kBotThreads + threadIdx.x, row = q / N, k = q - row * N, i = row / N, j = row - i * N;
        if (q < BotGrid<N>::CELLS)
            MG5_AT(dst, BotGrid<N>::idx(i, j, k)) = MG5_AT(src, q);
    }
}

// The visit of the grid of side N (level L of this launch) and all below it; its v is R v, its f R r.
template <int N, int L, bool LAST>
__device__ __forceinline__ void bot_visit(BotGrid<N> &g, const BotArgs &A, BotShared &sh, unsigned &clamps)
{
    using G = BotGrid<N>;
    const int p = threadIdx.x, lane = p & 31, warp = p >> 5;
    const CoefT<float> &cf = A.lv[L].cf;
    __syncthreads();
    // FAS right-hand side: f = op(v) + R r - m of the grid above; c = 0
    for (int q = p; q < G::CELLS; q += kBotThreads) {
        int colour;
        const BotNbr nb = bot_at<N>(q, colour);
        MG5_AT(g.f, q) = bot_op(g.v + colour * G::HC, g.v + (1 - colour) * G::HC, nb, MG5_AT(g.bs, q), MG5_AT(g.bd, q),
                        cf) + MG5_AT(g.f, q) - sh.mf;
    }
    __syncthreads();
    if constexpr (LAST) {
        bot_coarsest<N>(g, cf, A, sh, &sh.c[L], clamps);
        __syncthreads();
        g.turn(sh.iters);
        if (p == 0) {
            MG5_AT(A.lv[L].ls, 0).c = sh.c[L];
            if (A.sweeps)
                atomicAdd(&MG5_AT(A.sweeps, 0), sh.iters);
        }
    } else {
        bot_sweeps<N>(g, A.nu1, 0.0f, cf, clamps);
        g.turn(A.nu1);
        // residual, its mean (c -= m), and the 8-child means of v and r
        constexpr int NC = N / 2;
        using C = BotGrid<NC>;
        C c(g.v0 + G::CELLS);
        if constexpr (N != 8) {
            // a coarse cell a thread; the statistics as the launch of k_resid_restrict forms them: each
            // warp's shifted sums in FP32, combined in FP64 over the warps of a block of kBlock threads,
            // then over the blocks (the mean decides the FP32 rounding of all that follows)
            MomAcc<float> acc;
            if (p < C::CELLS) {
                const int row = p / NC, K = p - row * NC, I = row / NC, J = row - I * NC;
                float sv = 0.0f, sr = 0.0f;
#pragma unroll 2
                for (int ch = 0; ch < 8; ++ch) {
                    const int i = 2 * I + (ch >> 2), j = 2 * J + ((ch >> 1) & 1), k = 2 * K + (ch & 1);
                    const int colour = (i + j + k) & 1;
                    const BotNbr nb = bot_nbr<N>(i, j, k);
                    const int q = colour * G::HC + nb.r00 + nb.k0;
                    const float res = __fsub_rn(MG5_AT(g.f, q) + 0.0f, bot_op(g.v + colour * G::HC, g.v + (1 - colour) * G::HC,
                                                                       nb, MG5_AT(g.bs, q), MG5_AT(g.bd, q), cf));
                    sv += MG5_AT(g.v, q);
                    sr += res;
                    acc.add(res);
                }
                const int q = C::idx(I, J, K);
                MG5_AT(c.v, q) = MG5_AT(c.v0, q) = sv * 0.125f;
                MG5_AT(c.f, q) = sr * 0.125f;
            }
            MomT<float> v{(float)acc.n, acc.k, acc.s, acc.q};
            v = momt_shift(v, __shfl_sync(0xffffffffu, v.k, 0));
            for (int o = 16; o > 0; o >>= 1) {
                v.n += __shfl_down_sync(0xffffffffu, v.n, o);
                v.s += __shfl_down_sync(0xffffffffu, v.s, o);
            }
            if (lane == 0)
                sh.mom[warp] = Moments{(double)v.n, (double)v.k, (double)v.s, 0.0};
            __syncthreads();
            if (warp == 0) {
                // eight warps a block of the launch, at most two blocks: lanes 0 and 8 get a block's sums
                constexpr int blocks = (C::CELLS + kBlock - 1) / kBlock;
                static_assert(kBlock == 256 && blocks <= 2, "blocks of the launch");
                Moments u{0.0, 0.0, 0.0, 0.0};
                if (lane < 8 * blocks)
                    u = mom_shift(sh.mom[lane], sh.mom[lane & 8].k);
                for (int o = 4; o > 0; o >>= 1) {
                    u.n += __shfl_down_sync(0xffffffffu, u.n, o);
                    u.s += __shfl_down_sync(0xffffffffu, u.s, o);
                }
                const Moments u1{__shfl_sync(0xffffffffu, u.n, 8), sh.mom[8].k, __shfl_sync(0xffffffffu, u.s, 8), 0.0};
                if (lane == 0) {
                    if (blocks > 1) {
                        const Moments t = mom_shift(u1, u.k);
                        u.n += t.n;
                        u.s += t.s;
                    }
                    sh.m = u.n > 0.0 ? u.k + u.s / u.n : 0.0;
                }
            }
        } else {
            // 8^3: a cell a thread (its r in w), the sum in pairs
            static_assert(N != 8 || G::CELLS == kBotThreads, "a cell a thread");
            int colour;
            const BotNbr nb = bot_at<N>(p, colour);
            const float res = __fsub_rn(MG5_AT(g.f, p) + 0.0f, bot_op(g.v + colour * G::HC, g.v + (1 - colour) * G::HC, nb,
                                                               MG5_AT(g.bs, p), MG5_AT(g.bd, p), cf));
            MG5_AT(g.w, p) = res;
            float2 s = make_float2(res, 0.0f);
            for (int o = 16; o > 0; o >>= 1)
                s = pair_sum(s, pair_xor(s, o));
            if (lane == 0)
                sh.sum[warp] = s;
            __syncthreads();
            if (p < C::CELLS) {
                const int row = p / NC, K = p - row * NC, I = row / NC, J = row - I * NC;
                float sv = 0.0f, sr = 0.0f;
#pragma unroll
                for (int ch = 0; ch < 8; ++ch) {
                    const int q = G::idx(2 * I + (ch >> 2), 2 * J + ((ch >> 1) & 1), 2 * K + (ch & 1));
                    sv += MG5_AT(g.v, q);
                    sr += MG5_AT(g.w, q);
                }
                const int q = C::idx(I, J, K);
                MG5_AT(c.v, q) = MG5_AT(c.v0, q) = sv * 0.125f;
                MG5_AT(c.f, q) = sr * 0.125f;
            }
            if (warp == 0) {
                s = warps_pair_sum<kBotThreads / 32>(sh.sum);
                if (lane == 0)
                    sh.m = ((double)s.x + (double)s.y) / (double)G::CELLS;
            }
        }
        if (p == 0) {
            sh.c[L] = 0.0 - sh.m;
            sh.mf = (float)sh.m;
            MG5_AT(A.lv[L].ls, 0).m = sh.m;
        }
        bot_visit<NC, L + 1, NC == 4 || NC == 6>(c, A, sh, clamps);
        // prolongation of the correction (cell-centred trilinear), c += c of the grid below
        for (int q = p; q < C::CELLS; q += kBotThreads)
            MG5_AT(c.w, q) = MG5_AT(c.v, q) - MG5_AT(c.v0, q);
        if (p == 0) {
            sh.c[L] += sh.c[L + 1];
            sh.cf = (float)sh.c[L];
            MG5_AT(A.lv[L].ls, 0).c = sh.c[L];
        }
        __syncthreads();
        for (int q = p; q < G::CELLS; q += kBotThreads) {
            const int row = q / N, k = q - row * N, i = row / N, j = row - i * N;
            const int I = i >> 1, J = j >> 1, K = k >> 1;
            const int I2 = (i & 1) ? (I + 1 == NC ? 0 : I + 1) : (I == 0 ? NC - 1 : I - 1);
            const int J2 = (j & 1) ? (J + 1 == NC ? 0 : J + 1) : (J == 0 ? NC - 1 : J - 1);
            const int K2 = (k & 1) ? (K + 1 == NC ? 0 : K + 1) : (K == 0 ? NC - 1 : K - 1);
            const auto e = [&](int x, int y, int z) { return MG5_AT(c.w, C::idx(x, y, z)); };
            // weights (3/4, 1/4) per axis as 3x + y, one 1/64 at the end (as k_prolong_add)
            const float z00 = fmaf(3.0f, e(I, J, K), e(I, J, K2)), z01 = fmaf(3.0f, e(I, J2, K), e(I, J2, K2));
            const float z10 = fmaf(3.0f, e(I2, J, K), e(I2, J, K2)), z11 = fmaf(3.0f, e(I2, J2, K), e(I2, J2, K2));
            const float y0 = fmaf(3.0f, z00, z01), y1 = fmaf(3.0f, z10, z11);
            const float o = fmaf(3.0f, y0, y1);
            const int d = G::idx(i, j, k);
            MG5_AT(g.v, d) = fmaf(o, 1.0f / 64.0f, MG5_AT(g.v, d));
        }
        __syncthreads();
        bot_sweeps<N>(g, A.nu2, sh.cf, cf, clamps);
        g.turn(A.nu2);
    }
}

// N0: the side of the finest grid of the visit: 16 (8, 4 below it), 12 (6) or 8 (4)
template <int N0>
__global__ void __launch_bounds__(kBotThreads, 1) k_bottom(const __grid_constant__ BotArgs A)
{
    extern __shared__ __align__(16) unsigned char bot_raw[];
    __shared__ BotShared sh;
    unsigned clamps = 0;
    float *at = reinterpret_cast<float *>(bot_raw);
    // v and f of the finest of these grids, B of all (in v0 until its parts are formed)
    BotGrid<N0> g(at);
    BotGrid<N0 / 2> g1(at + BotGrid<N0>::FLOATS);
    bot_load<N0>(g.v0, A.lv[0].B);
    bot_load<N0>(g.v, A.v);
    bot_load<N0>(g.f, A.f);
    bot_load<N0 / 2>(g1.v0, A.lv[1].B);
    if constexpr (N0 == 16) {
        BotGrid<4> g2(at + BotGrid<16>::FLOATS + BotGrid<8>::FLOATS);
        bot_load<4>(g2.v0, A.lv[2].B);
    }
    if (threadIdx.x == 0)
        sh.mf = (float)MG5_AT(A.ls_up, 0).m;
    __syncthreads();
    bot_base<N0>(g);
    bot_base<N0 / 2>(g1);
    if constexpr (N0 == 16) {
        BotGrid<4> g2(at + BotGrid<16>::FLOATS + BotGrid<8>::FLOATS);
        bot_base<4>(g2);
    }
    bot_visit<N0, 0, false>(g, A, sh, clamps);
#pragma unroll
    for (int m = 0; m < (BotGrid<N0>::CELLS + kBotThreads - 1) / kBotThreads; ++m) {
        const int q = m * kBotThreads + threadIdx.x, row = q / N0, k = q - row * N0, i = row / N0, j = row - i * N0;
        if (q < BotGrid<N0>::CELLS)
            MG5_AT(A.v, q) = MG5_AT(g.v, BotGrid<N0>::idx(i, j, k));
    }
    if (clamps)
        atomicAdd(&MG5_AT(A.clamp, 0), (unsigned long long)clamps);
}

template <int N0>
constexpr int bot_smem()
{
    return (BotGrid<N0>::FLOATS + BotGrid<N0 / 2>::FLOATS + (N0 == 16 ? BotGrid<4>::FLOATS : 0)) * (int)sizeof(float);
}

template <int N0>
cudaError_t bot_prepare()
{
    return cudaFuncSetAttribute(k_bottom<N0>, cudaFuncAttributeMaxDynamicSharedMemorySize, bot_smem<N0>());
}

}  // namespace

bool bottom_ok(const int *n, int nlev)
{
    return (nlev == 3 && n[0] == 16 && n[2] == 4) || (nlev == 2 && ((n[0] == 12 && n[1] == 6) || (n[0] == 8 && n[1] == 4)));
}

cudaError_t prepare_bottom_kernel()
{
    cudaError_t e = bot_prepare<16>();
    if (e == cudaSuccess)
        e = bot_prepare<12>();
    return e == cudaSuccess ? bot_prepare<8>() : e;
}

cudaError_t launch_bottom(float *v, const float *f, const float *const *B, const int *n, int nlev,
                          const CoefT<float> *cf, const LevelScal *ls_up, LevelScal *ls, int nu1, int nu2,
                          int nu_coarse, double rtol, unsigned long long *clamp, int *sweeps, cudaStream_t st)
{
    if (!bottom_ok(n, nlev))
        return cudaErrorInvalidValue;
    BotArgs A{};
    for (int l = 0; l < nlev; ++l)
        A.lv[l] = BotLevel{cf[l], B[l], ls + l};
    A.v = v;
    A.f = f;
    A.ls_up = ls_up;
    A.nu1 = nu1;
    A.nu2 = nu2;
    A.nu_coarse = nu_coarse;
    A.rtol = rtol;
    A.clamp = clamp;
    A.sweeps = sweeps;
    if (n[0] == 16)
        k_bottom<16><<<1, kBotThreads, bot_smem<16>(), st>>>(A);
    else if (n[0] == 12)
        k_bottom<12><<<1, kBotThreads, bot_smem<12>(), st>>>(A);
    else
        k_bottom<8><<<1, kBotThreads, bot_smem<8>(), st>>>(A);
    count_launch(1);
    return cudaGetLastError();
}

}  // namespace mg5
