// k_visit.cu -- the coarse part of an FP64 V-cycle in one thread-block cluster: the visit of a
// coarse grid of up to 20000 cells and of every grid below it (FAS right-hand side, nu1 snapshot
// red-black sweeps, residual and 8-child restriction, ..., the coarsest iteration, ..., trilinear
// prolongation of the correction, nu2 sweeps; Sec. 3.1), for periodic grids and for the Dirichlet
// patch hierarchy.
//
// What bounds the level-by-level launches there is latency: 3 .. 12 us each for a few hundred ns of
// work, and FP64 at 2 lanes a clock per SM.  One kernel keeps every grid in shared memory:
//  * the planes of a grid are dealt to the 16 CTAs; grids of up to 8 planes or 512 cells and the
//    coarsest one live in CTA 0, where a barrier costs less than a cluster one and the cells still
//    fit the threads;
//  * a value is its three FP32 pieces (mg5_split.cuh) on a unit fixed for the visit (the top grid's
//    largest exponent, the size a correction can have, and two bits): the stencil is exact, an update
//    is a pair added to the pieces, rounded to 2^-58 of the largest value, and no FP64 instruction is
//    left in a sweep.  Three arrays hold the two colours and the one being written (a half-sweep reads
//    the old values of its own colour at the edges), 16 bytes a cell; a CTA's planes have copies of
//    their neighbours' planes beside them, which the neighbours write through distributed shared
//    memory as they update;
//  * the residual, its restriction and the correction pass between grids as pairs through the grids'
//    own global buffers (L2);
//  * a value that outgrows its unit raises a flag: at the end all CTAs agree and repeat the visit
//    with eight bits more, six times at most.  Where that is not enough, or values are not finite, the
//    visit leaves no correction: v = v0, c = 0 (the grid above keeps its own sweeps and its residual test).
//
// Measured on GB300 (a visit, launches -> cluster): top grid 16^3 periodic 130 -> 67 us, with the
// 32^3 patch's 16^3 grid below it 100 -> 46 us.  A half-sweep takes 2.1 kclk at 4^3, 2.95 at 8^3 and 3.6
// at 16^3: a chain of ~450 dependent instructions, and at 16^3 the cluster barrier.  Tried: two cells a
// thread in packed or in interleaved arithmetic (slower: the packed instructions' latency; the code
// outgrows the instruction cache).
//
// The FAS right-hand side is formed by the same pair arithmetic as the residual (relative 2^-47); the
// corrections it leads to vanish with the residual, so the V-cycles converge as before.
#include <cooperative_groups.h>

#include "mg5_fin.cuh"
#include "mg5_split.cuh"
#include "mg5_visit.cuh"

namespace mg5 {

namespace cg = cooperative_groups;
using namespace split::one;
using split::Kap;
using split::kUnitBias;

namespace {

constexpr int VT = 512;                 // threads
constexpr float kPieceMax = 1048576.0f; // 2^20: sums of 12 pieces stay exact
constexpr int kRestarts = 6;
constexpr int kHold = 4;                // top-grid cells a thread holds in registers

__device__ __forceinline__ int div_by(int t, unsigned m) { return m ? (int)__umulhi((unsigned)t, m) : t; }

struct VisitShared {
    Pr c[kVisitLevels];   // compatibility constants, units u / h^2 of their grids
    Kap kap;              // of the top grid
    int ebs[kVisitCtas];
    Pr sums[kVisitCtas];
    Pr red[2][2][VT / 32];
    int emax;
    int flags[kVisitCtas];
    int flag;
};

__device__ __forceinline__ double pow2d(int e) { return __hiloint2double((e + 1023) << 20, 0); }
__device__ __forceinline__ Pr shfl_down(const Pr &x, int q)
{
    return Pr{__shfl_down_sync(0xffffffffu, x.h, q), __shfl_down_sync(0xffffffffu, x.l, q)};
}
__device__ __forceinline__ float pow2f(int e)
{
    e = e < -126 ? -126 : (e > 127 ? 127 : e);
    return __int_as_float((e + 127) << 23);
}
__device__ __forceinline__ Pr pair_at(double x, int k)
{
    return pair_scaled((unsigned)__double2hiint(x), (unsigned)__double2loint(x), k);
}
// (x) 2^(eb - kUnitBias) as a double
__device__ __forceinline__ double to_f64(const Pr &x, int eb)
{
    unsigned h0, l0, h1, l1;
    split::unit_words(x.h, eb, h0, l0);
    split::unit_words(x.l, eb, h1, l1);
    const double d = __hiloint2double((int)h0, (int)l0) + __hiloint2double((int)h1, (int)l1);
    return fabsf(x.h) < 1e30f ? d : __longlong_as_double(0x7ff8000000000000ll);
}

// One visit.  Positions: p a plane of this CTA counted from its first one (-1 and np: the copies of the
// neighbours' planes, or a box's ghost planes), i = i0 + p; interior cells j, k.
template <bool BOX>
struct Visit {
    const VisitArgs &A;
    VisitShared &S;
    float4 *sm;
    cg::cluster_group cluster;
    int rank, tid;
    unsigned clamps = 0;
    int sweeps = 0;
    int eb = 0;      // the visit's exponent: u = 2^(eb - kUnitBias)
    bool finite = true;   // of the top grid's values
    int turn = 0;    // of the reduction buffers

    // the planes [i0, i0 + np) of level l this CTA owns
    struct Own {
        int i0, np;
    };
    __device__ __forceinline__ Own own(const VisitLevel &L, int r) const
    {
        if (L.single)
            return Own{0, r == 0 ? L.n0 : 0};
        const int i0 = r * L.P, np = min(L.n0 - i0, L.P);
        return Own{i0, np > 0 ? np : 0};
    }
    __device__ __forceinline__ void bar(const VisitLevel &L)
    {
        if (L.single)
            __syncthreads();
        else
            cluster.sync();
    }
    // Three arrays hold the two colours and the one a half-sweep writes, in turn: after b sweeps
    // (mod 3) colour 0 is array (3 - b) % 3, colour 1 (4 - b) % 3 and the free one (5 - b) % 3.
    static __device__ __forceinline__ int mod3(int x) { return x >= 3 ? x - 3 : x; }
    static __device__ __forceinline__ int arr(int colour, int b) { return mod3(3 + colour - b); }
    // a place in an array: a box keeps its ghost shell, a periodic grid wraps its indices; planes have
    // their neighbours on both sides unless CTA 0 holds the whole periodic grid
    __device__ __forceinline__ int at(const VisitLevel &L, int p, int j, int k) const
    {
        return BOX ? ((p + 1) * (L.n1 + 2) + j + 1) * L.wq + ((k + 1) >> 1)
                   : ((p + 1 - L.single) * L.n1 + j) * L.wq + (k >> 1);
    }
    __device__ __forceinline__ float4 *array(const VisitLevel &L, int a) const { return sm + L.pieces + a * L.sz; }
    static __device__ __forceinline__ P1 ld(const float4 &x) { return P1{x.x, x.y, x.z}; }
    static __device__ __forceinline__ float4 st(const P1 &x) { return make_float4(x.h, x.m, x.l, 0.0f); }
    // Interior cell into array a, and into the neighbours' copies of its plane.
    __device__ __forceinline__ void put(const VisitLevel &L, const Own &o, int a, int p, int j, int k, const P1 &x)
    {
        const float4 v = st(x);
        const int q = at(L, p, j, k);
        MG5_AT(array(L, a), q) = v;
        if (L.single)
            return;
        const int ps = (BOX ? L.n1 + 2 : L.n1) * L.wq;
        if (p == 0 && (!BOX || rank > 0)) {
            const int r = rank == 0 ? L.act - 1 : rank - 1;
            cluster.map_shared_rank(array(L, a), r)[q + own(L, r).np * ps] = v;
        }
        if (p == o.np - 1 && (!BOX || rank < L.act - 1)) {
            const int r = rank == L.act - 1 ? 0 : rank + 1;
            cluster.map_shared_rank(array(L, a), r)[q - o.np * ps] = v;
        }
    }
    // The stencil of cell (p, j, k): centre and edges from array ac, faces from array ao.
    __device__ __forceinline__ Lin1 lin_at(const VisitLevel &L, int ac, int ao, int p, int j, int k) const
    {
        const int ps = (BOX ? L.n1 + 2 : L.n1) * L.wq, row = L.wq;
        int xp = ps, xm = -ps, yp = row, ym = -row, zp, zm;
        if (BOX) {
            zp = (k + 1) & 1;
            zm = zp - 1;
        } else {
            if (L.single) {
                xp = p == L.n0 - 1 ? -(L.n0 - 1) * ps : ps;
                xm = p == 0 ? (L.n0 - 1) * ps : -ps;
            }
            yp = j == L.n1 - 1 ? -(L.n1 - 1) * row : row;
            ym = j == 0 ? (L.n1 - 1) * row : -row;
            zp = k == L.n2 - 1 ? -(k >> 1) : (k & 1);
            zm = k == 0 ? row - 1 : (k & 1) - 1;
        }
        const int q = at(L, p, j, k);
        const float4 *a = array(L, ac) + q, *b = array(L, ao) + q;
        const auto Av = [&](int x) { return ld(MG5_AT(a, x)); };
        const auto Ov = [&](int x) { return ld(MG5_AT(b, x)); };
        return lin_of(Av(0), Ov(xp) + Ov(xm), Ov(yp) + Ov(ym), Ov(zp) + Ov(zm),
                      (Av(xp + yp) - Av(xp + ym)) - (Av(xm + yp) - Av(xm + ym)),
                      (Av(xp + zp) - Av(xp + zm)) - (Av(xm + zp) - Av(xm + zm)),
                      (Av(yp + zp) - Av(yp + zm)) - (Av(ym + zp) - Av(ym + zm)));
    }
    __device__ __forceinline__ P1 centre(const VisitLevel &L, int b, int p, int j, int k, int colour) const
    {
        return ld(MG5_AT(array(L, arr(colour, b)), at(L, p, j, k)));
    }
    __device__ __forceinline__ float2 &Fat(const VisitLevel &L, int p, int j, int k) const
    {
        return MG5_AT(reinterpret_cast<float2 *>(sm + L.F), (p * L.n1 + j) * L.n2 + k);
    }
    __device__ __forceinline__ Pr Fget(const VisitLevel &L, int p, int j, int k) const
    {
        const float2 f = Fat(L, p, j, k);
        return Pr{f.x, f.y};
    }
    // every interior cell (p, j, k) of this CTA
    template <typename F>
    __device__ __forceinline__ void cells(const VisitLevel &L, const Own &o, const F &f)
    {
        const int n = o.np * L.n1 * L.n2;
#pragma unroll 1
        for (int t = tid; t < n; t += VT) {
            const int q = div_by(t, L.m2), k = t - q * L.n2, p = div_by(q, L.m1), j = q - p * L.n1;
            f(p, j, k);
        }
    }
    __device__ __forceinline__ long long gcell(const VisitLevel &L, int i, int j, int k) const
    {
        return ((long long)i * L.n1 + j) * L.n2 + k;
    }
    // a cell's place in the level's v0 and v (box: with its ghost shell)
    __device__ __forceinline__ long long vcell(const VisitLevel &L, int i, int j, int k) const
    {
        return BOX ? ((long long)(i + 1) * (L.n1 + 2) + j + 1) * (L.n2 + 2) + k + 1 : gcell(L, i, j, k);
    }
    __device__ __forceinline__ double v0_at(const VisitLevel &L, int i, int j, int k) const
    {
        return __ldcg(&MG5_AT(L.v0, vcell(L, i, j, k)));
    }
    // h^2 x / u as a pair
    __device__ __forceinline__ Pr in_units(const VisitLevel &L, double x) const
    {
        return mul_pair(pair_at(x, kUnitBias - eb + L.Hq), Pr{L.Hh, L.Hl});
    }
    __device__ __forceinline__ P1 split_f64(double x) const
    {
        return split1((unsigned)__double2hiint(x), (unsigned)__double2loint(x), eb);
    }
    // ... of a value that may not fit the unit
    __device__ __forceinline__ P1 split_checked(double x)
    {
        if (((__double2hiint(x) >> 20) & 0x7ff) > eb)
            S.flag = 1;
        return split_f64(x);
    }
    // the change of a cell since the visit began
    __device__ __forceinline__ Pr change(const P1 &now, double v0) const { return pair_of(now - split_f64(v0)); }
    // kappa of a grid: a quarter of the parent's, whose h is half of its own
    __device__ __forceinline__ Kap kap_of(const VisitLevel &L) const
    {
        const float s = pow2f(-2 * L.id);
        return Kap{S.kap.k3h * s, S.kap.k3l * s, S.kap.kh * s, S.kap.kl * s};
    }

    // ---- a box's ghosts: v0(g) + w^m (v(a) - v0(a)), a the nearest interior cell, m axes outside
    struct Ghost {
        int p, j, k, m;       // its place
        int pa, ja, ka, ca;   // the interior cell and its colour
    };
    // Ghost number t of this CTA: the rings around its planes and their two neighbours, then the
    // insides of a ghost plane.
    __device__ __forceinline__ int ghost_count(const VisitLevel &L, const Own &o) const
    {
        if (!BOX || o.np == 0)
            return 0;
        const int ends = (o.i0 == 0) + (o.i0 + o.np == L.n0);
        return (o.np + 2) * L.ring + ends * L.n1 * L.n2;
    }
    __device__ __forceinline__ Ghost ghost(const VisitLevel &L, const Own &o, int t) const
    {
        Ghost g;
        const int rings = (o.np + 2) * L.ring;
        if (t < rings) {
            const int pl = div_by(t, L.mring), r = t - pl * L.ring, row = L.n2 + 2;
            g.p = pl - 1;
            if (r < 2 * row) {
                g.j = r < row ? -1 : L.n1;
                g.k = (r < row ? r : r - row) - 1;
            } else {
                g.j = (r - 2 * row) >> 1;
                g.k = (r & 1) ? L.n2 : -1;   // 2 row is even
            }
        } else {
            const int inside = L.n1 * L.n2;
            int u = t - rings;
            const bool second = u >= inside || o.i0 != 0;
            if (u >= inside)
                u -= inside;
            g.p = second ? o.np : -1;
            g.j = div_by(u, L.m2);
            g.k = u - g.j * L.n2;
        }
        const int i = o.i0 + g.p, ia = min(max(i, 0), L.n0 - 1);
        g.ja = min(max(g.j, 0), L.n1 - 1);
        g.ka = min(max(g.k, 0), L.n2 - 1);
        g.pa = ia - o.i0;
        g.m = (i != ia) + (g.j != g.ja) + (g.k != g.ka);
        g.ca = (ia + g.ja + g.ka) & 1;
        return g;
    }
    __device__ __forceinline__ Pr weight(const VisitLevel &L, int m) const { return Pr{L.w[m - 1][0], L.w[m - 1][1]}; }
    // The ghosts after a half-sweep (k_patch_half's order): after the red one every ghost of the
    // sweep's result, after the black one those of the black cells.  a0, a1: the arrays of the two
    // colours' values; d0, d1: of the ghosts.  (v0 does not change any more, and the barrier after it was
    // written is an acquire: it may come from L1.)
    __device__ __forceinline__ void ghosts_follow(const VisitLevel &L, const Own &o, bool black, int a0, int a1,
                                                  int d0, int d1)
    {
        const int n = ghost_count(L, o);
#pragma unroll 1
        for (int t = tid; t < n; t += VT) {
            const Ghost g = ghost(L, o, t);
            if (black && g.ca == 0)
                continue;
            const double vg = MG5_AT(L.v0, vcell(L, o.i0 + g.p, g.j, g.k)),
                         va = MG5_AT(L.v0, vcell(L, o.i0 + g.pa, g.ja, g.ka));
            const P1 now = ld(MG5_AT(array(L, g.ca ? a1 : a0), at(L, g.pa, g.ja, g.ka)));
            const P1 x = add_change(split_f64(vg), mul_pair(weight(L, g.m), change(now, va)));
            MG5_AT(array(L, (g.ca ^ (g.m & 1)) ? d1 : d0), at(L, g.p, g.j, g.k)) = st(x);
        }
    }

    // The top grid from the caller's v and f; its exponent is the whole visit's (means and ghosts of
    // the grids below are no larger, nor are their corrections).
    __device__ __forceinline__ void enter_top(const VisitLevel &L, int margin)
    {
        const Own o = own(L, rank);
        if (tid == 0)
            S.emax = 0;
        __syncthreads();
        const int grow = L.nmax2 + L.Hq - 4;   // log2 of a correction's size over its residual's
        const int n = o.np * L.n1 * L.n2;
        int emax = 0;
        double x[kHold], f[kHold];   // the first kHold cells stay in registers
        const auto load = [&](int t, double &v, double &r) {
            const int q = div_by(t, L.m2), k = t - q * L.n2, p = div_by(q, L.m1), j = q - p * L.n1;
            v = v0_at(L, o.i0 + p, j, k);
            r = MG5_AT(L.f, gcell(L, o.i0 + p, j, k));
        };
        const auto see = [&](double v, double r) {
            const int ef = (__double2hiint(r) >> 20) & 0x7ff, ev = (__double2hiint(v) >> 20) & 0x7ff;
            emax = max(emax, max(ev, ef == 2047 ? 2047 : (ef > 0 ? min(ef + grow, 2046) : 0)));
        };
#pragma unroll
        for (int m = 0; m < kHold; ++m) {
            x[m] = f[m] = 0.0;
            if (tid + m * VT < n)
                load(tid + m * VT, x[m], f[m]);
        }
#pragma unroll
        for (int m = 0; m < kHold; ++m)
            see(x[m], f[m]);
#pragma unroll 1
        for (int t = tid + kHold * VT; t < n; t += VT) {
            double v, r;
            load(t, v, r);
            see(v, r);
        }
        const int ng = ghost_count(L, o);
#pragma unroll 1
        for (int t = tid; t < ng; t += VT) {   // the ghosts' fixed values
            const Ghost g = ghost(L, o, t);
            emax = max(emax, (__double2hiint(v0_at(L, o.i0 + g.p, g.j, g.k)) >> 20) & 0x7ff);
        }
        emax = __reduce_max_sync(0xffffffffu, emax);
        if ((tid & 31) == 0)
            atomicMax(&S.emax, emax);
        __syncthreads();
        // every CTA takes part, also where CTA 0 holds the grid alone
        if (tid < kVisitCtas)
            cluster.map_shared_rank(S.ebs, tid)[rank] = S.emax;
        cluster.sync();
        emax = 0;
        for (int r = 0; r < kVisitCtas; ++r)
            emax = max(emax, S.ebs[r]);
        eb = min(max((emax == 0 ? 1023 : emax) + margin, 200), 1800);
        finite = emax < 2047;
        if (tid == 0) {
            // (one thread: an FP64 instruction of every warp would take 256 clocks)
            const double k1 = L.k * pow2d(eb - kUnitBias), k3 = 3.0 * k1;
            S.kap.k3h = (float)k3;
            S.kap.k3l = (float)(k3 - (double)S.kap.k3h);
            S.kap.kh = (float)k1;
            S.kap.kl = (float)(k1 - (double)S.kap.kh);
        }
        const auto keep = [&](int t, double v, double r) {
            const int q = div_by(t, L.m2), k = t - q * L.n2, p = div_by(q, L.m1), j = q - p * L.n1;
            put(L, o, arr((o.i0 + p + j + k) & 1, 0), p, j, k, split_checked(v));
            const Pr F = in_units(L, r);
            Fat(L, p, j, k) = make_float2(F.h, F.l);
        };
#pragma unroll
        for (int m = 0; m < kHold; ++m)
            if (tid + m * VT < n)
                keep(tid + m * VT, x[m], f[m]);
#pragma unroll 1
        for (int t = tid + kHold * VT; t < n; t += VT) {
            double v, r;
            load(t, v, r);
            keep(t, v, r);
        }
    }
    // A grid below from its parent's values and residuals, 8-child means; r comes in the parent's unit
    // u / h^2, a quarter of its own.
    __device__ __forceinline__ void enter_below(const VisitLevel &L, const VisitLevel &U)
    {
        const Own o = own(L, rank);
        cells(L, o, [&](int p, int j, int k) {
            const int i = o.i0 + p;
            double s[8];
            float2 q[8];
#pragma unroll
            for (int ch = 0; ch < 8; ++ch) {
                const int fi = 2 * i + (ch >> 2), fj = 2 * j + ((ch >> 1) & 1), fk = 2 * k + (ch & 1);
                s[ch] = __ldcg(&MG5_AT(U.v, vcell(U, fi, fj, fk)));
                q[ch] = __ldcg(&MG5_AT(U.x, gcell(U, fi, fj, fk)));
            }
            const double x = 0.125 * (((s[0] + s[1]) + (s[2] + s[3])) + ((s[4] + s[5]) + (s[6] + s[7])));
            MG5_AT(L.v0, vcell(L, i, j, k)) = x;
            const auto add2 = [&](int a) { return add_pair(Pr{q[a].x, q[a].y}, Pr{q[a + 1].x, q[a + 1].y}); };
            const Pr r = add_pair(add_pair(add2(0), add2(2)), add_pair(add2(4), add2(6)));
            Fat(L, p, j, k) = make_float2(0.5f * r.h, 0.5f * r.l);
            put(L, o, arr((i + j + k) & 1, 0), p, j, k, split_checked(x));
        });
    }
    // ... then the ghosts' fixed values and c = 0
    __device__ __forceinline__ void entered(const VisitLevel &L)
    {
        const Own o = own(L, rank);
        const int ng = ghost_count(L, o);
#pragma unroll 1
        for (int t = tid; t < ng; t += VT) {
            const Ghost g = ghost(L, o, t);
            MG5_AT(array(L, arr(g.ca ^ (g.m & 1), 0)), at(L, g.p, g.j, g.k)) = st(split_checked(v0_at(L, o.i0 + g.p, g.j, g.k)));
        }
        if (tid == 0)
            S.c[L.id] = Pr{0.0f, 0.0f};
        bar(L);
    }

    // The residual of every cell.  RHS: F = op(v) + R r - m of the parent, entering a grid.  DOWN: r and
    // v for the restriction onto the next grid, sum of r.  TEST: sums of r and r^2 (c not counted).
    enum Mode { RHS, DOWN, TEST };
    __device__ __forceinline__ void residuals(const VisitLevel &L, int mode, int b, const Pr &Pm, Pr &sum, Pr &sq)
    {
        const Own o = own(L, rank);
        const Kap kap = kap_of(L);
        const Pr c = S.c[L.id];
        Pr mean{0.0f, 0.0f};
        if (!BOX && mode == RHS)   // (the parent's unit u / h^2 is four of L's)
            mean = L.id > 0 ? scale(Pm, 4.0f) : in_units(L, MG5_AT(A.m_up, 0));
        sum = Pr{0.0f, 0.0f};
        sq = Pr{0.0f, 0.0f};
        cells(L, o, [&](int p, int j, int k) {
            const int i = o.i0 + p, col = (i + j + k) & 1;
            Pr F;
            double v0 = 0.0;
            if (mode == RHS) {
                F = add_pair(mean, neg(Fget(L, p, j, k)));
            } else {
                F = Fget(L, p, j, k);
                if (mode == DOWN) {
                    v0 = v0_at(L, i, j, k);
                    F = add_pair(F, c);
                }
            }
            const Pr r = resid(lin_at(L, arr(col, b), arr(col ^ 1, b), p, j, k), F, kap);
            if (mode == RHS) {
                Fat(L, p, j, k) = make_float2(-r.h, -r.l);
                return;
            }
            if (mode == DOWN) {
                MG5_AT(L.x, gcell(L, i, j, k)) = make_float2(r.h, r.l);
                // v = v0 + the change since then
                MG5_AT(L.v, vcell(L, i, j, k)) = v0 + to_f64(change(centre(L, b, p, j, k, col), v0), eb);
            } else {
                sq = add_pair(sq, sqr(r));
            }
            sum = add_pair(sum, r);
        });
    }

    // `count` sweeps after b (mod 3); returns b + count (mod 3).  Where a thread's cells lie (plane,
    // row, k >> 1) is found once per call, for the first two.
    __device__ __forceinline__ int sweep(const VisitLevel &L, int count, int b)
    {
        const Own o = own(L, rank);
        const Kap kap = kap_of(L);
        const Pr c = S.c[L.id];
        const int nq = (L.n2 + 1) >> 1, n = o.np * L.n1 * nq;
        const auto find = [&](int t) {
            const int g = div_by(t, L.mq), p = div_by(g, L.m1);
            return (p << 20) | ((g - p * L.n1) << 10) | (t - g * nq);
        };
        const int pos0 = find(tid), pos1 = find(tid + VT);
#pragma unroll 1
        for (int s = 0; s < 2 * count; ++s) {
            const int black = s & 1, a0 = arr(0, b), a1 = arr(1, b), free_ = mod3(5 - b);
            // red: array a0 -> the free one; black: a1 -> what was a0
            const int ac = black ? a1 : a0, ao = black ? free_ : a1, ad = black ? a0 : free_;
#pragma unroll 1
            for (int t = tid; t < n; t += VT) {
                const int pos = t == tid ? pos0 : (t == tid + VT ? pos1 : find(t));
                const int p = pos >> 20, j = (pos >> 10) & 1023;
                const int k = 2 * (pos & 1023) + ((o.i0 + p + j + black) & 1);
                if (k >= L.n2)
                    continue;
                const Pr F = Fget(L, p, j, k);
                const P1 now = ld(MG5_AT(array(L, ac), at(L, p, j, k)));
                const Lin1 lin = lin_at(L, ac, ao, p, j, k);
                const Pr r = resid(lin, add_pair(F, c), kap);
                const Pr d = neg(mul_pair(root_change(lin, r, kap, clamps), Pr{L.wh, L.wl}));
                const P1 x = add_change(now, d);
                if (!(fabsf(x.h) <= kPieceMax && fabsf(d.h) <= 2.0f * kPieceMax))   // (NaN too)
                    S.flag = 1;
                put(L, o, ad, p, j, k, x);
            }
            bar(L);
            if (BOX) {
                // red: the result's arrays are free_ (red) and a0 (black); black values still in a1
                ghosts_follow(L, o, black, free_, black ? a0 : a1, free_, a0);
                __syncthreads();
            }
            if (black)
                b = mod3(b + 1);
        }
        return b;
    }
    // Sums of two pairs over the CTA, in every thread (fixed order; in pair arithmetic: an FP64
    // reduction of 16 warps would take over a microsecond).
    __device__ __forceinline__ void block_sums(Pr &x, Pr &y)
    {
        for (int q = 16; q > 0; q >>= 1) {
            x = add_pair(x, shfl_down(x, q));
            y = add_pair(y, shfl_down(y, q));
        }
        turn ^= 1;   // (the other buffer's readers have passed a barrier since)
        if ((tid & 31) == 0) {
            S.red[turn][0][tid >> 5] = x;
            S.red[turn][1][tid >> 5] = y;
        }
        __syncthreads();
        x = S.red[turn][0][tid & 15];
        y = S.red[turn][1][tid & 15];
        const auto other = [](const Pr &z, int q) {
            return Pr{__shfl_xor_sync(0xffffffffu, z.h, q), __shfl_xor_sync(0xffffffffu, z.l, q)};
        };
        for (int q = VT / 64; q > 0; q >>= 1) {
            x = add_pair(x, other(x, q));
            y = add_pair(y, other(y, q));
        }
    }
    // After the DOWN residuals: the mean residual (periodic), taken off c.
    __device__ __forceinline__ Pr mean_residual(const VisitLevel &L, Pr sum)
    {
        Pr mean{0.0f, 0.0f}, none{0.0f, 0.0f};
        if (BOX) {
            bar(L);
            return mean;
        }
        block_sums(sum, none);
        if (!L.single && tid < kVisitCtas)
            cluster.map_shared_rank(S.sums, tid)[rank] = sum;
        bar(L);
        if (!L.single) {
            sum = S.sums[0];
            for (int r = 1; r < L.act; ++r)
                sum = add_pair(sum, S.sums[r]);
        }
        mean = mul_pair(sum, Pr{L.inv_h, L.inv_l});
        if (tid == 0)
            S.c[L.id] = add_pair(S.c[L.id], neg(mean));
        __syncthreads();
        return mean;
    }
    // The correction since v0 as pairs, ghosts included, for the prolongation onto the grid above.
    __device__ __forceinline__ void leave_up(const VisitLevel &L, int b)
    {
        const Own o = own(L, rank);
        cells(L, o, [&](int p, int j, int k) {
            const int i = o.i0 + p;
            const Pr e = change(centre(L, b, p, j, k, (i + j + k) & 1), v0_at(L, i, j, k));
            MG5_AT(L.x, vcell(L, i, j, k)) = make_float2(e.h, e.l);
        });
        const int ng = ghost_count(L, o);
        for (int t = tid; t < ng; t += VT) {
            const Ghost g = ghost(L, o, t);
            const int i = o.i0 + g.p;
            if (i >= 0 && i < L.n0 && (g.p < 0 || g.p >= o.np))
                continue;   // a neighbour's plane
            const Pr e = change(centre(L, b, g.pa, g.ja, g.ka, g.ca), v0_at(L, o.i0 + g.pa, g.ja, g.ka));
            const Pr w = mul_pair(weight(L, g.m), e);
            MG5_AT(L.x, vcell(L, i, g.j, g.k)) = make_float2(w.h, w.l);
        }
    }
    // v += P (correction of the grid below), c += its c
    __device__ __forceinline__ void prolong(const VisitLevel &L, int b)
    {
        const Own o = own(L, rank);
        const VisitLevel &D = A.lev[L.id + 1];
        const auto three = [](const Pr &x, const Pr &y) {   // 3 x + y
            const float p = mul(3.0f, x.h), e = fma(3.0f, x.h, -p);
            const Pr s = two_sum(p, y.h);
            return Pr{s.h, add(s.l, add(e, fma(3.0f, x.l, y.l)))};
        };
        cells(L, o, [&](int p, int j, int k) {
            const int i = o.i0 + p, col = (i + j + k) & 1;
            int a[3] = {i >> 1, j >> 1, k >> 1};
            int n[3] = {(i & 1) ? a[0] + 1 : a[0] - 1, (j & 1) ? a[1] + 1 : a[1] - 1, (k & 1) ? a[2] + 1 : a[2] - 1};
            if (!BOX) {
                n[0] = n[0] < 0 ? D.n0 - 1 : (n[0] == D.n0 ? 0 : n[0]);
                n[1] = n[1] < 0 ? D.n1 - 1 : (n[1] == D.n1 ? 0 : n[1]);
                n[2] = n[2] < 0 ? D.n2 - 1 : (n[2] == D.n2 ? 0 : n[2]);
            }
            const auto E = [&](int x, int y, int z) {
                const float2 q = __ldcg(&MG5_AT(D.x, vcell(D, x, y, z)));
                return Pr{q.x, q.y};
            };
            const auto line = [&](int x, int y) { return three(E(x, y, a[2]), E(x, y, n[2])); };
            const Pr y0 = three(line(a[0], a[1]), line(a[0], n[1])), y1 = three(line(n[0], a[1]), line(n[0], n[1]));
            const Pr d = scale(three(y0, y1), 1.0f / 64.0f);
            const P1 x = add_change(centre(L, b, p, j, k, col), d);
            if (!(fabsf(x.h) <= kPieceMax && fabsf(d.h) <= 2.0f * kPieceMax))
                S.flag = 1;
            put(L, o, arr(col, b), p, j, k, x);   // (a box's ghosts follow in the next sweep, as in k_patch_half)
        });
        if (!BOX) {
            // c of the grid below from its unit u / h^2 (h^2 four times this one's)
            const Pr c = add_pair(S.c[L.id], scale(S.c[D.id], 0.25f));
            __syncthreads();
            if (tid == 0)
                S.c[L.id] = c;
        }
        bar(L);
    }
    // The coarsest grid's stopping rule (in CTA 0; as k_coarsest, k_pbox_coarsest): c = minus the mean
    // residual; stop at rtol times the first norm.  r0: the first squared norm (negative: none yet).
    __device__ __forceinline__ bool coarsest_done(const VisitLevel &L, Pr sum, Pr sq, float &r0)
    {
        block_sums(sum, sq);
        if (!BOX) {
            const Pr m = mul_pair(sum, Pr{L.inv_h, L.inv_l});
            sq = add_pair(sq, neg(mul_pair(sum, m)));
            if (tid == 0)
                S.c[L.id] = neg(m);
            __syncthreads();
        }
        const float rn = sq.h > 0.0f ? sq.h : 0.0f;
        if (r0 < 0.0f)
            r0 = rn;
        return rn <= (float)(A.rtol * A.rtol) * r0;
    }

    // One visit.  A loop over steps, so that the code of a residual pass and of a half-sweep exists
    // once: inlined at each of their uses it outgrew the instruction cache (a half-sweep of 8^3 took
    // 4400 clocks).
    enum Step { ENTER, DOWNWARD, COARSEST, UPWARD, DONE };
    __device__ __forceinline__ bool run(int margin, bool last_attempt)
    {
        if (tid == 0)
            S.flag = 0;
        cluster.sync();   // (also: every CTA of the cluster has started)
        const int last = A.nlev - 1, bdn = A.nu1 % 3;   // bdn: the arrays' turn a grid is left in on the way down
        int split_at = A.nlev;                          // first level held by CTA 0 alone
        while (split_at > 0 && A.lev[split_at - 1].single)
            --split_at;
        int l = 0, b = 0, it = 0, step = ENTER;
        float r0 = -1.0f;
        Pr mean{0.0f, 0.0f};
        enter_top(A.lev[0], margin);
        if (split_at == 0 && rank != 0)
            step = DONE;
#pragma unroll 1
        while (step != DONE) {
            const VisitLevel &L = A.lev[l];
            int count = 0;
            if (step == UPWARD) {
                if (l == split_at - 1) {
                    // CTA 0's correction, with its c, for the grid that the CTAs share
                    if (!BOX && rank == 0 && tid > 0 && tid < kVisitCtas)
                        cluster.map_shared_rank(S.c, tid)[split_at] = S.c[split_at];
                    cluster.sync();
                }
                prolong(L, bdn);
                b = bdn;
                count = A.nu2;
            } else {
                if (step == ENTER) {
                    if (l > 0)
                        enter_below(L, A.lev[l - 1]);
                    entered(L);
                }
                Pr sum, sq;
                residuals(L, step == ENTER ? RHS : (step == DOWNWARD ? DOWN : TEST), step == ENTER ? 0 : b, mean, sum,
                          sq);
                if (step == ENTER) {
                    __syncthreads();   // F, read by other threads in a sweep
                    b = 0;
                    if (l == last) {
                        step = COARSEST;
                        continue;
                    }
                    count = A.nu1;
                } else if (step == DOWNWARD) {
                    mean = mean_residual(L, sum);
                    ++l;
                    step = ENTER;
                    if (A.lev[l].single && rank != 0) {
                        l = split_at - 1;
                        step = UPWARD;
                    }
                    continue;
                } else {
                    if (it < A.nu_coarse && !coarsest_done(L, sum, sq, r0)) {
                        ++it;
                        count = 1;
                    } else {
                        if (l > 0)
                            leave_up(L, b);
                        __syncthreads();
                        step = l > 0 ? UPWARD : DONE;
                        --l;
                        continue;
                    }
                }
            }
            b = sweep(L, count, b);
            if (step == ENTER) {
                step = DOWNWARD;
            } else if (step == UPWARD) {
                if (l > 0) {
                    leave_up(L, b);
                    bar(L);
                }
                if (--l < 0 || (A.lev[l].single && rank != 0))
                    step = DONE;
            }
        }
        sweeps += it;
        // agree on the flag
        __syncthreads();
        if (tid < kVisitCtas)
            cluster.map_shared_rank(S.flags, tid)[rank] = S.flag;
        cluster.sync();
        int any = 0;
        for (int r = 0; r < kVisitCtas; ++r)
            any |= S.flags[r];
        if (any && !last_attempt && finite)
            return false;
        // the top grid's iterate and c
        const VisitLevel &L = A.lev[0];
        const Own o = own(L, rank);
        const int n = o.np * L.n1 * L.n2;
#pragma unroll 1
        for (int t0 = tid; t0 < n; t0 += kHold * VT) {
            double v0[kHold];
#pragma unroll
            for (int m = 0; m < kHold; ++m) {
                const int t = t0 + m * VT, q = div_by(t, L.m2), k = t - q * L.n2, p = div_by(q, L.m1), j = q - p * L.n1;
                v0[m] = t < n ? v0_at(L, o.i0 + p, j, k) : 0.0;
            }
#pragma unroll
            for (int m = 0; m < kHold; ++m) {
                const int t = t0 + m * VT, q = div_by(t, L.m2), k = t - q * L.n2, p = div_by(q, L.m1), j = q - p * L.n1;
                const int i = o.i0 + p;
                if (t < n)
                    MG5_AT(L.v, vcell(L, i, j, k)) =
                        any ? v0[m] : v0[m] + to_f64(change(centre(L, b, p, j, k, (i + j + k) & 1), v0[m]), eb);
            }
        }
        const int ng = ghost_count(L, o);
        for (int t = tid; t < ng; t += VT) {
            const Ghost g = ghost(L, o, t);
            const int i = o.i0 + g.p;
            if (i >= 0 && i < L.n0 && (g.p < 0 || g.p >= o.np))
                continue;
            const Pr e = change(centre(L, b, g.pa, g.ja, g.ka, g.ca), v0_at(L, o.i0 + g.pa, g.ja, g.ka));
            const double vg = v0_at(L, i, g.j, g.k);
            MG5_AT(L.v, vcell(L, i, g.j, g.k)) = any ? vg : vg + to_f64(mul_pair(weight(L, g.m), e), eb);
        }
        if (!BOX && rank == 0 && tid == 0)
            MG5_AT(A.c_out, 0) = any ? 0.0 : to_f64(S.c[0], eb) / L.h2;
        return true;
    }
};

template <bool BOX>
__global__ void __launch_bounds__(VT, 1) k_visit(const __grid_constant__ VisitArgs A)
{
    extern __shared__ __align__(16) float4 visit_sm[];
    __shared__ VisitShared S;
    cg::cluster_group cluster = cg::this_cluster();
    Visit<BOX> V{A, S, visit_sm, cluster, (int)cluster.block_rank(), (int)threadIdx.x};
    for (int it = 0;; ++it) {
        V.clamps = 0;
        V.sweeps = 0;
        if (V.run(A.headroom + 8 * it, it == kRestarts))
            break;
    }
    if (V.clamps)
        atomicAdd(&MG5_AT(A.clamp, 0), (unsigned long long)V.clamps);
    if (V.rank == 0 && V.tid == 0 && A.sweeps)
        atomicAdd(&MG5_AT(A.sweeps, 0), V.sweeps);
    cluster.sync();   // no CTA leaves while another may still write to its shared memory
}

cudaLaunchConfig_t cluster_config(int smem, cudaStream_t st, cudaLaunchAttribute *at)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kVisitCtas);
    cfg.blockDim = dim3(VT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = kVisitCtas;
    at->val.clusterDim.y = at->val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}

unsigned magic(int d) { return d < 2 ? 0u : (unsigned)((0x100000000ull + d - 1) / d); }

}  // namespace

bool visit_plan(const int (*q)[3], int nlev, bool box, VisitArgs *A)
{
    if (nlev < 1 || nlev > kVisitLevels)
        return false;
    int quads = 0;   // of 16 bytes
    for (int l = 0; l < nlev; ++l) {
        VisitLevel &L = A->lev[l];
        L.id = l;
        L.n0 = q[l][0];
        L.n1 = q[l][1];
        L.n2 = q[l][2];
        const long long cells = (long long)L.n0 * L.n1 * L.n2;
        const bool tail = l == nlev - 1;
        if (L.n0 < 2 || L.n1 < 2 || L.n2 < 2 || cells > 65536 || (tail && cells > kVisitCoarsest))
            return false;
        if (!box && ((L.n0 | L.n1 | L.n2) & 1))
            return false;
        L.single = tail || L.n0 <= 8 || cells <= 512;
        if (l > 0 && A->lev[l - 1].single)
            L.single = 1;
        L.P = L.single ? L.n0 : (L.n0 + kVisitCtas - 1) / kVisitCtas;
        L.act = L.single ? 1 : (L.n0 + L.P - 1) / L.P;
        L.wq = box ? (L.n2 + 3) / 2 : L.n2 / 2;
        L.sz = (box || !L.single ? L.P + 2 : L.P) * (box ? L.n1 + 2 : L.n1) * L.wq;
        L.pieces = quads;
        quads += 3 * L.sz;
        L.F = quads;
        quads += (L.P * L.n1 * L.n2 + 1) / 2;
        L.ring = 2 * (L.n2 + 2) + 2 * L.n1;
        L.mring = magic(L.ring);
        L.mq = magic((L.n2 + 1) / 2);
        L.m1 = magic(L.n1);
        L.m2 = magic(L.n2);
        L.inv_h = (float)(1.0 / (double)cells);
        L.inv_l = (float)(1.0 / (double)cells - (double)L.inv_h);
        int m = L.n0 > L.n1 ? L.n0 : L.n1;
        m = m > L.n2 ? m : L.n2;
        L.nmax2 = 0;
        while (m > 1) {
            m >>= 1;
            L.nmax2 += 2;
        }
    }
    A->nlev = nlev;
    A->smem = quads * 16;
    return A->smem <= kVisitSmem;
}

void visit_level_consts(VisitLevel *L, const CoefT<double> &cf, double w)
{
    const split::Coef cs = split::make_split_coef(cf);
    int ex = 0;
    const double H = 2.0 * std::frexp(cf.h2, &ex);
    L->h2 = cf.h2;
    L->k = cf.k23 * cf.inv_h2;
    L->Hq = ex - 1;
    L->Hh = (float)H;
    L->Hl = (float)(H - (double)L->Hh);
    L->wh = cs.wh;
    L->wl = cs.wl;
    double p = 1.0;
    for (int m = 0; m < 3; ++m) {
        p *= w;
        L->w[m][0] = (float)p;
        L->w[m][1] = (float)(p - (double)L->w[m][0]);
    }
}

cudaError_t prepare_visit_kernels(bool *fits)
{
    cudaError_t e = cudaSuccess;
    *fits = true;
    for (const void *k : {(const void *)k_visit<false>, (const void *)k_visit<true>}) {
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kVisitSmem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        cudaLaunchAttribute at;
        cudaLaunchConfig_t cfg = cluster_config(kVisitSmem, nullptr, &at);
        int n = 0;
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveClusters(&n, k, &cfg);
        *fits = *fits && n > 0;
    }
    return e;
}

cudaError_t launch_visit(const VisitArgs &A, bool box, cudaStream_t st)
{
    cudaLaunchAttribute at;
    const cudaLaunchConfig_t cfg = cluster_config(A.smem, st, &at);
    const cudaError_t e = box ? cudaLaunchKernelEx(&cfg, k_visit<true>, A) : cudaLaunchKernelEx(&cfg, k_visit<false>, A);
    count_launch(1);
    return e;
}

}  // namespace mg5
