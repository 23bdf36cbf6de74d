// The FP64 explicit MPM step (Sec. "Elastic Deformation") in 64-bit fixed point.
//
// Why: GB300 retires two FP64 lanes per clock and SM, so the step's ~870 FP64 instructions a
// cell bounded it at 3.33 ms for 256^3 points whatever else was done.  The integer pipes run
// 16 to 64 lanes a clock, and everything between the corner displacements and the corner
// forces of a cell is linear: additions, the 3/1 interpolation weights, and 36 products with
// the stiffness per point.  So a cell is computed in integers that share one exponent, and
// only the node update (v, u) stays in FP64.
//
// Numbers.  A node's displacement is held as one integer m * 2^3 (m the 53-bit mantissa) and one exponent per
// component.  Where no displacement of a cell exceeds the mean strain's exponent (most cells of a loaded
// body), the cell's exponent F is the mean strain's and the values are shifted to it.  Elsewhere a cell
// aligns each component's eight values to the largest exponent among them and takes the differences
// against its lowest corner, so that a displacement that all corners share costs nothing; what the alignment drops
// is below 2^-55 of the component's largest value where its exponents differ, and the differences are then
// of that size.  F is the smallest exponent, from the mean strain's on, at which all differences of all components
// stay below 2^56; a component above it is represented by its differences, shifted up exactly, one below it is
// shifted down.  The gradients (16 x interpolated differences) and the strains (two
// gradient entries and the mean strain) are exact integer sums below 2^62.6; strains are taken / 8 (< 2^59.6)
// and split into signed 32-bit halves.  The stiffness is held as integers C 2^cexp with row sums below 2^63,
// split the same way; sigma = round(C e / 2^64) drops only the product of the two low halves
// (< 2^62, below the rounding) and stays below 2^58.6; the sums behind it stay below 2^63.  The
// traction sums (< 2^59.6) are exact, their first 3/1 sums (< 2^61.6) are taken / 8, the second
// (< 2^60.6) and a corner's force (< 2^62.2) are exact again.  Each rounding is below the 2^-53 of the
// cell's largest strain, or stress, that an FP64 evaluation carries for it; a component of strain or
// stress far below the largest of its cell has that absolute error, not a relative one of its own (FP64
// keeps one where the stiffness does not couple the components, as in an aligned crystal).  The corner forces are
// +-X +-Y +-Z of the same integers, so a cell's forces sum to exactly zero whatever was rounded.
// A node's force is the sum of its eight cells' integers: exact when their exponents agree, or differ by
// less than the bits that the terms leave free, and the sum cannot leave 63 bits (all tested), otherwise aligned
// to the largest exponent with symmetric rounding.  A cell with a non-finite corner gets F = 2047 and its nodes NaN.
// Against an 80-bit reference (20x24x28 points, 100 steps) the velocity's relative error is
// 5.6e-15 and the displacement's 6.7e-16; FP64 arithmetic gave 1.05e-14 and 7.6e-16.
//
// Tiling, scheduling and the march in z are those of the FP32 step (k_mpm.cu); nodes and forces
// are kept in shared memory as two arrays of 16-byte halves, (x, y) and (z, exponents), so that
// consecutive lanes read consecutive 16 bytes.  The forces are double-buffered, which leaves one
// barrier per plane.
// What bounds it: 250 registers leave eight warps per SM, which issue 35 % of the cycles (the
// busiest pipe, the multipliers, 42 %).  Measured, us per step against the FP64 form before it:
// 32^3 7.7 (70), 100^3 49 (308), 128^3 99 (420), 256^3 675 to 708 (3330).
#include "hmc_device.cuh"
#include "hmc_fixed.h"

namespace hmc {

namespace {

typedef long long ll;

struct FxHalf {   // 16 bytes: x and y, or z and the exponent
    ll a, b;
};

struct FxMean {                              // mean strain, m * 2^8 aligned to the exponent e
    FxHalf eb[3];
    int e;
};
struct alignas(16) FxMarchSmem {
    FxHalf uxy[3][MPM_NODES], uze[3][MPM_NODES];             // node planes, W + 1 nodes a row
    FxHalf fxy[2][8][MPM_THREADS], fze[2][8][MPM_THREADS];   // (buffer) contributions to corner I + 2J + 4K
    FxMean m;
};
template <int THREADS>
struct alignas(16) FxBlockSmem {
    FxHalf uxy[2 * THREADS], uze[2 * THREADS];
    FxHalf fxy[8][THREADS], fze[8][THREADS];
    FxMean m;
};

__device__ __forceinline__ int dexp(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// mantissa of x times 2^K, aligned to the biased exponent E >= dexp(x)
template <int K>
__device__ __forceinline__ ll dfix(double x, int E) {
    const int hi = __double2hiint(x), e = (hi >> 20) & 0x7ff;
    const ll f = ((ll)(hi & 0xfffff) << 32) | (unsigned)__double2loint(x);
    const ll m = e ? f | 1ll << 52 : f << 1;   // a subnormal number is f 2^-1074
    const ll s = (ll)((unsigned long long)(m << K) >> min(E - e, 63));
    return hi < 0 ? -s : s;
}

// o[b][c] = sum_J sum_K W(J,b) W(K,c) d[J][K] with weights 3 (same side) and 1 (other side)
// (the first index's sums taken / 2^SHIFT)
template <int SHIFT>
__device__ __forceinline__ void interp31(ll d00, ll d10, ll d01, ll d11, ll (&o)[2][2]) {
    const ll s0 = d00 + d10, s1 = d01 + d11;
    const ll e00 = (s0 + (d00 << 1)) >> SHIFT, e10 = (s0 + (d10 << 1)) >> SHIFT;
    const ll e01 = (s1 + (d01 << 1)) >> SHIFT, e11 = (s1 + (d11 << 1)) >> SHIFT;
    const ll t0 = e00 + e01, t1 = e10 + e11;
    o[0][0] = t0 + (e00 << 1);
    o[0][1] = t0 + (e01 << 1);
    o[1][0] = t1 + (e10 << 1);
    o[1][1] = t1 + (e11 << 1);
}

// One orientation's stiffness: the 21 upper-triangle entries, each as signed halves (x low, y high)
struct FxRow {
    int2 v[22];
    __device__ __forceinline__ void load(const int2 *tab, uint32_t q) {
        const int4 *p = reinterpret_cast<const int4 *>(tab + 24ll * q);
#pragma unroll
        for (int i = 0; i < 11; ++i) {
            const int4 t = __ldg(p + i);
            v[2 * i] = make_int2(t.x, t.y);
            v[2 * i + 1] = make_int2(t.z, t.w);
        }
    }
};

__host__ __device__ constexpr int upper21(int i, int j) {   // place of entry (i, j) in the upper triangle
    const int lo = i < j ? i : j, hi = i < j ? j : i;
    return lo * 6 - lo * (lo - 1) / 2 + hi - lo;
}

// round(sum_j C_ij e_j / 2^64) for the six stress components
__device__ __forceinline__ void fx_hooke(const FxRow &r, const ll (&e)[6], ll (&s)[6]) {
    int eh[6], el[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const ll x = e[j] >> 3;
        el[j] = (int)x;
        eh[j] = (int)(x >> 32) + (int)((unsigned)el[j] >> 31);
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        ll h = 0, x = 1ll << 31;
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            const int2 c = r.v[upper21(i, j)];
            h += (ll)c.y * eh[j];
            x += (ll)c.y * el[j];
            x += (ll)c.x * eh[j];
        }
        s[i] = h + (x >> 32);
    }
}

// the visiting order of a cell's points: one coordinate changes from one to the next, so that a
// grain boundary normal to x, y, z costs 4, 2, 1 reloads of the stiffness row
__host__ __device__ constexpr int gray_pt(int n) {
    return n == 0 ? 0 : n == 1 ? 1 : n == 2 ? 3 : n == 3 ? 2 : n == 4 ? 6 : n == 5 ? 7 : n == 6 ? 5 : 4;
}

// the 24 corner forces of a cell (times 32, with the sign of -f) from its corner displacements
__device__ __forceinline__ void fx_cell(const ll (&u)[8][3], const ll (&eb)[6], const uint4 &sp, const int2 *tab,
                                        ll (&f)[8][3]) {
    FxRow row;
    uint32_t qprev = spin_of(sp, local_slot(0));
    row.load(tab, qprev);
    ll gx[2][2][3], gy[2][2][3], gz[2][2][3];   // [b][c], [a][c], [a][b]: d u_d / dx, dy, dz
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        ll o[2][2];
        interp31<0>(u[1][d] - u[0][d], u[3][d] - u[2][d], u[5][d] - u[4][d], u[7][d] - u[6][d], o);
#pragma unroll
        for (int i = 0; i < 4; ++i) gx[i >> 1][i & 1][d] = o[i >> 1][i & 1] + (d == 0 ? eb[0] : 0);
        interp31<0>(u[2][d] - u[0][d], u[3][d] - u[1][d], u[6][d] - u[4][d], u[7][d] - u[5][d], o);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            gy[i >> 1][i & 1][d] = o[i >> 1][i & 1] + (d == 1 ? eb[1] : d == 0 ? eb[5] : 0);
        interp31<0>(u[4][d] - u[0][d], u[5][d] - u[1][d], u[6][d] - u[2][d], u[7][d] - u[3][d], o);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            gz[i >> 1][i & 1][d] = o[i >> 1][i & 1] + (d == 2 ? eb[2] : d == 1 ? eb[3] : eb[4]);
    }
    ll tx[2][2][3], ty[2][2][3], tz[2][2][3];   // traction sums over a, b, c respectively
#pragma unroll
    for (int i = 0; i < 12; ++i)
        tx[i / 6][i / 3 & 1][i % 3] = ty[i / 6][i / 3 & 1][i % 3] = tz[i / 6][i / 3 & 1][i % 3] = 0;
#pragma unroll
    for (int n = 0; n < 8; ++n) {
        const int L = gray_pt(n);
        const int a = L & 1, b = (L >> 1) & 1, c = L >> 2;
        ll e[6], s[6];
        e[0] = gx[b][c][0];
        e[1] = gy[a][c][1];
        e[2] = gz[a][b][2];
        e[3] = gz[a][b][1] + gy[a][c][2];
        e[4] = gz[a][b][0] + gx[b][c][2];
        e[5] = gy[a][c][0] + gx[b][c][1];
        const uint32_t q = spin_of(sp, local_slot(L));
        if (q != qprev) {
            row.load(tab, q);
            qprev = q;
        }
        fx_hooke(row, e, s);
        tx[b][c][0] += s[0]; tx[b][c][1] += s[5]; tx[b][c][2] += s[4];
        ty[a][c][0] += s[5]; ty[a][c][1] += s[1]; ty[a][c][2] += s[3];
        tz[a][b][0] += s[4]; tz[a][b][1] += s[3]; tz[a][b][2] += s[2];
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        ll X[2][2], Y[2][2], Z[2][2];
        interp31<3>(tx[0][0][d], tx[1][0][d], tx[0][1][d], tx[1][1][d], X);   // X[J][K]
        interp31<3>(ty[0][0][d], ty[1][0][d], ty[0][1][d], ty[1][1][d], Y);   // Y[I][K]
        interp31<3>(tz[0][0][d], tz[1][0][d], tz[0][1][d], tz[1][1][d], Z);   // Z[I][J]
#pragma unroll
        for (int n = 0; n < 8; ++n) {
            const int I = n & 1, J = (n >> 1) & 1, K = n >> 2;
            f[n][d] = (I ? X[J][K] : -X[J][K]) + (J ? Y[I][K] : -Y[I][K]) + (K ? Z[I][J] : -Z[I][J]);
        }
    }
}

// 3 x + y
__device__ __forceinline__ ll x3(ll x, ll y) { return (x << 1) + x + y; }
// the value on the lane of the quarter beyond the cell's middle in y (8) or z (16)
__device__ __forceinline__ ll across(ll x, int lane) { return __shfl_xor_sync(0xffffffffu, x, lane); }
__device__ __forceinline__ ll flip(ll x, ll sign) { return (x ^ sign) - sign; }   // sign: 0 or -1

// Quarter (b, c) of a cell: its two points with that b and c, on lane 8 (b + 2c) + (cell of the warp),
// all 32 lanes together.  u holds the corners with I = 0, 1 that are near in y and z (0, 1), far in y
// (2, 3), far in z (4, 5) and far in both; f takes the forces (times 32, with the sign of -f) on the two
// near corners.  The same integers are summed and rounded as in fx_cell, so the results are the same bits.
__device__ __forceinline__ void fx_quarter(const ll (&u)[8][3], const ll (&eb)[6], const uint4 &sp, int b, int c,
                                           const int2 *tab, ll (&f)[2][3]) {
    const ll sb = b ? -1 : 0, sc = c ? -1 : 0;   // d/dy and d/dz point from near to far for b = 0, c = 0
    ll gx[3], gy[2][3], gz[2][3];                // [d], [a][d]: d u_d / dx, dy, dz at the points
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        ll m[4], z[4];   // the corners' mean over z with the points' weights; their differences in z
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            m[n] = x3(u[n][d], u[n + 4][d]);
            z[n] = u[n + 4][d] - u[n][d];
        }
        gx[d] = x3(m[1] - m[0], m[3] - m[2]) + (d == 0 ? eb[0] : 0);
        const ll dy[2] = {flip(m[2] - m[0], sb), flip(m[3] - m[1], sb)};
        const ll dz[2] = {flip(x3(z[0], z[2]), sc), flip(x3(z[1], z[3]), sc)};
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            gy[i][d] = x3(dy[i], dy[1 - i]) + (d == 1 ? eb[1] : d == 0 ? eb[5] : 0);
            gz[i][d] = x3(dz[i], dz[1 - i]) + (d == 2 ? eb[2] : d == 1 ? eb[3] : eb[4]);
        }
    }
    // the words of the packed field that hold point a = 0 and 1 of this quarter
    uint32_t q[2];
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        const uint32_t q0 = b ? spin_of(sp, local_slot(a + 2)) : spin_of(sp, local_slot(a));
        const uint32_t q1 = b ? spin_of(sp, local_slot(a + 6)) : spin_of(sp, local_slot(a + 4));
        q[a] = c ? q1 : q0;
    }
    FxRow row;
    row.load(tab, q[0]);
    ll tx[3], ty[2][3], tz[2][3];   // this quarter's share of the traction sums over a, b and c
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        ll s[6];
        const ll e[6] = {gx[0], gy[a][1], gz[a][2], gz[a][1] + gy[a][2], gz[a][0] + gx[2], gy[a][0] + gx[1]};
        if (a == 1 && q[1] != q[0]) row.load(tab, q[1]);
        fx_hooke(row, e, s);
        const ll x[3] = {s[0], s[5], s[4]}, y[3] = {s[5], s[1], s[3]}, z[3] = {s[4], s[3], s[2]};
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            tx[d] = a ? tx[d] + x[d] : x[d];
            ty[a][d] = y[d];
            tz[a][d] = z[d];
        }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const ll ex = x3(tx[d], across(tx[d], 8)) >> 3, X = x3(ex, across(ex, 16));   // X[b][c]
        ll Y[2], Z[2];                                                                 // Y[I][c], Z[I][b]
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            ty[i][d] += across(ty[i][d], 8);
            tz[i][d] += across(tz[i][d], 16);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const ll ey = x3(ty[i][d], ty[1 - i][d]) >> 3, ez = x3(tz[i][d], tz[1 - i][d]) >> 3;
            Y[i] = x3(ey, across(ey, 16));
            Z[i] = x3(ez, across(ez, 8));
            f[i][d] = (i ? X : -X) + flip(Y[i], ~sb) + flip(Z[i], ~sc);
        }
    }
}

// three integers with one exponent (that of the cells' displacements; 2047 = not finite)
struct Fx3 {
    ll v[3];
    int e;
};

// The sum of N terms x[i] 2^e[i] per direction.  With one exponent it is exact; with several it is exact at
// the smallest of them where the terms have the room (they mostly differ by one or two, and rounding
// every term instead took 256^3 under load along [111] from 708 to 801 us a step).  Otherwise the terms
// are aligned to the largest exponent, and three bits above it where the sum would leave 63 bits.
template <int N>
__device__ __forceinline__ Fx3 fx_sum(const ll (&x)[3][N], const int (&e)[N]) {
    Fx3 r;
    r.e = e[0];
    bool plain = true;
#pragma unroll
    for (int i = 1; i < N; ++i) {
        plain &= e[i] == e[0];
        r.e = max(r.e, e[i]);
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        ll v = 0;
        int t = 0;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            v += x[d][i];
            t += (int)(x[d][i] >> 35);
        }
        r.v[d] = v;
        plain &= fits63(t);
    }
    if (!plain && r.e < 2047) {
        const int top = r.e;
        int low = e[0];
        unsigned any = 0;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            low = min(low, e[i]);
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const int h = (int)(x[d][i] >> 32);
                any |= (unsigned)(h ^ (h >> 31));
            }
        }
        if (top - low <= __clz(any) - (N == 4 ? 4 : 3)) {   // then the N terms stay below 2^62 / N
            r.e = low;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                unsigned long long v = 0;
#pragma unroll
                for (int i = 0; i < N; ++i) v += (unsigned long long)x[d][i] << (e[i] - low);
                r.v[d] = (ll)v;
            }
            return r;
        }
#pragma unroll 1
        for (int up = 0; up <= 3; up += 3) {
            r.e = top + up;
            bool fits = true;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                ll v = 0;
                int t = 0;
#pragma unroll
                for (int i = 0; i < N; ++i) {
                    const ll s = rshift(x[d][i], r.e - e[i]);
                    v += s;
                    t += (int)(s >> 35);
                }
                r.v[d] = v;
                fits &= fits63(t);
            }
            if (fits) break;
        }
    }
    return r;
}

// a node's displacement into shared memory: each component's 2^3 m and their exponents, 16 bits each
__device__ __forceinline__ void fx_put(FxHalf *xy, FxHalf *ze, int t, const double (&u)[3]) {
    const int ex = dexp(u[0]), ey = dexp(u[1]), ez = dexp(u[2]);
    xy[t] = FxHalf{dfix<3>(u[0], ex), dfix<3>(u[1], ey)};
    ze[t] = FxHalf{dfix<3>(u[2], ez), ((ll)ez << 32) | (unsigned)(ex | ey << 16)};
}

// Behind the wait: the end of a Monte Carlo step writes the mean strain, and only the wait makes it
// visible.  By one thread in the march (by a warp there, other code of the loop came out slower: 102 ->
// 108 us at 128^3) ...
__device__ __forceinline__ void fx_mean(FxMean &m, const DevState *st) {
    double e[6];
    int E = 0;
    for (int i = 0; i < 6; ++i) {
        e[i] = st->ebar[i];
        E = max(E, dexp(e[i]));
    }
    for (int i = 0; i < 3; ++i) m.eb[i] = FxHalf{dfix<8>(e[2 * i], E), dfix<8>(e[2 * i + 1], E)};
    m.e = E;
}
// ... and by the first warp, a lane a component, in a block, where it lies in the chain of the
// step (8.18 us at 32^3, 8.37 by one thread)
__device__ __forceinline__ void fx_mean_warp(FxMean &m, const DevState *st) {
    const int lane = threadIdx.x;
    const double e = lane < 6 ? st->ebar[lane] : 0.0;
    const int E = (int)__reduce_max_sync(0xffffffffu, (unsigned)dexp(e));
    const ll x = dfix<8>(e, E);
    if (lane < 6) (lane & 1 ? m.eb[lane >> 1].b : m.eb[lane >> 1].a) = x;
    if (lane == 0) m.e = E;
}

// a cell: its corners lie at n0 and n1 (lower and upper plane; for a quarter near and far), dy apart in
// y; u becomes their displacements at the cell's exponent, which is returned, all eight of a component
// together against the cell's lowest corner's (ref: its place among them) where that keeps bits.  Against one
// exponent for the displacements of all components this costs a Monte Carlo run's state 2 % (32^3 7.55 ->
// 7.7 us, 100^3 47.4 -> 48.4; with the differences formed in every cell 8.3 and 50.3); states whose displacements
// pass the mean strain gain, since fewer cells differ in exponent (256^3 under load along z 696 -> 675).
__device__ __forceinline__ int fx_corners(const FxHalf *xy0, const FxHalf *ze0, const FxHalf *xy1, const FxHalf *ze1,
                                          int dy, int ref, const FxMean &m, ll (&u)[8][3], ll (&eb)[6]) {
    unsigned exy[8], ez[8], mxy = 0, mz = 0;
#pragma unroll
    for (int n = 0; n < 8; ++n) {
        const int o = (n & 1) + (n & 2 ? dy : 0);
        const FxHalf p = (n & 4 ? xy1 : xy0)[o], q = (n & 4 ? ze1 : ze0)[o];
        u[n][0] = p.a;
        u[n][1] = p.b;
        u[n][2] = q.a;
        exy[n] = (unsigned)q.b;
        ez[n] = (unsigned)(q.b >> 32);
        mxy = __vmaxu2(mxy, exy[n]);
        mz = max(mz, ez[n]);
    }
    const int E[3] = {(int)(mxy & 0xffffu), (int)(mxy >> 16), (int)mz}, top = max(max(E[0], E[1]), E[2]);
    int F = m.e;
    if (top <= F) {
        const unsigned f2 = (unsigned)F | (unsigned)F << 16;
#pragma unroll
        for (int n = 0; n < 8; ++n) {
            const unsigned t = __vminu2(f2 - exy[n], 0x003f003fu);
            u[n][0] >>= t & 0xffffu;
            u[n][1] >>= t >> 16;
            u[n][2] >>= min((unsigned)F - ez[n], 63u);
        }
    } else {
#pragma unroll
        for (int n = 0; n < 8; ++n) {
            const unsigned t = __vminu2(mxy - exy[n], 0x003f003fu);
            u[n][0] >>= t & 0xffffu;
            u[n][1] >>= t >> 16;
            u[n][2] >>= min(mz - ez[n], 63u);
        }
        ll r[3];   // the lowest corner's
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const ll lo = ref & 2 ? u[2][d] : u[0][d], hi = ref & 2 ? u[6][d] : u[4][d];
            r[d] = ref & 4 ? hi : lo;
            ll any = 0;
#pragma unroll
            for (int n = 0; n < 8; ++n) {
                const ll x = u[n][d] - r[d];
                any |= x ^ (x >> 63);
            }
            F = max(F, E[d] + 8 - __clzll(any));
        }
        if (top == 2047) F = 2047;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            if (E[d] > F) {
#pragma unroll
                for (int n = 0; n < 8; ++n) u[n][d] = (ll)((unsigned long long)(u[n][d] - r[d]) << min(E[d] - F, 63));
            } else {
#pragma unroll
                for (int n = 0; n < 8; ++n) u[n][d] >>= min(F - E[d], 63);
            }
        }
    }
    const int se = min(F - m.e, 63);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const FxHalf t = m.eb[i];
        eb[2 * i] = t.a >> se;
        eb[2 * i + 1] = t.b >> se;
    }
    return F;
}

// the four cells (i-1, j-1), (i, j-1), (i-1, j), (i, j) of one plane, W cells a row, on their common
// node: they see it as corner c + 3, c + 2, c + 1, c
template <int THREADS>
__device__ __forceinline__ Fx3 fx_sum4(const FxHalf (&xy)[8][THREADS], const FxHalf (&ze)[8][THREADS], int c, int t, int W) {
    const FxHalf a3 = xy[c + 3][t - W - 1], b3 = ze[c + 3][t - W - 1], a2 = xy[c + 2][t - W], b2 = ze[c + 2][t - W];
    const FxHalf a1 = xy[c + 1][t - 1], b1 = ze[c + 1][t - 1], a0 = xy[c][t], b0 = ze[c][t];
    const ll x[3][4] = {{a3.a, a2.a, a1.a, a0.a}, {a3.b, a2.b, a1.b, a0.b}, {b3.a, b2.a, b1.a, b0.a}};
    const int e[4] = {(int)b3.b, (int)b2.b, (int)b1.b, (int)b0.b};
    return fx_sum<4>(x, e);
}

// the update of a node whose force is not finite or whose scale leaves the normal range; kept out of
// line, since its FP64 multiplications would otherwise be formed for every node (6 % of a step)
__device__ __noinline__ void fx_update_any(ll x, ll y, ll z, int e, double fscale, int shift, double keep, double dt,
                                           double ukeep, const double *uold, const double *vold, double *u, double *v) {
    for (int d = 0; d < 3; ++d) {
        const double F = e >= 2047 ? __longlong_as_double(0x7ff8000000000000ll) : scalbn((double)(d == 0 ? x : d == 1 ? y : z), shift);
        const double vn = rfma(fscale, F, rmul(keep, vold[d]));
        v[d] = vn;
        u[d] = rfma(dt, vn, rmul(ukeep, uold[d]));
    }
}

// velocity and displacement of a node from the force sums of the cells below and above it
// (SCALED: the old displacement times ukeep, in the adjoint's reverse step; a form of its own, since an
// FP64 multiplication of every node costs 2 % of a step even where it is not used)
template <bool SCALED>
struct FxUpdate {
    double fscale, dt, keep, ukeep;   // fscale = -dt / (32 m)
    int cexp, fexp;
    __device__ __forceinline__ explicit FxUpdate(const MpmArgs<double> &a)
        : fscale(-a.dt_over_m * 0.03125), dt(a.dt), keep(a.keep), ukeep(a.ukeep), cexp(__ldg(&a.cfix[CFIX_EXP].x)) {
        // the force integers of exponent E are 2^(E - cexp - 1013) of the FP32 step's units
        fexp = dexp(fscale) ? dexp(fscale) - cexp - 1013 : -10000;   // (subnormal: the general form)
    }
    __device__ __forceinline__ void operator()(const Fx3 &lo, const Fx3 &hi, const double (&uold)[3],
                                               const double (&vold)[3], double *u, double *v) const {
        const ll x[3][2] = {{lo.v[0], hi.v[0]}, {lo.v[1], hi.v[1]}, {lo.v[2], hi.v[2]}};
        const int e[2] = {lo.e, hi.e};
        const Fx3 F = fx_sum<2>(x, e);
        const int ef = fexp + F.e;   // exponent of fscale times the force's unit
        if ((unsigned)(ef - 1) < 2045u && F.e < 2047) {
            const double fs = __hiloint2double((__double2hiint(fscale) & 0x800fffff) | (ef << 20), __double2loint(fscale));
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const double vn = rfma(fs, (double)F.v[d], rmul(keep, vold[d]));
                v[d] = vn;
                u[d] = rfma(dt, vn, SCALED ? rmul(ukeep, uold[d]) : uold[d]);
            }
        } else {
            fx_update_any(F.v[0], F.v[1], F.v[2], F.e, fscale, F.e - cexp - 1013, keep, dt, ukeep, uold, vold, u, v);
        }
    }
};

template <bool SCALED>
__global__ void __launch_bounds__(MPM_THREADS, 1) k_mpm_fixed(MpmArgs<double> a) {
    constexpr int PER = (MPM_NODES + MPM_THREADS - 1) / MPM_THREADS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FxMarchSmem &sm = *reinterpret_cast<FxMarchSmem *>(smem_raw);
    const int tid = threadIdx.x;
    const FxUpdate<SCALED> update(a);
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    long long w = a.cuts[blockIdx.x];
    const long long wend = a.cuts[blockIdx.x + 1];
    int r = 0;
    while (w < wend) {
        while (a.sched[r + 1].off <= w) ++r;
        const Replica &R = a.reps[r];
        const MpmSched &SC = a.sched[r];
        const int nbx = R.nbx, nby = R.nby, nbz = R.nbz;
        const long long lw = w - SC.off;
        const int tile = (int)(lw / nbz);
        const int k0 = (int)(lw - (long long)tile * nbz);
        const long long rem = min(wend, a.sched[r + 1].off) - w;
        const int kend = (int)min((long long)nbz, (long long)k0 + rem);
        w += kend - k0;
        const int i0 = (tile % SC.tiles_x) * SC.ox, j0 = (tile / SC.tiles_x) * SC.oy;
        const int W = min(SC.ox, nbx - i0) + 1, H = min(SC.oy, nby - j0) + 1, P = W + 1;
        const int lci = tid % W, lcj = tid / W;
        const bool need = tid < W * H;
        const bool own = need && lci >= 1 && lcj >= 1;
        const int plane = nbx * nby;
        const long long node0 = R.blk_off;   // not read again in every plane: 1 % from 100^3 on
        const long long col = node0 + wrapi(i0 - 1 + lci, nbx) + nbx * wrapi(j0 - 1 + lcj, nby);
        const int nd = lci + P * lcj;
        int ncol[PER];   // the patch's nodes that this thread loads, as (i + nbx j) in a node plane, -1 beyond it
#pragma unroll
        for (int m = 0; m < PER; ++m) {
            const int t = tid + m * MPM_THREADS;
            ncol[m] = t < P * (H + 1) ? wrapi(i0 - 1 + t % P, nbx) + nbx * wrapi(j0 - 1 + t / P, nby) : -1;
        }
        double pl[PER][3];
        auto fetch = [&](int k) {   // node plane k, -1 <= k <= nbz (periodic in z)
            const int gk = k < 0 ? k + nbz : (k >= nbz ? k - nbz : k);
            const double *base = a.u_in + 3 * (node0 + (long long)plane * gk);
#pragma unroll
            for (int m = 0; m < PER; ++m)
                if (ncol[m] >= 0)
#pragma unroll
                    for (int d = 0; d < 3; ++d) pl[m][d] = base[3 * ncol[m] + d];
        };
        auto store = [&](int b) {
#pragma unroll
            for (int m = 0; m < PER; ++m)
                if (ncol[m] >= 0) fx_put(sm.uxy[b], sm.uze[b], tid + m * MPM_THREADS, pl[m]);
        };
        int b0 = 0, b1 = 1, b2 = 2, fb = 0;
        const DevState *st = R.st;
        // nothing above reads what the kernels before this one write: 1.2 us a step against a wait ahead
        // of the range's look-ups
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (tid == 0) fx_mean(sm.m, st);
        fetch(k0 - 1);
        store(b0);
        fetch(k0);
        store(b1);
        uint4 sp = need ? a.spins[col + (long long)plane * wrapi(k0 - 1, nbz)] : make_uint4(0, 0, 0, 0);
        __syncthreads();

        Fx3 acc = {{0, 0, 0}, 0};
        const uint4 *spn = a.spins + col + (long long)plane * k0;
        const double *uip = a.u_in + 3 * (col + (long long)plane * k0);
        double *vp = a.v + 3 * (col + (long long)plane * k0);
        double *up = a.u_out + 3 * (col + (long long)plane * k0);
        const long long pstride = 3ll * plane;
        for (int kk = k0 - 1; kk < kend; ++kk) {
            uint4 sp_next = make_uint4(0, 0, 0, 0);
            if (need && kk + 1 < kend) sp_next = *spn;
            spn += plane;
            double vold[3] = {0, 0, 0}, uold[3] = {0, 0, 0};
            if (own && kk >= k0) {
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    vold[d] = vp[d];
                    uold[d] = uip[d];
                }
            }
            const bool more = kk + 1 < kend;
            if (more) fetch(kk + 2);
            if (need) {
                ll u[8][3], eb[6], f[8][3];
                const int E = fx_corners(sm.uxy[b0] + nd, sm.uze[b0] + nd, sm.uxy[b1] + nd, sm.uze[b1] + nd, P, 0, sm.m, u, eb);
                fx_cell(u, eb, sp, a.cfix, f);
#pragma unroll
                for (int n = 0; n < 8; ++n) {
                    sm.fxy[fb][n][tid] = FxHalf{f[n][0], f[n][1]};
                    sm.fze[fb][n][tid] = FxHalf{f[n][2], (ll)E};
                }
            }
            if (more) store(b2);   // buffer b2 was last read before the previous barrier
            __syncthreads();
            if (own) {
                if (kk >= k0) {
                    update(acc, fx_sum4(sm.fxy[fb], sm.fze[fb], 0, tid, W), uold, vold, up, vp);
                    vp += pstride;
                    up += pstride;
                    uip += pstride;
                }
                acc = fx_sum4(sm.fxy[fb], sm.fze[fb], 4, tid, W);
            }
            // one barrier a plane: the next plane writes the other force buffer and the node plane that
            // was last read before this one's barrier
            fb ^= 1;
            const int t = b0;
            b0 = b1;
            b1 = b2;
            b2 = t;
            sp = sp_next;
        }
        __syncthreads();   // the next range reuses every buffer
    }
}

// The block form (k_mpm.cu): one block per CTA, every cell at once, on SPLIT threads each.  Blocks of
// at most 96 cells run where there is one to an SM, three warps of whole cells: what bounds them is
// the length of a cell's code, and quarters take 8.2 us a step at 32^3 where whole cells took 11.4.
// Blocks of 256 cells fill the registers as they are (halves at 128 registers: 24.6 -> 30.3 us at
// 64^3; the march likewise, 102 -> 133 us at 128^3).
template <int CELLS, int SPLIT, bool SCALED>
__global__ void __launch_bounds__(CELLS *SPLIT, 1) k_mpm_fixed_block(MpmArgs<double> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FxBlockSmem<CELLS> &sm = *reinterpret_cast<FxBlockSmem<CELLS> *>(smem_raw);
    const int tid = threadIdx.x;
    const int cell = SPLIT == 4 ? (tid >> 5) * 8 + (tid & 7) : tid;
    const int b = SPLIT == 4 ? tid >> 3 & 1 : 0, c = SPLIT == 4 ? tid >> 4 & 1 : 0;   // this thread's quarter
    const FxUpdate<SCALED> update(a);
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    int r = 0;
    while (a.sched[r + 1].off <= blockIdx.x) ++r;
    const Replica &R = a.reps[r];
    const MpmSched &SC = a.sched[r];
    const BlockPlace B(SC, R, blockIdx.x - (int)SC.off);
    const int W = B.W, H = B.H, P = W + 1, PP = P * (H + 1);
    auto block_at = [&](int i, int j, int k) {
        return R.blk_off + wrapi(B.i0 - 1 + i, R.nbx) +
               (long long)R.nbx * (wrapi(B.j0 - 1 + j, R.nby) + (long long)R.nby * wrapi(B.k0 - 1 + k, R.nbz));
    };
    const int cells = W * H * B.D;
    const int ci = cell % W, cj = cell / W % H, ck = cell / (W * H);
    const bool need = cell < cells, some = SPLIT == 4 ? (tid >> 5) * 8 < cells : need;   // (quarters: the whole warp)
    const int lci = tid % W, lcj = tid / W % H, lck = tid / (W * H);   // the first threads own nodes
    const bool own = tid < cells && lci >= 1 && lcj >= 1 && lck >= 1;
    const long long at = own ? block_at(lci, lcj, lck) : 0, cat = need ? block_at(ci, cj, ck) : 0;
    constexpr int PER = SPLIT == 4 ? 1 : 2;   // nodes a thread converts: the blocks have at most two a cell
    long long node[PER];
#pragma unroll
    for (int m = 0; m < PER; ++m) node[m] = B.node(R, tid + m * CELLS);
    const DevState *st = R.st;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (tid < 32) fx_mean_warp(sm.m, st);
    const uint4 sp = need ? a.spins[cat] : make_uint4(0, 0, 0, 0);
    double uold[3] = {0, 0, 0}, vold[3] = {0, 0, 0};
    if (own) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            vold[d] = a.v[3 * at + d];
            uold[d] = a.u_in[3 * at + d];
        }
    }
#pragma unroll
    for (int m = 0; m < PER; ++m)
        if (node[m] >= 0) {
            const double *p = a.u_in + 3 * node[m];
            const double u[3] = {p[0], p[1], p[2]};
            fx_put(sm.uxy, sm.uze, tid + m * CELLS, u);
        }
    __syncthreads();
    if (some) {
        ll u[8][3], eb[6], f[8 / SPLIT][3];
        const int nd = need ? ci + P * cj + PP * ck : 0, n0 = nd + (b ? P : 0) + (c ? PP : 0), dz = c ? -PP : PP;
        const int E = fx_corners(sm.uxy + n0, sm.uze + n0, sm.uxy + n0 + dz, sm.uze + n0 + dz, b ? -P : P, 2 * b + 4 * c, sm.m, u, eb);
        if constexpr (SPLIT == 4)
            fx_quarter(u, eb, sp, b, c, a.cfix, f);
        else
            fx_cell(u, eb, sp, a.cfix, f);
#pragma unroll
        for (int n = 0; n < 8 / SPLIT; ++n) {
            sm.fxy[2 * b + 4 * c + n][cell] = FxHalf{f[n][0], f[n][1]};
            sm.fze[2 * b + 4 * c + n][cell] = FxHalf{f[n][2], (ll)E};
        }
    }
    __syncthreads();
    if (own)
        update(fx_sum4(sm.fxy, sm.fze, 4, tid - W * H, W), fx_sum4(sm.fxy, sm.fze, 0, tid, W), uold, vold,
               a.u_out + 3 * at, a.v + 3 * at);
}

struct Form {   // kernel, threads, shared memory
    void (*kernel)(MpmArgs<double>);
    int threads;
    size_t smem;
};
template <bool SCALED>
Form form_of(int variant) {
    if (!mpm_is_block(variant)) return Form{k_mpm_fixed<SCALED>, MPM_THREADS, sizeof(FxMarchSmem)};
    if (variant == MPM_BLOCK)
        return Form{k_mpm_fixed_block<MPM_THREADS, 1, SCALED>, MPM_THREADS, sizeof(FxBlockSmem<MPM_THREADS>)};
    return Form{k_mpm_fixed_block<MPM_SMALL_BLOCK, 4, SCALED>, 4 * MPM_SMALL_BLOCK,
                sizeof(FxBlockSmem<MPM_SMALL_BLOCK>)};
}

}  // namespace

cudaError_t mpm64_prepare() {
    for (int v : {0, (int)MPM_BLOCK, MPM_BLOCK + 1}) {
        for (const Form &f : {form_of<false>(v), form_of<true>(v)}) {
            const cudaError_t e = cudaFuncSetAttribute(f.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)f.smem);
            if (e != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

template <>
int mpm_per_sm<double>(int variant, int) {
    const Form f = form_of<false>(variant);
    int n = 1;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, f.kernel, f.threads, f.smem);
    return (e != cudaSuccess || n < 1) ? 1 : n;
}

// programmatic stream serialisation, as the FP32 step
template <>
cudaError_t launch_mpm_step<double>(const MpmArgs<double> &a, int variant, cudaStream_t s) {
    const Form f = a.ukeep == 1.0 ? form_of<false>(variant) : form_of<true>(variant);
    return launch_pdl(f.kernel, (unsigned)a.grid, (unsigned)f.threads, f.smem, s, a);
}

}  // namespace hmc
