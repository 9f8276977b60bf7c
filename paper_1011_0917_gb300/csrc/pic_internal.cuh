// pic_internal.cuh -- device-side data layout and helpers of the PIC library.
//
// Layout in HBM (all caller-owned):
//   fields:  9 components (Ex Ey Ez Bx By Bz Jx Jy Jz), each (nz+1) x ny x nx
//            elements in [k][j][i] order.  Yee staggering of component c at
//            array index (i, j, k): Ex (i+1/2, j, k), Ey (i, j+1/2, k),
//            Ez (i, j, k+1/2), Bx (i, j+1/2, k+1/2), By (i+1/2, j, k+1/2),
//            Bz (i+1/2, j+1/2, k); J like E.
//   species: per species two "sides" (double buffer).  A side holds `slots`
//            records in blocks of 32: a block is 32 values of the first
//            attribute, 32 of the next, ... (Rec), so that the 32 records a
//            warp works on are one contiguous piece (1 KB for an FP32
//            electron in 3D) reached with one address.  Tile t owns slots
//            [t*cap, (t+1)*cap) and keeps its particles in two runs: a bottom
//            run [0, lo) that the tile's own CTA writes (particles that stayed
//            in the tile, counted in shared memory) and a top run
//            [cap - hi, cap) that others append to with global atomics
//            (particles that arrived from a neighbour, were loaded or were
//            injected).  A particle is an int32 packed cell index plus its
//            offsets in [0,1) inside that cell (real), its weight and
//            (electrons) u = gamma v; with drift-relative z (below) an
//            electron also carries its departure from the drift.
//   scratch: per-side tile counters, the filter ping-pong buffer, per-tile
//            offsets for compaction, reduction partials and the error word.
#pragma once

#include <cstdint>
#include <cstring>
#include <cuda_runtime.h>
#include <type_traits>
#include <vector>

namespace pic {

enum : unsigned { ERR_CAPACITY = 1u, ERR_CFL = 2u, ERR_NAN = 4u, ERR_TILE = 8u };

// Bit 31 of an electron's cell word: the electron is paired with a drifting ion
// at its own position that has moved exactly like it since both were placed
// (the plasma no field has touched).  Such a pair carries no current and is
// stored as the electron record alone; its ion gets a record of its own (at the
// electron's position) the first time the electron gathers a non-zero field.
constexpr uint32_t kPaired = 0x80000000u;

struct Geom {
    int dim;            // 2 or 3
    int nx, ny, nz;     // cells (ny = 1 in 2D)
    int bc_z;           // 0 periodic, 1 Mur
    int shape;          // 1 or 2
    int bx, by;         // bits of i and j in a packed cell index
    int lt[3];          // log2 of the tile shape
    int nt[3];          // tiles per axis
    int cap;            // slots per tile
    int early;          // its kernels let the next one on the stream in early (see launch_chained)
    int64_t plane;      // nx * ny
    int64_t ncomp;      // (nz + 1) * plane, elements per field component
    int64_t ntiles;
};

// attribute arrays of a species side, in this order: ox oy oz w ux uy uz cell
// id dlx dly dlz (absent ones are null)
constexpr int kAttrs = 12;

// Record d of an attribute is at pointer[r(d)] (the cell word at cell[c(d)]):
// in a side of the store the pointers are the attribute's row of block 0 and
// sr, sc the elements from one block to the next; in a flat list (staging of
// uploads and downloads, one array per attribute) sr = sc = 32, so r(d) =
// c(d) = d.  Ids are a plain array in both.
template <typename real>
struct Species {
    real *ox, *oy, *oz, *w;     // oy is null in 2D
    real *ux, *uy, *uz;         // null for ions (constant drift)
    int32_t *cell;
    int64_t *id;                // null unless ids are tracked
    real *dlx, *dly, *dlz;      // relative positions only (see rel_actual); dly null in 2D
    int sr, sc;
    __host__ __device__ __forceinline__ int64_t r(int64_t d) const { return (d >> 5) * sr + (d & 31); }
    __host__ __device__ __forceinline__ int64_t c(int64_t d) const { return (d >> 5) * sc + (d & 31); }
};

// Byte offsets of the attribute rows in a block of 32 records and the block's
// size RB: reals ox oy oz w, for electrons ux uy uz, in relative form dlx dly
// dlz (oy, dly in 3D only), then the cell words.
template <typename real, int DIM, bool ELECTRON, bool REL>
struct Rec {
    static constexpr int NR = DIM + 1 + (ELECTRON ? 3 : 0) + (ELECTRON && REL ? DIM : 0);
    static constexpr int ROW = 32 * (int)sizeof(real);
    static constexpr int OX = 0, OY = ROW, OZ = (DIM - 1) * ROW, W = DIM * ROW;
    static constexpr int UX = (DIM + 1) * ROW, UY = UX + ROW, UZ = UX + 2 * ROW;
    static constexpr int DLX = (DIM + 4) * ROW, DLY = DLX + ROW, DLZ = DLX + (DIM - 1) * ROW;
    static constexpr int CELL = NR * ROW, RB = CELL + 128;
};

// Relative positions of an electron record.  In a strongly boosted frame the
// plasma (electrons and ions, gamma n each) streams through a good part of a
// cell every step, while the wake is made of the difference between the two
// species' currents: ~1/(2 gamma^2) of the plasma's response in the lab, so
// at gamma = 130 about 3e-8 of either species' current.  Each particle's
// current must then be formed from a position exact far beyond FP32, and in
// arithmetic far finer than FP32 (pairs of FP32 words in the FP32 build, see
// ff; FP64 in the FP64 build), or the difference is rounding noise.  A record
// in relative form holds, per axis, a reference offset o in [0, 1) -- along z
// it moves with exactly the arithmetic of a drifting ion, across it stays
// where the particle was placed, i.e. it is its ion's path -- plus the
// departure dl from it, |dl| <= 1/2 (whole cells move between dl and the
// reference cell, which is exact).  The position is c_ref + o + dl with c_ref =
// c + r, c the stored cell (the one the electron is in, so that tiles and
// stencils are as for any record) and r the shift this function returns; its
// result is the electron's offset in cell c, in [0, 1), for the gather.  The
// rounding of o + dl here does not accumulate: it is redone from the exact
// pair every step, and the current is deposited from the pair itself.
template <typename real>
__host__ __device__ inline real rel_actual(real o, real dl, int &r)
{
    const real a = o + dl;
    if (a < real(0)) {
        const real t = a + real(1);
        if (t < real(1)) {
            r = 1;
            return t;
        }
        r = 0;  // within rounding of the cell's lower face
        return real(0);
    }
    if (a >= real(1)) {
        r = -1;
        return a - real(1);
    }
    r = 0;
    return a;
}

__host__ __device__ inline int32_t pack_cell(const Geom &g, int i, int j, int k)
{
    return (int32_t)((uint32_t)i | ((uint32_t)j << g.bx) | ((uint32_t)k << (g.bx + g.by)));
}

__host__ __device__ inline void unpack_cell(const Geom &g, int32_t c, int &i, int &j, int &k)
{
    uint32_t u = (uint32_t)c & ~kPaired;
    i = (int)(u & ((1u << g.bx) - 1u));
    j = g.by ? (int)((u >> g.bx) & ((1u << g.by) - 1u)) : 0;
    k = (int)(u >> (g.bx + g.by));
}

__host__ __device__ inline int64_t tile_of(const Geom &g, int i, int j, int k)
{
    return ((int64_t)(k >> g.lt[2]) * g.nt[1] + (j >> g.lt[1])) * g.nt[0] + (i >> g.lt[0]);
}

__host__ __device__ inline int64_t fidx(const Geom &g, int i, int j, int k)
{
    return ((int64_t)k * g.ny + j) * g.nx + i;
}

// z index range of a component: half-integer-z components (Ez, Bx, By, Jz)
// live on k = 0..nz-1, the others on 0..nz; periodic z wraps over nz.
__host__ __device__ inline int zmax_of(const Geom &g, bool half_z)
{
    if (g.bc_z == 0) return g.nz - 1;
    return half_z ? g.nz - 1 : g.nz;
}

__host__ __device__ inline int wrapi(int i, int n)
{
    i %= n;
    return i < 0 ? i + n : i;
}

// ------------------------------------------------------------- buckets

__device__ __forceinline__ unsigned lane_id() { return threadIdx.x & 31u; }

// Reserve one slot per lane in the bucket of `dest` (dest < 0: no slot),
// one atomic per distinct destination in the warp.  All 32 lanes must call.
__device__ __forceinline__ int reserve_slot(int *cnt, int64_t dest)
{
    const unsigned lane = lane_id();
    const unsigned peers = __match_any_sync(0xffffffffu, (unsigned long long)dest);
    const int leader = __ffs(peers) - 1;
    const int rank = __popc(peers & ((1u << lane) - 1u));
    int base = 0;
    if (dest >= 0 && (int)lane == leader) base = atomicAdd(&cnt[dest], __popc(peers));
    base = __shfl_sync(peers, base, leader);
    return base + rank;
}

// slot of the p-th live particle of tile t (bottom run first, then top run)
__device__ __forceinline__ int64_t bucket_slot(int64_t t, int cap, int n_lo, int n_hi, int p)
{
    return t * (int64_t)cap + (p < n_lo ? p : cap - n_hi + (p - n_lo));
}

// run lengths of tile t; runs that overlap mean the bucket overflowed: that is
// reported and the runs are clamped so that no slot is read twice
__device__ __forceinline__ void bucket_counts(const int *lo, const int *hi, int64_t t, int cap, int &n_lo,
                                              int &n_hi, unsigned *err)
{
    n_lo = lo[t];
    n_hi = hi[t];
    if (n_lo > cap) n_lo = cap;
    if (n_hi > cap - n_lo) {
        if (err) atomicOr(err, ERR_CAPACITY);
        n_hi = cap - n_lo;
    }
}

// ---------------------------------------------------------------- shapes

// 1D B-spline weights of order S at a position p measured from node 0 of a
// window; returns the first node of the support and fills S+1 weights.
template <int S, typename real>
__device__ __forceinline__ int spline_weights(real p, real w[S + 1])
{
    if (S == 1) {
        real f = floor(p);
        real d = p - f;
        w[0] = real(1) - d;
        w[1] = d;
        return (int)f;
    } else {
        real c = floor(p + real(0.5));
        real d = p - c;
        real a = real(0.5) - d, b = real(0.5) + d;
        w[0] = real(0.5) * a * a;
        w[1] = real(0.75) - d * d;
        w[2] = real(0.5) * b * b;
        return (int)c - 1;
    }
}

// The same at an in-cell offset o in [0, 1) (the particle's own cell, an
// invariant of the store): for CIC the support starts at the cell's node, so
// the floor is 0 and the weights are those of spline_weights<1>(o) bit for bit.
template <int S, typename real>
__device__ __forceinline__ int offset_weights(real o, real w[S + 1])
{
    if (S == 1) {
        w[0] = real(1) - o;
        w[1] = o;
        return 0;
    }
    return spline_weights<S>(o, w);
}

// And at o - 1/2 (components staggered by half a cell), o in [0, 1): for CIC
// the floor is -1 or 0; the weights are those of spline_weights<1>(o - 1/2)
// bit for bit.
template <int S, typename real>
__device__ __forceinline__ int half_weights(real o, real w[S + 1])
{
    if (S == 1) {
        const real p = o - real(0.5);
        const bool lo = p < real(0);
        const real d = lo ? p + real(1) : p;
        w[0] = real(1) - d;
        w[1] = d;
        return lo ? -1 : 0;
    }
    return spline_weights<S>(o - real(0.5), w);
}

// Esirkepov window along one axis: old offset x0 in [0,1), new position x1 =
// x0 + d (|d| < 1), both relative to the old cell.  Returns the first node of
// a window of S+2 nodes that holds both supports, with S0 and DS = S1 - S0 on
// it, and whether the support moved to another first node.
template <int S, typename real>
__device__ __forceinline__ int esirk_axis_c(real x0, real x1, real S0[S + 2], real DS[S + 2], bool &crossed)
{
    real w0[S + 1], w1[S + 1];
    const int b0 = offset_weights<S>(x0, w0);  // x0: the in-cell offset at the start
    const int b1 = spline_weights<S>(x1, w1);
    const int anchor = b0 < b1 ? b0 : b1;
    const bool s0 = b0 != anchor, s1 = b1 != anchor;
    crossed = b0 != b1;
#pragma unroll
    for (int q = 0; q < S + 2; ++q) {
        const real v0 = s0 ? (q >= 1 ? w0[q - 1 < S ? q - 1 : S] : real(0)) : (q <= S ? w0[q <= S ? q : S] : real(0));
        const real v1 = s1 ? (q >= 1 ? w1[q - 1 < S ? q - 1 : S] : real(0)) : (q <= S ? w1[q <= S ? q : S] : real(0));
        S0[q] = v0;
        DS[q] = v1 - v0;
    }
    return anchor;
}

// The same for a start position x0 that need not lie in [0, 1) (within a
// cell of it): both supports from the spline itself.
template <int S, typename real>
__device__ __forceinline__ int esirk_axis_g(real x0, real x1, real S0[S + 2], real DS[S + 2], bool &crossed)
{
    real w0[S + 1], w1[S + 1];
    const int b0 = spline_weights<S>(x0, w0);
    const int b1 = spline_weights<S>(x1, w1);
    const int anchor = b0 < b1 ? b0 : b1;
    const bool s0 = b0 != anchor, s1 = b1 != anchor;
    crossed = b0 != b1;
#pragma unroll
    for (int q = 0; q < S + 2; ++q) {
        const real v0 = s0 ? (q >= 1 ? w0[q - 1 < S ? q - 1 : S] : real(0)) : (q <= S ? w0[q <= S ? q : S] : real(0));
        const real v1 = s1 ? (q >= 1 ? w1[q - 1 < S ? q - 1 : S] : real(0)) : (q <= S ? w1[q <= S ? q : S] : real(0));
        S0[q] = v0;
        DS[q] = v1 - v0;
    }
    return anchor;
}

// periodic index for i in [-n, 2n)
__device__ __forceinline__ int wrap1(int i, int n)
{
    return i < 0 ? i + n : (i >= n ? i - n : i);
}

// ----------------------------------------------------------------- Boris

// reciprocals used by the push: IEEE in FP64 (the debug path).  In FP32 the
// hardware reciprocal square root refined by one Newton-Raphson step for
// f(y) = 1/y^2 - x, y <- y (3 - x y^2) / 2, which squares its relative error
// (to below the FP32 rounding), so that the systematic error of v = u/gamma
// does not accumulate over many steps of a drifting plasma; and the correctly
// rounded reciprocal intrinsic.
__device__ __forceinline__ double rsqrt_p(double x) { return 1.0 / sqrt(x); }
__device__ __forceinline__ float rsqrt_p(float x)
{
    const float y = rsqrtf(x);
    return y * fmaf(-0.5f * x * y, y, 1.5f);
}
__device__ __forceinline__ double div_p(double a, double b) { return a / b; }
__device__ __forceinline__ float div_p(float a, float b) { return a * __frcp_rn(b); }

// Momenta are stored relative to the plasma drift u_d = (0, 0, U) (U = 0 in
// the lab frame, -gamma beta in the boosted frame): a record holds
// du = u - u_d.  In FP32 a momentum near -gamma beta resolves changes of one
// ulp of gamma beta, and v = u / gamma of it only ~6e-8, while a change du
// moves v_z by du / gamma^3; relative storage and the velocity formula below
// keep the plasma response at the relative precision of du itself.

// relativistic Boris rotation for du/dt = 2 pi (q/m)(E + u x B / gamma) on
// the stored du; eps = pi (q/m) dt is half the impulse factor.  The rotation
// acts on the full u^- = u_d + du^-; its increments are added to du, so zero
// fields leave du unchanged bit for bit.
template <typename real>
__device__ __forceinline__ void boris(real &dux, real &duy, real &duz, real U, real ex, real ey, real ez,
                                      real bx, real by, real bz, real eps)
{
    const real dmx = dux + eps * ex, dmy = duy + eps * ey, dmz = duz + eps * ez;
    const real umx = dmx, umy = dmy, umz = U + dmz;
    real f = eps * rsqrt_p(real(1) + umx * umx + umy * umy + umz * umz);
    real tx = f * bx, ty = f * by, tz = f * bz;
    real t2 = tx * tx + ty * ty + tz * tz;
    real s = div_p(real(2), real(1) + t2);
    real sx = s * tx, sy = s * ty, sz = s * tz;
    real upx = umx + (umy * tz - umz * ty);
    real upy = umy + (umz * tx - umx * tz);
    real upz = umz + (umx * ty - umy * tx);
    dux = dmx + (upy * sz - upz * sy) + eps * ex;
    duy = dmy + (upz * sx - upx * sz) + eps * ey;
    duz = dmz + (upx * sy - upy * sx) + eps * ez;
}

// correctly rounded add and multiply that the compiler may not contract into
// a fused multiply-add (the drift's displacement must round the same way in
// every kernel that applies it)
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// gamma_d^2 = 1 + U^2, 1 / gamma_d and the displacement per step dz (in
// cells, dtdh = dt / h_z) of the drift; the drifting ions and the electrons
// take all from here, and move by add_rn(offset, dz), so that a field-free
// electron and its ion move bit-identically
template <typename real>
struct Drift {
    real U, g2, ig, g, dz;
    __device__ __forceinline__ Drift(real u, real dtdh) : U(u)
    {
        g2 = add_rn(real(1), mul_rn(U, U));
        ig = rsqrt_p(g2);
        g = mul_rn(g2, ig);
        dz = mul_rn(mul_rn(U, ig), dtdh);
    }
};

// Velocity of a record with momentum u_d + du: returns v_z - v_d and sets
// vx, vy.  With gamma^2 = gamma_d^2 + D, D = du_z (2U + du_z) + p2,
// p2 = du_x^2 + du_y^2, and s = gamma + gamma_d,
//   v_z - v_d = [du_z (2 + E) - U p2] / (gamma gamma_d s),
//   E = gamma_d (gamma - gamma_d) - U du_z = (gamma_d (du_z^2 + p2) - U du_z D / s) / s,
// an exact rearrangement in which no term cancels the drift (E is of second
// order in du).  du = 0 gives exactly 0.  In the lab frame (U = 0) it is the
// plain du_z / gamma.
template <typename real>
__device__ __forceinline__ real drift_velocity(const Drift<real> &d, real dux, real duy, real duz, real &vx,
                                               real &vy)
{
    const real p2 = dux * dux + duy * duy;
    const real D = duz * (real(2) * d.U + duz) + p2;
    const real ig = rsqrt_p(d.g2 + D);
    vx = dux * ig;
    vy = duy * ig;
    if (d.U == real(0)) return duz * ig;
    const real is = div_p(real(1), (d.g2 + D) * ig + d.g);
    const real E = (d.g * (duz * duz + p2) - d.U * duz * D * is) * is;
    return (duz * (real(2) + E) - d.U * p2) * (ig * d.ig * is);
}

// An unevaluated sum h + l of two FP32 values, |l| <= ulp(h) / 2: 48 bits,
// from the error-free sum and product (Knuth, TAOCP 2, 4.2.2; Dekker, Numer.
// Math. 18, 1971, with a fused multiply-add for the product's error).  Sums and
// products of pairs round their low words and drop a.l b.l: each is good to
// about 46 bits of its larger operand.
// FP64 arithmetic gives 2 lanes per SM and cycle here, FP32 128, of which one
// of these operations takes 7 to 11.  The currents of records in relative
// form use them: they need the records' exact positions and far more than
// FP32's bits (see rel_actual), and end in fixed-point words that carry at
// most 43.
struct ff {
    float h, l;
    __device__ __forceinline__ ff() {}
    __device__ __forceinline__ ff(float x) : h(x), l(0.0f) {}
    __device__ __forceinline__ ff(int x) : h((float)x), l(0.0f) {}
    __device__ __forceinline__ ff(double x) : h((float)x), l((float)(x - (double)(float)x)) {}
    __device__ __forceinline__ ff(float x, float y) : h(x), l(y) {}
};
__device__ __forceinline__ ff two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b), z = __fsub_rn(s, a);
    return ff(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z)));
}
// |a| >= |b| or a = 0
__device__ __forceinline__ ff quick_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    return ff(s, __fsub_rn(b, __fsub_rn(s, a)));
}
__device__ __forceinline__ ff operator+(ff a, ff b)
{
    const ff s = two_sum(a.h, b.h);
    return quick_sum(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ ff operator-(ff a) { return ff(-a.h, -a.l); }
__device__ __forceinline__ ff operator-(ff a, ff b) { return a + -b; }
__device__ __forceinline__ ff operator*(ff a, ff b)
{
    const float p = __fmul_rn(a.h, b.h);
    float e = __fmaf_rn(a.h, b.h, -p);
    e = __fmaf_rn(a.h, b.l, e);
    e = __fmaf_rn(a.l, b.h, e);
    return quick_sum(p, e);
}
__device__ __forceinline__ ff &operator+=(ff &a, ff b)
{
    a = a + b;
    return a;
}
__device__ __forceinline__ bool operator==(ff a, ff b) { return a.h == b.h && a.l == b.l; }
// the exact floor (the low word decides where the high one is an integer)
__device__ __forceinline__ float floor_ff(ff a)
{
    const float f = floorf(a.h);
    return a.h == f && a.l < 0.0f ? f - 1.0f : f;
}

// Sums of many values of the working precision in FP64, compensated.  The
// FP64 pipe takes 2 lanes per SM and cycle, so an FP32 value is not converted
// and added by itself: up to kSumRun of them go into an unevaluated sum of
// three FP32 words by error-free two-sums (Knuth, TAOCP 2, 4.2.2), exact to
// far below FP64's last bit, and the three into an FP64 Kahan sum.  (With two
// words the totals were off by 4e-16 to 9e-16 of the sum, all to one side;
// FP64 Kahan sums of every value by 2e-16.)  FP64 values are added by Kahan
// directly.
constexpr int kSumRun = 32;
struct Kahan {
    double s = 0, c = 0;
    __device__ __forceinline__ void add(double v)
    {
        const double y = v - c, t = s + y;
        c = (t - s) - y;
        s = t;
    }
    __device__ __forceinline__ double value() const { return s - c; }
};
template <typename real> struct RunSum {
    Kahan k;
    __device__ __forceinline__ void add(double v) { k.add(v); }
    __device__ __forceinline__ void add_square(double v) { k.add(v * v); }
    __device__ __forceinline__ void flush() {}
};
template <> struct RunSum<float> {
    Kahan k;
    float h = 0, l = 0, m = 0;
    // a += b, the rounding error returned
    static __device__ __forceinline__ float add_to(float &a, float b)
    {
        const float t = __fadd_rn(a, b), z = __fsub_rn(t, a);
        const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(t, z)), __fsub_rn(b, z));
        a = t;
        return e;
    }
    __device__ __forceinline__ void add(float v) { m = __fadd_rn(m, add_to(l, add_to(h, v))); }
    // v^2 exactly: its rounded product and the product's error (in FP64
    // where either might leave the FP32 range)
    __device__ __forceinline__ void add_square(float v)
    {
        const float a = fabsf(v);
        if (!(a > 1e-12f && a < 1e15f) && a != 0.0f) {
            k.add((double)v * (double)v);
            return;
        }
        const float p = __fmul_rn(v, v);
        m = __fadd_rn(m, add_to(l, __fmaf_rn(v, v, -p)));
        add(p);
    }
    __device__ __forceinline__ void flush()
    {
        k.add((double)h + ((double)l + (double)m));
        h = l = m = 0.0f;
    }
};

// largest value below one, for offsets that round up to 1
template <typename real> __host__ __device__ inline real below_one();
template <> __host__ __device__ inline float below_one<float>() { return 0.99999994f; }
template <> __host__ __device__ inline double below_one<double>() { return 0.99999999999999989; }

// ---------------------------------------------------- kernel argument packs

template <typename real>
struct IonSide {         // the drifting-ion species of a step
    Species<real> in, out;
    int *in_lo, *in_hi, *out_lo, *out_hi;
    real jfac_z;         // -q h_z / (dt V) of the ions
};

template <typename real>
struct PushArgs {
    Geom g;
    const real *E[3];
    const real *B[3];
    real *J[3];
    Species<real> in, out;
    int *in_lo, *in_hi, *out_lo, *out_hi;   // run lengths per tile (see the layout note)
    real dtdh[3];       // dt / h_d
    real eps;           // pi (q/m) dt
    real jfac[3];       // -q h_d / (dt V): multiplied by w and the running sum
    real jyfac;         // q / V (2D out-of-plane current, times w vy)
    real u_drift;       // U: the plasma's drift momentum (0, 0, U); electron
                        // records store u - (0, 0, U), ions move with it
    // fixed-point current accumulation (FP32; FP64 uses 1): the per-particle
    // factors of Jx, Jy (2D: the out-of-plane factor), Jz are multiplied by
    // fx_scale[c]; a shared-tile node's integer sum times fx_quant[c] =
    // 1 / fx_scale[c] is its current; fx_lo = {2^K, 2^-K} scales the "lo" words
    real fx_scale[3], fx_quant[3], fx_lo[2];
    Species<real> ion_in;  // ion side the IONS phase reads next (released ions go there)
    int *ion_in_hi;        // its top-run lengths
    int fuse_ions;         // 1: the same CTA then moves and deposits the tile's ions
    IonSide<real> ions;    // (with fuse_ions) the ion sides and counters
    int rel;               // 1: electron records in relative form (rel_actual), currents
                           //    of electrons and ions in pairs of FP32 words (ff; FP64 build: FP64)
    unsigned *err;
};

template <typename real>
struct BucketArgs {      // re-bucket a flat list into tiles
    Geom g;
    Species<real> src, dst;
    int64_t n;
    int *dst_hi;         // top-run lengths of the destination side
    unsigned *err;
};

template <typename real>
struct CompactArgs {     // copy tiles into a flat list
    Geom g;
    Species<real> src, dst;
    const int *lo, *hi;
    const int64_t *offset;
};

template <typename real>
struct SortArgs {        // order every tile's bucket by cell (into the other side)
    Geom g;
    Species<real> in, out;
    int *in_lo, *in_hi, *out_lo;
    unsigned *err;
};

template <typename real>
struct BtdArgs {         // lab-frame snapshots filled during one step
    Geom g;
    const real *E0[3], *B0[3];  // fields at the start of the step
    const real *E1[3], *B1[3];  // and at its end
    real *data;                 // [nsnap][6][nz][nxs]
    int *flags;                 // [nsnap][nz]
    double gam, beta, hz;
    double zwin;                // window displacement (simulation-frame positions are relative to it)
    double t0, dt;              // the step's simulation-frame interval [t0, t0 + dt)
    double T0, dT, Z0, dZ;      // lab times and positions of the snapshots
    int nsnap, nz, nxs;
    int klo[64], kn[64];        // per snapshot, the lab points this step may fill
};

// per-step scalars of a captured step (CUDA graph): the antenna amplitude and
// the injection's times and lattice band, read by the kernels from device
// memory that the host refills before each replay
struct StepScal {
    double j0, t, t1;
    int64_t m_lo, m_hi;
};

struct InjectArgs {      // lattice load / boosted injection, FP64
    Geom g;
    double hx, hy, hz, Lx, Ly, Lz, gam, beta;
    int ppx, ppy, ppz;
    int64_t NX, NY, m_lo, m_hi;
    double z_start, z_end, ramp, ne, jitter, dzl, hz_lab, wfac;
    int nprof;
    double prof[16];
    // of the launch, rounded as the kernel's expressions would: the lattice
    // spacings across, the jitters, and the reciprocals of the divisors (with
    // fast set: see quotient)
    double spx, spy, jx, jy, jz, rhx, rhy, rhz, rgam, rlen;
    int fast;
    uint64_t seed;
    int mode;           // 0: in [zmin, Lz) at t; 1: crossing z = Lz during (t, t1]
    double t, t1;
    double zwin;        // window displacement (positions are relative to it)
    double zmin;        // lower end of a mode-0 load (0, or the layer a window move uncovers)
    int drift_ions;     // ions drift with the plasma
    int paired;         // electrons are placed paired with their ion (no ion record)
    int precision;      // 0 float, 1 double
    void *sp_e[kAttrs];  // ox oy oz w ux uy uz cell id dlx dly dlz of the electron side
    void *sp_i[kAttrs];  // same for the ion side (ux..uz, dl* unused)
    int sr_e, sc_e, sr_i, sc_i;  // elements from one block of 32 records to the next (reals, cell words)
    int *hi_e, *hi_i;    // top-run lengths of the electron / ion sides
    unsigned *err;
    // fixed-order ("flat") output of an adjoint run (flat_base >= 0, 2D):
    // lattice point q of the band goes to slot flat_base + q, alive or not
    int64_t flat_base;
    int *fe_ci, *fe_cj, *fe_ck;  // electron state (cj, oy in 3D)
    void *fe_ox, *fe_oy, *fe_oz, *fe_ux, *fe_uy, *fe_uz;
    unsigned char *fe_alive;
    int *fi_ck;                  // ion state
    void *fi_oz;
    unsigned char *fi_alive;
    int *f_ion_ci, *f_ion_cj;    // per slot, constant: the ion's transverse cells
    void *f_ion_ox, *f_ion_oy;   // and offsets,
    void *f_w;                   // the weight (shared by the pair)
    double *f_zeta;              // and the lab profile coordinate
    const StepScal *scal;        // non-null: t, t1, m_lo, m_hi from here (a captured
                                 // step; m_lo, m_hi above then bound the launch)
};

// One state of the flat particle store of an adjoint run (slot p is the same
// particle at every step; cj, oy only in 3D)
template <typename real>
struct FlatE {
    int *ci, *cj, *ck;
    real *ox, *oy, *oz, *ux, *uy, *uz;  // offsets; momenta relative to the drift
    unsigned char *alive;
};
template <typename real>
struct FlatI {
    int *ck;
    real *oz;
    unsigned char *alive;
};

template <typename real>
struct AdjArgs {
    Geom g;
    const real *E[3], *B[3];        // E^n, B^n
    real *J[3];                     // forward: current; reverse: its cotangent
    FlatE<real> in, out;            // electron states n and n+1
    FlatI<real> iin, iout;          // ion states n and n+1
    const real *w;                  // weights per slot
    const int *ion_ci, *ion_cj;     // ion transverse cells / offsets per slot
    const real *ion_ox, *ion_oy;
    int64_t n;                      // slots
    real dtdh[3];                   // dt / h_d
    real eps, u_drift;
    real jfac[3], jyfac, jfac_iz;   // electrons' -q h_d / (dt V), 2D q / V; ions' Jz factor
    real *lE[3], *lB[3];            // reverse: field cotangents at n
    real *lx, *ly, *lz, *lux, *luy, *luz;  // reverse: particle cotangents
    double *lw;                     // reverse: weight cotangents per slot
    const unsigned char *lj_plane;  // reverse: 1 for the cells ck within reach of a plane where lJ is not zero
    const unsigned char *f_plane;   // 1 for the cells ck within reach of a plane where E or B is not zero
    int with_ions;                  // the drifting ion of every slot too
};

// ------------------------------------------------- batched launch recording
//
// A batch of independent runs can step together with one launch per phase
// over the work items of all of them.  Such a step is built by running each
// run's own step on the host with a recorder installed on the calling
// thread: every launch function then appends what it would launch -- its
// phase, the batched form of its kernel, its argument struct and its number
// of work items (blocks, or tiles for the persistent particle kernels) --
// instead of launching.  A batched kernel maps its block (or the next item
// of a device-wide queue) to (run, item) through the runs' prefix sums of
// work items, copies that run's argument struct into shared memory and runs
// the same per-block body as the single-run kernel, so both give identical
// results.
//
// BatchLaunch(args, start, n, total, queue, stream): args = n argument
// structs (device), start = n + 1 prefix sums of the runs' work items
// (device), total = start[n], queue = a zeroed device counter (persistent
// kernels) or null.
using BatchLaunch = void (*)(const void *args, const int64_t *start, int n, int64_t total, unsigned *queue,
                             cudaStream_t s);
// phases in the order a step issues them
enum BatchPhase : int { kBPZero = 0, kBPPush, kBPIons, kBPAntenna, kBPFilter, kBPYee, kBPInject, kBPCount };
struct LaunchRecord {
    int chain, step, phase;
    BatchLaunch fn;
    std::vector<unsigned char> args;
    int64_t items;
    bool queue;  // the batched kernel pulls its items from a device counter
};
struct BatchRecorder {
    int chain = 0;             // the launch chain (stream) the current run belongs to
    int step = 0;
    int nctx = 1;              // runs in the batch (field kernels size their z chunks for all of them)
    bool unsupported = false;  // the step asked for something the batched step does not do
    std::vector<LaunchRecord> recs;
};
extern thread_local BatchRecorder *g_rec;

// true (and recorded) while a recorder is installed
template <typename A>
inline bool record_launch(int phase, BatchLaunch fn, const A &a, int64_t items, bool queue = false)
{
    static_assert(std::is_trivially_copyable<A>::value, "argument structs are copied as bytes");
    BatchRecorder *r = g_rec;
    if (!r) return false;
    LaunchRecord L;
    L.chain = r->chain;
    L.step = r->step;
    L.phase = phase;
    L.fn = fn;
    L.args.resize(sizeof(A));
    std::memcpy(L.args.data(), &a, sizeof(A));
    L.items = items;
    L.queue = queue;
    r->recs.push_back(std::move(L));
    return true;
}
// for launches with no batched form: true (the step is then not batched)
// while a recorder is installed
inline bool record_unsupported()
{
    if (!g_rec) return false;
    g_rec->unsupported = true;
    return true;
}
// runs whose field kernels share one launch (z chunks are sized for all)
inline int batch_runs() { return g_rec ? g_rec->nctx : 1; }

// true while this thread captures a batch's per-context graph
extern thread_local bool g_capture;

#ifdef __CUDACC__
// Launches that follow one another on a stream.  A step on a small grid is a
// chain of kernels of a few microseconds, and between two of them the GPU
// stood still for one to two.  A kernel launched by launch_chained may start
// as soon as every CTA of the one before it has left (a plain launch waits
// until that kernel's memory is flushed and it is retired as well); it begins
// with chain_begin(), which waits until the kernel before has completed and
// its writes are visible.  Every such kernel calls it first, in every thread,
// so a kernel that completes implies that all before it did, and what the
// stream holds afterwards (copies, events, other kernels) is ordered as ever.
// A batch's graph captures take plain launches.
//
// The next kernel is not let in earlier (griddepcontrol.launch_dependents):
// its CTAs then settle, waiting, on the first SMs that come free, and it runs
// with most of them on a few SMs.  us a step, plain launches / let in at the
// start of the kernel before / not let in early: 3D 48 x 48 x 64 cells 112 /
// 154 / 99, 128 x 128 x 256 1073 / 1083 / 1059, 256 x 256 x 512 6847 / 6953 /
// 6826; 2D 64 x 256 39.8 / 32.4 / 28.9, in FP64 125 / 146 / 115, 160 x 512
// quadratic 59 / 77 / 48, 256 x 8192 198 / 187 / 183, 1024 x 8192 652 / 644 /
// 638.  (In a process that has used more than about 8 streams every dependent
// launch takes the GPU's front end longer.  There the early start would hide
// more of it on 2D grids of some thousand tiles: 256 x 2048 80 / 66 / 69, 256 x
// 4096 118 / 105 / 108, 256 x 8192 200 / 186 / 188; with one stream 79 / 68 /
// 65, 118 / 110 / 103, 198 / 187 / 183.)
//
// A gradient's kernels on 2D grids of kEarlyNodes nodes or more do let the next
// one in (Geom::early): most of their grids cover every SM evenly, and
// gradients are run from programs with a stream per run, where launches take
// longer.  128 x 1536 cells, a forward and a reverse run of 100 steps, early /
// not: 14.1 / 14.7 ms on a process's sixth stream, 14.3 / 13.3 on its first.
constexpr int64_t kEarlyNodes = 150000;  // (64 x 600 cells: 9.4 / 8.2 ms on any stream)
__device__ __forceinline__ void chain_begin(int early)
{
    if (early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
// (cluster: CTAs per thread-block cluster)
template <typename... P, typename... A>
inline void launch_clusters(unsigned cluster, void (*kernel)(P...), unsigned grid, unsigned block, size_t smem,
                            cudaStream_t s, A... args)
{
    cudaLaunchConfig_t c{};
    c.gridDim = dim3(grid);
    c.blockDim = dim3(block);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    cudaLaunchAttribute at[2] = {};
    c.attrs = at;
    if (!g_capture) {
        at[c.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[c.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        at[c.numAttrs].id = cudaLaunchAttributeClusterDimension;
        at[c.numAttrs].val.clusterDim.x = cluster;
        at[c.numAttrs].val.clusterDim.y = 1;
        at[c.numAttrs++].val.clusterDim.z = 1;
    }
    (void)cudaLaunchKernelEx(&c, kernel, P(args)...);
}
template <typename... P, typename... A>
inline void launch_chained(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t s, A... args)
{
    launch_clusters(1, kernel, grid, block, smem, s, args...);
}

// the run owning work item `item`: the last r with start[r] <= item
__device__ __forceinline__ int batch_run_of(const int64_t *start, int n, int64_t item)
{
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (start[mid] <= item) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// all threads of the CTA copy an argument struct (global -> shared)
template <typename A>
__device__ __forceinline__ void batch_copy_args(A *dst, const A *src)
{
    static_assert(sizeof(A) % 4 == 0, "argument structs are copied as words");
    const int *s = reinterpret_cast<const int *>(src);
    int *d = reinterpret_cast<int *>(dst);
    for (int i = (int)threadIdx.x; i < (int)(sizeof(A) / 4); i += (int)blockDim.x) d[i] = s[i];
}

// block blockIdx.x of a batched launch with one block per work item: its
// run's arguments into *sa (shared), returns the block's index in its run
template <typename A>
__device__ __forceinline__ int64_t batch_block(const A *runs, const int64_t *start, int n, A *sa)
{
    __shared__ int s_r;
    if (threadIdx.x == 0) s_r = batch_run_of(start, n, (int64_t)blockIdx.x);
    __syncthreads();
    const int r = s_r;
    batch_copy_args(sa, runs + r);
    __syncthreads();
    return (int64_t)blockIdx.x - start[r];
}
#endif

// the zeroing of a current buffer as a batchable launch (cudaMemsetAsync
// otherwise)
template <typename real>
struct ZeroArgs {
    real *p;
    int64_t n;
};
// (returns the kernels it launches: none where a memset does it)
template <typename real> int launch_zero(real *p, int64_t n, cudaStream_t s);
// the same for two arrays in one launch (q: m bytes)
template <typename real> void launch_zero2(real *p, int64_t n, unsigned char *q, int64_t m, int early, cudaStream_t s);
// SMs of the current device (cached per device)
int device_sms();

// host launchers (defined in the .cu files)
template <typename real> void launch_push(const PushArgs<real> &a, cudaStream_t s);
template <typename real> void launch_ions(const PushArgs<real> &a, cudaStream_t s);
template <typename real> void launch_bucket(const BucketArgs<real> &a, cudaStream_t s);
template <typename real> void launch_compact(const CompactArgs<real> &a, cudaStream_t s);
template <typename real> void launch_sort_cells(const SortArgs<real> &a, cudaStream_t s);
template <typename real>
void launch_rho(const Geom &g, const Species<real> &sp, const int *lo, const int *hi, real qfac, real *rho,
                cudaStream_t s);
template <typename real>
int launch_particle_sums(const Geom &g, const Species<real> &sp, const int *lo, const int *hi, double q,
                          real u_drift, double wmax, double *partials, int max_blocks, cudaStream_t s);
void launch_inject(const InjectArgs &a, cudaStream_t s);
template <typename real>
void launch_btd(const BtdArgs<real> &a, cudaStream_t s);
// n components of the lab-frame E, B on the grid (comp[q] in 0..5, F the
// component, P its partner: By, Bx, -, Ey, Ex, -) into out[q]
template <typename real>
struct LabArgs {
    Geom g;
    int comp[6];
    const real *F[6], *P[6];
    real *out[6];
    double gam, beta;
};
template <typename real> void launch_lab_fields(const LabArgs<real> &a, int n, int sms, cudaStream_t s);
// moving window: every field plane k of dst takes plane k + S of src (zero
// above), for the nine components
template <typename real>
void launch_window_fields(const Geom &g, real *const src[9], real *const dst[9], int S, cudaStream_t s);
// moving window: the bucket of tile t of the output side takes the bucket of
// tile t + m ntx nty of the input side with every cell index S = m tz lower
template <typename real>
void launch_window_particles(const Geom &g, const Species<real> &in, const Species<real> &out, const int *in_lo,
                             const int *in_hi, int *out_lo, int *out_hi, int m, int S, cudaStream_t s);

template <typename real>
void launch_yee(const Geom &g, real *const F[9], real *const F1[6], double dt, double hx, double hy, double hz,
                cudaStream_t s);
template <typename real>
void launch_filter(const Geom &g, real *const J[3], real *tmp, int npass, cudaStream_t s);
// all passes from src (3 contiguous components, left unchanged) into J;
// false (nothing launched) where only the per-pass path applies (npass > 4)
template <typename real>
bool launch_filter_from(const Geom &g, const real *src, real *const J[3], int npass, cudaStream_t s);
// j0p non-null: the amplitude is read from device memory (a captured step)
template <typename real>
void launch_antenna(const Geom &g, real *J, int pol, int ka, double j0, double hx, double hy,
                    double xc, double yc, double waist, cudaStream_t s, const double *j0p = nullptr);
template <typename real>
int launch_field_sums(const Geom &g, real *const F[9], double *partials, int nblocks,
                       cudaStream_t s);
// adjoint: flat forward steps (electrons, and the slots' ions) and their transposes
template <typename real> void launch_adj_push(const AdjArgs<real> &a, cudaStream_t s);
template <typename real> void launch_adj_push_vjp(const AdjArgs<real> &a, cudaStream_t s);
template <typename real>
void launch_adj_yee(const Geom &g, real *lE[3], real *lB[3], real *lE0[3], real *pE[3], real *lJ[3], double dt,
                    double hx, double hy, double hz, unsigned char *near, cudaStream_t s);
template <typename real>
void launch_adj_antenna(const Geom &g, const real *lJ, int pol, int ka, double hx, double hy, double xc, double yc,
                        double waist, double fa, double fw, double *s, cudaStream_t st);
void launch_adj_profile(int64_t n, const double *lw, const void *w, int precision, const double *zeta, int M,
                        const double *coef, double *out, cudaStream_t s);
// planes[k] = 1 where any of the three components of lJ is non-zero on plane k
template <typename real>
void launch_adj_planes(const Geom &g, const real *F, int nc, unsigned char *near, cudaStream_t s);

}  // namespace pic
