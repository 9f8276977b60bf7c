// pic_fields.cu -- field kernels: Yee leapfrog with Mur boundaries, binomial
// current filter, laser antenna and the FP64 field-energy reduction.
//
// Yee (1966) on the staggered lattice of pic_internal.cuh, B split in two half
// steps so that E and B both live at integer times:
//   B -= (dt/2) curl E;   E += dt (curl B - 2 pi J);   B -= (dt/2) curl E,
// all three in one kernel that reads E^n, B^n from one field buffer and writes
// E^{n+1}, B^{n+1} to another (yee2d_kernel, yee3d_kernel).  With absorbing z
// the tangential E (Ex, Ey) on the end planes k = 0 and k = nz follows Mur's
// first-order condition (Mur 1981).
#include "pic.h"
#include "pic_internal.cuh"


namespace pic {

template <typename real>
struct Ptr9 {
    real *p[9];
};

template <typename real>
struct YeeArgs {
    Geom g;
    const real *E[3], *B[3];  // E^n, B^n
    real *E1[3], *B1[3];      // E^{n+1}, B^{n+1} (another buffer)
    const real *J[3];
    real hb, he;              // dt/2 (B half steps), dt (E step)
    real ihx, ihy, ihz;       // 1 / h_d
    real twopi;               // 2 pi
    real mur;                 // (dt - hz) / (dt + hz)
    int cz, nchunks;          // z planes per chunk, chunks
};

// CTAs of a grid-stride loop over n items: all of them, at most 32 per SM
static unsigned grid_for(int64_t n, int block)
{
    int64_t b = (n + block - 1) / block;
    const int64_t cap = (int64_t)device_sms() * 32;
    return (unsigned)(b < cap ? (b > 0 ? b : 1) : cap);
}

// A march loads each plane one iteration ahead, which covers the L2's latency
// but not the memory's under load; so the lines of the planes kAhead further
// on are brought into the L2, one line per lane (each row of 32 columns lies
// in two lines at most).
constexpr int kAhead = 3;
__device__ __forceinline__ void prefetch_l2(const void *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// Longest chunk of the 3D marches.  The columns next to each other share their
// halo through the L2 only while they are at about the same plane; in longer
// chunks they drift apart.  256 x 256 x 512 nodes, chunks as the waves alone
// would have them (103 planes) / at most 64 / 32 / 16: Yee 456 / 436 / 435 /
// 441 us, filter (2 passes) 324 / 271 / 268 / 295.
constexpr int kChunk3 = 32;

// Planes per chunk of a march over nzo planes in ncol columns, each chunk
// walking `halo` planes more than its own and `resident` chunks running at a
// time: the length that makes the number of waves times a wave's length
// smallest (at least cmin planes, about cmax at most where cmax > 0).
static int chunk_planes(int64_t nzo, int64_t ncol, int64_t resident, int halo, int cmin, int cmax = 0)
{
    int64_t m0 = (ncol + resident - 1) / resident;
    if (cmax > 0) {
        const int64_t need = ((nzo + cmax - 1) / cmax * ncol + resident - 1) / resident;
        if (need > m0) m0 = need;
    }
    int64_t best = cmax > 0 && cmax < nzo ? cmax : nzo, cost = INT64_MAX;
    for (int64_t m = m0; m < m0 + 16; ++m) {
        const int64_t chunks = m * resident / ncol;
        if (chunks < 1) continue;
        int64_t cz = (nzo + chunks - 1) / chunks;
        if (cz < cmin) cz = cmin;
        if (cz > nzo) cz = nzo;
        const int64_t waves = (ncol * ((nzo + cz - 1) / cz) + resident - 1) / resident;
        if (waves * (cz + halo) < cost) {
            cost = waves * (cz + halo);
            best = cz;
        }
    }
    return (int)best;
}

// --------------------------------------------------- 2D Yee, column march

// One Yee step in one pass over the grid, as a march up z with the planes in
// registers: each thread holds one (x, y) column and a chunk of z planes,
// and at plane k of the march computes
//   Bh(k)   = B^n(k) - (dt/2) curl E^n       (E^n at k and k+1)
//   E'(k)   = E^n(k) + dt (curl Bh - 2 pi J)  (Bh at k and k-1)
//   B'(k-1) = Bh(k-1) - (dt/2) curl E'       (E' at k-1 and k)
// and writes E'(k-1), B'(k-1) to the other field buffer, so that no thread
// reads a value another one writes.  Every z neighbour is a register of the
// previous iteration, every x neighbour a warp shuffle (lane l holds column
// x0 + l - 1), and the loads of a plane are issued an iteration ahead of
// their use.  Each curl takes the next neighbour on one side, so the columns
// at a strip's edges are its halo: Bh is exact on lanes 0-30, E' on lanes
// 1-30 and B' on lanes 1-29, the strip's own kColOwn columns.  With absorbing
// z the tangential E (Ex, Ey) of the end planes follows Mur's first-order
// condition
//   E0^{n+1} = E1^n + (dt - dz)/(dt + dz) (E1^{n+1} - E0^n)
// (Mur 1981), evaluated from the registers once E' of the neighbouring plane
// is known.  The chunk [z0, z1) starts two planes early (E' of plane z0 - 1
// for Mur's upper plane when nz - 1 is the plane before the chunk) and ends
// one late.  The arithmetic per node is that of the split-B leapfrog written
// out term by term; planes a component does not have (Ez, Bx, By at k = nz;
// every component at k = nz with periodic z) are neither read nor written.
//
// In 2D (d/dy = 0) a warp is independent of the others: no shared memory
// and no barrier.
constexpr int kColOwn = 29;

template <typename real>
__device__ __forceinline__ void yee2d_body(const YeeArgs<real> &a, const int strip, const int chunk)
{
    const Geom &g = a.g;
    const bool per = g.bc_z == 0;
    const int nzo = per ? g.nz : g.nz + 1;
    const unsigned lane = threadIdx.x & 31u;
    const int x = strip * kColOwn + (int)lane - 1;
    const int gx = x >= 0 && x < g.nx ? x : wrapi(x, g.nx);
    const bool own = lane >= 1u && lane <= (unsigned)kColOwn && x < g.nx;
    const int z0 = chunk * a.cz;
    const int z1 = chunk == a.nchunks - 1 ? nzo : z0 + a.cz;
    // offset of this lane's node of plane k of a component with integer
    // (half = false) or half-integer z, -1 where the component has no plane k
    auto off = [&](int k, bool half) -> int64_t {
        const int kk = per ? wrapi(k, g.nz) : (k >= 0 && k <= zmax_of(g, half) ? k : -1);
        return kk >= 0 ? (int64_t)kk * g.plane + gx : int64_t(-1);
    };
    auto ld = [&](const real *p, int64_t o) { return o >= 0 ? p[o] : real(0); };
    auto dn = [&](real v) { return __shfl_down_sync(0xffffffffu, v, 1); };  // the value at x + 1
    auto up = [&](real v) { return __shfl_up_sync(0xffffffffu, v, 1); };    // the value at x - 1
    const real zero = real(0);
    const int kb = z0 - 2;
    // offsets of planes k and k + 1 (carried along the march)
    int64_t oi0 = off(kb, false), oh0 = off(kb, true), oi1 = off(kb + 1, false), oh1 = off(kb + 1, true);
    // E^n of planes k - 1 (for Mur), k and k + 1; B^n and J of plane k;
    // Bh and E' of plane k - 1
    real emx = 0, emy = 0;
    real ex0 = ld(a.E[0], oi0), ey0 = ld(a.E[1], oi0), ez0 = ld(a.E[2], oh0);
    real ex1 = ld(a.E[0], oi1), ey1 = ld(a.E[1], oi1), ez1 = ld(a.E[2], oh1);
    real bx = ld(a.B[0], oh0), by = ld(a.B[1], oh0), bz = ld(a.B[2], oi0);
    real jx = ld(a.J[0], oi0), jy = ld(a.J[1], oi0), jz = ld(a.J[2], oh0);
    real bmx = 0, bmy = 0, bmz = 0, fpx = 0, fpy = 0, fpz = 0;
    real murx = 0, mury = 0;  // E'(nz) x, y by Mur's condition (from plane nz - 1)
    for (int k = kb; k <= z1; ++k) {
        // the next plane's loads, used one iteration later
        const int64_t oi2 = off(k + 2, false), oh2 = off(k + 2, true);
        const real nex = ld(a.E[0], oi2), ney = ld(a.E[1], oi2), nez = ld(a.E[2], oh2);
        const real nbx = ld(a.B[0], oh1), nby = ld(a.B[1], oh1), nbz = ld(a.B[2], oi1);
        const real njx = ld(a.J[0], oi1), njy = ld(a.J[1], oi1), njz = ld(a.J[2], oh1);
        // ---- Bh(k)
        const bool vxy = oh0 >= 0, vz = oi0 >= 0;
        const real eyr = dn(ey0), ezr = dn(ez0);
        const real dEy_dz = (ey1 - ey0) * a.ihz;
        const real dEx_dz = (ex1 - ex0) * a.ihz;
        const real dEz_dx = (ezr - ez0) * a.ihx;
        const real dEy_dx = (eyr - ey0) * a.ihx;
        const real hx = vxy ? bx - a.hb * (zero - dEy_dz) : real(0);
        const real hy = vxy ? by - a.hb * (dEx_dz - dEz_dx) : real(0);
        const real hz = vz ? bz - a.hb * (dEy_dx - zero) : real(0);
        // ---- E'(k)
        real fx = ex0, fy = ey0, fz = 0;
        {
            const real hyl = up(hy), hzl = up(hz);
            const bool ve = per || (k >= 1 && k <= g.nz - 1), vze = oh0 >= 0;
            if (ve) {
                const real dBy_dz = (hy - bmy) * a.ihz;
                fx = ex0 + a.he * ((zero - dBy_dz) - a.twopi * jx);
                const real dBx_dz = (hx - bmx) * a.ihz;
                const real dBz_dx = (hz - hzl) * a.ihx;
                fy = ey0 + a.he * ((dBx_dz - dBz_dx) - a.twopi * jy);
            }
            const real dBy_dx = (hy - hyl) * a.ihx;
            fz = vze ? ez0 + a.he * ((dBy_dx - zero) - a.twopi * jz) : real(0);
            if (!per) {
                if (k == 1) {  // E'(0) x, y from plane 1
                    fpx = ex0 + a.mur * (fx - emx);
                    fpy = ey0 + a.mur * (fy - emy);
                }
                if (k == g.nz - 1) {  // E'(nz) x, y from plane nz - 1
                    murx = ex0 + a.mur * (fx - ex1);
                    mury = ey0 + a.mur * (fy - ey1);
                }
                if (k == g.nz) {
                    fx = murx;
                    fy = mury;
                }
            }
        }
        // ---- E'(k - 1), B'(k - 1) of the own columns
        {
            const int kw = k - 1;
            const real fpyr = dn(fpy), fpzr = dn(fpz);
            if (kw >= z0 && kw < z1 && own) {
                const int64_t o = (int64_t)kw * g.plane + x;
                const bool wxy = kw <= zmax_of(g, false), wz = kw <= zmax_of(g, true);
                if (wxy) {
                    a.E1[0][o] = fpx;
                    a.E1[1][o] = fpy;
                }
                if (wz) {
                    a.E1[2][o] = fpz;
                    const real dEy_dz1 = (fy - fpy) * a.ihz;
                    a.B1[0][o] = bmx - a.hb * (zero - dEy_dz1);
                    const real dEx_dz1 = (fx - fpx) * a.ihz;
                    const real dEz_dx1 = (fpzr - fpz) * a.ihx;
                    a.B1[1][o] = bmy - a.hb * (dEx_dz1 - dEz_dx1);
                }
                if (wxy) {
                    const real dEy_dx1 = (fpyr - fpy) * a.ihx;
                    a.B1[2][o] = bmz - a.hb * (dEy_dx1 - zero);
                }
            }
        }
        // ---- shift the march by one plane
        oi0 = oi1;
        oh0 = oh1;
        oi1 = oi2;
        oh1 = oh2;
        emx = ex0;
        emy = ey0;
        ex0 = ex1;
        ey0 = ey1;
        ez0 = ez1;
        ex1 = nex;
        ey1 = ney;
        ez1 = nez;
        bx = nbx;
        by = nby;
        bz = nbz;
        jx = njx;
        jy = njy;
        jz = njz;
        bmx = hx;
        bmy = hy;
        bmz = hz;
        fpx = fx;
        fpy = fy;
        fpz = fz;
    }
}

// The march of a chunk whose planes k - 1 .. k + 2 all lie in the grid (every
// chunk but the ones at the z ends): the same arithmetic without validity
// tests and Mur's planes, one 32-bit byte offset for all components (the
// components' bases are uniform), the registers of two planes renamed by
// unrolling: about 80 instructions per node where the general march takes 330.
// 64 x 512 cells 9.2 -> 4.8 us, 256 x 1000 10.6 -> 5.9 us (with chunks of 4
// planes instead of 12); 256 x 8192 31 us before and after (the memory's rate).
template <typename real>
__device__ __forceinline__ bool yee2d_inner(const YeeArgs<real> &a, const int strip, const int chunk)
{
    const Geom &g = a.g;
    const int z0 = chunk * a.cz, z1 = z0 + a.cz;
    if (z0 < 1 || z1 + 2 > g.nz - 1 || chunk == a.nchunks - 1 || g.ncomp * (int64_t)sizeof(real) >= (int64_t(1) << 32))
        return false;
    const unsigned lane = threadIdx.x & 31u;
    const int x = strip * kColOwn + (int)lane - 1;
    const int gx = x >= 0 && x < g.nx ? x : wrapi(x, g.nx);
    const bool own = lane >= 1u && lane <= (unsigned)kColOwn && x < g.nx;
    auto dn = [&](real v) { return __shfl_down_sync(0xffffffffu, v, 1); };  // the value at x + 1
    auto up = [&](real v) { return __shfl_up_sync(0xffffffffu, v, 1); };    // the value at x - 1
    auto ld = [](const real *p, unsigned b) {
        return *reinterpret_cast<const real *>(reinterpret_cast<const char *>(p) + b);
    };
    auto st = [](real *p, unsigned b, real v) { *reinterpret_cast<real *>(reinterpret_cast<char *>(p) + b) = v; };
    const real zero = real(0);
    const unsigned dp = (unsigned)(g.plane * sizeof(real));
    unsigned o = (unsigned)(((int64_t)(z0 - 1) * g.plane + gx) * sizeof(real));  // plane k
    real ex0 = ld(a.E[0], o), ey0 = ld(a.E[1], o), ez0 = ld(a.E[2], o);
    real ex1 = ld(a.E[0], o + dp), ey1 = ld(a.E[1], o + dp), ez1 = ld(a.E[2], o + dp);
    real bx = ld(a.B[0], o), by = ld(a.B[1], o), bz = ld(a.B[2], o);
    real jx = 0, jy = 0, jz = 0;  // (E' of the first plane is not used)
    real bmx = 0, bmy = 0, bmz = 0, fpx = 0, fpy = 0, fpz = 0;
    // lane l < 18 prefetches a line of row l / 2 of Ex .. Jz
    const char *pf;
    {
        const int c = (int)(lane >> 1);
        const real *base = c == 0 ? a.E[0] : c == 1 ? a.E[1] : c == 2 ? a.E[2] : c == 3 ? a.B[0] : c == 4 ? a.B[1]
                         : c == 5 ? a.B[2] : c == 6 ? a.J[0] : c == 7 ? a.J[1] : a.J[2];
        const unsigned oa = __shfl_sync(0xffffffffu, o, 0), ob = __shfl_sync(0xffffffffu, o, 31);
        pf = reinterpret_cast<const char *>(base) + ((lane & 1u) ? ob : oa) + (kAhead + 1) * (size_t)dp;
    }
#pragma unroll 2
    for (int k = z0 - 1; k <= z1; ++k) {
        if (lane < 18u && k + kAhead <= z1) prefetch_l2(pf);
        pf += dp;
        // the next plane's loads, used one iteration later
        const real nex = ld(a.E[0], o + 2 * dp), ney = ld(a.E[1], o + 2 * dp), nez = ld(a.E[2], o + 2 * dp);
        const real nbx = ld(a.B[0], o + dp), nby = ld(a.B[1], o + dp), nbz = ld(a.B[2], o + dp);
        const real njx = ld(a.J[0], o + dp), njy = ld(a.J[1], o + dp), njz = ld(a.J[2], o + dp);
        // ---- Bh(k)
        const real eyr = dn(ey0), ezr = dn(ez0);
        const real dEy_dz = (ey1 - ey0) * a.ihz;
        const real dEx_dz = (ex1 - ex0) * a.ihz;
        const real dEz_dx = (ezr - ez0) * a.ihx;
        const real dEy_dx = (eyr - ey0) * a.ihx;
        const real hx = bx - a.hb * (zero - dEy_dz);
        const real hy = by - a.hb * (dEx_dz - dEz_dx);
        const real hz = bz - a.hb * (dEy_dx - zero);
        // ---- E'(k)
        const real hyl = up(hy), hzl = up(hz);
        const real dBy_dz = (hy - bmy) * a.ihz;
        const real fx = ex0 + a.he * ((zero - dBy_dz) - a.twopi * jx);
        const real dBx_dz = (hx - bmx) * a.ihz;
        const real dBz_dx = (hz - hzl) * a.ihx;
        const real fy = ey0 + a.he * ((dBx_dz - dBz_dx) - a.twopi * jy);
        const real dBy_dx = (hy - hyl) * a.ihx;
        const real fz = ez0 + a.he * ((dBy_dx - zero) - a.twopi * jz);
        // ---- E'(k - 1), B'(k - 1) of the own columns
        const real fpyr = dn(fpy), fpzr = dn(fpz);
        if (k > z0 && own) {
            const unsigned ow = o - dp;
            st(a.E1[0], ow, fpx);
            st(a.E1[1], ow, fpy);
            st(a.E1[2], ow, fpz);
            const real dEy_dz1 = (fy - fpy) * a.ihz;
            st(a.B1[0], ow, bmx - a.hb * (zero - dEy_dz1));
            const real dEx_dz1 = (fx - fpx) * a.ihz;
            const real dEz_dx1 = (fpzr - fpz) * a.ihx;
            st(a.B1[1], ow, bmy - a.hb * (dEx_dz1 - dEz_dx1));
            const real dEy_dx1 = (fpyr - fpy) * a.ihx;
            st(a.B1[2], ow, bmz - a.hb * (dEy_dx1 - zero));
        }
        o += dp;
        ex0 = ex1;
        ey0 = ey1;
        ez0 = ez1;
        ex1 = nex;
        ey1 = ney;
        ez1 = nez;
        bx = nbx;
        by = nby;
        bz = nbz;
        jx = njx;
        jy = njy;
        jz = njz;
        bmx = hx;
        bmy = hy;
        bmz = hz;
        fpx = fx;
        fpy = fy;
        fpz = fz;
    }
    return true;
}

// ------------------------------------------------------ 3D Yee, column march

// The Yee step on 3D grids with the planes in registers: a CTA of 16 warps
// owns kCol3Y x kColOwn (y, x) columns and a chunk of z planes; warp w holds
// row y = y0 + w - 1 and lane l column x = x0 + l - 1 (both wrapped), so that
// the x neighbours are shuffles and the y neighbours come through shared
// memory, two exchanges per plane (E^n(k) and E'(k-1) with the row above;
// Bh(k) with the row below).  Bh is exact on lanes 0-30 and warps 0-14, E' on
// lanes 1-30 and warps 1-14, B' on lanes 1-29 and warps 1-13, the own
// columns.  The march, its chunk ends, Mur's planes and the arithmetic are
// yee2d_body's with the y terms of the curls.
constexpr int kCol3Y = 13, kCol3Warps = 16;

template <typename real>
__device__ __forceinline__ void yee3d_body(const YeeArgs<real> &a, real (*xs)[6][kCol3Warps][32], const int sx,
                                           const int sy, const int chunk)
{
    const Geom &g = a.g;
    const bool per = g.bc_z == 0;
    const int nzo = per ? g.nz : g.nz + 1;
    const unsigned lane = threadIdx.x & 31u;
    const int w = (int)(threadIdx.x >> 5);
    const int x = sx * kColOwn + (int)lane - 1, y = sy * kCol3Y + w - 1;
    const int gx = x >= 0 && x < g.nx ? x : wrapi(x, g.nx);
    const int gy = y >= 0 && y < g.ny ? y : wrapi(y, g.ny);
    const int64_t col = (int64_t)gy * g.nx + gx;
    const bool own = lane >= 1u && lane <= (unsigned)kColOwn && w >= 1 && w <= kCol3Y && x < g.nx && y < g.ny;
    const int wu = w + 1 < kCol3Warps ? w + 1 : w, wd = w >= 1 ? w - 1 : w;  // rows above and below (halo: own)
    const int z0 = chunk * a.cz;
    const int z1 = chunk == a.nchunks - 1 ? nzo : z0 + a.cz;
    auto off = [&](int k, bool half) -> int64_t {
        const int kk = per ? wrapi(k, g.nz) : (k >= 0 && k <= zmax_of(g, half) ? k : -1);
        return kk >= 0 ? (int64_t)kk * g.plane + col : int64_t(-1);
    };
    auto ld = [&](const real *p, int64_t o) { return o >= 0 ? p[o] : real(0); };
    auto dn = [&](real v) { return __shfl_down_sync(0xffffffffu, v, 1); };  // x + 1
    auto up = [&](real v) { return __shfl_up_sync(0xffffffffu, v, 1); };    // x - 1
    const real zero = real(0);
    const int kb = z0 - 2;
    int64_t oi0 = off(kb, false), oh0 = off(kb, true), oi1 = off(kb + 1, false), oh1 = off(kb + 1, true);
    real emx = 0, emy = 0;
    real ex0 = ld(a.E[0], oi0), ey0 = ld(a.E[1], oi0), ez0 = ld(a.E[2], oh0);
    real ex1 = ld(a.E[0], oi1), ey1 = ld(a.E[1], oi1), ez1 = ld(a.E[2], oh1);
    real bx = ld(a.B[0], oh0), by = ld(a.B[1], oh0), bz = ld(a.B[2], oi0);
    real jx = ld(a.J[0], oi0), jy = ld(a.J[1], oi0), jz = ld(a.J[2], oh0);
    real bmx = 0, bmy = 0, bmz = 0, fpx = 0, fpy = 0, fpz = 0;
    real murx = 0, mury = 0;
    for (int k = kb; k <= z1; ++k) {
        const int P = k & 1;
        const int64_t oi2 = off(k + 2, false), oh2 = off(k + 2, true);
        const real nex = ld(a.E[0], oi2), ney = ld(a.E[1], oi2), nez = ld(a.E[2], oh2);
        const real nbx = ld(a.B[0], oh1), nby = ld(a.B[1], oh1), nbz = ld(a.B[2], oi1);
        const real njx = ld(a.J[0], oi1), njy = ld(a.J[1], oi1), njz = ld(a.J[2], oh1);
        // ---- exchange 1: E^n(k) and E'(k - 1) with the row above
        xs[P][0][w][lane] = ex0;
        xs[P][1][w][lane] = ez0;
        xs[P][2][w][lane] = fpx;
        xs[P][3][w][lane] = fpz;
        __syncthreads();
        const real exu = xs[P][0][wu][lane], ezu = xs[P][1][wu][lane];
        const real fpxu = xs[P][2][wu][lane], fpzu = xs[P][3][wu][lane];
        // ---- Bh(k)
        const bool vxy = oh0 >= 0, vz = oi0 >= 0;
        const real eyr = dn(ey0), ezr = dn(ez0);
        const real dEz_dy = (ezu - ez0) * a.ihy;
        const real dEx_dy = (exu - ex0) * a.ihy;
        const real dEy_dz = (ey1 - ey0) * a.ihz;
        const real dEx_dz = (ex1 - ex0) * a.ihz;
        const real dEz_dx = (ezr - ez0) * a.ihx;
        const real dEy_dx = (eyr - ey0) * a.ihx;
        const real hx = vxy ? bx - a.hb * (dEz_dy - dEy_dz) : real(0);
        const real hy = vxy ? by - a.hb * (dEx_dz - dEz_dx) : real(0);
        const real hz = vz ? bz - a.hb * (dEy_dx - dEx_dy) : real(0);
        // ---- exchange 2: Bh(k) with the row below
        xs[P][4][w][lane] = hx;
        xs[P][5][w][lane] = hz;
        __syncthreads();
        const real hxd = xs[P][4][wd][lane], hzd = xs[P][5][wd][lane];
        // ---- E'(k)
        real fx = ex0, fy = ey0, fz = 0;
        {
            const real hyl = up(hy), hzl = up(hz);
            const bool ve = per || (k >= 1 && k <= g.nz - 1), vze = oh0 >= 0;
            if (ve) {
                const real dBz_dy = (hz - hzd) * a.ihy;
                const real dBy_dz = (hy - bmy) * a.ihz;
                fx = ex0 + a.he * ((dBz_dy - dBy_dz) - a.twopi * jx);
                const real dBx_dz = (hx - bmx) * a.ihz;
                const real dBz_dx = (hz - hzl) * a.ihx;
                fy = ey0 + a.he * ((dBx_dz - dBz_dx) - a.twopi * jy);
            }
            const real dBy_dx = (hy - hyl) * a.ihx;
            const real dBx_dy = (hx - hxd) * a.ihy;
            fz = vze ? ez0 + a.he * ((dBy_dx - dBx_dy) - a.twopi * jz) : real(0);
            if (!per) {
                if (k == 1) {
                    fpx = ex0 + a.mur * (fx - emx);
                    fpy = ey0 + a.mur * (fy - emy);
                }
                if (k == g.nz - 1) {
                    murx = ex0 + a.mur * (fx - ex1);
                    mury = ey0 + a.mur * (fy - ey1);
                }
                if (k == g.nz) {
                    fx = murx;
                    fy = mury;
                }
            }
        }
        // ---- E'(k - 1), B'(k - 1) of the own columns.  At k = 1 Mur's
        // condition has just set E'(0) x, y: the row above's E'x(0), which B'z
        // reads, is exchanged again (k is the same for the whole CTA)
        real fpxu2 = fpxu;
        if (!per && k == 1) {
            xs[P][2][w][lane] = fpx;
            __syncthreads();
            fpxu2 = xs[P][2][wu][lane];
        }
        {
            const int kw = k - 1;
            const real fpyr = dn(fpy), fpzr = dn(fpz);
            if (kw >= z0 && kw < z1 && own) {
                const int64_t o = (int64_t)kw * g.plane + col;
                const bool wxy = kw <= zmax_of(g, false), wz = kw <= zmax_of(g, true);
                if (wxy) {
                    a.E1[0][o] = fpx;
                    a.E1[1][o] = fpy;
                }
                if (wz) {
                    a.E1[2][o] = fpz;
                    const real dEz_dy1 = (fpzu - fpz) * a.ihy;
                    const real dEy_dz1 = (fy - fpy) * a.ihz;
                    a.B1[0][o] = bmx - a.hb * (dEz_dy1 - dEy_dz1);
                    const real dEx_dz1 = (fx - fpx) * a.ihz;
                    const real dEz_dx1 = (fpzr - fpz) * a.ihx;
                    a.B1[1][o] = bmy - a.hb * (dEx_dz1 - dEz_dx1);
                }
                if (wxy) {
                    const real dEy_dx1 = (fpyr - fpy) * a.ihx;
                    const real dEx_dy1 = (fpxu2 - fpx) * a.ihy;
                    a.B1[2][o] = bmz - a.hb * (dEy_dx1 - dEx_dy1);
                }
            }
        }
        oi0 = oi1;
        oh0 = oh1;
        oi1 = oi2;
        oh1 = oh2;
        emx = ex0;
        emy = ey0;
        ex0 = ex1;
        ey0 = ey1;
        ez0 = ez1;
        ex1 = nex;
        ey1 = ney;
        ez1 = nez;
        bx = nbx;
        by = nby;
        bz = nbz;
        jx = njx;
        jy = njy;
        jz = njz;
        bmx = hx;
        bmy = hy;
        bmz = hz;
        fpx = fx;
        fpy = fy;
        fpz = fz;
    }
}

// yee3d_body for a chunk whose planes k - 1 .. k + 2 all lie in the grid, as
// yee2d_inner
template <typename real>
__device__ __forceinline__ bool yee3d_inner(const YeeArgs<real> &a, real (*xs)[6][kCol3Warps][32], const int sx,
                                            const int sy, const int chunk)
{
    const Geom &g = a.g;
    const int z0 = chunk * a.cz, z1 = z0 + a.cz;
    if (z0 < 1 || z1 + 2 > g.nz - 1 || chunk == a.nchunks - 1 || g.ncomp * (int64_t)sizeof(real) >= (int64_t(1) << 32))
        return false;
    const unsigned lane = threadIdx.x & 31u;
    const int w = (int)(threadIdx.x >> 5);
    const int x = sx * kColOwn + (int)lane - 1, y = sy * kCol3Y + w - 1;
    const int gx = x >= 0 && x < g.nx ? x : wrapi(x, g.nx);
    const int gy = y >= 0 && y < g.ny ? y : wrapi(y, g.ny);
    const bool own = lane >= 1u && lane <= (unsigned)kColOwn && w >= 1 && w <= kCol3Y && x < g.nx && y < g.ny;
    const int du = w + 1 < kCol3Warps ? 32 : 0, dd = w >= 1 ? -32 : 0;  // rows above and below (halo: own)
    auto dn = [&](real v) { return __shfl_down_sync(0xffffffffu, v, 1); };  // x + 1
    auto up = [&](real v) { return __shfl_up_sync(0xffffffffu, v, 1); };    // x - 1
    auto ld = [](const real *p, unsigned b) {
        return *reinterpret_cast<const real *>(reinterpret_cast<const char *>(p) + b);
    };
    auto st = [](real *p, unsigned b, real v) { *reinterpret_cast<real *>(reinterpret_cast<char *>(p) + b) = v; };
    const unsigned dp = (unsigned)(g.plane * sizeof(real));
    unsigned o = (unsigned)(((int64_t)(z0 - 1) * g.plane + (int64_t)gy * g.nx + gx) * sizeof(real));  // plane k
    real ex0 = ld(a.E[0], o), ey0 = ld(a.E[1], o), ez0 = ld(a.E[2], o);
    real ex1 = ld(a.E[0], o + dp), ey1 = ld(a.E[1], o + dp), ez1 = ld(a.E[2], o + dp);
    real bx = ld(a.B[0], o), by = ld(a.B[1], o), bz = ld(a.B[2], o);
    real jx = 0, jy = 0, jz = 0;  // (E' of the first plane is not used)
    real bmx = 0, bmy = 0, bmz = 0, fpx = 0, fpy = 0, fpz = 0;
    // lane l < 18 prefetches a line of row l / 2 of Ex .. Jz
    const char *pf;
    {
        const int c = (int)(lane >> 1);
        const real *base = c == 0 ? a.E[0] : c == 1 ? a.E[1] : c == 2 ? a.E[2] : c == 3 ? a.B[0] : c == 4 ? a.B[1]
                         : c == 5 ? a.B[2] : c == 6 ? a.J[0] : c == 7 ? a.J[1] : a.J[2];
        const unsigned oa = __shfl_sync(0xffffffffu, o, 0), ob = __shfl_sync(0xffffffffu, o, 31);
        pf = reinterpret_cast<const char *>(base) + ((lane & 1u) ? ob : oa) + (kAhead + 1) * (size_t)dp;
    }
#pragma unroll 2
    for (int k = z0 - 1; k <= z1; ++k) {
        if (lane < 18u && k + kAhead <= z1) prefetch_l2(pf);
        pf += dp;
        real *s = &xs[k & 1][0][w][lane];
        constexpr int C = kCol3Warps * 32;  // one component of the exchange
        const real nex = ld(a.E[0], o + 2 * dp), ney = ld(a.E[1], o + 2 * dp), nez = ld(a.E[2], o + 2 * dp);
        const real nbx = ld(a.B[0], o + dp), nby = ld(a.B[1], o + dp), nbz = ld(a.B[2], o + dp);
        const real njx = ld(a.J[0], o + dp), njy = ld(a.J[1], o + dp), njz = ld(a.J[2], o + dp);
        // ---- exchange 1: E^n(k) and E'(k - 1) with the row above
        s[0 * C] = ex0;
        s[1 * C] = ez0;
        s[2 * C] = fpx;
        s[3 * C] = fpz;
        __syncthreads();
        const real exu = s[0 * C + du], ezu = s[1 * C + du], fpxu = s[2 * C + du], fpzu = s[3 * C + du];
        // ---- Bh(k)
        const real eyr = dn(ey0), ezr = dn(ez0);
        const real dEz_dy = (ezu - ez0) * a.ihy, dEx_dy = (exu - ex0) * a.ihy;
        const real dEy_dz = (ey1 - ey0) * a.ihz, dEx_dz = (ex1 - ex0) * a.ihz;
        const real dEz_dx = (ezr - ez0) * a.ihx, dEy_dx = (eyr - ey0) * a.ihx;
        const real hx = bx - a.hb * (dEz_dy - dEy_dz);
        const real hy = by - a.hb * (dEx_dz - dEz_dx);
        const real hz = bz - a.hb * (dEy_dx - dEx_dy);
        // ---- exchange 2: Bh(k) with the row below
        s[4 * C] = hx;
        s[5 * C] = hz;
        __syncthreads();
        const real hxd = s[4 * C + dd], hzd = s[5 * C + dd];
        // ---- E'(k)
        const real hyl = up(hy), hzl = up(hz);
        const real dBz_dy = (hz - hzd) * a.ihy, dBy_dz = (hy - bmy) * a.ihz;
        const real fx = ex0 + a.he * ((dBz_dy - dBy_dz) - a.twopi * jx);
        const real dBx_dz = (hx - bmx) * a.ihz, dBz_dx = (hz - hzl) * a.ihx;
        const real fy = ey0 + a.he * ((dBx_dz - dBz_dx) - a.twopi * jy);
        const real dBy_dx = (hy - hyl) * a.ihx, dBx_dy = (hx - hxd) * a.ihy;
        const real fz = ez0 + a.he * ((dBy_dx - dBx_dy) - a.twopi * jz);
        // ---- E'(k - 1), B'(k - 1) of the own columns
        const real fpyr = dn(fpy), fpzr = dn(fpz);
        if (k > z0 && own) {
            const unsigned ow = o - dp;
            st(a.E1[0], ow, fpx);
            st(a.E1[1], ow, fpy);
            st(a.E1[2], ow, fpz);
            const real dEz_dy1 = (fpzu - fpz) * a.ihy, dEy_dz1 = (fy - fpy) * a.ihz;
            st(a.B1[0], ow, bmx - a.hb * (dEz_dy1 - dEy_dz1));
            const real dEx_dz1 = (fx - fpx) * a.ihz, dEz_dx1 = (fpzr - fpz) * a.ihx;
            st(a.B1[1], ow, bmy - a.hb * (dEx_dz1 - dEz_dx1));
            const real dEy_dx1 = (fpyr - fpy) * a.ihx, dEx_dy1 = (fpxu - fpx) * a.ihy;
            st(a.B1[2], ow, bmz - a.hb * (dEy_dx1 - dEx_dy1));
        }
        o += dp;
        ex0 = ex1;
        ey0 = ey1;
        ez0 = ez1;
        ex1 = nex;
        ey1 = ney;
        ez1 = nez;
        bx = nbx;
        by = nby;
        bz = nbz;
        jx = njx;
        jy = njy;
        jz = njz;
        bmx = hx;
        bmy = hy;
        bmz = hz;
        fpx = fx;
        fpy = fy;
        fpz = fz;
    }
    return true;
}

template <typename real>
__device__ __forceinline__ void yee3d_item(const YeeArgs<real> &a, int64_t item)
{
    const int nsx = (a.g.nx + kColOwn - 1) / kColOwn, nsy = (a.g.ny + kCol3Y - 1) / kCol3Y;
    const int sx = (int)(item % nsx), sy = (int)((item / nsx) % nsy), ch = (int)(item / ((int64_t)nsx * nsy));
    __shared__ real xs[2][6][kCol3Warps][32];  // per parity: Ex, Ez, E'x, E'z of each row; Bh x, z
    if (!yee3d_inner(a, xs, sx, sy, ch)) yee3d_body(a, xs, sx, sy, ch);
}

template <typename real>
__global__ void __launch_bounds__(512, 2) yee3d_kernel(YeeArgs<real> a)
{
    chain_begin(a.g.early);
    yee3d_item(a, (int64_t)blockIdx.x);
}

template <typename real>
__global__ void __launch_bounds__(512, 2) yee3d_batch_kernel(const YeeArgs<real> *__restrict__ runs,
                                                             const int64_t *__restrict__ start, int n)
{
    __shared__ __align__(16) YeeArgs<real> sa;
    const int64_t b = batch_block(runs, start, n, &sa);
    yee3d_item(sa, b);
}

template <typename real>
static void launch_yee3d_batch(const void *args, const int64_t *start, int n, int64_t total, unsigned *,
                               cudaStream_t s)
{
    yee3d_batch_kernel<real><<<(unsigned)total, 512, 0, s>>>(static_cast<const YeeArgs<real> *>(args), start, n);
}

// one warp per (strip, chunk) item; YeeArgs::cz holds the planes per chunk,
// nchunks the chunks (the strips follow from the grid)
template <typename real>
__device__ __forceinline__ void yee2d_items(const YeeArgs<real> &a, int64_t item, int64_t nitems)
{
    if (item >= nitems) return;
    const int nstrip = (a.g.nx + kColOwn - 1) / kColOwn;
    const int strip = (int)(item % nstrip), chunk = (int)(item / nstrip);
    if (!yee2d_inner(a, strip, chunk)) yee2d_body(a, strip, chunk);
}

template <typename real>
__global__ void __launch_bounds__(256) yee2d_kernel(YeeArgs<real> a, int64_t nitems)
{
    chain_begin(a.g.early);
    yee2d_items(a, (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5), nitems);
}

template <typename real>
__global__ void __launch_bounds__(256) yee2d_batch_kernel(const YeeArgs<real> *__restrict__ runs,
                                                          const int64_t *__restrict__ start, int n)
{
    __shared__ __align__(16) YeeArgs<real> sa;
    const int64_t b = batch_block(runs, start, n, &sa);
    const int nstrip = (sa.g.nx + kColOwn - 1) / kColOwn;
    yee2d_items(sa, b * 8 + (threadIdx.x >> 5), (int64_t)nstrip * sa.nchunks);
}

template <typename real>
static void launch_yee2d_batch(const void *args, const int64_t *start, int n, int64_t total, unsigned *,
                               cudaStream_t s)
{
    yee2d_batch_kernel<real><<<(unsigned)total, 256, 0, s>>>(static_cast<const YeeArgs<real> *>(args), start, n);
}

template <typename real>
void launch_yee(const Geom &g, real *const F[9], real *const F1[6], double dt, double hx, double hy, double hz,
                cudaStream_t s)
{
    YeeArgs<real> a;
    a.g = g;
    for (int c = 0; c < 3; ++c) {
        a.E[c] = F[c];
        a.B[c] = F[3 + c];
        a.J[c] = F[6 + c];
        a.E1[c] = F1[c];
        a.B1[c] = F1[3 + c];
    }
    a.hb = (real)(0.5 * dt);
    a.he = (real)dt;
    a.ihx = (real)(1.0 / hx);
    a.ihy = (real)(1.0 / hy);
    a.ihz = (real)(1.0 / hz);
    a.twopi = (real)6.283185307179586;
    a.mur = (real)((dt - hz) / (dt + hz));
    const int nzo = g.bc_z == 0 ? g.nz : g.nz + 1;
    const bool is3 = g.dim == 3;
    if (!is3) {
        // chunks of 4..64 planes, as many as leave about 24 warps per SM
        const int nstrip = (g.nx + kColOwn - 1) / kColOwn;
        int64_t czl = (int64_t)nzo * nstrip * batch_runs() / ((int64_t)device_sms() * 24);
        a.cz = (int)(czl < 4 ? 4 : (czl > 64 ? 64 : czl));
        if (a.cz > nzo) a.cz = nzo;
        a.nchunks = (nzo + a.cz - 1) / a.cz;
        const int64_t nitems = (int64_t)nstrip * a.nchunks, nblocks = (nitems + 7) / 8;
        if (record_launch(kBPYee, launch_yee2d_batch<real>, a, nblocks)) return;
        launch_chained(yee2d_kernel<real>, (unsigned)nblocks, 256, 0, s, a, nitems);
        return;
    }
    {
        const int64_t ncol = (int64_t)((g.nx + kColOwn - 1) / kColOwn) * ((g.ny + kCol3Y - 1) / kCol3Y);
        a.cz = chunk_planes(nzo, ncol * batch_runs(), (int64_t)device_sms() * 2, 3, 4, kChunk3);
        a.nchunks = (nzo + a.cz - 1) / a.cz;
        const int64_t nblocks = ncol * a.nchunks;
        if (record_launch(kBPYee, launch_yee3d_batch<real>, a, nblocks)) return;
        launch_chained(yee3d_kernel<real>, (unsigned)nblocks, 512, 0, s, a);
    }
}

// ---------------------------------------------------------- moving window

// dst plane k = src plane k + S (zero for k + S > nz), nine components
template <typename real>
__global__ void window_fields_kernel(Geom g, Ptr9<real> src, Ptr9<real> dst, int S)
{
    const int64_t n = 9 * g.ncomp;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(q / g.ncomp);
        const int64_t o = q - c * g.ncomp;
        const int64_t k = o / g.plane;
        dst.p[c][o] = k + S <= g.nz ? src.p[c][o + S * g.plane] : real(0);
    }
}

template <typename real>
void launch_window_fields(const Geom &g, real *const src[9], real *const dst[9], int S, cudaStream_t s)
{
    Ptr9<real> a, b;
    for (int c = 0; c < 9; ++c) {
        a.p[c] = src[c];
        b.p[c] = dst[c];
    }
    window_fields_kernel<real><<<grid_for(9 * g.ncomp, 256), 256, 0, s>>>(g, a, b, S);
}

// ---------------------------------------------------------------- filter

// One (1/4, 1/2, 1/4) pass of Jx, Jy, Jz along `axis` from `in` to `out`.
// Periodic axes wrap; with absorbing z the values outside a component's valid
// z range are zero (and the unused plane nz of Jz stays zero).
template <typename real>
__global__ void filter_kernel(Geom g, const real *in0, const real *in1, const real *in2, real *out0,
                              real *out1, real *out2, int axis)
{
    const int64_t n = g.ncomp;
    for (int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; o < 3 * n; o += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(o / n);
        const int64_t r = o - c * n;
        const real *in = c == 0 ? in0 : (c == 1 ? in1 : in2);
        real *out = c == 0 ? out0 : (c == 1 ? out1 : out2);
        const int i = (int)(r % g.nx);
        const int j = (int)((r / g.nx) % g.ny);
        const int k = (int)(r / g.plane);
        const int zmax = zmax_of(g, c == 2);
        if (k > zmax) {
            out[r] = 0;
            continue;
        }
        real lo, hi;
        if (axis == 0) {
            lo = in[fidx(g, i == 0 ? g.nx - 1 : i - 1, j, k)];
            hi = in[fidx(g, i + 1 == g.nx ? 0 : i + 1, j, k)];
        } else if (axis == 1) {
            lo = in[fidx(g, i, j == 0 ? g.ny - 1 : j - 1, k)];
            hi = in[fidx(g, i, j + 1 == g.ny ? 0 : j + 1, k)];
        } else if (g.bc_z == 0) {
            lo = in[fidx(g, i, j, k == 0 ? g.nz - 1 : k - 1)];
            hi = in[fidx(g, i, j, k + 1 == g.nz ? 0 : k + 1)];
        } else {
            lo = k > 0 ? in[fidx(g, i, j, k - 1)] : real(0);
            hi = k < zmax ? in[fidx(g, i, j, k + 1)] : real(0);
        }
        out[r] = real(0.25) * lo + real(0.5) * in[r] + real(0.25) * hi;
    }
}

template <typename real>
struct MarchArgs {
    Geom g;
    const real *in;
    real *out;
    int cz, nchunks;
};

// --------------------------------------- binomial passes, column march
//
// All H passes (H <= 4) along all axes in one march up z with the planes in
// registers.  A pass (1/4, 1/2, 1/4) is a sum with the neighbour on one side
// and then on the other, (v_i + v_i-1) + (v_i+1 + v_i): two adds, and one
// exact scaling by a power of two ends all of them (until then the sums grow
// by 2^(2H) per axis: FP32 currents beyond 2^(128 - 6H), 2e31 in 3D with four
// passes, leave the range).  Along x the neighbours
// are the lanes next door (shuffles: lane l holds column x0 + l - H, wrapped;
// lanes H .. 31 - H own theirs).  Along z a pass keeps two registers of the
// planes below and gives its result one plane late; with absorbing z a
// pass's result outside the component's valid planes is zero (k is uniform,
// so that is a uniform test, and none in a chunk inside the grid).  A plane's
// loads are issued an iteration ahead of their use.
//
// 2D, FP32: 64 x 512 cells (H = 1) 9.0 -> 3.7 us, 256 x 8192 (H = 2) 27.4 ->
// 19.5 us, 512 x 2048 (H = 4) 38 -> 25 us against a march that kept every
// pass's three planes and tested every node.  3D, against planes staged by TMA
// in a ring of shared buffers with a stencil of width 2H + 1 per axis: 75 x 52
// x 99 (H = 1) 24.5 -> 6.9 us, 128 x 128 x 256 (H = 2) 77 -> 40 us, 256 x 256 x
// 512 349 -> 268 us (bound by issue slots: 3.0 TB/s of its 24 bytes a node,
// which at the copy rate take 120 us).

// one chunk of planes of the march: walks k from z0 - H to z1 - 1 + H
template <typename real>
struct FilterWalk {
    bool per;
    int zmax_xy, zmax_z, nz;
    int64_t plane, off;  // offset of plane kk (wrapped)
    int kk;
    __device__ __forceinline__ FilterWalk(const Geom &g, int k)
        : per(g.bc_z == 0), zmax_xy(zmax_of(g, false)), zmax_z(zmax_of(g, true)), nz(g.nz), plane(g.plane),
          kk(g.bc_z == 0 ? wrapi(k, g.nz) : k)
    {
        off = (int64_t)kk * plane;
    }
    __device__ __forceinline__ void next()
    {
        ++kk;
        off += plane;
        if (per && kk == nz) {
            kk = 0;
            off = 0;
        }
    }
    // is plane k of component c (0, 1 on integer z, 2 on half-integer z) in the grid?
    __device__ __forceinline__ bool valid(int c, int k) const
    {
        return per || (k >= 0 && k <= (c == 2 ? zmax_z : zmax_xy));
    }
};

template <typename real, int H>
__device__ __forceinline__ real filter_x(real v)
{
#pragma unroll
    for (int p = 0; p < H; ++p) {
        v += __shfl_up_sync(0xffffffffu, v, 1);
        v += __shfl_down_sync(0xffffffffu, v, 1);
    }
    return v;
}

// the z passes of a value of plane k: the result belongs to plane k - H
template <typename real, int H, bool INNER>
__device__ __forceinline__ real filter_z(real v, real pa[H], real pb[H], const FilterWalk<real> &w, int c, int k)
{
#pragma unroll
    for (int p = 0; p < H; ++p) {
        const real u = v + pa[p];
        pa[p] = v;
        v = u + pb[p];
        pb[p] = u;
        if (!INNER && !w.valid(c, k - 1 - p)) v = real(0);
    }
    return v;
}

// an element at a 32-bit byte offset from a uniform base: one add per plane
// addresses all components (an inner march; the grid's components are below
// 4 GB each, or every chunk takes the general march)
template <typename real> __device__ __forceinline__ const real &elem(const real *p, unsigned b)
{
    return *reinterpret_cast<const real *>(reinterpret_cast<const char *>(p) + b);
}
template <typename real> __device__ __forceinline__ real &elem(real *p, unsigned b)
{
    return *reinterpret_cast<real *>(reinterpret_cast<char *>(p) + b);
}
template <typename real> __device__ __forceinline__ bool small_offsets(const Geom &g)
{
    return g.ncomp * (int64_t)sizeof(real) < (int64_t(1) << 32);
}

template <typename real, int H, bool INNER>
__device__ __forceinline__ void filter2d_march(const Geom &g, const real *in, real *out, const int strip, const int z0,
                                               const int z1)
{
    const int lane = (int)(threadIdx.x & 31u);
    const int x = strip * (32 - 2 * H) + lane - H;
    const int gx = x >= 0 && x < g.nx ? x : wrapi(x, g.nx);
    const bool own = lane >= H && lane < 32 - H && x < g.nx;
    const real scale = real(1.0 / (double)(1 << (4 * H)));
    FilterWalk<real> w(g, z0 - H);
    const unsigned dp = (unsigned)(g.plane * sizeof(real));
    unsigned b = (unsigned)((w.off + gx) * (int64_t)sizeof(real));  // of plane k (INNER)
    auto ld = [&](int c, int k) {
        if (INNER) return elem(in + c * g.ncomp, b);
        return w.valid(c, k) ? in[c * g.ncomp + w.off + gx] : real(0);
    };
    real pa[3][H], pb[3][H], cur[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        cur[c] = ld(c, z0 - H);
#pragma unroll
        for (int p = 0; p < H; ++p) pa[c][p] = pb[c][p] = real(0);
    }
    // lane l < 6 prefetches a line of component l / 2's row
    const int cl = __shfl_sync(0xffffffffu, gx, (lane & 1) ? 31 : 0);
    const real *pf = in + (lane >> 1) * g.ncomp + w.off + (kAhead + 1) * g.plane + cl;
    int64_t o = (int64_t)(z0 - 2 * H) * g.plane + x;  // plane k - H
#pragma unroll 2
    for (int k = z0 - H; k < z1 + H; ++k) {
        if (INNER && lane < 6 && k + kAhead + 1 < z1 + H) prefetch_l2(pf);
        pf += g.plane;
        const unsigned bo = b - H * dp;  // plane k - H (x = gx on the own lanes)
        b += dp;
        if (!INNER) w.next();
        real nxt[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) nxt[c] = ld(c, k + 1);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const real v = filter_z<real, H, INNER>(filter_x<real, H>(cur[c]), pa[c], pb[c], w, c, k);
            if (own && k >= z0 + H) {
                if (INNER) elem(out + c * g.ncomp, bo) = v * scale;
                else out[c * g.ncomp + o] = k - H > (c == 2 ? w.zmax_z : w.zmax_xy) ? real(0) : v * scale;
            }
            cur[c] = nxt[c];
        }
        o += g.plane;
    }
}

// a warp's strip of 32 - 2H columns and chunk of planes (2D); the plane after
// the last one it needs is loaded too, so an inner chunk ends a plane early
template <typename real, int H>
__device__ __forceinline__ void filter2d_body(const Geom &g, const real *in, real *out, const int strip,
                                              const int chunk, const int cz, const int nchunks)
{
    const int z0 = chunk * cz, z1 = chunk == nchunks - 1 ? g.nz + 1 : z0 + cz;
    if (z0 >= H && z1 + H <= g.nz - 1 && small_offsets<real>(g)) filter2d_march<real, H, true>(g, in, out, strip, z0, z1);
    else filter2d_march<real, H, false>(g, in, out, strip, z0, z1);
}

// In 3D a CTA holds rows of 32 columns, two rows a warp: the x passes are done
// for every row and the rows pass through shared memory (one barrier per
// plane, two buffers in turn), where a warp takes the H rows on either side of
// its own two for the y passes.  Only columns H .. 31 - H and rows H .. rows -
// 1 - H are the CTA's own (FP32, H = 2: 28^2 of 32^2).  Where the adds bound
// it (FP64, and FP32 with H = 4; kFilterLean) the y passes of a row are the
// binomial stencil of 2H + 1 rows, 2H adds and fused multiply-adds where
// passes as sums take 2H^2 + 3H for two rows, and warps without an own row in
// the grid leave out the y and z passes.  (In FP32 with H <= 3 the tests cost
// more than they save: 200^3 cells, H = 2 116 us without, 123 with.)  FP64
// takes 8 warps (16 rows): its pipe is full with one CTA per SM, and a grid of
// 40^3 cells is 4 columns of 32 rows but 8 to 20 of 16.  FP64, us, sums over
// 32 rows / this: 40^3 cells H = 1 66 / 40, H = 4 436 / 115; 100^3 H = 2 250 /
// 176; 200^3 H = 4 5177 / 3306, H = 1 550 / 559.  FP32, H = 4: 200^3 239 / 213.
template <typename real> constexpr int kFilterWarps = sizeof(real) == 4 ? 16 : 8;
// resident CTAs per SM that the kernels are compiled for
template <typename real, int H> constexpr int kFilterBlocks = H <= 2 ? 2 : 1;
template <typename real, int H> constexpr bool kFilterLean = sizeof(real) == 8 || H == 4;
// the binomial coefficient C(2H, i)
template <int H> __device__ __forceinline__ constexpr int binomial(int i)
{
    int c = 1;
    for (int q = 0; q < i; ++q) c = c * (2 * H - q) / (q + 1);
    return c;
}
template <typename real, int H, bool INNER>
__device__ __forceinline__ void filter3d_march(const Geom &g, const real *in, real *out, real *xs, const int sx,
                                               const int sy, const int z0, const int z1)
{
    // rows of a component in shared memory: H more on either side of the
    // CTA's, never written (only rows the CTA does not own would take them)
    constexpr int ROWS = 2 * kFilterWarps<real>, OWNX = 32 - 2 * H, OWNY = ROWS - 2 * H, CS = (ROWS + 2 * H) * 32;
    const int lane = (int)(threadIdx.x & 31u), r0 = 2 * (int)(threadIdx.x >> 5);
    const int x = sx * OWNX + lane - H, y = sy * OWNY + r0 - H;
    const int gx = x >= 0 && x < g.nx ? x : wrapi(x, g.nx);
    const bool ownx = lane >= H && lane < 32 - H && x < g.nx;
    int64_t col[2];
    bool own[2], row[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int yy = y + j, gy = yy >= 0 && yy < g.ny ? yy : wrapi(yy, g.ny);
        col[j] = (int64_t)gy * g.nx + gx;
        row[j] = r0 + j >= H && r0 + j < ROWS - H && yy < g.ny;
        own[j] = ownx && row[j];
    }
    // (uniform over the warp)
    const bool used = !kFilterLean<real, H> || y < g.ny + H, mine = !kFilterLean<real, H> || row[0] || row[1];
    const real scale = real(1.0 / (double)(1 << (6 * H)));
    FilterWalk<real> w(g, z0 - H);
    const unsigned dp = (unsigned)(g.plane * sizeof(real));
    unsigned b[2] = {(unsigned)((w.off + col[0]) * (int64_t)sizeof(real)),
                     (unsigned)((w.off + col[1]) * (int64_t)sizeof(real))};  // of plane k (INNER)
    auto ld = [&](int c, int j, int k) {
        if (INNER) return elem(in + c * g.ncomp, b[j]);
        return w.valid(c, k) ? in[c * g.ncomp + w.off + col[j]] : real(0);
    };
    real pa[3][2][H], pb[3][2][H], cur[3][2];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            cur[c][j] = used ? ld(c, j, z0 - H) : real(0);
#pragma unroll
            for (int p = 0; p < H; ++p) pa[c][j][p] = pb[c][j][p] = real(0);
        }
    real *at = xs + (r0 + H) * 32 + lane;  // [buffer][component][row][lane]
    // lane l < 12 prefetches a line of component l / 4's row r0 + (l / 2) % 2
    const int64_t ca = __shfl_sync(0xffffffffu, col[0], (lane & 1) ? 31 : 0),
                  cb = __shfl_sync(0xffffffffu, col[1], (lane & 1) ? 31 : 0);
    const real *pf = in + (lane >> 2) * g.ncomp + w.off + (kAhead + 1) * g.plane + ((lane & 2) ? cb : ca);
    int64_t o = (int64_t)(z0 - 2 * H) * g.plane;  // plane k - H
    for (int k = z0 - H; k < z1 + H; ++k) {
        if (INNER && used && lane < 12 && k + kAhead + 1 < z1 + H) prefetch_l2(pf);
        pf += g.plane;
        const unsigned bo[2] = {b[0] - H * dp, b[1] - H * dp};  // plane k - H
        b[0] += dp;
        b[1] += dp;
        if (!INNER) w.next();
        real *buf = at + (k & 1) * 3 * CS;
        real nxt[3][2];
        if (used) {
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
                for (int j = 0; j < 2; ++j) nxt[c][j] = ld(c, j, k + 1);
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    cur[c][j] = filter_x<real, H>(cur[c][j]);
                    buf[c * CS + j * 32] = cur[c][j];
                }
        }
        __syncthreads();
        if (mine) {
            const bool w0 = own[0] && k >= z0 + H, w1 = own[1] && k >= z0 + H;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                real v[2 * H + 2];  // rows r0 - H .. r0 + 1 + H
#pragma unroll
                for (int q = 0; q < 2 * H + 2; ++q) {
                    const int d = q - H;
                    v[q] = d == 0 || d == 1 ? cur[c][d & 1] : buf[c * CS + d * 32];
                }
                if (!kFilterLean<real, H>) {
#pragma unroll
                    for (int p = 0; p < 2 * H; ++p)
#pragma unroll
                        for (int q = 0; q < 2 * H + 1 - p; ++q) v[q] = v[q] + v[q + 1];
                }
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    real t = v[j];
                    if (kFilterLean<real, H>) {
                        t += v[j + 2 * H];
#pragma unroll
                        for (int q = 1; q < H; ++q) t += real(binomial<H>(q)) * (v[j + q] + v[j + 2 * H - q]);
                        t += real(binomial<H>(H)) * v[j + H];
                    }
                    t = filter_z<real, H, INNER>(t, pa[c][j], pb[c][j], w, c, k);
                    if (j == 0 ? w0 : w1) {
                        if (INNER) elem(out + c * g.ncomp, bo[j]) = t * scale;
                        else out[c * g.ncomp + o + col[j]] = k - H > (c == 2 ? w.zmax_z : w.zmax_xy) ? real(0) : t * scale;
                    }
                }
            }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int j = 0; j < 2; ++j) cur[c][j] = nxt[c][j];
        o += g.plane;
    }
}

template <typename real, int H>
__device__ __forceinline__ void filter3d_item(const Geom &g, const real *in, real *out, int cz, int nchunks,
                                              int64_t item)
{
    constexpr int ROWS = 2 * kFilterWarps<real>, OWNX = 32 - 2 * H, OWNY = ROWS - 2 * H;
    __shared__ real xs[2 * 3 * (ROWS + 2 * H) * 32];
    const int nsx = (g.nx + OWNX - 1) / OWNX, nsy = (g.ny + OWNY - 1) / OWNY;
    const int sx = (int)(item % nsx), sy = (int)((item / nsx) % nsy), ch = (int)(item / ((int64_t)nsx * nsy));
    const int z0 = ch * cz, z1 = ch == nchunks - 1 ? g.nz + 1 : z0 + cz;
    if (z0 >= H && z1 + H <= g.nz - 1 && small_offsets<real>(g)) filter3d_march<real, H, true>(g, in, out, xs, sx, sy, z0, z1);
    else filter3d_march<real, H, false>(g, in, out, xs, sx, sy, z0, z1);
}

template <typename real, int H>
__global__ void __launch_bounds__((32 * kFilterWarps<real>), (kFilterBlocks<real, H>))
    filter3d_kernel(Geom g, const real *in, real *out, int cz, int nchunks)
{
    chain_begin(g.early);
    filter3d_item<real, H>(g, in, out, cz, nchunks, (int64_t)blockIdx.x);
}

template <typename real, int H>
__global__ void __launch_bounds__((32 * kFilterWarps<real>), (kFilterBlocks<real, H>))
    filter3d_batch_kernel(const MarchArgs<real> *__restrict__ runs, const int64_t *__restrict__ start, int n)
{
    __shared__ __align__(16) MarchArgs<real> sa;
    const int64_t b = batch_block(runs, start, n, &sa);
    filter3d_item<real, H>(sa.g, sa.in, sa.out, sa.cz, sa.nchunks, b);
}

template <typename real, int H>
static void launch_filter3d_batch(const void *args, const int64_t *start, int n, int64_t total, unsigned *,
                                  cudaStream_t s)
{
    filter3d_batch_kernel<real, H>
        <<<(unsigned)total, 32 * kFilterWarps<real>, 0, s>>>(static_cast<const MarchArgs<real> *>(args), start, n);
}

// one warp per (strip, chunk) item; in FP64 two warps a CTA, so that few items
// share no SM's FP64 pipe while others idle
template <typename real> constexpr int kFilter2Warps = sizeof(real) == 4 ? 8 : 2;
// (FP64) warps that fill an SM's FP64 pipe; us, 4 / 8: 1000 x 1000 cells (H =
// 1) 78 / 62, 256 x 8192 (H = 4) 374 / 549, else within 15%
template <int H> constexpr int kFilter2Resident = H <= 3 ? 8 : 4;
template <typename real, int H>
__device__ __forceinline__ void filter2d_items(const Geom &g, const real *in, real *out, int cz, int nchunks,
                                               int64_t item)
{
    const int nstrip = (g.nx + (32 - 2 * H) - 1) / (32 - 2 * H);
    if (item >= (int64_t)nstrip * nchunks) return;
    filter2d_body<real, H>(g, in, out, (int)(item % nstrip), (int)(item / nstrip), cz, nchunks);
}

template <typename real, int H>
__global__ void __launch_bounds__((32 * kFilter2Warps<real>))
    filter2d_kernel(Geom g, const real *in, real *out, int cz, int nchunks)
{
    chain_begin(g.early);
    filter2d_items<real, H>(g, in, out, cz, nchunks, (int64_t)blockIdx.x * kFilter2Warps<real> + (threadIdx.x >> 5));
}

template <typename real, int H>
__global__ void __launch_bounds__((32 * kFilter2Warps<real>))
    filter2d_batch_kernel(const MarchArgs<real> *__restrict__ runs, const int64_t *__restrict__ start, int n)
{
    __shared__ __align__(16) MarchArgs<real> sa;
    const int64_t b = batch_block(runs, start, n, &sa);
    filter2d_items<real, H>(sa.g, sa.in, sa.out, sa.cz, sa.nchunks, b * kFilter2Warps<real> + (threadIdx.x >> 5));
}

template <typename real, int H>
static void launch_filter2d_batch(const void *args, const int64_t *start, int n, int64_t total, unsigned *,
                                  cudaStream_t s)
{
    filter2d_batch_kernel<real, H>
        <<<(unsigned)total, 32 * kFilter2Warps<real>, 0, s>>>(static_cast<const MarchArgs<real> *>(args), start, n);
}

template <typename real, int DIM, int H>
static void launch_march(const Geom &g, const real *in, real *out, cudaStream_t s)
{
    const int nzo = g.nz + 1;
    if constexpr (DIM == 2) {
        // FP32: chunks of 4..64 planes, as many as leave about 24 warps per SM.
        // FP64: the FP64 pipe of an SM is full with a few warps, beyond which
        // shorter chunks only repeat their halos.
        constexpr int OWN = 32 - 2 * H, NW = kFilter2Warps<real>;
        const int nstrip = (g.nx + OWN - 1) / OWN;
        int cz;
        if (sizeof(real) == 4) {
            const int64_t czl = (int64_t)nzo * nstrip * batch_runs() / ((int64_t)device_sms() * 24);
            cz = (int)(czl < 4 ? 4 : (czl > 64 ? 64 : czl));
        } else {
            cz = chunk_planes(nzo, (int64_t)nstrip * batch_runs(), (int64_t)device_sms() * kFilter2Resident<H>, 2 * H, 4, 64);
        }
        if (cz > nzo) cz = nzo;
        const int nchunks = (nzo + cz - 1) / cz;
        const int64_t nblocks = ((int64_t)nstrip * nchunks + NW - 1) / NW;
        if (record_launch(kBPFilter, launch_filter2d_batch<real, H>, MarchArgs<real>{g, in, out, cz, nchunks},
                          nblocks))
            return;
        launch_chained(filter2d_kernel<real, H>, (unsigned)nblocks, 32 * NW, 0, s, g, in, out, cz, nchunks);
    } else {
        // (FP64: waves of one CTA per SM, whose FP64 pipe it fills)
        constexpr int OWNX = 32 - 2 * H, OWNY = 2 * kFilterWarps<real> - 2 * H;
        const int64_t ncol = (int64_t)((g.nx + OWNX - 1) / OWNX) * ((g.ny + OWNY - 1) / OWNY);
        const int cz = chunk_planes(nzo, ncol * batch_runs(),
                                    (int64_t)device_sms() * (sizeof(real) == 4 ? kFilterBlocks<real, H> : 1), 2 * H, 4, kChunk3);
        const int nchunks = (nzo + cz - 1) / cz;
        const int64_t nblocks = ncol * nchunks;
        if (record_launch(kBPFilter, launch_filter3d_batch<real, H>, MarchArgs<real>{g, in, out, cz, nchunks},
                          nblocks))
            return;
        launch_chained(filter3d_kernel<real, H>, (unsigned)nblocks, 32 * kFilterWarps<real>, 0, s, g, in, out, cz, nchunks);
    }
}

template <typename real>
static bool fused_passes(const Geom &g, const real *in, real *out, int npass, cudaStream_t s)
{
    if (npass < 1 || npass > 4) return false;
    if (g.dim == 3) {
        switch (npass) {
        case 1: launch_march<real, 3, 1>(g, in, out, s); break;
        case 2: launch_march<real, 3, 2>(g, in, out, s); break;
        case 3: launch_march<real, 3, 3>(g, in, out, s); break;
        default: launch_march<real, 3, 4>(g, in, out, s); break;
        }
    } else {
        switch (npass) {
        case 1: launch_march<real, 2, 1>(g, in, out, s); break;
        case 2: launch_march<real, 2, 2>(g, in, out, s); break;
        case 3: launch_march<real, 2, 3>(g, in, out, s); break;
        default: launch_march<real, 2, 4>(g, in, out, s); break;
        }
    }
    return true;
}

template <typename real>
bool launch_filter_from(const Geom &g, const real *src, real *const J[3], int npass, cudaStream_t s)
{
    const bool contiguous = J[1] == J[0] + g.ncomp && J[2] == J[1] + g.ncomp;
    return contiguous && fused_passes<real>(g, src, J[0], npass, s);
}

template <typename real>
void launch_filter(const Geom &g, real *const J[3], real *tmp, int npass, cudaStream_t s)
{
    if (npass <= 0) return;
    // the three components are contiguous in the field buffer; the fused
    // kernel covers 1..4 passes, more fall back to one launch per pass
    if (record_unsupported()) return;  // (a copy back, or one launch per pass)
    const bool contiguous = J[1] == J[0] + g.ncomp && J[2] == J[1] + g.ncomp;
    if (contiguous && fused_passes<real>(g, J[0], tmp, npass, s)) {
        cudaMemcpyAsync(J[0], tmp, 3 * sizeof(real) * g.ncomp, cudaMemcpyDeviceToDevice, s);
        return;
    }
    real *src[3] = {J[0], J[1], J[2]};
    real *dst[3] = {tmp, tmp + g.ncomp, tmp + 2 * g.ncomp};
    const unsigned grid = grid_for(3 * g.ncomp, 256);
    int passes = 0;
    for (int axis = 0; axis < 3; ++axis) {
        if (axis == 1 && g.dim != 3) continue;
        for (int p = 0; p < npass; ++p) {
            filter_kernel<real><<<grid, 256, 0, s>>>(g, src[0], src[1], src[2], dst[0], dst[1], dst[2], axis);
            for (int c = 0; c < 3; ++c) {
                real *t = src[c];
                src[c] = dst[c];
                dst[c] = t;
            }
            ++passes;
        }
    }
    if (passes & 1)
        for (int c = 0; c < 3; ++c)
            cudaMemcpyAsync(J[c], src[c], sizeof(real) * g.ncomp, cudaMemcpyDeviceToDevice, s);
}

// ---------------------------------------------------------------- antenna

// Current sheet on plane ka: J_pol += j0 exp(-r^2 / w0^2) at each node of the
// polarisation component (its own staggered transverse position).  One plane
// per step: the profile is evaluated in FP64 and rounded once.
template <typename real>
struct AntennaArgs {
    Geom g;
    real *J;
    int pol, ka;
    double j0, hx, hy, xc, yc, inv_w2;
    const double *j0p;
};

template <typename real>
__device__ __forceinline__ void antenna_body(const AntennaArgs<real> &a, int64_t b, int64_t nb)
{
    const Geom &g = a.g;
    const double j0 = a.j0p ? *a.j0p : a.j0;
    const int64_t n = g.plane;
    for (int64_t o = b * blockDim.x + threadIdx.x; o < n; o += nb * blockDim.x) {
        const int i = (int)(o % g.nx), j = (int)(o / g.nx);
        const double x = ((double)i + (a.pol == 0 ? 0.5 : 0.0)) * a.hx - a.xc;
        double r2 = x * x;
        if (g.dim == 3) {
            const double y = ((double)j + (a.pol == 1 ? 0.5 : 0.0)) * a.hy - a.yc;
            r2 += y * y;
        }
        a.J[(int64_t)a.ka * g.plane + o] += (real)(j0 * exp(-r2 * a.inv_w2));
    }
}

template <typename real>
__global__ void antenna_kernel(AntennaArgs<real> a)
{
    chain_begin(a.g.early);
    antenna_body(a, (int64_t)blockIdx.x, (int64_t)gridDim.x);
}

template <typename real>
__global__ void antenna_batch_kernel(const AntennaArgs<real> *__restrict__ runs, const int64_t *__restrict__ start,
                                     int n)
{
    __shared__ __align__(16) AntennaArgs<real> sa;
    const int64_t b = batch_block(runs, start, n, &sa);
    const int r = batch_run_of(start, n, (int64_t)blockIdx.x);
    antenna_body(sa, b, start[r + 1] - start[r]);
}

template <typename real>
static void launch_antenna_batch(const void *args, const int64_t *start, int n, int64_t total, unsigned *,
                                 cudaStream_t s)
{
    antenna_batch_kernel<real><<<(unsigned)total, 256, 0, s>>>(static_cast<const AntennaArgs<real> *>(args), start, n);
}

template <typename real>
void launch_antenna(const Geom &g, real *J, int pol, int ka, double j0, double hx, double hy, double xc,
                    double yc, double waist, cudaStream_t s, const double *j0p)
{
    const AntennaArgs<real> a{g, J, pol, ka, j0, hx, hy, xc, yc, 1.0 / (waist * waist), j0p};
    const unsigned nb = grid_for(g.plane, 256);
    if (record_launch(kBPAntenna, launch_antenna_batch<real>, a, (int64_t)nb)) return;
    launch_chained(antenna_kernel<real>, (unsigned)nb, 256, 0, s, a);
}

// ---------------------------------------------------------------- zeroing

// blocks of kZeroChunk elements; the batched form zeroes every run's buffer
constexpr int kZeroChunk = 8192;

template <typename real>
__global__ void __launch_bounds__(256) zero_batch_kernel(const ZeroArgs<real> *__restrict__ runs,
                                                         const int64_t *__restrict__ start, int n)
{
    __shared__ __align__(16) ZeroArgs<real> sa;
    const int64_t b = batch_block(runs, start, n, &sa);
    const int64_t lo = b * kZeroChunk;
    const int64_t hi = lo + kZeroChunk < sa.n ? lo + kZeroChunk : sa.n;
    for (int64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) sa.p[i] = real(0);
}

template <typename real>
static void launch_zero_batch(const void *args, const int64_t *start, int n, int64_t total, unsigned *, cudaStream_t s)
{
    zero_batch_kernel<real><<<(unsigned)total, 256, 0, s>>>(static_cast<const ZeroArgs<real> *>(args), start, n);
}

// n values at p (16-byte aligned) and m bytes at q
template <typename real>
__global__ void __launch_bounds__(256) zero_kernel(real *p, int64_t n, unsigned char *q, int64_t m, int early)
{
    chain_begin(early);
    const int64_t first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    constexpr int V = 16 / (int)sizeof(real);
    for (int64_t o = first; o < n / V; o += stride) reinterpret_cast<int4 *>(p)[o] = make_int4(0, 0, 0, 0);
    for (int64_t o = n / V * V + first; o < n; o += stride) p[o] = real(0);
    for (int64_t o = first; o < m; o += stride) q[o] = 0;
}

// Values that zero_kernel takes, at most.  On small arrays it saves the gap
// that a memset makes between two kernels (3D 16 x 16 x 32 cells 65 -> 62 us a
// step); on large ones the two are alike (12.6M values 1056 us a step with the
// kernel, 1059 with the memset; 100M values 6827 and 6826).
constexpr int64_t kZeroKernelMax = 9 << 20;

// returns the kernels it launches
template <typename real>
static int zero_launch(real *p, int64_t n, unsigned char *q, int64_t m, int early, cudaStream_t s)
{
    // a large array, or one off the 16-byte grid (J of an odd grid, zeroed
    // by itself): a plain memset
    if (n > kZeroKernelMax || reinterpret_cast<uintptr_t>(p) % 16 != 0) {
        cudaMemsetAsync(p, 0, (size_t)n * sizeof(real), s);
        n = 0;
        if (m == 0) return 0;
    }
    launch_chained(zero_kernel<real>, grid_for(n / 4 + 1, 256), 256, 0, s, p, n, q, m, early);
    return 1;
}

template <typename real>
int launch_zero(real *p, int64_t n, cudaStream_t s)
{
    if (n <= 0) return 0;
    if (record_launch(kBPZero, launch_zero_batch<real>, ZeroArgs<real>{p, n}, (n + kZeroChunk - 1) / kZeroChunk))
        return 1;
    return zero_launch(p, n, nullptr, 0, 0, s);
}

template <typename real>
void launch_zero2(real *p, int64_t n, unsigned char *q, int64_t m, int early, cudaStream_t s)
{
    zero_launch(p, n, q, m, early, s);
}

// ------------------------------------------------------------ field sums

// Compensated FP64 partials of sum (E^2 + B^2) over the valid nodes of each
// component (its first zmax + 1 planes: one contiguous piece); the host
// multiplies by V/2 and adds the partials.  Every block takes one component.
// The squares are summed exactly in FP32 words (RunSum), eight loads in
// flight per thread: an FP64 Kahan sum of every value and two divisions for
// its place took 148 us on 256 x 8192 cells, where the 50 MB take 8.
template <typename real>
__global__ void field_sums_kernel(Geom g, const real *F0, const real *F1, const real *F2, const real *F3,
                                  const real *F4, const real *F5, double *partials)
{
    RunSum<real> sum;
    constexpr int U = 8;
    static_assert(kSumRun % U == 0, "whole groups of loads between flushes");
    const int comp = (int)(blockIdx.x % 6u);
    const int64_t blocks = (gridDim.x - comp + 5) / 6;  // that take this component
    const int64_t stride = blocks * blockDim.x, first = (int64_t)(blockIdx.x / 6) * blockDim.x + threadIdx.x;
    const real *F = comp == 0 ? F0 : comp == 1 ? F1 : comp == 2 ? F2 : comp == 3 ? F3 : comp == 4 ? F4 : F5;
    const int64_t n = (int64_t)(zmax_of(g, comp >= 2 && comp <= 4) + 1) * g.plane;
    int64_t o = first;
    int run = 0;
    for (; o + (U - 1) * stride < n; o += U * stride) {
        real v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = F[o + u * stride];
#pragma unroll
        for (int u = 0; u < U; ++u) sum.add_square(v[u]);
        run += U;
        if (run == kSumRun) {
            sum.flush();
            run = 0;
        }
    }
    if (run) sum.flush();
    for (; o < n; o += stride) sum.add_square(F[o]);
    sum.flush();
    __shared__ double red[256];
    red[threadIdx.x] = sum.k.value();
    __syncthreads();
    for (int off = blockDim.x / 2; off > 0; off >>= 1) {
        if ((int)threadIdx.x < off) red[threadIdx.x] += red[threadIdx.x + off];
        __syncthreads();
    }
    if (threadIdx.x == 0) partials[blockIdx.x] = red[0];
}

// returns the blocks whose partials it writes
template <typename real>
int launch_field_sums(const Geom &g, real *const F[9], double *partials, int max_blocks, cudaStream_t s)
{
    // about 16 values per thread, at least one block per component
    int64_t n = 6 * (g.ncomp / (256 * 16) + 1);
    const int nblocks = (int)(n < max_blocks ? n : max_blocks);
    field_sums_kernel<real><<<nblocks, 256, 0, s>>>(g, F[0], F[1], F[2], F[3], F[4], F[5], partials);
    return nblocks;
}

#define PIC_FIELDS_INSTANTIATE(real)                                                                    \
    template void launch_yee<real>(const Geom &, real *const[9], real *const[6], double, double, double, \
                                   double, cudaStream_t);                                               \
    template void launch_filter<real>(const Geom &, real *const[3], real *, int, cudaStream_t);          \
    template bool launch_filter_from<real>(const Geom &, const real *, real *const[3], int, cudaStream_t); \
    template void launch_window_fields<real>(const Geom &, real *const[9], real *const[9], int, cudaStream_t); \
    template void launch_antenna<real>(const Geom &, real *, int, int, double, double, double, double,  \
                                       double, double, cudaStream_t, const double *);                   \
    template int launch_field_sums<real>(const Geom &, real *const[9], double *, int, cudaStream_t); \
    template int launch_zero<real>(real *, int64_t, cudaStream_t);                                      \
    template void launch_zero2<real>(real *, int64_t, unsigned char *, int64_t, int, cudaStream_t);
PIC_FIELDS_INSTANTIATE(float)
PIC_FIELDS_INSTANTIATE(double)

// ------------------------------------------------ bounded-wait self-check

// The wait on an mbarrier that callers can check on their device: it never
// spins without a limit, but polls up to a time budget (globaltimer,
// nanoseconds) and reports failure.  No kernel of a step waits on one.
namespace {
__device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

// true once the phase with the given parity has completed; false after the
// time budget (from t0) is spent
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, uint64_t t0, uint64_t budget_ns)
{
    const uint32_t a = smem_addr(bar);
    for (;;) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
        if (global_ns() - t0 > budget_ns) return false;
    }
}

__device__ unsigned g_wait_result;

// one CTA: an mbarrier expecting one arrival, which this kernel makes or
// withholds; the wait gives up after budget_ns
__global__ void wait_check_kernel(int arrive, uint64_t budget_ns)
{
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) mbar_init(&bar, 1);
    __syncthreads();
    if (threadIdx.x == 0 && arrive)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&bar)) : "memory");
    const bool ok = mbar_wait(&bar, 0u, global_ns(), budget_ns);
    if (__syncthreads_or(!ok) && threadIdx.x == 0) g_wait_result = 1u;
}
}  // namespace

}  // namespace pic

extern "C" pic_status pic_wait_check(int arrive, double budget_ms, void *stream)
{
    if (!(budget_ms > 0.0) || budget_ms > 10000.0) return PIC_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const unsigned zero = 0u;
    if (cudaMemcpyToSymbolAsync(pic::g_wait_result, &zero, sizeof(zero), 0, cudaMemcpyHostToDevice, s) != cudaSuccess)
        return PIC_ERR_CUDA;
    pic::wait_check_kernel<<<1, 64, 0, s>>>(arrive ? 1 : 0, (uint64_t)(budget_ms * 1e6));
    unsigned r = 0;
    if (cudaGetLastError() != cudaSuccess ||
        cudaMemcpyFromSymbolAsync(&r, pic::g_wait_result, sizeof(r), 0, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return PIC_ERR_CUDA;
    return r ? PIC_ERR_TIMEOUT : PIC_OK;
}
