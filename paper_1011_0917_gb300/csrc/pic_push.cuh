// pic_push.cuh -- the per-tile bodies of the particle kernels and their
// helpers: fused gather / Boris push / Esirkepov deposit / re-bucketing of a
// tile's electrons (with its paired and released ions), and the drifting-ion
// deposit.  The single-run kernels (pic_particles.cu) and the batched ones
// (pic_batch.cu) run the same bodies.
//
// One CTA owns one tile of cells.  It stages E and B of the tile plus guard
// nodes in shared memory, pushes every particle of the tile, accumulates the
// current of all of them in a shared-memory J tile (tile plus the guard nodes
// a one-cell move can reach) and adds that tile to J in HBM once.  Each pushed
// particle is written straight into the bucket of the tile it now lies in, on
// the other side of the double buffer, so the store stays tile-sorted without
// a separate sort pass.
#pragma once

#include "pic_internal.cuh"

#include <cuda_pipeline.h>
#include <type_traits>

namespace pic {

// Threads per CTA of the particle kernels (one CTA per tile) and resident CTAs
// per SM the push kernel is compiled for: 24 warps of 80 registers in FP32
// (the FP64 debug path keeps more registers).  In 3D that is 3 CTAs of 8
// warps, which is what their shared memory allows; a 2D tile holds a quarter
// of the particles, so its start and end (staging, zeroing, the flush) are
// hidden behind more and smaller CTAs: 6 of 4 warps.
template <typename real, int DIM> struct BlockOf {
    static constexpr int value = DIM == 3 || sizeof(real) == 8 ? 256 : 128;
};
template <typename real, int DIM> struct MinBlocks {
    static constexpr int value = (sizeof(real) == 4 ? 3 : 2) * 256 / BlockOf<real, DIM>::value;
};

// ------------------------------------------------- a tile by several CTAs
//
// A grid of few tiles leaves most SMs idle at one CTA per tile.  There kSplit
// CTAs share a tile as a cluster: they take its blocks of records in turn,
// reserve the slots of the records that stay from one counter (in the first
// CTA's shared memory), and their current tiles are added word by word over
// the cluster before they are flushed, so an electron and its ion cancel
// exactly whichever CTA deposits them.
constexpr int kSplit = 4;

template <int SPLIT> __device__ __forceinline__ void cluster_sync()
{
    if (SPLIT > 1) {
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    } else {
        __syncthreads();
    }
}
__device__ __forceinline__ unsigned cluster_rank()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// the address of this CTA's shared variable p in CTA `rank` of the cluster
__device__ __forceinline__ unsigned cluster_map(const void *p, unsigned rank)
{
    unsigned a = (unsigned)__cvta_generic_to_shared(p), d;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(rank));
    return d;
}
__device__ __forceinline__ int cluster_ld(unsigned a, int)
{
    int v;
    asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ double cluster_ld(unsigned a, double)
{
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a));
    return v;
}
// the tile's counter of records that stay: *p of the cluster's first CTA
template <int SPLIT> __device__ __forceinline__ int stay_add(int *p, int n)
{
    if (SPLIT == 1) return atomicAdd(p, n);
    int old;
    asm volatile("atom.shared::cluster.add.s32 %0, [%1], %2;" : "=r"(old) : "r"(cluster_map(p, 0)), "r"(n) : "memory");
    return old;
}

// ---------------------------------------------------------------- helpers

// Shared-memory current accumulators.  FP32 currents are accumulated exactly,
// in 64-bit fixed point split over two 32-bit integer words per node: a
// contribution p = a*b, already multiplied by the launch's fixed-point scale
// (PushArgs::fx_scale, |p| < 2^21), is split into its nearest integer h and
// the remainder r = p - h (exact, |r| <= 1/2), and h and round(r 2^K) go to
// the "hi" and "lo" words with native integer atomics.  Integer addition is
// exact and associative, so a tile's sums do not depend on the order in which
// its particles are processed, and they carry the contributions to 2^-K.
// The "lo" word of a node sits LOFF words after its "hi" word.  FP64
// accumulates in double, and does not add zeros (e.g. nodes of a window
// outside both supports); the FP32 words are added without a test.
template <typename real> struct Acc { using type = double; };
template <> struct Acc<float> { using type = int; };
// bytes of a shared current tile of n values ("hi" and "lo" words in FP32), a multiple of 16
template <typename real> __host__ __device__ constexpr int j_tile_bytes(int n) { return (n * 8 + 15) / 16 * 16; }

// adding 1.5 * 2^23 to x (|x| <= 2^22) leaves round(x) in the low mantissa
// bits, which are read back as an integer
constexpr float kRoundMagic = 12582912.0f;
constexpr int kRoundMagicBits = 0x4B400000;

// adds v to a shared word (no test for zero: the compiler's branch around
// each atomic cost more than the atomics it saved)
__device__ __forceinline__ void sh_add(int *p, int v)
{
    asm volatile("red.shared.add.s32 [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(p)), "r"(v) : "memory");
}

template <int LOFF>
__device__ __forceinline__ void sh_acc(int *p, float a, float b, float lo_scale)
{
    const float t = fmaf(a, b, kRoundMagic);
    const int h = __float_as_int(t) - kRoundMagicBits;
    const float r = fmaf(a, b, -(t - kRoundMagic));
    const int l = __float_as_int(fmaf(r, lo_scale, kRoundMagic)) - kRoundMagicBits;
    sh_add(p, h);
    sh_add(p + LOFF, l);
}

// Two FP32 values in one 64-bit register: Blackwell's packed FP32 instructions
// take one issue slot for both, and the particle loop is bound by issue slots.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pk(float x, float y)
{
    f32x2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
    return d;
}
__device__ __forceinline__ f32x2 pk(float x) { return pk(x, x); }
__device__ __forceinline__ void upk(f32x2 v, float &x, float &y)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b)
{
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// sh_acc of the contributions a b.x to p and a b.y to p + STRIDE: the same
// values as two calls of the scalar form
template <int LOFF, int STRIDE>
__device__ __forceinline__ void sh_acc2(int *p, f32x2 a, f32x2 b, f32x2 lo_scale)
{
    const f32x2 t = fma2(a, b, pk(kRoundMagic));
    const f32x2 r = fma2(a, b, fma2(t, pk(-1.0f), pk(kRoundMagic)));
    const f32x2 l = fma2(r, lo_scale, pk(kRoundMagic));
    sh_add(p, (int)(unsigned)t - kRoundMagicBits);
    sh_add(p + STRIDE, (int)(unsigned)(t >> 32) - kRoundMagicBits);
    sh_add(p + LOFF, (int)(unsigned)l - kRoundMagicBits);
    sh_add(p + LOFF + STRIDE, (int)(unsigned)(l >> 32) - kRoundMagicBits);
}

// contributions of records in relative form into the same fixed-point words
template <int LOFF>
__device__ __forceinline__ void sh_acc(int *p, ff a, ff b, ff lo_scale)
{
    const float v = __fmul_rn(a.h, b.h);
    float e = __fmaf_rn(a.h, b.h, -v);
    e = __fmaf_rn(a.h, b.l, e);
    e = __fmaf_rn(a.l, b.h, e);
    const float t = __fadd_rn(v, kRoundMagic);
    const float r = __fadd_rn(__fsub_rn(v, __fsub_rn(t, kRoundMagic)), e);
    sh_add(p, __float_as_int(t) - kRoundMagicBits);
    sh_add(p + LOFF, __float_as_int(__fmaf_rn(r, lo_scale.h, kRoundMagic)) - kRoundMagicBits);
}

template <int LOFF>
__device__ __forceinline__ void sh_acc(double *p, double a, double b, double)
{
    const double v = a * b;
    if (v != 0.0) atomicAdd(p, v);
}


template <typename real>
struct Ptr6 {
    const real *p0, *p1, *p2, *p3, *p4, *p5;
    __device__ __forceinline__ const real *operator[](int c) const
    {
        return c == 0 ? p0 : c == 1 ? p1 : c == 2 ? p2 : c == 3 ? p3 : c == 4 ? p4 : p5;
    }
};

template <typename real>
struct Ptr3 {
    real *p0, *p1, *p2;
    __device__ __forceinline__ real *operator[](int c) const { return c == 0 ? p0 : c == 1 ? p1 : p2; }
};

// Stage NC field components of the box [lo - L, lo - L + F) (per axis) into
// shared memory.  Element-wise over all threads with compile-time extents, so
// the index decomposition is a few multiply-shifts; consecutive threads read
// consecutive x.  Nodes outside the valid z range of a component (absorbing z)
// are zero; x and y wrap.  Returns whether this thread staged a non-zero value.
template <typename real, int DIM, int NC, int FX, int FY, int FZ, int L>
__device__ __forceinline__ bool stage_tile(const Geom &g, const Ptr6<real> src, unsigned half_z, real *dst, int lox,
                                           int loy, int loz)
{
    constexpr int FN = FX * FY * FZ;
    const bool tiny = g.nx < FX || (DIM == 3 && g.ny < FY);
    bool nonzero = false;
    unsigned bits = 0;
    // each node of the box once, all components of it together; the loads of
    // NU nodes are issued before their values are stored (the tile's start
    // waits for memory about FN / (NU kBlock) times)
    constexpr int kBlock = BlockOf<real, DIM>::value, NI = (FN + kBlock - 1) / kBlock;
    constexpr int NU = sizeof(real) == 4 ? (NI < 4 ? NI : 4) : 2;
    for (int r0 = threadIdx.x; r0 < FN; r0 += NU * kBlock) {
        real v[NU][NC];
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            const int r = r0 + u * kBlock;
            const int lz = r / (FX * FY), r2 = r - lz * (FX * FY);
            const int ly = r2 / FX, lx = r2 - ly * FX;
            int gk = loz - L + lz;
            const bool inz = r < FN && (g.bc_z == 0 || gk >= 0);
            if (g.bc_z == 0) gk = wrapi(gk, g.nz);
            const int gi = tiny ? wrapi(lox - L + lx, g.nx) : wrap1(lox - L + lx, g.nx);
            const int gj = DIM == 3 ? (tiny ? wrapi(loy - L + ly, g.ny) : wrap1(loy - L + ly, g.ny)) : 0;
            const int64_t o = fidx(g, gi, gj, inz ? gk : 0);
#pragma unroll
            for (int c = 0; c < NC; ++c)
                v[u][c] = inz && (g.bc_z == 0 || gk <= zmax_of(g, (half_z >> c) & 1u)) ? src[c][o] : real(0);
        }
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            const int r = r0 + u * kBlock;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                if (r < FN) dst[c * FN + r] = v[u][c];
                if constexpr (sizeof(real) == 4) bits |= __float_as_uint(v[u][c]);
                else nonzero = nonzero || v[u][c] != real(0);
            }
        }
    }
    return nonzero || (bits << 1) != 0u;  // (-0 is a zero)
}

// Add NC shared-memory tiles (box [lo - L, lo - L + Q) per axis) to the global
// arrays, element-wise over all threads: non-zero nodes only, periodic x and y,
// nodes outside a component's valid z range dropped (absorbing z).  FP32
// tiles hold fixed-point "hi" and "lo" words (see sh_acc): the node's value is
// (hi + lo lo_inv) times the component's quantum q_c.
template <typename real, int DIM, int NC, int QX, int QY, int QZ, int L, int SPLIT>
__device__ __forceinline__ void flush_tile(const Geom &g, const Ptr3<real> dstJ, unsigned half_z,
                                           const typename Acc<real>::type *src, real q0, real q1, real q2,
                                           real lo_inv, int lox, int loy, int loz)
{
    constexpr int QN = QX * QY * QZ;
    const bool tiny = g.nx < QX || (DIM == 3 && g.ny < QY);
    // each node of the box once, all components of it together
    using acc_t = typename Acc<real>::type;
    // word w of the tile, summed over the cluster (each CTA flushes its share of the nodes)
    auto word = [&](int w) -> acc_t {
        if (SPLIT == 1) return src[w];
        acc_t v = 0;
#pragma unroll
        for (unsigned p = 0; p < (unsigned)SPLIT; ++p) v += cluster_ld(cluster_map(src + w, p), acc_t(0));
        return v;
    };
    const int first = (SPLIT > 1 ? (int)(cluster_rank() * blockDim.x) : 0) + (int)threadIdx.x;
    for (int r = first; r < QN; r += SPLIT * (int)blockDim.x) {
        real v[NC];
        bool any = false;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            if constexpr (sizeof(real) == 4) {
                const int h = word(c * QN + r), l = word(NC * QN + c * QN + r);  // "hi" and "lo" words
                v[c] = (h | l) == 0 ? real(0) : fmaf((float)l, lo_inv, (float)h);
            } else {
                v[c] = word(c * QN + r);
            }
            any = any || v[c] != real(0);
        }
        if (!any) continue;
        const int lz = r / (QX * QY), r2 = r - lz * (QX * QY);
        const int ly = r2 / QX, lx = r2 - ly * QX;
        int gk = loz - L + lz;
        if (g.bc_z == 0) gk = wrapi(gk, g.nz);
        else if (gk < 0) continue;
        const int gi = tiny ? wrapi(lox - L + lx, g.nx) : wrap1(lox - L + lx, g.nx);
        const int gj = DIM == 3 ? (tiny ? wrapi(loy - L + ly, g.ny) : wrap1(loy - L + ly, g.ny)) : 0;
        const int64_t o = fidx(g, gi, gj, gk);
#pragma unroll
        for (int c = 0; c < NC; ++c)
            if (v[c] != real(0) && (g.bc_z == 0 || gk <= zmax_of(g, (half_z >> c) & 1u)))
                atomicAdd(dstJ[c] + o, v[c] * (c == 0 ? q0 : c == 1 ? q1 : q2));
    }
}

// ---------------------------------------------------------------- gather

// interpolate one component from the shared field tile: node (a, b, c) of the
// support of each axis starts at base + cell-local index (+ guard FL)
template <int DIM, int S, typename real>
__device__ __forceinline__ real gather_comp(const real *F, int FX, int FY, int ix, int iy, int iz,
                                            const real *wx, const real *wy, const real *wz)
{
    if constexpr (S == 1 && sizeof(real) == 4) {
        // the two rows of a plane (3D), the two planes (2D), packed
        const f32x2 a0 = pk(wx[0]), a1 = pk(wx[1]);
        float u, v;
        if (DIM == 3) {
            const f32x2 y = pk(wy[0], wy[1]);
            f32x2 acc = 0;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const real *r0 = F + ((iz + c) * FY + iy) * FX + ix, *r1 = r0 + FX;
                const f32x2 r = fma2(a1, pk(r0[1], r1[1]), mul2(a0, pk(r0[0], r1[0])));
                acc = c ? fma2(mul2(y, pk(wz[c])), r, acc) : mul2(mul2(y, pk(wz[c])), r);
            }
            upk(acc, u, v);
        } else {
            const real *r0 = F + iz * FX + ix, *r1 = r0 + FX;
            upk(mul2(pk(wz[0], wz[1]), fma2(a1, pk(r0[1], r1[1]), mul2(a0, pk(r0[0], r1[0])))), u, v);
        }
        return u + v;
    }
    real sum = 0;
    if (DIM == 3) {
#pragma unroll
        for (int c = 0; c <= S; ++c) {
#pragma unroll
            for (int b = 0; b <= S; ++b) {
                const real *row = F + ((int64_t)(iz + c) * FY + (iy + b)) * FX + ix;
                real r = 0;
#pragma unroll
                for (int a = 0; a <= S; ++a) r += wx[a] * row[a];
                sum += wz[c] * wy[b] * r;
            }
        }
    } else {
#pragma unroll
        for (int c = 0; c <= S; ++c) {
            const real *row = F + (int64_t)(iz + c) * FX + ix;
            real r = 0;
#pragma unroll
            for (int a = 0; a <= S; ++a) r += wx[a] * row[a];
            sum += wz[c] * r;
        }
    }
    return sum;
}

// --------------------------------------------------------- Esirkepov

// The FP32 form of deposit_w below, two nodes of a row at a time (a window of
// three ends in a single one): the same values.
template <int W>
__device__ __forceinline__ void pairs(const float *S0, const float *DS, f32x2 *s, f32x2 *d)
{
#pragma unroll
    for (int q = 0; q < W / 2; ++q) {
        s[q] = pk(S0[2 * q], S0[2 * q + 1]);
        d[q] = pk(DS[2 * q], DS[2 * q + 1]);
    }
}

// contributions P * T(n) of the W nodes n of a row STRIDE words apart, T(n) =
// S0[n] a + DS[n] b
template <int LOFF, int STRIDE, int W>
__device__ __forceinline__ void row_acc(int *p, float P, const f32x2 *T, float Tl, float los)
{
#pragma unroll
    for (int q = 0; q < W / 2; ++q) sh_acc2<LOFF, STRIDE>(p + 2 * q * STRIDE, pk(P), T[q], pk(los));
    if (W & 1) sh_acc<LOFF>(p + (W - 1) * STRIDE, P, Tl, los);
}

template <int DIM, int QX, int QY, int QN, int WX, int WY, int WZ>
__device__ __forceinline__ void deposit_w2(int *sJ, const float *S0x, const float *DSx, const float *S0y,
                                           const float *DSy, const float *S0z, const float *DSz, int ax, int ay,
                                           int az, float fx, float fy, float fz, float fyv, float los)
{
    constexpr int LOFF = 3 * QN;
    constexpr float half = 0.5f, third = 1.0f / 3.0f;
    constexpr int NX = WX / 2 > 0 ? WX / 2 : 1, NY = WY / 2 > 0 ? WY / 2 : 1, NZ = WZ / 2;
    int *Jx = sJ, *Jy = sJ + QN, *Jz = sJ + 2 * QN;
    f32x2 sx[NX], dx[NX], T[NX > NY ? (NX > NZ ? NX : NZ) : (NY > NZ ? NY : NZ)];
    pairs<WX>(S0x, DSx, sx, dx);
    float Px[WX], Pz[WZ], acc = 0, Tl = 0;
#pragma unroll
    for (int q = 0; q < WX; ++q) { acc += DSx[q]; Px[q] = fx * acc; }
    acc = 0;
#pragma unroll
    for (int c = 0; c < WZ; ++c) { acc += DSz[c]; Pz[c] = fz * acc; }
    if (DIM == 3) {
        f32x2 sy[NY], dy[NY];
        pairs<WY>(S0y, DSy, sy, dy);
        float Py[WY];
        acc = 0;
#pragma unroll
        for (int b = 0; b < WY; ++b) { acc += DSy[b]; Py[b] = fy * acc; }
#pragma unroll
        for (int c = 0; c < WZ; ++c) {
            const float za = S0z[c] + half * DSz[c], zb = half * S0z[c] + third * DSz[c];
            const int o = ((az + c) * QY + ay) * QX + ax;
#pragma unroll
            for (int b = 0; b < WY / 2; ++b) T[b] = fma2(sy[b], pk(za), mul2(dy[b], pk(zb)));
            if (WY & 1) Tl = S0y[WY - 1] * za + DSy[WY - 1] * zb;
#pragma unroll
            for (int q = 0; q < WX - 1; ++q) row_acc<LOFF, QX, WY>(Jx + o + q, Px[q], T, Tl, los);
#pragma unroll
            for (int q = 0; q < WX / 2; ++q) T[q] = fma2(sx[q], pk(za), mul2(dx[q], pk(zb)));
            if (WX & 1) Tl = S0x[WX - 1] * za + DSx[WX - 1] * zb;
#pragma unroll
            for (int b = 0; b < WY - 1; ++b) row_acc<LOFF, 1, WX>(Jy + o + b * QX, Py[b], T, Tl, los);
        }
#pragma unroll
        for (int b = 0; b < WY; ++b) {
            const float ya = S0y[b] + half * DSy[b], yb = half * S0y[b] + third * DSy[b];
            const int o = (az * QY + ay + b) * QX + ax;
#pragma unroll
            for (int q = 0; q < WX / 2; ++q) T[q] = fma2(sx[q], pk(ya), mul2(dx[q], pk(yb)));
            if (WX & 1) Tl = S0x[WX - 1] * ya + DSx[WX - 1] * yb;
#pragma unroll
            for (int c = 0; c < WZ - 1; ++c) row_acc<LOFF, 1, WX>(Jz + o + c * QX * QY, Pz[c], T, Tl, los);
        }
    } else {
        const int o = az * QX + ax;
        f32x2 sz[NZ], dz[NZ];
        pairs<WZ>(S0z, DSz, sz, dz);
#pragma unroll
        for (int c = 0; c < WZ / 2; ++c) T[c] = fma2(dz[c], pk(half), sz[c]);
        if (WZ & 1) Tl = S0z[WZ - 1] + half * DSz[WZ - 1];
#pragma unroll
        for (int q = 0; q < WX - 1; ++q) row_acc<LOFF, QX, WZ>(Jx + o + q, Px[q], T, Tl, los);
#pragma unroll
        for (int c = 0; c < WZ; ++c) {
            const float za = S0z[c] + half * DSz[c], zb = half * S0z[c] + third * DSz[c];
#pragma unroll
            for (int q = 0; q < WX / 2; ++q) T[q] = fma2(sx[q], pk(za), mul2(dx[q], pk(zb)));
            if (WX & 1) Tl = S0x[WX - 1] * za + DSx[WX - 1] * zb;
            row_acc<LOFF, 1, WX>(Jy + o + c * QX, fyv, T, Tl, los);
        }
#pragma unroll
        for (int q = 0; q < WX / 2; ++q) T[q] = fma2(dx[q], pk(half), sx[q]);
        if (WX & 1) Tl = S0x[WX - 1] + half * DSx[WX - 1];
#pragma unroll
        for (int c = 0; c < WZ - 1; ++c) row_acc<LOFF, 1, WX>(Jz + o + c * QX, Pz[c], T, Tl, los);
    }
}

// Current of one particle into the shared J tile.  Along an axis the window
// has W nodes: S+1 when no lane of the warp moved its support to another first
// node along that axis (the last node is then outside both supports), else
// S+2.  The running sum along an axis is taken over DS first:
//   Jx(a,b,c) = fx * (sum_{a'<=a} DSx[a']) * T_yz(b,c),
//   T_yz = S0y (S0z + DSz/2) + DSy (S0z/2 + DSz/3)        (and cyclically),
// which is Esirkepov's decomposition rearranged; the last running sum of a
// window is zero and is not added.  In 2D3V the out-of-plane current is the
// path average of the shape times q w vy / V.
template <typename real, typename accT, int DIM, int S, int QX, int QY, int QN, int WX, int WY, int WZ>
__device__ __forceinline__ void deposit_w(accT *sJ, const real *S0x, const real *DSx, const real *S0y,
                                          const real *DSy, const real *S0z, const real *DSz, int ax, int ay, int az,
                                          real fx, real fy, real fz, real fyv, real los)
{
    constexpr int LOFF = 3 * QN;  // "lo" words follow the three components' "hi" words
    const real half = real(0.5), third = real(1.0 / 3.0);
    auto *Jx = sJ, *Jy = sJ + QN, *Jz = sJ + 2 * QN;
    if constexpr (sizeof(real) == 4) {
        deposit_w2<DIM, QX, QY, QN, WX, WY, WZ>(sJ, S0x, DSx, S0y, DSy, S0z, DSz, ax, ay, az, fx, fy, fz, fyv, los);
        return;
    }
    real Px[WX], Pz[WZ];
    real acc = 0;
#pragma unroll
    for (int q = 0; q < WX; ++q) { acc += DSx[q]; Px[q] = fx * acc; }
    acc = 0;
#pragma unroll
    for (int c = 0; c < WZ; ++c) { acc += DSz[c]; Pz[c] = fz * acc; }
    if (DIM == 3) {
        real Py[WY];
        acc = 0;
#pragma unroll
        for (int b = 0; b < WY; ++b) { acc += DSy[b]; Py[b] = fy * acc; }
#pragma unroll
        for (int c = 0; c < WZ; ++c) {
            const real za = S0z[c] + half * DSz[c], zb = half * S0z[c] + third * DSz[c];
#pragma unroll
            for (int b = 0; b < WY; ++b) {
                const real tyz = S0y[b] * za + DSy[b] * zb;
                auto *row = Jx + ((az + c) * QY + (ay + b)) * QX + ax;
#pragma unroll
                for (int q = 0; q < WX - 1; ++q) sh_acc<LOFF>(row + q, Px[q], tyz, los);
            }
#pragma unroll
            for (int q = 0; q < WX; ++q) {
                const real tzx = S0z[c] * (S0x[q] + half * DSx[q]) + DSz[c] * (half * S0x[q] + third * DSx[q]);
                auto *col = Jy + ((az + c) * QY + ay) * QX + ax + q;
#pragma unroll
                for (int b = 0; b < WY - 1; ++b) sh_acc<LOFF>(col + b * QX, Py[b], tzx, los);
            }
        }
#pragma unroll
        for (int b = 0; b < WY; ++b) {
            const real ya = S0y[b] + half * DSy[b], yb = half * S0y[b] + third * DSy[b];
#pragma unroll
            for (int q = 0; q < WX; ++q) {
                const real txy = S0x[q] * ya + DSx[q] * yb;
                auto *col = Jz + (az * QY + (ay + b)) * QX + ax + q;
#pragma unroll
                for (int c = 0; c < WZ - 1; ++c) sh_acc<LOFF>(col + c * QX * QY, Pz[c], txy, los);
            }
        }
    } else {
#pragma unroll
        for (int c = 0; c < WZ; ++c) {
            const real za = S0z[c] + half * DSz[c], zb = half * S0z[c] + third * DSz[c];
            auto *row = Jx + (az + c) * QX + ax;
#pragma unroll
            for (int q = 0; q < WX - 1; ++q) sh_acc<LOFF>(row + q, Px[q], za, los);
#pragma unroll
            for (int q = 0; q < WX; ++q) sh_acc<LOFF>(Jy + (az + c) * QX + ax + q, fyv, S0x[q] * za + DSx[q] * zb, los);
        }
#pragma unroll
        for (int q = 0; q < WX; ++q) {
            const real xa = S0x[q] + half * DSx[q];
#pragma unroll
            for (int c = 0; c < WZ - 1; ++c) sh_acc<LOFF>(Jz + (az + c) * QX + ax + q, Pz[c], xa, los);
        }
    }
}

// The current of particles that did not move across z (3D): Wx = Wy = 0
// exactly, so Jx = Jy = 0 and Jz(q,b,c) = fz (sum_{c'<=c} DSz[c']) S0x[q] S0y[b]
// -- the general formula's values with DSx = DSy = 0.  Windows along x and y
// have S+1 nodes (their supports did not move).
template <typename real, typename accT, int S, int QX, int QY, int QN, int WZ>
__device__ __forceinline__ void deposit_z(accT *sJ, const real *S0x, const real *S0y, const real *S0z,
                                          const real *DSz, int ax, int ay, int az, real fz, real los)
{
    constexpr int LOFF = 3 * QN;
    auto *Jz = sJ + 2 * QN;
    real Pz[WZ];
    real acc = 0;
#pragma unroll
    for (int c = 0; c < WZ; ++c) { acc += DSz[c]; Pz[c] = fz * acc; }
    (void)S0z;
    if constexpr (sizeof(real) == 4) {
        f32x2 sx[(S + 1) / 2], T[(S + 1) / 2];
#pragma unroll
        for (int q = 0; q < (S + 1) / 2; ++q) sx[q] = pk(S0x[2 * q], S0x[2 * q + 1]);
#pragma unroll
        for (int b = 0; b < S + 1; ++b) {
#pragma unroll
            for (int q = 0; q < (S + 1) / 2; ++q) T[q] = mul2(sx[q], pk(S0y[b]));
            const float Tl = S0x[S] * S0y[b];
#pragma unroll
            for (int c = 0; c < WZ - 1; ++c)
                row_acc<LOFF, 1, S + 1>(Jz + ((az + c) * QY + (ay + b)) * QX + ax, Pz[c], T, Tl, los);
        }
        return;
    }
#pragma unroll
    for (int b = 0; b < S + 1; ++b) {
#pragma unroll
        for (int q = 0; q < S + 1; ++q) {
            const real txy = S0x[q] * S0y[b];
            auto *col = Jz + (az * QY + (ay + b)) * QX + ax + q;
#pragma unroll
            for (int c = 0; c < WZ - 1; ++c) sh_acc<LOFF>(col + c * QX * QY, Pz[c], txy, los);
        }
    }
}

// picks the window lengths for the warp: bit 2 x, bit 1 y, bit 0 z crossed
template <typename real, typename accT, int DIM, int S, int QX, int QY, int QN>
__device__ __forceinline__ void deposit_sel(unsigned sel, accT *sJ, const real *S0x, const real *DSx, const real *S0y,
                                            const real *DSy, const real *S0z, const real *DSz, int ax, int ay, int az,
                                            real fx, real fy, real fz, real fyv, real los)
{
    constexpr int A = S + 1, B = S + 2;
#define PIC_DEP(wx, wy, wz) \
    deposit_w<real, accT, DIM, S, QX, QY, QN, wx, wy, wz>(sJ, S0x, DSx, S0y, DSy, S0z, DSz, ax, ay, az, fx, fy, fz, fyv, los)
    if (DIM == 3) {
        switch (sel) {
        case 0: PIC_DEP(A, A, A); break;
        case 1: PIC_DEP(A, A, B); break;
        case 2: PIC_DEP(A, B, A); break;
        case 3: PIC_DEP(A, B, B); break;
        case 4: PIC_DEP(B, A, A); break;
        case 5: PIC_DEP(B, A, B); break;
        case 6: PIC_DEP(B, B, A); break;
        default: PIC_DEP(B, B, B); break;
        }
    } else {
        switch (sel & 5u) {
        case 0: PIC_DEP(A, 1, A); break;
        case 1: PIC_DEP(A, 1, B); break;
        case 4: PIC_DEP(B, 1, A); break;
        default: PIC_DEP(B, 1, B); break;
        }
    }
#undef PIC_DEP
}

// Esirkepov's window along one axis for records in relative form: both ends
// in ff or FP64, each within a cell of [0, 1) (esirk_axis_g, whose FP64 form
// the debug path takes).
template <int S>
__device__ __forceinline__ float spline_ff(ff p, ff w[S + 1])
{
    if (S == 1) {
        const float f = floor_ff(p);
        const ff d = p - ff(f);
        w[0] = ff(1.0f) - d;
        w[1] = d;
        return f;
    }
    const float c = floor_ff(p + ff(0.5f));
    const ff d = p - ff(c), a = ff(0.5f) - d, b = ff(0.5f) + d;
    w[0] = ff(0.5f) * (a * a);
    w[1] = ff(0.75f) - d * d;
    w[2] = ff(0.5f) * (b * b);
    return c - 1.0f;
}
template <int S>
__device__ __forceinline__ int esirk_rel(ff x0, ff x1, ff S0[S + 2], ff DS[S + 2], bool &crossed)
{
    ff w0[S + 1], w1[S + 1];
    const float b0 = spline_ff<S>(x0, w0), b1 = spline_ff<S>(x1, w1);
    const bool s0 = b0 > b1, s1 = b1 > b0;  // which support starts a node above the window
    crossed = b0 != b1;
#pragma unroll
    for (int q = 0; q < S + 2; ++q) {
        const ff lo0 = q <= S ? w0[q <= S ? q : S] : ff(0.0f), hi0 = q >= 1 ? w0[q >= 1 ? q - 1 : 0] : ff(0.0f);
        const ff lo1 = q <= S ? w1[q <= S ? q : S] : ff(0.0f), hi1 = q >= 1 ? w1[q >= 1 ? q - 1 : 0] : ff(0.0f);
        const ff v1 = ff(s1 ? hi1.h : lo1.h, s1 ? hi1.l : lo1.l);
        S0[q] = ff(s0 ? hi0.h : lo0.h, s0 ? hi0.l : lo0.l);
        DS[q] = v1 - S0[q];
    }
    return (int)fminf(b0, b1);
}
template <int S>
__device__ __forceinline__ int esirk_rel(double x0, double x1, double S0[S + 2], double DS[S + 2], bool &crossed)
{
    return esirk_axis_g<S>(x0, x1, S0, DS, crossed);
}
// a position in the arithmetic of the deposit: r + (o + dl).  The pair of o and
// dl is exact; adding the cell shift r (0 for most records) rounds its low word,
// by at most 2^-48 of the position.
template <typename T> __device__ __forceinline__ T rel_pos(int r, double o, double dl) { return (T)r + (o + dl); }
template <typename T> __device__ __forceinline__ T rel_pos(int r, float o, float dl)
{
    return T(r) + two_sum(o, dl);
}

// One axis of the CIC window from the in-cell offset o, the offset d in the
// new cell and that cell f in {-1, 0, 1}: a window of two nodes when no lane
// of the warp changes cell (f = 0), else of three whose first node is f's or
// the old cell's, the lower.  The values of esirk_axis_c.
template <int W>
__device__ __forceinline__ int cic_axis(float o, float d, float f, float *S0, float *DS)
{
    const float a0 = 1.0f - o, a1 = o, b0 = 1.0f - d, b1 = d;
    if (W == 2) {
        S0[0] = a0;
        S0[1] = a1;
        DS[0] = b0 - a0;
        DS[1] = b1 - a1;
        return 0;
    }
    const bool dn = f < 0.0f, up = f > 0.0f;
    S0[0] = dn ? 0.0f : a0;
    S0[1] = dn ? a0 : a1;
    S0[2] = dn ? a1 : 0.0f;
    DS[0] = (up ? 0.0f : b0) - S0[0];
    DS[1] = (up ? b0 : b1) - S0[1];
    DS[2] = (up ? b1 : 0.0f) - S0[2];
    return dn ? -1 : 0;
}

template <int DIM, int QX, int QY, int QN, int WX, int WY, int WZ>
__device__ __forceinline__ void deposit_cic_w(int *sJ, float ox, float dx, float fx, int li, float oy, float dy, float fy,
                                              int lj, float oz, float dz, float fz, int lk, float jx, float jy, float jz,
                                              float jyv, float los)
{
    float S0x[WX], DSx[WX], S0y[WY], DSy[WY], S0z[WZ], DSz[WZ];
    const int ax = cic_axis<WX>(ox, dx, fx, S0x, DSx) + li + 1;
    const int az = cic_axis<WZ>(oz, dz, fz, S0z, DSz) + lk + 1;
    int ay = 0;
    if constexpr (DIM == 3) ay = cic_axis<WY>(oy, dy, fy, S0y, DSy) + lj + 1;
    deposit_w2<DIM, QX, QY, QN, WX, WY, WZ>(sJ, S0x, DSx, S0y, DSy, S0z, DSz, ax, ay, az, jx, jy, jz, jyv, los);
}

// the CIC current of one particle, FP32 (sel: bit 2 x, bit 1 y, bit 0 z
// crossed by a lane of the warp)
template <int DIM, int QX, int QY, int QN>
__device__ __forceinline__ void deposit_cic(bool z_only, unsigned sel, int *sJ, float ox, float dx, float fx, int li,
                                            float oy, float dy, float fy, int lj, float oz, float dz, float fz, int lk,
                                            float jx, float jy, float jz, float jyv, float los)
{
    if (DIM == 3 && z_only) {
        float S0z[3], DSz[3];
        const float wx[2] = {1.0f - ox, ox}, wy[2] = {1.0f - oy, oy};
        const int az = cic_axis<3>(oz, dz, fz, S0z, DSz) + lk + 1;
        deposit_z<float, int, 1, QX, QY, QN, 3>(sJ, wx, wy, S0z, DSz, li + 1, lj + 1, az, jz, los);
        return;
    }
#define PIC_DEP(wx, wy, wz)                                                                                          \
    deposit_cic_w<DIM, QX, QY, QN, wx, wy, wz>(sJ, ox, dx, fx, li, oy, dy, fy, lj, oz, dz, fz, lk, jx, jy, jz, jyv, los)
    if (DIM == 3) {
        switch (sel) {
        case 0: PIC_DEP(2, 2, 2); break;
        case 1: PIC_DEP(2, 2, 3); break;
        case 2: PIC_DEP(2, 3, 2); break;
        case 3: PIC_DEP(2, 3, 3); break;
        case 4: PIC_DEP(3, 2, 2); break;
        case 5: PIC_DEP(3, 2, 3); break;
        case 6: PIC_DEP(3, 3, 2); break;
        default: PIC_DEP(3, 3, 3); break;
        }
    } else {
        switch (sel & 5u) {
        case 0: PIC_DEP(2, 1, 2); break;
        case 1: PIC_DEP(2, 1, 3); break;
        case 4: PIC_DEP(3, 1, 2); break;
        default: PIC_DEP(3, 1, 3); break;
        }
    }
#undef PIC_DEP
}

// --------------------------------------------------- a tile's records by warp
//
// The warps of a CTA take the blocks of 32 records of the tile's two runs in
// turn, each warp on its own.  A block (one contiguous piece, see Rec) is
// copied into the warp's buffer with 16-byte cp.async while the block before
// it is worked on: its values go to registers at the start of an iteration,
// so one buffer per warp is enough.  Records that stay in the tile are
// written at once, to slots from a shared-memory counter.  Records that leave
// it are put aside in a queue of 32 per warp and written when it is full (or
// the tile is done): their slots come from global atomics, whose latency
// (the largest stall of the loop when every iteration waited for it: 2000 of
// its 5300 cycles on a 3D gamma = 13 plasma, where 9% of the records cross a
// tile face per step) and whose code a warp then pays once per 32 of them.

// the lane and the mask of the lanes below it, read once: the special
// registers are slow, and the compiler would read them again at every use
__device__ __forceinline__ int lane_reg()
{
    int v;
    asm volatile("mov.u32 %0, %%laneid;" : "=r"(v));
    return v;
}
__device__ __forceinline__ unsigned lanemask_lt_reg()
{
    unsigned v;
    asm volatile("mov.u32 %0, %%lanemask_lt;" : "=r"(v));
    return v;
}

// shared memory of a warp: a block, the queue's records, their moves and
// their input slots
template <typename R> __host__ __device__ constexpr int warp_bytes() { return 2 * R::RB + 256; }

struct Blocks {          // the blocks that hold the two runs of a bucket
    int n_lo, hi_first;  // bottom run [0, n_lo), top run [hi_first, cap)
    int nb_lo, hi0, n;   // blocks of the bottom run, first further block of the top run, blocks in all
    __device__ __forceinline__ Blocks(int lo, int hi, int cap)
    {
        n_lo = lo;
        hi_first = cap - hi;
        nb_lo = (lo + 31) >> 5;
        hi0 = max(hi_first >> 5, nb_lo);
        n = nb_lo + (cap >> 5) - hi0;
    }
    __device__ __forceinline__ int block(int i) const { return i < nb_lo ? i : hi0 + (i - nb_lo); }
    __device__ __forceinline__ bool valid(int slot) const { return slot < n_lo || slot >= hi_first; }
};

// (dst, src: already at the lane's 16 bytes)
template <int RB>
__device__ __forceinline__ void fetch_block(unsigned char *dst, const unsigned char *src, int lane)
{
#pragma unroll
    for (int q = 0; q < RB; q += 512)
        if (q + 512 <= RB || q + lane * 16 < RB) __pipeline_memcpy_async(dst + q, src + q, 16);
    __pipeline_commit();
}

// byte offset of slot s of a bucket: its block, then the lane's element of a row
template <int RB, typename T> __device__ __forceinline__ int slot_off(int s)
{
    return (s >> 5) * RB + (s & 31) * (int)sizeof(T);
}

template <typename T> __device__ __forceinline__ T &row(unsigned char *block, int off, int i)
{
    return *reinterpret_cast<T *>(block + off + i * (int)sizeof(T));
}
// at: a pointer already at the lane's element of the block's first row
template <typename T> __device__ __forceinline__ T &at(unsigned char *p, int off)
{
    return *reinterpret_cast<T *>(p + off);
}

// the tile's place: first cell, extents (smaller at a ragged end) and the
// packed cell word of its first cell.  A record's cell word minus that word
// holds its local indices in the same bit fields; any bit outside `mask`
// means another tile (tile corners are multiples of the tile shape, so no
// other cell's difference looks like a local one).
template <int DIM, int TX, int TY, int TZ>
struct TilePos {
    int lox, loy, loz, ex, ey, ez, tix, tiy, tiz;
    uint32_t word0, mask;
    __device__ __forceinline__ TilePos(const Geom &g, int64_t t)
    {
        const int n2 = g.nt[0] * g.nt[1];
        tiz = (int)(t / n2);
        const int r = (int)(t - (int64_t)tiz * n2);
        tiy = DIM == 3 ? r / g.nt[0] : 0;
        tix = r - tiy * g.nt[0];
        lox = tix * TX;
        loy = tiy * TY;
        loz = tiz * TZ;
        ex = min(TX, g.nx - lox);
        ey = DIM == 3 ? min(TY, g.ny - loy) : 1;
        ez = min(TZ, g.nz - loz);
        word0 = (uint32_t)pack_cell(g, lox, loy, loz);
        mask = (uint32_t)min(TX - 1, (1 << g.bx) - 1) | (uint32_t)(TZ - 1) << (g.bx + g.by);
        if (DIM == 3) mask |= (uint32_t)min(TY - 1, (1 << g.by) - 1) << g.bx;
    }
    // local indices of a cell word (pair bit cleared); false: another tile's
    __device__ __forceinline__ bool local(const Geom &g, uint32_t word, int &li, int &lj, int &lk) const
    {
        const uint32_t d = word - word0;
        li = (int)(d & (uint32_t)min(TX - 1, (1 << g.bx) - 1));
        lj = DIM == 3 ? (int)((d >> g.bx) & (uint32_t)min(TY - 1, (1 << g.by) - 1)) : 0;
        lk = (int)(d >> (g.bx + g.by));
        return (d & ~mask) == 0u;
    }
};

// ------------------------------------------------------------- drifting ions

// Ions immobile in the lab move at the species' constant u = (0, 0, -gamma
// beta) in the boosted frame: every ion of a step moves by the same
// dz = u_z dt / (gamma h_z), in (-1, 0) cells, and its transverse position
// never changes.  So only Jz is deposited, Wz = DSz (S0x S0y) (the general
// formula with DSx = DSy = 0, in the arithmetic order of the electrons'
// z-only deposit), and an ion either stays in its tile or moves to the one
// tile below it (the top tile when z wraps, none when it leaves the box): the
// slots of a queue of leavers come from one atomic.

// Jz of one ion moving along z from z0 to z1 (both relative to its cell, z0 in
// [0, 1)), in arithmetic ar, into the current tile Jz (QX x QY rows)
template <typename ar, typename accT, int DIM, int S, int QX, int QY, int LOFF>
__device__ __forceinline__ void ion_deposit(accT *Jz, ar z0, ar z1, ar ox, ar oy, int li, int lj, int lk, ar fz,
                                            ar lo_scale)
{
    constexpr int JL = S;
    ar S0z[S + 2], DSz[S + 2], wx[S + 1], wy[S + 1];
    bool crossed;
    int az, bx, by = 0;
    if constexpr (std::is_same<ar, ff>::value) {
        az = esirk_rel<S>(z0, z1, S0z, DSz, crossed) + lk + JL;
        bx = (int)spline_ff<S>(ox, wx) + li + JL;
        if (DIM == 3) by = (int)spline_ff<S>(oy, wy) + lj + JL;
    } else {
        az = esirk_axis_c<S>(z0, z1, S0z, DSz, crossed) + lk + JL;
        bx = offset_weights<S>(ox, wx) + li + JL;
        if (DIM == 3) by = offset_weights<S>(oy, wy) + lj + JL;
    }
    ar Pz[S + 2];
    ar run = 0;
#pragma unroll
    for (int c = 0; c < S + 2; ++c) {
        run += DSz[c];
        Pz[c] = fz * run;
    }
    if constexpr (std::is_same<ar, float>::value) {
        f32x2 T[(S + 1) / 2];
#pragma unroll
        for (int b = 0; b < (DIM == 3 ? S + 1 : 1); ++b) {
#pragma unroll
            for (int q = 0; q < (S + 1) / 2; ++q) {
                T[q] = pk(wx[2 * q], wx[2 * q + 1]);
                if (DIM == 3) T[q] = mul2(T[q], pk(wy[b]));
            }
            const float Tl = DIM == 3 ? wx[S] * wy[b] : wx[S];
#pragma unroll
            for (int c = 0; c < S + 1; ++c)
                row_acc<LOFF, 1, S + 1>(Jz + ((az + c) * QY + (by + b)) * QX + bx, Pz[c], T, Tl, lo_scale);
        }
        return;
    }
#pragma unroll
    for (int b = 0; b < (DIM == 3 ? S + 1 : 1); ++b) {
#pragma unroll
        for (int q = 0; q < S + 1; ++q) {
            const ar sxy = DIM == 3 ? wx[q] * wy[b] : wx[q];
#pragma unroll
            for (int c = 0; c < S + 1; ++c)
                sh_acc<LOFF>(Jz + ((az + c) * QY + (by + b)) * QX + bx + q, Pz[c], sxy, lo_scale);
        }
    }
}

// The ions of tile t (all threads of the CTA call it): their Jz into the
// current tile at Jz (the "hi" words; the "lo" words LOFF further), records
// into the output side.  wbuf: the warp's buffer.  REL: the tile's electrons
// are in relative form; the ions' currents are then formed in their arithmetic
// (ff) from their stored positions (the end of one step's path is exactly the start of the
// next one's).  Returns false (nothing done) for an empty bucket.  The loop
// runs all lanes of a warp (as the electrons', see push_tile).
template <typename real, int DIM, int S, int TX, int TY, int TZ, int LOFF, bool REL, int SPLIT>
__device__ __forceinline__ bool ions_of_tile(const Geom &g, const IonSide<real> &is, int64_t t,
                                             const TilePos<DIM, TX, TY, TZ> &tp, typename Acc<real>::type *Jz,
                                             unsigned char *wbuf, real dz, real scale_z, real lo_scale, unsigned *err,
                                             int *s_stay)
{
    constexpr int JL = S, JH = S + 1;
    constexpr int QX = TX + JL + JH, QY = DIM == 3 ? TY + JL + JH : 1;
    using acc_t = typename Acc<real>::type;
    using R = Rec<real, DIM, false, false>;
    using rel_t = typename std::conditional<sizeof(real) == 4, ff, double>::type;
    constexpr int ES = (int)sizeof(real), kBlock = BlockOf<real, DIM>::value;
    int n_lo, n_hi;
    bucket_counts(is.in_lo, is.in_hi, t, g.cap, n_lo, n_hi, err);
    if (n_lo + n_hi == 0) return false;
    const int lane = lane_reg();
    const unsigned lt = lanemask_lt_reg();
    const Blocks bl(n_lo, n_hi, g.cap);
    const int64_t bucket = (int64_t)(g.cap >> 5) * R::RB;
    const unsigned char *in = reinterpret_cast<const unsigned char *>(is.in.ox) + t * bucket + lane * 16;
    unsigned char *out = reinterpret_cast<unsigned char *>(is.out.ox) + t * bucket;
    const int kbit = g.bx + g.by;
    unsigned char *fbuf = wbuf + lane * 16, *rbuf = wbuf + lane * ES, *q = wbuf + R::RB;
    int *qslot = reinterpret_cast<int *>(q + R::RB) + 32;
    const int ntxy = g.nt[0] * g.nt[1];
    // the tile an ion leaving this one through its lower z face enters
    // (-1: it leaves the box), and the cell word's jump there through the
    // periodic end
    const int64_t below = tp.tiz > 0 ? t - ntxy : (g.bc_z == 0 ? t + (int64_t)(g.nt[2] - 1) * ntxy : -1);
    const int32_t jump = tp.tiz == 0 && g.bc_z == 0 ? g.nz << kbit : 0;
    auto put = [&](unsigned char *b, int slot, real ox, real oy, real oz, real w, int32_t cell) {
        b += slot_off<R::RB, real>(slot);
        at<real>(b, R::OX) = ox;
        if (DIM == 3) at<real>(b, R::OY) = oy;
        at<real>(b, R::OZ) = oz;
        at<real>(b, R::W) = w;
        at<int32_t>(ES == 4 ? b : b - (slot & 31) * 4, R::CELL) = cell;
    };
    const int rank = SPLIT > 1 ? (int)cluster_rank() : 0;
    __syncthreads();
    if (threadIdx.x == 0) *s_stay = 0;
    cluster_sync<SPLIT>();
    int i = rank * (kBlock / 32) + (int)(threadIdx.x >> 5), qn = 0;
    // the queue's records into the tile below
    auto flush = [&]() {
        __syncwarp();
        int b = 0;
        if (lane == 0) b = atomicAdd(&is.out_hi[below], qn);
        b = g.cap - 1 - (__shfl_sync(0xffffffffu, b, 0) + lane);
        if (lane < qn) {
            if (b >= 0) {
                unsigned char *p = q + lane * ES;
                put(out + (below - t) * bucket, b, at<real>(p, R::OX), DIM == 3 ? at<real>(p, R::OY) : real(0),
                    at<real>(p, R::OZ), at<real>(p, R::W), row<int32_t>(q, R::CELL, lane));
                if (is.out.id)
                    is.out.id[below * (int64_t)g.cap + b] = is.in.id ? is.in.id[t * (int64_t)g.cap + qslot[lane]] : 0;
            } else {
                atomicOr(err, ERR_CAPACITY);
            }
        }
        __syncwarp();
        qn = 0;
    };
    if (i < bl.n) fetch_block<R::RB>(fbuf, in + (int64_t)bl.block(i) * R::RB, lane);
    while (i < bl.n) {
        const int slot = bl.block(i) * 32 + lane;
        bool valid = bl.valid(slot);
        __pipeline_wait_prior(0);
        __syncwarp();
        real ox = at<real>(rbuf, R::OX), oy = DIM == 3 ? at<real>(rbuf, R::OY) : real(0);
        real oz = at<real>(rbuf, R::OZ), w = at<real>(rbuf, R::W);
        uint32_t cell = row<uint32_t>(wbuf, R::CELL, lane);
        __syncwarp();
        i += SPLIT * (kBlock / 32);
        if (i < bl.n) fetch_block<R::RB>(fbuf, in + (int64_t)bl.block(i) * R::RB, lane);
        int li, lj, lk;
        bool here = tp.local(g, cell, li, lj, lk);
        if (!__all_sync(0xffffffffu, valid && here)) {  // a run's end, or a record in the wrong bucket
            if (valid && !here) atomicOr(err, ERR_TILE);
            valid = valid && here;
            if (!valid) {
                ox = oy = oz = w = real(0);
                li = lj = lk = 0;
            }
        }
        const real z0 = oz, z1 = add_rn(oz, dz);
        // z1 in (-1, 1): the same cell or the one below; an offset that
        // rounds to 1 stays in the cell with offset 0
        const real up = z1 + real(1);
        const int sz = z1 < real(0) && up < real(1) ? -1 : 0;
        oz = z1 < real(0) ? (sz ? up : real(0)) : z1;
        if (valid) {
            if (REL)  // from the stored position to the stored position
                ion_deposit<rel_t, acc_t, DIM, S, QX, QY, LOFF>(Jz, rel_t(z0), rel_pos<rel_t>(sz, oz, real(0)), rel_t(ox),
                                                                rel_t(oy), li, lj, lk,
                                                                rel_t(is.jfac_z) * rel_t(w) * rel_t(scale_z),
                                                                rel_t(lo_scale));
            else
                ion_deposit<real, acc_t, DIM, S, QX, QY, LOFF>(Jz, z0, z1, ox, oy, li, lj, lk, is.jfac_z * w * scale_z,
                                                               lo_scale);
        }
        const bool in_tile = lk + sz >= 0;
        const bool stay = valid && in_tile, leave = valid && !in_tile && below >= 0;
        cell += (uint32_t)sz << kbit;
        const unsigned ms = __ballot_sync(0xffffffffu, stay), ml = __ballot_sync(0xffffffffu, leave);
        int bs = 0;
        if (lane == 0) bs = stay_add<SPLIT>(s_stay, __popc(ms));
        bs = __shfl_sync(0xffffffffu, bs, 0) + __popc(ms & lt);
        if (stay) {
            put(out, bs, ox, oy, oz, w, (int32_t)cell);
            if (is.out.id)
                is.out.id[t * (int64_t)g.cap + bs] = is.in.id ? is.in.id[t * (int64_t)g.cap + slot] : 0;
        }
        if (ml) {
            const int nl = __popc(ml);
            if (qn + nl > 32) flush();
            if (leave) {
                const int e = qn + __popc(ml & lt);
                unsigned char *p = q + e * ES;
                at<real>(p, R::OX) = ox;
                if (DIM == 3) at<real>(p, R::OY) = oy;
                at<real>(p, R::OZ) = oz;
                at<real>(p, R::W) = w;
                row<int32_t>(q, R::CELL, e) = (int32_t)cell + jump;
                qslot[e] = slot;
            }
            qn += nl;
        }
    }
    if (qn) flush();
    cluster_sync<SPLIT>();
    if (threadIdx.x == 0 && rank == 0) {
        is.out_lo[t] = *s_stay;
        is.in_lo[t] = 0;
        is.in_hi[t] = 0;
    }
    return true;
}

// ------------------------------------------------------------ push kernel

// one axis of a record in relative form: the departure takes the step's
// displacement d; whole cells move to the reference (exact: |dl| <= 3/2)
template <typename real>
__device__ __forceinline__ real rel_step(real dl, real d, int &fold)
{
    real v = dl + d;
    fold = 0;
    if (v > real(0.5)) {
        v = v - real(1);
        fold = 1;
    } else if (v < real(-0.5)) {
        v = v + real(1);
        fold = -1;
    }
    return v;
}

// REL: electron records in relative form (rel_actual): the gather uses the
// offsets in the stored cell, the current is deposited in ff arithmetic from
// the exact positions reference + departure.
//
// The loop is bound by issue slots and the latency they hide, so it runs all
// 32 lanes of a warp without per-lane branches: lanes without a record (the
// ends of the runs) take a record at rest of weight zero that goes nowhere,
// and what happens to few lanes of few warps (a bad record, a step beyond a
// cell, a released pair) is behind a vote.  The record is written, or put in
// the queue of leavers, before its current is deposited, so that the
// momentum's registers are free by then.  Measured on a 128 x 128 x 256 slab
// (33.6M electrons, gamma = 13): half of them still paired 1245 -> 955 us a
// launch, all paired 703 -> 487 us (57% of the DRAM rate), from 1054M to 702M
// and 503M to 362M warp instructions.
template <typename real, int DIM, int S, int TX, int TY, int TZ, bool REL, int SPLIT = 1>
__device__ __forceinline__ void push_tile(const PushArgs<real> &a, const int64_t t, unsigned char *smem_raw)
{
    const Geom &g = a.g;
    // tile shape and shared-tile extents are compile-time constants, so every
    // stencil offset below folds into an immediate
    constexpr int FL = 1, FH = S;        // field guards below / above the tile
    constexpr int JL = S, JH = S + 1;    // current guards below / above the tile
    constexpr int FX = TX + FL + FH, FY = DIM == 3 ? TY + FL + FH : 1, FZ = TZ + FL + FH;
    constexpr int QX = TX + JL + JH, QY = DIM == 3 ? TY + JL + JH : 1, QZ = TZ + JL + JH;
    constexpr int FN = FX * FY * FZ, QN = QX * QY * QZ;
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int kBlock = BlockOf<real, DIM>::value;
    using acc_t = typename Acc<real>::type;
    using R = Rec<real, DIM, true, REL>;
    using RI = Rec<real, DIM, false, false>;
    constexpr int ES = (int)sizeof(real);
    // arithmetic of the deposit: pairs of FP32 words for records in relative
    // form (FP64 in the debug path)
    using dep_t = typename std::conditional<REL && sizeof(real) == 4, ff, real>::type;
    unsigned char *wbuf = smem_raw + (threadIdx.x >> 5) * warp_bytes<R>();
    unsigned char *q = wbuf + R::RB;
    int *qmove = reinterpret_cast<int *>(q + R::RB), *qslot = qmove + 32;
    constexpr int JB = j_tile_bytes<real>(3 * QN);
    acc_t *sJ = reinterpret_cast<acc_t *>(smem_raw + (kBlock / 32) * warp_bytes<R>());
    real *sF = reinterpret_cast<real *>(reinterpret_cast<unsigned char *>(sJ) + JB);
    __shared__ int s_stay, s_stay_i;
    // the plasma drift and its displacement per step (the drifting ions')
    const Drift<real> drift(a.u_drift, a.dtdh[2]);
    const real dz_drift = drift.dz;

    int n_lo, n_hi;
    bucket_counts(a.in_lo, a.in_hi, t, g.cap, n_lo, n_hi, a.err);
    // uniform over the CTA
    if (n_lo + n_hi == 0 && !(a.fuse_ions && a.ions.in_lo[t] + a.ions.in_hi[t] > 0)) return;
    const int lane = lane_reg();
    const unsigned lt = lanemask_lt_reg();
    const Blocks bl(n_lo, n_hi, g.cap);
    const TilePos<DIM, TX, TY, TZ> tp(g, t);
    const int64_t bucket = (int64_t)(g.cap >> 5) * R::RB;
    const unsigned char *in = reinterpret_cast<const unsigned char *>(a.in.ox) + t * bucket + lane * 16;
    unsigned char *out = reinterpret_cast<unsigned char *>(a.out.ox) + t * bucket;
    const int kbit = g.bx + g.by;
    unsigned char *fbuf = wbuf + lane * 16, *rbuf = wbuf + lane * ES;

    const int rank = SPLIT > 1 ? (int)cluster_rank() : 0;
    __syncthreads();  // previous tile finished with shared memory
    int i = rank * (kBlock / 32) + (int)(threadIdx.x >> 5), qn = 0;
    if (i < bl.n) fetch_block<R::RB>(fbuf, in + (int64_t)bl.block(i) * R::RB, lane);
    if (threadIdx.x == 0) s_stay = 0;
    // Ez, Bx, By live on half-integer z (bits 2, 3, 4)
    const bool staged_nonzero = stage_tile<real, DIM, 6, FX, FY, FZ, FL>(
        g, Ptr6<real>{a.E[0], a.E[1], a.E[2], a.B[0], a.B[1], a.B[2]}, 0x1Cu, sF, tp.lox, tp.loy, tp.loz);
    for (int z = threadIdx.x; z < JB / 16; z += kBlock) reinterpret_cast<int4 *>(sJ)[z] = make_int4(0, 0, 0, 0);
    const bool field_in_tile = __syncthreads_or(staged_nonzero) != 0;
    if (SPLIT > 1) cluster_sync<SPLIT>();  // the first CTA's counter is set
    bool deposited = false;

    // a record into slot s of the bucket at b
    auto put = [&](unsigned char *b, int s, real vox, real voy, real voz, real vw, real vux, real vuy, real vuz,
                   real vdx, real vdy, real vdz, uint32_t vword) {
        b += slot_off<R::RB, real>(s);
        at<real>(b, R::OX) = vox;
        if (DIM == 3) at<real>(b, R::OY) = voy;
        at<real>(b, R::OZ) = voz;
        at<real>(b, R::W) = vw;
        at<real>(b, R::UX) = vux;
        at<real>(b, R::UY) = vuy;
        at<real>(b, R::UZ) = vuz;
        if (REL) {
            at<real>(b, R::DLX) = vdx;
            if (DIM == 3) at<real>(b, R::DLY) = vdy;
            at<real>(b, R::DLZ) = vdz;
        }
        at<uint32_t>(ES == 4 ? b : b - (s & 31) * 4, R::CELL) = vword;
    };
    // the queue's records into the top runs of their tiles
    auto flush = [&]() {
        __syncwarp();
        int64_t dest = -1;
        uint32_t qw = 0;
        if (lane < qn) {
            qw = row<uint32_t>(q, R::CELL, lane);
            const int mv = qmove[lane];
            int ni, nj, nk;
            unpack_cell(g, (int32_t)qw, ni, nj, nk);
            ni += (mv & 15) - 4;
            nk += (mv >> 8) - 4;
            if (ni < 0) ni += g.nx; else if (ni >= g.nx) ni -= g.nx;
            if (DIM == 3) {
                nj += ((mv >> 4) & 15) - 4;
                if (nj < 0) nj += g.ny; else if (nj >= g.ny) nj -= g.ny;
            }
            bool alive = true;
            if (g.bc_z == 0) {
                if (nk < 0) nk += g.nz; else if (nk >= g.nz) nk -= g.nz;
            } else if (nk < 0 || nk >= g.nz) {
                alive = false;
            }
            if (alive) {
                dest = tile_of(g, ni, nj, nk);
                qw = (qw & kPaired) | (uint32_t)pack_cell(g, ni, nj, nk);
            }
        }
        const int r = g.cap - 1 - reserve_slot(a.out_hi, dest);
        if (dest >= 0) {
            if (r >= 0) {
                unsigned char *p = q + lane * ES;
                put(out + (dest - t) * bucket, r, at<real>(p, R::OX), DIM == 3 ? at<real>(p, R::OY) : real(0),
                    at<real>(p, R::OZ), at<real>(p, R::W), at<real>(p, R::UX), at<real>(p, R::UY), at<real>(p, R::UZ),
                    REL ? at<real>(p, R::DLX) : real(0), REL && DIM == 3 ? at<real>(p, R::DLY) : real(0),
                    REL ? at<real>(p, R::DLZ) : real(0), qw);
                if (a.out.id)
                    a.out.id[dest * (int64_t)g.cap + r] = a.in.id ? a.in.id[t * (int64_t)g.cap + qslot[lane]] : 0;
            } else {
                atomicOr(a.err, ERR_CAPACITY);
            }
        }
        __syncwarp();
        qn = 0;
    };

    while (i < bl.n) {  // uniform over the warp
        const int slot = bl.block(i) * 32 + lane;
        bool valid = bl.valid(slot);
        // ---- load (the prefetched block), then fetch the next block
        __pipeline_wait_prior(0);
        __syncwarp();
        uint32_t word = row<uint32_t>(wbuf, R::CELL, lane);
        real ox = at<real>(rbuf, R::OX), oy = DIM == 3 ? at<real>(rbuf, R::OY) : real(0), oz = at<real>(rbuf, R::OZ);
        real w = at<real>(rbuf, R::W);
        real ux = at<real>(rbuf, R::UX), uy = at<real>(rbuf, R::UY), uz = at<real>(rbuf, R::UZ);
        real dlx = 0, dly = 0, dlz = 0;
        if (REL) {
            dlx = at<real>(rbuf, R::DLX);
            dlz = at<real>(rbuf, R::DLZ);
            if (DIM == 3) dly = at<real>(rbuf, R::DLY);
        }
        __syncwarp();
        i += SPLIT * (kBlock / 32);
        if (i < bl.n) fetch_block<R::RB>(fbuf, in + (int64_t)bl.block(i) * R::RB, lane);
        bool paired = (int32_t)word < 0;
        word &= ~kPaired;
        int li, lj, lk;
        const bool here = tp.local(g, word, li, lj, lk);
        if (!__all_sync(kAll, valid && here)) {  // a run's end, or a record in the wrong bucket
            if (valid && !here) atomicOr(a.err, ERR_TILE);
            valid = valid && here;
            if (!valid) {
                ox = oy = oz = w = ux = uy = uz = dlx = dly = dlz = real(0);
                li = lj = lk = 0;
                paired = false;
            }
        }
        // relative form: reference offsets and the reference cell's shift
        // from the stored cell
        const real orx = ox, ory = oy, orz = oz;
        int rx = 0, ry = 0, rz = 0;
        if (REL) {
            ox = rel_actual(orx, dlx, rx);
            oz = rel_actual(orz, dlz, rz);
            if (DIM == 3) oy = rel_actual(ory, dly, ry);
        }
        // ---- gather E^n, B^n at x^n, Boris
        bool release = false;
        // a tile whose staged E and B are all zero gathers exactly zero
        // everywhere: Boris is then the identity and no pair is released
        if (field_in_tile) {
            real wxu[S + 1], wxh[S + 1], wyu[S + 1], wyh[S + 1], wzu[S + 1], wzh[S + 1];
            const int bxu = offset_weights<S>(ox, wxu) + li + FL;
            const int bxh = half_weights<S>(ox, wxh) + li + FL;
            const int bzu = offset_weights<S>(oz, wzu) + lk + FL;
            const int bzh = half_weights<S>(oz, wzh) + lk + FL;
            int byu = 0, byh = 0;
            if (DIM == 3) {
                byu = offset_weights<S>(oy, wyu) + lj + FL;
                byh = half_weights<S>(oy, wyh) + lj + FL;
            } else {
#pragma unroll
                for (int c = 0; c <= S; ++c) wyu[c] = wyh[c] = real(c == 0);
            }
            const real ex = gather_comp<DIM, S>(sF + 0 * FN, FX, FY, bxh, byu, bzu, wxh, wyu, wzu);
            const real ey = gather_comp<DIM, S>(sF + 1 * FN, FX, FY, bxu, byh, bzu, wxu, wyh, wzu);
            const real ez = gather_comp<DIM, S>(sF + 2 * FN, FX, FY, bxu, byu, bzh, wxu, wyu, wzh);
            const real bx = gather_comp<DIM, S>(sF + 3 * FN, FX, FY, bxu, byh, bzh, wxu, wyh, wzh);
            const real by = gather_comp<DIM, S>(sF + 4 * FN, FX, FY, bxh, byu, bzh, wxh, wyu, wzh);
            const real bz = gather_comp<DIM, S>(sF + 5 * FN, FX, FY, bxh, byh, bzu, wxh, wyh, wzu);
            // a paired electron that gathers a non-zero field leaves its
            // ion behind: the pair's current is no longer zero
            release = paired && !(ex == real(0) && ey == real(0) && ez == real(0) && bx == real(0) && by == real(0) &&
                                  bz == real(0));
            boris(ux, uy, uz, drift.U, ex, ey, ez, bx, by, bz, a.eps);
        }
        // ---- move
        real vx, vy;
        const real dvz = drift_velocity(drift, ux, uy, uz, vx, vy);
        real dx = vx * a.dtdh[0];
        real dy = DIM == 3 ? vy * a.dtdh[1] : real(0);
        // the drift's displacement (the ions' own) plus the record's
        // departure from it
        real ddz = dvz * a.dtdh[2];
        {
            const real dz = dz_drift + ddz;
            const bool ok = fabs(dx) < real(1) && fabs(dy) < real(1) && fabs(dz) < real(1);
            if (!__all_sync(kAll, ok)) {
                if (!ok) {
                    if (valid) atomicOr(a.err, (dx == dx && dy == dy && dz == dz) ? ERR_CFL : ERR_NAN);
                    valid = release = false;
                    dx = dy = ddz = real(0);
                }
            }
        }
        // new offsets nox .. and the new cell relative to the old (mx ..);
        // relative form: new departures, and the shift of the reference cell
        // at the path's end (rx1 ..), relative to the old cell; else the end
        // of the path and its cell (fx ..)
        real nox, noy = 0, noz, dlx1 = 0, dly1 = 0, dlz1 = 0;
        real x1 = 0, y1 = 0, z1 = 0, fx = 0, fy = 0, fz = 0;
        int mx, my = 0, mz;
        int rx1 = 0, ry1 = 0, rz1 = 0;
        if (REL) {
            // across z the reference stays, the departure moves
            int f, r1;
            dlx1 = rel_step(dlx, dx, f);
            (void)rel_actual(orx, dlx1, r1);
            mx = rx + f - r1;
            rx1 = rx + f;
            if (DIM == 3) {
                dly1 = rel_step(dly, dy, f);
                (void)rel_actual(ory, dly1, r1);
                my = ry + f - r1;
                ry1 = ry + f;
            }
            // along z the reference moves exactly like a drifting ion
            // (same rounding, same cell changes)
            real sref = add_rn(orz, dz_drift);
            int sr = 0;
            if (sref < real(0)) {
                sref = sref + real(1);
                sr = -1;
                if (sref >= real(1)) { sref = 0; sr = 0; }
            } else if (sref >= real(1)) {
                sref = sref - real(1);
                sr = 1;
            }
            dlz1 = rel_step(dlz, ddz, f);
            (void)rel_actual(sref, dlz1, r1);
            mz = rz + sr + f - r1;
            rz1 = rz + sr + f;
            nox = orx;  // x, y references do not move
            noy = ory;
            noz = sref;
        } else {
            x1 = ox + dx;
            y1 = oy + dy;
            z1 = add_rn(oz, dz_drift) + ddz;
            // an offset that rounds to 1 moves on
            fx = floor(x1);
            nox = x1 - fx;
            mx = (int)fx + (nox >= real(1) ? 1 : 0);
            nox = nox >= real(1) ? real(0) : nox;
            if (DIM == 3) {
                fy = floor(y1);
                noy = y1 - fy;
                my = (int)fy + (noy >= real(1) ? 1 : 0);
                noy = noy >= real(1) ? real(0) : noy;
            }
            fz = floor(z1);
            noz = z1 - fz;
            mz = (int)fz + (noz >= real(1) ? 1 : 0);
            noz = noz >= real(1) ? real(0) : noz;
        }
        // ---- released ion: a record at the pair's position x^n, in the ion
        // side the IONS phase of this step reads (it moves and deposits it)
        if (__any_sync(kAll, release)) {
            const int r = g.cap - 1 - reserve_slot(a.ion_in_hi, release ? t : -1);
            if (release) {
                if (r < 0) {
                    atomicOr(a.err, ERR_CAPACITY);
                } else {
                    // (a paired record sits on its reference: orx = ox, ...)
                    unsigned char *b = reinterpret_cast<unsigned char *>(a.ion_in.ox) +
                                       t * ((int64_t)(g.cap >> 5) * RI::RB) + slot_off<RI::RB, real>(r);
                    at<real>(b, RI::OX) = orx;
                    if (DIM == 3) at<real>(b, RI::OY) = ory;
                    at<real>(b, RI::OZ) = orz;
                    at<real>(b, RI::W) = w;
                    at<uint32_t>(ES == 4 ? b : b - (r & 31) * 4, RI::CELL) = word;
                    if (a.ion_in.id)
                        a.ion_in.id[t * (int64_t)g.cap + r] = a.in.id ? a.in.id[t * (int64_t)g.cap + slot] : 0;
                }
            }
        }
        const bool keep_pair = paired && !release;  // exactly zero net current
        const bool dep = valid && !keep_pair;
        // ---- write the record, or put it in the queue
        {
            const uint32_t pair_bit = keep_pair ? kPaired : 0u;
            const bool in_tile = (unsigned)(li + mx) < (unsigned)tp.ex && (unsigned)(lk + mz) < (unsigned)tp.ez &&
                                 (DIM == 2 || (unsigned)(lj + my) < (unsigned)tp.ey);
            const bool stay = valid && in_tile, leave = valid && !in_tile;
            const unsigned ms = __ballot_sync(kAll, stay), ml = __ballot_sync(kAll, leave);
            int bs = 0;
            if (lane == 0) bs = stay_add<SPLIT>(&s_stay, __popc(ms));
            bs = __shfl_sync(kAll, bs, 0) + __popc(ms & lt);
            if (stay) {
                uint32_t nw = word + (uint32_t)mx + ((uint32_t)mz << kbit);
                if (DIM == 3) nw += (uint32_t)my << g.bx;
                put(out, bs, nox, noy, noz, w, ux, uy, uz, dlx1, dly1, dlz1, nw | pair_bit);
                if (a.out.id)
                    a.out.id[t * (int64_t)g.cap + bs] = a.in.id ? a.in.id[t * (int64_t)g.cap + slot] : 0;
            }
            if (ml) {
                const int nl = __popc(ml);
                if (qn + nl > 32) flush();
                if (leave) {
                    const int e = qn + __popc(ml & lt);
                    unsigned char *p = q + e * ES;
                    at<real>(p, R::OX) = nox;
                    if (DIM == 3) at<real>(p, R::OY) = noy;
                    at<real>(p, R::OZ) = noz;
                    at<real>(p, R::W) = w;
                    at<real>(p, R::UX) = ux;
                    at<real>(p, R::UY) = uy;
                    at<real>(p, R::UZ) = uz;
                    if (REL) {
                        at<real>(p, R::DLX) = dlx1;
                        if (DIM == 3) at<real>(p, R::DLY) = dly1;
                        at<real>(p, R::DLZ) = dlz1;
                    }
                    row<uint32_t>(q, R::CELL, e) = word | pair_bit;
                    qmove[e] = (mx + 4) | ((my + 4) << 4) | ((mz + 4) << 8);
                    qslot[e] = slot;
                }
                qn += nl;
            }
        }
        // ---- Esirkepov current; the warp agrees on the windows' lengths
        if (!__any_sync(kAll, dep)) continue;
        deposited = true;
        // (the fixed-point factors are read from the parameters at each use:
        // held in registers they would cost spills here)
        const dep_t jx = dep_t(a.jfac[0]) * dep_t(w) * dep_t(a.fx_scale[0]);
        const dep_t jy = dep_t(a.jfac[1]) * dep_t(w) * dep_t(a.fx_scale[1]);
        const dep_t jz = dep_t(a.jfac[2]) * dep_t(w) * dep_t(a.fx_scale[2]);
        const dep_t jyv = dep_t(a.jyfac) * dep_t(w) * dep_t(vy) * dep_t(a.fx_scale[1]);
        if constexpr (S == 1 && !REL && ES == 4) {
            const bool z_only = DIM == 3 && __all_sync(kAll, !dep || (x1 == ox && y1 == oy));
            const unsigned sel = (__any_sync(kAll, dep && fx != 0.0f) ? 4u : 0u) |
                                 (DIM == 3 && __any_sync(kAll, dep && fy != 0.0f) ? 2u : 0u) |
                                 (__any_sync(kAll, dep && fz != 0.0f) ? 1u : 0u);
            if (dep)
                deposit_cic<DIM, QX, QY, QN>(z_only, sel, sJ, ox, x1 - fx, fx, li, oy, y1 - fy, fy, lj, oz, z1 - fz, fz, lk,
                                             jx, jy, jz, jyv, a.fx_lo[0]);
        } else {
            dep_t S0x[S + 2], DSx[S + 2], S0y[S + 2], DSy[S + 2], S0z[S + 2], DSz[S + 2];
            int ax = 0, ay = 0, az = 0;
            bool cx = false, cy = false, cz = false;
            if (dep) {
                if constexpr (REL) {
                    ax = esirk_rel<S>(rel_pos<dep_t>(rx, orx, dlx), rel_pos<dep_t>(rx1, orx, dlx1), S0x, DSx, cx) + li +
                         JL;
                    az = esirk_rel<S>(rel_pos<dep_t>(rz, orz, dlz), rel_pos<dep_t>(rz1, noz, dlz1), S0z, DSz, cz) + lk +
                         JL;
                    if (DIM == 3)
                        ay = esirk_rel<S>(rel_pos<dep_t>(ry, ory, dly), rel_pos<dep_t>(ry1, ory, dly1), S0y, DSy, cy) +
                             lj + JL;
                } else {
                    ax = esirk_axis_c<S, dep_t>(ox, x1, S0x, DSx, cx) + li + JL;
                    az = esirk_axis_c<S, dep_t>(oz, z1, S0z, DSz, cz) + lk + JL;
                    if (DIM == 3) ay = esirk_axis_c<S, dep_t>(oy, y1, S0y, DSy, cy) + lj + JL;
                }
            }
            const unsigned sel = (__any_sync(kAll, cx) ? 4u : 0u) | (__any_sync(kAll, cy) ? 2u : 0u) |
                                 (__any_sync(kAll, cz) ? 1u : 0u);
            // 3D: no lane moved in x or y (e.g. plasma the laser has not reached)
            const bool z_only =
                DIM == 3 && __all_sync(kAll, !dep || (REL ? (rx1 == rx && dlx1 == dlx && ry1 == ry && dly1 == dly)
                                                         : (x1 == ox && y1 == oy)));
            if (dep) {
                if (z_only) {
                    if (sel & 1u)
                        deposit_z<dep_t, acc_t, S, QX, QY, QN, S + 2>(sJ, S0x, S0y, S0z, DSz, ax, ay, az, jz,
                                                                      (dep_t)a.fx_lo[0]);
                    else
                        deposit_z<dep_t, acc_t, S, QX, QY, QN, S + 1>(sJ, S0x, S0y, S0z, DSz, ax, ay, az, jz,
                                                                      (dep_t)a.fx_lo[0]);
                } else {
                    deposit_sel<dep_t, acc_t, DIM, S, QX, QY, QN>(sel, sJ, S0x, DSx, S0y, DSy, S0z, DSz, ax, ay, az, jx,
                                                                  jy, jz, jyv, (dep_t)a.fx_lo[0]);
                }
            }
        }
    }
    if (qn) flush();
    deposited = __syncthreads_or(deposited) != 0 || SPLIT > 1;
    if (SPLIT > 1) cluster_sync<SPLIT>();  // every CTA's records are written
    // the drifting ions of the tile, into the same current tile
    if (a.fuse_ions)
        deposited |= ions_of_tile<real, DIM, S, TX, TY, TZ, 3 * QN, REL, SPLIT>(g, a.ions, t, tp, sJ + 2 * QN, wbuf, dz_drift,
                                                                          a.fx_scale[2], a.fx_lo[0], a.err, &s_stay_i);
    // flush the J tile: one global add per non-zero node
    if (deposited)
        flush_tile<real, DIM, 3, QX, QY, QZ, JL, SPLIT>(g, Ptr3<real>{a.J[0], a.J[1], a.J[2]}, 0x4u, sJ, a.fx_quant[0],
                                                 a.fx_quant[1], a.fx_quant[2], a.fx_lo[1], tp.lox, tp.loy, tp.loz);
    if (threadIdx.x == 0 && rank == 0) {
        a.out_lo[t] = s_stay;
        a.in_lo[t] = 0;
        a.in_hi[t] = 0;
    }
    if (SPLIT > 1) cluster_sync<SPLIT>();  // no CTA leaves while another reads its tile
}

// ------------------------------------------------------ drifting-ion tile

template <typename real, int DIM, int S, int TX, int TY, int TZ, bool REL>
__device__ __forceinline__ void ion_tile(const PushArgs<real> &a, const int64_t t, unsigned char *smem_raw)
{
    const Geom &g = a.g;
    constexpr int JL = S, JH = S + 1;
    constexpr int QX = TX + JL + JH, QY = DIM == 3 ? TY + JL + JH : 1, QZ = TZ + JL + JH;
    constexpr int QN = QX * QY * QZ, kBlock = BlockOf<real, DIM>::value;
    using acc_t = typename Acc<real>::type;
    using RI = Rec<real, DIM, false, false>;
    // the warps' buffers, then the Jz tile ("hi" and, in FP32, "lo" words)
    unsigned char *wbuf = smem_raw + (threadIdx.x >> 5) * warp_bytes<RI>();
    constexpr int JB = j_tile_bytes<real>(QN);
    acc_t *sJ = reinterpret_cast<acc_t *>(smem_raw + (kBlock / 32) * warp_bytes<RI>());
    const Drift<real> drift(a.u_drift, a.dtdh[2]);
    const real dz = drift.dz;
    const IonSide<real> &is = a.ions;
    __shared__ int s_stay;

    if (is.in_lo[t] + is.in_hi[t] == 0) return;  // uniform over the CTA
    const TilePos<DIM, TX, TY, TZ> tp(g, t);
    __syncthreads();
    for (int z = threadIdx.x; z < JB / 16; z += kBlock) reinterpret_cast<int4 *>(sJ)[z] = make_int4(0, 0, 0, 0);
    ions_of_tile<real, DIM, S, TX, TY, TZ, QN, REL, 1>(g, is, t, tp, sJ, wbuf, dz, a.fx_scale[2], a.fx_lo[0], a.err,
                                                    &s_stay);
    flush_tile<real, DIM, 1, QX, QY, QZ, JL, 1>(g, Ptr3<real>{a.J[2], a.J[2], a.J[2]}, 0x1u, sJ, a.fx_quant[2],
                                             a.fx_quant[2], a.fx_quant[2], a.fx_lo[1], tp.lox, tp.loy, tp.loz);
}

// the tile shapes the kernels are compiled for (pic_init_grid accepts these):
// 8 x 8 x 8 in 3D, and for CIC also 8 x 8 x 4; 16 x 16 in 2D, and for CIC
// also 32 x 8 and 8 x 32 (x, z)
constexpr int kTile3[3] = {8, 8, 8};
constexpr int kTile2[3] = {16, 1, 16};

template <typename real, int DIM, int S, int TX, int TY, int TZ, bool REL>
static size_t push_smem(bool ions)
{
    const int FN = (TX + 1 + S) * (DIM == 3 ? TY + 1 + S : 1) * (TZ + 1 + S);
    const int QN = (TX + 2 * S + 1) * (DIM == 3 ? TY + 2 * S + 1 : 1) * (TZ + 2 * S + 1);
    constexpr int warps = BlockOf<real, DIM>::value / 32;
    return ions ? (size_t)warps * warp_bytes<Rec<real, DIM, false, false>>() + j_tile_bytes<real>(QN)
                : (size_t)warps * warp_bytes<Rec<real, DIM, true, REL>>() + j_tile_bytes<real>(3 * QN) +
                      sizeof(real) * (size_t)(6 * FN);
}

// the batched particle launches (pic_batch.cu): a persistent grid over the
// (run, tile) items of all runs; IONS selects the drifting-ion kernel
template <typename real, int DIM, int S, int TX, int TY, int TZ, bool REL, bool IONS>
void launch_push_batch(const void *args, const int64_t *start, int n, int64_t total, unsigned *queue, cudaStream_t s);

}  // namespace pic
