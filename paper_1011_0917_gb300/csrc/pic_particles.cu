// pic_particles.cu -- particle kernels of a single run: fused gather / Boris
// push / Esirkepov deposit / re-bucketing per tile (bodies in pic_push.cuh),
// the drifting-ion deposit, bucketing of flat lists, compaction, charge
// density and particle sums.
#include "pic_push.cuh"

#include <algorithm>
#include <cmath>

namespace pic {

template <typename real, int DIM, int S, int TX, int TY, int TZ, bool REL>
__global__ void __launch_bounds__((BlockOf<real, DIM>::value), (MinBlocks<real, DIM>::value)) push_kernel(PushArgs<real> a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    chain_begin(a.g.early);
    for (int64_t t = blockIdx.x; t < a.g.ntiles; t += gridDim.x) push_tile<real, DIM, S, TX, TY, TZ, REL>(a, t, smem_raw);
}

// few tiles: kSplit CTAs per tile
template <typename real, int DIM, int S, int TX, int TY, int TZ, bool REL>
__global__ void __launch_bounds__((BlockOf<real, DIM>::value), (MinBlocks<real, DIM>::value))
    push_split_kernel(PushArgs<real> a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    chain_begin(a.g.early);
    push_tile<real, DIM, S, TX, TY, TZ, REL, kSplit>(a, (int64_t)(blockIdx.x / kSplit), smem_raw);
}

// ----------------------------------------------------- drifting-ion kernel

template <typename real, int DIM, int S, int TX, int TY, int TZ, bool REL>
__global__ void __launch_bounds__((BlockOf<real, DIM>::value)) ion_kernel(PushArgs<real> a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    chain_begin(a.g.early);
    for (int64_t t = blockIdx.x; t < a.g.ntiles; t += gridDim.x) ion_tile<real, DIM, S, TX, TY, TZ, REL>(a, t, smem_raw);
}

template <typename real, int DIM, int S, int TX, int TY, int TZ, bool REL>
static void launch_push_z(const PushArgs<real> &a, bool ions, cudaStream_t s)
{
    if (ions ? record_launch(kBPIons, launch_push_batch<real, DIM, S, TX, TY, TZ, REL, true>, a, a.g.ntiles, true)
             : record_launch(kBPPush, launch_push_batch<real, DIM, S, TX, TY, TZ, REL, false>, a, a.g.ntiles, true))
        return;
    const size_t smem = push_smem<real, DIM, S, TX, TY, TZ, REL>(ions);
    auto k = ions ? ion_kernel<real, DIM, S, TX, TY, TZ, REL> : push_kernel<real, DIM, S, TX, TY, TZ, REL>;
    if (smem > 48 * 1024) cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    // One CTA per tile, or kSplit (the default tile shapes) where the tiles are
    // fewer than the SMs or kSplit CTAs for each fit the CTAs per SM that the
    // kernel is compiled for (in 3D FP64 shared memory holds one of the two);
    // beyond that the tiles fill the device and splitting them repeats their
    // staging.  us per step, one CTA / kSplit: 2D 64 tiles 34.0 / 28.9, 200
    // tiles 34.3 / 31.5, 384 tiles 36.0 / 40.0; FP64 64 tiles 159 / 115; 3D 16
    // tiles 72 / 48, 96 tiles 74 / 63.  us per pass of thermal plasmas: FP64, 900
    // particles a tile, 96 tiles 1488 / 1067, 152 tiles 1069 / 1293; 3D 125 tiles
    // 422 / 387, 432 tiles 500 / 581.  (Other tile shapes, which a caller asks
    // for, are not compiled for it, to keep the kernels' number down: 32 x 8
    // tiles of 64 x 512 cells would gain 8%, 8 x 8 x 4 tiles nothing.)
    constexpr bool kDefaultTile = DIM == 3 ? TZ == 8 : TX == 16;
    if constexpr (kDefaultTile) {
        const int64_t sms = device_sms();
        if (!ions && (a.g.ntiles < sms || a.g.ntiles * kSplit <= sms * MinBlocks<real, DIM>::value)) {
            auto ks = push_split_kernel<real, DIM, S, TX, TY, TZ, REL>;
            if (smem > 48 * 1024) cudaFuncSetAttribute(ks, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            launch_clusters(kSplit, ks, (unsigned)(a.g.ntiles * kSplit), BlockOf<real, DIM>::value, smem, s, a);
            return;
        }
    }
    const int64_t grid = a.g.ntiles < 2147483647LL ? a.g.ntiles : 2147483647LL;
    launch_chained(k, (unsigned)grid, BlockOf<real, DIM>::value, smem, s, a);
}

// records in relative form (and their ions) take the REL kernels
template <typename real, int DIM, int S, int TX, int TY, int TZ>
static void launch_push_t(const PushArgs<real> &a, bool ions, cudaStream_t s)
{
    if (a.rel) launch_push_z<real, DIM, S, TX, TY, TZ, true>(a, ions, s);
    else launch_push_z<real, DIM, S, TX, TY, TZ, false>(a, ions, s);
}

template <typename real>
static void dispatch_push(const PushArgs<real> &a, bool ions, cudaStream_t s)
{
    if (a.g.dim == 3) {
        if (a.g.shape == 2) launch_push_t<real, 3, 2, kTile3[0], kTile3[1], kTile3[2]>(a, ions, s);
        else if (a.g.lt[2] == 2) launch_push_t<real, 3, 1, 8, 8, 4>(a, ions, s);  // 8 x 8 x 4
        else launch_push_t<real, 3, 1, kTile3[0], kTile3[1], kTile3[2]>(a, ions, s);
    } else if (a.g.shape == 2) {
        launch_push_t<real, 2, 2, kTile2[0], kTile2[1], kTile2[2]>(a, ions, s);
    } else if (a.g.lt[0] == 5) {  // 32 x 8
        launch_push_t<real, 2, 1, 32, 1, 8>(a, ions, s);
    } else if (a.g.lt[0] == 3) {  // 8 x 32
        launch_push_t<real, 2, 1, 8, 1, 32>(a, ions, s);
    } else {
        launch_push_t<real, 2, 1, kTile2[0], kTile2[1], kTile2[2]>(a, ions, s);
    }
}

template <typename real> void launch_push(const PushArgs<real> &a, cudaStream_t s) { dispatch_push(a, false, s); }
template <typename real> void launch_ions(const PushArgs<real> &a, cudaStream_t s) { dispatch_push(a, true, s); }

// --------------------------------------------------------- moving window

// One CTA per output tile: it copies the bucket of the input tile m layers
// above (same slots, both runs) with the cell index S = m tz lower; the top m
// layers are left empty and the bottom m layers of the input are dropped.
template <typename real>
__global__ void window_particles_kernel(Geom g, Species<real> in, Species<real> out, const int *in_lo,
                                        const int *in_hi, int *out_lo, int *out_hi, int m, int S)
{
    const int64_t ntxy = (int64_t)g.nt[0] * g.nt[1];
    const int64_t t = blockIdx.x;
    const int64_t tz = t / ntxy;
    int n_lo = 0, n_hi = 0;
    if (tz + m < g.nt[2]) bucket_counts(in_lo, in_hi, t + m * ntxy, g.cap, n_lo, n_hi, nullptr);
    if (threadIdx.x == 0) {
        out_lo[t] = n_lo;
        out_hi[t] = n_hi;
    }
    const int n = n_lo + n_hi;
    const uint32_t dk = (uint32_t)S << (g.bx + g.by);
    for (int p = threadIdx.x; p < n; p += blockDim.x) {
        const int64_t d0 = bucket_slot(t, g.cap, n_lo, n_hi, p);
        const int64_t s0 = d0 + m * ntxy * (int64_t)g.cap;
        const int64_t d = out.r(d0), s = in.r(s0);
        out.ox[d] = in.ox[s];
        if (g.dim == 3) out.oy[d] = in.oy[s];
        out.oz[d] = in.oz[s];
        out.w[d] = in.w[s];
        if (in.ux) {
            out.ux[d] = in.ux[s];
            out.uy[d] = in.uy[s];
            out.uz[d] = in.uz[s];
        }
        if (in.dlx) {
            out.dlx[d] = in.dlx[s];
            if (in.dly) out.dly[d] = in.dly[s];
            out.dlz[d] = in.dlz[s];
        }
        out.cell[out.c(d0)] = (int32_t)((uint32_t)in.cell[in.c(s0)] - dk);  // keeps the pair bit
        if (in.id) out.id[d0] = in.id[s0];
    }
}

template <typename real>
void launch_window_particles(const Geom &g, const Species<real> &in, const Species<real> &out, const int *in_lo,
                             const int *in_hi, int *out_lo, int *out_hi, int m, int S, cudaStream_t s)
{
    window_particles_kernel<real><<<(unsigned)g.ntiles, 256, 0, s>>>(g, in, out, in_lo, in_hi, out_lo, out_hi, m, S);
}

// ------------------------------------------------------ bucket / compact

// A warp takes kBucketRun runs of 32 consecutive records.  A list that was
// compacted tile by tile (a snapshot) has nearly all of them in one tile:
// then one atomic reserves the slots of all runs, and every attribute's loads
// are in flight together (one run at a time waited for an atomic per 32
// records: 4.5 ms for the 268M electrons of 256 x 256 x 512 cells, whose 17 GB
// take 2.6).
constexpr int kBucketRun = 4;

template <typename real>
__global__ void __launch_bounds__(256) bucket_kernel(BucketArgs<real> a)
{
    constexpr int U = kBucketRun;
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = (int)(threadIdx.x & 31u);
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t w = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); w * 32 * U < a.n; w += warps) {
        const int64_t p0 = w * 32 * U + lane;
        int32_t cell[U];
        int64_t slot[U];  // of the record in the store, -1: none
#pragma unroll
        for (int u = 0; u < U; ++u) cell[u] = p0 + 32 * u < a.n ? a.src.cell[p0 + 32 * u] : 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            int ci, cj, ck;
            unpack_cell(a.g, cell[u], ci, cj, ck);
            slot[u] = p0 + 32 * u < a.n ? tile_of(a.g, ci, cj, ck) : -1;
        }
        const int64_t tile = __shfl_sync(kAll, slot[0], 0);
        bool same = true;
#pragma unroll
        for (int u = 0; u < U; ++u) same = same && slot[u] == tile;
        int bucket[U];  // place in the top run
        if (__all_sync(kAll, same)) {
            int b = 0;
            if (lane == 0) b = atomicAdd(&a.dst_hi[tile], 32 * U);
            b = __shfl_sync(kAll, b, 0) + lane;
#pragma unroll
            for (int u = 0; u < U; ++u) bucket[u] = b + 32 * u;
        } else {
#pragma unroll
            for (int u = 0; u < U; ++u) bucket[u] = reserve_slot(a.dst_hi, slot[u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (slot[u] >= 0 && bucket[u] >= a.g.cap) {
                atomicOr(a.err, ERR_CAPACITY);
                slot[u] = -1;
            }
            if (slot[u] >= 0) slot[u] = slot[u] * (int64_t)a.g.cap + (a.g.cap - 1 - bucket[u]);
        }
        auto copy = [&](real *dst, const real *src) {
            if (!dst) return;
            real v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) v[u] = slot[u] >= 0 ? src[p0 + 32 * u] : real(0);
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (slot[u] >= 0) dst[a.dst.r(slot[u])] = v[u];
        };
        copy(a.dst.ox, a.src.ox);
        copy(a.dst.oy, a.src.oy);
        copy(a.dst.oz, a.src.oz);
        copy(a.dst.w, a.src.w);
        copy(a.dst.ux, a.src.ux);
        copy(a.dst.uy, a.src.uy);
        copy(a.dst.uz, a.src.uz);
        copy(a.dst.dlx, a.src.dlx);
        copy(a.dst.dly, a.src.dly);
        copy(a.dst.dlz, a.src.dlz);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (slot[u] < 0) continue;
            a.dst.cell[a.dst.c(slot[u])] = cell[u];
            if (a.dst.id) a.dst.id[slot[u]] = a.src.id ? a.src.id[p0 + 32 * u] : 0;
        }
    }
}

template <typename real>
void launch_bucket(const BucketArgs<real> &a, cudaStream_t s)
{
    if (a.n <= 0) return;
    int64_t blocks = (a.n + 256 * kBucketRun - 1) / (256 * kBucketRun);
    if (blocks > (int64_t)device_sms() * 64) blocks = (int64_t)device_sms() * 64;
    bucket_kernel<real><<<(unsigned)blocks, 256, 0, s>>>(a);
}

template <typename real>
__global__ void compact_kernel(CompactArgs<real> a)
{
    for (int64_t t = blockIdx.x; t < a.g.ntiles; t += gridDim.x) {
        int n_lo, n_hi;
        bucket_counts(a.lo, a.hi, t, a.g.cap, n_lo, n_hi, nullptr);
        const int n = n_lo + n_hi;
        const int64_t o = a.offset[t];
        for (int p = threadIdx.x; p < n; p += blockDim.x) {
            const int64_t s0 = bucket_slot(t, a.g.cap, n_lo, n_hi, p), s = a.src.r(s0), d = o + p;
            a.dst.ox[d] = a.src.ox[s];
            if (a.src.oy) a.dst.oy[d] = a.src.oy[s];
            a.dst.oz[d] = a.src.oz[s];
            a.dst.w[d] = a.src.w[s];
            if (a.src.ux) {
                a.dst.ux[d] = a.src.ux[s];
                a.dst.uy[d] = a.src.uy[s];
                a.dst.uz[d] = a.src.uz[s];
            }
            if (a.src.dlx) {
                a.dst.dlx[d] = a.src.dlx[s];
                if (a.src.dly) a.dst.dly[d] = a.src.dly[s];
                a.dst.dlz[d] = a.src.dlz[s];
            }
            a.dst.cell[d] = a.src.cell[a.src.c(s0)];
            if (a.src.id) a.dst.id[d] = a.src.id[s0];
        }
    }
}

template <typename real>
void launch_compact(const CompactArgs<real> &a, cudaStream_t s)
{
    const int64_t grid = a.g.ntiles < 1048576 ? a.g.ntiles : 1048576;
    if (grid > 0) compact_kernel<real><<<(unsigned)grid, 256, 0, s>>>(a);
}

// ------------------------------------------------------------ cell order

// Counting sort of every tile's bucket by cell -- the cell's index inside
// its tile, x fastest, then y, then z -- into the bottom run of the same
// tile on the other side of the double buffer.  One CTA per tile: a
// histogram of the cells in shared memory, its exclusive scan, then every
// record copied to its cell's next slot (the order inside a cell is the
// order of the slot claims, which the results of a step do not depend on).
// A bucket of more than kSortKeys records is copied in its own order.
constexpr int kSortKeys = 8192;
constexpr int kSortCells = 512;  // the largest compiled tile (8 x 8 x 8, 16 x 16, 32 x 8)

template <typename real>
__global__ void __launch_bounds__(256) sort_cells_kernel(SortArgs<real> a)
{
    __shared__ int cnt[kSortCells];
    __shared__ unsigned short key[kSortKeys];
    __shared__ int wsum[8];
    const Geom &g = a.g;
    const int ncell = 1 << (g.lt[0] + g.lt[1] + g.lt[2]);
    const int tid = (int)threadIdx.x;
    for (int64_t t = blockIdx.x; t < g.ntiles; t += gridDim.x) {
        int n_lo, n_hi;
        bucket_counts(a.in_lo, a.in_hi, t, g.cap, n_lo, n_hi, a.err);
        const int n = n_lo + n_hi;
        const int tix = (int)(t % g.nt[0]);
        const int tiy = (int)((t / g.nt[0]) % g.nt[1]);
        const int tiz = (int)(t / ((int64_t)g.nt[0] * g.nt[1]));
        const int lox = tix << g.lt[0], loy = tiy << g.lt[1], loz = tiz << g.lt[2];
        const bool sorted = n <= kSortKeys;
        __syncthreads();  // the previous tile is done with shared memory
        for (int q = tid; q < ncell; q += blockDim.x) cnt[q] = 0;
        __syncthreads();
        if (sorted) {
            for (int p = tid; p < n; p += blockDim.x) {
                int ci, cj, ck;
                unpack_cell(g, a.in.cell[a.in.c(bucket_slot(t, g.cap, n_lo, n_hi, p))], ci, cj, ck);
                int li = ci - lox, lj = cj - loy, lk = ck - loz;
                if (li < 0 || li >= (1 << g.lt[0]) || lj < 0 || lj >= (1 << g.lt[1]) || lk < 0 ||
                    lk >= (1 << g.lt[2])) {
                    atomicOr(a.err, ERR_TILE);
                    li = lj = lk = 0;
                }
                const int lc = (((lk << g.lt[1]) | lj) << g.lt[0]) | li;
                key[p] = (unsigned short)lc;
                atomicAdd(&cnt[lc], 1);
            }
            __syncthreads();
            // exclusive scan of the counts: each thread two cells, then the
            // warps' totals
            const int c0 = 2 * tid, v0 = c0 < ncell ? cnt[c0] : 0, v1 = c0 + 1 < ncell ? cnt[c0 + 1] : 0;
            int x = v0 + v1;
            const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if ((int)lane >= o) x += y;
            }
            if (lane == 31) wsum[warp] = x;
            __syncthreads();
            int before = 0;
            for (unsigned w = 0; w < warp; ++w) before += wsum[w];
            const int excl = before + x - (v0 + v1);
            __syncthreads();  // every count has been read
            if (c0 < ncell) cnt[c0] = excl;
            if (c0 + 1 < ncell) cnt[c0 + 1] = excl + v0;
            __syncthreads();
        }
        for (int p = tid; p < n; p += blockDim.x) {
            const int64_t s0 = bucket_slot(t, g.cap, n_lo, n_hi, p), s = a.in.r(s0);
            const int64_t d0 = t * (int64_t)g.cap + (sorted ? atomicAdd(&cnt[key[p]], 1) : p), d = a.out.r(d0);
            // (all of a record's loads before its stores, which might alias them)
            const real ox = a.in.ox[s], oy = a.in.oy ? a.in.oy[s] : real(0), oz = a.in.oz[s], w = a.in.w[s];
            real ux = 0, uy = 0, uz = 0, dlx = 0, dly = 0, dlz = 0;
            const int32_t cell = a.in.cell[a.in.c(s0)];
            if (a.in.ux) {
                ux = a.in.ux[s];
                uy = a.in.uy[s];
                uz = a.in.uz[s];
            }
            if (a.in.dlx) {
                dlx = a.in.dlx[s];
                dly = a.in.dly ? a.in.dly[s] : real(0);
                dlz = a.in.dlz[s];
            }
            a.out.ox[d] = ox;
            if (a.in.oy) a.out.oy[d] = oy;
            a.out.oz[d] = oz;
            a.out.w[d] = w;
            if (a.in.ux) {
                a.out.ux[d] = ux;
                a.out.uy[d] = uy;
                a.out.uz[d] = uz;
            }
            if (a.in.dlx) {
                a.out.dlx[d] = dlx;
                if (a.in.dly) a.out.dly[d] = dly;
                a.out.dlz[d] = dlz;
            }
            a.out.cell[a.out.c(d0)] = cell;
            if (a.in.id) a.out.id[d0] = a.in.id[s0];
        }
        if (tid == 0) {
            a.out_lo[t] = n;
            a.in_lo[t] = 0;
            a.in_hi[t] = 0;
        }
    }
}

template <typename real>
void launch_sort_cells(const SortArgs<real> &a, cudaStream_t s)
{
    const int64_t grid = a.g.ntiles < 1048576 ? a.g.ntiles : 1048576;
    if (grid > 0) sort_cells_kernel<real><<<(unsigned)grid, 256, 0, s>>>(a);
}

// ------------------------------------------------------- charge density

template <typename real, int DIM, int S>
__global__ void rho_kernel(Geom g, Species<real> sp, const int *lo, const int *hi, real qfac, real *rho)
{
    for (int64_t t = blockIdx.x; t < g.ntiles; t += gridDim.x) {
        int n_lo, n_hi;
        bucket_counts(lo, hi, t, g.cap, n_lo, n_hi, nullptr);
        const int n = n_lo + n_hi;
        for (int p = threadIdx.x; p < n; p += blockDim.x) {
            const int64_t s0 = bucket_slot(t, g.cap, n_lo, n_hi, p), s = sp.r(s0);
            const int32_t word = sp.cell[sp.c(s0)];
            if ((uint32_t)word & kPaired) continue;  // with its ion: no net charge
            int ci, cj, ck;
            unpack_cell(g, word, ci, cj, ck);
            real wx[S + 1], wy[S + 1], wz[S + 1];
            real ox = sp.ox[s], oy = DIM == 3 ? sp.oy[s] : real(0), oz = sp.oz[s];
            if (sp.dlx) {  // relative form: the offsets in the stored cell
                int r;
                ox = rel_actual(ox, sp.dlx[s], r);
                oz = rel_actual(oz, sp.dlz[s], r);
                if (DIM == 3) oy = rel_actual(oy, sp.dly[s], r);
            }
            const int bx = spline_weights<S>(ox, wx) + ci;
            const int bz = spline_weights<S>(oz, wz) + ck;
            int by = 0;
            if (DIM == 3) by = spline_weights<S>(oy, wy) + cj;
            const real q = qfac * sp.w[s];
            for (int c = 0; c <= S; ++c) {
                int k = bz + c;
                if (g.bc_z == 0) k = wrapi(k, g.nz);
                else if (k < 0 || k > g.nz) continue;
                for (int b = 0; b < (DIM == 3 ? S + 1 : 1); ++b) {
                    const int j = DIM == 3 ? wrapi(by + b, g.ny) : 0;
                    for (int a = 0; a <= S; ++a) {
                        const int i = wrapi(bx + a, g.nx);
                        const real wt = DIM == 3 ? wx[a] * wy[b] * wz[c] : wx[a] * wz[c];
                        atomicAdd(rho + fidx(g, i, j, k), q * wt);
                    }
                }
            }
        }
    }
}

template <typename real>
void launch_rho(const Geom &g, const Species<real> &sp, const int *lo, const int *hi, real qfac, real *rho,
                cudaStream_t s)
{
    const int64_t grid = g.ntiles < 1048576 ? g.ntiles : 1048576;
    if (grid <= 0) return;
    if (g.dim == 3) {
        if (g.shape == 1) rho_kernel<real, 3, 1><<<(unsigned)grid, 128, 0, s>>>(g, sp, lo, hi, qfac, rho);
        else rho_kernel<real, 3, 2><<<(unsigned)grid, 128, 0, s>>>(g, sp, lo, hi, qfac, rho);
    } else {
        if (g.shape == 1) rho_kernel<real, 2, 1><<<(unsigned)grid, 128, 0, s>>>(g, sp, lo, hi, qfac, rho);
        else rho_kernel<real, 2, 2><<<(unsigned)grid, 128, 0, s>>>(g, sp, lo, hi, qfac, rho);
    }
}

// -------------------------------------------------------- particle sums

// Compensated FP64 partial sums per block: [0] sum w (gamma-1), [1] sum q w (a
// paired electron and its ion carry no net charge), [2] the number of paired
// electrons, [3] the number of records (negative: a bucket overflowed).  The
// host adds the block partials, also with compensation.
// Records at rest relative to the drift (all ions; the electrons no field has
// reached, most of a boosted plasma) share one gamma - 1, rest_ke: only their
// weights are summed.  (256 x 8192 cells, 8.4M electrons, 6% of them moving: 324 us
// per species with the FP64 kinetic energy of every record.)
// run_len: records whose weights a thread adds between two flushes, at most
// kSumRun (fewer for weights whose sums would leave the FP32 range)
template <typename real>
__global__ void particle_sums_kernel(Geom g, Species<real> sp, const int *lo, const int *hi, double q, double iuz,
                                     double rest_ke, int run_len, double *partials)
{
    RunSum<real> rest, charge;
    Kahan moving;
    unsigned npair = 0;
    int run = 0;
    double records = 0;
    unsigned overflow = 0;
    for (int64_t t = blockIdx.x; t < g.ntiles; t += gridDim.x) {
        int n_lo, n_hi;
        bucket_counts(lo, hi, t, g.cap, n_lo, n_hi, nullptr);
        if (hi[t] > n_hi) overflow = 1;  // (clamped: the runs meet)
        const int n = n_lo + n_hi;
        if (threadIdx.x == 0) records += n;
        for (int p = threadIdx.x; p < n; p += blockDim.x) {
            const int64_t slot = bucket_slot(t, g.cap, n_lo, n_hi, p), s = sp.r(slot);
            const real w = sp.w[s];
            const bool pair = ((uint32_t)sp.cell[sp.c(slot)] & kPaired) != 0u;
            real ux = 0, uy = 0, uz = 0;  // records hold u - u_drift
            if (sp.ux) {
                ux = sp.ux[s];
                uy = sp.uy[s];
                uz = sp.uz[s];
            }
            npair += pair ? 1u : 0u;
            if (!pair) charge.add(w);
            if (ux == real(0) && uy == real(0) && uz == real(0)) {
                rest.add(w);
            } else {
                const double vx = (double)ux, vy = (double)uy, vz = iuz + (double)uz;
                const double u2 = vx * vx + vy * vy + vz * vz;
                moving.add((double)w * (u2 / (sqrt(1.0 + u2) + 1.0)));  // gamma - 1 without cancellation
            }
            if (++run == run_len) {
                rest.flush();
                charge.flush();
                run = 0;
            }
        }
    }
    rest.flush();
    charge.flush();
    __shared__ double red[2][256];
    __shared__ unsigned pairs;
    red[0][threadIdx.x] = moving.value() + rest_ke * rest.k.value();
    red[1][threadIdx.x] = q * charge.k.value();
    if (threadIdx.x == 0) pairs = 0;
    __syncthreads();
    npair = __reduce_add_sync(0xffffffffu, npair);
    if ((threadIdx.x & 31u) == 0u) atomicAdd(&pairs, npair);
    for (int off = blockDim.x / 2; off > 0; off >>= 1) {
        if ((int)threadIdx.x < off) {
            red[0][threadIdx.x] += red[0][threadIdx.x + off];
            red[1][threadIdx.x] += red[1][threadIdx.x + off];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        partials[4 * blockIdx.x] = red[0][0];
        partials[4 * blockIdx.x + 1] = red[1][0];
        partials[4 * blockIdx.x + 2] = (double)pairs;
        partials[4 * blockIdx.x + 3] = overflow ? -1.0 : records;
    }
}

// returns the blocks whose partials (4 each) it writes: four per SM at most
// (an idle block costs FP64 additions too)
template <typename real>
int launch_particle_sums(const Geom &g, const Species<real> &sp, const int *lo, const int *hi, double q, real u_drift,
                         double wmax, double *partials, int max_blocks, cudaStream_t s)
{
    const int64_t cap = std::min<int64_t>(max_blocks, (int64_t)device_sms() * 4);
    const int nblocks = (int)std::min(cap, g.ntiles);
    const double u = (double)u_drift;
    particle_sums_kernel<real><<<nblocks, 256, 0, s>>>(g, sp, lo, hi, q, u, u * u / (std::sqrt(1.0 + u * u) + 1.0),
                                                       wmax * kSumRun < 1e38 ? kSumRun : 1, partials);
    return nblocks;
}

#define PIC_INSTANTIATE(real)                                                                       \
    template void launch_push<real>(const PushArgs<real> &, cudaStream_t);                          \
    template void launch_window_particles<real>(const Geom &, const Species<real> &, const Species<real> &, \
                                                const int *, const int *, int *, int *, int, int, cudaStream_t); \
    template void launch_ions<real>(const PushArgs<real> &, cudaStream_t);                          \
    template void launch_bucket<real>(const BucketArgs<real> &, cudaStream_t);                      \
    template void launch_compact<real>(const CompactArgs<real> &, cudaStream_t);                    \
    template void launch_sort_cells<real>(const SortArgs<real> &, cudaStream_t);                    \
    template void launch_rho<real>(const Geom &, const Species<real> &, const int *, const int *, real, \
                                   real *, cudaStream_t);                                            \
    template int launch_particle_sums<real>(const Geom &, const Species<real> &, const int *,      \
                                             const int *, double, real, double, double *, int, \
                                             cudaStream_t);
PIC_INSTANTIATE(float)
PIC_INSTANTIATE(double)

}  // namespace pic
