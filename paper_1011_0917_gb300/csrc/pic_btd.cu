// pic_btd.cu -- lab-frame ("back-transformed") snapshots of a boosted run.
//
// After the Yee update of step n both (E^n, B^n) and (E^{n+1}, B^{n+1}) are
// in memory (the two field buffers).  Every lab snapshot point (T_j, Z_k)
// whose simulation-frame event time t' = gamma (T - beta Z) lies in
// [t'^n, t'^{n+1}) is filled now: the fields at z' = gamma (Z - beta T),
// linear in z' between the planes of each component and linear in t' between
// the two times, transformed to the lab frame (the simulation frame moves at
// +beta along z):
//   Ex = gamma (Ex' + beta By'),  Ey = gamma (Ey' - beta Bx'),  Ez = Ez',
//   Bx = gamma (Bx' - beta Ey'),  By = gamma (By' + beta Ex'),  Bz = Bz'.
// Event times, heights and weights are FP64 and this file is compiled without
// FMA contraction, so which points a step fills is decided exactly as the
// FP64 reference decides it.
#include "pic_internal.cuh"

namespace pic {

template <typename real>
__global__ void btd_kernel(BtdArgs<real> a)
{
    chain_begin(a.g.early);
    const int js = (int)blockIdx.y;
    const int idx = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    const int kk = idx / a.nxs, is = idx - kk * a.nxs;
    if (kk >= a.kn[js]) return;
    const int k = a.klo[js] + kk;
    const Geom &g = a.g;
    const double T = a.T0 + js * a.dT;
    const double Z = a.Z0 + k * a.dZ;
    const double tp = a.gam * (T - a.beta * Z);
    if (!(tp >= a.t0 && tp < a.t0 + a.dt)) return;
    const double zp = a.gam * (Z - a.beta * T) - a.zwin;
    const double th = (tp - a.t0) / a.dt;
    const int i = a.nxs == 1 ? g.nx / 2 : is;
    const int jc = g.ny / 2;
    real v[6];
    for (int c = 0; c < 6; ++c) {
        // Ez, Bx, By sit half a cell up in z
        const double sz = (c == 2 || c == 3 || c == 4) ? 0.5 : 0.0;
        const double u = zp / a.hz - sz;
        const double k0 = floor(u);
        const double fz = u - k0;
        const int zmax = g.bc_z == 0 ? g.nz - 1 : (sz > 0.0 ? g.nz - 1 : g.nz);
        if (k0 < 0.0 || k0 + 1.0 > (double)zmax) return;  // the same for every column
        const int64_t o0 = fidx(g, i, jc, (int)k0), o1 = o0 + g.plane;
        const real *F0 = c < 3 ? a.E0[c] : a.B0[c - 3];
        const real *F1 = c < 3 ? a.E1[c] : a.B1[c - 3];
        const real w0 = (real)(1.0 - fz), w1 = (real)fz;
        const real f0 = w0 * F0[o0] + w1 * F0[o1];
        const real f1 = w0 * F1[o0] + w1 * F1[o1];
        v[c] = (real)(1.0 - th) * f0 + (real)th * f1;
    }
    const real gam = (real)a.gam, beta = (real)a.beta;
    const real lab[6] = {gam * (v[0] + beta * v[4]), gam * (v[1] - beta * v[3]), v[2],
                         gam * (v[3] - beta * v[1]), gam * (v[4] + beta * v[0]), v[5]};
    real *d = a.data + (size_t)js * 6 * a.nz * a.nxs;
    for (int c = 0; c < 6; ++c) d[((size_t)c * a.nz + k) * a.nxs + is] = lab[c];
    if (is == 0) a.flags[(size_t)js * a.nz + k] = 1;
}

template <typename real>
void launch_btd(const BtdArgs<real> &a, cudaStream_t s)
{
    int span = 0;
    for (int j = 0; j < a.nsnap; ++j) span = a.kn[j] > span ? a.kn[j] : span;
    if (span == 0) return;
    const int64_t n = (int64_t)span * a.nxs;
    dim3 grid((unsigned)((n + 255) / 256), (unsigned)a.nsnap);
    btd_kernel<real><<<grid, 256, 0, s>>>(a);
}

template void launch_btd<float>(const BtdArgs<float> &, cudaStream_t);
template void launch_btd<double>(const BtdArgs<double> &, cudaStream_t);

// ----------------------------------------------- lab-frame view of the grid

// gam (f + sgn beta (p0 + p1) / 2), rounded once to the working precision:
// FP64 in FP64, pairs of FP32 words (about 46 bits) in FP32, where the FP64
// pipe bounded it (1.2M nodes, six components: 6 launches of 17.6 us; one
// launch of 35 us with the pairs, 1.7 TB/s: 5.8 us a component).  The pairs'
// error words turn an infinite term into NaN, so what does not come out finite
// is taken in FP64 again.
__device__ __forceinline__ double lab_value(double f, double p0, double p1, double gam, double sb)
{
    return gam * (f + sb * (0.5 * (p0 + p1)));
}
__device__ __forceinline__ float lab_value(float f, float p0, float p1, ff gam, ff sb)
{
    return (gam * (ff(f) + sb * two_sum(0.5f * p0, 0.5f * p1))).h;
}

// The lab-frame fields on the simulation grid at the current time, each
// component at its own Yee position, by the inverse field transformation.  The
// partner a component mixes with is half a cell away in z: the mean of its
// planes k - 1, k (component on integer z) or k, k + 1, the nearer plane alone
// at an absorbing end, planes wrapped when z is periodic.  Nodes beyond the
// component's z range are zero.  blockIdx.y: the component.
template <typename real>
__global__ void lab_fields_kernel(LabArgs<real> a)
{
    using T = typename std::conditional<sizeof(real) == 4, ff, double>::type;
    const Geom &g = a.g;
    const int comp = a.comp[blockIdx.y];
    const real *F = a.F[blockIdx.y], *P = a.P[blockIdx.y];
    real *out = a.out[blockIdx.y];
    const bool half = comp == 2 || comp == 3 || comp == 4;
    const int km = zmax_of(g, half), kmp = zmax_of(g, !half);  // its range, its partner's
    const double sbeta = comp == 1 || comp == 3 ? -a.beta : a.beta;
    const T gam(a.gam), sb(sbeta);
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < g.ncomp; r += (int64_t)gridDim.x * blockDim.x) {
        const int k = g.ncomp <= 0x7fffffffLL ? (int)((unsigned)r / (unsigned)g.plane) : (int)(r / g.plane);
        real v = real(0);
        if (k <= km) {
            v = F[r];
            if (comp != 2 && comp != 5) {
                int lo = half ? k : k - 1, hi = half ? k + 1 : k;
                if (g.bc_z == 0) {
                    lo = wrapi(lo, g.nz);
                    hi = wrapi(hi, g.nz);
                } else {
                    if (lo < 0) lo = hi;
                    if (hi > kmp) hi = lo;
                    if (lo > kmp) lo = hi = kmp;
                }
                const real f = v, p0 = P[r + (lo - k) * g.plane], p1 = P[r + (hi - k) * g.plane];
                v = lab_value(f, p0, p1, gam, sb);
                if (sizeof(real) == 4 && !isfinite(v)) v = (real)lab_value((double)f, (double)p0, (double)p1, a.gam, sbeta);
            }
        }
        out[r] = v;
    }
}

template <typename real>
void launch_lab_fields(const LabArgs<real> &a, int n, int sms, cudaStream_t s)
{
    int64_t blocks = (a.g.ncomp + 255) / 256;
    if (blocks > 8LL * sms) blocks = 8LL * sms;
    lab_fields_kernel<real><<<dim3((unsigned)blocks, (unsigned)n), 256, 0, s>>>(a);
}

template void launch_lab_fields<float>(const LabArgs<float> &, int, int, cudaStream_t);
template void launch_lab_fields<double>(const LabArgs<double> &, int, int, cudaStream_t);

}  // namespace pic
