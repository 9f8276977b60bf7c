// restore_route_host.cu -- pic_capi.cu's object linked against a CUDA runtime
// of host memory: which memory does pic_set_state hand to the kernel that
// buckets a device snapshot?  Memory is host memory throughout; where it
// "lies" is what cudaPointerGetAttributes answers, and the bucket kernel's
// launch looks at the pointers it gets.  Prints one line per precision and
// kind of memory: direct (the snapshot itself) or staged (a copy of it).
// (Compiled twice: by the host compiler for the runtime, by nvcc for the rest.)
#include <cuda_runtime_api.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>

constexpr int kOwnDevice = 1;
extern cudaPointerAttributes answer;
extern cudaError_t answer_status;

#ifndef __CUDACC__

cudaPointerAttributes answer;
cudaError_t answer_status = cudaSuccess;

extern "C" cudaError_t cudaGetDevice(int *d)
{
    *d = kOwnDevice;
    return cudaSuccess;
}
extern "C" cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int)
{
    *v = 152;
    return cudaSuccess;
}
extern "C" cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *)
{
    *a = answer;
    return answer_status;
}
extern "C" cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t)
{
    std::memmove(d, s, n);
    return cudaSuccess;
}
extern "C" cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t)
{
    std::memset(d, v, n);
    return cudaSuccess;
}
extern "C" cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
extern "C" cudaError_t cudaGetLastError() { return cudaSuccess; }
extern "C" const char *cudaGetErrorString(cudaError_t) { return "error"; }
extern "C" void **__cudaRegisterFatBinary(void *) { return nullptr; }
extern "C" void __cudaRegisterFatBinaryEnd(void **) {}
extern "C" void __cudaUnregisterFatBinary(void **) {}

#else

#include "pic.h"
#include "pic_internal.cuh"

static const unsigned char *snap, *columns;  // the snapshot, its first attribute column
static int calls, direct, staged;

namespace pic {
template <typename real> static void look(const BucketArgs<real> &a)
{
    ++calls;
    // species 0 is bucketed first: its ox column is the snapshot's first
    if (calls > 1) return;
    const unsigned char *p = reinterpret_cast<const unsigned char *>(a.src.ox);
    if (p == columns) ++direct;
    else if (std::memcmp(p, columns, (size_t)a.n * sizeof(real)) == 0) ++staged;
}
template <> void launch_bucket<float>(const BucketArgs<float> &a, cudaStream_t) { look(a); }
template <> void launch_bucket<double>(const BucketArgs<double> &a, cudaStream_t) { look(a); }
template <> void launch_compact<float>(const CompactArgs<float> &, cudaStream_t) {}
template <> void launch_compact<double>(const CompactArgs<double> &, cudaStream_t) {}
}  // namespace pic

static void *memory(size_t bytes) { return std::aligned_alloc(256, (bytes + 255) / 256 * 256); }

int main()
{
    const struct {
        const char *name;
        cudaMemoryType type;
        int device;
        cudaError_t status;
    } kinds[] = {{"own", cudaMemoryTypeDevice, kOwnDevice, cudaSuccess},
                 {"other", cudaMemoryTypeDevice, kOwnDevice - 1, cudaSuccess},
                 {"managed", cudaMemoryTypeManaged, kOwnDevice - 1, cudaSuccess},
                 {"pinned", cudaMemoryTypeHost, kOwnDevice, cudaSuccess},
                 {"unknown", cudaMemoryTypeUnregistered, kOwnDevice, cudaSuccess},
                 {"refused", cudaMemoryTypeDevice, kOwnDevice, cudaErrorInvalidValue}};
    for (int precision : {PIC_FP32, PIC_FP64}) {
        pic_grid_params p{};
        p.dim = 2;
        p.nx = p.nz = 32;
        p.ny = 1;
        p.dx = p.dy = p.dz = 1.0;
        p.cfl = 0.99;
        p.gamma_boost = 5.0;
        p.shape_order = 1;
        p.bc_z = PIC_BC_PERIODIC;
        p.precision = precision;
        p.slots_per_cell = 1.0;
        pic_ctx *c = nullptr;
        pic_sizes s;
        if (pic_init_grid(&p, &c) != PIC_OK || pic_query_sizes(c, &s) != PIC_OK) return 1;
        pic_buffers b{};
        b.fields = memory(s.field_bytes);
        b.species[0] = memory(s.species_bytes[0]);
        b.species[1] = memory(s.species_bytes[1]);
        b.scratch = memory(s.scratch_bytes);
        std::memset(b.species[0], 1, s.species_bytes[0]);
        std::memset(b.species[1], 1, s.species_bytes[1]);
        if (pic_bind_buffers(c, &b) != PIC_OK) return 2;
        // 40 electrons in the first tile (the counters lead the scratch buffer)
        static_cast<int *>(b.scratch)[0] = 40;
        size_t bytes = 0;
        if (pic_state_bytes(c, &bytes) != PIC_OK) return 3;
        unsigned char *state = static_cast<unsigned char *>(memory(bytes));
        if (pic_get_state(c, state, bytes, 0) != PIC_OK) return 4;
        snap = state;
        columns = snap + 512 + s.field_bytes;
        for (size_t o = 512 + s.field_bytes; o < bytes; ++o) state[o] = (unsigned char)(o * 37);
        for (const auto &k : kinds) {
            answer = cudaPointerAttributes{};
            answer.type = k.type;
            answer.device = k.device;
            answer_status = k.status;
            calls = direct = staged = 0;
            if (pic_set_state(c, snap, bytes, 1) != PIC_OK) return 5;
            std::printf("%d %s %s\n", precision, k.name, direct ? "direct" : staged ? "staged" : "neither");
        }
        pic_destroy(c);
    }
    return 0;
}

#endif
