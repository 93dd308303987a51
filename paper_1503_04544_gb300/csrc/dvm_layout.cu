// Conversion between the public state layout [cell][component][p] of dvm.h
// and the device layout (slabs of one velocity group, W velocities of a cell
// contiguous, cells of a row consecutive; see dvm_internal.h).
//
// The conversion is a transpose, bound by memory: it reads and writes the
// state once.  A block moves a tile of 32 consecutive cells of a row times
// kTileBytes of velocities of one component through shared memory, so that
// both sides are whole lines: 512 contiguous bytes of a cell on the public
// side, 512 contiguous bytes of a group (32 cells of W velocities) on the
// device side.  One element per thread, as before, touched 16 bytes of a
// 32-byte sector in another slab with every fourth thread: 2D, 256^2 x 32^2
// FP32 (0.54 GB each way) 469 us, 3D, 64^3 x 20^3 FP32 10.8 ms.
#include <cudaTypedefs.h>

#include "dvm_device.cuh"

namespace dvm {
namespace {

constexpr int kTileBytes = 512;      // velocities of a cell per tile
constexpr int kTileVec = kTileBytes / 16;
constexpr int kLayThreads = 256;

struct LayArgs {
    int nx, ny, nz;          // nz = 1 in 2D
    int dim, ncomp;
    int nv, nvp;             // public and device velocities of a component
    int nvx, nvxp;           // a device row of nvxp velocities holds nvx public ones
    long slab;
    int nxt;                 // cell tiles of a row
    int nchunk;              // tiles of a component's device velocities
};

// What a transfer does with the values.
enum LayMode { kToDevice, kToPublic, kAddToDevice };

// VEC: whole 16-byte vectors on the public side too (public rows without
// padding and 16-byte aligned); else one element at a time there.
template <typename T, LayMode MODE, bool VEC>
__global__ void __launch_bounds__(kLayThreads) k_layout(LayArgs a, T *pub, T *dev)
{
    constexpr int W = Vec<T>::W, L = kTileVec * W, NW = kLayThreads / 32;
    using V = typename Vec<T>::type;
    // rows of kTileVec + 1 vectors: eight lanes of a quarter-warp phase hit
    // eight different 16-byte bank groups, by rows and by columns
    __shared__ V tile[32][kTileVec + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long row = blockIdx.x / a.nxt;
    const int i0 = (int)(blockIdx.x % a.nxt) * 32;
    const int comp = blockIdx.y / a.nchunk, d0 = (int)(blockIdx.y % a.nchunk) * L;
    const int k = (int)(row / a.ny), j = (int)(row - (long)k * a.ny);
    const long prow = a.dim == 2 ? j + 2 : (long)(k + 2) * (a.ny + 4) + (j + 2);
    const long pc0 = prow * (a.nx + 4) + 2 + i0;            // slab index of the tile's first cell
    const long cell0 = row * a.nx + i0;
    const int ncell = min(32, a.nx - i0);
    const int nvec = min(kTileVec, (a.nvp - d0) / W);       // vectors of the tile
    V *const dv = reinterpret_cast<V *>(dev);
    const auto dev_at = [&](int v) { return ((long)(d0 / W + v) * a.ncomp + comp) * a.slab + pc0 + lane; };

    if constexpr (MODE == kToPublic) {
        V r[kTileVec / NW];
#pragma unroll
        for (int q = 0; q < kTileVec / NW; ++q) {
            const int v = warp + q * NW;
            if (v < nvec && lane < ncell) r[q] = dv[dev_at(v)];
        }
#pragma unroll
        for (int q = 0; q < kTileVec / NW; ++q) tile[lane][warp + q * NW] = r[q];
        __syncthreads();
    }
    if constexpr (VEC) {
        V r[32 / NW];
#pragma unroll
        for (int q = 0; q < 32 / NW; ++q) {
            const int c = warp + q * NW;
            if (lane >= nvec || c >= ncell) continue;
            V *const p = reinterpret_cast<V *>(pub + ((cell0 + c) * a.ncomp + comp) * a.nv + d0) + lane;
            if constexpr (MODE == kToPublic) *p = tile[c][lane];
            else r[q] = *p;
        }
        if constexpr (MODE != kToPublic) {
#pragma unroll
            for (int q = 0; q < 32 / NW; ++q) tile[warp + q * NW][lane] = r[q];
        }
    } else {
        // element d of a device row of nvxp velocities is public element d of
        // the row's nvx, or padding (zero)
#pragma unroll 4
        for (int q = 0; q < 32 / NW; ++q) {
            const int c = warp + q * NW;
            if (c >= ncell) break;
            T *const p = pub + ((cell0 + c) * a.ncomp + comp) * a.nv;
            T *const t = reinterpret_cast<T *>(&tile[c][0]);
#pragma unroll
            for (int u = 0; u < W; ++u) {
                const int d = d0 + u * 32 + lane;
                if (d >= a.nvp) continue;
                const int r = d / a.nvxp, p1 = d - r * a.nvxp, s = r * a.nvx + p1;
                const bool in = p1 < a.nvx && s < a.nv;
                if constexpr (MODE == kToPublic) {
                    if (in) p[s] = t[u * 32 + lane];
                } else {
                    t[u * 32 + lane] = in ? p[s] : T(0);
                }
            }
        }
    }
    if constexpr (MODE != kToPublic) {
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kTileVec / NW; ++q) {
            const int v = warp + q * NW;
            if (v >= nvec || lane >= ncell) continue;
            V x = tile[lane][v];
            V *const o = dv + dev_at(v);
            if constexpr (MODE == kAddToDevice) {
                const V y = *o;
                x.x = y.x + x.x;
                x.y = y.y + x.y;
                if constexpr (W == 4) { x.z = y.z + x.z; x.w = y.w + x.w; }
            }
            *o = x;
        }
    }
}

// A function of the driver, or null.
template <typename F> F driver_entry(const char *name, unsigned version)
{
    cudaDriverEntryPointQueryResult q;
    void *fn = nullptr;
    const cudaError_t e = cudaGetDriverEntryPointByVersion(name, &fn, version, cudaEnableDefault, &q);
    if (e == cudaSuccess && q == cudaDriverEntryPointSuccess) return reinterpret_cast<F>(fn);
    cudaGetLastError();
    return nullptr;
}

template <typename T, LayMode MODE>
cudaError_t layout_t(dvm_ctx *c, T *pub, T *dev)
{
    LayArgs a{};
    a.nx = c->nx; a.ny = c->ny; a.nz = c->dim == 3 ? c->nz : 1;
    a.dim = c->dim; a.ncomp = c->ncomp;
    a.nv = c->nv; a.nvp = c->nvp;
    // 2D pads the whole velocity index at its end, 3D every v_x row
    a.nvx = c->dim == 3 ? c->nvx : c->nv;
    a.nvxp = c->dim == 3 ? c->nvxp : c->nvp;
    a.slab = c->slab;
    a.nxt = (c->nx + 31) / 32;
    constexpr int L = kTileVec * Vec<T>::W;
    a.nchunk = (c->nvp + L - 1) / L;
    const dim3 grid((unsigned)((long)a.nxt * a.ny * a.nz), (unsigned)(a.nchunk * a.ncomp));
    // vectors on both sides when no velocity row is padded and the public
    // array starts on a vector
    if (a.nvx == a.nvxp && reinterpret_cast<uintptr_t>(pub) % 16 == 0)
        k_layout<T, MODE, true><<<grid, kLayThreads, 0, c->stream>>>(a, pub, dev);
    else
        k_layout<T, MODE, false><<<grid, kLayThreads, 0, c->stream>>>(a, pub, dev);
    return cudaGetLastError();
}

}  // namespace

cudaError_t pack_state(dvm_ctx *c, const void *pub, void *dev)
{
    if (c->prec == DVM_FP32) return layout_t<float, kToDevice>(c, (float *)const_cast<void *>(pub), (float *)dev);
    return layout_t<double, kToDevice>(c, (double *)const_cast<void *>(pub), (double *)dev);
}

cudaError_t unpack_state(dvm_ctx *c, const void *dev, void *pub)
{
    if (c->prec == DVM_FP32) return layout_t<float, kToPublic>(c, (float *)pub, (float *)const_cast<void *>(dev));
    return layout_t<double, kToPublic>(c, (double *)pub, (double *)const_cast<void *>(dev));
}

cudaError_t add_state(dvm_ctx *c, const void *pub, void *dev)
{
    if (c->prec == DVM_FP32) return layout_t<float, kAddToDevice>(c, (float *)const_cast<void *>(pub), (float *)dev);
    return layout_t<double, kAddToDevice>(c, (double *)const_cast<void *>(pub), (double *)dev);
}

// How the kernels here may use a caller's device array of `bytes` bytes.  In
// place: whole elements, every byte in memory of this context's device.
// Anything else a copy can read (another device's memory, managed memory, an
// odd address) goes through the staging buffer.  An array that runs past the
// end of its allocation, say a tensor of one element expanded, is an error
// here: a copy of it is refused, a kernel would fault.  In a reserved address
// range the pieces of memory that are mapped into it are followed to the
// array's end.
ArrayAccess array_access(const dvm_ctx *c, const void *p, size_t bytes)
{
    static const auto piece = driver_entry<PFN_cuMemGetAddressRange_v3020>("cuMemGetAddressRange", 3020);
    static const auto attribute = driver_entry<PFN_cuPointerGetAttribute_v4000>("cuPointerGetAttribute", 4000);
    int dev = -1;
    if (!attribute || !piece || reinterpret_cast<uintptr_t>(p) % c->elem != 0 || cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return ArrayAccess::kStaged;
    }
    const auto on_device = [dev](CUdeviceptr at) {
        cudaPointerAttributes attr;
        if (cudaPointerGetAttributes(&attr, reinterpret_cast<const void *>(at)) == cudaSuccess)
            return attr.type == cudaMemoryTypeDevice && attr.device == dev;
        cudaGetLastError();
        return false;
    };
    CUdeviceptr at = reinterpret_cast<CUdeviceptr>(p), start = 0;
    const CUdeviceptr end = at + bytes;
    size_t size = 0;
    if (!on_device(at) || piece(&start, &size, at) != CUDA_SUCCESS) return ArrayAccess::kStaged;
    if (end <= start + size) return ArrayAccess::kDirect;
    at = start + size;
    if (attribute(&start, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, reinterpret_cast<CUdeviceptr>(p)) != CUDA_SUCCESS ||
        attribute(&size, CU_POINTER_ATTRIBUTE_RANGE_SIZE, reinterpret_cast<CUdeviceptr>(p)) != CUDA_SUCCESS)
        return ArrayAccess::kStaged;
    if (end > start + size) return ArrayAccess::kShort;
    while (at < end) {
        if (piece(&start, &size, at) != CUDA_SUCCESS || start + size <= at) return ArrayAccess::kShort;
        if (!on_device(at)) return ArrayAccess::kStaged;
        at = start + size;
    }
    return ArrayAccess::kDirect;
}

}  // namespace dvm
