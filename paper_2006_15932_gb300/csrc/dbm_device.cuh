// dbm_device.cuh -- device building blocks of the D2V16 DBM step:
// chained launches, the equilibrium moments f-hat, conversions by bits and
// the ghost-image bookkeeping of the boundary conditions.  The NND flux
// differences are in dbm_step_impl.cuh.
#pragma once

#include <atomic>
#include <type_traits>

#include "dbm_internal.h"

namespace dbm {

// Chained launches: a step kernel launched with programmatic serialization
// may start while the kernel before it on the stream still drains.  It sets
// up its barriers and touches no memory that another kernel reads or writes
// before its wait (ChainedIn::wait, chain_begin) has returned: by then the
// kernel before it has completed and its writes are visible.  Its own successor
// may start once every CTA has passed chain_end, which sits late in the step:
// CTAs that start early take the free SMs and the rest of their grid doubles up
// on others, which costs a grid of fewer CTAs than the chip holds more than the
// launch it hides (FP64, 64 x 64, two species: 29 us a step unchained, 54 with
// the successor let in at once).
//
// The input of a chained kernel is still being written when the kernel starts,
// so it is not read-only for the kernel's lifetime: a const __restrict__
// parameter would promise that, and would let the compiler move loads above the
// wait or send them through the non-coherent cache.  A chained kernel takes it
// as ChainedIn, which gives the pointer out of the wait itself: every load
// depends on the wait's result.  launch_chained takes no bare pointer to const.
// (Plain pointers in a struct, as the compact step's BfState, promise nothing:
// their loads stay behind the memory clobber of chain_begin.)
template <class T>
class ChainedIn {
    const T *p;

  public:
    explicit ChainedIn(const void *q) : p(static_cast<const T *>(q)) {}
    __device__ __forceinline__ const T *wait() const  // chain_begin, and the input after it
    {
        size_t g = __cvta_generic_to_global(p);  // stays a global address across the asm
        asm volatile("griddepcontrol.wait;" : "+l"(g)::"memory");
        return static_cast<const T *>(__cvta_global_to_generic(g));
    }
};
__device__ __forceinline__ void chain_begin() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_end() { asm volatile("griddepcontrol.launch_dependents;"); }

// Raise a kernel's dynamic shared-memory limit, once per device (`done`: one
// bit per device, a static of the launcher).
template <class K>
cudaError_t allow_smem(K kernel, size_t bytes, std::atomic<unsigned long long> &done)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
    if (bit != 0 && (done.load(std::memory_order_relaxed) & bit) != 0) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_relaxed);
    return e;
}

// Dynamic shared memory that keeps a grid of at most one CTA per SM from
// doubling up: more than half of an SM's.
constexpr size_t ALONE_SMEM = 116 * 1024;

template <class P>
constexpr bool bare_input()  // a pointer to const
{
    return std::is_pointer<P>::value && std::is_const<typename std::remove_pointer<P>::type>::value;
}

template <class... P, class... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A &&...args)
{
    static_assert(!(bare_input<P>() || ...), "a chained kernel takes its input as ChainedIn");
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// f-hat_1..16 of the moment relations (section "Discrete Boltzmann model",
// the f-hat list restating Eqs. relation1..relation7) at (n, u, theta = T/m)
// with dpi = D + I.  Factored for the GPU; the same polynomials as printed.
template <typename real>
__device__ __forceinline__ void fhat16(real n, real ux, real uy, real th, real dpi, real fh[Q])
{
    const real u2 = ux * ux + uy * uy;
    const real a2 = (dpi + real(2)) * th + u2;  // (D+I+2) T/m + u.u
    const real a4 = (dpi + real(4)) * th + u2;  // (D+I+4) T/m + u.u
    const real nux = n * ux, nuy = n * uy;
    const real xx = ux * ux, yy = uy * uy;
    fh[0] = n;
    fh[1] = nux;
    fh[2] = nuy;
    fh[3] = n * (dpi * th + u2);
    fh[4] = n * (th + xx);
    fh[5] = nux * uy;
    fh[6] = n * (th + yy);
    fh[7] = nux * a2;
    fh[8] = nuy * a2;
    fh[9] = nux * (real(3) * th + xx);
    fh[10] = nuy * (th + xx);
    fh[11] = nux * (th + yy);
    fh[12] = nuy * (real(3) * th + yy);
    fh[13] = n * (a2 * th + xx * a4);
    fh[14] = nux * uy * a4;
    fh[15] = n * (a2 * th + yy * a4);
}

// (double)x on the integer pipe.  The conversion instruction shares the FP64
// pipe, two lanes per SM and cycle here, and the output kernels convert every
// value they read or write: exponent and mantissa are moved over instead
// (k_moments_f32: half its time; k_get_f on 4096^2: 1.05 -> 0.99 ms).
// Zeros keep their sign; subnormal, infinite and NaN values take the
// instruction.
__device__ __forceinline__ bool widens_by_bits(float x)
{
    const unsigned a = __float_as_uint(x) & 0x7fffffffu;
    return a - 1u >= 0x007fffffu && a < 0x7f800000u;
}
__device__ __forceinline__ double widen_bits(float x)
{
    const unsigned u = __float_as_uint(x), a = u & 0x7fffffffu;
    const unsigned hi = a == 0u ? u : (u & 0x80000000u) | ((a >> 3) + 0x38000000u);
    return __hiloint2double((int)hi, (int)(u << 29));
}
__device__ __forceinline__ double widen(float x) { return widens_by_bits(x) ? widen_bits(x) : (double)x; }

// Ghost images of interior index k along an axis of n cells: the ghost
// indices g in {-2, -1, n, n+1} whose source cell is k (periodic wrap, or
// the edge cell for outflow).  Returns the count (0..4) and the indices.
__device__ __forceinline__ int ghost_images(int k, int n, int bc, int g[4])
{
    int cnt = 0;
    const int cand[4] = {-2, -1, n, n + 1};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int c = cand[j];
        int src;
        if (bc == DBM_BC_PERIODIC)
            src = ((c % n) + n) % n;
        else
            src = c < 0 ? 0 : n - 1;
        if (src == k) g[cnt++] = c;
    }
    return cnt;
}

struct Images {
    int gx[4], gy[4];
    int ngx, ngy;
};

__device__ __forceinline__ Images cell_images(int x, int y, int nx, int ny, int bc_x, int bc_y)
{
    Images im;
    im.ngx = ghost_images(x, nx, bc_x, im.gx);
    im.ngy = ghost_images(y, ny, bc_y, im.gy);
    return im;
}

// Store v at interior cell (x, y) of plane base `pl` and at its ghost images.
template <typename T>
__device__ __forceinline__ void store_with_images(T *pl, long long cell, int x, int y, int pitch,
                                                  const Images &im, T v)
{
    pl[cell] = v;
    for (int j = 0; j < im.ngx; ++j) pl[(long long)(y + GY) * pitch + (im.gx[j] + GX)] = v;
    for (int j = 0; j < im.ngy; ++j) pl[(long long)(im.gy[j] + GY) * pitch + (x + GX)] = v;
}

__device__ __forceinline__ void raise_flag(unsigned *flag, unsigned bits)
{
    if (bits) atomicOr(flag, bits);
}

// Checked builds (-DDBM_CHECKED, a debugging aid that stands in for a
// memory checker): every index into a shared-memory tile, a state buffer or
// a ghost image is compared with the extent of what it addresses; one
// outside it raises DBM_HEALTH_BOUNDS and the access is skipped (a load
// gives 0).  The default build compiles the checks away.
__device__ __forceinline__ bool in_bounds(long long i, long long n, unsigned *flag)
{
#ifdef DBM_CHECKED
    if (i >= 0 && i < n) return true;
    raise_flag(flag, DBM_HEALTH_BOUNDS);
    return false;
#else
    return true;
#endif
}

}  // namespace dbm
