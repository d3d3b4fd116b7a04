// Shared definitions of the sm_103a library: complex arithmetic, mesh state, launch helpers.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

#include "nmgb.h"

namespace nm {

constexpr double kMu0 = 4.0e-7 * 3.14159265358979323846;

template <typename T> struct Cx;
template <> struct alignas(8) Cx<float> { float x, y; };
template <> struct alignas(16) Cx<double> { double x, y; };

template <typename T> __host__ __device__ __forceinline__ Cx<T> cx(T a, T b) { Cx<T> r; r.x = a; r.y = b; return r; }
template <typename T> __host__ __device__ __forceinline__ Cx<T> operator+(Cx<T> a, Cx<T> b) { return cx<T>(a.x + b.x, a.y + b.y); }
template <typename T> __host__ __device__ __forceinline__ Cx<T> operator-(Cx<T> a, Cx<T> b) { return cx<T>(a.x - b.x, a.y - b.y); }
template <typename T> __host__ __device__ __forceinline__ Cx<T> operator*(Cx<T> a, Cx<T> b)
{
    return cx<T>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename T> __host__ __device__ __forceinline__ Cx<T> scale(Cx<T> a, T s) { return cx<T>(a.x * s, a.y * s); }
template <typename T> __host__ __device__ __forceinline__ Cx<T> conj(Cx<T> a) { return cx<T>(a.x, -a.y); }
// multiply by s*i for s = +-1
template <typename T> __host__ __device__ __forceinline__ Cx<T> mul_si(Cx<T> a, int s)
{
    return s > 0 ? cx<T>(-a.y, a.x) : cx<T>(a.y, -a.x);
}

// Division by a run-time constant through a multiply-high (round-up method): valid for n + d < 2^32.
struct FastDiv {
    unsigned d, m, s;
    FastDiv() = default;
    __host__ __device__ explicit FastDiv(unsigned d_) : d(d_), m(0), s(0)
    {
        while ((1u << s) < d) ++s;
        m = (unsigned)(((1ull << 32) * ((1ull << s) - d)) / d + 1);
    }
    __device__ __forceinline__ unsigned div(unsigned n) const { return (__umulhi(n, m) + n) >> s; }
    __device__ __forceinline__ unsigned mod(unsigned n) const { return n - div(n) * d; }
};

// Device-resident step control: every kernel of an RK step reads t and dt from here, so a whole step
// (or many) can be launched without a host round trip.
struct StepCtl {
    double t;        // time at the start of the step being attempted
    double dt;       // size of the step being attempted
    double dt_used;  // size of the last attempted step (read by the update after control)
    double dt_prop;  // controller proposal before clipping to t_end
    double err;      // error norm of the last attempt
    double t_end;    // integration end (run_until); steps are clipped to it and to sample times
    double sample_dt;
    double dt_min;
    long n_acc, n_rej;
    long next_sample;  // index of the next sample time (run_until)
    long max_samples;
    int accepted;    // last attempt accepted
    int done;        // t reached t_end: later steps do nothing
    int status;      // NM_OK or an NM_ERR_* code set on the device
    int consecutive_rej;
    double rtol, atol;
    unsigned ticket;  // blocks of the running reduction that have arrived (zero between launches)
};

// Optional per-launch hook, called after every kernel launch with the kernel's name (profiling).
struct Marker {
    void (*fn)(void *ctx, const char *name) = nullptr;
    void *ctx = nullptr;
    void operator()(const char *name) const
    {
        if (fn) fn(ctx, name);
    }
};

// Programmatic dependent launch.  The passes of a step are short kernels that each need all of the one
// before, so on small meshes the gap between two kernels costs as much as a kernel.  A kernel launched with
// launch_pdl may be scheduled while its predecessor in the stream still runs; its first statement pdl_enter
// waits until that predecessor has finished and its writes are visible (every thread calls it, before any
// access to global memory).  Because each kernel waits for its predecessor, which waited for its own,
// everything earlier in the stream is finished too.
//
// A grid of many waves lets its successor be scheduled as soon as its last blocks have started, so that the
// successor's blocks fill the SMs that drain (1024x1024x32 step 26.83 -> 26.24 ms, 512x512x16 3.90 -> 3.83
// ms).  Smaller grids do not: blocks of the successor that settle early crowd the SMs the running grid left
// free and stay there (FP64 step on 512x33x3 1.44 -> 2.12 ms, 256x256x8 in FP32 634 -> 656 us with the
// early trigger everywhere); for them the successor comes when the grid has ended (64x64x1 step 172 -> 162
// us, 16x16x4 RK4 step 84 -> 80 us against plain launches).
constexpr unsigned kPdlEarlyBlocks = 4096;
__device__ __forceinline__ void pdl_enter()
{
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    if (gridDim.x * gridDim.y * gridDim.z >= kPdlEarlyBlocks)
        asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}
template <typename... KA, typename... A>
inline void launch_pdl(void (*kernel)(KA...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A &&...args)
{
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<KA>(std::forward<A>(args))...);  // (a failure is left for cudaGetLastError)
}

// Launch-shape helpers
inline int div_up(long a, long b) { return (int)((a + b - 1) / b); }
inline long round_up(long a, long b) { return (a + b - 1) / b * b; }

}  // namespace nm
