// Error terms, reduction and step control of a Dormand-Prince attempt, and the end of an RK4 step: shared by the kernels
// of the Runge-Kutta bookkeeping and by the node kernels that do that work themselves.
#pragma once
#include "rk.cuh"

namespace nm {

// Sum over the block in a fixed order, the same value in every thread; sh holds 33 values.
__device__ __forceinline__ double block_sum(double v, double *sh)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if ((threadIdx.x & 31) == 0) sh[w] = v;
    __syncthreads();
    if (w == 0) {
        v = (int)threadIdx.x < nw ? sh[threadIdx.x] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (threadIdx.x == 0) sh[32] = v;
    }
    __syncthreads();
    const double r = sh[32];
    __syncthreads();
    return r;
}

// err^(-1/5) for err within [1e-4, 1e4]: the FP32 power and two Newton steps in FP64 (relative error 1e-6 ->
// 1e-12 -> rounding), a dozen operations where the FP64 power takes hundreds at GB300's FP64 rate
__device__ __forceinline__ double inv_fifth_root(double err)
{
    double r = (double)powf((float)err, -0.2f);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const double r2 = r * r;
        r = r * (1.2 - 0.2 * err * r2 * r2 * r);
    }
    return r;
}

// Step control from s = the sum of the squared error terms (one thread): err = sqrt(s / (3 n_active)); accept
// when err <= 1; new dt from dt * clamp(0.9 err^(-1/5), 0.2, 5); clipping to t_end; failure after too many
// rejections.
__device__ __forceinline__ void dp5_decide(double s, double n_active, StepCtl *ctl, int max_rej)
{
    const double err = n_active > 0 ? sqrt(s / (3.0 * n_active)) : 0.0;
    const bool fin = isfinite(err), acc = fin && err <= 1.0;
    // (below 1e-4 and above 1e4 the factor is at its bounds)
    const double fac =
        !fin || err > 1e4 ? 0.2 : (err < 1e-4 ? 5.0 : fmin(5.0, fmax(0.2, 0.9 * inv_fifth_root(err))));
    const double dt = ctl->dt;
    ctl->err = err;
    ctl->accepted = acc;
    ctl->dt_used = dt;
    double t = ctl->t;
    int rej = ctl->consecutive_rej;
    if (acc) {
        t += dt;
        ctl->t = t;
        ctl->n_acc += 1;
        rej = 0;
    } else {
        ctl->n_rej += 1;
        rej += 1;
    }
    ctl->consecutive_rej = rej;
    double dtn = dt * fac;
    ctl->dt_prop = dtn;
    const double t_end = ctl->t_end;
    bool done = false;
    if (t_end > 0.0) {
        const double rem = t_end - t;
        if (rem <= 1e-12 * fmax(fabs(t_end), 1e-30)) done = true;
        else if (dtn > rem) dtn = rem;
    }
    if (rej > max_rej || (!done && dtn < ctl->dt_min)) {
        ctl->status = NM_ERR_STEP_UNDERFLOW;
        done = true;
    }
    if (done) ctl->done = 1;
    ctl->dt = dtn;
}

// End of an error kernel: the block's sum goes to partials, and the block that arrives last adds them up in
// order and takes the step decision (a launch of its own before: on small meshes it took as long as a pass).
// Every block has read what it needs of ctl before it arrives.
__device__ __forceinline__ void dp5_finish(double acc, double *partials, double n_active, StepCtl *ctl, int max_rej,
                                           double *sh)
{
    __shared__ bool last;
    const double s = block_sum(acc, sh);
    if (threadIdx.x == 0) {
        partials[blockIdx.x] = s;
        __threadfence();
        last = atomicAdd(&ctl->ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double v = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) v += __ldcg(partials + i);
    const double total = block_sum(v, sh);
    if (threadIdx.x == 0) {
        ctl->ticket = 0;
        dp5_decide(total, n_active, ctl, max_rej);
    }
}
// a finished integration: the attempt counts for nothing
__device__ __forceinline__ bool dp5_idle(StepCtl *ctl)
{
    if (!ctl->done) return false;
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl->accepted = 0;
    return true;
}

// The error combination sum_j e_j k_j (e_j = b_j - b*_j, first slope k_1) is formed in FP32 as
// sum_{j>1} e_j (k_j - k_1).  The weights sum to zero, so this is the same quantity; the slopes of one
// step are close to each other, so their differences are exact in FP32 and the combination keeps its
// relative accuracy when it is far smaller than the slopes (small steps), where the direct sum with
// FP32-rounded weights would leave a residue of about 1e-8 |k_1|.
__device__ __forceinline__ float dp5_err_term5(float m0, float m5, float se, float dtf, float rtol, float atol)
{
    const float sc = atol + rtol * fmaxf(fabsf(m0), fabsf(m5));
    const float q = __fdividef(dtf * se, sc);  // a weight of the norm: fast division
    return q * q;
}
__device__ __forceinline__ float dp5_err_term(float m0, float sb, float se, float dtf, float rtol, float atol)
{
    return dp5_err_term5(m0, m0 + dtf * sb, se, dtf, rtol, atol);
}

// 1/sqrt(s) for s > 0 in FP64 from an FP32 estimate and one Newton step (relative error ~1e-14), so
// the FP32 path renormalises without FP64 division or square root.
__device__ __forceinline__ double rsqrt_refined(double s)
{
    const double r0 = (double)rsqrtf((float)s);
    return r0 * (1.5 - 0.5 * s * r0 * r0);
}

// v / |v| (v unchanged when zero): FP32 meshes through rsqrt_refined
template <typename T>
__device__ __forceinline__ void renormalise(double v[3])
{
    const double s = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
    if (s > 0.0) {
        const double r = sizeof(T) == 8 ? 1.0 / sqrt(s) : rsqrt_refined(s);
        v[0] *= r; v[1] *= r; v[2] *= r;
    }
}

// End of an RK4 step, called by every thread of the grid: the block that arrives last (every thread of every block has
// read t and dt by then) advances the time
__device__ __forceinline__ void rk4_finish(StepCtl *ctl)
{
    __syncthreads();
    if (threadIdx.x != 0 || atomicAdd(&ctl->ticket, 1u) != gridDim.x - 1) return;
    ctl->ticket = 0;
    ctl->t += ctl->dt;
    ctl->n_acc += 1;
    ctl->accepted = 1;
    ctl->dt_used = ctl->dt;
    if (ctl->t_end > 0.0) {
        double rem = ctl->t_end - ctl->t;
        if (rem <= 1e-12 * fmax(fabs(ctl->t_end), 1e-30)) ctl->done = 1;
        else if (ctl->dt > rem) ctl->dt = rem;
    }
}

}  // namespace nm
