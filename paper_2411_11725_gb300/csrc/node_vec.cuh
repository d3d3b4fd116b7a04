// Shared parts of the node kernels: 3-vectors, rotating planes in shared memory, arguments, outputs and the split of
// their walk along z.
#pragma once
#include <type_traits>

#include "dp5_control.cuh"
#include "local.cuh"

namespace nm {

// tile of nodes walked along z by one block
constexpr int kUX = 32, kUY = 4, kUThreads = kUX * kUY;

// A 3-vector of the working precision.  FP32: x and y as one packed pair (fma.rn.f32x2: one instruction for
// both, rounded as the scalar ones) and z apart, the layout of the shared planes.
template <typename T>
struct Vec {
    T x, y, z;
};
template <>
struct Vec<float> {
    unsigned long long xy;
    float z;
};
__device__ __forceinline__ unsigned long long pk(float a, float b)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpk(unsigned long long r, float &a, float &b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
template <typename T>
__device__ __forceinline__ Vec<T> vadd(const Vec<T> &a, const Vec<T> &b)
{
    if constexpr (sizeof(T) == 4) {
        Vec<float> r;
        asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.xy) : "l"(a.xy), "l"(b.xy));
        r.z = a.z + b.z;
        return r;
    } else {
        return Vec<T>{a.x + b.x, a.y + b.y, a.z + b.z};
    }
}
// c v + w
template <typename T>
__device__ __forceinline__ Vec<T> vfma(T c, const Vec<T> &v, const Vec<T> &w)
{
    if constexpr (sizeof(T) == 4) {
        Vec<float> r;
        asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.xy) : "l"(pk(c, c)), "l"(v.xy), "l"(w.xy));
        r.z = fmaf(c, v.z, w.z);
        return r;
    } else {
        return Vec<T>{fma(c, v.x, w.x), fma(c, v.y, w.y), fma(c, v.z, w.z)};
    }
}
template <typename T>
__device__ __forceinline__ Vec<T> vmul(T c, const Vec<T> &v)
{
    if constexpr (sizeof(T) == 4) {
        Vec<float> r;
        asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.xy) : "l"(pk(c, c)), "l"(v.xy));
        r.z = c * v.z;
        return r;
    } else {
        return Vec<T>{c * v.x, c * v.y, c * v.z};
    }
}
template <typename T>
__device__ __forceinline__ Vec<T> vsub(const Vec<T> &a, const Vec<T> &b)
{
    if constexpr (sizeof(T) == 4) {
        Vec<float> r;
        asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.xy) : "l"(a.xy), "l"(b.xy));
        r.z = a.z - b.z;
        return r;
    } else {
        return Vec<T>{a.x - b.x, a.y - b.y, a.z - b.z};
    }
}
template <typename T>
__device__ __forceinline__ Vec<T> vzero()
{
    if constexpr (sizeof(T) == 4) return Vec<float>{0ull, 0.f};
    else return Vec<T>{T(0), T(0), T(0)};
}
template <typename T>
__device__ __forceinline__ void vget(const Vec<T> &v, T &x, T &y, T &z)
{
    if constexpr (sizeof(T) == 4) {
        unpk(v.xy, x, y);
        z = v.z;
    } else {
        x = v.x;
        y = v.y;
        z = v.z;
    }
}

// NS planes of R x C 3-vectors in shared memory
template <typename T, int R, int C, int NS>
struct VPlanes {
    T v[NS][R * C][3];
    __device__ __forceinline__ Vec<T> get(int s, int i) const { return Vec<T>{v[s][i][0], v[s][i][1], v[s][i][2]}; }
    __device__ __forceinline__ T *p(int s, int i, int c) { return &v[s][i][c]; }
};
template <int R, int C, int NS>
struct VPlanes<float, R, C, NS> {
    unsigned long long xy[NS][R * C];
    float z[NS][R * C];
    __device__ __forceinline__ Vec<float> get(int s, int i) const { return Vec<float>{xy[s][i], z[s][i]}; }
    __device__ __forceinline__ float *p(int s, int i, int c)
    {
        return c == 2 ? &z[s][i] : reinterpret_cast<float *>(&xy[s][i]) + c;
    }
};

template <typename T>
struct NodeUArgs {
    int nn1, nn2, nn3, N1, N2, N3, ns, cs;
    int bxn, full, chunks, zc;  // blocks b < full walk tile b over all planes; the other tiles are split into
                                // `chunks` blocks of zc planes
    // uniform materials (node_uniform.cu), over a nodal mass unless raw.  2D basis, of a node with one cell column: exchange
    // weights w of the sums of differences, by the cells along the other axis.  3D basis, of a node inside: FP32 the same
    // in the node's own plane (w, index 0) and in the planes beside it (v), and of the difference along z (vz, and vzl:
    // what its rounding left); FP64 2 A x element constants of the axes (c)
    T w1[2], w2[2], ws;
    T can;                      // 2 Ku V / 216 (2D basis: / 36 per layer)
    T v1, v2, vs, vz, vzl, cx, cy, cz;
    T canl, wl;                 // 3D basis, FP32: what the rounding of can left, and of w and v together (relative)
    T e0, e1, e2;
    T im1, mu0V8;               // 1 / mass of such a node (1 when raw); mu0 V/8 (2D basis: mu0 V/4)
    T gam, alpha;
    const T *y, *MsH, *Msh, *hdmi;
    T *out, *y_next;
    const double *m;
    const float *mf;
    const T *k[4];              // earlier slopes with non-zero coefficients in the next stage input
    T a[4], as;                 // their coefficients, and that of the slope being written
    const StepCtl *ctl;
    double c_s, t_fixed, hu0, hu1, hu2, hu_freq, hu_phase, hc_freq, hc_phase;
    int raw, zee, nk;
    // error of a Dormand-Prince step (StageArgs)
    float *se, *dinc;
    float e[5];
    StepCtl *control;
    double *partials, n_active;
    int max_rej;
    // end of an RK4 step (StageArgs)
    double *m_out;
    float *mf_out;
    int renorm;
};

template <typename T>
__device__ __forceinline__ double u_time_factor(double f, double ph, double t)
{
    return f == 0.0 ? 1.0 : sin(2.0 * 3.14159265358979323846 * f * t + ph);
}

// asynchronous copy of one value, or zero fill when !in
template <typename T>
__device__ __forceinline__ void cp_elem(T *dst, const T *src, bool in)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const int n = in ? (int)sizeof(T) : 0;
    if (sizeof(T) == 4)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src), "r"(n) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(d), "l"(src), "r"(n) : "memory");
}

// What a kernel instance writes: the field (kHeff), the slope (kSlope), or the slope and the next stage input
// formed from NK >= 0 earlier slopes.  M64: the next input is formed from the FP64 m (always in FP64, and in
// FP32 where no FP32 copy of m is kept).
// kLast: the slope k_6, the next stage input from four earlier slopes, the step's increment and its error so far; kErr:
// the slope k_7 and the error terms.
// kRk4: the new state of an RK4 step from three earlier slopes and k_4, which is not written.
constexpr int kHeff = -2, kSlope = -1, kErr = -3, kLast = 5, kRk4 = 6;
// earlier slopes that an instance combines
constexpr int node_slopes(int NK) { return NK == kLast ? 4 : (NK == kRk4 ? 3 : (NK > 0 ? NK : 0)); }

// what kErr reads of a node, loaded ahead of its field
struct ErrIn {
    float k1[3], se[3], m0[3];
};

template <typename T>
__device__ __forceinline__ ErrIn load_err(const NodeUArgs<T> &p, int n)
{
    ErrIn e;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        e.k1[c] = p.k[0][c * p.ns + n];
        e.se[c] = p.se[c * p.ns + n];
        e.m0[c] = p.mf[c * p.ns + n];
    }
    return e;
}

// The node's output from its field: H itself, or the LLG slope k (zero without magnetic material) and the next
// stage input.  Returns the node's error terms (kErr; 0 otherwise).
template <typename T, int NK, bool M64>
__device__ __forceinline__ T node_u_out(const NodeUArgs<T> &p, int n, T hx, T hy, T hz, T mx, T my, T mz, T dt,
                                     double dt64, bool magnetic = true, const ErrIn &ei = ErrIn())
{
    constexpr int NS = node_slopes(NK);
    if (NK == kHeff) {
        p.out[n] = hx;
        p.out[p.ns + n] = hy;
        p.out[2 * p.ns + n] = hz;
        return T(0);
    } else {
        // the next stage input's own values, all loads issued together
        T kv[NS > 0 ? NS : 1][3], m0[3];
        double md[3];
        if (NK >= 0) {
#pragma unroll
            for (int i = 0; i < NS; ++i)
#pragma unroll
                for (int c = 0; c < 3; ++c) kv[i][c] = p.k[i][c * p.ns + n];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                if (M64) md[c] = p.m[c * p.ns + n];
                else m0[c] = (T)p.mf[c * p.ns + n];
            }
        }
        // k = -gamma' (m x H + alpha m x (m x H))
        const T ax = my * hz - mz * hy, ay = mz * hx - mx * hz, az = mx * hy - my * hx;
        const T bx = my * az - mz * ay, by = mz * ax - mx * az, bz = mx * ay - my * ax;
        T kk[3];
        kk[0] = -p.gam * (ax + p.alpha * bx);
        kk[1] = -p.gam * (ay + p.alpha * by);
        kk[2] = -p.gam * (az + p.alpha * bz);
        if (!magnetic) kk[0] = kk[1] = kk[2] = T(0);
        if constexpr (NK == kRk4) {
            double v[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                T sum = 0;
#pragma unroll
                for (int i = 0; i < NS; ++i) sum += p.a[i] * kv[i][c];
                sum += p.as * kk[c];
                v[c] = md[c] + dt64 * (double)sum;
            }
            if (p.renorm) renormalise<T>(v);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                p.m_out[c * p.ns + n] = v[c];
                if (p.mf_out) p.mf_out[c * p.ns + n] = (float)v[c];
            }
            return T(0);
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) p.out[c * p.ns + n] = kk[c];
        if (NK >= 0) {
            // y_{s+1} = m + dt sum_j a_j k_j, the slope combination in the working precision
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                T sum = 0;
#pragma unroll
                for (int i = 0; i < NS; ++i) sum += p.a[i] * kv[i][c];
                sum += p.as * kk[c];
                if constexpr (NK == kLast) {
                    // this sum is the step's increment; the error so far in difference form, operation by operation as
                    // in dp5_err_node (the rounded slopes: no contraction into their last product)
                    const T x = kv[0][c];
                    T e = __fmul_rn(p.e[0], __fsub_rn(kv[1][c], x));
                    e = __fmaf_rn(p.e[1], __fsub_rn(kv[2][c], x), e);
                    e = __fmaf_rn(p.e[2], __fsub_rn(kv[3][c], x), e);
                    p.se[c * p.ns + n] = __fmaf_rn(p.e[3], __fsub_rn(kk[c], x), e);
                    p.dinc[c * p.ns + n] = dt * sum;
                }
                p.y_next[c * p.ns + n] = M64 ? (T)(md[c] + dt64 * (double)sum) : m0[c] + dt * sum;
            }
        }
        T part = 0;
        if constexpr (NK == kErr) {
            // the stage's input is the step's result
            const float m5[3] = {mx, my, mz}, rtol = (float)p.ctl->rtol, atol = (float)p.ctl->atol;
#pragma unroll
            for (int c = 0; c < 3; ++c)
                part += dp5_err_term5(ei.m0[c], m5[c], __fmaf_rn(p.e[4], __fsub_rn(kk[c], ei.k1[c]), ei.se[c]), dt, rtol,
                                      atol);
        }
        return part;
    }
}

// the arguments that both node kernels take from the mesh, the stage and the evaluation time
template <typename T>
inline NodeUArgs<T> node_u_args(const LocalParams<T> &p, const T *y, T *out, T *y_next, const StageArgs *sa, double t)
{
    const Geom &g = p.g;
    NodeUArgs<T> a{};
    a.nn1 = g.nn1; a.nn2 = g.nn2; a.nn3 = g.nn3;
    a.N1 = g.N1; a.N2 = g.N2; a.N3 = g.N3;
    a.ns = (int)g.ns;
    a.cs = (int)g.cs;
    a.e0 = p.e0; a.e1 = p.e1; a.e2 = p.e2;
    a.mu0V8 = g.basis == 3 ? p.mu0V8 : p.mu0V4;
    a.gam = p.gam_t;
    a.alpha = p.alpha_t;
    a.y = y;
    a.MsH = (p.terms & NM_DEMAG) ? p.MsH : nullptr;
    a.Msh = p.Msh;
    a.hdmi = p.hdmi;
    a.out = out;
    a.y_next = y_next;
    a.hu0 = p.hu0; a.hu1 = p.hu1; a.hu2 = p.hu2;
    a.hu_freq = p.hu_freq; a.hu_phase = p.hu_phase;
    a.hc_freq = p.hc_freq; a.hc_phase = p.hc_phase;
    a.raw = p.raw;
    a.zee = (p.terms & NM_ZEE) != 0;
    a.t_fixed = t;
    if (!sa) return a;
    a.ctl = sa->ctl;
    a.c_s = sa->c_s;
    a.t_fixed = sa->t_fixed;
    a.se = sa->se;
    a.dinc = sa->dinc;
    for (int j = 0; j < 5; ++j) a.e[j] = sa->e[j];
    a.control = sa->control;
    a.partials = sa->partials;
    a.n_active = sa->n_active;
    a.max_rej = sa->max_rej;
    a.mf = sa->mf;
    a.m_out = sa->m_out;
    a.mf_out = sa->mf_out;
    a.renorm = sa->renorm;
    if (!y_next && !sa->m_out) {
        a.k[0] = (const T *)sa->k[0];
        return a;
    }
    a.m = sa->m;
    a.as = sizeof(T) == 4 ? (T)sa->af_s : (T)sa->a_s;
    for (int j = 0; j + 1 < sa->s && j < 7; ++j) {
        const T c = sizeof(T) == 4 ? (T)sa->af[j] : (T)sa->a[j];
        if (c == T(0)) continue;
        a.k[a.nk] = (const T *)sa->k[j];
        a.a[a.nk] = c;
        ++a.nk;
    }
    return a;
}

// go(NK, M64) with the instance that the arguments need (ERR: kErr among them)
template <typename T, bool ERR, typename F>
inline void node_u_dispatch(const NodeUArgs<T> &a, bool stage, F &&go)
{
    if (!stage) return go(std::integral_constant<int, kHeff>{}, std::true_type{});
    if (a.m_out) return go(std::integral_constant<int, kRk4>{}, std::true_type{});
    if (!a.y_next) {
        if constexpr (sizeof(T) == 4 && ERR) {
            if (a.control) return go(std::integral_constant<int, kErr>{}, std::false_type{});
        }
        return go(std::integral_constant<int, kSlope>{}, std::true_type{});
    }
    if constexpr (sizeof(T) == 4 && ERR) {
        if (a.se) return go(std::integral_constant<int, kLast>{}, std::false_type{});
    }
    auto slopes = [&](auto n) {
        if constexpr (sizeof(T) == 4) {
            if (a.mf) return go(n, std::false_type{});
        }
        go(n, std::true_type{});
    };
    switch (a.nk) {
    case 0: return slopes(std::integral_constant<int, 0>{});
    case 1: return slopes(std::integral_constant<int, 1>{});
    case 2: return slopes(std::integral_constant<int, 2>{});
    case 3: return slopes(std::integral_constant<int, 3>{});
    default: return slopes(std::integral_constant<int, 4>{});
    }
}

// Split of the walk: cost in plane units of a grid whose tiles are cut into `chunks` pieces, from the latency
// of one block (its planes, two more for the halo, and the start of the walk) and the planes an SM works
// through when the blocks are dealt out evenly (about four planes of one block cost an SM as much time as the
// latency of one).
//
// FP64 is bound by the FP64 rate, not by the latency of a block, and pays for the planes that neighbouring chunks
// both work on: its cost counts the planes a chunk really works on (128x128x4: 68 -> 46 us a stage, events around each launch).
inline void node_u_grid(int nn1, int nn2, int nn3, bool fp64, int *bxn, int *full, int *chunks, int *zc, int *blocks)
{
    static const int sms = [] {
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        return cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0 ? v : 152;
    }();
    *bxn = div_up(nn1, kUX);
    const int tiles = *bxn * div_up(nn2, kUY);
    double best = 1e300;
    for (int f = 0; f < 2; ++f) {
        const int fl = f ? tiles - tiles % sms : 0, rest = tiles - fl;
        if (f && fl == 0) break;
        for (int c = 1; c <= nn3; ++c) {
            const int z = div_up(nn3, c), ch = div_up(nn3, z);
            if (c > 1 && ch != c) continue;  // (the same split as fewer chunks)
            const double pf = fp64 ? nn3 + 0.5 : nn3 + 2, pc = fp64 ? (nn3 + 2.0 * (ch - 1)) / ch + 0.5 : z + 2;
            const double work = (double)(fl / sms) * pf + div_up((long)rest * ch, sms) * pc;
            const double lat = (fp64 ? 1.0 : 4.0) * ((fl ? nn3 : z) + 4);
            const double cost = work > lat ? work : lat;
            if (cost < best * 0.999) {
                best = cost;
                *full = fl;
                *zc = z;
                *chunks = ch;
                *blocks = fl + rest * ch;
            }
        }
    }
}

}  // namespace nm
