// Node kernels of the trilinear and of the 2D basis for a uniform material (no cell maps, Ms > 0): exchange, uniaxial
// anisotropy, Zeeman and the cell->node demag average, divided by the lumped nodal mass (Eqs.
// weak_form_impl_f, weak_form_impl, mass_lumping), followed by the LLG right-hand side (Eq. llg) and the next
// Runge-Kutta stage input.
//
// With one A and one Ku on a box of cells the assembled operators are sums of tensor products of the
// one-dimensional stiffness and mass matrices, which at a node with n adjacent cells along the axis (n = 2
// inside, 1 at an end) act as
//   K u = -D u / dx,      M u = (3 n u0 + D u) dx / 6,      D u = the sum of u' - u0 over the neighbours u' (n of them).
// The field is
//   -dE_ex = -2 A (K1 M2 M3 + M1 K2 M3 + M1 M2 K3) m,   -dE_an = 2 Ku e (M1 M2 M3) (e . m).
// A node at an end of the x or y axis has half the cells and half the mass of one inside, so its field is that of a node
// inside whose missing neighbours mirror the ones it has; along z the ends keep their own weights.  In a node plane every
// operator is a combination of sums of differences to the node itself, X of the neighbours along x, Y along y and C of
// the corners; along z two partial sums per component and the node's own value are carried up the walk:
//   exchange at z:  n3 (w1 X + w2 Y + ws C)(z) + sum over the planes z' beside of  (v1 X + v2 Y + vs C)(z') + vz (u0(z') - u0(z)),
//   36 M1 M2 u / (dx dy) = 36 u0 + 4 X + 4 Y + C.
// That is about 75 multiply-adds and 9 shared-memory vectors per node instead of the 162 and 27 of the assembled
// 27-point form.  Differences of close values are exact, so the exchange field keeps its relative accuracy on smooth
// states; sums of the values themselves cancel (FP32, 64x64x16 cells, a rotation by 0.01 rad a cell: relative error inside
// 7.7e-4 with such sums, 1.6e-6 here; random state 7.1e-8, 5.3e-8).  FP64 keeps the sums: it is bound by the FP64 rate
// (stage at 128x128x4: 54.5 us with differences, 48.5 us), and their rounding is 1e-16 of the values.
#include "node_vec.cuh"

namespace nm {

// Tile of 32 x 4 nodes walked along z by 128 threads, eight FP32 blocks per SM at 64 registers.  Measured per
// stage at 1024x1024x32 (FP32) / 512x512x16, with sums of the values: 0.59 ms / 87 us, against 1.04 ms / 154 us for the
// assembled 27-point form and 0.64 ms / 99 us with two rows per thread (96 registers, five blocks per SM).  The
// differences cost 1.5 / 2.5 %: mean stage of a Dormand-Prince step, with its error terms, 0.648 -> 0.657 ms / 96 -> 98 us
// (100 us with reads for the elements past the mirror nodes too, and 13.4 instead of 11.5 us at 15x200x13).
constexpr int kUSlots = 3;

template <typename T>
struct NodeUSmem {
    static constexpr int SX = kUX + 2, SY = kUY + 2, CX = kUX + 1, CY = kUY + 1;
    VPlanes<T, SY, SX, kUSlots> y;  // node plane p in slot p mod 3 (counted from the first plane of the walk)
    VPlanes<T, CY, CX, kUSlots> c;  // cell plane p - 1 (Ms_c H_c) beside node plane p
    T hf[4];               // uniform applied field, time factor of the cell field
};

// the node that stands for index i >= -1 of an axis of n nodes: its mirror image beside an end, none (-1) beyond that
__device__ __forceinline__ int mirror(int i, int n) { return i < 0 ? 1 : (i < n ? i : (i == n ? n - 2 : -1)); }

// (The instances of the last two Dormand-Prince stages take 72 registers, seven blocks: at 64 kLast spilled and took
// 219 us at 512x512x16 where stage 5 took 101; with 72 it takes 119 where stage 5 takes 106, and kErr 102.)
template <typename T, int NK, bool M64>
__global__ void __launch_bounds__(kUThreads, sizeof(T) == 4 ? (NK == kLast || NK == kErr || NK == kRk4 ? 7 : 8) : 4) k_node_u(const __grid_constant__ NodeUArgs<T> p)
{
    pdl_enter();
    if constexpr (NK == kErr) {
        if (dp5_idle(p.control)) return;
    } else if (NK != kHeff && p.ctl && p.ctl->done) {
        return;
    }
    using S = NodeUSmem<T>;
    __shared__ S sm;
    const int b = blockIdx.x, split = b >= p.full;
    const int tile = split ? p.full + (b - p.full) / p.chunks : b;
    const int z0 = split ? (b - p.full) % p.chunks * p.zc : 0, z1 = split ? min(p.nn3, z0 + p.zc) : p.nn3;
    const int x0 = tile % p.bxn * kUX, y0 = tile / p.bxn * kUY;
    const int tx = threadIdx.x % kUX, ty = threadIdx.x / kUX;
    const int n1 = x0 + tx, n2 = y0 + ty;
    if (threadIdx.x == 0) {
        const double t = p.ctl ? p.ctl->t + p.c_s * p.ctl->dt : p.t_fixed;
        const double su = u_time_factor<T>(p.hu_freq, p.hu_phase, t);
        sm.hf[0] = (T)(p.hu0 * su);
        sm.hf[1] = (T)(p.hu1 * su);
        sm.hf[2] = (T)(p.hu2 * su);
        sm.hf[3] = (T)u_time_factor<T>(p.hc_freq, p.hc_phase, t);
    }
    // the elements of every node and cell plane that this thread copies: offset within the plane (of the mirror node
    // beside an end of the mesh), or -1 where there is none (zero fill)
    constexpr int EN = (S::SX * S::SY + kUThreads - 1) / kUThreads, EC = (S::CX * S::CY + kUThreads - 1) / kUThreads;
    int no[EN], co[EC];
#pragma unroll
    for (int k = 0; k < EN; ++k) {
        const int t = threadIdx.x + k * kUThreads, r = t / S::SX, c = t - r * S::SX;
        const int i = mirror(x0 - 1 + c, p.nn1), j = mirror(y0 - 1 + r, p.nn2);
        no[k] = i >= 0 && j >= 0 ? j * p.nn1 + i : -1;
    }
#pragma unroll
    for (int k = 0; k < EC; ++k) {
        const int t = threadIdx.x + k * kUThreads, r = t / S::CX, c = t - r * S::CX;
        const int i = x0 - 1 + c, j = y0 - 1 + r;
        co[k] = (i >= 0 && i < p.N1 && j >= 0 && j < p.N2) ? j * p.N1 + i : -1;
    }
    const int np = p.nn1 * p.nn2, ncp = p.N1 * p.N2;
    // node plane q and cell plane q - 1 into slot s (planes outside the mesh are not read: their terms are
    // skipped)
    auto load_plane = [&](int q, int s) {
        if (q >= 0 && q < p.nn3) {
#pragma unroll
            for (int k = 0; k < EN; ++k) {
                const int t = threadIdx.x + k * kUThreads;
                if (t < S::SX * S::SY) {
                    const bool in = no[k] >= 0;
                    const T *src = p.y + (in ? q * np + no[k] : 0);
#pragma unroll
                    for (int c = 0; c < 3; ++c) cp_elem(sm.y.p(s, t, c), src + c * p.ns, in);
                }
            }
        }
        if (p.MsH && q >= 1 && q - 1 < p.N3) {
#pragma unroll
            for (int k = 0; k < EC; ++k) {
                const int t = threadIdx.x + k * kUThreads;
                if (t < S::CX * S::CY) {
                    const bool in = co[k] >= 0;
                    const T *src = p.MsH + (in ? (q - 1) * ncp + co[k] : 0);
#pragma unroll
                    for (int c = 0; c < 3; ++c) cp_elem(sm.c.p(s, t, c), src + c * p.cs, in);
                }
            }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    load_plane(z0 - 1, 0);
    load_plane(z0, 1);
    const T dt = (NK >= 0 || NK == kErr) && p.ctl ? (T)p.ctl->dt : T(0);
    const double dt64 = NK >= 0 && p.ctl ? p.ctl->dt : 0.0;
    // cells on both sides of the node along x and y
    const bool bx = n1 >= 1 && n1 < p.N1, by = n2 >= 1 && n2 < p.N2;
    const bool active = n1 < p.nn1 && n2 < p.nn2;
    // carried up the walk: the part of the node being completed that planes z - 1 and z gave, the share of plane z in the
    // node above, m and the cell sum of plane z
    Vec<T> acc = vzero<T>(), up = acc, mc = acc, cc = acc;
    T accR = 0, upR = 0;
    double err = 0.0;  // (kErr; unused and gone otherwise)
    int s = 0;
    for (int q = z0 - 1; q <= z1; ++q) {
        ErrIn ei;
        if constexpr (NK == kErr) {
            if (q - 1 >= z0 && active) ei = load_err<T>(p, (q - 1) * np + n2 * p.nn1 + n1);
        }
        asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        __syncthreads();  // plane q has arrived for all; slot (s + 2) mod 3 (plane q - 1) is free
        load_plane(q + 2 <= z1 ? q + 2 : -1, s + 2 >= kUSlots ? s + 2 - kUSlots : s + 2);
        Vec<T> own = vzero<T>(), fin = own, mnew = own, ccur = own, dz = own;
        T nz = 1;
        T ownR = 0, finR = 0;
        if (q >= 0 && q < p.nn3) {
            const int i = (ty + 1) * S::SX + tx + 1;
            mnew = sm.y.get(s, i);
            nz = q >= 1 && q < p.N3 ? T(2) : T(1);  // cells on both sides along z
            Vec<T> P;                               // 36 M1 M2 m / (dx dy)
            if constexpr (sizeof(T) == 4) {
                auto diff = [&](int o) { return vsub(sm.y.get(s, i + o), mnew); };
                const Vec<T> X = vadd(diff(-1), diff(1)), Y = vadd(diff(-S::SX), diff(S::SX));
                const Vec<T> C = vadd(vadd(diff(-S::SX - 1), diff(S::SX + 1)), vadd(diff(1 - S::SX), diff(S::SX - 1)));
                fin = vfma(p.vs, C, vfma(p.v2, Y, vmul(p.v1, X)));     // share in the nodes of the planes beside
                own = vfma(p.ws, C, vfma(p.w2[0], Y, vmul(p.w1[0], X)));  // share in the plane's own node
                if (q >= 1) {
                    const Vec<T> d = vsub(mnew, mc);
                    dz = vfma(p.vz, d, vmul(p.vzl, d));
                }
                P = vfma(T(36), mnew, vfma(T(4), vadd(X, Y), C));
            } else {
                // row sums along x of rows n2 - 1 .. n2 + 1: a = 6 M1 m / dx, d = -dx K1 m
                Vec<T> a[3], d[3];
#pragma unroll
                for (int r = 0; r < 3; ++r) {
                    const int j = i + (r - 1) * S::SX;
                    const Vec<T> c = sm.y.get(s, j), e = vadd(sm.y.get(s, j - 1), sm.y.get(s, j + 1));
                    a[r] = vfma(T(4), c, e);
                    d[r] = vfma(T(-2), c, e);
                }
                const Vec<T> as = vadd(a[0], a[2]), ds = vadd(d[0], d[2]);
                P = vfma(T(4), a[1], as);
                const Vec<T> Q = vfma(p.cx, vfma(T(4), d[1], ds), vmul(p.cy, vfma(T(-2), a[1], as)));
                fin = vfma(p.cz, P, Q);
                own = vfma(T(2), Q, vmul(-p.cz, P));
            }
            T px, py, pz;
            vget(P, px, py, pz);
            finR = p.e0 * px + p.e1 * py + p.e2 * pz;
            ownR = T(2) * nz * finR;
        }
        // Ms H over the four cells of plane q - 1 around the node
        if (p.MsH && q >= 1 && q - 1 < p.N3) {
            const int i = ty * S::CX + tx;
            ccur = vadd(vadd(sm.c.get(s, i), sm.c.get(s, i + 1)),
                        vadd(sm.c.get(s, i + S::CX), sm.c.get(s, i + S::CX + 1)));
        }
        const int z = q - 1;
        if (z >= z0 && active) {
            const int n = z * np + n2 * p.nn1 + n1;
            T hx, hy, hz, cx, cy, cz, mx, my, mz;
            vget(vadd(acc, sizeof(T) == 4 ? vadd(dz, fin) : fin), hx, hy, hz);
            const T ps = accR + finR, pe = sizeof(T) == 4 ? fma(p.can, ps, p.canl * ps) : p.can * ps;
            hx += p.e0 * pe;
            hy += p.e1 * pe;
            hz += p.e2 * pe;
            vget(vadd(cc, ccur), cx, cy, cz);
            vget(mc, mx, my, mz);
            if (p.Msh && p.zee) {
                T sx = 0, sy = 0, sz = 0;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int c1 = n1 - ((i >> 2) & 1), c2 = n2 - ((i >> 1) & 1), c3 = z - (i & 1);
                    if (c1 >= 0 && c1 < p.N1 && c2 >= 0 && c2 < p.N2 && c3 >= 0 && c3 < p.N3) {
                        const int c = (c3 * p.N2 + c2) * p.N1 + c1;
                        sx += p.Msh[c];
                        sy += p.Msh[p.cs + c];
                        sz += p.Msh[2 * p.cs + c];
                    }
                }
                cx += sm.hf[3] * sx;
                cy += sm.hf[3] * sy;
                cz += sm.hf[3] * sz;
            }
            cx *= p.mu0V8;
            cy *= p.mu0V8;
            cz *= p.mu0V8;
            if (p.hdmi) {
                cx += p.hdmi[n];
                cy += p.hdmi[p.ns + n];
                cz += p.hdmi[2 * p.ns + n];
            }
            // f (1 + wl) h + c, where f (1 + wl) is no FP32 number
            auto corrected = [&](T &x, T &y, T &z, T f, T ax, T ay, T az) {
                const T l = f * p.wl;
                x = fma(f, x, sizeof(T) == 4 ? fma(l, x, ax) : ax);
                y = fma(f, y, sizeof(T) == 4 ? fma(l, y, ay) : ay);
                z = fma(f, z, sizeof(T) == 4 ? fma(l, z, az) : az);
            };
            // (powers of two: the share of the node's cells in those of a node inside, and its inverse)
            if (p.raw) {
                const T f = (bx ? T(1) : T(0.5)) * (by ? T(1) : T(0.5));
                corrected(hx, hy, hz, f, cx, cy, cz);
            } else {
                const T fz = z >= 1 && z < p.N3 ? T(1) : T(2), im = p.im1 * fz * (bx ? T(1) : T(2)) * (by ? T(1) : T(2));
                corrected(hx, hy, hz, fz, im * cx, im * cy, im * cz);
                if (p.zee) {
                    hx += sm.hf[0];
                    hy += sm.hf[1];
                    hz += sm.hf[2];
                }
            }
            err += (double)node_u_out<T, NK, M64>(p, n, hx, hy, hz, mx, my, mz, dt, dt64, true, ei);
        }
        acc = vfma(nz, own, sizeof(T) == 4 ? vsub(up, dz) : up);
        accR = upR + ownR;
        up = fin;
        upR = finR;
        mc = mnew;
        cc = ccur;
        s = s + 1 >= kUSlots ? 0 : s + 1;
    }
    if constexpr (NK == kErr) {
        __shared__ double sh[33];
        dp5_finish(err, p.partials, p.n_active, p.control, p.max_rej, sh);
    }
    if constexpr (NK == kRk4) rk4_finish(p.control);
}

// The same operators for the 2D nodal basis (one node layer, constant over the N3 cell layers): the field is
//   -2 A (K1 M2 + M1 K2) m + 2 Ku e (M1 M2) (e . m), both times the film's thickness,
// one thread per node, neighbours and cells through L1.  Each operator is a combination of sums of differences to
// the node itself, X of the neighbours along x, Y along y and C of the corners, in which an index beyond an end is
// moved to the end (the weights take out what that adds):
//   exchange w1 X + w2 Y + ws C,   36 M1 M2 u / (dx dy) = 9 nx ny u + (3 ny - 2) X + (3 nx - 2) Y + C.
// Differences of close values are exact, so the exchange field keeps its relative accuracy on smooth states, where sums
// of the values themselves cancel (FP32, 200x200 cells, a rotation by 0.01 rad a cell: relative error inside 6.8e-4
// with such sums, 3.1e-7 here).  Bound by instruction issue and L1 latency: 30.2 us a stage of a Dormand-Prince step at
// 1024x1024x1 (events around each launch; 29.7 us with sums of values), against 52.4 us with the assembled 9-point
// weights of the general 2D kernel, which sums A, Ku and the cell weights of every layer at every node.
constexpr int kU2X = 32, kU2Y = 4;
constexpr int kErrBlocks = 8 * 152;  // blocks of the instances that end a step: eight per SM
template <typename T, int NK, bool M64>
__device__ __forceinline__ T node2d_u(const NodeUArgs<T> &p, int n1, int n2)
{
    const int n = n2 * p.nn1 + n1;
    ErrIn ei;
    if constexpr (NK == kErr) ei = load_err<T>(p, n);
    const T dt = (NK >= 0 || NK == kErr) && p.ctl ? (T)p.ctl->dt : T(0);
    const double dt64 = NK >= 0 && p.ctl ? p.ctl->dt : 0.0;
    const bool xl = n1 >= 1, xh = n1 < p.N1, yl = n2 >= 1, yh = n2 < p.N2;
    const T nx = xl && xh ? T(2) : T(1), ny = yl && yh ? T(2) : T(1);
    const int xm = xl ? -1 : 0, xp = xh ? 1 : 0, rm = yl ? -p.nn1 : 0, rp = yh ? p.nn1 : 0;
    const T w1 = ny == T(2) ? p.w1[0] : p.w1[1], w2 = nx == T(2) ? p.w2[0] : p.w2[1];
    T h[3], m[3], P[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const T *q = p.y + c * p.ns + n;
        const T u = q[0], X = (q[xm] - u) + (q[xp] - u), Y = (q[rm] - u) + (q[rp] - u);
        const T C = ((q[rm + xm] - u) + (q[rp + xp] - u)) + ((q[rm + xp] - u) + (q[rp + xm] - u));
        m[c] = u;
        h[c] = fma(p.ws, C, fma(w2, Y, w1 * X));
        P[c] = fma(T(9) * nx * ny, u, fma(T(3) * nx - T(2), Y, fma(T(3) * ny - T(2), X, C)));
    }
    const T pe = p.can * (p.e0 * P[0] + p.e1 * P[1] + p.e2 * P[2]);
    h[0] += p.e0 * pe;
    h[1] += p.e1 * pe;
    h[2] += p.e2 * pe;
    // Ms H (and the cell field) over the in-plane cells of every layer
    auto cells = [&](const T *f, T s) {
        T sum[3] = {0, 0, 0};
        for (int c3 = 0; c3 < p.N3; ++c3) {
            const T *q = f + (c3 * p.N2 + n2) * p.N1 + n1;
#pragma unroll
            for (int c = 0; c < 3; ++c, q += p.cs)
                sum[c] += ((xl && yl ? q[-p.N1 - 1] : T(0)) + (xh && yl ? q[-p.N1] : T(0))) +
                          ((xl && yh ? q[-1] : T(0)) + (xh && yh ? q[0] : T(0)));
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) h[c] += p.im1 * (p.mu0V8 * s * sum[c]);
    };
    const double t = NK != kHeff && p.ctl ? p.ctl->t + p.c_s * p.ctl->dt : p.t_fixed;
    if (p.MsH) cells(p.MsH, T(1));
    if (p.Msh && p.zee) cells(p.Msh, (T)u_time_factor<T>(p.hc_freq, p.hc_phase, t));
    if (!p.raw) {
        // (the weights hold 1 / mass of a node with one cell column; the others have two or four)
        const T im = (nx == T(2) ? T(0.5) : T(1)) * (ny == T(2) ? T(0.5) : T(1));
#pragma unroll
        for (int c = 0; c < 3; ++c) h[c] *= im;
        if (p.zee) {
            const double su = u_time_factor<T>(p.hu_freq, p.hu_phase, t);
            h[0] += (T)(p.hu0 * su);
            h[1] += (T)(p.hu1 * su);
            h[2] += (T)(p.hu2 * su);
        }
    }
    return node_u_out<T, NK, M64>(p, n, h[0], h[1], h[2], m[0], m[1], m[2], dt, dt64, true, ei);
}
template <typename T, int NK, bool M64>
__global__ void __launch_bounds__(kU2X *kU2Y) k_node2d_u(const __grid_constant__ NodeUArgs<T> p)
{
    pdl_enter();
    if constexpr (NK == kErr) {
        if (dp5_idle(p.control)) return;
    } else if (NK != kHeff && p.ctl && p.ctl->done) {
        return;
    }
    auto node = [&](int tile) {
        const int n1 = tile % p.bxn * kU2X + threadIdx.x % kU2X, n2 = tile / p.bxn * kU2Y + threadIdx.x / kU2X;
        return n1 < p.nn1 && n2 < p.nn2 ? node2d_u<T, NK, M64>(p, n1, n2) : T(0);
    };
    if constexpr (NK == kErr) {
        // (a block for every tile spends more on its part of the reduction than on its 128 nodes)
        __shared__ double sh[33];
        double err = 0.0;
        for (int tile = blockIdx.x; tile < p.full; tile += gridDim.x) err += (double)node(tile);
        dp5_finish(err, p.partials, p.n_active, p.control, p.max_rej, sh);
    } else if constexpr (NK == kRk4) {
        for (int tile = blockIdx.x; tile < p.full; tile += gridDim.x) node(tile);
        rk4_finish(p.control);
    } else {
        node(blockIdx.x);
    }
}

template <typename T>
static void uniform_grid(const Geom &g, NodeUArgs<T> &a, int *blocks)
{
    if (g.basis == 3) {
        node_u_grid(g.nn1, g.nn2, g.nn3, sizeof(T) == 8, &a.bxn, &a.full, &a.chunks, &a.zc, blocks);
    } else {
        a.bxn = div_up(g.nn1, kU2X);
        a.full = *blocks = a.bxn * div_up(g.nn2, kU2Y);
    }
}

template <typename T>
bool uniform_error_fits(const LocalParams<T> &p)
{
    if (!p.uniform) return false;
    NodeUArgs<T> a{};
    int blocks = 0;
    uniform_grid<T>(p.g, a, &blocks);
    return blocks <= kMaxPartials;
}
template bool uniform_error_fits<float>(const LocalParams<float> &);
template bool uniform_error_fits<double>(const LocalParams<double> &);

template <typename T>
static void launch_node_uniform(const LocalParams<T> &p, const T *y, T *out, T *y_next, const StageArgs *sa, double t,
                                cudaStream_t st)
{
    const Geom &g = p.g;
    NodeUArgs<T> a = node_u_args<T>(p, y, out, y_next, sa, t);
    // weights of the sums of differences, one rounding each
    if (g.basis == 3) {
        const double f = p.raw ? 1.0 : p.uim / 8.0, cx = f * p.ucx, cy = f * p.ucy, cz = f * p.ucz;
        a.cx = (T)cx;
        a.cy = (T)cy;
        a.cz = (T)cz;
        a.w1[0] = (T)(8.0 * cx - 4.0 * cy - 4.0 * cz);
        a.w2[0] = (T)(8.0 * cy - 4.0 * cx - 4.0 * cz);
        a.ws = (T)(2.0 * cx + 2.0 * cy - cz);
        a.v1 = (T)(4.0 * cx - 2.0 * cy + 4.0 * cz);
        a.v2 = (T)(4.0 * cy - 2.0 * cx + 4.0 * cz);
        a.vs = (T)(cx + cy + cz);
        // 1 + wl: the factor that brings the rounded weights closest to the true ones, neighbour by neighbour and at the node
        // itself (with cubic cells they are multiples of one number and share its rounding, up to 6e-8: an error of every
        // exchange field that does not average out)
        const double w[6] = {8.0 * cx - 4.0 * cy - 4.0 * cz, 8.0 * cy - 4.0 * cx - 4.0 * cz, 2.0 * cx + 2.0 * cy - cz,
                             4.0 * cx - 2.0 * cy + 4.0 * cz, 4.0 * cy - 2.0 * cx + 4.0 * cz, cx + cy + cz};
        const double r[6] = {(double)a.w1[0], (double)a.w2[0], (double)a.ws, (double)a.v1, (double)a.v2, (double)a.vs};
        auto sums = [](const double *v, double *out) {
            for (int i = 0; i < 6; ++i) out[i] = (i < 3 ? 2.0 : 1.0) * v[i];
            out[6] = 2.0 * v[3] + 2.0 * v[4] + 4.0 * v[5];        // (from the node straight above or below)
            out[7] = 4.0 * v[0] + 4.0 * v[1] + 8.0 * v[2];        // (from the node itself)
        };
        const double many[8] = {2, 2, 4, 4, 4, 8, 2, 1};
        double sw[8], sr[8], rw = 0.0, rr = 0.0;
        sums(w, sw);
        sums(r, sr);
        for (int i = 0; i < 8; ++i) {
            rw += many[i] * sr[i] * sw[i];
            rr += many[i] * sr[i] * sr[i];
        }
        const double one = sizeof(T) == 4 && rr > 0.0 ? rw / rr : 1.0;
        a.wl = (T)(one - 1.0);
        a.vz = (T)(36.0 * cz / one);
        a.vzl = (T)(36.0 * cz / one - (double)a.vz);
        a.can = (T)(f * p.uan / one);
        a.canl = (T)(f * p.uan / one - (double)a.can);
        a.im1 = (T)f;
    } else {
        const double f = p.raw ? 1.0 : p.uim, cx = f * p.ucx, cy = f * p.ucy;
        a.w1[0] = (T)(4.0 * cx - 2.0 * cy);  // cells on both sides of the node along the other axis
        a.w1[1] = (T)(cx - 2.0 * cy);        // on one side
        a.w2[0] = (T)(4.0 * cy - 2.0 * cx);
        a.w2[1] = (T)(cy - 2.0 * cx);
        a.ws = (T)(cx + cy);
        a.can = (T)(f * p.uan);
        a.im1 = (T)f;
    }
    int blocks = 0;
    uniform_grid<T>(g, a, &blocks);
    node_u_dispatch<T, true>(a, sa != nullptr, [&](auto nk, auto m64) {
        constexpr int NK = decltype(nk)::value;
        constexpr bool M64 = decltype(m64)::value;
        if (g.basis == 3)
            launch_pdl(k_node_u<T, NK, M64>, blocks, kUThreads, 0, st, a);
        else
            launch_pdl(k_node2d_u<T, NK, M64>, (NK == kErr || NK == kRk4) && blocks > kErrBlocks ? kErrBlocks : blocks, kU2X * kU2Y, 0,
                       st, a);
    });
}

template <typename T>
void launch_heff_uniform(const LocalParams<T> &p, const T *y, T *h_out, double t, cudaStream_t st)
{
    launch_node_uniform<T>(p, y, h_out, nullptr, nullptr, t, st);
}
template <typename T>
void launch_llg_stage_uniform(const LocalParams<T> &p, const T *y, T *k_out, T *y_next, const StageArgs &sa,
                              cudaStream_t st)
{
    launch_node_uniform<T>(p, y, k_out, y_next, &sa, 0.0, st);
}

template void launch_heff_uniform<float>(const LocalParams<float> &, const float *, float *, double, cudaStream_t);
template void launch_heff_uniform<double>(const LocalParams<double> &, const double *, double *, double, cudaStream_t);
template void launch_llg_stage_uniform<float>(const LocalParams<float> &, const float *, float *, float *,
                                              const StageArgs &, cudaStream_t);
template void launch_llg_stage_uniform<double>(const LocalParams<double> &, const double *, double *, double *,
                                               const StageArgs &, cudaStream_t);

}  // namespace nm
