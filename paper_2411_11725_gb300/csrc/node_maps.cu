// Node kernel of the trilinear basis for cell maps of Ms, A and Ku (vacuum included): exchange, uniaxial anisotropy,
// Zeeman, DMI field and the cell->node demag average, divided by the lumped nodal mass (Eqs. weak_form_impl_f,
// weak_form_impl, mass_lumping), followed by the LLG right-hand side (Eq. llg) and the next Runge-Kutta stage input.
//
// The element integrals are tensor products of the one-dimensional 2 x 2 matrices K = [1 -1; -1 1] / dx and
// M = [2 1; 1 2] dx / 6, so the cells of layer L, between node planes L and L + 1, act on both planes through sums
// over the nine in-plane neighbours o of a node,
//   A(q) = sum_o S_o wP_o (u_o(q) - u(q)),   B = sum_o S_o wZ_o (u_o(L) - u_o(L+1)),   R(q) = sum_o K_o wK_o u_o(q),
// S_o and K_o the sums of A and Ku over the (one, two or four) magnetic cells of the layer that hold n and n + o:
//   plane L gets 2 A(L) + A(L+1) + B and 2 R(L) + R(L+1), plane L + 1 gets A(L) + 2 A(L+1) - B and R(L) + 2 R(L+1).
// (The rows of the in-plane stiffness sum to zero, hence the differences.)  A block walks the layers upwards and
// carries the upper plane's share, so each layer's weights are formed once: a third of the instructions of the
// 27-point gather with the weights of eight cells at every node.  Bound by instruction issue (six blocks per SM at 80
// registers): 24 against 43 us per stage on 256x256x8 cells, 8.7 / 10.5 us on 256x64x1 (events around each launch,
// about 5 us of each figure the gap between them).
#include "node_vec.cuh"

namespace nm {

constexpr int kMNodeSlots = 4, kMCellSlots = 3;

template <typename T>
struct NodeMSmem {
    static constexpr int SX = kUX + 2, SY = kUY + 2, CX = kUX + 1, CY = kUY + 1;
    VPlanes<T, SY, SX, kMNodeSlots> y;  // node plane q in slot q - first mod 4
    VPlanes<T, CY, CX, kMCellSlots> c;  // Ms_c H_c of cell layer q - 1 in slot q - first mod 3
    T par[kMCellSlots][3][CY * CX];     // Ms, A, Ku of the same layer (where they are maps)
    T hf[4];                            // uniform applied field, time factor of the cell field
};

template <typename T>
struct NodeMArgs {
    NodeUArgs<T> u;
    const T *Ms, *A, *Ku, *inv_mass;  // cell maps or NULL: the uniform value
    T Ms0, A0, Ku0;
    T wP[4], wZ[4], wK[4];            // by pattern 2 |o1| + |o2|
    int exch, anis;
};

template <typename T, int NK, bool M64>
__global__ void __launch_bounds__(kUThreads, sizeof(T) == 4 ? 6 : 4) k_node_m(const __grid_constant__ NodeMArgs<T> a)
{
    pdl_enter();
    const NodeUArgs<T> &p = a.u;
    if (NK != kHeff && p.ctl && p.ctl->done) return;
    using S = NodeMSmem<T>;
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
    // the elements of every node plane and cell layer that this thread copies: offset within it, or -1 outside the
    // mesh (zero fill)
    constexpr int EN = (S::SX * S::SY + kUThreads - 1) / kUThreads, EC = (S::CX * S::CY + kUThreads - 1) / kUThreads;
    int no[EN], co[EC];
#pragma unroll
    for (int k = 0; k < EN; ++k) {
        const int t = threadIdx.x + k * kUThreads, r = t / S::SX, c = t - r * S::SX;
        const int i = x0 - 1 + c, j = y0 - 1 + r;
        no[k] = (i >= 0 && i < p.nn1 && j >= 0 && j < p.nn2) ? j * p.nn1 + i : -1;
    }
#pragma unroll
    for (int k = 0; k < EC; ++k) {
        const int t = threadIdx.x + k * kUThreads, r = t / S::CX, c = t - r * S::CX;
        const int i = x0 - 1 + c, j = y0 - 1 + r;
        co[k] = (i >= 0 && i < p.N1 && j >= 0 && j < p.N2) ? j * p.N1 + i : -1;
    }
    const int np = p.nn1 * p.nn2, ncp = p.N1 * p.N2;
    // node plane q into slot s, cell layer q - 1 into slot sc (planes and layers outside the mesh are not read)
    auto load_plane = [&](int q, int s, int sc) {
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
        if (q >= 1 && q - 1 < p.N3) {
#pragma unroll
            for (int k = 0; k < EC; ++k) {
                const int t = threadIdx.x + k * kUThreads;
                if (t < S::CX * S::CY) {
                    const bool in = co[k] >= 0;
                    const int c0 = in ? (q - 1) * ncp + co[k] : 0;
                    if (p.MsH) {
#pragma unroll
                        for (int c = 0; c < 3; ++c) cp_elem(sm.c.p(sc, t, c), p.MsH + c0 + c * p.cs, in);
                    }
                    if (a.Ms) cp_elem(&sm.par[sc][0][t], a.Ms + c0, in);
                    if (a.A) cp_elem(&sm.par[sc][1][t], a.A + c0, in);
                    if (a.Ku) cp_elem(&sm.par[sc][2][t], a.Ku + c0, in);
                }
            }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    // the walk takes layers z0 - 1 .. z1 - 1: planes q - 1 and q at step q = z0 .. z1
    load_plane(z0 - 1, 0, 0);
    load_plane(z0, 1, 1);
    load_plane(z0 + 1 <= z1 ? z0 + 1 : -1, 2, 2);
    const T dt = NK >= 0 && p.ctl ? (T)p.ctl->dt : T(0);
    const double dt64 = NK >= 0 && p.ctl ? p.ctl->dt : 0.0;
    const bool active = n1 < p.nn1 && n2 < p.nn2;
    // the cells (i1, i2) around the node, c = n - i, that lie in the mesh
    bool in[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int c1 = n1 - (i >> 1), c2 = n2 - (i & 1);
        in[i] = c1 >= 0 && c1 < p.N1 && c2 >= 0 && c2 < p.N2;
    }
    // carried up the walk: the lower layer's share in plane q and its cell sum
    Vec<T> up = vzero<T>(), cc = up;
    T upR = 0;
    int s1 = 1, sc = 1;  // slots of plane q and of layer q - 1
    for (int q = z0; q <= z1; ++q) {
        asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        __syncthreads();  // plane q has arrived for all; the slots of plane q - 2 and layer q - 2 are free
        load_plane(q + 2 <= z1 ? q + 2 : -1, (s1 + 2) & 3, sc + 2 >= kMCellSlots ? sc + 2 - kMCellSlots : sc + 2);
        const int s0 = (s1 + 3) & 3;
        const int z = q - 1;                       // the node plane that this layer completes
        const bool write = z >= z0 && active;
        const int n = z * np + n2 * p.nn1 + n1;
        const T im = write ? a.inv_mass[n] : T(0);
        Vec<T> A0 = vzero<T>(), A1 = A0, B = A0, R0 = A0, R1 = A0, ccur = A0;
        const int ic = (ty + 1) * S::SX + tx + 1;  // the node itself
        const Vec<T> lc = sm.y.get(s0, ic);
        if (z >= 0 && z < p.N3) {
            const Vec<T> hc = sm.y.get(s1, ic);
            // A and Ku of the four cells, zero where not magnetic
            T ca[4], ck[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int t = (ty + 1 - (i & 1)) * S::CX + tx + 1 - (i >> 1);
                const bool mag = in[i] && (a.Ms ? sm.par[sc][0][t] : a.Ms0) > T(0);
                ca[i] = mag && a.exch ? (a.A ? sm.par[sc][1][t] : a.A0) : T(0);
                ck[i] = mag && a.anis ? (a.Ku ? sm.par[sc][2][t] : a.Ku0) : T(0);
            }
#pragma unroll
            for (int o2 = -1; o2 <= 1; ++o2)
#pragma unroll
                for (int o1 = -1; o1 <= 1; ++o1) {
                    T So = 0, Ko = 0;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int i1 = i >> 1, i2 = i & 1;
                        if ((o1 == 0 || (o1 < 0) == (i1 == 1)) && (o2 == 0 || (o2 < 0) == (i2 == 1))) {
                            So += ca[i];
                            Ko += ck[i];
                        }
                    }
                    const int d = 2 * (o1 != 0) + (o2 != 0), io = ic + o2 * S::SX + o1;
                    const Vec<T> lo = sm.y.get(s0, io), hi = sm.y.get(s1, io);
                    if (d != 0) {
                        const T w = a.wP[d] * So;
                        A0 = vfma(w, vsub(lo, lc), A0);
                        A1 = vfma(w, vsub(hi, hc), A1);
                    }
                    B = vfma(a.wZ[d] * So, vsub(lo, hi), B);
                    const T k = a.wK[d] * Ko;
                    R0 = vfma(k, lo, R0);
                    R1 = vfma(k, hi, R1);
                }
            if (p.MsH) {
                const int i = ty * S::CX + tx;
                ccur = vadd(vadd(sm.c.get(sc, i), sm.c.get(sc, i + 1)),
                            vadd(sm.c.get(sc, i + S::CX), sm.c.get(sc, i + S::CX + 1)));
            }
        }
        T rx, ry, rz, sx, sy, sz;
        vget(R0, rx, ry, rz);
        vget(R1, sx, sy, sz);
        const T r0 = p.e0 * rx + p.e1 * ry + p.e2 * rz, r1 = p.e0 * sx + p.e1 * sy + p.e2 * sz;
        if (write) {
            T hx, hy, hz, dx, dy, dz, mx, my, mz;
            vget(vadd(up, vadd(vfma(T(2), A0, A1), B)), hx, hy, hz);
            const T pe = upR + (T(2) * r0 + r1);
            hx += p.e0 * pe;
            hy += p.e1 * pe;
            hz += p.e2 * pe;
            vget(vadd(cc, ccur), dx, dy, dz);
            vget(lc, mx, my, mz);
            if (p.Msh && p.zee) {
                T fx = 0, fy = 0, fz = 0;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int c1 = n1 - ((i >> 2) & 1), c2 = n2 - ((i >> 1) & 1), c3 = z - (i & 1);
                    if (c1 >= 0 && c1 < p.N1 && c2 >= 0 && c2 < p.N2 && c3 >= 0 && c3 < p.N3) {
                        const int c = (c3 * p.N2 + c2) * p.N1 + c1;
                        fx += p.Msh[c];
                        fy += p.Msh[p.cs + c];
                        fz += p.Msh[2 * p.cs + c];
                    }
                }
                dx += sm.hf[3] * fx;
                dy += sm.hf[3] * fy;
                dz += sm.hf[3] * fz;
            }
            hx += p.mu0V8 * dx;
            hy += p.mu0V8 * dy;
            hz += p.mu0V8 * dz;
            if (p.hdmi) {
                hx += p.hdmi[n];
                hy += p.hdmi[p.ns + n];
                hz += p.hdmi[2 * p.ns + n];
            }
            const bool magnetic = im > T(0);
            if (!p.raw) {
                hx *= im;
                hy *= im;
                hz *= im;
                if (p.zee && magnetic) {
                    hx += sm.hf[0];
                    hy += sm.hf[1];
                    hz += sm.hf[2];
                }
            }
            node_u_out<T, NK, M64>(p, n, hx, hy, hz, mx, my, mz, dt, dt64, magnetic);
        }
        up = vsub(vfma(T(2), A1, A0), B);
        upR = r0 + T(2) * r1;
        cc = ccur;
        s1 = (s1 + 1) & 3;
        sc = sc + 1 >= kMCellSlots ? 0 : sc + 1;
    }
    if constexpr (NK == kRk4) rk4_finish(p.control);
}

template <typename T>
static void launch_node_maps(const LocalParams<T> &p, const T *y, T *out, T *y_next, const StageArgs *sa, double t,
                             cudaStream_t st)
{
    const Geom &g = p.g;
    NodeMArgs<T> a{};
    a.u = node_u_args<T>(p, y, out, y_next, sa, t);
    a.Ms = p.Ms;
    a.A = p.A;
    a.Ku = p.Ku;
    a.Ms0 = p.Ms0;
    a.A0 = p.A0;
    a.Ku0 = p.Ku0;
    a.inv_mass = p.inv_mass;
    a.exch = (p.terms & NM_EXCH) != 0;
    a.anis = (p.terms & NM_ANIS) != 0;
    for (int d = 0; d < 4; ++d) {
        a.wP[d] = (T)p.mP[d];
        a.wZ[d] = (T)p.mZ[d];
        a.wK[d] = (T)p.mK[d];
    }
    int blocks = 0;
    node_u_grid(g.nn1, g.nn2, g.nn3, sizeof(T) == 8, &a.u.bxn, &a.u.full, &a.u.chunks, &a.u.zc, &blocks);
    node_u_dispatch<T, false>(a.u, sa != nullptr, [&](auto nk, auto m64) {
        launch_pdl(k_node_m<T, decltype(nk)::value, decltype(m64)::value>, blocks, kUThreads, 0, st, a);
    });
}

template <typename T>
void launch_heff_maps(const LocalParams<T> &p, const T *y, T *h_out, double t, cudaStream_t st)
{
    launch_node_maps<T>(p, y, h_out, nullptr, nullptr, t, st);
}
template <typename T>
void launch_llg_stage_maps(const LocalParams<T> &p, const T *y, T *k_out, T *y_next, const StageArgs &sa,
                           cudaStream_t st)
{
    launch_node_maps<T>(p, y, k_out, y_next, &sa, 0.0, st);
}

#define NM_MAPS_INST(T)                                                                                            \
    template void launch_heff_maps<T>(const LocalParams<T> &, const T *, T *, double, cudaStream_t);              \
    template void launch_llg_stage_maps<T>(const LocalParams<T> &, const T *, T *, T *, const StageArgs &,        \
                                           cudaStream_t);
NM_MAPS_INST(float)
NM_MAPS_INST(double)

}  // namespace nm
