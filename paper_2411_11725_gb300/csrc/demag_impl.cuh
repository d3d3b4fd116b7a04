// Demag passes (section "Demagnetization Field"): node->cell averaging fused into a pruned
// real-to-complex x transform, pruned y transforms, a z pass that fuses forward z, the pointwise
// product with the symmetric tensor spectrum and inverse z (or, for one cell layer and for small meshes, one
// pass that fuses all of y and z), and a pruned complex-to-real x transform that writes Ms_c H_c per cell.
//
// Every kernel is instantiated per log2 transform length (the f3 engine), so the index arithmetic of
// the FFT stages is resolved at compile time.  The x passes read their input in the first FFT stage
// straight from global memory (the zero padding is never read); the forward y pass and the z passes
// stage their strided tiles in shared memory with cp.async (all copies of a tile in flight at once), the
// inverse y pass with one TMA tensor copy per tile, and the forward y pass writes its tile back with one
// TMA tensor store.  Every pass writes its
// output from the last FFT stage straight to global memory, and only the part that later passes read.
//
// Templates only: demag_f32.cu and demag_f64.cu instantiate them (two translation units, compiled in
// parallel).
#pragma once
#include <string.h>

#include "demag.cuh"
#include "fft3.cuh"

namespace nm {

// x passes: small blocks hide the gather and barrier latency best (measured against 256 and 512
// threads): the forward pass takes 128 threads (two 1024-point lines, eight blocks per SM), the inverse
// pass 64 in FP32 (one line, sixteen blocks per SM; FP64 keeps 128 threads for its 8 values per thread)
constexpr int kXThreads = 128;
template <typename T>
constexpr int kXiThreads = sizeof(T) == 4 ? 64 : 128;
// y and z passes: 512-thread blocks, two per SM in FP32 (one block's loads and barriers overlap the
// other's arithmetic); the longest y lines (2^11) take 1024 threads so that a block still spans 4 columns.
template <typename T, int LG = 0>
constexpr int kMaxThreads = 512;
template <typename T, int LG = 0>
constexpr int kMinBlocks = sizeof(T) == 4 ? 2 : 1;
// values per thread per FFT stage in the y passes: radix-16 stages for the FP32 lengths where they save a stage
// (2^10 and 2^11; 2^7 and 2^8: 12.5 against 14.8 us a pass at 512x100x8, 14.2 / 17.7 at 1000x60x12, 8.5 / 9.4 at
// 131x67x5)
template <typename T, int LG>
constexpr int kYEpt = (sizeof(T) == 4 && (LG >= 10 || LG == 7 || LG == 8)) ? 16 : 8;
constexpr int pow2_floor_c(int v)
{
    int p = 1;
    while (2 * p <= v) p *= 2;
    return p;
}
// Compile-time tile of the z convolution for lines of 2^LG: G kx columns x KY octant rows (each with its
// mirror) x 3 components, 8 values per thread, 64-byte rows where they fit (lines beyond the register tiles: ZRTile).
template <typename T, int LG>
struct ZTile {
    static constexpr int P3 = 1 << LG;
    static constexpr int EPT = 8;
    static constexpr int BUDGET = EPT * kMaxThreads<T>;
    static constexpr int G0 = (int)(64 / sizeof(Cx<T>));
    static constexpr int fit_g(int g) { return (g > 1 && 6 * g * P3 > BUDGET) ? fit_g(g / 2) : g; }
    static constexpr int G = fit_g(G0);
    static constexpr int KY = pow2_floor_c(BUDGET / (6 * G * P3)) > 0 ? pow2_floor_c(BUDGET / (6 * G * P3)) : 1;
    static constexpr int NL = 6 * KY * G;
    static constexpr int THREADS = ((NL * P3 / EPT > 32 ? NL * P3 / EPT : 32) + 31) / 32 * 32;
    static constexpr size_t SMEM = (size_t)NL * P3 * sizeof(Cx<T>) + (size_t)6 * (P3 / 2 + 1) * KY * G * sizeof(T);
    static_assert(NL * P3 <= EPT * THREADS && THREADS <= kMaxThreads<T>, "z tile exceeds the block");
};

// Compile-time tile of the y passes for lines of 2^LG: G kx columns, EPT values per thread.  Tiles of
// fewer than 16 columns pad the lines-fastest layout with one row every 8 elements (LFP = 3): the first
// stage stores with a stride of radix x G elements, which otherwise hits the same banks.
template <typename T, int LG>
struct YTile {
    static constexpr int P2 = 1 << LG;
    static constexpr int EPT = kYEpt<T, LG>;
    static constexpr int MAXT = kMaxThreads<T, LG>;
    static constexpr int G0 = pow2_floor_c(EPT * MAXT / P2);
    static constexpr int G = G0 > 16 ? 16 : (G0 < 1 ? 1 : G0);
    static constexpr int LFP = G < 16 ? 3 : 0;
    static constexpr int THREADS = ((G * P2 / EPT > 32 ? G * P2 / EPT : 32) + 31) / 32 * 32;
    static constexpr size_t SMEM = (size_t)G * f3::lf_rows(P2, LFP) * sizeof(Cx<T>), TILE_BYTES = SMEM;
    // inverse pass: the tile, up to 128 bytes to align it for the TMA copy, and the copy's barrier
    static constexpr size_t SMEM_TMA = TILE_BYTES + 128 + 16;
    static_assert(G * P2 <= EPT * THREADS && THREADS <= MAXT, "y tile exceeds the block");
    static_assert(TILE_BYTES % 8 == 0, "barrier alignment");
};

// x passes, values per thread: radix-16 stages (16) for FP32 lines of 2^10 complex values, and for those of 2^7 and 2^8,
// where they save a stage, once the lines fill the GPU with half the threads (kXWide threads or more).  Steps with 8 and 16
// values: 256x256x8 (98k threads) 489 / 472 us, 128x200x17 (82k) 594 / 590, but 128x128x16 (49k) 306 / 316, 256x256x4 (49k)
// 278 / 294, 200x50x1 (2k) 121 / 150.
constexpr long kXWide = 152 * 512;
template <typename T>
constexpr bool x_ept_choice(int LG)
{
    return sizeof(T) == 4 && (LG == 7 || LG == 8);
}
template <typename T>
static int x_ept(const Geom &g)
{
    if (sizeof(T) == 4 && g.lgQ >= 10) return 16;
    return x_ept_choice<T>(g.lgQ) && 3L * g.N2 * g.N3 * g.Q / 16 >= kXWide ? 16 : 8;
}

// Asynchronous global -> shared copies (cp.async): many in flight per thread without registers.
__device__ __forceinline__ void cpa16(void *sm, const void *gm)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(sm)),
                 "l"(gm)
                 : "memory");
}
__device__ __forceinline__ void cpa8(void *sm, const void *gm)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((unsigned)__cvta_generic_to_shared(sm)),
                 "l"(gm)
                 : "memory");
}
__device__ __forceinline__ void cpa_wait_all()
{
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}
// copy `bytes` (a multiple of 8; both addresses aligned to min(bytes, 16)) as copy number ch of a row
__device__ __forceinline__ void cpa_chunk(void *sm, const void *gm, int cb)
{
    if (cb == 16) cpa16(sm, gm);
    else cpa8(sm, gm);
}

// x-pass line L = c * (N2 N3) + row, row = zz * N2 + yy: consecutive lines of a block are consecutive
// cell rows of one component, so the node rows they average overlap.  Offsets (elements, int32: every
// supported size fits) of the line's start in the node array, the cell arrays and the spectrum.
struct XInfo {
    int in;    // node array (forward pass) or cell array (inverse pass), component included
    int cell;  // cell index of the row start (Ms map)
    int spec;  // spectrum row start
};
__device__ __forceinline__ XInfo x_info(const Geom &g, int L, bool cell)
{
    const int NR = g.N2 * g.N3;
    const int c = (int)g.nrf.div((unsigned)L);
    const int row = L - c * NR;
    const int zz = (int)g.n2f.div((unsigned)row);
    const int yy = row - zz * g.N2;
    XInfo x;
    x.cell = row * g.N1;
    x.in = cell ? c * (int)g.cs + x.cell : c * (int)g.ns + zz * g.zsn + yy * g.ysn;
    x.spec = c * (int)g.s_comp + (zz * g.P2 + yy) * g.Xp;
    return x;
}

// M of the cell pair (x, x+1) of a row: M_c = Ms_c * (1/8) sum_{i in {0,1}^3} y_{c+i}.  p points at node
// (x, yy, zz) of one component; `row` is the node offset of the upper y corners (0 with the 1D basis) and
// `plane` that of the upper z corners (0 with the 2D and 1D bases, where the 8-corner mean is the mean of
// the 4 in-plane corners, or of the 2 corners along x).
template <typename T>
__device__ __forceinline__ Cx<T> cell_M_pair(const T *__restrict__ p, int row, int plane, const T *__restrict__ Ms,
                                             T Ms0, int cell, bool has2)
{
    const T a0 = (p[0] + p[row]) + (p[plane] + p[plane + row]);
    const T a1 = (p[1] + p[row + 1]) + (p[plane + 1] + p[plane + row + 1]);
    const T ms0 = Ms ? Ms[cell] : Ms0;
    T m0 = ms0 * T(0.125) * (a0 + a1), m1 = T(0);
    if (has2) {
        const T a2 = (p[2] + p[row + 2]) + (p[plane + 2] + p[plane + row + 2]);
        const T ms1 = Ms ? Ms[cell + 1] : Ms0;
        m1 = ms1 * T(0.125) * (a1 + a2);
    }
    return cx<T>(m0, m1);
}

// Pass 1: x transform (R2C of length P1 = 2Q via a complex FFT of length Q = 2^LG on even/odd pairs).
// One block holds `lpb` consecutive lines.
template <typename T, int LG, int EPT>
__global__ void __launch_bounds__(kXThreads, sizeof(T) == 4 ? 8 : 4)
    k_x_fwd(Geom g, DemagBufs<T> b, const T *__restrict__ in, int lpb)
{
    pdl_enter();
    if (b.ctl && b.ctl->done) return;
    constexpr int Q = 1 << LG, H = Q / 2, LSZ = f3::padded(Q);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Cx<T> *buf = reinterpret_cast<Cx<T> *>(smem_raw);
    XInfo *info = reinterpret_cast<XInfo *>(buf + lpb * LSZ);
    const int nlines = 3 * g.N2 * g.N3;
    const int l0 = blockIdx.x * lpb;
    const int nl = min(lpb, nlines - l0);
    if (nl <= 0) return;
    if (threadIdx.x < nl) info[threadIdx.x] = x_info(g, l0 + threadIdx.x, false);
    __syncthreads();
    const int N1 = g.N1, row = g.ysn, plane = g.zsn;  // 2D (1D) basis: both z (y and z) corners are the node
    const T *Ms = b.Ms;
    const T Ms0 = b.Ms0;
    auto src = [&](int l, int i) -> Cx<T> {
        const int x = 2 * i;
        const XInfo xi = info[l];
        const T *p = in + xi.in + x;
        return cell_M_pair<T>(p, row, plane, Ms, Ms0, xi.cell + x, x + 1 < N1);
    };
    f3::fft<T, LG, -1, false, false, true, EPT>(buf, nl, FastDiv(1u), b.tw, g.twlg, (N1 + 1) >> 1, Q, src,
                                                         f3::NoFn<T>());
    // X_k = (Z_k + conj Z_{Q-k})/2 - (i/2) W^k (Z_k - conj Z_{Q-k}),  W = e^{-2 pi i / P1},  k = 0..Q;
    // thread (l, k) with k < Q/2 writes X_k and X_{Q-k}; k = 0 also writes X_{Q/2} (and X_0, X_Q)
    const int wsh = g.twlg - (LG + 1);
    const Cx<T> *tw = b.tw;
    auto xk = [&](Cx<T> Zk, Cx<T> Zq, int k) -> Cx<T> {
        const Cx<T> Zc = conj(Zq);
        const Cx<T> E = scale(Zk + Zc, T(0.5));
        const Cx<T> O = scale(mul_si(Zk - Zc, -1), T(0.5));
        return E + tw[k << wsh] * O;
    };
    for (int t = threadIdx.x; t < nl * H; t += blockDim.x) {
        const int l = t >> (LG - 1 < 0 ? 0 : LG - 1), k = t & (H - 1);
        const Cx<T> *z = buf + l * LSZ;
        Cx<T> *out = b.S + info[l].spec;
        if (k == 0) {
            const Cx<T> Z0 = z[0];
            out[0] = xk(Z0, Z0, 0);
            out[Q] = xk(Z0, Z0, Q);
            if (H > 0 && Q > 1) {
                const Cx<T> Zh = z[f3::pad16c(H)];
                out[H] = xk(Zh, Zh, H);
            }
        } else {
            const Cx<T> Zk = z[f3::pad16c(k)], Zq = z[f3::pad16c(Q - k)];
            out[k] = xk(Zk, Zq, k);
            out[Q - k] = xk(Zq, Zk, Q - k);
        }
    }
}

// N1 == 1 (P1 == 1): the x "transform" is a copy of the cell value (real) into kx = 0.
template <typename T>
__global__ void k_x_fwd1(Geom g, DemagBufs<T> b, const T *__restrict__ in)
{
    pdl_enter();
    if (b.ctl && b.ctl->done) return;
    const int nlines = 3 * g.N2 * g.N3;
    const int L = blockIdx.x * blockDim.x + threadIdx.x;
    if (L >= nlines) return;
    const XInfo xi = x_info(g, L, false);
    const T v = cell_M_pair<T>(in + xi.in, g.ysn, g.zsn, b.Ms, b.Ms0, xi.cell, false).x;
    b.S[xi.spec] = cx<T>(v, T(0));
}

// Pass 5: inverse x transform (C2R of length P1 via a complex FFT of length Q), keeping x < N1.
// Output per cell: Ms_c H_c and, when H is not NULL, H_c itself there.
template <typename T, int LG, int EPT>
__global__ void __launch_bounds__(kXiThreads<T>, sizeof(T) == 4 ? 16 : 4)
    k_x_inv(Geom g, DemagBufs<T> b, T *__restrict__ out, T *__restrict__ H_out, int lpb)
{
    pdl_enter();
    if (b.ctl && b.ctl->done) return;
    constexpr int Q = 1 << LG, H = Q / 2, LSZ = f3::padded(Q);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Cx<T> *buf = reinterpret_cast<Cx<T> *>(smem_raw);
    XInfo *info = reinterpret_cast<XInfo *>(buf + lpb * LSZ);
    const int nlines = 3 * g.N2 * g.N3;
    const int l0 = blockIdx.x * lpb;
    const int nl = min(lpb, nlines - l0);
    if (nl <= 0) return;
    if (threadIdx.x < nl) info[threadIdx.x] = x_info(g, l0 + threadIdx.x, true);
    __syncthreads();
    // Z_k = (X_k + conj X_{Q-k}) + i conj(W^k) (X_k - conj X_{Q-k}), k < Q, into shared memory
    const int wsh = g.twlg - (LG + 1);
    const Cx<T> *tw = b.tw;
    auto zk = [&](Cx<T> Xk, Cx<T> Xq, int k) -> Cx<T> {
        const Cx<T> Xc = conj(Xq);
        return (Xk + Xc) + mul_si((Xk - Xc) * conj(tw[k << wsh]), 1);
    };
    // the spectrum reads of KB pairs per thread are issued together, before any of them is used
    constexpr int KB = 8;
    for (int t0 = threadIdx.x; t0 < nl * H; t0 += KB * blockDim.x) {
        Cx<T> xa[KB], xb[KB];
#pragma unroll
        for (int u = 0; u < KB; ++u) {
            const int t = t0 + u * blockDim.x;
            if (t >= nl * H) break;
            const int l = t >> (LG - 1 < 0 ? 0 : LG - 1), k = t & (H - 1);
            const Cx<T> *s = b.S + info[l].spec;
            xa[u] = s[k];
            xb[u] = s[k == 0 ? Q : Q - k];
        }
#pragma unroll
        for (int u = 0; u < KB; ++u) {
            const int t = t0 + u * blockDim.x;
            if (t >= nl * H) break;
            const int l = t >> (LG - 1 < 0 ? 0 : LG - 1), k = t & (H - 1);
            Cx<T> *z = buf + l * LSZ;
            if (k == 0) {
                z[0] = zk(xa[u], xb[u], 0);
                if (H > 0 && Q > 1) {
                    const Cx<T> Xh = b.S[info[l].spec + H];
                    z[f3::pad16c(H)] = zk(Xh, Xh, H);
                }
            } else {
                z[f3::pad16c(k)] = zk(xa[u], xb[u], k);
                z[f3::pad16c(Q - k)] = zk(xb[u], xa[u], Q - k);
            }
        }
    }
    __syncthreads();
    const int N1 = g.N1;
    const T *Ms = b.Ms;
    const T Ms0 = b.Ms0;
    auto dst = [&](int l, int j, Cx<T> v) {
        const XInfo xi = info[l];
        const int x = 2 * j;
        T v0 = v.x, v1 = v.y;
        if (H_out) {
            H_out[xi.in + x] = v0;
            if (x + 1 < N1) H_out[xi.in + x + 1] = v1;
        }
        v0 *= Ms ? Ms[xi.cell + x] : Ms0;
        if (x + 1 < N1) v1 *= Ms ? Ms[xi.cell + x + 1] : Ms0;
        out[xi.in + x] = v0;
        if (x + 1 < N1) out[xi.in + x + 1] = v1;
    };
    f3::fft<T, LG, +1, false, true, false, EPT>(buf, nl, FastDiv(1u), b.tw, g.twlg, Q, (N1 + 1) >> 1, f3::NoFn<T>(), dst);
}

template <typename T>
__global__ void k_x_inv1(Geom g, DemagBufs<T> b, T *__restrict__ out, T *__restrict__ H_out)
{
    pdl_enter();
    if (b.ctl && b.ctl->done) return;
    const int nlines = 3 * g.N2 * g.N3;
    const int L = blockIdx.x * blockDim.x + threadIdx.x;
    if (L >= nlines) return;
    const XInfo xi = x_info(g, L, true);
    T v = b.S[xi.spec].x;
    if (H_out) H_out[xi.in] = v;
    v *= b.Ms ? b.Ms[xi.cell] : b.Ms0;
    out[xi.in] = v;
}

// Shared-memory barriers and TMA tile copies (cp.async.bulk.tensor): one thread issues the copy of a
// block's whole tile, which completes on an mbarrier with its byte count; the threads wait on the
// barrier's phase.  Every wait is bounded (about a second of SM clock): a wait that runs out reports
// NM_ERR_TIMEOUT through the status word and the block writes nothing.
__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned bar, unsigned parity)
{
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool mbar_wait_bounded(unsigned bar, unsigned parity)
{
    const long long t0 = clock64();
    for (unsigned it = 0; it < (1u << 26); ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if (clock64() - t0 > (2LL << 30)) break;
    }
    return false;
}
__device__ __forceinline__ void tma_load_3d(unsigned dst, const CUtensorMap *tm, int c0, int c1, int c2, unsigned bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];\n" ::"r"(dst),
        "l"((unsigned long long)tm), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void tma_load_4d(unsigned dst, const CUtensorMap *tm, int c0, int c1, int c2, int c3,
                                            unsigned bar)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
        "%5}], [%6];\n" ::"r"(dst),
        "l"((unsigned long long)tm), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
        : "memory");
}

// TMA tile store from shared memory (bulk group); the writes of the threads that filled the tile must
// be made visible to the copy first (fence_proxy_async by every writer, then a barrier)
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }
__device__ __forceinline__ void tma_store_3d(const CUtensorMap *tm, int c0, int c1, int c2, unsigned src)
{
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3}], [%4];\n" ::"l"(
                     (unsigned long long)tm),
                 "r"(c0), "r"(c1), "r"(c2), "r"(src)
                 : "memory");
}
__device__ __forceinline__ void tma_store_4d(const CUtensorMap *tm, int c0, int c1, int c2, int c3, unsigned src)
{
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3, %4}], [%5];\n" ::"l"(
                     (unsigned long long)tm),
                 "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(src)
                 : "memory");
}
// commit the issued stores and wait until they have read their shared-memory source
__device__ __forceinline__ void tma_store_commit_wait_read()
{
    asm volatile("cp.async.bulk.commit_group;\ncp.async.bulk.wait_group.read 0;\n" ::: "memory");
}

// Bytes of the inverse y pass's TMA tile copy (all P2 rows): groups of 8 rows plus the zero-filled
// padding row when the tile pads its rows (LFP = 3), plain rows otherwise (the box of demag_encode_ymap)
template <typename T, int LG>
__host__ __device__ constexpr unsigned y_tile_bytes()
{
    constexpr unsigned rowb = YTile<T, LG>::G * (unsigned)sizeof(Cx<T>), rows = 1u << LG;
    return YTile<T, LG>::LFP > 0 ? rows / 8 * 9u * rowb : rows * rowb;
}

// Passes 2 and 4: y transform of G consecutive kx columns of one (component, z) plane, in place.
// Forward reads y < N2 (zero padding above) and writes all P2; inverse reads all P2, writes y < N2.
// Shared layout: row y at buf + lfpad(y) * G (lines = columns, fastest; padded rows for narrow tiles).
//
// Forward y pass: the N2 input rows of the tile are staged with cp.async (all copies in flight at once;
// a TMA copy of the same rows measured slower here, 0.693 against 0.674 ms at 1024x1024x32).  The last
// stage writes the P2 outputs back into the tile, and one TMA store writes the whole tile (the box of
// the inverse pass's load, descriptor tm: its ninth row per group of 8 lies outside the tensor and is
// not written): 0.588 against 0.674 ms with the last stage storing to global memory itself.
template <typename T, int LG>
__global__ void __launch_bounds__(kMaxThreads<T, LG>, kMinBlocks<T, LG>)
    k_y_fwd(Geom g, DemagBufs<T> b, const __grid_constant__ CUtensorMap tm)
{
    pdl_enter();
    if (b.ctl && b.ctl->done) return;
    constexpr int P2 = 1 << LG, G = YTile<T, LG>::G, LFP = YTile<T, LG>::LFP;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // the tile at the first 128-byte boundary of the dynamic buffer (the source of the TMA store)
    const unsigned pad = (128u - (smem_u32(smem_raw) & 127u)) & 127u;
    Cx<T> *buf = reinterpret_cast<Cx<T> *>(smem_raw + pad);
    const Cx<T> *base = b.S + (long)blockIdx.y * P2 * g.Xp + blockIdx.x * G;
    const int nin = g.N2;
    const int Xp = g.Xp;
    constexpr int rowb = G * (int)sizeof(Cx<T>);
    constexpr int cb = rowb >= 16 ? 16 : rowb;
    constexpr int cpr = rowb / cb;  // copies per row
    for (int t = threadIdx.x; t < nin * cpr; t += blockDim.x) {
        const int y = t / cpr, ch = t - y * cpr;
        cpa_chunk((char *)(buf + f3::lfpad<LFP>(y) * G) + ch * cb, (const char *)(base + y * Xp) + ch * cb, cb);
    }
    cpa_wait_all();
    __syncthreads();
    f3::fft<T, LG, -1, true, true, true, kYEpt<T, LG>, G, LFP>(buf, G, FastDiv(1u), b.tw, g.twlg, nin, P2,
                                                               f3::NoFn<T>(), f3::NoFn<T>());
    fence_proxy_async();  // (the transform ends with a barrier; this one orders the copy after every fence)
    __syncthreads();
    if (threadIdx.x == 0) {
        const int x0 = 2 * G * blockIdx.x;  // real elements: a multiple of 2G, i.e. of 16 bytes
        if constexpr (LFP > 0) tma_store_4d(&tm, x0, 0, 0, blockIdx.y, smem_u32(buf));
        else tma_store_3d(&tm, x0, 0, blockIdx.y, smem_u32(buf));
        tma_store_commit_wait_read();
    }
}

// Inverse y pass: the whole P2-row tile arrives by one TMA copy (descriptor tm, built by
// demag_encode_ymap) that completes on a shared-memory barrier.  With padded rows the copy's box spans
// 9 rows of each group of 8, the ninth outside the tensor and zero-filled by the copy, so the box lands
// in the padded layout as it is.  0.610 against 0.658 ms with cp.async staging at 1024x1024x32.
template <typename T, int LG>
__global__ void __launch_bounds__(kMaxThreads<T, LG>, kMinBlocks<T, LG>)
    k_y_inv(Geom g, DemagBufs<T> b, const __grid_constant__ CUtensorMap tm)
{
    pdl_enter();
    if (b.ctl && b.ctl->done) return;
    constexpr int G = YTile<T, LG>::G, LFP = YTile<T, LG>::LFP;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // the tile at the first 128-byte boundary of the dynamic buffer, the barrier behind it
    const unsigned pad = (128u - (smem_u32(smem_raw) & 127u)) & 127u;
    Cx<T> *buf = reinterpret_cast<Cx<T> *>(smem_raw + pad);
    const unsigned bar = smem_u32(smem_raw + pad + YTile<T, LG>::TILE_BYTES);
    if (threadIdx.x == 0) mbar_init(bar, 1);
    __syncthreads();
    if (threadIdx.x == 0) {
        mbar_expect_tx(bar, y_tile_bytes<T, LG>());
        const int x0 = 2 * G * blockIdx.x;  // real elements: a multiple of 2G, i.e. of 16 bytes
        if constexpr (LFP > 0) tma_load_4d(smem_u32(buf), &tm, x0, 0, 0, blockIdx.y, bar);
        else tma_load_3d(smem_u32(buf), &tm, x0, 0, blockIdx.y, bar);
    }
    const bool arrived = mbar_wait_bounded(bar, 0);
    if (__syncthreads_or(!arrived)) {
        if (threadIdx.x == 0 && b.wait_err) atomicExch(b.wait_err, NM_ERR_TIMEOUT);
        mbar_wait_bounded(bar, 0);  // the copy may still land: let it finish before the block exits
        return;
    }
    constexpr int P2 = 1 << LG;
    Cx<T> *base = b.S + (long)blockIdx.y * P2 * g.Xp + blockIdx.x * G;
    const int Xp = g.Xp;
    auto dst = [&](int l, int i, Cx<T> v) { base[i * Xp + l] = v; };
    f3::fft<T, LG, +1, true, true, false, kYEpt<T, LG>, G, LFP>(buf, G, FastDiv(1u), b.tw, g.twlg, P2, g.N2,
                                                                f3::NoFn<T>(), dst);
}

// The six real tensor components at octant frequency (kx, a2, kz), with the sign of the odd ones in
// kz restored (Nxz odd in kz, Nyz odd in kz); the y parity is applied by the caller (s2).
template <typename T>
struct Ten6 {
    T xx, yy, zz, xy, xz, yz;
};
// H^ = N~ M^ with N~ real symmetric; s2 = -1 on the mirrored frequency P2 - a2 (Nxy and Nyz odd in ky)
template <typename T>
__device__ __forceinline__ void tensor_mul(const Ten6<T> &t, T s2, Cx<T> *px, Cx<T> *py, Cx<T> *pz)
{
    const Cx<T> mx = *px, my = *py, mz = *pz;
    const T nxy = t.xy * s2, nyz = t.yz * s2;
    *px = cx<T>(t.xx * mx.x + nxy * my.x + t.xz * mz.x, t.xx * mx.y + nxy * my.y + t.xz * mz.y);
    *py = cx<T>(nxy * mx.x + t.yy * my.x + nyz * mz.x, nxy * mx.y + t.yy * my.y + nyz * mz.y);
    *pz = cx<T>(t.xz * mx.x + nyz * my.x + t.zz * mz.x, t.xz * mx.y + nyz * my.y + t.zz * mz.y);
}

// ky of row r of a z tile whose octant rows start at a20: rows r < KY are ky = a20 + r, rows KY + r are
// the mirrors P2 - (a20 + r), present when 0 < a2 < P2/2; -1 marks an absent row
template <int KY>
__device__ __forceinline__ int z_row_ky(const Geom &g, int a20, int r)
{
    const int a2 = a20 + (r < KY ? r : r - KY);
    if (a2 >= g.H2) return -1;
    if (r < KY) return a2;
    return (a2 > 0 && a2 < (g.P2 >> 1)) ? g.P2 - a2 : -1;
}

// Stage a z tile in shared memory with cp.async: the N3 spectrum rows of its 3 x 2KY lines of G kx
// columns (element z of line l = (c * 2KY + r) * G + g at buf[z * nl + l]), then the tensor slice
// [component][a3][row][kx] behind the NL * P3 spectrum values; ends with a barrier.
template <typename T, int G, int KY, int P3>
__device__ __forceinline__ void z_tile_load(const Geom &g, const DemagBufs<T> &b, Cx<T> *buf, int kx0, int a20)
{
    constexpr int R2 = 2 * KY, nl = 3 * R2 * G, H3 = P3 / 2 + 1;
    constexpr int rowb = G * (int)sizeof(Cx<T>);
    constexpr int cb = rowb >= 16 ? 16 : rowb, lcpr = rowb / cb == 1 ? 0 : (rowb / cb == 2 ? 1 : (rowb / cb == 4 ? 2 : 3));
    const int nrow = g.N3 * 3 * R2;
    for (int t = threadIdx.x; t < (nrow << lcpr); t += blockDim.x) {
        const int rr = t >> lcpr, ch = t - (rr << lcpr);
        const int r = rr % R2, cz = rr / R2, z = cz / 3, c = cz - 3 * z;
        const int ky = z_row_ky<KY>(g, a20, r);
        if (ky < 0) continue;
        const long ga = c * g.s_comp + ((long)z * g.P2 + ky) * g.Xp + kx0;
        cpa_chunk((char *)(buf + z * nl + (c * R2 + r) * G) + ch * cb, (const char *)(b.S + ga) + ch * cb, cb);
    }
    // the tensor slice of this tile, copied while the spectrum rows arrive
    T *ten = reinterpret_cast<T *>(buf + nl * P3);
    constexpr int trowb = G * (int)sizeof(T);
    constexpr int tcb = trowb >= 16 ? 16 : trowb, tch = trowb / tcb;
    for (int t = threadIdx.x; t < 6 * H3 * KY * tch; t += blockDim.x) {
        const int row = t / tch, ch = t - row * tch;
        const int rr = row % KY, kq = row / KY, a3 = kq % H3, comp = kq / H3;
        const int a2 = a20 + rr;
        if (a2 >= g.H2) continue;
        cpa_chunk((char *)(ten + row * G) + ch * tcb,
                  (const char *)(b.Nk + comp * g.t_comp + ((long)a3 * g.H2 + a2) * g.Xp + kx0) + ch * tcb, tcb);
    }
    cpa_wait_all();
    __syncthreads();
}

// Pass 3 (N3 > 1): G kx columns x KY octant rows a2 (each with its mirror P2 - a2, so the tensor is
// read once): forward z (N3 non-zero inputs), tensor product, inverse z keeping z < N3.
// Rows r < KY are ky = a2_0 + r, rows KY + r are ky = P2 - (a2_0 + r) (present when 0 < a2 < P2/2).
// Lines l = (c * 2KY + r) * G + g; element kz of line l at buf[kz * nl + l].
template <typename T, int LG>
__global__ void __launch_bounds__(kMaxThreads<T>, kMinBlocks<T>) k_z_conv(Geom g, DemagBufs<T> b)
{
    pdl_enter();
    if (b.ctl && b.ctl->done) return;
    using Z = ZTile<T, LG>;
    constexpr int P3 = 1 << LG, H3 = P3 / 2 + 1, G = Z::G, KY = Z::KY;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Cx<T> *buf = reinterpret_cast<Cx<T> *>(smem_raw);
    const int kx0 = blockIdx.x * G, a20 = blockIdx.y * KY;
    constexpr int R2 = 2 * KY, nl = 3 * R2 * G;
    const int h2 = g.P2 >> 1;
    auto row_ky = [&](int r) -> int { return z_row_ky<KY>(g, a20, r); };
    auto gaddr = [&](int c, int ky, int z) -> long { return c * g.s_comp + ((long)z * g.P2 + ky) * g.Xp + kx0; };
    z_tile_load<T, G, KY, P3>(g, b, buf, kx0, a20);
    const FastDiv nlf(1u);  // unused: the line count is a compile-time constant
    f3::fft<T, LG, -1, true, true, true, Z::EPT, nl>(buf, nl, nlf, b.tw, g.twlg, g.N3, P3, f3::NoFn<T>(),
                                                    f3::NoFn<T>());
    constexpr int npts = KY * G * P3;
    const T *ten = reinterpret_cast<const T *>(buf + nl * P3);
    constexpr int tstride = H3 * KY * G;
    for (int t = threadIdx.x; t < npts; t += blockDim.x) {
        const int gg = t % G, q = t / G, rr = q % KY, kz = q / KY;
        const int a2 = a20 + rr;
        if (a2 >= g.H2) continue;
        const int a3 = kz <= (P3 >> 1) ? kz : P3 - kz;
        const T s3 = kz <= (P3 >> 1) ? T(1) : T(-1);
        const T *tp = ten + (a3 * KY + rr) * G + gg;
        Ten6<T> tt;
        tt.xx = tp[0];
        tt.yy = tp[tstride];
        tt.zz = tp[2 * tstride];
        tt.xy = tp[3 * tstride];
        tt.xz = tp[4 * tstride] * s3;
        tt.yz = tp[5 * tstride] * s3;
        const Ten6<T> &ten6 = tt;
        Cx<T> *p = buf + kz * nl + rr * G + gg;
        tensor_mul(ten6, T(1), p, p + R2 * G, p + 2 * R2 * G);
        if (a2 > 0 && a2 < h2) {
            Cx<T> *pm = p + KY * G;
            tensor_mul(ten6, T(-1), pm, pm + R2 * G, pm + 2 * R2 * G);
        }
    }
    __syncthreads();
    auto dst = [&](int l, int z, Cx<T> v) {
        const int gg = l % G, q = l / G, r = q % R2, c = q / R2;
        const int ky = row_ky(r);
        if (ky >= 0) b.S[gaddr(c, ky, z) + gg] = v;
    };
    f3::fft<T, LG, +1, true, true, false, Z::EPT, nl>(buf, nl, nlf, b.tw, g.twlg, P3, g.N3, f3::NoFn<T>(), dst);
}

// Register z convolution.  A thread holds all three components of one (kx, ky) line, or of the part r of it
// that a split over S threads leaves, so the tensor product needs no exchange.  The z input is zero above
// N3 <= P3/2; with S threads per line and D = P3/S the spectrum splits into S interleaved parts
//   X_{Sk+r} = sum_{m<D} e^{-2 pi i mk/D} w^{mr} sum_{j<S/2} w_S^{jr} x_{m+jD},
// w = e^{-2 pi i/P3}, w_S = w^D, and the inverse kept for z = m + jD < N3 is
//   y_{m+jD} = sum_r conj(w_S)^{jr} conj(w)^{mr} u_r[m],   u_r = length-D inverse transform of part r.
// A warp is one part of 16 kx columns of an octant row a2 (lanes 0-15) and of its mirror P2 - a2 (lanes
// 16-31), whose tensor reads coincide.
//
// Bound by latency and HBM together: four 128-thread blocks per SM at 128 registers (48 or 96 of them the spectrum).
// The tensor slice is staged with cp.async while the forward transforms run; read straight from L2 inside the
// product, its latency was exposed at every frequency (1.26 ms at 1024x1024x32).  Against the version that held one
// component's line per thread and exchanged spectra through shared memory for the product (4x the shared traffic;
// FP64 and P3 <= 4 had their own): 1.07 -> 0.89 ms at 1024x1024x32 (S = 4), 144 -> 107 us at 512x512x16 (S = 2),
// 24.7 -> 16.5 us at 256x256x8 and FP64 53 -> 39 us at 128x128x4 (S = 1, no exchange at all).
template <typename T, int LG>
struct ZRTile {
    static constexpr int P3 = 1 << LG, G = 16, THREADS = 128;
    static constexpr int DMAX = sizeof(T) == 4 ? 16 : 8;  // values per component that fit the registers
    static constexpr int S = P3 <= DMAX ? 1 : P3 / DMAX, D = P3 / S;
    static constexpr int KY = THREADS / 32 / S;  // octant rows per block
    static constexpr bool STAGE = S == 4;        // inputs staged in shared memory: every part reads all of them
    static constexpr int NZ = P3 / 2;
    static constexpr size_t IN_BYTES = STAGE ? (size_t)3 * NZ * KY * 32 * sizeof(Cx<T>) : 0;
    static constexpr size_t TEN_BYTES = (size_t)6 * (P3 / 2 + 1) * KY * G * sizeof(T);
    static constexpr size_t EX_BYTES =  // over the inputs and the tensor, once they are consumed
        S == 1 ? 0 : (size_t)3 * (S == 2 ? D : P3) * KY * 32 * sizeof(Cx<T>);
    static constexpr size_t SMEM = IN_BYTES + TEN_BYTES > EX_BYTES ? IN_BYTES + TEN_BYTES : EX_BYTES;
    static_assert(LG >= 2 && (S == 1 || S == 2 || S == 4), "register z tile");
};
// longest register z line
template <typename T>
constexpr int kZRMaxLg = sizeof(T) == 4 ? 6 : 5;

// c v for a real c, c v + w
__device__ __forceinline__ Cx<float> rmul(float c, Cx<float> v)
{
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f3::pack2(cx<float>(c, c))), "l"(f3::pack2(v)));
    return f3::unpack2(d);
}
__device__ __forceinline__ Cx<float> rfma(float c, Cx<float> v, Cx<float> w)
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;"
        : "=l"(d)
        : "l"(f3::pack2(cx<float>(c, c))), "l"(f3::pack2(v)), "l"(f3::pack2(w)));
    return f3::unpack2(d);
}
__device__ __forceinline__ Cx<double> rmul(double c, Cx<double> v) { return cx<double>(c * v.x, c * v.y); }
__device__ __forceinline__ Cx<double> rfma(double c, Cx<double> v, Cx<double> w)
{
    return cx<double>(fma(c, v.x, w.x), fma(c, v.y, w.y));
}

// H^ = N~ M^ at the frequencies kz = Sk + r held in v[component][bitrev(k)]: N~ at a3 = kz or P3 - kz, xz and
// yz odd in kz, xy and yz odd in ky (s2 = -1 on the mirrored row); the result is left in natural order, v[c][k].
// n points at the tensor of (a3 = 0, a2, kx);
// pl and tc are its strides in a3 and between components.
template <typename T, int LG, int S>
__device__ __forceinline__ void z_product(Cx<T> (&v)[3][(1 << LG) / S], const T *n, int pl, int tc, int r, T s2)
{
    constexpr int P3 = 1 << LG, D = P3 / S, H = P3 / 2;
    auto mul = [&](int k, const Ten6<T> &t, T s3) {
        Cx<T> &x = v[0][f3::bitrev<D>(k)], &y = v[1][f3::bitrev<D>(k)], &z = v[2][f3::bitrev<D>(k)];
        const T xy = t.xy * s2, yz = t.yz * (s2 * s3), xz = t.xz * s3;
        const Cx<T> a = rfma(xz, z, rfma(xy, y, rmul(t.xx, x)));
        const Cx<T> c = rfma(yz, z, rfma(t.yy, y, rmul(xy, x)));
        z = rfma(t.zz, z, rfma(yz, y, rmul(xz, x)));
        x = a;
        y = c;
    };
    auto load = [&](const T *p) {
        Ten6<T> t;
        t.xx = p[0];
        t.yy = p[tc];
        t.zz = p[2 * tc];
        t.xy = p[3 * tc];
        t.xz = p[4 * tc];
        t.yz = p[5 * tc];
        return t;
    };
    if constexpr (S == 1) {
        // (kz and P3 - kz share a tensor value)
#pragma unroll
        for (int k = 0; k <= H; ++k) {
            const Ten6<T> t = load(n + k * pl);
            mul(k, t, T(1));
            if (k > 0 && k < H) mul(P3 - k, t, T(-1));
        }
    } else {
        const T *lo = n + r * pl, *hi = n + (P3 - r) * pl;  // a3 = Sk + r up to H, P3 - r - Sk above
#pragma unroll
        for (int k = 0; k < D; ++k) {
            // (kz = H itself, k = D/2 of part 0, counts as the lower half)
            const Ten6<T> t = load(2 * k < D ? lo + S * k * pl : hi - S * k * pl);
            mul(k, t, 2 * k < D ? T(1) : (2 * k == D && r == 0 ? T(1) : T(-1)));
        }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int k = 0; k < D; ++k) {
            const int j = f3::bitrev<D>(k);
            if (j > k) {
                const Cx<T> t = v[c][k];
                v[c][k] = v[c][j];
                v[c][j] = t;
            }
        }
}

// (16-point FP32 lines spill at the 128 registers of four blocks: three blocks, 9.1 -> 8.6 us at 128x128x8)
template <typename T, int LG>
__global__ void __launch_bounds__(ZRTile<T, LG>::THREADS, sizeof(T) == 4 && LG == 4 ? 3 : 4) k_z_conv_r(Geom g, DemagBufs<T> b)
{
    pdl_enter();
    if (b.ctl && b.ctl->done) return;
    using Z = ZRTile<T, LG>;
    constexpr int P3 = Z::P3, D = Z::D, S = Z::S, H = P3 / 2, KY = Z::KY, G = Z::G, NZ = Z::NZ;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Cx<T> *buf = reinterpret_cast<Cx<T> *>(smem_raw);
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, r = wp % S, rw = wp / S;
    const int h2 = g.P2 >> 1, N3 = g.N3;
    const int mir = lane >> 4;
    int a2 = blockIdx.y * KY + rw;
    // rows past the octant and mirrors of the rows without one compute on row 0 and write nothing
    const bool valid = a2 < g.H2 && (!mir || (a2 > 0 && a2 < h2));
    if (a2 >= g.H2) a2 = 0;
    const int kx = blockIdx.x * G + (lane & 15);
    const int ky = valid && mir ? g.P2 - a2 : a2;
    const int zs = g.P2 * g.Xp;
    const int line = ky * g.Xp + kx, cstr = N3 * zs;
    if constexpr (Z::STAGE) {
        // rows of 32 lanes: element (c, z) of the block's row and mirror; zero above N3
        const int kx0 = blockIdx.x * G;
        constexpr int CP = G * (int)sizeof(Cx<T>) / 16;  // 16-byte copies per row of 16 columns
        static_assert(KY == 1 && (2 * CP) % 16 == 0 && Z::THREADS % (2 * CP) == 0, "staging");
        const int ch = threadIdx.x % (2 * CP), t0 = threadIdx.x / (2 * CP);
        const int my = ch < CP ? a2 : ((a2 > 0 && a2 < h2) ? g.P2 - a2 : a2);
        const char *src = (const char *)(b.S + my * g.Xp + kx0) + (ch % CP) * 16;
        const unsigned dst = (unsigned)__cvta_generic_to_shared(smem_raw) + ch * 16;
#pragma unroll
        for (int i = 0; i < 3 * NZ * 2 * CP / Z::THREADS; ++i) {
            const int t = t0 + i * (Z::THREADS / (2 * CP)), c = t / NZ, z = t % NZ;
            const int n = z < N3 ? 16 : 0;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst + t * (unsigned)(32 * sizeof(Cx<T>))),
                         "l"(src + (z < N3 ? (size_t)(c * cstr + z * zs) * sizeof(Cx<T>) : 0)), "r"(n)
                         : "memory");
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
    // the tensor slice [component][a3][row][kx] arrives while the forward transforms run
    T *ten = reinterpret_cast<T *>(smem_raw + Z::IN_BYTES);
    {
        constexpr int CP = G * (int)sizeof(T) / 16, RT = Z::THREADS / CP, ROWS = 6 * (H + 1) * KY;
        const int ch = threadIdx.x % CP, t0 = threadIdx.x / CP;
        const T *src = b.Nk + blockIdx.x * G + ch * (16 / (int)sizeof(T));
        const unsigned dst = (unsigned)__cvta_generic_to_shared(ten) + ch * 16;
#pragma unroll
        for (int i = 0; i < (ROWS + RT - 1) / RT; ++i) {
            const int t = t0 + i * RT, rr = t % KY, q = t / KY, a3 = q % (H + 1), c = q / (H + 1);
            const int aa = blockIdx.y * KY + rr;
            if (t < ROWS)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst + t * (unsigned)(G * sizeof(T))),
                             "l"(src + c * (int)g.t_comp + (a3 * g.H2 + (aa < g.H2 ? aa : 0)) * g.Xp)
                             : "memory");
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
    if constexpr (Z::STAGE) {
        asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        __syncthreads();
    }
    Cx<T> v[3][D];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const Cx<T> *in = b.S + line + c * cstr;
#pragma unroll
        for (int m = 0; m < D; ++m) {
            if constexpr (Z::STAGE) {
                const Cx<T> x0 = buf[(c * NZ + m) * 32 + lane], x1 = buf[(c * NZ + m + D) * 32 + lane];
                // x_m + w_4^r x_{m+D}, w_4 = -i
                const T p = r & 1 ? x1.y : x1.x, q = r & 1 ? x1.x : x1.y;
                const T sp = r == 2 || r == 3 ? T(-1) : T(1), sq = r == 1 || r == 2 ? T(-1) : T(1);
                v[c][m] = cx<T>(fma(sp, p, x0.x), fma(sq, q, x0.y));
            } else {
                v[c][m] = m < H && m < N3 ? in[m * zs] : cx<T>(T(0), T(0));
            }
        }
    }
    // twist by w^{mr}; r is the same for a whole warp.  Two parts: constants for part 1.  Four parts: from the table, the
    // same instructions for every part; with a branch of constants for each the kernel waited for its instructions more
    // than for anything else (1.03 -> 0.89 ms at 1024x1024x32; two parts 107 -> 117 us at 512x512x16, so not there).
    auto twist = [&](auto dir) {
        constexpr int DIR = decltype(dir)::value;
        if (r == 0) return;
        if constexpr (S == 4) {
            const Cx<T> *tw = b.tw;
            const int step = r << (g.twlg - LG);
#pragma unroll
            for (int m = 1; m < D; ++m) {
                const Cx<T> w = tw[m * step];
                const int i = DIR < 0 ? m : f3::bitrev<D>(m);
#pragma unroll
                for (int c = 0; c < 3; ++c) v[c][i] = f3::twmul<T, DIR>(v[c][i], w);
            }
        } else {
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
                for (int m = 1; m < D; ++m) {
                    const int i = DIR < 0 ? m : f3::bitrev<D>(m);
                    v[c][i] = f3::rot<T, P3, DIR>(v[c][i], m);
                }
        }
    };
    if constexpr (S > 1) twist(std::integral_constant<int, -1>{});
    // (two parts: the radix-4 first level takes 116 instead of 107 us at 512x512x16)
#pragma unroll
    for (int c = 0; c < 3; ++c) f3::dft_reg<T, D, -1, S != 2>(v[c]);
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    z_product<T, LG, S>(v, ten + rw * G + (lane & 15), KY * G, (H + 1) * KY * G, r, mir ? T(-1) : T(1));
#pragma unroll
    for (int c = 0; c < 3; ++c) f3::dft_reg<T, D, +1, S != 2>(v[c]);
    if constexpr (S > 1) twist(std::integral_constant<int, +1>{});
    if constexpr (S == 1) {
        if (!valid) return;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            Cx<T> *out = b.S + line + c * cstr;
#pragma unroll
            for (int m = 0; m < NZ; ++m)
                if (m < N3) out[m * zs] = v[c][f3::bitrev<D>(m)];
        }
    } else if constexpr (S == 2) {
        // part 0 writes z < D/2, part 1 the others: each sends the half that it does not write
        constexpr int F = D / 2;
        Cx<T> *ex = buf + (rw * 2) * (3 * F * 32) + lane;
        __syncthreads();  // the tensor has been read
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int i = 0; i < F; ++i) {
                const Cx<T> u0 = v[c][f3::bitrev<D>(i)], u1 = v[c][f3::bitrev<D>(i + F)];
                ex[(r * 3 + c) * F * 32 + i * 32] = r == 0 ? u1 : u0;
            }
        __syncthreads();
        if (!valid) return;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            Cx<T> *out = b.S + line + c * cstr;
#pragma unroll
            for (int i = 0; i < F; ++i) {
                const Cx<T> u0 = v[c][f3::bitrev<D>(i)], u1 = v[c][f3::bitrev<D>(i + F)];
                const Cx<T> own = r == 0 ? u0 : u1;
                const int z = i + r * F;
                if (z < N3) out[z * zs] = f3::csum(own, ex[((r ^ 1) * 3 + c) * F * 32 + i * 32]);
            }
        }
    } else {
        // thread r writes z = m and m + D for its quarter of the m: the four parts meet in shared memory
        constexpr int F = D / 4;
        __syncthreads();  // every part has read the staged inputs and the tensor
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int m = 0; m < D; ++m) buf[((c * 4 + r) * D + m) * 32 + lane] = v[c][f3::bitrev<D>(m)];
        __syncthreads();
        if (!valid) return;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            Cx<T> *out = b.S + line + c * cstr;
#pragma unroll
            for (int i = 0; i < F; ++i) {
                const int m = r * F + i;
                const Cx<T> *p = buf + (c * 4 * D + m) * 32 + lane;
                const Cx<T> t0 = p[0], t1 = p[D * 32], t2 = p[2 * D * 32], t3 = p[3 * D * 32];
                // j = 0: plain sum; j = 1: conj(w_4)^r = (i)^r
                if (m < N3) out[m * zs] = f3::csum(f3::csum(t0, t2), f3::csum(t1, t3));
                if (m + D < N3) out[(m + D) * zs] = f3::csum(f3::cdiff(t0, t2), mul_si(f3::cdiff(t1, t3), 1));
            }
        }
    }
}

// Fused y-z convolution (FP32 P3 <= 16, FP64 P3 <= 8): one block holds all N3 planes of the three components of
// G kx columns, P2 rows each, in shared memory and runs forward y, z convolution and inverse y on them, so
// the spectrum padded along y never reaches global memory and three launches become one.
//
// One block of 512 threads (FP64: 256) works through its phases in turn, so their latencies bound it.  Against the
// passes it replaces (for one layer a fused y pass that held a line's stage in registers, one column per block at
// this length): 76 against 126 us at 1024x1024x1, 23 / 31 at 512x512x1, FP64 19 / 53 at 64x64x1 and 46 / 63 (three
// launches) at 64x64x4.  (Events around each launch, about 5 us of each figure the gap between them.)
//
// The y transforms are in place: decimation in frequency forward (the frequencies end in digit-reversed
// rows), decimation in time inverse (from digit-reversed rows back to natural ones), one barrier per stage
// and any number of butterflies per thread.  The first stage reads the N2 input rows from global memory, the
// last one writes the N2 output rows there.  In between a thread takes the three z lines of a (row, kx) into
// registers for the z transforms and the product.
// Row y at buf + y * nlp, line l = (c N3 + z) G + g within it; nlp = G x an odd number, so that the G columns
// of consecutive rows fall into different banks.
template <typename T>
constexpr int kYZThreads = sizeof(T) == 4 ? 512 : 256;
template <typename T>
constexpr int kYZMaxLg3 = sizeof(T) == 4 ? 4 : 3;

// One radix-2^LR stage over sub-transforms of 2^lgM rows (of 2^lgP rows in all) of nl lines.
template <typename T, int LR, int DIR, typename Ld, typename St>
__device__ __forceinline__ void yz_stage(int lgP, int lgM, int nl, const FastDiv &nlf, const Cx<T> *__restrict__ tw,
                                         int twlg, const Ld &ld, const St &st)
{
    constexpr int R = 1 << LR;
    const int lgq = lgM - LR, nb = nl << (lgP - LR), sh = twlg - lgM;
#pragma unroll 1  // (two butterflies at a time would not fit the registers)
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
        const int q = (int)nlf.div((unsigned)b), l = b - q * nl;
        const int j = q & ((1 << lgq) - 1), row = ((q >> lgq) << lgM) + j;
        Cx<T> v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = ld(l, row + (r << lgq));
        Cx<T> w[R];
        if (DIR < 0) f3::dft<T, R, DIR>(v);
        if (lgq > 0) {
            const int jj = j << sh;
            if constexpr (R == 16) {
                // (powers from four table values: see f3::stage)
                w[1] = tw[jj];
                w[2] = tw[2 * jj];
                w[4] = tw[4 * jj];
                w[8] = tw[8 * jj];
                w[3] = w[1] * w[2];
                w[5] = w[4] * w[1];
                w[6] = w[4] * w[2];
                w[7] = w[4] * w[3];
#pragma unroll
                for (int r = 9; r < 16; ++r) w[r] = w[8] * w[r - 8];
            } else {
#pragma unroll
                for (int r = 1; r < R; ++r) w[r] = tw[jj * r];
            }
        }
        if (DIR > 0 && lgq > 0) {
#pragma unroll
            for (int r = 1; r < R; ++r) v[r] = f3::twmul<T, DIR>(v[r], w[r]);
        }
        if (DIR > 0) f3::dft<T, R, DIR>(v);
        if (DIR < 0 && lgq > 0) {
#pragma unroll
            for (int r = 1; r < R; ++r) v[f3::bitrev<R>(r)] = f3::twmul<T, DIR>(v[f3::bitrev<R>(r)], w[r]);
        }
#pragma unroll
        for (int r = 0; r < R; ++r) st(l, row + (r << lgq), v[f3::bitrev<R>(r)]);
    }
}
template <typename T, int DIR, typename Ld, typename St>
__device__ __forceinline__ void yz_stage_any(int lr, int lgP, int lgM, int nl, const FastDiv &nlf,
                                             const Cx<T> *__restrict__ tw, int twlg, const Ld &ld, const St &st)
{
    if (lr == 1) yz_stage<T, 1, DIR>(lgP, lgM, nl, nlf, tw, twlg, ld, st);
    else if (lr == 2) yz_stage<T, 2, DIR>(lgP, lgM, nl, nlf, tw, twlg, ld, st);
    else if (lr == 3) yz_stage<T, 3, DIR>(lgP, lgM, nl, nlf, tw, twlg, ld, st);
    else if constexpr (sizeof(T) == 4) yz_stage<T, 4, DIR>(lgP, lgM, nl, nlf, tw, twlg, ld, st);
}

// plan: log2 radices of the forward stages, four bits each, first stage lowest
template <typename T, int LG3>
__global__ void __launch_bounds__(kYZThreads<T>, 1) k_yz_conv(Geom g, DemagBufs<T> b, int lgG, int nlp, FastDiv nlf, unsigned plan)
{
    pdl_enter();
    if (b.ctl && b.ctl->done) return;
    constexpr int P3 = 1 << LG3, NZ = P3 > 1 ? P3 / 2 : 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Cx<T> *buf = reinterpret_cast<Cx<T> *>(smem_raw);
    const int G = 1 << lgG, N3 = g.N3, N2 = g.N2, lgP = g.lgP2, zs = g.P2 * g.Xp, Xp = g.Xp;
    const int nl = 3 * N3 * G;
    Cx<T> *S = b.S + (blockIdx.x << lgG);
    auto gl = [&](int l, int y) { return (l >> lgG) * zs + (l & (G - 1)) + y * Xp; };
    auto sld = [&](int l, int y) { return buf[y * nlp + l]; };
    auto sst = [&](int l, int y, Cx<T> v) { buf[y * nlp + l] = v; };
    auto gld = [&](int l, int y) { return y < N2 ? S[gl(l, y)] : cx<T>(T(0), T(0)); };
    auto gst = [&](int l, int y, Cx<T> v) {
        if (y < N2) S[gl(l, y)] = v;
    };
    if (lgP == 0) {
        for (int l = threadIdx.x; l < nl; l += blockDim.x) sst(l, 0, gld(l, 0));
        __syncthreads();
    }
    {
        int lgM = lgP;
        for (unsigned p = plan; p; p >>= 4) {
            const int lr = p & 15;
            if (lgM == lgP) yz_stage_any<T, -1>(lr, lgP, lgM, nl, nlf, b.tw, g.twlg, gld, sst);
            else yz_stage_any<T, -1>(lr, lgP, lgM, nl, nlf, b.tw, g.twlg, sld, sst);
            lgM -= lr;
            __syncthreads();
        }
    }
    auto freq = [&](int row) {
        int ky = 0, sh = 0, rem = lgP;
        for (unsigned p = plan; p; p >>= 4) {
            const int lr = p & 15;
            rem -= lr;
            ky |= ((row >> rem) & ((1 << lr) - 1)) << sh;
            sh += lr;
        }
        return ky;
    };
    const T *nk = b.Nk + (int)(blockIdx.x << lgG);
    const int tc = (int)g.t_comp, h2 = g.P2 >> 1;
    if constexpr (P3 == 1) {
        // one layer: the product alone, the tensor values of NB points in flight together
        constexpr int NB = 4;
        const int ni = G << lgP;
        for (int i0 = threadIdx.x; i0 < ni; i0 += NB * blockDim.x) {
            Ten6<T> t[NB];
            T s2[NB];
#pragma unroll
            for (int u = 0; u < NB; ++u) {
                const int i = i0 + u * blockDim.x;
                if (i >= ni) break;
                const int ky = freq(i >> lgG), a2 = ky > h2 ? g.P2 - ky : ky;
                const T *q = nk + a2 * Xp + (i & (G - 1));
                s2[u] = ky > h2 ? T(-1) : T(1);
                t[u] = Ten6<T>{q[0], q[tc], q[2 * tc], q[3 * tc], q[4 * tc], q[5 * tc]};
            }
#pragma unroll
            for (int u = 0; u < NB; ++u) {
                const int i = i0 + u * blockDim.x;
                if (i >= ni) break;
                Cx<T> *p = buf + (i >> lgG) * nlp + (i & (G - 1));
                tensor_mul(t[u], s2[u], p, p + G, p + 2 * G);
            }
        }
    } else {
        for (int i = threadIdx.x; i < (G << lgP); i += blockDim.x) {
            const int gg = i & (G - 1), row = i >> lgG, ky = freq(row);
            const bool mir = ky > h2;
            const int a2 = mir ? g.P2 - ky : ky;
            Cx<T> *p = buf + row * nlp + gg;
            Cx<T> v[3][P3];
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
                for (int m = 0; m < P3; ++m) v[c][m] = m < NZ && m < N3 ? p[(c * N3 + m) << lgG] : cx<T>(T(0), T(0));
#pragma unroll
            for (int c = 0; c < 3; ++c) f3::dft_reg<T, P3, -1>(v[c]);
            z_product<T, LG3, 1>(v, nk + a2 * Xp + gg, g.H2 * Xp, tc, 0, mir ? T(-1) : T(1));
#pragma unroll
            for (int c = 0; c < 3; ++c) f3::dft_reg<T, P3, +1>(v[c]);
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
                for (int m = 0; m < NZ; ++m)
                    if (m < N3) p[(c * N3 + m) << lgG] = v[c][f3::bitrev<P3>(m)];
        }
    }
    __syncthreads();
    if (lgP == 0) {
        for (int l = threadIdx.x; l < nl; l += blockDim.x) gst(l, 0, sld(l, 0));
        return;
    }
    {
        // the stages in reverse order
        int lgM = 0, ns = 0;
        for (unsigned p = plan; p; p >>= 4) ++ns;
        for (int s = ns - 1; s >= 0; --s) {
            const int lr = (plan >> (4 * s)) & 15;
            lgM += lr;
            if (s > 0) {
                yz_stage_any<T, +1>(lr, lgP, lgM, nl, nlf, b.tw, g.twlg, sld, sst);
                __syncthreads();
            } else {
                yz_stage_any<T, +1>(lr, lgP, lgM, nl, nlf, b.tw, g.twlg, sld, gst);
            }
        }
    }
}

// ---------------------------------------------------------------------------------------------
static void set_smem(const void *f) { cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024); }

template <typename T>
static void init_attributes_t()
{
    f3::lg_for_each<1, 10>([&](auto c) {
        constexpr int LG = decltype(c)::value;
        constexpr int E = sizeof(T) == 4 && LG >= 10 ? 16 : 8;
        set_smem((const void *)k_x_fwd<T, LG, E>);
        set_smem((const void *)k_x_inv<T, LG, E>);
        if constexpr (x_ept_choice<T>(LG)) {
            set_smem((const void *)k_x_fwd<T, LG, 16>);
            set_smem((const void *)k_x_inv<T, LG, 16>);
        }
    });
    f3::lg_for_each<1, 11>([&](auto c) {
        constexpr int LG = decltype(c)::value;
        set_smem((const void *)k_y_fwd<T, LG>);
        set_smem((const void *)k_y_inv<T, LG>);
    });
    f3::lg_for_each<kZRMaxLg<T> + 1, 7>([&](auto c) { set_smem((const void *)k_z_conv<T, decltype(c)::value>); });
    f3::lg_for_each<2, kZRMaxLg<T>>([&](auto c) { set_smem((const void *)k_z_conv_r<T, decltype(c)::value>); });
    f3::lg_for_each<0, kYZMaxLg3<T>>([&](auto c) { set_smem((const void *)k_yz_conv<T, decltype(c)::value>); });
}


// Tile of the fused y-z convolution.  Single-layer meshes always take it.  Meshes of several layers take it where
// a column's tile is so small that the three launches it replaces cost more than its serial phases (FP32 steps,
// fused against separate: 16x16x4 107 against 117 us, 64x32x4 117 / 129, 64x64x2 125 / 132, but 128x64x4 150 / 152, 131x67x5
// 214 / 187 and 128x128x8 252 / 213; FP64: 64x64x4 602 / 664, 128x128x4 1103 / 1208, 256x256x4 3593 / 3638).  G is the widest
// tile that leaves at least 128 blocks: wider rows move whole sectors, narrower ones fill the GPU (FP32 steps with G = 1, 2,
// 4: 64x64x1 111, 115, 117 us; 200x50x1 120, 121, 123; 512x512x1 511, 392, 330; 1024x1024x1 1547, 1252, 1087).
template <typename T>
static void plan_yz(const Geom &g, DemagPlan &p)
{
    constexpr long kMaxTile = sizeof(T) == 4 ? 768 : 4096;  // values of one column, several layers
    p.yz = g.lgP3 <= kYZMaxLg3<T> && g.lgP2 <= 11 && (g.N3 == 1 || 3L * g.N3 * g.P2 <= kMaxTile);
    if (!p.yz) return;
    int lgG = sizeof(T) == 4 ? 2 : 1;
    auto bytes = [&](int lg) { return ((size_t)((3L * g.N3) | 1) << lg) * g.P2 * sizeof(Cx<T>); };
    while (lgG > 0 && (div_up(g.X, 1 << lgG) < 128 || bytes(lgG) > 200 * 1024)) --lgG;
    p.yz_lgG = lgG;
    p.yz_nlp = ((3 * g.N3) | 1) << lgG;
    p.yz_smem = bytes(lgG);
    // as many threads as a radix-8 stage has butterflies
    const int want = (((3 * g.N3) << lgG) * g.P2 / 8 + 31) / 32 * 32;
    p.yz_threads = want < 128 ? 128 : (want > kYZThreads<T> ? kYZThreads<T> : want);
    // As few stages as radix 8 (FP64 and lines up to 2^9) or 16 allows, split evenly.  2^8 in three stages with table
    // twiddles: two of radix 16 save 2 us of 131 a step at 200x100x1, but cost a quarter of the accuracy with products and a
    // tenth with table values (error of a random state's demag field at 30x100x1: 1.50e-7 and 1.30e-7 against 1.18e-7).
    // FP32: the larger radices first, more reads in flight (200x50x1 step 115 against 117 us, 200x100x1 130 / 132, 111x528x1
    // 203 / 214), but for 2^10, whose one radix-16 stage comes last, where it has no twiddles (512x512x1 255 against 260 us,
    // and more accurate: 30x400x1 1.25e-7 against 1.42e-7).  FP64: last (64x64x1 359 / 368 us, 128x128x4 1099 / 1133).
    const int RM = sizeof(T) == 4 && g.lgP2 > 8 ? 4 : 3;
    const bool larger_first = sizeof(T) == 4 && g.lgP2 != 10;
    p.yz_plan = 0;
    for (int left = g.lgP2, s = 0, ns = div_up(left, RM); left > 0; ++s, --ns) {
        const int lr = larger_first ? div_up(left, ns) : left / ns;
        p.yz_plan |= (unsigned)lr << (4 * s);
        left -= lr;
    }
}

// Launch shapes: every block transforms at most 8 (16) complex values per thread; the y and z passes take
// up to kMaxThreads<T> threads so that their rows span at least 64 bytes where the size allows.
template <typename T>
DemagPlan demag_plan(const Geom &g)
{
    DemagPlan p{};
    p.ok = true;
    const size_t cs = sizeof(Cx<T>);
    if (g.P1 > 1) {
        const int xept = x_ept<T>(g);
        p.x_ept = xept;
        int lpb = (int)((long)xept * kXThreads / g.Q);
        lpb = lpb > 64 ? 64 : lpb;
        if (lpb < 1 || g.lgQ > 10) p.ok = false;
        p.x_lpb = lpb < 1 ? 1 : lpb;
        p.x_threads = kXThreads;
        p.x_smem = (size_t)p.x_lpb * f3::padded(g.Q) * cs + (size_t)p.x_lpb * 3 * sizeof(int);
        int lpbi = (int)((long)xept * kXiThreads<T> / g.Q);  // the inverse takes the same stages (measured)
        lpbi = lpbi > 64 ? 64 : lpbi;
        if (lpbi < 1) p.ok = false;
        p.xi_lpb = lpbi < 1 ? 1 : lpbi;
        p.xi_threads = kXiThreads<T>;
        p.xi_smem = (size_t)p.xi_lpb * f3::padded(g.Q) * cs + (size_t)p.xi_lpb * 3 * sizeof(int);
    } else {
        p.x_lpb = 1;
        p.xi_lpb = 1;
        p.xi_threads = 256;
        p.xi_smem = 0;
        p.x_threads = 256;
        p.x_smem = 0;
    }
    if (g.N3 > 1) {
        // (P2 == 1: no y passes)
        p.y_G = 1;
        if (g.lgP2 > 11) p.ok = false;
        f3::lg_dispatch<1, 11>(g.lgP2, [&](auto c) {
            using Y = YTile<T, decltype(c)::value>;
            p.y_G = Y::G;
            p.y_threads = Y::THREADS;
            p.y_smem = Y::SMEM;
            p.yi_smem = Y::SMEM_TMA;
        });
        if (g.lgP3 < 2 || g.lgP3 > 7) p.ok = false;
        f3::lg_dispatch<kZRMaxLg<T> + 1, 7>(g.lgP3, [&](auto c) {
            using Z = ZTile<T, decltype(c)::value>;
            p.z_G = Z::G;
            p.z_KY = Z::KY;
            p.z_threads = Z::THREADS;
            p.z_smem = Z::SMEM;
        });
        p.z_reg = g.lgP3 <= kZRMaxLg<T>;
        if (p.z_reg) {
            f3::lg_dispatch<2, kZRMaxLg<T>>(g.lgP3, [&](auto c) {
                using Z = ZRTile<T, decltype(c)::value>;
                p.z_G = Z::G;
                p.z_KY = Z::KY;
                p.z_threads = Z::THREADS;
                p.z_smem = Z::SMEM;
            });
        }
    }
    plan_yz<T>(g, p);
    // every block holds at most (values per thread) x (threads) values of its transforms
    if (g.P1 > 1) {
        const long xept = p.x_ept;
        if ((long)p.x_lpb * g.Q > xept * p.x_threads || (long)p.xi_lpb * g.Q > xept * p.xi_threads) p.ok = false;
    }
    if (g.N3 > 1) {
        if (p.y_threads > kMaxThreads<T> * ((sizeof(T) == 4 && g.lgP2 >= 11) ? 2 : 1) ||
            p.z_threads > (p.z_reg ? 1024 : kMaxThreads<T>))
            p.ok = false;
    } else if (!p.yz) {
        p.ok = false;
    }
    // the kx grouping divides Xp (a multiple of 16)
    const int Gmax = g.N3 > 1 ? (p.y_G > p.z_G ? p.y_G : p.z_G) : 1 << p.yz_lgG;
    if (g.Xp % Gmax != 0) p.ok = false;
    if (p.x_smem > 200 * 1024 || p.xi_smem > 200 * 1024 || p.y_smem > 200 * 1024 || p.yi_smem > 200 * 1024 ||
        p.z_smem > 200 * 1024 || (p.yz && p.yz_smem > 200 * 1024))
        p.ok = false;
    return p;
}

// ---------------------------------------------------------------------------------------------
// TMA descriptor of a y-pass tile (the inverse pass's load, the forward pass's store) over
// S = [3][N3][P2][Xp] complex: every (component, z) plane holds P2 rows of Xp complex values (rows of
// Xp * sizeof(Cx<T>) bytes, a multiple of 128).  Dimensions in real elements, innermost first: the 2 Xp
// reals of a row, then (LFP = 3) the row within its group of 8 and the group, or (LFP = 0) the row, then
// the 3 N3 planes.  The box is the 2G reals of a block's G kx columns by all P2 rows of one plane: P2 / 8
// groups of 9 rows (the ninth outside the tensor, zero-filled by a load and skipped by a store: the
// padding row of the shared layout), or P2 plain rows.
using EncodeTiledFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                   const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn encode_tiled_fn()
{
    static EncodeTiledFn fn = [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return (EncodeTiledFn) nullptr;
        return (EncodeTiledFn)f;
    }();
    return fn;
}

template <typename T>
int demag_encode_ymap(const Geom &g, void *S, CUtensorMap *map)
{
    memset(map, 0, sizeof(CUtensorMap));
    if (g.N3 <= 1 || g.P2 <= 1) return 0;  // no y passes
    const EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) return -1;
    const DemagPlan p = demag_plan<T>(g);
    if (!p.ok) return -1;
    int LFP = 0;
    f3::lg_dispatch<1, 11>(g.lgP2, [&](auto c) { LFP = YTile<T, decltype(c)::value>::LFP; });
    const CUtensorMapDataType dt = sizeof(T) == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_FLOAT64;
    const cuuint64_t rowb = (cuuint64_t)g.Xp * sizeof(Cx<T>);
    const cuuint32_t ones[4] = {1, 1, 1, 1};
    CUresult r;
    if (LFP > 0) {
        const cuuint64_t dims[4] = {(cuuint64_t)2 * g.Xp, 8, (cuuint64_t)g.P2 / 8, (cuuint64_t)3 * g.N3};
        const cuuint64_t strides[3] = {rowb, 8 * rowb, (cuuint64_t)g.P2 * rowb};
        const cuuint32_t box[4] = {(cuuint32_t)(2 * p.y_G), 9, (cuuint32_t)(g.P2 / 8), 1};
        r = enc(map, dt, 4, S, dims, strides, box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    } else {
        const cuuint64_t dims[3] = {(cuuint64_t)2 * g.Xp, (cuuint64_t)g.P2, (cuuint64_t)3 * g.N3};
        const cuuint64_t strides[2] = {rowb, (cuuint64_t)g.P2 * rowb};
        const cuuint32_t box[3] = {(cuuint32_t)(2 * p.y_G), (cuuint32_t)g.P2, 1};
        r = enc(map, dt, 3, S, dims, strides, box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    }
    return r == CUDA_SUCCESS ? 0 : (int)r;
}

template <typename T>
void demag_forward(const Geom &g, const DemagBufs<T> &b, const T *y, T *MsH, cudaStream_t st, T *H)
{
    const DemagPlan p = demag_plan<T>(g);
    if (!p.ok) return;
    // (create_mesh refuses shapes without a plan or, where there are y passes, without their descriptors)
    if (g.N3 > 1 && g.P2 > 1 && !b.ymap) return;
    const int nlines = 3 * g.N2 * g.N3;
    if (g.P1 == 1) {
        launch_pdl(k_x_fwd1<T>, div_up(nlines, 256), 256, 0, st, g, b, y);
    } else {
        f3::lg_dispatch<1, 10>(g.lgQ, [&](auto c) {
            constexpr int LG = decltype(c)::value, E = sizeof(T) == 4 && LG >= 10 ? 16 : 8;
            auto kernel = k_x_fwd<T, LG, E>;
            if constexpr (x_ept_choice<T>(LG)) {
                if (p.x_ept == 16) kernel = k_x_fwd<T, LG, 16>;
            }
            launch_pdl(kernel, div_up(nlines, p.x_lpb), p.x_threads, p.x_smem, st, g, b, y, p.x_lpb);
        });
    }
    b.mark("demag_x_fwd");
    if (p.yz) {
        f3::lg_dispatch<0, kYZMaxLg3<T>>(g.lgP3, [&](auto c) {
            constexpr int LG3 = decltype(c)::value;
            launch_pdl(k_yz_conv<T, LG3>, div_up(g.X, 1 << p.yz_lgG), p.yz_threads, p.yz_smem, st, g, b, p.yz_lgG,
                       p.yz_nlp, FastDiv((unsigned)((3 * g.N3) << p.yz_lgG)), p.yz_plan);
        });
        b.mark("demag_yz_conv");
    } else {
        if (g.P2 > 1) {
            f3::lg_dispatch<1, 11>(g.lgP2, [&](auto c) {
                constexpr int LG = decltype(c)::value;
                launch_pdl(k_y_fwd<T, LG>, dim3(g.Xp / p.y_G, 3 * g.N3), p.y_threads, p.yi_smem, st, g, b, *b.ymap);
            });
            b.mark("demag_y_fwd");
        }
        if (p.z_reg) {
            f3::lg_dispatch<2, kZRMaxLg<T>>(g.lgP3, [&](auto c) {
                constexpr int LG = decltype(c)::value;
                launch_pdl(k_z_conv_r<T, LG>, dim3(g.Xp / p.z_G, div_up(g.H2, p.z_KY)), p.z_threads, p.z_smem, st, g, b);
            });
        }
        if (!p.z_reg) {
            f3::lg_dispatch<kZRMaxLg<T> + 1, 7>(g.lgP3, [&](auto c) {
                constexpr int LG = decltype(c)::value;
                launch_pdl(k_z_conv<T, LG>, dim3(g.Xp / p.z_G, div_up(g.H2, p.z_KY)), p.z_threads, p.z_smem, st, g, b);
            });
        }
        b.mark("demag_z_conv");
        if (g.P2 > 1) {
            f3::lg_dispatch<1, 11>(g.lgP2, [&](auto c) {
                constexpr int LG = decltype(c)::value;
                launch_pdl(k_y_inv<T, LG>, dim3(g.Xp / p.y_G, 3 * g.N3), p.y_threads, p.yi_smem, st, g, b, *b.ymap);
            });
            b.mark("demag_y_inv");
        }
    }
    if (g.P1 == 1) {
        launch_pdl(k_x_inv1<T>, div_up(nlines, 256), 256, 0, st, g, b, MsH, H);
    } else {
        f3::lg_dispatch<1, 10>(g.lgQ, [&](auto c) {
            constexpr int LG = decltype(c)::value, E = sizeof(T) == 4 && LG >= 10 ? 16 : 8;
            auto kernel = k_x_inv<T, LG, E>;
            if constexpr (x_ept_choice<T>(LG)) {
                if (p.x_ept == 16) kernel = k_x_inv<T, LG, 16>;
            }
            launch_pdl(kernel, div_up(nlines, p.xi_lpb), p.xi_threads, p.xi_smem, st, g, b, MsH, H, p.xi_lpb);
        });
    }
    b.mark("demag_x_inv");
}

}  // namespace nm
