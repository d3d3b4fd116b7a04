// Local field terms and the LLG right-hand side, fused per node.
#pragma once
#include "demag.cuh"

namespace nm {

// Per-mesh constants of the local terms.  The element integrals are tensor products of one-dimensional 2 x 2
// stiffness and mass matrices; they depend only on d = |i - i'| per direction.
template <typename T>
struct LocalParams {
    Geom g;
    // trilinear basis, by in-plane pattern d = 2 |o1| + |o2| (node_maps.cu): -2 (K1 M2 + M1 K2) dz/6 and
    // -2 M1 M2 / dz per unit A, 2 M1 M2 dz/6 per unit Ku
    T mP[4], mZ[4], mK[4];
    // Uniform material (no cell maps, Ms0 > 0; trilinear basis): node_uniform.cu.  2 A and 2 Ku (0 for terms
    // that are off) times the constants of the one-dimensional element matrices, and 1 / (mu0 V/8 Ms0).
    int uniform;
    double ucx, ucy, ucz, uan, uim;
    T mu0V8;           // mu0 * V / 8
    // 2D basis (section "Low-Dimensional Geometries"): the in-plane pattern integrals per cell layer
    // (pattern d = 2 |o1| + |o2|), through the layer's thickness, and mu0 V / 4
    T Wex2[4], Wm2[4], mu0V4;
    // interfacial DMI: raw field buffer (NULL: term off), cell map or uniform value, and the pattern
    // weights of the antisymmetric element integrals (dmx by (|o2|,|o3|), dmy by (|o1|,|o3|))
    T *hdmi;
    const T *Dm;
    T D0, dmx[4], dmy[4];
    const T *A;        // cell maps (n_cells) or NULL for the uniform value
    const T *Ku;
    const T *Ms;
    T A0, Ku0, Ms0;
    T e0, e1, e2;      // easy axis
    const T *inv_mass; // 1/mass_n, 0 where no magnetic cell touches n
    const T *MsH;      // demag: Ms_c H_c (3 x cs) or NULL
    const T *Msh;      // cell applied field times Ms: Ms_c h_c (3 x cs) or NULL
    double hu0, hu1, hu2, hu_freq, hu_phase, hc_freq, hc_phase;
    unsigned terms;
    double gam;        // gamma / (1 + alpha^2)
    T gam_t, alpha_t;  // the same in the working precision
    int raw;           // 1: output -dE (no division by the mass, no uniform applied field)
    double alpha;
    // 1D basis: the pattern integrals along x (d = |o1|) per cell of the cross-section, through its
    // area, and mu0 V / 2 (last, so that the fields above keep the offsets the other kernels were tuned
    // with)
    T Wex1[2], Wm1[2], mu0V2;
};

// What the node kernel writes.
//   out_h:   H (3 x ns) -- effective-field evaluation
//   k_out:   LLG slope k_s (3 x ns)
//   y_next:  next stage input y_{s+1} = m + dt sum_{j<=s} a_j k_j (3 x ns), when non-NULL
struct StageArgs {
    const double *m;          // FP64 master magnetisation (3 x ns)
    const float *mf;          // its FP32 copy (FP32 path; NULL = form the next input from m in FP64)
    const void *k[8];         // k_1 .. k_s (k[s-1] is the one being written)
    double a[8];              // a_{s+1, j}, j = 1 .. s
    int s;                    // stage index (1-based) of the slope being computed
    double c_s;               // time fraction of stage s
    float af[8];              // the same coefficients in FP32 (used by the FP32 path)
    double a_s;               // a_{s+1, s}: the coefficient of the slope being written (a[s - 1])
    float af_s;
    const StepCtl *ctl;       // t, dt
    double t_fixed;           // time when ctl == NULL
    // Dormand-Prince error (FP32, uniform materials): stage 6 also writes the increment dt sum_j b_j k_j of the step to
    // dinc and its part of the error combination to se; stage 7 (y_next NULL) reads se and takes the step decision
    float *se, *dinc;
    float e[5];               // error weights of k_3 .. k_7
    StepCtl *control;         // ctl, to be written by stage 7 (RK4: by stage 4)
    // RK4 (node kernels of node_uniform.cu and node_maps.cu): stage 4 ends the step when m_out is set: a and a_s are then
    // the weights b of the four slopes, m_out (= m) and its FP32 copy receive the new state, and the time advances
    double *m_out;
    float *mf_out;
    int renorm;
    double *partials;
    double n_active;
    int max_rej;
};
constexpr int kMaxPartials = 16384;  // partial sums of a reduction (the mesh's partials buffer)
// whether the uniform node kernels can form the error of a step on this mesh: a partial sum per block has a place
template <typename T>
bool uniform_error_fits(const LocalParams<T> &p);

template <typename T>
void launch_heff(const LocalParams<T> &p, const T *y, T *h_out, double t, cudaStream_t st);

template <typename T>
void launch_llg_stage(const LocalParams<T> &p, const T *y, T *k_out, T *y_next, const StageArgs &sa,
                      cudaStream_t st);

// the same for a uniform material (p.uniform) on the trilinear or 2D basis; DMI reads the raw field p.hdmi
template <typename T>
void launch_heff_uniform(const LocalParams<T> &p, const T *y, T *h_out, double t, cudaStream_t st);
template <typename T>
void launch_llg_stage_uniform(const LocalParams<T> &p, const T *y, T *k_out, T *y_next, const StageArgs &sa,
                              cudaStream_t st);

// the same for cell maps on the trilinear basis
template <typename T>
void launch_heff_maps(const LocalParams<T> &p, const T *y, T *h_out, double t, cudaStream_t st);
template <typename T>
void launch_llg_stage_maps(const LocalParams<T> &p, const T *y, T *k_out, T *y_next, const StageArgs &sa,
                           cudaStream_t st);

// lumped mass: inv_mass_n = 1 / (mu0 V/8 sum_{c∋n} Ms_c); counts magnetic nodes into *n_active (device)
template <typename T>
void launch_mass(const Geom &g, const double *Ms_d, double Ms0, double V, T *inv_mass, unsigned long long *n_active,
                 cudaStream_t st);

}  // namespace nm
