// fdm_step.cuh -- pieces of the step that its kernels share: instance addressing, the loading
// law, the column pass's symbols, the celerity law and the time-step rule.
#pragma once
#include "fdm_device.cuh"
#include "fdm_fix.cuh"
#include "fdm_internal.h"

namespace fdm {

// ------------------------------------------------------------------ small helpers
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// block-wide sum, fixed order (deterministic); result valid in thread 0
__device__ __forceinline__ double block_sum(double v, double* red) {
    v = warp_sum(v);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    __syncthreads();
    if (lane == 0) red[w] = v;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x == 0) for (int i = 0; i < nw; ++i) r += red[i];
    __syncthreads();
    return r;
}
// max of non-negative values, NaN-propagating through the bit order (NaN > +inf)
__device__ __forceinline__ unsigned long long abs_bits(double v) {
    return (unsigned long long)__double_as_longlong(fabs(v));
}

// mu = E / (2 (1 + nu)) and frac = nh / nz come from the host: a division is about 12 FP64
// instructions in a chain, 64 cycles each, and the chain that ends here is what the step's column
// pass waits for on a small grid (128^2, us per step, with the divisions here and now: double words
// 45 and 42, mixed 23.6 and 22)
__device__ __forceinline__ void loading_state(const fdm_params& p, double mu, double frac, long long step, double t,
                                              double mean, double* eps, double* sig) {
    if (p.loading_mode == FDM_LOAD_STRESS) {
        *sig = p.sigma_bar13;
        *eps = (p.sigma_bar13 + mu * frac * mean) / (2.0 * mu);
    } else if (p.loading_mode == FDM_LOAD_STRAIN_RAMP || p.loading_mode == FDM_LOAD_STRAIN_RATE) {
        *eps = p.eps_bar13_0 + p.eps_bar13_rate * (p.loading_mode == FDM_LOAD_STRAIN_RAMP ? (double)step : t);
        *sig = 2.0 * mu * (*eps) - mu * frac * mean;
    } else {
        *eps = 0.5 * frac * mean;
        *sig = 0.0;
    }
}


// Instance addressing of the step kernels: a launch covers `count` instances (grid y, or z
// for the stencil).  sc == nullptr marks a set-up launch (one instance, buffer 0, always
// runs).  Otherwise instance i reads U13 from buffer sc[i].cur, and with gating on it runs
// only while its step budget sc[i].steps_left is non-zero.  Read by thread 0 only and
// broadcast, so that every thread of a block sees the same values.
struct InstCtl {
    fdm_dev_scalars* sc;
    int gated;
};

__device__ __forceinline__ void inst_state(const InstCtl& c, int inst, int* run, int* cur) {
    int r = 1, k = 0;
    if (c.sc) {
        const fdm_dev_scalars* si = c.sc + inst;
        k = si->cur;
        if (c.gated && si->steps_left == 0) r = 0;
    }
    *run = r;
    *cur = k;
}

// Neumaier step s + x with compensation c (FP64; the magnitude test on bit patterns)
__device__ __forceinline__ void neumaier_add(double& s, double& c, double x) {
    const double t = s + x;
    c += ((ubits(s) & kMagBits) >= (ubits(x) & kMagBits)) ? (s - t) + x : (x - t) + s;
    s = t;
}
// the first step, 0 + x with compensation 0 (not 0 for an infinite x)
__device__ __forceinline__ void neumaier_start(double& s, double& c, double x) {
    s = x;
    c = x - x;
}

// Multiplier modes (all include the 1/(n1 n2) normalisation):
//   COL_K         tau-hat = K U-hat, DC = sigma_bar13 (block 0 computes <U13> and loading)
//   COL_DERIV1    alpha12-hat = i xi1 U-hat  (odd symbol, 0 at the x1 Nyquist index)
//   COL_DERIV2N   alpha11-hat = -i xi2 U-hat (odd symbol, 0 at the x2 Nyquist index)
//   COL_FWD       forward transform only (no normalisation)
//   COL_INV       inverse transform only
//   COL_SYM       stress component on a plane of the 3-D cell: the quarter table Kh holds
//                 |symbol| for kx, ky >= 0 (normalisation folded in); the symbol is i times
//                 it when sym_imag, and changes sign with ky when sym_odd2 (the sign in kx
//                 never enters: kx >= 0 in the half spectrum); DC is zero
constexpr int kRedLanes = 256;  // lanes of the <U13> reduction in the column kernel
enum ColMode { COL_K = 0, COL_DERIV1 = 1, COL_DERIV2N = 2, COL_FWD = 3, COL_INV = 4, COL_SYM = 5 };

template <typename T>
struct ColArgs {
    fdm_params p;
    int mode;
    const double* row_partials;  // COL_K: per-row sums of U13 (nparts = n2 entries)
    int nparts;
    fdm_dev_scalars* sc;         // COL_K: scalars of instance 0 (block 0 writes mean/eps/sigma)
    int gated;                   // COL_K: honour the instances' step budgets
    T scl;                       // 1 / (n1 n2)
    double inv_n;                // the same (a power of two: a product with it is the quotient)
    double mu, frac;             // COL_K: shear modulus; the layer's share of the cell
    T xi1_unit, xi2_unit;        // 2 pi / (n dx): xi = k~ * unit
    int sym_odd2, sym_imag;      // COL_SYM: symbol odd in xi2; symbol imaginary
    int moderate;                // the symbol's unit (mu, xi) lies in [2^-200, 2^200]
};

template <typename T>
__device__ __forceinline__ cpx<T> col_multiplier(const ColArgs<T>& a, const T* __restrict__ Kh, int kxi,
                                                 int ky, int n1, int n2) {
    // kxi in [0, n1/2]; ky in [0, n2)
    if (a.mode == COL_K) {   // the table carries the 1/(n1 n2) normalisation
        int kyf = ky <= n2 / 2 ? ky : n2 - ky;
        return mk(Kh[(size_t)kxi * (n2 / 2 + 1) + kyf], T(0));
    }
    if (a.mode == COL_SYM) {
        int kyf = ky <= n2 / 2 ? ky : n2 - ky;
        T v = Kh[(size_t)kxi * (n2 / 2 + 1) + kyf];
        if (a.sym_odd2 && ky > n2 / 2) v = -v;
        return a.sym_imag ? mk(T(0), v) : mk(v, T(0));
    }
    if (a.mode == COL_DERIV1) {
        if (2 * kxi == n1) return mk(T(0), T(0));
        return mk(T(0), T(kxi) * a.xi1_unit * a.scl);
    }
    // COL_DERIV2N
    if (2 * ky == n2) return mk(T(0), T(0));
    int kys = ky <= n2 / 2 ? ky : ky - n2;
    return mk(T(0), -(T(kys) * a.xi2_unit) * a.scl);
}

// the symbol applied to one coefficient: real (K) or imaginary (derivatives), so two
// multiplications rather than a general complex product
template <typename T>
__device__ __forceinline__ cpx<T> col_apply(const ColArgs<T>& a, const T* __restrict__ Kh, int kxi, int ky,
                                            int n1, int n2, cpx<T> z) {
    const cpx<T> m = col_multiplier<T>(a, Kh, kxi, ky, n1, n2);
    if (a.mode == COL_K || (a.mode == COL_SYM && !a.sym_imag)) return mk(m.x * z.x, m.x * z.y);
    return mk(-(m.y * z.y), m.y * z.x);
}

// COL_K, by all threads of the block that holds the column kx = 0: <U13> from the row sums, then
// the loading state of this step; *s_sigma is set by thread 0 (a barrier must follow)
template <typename T>
__device__ __forceinline__ void loading_from_rows(const ColArgs<T>& a, int n1, int n2, int inst, double* s_red,
                                                  double* s_sigma) {
    fdm_dev_scalars* sci = a.sc + inst;
    const double* parts = a.row_partials ? a.row_partials + (size_t)inst * a.nparts : nullptr;
    // <U13> from the row sums, then the loading state of this step (Sec. 5.1).  The
    // order is fixed by n2 alone: kRedLanes compensated lane sums over a stride, then a
    // fixed tree (results do not depend on the launch shape)
    for (int v = threadIdx.x; v < kRedLanes; v += blockDim.x) {
        double s = 0.0, c = 0.0;
        if (parts && v < a.nparts) neumaier_start(s, c, parts[v]);
        for (int i = v + kRedLanes; parts && i < a.nparts; i += kRedLanes) neumaier_add(s, c, parts[i]);
        s_red[v] = s + c;
    }
    __syncthreads();
    double tot = 0.0;
    if (threadIdx.x < 32) {
        double s = 0.0, c = 0.0;
        neumaier_start(s, c, s_red[threadIdx.x]);
        for (int v = threadIdx.x + 32; v < kRedLanes; v += 32) neumaier_add(s, c, s_red[v]);
        tot = warp_sum(s + c);
    }
    if (threadIdx.x == 0) {
        double mean = parts ? sci->phi_ref + tot * a.inv_n : sci->mean_up13;
        double eps, sig;
        loading_state(a.p, a.mu, a.frac, sci->step, sci->t, mean, &eps, &sig);
        sci->mean_up13 = mean;
        sci->eps_bar13 = eps;
        sci->sigma_bar13 = sig;
        *s_sigma = sig;
    }
}
// the symbol on the packed column, z = C0 + i CN (C0, CN transforms of the real columns kx = 0 and
// kx = n1/2): each multiplied by its own symbol and repacked,
// out(ky) = (m0 + mN)/2 z(ky) + (m0 - mN)/2 conj(z(-ky))
template <typename T>
__device__ __forceinline__ cpx<T> packed_symbol(const ColArgs<T>& a, const T* __restrict__ Kh, int ky, int n1, int n2,
                                                cpx<T> z, cpx<T> zr) {
    cpx<T> m0 = col_multiplier<T>(a, Kh, 0, ky, n1, n2);
    cpx<T> mN = col_multiplier<T>(a, Kh, n1 / 2, ky, n1, n2);
    return cmul(scale(m0 + mN, T(0.5)), z) + cmul(scale(m0 - mN, T(0.5)), conj(zr));
}

enum RowMode { ROW_PLAIN = 0, ROW_TAU = 1 };

// celerity law (Sec. 3.2.3 Hamiltonian; Sec. 4.1 prescribed), parameters in the field type
template <typename T>
struct VelLaw {
    int mode;            // FDM_V_PRESCRIBED or FDM_V_STRESS
    int friction;        // tau_y != 0 and stress driven
    T v0, mobility;
    double tau_y, beta;  // lattice friction (FP64; evaluated only when friction != 0)
    FixTurns turns;      // beta for fix_cos (FP64 fields)
    const T* mfac;       // per-cell mobility factor m(x) (heterogeneous drag, Sec. 5.3), or null
};

template <typename T> VelLaw<T> make_vel(const fdm_params& p, const void* mfac = nullptr) {
    VelLaw<T> v;
    v.mfac = static_cast<const T*>(mfac);
    v.mode = p.velocity_mode;
    v.friction = (p.tau_y != 0.0 && p.velocity_mode == FDM_V_STRESS) ? 1 : 0;
    v.v0 = T(p.v0);
    v.mobility = T(p.mobility);
    v.tau_y = p.tau_y;
    v.beta = p.beta;
    v.turns = fix_turns(p.beta);
    return v;
}

// cos(x / beta).  FP64 instructions are what a friction node costs (two lanes per SM): cos() and
// the division are about 45 of them, fix_cos two and 170 integer ones.  512 x 256 in FP64 with
// mobility factors: rows inverse 41.0 us and stencil 47.2 with cos(), 32.8 and 43.0 with fix_cos (22.5
// and 38.9 without friction).  The other paths keep cos(), whose roundings their long runs amplify.
template <typename T> __device__ __forceinline__ double friction_cos(const VelLaw<T>& v, double x) {
    if constexpr (std::is_same<T, double>::value) {
        long long c;
        if (fix_cos(x, v.turns, &c)) return fix_to(c, -62);
    }
    return cos(x / v.beta);
}

template <typename T>
__device__ __forceinline__ T celerity(const VelLaw<T>& v, T tau, T up, double phi_ref) {
    if (v.mode == FDM_V_PRESCRIBED) return v.v0;
    if (!v.friction) return -(v.mobility * tau);
    const T fr = T(v.tau_y * friction_cos(v, (double)up + phi_ref));
    return v.mobility * (fr - tau);
}

// dt from the CFL rule |v0|max dt / dx = CFL (Sec. 4.3, Sec. 5.2), in FP64
__device__ __forceinline__ double cfl_dt(double vmax, double cfl, double dx, double dt_max) {
    double dtd;
    if (vmax > 0.0) {
        dtd = cfl * dx / vmax;
        if (dt_max > 0.0 && dtd > dt_max) dtd = dt_max;
    } else {
        dtd = dt_max > 0.0 ? dt_max : 0.0;
    }
    return dtd;
}

// the step's time step: the block's largest |v0| (magnitude bits of a double per thread, NaN
// above all) into the instance's maximum, and the last of the instance's `ntiles` blocks to
// finish turns it into dt, once (every block's maximum is in before its fenced increment)
__device__ __forceinline__ void step_dt_from_max(unsigned long long bits, fdm_dev_scalars* sci, unsigned ntiles,
                                                 double cfl, double dx, double dt_max) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long other = __shfl_xor_sync(0xffffffffu, bits, o);
        bits = other > bits ? other : bits;
    }
    if ((threadIdx.x & 31) == 0) atomicMax(&sci->vmax_bits, bits);
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&sci->ri_count, 1u) == ntiles - 1u) {
            __threadfence();
            const double vmax = __longlong_as_double((long long)atomicAdd(&sci->vmax_bits, 0ull));
            const double dtd = cfl_dt(vmax, cfl, dx, dt_max);
            sci->dt_next = dtd;
            sci->dt_h_next = dtd / dx;   // the stencil works in cell units
            sci->ri_count = 0u;
        }
    }
}

template <typename T>
struct RowArgs {
    VelLaw<T> vel;
    int mode;
    const void* phi0;          // ROW_TAU: the two state buffers (U13 is needed for friction)
    const void* phi1;
    fdm_dev_scalars* sc;       // ROW_TAU: scalars of instance 0
    int gated;
    int add_sigma;             // FP64: add sc's sigma_bar13 to the mean (the column pass left it out)
    T offset;                  // ROW_PLAIN: added to every output value
    double cfl, dx, dt_max;    // ROW_TAU: time-step rule (FP64)
};

// the FP64 path's transforms in block fixed point (fdm_fix.cu): launch_row_forward, launch_col
// and launch_row_inverse of double fields
cudaError_t fix_preload(int side);
cudaError_t fix_configure(int n1, int n2);
void fix_row_forward(const Dev& d, const double* src0, const double* src1, cpx<double>* spec, double* partials,
                     InstCtl ctl, int count, cudaStream_t s);
void fix_col(const Dev& d, const cpx<double>* in, cpx<double>* out, const ColArgs<double>& a, int count,
             cudaStream_t s);
void fix_row_inverse(const Dev& d, const cpx<double>* spec, double* dst, const RowArgs<double>& a, int count,
                     cudaStream_t s);
// the mixed path's transforms (fdm_f32.cu): the same for float fields
cudaError_t f32_configure(int n1, int n2);
void f32_row_forward(const Dev& d, const float* src0, const float* src1, cpx<float>* spec, double* partials,
                     InstCtl ctl, int count, cudaStream_t s);
void f32_col(const Dev& d, const cpx<float>* in, cpx<float>* out, const ColArgs<float>& a, int count, cudaStream_t s);
void f32_row_inverse(const Dev& d, const cpx<float>* spec, float* dst, const RowArgs<float>& a, int count,
                     cudaStream_t s);
void fix_tables(void* tw, int n, void* pt, int L, cudaStream_t s);

}  // namespace fdm
