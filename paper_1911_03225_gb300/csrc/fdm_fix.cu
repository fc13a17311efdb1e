// fdm_fix.cu -- the FP64 path's transform kernels in 64-bit block fixed point (fdm_fix.cuh):
// rows of U13 to the packed half spectrum, the column pass with its symbol, and rows back to
// tau13.  Same data layouts and results (to rounding) as the kernels of fdm_kernels.cu.
//
// A block holds RB rows (or CB columns), L / 8 threads each, eight complex values per thread
// in registers; the passes exchange through two shared buffers.  The first pass takes its
// values from, and the last leaves them for, global memory in coalesced order, so shared
// memory sees only the exchanges between passes and the transposition.
//
// What bounds them: instruction issue (about 250 instructions per complex point and transform,
// half of them 64-bit additions), no longer the FP64 pipe, which keeps the conversions to
// double.  2048^2, one launch (events between the kernels), FP64 -> fixed point: rows 190 -> 50 us,
// column pass 303 -> 88, inverse rows 190 -> 64; 1024^2: 52 -> 21, 94 -> 39, 55 -> 27.
#include <type_traits>

#include "fdm_fix.cuh"
#include "fdm_step.cuh"

namespace fdm {
namespace {

// waits for the T threads of one sequence (its id in the block)
template <int T> __device__ __forceinline__ void sync_seq(int id) {
    if constexpr (T >= 32) asm volatile("bar.sync %0, %1;" ::"r"(id + 1), "n"(T) : "memory");
    else __syncwarp();
}

// The scale of one sequence: E, the exponent its integers are held at; need, the bits its
// transform may grow beyond the first pass's three (see FixPlan::shift): the sum over the
// threads of each one's largest exponent bounds the sum of all magnitudes, which bounds every
// partial transform.  pre = +-1 asks for a factor 2^(600 pre) on the values first (magnitudes
// near the ends of FP64's range); nan marks a sequence with an infinity, a NaN or a magnitude
// of 2^1023 and more (whose sums overflow FP64): its transform is NaN throughout.
struct FixScale { int E, need, pre; bool nan; };
constexpr double kUp = 0x1p600, kDown = 0x1p-600;

__device__ __forceinline__ FixScale fix_scale_of(int E, unsigned sum, int most) {
    FixScale f;
    f.nan = E >= 0x7fe;
    f.pre = 0;
    f.E = E;
    if (E < kFixLowExp) { f.pre = 1; f.E = E == 0 ? 601 : E + 600; }
    else if (E > kFixHighExp && !f.nan) { f.pre = -1; f.E = E - 600; }
    const int b = 12 - __clz((int)(sum - 1u));   // ceil(log2(sum)) - 20
    f.need = b < 0 ? 0 : (b > most ? most : b);
    return f;
}
__device__ __forceinline__ unsigned exp_unit(int E, unsigned m) {   // 2^(20 - (E - exponent)), at least 1
    const int d = E - (int)(m >> 20);
    return m == 0u ? 0u : (d > 20 ? 1u : 1u << (20 - d));
}
struct WarpStat { unsigned m, s; };

// scale of a sequence held by T consecutive threads; m: the largest fix_mag of the thread's values
template <int T>
__device__ __forceinline__ FixScale seq_scale(unsigned m, int seq, int tid, WarpStat* stat, int most) {
    if constexpr (T >= 32) {
        const unsigned wm = __reduce_max_sync(0xffffffffu, m);
        const unsigned ws = __reduce_add_sync(0xffffffffu, exp_unit((int)(wm >> 20), m));
        constexpr int NW = T / 32;
        if constexpr (NW == 1) return fix_scale_of((int)(wm >> 20), ws, most);
        if ((tid & 31) == 0) stat[tid >> 5] = WarpStat{wm, ws};
        sync_seq<T>(seq);
        int E = 0;
        unsigned s = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) E = max(E, (int)(stat[seq * NW + w].m >> 20));
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            const WarpStat q = stat[seq * NW + w];
            const int d = E - (int)(q.m >> 20);
            s += (d > 31 ? 0u : q.s >> d) + 1u;
        }
        return fix_scale_of(E, s, most);
    } else {
        unsigned wm = m;
#pragma unroll
        for (int o = 1; o < T; o <<= 1) wm = max(wm, __shfl_xor_sync(0xffffffffu, wm, o));
        unsigned ws = exp_unit((int)(wm >> 20), m);
#pragma unroll
        for (int o = 1; o < T; o <<= 1) ws += __shfl_xor_sync(0xffffffffu, ws, o);
        return fix_scale_of((int)(wm >> 20), ws, most);
    }
}

__device__ __forceinline__ unsigned mag_of(const cpx<double>* x) {
    unsigned m = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) m = max(m, max(fix_mag(x[u].x), fix_mag(x[u].y)));
    return m;
}
// eight values in the sequence's units, and, if asked for, what their rounding left (fix_from_lost);
// the branch for its rare scales keeps their products off the common path
template <bool LOST = false>
__device__ __forceinline__ void to_fixed(cpx<double>* x, cfx* v, const FixScale& f, int* lost = nullptr) {
    if (f.pre) {
        const double p = f.pre > 0 ? kUp : kDown;
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = mk(x[u].x * p, x[u].y * p);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        if constexpr (LOST) v[u] = mkx(fix_from_lost(x[u].x, f.E, *lost), fix_from_lost(x[u].y, f.E, *lost));
        else v[u] = mkx(fix_from<kFixBits, true>(x[u].x, f.E), fix_from<kFixBits, true>(x[u].y, f.E));
    }
}
// N results as doubles: integers that carry the scale sc (the sequence's units included)
template <int N> __device__ __forceinline__ void from_fixed(const cfx* v, cpx<double>* x, int sc, const FixScale& f) {
#pragma unroll
    for (int u = 0; u < N; ++u) x[u] = mk(fix_to(v[u].x, sc), fix_to(v[u].y, sc));
    if (f.pre | (int)f.nan) {
        const double p = f.nan ? __longlong_as_double(0x7ff8000000000000ll) : (f.pre > 0 ? kDown : kUp);
#pragma unroll
        for (int u = 0; u < N; ++u) x[u] = mk(f.nan ? p : x[u].x * p, f.nan ? p : x[u].y * p);
    }
}

// a sum of a row's integers as a double
__device__ __forceinline__ double row_sum(double d, const FixScale& f) {
    const cfx one = mkx(1ll << 57, 0);
    cpx<double> r;
    from_fixed<1>(&one, &r, f.E - 1080, f);
    return d * 0x1p-57 * r.x;
}

// passes p.. of the transform of the eight values of thread j of sequence `seq`; A, B: the
// sequence's places in the two shared buffers
template <int L, int S, int p = 0>
__device__ __forceinline__ void fix_transform(cfx* v, int j, int seq, cfx* A, cfx* B, const twx* __restrict__ tab,
                                              int need) {
    using Pl = FixPlan<L>;
    fix_pass<L, p, S>(v, j, tab, need);
    if constexpr (p + 1 < Pl::P) {
#pragma unroll
        for (int u = 0; u < 8; ++u) A[fix_pad(fix_place<L, p>(j, u))] = v[u];
        sync_seq<Pl::T>(seq);
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = A[fix_pad(j + u * Pl::T)];
        fix_transform<L, S, p + 1>(v, j, seq, B, A, tab, need);
    }
}

__host__ __device__ constexpr int log2i(int v) { return v <= 1 ? 0 : 1 + log2i(v / 2); }
// threads of a block: enough sequences for a full warp and up to 256 threads, three blocks per
// SM (80 registers, a few spilled: the rows of 2048^2 took 44 us so and 51 with two blocks of
// 128); 512 where one row takes 256, because the transposed accesses need two rows for 32-byte
// segments, and where one column takes 512
template <int L, bool ROWS> struct FixBlock {
    static constexpr int T = L / 8;
    static constexpr int most = T > 256 || (ROWS && T == 256) ? 512 : 256;
    static constexpr int minb = most == 512 ? 1 : 3;
};
__host__ __device__ constexpr int fix_seqs(int L, int R, bool rows) {   // sequences a block works on at a time
    int rb = (L / 8 > 256 || (rows && L / 8 == 256) ? 512 : 256) / (L / 8);
    if (rb > 8) rb = 8;
    return rb < R ? rb : R;
}
// stride of a sequence in shared memory: padded, and offset so that the transposed accesses of
// rb sequences (a power of two) fall into different banks
__host__ __device__ constexpr int fix_ld(int L, int rb) { return L + L / 8 + (rb > 1 ? 8 / rb : 0); }
__host__ __device__ constexpr int fix_threads(int L, int rb) { return rb * (L / 8) < 32 ? 32 : rb * (L / 8); }
// sequences the block's threads cover: a block of one warp may hold idle ones, which run the
// transform of zeros in places of their own
__host__ __device__ constexpr int fix_slots(int L, int rb) { return fix_threads(L, rb) / (L / 8); }
__host__ __device__ constexpr size_t fix_smem(int L, int rb) {
    return (size_t)2 * fix_slots(L, rb) * fix_ld(L, rb) * sizeof(cfx);
}
constexpr size_t fix_max_smem(int L, bool rows) {   // of any R
    size_t m = 0;
    for (int R = 1; R <= 16; R *= 2) {
        const size_t b = fix_smem(L, fix_seqs(L, R, rows));
        if (b > m) m = b;
    }
    return m;
}

// ------------------------------------------------------------------ row forward (R2C)
// grid (n2 / R, instances); see row_forward_kernel.  The row's sum (for <U13>) is taken from
// the integers and what their rounding left, to 2^-64 of the row's largest value each, and rounded
// once per thread.
template <int L>
__global__ void __launch_bounds__(FixBlock<L, true>::most, FixBlock<L, true>::minb)
    fix_row_forward_kernel(const double* src0, const double* src1, cpx<double>* spec, int n2, int R,
                           const twx* __restrict__ tw1, const twx* __restrict__ pt1, double* row_partials,
                           InstCtl ctl) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_run, s_cur;
    __shared__ WarpStat s_stat[16];
    __shared__ FixScale s_scale[8];
    __shared__ double s_sum[16];
    constexpr int T = L / 8, NW = T >= 32 ? T / 32 : 1;
    const int inst = blockIdx.y, tid = threadIdx.x;
    if (tid == 0) inst_state(ctl, inst, &s_run, &s_cur);
    __syncthreads();
    if (!s_run) return;
    const size_t nn = (size_t)(2 * L) * n2;
    const cpx<double>* src = reinterpret_cast<const cpx<double>*>((s_cur ? src1 : src0) + inst * nn);
    spec += inst * (nn / 2);
    const int RB = fix_seqs(L, R, true), lRB = 31 - __clz(RB), ld = fix_ld(L, RB);
    cfx* A = reinterpret_cast<cfx*>(smem_raw);
    cfx* B = A + fix_slots(L, RB) * ld;
    const int row = tid / T, j = tid & (T - 1);
    const bool on = row < RB;
    for (int r0 = 0; r0 < R; r0 += RB) {
        const int y0 = blockIdx.x * R + r0;
        cpx<double> x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
            x[u] = on ? src[(size_t)(y0 + row) * L + j + u * T] : mk(0.0, 0.0);
        const FixScale f = seq_scale<T>(mag_of(x), row, tid, s_stat, log2i(T));
        cfx v[8];
        int lost = 0;
        to_fixed<true>(x, v, f, &lost);
        if (row_partials) {
            long long s = 0;   // |components| <= 2^58: 16 of them fit
#pragma unroll
            for (int u = 0; u < 8; ++u) s += v[u].x + v[u].y;
            double d = (double)s + (double)lost * 0x1p-6;
#pragma unroll
            for (int o = (T < 32 ? T : 32) / 2; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
            if ((tid & 31) == 0) s_sum[tid >> 5] = d;
            if (T < 32 && on && j == 0) row_partials[(size_t)inst * n2 + y0 + row] = row_sum(d, f);
        }
        if (on && j == 0) s_scale[row] = f;
        fix_transform<L, -1>(v, j, row, A + row * ld, B + row * ld, pt1, f.need);
        // the last exchange read buffer A or B; the results go to the other one
        cfx* F = (FixPlan<L>::P & 1) ? A : B;
        if (on) {
#pragma unroll
            for (int u = 0; u < 8; ++u) F[row * ld + fix_pad(j + u * T)] = v[u];
        }
        __syncthreads();
        if (T >= 32 && row_partials && on && j == 0) {
            double d = 0.0;
#pragma unroll
            for (int w = 0; w < NW; ++w) d += s_sum[row * NW + w];
            row_partials[(size_t)inst * n2 + y0 + row] = row_sum(d, f);
        }
        // pairs (k, L - k) of each row, rows fastest: X(k), X(L - k) to the transposed spectrum
        for (int e = tid; e < RB * (L / 2); e += blockDim.x) {
            const int r = e & (RB - 1), k = e >> lRB;
            const cfx* Z = F + r * ld;
            const FixScale g = s_scale[r];
            const int sc = g.E - 1080 + g.need;
            cpx<double>* out = spec + y0 + r;
            int kc = L - k;
            cfx w[2];
            if (k == 0) {
                const cfx z0 = Z[0], zm = Z[fix_pad(L / 2)];
                cfx xc;
                w[0] = mkx(z0.x + z0.y, z0.x - z0.y);
                fix_r2c(zm, zm, tw1[L / 2], &w[1], &xc);
                kc = L / 2;
            } else {
                fix_r2c(Z[fix_pad(k)], Z[fix_pad(L - k)], tw1[k], &w[0], &w[1]);
            }
            cpx<double> o[2];
            from_fixed<2>(w, o, sc, g);
            out[(size_t)k * n2] = o[0];
            out[(size_t)kc * n2] = o[1];
        }
        if (r0 + RB < R) __syncthreads();
    }
}

// ------------------------------------------------------------------ column pass
// the exact sum of two doubles and its rounding error
__device__ __forceinline__ void sum_err(double a, double b, double& s, double& e) {
    s = a + b;
    const double t = s - a;
    e = (a - (s - t)) + (b - t);
}
// <U13> from the row sums and the loading state of this step (Sec. 5.1): eight sums per thread
// of the first T (compensated), then pairs of (sum, error) over the warp and the warps; an
// order fixed by n2 alone.  A chain of dependent FP64 operations: in a block of its own beside
// the columns', it is off the column pass's critical path (the stress enters each row's zero
// frequency in the inverse row kernel).
template <int T>
__device__ __forceinline__ void loading_block(const ColArgs<double>& a, int n1, int n2, int inst,
                                              double (*s_part)[16]) {
    const int tid = threadIdx.x;
    const double* parts = a.row_partials ? a.row_partials + (size_t)inst * a.nparts : nullptr;
    double s = 0.0, e = 0.0;
    if (parts && tid < T) {
        neumaier_start(s, e, parts[tid]);
#pragma unroll
        for (int u = 1; u < 8; ++u) neumaier_add(s, e, parts[tid + u * T]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        double t, f;
        sum_err(s, __shfl_xor_sync(0xffffffffu, s, o), t, f);
        e = (e + __shfl_xor_sync(0xffffffffu, e, o)) + f;
        s = t;
    }
    if ((tid & 31) == 0) { s_part[0][tid >> 5] = s; s_part[1][tid >> 5] = e; }
    __syncthreads();
    if (tid != 0) return;
    double tot = s_part[0][0], err = s_part[1][0];
    for (int w = 1; w < (T + 31) / 32; ++w) {
        double t, f;
        sum_err(tot, s_part[0][w], t, f);
        err += s_part[1][w] + f;
        tot = t;
    }
    fdm_dev_scalars* sci = a.sc + inst;
    const double mean = parts ? sci->phi_ref + (tot + err) * a.scl : sci->mean_up13;
    double eps, sig;
    loading_state(a.p, a.mu, a.frac, sci->step, sci->t, mean, &eps, &sig);
    sci->mean_up13 = mean;
    sci->eps_bar13 = eps;
    sci->sigma_bar13 = sig;
}

// grid (n1 / 2 / C (+ 1 for COL_K), instances); see col_pass_kernel.  The symbol acts on doubles between the
// two transforms: each thread's results of the forward one sit where the inverse one starts,
// so only the packed column kx = 0 exchanges values there.
template <int L>
__global__ void __launch_bounds__(FixBlock<L, false>::most, FixBlock<L, false>::minb)
    fix_col_kernel(const cpx<double>* in, cpx<double>* out, int n1, int C, const twx* __restrict__ pt2,
                   const double* __restrict__ Kh, ColArgs<double> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_run, s_cur;
    __shared__ WarpStat s_stat[2][16];
    __shared__ double s_part[2][16];
    constexpr int T = L / 8, n2 = L;
    const int inst = blockIdx.y, tid = threadIdx.x;
    if (tid == 0) {
        InstCtl ctl{a.mode == COL_K ? a.sc : nullptr, a.gated};
        inst_state(ctl, inst, &s_run, &s_cur);
    }
    __syncthreads();
    if (!s_run) return;
    if ((int)blockIdx.x * C == n1 / 2) {   // COL_K: one block more, for the loading
        loading_block<T>(a, n1, n2, inst, s_part);
        return;
    }
    const size_t half_n = (size_t)n1 * n2 / 2;
    in += inst * half_n;
    out += inst * half_n;
    const int CB = fix_seqs(L, C, false), ld = fix_ld(L, CB);
    cfx* A = reinterpret_cast<cfx*>(smem_raw);
    cfx* B = A + fix_slots(L, CB) * ld;
    const int c = tid / T, j = tid & (T - 1);
    const bool on = c < CB;
    const bool symbol = a.mode != COL_FWD && a.mode != COL_INV;
    for (int c0 = 0; c0 < C; c0 += CB) {
        const int kx = blockIdx.x * C + c0 + c;
        const bool packed_block = symbol && blockIdx.x == 0 && c0 == 0;   // holds the column kx = 0
        cpx<double> x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = on ? in[(size_t)kx * n2 + j + u * T] : mk(0.0, 0.0);
        FixScale f{};
        cfx v[8];
        int sc = 0;      // the doubles x stand for x 2^sc (kx > 0 between the transforms)
        if (a.mode != COL_INV) {
            f = seq_scale<T>(mag_of(x), c, tid, s_stat[0], log2i(T));
            to_fixed(x, v, f);
            fix_transform<L, -1>(v, j, c, A + c * ld, B + c * ld, pt2, f.need);
            sc = f.E - 1080 + f.need;
            // the power stays out of the symbol's products and joins the inverse transform's, where
            // the two together cannot leave FP64's range (8 FP64 products a thread)
            const bool apart = a.moderate && sc >= -500 && sc <= 700;
            if (!symbol || !apart || f.nan || f.pre || (packed_block && c == 0)) {
                from_fixed<8>(v, x, sc, f);
                sc = 0;
            } else {
#pragma unroll
                for (int u = 0; u < 8; ++u) x[u] = mk((double)v[u].x, (double)v[u].y);
            }
        }
        if (symbol) {
            if (packed_block) {   // exchange the packed column: z(ky) and z(-ky)
                cpx<double>* W = reinterpret_cast<cpx<double>*>((FixPlan<L>::P & 1) ? A : B);
                if (on && c == 0) {
#pragma unroll
                    for (int u = 0; u < 8; ++u) W[fix_pad(j + u * T)] = x[u];
                }
                __syncthreads();
                if (on && c == 0) {
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        // z = C0 + i CN: out(ky) = (m0 + mN)/2 z(ky) + (m0 - mN)/2 conj(z(-ky)),
                        // the symbols real (K, some stress components) or imaginary
                        const int ky = j + u * T;
                        const cpx<double> m0 = col_multiplier<double>(a, Kh, 0, ky, n1, n2);
                        const cpx<double> mN = col_multiplier<double>(a, Kh, n1 / 2, ky, n1, n2);
                        const cpx<double> z = x[u], zr = W[fix_pad((n2 - ky) & (n2 - 1))];
                        if (a.mode == COL_K || (a.mode == COL_SYM && !a.sym_imag)) {
                            const double p = 0.5 * (m0.x + mN.x), d = 0.5 * (m0.x - mN.x);
                            x[u] = mk(p * z.x + d * zr.x, p * z.y - d * zr.y);
                        } else {
                            const double p = 0.5 * (m0.y + mN.y), d = 0.5 * (m0.y - mN.y);
                            x[u] = mk(d * zr.y - p * z.y, p * z.x + d * zr.x);
                        }
                        // the macroscopic stress: see fix_row_inverse_kernel
                        if (ky == 0 && a.mode == COL_K) x[u].x = 0.0;
                    }
                }
                __syncthreads();
            }
            if (on && kx > 0) {
#pragma unroll
                for (int u = 0; u < 8; ++u) x[u] = col_apply<double>(a, Kh, kx, j + u * T, n1, n2, x[u]);
            }
        }
        if (a.mode != COL_FWD) {
            f = seq_scale<T>(mag_of(x), c, tid, s_stat[1], log2i(T));
            to_fixed(x, v, f);
            fix_transform<L, +1>(v, j, c, A + c * ld, B + c * ld, pt2, f.need);
            sc += f.E - 1080 + f.need;
            from_fixed<8>(v, x, sc, f);
        }
        if (on) {
#pragma unroll
            for (int u = 0; u < 8; ++u) out[(size_t)kx * n2 + j + u * T] = x[u];
        }
        if (c0 + CB < C) __syncthreads();
    }
}

// ------------------------------------------------------------------ row inverse (C2R)
// grid (n2 / R, instances); see row_inverse_kernel.
template <int L>
__global__ void __launch_bounds__(FixBlock<L, true>::most, FixBlock<L, true>::minb)
    fix_row_inverse_kernel(const cpx<double>* spec, double* dst, int n2, int R, const twx* __restrict__ tw1,
                           const twx* __restrict__ pt1, RowArgs<double> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_run, s_cur;
    __shared__ WarpStat s_stat[8][16];
    constexpr int T = L / 8;
    const int inst = blockIdx.y, tid = threadIdx.x;
    if (tid == 0) {
        InstCtl ctl{a.mode == ROW_TAU ? a.sc : nullptr, a.gated};
        inst_state(ctl, inst, &s_run, &s_cur);
    }
    __syncthreads();
    if (!s_run) return;
    const size_t nn = (size_t)(2 * L) * n2;
    spec += inst * (nn / 2);
    dst += inst * nn;
    fdm_dev_scalars* sci = (a.mode == ROW_TAU) ? a.sc + inst : nullptr;
    const int RB = fix_seqs(L, R, true), lRB = 31 - __clz(RB), ld = fix_ld(L, RB);
    cfx* A = reinterpret_cast<cfx*>(smem_raw);
    cfx* B = A + fix_slots(L, RB) * ld;
    const int row = tid / T, j = tid & (T - 1);
    const bool on = row < RB;
    const int lr = tid & (RB - 1), lk = tid >> lRB;   // the thread's row and first pair while loading
    const int NWB = (blockDim.x + 31) >> 5;
    unsigned long long vbits = 0ull;                  // max of |v0| as magnitude bits (a NaN wins)
    const double* up = s_cur ? (const double*)a.phi1 : (const double*)a.phi0;
    if (up) up += inst * nn;
    const double phi_ref = (sci && a.vel.friction) ? sci->phi_ref : 0.0;
    // without friction and mobility factors |v0| = |M tau| (rounded once, monotone in |tau|), or
    // the prescribed |v0|: the largest |tau| is enough
    const bool law = a.mode == ROW_TAU && (a.vel.friction || a.vel.mfac);
    VelLaw<double> plain = a.vel;
    plain.friction = 0;
    for (int r0 = 0; r0 < R; r0 += RB) {
        const int y0 = blockIdx.x * R + r0;
        // pairs (k, L - k), k = lk + i T < L / 2, of row lr; k = 0 takes the middle L / 2.  After
        // the layer kernel the macroscopic stress joins each row's zero frequency here
        cpx<double> x[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int k = lk + i * T;
            const cpx<double>* col = spec + y0 + lr;
            x[2 * i] = on ? col[(size_t)k * n2] : mk(0.0, 0.0);
            x[2 * i + 1] = on ? col[(size_t)(k == 0 ? L / 2 : L - k) * n2] : mk(0.0, 0.0);
        }
        if (a.add_sigma && lk == 0) x[0].x += a.sc[inst].sigma_bar13;
        const unsigned m = mag_of(x);
        // the row's scale: over the lanes of equal lr, then over the warps
        unsigned wm = m;
        for (int o = RB; o < 32; o <<= 1) wm = max(wm, __shfl_xor_sync(0xffffffffu, wm, o));
        unsigned ws = exp_unit((int)(wm >> 20), m);
        for (int o = RB; o < 32; o <<= 1) ws += __shfl_xor_sync(0xffffffffu, ws, o);
        if ((tid & 31) < RB) s_stat[tid & 31][tid >> 5] = WarpStat{wm, ws};
        __syncthreads();
        auto scale_row = [&](int r) {
            int E = 0;
            unsigned s = 0;
            for (int w = 0; w < NWB; ++w) E = max(E, (int)(s_stat[r][w].m >> 20));
            for (int w = 0; w < NWB; ++w) {
                const int d = E - (int)(s_stat[r][w].m >> 20);
                s += (d > 31 ? 0u : s_stat[r][w].s >> d) + 1u;
            }
            return fix_scale_of(E, s, log2i(T));
        };
        FixScale f = scale_row(lr);
        cfx v[8];
        to_fixed(x, v, f);
        if (on) {
            cfx* Z = A + lr * ld;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int k = lk + i * T;
                const cfx p = v[2 * i], q = v[2 * i + 1];
                cfx zk, zc;
                if (k == 0) {
                    Z[0] = mkx(fix_shr(p.x + p.y, 1), fix_shr(p.x - p.y, 1));
                    fix_c2r(q, q, tw1[L / 2], &zk, &zc);
                    Z[fix_pad(L / 2)] = zk;
                } else {
                    fix_c2r(p, q, tw1[k], &zk, &zc);
                    Z[fix_pad(k)] = zk;
                    Z[fix_pad(L - k)] = zc;
                }
            }
        }
        f = scale_row(on ? row : 0);
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = A[(on ? row : 0) * ld + fix_pad(j + u * T)];
        fix_transform<L, +1>(v, j, row, B + row * ld, A + row * ld, pt1, f.need);
        const int sc = f.E - 1080 + 1 + f.need;
        from_fixed<8>(v, x, sc, f);
        if (on) {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const size_t o = (size_t)(y0 + row) * (2 * L) + 2 * (j + u * T);
                cpx<double> t = x[u];
                if (a.mode != ROW_TAU) {
                    t = mk(t.x + a.offset, t.y + a.offset);
                } else if (!a.vel.friction) {
                    double c0 = t.x, c1 = t.y;
                    if (a.vel.mfac) {
                        const cpx<double> mf = *reinterpret_cast<const cpx<double>*>(a.vel.mfac + inst * nn + o);
                        c0 = celerity(plain, t.x, 0.0, 0.0) * mf.x;
                        c1 = celerity(plain, t.y, 0.0, 0.0) * mf.y;
                    }
                    vbits = max(vbits, max(ubits(c0) & kMagBits, ubits(c1) & kMagBits));
                }
                *reinterpret_cast<cpx<double>*>(dst + o) = t;
            }
            if (a.mode == ROW_TAU && a.vel.friction) {   // from what was stored, one body for all values
#pragma unroll 1
                for (int u = 0; u < 8; ++u) {
                    const size_t o = (size_t)(y0 + row) * (2 * L) + 2 * (j + u * T);
                    const cpx<double> t = *reinterpret_cast<const cpx<double>*>(dst + o);
                    const cpx<double> w = *reinterpret_cast<const cpx<double>*>(up + o);
                    double c0 = celerity(a.vel, t.x, w.x, phi_ref), c1 = celerity(a.vel, t.y, w.y, phi_ref);
                    if (a.vel.mfac) {
                        const cpx<double> mf = *reinterpret_cast<const cpx<double>*>(a.vel.mfac + inst * nn + o);
                        c0 = c0 * mf.x;
                        c1 = c1 * mf.y;
                    }
                    vbits = max(vbits, max(ubits(c0) & kMagBits, ubits(c1) & kMagBits));
                }
            }
        }
        if (r0 + RB < R) __syncthreads();
    }
    if (a.mode == ROW_TAU) {
        if (!law) vbits = ubits(celerity(a.vel, dbits(vbits), 0.0, 0.0)) & kMagBits;
        step_dt_from_max(vbits, sci, gridDim.x, a.cfl, a.dx, a.dt_max);
    }
}

// Runs BODY with the constant FL = L
#define FIX_SWITCH(L, BODY)                                  \
    switch (L) {                                             \
        case 8: { constexpr int FL = 8; BODY; break; }       \
        case 16: { constexpr int FL = 16; BODY; break; }     \
        case 32: { constexpr int FL = 32; BODY; break; }     \
        case 64: { constexpr int FL = 64; BODY; break; }     \
        case 128: { constexpr int FL = 128; BODY; break; }   \
        case 256: { constexpr int FL = 256; BODY; break; }   \
        case 512: { constexpr int FL = 512; BODY; break; }   \
        case 1024: { constexpr int FL = 1024; BODY; break; } \
        default: { constexpr int FL = 2048; BODY; break; }   \
    }
#define FIX_SWITCH_COL(L, BODY)                              \
    if ((L) == 4096) { constexpr int FL = 4096; BODY; }      \
    else FIX_SWITCH(L, BODY)

template <typename K> cudaError_t allow_smem(K* k, size_t bytes) {
    if (bytes <= 48 * 1024) return cudaSuccess;   // allowed as it is
    cudaError_t e = cudaFuncSetAttribute((const void*)k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute((const void*)k, cudaFuncAttributePreferredSharedMemoryCarveout,
                                cudaSharedmemCarveoutMaxShared);
}

}  // namespace

// loads the kernels of grids up to `side` x `side` onto the device (CUDA loads them lazily)
cudaError_t fix_preload(int side) {
    cudaError_t e = cudaSuccess;
    cudaFuncAttributes at;
    for (int L = 8; L <= side && e == cudaSuccess; L *= 2) {
        if (2 * L <= side)
            FIX_SWITCH(L, e = cudaFuncGetAttributes(&at, (const void*)fix_row_forward_kernel<FL>);
                       if (e == cudaSuccess) e = cudaFuncGetAttributes(&at, (const void*)fix_row_inverse_kernel<FL>));
        if (e == cudaSuccess && L >= 16)
            FIX_SWITCH_COL(L, e = cudaFuncGetAttributes(&at, (const void*)fix_col_kernel<FL>));
    }
    return e;
}
// shared-memory limits of the kernels of one grid
cudaError_t fix_configure(int n1, int n2) {
    const int L = n1 / 2;
    cudaError_t e = cudaSuccess;
    FIX_SWITCH(L, e = allow_smem(fix_row_forward_kernel<FL>, fix_max_smem(FL, true));
               if (e == cudaSuccess) e = allow_smem(fix_row_inverse_kernel<FL>, fix_max_smem(FL, true)));
    if (e != cudaSuccess) return e;
    FIX_SWITCH_COL(n2, e = allow_smem(fix_col_kernel<FL>, fix_max_smem(FL, false)));
    return e;
}

void fix_row_forward(const Dev& d, const double* src0, const double* src1, cpx<double>* spec, double* partials,
                     InstCtl ctl, int count, cudaStream_t s) {
    const LaunchGeom& g = d.geom;
    const int L = d.p.n1 / 2, rb = fix_seqs(L, g.R, true);
    const dim3 grid(g.row_blocks, count);
    FIX_SWITCH(L, (fix_row_forward_kernel<FL><<<grid, fix_threads(L, rb), fix_smem(L, rb), s>>>(
                      src0, src1, spec, d.p.n2, g.R, (const twx*)d.tw1, (const twx*)d.pt1, partials, ctl)));
}
void fix_col(const Dev& d, const cpx<double>* in, cpx<double>* out, const ColArgs<double>& a, int count,
             cudaStream_t s) {
    const LaunchGeom& g = d.geom;
    const int L = d.p.n2, cb = fix_seqs(L, g.C, false);
    const dim3 grid(g.col_blocks + (a.mode == COL_K ? 1 : 0), count);
    FIX_SWITCH_COL(L, (fix_col_kernel<FL><<<grid, fix_threads(L, cb), fix_smem(L, cb), s>>>(
                          in, out, d.p.n1, g.C, (const twx*)d.pt2, (const double*)d.Kh, a)));
}
void fix_row_inverse(const Dev& d, const cpx<double>* spec, double* dst, const RowArgs<double>& a, int count,
                     cudaStream_t s) {
    const LaunchGeom& g = d.geom;
    const int L = d.p.n1 / 2, rb = fix_seqs(L, g.R, true);
    const dim3 grid(g.row_blocks, count);
    FIX_SWITCH(L, (fix_row_inverse_kernel<FL><<<grid, fix_threads(L, rb), fix_smem(L, rb), s>>>(
                      spec, dst, d.p.n2, g.R, (const twx*)d.tw1, (const twx*)d.pt1, a)));
}

// the integer twiddle tables of an n-point twist and an L-point transform (launch_twiddle_tables)
__global__ void fix_tables_kernel(twx* __restrict__ tw, int n, twx* __restrict__ pt, int L) {
    const int len = pt ? pass_table_len(L) : 0;
    const int top = n > len ? n : len;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < top; i += gridDim.x * blockDim.x) {
        double sn, cs;
        if (tw && i < n) {
            sincospi(2.0 * (double)i / (double)n, &sn, &cs);
            tw[i] = fix_factor(cs, -sn, 2);
        }
        if (i < len) {
            int num, den;
            pass_table_entry(L, i, &num, &den);
            sincospi(2.0 * (double)num / (double)den, &sn, &cs);
            int Ns = 1, o = i;   // the radix of the entry's pass sets its scale
            while (o >= (pass_radix(L, Ns) - 1) * Ns) {
                const int r = pass_radix(L, Ns);
                o -= (r - 1) * Ns;
                Ns *= r;
            }
            pt[i] = fix_factor(cs, -sn, pass_radix(L, Ns) == 8 ? 3 : 2);
        }
    }
}
void fix_tables(void* tw, int n, void* pt, int L, cudaStream_t s) {
    fix_tables_kernel<<<8, 256, 0, s>>>((twx*)tw, n, (twx*)pt, L);
}

}  // namespace fdm
