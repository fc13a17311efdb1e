// fdm_f32.cu -- the mixed path's FP32 transform kernels: rows of U13 to the packed half spectrum,
// the column pass with its symbol, and rows back to tau13.  The same passes, products and sums as
// the generic kernels of fdm_kernels.cu, bit for bit (long coupled runs amplify any change of
// 32-bit rounding), in another arrangement: lengths are compile-time constants, a thread keeps
// eight values in registers, the first pass takes them from and the last leaves them for global
// memory, and shared memory, padded instead of swizzled, sees only the exchanges between passes
// and the transposition.
//
// What bounds them: latency, of global memory at the ends and of the barriers between passes, at
// 36 to 49 percent of the issue slots.  The arrangement's point is that an access or an index costs
// no arithmetic of its own: 7.9, 10.1 and 7.9 million warp instructions at 2048^2 (rows forward,
// columns, rows inverse) against 13.1, 21.3 and 14.5 of the generic kernels.  Measured at 2048^2
// (bytes read and written at the copy bandwidth: 5 us each): 24.4, 28.3, 29.7 us before, 25.6, 24.2,
// 22.5 now; at 4096^2 92, 108, 111 before, 70, 68, 76 now.
#include <type_traits>

#include "fdm_fix.cuh"
#include "fdm_step.cuh"

namespace fdm {
namespace {

using cf = cpx<float>;

template <int T> __device__ __forceinline__ void sync_seq(int id) {
    if constexpr (T >= 32) asm volatile("bar.sync %0, %1;" ::"r"(id + 1), "n"(T) : "memory");
    else __syncwarp();
}
__host__ __device__ __forceinline__ int f32_pad(int i) { return i + (i >> 4); }

// data pass through once, past the L1 cache, which the twiddles keep
__device__ __forceinline__ cf load_once(const cf* p) {
    const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
    return mk(v.x, v.y);
}

// threads of a block and sequences it works on at a time
template <int L> struct F32Block {
    static constexpr int T = L / 8;
    static constexpr int most = T >= 256 ? 512 : 256;
    static constexpr int minb = most == 512 ? 2 : 4;
};
__host__ __device__ constexpr int f32_seqs(int L, int R) {
    int rb = (L / 8 >= 256 ? 512 : 256) / (L / 8);
    if (rb > 8) rb = 8;
    return rb < R ? rb : R;
}
__host__ __device__ constexpr int f32_threads(int L, int rb) { return rb * (L / 8) < 32 ? 32 : rb * (L / 8); }
__host__ __device__ constexpr int f32_slots(int L, int rb) { return f32_threads(L, rb) / (L / 8); }
// stride of a sequence: padded, and such that the transposed accesses of rb sequences (a power of
// two) fall into different banks
__host__ __device__ constexpr int f32_ld(int L, int rb) {
    return (L + L / 16 + 15) / 16 * 16 + (rb > 1 ? 16 / rb : 0);
}
__host__ __device__ constexpr size_t f32_smem(int L, int rb) {
    return (size_t)2 * f32_slots(L, rb) * f32_ld(L, rb) * sizeof(cf);
}
constexpr size_t f32_max_smem(int L) {   // of any R
    size_t m = 0;
    for (int R = 1; R <= 16; R *= 2) {
        const size_t b = f32_smem(L, f32_seqs(L, R));
        if (b > m) m = b;
    }
    return m;
}

// pass p of direction S on the eight values of thread j (stockham_pass_pp's arithmetic)
template <int L, int p, int S> __device__ __forceinline__ void f32_pass(cf* v, int j, const cf* __restrict__ tab) {
    using Pl = FixPlan<L>;
    constexpr int R = Pl::radix(p), Ns = Pl::ns(p), PER = 8 / R;
#pragma unroll
    for (int b = 0; b < PER; ++b) {
        cf w[R];
#pragma unroll
        for (int r = 0; r < R; ++r) w[r] = v[b + r * PER];
        if (p > 0) {
            const int k = (j + b * Pl::T) & (Ns - 1);
#pragma unroll
            for (int r = 1; r < R; ++r) w[r] = cmul(w[r], twiddle<S>(tab + Pl::off(p), (r - 1) * Ns + k));
        }
        Dft<float, R>::template run<S>(w);
#pragma unroll
        for (int r = 0; r < R; ++r) v[b + r * PER] = w[r];
    }
}
// the transform of the eight values of thread j of sequence seq; A, B: its places in the buffers
template <int L, int S, int p = 0>
__device__ __forceinline__ void f32_transform(cf* v, int j, int seq, cf* A, cf* B, const cf* __restrict__ tab) {
    using Pl = FixPlan<L>;
    f32_pass<L, p, S>(v, j, tab);
    if constexpr (p + 1 < Pl::P) {
#pragma unroll
        for (int u = 0; u < 8; ++u) A[f32_pad(fix_place<L, p>(j, u))] = v[u];
        sync_seq<Pl::T>(seq);
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = A[f32_pad(j + u * Pl::T)];
        f32_transform<L, S, p + 1>(v, j, seq, B, A, tab);
    }
}

// ------------------------------------------------------------------ row forward (R2C)
template <int L>
__global__ void __launch_bounds__(F32Block<L>::most, F32Block<L>::most == 512 ? 2 : 5)
    f32_row_forward_kernel(const float* src0, const float* src1, cf* spec, int n2, int R, const cf* __restrict__ tw1,
                           const cf* __restrict__ pt1, double* row_partials, InstCtl ctl) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_run, s_cur;
    constexpr int T = L / 8;
    const int inst = blockIdx.y, tid = threadIdx.x;
    if (tid == 0) inst_state(ctl, inst, &s_run, &s_cur);
    __syncthreads();
    if (!s_run) return;
    const size_t nn = (size_t)(2 * L) * n2;
    const cf* src = reinterpret_cast<const cf*>((s_cur ? src1 : src0) + inst * nn);
    spec += inst * (nn / 2);
    const int RB = f32_seqs(L, R), lRB = 31 - __clz(RB), ld = f32_ld(L, RB);
    cf* A = reinterpret_cast<cf*>(smem_raw);
    cf* B = A + f32_slots(L, RB) * ld;
    const int row = tid / T, j = tid & (T - 1);
    const bool on = row < RB;
    for (int r0 = 0; r0 < R; r0 += RB) {
        const int y0 = blockIdx.x * R + r0;
        cf v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = on ? load_once(src + (size_t)(y0 + row) * L + j + u * T) : mk(0.0f, 0.0f);
        cf* X = A + row * ld;
        cf* Y = B + row * ld;
        if (row_partials) {
            // the row's values, for its sum; the transform's exchanges start in the other buffer
#pragma unroll
            for (int u = 0; u < 8; ++u) X[f32_pad(j + u * T)] = v[u];
            sync_seq<T>(row);
            // one warp of the row's own threads: lane l sums the pairs l, l + 32, ...
            // (compensated), then a fixed FP64 butterfly over the lanes
            const int lane = tid & 31;
            const int first = T >= 32 ? (j < 32 ? row : RB) : (tid >> 5) * (32 / (T < 32 ? T : 32));
            const int last = T >= 32 ? first + 1 : first + 32 / (T < 32 ? T : 32);
            for (int r = first; r < last && r < RB; ++r) {
                float acc = 0.0f, comp = 0.0f;
#pragma unroll 8
                for (int m = lane; m < L; m += 32) {
                    const cf z = A[r * ld + f32_pad(m)];
                    const float y = __fsub_rn(__fadd_rn(z.x, z.y), comp);
                    const float t = __fadd_rn(acc, y);
                    comp = __fsub_rn(__fsub_rn(t, acc), y);
                    acc = t;
                }
                const double rs = warp_sum((double)acc - (double)comp);
                if (lane == 0) row_partials[(size_t)inst * n2 + y0 + r] = rs;
            }
            cf* t = X; X = Y; Y = t;
        }
        f32_transform<L, -1>(v, j, row, X, Y, pt1);
        // the last exchange read X (P even) or Y; the results go to the other one
        cf* F = ((FixPlan<L>::P & 1) ? X : Y) - row * ld;
        if (on) {
#pragma unroll
            for (int u = 0; u < 8; ++u) F[row * ld + f32_pad(j + u * T)] = v[u];
        }
        __syncthreads();
        // pairs (k, L - k) of each row, rows fastest: X(k), X(L - k) to the transposed spectrum
        for (int e = tid; e < RB * (L / 2); e += blockDim.x) {
            const int r = e & (RB - 1), k = e >> lRB;
            const cf* Z = F + r * ld;
            cf* out = spec + y0 + r;
            if (k == 0) {
                const cf z0 = Z[0];
                out[0] = mk(z0.x + z0.y, z0.x - z0.y);
                const cf zm = Z[f32_pad(L / 2)];
                out[(size_t)(L / 2) * n2] = r2c_pair(zm, conj(zm), tw1[L / 2]).a;
            } else {
                const cpair<float> q = r2c_pair(Z[f32_pad(k)], conj(Z[f32_pad(L - k)]), tw1[k]);
                out[(size_t)k * n2] = q.a;
                out[(size_t)(L - k) * n2] = q.b;
            }
        }
        if (r0 + RB < R) __syncthreads();
    }
}

// ------------------------------------------------------------------ column pass
template <int L>
__global__ void __launch_bounds__(F32Block<L>::most, F32Block<L>::minb)
    f32_col_kernel(const cf* in, cf* out, int n1, int C, const cf* __restrict__ pt2, const float* __restrict__ Kh,
                   ColArgs<float> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_run, s_cur;
    __shared__ double s_sigma;
    __shared__ double s_red[kRedLanes];
    constexpr int T = L / 8, n2 = L;
    const int inst = blockIdx.y, tid = threadIdx.x;
    const size_t half_n = (size_t)n1 * n2 / 2;
    in += inst * half_n;
    out += inst * half_n;
    const int CB = f32_seqs(L, C), ld = f32_ld(L, CB);
    cf* A = reinterpret_cast<cf*>(smem_raw);
    cf* B = A + f32_slots(L, CB) * ld;
    const int c = tid / T, j = tid & (T - 1);
    const bool on = c < CB;
    cf v[8];
    auto load = [&](int kx) {
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = on ? load_once(in + (size_t)kx * n2 + j + u * T) : mk(0.0f, 0.0f);
    };
    load(blockIdx.x * C + c);   // on its way while thread 0 reads the instance's state
    if (tid == 0) {
        InstCtl ctl{a.mode == COL_K ? a.sc : nullptr, a.gated};
        inst_state(ctl, inst, &s_run, &s_cur);
    }
    __syncthreads();
    if (!s_run) return;
    const bool symbol = a.mode != COL_FWD && a.mode != COL_INV;
    for (int c0 = 0; c0 < C; c0 += CB) {
        const int kx = blockIdx.x * C + c0 + c;
        const bool packed_block = symbol && blockIdx.x == 0 && c0 == 0;   // holds the column kx = 0
        if (c0 > 0) load(kx);
        if (packed_block && a.mode == COL_K) loading_from_rows(a, n1, n2, inst, s_red, &s_sigma);
        cf* X = A + c * ld;
        cf* Y = B + c * ld;
        if (a.mode != COL_INV) f32_transform<L, -1>(v, j, c, X, Y, pt2);
        if (symbol) {
            if (packed_block) {   // exchange the packed column: z(ky) and z(-ky)
                cf* W = (FixPlan<L>::P & 1) ? A : B;   // the last exchange read the other buffer
                if (on && c == 0) {
#pragma unroll
                    for (int u = 0; u < 8; ++u) W[f32_pad(j + u * T)] = v[u];
                }
                __syncthreads();
                if (on && c == 0) {
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int ky = j + u * T;
                        v[u] = packed_symbol(a, Kh, ky, n1, n2, v[u], W[f32_pad((n2 - ky) & (n2 - 1))]);
                        if (ky == 0 && a.mode == COL_K) v[u].x = (float)s_sigma;   // macroscopic stress
                    }
                }
                __syncthreads();
            }
            if (on && kx > 0) {
                const bool real = a.mode == COL_K || (a.mode == COL_SYM && !a.sym_imag);
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    // rounded products: the next pass's sums must not take them in unrounded
                    const cf m = col_multiplier<float>(a, Kh, kx, j + u * T, n1, n2);
                    v[u] = real ? mk(__fmul_rn(m.x, v[u].x), __fmul_rn(m.x, v[u].y))
                                : mk(-__fmul_rn(m.y, v[u].y), __fmul_rn(m.y, v[u].x));
                }
            }
        }
        if (a.mode != COL_FWD) {
            // the forward exchanges end with a read of Y (P even: X); the inverse ones start with
            // a write to X, behind one more meeting of the sequence's threads
            if (a.mode != COL_INV) sync_seq<T>(c);
            f32_transform<L, +1>(v, j, c, X, Y, pt2);
        }
        if (on) {
#pragma unroll
            for (int u = 0; u < 8; ++u) out[(size_t)kx * n2 + j + u * T] = v[u];
        }
        if (c0 + CB < C) __syncthreads();
    }
}

// ------------------------------------------------------------------ row inverse (C2R)
template <int L>
__global__ void __launch_bounds__(F32Block<L>::most, F32Block<L>::minb)
    f32_row_inverse_kernel(const cf* spec, float* dst, int n2, int R, const cf* __restrict__ tw1,
                           const cf* __restrict__ pt1, RowArgs<float> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_run, s_cur;
    constexpr int T = L / 8;
    const int inst = blockIdx.y, tid = threadIdx.x;
    const size_t nn = (size_t)(2 * L) * n2;
    spec += inst * (nn / 2);
    dst += inst * nn;
    fdm_dev_scalars* sci = (a.mode == ROW_TAU) ? a.sc + inst : nullptr;
    const int RB = f32_seqs(L, R), lRB = 31 - __clz(RB), ld = f32_ld(L, RB);
    cf* A = reinterpret_cast<cf*>(smem_raw);
    cf* B = A + f32_slots(L, RB) * ld;
    const int row = tid / T, j = tid & (T - 1);
    const bool on = row < RB;
    const int lr = tid & (RB - 1), lk = tid >> lRB;   // the thread's row and first pair while loading
    // pairs (k, L - k), k = lk + i T < L / 2, of row lr; k = 0 takes the middle L / 2
    cf x[8];
    auto load = [&](int y0) {
        const cf* col = spec + y0 + lr;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int k = lk + i * T;
            x[2 * i] = on ? load_once(col + (size_t)k * n2) : mk(0.0f, 0.0f);
            x[2 * i + 1] = on ? load_once(col + (size_t)(k == 0 ? L / 2 : L - k) * n2) : mk(0.0f, 0.0f);
        }
    };
    load(blockIdx.x * R);   // on its way while thread 0 reads the instance's state
    if (tid == 0) {
        InstCtl ctl{a.mode == ROW_TAU ? a.sc : nullptr, a.gated};
        inst_state(ctl, inst, &s_run, &s_cur);
    }
    __syncthreads();
    if (!s_run) return;
    float vmax = 0.0f;
    bool bad = false;
    const float* up = s_cur ? (const float*)a.phi1 : (const float*)a.phi0;
    if (up) up += inst * nn;
    const double phi_ref = (sci && a.vel.friction) ? sci->phi_ref : 0.0;
    const bool law = a.vel.friction || a.vel.mfac;
    VelLaw<float> plain = a.vel;   // without friction: no FP64 instruction per node
    plain.friction = 0;
    for (int r0 = 0; r0 < R; r0 += RB) {
        const int y0 = blockIdx.x * R + r0;
        if (r0 > 0) load(y0);
        if (on) {
            cf* Z = A + lr * ld;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int k = lk + i * T;
                if (k == 0) {
                    Z[0] = mk(x[2 * i].x + x[2 * i].y, x[2 * i].x - x[2 * i].y);
                    Z[f32_pad(L / 2)] = c2r_pair(x[2 * i + 1], conj(x[2 * i + 1]), conj(tw1[L / 2])).a;
                } else {
                    const cpair<float> q = c2r_pair(x[2 * i], conj(x[2 * i + 1]), conj(tw1[k]));
                    Z[f32_pad(k)] = q.a;
                    Z[f32_pad(L - k)] = q.b;
                }
            }
        }
        __syncthreads();
        cf v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = A[(on ? row : 0) * ld + f32_pad(j + u * T)];
        f32_transform<L, +1>(v, j, row, B + row * ld, A + row * ld, pt1);
        if (on) {
            float* o = dst + (size_t)(y0 + row) * (2 * L) + 2 * j;
            if (a.mode != ROW_TAU) {
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = mk(v[u].x + a.offset, v[u].y + a.offset);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) *reinterpret_cast<cf*>(o + 2 * u * T) = v[u];
            if (a.mode == ROW_TAU && !law) {
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const float c0 = celerity(plain, v[u].x, 0.0f, 0.0), c1 = celerity(plain, v[u].y, 0.0f, 0.0);
                    vmax = tmax(vmax, tmax(tabs(c0), tabs(c1)));
                    bad |= (c0 != c0) || (c1 != c1);
                }
            } else if (a.mode == ROW_TAU) {   // friction or mobility factors: from what was stored
#pragma unroll 1
                for (int u = 0; u < 8; ++u) {
                    const size_t at = (size_t)(y0 + row) * (2 * L) + 2 * (j + u * T);
                    const cf t = *reinterpret_cast<const cf*>(dst + at);
                    cf w = mk(0.0f, 0.0f);
                    if (a.vel.friction) w = *reinterpret_cast<const cf*>(up + at);
                    float c0 = celerity(a.vel, t.x, w.x, phi_ref), c1 = celerity(a.vel, t.y, w.y, phi_ref);
                    if (a.vel.mfac) {
                        const cf mf = *reinterpret_cast<const cf*>(a.vel.mfac + inst * nn + at);
                        c0 = c0 * mf.x;
                        c1 = c1 * mf.y;
                    }
                    vmax = tmax(vmax, tmax(tabs(c0), tabs(c1)));
                    bad |= (c0 != c0) || (c1 != c1);
                }
            }
        }
        if (r0 + RB < R) __syncthreads();
    }
    if (a.mode == ROW_TAU)
        step_dt_from_max(bad ? 0x7ff8000000000000ull : abs_bits((double)vmax), sci, gridDim.x, a.cfl, a.dx, a.dt_max);
}

#define F32_SWITCH(L, BODY)                                  \
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
#define F32_SWITCH_COL(L, BODY)                              \
    if ((L) == 4096) { constexpr int FL = 4096; BODY; }      \
    else F32_SWITCH(L, BODY)

template <typename K> cudaError_t allow_smem(K* k, size_t bytes) {
    if (bytes > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute((const void*)k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e != cudaSuccess) return e;
    }
    // shared memory for the blocks that registers let live on an SM; the rest is cache for the
    // twiddles, which every pass reads.  4096^2, all three kernels: 264 us with all of it shared,
    // 221 with 80 percent, 215 with 60, 299 with 40 (too few blocks); 2048^2: 78, 72, 73, 85.
    return cudaFuncSetAttribute((const void*)k, cudaFuncAttributePreferredSharedMemoryCarveout, 60);
}

}  // namespace

// shared-memory limits of the kernels of one grid
cudaError_t f32_configure(int n1, int n2) {
    const int L = n1 / 2;
    cudaError_t e = cudaSuccess;
    F32_SWITCH(L, e = allow_smem(f32_row_forward_kernel<FL>, f32_max_smem(FL));
               if (e == cudaSuccess) e = allow_smem(f32_row_inverse_kernel<FL>, f32_max_smem(FL)));
    if (e != cudaSuccess) return e;
    F32_SWITCH_COL(n2, e = allow_smem(f32_col_kernel<FL>, f32_max_smem(FL)));
    return e;
}
void f32_row_forward(const Dev& d, const float* src0, const float* src1, cf* spec, double* partials, InstCtl ctl,
                     int count, cudaStream_t s) {
    const LaunchGeom& g = d.geom;
    const int L = d.p.n1 / 2, rb = f32_seqs(L, g.R);
    const dim3 grid(g.row_blocks, count);
    F32_SWITCH(L, (f32_row_forward_kernel<FL><<<grid, f32_threads(L, rb), f32_smem(L, rb), s>>>(
                      src0, src1, spec, d.p.n2, g.R, (const cf*)d.tw1, (const cf*)d.pt1, partials, ctl)));
}
void f32_col(const Dev& d, const cf* in, cf* out, const ColArgs<float>& a, int count, cudaStream_t s) {
    const LaunchGeom& g = d.geom;
    const int L = d.p.n2, cb = f32_seqs(L, g.C);
    const dim3 grid(g.col_blocks, count);
    F32_SWITCH_COL(L, (f32_col_kernel<FL><<<grid, f32_threads(L, cb), f32_smem(L, cb), s>>>(
                          in, out, d.p.n1, g.C, (const cf*)d.pt2, (const float*)d.Kh, a)));
}
void f32_row_inverse(const Dev& d, const cf* spec, float* dst, const RowArgs<float>& a, int count, cudaStream_t s) {
    const LaunchGeom& g = d.geom;
    const int L = d.p.n1 / 2, rb = f32_seqs(L, g.R);
    const dim3 grid(g.row_blocks, count);
    F32_SWITCH(L, (f32_row_inverse_kernel<FL><<<grid, f32_threads(L, rb), f32_smem(L, rb), s>>>(
                      spec, dst, d.p.n2, g.R, (const cf*)d.tw1, (const cf*)d.pt1, a)));
}

}  // namespace fdm
