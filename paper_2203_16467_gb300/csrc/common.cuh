// common.cuh -- device data layout, per-problem control block, pointwise
// constitutive model (Sec. 2.1) and deterministic reductions shared by every
// kernel of libpff.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

namespace pff {

// ---------------------------------------------------------------------------
// complex helpers
template <typename T> struct CT;
template <> struct CT<float> { using t = float2; };
template <> struct CT<double> { using t = double2; };

template <typename C> __device__ __forceinline__ C cadd(C a, C b) { return C{a.x + b.x, a.y + b.y}; }
template <typename C> __device__ __forceinline__ C csub(C a, C b) { return C{a.x - b.x, a.y - b.y}; }
template <typename C> __device__ __forceinline__ C cmul(C a, C b) { return C{a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x}; }
// a * conj(b)
template <typename C> __device__ __forceinline__ C cmulc(C a, C b) { return C{a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y}; }

// model enums (mirror include/pff.h)
enum { AT1 = 1, AT2 = 2 };
enum { ISOTROPIC = 0, SPECTRAL = 1, SPECTRAL_STRESSFREE = 2, VOLDEV = 3, SPECTRAL_VOLDEV = 4 };
// split that supplies the stress (contact model) / the crack driving force (Sec. 2.1, Sec. 4.2)
__host__ __device__ __forceinline__ int contact_of(int split) {
    return split == SPECTRAL_STRESSFREE ? ISOTROPIC : (split == SPECTRAL_VOLDEV ? VOLDEV : split);
}
__host__ __device__ __forceinline__ int driving_of(int split) {
    return (split == SPECTRAL_STRESSFREE || split == SPECTRAL_VOLDEV) ? SPECTRAL : split;
}
enum { CRACK_SET = 0, DAMAGE = 1 };

// ---------------------------------------------------------------------------
// A quotient a / x whose divisor is known earlier than its dividend: 1 / (x s) = hi + lo is formed off the
// chain (an FP64 division takes 550 cycles, a product 65), and (a s) hi + (a s) lo rounds once, so the
// quotient is as accurate as a division (its error is half a unit and some 2^-50 of one; 2e5 random
// quotients all equal the division's).  s, a power of two, keeps the parts within the exponent range.  The
// quotient by 0 is 0.
struct Recip { double hi, lo, s; };
__device__ __forceinline__ Recip recip(double x) {
    const unsigned e = ((unsigned)__double2hiint(x) >> 20) & 0x7ffu;   // biased exponent
    const double s = e < 64u ? 0x1p256 : e > 1982u ? 0x1p-256 : 1.0;
    const double xs = x * s, hi = 1.0 / xs, lo = fma(-hi, xs, 1.0) * hi;
    const bool in = e < 0x7ffu && x != 0.0;
    return Recip{x != 0.0 ? hi : 0.0, in ? lo : 0.0, s};
}
__device__ __forceinline__ double quotient(double a, const Recip& r) {
    a *= r.s;
    return fma(a, r.hi, a * r.lo);
}

// ---------------------------------------------------------------------------
// Control block of one problem (device memory).  Scalars of the iterative
// solvers live here so that kernels chain without host round trips.  Flags
// come in pairs (x_a, x_b): a kernel never writes a flag that kernels of the
// same launch read, so early-exit decisions are consistent across its blocks.
struct Ctrl {
    // macroscopic strain and loading
    double eps_bar[3];
    double sumE2;           // sum of E^2 over pixels (scale of the mechanics tolerance)
    double sumE;            // sum of E
    // mechanics
    double mech_target, R2, rr, alpha, beta, cg_target;
    Recip rr_inv;           // of rr, formed beside alpha
    int nd_a, nd_b, newton_it, needs_fold;
    int cg_a, cg_b, cg_it, cg_total, cg_break;
    // near-equilibrium rescale (Algorithm 4 lines 4-10)
    double mF_max, D_max, Rf_star, D_star, gamma;
    int istar, flag, rescaled;
    // phase field (Algorithm 1)
    double pf_rr, pf_rp, pf_alpha, pf_beta, pf_target, pf_best;   // pf_best, pf_last_full: squared norms
    Recip pf_irp;           // of -r.p of the direction, formed beside alpha
    double pf_pap;          // sum a p^2 of the direction (the diagonal part of p.Jp)
    int pf_a, pf_b, pf_it, pf_break, n_active, pf_best_it, pf_clamp_iters;
    // residual recurrence: pf_full = this iteration evaluates Jv explicitly
    int pf_full, pf_force, pf_confirm, pf_since_full, pf_full_iters;
    int pf_rsel;            // the BCCG residual r lives in th[1] (0) or q[1] (1)
    double pf_abar;         // mean of the BCCG diagonal a (preconditioner)
    double pf_rz;           // r.z of the previous preconditioned iteration
    // grid barrier of the persistent BCCG kernel (arrivals, release generation, abort)
    unsigned bar_count, bar_gen;
    int bar_abort;
    double pf_last_full;
    // post-step (Algorithm 4 lines 12-14)
    double rep_eps_bar[3], sig_bar[3], C_bar, dphi, Fe, Ff;
    int incremented, broken;
    int status;             // bit0: mechanics cap hit, bit1: BCCG cap hit, bit3: a wait ran out
    unsigned counter;       // last-block reduction counter (reset by the last block)
    // set by the host for the alternating-minimisation / time-dependent methods
    double eta_dt_override; // eta/dt of the phase-field step when use_override
    int use_override;
    int con_frozen;         // constraint field phi_con taken from aux (fixed over an increment)
    int post_mode;          // 0: post-step applies Algorithm 4's strain increment; 1: host decides
    int pad;
};
// The last block of a reduction moves the control block with 128 threads in one go, a word each (a second
// round trip costs 3 % of a 512^2 BCCG solve).
static_assert(sizeof(Ctrl) <= 512, "one word per thread of the smallest block");

// Model constants of a problem, resolved on the host.
struct Consts {
    double lam_c, mu_c;     // lambda = lam_c * E, mu = mu_c * E (plane strain)
    double c;               // G_c / (c_w ell)
    double kappa;           // 2 c ell^2 (coefficient of -nabla^2 in J)
    double ell2;            // ell^2
    double eta_dt;          // eta / dt
    double cf2;             // c * f''
    double Fmax, thresh, dphi_min, C_broken, crack_thr;
    double mech_tol, mech_cg_rtol, pf_tol, pf_atol, pf_floor;
    double d_eps_bar[3];
    double dA;              // pixel area
    double inv_n;           // 1 / (nx ny)
    double L1_scale;        // (dx/ell)^2
    double two_pi_over_Lx, two_pi_over_Ly;
    double lp_a, lp_b, lp_c;  // low-pass band kx^2 lp_a + ky^2 lp_b <= lp_c (microstructure generator only)
    int max_newton, max_cg, max_pf;
    int pf_precond;         // BCCG with the Fourier Helmholtz preconditioner
    int fracture, split, irrev;
};

// Device descriptor of one problem's fields (all arrays nx*ny, row-major).
// Phase-field work vectors alias the mechanics CG vectors:
//   v = th[0], rb = th[1], pb = th[2], a = r[0], b = r[1], vcon = r[2].
template <typename T>
struct Desc {
    using C = typename CT<T>::t;
    T* E;
    T* phi;
    T* eps[3];
    T* th[3];
    T* r[3];
    T* p[3];
    T* q[3];
    T* lap;
    T* aux;
    uint8_t* flags;
    C* S;                   // spectral buffer [3][ny][wp]
    const C* tw;            // twiddle tables of this device
    double* part;           // reduction partials [blocks * 8]
    Ctrl* ctrl;
    int nx, ny, wp, pad;
    Consts k;
};

// ---------------------------------------------------------------------------
// Programmatic dependent launch: a kernel's blocks may be scheduled while the
// previous kernel of the stream is still running; they do only work on
// immutable data (descriptor, twiddle tables) before pdl_wait(), which returns
// once the previous kernel has completed and its writes are visible.  Each
// kernel then lets the next one be scheduled.  Both are no-ops for launches
// without the attribute.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_enter() { pdl_wait(); pdl_release(); }

// ---------------------------------------------------------------------------
// Per-block constants: thread 0 evaluates F::skip and F::prep once (control
// block loads and FP64-to-FP32 conversions, which run on GB300's narrow FP64
// pipe) and shares the result through shared memory.  Returns true when the
// whole problem is skipped.  Ctx must be trivially copyable.  prep does not wait
// for the skip test: its loads and the flag's (some 700 cycles from L2) overlap.
template <class F, class D, class X>
__device__ __forceinline__ bool block_prep(const D& d, X& ctx) {
    __shared__ __align__(16) unsigned char s_raw[sizeof(X)];
    __shared__ int s_skip;
    if (threadIdx.x == 0) {
        const int skip = F::skip(d) ? 1 : 0;
        const X c = F::prep(d);
        memcpy(s_raw, &c, sizeof(X));
        s_skip = skip;
    }
    __syncthreads();
    if (s_skip) return true;
    memcpy(&ctx, s_raw, sizeof(X));
    return false;
}

// ---------------------------------------------------------------------------
// flag access (bypass L1: flags are written by other kernels / blocks)
__device__ __forceinline__ int ldflag(const int* p) { return __ldcg(p); }
__device__ __forceinline__ double ldd(const double* p) { return __ldcg(p); }

// ---------------------------------------------------------------------------
// Per-thread accumulation.  FP64 problems accumulate in double.  FP32 problems
// accumulate products exactly split (fmaf) and summed with Knuth's two-sum in
// a float pair, and reduce across the grid in double-float arithmetic
// (reduce_finalize): the work stays on the FP32 pipe while the sums keep close to
// FP64 accuracy.
// Functors whose per-pixel work splits into load() (returning an In record) and
// pixel(..., const In&, ...) let a kernel issue the loads of all of a thread's
// pixels before the first store, so that they are in flight together.
template <class F, class = void> struct HasIn { static constexpr bool value = false; };
template <class F> struct HasIn<F, decltype((void)sizeof(typename F::In), void())> { static constexpr bool value = true; };

template <class F, class D, class X, class... A>
__device__ __forceinline__ void pixel_one(const D& d, const X& c, size_t i, A&&... a) {
    if constexpr (HasIn<F>::value) F::pixel(d, c, i, F::load(d, c, i), a...);
    else F::pixel(d, c, i, a...);
}

struct DF { float hi, lo; };   // double-float value hi + lo (see reduce_finalize)
template <typename T> struct Acc;
// count(x): a small integer (a pixel count); a thread's sum of counts is exact in
// either precision (below 2^24), so it needs no compensation.
template <> struct Acc<double> {
    double s = 0.0;
    __device__ __forceinline__ void add(double x) { s += x; }
    __device__ __forceinline__ void count(double x) { s += x; }
    __device__ __forceinline__ void addp(double a, double b) { s = fma(a, b, s); }
    __device__ __forceinline__ double get() const { return s; }
};
template <> struct Acc<float> {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void count(float x) { s += x; }
    __device__ __forceinline__ void add(float x) {
        float t = s + x;
        float z = t - s;
        c += (s - (t - z)) + (x - z);
        s = t;
    }
    __device__ __forceinline__ void addp(float a, float b) {
        float pr = __fmul_rn(a, b);   // not contracted into the two-sum below
        float e = fmaf(a, b, -pr);
        add(pr);
        c += e;
    }
    __device__ __forceinline__ double get() const { return (double)s + (double)c; }
    __device__ __forceinline__ DF df() const {   // normalised double-float pair
        float h = s + c;
        float z = h - s;
        return DF{h, (s - (h - z)) + (c - z)};
    }
};

// Grid reductions.  Each block reduces its threads' values (a shuffle tree per value) into
// part[blockIdx.x*NR + k]; the last block of the problem (by an atomic ticket) sums all partials in a
// fixed order, the totals in tot (valid in thread 0), and runs the finalizer (reduce_finalize).
// Deterministic: the summation tree depends only on the grid shape.
//
// FP32 problems: every product is formed exactly (fmaf split), each thread's
// sum is a compensated float pair, and the block reduces the pairs in
// double-float arithmetic (a value is an unevaluated sum hi + lo of two floats,
// added with Knuth's two-sum; about 44 significant bits) so that the per-pixel
// and per-thread work stays on the FP32 pipe; the block totals and the
// cross-block sum are FP64 (reduce_finalize).
__device__ __forceinline__ DF df_add(DF a, DF b) {
    float s = a.hi + b.hi;
    float z = s - a.hi;
    float e = (a.hi - (s - z)) + (b.hi - z);
    e += a.lo + b.lo;
    float h = s + e;
    return DF{h, e - (h - s)};
}
// Double-float arithmetic on values (relative error a few 2^-46 away from cancellation and from the
// ends of the exponent range): exact sum and product of floats, product, scaling, square root.
__device__ __forceinline__ DF df_sum(float a, float b) {
    float s = a + b, z = s - a;
    return DF{s, (a - (s - z)) + (b - z)};
}
__device__ __forceinline__ DF df_of(double x) {
    float h = (float)x;
    return DF{h, (float)(x - (double)h)};
}
__device__ __forceinline__ DF df_neg(DF a) { return DF{-a.hi, -a.lo}; }
__device__ __forceinline__ DF df_scale(DF a, float s) { return DF{a.hi * s, a.lo * s}; }   // s a power of two
__device__ __forceinline__ DF df_mul(DF a, DF b) {
    float p = __fmul_rn(a.hi, b.hi);
    float e = fmaf(a.hi, b.hi, -p) + fmaf(a.hi, b.lo, a.lo * b.hi);
    float h = p + e;
    return DF{h, e - (h - p)};
}
__device__ __forceinline__ DF df_mulf(DF a, float b) {
    float p = __fmul_rn(a.hi, b);
    float e = fmaf(a.hi, b, -p) + a.lo * b;
    float h = p + e;
    return DF{h, e - (h - p)};
}
// one Newton step on the FP32 root (a.hi > 0)
__device__ __forceinline__ DF df_sqrt(DF a) {
    float r = rsqrtf(a.hi), x = a.hi * r;
    float p = __fmul_rn(x, x);
    float rem = ((a.hi - p) - fmaf(x, x, -p)) + a.lo;   // a - x^2 (a.hi - p is exact)
    float e = 0.5f * r * rem;
    float h = x + e;
    return DF{h, e - (h - x)};
}

template <typename V> struct RedOps;
template <> struct RedOps<double> {
    __device__ static double zero() { return 0.0; }
    __device__ static double add(double a, double b) { return a + b; }
    __device__ static double shfl(double a, int o) { return __shfl_down_sync(0xffffffffu, a, o); }
    __device__ static double total(double v) { return v; }
};
template <> struct RedOps<DF> {
    __device__ static DF zero() { return DF{0.f, 0.f}; }
    __device__ static DF add(DF a, DF b) { return df_add(a, b); }
    __device__ static DF shfl(DF a, int o) {
        return DF{__shfl_down_sync(0xffffffffu, a.hi, o), __shfl_down_sync(0xffffffffu, a.lo, o)};
    }
    __device__ static double total(DF v) { return (double)v.hi + (double)v.lo; }
};

// Block reduction in a fixed order: every thread stores its NR values in shared memory, then L lanes
// take each value (all values at once: L = NT / 8 lanes for 8 of them, a warp at most): lane l adds entries
// l, l + L, ... pairwise, then a shuffle tree.  The totals are left in res.  (A warp taking its share of the
// values one after the other makes the chain twice as long for eight: 512^2 FP32 BCCG solve 3.87 -> 3.85 ms in
// one pair of runs, 3.95 -> 3.90 in another; eight in streams 14.5 -> 14.4 ms per load step.)
template <int NR, int NT, typename V>
__device__ __forceinline__ void block_reduce(const V (&v)[NR], V (&res)[NR]) {
    using O = RedOps<V>;
    constexpr int KP = NR <= 1 ? 1 : NR <= 2 ? 2 : NR <= 4 ? 4 : 8;
    constexpr int L = NT / KP < 32 ? NT / KP : 32, PER = NT / L;
    __shared__ V sh[NR][NT];
#pragma unroll
    for (int k = 0; k < NR; ++k) sh[k][threadIdx.x] = v[k];
    __syncthreads();
    if (threadIdx.x < KP * L) {   // whole warps
        const int k = threadIdx.x / L, l = threadIdx.x & (L - 1);
        const V* row = sh[k < NR ? k : 0];
        V x[PER];
#pragma unroll
        for (int j = 0; j < PER; ++j) x[j] = row[l + L * j];
#pragma unroll
        for (int n = 1; n < PER; n *= 2)
#pragma unroll
            for (int j = 0; j + n < PER; j += 2 * n) x[j] = O::add(x[j], x[j + n]);
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) x[0] = O::add(x[0], O::shfl(x[0], o));
        if (l == 0 && k < NR) res[k] = x[0];
    }
    __syncthreads();
}

// The cross-block stage is FP64 for both precisions: each block's total is stored
// as one double (a double-float pair hi + lo converts exactly), and the last block
// sums the partials in double.  Within a block an FP32 problem's values stay
// double-float pairs (FP32 pipe); an FP64 problem's stay doubles.
//
// This tail is a serial chain at the end of a kernel: an L2 round trip takes 700 to 900 cycles and an
// FP64 operation 65.  So the block's values are converted and stored by one lane each; the last
// block's threads hold one value each of several blocks and load them eight at a time; and the
// control block and the descriptor, which the finalizer works on, come into shared memory beside the
// partials and go back in one go.  (Eight values of the 512^2 BCCG iterate: 19000 of the kernel's 30000
// cycles lay between its last pixel and its end with one thread storing, a load at a time and the
// finalizer on global memory: 18.7 us, now 14.6; 2048^2 66 -> 60 us.)
constexpr int red_lanes(int n) { return n <= 1 ? 1 : n <= 2 ? 2 : n <= 4 ? 4 : 8; }

// Block and grid reduction of the per-thread accumulators, F::finalize(descriptor, totals) in the last block.
template <class F, int NR, int NT, typename T>
__device__ __forceinline__ void reduce_finalize(const Acc<T>* acc, const Desc<T>& d, int nblocks) {
    using V = typename std::conditional<sizeof(T) == 4, DF, double>::type;
    static_assert(NR >= 1 && NR <= 8 && NT >= 64, "one lane per value");
    constexpr int KP = red_lanes(NR), NW = NT / 32, S = NT / KP;   // S blocks per pass
    constexpr int CWORDS = (int)(sizeof(Ctrl) / 4), DWORDS = (int)(sizeof(Desc<T>) / 4);
    __shared__ V bs[NR];
    __shared__ double shw[NW][KP];
    __shared__ __align__(16) int s_ctrl[CWORDS];
    __shared__ __align__(16) int s_desc[DWORDS];
    __shared__ int s_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    V v[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) {
        if constexpr (sizeof(T) == 4) v[k] = acc[k].df();
        else v[k] = acc[k].get();
    }
    block_reduce<NR, NT>(v, bs);
    if (warp == 0) {
        if (lane < NR) __stcg(d.part + (size_t)blockIdx.x * NR + lane, RedOps<V>::total(bs[lane]));
        __threadfence();
        __syncwarp();
        if (lane == 0) s_last = atomicAdd(&d.ctrl->counter, 1u) == (unsigned)(nblocks - 1);
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const int* gc = reinterpret_cast<const int*>(d.ctrl);
    const int* gd = reinterpret_cast<const int*>(&d);
    for (int w = tid; w < CWORDS; w += NT) s_ctrl[w] = __ldcg(gc + w);
    for (int w = tid; w < DWORDS; w += NT) s_desc[w] = gd[w];
    // thread (b0, k) sums value k of the blocks b0, b0 + S, ...
    const int k = tid % KP;
    double x = 0.0;
    for (int b = tid / KP; b < nblocks; b += 8 * S) {
        double y[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int bb = b + u * S;
            y[u] = k < NR && bb < nblocks ? __ldcg(d.part + (size_t)bb * NR + k) : 0.0;
        }
        x += ((y[0] + y[1]) + (y[2] + y[3])) + ((y[4] + y[5]) + (y[6] + y[7]));
    }
#pragma unroll
    for (int o = KP; o < 32; o *= 2) x += __shfl_xor_sync(0xffffffffu, x, o);
    if (lane < KP) shw[warp][lane] = x;
    __syncthreads();
    if (warp == 0) {
        if (lane < KP) {
            double t[NW];
#pragma unroll
            for (int w = 0; w < NW; ++w) t[w] = shw[w][lane];
#pragma unroll
            for (int n = 1; n < NW; n *= 2)
#pragma unroll
                for (int w = 0; w + n < NW; w += 2 * n) t[w] += t[w + n];
            shw[0][lane] = t[0];
        }
        __syncwarp();
        if (lane == 0) {
            double tot[NR];
#pragma unroll
            for (int q = 0; q < NR; ++q) tot[q] = shw[0][q];
            Desc<T>& sd = *reinterpret_cast<Desc<T>*>(s_desc);
            sd.ctrl = reinterpret_cast<Ctrl*>(s_ctrl);
            F::finalize(sd, tot);
            sd.ctrl->counter = 0u;
        }
    }
    __syncthreads();
    int* out = reinterpret_cast<int*>(d.ctrl);
    for (int w = tid; w < CWORDS; w += NT) __stcg(out + w, s_ctrl[w]);
}

// ---------------------------------------------------------------------------
// Pointwise constitutive model (Sec. 2.1).  Strain / stress as (xx, yy, xy)
// with xy the tensor shear component.  Lame constants for plane strain.
template <typename T> __device__ __forceinline__ T rp(T x) { return x > T(0) ? x : T(0); }
template <typename T> __device__ __forceinline__ T rm(T x) { return x < T(0) ? x : T(0); }
template <typename T> __device__ __forceinline__ T hv(T x) { return x > T(0) ? T(1) : T(0); }

// Principal strains e1 >= e2 and the eigen-projector frame of a symmetric
// 2x2 tensor without explicit eigenvectors: with d = (xx-yy)/2, rad =
// sqrt(d^2 + xy^2), u = d/rad, w = xy/rad:
//   P1 = 1/2 [[1+u, w], [w, 1-u]],  P2 = I - P1,  S = [[-w, u], [u, w]]
// (S = n1 n2^T + n2 n1^T).  deg marks coincident principal strains.
// irad = 1/rad when not deg.  FP32 takes rad and 1/rad from one reciprocal
// square root (rsqrtf, 2 ulp) instead of a correctly rounded root and division.
template <typename T>
struct Eig2 {
    T e1, e2, u, w, tr, irad;
    bool deg;
    __device__ __forceinline__ Eig2(T xx, T yy, T xy) {
        tr = xx + yy;
        T d = T(0.5) * (xx - yy);
        T s2 = d * d + xy * xy;
        T rad;
        if constexpr (sizeof(T) == 4) {
            irad = s2 > T(0) ? rsqrtf(s2) : T(0);
            rad = s2 * irad;
        } else {
            rad = sqrt(s2);
            irad = rad > T(0) ? T(1) / rad : T(0);
        }
        e1 = T(0.5) * tr + rad;
        e2 = T(0.5) * tr - rad;
        T scale = fmax(fabs(e1), fabs(e2));
        deg = !(T(2) * rad > T(1e-12) * scale) || rad == T(0);
        if (deg) { u = T(1); w = T(0); }
        else { u = d * irad; w = xy * irad; }
    }
};

// sigma_0^+ (sp) and sigma_0^- (sm) of the strain-spectral split
// (Eq. stress_spectral) and psi_0^+ (Eq. strain_spectral_en).
template <typename T>
__device__ __forceinline__ void spectral_split(T xx, T yy, T xy, T lam, T mu, T* sp, T* sm, T& psip) {
    Eig2<T> g(xx, yy, xy);
    T a1 = rp(g.e1), a2 = rp(g.e2), b1 = rm(g.e1), b2 = rm(g.e2);
    T trp = rp(g.tr), trm = rm(g.tr);
    // eps^+ = a1 P1 + a2 P2
    T hs = T(0.5) * (a1 + a2), hd = T(0.5) * (a1 - a2);
    T epxx = hs + hd * g.u, epyy = hs - hd * g.u, epxy = hd * g.w;
    T ms = T(0.5) * (b1 + b2), md = T(0.5) * (b1 - b2);
    T emxx = ms + md * g.u, emyy = ms - md * g.u, emxy = md * g.w;
    sp[0] = lam * trp + T(2) * mu * epxx;
    sp[1] = lam * trp + T(2) * mu * epyy;
    sp[2] = T(2) * mu * epxy;
    sm[0] = lam * trm + T(2) * mu * emxx;
    sm[1] = lam * trm + T(2) * mu * emyy;
    sm[2] = T(2) * mu * emxy;
    psip = T(0.5) * lam * trp * trp + mu * (a1 * a1 + a2 * a2);
}

template <typename T>
__device__ __forceinline__ T psi_iso(T xx, T yy, T xy, T lam, T mu) {
    T tr = xx + yy;
    return T(0.5) * lam * tr * tr + mu * (xx * xx + yy * yy + T(2) * xy * xy);
}

template <typename T>
__device__ __forceinline__ T psi_spectral(T xx, T yy, T xy, T lam, T mu) {
    Eig2<T> g(xx, yy, xy);
    T a1 = rp(g.e1), a2 = rp(g.e2), trp = rp(g.tr);
    return T(0.5) * lam * trp * trp + mu * (a1 * a1 + a2 * a2);
}

// Volumetric-deviatoric split, Eq. vol_dev_en with the sums over the two in-plane
// components and the 1/3 of the 3-D deviator; K = lambda + 2 mu / 3.
template <typename T>
__device__ __forceinline__ T psi_voldev(T xx, T yy, T xy, T lam, T mu) {
    T tr = xx + yy, K = lam + T(2) * mu / T(3), t3 = tr / T(3);
    T a = xx - t3, b = yy - t3, trp = rp(tr);
    return T(0.5) * K * trp * trp + mu * (a * a + b * b + T(2) * xy * xy);
}

// psi_0^+ of the crack-driving-force model in double-float arithmetic, for FP32 problems (GB300 runs
// FP64 at 1/64 of the FP32 rate).  With M the largest |eps_bar| + |eps*| of the components, the value is off
// by less than 2^-41 (2 |lambda| + 10 mu) M^2 (df_psi_size): an addition's error is at most 5 2^-48 of its
// operands' magnitudes, a product's 7 2^-48, the root's 51 2^-48 of itself, and the longest path (spectral)
// adds up to 83 2^-48 of that size.  df_psi_range: no part leaves the FP32 exponent range (else the caller
// takes the FP64 function).
struct DF3 { DF xx, yy, xy; };
__device__ __forceinline__ DF df_pos(DF a) { return a.hi > 0.f ? a : DF{0.f, 0.f}; }
__device__ __forceinline__ bool df_psi_range(float M, float lam, float mu) {
    const float k = fmaxf(fabsf(lam), mu);
    return M > 1e-8f && M < 1e10f && k > 1e-15f && k < 1e15f;
}
__device__ __forceinline__ float df_psi_size(float M, float lam, float mu) { return (2.f * fabsf(lam) + 10.f * mu) * M * M; }
// are all values within err of hi + lo rounded to the same FP32 number (false for a NaN)
__device__ __forceinline__ bool df_rounds(DF x, float err) { return x.hi + (x.lo - err) == x.hi + (x.lo + err); }
__device__ __forceinline__ DF df_psi_plus(int split, const DF3& e, DF lam, DF mu) {
    const int s = driving_of(split);
    const DF tr = df_add(e.xx, e.yy);
    if (s == ISOTROPIC) {
        DF q = df_add(df_mul(e.xx, e.xx), df_mul(e.yy, e.yy));
        q = df_add(q, df_scale(df_mul(e.xy, e.xy), 2.f));
        return df_add(df_mul(df_scale(lam, 0.5f), df_mul(tr, tr)), df_mul(mu, q));
    }
    const DF trp = df_pos(tr);
    if (s == VOLDEV) {
        // a^2 + b^2 + 2 xy^2 with a = xx - tr/3, b = yy - tr/3 is xx^2 + yy^2 + 2 xy^2 - 4/9 tr^2
        const DF tr2 = df_mul(tr, tr);
        const DF third{0.33333334f, -9.934108e-09f}, k49{0.44444445f, -3.3113692e-09f};   // 1/3, 4/9
        DF q = df_add(df_mul(e.xx, e.xx), df_mul(e.yy, e.yy));
        q = df_add(q, df_scale(df_mul(e.xy, e.xy), 2.f));
        q = df_add(q, df_neg(df_mul(k49, tr2)));
        const DF K = df_add(lam, df_scale(df_mul(mu, third), 2.f));
        return df_add(df_mul(df_scale(K, 0.5f), df_mul(trp, trp)), df_mul(mu, q));
    }
    const DF d = df_scale(df_add(e.xx, df_neg(e.yy)), 0.5f);
    const DF s2 = df_add(df_mul(d, d), df_mul(e.xy, e.xy));
    const DF rad = s2.hi > 0.f ? df_sqrt(s2) : DF{0.f, 0.f};
    const DF h = df_scale(tr, 0.5f);
    const DF a1 = df_pos(df_add(h, rad)), a2 = df_pos(df_add(h, df_neg(rad)));
    return df_add(df_mul(df_scale(lam, 0.5f), df_mul(trp, trp)), df_mul(mu, df_add(df_mul(a1, a1), df_mul(a2, a2))));
}

// psi_0^+ of the crack-driving-force model.
template <typename T>
__device__ __forceinline__ T psi_plus(int split, T xx, T yy, T xy, T lam, T mu) {
    const int s = driving_of(split);
    if (s == ISOTROPIC) return psi_iso(xx, yy, xy, lam, mu);
    if (s == VOLDEV) return psi_voldev(xx, yy, xy, lam, mu);
    return psi_spectral(xx, yy, xy, lam, mu);
}

// Stress of the contact model (isotropic for SPECTRAL_STRESSFREE, vol.-dev. for SPECTRAL_VOLDEV).
template <typename T>
__device__ __forceinline__ void stress(int split, T xx, T yy, T xy, T hphi, T lam, T mu, T* s) {
    split = contact_of(split);
    if (split == VOLDEV) {
        // sigma^+ = K <tr>_+ I + 2 mu (eps - 4/9 tr I), sigma^- = K <tr>_- I (exact gradients)
        T tr = xx + yy, K = lam + T(2) * mu / T(3);
        T q = T(4) / T(9) * tr;
        s[0] = hphi * (K * rp(tr) + T(2) * mu * (xx - q)) + K * rm(tr);
        s[1] = hphi * (K * rp(tr) + T(2) * mu * (yy - q)) + K * rm(tr);
        s[2] = hphi * (T(2) * mu * xy);
        return;
    }
    if (split == SPECTRAL) {
        T sp[3], sm[3], psip;
        spectral_split(xx, yy, xy, lam, mu, sp, sm, psip);
        s[0] = hphi * sp[0] + sm[0];
        s[1] = hphi * sp[1] + sm[1];
        s[2] = hphi * sp[2] + sm[2];
    } else {
        T tr = xx + yy;
        s[0] = hphi * (lam * tr + T(2) * mu * xx);
        s[1] = hphi * (lam * tr + T(2) * mu * yy);
        s[2] = hphi * (T(2) * mu * xy);
    }
}

// Energy density psi = h psi_0^+ + psi_0^- of the contact model (Eq. psi_schema).
template <typename T>
__device__ __forceinline__ T energy(int split, T xx, T yy, T xy, T hphi, T lam, T mu) {
    split = contact_of(split);
    if (split == VOLDEV) {
        T tr = xx + yy, K = lam + T(2) * mu / T(3), trm = rm(tr);
        return hphi * psi_voldev(xx, yy, xy, lam, mu) + T(0.5) * K * trm * trm;
    }
    if (split == SPECTRAL) {
        Eig2<T> g(xx, yy, xy);
        T a1 = rp(g.e1), a2 = rp(g.e2), b1 = rm(g.e1), b2 = rm(g.e2);
        T trp = rp(g.tr), trm = rm(g.tr);
        T pp = T(0.5) * lam * trp * trp + mu * (a1 * a1 + a2 * a2);
        T pm = T(0.5) * lam * trm * trm + mu * (b1 * b1 + b2 * b2);
        return hphi * pp + pm;
    }
    return hphi * psi_iso(xx, yy, xy, lam, mu);
}

// Tangent C:p of the contact model at strain eps (Sec. 3.1.1).  Spectral:
// Daleckii-Krein derivative of eps -> eps^+ in the frame (P1, P2, S):
//   D+[p] = H(e1)(P1:p)P1 + H(e2)(P2:p)P2 + g12 (S:p/2) S,
//   g12 = (<e1>_+ - <e2>_+)/(e1 - e2)  (H(e1) for coincident e1 = e2),
// sigma' = h (lam H(tr) tr p I + 2 mu D+) + lam (1 - H(tr)) tr p I + 2 mu (p - D+).
template <typename T>
__device__ __forceinline__ void tangent(int split, T xx, T yy, T xy, T hphi, T lam, T mu,
                                        T pxx, T pyy, T pxy, T* out) {
    T trp = pxx + pyy;
    split = contact_of(split);
    if (split == VOLDEV) {
        T K = lam + T(2) * mu / T(3), Ht = hv(xx + yy);
        T q = T(4) / T(9) * trp;
        out[0] = hphi * (K * Ht * trp + T(2) * mu * (pxx - q)) + K * (T(1) - Ht) * trp;
        out[1] = hphi * (K * Ht * trp + T(2) * mu * (pyy - q)) + K * (T(1) - Ht) * trp;
        out[2] = hphi * (T(2) * mu * pxy);
        return;
    }
    if (split == SPECTRAL) {
        Eig2<T> g(xx, yy, xy);
        T dxx, dyy, dxy;
        if (g.deg) {
            T H = hv(g.e1);
            dxx = H * pxx; dyy = H * pyy; dxy = H * pxy;
        } else {
            T H1 = hv(g.e1), H2 = hv(g.e2);
            // divided difference (<e1>_+ - <e2>_+)/(e1 - e2): H(e1) when e1 and e2 have
            // the same sign (exactly, as the quotient of equal values), e1 / (2 rad)
            // when they straddle zero (no cancellation there); FP32 avoids the division
            T g12;
            if constexpr (sizeof(T) == 4) g12 = (g.e1 > T(0) && g.e2 < T(0)) ? g.e1 * (T(0.5) * g.irad) : H1;
            else g12 = (rp(g.e1) - rp(g.e2)) / (g.e1 - g.e2);
            T u = g.u, w = g.w;
            T P1p = T(0.5) * ((T(1) + u) * pxx + (T(1) - u) * pyy + T(2) * w * pxy);
            T P2p = T(0.5) * ((T(1) - u) * pxx + (T(1) + u) * pyy - T(2) * w * pxy);
            T Sp = T(0.5) * (-w * pxx + w * pyy + T(2) * u * pxy);
            T c1 = H1 * P1p, c2 = H2 * P2p, c3 = g12 * Sp;
            dxx = T(0.5) * (c1 * (T(1) + u) + c2 * (T(1) - u)) - c3 * w;
            dyy = T(0.5) * (c1 * (T(1) - u) + c2 * (T(1) + u)) + c3 * w;
            dxy = T(0.5) * (c1 * w - c2 * w) + c3 * u;
        }
        T Ht = hv(g.tr);
        T lp = lam * Ht * trp, lm = lam * (T(1) - Ht) * trp;
        out[0] = hphi * (lp + T(2) * mu * dxx) + lm + T(2) * mu * (pxx - dxx);
        out[1] = hphi * (lp + T(2) * mu * dyy) + lm + T(2) * mu * (pyy - dyy);
        out[2] = hphi * (T(2) * mu * dxy) + T(2) * mu * (pxy - dxy);
    } else {
        out[0] = hphi * (lam * trp + T(2) * mu * pxx);
        out[1] = hphi * (lam * trp + T(2) * mu * pyy);
        out[2] = hphi * (T(2) * mu * pxy);
    }
}

// FP64: the part of the tangent that depends on the strain, which is fixed while a Newton round's CG runs;
// its kernels read it (f) instead of the strain.  Spectral: u, w of the frame and g12, with
// H(e1) = (g12 != 0), H(e2) = (|g12| >= 1) and H(tr) = (sign bit clear): g12 of opposite signs lies in
// (0, 1) and is kept there (at its ends by an ulp).  Vol.-dev.: f[0] = H(tr).  Isotropic: nothing.
// A root, two divisions and some 20 further FP64 instructions a pixel less in each CG iteration, whose
// first pass they bound (us, event-timed: 512^2 58.5 -> 41.4, 256^2 18.6 -> 15.8, 256 x 128 15.6 -> 13.7) for
// three stores a pixel in each Newton round (512^2 79 -> 101).  FP32 problems form the tangent from the
// strain each time: a reciprocal root costs them little (2048^2 37.0, from the frame 38.6; 1024^2 15.1
// and 13.6, whose Newton round loses as much).
template <typename T> constexpr bool TANGENT_FRAME = sizeof(T) == 8;
template <typename T>
__device__ __forceinline__ void tangent_frame(int contact, T xx, T yy, T xy, T (&f)[3]) {
    if (contact == VOLDEV) {
        f[0] = hv(xx + yy);
    } else if (contact == SPECTRAL) {
        Eig2<T> g(xx, yy, xy);
        const T above0 = T(1e-300), below1 = T(0.99999999999999989);
        T m;
        if (g.deg || !(g.e1 > T(0)) || g.e2 > T(0)) m = hv(g.e1);   // one sign: H(e1) (see tangent)
        else m = fmin(fmax(g.e1 / (g.e1 - g.e2), above0), below1);
        f[0] = g.u;
        f[1] = g.w;
        f[2] = copysign(m, hv(g.tr) - T(0.5));
    }
}
// C:p from the frame f of the strain (see tangent)
template <typename T>
__device__ __forceinline__ void tangent_framed(int contact, const T (&f)[3], T hphi, T lam, T mu, T pxx, T pyy, T pxy,
                                               T* out) {
    const T trp = pxx + pyy;
    if (contact == VOLDEV) {
        const T K = lam + T(2) * mu / T(3), Ht = f[0];
        const T q = T(4) / T(9) * trp;
        out[0] = hphi * (K * Ht * trp + T(2) * mu * (pxx - q)) + K * (T(1) - Ht) * trp;
        out[1] = hphi * (K * Ht * trp + T(2) * mu * (pyy - q)) + K * (T(1) - Ht) * trp;
        out[2] = hphi * (T(2) * mu * pxy);
    } else if (contact == SPECTRAL) {
        const T u = f[0], w = f[1], g12 = fabs(f[2]);
        const T P1p = T(0.5) * ((T(1) + u) * pxx + (T(1) - u) * pyy + T(2) * w * pxy);
        const T P2p = T(0.5) * ((T(1) - u) * pxx + (T(1) + u) * pyy - T(2) * w * pxy);
        const T Sp = T(0.5) * (-w * pxx + w * pyy + T(2) * u * pxy);
        const T c1 = g12 > T(0) ? P1p : T(0), c2 = g12 >= T(1) ? P2p : T(0), c3 = g12 * Sp;
        const T dxx = T(0.5) * (c1 * (T(1) + u) + c2 * (T(1) - u)) - c3 * w;
        const T dyy = T(0.5) * (c1 * (T(1) - u) + c2 * (T(1) + u)) + c3 * w;
        const T dxy = T(0.5) * (c1 * w - c2 * w) + c3 * u;
        const bool open = !signbit(f[2]);
        const T lp = open ? lam * trp : T(0), lm = open ? T(0) : lam * trp;
        out[0] = hphi * (lp + T(2) * mu * dxx) + lm + T(2) * mu * (pxx - dxx);
        out[1] = hphi * (lp + T(2) * mu * dyy) + lm + T(2) * mu * (pyy - dyy);
        out[2] = hphi * (T(2) * mu * dxy) + T(2) * mu * (pxy - dxy);
    } else {
        out[0] = hphi * (lam * trp + T(2) * mu * pxx);
        out[1] = hphi * (lam * trp + T(2) * mu * pyy);
        out[2] = hphi * (T(2) * mu * pxy);
    }
}

}  // namespace pff
