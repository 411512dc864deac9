// fft.cuh -- shared-memory batched FFTs and the three kernel shapes of a
// 2-D spectral operator F^-1 M F (Sec. 3.1: the DFT pair; the normalisation
// 1/(nx ny) is folded into the mode multiplier M):
//   k_row_fwd : per-pixel prologue -> real FFT along x  -> half spectrum S
//   k_col     : FFT along y -> mode multiplier (Gamma, -|2 pi q|^2 or the band
//               limit) -> inverse FFT along y (k_col512: register radix-8 stages
//               for 512-point FP32 columns)
//   k_row_inv : half spectrum -> real inverse FFT along x -> per-pixel epilogue (+ reductions)
// The kernels' bodies are per-item device functions (a row group, a column
// group) that the persistent solve shares.  FFTs are radix-8 Stockham passes
// (one radix-2 or radix-4 pass first when log2 of the length is not a multiple
// of 3), register staged and in place in shared memory with padded indices,
// with twiddles from FP64-accurate tables.
#pragma once
#include "common.cuh"

namespace pff {

// Twiddle tables (per device, built on the host in FP64): the table of
// length M sits at offset M and holds exp(-2 pi i j / M), j < M.
constexpr int TW_MAX = 4096;                 // longest transform

constexpr int ilog2(int n) { return n <= 1 ? 0 : 1 + ilog2(n / 2); }
constexpr int pow2floor(int n) { return n <= 1 ? 1 : 2 * pow2floor(n / 2); }
constexpr int cmin(int a, int b) { return a < b ? a : b; }
constexpr int cmax(int a, int b) { return a > b ? a : b; }

// Padded index of element e of a sequence in shared memory: one empty slot per
// 16 elements.  With this padding every read and write pattern of the mixed
// radix-8/4/2 Stockham passes below touches each 8-byte slot column at most
// twice per warp (the minimum for 8-byte elements).
__device__ __forceinline__ int pidx(int e) { return e + (e >> 4); }
constexpr int padded_len(int M) { return M + M / 16; }

template <typename C, bool INV>
__device__ __forceinline__ void dft4(C& a0, C& a1, C& a2, C& a3) {
    C s02 = cadd(a0, a2), d02 = csub(a0, a2), s13 = cadd(a1, a3), d13 = csub(a1, a3);
    // forward: multiply d13 by -i; inverse: by +i
    C t = INV ? C{-d13.y, d13.x} : C{d13.y, -d13.x};
    a0 = cadd(s02, s13);
    a2 = csub(s02, s13);
    a1 = cadd(d02, t);
    a3 = csub(d02, t);
}

// 8-point DFT in registers: two 4-point DFTs of the even and odd samples and
// the twiddles W8^k (W8 = exp(-+ 2 pi i / 8)).
template <typename C, bool INV>
__device__ __forceinline__ void dft8(C (&u)[8]) {
    using T = decltype(u[0].x);
    const T h = T(0.70710678118654752440);
    C e0 = u[0], e1 = u[2], e2 = u[4], e3 = u[6];
    C o0 = u[1], o1 = u[3], o2 = u[5], o3 = u[7];
    dft4<C, INV>(e0, e1, e2, e3);
    dft4<C, INV>(o0, o1, o2, o3);
    C t1, t2, t3;
    if (!INV) {
        t1 = C{h * (o1.x + o1.y), h * (o1.y - o1.x)};
        t2 = C{o2.y, -o2.x};
        t3 = C{h * (o3.y - o3.x), -h * (o3.x + o3.y)};
    } else {
        t1 = C{h * (o1.x - o1.y), h * (o1.x + o1.y)};
        t2 = C{-o2.y, o2.x};
        t3 = C{-h * (o3.x + o3.y), h * (o3.x - o3.y)};
    }
    u[0] = cadd(e0, o0); u[4] = csub(e0, o0);
    u[1] = cadd(e1, t1); u[5] = csub(e1, t1);
    u[2] = cadd(e2, t2); u[6] = csub(e2, t2);
    u[3] = cadd(e3, t3); u[7] = csub(e3, t3);
}

// One Stockham pass of radix R over sequences [s0, s0+G) of length M stored at
// buf[s*SP + pidx(j)]; p = product of the radices of the previous passes.
//   butterfly i in [0, M/R): k = i mod p; inputs x[i + r M/R]; twiddle
//   w^(r k) with w = exp(-+2 pi i/(p R)); outputs y[(i - k) R + k + r p].
// Twiddles: w^k, w^2k (and w^4k for radix 8) from the table, the rest as products (FP32).
// TWP: the twiddle table is stored with padded indices (pidx), as when staged in
// shared memory, so that the strided reads of a warp spread over the banks.
template <typename T, int M, int R, int G, int NSEQ, int SP, int NT, bool INV, bool TWP = false>
__device__ __forceinline__ void stockham_pass(typename CT<T>::t* buf, int s0, int p, const typename CT<T>::t* tw, int tid) {
    using C = typename CT<T>::t;
    constexpr int NBS = M / R;           // butterflies per sequence
    constexpr int NB = G * NBS;          // butterflies in the round
    constexpr int PER = (NB + NT - 1) / NT;
    // FP64: all twiddles from the table (16 of a radix-8 butterfly's 100 FP64 instructions formed the
    // products; that pipe bounds its passes)
    constexpr bool TABLE = sizeof(T) == 8;
    C u[PER][8];
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        int b = tid + j * NT;
        int s = s0 + b / NBS, i = b % NBS;
        if ((NB % NT == 0 || b < NB) && s < NSEQ) {
#pragma unroll
            for (int r = 0; r < R; ++r) u[j][r] = buf[s * SP + pidx(i + r * NBS)];
        }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        int b = tid + j * NT;
        int s = s0 + b / NBS, i = b % NBS;
        if ((NB % NT == 0 || b < NB) && s < NSEQ) {
            const int k = i & (p - 1);
            if (p > 1) {
                const int idx = k * (M / (p * R));
                C w1 = tw[TWP ? pidx(idx) : idx];
                if (INV) w1.y = -w1.y;
                if (R == 2) {
                    u[j][1] = cmul(u[j][1], w1);
                } else {
                    C w2 = tw[TWP ? pidx(2 * idx) : 2 * idx];
                    if (INV) w2.y = -w2.y;
                    C w3;
                    if constexpr (TABLE) {
                        w3 = tw[TWP ? pidx(3 * idx) : 3 * idx];
                        if (INV) w3.y = -w3.y;
                    } else {
                        w3 = cmul(w1, w2);
                    }
                    u[j][1] = cmul(u[j][1], w1);
                    u[j][2] = cmul(u[j][2], w2);
                    u[j][3] = cmul(u[j][3], w3);
                    if (R == 8) {
                        C w4 = tw[TWP ? pidx(4 * idx) : 4 * idx];
                        if (INV) w4.y = -w4.y;
                        u[j][4] = cmul(u[j][4], w4);
                        if constexpr (TABLE) {
#pragma unroll
                            for (int r = 5; r < 8; ++r) {
                                C w = tw[TWP ? pidx(r * idx) : r * idx];
                                if (INV) w.y = -w.y;
                                u[j][r] = cmul(u[j][r], w);
                            }
                        } else {
                            u[j][5] = cmul(u[j][5], cmul(w1, w4));
                            u[j][6] = cmul(u[j][6], cmul(w2, w4));
                            u[j][7] = cmul(u[j][7], cmul(w3, w4));
                        }
                    }
                }
            }
            if (R == 8) {
                dft8<C, INV>(u[j]);
            } else if (R == 4) {
                dft4<C, INV>(u[j][0], u[j][1], u[j][2], u[j][3]);
            } else {
                C a = u[j][0], c = u[j][1];
                u[j][0] = cadd(a, c);
                u[j][1] = csub(a, c);
            }
            const int o = (i - k) * R + k;
#pragma unroll
            for (int r = 0; r < R; ++r) buf[s * SP + pidx(o + r * p)] = u[j][r];
        }
    }
    __syncthreads();
}

// NSEQ in-place complex FFTs of length M (unnormalised; forward e^-, inverse e^+),
// radix-8 passes after one radix-2 or radix-4 pass when log2 M is not a multiple
// of 3.  Sequences are processed in rounds of G; each thread holds at most PER8
// radix-8 butterflies of a round in registers.
template <typename T, int M, int NSEQ, int SP, int NT, bool INV, bool TWP = false>
__device__ __forceinline__ void fft_smem(typename CT<T>::t* buf, const typename CT<T>::t* tw, int tid = threadIdx.x) {
    constexpr int LOG = ilog2(M);
    constexpr int PER8 = sizeof(T) == 4 ? 2 : 1;
    constexpr int G = cmax(1, cmin(NSEQ, (8 * NT * PER8) / M));   // sequences per round
    for (int s0 = 0; s0 < NSEQ; s0 += G) {
        int p = 1;
        if (LOG % 3 == 1) {
            stockham_pass<T, M, 2, G, NSEQ, SP, NT, INV, TWP>(buf, s0, 1, tw, tid);
            p = 2;
        } else if (LOG % 3 == 2) {
            stockham_pass<T, M, 4, G, NSEQ, SP, NT, INV, TWP>(buf, s0, 1, tw, tid);
            p = 4;
        }
        for (; p < M; p *= 8) stockham_pass<T, M, 8, G, NSEQ, SP, NT, INV, TWP>(buf, s0, p, tw, tid);
    }
}

// cp.async: asynchronous global -> shared copies (no register staging)
// (PFF_L2_ONLY: translation units whose kernels read data written by other blocks of
// the same launch copy 8-byte elements with L2-only loads instead: cp.async.ca
// would go through L1, which is not coherent between SMs within a kernel.)
template <int BYTES>
__device__ __forceinline__ void cp_async(void* smem, const void* gmem) {
#ifdef PFF_L2_ONLY
    if constexpr (BYTES == 8) {
        *reinterpret_cast<unsigned long long*>(smem) = __ldcg(reinterpret_cast<const unsigned long long*>(gmem));
        return;
    }
#endif
    unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(sa), "l"(gmem), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

// ---------------------------------------------------------------------------
// launch geometry
// Passes of up to 512 points ask for their half spectra beside the skip test (a skipped launch reads them
// for nothing): the flag's load and the spectrum's, some 800 cycles each, then overlap.  Solves, ms, after -> beside:
// phase field 512^2 FP32 3.90 -> 3.79, 256^2 FP64 5.09 -> 5.01; mechanics 256 x 128 FP64 1.87 -> 1.84; eight 512^2
// problems in streams 14.25 -> 13.94 a load step.  Not FP32 with three components (512^2 mechanics 2.42 -> 2.48).
template <typename T, int N, int NC> constexpr bool EARLY_SPECTRUM = N <= 512 && (NC == 1 || sizeof(T) == 8);

template <typename T, int NX, int NC>
struct RowCfg {
    static constexpr int M = NX / 2;
    static constexpr bool F32 = sizeof(T) == 4;
    // rows per block: about 512 complex values per block so that a 512^2 grid
    // already gives 128+ blocks per component plane.  FP64 rows of up to 256 points: 256 values, so
    // that the phases of two or more blocks on an SM overlap (FP64 256^2, us, event-timed: BCCG
    // iterate 22.1 -> 18.8, direction 13.4 -> 12.6; eight of them 55 -> 49; 512-point rows are
    // better off with 512: iterate 29.8, with 256 values 31.1)
    static constexpr int VALUES = !F32 && NX <= 256 ? 256 : 512;
    static constexpr int ROWS = pow2floor(cmax(1, cmin(16, VALUES / (NC * M))));   // divides every ny >= 16
    // 128 threads for up to 1024 complex values (and the 1536 of an FP32 1024-point three-component
    // row, whose passes then hold seven blocks per SM), else 256
    static constexpr int NT = (NC * ROWS * M >= 1024 && !(F32 && NX == 1024)) ? 256 : 128;
    // FP32 forward passes: ask the register allocator for 8 resident 128-thread
    // blocks per SM (64 registers), so that enough loads are in flight, on the
    // sizes where the tangent of the mechanics pass fits without spilling; the
    // 512-point three-component pass takes 9 (56 registers, 8 bytes of spill:
    // measured 0.7 % faster in the concurrent-stream launch mode), the 2048-point
    // one-component pass 5 of 256 threads (BCCG direction 24.1 -> 22.1 us)
    static constexpr int MINB = !F32 ? 1
                                : NX == 128 || NX == 512 || NX == 1024 ? (NX == 512 && NC == 3 ? 9 : 8)
                                : NX == 2048 && NC == 1                ? 5
                                                                       : 1;
    // FP32 inverse passes of 256 points on take their epilogue's loads a few pixels at a time after
    // the FFT and ask for enough resident blocks to overlap it with other blocks' transforms, instead
    // of prefetching all of a thread's pixels (up to 8, 70 registers) before it: one launch with every
    // problem active, us, prefetching -> here: CG update 2048^2 143 -> 80, 1024^2 36 -> 25, eight 512^2
    // 22.5 -> 20.3; BCCG iterate 2048^2 85 -> 66, 1024^2 31 -> 27, one 512^2 21 -> 18, eight 40 -> 35.
    // (Fewer blocks: 2048-point iterate at 2 blocks 79 us; more: spills, 4 blocks 71 us; 512 threads 81.)
    static constexpr int PREFETCH = F32 && NX >= 256 ? 2 : 8;   // most pixels per thread that are prefetched
    static constexpr int MINB_INV = !F32 ? 1
                                    : NX == 2048 ? (NC == 3 ? 4 : 3)
                                    : NX == 1024 ? 7
                                    : NX == 512  ? (NC == 3 ? 9 : 7)
                                    : NX == 256  ? (NC == 3 ? 10 : 6)
                                                 : 1;
    static constexpr bool EARLY = EARLY_SPECTRUM<T, NX, NC>;   // (inverse passes)
    static constexpr int SP = padded_len(M) + 2;            // pitch (complex): padded M values + slot for k = M
    static constexpr int NSEQ = NC * ROWS;
    // twiddles staged in shared memory: length-M FFT table (padded indices) + the
    // real-FFT factors exp(-2 pi i k / NX), k < M/2 (the split handles k and M - k together)
    static constexpr int TWF = padded_len(M);
    static constexpr int TWS = TWF + M / 2;
    static constexpr size_t SMEM = (size_t)(NSEQ * SP + TWS) * sizeof(typename CT<T>::t);
};

template <typename T, int NY, int NC>
struct ColCfg {
    static constexpr int CSZ = (int)sizeof(typename CT<T>::t);
    static constexpr int CWMIN = 32 / CSZ;                   // one 32-byte sector per row segment
    // one 32-byte sector per row segment: enough columns per block for full
    // sectors, and as many blocks as possible.  FP64 columns of 256 points on: one per block, half a
    // sector (the other half comes from L2 for the next block), since twice the blocks fill the chip
    // and overlap (us, event-timed, two columns -> one: CG pass 256^2 21.1 -> 14.2, 256 x 512 34.8 -> 24.3,
    // 512^2 39, 1024^2 135 -> 129, four 512^2 119 -> 108, 2048 x 256 61 -> 54).  Shorter columns keep two
    // (1024 x 128: 20.7, one column 25.2).
    static constexpr int CWE = sizeof(T) == 8 && NY >= 256 ? 1 : CWMIN;
    static constexpr int SP = ((padded_len(NY) + 7) / 16) * 16 + 8;   // pitch = 8 (mod 16) slots
    static constexpr int NSEQ = NC * CWE;
    static constexpr int NT = (NSEQ * NY >= 8192) ? 512 : (NSEQ * NY >= 2048 ? 256 : 128);
    // twiddles in shared memory when they fit next to the data (not for FP64 at 2048)
    static constexpr bool TW_SMEM = (size_t)(NSEQ * SP + padded_len(NY)) * CSZ <= 225 * 1024;
    static constexpr size_t SMEM = (size_t)(NSEQ * SP + (TW_SMEM ? padded_len(NY) : 0)) * CSZ;
};

constexpr int WP_ALIGN = 16;   // spectral row pitch multiple (largest column tile)

// Per-block mode constants in the storage precision (converted from FP64 once
// per thread, never per element: the FP64 pipe is narrow).
template <typename T>
struct ModeK {
    T cx, cy, inv_n;
    int nx, ny;
    const Consts* kc;       // the problem constants (read only by rarely used multipliers)
    T pre_a, pre_k;         // preconditioner (a_mean, 2 c ell^2), set by multipliers that need them
    int full = 0;           // an explicit residual's slot (FColLapPFS)
    __device__ __forceinline__ ModeK() {}
    __device__ __forceinline__ explicit ModeK(const Desc<T>& d)
        : cx(T(d.k.two_pi_over_Lx)), cy(T(d.k.two_pi_over_Ly)), inv_n(T(d.k.inv_n)), nx(d.nx), ny(d.ny), kc(&d.k) {}
};


// real value x of a real sequence stored as complex pairs z[n] = x[2n] + i x[2n+1]
__device__ __forceinline__ int ridx(int x) { return 2 * pidx(x >> 1) + (x & 1); }

// ---------------------------------------------------------------------------
// Functor interface (F):
//   static constexpr int NR;                      // reduced doubles (0: none)
//   struct Ctx; static Ctx prep(const Desc<T>&);  // per-block constants
//   static bool skip(const Desc<T>&);             // whole-problem early exit
//   static void pixel(const Desc<T>&, const Ctx&, size_t i, T (&v)[NC], Acc<T> (&acc)[NR]);
//   static void finalize(const Desc<T>&, const double (&tot)[NR]);   // one thread
#ifndef PFF_ROW_G
#define PFF_ROW_G 2
#endif
template <class F, bool TWO> struct InOf { struct type {}; };
template <class F> struct InOf<F, true> { using type = typename F::In; };

// Row-forward pass of one row group y0 (ROWS rows): pixel prologue into the
// sequence buffer (accumulating F's reductions in acc) ...
template <typename T, int NX, int NC, class F>
__device__ __forceinline__ void row_fwd_pixels(const Desc<T>& d, const typename F::Ctx& ctx, int y0,
                                               typename CT<T>::t* buf, Acc<T>* acc) {
    using Cfg = RowCfg<T, NX, NC>;
    constexpr int SP = Cfg::SP, ROWS = Cfg::ROWS, NT = Cfg::NT;
    T* rb = reinterpret_cast<T*>(buf);
    if constexpr (HasIn<F>::value && (ROWS * NX) % NT == 0) {
        constexpr int PPT = ROWS * NX / NT;
        // pixels whose loads are in flight together: PFF_ROW_G, or as many as about 32
        // registers of loaded values allow (a power of two, so that it divides PPT)
        constexpr int WORDS = (int)((sizeof(typename F::In) + 3) / 4);
        constexpr int G = pow2floor(cmin(PPT, cmax(PFF_ROW_G, 32 / WORDS)));
#pragma unroll
        for (int j0 = 0; j0 < PPT; j0 += G) {
            typename F::In in[G];
#pragma unroll
            for (int j = 0; j < G; ++j) {
                const int t = threadIdx.x + (j0 + j) * NT;
                in[j] = F::load(d, ctx, (size_t)(y0 + t / NX) * NX + t % NX);
            }
#pragma unroll
            for (int j = 0; j < G; ++j) {
                const int t = threadIdx.x + (j0 + j) * NT;
                const int row = t / NX, x = t % NX;
                T v[NC];
                F::pixel(d, ctx, (size_t)(y0 + row) * NX + x, in[j], v, acc);
#pragma unroll
                for (int c = 0; c < NC; ++c) rb[(c * ROWS + row) * 2 * SP + ridx(x)] = v[c];
            }
        }
    } else {
#pragma unroll 4
        for (int t = threadIdx.x; t < ROWS * NX; t += NT) {
            const int row = t / NX, x = t % NX;
            const size_t pix = (unsigned)(y0 + row) * NX + x;
            T v[NC];
            pixel_one<F>(d, ctx, pix, v, acc);
#pragma unroll
            for (int c = 0; c < NC; ++c) rb[(c * ROWS + row) * 2 * SP + ridx(x)] = v[c];
        }
    }
}

// ... then (after a barrier) the real FFT along x and the half-spectrum store.
template <typename T, int NX, int NC>
__device__ __forceinline__ void row_fwd_fft_store(const Desc<T>& d, int y0, typename CT<T>::t* buf,
                                                  const typename CT<T>::t* tws) {
    using Cfg = RowCfg<T, NX, NC>;
    using C = typename CT<T>::t;
    constexpr int M = Cfg::M, SP = Cfg::SP, ROWS = Cfg::ROWS, NT = Cfg::NT;
    fft_smem<T, M, Cfg::NSEQ, SP, NT, false, true>(buf, tws);
    // real-to-complex post-processing of z = FFT(x[2n] + i x[2n+1]):
    //   X[k] = e + t,  e = (z[k] + conj z[M-k]) / 2,  t = W_N^k (z[k] - conj z[M-k]) / 2i,
    // and, from the same two values, X[M-k] = conj(e - t) (W_N^(M-k) = -conj W_N^k);
    // k = 0 gives X[0] and X[M], and its lane also writes the self-paired X[M/2] = conj z[M/2].
    constexpr int H = M / 2;
    const C* twN = tws + Cfg::TWF;
    const unsigned plane = (unsigned)d.ny * d.wp;   // 32-bit indices: < 2^32 elements
    for (int t = threadIdx.x; t < Cfg::NSEQ * H; t += NT) {
        const int s = t / H, k = t % H;
        const int c = s / ROWS, row = s % ROWS;
        C* out = d.S + (c * plane + (unsigned)(y0 + row) * d.wp);
        C zk = buf[s * SP + pidx(k)];
        C zm = buf[s * SP + pidx(k == 0 ? 0 : M - k)];
        zm.y = -zm.y;
        C e = C{T(0.5) * (zk.x + zm.x), T(0.5) * (zk.y + zm.y)};
        C o = C{T(0.5) * (zk.y - zm.y), T(-0.5) * (zk.x - zm.x)};
        C tk = cmul(twN[k], o);
        out[k] = cadd(e, tk);
        out[M - k] = C{e.x - tk.x, tk.y - e.y};
        if (k == 0) {
            C zh = buf[s * SP + pidx(H)];
            out[H] = C{zh.x, -zh.y};
        }
    }
}

// staged row twiddles: FFT table of length M at pidx(j), then exp(-2 pi i k / NX), k < M/2
template <typename T, int NX, int NC>
__device__ __forceinline__ void stage_row_twiddles(const Desc<T>& d, typename CT<T>::t* tws) {
    using Cfg = RowCfg<T, NX, NC>;
    using C = typename CT<T>::t;
    constexpr int M = Cfg::M;
    for (int t = threadIdx.x; t < M + M / 2; t += blockDim.x)
        cp_async<sizeof(C)>(t < M ? &tws[pidx(t)] : &tws[Cfg::TWF + (t - M)], t < M ? &d.tw[M + t] : &d.tw[NX + (t - M)]);
}

template <typename T, int NX, int NC, class F>
__device__ __forceinline__ void row_fwd_body(const Desc<T>& d) {
    using Cfg = RowCfg<T, NX, NC>;
    using C = typename CT<T>::t;
    constexpr int NT = Cfg::NT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* buf = reinterpret_cast<C*>(smem_raw);
    C* tws = buf + Cfg::NSEQ * Cfg::SP;
    pdl_enter();
    typename F::Ctx ctx;
    if (block_prep<F>(d, ctx)) return;
    // twiddles are needed only after the pixel phase: staged after the skip test,
    // so that the blocks of a skipped problem return at once
    stage_row_twiddles<T, NX, NC>(d, tws);
    const int y0 = blockIdx.x * Cfg::ROWS;
    constexpr int NRA = F::NR > 0 ? F::NR : 1;
    Acc<T> acc[NRA];
    row_fwd_pixels<T, NX, NC, F>(d, ctx, y0, buf, &acc[0]);
    if constexpr (F::NR > 0) reduce_finalize<F, F::NR, NT>(acc, d, gridDim.x);
    cp_async_wait_all();
    __syncthreads();
    row_fwd_fft_store<T, NX, NC>(d, y0, buf, tws);
}

// Each row kernel comes in two forms: with the register cap of its configuration (minimum
// resident blocks per SM; the FP32 sizes whose caps were chosen by measurement) and, suffix
// _u, without a minimum (the compiler's own choice: a minimum of one block is not the same as
// no bound to ptxas, which then takes more registers).
template <typename T, int NX, int NC, class F>
__global__ void __launch_bounds__(RowCfg<T, NX, NC>::NT, RowCfg<T, NX, NC>::MINB) k_row_fwd(const Desc<T>* __restrict__ descs) {
    row_fwd_body<T, NX, NC, F>(descs[blockIdx.y]);
}
template <typename T, int NX, int NC, class F>
__global__ void __launch_bounds__(RowCfg<T, NX, NC>::NT) k_row_fwd_u(const Desc<T>* __restrict__ descs) {
    row_fwd_body<T, NX, NC, F>(descs[blockIdx.y]);
}

// the half-spectrum rows of a row group on their way to shared memory (asynchronous copies)
template <typename T, int NX, int NC>
__device__ __forceinline__ void row_inv_stage(const Desc<T>& d, int y0, typename CT<T>::t* buf) {
    using Cfg = RowCfg<T, NX, NC>;
    using C = typename CT<T>::t;
    constexpr int M = Cfg::M, SP = Cfg::SP, ROWS = Cfg::ROWS;
    const unsigned plane = (unsigned)d.ny * d.wp;   // 32-bit indices: < 2^32 elements
    for (int t = threadIdx.x; t < Cfg::NSEQ * (M + 1); t += Cfg::NT) {
        const int s = t / (M + 1), k = t % (M + 1);
        const int c = s / ROWS, row = s % ROWS;
        cp_async<sizeof(C)>(&buf[s * SP + pidx(k)], &d.S[c * plane + (unsigned)(y0 + row) * d.wp + k]);
    }
}

// Row-inverse pass of one row group y0: a few pixels' epilogue loads are issued
// first (they land during the staging and the FFT; see PREFETCH), the half-spectrum rows are
// staged (STAGED: already on their way), combined for the complex-to-real transform, transformed back
// along x, and the epilogue runs on the real values (accumulating F's reductions in acc).
template <typename T, int NX, int NC, class F, bool STAGED = false>
__device__ __forceinline__ void row_inv_item(const Desc<T>& d, const typename F::Ctx& ctx, int y0,
                                             typename CT<T>::t* buf, const typename CT<T>::t* tws, Acc<T>* acc) {
    using Cfg = RowCfg<T, NX, NC>;
    using C = typename CT<T>::t;
    constexpr int M = Cfg::M, SP = Cfg::SP, ROWS = Cfg::ROWS, NT = Cfg::NT;
    const T* rb = reinterpret_cast<const T*>(buf);
    constexpr bool TWO = HasIn<F>::value && (ROWS * NX) % NT == 0 && ROWS * NX / NT <= Cfg::PREFETCH;
    constexpr int PPT = TWO ? ROWS * NX / NT : 1;
    using InT = typename InOf<F, TWO>::type;
    InT in[PPT];
    if constexpr (TWO) {
#pragma unroll
        for (int j = 0; j < PPT; ++j) {
            const int t = threadIdx.x + j * NT;
            in[j] = F::load(d, ctx, (size_t)((unsigned)(y0 + t / NX) * NX + t % NX));
        }
    }
    const C* twN = tws + Cfg::TWF;
    // complex-to-real pre-processing: Z[k] = A + i B,
    //   A = X[k] + conj(X[M-k]),  B = (X[k] - conj(X[M-k])) e^{+2 pi i k/N}
    // (imaginary parts of X[0] and X[M] are dropped, as for a real inverse); the same two
    // values give Z[M-k] = conj(A) + i conj(B), and Z[M/2] = 2 conj(X[M/2]) (k and M - k
    // together, k < M/2; the k = 0 lane forms Z[0] and Z[M/2]).
    // stage the half spectrum rows in shared memory, then combine
    if constexpr (!STAGED) row_inv_stage<T, NX, NC>(d, y0, buf);
    cp_async_wait_all();
    __syncthreads();
    // (a lane's two values replace the two that it read, so the combination runs in place)
    constexpr int H = M / 2, NI = (Cfg::NSEQ * H + NT - 1) / NT;
#pragma unroll
    for (int u = 0; u < NI; ++u) {
        const int t = threadIdx.x + u * NT;
        if ((Cfg::NSEQ * H) % NT == 0 || t < Cfg::NSEQ * H) {
            const int s = t / H, k = t % H;
            C *lo = &buf[s * SP + pidx(k)], *hi = &buf[s * SP + pidx(M - k)];
            C xk = *lo, xm = *hi;
            if (k == 0) { xk.y = T(0); xm.y = T(0); }
            xm.y = -xm.y;
            C A = cadd(xk, xm);
            C B = cmulc(csub(xk, xm), twN[k]);
            *lo = C{A.x - B.y, A.y + B.x};
            if (k > 0) {
                *hi = C{A.x + B.y, B.x - A.y};
            } else {
                C* h = &buf[s * SP + pidx(H)];
                *h = C{T(2) * h->x, T(-2) * h->y};
            }
        }
    }
    __syncthreads();
    fft_smem<T, M, Cfg::NSEQ, SP, NT, true, true>(buf, tws);
    if constexpr (TWO) {
#pragma unroll
        for (int j = 0; j < PPT; ++j) {
            const int t = threadIdx.x + j * NT;
            const int row = t / NX, x = t % NX;
            T v[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) v[c] = rb[(c * ROWS + row) * 2 * SP + ridx(x)];
            F::pixel(d, ctx, (size_t)((unsigned)(y0 + row) * NX + x), in[j], v, acc);
        }
    } else if constexpr (HasIn<F>::value && (ROWS * NX) % NT == 0) {
        (void)in;
        // the loads of a few pixels at a time (about 32 registers) are in flight together
        constexpr int N = ROWS * NX / NT, WORDS = (int)((sizeof(typename F::In) + 3) / 4);
        constexpr int G = pow2floor(cmin(N, cmax(2, 32 / WORDS)));
#pragma unroll 1
        for (int j0 = 0; j0 < N; j0 += G) {
            typename F::In b[G];
#pragma unroll
            for (int j = 0; j < G; ++j) {
                const int t = threadIdx.x + (j0 + j) * NT;
                b[j] = F::load(d, ctx, (size_t)((unsigned)(y0 + t / NX) * NX + t % NX));
            }
#pragma unroll
            for (int j = 0; j < G; ++j) {
                const int t = threadIdx.x + (j0 + j) * NT;
                const int row = t / NX, x = t % NX;
                T v[NC];
#pragma unroll
                for (int c = 0; c < NC; ++c) v[c] = rb[(c * ROWS + row) * 2 * SP + ridx(x)];
                F::pixel(d, ctx, (size_t)((unsigned)(y0 + row) * NX + x), b[j], v, acc);
            }
        }
    } else {
        (void)in;
#pragma unroll 4
        for (int t = threadIdx.x; t < ROWS * NX; t += NT) {
            const int row = t / NX, x = t % NX;
            const size_t pix = (unsigned)(y0 + row) * NX + x;
            T v[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) v[c] = rb[(c * ROWS + row) * 2 * SP + ridx(x)];
            pixel_one<F>(d, ctx, pix, v, acc);
        }
    }
}

template <typename T, int NX, int NC, class F>
__device__ __forceinline__ void row_inv_body(const Desc<T>& d) {
    using Cfg = RowCfg<T, NX, NC>;
    using C = typename CT<T>::t;
    constexpr int NT = Cfg::NT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* buf = reinterpret_cast<C*>(smem_raw);
    C* tws = buf + Cfg::NSEQ * Cfg::SP;
    pdl_enter();
    if constexpr (Cfg::EARLY) {
        row_inv_stage<T, NX, NC>(d, blockIdx.x * Cfg::ROWS, buf);
        stage_row_twiddles<T, NX, NC>(d, tws);
    }
    typename F::Ctx ctx;
    if (block_prep<F>(d, ctx)) {
        if constexpr (Cfg::EARLY) cp_async_wait_all();
        return;
    }
    if constexpr (!Cfg::EARLY) stage_row_twiddles<T, NX, NC>(d, tws);
    constexpr int NRA = F::NR > 0 ? F::NR : 1;
    Acc<T> acc[NRA];
    row_inv_item<T, NX, NC, F, Cfg::EARLY>(d, ctx, blockIdx.x * Cfg::ROWS, buf, tws, &acc[0]);
    if constexpr (F::NR > 0) reduce_finalize<F, F::NR, NT>(acc, d, gridDim.x);
}
template <typename T, int NX, int NC, class F>
__global__ void __launch_bounds__(RowCfg<T, NX, NC>::NT, RowCfg<T, NX, NC>::MINB_INV) k_row_inv(const Desc<T>* __restrict__ descs) {
    row_inv_body<T, NX, NC, F>(descs[blockIdx.y]);
}
template <typename T, int NX, int NC, class F>
__global__ void __launch_bounds__(RowCfg<T, NX, NC>::NT) k_row_inv_u(const Desc<T>* __restrict__ descs) {
    row_inv_body<T, NX, NC, F>(descs[blockIdx.y]);
}

// Column pass: CWE adjacent columns kx of the half spectrum, all NC planes.
// OP::apply(d, kx, ky, vals[NC]) multiplies one mode (normalisation included).
// column multipliers may read further per-problem constants into the ModeK (mode_prep)
template <class OP, class = void> struct HasModePrep { static constexpr bool value = false; };
template <class OP> struct HasModePrep<OP, decltype((void)&OP::template mode_prep<float>, void())> {
    static constexpr bool value = true;
};

// Column multipliers may also reduce over the modes they see (before multiplying):
// OP::NR values, OP::accum(mk, kx, ky, v, acc) per mode, OP::finalize(d, tot) once.
template <class OP, class = void> struct ColNR { static constexpr int value = 0; };
template <class OP> struct ColNR<OP, decltype((void)OP::NR, void())> { static constexpr int value = OP::NR; };

// skip test and mode constants of a column pass, evaluated once per block
template <typename T, class OP>
struct ColPrep {
    __device__ static bool skip(const Desc<T>& d) { return OP::skip(d); }
    __device__ static ModeK<T> prep(const Desc<T>& d) {
        ModeK<T> m(d);
        if constexpr (HasModePrep<OP>::value) OP::mode_prep(d, m);
        return m;
    }
};

template <typename T, int NY, int NC, class OP>
__device__ __forceinline__ void col_body(const Desc<T>& d) {
    using Cfg = ColCfg<T, NY, NC>;
    using C = typename CT<T>::t;
    constexpr int CW = Cfg::CWE, SP = Cfg::SP, NT = Cfg::NT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* buf = reinterpret_cast<C*>(smem_raw);
    pdl_enter();
    ModeK<T> mk;
    constexpr bool EARLY = EARLY_SPECTRUM<T, NY, NC>;
    if constexpr (!EARLY)
        if (block_prep<ColPrep<T, OP>>(d, mk)) return;
    const C* tw = d.tw + NY;
    if constexpr (Cfg::TW_SMEM) {
        C* tws = buf + Cfg::NSEQ * SP;
        for (int t = threadIdx.x; t < NY; t += NT) cp_async<sizeof(C)>(&tws[pidx(t)], &d.tw[NY + t]);
        tw = tws;
    }
    const int kx0 = blockIdx.x * CW;
    const unsigned plane = (unsigned)d.ny * d.wp;   // 32-bit indices: < 2^32 elements
    constexpr int TOT = NC * NY * CW;
    for (int t = threadIdx.x; t < TOT; t += NT) {
        const int j = t % CW, ky = (t / CW) % NY, c = t / (CW * NY);
        cp_async<sizeof(C)>(&buf[(c * CW + j) * SP + pidx(ky)], &d.S[c * plane + (unsigned)ky * d.wp + kx0 + j]);
    }
    if constexpr (EARLY)
        if (block_prep<ColPrep<T, OP>>(d, mk)) {
            cp_async_wait_all();
            return;
        }
    cp_async_wait_all();
    __syncthreads();
    fft_smem<T, NY, Cfg::NSEQ, SP, NT, false, Cfg::TW_SMEM>(buf, tw);
    constexpr int NRA = ColNR<OP>::value > 0 ? ColNR<OP>::value : 1;
    Acc<T> acc[NRA];
    for (int t = threadIdx.x; t < CW * NY; t += NT) {
        const int ky = t % NY, j = t / NY;
        C v[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) v[c] = buf[(c * CW + j) * SP + pidx(ky)];
        if constexpr (ColNR<OP>::value > 0) OP::accum(mk, kx0 + j, ky, v, acc);
        OP::apply(mk, kx0 + j, ky, v);
#pragma unroll
        for (int c = 0; c < NC; ++c) buf[(c * CW + j) * SP + pidx(ky)] = v[c];
    }
    __syncthreads();
    fft_smem<T, NY, Cfg::NSEQ, SP, NT, true, Cfg::TW_SMEM>(buf, tw);
#pragma unroll 4
    for (int t = threadIdx.x; t < TOT; t += NT) {
        const int j = t % CW, ky = (t / CW) % NY, c = t / (CW * NY);
        d.S[c * plane + (unsigned)ky * d.wp + kx0 + j] = buf[(c * CW + j) * SP + pidx(ky)];
    }
    if constexpr (ColNR<OP>::value > 0) reduce_finalize<OP, ColNR<OP>::value, NT>(acc, d, gridDim.x);
}
template <typename T, int NY, int NC, class OP>
__global__ void __launch_bounds__(ColCfg<T, NY, NC>::NT) k_col(const Desc<T>* __restrict__ descs) {
    col_body<T, NY, NC, OP>(descs[blockIdx.y]);
}

// ---------------------------------------------------------------------------
// Column pass for ny = 512 with register-resident radix-8 stages (512 = 8 x 8 x 8).
// Thread (column j, lane t) loads rows t + 64 m (m < 8) of every component
// straight into registers and runs the three radix-8 stages with two
// shared-memory exchanges:
//   stage 1: DFT8 over m, twiddle W512^(n0 k1)           (n0 = the lane's index)
//   stage 2: lane (k1, a): DFT8 over b of stage-1 values at n0 = a + 8 b, twiddle W64^(a c)
//   stage 3: lane (k1, c): DFT8 over a -> modes k1 + 8 c + 64 e, e < 8
// (k1 = t / 8, a or c = t % 8).  The mode multiplier acts on the NC components a
// lane holds; the inverse runs the same stages with lane index t' = k1 + 8 c (the
// lane holds modes t' + 64 e) and ends on rows t' + 64 e, stored straight from
// registers.  Exchange layouts (per component and column, stride COL512_XS = 8
// mod 16 complex slots): stage-1 value (k1, n0) at 72 k1 + n0 + n0/8, stage-2
// value (k1, a, c) at 72 k1 + 9 a + c; every access of a warp touches each
// bank pair at most twice (FP32).
constexpr int COL512_CW = 4;       // default columns per block (one 32-byte sector per row in FP32; 2 selectable)
constexpr int COL512_XS = 584;     // exchange slots per component and column

template <typename C, bool INV>
__device__ __forceinline__ void tw8(const C* tws, int base, C (&w)[8]) {
    // W512^(base r) for r < 8 from the entries for r = 1, 2, 4 (conjugated for the
    // inverse); the staged table is padded like the sequences (pidx), so that the
    // strided reads of a warp do not collide in the shared-memory banks
    C w1 = tws[pidx(base)], w2 = tws[pidx(2 * base)], w4 = tws[pidx(4 * base)];
    if (INV) { w1.y = -w1.y; w2.y = -w2.y; w4.y = -w4.y; }
    const C w3 = cmul(w1, w2);
    w[1] = w1; w[2] = w2; w[3] = w3; w[4] = w4;
    w[5] = cmul(w1, w4); w[6] = cmul(w2, w4); w[7] = cmul(w3, w4);
}

template <typename T, bool INV, int NC, int CW>
__device__ __forceinline__ void fft512_reg(typename CT<T>::t (&u)[NC][8], int n0, int t, typename CT<T>::t* xb,
                                           const typename CT<T>::t* tws) {
    using C = typename CT<T>::t;
    constexpr int CS = CW * COL512_XS;   // component stride
    C w[8];
    // stage 1
    tw8<C, INV>(tws, n0, w);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        dft8<C, INV>(u[c]);
#pragma unroll
        for (int r = 1; r < 8; ++r) u[c][r] = cmul(u[c][r], w[r]);
    }
    __syncthreads();   // earlier readers of xb are done
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int k1 = 0; k1 < 8; ++k1) xb[c * CS + 72 * k1 + n0 + (n0 >> 3)] = u[c][k1];
    __syncthreads();
    // stage 2
    const int k1 = t >> 3, a = t & 7;
    tw8<C, INV>(tws, 8 * a, w);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
#pragma unroll
        for (int b = 0; b < 8; ++b) u[c][b] = xb[c * CS + 72 * k1 + a + 9 * b];
        dft8<C, INV>(u[c]);
#pragma unroll
        for (int r = 1; r < 8; ++r) u[c][r] = cmul(u[c][r], w[r]);
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int cc = 0; cc < 8; ++cc) xb[c * CS + 72 * k1 + 9 * a + cc] = u[c][cc];
    __syncthreads();
    // stage 3 (lane (k1, c) with c = a)
#pragma unroll
    for (int c = 0; c < NC; ++c) {
#pragma unroll
        for (int aa = 0; aa < 8; ++aa) u[c][aa] = xb[c * CS + 72 * k1 + 9 * aa + a];
        dft8<C, INV>(u[c]);
    }
}

template <typename T, int NC, int CW = COL512_CW>
struct Col512Cfg {
    static constexpr int NT = 64 * CW;
    static constexpr size_t SMEM = (size_t)(padded_len(512) + NC * CW * COL512_XS) * sizeof(typename CT<T>::t);
};

// staged column twiddles: exp(-2 pi i k / 512) at pidx(k), k < 512
template <typename T>
__device__ __forceinline__ void stage_col512_twiddles(const Desc<T>& d, typename CT<T>::t* tws) {
    for (int i = threadIdx.x; i < 512; i += blockDim.x) cp_async<sizeof(typename CT<T>::t)>(&tws[pidx(i)], &d.tw[512 + i]);
}

// Column pass of the CW columns kx0.. of the half spectrum (64 CW threads).
template <typename T, int NC, int CW>
__device__ __forceinline__ void col512_load(const Desc<T>& d, int kx0, typename CT<T>::t (&u)[NC][8]) {
    const int t = threadIdx.x / CW, kx = kx0 + threadIdx.x % CW;
    const unsigned plane = (unsigned)d.ny * d.wp;   // 32-bit indices: < 2^32 elements
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int m = 0; m < 8; ++m) u[c][m] = d.S[c * plane + (unsigned)(t + 64 * m) * d.wp + kx];
}
// (u: the columns, from col512_load)
template <typename T, int NC, class OP, int CW>
__device__ __forceinline__ void col512_item(const Desc<T>& d, const ModeK<T>& mk, int kx0, typename CT<T>::t* xb,
                                            const typename CT<T>::t* tws, typename CT<T>::t (&u)[NC][8],
                                            Acc<T>* acc = nullptr) {
    using C = typename CT<T>::t;
    const int j = threadIdx.x % CW, t = threadIdx.x / CW;
    const int kx = kx0 + j;
    const unsigned plane = (unsigned)d.ny * d.wp;
    cp_async_wait_all();   // staged twiddles (a no-op when the caller has waited already)
    __syncthreads();
    fft512_reg<T, false, NC, CW>(u, t, t, xb + j * COL512_XS, tws);
    const int k1 = t >> 3, cc = t & 7;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        C v[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) v[c] = u[c][e];
        if constexpr (ColNR<OP>::value > 0) OP::accum(mk, kx, k1 + 8 * cc + 64 * e, v, acc);
        OP::apply(mk, kx, k1 + 8 * cc + 64 * e, v);
#pragma unroll
        for (int c = 0; c < NC; ++c) u[c][e] = v[c];
    }
    const int tp = k1 + 8 * cc;
    fft512_reg<T, true, NC, CW>(u, tp, t, xb + j * COL512_XS, tws);
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int e = 0; e < 8; ++e) d.S[c * plane + (unsigned)(tp + 64 * e) * d.wp + kx] = u[c][e];
}

template <typename T, int NC, class OP, int CW>
__device__ __forceinline__ void col512_body(const Desc<T>& d) {
    using C = typename CT<T>::t;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* tws = reinterpret_cast<C*>(smem_raw);
    C* xb = tws + padded_len(512);
    pdl_enter();
    ModeK<T> mk;
    C u[NC][8];
    constexpr bool EARLY = EARLY_SPECTRUM<T, 512, NC>;
    if constexpr (EARLY) {
        stage_col512_twiddles<T>(d, tws);   // waited for inside the item
        col512_load<T, NC, CW>(d, blockIdx.x * CW, u);
    }
    if (block_prep<ColPrep<T, OP>>(d, mk)) {
        if constexpr (EARLY) cp_async_wait_all();
        return;
    }
    if constexpr (!EARLY) {
        stage_col512_twiddles<T>(d, tws);
        col512_load<T, NC, CW>(d, blockIdx.x * CW, u);
    }
    constexpr int NRA = ColNR<OP>::value > 0 ? ColNR<OP>::value : 1;
    Acc<T> acc[NRA];
    col512_item<T, NC, OP, CW>(d, mk, blockIdx.x * CW, xb, tws, u, acc);
    if constexpr (ColNR<OP>::value > 0) reduce_finalize<OP, ColNR<OP>::value, 64 * CW>(acc, d, gridDim.x);
}
template <typename T, int NC, class OP, int CW = COL512_CW>
__global__ void __launch_bounds__(64 * CW) k_col512(const Desc<T>* __restrict__ descs) {
    col512_body<T, NC, OP, CW>(descs[blockIdx.y]);
}

// ---------------------------------------------------------------------------
// Column pass for ny = 1024 and 2048 (FP32) with sixteen values of every component in a thread's
// registers: ny = 16 x 16 x R3 (R3 = 4 or 8), N1 = ny / 16 threads per column.
//   stage 1: thread t holds rows t + N1 m (m < 16): DFT16 over m -> k1, twiddle W_ny^(t k1)
//   stage 2: thread (k1, a), a < R3, holds t = a + R3 b (b < 16): DFT16 over b -> k2, twiddle W_N1^(a k2)
//   stage 3: thread t holds the groups g = k1 + 16 k2 = t + N1 q (q < 16 / R3): DFT R3 over a -> k3,
//            modes ky = g + 256 k3
// The multiplier acts on the NC components of a mode, which one thread holds, and the inverse runs the
// stages backwards with the same twiddles conjugated, so a column makes two exchanges through shared
// memory each way instead of the eight to ten passes of the Stockham form.  Exchange layouts per
// component and column (column stride XS): stage-1 value (k1, t) at (N1 + R3) k1 + t, stage-2 value
// (a, g) at (256 + P2) a + g; with XS = 16 / CW (mod 16) a half-warp's 8-byte accesses touch 16
// different bank pairs.  Four columns (one 32-byte sector per row and access): with two, and two
// blocks per SM, the line accesses of the loads and stores lead (2048^2 three components 77-104 us).
// One launch, us, Stockham pass -> here: three components 2048^2 107 -> 75, 1024^2 27 -> 18; one
// component 2048^2 33 -> 22, with the BCCG's sum 42 -> 26 (two blocks per SM; 1024^2 18 -> 14).  What is
// left is latency: 16 warps per SM (98 registers of data a thread, 200 KB of exchange buffers).
template <typename C, bool INV>
__device__ __forceinline__ void dft16(C* u) {   // X[k] ends at u[4 (k mod 4) + k / 4]
    using T = decltype(u[0].x);
    const T c1 = T(0.92387953251128675613), s1 = T(0.38268343236508977173), h = T(0.70710678118654752440);
    const C w1{c1, INV ? s1 : -s1}, w2{h, INV ? h : -h}, w3{s1, INV ? c1 : -c1};
#pragma unroll
    for (int n = 0; n < 4; ++n) dft4<C, INV>(u[n], u[4 + n], u[8 + n], u[12 + n]);
    u[5] = cmul(u[5], w1);
    u[6] = cmul(u[6], w2);
    u[7] = cmul(u[7], w3);
    u[9] = cmul(u[9], w2);
    u[10] = INV ? C{-u[10].y, u[10].x} : C{u[10].y, -u[10].x};
    u[11] = cmul(u[11], C{-h, INV ? h : -h});
    u[13] = cmul(u[13], w3);
    u[14] = cmul(u[14], C{-h, INV ? h : -h});
    u[15] = cmul(u[15], C{-c1, INV ? -s1 : s1});
#pragma unroll
    for (int k = 0; k < 4; ++k) dft4<C, INV>(u[4 * k], u[4 * k + 1], u[4 * k + 2], u[4 * k + 3]);
}
__host__ __device__ constexpr int at16(int k) { return 4 * (k & 3) + (k >> 2); }   // place of X[k] after dft16

template <typename T, int NY, int NC, int CW>
struct Col16Cfg {
    static constexpr int N1 = NY / 16, R3 = NY / 256, NT = CW * N1;
    static constexpr int P1 = N1 + R3;                       // pitch of a stage-1 row
    static constexpr int P2 = 256 + (CW == 2 && R3 == 4 ? 2 : 1);
    static constexpr int NEED = cmax(16 * P1, R3 * P2), OFF = 16 / CW;
    static constexpr int XS = ((NEED - OFF + 15) / 16) * 16 + OFF;
    static constexpr size_t SMEM = (size_t)NC * CW * XS * sizeof(typename CT<T>::t);
};

// u[c][at(r)] *= w^r for r = 1 .. 15.  TABLE: all from the table tw[r step]; else w^1, w^2, w^3, w^4, w^8,
// w^12, and the others as products of two of these.  Products of three (from w^1, w^2, w^4, w^8) made the
// Laplacian of a field with 1024 rows 8 % and with 2048 rows 4 % less accurate than the Stockham pass; now they
// are 4 % and 2 % more accurate.  With 2048 points the whole table costs 5 % of a load step (registers), with
// 1024 points 0.9 % (1024^2 4330 -> 4367 us), the products there 0.5 % of accuracy.
template <typename C, int NC, bool CONJ, bool PERM, bool TABLE>
__device__ __forceinline__ void twiddle16(C (&u)[NC][16], const C* tw, int step) {
    auto from_table = [](int r) { return TABLE || r < 4 || r % 4 == 0; };
    C w[16];
#pragma unroll
    for (int r = 1; r < 16; ++r) {
        if (!from_table(r)) continue;
        const C x = __ldg(tw + r * step);
        w[r] = CONJ ? C{x.x, -x.y} : x;
    }
#pragma unroll
    for (int r = 1; r < 16; ++r) {
        if (!from_table(r)) w[r] = cmul(w[r & ~3], w[r & 3]);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            C& x = u[c][PERM ? at16(r) : r];
            x = cmul(x, w[r]);
        }
    }
}

template <typename T, int NY, int NC, class OP, int CW>
__global__ void __launch_bounds__(CW * NY / 16, NC == 1 && NY == 2048 ? 2 : 1) k_col16(const Desc<T>* __restrict__ descs) {
    using Cfg = Col16Cfg<T, NY, NC, CW>;
    using C = typename CT<T>::t;
    constexpr int N1 = Cfg::N1, R3 = Cfg::R3, P1 = Cfg::P1, P2 = Cfg::P2, CS = CW * Cfg::XS, Q = 16 / R3;
    const Desc<T>& d = descs[blockIdx.y];
    extern __shared__ __align__(16) unsigned char smem_raw[];
    pdl_enter();
    ModeK<T> mk;
    if (block_prep<ColPrep<T, OP>>(d, mk)) return;
    const int j = threadIdx.x % CW, t = threadIdx.x / CW;
    const int kx = blockIdx.x * CW + j;
    C* xb = reinterpret_cast<C*>(smem_raw) + j * Cfg::XS;
    const unsigned plane = (unsigned)d.ny * d.wp;   // 32-bit indices: < 2^32 elements
    C* S = d.S + ((unsigned)t * d.wp + kx);
    const unsigned step = (unsigned)N1 * d.wp;
    const C* tw = d.tw + NY;
    const int k1 = t / R3, a = t % R3;              // stage-2 role
    C u[NC][16];
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int m = 0; m < 16; ++m) u[c][m] = S[c * plane + m * step];
    // forward
#pragma unroll
    for (int c = 0; c < NC; ++c) dft16<C, false>(u[c]);
    twiddle16<C, NC, false, true, NY == 1024>(u, tw, t);
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int k = 0; k < 16; ++k) xb[c * CS + P1 * k + t] = u[c][at16(k)];
    __syncthreads();
#pragma unroll
    for (int c = 0; c < NC; ++c) {
#pragma unroll
        for (int b = 0; b < 16; ++b) u[c][b] = xb[c * CS + P1 * k1 + a + R3 * b];
        dft16<C, false>(u[c]);
    }
    twiddle16<C, NC, false, true, NY == 1024>(u, tw, 16 * a);
    __syncthreads();
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int k = 0; k < 16; ++k) xb[c * CS + P2 * a + 16 * k + k1] = u[c][at16(k)];
    __syncthreads();
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int q = 0; q < Q; ++q) {
#pragma unroll
            for (int r = 0; r < R3; ++r) u[c][q * R3 + r] = xb[c * CS + P2 * r + t + N1 * q];
            if constexpr (R3 == 4) dft4<C, false>(u[c][4 * q], u[c][4 * q + 1], u[c][4 * q + 2], u[c][4 * q + 3]);
            else dft8<C, false>(*reinterpret_cast<C(*)[8]>(&u[c][8 * q]));
        }
    // modes
    constexpr int NRA = ColNR<OP>::value > 0 ? ColNR<OP>::value : 1;
    Acc<T> acc[NRA];
#pragma unroll
    for (int q = 0; q < Q; ++q)
#pragma unroll
        for (int r = 0; r < R3; ++r) {
            const int ky = t + N1 * q + 256 * r;
            C v[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) v[c] = u[c][q * R3 + r];
            if constexpr (ColNR<OP>::value > 0) OP::accum(mk, kx, ky, v, acc);
            OP::apply(mk, kx, ky, v);
#pragma unroll
            for (int c = 0; c < NC; ++c) u[c][q * R3 + r] = v[c];
        }
    // inverse
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            if constexpr (R3 == 4) dft4<C, true>(u[c][4 * q], u[c][4 * q + 1], u[c][4 * q + 2], u[c][4 * q + 3]);
            else dft8<C, true>(*reinterpret_cast<C(*)[8]>(&u[c][8 * q]));
#pragma unroll
            for (int r = 0; r < R3; ++r) xb[c * CS + P2 * r + t + N1 * q] = u[c][q * R3 + r];
        }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int k = 0; k < 16; ++k) u[c][k] = xb[c * CS + P2 * a + 16 * k + k1];
    twiddle16<C, NC, true, false, NY == 1024>(u, tw, 16 * a);
    __syncthreads();
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        dft16<C, true>(u[c]);
#pragma unroll
        for (int b = 0; b < 16; ++b) xb[c * CS + P1 * k1 + a + R3 * b] = u[c][at16(b)];
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int k = 0; k < 16; ++k) u[c][k] = xb[c * CS + P1 * k + t];
    twiddle16<C, NC, true, false, NY == 1024>(u, tw, t);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        dft16<C, true>(u[c]);
#pragma unroll
        for (int m = 0; m < 16; ++m) S[c * plane + m * step] = u[c][at16(m)];
    }
    if constexpr (ColNR<OP>::value > 0) reduce_finalize<OP, ColNR<OP>::value, Cfg::NT>(acc, d, gridDim.x);
}

// ---------------------------------------------------------------------------
// mode multipliers
// Signed wavenumber index of row ky (numpy fftfreq order); Nyquist flagged.
__device__ __forceinline__ int signed_k(int k, int n) { return k < n / 2 ? k : k - n; }

// Compatibility projection Gamma(n) (Sec. 3.1.1), zero at q = 0 and on
// Nyquist modes; scaled by 1/(nx ny).
template <typename T>
__device__ __forceinline__ void gamma_apply(const ModeK<T>& m, int kx, int ky, typename CT<T>::t (&v)[3]) {
    using C = typename CT<T>::t;
    const int M = m.nx / 2;
    if (kx >= M || ky == m.ny / 2 || (kx == 0 && ky == 0)) {
        v[0] = C{T(0), T(0)}; v[1] = v[0]; v[2] = v[0];
        return;
    }
    T qx = T(kx) * m.cx;
    T qy = T(signed_k(ky, m.ny)) * m.cy;
    if constexpr (sizeof(T) == 8) {
        // Gamma zeta = zeta - (t . zeta t) t (x) t with t the unit tangent: a division and some 35 FP64
        // instructions (a root, a division and some 80 in the form below, 40 % of a column pass's FP64 work)
        const T iq = T(1) / (qx * qx + qy * qy), sc = m.inv_n;
        const T t11 = qy * qy * iq, t22 = qx * qx * iq, t12 = qx * qy * iq;   // t = n turned by 90 degrees; t12 = -t1 t2
        const C a = v[0], b = v[1], c = v[2];
        const C s{sc * (t11 * a.x + t22 * b.x - T(2) * t12 * c.x), sc * (t11 * a.y + t22 * b.y - T(2) * t12 * c.y)};
        v[0] = C{sc * a.x - t11 * s.x, sc * a.y - t11 * s.y};
        v[1] = C{sc * b.x - t22 * s.x, sc * b.y - t22 * s.y};
        v[2] = C{sc * c.x + t12 * s.x, sc * c.y + t12 * s.y};
    } else {
        const T inv = rsqrtf(qx * qx + qy * qy);   // 2 ulp, one instruction
        T n1 = qx * inv, n2 = qy * inv;
        T sc = m.inv_n;
        C a = v[0], b = v[1], c = v[2];
        C s1{n1 * a.x + n2 * c.x, n1 * a.y + n2 * c.y};      // zeta n
        C s2{n1 * c.x + n2 * b.x, n1 * c.y + n2 * b.y};
        C t{n1 * s1.x + n2 * s2.x, n1 * s1.y + n2 * s2.y};   // n . zeta n
        T n11 = n1 * n1, n22 = n2 * n2, n12 = n1 * n2;
        v[0] = C{sc * (T(2) * n1 * s1.x - t.x * n11), sc * (T(2) * n1 * s1.y - t.y * n11)};
        v[1] = C{sc * (T(2) * n2 * s2.x - t.x * n22), sc * (T(2) * n2 * s2.y - t.y * n22)};
        v[2] = C{sc * (n1 * s2.x + n2 * s1.x - t.x * n12), sc * (n1 * s2.y + n2 * s1.y - t.y * n12)};
    }
}

// Collocation Laplacian multiplier -|2 pi q|^2 / (nx ny) (Sec. 3.1.2).
template <typename T>
__device__ __forceinline__ void lap_apply(const ModeK<T>& m, int kx, int ky, typename CT<T>::t (&v)[1]) {
    T qx = T(kx) * m.cx;
    T qy = T(signed_k(ky, m.ny)) * m.cy;
    T f = -(qx * qx + qy * qy) * m.inv_n;
    v[0].x *= f;
    v[0].y *= f;
}

}  // namespace pff
