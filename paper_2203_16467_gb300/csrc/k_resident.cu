// k_resident.cu -- the two sub-problem solves of small FP32 grids (up to 2^14 pixels), each solve of
// a problem in one launch of one thread-block cluster (8 or 16 CTAs) that keeps the iteration's
// state on chip.
//
// Why.  At these sizes the kernels of an iteration hold well under a microsecond of work each and
// cost 6-10 us (launch, control block read, load latency, reduction tail).  One load step, per-kernel path
// -> here, us, host calls included: 16^2 1845 -> 528, 64^2 2468 -> 671, 128^2 2953 -> 1092, 64 x 256 3293 ->
// 1516.  At 256^2 the 16 SMs of a cluster no longer keep up with the whole chip (64 problems of 256^2 in
// groups of eight, 40 against 20 ms per load step), hence the limit of 2^14 pixels.
// A cluster has its SMs to itself (at 2^14 pixels a CTA's registers fill one), so the chip runs nine
// clusters of 16 at a time and a group's others queue, while the per-kernel path hardly slows until a launch
// holds some 2^19 pixels.  Groups in one launch, per-kernel -> here, ms: 64^2 64 problems 7.0 -> 6.1, 128 11.4
// -> 11.9; 128^2 16 4.9 -> 3.5, 32 6.6 -> 6.1, 64 10.5 -> 11.9; 64 x 256 16 4.9 -> 4.6, 32 6.6 -> 8.0, 64 10.3 ->
// 15.0.  Groups of one in streams are faster here throughout (64 of 128^2 26.2 -> 13.2).  The number of
// problems still does not choose the path: the two differ in the last bits, and a simulation's result must not
// depend on the grouping of its batch (pff_batch_autotune changes that as it goes).
// (Registers: the 17 warps at 64 x 256 leave 96 a thread, which spills 716 bytes in the mechanics solve and 248
// in the BCCG; the nine warps at 128^2 leave 168, which spills 160 bytes in the mechanics solve.)
// A cluster exchanges through its own shared memory instead:
//   rows     CTA c owns the rows [c RPC, (c+1) RPC), a row per warp (several short rows); the vectors
//            of the iteration (p, r, theta, or p, r, v, R) of its pixels and the constants stay in
//            registers for the whole solve;
//   columns  CTA c owns CPC adjacent mode columns kx of the half spectrum (all components), a column
//            per warp;
//   the forward row FFTs store their modes straight into the column owners' shared memory, the
//   column pass (FFT along y, mode multiplier, inverse) stores its rows straight into the row owners'.
// What bounds it: the chain of dependent exchanges and scalars of an iteration (7300 cycles of a 64^2
// CG iteration, of which the two spectrum exchanges take 1900 and the sums' 1500; at 128^2 the bytes
// of the exchanges too: scattered remote stores move about 6 B per cycle and SM).  Measured on the
// chip: a cluster barrier with stores before it 960 (8 CTAs) to 1480 (16) cycles, a store with
// transaction count (st.async) seen by the receiver after 240; an FP64 add 65, a division 550, a
// square root 600 cycles.  Hence
//   * every exchange is st.async with the bytes counted by an mbarrier of the receiver;
//   * FFTs run within a warp (registers and shuffles, lengths 8 to 256), so no phase needs a block
//     barrier;
//   * one more warp does nothing but the scalars: it sums, sends and receives the partial sums and
//     runs the finalizers, beside the column pass where the iteration allows it.
// An iteration has three exchanges: modes there, rows back, sums (BCCG: six when J v - b is
// evaluated explicitly).
//
// Order of the exchanges.  A CTA sends into a buffer of another only after that one has read the
// buffer's previous contents; and a receiver arms an mbarrier's phase when it waits for it, so that
// bytes that arrive earlier already count for the phase they belong to (the previous one has completed).
//   modes, rows: a CTA that has all its rows knows that every CTA has read its modes (the rows are
//     made of them) and its previous rows (a CTA sends its modes after reading those);
//   sums, slot 0 (p.Ap, p.Jp): sent beside an operator, when all that a CTA knows of the others are the
//     sums it has received; those before it were slot 1's, and each CTA contributed to them after reading
//     slot 0.  The wait for the modes would not do: a CTA without mode columns (1 to 7 of each cluster)
//     waits for none;
//   sums, slot 1 (everything else): sent after an operator, of which each CTA has received all rows,
//     which every CTA made possible after reading slot 1.
// (tests/test_resident_exchanges.py plays this order with late CTAs.)  Every CTA sums the
// same partials in the same order, so all take the same decisions.
//
// Waits are bounded (pff_set_barrier_spin_limit; about two seconds by default).  A CTA whose wait ran
// out goes on to the next block barrier that asks for it (the answer is the barrier's, so all its warps
// leave together), stops sending, and so makes the others' waits run out; a CTA that was sent partial
// results meanwhile learns of it at the end (leave).  Nothing of a solve is stored before that: eps*, v
// and the control block stay as they were, status bit 8 is set, and the kernels that follow in a load
// step leave the state alone.  The cluster barriers at the start and the end are reached by every thread
// once.
//
// Arithmetic: the pixel functions, mode multipliers and finalizers of the per-kernel path; a
// private copy of the control block in each CTA's shared memory takes the finalizers' results and
// rank 0 stores it at the end.  Sums: compensated pairs per thread, double-float within a CTA,
// FP64 across the CTAs in a fixed order.
#include <atomic>

#include "kernels.cuh"
#include "launch.h"

namespace pff {
namespace {

using C = float2;
constexpr int MAXR = 8;                             // values of a reduction
constexpr unsigned FULLW = 0xffffffffu;

// ---------------------------------------------------------------- cluster primitives
__device__ __forceinline__ unsigned s32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
// the address of this CTA's shared-memory location a in CTA `rank` of the cluster
__device__ __forceinline__ unsigned at_rank(unsigned a, unsigned rank) {
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
// stores of 8 bytes whose arrival counts on the mbarrier bar (of the same CTA as a)
__device__ __forceinline__ void send(unsigned a, C v, unsigned bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(a), "f"(v.x),
                 "f"(v.y), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void send(unsigned a, double v, unsigned bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f64 [%0], %1, [%2];" ::"r"(a), "d"(v), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void bar_init(unsigned bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void bar_arm(unsigned bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// has the phase completed: now, and waiting a little for it
__device__ __forceinline__ bool bar_test(unsigned bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool bar_try(unsigned bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// a plain store to the shared memory of a CTA of the cluster
__device__ __forceinline__ void put(unsigned a, int v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned cta_rank() {
    unsigned r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// ---------------------------------------------------------------- geometry
// 16 CTAs from 1024 pixels on (8 below), a warp per row (or per 32 / (nx/2) short rows).
template <int NX, int NY, int NC>
struct RG {
    static constexpr int CS = NX * NY >= 1024 && NY >= 16 ? 16 : 8;
    static constexpr int RPC = NY / CS;                  // rows per CTA
    static constexpr int M = NX / 2, NM = M + 1;         // row FFT length, mode columns
    static constexpr int LR = M < 32 ? M : 32, ER = M / LR;      // lanes and values per lane of a row
    static constexpr int RW = 32 / LR;                   // rows per warp
    static constexpr int W = RPC >= RW ? RPC / RW : 1;   // row warps
    static constexpr int CPC = (NM + CS - 1) / CS;       // mode columns per CTA
    static constexpr int LC = NY < 32 ? NY : 32, EC = NY / LC;   // lanes and values per lane of a column
    static constexpr int CW = 32 / LC;                   // columns per warp
    static constexpr int NT = (W + 1) * 32;              // with the scalar warp
    static constexpr int SPR = NM | 1, SPC = NY + 1;     // odd pitches: strided accesses spread over the banks
    static constexpr int O_KB = NC * RPC * SPR, O_TWC = O_KB + NC * CPC * SPC;
    static constexpr size_t SMEM = (size_t)(O_TWC + NY) * sizeof(C);
    static_assert(NY % CS == 0 && RPC >= 1 && (RPC % RW == 0 || RPC < RW), "whole rows per warp");
};

struct Shared {              // per-CTA scalars
    double red[2][16][MAXR]; // CTA totals of the cluster, by rank (two slots)
    double alpha_d;          // what the scalar warp tells the row warps
    float alpha, beta;
    int stop, full;
    unsigned long long bar[4];   // mbarriers: modes, rows, sums slot 0, sums slot 1
    Ctrl ctrl;
    Desc<float> d;           // the problem's descriptor with ctrl pointing here
    long long spin;          // wait limit in clock cycles
    volatile int dead;       // a wait of this CTA ran out
    volatile int any;        // a wait of some CTA ran out (written before the last cluster barrier)
};
enum { B_MODES = 0, B_ROWS = 1, B_SUM0 = 2, B_SUM1 = 3 };

// Wait for `parity` of an mbarrier; every lane polls, at most s.spin cycles (then s.dead).
__device__ __forceinline__ void await(Shared& s, int which, unsigned parity) {
    const unsigned bar = s32(&s.bar[which]);
    if (bar_test(bar, parity)) return;
    const long long t0 = clock64();
    while (!s.dead) {
        if (clock64() - t0 > s.spin) s.dead = 1;
        else if (bar_try(bar, parity)) return;
    }
}
// A block barrier: has a wait of this CTA run out (the same answer in every thread)?
__device__ __forceinline__ bool sync_dead(const Shared& s) { return __syncthreads_or(s.dead) != 0; }

// ---------------------------------------------------------------- FFTs within a warp
// Stage twiddles of the lane FFT: w[i] for the half-width h = 16 >> i: exp(-pi i (lane mod h) / h) in
// the lanes with bit h set, 1 in the others.
__device__ __forceinline__ void lane_twiddles(const Desc<float>& d, int lane, C (&w)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int h = 16 >> i;
        w[i] = (lane & h) ? d.tw[2 * h + (lane & (h - 1))] : C{1.f, 0.f};
    }
}
// K transforms at once over groups of L lanes, in place; the results are in bit-reversed lane order
// (forward, decimation in frequency) or are taken in it (inverse, unnormalised).
template <int L, int K, bool INV>
__device__ __forceinline__ void lane_fft(C (&v)[K], int lane, const C (&w)[4]) {
#pragma unroll
    for (int q = 0; (1 << q) < L; ++q) {
        const int h = INV ? (1 << q) : (L >> (q + 1));
        const float sg = (lane & h) ? -1.f : 1.f;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            if (INV && h > 1) v[k] = cmulc(v[k], w[h == 2 ? 3 : h == 4 ? 2 : h == 8 ? 1 : 0]);
            const C o{__shfl_xor_sync(FULLW, v[k].x, h), __shfl_xor_sync(FULLW, v[k].y, h)};
            v[k] = C{fmaf(sg, v[k].x, o.x), fmaf(sg, v[k].y, o.y)};
            if (!INV && h > 1) v[k] = cmul(v[k], w[h == 2 ? 3 : h == 4 ? 2 : h == 8 ? 1 : 0]);
        }
    }
}
template <int E, bool INV>
__device__ __forceinline__ void dft_regs(C* u) {
    if constexpr (E == 2) {
        const C a = u[0], b = u[1];
        u[0] = cadd(a, b);
        u[1] = csub(a, b);
    } else if constexpr (E == 4) {
        dft4<C, INV>(u[0], u[1], u[2], u[3]);
    } else if constexpr (E == 8) {
        dft8<C, INV>(*reinterpret_cast<C(*)[8]>(u));
    }
}
// NC transforms of length N = E L: forward from value e of lane l = element e L + l to value k1 of lane
// l = mode k1 + E bitrev(l); the inverse back.  tw[k1 - 1] = exp(-2 pi i l k1 / N).
template <int L, int E, int NC, bool INV>
__device__ __forceinline__ void warp_fft(C (&v)[NC * E], int lane, const C (&w)[4], const C* tw) {
    if constexpr (!INV && E > 1) {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            dft_regs<E, false>(&v[c * E]);
#pragma unroll
            for (int k = 1; k < E; ++k) v[c * E + k] = cmul(v[c * E + k], tw[k - 1]);
        }
    }
    lane_fft<L, NC * E, INV>(v, lane, w);
    if constexpr (INV && E > 1) {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
#pragma unroll
            for (int k = 1; k < E; ++k) v[c * E + k] = cmulc(v[c * E + k], tw[k - 1]);
            dft_regs<E, true>(&v[c * E]);
        }
    }
}
template <int L>
__device__ __forceinline__ int bitrev(int l) { return (int)(__brev((unsigned)l) >> (32 - ilog2(L))); }

// ---------------------------------------------------------------- the exchange phases
// Per-thread constants of a solve.
template <class G>
struct Lane {
    int lane, warp, li, row;          // lane, warp, lane within the row's group, row within the CTA
    bool on;                          // holds pixels
    unsigned rank, rb, kb;            // cluster rank, buffers of this CTA
    C w[4];                           // lane FFT twiddles
    C te[G::ER > 1 ? G::ER - 1 : 1];  // row FFT twiddles across the lanes
    C tn[G::ER];                      // exp(-2 pi i k / NX) of this lane's modes
    unsigned to[G::ER], tb[G::ER];    // where this lane's modes of component 0 go, and their mbarrier
    unsigned to_m, tb_m;              // the same of mode nx/2 (lane 0 of a group)
    int zero;                         // the lane with the conjugate partner of this lane's mode k1 = 0
};

template <int NX, int NY, int NC>
__device__ __forceinline__ void lane_setup(Lane<RG<NX, NY, NC>>& t, const Desc<float>& d, Shared& s, const C* sm) {
    using G = RG<NX, NY, NC>;
    constexpr int L = G::LR, E = G::ER, M = G::M;
    t.lane = threadIdx.x & 31;
    t.warp = threadIdx.x >> 5;
    t.li = t.lane & (L - 1);
    t.row = t.warp * G::RW + t.lane / L;
    t.on = t.warp < G::W && t.row < G::RPC;
    t.rank = cta_rank();
    t.rb = s32(sm);
    t.kb = s32(sm + G::O_KB);
    lane_twiddles(d, t.lane, t.w);
    const int br = bitrev<L>(t.li);
    t.zero = (t.lane & ~(L - 1)) | bitrev<L>((L - br) & (L - 1));
    const int y = (int)t.rank * G::RPC + t.row;
    const unsigned bar = s32(&s.bar[B_MODES]);
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int k = e + E * br;
        if (e > 0) t.te[e - 1] = d.tw[M + t.li * e];
        t.tn[e] = d.tw[NX + k];
        t.to[e] = at_rank(t.kb + (unsigned)(((k % G::CPC) * G::SPC + y) * sizeof(C)), k / G::CPC);
        t.tb[e] = at_rank(bar, k / G::CPC);
    }
    t.to_m = at_rank(t.kb + (unsigned)(((M % G::CPC) * G::SPC + y) * sizeof(C)), M / G::CPC);
    t.tb_m = at_rank(bar, M / G::CPC);
}

// Forward row FFTs of the real pixels z[c E + e] = (x, x + 1), x = 2 (e L + li), and the modes to the
// column owners.
template <class G, int NC>
__device__ __forceinline__ void rows_forward(const Lane<G>& t, C (&z)[NC * G::ER]) {
    constexpr int L = G::LR, E = G::ER;
    constexpr unsigned CST = G::CPC * G::SPC * sizeof(C);   // component stride of the column buffer
    warp_fft<L, E, NC, false>(z, t.lane, t.w, t.te);
    // split of the half-length complex FFT: X[k] = e + w o with z[M-k] from its lane
#pragma unroll
    for (int c = 0; c < NC; ++c) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const C zk = z[c * E + e];
            const C zp = z[c * E + (E - e) % E];
            const int src = e == 0 ? t.zero : (t.lane ^ (L - 1));
            const C zm{__shfl_sync(FULLW, zp.x, src), -__shfl_sync(FULLW, zp.y, src)};
            const C ev{0.5f * (zk.x + zm.x), 0.5f * (zk.y + zm.y)};
            const C od{0.5f * (zk.y - zm.y), -0.5f * (zk.x - zm.x)};
            const C tk = cmul(t.tn[e], od);
            if (t.on) {
                send(t.to[e] + c * CST, cadd(ev, tk), t.tb[e]);
                if (e == 0 && t.li == 0) send(t.to_m + c * CST, C{ev.x - tk.x, tk.y - ev.y}, t.tb_m);
            }
        }
    }
}

// Column pass of this CTA's mode columns (one per warp and round) and the rows back to their owners.
// mid(): run once per warp, as soon as OP has seen its last modes.
template <class G, int NX, int NY, int NC, class OP, class MID>
__device__ __forceinline__ void columns(const Lane<G>& t, Shared& s, const C* sm, const ModeK<float>& mk, Acc<float>* acc,
                                        MID mid) {
    constexpr int L = G::LC, E = G::EC;
    const C* kb = sm + G::O_KB;
    const C* twc = sm + G::O_TWC;
    const int l = t.lane & (L - 1), br = bitrev<L>(l);
    C te[E > 1 ? E - 1 : 1];
#pragma unroll
    for (int k = 1; k < E; ++k) te[k - 1] = twc[l * k];
    const unsigned bar = s32(&s.bar[B_ROWS]);
    if (t.warp * G::CW >= G::CPC) mid();   // no columns
#pragma unroll 1
    for (int j0 = t.warp * G::CW; j0 < G::CPC; j0 += G::W * G::CW) {
        const int j = j0 + t.lane / L, kx = (int)t.rank * G::CPC + j;
        const bool on = j < G::CPC && kx <= G::M;
        C u[NC * E];
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
            for (int e = 0; e < E; ++e)
                u[c * E + e] = on ? kb[(c * G::CPC + j) * G::SPC + e * L + l] : C{0.f, 0.f};
        warp_fft<L, E, NC, false>(u, t.lane, t.w, te);
#pragma unroll
        for (int k = 0; k < E; ++k) {
            const int ky = k + E * br;
            C v[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) v[c] = u[c * E + k];
            if constexpr (ColNR<OP>::value > 0) OP::accum(mk, kx, ky, v, acc);
            OP::apply(mk, kx, ky, v);
#pragma unroll
            for (int c = 0; c < NC; ++c) u[c * E + k] = v[c];
        }
        if (j0 + G::W * G::CW >= G::CPC) mid();
        warp_fft<L, E, NC, true>(u, t.lane, t.w, te);
        if (on) {
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int y = e * L + l;
                const unsigned rk = (unsigned)(y / G::RPC);
                const unsigned a = at_rank(t.rb + (unsigned)(((y % G::RPC) * G::SPR + kx) * sizeof(C)), rk);
                const unsigned b = at_rank(bar, rk);
#pragma unroll
                for (int c = 0; c < NC; ++c) send(a + (unsigned)(c * G::RPC * G::SPR * sizeof(C)), u[c * E + e], b);
            }
        }
    }
}

// Inverse row FFTs from the half spectra in this CTA's row buffer to the pixels.
template <class G, int NC>
__device__ __forceinline__ void rows_inverse(const Lane<G>& t, const C* rb, C (&z)[NC * G::ER]) {
    constexpr int L = G::LR, E = G::ER, M = G::M;
    const int br = bitrev<L>(t.li), row = t.row < G::RPC ? t.row : 0;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        const C* x = rb + (c * G::RPC + row) * G::SPR;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int k = e + E * br;
            C xk = x[k], xm = x[M - k];
            if (k == 0) { xk.y = 0.f; xm.y = 0.f; }
            xm.y = -xm.y;
            const C A = cadd(xk, xm);
            const C B = cmulc(csub(xk, xm), t.tn[e]);
            z[c * E + e] = C{A.x - B.y, A.y + B.x};
        }
    }
    warp_fft<L, E, NC, true>(z, t.lane, t.w, t.te);
}

// The operator F^-1 M F on the pixels z (row warps); par: parity of the two mbarriers' next phases.
template <int NX, int NY, int NC, class OP, class MID>
__device__ __forceinline__ void operate(const Lane<RG<NX, NY, NC>>& t, Shared& s, const C* sm, const ModeK<float>& mk,
                                        C (&z)[NC * RG<NX, NY, NC>::ER], unsigned& par, Acc<float>* acc, MID mid) {
    using G = RG<NX, NY, NC>;
    rows_forward<G, NC>(t, z);
    // columns this CTA owns (the last CTAs may own fewer, or none)
    const int own = max(0, min(G::CPC, G::NM - (int)t.rank * G::CPC));
    if (threadIdx.x == 0) {
        bar_arm(s32(&s.bar[B_MODES]), (unsigned)(own * NC * NY * sizeof(C)));
        bar_arm(s32(&s.bar[B_ROWS]), (unsigned)(NC * G::RPC * G::NM * sizeof(C)));
    }
    await(s, B_MODES, par);
    columns<G, NX, NY, NC, OP>(t, s, sm, mk, acc, mid);
    await(s, B_ROWS, par);
    par ^= 1u;
    rows_inverse<G, NC>(t, sm, z);
}

// ---------------------------------------------------------------- sums
__device__ __forceinline__ DF warp_sum(DF x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = df_add(x, RedOps<DF>::shfl(x, o));
    return x;
}
// total of value k of this CTA to slot `slot` of every CTA (a whole warp; x valid in lane 0)
template <int CS>
__device__ __forceinline__ void send_sum(Shared& s, int slot, int k, DF x, unsigned rank, int lane) {
    x.hi = __shfl_sync(FULLW, x.hi, 0);
    x.lo = __shfl_sync(FULLW, x.lo, 0);
    if (lane < CS)
        send(at_rank(s32(&s.red[slot][rank][k]), lane), RedOps<DF>::total(x), at_rank(s32(&s.bar[B_SUM0 + slot]), lane));
}
__device__ __forceinline__ double lane_add(double x, int o) { return x + __shfl_xor_sync(FULLW, x, o); }
// Cluster total of one value in FP64, in every lane of the scalar warp.
template <int CS>
__device__ __forceinline__ double take_one(Shared& s, int slot, unsigned parity, int lane) {
    if (lane == 0) bar_arm(s32(&s.bar[B_SUM0 + slot]), (unsigned)(CS * sizeof(double)));
    __syncwarp();
    await(s, B_SUM0 + slot, parity);
    double x = s.red[slot][lane & (CS - 1)][0];
#pragma unroll
    for (int o = 1; o < CS; o *= 2) x = lane_add(x, o);
    return x;
}
// Cluster totals of NR values: value k in the lanes 4 k .. 4 k + 3.
template <int NR, int CS>
__device__ __forceinline__ double take_many(Shared& s, int slot, unsigned parity, int lane) {
    if (lane == 0) bar_arm(s32(&s.bar[B_SUM0 + slot]), (unsigned)(NR * CS * sizeof(double)));
    __syncwarp();
    await(s, B_SUM0 + slot, parity);
    const int k = lane >> 2, g = lane & 3;
    double x = 0.0;
    if (k < NR) {
        x = s.red[slot][g * (CS / 4)][k];
#pragma unroll
        for (int q = 1; q < CS / 4; ++q) x += s.red[slot][g * (CS / 4) + q][k];
    }
    return lane_add(lane_add(x, 1), 2);
}
// This lane's share (entries lane, lane + 32, ...) of a value that every row thread stored in sh.
template <int W>
__device__ __forceinline__ DF lane_share(const DF* sh, int lane) {
    DF x[W];
#pragma unroll
    for (int j = 0; j < W; ++j) x[j] = sh[32 * j + lane];
#pragma unroll
    for (int n = 1; n < W; n *= 2)
#pragma unroll
        for (int j = 0; j + n < W; j += 2 * n) x[j] = df_add(x[j], x[j + n]);
    return x[0];
}
// A single value that every row thread stored in sh (before a barrier): the scalar warp sums it.
template <int W, int CS>
__device__ __forceinline__ double one_sum(Shared& s, const DF* sh, int slot, unsigned parity, unsigned rank, int lane) {
    send_sum<CS>(s, slot, 0, warp_sum(lane_share<W>(sh, lane)), rank, lane);
    return take_one<CS>(s, slot, parity, lane);
}
// x <= y of non-negative doubles (false for a NaN in either), without the FP64 pipe
__device__ __forceinline__ bool le_bits(double x, double y) {
    const unsigned long long a = (unsigned long long)__double_as_longlong(x), b = (unsigned long long)__double_as_longlong(y);
    return a <= b && b <= 0x7ff0000000000000ull;
}
// NR values, value k of every row thread in sh[k 32 W ...] (before a barrier): each warp sums some of them.
template <int NR, int W, int CS>
__device__ __forceinline__ void many_sums(Shared& s, const DF* sh, int slot, unsigned rank, int warp, int lane) {
    constexpr int ROUNDS = (NR + W) / (W + 1);
    DF x[ROUNDS];
#pragma unroll
    for (int u = 0; u < ROUNDS; ++u) {   // a warp's values together: their chains overlap
        const int k = warp + u * (W + 1);
        x[u] = warp_sum(lane_share<W>(sh + (k < NR ? k : 0) * W * 32, lane));
    }
#pragma unroll
    for (int u = 0; u < ROUNDS; ++u) {
        const int k = warp + u * (W + 1);
        if (k < NR) send_sum<CS>(s, slot, k, x[u], rank, lane);
    }
}
template <int NT>
__device__ __forceinline__ void scalar_arrive() { asm volatile("bar.arrive 1, %0;" ::"n"(NT) : "memory"); }
template <int NT>
__device__ __forceinline__ void scalar_join() { asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory"); }

__device__ __forceinline__ void init(Shared& s, long long spin) {   // one thread, before the cluster's start
    s.spin = spin;
    s.dead = 0;
    s.any = 0;
    for (int b = 0; b < 4; ++b) bar_init(s32(&s.bar[b]));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// Control block, descriptor, column twiddles; mbarriers; then the cluster's start.
template <class G, int NY>
__device__ __forceinline__ void stage(const Desc<float>& d, Shared& s, C* sm, long long spin) {
    const int* src = reinterpret_cast<const int*>(d.ctrl);
    int* dst = reinterpret_cast<int*>(&s.ctrl);
    for (int i = threadIdx.x; i < (int)(sizeof(Ctrl) / 4); i += G::NT) dst[i] = __ldcg(src + i);
    const int* sd = reinterpret_cast<const int*>(&d);
    int* dd = reinterpret_cast<int*>(&s.d);
    for (int i = threadIdx.x; i < (int)(sizeof(Desc<float>) / 4); i += G::NT) dd[i] = sd[i];
    for (int i = threadIdx.x; i < NY; i += G::NT) sm[G::O_TWC + i] = d.tw[NY + i];
    if (threadIdx.x == 0) init(s, spin);
    __syncthreads();
    if (threadIdx.x == 0) s.d.ctrl = &s.ctrl;
    __syncthreads();
    cluster_sync_all();
}

// The cluster's end: true when no wait of any CTA ran out.  Otherwise what is still on its way to a CTA
// gets time to arrive before that one exits.
template <int CS>
__device__ __forceinline__ bool finished(Shared& s) {
    __syncthreads();   // no wait of this CTA from here on
    if (s.dead && threadIdx.x < CS) put(at_rank(s32((const void*)&s.any), threadIdx.x), 1);
    cluster_sync_all();
    if (!s.any) return true;
    const long long t0 = clock64();
    while (clock64() - t0 < 1000000) {}
    return false;
}
// ... and the control block back (rank 0), or status bit 8 alone.
template <class G>
__device__ __forceinline__ bool leave(const Desc<float>& d, Shared& s, unsigned rank) {
    if (!finished<G::CS>(s)) {
        if (rank == 0 && threadIdx.x == 0) atomicOr(&d.ctrl->status, 8);
        return false;
    }
    if (rank == 0) {
        const int* src = reinterpret_cast<const int*>(&s.ctrl);
        int* dst = reinterpret_cast<int*>(d.ctrl);
        for (int i = threadIdx.x; i < (int)(sizeof(Ctrl) / 4); i += G::NT) dst[i] = src[i];
    }
    return true;
}

// ---------------------------------------------------------------- mechanics (Sec. 3.1.1)
template <int NX, int NY>
__global__ void __launch_bounds__(RG<NX, NY, 3>::NT, 1) k_res_mech(const Desc<float>* __restrict__ descs, long long spin) {
    using G = RG<NX, NY, 3>;
    constexpr int E = G::ER, PP = 2 * E, NT = G::NT, CS = G::CS, W = G::W;
    const Desc<float>& d = descs[blockIdx.y];
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ Shared s;
    __shared__ DF sh[W * 32];
    C* sm = reinterpret_cast<C*>(smem_raw);
    stage<G, NY>(d, s, sm, spin);
    Lane<G> t;
    lane_setup<NX, NY, 3>(t, d, s, sm);
    const ModeK<float> mk(s.d);
    const LameC<float> lm(s.d);
    const int split = s.d.k.split;
    const bool linear = contact_of(split) == ISOTROPIC, scalar = t.warp == W;
    const float eb[3] = {(float)s.ctrl.eps_bar[0], (float)s.ctrl.eps_bar[1], (float)s.ctrl.eps_bar[2]};
    const unsigned pix = (t.rank * G::RPC + t.row) * NX + 2 * t.li;   // first pixel pair of this lane
    float p[PP][3], r[PP][3], th[PP][3], ep[PP][3], h[PP], Em[PP];
#pragma unroll
    for (int q = 0; q < PP; ++q) {
        const unsigned i = pix + (q >> 1) * 2 * G::LR + (q & 1);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            p[q][k] = r[q][k] = th[q][k] = 0.f;
            ep[q][k] = t.on ? d.eps[k][i] : 0.f;
        }
        h[q] = t.on ? hdeg(d.phi[i]) : 1.f;
        Em[q] = t.on ? d.E[i] : 1.f;
    }
    unsigned par = 0, p0 = 0, p1 = 0;   // parities: modes and rows, sums slot 0, sums slot 1
    // The scalar warp's state (the same in its lanes): FNewtonOut, FCgIn and FCgOut with norms compared
    // by their squares, the divisions off the chain of the iteration, and no control block between.
    double target = 0.0, target2 = 0.0, cg2 = 0.0, R2 = 0.0, rr = 0.0;
    Recip rr_inv{0.0, 0.0, 1.0};
    int cg_it = 0, cg_total = 0, newton_it = 0, status = 0;
    if (scalar) {
        const Consts& k = s.d.k;
        const double* e = s.ctrl.eps_bar;
        const double tr = e[0] + e[1];
        const double s0 = k.lam_c * tr + 2.0 * k.mu_c * e[0], s1 = k.lam_c * tr + 2.0 * k.mu_c * e[1], s2 = 2.0 * k.mu_c * e[2];
        target = k.mech_tol * sqrt(s.ctrl.sumE2) * sqrt(s0 * s0 + s1 * s1 + 2.0 * s2 * s2);
        target2 = target * target;
    }
    C z[3 * E];
    bool fold = false, dead = false;
    for (;; fold = true) {                   // Newton rounds
        if (fold) {
#pragma unroll
            for (int q = 0; q < PP; ++q)
#pragma unroll
                for (int k = 0; k < 3; ++k) ep[q][k] += th[q][k];
        }
        if (fold && linear) break;   // a linear model takes one Newton step: folded, done
        if (!scalar) {
#pragma unroll
            for (int q = 0; q < PP; ++q) {
                float sg[3];
                stress(split, eb[0] + ep[q][0], eb[1] + ep[q][1], eb[2] + ep[q][2], h[q], lm.lc * Em[q], lm.mc * Em[q], sg);
#pragma unroll
                for (int c = 0; c < 3; ++c) (q & 1 ? z[c * E + (q >> 1)].y : z[c * E + (q >> 1)].x) = sg[c];
            }
            operate<NX, NY, 3, FColGammaCG>(t, s, sm, mk, z, par, nullptr, [] {});
            Acc<float> acc;
            if (t.on) {
#pragma unroll
                for (int q = 0; q < PP; ++q) {
                    float v[3];
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        v[c] = q & 1 ? z[c * E + (q >> 1)].y : z[c * E + (q >> 1)].x;
                        r[q][c] = p[q][c] = -v[c];
                        th[q][c] = 0.f;
                    }
                    wdot(acc, v[0], v[1], v[2], v[0], v[1], v[2]);
                }
            }
            sh[threadIdx.x] = acc.df();
        }
        __syncthreads();
        if (scalar) {
            R2 = one_sum<W, CS>(s, sh, 1, p1, t.rank, t.lane);
            p1 ^= 1u;
            const bool conv = le_bits(R2, target2), stop = conv || newton_it >= s.d.k.max_newton;
            if (stop) {
                if (!conv) status |= 1;
            } else {
                const double rt = s.d.k.mech_cg_rtol;
                cg2 = linear ? target2 : fmax(target2, rt * rt * R2);
                rr = R2;
                cg_it = 0;
                ++newton_it;
            }
            if (t.lane == 0) s.stop = stop;
        }
        dead = sync_dead(s);
        if (s.stop || dead) break;     // Newton stopping test (or the round limit)
        bool first = true;
        do {                                // CG iterations
            if (!scalar) {
                const float beta = s.beta;
                Acc<float> acc;
#pragma unroll
                for (int q = 0; q < PP; ++q) {
                    float v[3];
                    if (!first) {
#pragma unroll
                        for (int k = 0; k < 3; ++k) p[q][k] = r[q][k] + beta * p[q][k];
                    }
                    tangent(split, eb[0] + ep[q][0], eb[1] + ep[q][1], eb[2] + ep[q][2], h[q], lm.lc * Em[q], lm.mc * Em[q],
                            p[q][0], p[q][1], p[q][2], v);
                    wdot(acc, p[q][0], p[q][1], p[q][2], v[0], v[1], v[2]);
#pragma unroll
                    for (int c = 0; c < 3; ++c) (q & 1 ? z[c * E + (q >> 1)].y : z[c * E + (q >> 1)].x) = v[c];
                }
                sh[threadIdx.x] = t.on ? acc.df() : DF{0.f, 0.f};
                scalar_arrive<NT>();
                operate<NX, NY, 3, FColGammaCG>(t, s, sm, mk, z, par, nullptr, [] {});
            } else {                        // alpha, beside the operator
                scalar_join<NT>();
                const double pAp = one_sum<W, CS>(s, sh, 0, p0, t.rank, t.lane);
                p0 ^= 1u;
                const bool go_on = pAp > 0.0;
                rr_inv = recip(rr);
                const float alpha = go_on ? (float)(rr / pAp) : 0.f;
                if (t.lane == 0) {
                    s.alpha = alpha;
                    s.stop = !go_on;
                }
            }
            first = false;
            dead = sync_dead(s);
            if (s.stop || dead) break;      // p.Ap <= 0: no update
            if (!scalar) {
                const float alpha = s.alpha;
                Acc<float> acc;
#pragma unroll
                for (int q = 0; q < PP; ++q) {
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        th[q][k] += alpha * p[q][k];
                        r[q][k] -= alpha * (q & 1 ? z[k * E + (q >> 1)].y : z[k * E + (q >> 1)].x);
                    }
                    wdot(acc, r[q][0], r[q][1], r[q][2], r[q][0], r[q][1], r[q][2]);
                }
                sh[threadIdx.x] = t.on ? acc.df() : DF{0.f, 0.f};
            }
            __syncthreads();
            if (scalar) {
                rr = one_sum<W, CS>(s, sh, 1, p1, t.rank, t.lane);
                p1 ^= 1u;
                const float beta = (float)quotient(rr, rr_inv);
                ++cg_it;
                ++cg_total;
                const bool conv = le_bits(rr, cg2), stop = conv || cg_it >= s.d.k.max_cg;
                if (stop && !conv) status |= 1;
                if (t.lane == 0) {
                    s.beta = beta;
                    s.stop = stop;
                }
            }
            dead = sync_dead(s);
        } while (!s.stop && !dead);
        if (dead) break;
    }
    __syncthreads();
    if (scalar && t.lane == 0) {    // results, and the flags as the per-kernel path leaves them
        Ctrl& c = s.ctrl;
        c.mech_target = target;
        c.R2 = R2;
        c.rr = rr;
        c.newton_it = newton_it;
        c.cg_it = cg_it;
        c.cg_total += cg_total;
        c.status |= status;
        c.nd_a = c.nd_b = c.cg_a = c.cg_b = 1;
        c.needs_fold = 0;
    }
    if (leave<G>(d, s, t.rank) && fold && t.on) {
#pragma unroll
        for (int q = 0; q < PP; ++q) {
            const unsigned i = pix + (q >> 1) * 2 * G::LR + (q & 1);
#pragma unroll
            for (int k = 0; k < 3; ++k) d.eps[k][i] = ep[q][k];
        }
    }
}

// ---------------------------------------------------------------- phase field (Algorithm 1)
// From the start that FPfInit leaves: v, r, p, a, b, v_con, R and the flags.
template <int NX, int NY>
__global__ void __launch_bounds__(RG<NX, NY, 1>::NT, 1) k_res_bccg(const Desc<float>* __restrict__ descs, long long spin) {
    using G = RG<NX, NY, 1>;
    constexpr int E = G::ER, PP = 2 * E, NT = G::NT, CS = G::CS, W = G::W;
    const Desc<float>& d = descs[blockIdx.y];
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ Shared s;
    __shared__ DF sh[MAXR * W * 32];
    C* sm = reinterpret_cast<C*>(smem_raw);
    stage<G, NY>(d, s, sm, spin);
    Lane<G> t;
    lane_setup<NX, NY, 1>(t, d, s, sm);
    const ModeK<float> mk(s.d);
    const float kappa = (float)s.d.k.kappa;
    const bool scalar = t.warp == W;
    const unsigned pix = (t.rank * G::RPC + t.row) * NX + 2 * t.li;
    float p[PP], r[PP], ro[PP], v[PP], R[PP], a[PP], b[PP], vc[PP];
    uint8_t fl[PP];
#pragma unroll
    for (int q = 0; q < PP; ++q) {
        const unsigned i = pix + (q >> 1) * 2 * G::LR + (q & 1);
        v[q] = t.on ? d.th[0][i] : 0.f;
        r[q] = t.on ? d.th[1][i] : 0.f;
        p[q] = t.on ? d.th[2][i] : 0.f;
        a[q] = t.on ? d.r[0][i] : 0.f;
        b[q] = t.on ? d.r[1][i] : 0.f;
        vc[q] = t.on ? d.r[2][i] : 0.f;
        R[q] = t.on ? d.lap[i] : 0.f;
        fl[q] = t.on ? d.flags[i] : 0;
        ro[q] = 0.f;
    }
    unsigned par = 0, p0 = 0, p1 = 0;
    // The scalar warp's state (the same in its lanes): FColLapPFQ's and FPfSlotOut's finalizers with
    // the next step's flags and beta first and everything else after the row warps have gone on.
    double target2 = 0.0, kin = 0.0, pap = 0.0, rp = 0.0, beta = 0.0, rr = 0.0, best = 0.0, last = 0.0, nact = 0.0;
    Recip irp{0.0, 0.0, 1.0};   // of -rp
    int it = 0, best_it = 0, since_full = 0, full_iters = 0, clamp_iters = 0, status = 0;
    bool confirm = false, broke = false;
    if (scalar) {
        const Ctrl& c = s.ctrl;
        target2 = c.pf_target * c.pf_target;
        kin = s.d.k.kappa * s.d.k.inv_n;
        pap = c.pf_pap;
        rp = c.pf_rp;
        irp = recip(-rp);
        rr = c.pf_rr;
        best = last = rr;
        if (t.lane == 0) s.stop = c.pf_b;
    }
    __syncthreads();
    // sums 4 .. 7 (or 3 .. 6) of a pass over the pixels -> sum a p'^2 and r'.p' of the next direction
    auto next_dir = [&](double x, int k0) {
        const double S0 = __shfl_sync(FULLW, x, 4 * k0), S1 = __shfl_sync(FULLW, x, 4 * k0 + 4),
                     S2 = __shfl_sync(FULLW, x, 4 * k0 + 8), S3 = __shfl_sync(FULLW, x, 4 * k0 + 12);
        pap = S0 - 2.0 * beta * S1 + beta * beta * S2;
        rp = -rr + beta * S3;
        irp = recip(-rp);
    };
    C z[E];
    bool dead = false;
    for (bool first = true; !s.stop && !dead; first = false) {
        if (!scalar) {
            if (!first) {   // p = -r + beta p, zero on the active set
                const float bt = s.beta;
#pragma unroll
                for (int q = 0; q < PP; ++q) p[q] = (fl[q] & 2) ? 0.f : -r[q] + bt * p[q];
            }
#pragma unroll
            for (int e = 0; e < E; ++e) z[e] = C{p[2 * e], p[2 * e + 1]};
            Acc<float> acc;
            operate<NX, NY, 1, FColLapPFQ>(t, s, sm, mk, z, par, &acc, [&] {
                sh[threadIdx.x] = acc.df();
                scalar_arrive<NT>();
            });
        } else {                      // alpha, beside the rows' way back
            scalar_join<NT>();
            const double pJp = fma(kin, one_sum<W, CS>(s, sh, 0, p0, t.rank, t.lane), pap);
            p0 ^= 1u;
            broke = !(pJp > 0.0);
            const double al = broke ? 0.0 : -rp / pJp;
            if (t.lane == 0) {
                s.alpha_d = al;
                s.alpha = (float)al;
            }
        }
        __syncthreads();
        if (!scalar) {
            const double alpha_d = s.alpha_d;
            const float alpha = s.alpha;
            Acc<float> acc[8];
#pragma unroll
            for (int q = 0; q < PP; ++q) {
                float x, Rn, rn;
                ro[q] = r[q];
                fl[q] = pf_iterate_px(kappa, alpha, alpha_d, p[q], a[q], v[q], vc[q], R[q], r[q],
                                      q & 1 ? z[q >> 1].y : z[q >> 1].x, x, Rn, rn, acc);
                v[q] = x;
                R[q] = Rn;
                r[q] = rn;
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) sh[k * W * 32 + threadIdx.x] = t.on ? acc[k].df() : DF{0.f, 0.f};
        }
        __syncthreads();
        many_sums<8, W, CS>(s, sh, 1, t.rank, t.warp, t.lane);
        double x8 = 0.0;
        bool full_now = false;
        if (scalar) {
            x8 = take_many<8, CS>(s, 1, p1, t.lane);
            p1 ^= 1u;
            const double r2 = __shfl_sync(FULLW, x8, 4), rro = __shfl_sync(FULLW, x8, 8);
            const bool clamped = __double_as_longlong(__shfl_sync(FULLW, x8, 0)) > 0;
            const bool rec_conv = le_bits(r2, target2);
            full_now = clamped || rec_conv || since_full + 1 >= PF_REFRESH;
            bool stop = false;
            if (!full_now) {
                beta = quotient(r2 - rro, irp);
                rr = r2;
                ++it;
                ++since_full;
                const bool stalled = it - best_it >= PF_STALL;
                stop = stalled || it >= s.d.k.max_pf || broke;
                if (stop && !stalled && !broke) status |= 2;
            }
            const float bt = (float)beta;
            if (t.lane == 0) {
                s.beta = bt;
                s.full = full_now;
                s.stop = stop;
            }
            clamp_iters += clamped;
            confirm = rec_conv;
        }
        dead = sync_dead(s);
        if (!s.full || dead) {
            if (scalar) {   // beside the next direction's way to the columns
                nact = __shfl_sync(FULLW, x8, 12);
                next_dir(x8, 4);
            }
            continue;
        }
        // explicit R = J v - b (some value was clamped, the refresh interval, or a confirmation)
        if (!scalar) {
#pragma unroll
            for (int e = 0; e < E; ++e) z[e] = C{v[2 * e], v[2 * e + 1]};
            operate<NX, NY, 1, FColLapPFFull>(t, s, sm, mk, z, par, nullptr, [] {});
            Acc<float> acc[7];
#pragma unroll
            for (int q = 0; q < PP; ++q) {
                float Rn, rn;
                fl[q] = pf_explicit_px(kappa, s.d.k.kappa, ro[q], v[q], a[q], b[q], p[q], (fl[q] & 1) != 0,
                                       q & 1 ? z[q >> 1].y : z[q >> 1].x, Rn, rn, acc);
                R[q] = Rn;
                r[q] = rn;
            }
#pragma unroll
            for (int k = 0; k < 7; ++k) sh[k * W * 32 + threadIdx.x] = t.on ? acc[k].df() : DF{0.f, 0.f};
        }
        __syncthreads();
        many_sums<7, W, CS>(s, sh, 1, t.rank, t.warp, t.lane);
        if (scalar) {
            x8 = take_many<7, CS>(s, 1, p1, t.lane);
            p1 ^= 1u;
            rr = __shfl_sync(FULLW, x8, 0);
            beta = quotient(rr - __shfl_sync(FULLW, x8, 4), irp);
            ++it;
            ++full_iters;
            since_full = 0;
            // FP32: a confirming evaluation that improved little on the previous explicit residual has
            // reached the rounding level of J v - b
            const bool conv = le_bits(rr, target2) || (confirm && rr >= 0.25 * last);
            if (rr < best) { best = rr; best_it = it; }
            const bool stalled = it - best_it >= PF_STALL;
            const bool stop = conv || stalled || it >= s.d.k.max_pf || broke;
            if (stop && !conv && !stalled && !broke) status |= 2;
            const float bt = (float)beta;
            if (t.lane == 0) {
                s.beta = bt;
                s.stop = stop;
            }
        }
        dead = sync_dead(s);
        if (scalar) {
            last = rr;
            nact = __shfl_sync(FULLW, x8, 8);
            next_dir(x8, 3);
        }
    }
    if (scalar && t.lane == 0) {
        Ctrl& c = s.ctrl;
        c.pf_rr = rr;
        c.pf_it = it;
        c.pf_beta = beta;
        c.pf_rp = rp;
        c.pf_pap = pap;
        c.n_active = (int)nact;
        c.pf_clamp_iters += clamp_iters;
        c.pf_full_iters = full_iters;
        c.pf_break = broke;
        c.status |= status;
        c.pf_a = c.pf_b = 1;
    }
    if (leave<G>(d, s, t.rank) && t.on) {
#pragma unroll
        for (int q = 0; q < PP; ++q) {
            const unsigned i = pix + (q >> 1) * 2 * G::LR + (q & 1);
            d.th[0][i] = v[q];
            d.flags[i] = fl[q];
        }
    }
}

// ---------------------------------------------------------------- one Laplacian
// out = nabla^2 in of one field, in = d.r[0], out = d.q[0] (the allocation-free entry point): the
// operator alone, without the scalar warp.  A wait that runs out in any CTA leaves NaN in all of them, never
// a wrong field.
// Bound by its two exchanges and the launch: everything that does not depend on the input (twiddles,
// lane constants, the cluster's start) runs before the wait for the stream's previous work.  The rate of a
// row of calls, whose prologues overlap, three passes -> one launch: 16^2 6.1 -> 2.6 us, 64^2 5.9 -> 2.7, 128^2
// 6.8 -> 3.7, 256 x 64 6.6 -> 4.0.  One call that is waited for (host call, launch and wait included): 16^2 14.2
// -> 12.1 us, 64^2 15.5 -> 12.9, 128^2 16.8 -> 14.2, 256 x 64 16.7 -> 14.5.
template <int NX, int NY>
__global__ void __launch_bounds__(RG<NX, NY, 1>::W * 32, 1) k_res_lap(const __grid_constant__ Desc<float> d, long long spin) {
    using G = RG<NX, NY, 1>;
    constexpr int E = G::ER;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ Shared s;
    C* sm = reinterpret_cast<C*>(smem_raw);
    if (threadIdx.x == 0) init(s, spin);
    Lane<G> t;
    lane_setup<NX, NY, 1>(t, d, s, sm);
    const unsigned pix = (t.rank * G::RPC + t.row) * NX + 2 * t.li;
    C z[E];
    for (int i = threadIdx.x; i < NY; i += G::W * 32) sm[G::O_TWC + i] = d.tw[NY + i];
    const ModeK<float> mk(d);
    __syncthreads();
    cluster_sync_all();
    pdl_enter();   // the stream's previous work is complete from here on
#pragma unroll
    for (int e = 0; e < E; ++e)
        z[e] = t.on ? *reinterpret_cast<const C*>(d.r[0] + pix + e * 2 * G::LR) : C{0.f, 0.f};
    unsigned par = 0;
    operate<NX, NY, 1, FColLapPlain>(t, s, sm, mk, z, par, nullptr, [] {});
    const bool ok = finished<G::CS>(s);
    if (t.on) {
#pragma unroll
        for (int e = 0; e < E; ++e)
            *reinterpret_cast<C*>(d.q[0] + pix + e * 2 * G::LR) = ok ? z[e] : C{NAN, NAN};
    }
}

// ---------------------------------------------------------------- launch
// One cluster of CS CTAs per problem.  cudaErrorNotSupported where the device cannot host the
// cluster (the caller then runs the per-kernel path).  pdl: may be scheduled while the stream's
// previous kernel runs.
constexpr int MAX_DEVICES = 64;
enum : signed char { UNKNOWN = 0, RUNS = 1, REFUSED = 2 };
template <typename A>
cudaError_t go(void (*fn)(A, long long), std::atomic<signed char>* known, int cs, int nt, size_t smem, const A& d, int np,
               cudaStream_t st, bool pdl = false) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) return cudaErrorNotSupported;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cs, np);
    cfg.blockDim = dim3(nt);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (known[dev] == UNKNOWN) {   // two threads may both ask: the answers agree
        int n = 0;
        const bool ok = cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) ==
                            cudaSuccess &&
                        (cs <= 8 || cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeNonPortableClusterSizeAllowed,
                                                         1) == cudaSuccess) &&
                        cudaOccupancyMaxActiveClusters(&n, (const void*)fn, &cfg) == cudaSuccess && n >= 1;
        if (!ok) cudaGetLastError();
        known[dev] = ok ? RUNS : REFUSED;
    }
    if (known[dev] == REFUSED) return cudaErrorNotSupported;
    cfg.numAttrs = pdl ? 2 : 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, fn, d, barrier_spin_limit());
    if (e == cudaSuccess) count_launch();
    return e;
}

#if PFF_RESIDENT == 2
using Arg = Desc<float>;
#else
using Arg = const Desc<float>*;
#endif

template <int NX, int NY>
cudaError_t go_size(const Arg& d, int np, cudaStream_t st) {
    if constexpr (NX * NY <= RESIDENT_PIXELS) {
        static std::atomic<signed char> known[MAX_DEVICES];   // per device: can the cluster run
#if PFF_RESIDENT == 0
        using G = RG<NX, NY, 3>;
        return go<Arg>(k_res_mech<NX, NY>, known, G::CS, G::NT, G::SMEM, d, np, st);
#elif PFF_RESIDENT == 1
        using G = RG<NX, NY, 1>;
        return go<Arg>(k_res_bccg<NX, NY>, known, G::CS, G::NT, G::SMEM, d, np, st);
#else
        using G = RG<NX, NY, 1>;
        return go<Arg>(k_res_lap<NX, NY>, known, G::CS, G::W * 32, G::SMEM, d, np, st, pdl_on());
#endif
    } else {
        return cudaErrorNotSupported;
    }
}

template <int NX>
cudaError_t go_nx(int ny, const Arg& d, int np, cudaStream_t st) {
    switch (ny) {
        case 16: return go_size<NX, 16>(d, np, st);
        case 32: return go_size<NX, 32>(d, np, st);
        case 64: return go_size<NX, 64>(d, np, st);
        case 128: return go_size<NX, 128>(d, np, st);
        case 256: return go_size<NX, 256>(d, np, st);
        default: return cudaErrorNotSupported;
    }
}

cudaError_t go_any(int nx, int ny, const Arg& d, int np, cudaStream_t st) {
    switch (nx) {
        case 16: return go_nx<16>(ny, d, np, st);
        case 32: return go_nx<32>(ny, d, np, st);
        case 64: return go_nx<64>(ny, d, np, st);
        case 128: return go_nx<128>(ny, d, np, st);
        case 256: return go_nx<256>(ny, d, np, st);
        default: return cudaErrorNotSupported;
    }
}

}  // namespace

#if PFF_RESIDENT == 0
cudaError_t launch_resident_mech(const Desc<float>* d, int nx, int ny, int np, cudaStream_t st) {
    return go_any(nx, ny, d, np, st);
}
#elif PFF_RESIDENT == 1
cudaError_t launch_resident_bccg(const Desc<float>* d, int nx, int ny, int np, cudaStream_t st) {
    return go_any(nx, ny, d, np, st);
}
#else
cudaError_t launch_resident_laplacian(const Desc<float>& d, cudaStream_t st) { return go_any(d.nx, d.ny, d, 1, st); }
#endif

}  // namespace pff
