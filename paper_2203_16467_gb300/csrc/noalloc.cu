// noalloc.cu -- pff_apply_laplacian_noalloc (FP64) and _f32: the collocation
// Laplacian of a caller-owned device field, computed without allocating memory.
//
// Some callers cannot call cudaMalloc: a framework that has reserved the whole
// device memory for its own pool, a latency-critical loop that cannot afford
// the implicit device synchronisation an allocation may cause, or a caller
// that must not leave allocations behind.  These entry points run the same
// three passes as pff_apply_laplacian, but their scratch (one half spectrum of
// at most PFF_NOALLOC_MAX_N x (PFF_NOALLOC_MAX_N/2 + 16) complex values per
// precision, about 2.2 MB in FP64 and 1.1 MB in FP32) and twiddle tables are
// file-scope device arrays that every GPU loading the library keeps until exit.
//
// A call is launch-bound (a 64^2 field holds under a microsecond of work), so the
// descriptor is a kernel argument (its copy to the device was a fourth operation
// in the stream), and FP32 fields up to 2^14 pixels take one launch of one
// cluster (k_resident.cu): a 64^2 FP32 call in a row of calls 11.3 -> 2.7 us (5.9
// with the argument alone), one that is waited for 12.9 us (15.5), 512 x 256 FP64
// 49 -> 45 us (now 43; the FP64 pipe bounds its passes).
#include <cmath>
#include <cstring>
#include <mutex>

#include "../../include/pff.h"
#include "kernels.cuh"

namespace pff {
cudaError_t take_launch_error();   // launches rejected by the runtime on this host thread
namespace {

constexpr int NA_MAX = PFF_NOALLOC_MAX_N;
constexpr int NA_WP = ((NA_MAX / 2 + 1 + 15) / 16) * 16;
constexpr int NA_TW = 2 * NA_MAX;   // twiddle tables for lengths up to NA_MAX

static __device__ __align__(256) double2 g_na_spectrum[(size_t)NA_MAX * NA_WP];
static __device__ __align__(256) double2 g_na_twiddles[NA_TW];
static __device__ __align__(256) float2 g_na_spectrum_f[(size_t)NA_MAX * NA_WP];
static __device__ __align__(256) float2 g_na_twiddles_f[NA_TW];

struct DeviceSymbols {
    bool ready = false;
    double2* spectrum = nullptr;
    double2* twiddles = nullptr;
    float2* spectrum_f = nullptr;
    float2* twiddles_f = nullptr;
};
constexpr int NA_MAX_DEVICES = 64;
DeviceSymbols g_symbols[NA_MAX_DEVICES];
std::mutex g_mu;

template <typename S>
bool symbol(const S& sym, void** p) {
    if (cudaGetSymbolAddress(p, sym) == cudaSuccess) return true;
    cudaGetLastError();
    return false;
}

// Once per device, with that device current: device addresses of the arrays
// (the names are host-side stand-ins in host code) and the twiddle tables.
int setup(int dev, DeviceSymbols& out, const char** msg) {
    std::lock_guard<std::mutex> g(g_mu);
    DeviceSymbols& s = g_symbols[dev];
    if (!s.ready) {
        void* p[4] = {};
        if (!symbol(g_na_spectrum, &p[0]) || !symbol(g_na_twiddles, &p[1]) || !symbol(g_na_spectrum_f, &p[2]) ||
            !symbol(g_na_twiddles_f, &p[3])) {
            *msg = "cudaGetSymbolAddress failed";
            return PFF_ERR_CUDA;
        }
        s.spectrum = (double2*)p[0];
        s.twiddles = (double2*)p[1];
        s.spectrum_f = (float2*)p[2];
        s.twiddles_f = (float2*)p[3];
        static double2 tw[NA_TW];   // host staging without a heap allocation
        static float2 twf[NA_TW];
        tw[0] = make_double2(1.0, 0.0);
        tw[1] = make_double2(1.0, 0.0);
        for (int M = 2; M <= NA_MAX; M *= 2)
            for (int j = 0; j < M; ++j) {
                double a = -2.0 * M_PI * (double)j / (double)M;
                tw[M + j] = make_double2(std::cos(a), std::sin(a));
            }
        for (int j = 0; j < NA_TW; ++j) twf[j] = make_float2((float)tw[j].x, (float)tw[j].y);
        // a copy from pageable memory may return before its DMA has landed, and kernels on
        // non-blocking streams do not wait for the legacy stream: the device synchronisation
        // makes the tables complete before any call can read them
        if (cudaMemcpyToSymbol(g_na_twiddles, tw, sizeof(double2) * NA_TW) != cudaSuccess ||
            cudaMemcpyToSymbol(g_na_twiddles_f, twf, sizeof(float2) * NA_TW) != cudaSuccess ||
            cudaDeviceSynchronize() != cudaSuccess) {
            *msg = "twiddle upload failed";
            cudaGetLastError();
            return PFF_ERR_CUDA;
        }
        s.ready = true;
    }
    out = s;
    return PFF_OK;
}

bool pow2_in_range(int n) { return n >= 16 && n <= NA_MAX && (n & (n - 1)) == 0; }

// the passes with the descriptor as an argument
template <typename T, int NX>
__global__ void __launch_bounds__(RowCfg<T, NX, 1>::NT) k_na_row_fwd(const __grid_constant__ Desc<T> d) {
    row_fwd_body<T, NX, 1, FCopyIn<T, 1>>(d);
}
template <typename T, int NX>
__global__ void __launch_bounds__(RowCfg<T, NX, 1>::NT) k_na_row_inv(const __grid_constant__ Desc<T> d) {
    row_inv_body<T, NX, 1, FCopyOut<T, 1>>(d);
}
template <typename T, int NY>
__global__ void __launch_bounds__(ColCfg<T, NY, 1>::NT) k_na_col(const __grid_constant__ Desc<T> d) {
    col_body<T, NY, 1, FColLapPlain>(d);
}
__global__ void __launch_bounds__(64 * COL512_CW) k_na_col512(const __grid_constant__ Desc<float> d) {
    col512_body<float, 1, FColLapPlain, COL512_CW>(d);
}

template <typename T>
void go(void (*fn)(Desc<T>), unsigned blocks, unsigned threads, size_t smem, cudaStream_t st, const Desc<T>& d, int key) {
    smem_optin((const void*)fn, smem);
    const bool tm = timing_on();
    if (tm) timing_begin(key, st);
    launch_pdl<T>(fn, dim3(blocks), dim3(threads), smem, st, d);
    if (tm) timing_end(key, st);
    count_launch();
}
template <typename T, int N>
void rows(bool forward, const Desc<T>& d, cudaStream_t st) {
    using Cfg = RowCfg<T, N, 1>;
    go<T>(forward ? k_na_row_fwd<T, N> : k_na_row_inv<T, N>, d.ny / Cfg::ROWS, Cfg::NT, Cfg::SMEM, st, d,
          forward ? FAM_ROW_FWD * 16 + RF_COPY1 : FAM_ROW_INV * 16 + RI_COPY1);
}
template <typename T, int N>
void columns(const Desc<T>& d, cudaStream_t st) {
    const int nm = d.nx / 2 + 1, key = FAM_COL * 16 + CO_LAP_PLAIN;
    if constexpr (N == 512 && sizeof(T) == 4) {
        using Cfg = Col512Cfg<T, 1, COL512_CW>;
        go<T>(k_na_col512, (nm + COL512_CW - 1) / COL512_CW, Cfg::NT, Cfg::SMEM, st, d, key);
    } else {
        using Cfg = ColCfg<T, N, 1>;
        go<T>(k_na_col<T, N>, (nm + Cfg::CWE - 1) / Cfg::CWE, Cfg::NT, Cfg::SMEM, st, d, key);
    }
}
#define NA_SIZES(n, CALL)                                  \
    switch (n) {                                           \
        case 16: { constexpr int N_ = 16; CALL; } break;   \
        case 32: { constexpr int N_ = 32; CALL; } break;   \
        case 64: { constexpr int N_ = 64; CALL; } break;   \
        case 128: { constexpr int N_ = 128; CALL; } break; \
        case 256: { constexpr int N_ = 256; CALL; } break; \
        case 512: { constexpr int N_ = 512; CALL; } break; \
        default: break;                                    \
    }

template <typename T, typename C>
int apply(int nx, int ny, double dx, const T* in_dev, T* out_dev, void* cuda_stream, const char** err_msg,
          C* spectrum, C* twiddles) {
    const char* dummy = nullptr;
    const char** msg = err_msg ? err_msg : &dummy;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    Desc<T> d;
    std::memset(&d, 0, sizeof(d));
    d.r[0] = const_cast<T*>(in_dev);   // FCopyIn reads r[0]
    d.q[0] = out_dev;                  // FCopyOut writes q[0]
    d.S = spectrum;
    d.tw = twiddles;
    d.nx = nx;
    d.ny = ny;
    d.wp = ((nx / 2 + 1 + 15) / 16) * 16;
    d.k.inv_n = 1.0 / ((double)nx * (double)ny);
    d.k.two_pi_over_Lx = 2.0 * M_PI / (nx * dx);
    d.k.two_pi_over_Ly = 2.0 * M_PI / (ny * dx);
    bool done = false;
    if constexpr (sizeof(T) == 4) {
        if (nx * ny <= RESIDENT_PIXELS && resident_aligned(in_dev, out_dev) && !timing_on()) {
            done = launch_resident_laplacian(d, st) == cudaSuccess;
            if (!done) cudaGetLastError();   // no such size or no such cluster here: the three passes
        }
    }
    if (!done) {
        NA_SIZES(nx, (rows<T, N_>(true, d, st)));
        NA_SIZES(ny, (columns<T, N_>(d, st)));
        NA_SIZES(nx, (rows<T, N_>(false, d, st)));
    }
    if (take_launch_error() != cudaSuccess) {
        *msg = "kernel launch failed";
        return PFF_ERR_CUDA;
    }
    return PFF_OK;
}

int check(int nx, int ny, double dx, const void* in_dev, const void* out_dev, const char** msg,
          DeviceSymbols& sym) {
    if (!pow2_in_range(nx) || !pow2_in_range(ny)) {
        *msg = "nx and ny must be powers of two from 16 to PFF_NOALLOC_MAX_N (512)";
        return PFF_ERR_INVALID_ARG;
    }
    if (!(dx > 0.0) || !in_dev || !out_dev) {
        *msg = "dx must be positive and both device pointers non-null";
        return PFF_ERR_INVALID_ARG;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NA_MAX_DEVICES) {
        cudaGetLastError();
        *msg = "no usable current CUDA device";
        return PFF_ERR_CUDA;
    }
    return setup(dev, sym, msg);
}

}  // namespace
}  // namespace pff

extern "C" int pff_apply_laplacian_noalloc(int nx, int ny, double dx, const double* in_dev, double* out_dev,
                                           void* cuda_stream, const char** err_msg) {
    using namespace pff;
    const char* dummy = nullptr;
    const char** msg = err_msg ? err_msg : &dummy;
    *msg = nullptr;
    DeviceSymbols sym;
    int rc = check(nx, ny, dx, in_dev, out_dev, msg, sym);
    if (rc) return rc;
    return apply<double>(nx, ny, dx, in_dev, out_dev, cuda_stream, msg, sym.spectrum, sym.twiddles);
}

extern "C" int pff_apply_laplacian_noalloc_f32(int nx, int ny, double dx, const float* in_dev, float* out_dev,
                                               void* cuda_stream, const char** err_msg) {
    using namespace pff;
    const char* dummy = nullptr;
    const char** msg = err_msg ? err_msg : &dummy;
    *msg = nullptr;
    DeviceSymbols sym;
    int rc = check(nx, ny, dx, in_dev, out_dev, msg, sym);
    if (rc) return rc;
    return apply<float>(nx, ny, dx, in_dev, out_dev, cuda_stream, msg, sym.spectrum_f, sym.twiddles_f);
}
