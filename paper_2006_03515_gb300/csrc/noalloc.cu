// kifmm_direct_noalloc: the photoionization sum by direct summation, without any
// device allocation.
//
// Some callers cannot call cudaMalloc at the moment they need S: code running while a
// CUDA graph is being captured on its stream (allocation would break or be illegal in the
// capture), real-time loops that forbid allocation after start-up, and processes whose
// device memory is fully reserved by another allocator. For them this entry point keeps
// its only work space, the cell weights q_j = I_j h^3 and the self-cell value, in one
// fixed array in device global memory that exists for as long as the library is loaded
// (on every GPU that loads it). The caller passes inputs and outputs as device pointers.
#include <cmath>
#include <mutex>

#include <cooperative_groups.h>

#include "internal.cuh"
#include "kernel.cuh"
#include "pair64.cuh"

namespace kifmm {

namespace cg = cooperative_groups;

// Work space: n weights followed by the partial sums of the self-cell value; every call writes it
// before reading it, so nothing needs clearing, but two calls that overlap on the GPU race on it.
static __device__ __align__(256) double g_noalloc_scratch[KIFMM_NOALLOC_MAX_POINTS + 32];
constexpr int NA_SIG = 32;   // partial sums of sigma

// positive nodes and their weights of the 32-point Gauss-Legendre rule; the 16-point rule
__device__ const double kGlX32[16] = {
    0.04830766568773832, 0.1444719615827965, 0.23928736225213706, 0.33186860228212767, 0.42135127613063533,
    0.5068999089322294, 0.5877157572407623, 0.6630442669302152, 0.7321821187402897, 0.7944837959679424,
    0.84936761373257, 0.8963211557660521, 0.9349060759377397, 0.9647622555875064, 0.9856115115452684,
    0.9972638618494816};
__device__ const double kGlW32[16] = {
    0.0965400885147278, 0.09563872007927486, 0.09384439908080457, 0.09117387869576389, 0.08765209300440381,
    0.08331192422694675, 0.07819389578707031, 0.0723457941088485, 0.06582222277636185, 0.058684093478535544,
    0.050998059262376175, 0.04283589802222668, 0.03427386291302143, 0.02539206530926206, 0.01627439473090567,
    0.007018610009470096};
__device__ const double kGlX16[8] = {
    0.09501250983763744, 0.2816035507792589, 0.45801677765722737, 0.6178762444026438, 0.755404408355003,
    0.8656312023878318, 0.9445750230732326, 0.9894009349916499};
__device__ const double kGlW16[8] = {
    0.1894506104550685, 0.18260341504492358, 0.16915651939500254, 0.14959598881657674, 0.12462897125553388,
    0.09515851168249279, 0.062253523938647894, 0.027152459411754096};

// q_j = I_j h^3 into the work space (S may be I itself), and sigma(h) as NA_SIG partial sums behind
// them, one block each. cell_exact: over the six faces, the solid angle
// times F(R) / (4 pi ln(b/a)), F(R) = int_0^R (e^{-ar} - e^{-br}) / r dr. Written
// F(R) = int_{ln a}^{ln b} (1 - exp(-e^t R)) dt it is a smooth integral (analytic for |Im t| < pi/2):
// panels of length <= 1.5 with 16 nodes reach rounding, and all (face node, t node) pairs are
// independent, 12288 exponentials over 32 blocks, where the two exponential integrals per node were
// series and continued fractions of some sixty dependent divisions in one block (3.2 ms of a call;
// now 16 us). The face integrand is analytic within a Bernstein ellipse of 1 + sqrt(2): 32 nodes a
// side (16 by symmetry) leave 1e-24.
__global__ void __launch_bounds__(256) k_na_prepare(const double* I, int64_t n, double h, double a, double b, int mode,
                                                    double* ws) {
    __shared__ double red[256];
    const double w = h * h * h;
    for (int64_t j = (int64_t)blockIdx.x * 256 + threadIdx.x; j < n; j += 256 * NA_SIG) ws[j] = I[j] * w;
    ws += n;
    const double lba = log(b / a);
    if (mode == KIFMM_SELF_PAPER_GL2) {   // h^3 K(h / 2), the paper's two-point rule
        if (threadIdx.x == 0) {
            const double rho = 0.5 * h;
            const double v = (exp(-a * rho) - exp(-b * rho)) / (rho * lba);
            ws[blockIdx.x] = blockIdx.x == 0 ? h * h * h * v / (3.14159265358979323846 * h * h) : 0.0;
        }
        return;
    }
    const int np = max(1, (int)ceil(lba / 1.5));
    const double half = 0.5 * lba / np;
    double acc = 0.0;
    for (int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x; e < 256LL * 16 * np; e += 256 * NA_SIG) {
        const int node = (int)(e % 256), k = (int)((e / 256) % 16), panel = (int)(e / 4096);
        const int i = node % 16, j = node / 16;
        const double u = 0.5 * h * kGlX32[i], v = 0.5 * h * kGlX32[j];
        const double R = sqrt(u * u + v * v + 0.25 * h * h);
        const double tk = k < 8 ? -kGlX16[7 - k] : kGlX16[k - 8], wk = kGlW16[k < 8 ? 7 - k : k - 8];
        const double s = a * exp(half * (2 * panel + 1 + tk));
        acc += (0.25 * h * h) * kGlW32[i] * kGlW32[j] * (0.5 * h) / (R * R * R) * (half * wk) * -expm1(-s * R);
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    // six faces, four quadrants
    if (threadIdx.x == 0) ws[blockIdx.x] = 24.0 * red[0] / (4.0 * 3.14159265358979323846 * lba);
}

// S_i = C * (sum_{j != i} K(|x_i - x_j|) q_j + sigma I_i), FP64: a cluster of CS blocks per 32 targets
// (a target per lane), every warp of it a contiguous share of the sources, which its lanes load and
// pass on by shuffles; the shares' sums are added in order, through distributed shared memory. One
// block of 256 targets each left 4096 points on 16 of the 152 SMs (14.0 ms; with the pairs of
// pair64.cuh 1.4 ms). CS = 8 below 1216 target groups, eight blocks on each of 152 SMs, else 1: 1000 points
// 0.12 ms with CS = 8 and 0.36 with 1, 16384 20.6 and 21.6, 30000 68.5 and 69.1, 38912 (1216 groups, one whole wave
// of single blocks) 115 and 102, 50000 189 and 181, 60000 273 and 256.
constexpr int NA_CLUSTER_GROUPS = 1216;
constexpr int NA_T = 256, NA_W = NA_T / 32;
template <int CS>
__global__ void __launch_bounds__(NA_T) k_na_direct(const double* __restrict__ pts, const double* I, int n, Pair64 kp,
                                                    double C, const double* __restrict__ ws, double* S) {
    __shared__ Pair64Tab tab;
    __shared__ double red[NA_W][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rank = blockIdx.x % CS;
    const int i = (int)(blockIdx.x / CS) * 32 + lane;
    pair64_tab_fill(tab);
    __syncthreads();
    const bool act = i < n;
    const double x = act ? pts[3 * (int64_t)i] : 0.0, y = act ? pts[3 * (int64_t)i + 1] : 0.0,
                 z = act ? pts[3 * (int64_t)i + 2] : 0.0;
    constexpr int SH = CS * NA_W;   // shares
    const int share = rank * NA_W + warp;
    const int j0 = (int)((int64_t)n * share / SH), j1 = (int)((int64_t)n * (share + 1) / SH);
    double acc = 0.0;
    for (int jb = j0; jb < j1; jb += 32) {
        const int j = jb + lane, m = min(32, j1 - jb);
        double sx = 0.0, sy = 0.0, sz = 0.0, sq = 0.0;
        if (j < j1) {
            sx = pts[3 * (int64_t)j];
            sy = pts[3 * (int64_t)j + 1];
            sz = pts[3 * (int64_t)j + 2];
            sq = ws[j];
        }
#pragma unroll 2
        for (int k = 0; k < m; ++k) {
            const double dx = x - __shfl_sync(0xffffffffu, sx, k), dy = y - __shfl_sync(0xffffffffu, sy, k),
                         dz = z - __shfl_sync(0xffffffffu, sz, k), q = __shfl_sync(0xffffffffu, sq, k);
            const double r2 = dx * dx + dy * dy + dz * dz;
            const double v = pair64_kernel(r2, kp, tab) * q;
            if (jb + k != i) acc += v;
        }
    }
    red[warp][lane] = acc;
    if (CS > 1) cg::this_cluster().sync();
    else __syncthreads();
    if (rank == 0 && warp == 0 && act) {
        double s = 0.0, sig = 0.0;
        for (int r = 0; r < CS; ++r) {
            const double* o = CS > 1 ? cg::this_cluster().map_shared_rank(&red[0][0], r) : &red[0][0];
            for (int k = 0; k < NA_W; ++k) s += o[k * 32 + lane];
        }
        for (int k = 0; k < NA_SIG; ++k) sig += ws[n + k];
        S[i] = C * (s + sig * I[i]);
    }
    if (CS > 1) cg::this_cluster().sync();   // (the other blocks' sums are read above)
}

template <int CS>
static cudaError_t launch_na_direct(cudaStream_t st, const double* pts, const double* I, int n, const Pair64& kp,
                                    double C, const double* ws, double* S) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)((n + 31) / 32 * CS));
    cfg.blockDim = dim3(NA_T);
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = CS;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_na_direct<CS>, pts, I, n, kp, C, ws, S);
}

// Device address of the work space, looked up once per device (with that device current).
static std::mutex g_na_mutex;
static double* g_na_addr[64] = {};

static int scratch_address(double** out) {
    int dev = 0;
    KF_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) {
        set_error("kifmm_direct_noalloc: device index out of range");
        return KIFMM_ERR_ARG;
    }
    std::lock_guard<std::mutex> lock(g_na_mutex);
    if (!g_na_addr[dev]) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) {
            set_error(std::string("kifmm_direct_noalloc: cudaGetSymbolAddress: ") + cudaGetErrorString(e));
            return KIFMM_ERR_CUDA;
        }
        g_na_addr[dev] = static_cast<double*>(p);
    }
    *out = g_na_addr[dev];
    return KIFMM_OK;
}

}  // namespace kifmm

using namespace kifmm;

extern "C" int kifmm_direct_noalloc(const double* points_dev, int64_t n, double h, const double* I_dev,
                                    double* S_dev, double a, double b, double C, int self_mode, void* stream) {
    set_error("");
    if (!points_dev || !I_dev || !S_dev || n < 1) {
        set_error("kifmm_direct_noalloc: need non-NULL pointers and n >= 1");
        return KIFMM_ERR_ARG;
    }
    if (n > KIFMM_NOALLOC_MAX_POINTS) {
        set_error("kifmm_direct_noalloc: n = " + std::to_string(n) + " exceeds the fixed work space of " +
                  std::to_string(KIFMM_NOALLOC_MAX_POINTS) + " points");
        return KIFMM_ERR_ARG;
    }
    if (!(h > 0.0) || !std::isfinite(h) || !(a > 0.0) || !(b > a) || !std::isfinite(b) || !std::isfinite(C)) {
        set_error("kifmm_direct_noalloc: need h > 0, 0 < a < b and finite C");
        return KIFMM_ERR_ARG;
    }
    if (self_mode != KIFMM_SELF_CELL_EXACT && self_mode != KIFMM_SELF_PAPER_GL2) {
        set_error("kifmm_direct_noalloc: unknown self_mode");
        return KIFMM_ERR_ARG;
    }
    double* ws = nullptr;
    KF_TRY(scratch_address(&ws));
    cudaStream_t st = (cudaStream_t)stream;
    k_na_prepare<<<NA_SIG, 256, 0, st>>>(I_dev, n, h, a, b, self_mode, ws);
    KF_LAUNCH();
    const Pair64 kp = make_pair64(make_kparams(a, b));
    auto* fn = (n + 31) / 32 < NA_CLUSTER_GROUPS ? launch_na_direct<8> : launch_na_direct<1>;
    KF_CUDA(fn(st, points_dev, I_dev, (int)n, kp, C, ws, S_dev));
    return KIFMM_OK;
}
