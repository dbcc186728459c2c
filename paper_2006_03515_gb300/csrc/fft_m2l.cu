// M2L of the FP64 form by Fourier transforms (the remark after Eq. (m2l), as in the cited KIFMM).
//
// The upward equivalent surface of a source box and the downward check surface of a target box are the
// boundary points of m0^3 lattices of one spacing, so a translation is a linear convolution of the
// densities phi (on the full lattice, zero inside) with the kernel at the lattice offsets. On a periodic
// lattice of n = 2 m0 - 1 points per axis nothing wraps around onto the m0^3 outputs:
//
//   q^{B,d} = sample IDFT( sum over V(B) of DFT(K_slot) DFT(phi^A) ),
//
// one forward transform per box, the kernel transforms tabulated per level and offset slot at plan time,
// the products summed in frequency space, one inverse transform per box. Coefficients enter and leave by
// the basis changes phi = V c and d = V^T q of the dense form.
//
// What bounds the FP64 M2L is the FP64 pipe (two lanes an SM). A V pair takes 4 n^2 m0 fused
// multiply-adds (m0 = 6: 2904) instead of R^2 (16,384 at R = 128) in the rank basis, and a box about
// 60,000 for its transforms, taken as n-term sums (a box has some 130 to 189 pairs). Measured on one
// GB300, 48^3 points in 4096 leaves of 27, m0 = 6: 3.65 ms and
// 0.25 ms for the boxes' transforms (and 0.6 ms for the basis changes), against 124.7 ms for the dense form, whose tiles
// of 64 boxes also left half of each operand zero and most SMs idle. A block takes one target box: a
// frequency per thread and register, so that the pair loop reads 32 bytes from L2 per four FP64
// instructions (16 bytes a cycle and SM).
#include <cmath>
#include <cstdlib>
#include <string>
#include <vector>

#include "internal.cuh"
#include "kernel.cuh"

namespace kifmm {

static inline unsigned nbf(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

constexpr int FF_T = 256, FF_MAXM0 = 8, FF_MAXN = 2 * FF_MAXM0 - 1;
// the half spectrum along x, [kz][ky][kx], kx < m0 (n odd)
__host__ __device__ inline int ff_nf(int m0) { return (2 * m0 - 1) * (2 * m0 - 1) * m0; }

// e^{-2 pi i k / n}, k < n, in shared memory
__device__ __forceinline__ void ff_twiddles(int n, double2* tw) {
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        double s, c;
        sincospi(-2.0 * k / n, &s, &c);
        tw[k] = make_double2(c, s);
    }
}

__device__ __forceinline__ void cfma(double2& a, const double2& x, const double2& y) {
    a.x = fma(x.x, y.x, a.x);
    a.x = fma(-x.y, y.y, a.x);
    a.y = fma(x.x, y.y, a.y);
    a.y = fma(x.y, y.x, a.y);
}

// DFT of a real array g[nz][ny][nx] (zero beyond, up to n) into out[kz][ky][kx], kx < m0; A, B: scratch of
// nz ny m0 and nz n m0 values
__device__ void ff_forward(const double* g, int nz, int ny, int nx, int n, int m0, const double2* tw, double2* A,
                           double2* B, double2* out) {
    for (int e = threadIdx.x; e < nz * ny * m0; e += blockDim.x) {
        const int kx = e % m0, l = e / m0;
        double2 a = make_double2(0.0, 0.0);
        for (int x = 0, t = 0; x < nx; ++x, t = (t + kx) % n) {
            a.x = fma(g[l * nx + x], tw[t].x, a.x);
            a.y = fma(g[l * nx + x], tw[t].y, a.y);
        }
        A[e] = a;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < nz * n * m0; e += blockDim.x) {
        const int kx = e % m0, ky = (e / m0) % n, z = e / (m0 * n);
        double2 a = make_double2(0.0, 0.0);
        for (int y = 0, t = 0; y < ny; ++y, t = (t + ky) % n) cfma(a, A[(z * ny + y) * m0 + kx], tw[t]);
        B[e] = a;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < n * n * m0; e += blockDim.x) {
        const int q = e % (n * m0), kz = e / (n * m0);
        double2 a = make_double2(0.0, 0.0);
        for (int z = 0, t = 0; z < nz; ++z, t = (t + kz) % n) cfma(a, B[z * n * m0 + q], tw[t]);
        out[e] = a;
    }
}

// Transforms of the kernel at the lattice offsets u in {-(m0-1)..m0-1}^3 (stored at u mod n) of one
// level's offset slots: K(|delta u - 2 r slot offset|); near slots stay zero.
__global__ void __launch_bounds__(FF_T) k_fft_table(int m0, double delta, double r, KParams kp, double2* out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = 2 * m0 - 1, nf = ff_nf(m0), slot = blockIdx.x;
    const int off[3] = {slot % 7 - 3, (slot / 7) % 7 - 3, slot / 49 - 3};
    double2* A = reinterpret_cast<double2*>(smem_raw);
    double2* B = A + nf;
    double* g = reinterpret_cast<double*>(B + nf);
    __shared__ double2 tw[FF_MAXN];
    out += (int64_t)slot * nf;
    if (abs(off[0]) <= 1 && abs(off[1]) <= 1 && abs(off[2]) <= 1) {
        for (int e = threadIdx.x; e < nf; e += FF_T) out[e] = make_double2(0.0, 0.0);
        return;
    }
    ff_twiddles(n, tw);
    for (int e = threadIdx.x; e < n * n * n; e += FF_T) {
        const int v[3] = {e % n, (e / n) % n, e / (n * n)};
        double d2 = 0.0;
        for (int k = 0; k < 3; ++k) {
            const double d = delta * (v[k] < m0 ? v[k] : v[k] - n) - 2.0 * r * off[k];
            d2 += d * d;
        }
        g[e] = kern_f64(sqrt(d2), kp);
    }
    __syncthreads();
    ff_forward(g, n, n, n, n, m0, tw, A, B, out);
}

// spectrum of each box's densities phi ([box - b0][S]) on the lattice
__global__ void __launch_bounds__(FF_T) k_fft_boxes(int m0, int S, const int32_t* lidx, const double* phi, double2* spec) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = 2 * m0 - 1, m3 = m0 * m0 * m0;
    double2* A = reinterpret_cast<double2*>(smem_raw);
    double2* B = A + m3;
    double* g = reinterpret_cast<double*>(B + m0 * n * m0);
    __shared__ double2 tw[FF_MAXN];
    ff_twiddles(n, tw);
    phi += (int64_t)blockIdx.x * S;
    for (int e = threadIdx.x; e < m3; e += FF_T) g[e] = lidx[e] >= 0 ? phi[lidx[e]] : 0.0;
    __syncthreads();
    ff_forward(g, m0, m0, m0, n, m0, tw, A, B, spec + (int64_t)blockIdx.x * ff_nf(m0));
}

// check potentials q[box - b0][S] of each target box: the products over its V list (vtab row), KF
// frequencies a thread, then the inverse transform at the surface points
template <int KF>
__global__ void __launch_bounds__(FF_T) k_fft_m2l(int m0, int S, int64_t b0, const int32_t* __restrict__ level,
                                                  const int32_t* __restrict__ vtab, const int32_t* __restrict__ lidx,
                                                  const double2* __restrict__ tab, const double2* __restrict__ spec,
                                                  double* __restrict__ q) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = 2 * m0 - 1, nf = ff_nf(m0);
    double2* D = reinterpret_cast<double2*>(smem_raw);   // [kz][ky][kx], then [z][y][kx]
    double2* M = D + nf;                                 // [z][ky][kx]
    __shared__ double2 tw[FF_MAXN];
    __shared__ int32_t lsrc[kOffsetSlots], lslot[kOffsetSlots];
    __shared__ int count;
    const int64_t box = b0 + blockIdx.x;
    ff_twiddles(n, tw);
    if (threadIdx.x < 32) {   // the V list in slot order
        int c = 0;
        for (int s0 = 0; s0 < kOffsetSlots; s0 += 32) {
            const int s = s0 + threadIdx.x;
            const int a = s < kOffsetSlots ? vtab[box * kOffsetSlots + s] : -1;
            const unsigned m = __ballot_sync(0xffffffffu, a >= 0);
            if (a >= 0) {
                const int at = c + __popc(m & ((1u << threadIdx.x) - 1));
                lsrc[at] = a;
                lslot[at] = s;
            }
            c += __popc(m);
        }
        if (threadIdx.x == 0) count = c;
    }
    __syncthreads();
    const double2* T = tab + (int64_t)(level[box] - 2) * kOffsetSlots * nf;
    double2 acc[KF];
#pragma unroll
    for (int k = 0; k < KF; ++k) acc[k] = make_double2(0.0, 0.0);
    const int nv = count;
#pragma unroll 2
    for (int v = 0; v < nv; ++v) {
        const double2* t = T + (int64_t)lslot[v] * nf;
        const double2* c = spec + ((int64_t)lsrc[v] - b0) * nf;
#pragma unroll
        for (int k = 0; k < KF; ++k) {
            const int f = threadIdx.x + FF_T * k;
            if (f < nf) cfma(acc[k], t[f], c[f]);
        }
    }
#pragma unroll
    for (int k = 0; k < KF; ++k) {
        const int f = threadIdx.x + FF_T * k;
        if (f < nf) D[f] = acc[k];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < m0 * n * m0; e += FF_T) {   // over kz (conjugate twiddles)
        const int r = e % (n * m0), z = e / (n * m0);
        double2 a = make_double2(0.0, 0.0);
        for (int kz = 0, t = 0; kz < n; ++kz, t = (t + z) % n) cfma(a, D[kz * n * m0 + r], make_double2(tw[t].x, -tw[t].y));
        M[e] = a;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < m0 * m0 * m0; e += FF_T) {   // over ky
        const int kx = e % m0, y = (e / m0) % m0, z = e / (m0 * m0);
        double2 a = make_double2(0.0, 0.0);
        for (int ky = 0, t = 0; ky < n; ++ky, t = (t + y) % n)
            cfma(a, M[(z * n + ky) * m0 + kx], make_double2(tw[t].x, -tw[t].y));
        D[e] = a;
    }
    __syncthreads();
    const double scale = 1.0 / ((double)n * n * n);
    for (int e = threadIdx.x; e < m0 * m0 * m0; e += FF_T) {   // over kx: kx and -kx are conjugates
        if (lidx[e] < 0) continue;
        const int x = e % m0, l = e / m0;
        double s = 0.0;
        for (int kx = 1, t = x; kx < m0; ++kx, t = (t + x) % n) {
            const double2 d = D[l * m0 + kx];
            s += d.x * tw[t].x + d.y * tw[t].y;   // Re(d conj(tw))
        }
        q[(int64_t)blockIdx.x * S + lidx[e]] = scale * (D[l * m0].x + 2.0 * s);
    }
}

// The FP64 form of the surface representation takes the transforms up to m0 = 8 (the evaluation's kernels
// then stay within 48 KB of shared memory), where their memory, which grows with the boxes (12.8 KB each at
// m0 = 6), is no more than that of the dense products' tables (45 MB a level), or else at most 16 GB of spectra
// and an eighth of what the device has free, so that plans made side by side do not crowd out one another; a plan that
// still runs out of memory is made again without them (kifmm_plan). KIFMM_M2L=simt keeps the dense products.
bool fft_m2l_wanted(const Plan& p) {
    const char* m2l = std::getenv("KIFMM_M2L");
    if (p.precision != KIFMM_FP64 || p.cheb || p.m0 > FF_MAXM0 || p.no_fft || (m2l && std::string(m2l) == "simt"))
        return false;
    const double nf = ff_nf(p.m0), slots = (double)(p.tree.nlevels - 2) * kOffsetSlots, spec = p.tree.nboxes * nf * 16.0;
    const double need = spec + p.tree.nboxes * p.S * 8.0 + slots * nf * 16.0;
    if (need <= slots * p.R * p.R * 8.0) return true;
    size_t free_b = 0, total_b = 0;
    if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return spec <= 16e9 && need <= free_b / 8.0;
}

int fft_m2l_plan(Plan& p) {
    p.fft_m2l = true;
    cudaStream_t st = p.stream;
    const int m0 = p.m0, nf = ff_nf(m0), n = 2 * m0 - 1, L = p.tree.nlevels;
    std::vector<int32_t> lidx((size_t)m0 * m0 * m0, -1);
    int s = 0;
    for (int z = 0; z < m0; ++z)
        for (int y = 0; y < m0; ++y)
            for (int x = 0; x < m0; ++x) {
                const bool in = x > 0 && x < m0 - 1 && y > 0 && y < m0 - 1 && z > 0 && z < m0 - 1;
                if (!in) lidx[(z * m0 + y) * m0 + x] = s++;
            }
    const int64_t nb = p.tree.nboxes - p.tree.level_start[2];
    KF_TRY(dev_alloc(p.fft_idx, lidx.size() * 4));
    KF_TRY(dev_alloc(p.fft_tab, (size_t)(L - 2) * kOffsetSlots * nf * 16));
    KF_TRY(dev_alloc(p.fft_spec, (size_t)nb * nf * 16));
    KF_TRY(dev_alloc(p.fft_q, (size_t)p.tree.nboxes * p.S * 8));
    KF_CUDA(cudaMemcpyAsync(p.fft_idx.p, lidx.data(), lidx.size() * 4, cudaMemcpyHostToDevice, st));
    const int smem = 2 * nf * 16 + n * n * n * 8;
    KF_CUDA(cudaFuncSetAttribute(k_fft_table, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    for (int l = 2; l < L; ++l) {
        const double r = p.tree.side / (double)(2ll << l);
        k_fft_table<<<kOffsetSlots, FF_T, smem, st>>>(m0, 2.0 * p.r_in * r / (m0 - 1), r,
                                                      make_kparams_kind(p.kind, p.a, p.b),
                                                      ptr<double2>(p.fft_tab) + (int64_t)(l - 2) * kOffsetSlots * nf);
        KF_LAUNCH();
    }
    KF_CUDA(cudaStreamSynchronize(st));
    return KIFMM_OK;
}

// fft_q rows of the boxes of level >= 2: densities in, downward check potentials out
int fft_m2l_apply(Plan& p, int64_t& nl) {
    cudaStream_t st = p.stream;
    const int m0 = p.m0, nf = ff_nf(m0), n = 2 * m0 - 1, m3 = m0 * m0 * m0;
    const int64_t b0 = p.tree.level_start[2], nb = p.tree.nboxes - b0;
    double* q = ptr<double>(p.fft_q) + b0 * p.S;
    const int sf = (m3 + m0 * n * m0) * 16 + m3 * 8, sm = (nf + m0 * n * m0) * 16;   // (below 48 KB for m0 <= 8)
    k_fft_boxes<<<(unsigned)nb, FF_T, sf, st>>>(m0, p.S, ptr<int32_t>(p.fft_idx), q, ptr<double2>(p.fft_spec));
    KF_LAUNCH();
    const int kf = (nf + FF_T - 1) / FF_T;
    auto* fn = kf <= 1 ? k_fft_m2l<1> : kf <= 2 ? k_fft_m2l<2> : kf <= 3 ? k_fft_m2l<3> : kf <= 5 ? k_fft_m2l<5> : k_fft_m2l<8>;
    fn<<<(unsigned)nb, FF_T, sm, st>>>(m0, p.S, b0, ptr<int32_t>(p.tree.level), ptr<int32_t>(p.vtab),
                                       ptr<int32_t>(p.fft_idx), ptr<double2>(p.fft_tab), ptr<double2>(p.fft_spec), q);
    KF_LAUNCH();
    nl += 2;
    return KIFMM_OK;
}

}  // namespace kifmm
