// Learned surrogate: a 3D spectral neural operator (forward, backward, Adam) and the
// surrogate-first photoionization solve with the FMM as judge and fallback.
//
// Network on an n^3 grid, width C, m modes per axis, L layers, projection width P:
//   v_0 = Wl u + bl;  z_l = SpecConv_l(v_l) + W_l v_l + b_l;  v_{l+1} = GELU(z_l) (l < L-1),
//   v_L = z_{L-1};  y = Q2 . GELU(Q1 v_L + q1) + q2,
//   SpecConv(v)(o, x) = (1/n^3) sum_{k in K} w_kz Re[ (R(k) V(k))_o e^{+2 pi i k.x/n} ],
//   V(c, k) = sum_x v(c, x) e^{-2 pi i k.x/n},  K = Kx x Ky x Kz,
//   Kx = Ky = {0..m-1} U {n-m..n-1}, Kz = {0..m-1}, w_0 = 1, w_{kz>=1} = 2.
// The truncated transforms run axis by axis as small dense DFTs against twiddle tables (a
// partial DFT keeps 2m of n frequencies, so a full FFT would be wasted work); the work is
// bound by memory traffic, so the kernels are organised to touch each field once:
//  * the z-row kernel owns the n values along the last axis of every channel at one (b, x, y): it
//    fuses the inverse last-axis DFT, the pointwise layer W v + b (or its transpose), GELU (or its
//    derivative), the projection and the next layer's forward last-axis DFT;
//  * the "fold" kernels do the DFTs along the first two axes on the m-wide spectra, staged through
//    shared memory;
//  * the per-mode channel mix is tiled over a few modes, with R in shared memory;
//  * the weights' gradients are sums over chunks of points, in register tiles.
// Spectral weights R are held in FP32 (master) and used rounded to BF16 (FP32
// accumulation) unless the model is switched to FP32 weights.
//
// Period: the transforms may take a period N >= n (angles 2 pi k x / N, negative
// frequencies N - m..N - 1, factor 1/N^3): the n^3 grid is then the corner of a zero-padded
// N^3 grid, so that the spectral convolution is not periodic on the grid itself.
// Near part: the model may add near(u) = sigma u + sum_{0 < |d| <= r_out} K(h|d|) w(|d|) h^3
// u(x + d) to its output (w = 1 up to r_in, cos^2 taper to 0 at r_out; u = 0 outside the
// grid), the exact short-range part of the photoionization sum (Sec. 3, Eq. (summation)) in
// the amplitude-normalised form u = I / max I, y = S / (C max I); the network then carries
// the smooth far part, whose Fourier multiplier on the N-periodic grid can initialise it
// (sno_init_far_field).
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "internal.cuh"
#include "kernel.cuh"
#include "selfcell.cuh"

namespace kifmm {

constexpr int MAXC = 64;              // widest layer
constexpr int MAXP = 128;             // widest projection
constexpr int SNO_MAX_JUDGE = 4096;   // most judge targets per photo_solve
constexpr int ZR_T = 256;             // threads of the z-row kernels
constexpr int ZR_RG = 4;              // z-row groups (b, x, y) per block

struct SnoModel {
    int n = 64, C = 32, m = 12, L = 4, P = 64, maxB = 32;
    int bf16 = 1;
    cudaStream_t st = nullptr;
    int64_t K = 0, np3 = 0;          // modes, grid points
    int64_t nparam = 0;
    std::vector<int64_t> off;        // offsets: Wl, bl, then per layer Rr, Ri, W, b, then Q1, q1, Q2, q2
    DevBuf theta, grad, adam_m, adam_v, rbf;   // rbf: BF16 copies of Rr, Ri per layer
    DevBuf tabs;                     // float2 twiddle tables
    int64_t tzf, tyf, tfo, tph;   // table offsets (float2 units)
    // fields (FP32): v[L+1][B][C][np3], z[L][B][C][np3], dz ping-pong [2][B][C][np3], y and dy [B][np3]
    DevBuf v, z, dz, yb, dy, loss;
    // spectra (float2): cz [B][C][n][n][m], cy / gx [B][C][n][2m][m], gy [B][C][n][n][m],
    // V per layer [L][B][C][K], g / ga [B][C][K]
    DevBuf cz, cy, gx, gy, Vst, g, ga;
    DevBuf m0ab;                     // inference, layer 0: A = R Wl and Bc = (R bl) O, [2][C][K] complex
    DevBuf jt, jref, jorig, jerr;    // photo_solve judge: targets, reference values, caller indices, error
    int mix_mb = 1;                  // modes per block of k_mix_grad
    size_t lift_smem = 0, mixg_smem = 0;
    int num_sms = 1;
    int64_t steps = 0;
    int period = 0;                  // N of the transforms (>= n)
    // exact near part (amplitude-normalised linear form): y += near(u)
    int near_on = 0;
    double na = 0, nb = 0, nh = 0, nsig = 0, nr_in = 0, nr_out = 0;
    int nself = KIFMM_SELF_CELL_EXACT, nR = 0, ntaps = 0, ngroups = 0;   // halo (cells), stencil columns
    DevBuf near_d, near_w;           // bounds and int2 (di, dj) of the groups of stencil columns, a group's weights
    DevBuf scal;                     // photo_solve: amplitude scale (double)
    DevBuf jws;                      // photo_solve: the judge's work space (sized at creation)
};

// ---- layout ----------------------------------------------------------------------------
static void sno_layout(SnoModel& M) {
    const int64_t C = M.C, K = M.K;
    M.off.clear();
    int64_t o = 0;
    auto add = [&](int64_t k) {
        M.off.push_back(o);
        o += k;
    };
    add(C);
    add(C);
    for (int l = 0; l < M.L; ++l) {
        add(K * C * C);
        add(K * C * C);
        add(C * C);
        add(C);
    }
    add((int64_t)M.P * C);
    add(M.P);
    add(M.P);
    add(1);
    M.nparam = o;
}
enum { O_WL = 0, O_BL = 1 };
static inline int o_rr(int l) { return 2 + 4 * l; }
static inline int o_ri(int l) { return 3 + 4 * l; }
static inline int o_w(int l) { return 4 + 4 * l; }
static inline int o_b(int l) { return 5 + 4 * l; }
static inline int o_q1(const SnoModel& M) { return 2 + 4 * M.L; }

static inline unsigned nbs(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

// ---- kernels ---------------------------------------------------------------------------
__device__ __forceinline__ float gelu_f(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_d(float x) {
    return 0.5f * (1.0f + erff(x * 0.70710678118654752f)) + x * 0.3989422804014327f * expf(-0.5f * x * x);
}

// Twiddle tables: tzf[kz][z] = e^{-i kz z}, tyf[k][y] = e^{-i k y} (k = 0..2m-1 mapped to
// {0..m-1} U {N-m..N-1}),
// tfo[j][k] = (cos, sin)(k (zc - j)) for j < n / 2 and k = 0..m with zc = (n - 1) / 2,
// tph[k] = (cos, sin)(k zc) (angles in 2 pi / N units, N the period, grid indices 0..n-1).
__global__ void k_tables(int n, int N, int m, float2* t, int64_t tzf, int64_t tyf, int64_t tfo, int64_t tph) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const double tw = 6.283185307179586476925286766559 / N;
    auto kxy = [&](int k) { return k < m ? k : N - 2 * m + k; };
    if (i < m * n) {
        int kz = i / n, z = i % n;
        double a = tw * kz * z;
        t[tzf + i] = make_float2((float)cos(a), (float)-sin(a));
    }
    if (i < 2 * m * n) {
        int k = i / n, y = i % n;
        double a = tw * kxy(k) * y;
        t[tyf + i] = make_float2((float)cos(a), (float)-sin(a));
    }
    if (i < n / 2 * (m + 1)) {
        int j = i / (m + 1), k = i % (m + 1);
        double a = tw * k * (0.5 * (n - 1) - j);
        t[tfo + i] = make_float2((float)cos(a), (float)sin(a));
    }
    if (i <= m) {
        double a = tw * i * (0.5 * (n - 1));
        t[tph + i] = make_float2((float)cos(a), (float)sin(a));
    }
}

// 8-byte asynchronous global-to-shared copies (the plane and z-row kernels' prefetch)
__device__ __forceinline__ void sno_cp8(void* dst, const void* src) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void sno_cp16(void* dst, const void* src) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
// (zeros in place of the source where it is not there)
__device__ __forceinline__ void sno_cp16z(void* dst, const void* src, bool there) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(there ? 16 : 0) : "memory");
}
__device__ __forceinline__ void sno_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void sno_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Plane DFTs along x and y, folded: in[p][q][i] -> out[p][j][i] with p < P planes and i < inner
// columns. About the grid's centre zc = (n - 1) / 2 the points q and n - 1 - q lie at -t and
// +t, so a frequency pair +-k needs only P_k = sum_t cos(k t) s_t and Q_k = sum_t sin(k t) d_t
// of the sums and differences s, d of the two points (forward: F(+-k) = e^{-+i k zc} (P_k -+ i Q_k)),
// and a point pair only U_t = sum_k cos(k t) a_k and V_t = sum_k sin(k t) b_k of those of the two
// frequencies (inverse: f(+-t) = U_t +- i V_t): a quarter of the dense form's FMAs. What is
// left is bound by memory: persistent blocks copy the next tile of columns (whole planes
// where they are short, else a chunk of columns of one plane) in 16-byte pieces, the way it
// lies in memory, while they compute the current one.
// One GB300, 32 fields of 64^3 at width 32 and 12 modes: 16 passes 3.55 -> 1.66 ms
// (the dense form read its tiles in 8-byte pieces); the largest, 554 MB, 419 -> 176 us = 3.1 TB/s.
struct FoldTile {
    int64_t P, ntiles;
    int L, inner, PB, W, nch, ps;   // rows in, columns in all, planes and columns a tile, chunks, plane stride
};
__device__ __forceinline__ void fold_shape(const FoldTile& f, int64_t t, int64_t& p0, int& np, int& i0, int& w) {
    const int64_t pb = t / f.nch;
    p0 = pb * f.PB;
    np = (int)min((int64_t)f.PB, f.P - p0);
    i0 = (int)(t - pb * f.nch) * f.W;
    w = min(f.W, f.inner - i0);
}
// copies tile t to dst[pl][q][w] (rows of f.W, planes of f.ps elements)
__device__ __forceinline__ void fold_issue(const FoldTile& f, int64_t t, const float2* __restrict__ in, float2* dst) {
    int64_t p0;
    int np, i0, w;
    fold_shape(f, t, p0, np, i0, w);
    if (f.nch == 1) {   // whole planes: contiguous, an even number of elements (L is even)
        const int half = f.L * f.inner / 2;
        for (int pl = 0; pl < np; ++pl) {
            const float2* src = in + (p0 + pl) * f.L * (int64_t)f.inner;
            for (int r = threadIdx.x; r < half; r += blockDim.x) sno_cp16(dst + pl * f.ps + 2 * r, src + 2 * r);
        }
        return;
    }
    const float2* src = in + p0 * f.L * (int64_t)f.inner + i0;
    const int lane = threadIdx.x & 31;
    if (f.inner % 2 == 0) {   // (f.W is even, so is the last chunk's width)
        for (int q = threadIdx.x >> 5; q < f.L; q += blockDim.x >> 5)
            for (int r = lane; r < w / 2; r += 32) sno_cp16(dst + q * f.W + 2 * r, src + (int64_t)q * f.inner + 2 * r);
    } else {
        for (int q = threadIdx.x >> 5; q < f.L; q += blockDim.x >> 5)
            for (int r = lane; r < w; r += 32) sno_cp8(dst + q * f.W + r, src + (int64_t)q * f.inner + r);
    }
}

// Factor of column i (kz = i mod m): the z rows' transforms are taken about their centre as well, and
// their phase e^{+i kz zc} belongs to the x transforms, where the spectra are smallest. zscale = 0: the
// rows' transforms are not centred, factor 1; else zscale, twice that for kz > 0 where it is not 1
// (1 / N^3 of the inverse transform and the conjugate half of the spectrum).
__device__ __forceinline__ float2 fold_zphase(const float2* __restrict__ tph, int m, int i, float zscale) {
    if (zscale == 0.f) return make_float2(1.f, 0.f);
    const int kz = i % m;
    const float w = zscale != 1.f && kz > 0 ? 2.f * zscale : zscale;
    const float2 ph = __ldg(tph + kz);
    return make_float2(w * ph.x, w * ph.y);
}

constexpr int FF_T = 128;   // threads of the forward kernel
constexpr int FV_T = 256;   // and of the inverse
constexpr int FV_J = 8;     // point pairs a thread of the inverse

// n points to 2m frequencies; a thread takes one column and KB frequencies (of 0..m)
template <int KB>
__global__ void __launch_bounds__(FF_T) k_fold_fwd(const float2* __restrict__ in, float2* __restrict__ out,
                                                   const float2* __restrict__ tfo, const float2* __restrict__ tph,
                                                   int m, int nkb, float zscale, FoldTile f) {
    constexpr int KP = (KB + 1) & ~1;   // (a table row is read in 16-byte pieces)
    extern __shared__ __align__(16) float2 psh[];
    const int n = f.L, nh = n / 2, bufn = f.PB * f.ps;
    float2* T = psh;                    // [nkb][n / 2][KP], zero past m
    float2* buf = T + nkb * nh * KP;    // two tiles
    for (int e = threadIdx.x; e < nkb * nh * KP; e += FF_T) {
        const int u = e % KP, j = (e / KP) % nh, k = (e / (KP * nh)) * KB + u;
        T[e] = u < KB && k <= m ? tfo[j * (m + 1) + k] : make_float2(0.f, 0.f);
    }
    int64_t t = blockIdx.x;
    if (t < f.ntiles) fold_issue(f, t, in, buf);
    sno_commit();
    for (int it = 0; t < f.ntiles; t += gridDim.x, ++it) {
        sno_wait_all();
        __syncthreads();   // the tile is there, and the other buffer has been read
        if (t + gridDim.x < f.ntiles) fold_issue(f, t + gridDim.x, in, buf + ((it + 1) & 1) * bufn);
        sno_commit();
        int64_t p0;
        int np, i0, w;
        fold_shape(f, t, p0, np, i0, w);
        const int ncol = np * w;
        for (int e = threadIdx.x; e < nkb * ncol; e += FF_T) {
            const int kb = e / ncol, col = e - kb * ncol, pl = col / w, i = col - pl * w;
            const float2* lo = buf + (it & 1) * bufn + pl * f.ps + i;
            const float2* hi = lo + (n - 1) * f.W;
            const float4* tk = reinterpret_cast<const float4*>(T + kb * nh * KP);
            float pr[KP], pi[KP], qr[KP], qi[KP];
#pragma unroll
            for (int u = 0; u < KP; ++u) pr[u] = pi[u] = qr[u] = qi[u] = 0.f;
            for (int j = 0; j < nh; ++j, lo += f.W, hi -= f.W, tk += KP / 2) {
                const float2 x0 = *lo, x1 = *hi;
                const float sr = x1.x + x0.x, si = x1.y + x0.y, dr = x1.x - x0.x, di = x1.y - x0.y;
#pragma unroll
                for (int u = 0; u < KP; u += 2) {
                    const float4 c = tk[u / 2];
                    pr[u] = fmaf(c.x, sr, pr[u]);
                    pi[u] = fmaf(c.x, si, pi[u]);
                    qr[u] = fmaf(c.y, dr, qr[u]);
                    qi[u] = fmaf(c.y, di, qi[u]);
                    if (u + 1 < KB) {
                        pr[u + 1] = fmaf(c.z, sr, pr[u + 1]);
                        pi[u + 1] = fmaf(c.z, si, pi[u + 1]);
                        qr[u + 1] = fmaf(c.w, dr, qr[u + 1]);
                        qi[u + 1] = fmaf(c.w, di, qi[u + 1]);
                    }
                }
            }
            float2* o = out + (p0 + pl) * 2 * m * (int64_t)f.inner + i0 + i;
            const float2 z = fold_zphase(tph, m, i0 + i, zscale);   // (conjugated: this is the forward direction)
#pragma unroll
            for (int u = 0; u < KB; ++u) {
                const int k = kb * KB + u;
                if (k > m) break;
                const float2 ph = __ldg(tph + k);
                const float ar = pr[u] + qi[u], ai = pi[u] - qr[u], br = pr[u] - qi[u], bi = pi[u] + qr[u];
                const float2 a = make_float2(fmaf(ar, ph.x, ai * ph.y), fmaf(ai, ph.x, -ar * ph.y));
                const float2 b = make_float2(fmaf(br, ph.x, -bi * ph.y), fmaf(bi, ph.x, br * ph.y));
                if (k < m) o[(int64_t)k * f.inner] = make_float2(fmaf(a.x, z.x, a.y * z.y), fmaf(a.y, z.x, -a.x * z.y));
                if (k > 0)
                    o[(int64_t)(2 * m - k) * f.inner] = make_float2(fmaf(b.x, z.x, b.y * z.y), fmaf(b.y, z.x, -b.x * z.y));
            }
        }
    }
}

// 2m frequencies to n points; the tile's frequency pairs are folded once, then a thread takes
// one column and FV_J point pairs
__global__ void __launch_bounds__(FV_T) k_fold_inv(const float2* __restrict__ in, float2* __restrict__ out,
                                                   const float2* __restrict__ tfo, const float2* __restrict__ tph,
                                                   int m, int n, int njb, float zscale, FoldTile f) {
    extern __shared__ __align__(16) float2 psh[];
    const int m1 = m + 1, nh = n / 2, bufn = f.PB * f.ps, NJ = njb * FV_J;
    float2* T = psh;                                       // [m + 1][NJ], zero past n / 2
    float4* F = reinterpret_cast<float4*>(T + m1 * NJ);    // [m + 1][PB W]: a, b
    float2* buf = reinterpret_cast<float2*>(F + m1 * f.PB * f.W);
    for (int e = threadIdx.x; e < m1 * NJ; e += FV_T) {
        const int k = e / NJ, j = e - k * NJ;
        T[e] = j < nh ? tfo[j * m1 + k] : make_float2(0.f, 0.f);
    }
    int64_t t = blockIdx.x;
    if (t < f.ntiles) fold_issue(f, t, in, buf);
    sno_commit();
    for (int it = 0; t < f.ntiles; t += gridDim.x, ++it) {
        sno_wait_all();
        __syncthreads();   // the tile is there, the other buffer and F have been read
        if (t + gridDim.x < f.ntiles) fold_issue(f, t + gridDim.x, in, buf + ((it + 1) & 1) * bufn);
        sno_commit();
        int64_t p0;
        int np, i0, w;
        fold_shape(f, t, p0, np, i0, w);
        const int ncol = np * w;
        for (int e = threadIdx.x; e < m1 * ncol; e += FV_T) {
            const int k = e / ncol, col = e - k * ncol, pl = col / w, i = col - pl * w;
            const float2* x = buf + (it & 1) * bufn + pl * f.ps + i;
            const float2 g = k < m ? x[k * f.W] : make_float2(0.f, 0.f);
            const float2 h = k > 0 ? x[(2 * m - k) * f.W] : make_float2(0.f, 0.f);
            const float2 ph = __ldg(tph + k);
            const float gr = fmaf(g.x, ph.x, -g.y * ph.y), gi = fmaf(g.x, ph.y, g.y * ph.x);
            const float hr = fmaf(h.x, ph.x, h.y * ph.y), hi = fmaf(h.y, ph.x, -h.x * ph.y);
            const float2 z = fold_zphase(tph, m, i0 + i, zscale);
            const float ar = gr + hr, ai = gi + hi, br = gr - hr, bi = gi - hi;
            F[e] = make_float4(fmaf(ar, z.x, -ai * z.y), fmaf(ar, z.y, ai * z.x), fmaf(br, z.x, -bi * z.y),
                               fmaf(br, z.y, bi * z.x));
        }
        __syncthreads();
        for (int e = threadIdx.x; e < njb * ncol; e += FV_T) {
            const int jb = e / ncol, col = e - jb * ncol, pl = col / w, i = col - pl * w;
            float ur[FV_J], ui[FV_J], vr[FV_J], vi[FV_J];
#pragma unroll
            for (int u = 0; u < FV_J; ++u) ur[u] = ui[u] = vr[u] = vi[u] = 0.f;
            for (int k = 0; k < m1; ++k) {
                const float4 x = F[k * ncol + col];
                const float4* tk = reinterpret_cast<const float4*>(T + k * NJ + jb * FV_J);
#pragma unroll
                for (int u = 0; u < FV_J; u += 2) {
                    const float4 c = tk[u / 2];
                    ur[u] = fmaf(c.x, x.x, ur[u]);
                    ui[u] = fmaf(c.x, x.y, ui[u]);
                    vr[u] = fmaf(c.y, x.z, vr[u]);
                    vi[u] = fmaf(c.y, x.w, vi[u]);
                    ur[u + 1] = fmaf(c.z, x.x, ur[u + 1]);
                    ui[u + 1] = fmaf(c.z, x.y, ui[u + 1]);
                    vr[u + 1] = fmaf(c.w, x.z, vr[u + 1]);
                    vi[u + 1] = fmaf(c.w, x.w, vi[u + 1]);
                }
            }
            float2* o = out + (p0 + pl) * n * (int64_t)f.inner + i0 + i;
#pragma unroll
            for (int u = 0; u < FV_J; ++u) {
                const int j = jb * FV_J + u;
                if (j >= nh) break;
                o[(int64_t)j * f.inner] = make_float2(ur[u] + vi[u], ui[u] - vr[u]);
                o[(int64_t)(n - 1 - j) * f.inner] = make_float2(ur[u] - vi[u], ui[u] + vr[u]);
            }
        }
    }
}

// ---- inference, layer 0: the lift v0 = Wl u + bl has rank one in the channels, so its
// spectrum is V0[c][k] = Wl[c] U[k] + bl[c] O[k] (U the truncated transform of u, O that of
// the field of ones, separable: O = Sx[kx] Sy[ky] Sz[kz] with S the sums of the tables' rows)
// and the layer's mix G[o][k] = sum_c R[k][o][c] V0[c][k] = A[o][k] U[k] + Bc[o][k].
// cu[b][x][y][kz] = sum_z e^{-i kz (z - zc)} u[b][x][y][z], folded as in k_fold_fwd; a block stages the
// sums and differences of LU rows, a thread takes 4 rows and 2 modes
constexpr int LU = 32;
__global__ void __launch_bounds__(256) k_lift_u(const float* __restrict__ u, const float2* __restrict__ tfo,
                                                float2* __restrict__ cu, int64_t rows, int n, int m) {
    extern __shared__ __align__(16) float2 lsh[];
    const int nh = n / 2, ns = nh + 1, mh = (m + 1) / 2;
    float2* sd = lsh;               // [LU][n / 2 + 1]
    float2* tf = sd + LU * ns;      // [n / 2][m + 1]
    for (int e = threadIdx.x; e < nh * (m + 1); e += blockDim.x) tf[e] = tfo[e];
    const int64_t r0 = (int64_t)blockIdx.x * LU;
    const int nr = (int)min((int64_t)LU, rows - r0);
    for (int e = threadIdx.x; e < nr * nh; e += blockDim.x) {
        const int rq = e / nh, j = e - rq * nh;
        const float lo = u[(r0 + rq) * n + j], hi = u[(r0 + rq) * n + n - 1 - j];
        sd[rq * ns + j] = make_float2(hi + lo, hi - lo);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < ((nr + 3) / 4) * mh; e += blockDim.x) {
        const int rb = e / mh, k0 = e - rb * mh, k1 = min(k0 + mh, m - 1);
        float re[4][2] = {}, im[4][2] = {};
        for (int j = 0; j < nh; ++j) {
            const float2 t0 = tf[j * (m + 1) + k0], t1 = tf[j * (m + 1) + k1];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 x = sd[min(4 * rb + q, nr - 1) * ns + j];
                re[q][0] = fmaf(t0.x, x.x, re[q][0]);
                im[q][0] = fmaf(-t0.y, x.y, im[q][0]);
                re[q][1] = fmaf(t1.x, x.x, re[q][1]);
                im[q][1] = fmaf(-t1.y, x.y, im[q][1]);
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (4 * rb + q >= nr) break;
            cu[(r0 + 4 * rb + q) * m + k0] = make_float2(re[q][0], im[q][0]);
            if (k0 + mh < m) cu[(r0 + 4 * rb + q) * m + k0 + mh] = make_float2(re[q][1], im[q][1]);
        }
    }
}
// A[o][k] = sum_c R[k][o][c] Wl[c], Bc[o][k] = (sum_c R[k][o][c] bl[c]) O[k]; a block per mode, whose
// C x C weights lie together: a warp per row o, its lanes along c; O's three row sums once a block.
// Width 32, 12 modes: 99 -> 43 us (a thread per (o, k) read R with a stride of C^2).
constexpr int M0_T = 256;
__device__ __forceinline__ float warp_sum(float a) {
    for (int o = 16; o > 0; o /= 2) a += __shfl_xor_sync(0xffffffffu, a, o);
    return a;
}
template <class TR>
__global__ void __launch_bounds__(M0_T) k_mix0_prep(const TR* __restrict__ Rr, const TR* __restrict__ Ri,
                                                    const float* __restrict__ Wl, const float* __restrict__ bl,
                                                    const float2* __restrict__ tyf, const float2* __restrict__ tzf,
                                                    int C, int64_t K, int n, int m, float2* __restrict__ A,
                                                    float2* __restrict__ Bc) {
    __shared__ float2 sums[3];
    const int64_t k = blockIdx.x;
    const int M2 = 2 * m, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (w < 3) {
        const int j = (int)(w == 0 ? k / ((int64_t)M2 * m) : w == 1 ? (k / m) % M2 : k % m);
        const float2* T = (w < 2 ? tyf : tzf) + j * n;
        float sr = 0.f, si = 0.f;
        for (int q = lane; q < n; q += 32) {
            sr += T[q].x;
            si += T[q].y;
        }
        sr = warp_sum(sr);
        si = warp_sum(si);
        if (lane == 0) sums[w] = make_float2(sr, si);
    }
    __syncthreads();
    const float2 sx = sums[0], sy = sums[1], sz = sums[2];
    const float2 sxy = make_float2(sx.x * sy.x - sx.y * sy.y, sx.x * sy.y + sx.y * sy.x);
    const float2 O = make_float2(sxy.x * sz.x - sxy.y * sz.y, sxy.x * sz.y + sxy.y * sz.x);
    for (int o = w; o < C; o += M0_T / 32) {
        float ar = 0.f, ai = 0.f, br = 0.f, bi = 0.f;
        for (int c = lane; c < C; c += 32) {
            const int64_t ri = (k * C + o) * C + c;
            const float xr = (float)Rr[ri], xi = (float)Ri[ri];
            ar = fmaf(xr, Wl[c], ar);
            ai = fmaf(xi, Wl[c], ai);
            br = fmaf(xr, bl[c], br);
            bi = fmaf(xi, bl[c], bi);
        }
        ar = warp_sum(ar);
        ai = warp_sum(ai);
        br = warp_sum(br);
        bi = warp_sum(bi);
        if (lane == 0) {
            A[(int64_t)o * K + k] = make_float2(ar, ai);
            Bc[(int64_t)o * K + k] = make_float2(br * O.x - bi * O.y, br * O.y + bi * O.x);
        }
    }
}
// G[b][o][k] = A[o][k] U[b][k] + Bc[o][k]
__global__ void k_mix0(const float2* __restrict__ U, const float2* __restrict__ A, const float2* __restrict__ Bc,
                       float2* __restrict__ G, int B, int C, int64_t K) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (int64_t)B * C * K) return;
    const int64_t k = e % K, ok = e % ((int64_t)C * K), b = e / ((int64_t)C * K);
    const float2 a = A[ok], c = Bc[ok], x = U[b * K + k];
    G[e] = make_float2(fmaf(a.x, x.x, fmaf(-a.y, x.y, c.x)), fmaf(a.x, x.y, fmaf(a.y, x.x, c.y)));
}

// Channel mix per mode, MB modes and up to MIX_B fields (blockIdx.y) per block: G[b][o][k] =
// sum_c R[k][o][c] V[b][c][k] (adj = 1: G[b][c][k] = sum_o conj(R[k][o][c]) V[b][o][k]). A thread takes
// 4 outputs x 4 fields (two pairs of each, so that the lanes' 16-byte loads are contiguous): 64 FMAs for 4
// of them, where one output a thread was bound by its two loads for 4 FMAs. R is staged as complex
// [kk][in][C + 2], V as [kk][c][BS] over a whole number of pairs; G takes V's place on the way out.
// One GB300, width 32, 12 modes, 32 fields: 199 -> 139 us a layer.
constexpr int MIX_B = 32;
struct MixDims {
    int MB, BT, BS;   // modes and fields a block, row of V
    size_t smem;
};
static MixDims mix_dims(int C, int B) {
    MixDims d;
    d.BT = std::min(MIX_B, (B + 3) & ~3);
    d.BS = d.BT + 2;
    const size_t per = ((size_t)C * (C + 2) + C * d.BS + 8) * sizeof(float2);   // (52 KB at C = 64 and 32 fields)
    // one item a thread (at most 128 a mode), two blocks an SM
    d.MB = (int)std::max<size_t>(1, std::min<size_t>({16, (size_t)(256 / ((C / 4) * (d.BT / 4))), (96u << 10) / per}));
    d.smem = d.MB * per;
    return d;
}
template <class TR>
__global__ void __launch_bounds__(256) k_mix(const TR* __restrict__ Rr, const TR* __restrict__ Ri,
                                             const float2* __restrict__ V, float2* __restrict__ G, int B, int C,
                                             int64_t K, int adj, MixDims d) {
    extern __shared__ __align__(16) float2 msh[];
    const int CS = C + 2, VS = C * d.BS + 8;             // rows of R, modes of V
    float2* Rs = msh;                                    // [MB][C][C + 2]
    float2* Vs = msh + (size_t)d.MB * C * CS;            // [MB][C][BS]
    const int64_t k0 = (int64_t)blockIdx.x * d.MB;
    const int nk = (int)min((int64_t)d.MB, K - k0);
    const int b0 = blockIdx.y * d.BT, nb = min(d.BT, B - b0);
    for (int e = threadIdx.x; e < nk * C * C; e += blockDim.x) {
        const int c = e % C, o = (e / C) % C, kk = e / (C * C);
        const int64_t ri = k0 * C * C + e;
        const float xr = (float)Rr[ri], xi = (float)Ri[ri];
        Rs[(kk * C + (adj ? o : c)) * CS + (adj ? c : o)] = make_float2(xr, adj ? -xi : xi);
    }
    for (int e = threadIdx.x; e < d.BT * C * nk; e += blockDim.x) {
        const int kk = e % nk, b = (e / nk) % d.BT, c = e / (nk * d.BT);
        Vs[kk * VS + c * d.BS + b] = b < nb ? V[((int64_t)(b0 + b) * C + c) * K + k0 + kk] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    const int nob = C / 4, nbb = d.BT / 4;
    const int ob = threadIdx.x % nob, bb = (threadIdx.x / nob) % nbb, kk = threadIdx.x / (nob * nbb);
    float2 acc[4][4] = {};   // [output][field]: 2 ob + {0, 1}, C / 2 + 2 ob + {0, 1}; the fields alike
    if (kk < nk) {
        const float2* r = Rs + kk * C * CS + 2 * ob;
        const float2* x = Vs + kk * VS + 2 * bb;
        for (int c = 0; c < C; ++c, r += CS, x += d.BS) {
            const float4 r0 = *reinterpret_cast<const float4*>(r), r1 = *reinterpret_cast<const float4*>(r + C / 2);
            const float4 x0 = *reinterpret_cast<const float4*>(x), x1 = *reinterpret_cast<const float4*>(x + d.BT / 2);
            const float2 a[4] = {{r0.x, r0.y}, {r0.z, r0.w}, {r1.x, r1.y}, {r1.z, r1.w}};
            const float2 v[4] = {{x0.x, x0.y}, {x0.z, x0.w}, {x1.x, x1.y}, {x1.z, x1.w}};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    acc[i][j].x = fmaf(a[i].x, v[j].x, fmaf(-a[i].y, v[j].y, acc[i][j].x));
                    acc[i][j].y = fmaf(a[i].x, v[j].y, fmaf(a[i].y, v[j].x, acc[i][j].y));
                }
        }
    }
    __syncthreads();   // V has been read
    if (kk < nk)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float2* o = Vs + kk * VS + ((i < 2 ? 0 : C / 2) + 2 * ob + (i & 1)) * d.BS + 2 * bb;
            *reinterpret_cast<float4*>(o) = make_float4(acc[i][0].x, acc[i][0].y, acc[i][1].x, acc[i][1].y);
            *reinterpret_cast<float4*>(o + d.BT / 2) = make_float4(acc[i][2].x, acc[i][2].y, acc[i][3].x, acc[i][3].y);
        }
    __syncthreads();
    for (int e = threadIdx.x; e < d.BT * C * nk; e += blockDim.x) {
        const int q = e % nk, b = (e / nk) % d.BT, o = e / (nk * d.BT);
        if (b < nb) G[((int64_t)(b0 + b) * C + o) * K + k0 + q] = Vs[q * VS + o * d.BS + b];
    }
}

// dR[k][o][c] = sum_b dG[b][o][k] conj(V[b][c][k]) (real and imaginary planes, stored)
__global__ void __launch_bounds__(256) k_mix_grad(const float2* __restrict__ dG, const float2* __restrict__ V,
                                                  float* dRr, float* dRi, int B, int C, int64_t K, int MB) {
    extern __shared__ float2 msh[];
    float2* Gs = msh;                           // [B][MB][C]
    float2* Vs = msh + (size_t)B * MB * C;      // [B][MB][C]
    const int64_t k0 = (int64_t)blockIdx.x * MB;
    const int nk = (int)min((int64_t)MB, K - k0);
    for (int e = threadIdx.x; e < B * C * nk; e += blockDim.x) {
        const int kk = e % nk, c = (e / nk) % C, b = e / (nk * C);
        const int64_t gi = ((int64_t)b * C + c) * K + k0 + kk;
        Gs[((size_t)b * MB + kk) * C + c] = dG[gi];
        Vs[((size_t)b * MB + kk) * C + c] = V[gi];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < nk * C * C; e += blockDim.x) {
        const int c = e % C, o = (e / C) % C, kk = e / (C * C);
        float re = 0.f, im = 0.f;
        for (int b = 0; b < B; ++b) {
            const float2 g = Gs[((size_t)b * MB + kk) * C + o];
            const float2 x = Vs[((size_t)b * MB + kk) * C + c];
            re = fmaf(g.x, x.x, fmaf(g.y, x.y, re));
            im = fmaf(g.y, x.x, fmaf(-g.x, x.y, im));
        }
        const int64_t ri = ((k0 + kk) * C + o) * C + c;
        dRr[ri] = re;
        dRi[ri] = im;
    }
}

// z-row kernels: shared-memory fields as [rows][n + 1] floats and tables as [rows][cols + 1]
// float2 (odd strides keep column access free of bank conflicts); the float2 region starts
// on an 8-byte boundary. Inner products are register-blocked (several outputs per thread
// share each shared-memory load).

// out[c][kz] = sum_z tf[kz][z] X[c][z] for c < C, kz < m (X real [C][n + 1], tf [m][n + 1]);
// a thread takes one c and the pair kz, kz + mh. Written to dst + (c * rs) + kz.
__device__ __forceinline__ void zfwd_rows(const float* X, const float2* tf, int C, int n, int m, float2* dst,
                                          int64_t rs) {
    const int ns = n + 1, mh = (m + 1) / 2;
    for (int e = threadIdx.x; e < C * mh; e += blockDim.x) {
        const int k0 = e % mh, c = e / mh;
        const int k1 = k0 + mh;
        const bool h1 = k1 < m;
        const float2* t0 = tf + k0 * ns;
        const float2* t1 = tf + (h1 ? k1 : k0) * ns;
        const float* x = X + c * ns;
        float r0 = 0.f, i0 = 0.f, r1 = 0.f, i1 = 0.f;
        for (int zz = 0; zz < n; ++zz) {
            const float xv = x[zz];
            const float2 a = t0[zz], b = t1[zz];
            r0 = fmaf(a.x, xv, r0);
            i0 = fmaf(a.y, xv, i0);
            r1 = fmaf(b.x, xv, r1);
            i1 = fmaf(b.y, xv, i1);
        }
        dst[c * rs + k0] = make_float2(r0, i0);
        if (h1) dst[c * rs + k1] = make_float2(r1, i1);
    }
}

// forward, layer input side: v0 = Wl u + bl (lift) and its last-axis DFT cz = Tzf v0
__global__ void __launch_bounds__(ZR_T) k_lift_z(const float* __restrict__ u, const float* __restrict__ Wl,
                                                 const float* __restrict__ bl, float* __restrict__ v0,
                                                 float2* __restrict__ cz, const float2* __restrict__ Tzf, int B, int C,
                                                 int n, int m) {
    extern __shared__ float zsh[];
    const int ns = n + 1;
    float* vs = zsh;                                                 // [C][n + 1]
    float* us = vs + C * ns;                                         // [n]
    size_t fo = (size_t)(C * ns + n);
    fo = (fo + 1) & ~(size_t)1;
    float2* tf = reinterpret_cast<float2*>(zsh + fo);                // [m][n + 1]
    for (int e = threadIdx.x; e < m * n; e += blockDim.x) tf[(e / n) * ns + e % n] = Tzf[e];
    const int64_t n2 = (int64_t)n * n, rows = (int64_t)B * n2, np3 = n2 * n;
    for (int64_t r = (int64_t)blockIdx.x * ZR_RG; r < min(rows, (int64_t)(blockIdx.x + 1) * ZR_RG); ++r) {
        const int64_t b = r / n2, xy = r % n2;
        __syncthreads();
        for (int e = threadIdx.x; e < n; e += blockDim.x) us[e] = u[b * np3 + xy * n + e];
        __syncthreads();
        for (int e = threadIdx.x; e < C * n; e += blockDim.x) {
            const int c = e / n, zz = e % n;
            const float val = fmaf(Wl[c], us[zz], bl[c]);
            vs[c * ns + zz] = val;
            v0[((b * C + c) * n2 + xy) * n + zz] = val;
        }
        __syncthreads();
        zfwd_rows(vs, tf, C, n, m, cz + (b * C * n2 + xy) * m, n2 * m);
    }
}

// Forward, layer output side: persistent blocks over R row groups (b, x, y) at a time,
// z = Re(sum_kz g e^{i kz (z - zc)}) + W v + b with v_next = GELU(z) (or z for the last layer), then the
// next layer's cz = sum_z e^{-i kz (z - zc)} v_next or the projection y; z itself is stored when zio is
// given (training). Layer 0 of the inference takes W v0 + b = (W Wl) u + (W bl + b) from u.
// The transforms are folded about the row's centre zc = (n - 1) / 2 as in k_fold_fwd (half the FMAs; the
// phases e^{+-i kz zc} and the weights are in the spectra). A thread computes 8 channels x 4 point pairs:
// the pairs' shared cosine and sine sums become the two points' values in the same 64 registers, 16 FMAs a
// 16-byte shared load in W v, and their sums and differences go to shared memory ready for the next
// transform (4 channels x 3 modes a thread, lanes 8 x 4 so that a warp reads few distinct words). Three
// blocks an SM cover each other's loads: bound by FP32 issue (FMAs and GELU's erf).
// One GB300, 32 fields of 64^3 at width 32 and 12 modes: layers 1 and 2 2.28 -> 1.25 ms each,
// the last with the projection 2.27 -> 1.92 ms, layer 0 0.87 ms; the four launches 6.83 -> 5.3 ms.
// The backward pass runs the same rows with W transposed: dv = Re(sum_kz g e^{i kz (z - zc)}) + W^T dz, then
// dz_prev = dv GELU'(z_prev) and its transform (layer 0: dv alone, zio and cznext null).
constexpr int ZF_T = 128;
enum { ZR_FWD = 0, ZR_PROJ = 1, ZR_BWD = 2 };   // k_zrow's MODE; zio: z written (forward), z_prev read (backward)
struct ZRowDims {
    int nh, nhp, nzb, nob, CP, CG, nz4, TS, PP, R;   // (see zrow_dims)
    size_t smem;
};
static ZRowDims zrow_dims(int n, int C, int m, int P, bool proj) {
    ZRowDims d;
    d.nh = n / 2;
    d.nhp = (d.nh + 3) & ~3;       // point pairs, in blocks of 4
    d.nzb = d.nhp / 4;
    d.nob = (C + 7) / 8;           // channel blocks
    d.CP = 8 * d.nob;
    d.CG = d.CP + 2;               // row of a mode's spectra (2-way conflicts in the transposing copy)
    d.nz4 = n + 4;
    d.TS = d.nhp + 4;              // row of the cosine and sine tables
    d.PP = (P + 7) & ~7;
    d.R = ZF_T / (d.nob * d.nzb);  // one tile a thread (n <= 128 and C <= 64: at least one row)
    size_t f = (size_t)d.R * C * d.nz4 + (size_t)C * d.CP + 2 * d.CP + 2 * (size_t)m * d.TS +
               2 * (size_t)d.R * m * d.CG;
    f = (f + 3) & ~(size_t)3;      // (the projection's rows are read in 16-byte pieces)
    if (proj) f += (size_t)C * d.PP + 2 * d.PP + (size_t)d.R * (d.PP / 8) * n;
    d.smem = f * 4;
    return d;
}
__device__ __forceinline__ float4 rev4(float4 a) { return make_float4(a.w, a.z, a.y, a.x); }
template <int MODE>
__global__ void __launch_bounds__(ZF_T, 3) k_zrow(const float2* __restrict__ gy, const float* __restrict__ v,
                                                  const float* __restrict__ W, const float* __restrict__ bias,
                                                  const float2* __restrict__ tfo, float* __restrict__ zio,
                                                  float* __restrict__ vnext, float2* __restrict__ cznext,
                                                  const float* __restrict__ Q1, const float* __restrict__ q1,
                                                  const float* __restrict__ Q2, const float* __restrict__ q2,
                                                  float* __restrict__ y, const float* __restrict__ u0,
                                                  const float* __restrict__ Wl, const float* __restrict__ bl, int rows,
                                                  int C, int n, int m, int P, ZRowDims d) {
    constexpr bool PROJ = MODE == ZR_PROJ, BWD = MODE == ZR_BWD;
    extern __shared__ __align__(16) float zsh[];
    float* vs = zsh;                                              // [R][C][n + 4]
    float* Ws = vs + d.R * C * d.nz4;                             // [C][CP], transposed
    float* bs = Ws + C * d.CP;                                    // [CP] bias, [CP] W Wl
    float* tc = bs + 2 * d.CP;                                    // [m][TS] cosines, then sines
    float* tn = tc + m * d.TS;
    float2* gs = reinterpret_cast<float2*>(tn + m * d.TS);        // [R][m][CG]
    float* Qs = zsh + (((d.R * C * d.nz4 + C * d.CP + 2 * d.CP + 2 * m * d.TS + 2 * d.R * m * d.CG) + 3) & ~3);
    float* pq = Qs + C * d.PP;                                    // [C][PP] Q1 transposed; q1, Q2
    float* ys = pq + 2 * d.PP;                                    // [R][PP / 8][n]
    const int tid = threadIdx.x, n4 = n / 4, n2 = n * n;
    for (int e = tid; e < C * d.CP; e += ZF_T) {
        const int c = e / d.CP, o = e - c * d.CP;
        Ws[e] = o < C ? W[BWD ? c * C + o : o * C + c] : 0.f;
    }
    for (int o = tid; o < d.CP; o += ZF_T) {
        float w0 = !BWD && o < C ? bias[o] : 0.f, w1 = 0.f;
        if (u0 && o < C)
            for (int c = 0; c < C; ++c) {
                w1 = fmaf(W[o * C + c], Wl[c], w1);
                w0 = fmaf(W[o * C + c], bl[c], w0);
            }
        bs[o] = w0;
        bs[d.CP + o] = w1;
    }
    for (int e = tid; e < m * d.nhp; e += ZF_T) {   // (the last block's pairs past n / 2 are mirrored ones)
        const int k = e / d.nhp, j = e - k * d.nhp;
        const float2 t = tfo[(j < d.nh ? j : n - 1 - j) * (m + 1) + k];
        tc[k * d.TS + j] = t.x;
        tn[k * d.TS + j] = j < d.nh ? t.y : -t.y;
    }
    if (PROJ) {
        for (int e = tid; e < C * d.PP; e += ZF_T) {
            const int c = e / d.PP, p = e - c * d.PP;
            Qs[e] = p < P ? Q1[p * C + c] : 0.f;
        }
        for (int p = tid; p < d.PP; p += ZF_T) {
            pq[p] = p < P ? q1[p] : 0.f;
            pq[d.PP + p] = p < P ? Q2[p] : 0.f;
        }
    }
    const bool aligned = (reinterpret_cast<uintptr_t>(u0) & 15) == 0;   // (a caller's field may lie anywhere)
    // lanes of the copies: 16-byte pieces of a row and modes of a spectrum, in powers of two
    const int lv = 32 - __clz(n4 - 1), lm = m > 1 ? 32 - __clz(m - 1) : 0;
    const int zb = tid % d.nzb, ob = (tid / d.nzb) % d.nob, rg = tid / (d.nzb * d.nob);
    const int z0 = 4 * zb, z1 = n - 4 - z0, o0 = 8 * ob;
    for (int r0 = blockIdx.x * d.R; r0 < rows; r0 += gridDim.x * d.R) {
        const int nr = min(d.R, rows - r0);
        __syncthreads();   // the previous rows have been read
        for (int rr = 0; rr < nr; ++rr) {
            const int b = (r0 + rr) / n2, xy = (r0 + rr) - b * n2;
            const int q = tid & ((1 << lv) - 1);
            if (u0) {
                float* row = vs + rr * C * d.nz4;
                const float* src = u0 + (int64_t)(r0 + rr) * n;
                if (aligned) {
                    if (tid < n4) sno_cp16(row + 4 * tid, src + 4 * tid);
                } else {
                    for (int z = tid; z < n; z += ZF_T) row[z] = src[z];
                }
            } else if (q < n4) {
                for (int c = tid >> lv; c < C; c += ZF_T >> lv)
                    sno_cp16(vs + (rr * C + c) * d.nz4 + 4 * q, v + (((int64_t)b * C + c) * n2 + xy) * n + 4 * q);
            }
            const int kz = tid & ((1 << lm) - 1);
            if (kz < m)
                for (int c = tid >> lm; c < C; c += ZF_T >> lm)
                    sno_cp8(gs + (rr * m + kz) * d.CG + c, gy + (((int64_t)b * C + c) * n2 + xy) * m + kz);
        }
        sno_commit();
        sno_wait_all();
        __syncthreads();
        float lo[8][4], hi[8][4];
        if (rg < nr) {
#pragma unroll
            for (int j = 0; j < 8; ++j)
#pragma unroll
                for (int i = 0; i < 4; ++i) lo[j][i] = hi[j][i] = 0.f;
            const float4* g = reinterpret_cast<const float4*>(gs + rg * m * d.CG + o0);
            for (int kz = 0; kz < m; ++kz, g += d.CG / 2) {
                const float4 c4 = *reinterpret_cast<const float4*>(tc + kz * d.TS + z0);
                const float4 s4 = *reinterpret_cast<const float4*>(tn + kz * d.TS + z0);
                const float cv[4] = {c4.x, c4.y, c4.z, c4.w}, sv[4] = {s4.x, s4.y, s4.z, s4.w};
#pragma unroll
                for (int j = 0; j < 8; j += 2) {
                    const float4 x = g[j / 2];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        lo[j][i] = fmaf(cv[i], x.x, lo[j][i]);
                        hi[j][i] = fmaf(sv[i], x.y, hi[j][i]);
                        lo[j + 1][i] = fmaf(cv[i], x.z, lo[j + 1][i]);
                        hi[j + 1][i] = fmaf(sv[i], x.w, hi[j + 1][i]);
                    }
                }
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {   // points z0 + i (at -t) and n - 1 - z0 - i (at +t)
                const float bj = bs[o0 + j];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float a = lo[j][i] + bj, b = hi[j][i];
                    lo[j][i] = a + b;
                    hi[j][i] = a - b;
                }
            }
            const float* vr = vs + rg * C * d.nz4;
            const float* wr = (u0 ? bs + d.CP : Ws) + o0;
            const int nc = u0 ? 1 : C;
            for (int c = 0; c < nc; ++c, vr += d.nz4, wr += d.CP) {
                const float4 a = *reinterpret_cast<const float4*>(vr + z0);
                const float4 b = rev4(*reinterpret_cast<const float4*>(vr + z1));
                const float4 w0 = *reinterpret_cast<const float4*>(wr), w1 = *reinterpret_cast<const float4*>(wr + 4);
                const float wv[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
                const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
                for (int j = 0; j < 8; ++j)
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        lo[j][i] = fmaf(wv[j], av[i], lo[j][i]);
                        hi[j][i] = fmaf(wv[j], bv[i], hi[j][i]);
                    }
            }
        }
        __syncthreads();   // every tile is in registers: v_next (or its sums and differences) replaces v
        if (rg < nr) {
            const int b = (r0 + rg) / n2, xy = (r0 + rg) - b * n2;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                if (o0 + j >= C) break;
                const int64_t gi = (((int64_t)b * C + o0 + j) * n2 + xy) * n;
                float4 a = make_float4(lo[j][0], lo[j][1], lo[j][2], lo[j][3]);
                float4 h = make_float4(hi[j][0], hi[j][1], hi[j][2], hi[j][3]);
                if (BWD) {
                    if (zio) {
                        const float4 x = *reinterpret_cast<const float4*>(zio + gi + z0);
                        const float4 w = rev4(*reinterpret_cast<const float4*>(zio + gi + z1));
                        a = make_float4(a.x * gelu_d(x.x), a.y * gelu_d(x.y), a.z * gelu_d(x.z), a.w * gelu_d(x.w));
                        h = make_float4(h.x * gelu_d(w.x), h.y * gelu_d(w.y), h.z * gelu_d(w.z), h.w * gelu_d(w.w));
                    }
                } else if (zio) {
                    *reinterpret_cast<float4*>(zio + gi + z0) = a;
                    *reinterpret_cast<float4*>(zio + gi + z1) = rev4(h);
                }
                if (MODE == ZR_FWD) {
                    a = make_float4(gelu_f(a.x), gelu_f(a.y), gelu_f(a.z), gelu_f(a.w));
                    h = make_float4(gelu_f(h.x), gelu_f(h.y), gelu_f(h.z), gelu_f(h.w));
                }
                if (vnext) {
                    *reinterpret_cast<float4*>(vnext + gi + z0) = a;
                    *reinterpret_cast<float4*>(vnext + gi + z1) = rev4(h);
                }
                float* sr = vs + (rg * C + o0 + j) * d.nz4;
                if (!PROJ) {   // sums at [0, nhp), differences at [nhp, 2 nhp), zero past n / 2
                    const bool two = z0 + 4 > d.nh;   // (n / 2 is even)
                    *reinterpret_cast<float4*>(sr + z0) =
                        make_float4(h.x + a.x, h.y + a.y, two ? 0.f : h.z + a.z, two ? 0.f : h.w + a.w);
                    *reinterpret_cast<float4*>(sr + d.nhp + z0) =
                        make_float4(h.x - a.x, h.y - a.y, two ? 0.f : h.z - a.z, two ? 0.f : h.w - a.w);
                } else {
                    *reinterpret_cast<float4*>(sr + z0) = a;
                    *reinterpret_cast<float4*>(sr + z1) = rev4(h);
                }
            }
        }
        __syncthreads();
        if (!PROJ && cznext) {   // channels cg + ncg i, modes 3 kb + i
            const int ncg = C / 4, nkb = (m + 2) / 3;
            for (int e = tid; e < nr * ncg * nkb; e += ZF_T) {
                const int cg = e % ncg, kb = (e / ncg) % nkb, rq = e / (ncg * nkb);
                int kc[3];
#pragma unroll
                for (int i = 0; i < 3; ++i) kc[i] = min(3 * kb + i, m - 1) * d.TS;
                float re[4][3] = {}, im[4][3] = {};
                const float* vr = vs + (rq * C + cg) * d.nz4;
                for (int j = 0; j < d.nhp; j += 4) {
                    float4 x[4], w[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        x[i] = *reinterpret_cast<const float4*>(vr + i * ncg * d.nz4 + j);
                        w[i] = *reinterpret_cast<const float4*>(vr + i * ncg * d.nz4 + d.nhp + j);
                    }
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        const float4 c4 = *reinterpret_cast<const float4*>(tc + kc[k] + j);
                        const float4 s4 = *reinterpret_cast<const float4*>(tn + kc[k] + j);
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            re[i][k] = fmaf(c4.x, x[i].x, fmaf(c4.y, x[i].y, fmaf(c4.z, x[i].z, fmaf(c4.w, x[i].w, re[i][k]))));
                            im[i][k] = fmaf(s4.x, w[i].x, fmaf(s4.y, w[i].y, fmaf(s4.z, w[i].z, fmaf(s4.w, w[i].w, im[i][k]))));
                        }
                    }
                }
                const int b = (r0 + rq) / n2, xy = (r0 + rq) - b * n2;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float2* o = cznext + (((int64_t)b * C + cg + i * ncg) * n2 + xy) * m + 3 * kb;
#pragma unroll
                    for (int k = 0; k < 3; ++k)
                        if (3 * kb + k < m) o[k] = make_float2(re[i][k], -im[i][k]);
                }
            }
        }
        if (PROJ) {   // projection: 8 rows of Q1 x 8 points a thread, partial sums per row block
            const int npb = d.PP / 8, nq = (n4 + 1) / 2;
            for (int e = tid; e < nr * npb * nq; e += ZF_T) {
                const int q = e % nq, pb = (e / nq) % npb, rq = e / (nq * npb);
                const int za = 4 * q, zc = 4 * min(q + nq, n4 - 1), p0 = 8 * pb;
                float a[8][8];
#pragma unroll
                for (int j = 0; j < 8; ++j)
#pragma unroll
                    for (int i = 0; i < 8; ++i) a[j][i] = pq[p0 + j];
                const float* vr = vs + rq * C * d.nz4;
                const float* qr = Qs + p0;
                for (int c = 0; c < C; ++c, vr += d.nz4, qr += d.PP) {
                    const float4 xa = *reinterpret_cast<const float4*>(vr + za);
                    const float4 xc = *reinterpret_cast<const float4*>(vr + zc);
                    const float4 w0 = *reinterpret_cast<const float4*>(qr), w1 = *reinterpret_cast<const float4*>(qr + 4);
                    const float wv[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
                    const float xv[8] = {xa.x, xa.y, xa.z, xa.w, xc.x, xc.y, xc.z, xc.w};
#pragma unroll
                    for (int j = 0; j < 8; ++j)
#pragma unroll
                        for (int i = 0; i < 8; ++i) a[j][i] = fmaf(wv[j], xv[i], a[j][i]);
                }
                float part[8] = {};
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float w = pq[d.PP + p0 + j];
#pragma unroll
                    for (int i = 0; i < 8; ++i) part[i] = fmaf(w, gelu_f(a[j][i]), part[i]);
                }
                float* yo = ys + (rq * npb + pb) * n;
                *reinterpret_cast<float4*>(yo + za) = make_float4(part[0], part[1], part[2], part[3]);
                *reinterpret_cast<float4*>(yo + zc) = make_float4(part[4], part[5], part[6], part[7]);
            }
            __syncthreads();
            for (int e = tid; e < nr * n; e += ZF_T) {
                const int rq = e / n, zz = e - rq * n;
                float sum = 0.f;
                for (int pb = 0; pb < npb; ++pb) sum += ys[(rq * npb + pb) * n + zz];
                y[(int64_t)(r0 + rq) * n + zz] = q2[0] + sum;   // (b n^3 + xy n + z)
            }
        }
    }
}

// ---- backward: the weights' gradients are sums over all points, C x C or P x C at a time. Persistent
// blocks walk chunks of GP points with 4 x 4 tiles of the sum in registers; where the tiles are fewer
// than the threads, the chunk's points are split over 2^k lanes a tile (added by shuffles at the end),
// and a block adds its sums to the gradient once (the row-by-row form added 16384 times 4 rows' sums).
constexpr int GP = 64;            // points a chunk (n^3 is a multiple of 64); a row in shared memory has 4 more
constexpr int GPS = GP + 4;
constexpr int GD_T = 256;
__device__ __forceinline__ int grad_splits(int tiles) {   // lanes a tile, a power of two up to GP / 4
    int S = GP / 4;
    while (S > 1 && tiles * S > GD_T) S /= 2;
    return S;
}
// acc[4 i + j] += sum over the lane's points of X[i][.] Y[j][.]
template <int NP>
__device__ __forceinline__ void grad_tile(const float* X, const float* Y, int s, int S, float* acc) {
    constexpr int GPS = NP + 4;
    for (int q = 4 * s; q < NP; q += 4 * S) {
        float4 x[4], w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            x[i] = *reinterpret_cast<const float4*>(X + i * GPS + q);
            w[i] = *reinterpret_cast<const float4*>(Y + i * GPS + q);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
                acc[4 * i + j] = fmaf(x[i].x, w[j].x, fmaf(x[i].y, w[j].y, fmaf(x[i].z, w[j].z, fmaf(x[i].w, w[j].w, acc[4 * i + j]))));
    }
}
__device__ __forceinline__ float lane_sum(float a, int S) {   // over S consecutive lanes (a power of two)
    for (int o = 1; o < S; o *= 2) a += __shfl_xor_sync(0xffffffffu, a, o);
    return a;
}

// dW[o][c] += sum_pt dz[o][pt] v[c][pt], db[o] += sum_pt dz[o][pt]: reads both fields once, the next
// chunk on its way. Width 16, 4 fields of 64^3: 134 MB, 60 us at worst (4 layers 235 us).
__global__ void __launch_bounds__(GD_T) k_grad_w(const float* __restrict__ dz, const float* __restrict__ v, float* gW,
                                                 float* gb, int B, int C, int64_t np3) {
    extern __shared__ __align__(16) float zsh[];   // two buffers of dz [C][GPS], v [C][GPS]
    const int nt = C / 4, tiles = nt * nt, S = grad_splits(tiles);
    const int s = threadIdx.x % S, t = threadIdx.x / S;
    const int i0 = 4 * (t / nt), j0 = 4 * (t % nt);
    const int64_t per = np3 / GP, nchunk = per * B;
    auto issue = [&](int64_t k, float* dst) {
        const int64_t b = k / per, p = (k - b * per) * GP;
        const int q = threadIdx.x % (GP / 4);
        for (int c = threadIdx.x / (GP / 4); c < C; c += GD_T / (GP / 4)) {
            const int64_t g = (b * C + c) * np3 + p + 4 * q;
            sno_cp16(dst + c * GPS + 4 * q, dz + g);
            sno_cp16(dst + (C + c) * GPS + 4 * q, v + g);
        }
    };
    float acc[16], ab[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[i] = 0.f;
    int64_t k = blockIdx.x;
    if (k < nchunk) issue(k, zsh);
    sno_commit();
    for (int it = 0; k < nchunk; k += gridDim.x, ++it) {
        sno_wait_all();
        __syncthreads();   // the chunk is there, and the other buffer has been read
        if (k + gridDim.x < nchunk) issue(k + gridDim.x, zsh + ((it + 1) & 1) * 2 * C * GPS);
        sno_commit();
        const float* X = zsh + (it & 1) * 2 * C * GPS;
        if (t < tiles) {
            grad_tile<GP>(X + i0 * GPS, X + (C + j0) * GPS, s, S, acc);
            if (j0 == 0)
                for (int q = 4 * s; q < GP; q += 4 * S)
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float4 x = *reinterpret_cast<const float4*>(X + (i0 + i) * GPS + q);
                        ab[i] += (x.x + x.y) + (x.z + x.w);
                    }
        }
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[i] = lane_sum(acc[i], S);
#pragma unroll
    for (int i = 0; i < 4; ++i) ab[i] = lane_sum(ab[i], S);
    if (t >= tiles || s) return;
#pragma unroll
    for (int i = 0; i < 16; ++i) atomicAdd(gW + (i0 + i / 4) * C + j0 + i % 4, acc[i]);
    if (j0 == 0)
#pragma unroll
        for (int i = 0; i < 4; ++i) atomicAdd(gb + i0 + i, ab[i]);
}

// the lift's gradients: dWl[c] += sum_pt dv[c][pt] u[pt], dbl[c] += sum_pt dv[c][pt]; blockIdx.y = c
__global__ void __launch_bounds__(256) k_grad_lift(const float* __restrict__ dv, const float* __restrict__ u,
                                                   float* gWl, float* gbl, int B, int C, int64_t np3) {
    __shared__ float red[2][8];
    const int c = blockIdx.y;
    float sw = 0.f, sb = 0.f;
    for (int b = 0; b < B; ++b) {
        const float4* d = reinterpret_cast<const float4*>(dv + ((int64_t)b * C + c) * np3);
        const float* x = u + b * np3;
        for (int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x; e < np3 / 4; e += (int64_t)gridDim.x * 256) {
            const float4 a = d[e];
            sw = fmaf(a.x, x[4 * e], fmaf(a.y, x[4 * e + 1], fmaf(a.z, x[4 * e + 2], fmaf(a.w, x[4 * e + 3], sw))));
            sb += (a.x + a.y) + (a.z + a.w);
        }
    }
    sw = lane_sum(sw, 32);
    sb = lane_sum(sb, 32);
    if (threadIdx.x % 32 == 0) {
        red[0][threadIdx.x / 32] = sw;
        red[1][threadIdx.x / 32] = sb;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        float a = 0.f;
        for (int w = 0; w < 8; ++w) a += red[threadIdx.x][w];
        atomicAdd((threadIdx.x ? gbl : gWl) + c, a);
    }
}

// backward of the projection: a = Q1 v_L + q1, h = GELU(a), da = dy Q2 GELU'(a), dz_{L-1} = Q1^T da, and the
// sums dQ1 = da v_L, dq1 = da, dQ2 = dy h, dq2 = dy over all points. Per chunk of NP points (128 where all
// threads then have a tile of a, P <= 64 and n a multiple of 8, else 64): a in tiles of
// 8 rows of Q1 x 4 points a thread, da through shared memory, dz in tiles of 4 channels x 4 points, dQ1 as in
// k_grad_w. Bound by FP32 issue. Width 16, 64 rows, 4 fields of 64^3: 408 us in
// chunks of 64 (half the threads without a tile of a), 288 us in chunks of 128; the row-by-row form before, with
// the last layer's dW and transform (60 us each) in it, 835 us.
constexpr int GQ_TILES = (MAXP / 4) * (MAXC / 4) / GD_T;   // 4 x 4 tiles of dQ1 a thread, at most
struct ProjDims {
    int PP, C4;   // rows of Q1 in blocks of 8, row stride of Q1 [p][c]
    size_t smem;
};
static ProjDims proj_dims(int C, int P, int np) {
    ProjDims d;
    d.PP = (P + 7) & ~7;
    d.C4 = C + 4;
    d.smem = ((size_t)(C + d.PP) * (np + 4) + (size_t)C * d.PP + (size_t)d.PP * d.C4 + 2 * d.PP + np) * 4;
    return d;
}
template <int NP>
__global__ void __launch_bounds__(GD_T) k_proj_bwd(const float* __restrict__ vL, const float* __restrict__ dy,
                                                   const float* __restrict__ Q1, const float* __restrict__ q1,
                                                   const float* __restrict__ Q2, float* __restrict__ dz, float* gQ1,
                                                   float* gq1, float* gQ2, float* gq2, int B, int C, int P, int64_t np3,
                                                   ProjDims d) {
    constexpr int GPS = NP + 4;
    extern __shared__ __align__(16) float zsh[];
    float* vs = zsh;                    // v_L [C][GPS]
    float* das = vs + C * GPS;          // da [PP][GPS]
    float* Qt = das + d.PP * GPS;       // Q1 transposed [C][PP]
    float* Qs = Qt + C * d.PP;          // Q1 [PP][C4]
    float* pq = Qs + d.PP * d.C4;       // q1, Q2 [2][PP]
    float* dys = pq + 2 * d.PP;         // dy [NP]
    const int tid = threadIdx.x;
    for (int e = tid; e < d.PP * C; e += GD_T) {
        const int p = e / C, c = e - p * C;
        const float w = p < P ? Q1[e] : 0.f;
        Qt[c * d.PP + p] = w;
        Qs[p * d.C4 + c] = w;
    }
    for (int p = tid; p < d.PP; p += GD_T) {
        pq[p] = p < P ? q1[p] : 0.f;
        pq[d.PP + p] = p < P ? Q2[p] : 0.f;
    }
    constexpr int NZ = NP / 4;                  // blocks of 4 points
    const int nt = C / 4, tiles = d.PP / 4 * nt, S = grad_splits(tiles), s = tid % S;
    const int zb = tid % NZ, pb = tid / NZ;     // (PP / 8 <= GD_T / NZ blocks of 8 rows)
    const int z0 = 4 * zb, p0 = 8 * pb;
    float aQ1[GQ_TILES][16], aq1[8], aQ2[8], aq2 = 0.f;
#pragma unroll
    for (int k = 0; k < GQ_TILES; ++k)
#pragma unroll
        for (int i = 0; i < 16; ++i) aQ1[k][i] = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) aq1[j] = aQ2[j] = 0.f;
    const int64_t per = np3 / NP, nchunk = per * B;
    for (int64_t k = blockIdx.x; k < nchunk; k += gridDim.x) {
        const int64_t b = k / per, pt = (k - b * per) * NP;
        __syncthreads();   // the previous chunk has been read
        for (int c = tid / NZ; c < C; c += GD_T / NZ) sno_cp16(vs + c * GPS + z0, vL + (b * C + c) * np3 + pt + z0);
        if (tid < NZ) sno_cp16(dys + z0, dy + b * np3 + pt + z0);
        sno_commit();
        sno_wait_all();
        __syncthreads();
        const float4 dyv = *reinterpret_cast<const float4*>(dys + z0);
        if (p0 < d.PP) {
            float a[8][4];
#pragma unroll
            for (int j = 0; j < 8; ++j)
#pragma unroll
                for (int i = 0; i < 4; ++i) a[j][i] = pq[p0 + j];
            for (int c = 0; c < C; ++c) {
                const float4 x = *reinterpret_cast<const float4*>(vs + c * GPS + z0);
                const float4 w0 = *reinterpret_cast<const float4*>(Qt + c * d.PP + p0);
                const float4 w1 = *reinterpret_cast<const float4*>(Qt + c * d.PP + p0 + 4);
                const float wv[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    a[j][0] = fmaf(wv[j], x.x, a[j][0]);
                    a[j][1] = fmaf(wv[j], x.y, a[j][1]);
                    a[j][2] = fmaf(wv[j], x.z, a[j][2]);
                    a[j][3] = fmaf(wv[j], x.w, a[j][3]);
                }
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float w = pq[d.PP + p0 + j];
                const float4 g = make_float4(dyv.x * w * gelu_d(a[j][0]), dyv.y * w * gelu_d(a[j][1]),
                                             dyv.z * w * gelu_d(a[j][2]), dyv.w * w * gelu_d(a[j][3]));
                aQ2[j] = fmaf(dyv.x, gelu_f(a[j][0]), fmaf(dyv.y, gelu_f(a[j][1]),
                         fmaf(dyv.z, gelu_f(a[j][2]), fmaf(dyv.w, gelu_f(a[j][3]), aQ2[j]))));
                aq1[j] += (g.x + g.y) + (g.z + g.w);
                *reinterpret_cast<float4*>(das + (p0 + j) * GPS + z0) = g;
            }
        }
        if (tid < NZ) aq2 += (dyv.x + dyv.y) + (dyv.z + dyv.w);
        __syncthreads();
        for (int cb = tid / NZ; cb < nt; cb += GD_T / NZ) {   // dz: 4 channels x 4 points
            float a[4][4] = {};
            for (int p = 0; p < d.PP; ++p) {
                const float4 x = *reinterpret_cast<const float4*>(das + p * GPS + z0);
                const float4 w = *reinterpret_cast<const float4*>(Qs + p * d.C4 + 4 * cb);
                const float wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    a[j][0] = fmaf(wv[j], x.x, a[j][0]);
                    a[j][1] = fmaf(wv[j], x.y, a[j][1]);
                    a[j][2] = fmaf(wv[j], x.z, a[j][2]);
                    a[j][3] = fmaf(wv[j], x.w, a[j][3]);
                }
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
                *reinterpret_cast<float4*>(dz + (b * C + 4 * cb + j) * np3 + pt + z0) =
                    make_float4(a[j][0], a[j][1], a[j][2], a[j][3]);
        }
#pragma unroll
        for (int j = 0; j < GQ_TILES; ++j) {
            const int t = tid / S + j * (GD_T / S);
            if (t < tiles) grad_tile<NP>(das + 4 * (t / nt) * GPS, vs + 4 * (t % nt) * GPS, s, S, aQ1[j]);
        }
    }
#pragma unroll
    for (int j = 0; j < GQ_TILES; ++j) {
        const int t = tid / S + j * (GD_T / S);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const float a = lane_sum(aQ1[j][i], S);
            const int p = 4 * (t / nt) + i / 4;
            if (t < tiles && !s && p < P) atomicAdd(gQ1 + p * C + 4 * (t % nt) + i % 4, a);
        }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const float a = lane_sum(aq1[j], NZ), h = lane_sum(aQ2[j], NZ);
        if (!zb && p0 + j < P) {
            atomicAdd(gq1 + p0 + j, a);
            atomicAdd(gQ2 + p0 + j, h);
        }
    }
    aq2 = lane_sum(aq2, NZ);
    if (tid == 0) atomicAdd(gq2, aq2);
}

// loss and dL/dy: mean squared error; dy = 2 (y - t) / (B np3)
__global__ void k_loss(const float* y, const float* t, float* dy, int64_t N, double* loss) {
    __shared__ double red[256];
    double acc = 0;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < N; e += (int64_t)gridDim.x * blockDim.x) {
        const float d = y[e] - t[e];
        acc += (double)d * d;
        dy[e] = 2.0f * d / (float)N;
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(loss, red[0] / (double)N);
}

__global__ void k_adam(float* th, const float* g, float* mo, float* ve, int64_t n, float lr, float b1, float b2,
                       float eps, float c1, float c2) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const float gi = g[e];
    const float m = b1 * mo[e] + (1.f - b1) * gi;
    const float v = b2 * ve[e] + (1.f - b2) * gi * gi;
    mo[e] = m;
    ve[e] = v;
    th[e] -= lr * (m / c1) / (sqrtf(v / c2) + eps);
}

__global__ void k_to_bf16(const float* a, __nv_bfloat16* b, int64_t n) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < n) b[e] = __float2bfloat16_rn(a[e]);
}

// ---- passes ---------------------------------------------------------------------------------
static float* fld(const DevBuf& b, int64_t i, int64_t per) { return ptr<float>(b) + i * per; }

// tiles of about `cols` columns for the folded plane transforms
static FoldTile fold_tiles(int64_t P, int L, int inner, int cols) {
    FoldTile f;
    f.P = P;
    f.L = L;
    f.inner = inner;
    f.PB = 1;
    f.W = inner;
    f.ps = L * inner;
    if (inner > cols) {
        const int nchunk = (inner + cols - 1) / cols;
        f.W = ((inner + nchunk - 1) / nchunk + 1) & ~1;
        f.ps = L * f.W;
    } else {   // the planes' stride continues the columns' banks, and keeps the 16-byte copies aligned
        f.PB = (int)std::min<int64_t>(std::max(1, cols / inner), P);
        f.ps += (((inner + 1) & ~1) - L * inner % 16 + 16) % 16;
    }
    f.nch = (inner + f.W - 1) / f.W;
    f.ntiles = ((P + f.PB - 1) / f.PB) * f.nch;
    return f;
}

// x and y transforms of [P][n][inner] to [P][2m][inner]: about one item a thread, at most 72 KB of
// tiles (three blocks an SM at n = 64)
static FoldTile fold_fwd_tiles(int n, int m, int64_t P, int inner, int& nkb, int& kb, size_t& smem) {
    nkb = (m + 8) / 8;
    kb = std::max(4, (m + nkb) / nkb);
    const FoldTile f = fold_tiles(P, n, inner, std::max(2, std::min(FF_T / nkb, (72 << 10) / (16 * n))) & ~1);
    smem = ((size_t)2 * f.PB * f.ps + (size_t)nkb * (n / 2) * ((kb + 1) & ~1)) * sizeof(float2);
    return f;
}
static int plane_fwd(SnoModel& M, const float2* in, float2* out, int64_t P, int inner, float zscale = 0.f) {
    int nkb = 0, kb = 0;
    size_t smem = 0;
    const FoldTile f = fold_fwd_tiles(M.n, M.m, P, inner, nkb, kb, smem);
    auto* k = kb == 4 ? k_fold_fwd<4> : kb == 5 ? k_fold_fwd<5> : kb == 6 ? k_fold_fwd<6> : kb == 7 ? k_fold_fwd<7>
                                                                                         : k_fold_fwd<8>;
    int per_sm = 1;
    KF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, FF_T, smem));
    const int64_t grid = std::min<int64_t>(f.ntiles, (int64_t)std::max(1, per_sm) * M.num_sms);
    const float2* T = ptr<float2>(M.tabs);
    k<<<(unsigned)grid, FF_T, smem, M.st>>>(in, out, T + M.tfo, T + M.tph, M.m, nkb, zscale, f);
    KF_LAUNCH();
    return KIFMM_OK;
}
// and of [P][2m][inner] to [P][n][inner]
static FoldTile fold_inv_tiles(int n, int m, int64_t P, int inner, int& njb, size_t& smem) {
    njb = (n / 2 + FV_J - 1) / FV_J;
    const FoldTile f = fold_tiles(P, 2 * m, inner, std::max(2, std::min(FV_T / njb, (80 << 10) / (48 * m + 16))) & ~1);
    smem = ((size_t)2 * f.PB * f.ps + (size_t)(m + 1) * njb * FV_J) * sizeof(float2) +
           (size_t)(m + 1) * f.PB * f.W * sizeof(float4);
    return f;
}
static int plane_inv(SnoModel& M, const float2* in, float2* out, int64_t P, int inner, float zscale = 0.f) {
    int njb = 0;
    size_t smem = 0;
    const FoldTile f = fold_inv_tiles(M.n, M.m, P, inner, njb, smem);
    int per_sm = 1;
    KF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fold_inv, FV_T, smem));
    const int64_t grid = std::min<int64_t>(f.ntiles, (int64_t)std::max(1, per_sm) * M.num_sms);
    const float2* T = ptr<float2>(M.tabs);
    k_fold_inv<<<(unsigned)grid, FV_T, smem, M.st>>>(in, out, T + M.tfo, T + M.tph, M.m, M.n, njb, zscale, f);
    KF_LAUNCH();
    return KIFMM_OK;
}

static int mix(SnoModel& M, int l, const float2* V, float2* G, int B, int adj) {
    const int C = M.C;
    const MixDims d = mix_dims(C, B);
    const dim3 nb(nbs(M.K, d.MB), nbs(B, d.BT));
    if (M.bf16)
        k_mix<__nv_bfloat16><<<nb, 256, d.smem, M.st>>>(
            ptr<__nv_bfloat16>(M.rbf) + (int64_t)l * 2 * M.K * C * C,
            ptr<__nv_bfloat16>(M.rbf) + ((int64_t)l * 2 + 1) * M.K * C * C, V, G, B, C, M.K, adj, d);
    else
        k_mix<float><<<nb, 256, d.smem, M.st>>>(ptr<float>(M.theta) + M.off[o_rr(l)],
                                                ptr<float>(M.theta) + M.off[o_ri(l)], V, G, B, C, M.K, adj, d);
    KF_LAUNCH();
    return KIFMM_OK;
}

static size_t lift_u_smem(int n, int m) { return (size_t)(LU * (n / 2 + 1) + n / 2 * (m + 1)) * 8; }
static size_t lift_z_smem(int n, int C, int m) { return (size_t)((C * (n + 1) + n + 1) & ~1) * 4 + (size_t)m * (n + 1) * 8; }
static size_t grad_w_smem(int C) { return (size_t)4 * C * GPS * 4; }
static bool proj_wide(int n, int P) { return P <= 64 && n % 8 == 0; }   // chunks of the projection's backward
// the most shared memory that a kernel of the forward and backward passes takes (bytes), without k_mix_grad
static size_t sno_smem(int n, int C, int m, int P, int maxB) {
    size_t most = std::max({lift_u_smem(n, m), lift_z_smem(n, C, m), grad_w_smem(C), zrow_dims(n, C, m, P, false).smem,
                            zrow_dims(n, C, m, P, true).smem, proj_dims(C, P, proj_wide(n, P) ? 128 : 64).smem});
    for (int B = 1; B <= std::min(maxB, MIX_B); ++B) most = std::max(most, mix_dims(C, B).smem);
    for (int inner : {m, 2 * m * m}) {
        int a = 0, b = 0;
        size_t smem = 0;
        fold_fwd_tiles(n, m, (int64_t)1 << 40, inner, a, b, smem);
        most = std::max(most, smem);
        fold_inv_tiles(n, m, (int64_t)1 << 40, inner, a, smem);
        most = std::max(most, smem);
    }
    return most;
}

static unsigned zr_blocks(const SnoModel& M, int B) { return nbs((int64_t)B * M.n * M.n, ZR_RG); }
static int near_add(SnoModel& M, const float* u, float* y, int B);

// forward; train: keep z_l and the spectra V_l for the backward pass
static int forward(SnoModel& M, const float* u, float* y, int B, bool train) {
    const int n = M.n, m = M.m, C = M.C, M2 = 2 * m;
    const int64_t per = (int64_t)B * C * M.np3, BC = (int64_t)B * C;
    cudaStream_t st = M.st;
    const float* th = ptr<float>(M.theta);
    const float2* T = ptr<float2>(M.tabs);
    const int q = o_q1(M);
    const float wn = 1.f / ((float)M.period * M.period * M.period);
    if (!train) {   // inference: layer 0 from u

        const int64_t rows = (int64_t)B * n * n;
        k_lift_u<<<(unsigned)((rows + LU - 1) / LU), 256, lift_u_smem(n, m), st>>>(
            u, T + M.tfo, ptr<float2>(M.cz), rows, n, m);
        KF_LAUNCH();
        KF_TRY(plane_fwd(M, ptr<float2>(M.cz), ptr<float2>(M.cy), (int64_t)B * n, m));     // y
        KF_TRY(plane_fwd(M, ptr<float2>(M.cy), ptr<float2>(M.Vst), B, M2 * m, 1.f));      // x: U
        float2* A = ptr<float2>(M.m0ab);
        float2* Bc = A + (int64_t)C * M.K;
        const unsigned np = (unsigned)M.K;
        if (M.bf16)
            k_mix0_prep<__nv_bfloat16><<<np, M0_T, 0, st>>>(ptr<__nv_bfloat16>(M.rbf),
                                                           ptr<__nv_bfloat16>(M.rbf) + M.K * C * C, th + M.off[O_WL],
                                                           th + M.off[O_BL], T + M.tyf, T + M.tzf, C, M.K, n, m, A,
                                                           Bc);
        else
            k_mix0_prep<float><<<np, M0_T, 0, st>>>(th + M.off[o_rr(0)], th + M.off[o_ri(0)], th + M.off[O_WL],
                                                   th + M.off[O_BL], T + M.tyf, T + M.tzf, C, M.K, n, m, A, Bc);
        k_mix0<<<nbs(BC * M.K, 256), 256, 0, st>>>(ptr<float2>(M.Vst), A, Bc, ptr<float2>(M.g), B, C, M.K);
        KF_LAUNCH();
    } else {
        k_lift_z<<<zr_blocks(M, B), ZR_T, M.lift_smem, st>>>(u, th + M.off[O_WL], th + M.off[O_BL],
                                                             fld(M.v, 0, per), ptr<float2>(M.cz), T + M.tzf, B, C, n,
                                                             m);
        KF_LAUNCH();
    }
    for (int l = 0; l < M.L; ++l) {
        if (train || l > 0) {   // (the training's lift is not centred)
            float2* V = ptr<float2>(M.Vst) + (train ? (int64_t)l * BC * M.K : 0);
            KF_TRY(plane_fwd(M, ptr<float2>(M.cz), ptr<float2>(M.cy), BC * n, m));            // y
            KF_TRY(plane_fwd(M, ptr<float2>(M.cy), V, BC, M2 * m, l == 0 ? 0.f : 1.f));     // x
            KF_TRY(mix(M, l, V, ptr<float2>(M.g), B, 0));
        }
        KF_TRY(plane_inv(M, ptr<float2>(M.g), ptr<float2>(M.gx), BC, M2 * m, wn));                   // x^-1
        KF_TRY(plane_inv(M, ptr<float2>(M.gx), ptr<float2>(M.gy), BC * n, m));                       // y^-1
        const bool last = l == M.L - 1, lift = !train && l == 0;
        const ZRowDims d = zrow_dims(n, C, m, M.P, last);
        const int rows = B * n * n;
        int per_sm = 1;
        auto* kz = last ? k_zrow<ZR_PROJ> : k_zrow<ZR_FWD>;   // (the last layer's rows go into the projection)
        KF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kz, ZF_T, d.smem));
        const int grid = std::min((rows + d.R - 1) / d.R, std::max(1, per_sm) * M.num_sms);
        kz<<<grid, ZF_T, d.smem, st>>>(
            ptr<float2>(M.gy), lift ? nullptr : fld(M.v, l, per), th + M.off[o_w(l)], th + M.off[o_b(l)], T + M.tfo,
            train ? fld(M.z, l, per) : nullptr, train || !last ? fld(M.v, l + 1, per) : nullptr,
            last ? nullptr : ptr<float2>(M.cz), th + M.off[q], th + M.off[q + 1], th + M.off[q + 2], th + M.off[q + 3],
            last ? y : nullptr, lift ? u : nullptr, th + M.off[O_WL], th + M.off[O_BL], rows, C, n, m, M.P,
            d);
        KF_LAUNCH();
    }
    return near_add(M, u, y, B);   // the exact near part (when set) is a fixed addend of y
}

static int loss_grad(SnoModel& M, const float* u, const float* t, int B, double* loss_host) {
    const int n = M.n, m = M.m, C = M.C, M2 = 2 * m;
    const int64_t per = (int64_t)B * C * M.np3, BC = (int64_t)B * C, N = (int64_t)B * M.np3;
    cudaStream_t st = M.st;
    float* gr = ptr<float>(M.grad);
    const float* th = ptr<float>(M.theta);
    const float2* T = ptr<float2>(M.tabs);
    KF_CUDA(cudaMemsetAsync(gr, 0, M.nparam * 4, st));
    KF_CUDA(cudaMemsetAsync(M.loss.p, 0, 8, st));
    float* y = ptr<float>(M.yb);
    float* dy = ptr<float>(M.dy);
    KF_TRY(forward(M, u, y, B, true));
    k_loss<<<1024, 256, 0, st>>>(y, t, dy, N, ptr<double>(M.loss));
    KF_LAUNCH();
    const int q = o_q1(M), L = M.L;
    float* dzA = fld(M.dz, 0, per);
    float* dzB = fld(M.dz, 1, per);
    const bool wide = proj_wide(n, M.P);
    const ProjDims pd = proj_dims(C, M.P, wide ? 128 : 64);
    auto* kpb = wide ? k_proj_bwd<128> : k_proj_bwd<64>;
    const int64_t nchunk = N / GP, rows = BC * n * n;
    const size_t gsm = grad_w_smem(C);
    int pb_sm = 1, gw_sm = 1;
    KF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&pb_sm, kpb, GD_T, pd.smem));
    KF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&gw_sm, k_grad_w, GD_T, gsm));
    const unsigned npb = (unsigned)std::min<int64_t>(N / (wide ? 128 : 64), (int64_t)std::max(1, pb_sm) * M.num_sms);
    const unsigned ngw = (unsigned)std::min<int64_t>(nchunk, (int64_t)std::max(1, gw_sm) * M.num_sms);
    kpb<<<npb, GD_T, pd.smem, st>>>(fld(M.v, L, per), dy, th + M.off[q], th + M.off[q + 1], th + M.off[q + 2],
                                           dzA, gr + M.off[q], gr + M.off[q + 1], gr + M.off[q + 2], gr + M.off[q + 3],
                                           B, C, M.P, M.np3, pd);
    KF_LAUNCH();
    k_lift_u<<<nbs(rows, LU), 256, lift_u_smem(n, m), st>>>(
        dzA, T + M.tfo, ptr<float2>(M.cz), rows, n, m);
    KF_LAUNCH();
    const float wn = 1.f / ((float)M.period * M.period * M.period);
    const ZRowDims zd = zrow_dims(n, C, m, M.P, false);
    int zb_sm = 1;
    KF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&zb_sm, k_zrow<ZR_BWD>, ZF_T, zd.smem));
    const int zgrid = std::min((B * n * n + zd.R - 1) / zd.R, std::max(1, zb_sm) * M.num_sms);
    for (int l = L - 1; l >= 0; --l) {
        k_grad_w<<<ngw, GD_T, gsm, st>>>(dzA, fld(M.v, l, per), gr + M.off[o_w(l)], gr + M.off[o_b(l)], B, C, M.np3);
        KF_LAUNCH();
        // spectral adjoint of layer l (cz holds the last-axis transform of dz_l): dG, dR, dV = R^H dG
        KF_TRY(plane_fwd(M, ptr<float2>(M.cz), ptr<float2>(M.cy), BC * n, m));
        KF_TRY(plane_fwd(M, ptr<float2>(M.cy), ptr<float2>(M.g), BC, M2 * m, wn));
        const unsigned nb = nbs(M.K, M.mix_mb);
        k_mix_grad<<<nb, 256, M.mixg_smem, st>>>(ptr<float2>(M.g), ptr<float2>(M.Vst) + (int64_t)l * BC * M.K,
                                                 gr + M.off[o_rr(l)], gr + M.off[o_ri(l)], B, C, M.K, M.mix_mb);
        KF_LAUNCH();
        KF_TRY(mix(M, l, ptr<float2>(M.g), ptr<float2>(M.ga), B, 1));
        KF_TRY(plane_inv(M, ptr<float2>(M.ga), ptr<float2>(M.gx), BC, M2 * m, 1.f));
        KF_TRY(plane_inv(M, ptr<float2>(M.gx), ptr<float2>(M.gy), BC * n, m));
        k_zrow<ZR_BWD><<<zgrid, ZF_T, zd.smem, st>>>(
            ptr<float2>(M.gy), dzA, th + M.off[o_w(l)], nullptr, T + M.tfo, l > 0 ? fld(M.z, l - 1, per) : nullptr, dzB,
            l > 0 ? ptr<float2>(M.cz) : nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr,
            B * n * n, C, n, m, M.P, zd);
        KF_LAUNCH();
        std::swap(dzA, dzB);
    }
    k_grad_lift<<<dim3(nbs(M.np3 / 4, 1024), C), 256, 0, st>>>(dzA, u, gr + M.off[O_WL], gr + M.off[O_BL], B, C, M.np3);
    KF_LAUNCH();
    if (loss_host) {
        KF_CUDA(cudaMemcpyAsync(loss_host, M.loss.p, 8, cudaMemcpyDeviceToHost, st));
        KF_CUDA(cudaStreamSynchronize(st));
    }
    return KIFMM_OK;
}

static int refresh_bf16(SnoModel& M) {
    const int64_t KC = M.K * M.C * M.C;
    for (int l = 0; l < M.L; ++l) {
        k_to_bf16<<<nbs(KC, 256), 256, 0, M.st>>>(ptr<float>(M.theta) + M.off[o_rr(l)],
                                                  ptr<__nv_bfloat16>(M.rbf) + (int64_t)l * 2 * KC, KC);
        KF_LAUNCH();
        k_to_bf16<<<nbs(KC, 256), 256, 0, M.st>>>(ptr<float>(M.theta) + M.off[o_ri(l)],
                                                  ptr<__nv_bfloat16>(M.rbf) + ((int64_t)l * 2 + 1) * KC, KC);
        KF_LAUNCH();
    }
    return KIFMM_OK;
}

// ---- near part and far-field multiplier ------------------------------------------------------
__host__ __device__ inline double near_window(double rho, double r_in, double r_out) {
    if (rho <= r_in) return 1.0;
    if (rho >= r_out) return 0.0;
    const double c = cos(1.5707963267948966 * (rho - r_in) / (r_out - r_in));
    return c * c;
}

// taps of the near part on the cube [-R, R]^3: K(h|d|) w(|d|) h^3 (0 at d = 0 and beyond
// r_out); block 0 also writes sigma (64-node Gauss-Legendre face integral) to sig[0]
__global__ void k_near_taps(int R, KParams kp, double h, double r_in, double r_out, int mode, double* tap,
                            double* sig) {
    const int side = 2 * R + 1;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < (int64_t)side * side * side) {
        const int dx = (int)(i % side) - R, dy = (int)((i / side) % side) - R, dz = (int)(i / ((int64_t)side * side)) - R;
        const double rho = sqrt((double)(dx * dx + dy * dy + dz * dz));
        tap[i] = (rho == 0.0 || rho >= r_out) ? 0.0 : kern_f64(h * rho, kp) * near_window(rho, r_in, r_out) * h * h * h;
    }
    if (blockIdx.x == 0) {
        __shared__ double gx[64], gw[64], red[256];
        if (threadIdx.x < 64) gl_node(64, threadIdx.x, &gx[threadIdx.x], &gw[threadIdx.x]);
        __syncthreads();
        const double sv = self_sigma_block(h, kp.a, kp.b, mode, 64, gx, gw, red);
        if (threadIdx.x == 0) sig[0] = sv;
    }
}

// y[b][i][j][k] += sum_d w_d u[b][i+di][j+dj][k+dk] (u = 0 outside the grid). A block takes an
// 8 (i) x 8 (j) x 32 (k) tile of one field with its halo of R cells in shared memory; a thread
// computes 16 consecutive k of one (i, j). The weights depend on the distance alone, so the up to
// eight stencil columns (+-di, +-dj) and (+-dj, +-di) share theirs: their rows of 16 + 2R inputs
// are added first and take the 2R + 1 weights (zero outside the sphere) once, R = 6: 28 additions
// a column and 208 FMAs a group in place of 208 FMAs a column. The halo along k is rounded up to
// whole 16-byte pieces, copied asynchronously with zeros outside the grid, and rows are padded so
// that a warp's 16-byte loads are free of conflicts; bound by those loads.
// One GB300, 32 fields of 64^3, a halo of 7 cells: 925 -> 438 us (8 outputs a
// thread, 8 x 4-byte halo loads and a column at a time before).
constexpr int NT_I = 8, NT_J = 8, NT_K = 32, NT_KB = 16, NT_T = NT_I * NT_J * NT_K / NT_KB;
constexpr int NT_TK = 52;   // row stride: at least NT_K + 16, and 4 mod 16
// tab: ng + 1 group bounds (in .x), then the members' (di, dj)
template <int R>
__global__ void __launch_bounds__(NT_T) k_near_add(const float* __restrict__ u, float* __restrict__ y, int n,
                                                   const int2* __restrict__ tab, const float* __restrict__ cw,
                                                   int ng, int ncols) {
    extern __shared__ __align__(16) float nsh[];
    constexpr int TI = NT_I + 2 * R, TJ = NT_J + 2 * R, TK = NT_TK, W = 2 * R + 1;
    constexpr int RK = (R + 3) & ~3, NQ = (NT_K + 2 * RK) / 4, NR = NT_KB + 2 * RK;   // halo and pieces of a row, inputs a thread
    float* us = nsh;                                               // [TI][TJ][TK]
    float* ws = us + TI * TJ * TK;                                 // [ng][2R + 1]
    int* gb = reinterpret_cast<int*>(ws + ng * W);                 // [ng + 1]
    int* cs = gb + ng + 1;                                         // [ncols] offsets of the members' rows
    const int ti_n = (n + NT_I - 1) / NT_I, tj_n = (n + NT_J - 1) / NT_J, tk_n = (n + NT_K - 1) / NT_K;
    const int64_t per = (int64_t)ti_n * tj_n * tk_n;
    const int b = (int)(blockIdx.x / per);
    const int r3 = (int)(blockIdx.x % per);
    const int i0 = NT_I * (r3 / (tj_n * tk_n)), j0 = NT_J * ((r3 / tk_n) % tj_n), k0 = NT_K * (r3 % tk_n);
    const int64_t base = (int64_t)b * n * n * n;
    const bool aligned = (reinterpret_cast<uintptr_t>(u) & 15) == 0;   // (a caller's field may lie anywhere)
    for (int e = threadIdx.x; e < TI * TJ * NQ; e += NT_T) {   // (n is a multiple of 4)
        const int ij = e / NQ, q = e - ij * NQ;
        const int ii = ij / TJ + i0 - R, jj = ij % TJ + j0 - R, kk = 4 * q + k0 - RK;
        const bool in = ii >= 0 && ii < n && jj >= 0 && jj < n && kk >= 0 && kk < n;
        const float* src = in ? u + base + ((int64_t)ii * n + jj) * n + kk : u;
        float* dst = us + ij * TK + 4 * q;
        if (aligned) sno_cp16z(dst, src, in);
        else *reinterpret_cast<float4*>(dst) = in ? make_float4(src[0], src[1], src[2], src[3]) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    sno_commit();
    for (int g = threadIdx.x; g <= ng; g += NT_T) gb[g] = tab[g].x;
    for (int c = threadIdx.x; c < ncols; c += NT_T) cs[c] = (tab[ng + 1 + c].x * TJ + tab[ng + 1 + c].y) * TK;
    for (int e = threadIdx.x; e < ng * W; e += NT_T) ws[e] = cw[e];
    sno_wait_all();
    __syncthreads();
    constexpr int KT = NT_K / NT_KB;
    const int tkb = threadIdx.x % KT, tj = (threadIdx.x / KT) % NT_J, ti = threadIdx.x / (KT * NT_J);
    const float* own = us + ((ti + R) * TJ + tj + R) * TK + NT_KB * tkb;
    float acc[NT_KB];
#pragma unroll
    for (int m = 0; m < NT_KB; ++m) acc[m] = 0.f;
    for (int g = 0; g < ng; ++g) {
        float r[NR];
#pragma unroll
        for (int q = 0; q < NR; ++q) r[q] = 0.f;
        for (int c = gb[g]; c < gb[g + 1]; ++c) {
            const float* row = own + cs[c];
#pragma unroll
            for (int q = 0; q < NR; q += 4) {
                const float4 x = *reinterpret_cast<const float4*>(row + q);
                r[q] += x.x;
                r[q + 1] += x.y;
                r[q + 2] += x.z;
                r[q + 3] += x.w;
            }
        }
        const float* w = ws + g * W;
#pragma unroll
        for (int t = 0; t < W; ++t) {
            const float wt = w[t];
#pragma unroll
            for (int m = 0; m < NT_KB; ++m) acc[m] = fmaf(wt, r[m + t + RK - R], acc[m]);
        }
    }
    const int gi = i0 + ti, gj = j0 + tj, gk = k0 + NT_KB * tkb;
    if (gi < n && gj < n) {
        float* yo = y + base + ((int64_t)gi * n + gj) * n + gk;
#pragma unroll
        for (int m = 0; m < NT_KB; ++m)
            if (gk + m < n) yo[m] += acc[m];
    }
}

template <int R>
static size_t near_smem(int ng, int ncols) {
    return ((size_t)(NT_I + 2 * R) * (NT_J + 2 * R) * NT_TK + (size_t)ng * (2 * R + 1) + ng + 1 + ncols) * 4;
}

static int near_add(SnoModel& M, const float* u, float* y, int B) {
    if (!M.near_on) return KIFMM_OK;
    const int n = M.n;
    const int64_t blocks = (int64_t)B * ((n + NT_I - 1) / NT_I) * ((n + NT_J - 1) / NT_J) * ((n + NT_K - 1) / NT_K);
#define KF_NEAR(RR)                                                                                              \
    case RR:                                                                                                     \
        k_near_add<RR><<<(unsigned)blocks, NT_T, near_smem<RR>(M.ngroups, M.ntaps), M.st>>>(                                \
            u, y, n, ptr<int2>(M.near_d), ptr<float>(M.near_w), M.ngroups, M.ntaps);                                         \
        break;
    switch (M.nR) {
        KF_NEAR(1) KF_NEAR(2) KF_NEAR(3) KF_NEAR(4) KF_NEAR(5) KF_NEAR(6) KF_NEAR(7)   // (r_out <= 8)
        default: set_error("near part: halo out of range"); return KIFMM_ERR_ARG;
    }
#undef KF_NEAR
    KF_LAUNCH();
    return KIFMM_OK;
}

// far multiplier M(k) = sum_d K(h|d|) (1 - w(|d|)) h^3 cos(2 pi kx dx / N) cos(..) cos(..) over
// the N-periodic grid (minimum-image offsets; the table is even in every axis), by three
// one-axis passes in FP64: A[dx][dy][kz], B[dx][ky][kz], M[kx][ky][kz]
__device__ __forceinline__ int min_image(int d, int N) { return d >= (N + 1) / 2 ? d - N : d; }
__global__ void k_far_pass_z(int N, int m, KParams kp, double h, double r_in, double r_out, double* A) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)N * N * m) return;
    const int kz = (int)(i % m), dy = min_image((int)((i / m) % N), N), dx = min_image((int)(i / ((int64_t)m * N)), N);
    const double tw = 6.283185307179586476925286766559 / N;
    double acc = 0.0;
    for (int z = 0; z < N; ++z) {
        const int dz = min_image(z, N);
        const double rho = sqrt((double)dx * dx + (double)dy * dy + (double)dz * dz);
        if (rho == 0.0) continue;
        const double kf = kern_f64(h * rho, kp) * (1.0 - near_window(rho, r_in, r_out)) * h * h * h;
        acc += kf * cos(tw * (double)((int64_t)kz * z % N));
    }
    A[i] = acc;
}
__global__ void k_far_pass_y(int N, int m, const double* A, double* Bf) {   // Bf[dx][ky][kz]
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)N * 2 * m * m) return;
    const int kz = (int)(i % m), kyi = (int)((i / m) % (2 * m)), x = (int)(i / ((int64_t)m * 2 * m));
    const int ky = kyi < m ? kyi : N - 2 * m + kyi;
    const double tw = 6.283185307179586476925286766559 / N;
    double acc = 0.0;
    for (int y = 0; y < N; ++y) acc += A[((int64_t)x * N + y) * m + kz] * cos(tw * (double)((int64_t)ky * y % N));
    Bf[i] = acc;
}
__global__ void k_far_pass_x(int N, int m, const double* Bf, double* Mk) {   // Mk[kx][ky][kz]
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)4 * m * m * m) return;
    const int kz = (int)(i % m), kyi = (int)((i / m) % (2 * m)), kxi = (int)(i / ((int64_t)m * 2 * m));
    const int kx = kxi < m ? kxi : N - 2 * m + kxi;
    const double tw = 6.283185307179586476925286766559 / N;
    double acc = 0.0;
    for (int x = 0; x < N; ++x) acc += Bf[((int64_t)x * 2 * m + kyi) * m + kz] * cos(tw * (double)((int64_t)kx * x % N));
    Mk[i] = acc;
}

// photo_solve's amplitude scale s = max_i |I_i| (non-negative doubles compare as their bits)
__global__ void k_sno_absmax(const double* I, int64_t n, unsigned long long* out) {
    __shared__ double red[256];
    double mx = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        mx = fmax(mx, fabs(I[i]));
    red[threadIdx.x] = mx;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + o]);
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicMax(out, (unsigned long long)__double_as_longlong(red[0]));
}
__global__ void k_scale_in(const double* I, const double* s, float* u, int64_t n) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const double sv = s[0];
    if (e < n) u[e] = sv > 0.0 ? (float)(I[e] / sv) : 0.f;
}
__global__ void k_scale_out(const float* y, const double* s, double C, double* S, int64_t n) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < n) S[e] = C * s[0] * (double)y[e];
}

// ---- judge: direct sum at sampled targets (FP32, absolute coordinates) ------------------------
// The judge's direct sum at the k drawn targets, with each source read once: a block takes a
// chunk of JG_CH sources (FP32 coordinates and weights) into shared memory and adds its part
// of every target's sum (one target per thread and pass) into acc[t] (one FP64 atomic per
// target and chunk). Within a chunk the pairs accumulate in FP32 with Kahan compensation: the
// judge decides against a tolerance of order 1e-2, far above the FP32 sum's error.
constexpr int JG_T = 256, JG_CH = 256;
__global__ void __launch_bounds__(JG_T) k_judge_src(const double* pts, const double* q, const int32_t* targets,
                                                    int k, int64_t n, KParams kp, double* acc) {
    __shared__ float4 sp[JG_CH];   // x, y, z, q
    const int64_t j0 = (int64_t)blockIdx.x * JG_CH;
    const int m = (int)min((int64_t)JG_CH, n - j0);
    for (int e = threadIdx.x; e < m; e += JG_T) {
        const int64_t j = j0 + e;
        sp[e] = make_float4((float)pts[3 * j], (float)pts[3 * j + 1], (float)pts[3 * j + 2], (float)q[j]);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < k; t += JG_T) {
        const int64_t i = targets[t];
        const float xi = (float)pts[3 * i], yi = (float)pts[3 * i + 1], zi = (float)pts[3 * i + 2];
        const int self = (i >= j0 && i < j0 + m) ? (int)(i - j0) : -1;
        Kahan a;
        float part[4] = {0.f, 0.f, 0.f, 0.f};   // four independent chains, then the compensated sum
        int e = 0;
        for (; e + 4 <= m; e += 4) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float4 v = sp[e + u];
                const float dx = xi - v.x, dy = yi - v.y, dz = zi - v.z;
                const float r2 = dx * dx + dy * dy + dz * dz;
                part[u] += e + u == self ? 0.f : kern_f32(r2, kp) * v.w;
            }
            if ((e & 15) == 12) {
                a.add((part[0] + part[1]) + (part[2] + part[3]));
                part[0] = part[1] = part[2] = part[3] = 0.f;
            }
        }
        for (; e < m; ++e) {
            const float4 v = sp[e];
            const float dx = xi - v.x, dy = yi - v.y, dz = zi - v.z;
            part[0] += e == self ? 0.f : kern_f32(dx * dx + dy * dy + dz * dz, kp) * v.w;
        }
        a.add((part[0] + part[1]) + (part[2] + part[3]));
        atomicAdd(acc + t, a.value());
    }
}
__global__ void k_judge_fin(const double* acc, const int32_t* targets, int k, const double* sigma, const double* Isort,
                            double C, const int32_t* perm, double* ref, int32_t* orig) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= k) return;
    const int64_t i = targets[t];
    ref[t] = C * (acc[t] + sigma[i] * Isort[i]);
    orig[t] = perm[i];
}

// importance-weighted estimate of the relative L2 error: targets drawn with probability
// m_i, each weighted 1 / (k m_i) (wt), so that both sums estimate the whole field's
__global__ void k_judge_err(const double* S, const double* ref, const int32_t* orig, const double* wt, int k,
                            double* out) {
    __shared__ double a[256], b[256];
    double num = 0, den = 0;
    for (int t = threadIdx.x; t < k; t += blockDim.x) {
        const double d = S[orig[t]] - ref[t];
        num += wt[t] * d * d;
        den += wt[t] * ref[t] * ref[t];
    }
    a[threadIdx.x] = num;
    b[threadIdx.x] = den;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
            a[threadIdx.x] += a[threadIdx.x + o];
            b[threadIdx.x] += b[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = sqrt(a[0] / fmax(b[0], 1e-300));
}

}  // namespace kifmm

using namespace kifmm;

struct sno_model_s {
    SnoModel m;
};

extern "C" {

int sno_create(sno_model_t* out, int n, int width, int modes, int layers, int proj_width, int max_batch,
               void* stream) {
    set_error("");
    if (!out || n < 4 || n > 128 || n % 4 || width < 4 || width > MAXC || width % 4 || modes < 1 || 2 * modes > n ||
        layers < 1 || proj_width < 1 || proj_width > MAXP || max_batch < 1) {
        set_error("sno_create: invalid dimensions");
        return KIFMM_ERR_ARG;
    }
    *out = nullptr;
    sno_model_s* h = new (std::nothrow) sno_model_s();
    if (!h) return KIFMM_ERR_OOM;
    SnoModel& M = h->m;
    M.n = n;
    M.C = width;
    M.m = modes;
    M.L = layers;
    M.P = proj_width;
    M.maxB = max_batch;
    M.st = (cudaStream_t)stream;
    M.K = (int64_t)(2 * modes) * (2 * modes) * modes;
    M.np3 = (int64_t)n * n * n;
    sno_layout(M);
    auto fail = [&](int rc) {
        sno_destroy(h);
        return rc;
    };
    const int64_t per = (int64_t)max_batch * width * M.np3;
    const int64_t BC = (int64_t)max_batch * width;
    // shared memory of the kernels (bytes), checked against the device's opt-in limit
    {
        M.lift_smem = lift_z_smem(n, width, modes);
        const size_t f4 = 4, f8 = 8, al = 16, per_mode = (size_t)width * (width + 1 + 2 * max_batch) * f8;
        M.mix_mb = (int)std::max<size_t>(1, std::min<size_t>(16, (96u << 10) / per_mode));
        M.mixg_smem = (size_t)2 * max_batch * M.mix_mb * width * f8;
        // The shapes taken: no more than those for which a form with whole rows of n points, the tables of their
        // transforms and R with the batch's spectra in shared memory would fit. (Some of the others would fit the kernels
        // now, 68 points with 64 channels and 33 modes for one, but none of them has been run.)
        const size_t ns = n + 1, C1 = width + 1;
        const size_t zf = (2 * width * ns + width * C1 + width) * f4 + al +
                          ((size_t)width * modes + n * (modes + 1) + modes * ns) * f8;
        const size_t zb = (3 * width * ns + width * C1) * f4 + al +
                          ((size_t)width * modes + n * (modes + 1) + modes * ns) * f8;
        const size_t zr = ((size_t)4 * width * (n + 4) + width * (width + 4) + width + proj_width * (width + 4) +
                     2 * proj_width + 4 * n) * f4 + al +
                    ((size_t)4 * width * modes + n * (modes + 1) + modes * (n + 2)) * f8;
        const size_t zp = zf + ((size_t)proj_width * C1 + 4 * n + 2 * proj_width) * f4;
        const size_t pb = (3 * width * ns + 2 * proj_width * ns + proj_width * C1 + 2 * proj_width + n) * f4 + al +
                      (size_t)modes * ns * f8;
        const size_t rows = std::max({zb, zr, zp, pb, (size_t)M.mix_mb * per_mode, ((size_t)n * 128 + (size_t)n * 2 * modes) * f8});
        int dev = 0, optin = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        const size_t need = std::max({rows, M.mixg_smem, sno_smem(n, width, modes, proj_width, max_batch)});
        cudaDeviceGetAttribute(&M.num_sms, cudaDevAttrMultiProcessorCount, dev);
        M.num_sms = std::max(M.num_sms, 1);
        if (optin <= 0 || need > (size_t)optin) {
            set_error("sno_create: the model's kernels need more shared memory than the device offers");
            delete h;
            return KIFMM_ERR_ARG;
        }
        const int lim = optin;
        cudaFuncSetAttribute(k_lift_z, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        for (auto* k : {k_zrow<ZR_FWD>, k_zrow<ZR_PROJ>, k_zrow<ZR_BWD>})
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        cudaFuncSetAttribute(k_grad_w, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        cudaFuncSetAttribute(k_proj_bwd<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        cudaFuncSetAttribute(k_proj_bwd<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        for (auto* k : {k_fold_fwd<4>, k_fold_fwd<5>, k_fold_fwd<6>, k_fold_fwd<7>, k_fold_fwd<8>})
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        cudaFuncSetAttribute(k_fold_inv, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        cudaFuncSetAttribute(k_lift_u, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        cudaFuncSetAttribute(k_mix<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        cudaFuncSetAttribute(k_mix<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        cudaFuncSetAttribute(k_mix_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        cudaFuncSetAttribute(k_near_add<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        cudaFuncSetAttribute(k_near_add<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        cudaFuncSetAttribute(k_near_add<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        cudaFuncSetAttribute(k_near_add<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        cudaFuncSetAttribute(k_near_add<5>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        cudaFuncSetAttribute(k_near_add<6>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        cudaFuncSetAttribute(k_near_add<7>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        if (cudaGetLastError() != cudaSuccess) {
            set_error("sno_create: cannot configure the kernels");
            delete h;
            return KIFMM_ERR_CUDA;
        }
    }
    int rc = KIFMM_OK;
    for (auto* pr : {&M.theta, &M.grad, &M.adam_m, &M.adam_v}) {
        rc = dev_alloc(*pr, M.nparam * 4);
        if (rc) return fail(rc);
        if (cudaMemsetAsync(pr->p, 0, M.nparam * 4, M.st) != cudaSuccess) return fail(KIFMM_ERR_CUDA);
    }
    if ((rc = dev_alloc(M.rbf, (size_t)layers * 2 * M.K * width * width * 2))) return fail(rc);
    M.tzf = 0;
    M.tyf = M.tzf + (int64_t)modes * n;
    M.tfo = M.tyf + (int64_t)2 * modes * n;
    M.tph = M.tfo + (int64_t)n / 2 * (modes + 1);
    if ((rc = dev_alloc(M.tabs, (M.tph + modes + 1) * sizeof(float2)))) return fail(rc);
    M.period = n;
    k_tables<<<nbs(2 * modes * n, 128), 128, 0, M.st>>>(n, n, modes, ptr<float2>(M.tabs), M.tzf, M.tyf, M.tfo,
                                                          M.tph);
    if (cudaGetLastError() != cudaSuccess) return fail(KIFMM_ERR_CUDA);
    if ((rc = dev_alloc(M.v, (size_t)(layers + 1) * per * 4))) return fail(rc);
    if ((rc = dev_alloc(M.z, (size_t)layers * per * 4))) return fail(rc);
    if ((rc = dev_alloc(M.dz, (size_t)2 * per * 4))) return fail(rc);
    if ((rc = dev_alloc(M.yb, (size_t)max_batch * M.np3 * 4))) return fail(rc);
    if ((rc = dev_alloc(M.dy, (size_t)max_batch * M.np3 * 4))) return fail(rc);
    if ((rc = dev_alloc(M.cz, (size_t)BC * n * n * modes * 8))) return fail(rc);
    if ((rc = dev_alloc(M.cy, (size_t)BC * n * 2 * modes * modes * 8))) return fail(rc);
    if ((rc = dev_alloc(M.gx, (size_t)BC * n * 2 * modes * modes * 8))) return fail(rc);
    if ((rc = dev_alloc(M.gy, (size_t)BC * n * n * modes * 8))) return fail(rc);
    if ((rc = dev_alloc(M.Vst, (size_t)layers * BC * M.K * 8))) return fail(rc);
    if ((rc = dev_alloc(M.g, (size_t)BC * M.K * 8))) return fail(rc);
    if ((rc = dev_alloc(M.ga, (size_t)BC * M.K * 8))) return fail(rc);
    if ((rc = dev_alloc(M.m0ab, (size_t)2 * width * M.K * 8))) return fail(rc);
    if ((rc = dev_alloc(M.loss, 16))) return fail(rc);
    // judge buffers for a batch of max_batch fields: targets, references, caller indices, errors, scales
    if ((rc = dev_alloc(M.jt, (size_t)max_batch * SNO_MAX_JUDGE * 4))) return fail(rc);
    if ((rc = dev_alloc(M.jref, (size_t)max_batch * SNO_MAX_JUDGE * 8))) return fail(rc);
    if ((rc = dev_alloc(M.jorig, (size_t)max_batch * SNO_MAX_JUDGE * 4))) return fail(rc);
    if ((rc = dev_alloc(M.jerr, (size_t)max_batch * 8))) return fail(rc);
    if ((rc = dev_alloc(M.scal, (size_t)max_batch * 8 + 8))) return fail(rc);
    {   // judge work space: the target draw's (reused field by field), then per field the
        // weights and the targets' sums (8 k each)
        const size_t ws = importance_ws_bytes(M.np3, SNO_MAX_JUDGE) + 2 * 8 * (size_t)max_batch * SNO_MAX_JUDGE;
        if ((rc = dev_alloc(M.jws, ws))) return fail(rc);
    }
    if (cudaStreamSynchronize(M.st) != cudaSuccess) return fail(KIFMM_ERR_CUDA);
    *out = h;
    return KIFMM_OK;
}

int sno_set_period(sno_model_t h, int period) {
    set_error("");
    if (!h) return KIFMM_ERR_ARG;
    SnoModel& M = h->m;
    if (period < M.n || period > 4 * M.n || 2 * M.m > period) {
        set_error("sno_set_period: need n <= period <= 4 n and 2 modes <= period");
        return KIFMM_ERR_ARG;
    }
    M.period = period;
    k_tables<<<nbs(2 * M.m * M.n, 128), 128, 0, M.st>>>(M.n, period, M.m, ptr<float2>(M.tabs), M.tzf, M.tyf, M.tfo,
                                                          M.tph);
    KF_LAUNCH();
    KF_CUDA(cudaStreamSynchronize(M.st));
    return KIFMM_OK;
}

int sno_set_near_field(sno_model_t h, double a, double b, double cell_h, int self_mode, double r_in, double r_out) {
    set_error("");
    if (!h) return KIFMM_ERR_ARG;
    SnoModel& M = h->m;
    if (a == 0.0 && b == 0.0) {   // off
        M.near_on = 0;
        return KIFMM_OK;
    }
    if (!(a > 0.0) || !(b > a) || !std::isfinite(b) || !(cell_h > 0.0) || !std::isfinite(cell_h) ||
        (self_mode != KIFMM_SELF_CELL_EXACT && self_mode != KIFMM_SELF_PAPER_GL2) || !(r_in >= 0.0) ||
        !(r_out > r_in) || !(r_out <= 8.0)) {
        set_error("sno_set_near_field: need 0 < a < b, h > 0, a known self_mode and 0 <= r_in < r_out <= 8");
        return KIFMM_ERR_ARG;
    }
    // (taps at r_out itself are zero)
    const int R = r_out < 1.0 ? 0 : std::max(1, (int)std::ceil(r_out) - 1), side = 2 * R + 1;
    const int64_t nc = (int64_t)side * side * side;
    DevBuf tap, sig;
    KF_TRY(dev_alloc(tap, nc * 8));
    int rc = dev_alloc(sig, 8);
    if (rc) {
        dev_free(tap);
        return rc;
    }
    k_near_taps<<<nbs(nc, 256), 256, 0, M.st>>>(R, make_kparams(a, b), cell_h, r_in, r_out, self_mode,
                                               ptr<double>(tap), ptr<double>(sig));
    std::vector<double> tv(nc);
    double sv = 0.0;
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(tv.data(), tap.p, nc * 8, cudaMemcpyDeviceToHost, M.st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&sv, sig.p, 8, cudaMemcpyDeviceToHost, M.st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(M.st);
    dev_free(tap);
    dev_free(sig);
    KF_CUDA(e);
    // stencil columns (di, dj) on the [i][j][k] grid, in groups of equal max and min of |di|, |dj|: a
    // group's taps are the same, the 2R + 1 over dk = -R..R (sigma at the centre; zero outside the
    // sphere); groups without a nonzero tap are left out
    tv[(size_t)R * side * side + (size_t)R * side + R] = sv;
    std::vector<int2> bounds, cd;
    std::vector<float> cw;
    for (int hi = 0; hi <= R; ++hi)
        for (int lo = 0; lo <= hi; ++lo) {
            const double* col = tv.data() + ((size_t)(hi + R) * side + (lo + R)) * side;
            bool any = false;
            for (int t = 0; t < side; ++t) any = any || col[t] != 0.0;
            if (!any) continue;
            bounds.push_back(make_int2((int)cd.size(), 0));
            for (int di = -hi; di <= hi; ++di)
                for (int dj = -hi; dj <= hi; ++dj)
                    if (std::max(std::abs(di), std::abs(dj)) == hi && std::min(std::abs(di), std::abs(dj)) == lo)
                        cd.push_back(make_int2(di, dj));
            for (int t = 0; t < side; ++t) cw.push_back((float)col[t]);
        }
    const int ng = (int)bounds.size(), ncol = (int)cd.size();
    bounds.push_back(make_int2(ncol, 0));
    cd.insert(cd.begin(), bounds.begin(), bounds.end());
    dev_free(M.near_d);
    dev_free(M.near_w);
    KF_TRY(dev_alloc(M.near_d, cd.size() * sizeof(int2)));
    KF_TRY(dev_alloc(M.near_w, cw.size() * 4));
    KF_CUDA(cudaMemcpyAsync(M.near_d.p, cd.data(), cd.size() * sizeof(int2), cudaMemcpyHostToDevice, M.st));
    KF_CUDA(cudaMemcpyAsync(M.near_w.p, cw.data(), cw.size() * 4, cudaMemcpyHostToDevice, M.st));
    KF_CUDA(cudaStreamSynchronize(M.st));
    M.na = a;
    M.nb = b;
    M.nh = cell_h;
    M.nsig = sv;
    M.nr_in = r_in;
    M.nr_out = r_out;
    M.nself = self_mode;
    M.nR = R;
    M.ngroups = ng;
    M.ntaps = ncol;
    M.near_on = 1;
    return KIFMM_OK;
}

int sno_init_far_field(sno_model_t h, double shift) {
    set_error("");
    if (!h) return KIFMM_ERR_ARG;
    SnoModel& M = h->m;
    if (!M.near_on || !(shift > 0.0) || !std::isfinite(shift)) {
        set_error("sno_init_far_field: needs the near part (sno_set_near_field) and shift > 0");
        return KIFMM_ERR_ARG;
    }
    const int N = M.period, m = M.m, C = M.C, P = M.P;
    const int64_t nA = (int64_t)N * N * m, nB = (int64_t)N * 2 * m * m, K = M.K;
    DevBuf A, Bf, Mk;
    KF_TRY(dev_alloc(A, nA * 8));
    int rc = dev_alloc(Bf, nB * 8);
    if (!rc) rc = dev_alloc(Mk, K * 8);
    std::vector<double> mult(K);
    if (!rc) {
        const KParams kp = make_kparams(M.na, M.nb);
        k_far_pass_z<<<nbs(nA, 128), 128, 0, M.st>>>(N, m, kp, M.nh, M.nr_in, M.nr_out, ptr<double>(A));
        k_far_pass_y<<<nbs(nB, 128), 128, 0, M.st>>>(N, m, ptr<double>(A), ptr<double>(Bf));
        k_far_pass_x<<<nbs(K, 128), 128, 0, M.st>>>(N, m, ptr<double>(Bf), ptr<double>(Mk));
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(mult.data(), Mk.p, K * 8, cudaMemcpyDeviceToHost, M.st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(M.st);
        if (e != cudaSuccess) {
            set_error(std::string("sno_init_far_field: ") + cudaGetErrorString(e));
            rc = KIFMM_ERR_CUDA;
        }
    }
    dev_free(A);
    dev_free(Bf);
    dev_free(Mk);
    KF_TRY(rc);
    // channel 0 carries the far convolution: lift 1; layer 0 spectral weight M(k) at (0, 0) and
    // bias `shift` (GELU(shift + x) = shift + x to 1e-12 for |x| <= 2); later layers pass it
    // through (W[0][0] = 1); projection row 0 reads it and q2 removes the shift. Every weight
    // into or out of channel 0 and projection row 0 other than these is 0; the others keep
    // their values.
    std::vector<float> th(M.nparam);
    KF_CUDA(cudaMemcpyAsync(th.data(), M.theta.p, M.nparam * 4, cudaMemcpyDeviceToHost, M.st));
    KF_CUDA(cudaStreamSynchronize(M.st));
    float* t = th.data();
    t[M.off[O_WL]] = 1.f;
    t[M.off[O_BL]] = 0.f;
    for (int l = 0; l < M.L; ++l) {
        float* Rr = t + M.off[o_rr(l)];
        float* Ri = t + M.off[o_ri(l)];
        float* W = t + M.off[o_w(l)];
        for (int64_t k = 0; k < K; ++k)
            for (int c = 0; c < C; ++c) {
                Rr[(k * C + 0) * C + c] = Ri[(k * C + 0) * C + c] = 0.f;
                Rr[(k * C + c) * C + 0] = Ri[(k * C + c) * C + 0] = 0.f;
            }
        for (int c = 0; c < C; ++c) W[0 * C + c] = W[c * C + 0] = 0.f;
        if (l == 0)
            for (int64_t k = 0; k < K; ++k) Rr[k * C * C] = (float)mult[k];
        else
            W[0] = 1.f;
        t[M.off[o_b(l)]] = l == 0 ? (float)shift : 0.f;
    }
    const int q = o_q1(M);
    float* Q1 = t + M.off[q];
    for (int p = 0; p < P; ++p) Q1[p * C + 0] = 0.f;
    for (int c = 0; c < C; ++c) Q1[0 * C + c] = 0.f;
    Q1[0] = 1.f;
    t[M.off[q + 1]] = 0.f;
    t[M.off[q + 2]] = 1.f;
    t[M.off[q + 3]] = (float)-shift;
    return sno_set_params(h, th.data());
}

void sno_destroy(sno_model_t h) {
    if (!h) return;
    SnoModel& M = h->m;
    if (M.st) cudaStreamSynchronize(M.st);
    for (DevBuf* b : {&M.theta, &M.grad, &M.adam_m, &M.adam_v, &M.rbf, &M.tabs, &M.v, &M.z, &M.dz, &M.yb, &M.dy,
                      &M.loss, &M.cz, &M.cy, &M.gx, &M.gy, &M.Vst, &M.g, &M.ga, &M.m0ab, &M.jt, &M.jref, &M.jorig,
                      &M.jerr, &M.near_d, &M.near_w, &M.scal, &M.jws})
        dev_free(*b);
    delete h;
}

int64_t sno_num_params(sno_model_t h) { return h ? h->m.nparam : -1; }

int sno_set_params(sno_model_t h, const float* theta_host) {
    if (!h || !theta_host) {
        set_error("sno_set_params: invalid argument");
        return KIFMM_ERR_ARG;
    }
    SnoModel& M = h->m;
    KF_CUDA(cudaMemcpyAsync(M.theta.p, theta_host, M.nparam * 4, cudaMemcpyHostToDevice, M.st));
    KF_CUDA(cudaMemsetAsync(M.adam_m.p, 0, M.nparam * 4, M.st));
    KF_CUDA(cudaMemsetAsync(M.adam_v.p, 0, M.nparam * 4, M.st));
    M.steps = 0;
    KF_TRY(refresh_bf16(M));
    KF_CUDA(cudaStreamSynchronize(M.st));
    return KIFMM_OK;
}

int sno_get_params(sno_model_t h, float* theta_host) {
    if (!h || !theta_host) return KIFMM_ERR_ARG;
    KF_CUDA(cudaMemcpyAsync(theta_host, h->m.theta.p, h->m.nparam * 4, cudaMemcpyDeviceToHost, h->m.st));
    KF_CUDA(cudaStreamSynchronize(h->m.st));
    return KIFMM_OK;
}

int sno_get_grads(sno_model_t h, float* grad_host) {
    if (!h || !grad_host) return KIFMM_ERR_ARG;
    KF_CUDA(cudaMemcpyAsync(grad_host, h->m.grad.p, h->m.nparam * 4, cudaMemcpyDeviceToHost, h->m.st));
    KF_CUDA(cudaStreamSynchronize(h->m.st));
    return KIFMM_OK;
}

// file: "SNO1", int32 n, width, modes, layers, proj_width, int64 parameter count, FP32 parameters
int sno_save(sno_model_t h, const char* path) {
    set_error("");
    if (!h || !path) return KIFMM_ERR_ARG;
    SnoModel& M = h->m;
    std::vector<float> th(M.nparam);
    KF_CUDA(cudaMemcpyAsync(th.data(), M.theta.p, M.nparam * 4, cudaMemcpyDeviceToHost, M.st));
    KF_CUDA(cudaStreamSynchronize(M.st));
    FILE* fp = fopen(path, "wb");
    if (!fp) {
        set_error("sno_save: cannot open the file");
        return KIFMM_ERR_ARG;
    }
    const int32_t hdr[6] = {0x314f4e53, M.n, M.C, M.m, M.L, M.P};
    bool ok = fwrite(hdr, 4, 6, fp) == 6 && fwrite(&M.nparam, 8, 1, fp) == 1 &&
              fwrite(th.data(), 4, M.nparam, fp) == (size_t)M.nparam;
    ok = (fclose(fp) == 0) && ok;
    if (!ok) {
        set_error("sno_save: write failed");
        return KIFMM_ERR_ARG;
    }
    return KIFMM_OK;
}

int sno_load(sno_model_t h, const char* path) {
    set_error("");
    if (!h || !path) return KIFMM_ERR_ARG;
    SnoModel& M = h->m;
    FILE* fp = fopen(path, "rb");
    if (!fp) {
        set_error("sno_load: cannot open the file");
        return KIFMM_ERR_ARG;
    }
    int32_t hdr[6] = {0};
    int64_t np = -1;
    std::vector<float> th(M.nparam);
    bool ok = fread(hdr, 4, 6, fp) == 6 && fread(&np, 8, 1, fp) == 1;
    ok = ok && hdr[0] == 0x314f4e53 && hdr[1] == M.n && hdr[2] == M.C && hdr[3] == M.m && hdr[4] == M.L &&
         hdr[5] == M.P && np == M.nparam;
    ok = ok && fread(th.data(), 4, M.nparam, fp) == (size_t)M.nparam;
    fclose(fp);
    if (!ok) {
        set_error("sno_load: not a parameter file of this model's shape");
        return KIFMM_ERR_ARG;
    }
    return sno_set_params(h, th.data());
}

// checkpoint: "SNO2", the sizes as in "SNO1", int64 parameter count, int64 Adam step count,
// then the FP32 parameters and Adam's first and second moments (training resumes exactly)
int sno_save_checkpoint(sno_model_t h, const char* path) {
    set_error("");
    if (!h || !path) return KIFMM_ERR_ARG;
    SnoModel& M = h->m;
    const size_t np = (size_t)M.nparam;
    std::vector<float> buf(3 * np);
    KF_CUDA(cudaMemcpyAsync(buf.data(), M.theta.p, np * 4, cudaMemcpyDeviceToHost, M.st));
    KF_CUDA(cudaMemcpyAsync(buf.data() + np, M.adam_m.p, np * 4, cudaMemcpyDeviceToHost, M.st));
    KF_CUDA(cudaMemcpyAsync(buf.data() + 2 * np, M.adam_v.p, np * 4, cudaMemcpyDeviceToHost, M.st));
    KF_CUDA(cudaStreamSynchronize(M.st));
    FILE* fp = fopen(path, "wb");
    if (!fp) {
        set_error("sno_save_checkpoint: cannot open the file");
        return KIFMM_ERR_ARG;
    }
    const int32_t hdr[6] = {0x324f4e53, M.n, M.C, M.m, M.L, M.P};
    bool ok = fwrite(hdr, 4, 6, fp) == 6 && fwrite(&M.nparam, 8, 1, fp) == 1 && fwrite(&M.steps, 8, 1, fp) == 1 &&
              fwrite(buf.data(), 4, buf.size(), fp) == buf.size();
    ok = (fclose(fp) == 0) && ok;
    if (!ok) {
        set_error("sno_save_checkpoint: write failed");
        return KIFMM_ERR_ARG;
    }
    return KIFMM_OK;
}

int sno_load_checkpoint(sno_model_t h, const char* path) {
    set_error("");
    if (!h || !path) return KIFMM_ERR_ARG;
    SnoModel& M = h->m;
    FILE* fp = fopen(path, "rb");
    if (!fp) {
        set_error("sno_load_checkpoint: cannot open the file");
        return KIFMM_ERR_ARG;
    }
    const size_t np = (size_t)M.nparam;
    int32_t hdr[6] = {0};
    int64_t nfile = -1, steps = -1;
    std::vector<float> buf(3 * np);
    bool ok = fread(hdr, 4, 6, fp) == 6 && fread(&nfile, 8, 1, fp) == 1 && fread(&steps, 8, 1, fp) == 1;
    ok = ok && hdr[0] == 0x324f4e53 && hdr[1] == M.n && hdr[2] == M.C && hdr[3] == M.m && hdr[4] == M.L &&
         hdr[5] == M.P && nfile == M.nparam && steps >= 0;
    ok = ok && fread(buf.data(), 4, buf.size(), fp) == buf.size();
    fclose(fp);
    if (!ok) {
        set_error("sno_load_checkpoint: not a checkpoint of this model's shape");
        return KIFMM_ERR_ARG;
    }
    KF_TRY(sno_set_params(h, buf.data()));   // parameters and their BF16 copies (clears the moments)
    KF_CUDA(cudaMemcpyAsync(M.adam_m.p, buf.data() + np, np * 4, cudaMemcpyHostToDevice, M.st));
    KF_CUDA(cudaMemcpyAsync(M.adam_v.p, buf.data() + 2 * np, np * 4, cudaMemcpyHostToDevice, M.st));
    KF_CUDA(cudaStreamSynchronize(M.st));
    M.steps = steps;
    return KIFMM_OK;
}

int sno_set_bf16(sno_model_t h, int on) {
    if (!h) return KIFMM_ERR_ARG;
    h->m.bf16 = on ? 1 : 0;
    return refresh_bf16(h->m);
}

int sno_forward(sno_model_t h, const float* u_dev, float* y_dev, int batch) {
    if (!h || !u_dev || !y_dev || batch < 1 || batch > h->m.maxB) {
        set_error("sno_forward: invalid argument");
        return KIFMM_ERR_ARG;
    }
    return forward(h->m, u_dev, y_dev, batch, false);
}

int sno_loss_grad(sno_model_t h, const float* u_dev, const float* t_dev, int batch, double* loss) {
    if (!h || !u_dev || !t_dev || batch < 1 || batch > h->m.maxB) {
        set_error("sno_loss_grad: invalid argument");
        return KIFMM_ERR_ARG;
    }
    return loss_grad(h->m, u_dev, t_dev, batch, loss);
}

int sno_adam_step(sno_model_t h, float lr, float beta1, float beta2, float eps) {
    if (!h) return KIFMM_ERR_ARG;
    SnoModel& M = h->m;
    M.steps += 1;
    const float c1 = 1.f - powf(beta1, (float)M.steps), c2 = 1.f - powf(beta2, (float)M.steps);
    k_adam<<<nbs(M.nparam, 256), 256, 0, M.st>>>(ptr<float>(M.theta), ptr<float>(M.grad), ptr<float>(M.adam_m),
                                                 ptr<float>(M.adam_v), M.nparam, lr, beta1, beta2, eps, c1, c2);
    KF_LAUNCH();
    return refresh_bf16(M);
}

// Surrogate-first solves of `count` fields (one plan each, the model's grid) on plans[0]'s
// stream: the batched forward pass, then per field the importance-sampled judge, then one
// FMM batch for the fields judged above tol.
static int photo_solve_impl(kifmm_plan_t* plans, int count, SnoModel& M, const double* const* I, double* const* S,
                            const double* Cs, double tol, int k_samples, uint64_t seed, int* used_fallback,
                            double* judged_err) {
    if (!plans || count < 1 || count > M.maxB || !I || !S || k_samples < 1 || k_samples > SNO_MAX_JUDGE) {
        set_error("photo_solve: invalid argument");
        return KIFMM_ERR_ARG;
    }
    for (int b = 0; b < count; ++b) {
        if (!plans[b] || !I[b] || !S[b]) {
            set_error("photo_solve: invalid argument");
            return KIFMM_ERR_ARG;
        }
        Plan& p = *kifmm_plan_internal(plans[b]);
        if (p.n_real != p.tree.n) {
            set_error("photo_solve: the plan holds padding cells (pad_lattice); the surrogate's grid is the plan's own");
            return KIFMM_ERR_ARG;
        }
        if (p.tree.n != M.np3) {
            set_error("photo_solve: the plan's point count differs from the model's grid");
            return KIFMM_ERR_ARG;
        }
        if (p.kind != 0) {
            set_error("photo_solve: the surrogate and its judge take the paper's kernel");
            return KIFMM_ERR_ARG;
        }
        if (M.near_on) {   // the model's near part must be the plan's kernel and cells
            auto same = [](double x, double y) { return std::fabs(x - y) <= 1e-12 * std::fabs(y); };
            if (!same(M.na, p.a) || !same(M.nb, p.b) || !same(M.nh, p.uniform_h) || p.self_mode != M.nself) {
                set_error("photo_solve: the model's near part was set for another kernel, cell size or self term");
                return KIFMM_ERR_ARG;
            }
        }
    }
    const int64_t n = M.np3;
    const int K = SNO_MAX_JUDGE;
    cudaStream_t st = kifmm_plan_internal(plans[0])->stream;
    cudaStream_t saved = M.st;
    M.st = st;
    // surrogate in the amplitude-normalised linear form: s = max |I|, u = I / s (caller's
    // grid order), S = C s y
    float* u = ptr<float>(M.dz);
    float* y = ptr<float>(M.yb);
    double* sc = ptr<double>(M.scal);
    KF_CUDA(cudaMemsetAsync(sc, 0, (size_t)count * 8, st));
    for (int b = 0; b < count; ++b) {
        k_sno_absmax<<<std::min<int64_t>(nbs(n, 256), 4LL * M.num_sms), 256, 0, st>>>(
            I[b], n, reinterpret_cast<unsigned long long*>(sc + b));
        k_scale_in<<<nbs(n, 256), 256, 0, st>>>(I[b], sc + b, u + b * n, n);
    }
    KF_LAUNCH();
    int rc = forward(M, u, y, count, false);
    M.st = saved;
    KF_TRY(rc);
    for (int b = 0; b < count; ++b) {
        const double C = Cs ? Cs[b] : 1.0;
        k_scale_out<<<nbs(n, 256), 256, 0, st>>>(y + b * n, sc + b, C, S[b], n);
    }
    KF_LAUNCH();
    // judge: the direct sum at k targets drawn with probability m_i = 0.5 |S_i| / sum |S| + 0.5 / n
    // (systematic sampling from the surrogate's own field, offset from a fixed LCG of seed + b),
    // each weighted 1 / (k m_i): an importance-sampled estimate of the whole field's relative
    // L2 error that does not miss a concentrated source the way uniform samples do
    double* wts = reinterpret_cast<double*>(static_cast<char*>(M.jws.p) + importance_ws_bytes(n, K));
    double* accs = wts + (size_t)M.maxB * K;
    KF_CUDA(cudaMemsetAsync(accs, 0, (size_t)count * K * 8, st));
    for (int b = 0; b < count; ++b) {
        Plan& p = *kifmm_plan_internal(plans[b]);
        const double C = Cs ? Cs[b] : 1.0;
        int32_t* tb = ptr<int32_t>(M.jt) + (size_t)b * K;
        double* wb = wts + (size_t)b * K;
        double* ab = accs + (size_t)b * K;
        KF_TRY(importance_targets(st, S[b], n, k_samples, seed + (uint64_t)b, ptr<int32_t>(p.tree.perm), n, M.jws.p,
                                  nullptr, tb, wb, M.num_sms));
        // weights q = I h^3 in sorted order (the evaluation's own scatter kernel)
        KF_TRY(kifmm_scatter_weights(p, I[b], st));
        k_judge_src<<<nbs(n, JG_CH), JG_T, 0, st>>>(ptr<double>(p.pts), ptr<double>(p.q), tb, k_samples, n,
                                                      make_kparams(p.a, p.b), ab);
        k_judge_fin<<<nbs(k_samples, 128), 128, 0, st>>>(ab, tb, k_samples, ptr<double>(p.sigma), ptr<double>(p.Isort),
                                                         C, ptr<int32_t>(p.tree.perm), ptr<double>(M.jref) + (size_t)b * K,
                                                         ptr<int32_t>(M.jorig) + (size_t)b * K);
        k_judge_err<<<1, 256, 0, st>>>(S[b], ptr<double>(M.jref) + (size_t)b * K, ptr<int32_t>(M.jorig) + (size_t)b * K,
                                       wb, k_samples, ptr<double>(M.jerr) + b);
        KF_LAUNCH();
    }
    std::vector<double> err(count);
    KF_CUDA(cudaMemcpyAsync(err.data(), M.jerr.p, (size_t)count * 8, cudaMemcpyDeviceToHost, st));
    KF_CUDA(cudaStreamSynchronize(st));
    std::vector<kifmm_plan_t> fp;
    std::vector<const void*> fi;
    std::vector<void*> fs;
    std::vector<double> fc;
    for (int b = 0; b < count; ++b) {
        const int fb = !(err[b] <= tol);
        if (judged_err) judged_err[b] = err[b];
        if (used_fallback) used_fallback[b] = fb;
        if (fb) {
            fp.push_back(plans[b]);
            fi.push_back(I[b]);
            fs.push_back(S[b]);
            fc.push_back(Cs ? Cs[b] : 1.0);
        }
    }
    if (!fp.empty()) {   // the FMM for the rejected fields, as one batch (ordered on st after the judge)
        const int nf = (int)fp.size();
        KF_TRY(kifmm_eval_batch(fp.data(), fi.data(), fs.data(), nf, KIFMM_F64, fc.data(), 0,
                                std::min(nf, KIFMM_MAX_LANES)));
        KF_CUDA(cudaStreamSynchronize(kifmm_plan_internal(fp[0])->stream));
    }
    return KIFMM_OK;
}

int photo_solve(kifmm_plan_t plan, sno_model_t model, const double* I_dev, double* S_dev, double C, double tol,
                int k_samples, uint64_t seed, int* used_fallback, double* judged_err) {
    set_error("");
    if (!plan || !model || !I_dev || !S_dev) {
        set_error("photo_solve: invalid argument");
        return KIFMM_ERR_ARG;
    }
    double* Sp = S_dev;
    return photo_solve_impl(&plan, 1, model->m, &I_dev, &Sp, &C, tol, k_samples, seed, used_fallback, judged_err);
}

int photo_solve_batch(kifmm_plan_t* plans, int count, sno_model_t model, const double* const* I_dev,
                      double* const* S_dev, const double* C, double tol, int k_samples, uint64_t seed,
                      int* used_fallback, double* judged_err) {
    set_error("");
    if (!model) {
        set_error("photo_solve_batch: invalid argument");
        return KIFMM_ERR_ARG;
    }
    return photo_solve_impl(plans, count, model->m, I_dev, S_dev, C, tol, k_samples, seed, used_fallback,
                            judged_err);
}

}  // extern "C"
