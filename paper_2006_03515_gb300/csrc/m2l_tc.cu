// M2L (Eq. (m2l)) on the 5th-generation tensor cores: a 3-term FP16 split with FP32
// accumulation (x = x_hi + x_lo, both FP16 with the 11-bit significand of TF32, products
// hi*hi + hi*lo + lo*hi), so the result carries the accuracy of a 3xTF32 product at half
// the operand bytes and twice the MMA rate of kind::tf32. FP16's exponent range is handled by
// exact power-of-two scaling: each box's coefficient row c[A] by 2^{e_A} and each level's T
// table by 2^{e_T} (largest magnitude near 2^14); the epilogue undoes 2^{e_A + e_T} per slot.
//
// In the coefficient basis the translation of one level is, for every target box B,
//   d[B] = sum over the offset slots of V(B):  T[slot] c[A(B, slot)],
// with T[slot] (R x R) shared by every pair with that relative offset. One CTA takes a
// tile of 128 target boxes of a level (boxes grouped by their octant inside the parent,
// so that the tile's boxes share one set of about 189 offsets) and a block of NT <= 256
// output rows (one block when R <= 256), and, per offset slot and 32-wide k-chunk,
// multiplies the gathered source rows c[A] (A operand, 128 x 32) by the chunk's rows of
// T[slot] (B operand, NT x 32), both K-major in the 128-byte swizzled layout. A 128-byte row
// holds the chunk's 32 hi halves, then its 32 lo halves, in global memory as in shared memory:
// a source row's piece is one line, a stage 16 KB + NT 128 B, and six stages of R = 128 fit (with
// 64-wide chunks and hi and lo apart, three of 64 KB did: a slot waited for the refill of a stage).
//
// The launch's work is the sequence of all (tile, offset slot) pairs, tile after tile; CTA c of n
// takes the slots [c T / n, (c + 1) T / n) of the T in it, so that every SM gets the same number
// whatever the tile count (a 32^3 grid has 5 tiles of about 250 slots, a 128^3 grid 293 of 189).
// A tile that lies wholly in one CTA's range is written to d; the pieces of a tile that is cut go
// to a work space and k_tc_finish adds them in slot order (no atomics: the result is the same
// on every run).
//
// Roles (warp specialization, 10 + PW warps):
//  * index warp: source box and scale 2^{-(e_A + e_T)} of the tile's 128 rows for each slot, four
//    slots at a time, into a ring in shared memory. The sources of every slot are tabulated at plan
//    time in the launch's order, so their loads are contiguous and run a group ahead; only the
//    exponents are gathered. In the consumers, the chain of dependent look-ups (slot, source box,
//    exponent) stalled every slot by two or three L2 latencies.
//  * PW producer warps: eight lanes copy one source row's 128-byte piece with 16-byte cp.async
//    (zero-filled where the box has no source at this offset), so a warp instruction touches four
//    lines; with a row per lane it touched 32. Thread 0 also moves the pre-swizzled B chunk with one
//    1-D bulk copy. A thread's arrival on the stage's "full" mbarrier is left to the hardware, when its
//    copies are there (cp.async.mbarrier.arrive.noinc), so it goes on to the next free stage at once.
//  * MMA warp, lane 0: waits for a full stage, issues its k-steps x 3 MMAs into the slot's two
//    tensor-memory accumulators (hi x hi terms; cross terms) and commits the stage's "empty"
//    mbarrier; after the last chunk of a slot it commits the accumulators' "ready" mbarrier. MMAs are
//    issued nearly in step with their execution, so the thread tests the next stage's and the next
//    slot's mbarriers before it issues the current MMAs (waiting where they were used, and with the
//    descriptors formed in 64 bits, it took 4300 cycles a slot for 1536 of MMAs).
//  * warps 0-7, epilogue: rings of accumulators take the slots in turn; the epilogue scales a
//    finished pair by the slot's 2^{-(e_A + e_T)} into FP32 registers (round-to-nearest) and
//    releases it. The tensor core's own (truncating) accumulation thus spans the R / 16 hi x hi
//    products of one slot: the cross terms, 2^-11 of them, are summed apart. (In one accumulator
//    a slot of R = 128 took 24 truncating additions, and the mixed form's error at 7.6 Torr
//    followed their order: 8.9e-7 of FP64 with the cross terms of 64 columns first, 1.07e-6 with
//    those of 32 first.)
// Measured on one GB300 (ncu, cold cache), before and after these changes: the 6.0 M V pairs of 128^3
// (R = 128) 985 -> 599 us, one wave of the chip at 64^3 506 -> 92 us, 1250 slots in five tiles at 32^3
// 507 -> 25 us, the near field's 6912 slots at 128^3 (R = 64) 78 -> 50 us. At 128^3 the tensor pipe is
// active half of the time; the MMA thread's waits and proxy fences take most of the rest.
// Every wait is bounded; a timeout sets an abort flag that ends the other roles' waits (lanes whose wait
// ran out go through their role's warp-wide instructions all the same, or leave by the warp's vote),
// records an error code, and the tensor memory is freed before the CTA exits.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "internal.cuh"
#include "tc_split.h"
#include "tcgen05.cuh"

namespace kifmm {

constexpr int TC_M = 128;                 // target boxes per tile = MMA M
constexpr int TC_KC = 32;                 // k-chunk: 32 hi and 32 lo FP16 = one 128-byte swizzle row
constexpr int TC_HI_EXP = 14;             // scaled operands keep their largest magnitude near 2^14
constexpr int TC_EPI = 256;               // epilogue threads (warps 0-7)
constexpr int TC_RING = 8;                // slots whose source indices and scales are held in shared memory
constexpr int TC_GRP = 4;                 // slots the index warp looks up at a time
constexpr int TC_PW = 2;                  // producer warps
constexpr int TC_THREADS = TC_EPI + 32 * TC_PW + 64;

// ------------------------------------------------------------------------------------
// plan and per-evaluation operand preparation
// ------------------------------------------------------------------------------------
// largest |T| of a level's table, as the bits of a non-negative double (ordered like integers)
__global__ void k_absmax(const double* x, int64_t n, unsigned long long* out) {
    double m = 0.0;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
        m = fmax(m, fabs(x[e]));
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, (unsigned long long)__double_as_longlong(m));
}

// T (FP64 [nslots][R][R]) * 2^sT as FP16 hi / lo in the order [slot][k-chunk][row][128-byte swizzled
// row of 32 hi, 32 lo], so that one chunk of one slot is a contiguous R * 128-byte image of the
// shared-memory B tile.
__global__ void k_swizzle_T(const double* T, int R, int nslots, int sT, __half* out) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t per = (int64_t)R * R;
    if (e >= (int64_t)nslots * per) return;
    const int64_t slot = e / per;
    const int row = (int)((e % per) / R), k = (int)(e % R);
    const float x = (float)ldexp(T[e], sT);
    const __half h = __float2half_rn(x);
    char* o = reinterpret_cast<char*>(out) + (slot * (R / TC_KC) + k / TC_KC) * (int64_t)R * 128;
    *reinterpret_cast<__half*>(o + sw128_off_h(row, k % TC_KC)) = h;
    *reinterpret_cast<__half*>(o + sw128_off_h(row, TC_KC + k % TC_KC)) = __float2half_rn(x - __half2float(h));
}

// coefficient rows (R values) scaled by 2^{e_b} per box (largest magnitude near 2^14) and split
// into FP16 hi / lo: rows of 2 ldo halves, per 32 columns the 32 hi then the 32 lo (columns
// R..ldo-1 zero); one warp per box
template <class TIN>
__global__ void k_split_c(const TIN* c, int64_t nb, int R, __half* out, int* cexp, int ldo) {
    const int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (b >= nb) return;
    const TIN* row = c + b * R;
    float m = 0.f;
    for (int k = lane; k < R; k += 32) m = fmaxf(m, fabsf((float)row[k]));
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    int e = 0;
    if (m > 0.f) {
        int ex;
        frexpf(m, &ex);             // m = f 2^ex, f in [0.5, 1)
        e = TC_HI_EXP + 1 - ex;     // m 2^e in [2^13, 2^14)
    }
    __half* o = out + b * 2 * ldo;
    for (int k = lane; k < ldo; k += 32) {
        const float x = k < R ? ldexpf((float)row[k], e) : 0.f;
        const __half h = __float2half_rn(x);
        o[2 * (k - lane) + lane] = h;
        o[2 * (k - lane) + TC_KC + lane] = __float2half_rn(x - __half2float(h));
    }
    if (lane == 0) cexp[b] = e;
}

// Source box of every row of every (tile, slot) of a launch, in the launch's order ([T][128], -1:
// none), and the slot with its level; vtab: rows of vstride source boxes per target box
__global__ void __launch_bounds__(128) k_tc_sources(const int4* tiles, const int32_t* pre, const int32_t* boxes,
                                                    const int32_t* vtab, int vstride, const int32_t* slots, int32_t* src,
                                                    int32_t* meta) {
    const int t = blockIdx.x, row = threadIdx.x;
    const int4 tile = tiles[t];
    const int p0 = pre[t], ns = pre[t + 1] - p0;
    const int64_t v = row < tile.z ? (int64_t)boxes[tile.y + row] * vstride : -1;
    for (int si = 0; si < ns; ++si) {
        const int slot = slots[(int64_t)t * kSlotStride + 1 + si];
        src[((int64_t)p0 + si) * TC_M + row] = v >= 0 ? vtab[v + slot] : -1;
        if (row == 0) meta[p0 + si] = slot | (tile.x << 16);
    }
}

// ------------------------------------------------------------------------------------
// the kernel
// ------------------------------------------------------------------------------------
// R = NB NT coefficients per box; each CTA computes the NT = 32 NC output rows
// n0 = blockIdx.y NT .. of its tiles (NB > 1 where R exceeds the MMA's N of 256).
template <int NC, int NS, int NB>
__global__ void __launch_bounds__(TC_THREADS, 1)
    k_m2l_tc(M2LTables tabs, const int4* __restrict__ tiles, const int32_t* __restrict__ first,
             const int32_t* __restrict__ pre, int T, const int32_t* __restrict__ all_boxes,
             const int4* __restrict__ src, const int32_t* __restrict__ meta, const __half* __restrict__ chl,
             const int* __restrict__ cexp, float* __restrict__ d, int accum, float* __restrict__ part, int* err) {
    constexpr int NT = 32 * NC;
    constexpr int R = NB * NT;
    constexpr int NK = R / TC_KC;
    constexpr int PW = TC_PW;
    const int n0 = blockIdx.y * NT;
    constexpr int A_BYTES = TC_M * 128, B_BYTES = NT * 128;
    constexpr int STAGE = A_BYTES + B_BYTES;
    // rings of NH hi x hi and NX cross-term accumulators of ACC columns in the 512 TMEM columns, so that
    // the MMAs of a slot wait for the drain of the slot NH (NX) back
    constexpr int ACC = NT;
    constexpr int NH = 8 * ACC <= 512 ? 4 : (4 * ACC <= 512 ? 2 : (3 * ACC <= 512 ? 2 : 1));
    constexpr int NX = 3 * ACC <= 512 && 4 * ACC > 512 ? 1 : NH;
    constexpr int USED = (NH + NX) * ACC;
    constexpr uint32_t NCOLS = USED <= 32 ? 32 : (USED <= 64 ? 64 : (USED <= 128 ? 128 : (USED <= 256 ? 256 : 512)));
    static_assert(USED <= 512, "tensor memory");
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ uint64_t full[NS], empty[NS], ready[NH], freed[NH], freedx[NX], rfull[TC_RING], rempty[TC_RING];
    __shared__ uint32_t tmem_base;
    __shared__ volatile int abort_flag;
    __shared__ int rmeta[TC_RING];   // offset slot and level
    unsigned char* base = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    int (*ridx)[TC_M] = reinterpret_cast<int(*)[TC_M]>(base + NS * STAGE);
    float (*rscale)[TC_M] = reinterpret_cast<float(*)[TC_M]>(base + NS * STAGE + TC_RING * TC_M * 4);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int cta = blockIdx.x, ncta = gridDim.x;
    const int g0 = tc_range(cta, T, ncta), g1 = tc_range(cta + 1, T, ncta);
    const int total = g1 - g0;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(NCOLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        abort_flag = 0;
        for (int s = 0; s < NS; ++s) {
            mbar_init(smem_u32(&full[s]), 32 * PW + 1);
            mbar_init(smem_u32(&empty[s]), 1);
        }
        for (int j = 0; j < NH; ++j) {
            mbar_init(smem_u32(&ready[j]), 1);
            mbar_init(smem_u32(&freed[j]), TC_EPI / 32);
        }
        for (int j = 0; j < NX; ++j) mbar_init(smem_u32(&freedx[j]), TC_EPI / 32);
        for (int r = 0; r < TC_RING; ++r) {
            mbar_init(smem_u32(&rfull[r]), 1);
            mbar_init(smem_u32(&rempty[r]), PW + TC_EPI / 32);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;

    if (warp >= 8 && warp < 8 + PW) {
        // ---------------- producers ----------------
        constexpr int RPT = TC_M / (4 * PW);   // rows a thread copies a 16-byte piece of: 4 (j PW + w) + lane / 8
        const int w = warp - 8, piece = 8 * (lane & 7);
        static_assert(4 * PW % 8 == 0, "rows of a thread share the swizzle phase");
        uint32_t s = 0, sp = 0;   // running stage and the parity of its current use
        bool ok = true, filled = false;
        // (every lane runs through every slot, those whose wait ran out without another wait or a copy: one that left
        // would keep the others in the __syncwarp for ever; a vote on leaving instead, here or in the index warp, took
        // 128^3 from 1154 to 1166 us)
        for (int n = 0; n < total; ++n) {
            const int r = n % TC_RING;
            ok = ok && mbar_wait(smem_u32(&rfull[r]), (uint32_t)((n / TC_RING) & 1), &abort_flag);
            // this thread's piece of each of its rows (row 0 with no bytes copied, so zeros, where the box has
            // no source); the rows of a thread are 4 PW apart, a multiple of the swizzle's 8
            const __half* from[RPT];
            uint32_t none = 0;
#pragma unroll
            for (int j = 0; j < RPT; ++j) {
                const int a = ridx[r][4 * (j * PW + w) + (lane >> 3)];
                from[j] = chl + (int64_t)(a >= 0 ? a : 0) * (2 * R) + piece;
                none |= a >= 0 ? 0u : 1u << j;
            }
            const int slot = rmeta[r] & 0xFFFF, lev = rmeta[r] >> 16;
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&rempty[r]));
            if (!ok) continue;
            const char* tb = reinterpret_cast<const char*>(tabs.t[lev]) + ((int64_t)slot * NK * R + n0) * 128;
#pragma unroll(NK <= 8 ? NK : 1)
            for (int kc = 0; kc < NK; ++kc) {
                if (filled && !mbar_wait(smem_u32(&empty[s]), sp ^ 1u, &abort_flag)) {
                    ok = false;
                    break;
                }
                const uint32_t st = smem_u32(base + s * STAGE), fb = smem_u32(&full[s]);
                if (w == 0 && lane == 0) {   // B: one pre-swizzled bulk copy of rows n0 .. n0 + NT - 1, 128 bytes each
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb), "r"(B_BYTES)
                                 : "memory");
                    asm volatile(
                        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                            st + A_BYTES),
                        "l"(tb + (int64_t)kc * R * 128), "r"(B_BYTES), "r"(fb)
                        : "memory");
                }
                // A: row = c[source of the row's box at this slot], columns 32 kc .. 32 kc + 31, hi and lo
                const uint32_t to = st + sw128_off_h(4 * w + (lane >> 3), piece);
#pragma unroll
                for (int j = 0; j < RPT; ++j)
                    cp_async16(to + j * (4 * PW * 128), from[j] + kc * (2 * TC_KC), (none >> j) & 1u ? 0u : 16u);
                asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(fb) : "memory");
                if (++s == NS) {
                    s = 0;
                    sp ^= 1u;
                    filled = true;
                }
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    } else if (warp == 8 + PW) {
        // ---------------- index warp: rows 4 lane .. 4 lane + 3 ----------------
        int4 a[TC_GRP], nx[TC_GRP];
        int m[TC_GRP], mx[TC_GRP];
        auto fetch = [&](int g) {
#pragma unroll
            for (int q = 0; q < TC_GRP; ++q) {
                nx[q] = g + q < g1 ? src[(int64_t)(g + q) * (TC_M / 4) + lane] : make_int4(-1, -1, -1, -1);
                mx[q] = g + q < g1 ? meta[g + q] : 0;
            }
        };
        fetch(g0);
        bool ok = true;
        for (int g = g0; g < g1; g += TC_GRP) {   // (every lane to the end, as the producers)
#pragma unroll
            for (int q = 0; q < TC_GRP; ++q) {
                a[q] = nx[q];
                m[q] = mx[q];
            }
            int4 e[TC_GRP];
#pragma unroll
            for (int q = 0; q < TC_GRP; ++q)
                e[q] = make_int4(a[q].x >= 0 ? cexp[a[q].x] : 0, a[q].y >= 0 ? cexp[a[q].y] : 0,
                                 a[q].z >= 0 ? cexp[a[q].z] : 0, a[q].w >= 0 ? cexp[a[q].w] : 0);
            fetch(g + TC_GRP);
#pragma unroll
            for (int q = 0; q < TC_GRP; ++q) {
                if (g + q >= g1) break;
                const int n = g - g0 + q, r = n % TC_RING;
                if (n >= TC_RING) ok = ok && mbar_wait(smem_u32(&rempty[r]), (uint32_t)((n / TC_RING - 1) & 1), &abort_flag);
                const int sT = tabs.sT[m[q] >> 16];
                reinterpret_cast<int4*>(ridx[r])[lane] = a[q];
                reinterpret_cast<float4*>(rscale[r])[lane] =
                    make_float4(a[q].x >= 0 ? pow2i(-(e[q].x + sT)) : 0.f, a[q].y >= 0 ? pow2i(-(e[q].y + sT)) : 0.f,
                                a[q].z >= 0 ? pow2i(-(e[q].z + sT)) : 0.f, a[q].w >= 0 ? pow2i(-(e[q].w + sT)) : 0.f);
                if (lane == 0) rmeta[r] = m[q];
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&rfull[r]));
            }
        }
    } else if (warp == 9 + PW) {
        // ---------------- MMA issuer ----------------
        if (lane == 0) {
            constexpr uint32_t idesc = f16_idesc(TC_M, NT);
            const uint32_t a0 = sw128_desc_lo(smem_u32(base));
            const uint32_t fullb = smem_u32(full), emptyb = smem_u32(empty), readyb = smem_u32(ready);
            const uint32_t freedb = smem_u32(freed), freedxb = smem_u32(freedx);
            // running stage and accumulator numbers, with the parity of their current use
            uint32_t s = 0, sp = 0, j = 0, jp = 0, jx = 0, jxp = 0;
            bool ok = true, full_next = false, acc_next = false;
            for (int si = 0; si < total && ok; ++si) {
                if (si >= NH && !acc_next && !mbar_wait(freedb + 8 * j, jp ^ 1u, &abort_flag)) break;
                if (si >= NX && !acc_next && !mbar_wait(freedxb + 8 * jx, jxp ^ 1u, &abort_flag)) break;
                const uint32_t dh = tmem + j * ACC, dx = tmem + (NH + jx) * ACC;
                const uint32_t rj = readyb + 8 * j;
                if (++j == NH) {
                    j = 0;
                    jp ^= 1u;
                }
                if (++jx == NX) {
                    jx = 0;
                    jxp ^= 1u;
                }
#pragma unroll 1
                for (int kc = 0; kc < NK; ++kc) {
                    if (!full_next && !mbar_wait(fullb + 8 * s, sp, &abort_flag)) {
                        ok = false;
                        break;
                    }
                    // A's copies are generic-proxy writes, read here by the async proxy
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t a = a0 + s * (STAGE >> 4), b = a + (A_BYTES >> 4), es = emptyb + 8 * s;
                    const uint32_t acc = kc > 0 ? 1u : 0u;
                    if (++s == NS) {
                        s = 0;
                        sp ^= 1u;
                    }
                    full_next = mbar_test(fullb + 8 * s, sp);
                    if (kc == NK - 1)
                        acc_next = (si + 1 >= NH) & mbar_test(freedb + 8 * j, jp ^ 1u) & mbar_test(freedxb + 8 * jx, jxp ^ 1u);
                    // (16 FP16 = 32 bytes along K inside the swizzle row, lo parts 64 bytes on; offsets >> 4)
                    mma_f16_lo<false>(dh, a, b, idesc, acc);
                    mma_f16_lo<false>(dx, a, b + 4, idesc, acc);
                    mma_f16_lo<true>(dx, a + 4, b, idesc, 1u);
                    mma_f16_lo<true>(dh, a + 2, b + 2, idesc, 1u);
                    mma_f16_lo<true>(dx, a + 2, b + 6, idesc, 1u);
                    mma_f16_lo<true>(dx, a + 6, b + 2, idesc, 1u);
                    mma_commit(es);
                }
                if (!ok) break;
                mma_commit(rj);
            }
        }
        __syncwarp();
    } else {
        // ---------------- epilogue: warps 0-7 ----------------
        const int q = warp & 3, half = warp >> 2;
        const uint32_t t_row = (uint32_t)(32 * q) << 16;
        const int col0 = half * (NT / 2);
        const int row = 32 * q + lane;
        constexpr int LDW = (NT / 2) % 32 == 0 && NC <= 4 ? 32 : 16;   // columns a tensor-memory load takes
        float acc[NT / 2];
        int n = 0, t = first[cta];
        bool ok = true;
        for (int g = g0; g < g1 && ok; ++t) {
            const int p0 = pre[t], p1 = pre[t + 1], e = min(p1, g1);
            if (e <= g) continue;   // (a tile without slots)
            const int4 tile = tiles[t];
            const int box = row < tile.z ? all_boxes[tile.y + row] : -1;
#pragma unroll
            for (int k = 0; k < NT / 2; ++k) acc[k] = 0.f;
            for (; g < e; ++g, ++n) {
                const int j = n % NH, jx = n % NX, r = n % TC_RING;
                ok = mbar_wait(smem_u32(&rfull[r]), (uint32_t)((n / TC_RING) & 1), &abort_flag);
                const float f = rscale[r][row];
                ok = ok && mbar_wait(smem_u32(&ready[j]), (uint32_t)((n / NH) & 1), &abort_flag);
                ok = __all_sync(0xffffffffu, ok);   // warp-uniform exit (tcgen05.ld is .sync.aligned)
                if (!ok) break;
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&rempty[r]));
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (int h = 0; h < 2; ++h) {   // the cross terms, then the hi x hi terms
                    const uint32_t ta = tmem + t_row + (uint32_t)((h ? j : NH + jx) * ACC + col0);
#pragma unroll
                    for (int cc = 0; cc < NT / 2; cc += LDW) {
                        uint32_t v[LDW];
                        if (LDW == 32) tmem_ld32(v, ta + cc);
                        else tmem_ld16(v, ta + cc);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                        for (int k = 0; k < LDW; ++k) acc[cc + k] = fmaf(__uint_as_float(v[k]), f, acc[cc + k]);
                    }
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(h ? &freed[j] : &freedx[jx]));
                }
            }
            if (!ok || box < 0) continue;
            const bool cut = p0 < g0 || p1 > g1;   // a piece of the tile: into the work space
            float4* o = cut ? reinterpret_cast<float4*>(part + ((int64_t)tc_piece(cta, p0, T, ncta) * TC_M + row) * R + n0 + col0)
                            : reinterpret_cast<float4*>(d + (int64_t)box * R + n0 + col0);
#pragma unroll
            for (int k = 0; k < NT / 8; ++k) {
                float4 v = make_float4(acc[4 * k], acc[4 * k + 1], acc[4 * k + 2], acc[4 * k + 3]);
                if (accum && !cut) {   // add to the row already there (L2L onto the M2L result)
                    const float4 u = o[k];
                    v = make_float4(u.x + v.x, u.y + v.y, u.z + v.z, u.w + v.w);
                }
                o[k] = v;
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (abort_flag) {
        if (tid == 0) atomicExch(err, 1);
        for (int k = 0; k < 32; ++k) __nanosleep(1000);   // (copies and MMAs that another role had just issued)
    }
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(NCOLS));
}

// The rows of every tile that k_m2l_tc cut between CTAs: its pieces added in slot order. Tiles
// without a slot get zeros (unless added onto d).
__global__ void __launch_bounds__(256) k_tc_finish(const int4* __restrict__ tiles, const int32_t* __restrict__ pre, int T,
                                                   int ncta, const int32_t* __restrict__ all_boxes,
                                                   const float* __restrict__ part, int R, float* __restrict__ d, int accum) {
    const int t = blockIdx.x, p0 = pre[t], p1 = pre[t + 1];
    const bool none = p0 == p1;
    if (none && accum) return;
    const int c0 = none ? 0 : tc_cta_of(p0, T, ncta), c1 = none ? -1 : tc_cta_of(p1 - 1, T, ncta);
    if (c0 == c1) return;
    const int4 tile = tiles[t];
    const int per = R / 4, e = blockIdx.y * blockDim.x + threadIdx.x;   // one float4 a thread
    const int row = e / per, col = e % per;
    if (row >= tile.z) return;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int c = c0; c <= c1; c += 8) {   // eight pieces' loads in flight
        float4 u[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            u[q] = c + q <= c1 ? reinterpret_cast<const float4*>(part + ((int64_t)tc_piece(c + q, p0, T, ncta) * TC_M + row) * R)[col]
                               : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) v = make_float4(v.x + u[q].x, v.y + u[q].y, v.z + u[q].z, v.w + u[q].w);
    }
    float4* o = reinterpret_cast<float4*>(d + (int64_t)all_boxes[tile.y + row] * R) + col;
    if (accum) {
        const float4 u = *o;
        v = make_float4(u.x + v.x, u.y + v.y, u.z + v.z, u.w + v.w);
    }
    *o = v;
}

// ------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------
static constexpr size_t kRingBytes = (size_t)TC_RING * TC_M * 8;

static constexpr int stages_for(int R) {
    const size_t stage = (size_t)TC_M * 128 + (size_t)R * 128;
    const size_t avail = 227 * 1024 - 1024 - 1024 - kRingBytes;
    int ns = (int)(avail / stage);
    return ns > 8 ? 8 : ns;
}

size_t m2l_tc_smem(int R) {
    const size_t stage = (size_t)TC_M * 128 + (size_t)R * 128;
    return 1024 + (size_t)stages_for(R) * stage + kRingBytes;
}

// row blocks per tile: the MMA's N is at most 256
static int row_blocks(int R) { return (R + 255) / 256; }

// coefficient counts with a compiled kernel: R <= 256 in one row block, and the Chebyshev
// counts 384, 512, 768, 1024 in blocks of 192 or 256 rows
int m2l_tc_supported(int R) {
    if (R % 32 != 0 || R < 32) return 0;
    if (R > 256 && R != 384 && R != 512 && R != 768 && R != 1024) return 0;
    const int nb = row_blocks(R);
    return (R % (32 * nb) == 0 && stages_for(R / nb) >= 2) ? 1 : 0;
}

int64_t m2l_tc_table_elems(int R, int nslots) { return (int64_t)nslots * R * R * 2; }

int m2l_tc_prepare(cudaStream_t st, const double* T, int R, void* out, int* sT_out, int nslots) {
    const int64_t n = (int64_t)nslots * R * R;
    DevBuf mx;
    KF_TRY(dev_alloc(mx, 8));
    KF_CUDA(cudaMemsetAsync(mx.p, 0, 8, st));
    k_absmax<<<1024, 256, 0, st>>>(T, n, ptr<unsigned long long>(mx));
    KF_LAUNCH();
    unsigned long long bits = 0;
    KF_CUDA(cudaMemcpyAsync(&bits, mx.p, 8, cudaMemcpyDeviceToHost, st));
    KF_CUDA(cudaStreamSynchronize(st));
    dev_free(mx);
    double m;
    std::memcpy(&m, &bits, 8);
    int ex = 0;
    if (m > 0.0) std::frexp(m, &ex);
    const int sT = m > 0.0 ? TC_HI_EXP + 1 - ex : 0;   // max |T| 2^sT in [2^13, 2^14)
    *sT_out = sT;
    k_swizzle_T<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(T, R, nslots, sT, reinterpret_cast<__half*>(out));
    KF_LAUNCH();
    return KIFMM_OK;
}

int m2l_tc_split(cudaStream_t st, const double* c, int64_t nb, int R, void* out, int* cexp) {
    return m2l_tc_split_pad(st, c, nb, R, R, out, cexp);
}

int m2l_tc_split_pad(cudaStream_t st, const double* c, int64_t nb, int R, int ldo, void* out, int* cexp) {
    if (nb <= 0) return KIFMM_OK;
    k_split_c<double><<<(unsigned)((nb * 32 + 255) / 256), 256, 0, st>>>(c, nb, R, reinterpret_cast<__half*>(out), cexp, ldo);
    KF_LAUNCH();
    return KIFMM_OK;
}

int m2l_tc_split_f32(cudaStream_t st, const float* c, int64_t nb, int R, void* out, int* cexp) {
    if (nb <= 0) return KIFMM_OK;
    k_split_c<float><<<(unsigned)((nb * 32 + 255) / 256), 256, 0, st>>>(c, nb, R, reinterpret_cast<__half*>(out), cexp, R);
    KF_LAUNCH();
    return KIFMM_OK;
}

int tc_sched_build(cudaStream_t st, const int4* tiles, const int32_t* boxes, const int32_t* vtab, int vstride,
                   const int32_t* slots, int ntiles, int R, int num_sms, TcSched& s) {
    s.ntiles = ntiles;
    s.total = s.ncta = 0;
    s.finish = false;
    if (ntiles <= 0) return KIFMM_OK;
    std::vector<int32_t> cnt(ntiles), pre(ntiles + 1, 0);
    KF_CUDA(cudaMemcpy2DAsync(cnt.data(), 4, slots, kSlotStride * 4, 4, ntiles, cudaMemcpyDeviceToHost, st));
    KF_CUDA(cudaStreamSynchronize(st));
    int64_t sum = 0;
    for (int k = 0; k < ntiles; ++k) {
        sum += cnt[k];
        if (sum >= (int64_t)1 << 31) {
            set_error("tensor-core translations: more than 2^31 tile slots");
            return KIFMM_ERR_ARG;
        }
        pre[k + 1] = (int32_t)sum;
    }
    const int T = s.total = (int)sum;
    s.ncta = tc_num_ctas(T, ntiles, num_sms / row_blocks(R));
    bool cut = false;
    std::vector<int32_t> first(s.ncta, 0);   // each CTA's first tile
    for (int k = 0; k < ntiles; ++k) {
        const bool none = pre[k] == pre[k + 1];
        for (int c = 0; !none && c < s.ncta; ++c)
            if (tc_range(c, T, s.ncta) >= pre[k] && tc_range(c, T, s.ncta) < pre[k + 1]) first[c] = k;
        s.finish = s.finish || none;
        if (!none && tc_cta_of(pre[k], T, s.ncta) != tc_cta_of(pre[k + 1] - 1, T, s.ncta)) cut = true;
    }
    s.finish = s.finish || cut;
    KF_TRY(dev_alloc(s.pre, pre.size() * 4));
    KF_CUDA(cudaMemcpyAsync(s.pre.p, pre.data(), pre.size() * 4, cudaMemcpyHostToDevice, st));
    KF_TRY(dev_alloc(s.first, first.size() * 4));
    KF_CUDA(cudaMemcpyAsync(s.first.p, first.data(), first.size() * 4, cudaMemcpyHostToDevice, st));
    if (cut) KF_TRY(dev_alloc(s.part, (size_t)2 * s.ncta * TC_M * R * 4));
    if (T > 0) {
        KF_TRY(dev_alloc(s.src, (size_t)T * TC_M * 4));
        KF_TRY(dev_alloc(s.meta, (size_t)T * 4));
        k_tc_sources<<<ntiles, 128, 0, st>>>(tiles, ptr<int32_t>(s.pre), boxes, vtab, vstride, slots,
                                             ptr<int32_t>(s.src), ptr<int32_t>(s.meta));
        KF_LAUNCH();
    }
    KF_CUDA(cudaStreamSynchronize(st));
    return KIFMM_OK;
}

// Launch arguments other than the tables and tiles: the split, the coefficient rows, the output and
// whether it is added to.
struct TcArgs {
    const TcSched& s;
    const void* chl;
    const int* cexp;
    float* d;
    int accum;
    int* err;
};

template <int NC, int NB>
static int launch_nc(cudaStream_t st, const M2LTables& tabs, const int4* tiles, const int32_t* boxes, const TcArgs& a) {
    constexpr int NS = stages_for(32 * NC);
    const size_t smem = m2l_tc_smem(32 * NC);
    static bool configured = false;   // one attribute per instantiation (its size never changes)
    if (!configured) {
        KF_CUDA(cudaFuncSetAttribute(k_m2l_tc<NC, NS, NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        configured = true;
    }
    if (a.s.total > 0) {
        k_m2l_tc<NC, NS, NB><<<dim3(a.s.ncta, NB), TC_THREADS, smem, st>>>(
            tabs, tiles, ptr<int32_t>(a.s.first), ptr<int32_t>(a.s.pre), a.s.total, boxes, ptr<int4>(a.s.src),
            ptr<int32_t>(a.s.meta), reinterpret_cast<const __half*>(a.chl), a.cexp, a.d, a.accum, ptr<float>(a.s.part),
            a.err);
        KF_LAUNCH();
    }
    if (a.s.finish) {
        k_tc_finish<<<dim3(a.s.ntiles, TC_M * 32 * NC * NB / 4 / 256), 256, 0, st>>>(tiles, ptr<int32_t>(a.s.pre), a.s.total, a.s.ncta, boxes,
                                                         ptr<float>(a.s.part), 32 * NC * NB, a.d, a.accum);
        KF_LAUNCH();
    }
    return KIFMM_OK;
}

int launch_tc_translate(cudaStream_t st, const M2LTables& tabs, int R, const TcSched& sched, const int4* tiles,
                        const int32_t* boxes, const void* chl, const int* cexp, float* d, int accum, int* err,
                        int64_t& nl) {
    if (sched.ntiles <= 0) return KIFMM_OK;
    nl += (sched.total > 0) + (sched.finish ? 1 : 0);
    const TcArgs a{sched, chl, cexp, d, accum, err};
#define KF_M2L_TC(NC, NB) return launch_nc<NC, NB>(st, tabs, tiles, boxes, a)
    switch (m2l_tc_supported(R) ? R : 0) {
        case 32: KF_M2L_TC(1, 1);
        case 64: KF_M2L_TC(2, 1);
        case 96: KF_M2L_TC(3, 1);
        case 128: KF_M2L_TC(4, 1);
        case 160: KF_M2L_TC(5, 1);
        case 192: KF_M2L_TC(6, 1);
        case 224: KF_M2L_TC(7, 1);
        case 256: KF_M2L_TC(8, 1);
        case 384: KF_M2L_TC(6, 2);    // Chebyshev p = 7
        case 512: KF_M2L_TC(8, 2);    // p = 8
        case 768: KF_M2L_TC(8, 3);    // p = 9
        case 1024: KF_M2L_TC(8, 4);   // p = 10
        default: set_error("M2L tensor path: unsupported coefficient count"); return KIFMM_ERR_ARG;
    }
#undef KF_M2L_TC
}

}  // namespace kifmm
