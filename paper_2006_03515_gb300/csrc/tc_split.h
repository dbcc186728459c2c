// The split of a tensor-core translation launch (m2l_tc.cu) over the SMs: T slots, tile after tile, over n
// CTAs, and the pieces of the tiles that it cuts. Host and device, without CUDA headers.
#pragma once
#include <algorithm>
#include <cstdint>

#ifdef __CUDACC__
#define KF_HD __host__ __device__ __forceinline__
#else
#define KF_HD inline
#endif

namespace kifmm {

// A tile is cut into pieces of at least this many slots: the start of a CTA (tensor memory, first
// copies) and the addition of a piece cost about three (32^3, 1250 slots: M2L and addition 76 us
// with pieces of 6 slots, 34 us with 12). Whole evaluations with pieces of 6, 12 and 24 slots: 16^3 93, 95 and
// 114 us, 24^3 148, 152 and 168, 32^3 165, 165 and 183, 40^3 247, 245 and 256, 64^3 306, 295 and 294, 80^3 512, 499 and 496.
constexpr int kTcMinSlots = 12;

// CTAs of a launch. No more than slots: tiles without a slot count among the ntiles, and a CTA with an
// empty range would write no piece of a cut tile that it lies in, while the addition reads one of every CTA
// from the tile's first to its last.
inline int tc_num_ctas(int T, int ntiles, int max_ctas) {
    return std::max(1, std::min({max_ctas, T, std::max(ntiles, T / kTcMinSlots)}));
}

// first slot of CTA c's range, and the CTA whose range holds slot g
KF_HD int tc_range(int c, int T, int n) { return (int)((int64_t)c * T / n); }
KF_HD int tc_cta_of(int g, int T, int n) { return (int)((((int64_t)g + 1) * n - 1) / T); }

// A CTA's range cuts at most two tiles: where its piece of a cut tile whose slots start at p0 lies in the
// work space
KF_HD int tc_piece(int c, int p0, int T, int n) { return 2 * c + (p0 < tc_range(c, T, n) ? 0 : 1); }

}  // namespace kifmm
