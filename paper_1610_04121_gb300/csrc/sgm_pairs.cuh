// Path aggregation (Eq. 3), the sum S and the winner-take-all disparity
// (Eq. 4) of the SGM path of arXiv 1610.04121 with two lines per warp, for
// sm_103a; 2, 4 and 8 paths.
//
// Parallel scheme (Section 3.2's CTA-to-warp conversion, with the paper's
// byte-SIMD replaced by packed 16-bit lanes): a warp carries two adjacent
// lines of one direction, line A in the low u16 half of every packed word
// and line B in the high half.  Lane l holds the path costs of disparities
// d = K l + j, j < K = D / 32, of both lines, so word j of lane l is
// (L_A(d), L_B(d)).  The disparity neighbours d - 1 and d + 1 sit in the
// neighbouring words of the lane, or one lane over (two shuffles per step);
// the two per-line minima m(q) are two warp reductions.  No byte of a word
// ever crosses into the other line's half: every value stays below 2^14.
//
// Data layout (sgm_internal.h): the cost cube lives in quads of 2 x 2 pixels,
// so that a walk along rows or columns reads one quad (4 K bytes per lane)
// per two steps; a walk along diagonals reads two neighbouring quads per two
// steps.  Rows and columns are padded to even counts; the padding pixels have
// MC = 0, so a path that starts on one (a walk from the bottom or right edge
// of an odd-sized image) passes through it unchanged: from the reset state a
// zero-cost step leaves L = 0 and m = 0, which is the reset state again.
//
// Schedule:
//   walks     every direction of every line pair at once.  The vertical and
//             diagonal walkers store r = L_r - MC (0 <= r <= P2, a byte); the
//             horizontal walkers store nothing but their state at every
//             segment boundary (at most seg_quads(D) quads, pairs_geometry);
//   finish    a warp per segment of a row pair walks left to right and right
//             to left again from the stored states, adds the stored r of the
//             other directions and takes the winner.
// Walking a horizontal direction twice costs its integer work again (640x480
// D=128, 4 paths: the finishing launch is bound by issue, not by its 51 MB), and
// saves writing and reading back two bytes per pixel and disparity.
//
// Bounds: a step takes about 45 instructions per warp and 256 (pixel,
// disparity) pairs, 15-19 of them on the integer ALU, where each takes two
// cycles; two warps per scheduler (a 640x480 frame) are bound by that and by
// the chain of a step (two shuffles and two reductions), full schedulers by
// the ALU.  Measured, whole frame, against the per-line sweeps (one line per
// warp, sums in records): 1242x375 D=128 8 paths 390 -> 202 us, 1920x1080
// D=128 8 paths 1440 -> 935 us, 640x480 D=128 2 paths 84 -> 60 us, the same
// with 4 paths and all post-filters 257 -> 163 us; alone the horizontal walks of
// the 640x480 4-path frame take 30 us, the vertical ones 34 us, the finishing
// launch 27 us.
#pragma once

#include "sgm_device.cuh"
#include "sgm_internal.h"

namespace sgm {
namespace pairs {

constexpr uint32_t kInf2 = kInf16 * 0x10001u;
constexpr unsigned kFull = 0xffffffffu;

// Walk kinds of the first launch.
enum Kind { kHor = 0, kVer = 1, kDiag = 2 };

// Byte selectors: two bytes of a quad [x0y0, x1y0, x0y1, x1y1] as the u16x2 word
// of a step, columns of row j (vertical walks) or rows of column i (horizontal
// walks).  The zero bytes replicate the sign of a cost (MC <= 62).
constexpr uint32_t kSelRow0 = 0x9180u, kSelRow1 = 0xB3A2u, kSelCol0 = 0xA280u, kSelCol1 = 0xB391u;
// Diagonal walks take row 2j from quad a and row 2j + 1 from quads (a, a + 1)
// (lines moving right with increasing row) or (a, a - 1) (moving left).
constexpr uint32_t kSelNext = 0xE6B3u, kSelPrev = 0xA2F7u;

// ---------------------------------------------------------------------------
// Unit copies: a unit of a field (a quad, 4 D contiguous bytes) goes to
// shared memory with asynchronous 16-byte copies through L2 only, one group
// per unit.  Completion is counted per group, so a warp waits for exactly the
// unit it needs however many are in flight (register prefetch shares six
// scoreboards among all loads in flight and waits for later ones too).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

template <int N>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
    __syncwarp();
}

// L2 policy of data read for the last time: its lines go first, so that they do
// not push out what the other warps are about to read (the finishing launch of
// a 1242x375 8-path frame reads 7 bytes per pixel and disparity, most of it
// past what L2 holds: 216 -> 206 us for the frame).
__device__ __forceinline__ uint64_t last_read() {
    uint64_t pol;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

// Extents for the bounds-checked build.
__device__ __forceinline__ const uint8_t* cubes_end(const PairsArgs& a) {
    return a.rec + pairs_fields(a.n_paths) * a.FS - a.check_shrink;
}

// 64-bit base + 32-bit offset in one instruction.
__device__ __forceinline__ uint8_t* at(uint8_t* base, uint32_t off) {
    uint64_t r;
    asm("mad.wide.u32 %0, %1, 1, %2;" : "=l"(r) : "r"(off), "l"(reinterpret_cast<uint64_t>(base)));
    return reinterpret_cast<uint8_t*>(r);
}

// base: the lane's base (field + 16 lane); dst: shared address of the slot + 16 lane.
template <int D, bool LAST = false>
__device__ __forceinline__ void cp_unit(const PairsArgs& a, uint32_t dst, uint8_t* base, uint32_t off, unsigned site,
                                        uint64_t pol = 0) {
    constexpr int NC = D / 4;  // 16-byte pieces of a unit
    const int lane = threadIdx.x & 31;
    uint8_t* const g = at(base, off);
#pragma unroll
    for (int i = 0; i < (NC + 31) / 32; ++i)
        if (NC % 32 == 0 || lane + 32 * i < NC)
            if (SGM_GUARD(g + 512 * i, 16, a.rec, cubes_end(a), site))
            {
                if constexpr (LAST)
                    asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"(dst + 512 * i),
                                 "l"(g + 512 * i), "l"(pol)
                                 : "memory");
                else
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 512 * i), "l"(g + 512 * i)
                                 : "memory");
            }
}

// A lane's 4 K bytes of a unit in shared memory (address of the lane's bytes).
template <int K>
__device__ __forceinline__ void lds_unit(uint32_t s, uint32_t (&r)[K]) {
    if constexpr (K % 4 == 0) {
#pragma unroll
        for (int i = 0; i < K / 4; ++i)
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(r[4 * i]), "=r"(r[4 * i + 1]), "=r"(r[4 * i + 2]), "=r"(r[4 * i + 3])
                         : "r"(s + 16 * i));
    } else if constexpr (K % 2 == 0) {
#pragma unroll
        for (int i = 0; i < K / 2; ++i)
            asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(r[2 * i]), "=r"(r[2 * i + 1]) : "r"(s + 8 * i));
    } else {
#pragma unroll
        for (int i = 0; i < K; ++i) asm volatile("ld.shared.u32 %0, [%1];" : "=r"(r[i]) : "r"(s + 4 * i));
    }
}

template <int K>
__device__ __forceinline__ void sts_unit(uint32_t s, const uint32_t (&r)[K]) {
    if constexpr (K % 4 == 0) {
#pragma unroll
        for (int i = 0; i < K / 4; ++i)
            asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(s + 16 * i), "r"(r[4 * i]),
                         "r"(r[4 * i + 1]), "r"(r[4 * i + 2]), "r"(r[4 * i + 3])
                         : "memory");
    } else if constexpr (K % 2 == 0) {
#pragma unroll
        for (int i = 0; i < K / 2; ++i)
            asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(s + 8 * i), "r"(r[2 * i]), "r"(r[2 * i + 1])
                         : "memory");
    } else {
#pragma unroll
        for (int i = 0; i < K; ++i) asm volatile("st.shared.u32 [%0], %1;" ::"r"(s + 4 * i), "r"(r[i]) : "memory");
    }
}

// n contiguous bytes (a multiple of 16) from DRAM into L2.
__device__ __forceinline__ void prefetch_l2(const PairsArgs& a, const uint8_t* p, uint32_t n, unsigned site) {
    if (SGM_GUARD(p, n, a.rec, cubes_end(a), site))
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(n) : "memory");
}

// A lane's 4 K bytes of a unit from global memory, through L2 only.
template <int K>
__device__ __forceinline__ void ldg_unit(const PairsArgs& a, const uint8_t* p, uint32_t (&r)[K], uint64_t pol,
                                         unsigned site) {
    if (!SGM_GUARD(p, 4 * K, a.rec, cubes_end(a), site)) {
#pragma unroll
        for (int i = 0; i < K; ++i) r[i] = 0u;
    } else if constexpr (K % 4 == 0) {
#pragma unroll
        for (int i = 0; i < K / 4; ++i) {
            asm volatile("ld.global.cg.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
                         : "=r"(r[4 * i]), "=r"(r[4 * i + 1]), "=r"(r[4 * i + 2]), "=r"(r[4 * i + 3])
                         : "l"(p + 16 * i), "l"(pol));
        }
    } else if constexpr (K % 2 == 0) {
#pragma unroll
        for (int i = 0; i < K / 2; ++i) {
            asm volatile("ld.global.cg.L2::cache_hint.v2.u32 {%0, %1}, [%2], %3;"
                         : "=r"(r[2 * i]), "=r"(r[2 * i + 1])
                         : "l"(p + 8 * i), "l"(pol));
        }
    } else {
#pragma unroll
        for (int i = 0; i < K; ++i)
            asm volatile("ld.global.cg.L2::cache_hint.u32 %0, [%1], %2;" : "=r"(r[i]) : "l"(p + 4 * i), "l"(pol));
    }
}

// L2 policy of the stored r: of a cube larger than L2 they are gone before they
// are read, so their lines make way for the costs that the other walkers read
// (1920x1080 D=128 8 paths 974 -> 965 us); of a smaller one they stay.
__device__ __forceinline__ uint64_t store_policy(const PairsArgs& a) {
    uint64_t pol;
    if (larger_than_l2(a.FS))
        asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    else
        asm("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

// A lane's 4 K bytes of a unit to global memory.
template <int K>
__device__ __forceinline__ void stg_unit(const PairsArgs& a, uint8_t* p, const uint32_t (&r)[K], uint64_t pol,
                                         unsigned site) {
    if (!SGM_GUARD(p, 4 * K, a.rec, cubes_end(a), site)) return;
    if constexpr (K % 4 == 0) {
#pragma unroll
        for (int i = 0; i < K / 4; ++i)
            asm volatile("st.global.L2::cache_hint.v4.u32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(p + 16 * i),
                         "r"(r[4 * i]), "r"(r[4 * i + 1]), "r"(r[4 * i + 2]), "r"(r[4 * i + 3]), "l"(pol)
                         : "memory");
    } else if constexpr (K % 2 == 0) {
#pragma unroll
        for (int i = 0; i < K / 2; ++i)
            asm volatile("st.global.L2::cache_hint.v2.u32 [%0], {%1, %2}, %3;" ::"l"(p + 8 * i), "r"(r[2 * i]),
                         "r"(r[2 * i + 1]), "l"(pol)
                         : "memory");
    } else {
#pragma unroll
        for (int i = 0; i < K; ++i)
            asm volatile("st.global.L2::cache_hint.u32 [%0], %1, %2;" ::"l"(p + 4 * i), "r"(r[i]), "l"(pol) : "memory");
    }
}

__device__ __forceinline__ uint32_t mad(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t d;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}
// Byte permute with the sign-replicating selectors (__byte_perm masks them off).
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
}
// Minimum of three u16 pairs: one ALU instruction, as a minimum of two is.
__device__ __forceinline__ uint32_t vmin3(uint32_t a, uint32_t b, uint32_t c) { return __vimin3_u16x2(a, b, c); }

// ---------------------------------------------------------------------------
// Two chains (lines A and B) of Eq. 3 in one warp.  The first pixel of a path
// starts from the reset state (L = 0, m = 0), which gives L = MC.  A constant
// added to the w and m of a line changes no r (below): a chain that stores no
// r may leave the subtraction of m out and take it off now and then.
// ---------------------------------------------------------------------------
template <int K>
struct Chain2 {
    static constexpr int CW = (K + 1) / 2;  // words of a stored state: two bytes per word and lane
    uint32_t w[K];
    uint32_t up, dn;  // word K-1 of lane l-1 and word 0 of lane l+1, exchanged after every step
    uint32_t mpx2;    // (m_A, m_B)
    uint32_t mul_up, add_up, mul_dn, add_dn, k16;

    __device__ __forceinline__ void init(int lane) {
        // d = 0 has no d - 1 (lane 0) and d = D - 1 no d + 1 (lane 31): those
        // neighbours read "infinity" through a multiply-add on the FMA pipe
        // (opaque: a known 0 or 1 becomes a select on the ALU)
        mul_up = opaque(lane == 0 ? 0u : 1u);
        add_up = lane == 0 ? kInf2 : 0u;
        mul_dn = opaque(lane == 31 ? 0u : 1u);
        add_dn = lane == 31 ? kInf2 : 0u;
        k16 = opaque(0x10000u);
        reset();
    }

    __device__ __forceinline__ void reset() {
#pragma unroll
        for (int j = 0; j < K; ++j) w[j] = 0u;
        up = dn = 0u;
        mpx2 = 0u;
    }

    // Lines outside `keep` (a mask over the two halves) start a path at the next step.
    __device__ __forceinline__ void restart(uint32_t keep) {
#pragma unroll
        for (int j = 0; j < K; ++j) w[j] &= keep;
        up &= keep;
        dn &= keep;
        mpx2 &= keep;
    }

    // Neighbour words and per-line minima of the state in w.
    __device__ __forceinline__ void exchange() {
        up = __shfl_up_sync(kFull, w[K - 1], 1);
        dn = __shfl_down_sync(kFull, w[0], 1);
        uint32_t r = w[0];
        if constexpr (K == 2) {
            r = vmin2(w[0], w[1]);
        } else if constexpr (K > 2) {
            r = vmin3(w[0], w[1], w[2]);
#pragma unroll
            for (int j = 3; j + 1 < K; j += 2) r = vmin3(r, w[j], w[j + 1]);
            if constexpr (K % 2 == 0) r = vmin2(r, w[K - 1]);
        }
        // the 32-bit minimum orders by the high half first
        const uint32_t hi = __reduce_min_sync(kFull, r);
        const uint32_t lo = __reduce_min_sync(kFull, mad(r, k16, 0u));
        mpx2 = __byte_perm(lo, hi, 0x7632u);
    }

    // x(d) = min(L(q, d), L(q, d-1) + P1, L(q, d+1) + P1, m(q) + P2), the step's costs before MC and m(q)
    __device__ __forceinline__ void relax(uint32_t P1x2, uint32_t P2x2, uint32_t (&x)[K]) const {
        const uint32_t u = mad(up, mul_up, add_up);
        const uint32_t d = mad(dn, mul_dn, add_dn);
        const uint32_t mp2 = mpx2 + P2x2;
#pragma unroll
        for (int j = 0; j < K; ++j) {
            const uint32_t dm1 = j == 0 ? u : w[j - 1];
            const uint32_t dp1 = j == K - 1 ? d : w[j + 1];
            x[j] = vmin3(vmin2(dm1, dp1) + P1x2, w[j], mp2);
        }
    }

    // One step with r(p, d) = L(p, d) - MC(p, d), 0 <= r <= P2.
    __device__ __forceinline__ void step(const uint32_t (&mc)[K], uint32_t P1x2, uint32_t P2x2, uint32_t (&r)[K]) {
        uint32_t x[K];
        relax(P1x2, P2x2, x);
        // every candidate is >= m(q) in each half, so the packed subtraction never borrows
#pragma unroll
        for (int j = 0; j < K; ++j) r[j] = x[j] - mpx2;
#pragma unroll
        for (int j = 0; j < K; ++j) w[j] = r[j] + mc[j];
        exchange();
    }

    // One step that leaves m(q) in w and m; at most 16 between rebase() calls
    // (16 steps add at most 16 * 62, far below the infinity of the border lanes).
    __device__ __forceinline__ void step_raw(const uint32_t (&mc)[K], uint32_t P1x2, uint32_t P2x2) {
        uint32_t x[K];
        relax(P1x2, P2x2, x);
#pragma unroll
        for (int j = 0; j < K; ++j) w[j] = x[j] + mc[j];
        exchange();
    }

    __device__ __forceinline__ void rebase() {
#pragma unroll
        for (int j = 0; j < K; ++j) w[j] -= mpx2;
        up -= mpx2;
        dn -= mpx2;
        mpx2 = 0u;
    }

    // A stored state: every L_r fits a byte.  Word i of lane l at p[32 i + l].
    __device__ __forceinline__ void save(uint32_t* p) const {
#pragma unroll
        for (int i = 0; i < CW; ++i)
            p[32 * i] = __byte_perm(w[2 * i], 2 * i + 1 < K ? w[2 * i + 1 < K ? 2 * i + 1 : 0] : 0u, 0x6420u);
    }
    __device__ __forceinline__ void restore(const uint32_t (&c)[CW]) {
#pragma unroll
        for (int j = 0; j < K; ++j) w[j] = __byte_perm(c[j / 2], 0u, (j & 1) ? 0x4342u : 0x4140u);
        exchange();
    }
};

// A word of bytes [b0, b1, b2, b3] as (b0, b2) and (b1, b3): one permute on the
// ALU, one multiply-add on the FMA pipe (m256 = -256, opaque).
__device__ __forceinline__ void split(uint32_t q, uint32_t m256, uint32_t& even, uint32_t& odd) {
    odd = __byte_perm(q, 0u, 0x4341u);
    even = mad(odd, m256, q);
}

// Segment states of the horizontal walks: slot s of (direction, row pair) is
// the state in front of segment s in the direction's order.
template <int D>
__device__ __forceinline__ uint32_t* state_slot(const PairsArgs& a, int dir, int r, int s) {
    constexpr int CW = Chain2<D / 32>::CW;
    return a.state + ((static_cast<size_t>(dir) * a.QH + r) * a.NS + s) * (32 * CW) + (threadIdx.x & 31);
}
template <int D>
__device__ __forceinline__ bool state_ok(const PairsArgs& a, const uint32_t* p, unsigned site) {
    return SGM_GUARD(p, 4 * (32 * (Chain2<D / 32>::CW - 1) + 1), a.state,
                     a.state + pairs_state_words(a), site);
}

// The walks' ring of units in shared memory, per warp, at most 16 units.  D >
// 128: 16 KB, which also keeps the warps of an SM at twelve and their reads near
// one another (1920x1080 D=256 4 paths 893 us per frame; 12 KB 944, 8 KB 924,
// 24 KB 905); 8 KB for each of the three warps of a block that walks rows (8
// and 12 KB measure alike).  A walk's loop is UN units long: eight (640x480
// D=128 frame 79.5 us, four 81.8), four for D > 128 (1920x1080 D=256 892 us,
// eight 905), but two for diagonals that run beside the other walks (1242x375 8
// paths 204 us; eight no longer fit the instruction caches with them: 214), and
// no more than a segment or the ring holds.  SHORT (frames with shorter segments,
// pairs_geometry): a walk's last DEPTH units run outside the loop, one by one, so
// their rings hold eight units, four for D > 128, and their loops are four long
// (64x100 D=96 frame 14.9 us; rings of sixteen and loops of eight 16.7, eight and
// eight 15.2, four and four 15.5; 100x100 D=192 18.5, rings of eight 18.9).
template <int D>
__host__ __device__ constexpr int ring_bytes(bool rows = false) {
    return D <= 128 || rows ? 8192 : 16384;
}
template <int D, int KIND, bool ROWS, bool SHORT>
struct Ring {
    static constexpr int SB = (KIND == kDiag ? 2 : 1) * 4 * D;  // bytes of a slot
    static constexpr int WANT = KIND == kDiag && !ROWS ? 2 : (D <= 128 && !SHORT ? 8 : 4), FIT = ring_bytes<D>(ROWS) / SB;
    static constexpr int UN = WANT <= FIT && (KIND != kHor || WANT <= seg_quads(D)) ? WANT : (WANT < 4 ? WANT : 4);
    static constexpr int DEPTH = SHORT ? (D <= 128 ? 8 : 4) : (FIT / UN * UN > 16 ? 16 : FIT / UN * UN);
};

// ---------------------------------------------------------------------------
// One walk of the first launch: line pair `line` of a direction (fwd:
// increasing row or column).  Diagonals: kd = 0 moves right with increasing
// row, 1 left; line pair p starts at columns 2p, 2p + 1 of row 0 and wraps
// around at the padded width, each line starting a new path there
// (Section 3.2).  AP2: the jump penalty of every step comes from a.p2map.
// One body of code serves both directions (the byte selectors are registers):
// with a copy per direction the walks that run side by side no longer fit the
// instruction caches (164 against 144 us for the walks of a 1242x375 8-path
// frame, although each ran faster alone).
// ---------------------------------------------------------------------------
template <int D, int KIND, bool AP2, bool ROWS = false, bool SHORT = false>
__device__ __forceinline__ void walk(const PairsArgs& a, int line, int kd, bool fwd, uint32_t ring) {
    using R = Ring<D, KIND, ROWS, SHORT>;
    constexpr int K = D / 32, SB = R::SB, DEPTH = R::DEPTH, UN = R::UN;
    static_assert((KIND != kHor || (seg_quads(D) % UN == 0 && UN % kShortSeg == 0)) && DEPTH >= UN,
                  "segments end where groups of units end, short ones inside them too");
    const int CQ = SHORT ? a.CQ : seg_quads(D);
    const int lane = threadIdx.x & 31;
    const uint32_t QB = static_cast<uint32_t>(a.QB), rowb = static_cast<uint32_t>(a.QW) * QB;
    int nu;               // units of the walk
    uint32_t off, ustep;  // offset of the first unit and from unit to unit (in the output field for diagonals)
    if constexpr (KIND == kHor) {
        // the states in front of segments 1 .. NS - 1 (forward) and NS - 2 .. 0 (backward)
        nu = fwd ? (a.NS - 1) * CQ : max(a.QW - CQ, 0);
        off = static_cast<uint32_t>(line) * rowb + (fwd ? 0u : rowb - QB);
        ustep = fwd ? QB : 0u - QB;
    } else {
        nu = a.QH;
        off = static_cast<uint32_t>(line) * QB + (fwd ? 0u : (a.QH - 1) * rowb);
        ustep = fwd ? rowb : 0u - rowb;
    }
    if (nu <= 0) return;
    // the two steps' words of a unit, and the two steps' r as a unit (vertical
    // units are quads, diagonal ones [A0, A1, B0, B1])
    const uint32_t s_lo = KIND == kHor ? kSelCol0 : kSelRow0;
    const uint32_t s_hi = KIND == kHor ? kSelCol1 : (KIND == kVer ? kSelRow1 : (kd == 0 ? kSelNext : kSelPrev));
    const uint32_t sel0 = fwd ? s_lo : s_hi, sel1 = fwd ? s_hi : s_lo;
    const uint32_t selq = KIND == kVer ? (fwd ? 0x6420u : 0x2064u) : (fwd ? 0x6240u : 0x2604u);
    const uint64_t pol = store_policy(a);
    uint8_t* const src = a.rec + 16 * lane;
    uint8_t* const out =
        a.rec + (KIND == kVer ? 1 : 3 + 2 * kd) * a.FS + (fwd ? 0 : a.FS) + 4 * K * lane;  // stored r

    // Diagonals read quads qa and qb of every unit, both one column further in
    // every row, kd = 0: qb = qa + 1, kd = 1: qb = qa - 1.  Around the rows' end
    // one of them wraps a unit before the other: forward walks qb first, then
    // qa; backward walks qa, then qb.  ld_n / cp_n count the units up to the
    // first of the two for the unit being loaded / computed.
    uint32_t off_a = off, off_b = 0, lstep = ustep, wrap = 0, keep1 = 0;
    int ld_n = 0, cp_n = 0;
    if constexpr (KIND == kDiag) {
        const int j0 = fwd ? 0 : a.QH - 1, jm = j0 % a.QW;
        const bool right = (kd == 0) == fwd;  // the walk moves right
        int qa = kd == 0 ? line + jm : line - jm;
        qa = qa >= a.QW ? qa - a.QW : (qa < 0 ? qa + a.QW : qa);
        off_a = static_cast<uint32_t>(j0) * rowb + static_cast<uint32_t>(qa) * QB;
        lstep = ustep + (right ? QB : 0u - QB);
        wrap = right ? 0u - rowb : rowb;
        if (fwd) {
            ld_n = right ? a.QW - 1 - qa : qa;
            off_b = off_a + (right ? QB : 0u - QB);  // past the row's end where n = 0: wraps in that unit
        } else {
            ld_n = right ? (a.QW - qa) % a.QW : (qa + 1) % a.QW;
            const int qb = kd == 0 ? (qa + 1 == a.QW ? 0 : qa + 1) : (qa == 0 ? a.QW - 1 : qa - 1);
            off_b = off_a + static_cast<uint32_t>(qb - qa) * QB;
            if (ld_n == 0) off_a -= wrap;  // the first unit adds it
        }
        if (a.QW == 1) {  // one quad per row: never past its end
            off_a = off_b = static_cast<uint32_t>(j0) * rowb;
            lstep = ustep;
            wrap = 0u;
        }
        cp_n = ld_n;
        // the line that goes on at the first wrap: forward, in the unit's second
        // step (kd = 0: line A, 1: line B); backward, in its first step (kd = 0:
        // line B, 1: line A); the other line's path starts one step later
        keep1 = right ? 0x0000ffffu : 0xffff0000u;
    }
    const uint32_t sdst = ring + 16 * lane, ssrc = ring + 4 * K * lane;
    auto issue = [&](int slot, bool near) {
        if constexpr (KIND == kDiag) {
            if (near) {  // forward: qb wraps at n = 0, qa one unit later; backward: qa, then qb
                if (ld_n == 0) (fwd ? off_b : off_a) += wrap;
                if (ld_n < 0) {
                    (fwd ? off_a : off_b) += wrap;
                    ld_n = a.QW - 1;
                }
            }
            cp_unit<D>(a, sdst + slot, src, off_a, 101);
            cp_unit<D>(a, sdst + slot + 4 * D, src, off_b, 102);
            off_b += lstep;
            --ld_n;
        } else {
            cp_unit<D>(a, sdst + slot, src, off_a, 103);
        }
        off_a += lstep;
    };
    // a unit's costs from its slot
    constexpr int KB = KIND == kDiag ? K : 1;
    struct Cost {
        uint32_t a[K], b[KB];
    };
    auto read = [&](int slot, Cost& c) {
        lds_unit<K>(ssrc + slot, c.a);
        if constexpr (KIND == kDiag) lds_unit<K>(ssrc + slot + 4 * D, c.b);
    };
    auto words = [&](const Cost& c, uint32_t sel, uint32_t (&m)[K]) {
#pragma unroll
        for (int j = 0; j < K; ++j) m[j] = prmt(c.a[j], KIND == kDiag ? c.b[j < KB ? j : 0] : 0u, sel);
    };
    // jump penalties (AP2): lane l holds the word of unit 32 b + l, one batch ahead
    uint32_t p2c = 0, p2n = 0;
    const size_t units = static_cast<size_t>(a.QW) * a.QH;
    int p2i = 0, p2s = 0;
    const uint32_t* p2m = nullptr;
    auto p2_load = [&](int k) -> uint32_t {
        const int i = p2i + min(k, nu - 1) * p2s;
        return SGM_GUARD_INDEX(i, static_cast<long long>(units), 104) ? __ldcg(p2m + i) : 0u;  // see Side
    };
    if constexpr (AP2) {
        const int m = (KIND == kHor ? 0 : (KIND == kVer ? 2 : 4 + 2 * kd)) + (fwd ? 0 : 1);
        p2m = a.p2map + m * units;
        p2i = KIND == kHor ? line * a.QW + (fwd ? 0 : a.QW - 1) : line + (fwd ? 0 : (a.QH - 1) * a.QW);
        p2s = (KIND == kHor ? 1 : a.QW) * (fwd ? 1 : -1);
        p2n = p2_load(lane);
    }
    // selectors of the penalties (up to 255) in the order of the steps
    const uint32_t p_lo = KIND == kVer ? 0x4140u : 0x4240u, p_hi = KIND == kVer ? 0x4342u : 0x4341u;
    const uint32_t psel0 = fwd ? p_lo : p_hi, psel1 = fwd ? p_hi : p_lo;

    Chain2<K> ch;
    ch.init(lane);
    // one unit; `near`: a diagonal's lines may start a path in it
    auto unit = [&](const Cost& cur, int k, bool near) {
        uint32_t pa = a.P2x2, pb = a.P2x2;
        if constexpr (AP2) {
            if ((k & 31) == 0) {
                p2c = p2n;
                p2n = p2_load(k + 32 + lane);
            }
            const uint32_t p = __shfl_sync(kFull, p2c, k & 31);
            pa = __byte_perm(p, 0u, psel0);
            pb = __byte_perm(p, 0u, psel1);
        }
        uint32_t m[K];
        words(cur, sel0, m);
        if constexpr (KIND == kHor) {
            ch.step_raw(m, a.P1x2, pa);
            words(cur, sel1, m);
            ch.step_raw(m, a.P1x2, pb);
        } else {
            uint32_t r0[K], r1[K];
            if (KIND == kDiag && near) {
                if (a.QW == 1 || (fwd ? cp_n < 0 : cp_n == 0)) ch.restart(fwd ? ~keep1 : keep1);
            }
            ch.step(m, a.P1x2, pa, r0);
            if (KIND == kDiag && near) {
                if (a.QW == 1 || cp_n == 0) ch.restart(fwd ? keep1 : ~keep1);
                if (cp_n < 0) cp_n = a.QW - 1;
            }
            words(cur, sel1, m);
            ch.step(m, a.P1x2, pb, r1);
#pragma unroll
            for (int j = 0; j < K; ++j) r0[j] = prmt(r0[j], r1[j], selq);
            stg_unit<K>(a, at(out, off), r0, pol, 106);
            off += ustep;
            if constexpr (KIND == kDiag) --cp_n;
        }
    };
    // horizontal: the state where a segment ends, seg_n units further on
    int seg_n = 0;
    uint32_t* seg_st = nullptr;
    if constexpr (KIND == kHor) {
        seg_n = fwd ? CQ : (a.QW - 1) % CQ + 1;
        seg_st = state_slot<D>(a, fwd ? 0 : 1, line, fwd ? 1 : (a.QW - 1) / CQ - 1);
    }
    auto segment_end = [&](int n) {
        seg_n -= n;
        if (seg_n == 0) {
            seg_n = CQ;
            ch.rebase();
            if (state_ok<D>(a, seg_st, 105)) ch.save(seg_st);
            seg_st += (fwd ? 32 : -32) * Chain2<K>::CW;
        }
    };

    // backward row walks start inside a group of UN columns: the first slot
    // is chosen so that groups of slots and of columns end together
    const int s0 = KIND == kHor && !fwd ? (UN - a.QW % UN) % UN : 0;
    int slot = s0 * SB;
#pragma unroll 1
    for (int i = 0; i < DEPTH; ++i) {
        const int si = s0 + i < DEPTH ? s0 + i : s0 + i - DEPTH;
        if (i < nu) issue(si * SB, true);
        cp_commit();
    }
    Cost cur, nxt;
    cp_wait<DEPTH - 1>();
    read(slot, cur);
    // every unit: the next unit's costs into registers, its slot refilled, then its two steps
#pragma unroll 1
    for (int k = 0; k < nu;) {
        // groups of UN units that need no care: refills in range, no path starts
        int groups = 0;
        if (slot % (UN * SB) == 0) {
            int n = nu - DEPTH - k;
            if constexpr (KIND == kDiag) n = min(n, min(ld_n, cp_n));
            groups = n / UN;
        }
#pragma unroll 1
        for (; groups > 0; --groups) {
#pragma unroll
            for (int i = 0; i < UN; ++i) {
                const int s = slot + i * SB;
                cp_wait<DEPTH - 2>();
                read(i + 1 < UN ? s + SB : (s + SB == DEPTH * SB ? 0 : s + SB), nxt);
                issue(s, false);
                cp_commit();
                unit(cur, k + i, false);
                cur = nxt;
                if constexpr (KIND == kHor && SHORT)
                    if ((i + 1) % kShortSeg == 0) segment_end(kShortSeg);
            }
            k += UN;
            slot += UN * SB;
            if (slot == DEPTH * SB) slot = 0;
            if constexpr (KIND == kHor && !SHORT) segment_end(UN);
        }
        if (k < nu) {
            const int ns = slot + SB == DEPTH * SB ? 0 : slot + SB;
            cp_wait<DEPTH - 2>();
            read(ns, nxt);
            if (k + DEPTH < nu) issue(slot, true);
            cp_commit();
            unit(cur, k, true);
            cur = nxt;
            if constexpr (KIND == kHor) segment_end(1);
            ++k;
            slot = ns;
        }
    }
}

// The order of the walks' launches (launch_pairs_walks): the first one waits for
// the costs; a later one starts when every block of the one before has come
// past that wait and does without one of its own (which would wait for the end
// of the walks before, too), but its last block waits for the end of the one
// before, so that its own end means both.  PTX promises the writes of earlier
// kernels to a kernel that waits.  What a later walk reads without a wait, the
// costs and the penalties, was complete and visible to the whole device when the
// first walk's wait ended, before that walk let this one start; the assumption is
// that a kernel started after that moment sees it through L2.  So these reads
// take L2 only, never a line that an L1 may have kept from an earlier frame.
struct Side {
    int later, trigger;  // not the first launch; another one follows
    __device__ __forceinline__ void begin() const {
        if (!later) pdl_wait();
        if (trigger) pdl_trigger();
    }
    __device__ __forceinline__ void end() const {
        if (later && blockIdx.x == gridDim.x - 1 && blockIdx.y == gridDim.y - 1) pdl_wait();
    }
};

// The walks: one chain per warp.  Chains [0, nh) are horizontal line pairs
// (row pair c / nd, direction c % nd), [nh, nh + nv) vertical ones, nd
// directions each (1 with 2 paths).
template <int D, bool AP2, bool SHORT>
__global__ void __launch_bounds__(64) walk_hv_kernel(const __grid_constant__ PairsJobs f, int nh, int nv, Side side) {
    __shared__ __align__(16) uint8_t ring[2][ring_bytes<D>()];
    side.begin();
    const int warp = threadIdx.x >> 5;
    const PairsArgs& a = f.job[blockIdx.y];
    const uint32_t r = static_cast<uint32_t>(__cvta_generic_to_shared(ring[warp]));
    const int nd = a.n_paths == 2 ? 1 : 2, c = blockIdx.x * 2 + warp, v = c - nh;
    if (c < nh)
        walk<D, kHor, AP2, false, SHORT>(a, c / nd, 0, c % nd == 0, r);
    else if (v < nv)
        walk<D, kVer, AP2, false, SHORT>(a, v / nd, 0, v % nd == 0, r);
    side.end();
}

// Diagonal line pairs (8 paths): chain c is line pair c / 4, line set (c / 2) % 2, direction c % 2.
template <int D, bool AP2>
__global__ void __launch_bounds__(64) walk_d_kernel(const __grid_constant__ PairsJobs f, Side side) {
    __shared__ __align__(16) uint8_t ring[2][ring_bytes<D>()];
    side.begin();
    const int warp = threadIdx.x >> 5;
    const PairsArgs& a = f.job[blockIdx.y];
    const uint32_t r = static_cast<uint32_t>(__cvta_generic_to_shared(ring[warp]));
    const int c = blockIdx.x * 2 + warp;
    if (c < 4 * a.QW) walk<D, kDiag, AP2>(a, c / 4, (c / 2) % 2, c % 2 == 0, r);
    side.end();
}

// 8 paths, cubes larger than L2: the three directions that go down (fwd) or up
// from one column pair, a warp each.  They pass every row together, so that
// its costs come from DRAM once for the three.  Cubes that L2 holds walk the
// vertical pair beside the diagonals instead (fewer code paths per block and
// shorter blocks): 1920x1080 D=128 974 against 1008 us per frame, but 1242x375
// D=128 (60 MB of costs) 216 against 208.
template <int D, bool AP2>
__global__ void __launch_bounds__(96) walk_rows_kernel(const __grid_constant__ PairsJobs f, bool fwd, Side side) {
    __shared__ __align__(16) uint8_t ring[3][ring_bytes<D>(true)];
    side.begin();
    const int warp = threadIdx.x >> 5;
    const PairsArgs& a = f.job[blockIdx.y];
    const uint32_t r = static_cast<uint32_t>(__cvta_generic_to_shared(ring[warp]));
    if (warp == 0)
        walk<D, kVer, AP2, true>(a, blockIdx.x, 0, fwd, r);
    else
        walk<D, kDiag, AP2, true>(a, blockIdx.x, warp - 1, fwd, r);
    side.end();
}

// ---------------------------------------------------------------------------
// Finish: one segment (CQ quads) of a row pair per warp.  The segment's costs
// come into shared memory; left to right from the stored state, each step's r
// is kept there too; then right to left, adding everything and taking the
// winner (2 paths have no second walk: the first one finishes).  The stored r
// of the other directions come a quad ahead straight into registers, so that
// their reads are spread over the walk and shared memory allows 28 warps per
// SM (all of them loaded up front let every warp of a wave wait, then compute,
// in step: 31 us for a 640x480 D=128 frame).  S = own r + n MC + the r of the
// other n - 1 directions.  GS r may be added in a byte: GS P2 <= 255.  K16:
// S D + d fits 16 bits, so that one packed minimum serves both lines.  SHORT:
// segments of a.CQ quads, fewer than seg_quads(D).
// ---------------------------------------------------------------------------
template <int D, int NP>
struct Finish {
    static constexpr int UB = 4 * D, CQ = seg_quads(D);
    static constexpr int NV = NP == 2 ? 1 : 2, NF = NV + (NP == 8 ? 4 : 0);  // stored r of a quad
    static constexpr int KEPT = CQ * UB, BYTES = KEPT + (NP == 2 ? 0 : CQ * UB);
};

template <int D, int NP, int GS, bool K16, bool POST, bool SHORT>
__device__ __forceinline__ void finish(const PairsArgs& a, int r, int s, uint32_t smem) {
    using F = Finish<D, NP>;
    constexpr int K = D / 32, UB = F::UB, CQ = F::CQ, NV = F::NV, NF = F::NF;
    constexpr bool DIAG = NP == 8;
    const int lane = threadIdx.x & 31;
    const int q0 = s * (SHORT ? a.CQ : CQ), nq = min(SHORT ? a.CQ : CQ, a.QW - q0);
    const uint32_t QB = static_cast<uint32_t>(a.QB), rowoff = static_cast<uint32_t>(r) * a.QW * QB;
    const uint32_t off0 = rowoff + static_cast<uint32_t>(q0) * QB;
    const uint32_t ssrc = smem + 4 * K * lane;
    const uint32_t m256 = opaque(0xffffff00u), k256 = opaque(256u), k16 = opaque(0x10000u);
    const uint64_t pol = last_read();
#pragma unroll
    for (int i = 0; i < CQ; ++i)
        if (i < nq) cp_unit<D, true>(a, smem + 16 * lane + i * UB, a.rec + 16 * lane, off0 + i * UB, 111, pol);
    cp_commit();

    // the states in front of this segment, and its jump penalties
    Chain2<K> ch;
    ch.init(lane);
    constexpr int CW = Chain2<K>::CW;
    uint32_t cl[CW], cr[CW];
#pragma unroll
    for (int i = 0; i < CW; ++i) cl[i] = cr[i] = 0u;
    if (s > 0) {
        const uint32_t* st = state_slot<D>(a, 0, r, s);
        if (state_ok<D>(a, st, 114))
#pragma unroll
            for (int i = 0; i < CW; ++i) cl[i] = __ldcg(st + 32 * i);
    }
    if (NP > 2 && s + 1 < a.NS) {
        const uint32_t* st = state_slot<D>(a, 1, r, s);
        if (state_ok<D>(a, st, 115))
#pragma unroll
            for (int i = 0; i < CW; ++i) cr[i] = __ldcg(st + 32 * i);
    }
    uint32_t p2l = 0, p2r = 0;
    if constexpr (POST) {
        if (a.p2map) {
            const size_t i = static_cast<size_t>(r) * a.QW + q0 + min(lane, nq - 1);
            const size_t units = static_cast<size_t>(a.QW) * a.QH;
            if (SGM_GUARD_INDEX(static_cast<long long>(i), static_cast<long long>(units), 119)) {
                p2l = __ldg(a.p2map + i);
                if (NP > 2) p2r = __ldg(a.p2map + units + i);
            }
        }
    }
    auto p2_at = [&](uint32_t words, int i, uint32_t sel) -> uint32_t {
        if constexpr (POST) {
            const uint32_t p = __shfl_sync(kFull, words, i);
            return a.p2map ? __byte_perm(p, 0u, sel) : a.P2x2;
        } else {
            return a.P2x2;
        }
    };

    // stored r, in the order of the finishing walk.  Diagonal units are shared
    // by the two quads of a row that a line pair crosses: fv holds the one a
    // quad shares with its left neighbour, `carry` the one it shares with the
    // right, so each is read once, starting one quad past the segment.
    uint32_t fv[NF][K];
    uint8_t* const base = a.rec + 4 * K * lane;
    int up = 0, um = 0;  // next units of the right- and left-moving lines
    if constexpr (DIAG) {
        const int rm = r % a.QW;
        up = q0 + nq - 1 - rm;
        up = up < 0 ? up + a.QW : up;
        um = q0 + nq + rm;
        um = um >= a.QW ? um - a.QW : um;
        um = um >= a.QW ? um - a.QW : um;
    }
    auto load_v = [&](int i) {
#pragma unroll
        for (int v = 0; v < NV; ++v) ldg_unit<K>(a, at(base + (1 + v) * a.FS, off0 + i * QB), fv[v], pol, 112);
    };
    auto load_d = [&]() {
        if constexpr (DIAG) {
#pragma unroll
            for (int v = 0; v < 4; ++v)
                ldg_unit<K>(a, at(base + (3 + v) * a.FS, rowoff + static_cast<uint32_t>(v < 2 ? up : um) * QB),
                            fv[NF - 4 + v], pol, 113);
            up = up == 0 ? a.QW - 1 : up - 1;
            um = um == 0 ? a.QW - 1 : um - 1;
        }
    };
    // 4 paths: the whole segment's stored r on its way into L2 (lane v: field v),
    // which a quad ahead in registers leaves short of bytes in flight: 1920x1080
    // D=256 336 -> 260 us, 640x480 frame 84.2 -> 82.7.  With 8 paths the six
    // fields would push one another out (1242x375: 208 -> 221), with 2 paths L2
    // holds the one field already.
    if (NP == 4 && lane < NV) prefetch_l2(a, a.rec + (1 + lane) * a.FS + off0, nq * UB, 118);
    load_v(NP == 2 ? 0 : nq - 1);
    load_d();

    ch.restore(cl);
    cp_wait<0>();
    if constexpr (NP > 2) {
#pragma unroll 1
        for (int i = 0; i < nq; ++i) {
            uint32_t mc[K], lo[K], hi[K], r0[K], r1[K];
            lds_unit<K>(ssrc + i * UB, mc);
#pragma unroll
            for (int j = 0; j < K; ++j) split(mc[j], m256, lo[j], hi[j]);
            ch.step(lo, a.P1x2, p2_at(p2l, i, 0x4240u), r0);
            ch.step(hi, a.P1x2, p2_at(p2l, i, 0x4341u), r1);
#pragma unroll
            for (int j = 0; j < K; ++j) r0[j] = mad(r1[j], k256, r0[j]);
            sts_unit<K>(ssrc + F::KEPT + i * UB, r0);
        }
        ch.restore(cr);
    }

    // groups of r that add in bytes: the kept and the vertical ones, then each line set's
    constexpr int NB = NP == 2 ? 1 : (GS == 3 ? 1 : (GS == 2 ? 2 : 3)), NC = GS >= 2 ? 1 : 2;
    constexpr int NG = NB + (DIAG ? 2 * NC : 0);
    uint32_t carry[2][NC][K];
    auto diag_sums = [&](uint32_t (&u)[2][NC][K]) {
#pragma unroll
        for (int l = 0; l < 2; ++l)
#pragma unroll
            for (int j = 0; j < K; ++j) {
                const uint32_t x = fv[NF - 4 + 2 * l][j], y = fv[NF - 3 + 2 * l][j];
                if constexpr (GS >= 2) {
                    u[l][0][j] = x + y;
                } else {
                    u[l][0][j] = x;
                    u[l][NC - 1][j] = y;
                }
            }
    };
    if constexpr (DIAG) {
        diag_sums(carry);
        load_d();
    }
    uint32_t rawv = 0;
#pragma unroll 1
    for (int n = 0; n < nq; ++n) {
        const int i = NP == 2 ? n : nq - 1 - n;
        uint32_t mc[K], g[NG][K], mlo[K], mhi[K];
        lds_unit<K>(ssrc + i * UB, mc);
        if constexpr (NP == 2) {
#pragma unroll
            for (int j = 0; j < K; ++j) g[0][j] = fv[0][j];
        } else {
            uint32_t kept[K];
            lds_unit<K>(ssrc + F::KEPT + i * UB, kept);
#pragma unroll
            for (int j = 0; j < K; ++j) {
                if constexpr (GS == 3) {
                    g[0][j] = fv[0][j] + fv[1][j] + kept[j];
                } else if constexpr (GS == 2) {
                    g[0][j] = fv[0][j] + fv[1][j];
                    g[1][j] = kept[j];
                } else {
                    g[0][j] = fv[0][j];
                    g[1][j] = fv[1][j];
                    g[2][j] = kept[j];
                }
            }
        }
        if constexpr (DIAG) {
            uint32_t u[2][NC][K];
            diag_sums(u);
#pragma unroll
            for (int c = 0; c < NC; ++c)
#pragma unroll
                for (int j = 0; j < K; ++j) {
                    // units hold [A0, A1, B0, B1]; a quad [A0, B0, row 1 of the two lines crossing it]
                    g[NB + c][j] = __byte_perm(carry[0][c][j], u[0][c][j], 0x1720u);
                    g[NB + NC + c][j] = __byte_perm(u[1][c][j], carry[1][c][j], 0x5320u);
                    carry[0][c][j] = u[0][c][j];
                    carry[1][c][j] = u[1][c][j];
                }
        }
        if (n + 1 < nq) {
            load_v(NP == 2 ? i + 1 : i - 1);
            load_d();
        }
#pragma unroll
        for (int j = 0; j < K; ++j) split(mc[j], m256, mlo[j], mhi[j]);
        // sums of the other directions' r, both columns
        uint32_t slo[K], shi[K];
#pragma unroll
        for (int j = 0; j < K; ++j) {
            split(g[0][j], m256, slo[j], shi[j]);
#pragma unroll
            for (int q = 1; q < NG; ++q) {
                uint32_t e, o;
                split(g[q][j], m256, e, o);
                slo[j] += e;
                shi[j] += o;
            }
        }
        uint32_t word = 0;
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const int h = NP == 2 ? t : 1 - t;  // column of the quad
            uint32_t S[K];
            ch.step(h ? mhi : mlo, a.P1x2, p2_at(NP == 2 ? p2l : p2r, i, h ? 0x4341u : 0x4240u), S);
#pragma unroll
            for (int j = 0; j < K; ++j) S[j] = mad(h ? mhi[j] : mlo[j], NP, S[j]) + (h ? shi[j] : slo[j]);
            // the smallest S, then the lowest d, of both lines
            uint32_t dd, kA = 0xffffffffu, kB = 0xffffffffu;
            if constexpr (K16) {
                uint32_t key[K];
#pragma unroll
                for (int j = 0; j < K; ++j)
                    key[j] = mad(S[j], D, static_cast<uint32_t>(K * lane + j) * 0x10001u);
                uint32_t best = key[0];
#pragma unroll
                for (int j = 1; j + 1 < K; j += 2) best = vmin3(best, key[j], key[j + 1]);
                if constexpr (K % 2 == 0) best = vmin2(best, key[K - 1]);
                kB = __reduce_min_sync(kFull, best);
                kA = __reduce_min_sync(kFull, mad(best, k16, 0u));
                dd = __byte_perm(kA, kB, 0x7632u);
                if constexpr ((D & (D - 1)) == 0)
                    dd &= static_cast<uint32_t>(D - 1) * 0x10001u;
                else
                    dd = ((dd & 0xffffu) % static_cast<uint32_t>(D)) | (((dd >> 16) % static_cast<uint32_t>(D)) << 16);
            } else {  // 32-bit keys S << 16 | d
#pragma unroll
                for (int j = 0; j < K; ++j) {
                    const uint32_t d = static_cast<uint32_t>(K * lane + j);
                    kA = min(kA, mad(S[j], k16, d));
                    kB = min(kB, (S[j] & 0xffff0000u) | d);
                }
                kA = __reduce_min_sync(kFull, kA);
                kB = __reduce_min_sync(kFull, kB);
                dd = prmt(kA, kB, 0x5410u) & 0x00ff00ffu;
            }
            word |= dd << (8 * h);
            if (POST && a.Sdbg) {  // debug: natural-order S
                const int x = 2 * (q0 + i) + h, y = 2 * r;
                auto put = [&](size_t p, uint32_t v) {
                    if (SGM_GUARD_INDEX(static_cast<long long>(p), static_cast<long long>(a.W) * a.H * D, 120))
                        a.Sdbg[p] = static_cast<uint16_t>(v);
                };
                if (x < a.W) {
#pragma unroll
                    for (int j = 0; j < K; ++j) {
                        const size_t p = (static_cast<size_t>(y) * a.W + x) * D + static_cast<size_t>(K * lane + j);
                        put(p, S[j] & 0xffffu);
                        if (y + 1 < a.H) put(p + static_cast<size_t>(a.W) * D, S[j] >> 16);
                    }
                }
            }
            if constexpr (POST) {
                if (a.subq) {
                    // S(d-1) - S(d) | (S(d+1) - S(d)) << 16 at each line's winner: S by
                    // disparity in shared memory, lane 2 h takes S(d-1) of line h,
                    // lane 2 h + 1 S(d+1)
                    const uint32_t sums = smem + F::BYTES;
                    __syncwarp();
                    sts_unit<K>(sums + 4 * K * lane, S);
                    __syncwarp();
                    const uint32_t key = lane & 2 ? kB : kA;
                    const int d = static_cast<int>(key & 0xffu), e = lane & 1 ? d + 1 : d - 1;
                    uint32_t v = 0;
                    if (lane < 4 && e >= 0 && e < D) {
                        uint32_t w;
                        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(w) : "r"(sums + 4 * e));
                        v = (lane & 2 ? w >> 16 : w & 0xffffu) - (key >> 16);
                    }
                    v |= __shfl_down_sync(kFull, v, 1) << 16;
                    const size_t q = 4 * (static_cast<size_t>(r) * a.QW + q0 + i) + h + (lane & 2);
                    if ((lane == 0 || lane == 2) &&
                        SGM_GUARD_INDEX(static_cast<long long>(q), 4ll * a.QW * a.QH, 117))
                        a.subq[q] = v;
                }
            }
        }
        rawv = lane == i ? word : rawv;
    }
    const size_t q = static_cast<size_t>(r) * a.QW + q0 + lane;
    if (lane < nq && SGM_GUARD_INDEX(static_cast<long long>(q), static_cast<long long>(a.QW) * a.QH, 116))
        reinterpret_cast<uint32_t*>(a.rawq)[q] = rawv;
}

template <int D, int NP, int GS, bool K16, bool POST, bool SHORT>
__global__ void __launch_bounds__(64) finish_kernel(const __grid_constant__ PairsJobs f) {
    __shared__ __align__(16) uint8_t smem[2][Finish<D, NP>::BYTES + (POST ? 4 * D : 0)];  // post form: S of a column
    pdl_wait();
    const int warp = threadIdx.x >> 5;
    const PairsArgs& a = f.job[blockIdx.z];
    const int r = blockIdx.y * 2 + warp;  // two row pairs
    if (r < a.QH)
        finish<D, NP, GS, K16, POST, SHORT>(a, r, blockIdx.x,
                                            static_cast<uint32_t>(__cvta_generic_to_shared(smem[warp])));
}

// ---------------------------------------------------------------------------
// Work-list forms (batched pairs, sgm_internal.h): a persistent grid takes
// blocks of chains or, warp by warp, runs of segments.
// ---------------------------------------------------------------------------
template <int D>
__global__ void __launch_bounds__(64) walk_hv_list_kernel(const WorkList<PairsArgs>* __restrict__ Lp,
                                                          uint32_t* __restrict__ next, uint32_t* __restrict__ status,
                                                          bool ver) {
    __shared__ __align__(16) uint8_t ring[2][ring_bytes<D>()];
    const WorkList<PairsArgs> L = *Lp;
    const int warp = threadIdx.x >> 5;
    const uint32_t r = static_cast<uint32_t>(__cvta_generic_to_shared(ring[warp]));
    int p, u;
    while (take_unit(L, next, p, u)) {
        const PairsArgs a = L.job[p];
        if (a.D != D) {
            report_bad_job(status);
            continue;
        }
        const int nd = a.n_paths == 2 ? 1 : 2, nh = a.NS > 1 ? a.QH * nd : 0, c = u * 2 + warp, v = c - nh;
        if (c < nh)
            walk<D, kHor, false>(a, c / nd, 0, c % nd == 0, r);
        else if (ver && v < a.QW * nd)
            walk<D, kVer, false>(a, v / nd, 0, v % nd == 0, r);
    }
}

template <int D>
__global__ void __launch_bounds__(96) walk_rows_list_kernel(const WorkList<PairsArgs>* __restrict__ Lp,
                                                            uint32_t* __restrict__ next,
                                                            uint32_t* __restrict__ status, bool fwd) {
    __shared__ __align__(16) uint8_t ring[3][ring_bytes<D>(true)];
    const WorkList<PairsArgs> L = *Lp;
    const int warp = threadIdx.x >> 5;
    const uint32_t r = static_cast<uint32_t>(__cvta_generic_to_shared(ring[warp]));
    int p, u;
    while (take_unit(L, next, p, u)) {
        const PairsArgs a = L.job[p];
        if (a.D != D) {
            report_bad_job(status);
            continue;
        }
        if (warp == 0)
            walk<D, kVer, false, true>(a, u, 0, fwd, r);
        else
            walk<D, kDiag, false, true>(a, u, warp - 1, fwd, r);
    }
}

// Blocks per SM of the finishing list: its descriptors take registers where the
// single pair's sit in constant memory, so the count is forced.
template <int D, int NP>
constexpr int finish_list_blocks() {
    return D <= 128 ? (NP == 8 ? 10 : 14) : (NP == 8 ? 7 : 9);
}
template <int D, int NP, int GS, bool K16>
__global__ void __launch_bounds__(64, finish_list_blocks<D, NP>()) finish_list_kernel(const WorkList<PairsArgs>* __restrict__ Lp,
                                                         uint32_t* __restrict__ next, uint32_t* __restrict__ status) {
    __shared__ __align__(16) uint8_t smem[2][Finish<D, NP>::BYTES];
    const WorkList<PairsArgs> L = *Lp;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (L.n <= 0) return;
    const uint32_t end = L.start[L.n];
    // the next run is taken while this one is on its way
    uint32_t i = lane == 0 ? atomicAdd(next, 1u) : 0u;
    i = __shfl_sync(kFull, i, 0);
    int p = 0;
    while (i < end) {
        const uint32_t nx = lane == 0 ? atomicAdd(next, 1u) : 0u;
        while (L.start[p + 1] <= i) ++p;  // runs come in order
        const PairsArgs a = L.job[p];
        if (a.D != D || a.n_paths != NP) {
            report_bad_job(status);
        } else {
            const int u = static_cast<int>(i - L.start[p]), runs = (a.NS + a.run - 1) / a.run;
            const int r = u / runs, s0 = (u - r * runs) * a.run;
#pragma unroll 1
            for (int s = s0; s < min(s0 + a.run, a.NS); ++s)
                finish<D, NP, GS, K16, false, false>(a, r, s, static_cast<uint32_t>(__cvta_generic_to_shared(smem[warp])));
        }
        i = __shfl_sync(kFull, nx, 0);
    }
}

template <int D>
struct PairsD {
    static cudaError_t walks(const PairsJobs& f, Walks w, Stream s) {
        const PairsArgs& a = f.job[0];
        const int nd = a.n_paths == 2 ? 1 : 2;
        const bool rows = w == Walks::kDown || w == Walks::kUp;
        const Side side{w != Walks::kHor && w != Walks::kHorVer,
                        w == Walks::kHor || (a.n_paths == 8 && (w == Walks::kVer || w == Walks::kDown))};
        if (side.later) s.pdl = true;
        if (rows) {
            launch(a.p2map ? walk_rows_kernel<D, true> : walk_rows_kernel<D, false>, dim3(a.QW, f.n), 96, s, f,
                   w == Walks::kDown, side);
        } else if (w == Walks::kDiag) {
            launch(a.p2map ? walk_d_kernel<D, true> : walk_d_kernel<D, false>, dim3(2 * a.QW, f.n), 64, s, f, side);
        } else {
            const int nh = w != Walks::kVer && a.NS > 1 ? a.QH * nd : 0, nv = w != Walks::kHor ? a.QW * nd : 0;
            const dim3 grid(nh + nv > 0 ? (nh + nv + 1) / 2 : 1, f.n);  // images of one segment have no horizontal states
            const auto kernel = a.CQ != seg_quads(D)
                                    ? (a.p2map ? walk_hv_kernel<D, true, true> : walk_hv_kernel<D, false, true>)
                                    : (a.p2map ? walk_hv_kernel<D, true, false> : walk_hv_kernel<D, false, false>);
            launch(kernel, grid, 64, s, f, nh, nv, side);
        }
        return cudaGetLastError();
    }
    template <int NP, int GS, bool K16>
    static void finish_t(const PairsJobs& f, Stream s) {
        const PairsArgs& a = f.job[0];
        const dim3 grid(a.NS, (a.QH + 1) / 2, f.n);
        const bool post = a.p2map || a.subq || a.Sdbg;  // the post form serves the debug sums too
        if (a.CQ == seg_quads(D))
            launch(post ? finish_kernel<D, NP, GS, false, true, false> : finish_kernel<D, NP, GS, K16, false, false>, grid,
                   64, s, f);
        else
            launch(post ? finish_kernel<D, NP, GS, false, true, true> : finish_kernel<D, NP, GS, K16, false, true>, grid,
                   64, s, f);
    }
    template <int NP>
    static void finish_np(const PairsJobs& f, Stream s) {
        const int cls = f.job[0].cls;
        if constexpr (NP == 2) {
            if (cls == 0)
                finish_t<2, 1, true>(f, s);
            else
                finish_t<2, 1, false>(f, s);
        } else if (cls == 0) {
            finish_t<NP, 3, true>(f, s);
        } else if (cls == 1) {
            finish_t<NP, 2, false>(f, s);
        } else {
            finish_t<NP, 1, false>(f, s);
        }
    }
    static cudaError_t fin(const PairsJobs& f, Stream s) {
        switch (f.job[0].n_paths) {
            case 2: finish_np<2>(f, s); break;
            case 4: finish_np<4>(f, s); break;
            default: finish_np<8>(f, s);
        }
        return cudaGetLastError();
    }
    static cudaError_t walks_list(const ListLaunch& l, Walks w, NodeChain& chain) {
        const auto* L = static_cast<const WorkList<PairsArgs>*>(l.list);
        if (w == Walks::kDown || w == Walks::kUp)
            return add_kernel(chain, walk_rows_list_kernel<D>, l.grid, 96, L, l.next, l.status, w == Walks::kDown);
        return add_kernel(chain, walk_hv_list_kernel<D>, l.grid, 64, L, l.next, l.status, w == Walks::kHorVer);
    }
    template <int NP, int GS, bool K16>
    static cudaError_t finish_list_t(const ListLaunch& l, NodeChain& chain) {
        return add_kernel(chain, finish_list_kernel<D, NP, GS, K16>, l.grid, 64,
                          static_cast<const WorkList<PairsArgs>*>(l.list), l.next, l.status);
    }
    template <int NP>
    static cudaError_t finish_list_np(const ListLaunch& l, NodeChain& chain) {
        if (l.cls == 0) return finish_list_t<NP, 3, true>(l, chain);
        return l.cls == 1 ? finish_list_t<NP, 2, false>(l, chain) : finish_list_t<NP, 1, false>(l, chain);
    }
    static cudaError_t fin_list(const ListLaunch& l, NodeChain& chain) {
        if (l.n_paths == 8) return finish_list_np<8>(l, chain);
        if (l.n_paths == 4) return finish_list_np<4>(l, chain);
        return l.cls == 0 ? finish_list_t<2, 1, true>(l, chain) : finish_list_t<2, 1, false>(l, chain);
    }
};

}  // namespace pairs

// defined in sgm_sweeps_d<D>.cu; internal to the library (not part of the C ABI)
#define SGM_INTERNAL_P __attribute__((visibility("hidden")))
template <int D>
SGM_INTERNAL_P cudaError_t pairs_walks(const PairsJobs& f, Walks w, Stream s);
template <int D>
SGM_INTERNAL_P cudaError_t pairs_finish(const PairsJobs& f, Stream s);
template <int D>
SGM_INTERNAL_P cudaError_t pairs_walks_list(const ListLaunch& l, Walks w, NodeChain& chain);
template <int D>
SGM_INTERNAL_P cudaError_t pairs_finish_list(const ListLaunch& l, NodeChain& chain);

#define SGM_INSTANTIATE_PAIRS(D)                                                                   \
    template <>                                                                                    \
    SGM_INTERNAL_P cudaError_t pairs_walks<D>(const PairsJobs& f, Walks w, Stream s) {             \
        return pairs::PairsD<D>::walks(f, w, s);                                                   \
    }                                                                                              \
    template <>                                                                                    \
    SGM_INTERNAL_P cudaError_t pairs_finish<D>(const PairsJobs& f, Stream s) {                     \
        return pairs::PairsD<D>::fin(f, s);                                                        \
    }                                                                                              \
    template <>                                                                                    \
    SGM_INTERNAL_P cudaError_t pairs_walks_list<D>(const ListLaunch& l, Walks w, NodeChain& chain) { \
        return pairs::PairsD<D>::walks_list(l, w, chain);                                          \
    }                                                                                              \
    template <>                                                                                    \
    SGM_INTERNAL_P cudaError_t pairs_finish_list<D>(const ListLaunch& l, NodeChain& chain) {         \
        return pairs::PairsD<D>::fin_list(l, chain);                                               \
    }

}  // namespace sgm
