// Host-side declarations shared by the library's translation units.
#pragma once

#include <cstdint>
#include <tuple>
#include <vector>
#include <cuda_runtime.h>

namespace sgm {

// A chain of nodes in a graph under construction: the next kernel runs after
// the nodes in `after`.  Graphs are built node by node, not captured: they are
// built on the scheduler's thread and on those of the callers, and a capture
// there fails a cudaDeviceSynchronize that another thread happens to make.
struct NodeChain {
    cudaGraph_t graph;
    std::vector<cudaGraphNode_t> after;
    bool kernel = false;            // `after` is the one kernel before
    cudaError_t err = cudaSuccess;  // the first error of launch()
};

// A path's kernels follow one another in a stream, each launched with
// programmatic stream serialization (pdl): its launch work overlaps the kernel
// before it, and its first instruction waits until that one has ended and its
// writes are visible (pdl_wait, sgm_device.cuh).  In plain order, and at every
// graph launch, the device releases a kernel in steps of 2.05 us, 4.1 us at
// least; measured for five kernels of 1.5 us back to back: 20.5 us launched
// plainly, 14.3 us as a replayed graph, 11.3 us this way.
// With a chain, the kernels become nodes of its graph instead, one after the
// other, by programmatic edges where the launch would be a programmatic one.
struct Stream {
    cudaStream_t s;
    bool pdl;
    NodeChain* chain;
    Stream(cudaStream_t stream, bool p = false, NodeChain* c = nullptr) : s(stream), pdl(p), chain(c) {}
};

// Adds a kernel to a chain.
template <class... P, class... A>
inline cudaError_t add_kernel(NodeChain& c, void (*kernel)(P...), dim3 grid, dim3 block, A&&... args) {
    std::tuple<P...> v{static_cast<P>(args)...};
    cudaKernelNodeParams n{};
    n.func = reinterpret_cast<void*>(kernel);
    n.gridDim = grid;
    n.blockDim = block;
    void* ptrs[sizeof...(P)];
    std::apply([&](auto&... x) { int i = 0; ((ptrs[i++] = &x), ...); }, v);
    n.kernelParams = ptrs;  // the values are copied into the node
    cudaGraphNode_t node = nullptr;
    const cudaError_t e = cudaGraphAddKernelNode(&node, c.graph, c.after.data(), c.after.size(), &n);
    if (e == cudaSuccess) c.after.assign(1, node);
    return e;
}

// Launches a kernel, or adds it to the stream's chain; the caller reads the
// error with cudaGetLastError, or in the chain.
template <class... P, class... A>
inline void launch(void (*kernel)(P...), dim3 grid, dim3 block, Stream st, A&&... args) {
    if (st.chain) {
        NodeChain& c = *st.chain;
        if (c.err != cudaSuccess) return;
        const bool side = st.pdl && c.kernel;
        const std::vector<cudaGraphNode_t> before = c.after;
        if (side) c.after.clear();
        c.err = add_kernel(c, kernel, grid, block, args...);
        if (side && c.err == cudaSuccess) {
            cudaGraphEdgeData edge{};
            edge.type = cudaGraphDependencyTypeProgrammatic;
            edge.from_port = cudaGraphKernelNodePortProgrammatic;
            c.err = cudaGraphAddDependencies(c.graph, before.data(), c.after.data(), &edge, 1);
        }
        c.kernel = true;
        return;
    }
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = block;
    c.stream = st.s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    c.attrs = attr;
    c.numAttrs = st.pdl ? 1 : 0;
    cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}

// The sweeps keep every per-(pixel, disparity) cube of a pair in one array of
// per-pixel records [H][W][RB] bytes: the paired costs MC (D bytes, offset 0),
// the sums S (offset D: D paired bytes when s8, else D/2 packed u16x2 words),
// then one stored-L_r field (D paired bytes) per pair of opposite paths that
// needs its own.  One offset then addresses every field of a step's pixel.
inline int record_bytes(int D, bool s8, int n_lx) { return D + (s8 ? D : 2 * D) + n_lx * D; }

// Arguments of the aggregation sweeps (Eq. 3) over one pair.
struct SweepArgs {
    uint8_t* rec;       // per-pixel records [H][W][RB]
    uint8_t* raw;       // winner-take-all disparity [H][W] (final vertical sweep)
    uint16_t* Sdbg;     // optional natural-order S [H][W][D] (debug)
    int RB;             // record bytes (W * H * RB < 2^32)
    int lx_off;         // byte offset of this pair's stored-L_r field in a record
    int W, H, D;
    uint32_t P1x2, P2x2;  // penalties replicated in both u16 halves
    int rx;               // vertical-type sweeps: 0 (vertical), +1 / -1 (diagonals)
    int pair;             // 1: both opposite directions, 0: the forward one only
    int wta;              // vertical-type sweeps: 1 = finish with Eq. 4, 0 = add into S
    int phase;            // vertical-type pairs: 0 = both phases, 1 = first half of each path
                          // (saves the path state), 2 = second half (restores it)
    uint32_t* state;      // path states between phases 1 and 2 (sweep_state_words)
    uint32_t* state_end;  // the end of the state array (bounds-checked build)
    int s8;               // S kept as paired bytes instead of u16x2 words
    // Post-filter form of the sweeps (sgm_compute_ex): post = 1 selects it.
    // Every step q -> p then takes its jump penalty from a per-block table
    // indexed by |I(p) - I(q)| of the base image img (max(P1, P2 / (1 + g))
    // with ap2, else P2 throughout), and a winner-take-all sweep with
    // sub != nullptr also writes, per pixel, S(d-1) - S(d) | (S(d+1) - S(d)) << 16
    // at the winner d (each half 0 when that neighbour is outside [0, D)).
    int post;
    const uint8_t* img;   // base image [H][W] (post form)
    int ap2;              // adaptive P2: P2(g) = max(P1, P2 / (1 + g)); else P2
    uint32_t* sub;        // [H][W] (post form, winner-take-all sweeps; optional)
};

// Every sum S held between sweeps fits a byte: with 2 paths S = L_LR <= 31 + P2
// <= 255 always; with 4 paths S = L_LR + L_RL <= 2 * (31 + P2) before the
// vertical pair's winner-take-all (L_r - MC <= P2 from Eq. 3, MC <= 31).
// With the full Census MC <= 62 instead of 31 (mc_max).
inline bool sum_fits_u8(int n_paths, int P2, int mc_max = 31) {
    return (n_paths == 2 && mc_max + P2 <= 255) || (n_paths == 4 && 2 * (mc_max + P2) <= 255);
}

// ---------------------------------------------------------------------------
// Batched execution over device work lists.  A stage of a group of pairs (one
// D, path count, sum width and Census type) is one persistent grid: every
// block takes the next unit of the stage's list (a Census tile, a cost row
// segment, a block of sweep lines, a median tile) with an atomic counter
// until the list is exhausted.  The list lives in device memory: the pairs'
// descriptors in the list's order (longest chains first) and the prefix sums
// of their unit counts.  A kernel skips a descriptor whose D is not its own
// and sets bit 0 of the device status word.
// ---------------------------------------------------------------------------
template <class Job>
struct WorkList {
    const Job* job;         // [n] descriptors
    const uint32_t* start;  // [n + 1]: jobs [0, k) hold units [0, start[k])
    int n;
};

// Features are uint32 (CSCT) or uint64 (full Census) as the launch's ct62 says.
struct CensusJob {
    const uint8_t *left, *right;
    void *Fb, *Fm;
    int W, H;
};
struct CostJob {
    const void *Fb, *Fm;
    uint8_t* rec;  // MC is written at offset 0 of each RB-byte record
    int RB, W, H, D;
};
struct MedianJob {
    const uint8_t* raw;
    uint8_t* out;
    int W, H;
};

// One stage of a group over its work list.
struct ListLaunch {
    const void* list;  // device WorkList<Job> of the stage
    uint32_t* next;    // the list's unit counter, 0 before the launch
    uint32_t* status;  // device status word
    int grid;          // persistent blocks
    int D;
    bool ct62, pair, s8;
    int rx;            // vertical-type sweeps: 0 (vertical, finishing with Eq. 4), +1 / -1 (diagonals)
    int n_paths, cls;  // paired schedule: paths and class of the sums (pairs_class)
};

// Each launcher enqueues one kernel on `stream` and returns the launch error;
// the list launchers add it to a chain of nodes.
// ct62 = false: the CSCT of Eq. 1, uint32 features; true: the full 9x7
// Census, uint64 features.
cudaError_t launch_census(const uint8_t* left, const uint8_t* right, void* Fb, void* Fm, int W, int H, bool ct62,
                          Stream stream);
// MC goes to offset 0 of the RB-byte record of each pixel.
cudaError_t launch_cost(const void* Fb, const void* Fm, uint8_t* rec, int RB, int W, int H, int D, bool ct62,
                        Stream stream);
cudaError_t launch_sweep_h(const SweepArgs& a, Stream stream);
// The first sweep stage of a path with pairs (4 or 8 directions): the
// horizontal pair and the first halves (phase 1) of up to three vertical-type
// pairs in one launch; blocks [start[0], start[1]) run the horizontal pair,
// blocks [start[k + 1], start[k + 2]) the first halves of v[k].  `start` is
// filled in by the launcher.
struct FirstStageArgs {
    SweepArgs h;
    SweepArgs v[3];
    int nv;
    int start[5];
};
cudaError_t launch_sweep_first(FirstStageArgs& f, Stream stream);
// 4 paths: the horizontal first halves (saving their state in f.h.state) beside
// the whole vertical pair f.v[0], which writes S; then the horizontal second
// halves finish with Eq. 4 (launch_sweep_h2, a.state as in the first stage).
cudaError_t launch_sweep_first4(FirstStageArgs& f, Stream stream);
cudaError_t launch_sweep_h2(const SweepArgs& a, Stream stream);
cudaError_t launch_sweep_v(const SweepArgs& a, Stream stream);
// Words of saved path state per vertical-type pair between its two phases:
// per line, 32 lanes x (K + 3) words for each warp carrying it (one warp of
// 16-lane paths, K = D/32; or two warps of 32-lane paths, K = D/64).
inline size_t sweep_state_words(int W, int D) {
    return (D % 64 == 0) ? static_cast<size_t>(W) * 64 * (D / 64 + 3) : static_cast<size_t>(W) * 32 * (D / 32 + 3);
}
cudaError_t launch_median(const uint8_t* raw, uint8_t* disp, int W, int H, Stream stream);
// Post-filters (sgm_compute_ex).  Mirror: mr[y][x] = right[y][W-1-x],
// ml[y][x] = left[y][W-1-x].
cudaError_t launch_mirror(const uint8_t* left, const uint8_t* right, uint8_t* ml, uint8_t* mr, int W, int H,
                          Stream stream);
// out16 = 3x3 median of v, v = 16 d + the sub-pixel offset from sub (when
// sub != nullptr) with d = rawL; then, when rawRm != nullptr (the right
// pass's disparity in mirrored columns), 0xFFFF where the left-right check
// fails.  quads: the three inputs are in quads of 2 x 2 pixels, else row-major.
cudaError_t launch_post(const uint8_t* rawL, const uint32_t* sub, const uint8_t* rawRm, uint16_t* out16, bool quads,
                        int W, int H, int D, Stream stream);
// The work-list kernels: every job of a list has the launch's D (and, for
// sweeps, its pair / s8 settings; a vertical-type list runs both halves of
// its pair in one unit, the vertical one finishing with Eq. 4).
cudaError_t launch_census_list(const ListLaunch& l, NodeChain& chain);
cudaError_t launch_cost_list(const ListLaunch& l, NodeChain& chain);
cudaError_t launch_sweep_h_list(const ListLaunch& l, NodeChain& chain);
cudaError_t launch_sweep_v_list(const ListLaunch& l, NodeChain& chain);
cudaError_t launch_median_list(const ListLaunch& l, NodeChain& chain);
// Units of one pair in each list; blocks of each list kernel resident per SM.
int census_units(int W, int H);
int cost_units(int W, int H);
int sweep_units(int lines, int D, bool pair);
int median_units(int W, int H);
int median_quads_units(int W, int H);
constexpr int kCensusListPerSM = 16, kCostListPerSM = 8, kMedianListPerSM = 8, kSweepListMaxPerSM = 5;
// Debug: paired costs (offset 0 of RB-byte records) -> natural order [H][W][D].
cudaError_t launch_unpair_cost(const uint8_t* rec, int RB, uint8_t* out, int W, int H, int D, cudaStream_t stream);

// ---------------------------------------------------------------------------
// The paired-line schedule (sgm_pairs.cuh).  Every warp carries two adjacent
// lines of one direction, one per u16 half of each packed word.  The
// per-(pixel, disparity) cubes live in quads of 2 x 2 pixels over the grid
// padded to even sizes W2 x H2: quad (qx, qy) holds, per disparity d, the four
// bytes of pixels (2qx + i, 2qy + j) at byte i + 2j of a 32-bit word, so a
// quad takes QB = 4D bytes of a cube.  Each cube is its own array of
// [QH][QW] quads (FS bytes), at rec + f FS for field f:
//   0     MC      matching costs (Eq. 2); 0 at padding pixels
//   1, 2  vertical   r = L_r - MC of the top-to-bottom and bottom-to-top paths
//   3, 4  diagonal   r of the down-right and the up-left paths
//   5, 6  diagonal   r of the down-left and the up-right paths
// (2 paths: fields 0, 1; 4 paths: 0-2; 8 paths: all).  One 32-bit offset
// q QB then addresses quad q in every field.  The diagonal fields hold units
// of a line pair instead of quads: unit (j, p) at [j][p] holds, per disparity,
// line 2p at rows 2j and 2j + 1, then line 2p + 1 (sgm_pairs.cuh).
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int pairs_fields(int n_paths) { return n_paths == 2 ? 2 : (n_paths == 4 ? 3 : 7); }

// Quads of a segment: the horizontal walks store their state at every segment
// boundary and the finishing launch walks each segment again.  Sixteen columns
// keep the states at 1/16 of a stored field per direction; with more than 128
// disparities a warp's segment has to fit its shared memory.
__host__ __device__ constexpr int seg_quads(int D) { return D <= 128 ? 8 : 4; }
// Small frames walk shorter segments, a multiple of kShortSeg quads (pairs_geometry).
constexpr int kShortSeg = 2;

struct PairsArgs {
    uint8_t* rec;          // the field arrays (pairs_fields of FS bytes each)
    uint8_t* rawq;         // winner-take-all disparity in quads [QH][QW][4]
    uint16_t* Sdbg;        // optional natural-order S [H][W][D] (debug)
    uint32_t* state;       // horizontal states [2 (1 with 2 paths)][QH][NS][(D/32 + 1) / 2][32]
    // Post-filters: the jump penalty of every step, [8][QH][QW] words of the
    // four pixels of a quad or diagonal unit (direction: left to right, right to
    // left, then the order of the fields), or null (P2 throughout); S(d-1) - S(d)
    // | (S(d+1) - S(d)) << 16 at the winner in quads [QH][QW][4], or null.
    const uint32_t* p2map;
    uint32_t* subq;
    int W, H, W2, H2, QW, QH, D, n_paths;
    int CQ, NS;            // quads of a segment, segments of a row pair
    size_t FS;             // bytes of one field array (QH * QW * QB, rounded up)
    int QB;                // bytes of one quad in a field: 4D (W2 * H2 * D < 2^32)
    uint32_t P1x2, P2x2;
    int cls;               // class of the sums (pairs_class)
    int run;               // batched: segments of a unit of the finishing list
    int check_shrink;      // bounds-checked build, test hook: bytes taken off the declared end of the fields
};
// One launch over one or two problems of the same shape (the two passes of the
// left-right check).
struct PairsJobs {
    PairsArgs job[2];
    int n;
};
// Geometry of a W x H problem; `lists`: as the work lists walk it (segments of seg_quads).
PairsArgs pairs_geometry(int W, int H, int D, int n_paths, bool lists);
__host__ __device__ inline size_t pairs_state_words(const PairsArgs& a) {
    return static_cast<size_t>(a.n_paths == 2 ? 1 : 2) * a.QH * a.NS * 32 * ((a.D / 32 + 1) / 2);
}
// How the finishing launch sums and takes the winner.  4 and 8 paths: 0 = three
// r add in a byte (3 P2 <= 255) and the keys S D + d fit 16 bits, 1 = two r add
// in a byte, 2 = neither; 2 paths: 0 = 16-bit keys, 1 = 32-bit keys.
// S <= n_paths (MC_max + P2).
inline int pairs_class(int n_paths, int D, int p2_max, int mc_max) {
    const bool k16 = n_paths * (mc_max + p2_max) * D + D - 1 <= 65535;
    if (n_paths == 2) return k16 ? 0 : 1;
    return 3 * p2_max <= 255 && k16 ? 0 : (2 * p2_max <= 255 ? 1 : 2);
}
// A cube (or a field) that the 126 MB L2 does not hold beside what streams through it.
__host__ __device__ inline bool larger_than_l2(size_t bytes) { return bytes > (size_t(96) << 20); }
// Features of one or both passes: image z of F + z fstride bytes is left (0),
// right (1), and with n = 4 the mirrored pair of the right pass (right, left).
cudaError_t launch_census_passes(const uint8_t* left, const uint8_t* right, void* F, size_t fstride, int n, int W,
                                 int H, bool ct62, Stream stream);
// Quad-layout matching cost (Eq. 2): pass k from feature images 2k and 2k + 1
// into mc + k mcstride, quad q at + q QB.
cudaError_t launch_cost_quads(const void* F, size_t fstride, uint8_t* mc, size_t mcstride, int passes, int QB, int W,
                              int H, int D, bool ct62, Stream stream);
// Jump penalties max(P1, P2 / (1 + g)) of every step (PairsArgs::p2map), pass k
// into map + k stride words: base image left, and for the second pass the
// mirrored right image.
cudaError_t launch_p2map(const uint8_t* left, const uint8_t* right, uint32_t* map, size_t stride, int passes,
                         int n_paths, int W, int H, int P1, int P2, Stream stream);
// The walks of a path, side by side: horizontal, vertical and, with 8 paths,
// diagonal pairs; with 8 paths over a cube larger than L2, horizontal pair,
// directions that go down and directions that go up; or both directions of 2
// paths in one launch.  The first launch waits for the costs, each lets the
// next one start as soon as its own blocks have, and the last block of a later
// one waits for the one before it, so that the last launch ends when all have.
enum class Walks { kHor, kVer, kDiag, kDown, kUp, kHorVer };
inline bool walks_by_rows(const PairsArgs& a) { return a.n_paths == 8 && larger_than_l2(a.FS); }
cudaError_t launch_pairs_walks(const PairsJobs& f, Walks w, Stream stream);
cudaError_t launch_pairs_finish(const PairsJobs& f, Stream stream);
// Work-list forms.  Walks: kHorVer (2 and 4 paths), or kHor, kDown and kUp (8
// paths; kHor and kHorVer take pairs_hv_units, kDown and kUp QW units a pair).
struct CostQuadsJob {
    const void *Fb, *Fm;
    uint8_t* mc;
    int QB, W, H, D;
};
constexpr int kCostQuadsRun = 4; // 32-quad segments of a unit of the cost list
cudaError_t launch_cost_quads_list(const ListLaunch& l, NodeChain& chain);
cudaError_t launch_pairs_walks_list(const ListLaunch& l, Walks w, NodeChain& chain);
cudaError_t launch_pairs_finish_list(const ListLaunch& l, NodeChain& chain);
cudaError_t launch_median_quads_list(const ListLaunch& l, NodeChain& chain);
int cost_quads_units(int W, int H);
int pairs_hv_units(const PairsArgs& a, bool ver);
// Segments a warp takes at once: four, unless that leaves a pair with fewer
// units than the list's grid has warps.
inline int pairs_finish_run(const PairsArgs& a) { return a.QH * a.NS >= 16384 ? 4 : (a.QH * a.NS >= 8192 ? 2 : 1); }
inline int pairs_finish_units(const PairsArgs& a) { return a.QH * ((a.NS + a.run - 1) / a.run); }
constexpr int kFinishListPerSM = 14, kCostQuadsListPerSM = 12;
// 3x3 median of a quad-layout raw disparity.
cudaError_t launch_median_quads(const uint8_t* rawq, uint8_t* disp, int W, int H, Stream stream);
// Debug: a quad-layout cube (quad q at cube + q QB) -> natural order [H][W][D].
cudaError_t launch_unquad_cost(const uint8_t* cube, int QB, uint8_t* out, int W, int H, int D, cudaStream_t stream);

bool supported_D(int D);

// One-time kernel attributes; call before any launch or stream capture on the
// current device.
cudaError_t init_kernel_attributes();

}  // namespace sgm
