// Dispatch of the aggregation sweeps (Eq. 3, Eq. 4) by disparity count; the
// kernels themselves are in sgm_sweeps.cuh, instantiated per D in
// sgm_sweeps_d<D>.cu so that the translation units compile in parallel.
#include <algorithm>

#include "sgm_pairs.cuh"
#include "sgm_sweeps.cuh"

namespace sgm {

cudaError_t init_kernel_attributes() {
    cudaError_t e = sweep_set_attrs<32>();
    if (e == cudaSuccess) e = sweep_set_attrs<64>();
    if (e == cudaSuccess) e = sweep_set_attrs<96>();
    if (e == cudaSuccess) e = sweep_set_attrs<128>();
    if (e == cudaSuccess) e = sweep_set_attrs<160>();
    if (e == cudaSuccess) e = sweep_set_attrs<192>();
    if (e == cudaSuccess) e = sweep_set_attrs<224>();
    if (e == cudaSuccess) e = sweep_set_attrs<256>();
    return e;
}

#define SGM_DISPATCH_D(FN, D, arg, s)          \
    switch (D) {                               \
        case 32: return FN<32>(arg, s);        \
        case 64: return FN<64>(arg, s);        \
        case 96: return FN<96>(arg, s);        \
        case 128: return FN<128>(arg, s);      \
        case 160: return FN<160>(arg, s);      \
        case 192: return FN<192>(arg, s);      \
        case 224: return FN<224>(arg, s);      \
        case 256: return FN<256>(arg, s);      \
        default: return cudaErrorInvalidValue; \
    }

cudaError_t launch_sweep_h(const SweepArgs& a, Stream stream) { SGM_DISPATCH_D(sweep_launch_h, a.D, a, stream) }

cudaError_t launch_sweep_v(const SweepArgs& a, Stream stream) { SGM_DISPATCH_D(sweep_launch_v, a.D, a, stream) }

cudaError_t launch_sweep_first(FirstStageArgs& f, Stream stream) {
    SGM_DISPATCH_D(sweep_launch_first, f.h.D, f, stream)
}

cudaError_t launch_sweep_first4(FirstStageArgs& f, Stream stream) {
    SGM_DISPATCH_D(sweep_launch_first4, f.h.D, f, stream)
}

cudaError_t launch_sweep_h2(const SweepArgs& a, Stream stream) { SGM_DISPATCH_D(sweep_launch_h2, a.D, a, stream) }

cudaError_t launch_sweep_h_list(const ListLaunch& l, NodeChain& chain) {
    SGM_DISPATCH_D(sweep_launch_h_list, l.D, l, chain)
}

cudaError_t launch_sweep_v_list(const ListLaunch& l, NodeChain& chain) {
    SGM_DISPATCH_D(sweep_launch_v_list, l.D, l, chain)
}

int sweep_units(int lines, int D, bool pair) {
    // lines per block: a path takes G = 32 lanes (D % 64 == 0) or 16, a pair two paths
    const int G = (D % 64 == 0) ? 32 : 16, per_warp = 32 / G, per = kWarpsPerBlock * per_warp / (pair ? 2 : 1);
    return (lines + per - 1) / per;
}

// Quads of a segment.  The finishing launch walks a segment in both directions,
// one step after the other, and with few segments most of the chip is empty
// meanwhile: they are halved while they give at most two warps for each of the
// chip's 608 schedulers; beyond that the states cost more than the shorter
// walks gain.  us per frame, 4 paths, eight / four / two quads, by the warps of
// eight: 64x48 D=32 (96) 15.7 / 13.2 / 12.9, 64x128 D=96 (256) 20.2 / 17.1 / 16.2,
// 100x150 D=96 (525) 21.9 / 18.7 / 18.2, 160x120 D=64 (600) 20.3 / 18.8 / 18.8, 200x150
// D=128 (975) 24.6 / 22.9 / 23.0, 256x160 D=96 (1280) 27.1 / 26.9 / 27.4, 320x240
// D=64 (2400) 28.1 / 29.1 / 30.2; four / two quads, by the warps of four: 100x100
// D=192 (650) 21.1 / 18.4, 128x96 D=224 (768) 24.6 / 23.1, 200x100 D=160 (1250)
// 25.4 / 25.3, 240x200 D=160 (3000) 30.7 / 31.6.
static int segment_quads(const PairsArgs& a) {
    int quads = seg_quads(a.D);
    while (quads > kShortSeg && a.QH * ((a.QW + quads - 1) / quads) <= 2 * 608) quads /= 2;
    return quads;
}

PairsArgs pairs_geometry(int W, int H, int D, int n_paths, bool lists) {
    PairsArgs a{};
    a.W = W;
    a.H = H;
    a.D = D;
    a.n_paths = n_paths;
    a.W2 = W + (W & 1);
    a.H2 = H + (H & 1);
    a.QW = a.W2 / 2;
    a.QH = a.H2 / 2;
    a.CQ = lists ? seg_quads(D) : segment_quads(a);
    a.NS = (a.QW + a.CQ - 1) / a.CQ;
    return a;
}

#define SGM_DISPATCH_PAIRS(FN, D, ...)             \
    switch (D) {                                   \
        case 32: return FN<32>(__VA_ARGS__);       \
        case 64: return FN<64>(__VA_ARGS__);       \
        case 96: return FN<96>(__VA_ARGS__);       \
        case 128: return FN<128>(__VA_ARGS__);     \
        case 160: return FN<160>(__VA_ARGS__);     \
        case 192: return FN<192>(__VA_ARGS__);     \
        case 224: return FN<224>(__VA_ARGS__);     \
        case 256: return FN<256>(__VA_ARGS__);     \
        default: return cudaErrorInvalidValue;     \
    }

cudaError_t launch_pairs_walks(const PairsJobs& f, Walks w, Stream stream) {
    SGM_DISPATCH_PAIRS(pairs_walks, f.job[0].D, f, w, stream)
}

cudaError_t launch_pairs_finish(const PairsJobs& f, Stream stream) {
    SGM_DISPATCH_PAIRS(pairs_finish, f.job[0].D, f, stream)
}

cudaError_t launch_pairs_walks_list(const ListLaunch& l, Walks w, NodeChain& chain) {
    SGM_DISPATCH_PAIRS(pairs_walks_list, l.D, l, w, chain)
}

cudaError_t launch_pairs_finish_list(const ListLaunch& l, NodeChain& chain) {
    SGM_DISPATCH_PAIRS(pairs_finish_list, l.D, l, chain)
}

int pairs_hv_units(const PairsArgs& a, bool ver) {
    const int nd = a.n_paths == 2 ? 1 : 2;
    return ((a.NS > 1 ? a.QH * nd : 0) + (ver ? a.QW * nd : 0) + 1) / 2;
}

}  // namespace sgm
