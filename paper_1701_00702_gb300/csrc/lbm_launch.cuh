// Kernel launchers shared by the per-mode translation units.  Each unit
// includes this file and instantiates the launchers for its storage modes.
#pragma once

#include "lbm_kernels.cuh"

namespace lbmk {

constexpr int kBlockX = 128;
constexpr int kBlockY = 2;

inline dim3 grid_for(int nx, int ny) {
    return dim3((unsigned)((nx + kBlockX - 1) / kBlockX), (unsigned)((ny + kBlockY - 1) / kBlockY), 1u);
}

// Rows per thread of the diagnostics: one where the grid hardly fills the
// device (in blocks of 128 x 2 threads), up to eight where blocks abound (a
// block's reduction costs as much FP64 time as two rows), in blocks of 128 x 1.
inline int diag_rows(int nx, int ny) {
    const long long nodes = (long long)nx * ny;
    return nodes <= 65536 && ny <= 32768 ? 1 : nodes <= 524288 ? 4 : 8;   // (at most 65,535 blocks along y)
}

inline dim3 diag_block(int nx, int ny) { return dim3(128, diag_rows(nx, ny) == 1 ? 2 : 1); }

inline dim3 diag_grid(int nx, int ny) {
    const int r = diag_rows(nx, ny) * (int)diag_block(nx, ny).y;
    return dim3((unsigned)((nx + 127) / 128 + 1), (unsigned)((ny + r - 1) / r), 1u);   // and a column for the wall flux
}

// Rows of four partial sums that a run's scratch holds: one per 128 x 2 nodes,
// which every grid above needs at most.
inline int diag_blocks(int nx, int ny) { return ((nx + 127) / 128) * ((ny + 1) / 2); }

// Uniform initial state: one value per logical population (9 flow, Q PCM, Q
// metal, in the order of Eq. 11), the low part of the PCM rest population
// (MODE_F32), and zero history.
struct InitVals {
    double f[9], g[9], h[9], g0_lo;
};

template <int M, int QT, bool FLOW>
__global__ void init_kernel(const __grid_constant__ StepParams<typename ModeTraits<M>::R> P,
                            const __grid_constant__ InitVals V) {
    using R = typename ModeTraits<M>::R;
    using PL = Planes<M, QT, FLOW>;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= P.nx || y >= P.ny) return;
    auto* db = bulk_at<M, QT, FLOW>(const_cast<char*>(P.src), P, x, y);
    if constexpr (FLOW)
        for (int q = 0; q < 9; ++q) stb<M>(db + q * kChunk, (R)(V.f[q] * (double)P.fscale));
    if constexpr (kSplit<M>) {
        float* dw = wide_at<M, QT, FLOW>(const_cast<char*>(P.src), P, x, y);
        const float g0 = (float)V.g[0], h0 = (float)V.h[0];
        dw[0] = g0;
        dw[kChunk] = h0;
        for (int q = 1; q < QT; ++q) {
            stb<M>(db + PL::pcm(q) * kChunk, (float)V.g[q] - P.w_move[q] * pcm_ref(P, g0));
            stb<M>(db + PL::met(q) * kChunk, (float)V.h[q] - P.w_move[q] * P.kappa_m * h0);
        }
    } else {
        for (int q = 0; q < QT; ++q) {
            stb<M>(db + PL::pcm(q) * kChunk, (R)V.g[q]);
            stb<M>(db + PL::met(q) * kChunk, (R)V.h[q]);
        }
        if constexpr (kComp<M>) stb<M>(db + PL::lo * kChunk, (R)V.g0_lo);
    }
    P.dT[y * P.pitch + x] = R(0);
}

// Dense copy of the state, [q][ny][nx] per lattice in the run's arithmetic
// type (state I/O converts through it).  to_dense = 1 reads the current copy
// into the dense arrays, 0 writes the dense arrays into the copy; a null
// array is skipped.  The 16-bit modes decode (encode) the moving thermal
// populations with the reference of their node; FP32 carries the low part
// of the PCM rest population in lo (taken as zero on writing when lo is null
// and g is given).
template <typename R>
struct DenseState {
    R* f;      // 9 planes (deviations f_i - w_i)
    R* g;      // Q planes
    R* h;      // Q planes
    R* lo;     // FP32 only: low part of g_0
};

template <int M, int QT, bool FLOW>
__global__ void convert_state(const __grid_constant__ StepParams<typename ModeTraits<M>::R> P,
                              const __grid_constant__ DenseState<typename ModeTraits<M>::R> D, int to_dense) {
    using R = typename ModeTraits<M>::R;
    using B = typename ModeTraits<M>::B;
    using PL = Planes<M, QT, FLOW>;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= P.nx || y >= P.ny) return;
    const long long k = (long long)y * P.nx + x, dpl = (long long)P.nx * P.ny;
    B* db = bulk_at<M, QT, FLOW>(const_cast<char*>(P.src), P, x, y);
    if (to_dense) {
        if (FLOW && D.f)
            for (int q = 0; q < 9; ++q) D.f[q * dpl + k] = to_f(db[q * kChunk]) * P.finv;
        if constexpr (kSplit<M>) {
            const float* dw = wide_at<M, QT, FLOW>(P.src, P, x, y);
            if (D.g) {
                const float rg = pcm_ref(P, dw[0]);
                D.g[k] = dw[0];
                for (int q = 1; q < QT; ++q) D.g[q * dpl + k] = to_f(db[PL::pcm(q) * kChunk]) + P.w_move[q] * rg;
            }
            if (D.h) {
                const float rm = P.kappa_m * dw[kChunk];
                D.h[k] = dw[kChunk];
                for (int q = 1; q < QT; ++q) D.h[q * dpl + k] = to_f(db[PL::met(q) * kChunk]) + P.w_move[q] * rm;
            }
        } else {
            if (D.g)
                for (int q = 0; q < QT; ++q) D.g[q * dpl + k] = to_f(db[PL::pcm(q) * kChunk]);
            if (D.h)
                for (int q = 0; q < QT; ++q) D.h[q * dpl + k] = to_f(db[PL::met(q) * kChunk]);
            if constexpr (kComp<M>)
                if (D.lo) D.lo[k] = db[PL::lo * kChunk];
        }
    } else {
        if (FLOW && D.f)
            for (int q = 0; q < 9; ++q) db[q * kChunk] = from_f<B>(D.f[q * dpl + k] * P.fscale);
        if constexpr (kSplit<M>) {
            float* dw = wide_at<M, QT, FLOW>(const_cast<char*>(P.src), P, x, y);
            if (D.g) {
                const float rg = pcm_ref(P, D.g[k]);
                dw[0] = D.g[k];
                for (int q = 1; q < QT; ++q) db[PL::pcm(q) * kChunk] = from_f<B>(D.g[q * dpl + k] - P.w_move[q] * rg);
            }
            if (D.h) {
                const float rm = P.kappa_m * D.h[k];
                dw[kChunk] = D.h[k];
                for (int q = 1; q < QT; ++q) db[PL::met(q) * kChunk] = from_f<B>(D.h[q * dpl + k] - P.w_move[q] * rm);
            }
        } else {
            if (D.g)
                for (int q = 0; q < QT; ++q) db[PL::pcm(q) * kChunk] = from_f<B>(D.g[q * dpl + k]);
            if (D.h)
                for (int q = 0; q < QT; ++q) db[PL::met(q) * kChunk] = from_f<B>(D.h[q * dpl + k]);
            if constexpr (kComp<M>)
                if (D.lo || D.g) db[PL::lo * kChunk] = D.lo ? D.lo[k] : R(0);
        }
    }
}

template <int M, typename Fn>
inline cudaError_t dispatch(int qt, int flow, Fn&& fn) {
    if (qt == 5) return flow ? fn.template operator()<M, 5, true>() : fn.template operator()<M, 5, false>();
    return flow ? fn.template operator()<M, 9, true>() : fn.template operator()<M, 9, false>();
}

// The step kernels also take PH (the Eq. 9 per-node rates compiled in or not).
template <int M, typename Fn>
inline cudaError_t dispatch_step(int qt, int flow, int ph, Fn&& fn) {
    return dispatch<M>(qt, flow, [&]<int MM, int Q, bool F>() {
        return ph ? fn.template operator()<MM, Q, F, true>() : fn.template operator()<MM, Q, F, false>();
    });
}

// Block shape of the one-node-per-thread step kernel (GB300, us per step).
// FP64: 64 x 1; two warps spread over the SMs' schedulers better than four where
// each scheduler has only a few, 64 cycles an operation each (128 x 1 / 64 x 1:
// 150^2 15.9 / 12.6, 256^2 30.1 / 28.3).  Others: 64 x 2 up to 40,000 nodes
// (128^2 in one step per launch 1.63, 128 x 1 1.73); 128 x 1 from there; where
// the grid takes more than a wave of blocks (131,072 nodes, or columns so idle
// that its blocks of 128 x 1 are more than 8 per SM), the width of 128, 64 and 32 that
// leaves the fewest columns idle (128 x 1 / 64 x 1 / 32 x 2, FP32: 400 x 390
// 4.11 / 3.62 / 3.61, 777 x 501 7.10 / 7.03 / 6.80, 512^2 5.00 all; 128 x 1 / chosen,
// D2Q9 137 x 689 4.76 / 3.37, 290 x 420 4.30 / 3.72, D2Q5 150 x 800 3.95 / 3.02).
constexpr int kNumSMs = 152;

inline dim3 step_block(int mode, int nx, int ny) {
    const long long nodes = (long long)nx * ny;
    if (mode == MODE_F64) return dim3(64, 1);
    if (nodes <= 40000) return dim3(64, 2);
    auto cover = [&](int w) { return (nx + w - 1) / w * w; };
    if (nodes <= 1ll << 17 && cover(128) / 128 * (long long)ny <= 8 * kNumSMs) return dim3(128, 1);
    if (cover(128) <= cover(64)) return dim3(128, 1);
    return cover(64) <= cover(32) ? dim3(64, 1) : dim3(32, 2);
}

// Step forms.  FORM_SINGLE is one step per launch, one node per thread,
// FORM_PAIRS that with node pairs (fused_step_pair, the default configuration
// only: flow, D2Q5, volumetric blend, FP32 arithmetic) and the L2 prefetch.
// Automatic: pairs
// with the prefetch for the 16-bit forms from 1536 x 1024 nodes up (at 1024^2,
// whose state nearly fits in L2, the prefetch gains nothing; in FP32, bound by
// HBM, one node per thread is faster at every size).
enum : int { FORM_AUTO = 0, FORM_SINGLE = 1, FORM_PAIRS = 2, FORM_TWO_STEPS = 3 };
constexpr long long kPairMinNodes = 3ll << 19;

// The rule (host code; lbm_step_form_for reports it): the form a run takes,
// FORM_SINGLE (one step per launch, pairs without the prefetch among them) or
// FORM_PAIRS.  mode: MODE_*.
inline int form_for(int mode, int qt, int flow, int solid_scheme, long long nodes, int form) {
    const bool pairs = mode != MODE_F64 && qt == 5 && flow && !solid_scheme;
    if (form == FORM_PAIRS) return pairs ? FORM_PAIRS : FORM_SINGLE;
    if (form == FORM_SINGLE || form == FORM_TWO_STEPS) return FORM_SINGLE;
    if (pairs && (mode == MODE_F16 || mode == MODE_BF16) && nodes >= kPairMinNodes) return FORM_PAIRS;
    return FORM_SINGLE;
}

// Two time steps per launch (fused_step2) for runs with flow in FP32, FP16
// or BF16 storage: forced by FORM_TWO_STEPS; automatic, for the D2Q5 thermal
// lattices, on grids of up to kTwoStepSmallMaxNodes nodes (the launch floor and
// one dependency chain per step dominate there) and for FP32 on grids of at
// least kTwoStepF32MinNodes (two state copies, 168 bytes per node, exceed the
// 129 MB L2, and two steps per launch move the state through HBM once per two
// steps).  Between the two the state sits in L2 and the step is bound by
// instruction issue, which the redundant ring only adds to.  The thresholds
// were set on an earlier node update's times (us per step, one against two
// steps per launch; FP32: 256^2 2.40 / 2.02, 320^2 3.01 / 2.74,
// 352^2 3.16 / 3.30, 384^2 3.39 / 4.26, 512^2 4.99 / 5.98, 768^2 11.1 / 12.2,
// 896^2 19.1 / 16.9, 1024^2 26.5 / 21.9, 2048^2 99.7 / 81.2; FP16: 320^2
// 3.14 / 2.91, 352^2 3.20 / 4.25).  The current one takes FP32 256^2 2.21 / 1.82,
// 320^2 2.83 / 2.43, 352^2 2.94 / 3.10, 768^2 9.3 / 10.9, 896^2 13.1 / 14.2, 1024^2
// 21.6 / 18.2, 2048^2 99.3 / 70.5, FP16 320^2 2.97 / 2.62, 352^2 2.98 / 3.72: by it the
// FP32 line would lie some way above 896^2 (802,816 nodes).  Single steps (an odd
// remainder, batches) keep the form above.
constexpr long long kTwoStepSmallMaxNodes = 320 * 320;
constexpr long long kTwoStepF32MinNodes = 3ll << 18;

inline bool two_steps_for(int mode, int qt, int flow, long long nodes, int form) {
    const bool can = mode != MODE_F64 && flow;
    if (form == FORM_TWO_STEPS) return can;
    if (form != FORM_AUTO || !can || qt != 5) return false;
    return nodes <= kTwoStepSmallMaxNodes || (mode == MODE_F32 && nodes >= kTwoStepF32MinNodes);
}

// The automatic single step, and the single steps of FORM_TWO_STEPS, take pairs
// without the prefetch too, in 16-bit runs of kPairPlainMinNodes nodes and more
// where they are the faster form (GB300, us per step, one node / pairs, FP16):
//   * beyond about one wave of one-node blocks (10 of 128 threads per SM) always:
//     1000 x 200 4.42 / 3.98, 512^2 5.1 / 4.7, 640^2 7.33 / 6.35, 1217 x 1011 20.3 / 16.3;
//   * within the wave, where a step takes as long as the busiest SM's blocks one
//     after another, if those of pairs are half as many or fewer: 600 x 240 (8 and
//     4) 3.45 / 3.27, 600 x 300 (10 and 5) 3.93 / 3.63, but 512 x 256 (7 and 4) 3.02 /
//     3.40, 512 x 340 (9 and 5) 3.62 / 3.78, 448 x 300 (7 and 4) 3.02 / 3.28;
//   * in odd widths the last node is a second chain for its warp of pairs, unless
//     it has the warp for itself (nx mod 64 = 1: 513 x 300 3.69 / 3.54, 577^2 6.64 /
//     5.85): from kPairOddMinNodes (333 x 700 5.27 / 5.87, 593 x 411 5.14 / 5.37, 901 x
//     360 6.22 / 6.27, 1201 x 300 6.63 / 6.35, 777 x 501 7.24 / 7.15, 865 x 801 11.9 / 10.7).
// In FP32 one node per thread is faster (512^2 4.83 / 5.23).
constexpr long long kPairPlainMinNodes = 1ll << 17, kPairOddMinNodes = 360000;

inline bool plain_pairs(int nx, int ny) {
    const long long nodes = (long long)nx * ny;
    if (nodes < kPairPlainMinNodes) return false;
    if (nx & 1) return nx % 64 == 1 || nodes >= kPairOddMinNodes;
    const dim3 b = step_block(MODE_F16, nx, ny);
    auto busiest = [](long long blocks) { return (blocks + kNumSMs - 1) / kNumSMs; };
    auto blocks = [&](int w, int h) { return (long long)((nx + w - 1) / w) * ((ny + h - 1) / h); };
    // in blocks of 64 threads, as which those of 128 count twice
    const long long one = busiest(blocks((int)b.x, (int)b.y)) * (b.x * b.y / 64), pairs = 2 * busiest(blocks(64, 4));
    return one > 18 || 2 * pairs <= one;
}

// Whether a run's one-step kernel takes node pairs (chosen: see step_launch).
template <int M>
inline bool pairs_of(const StepParams<typename ModeTraits<M>::R>& P, int qt, int flow, int form, bool chosen) {
    if (form_for(M, qt, flow, P.solid_scheme, (long long)P.nx * P.ny, form) == FORM_PAIRS) return true;
    return form != FORM_SINGLE && !chosen && kSplit<M> && qt == 5 && flow && !P.solid_scheme && plain_pairs(P.nx, P.ny);
}

// Whether a run's launches mark their reads evict-first (read_state): from
// kStreamMinBytes, where the two copies and the history begin to overflow L2, to
// kStreamMaxBytes, beyond which they stream through it anyway and the marking
// costs (GB300, us per step without / with.  FP32: 700^2, 80 MB, 8.60 / 8.69,
// 740^2, 90 MB, 11.2 / 10.5, 768^2 11.7 / 9.3, 1024^2 in two steps per launch, 172
// MB, 19.4 / 18.4, 1150^2, 217 MB, 24.1 / 25.9; with D2Q9 700^2, 112 MB, 16.2 /
// 12.7, 900^2, 185 MB, 29.6 / 28.4, 1100^2, 276 MB, 42.5 / 45.6, in two steps per
// launch (forced) 700^2 16.3 / 15.2, 800^2, 146 MB, 20.2 / 18.2.  FP16: 900^2, 71
// MB, 11.7 / 11.6, 1000^2, 88 MB, 14.7 / 13.7, 1200^2, 127 MB, 25.3 / 18.6.)  A
// marked line is not prefetched: it would be dropped before its block reads it.
// The runs of a batch share L2: grouped launches go by the nodes of all runs
// (12 cavities of 106-471 nodes a side, us per step of all: FP16 map 4, 90 MB,
// 17.7 / 16.1, FP32 map 5, 167 MB, 22.8 / 20.0, FP32 map 4 25.5 / 24.5), the other
// maps' kernels don't mark.
constexpr long long kStreamMinBytes = 84000000, kStreamMaxBytes = 180000000;

inline bool streams(int mode, int qt, int flow, long long nodes) {
    const int fb = flow ? 9 : 0;
    const long long copy = mode == MODE_F32 ? 4 * (fb + 2 * qt + 1) : 2 * (fb + 2 * (qt - 1)) + 8;
    const long long bytes = (2 * copy + 4) * nodes;
    return flow && mode != MODE_F64 && bytes >= kStreamMinBytes && bytes <= kStreamMaxBytes;
}

// L2 prefetch distance of the node-pair kernel in rows (0: off): grids of at
// least kPrefetchMinNodes nodes, whose state is far larger than L2, prefetch
// each block's chunk rows this far ahead, past most of the blocks resident at
// the same time.  One node per thread takes no prefetch: in FP32 it already
// runs at the copy bandwidth, and the extra requests slowed it down.
constexpr long long kPrefetchMinNodes = 3ll << 19;
constexpr int kPrefetchRowsPairs = 48;

inline int prefetch_rows_for(int mode, int qt, int flow, int solid_scheme, long long nodes, int form) {
    if (nodes < kPrefetchMinNodes) return 0;
    return form_for(mode, qt, flow, solid_scheme, nodes, form) == FORM_PAIRS ? kPrefetchRowsPairs : 0;
}

// The two-step kernel's distance, for FP32 grids whose state exceeds L2 (GB300,
// us per step without / with: 2048^2 80.8 / 71.3, 4096^2 317 / 279; distances of
// 10 to 40 rows within 1 % of each other but for the widest).  The blocks that read the rows start about 2 us later.
constexpr int kPrefetchRowsTwoSteps = 20;

inline int prefetch_rows_two_steps(int mode, long long nodes) {
    return mode == MODE_F32 && nodes >= kTwoStepF32MinNodes ? kPrefetchRowsTwoSteps : 0;
}

// FP64 runs without flow take conduction_step_lanes while its warps, of 16
// nodes, find a scheduler each (152 SMs x 4; 200 x 4 2.63 us per step against
// 3.46 with one lane per node); beyond, two warps of one lattice's FP64
// operations in turn take longer than one warp of both lattices', which share
// some.
constexpr long long kConductionLanesMaxNodes = kNumSMs * 4 * 16;

// The one-step kernel of a run, with its grid: one node per thread in blocks of
// b threads, node pairs in blocks of 32 x 4, or two lanes per node.  chosen: b is
// the caller's choice for this run, which then steps one node per thread unless
// its form is FORM_PAIRS.
struct StepLaunch {
    const void* fn;
    dim3 grid, block;
};

template <int M>
StepLaunch step_launch(const StepParams<typename ModeTraits<M>::R>& P, int qt, int flow, int form, dim3 b,
                       bool stream = false, bool chosen = false) {
    while (P.ny > 65535ll * b.y) b = dim3(b.x / 2, b.y * 2);   // (65,536 rows are admitted, 65,535 blocks along y)
    StepLaunch L{nullptr, dim3(), b};
    if constexpr (M != MODE_F64) {
        if (pairs_of<M>(P, qt, flow, form, chosen)) {
            if (stream) L.fn = P.phase_k ? (const void*)fused_step_pair<M, true, true> : (const void*)fused_step_pair<M, false, true>;
            else L.fn = P.phase_k ? (const void*)fused_step_pair<M, true> : (const void*)fused_step_pair<M, false>;
            L.block = dim3(32, 4);   // 2048^2 FP16 61.25 us per step (64 x 2: 61.98)
            L.grid = dim3((unsigned)(((P.nx + 1) / 2 + 31) / 32), (unsigned)((P.ny + 3) / 4), 1u);
            return L;
        }
    }
    if constexpr (M == MODE_F64) {
        if (!chosen && qt == 5 && !flow && !P.phase_k && (long long)P.nx * P.ny <= kConductionLanesMaxNodes) {
            L.fn = (const void*)conduction_step_lanes<M>;
            L.block = dim3(64, 1);
            L.grid = dim3((unsigned)((P.nx + 31) / 32), (unsigned)P.ny, 1u);
            return L;
        }
    }
    dispatch_step<M>(qt, flow, P.phase_k, [&]<int MM, int Q, bool F, bool PH>() {
        L.fn = (const void*)fused_step<MM, Q, F, PH>;
        if constexpr (F && MM != MODE_F64)
            if (stream) L.fn = (const void*)fused_step<MM, Q, F, PH, true>;
        return cudaSuccess;
    });
    L.grid = dim3((unsigned)((P.nx + b.x - 1) / b.x), (unsigned)((P.ny + b.y - 1) / b.y), 1u);
    return L;
}

// Grouped launches (map 4 of a batch): runs below kGroupMaxNodes nodes share
// grouped launches; larger runs, whose own step kernel fills the device,
// keep it (a chain of their own, as under map 3).
constexpr long long kGroupMaxNodes = 1ll << 20;

// The tile of a run in a grouped launch: the narrowest waste of threads among
// tiles 32, 64 and 128 nodes wide (ties to the wider); the idle fraction of the
// covered columns, (cover - nx) / cover, compared exactly.
inline int group_tile(int nx) {
    int best = 2;
    long long best_cover = ((nx + 127) / 128) * 128ll;
    for (int k = 1; k >= 0; --k) {
        const int w = 32 << k;
        const long long cover = (long long)((nx + w - 1) / w) * w;
        if ((cover - nx) * best_cover < (best_cover - nx) * cover) {
            best = k;
            best_cover = cover;
        }
    }
    return best;
}

// Whether the grouped launches of a batch take node pairs, by the nodes of all
// its grouped runs, whose launches run side by side: below kGroupPairsMinNodes
// one warp's chain bounds them, not instruction issue (GB300, us per step of all,
// one node / pairs, FP16: one run of 25,600 nodes 2.05 / 2.29, two of 17,416 together
// 2.11 / 3.15, 8 of 284,456 5.44 / 5.96, 3 of 380,495 6.72 / 6.98, 16 of 560,742 10.72 /
// 9.17, 5 of 580,808 10.21 / 8.74, 30 of 2,683,681 53.9 / 51.1; BF16 within 3 % of these).
constexpr long long kGroupPairsMinNodes = 7ll << 16;

inline bool group_pairs(int mode, int qt, int flow, long long nodes) {
    return (mode == MODE_F16 || mode == MODE_BF16) && qt == 5 && flow && nodes >= kGroupPairsMinNodes;
}

// Blocks of one run in a grouped launch (blocks of 128 threads, one node or one
// pair each).
inline long long group_blocks(int nx, int ny, int tile, bool pairs) {
    const int w = 32 << tile, h = (pairs ? 256 : 128) / w;
    return (long long)((nx + w - 1) / w) * ((ny + h - 1) / h);
}

// stream: reads marked evict-first (runs with flow, not in FP64; 16-bit runs of
// D2Q5 then take pairs, since they are beyond kGroupPairsMinNodes).
template <int M, int NR, bool EV>
const void* group_kernel_nr(int qt, int flow, int ph, bool pairs) {
    if constexpr (kSplit<M>)
        if (pairs)
            return ph ? (const void*)group_step_pair<M, true, NR, EV> : (const void*)group_step_pair<M, false, NR, EV>;
    const void* fn = nullptr;
    dispatch_step<M>(qt, flow, ph, [&]<int MM, int Q, bool F, bool PH>() {
        fn = (const void*)group_step<MM, Q, F, PH, NR, (EV && F && !(kSplit<MM> && Q == 5))>;
        return cudaSuccess;
    });
    return fn;
}

// few: the build for at most kGroupFew runs.
template <int M>
const void* group_kernel(int qt, int flow, int ph, bool few, bool stream, bool pairs) {
    constexpr int all = kGroupRuns<typename ModeTraits<M>::R>;
    if constexpr (M != MODE_F64)
        if (stream)
            return few ? group_kernel_nr<M, kGroupFew, true>(qt, flow, ph, pairs)
                       : group_kernel_nr<M, all, true>(qt, flow, ph, pairs);
    return few ? group_kernel_nr<M, kGroupFew, false>(qt, flow, ph, pairs)
               : group_kernel_nr<M, all, false>(qt, flow, ph, pairs);
}

// Launched as a programmatic dependent of the previous step (the kernels wait
// for it before touching the state), so the launch overlaps its tail.
template <int M>
cudaError_t launch_step(const StepParams<typename ModeTraits<M>::R>& P, int qt, int flow, int form, cudaStream_t s) {
    const bool stream = streams(M, qt, flow, (long long)P.nx * P.ny);
    const StepLaunch L = step_launch<M>(P, qt, flow, form, step_block(M, P.nx, P.ny), stream);
    void* args[1] = {const_cast<StepParams<typename ModeTraits<M>::R>*>(&P)};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = L.grid;
    cfg.blockDim = L.block;
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, L.fn, args);
}

// Block height of the two-step kernel (blocks of kT2W x H threads, inner
// tiles of (kT2W - 2) x (H - 2) nodes) for an nx x ny grid on nsm SMs.  Among
// the heights that leave at most two tiles per SM, the one whose busiest SM
// runs the fewest node updates (its tiles, rounded up over the SMs, times the
// block's warps for the first step and the inner tile for the second), with
// the work of two tiles per SM counted at kT2Overlap: two resident blocks
// overlap each other's L2 loads and barrier.  On 152 SMs: 128^2 takes H = 6
// (128 tiles), 192^2 H = 10 (144), 256^2 H = 9 (296; fitted on FP32 times of
// 2.04 us per step against 2.21 for H = 16 and one tile per SM, now 1.82).  One
// tile per SM takes up to kT2H rows, two up to kT2HTwo (what their registers
// allow).  Other grids take H = kT2HMany = 12, measured fastest there (FP32:
// three resident blocks of 13 warps per SM; 1024^2 and 2048^2 against H = 6, 8,
// 10, 14, 16; 65 x 1400, two tiles of 16 rows per SM before: 3.37 / 3.17).
constexpr double kT2Overlap = 0.87;

inline long long t2_tiles(int n, int inner) { return t2_count(n, inner); }

inline dim3 t2_grid(int nx, int ny, int h) {
    return dim3((unsigned)t2_tiles(nx, kT2W - 2), (unsigned)t2_tiles(ny, h - 2), 1u);
}

struct T2Shape {
    int h;    // block height
    int hm;   // the build, kT2H, kT2HTwo or kT2HMany
    bool stream;   // kT2HMany in FP32: reads marked evict-first
    bool thermal;  // kT2H in FP32, D2Q5: the thermal lattices collide first
};

// Height from which two blocks of the first build don't fit an SM's registers
// (FP32 64, with D2Q9 76; 16-bit 75, with D2Q9 94), so that two tiles per SM take
// the build capped for them (D2Q9, us per step uncapped / capped: FP32 300^2 4.04 /
// 3.30, 320^2 4.20 / 3.39, 334 x 303 4.39 / 3.74, FP16 300 x 260 3.91 / 3.21, 320^2 4.55 /
// 3.75, BF16 334 x 303 4.68 / 4.08).
inline int t2_two_from(int mode, int qt) { return mode == MODE_F32 ? (qt == 5 ? kT2HTwo + 1 : 12) : (qt == 5 ? 12 : 10); }

// Rows of tiles per SM from which the FP32 D2Q5 tiles let the thermal lattices
// collide first: with the schedulers full the order that frees registers
// early wins, with a few warps the one whose chain is shorter (us per step,
// flow / thermal lattices first: 64^2, 4 rows, 1.09 / 1.12, 128^2, 6, 1.22 / 1.25,
// 150^2, 7, and 200^2, 10, the same, 256 x 242, 15, 1.89 / 1.86, 256^2, 18, 1.86 /
// 1.82, 300^2, 24, 2.41 / 2.38, 320^2, 26, 2.47 / 2.43; with Eq. 9 256^2 1.89 /
// 1.91, not taken).
constexpr int kT2ThermalRows = 15;

inline T2Shape t2_block(int mode, int qt, int nx, int ny, int nsm) {
    if (nsm < 1) nsm = 1;
    T2Shape best = {kT2HMany, kT2HMany, mode == MODE_F32 && streams(mode, qt, 1, (long long)nx * ny), false};
    double best_cost = -1.0;
    for (int h = 4; h <= kT2H; ++h) {
        const long long tiles = t2_tiles(nx, kT2W - 2) * t2_tiles(ny, h - 2);
        const long long per_sm = (tiles + nsm - 1) / nsm;
        if (per_sm > 2 || (per_sm == 2 && h > kT2HTwo)) continue;
        const long long work = per_sm * ((kT2W * h + 31) / 32 * 32 + (long long)(kT2W - 2) * (h - 2));
        const double cost = per_sm > 1 ? kT2Overlap * (double)work : (double)work;
        if (best_cost < 0.0 || cost < best_cost) {
            best = {h, per_sm == 2 && h >= t2_two_from(mode, qt) ? kT2HTwo : kT2H, false,
                    mode == MODE_F32 && qt == 5 && per_sm * h >= kT2ThermalRows};
            best_cost = cost;
        }
    }
    return best;
}

// The build of the kernel and its dynamic shared memory (300^2 with 12 rows and
// two tiles per SM takes 2.53 us per step in the many-tiles build, 2.44 in the
// first).
template <int M, int HM, bool EV = false>
const void* step2_kernel_hm(int qt, int phase_k) {
    if (qt == 9)
        return phase_k ? (const void*)fused_step2<M, 9, true, HM, EV> : (const void*)fused_step2<M, 9, false, HM, EV>;
    if constexpr (HM == kT2HTwo && M == MODE_F32) return nullptr;   // (two blocks of up to 14 rows fit as they are)
    else return phase_k ? (const void*)fused_step2<M, 5, true, HM, EV> : (const void*)fused_step2<M, 5, false, HM, EV>;
}

template <int M>
const void* step2_kernel(int qt, int phase_k, T2Shape t) {
    const int hm = t.hm;
    if constexpr (M == MODE_F32) {
        if (t.stream) return step2_kernel_hm<M, kT2HMany, true>(qt, phase_k);
        if (t.thermal && !phase_k) return (const void*)fused_step2<M, 5, false, kT2H, false, true>;
    }
    if constexpr (M != MODE_F64) {
        if (hm == kT2HMany) return step2_kernel_hm<M, kT2HMany>(qt, phase_k);
        return hm == kT2HTwo ? step2_kernel_hm<M, kT2HTwo>(qt, phase_k) : step2_kernel_hm<M, kT2H>(qt, phase_k);
    }
    return nullptr;
}

template <int M, int HM>
constexpr size_t step2_smem_hm(int qt) {
    return qt == 5 ? Tile2<M, 5, HM>::bytes : Tile2<M, 9, HM>::bytes;
}

template <int M>
size_t step2_smem(int qt, int hm) {
    if constexpr (M != MODE_F64) {
        if (hm == kT2HMany) return step2_smem_hm<M, kT2HMany>(qt);
        return hm == kT2HTwo ? step2_smem_hm<M, kT2HTwo>(qt) : step2_smem_hm<M, kT2H>(qt);
    }
    return 0;
}

// Batch map 5: the grouped two-step kernel and its shared memory (the 12-row
// build; blocks of kT2W x kT2HMany threads).
template <int M, int NR, bool EV>
const void* group2_kernel_nr(int qt, int phase_k) {
    if (qt == 5) return phase_k ? (const void*)group_step2<M, 5, true, NR, EV> : (const void*)group_step2<M, 5, false, NR, EV>;
    return phase_k ? (const void*)group_step2<M, 9, true, NR, EV> : (const void*)group_step2<M, 9, false, NR, EV>;
}

template <int M>
const void* group2_kernel(int qt, int phase_k, bool few, bool stream) {
    if constexpr (M == MODE_F32)
        if (stream)
            return few ? group2_kernel_nr<M, kGroupFew, true>(qt, phase_k)
                       : group2_kernel_nr<M, kGroupRuns<float>, true>(qt, phase_k);
    if constexpr (M != MODE_F64)
        return few ? group2_kernel_nr<M, kGroupFew, false>(qt, phase_k)
                   : group2_kernel_nr<M, kGroupRuns<float>, false>(qt, phase_k);
    return nullptr;
}

inline long long group2_blocks(int nx, int ny) { return t2_tiles(nx, kT2W - 2) * t2_tiles(ny, kT2HMany - 2); }

// Lets the kernel of a run's two-step launches take its shared memory; once,
// before the first of them on the device.
template <int M>
cudaError_t prepare_step2(int qt, int phase_k, T2Shape t) {
    const void* fn = step2_kernel<M>(qt, phase_k, t);
    if (!fn) return cudaErrorInvalidConfiguration;
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)step2_smem<M>(qt, t.hm));
}

// Two steps from copy P.src to P.dst, history P.dT -> P.dT_out, in blocks of
// kT2W x t.h threads, as a programmatic dependent of the previous launch in the
// stream.
template <int M>
cudaError_t launch_step2(const StepParams<typename ModeTraits<M>::R>& P, int qt, T2Shape t, cudaStream_t s) {
    if (t.h < 4 || t.h > t.hm) return cudaErrorInvalidConfiguration;
    const void* fn = step2_kernel<M>(qt, P.phase_k, t);
    if (!fn) return cudaErrorInvalidConfiguration;
    const size_t smem = step2_smem<M>(qt, t.hm);
    void* args[1] = {const_cast<StepParams<typename ModeTraits<M>::R>*>(&P)};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = t2_grid(P.nx, P.ny, t.h);
    cfg.blockDim = dim3((unsigned)kT2W, (unsigned)t.h, 1u);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, fn, args);
}

template <int M>
cudaError_t launch_fields(const StepParams<typename ModeTraits<M>::R>& P,
                          const FieldOut<typename ModeTraits<M>::R>& o, int qt, int flow, cudaStream_t s) {
    const dim3 g = grid_for(P.nx, P.ny), b(kBlockX, kBlockY);
    return dispatch<M>(qt, flow, [&]<int MM, int Q, bool F>() {
        fields_kernel<MM, Q, F><<<g, b, 0, s>>>(P, o);
        return cudaGetLastError();
    });
}

template <int M>
cudaError_t launch_diag(const StepParams<typename ModeTraits<M>::R>& P, const DiagConst& C, double* scratch,
                        double* out, int qt, int flow, cudaStream_t s) {
    const dim3 g = diag_grid(P.nx, P.ny), b = diag_block(P.nx, P.ny);
    cudaError_t e = dispatch<M>(qt, flow, [&]<int MM, int Q, bool F>() {
        diag_partial<MM, Q, F><<<g, b, 0, s>>>(P, C, scratch);
        return cudaGetLastError();
    });
    if (e != cudaSuccess) return e;
    diag_finalize<<<1, 512, 0, s>>>(scratch, (int)((g.x - 1) * g.y), (double)P.nx * P.ny, out);
    return cudaGetLastError();
}

template <int M>
cudaError_t launch_init(const StepParams<typename ModeTraits<M>::R>& P, const InitVals& V, int qt, int flow,
                        cudaStream_t s) {
    const dim3 g = grid_for(P.nx, P.ny), b(kBlockX, kBlockY);
    return dispatch<M>(qt, flow, [&]<int MM, int Q, bool F>() {
        init_kernel<MM, Q, F><<<g, b, 0, s>>>(P, V);
        return cudaGetLastError();
    });
}

template <int M>
cudaError_t launch_convert(const StepParams<typename ModeTraits<M>::R>& P,
                           const DenseState<typename ModeTraits<M>::R>& D, int to_dense, int qt, int flow,
                           cudaStream_t s) {
    const dim3 g = grid_for(P.nx, P.ny), b(kBlockX, kBlockY);
    return dispatch<M>(qt, flow, [&]<int MM, int Q, bool F>() {
        convert_state<MM, Q, F><<<g, b, 0, s>>>(P, D, to_dense);
        return cudaGetLastError();
    });
}

// ph: some run of the batch uses the Eq. 9 per-node rates.
template <int M>
cudaError_t launch_batch(const StepParams<typename ModeTraits<M>::R>* runs, const Tile* tiles, int ntiles,
                         int chunk, int grid, int parity, int qt, int flow, int ph, cudaStream_t s) {
    return dispatch_step<M>(qt, flow, ph, [&]<int MM, int Q, bool F, bool PH>() {
        batch_step<MM, Q, F, PH><<<grid, 256, 0, s>>>(runs, tiles, ntiles, chunk, parity);
        return cudaGetLastError();
    });
}


template <int M>
int batch_blocks_per_sm(int qt, int flow, int ph) {
    int n = 0;
    dispatch_step<M>(qt, flow, ph, [&]<int MM, int Q, bool F, bool PH>() {
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, batch_step<MM, Q, F, PH>, 256, 0);
    });
    return n;
}

// Explicit instantiations of the launchers (KW empty: in the kernel units) and
// the matching declarations (KW = extern: in the units that call them, so
// that the kernels are compiled once, in their own units).
#define LBMK_TEMPLATES(KW, M)                                                                                 \
    KW template cudaError_t launch_step<M>(const StepParams<ModeTraits<M>::R>&, int, int, int, cudaStream_t);   \
    KW template cudaError_t launch_fields<M>(const StepParams<ModeTraits<M>::R>&, const FieldOut<ModeTraits<M>::R>&, \
                                          int, int, cudaStream_t);                                            \
    KW template cudaError_t launch_diag<M>(const StepParams<ModeTraits<M>::R>&, const DiagConst&, double*, double*, \
                                        int, int, cudaStream_t);                                              \
    KW template cudaError_t launch_init<M>(const StepParams<ModeTraits<M>::R>&, const InitVals&, int, int, cudaStream_t); \
    KW template cudaError_t launch_batch<M>(const StepParams<ModeTraits<M>::R>*, const Tile*, int, int, int, int, int, \
                                         int, int, cudaStream_t);                                               \
    KW template int batch_blocks_per_sm<M>(int, int, int);                                                   \
    KW template const void* group_kernel<M>(int, int, int, bool, bool, bool);                                                  \
    KW template cudaError_t launch_step2<M>(const StepParams<ModeTraits<M>::R>&, int, T2Shape, cudaStream_t); \
    KW template cudaError_t prepare_step2<M>(int, int, T2Shape);                                              \
    KW template const void* group2_kernel<M>(int, int, bool, bool);                                                        \
    KW template size_t step2_smem<M>(int, int);                                                               \
    KW template StepLaunch step_launch<M>(const StepParams<ModeTraits<M>::R>&, int, int, int, dim3, bool, bool);

#define LBMK_CONVERT_TEMPLATES(KW, M)                                                                         \
    KW template cudaError_t launch_convert<M>(const StepParams<ModeTraits<M>::R>&, const DenseState<ModeTraits<M>::R>&, \
                                           int, int, int, cudaStream_t);


#define LBMK_INSTANTIATE(M) LBMK_TEMPLATES(, M)
#define LBMK_INSTANTIATE_CONVERT(M) LBMK_CONVERT_TEMPLATES(, M)
#define LBMK_EXTERN(M) LBMK_TEMPLATES(extern, M) LBMK_CONVERT_TEMPLATES(extern, M)

}  // namespace lbmk
