// hg_steps.h -- the resident multi-step kernel (hg_steps.cu) as the host runtime launches it.
#pragma once

#include "hg_internal.h"

namespace hg {

constexpr uint32_t kWaitLimit = 1u << 22;  // polls after which a wait gives up (seconds), unless a test sets fewer
constexpr int kStepsThreads = 512;  // most threads per block
constexpr int kStepsPerSm = 3;      // blocks of that size per SM (links in shared memory: 40 registers; else 2)
constexpr int kStepsTiles = 8;      // most tiles a site block owns
constexpr int kStepsIolets = 8;     // most iolets an iolet block owns
constexpr int kStepsSmem = 200 * 1024;  // most dynamic shared memory of a block
constexpr int kStashRows = 20;      // words of shared memory per site: 18 links, boundary slot, its word
constexpr int kStepsChunks = 16;    // iolet chunks summed at a time
constexpr int kStepsLag = 4;        // steps the iolet means may trail the sites (boundary-moment buffers)
constexpr int kStepsMax = 1024;     // most steps of one launch (bounds the table of boundary values)

// A domain of the set: its descriptor, its boundary values of steps 1 .. of a launch (n_io
// each; step 0 reads, and the last step leaves, D.bcv), and the boundary moments of the last
// kStepsLag steps (n_adj each; the last step's are left in D.bnd).
// coupled: it has inlets that follow another domain's means.
struct StepsDom {
    DomDev D;
    float *values;
    float4 *moments;
    int64_t n_adj;
    int64_t coupled;
};
// Iolet of the set (beside its IoDev): domain and index, and the coupled inlets it feeds.
struct StepsIo {
    int32_t dom, iolet, fed0, n_fed;
};
struct StepsFed {
    int32_t dom, iolet;
    double factor;
};
// Counters, zero before and after a launch.
struct StepsSync {
    alignas(128) unsigned arrived;          // site blocks that ended a step
    alignas(128) unsigned done[kStepsLag];  // iolet means of steps j = i (mod kStepsLag)
    unsigned values;                        // iolet blocks that have written their boundary values
    alignas(128) unsigned ready;            // source iolets whose coupled values are written
    alignas(128) unsigned left;             // blocks that left
};
struct StepsArgs {
    const StepsDom *doms;
    const TileDev *tiles;  // TileDev::dom indexes doms
    const IoDev *ios;
    const StepsIo *sios;
    const StepsFed *fed;
    StepsSync *sync;
    int32_t *err;
    int32_t n_doms, n_tiles, n_ios, n_sources, n_site_blocks, n_steps;
    int32_t n_groups;     // iolet blocks that take the same iolets' steps in turn
    int32_t stash_words;  // dynamic shared memory of a block
    uint32_t wait_limit;  // kWaitLimit
};
struct StepsShape {
    int grid = 0, threads = 0, groups = 1;
    size_t smem = 0;
    bool stash = false;
};

template <int S, int SCHEME>
cudaError_t steps_blocks_per_sm(bool stash, int threads, size_t smem, int *out);
template <int S, int SCHEME> cudaError_t launch_steps(const StepsArgs &a, const StepsShape &sh, cudaStream_t st);
#define HG_STEPS_DECL(S_, C_)                                                              \
    template <> cudaError_t steps_blocks_per_sm<S_, C_>(bool, int, size_t, int *);         \
    template <> cudaError_t launch_steps<S_, C_>(const StepsArgs &, const StepsShape &, cudaStream_t);
HG_STEPS_DECL(0, 0) HG_STEPS_DECL(0, 1) HG_STEPS_DECL(1, 0) HG_STEPS_DECL(1, 1) HG_STEPS_DECL(2, 0) HG_STEPS_DECL(2, 1)
#undef HG_STEPS_DECL

}  // namespace hg
