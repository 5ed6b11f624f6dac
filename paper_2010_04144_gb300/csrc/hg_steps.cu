// hg_steps.cu -- many steps of a set of small domains in one launch, for one (storage,
// scheme) combination given by HG_PART_S and HG_PART_SCHEME (compiled once per combination,
// in parallel).
//
// What bounds a step of a small domain is not memory: at 4.5 thousand sites a stream-collide
// launch and an iolet-update launch take 11.4 us per step, nearly all of it launch, drain and
// the chain of dependent latencies in the iolet update.  Here a cooperative grid stays
// resident for all the steps: most blocks own fixed tiles of sites and keep their links in
// shared memory, a few blocks do the iolet work, and one grid barrier (1.4 us) ends each step.
// Per step, launches -> resident: 4.5k sites FP32 A/B 11.4 -> 2.8 us, 13k FP32 AA 12.0 -> 2.8,
// 166k FP32 A/B 15.0 -> 6.1, 16 tubes of 279k FP16 AA 21.9 -> 11.2, coupled pair of 339k FP16
// AA 22.9 -> 11.2.  What bounds it now: the barrier and one round of L2 latencies up to ~50k
// sites, then L2 traffic.
//
//   step j:  site blocks   stream-collide (moments of iolet sites -> ring[j mod lag]), then
//                          arrive and wait for the other site blocks
//            iolet blocks  once every site block has arrived: the means of step j and the
//                          coupled values of step j + 1 that follow from them
//
// The iolet blocks trail: a site block waits for the means of step j - lag only (before it
// overwrites their ring entry), and a site next to a coupled inlet waits, in step j, for the
// values published from step j - 1.  Uncoupled boundary values depend on time alone; the
// iolet blocks write those of all the launch's steps first.  All waits are bounded: one that
// gives up sets the context's error word and the block leaves (a site that waited for a coupled
// value goes on with what is there).  Waits for a block that left run out too, and the last block
// to leave advances the step counters, as the host has, and clears the counters: the states are
// not to be trusted, the next launch is sound.  The arithmetic and every order of summation are
// those of the per-step kernels: the same bits.
#include "hg_device.cuh"
#include "hg_iolet.cuh"
#include "hg_steps.h"

#if !defined(HG_PART_S) || !defined(HG_PART_SCHEME)
#error "compile with -DHG_PART_S=.. -DHG_PART_SCHEME=.."
#endif

namespace hg {
namespace {

// Polls after which a wait gives up (StepsArgs::wait_limit).  In shared memory: as one more value
// held across the site's registers it cost 1.7 % at 166k sites FP32 A/B.
__shared__ volatile uint32_t s_wait_limit;
__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
// Counts one up after everything this thread, and every thread it has synchronised with, wrote.
__device__ __forceinline__ void add_release(unsigned *p) {
    fence_gpu();
    asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}
// Until *p >= target; false when it gave up.  (Acquiring polls: relaxed ones with a fence after
// the last measured 0.2 us per step slower.)
__device__ __forceinline__ bool wait_at_least(const unsigned *p, unsigned target) {
    for (uint32_t it = 0; it < s_wait_limit; ++it)
        if (ld_acquire(p) >= target) return true;
    return false;
}

// Which buffer holds the boundary values step j reads (0 <= j <= n; n: the step after the
// launch), and the moments step j writes.
__device__ __forceinline__ float *values_of(const StepsDom &d, int j, int n) {
    return j == 0 || j == n ? const_cast<float *>(d.D.bcv) : d.values + (int64_t)j * d.D.n_io;
}
__device__ __forceinline__ float4 *moments_of(const StepsDom &d, int j, int n) {
    return j == n - 1 ? d.D.bnd : d.moments + (j % kStepsLag) * d.n_adj;
}
// The end of step j in a site block: arrive, then wait for what step j + 1 needs.  False (for
// all threads of the block) when the wait gave up.
__device__ __forceinline__ bool end_step(const StepsArgs &a, int j) {
    bool ok = true;
    __syncthreads();
    if (threadIdx.x == 0) {
        add_release(&a.sync->arrived);
        if (j + 1 < a.n_steps) {
            const unsigned target = (unsigned)(j + 1) * (unsigned)a.n_site_blocks;
            const int old = j + 1 - kStepsLag;  // the ring entry step j + 1 overwrites
            const unsigned *also = a.n_ios == 0 ? nullptr : j == 0 ? &a.sync->values
                                   : old >= 0   ? &a.sync->done[old % kStepsLag] : nullptr;
            const unsigned also_target = j == 0 ? gridDim.x - (unsigned)a.n_site_blocks
                                                : (unsigned)(old / kStepsLag + 1) * (unsigned)a.n_ios;
            ok = false;
            for (uint32_t it = 0; it < s_wait_limit && !ok; ++it) {
                const unsigned x = also ? ld_acquire(also) : 0u;
                ok = ld_acquire(&a.sync->arrived) >= target && (!also || x >= also_target);
            }
            if (!ok) atomicExch(a.err, 1);
        }
    }
    return __syncthreads_and(ok) != 0;
}

// ---- the 18 links of a site as element indices into the distributions (row included) ----
struct StashLinks {  // one bank per thread
    const int32_t *p;
    template <typename F> __device__ __forceinline__ void each(F &&f) const {
        unroll<1, 19>([&](auto ic) { f(ic, p[(decltype(ic)::v - 1) * blockDim.x]); });
    }
};
template <int SCHEME> struct TableLinks {
    const int32_t *p;  // entry 1 of the site
    int32_t np;
    template <typename F> __device__ __forceinline__ void each(F &&f) const {
        unroll<1, 19>([&](auto ic) {
            constexpr int I = decltype(ic)::v;
            f(ic, (SCHEME == kAB ? I : OPP(I)) * np + __ldg(p + (int64_t)(I - 1) * np));
        });
    }
};
template <int SCHEME> struct RunLinks {
    RunSite r;
    int32_t s, np;
    template <typename F> __device__ __forceinline__ void each(F &&f) const {
        unroll<0, 5>([&](auto kc) {
            run_links4<decltype(kc)::v>(r.row, [&](auto ic, int32_t d) {
                constexpr int I = decltype(ic)::v;
                f(ic, ((I - 1) / 2 * 2 + 1) * np + s + run_offset<SCHEME, I>(r.w, d, np));
            });
        });
    }
};

// What a site block does at a site next to an iolet before and after the collision.
struct IoSite {
    int slot;               // -1: none
    uint32_t word;          // io_words of the slot
    const float *bcv;
    float4 *bnd;
    const unsigned *ready;  // null: no wait
    unsigned target;
    int32_t *err;
    template <int S> __device__ __forceinline__ void links(const DomDev &D, float g[19]) const {
        if (slot < 0) return;
        if (ready && !wait_at_least(ready, target)) atomicExch(err, 1);
        apply_iolet_links<S, true>(D, bcv, slot, word, g);
    }
};

// A/B step or AA odd step of site s; `again` gives the links a second time (AA scatter).
template <int S, int SCHEME, typename L>
__device__ __forceinline__ void step_site(const DomDev &D, const typename St<S>::T *src, typename St<S>::T *dst,
                                          int64_t s, L links, const IoSite &io) {
    using Tr = St<S>;
    using T = typename Tr::T;
    float g[19];
    g[0] = Tr::template ld<0>(src[s]);
    links.each([&](auto ic, int32_t at) {
        constexpr int I = decltype(ic)::v;
        g[I] = Tr::template ld<I>(src[at]);
    });
    io.template links<S>(D, g);
    const float4 m = collide_s<S>(g, D.omega);
    if constexpr (SCHEME == kAB) {
        const uint32_t npb = (uint32_t)D.np * sizeof(T);
        T *q = opaque(dst + s);
        unroll<0, 19>([&](auto ic) {
            constexpr int I = decltype(ic)::v;
            *row_at<I>(q, npb) = Tr::template st<I>(g[I]);
        });
    } else {
        T *q = opaque(dst);
        asm volatile("" ::"f"(m.x) : "memory");  // the links are read again, not kept
        q[s] = Tr::template st<0>(g[0]);
        links.each([&](auto ic, int32_t at) {
            constexpr int J = OPP(decltype(ic)::v);  // direction J goes where its opposite was read
            q[at] = Tr::template st<J>(g[J]);
        });
    }
    if (io.slot >= 0) io.bnd[io.slot] = m;
}
template <int S>
__device__ __forceinline__ void step_even(const DomDev &D, typename St<S>::T *buf, int64_t s, const IoSite &io) {
    using Tr = St<S>;
    using T = typename Tr::T;
    const uint32_t npb = (uint32_t)D.np * sizeof(T);
    float g[19];
    unroll<0, 19>([&](auto ic) {
        constexpr int I = decltype(ic)::v;
        g[I] = Tr::template ld<I>(*row_at<I>(buf + s, npb));
    });
    io.template links<S>(D, g);
    const float4 m = collide_s<S>(g, D.omega);
    T *q = opaque(buf + s);
    unroll<0, 19>([&](auto ic) {
        constexpr int I = decltype(ic)::v;
        *row_at<OPP(I)>(q, npb) = Tr::template st<I>(g[I]);
    });
    if (io.slot >= 0) io.bnd[io.slot] = m;
}

// One tile a site block owns.
struct OwnTile {
    StepsDom d;
    int64_t start;
    int32_t count, parity;  // parity: of the steps completed before the launch
};

template <int S, int SCHEME, bool STASH>
__device__ __forceinline__ void site_block(const StepsArgs &a, OwnTile *own, int32_t *stash) {
    using T = typename St<S>::T;
    const int tid = threadIdx.x, B = blockDim.x;
    int n_own = 0;
    for (int t = blockIdx.x; t < a.n_tiles; t += a.n_site_blocks) ++n_own;
    if (tid < n_own) {
        const TileDev tl = a.tiles[blockIdx.x + tid * a.n_site_blocks];
        OwnTile &o = own[tid];
        o.d = a.doms[tl.dom];
        o.start = tl.start;
        o.count = tl.count;
        o.parity = (int32_t)(*o.d.D.step & 1);
    }
    __syncthreads();
    // links (and boundary slot) of every own site into shared memory, once
    auto with_links = [&](const DomDev &D, int64_t s, auto &&f) {
        if (D.lword) f(RunLinks<SCHEME>{run_site(D, s), (int32_t)s, (int32_t)D.np});
        else f(TableLinks<SCHEME>{D.nbr + s, (int32_t)D.np});
    };
    auto slot_of = [&](const DomDev &D, int64_t s) {
        uint32_t word;
        return site_flag(D, s, word) ? site_slot(D, s, word) : -1;
    };
    if constexpr (STASH) {
        for (int i = 0; i < n_own; ++i) {
            if (tid >= own[i].count) continue;
            int32_t *p = stash + (int64_t)i * kStashRows * B + tid;
            const int64_t s = own[i].start + tid;
            with_links(own[i].d.D, s, [&](const auto &links) {
                links.each([&](auto ic, int32_t at) { p[(decltype(ic)::v - 1) * B] = at; });
            });
            const int slot = slot_of(own[i].d.D, s);
            p[18 * B] = slot;
            p[19 * B] = slot < 0 ? 0 : (int32_t)io_word(own[i].d.D, slot);
        }
    }
    for (int j = 0; j < a.n_steps; ++j) {
        for (int i = 0; i < n_own; ++i) {
            if (tid >= own[i].count) continue;
            const StepsDom &d = own[i].d;
            const DomDev &D = d.D;
            const int64_t s = own[i].start + tid;
            const bool odd = ((own[i].parity + j + 1) & 1) != 0;
            int32_t *p = stash + (int64_t)i * kStashRows * B + tid;
            IoSite io;
            io.slot = STASH ? p[18 * B] : slot_of(D, s);
            io.word = io.slot < 0 ? 0u : STASH ? (uint32_t)p[19 * B] : io_word(D, io.slot);
            io.bcv = values_of(d, j, a.n_steps);
            io.bnd = moments_of(d, j, a.n_steps);
            io.ready = d.coupled && j > 0 ? &a.sync->ready : nullptr;
            io.target = (unsigned)j * (unsigned)a.n_sources;
            io.err = a.err;
            if (SCHEME == kAA && !odd) {
                step_even<S>(D, (T *)D.f[0], s, io);
                continue;
            }
            const T *src = (const T *)D.f[SCHEME == kAA || odd ? 0 : 1];
            T *dst = (T *)D.f[SCHEME == kAA || !odd ? 0 : 1];
            if constexpr (STASH) step_site<S, SCHEME>(D, src, dst, s, StashLinks{p}, io);
            else with_links(D, s, [&](const auto &links) { step_site<S, SCHEME>(D, src, dst, s, links, io); });
        }
        if (!end_step(a, j)) return;
    }
}

// An iolet an iolet block owns.
struct OwnIolet {
    IoDev I;
    StepsIo Q;
    StepsDom d;            // its domain
    int64_t done;          // steps completed before the launch
    const int32_t *slots;  // I.slots, or their copy in shared memory
};

// The means of step j, and the values of step j + 1 of the inlets they feed.
__device__ __forceinline__ void iolet_means(const StepsArgs &a, const OwnIolet &o, int j) {
    __shared__ double2 s_warp[8 * kStepsChunks], s_chunk[kStepsChunks];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    const IoDev &I = o.I;
    const float4 *bnd = moments_of(o.d, j, a.n_steps);
    double sum_u = 0.0, sum_r = 0.0;
    for (int c0 = 0; c0 < I.n_chunks; c0 += kStepsChunks) {
        const int nc = min(kStepsChunks, I.n_chunks - c0);
        for (int q = warp; q < 8 * nc; q += n_warps) {
            const int slot = c0 * kIoChunk + q * 32 + lane;
            double su = 0.0, sr = 0.0;
            if (slot < I.n_slots) iolet_terms(I, bnd[o.slots[slot]], su, sr);
            warp_sum2(su, sr);
            if (lane == 0) s_warp[q] = make_double2(su, sr);
        }
        __syncthreads();
        for (int c = warp; c < nc; c += n_warps) {
            double su = lane < 8 ? s_warp[8 * c + lane].x : 0.0, sr = lane < 8 ? s_warp[8 * c + lane].y : 0.0;
            warp_sum2(su, sr);
            if (lane == 0) s_chunk[c] = make_double2(su, sr);
        }
        __syncthreads();
        if (threadIdx.x == 0)
            for (int c = 0; c < nc; ++c) {
                sum_u += s_chunk[c].x;
                sum_r += s_chunk[c].y;
            }
        if (c0 + kStepsChunks < I.n_chunks) __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double mean = iolet_mean(I, sum_u);
        if (j == a.n_steps - 1) iolet_store_means(I, mean, sum_r);  // the ones that can be read
        for (int f = 0; f < o.Q.n_fed; ++f) {
            const StepsFed &F = a.fed[o.Q.fed0 + f];
            values_of(a.doms[F.dom], j + 1, a.n_steps)[F.iolet] = (float)(F.factor * mean);
        }
        if (o.Q.n_fed) add_release(&a.sync->ready);
        add_release(&a.sync->done[j % kStepsLag]);
    }
    __syncthreads();  // s_warp and s_chunk are reused
}

__device__ __forceinline__ void iolet_block(const StepsArgs &a, int32_t *copy) {
    __shared__ __align__(16) OwnIolet own[kStepsIolets];
    const int stride = ((int)gridDim.x - a.n_site_blocks) / a.n_groups;
    const int first = ((int)blockIdx.x - a.n_site_blocks) % stride, group = ((int)blockIdx.x - a.n_site_blocks) / stride;
    const int n_own = (a.n_ios - first + stride - 1) / stride;  // at most kStepsIolets (host)
    if ((int)threadIdx.x < n_own) {
        const int k = first + (int)threadIdx.x * stride;
        OwnIolet &o = own[threadIdx.x];
        o.I = a.ios[k];
        o.Q = a.sios[k];
        o.d = a.doms[o.Q.dom];
        o.done = *o.I.step;
        o.slots = o.I.slots;
    }
    __syncthreads();
    for (int i = 0, room = a.stash_words; i < n_own; ++i) {
        const int n = own[i].I.n_slots;
        if (n > room) break;
        for (int q = threadIdx.x; q < n; q += blockDim.x) copy[q] = __ldg(own[i].I.slots + q);
        __syncthreads();
        if (threadIdx.x == 0) own[i].slots = copy;
        copy += n;
        room -= n;
    }
    __syncthreads();
    for (int i = 0; i < n_own && group == 0; ++i)  // FP64 remainder and cosine: one step per thread
        if (!own[i].I.coupled)
            for (int j = 1 + (int)threadIdx.x; j < a.n_steps; j += blockDim.x)
                values_of(own[i].d, j, a.n_steps)[own[i].Q.iolet] = iolet_value(own[i].I, own[i].done + j);
    __syncthreads();
    if (threadIdx.x == 0) add_release(&a.sync->values);
    for (int j = group; j < a.n_steps; j += a.n_groups) {
        bool ok = true;
        if (threadIdx.x == 0) {
            ok = wait_at_least(&a.sync->arrived, (unsigned)(j + 1) * (unsigned)a.n_site_blocks);
            if (!ok) atomicExch(a.err, 1);
        }
        if (!__syncthreads_and(ok)) return;
        for (int i = 0; i < n_own; ++i) iolet_means(a, own[i], j);
    }
    // (the last step's group: step 0 has been read by then)
    if ((a.n_steps - 1) % a.n_groups == group && (int)threadIdx.x < n_own && !own[threadIdx.x].I.coupled) {
        const OwnIolet &o = own[threadIdx.x];
        values_of(o.d, a.n_steps, a.n_steps)[o.Q.iolet] = iolet_value(o.I, o.done + a.n_steps);
    }
}

template <int S, int SCHEME, bool STASH>
__global__ void __launch_bounds__(kStepsThreads, STASH ? kStepsPerSm : 2) k_steps(const __grid_constant__ StepsArgs a) {
    __shared__ __align__(16) OwnTile own[kStepsTiles];
    extern __shared__ __align__(128) int32_t link_stash[];
    if (threadIdx.x == 0) s_wait_limit = a.wait_limit;
    __syncthreads();
    if ((int)blockIdx.x < a.n_site_blocks) site_block<S, SCHEME, STASH>(a, own, link_stash);
    else iolet_block(a, link_stash);
    // the last block to leave advances the step counters and clears the counters for the
    // next launch: every other block has read them for the last time
    __syncthreads();
    if (threadIdx.x == 0) {
        fence_gpu();
        if (atomicAdd(&a.sync->left, 1u) == gridDim.x - 1) {
            fence_gpu();
            for (int i = 0; i < a.n_doms; ++i) *const_cast<int64_t *>(a.doms[i].D.step) += a.n_steps;
            for (unsigned &d : a.sync->done) d = 0;
            a.sync->arrived = 0;
            a.sync->values = 0;
            a.sync->ready = 0;
            a.sync->left = 0;
        }
    }
}

template <bool STASH> cudaError_t blocks_per_sm(int threads, size_t smem, int *out) {
    auto k = k_steps<HG_PART_S, HG_PART_SCHEME, STASH>;
    // one allowance for every shape: sets of several shapes may be stepped in turn
    cudaError_t e = cudaSuccess;
    if (STASH) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kStepsSmem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k, threads, smem);
    return e;
}

}  // namespace

template <>
cudaError_t steps_blocks_per_sm<HG_PART_S, HG_PART_SCHEME>(bool stash, int threads, size_t smem, int *out) {
    return stash ? blocks_per_sm<true>(threads, smem, out) : blocks_per_sm<false>(threads, smem, out);
}

template <>
cudaError_t launch_steps<HG_PART_S, HG_PART_SCHEME>(const StepsArgs &a, const StepsShape &sh, cudaStream_t st) {
    StepsArgs arg = a;
    void *args[] = {&arg};
    const void *k = sh.stash ? (const void *)k_steps<HG_PART_S, HG_PART_SCHEME, true>
                             : (const void *)k_steps<HG_PART_S, HG_PART_SCHEME, false>;
    return cudaLaunchCooperativeKernel(k, dim3((unsigned)sh.grid), dim3((unsigned)sh.threads), args, sh.smem, st);
}

}  // namespace hg
