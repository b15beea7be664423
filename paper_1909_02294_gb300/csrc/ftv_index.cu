// Data preparation kernels: texel packing, the per-reference segment index, the work plan of the persistent
// cost kernel and the tile records it reads.
//
// Paper: segments are the estimation units (Sec. III-A: "depth is estimated for segments"; Sec. IV-C:
// segments come from any superpixel method, one label map per view). The index groups each
// reference's pixels by segment so that a cost tile reads consecutive pixels of few segments.
// Every stage takes all views or references of a call in one launch: they are short kernels, and one after
// the other per view they cost more in launches and idle SMs than in work (8 references at 1920x1080: the
// index alone 380 us in 24 launches).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "ftv_internal.h"
#include "ftv_strip.cuh"

namespace ftv {
namespace {

constexpr unsigned kFull = 0xffffffffu;

// ------------------------------------------------------------------------------------------ packing

struct PackArgs {
    PackView v[FTV_MAX_VIEWS];
};

// Four adjacent pixels of a row per thread; blockIdx.y is the row, blockIdx.z the view. Samples above max_value
// are reported and clamped so that they cannot spill into a neighbouring packed field. Memory-bound; a thread's
// four samples of a plane come in one load and leave as one 16-byte store (or two) where the pointers, the
// pitches and the width allow (every pixel of such a view then has 4-aligned company).
template <int SB, int FMT>
__global__ void __launch_bounds__(128) pack_kernel(const __grid_constant__ PackArgs args, uint32_t max_value,
                                                   uint32_t* status) {
    const PackView& V = args.v[blockIdx.z];
    const int x = (blockIdx.x * blockDim.x + threadIdx.x) * 4, y = blockIdx.y;
    if (x >= V.W || y >= V.H) return;
    const int n = min(4, V.W - x);
    const bool vec = V.vec != 0;  // then W is a multiple of 4
    uint32_t s[3][4];
#pragma unroll
    for (int c = 0; c < 3; ++c)
        load4<SB>(static_cast<const char*>(V.planes[c]) + (int64_t)y * V.pitch[c] + (int64_t)x * SB, n, vec, s[c]);
    if (clamp4(s, max_value)) atomicOr(status, ST_BAD_SAMPLE);
    store4<FMT>(V.out, (int64_t)y * V.W + x, n, vec, s);
}

// ------------------------------------------------------------------------------------ segment index

struct IndexArgs {
    IndexRef r[FTV_MAX_VIEWS];
};

// Four adjacent labels of a row (-1 past its end), in one load where the map allows.
__device__ __forceinline__ void load_labels(const IndexRef& R, int x, int y, int* l) {
    const int32_t* p = R.labels + (int64_t)y * R.W + x;
    if (R.vec && x + 4 <= R.W) {
        const int4 t = __ldg(reinterpret_cast<const int4*>(p));
        l[0] = t.x;
        l[1] = t.y;
        l[2] = t.z;
        l[3] = t.w;
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) l[k] = x + k < R.W ? __ldg(p + k) : -1;
    }
}

// Per-segment pixel counts (blockIdx.z: the reference): one addition per run of equal labels among the 128 adjacent
// pixels of a warp, four to a thread. A thread that starts a run counts the threads it goes on through from two ballots:
// those whose pixels all continue it, and the first one that continues it only in part.
// Runs joined within a thread only took one addition per four pixels of a large segment, all at a few addresses: three
// 961x541 maps of 8 segments each 223 us, this 12; of 60 px segments 8, of 10 px ones 5.
__global__ void __launch_bounds__(128) histogram_kernel(const __grid_constant__ IndexArgs args, uint32_t* status) {
    const IndexRef& R = args.r[blockIdx.z];
    const int x = (blockIdx.x * blockDim.x + threadIdx.x) * 4, y = blockIdx.y, lane = threadIdx.x & 31;
    if (y >= R.H || x - 4 * lane >= R.W) return;  // uniform over the warp
    int l[4] = {-1, -1, -1, -1};
    if (x < R.W) load_labels(R, x, y, l);
    bool bad = false;
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if ((unsigned)l[k] >= (unsigned)R.S) {
            bad = bad || x + k < R.W;
            l[k] = -1;
        }
    if (bad) atomicOr(status, ST_BAD_LABEL);
    const int lead = l[0] != l[1] ? 1 : l[0] != l[2] ? 2 : l[0] != l[3] ? 3 : 4;  // pixels of the thread's first run
    const int left = __shfl_up_sync(kFull, l[3], 1);
    const bool cont = lane > 0 && l[0] == left;  // the first run is the left thread's last one going on
    const unsigned conts = __ballot_sync(kFull, cont), whole = __ballot_sync(kFull, cont && lead == 4);
    const unsigned ends = ~whole & (kFull << lane << 1);  // the threads after this one that a run does not fill
    const int end = ends ? __ffs(ends) - 1 : 32;
    const int part = __shfl_sync(kFull, lead, end & 31);
    const int more = 4 * (end - 1 - lane) + (end < 32 && (conts >> end & 1u) ? part : 0);
    int n = 0;
    bool mine = !cont;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        ++n;
        if (k == 3 || l[k + 1 < 4 ? k + 1 : k] != l[k]) {
            if (mine && l[k] >= 0) atomicAdd(&R.counts[l[k]], k == 3 ? n + more : n);
            n = 0;
            mine = true;
        }
    }
}

// Exclusive prefix of n counts by blocks of 1024, each of kScanChunk counts (eight consecutive ones per thread, read and
// written coalesced through shared memory): block b adds up the counts of the blocks before it (independent loads),
// then scans its own. out, and out2 where it is given, receive the prefix, *total (by the last block) the sum.
// One block walking the counts took 25 us for 20736 segments one stretch per thread, 9 us chunk by chunk; this 5.
constexpr int kScanPer = 8, kScanChunk = 1024 * kScanPer;
__device__ void scan_counts(const int32_t* __restrict__ in, int n, int32_t* out, int32_t* out2, int32_t* total, int* mx) {
    __shared__ int sm[kScanChunk + kScanChunk / 32];
    __shared__ int s_before;
    auto at = [](int i) { return i + (i >> 5); };  // padded against bank conflicts
    const int b = blockIdx.x * kScanChunk;
    if (b >= n && b > 0) return;  // uniform: past this reference's counts
    if (threadIdx.x == 0) s_before = 0;
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        const int i = k * 1024 + threadIdx.x;
        sm[at(i)] = b + i < n ? in[b + i] : 0;
    }
    int before = 0;
#pragma unroll 8
    for (int i = threadIdx.x; i < b; i += 1024) before += in[i];
    before = __reduce_add_sync(kFull, before);
    __syncthreads();
    if ((threadIdx.x & 31) == 0 && before) atomicAdd(&s_before, before);
    int c[kScanPer], sum = 0;
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        c[k] = sm[at(threadIdx.x * kScanPer + k)];
        sum += c[k];
        *mx = max(*mx, c[k]);
    }
    int all;
    int p = block_exclusive_scan(sum, &all);
    p += s_before;  // a statement of its own: the scan's barriers come between the additions to s_before and this read
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        sm[at(threadIdx.x * kScanPer + k)] = p;
        p += c[k];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        const int i = k * 1024 + threadIdx.x;
        if (b + i < n) {
            out[b + i] = sm[at(i)];
            if (out2) out2[b + i] = sm[at(i)];
        }
    }
    if (b + kScanChunk >= n && threadIdx.x == 0) *total = s_before + all;
}

// Counts -> offsets[S + 1]; cursor[s] = offsets[s] for the scatter. Also checks that no segment is large enough for its
// int32 cost sum to overflow.
__global__ void __launch_bounds__(1024) offsets_kernel(const __grid_constant__ IndexArgs args, uint32_t* status) {
    const IndexRef& R = args.r[blockIdx.y];
    int mx = 0;
    scan_counts(R.counts, R.S, R.offs, R.cursor, R.offs + R.S, &mx);
    mx = __reduce_max_sync(kFull, mx);
    if ((threadIdx.x & 31) == 0 && (int64_t)mx * R.max_pix_cost > (int64_t)INT32_MAX) atomicOr(status, ST_OVERFLOW);
}

__global__ void __launch_bounds__(1024) prefix_kernel(const int32_t* counts, int n, int32_t* offs, int32_t* total) {
    int mx = 0;
    scan_counts(counts, n, offs, nullptr, total, &mx);
}

// Scatter (y << 16 | x) records into their segment's range. A warp's run of equal labels takes one atomic and keeps
// its left-to-right order (the cost kernel's gathers follow this order: one atomic per run of a thread's four pixels
// made it 3 % slower on the 1920x1080 rig). kScatterRows rows per warp, their atomics in flight together.
constexpr int kScatterRows = 4;
__global__ void __launch_bounds__(256) scatter_kernel(const __grid_constant__ IndexArgs args) {
    const IndexRef& R = args.r[blockIdx.z];
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y0 = blockIdx.y * kScatterRows;
    if (y0 >= R.H) return;
    const int lane = threadIdx.x & 31;
    int l[kScatterRows], at[kScatterRows];
    unsigned peers[kScatterRows];
#pragma unroll
    for (int r = 0; r < kScatterRows; ++r) l[r] = x < R.W && y0 + r < R.H ? __ldg(&R.labels[(int64_t)(y0 + r) * R.W + x]) : -1;
#pragma unroll
    for (int r = 0; r < kScatterRows; ++r) {
        if ((unsigned)l[r] >= (unsigned)R.S) l[r] = -1;
        peers[r] = __match_any_sync(kFull, l[r]);
        at[r] = 0;
        if (l[r] >= 0 && lane == __ffs(peers[r]) - 1) at[r] = atomicAdd(&R.cursor[l[r]], __popc(peers[r]));
    }
#pragma unroll
    for (int r = 0; r < kScatterRows; ++r) {
        const int base = __shfl_sync(kFull, at[r], __ffs(peers[r]) - 1);
        if (l[r] >= 0) R.pix[base + __popc(peers[r] & ((1u << lane) - 1u))] = ((uint32_t)(y0 + r) << 16) | (uint32_t)x;
    }
}

// ---------------------------------------------------------------------------------------------- plan

template <int CAP>
struct PlanArgs {
    RefJob jobs[CAP];
};

// An item's fixed work (staging, pixel loads, barriers) in staged entries: between fits to label-block sweeps on the
// 1920x1080 8-view rig (9.6) and a 957x541 one with two neighbours (4.3). Against 8, a value of 4 makes the latter 2 %
// faster (975 -> 956 us) and a 960x540 frame of few changed segments 4 % slower (156 -> 161), 12 changes nothing.
constexpr int kItemOverhead = 8;
constexpr int kMaxSplit = 16;

// Completes the plan of one launch. Block u computes unit u's listed pixel prefix (woffs) and pixel count; the
// last block to finish chooses the label blocks and gives every unit its first tile and item.
// Label blocks: an item is one tile times LB labels. The host's LB is the largest the stage holds, right for
// launches of many waves; a launch of few tiles would leave most CTAs idle (a 480x270 frame has 127 tiles for 608
// CTAs), so the blocks are split f-fold, f minimising the modelled time (items' work and fixed overhead spread
// over the CTAs, plus three quarters of the largest item for the last wave). 480x270 with 64 labels and 2
// neighbours: 151 us at f = 1, 51 us at f = 4 to 8.
__device__ void plan_block(const RefJob& J, RefJob* out, int u, int n_jobs, int slots, Plan* plan) {
    if (u < n_jobs) {
        int n_work = J.S;
        if (J.list != nullptr) n_work = min(max(*J.n_listed, 0), J.S);
        int n_rec;
        if (J.list == nullptr) {
            n_rec = J.offs[J.S];
        } else {
            // A strictly increasing list (every changed list is) names each segment once. Another one is checked
            // for repeats: a repeated segment's pixels belong to its first entry, the others have none.
            bool mine = false;
            for (int i = threadIdx.x; i + 1 < n_work; i += 1024) mine = mine || J.list[i] >= J.list[i + 1];
            const bool repeats = __syncthreads_or(mine);
            if (repeats) {
                for (int s = threadIdx.x; s < J.S; s += 1024) J.first[s] = INT32_MAX;
                __syncthreads();
                for (int i = threadIdx.x; i < n_work; i += 1024)
                    if ((unsigned)J.list[i] < (unsigned)J.S) atomicMin(&J.first[J.list[i]], i);
                __syncthreads();
            }
            int run = 0;
            for (int b = 0; b < n_work; b += 1024) {
                const int i = b + threadIdx.x;
                int c = 0;
                if (i < n_work) {
                    const int s = J.list[i];
                    if ((unsigned)s < (unsigned)J.S && (!repeats || J.first[s] == i)) c = J.offs[s + 1] - J.offs[s];
                }
                int total;
                const int at = run + block_exclusive_scan(c, &total);
                if (i < n_work) J.woffs[i] = at;
                run += total;
            }
            if (threadIdx.x == 0) J.woffs[n_work] = run;
            n_rec = run;
        }
        if (threadIdx.x == 0) {
            RefJob o = J;
            if (o.list == nullptr) o.woffs = const_cast<int32_t*>(o.offs);
            o.n_work = n_work;
            o.n_rec = n_rec;
            out[u] = o;
        }
    }
    __shared__ int s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(&plan->ticket, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const volatile RefJob* units = out;
    __shared__ float s_time[kMaxSplit];
    if (threadIdx.x < kMaxSplit) {
        const int f = threadIdx.x + 1;
        float work = 0.0f, top = 0.0f;
        for (int k = 0; k < n_jobs; ++k) {
            const int tiles = (units[k].n_rec + kTile - 1) / kTile, L = units[k].L;
            const int n = (L * f + units[k].LB - 1) / units[k].LB, lb = (L + n - 1) / n;
            const float w = (float)(max(1, units[k].N) * lb + kItemOverhead);
            work += (float)tiles * (float)((L + lb - 1) / lb) * w;
            if (tiles > 0) top = fmaxf(top, w);
        }
        s_time[threadIdx.x] = work / (float)slots + 0.75f * top;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int f = 1;
        for (int k = 2; k <= kMaxSplit; ++k)
            if (s_time[k - 1] < s_time[f - 1]) f = k;
        int items = 0, base = 0;
        for (int k = 0; k < n_jobs; ++k) {
            RefJob& o = out[k];
            const int tiles = (units[k].n_rec + kTile - 1) / kTile, L = units[k].L;
            const int n = (L * f + units[k].LB - 1) / units[k].LB;
            o.LB = (L + n - 1) / n;
            o.nLB = (L + o.LB - 1) / o.LB;
            o.item_base = items;
            o.tile_base = base;
            items += tiles * o.nLB;
            base += max(1, tiles);  // a unit without pixels has one tile, which clears its rows
        }
        plan->total_items = items;
        plan->total_tiles = base;
        for (int k = 0; k < kMaxChunks; ++k) plan->counter[k] = 0;
        plan->n_jobs = n_jobs;
        plan->culled = 0;
        plan->skipped = 0;
        plan->recomputed = 0;
        plan->checked = 0;
        plan->ticket = 0;
    }
}

// One block of 1024 threads per unit; descriptors arrive as kernel parameters and are written, completed, to `out`.
template <int CAP>
__global__ void __launch_bounds__(1024) plan_kernel(const __grid_constant__ PlanArgs<CAP> args, int n_jobs, int slots,
                                                    RefJob* out, Plan* plan) {
    plan_block(args.jobs[blockIdx.x], out, blockIdx.x, n_jobs, slots, plan);
}

// Descriptors already in device memory are completed in place; blocks past the launch's units only take part in
// the count.
__global__ void __launch_bounds__(1024) plan_device_kernel(RefJob* jobs, const int32_t* n_jobs_ptr, int slots, Plan* plan) {
    const RefJob J = jobs[blockIdx.x];
    __syncthreads();
    plan_block(J, jobs, blockIdx.x, *n_jobs_ptr, slots, plan);
}

// Largest k in [lo, hi) with a[k] <= w (a nondecreasing, a[lo] <= w).
__device__ __forceinline__ int upper_index(const int32_t* a, int lo, int hi, int w) {
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (a[mid] <= w) lo = mid;
        else hi = mid;
    }
    return lo;
}

// Warp-cooperative version (all 32 lanes call it): 32 probes per round narrow the range ~33-fold, so a
// search over n entries takes about log33(n) dependent loads instead of log2(n).
__device__ __forceinline__ int warp_upper_index(const int32_t* a, int lo, int hi, int w) {
    const int lane = threadIdx.x & 31;
    while (hi - lo > 32) {
        const int64_t span = hi - lo;
        const bool le = a[lo + (int)(span * (lane + 1) / 33)] <= w;
        const int cnt = __popc(__ballot_sync(kFull, le));  // the true probes are a prefix
        const int nlo = cnt ? lo + (int)(span * cnt / 33) : lo;
        const int nhi = cnt < 32 ? lo + (int)(span * (cnt + 1) / 33) : hi;
        lo = nlo;
        hi = nhi;
    }
    const int p = lo + lane;
    const unsigned m = __ballot_sync(kFull, p < hi && a[p] <= w);
    return lo + 31 - __clz(m);
}

constexpr int kTileThreads = 256;
constexpr int kLocCache = 1025;  // segments of a tile whose offsets are cached (more: search in global memory)

// The tile records of every unit, one CTA per tile (persistent over the launch's tiles): each listed pixel's
// position and segment, and per tile its segments and pixel box, which the cost kernel would otherwise search for
// once per label block. Each tile also clears its share of the unit's cost rows (segments cut by a tile boundary
// are summed with atomics), in place of one clear per reference.
// The records stay in list order. Ordering a tile's pixels by 16- or 32-pixel wide blocks, so that a gather meets
// fewer rows, measured slower (1920x1080 rig 21.8 and 24.0 against 20.6 ms): a warp then meets more segments.
__global__ void __launch_bounds__(kTileThreads) tile_kernel(const RefJob* __restrict__ jobs, const Plan* __restrict__ plan) {
    __shared__ int sWoffs[kLocCache + 1], sFrom[kLocCache + 1];  // sFrom: list position - record position
    __shared__ int s_k0, s_k1, s_box[4];
    const int tid = threadIdx.x, lane = tid & 31;
    const int total = plan->total_tiles, n_jobs = plan->n_jobs;
    for (int t = blockIdx.x; t < total; t += gridDim.x) {
        int lo = 0, hi = n_jobs - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (__ldg(&jobs[mid].tile_base) <= t) lo = mid;
            else hi = mid - 1;
        }
        const RefJob& J = jobs[lo];
        const int tile = t - J.tile_base, n_work = J.n_work, n_rec = J.n_rec, L = J.L;
        const int tiles = max(1, (n_rec + kTile - 1) / kTile);
        const int32_t* __restrict__ list = J.list;
        const int32_t* __restrict__ woffs = J.woffs;
        {  // this tile's share of the cost rows to clear
            if (list == nullptr) {
                const int64_t words = (int64_t)n_work * L, b = words * tile / tiles, e = words * (tile + 1) / tiles;
                const bool vec = (reinterpret_cast<uintptr_t>(J.cost) & 15) == 0;
                const int64_t vb = vec ? (b + 3) / 4 : 0, ve = vec ? e / 4 : 0;
                if (vec && vb < ve) {
                    for (int64_t i = vb + tid; i < ve; i += kTileThreads)
                        reinterpret_cast<int4*>(J.cost)[i] = make_int4(0, 0, 0, 0);
                    for (int64_t i = b + tid; i < vb * 4; i += kTileThreads) J.cost[i] = 0;
                    for (int64_t i = ve * 4 + tid; i < e; i += kTileThreads) J.cost[i] = 0;
                } else {
                    for (int64_t i = b + tid; i < e; i += kTileThreads) J.cost[i] = 0;
                }
            } else {
                // whole rows, one per warp
                const int kb = (int)((int64_t)n_work * tile / tiles), ke = (int)((int64_t)n_work * (tile + 1) / tiles);
                for (int k = kb + (tid >> 5); k < ke; k += kTileThreads / 32) {
                    const int s = list[k];
                    if ((unsigned)s < (unsigned)J.S)
                        for (int d = lane; d < L; d += 32) J.cost[(int64_t)s * L + d] = 0;
                }
            }
        }
        const int w0 = tile * kTile, w1 = min(w0 + kTile, n_rec);
        if (w0 >= w1) continue;  // uniform: a unit without pixels
        if (tid < 32) {
            const int k = warp_upper_index(woffs, 0, n_work + 1, w0);
            if (lane == 0) s_k0 = k;
        } else if (tid < 64) {
            const int k = warp_upper_index(woffs, 0, n_work + 1, w1 - 1);
            if (lane == 0) s_k1 = k;
        }
        if (tid == 0) {
            s_box[0] = s_box[2] = INT32_MAX;
            s_box[1] = s_box[3] = -1;
        }
        __syncthreads();
        const int k0 = s_k0, k1 = s_k1, nk = k1 - k0 + 1;
        const bool cached = nk + 1 <= kLocCache;
        if (cached)
            for (int i = tid; i <= nk; i += kTileThreads) {
                const int at = woffs[k0 + i];
                sWoffs[i] = at;
                if (list != nullptr && i < nk) {
                    const int l = list[k0 + i];  // an entry outside the segments owns no pixels: its offset is not read
                    sFrom[i] = (unsigned)l < (unsigned)J.S ? J.offs[l] - at : 0;
                }
            }
        __syncthreads();
        int x0 = INT32_MAX, x1 = -1, y0 = INT32_MAX, y1 = -1;
#pragma unroll
        for (int j = 0; j < kTile / kTileThreads; ++j) {
            const int w = w0 + j * kTileThreads + tid;
            if (w < w1) {
                const int k = cached ? k0 + upper_index(sWoffs, 0, nk + 1, w) : upper_index(woffs, k0, k1 + 1, w);
                int i = w;
                if (list != nullptr) i = cached ? w + sFrom[k - k0] : J.offs[list[k]] + (w - woffs[k]);
                const uint32_t xy = J.pix[i];
                J.recs[w] = make_int2((int)xy, k);
                const int x = xy & 0xffff, y = xy >> 16;
                x0 = min(x0, x);
                x1 = max(x1, x);
                y0 = min(y0, y);
                y1 = max(y1, y);
            }
        }
        x0 = __reduce_min_sync(kFull, x0);
        x1 = __reduce_max_sync(kFull, x1);
        y0 = __reduce_min_sync(kFull, y0);
        y1 = __reduce_max_sync(kFull, y1);
        if (lane == 0) {
            atomicMin(&s_box[0], x0);
            atomicMax(&s_box[1], x1);
            atomicMin(&s_box[2], y0);
            atomicMax(&s_box[3], y1);
        }
        __syncthreads();
        if (tid == 0) J.tiles[tile] = make_int4(k0, k1, s_box[0] | (s_box[1] << 16), s_box[2] | (s_box[3] << 16));
        __syncthreads();  // the shared arrays are reused by the next tile
    }
}

}  // namespace

cudaError_t launch_pack(const PackView* views, int n, int sample_bytes, int bit_depth, int fmt, uint32_t* status,
                        cudaStream_t s, int64_t* launches) {
    if (n <= 0) return cudaSuccess;
    if (n > FTV_MAX_VIEWS) return cudaErrorInvalidValue;
    PackArgs args;
    int W = 0, H = 0;
    for (int k = 0; k < n; ++k) {
        PackView v = views[k];
        uintptr_t a = reinterpret_cast<uintptr_t>(v.out) & 15;
        for (int c = 0; c < 3; ++c)
            a |= (reinterpret_cast<uintptr_t>(v.planes[c]) | (uintptr_t)v.pitch[c]) & (uintptr_t)(4 * sample_bytes - 1);
        v.vec = a == 0 && v.W % 4 == 0;
        args.v[k] = v;
        W = std::max(W, v.W);
        H = std::max(H, v.H);
    }
    if (W <= 0 || H <= 0) return cudaSuccess;
    const dim3 block(128), grid((W + 511) / 512, H, n);
    const uint32_t maxv = (1u << bit_depth) - 1u;
    if (sample_bytes == 1) pack_kernel<1, FMT_U8X4><<<grid, block, 0, s>>>(args, maxv, status);
    else if (fmt == FMT_P10) pack_kernel<2, FMT_P10><<<grid, block, 0, s>>>(args, maxv, status);
    else if (fmt == FMT_U16S) pack_kernel<2, FMT_U16S><<<grid, block, 0, s>>>(args, maxv, status);
    else pack_kernel<2, FMT_U16X4><<<grid, block, 0, s>>>(args, maxv, status);
    *launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_segment_index(const IndexRef* refs, int n, uint32_t* status, cudaStream_t s, int64_t* launches) {
    if (n <= 0) return cudaSuccess;
    if (n > FTV_MAX_VIEWS) return cudaErrorInvalidValue;
    IndexArgs args;
    int W = 1, H = 1, S = 1;
    for (int k = 0; k < n; ++k) {
        args.r[k] = refs[k];
        args.r[k].vec = (reinterpret_cast<uintptr_t>(refs[k].labels) & 15) == 0 && refs[k].W % 4 == 0;
        W = std::max(W, refs[k].W);
        H = std::max(H, refs[k].H);
        S = std::max(S, refs[k].S);
        // the references' counts lie one after the other: one clear for a run of them
        if (k == 0 || refs[k].counts != refs[k - 1].counts + refs[k - 1].stride) {
            size_t words = refs[k].S > 0 ? refs[k].S : 1;
            for (int j = k + 1; j < n && refs[j].counts == refs[j - 1].counts + refs[j - 1].stride; ++j)
                words = (size_t)(refs[j].counts - refs[k].counts) + refs[j].S;
            const cudaError_t e = cudaMemsetAsync(refs[k].counts, 0, sizeof(int32_t) * words, s);
            if (e != cudaSuccess) return e;
        }
    }
    const dim3 block(128), grid((W + 511) / 512, H, n);
    histogram_kernel<<<grid, block, 0, s>>>(args, status);
    offsets_kernel<<<dim3((S + kScanChunk - 1) / kScanChunk, n), 1024, 0, s>>>(args, status);
    scatter_kernel<<<dim3((W + 255) / 256, (H + kScatterRows - 1) / kScatterRows, n), 256, 0, s>>>(args);
    *launches += 3;
    return cudaGetLastError();
}

template <int CAP>
static cudaError_t launch_plan_cap(const RefJob* host_jobs, int n_jobs, int slots, RefJob* d_jobs, Plan* plan,
                                   cudaStream_t s) {
    static_assert(sizeof(PlanArgs<CAP>) + 64 <= 32764, "kernel parameter space");
    PlanArgs<CAP> args;
    for (int j = 0; j < n_jobs; ++j) args.jobs[j] = host_jobs[j];
    plan_kernel<CAP><<<std::max(1, n_jobs), 1024, 0, s>>>(args, n_jobs, slots, d_jobs, plan);
    return cudaGetLastError();
}

cudaError_t launch_plan_device(RefJob* d_jobs, const int32_t* n_jobs, int max_jobs, int slots, Plan* plan,
                               cudaStream_t s) {
    plan_device_kernel<<<std::max(1, max_jobs), 1024, 0, s>>>(d_jobs, n_jobs, slots, plan);
    return cudaGetLastError();
}

cudaError_t launch_plan(const RefJob* host_jobs, int n_jobs, int slots, RefJob* d_jobs, Plan* plan, cudaStream_t s) {
    if (n_jobs < 0 || n_jobs > FTV_MAX_VIEWS) return cudaErrorInvalidValue;  // one unit per reference
    if (n_jobs <= 16) return launch_plan_cap<16>(host_jobs, n_jobs, slots, d_jobs, plan, s);
    return launch_plan_cap<FTV_MAX_VIEWS>(host_jobs, n_jobs, slots, d_jobs, plan, s);
}

cudaError_t launch_prefix(const int32_t* counts, int n, int32_t* offs, int32_t* total, cudaStream_t s) {
    prefix_kernel<<<std::max(1, (n + kScanChunk - 1) / kScanChunk), 1024, 0, s>>>(counts, n, offs, total);
    return cudaGetLastError();
}

cudaError_t launch_tiles(const RefJob* jobs, const Plan* plan, int grid, cudaStream_t s) {
    tile_kernel<<<std::max(1, grid), kTileThreads, 0, s>>>(jobs, plan);
    return cudaGetLastError();
}

}  // namespace ftv
