// Temporal consistency test, winner-take-all readout and per-pixel depth maps.
//
// Paper, Sec. III-E: a segment is left out of the new estimate when every component of its mean
// (Y, Cb, Cr) vector changed by less than T_P against the collocated segment of the previous P frame,
// or by less than T_I against the I frame; it then adopts that frame's depth. With the segment's
// pixel set fixed by the current label map, n pixels and channel sums S, "mean changed by less than
// T" is |S_cur - S_ref| < T * n, which the kernels below evaluate exactly in 64-bit integers.
// The winner-take-all readout stands in for the paper's graph-cut optimisation (Sec. IV-B), which is
// not part of this library: it returns the label of least cost per segment.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <climits>

#include "ftv_internal.h"
#include "ftv_strip.cuh"

namespace ftv {
namespace {

constexpr unsigned kFull = 0xffffffffu;

template <int SB>
__device__ __forceinline__ int load_sample(const char* p) {
    if (SB == 1) return __ldg(reinterpret_cast<const uint8_t*>(p));
    return __ldg(reinterpret_cast<const uint16_t*>(p));
}

__device__ __forceinline__ void add64(int64_t* dst, int v) {
    atomicAdd(reinterpret_cast<unsigned long long*>(dst), (unsigned long long)(long long)v);
}

// Per-segment sums over a tile of kAccCols x kAccRowsTile pixels per CTA: each thread walks a strip of four adjacent
// columns down kAccRows rows. A row of the strip meets at most two segments almost always (segments are many pixels
// wide): the pixels that share the first one's label form part A, the others part B, and each part's sum over the
// strip's row is a pair of dot products of the packed samples with the part's 0/1 weights per plane. Parts of equal
// label in successive rows are summed in registers; a finished run is added to the CTA's bins in shared memory,
// indexed by label - (the tile's least label); labels beyond kBins of it go to global memory directly. A row whose
// B pixels differ in label adds them one by one. At the end each non-empty bin is added to the segment's 64-bit sums,
// once per tile. All sums are exact integers, so the order of the additions does not change the result. Tile bins are
// 32-bit: a tile has 1024 pixels of differences below 2^16.
// Segments of fewer than three pixels on average take the columns of a strip 32 apart (STEP): nearly every pixel is a run
// of its own then and goes to global memory, where a warp's additions of four columns each touch four times the
// sectors. Four 960x540 references of one-pixel segments: adjacent columns 129 us, 32 apart 105; of 2 x 2 pixel ones 98
// and 106 (L2 flushed).
// Single columns took 61 instructions per pixel and 127 us for eight 1920x1080 references; the strips take 72, of which
// the bytes need 54. Two rows per thread and six CTAs per SM: the loads of a strip are all in flight at once, so that
// more rows cost warps (four rows 107 us; four CTAs 80, eight 76; all measured on three planes with an I frame. Luma
// alone gains little: eight 1920x1080 references with an I frame and a flushed L2 135 -> 131 us).
constexpr int kAccCols = 128;      // pixels per tile row
constexpr int kStrips = kAccCols / 4;
constexpr int kAccRows = 2;        // rows per thread
constexpr int kAccRowsTile = 8;    // rows per tile
constexpr int kAccThreads = kStrips * (kAccRowsTile / kAccRows);
constexpr int kBins = 512;
static_assert(kAccThreads == 128, "one CTA of 128 threads per tile");

// The references of one launch (kernel parameters, read in place).
struct TemporalRefs {
    TemporalRef r[kMaxTemporalRefs];
};

// Four samples of a row, STEP columns apart, packed in 16-bit lanes; n of them lie in the view (the rest repeat the last).
template <int SB, bool VEC, int STEP>
__device__ __forceinline__ uint2 load_strip(const char* p, int n) {
    if constexpr (VEC && SB == 2) {
        return __ldg(reinterpret_cast<const uint2*>(p));
    } else if constexpr (VEC) {
        const uint32_t t = __ldg(reinterpret_cast<const uint32_t*>(p));
        return make_uint2(__byte_perm(t, 0, 0x4140), __byte_perm(t, 0, 0x4342));
    } else {
        uint32_t v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = (uint32_t)load_sample<SB>(p + (int64_t)min(k, n - 1) * (STEP * SB));
        return make_uint2(v[0] | (v[1] << 16), v[2] | (v[3] << 16));
    }
}

// c + the sum of the four samples times the weights (bytes 0/1 of the pixels, or their negatives).
__device__ __forceinline__ int strip_dot(const uint2& v, uint32_t weights, int c) {
    int d;
    asm("dp2a.lo.u32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(v.x), "r"(weights), "r"(c));
    asm("dp2a.hi.u32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(v.y), "r"(weights), "r"(d));
    return d;
}

template <int SB, int NCH, bool HAS_I, bool VEC, int STEP>
__global__ void __launch_bounds__(kAccThreads, 6) temporal_accumulate_kernel(const __grid_constant__ TemporalRefs p,
                                                                          uint32_t* status) {
    constexpr int Q = 1 + NCH * (HAS_I ? 2 : 1);  // per segment: n, dP[NCH], dI[NCH]
    __shared__ __align__(16) int bins[Q][kBins];
    __shared__ int s_base, s_top;
    const TemporalRef& f = p.r[blockIdx.z];  // blockIdx.z: the reference
    const int W = f.W, H = f.H, S = f.S;
    if ((int)blockIdx.x * kAccCols >= W || (int)blockIdx.y * kAccRowsTile >= H) return;  // past this view
    int64_t* __restrict__ stats = f.stats;
    const int tid = threadIdx.x;
    const int x = blockIdx.x * kAccCols + tid % kStrips * (STEP == 1 ? 4 : 1);  // columns x, x + STEP, ..
    const int y0 = blockIdx.y * kAccRowsTile + (tid / kStrips) * kAccRows;
    // Positions past the view's edge are clamped into it, so the loads need no branch, and those pixels are then
    // dropped through their label.
    // A vector load's strip is clamped as a whole: W is then a multiple of four.
    const int xc = VEC ? min(x, W - 4) : min(x, W - 1), nx = min(4, (W - xc + STEP - 1) / STEP), yc0 = min(y0, H - 1);
    int lab[kAccRows][4];
    uint2 a[kAccRows][NCH], b[kAccRows][NCH], e[kAccRows][HAS_I ? NCH : 1];
#pragma unroll
    for (int r = 0; r < kAccRows; ++r) {
        const int64_t y = min(yc0 + r, H - 1);
        const int32_t* pl = f.labels + y * W + xc;
        if (VEC) {
            const int4 t = __ldg(reinterpret_cast<const int4*>(pl));
            lab[r][0] = t.x;
            lab[r][1] = t.y;
            lab[r][2] = t.z;
            lab[r][3] = t.w;
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) lab[r][k] = __ldg(pl + min(k, nx - 1) * STEP);
        }
#pragma unroll
        for (int c = 0; c < NCH; ++c) {
            a[r][c] = load_strip<SB, VEC, STEP>(static_cast<const char*>(f.cur[c]) + y * f.pc[c] + (int64_t)xc * SB, nx);
            b[r][c] = load_strip<SB, VEC, STEP>(static_cast<const char*>(f.prev[c]) + y * f.pp[c] + (int64_t)xc * SB, nx);
            if (HAS_I) e[r][c] = load_strip<SB, VEC, STEP>(static_cast<const char*>(f.ifr[c]) + y * f.pi[c] + (int64_t)xc * SB, nx);
        }
    }
    int lmin = INT_MAX, lmax = -1;
    bool bad = false;
#pragma unroll
    for (int r = 0; r < kAccRows; ++r)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const bool in = x + k * STEP < W && y0 + r < H;
            if (in && (unsigned)lab[r][k] < (unsigned)S) {
                lmin = min(lmin, lab[r][k]);
                lmax = max(lmax, lab[r][k]);
            } else {
                bad = bad || in;
                lab[r][k] = -1;
            }
        }
    if (bad) atomicOr(status, ST_BAD_LABEL);
    if (tid == 0) {
        s_base = INT_MAX;
        s_top = -1;
    }
    __syncthreads();
    lmin = __reduce_min_sync(kFull, lmin);
    lmax = __reduce_max_sync(kFull, lmax);
    if ((tid & 31) == 0 && lmax >= 0) {
        atomicMin(&s_base, lmin);
        atomicMax(&s_top, lmax);
    }
    __syncthreads();
    // the bins in use: the tile's labels from base to s_top (those beyond kBins go to global memory)
    const int base = s_base, used = min(kBins, s_top - base + 1);
    for (int i = tid; i < used; i += kAccThreads)
#pragma unroll
        for (int q = 0; q < Q; ++q) bins[q][i] = 0;
    __syncthreads();

    // word q of segment s: stats[q * ms + s] (q = 0: n, 1 + c: dP[c], 4 + c: dI[c])
    const int64_t ms = f.ms;
    {
        auto flush = [&](int l, int (&acc)[Q]) {
            if (l >= 0) {
                const unsigned bi = (unsigned)(l - base);
                if (bi < (unsigned)kBins) {
#pragma unroll
                    for (int q = 0; q < Q; ++q)
                        if (q == 0 || acc[q] != 0) atomicAdd(&bins[q][bi], acc[q]);
                } else {
                    add64(&stats[l], acc[0]);
#pragma unroll
                    for (int c = 0; c < NCH; ++c) {
                        add64(&stats[(1 + c) * ms + l], acc[1 + c]);
                        if (HAS_I) add64(&stats[(4 + c) * ms + l], acc[1 + NCH + c]);
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < Q; ++q) acc[q] = 0;
        };
        // adds the pixels of row r with the given 0/1 byte weights to a run of label l
        auto add = [&](int r, uint32_t w, int (&acc)[Q]) {
            const uint32_t neg = w * 255u;  // the weights' negatives
            acc[0] += __popc(w);
#pragma unroll
            for (int c = 0; c < NCH; ++c) {
                const int cur = strip_dot(a[r][c], w, 0);
                acc[1 + c] = strip_dot(b[r][c], neg, acc[1 + c] + cur);
                if (HAS_I) acc[1 + NCH + c] = strip_dot(e[r][c], neg, acc[1 + NCH + c] + cur);
            }
        };
        int la = -1, lb = -1, accA[Q], accB[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) accA[q] = accB[q] = 0;
#pragma unroll
        for (int r = 0; r < kAccRows; ++r) {
            // part A: the label of the first pixel; part B: that of the last one not in A
            const int l0 = lab[r][0];
            uint32_t wa = 0, wb = 0;
            int l1 = -1;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (lab[r][k] == l0) wa |= 1u << (8 * k);
                else l1 = lab[r][k];
            }
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (lab[r][k] == l1) wb |= 1u << (8 * k);
            if (l0 < 0) wa = 0;
            if (l1 < 0 || l1 == l0) wb = 0;
            if (l0 != la) {
                flush(la, accA);
                la = l0;
            }
            add(r, wa, accA);
            if (wb) {
                if (l1 != lb) {
                    flush(lb, accB);
                    lb = l1;
                }
                add(r, wb, accB);
            }
            // a third label (narrow segments): pixel by pixel
#pragma unroll
            for (int k = 1; k < 4; ++k)
                if (lab[r][k] >= 0 && !((wa | wb) >> (8 * k) & 1u)) {
                    int one[Q];
#pragma unroll
                    for (int q = 0; q < Q; ++q) one[q] = 0;
                    add(r, 1u << (8 * k), one);
                    flush(lab[r][k], one);
                }
        }
        flush(la, accA);
        flush(lb, accB);
    }
    __syncthreads();
    for (int i = tid; i < used; i += kAccThreads) {
        const int n = bins[0][i];
        if (n == 0) continue;
        const int64_t sg = base + i;
        add64(&stats[sg], n);
#pragma unroll
        for (int c = 0; c < NCH; ++c) {
            if (bins[1 + c][i] != 0) add64(&stats[(1 + c) * ms + sg], bins[1 + c][i]);
            if (HAS_I && bins[1 + NCH + c][i] != 0) add64(&stats[(4 + c) * ms + sg], bins[1 + NCH + c][i]);
        }
    }
}

__device__ __forceinline__ int64_t abs64(int64_t v) { return v < 0 ? -v : v; }

// The masks and the ordered list of changed segments, in two passes over blocks of kChunk segments.
// decide: one thread per segment reads its sums (one word from each plane in use, coalesced over the block),
// sets its mask and clears those words, so that the next call needs no clearing pass; each block's count of
// changed segments goes to plane 7 at the block's index. compact: each block adds up the counts of the
// blocks before it, scans its own changed flags and writes their positions; the last block writes the total.
constexpr int kChunk = 256;

// blockIdx.y: the reference; blocks past its segments return.
template <int NCH, bool HAS_I>
__global__ void __launch_bounds__(kChunk) temporal_decide_kernel(const __grid_constant__ TemporalRefs p, int t_p,
                                                                 int t_i) {
    const TemporalRef& R = p.r[blockIdx.y];
    const int S = R.S;
    if ((int)blockIdx.x * kChunk >= S) return;
    int64_t* __restrict__ stats = R.stats;
    const int64_t ms = R.ms;
    const int s = blockIdx.x * kChunk + threadIdx.x;
    int m = FTV_MASK_CHANGED;
    if (s < S) {
        int64_t dp[NCH], di[HAS_I ? NCH : 1];
        const int64_t n = stats[s];
#pragma unroll
        for (int c = 0; c < NCH; ++c) {
            dp[c] = stats[(1 + c) * ms + s];
            if (HAS_I) di[c] = stats[(4 + c) * ms + s];
        }
        if (n > 0) {
            bool okp = true, oki = HAS_I;
#pragma unroll
            for (int c = 0; c < NCH; ++c) {
                okp = okp && abs64(dp[c]) < (int64_t)t_p * n;
                if (HAS_I) oki = oki && abs64(di[c]) < (int64_t)t_i * n;
            }
            m = okp ? FTV_MASK_REUSE_P : (oki ? FTV_MASK_REUSE_I : FTV_MASK_CHANGED);
        }
        R.mask[s] = (uint8_t)m;
        // leave the sums zero for the next call
        stats[s] = 0;
#pragma unroll
        for (int c = 0; c < NCH; ++c) {
            stats[(1 + c) * ms + s] = 0;
            if (HAS_I) stats[(4 + c) * ms + s] = 0;
        }
    }
    const int cnt = __syncthreads_count(s < S && m == FTV_MASK_CHANGED);
    if (threadIdx.x == 0) stats[7 * ms + blockIdx.x] = cnt;
}

// blockIdx.y: the reference; blocks past its chunks return (a reference without segments has one chunk).
__global__ void __launch_bounds__(kChunk) temporal_compact_kernel(const __grid_constant__ TemporalRefs p) {
    __shared__ int s_base;
    const TemporalRef& R = p.r[blockIdx.y];
    const int S = R.S, chunks = S > 0 ? (S + kChunk - 1) / kChunk : 1;
    if ((int)blockIdx.x >= chunks) return;
    const int64_t* __restrict__ counts = R.stats + 7 * (int64_t)R.ms;
    const uint8_t* __restrict__ mask = R.mask;
    int32_t* __restrict__ changed = R.changed;
    if (threadIdx.x == 0) s_base = 0;
    __syncthreads();
    int before = 0;  // changed segments of the blocks before this one
    for (int b = threadIdx.x; b < (int)blockIdx.x; b += kChunk) before += (int)counts[b];
    before = __reduce_add_sync(kFull, before);
    if ((threadIdx.x & 31) == 0 && before) atomicAdd(&s_base, before);
    __syncthreads();
    const int s = blockIdx.x * kChunk + threadIdx.x;
    const int flag = s < S && mask[s] == FTV_MASK_CHANGED;
    int total;
    const int pos = block_exclusive_scan(flag, &total);
    if (flag) changed[s_base + pos] = s;
    if ((int)blockIdx.x == chunks - 1 && threadIdx.x == 0) *R.n_changed = s_base + total;
}

// One warp per listed segment: least-cost label, smallest on ties; masked segments adopt.
__global__ void wta_kernel(const int32_t* __restrict__ cost, int S, int L, const uint8_t* __restrict__ mask,
                           const uint16_t* __restrict__ prev_label, const uint16_t* __restrict__ ifr_label,
                           const int32_t* __restrict__ list, const int32_t* __restrict__ n_listed,
                           uint16_t* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    const int n = list ? min(max(*n_listed, 0), S) : S;
    for (int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n; i += (gridDim.x * blockDim.x) >> 5) {
        const int s = list ? list[i] : i;
        if ((unsigned)s >= (unsigned)S) continue;
        const int m = mask ? mask[s] : FTV_MASK_CHANGED;
        if (m == FTV_MASK_REUSE_P && prev_label) {
            if (lane == 0) out[s] = prev_label[s];
            continue;
        }
        if (m == FTV_MASK_REUSE_I && ifr_label) {
            if (lane == 0) out[s] = ifr_label[s];
            continue;
        }
        const int d = least_label(cost + (int64_t)s * L, L, lane);
        if (lane == 0) out[s] = (uint16_t)d;
    }
}

// Four adjacent pixels of a row per thread.
__global__ void __launch_bounds__(128) depth_map_kernel(const int32_t* __restrict__ labels, int W, int S,
                                                        const uint16_t* __restrict__ seg_label,
                                                        const float* __restrict__ label_z, int L,
                                                        float* __restrict__ depth, bool vec, uint32_t* status) {
    const int x = (blockIdx.x * blockDim.x + threadIdx.x) * 4;
    if (x >= W) return;
    depth4(labels, (int64_t)blockIdx.y * W + x, min(4, W - x), vec, S, seg_label, label_z, L, depth, status);
}

}  // namespace

cudaError_t launch_temporal_refs(const TemporalRef* refs, int n, int sample_bytes, int mode, bool has_i, int t_p,
                                 int t_i, uint32_t* status, cudaStream_t s, int64_t* launches) {
    if (n <= 0) return cudaSuccess;
    if (n > kMaxTemporalRefs) return cudaErrorInvalidValue;
    TemporalRefs p{};
    int tx = 0, ty = 0, chunks = 1;
    bool any_s = false, vec = true, fine = false;
    for (int k = 0; k < n; ++k) {
        p.r[k] = refs[k];
        tx = std::max(tx, (refs[k].W + kAccCols - 1) / kAccCols);
        ty = std::max(ty, (refs[k].H + kAccRowsTile - 1) / kAccRowsTile);
        // four samples (labels) per load where every row of every plane starts on such a boundary
        uintptr_t at = (reinterpret_cast<uintptr_t>(refs[k].labels) & 15) | (uintptr_t)(refs[k].W & 3);
        for (int c = 0; c < (mode == FTV_TM_ALL_YUV ? 3 : 1); ++c) {
            uintptr_t u = reinterpret_cast<uintptr_t>(refs[k].cur[c]) | reinterpret_cast<uintptr_t>(refs[k].prev[c]) |
                          (uintptr_t)refs[k].pc[c] | (uintptr_t)refs[k].pp[c];
            if (has_i) u |= reinterpret_cast<uintptr_t>(refs[k].ifr[c]) | (uintptr_t)refs[k].pi[c];
            at |= u & (uintptr_t)(4 * sample_bytes - 1);
        }
        vec = vec && at == 0;
        fine = fine || (int64_t)refs[k].S * 3 > (int64_t)refs[k].W * refs[k].H;
        chunks = std::max(chunks, (refs[k].S + kChunk - 1) / kChunk);
        any_s = any_s || refs[k].S > 0;
    }
    const int nch = mode == FTV_TM_ALL_YUV ? 3 : 1;
    if (tx > 0 && ty > 0) {
        const dim3 block(kAccThreads), grid(tx, ty, n);
#define FTV_T(SB, NCH, HI) \
    if (fine) temporal_accumulate_kernel<SB, NCH, HI, false, kStrips><<<grid, block, 0, s>>>(p, status); \
    else if (vec) temporal_accumulate_kernel<SB, NCH, HI, true, 1><<<grid, block, 0, s>>>(p, status); \
    else temporal_accumulate_kernel<SB, NCH, HI, false, 1><<<grid, block, 0, s>>>(p, status)
        if (sample_bytes == 1) {
            if (nch == 1) { if (has_i) { FTV_T(1, 1, true); } else { FTV_T(1, 1, false); } }
            else { if (has_i) { FTV_T(1, 3, true); } else { FTV_T(1, 3, false); } }
        } else {
            if (nch == 1) { if (has_i) { FTV_T(2, 1, true); } else { FTV_T(2, 1, false); } }
            else { if (has_i) { FTV_T(2, 3, true); } else { FTV_T(2, 3, false); } }
        }
#undef FTV_T
        *launches += 1;
    }
    if (any_s) {
        const dim3 grid(chunks, n);
        if (nch == 1) {
            if (has_i) temporal_decide_kernel<1, true><<<grid, kChunk, 0, s>>>(p, t_p, t_i);
            else temporal_decide_kernel<1, false><<<grid, kChunk, 0, s>>>(p, t_p, t_i);
        } else {
            if (has_i) temporal_decide_kernel<3, true><<<grid, kChunk, 0, s>>>(p, t_p, t_i);
            else temporal_decide_kernel<3, false><<<grid, kChunk, 0, s>>>(p, t_p, t_i);
        }
        *launches += 1;
    }
    temporal_compact_kernel<<<dim3(chunks, n), kChunk, 0, s>>>(p);
    *launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_temporal(const void* const* cur, const int64_t* cur_pitch, const void* const* prev,
                            const int64_t* prev_pitch, const void* const* ifr, const int64_t* ifr_pitch,
                            int sample_bytes, const int32_t* labels, int W, int H, int S, int t_p, int t_i,
                            int mode, int64_t* stats, int ms, uint8_t* mask, int32_t* changed, int32_t* n_changed,
                            uint32_t* status, bool clear, cudaStream_t s, int64_t* launches) {
    if (clear) {  // planes 0 to 6 over the call's segments
        const cudaError_t e = cudaMemsetAsync(stats, 0, sizeof(int64_t) * (6 * (size_t)ms + (size_t)S), s);
        if (e != cudaSuccess) return e;
    }
    TemporalRef r{};
    for (int c = 0; c < 3; ++c) {
        r.cur[c] = cur[c];
        r.prev[c] = prev[c];
        r.ifr[c] = ifr ? ifr[c] : nullptr;
        r.pc[c] = cur_pitch[c];
        r.pp[c] = prev_pitch[c];
        r.pi[c] = ifr ? ifr_pitch[c] : 0;
    }
    r.labels = labels;
    r.stats = stats;
    r.mask = mask;
    r.changed = changed;
    r.n_changed = n_changed;
    r.W = W;
    r.H = H;
    r.S = S;
    r.ms = ms;
    return launch_temporal_refs(&r, 1, sample_bytes, mode, ifr != nullptr, t_p, t_i, status, s, launches);
}

cudaError_t launch_wta(const int32_t* cost, int S, int L, const uint8_t* mask, const uint16_t* prev_label,
                       const uint16_t* ifr_label, const int32_t* list, const int32_t* n_listed, uint16_t* out,
                       cudaStream_t s) {
    const int warps_per_block = 8;
    const int blocks = std::max(1, std::min(65535, (S + warps_per_block - 1) / warps_per_block));
    wta_kernel<<<blocks, warps_per_block * 32, 0, s>>>(cost, S, L, mask, prev_label, ifr_label, list, n_listed, out);
    return cudaGetLastError();
}

cudaError_t launch_depth_map(const int32_t* labels, int W, int H, int S, const uint16_t* seg_label,
                             const float* label_z, int L, float* depth, uint32_t* status, cudaStream_t s) {
    if (W <= 0 || H <= 0) return cudaSuccess;
    const dim3 block(128), grid((W + 511) / 512, H);
    const bool vec = ((reinterpret_cast<uintptr_t>(labels) | reinterpret_cast<uintptr_t>(depth)) & 15) == 0 && W % 4 == 0;
    depth_map_kernel<<<grid, block, 0, s>>>(labels, W, S, seg_label, label_z, L, depth, vec, status);
    return cudaGetLastError();
}

}  // namespace ftv
