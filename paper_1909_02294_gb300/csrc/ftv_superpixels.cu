// Superpixel segmentation (Sec. IV-C): the label maps the method consumes, as SNIC-like superpixels in
// (Y, Cb, Cr) with compactness factor m and 8-connected segments.
//
// SNIC grows every cluster from its seed through a single priority queue, which is sequential. This is
// its data-parallel reformulation (the clustering SNIC itself derives from), with SNIC's seeds, distance
// and connectivity:
//   - seeds on an S x S grid: cell (i, j) of width w and height h has label j * ceil(W/S) + i and seed
//     (iS + (w-1)/2, jS + (h-1)/2);
//   - D = S^2 ||c_p - c_k||^2 + m^2 ||x_p - x_k||^2 on the 8-bit colour scale (the spatial weight times
//     4^(bd-8) above 8 bits, the colour weight times 4^(8-bd) below), evaluated exactly in 64-bit
//     integers on 16 * (pixel value) - (cluster mean in 1/16 units);
//   - assignment passes: a pixel of cell (i, j) joins the least-D cluster among cells (i+a, j+b),
//     a, b in {-1, 0, 1} (smallest label on ties); between passes every cluster mean becomes
//     floor((32 sum + n) / (2 n)) of its pixels (an empty cluster keeps its mean);
//   - connectivity: components are the 8-connected sets of equally labelled pixels (named by their first
//     pixel); a label's largest component (earliest on ties) is anchored with that label; the other
//     components merge in rounds, each unanchored group joining the 8-adjacent group of nearest mean
//     colour (L1 of the rounded 1/16 means; on ties the group of smallest name, a group's name being its
//     smallest component name), all picks of a round at once, until every group is anchored.
// The result is unique (integer arithmetic, order-free rules), so it equals the CPU definition exactly.
//
// Kernels: one assignment launch per pass (a thread takes a column of a cell row's pixels, the candidates' centres staged
// in shared memory; D in 32-bit integers when the weights reduced by their gcd provably keep it below 2^32, else in
// 64-bit; runs of equal labels summed in registers, then into per-tile shared accumulators, then one global add per
// cluster and pair of fields), which also forms the means of the pass before; components_kernel, the components of each
// 32 x 32 tile by union-find in shared memory (atomicMin linking, so a root is its component's first pixel); and
// regions_kernel, one cooperative launch that links the tiles, sums the components, picks every label's main component,
// runs the merge rounds (round 0 over every pixel, later rounds over the pixels of unanchored groups that still
// touched another group, a list that shrinks every round) and writes the labels.
// 8 images of 1920x1080, 10 passes: 4.28 -> 2.47 ms; one of 480x270: 0.55 -> 0.26 ms, 113 launches -> 12.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cstring>
#include <numeric>
#include <vector>

#include "ftv_internal.h"

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kThreads = 256;
constexpr int kTileW = 32, kTileH = 4;           // pixel tiles of a warp in regions_kernel
constexpr int kPY = 5;                           // assignment: vertically adjacent pixels per thread, at most
constexpr int kAGroups = 4;                      // assignment: row groups per thread (one where images are small)
constexpr int kATileW = 64;                      // assignment: columns per CTA, one thread each
static_assert(kATileW * kAGroups * kPY <= 1280 && kAGroups * kPY <= 20 && kATileW <= 64, "packed tile sums");
constexpr int kCTile = 32;                       // component tiles
constexpr int kLoopCap = 1 << 26;                // bound of every union-find walk (parents strictly decrease)
// One CTA of 1024 threads per SM: a barrier costs by the CTAs that meet at it (about 10 us with 912 CTAs of 256).
constexpr int kRegionThreads = 1024;  // 152 of 1024: about 1 us
constexpr int kRun = 128;             // entries that a warp of regions_kernel appends to a list at a time
constexpr unsigned long long kNone = ~0ull;

enum : uint32_t { SP_LOOP_CAP = 1u, SP_ROUND_CAP = 2u, SP_BARRIER = 4u };
enum : int { DIST_DOT32 = 0, DIST_NARROW = 1, DIST_WIDE = 2, DIST_WIDE_COLOUR = 3 };

struct SegImage {
    const void* plane[3];
    int64_t pitch[3];
    int32_t* out;
    int32_t W, H, gw, gh;
    int32_t pix_base, seg_base, K;
    int32_t tile_base, ctile_base;  // first pixel tile and first component tile of the image, flattened over the images
    int32_t pad;
};

struct alignas(32) Centre {  // one 32-byte sector each
    int x, y, c0, c1, c2;
};

struct alignas(32) Sums {
    uint32_t n, x, y, c0, c1, c2;
};

struct alignas(32) GSum {
    unsigned long long n, c0, c1, c2;
};

// counters: [4 + 2 rounds] tile components, [6 + 2 rounds + r] anchored groups that gained members in round r, [0]
// components, [1 + r] unanchored groups at the start of round r (r = 0..rounds), which
// is also the length of the round's list uroots, [2 + rounds + r] length of round r's pick list (r = 0..rounds)
struct Scratch {
    const SegImage* img;
    Centre* cen[2];               // [K] cluster means before an assignment pass, alternating between passes
    Sums* sums[3];                // [K] cluster sums: of the previous pass, of this one, cleared for the next
    unsigned long long* mainkey;  // [K]: (size << 32) | ~name of the label's largest component
    int32_t* lab;                 // [P] global segment id of each pixel
    int32_t* par;                 // [P] union-find over pixels; then -1 - (component index) at a component's name
    int32_t* comp;                // [P] component index of each pixel
    ulonglong2* csum;             // [P] per component name: (n << 40) + sum Y, (sum Cb << 32) + sum Cr
                                  // (a component lies in one cluster: n < 2^24, each sum < 2^32)
    int32_t* comps;               // [P] component names (first pixels), by component index
    // Groups live at the index of one of their components, so that their fields lie close together:
    int32_t* gpar;                // [P] union-find over component indexes
    int32_t* glab;                // [P] anchored label of a group (-1 unanchored)
    GSum* gsum;                   // [P] group sums (valid at group roots)
    int4* gmean;                  // [P] group mean colour in 1/16 units, and its name (its smallest component name)
    unsigned long long* best;     // [P] (distance << 32) | name picked by an unanchored group
    int32_t* uroots[2];           // [P] unanchored group roots at the start of a round, alternating; before the
                                  // rounds uroots[1] lists the tile components' roots
    int32_t* dirty;               // [P] an anchored root gained members in the current round (then listed)
    int32_t* dirty_list;          // [P]
    int2* orph[2];                // [P] pick lists of (pixel, image), alternating between rounds
    int32_t* cnt;
    uint32_t* barrier;            // arrivals at the grid barriers of regions_kernel (cleared with cnt)
    int32_t* work;                // [2 phases] items drawn from for_items (cleared with cnt)
    uint32_t* status;
    int32_t polls;                // bound of the grid barriers' waits
    int32_t n_images, tiles, ctiles;  // images, and pixel tiles and component tiles of all of them
    int64_t pixels;
    int32_t S, sb, rounds, max_cells;
    int32_t G, PY;                // row groups per cell row, rows per group
    int32_t packed;               // a tile's count and Cr sum share a word (bit depth <= 10)
    unsigned long long wc, ws;    // distance weights
    uint32_t wcn, wsn;            // the weights divided by their gcd (32-bit distance)
};

__device__ __forceinline__ int sample(const SegImage& im, int c, int x, int y, int sb) {
    const char* row = static_cast<const char*>(im.plane[c]) + (int64_t)y * im.pitch[c];
    return sb == 1 ? (int)reinterpret_cast<const uint8_t*>(row)[x] : (int)reinterpret_cast<const uint16_t*>(row)[x];
}

__device__ __forceinline__ int seed_coord(int n, int S, int i) {
    const int w = min(S, n - i * S);
    return i * S + (w - 1) / 2;
}

// round(16 * s / n), halves up: floor((32 s + n) / (2 n)); 32-bit division when it fits
__device__ __forceinline__ int mean16(unsigned long long s, unsigned long long n) {
    const unsigned long long num = 32ull * s + n, den = 2ull * n;
    if ((num >> 32) == 0 && (den >> 32) == 0) return (int)((uint32_t)num / (uint32_t)den);
    return (int)(num / den);
}

// Walk to the root. Reads may be stale while other threads link (a stale parent is still an ancestor),
// so a walk always ends at a node that is or was a root; unite() then corrects itself through the atomic.
// CG: read parents from L2 (ld.global.cg), for walks that run while other SMs link.
template <bool CG = false>
__device__ int find_root(const int32_t* par, int32_t x, uint32_t* status) {
    for (int it = 0; it < kLoopCap; ++it) {
        const int32_t p = CG ? __ldcg(&par[x]) : par[x];
        if (p == x) return x;
        x = p;
    }
    atomicOr(status, SP_LOOP_CAP);
    return x;
}

// Link the sets of a and b; the smaller root becomes the parent (so a root is its set's smallest name).
__device__ void unite(int32_t* par, int32_t a, int32_t b, uint32_t* status) {
    for (int it = 0; it < kLoopCap; ++it) {
        a = find_root<true>(par, a, status);
        b = find_root<true>(par, b, status);
        if (a == b) return;
        if (a > b) {
            const int32_t t = a;
            a = b;
            b = t;
        }
        const int32_t old = atomicMin(&par[b], a);
        if (old == b) return;  // b was a root and now hangs under a
        b = old;               // b was linked meanwhile: join a with b's new parent instead
    }
    atomicOr(status, SP_LOOP_CAP);
}

// A warp's share of a list that grows in global memory: entries gather in shared memory (RUN + 32 words of it) and leave
// RUN at a time, coalesced, with one atomic (an append of the whole CTA waited at three barriers per call). All warps of
// the chip meet at that atomic, so a long list takes long runs (15 fragmented images of
// 3840x2160: 54.5 ms with runs of 32, 44.2 of 128).
template <class T, int RUN>
struct WarpList {
    T* buf;
    T* list;
    int32_t* counter;
    int n;

    __device__ __forceinline__ void flush() {
        const int lane = threadIdx.x & 31, k = min(n, RUN);
        __syncwarp();
        int base = 0;
        if (lane == 0) base = atomicAdd(counter, k);
        base = __shfl_sync(kFull, base, 0);
        for (int i = lane; i < k; i += 32) list[base + i] = buf[i];
        T rest{};
        if (lane < n - k) rest = buf[k + lane];
        __syncwarp();
        if (lane < n - k) buf[lane] = rest;
        n -= k;
        __syncwarp();
    }
    // all lanes of the warp call it
    __device__ __forceinline__ void append(bool keep, const T& v) {
        const unsigned m = __ballot_sync(kFull, keep);
        if (m == 0) return;
        if (keep) buf[n + __popc(m & ((1u << (threadIdx.x & 31)) - 1u))] = v;
        n += __popc(m);
        if (n >= RUN) flush();
    }
    __device__ __forceinline__ void finish() {
        while (n > 0) flush();
    }
};

// ---------------------------------------------------------------------------------------- clustering

// D of one candidate, from the staged cell (a, b). Direct forms (a = x, y, Y, Cb of the mean; b.x = Cr):
// NARROW uses the gcd-reduced weights in 32 bits (the host has shown that D stays below 2^32); WIDE
// 32-bit squares and a 64-bit weighted sum; WIDE_COLOUR 64-bit colour squares (bit depth > 11).
// DOT32 drops the pixel's own squares, common to all candidates: with tile-relative positions,
// D - wc' |v|^2 - ws' |p|^2 = K - 2 (wc' <v, c> + ws' <p, x>) where K = wc' |c|^2 + ws' |x|^2, so
// a = (K, -2 ws' x, -2 ws' y, -2 wc' Y), b = (-2 wc' Cb, -2 wc' Cr): five multiply-adds in 32 bits
// (the host has shown that every partial sum stays below 2^31 in magnitude).
template <int DM>
struct Dist {
    using T = unsigned long long;
};
template <>
struct Dist<DIST_NARROW> {
    using T = uint32_t;
};
template <>
struct Dist<DIST_DOT32> {
    using T = int;
};

template <int DM>
__device__ __forceinline__ typename Dist<DM>::T distance(const int4 a, const int4 b, int vx, int vy, int w0, int w1,
                                                         int w2, const Scratch& s) {
    static_assert(DM != DIST_DOT32, "assign_kernel steps that form from row to row");
    const int dx = vx - a.x, dy = vy - a.y;
    const uint32_t dsp = (uint32_t)dx * (uint32_t)dx + (uint32_t)dy * (uint32_t)dy;
    const int d0 = w0 - a.z, d1 = w1 - a.w, d2 = w2 - b.x;
    if (DM == DIST_NARROW) {
        const uint32_t dcol = (uint32_t)d0 * (uint32_t)d0 + (uint32_t)d1 * (uint32_t)d1 + (uint32_t)d2 * (uint32_t)d2;
        return (typename Dist<DM>::T)(s.wcn * dcol + s.wsn * dsp);
    } else if (DM == DIST_WIDE) {
        const uint32_t dcol = (uint32_t)d0 * (uint32_t)d0 + (uint32_t)d1 * (uint32_t)d1 + (uint32_t)d2 * (uint32_t)d2;
        return (typename Dist<DM>::T)(s.wc * dcol + s.ws * dsp);
    } else {
        const unsigned long long dcol = (unsigned long long)((long long)d0 * d0) +
                                        (unsigned long long)((long long)d1 * d1) +
                                        (unsigned long long)((long long)d2 * d2);
        return (typename Dist<DM>::T)(s.wc * dcol + s.ws * dsp);
    }
}

// Field f (x, y, Y, Cb, Cr in 1/16 units) of cell (i, j)'s cluster mean before pass `pass`: its seed pixel, or the
// rounded mean of the pixels that joined it in the previous pass (a cluster without pixels keeps its mean).
template <int SB>
__device__ __forceinline__ int centre_field(const Scratch& s, const SegImage& im, int i, int j, int f, int pass) {
    if (pass == 0) {
        const int x = seed_coord(im.W, s.S, i), y = seed_coord(im.H, s.S, j);
        return 16 * (f == 0 ? x : f == 1 ? y : sample(im, f - 2, x, y, SB));
    }
    const int k = im.seg_base + j * im.gw + i;
    const uint32_t* t = &s.sums[(pass + 2) % 3][k].n;  // n, x, y, c0, c1, c2
    const uint32_t n = t[0];
    return n ? mean16(t[1 + f], n) : reinterpret_cast<const int*>(&s.cen[(pass + 1) & 1][k])[f];
}

// One assignment pass. A thread takes up to kPY vertically adjacent pixels of one cell row (a group: the rows of a
// cell row are split into s.G groups), so that its nine candidates are the same for all of them: each staged
// candidate is read once, its column term is formed once and its row term steps by an addition. A CTA takes kATileW
// columns of kAGroups consecutive groups, a thread its column through all of them (what a thread computes once, image,
// cells and divisions, weighed a quarter of the pass with one group per thread; an image too small to fill the chip with
// such columns keeps one group: AG). accumulate: add every pixel to its cluster's sums for the next pass, as runs
// in registers, then the tile's bins in shared memory (counts and positions relative to the tile, two sums to a
// word), then one 64-bit add per pair of sums and cluster. last: write the labels.
// The cluster means of the previous pass are formed here, by every CTA for the cells it can see (no kernel between the
// passes); the cell's own tile stores them and clears the sums of the pass after this one.
// The 3 x 3 candidates are visited unrolled in increasing label order; a candidate outside the grid is
// replaced by the nearest existing cell, a repeat of a label already visited with the same D, which the
// strict comparison ignores.
// Bound by instruction issue (about seven per candidate and pixel): 101 us per pass over eight 1920x1080 images, where
// four horizontal pixels per thread, each with its own candidates, took 280 instructions per pixel and 184 us.
template <int DM, int SB, int AG, int ROWS>
__global__ void __launch_bounds__(kATileW) assign_kernel(Scratch s, int pass, int accumulate, int last) {
    extern __shared__ __align__(16) unsigned char smem[];
    const SegImage& im = s.img[blockIdx.z];
    const int S = s.S, G = s.G, PY = s.PY, MC = s.max_cells;
    const int x0 = blockIdx.x * kATileW, g0 = blockIdx.y * AG;
    const int cj0 = g0 / G;
    if (x0 >= im.W || cj0 >= im.gh) return;  // uniform over the CTA
    const int cx0 = max(0, x0 / S - 1), cx1 = min(im.gw - 1, min(im.W - 1, x0 + kATileW - 1) / S + 1);
    const int cy0 = max(0, cj0 - 1), cy1 = min(im.gh - 1, (g0 + AG - 1) / G + 1);
    const int ncx = cx1 - cx0 + 1, ncells = ncx * (cy1 - cy0 + 1);
    const int y0 = cj0 * S + (g0 - cj0 * G) * PY;  // first row of the tile
    int4* sA = reinterpret_cast<int4*>(smem);
    int4* sB = sA + MC;
    uint32_t* acc = reinterpret_cast<uint32_t*>(sB + MC);  // [5][MC]: (y, x), Y, Cb, Cr or (n, Cr), n
    const int tid = threadIdx.x;
    // one field of one mean per thread (a division each), then one cell per thread
    for (int q = tid; q < 5 * ncells; q += kATileW) {
        const int f = q / ncells, e = q - f * ncells, j = e / ncx;
        acc[f * MC + e] = (uint32_t)centre_field<SB>(s, im, cx0 + e - j * ncx, cy0 + j, f, pass);
    }
    __syncthreads();
    for (int e = tid; e < ncells; e += kATileW) {
        const int j = cy0 + e / ncx, i = cx0 + e % ncx;
        const Centre c{(int)acc[e], (int)acc[MC + e], (int)acc[2 * MC + e], (int)acc[3 * MC + e], (int)acc[4 * MC + e]};
        // the cell's own tile: its first group's rows, its first column
        if (j * G >= g0 && j * G < g0 + AG && i * S >= x0 && i * S < x0 + kATileW) {
            const int k = im.seg_base + j * im.gw + i;
            s.cen[pass & 1][k] = c;
            s.sums[(pass + 1) % 3][k] = Sums{};
            if (pass == 0) s.mainkey[k] = 0;
        }
        if (DM == DIST_DOT32) {
            const int xr = c.x - 16 * x0, yr = c.y - 16 * y0;
            const long long K = (long long)s.wcn * ((long long)c.c0 * c.c0 + (long long)c.c1 * c.c1 +
                                                    (long long)c.c2 * c.c2) +
                                (long long)s.wsn * ((long long)xr * xr + (long long)yr * yr);
            const int wc2 = 32 * (int)s.wcn, ws2 = 32 * (int)s.wsn;  // times the pixel's own 16
            sA[e] = make_int4((int)K, -ws2 * xr, -ws2 * yr, -wc2 * c.c0);
            sB[e] = make_int4(-wc2 * c.c1, -wc2 * c.c2, 0, 0);
        } else {
            sA[e] = make_int4(c.x, c.y, c.c0, c.c1);
            sB[e] = make_int4(c.c2, 0, 0, 0);
        }
        if (accumulate)
            for (int f = 0; f < 5; ++f) acc[f * MC + e] = 0;
    }
    __syncthreads();

    const int x = x0 + tid;
    if (x < im.W) {
        const int ci = x / S, W = im.W, H = im.H, gh = im.gh;
        const int i0 = max(ci - 1, 0) - cx0, i1 = ci - cx0, i2 = min(ci + 1, im.gw - 1) - cx0;
        int cj = cj0, gi = g0 - cj0 * G;  // cell row and group within it
        const char* col[3];               // the column in each plane
        int64_t pitch[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            pitch[c] = im.pitch[c];
            col[c] = static_cast<const char*>(im.plane[c]) + (int64_t)x * SB;
        }
        auto load = [&](int c, int y) {
            const char* at = col[c] + (int64_t)y * pitch[c];
            return SB == 1 ? (int)__ldg(reinterpret_cast<const uint8_t*>(at)) : (int)__ldg(reinterpret_cast<const uint16_t*>(at));
        };
#pragma unroll 1
        for (int g = 0; g < AG && cj < gh; ++g) {
            const int ya = cj * S + gi * PY, rows = min(min(PY, S - gi * PY), H - ya);
            if (rows > 0) {
                int v0[ROWS], v1[ROWS], v2[ROWS], be[ROWS];
                typename Dist<DM>::T bd[ROWS];
#pragma unroll
                for (int r = 0; r < ROWS; ++r) {
                    const bool in = r < rows;
                    v0[r] = in ? load(0, ya + r) : 0;
                    v1[r] = in ? load(1, ya + r) : 0;
                    v2[r] = in ? load(2, ya + r) : 0;
                    be[r] = 0;
                    bd[r] = 0;
                }
#pragma unroll
                for (int c = 0; c < 9; ++c) {
                    const int j = c / 3 == 0 ? max(cj - 1, 0) : (c / 3 == 1 ? cj : min(cj + 1, gh - 1));
                    const int i = c % 3 == 0 ? i0 : (c % 3 == 1 ? i1 : i2);
                    const int e = (j - cy0) * ncx + i;
                    const int4 a = sA[e], b = sB[e];
                    int t = 0;
                    if (DM == DIST_DOT32) t = a.x + (x - x0) * a.y + (ya - y0) * a.z;
#pragma unroll
                    for (int r = 0; r < ROWS; ++r) {
                        typename Dist<DM>::T D;
                        if constexpr (DM == DIST_DOT32) {
                            D = (typename Dist<DM>::T)(t + v0[r] * a.w + v1[r] * b.x + v2[r] * b.y);
                            t += a.z;
                        } else {
                            D = distance<DM>(a, b, 16 * x, 16 * (ya + r), 16 * v0[r], 16 * v1[r], 16 * v2[r], s);
                        }
                        if (c == 0 || D < bd[r]) {
                            bd[r] = D;
                            be[r] = e;
                        }
                    }
                }
                if (last) {
#pragma unroll
                    for (int r = 0; r < ROWS; ++r)
                        if (r < rows) {
                            const int bj = be[r] / ncx;
                            const int64_t gp = (int64_t)im.pix_base + (int64_t)(ya + r) * W + x;
                            s.lab[gp] = im.seg_base + (cy0 + bj) * im.gw + cx0 + be[r] - bj * ncx;
                        }
                }
                if (accumulate) {
                    uint32_t n = 0, q0 = 0, q1 = 0, q2 = 0, qy = 0;
#pragma unroll
                    for (int r = 0; r < ROWS; ++r) {
                        if (r < rows) {
                            n += 1;
                            q0 += v0[r];
                            q1 += v1[r];
                            q2 += v2[r];
                            qy += ya + r - y0;
                            if (r + 1 >= rows || be[r + 1 < ROWS ? r + 1 : r] != be[r]) {
                                // a tile has at most 64 x 20 pixels, so that n < 2^11, the relative y sum < 2^15 and the
                                // relative x sum < 2^17; at 10 bits a colour sum is below 2^21
                                const int e = be[r];
                                atomicAdd(&acc[e], (qy << 17) + n * (uint32_t)(x - x0));
                                atomicAdd(&acc[MC + e], q0);
                                atomicAdd(&acc[2 * MC + e], q1);
                                if (s.packed) {
                                    atomicAdd(&acc[3 * MC + e], (n << 21) + q2);
                                } else {
                                    atomicAdd(&acc[3 * MC + e], q2);
                                    atomicAdd(&acc[4 * MC + e], n);
                                }
                                n = q0 = q1 = q2 = qy = 0;
                            }
                        }
                    }
                }
            }
            if (++gi == G) {
                gi = 0;
                ++cj;
            }
        }
    }
    if (!accumulate) return;
    __syncthreads();
    for (int e = tid; e < ncells; e += kATileW) {
        const uint32_t cr = acc[3 * MC + e];
        const uint32_t n = s.packed ? cr >> 21 : acc[4 * MC + e];
        if (n == 0) continue;
        const uint32_t yx = acc[e], c2 = s.packed ? cr & 0x1fffffu : cr;
        const unsigned long long X = (unsigned long long)(yx & 0x1ffffu) + (unsigned long long)n * (unsigned)x0;
        const unsigned long long Y = (unsigned long long)(yx >> 17) + (unsigned long long)n * (unsigned)y0;
        const int j = cy0 + e / ncx, i = cx0 + e % ncx;
        // a cluster's pixels lie in 3 x 3 cells of 64 x 64, so that each of its sums stays below 2^32
        unsigned long long* t = reinterpret_cast<unsigned long long*>(&s.sums[pass % 3][im.seg_base + j * im.gw + i]);
        atomicAdd(&t[0], n | (X << 32));
        atomicAdd(&t[1], Y | ((unsigned long long)acc[MC + e] << 32));
        atomicAdd(&t[2], (unsigned long long)acc[2 * MC + e] | ((unsigned long long)c2 << 32));
    }
}

// ------------------------------------------------------------------------------------- connectivity

// Root of a tile's pixel in its shared union-find.
__device__ __forceinline__ int tile_root(const volatile int* par, int x) {
    for (int p = par[x]; p != x; p = par[x]) x = p;  // parents strictly decrease
    return x;
}

__device__ __forceinline__ void tile_unite(int* par, int a, int b) {
    for (int it = 0; it < kCTile * kCTile; ++it) {  // every turn lowers a parent
        a = tile_root(par, a);
        b = tile_root(par, b);
        if (a == b) return;
        if (a > b) {
            const int t = a;
            a = b;
            b = t;
        }
        const int old = atomicMin(&par[b], a);
        if (old == b) return;
        b = old;
    }
}

// 8-connected components of equal labels within one 32 x 32 tile, in shared memory: every row of the tile is a warp's;
// a ballot finds each pixel's run start, runs are linked to the row above where they overlap (issued once, from the
// later of the two run starts) or touch diagonally (from the run's first and last pixel), and each run's count and
// colour sums are added to its root's. A tile component's root is its first pixel; par
// names it for every pixel, csum holds its sums, and the roots are listed. The links across tiles and the rest
// follow in regions_kernel. Bound by divergent walks and shared-memory latency: 0.40 ms for eight 1920x1080 images, where
// linking every run through global atomics took 0.54 ms and the sums of every run 0.29 ms.
__global__ void __launch_bounds__(kThreads) components_kernel(Scratch s) {
    constexpr int kRows = kCTile / (kThreads / 32);  // rows per warp
    __shared__ int s_lab[kCTile * kCTile], s_par[kCTile * kCTile];
    __shared__ uint32_t s_sum[4][kCTile * kCTile];
    __shared__ int32_t s_buf[kThreads / 32][64];
    const SegImage& im = s.img[blockIdx.z];
    const int x0 = blockIdx.x * kCTile, y0 = blockIdx.y * kCTile;
    if (x0 >= im.W || y0 >= im.H) return;  // uniform over the CTA
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, x = x0 + lane;
    const unsigned upto = kFull >> (31 - lane);
#pragma unroll
    for (int k = 0; k < kRows; ++k) {
        const int row = warp * kRows + k, y = y0 + row, i = row * kCTile + lane;
        const bool valid = x < im.W && y < im.H;
        const int l = valid ? s.lab[im.pix_base + y * im.W + x] : -1;
        const int left = __shfl_up_sync(kFull, l, 1);
        const unsigned cont = __ballot_sync(kFull, valid && lane > 0 && left == l);  // continues the run on its left
        s_lab[i] = l;
        s_par[i] = row * kCTile + 31 - __clz(~cont & upto);
#pragma unroll
        for (int f = 0; f < 4; ++f) s_sum[f][i] = 0;
    }
    // the runs of row `row` with those of the row above
    auto link_rows = [&](int row) {
        const int i = row * kCTile + lane, l = s_lab[i];
        if (l < 0) return;
        const int* up = &s_lab[i - kCTile];
        const bool first = lane == 0 || s_lab[i - 1] != l, end = lane == 31 || s_lab[i + 1] != l;
        if (up[0] == l && (first || up[-1] != l)) tile_unite(s_par, i, i - kCTile);
        if (first && lane > 0 && up[-1] == l) tile_unite(s_par, i, i - kCTile - 1);
        if (end && lane < 31 && up[1] == l) tile_unite(s_par, i, i - kCTile + 1);
    };
    // first within the warp's own rows, each row's parents shortened before the next row hangs under them
    __syncwarp();
#pragma unroll
    for (int k = 1; k < kRows; ++k) {
        link_rows(warp * kRows + k);
        __syncwarp();
        const int i = (warp * kRows + k) * kCTile + lane;
        const int r = tile_root(s_par, i);
        __syncwarp();
        s_par[i] = r;
        __syncwarp();
    }
    __syncthreads();
    if (warp > 0) link_rows(warp * kRows);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kRows; ++k) {
        const int row = warp * kRows + k, y = y0 + row, i = row * kCTile + lane, l = s_lab[i];
        const int left = __shfl_up_sync(kFull, l, 1);
        const unsigned cont = __ballot_sync(kFull, l >= 0 && lane > 0 && left == l);
        const int start = 31 - __clz(~cont & upto);
        const int r = tile_root(s_par, i);
        uint32_t v[3] = {0, 0, 0};
        if (l >= 0) {
#pragma unroll
            for (int c = 0; c < 3; ++c) v[c] = sample(im, c, x, y, s.sb);
            s.par[im.pix_base + y * im.W + x] = im.pix_base + (y0 + (r >> 5)) * im.W + x0 + (r & 31);
        }
        // a run's sums are differences of the row's prefix sums, taken by its last lane
#pragma unroll
        for (int o = 1; o < 32; o <<= 1)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const uint32_t t = __shfl_up_sync(kFull, v[c], o);
                if (lane >= o) v[c] += t;
            }
        const bool end = lane == 31 || !(cont >> (lane + 1) & 1u);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const uint32_t before = __shfl_sync(kFull, v[c], max(start - 1, 0));
            if (l >= 0 && end) atomicAdd(&s_sum[1 + c][r], v[c] - (start > 0 ? before : 0u));
        }
        if (l >= 0 && end) atomicAdd(&s_sum[0][r], (uint32_t)(lane - start + 1));
    }
    __syncthreads();
    WarpList<int32_t, 32> roots{s_buf[warp], s.uroots[1], &s.cnt[4 + 2 * s.rounds], 0};
#pragma unroll
    for (int k = 0; k < kRows; ++k) {
        const int row = warp * kRows + k, y = y0 + row, i = row * kCTile + lane;
        const bool root = s_lab[i] >= 0 && s_par[i] == i;
        const int32_t gp = im.pix_base + y * im.W + x;
        if (root)
            s.csum[gp] = make_ulonglong2(((unsigned long long)s_sum[0][i] << 40) + s_sum[1][i],
                                         ((unsigned long long)s_sum[2][i] << 32) + s_sum[3][i]);
        roots.append(root, gp);
    }
    roots.finish();
}

// Distance of two groups' mean colours in the high word, the second's name in the low one.
__device__ __forceinline__ unsigned long long pick_key(const int4& ma, const int4& mb) {
    return ((unsigned long long)(abs(ma.x - mb.x) + abs(ma.y - mb.y) + abs(ma.z - mb.z)) << 32) |
           (unsigned long long)(uint32_t)mb.w;
}

// The pick of one pixel p (component pc) of group a (unanchored): the neighbouring group of least
// (distance, name). The lookups run in stages over all eight neighbours at once (components, one step
// up the group forest, the rest of the walk where one is left, then means and names), so that each
// stage's independent loads are in flight together; neighbours in p's own component are skipped.
__device__ __forceinline__ bool pick_pixel(const Scratch& s, const SegImage& im, int32_t p, int32_t pc, int32_t a) {
    const int local = p - im.pix_base;
    const int x = local % im.W, y = local / im.W;
    int32_t g[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int dx = k < 3 ? k - 1 : (k == 3 ? -1 : (k == 4 ? 1 : k - 6));
        const int dy = k < 3 ? -1 : (k < 5 ? 0 : 1);
        const int qx = x + dx, qy = y + dy;
        g[k] = (qx >= 0 && qx < im.W && qy >= 0 && qy < im.H) ? s.comp[p + dy * im.W + dx] : -1;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) g[k] = (g[k] < 0 || g[k] == pc) ? -1 : s.gpar[g[k]];
#pragma unroll
    for (int k = 0; k < 8; ++k)
        if (g[k] >= 0) {
            const int32_t up = s.gpar[g[k]];
            if (up != g[k]) g[k] = find_root(s.gpar, up, s.status);
        }
    const int4 ma = s.gmean[a];
    unsigned long long best = kNone;
#pragma unroll
    for (int k = 0; k < 8; ++k)
        if (g[k] >= 0 && g[k] != a) best = min(best, pick_key(ma, s.gmean[g[k]]));
    if (best == kNone) return false;
    atomicMin(&s.best[a], best);
    return true;
}

// The mean colour of a group from its sums (they and the name were changed by atomics of other SMs).
__device__ __forceinline__ void set_mean(const Scratch& s, int32_t t) {
    const unsigned long long n = __ldcg(&s.gsum[t].n), c0 = __ldcg(&s.gsum[t].c0), c1 = __ldcg(&s.gsum[t].c1),
                             c2 = __ldcg(&s.gsum[t].c2);
    s.gmean[t] = make_int4(mean16(c0, n), mean16(c1, n), mean16(c2, n), __ldcg(&s.gmean[t].w));
}

// Group links order roots anchored first, then by smaller name, and hang the later root under the earlier
// one (compare-and-swap on a root): an anchored root therefore never gets a parent, and the order is total,
// so no cycle can form. Anchored status does not change while links are made.
__device__ void unite_groups(Scratch& s, int32_t a, int32_t b) {
    for (int it = 0; it < kLoopCap; ++it) {
        a = find_root<true>(s.gpar, a, s.status);
        b = find_root<true>(s.gpar, b, s.status);
        if (a == b) return;
        const bool aa = s.glab[a] >= 0, ab = s.glab[b] >= 0;
        if (ab > aa || (ab == aa && b < a)) {
            const int32_t t = a;
            a = b;
            b = t;
        }
        if (atomicCAS(&s.gpar[b], b, a) == b) return;
    }
    atomicOr(s.status, SP_LOOP_CAP);
}

// A barrier of the whole grid (a cooperative launch: every CTA is resident). Arrivals count up; `phase` is the number
// of barriers passed. Waits at most s.polls polls, then reports SP_BARRIER and returns false, on which the CTA leaves
// the kernel. The others may still pass this barrier, but not the next one, where its arrival is missing: no CTA ever
// works on a phase before every CTA has finished the one before it.
constexpr int kBarrierPolls = 1 << 23;  // seconds

__device__ bool grid_barrier(const Scratch& s, uint32_t& phase) {
    __shared__ int s_ok;
    __syncthreads();
    ++phase;
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(s.barrier, 1u);
        const uint32_t target = phase * gridDim.x;
        int polls = 0;
        while (*reinterpret_cast<volatile uint32_t*>(s.barrier) < target && ++polls < s.polls) {
        }
        s_ok = polls < s.polls;
        if (!s_ok) atomicOr(s.status, SP_BARRIER);
        __threadfence();
    }
    __syncthreads();
    return s_ok != 0;
}

// Calls f(t) for this warp's share of the turns 0 .. n - 1; all lanes make every call. The warps take turns. Where that
// would be more than kTurns each, they draw runs of kTurns turns from a counter instead: with fixed turns the SMs drift
// apart (a third of a phase on 15 images of 3840x2160 full of fragments), wait at the barrier, and the lists and groups
// in use at a time no longer fit the L2 (that call 76 ms with fixed turns, 54 with runs of 4 or 8, 57 of 2,
// 68 of 32).
constexpr uint32_t kTurns = 8;

template <class F>
__device__ __forceinline__ void for_turns(uint32_t n, int32_t* counter, F f) {
    const uint32_t warps = gridDim.x * (kRegionThreads / 32), w = blockIdx.x * (kRegionThreads / 32) + (threadIdx.x >> 5);
    const bool draw = n > warps * kTurns;
    uint32_t t = draw ? w * kTurns : w, left = kTurns;
    while (t < n) {
        f((int)t);
        if (!draw) {
            t += warps;
        } else if (--left > 0) {
            ++t;
        } else {
            uint32_t c = 0;
            if ((threadIdx.x & 31) == 0) c = warps + (uint32_t)atomicAdd(counter, 1);
            t = __shfl_sync(kFull, c, 0) * kTurns;
            left = kTurns;
        }
    }
}

// The same for n items (n < 2^31), 32 to a turn: f(base), items base .. base + 31, base < n.
template <class F>
__device__ __forceinline__ void for_items(int64_t n, int32_t* counter, F f) {
    for_turns((uint32_t)((n + 31) / 32), counter, [&](int t) { f(t * 32); });
}

// Calls f(image index, image, x, y0) for this warp's share of all images' 32 x 4 pixel tiles (column x of the lane, rows
// y0 .. y0 + 3; positions past the image's edges included); all lanes make every call.
template <class F>
__device__ __forceinline__ void for_tiles(const Scratch& s, int32_t* counter, F f) {
    const int lane = threadIdx.x & 31;
    for_turns((uint32_t)s.tiles, counter, [&](int t) {
        int lo = 0, hi = s.n_images - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s.img[mid].tile_base <= t) lo = mid;
            else hi = mid - 1;
        }
        const SegImage& im = s.img[lo];
        const int tw = (im.W + kTileW - 1) / kTileW, q = t - im.tile_base;
        f(lo, im, (q % tw) * kTileW + lane, (q / tw) * kTileH);
    });
}

// From the tile components to the labels, in one cooperative launch whose phases are separated by grid barriers: links
// across tiles, components and their main ones; groups start as single components (main components anchored with their label); then rounds of
//   pick    every unanchored group takes the 8-adjacent group of nearest mean colour. A pixel whose group is
//           anchored, or whose neighbours all lie in its own group, can never matter again (anchors are kept and
//           groups only merge): only the others enter the next round's list. Round 0 visits every pixel;
//   link    all picks at once (the round's unanchored roots with the groups they picked, found from the picked
//           group's name, which is one of its components);
//   merge   every unanchored root that now hangs under another root moves its sums and its name there;
//   finish  the round's roots point at their new roots; those still unanchored get their mean and form the next
//           round's list; anchored roots that gained members get their mean;
// until no group is unanchored; then every component points straight at its group's root and the labels are
// written. Four launches per possible round (the bound is the logarithm of the image, 18 to 23 rounds) cost a
// 480x270 image about 100 launches, most of them empty, of its 0.55 ms. The phases wait on dependent loads: 141 us for
// such an image (25 phases of 2 to 8 us, 1 us of them the barrier), 1.12 ms for eight of 1920x1080, a quarter of it the
// first pick (a third of these scenes' pixels lie outside their label's main component).
__global__ void __launch_bounds__(kRegionThreads, 1) regions_kernel(Scratch s) {
    __shared__ int2 s_buf[kRegionThreads / 32][kRun + 32];  // one list at a time
    uint32_t phase = 0;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, stride = gridDim.x * kRegionThreads;
    auto work = [&](int k) { return s.work + 2 * phase + k; };  // the phase's counters for for_items
    auto int_list = [&](int32_t* list, int32_t* counter) { return WarpList<int32_t, kRun>{reinterpret_cast<int32_t*>(s_buf[warp]), list, counter, 0}; };

    // links across the component tiles' borders: a tile's top row in three directions, its left column in two and its
    // right column in one, each a warp's task (a link waits on a chain of loads)
    for (int64_t task = blockIdx.x * (kRegionThreads / 32) + warp; task < 6 * (int64_t)s.ctiles;
         task += gridDim.x * (kRegionThreads / 32)) {
        const int t = (int)(task / 6), side = (int)(task - 6 * (int64_t)t);
        int lo = 0, hi = s.n_images - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s.img[mid].ctile_base <= t) lo = mid;
            else hi = mid - 1;
        }
        const SegImage& im = s.img[lo];
        const int W = im.W, H = im.H, tw = (W + kCTile - 1) / kCTile, q = t - im.ctile_base;
        const int x0 = (q % tw) * kCTile, y0 = (q / tw) * kCTile;
        auto link = [&](int x, int y, int dx, int dy) {
            const int px = x + dx, py = y + dy;
            if (x >= W || y >= H || px < 0 || px >= W || py < 0) return;
            const int32_t gp = im.pix_base + y * W + x, gq = im.pix_base + py * W + px;
            if (s.lab[gp] == s.lab[gq]) unite(s.par, gp, gq, s.status);
        };
        if (side < 3) link(x0 + lane, y0, side - 1, -1);
        else if (side == 3) link(x0, y0 + lane, -1, 0);
        else if (lane > 0) link(side == 4 ? x0 : x0 + kCTile - 1, y0 + lane, side == 4 ? -1 : 1, -1);
    }
    if (!grid_barrier(s, phase)) return;
    // the tile components' roots point at their component's name and add their sums there; the names are listed
    {
        const int n = __ldcg(&s.cnt[4 + 2 * s.rounds]);
        auto comps = int_list(s.comps, &s.cnt[0]);
        for_items(n, work(0), [&](int base) {
            const int i = base + lane;
            bool root = false;
            int32_t c = 0;
            if (i < n) {
                c = s.uroots[1][i];
                const int32_t r = find_root<true>(s.par, c, s.status);
                root = r == c;
                if (!root) {
                    const ulonglong2 t = s.csum[c];
                    s.par[c] = r;
                    atomicAdd(&s.csum[r].x, t.x);
                    atomicAdd(&s.csum[r].y, t.y);
                }
            }
            comps.append(root, c);
        });
        comps.finish();
    }
    if (!grid_barrier(s, phase)) return;
    // every component takes its index in the list and offers itself as its label's main component (the largest, the
    // earliest named on ties)
    const int n_comps = __ldcg(&s.cnt[0]);
    for_items(n_comps, work(0), [&](int base) {
        const int i = base + lane;
        if (i >= n_comps) return;
        const int32_t c = s.comps[i];
        const unsigned long long key = ((__ldcg(&s.csum[c].x) >> 40) << 32) | (unsigned long long)(~(uint32_t)c);
        atomicMax(&s.mainkey[s.lab[c]], key);
        s.par[c] = -1 - i;
    });
    if (!grid_barrier(s, phase)) return;
    // the groups, and every pixel's component index (a pixel's parent is its tile component's root, whose parent is
    // the component's name; four pixels per thread in flight)
    {
        auto orphans = int_list(s.uroots[0], &s.cnt[1]);
        for_items(n_comps, work(0), [&](int base) {
            const int i = base + lane;
            bool is_main = false;
            if (i < n_comps) {
                const int32_t c = s.comps[i];
                const int32_t k = s.lab[c];
                is_main = (uint32_t)(~s.mainkey[k]) == (uint32_t)c;
                const ulonglong2 t = __ldcg(&s.csum[c]);
                const unsigned long long n = t.x >> 40, sy = t.x & ((1ull << 40) - 1), scb = t.y >> 32,
                                         scr = t.y & 0xffffffffull;
                s.gpar[i] = i;
                s.glab[i] = is_main ? k : -1;
                s.gsum[i] = GSum{n, sy, scb, scr};
                s.gmean[i] = make_int4(mean16(sy, n), mean16(scb, n), mean16(scr, n), c);
                s.best[i] = kNone;
                s.dirty[i] = 0;
            }
            orphans.append(i < n_comps && !is_main, i);
        });
        orphans.finish();
    }
    for_items((s.pixels + 3) / 4, work(1), [&](int base) {
        const int64_t p0 = 4 * (int64_t)base + lane;
        int32_t r[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) r[k] = p0 + 32 * k < s.pixels ? s.par[p0 + 32 * k] : -1;
#pragma unroll
        for (int step = 0; step < 2; ++step)
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (r[k] >= 0) r[k] = s.par[r[k]];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (p0 + 32 * k < s.pixels) s.comp[p0 + 32 * k] = -1 - r[k];
    });
    if (!grid_barrier(s, phase)) return;
    for (int r = 0; r < s.rounds; ++r) {
        const int n_roots = __ldcg(&s.cnt[1 + r]);
        if (n_roots == 0) break;
        WarpList<int2, kRun> next{s_buf[warp], s.orph[(r + 1) & 1], &s.cnt[2 + s.rounds + r + 1], 0};
        if (r == 0) {
            // Every group is one component: no walks, and a pixel all of whose neighbours lie in its own component,
            // the common case, is done after loads that its warp shares: a lane holds four rows of a column and the
            // rows above and below, and takes its neighbours' columns by shuffles.
            for_tiles(s, work(0), [&](int k, const SegImage& im, int x, int y0) {
                const int W = im.W, H = im.H;
                const int32_t* comp = s.comp + im.pix_base;
                int32_t c[6], edge[6];  // rows y0 - 1 .. y0 + 4; edge: the column beyond the warp's, lanes 0 and 31
                const int xe = lane == 0 ? x - 1 : x + 1;
                const bool has_edge = (lane == 0 && x > 0) || (lane == 31 && x + 1 < W);
#pragma unroll
                for (int q = 0; q < 6; ++q) {
                    const int y = y0 - 1 + q;
                    const bool row = y >= 0 && y < H;
                    c[q] = row && x < W ? comp[(int64_t)y * W + x] : -1;
                    edge[q] = row && has_edge ? comp[(int64_t)y * W + xe] : -1;
                }
                int32_t l[6], r[6];
#pragma unroll
                for (int q = 0; q < 6; ++q) {
                    l[q] = __shfl_up_sync(kFull, c[q], 1);
                    r[q] = __shfl_down_sync(kFull, c[q], 1);
                    if (lane == 0) l[q] = edge[q];
                    if (lane == 31) r[q] = edge[q];
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int32_t pc = c[j + 1];
                    const int32_t g[8] = {l[j], c[j], r[j], l[j + 1], r[j + 1], l[j + 2], c[j + 2], r[j + 2]};
                    bool keep = false;
                    if (pc >= 0) {
                        bool other = false;
#pragma unroll
                        for (int q = 0; q < 8; ++q) other = other || (g[q] >= 0 && g[q] != pc);
                        if (other && s.glab[pc] < 0) {
                            const int4 ma = s.gmean[pc];
                            unsigned long long best = kNone;
#pragma unroll
                            for (int q = 0; q < 8; ++q)
                                if (g[q] >= 0 && g[q] != pc) best = min(best, pick_key(ma, s.gmean[g[q]]));
                            atomicMin(&s.best[pc], best);
                            keep = true;
                        }
                    }
                    next.append(keep, make_int2(im.pix_base + (y0 + j) * W + x, k));
                }
            });
        } else {
            const int n = __ldcg(&s.cnt[2 + s.rounds + r]);
            const int2* in = s.orph[r & 1];
            for_items(n, work(0), [&](int base) {
                const int i = base + lane;
                bool keep = false;
                int2 o = make_int2(0, 0);
                if (i < n) {
                    o = in[i];
                    const int32_t pc = s.comp[o.x];
                    const int32_t a = find_root(s.gpar, pc, s.status);
                    keep = s.glab[a] < 0 && pick_pixel(s, s.img[o.y], o.x, pc, a);
                }
                next.append(keep, o);
            });
        }
        next.finish();
        if (!grid_barrier(s, phase)) return;
        const int32_t* u = s.uroots[r & 1];
        for_items(n_roots, work(0), [&](int base) {
            if (base + lane >= n_roots) return;
            const int32_t c = u[base + lane];
            const unsigned long long b = s.best[c];
            if (b != kNone) unite_groups(s, c, s.comp[(uint32_t)b]);
        });
        if (!grid_barrier(s, phase)) return;
        auto dirty = int_list(s.dirty_list, &s.cnt[6 + 2 * s.rounds + r]);
        for_items(n_roots, work(0), [&](int base) {
            const int i = base + lane;
            bool first = false;
            int32_t t = 0;
            if (i < n_roots) {
                const int32_t c = u[i];
                t = find_root(s.gpar, c, s.status);
                if (t != c) {
                    const GSum g = s.gsum[c];
                    GSum* d = &s.gsum[t];
                    atomicAdd(&d->n, g.n);
                    atomicAdd(&d->c0, g.c0);
                    atomicAdd(&d->c1, g.c1);
                    atomicAdd(&d->c2, g.c2);
                    atomicMin(&s.gmean[t].w, s.gmean[c].w);
                    if (s.glab[t] >= 0) first = atomicExch(&s.dirty[t], 1) == 0;
                }
            }
            dirty.append(first, t);
        });
        dirty.finish();
        if (!grid_barrier(s, phase)) return;
        auto left = int_list(s.uroots[(r + 1) & 1], &s.cnt[2 + r]);
        for_items(n_roots, work(0), [&](int base) {
            const int i = base + lane;
            bool keep = false;
            int32_t c = 0;
            if (i < n_roots) {
                c = u[i];
                s.best[c] = kNone;
                const int32_t t = find_root(s.gpar, c, s.status);
                s.gpar[c] = t;
                if (t == c) {
                    set_mean(s, c);
                    keep = true;
                }
            }
            left.append(keep, c);
        });
        left.finish();
        const int n_dirty = __ldcg(&s.cnt[6 + 2 * s.rounds + r]);
        for (int i = blockIdx.x * kRegionThreads + tid; i < n_dirty; i += stride) {
            const int32_t t = s.dirty_list[i];
            s.dirty[t] = 0;
            set_mean(s, t);
        }
        if (!grid_barrier(s, phase)) return;
    }
    if (blockIdx.x == 0 && tid == 0 && __ldcg(&s.cnt[1 + s.rounds]) != 0) atomicOr(s.status, SP_ROUND_CAP);
    // every component takes its group's label (an anchored root keeps its own; it is not written here)
    for_items(n_comps, work(0), [&](int base) {
        const int i = base + lane;
        if (i >= n_comps) return;
        const int32_t t = find_root(s.gpar, i, s.status);
        if (t != i) s.glab[i] = s.glab[t];
    });
    if (!grid_barrier(s, phase)) return;
    for_tiles(s, work(0), [&](int, const SegImage& im, int x, int y0) {
        if (x >= im.W) return;
        const int W = im.W, H = im.H, base = im.pix_base + y0 * W + x;
        int32_t g[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) g[j] = y0 + j < H ? s.comp[base + j * W] : -1;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (g[j] >= 0) g[j] = s.glab[g[j]];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (y0 + j < H) im.out[(int64_t)(y0 + j) * W + x] = (g[j] >= 0 ? g[j] : s.lab[base + j * W]) - im.seg_base;
    });
}

}  // namespace

struct ftv_segmenter {
    int device = 0;
    int n_images = 0, sb = 1, bd = 8, S = 1, m = 0, T = 1;
    std::vector<SegImage> h_meta;  // sizes and bases (pointers filled per call)
    int64_t P = 0;
    int32_t K = 0;
    int max_W = 0, max_H = 0, rounds = 0, dist_mode = 0;
    size_t assign_smem = 0;
    int region_blocks = 0;  // CTAs of the cooperative launch: all that stay resident
    int groups = 1;         // row groups per thread of an assignment pass
    unsigned long long wc = 0, ws = 0;
    SegImage* h_img = nullptr;  // pinned staging of the per-call descriptors
    SegImage* d_img = nullptr;
    Scratch sc{};
    std::vector<void*> blocks;  // every device allocation, freed at destroy
    cudaEvent_t staged = nullptr;
    int64_t launches = 0;
    bool profiling = false;
    std::vector<cudaEvent_t> ev;  // profiling: call begin, call end, then a pair per assignment pass
    bool timed = false;
};

namespace {

// Counter words of a segmenter: the lists' and the barrier's, then two for each phase of regions_kernel (four barriers
// before the rounds, four in a round, one after).
size_t counters(int rounds) { return (size_t)(3 * rounds + 8) + 2 * (size_t)(4 * rounds + 6); }

template <class T>
bool dalloc(ftv_segmenter* g, T** p, size_t n) {
    void* q = nullptr;
    if (cudaMalloc(&q, sizeof(T) * std::max<size_t>(n, 1)) != cudaSuccess) return false;
    g->blocks.push_back(q);
    *p = static_cast<T*>(q);
    return true;
}

void release(ftv_segmenter* g) {
    for (void* q : g->blocks) cudaFree(q);
    g->blocks.clear();
    if (g->h_img) cudaFreeHost(g->h_img);
    if (g->staged) cudaEventDestroy(g->staged);
    for (cudaEvent_t e : g->ev) cudaEventDestroy(e);
    delete g;
}

// The rows of a group are compiled in: with five for all, steps of one and two pixels leave most of a thread's
// comparisons unused (8 images of 1920x1080, 12 bits, 10 passes: step 1 17.9 -> 13.7 ms, step 2 7.9 -> 5.3). Images small enough
// for one group per thread wait on the chain of passes instead and keep the one form.
template <int D, int SB>
const void* assign_function_of(int groups, int rows) {
    if (groups == 1) return reinterpret_cast<const void*>(assign_kernel<D, SB, 1, kPY>);
    if (rows == 1) return reinterpret_cast<const void*>(assign_kernel<D, SB, kAGroups, 1>);
    if (rows == 2) return reinterpret_cast<const void*>(assign_kernel<D, SB, kAGroups, 2>);
    return reinterpret_cast<const void*>(assign_kernel<D, SB, kAGroups, kPY>);
}

const void* assign_function(int dist_mode, int sb, int groups, int rows) {
    switch (dist_mode) {
        case DIST_DOT32: return sb == 1 ? assign_function_of<DIST_DOT32, 1>(groups, rows) : assign_function_of<DIST_DOT32, 2>(groups, rows);
        case DIST_NARROW: return sb == 1 ? assign_function_of<DIST_NARROW, 1>(groups, rows) : assign_function_of<DIST_NARROW, 2>(groups, rows);
        case DIST_WIDE: return sb == 1 ? assign_function_of<DIST_WIDE, 1>(groups, rows) : assign_function_of<DIST_WIDE, 2>(groups, rows);
        default: return sb == 1 ? assign_function_of<DIST_WIDE_COLOUR, 1>(groups, rows) : assign_function_of<DIST_WIDE_COLOUR, 2>(groups, rows);
    }
}

}  // namespace

extern "C" ftv_status ftv_segmenter_init(const ftv_segmenter_config* cfg, ftv_segmenter** out) {
    if (!cfg || !out) return FTV_ERR_INVALID_ARG;
    *out = nullptr;
    if (cfg->n_images < 1 || cfg->n_images > FTV_SEG_MAX_IMAGES || !cfg->widths || !cfg->heights)
        return FTV_ERR_INVALID_ARG;
    if (cfg->sample_bytes != 1 && cfg->sample_bytes != 2) return FTV_ERR_INVALID_ARG;
    if (cfg->bit_depth < 1 || cfg->bit_depth > 8 * cfg->sample_bytes) return FTV_ERR_INVALID_ARG;
    if (cfg->grid_step < 1 || cfg->grid_step > FTV_SEG_MAX_STEP) return FTV_ERR_INVALID_ARG;
    if (cfg->compactness < 0 || cfg->compactness > 255) return FTV_ERR_INVALID_ARG;
    if (cfg->iterations < 1 || cfg->iterations > 64) return FTV_ERR_INVALID_ARG;
    auto* g = new ftv_segmenter();
    g->n_images = cfg->n_images;
    g->sb = cfg->sample_bytes;
    g->bd = cfg->bit_depth;
    g->S = cfg->grid_step;
    g->m = cfg->compactness;
    g->T = cfg->iterations;
    int64_t P = 0, K = 0, tiles = 0, ctiles = 0;
    for (int i = 0; i < g->n_images; ++i) {
        const int W = cfg->widths[i], H = cfg->heights[i];
        if (W < 1 || H < 1 || W > FTV_MAX_DIM || H > FTV_MAX_DIM) {
            delete g;
            return FTV_ERR_INVALID_ARG;
        }
        SegImage m{};
        m.W = W;
        m.H = H;
        m.gw = (W + g->S - 1) / g->S;
        m.gh = (H + g->S - 1) / g->S;
        m.K = m.gw * m.gh;
        m.pix_base = (int32_t)std::min<int64_t>(P, INT32_MAX);
        m.seg_base = (int32_t)std::min<int64_t>(K, INT32_MAX);
        m.tile_base = (int32_t)std::min<int64_t>(tiles, INT32_MAX);
        P += (int64_t)W * H;
        K += m.K;
        m.ctile_base = (int32_t)std::min<int64_t>(ctiles, INT32_MAX);
        tiles += (int64_t)((W + kTileW - 1) / kTileW) * ((H + kTileH - 1) / kTileH);
        ctiles += (int64_t)((W + kCTile - 1) / kCTile) * ((H + kCTile - 1) / kCTile);
        g->max_W = std::max(g->max_W, W);
        g->max_H = std::max(g->max_H, H);
        g->h_meta.push_back(m);
    }
    // global pixel names must fit 31 bits (component names are packed into 32-bit key halves)
    if (P >= INT32_MAX || K >= INT32_MAX || tiles >= INT32_MAX) {
        delete g;
        return FTV_ERR_INVALID_ARG;
    }
    g->P = P;
    g->K = (int32_t)K;
    g->wc = (unsigned long long)g->S * g->S;
    g->ws = (unsigned long long)g->m * g->m;
    if (g->bd > 8) g->ws <<= 2 * (g->bd - 8);
    if (g->bd < 8) g->wc <<= 2 * (8 - g->bd);
    // unanchored groups at least halve every round
    int64_t maxP = 0;
    for (const auto& m : g->h_meta) maxP = std::max<int64_t>(maxP, (int64_t)m.W * m.H);
    int rounds = 1;
    while ((1LL << (rounds - 1)) < maxP) ++rounds;
    g->rounds = rounds + 1;
    cudaGetDevice(&g->device);

    Scratch& s = g->sc;
    bool ok = cudaMallocHost(reinterpret_cast<void**>(&g->h_img), sizeof(SegImage) * g->n_images) == cudaSuccess;
    ok = ok && cudaEventCreateWithFlags(&g->staged, cudaEventDisableTiming) == cudaSuccess;
    ok = ok && dalloc(g, &g->d_img, g->n_images);
    ok = ok && dalloc(g, &s.cen[0], K) && dalloc(g, &s.cen[1], K) && dalloc(g, &s.mainkey, K);
    ok = ok && dalloc(g, &s.sums[0], K) && dalloc(g, &s.sums[1], K) && dalloc(g, &s.sums[2], K);
    ok = ok && dalloc(g, &s.lab, P) && dalloc(g, &s.par, P) && dalloc(g, &s.comp, P) && dalloc(g, &s.csum, P);
    ok = ok && dalloc(g, &s.comps, P) && dalloc(g, &s.gpar, P) && dalloc(g, &s.glab, P) && dalloc(g, &s.gsum, P) &&
         dalloc(g, &s.gmean, P);
    ok = ok && dalloc(g, &s.best, P) && dalloc(g, &s.orph[0], P) && dalloc(g, &s.orph[1], P);
    ok = ok && dalloc(g, &s.uroots[0], P) && dalloc(g, &s.uroots[1], P) && dalloc(g, &s.dirty, P) &&
         dalloc(g, &s.dirty_list, P);
    ok = ok && dalloc(g, &s.cnt, counters(g->rounds)) && dalloc(g, &s.status, 1);
    ok = ok && cudaMemset(s.status, 0, sizeof(uint32_t)) == cudaSuccess;
    ok = ok && ftv::finish_setup() == cudaSuccess;
    if (!ok) {
        release(g);
        cudaGetLastError();
        return FTV_ERR_OUT_OF_MEMORY;
    }
    s.img = g->d_img;
    s.barrier = reinterpret_cast<uint32_t*>(s.cnt + 2 * g->rounds + 5);
    s.work = s.cnt + 3 * g->rounds + 8;
    s.polls = kBarrierPolls;
    s.n_images = g->n_images;
    s.tiles = (int32_t)tiles;
    s.ctiles = (int32_t)ctiles;
    s.pixels = P;
    int per_sm = 0, sms = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, regions_kernel, kRegionThreads, 0) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, g->device) != cudaSuccess || per_sm < 1) {
        release(g);
        return FTV_ERR_CUDA;
    }
    // four warps to a pixel tile, for images too small to fill the chip (a barrier of few CTAs costs no less)
    g->region_blocks = (int)std::min<int64_t>((int64_t)per_sm * sms, std::max<int64_t>(1, 4 * tiles * 32 / kRegionThreads));
    s.S = g->S;
    s.sb = g->sb;
    s.rounds = g->rounds;
    s.wc = g->wc;
    s.ws = g->ws;
    // Distance arithmetic. |x - X| < 3S in pixels for every candidate (a candidate's pixels, hence its
    // mean, lie within one cell of the candidate's cell), so in 1/16 units dsp < 2 (48 S)^2, and
    // dcol <= 3 (16 (2^bd - 1))^2 for samples within the bit depth. In the DOT32 form positions are
    // relative to the tile (64 columns, at most 20 rows and the one that the row term steps past them),
    // |position| <= 16 (63 + 3S) = R, and every partial sum is bounded by wc' 3 vmax^2 + ws' 6 R^2.
    {
        const unsigned long long gcd = std::gcd(g->wc, g->ws);
        const unsigned long long wcn = g->wc / gcd, wsn = g->ws / gcd;
        const unsigned long long vmax = 16ull * ((1ull << g->bd) - 1), dmax = 48ull * g->S;
        const unsigned long long R = 16ull * (kATileW - 1 + 3ull * g->S);
        const unsigned long long direct = wcn * 3ull * vmax * vmax + wsn * 2ull * dmax * dmax;
        const unsigned long long dot = wcn * 3ull * vmax * vmax + wsn * 6ull * R * R;
        g->dist_mode = dot < (1ull << 31) ? DIST_DOT32
                       : direct < (1ull << 32) ? DIST_NARROW
                       : (g->bd <= 11 ? DIST_WIDE : DIST_WIDE_COLOUR);
        s.wcn = (uint32_t)(g->dist_mode <= DIST_NARROW ? wcn : 0);
        s.wsn = (uint32_t)(g->dist_mode <= DIST_NARROW ? wsn : 0);
    }
    // row groups of a cell row: as few as kPY rows each allow, of equal size
    s.G = (g->S + kPY - 1) / kPY;
    s.PY = (g->S + s.G - 1) / s.G;
    s.packed = g->bd <= 10;
    // shared memory of an assignment tile: the cells it can see (kAGroups consecutive groups, from a multiple of
    // kAGroups, touch at most ceil((kAGroups - 1) / G) + 1 cell rows), 52 bytes each. At most 66 x 6 cells (step 1), 20.6
    // KB: below what every launch may ask for, so that no limit is set. A limit would belong to the kernel, and the
    // next segmenter's would replace it.
    {
        // One group per thread while the tiles of kAGroups would not give every SM a few warps: 480x270, 10 passes,
        // 72 against 125 us; 8 x 1920x1080, 1300 against 1010 us.
        int64_t ctas = 0;
        for (const auto& m : g->h_meta)
            ctas += (int64_t)((m.W + kATileW - 1) / kATileW) * ((m.gh * s.G + kAGroups - 1) / kAGroups);
        g->groups = ctas < 8 * sms ? 1 : kAGroups;
        const int ncx = (kATileW - 1 + g->S - 1) / g->S + 3, ncy = (g->groups - 1 + s.G - 1) / s.G + 3;
        s.max_cells = ncx * ncy;
        g->assign_smem = (size_t)s.max_cells * (2 * sizeof(int4) + 5 * sizeof(uint32_t));
    }
    *out = g;
    return FTV_OK;
}

extern "C" ftv_status ftv_segmenter_segments(const ftv_segmenter* g, int32_t* n_segments) {
    if (!g || !n_segments) return FTV_ERR_INVALID_ARG;
    for (int i = 0; i < g->n_images; ++i) n_segments[i] = g->h_meta[i].K;
    return FTV_OK;
}

extern "C" ftv_status ftv_superpixels(ftv_segmenter* g, const void* const* d_planes, const int64_t* pitch_bytes,
                                      int32_t* const* d_labels, ftv_stream stream) {
    if (!g || !d_planes || !pitch_bytes || !d_labels) return FTV_ERR_INVALID_ARG;
    for (int i = 0; i < g->n_images; ++i) {
        if (!d_labels[i]) return FTV_ERR_INVALID_ARG;
        for (int c = 0; c < 3; ++c)
            if (!d_planes[3 * i + c] || pitch_bytes[3 * i + c] < (int64_t)g->h_meta[i].W * g->sb)
                return FTV_ERR_INVALID_ARG;
    }
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != g->device) cudaSetDevice(g->device);
    ftv::NvtxRange range("ftv_superpixels");
    cudaStream_t st = (cudaStream_t)stream;
    // the staging copy of the previous call must have left before it is rewritten
    if (cudaEventSynchronize(g->staged) != cudaSuccess) {
        if (prev >= 0 && prev != g->device) cudaSetDevice(prev);
        return FTV_ERR_CUDA;
    }
    for (int i = 0; i < g->n_images; ++i) {
        SegImage m = g->h_meta[i];
        for (int c = 0; c < 3; ++c) {
            m.plane[c] = d_planes[3 * i + c];
            m.pitch[c] = pitch_bytes[3 * i + c];
        }
        m.out = d_labels[i];
        g->h_img[i] = m;
    }
    Scratch& s = g->sc;
    cudaError_t e = cudaMemcpyAsync(g->d_img, g->h_img, sizeof(SegImage) * g->n_images, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaEventRecord(g->staged, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(s.cnt, 0, sizeof(int32_t) * counters(g->rounds), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(s.sums[0], 0, sizeof(Sums) * (size_t)g->K, st);
    if (e != cudaSuccess) {
        if (prev >= 0 && prev != g->device) cudaSetDevice(prev);
        return FTV_ERR_CUDA;
    }
    const dim3 cgrid((g->max_W + kCTile - 1) / kCTile, (g->max_H + kCTile - 1) / kCTile, g->n_images);
    const int groups = (g->max_H + g->S - 1) / g->S * s.G;
    const dim3 agrid((g->max_W + kATileW - 1) / kATileW, (groups + g->groups - 1) / g->groups, g->n_images);
    int64_t n = 0;
    const bool prof = g->profiling;
    if (prof) cudaEventRecord(g->ev[0], st);
    for (int it = 0; it < g->T && e == cudaSuccess; ++it) {
        const int acc = it + 1 < g->T, last = it + 1 == g->T;
        if (prof) cudaEventRecord(g->ev[2 + 2 * it], st);
        int pass = it, add = acc, end = last;
        void* args[] = {&s, &pass, &add, &end};
        e = cudaLaunchKernel(assign_function(g->dist_mode, g->sb, g->groups, s.PY), agrid, dim3(kATileW), args, g->assign_smem, st);
        if (prof) cudaEventRecord(g->ev[3 + 2 * it], st);
        ++n;
    }
    components_kernel<<<cgrid, kThreads, 0, st>>>(s);
    n += 1;
    void* args[] = {&s};
    if (e == cudaSuccess)
        e = cudaLaunchCooperativeKernel(reinterpret_cast<void*>(regions_kernel), dim3(g->region_blocks), dim3(kRegionThreads), args, 0, st);
    n += 1;
    if (prof) cudaEventRecord(g->ev[1], st);
    g->timed = g->timed || prof;
    g->launches += n;
    const cudaError_t e2 = cudaGetLastError();
    if (e == cudaSuccess) e = e2;
    if (prev >= 0 && prev != g->device) cudaSetDevice(prev);
    return e == cudaSuccess ? FTV_OK : FTV_ERR_CUDA;
}

extern "C" ftv_status ftv_segmenter_check(ftv_segmenter* g, ftv_stream stream) {
    if (!g) return FTV_ERR_INVALID_ARG;
    if (cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) return FTV_ERR_CUDA;
    uint32_t st = 0;
    if (cudaMemcpy(&st, g->sc.status, sizeof(st), cudaMemcpyDeviceToHost) != cudaSuccess) return FTV_ERR_CUDA;
    if (st && cudaMemset(g->sc.status, 0, sizeof(st)) != cudaSuccess) return FTV_ERR_CUDA;
    return st ? FTV_ERR_TIMEOUT : FTV_OK;
}

extern "C" ftv_status ftv_segmenter_set_poll_limit(ftv_segmenter* g, int32_t polls) {
    if (!g || polls < 0) return FTV_ERR_INVALID_ARG;
    g->sc.polls = polls > 0 ? polls : kBarrierPolls;
    return FTV_OK;
}

extern "C" int64_t ftv_segmenter_launch_count(const ftv_segmenter* g) { return g ? g->launches : 0; }

extern "C" ftv_status ftv_segmenter_set_profiling(ftv_segmenter* g, int32_t enable) {
    if (!g) return FTV_ERR_INVALID_ARG;
    if (enable && g->ev.empty()) {
        g->ev.resize(2 + 2 * g->T, nullptr);
        for (auto& e : g->ev)
            if (cudaEventCreate(&e) != cudaSuccess) return FTV_ERR_CUDA;
    }
    g->profiling = enable != 0;
    return FTV_OK;
}

extern "C" ftv_status ftv_segmenter_kernel_ms(ftv_segmenter* g, float* assign_ms, float* total_ms) {
    if (!g || (!assign_ms && !total_ms)) return FTV_ERR_INVALID_ARG;
    if (!g->timed) return FTV_ERR_STATE;
    if (cudaEventSynchronize(g->ev[1]) != cudaSuccess) return FTV_ERR_CUDA;
    float ms = 0.f, sum = 0.f;
    for (int it = 0; it < g->T; ++it) {
        if (cudaEventElapsedTime(&ms, g->ev[2 + 2 * it], g->ev[3 + 2 * it]) != cudaSuccess) return FTV_ERR_CUDA;
        sum += ms;
    }
    if (assign_ms) *assign_ms = sum / g->T;
    if (total_ms) {
        if (cudaEventElapsedTime(&ms, g->ev[0], g->ev[1]) != cudaSuccess) return FTV_ERR_CUDA;
        *total_ms = ms;
    }
    return FTV_OK;
}

extern "C" ftv_status ftv_segmenter_destroy(ftv_segmenter* g) {
    if (!g) return FTV_ERR_INVALID_ARG;
    cudaEventSynchronize(g->staged);
    release(g);
    return FTV_OK;
}
