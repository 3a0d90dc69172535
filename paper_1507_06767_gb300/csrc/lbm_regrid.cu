// Regridding of one refinement level from the Knudsen sensor (Sec. 5.2): tags, buffer cells,
// proper nesting, Berger-Rigoutsos point clustering.
//
// The per-cell work runs on the GPU: tagging (max of the sensor over a tag cell against the
// threshold), the buffer (a Chebyshev-ball dilation, done as three 1-D passes since the ball is a
// product of segments), the nesting mask (the dual erosion, positions beyond a non-periodic edge
// counting as covered) and, for every round of candidate boxes, the slab counts (signatures)
// along each axis.  The cut decisions need only the signatures; the kernel that counts them makes
// them, or the host between rounds where there are too many boxes for that: shrink to the tags'
// bounding box, accept at the efficiency, else cut at the hole nearest the centre, else at the
// strongest inflection of the signature, else bisect the longest axis; cuts leaving a piece narrower
// than min_width are not admissible.  Boxes of one round are disjoint, so a round costs one pass over
// at most the tag grid.
#include <cuda_runtime.h>
#include <math.h>
#include <limits.h>
#include <stddef.h>
#include <stdint.h>
#include <stdlib.h>

#include <algorithm>
#include <new>
#include <vector>

#include "../../include/lbm.h"
#include "lbm_internal.h"
#include "lbm_traits.cuh"

namespace lbm {
namespace rg {

namespace {

constexpr int SIG_XCHUNK = 1024;  // x extent of one signature work item
constexpr int SIG_CELLS = 16384;  // cells of one signature work item (at most)
constexpr int SIG_THREADS = 256;

struct SigItem {
    int box, z, y0, y1, x0, x1;
};
struct SigBox {
    int lo[3];
    int w, h, off;  // sig x at off, y at off + w, z at off + w + h
};

template <class T>
__global__ void k_tag(const T *__restrict__ K, int nx, int ny, int nz, int r, int rz, int tx,
                      int ty, long long ntag, double thr, uint8_t *__restrict__ tags) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ntag) return;
    const int x = (int)(t % tx), y = (int)((t / tx) % ty), z = (int)(t / ((long long)tx * ty));
    const int x0 = x * r, y0 = y * r, z0 = z * rz;
    const int x1 = min(x0 + r, nx), y1 = min(y0 + r, ny), z1 = min(z0 + rz, nz);
    uint8_t hit = 0;
    for (int cz = z0; cz < z1 && !hit; ++cz)
        for (int cy = y0; cy < y1 && !hit; ++cy) {
            const T *row = K + ((size_t)cz * ny + cy) * nx;
            for (int cx = x0; cx < x1; ++cx) {
                const double v = (double)row[cx];
                if (v > thr || v != v) {
                    hit = 1;
                    break;
                }
            }
        }
    tags[t] = hit;
}

// The same for FP32 fields whose tag cells span whole groups of 4 cells along x (r % 4 == 0,
// nx % 4 == 0): 16-byte loads, all of a row's loads issued before any test.  thr_f is the largest
// float not above the double threshold, so v > thr_f decides exactly as (double)v > thr, without
// the FP64 pipe (a small fraction of the FP32 rate on this GPU).
__global__ void k_tag_f4(const float *__restrict__ K, int nx, int ny, int nz, int r, int rz,
                         int tx, int ty, long long ntag, float thr_f, uint8_t *__restrict__ tags) {
    const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;  // fewer tags than cells, which fit an int
    if (t >= ntag) return;
    const int x = t % tx, y = t / tx % ty, z = t / tx / ty;
    const int x0 = x * r, y0 = y * r, z0 = z * rz;
    const int x1 = min(x0 + r, nx), y1 = min(y0 + r, ny), z1 = min(z0 + rz, nz);
    int hit = 0;
    for (int cz = z0; cz < z1; ++cz)
#pragma unroll 4
        for (int cy = y0; cy < y1; ++cy) {
            const float4 *row = reinterpret_cast<const float4 *>(K + ((size_t)cz * ny + cy) * nx);
            for (int c4 = x0 / 4; c4 < x1 / 4; ++c4) {
                const float4 v = __ldg(row + c4);
                // NaN fails every comparison: !(v <= thr_f) is true for v > thr_f and for NaN
                hit |= !(v.x <= thr_f) | !(v.y <= thr_f) | !(v.z <= thr_f) | !(v.w <= thr_f);
            }
        }
    tags[t] = (uint8_t)(hit != 0);
}

// One 1-D pass along an axis of extent n and element stride `stride`: dilation (op 0: OR over the
// segment, nothing beyond a non-periodic edge) or erosion (op 1: AND over the segment, covered
// beyond a non-periodic edge).  Periodic axes wrap.
__global__ void k_morph(const uint8_t *__restrict__ in, uint8_t *__restrict__ out, long long total,
                        int n, long long stride, int radius, int periodic, int op) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= total) return;
    const int c = (int)((t / stride) % n);
    int acc = op;  // OR starts at 0, AND at 1
    for (int k = -radius; k <= radius; ++k) {
        int cc = c + k;
        if (cc < 0 || cc >= n) {
            if (!periodic) continue;  // beyond the edge: 0 for OR, 1 for AND, neither changes acc
            cc = ((cc % n) + n) % n;
        }
        const int v = in[t + (long long)(cc - c) * stride] != 0;
        acc = op ? (acc & v) : (acc | v);
    }
    out[t] = (uint8_t)acc;
}

__global__ void k_and(uint8_t *__restrict__ tags, const uint8_t *__restrict__ mask,
                      long long total) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < total) tags[t] = (uint8_t)(tags[t] && mask[t]);
}

__global__ void k_normalise(uint8_t *m, long long total) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < total) m[t] = (uint8_t)(m[t] != 0);
}

// Slab counts of one work item (a z plane, a run of rows, a run of x) of one box: one warp per
// row, x counts in shared memory, row counts written directly (each row belongs to one warp), the
// plane count added once per CTA.
__global__ void __launch_bounds__(SIG_THREADS)
    k_signatures(const uint8_t *__restrict__ tags, int tx, int ty, const SigItem *__restrict__ items,
                 const SigBox *__restrict__ boxes, int *__restrict__ sig) {
    __shared__ int sx[SIG_XCHUNK];
    __shared__ int sy[SIG_XCHUNK];
    __shared__ int plane;
    const SigItem it = items[blockIdx.x];
    const SigBox b = boxes[it.box];
    const int cw = it.x1 - it.x0, ch = it.y1 - it.y0;
    for (int i = threadIdx.x; i < SIG_XCHUNK; i += blockDim.x) sx[i] = 0;
    if (threadIdx.x == 0) plane = 0;
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    int cnt = 0;
    for (int y = warp; y < ch; y += nw) {
        const uint8_t *row = tags + ((size_t)it.z * ty + it.y0 + y) * tx + it.x0;
        int rc = 0;
        for (int x = lane; x < cw; x += 32) {
            const int v = row[x];
            if (v) atomicAdd(&sx[x], 1);
            rc += v;
        }
        rc = __reduce_add_sync(0xffffffffu, rc);
        if (lane == 0) sy[y] = rc;
        cnt += rc;
    }
    if (lane == 0 && cnt) atomicAdd(&plane, cnt);
    __syncthreads();
    for (int i = threadIdx.x; i < cw; i += blockDim.x)
        if (sx[i]) atomicAdd(&sig[b.off + it.x0 - b.lo[0] + i], sx[i]);
    for (int i = threadIdx.x; i < ch; i += blockDim.x)
        if (sy[i]) atomicAdd(&sig[b.off + b.w + it.y0 - b.lo[1] + i], sy[i]);
    if (threadIdx.x == 0 && plane) atomicAdd(&sig[b.off + b.w + b.h + it.z - b.lo[2]], plane);
}

inline unsigned nblk(long long n, int t) { return (unsigned)((n + t - 1) / t); }

// The largest float whose value does not exceed t (t itself if it is a float; NaN stays NaN).
inline float float_at_most(double t) {
    float f = (float)t;
    if ((double)f > t) f = nextafterf(f, -INFINITY);
    return f;
}

struct HBox {
    int lo[3], hi[3];
};

// Host side of one box: trim to the tags, then accept or cut.  Returns 0 (drop), 1 (accept,
// `box` trimmed) or 2 (cut into lower / upper).
int decide(HBox &box, const int *sx, const int *sy, const int *sz, double efficiency, int wmin,
           HBox *lower, HBox *upper) {
    const int *s[3] = {sx, sy, sz};
    int len[3];
    int first[3], last[3];
    long long total = 0;
    for (int a = 0; a < 3; ++a) {
        len[a] = box.hi[a] - box.lo[a];
        first[a] = -1;
        last[a] = -1;
        for (int i = 0; i < len[a]; ++i)
            if (s[a][i]) {
                if (first[a] < 0) first[a] = i;
                last[a] = i;
            }
    }
    for (int i = 0; i < len[0]; ++i) total += s[0][i];
    if (total == 0) return 0;
    const int *sig[3];
    for (int a = 0; a < 3; ++a) {
        sig[a] = s[a] + first[a];
        box.hi[a] = box.lo[a] + last[a] + 1;
        box.lo[a] += first[a];
        len[a] = last[a] - first[a] + 1;
    }
    const double vol = (double)len[0] * (double)len[1] * (double)len[2];
    if ((double)total >= efficiency * vol) return 1;

    int cut_axis = -1, cut_at = 0;
    // holes: least |2p - L|, then longer axis, lower axis, lower p
    long long bd = 0;
    int bl = 0;
    for (int a = 0; a < 3; ++a)
        for (int p = wmin; p <= len[a] - wmin; ++p) {
            if (p >= len[a] || sig[a][p] != 0) continue;
            const long long d = llabs(2LL * p - len[a]);
            const bool better = cut_axis < 0 || d < bd || (d == bd && len[a] > bl);
            if (better) {  // equal d and length: the earlier (axis, p) stays
                cut_axis = a;
                cut_at = p;
                bd = d;
                bl = len[a];
            }
        }
    if (cut_axis < 0) {
        // inflections: strongest |D[i+1] - D[i]| at a strict sign change, then as for holes
        long long bs = -1;
        for (int a = 0; a < 3; ++a) {
            const int *q = sig[a];
            for (int i = 1; i <= len[a] - 3; ++i) {
                const long long d0 = (long long)q[i - 1] - 2LL * q[i] + q[i + 1];
                const long long d1 = (long long)q[i] - 2LL * q[i + 1] + q[i + 2];
                if (!((d0 < 0 && d1 > 0) || (d0 > 0 && d1 < 0))) continue;
                const int p = i + 1;
                if (p < wmin || len[a] - p < wmin) continue;
                const long long st = llabs(d1 - d0);
                const long long d = llabs(2LL * p - len[a]);
                const bool better = cut_axis < 0 || st > bs ||
                                    (st == bs && (d < bd || (d == bd && len[a] > bl)));
                if (better) {
                    cut_axis = a;
                    cut_at = p;
                    bs = st;
                    bd = d;
                    bl = len[a];
                }
            }
        }
    }
    if (cut_axis < 0) {
        // bisection of the longest admissible axis (ties: lower axis)
        for (int a = 0; a < 3; ++a) {
            const int p = len[a] / 2;
            if (p < wmin || len[a] - p < wmin) continue;
            if (cut_axis < 0 || len[a] > bl) {
                cut_axis = a;
                cut_at = p;
                bl = len[a];
            }
        }
    }
    if (cut_axis < 0) return 1;
    *lower = box;
    *upper = box;
    lower->hi[cut_axis] = box.lo[cut_axis] + cut_at;
    upper->lo[cut_axis] = box.lo[cut_axis] + cut_at;
    return 2;
}

// ---- clustering on the device
//
// The boxes of a round are trimmed, accepted or cut by the kernel itself, so the rounds follow each
// other in the stream without the host.  The CTAs of a launch share the round's boxes evenly: a box
// is counted by `parts` CTAs, each taking a run of its rows, and the one that comes last decides (no
// CTA waits for another).  The decisions are those of decide(), over the same integers and the one
// product of doubles, so the boxes are the same.  Of a regrid of 64^3 tags in 12 rounds with its level
// map, 732 us, 132 us were kernels, the rest uploads, downloads and waits between the rounds and
// allocations; with the rounds and the buffers kept on the device it takes 280 us.  A round overlaps its
// start with the end of the one before, as most rounds of a regrid of few boxes have nothing to do: one
// box of 128^2 tags takes 90 us, 138 without the overlap and 121 with the rounds on the host; 175 boxes of
// 64^3 tags 359, 449 and 1042.
constexpr int CL_THREADS = 256;
constexpr int CL_CTAS = 608;         // four to an SM
constexpr int CL_MAX_PARTS = 152;    // CTAs of one box: each adds its x counts to the same few words
constexpr int CL_EXTENTS = 8192;     // extents of the tag grid in all: a box's signatures in shared memory
constexpr int CL_ROUNDS = 16;        // launches queued before the host looks (even: the queues alternate)
constexpr int CL_BOXES = 8192;       // boxes of a round at most, and accepted ones
constexpr int CL_SIG = 1 << 19;      // signature words of a round at most

struct DBox {
    int lo[3], hi[3];
    int off;      // signatures x, y, z in the round's pool
    int arrived;  // CTAs done counting
};
struct ClusterState {
    int count[CL_ROUNDS + 1];  // boxes of each round
    int used[CL_ROUNDS + 1];   // signature words of each round
    int accepted;
    int overflow;              // a queue or pool was too small: the host, which alone reads this,
                               // clusters instead
    long long tagged;
    HBox boxes[CL_BOXES];      // the accepted ones
};
struct ClusterWork {
    ClusterState state;
    DBox queue[2][CL_BOXES];
    int sig[2][CL_SIG];        // zero where no box of the current round counts
};
// What the host reads after a batch of rounds, with the first boxes in the same copy.
constexpr int CL_FIRST_BOXES = 1024;
constexpr size_t CL_HEAD = offsetof(ClusterState, boxes) + sizeof(HBox) * CL_FIRST_BOXES;

// The first batch starts from the whole tag grid, a later one from the boxes the last one left.
__global__ void k_cluster_start(ClusterWork *w, int tx, int ty, int tz, bool first) {
    ClusterState &s = w->state;
    const int left = s.count[CL_ROUNDS], used = s.used[CL_ROUNDS];
    for (int k = 0; k <= CL_ROUNDS; ++k) s.count[k] = s.used[k] = 0;
    s.count[0] = first ? 1 : left;
    s.used[0] = first ? tx + ty + tz : used;
    if (!first) return;
    s.accepted = s.overflow = 0;
    s.tagged = 0;
    w->queue[0][0] = DBox{{0, 0, 0}, {tx, ty, tz}, 0, 0};
}

struct Cut {
    long long strength;  // -1: none
    int d, len, axis, p;
};
__device__ __forceinline__ bool better_cut(const Cut &a, const Cut &b) {
    if (a.strength != b.strength) return a.strength > b.strength;
    if (a.d != b.d) return a.d < b.d;
    if (a.len != b.len) return a.len > b.len;
    return a.axis != b.axis ? a.axis < b.axis : a.p < b.p;
}
__device__ __forceinline__ Cut best_of_warp(Cut c) {
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) {
        Cut o;
        o.strength = __shfl_xor_sync(0xffffffffu, c.strength, off);
        o.d = __shfl_xor_sync(0xffffffffu, c.d, off);
        o.len = __shfl_xor_sync(0xffffffffu, c.len, off);
        o.axis = __shfl_xor_sync(0xffffffffu, c.axis, off);
        o.p = __shfl_xor_sync(0xffffffffu, c.p, off);
        if (better_cut(o, c)) c = o;
    }
    return c;
}

// decide() by one warp: s holds the box's signatures x, y, z.  The same value on every lane.
__device__ int decide_warp(HBox &box, const int *s, double efficiency, int wmin, long long &total,
                           HBox &lower, HBox &upper) {
    const int lane = threadIdx.x & 31;
    const int *sig[3];
    int len[3];
    total = 0;
    const int *at = s;
    int first[3];
    for (int a = 0; a < 3; ++a) {
        const int n = box.hi[a] - box.lo[a];
        int lo = INT_MAX, hi = -1;
        for (int i = lane; i < n; i += 32) {
            if (a == 0) total += at[i];
            if (at[i]) {
                lo = min(lo, i);
                hi = max(hi, i);
            }
        }
        first[a] = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        if (hi < 0) return 0;  // no tag on this axis, so none in the box
        len[a] = hi - first[a] + 1;
        sig[a] = at + first[a];
        at += n;
    }
    for (int off = 16; off >= 1; off >>= 1) total += __shfl_xor_sync(0xffffffffu, total, off);
    for (int a = 0; a < 3; ++a) {
        box.lo[a] += first[a];
        box.hi[a] = box.lo[a] + len[a];
    }
    const double vol = (double)len[0] * (double)len[1] * (double)len[2];
    if ((double)total >= efficiency * vol) return 1;
    Cut cut = {-1, 0, 0, 0, 0};
    for (int a = 0; a < 3; ++a)  // holes
        for (int p = wmin + lane; p <= len[a] - wmin; p += 32) {
            if (p >= len[a] || sig[a][p] != 0) continue;
            const Cut c = {0, abs(2 * p - len[a]), len[a], a, p};
            if (better_cut(c, cut)) cut = c;
        }
    cut = best_of_warp(cut);
    if (cut.strength < 0) {  // inflections
        for (int a = 0; a < 3; ++a) {
            const int *q = sig[a];
            for (int i = 1 + lane; i <= len[a] - 3; i += 32) {
                const long long d0 = (long long)q[i - 1] - 2LL * q[i] + q[i + 1];
                const long long d1 = (long long)q[i] - 2LL * q[i + 1] + q[i + 2];
                if (!((d0 < 0 && d1 > 0) || (d0 > 0 && d1 < 0))) continue;
                const int p = i + 1;
                if (p < wmin || len[a] - p < wmin) continue;
                const Cut c = {llabs(d1 - d0), abs(2 * p - len[a]), len[a], a, p};
                if (better_cut(c, cut)) cut = c;
            }
        }
        cut = best_of_warp(cut);
    }
    if (cut.strength < 0)  // bisection of the longest admissible axis (ties: lower axis)
        for (int a = 0; a < 3; ++a) {
            const int p = len[a] / 2;
            if (p < wmin || len[a] - p < wmin) continue;
            if (cut.strength < 0 || len[a] > cut.len) cut = {0, 0, len[a], a, p};
        }
    if (cut.strength < 0) return 1;
    lower = upper = box;
    for (int a = 0; a < 3; ++a)
        if (a == cut.axis) lower.hi[a] = upper.lo[a] = box.lo[a] + cut.p;
    return 2;
}

__global__ void __launch_bounds__(CL_THREADS)
    k_cluster_round(const uint8_t *__restrict__ tags, int tx, int ty, ClusterWork *w, int round,
                    bool root, double efficiency, int wmin) {
    __shared__ int sx[CL_EXTENTS];
    __shared__ int last;
    // the round before has ended (the tags are older: k_cluster_start has waited for them); the next
    // round's CTAs start as this one's end
    w = pdl_wait_only(w);
    ClusterState &st = w->state;
    // The round's boxes and signature words are what the launches before left, the same for every
    // thread of this one: all go on or all leave, whatever other CTAs of the launch queue meanwhile.
    // Counts beyond the limits are of boxes that have no place: the clustering has failed.
    const int count = st.count[round];
    if (count == 0 || count > CL_BOXES || st.used[round] > CL_SIG) return;
    const int parts = min(max((int)gridDim.x / count, 1), CL_MAX_PARTS);
    DBox *queue = w->queue[round & 1];
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    for (int job = blockIdx.x; job < count * parts; job += gridDim.x) {
        DBox &b = queue[job / parts];
        HBox box;
        for (int a = 0; a < 3; ++a) box.lo[a] = b.lo[a], box.hi[a] = b.hi[a];
        const int bw = box.hi[0] - box.lo[0], bh = box.hi[1] - box.lo[1], bd = box.hi[2] - box.lo[2];
        int *sig = w->sig[round & 1] + b.off;
        const int rows = bh * bd, part = job % parts;  // under CL_EXTENTS^2
        const int r0 = (int)((long long)rows * part / parts);
        const int r1 = (int)((long long)rows * (part + 1) / parts);
        __syncthreads();  // the last job's signatures have been read
        for (int i = threadIdx.x; i < bw; i += CL_THREADS) sx[i] = 0;
        __syncthreads();
        for (int r = r0 + warp; r < r1; r += CL_THREADS / 32) {
            const int y = r % bh, z = r / bh;
            const uint8_t *row = tags + ((size_t)(box.lo[2] + z) * ty + box.lo[1] + y) * tx + box.lo[0];
            int n = 0;
            for (int x = lane; x < bw; x += 32) {
                const int v = row[x];
                if (v) atomicAdd(&sx[x], 1);
                n += v;
            }
            n = __reduce_add_sync(0xffffffffu, n);
            if (lane == 0 && n) {
                atomicAdd(&sig[bw + y], n);
                atomicAdd(&sig[bw + bh + z], n);
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < bw; i += CL_THREADS)
            if (sx[i]) atomicAdd(&sig[i], sx[i]);
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) last = atomicAdd(&b.arrived, 1) == parts - 1;
        __syncthreads();
        if (!last) continue;
        __threadfence();
        const int words = bw + bh + bd;
        for (int i = threadIdx.x; i < words; i += CL_THREADS) {
            sx[i] = __ldcg(sig + i);
            sig[i] = 0;
        }
        __syncthreads();
        if (warp != 0) continue;
        HBox lower, upper;
        long long total;
        const int d = decide_warp(box, sx, efficiency, wmin, total, lower, upper);
        if (lane != 0) continue;
        if (root) st.tagged = total;
        if (d == 1) {
            const int k = atomicAdd(&st.accepted, 1);
            if (k < CL_BOXES)
                st.boxes[k] = box;
            else
                st.overflow = 1;
        } else if (d == 2) {
            const HBox half[2] = {lower, upper};
            int n[2];
            for (int j = 0; j < 2; ++j)
                n[j] = half[j].hi[0] - half[j].lo[0] + half[j].hi[1] - half[j].lo[1] +
                       half[j].hi[2] - half[j].lo[2];
            const int k = atomicAdd(&st.count[round + 1], 2);
            const int off = atomicAdd(&st.used[round + 1], n[0] + n[1]);
            if (k + 2 > CL_BOXES || off > CL_SIG - n[0] - n[1]) {
                st.overflow = 1;
            } else {
                for (int j = 0; j < 2; ++j) {
                    DBox &c = w->queue[(round + 1) & 1][k + j];
                    for (int a = 0; a < 3; ++a) c.lo[a] = half[j].lo[a], c.hi[a] = half[j].hi[a];
                    c.off = off + (j ? n[0] : 0);
                    c.arrived = 0;
                }
            }
        }
    }
}

struct DevBuf {
    void *p = nullptr;
    size_t cap = 0;
    ~DevBuf() { cudaFree(p); }
    cudaError_t ensure(size_t bytes) {
        if (bytes <= cap) return cudaSuccess;
        cudaFree(p);
        p = nullptr;
        cap = 0;
        cudaError_t e = lbm::dev_alloc(&p, bytes);
        if (e == cudaSuccess) cap = bytes;
        return e;
    }
};

#define RGCK(call, what)                                          \
    do {                                                          \
        cudaError_t e_ = (call);                                  \
        if (e_ != cudaSuccess) return report_cuda_error(e_, what); \
    } while (0)

}  // namespace

// The buffers of a handle's regrids, kept from one to the next and freed with the handle.
struct Work {
    DevBuf tags[2], mask, sig, items, boxes, cluster;
    void *head = nullptr;  // pinned copy of the clustering's state and first boxes
    bool sig_clear = false;  // the clustering's signature pools are zero
    ~Work() { cudaFreeHost(head); }
};
void destroy(Work *w) { delete w; }

namespace {

// Clusters the tags on the device; *done = false where a queue or pool was too small.
int cluster(Work &wk, const uint8_t *tags, int tx, int ty, int tz, const Params &p,
            std::vector<HBox> *accepted, long long *ntagged, bool *done, uint8_t *tags_out,
            long long ntag, cudaStream_t s) {
    const bool fresh = wk.cluster.cap == 0;
    RGCK(wk.cluster.ensure(sizeof(ClusterWork)), "cudaMalloc(clustering)");
    if (!wk.head) RGCK(cudaHostAlloc(&wk.head, CL_HEAD, cudaHostAllocDefault), "cudaHostAlloc(regrid)");
    ClusterWork *w = static_cast<ClusterWork *>(wk.cluster.p);
    if (fresh || !wk.sig_clear) RGCK(cudaMemsetAsync(w->sig, 0, sizeof(w->sig), s), "memset(signatures)");
    wk.sig_clear = false;
    const ClusterState *head = static_cast<const ClusterState *>(wk.head);
    // a piece wider than any extent is as inadmissible as one of INT_MAX, to which lanes cannot be added
    const int wmin = std::min(p.min_width, CL_EXTENTS + 1);
    for (bool first = true;; first = false) {
        k_cluster_start<<<1, 1, 0, s>>>(w, tx, ty, tz, first);
        for (int r = 0; r < CL_ROUNDS; ++r)
            RGCK(launch_pdl(k_cluster_round, CL_CTAS, CL_THREADS, 0, s, tags, tx, ty, w, r,
                            first && r == 0, p.efficiency, wmin),
                 "clustering kernel");
        RGCK(cudaGetLastError(), "clustering kernel");
        RGCK(cudaMemcpyAsync(wk.head, w, CL_HEAD, cudaMemcpyDeviceToHost, s), "boxes");
        if (first && tags_out)
            RGCK(cudaMemcpyAsync(tags_out, tags, ntag, cudaMemcpyDeviceToHost, s), "tags");
        RGCK(cudaStreamSynchronize(s), "regrid");
        if (head->overflow) return LBM_OK;
        if (head->count[CL_ROUNDS] == 0) break;
    }
    wk.sig_clear = true;
    *ntagged = head->tagged;
    const int n = head->accepted;
    accepted->resize(n);
    std::copy(head->boxes, head->boxes + std::min(n, CL_FIRST_BOXES), accepted->begin());
    if (n > CL_FIRST_BOXES) {
        RGCK(cudaMemcpyAsync(accepted->data() + CL_FIRST_BOXES, w->state.boxes + CL_FIRST_BOXES,
                             sizeof(HBox) * (n - CL_FIRST_BOXES), cudaMemcpyDeviceToHost, s),
             "boxes");
        RGCK(cudaStreamSynchronize(s), "regrid");
    }
    *done = true;
    return LBM_OK;
}

}  // namespace

int regrid(Work **work, const void *field, int field_type, int nx, int ny, int nz, int periodic,
           const Params &p, const uint8_t *allowed_host, std::vector<int> *boxes_out,
           long long *ntagged, uint8_t *tags_out, cudaStream_t s) {
    const int r = p.coarsen, rz = nz > 1 ? p.coarsen : 1;
    const int tx = (nx + r - 1) / r, ty = (ny + r - 1) / r, tz = (nz + rz - 1) / rz;
    const long long ntag = (long long)tx * ty * tz;
    if (!*work) *work = new (std::nothrow) Work();
    if (!*work) return report_error(LBM_ENOMEM, "regrid: out of host memory");
    Work &wk = **work;
    DevBuf (&tagbuf)[2] = wk.tags, &maskbuf = wk.mask, &sigbuf = wk.sig, &itembuf = wk.items,
           &boxbuf = wk.boxes;
    RGCK(tagbuf[0].ensure(ntag), "cudaMalloc(tags)");
    RGCK(tagbuf[1].ensure(ntag), "cudaMalloc(tags)");
    uint8_t *ta = (uint8_t *)tagbuf[0].p, *tb = (uint8_t *)tagbuf[1].p;

    // 1. tags
    if (field_type == LBM_F64)
        k_tag<double><<<nblk(ntag, 256), 256, 0, s>>>((const double *)field, nx, ny, nz, r, rz, tx,
                                                      ty, ntag, p.threshold, ta);
    else if (r % 4 == 0 && nx % 4 == 0 && ((uintptr_t)field & 15) == 0)
        k_tag_f4<<<nblk(ntag, 256), 256, 0, s>>>((const float *)field, nx, ny, nz, r, rz, tx, ty,
                                                  ntag, float_at_most(p.threshold), ta);
    else
        k_tag<float><<<nblk(ntag, 256), 256, 0, s>>>((const float *)field, nx, ny, nz, r, rz, tx,
                                                     ty, ntag, p.threshold, ta);
    RGCK(cudaGetLastError(), "tag kernel");
    const int ext[3] = {tx, ty, tz};
    const long long stride[3] = {1, tx, (long long)tx * ty};
    // 2. buffer: three 1-D dilations
    if (p.buffer > 0) {
        for (int a = 0; a < 3; ++a) {
            k_morph<<<nblk(ntag, 256), 256, 0, s>>>(ta, tb, ntag, ext[a], stride[a], p.buffer,
                                                    (periodic >> a) & 1, 0);
            std::swap(ta, tb);
        }
        RGCK(cudaGetLastError(), "buffer kernel");
    }
    // 3. proper nesting: erode the covered mask, keep the tags inside it
    if (allowed_host) {
        RGCK(maskbuf.ensure(2 * ntag), "cudaMalloc(mask)");
        uint8_t *ma = (uint8_t *)maskbuf.p, *mb = ma + ntag;
        RGCK(cudaMemcpyAsync(ma, allowed_host, ntag, cudaMemcpyHostToDevice, s), "mask upload");
        k_normalise<<<nblk(ntag, 256), 256, 0, s>>>(ma, ntag);
        if (p.nest > 0)
            for (int a = 0; a < 3; ++a) {
                k_morph<<<nblk(ntag, 256), 256, 0, s>>>(ma, mb, ntag, ext[a], stride[a], p.nest,
                                                        (periodic >> a) & 1, 1);
                std::swap(ma, mb);
            }
        k_and<<<nblk(ntag, 256), 256, 0, s>>>(ta, ma, ntag);
        RGCK(cudaGetLastError(), "nesting kernel");
    }

    // 4. clustering, on the device where a box's signatures fit its shared memory and the boxes its
    // queues; else in rounds of signature passes over the pending boxes, cut by the host
    std::vector<HBox> pending, accepted;
    bool done = false;
    long long tagged = 0;
    const bool device = (long long)tx + ty + tz <= CL_EXTENTS;
    if (device) {
        const int st = cluster(wk, ta, tx, ty, tz, p, &accepted, &tagged, &done, tags_out, ntag, s);
        if (st != LBM_OK) return st;
        if (done && ntagged) *ntagged = tagged;
    } else if (tags_out) {
        RGCK(cudaMemcpyAsync(tags_out, ta, ntag, cudaMemcpyDeviceToHost, s), "tags");
    }
    if (!done) {
        accepted.clear();
        pending.assign(1, HBox{{0, 0, 0}, {tx, ty, tz}});
    }
    std::vector<SigItem> items;
    std::vector<SigBox> sboxes;
    std::vector<int> sig;
    bool first_round = true;
    while (!pending.empty()) {
        items.clear();
        sboxes.clear();
        int off = 0;
        for (size_t k = 0; k < pending.size(); ++k) {
            const HBox &b = pending[k];
            SigBox sb;
            for (int a = 0; a < 3; ++a) sb.lo[a] = b.lo[a];
            sb.w = b.hi[0] - b.lo[0];
            sb.h = b.hi[1] - b.lo[1];
            sb.off = off;
            off += sb.w + sb.h + (b.hi[2] - b.lo[2]);
            sboxes.push_back(sb);
            for (int z = b.lo[2]; z < b.hi[2]; ++z)
                for (int x0 = b.lo[0]; x0 < b.hi[0]; x0 += SIG_XCHUNK) {
                    const int x1 = std::min(x0 + SIG_XCHUNK, b.hi[0]);
                    const int rows = std::max(1, std::min(SIG_XCHUNK, SIG_CELLS / (x1 - x0)));
                    for (int y0 = b.lo[1]; y0 < b.hi[1]; y0 += rows)
                        items.push_back({(int)k, z, y0, std::min(y0 + rows, b.hi[1]), x0, x1});
                }
        }
        RGCK(sigbuf.ensure(sizeof(int) * off), "cudaMalloc(signatures)");
        RGCK(itembuf.ensure(sizeof(SigItem) * items.size()), "cudaMalloc(items)");
        RGCK(boxbuf.ensure(sizeof(SigBox) * sboxes.size()), "cudaMalloc(boxes)");
        RGCK(cudaMemcpyAsync(itembuf.p, items.data(), sizeof(SigItem) * items.size(),
                             cudaMemcpyHostToDevice, s),
             "items upload");
        RGCK(cudaMemcpyAsync(boxbuf.p, sboxes.data(), sizeof(SigBox) * sboxes.size(),
                             cudaMemcpyHostToDevice, s),
             "boxes upload");
        RGCK(cudaMemsetAsync(sigbuf.p, 0, sizeof(int) * off, s), "memset(signatures)");
        k_signatures<<<(unsigned)items.size(), SIG_THREADS, 0, s>>>(
            ta, tx, ty, (const SigItem *)itembuf.p, (const SigBox *)boxbuf.p, (int *)sigbuf.p);
        RGCK(cudaGetLastError(), "signature kernel");
        sig.resize(off);
        RGCK(cudaMemcpyAsync(sig.data(), sigbuf.p, sizeof(int) * off, cudaMemcpyDeviceToHost, s),
             "signatures download");
        RGCK(cudaStreamSynchronize(s), "regrid round");
        std::vector<HBox> next;
        for (size_t k = 0; k < pending.size(); ++k) {
            HBox b = pending[k], lo, hi;
            const SigBox &sb = sboxes[k];
            const int *sx = sig.data() + sb.off;
            if (first_round && ntagged) {
                long long t = 0;
                for (int i = 0; i < sb.w; ++i) t += sx[i];
                *ntagged = t;
            }
            const int d = decide(b, sx, sx + sb.w, sx + sb.w + sb.h, p.efficiency, p.min_width,
                                 &lo, &hi);
            if (d == 1) accepted.push_back(b);
            if (d == 2) {
                next.push_back(lo);
                next.push_back(hi);
            }
        }
        first_round = false;
        pending.swap(next);
    }
    std::sort(accepted.begin(), accepted.end(), [](const HBox &a, const HBox &b) {
        if (a.lo[2] != b.lo[2]) return a.lo[2] < b.lo[2];
        if (a.lo[1] != b.lo[1]) return a.lo[1] < b.lo[1];
        return a.lo[0] < b.lo[0];
    });
    const int scale[3] = {r, r, rz}, lat[3] = {nx, ny, nz};
    boxes_out->clear();
    for (const HBox &b : accepted) {
        for (int a = 0; a < 3; ++a) boxes_out->push_back(b.lo[a] * scale[a]);
        for (int a = 0; a < 3; ++a)
            boxes_out->push_back((int)std::min<long long>((long long)b.hi[a] * scale[a], lat[a]));
    }
    return LBM_OK;
}

}  // namespace rg
}  // namespace lbm
