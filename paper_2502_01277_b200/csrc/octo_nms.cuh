// Per-image ordering + class-aware greedy NMS + cap + scale-back, as device code of one CTA (or of a
// thread-block cluster) per image.
//
// Latency / shared-memory bound; bytes are negligible.  Keys are (class | inverted score bits | anchor),
// so the ascending order of the keys of a class is its NMS order.
//
// At most kSmallMax candidates (the usual case in serving): every step is spread over the threads of the
// CTA.  Candidates are put in order (words of 32 by counting, then every candidate's place in every word by
// binary search); each is tested against the earlier candidates of its class (one bit each); which
// candidates survive is settled word by word of those bits (resolve_words), in a time that follows the
// length of the chains of overlapping boxes, not the number of candidates of a class.  us per launch (CUDA
// events), against one thread per class that walked its candidates: 200 candidates of one class 18.7 (67.4
// with 8 images), of 7 classes 14.6 (28.3), of 80 classes 12.6 (12.6); 90 candidates under class-agnostic
// NMS 13.3 (35.7).  What is left is bound by the latency of a dozen short phases and, in one large class,
// by the pair tests (shared-memory return bandwidth: 20 bytes per lane and test).
//
// More candidates: bucketed by class in shared memory (histogram, scan, scatter).  Most classes belong to
// one warp each: counting sort, boxes gathered from the head, then a greedy scan of 32 candidates at a
// time against the class's survivors.  A class that is large beside a warp's share of the image
// (`team_min`) is taken by the whole CTA, kTeamBlock candidates at a time: survivor tests, suppression
// bits and the settling above are spread over all warps (1200 candidates of one class, 4 images: 95 us;
// 464 when one warp had the class to itself).
// Survivors are compacted in place, re-keyed to (inverted score | anchor | class), packed and put in
// order by counting or, when there are many, by a CTA-wide bitonic network.
//
// Images with more candidates than fit in shared memory take the same code path with the arrays in a
// global-memory workspace.
//
// A cluster of CTAs per image (crowded scenes at small batches): every CTA buckets the image's keys for
// itself, the classes are handed out by one counter in the first CTA's shared memory to the warps of all
// CTAs (the large ones to the CTAs in turn), and every finished class is written into the first CTA's
// arrays through distributed shared memory.  The first CTA alone orders and writes the image's results.
#pragma once

#include <cooperative_groups.h>

#include "octo_common.cuh"
#include "octo_kernels.h"

namespace octo {

namespace cg = cooperative_groups;

constexpr int kNmsThreadsFull = 1024;
constexpr int kNmsSmemCap = 8192;   // candidates handled on chip: 8 B key + 16 B box each
// Batches of more images than the GPU has SMs that have held only sparse images lately run two
// smaller CTAs per SM (half the threads, half the on-chip capacity), so that the launch is one
// wave of CTAs instead of two; an image that exceeds the smaller capacity takes the global-memory
// path, and the launches after it are full-sized again.
constexpr int kNmsThreadsHalf = 512;
constexpr int kNmsSmemCapHalf = 4096;
constexpr int kSmallMax = 512;      // images with at most this many candidates take the short path
constexpr int kSmallWords = kSmallMax / 32;
constexpr int kTeamBlock = 128;     // candidates of a large class that the CTA works on together
constexpr int kTeamWords = kTeamBlock / 32;
constexpr int kTeamMax = 512;       // a class above this is always the whole CTA's
constexpr int kClusterMinCand = 1024;  // an image with more candidates than this makes clusters worth while

constexpr size_t kNmsSmemBytes = (size_t)kNmsSmemCap * (sizeof(float4) + sizeof(unsigned long long));
constexpr size_t kNmsSmemBytesHalf = (size_t)kNmsSmemCapHalf * (sizeof(float4) + sizeof(unsigned long long));

// What one image's NMS works on and writes (by value in kernel parameter space).
struct NmsParams {
    const float* head;
    int A, C, layout;
    IouTest iou_test;
    int max_det, key_stride;
    unsigned long long* gkeys;
    float4* gboxes;
    int* cand_count;
    octo_det_rec* dets;
    int* counts;
    int num_branches, class_agnostic;
    int full_branches;  // bit b: the mask of branch b holds every class
    BranchMasks masks;
    int* bcount;
    int* bidx;
    int max_batch;
    StageCounters* ctr;
    int* dense_seen;
    int launch_seq;
};

constexpr unsigned long long kKeyLow = (1ull << 57) - 1;  // score and anchor of a key

// class | inverted score | anchor  ->  inverted score | anchor | class
__device__ __forceinline__ unsigned long long global_key(unsigned long long k) { return ((k & kKeyLow) << 7) | (k >> 57); }

__device__ __forceinline__ void cmp_swap(unsigned long long* __restrict__ k, int i, int j) {
    const unsigned long long a = k[i], b = k[j];
    if (a > b) { k[i] = b; k[j] = a; }
}

// Ascending bitonic sort of k[0, m) for any m by the whole CTA.  Every comparator puts the smaller key
// at the lower index (the first stage of each merge pairs mirrored positions), so positions >= m can
// stand for +infinity and are simply skipped.
__device__ __forceinline__ void bitonic_cta(unsigned long long* __restrict__ k, int m, int tid, int nthreads) {
    int np2 = 2;
    while (np2 < m) np2 <<= 1;
    const int half = np2 >> 1;
    for (int size = 2; size <= np2; size <<= 1) {
        __syncthreads();
        const int h = size >> 1;
        for (int t = tid; t < half; t += nthreads) {
            const int off = t & (h - 1);
            const int i = 2 * t - off;             // block start + off
            const int j = i + size - 1 - 2 * off;  // mirrored position in the block
            if (j < m) cmp_swap(k, i, j);
        }
        for (int stride = size >> 2; stride > 0; stride >>= 1) {
            __syncthreads();
            for (int t = tid; t < half; t += nthreads) {
                const int i = 2 * t - (t & (stride - 1));
                const int j = i + stride;
                if (j < m) cmp_swap(k, i, j);
            }
        }
    }
    __syncthreads();
}

// Box of one anchor; es = distance between consecutive values of an anchor (1 in the rows
// layout, A in the planes layout).
__device__ __forceinline__ float4 gather_box(const float* __restrict__ p, size_t es) {
    return box_corners(__ldg(p), __ldg(p + es), __ldg(p + 2 * es), __ldg(p + 3 * es));
}

// Barrier of the first `threads` threads of the CTA (a multiple of 32); returns whether any of them
// passed `more`.
__device__ __forceinline__ bool bar_any(int threads, bool more) {
    int r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.s32 p, %1, 0;\n\t"
        "barrier.cta.red.or.pred q, 1, %2, p;\n\tselp.s32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"((int)more), "r"(threads)
        : "memory");
    return r != 0;
}

// Exclusive scan over 128 class counts by one warp: four neighbouring classes per lane.
__device__ __forceinline__ void scan_classes(int lane, const int* count, int* start) {
    const int4 v = *reinterpret_cast<const int4*>(count + 4 * lane);
    const int sum = v.x + v.y + v.z + v.w;
    int inc = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, inc, off);
        if (lane >= off) inc += u;
    }
    const int s = inc - sum;
    *reinterpret_cast<int4*>(start + 4 * lane) = make_int4(s, s + v.x, s + v.x + v.y, s + v.x + v.y + v.z);
}

// Part `part` of `parts` of the number of keys in k[lo, hi) below `own`, two keys per read (k is 16-byte
// aligned; k[hi] is readable and not below any key counted against it).  From an even position: when lo
// is odd, k[lo - 1] must be below `own` and is taken off again.
__device__ __forceinline__ int count_below(const unsigned long long* k, int lo, int hi, unsigned long long own, int part,
                                           int parts) {
    int r = part == 0 ? -(lo & 1) : 0;
#pragma unroll 2
    for (int j = (lo & ~1) + 2 * part; j < hi; j += 2 * parts) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(k + j);
        r += (v.x < own ? 1 : 0) + (v.y < own ? 1 : 0);
    }
    return r;
}

// Which candidates survive, by the first `words` warps of the CTA, one candidate per thread: `cand` (or
// none when cand >= n).  A candidate's bit is bit (lane) of word (warp) of its thread.  sup[w * LEN +
// cand]: the bits of the earlier candidates that suppress it, valid for the words w0 .. own.  fate[w] =
// (kept, gone): gone may already hold candidates that are out; `left` is scratch, one word per warp.
// A candidate is removed once one of its suppressors survives and survives once all of them are removed.
// All words settle at once what they can by themselves (ballots inside the warp, one per link of a chain
// of overlapping boxes), then once more with what the others found: that is all when the classes are
// small.  The words that are not done then take their turn in order, every later word learning from each
// what it kept, so that a word whose turn it is has only its own chains left.
template <int LEN>
__device__ __forceinline__ void resolve_words(const unsigned* sup, int cand, int n, int w0, volatile uint2* fate,
                                              volatile unsigned* left, int tid, int words) {
    const int lane = tid & 31, word = tid >> 5, threads = words * 32;
    unsigned kept = 0u, gone = fate[word].y;
    bool open = cand < n && !((gone >> lane) & 1u), out = false;
    const unsigned own = open ? sup[word * LEN + cand] : 0u;
    unsigned undecided = __ballot_sync(0xffffffffu, open);
    auto settle = [&](bool free) {  // free: no undecided suppressor in an earlier word
        while (undecided != 0u) {
            const bool dies = open && (out || (own & kept) != 0u);
            const bool lives = open && !dies && free && (own & ~gone) == 0u;
            const unsigned k = __ballot_sync(0xffffffffu, lives), g = __ballot_sync(0xffffffffu, dies);
            if ((k | g) == 0u) break;
            kept |= k;
            gone |= g;
            undecided &= ~(k | g);
            open = open && !dies && !lives;
        }
    };
    auto meet = [&]() { asm volatile("barrier.cta.sync 1, %0;" ::"r"(threads) : "memory"); };
    unsigned ask = 0u;  // earlier words with a suppressor
    if (open)
        for (int w = w0; w < word; ++w)
            if (sup[w * LEN + cand]) ask |= 1u << w;
    settle(ask == 0u);
    if (lane == 0) { fate[word].x = kept; fate[word].y = gone; }
    meet();
    unsigned later = 0u;  // ... that hold an undecided one
    if (open) {
        for (unsigned todo = ask; todo != 0u; todo &= todo - 1u) {
            const int w = __ffs(todo) - 1;
            const unsigned b = sup[w * LEN + cand];
            out |= (b & fate[w].x) != 0u;
            if (b & ~fate[w].y) later |= 1u << w;
        }
    }
    settle(later == 0u);
    // (kept only gains bits, so a warp that still looks at the first outcome may read either)
    if (lane == 0) { fate[word].x = kept; left[word] = undecided; }
    if (!bar_any(threads, open)) return;
    for (int w = 0; w < words; ++w) {
        if (left[w] != 0u) {
            if (word == w) {
                settle(true);
                if (lane == 0) fate[w].x = kept;
            }
            meet();
        }
        if ((later >> w) & 1u) out |= (sup[w * LEN + cand] & fate[w].x) != 0u;
    }
}

// Head boxes to source-frame pixels.
struct RegionMap {
    float fpl, fpt, gx, gy, x_lo, y_lo, x_hi, y_hi;
    __device__ __forceinline__ explicit RegionMap(const FrameDesc& fd)
        : fpl((float)fd.pad_l), fpt((float)fd.pad_t), gx(fd.gx), gy(fd.gy), x_lo((float)fd.ox), y_lo((float)fd.oy),
          x_hi((float)(fd.ox + fd.rw)), y_hi((float)(fd.oy + fd.rh)) {}
    // X = fl(fl(fl(x - pad) * gain) + origin), clamped to the region of the frame the detector input shows
    __device__ __forceinline__ void write(octo_det_rec* out, const float4 b, unsigned long long g, int cls) const {
        octo_det_rec d;
        d.x1 = fminf(fmaxf(__fadd_rn(__fmul_rn(__fsub_rn(b.x, fpl), gx), x_lo), x_lo), x_hi);
        d.y1 = fminf(fmaxf(__fadd_rn(__fmul_rn(__fsub_rn(b.y, fpt), gy), y_lo), y_lo), y_hi);
        d.x2 = fminf(fmaxf(__fadd_rn(__fmul_rn(__fsub_rn(b.z, fpl), gx), x_lo), x_lo), x_hi);
        d.y2 = fminf(fmaxf(__fadd_rn(__fmul_rn(__fsub_rn(b.w, fpt), gy), y_lo), y_lo), y_hi);
        d.score = __uint_as_float(~(unsigned)(g >> 32));
        d.cls = cls;
        d.anchor = (int)((g >> 7) & ((1ull << kKeyAnchorBits) - 1));
        d._pad = 0;
        *out = d;
    }
};

// NMS of image `img` by a CTA of NT threads (SMEM_CAP candidates on chip), or by the cluster the CTA
// belongs to when CLUSTER.  The image's candidate count, keys and (for the short path) boxes are in
// global memory.
template <int NT, int SMEM_CAP, bool CLUSTER>
__device__ __forceinline__ void nms_image(const NmsParams& P, const FrameDesc& fd, bool no_frame, int img,
                                          unsigned char* smem_raw) {
    __shared__ __align__(16) int seg_start[128], seg_cnt[128], cursor[128], nkept[128];
    __shared__ unsigned s_mask[OCTO_MAX_BRANCHES][4];
    __shared__ int s_total, s_next, s_nlarge;
    __shared__ unsigned char s_large[128];
    __shared__ uint2 s_fate[kSmallWords];  // see resolve_words
    __shared__ unsigned s_left[kSmallWords];
    unsigned int* const status = &P.ctr->status;
    (void)status;  // referenced by the range checks of the checked build only

    const unsigned csize = CLUSTER ? cg::this_cluster().num_blocks() : 1u;
    const unsigned crank = CLUSTER ? cg::this_cluster().block_rank() : 0u;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // rows layout [A][5 + C] or planes layout [4 + C][A]
    const int nbox = P.layout == OCTO_HEAD_PLANES ? 4 : 5;
    const size_t es = P.layout == OCTO_HEAD_PLANES ? (size_t)P.A : 1;           // value to value
    const size_t as = P.layout == OCTO_HEAD_PLANES ? 1 : (size_t)(nbox + P.C);  // anchor to anchor
    const float* __restrict__ hbase = P.head + (size_t)img * (size_t)P.A * (size_t)(nbox + P.C);
    unsigned long long* const gk = P.gkeys + (size_t)img * P.key_stride;
    const float4* const gb = P.gboxes + (size_t)img * P.key_stride;
    const int max_det = P.max_det;

    // the first kSmallMax keys and boxes travel beside the count: one round trip for the usual image
    int cnt = __ldcg(P.cand_count + img);
    unsigned long long first_key = kKeySentinel;
    float4 first_box = make_float4(0.f, 0.f, 0.f, 0.f);
    if (tid < kSmallMax && tid < P.key_stride) {
        first_key = __ldcg(gk + tid);
        first_box = __ldcg(gb + tid);
    }
    cnt = min(cnt, P.key_stride);
    if (no_frame) cnt = 0;
    if (tid < 128) { seg_cnt[tid] = 0; nkept[tid] = 0; }
    if (tid < kSmallWords) s_fate[tid] = make_uint2(0u, 0u);
    if (tid < OCTO_MAX_BRANCHES * 4) s_mask[tid >> 2][tid & 3] = P.masks.m[tid >> 2][tid & 3];
    if (tid == 0) { s_total = 0; s_next = 0; }
    // every CTA of the image has read the count, and the first CTA's counters are set, before the
    // count is cleared and before any CTA touches those counters
    if (CLUSTER && csize > 1) cg::this_cluster().sync(); else __syncthreads();
    if (tid == NT - 1 && crank == 0) {  // (a warp that has no other work on the short path)
        P.cand_count[img] = 0;  // ready for the next batch's decode
        atomicAdd(&P.ctr->candidates, (unsigned long long)cnt);
        atomicMax(&P.ctr->max_cand, cnt);
        // (only crowded images write: a store to host memory delays the end of the kernel by a PCIe
        // round trip, which a sparse launch of ten microseconds would feel)
        if (P.dense_seen && cnt > kClusterMinCand) *P.dense_seen = P.launch_seq;
    }

    octo_det_rec* const dets = P.dets + (size_t)img * max_det;
    const RegionMap map(fd);
    unsigned long long* ordered;  // survivors in output order (inverted score | anchor | class)
    int nout;
    if (cnt <= kSmallMax) {
        if (crank != 0) return;  // the first CTA alone; no cluster barrier follows on this path
        // Thread (candidate c = word * 32 + lane, part): the 4, 2 or 1 parts of a candidate's work are warps, and
        // the lanes of a warp read the same shared-memory words as they walk.  Part 0 of candidate c is thread
        // c, which holds its key and box in registers.
        const int words = (cnt + 31) >> 5;
        const int parts = 4 * words <= NT / 32 ? 4 : 2 * words <= NT / 32 ? 2 : 1;
        const int word = warp % max(words, 1), part = warp / max(words, 1);  // part >= parts: nothing to do
        const int c = word * 32 + lane;
        const bool busy = part < parts && c < cnt;
        unsigned long long* const ukey = reinterpret_cast<unsigned long long*>(smem_raw);  // as they came
        unsigned long long* const wkey = ukey + kSmallMax;      // each word of 32 in order
        unsigned long long* const skey = wkey + kSmallMax;      // all in order: by class, then NMS order
        unsigned long long* const surv = skey + kSmallMax;      // survivors' global-order keys, padded
        ordered = surv + kSmallMax + 2;
        float4* const sbox = reinterpret_cast<float4*>(ordered + kSmallMax);
        unsigned* const sup = reinterpret_cast<unsigned*>(sbox + kSmallMax);  // [kSmallWords][kSmallMax]
        float* const sshare = reinterpret_cast<float*>(sup + kSmallMax * kSmallWords);
        int* const rank = reinterpret_cast<int*>(sshare + kSmallMax);
        int* const rank2 = rank + kSmallMax;
        unsigned short* const sstart = reinterpret_cast<unsigned short*>(rank2 + kSmallMax);  // first of the class
        unsigned short* const spos = sstart + kSmallMax;
        if (warp < words) {
            if (tid >= cnt) first_key = kKeySentinel;
            if (tid < cnt) atomicAdd(&seg_cnt[(int)(first_key >> 57)], 1);
            ukey[tid] = first_key;
            rank[tid] = 0;
            rank2[tid] = 0;
            __syncwarp();
            // order inside the word: the keys of its 32 that are below one's own
            int r = 0;
#pragma unroll 4
            for (int j = 0; j < 32; j += 2) {
                const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(ukey + (tid & ~31) + j);
                r += (v.x < first_key ? 1 : 0) + (v.y < first_key ? 1 : 0);
            }
            wkey[tid < cnt ? (tid & ~31) + r : tid] = first_key;
        }
        if (busy)
            for (int w = part; w < words; w += parts) sup[w * kSmallMax + c] = 0u;
        __syncthreads();
        // place among all candidates: its place in every word, by binary search
        if (busy) {
            const unsigned long long key = ukey[c];
            int r = 0;
            for (int w = part; w < words; w += 2 * parts) {  // two words side by side
                const unsigned long long* const k0 = wkey + 32 * w;
                const unsigned long long* const k1 = wkey + 32 * min(w + parts, words - 1);
                int lo0 = 0, lo1 = 0;
#pragma unroll 1
                for (int step = 16; step > 0; step >>= 1) {
                    lo0 += k0[lo0 + step - 1] < key ? step : 0;
                    lo1 += k1[lo1 + step - 1] < key ? step : 0;
                }
                r += lo0 + (k0[lo0] < key ? 1 : 0);
                if (w + parts < words) r += lo1 + (k1[lo1] < key ? 1 : 0);
            }
            if (r) atomicAdd(&rank[c], r);
        }
        if (warp == NT / 32 - 1) scan_classes(lane, seg_cnt, seg_start);  // where each class starts
        __syncthreads();
        if (tid < cnt) {
            const int at = rank[tid];
            if (OCTO_IN_RANGE(at >= 0 && at < cnt, status)) {
                skey[at] = first_key;
                sbox[at] = first_box;
                sshare[at] = iou_share(first_box, P.iou_test);
                sstart[at] = (unsigned short)seg_start[(int)(first_key >> 57)];
            }
        }
        __syncthreads();
        // Suppression bits.  Candidates j % 4 = p give byte p of a word (candidate j of a word has bit (j & 3)
        // * 8 + j / 4), so that parts never share one; a byte is tested whole (the lanes read the same boxes)
        // and what is not an earlier candidate of the class is masked off.
        if (busy) {
            const float4 b = sbox[c];
            const float own_share = sshare[c];
            const int start = sstart[c];
            if (!__any_sync(__activemask(), c - start > 24)) {
                // small classes: only the pairs there are, bits of two words at most
                const int w0 = start >> 5;
                for (int p = part; p < 4; p += parts) {
                    const int first = start + ((p - start) & 3);
                    unsigned bits = 0u;
                    bool close = false;
                    for (int j = first; j < c; j += 4)
                        if (iou_by_share(sbox[j], sshare[j], b, own_share, close)) bits |= 1u << ((j >> 2) - 8 * w0);
                    if (close) {
                        bits = 0u;
                        for (int j = first; j < c; j += 4)
                            if (iou_above(sbox[j], b, P.iou_test)) bits |= 1u << ((j >> 2) - 8 * w0);
                    }
                    unsigned char* const to = reinterpret_cast<unsigned char*>(sup + w0 * kSmallMax + c) + p;
                    if (bits & 0xffu) to[0] = (unsigned char)bits;
                    if (bits >> 8) to[4 * kSmallMax] = (unsigned char)(bits >> 8);
                }
            } else for (int p = part; p < 4; p += parts) {
                for (int w = start >> 5; 32 * w + p < c; ++w) {
                    const int base = 32 * w + p;
                    const int lo = max((start - base + 3) >> 2, 0), hi = min((c - base + 3) >> 2, 8);
                    unsigned bits = 0u;
                    bool close = false;
#pragma unroll
                    for (int t = 0; t < 8; ++t)
                        if (iou_by_share(sbox[base + 4 * t], sshare[base + 4 * t], b, own_share, close)) bits |= 1u << t;
                    if (close) {  // rare: some pair lies too near the threshold for binary32
                        bits = 0u;
                        for (int t = lo; t < hi; ++t)
                            if (iou_above(sbox[base + 4 * t], b, P.iou_test)) bits |= 1u << t;
                    }
                    bits &= (0xffu << lo) & (0xffu >> (8 - hi));
                    if (bits) reinterpret_cast<unsigned char*>(sup + w * kSmallMax + c)[p] = (unsigned char)bits;
                }
            }
        }
        __syncthreads();
        const int cand = (tid & ~31) | ((lane & 7) << 2) | (lane >> 3);  // the candidate of this thread's bit
        if (warp < words) resolve_words<kSmallMax>(sup, cand, cnt, cand < cnt ? sstart[cand] >> 5 : 0, s_fate, s_left, tid, words);
        __syncthreads();
        int inc = lane < kSmallWords ? __popc(s_fate[lane].x) : 0;  // survivors up to and including word `lane`
#pragma unroll
        for (int off = 1; off < kSmallWords; off <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, inc, off);
            if (lane >= off) inc += u;
        }
        const int m = __shfl_sync(0xffffffffu, inc, kSmallWords - 1);
        const int before = warp == 0 ? 0 : __shfl_sync(0xffffffffu, inc, warp - 1);
        const unsigned kept = warp < words ? s_fate[warp].x : 0u;
        if ((kept >> lane) & 1u) {
            const int q = before + __popc(kept & ((1u << lane) - 1u));
            surv[q] = global_key(skey[cand]);
            spos[q] = (unsigned short)cand;
        }
        if (tid == 0) surv[m] = kKeySentinel;
        __syncthreads();
        nout = min(m, max_det);
        // the survivors' order by counting among themselves
        const int mwords = max((m + 31) >> 5, 1);
        const int q = (warp % mwords) * 32 + lane, mpart = warp / mwords, mparts = min((NT / 32) / mwords, 4);
        unsigned long long g = 0ull;
        if (q < m && mpart < mparts) {
            g = surv[q];
            const int r = count_below(surv, 0, m, g, mpart, mparts);
            if (r) atomicAdd(&rank2[q], r);
        }
        __syncthreads();
        if (q < m && mpart == 0) {
            const int r = rank2[q];
            if (r < max_det && OCTO_IN_RANGE(r >= 0 && r < m, status)) {
                ordered[r] = g;
                if (!P.class_agnostic) map.write(dets + r, sbox[spos[q]], g, (int)(g & 127u));
            }
        }
    } else {
        const bool on_chip = cnt <= SMEM_CAP;
        unsigned long long* keys;
        float4* boxes;
        if (on_chip) {
            boxes = reinterpret_cast<float4*>(smem_raw);
            keys = reinterpret_cast<unsigned long long*>(smem_raw + (size_t)SMEM_CAP * sizeof(float4));
        } else {
            boxes = P.gboxes + (size_t)img * P.key_stride;
            keys = gk;
            if (tid == 0 && crank == 0 && cnt > kNmsSmemCap) atomicOr(&P.ctr->status, 0x8u);
            if (crank != 0) return;  // the first CTA alone; no cluster barrier follows on this path
        }
        // where the other CTAs of the cluster put their finished classes: the first CTA's arrays
        const bool shared_work = CLUSTER && csize > 1 && on_chip;
        const unsigned team_ctas = shared_work ? csize : 1u;
        unsigned long long* keys0 = keys;
        int *nkept0 = nkept, *total0 = &s_total, *next0 = &s_next;
        if (shared_work) {
            cg::cluster_group cluster = cg::this_cluster();
            keys0 = cluster.map_shared_rank(keys, 0);
            nkept0 = cluster.map_shared_rank(nkept, 0);
            total0 = cluster.map_shared_rank(&s_total, 0);
            next0 = cluster.map_shared_rank(&s_next, 0);
        }

        // A class with more candidates than this is the whole CTA's work: about eight times a warp's share
        // of the image, at least kTeamBlock (a smaller class is a few chunks of a warp).
        const int team_min = min(max(cnt / (4 * (int)team_ctas), kTeamBlock), kTeamMax);

        // ---- bucket the keys by class: histogram, scan, scatter ----
        auto scan_counts = [&]() {
            if (warp != 0) return;
            scan_classes(lane, seg_cnt, seg_start);
            __syncwarp();
            int nb = 0;  // the large classes
            for (int base = 0; base < 128; base += 32) {
                cursor[base + lane] = seg_start[base + lane];
                const bool is = seg_cnt[base + lane] > team_min;
                const unsigned bal = __ballot_sync(0xffffffffu, is);
                if (is) s_large[nb + __popc(bal & ((1u << lane) - 1u))] = (unsigned char)(base + lane);
                nb += __popc(bal);
            }
            if (lane == 0) s_nlarge = nb;
        };
        constexpr int kHeld = SMEM_CAP / NT;  // keys a thread keeps between the two passes
        if (on_chip) {
            unsigned long long held[kHeld];
#pragma unroll
            for (int u = 0; u < kHeld; ++u) {
                const int i = tid + u * NT;
                held[u] = i < cnt ? __ldcg(gk + i) : kKeySentinel;
            }
#pragma unroll
            for (int u = 0; u < kHeld; ++u)
                if (tid + u * NT < cnt) atomicAdd(&seg_cnt[(int)(held[u] >> 57)], 1);
            __syncthreads();
            scan_counts();
            __syncthreads();
#pragma unroll
            for (int u = 0; u < kHeld; ++u) {
                if (tid + u * NT >= cnt) continue;
                const int pos = atomicAdd(&cursor[(int)(held[u] >> 57)], 1);
                if (OCTO_IN_RANGE(pos >= 0 && pos < cnt, status)) keys[pos] = held[u];
            }
        } else {
            for (int i = tid; i < cnt; i += NT) atomicAdd(&seg_cnt[(int)(__ldcg(gk + i) >> 57)], 1);
            __syncthreads();
            scan_counts();
            __syncthreads();
            // off chip the scatter goes through the box workspace and back into the key array
            unsigned long long* const dst = reinterpret_cast<unsigned long long*>(boxes);
            for (int i = tid; i < cnt; i += NT) {
                const unsigned long long k = __ldcg(gk + i);
                const int pos = atomicAdd(&cursor[(int)(k >> 57)], 1);
                if (OCTO_IN_RANGE(pos >= 0 && pos < cnt, status)) dst[pos] = k;
            }
            __syncthreads();
            for (int i = tid; i < cnt; i += NT) keys[i] = dst[i];
        }
        __syncthreads();
        // The first CTA's bucketing is finished before another CTA of the cluster writes a finished
        // class into its arrays.
        if (shared_work) cg::this_cluster().sync();

        // survivors of a class are compacted at [s, s + nk) of its segment; other CTAs hand them to the first
        auto finish_class = [&](int cls, int s, int nk, int t, int nt) {
            if (crank != 0)
                for (int p = s + t; p < s + nk; p += nt) keys0[p] = keys[p];
            if (t == 0 && nk > 0) {
                nkept0[cls] = nk;
                atomicAdd(total0, nk);
            }
        };

        // ---- large classes, by all warps of a CTA ----
        {
            __shared__ unsigned t_sup[kTeamBlock * kTeamWords];
            const int nlarge = s_nlarge;
            for (int q = (int)crank; q < nlarge; q += (int)team_ctas) {
                const int cls = s_large[q], m = seg_cnt[cls];
                const int s = seg_start[cls], e = s + m;
                // order: by counting where two threads or more share a key, else by a network
                if (2 * m <= NT) {
                    int per = 2;
                    while (2 * per * m <= NT && per < 32) per <<= 1;
                    unsigned long long* const tmp = reinterpret_cast<unsigned long long*>(boxes + s);
                    const int part = tid & (per - 1), i = tid / per;
                    const unsigned long long own = i < m ? keys[s + i] : 0ull;
                    int r = 0;
#pragma unroll 4
                    for (int j = part; j < m; j += per) r += keys[s + j] < own ? 1 : 0;
                    for (int off = per >> 1; off > 0; off >>= 1) r += __shfl_xor_sync(0xffffffffu, r, off);
                    __syncthreads();
                    if (part == 0 && i < m && OCTO_IN_RANGE(r < m, status)) tmp[r] = own;
                    __syncthreads();
                    const unsigned long long sorted = tid < m ? tmp[tid] : 0ull;
                    __syncthreads();
                    if (tid < m) keys[s + tid] = sorted;
                    __syncthreads();
                } else {
                    bitonic_cta(keys + s, m, tid, NT);
                }
                for (int p = s + tid; p < e; p += NT)
                    boxes[p] = gather_box(hbase + (size_t)(keys[p] & ((1ull << kKeyAnchorBits) - 1)) * as, es);
                int nk = 0;
                for (int c0 = s; c0 < e && nk < max_det; c0 += kTeamBlock) {
                    const int n = min(kTeamBlock, e - c0);
                    if (tid < kTeamWords) s_fate[tid] = make_uint2(0u, 0u);
                    __syncthreads();
                    {
                        // against the survivors so far: a quarter of the warps per 32 candidates
                        const int i = (warp & (kTeamWords - 1)) * 32 + lane;
                        const float4 b = i < n ? boxes[c0 + i] : make_float4(0.f, 0.f, 0.f, 0.f);
                        bool hit = false;
                        constexpr int kStep = NT / 32 / kTeamWords;
#pragma unroll 4
                        for (int j = warp / kTeamWords; j < nk; j += kStep) hit |= iou_above(boxes[s + j], b, P.iou_test);
                        const unsigned bits = __ballot_sync(0xffffffffu, hit && i < n);
                        if (lane == 0 && bits) atomicOr(&s_fate[warp & (kTeamWords - 1)].y, bits);
                    }
                    __syncthreads();
                    // among themselves
                    for (int i = warp; i < n; i += NT / 32) {
                        if ((s_fate[i >> 5].y >> (i & 31)) & 1u) continue;
                        const float4 b = boxes[c0 + i];
                        for (int w = 0; w <= i >> 5; ++w) {
                            const int j = (w << 5) + lane;
                            const bool hit = j < i && iou_above(boxes[c0 + j], b, P.iou_test);
                            const unsigned bits = __ballot_sync(0xffffffffu, hit);
                            if (lane == 0) t_sup[w * kTeamBlock + i] = bits;
                        }
                    }
                    float4 b = make_float4(0.f, 0.f, 0.f, 0.f);
                    unsigned long long k = 0ull;
                    if (tid < n) { b = boxes[c0 + tid]; k = keys[c0 + tid]; }
                    __syncthreads();
                    const int twords = (n + 31) >> 5;
                    if (warp < twords) resolve_words<kTeamBlock>(t_sup, tid, n, 0, s_fate, s_left, tid, twords);
                    __syncthreads();
                    int all = 0, before = 0;
#pragma unroll
                    for (int w = 0; w < kTeamWords; ++w) {
                        const int c = __popc(s_fate[w].x);
                        if (w < warp) before += c;
                        all += c;
                    }
                    if (tid < n && ((s_fate[warp].x >> lane) & 1u)) {
                        const int r = nk + before + __popc(s_fate[warp].x & ((1u << lane) - 1u));
                        if (r < max_det && OCTO_IN_RANGE(s + r < e, status)) {
                            boxes[s + r] = b;
                            keys[s + r] = global_key(k);
                        }
                    }
                    nk = min(nk + all, max_det);
                    __syncthreads();
                }
                finish_class(cls, s, nk, tid, NT);
            }
        }

        // ---- the other classes: one warp each, handed out by a counter, so that a warp that drew small
        // classes takes more of them ----
        for (;;) {
            int cls = 0;
            if (lane == 0) cls = atomicAdd(next0, 1);
            cls = __shfl_sync(0xffffffffu, cls, 0);
            if (cls >= 128) break;
            const int m = seg_cnt[cls];
            if (m == 0 || m > team_min) continue;
            const int s = seg_start[cls], e = s + m;
            if (m > 1) {
                // every key counts the keys below it and moves to that position, staged in the (not yet
                // used) box slots of the segment
                unsigned long long* const tmp = reinterpret_cast<unsigned long long*>(boxes + s);
                for (int i0 = lane; i0 < m; i0 += 128) {
                    // up to four keys per lane share one pass over the segment
                    const unsigned long long k0 = keys[s + i0];
                    const unsigned long long k1 = i0 + 32 < m ? keys[s + i0 + 32] : kKeySentinel;
                    const unsigned long long k2 = i0 + 64 < m ? keys[s + i0 + 64] : kKeySentinel;
                    const unsigned long long k3 = i0 + 96 < m ? keys[s + i0 + 96] : kKeySentinel;
                    int r0 = 0, r1 = 0, r2 = 0, r3 = 0;
                    for (int j = 0; j < m; ++j) {
                        const unsigned long long kj = keys[s + j];
                        r0 += kj < k0; r1 += kj < k1; r2 += kj < k2; r3 += kj < k3;
                    }
                    tmp[r0] = k0;
                    if (i0 + 32 < m) tmp[r1] = k1;
                    if (i0 + 64 < m) tmp[r2] = k2;
                    if (i0 + 96 < m) tmp[r3] = k3;
                }
                __syncwarp();
                for (int p = lane; p < m; p += 32) keys[s + p] = tmp[p];
                __syncwarp();
            }
            // boxes of the class from the head, four per lane in flight (a lone warp pays the full
            // round trip for every load it waits on)
            for (int p0 = s + lane; p0 < e; p0 += 128) {
                float4 b4[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int p = p0 + 32 * u;
                    if (p < e) {
                        const int anchor = (int)(keys[p] & ((1ull << kKeyAnchorBits) - 1));
                        b4[u] = gather_box(hbase + (size_t)anchor * as, es);
                    }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int p = p0 + 32 * u;
                    if (p < e) boxes[p] = b4[u];
                }
            }
            __syncwarp();
            int nk = 0;  // survivors of this class, compacted at [s, s + nk)
            for (int c0 = s; c0 < e && nk < max_det; c0 += 32) {
                const int p = c0 + lane;
                const bool valid = p < e;
                float4 b = make_float4(0.f, 0.f, 0.f, 0.f);
                unsigned long long k = kKeySentinel;
                if (valid) { b = boxes[p]; k = keys[p]; }
                bool alive = valid;
                // four survivors per round: the tests of a round are independent of one another, so
                // their latencies overlap (a lone warp is bound by the dependent chain, not by issue)
                for (int t = 0; t < nk; t += 4) {
                    if (!__any_sync(0xffffffffu, alive)) break;
                    const float4 k0 = boxes[s + t];
                    const float4 k1 = boxes[s + min(t + 1, nk - 1)];
                    const float4 k2 = boxes[s + min(t + 2, nk - 1)];
                    const float4 k3 = boxes[s + min(t + 3, nk - 1)];
                    bool close = false;
                    bool hit = iou_quick(k0, b, P.iou_test, close) | iou_quick(k1, b, P.iou_test, close) |
                               iou_quick(k2, b, P.iou_test, close) | iou_quick(k3, b, P.iou_test, close);
                    if (close)
                        hit = iou_above(k0, b, P.iou_test) | iou_above(k1, b, P.iou_test) |
                              iou_above(k2, b, P.iou_test) | iou_above(k3, b, P.iou_test);
                    if (hit) alive = false;
                }
                unsigned rem = __ballot_sync(0xffffffffu, alive);
                unsigned keptmask = 0;
                while (rem) {
                    const int l = __ffs(rem) - 1;
                    keptmask |= 1u << l;
                    const float4 lb = boxes[c0 + l];
                    if (alive && lane > l && iou_above(lb, b, P.iou_test)) alive = false;
                    rem = __ballot_sync(0xffffffffu, alive) & ~((2u << l) - 1u);
                }
                __syncwarp();
                const int allowed = min(__popc(keptmask), max_det - nk);
                if ((keptmask >> lane) & 1u) {
                    const int r = __popc(keptmask & ((1u << lane) - 1u));
                    if (r < allowed && OCTO_IN_RANGE(s + nk + r < e, status)) {
                        boxes[s + nk + r] = b;
                        keys[s + nk + r] = global_key(k);
                    }
                }
                __syncwarp();
                nk += allowed;
            }
            finish_class(cls, s, nk, lane, 32);
        }
        if (shared_work) {
            cg::this_cluster().sync();  // every class has arrived in the first CTA's arrays
            if (crank != 0) return;
        } else {
            __syncthreads();
        }

        // ---- global score order: the survivor lists are packed into the memory of the (dead) boxes and
        // put in order there ----
        if (warp == 0) scan_classes(lane, nkept, cursor);
        __syncthreads();
        const int total = s_total;
        unsigned long long* const packed = reinterpret_cast<unsigned long long*>(boxes);
        for (int cls = warp; cls < 128; cls += NT / 32) {
            const int m = nkept[cls], from = seg_start[cls], to = cursor[cls];
            for (int i = lane; i < m; i += 32)
                if (OCTO_IN_RANGE(to + i >= 0 && to + i < total && total <= cnt, status)) packed[to + i] = keys[from + i];
        }
        // (a box slot is twice a key, and total <= cnt: the padded list, its ranks and the ordered list fit)
        if (tid == 0) packed[total] = kKeySentinel;
        nout = min(total, max_det);
        const int mwords = max((total + 31) >> 5, 1);
        if (2 * mwords <= NT / 32) {
            int* const rank = reinterpret_cast<int*>(keys);  // (dead as well once packed)
            ordered = packed + ((total + 2) & ~1);
            __syncthreads();
            for (int i = tid; i < total; i += NT) rank[i] = 0;
            __syncthreads();
            const int q = (warp % mwords) * 32 + lane, part = warp / mwords, mparts = (NT / 32) / mwords;
            unsigned long long g = 0ull;
            if (q < total && part < mparts) {
                g = packed[q];
                const int r = count_below(packed, 0, total, g, part, mparts);
                if (r) atomicAdd(&rank[q], r);
            }
            __syncthreads();
            if (q < total && part == 0) {
                const int r = rank[q];
                if (r < max_det && OCTO_IN_RANGE(r >= 0 && r < total, status)) ordered[r] = g;
            }
            __syncthreads();
        } else {
            ordered = packed;
            bitonic_cta(ordered, total, tid, NT);
        }
        if (!P.class_agnostic) {
            for (int r = tid; r < nout; r += NT) {
                const unsigned long long g = ordered[r];
                const int anchor = (int)((g >> 7) & ((1ull << kKeyAnchorBits) - 1));
                map.write(dets + r, gather_box(hbase + (size_t)anchor * as, es), g, (int)(g & 127u));
            }
        }
    }
    __syncthreads();
    if (P.class_agnostic) {
        // NMS ran with every candidate in class 0: a warp recovers the real class (first maximum)
        for (int r = warp; r < nout; r += NT / 32) {
            const unsigned long long g = ordered[r];
            const int anchor = (int)((g >> 7) & ((1ull << kKeyAnchorBits) - 1));
            const float* __restrict__ row = hbase + (size_t)anchor * as;
            const float* __restrict__ cv = row + (size_t)nbox * es;
            float best = -INFINITY;
            int cls = 0x7fffffff;
            float v[OCTO_MAX_CLASSES / 32];
#pragma unroll
            for (int u = 0; u < OCTO_MAX_CLASSES / 32; ++u)
                v[u] = lane + 32 * u < P.C ? __ldg(cv + (size_t)(lane + 32 * u) * es) : -INFINITY;
            const float4 b = gather_box(row, es);
#pragma unroll
            for (int u = 0; u < OCTO_MAX_CLASSES / 32; ++u)
                if (v[u] > best) { best = v[u]; cls = lane + 32 * u; }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                const float ov = __shfl_xor_sync(0xffffffffu, best, off);
                const int oc = __shfl_xor_sync(0xffffffffu, cls, off);
                if (ov > best || (ov == best && oc < cls)) { best = ov; cls = oc; }
            }
            __syncwarp();
            if (lane == 0) {
                map.write(dets + r, b, g, cls);
                ordered[r] = (g & ~127ull) | (unsigned long long)cls;  // for the branch lists
            }
        }
        __syncthreads();
    }
    if (tid == NT - 1) {
        P.counts[img] = nout;
        // a branch that takes every class has no index list: item j of an image is its detection j
        for (int b = 0; b < P.num_branches; ++b)
            if ((P.full_branches >> b) & 1) P.bcount[b * P.max_batch + img] = nout;
        atomicAdd(&P.ctr->kept, (unsigned long long)nout);
    }
    // ---- index lists of the other branches, filtered by class (stable), one warp per branch ----
    if (warp < P.num_branches && !((P.full_branches >> warp) & 1)) {
        int m = 0;
        int* const list = P.bidx + ((size_t)warp * P.max_batch + img) * max_det;
        for (int r0 = 0; r0 < nout; r0 += 32) {
            const int r = r0 + lane;
            bool take = false;
            if (r < nout) {
                const unsigned cls = (unsigned)(ordered[r] & 127u);
                take = (s_mask[warp][cls >> 5] >> (cls & 31u)) & 1u;
            }
            const unsigned bal = __ballot_sync(0xffffffffu, take);
            if (take && OCTO_IN_RANGE(m + __popc(bal & ((1u << lane) - 1u)) < max_det, status))
                list[m + __popc(bal & ((1u << lane) - 1u))] = r;
            m += __popc(bal);
        }
        if (lane == 0) P.bcount[warp * P.max_batch + img] = m;
    }
}

}  // namespace octo
