// Per-image ordering + class-aware greedy NMS + cap + scale-back, as device code of one CTA (or of a
// thread-block cluster) per image.
//
// Latency / shared-memory bound; bytes are negligible.  Keys are (class | inverted score bits | anchor),
// so the ascending order of the keys of a class is its NMS order.
//
// Candidates are worked on in batches of whole classes, one thread (or up to four) per candidate
// (nms_batch): put in order (by counting inside a class, or inside its score bucket; where one is large, words
// of 32 by counting, then every candidate's place in every word by binary search); each tested against the
// earlier candidates of its class (one bit each); which survive is settled word by word of those bits
// (resolve_words), in a time that follows the length of the chains of overlapping
// boxes, not the number of candidates of a class.  Up to kSmallMax candidates (the usual case in serving) are
// one batch; more are bucketed by class first (histogram, scan, scatter) and cut into about as many
// batches as the image has CTAs; on one CTA many small classes are taken by a warp each instead (kWarpShare).
// Survivors are re-keyed to (inverted score | anchor | class) and put in order by counting, by score buckets or
// (more than threads) by a network.  Boxes: as the decode step left them beside the keys for the short path, for
// batches on chip and for records while no class went to a warp or to the whole CTA; from the head otherwise.
// us per launch (CUDA events), against one thread per class that walked its candidates (and one warp per
// class above 256): 200 candidates of one class, 8 images, 16.8 (67.4), of 7 classes 13.9 (28.3), of 80 classes
// 12.7 (12.6); 90 candidates under class-agnostic NMS 12.7 (35.7); 5000 candidates of 80 classes, one image
// on a cluster of 8, 38.8 (54).  What is left is bound by the latency of a dozen short phases and, in one
// large class, by the pair tests (shared-memory return bandwidth: 20 bytes per lane and test).
//
// A class of more candidates than half the CTA's threads is taken by the whole CTA, kTeamBlock at a time:
// sorted by a network, survivor tests, suppression bits and settling spread over all warps (1200 candidates
// of one class, 4 images: 87 us; 464 when one warp had the class to itself).
//
// Images with more candidates than fit in shared memory take the same code path with the arrays in a
// global-memory workspace.
//
// A cluster of CTAs per image (crowded scenes at small batches): every CTA buckets the image's keys for
// itself, the batches (and the large classes) go to the CTAs in turn, and the survivors of each are written
// into the first CTA's arrays through distributed shared memory.  The first CTA alone orders and writes the
// image's results.
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
constexpr int kSmallMax = 512;      // up to here an image takes the short path, above it a cluster is worth while
constexpr int kTeamBlock = 128;     // candidates of a large class that the CTA works on together
constexpr int kTeamWords = kTeamBlock / 32;
constexpr int kBatchRows = 17;      // words of 32 that a class of a batch reaches over (512 candidates)
constexpr int kMaxBatches = 128;    // 128 classes of at most half a CTA's threads, in batches that hold at least that
constexpr int kCountMax = 96;       // so many survivors are put in order by counting, more by score buckets
constexpr int kSubs = 16;           // score buckets of a class of a crowded image
constexpr float kSubScale = 20.0f;  // ... of 1 / 20 each; scores below 1/4 share the last
constexpr int kCountedMax = 128;    // a batch without larger classes orders its candidates by counting
// An image on one CTA whose largest class is at most kWarpShare of its candidates (above kSmallMax) and at most
// kWarpClassMax candidates has its classes worked on by one warp each, side by side, instead of in batches one
// after the other: a warp tests against survivors only, but has a class to itself.  Which is better depends on how
// many boxes survive, which is not known here.  Time of the batches over that of the warps (80 images): boxes in
// clusters of twenty, 5000 of 80 classes 1.26, 2000 of 10 1.34, 5000 of 7 0.99, 8000 of 10 1.02, of 6 (1340 a class) 0.58; boxes
// that hardly overlap, 5000 of 80 1.00, 2000 of 10 0.67.  The share lies above a fifth because five classes are rarely
// even (850 of 5, one image: 41 us in batches, 34 by warps).
constexpr float kWarpShare = 0.235f;
constexpr int kWarpClassMax = 1280;
constexpr int kWarpRankMax = 512;  // up to here a warp orders a class by counting, above by a network (80 images,
                                   // 8000 candidates of 10 clustered classes: 554 us by counting, 362 so)
constexpr int kCrowdedMin = 1024;  // an image with more candidates than this wants full-sized CTAs

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

// Bucket 0 .. buckets - 1 of a class | inverted score | anchor key by its score: falls as the score rises (the
// subtraction and the product round monotonously), so buckets are in the order of the keys of a class.
__device__ __forceinline__ int score_bucket(unsigned long long k, int buckets, float scale) {
    const float score = __uint_as_float(~(unsigned)(k >> kKeyAnchorBits));
    return min(max(__float2int_rz(__fmul_rn(__fsub_rn(1.0f, score), scale)), 0), buckets - 1);
}

__device__ __forceinline__ void cmp_swap(unsigned long long* __restrict__ k, int i, int j) {
    const unsigned long long a = k[i], b = k[j];
    if (a > b) { k[i] = b; k[j] = a; }
}

// Ascending bitonic sort of k[0, m) for any m by the whole CTA or (CTA = false) by one warp.  Every comparator puts
// the smaller key at the lower index (the first stage of each merge pairs mirrored positions), so positions >= m
// can stand for +infinity and are simply skipped.
template <bool CTA>
__device__ __forceinline__ void bitonic_range(unsigned long long* __restrict__ k, int m, int tid, int nthreads) {
    auto barrier = []() {
        if (CTA) __syncthreads(); else __syncwarp();
    };
    int np2 = 2;
    while (np2 < m) np2 <<= 1;
    const int half = np2 >> 1;
    for (int size = 2; size <= np2; size <<= 1) {
        barrier();
        const int h = size >> 1;
        for (int t = tid; t < half; t += nthreads) {
            const int off = t & (h - 1);
            const int i = 2 * t - off;             // block start + off
            const int j = i + size - 1 - 2 * off;  // mirrored position in the block
            if (j < m) cmp_swap(k, i, j);
        }
        for (int stride = size >> 2; stride > 0; stride >>= 1) {
            barrier();
            for (int t = tid; t < half; t += nthreads) {
                const int i = 2 * t - (t & (stride - 1));
                const int j = i + stride;
                if (j < m) cmp_swap(k, i, j);
            }
        }
    }
    barrier();
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
// cand] (w counted from w0): the bits of the earlier candidates that suppress it, in the words w0 .. own.
// fate[w] = (kept, gone): gone may already hold candidates that are out.
// A candidate is removed once one of its suppressors survives and survives once all of them are removed.
// In every round all words settle what they can (ballots inside the warp, one per link of a chain of
// overlapping boxes) and learn what the earlier words found in the round before.  The first undecided word
// of a class has only its own chains left, so there are at most as many rounds as a class has words.
template <int LEN>
__device__ __forceinline__ void resolve_words(const unsigned* sup, int cand, int n, int w0, volatile uint2* fate, int tid,
                                              int words) {
    const int lane = tid & 31, word = tid >> 5;
    unsigned kept = 0u, gone = fate[word].y;
    bool open = cand < n && !((gone >> lane) & 1u), out = false;
    const unsigned own = open ? sup[(word - w0) * LEN + cand] : 0u;
    unsigned undecided = __ballot_sync(0xffffffffu, open);
    unsigned ask = 0u;  // earlier words with a suppressor that is not decided yet
    if (open)
        for (int w = w0; w < word; ++w)
            if (sup[(w - w0) * LEN + cand]) ask |= 1u << w;
    for (;;) {
        while (undecided != 0u) {
            const bool dies = open && (out || (own & kept) != 0u);
            const bool lives = open && !dies && ask == 0u && (own & ~gone) == 0u;
            const unsigned k = __ballot_sync(0xffffffffu, lives), g = __ballot_sync(0xffffffffu, dies);
            if ((k | g) == 0u) break;
            kept |= k;
            gone |= g;
            undecided &= ~(k | g);
            open = open && !dies && !lives;
        }
        // (both words only gain bits, so a warp that still looks at the round before may read either)
        if (lane == 0) { fate[word].x = kept; fate[word].y = gone; }
        if (!bar_any(words * 32, open)) break;
        if (open) {
            for (unsigned todo = ask; todo != 0u; todo &= todo - 1u) {
                const int w = __ffs(todo) - 1;
                const unsigned b = sup[(w - w0) * LEN + cand], k = fate[w].x, g = fate[w].y;
                if (b & k) { out = true; break; }
                if ((b & ~g) == 0u) ask &= ~(1u << w);
            }
        }
    }
}

// Head boxes to source-frame pixels.
struct RegionMap {
    float fpl, fpt, gx, gy, x_lo, y_lo, x_hi, y_hi;
    __device__ __forceinline__ explicit RegionMap(const FrameDesc& fd)
        : fpl((float)fd.pad_l), fpt((float)fd.pad_t), gx(fd.gx), gy(fd.gy), x_lo((float)fd.ox), y_lo((float)fd.oy),
          x_hi((float)(fd.ox + fd.rw)), y_hi((float)(fd.oy + fd.rh)) {}
    // Word k of the record of a survivor (x1, y1, x2, y2, score, class, anchor, pad); box: its corners in head
    // pixels.  X = fl(fl(fl(x - pad) * gain) + origin), clamped to the region the detector input shows.
    __device__ __forceinline__ unsigned word(int k, float corner, unsigned long long g) const {
        if (k < 4) {
            const bool y = (k & 1) != 0;
            const float lo = y ? y_lo : x_lo, hi = y ? y_hi : x_hi;
            const float v = __fadd_rn(__fmul_rn(__fsub_rn(corner, y ? fpt : fpl), y ? gy : gx), lo);
            return __float_as_uint(fminf(fmaxf(v, lo), hi));
        }
        if (k == 4) return ~(unsigned)(g >> 32);
        if (k == 5) return (unsigned)(g & 127u);
        return k == 6 ? (unsigned)((g >> 7) & ((1ull << kKeyAnchorBits) - 1)) : 0u;
    }
    __device__ __forceinline__ void write(octo_det_rec* out, const float4 b, unsigned long long g) const {
        unsigned* const o = reinterpret_cast<unsigned*>(out);
        o[0] = word(0, b.x, g); o[1] = word(1, b.y, g); o[2] = word(2, b.z, g); o[3] = word(3, b.w, g);
        o[4] = word(4, 0.f, g); o[5] = word(5, 0.f, g); o[6] = word(6, 0.f, g); o[7] = 0u;
    }
};

// Finds the place of the m (<= NT) survivors in list / lpos in the output order: emit(place, key, pos), one
// thread per survivor.  Few by counting; more are dealt to 256 buckets by score first and counted inside their
// bucket (766 survivors of a crowded image: 8 K cycles; 28 K with a network over all of them).  list has room for
// a pad; tmp: NT + 2 keys, rank: NT integers.  All threads of the CTA; ends with a barrier.
template <int NT, typename Emit>
__device__ __forceinline__ void order_survivors(unsigned long long* list, const unsigned short* lpos, int m,
                                                unsigned long long* tmp, int* rank, int tid, Emit emit) {
    constexpr int kBuckets = 256;
    const int lane = tid & 31, warp = tid >> 5;
    if (m <= kCountMax) {
        if (tid < m) rank[tid] = 0;
        if (tid == 0) list[m] = kKeySentinel;
        __syncthreads();
        const int words = max((m + 31) >> 5, 1), q = (warp % words) * 32 + lane, part = warp / words;
        unsigned long long g = 0ull;
        if (q < m && part < 4) {
            g = list[q];
            const int r = count_below(list, 0, m, g, part, 4);
            if (r) atomicAdd(&rank[q], r);
        }
        __syncthreads();
        if (q < m && part == 0) emit(rank[q], g, lpos[q]);
    } else {
        if (tid < kBuckets) rank[tid] = 0;
        if (tid == 0) tmp[m] = kKeySentinel;
        unsigned long long g = 0ull;
        unsigned short pos = 0;
        int bucket = 0, at = 0;
        if (tid < m) {
            g = list[tid];
            pos = lpos[tid];
            bucket = score_bucket(g >> 7, kBuckets, (float)kBuckets);
        }
        __syncthreads();
        if (tid < m) at = atomicAdd(&rank[bucket], 1);
        __syncthreads();
        if (warp == 0) {
            int v[kBuckets / 32], sum = 0;
#pragma unroll
            for (int u = 0; u < kBuckets / 32; ++u) { v[u] = rank[lane * (kBuckets / 32) + u]; sum += v[u]; }
            int inc = sum;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, inc, off);
                if (lane >= off) inc += u;
            }
            int run = inc - sum;
#pragma unroll
            for (int u = 0; u < kBuckets / 32; ++u) {
                rank[lane * (kBuckets / 32) + u] = run;
                run += v[u];
            }
        }
        __syncthreads();
        const int lo = rank[bucket], hi = bucket + 1 < kBuckets ? rank[bucket + 1] : m;
        if (tid < m) tmp[lo + at] = g;
        __syncthreads();
        if (tid < m) emit(lo + count_below(tmp, lo, hi, g, 0, 1), g, pos);
    }
    __syncthreads();
}

// Shared memory of one batch of up to B candidates (nms_batch).
template <int B>
struct BatchMem {
    unsigned long long *wkey, *skey;  // every word of 32 in order; all in order (first: as they came)
    float4* sbox;                     // ... their boxes
    float* sshare;                    // ... and shares (iou_share)
    unsigned* sup;                    // [kBatchRows][B] suppression bits, rows counted from the class's first word
    int* rank;
    unsigned short* sstart;           // first candidate of the class
    __device__ __forceinline__ explicit BatchMem(unsigned char* p) {
        wkey = reinterpret_cast<unsigned long long*>(p);
        skey = wkey + B;
        sbox = reinterpret_cast<float4*>(skey + B);
        sshare = reinterpret_cast<float*>(sbox + B);
        sup = reinterpret_cast<unsigned*>(sshare + B);
        rank = reinterpret_cast<int*>(sup + kBatchRows * B);
        sstart = reinterpret_cast<unsigned short*>(rank + B);
    }
    static constexpr size_t kBytes = (size_t)B * (8 + 8 + 16 + 4 + 4 * kBatchRows + 4 + 2);
};

// Greedy NMS of m (<= B) candidates of whole classes, none of more than 512, by so many warps: thread c < m brings candidate
// c (key, box); on return mem.skey / mem.sbox hold them ordered by class and score and fate[w].x says which
// of them survive, as one bit each: bit l of word w is candidate batch_cand(32 w + l).  class_start: where a
// class begins.  bucketed: thread c's candidate lies in a bucket of mem.skey (which has a pad), buckets in
// ascending order of their keys; range(key, lo, hi) gives the bucket, and the order comes from counting
// inside it; else from words of 32 and binary search.  All threads of the CTA, after a barrier.
__device__ __forceinline__ int batch_cand(int tid) { return (tid & ~31) | ((tid & 7) << 2) | ((tid >> 3) & 3); }

template <int B, typename Start, typename Range>
__device__ __forceinline__ void nms_batch(const BatchMem<B>& mem, int warps, unsigned long long key, const float4 box, int m,
                                          bool bucketed, const IouTest& test, uint2* fate, unsigned int* status,
                                          Start class_start, Range range) {
    (void)status;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // Thread (candidate c = word * 32 + lane, part): the 4, 2 or 1 parts of a candidate's work are warps, and
    // the lanes of a warp read the same shared-memory words as they walk.  Part 0 of candidate c is thread
    // c, which holds its key and box in registers.
    const int words = (m + 31) >> 5;
    const int parts = 4 * words <= warps ? 4 : 2 * words <= warps ? 2 : 1;
    const int word = warp % max(words, 1), part = warp / max(words, 1);  // part >= parts: nothing to do
    const int c = word * 32 + lane;
    const bool busy = part < parts && c < m;
    if (tid < 32) fate[tid] = make_uint2(0u, 0u);
    if (!bucketed) {
        if (warp < words) {
            if (tid >= m) key = kKeySentinel;
            mem.skey[tid] = key;
            __syncwarp();
            // order inside the word: the keys of its 32 that are below one's own
            int r = 0;
#pragma unroll 4
            for (int j = 0; j < 32; j += 2) {
                const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(mem.skey + (tid & ~31) + j);
                r += (v.x < key ? 1 : 0) + (v.y < key ? 1 : 0);
            }
            mem.wkey[tid < m ? (tid & ~31) + r : tid] = key;
        }
        if (tid < m) mem.rank[tid] = 0;
        __syncthreads();
        // place among all candidates: its place in every word, by binary search
        if (busy) {
            const unsigned long long own = mem.skey[c];
            int r = 0;
            for (int w = part; w < words; w += 2 * parts) {  // two words side by side
                const unsigned long long* const k0 = mem.wkey + 32 * w;
                const unsigned long long* const k1 = mem.wkey + 32 * min(w + parts, words - 1);
                int lo0 = 0, lo1 = 0;
#pragma unroll 1
                for (int step = 16; step > 0; step >>= 1) {
                    lo0 += k0[lo0 + step - 1] < own ? step : 0;
                    lo1 += k1[lo1 + step - 1] < own ? step : 0;
                }
                r += lo0 + (k0[lo0] < own ? 1 : 0);
                if (w + parts < words) r += lo1 + (k1[lo1] < own ? 1 : 0);
            }
            if (r) atomicAdd(&mem.rank[c], r);
        }
    } else if (busy) {
        const unsigned long long own = mem.skey[c];
        int lo, hi;
        range(own, lo, hi);
        const int r = (part == 0 ? lo : 0) + count_below(mem.skey, lo, hi, own, part, parts);
        if (r) atomicAdd(&mem.rank[c], r);  // (zero on entry)
    }
    __syncthreads();
    if (tid < m) {
        const int at = mem.rank[tid];
        if (OCTO_IN_RANGE(at >= 0 && at < m, status)) {
            mem.skey[at] = key;
            mem.sbox[at] = box;
            mem.sshare[at] = iou_share(box, test);
            mem.sstart[at] = (unsigned short)class_start((int)(key >> 57));
        }
    }
    __syncthreads();
    // Suppression bits.  Candidates j % 4 = p give byte p of a word (candidate j of a word has bit (j & 3)
    // * 8 + j / 4), so that parts never share one.
    if (busy) {
        const float4 b = mem.sbox[c];
        const float own_share = mem.sshare[c];
        const int start = mem.sstart[c], w0 = start >> 5, rows = (c >> 5) - w0;
        unsigned char* const to = reinterpret_cast<unsigned char*>(mem.sup + c);
        const bool room = OCTO_IN_RANGE(rows >= 0 && rows < kBatchRows, status);
        if (!__any_sync(__activemask(), c - start > 96)) {
            // small classes: only the pairs there are, bits of four words at most
            for (int p = part; p < 4; p += parts) {
                const int first = start + ((p - start) & 3);
                unsigned bits = 0u;
                bool close = false;
#pragma unroll 2
                for (int j = first; j < c; j += 4)
                    if (iou_by_share(mem.sbox[j], mem.sshare[j], b, own_share, close)) bits |= 1u << ((j >> 2) - 8 * w0);
                if (close) {  // rare: some pair lies too near the threshold for binary32
                    bits = 0u;
                    for (int j = first; j < c; j += 4)
                        if (iou_above(mem.sbox[j], b, test)) bits |= 1u << ((j >> 2) - 8 * w0);
                }
                to[p] = (unsigned char)bits;
                for (int w = 1; w <= rows && room; ++w) to[4 * B * w + p] = (unsigned char)(bits >> (8 * w));
            }
        } else if (room) {
            // a byte is tested whole (the lanes read the same boxes) and what is not an earlier candidate of
            // the class is masked off
            for (int p = part; p < 4; p += parts) {
                for (int w = w0; w <= c >> 5; ++w) {
                    const int base = 32 * w + p;
                    const int lo = max((start - base + 3) >> 2, 0), hi = max(min((c - base + 3) >> 2, 8), 0);
                    unsigned bits = 0u;
                    bool close = false;
#pragma unroll
                    for (int t = 0; t < 8; ++t)
                        if (iou_by_share(mem.sbox[base + 4 * t], mem.sshare[base + 4 * t], b, own_share, close)) bits |= 1u << t;
                    if (close) {
                        bits = 0u;
                        for (int t = lo; t < hi; ++t)
                            if (iou_above(mem.sbox[base + 4 * t], b, test)) bits |= 1u << t;
                    }
                    to[4 * B * (w - w0) + p] = (unsigned char)(bits & (0xffu << lo) & (0xffu >> (8 - hi)));
                }
            }
        }
    }
    __syncthreads();
    const int cand = batch_cand(tid);
    if (warp < words) resolve_words<B>(mem.sup, cand, m, cand < m ? mem.sstart[cand] >> 5 : 0, fate, tid, words);
    __syncthreads();
}

// Number of survivors in the words of `fate` before word `warp`, and of all of them (`words` <= 32).
__device__ __forceinline__ int kept_before(const uint2* fate, int words, int lane, int warp, int& all) {
    int inc = lane < words ? __popc(fate[lane].x) : 0;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, inc, off);
        if (lane >= off) inc += u;
    }
    all = __shfl_sync(0xffffffffu, inc, 31);
    const int before = __shfl_sync(0xffffffffu, inc, max(warp - 1, 0));
    return warp == 0 ? 0 : before;
}

// One class, the candidates [s, s + m), by one warp: keys ordered, boxes gathered from the head, each candidate tested
// against the survivors before it.  Survivors (at most max_det) are left at the start, re-keyed; returns their number.
__device__ __forceinline__ int warp_class(unsigned long long* keys, float4* boxes, int s, int m, int max_det,
                                          const float* __restrict__ hbase, size_t as, size_t es, const IouTest& test,
                                          int lane, unsigned int* status) {
    (void)status;
    const int e = s + m;
    if (m > kWarpRankMax) {
        bitonic_range<false>(keys + s, m, lane, 32);
    } else if (m > 1) {
        // every key counts the keys below it and moves to that position, staged in the (not yet used) box slots
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
            if (OCTO_IN_RANGE(r0 < m, status)) tmp[r0] = k0;
            if (i0 + 32 < m && OCTO_IN_RANGE(r1 < m, status)) tmp[r1] = k1;
            if (i0 + 64 < m && OCTO_IN_RANGE(r2 < m, status)) tmp[r2] = k2;
            if (i0 + 96 < m && OCTO_IN_RANGE(r3 < m, status)) tmp[r3] = k3;
        }
        __syncwarp();
        for (int p = lane; p < m; p += 32) keys[s + p] = tmp[p];
        __syncwarp();
    }
    // four boxes per lane in flight (a lone warp pays the full round trip for every load it waits on)
    for (int p0 = s + lane; p0 < e; p0 += 128) {
        float4 b4[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int p = p0 + 32 * u;
            if (p < e) b4[u] = gather_box(hbase + (size_t)(int)(keys[p] & ((1ull << kKeyAnchorBits) - 1)) * as, es);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int p = p0 + 32 * u;
            if (p < e) boxes[p] = b4[u];
        }
    }
    __syncwarp();
    int nk = 0;
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
            bool hit = iou_quick(k0, b, test, close) | iou_quick(k1, b, test, close) | iou_quick(k2, b, test, close) |
                       iou_quick(k3, b, test, close);
            if (close) hit = iou_above(k0, b, test) | iou_above(k1, b, test) | iou_above(k2, b, test) | iou_above(k3, b, test);
            if (hit) alive = false;
        }
        unsigned rem = __ballot_sync(0xffffffffu, alive);
        unsigned keptmask = 0;
        while (rem) {
            const int l = __ffs(rem) - 1;
            keptmask |= 1u << l;
            const float4 lb = boxes[c0 + l];
            if (alive && lane > l && iou_above(lb, b, test)) alive = false;
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
    return nk;
}

// NMS of image `img` by a CTA of NT threads (SMEM_CAP candidates on chip), or by the cluster the CTA
// belongs to when CLUSTER.  The image's candidate count, keys and (for the short path) boxes are in
// global memory.
template <int NT, int SMEM_CAP, bool CLUSTER>
__device__ __forceinline__ void nms_image(const NmsParams& P, const FrameDesc& fd, bool no_frame, int img,
                                          unsigned char* smem_raw) {
    __shared__ __align__(16) int seg_start[128], seg_cnt[128], cursor[128], nkept[128];
    __shared__ unsigned s_mask[OCTO_MAX_BRANCHES][4];
    __shared__ int s_total, s_nlarge, s_nbatch, s_pack, s_most, s_next;
    __shared__ bool s_by_warps;
    __shared__ unsigned char s_large[128];
    __shared__ int s_lo[kMaxBatches], s_hi[kMaxBatches], s_kept[kMaxBatches];  // batches: range of keys, survivors
    __shared__ uint2 s_fate[32];  // see resolve_words
    __shared__ __align__(16) int s_sub[128 * kSubs];  // crowded images: keys per class and score bucket, then where it begins
    static_assert(BatchMem<NT>::kBytes + 16 + 2 * SMEM_CAP <= (size_t)SMEM_CAP * sizeof(float4),
                  "a batch and the slots of all keys fit the memory of the boxes");
    constexpr int kShort = kSmallMax;  // candidates of the short path, and threads of its smaller form
    static_assert(NT == kShort || NT == 2 * kShort, "a thread for every candidate of the short path");
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
    for (int i = tid; i < 128 * kSubs / 4; i += NT) reinterpret_cast<int4*>(s_sub)[i] = make_int4(0, 0, 0, 0);
    if (tid < OCTO_MAX_BRANCHES * 4) s_mask[tid >> 2][tid & 3] = P.masks.m[tid >> 2][tid & 3];
    if (tid < kMaxBatches) { s_lo[tid] = 0x7fffffff; s_hi[tid] = 0; s_kept[tid] = 0; }
    if (tid == 0) { s_total = 0; s_pack = 0; s_next = 0; }
    // every CTA of the image has read the count, and the first CTA's counters are set, before the
    // count is cleared and before any CTA touches those counters
    if (CLUSTER && csize > 1) cg::this_cluster().sync(); else __syncthreads();
    if (tid == NT - 1 && crank == 0) {  // (a warp that has no other work on the short path)
        P.cand_count[img] = 0;  // ready for the next batch's decode
        atomicAdd(&P.ctr->candidates, (unsigned long long)cnt);
        atomicMax(&P.ctr->max_cand, cnt);
        // (only images beyond the short path write: a store to host memory delays the end of the kernel by a PCIe
        // round trip, which a sparse launch of ten microseconds would feel)
        if (P.dense_seen && cnt > kSmallMax) P.dense_seen[1] = P.launch_seq;
        if (P.dense_seen && cnt > kCrowdedMin) P.dense_seen[0] = P.launch_seq;
    }

    octo_det_rec* const dets = P.dets + (size_t)img * max_det;
    const RegionMap map(fd);
    unsigned long long* ordered;  // survivors in output order (inverted score | anchor | class)
    unsigned short* opos = nullptr;    // ... and where their boxes lie in boxes_at (null: in the head)
    const float4* boxes_at = nullptr;
    bool written = false;  // the records are
    int nout;
    int nt = NT;  // threads that go on
    if (cnt <= kSmallMax) {
        // The first CTA alone (no cluster barrier follows on this path).  Up to 256 candidates 512 of its threads go on:
        // the barriers of the short phases are between 16 warps instead of 32, and a candidate still has two threads.
        // Decode and NMS of one image with 1024 threads / with 512, us: 40 candidates 8.4 / 7.3, 128 of 7 classes 9.1 / 8.0,
        // 256 of one class 17.2 / 16.9, 300 of one class 18.6 / 20.0, class-agnostic 20.1 / 22.2.
        if (NT > kShort && cnt <= kShort / 2) nt = kShort;
        if (crank != 0 || tid >= nt) return;
        const BatchMem<kShort> mem(smem_raw);
        int pos = 0;
        if (tid < cnt) pos = atomicAdd(&seg_cnt[(int)(first_key >> 57)], 1);
        if (tid < cnt) mem.rank[tid] = 0;
        if (tid == 0) mem.skey[cnt] = kKeySentinel;  // (a key more than fits when cnt is kShort: never read then)
        __syncthreads();
        if (warp == 0) {  // where each class starts, and the largest
            scan_classes(lane, seg_cnt, seg_start);
            const int4 v = *reinterpret_cast<const int4*>(&seg_cnt[4 * lane]);
            const int most = __reduce_max_sync(0xffffffffu, max(max(v.x, v.y), max(v.z, v.w)));
            if (lane == 0) s_most = most;
        }
        __syncthreads();
        const bool bucketed = s_most <= kCountedMax;
        if (bucketed) {
            float4* const ubox = reinterpret_cast<float4*>(mem.sup);
            if (tid < cnt) {
                const int at = seg_start[(int)(first_key >> 57)] + pos;
                if (OCTO_IN_RANGE(at >= 0 && at < cnt, status)) {
                    mem.skey[at] = first_key;
                    ubox[at] = first_box;
                }
            }
            __syncthreads();
            if (tid < cnt) {
                first_key = mem.skey[tid];
                first_box = ubox[tid];
            }
        }
        nms_batch<kShort>(mem, nt / 32, first_key, first_box, cnt, bucketed, P.iou_test, s_fate, status,
                      [&](int cls) { return seg_start[cls]; },
                      [&](unsigned long long k, int& lo, int& hi) {
                          lo = seg_start[(int)(k >> 57)];
                          hi = lo + seg_cnt[(int)(k >> 57)];
                      });
        // survivors (the ordered keys' other arrays are free again)
        unsigned long long* const surv = mem.wkey;
        unsigned short* const spos = reinterpret_cast<unsigned short*>(mem.sup);
        const int words = (cnt + 31) >> 5, cand = batch_cand(tid);
        int m = 0;
        const int before = kept_before(s_fate, words, lane, warp, m);
        const unsigned kept = warp < words ? s_fate[warp].x : 0u;
        if ((kept >> lane) & 1u) {
            const int q = before + __popc(kept & ((1u << lane) - 1u));
            surv[q] = global_key(mem.skey[cand]);
            spos[q] = (unsigned short)cand;
        }
        nout = min(m, max_det);
        opos = spos + kShort;
        unsigned long long* const tmp = reinterpret_cast<unsigned long long*>(spos + 2 * kShort);
        ordered = tmp + kShort + 2;
        __syncthreads();
        order_survivors<kShort>(surv, spos, m, tmp, mem.rank, tid, [&](int r, unsigned long long g, int at) {
            if (r >= max_det || !OCTO_IN_RANGE(r >= 0 && r < m && at < cnt, status)) return;
            ordered[r] = g;
            if (P.class_agnostic) opos[r] = (unsigned short)at;
            else map.write(dets + r, mem.sbox[at], g);
        });
        if (P.class_agnostic) boxes_at = mem.sbox;
        else written = true;
    } else {
        const bool on_chip = cnt <= SMEM_CAP;
        unsigned short* slots = nullptr;  // on chip: where a key came from, hence where its box lies
        unsigned long long* keys;
        float4* boxes;
        if (on_chip) {
            boxes = reinterpret_cast<float4*>(smem_raw);
            keys = reinterpret_cast<unsigned long long*>(smem_raw + (size_t)SMEM_CAP * sizeof(float4));
            slots = reinterpret_cast<unsigned short*>(smem_raw + ((BatchMem<NT>::kBytes + 15) & ~(size_t)15));
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
        unsigned short* slots0 = slots;
        int *nkept0 = nkept, *kept0 = s_kept, *total0 = &s_total;
        if (shared_work) {
            cg::cluster_group cluster = cg::this_cluster();
            keys0 = cluster.map_shared_rank(keys, 0);
            nkept0 = cluster.map_shared_rank(nkept, 0);
            total0 = cluster.map_shared_rank(&s_total, 0);
            kept0 = cluster.map_shared_rank(s_kept, 0);
            slots0 = cluster.map_shared_rank(slots, 0);
        }

        // ---- bucket the keys by class: histogram, scan, scatter.  Classes of more than kTeamMin candidates
        // come last; the others are cut into batches of whole classes, about as many as there are CTAs ----
        constexpr int kTeamMin = NT / 2;
        static_assert(kTeamMin <= 32 * (kBatchRows - 1), "rows of the suppression bits");
        auto scan_counts = [&]() {
            if (warp != 0) return;
            int nb = 0, most = 0;
            {
                const int4 v = *reinterpret_cast<const int4*>(&seg_cnt[4 * lane]);
                const int largest = __reduce_max_sync(0xffffffffu, max(max(v.x, v.y), max(v.z, v.w)));
                const bool by_warps = team_ctas == 1u && largest <= kWarpClassMax && (float)largest <= kWarpShare * (float)cnt;
                if (lane == 0) s_by_warps = by_warps;
                if (by_warps) {  // every class with candidates is listed, none is in a batch
                    scan_classes(lane, seg_cnt, seg_start);
                    __syncwarp();
                    for (int base = 0; base < 128; base += 32) {
                        const bool is = seg_cnt[base + lane] > 0;
                        const unsigned bal = __ballot_sync(0xffffffffu, is);
                        if (is) s_large[nb + __popc(bal & ((1u << lane) - 1u))] = (unsigned char)(base + lane);
                        nb += __popc(bal);
                        cursor[base + lane] = seg_start[base + lane];
                    }
                    if (lane == 0) {
                        s_nlarge = nb;
                        s_nbatch = 0;
                        s_most = largest;
                    }
                    return;
                }
            }
            for (int base = 0; base < 128; base += 32) {
                const int v = seg_cnt[base + lane];
                const bool is = v > kTeamMin;
                const unsigned bal = __ballot_sync(0xffffffffu, is);
                if (is) s_large[nb + __popc(bal & ((1u << lane) - 1u))] = (unsigned char)(base + lane);
                nb += __popc(bal);
                cursor[base + lane] = is ? 0 : v;
                if (!is) most = max(most, v);
            }
            most = __reduce_max_sync(0xffffffffu, most);
            if (lane == 0) s_most = most;
            __syncwarp();
            scan_classes(lane, cursor, seg_start);
            __syncwarp();
            const int small = seg_start[127] + cursor[127];
            // a batch is the classes that start in one range of this many keys
            // (an equal share of as few rounds over the CTAs as the threads allow)
            const int share = (small + (int)team_ctas - 1) / (int)team_ctas, rounds = max((share + NT - most - 1) / (NT - most), 1);
            const int quota = min(max((share + rounds - 1) / rounds, 128), NT - most);
            for (int base = 0; base < 128; base += 32) {
                const int v = cursor[base + lane], s = seg_start[base + lane];
                if (v > 0 && OCTO_IN_RANGE(s / quota < kMaxBatches, status)) {
                    atomicMin(&s_lo[s / quota], s);
                    atomicMax(&s_hi[s / quota], s + v);
                }
            }
            if (lane == 0) {
                s_nlarge = nb;
                s_nbatch = min((small + quota - 1) / quota, kMaxBatches);
                int at = small;
                for (int q = 0; q < nb; ++q) {
                    seg_start[s_large[q]] = at;
                    at += seg_cnt[s_large[q]];
                }
            }
            __syncwarp();
            for (int base = 0; base < 128; base += 32) cursor[base + lane] = seg_start[base + lane];
        };
        constexpr int kHeld = SMEM_CAP / NT;  // keys a thread keeps between the two passes
        if (on_chip) {
            unsigned long long held[kHeld];
            int place[kHeld];  // class and score bucket | place in it
#pragma unroll
            for (int u = 0; u < kHeld; ++u) {
                const int i = tid + u * NT;
                held[u] = i < cnt ? __ldcg(gk + i) : kKeySentinel;
            }
#pragma unroll
            for (int u = 0; u < kHeld; ++u) {
                if (tid + u * NT >= cnt) continue;
                const int at = (int)(held[u] >> 57) * kSubs + score_bucket(held[u], kSubs, kSubScale);
                place[u] = at << 16 | atomicAdd(&s_sub[at], 1);
            }
            __syncthreads();
            if (tid < 128) {
                int4* const sub = reinterpret_cast<int4*>(&s_sub[tid * kSubs]);
                int run = 0;
#pragma unroll
                for (int u = 0; u < kSubs / 4; ++u) {
                    const int4 v = sub[u];
                    sub[u] = make_int4(run, run + v.x, run + v.x + v.y, run + v.x + v.y + v.z);
                    run += v.x + v.y + v.z + v.w;
                }
                seg_cnt[tid] = run;
            }
            __syncthreads();
            scan_counts();
            __syncthreads();
#pragma unroll
            for (int u = 0; u < kHeld; ++u) {
                if (tid + u * NT >= cnt) continue;
                const int pos = seg_start[(int)(held[u] >> 57)] + s_sub[place[u] >> 16] + (place[u] & 0xffff);
                if (OCTO_IN_RANGE(pos >= 0 && pos < cnt, status)) {
                    keys[pos] = held[u];
                    slots[pos] = (unsigned short)(tid + u * NT);
                }
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

        // ---- many small classes on one CTA: one warp each, handed out by a counter ----
        if (s_by_warps) {
            auto by_warps = [&](unsigned long long* k, float4* b) {
                const int nclasses = s_nlarge;
                for (;;) {
                    int q = 0;
                    if (lane == 0) q = atomicAdd(&s_next, 1);
                    q = __shfl_sync(0xffffffffu, q, 0);
                    if (q >= nclasses) break;
                    const int cls = s_large[q];
                    const int nk = warp_class(k, b, seg_start[cls], seg_cnt[cls], max_det, hbase, as, es, P.iou_test, lane, status);
                    finish_class(cls, seg_start[cls], nk, lane, 32);
                }
            };
            // (in the half-sized form the code for pointers of shared memory alone is 5 to 10 % faster than the code for
            // both, in the full-sized form 10 % slower)
            if (NT == kNmsThreadsFull) by_warps(keys, boxes);
            else if (on_chip) by_warps(reinterpret_cast<unsigned long long*>(smem_raw + (size_t)SMEM_CAP * sizeof(float4)),
                                      reinterpret_cast<float4*>(smem_raw));
            else by_warps(gk, P.gboxes + (size_t)img * P.key_stride);
        } else {
            // ---- classes of at most kTeamMin, a batch of them at a time: one candidate per thread.  (Before the large
            // classes, whose boxes take the memory of the slots.) ----
            const int nbatch = s_nbatch;
            const bool bucketed = on_chip || s_most <= kCountedMax;
            for (int q = (int)crank; q < nbatch; q += (int)team_ctas) {
                const int lo = s_lo[q], m = s_hi[q] - lo;
                if (m <= 0) continue;
                const BatchMem<NT> mem(smem_raw);
                unsigned long long key = kKeySentinel;
                float4 box = make_float4(0.f, 0.f, 0.f, 0.f);
                int slot = 0;
                if (tid < m && OCTO_IN_RANGE(m <= NT && lo >= 0 && lo + m <= cnt, status)) {
                    key = keys[lo + tid];
                    if (on_chip) {
                        slot = slots[lo + tid];
                        box = __ldcg(gb + slot);
                    } else {
                        box = gather_box(hbase + (size_t)(key & ((1ull << kKeyAnchorBits) - 1)) * as, es);
                    }
                    mem.skey[tid] = key;
                    mem.rank[tid] = 0;
                }
                if (tid == 0) mem.skey[m] = kKeySentinel;  // (m = NT: the first word of the boxes, not read)
                __syncthreads();
                nms_batch<NT>(mem, NT / 32, key, box, m, bucketed, P.iou_test, s_fate, status,
                              [&](int cls) { return seg_start[cls] - lo; },
                              [&](unsigned long long k, int& from, int& to) {
                                  const int cls = (int)(k >> 57), start = seg_start[cls] - lo, all = seg_cnt[cls];
                                  if (on_chip) {
                                      const int b = score_bucket(k, kSubs, kSubScale), at = cls * kSubs + b;
                                      from = start + s_sub[at];
                                      to = b + 1 < kSubs ? start + s_sub[at + 1] : start + all;
                                  } else {
                                      from = start;
                                      to = start + all;
                                  }
                              });
                const int words = (m + 31) >> 5;
                int all = 0;
                const int before = kept_before(s_fate, words, lane, warp, all);
                // survivors and their slots: thread c still knows candidate c's slot, and its rank says where it went
                unsigned short* const sslot = reinterpret_cast<unsigned short*>(mem.sup);
                if (tid < m) sslot[mem.rank[tid]] = (unsigned short)slot;
                __syncthreads();
                const unsigned kept = warp < words ? s_fate[warp].x : 0u;
                if ((kept >> lane) & 1u) {
                    const int at = lo + before + __popc(kept & ((1u << lane) - 1u)), cand = batch_cand(tid);
                    keys0[at] = global_key(mem.skey[cand]);
                    // (a large class's boxes may take the first CTA's slots)
                    if (on_chip && s_nlarge == 0) slots0[at] = sslot[cand];
                }
                if (tid == 0) {
                    kept0[q] = all;
                    atomicAdd(total0, all);
                }
                __syncthreads();
            }

            // ---- large classes, by all warps of a CTA ----
            __shared__ unsigned t_sup[kTeamBlock * kTeamWords];
            const int nlarge = s_nlarge;
            for (int q = (int)crank; q < nlarge; q += (int)team_ctas) {
                const int cls = s_large[q], m = seg_cnt[cls];
                const int s = seg_start[cls], e = s + m;
                bitonic_range<true>(keys + s, m, tid, NT);
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
                    if (warp < twords) resolve_words<kTeamBlock>(t_sup, tid, n, 0, s_fate, tid, twords);
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

        if (shared_work) {
            cg::this_cluster().sync();  // every class has arrived in the first CTA's arrays
            if (crank != 0) return;
        } else {
            __syncthreads();
        }

        // ---- global score order: the survivor lists (batches, then large classes) are packed into the memory
        // of the (dead) boxes and put in order there ----
        const int total = s_total;
        nout = min(total, max_det);
        const bool in_smem = total <= NT;
        unsigned long long* const packed = in_smem ? reinterpret_cast<unsigned long long*>(smem_raw)
                                                   : reinterpret_cast<unsigned long long*>(boxes);
        ordered = packed + NT + 2;
        unsigned long long* const tmp = ordered + NT;
        unsigned short* const ppos = reinterpret_cast<unsigned short*>(tmp + NT + 2);
        const bool have_slots = in_smem && on_chip && s_nlarge == 0;
        const int lists = s_nbatch + s_nlarge;
        for (int q = warp; q < lists; q += NT / 32) {
            const int cls = q < s_nbatch ? 0 : s_large[q - s_nbatch];
            const int m = q < s_nbatch ? s_kept[q] : nkept[cls], from = q < s_nbatch ? s_lo[q] : seg_start[cls];
            int to = 0;
            if (lane == 0) to = atomicAdd(&s_pack, m);
            to = __shfl_sync(0xffffffffu, to, 0);
            for (int i = lane; i < m; i += 32)
                if (OCTO_IN_RANGE(to + i >= 0 && to + i < total && total <= cnt, status)) {
                    packed[to + i] = keys[from + i];
                    if (have_slots) ppos[to + i] = slots[from + i];
                }
        }
        __syncthreads();
        if (in_smem) {
            opos = ppos + NT;
            order_survivors<NT>(packed, ppos, total, tmp, reinterpret_cast<int*>(ppos + 2 * NT), tid,
                                [&](int r, unsigned long long g, int at) {
                                    if (!OCTO_IN_RANGE(r >= 0 && r < total, status)) return;
                                    ordered[r] = g;
                                    opos[r] = (unsigned short)at;
                                });
            if (have_slots) boxes_at = gb;
        } else {
            ordered = packed;
            bitonic_range<true>(ordered, total, tid, NT);
        }
    }
    if (P.class_agnostic) {
        // NMS ran with every candidate in class 0: a warp recovers the real class (first maximum)
        for (int r = warp; r < nout; r += nt / 32) {
            const unsigned long long g = ordered[r];
            const int anchor = (int)((g >> 7) & ((1ull << kKeyAnchorBits) - 1));
            const float* __restrict__ cv = hbase + (size_t)anchor * as + (size_t)nbox * es;
            float best = -INFINITY;
            int cls = 0x7fffffff;
            float v[OCTO_MAX_CLASSES / 32];
#pragma unroll
            for (int u = 0; u < OCTO_MAX_CLASSES / 32; ++u)
                v[u] = lane + 32 * u < P.C ? __ldg(cv + (size_t)(lane + 32 * u) * es) : -INFINITY;
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
            if (lane == 0) ordered[r] = (g & ~127ull) | (unsigned long long)cls;  // for the record and the branch lists
        }
        __syncthreads();
    }
    // Records: eight lanes each, one word per lane (a thread that writes a whole record touches eight sectors
    // of its own).
    for (int i = written ? 8 * nout : tid; i < 8 * nout; i += nt) {
        const int r = i >> 3, k = i & 7;
        const unsigned long long g = ordered[r];
        float corner = 0.0f;
        if (k < 4) {
            if (boxes_at) {
                corner = reinterpret_cast<const float*>(boxes_at + opos[r])[k];
            } else {
                const float* __restrict__ row = hbase + (size_t)((g >> 7) & ((1ull << kKeyAnchorBits) - 1)) * as;
                const float centre = __ldg(row + (size_t)(k & 1) * es);
                const float half = __fmul_rn(0.5f, __ldg(row + (size_t)(2 + (k & 1)) * es));
                corner = k < 2 ? __fsub_rn(centre, half) : __fadd_rn(centre, half);  // as box_corners
            }
        }
        if (OCTO_IN_RANGE(r < max_det, status)) reinterpret_cast<unsigned*>(dets + r)[k] = map.word(k, corner, g);
    }
    if (tid == nt - 1) {
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
