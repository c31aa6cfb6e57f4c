// Decode + confidence filter + compaction of a YOLOv5-layout head [n, A, 5 + C] fp32.
//
// HBM-bound scan.  For logit heads sigma <= 1 makes sigma(obj) > conf a necessary condition
// for score = fl(sigma(obj) * sigma(cls)) > conf, so the scan reads only the obj value of
// each 340-byte row (one DRAM sector) and fetches the whole row, 32 bytes at a time by a group
// of eight lanes (four passing rows per warp in flight together), for the few anchors that pass.
// Probability heads are read densely (decode_dense_kernel, where a 16-byte boundary allows it).  A passing row is
// reduced by eight lanes (finite check, first-maximum class), scored in the fixed binary32
// sequence and appended to the image's key list with one atomic; the key carries class,
// inverted score bits and anchor, so later steps need nothing else from this kernel and the
// nondeterministic append order is erased by the sort.
//
// Variants.  Multi-label: a passing row yields one key per class whose own score exceeds the
// threshold.  Planes layout [n, 4 + C, A] (anchor-free heads without objectness): consecutive
// anchors are contiguous in every plane, so the scan is a dense, coalesced read of the C class
// planes (the whole head must be read: the maximum over classes needs every value); the four
// box planes are read only for anchors whose score passes.
#include "octo_common.cuh"
#include <cmath>

#include "octo_kernels.h"

namespace octo {

constexpr int kDecThreads = 256;

// Read-only load that asks L2 to fetch 64 bytes around the address instead of the default
// 128: the obj scan touches 4 bytes per 340-byte row, so the smaller fill granularity cuts
// the DRAM traffic of the scan (measured: 27 % less time for the bare scan).  The values are used
// once, so they are kept out of L1 as well (another 3.6 %).
__device__ __forceinline__ float ld_obj(const float* p) {
    float v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::64B.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}

// Candidate key: class | inverted score bits | anchor (ascending key = descending score, then
// ascending anchor inside a class).
__device__ __forceinline__ unsigned long long make_key(int cls, float score, int anchor) {
    return ((unsigned long long)(unsigned)cls << 57) | ((unsigned long long)(~__float_as_uint(score)) << kKeyAnchorBits) |
           (unsigned long long)(unsigned)anchor;
}

// kDecPerThread anchors per thread: 4 for large batches, 1 when the grid would otherwise be
// too small to cover the SMs.
// Six (five) CTAs per SM: the scan lives on loads in flight, and one register more than 40 costs the large
// grids a CTA per SM ([32, 25200, 85] with 5000 candidates an image 74.7 against 66.5 us).
template <int kDecPerThread>
__global__ void __launch_bounds__(kDecThreads, kDecPerThread == 1 ? 5 : 6)
decode_kernel(const float* __restrict__ head, int A, int C, int mode, float conf, int key_stride,
              unsigned long long* __restrict__ keys, float4* __restrict__ boxes, int* __restrict__ cand_count,
              unsigned int* __restrict__ status) {
    pdl_wait();
    // mode bit 0: obj / class values are logits; bit 1: class-agnostic NMS (key class field 0);
    // bit 2: multi-label candidates
    const int logits = mode & 1;
    const bool agnostic = (mode & 2) != 0;
    const bool multi = (mode & 4) != 0;
    const int img = blockIdx.y;
    const int row_len = 5 + C;
    const float* __restrict__ hbase = head + (size_t)img * (size_t)A * (size_t)row_len;
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int grp = lane >> 3, gl = lane & 7, gbase = lane & 24;  // group of eight lanes, lane in it, its first lane
    const unsigned gmask = 0xffu << gbase;
    // each warp owns kDecPerThread consecutive groups of 32 anchors
    const int a_warp = blockIdx.x * (kDecThreads * kDecPerThread) + warp * (32 * kDecPerThread);

    float obj[kDecPerThread];
#pragma unroll
    for (int u = 0; u < kDecPerThread; ++u) {
        const int a = a_warp + u * 32 + lane;
        obj[u] = (logits && a < A) ? ld_obj(hbase + (size_t)a * row_len + 4) : 0.0f;
    }
    bool nonfinite_seen = false;
#pragma unroll
    for (int u = 0; u < kDecPerThread; ++u) {
        const int a = a_warp + u * 32 + lane;
        bool pass = a < A;
        if (logits && pass) {
            const bool fin = finite_f(obj[u]);
            nonfinite_seen |= !fin;
            pass = fin && sigmoid_fixed(obj[u]) > conf;
        }
        // Passing rows are reduced four at a time, one per group of eight lanes (a row is read in
        // 32-byte pieces, lane g of a group holds elements g, g + 8, ...): the four row fetches are in
        // flight together and a row costs a quarter of the warp's instructions.
        unsigned todo = __ballot_sync(0xffffffffu, pass);
        while (todo) {
            unsigned mine = todo;  // this group's row: the grp-th lowest set bit
            for (int i = 0; i < grp; ++i) mine &= mine - 1;
            const bool have = mine != 0u;
            const int src = have ? __ffs(mine) - 1 : 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) todo &= todo - 1;  // the four lowest rows are taken
            const int ra = a_warp + u * 32 + src;
            const float* __restrict__ row = hbase + (size_t)ra * row_len;
            bool fin = true;
            float best = -INFINITY;
            int best_k = 0x7fffffff;
            float e0 = 0.0f;
            if (have) {
                // the row is requested in batches of kPieces 32-byte pieces (48 values per group), so
                // a row of 85 values takes two round trips and the kernel stays at 32-40 registers
                // (the obj scan of large batches lives on occupancy); the small-grid form asks for
                // the whole row at once (any row of up to 5 + 128 values): one round trip less
                constexpr int kPieces = kDecPerThread == 1 ? 17 : 6;
                for (int e00 = 0; e00 < row_len; e00 += 8 * kPieces) {
                    float v[kPieces];
#pragma unroll
                    for (int j = 0; j < kPieces; ++j) {
                        const int e = e00 + gl + 8 * j;
                        v[j] = e < row_len ? __ldg(row + e) : 0.0f;
                    }
                    if (e00 == 0) e0 = v[0];
#pragma unroll
                    for (int j = 0; j < kPieces; ++j) {
                        const int e = e00 + gl + 8 * j;
                        if (e < row_len) {
                            fin &= finite_f(v[j]);
                            if (e >= 5 && v[j] > best) { best = v[j]; best_k = e - 5; }
                        }
                    }
                }
            }
            const unsigned bad = __ballot_sync(0xffffffffu, !fin) & gmask;
            const float bw = __shfl_sync(0xffffffffu, e0, gbase + 2);
            const float bh = __shfl_sync(0xffffffffu, e0, gbase + 3);
            const float ob = __shfl_sync(0xffffffffu, e0, gbase + 4);
            if (bad) nonfinite_seen = true;
            const bool ok = have && !bad && bw > 0.0f && bh > 0.0f;
            if (!multi) {
#pragma unroll
                for (int off = 4; off > 0; off >>= 1) {  // first maximum over the group's eight lanes
                    const float ov = __shfl_xor_sync(0xffffffffu, best, off);
                    const int ok2 = __shfl_xor_sync(0xffffffffu, best_k, off);
                    if (ov > best || (ov == best && ok2 < best_k)) { best = ov; best_k = ok2; }
                }
                const float cy = __shfl_sync(0xffffffffu, e0, gbase + 1);  // (the group's first lane holds cx)
                if (ok && gl == 0) {
                    const float score = logits ? __fmul_rn(sigmoid_fixed(ob), sigmoid_fixed(best))
                                               : __fmul_rn(ob, best);
                    if (score > conf) {
                        const int slot = atomicAdd(cand_count + img, 1);
                        if (slot < key_stride) {
                            keys[(size_t)img * key_stride + slot] = make_key(agnostic ? 0 : best_k, score, ra);
                            boxes[(size_t)img * key_stride + slot] = box_corners(e0, cy, bw, bh);
                        } else {
                            atomicOr(status, 0x10u);
                        }
                    }
                }
            } else {
                // one candidate per class whose own score passes; the keys of a row go out in
                // groups of up to eight with one counter update per group
                const float so = logits ? sigmoid_fixed(ob) : ob;
                const float4 box = box_corners(__shfl_sync(0xffffffffu, e0, gbase), __shfl_sync(0xffffffffu, e0, gbase + 1),
                                               bw, bh);
                for (int e0i = 0; e0i < row_len; e0i += 8) {  // the same trip count in every group
                    const int e = e0i + gl;
                    float score = 0.0f;
                    bool hit = false;
                    if (ok && e >= 5 && e < row_len) {
                        const float v = __ldg(row + e);  // second pass over the row: an L1 hit
                        score = __fmul_rn(so, logits ? sigmoid_fixed(v) : v);
                        hit = score > conf;
                    }
                    const unsigned hits = __ballot_sync(0xffffffffu, hit) & gmask;
                    int base = 0;
                    if (hits != 0u && gl == 0) base = atomicAdd(cand_count + img, __popc(hits));
                    base = __shfl_sync(0xffffffffu, base, gbase);
                    if (hit) {
                        const int slot = base + __popc(hits & ((1u << lane) - 1u));
                        if (slot < key_stride) {
                            keys[(size_t)img * key_stride + slot] = make_key(e - 5, score, ra);
                            boxes[(size_t)img * key_stride + slot] = box;
                        } else {
                            atomicOr(status, 0x10u);
                        }
                    }
                }
            }
        }
    }
    if (__any_sync(0xffffffffu, nonfinite_seen) && lane == 0) atomicOr(status, 0x1u);
}

// Planes layout [n, 4 + C, A].  A thread owns VEC consecutive anchors (VEC = 4 with 16-byte
// loads when A is a multiple of 4, else 1); the lanes of a warp and AW warps side by side read
// consecutive addresses of one plane, so a CTA fetches long contiguous runs (DRAM pages are used
// better the longer the run).  CW = 8 / AW groups of warps split the C class planes between them
// (group g takes classes g, g + CW, ...) and leave their running first maxima in shared memory, where
// one thread per anchor merges them.  Every thread keeps kBatch planes in flight.
// Bound by HBM for large batches of the vector form, by issue for large batches of the scalar form (a value
// costs a load, the multiply-add that turns NaN once a value is not finite, a comparison and two selects; with
// clamped plane numbers and a test of every exponent heads of odd A were slower than before the loads were
// batched), and by the number of planes a warp walks one after another for small ones.  So the split follows
// the size of the grid: side by side (four warps, or eight in the scalar form) where that gives every SM two
// CTAs (one), else one warp's width and eight groups.  us per decode + NMS pass without batches of loads / with
// batches of clamped plane numbers / now, [n, 84, A]: A = 8401, n = 8 12.3 / 13.6 / 10.1, n = 32 24.2 / 28.2 / 17.4, n = 256 116 /
// 156 / 109; A = 8400, n = 8 27.1 / 11.2 / 10.4, n = 32 31.1 / 21.9 / 16.4, n = 256 130 / 112 / 109; multi-label, n = 32 76.5 /
// 27.9 / 21.4; seven classes, A = 8401, n = 13 9.9 / 13.2 / 8.8.
// For multi-label heads in logit form a value is only run through the fixed logistic sequence when it
// lies above `pre`, a bound placed safely below the threshold's logit, so that the common case costs
// one comparison per value.
constexpr int kPlaneRepeat = 5;  // class planes a lane reads at a time the second time (multi-label)

template <int VEC, int AW, bool MULTI>
__global__ void __launch_bounds__(kDecThreads, 5)
decode_planes_kernel(const float* __restrict__ head, int A, int C, int mode, float conf, float pre, int key_stride,
                     unsigned long long* __restrict__ keys, float4* __restrict__ boxes, int* __restrict__ cand_count,
                     unsigned int* __restrict__ status) {
    pdl_wait();
    constexpr int CW = kDecThreads / 32 / AW;
    constexpr int kCtaAnchors = AW * 32 * VEC;
    constexpr int kBatch = VEC == 4 ? 5 : 8;
    __shared__ float s_best[CW][kCtaAnchors];
    __shared__ unsigned char s_k[CW][kCtaAnchors];
    __shared__ unsigned char s_flags[CW][AW * 32];  // bits 0..3: non-finite, 4..7: above `pre`
    __shared__ unsigned short s_list[MULTI ? kCtaAnchors : 1];  // multi-label: anchors with a value above `pre`
    __shared__ float4 s_box[MULTI ? kCtaAnchors : 1];           // ... and their boxes
    __shared__ int s_nlist;
    const int logits = mode & 1;
    const bool agnostic = (mode & 2) != 0;
    const int img = blockIdx.y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int aw = warp % AW, cw = warp / AW;
    const float* __restrict__ hbase = head + (size_t)img * (size_t)(4 + C) * (size_t)A;
    const int col = aw * 32 + lane;  // this thread's group of VEC anchors inside the CTA
    const int a0 = blockIdx.x * kCtaAnchors + col * VEC;

    float best[VEC], zero[VEC];  // zero: sum of 0 * value, a NaN once a value was not finite
    int best_k[VEC];
    unsigned flags = 0u;
#pragma unroll
    for (int u = 0; u < VEC; ++u) { best[u] = -INFINITY; zero[u] = 0.0f; best_k[u] = 255; }
    if (a0 < A) {
        auto load = [&](const float* __restrict__ p, float (&v)[VEC]) {
            if (VEC == 4) {
                const float4 q = __ldg(reinterpret_cast<const float4*>(p));
                v[0] = q.x; v[1 % VEC] = q.y; v[2 % VEC] = q.z; v[3 % VEC] = q.w;
            } else {
                v[0] = __ldg(p);
            }
        };
        auto take = [&](const float (&v)[VEC], int k) {
#pragma unroll
            for (int u = 0; u < VEC; ++u) {
                zero[u] = __fmaf_rn(v[u], 0.0f, zero[u]);
                if (v[u] > best[u]) { best[u] = v[u]; best_k[u] = k; }
                if (MULTI && v[u] > pre) flags |= 16u << u;
            }
        };
        const size_t step = (size_t)CW * (size_t)A;
        const float* __restrict__ p = hbase + (size_t)(4 + cw) * (size_t)A + a0;
        int k = cw;
        for (; k + (kBatch - 1) * CW < C; k += kBatch * CW) {
            float v[kBatch][VEC];
#pragma unroll
            for (int j = 0; j < kBatch; ++j) { load(p, v[j]); p += step; }
#pragma unroll
            for (int j = 0; j < kBatch; ++j) take(v[j], k + j * CW);
        }
        float v[kBatch - 1][VEC];  // what is left: fewer than a batch
#pragma unroll
        for (int j = 0; j < kBatch - 1; ++j) {
            if (k + j * CW < C) load(p, v[j]);
            p += step;
        }
#pragma unroll
        for (int j = 0; j < kBatch - 1; ++j)
            if (k + j * CW < C) take(v[j], k + j * CW);
#pragma unroll
        for (int u = 0; u < VEC; ++u)
            if (!(zero[u] == 0.0f)) flags |= 1u << u;
    }
#pragma unroll
    for (int u = 0; u < VEC; ++u) {
        s_best[cw][col * VEC + u] = best[u];
        s_k[cw][col * VEC + u] = (unsigned char)best_k[u];
    }
    s_flags[cw][col] = (unsigned char)flags;
    if (threadIdx.x == 0) s_nlist = 0;
    __syncthreads();

    auto emit = [&](int cls, float score, int anchor, const float4 box) {
        const int slot = atomicAdd(cand_count + img, 1);
        if (slot < key_stride) {
            keys[(size_t)img * key_stride + slot] = make_key(cls, score, anchor);
            boxes[(size_t)img * key_stride + slot] = box;
        } else {
            atomicOr(status, 0x10u);
        }
    };
    // one thread per anchor of the CTA
    for (int t = threadIdx.x; t < kCtaAnchors; t += kDecThreads) {
        const int u = t % VEC;
        const int anchor = blockIdx.x * kCtaAnchors + t;
        if (anchor >= A) break;
        float bv = -INFINITY;
        int bk = 255;
        unsigned fl = 0u;
#pragma unroll
        for (int w = 0; w < CW; ++w) {
            const float v = s_best[w][t];
            const int k = s_k[w][t];
            if (v > bv || (v == bv && k < bk)) { bv = v; bk = k; }  // first maximum over all classes
            fl |= s_flags[w][t / VEC];
        }
        const bool bad = (fl >> u) & 1u;
        if (bad) {
            atomicOr(status, 0x1u);
            continue;
        }
        float score = 0.0f;
        if (!MULTI) {
            score = logits ? sigmoid_fixed(bv) : bv;
            if (!(score > conf)) continue;
        } else if (!((fl >> (4 + u)) & 1u)) {
            continue;
        }
        // finite box with w, h > 0
        const float* __restrict__ bx = hbase + anchor;
        const float cx = __ldg(bx), cy = __ldg(bx + A), bw = __ldg(bx + 2 * (size_t)A), bh = __ldg(bx + 3 * (size_t)A);
        if (!(finite_f(cx) && finite_f(cy) && finite_f(bw) && finite_f(bh))) {
            atomicOr(status, 0x1u);
            continue;
        }
        if (!(bw > 0.0f && bh > 0.0f)) continue;
        const float4 box = box_corners(cx, cy, bw, bh);
        if (!MULTI) {
            emit(agnostic ? 0 : bk, score, anchor, box);
        } else {
            const int q = atomicAdd(&s_nlist, 1);
            s_list[q] = (unsigned short)t;
            s_box[q] = box;
        }
    }
    if (!MULTI) return;
    // Multi-label: every (listed anchor, class) pair is tested by its own lane, a warp taking a class
    // plane at a time and kPlaneRepeat planes in flight.  Bound by the latency of these second reads
    // (L2 hits, 4 bytes each): with one thread walking the C classes of its anchor in turn the launch
    // took 115 us on [32, 84, 8400] with 300 candidates an image, 32-34 us this way (31 without labels).
    __syncthreads();
    const int nlist = s_nlist;
    for (int k0 = warp; k0 < C; k0 += (kDecThreads / 32) * kPlaneRepeat) {
        for (int q = lane; q < nlist; q += 32) {
            const int anchor = blockIdx.x * kCtaAnchors + (int)s_list[q];
            const float* __restrict__ cv = hbase + (size_t)4 * A + anchor;
            float v[kPlaneRepeat];
#pragma unroll
            for (int j = 0; j < kPlaneRepeat; ++j) {
                const int k = k0 + j * (kDecThreads / 32);
                v[j] = k < C ? __ldg(cv + (size_t)k * A) : -INFINITY;
            }
#pragma unroll
            for (int j = 0; j < kPlaneRepeat; ++j) {
                if (!(v[j] > pre)) continue;
                const float score = logits ? sigmoid_fixed(v[j]) : v[j];
                if (score > conf) emit(k0 + j * (kDecThreads / 32), score, anchor, s_box[q]);
            }
        }
    }
}

// Rows layout, probabilities: nothing bounds a row's score before its class values are known, so the
// head is read whole and the scan is bound by HBM.  A CTA takes kDenseRows consecutive rows, which are
// one contiguous piece of memory: one bulk copy stages them (five CTAs of 85-value rows keep 218 KB per
// SM in flight), then a thread reduces a row out of shared memory.  A row of an odd number of values is
// read without bank conflicts as it stands (lane stride = row length); for the others the lanes start
// at rotated positions.  The scan of a row was the bound while it kept an index and tested every value's
// exponent (12 instructions a value); now a value costs a load, a multiply-add that turns NaN once a value is
// not finite, and a maximum, and the few rows that pass look for the class that holds the maximum.
// us per launch on [n, 25200, 5 + C], row groups of decode_kernel / that scan / this one: C = 80, n = 1 18.5 / 12.3 /
// 10.3, n = 4 22.6 / 18.5 / 14.3, n = 32 96 / 70.7 / 57.4; C = 27, n = 64 111 / 52.2 / 46; C = 128, n = 256 776 / 915 /
// 479 (7.2 TB/s).  Multi-label heads [32, 6300, 128]: 77.8 / 127 / 47.1 (every row had walked its classes a
// second time, rows of one bank one after the other).  64 rows per CTA measure the same.
constexpr int kDenseRows = 128;

__global__ void __launch_bounds__(kDenseRows)
decode_dense_kernel(const float* __restrict__ head, int A, int C, int mode, float conf, int key_stride,
                    unsigned long long* __restrict__ keys, float4* __restrict__ boxes, int* __restrict__ cand_count,
                    unsigned int* __restrict__ status) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) uint64_t bar;
    pdl_wait();
    const bool agnostic = (mode & 2) != 0;
    const bool multi = (mode & 4) != 0;
    const int img = blockIdx.y, t = threadIdx.x;
    const int row_len = 5 + C;
    const int a0 = blockIdx.x * kDenseRows;
    const int rows = min(kDenseRows, A - a0);
    const float* __restrict__ src = head + ((size_t)img * (size_t)A + (size_t)a0) * (size_t)row_len;
    float* const s = reinterpret_cast<float*>(smem);
    const int values = rows * row_len, bulk = values & ~3;  // the copy moves multiples of 16 bytes
    if (t == 0) {
        mbar_init(&bar, 1);
        mbar_fence_init();
        fence_proxy_async();
        mbar_expect_tx(&bar, (uint32_t)bulk * 4u);
        if (bulk) bulk_g2s(s, src, (uint32_t)bulk * 4u, &bar);
    }
    if (t < values - bulk) s[bulk + t] = __ldg(src + bulk + t);
    __syncthreads();
    if (!mbar_wait_or_report(&bar, 0, status)) return;
    if (t >= rows) return;
    const float* const row = s + t * row_len;
    const float* const cls = row + 5;
    float zero = 0.0f;  // sum of 0 * value: a NaN once a value was not finite
    float best = -INFINITY;
    if (row_len & 1) {
#pragma unroll
        for (int e = 0; e < 5; ++e) zero = __fmaf_rn(row[e], 0.0f, zero);
#pragma unroll 8
        for (int k = 0; k < C; ++k) {
            const float v = cls[k];
            zero = __fmaf_rn(v, 0.0f, zero);
            best = fmaxf(best, v);
        }
    } else {
        // lanes whose rows start in the same bank (32 / gcd(row_len, 32) lanes apart) start at different values
        const int banks = row_len & -row_len;  // gcd with a power of two
        int e = banks >= 32 ? (t & 31) : (t & 31) / (32 / banks);
#pragma unroll 8
        for (int i = 0; i < row_len; ++i) {
            const float v = row[e];
            zero = __fmaf_rn(v, 0.0f, zero);
            if (e >= 5) best = fmaxf(best, v);
            e = e + 1 == row_len ? 0 : e + 1;
        }
    }
    if (!(zero == 0.0f)) {
        atomicOr(status, 0x1u);
        return;
    }
    // (no class of a row scores above its best, unless both factors are negative)
    const float ob = row[4], top = __fmul_rn(ob, best);
    if (!(top > conf) && !(multi && ob < 0.0f)) return;
    if (!(row[2] > 0.0f) || !(row[3] > 0.0f)) return;
    auto emit = [&](int cls, float score) {
        const int slot = atomicAdd(cand_count + img, 1);
        if (slot < key_stride) {
            keys[(size_t)img * key_stride + slot] = make_key(cls, score, a0 + t);
            boxes[(size_t)img * key_stride + slot] = box_corners(row[0], row[1], row[2], row[3]);
        } else {
            atomicOr(status, 0x10u);
        }
    };
    if (!multi) {
        int k = 0;  // the first maximum
        while (!agnostic && k < C - 1 && cls[k] != best) ++k;
        emit(k, top);
    } else {
        for (int k = 0; k < C; ++k) {
            const float score = __fmul_rn(ob, cls[k]);
            if (score > conf) emit(k, score);
        }
    }
}

cudaError_t prepare_decode() {
    return cudaFuncSetAttribute(decode_dense_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                kDenseRows * (5 + OCTO_MAX_CLASSES) * (int)sizeof(float));
}

template <int VEC, int AW>
static cudaError_t launch_planes_split(const DecodeArgs& a, int mode, float pre, cudaStream_t stream) {
    dim3 grid((a.A + 32 * VEC * AW - 1) / (32 * VEC * AW), a.n);
    auto kernel = a.multi_label ? decode_planes_kernel<VEC, AW, true> : decode_planes_kernel<VEC, AW, false>;
    return launch_kernel(kernel, grid, dim3(kDecThreads), 0, stream, a.d_head, a.A, a.C, mode, a.conf, pre,
                         a.key_stride, a.d_keys, a.d_boxes, a.d_cand_count, a.d_status);
}

// Warps side by side along the anchors, by the number of CTAs that gives (see decode_planes_kernel).
template <int VEC>
static cudaError_t launch_planes(const DecodeArgs& a, int mode, float pre, cudaStream_t stream) {
    constexpr int kWide = VEC == 4 ? 4 : 8;
    const long long ctas = (long long)a.n * ((a.A + 32 * VEC * kWide - 1) / (32 * VEC * kWide));
    return ctas >= (VEC == 4 ? 2 : 1) * (long long)a.sm_count ? launch_planes_split<VEC, kWide>(a, mode, pre, stream)
                                                              : launch_planes_split<VEC, 1>(a, mode, pre, stream);
}

cudaError_t launch_decode(const DecodeArgs& a, cudaStream_t stream) {
    // d_cand_count is zero on entry: zeroed at stage creation and re-zeroed by the NMS kernel.
    const int mode = (a.logits ? 1 : 0) | (a.class_agnostic ? 2 : 0) | (a.multi_label ? 4 : 0);
    if (a.layout == OCTO_HEAD_PLANES) {
        // Multi-label prefilter in the head's own units: for probabilities the threshold itself;
        // for logits the threshold's logit lowered by a margin that dwarfs the few-ulp error of
        // the fixed logistic sequence (no prefilter where the logistic curve is too flat for that).
        float pre = a.conf;
        if (a.logits) {
            pre = -INFINITY;
            if (a.conf > 0.0f && a.conf <= 0.99f) {
                const double t = log((double)a.conf / (1.0 - (double)a.conf));
                pre = (float)(t - 1e-3 * (1.0 + fabs(t)));
            }
        }
        const bool vec = (a.A & 3) == 0 && (reinterpret_cast<uintptr_t>(a.d_head) & 15) == 0;
        return vec ? launch_planes<4>(a, mode, pre, stream) : launch_planes<1>(a, mode, pre, stream);
    }
    if (!a.logits && ((long long)a.A * (5 + a.C)) % 4 == 0 && (reinterpret_cast<uintptr_t>(a.d_head) & 15) == 0) {
        // (every image starts on a 16-byte boundary, as the bulk copies need; any other head is read
        // by the row groups of decode_kernel)
        dim3 grid((a.A + kDenseRows - 1) / kDenseRows, a.n);
        return launch_kernel(decode_dense_kernel, grid, dim3(kDenseRows), sizeof(float) * kDenseRows * (5 + (size_t)a.C),
                             stream, a.d_head, a.A, a.C, mode, a.conf, a.key_stride, a.d_keys, a.d_boxes, a.d_cand_count,
                             a.d_status);
    }
    const int per_cta4 = kDecThreads * 4;
    if ((long long)a.n * ((a.A + per_cta4 - 1) / per_cta4) >= 2ll * a.sm_count) {
        dim3 grid((a.A + per_cta4 - 1) / per_cta4, a.n);
        return launch_kernel(decode_kernel<4>, grid, dim3(kDecThreads), 0, stream, a.d_head, a.A, a.C, mode,
                             a.conf, a.key_stride, a.d_keys, a.d_boxes, a.d_cand_count, a.d_status);
    }
    dim3 grid((a.A + kDecThreads - 1) / kDecThreads, a.n);
    return launch_kernel(decode_kernel<1>, grid, dim3(kDecThreads), 0, stream, a.d_head, a.A, a.C, mode, a.conf,
                         a.key_stride, a.d_keys, a.d_boxes, a.d_cand_count, a.d_status);
}

}  // namespace octo
