// Letterbox kernel: n BGR uint8 frames -> fp16 NCHW [n, 3, S, S] detector batch.
//
// HBM-bound gather.  One CTA produces up to kLbRows output rows of one frame.  The source rows
// those output rows tap (one row where the vertical weight is zero, e.g. the 3:1 reduction
// of 1080p, else two) are fetched whole into shared memory by the bulk-copy (TMA) engine
// with 16-byte coalesced transactions and an mbarrier; rows that carry no weight are never
// read.  While the copies are in flight the CTA builds a table of horizontal taps (byte
// offset + exact integer weights per canvas column).  Threads then take pixel pairs (lane l
// of a warp owns pixels 2l, 2l+1 of a 64-pixel run): the horizontal lerp is an exact integer
// two-way dot product per channel, the vertical lerp and all scaling are two fp32
// operations, and each warp writes 128 contiguous bytes per colour plane.
#include "octo_common.cuh"
#include "octo_kernels.h"

namespace octo {

constexpr int kLbThreads = 256;
constexpr int kLbRows = 8;  // most output rows a CTA produces; fewer for very wide frames
static_assert(kLbRows <= kLbThreads / 32, "a warp for every row of a CTA");

// A warp stages its own output row, behind a barrier of its own, and waits for nothing else but the table of taps;
// where a CTA has fewer rows than warps (small batches), several warps share a row.  What needs no memory (barriers,
// which rows are tapped) comes before the wait for the previous kernel.  Large batches are bound by HBM, small
// ones by this chain.  One thread that walked the rows twice and issued every copy, and one barrier for all of them /
// a barrier and copies per warp / rows shared by warps too (us a launch over 1080p frames from memory): one 4.3 / 4.1 / 3.5, two 5.3 /
// 4.8 / 4.2, eight 11.5 / 9.4 / 9.2, 64 50.7 / - / 49.1.
template <int CAP>
__global__ void __launch_bounds__(kLbThreads)
letterbox_kernel(const __grid_constant__ FrameTable<CAP> tab, __half* __restrict__ out, int S, int band_rows,
                 int slot_bytes, int row_slots, int share, uint32_t fill_h2, int swap_rb, unsigned int* __restrict__ status) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) uint64_t bar[kLbRows];

    const FrameDesc& fd = tab.f[blockIdx.y];
    const int dy0 = blockIdx.x * band_rows;
    const int w = fd.w, h = fd.h, nw = fd.nw, nh = fd.nh, pad_l = fd.pad_l, pad_t = fd.pad_t;
    const int chunks = S >> 3;
    const size_t plane = (size_t)S * (size_t)S;
    __half* const out_img = out + (size_t)blockIdx.y * 3 * plane;
    const int nrows = min(band_rows, S - dy0);
    // the staged rows start after the table of horizontal taps
    XEntry* const s_xtab = reinterpret_cast<XEntry*>(smem);
    unsigned char* const s_rows = smem + (((size_t)S * sizeof(XEntry) + 127) & ~(size_t)127);

    // Does this band touch the image at all?
    const bool any_image = max(dy0, pad_t) < min(dy0 + nrows, pad_t + nh);
    if (!any_image) {
        pdl_wait();
        const uint4 fill4 = make_uint4(fill_h2, fill_h2, fill_h2, fill_h2);
        for (int t = threadIdx.x; t < nrows * chunks; t += kLbThreads) {
            const int r = t / chunks;
            __half* const o0 = out_img + (size_t)(dy0 + r) * S + ((t - r * chunks) << 3);
            *reinterpret_cast<uint4*>(o0) = fill4;
            *reinterpret_cast<uint4*>(o0 + plane) = fill4;
            *reinterpret_cast<uint4*>(o0 + 2 * plane) = fill4;
        }
        return;
    }

    if (threadIdx.x < kLbRows) mbar_init(&bar[threadIdx.x], 1);
    // this warp's row, and its share of it
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int parts = 1 << share, r = warp >> share, part = warp & (parts - 1);
    const int iy = dy0 + r - pad_t;
    const bool image = r < nrows && iy >= 0 && iy < nh;  // else a canvas row, or none
    int y0 = 0, ry = 0;
    if (image) src_coord(iy, h, nh, 1.0f / (float)(2 * nh), y0, ry);
    if (threadIdx.x < kLbRows) {
        mbar_fence_init();
        fence_proxy_async();
    }
    __syncthreads();  // barriers ready
    pdl_wait();
    const uint32_t rows_s = smem_u32(s_rows) + (uint32_t)(r * row_slots * slot_bytes);
    if (image && part == 0 && elect_one()) {
        const uint32_t row_bytes = (uint32_t)((3 * w + 15) & ~15);
        const uint8_t* const src = fd.data + (size_t)y0 * (size_t)fd.pitch;
        mbar_expect_tx(&bar[r], ry != 0 ? 2u * row_bytes : row_bytes);
        bool ok = true;
#ifdef OCTO_BOUNDS_CHECK
        ok = OCTO_IN_RANGE((ry != 0 ? 2 : 1) <= row_slots && (int)row_bytes + 16 <= slot_bytes && y0 + (ry != 0 ? 1 : 0) < h &&
                           (int)row_bytes <= fd.pitch, status);
        if (!ok)  // keep the barrier's byte count right without touching memory
            asm volatile("mbarrier.complete_tx.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&bar[r])),
                         "r"(row_bytes * (ry != 0 ? 2u : 1u)) : "memory");
#endif
        if (ok) {
            bulk_g2s(rows_s, src, row_bytes, smem_u32(&bar[r]));
            if (ry != 0) bulk_g2s(rows_s + (uint32_t)slot_bytes, src + fd.pitch, row_bytes, smem_u32(&bar[r]));
        }
    }
    // table of horizontal taps, built while the copies are in flight
    const float inv_dx = 1.0f / (float)(2 * nw);
    for (int dx = threadIdx.x; dx < S; dx += kLbThreads) {
        const int ix = dx - pad_l;
        XEntry e;
        if (ix < 0 || ix >= nw) { e.off = 0; e.wts = 0; }  // zero weights mark a canvas column
        else e = make_xentry<false>(ix, w, nw, inv_dx, 0);
        s_xtab[dx] = e;
    }
    __syncthreads();  // table visible
    if (r >= nrows) return;

    const int pairs = S >> 1;
    const size_t o = (size_t)(dy0 + r) * S;
    __half* const o0 = out_img + (swap_rb ? 2 : 0) * plane + o;  // plane of input channel 0
    __half* const o1 = out_img + plane + o;
    __half* const o2 = out_img + (swap_rb ? 0 : 2) * plane + o;  // plane of input channel 2
    if (!image || !mbar_wait_or_report(&bar[r], 0, status)) {
        for (int pair = lane + 32 * part; pair < pairs; pair += 32 * parts) {
            *reinterpret_cast<uint32_t*>(o0 + 2 * pair) = fill_h2;
            *reinterpret_cast<uint32_t*>(o1 + 2 * pair) = fill_h2;
            *reinterpret_cast<uint32_t*>(o2 + 2 * pair) = fill_h2;
        }
        return;
    }
    // every scale factor folded into the vertical weights: 1 / (255 * den_x * den_y)
    const float inv_all = 1.0f / (255.0f * (float)(2 * nw) * (float)(2 * nh));
    const float wx = (float)(2 * nh - ry) * inv_all, wy = (float)ry * inv_all;
    const uint32_t xtab_s = smem_u32(s_xtab);
    if (ry != 0) sample_row<true, true>(rows_s, (uint32_t)slot_bytes, wx, wy, xtab_s, pairs, lane, part, parts, o0, o1, o2, fill_h2);
    else sample_row<false, true>(rows_s, (uint32_t)slot_bytes, wx, wy, xtab_s, pairs, lane, part, parts, o0, o1, o2, fill_h2);
}

// Staging slots an output row needs: one when every row of every frame taps a single source
// row (the vertical ratio is an odd integer, e.g. 1080 -> 360), else two.
static int slots_per_row(const FrameDesc* frames, int n) {
    for (int i = 0; i < n; ++i) {
        const int h = frames[i].h, nh = frames[i].nh;
        const bool single = (h % nh == 0) && ((h / nh) & 1);
        if (!single) return 2;
    }
    return 1;
}

static size_t lb_smem_bytes(int S, int slots, int slot_bytes) {
    return (((size_t)S * sizeof(XEntry) + 127) & ~(size_t)127) + (size_t)slots * slot_bytes;
}

// Output rows of a CTA, when `fit` of them fit.  They are halved (7 and 6 to 3, 5 and 3 to 2) until there are eight
// CTAs per SM of more than four rows (five where the table of taps is longer than the source rows of an output row, so that
// it wants to be shared), two and a half of four, four of three (which two of the eight warps have no row of); single
// rows only where two do not fit.
// us a launch over frames that come from memory / lie in L2, by the rows of a CTA (* taken):
//   320x240    @ 640, 12 frames: 8 rows* 12.2 / 12.0, 4 rows 12.9 / 13.1
//   640x480    @ 640, 12 frames: 8 rows* 10.6 / 10.2, 4 rows 11.5 / 11.4;  8 frames: 8 rows 8.0 / 8.1, 4 rows* 8.5 / 8.6
//   800x600    @ 640, 12 frames: 8 rows* 13.6 / 13.7, 4 rows 13.8 / 13.6;  8 frames: 8 rows 10.6 / 10.6, 4 rows* 9.9 / 9.9
//   640x480    @ 640,  3 frames: 4 rows* 5.2 / 4.9, 2 rows 5.4 / 5.3
//   1080x1920  @ 640,  3 frames: 4 rows* 5.2 / 4.7, 2 rows 5.8 / 5.5;  8 frames: 8 rows 9.2 / 9.3, 4 rows* 9.6 / 9.3
//   1920x1080  @ 640,  1 frame:  4 rows 3.6 / 2.8, 2 rows* 3.4 / 2.9;  3 frames: 4 rows* 5.1 / 4.1, 2 rows 4.9 / 4.7
//   1920x1080  @ 640, 12 frames: 8 rows 13.3 / 12.7, 4 rows* 12.0 / 11.9;  32 frames: 8 rows* 27.3 / 26.1
//   1280x720   @ 640,  2 frames: 3 rows 4.8 / 4.0, 2 rows* 4.5 / 4.2, 1 row 5.1 / 5.2
//   1280x720   @ 640,  4 frames: 6 rows 7.0 / 5.5, 4 rows 6.4 / 5.6, 3 rows* 6.1 / 5.6, 2 rows 5.9 / 6.0
//   1280x720   @ 640,  8 frames: 6 rows 11.4 / 11.4, 4 rows 10.4 / 10.0, 3 rows* 9.6 / 9.6, 2 rows 10.4 / 10.2
//   1277x717   @ 416,  4 frames: 7 rows 6.2 / 5.3, 3 rows 5.8 / 4.7, 2 rows* 4.8 / 4.3, 1 row 5.7 / 5.3
//   2560x1440  @ 640,  2 frames: 3 rows 5.7 / 3.8, 2 rows* 5.2 / 4.5, 1 row 5.2 / 5.0
constexpr int letterbox_rows(int fit, int n, int S, bool long_table, int sm_count) {
    int rows = fit < kLbRows ? fit : kLbRows;
    while (rows > 2 && 2ll * n * ((S + rows - 1) / rows) < (rows > 4 ? long_table ? 10ll : 16ll : rows == 4 ? 5ll : 8ll) * sm_count)
        rows = rows > 4 ? rows / 2 : 2;
    return rows;
}
static_assert(letterbox_rows(8, 1, 640, false, 148) == 2 && letterbox_rows(8, 3, 640, false, 148) == 4 &&
              letterbox_rows(8, 14, 640, false, 148) == 4 && letterbox_rows(8, 15, 640, false, 148) == 8 &&
              letterbox_rows(8, 9, 640, true, 148) == 4 && letterbox_rows(8, 10, 640, true, 148) == 8 &&
              letterbox_rows(6, 2, 640, false, 148) == 2 && letterbox_rows(6, 3, 640, false, 148) == 3 &&
              letterbox_rows(7, 4, 416, false, 148) == 2 && letterbox_rows(5, 1, 640, false, 148) == 2 &&
              letterbox_rows(3, 1, 640, false, 148) == 2 && letterbox_rows(3, 3, 640, false, 148) == 3 &&
              letterbox_rows(2, 1, 640, false, 148) == 2 && letterbox_rows(1, 9, 640, false, 148) == 1, "rows as stated");

template <int CAP>
static cudaError_t launch_cap(const FrameDesc* frames, int n, void* d_out, int S, int max_w, int pad_value,
                              int swap_rb, int sm_count, unsigned int* d_status, cudaStream_t stream) {
    FrameTable<CAP> tab;  // built per call (copied into kernel parameter space by the launch)
    for (int i = 0; i < n; ++i) tab.f[i] = frames[i];
    const int slot_bytes = ((3 * max_w + 15) & ~15) + 16;  // 16 bytes of slack: a tap reads 12 bytes from its word
    // as many rows as fit about 56 KB of shared memory (four CTAs per SM), at least one (a single row of the widest
    // supported frame still fits)
    const int per_row = slots_per_row(frames, n) * slot_bytes;
    const long long room = 56 * 1024 - (long long)lb_smem_bytes(S, 0, slot_bytes);
    const int fit = (int)(room / per_row);
    const int band_rows = letterbox_rows(fit < 1 ? 1 : fit, n, S, S * (int)sizeof(XEntry) >= per_row, sm_count);
    int share = 0;  // 2^share warps to a row
    while ((band_rows << (share + 1)) <= kLbThreads / 32) ++share;
    const size_t smem = lb_smem_bytes(S, band_rows * slots_per_row(frames, n), slot_bytes);
    const __half hf = __double2half((double)pad_value / 255.0);  // one rounding, nearest even
    const uint32_t fb = *reinterpret_cast<const unsigned short*>(&hf);
    const uint32_t fill_h2 = fb | (fb << 16);
    dim3 grid((S + band_rows - 1) / band_rows, n);
    return launch_kernel(letterbox_kernel<CAP>, grid, dim3(kLbThreads), smem, stream, tab,
                         reinterpret_cast<__half*>(d_out), S, band_rows, slot_bytes,
                         slots_per_row(frames, n), share, fill_h2, swap_rb, d_status);
}

// largest dynamic shared memory a launch may ask for (see kLetterboxMaxWidth)
constexpr int kLbMaxSmem = 227 * 1024 - 1024;

cudaError_t prepare_letterbox() {
    cudaError_t e;
    e = cudaFuncSetAttribute(letterbox_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, kLbMaxSmem);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(letterbox_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, kLbMaxSmem);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(letterbox_kernel<512>, cudaFuncAttributeMaxDynamicSharedMemorySize, kLbMaxSmem);
}

cudaError_t launch_letterbox(const FrameDesc* frames, int n, void* d_out, int S, int max_w, int pad_value,
                             int swap_rb, int sm_count, unsigned int* d_status, cudaStream_t stream) {
    if (n <= 8) return launch_cap<8>(frames, n, d_out, S, max_w, pad_value, swap_rb, sm_count, d_status, stream);
    if (n <= 64) return launch_cap<64>(frames, n, d_out, S, max_w, pad_value, swap_rb, sm_count, d_status, stream);
    return launch_cap<512>(frames, n, d_out, S, max_w, pad_value, swap_rb, sm_count, d_status, stream);
}

}  // namespace octo
