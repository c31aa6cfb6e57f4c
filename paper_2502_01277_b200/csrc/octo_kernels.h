// Internal launcher interface between the stage object (octo_stage.cu) and the kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

#include "octo.h"
#include "octo_common.cuh"

namespace octo {

typedef octo_det_t octo_det_rec;

struct BranchMasks {
    uint32_t m[OCTO_MAX_BRANCHES][4];
};

struct DecodeArgs {
    const float* d_head;
    int n, A, C;
    int layout;  // OCTO_HEAD_ROWS / OCTO_HEAD_PLANES
    int logits, class_agnostic, multi_label;
    float conf;
    int key_stride;
    unsigned long long* d_keys;
    float4* d_boxes;  // box of every candidate, at its key's slot
    int* d_cand_count;
    unsigned int* d_status;
    int sm_count;
};

struct NmsArgs {
    const FrameDesc* frames;  // host
    const FrameDesc* d_tab;   // device-resident frame table of a chained stage, or null
    int n;
    const float* d_head;
    int A, C;
    int layout;  // OCTO_HEAD_ROWS / OCTO_HEAD_PLANES
    float iou_thr;
    int max_det, key_stride;
    unsigned long long* d_keys;
    float4* d_boxes;
    int* d_cand_count;
    octo_det_t* d_dets;
    int* d_counts;
    int num_branches;
    int class_agnostic;  // NMS across classes; the class of a survivor is recomputed for the output
    BranchMasks masks;
    int full_branches;  // bit b: the mask of branch b holds every class
    int* d_bcount;
    int* d_bidx;        // not written for those branches
    int max_batch;
    StageCounters* d_ctr;
    // CTAs per image (a thread-block cluster; 1, 2, 4 or 8).  More than one pays off when few
    // images carry many candidates each.  d_dense_seen (device pointer to two integers the host can
    // read, or null): the kernel stores launch_seq in [0] / [1] when an image had more than 1024 /
    // 512 candidates; the caller picks the form of later launches from them.
    int cluster;
    int* d_dense_seen;
    int launch_seq;
    // two half-sized CTAs per SM (half the threads and half the on-chip capacity each) instead of
    // one: for batches of more images than SMs whose images are sparse
    bool half_ctas;
};

// Branch options of the crop kernel, per INPUT channel c (output plane swap_rb ? 2 - c : c):
// value' = value * sc[c] + of[c]; fill[c] is the canvas value after the same mapping.
struct CropOpts {
    int keep_aspect;
    float sc[3], of[3], fill[3];
};

struct CropArgs {
    const FrameDesc* frames;  // host
    const FrameDesc* d_tab;   // device-resident frame table of a chained stage, or null
    int n;
    int max_w, max_h;  // largest frame
    int max_det, first_item, max_items;
    const int* d_bcount;  // this branch's [max_batch]
    const int* d_bidx;    // this branch's [max_batch][max_det], or null: item j of a frame is its detection j
    const octo_det_t* d_dets;
    int* d_offsets;
    int* d_n_items;
    octo_item_t* d_items;
    void* d_out;
    int out_w, out_h, swap_rb, sm_count;
    StageCounters* d_ctr;
    bool general;   // keep_aspect or normalize set for the branch
    CropOpts opts;
};

// Branch options -> kernel form (per input channel, see CropOpts).
void fill_crop_opts(const octo_branch_cfg_t& br, int swap_rb, int pad_value, CropOpts* out);
int validate_branch_options(const octo_branch_cfg_t& br);  // OCTO_OK or OCTO_E_INVALID_ARG

// Records the text that octo_last_cuda_error returns on this thread; returns OCTO_E_CUDA.
int report_cuda_error(cudaError_t e, const char* what);

// Opt the kernels of every table capacity into the shared memory they need (current device).
cudaError_t prepare_letterbox();
cudaError_t prepare_decode();
// clusters (optional): how many clusters of 2, 4 and 8 CTAs of the NMS kernel the current device holds at once.
constexpr int kNmsClusterSizes = 3;
cudaError_t prepare_nms(int* clusters = nullptr);
cudaError_t prepare_crop();

cudaError_t launch_letterbox(const FrameDesc* frames, int n, void* d_out, int S, int max_w, int pad_value,
                             int swap_rb, int sm_count, unsigned int* d_status, cudaStream_t stream);
cudaError_t launch_decode(const DecodeArgs& a, cudaStream_t stream);
cudaError_t launch_nms(const NmsArgs& a, cudaStream_t stream);
cudaError_t launch_crop(const CropArgs& a, cudaStream_t stream);  // batch assembler + crop-resize
cudaError_t launch_crop_queue(const QRecord* d_staged, const int* d_qpacked, int bz, void* d_out, int out_w,
                              int out_h, int swap_rb, int sm_count, unsigned int* d_status, int* d_sched,
                              const CropOpts* general, int max_w, int max_h, cudaStream_t stream);

constexpr int kLetterboxMaxWidth = 8192;  // widest frame the row staging supports

// One kernel launch with the programmatic stream serialisation attribute: the kernel may be scheduled
// while its predecessor in the stream ends (it waits for it in pdl_wait before it touches memory).  With
// `cluster` > 1, thread-block clusters of that many CTAs along x (grid.x is a multiple of it).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel_cluster(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                                         cudaStream_t stream, int cluster, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    unsigned na = 0;
    attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[na].val.programmaticStreamSerializationAllowed = 1;
    ++na;
    if (cluster > 1) {
        attr[na].id = cudaLaunchAttributeClusterDimension;
        attr[na].val.clusterDim.x = (unsigned)cluster;
        attr[na].val.clusterDim.y = 1;
        attr[na].val.clusterDim.z = 1;
        ++na;
    }
    cfg.attrs = attr;
    cfg.numAttrs = na;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                                 Args&&... args) {
    return launch_kernel_cluster(kernel, grid, block, smem, stream, 1, std::forward<Args>(args)...);
}

}  // namespace octo
