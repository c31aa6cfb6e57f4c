// NMS launch (one CTA or one thread-block cluster per image); the work is in octo_nms.cuh.
#include "octo_nms.cuh"

#include <cmath>
#include <cstring>

namespace octo {

template <int CAP, int NT>
__global__ void __launch_bounds__(NT, kNmsThreadsFull / NT)
nms_kernel(const __grid_constant__ FrameTable<CAP> tab, const FrameDesc* __restrict__ gtab,
           const __grid_constant__ NmsParams params) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // fetch the parameters' constant-cache lines while the launch waits for its predecessor
    asm volatile("" ::"l"(params.bidx), "l"(params.bcount), "l"(params.counts), "l"(params.dets), "l"(params.gkeys),
                 "l"(params.ctr), "r"(params.masks.m[0][0]), "r"(params.launch_seq), "r"(params.num_branches),
                 "f"(tab.f[0].gx), "r"(tab.f[0].w));
    pdl_wait();
    constexpr bool kCluster = NT == kNmsThreadsFull;  // half-sized CTAs never form clusters
    const int img = (int)(blockIdx.x / (kCluster ? cg::this_cluster().num_blocks() : 1u));
    // The frame table comes by value (first-level stages) or from device memory (chained stages,
    // where an entry without a frame stands for an unused slot of the batch: no detections).
    const FrameDesc fd = gtab ? gtab[img] : tab.f[img];
    nms_image<NT, kCluster ? kNmsSmemCap : kNmsSmemCapHalf, kCluster>(params, fd, gtab && fd.data == nullptr, img, smem_raw);
}

static NmsParams nms_params(const NmsArgs& a) {
    NmsParams p;
    p.head = a.d_head;
    p.A = a.A; p.C = a.C; p.layout = a.layout;
    // rounding boundary of the IoU test (see iou_exact)
    const float up = nextafterf(a.iou_thr, INFINITY);
    p.iou_test.mid = 0.5 * ((double)a.iou_thr + (double)up);
    const bool quick = p.iou_test.mid >= 0x1p-60;
    p.iou_test.midf = quick ? (float)p.iou_test.mid : NAN;
    p.iou_test.share = quick ? (float)(p.iou_test.mid / (1.0 + p.iou_test.mid)) : NAN;
    unsigned int up_bits;
    memcpy(&up_bits, &up, sizeof(up_bits));
    p.iou_test.tie_up = (up_bits & 1u) == 0u ? 1 : 0;
    p.max_det = a.max_det; p.key_stride = a.key_stride;
    p.gkeys = a.d_keys; p.gboxes = a.d_boxes; p.cand_count = a.d_cand_count;
    p.dets = reinterpret_cast<octo_det_rec*>(a.d_dets);
    p.counts = a.d_counts;
    p.num_branches = a.num_branches; p.class_agnostic = a.class_agnostic;
    p.masks = a.masks;
    p.full_branches = a.full_branches;
    p.bcount = a.d_bcount; p.bidx = a.d_bidx;
    p.max_batch = a.max_batch;
    p.ctr = a.d_ctr;
    p.dense_seen = a.d_dense_seen;
    p.launch_seq = a.launch_seq;
    return p;
}

cudaError_t prepare_nms(int* clusters) {
    cudaError_t e;
    e = cudaFuncSetAttribute(nms_kernel<8, kNmsThreadsFull>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kNmsSmemBytes);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(nms_kernel<64, kNmsThreadsFull>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kNmsSmemBytes);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(nms_kernel<512, kNmsThreadsFull>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kNmsSmemBytes);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(nms_kernel<512, kNmsThreadsHalf>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kNmsSmemBytesHalf);
    if (e != cudaSuccess) return e;
    if (clusters) {
        // (one CTA per SM: the kernel takes nearly all shared memory of an SM)
        for (int k = 0; k < kNmsClusterSizes; ++k) {
            const int c = 2 << k;
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3((unsigned)c);
            cfg.blockDim = dim3(kNmsThreadsFull);
            cfg.dynamicSmemBytes = kNmsSmemBytes;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = (unsigned)c;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            clusters[k] = 0;
            if (cudaOccupancyMaxActiveClusters(&clusters[k], nms_kernel<8, kNmsThreadsFull>, &cfg) != cudaSuccess) {
                clusters[k] = 0;
                (void)cudaGetLastError();
            }
        }
    }
    return cudaSuccess;
}

template <int CAP>
static cudaError_t launch_cap(const NmsArgs& a, cudaStream_t stream) {
    FrameTable<CAP> tab;  // built per call (copied into kernel parameter space by the launch)
    if (!a.d_tab)
        for (int i = 0; i < a.n; ++i) tab.f[i] = a.frames[i];
    const int cluster = a.cluster == 2 || a.cluster == 4 || a.cluster == 8 ? a.cluster : 1;
    // two half-sized CTAs per SM: only the largest table size has that form (more images than SMs)
    const bool half = CAP == 512 && a.half_ctas && cluster == 1;
    auto kernel = nms_kernel<CAP, kNmsThreadsFull>;
    if constexpr (CAP == 512) {
        if (half) kernel = nms_kernel<512, kNmsThreadsHalf>;
    }
    return launch_kernel_cluster(kernel, dim3((unsigned)(a.n * cluster)), dim3(half ? kNmsThreadsHalf : kNmsThreadsFull),
                                 half ? kNmsSmemBytesHalf : kNmsSmemBytes, stream,
                                 cluster, tab, a.d_tab, nms_params(a));
}

cudaError_t launch_nms(const NmsArgs& a, cudaStream_t stream) {
    if (a.n <= 8) return launch_cap<8>(a, stream);
    if (a.n <= 64) return launch_cap<64>(a, stream);
    return launch_cap<512>(a, stream);
}

}  // namespace octo
