// Host launcher and instantiations of the tiled forward projection (forward_tiled.cuh).
#include <algorithm>

#include "forward_tiled.cuh"
#include "tensor_map.h"

namespace radon {

namespace {

constexpr uint32_t kSpinLimit = 1u << 22;   // bounded mbarrier polls (~seconds) before giving up
constexpr long long kFwdFourMinCtas = 300;   // CTAs of four texel groups below which smaller ones fill the GPU better

// FP16 storage takes FP16 weights in mixed-precision FMAs only when the config asks for them and the
// epilogue adds nothing to the projection (a fused residual keeps FP32 weights); the default is FP32.
bool fp16_weights(const radon_launch_config* cfg, const Epilogue& ep) {
    return cfg != nullptr && cfg->weights == RADON_WEIGHTS_F16 && ep.add == nullptr;
}

template <typename T, int MODE>
cudaError_t launch_t(const CUtensorMap& mv, const CUtensorMap& mh, const FwdTiledArgs& a, dim3 grid, size_t smem,
                     cudaStream_t s) {
    auto kern = forward_tiled_kernel<T, MODE>;
    static size_t attr_bytes = 0;
    if (smem > attr_bytes) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        attr_bytes = smem;
    }
    kern<<<grid, kFwdThreads, smem, s>>>(mv, mh, a);
    return cudaGetLastError();
}

}  // namespace

radon_status launch_forward_tiled(radon_geometry* g, const void* img, void* sino, radon_dtype dt, int batch,
                                  const radon_launch_config* cfg, const Epilogue& ep, cudaStream_t s,
                                  std::string* why) {
    const int esz = dt == RADON_F32 ? 4 : 2;
    const int align = 16 / esz;
    const int BG = 16 / esz;
    if (g->n % align != 0) {
        *why = "image side must be a multiple of 16 bytes of storage for TMA rows";
        return RADON_ERR_UNSUPPORTED;
    }
    if (((uintptr_t)img & 15) != 0) {
        *why = "image pointer not 16-byte aligned";
        return RADON_ERR_UNSUPPORTED;
    }
    int G = cfg && cfg->views_per_cta ? cfg->views_per_cta : 4;
    if (G != 1 && G != 2 && G != 4 && G != 8) {
        *why = "views_per_cta must be 1, 2, 4 or 8 for the tiled forward";
        return RADON_ERR_UNSUPPORTED;
    }
    const int Dt = kFwdRays / G;
    const int R = cfg && cfg->rows_per_slab ? cfg->rows_per_slab : 8;
    if (R < 2 || R > 64 || (R & 1)) {
        *why = "rows_per_slab must be even and in [2, 64]";
        return RADON_ERR_UNSUPPORTED;
    }
    const int maxw = forward_band_width(g, G, Dt, R);
    const int wbox = (maxw + 2 + align - 1 + align - 1) / align * align;
    const int rbox_h = (R + align + align - 1) / align * align;   // R + 2 rows at an even offset < align
    if (wbox > 256 || rbox_h > 256) {
        *why = "working band wider than a TMA box";
        return RADON_ERR_UNSUPPORTED;
    }
    const int wc = (wbox + 7) / 8 * 8;   // row pitch = 0 (mod 8) texels: fewest shared-memory bank conflicts
    const int stage_bytes = std::max(wbox * (R + 2) * 16, rbox_h * wbox * 16);
    const size_t smem = fwd_smem_bytes(stage_bytes, R, wc);
    if (smem > 227 * 1024) {
        *why = "shared memory budget exceeded";
        return RADON_ERR_UNSUPPORTED;
    }
    int gi = 0;
    while ((1 << gi) < G) ++gi;
    const uint64_t dims[3] = {(uint64_t)g->n, (uint64_t)g->n, (uint64_t)batch};
    const uint64_t strides[2] = {(uint64_t)g->n * esz, (uint64_t)g->n * g->n * esz};
    const uint32_t box_v[3] = {(uint32_t)wbox, (uint32_t)(R + 2), (uint32_t)BG};
    const uint32_t box_h[3] = {(uint32_t)rbox_h, (uint32_t)wbox, (uint32_t)BG};
    CUtensorMap mv, mh;
    int rc = encode_tiled(&mv, tma_dtype(dt), 3, const_cast<void*>(img), dims, strides, box_v,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_128B);
    if (rc == 0)
        rc = encode_tiled(&mh, tma_dtype(dt), 3, const_cast<void*>(img), dims, strides, box_h,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_128B);
    if (rc != 0) {
        *why = "cuTensorMapEncodeTiled rejected the image descriptor (CUresult " + std::to_string(rc) + ")";
        return RADON_ERR_UNSUPPORTED;
    }
    FwdTiledArgs a;
    a.rays = g->d_ray;
    a.nks = g->d_nk;
    a.groups = g->d_groups + g->group_offset[gi];
    a.sino = sino;
    a.n = g->n;
    a.V = g->V;
    a.D = g->D;
    a.B = batch;
    a.h = (float)g->h;
    a.ep = ep;
    a.G = G;
    a.Dt = Dt;
    a.pair_views = G >= 2 && g->fwd_pair_views ? 1 : 0;
    a.n_dr = (g->D + Dt - 1) / Dt;
    a.R = R;
    a.n_slabs = (g->n + 4 + R - 1) / R;
    a.wbox = wbox;
    a.wc = wc;
    a.rbox_h = rbox_h;
    a.align = align;
    a.stage_bytes = stage_bytes;
    a.err = device_error_word();
    if (a.err == nullptr) {
        *why = "device error word unavailable";
        return RADON_ERR_CUDA;
    }
    a.spin_limit = kSpinLimit;
    a.stages = 2;
    a.vec_store = (g->D % 2 == 0 && ((uintptr_t)sino % (2 * esz)) == 0) ? 1 : 0;
    const long long nblk = (long long)g->group_count[gi] * a.n_dr;
    if (nblk > 0x7fffffffLL) {
        *why = "too many CTAs";
        return RADON_ERR_UNSUPPORTED;
    }
    dim3 grid((unsigned)nblk, (unsigned)((batch + BG - 1) / BG));
    cudaError_t e;
    switch (dt) {
        case RADON_F16:
            e = fp16_weights(cfg, ep) ? launch_t<__half, kMathF16W>(mv, mh, a, grid, smem, s)
                                      : launch_t<__half, kMathScalar>(mv, mh, a, grid, smem, s);
            break;
        case RADON_BF16: e = launch_t<__nv_bfloat16, kMathScalar>(mv, mh, a, grid, smem, s); break;
        default: e = launch_t<float, kMathScalar>(mv, mh, a, grid, smem, s); break;
    }
    if (e != cudaSuccess) {
        *why = std::string("tiled forward launch: ") + cudaGetErrorString(e);
        return RADON_ERR_CUDA;
    }
    return RADON_OK;
}

}  // namespace radon

namespace radon {

namespace {

template <typename T, int MODE, int NG, int LN, bool ROWS>
cudaError_t launch_packed_ng(const CUtensorMap& mr, const CUtensorMap& mc, const FwdTiledArgs& a, dim3 grid,
                             size_t smem, cudaStream_t s) {
    auto kern = forward_packed_kernel<T, MODE, NG, LN, ROWS>;
    static size_t attr_bytes = 0;
    if (smem > attr_bytes) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        attr_bytes = smem;
    }
    if constexpr (ROWS && NG < 4) {   // beside the launch of four groups before it
        cudaLaunchAttribute beside;
        beside.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        beside.val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t c = {};
        c.gridDim = grid;
        c.blockDim = dim3(kFwdThreads);
        c.dynamicSmemBytes = smem;
        c.stream = s;
        c.attrs = &beside;
        c.numAttrs = 1;
        return cudaLaunchKernelEx(&c, kern, mr, mc, a);
    }
    kern<<<grid, kFwdThreads, smem, s>>>(mr, mc, a);
    return cudaGetLastError();
}

template <typename T, int MODE>
cudaError_t launch_packed_t(const CUtensorMap& mr, const CUtensorMap& mc, const FwdTiledArgs& a, dim3 grid,
                            size_t smem, int NG, int LN, bool rows, cudaStream_t s) {
    if (LN == 2) return launch_packed_ng<T, MODE, 1, 2, false>(mr, mc, a, grid, smem, s);
    if constexpr (MODE == kMathScalar) {
        if (NG == 4) return launch_packed_ng<T, MODE, 4, 1, true>(mr, mc, a, grid, smem, s);
        if (rows)
            return NG == 2 ? launch_packed_ng<T, MODE, 2, 1, true>(mr, mc, a, grid, smem, s)
                           : launch_packed_ng<T, MODE, 1, 1, true>(mr, mc, a, grid, smem, s);
    }
    return NG == 2 ? launch_packed_ng<T, MODE, 2, 1, false>(mr, mc, a, grid, smem, s)
                   : launch_packed_ng<T, MODE, 1, 1, false>(mr, mc, a, grid, smem, s);
}

}  // namespace

radon_status packed_forward_shape(radon_geometry* g, radon_dtype dt, int batch, const radon_launch_config* cfg,
                                  bool f16w, int lanes, PackedFwdShape* out, std::string* why) {
    const int esz = dt == RADON_F32 ? 4 : 2;
    const int BG = 16 / esz;
    const int G = cfg && cfg->views_per_cta ? cfg->views_per_cta : 8;
    if (G != 1 && G != 2 && G != 4 && G != 8) {
        *why = "views_per_cta must be 1, 2, 4 or 8 for the tiled forward";
        return RADON_ERR_UNSUPPORTED;
    }
    if (lanes != 1 && lanes != 2) {
        *why = "lanes per ray must be 1 or 2";
        return RADON_ERR_UNSUPPORTED;
    }
    const int Dt = kFwdRays / (G * lanes);
    // images per CTA: one texel group (BG images) or two groups sharing each sample's index work
    const int ipc = cfg ? cfg->images_per_cta : 0;
    if (ipc != 0 && ipc != BG && ipc != 2 * BG) {
        *why = "images_per_cta must be 0, " + std::to_string(BG) + " or " + std::to_string(2 * BG) +
               " for the packed forward";
        return RADON_ERR_UNSUPPORTED;
    }
    if (lanes == 2 && ipc == 2 * BG) {
        *why = "two lanes per ray take one texel group";
        return RADON_ERR_UNSUPPORTED;
    }
    // Default: 16-bit batches of more than one group pair their groups (one sample's index and weight
    // work then serves 16 images; measured 7-9 % faster on the fan and parallel workloads); FP32
    // texels (4 images each) measured slower paired.  Rows per slab: 16 for one group; 14 for two
    // (2 CTAs/SM), 8 with FP16 weights (3 CTAs/SM), the fastest of 8-16 rows measured.  A default pair
    // whose buffers would not fit falls back to one group.
    // Four groups, row by row, where the batch fills most of one more CTA: 16-bit batches of more than 24 images
    // (parallel 32 x 512^2, 512 views: FP16 1.78 -> 1.35 ms, BF16 1.55 -> 1.20; three groups cost about what a pair
    // and a single do) and FP32 batches of more than 16 (2.33 -> 1.56 ms; 32 x 256^2, 256 views 376 -> 242 us; smaller
    // FP32 batches keep the one group that the query reports for them), in the highest slab of 8, 6 or 4 rows that
    // leaves two CTAs per SM (with the left-over groups still in the kernel, FP16: 8 rows 1.45 ms, 6 1.48, 4 1.56; 10
    // rows at one CTA 1.88).  FP16 weights keep two groups.  Not where the CTAs of four groups would not fill two per
    // SM (us, default -> four groups, FP16: 32 x 256^2, 128 views, 204 CTAs 177 -> 194; 192 views, 300 CTAs 242 ->
    // 239; 256 views, 396 CTAs 284 -> 246), nor, since a CTA costs the same with empty groups and thin slabs repeat
    // the rows between them, where groups are empty and the slab is low: FP32, against one group per CTA, needs 6 rows
    // (32 x 512^2, 100 views, 4 rows: 682 -> 891; 32 x 256^2, 128 views, 6 rows: 219 -> 178), either type two more
    // with two groups empty (FP32 24 x 256^2, 256 views, 8 rows: 289 -> 239; 24 x 266^2 fan, 586 views, 6 rows: 570 ->
    // 640) and FP32 never runs with three (20 x 512^2, 150 views: 579 -> 958).
    // Nor where too few of the samples lie on rays that go by rows: sample by sample four groups only leave fewer CTAs
    // (steps other than one pixel; us, default -> four groups at a share of 0 | 0.4 | 0.6 | 0.75 | 0.85: 32 x 512^2,
    // 300 views, FP32 2104 -> 2306 | 1858 -> 1608 | 1759 -> 1383; 25 x 215^2, 219 views, 314 -> 418 | 279 -> 311 | 266
    // -> 272 | 253 -> 237; 32 x 256^2, 256 views, FP16 438 -> 463 | 382 -> 469 | 357 -> 400 | 337 -> 337, and 512^2
    // 1686 -> 1753 | 1472 -> 1315 | 1382 -> 1151; with steps above one, where the rays nearest the rows' normal fall
    // out, 273 -> 322 and 1043 -> 1040 at 0.75; where some do not, twice the CTAs are needed to even out those that
    // take longer: at 0.85, 396 CTAs, 320 -> 357).  (One or two groups past whole CTAs now run beside them and cost
    // less: 24 x 256^2, 256 views, 201.)
    const int groups = (batch + BG - 1) / BG;
    const int empty = groups < 12 ? (4 - groups % 4) % 4 : 0;   // (of many, a few cost little)
    const int min_rows = 4 + (esz == 4 ? 2 : 0) + (empty >= 2 ? 2 : 0);
    const long long ctas4 = (long long)g->group_count[G >= 8 ? 3 : G >= 4 ? 2 : G >= 2 ? 1 : 0] * ((g->D + Dt - 1) / Dt) *
                            ((groups + 3) / 4);
    const int fixed_rows = cfg ? cfg->rows_per_slab : 0;
    const double min_share = esz == 4 ? 0.55 : g->h > 1.0 ? 0.9 : 0.7;
    const bool four = !f16w && g->row_share >= min_share && batch > (esz == 2 ? 24 : 16) && !(esz == 4 && empty == 3) &&
                      ctas4 >= kFwdFourMinCtas * (g->row_share < 0.98 ? 2 : 1) &&
                      (fixed_rows == 0 || fixed_rows >= min_rows);
    int NG = lanes == 2 ? 1
             : ipc != 0 ? (ipc == 2 * BG ? 2 : 1)
             : four     ? 4
                        : (esz == 2 && batch > BG ? 2 : 1);
    int R = fixed_rows ? fixed_rows : 8;   // of four groups, lowered until they fit
    for (;;) {
        if (NG != 4) R = fixed_rows ? fixed_rows : (NG == 2 ? (f16w ? 8 : 14) : 16);
        if (R < 2 || R > 64 || (R & 1)) {
            *why = "rows_per_slab must be even and in [2, 64]";
            return RADON_ERR_UNSUPPORTED;
        }
        const int maxw = forward_band_width(g, G, Dt, R);
        const int wbox = (maxw + 2 + 7) / 8 * 8;   // row pitch = 0 (mod 8) texels: fewest bank conflicts (measured)
        // As many ring stages (up to 4) as keep three CTAs resident per SM (3 x (smem + 1 KB) <= 228 KB), two
        // of four groups.
        const size_t room = (NG == 4 ? 113 : 75) * 1024;
        int stages = 2;
        while (stages < kFwdMaxStages && fwd_packed_smem_bytes(R, wbox, stages + 1, NG) <= room) ++stages;
        const size_t smem = fwd_packed_smem_bytes(R, wbox, stages, NG);
        if (NG == 4 && (wbox > 256 || smem > room)) {
            if (!fixed_rows && R > min_rows) R -= 2;
            else NG = esz == 2 ? 2 : 1;
            continue;
        }
        if (wbox > 256) {
            *why = "working band wider than a TMA box";
            return RADON_ERR_UNSUPPORTED;
        }
        if (smem <= 227 * 1024) {
            *out = PackedFwdShape{G, Dt, NG, lanes, R, wbox, stages, smem};
            return RADON_OK;
        }
        if (ipc == 0 && NG == 2) {
            NG = 1;
            continue;
        }
        *why = "shared memory budget exceeded";
        return RADON_ERR_UNSUPPORTED;
    }
}

radon_status launch_forward_packed(radon_geometry* g, const void* packed, void* sino, radon_dtype dt, int batch,
                                   const radon_launch_config* cfg, const Epilogue& ep, cudaStream_t s,
                                   std::string* why, int lanes) {
    const int esz = dt == RADON_F32 ? 4 : 2;
    const int BG = 16 / esz;
    if (((uintptr_t)packed & 15) != 0) {
        *why = "workspace not 16-byte aligned";
        return RADON_ERR_UNSUPPORTED;
    }
    PackedFwdShape sh;
    const radon_status st =
        packed_forward_shape(g, dt, batch, cfg, dt == RADON_F16 && fp16_weights(cfg, ep), lanes, &sh, why);
    if (st != RADON_OK) return st;
    const int G = sh.G, Dt = sh.Dt, LN = sh.LN, R = sh.R, wbox = sh.wbox;
    int gi = 0;
    while ((1 << gi) < G) ++gi;
    const int groups = (batch + BG - 1) / BG;
    const uint64_t n = (uint64_t)g->n;
    const uint64_t dims[4] = {(uint64_t)BG, n, n, (uint64_t)groups};
    const uint64_t strides[3] = {16, n * 16, n * n * 16};
    const unsigned char* rows = reinterpret_cast<const unsigned char*>(packed);
    const unsigned char* cols = rows + (size_t)groups * n * n * 16;
    FwdTiledArgs a;
    a.rays = g->d_ray;
    a.nks = g->d_nk;
    a.groups = g->d_groups + g->group_offset[gi];
    a.sino = sino;
    a.n = g->n;
    a.V = g->V;
    a.D = g->D;
    a.B = batch;
    a.h = (float)g->h;
    a.ep = ep;
    a.G = G;
    a.Dt = Dt;
    a.pair_views = LN == 1 && G >= 2 && g->fwd_pair_views ? 1 : 0;
    a.n_dr = (g->D + Dt - 1) / Dt;
    a.R = R;
    a.n_slabs = (g->n + 4 + R - 1) / R;
    a.wbox = wbox;
    a.wc = wbox;
    a.rbox_h = 0;
    a.align = 1;
    a.stage_bytes = 0;
    a.err = device_error_word();
    if (a.err == nullptr) {
        *why = "device error word unavailable";
        return RADON_ERR_CUDA;
    }
    a.spin_limit = kSpinLimit;
    a.vec_store = (g->D % 2 == 0 && ((uintptr_t)sino % (2 * esz)) == 0) ? 1 : 0;
    const long long nblk = (long long)g->group_count[gi] * a.n_dr;
    const bool f16w = dt == RADON_F16 && fp16_weights(cfg, ep);
    // Groups [g0, g0 + count) in CTAs of NG groups.
    auto launch = [&](int g0, int count, int NG, int stages, size_t smem, bool by_rows) {
        const uint32_t box[4] = {(uint32_t)BG, (uint32_t)wbox, (uint32_t)(R + 2), (uint32_t)NG};
        CUtensorMap mr, mc;
        int rc = encode_tiled(&mr, tma_dtype(dt), 4, const_cast<unsigned char*>(rows), dims, strides, box,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_128B);
        if (rc == 0)
            rc = encode_tiled(&mc, tma_dtype(dt), 4, const_cast<unsigned char*>(cols), dims, strides, box,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_128B);
        if (rc != 0) {
            *why = "cuTensorMapEncodeTiled rejected the packed-image descriptor (CUresult " + std::to_string(rc) + ")";
            return RADON_ERR_UNSUPPORTED;
        }
        a.g0 = g0;
        a.stages = stages;
        const dim3 grid((unsigned)nblk, (unsigned)((count + NG - 1) / NG));
        cudaError_t e;
        switch (dt) {
            case RADON_F16:
                e = f16w ? launch_packed_t<__half, kMathF16W>(mr, mc, a, grid, smem, NG, LN, by_rows, s)
                         : launch_packed_t<__half, kMathScalar>(mr, mc, a, grid, smem, NG, LN, by_rows, s);
                break;
            case RADON_BF16:
                e = launch_packed_t<__nv_bfloat16, kMathScalar>(mr, mc, a, grid, smem, NG, LN, by_rows, s);
                break;
            default: e = launch_packed_t<float, kMathScalar>(mr, mc, a, grid, smem, NG, LN, by_rows, s); break;
        }
        if (e != cudaSuccess) {
            *why = std::string("packed forward launch: ") + cudaGetErrorString(e);
            return RADON_ERR_CUDA;
        }
        return RADON_OK;
    };
    // One or two groups past whole CTAs of four run by themselves, row by row like the others with the same slabs, so
    // that equal images of a batch have equal projections; and with their code out of the kernel of four
    // groups it keeps its registers.  They start as the last CTAs of four do (their inputs were packed before
    // that launch, their outputs are other images) and fill the SMs that those leave.  (us, one launch that
    // takes them sample by sample -> two one after the other -> two so, FP16: 34 x 512^2, 512 views 1993 ->
    // 1941 -> 1782; 40 x 256^2, 202 views 283 -> 333 -> 274; 100 x 128^2, 162 views 148 -> 186 -> 152; no tail,
    // 32 x 512^2, 512 views 1387 -> 1345, BF16 1279 -> 1203.)
    const int tail = sh.NG == 4 && groups % 4 <= 2 ? groups % 4 : 0;
    radon_status done = launch(0, groups - tail, sh.NG, sh.stages, sh.smem, sh.NG == 4);
    if (done == RADON_OK && tail > 0) {
        int stages = 2;
        while (stages < kFwdMaxStages && fwd_packed_smem_bytes(R, wbox, stages + 1, tail) <= (tail == 2 ? 113 : 75) * 1024) ++stages;
        done = launch(groups - tail, tail, tail, stages, fwd_packed_smem_bytes(R, wbox, stages, tail), true);
        if (done == RADON_OK) count_launches(1);
        else if (done == RADON_ERR_UNSUPPORTED) done = RADON_ERR_CUDA;   // the first launch has run: no other path
    }
    return done;
}

}  // namespace radon
