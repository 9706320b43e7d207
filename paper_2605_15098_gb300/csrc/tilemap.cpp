// Tensor description of a pass's tiles (tilemap.h).
#include "tilemap.h"

#include <algorithm>
#include <cstring>

namespace sv {

void tile_dims(int n, int k, const int *slot_phys, size_t amp_bytes, TileDims *dims, TileBox *box) {
    constexpr int kMaxLen = 8;    // a box holds at most 256 elements per dimension
    constexpr int kMaxSpan = 30;  // a dimension's coordinate is a 32-bit signed integer
    const int w = amp_bytes == 16 ? 1 : 0;
    // local word bits, ascending; runs of at most kMaxLen
    int bits[kMaxTileQubits + 1], nb = 0;
    if (w) bits[nb++] = 0;
    for (int s = 0; s < k; s++) bits[nb++] = slot_phys[s] + w;
    std::memset(box, 0, sizeof *box);
    int start[kTileDims], len[kTileDims], nd = 0, b = 0;
    while (b < nb && nd < kTileDims) {
        // a gap too wide for one coordinate takes a dimension without a local run
        if (nd && bits[b] - start[nd - 1] > kMaxSpan) {
            start[nd] = start[nd - 1] + kMaxSpan;
            len[nd++] = 0;
            continue;
        }
        int e = b + 1;
        while (e < nb && bits[e] == bits[e - 1] + 1 && e - b < kMaxLen) e++;
        start[nd] = bits[b];
        len[nd++] = e - b;
        b = e;
    }
    int inside = 0;
    for (int i = 0; i < nd; i++) inside += len[i];
    for (; b < nb; b++) box->ext[box->next++] = (int8_t)bits[b];
    const int top = n + w;
    // the last dimension reaches the top of the state; where that is too wide
    // and a dimension is left, split it
    if (nd < kTileDims && top - start[nd - 1] > kMaxSpan) {
        start[nd] = start[nd - 1] + kMaxSpan;
        len[nd++] = 0;
    }
    for (int i = 0; i < kTileDims; i++) {
        if (i < nd) {
            const int end = i + 1 < nd ? start[i + 1] : top;
            dims->size[i] = UINT64_C(1) << (end - start[i]);
            dims->stride[i] = UINT64_C(8) << start[i];
            dims->width[i] = 1u << len[i];
            box->pos[i] = (int8_t)start[i];
        } else {
            dims->size[i] = 1;
            dims->stride[i] = UINT64_C(8) << top;
            dims->width[i] = 1;
            box->pos[i] = 0;
        }
        box->mask[i] = (uint32_t)(dims->size[i] - 1);
    }
    box->copy_bytes = 8u << inside;
}

namespace {
using EncodeFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                              const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeFn encode_fn() {
    static const EncodeFn fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            p = nullptr;
        }
        return reinterpret_cast<EncodeFn>(p);
    }();
    return fn;
}
}  // namespace

sv_status tile_map(void *amps, int n, int k, const int *slot_phys, size_t amp_bytes, CUtensorMap *map,
                   TileBox *box) {
    TileDims d;
    tile_dims(n, k, slot_phys, amp_bytes, &d, box);
    const EncodeFn fn = encode_fn();
    if (!fn) return fail(SV_ERR_CUDA, "the driver has no tensor map encoder");
    cuuint64_t size[kTileDims], stride[kTileDims - 1];
    cuuint32_t width[kTileDims], step[kTileDims];
    for (int i = 0; i < kTileDims; i++) {
        size[i] = d.size[i];
        width[i] = d.width[i];
        step[i] = 1;
        if (i) stride[i - 1] = d.stride[i];
    }
    const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, kTileDims, amps, size, stride, width, step,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(SV_ERR_CUDA, "tensor map of a tile pass refused (%d)", (int)r);
    return SV_OK;
}

}  // namespace sv
