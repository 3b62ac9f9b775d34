// The context's grow-only device workspace.
#pragma once

#include <cuda_runtime_api.h>

#include "ctx.h"
#include "pcl.h"

namespace pcl {

inline size_t ws_request(size_t bytes) { return bytes + bytes / 4 + 4096; }

inline pcl_status ensure_ws(pcl_ctx *ctx, size_t bytes) {
    if (bytes <= ctx->ws_bytes) return PCL_OK;
    if (ctx->ws) {
        cudaFree(ctx->ws);  // synchronises the device: no kernel still uses it
        ctx->ws = nullptr;
        ctx->ws_bytes = 0;
    }
    const size_t want = ws_request(bytes);
    if (cudaMalloc(&ctx->ws, want) != cudaSuccess) {
        cudaGetLastError();
        ctx->ws = nullptr;
        ctx->err = "workspace allocation of " + std::to_string(want) + " bytes failed";
        return PCL_ERR_OOM;
    }
    ctx->ws_bytes = want;
    return PCL_OK;
}

// A larger workspace for a faster path, if it can be had: not while st is being
// captured (an allocation would end the capture; a smaller one may be there
// from an earlier call).  Each try gives the present workspace back first, so a size
// that did not fit is tried again only once the device has the memory free.
inline bool ensure_ws_optional(pcl_ctx *ctx, size_t bytes, cudaStream_t st) {
    if (bytes <= ctx->ws_bytes) return true;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (cap != cudaStreamCaptureStatusNone) return false;
    if (ctx->ws_refused && bytes >= ctx->ws_refused) {
        size_t avail = 0, total = 0;
        if (cudaMemGetInfo(&avail, &total) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        if (avail + ctx->ws_bytes < ws_request(bytes)) return false;
    }
    if (ensure_ws(ctx, bytes) == PCL_OK) {
        ctx->ws_refused = 0;
        return true;
    }
    ctx->ws_refused = bytes;
    ctx->err.clear();
    return false;
}

}  // namespace pcl
