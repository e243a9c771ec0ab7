// Host-side helpers shared by the translation units of libshiftquant: error reporting,
// argument checks and the code-format rules.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <cstdio>

#include "../../include/shiftquant.h"

namespace sq {

// record a message for shiftquant_last_error() and return `status`
int fail(int status, const char* fmt, ...);

inline int cuda_fail(cudaError_t err, const char* what) {
  return fail(SQ_ECUDA, "%s failed: %s", what, cudaGetErrorString(err));
}

inline int q_of_bits(int bits) { return (1 << (bits - 1)) - 1; }

inline bool bits_ok(int bits) { return bits >= 2 && bits <= 8; }
inline bool groups_ok(int g) { return g >= 1 && g <= 8; }

// FP8 E4M3 represents every integer up to 16 and every 4-significant-bit integer up to
// 448, so it holds q (|q| <= 15) and the shifted weight codes q 2^(G-1) when those stay
// below 448; otherwise BF16 (8 significant bits) holds q 2^(G-1) for all bits <= 8.
inline int code_type(int bits, int groups) {
  const int Q = q_of_bits(bits);
  return (Q <= 15 && (Q << (groups - 1)) <= 448) ? SQ_CODE_E4M3 : SQ_CODE_BF16;
}

inline int code_bytes(int type) { return type == SQ_CODE_E4M3 ? 1 : 2; }

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// SMs of the current device (its index to *dev_out unless null), -1 without one
int device_sms(int* dev_out);

inline cudaStream_t as_stream(void* s) { return static_cast<cudaStream_t>(s); }

// ------------------------------------------------------------ one layer step's parts
// device memory a launch wants zeroed before it (16-byte aligned, a multiple of 16 bytes)
struct ZeroRegion {
  void* p;
  size_t bytes;
};

// The quantizer's argument checks of a layer step (non-empty, required pointers checked).
int check_layer_quant(const sq_layer_step* L);
// whether the passes of quantize_layer can index the layer's tiles
bool layer_quant_fits(const sq_layer_step* L);
// The quantizer passes of a checked layer step -- zeroed accumulators, ranges, codes: three
// launches, five where the codes of a large layer are three -- and the zero regions cleared.
// words: 256 bytes of device memory, of which the first 64 are left zero and the rest is the
// passes' own.
int quantize_layer(const sq_layer_step* L, uint64_t seed, unsigned* words, const ZeroRegion* zero, int nzero,
                   cudaStream_t s);

// The GEMM launch of a layer step: planned (checks included) into `plan`, then issued on the
// stream once the operands' launches are.  zero receives the regions (at most 3) that must be
// zeroed before, besides the counter word at the start of the workspace.
struct alignas(64) LayerPlan {
  char bytes[4096];
};
int plan_layer_gemms(const sq_layer_gemms* args, void* workspace, size_t workspace_bytes, int32_t* dev_status,
                     LayerPlan* plan, ZeroRegion* zero, int* nzero);
int issue_layer_gemms(const LayerPlan* plan, cudaStream_t s);

// Launch with programmatic stream serialization: the kernel may begin launching while the
// preceding kernel of the stream finishes, and waits for it (griddep_wait) before reading
// anything.
template <typename... Params, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(Params...), dim3 grid, dim3 block, cudaStream_t s,
                              Args... args) {
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace sq
