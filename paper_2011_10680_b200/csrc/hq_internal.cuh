// Internal declarations shared by the translation units of libhq.so (CUDA side only).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/hq.h"

// Device-side status word values (written by a kernel that gave up a bounded wait).
enum : uint32_t {
  HQ_DEV_OK = 0,
  HQ_DEV_TIMEOUT_PRODUCER = 1,   // TMA producer waited too long for a free stage
  HQ_DEV_TIMEOUT_MMA = 2,        // MMA issuer waited too long for operands or a free accumulator
  HQ_DEV_TIMEOUT_EPILOGUE = 3,   // epilogue waited too long for a finished accumulator
  HQ_DEV_TIMEOUT_DRAIN = 4,      // teardown waited too long for work in flight
  HQ_DEV_TIMEOUT_ELTWISE = 5     // a streaming kernel waited too long for a staged chunk or a free stage
};

struct hq_handle {
  int32_t device;
  int32_t conv_path;          // see hq_set_conv_path
  int32_t sm_count;
  uint32_t* dev_status;       // one word in device memory, sticky until hq_sync
  void* workspace;            // scratch owned by the handle (grown on demand, never inside a capture)
  size_t workspace_bytes;
  void* narrow_pairs;         // 2 x kNarrowChannels x 16 bytes: narrow pairs of a single element-wise call's two operands
  int32_t tile_order;         // tensor-core convolutions walk their pixel tiles 0: first to last, 1: last to first
};
constexpr int kNarrowChannels = 4096;
constexpr long long kIm2colMinTensorBytes = 128 * 1024;   // smaller activation tensors are not fetched in im2col mode

// ------------------------------------------------------------------------------------------
// Dyadic arithmetic (Eq. 4): dn(q, b, c) = (q*b + 2^(c-1)) >> c, 64-bit product, arithmetic shift.
// ------------------------------------------------------------------------------------------
// a * b + c as one multiply-add.  Spelled as a product and a sum, which the assembler joins; the fused PTX form (mad.wide) comes
// out as two multiplies and an add (product, shift by register and pack in a loop: 6.2 against 4.7 cycles per 32 values and
// scheduler), and plain C++ can become a full 64 x 64-bit multiply when the sign extension of `b` is hoisted out of a loop.
__device__ __forceinline__ long long hq_mad_wide(int a, int b, long long c) {
  long long d;
  asm("{\n\t.reg .s64 m;\n\tmul.wide.s32 m, %1, %2;\n\tadd.s64 %0, m, %3;\n\t}" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}
__device__ __forceinline__ long long hq_dn(int q, int b, int c) { return hq_mad_wide(q, b, 1LL << (c - 1)) >> c; }

// Byte permute with the full PTX selector: bit 3 of a selector nibble replicates the selected byte's sign bit over the
// target byte.  (The __byte_perm intrinsic keeps three bits per nibble and cannot sign-extend.)
__device__ __forceinline__ unsigned hq_prmt(unsigned a, unsigned b, unsigned sel) {
  unsigned d;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
  return d;
}

// Programmatic dependent launch of the kernels around the convolutions: the grid may be set up while the previous kernel
// of the stream still runs, and lets the next one do the same; nothing the previous kernel wrote is read before this.
// The wait comes first: a convolution behind this kernel fetches its weights without waiting, and whatever an earlier
// launch wrote into them is then complete.
// (A chain of small launches otherwise pays the full launch latency at every one of them.)
__device__ __forceinline__ void hq_pdl_entry() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <class... Params, class... Args>
cudaError_t hq_launch_pdl_if(bool overlap, void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s; cfg.attrs = attr; cfg.numAttrs = overlap ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, Params(args)...);
}
template <class... Params, class... Args>
cudaError_t hq_launch_pdl(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args... args) {
  return hq_launch_pdl_if(true, kernel, grid, block, smem, s, args...);
}

// Tensors of at least this many values: launches of the kernels that run between two convolutions are not overlapped.  The
// convolutions take every SM then and the early blocks only get in their way (ResNet-50, 256 images: 2.098 ms with the
// first layer's two helpers overlapped, 2.088 without; with the INT32 stream, 64 images: 3.00 against 2.93 ms).
constexpr long long kOverlapValues = 1ll << 23;

// Element access for dense tensors with 4, 8 or 32 bits per element (even element = low nibble).
__device__ __forceinline__ int hq_load_elem(const void* base, long long idx, int bits, int is_signed) {
  if (bits == 32) return ((const int*)base)[idx];
  if (bits == 8) return is_signed ? (int)((const signed char*)base)[idx] : (int)((const unsigned char*)base)[idx];
  const unsigned byte = ((const unsigned char*)base)[idx >> 1];
  int v = (idx & 1) ? (int)(byte >> 4) : (int)(byte & 0xF);
  if (is_signed && (v & 8)) v -= 16;
  return v;
}

__device__ __forceinline__ int hq_clamp_ll(long long y, int relu, int qmin, int qmax) {
  if (relu && y < 0) y = 0;
  if (y < (long long)qmin) y = qmin;
  if (y > (long long)qmax) y = qmax;
  return (int)y;
}

// What may be fused behind a convolution whose raw INT32 result feeds the residual add of Fig. 2 (an INT32 stream) and,
// through it, the requantization of the next block.  The add's main pair, residual, ReLU, clamp and INT32 result are the
// b / c / res / relu / qmin / qmax / out fields of ConvArgs (out NULL: nobody reads the stream itself).
struct WideArgs {
  void* q;                            // the stream requantized to one byte per value, or NULL
  const int32_t* qb; const int32_t* qc;
  int32_t q_relu, q_qmin, q_qmax;
};

// Launchers implemented in the other translation units.  All return a cudaError_t from the launch.
struct ConvArgs {
  const void* in; int32_t n, h, w, cin, in_bits, in_signed;
  const void* wgt; int32_t cout, kh, kw, stride, pad;
  const int32_t* bias; const int32_t* b; const int32_t* c;
  const void* res; int32_t res_bits, res_signed; const int32_t* rb; const int32_t* rc;
  int32_t relu, qmin, qmax;
  void* out; int32_t ho, wo, out_bits, out_signed;
  // internal (zero for calls that come straight from the ABI):
  const void* res_narrow;    // per-channel narrow residual pairs prepared by hq_launch_residual_narrow, or NULL
  int32_t res_narrow_fresh;  // nonzero: the pairs come from the launch just before on the same stream (the kernel waits for it)
  const void* wgt_widened;   // weights as the lowered form wants them, prepared once by a network, or NULL: 4-bit weights widened
                             // to one byte per value; for the first-layer form the virtual-channel weights and constants
  const WideArgs* wide;      // non-NULL: the convolution ends in the INT32 residual add (see WideArgs)
  int32_t pairs;             // nonzero: the pixel-pair form (hq_conv_pairs_applies): "pixels" are pairs, "channels" those of both; weights and constants are the layer's own
  int32_t in_slack;          // nonzero: a layer inside a network; the allocation behind `in` goes on for at least kIm2colMinTensorBytes + one image
  int32_t params_late;       // nonzero: weights, bias or pairs may be written by the launch just before: nothing is read ahead of its end
  int32_t pad_after_delta;   // padding after the last row/column minus `pad`
  // byte pitches of the activation tensor along W, H and N when it is not dense (0: dense NHWC).  A W pitch
  // below cin bytes makes neighbouring "pixels" overlap: a pixel is then a window of adjacent stored pixels.
  long long pitch_w, pitch_h, pitch_n;
};

struct EltArgs {
  const void* main_t; int32_t main_bits, main_signed; const int32_t* mb; const int32_t* mc;
  const void* res; int32_t res_bits, res_signed; const int32_t* rb; const int32_t* rc;
  long long pixels; int32_t ch; int32_t relu, qmin, qmax;
  void* out; int32_t out_bits;
  // optional narrow pairs {m, a, s, valid} per channel for 8-bit operands (see hq_launch_residual_narrow), or NULL
  const void* m_narrow; const void* r_narrow;
  int32_t narrow_fresh;      // nonzero: they are written by the launch just before (residual_narrow_kernel)
  int32_t overlap;           // set by the launcher: this launch overlaps its neighbours (hq_pdl_entry)
  uint32_t* status;          // the handle's device status word (bounded waits report here), or NULL
};

// Bytes of K per stage of the tensor-core convolutions: the shortest power of two up to 128 that holds a tap's channels, else
// 128 with the last block reaching past them (the copies fill zeros, the MMA steps beyond the channels are left out, and what
// the weight box picks up of the next tap meets nothing).  An SM takes in one operand row per two cycles whatever its length, so
// the rows have to be long: 3x3 over 96 channels in 32-byte rows 82 us, over 192 in 64-byte rows 42 us (35x35 and 17x17, 256
// images); in 128-byte rows 58 and 36 us.  5x5 over 48 channels as a patch matrix (three launches) 161 us, fetched directly 135 us.
inline int hq_conv_bkb(int cin) { return cin > 64 ? 128 : cin > 32 ? 64 : 32; }

cudaError_t hq_launch_conv_cuda_core(const ConvArgs& a, cudaStream_t s);
bool hq_conv_tc_init();
bool hq_conv_tc_supported(const ConvArgs& a);
// True for a layer the direct kernel declines although its shape is supported: it would fetch a tensor below
// 128 KiB through an im2col-mode map.  Such a layer runs in its lowered (patch-matrix) form.
bool hq_conv_tc_small_im2col(const ConvArgs& a);
bool hq_conv_tc_declines(const ConvArgs& a);      // ... or whose patch matrix is cheaper than its short rows
// The layer can end in the INT32 residual add (ConvArgs::wide): there is no other kernel for that, so the launcher takes
// exactly these.
bool hq_conv_wide_applies(const ConvArgs& a, int sm_count);
// Tensor-core path; returns HQ_OK, HQ_ERR_UNSUPPORTED (nothing was launched) or HQ_ERR_CUDA.
hq_status hq_launch_conv_tc(hq_handle* h, const ConvArgs& a, cudaStream_t s);
hq_status hq_conv_tc_plan(const ConvArgs& a, int sm_count, hq_conv_plan* out);     // what it would launch; host arithmetic only
// One tile per CTA, reduction split over a cluster: small problems (conv_small.cu).  Same status convention.
bool hq_conv_small_init();
bool hq_conv_small_supported(const ConvArgs& a, int sm_count);
bool hq_conv_small_wanted(const ConvArgs& a, int sm_count);    // the automatic path's choice
hq_status hq_launch_conv_small(hq_handle* h, const ConvArgs& a, cudaStream_t s);
// Fills `out` (channels x 16 bytes) with the narrow residual pairs of an 8-bit residual branch.
cudaError_t hq_launch_residual_narrow(const int32_t* rb, const int32_t* rc, int res_signed, int channels, void* out,
                                      cudaStream_t s);
// The same for the two operands of an element-wise call in one launch (`out1` NULL: first operand only).
cudaError_t hq_launch_residual_narrow2(const int32_t* b0, const int32_t* c0, int signed0, void* out0,
                                       const int32_t* b1, const int32_t* c1, int signed1, void* out1, int channels,
                                       cudaStream_t s);
// Lowered path for thin first layers: patch matrix + padded weights in scratch, then the tensor-core kernel.
bool hq_conv_lowering_applies(const ConvArgs& a);
size_t hq_conv_lowering_bytes(const ConvArgs& a);
hq_status hq_launch_conv_lowered(hq_handle* h, const ConvArgs& a, void* scratch, cudaStream_t s);
// 7x7 / stride 2 / 3-channel first layer as a 4x4 stride-1 conv over a space-to-depth copy of the image.
bool hq_conv_s2d_applies(const ConvArgs& a);
size_t hq_conv_s2d_bytes(const ConvArgs& a);
hq_status hq_launch_conv_s2d(hq_handle* h, const ConvArgs& a, void* scratch, cudaStream_t s);
size_t hq_conv_s2d_prepared_bytes(const ConvArgs& a);
cudaError_t hq_prepare_conv_s2d(const ConvArgs& a, void* buf, cudaStream_t s);
// 3x3 / stride 1 layers over 64 channels, 64 to 64, as convolutions over pixel pairs (inside networks).
bool hq_conv_pairs_applies(const ConvArgs& a, int sm_count);
hq_status hq_launch_conv_pairs(hq_handle* h, const ConvArgs& a, cudaStream_t s);
// 4-bit operands: widen to bytes in scratch, then the tensor-core kernel.
bool hq_conv_widen4_applies(const ConvArgs& a);
size_t hq_conv_widen4_bytes(const ConvArgs& a);
hq_status hq_launch_conv_widen4(hq_handle* h, const ConvArgs& a, void* scratch, cudaStream_t s);
// Widen packed 4-bit weights (cout*kh*kw*cin values, a multiple of 16) to bytes, once, for ConvArgs::wgt_widened.
cudaError_t hq_launch_widen_weights(const void* wgt, long long values, void* out, int sm_count, cudaStream_t s);
// Bytes holding 4-bit values (one per byte) -> packed 4-bit tensor; `values` a multiple of 8.
cudaError_t hq_launch_expire_wait(uint32_t* status, int budget_ms, cudaStream_t s);
cudaError_t hq_launch_pack4(const void* in, long long values, void* out, int sm_count, cudaStream_t s);
// Grow the handle's scratch buffer (not allowed while `s` is capturing).
hq_status hq_reserve_workspace(hq_handle* h, size_t bytes, cudaStream_t s);
// hq_concat_requant as a network runs it: `skip` is a branch written by somebody else (-1: none); `narrow` the branches' narrow
// pairs, out->c x 16 bytes (NULL: a large call works them out itself), only computed with `prepare`.
struct ConcatPlan { int32_t skip; void* narrow; bool prepare; };
hq_status hq_concat_requant_planned(hq_handle* h, int32_t n_branches, const hq_tensor* branches, const hq_dyadic* rescale, int32_t relu,
                                    int32_t qmin, int32_t qmax, hq_tensor* out, void* stream, const ConcatPlan& plan);
// 3x3 / stride 1 / pad 1 window sums of an 8-bit tensor rescaled by `r` straight into channels [ch_off, ch_off + in->c) of an
// 8-bit concatenation (sumpool.cu); false: the shapes do not allow it.
bool hq_sumpool_concat_applies(const hq_tensor& in, const hq_tensor& out, int32_t ch_off);
hq_status hq_launch_sumpool_concat(hq_handle* h, const hq_tensor& in, hq_dyadic r, int32_t relu, int32_t qmin, int32_t qmax,
                                   const hq_tensor& out, int32_t ch_off, cudaStream_t s);
cudaError_t hq_launch_residual_add(const EltArgs& a, int sm_count, cudaStream_t s);
cudaError_t hq_launch_avgpool(const void* in, int n, int h, int w, int ch, int in_bits, int in_signed,
                              const int32_t* b, const int32_t* c, int qmin, int qmax,
                              void* out, int out_bits, int sm_count, cudaStream_t s);
cudaError_t hq_launch_maxpool(const void* in, int n, int h, int w, int ch, int bits, int is_signed,
                              int k, int stride, int pad, void* out, int ho, int wo, cudaStream_t s);
