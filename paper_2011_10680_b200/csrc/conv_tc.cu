// Tensor-core convolution for sm_100a: implicit GEMM
//     D[ch][px] = sum_k W[ch][k] * X[px][k]
// with ch = output channel, px = output pixel (n, oh, ow) in NHWC order and k = (kh, kw, cin): the
// contraction of Eq. 3 on tcgen05.mma kind::i8 (s8 weights x u8/s8 activations, INT32 accumulators in
// tensor memory), fused with the integer epilogue: INT32 bias (Appendix D), dyadic multiply-shift
// (Eq. 4), dyadically rescaled residual branch (Section 3.3), ReLU, clamp, pack.
//
// Orientation.  The output channels sit on the M side of the MMA, i.e. on the 128 lanes of tensor
// memory, and the pixels on the N side (columns).  An epilogue thread therefore owns ONE channel:
// its dyadic pair, bias and residual pair live in registers for the whole kernel, no per-element
// constant fetch is needed, and the 32 lanes of a warp hold 32 consecutive channels of the same
// pixel, which is a contiguous 32-byte run of the NHWC output.
//
// One persistent CTA per SM, twelve warps (six in the two-CTAs-per-SM shape):
//   warp 0      TMA producer.  X tile = PT consecutive output pixels x BK bytes of one filter tap,
//               fetched by an im2col-mode tensor map straight from the NHWC activation tensor (the
//               hardware walks pixels across rows and images, applies the stride and zero-fills the
//               padding; zero is the right padding value because activations have zero point 0), or by
//               a plain tiled map when the conv is 1x1 / stride 1.  W tile = 128 output channels x BK
//               bytes of the [cout][kh*kw*cin] weight matrix.  When a residual is fused, its
//               [PT][128] tile of the stored 8-bit tensor is prefetched as well.
//   warps 1-3   MMA issuers (one lane each; a single issuer for layers whose weights stream from L2).
//               BK/32 instructions of shape 128 x PT x 32 per stage; two (PT = 256) or four
//               (PT <= 128) accumulator buffers in tensor memory, so the MMAs of the next tiles run
//               while the epilogue works on the current ones.  3x3 / stride 1 layers with resident
//               weights use the strip form: one padded input patch per cin chunk, read by all nine
//               taps as row offsets (see the issuer loop).
//   warps 4-11  epilogue.  Warp (q, half) reads lanes 32q..32q+31 (tcgen05.ld 32x32b) of one half
//               of the tile's pixel columns, applies the integer epilogue in registers and writes
//               bytes to a private staging box that leaves through its own TMA store; no CTA-wide
//               barrier per tile.  The loop is software-pipelined: the accumulator buffer goes back
//               to the MMA issuer as soon as its last chunk has been read, and the first chunk of
//               the next tile is requested from tensor memory before the current tile's staging
//               writes and store hand-over, whose latency it hides.
// The CTA keeps one channel tile for its whole life (grid = multiple of the channel tiles).
// Every wait on an mbarrier is bounded: after the budget the waiter records a code in the
// handle's status word, raises a CTA-wide abort flag and every role leaves its loop, drains what
// it has in flight (again bounded), and the CTA frees its tensor memory and returns.
#include <type_traits>

#include "tc_common.cuh"

namespace {

constexpr int kMaxStages = 8;
// Dynamic shared memory of a one-CTA-per-SM launch: 224 KiB for the pipeline's pieces + 1 KiB of alignment slack, inside
// the 226 KiB the kernels ask for (227 KiB per block is the limit, the control block is static).
constexpr int kSmemBudget = 224 * 1024;
constexpr int kSmemAttr = 226 * 1024;
constexpr int kMaxAccBufs = 4;                                 // accumulator buffers: 4 x 128 or 2 x 256 columns
constexpr int kMaxResBufs = 8;                                 // residual / output tiles in shared memory
// Launch shapes of the same kernel:
//   solo  8 epilogue warps, one CTA per SM, up to 512 tensor-memory columns, up to 224 KiB of shared memory;
//   pair  4 epilogue warps, two CTAs per SM with 256 columns and at most 110 KiB each.  Layers with a short
//         reduction are bound by the latency of the hand-over chain between the MMA issuer and the epilogue
//         (barrier, fences, MMA, commit), not by any throughput; two independent CTAs hide each other's chain.
//   frag  16 epilogue warps in two groups on alternate tiles, two issuers and a store warp, one CTA per SM, 128-pixel tiles
//         in four accumulators: fused 8-bit residuals with a short reduction, and 8-bit results without a residual whose
//         weights stay resident.  The epilogue works on 16 x 8 fragments, reads the residual with transposing matrix loads and
//         writes over it with transposing matrix stores; the store warp fetches the residual tiles.
//   wide  16 epilogue warps on boxes of 16 pixels: INT32 results, raw or through the residual add (see epilogue_loop_wide).
//   duo   the solo roles in clusters of two CTAs that share every MMA (cta_group::2): long reductions whose weights
//         stream; each CTA fetches its own weight rows and half of the pixel rows.
constexpr int kSoloEpilogueWarps = 8;
constexpr int kPairEpilogueWarps = 4;
constexpr int kFragWarps = 16, kFragIssuers = 2, kFragGroups = 2, kFragAccs = 4;   // the frag shape: epilogue warps, in two groups; issuers; accumulator buffers
constexpr int kSoloIssuerWarps = 3;     // 1 + 3 + 8 warps = 384 threads: 168 registers per thread remain
constexpr int kPairIssuerWarps = 1;

struct TcParams {
  int32_t P, C;          // output pixels (n*ho*wo) and output channels
  int32_t howo, wo, stride, pad, kw;
  int32_t cin;
  int32_t cchunks;       // K blocks per filter tap; the last one may reach past the channels (the copies fill zeros there)
  int32_t tail_steps;    // 32-byte MMA steps of a tap's last K block
  int32_t bkb;           // bytes of K per stage (32, 64 or 128) = swizzle span
  int32_t k_blocks;      // kh * kw * cchunks
  int32_t pt;            // pixel tile = MMA N: 64, 128 or 256
  int32_t p_tiles, c_tiles, stages;
  int32_t rev;           // 1: a CTA's t-th pixel tile is tile p_tiles - 1 - t: the layer walks its tensors from the end, so
                         //    that it reads first what the kernel before it wrote last (still in the L2)
  int32_t wres;          // 1: the CTA's whole weight slab [k_blocks][128][bkb] is loaded once and stays in shared memory
  uint32_t wres_off;     // its offset from the 1024-aligned dynamic base
  int32_t fold;          // 1: at most 64 output channels: W rows loaded twice, lane quarters 2-3 share the pixel columns
  int32_t halves;        // warps that share a lane quarter's pixel columns: 2, 4 with INT32 boxes, 1 for the 64-pixel tile (the others idle)
  int32_t lg_rbufs;      // log2 of the residual-tile buffer count (<= lg_bufs; 0 when a long reduction leaves no room)
  int32_t frag, deal;    // 1: the launch shape of epilogue_loop_frag; its two issuers take alternate K blocks (see frag_issue)
  int32_t acc_bits;      // |accumulator| < 2^acc_bits for every 8-bit operand pair: ceil(log2(K * 255 * 128 + 1))
  int32_t acc_stride;    // tensor-memory columns between accumulator buffers
  int32_t duo;           // 1: two CTAs of a cluster (adjacent SMs) share every MMA: 256 channels x 256 pixels per pair
  int32_t ni;            // MMA issuer warps in use: min(issuer warps of the launch shape, k_blocks)
  int32_t lg_bufs;       // log2 of the accumulator / residual buffer count: tile t of a CTA uses buffer t mod 2^lg_bufs
  int32_t x_signed;      // activations signed?
  int32_t x_tiled;       // 1: X is a dense [P][cin] matrix (1x1, stride 1, no padding) fetched by a tiled map
  // Strip mode (3x3, stride 1, pad 1): a tile is `rows` output rows of one image, laid out with a power-of-two
  // pitch of 2^lg_wp positions (columns >= wo are scratch); one padded input patch per cin chunk feeds all nine taps.
  int32_t strip;         // 1: strip mode
  int32_t lg_wp, rows;   // log2 of the position pitch; output rows per tile (pt = rows << lg_wp)
  int32_t tpi;           // tiles per image = ceil(ho / rows)
  int32_t ho;            // output (= input) height
  int32_t pairs;         // 1: strip mode over pixel pairs (lowering.cu): twelve blocks (filter row, pixel of four) of 64 bytes
  int32_t w_blocks;      // K blocks of the resident weight slab
  int32_t npatch;        // patch buffers (2 or 3)
  uint32_t patch_bytes, patch_off;   // bytes of one patch [(rows+3) << lg_wp][bkb]; offset from the 1024-aligned base
  uint32_t tmem_cols;
  // epilogue
  int32_t staged_out;    // 1: bytes leave through per-warp staging boxes and TMA stores
  int32_t staged_res;    // 1: the 8-bit residual tile arrives through a TMA load
  int32_t sat_pack;      // 1: clamp bounds equal the 8-bit output type's range (a saturating convert does the clamp)
  int32_t out_signed;
  uint32_t out_stage_off, res_stage_off;   // offsets from the 1024-aligned dynamic base
  const int32_t* bias; const int32_t* b; const int32_t* c;
  const void* res; int32_t res_bits, res_signed; const int32_t* rb; const int32_t* rc;
  const int4* res_narrow;   // optional per-channel {m, a, s, valid} from residual_narrow_kernel
  int32_t narrow_fresh;     // 1: the pairs are written by the kernel launched just before this one
  int32_t params_late;      // 1: so may be weights, bias or pairs (see ConvArgs)
  int32_t relu, qmin, qmax;
  void* out; int32_t out_bits;
  void* q_out; const int32_t* qb; const int32_t* qc; int32_t q_lo, q_hi, q_sat;   // wide: the stream requantized to bytes, or NULL
  uint32_t* status;
};

struct SharedCtl {
  unsigned long long full[kMaxStages];
  unsigned long long empty[kMaxStages];
  unsigned long long tfull[kMaxAccBufs];
  unsigned long long tempty[kMaxAccBufs];
  unsigned long long tstart[kMaxAccBufs];   // the tile's first (overwriting) MMA has been issued
  unsigned long long rfull[kMaxResBufs];
  unsigned long long rempty[kMaxResBufs];
  unsigned long long ofull[kMaxResBufs];    // frag: every epilogue warp of the tile's group has written its pieces of the output tile
  unsigned long long drain;
  unsigned long long wfull;              // resident weight slab landed
  unsigned long long pfull[3], pempty[3];  // strip mode: input patches
  unsigned long long wbox[16][3];         // INT32 results: residual boxes of the epilogue warps (kWideSlots each)
  uint32_t tmem_base;
  volatile uint32_t abort_flag;
};

// Pixel tile behind position `t` of the tile order (see TcParams::rev).
__device__ __forceinline__ int tile_at(const TcParams& p, int t) { return p.rev ? p.p_tiles - 1 - t : t; }

// The finished staging box of one warp leaves for global memory.  Dense tiles: one [columns][32 B] box at pixel
// `p_tile * pt + col0`.  Strip tiles: one box per 32 positions (a row, half a row or two rows of the pitch-2^lg_wp
// raster); columns at or beyond the image width and rows at or beyond its height fall outside the tensor map
// and are clipped by the copy.
__device__ __forceinline__ void store_warp_box(const TcParams& p, const CUtensorMap* map_out, uint32_t my_stage, int chx,
                                               int p_tile, int col0, int px_per_warp) {
  if (!p.strip) {
    const int p_base = p_tile * p.pt + col0;
    if (p_base < p.P) { tma_store_2d(map_out, my_stage, chx, p_base); tma_store_commit(); }
    return;
  }
  const int img = p_tile / p.tpi, y0 = (p_tile - img * p.tpi) * p.rows;
  bool any = false;
  for (int c = 0; c < (px_per_warp >> 5); ++c) {
    const int j0 = col0 + 32 * c;
    const int y = y0 + (j0 >> p.lg_wp), x = j0 & ((1 << p.lg_wp) - 1);
    if (y < p.ho && x < p.wo) { tma_store_4d(map_out, my_stage + (uint32_t)c * 1024u, chx, x, y, img); any = true; }
  }
  if (any) tma_store_commit();
}

// An epilogue warp hands its part of accumulator buffer `as` back.  The barrier that counts is the one the MMA issuer
// waits on: this CTA's, or the leading CTA's when two CTAs share the MMAs.
__device__ __forceinline__ void release_accumulator(const TcParams& p, SharedCtl& ctl, uint32_t as) {
  const uint32_t bar = smem_u32(&ctl.tempty[as]);
  if (p.duo) mbar_arrive_cluster(in_cta(bar, 0)); else mbar_arrive(bar);
}

// Everything an epilogue warp needs, gathered once so the tile loops can live in their own functions.
struct EpiCtx {
  const TcParams* p; SharedCtl* ctl; const CUtensorMap* map_out;
  uint8_t* smem_raw; uint32_t raw, out_stage, res_stage, res_tile_bytes, tmem_base;
  int warp, lane, q, cq, ew, half, col0, px_per_warp, ch, c_tile, p_tile0, p_step, lo, hi;
  bool ch_live, warp_live;
};

// Lean tile loop for the common case: 8-bit output through the staging box, 32-bit fast arithmetic,
// clamp by saturating convert or by min/max, optional 8-bit residual from the prefetched tile.
// Software-pipelined across chunks and tiles: while one 32-pixel accumulator chunk is processed, the
// next one (of this tile, or the first of the group's next tile) streams from tensor memory into the
// other register set; the accumulator buffer is handed back as soon as its last chunk has been read,
// the residual tile as soon as its last bytes have been used, both before the tile's store is issued.
template <bool RES, bool RSIGNED, bool SAT, bool OSIGNED, int SMALL, bool RN, bool OUT4 = false>
__device__ __forceinline__ void epilogue_loop_fast8(const EpiCtx& e_in, const ChanConst& k_in) {
  // Private copies: the caller's objects live in local memory (their address is passed to the general
  // loop), so every asm statement with a memory clobber would force their fields to be re-read.
  const EpiCtx e = e_in;
  ChanConst k_own = k_in;
  if (SMALL == 2) k_own.r0 <<= k_own.pre;          // the pre-shift form of requant_fast
  const ChanConst k = k_own;
  const TcParams& p = *e.p;
  SharedCtl& ctl = *e.ctl;
  const int lane = e.lane, q = e.q, cq = e.cq, col0 = e.col0, px_per_warp = e.px_per_warp;
  const uint32_t my_stage = e.out_stage + (uint32_t)e.ew * (uint32_t)(px_per_warp * 32);
  uint8_t* const my_stage_ptr = e.smem_raw + (my_stage - e.raw);
  const uint8_t* const res_stage_ptr = e.smem_raw + (e.res_stage - e.raw);
  const int nchunks = px_per_warp >> 5;           // 2 or 4
  const uint32_t bmask = (1u << p.lg_bufs) - 1u, rmask = (1u << p.lg_rbufs) - 1u;
  const int tile_step = e.p_step;
  int p_tile = e.p_tile0;
  if (p_tile >= p.p_tiles) return;
  uint32_t tcount = 0;
  uint32_t as = 0, aph = 0;
  const uint32_t t_warp = e.tmem_base + ((uint32_t)(q * 32) << 16) + col0;

  auto wait_bar = [&](unsigned long long* bar, uint32_t ph) -> bool {
    uint32_t w = 1;
    if (lane == 0) w = mbar_wait(smem_u32(bar), ph, &ctl, p.status, HQ_DEV_TIMEOUT_EPILOGUE) ? 1u : 0u;
    return __shfl_sync(0xffffffffu, w, 0) != 0;
  };
  auto chunk = [&](const int (&v)[32], const uint8_t* res_tile, int c) {
    if (!e.warp_live) return;
    int y[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      const int r = !RES ? 0 : RSIGNED ? (int)(signed char)res_tile[(c * 32 + j) * kTileC] : (int)res_tile[(c * 32 + j) * kTileC];
      const int s = requant_fast<RES, RSIGNED, SMALL, RN>(v[j], r, k);
      y[j] = SAT ? (OSIGNED ? sat_s8(s) : sat_u8(s)) : min(max(s, e.lo), e.hi);
    }
    if (!OUT4) {
#pragma unroll
      for (int j = 0; j < 32; ++j) my_stage_ptr[(c * 32 + j) * 32 + lane] = (uint8_t)y[j];
    } else {
      // Unsigned 4-bit output (0 <= y <= 15 after the clamp): a byte holds the channel pair of two neighbouring
      // lanes.  Each lane packs its 32 pixels into four words of eight nibbles, the pair exchanges the words
      // (4 shuffles instead of 32), both interleave them into bytes, and the even lane stores pixels 0-3 of every
      // eight, the odd lane pixels 4-7: rows of 16 bytes per pixel in the staging box.
      const bool odd = lane & 1;
      const unsigned sel = odd ? 0x7362u : 0x5140u;
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        unsigned mine = (unsigned)y[8 * w + 7];
#pragma unroll
        for (int i = 6; i >= 0; --i) mine = mine * 16u + (unsigned)y[8 * w + i];
        const unsigned other = __shfl_xor_sync(0xffffffffu, mine, 1);
        const unsigned a = odd ? other : mine, b = odd ? mine : other;        // even channel, odd channel
        const unsigned t = (a & 0x0F0F0F0Fu) | ((b << 4) & 0xF0F0F0F0u);        // pixels 0, 2, 4, 6
        const unsigned u = ((a >> 4) & 0x0F0F0F0Fu) | (b & 0xF0F0F0F0u);        // pixels 1, 3, 5, 7
        const unsigned four = __byte_perm(t, u, sel);                          // pixels 0-3 (even lane) or 4-7 (odd lane)
        const int px = c * 32 + 8 * w + (odd ? 4 : 0);
#pragma unroll
        for (int i = 0; i < 4; ++i) my_stage_ptr[(px + i) * 16 + (lane >> 1)] = (uint8_t)(four >> (8 * i));
      }
    }
  };

  int va[32], vb[32];
  bool ok = wait_bar(&ctl.tfull[as], aph);
  if (!ok) return;
  tc_fence_after();
  tmem_ld32_issue(t_warp + as * p.pt, va);
  bool pending = true;                            // a tensor-memory load into va is in flight
  while (true) {
    const uint32_t rs = tcount & rmask, rph = (tcount >> p.lg_rbufs) & 1u;       // residual buffer and its phase
    if (RES && !wait_bar(&ctl.rfull[rs], rph)) break;
    const uint8_t* const res_tile = res_stage_ptr + rs * e.res_tile_bytes + (uint32_t)col0 * kTileC + cq * 32 + lane;
    const uint32_t t_addr = t_warp + as * p.pt;
    const bool has_next = p_tile + tile_step < p.p_tiles;
    const uint32_t nas = (tcount + 1u) & bmask, naph = ((tcount + 1u) >> p.lg_bufs) & 1u;

    for (int c = 0; c < nchunks; c += 2) {
      // ---- chunk c (registers va), while chunk c+1 streams into vb
      tmem_ld_wait();
      tie(va);
      tmem_ld32_issue(t_addr + (c + 1) * 32, vb);
      if (c == 0) {                               // the previous tile's store must have read the staging box
        if (lane == 0) tma_store_wait_read0();
        __syncwarp();
      }
      chunk(va, res_tile, c);
      // ---- chunk c+1 (registers vb), while the next chunk streams into va
      tmem_ld_wait();
      tie(vb);
      pending = false;
      if (c + 2 < nchunks) {
        tmem_ld32_issue(t_addr + (c + 2) * 32, va);
        pending = true;
      } else {
        // every lane has read its last accumulator columns of this tile: hand the buffer back
        tc_fence_before();
        __syncwarp();
        if (lane == 0) release_accumulator(p, ctl, as);
      }
      chunk(vb, res_tile, c + 1);
    }
    if (RES) {                                    // every lane has used its last residual bytes of this tile
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&ctl.rempty[rs]));
    }
    // Only now wait for the group's next tile: its copies may be queued behind the buffers released above.
    if (has_next) {
      ok = wait_bar(&ctl.tfull[nas], naph);
      if (ok) { tc_fence_after(); tmem_ld32_issue(t_warp + nas * p.pt, va); pending = true; }
    }
    fence_async_smem();                           // make this lane's box writes visible to the TMA engine
    __syncwarp();
    if (lane == 0 && e.warp_live) store_warp_box(p, e.map_out, my_stage, (e.c_tile * kTileC + cq * 32) >> (OUT4 ? 1 : 0), tile_at(p, p_tile), col0, px_per_warp);
    if (!has_next || !ok) break;
    p_tile += tile_step; ++tcount; as = nas; aph = naph;
  }
  if (pending) tmem_ld_wait();
  if (lane == 0) tma_store_wait_all();
}

// The shared per-channel constants, with the checked narrow residual pair of the channel where the loops use it.
__device__ __forceinline__ ChanConst chan_const_for(const TcParams& p, int ch, bool fast, bool narrow, bool pre = false) {
  ChanConst k = chan_const(p, ch, fast, pre);
  if (narrow) {
    const int4 nr = ch < p.C ? p.res_narrow[ch] : make_int4(0, 0, 0, 1);
    k.rb = nr.x; k.rh = nr.y; k.rsh = nr.z;
  }
  return k;
}

// Tile loop of the frag shape (sixteen epilogue warps, a store warp, 128-pixel tiles).
//
// Nothing moves byte by byte here.  A warp reads 16 accumulator lanes with 16x256b loads, which hand thread T the values of
// lanes t4, t4 + 8 for pixel pairs -- the fragment of a 16 x 8 matrix.  The weight rows lie on the lanes in the order of
// encode_paired_rows_map, so that the two lanes are neighbouring channels and a matrix element of 16 bits is the channel pair
// of one pixel: ldmatrix (transposing) delivers the residual tile [128 pixels][128 channels], as TMA left it with the 128-byte
// swizzle, in exactly the accumulator's fragments, and stmatrix writes the packed results over it in place, 16-byte row pieces
// of 32 pixels at a time.  The constants of a thread's two channels stay in registers.  Two groups of eight warps take
// alternate tiles, four accumulators of 128 columns let the MMAs run ahead.  Warps do not wait for each other: each arrives on
// the tile's `ofull` barrier when its pieces are written, and the store warp alone waits there, stores the [128][128] box and
// hands the buffer back.  Up to eight residual / output tiles circulate: their loads in flight cover the memory latency.
//
// What bounds it: instructions and their latency together.  All warps execute 10.2 warp instructions per 32 values (5.3 without a
// residual) in 52 % (46 %) of the issue slots, no unit is saturated, tensor pipe 5 %, DRAM 30 % (counters at 128 images); 1x1 64 -> 256 at
// 56x56, 256 images, L2 flushed, takes 97 us, with no arithmetic 82, with no memory traffic 95.  Twenty-four warps in three groups: no
// faster.  Inside ResNet-50 at 256 images, us a layer:
// 1x1 64 -> 256 at 56x56 / 128 -> 512 at 28x28 / 256 -> 1024 at 14x14 / 512 -> 2048 at 7x7 with residual 94 / 55 / 34 / 25, 64 -> 256 without 67.  The
// shape before this one - eight warps, the residual widened into tensor memory by an MMA with the identity matrix, two accumulators, one
// issuer, multiply-adds of three instructions - took 122 / 70 / 42 / 33 and, for the last, the solo shape 88; the issuer's own instruction
// latency (2.5 k cycles a tile) set its tile rate, whatever the epilogue did (sixteen warps or another matrix store: the same).
// GEN: 64-bit arithmetic for every shift 1..62 (a residual shift below 9).  SMALL: some channel of the warp has c < 32 (common
// with 4-bit operands, whose accumulators are small): funnel-shift or pre-shift form of Eq. 4.
template <bool RES, bool GEN, bool RSIGNED, bool SAT, bool OSIGNED, bool RN, int SMALL = 0>
__device__ __forceinline__ void epilogue_loop_frag(const EpiCtx& e_in) {
  const EpiCtx e = e_in;
  const TcParams& p = *e.p;
  SharedCtl& ctl = *e.ctl;
  const int lane = e.lane, q = e.q, hh = (e.ew >> 2) & 1, group = e.ew >> 3;
  const int t4 = lane >> 2;
  ChanConst k[2];                                   // channels 32 q + 16 hh + 2 t4 + r, on lanes 32 q + 16 hh + t4 + 8 r (see encode_paired_rows_map)
#pragma unroll
  for (int r = 0; r < 2; ++r) k[r] = chan_const_for(p, e.c_tile * kTileC + 32 * q + 16 * hh + 2 * t4 + r, !GEN, RN, SMALL == 2);
  const uint32_t rmask = (1u << p.lg_rbufs) - 1u;
  constexpr int units = 4;                          // 32 pixel columns per unit, 128-pixel tiles
  const uint32_t t_lane = e.tmem_base + ((uint32_t)(q * 32 + 16 * hh) << 16);
  // byte offset of this thread's 16-byte piece in a unit's 32 rows: row `lane`, chunk (2 q + hh) ^ (row % 8)
  const uint32_t row_off = (uint32_t)lane * 128u + ((uint32_t)((2 * q + hh) ^ (lane & 7)) << 4);
  auto wait_bar = [&](unsigned long long* bar, uint32_t ph) -> bool {
    uint32_t w = 1;
    if (lane == 0) w = mbar_wait(smem_u32(bar), ph, &ctl, p.status, HQ_DEV_TIMEOUT_EPILOGUE) ? 1u : 0u;
    return __shfl_sync(0xffffffffu, w, 0) != 0;
  };
  auto one = [&](int acc, unsigned word, int i, const ChanConst& c) -> int {
    const int r = !RES ? 0 : (int)hq_prmt(word, 0u, RSIGNED ? 0x8880u + 0x1111u * i : 0x4440u + i);
    if (GEN) {
      const long long y = (hq_mad_wide(acc, c.b, c.r0) >> c.sh) + (hq_mad_wide(r, c.rb, c.rr0) >> c.rsh);
      return hq_clamp_ll(y, p.relu, p.qmin, p.qmax);
    }
    const int y = requant_fast<RES, RSIGNED, SMALL, RN>(acc, r, c);
    return SAT ? y : min(max(y, e.lo), e.hi);
  };
  // one unit: 16 values per thread -> four words -> one transposing store of 32 pixel rows x 16 channel bytes
  auto unit = [&](const int (&v)[16], const unsigned (&r)[4], uint32_t at) {
    unsigned w[4];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      // bytes of a word: (pixel 2 q2, even channel), (2 q2, odd), (2 q2 + 1, even), (2 q2 + 1, odd)
      const int y0 = one(v[4 * g + 0], r[g], 0, k[0]), y1 = one(v[4 * g + 2], r[g], 1, k[1]);
      const int y2 = one(v[4 * g + 1], r[g], 2, k[0]), y3 = one(v[4 * g + 3], r[g], 3, k[1]);
      w[g] = sat_pack4<OSIGNED>(y0, y1, y2, y3);
    }
    if (e.warp_live) stmatrix_t_x4(at, w[0], w[1], w[2], w[3]);
  };

  int a0[16], a1[16];
  unsigned r0[4] = {0u, 0u, 0u, 0u}, r1[4] = {0u, 0u, 0u, 0u};
  uint32_t tcount = (uint32_t)group;
  for (int p_tile = e.p_tile0 + group * e.p_step; p_tile < p.p_tiles; p_tile += kFragGroups * e.p_step, tcount += kFragGroups) {
    const uint32_t as = tcount & (kFragAccs - 1), aph = (tcount / kFragAccs) & 1u;
    const uint32_t rs = tcount & rmask, rph = (tcount >> p.lg_rbufs) & 1u;
    const uint32_t at = e.res_stage + rs * e.res_tile_bytes + row_off;  // tile: [128 pixels][128 bytes], 128-byte swizzle
    if (!wait_bar(&ctl.tfull[as], aph)) break;
    if (!(RES ? wait_bar(&ctl.rfull[rs], rph) : wait_bar(&ctl.rempty[rs], rph ^ 1u))) break;
    tc_fence_after();
    const uint32_t t_addr = t_lane + as * kTileC;
    tmem_ld_frag16(t_addr, a0);
    if (RES) ldmatrix_t_x4(at, r0);
#pragma unroll 1                                    // (unrolled: 103 / 60 instead of 99 / 57 us on the first two layers above)
    for (int u = 0; u < units; u += 2) {
      tmem_ld_wait();
      tie(a0);
      tmem_ld_frag16(t_addr + 32 * (u + 1), a1);
      if (RES) ldmatrix_t_x4(at + (u + 1) * 4096u, r1);
      unit(a0, r0, at + u * 4096u);
      tmem_ld_wait();
      tie(a1);
      if (u + 2 < units) {
        tmem_ld_frag16(t_addr + 32 * (u + 2), a0);
        if (RES) ldmatrix_t_x4(at + (u + 2) * 4096u, r0);
      } else {
        // every lane has read its last columns of this tile: hand the accumulator buffer back
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&ctl.tempty[as]));
      }
      unit(a1, r1, at + (u + 1) * 4096u);
    }
    fence_async_smem();                             // make this lane's pieces visible to the TMA engine
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&ctl.ofull[rs]));
  }
}

// Tile loop of the instantiation for INT32 results.  Two uses:
//   - a convolution that ends in the INT32 residual add of Fig. 2 (Section 3.3) and the requantization of the next block
//     (WideArgs): y = clamp(relu(dn(acc + bias, b, c) + dn(res, rb, rc))) to INT32, z = clamp(dn(y, qb, qc)) to bytes;
//   - a raw INT32 result, acc + bias (FORM 3).
// Sixteen warps; a warp works on boxes of 16 pixels x 32 channels, one channel per lane.  The residual box arrives by TMA in one of the
// warp's own three 2 KiB slots (two boxes ahead), the sums are written over it in place and leave by TMA from there;
// the requantized bytes are turned round in lane quads and leave from a 512-byte box.  No CTA-wide barrier, no predicates at the
// tensor's edges (the copies clip), and 64 KiB of loads in flight per SM.
// What bounds it: nine bytes of HBM traffic per value against three wide multiplies and about fifteen plain instructions.
// 64 images of 56x56x256 (461 MB): loads and stores by the lanes (16 KiB in flight per SM) 172-261 us; boxes on eight warps
// 131-135 us, on sixteen 113-119 us (4.0 TB/s, issue slots 47 % busy); raw result 110 us with direct stores, 43 us here.
// FORM 0: every shift of the warp's channels is at least 32 (no 64-bit step).  1: c or rc below 32: 64-bit sum of the two terms,
// saturated.  2: qc below 32 as well.  3: raw.  (The loop works on 16 pixels at a time: with 32 unrolled, and the 64-bit form as
// a second pass, it ran out of the instruction cache: 2.9 stalls per issue.)
constexpr int kWideSlots = 3;
constexpr int kWideWarps = 16;          // 640 threads: 96 registers each
constexpr int kWideBox = 16 * 32 * 4, kWideQBox = 16 * 32;
// (t >> c) as upper and lower word: c1 = min(c, 32), c2 = c - c1, cm = min(c, 31)
__device__ __forceinline__ void shift64(long long t, int c1, int c2, int cm, int& up, unsigned& low) {
  const int hi = (int)(t >> 32);
  low = (unsigned)((int)__funnelshift_rc((unsigned)t, (unsigned)hi, c1) >> c2);
  up = hi >> cm;
}
// a 64-bit value saturated to INT32
__device__ __forceinline__ int sat32(int up, unsigned low) {
  return up == ((int)low >> 31) ? (int)low : (up >> 31) ^ INT_MAX;
}
template <int FORM, bool Q>
__device__ __forceinline__ void epilogue_loop_wide(const EpiCtx& e_in, const ChanConst& k_in, const CUtensorMap* map_res, const CUtensorMap* map_q) {
  const EpiCtx e = e_in;
  const ChanConst k = k_in;
  const TcParams& p = *e.p;
  SharedCtl& ctl = *e.ctl;
  constexpr bool RAW = FORM == 3;
  const int lane = e.lane;
  const int qb = Q && e.ch_live ? p.qb[e.ch] : 0, qc = Q && e.ch_live ? p.qc[e.ch] : 32;
  const long long qr0 = 1LL << (qc - 1);
  const int qsh = qc - 32, qsh1 = min(qc, 32), qsh2 = qc - qsh1, qcm = min(qc, 31);
  const int msh1 = min(k.sh, 32), msh2 = k.sh - msh1, mcm = min(k.sh, 31);
  const int rsh1 = min(k.rsh, 32), rsh2 = k.rsh - rsh1, rcm = min(k.rsh, 31);
  const uint32_t bmask = (1u << p.lg_bufs) - 1u;
  const int nb = e.px_per_warp >> 4;                                   // boxes per tile: 1 or 2
  const bool sum_out = p.out != nullptr, live = e.warp_live;
  if (e.p_tile0 >= p.p_tiles) return;
  const uint32_t t_warp = e.tmem_base + ((uint32_t)(e.q * 32) << 16) + (uint32_t)e.col0;
  const int ch0 = e.c_tile * kTileC + e.cq * 32;                       // first channel of the warp
  const uint32_t slots = e.out_stage + (uint32_t)(e.ew * kWideSlots * kWideBox);
  const uint32_t qboxes = e.out_stage + (uint32_t)(kWideWarps * kWideSlots * kWideBox + e.ew * 2 * kWideQBox);
  const bool res8 = !RAW && p.res_bits == 8;
  const uint32_t res_bytes = res8 ? kWideQBox : kWideBox, res_at = res8 ? kWideBox - kWideQBox : 0;   // bytes lie at the slot's end
  const unsigned long long pol = policy_evict_first();
  auto wait_bar = [&](unsigned long long* bar, uint32_t ph) -> bool {
    uint32_t w = 1;
    if (lane == 0) w = mbar_wait(smem_u32(bar), ph, &ctl, p.status, HQ_DEV_TIMEOUT_EPILOGUE) ? 1u : 0u;
    return __shfl_sync(0xffffffffu, w, 0) != 0;
  };
  // lane 0: the next residual box, in order of use
  int pf_tile = e.p_tile0, pf_sub = 0, pf_slot = 0, issued = 0;
  auto prefetch = [&]() {
    if (RAW || !live || pf_tile >= p.p_tiles) return;
    const uint32_t bar = smem_u32(&ctl.wbox[e.ew][pf_slot]);
    mbar_expect_tx(bar, res_bytes);
    tma_load_2d_hint(slots + (uint32_t)(pf_slot * kWideBox) + res_at, map_res, bar, res8 ? ch0 : ch0 * 4,
                     tile_at(p, pf_tile) * p.pt + e.col0 + 16 * pf_sub, pol);
    ++issued;
    if (++pf_slot == kWideSlots) pf_slot = 0;
    if (++pf_sub == nb) { pf_sub = 0; pf_tile += e.p_step; }
  };
  if (lane == 0) { prefetch(); prefetch(); }

  int done = 0, slot = 0;
  uint32_t sph = 0;
  bool ok = true;
  // 8 pixels of a box: its h-th half
  auto unit = [&](const int (&v)[8], int h) {
    uint8_t* const sp = e.smem_raw + (slots - e.raw) + slot * kWideBox;
    int* const words = (int*)sp + 256 * h + lane;
    int y[8];
    if constexpr (RAW) {
#pragma unroll
      for (int j = 0; j < 8; ++j) y[j] = v[j] + k.bias;
    } else {
      int r[8];
      if (!res8) {
#pragma unroll
        for (int j = 0; j < 8; ++j) r[j] = words[32 * j];
      } else {
        const uint8_t* const bytes = sp + res_at + 256 * h + lane;
#pragma unroll
        for (int j = 0; j < 8; ++j) r[j] = p.res_signed ? (int)(signed char)bytes[32 * j] : (int)bytes[32 * j];
        __syncwarp();                                // these byte rows may be overwritten by the sums below
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const long long t = hq_mad_wide(v[j], k.b, k.r0), u = hq_mad_wide(r[j], k.rb, k.rr0);
        if constexpr (FORM == 0) {
          y[j] = ((int)(t >> 32) >> msh2) + ((int)(u >> 32) >> rsh2);                // each within [-2^30, 2^30)
        } else {
          int tu, uu;
          unsigned tl, ul;
          shift64(t, msh1, msh2, mcm, tu, tl);
          shift64(u, rsh1, rsh2, rcm, uu, ul);
          unsigned low;
          int up;
          asm("add.cc.u32 %0, %2, %3;\n\taddc.s32 %1, %4, %5;" : "=r"(low), "=r"(up) : "r"(tl), "r"(ul), "r"(tu), "r"(uu));
          y[j] = sat32(up, low);
        }
        y[j] = min(max(y[j], e.lo), e.hi);
      }
    }
    if (RAW || sum_out) {
#pragma unroll
      for (int j = 0; j < 8; ++j) words[32 * j] = y[j];
    }
    if constexpr (Q) {
      const uint32_t qrow = qboxes + (uint32_t)((done & 1) * kWideQBox + 256 * h + (lane & 3) * 32 + (lane & ~3));
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        int z[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          long long t = hq_mad_wide(y[4 * g + j], qb, qr0);
          if constexpr (FORM < 2) z[j] = (int)(t >> 32) >> qsh;
          else { int up; unsigned low; shift64(t, qsh1, qsh2, qcm, up, low); z[j] = sat32(up, low); }
        }
        unsigned w;
        if (p.q_sat == 1) w = sat_pack4<false>(z[0], z[1], z[2], z[3]);
        else {
#pragma unroll
          for (int j = 0; j < 4; ++j) z[j] = min(max(z[j], p.q_lo), p.q_hi);
          w = __byte_perm(__byte_perm((unsigned)z[0], (unsigned)z[1], 0x0040), __byte_perm((unsigned)z[2], (unsigned)z[3], 0x0040), 0x5410);
        }
        w = quad_transpose(w, lane);                                      // four channels of pixel 8 h + 4 g + lane % 4
        asm volatile("st.shared.b32 [%0], %1;" ::"r"(qrow + 128u * g), "r"(w) : "memory");
      }
    }
  };
  // the finished box leaves, the box after next is fetched
  auto ship = [&](int px0) {
    fence_async_smem();                              // make this lane's writes visible to the TMA engine
    __syncwarp();
    if (lane == 0) {
      if (px0 < p.P) {
        if (RAW || sum_out) tma_store_2d(e.map_out, slots + (uint32_t)(slot * kWideBox), ch0 * 4, px0);
        if (Q) tma_store_2d(map_q, qboxes + (uint32_t)((done & 1) * kWideQBox), ch0, px0);
      }
      tma_store_commit();
      // the store before this one has been read: its slot takes the box after next, and the other byte box is free
      asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
      prefetch();
    }
    __syncwarp();
    ++done;
    if (++slot == kWideSlots) { slot = 0; sph ^= 1u; }
  };

  int va[8], vb[8];
  uint32_t tcount = 0, as = 0;
  int p_tile = e.p_tile0;
  if (wait_bar(&ctl.tfull[0], 0)) {
    tc_fence_after();
    tmem_ld8_issue(t_warp, va);
    bool pending = true;
    while (true) {
      const int px_first = tile_at(p, p_tile) * p.pt + e.col0;
      const bool has_next = p_tile + e.p_step < p.p_tiles;
      const uint32_t nas = (tcount + 1u) & bmask, naph = ((tcount + 1u) >> p.lg_bufs) & 1u;
      const uint32_t t_addr = t_warp + as * p.acc_stride;
#pragma unroll 1
      for (int c = 0; c < nb; ++c) {
        if (!RAW && live) { ok = wait_bar(&ctl.wbox[e.ew][slot], sph); if (!ok) break; }
        tmem_ld_wait();
        tie(va);
        tmem_ld8_issue(t_addr + 16 * c + 8, vb);
        if (live) unit(va, 0);
        tmem_ld_wait();
        tie(vb);
        pending = false;
        if (c + 1 < nb) { tmem_ld8_issue(t_addr + 16 * (c + 1), va); pending = true; }
        else {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) release_accumulator(p, ctl, as);
        }
        if (live) unit(vb, 1);
        if (live) ship(px_first + 16 * c);
      }
      if (!ok || !has_next) break;
      if (!wait_bar(&ctl.tfull[nas], naph)) break;
      tc_fence_after();
      tmem_ld8_issue(t_warp + nas * p.acc_stride, va);
      pending = true;
      p_tile += e.p_step; ++tcount; as = nas;
    }
    if (pending) tmem_ld_wait();
  }
  if (lane == 0) {
    // every copy this thread started must have landed before the CTA may exit (all consumed unless a wait ran out)
    for (int i = done; !RAW && i < issued; ++i) {
      const uint32_t bar = smem_u32(&ctl.wbox[e.ew][i % kWideSlots]), ph = (uint32_t)(i / kWideSlots) & 1u;
      const unsigned long long t0 = global_ns();
      while (!mbar_try_wait(bar, ph))
        if (global_ns() - t0 > kWaitBudgetNs) { atomicCAS(p.status, 0u, (uint32_t)HQ_DEV_TIMEOUT_DRAIN); break; }
    }
    tma_store_wait_all();
  }
}

// General tile loop: every output type, direct stores, 64-bit arithmetic, INT32 residuals.
__device__ __noinline__ void epilogue_loop_general(const EpiCtx& e, const ChanConst& k, uint32_t fast) {
  const TcParams& p = *e.p;
  SharedCtl& ctl = *e.ctl;
  const CUtensorMap& map_out = *e.map_out;
  uint8_t* const smem_raw = e.smem_raw;
  const uint32_t raw = e.raw, out_stage = e.out_stage, res_stage = e.res_stage, res_tile_bytes = e.res_tile_bytes;
  const uint32_t tmem_base = e.tmem_base;
  const int lane = e.lane, q = e.q, cq = e.cq, ew = e.ew, col0 = e.col0, px_per_warp = e.px_per_warp, ch = e.ch;
  const int c_tile = e.c_tile, p_tile0 = e.p_tile0, p_step = e.p_step, lo = e.lo, hi = e.hi;
  const bool ch_live = e.ch_live, warp_live = e.warp_live;
  const bool staged_out = p.staged_out != 0;
    // staging box of this warp: [px_per_warp pixels][32 channels] bytes (16 bytes per pixel at 4 bit)
    const int row_b = (p.out_bits == 4) ? 16 : 32;
    const uint32_t my_stage = out_stage + (uint32_t)ew * (uint32_t)(px_per_warp * 32);   // px_per_warp rows x 32 bytes reserved per warp
    // plain pointers to the same bytes: ordinary loads / stores that the compiler may schedule freely
    uint8_t* const my_stage_ptr = smem_raw + (my_stage - raw);
    const uint8_t* const res_stage_ptr = smem_raw + (res_stage - raw);
    const uint32_t bmask = (1u << p.lg_bufs) - 1u;
    uint32_t tcount = 0;
    for (int p_tile = p_tile0; p_tile < p.p_tiles; p_tile += p_step, ++tcount) {
      const uint32_t as = tcount & bmask, aph = (tcount >> p.lg_bufs) & 1u;
      const uint32_t rs = tcount & ((1u << p.lg_rbufs) - 1u), rph = (tcount >> p.lg_rbufs) & 1u;
      uint32_t w = 1;
      if (lane == 0) {
        if (staged_out) tma_store_wait_read0();   // the previous store has read this warp's staging box
        w = mbar_wait(smem_u32(&ctl.tfull[as]), aph, &ctl, p.status, HQ_DEV_TIMEOUT_EPILOGUE) ? 1u : 0u;
        if (w && p.staged_res)
          w = mbar_wait(smem_u32(&ctl.rfull[rs]), rph, &ctl, p.status, HQ_DEV_TIMEOUT_EPILOGUE) ? 1u : 0u;
      }
      w = __shfl_sync(0xffffffffu, w, 0);
      if (!w) break;
      tc_fence_after();                            // lane 0 observed the barriers; the shuffle ordered the warp
      const int p_base = tile_at(p, p_tile) * p.pt + col0;              // first pixel of this warp's columns
      const uint8_t* const res_tile = res_stage_ptr + rs * res_tile_bytes + (uint32_t)col0 * kTileC + cq * 32 + lane;

      for (int cc0 = 0; cc0 < px_per_warp; cc0 += 32) {
        int v[32];
        tmem_ld32_issue(tmem_base + ((uint32_t)(q * 32) << 16) + as * p.pt + col0 + cc0, v);
        tmem_ld_wait();
        tie(v);
        if (!warp_live) continue;
        const int px0 = p_base + cc0;                                     // global pixel of v[0]

        if (p.out_bits == 32) {
          // raw accumulator + bias: 32 lanes write 32 consecutive INT32 channels of one pixel
          if (ch_live) {
            int* dst = (int*)p.out + (long long)px0 * p.C + ch;
#pragma unroll
            for (int j = 0; j < 32; ++j) if (px0 + j < p.P) dst[(long long)j * p.C] = v[j] + k.bias;
          }
          continue;
        }

        int y[32];
        if (fast) {
          unsigned rb8[32];
          if (p.res) {
            if (p.staged_res) {
#pragma unroll
              for (int j = 0; j < 32; ++j) rb8[j] = res_tile[(cc0 + j) * kTileC];
            } else {
              const unsigned char* rp = (const unsigned char*)p.res + (long long)px0 * p.C + ch;
#pragma unroll
              for (int j = 0; j < 32; ++j) rb8[j] = (ch_live && px0 + j < p.P) ? (unsigned)__ldg(rp + (long long)j * p.C) : 0u;
            }
          }
          const int variant = (p.res ? 2 : 0) | (p.res_signed ? 1 : 0);
          if (variant == 2) {
#pragma unroll
            for (int j = 0; j < 32; ++j) y[j] = requant_fast<true, false, true>(v[j], (int)rb8[j], k);
          } else if (variant == 3) {
#pragma unroll
            for (int j = 0; j < 32; ++j) y[j] = requant_fast<true, true, true>(v[j], (int)(signed char)rb8[j], k);
          } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) y[j] = requant_fast<false, false, true>(v[j], 0, k);
          }
          if (p.sat_pack) {
            if (p.out_signed) {
#pragma unroll
              for (int j = 0; j < 32; ++j) y[j] = sat_s8(y[j]);
            } else {
#pragma unroll
              for (int j = 0; j < 32; ++j) y[j] = sat_u8(y[j]);
            }
          } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) y[j] = min(max(y[j], lo), hi);
          }
        } else {
          // general CTA: full 64-bit results (any 1 <= c <= 62, INT32 residual operands)
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            long long s = ((long long)v[j] * (long long)k.b + k.r0) >> k.sh;
            if (p.res) {
              int r = 0;
              if (p.staged_res) {
                const unsigned byte = res_tile[(cc0 + j) * kTileC];
                r = p.res_signed ? (int)(signed char)byte : (int)byte;
              } else if (ch_live && px0 + j < p.P) {
                r = hq_load_elem(p.res, (long long)(px0 + j) * p.C + ch, p.res_bits, p.res_signed);
              }
              s += ((long long)r * (long long)k.rb + k.rr0) >> k.rsh;
            }
            y[j] = hq_clamp_ll(s, p.relu, p.qmin, p.qmax);
          }
        }

        if (p.out_bits == 4) {
          // neighbouring channels share a byte: even lanes collect the odd lane's nibble
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const int other = __shfl_xor_sync(0xffffffffu, y[j], 1);
            y[j] = (y[j] & 0xF) | ((other & 0xF) << 4);
          }
          if (staged_out) {
            if (!(lane & 1)) {
#pragma unroll
              for (int j = 0; j < 32; ++j) my_stage_ptr[(cc0 + j) * row_b + (lane >> 1)] = (uint8_t)y[j];
            }
          } else if (ch_live && !(lane & 1)) {
            unsigned char* dst = (unsigned char*)p.out + (((long long)px0 * p.C + ch) >> 1);
#pragma unroll
            for (int j = 0; j < 32; ++j) if (px0 + j < p.P) dst[((long long)j * p.C) >> 1] = (unsigned char)y[j];
          }
        } else if (staged_out) {
#pragma unroll
          for (int j = 0; j < 32; ++j) my_stage_ptr[(cc0 + j) * 32 + lane] = (uint8_t)y[j];
        } else if (ch_live) {
          unsigned char* dst = (unsigned char*)p.out + (long long)px0 * p.C + ch;
#pragma unroll
          for (int j = 0; j < 32; ++j) if (px0 + j < p.P) dst[(long long)j * p.C] = (unsigned char)(y[j] & 0xFF);
        }
      }
      // accumulator columns (and the residual tile) are no longer needed by this warp: hand them back
      tc_fence_before();
      if (staged_out) fence_async_smem();        // make this lane's box writes visible to the TMA engine
      __syncwarp();
      if (lane == 0) {
        release_accumulator(p, ctl, as);
        if (p.staged_res) mbar_arrive(smem_u32(&ctl.rempty[rs]));
        if (staged_out && warp_live)
          store_warp_box(p, &map_out, my_stage, ((c_tile * kTileC + cq * 32) * p.out_bits) >> 3, tile_at(p, p_tile), col0, px_per_warp);
      }
    }

    if (staged_out && lane == 0) tma_store_wait_all();
}

// MMA issue of the frag shape.  One thread needs about 1 k cycles per K block, nearly all of it the latency of its own
// instructions between one barrier and the next, so two issuers share the work:
//   - DEAL false: issuer `c` of `n` takes the tiles c, c + n, ...  The stage count is a multiple of n * k_blocks;
//   - DEAL true: the K blocks of the CTA, numbered through its tiles, alternate between the two issuers, whose number divides
//     the stage count; the tile's first, overwriting MMA signals `tstart`, which the other one awaits.
// Either way a stage belongs to one issuer for the whole launch.  It has to: a wait for a stage's m-th fill looks at a parity and
// cannot tell it from the (m-2)-nd, so the waiting thread must have seen the (m-1)-st itself.  (No other barrier shows that one: copies
// land out of order, and with five stages of one-block tiles the fill before is the other issuer's, five tiles back, while the
// accumulator's barrier speaks of the tile four back.)
template <int STEPS, bool DEAL>
__device__ __forceinline__ void frag_issue(const TcParams& p, SharedCtl& ctl, int c, int n, uint32_t tiles, uint32_t stage_bytes,
                                           uint32_t w_bytes, uint32_t tmem_base, int p_tile0, int p_step) {
  const uint32_t idesc = (2u << 4) | (1u << 7) | ((uint32_t)(p.x_signed ? 1 : 0) << 10) | ((uint32_t)(kTileC >> 3) << 17) |
                         ((uint32_t)(kTileC >> 4) << 24);
  const uint64_t hi = smem_desc(0, STEPS * 32);
  const uint32_t x_off = p.wres ? 0u : w_bytes;
  const uint32_t nstages = (uint32_t)p.stages;
  const int k_blocks = p.k_blocks;
  const bool tail = p.tail_steps != STEPS;
  const int per = DEAL ? 2 : 1, tiles_per = DEAL ? 1 : n;
  if (p.wres && !mbar_wait(smem_u32(&ctl.wfull), 0, &ctl, p.status, HQ_DEV_TIMEOUT_MMA)) return;
  uint32_t s = 0, ph = 0, tcount = DEAL ? 0u : (uint32_t)c;
  auto skip = [&](int blocks) { for (int i = 0; i < blocks; ++i) if (++s == nstages) { s = 0; ph ^= 1u; } };
  skip(DEAL ? c : c * k_blocks);
  int kb = DEAL ? c : 0;
  for (int p_tile = p_tile0 + (DEAL ? 0 : c * p_step); p_tile < p.p_tiles; p_tile += tiles_per * p_step, tcount += (uint32_t)tiles_per) {
    const uint32_t as = tcount & (kFragAccs - 1), aph = (tcount / kFragAccs) & 1u;
    const uint32_t d = tmem_base + as * kTileC;
    if (!mbar_wait(smem_u32(&ctl.tempty[as]), aph ^ 1u, &ctl, p.status, HQ_DEV_TIMEOUT_MMA)) return;
    bool first = DEAL && kb != 0;
    for (; kb < k_blocks; kb += per) {
      if (!mbar_wait(smem_u32(&ctl.full[s]), ph, &ctl, p.status, HQ_DEV_TIMEOUT_MMA)) return;
      if (DEAL && first) {
        if (!mbar_wait(smem_u32(&ctl.tstart[as]), aph, &ctl, p.status, HQ_DEV_TIMEOUT_MMA)) return;
        first = false;
      }
      tc_fence_after();
      const uint32_t x = tiles + s * stage_bytes, w = p.wres ? tiles + p.wres_off + (uint32_t)kb * w_bytes : x;
      const uint64_t ad = hi | (uint64_t)((w >> 4) & 0x3FFF), bd = hi | (uint64_t)(((x + x_off) >> 4) & 0x3FFF);
      if (tail && (kb + 1) % p.cchunks == 0) {
        for (int k = 0; k < p.tail_steps; ++k) mma_i8(d, ad + 2 * k, bd + 2 * k, idesc, (kb | k) ? 1u : 0u);
      } else {
#pragma unroll
        for (int k = 0; k < STEPS; ++k) mma_i8(d, ad + 2 * k, bd + 2 * k, idesc, k ? 1u : kb ? 1u : 0u);
      }
      if (DEAL && kb == 0) { tc_fence_before(); mbar_arrive(smem_u32(&ctl.tstart[as])); }    // (the other issuer fences behind its wait)
      if (kb + per >= k_blocks) mma_commit(smem_u32(&ctl.tfull[as]));
      mma_commit(smem_u32(&ctl.empty[s]));
      s += (uint32_t)per;
      if (s >= nstages) { s -= nstages; ph ^= 1u; }
    }
    kb -= k_blocks;
    if (!DEAL) { kb = 0; skip((n - 1) * k_blocks); }
  }
}

// ---------------------------------------------------------------- the kernel -----------------
// DUO: the instantiation that may be launched as clusters of two CTAs sharing their MMAs; only it contains the
// cta_group::2 instructions (a kernel that contains them cannot be launched without clusters).
// FRAG: the instantiation of the frag shape; it has one more warp, which stores the finished output tiles.
// WIDE: the instantiations for INT32 results (epilogue_loop_wide), kRaw32 or through the residual add of Fig. 2, kAdd32.  (One for
// both ran the add 0.6 % slower as soon as the raw form's waits for parameters were in it; the add only runs in networks.)
constexpr int kRaw32 = 1, kAdd32 = 2;
template <int EPI_WARPS, int MIN_CTAS, int MMA_WARPS, bool DUO = false, bool FRAG = false, int WIDE = 0>
__global__ void __launch_bounds__(32 * (1 + MMA_WARPS + EPI_WARPS + (FRAG ? 1 : 0)), MIN_CTAS)
conv_tc_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w,
               const __grid_constant__ CUtensorMap map_out, const __grid_constant__ CUtensorMap map_res,
               const __grid_constant__ CUtensorMap map_q, const __grid_constant__ TcParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ SharedCtl ctl;

  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t tiles = (raw + 1023u) & ~1023u;          // operand stages, 1024-byte aligned
  const uint32_t w_bytes = kTileC * p.bkb;
  // strip mode: the stages carry weights only; duo: each CTA of the pair holds half of the pixel rows
  const uint32_t x_bytes = p.strip ? 0u : (uint32_t)((p.pt >> p.duo) * p.bkb);
  uint32_t rank = 0u;                                      // 0 = the CTA that issues the pair's MMAs
  if constexpr (DUO) rank = cluster_ctarank();
  const uint32_t x_off = p.wres ? 0u : w_bytes;          // offset of the X tile inside a stage
  const uint32_t stage_bytes = x_off + x_bytes;
  const uint32_t out_stage = tiles + p.out_stage_off;
  const uint32_t res_stage = tiles + p.res_stage_off;
  const uint32_t res_tile_bytes = p.pt * kTileC;          // [pt pixels][128 channels] bytes
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // Tile schedule: the grid is a multiple of c_tiles, so a CTA keeps one channel tile for its whole
  // life (its weights' rows and per-channel constants never change) and strides over the pixel tiles.
  const int c_tile = blockIdx.x % p.c_tiles;
  const int p_tile0 = blockIdx.x / p.c_tiles;
  const int p_step = gridDim.x / p.c_tiles;

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) { mbar_init(smem_u32(&ctl.full[s]), 1); mbar_init(smem_u32(&ctl.empty[s]), 1); }
    for (int s = 0; s < (1 << p.lg_bufs); ++s) {
      mbar_init(smem_u32(&ctl.tfull[s]), FRAG && !p.deal ? 1 : p.ni); mbar_init(smem_u32(&ctl.tempty[s]), (4 * p.halves) << p.duo);
      mbar_init(smem_u32(&ctl.tstart[s]), 1);
    }
    for (int s = 0; s < (1 << p.lg_rbufs); ++s) {
      mbar_init(smem_u32(&ctl.rfull[s]), 1);
      mbar_init(smem_u32(&ctl.rempty[s]), FRAG ? 1 : 4 * p.halves);
      mbar_init(smem_u32(&ctl.ofull[s]), EPI_WARPS / kFragGroups);
    }
    mbar_init(smem_u32(&ctl.drain), FRAG ? MMA_WARPS : p.ni);
    mbar_init(smem_u32(&ctl.wfull), 1);
    if constexpr (WIDE) for (int s = 0; s < kWideWarps * kWideSlots; ++s) mbar_init(smem_u32(&ctl.wbox[s / kWideSlots][s % kWideSlots]), 1);
    for (int s = 0; s < 3; ++s) { mbar_init(smem_u32(&ctl.pfull[s]), 1); mbar_init(smem_u32(&ctl.pempty[s]), p.ni); }
    ctl.abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) { if constexpr (DUO) tmem_alloc2(smem_u32(&ctl.tmem_base), p.tmem_cols); else tmem_alloc(smem_u32(&ctl.tmem_base), p.tmem_cols); }
  tc_fence_before();
  __syncthreads();
  if constexpr (DUO) cluster_sync_all();   // both CTAs' barriers exist before either touches the other's
  tc_fence_after();
  const uint32_t tmem_base = ctl.tmem_base;
  // Programmatic dependent launch: this grid may have started while the previous kernel of the stream was
  // still finishing (its CTAs leave the SMs one by one); everything above touched only this CTA's own
  // resources.  The threads that read what the previous kernel wrote -- the producer lane (activations and
  // residual tiles by TMA) and epilogue warps that load a residual directly -- wait for that grid to complete
  // first; the other roles only consume what arrives behind the producer's barriers.  The next kernel's CTAs
  // may start filling SMs as ours leave.  Weights and constants are read ahead of that inside a network; a call of its own
  // (params_late) may follow the kernel that wrote them: its producer and epilogue wait before they read those too, and the
  // next kernel is let in after the producer's wait only (a network's second layer would read its own parameters at once).
  const bool params_late = WIDE != kAdd32 && p.params_late != 0;
  if (!params_late) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (elect_one()) {
      // No division or modulo in this loop: one thread runs it and every dependent instruction
      // costs its full latency, so stage / phase / filter-tap indices are carried incrementally.
      uint32_t it = 0, tcount = 0, s = 0, ph = 0;
      const uint32_t rmask = (1u << p.lg_rbufs) - 1u;
      bool ok = true;
      // (image, row, column) of the tile's first output pixel, advanced by a fixed step per tile
      const int ho = p.howo / p.wo;
      // (duo: this CTA fetches the half of the tile's pixel rows that starts at half_off)
      const int half_off = p.duo ? (int)rank * (p.pt >> 1) : 0;
      const int px_first = tile_at(p, p_tile0) * p.pt + half_off;
      int img = px_first / p.howo;
      int oh = (px_first - img * p.howo) / p.wo;
      int ow = px_first - img * p.howo - oh * p.wo;
      const int step = p_step * p.pt;
      const int d_img = step / p.howo, d_oh = (step - d_img * p.howo) / p.wo, d_ow = step - d_img * p.howo - d_oh * p.wo;
      if (params_late) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
      }
      if (p.wres) {              // the channel tile's weights for every K block, once
        const uint32_t bar = smem_u32(&ctl.wfull);
        mbar_expect_tx(bar, (uint32_t)p.w_blocks * w_bytes);
        int wx = 0, tap_x = 0, left = p.cchunks;
        for (int kb = 0; kb < p.w_blocks; ++kb) {
          const uint32_t w_dst = tiles + p.wres_off + (uint32_t)kb * w_bytes;
          if (p.pairs) {           // block (filter row, half of the four pixels): rows of output 2q, then of output 2q + 1
            tma_load_3d(w_dst, &map_w, bar, (kb & 1) * 128, kb >> 1, 0);
            tma_load_3d(w_dst + 64 * 128, &map_w, bar, (kb & 1) * 128 - 64, kb >> 1, 0);
          } else if (p.fold) {
            tma_load_2d(w_dst, &map_w, bar, wx, 0);
            tma_load_2d(w_dst + 64 * p.bkb, &map_w, bar, wx, 0);
          } else if constexpr (FRAG) {
            tma_load_4d(w_dst, &map_w, bar, wx, 0, 0, c_tile * (kTileC / 16));
          } else {
            tma_load_2d(w_dst, &map_w, bar, wx, c_tile * kTileC);
          }
          wx += p.bkb;
          if (--left == 0) { left = p.cchunks; tap_x += p.cin; wx = tap_x; }
        }
      }
      // The resident weights above do not wait for the previous kernel unless it may have written them (params_late; the
      // helper kernels that prepare weights are always followed by another launch).
      // Everything below reads activations, which the previous kernel may still be writing.
      asm volatile("griddepcontrol.wait;" ::: "memory");
      const unsigned long long pol_first = policy_evict_first();
      uint32_t pit = 0;                                // strip mode: patches started
      if (p.strip) {
        uint32_t ps = 0, pph = 0;
        for (int p_tile = p_tile0; p_tile < p.p_tiles && ok; p_tile += p_step, ++tcount) {
          const int t_act = tile_at(p, p_tile);
          const int img_s = t_act / p.tpi, y0 = (t_act - img_s * p.tpi) * p.rows;
          for (int chunk = 0; chunk < p.cchunks && ok; ++chunk) {
            // the padded patch of this cin chunk: columns -1 .. 2^lg_wp - 2, rows y0-1 .. y0+rows+1 (zeros outside the image)
            if (!mbar_wait(smem_u32(&ctl.pempty[ps]), pph ^ 1u, &ctl, p.status, HQ_DEV_TIMEOUT_PRODUCER)) { ok = false; break; }
            const uint32_t pbar = smem_u32(&ctl.pfull[ps]);
            mbar_expect_tx(pbar, p.patch_bytes);
            tma_load_4d(tiles + p.patch_off + ps * p.patch_bytes, &map_x, pbar, chunk * p.bkb, -1, y0 - 1, img_s);
            ++pit;
            if (++ps == (uint32_t)p.npatch) { ps = 0; pph ^= 1u; }
            if (p.wres) continue;
            for (int tap = 0; tap < 9; ++tap, ++it) {      // the nine weight blocks that meet this patch
              if (!mbar_wait(smem_u32(&ctl.empty[s]), ph ^ 1u, &ctl, p.status, HQ_DEV_TIMEOUT_PRODUCER)) { ok = false; break; }
              const uint32_t bar = smem_u32(&ctl.full[s]);
              const uint32_t w_dst = tiles + s * stage_bytes;
              const int kb = tap * p.cchunks + chunk;
              mbar_expect_tx(bar, stage_bytes);
              if (p.fold) {
                tma_load_2d(w_dst, &map_w, bar, kb * p.bkb, 0);
                tma_load_2d(w_dst + 64 * p.bkb, &map_w, bar, kb * p.bkb, 0);
              } else {
                tma_load_2d(w_dst, &map_w, bar, kb * p.bkb, c_tile * kTileC);
              }
              if (++s == (uint32_t)p.stages) { s = 0; ph ^= 1u; }
            }
          }
        }
      }
      if (FRAG && p.wres && p.x_tiled) {
        // the leanest form for the layers with the most tiles: this thread's instructions are on the tile's path
        const int k_blocks = p.k_blocks, bkb = p.bkb;
        for (int p_tile = p_tile0; p_tile < p.p_tiles && ok; p_tile += p_step) {
          const int p0 = tile_at(p, p_tile) * kTileC;
          for (int kb = 0; kb < k_blocks; ++kb, ++it) {
            if (!mbar_wait(smem_u32(&ctl.empty[s]), ph ^ 1u, &ctl, p.status, HQ_DEV_TIMEOUT_PRODUCER)) { ok = false; break; }
            const uint32_t bar = smem_u32(&ctl.full[s]);
            mbar_expect_tx(bar, stage_bytes);
            tma_load_2d_hint(tiles + s * stage_bytes, &map_x, bar, kb * bkb, p0, pol_first);
            if (++s == (uint32_t)p.stages) { s = 0; ph ^= 1u; }
          }
        }
      } else
      for (int p_tile = p_tile0; p_tile < p.p_tiles && ok && !p.strip; p_tile += p_step, ++tcount) {
        const int p0 = tile_at(p, p_tile) * p.pt;
        const int cw = ow * p.stride - p.pad, chh = oh * p.stride - p.pad, img_now = img;
        if (!p.rev) {
          ow += d_ow; if (ow >= p.wo) { ow -= p.wo; ++oh; }
          oh += d_oh; if (oh >= ho) { oh -= ho; ++img; }
          img += d_img;
        } else {                                     // the same step backwards, with borrows (unused after the last tile)
          ow -= d_ow; if (ow < 0) { ow += p.wo; --oh; }
          oh -= d_oh; if (oh < 0) { oh += ho; --img; }
          img -= d_img;
        }
        int chunk = 0, tap_s = 0, tap_r = 0, wx = 0, tap_x = 0;     // wx: the block's first byte in a weight row
        // The residual tile of this output tile is fetched as soon as its buffer is free, but this thread only
        // blocks for the buffer after the tile's last operand block is on its way: the buffer comes back when the
        // epilogue of an earlier tile ends, and the operand copies must not queue behind that.
        bool res_due = !FRAG && p.staged_res != 0;                  // (frag: the store warp fetches them)
        auto residual = [&](bool must) -> bool {
          const uint32_t rbuf = tcount & rmask, rph = (tcount >> p.lg_rbufs) & 1u;
          const uint32_t rb = smem_u32(&ctl.rempty[rbuf]);
          if (!mbar_try_wait(rb, rph ^ 1u)) {
            if (!must) return true;
            if (!mbar_wait(rb, rph ^ 1u, &ctl, p.status, HQ_DEV_TIMEOUT_PRODUCER)) return false;
          }
          const uint32_t bar = smem_u32(&ctl.rfull[rbuf]);
          mbar_expect_tx(bar, res_tile_bytes);
          tma_load_2d_hint(res_stage + rbuf * res_tile_bytes, &map_res, bar, c_tile * kTileC, p0, pol_first);
          res_due = false;
          return true;
        };
        for (int kb = 0; kb < p.k_blocks; ++kb, ++it) {
          if (res_due && !residual(false)) { ok = false; break; }
          if (!mbar_wait(smem_u32(&ctl.empty[s]), ph ^ 1u, &ctl, p.status, HQ_DEV_TIMEOUT_PRODUCER)) { ok = false; break; }
          const uint32_t bar = smem_u32(&ctl.full[s]);
          const uint32_t w_dst = tiles + s * stage_bytes;
          if constexpr (DUO) {
            // Both CTAs of the pair fetch their own weight rows and their half of the pixel rows into their own
            // stage; all four copies are counted on the leading CTA's barrier, which alone expects the bytes.
            if (rank == 0) mbar_expect_tx(bar, 2u * stage_bytes);
            if (p.x_tiled) tma_load_2d_2cta(w_dst + x_off, &map_x, bar, chunk * p.bkb, p0 + half_off);
            else tma_load_im2col_2cta(w_dst + x_off, &map_x, bar, chunk * p.bkb, cw, chh, img_now, (uint16_t)tap_s, (uint16_t)tap_r);
            tma_load_2d_2cta(w_dst, &map_w, bar, wx, c_tile * kTileC);
            wx += p.bkb;
            if (++chunk == p.cchunks) { chunk = 0; tap_x += p.cin; wx = tap_x; if (++tap_s == p.kw) { tap_s = 0; ++tap_r; } }
            if (++s == (uint32_t)p.stages) { s = 0; ph ^= 1u; }
            if (res_due && kb + 1 == p.k_blocks && !residual(true)) { ok = false; break; }
            continue;
          }
          mbar_expect_tx(bar, stage_bytes);
          if (p.x_tiled) {
            tma_load_2d_hint(w_dst + x_off, &map_x, bar, chunk * p.bkb, p0, pol_first);
          } else {
            tma_load_im2col(w_dst + x_off, &map_x, bar, chunk * p.bkb, cw, chh, img_now, (uint16_t)tap_s, (uint16_t)tap_r);
          }
          if (p.wres) {
            // weights are resident
          } else if (p.fold) {   // 64-row box, twice: accumulator lanes 64-127 repeat lanes 0-63
            tma_load_2d(w_dst, &map_w, bar, wx, 0);
            tma_load_2d(w_dst + 64 * p.bkb, &map_w, bar, wx, 0);
          } else if constexpr (FRAG) {
            tma_load_4d(w_dst, &map_w, bar, wx, 0, 0, c_tile * (kTileC / 16));
          } else {
            tma_load_2d(w_dst, &map_w, bar, wx, c_tile * kTileC);
          }
          wx += p.bkb;
          if (++chunk == p.cchunks) { chunk = 0; tap_x += p.cin; wx = tap_x; if (++tap_s == p.kw) { tap_s = 0; ++tap_r; } }
          if (++s == (uint32_t)p.stages) { s = 0; ph ^= 1u; }
          if (res_due && kb + 1 == p.k_blocks && !residual(true)) { ok = false; break; }
        }
      }
      // Drain: every copy this thread started must have landed before the CTA may exit.
      // (the odd CTA of a pair sees no completion of its own copies: they are counted on the leading CTA's barriers,
      // whose MMAs consume them before the pair's closing cluster barrier)
      const uint32_t issued = (p.duo && rank != 0) ? 0u : (it < (uint32_t)p.stages ? it : (uint32_t)p.stages);
      for (uint32_t j = 0; j < (p.npatch > 0 ? (pit < (uint32_t)p.npatch ? pit : (uint32_t)p.npatch) : 0u); ++j) {
        const uint32_t k = pit - 1 - j;
        const unsigned long long t0 = global_ns();
        while (!mbar_try_wait(smem_u32(&ctl.pfull[k % p.npatch]), (k / p.npatch) & 1u)) {
          if (global_ns() - t0 > kWaitBudgetNs) { atomicCAS(p.status, 0u, (uint32_t)HQ_DEV_TIMEOUT_DRAIN); break; }
        }
      }
      for (uint32_t j = 0; j < issued; ++j) {
        const uint32_t k = it - 1 - j;
        const uint32_t ds = k % p.stages, dph = (k / p.stages) & 1u;
        const unsigned long long t0 = global_ns();
        while (!mbar_try_wait(smem_u32(&ctl.full[ds]), dph)) {
          if (global_ns() - t0 > kWaitBudgetNs) { atomicCAS(p.status, 0u, (uint32_t)HQ_DEV_TIMEOUT_DRAIN); break; }
        }
      }
      if (p.wres) {
        const unsigned long long t0 = global_ns();
        while (!mbar_try_wait(smem_u32(&ctl.wfull), 0)) {
          if (global_ns() - t0 > kWaitBudgetNs) { atomicCAS(p.status, 0u, (uint32_t)HQ_DEV_TIMEOUT_DRAIN); break; }
        }
      }
      if (!FRAG && p.staged_res) {
        const uint32_t tiles_done = tcount < rmask + 1u ? tcount : rmask + 1u;
        for (uint32_t j = 0; j < tiles_done; ++j) {
          const uint32_t k = tcount - 1 - j;
          const unsigned long long t0 = global_ns();
          while (!mbar_try_wait(smem_u32(&ctl.rfull[k & rmask]), (k >> p.lg_rbufs) & 1u)) {
            if (global_ns() - t0 > kWaitBudgetNs) { atomicCAS(p.status, 0u, (uint32_t)HQ_DEV_TIMEOUT_DRAIN); break; }
          }
        }
      }
    }
  } else if (warp <= MMA_WARPS) {
    // ------------------------------------------------------------ MMA issuers
    // The K blocks of the CTA's tiles, numbered through (g = tile * k_blocks + b), are dealt round-robin to p.ni
    // issuer warps (one lane each).  A single thread cannot keep the tensor pipe busy: every shared-memory
    // operation it executes between two batches of MMAs (the wait for the next operands) holds it for a few hundred
    // cycles while its own MMAs are in flight, and the pipe drains meanwhile; with the waits of one issuer falling
    // into the MMAs of the others the pipe stays fed.  The stage count is a multiple of p.ni, so a stage is always
    // read by the same issuer: its parity waits then follow one another like a single thread's (a thread that
    // looked at a stage's barrier a whole fill early would take the fill before for its own).  Integer accumulation
    // does not care about the order of the blocks; only the tile's first MMA, which overwrites the accumulator,
    // must come first: whoever issues it signals `tstart` and the others wait for that.
    const int iss = warp - 1;
    if constexpr (FRAG) {
      if (elect_one()) {
        if (iss < p.ni) {
#define HQ_ISSUE(STEPS) do { if (p.deal) frag_issue<STEPS, true>(p, ctl, iss, p.ni, tiles, stage_bytes, w_bytes, tmem_base, p_tile0, p_step); \
                             else frag_issue<STEPS, false>(p, ctl, iss, p.ni, tiles, stage_bytes, w_bytes, tmem_base, p_tile0, p_step); } while (0)
          if (p.bkb == 128) HQ_ISSUE(4); else if (p.bkb == 64) HQ_ISSUE(2); else HQ_ISSUE(1);
#undef HQ_ISSUE
        }
        // Drain: all issued MMAs must have completed before tensor memory is freed.
        mma_commit(smem_u32(&ctl.drain));
        const unsigned long long t0 = global_ns();
        while (!mbar_try_wait(smem_u32(&ctl.drain), 0)) {
          if (global_ns() - t0 > kWaitBudgetNs) { atomicCAS(p.status, 0u, (uint32_t)HQ_DEV_TIMEOUT_DRAIN); break; }
        }
      }
    } else if (iss < p.ni && rank == 0 && elect_one()) {
      // instruction descriptor: D = S32, A = s8 weights, B = u8/s8 activations, both K-major, N = pt,
      // M = 128 (256 over the two CTAs of a pair)
      const uint32_t idesc = (2u << 4) | (1u << 7) | ((uint32_t)(p.x_signed ? 1 : 0) << 10) |
                             ((uint32_t)(p.pt >> 3) << 17) | ((uint32_t)((kTileC << p.duo) >> 4) << 24);
      // completion of the MMAs issued so far, signalled on a barrier of this CTA -- and of its partner in a pair
      auto commit = [&](uint32_t bar) {
        if constexpr (DUO) { mma_commit_2cta(in_cta(bar, 0)); mma_commit_2cta(in_cta(bar, 1)); }
        else mma_commit(bar);
      };
      const uint32_t ni = (uint32_t)p.ni, nstages = (uint32_t)p.stages;
      const bool ring = !(p.strip && p.wres);                 // do the blocks travel through the stage ring?
      uint32_t tcount = 0, s = 0, ph = 0;
      auto advance = [&](uint32_t d) { s += d; while (s >= nstages) { s -= nstages; ph ^= 1u; } };
      if (ring) advance((uint32_t)iss);
      int b = iss;                                           // my next block of the current tile
      const uint32_t bmask = (1u << p.lg_bufs) - 1u;
      bool ok = true;
      const uint64_t desc_hi = smem_desc(0, p.bkb);           // everything but the start address
      const int ksteps = p.pairs ? 2 : p.bkb >> 5;
      const bool tail = !p.pairs && p.tail_steps != ksteps;              // a tap's last block holds fewer steps
      if (p.wres && !mbar_wait(smem_u32(&ctl.wfull), 0, &ctl, p.status, HQ_DEV_TIMEOUT_MMA)) ok = false;
      // One issuer, plain form: the lean loop (the hand-over chain of short reductions is latency bound, every
      // instruction on it counts).
      const bool lean = ni == 1 && !p.strip;
      auto lean_tiles = [&](auto tail_tag) {
        constexpr bool TAIL = decltype(tail_tag)::value;
      for (int p_tile = p_tile0; p_tile < p.p_tiles && ok; p_tile += p_step, ++tcount) {
        const uint32_t as = tcount & bmask, aph = (tcount >> p.lg_bufs) & 1u;
        // The operands of the tile's first K block have usually landed long ago; looking at them first
        // keeps that check off the path between the epilogue's hand-back and the first MMA.
        if (!mbar_wait(smem_u32(&ctl.full[s]), ph, &ctl, p.status, HQ_DEV_TIMEOUT_MMA)) { ok = false; break; }
        if (!mbar_wait(smem_u32(&ctl.tempty[as]), aph ^ 1u, &ctl, p.status, HQ_DEV_TIMEOUT_MMA)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + as * p.acc_stride;
        int chunk = 0;
        for (int kb = 0; kb < p.k_blocks; ++kb) {
          int nsteps = ksteps;
          if (TAIL && ++chunk == p.cchunks) { chunk = 0; nsteps = p.tail_steps; }
          if (kb > 0 && !mbar_wait(smem_u32(&ctl.full[s]), ph, &ctl, p.status, HQ_DEV_TIMEOUT_MMA)) { ok = false; break; }
          const uint32_t w_addr = tiles + s * stage_bytes;
          const uint32_t a_addr = p.wres ? tiles + p.wres_off + (uint32_t)kb * w_bytes : w_addr;
          uint64_t adesc = desc_hi | (uint64_t)((a_addr >> 4) & 0x3FFF);
          uint64_t bdesc = desc_hi | (uint64_t)(((w_addr + x_off) >> 4) & 0x3FFF);
          if constexpr (DUO) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
              if (k < nsteps) mma_i8_2cta(d_tmem, adesc + 2 * k, bdesc + 2 * k, idesc, k ? 1u : kb ? 1u : 0u);
          } else {
            for (int k = 0; k < nsteps; ++k, adesc += 2, bdesc += 2)     // 32 bytes of K per instruction
              mma_i8(d_tmem, adesc, bdesc, idesc, (kb | k) ? 1u : 0u);
          }
          // the accumulator's barrier first on the last K block: the epilogue is the one waiting
          if (kb + 1 == p.k_blocks) commit(smem_u32(&ctl.tfull[as]));
          commit(smem_u32(&ctl.empty[s]));         // frees the stage when these MMAs have read it
          if (++s == nstages) { s = 0; ph ^= 1u; }
        }
      }
      };
      if (lean) { if (tail) lean_tiles(std::true_type{}); else lean_tiles(std::false_type{}); }
      for (int p_tile = p_tile0; p_tile < p.p_tiles && ok && !lean; p_tile += p_step, ++tcount) {
        const uint32_t as = tcount & bmask, aph = (tcount >> p.lg_bufs) & 1u;
        const uint32_t d_tmem = tmem_base + as * p.pt;
        bool first = true;
        int cur_chunk = -1;
        uint32_t ps = 0;
        for (; b < p.k_blocks; b += (int)ni) {
          uint32_t a_addr, b_addr;
          if (p.strip) {
            // block b = (cin chunk, filter tap): the chunk's patch, read from (tr << lg_wp) + ts rows further on.
            // The start is then not aligned to the swizzle pattern's eight rows, which needs nothing more: the
            // pattern is a function of the shared-memory address, for the copy that wrote the patch and for the
            // MMA that reads it alike (the descriptor's base-offset field stays 0; a phase there gives wrong sums).
            const int chunk = p.pairs ? 0 : b / 9, tap = b - 9 * chunk, tr = p.pairs ? b >> 2 : tap / 3, ts = p.pairs ? b & 3 : tap - 3 * tr;
            if (chunk != cur_chunk) {
              if (cur_chunk >= 0) mma_commit(smem_u32(&ctl.pempty[ps]));    // my MMAs on the previous patch
              cur_chunk = chunk;
              const uint32_t pidx = tcount * (uint32_t)p.cchunks + (uint32_t)chunk;
              ps = pidx % (uint32_t)p.npatch;
              if (!mbar_wait(smem_u32(&ctl.pfull[ps]), (pidx / (uint32_t)p.npatch) & 1u, &ctl, p.status, HQ_DEV_TIMEOUT_MMA)) { ok = false; break; }
            }
            b_addr = tiles + p.patch_off + ps * p.patch_bytes + (uint32_t)(((tr << p.lg_wp) + ts) * p.bkb);
            if (p.pairs) {
              // pixel ts - 1 of the pair: second half of the pair before, the pair itself, first half of the pair after
              b_addr = tiles + p.patch_off + ps * p.patch_bytes + (uint32_t)(((tr << p.lg_wp) + ((ts + 1) >> 1)) * 128 + (((ts + 1) & 1) << 6));
              a_addr = tiles + p.wres_off + (uint32_t)(2 * tr + (ts >> 1)) * w_bytes + (uint32_t)((ts & 1) << 6);
            } else if (p.wres) {
              a_addr = tiles + p.wres_off + (uint32_t)(tap * p.cchunks + chunk) * w_bytes;
            } else {
              if (!mbar_wait(smem_u32(&ctl.full[s]), ph, &ctl, p.status, HQ_DEV_TIMEOUT_MMA)) { ok = false; break; }
              a_addr = tiles + s * stage_bytes;
            }
          } else {
            if (!mbar_wait(smem_u32(&ctl.full[s]), ph, &ctl, p.status, HQ_DEV_TIMEOUT_MMA)) { ok = false; break; }
            const uint32_t w_addr = tiles + s * stage_bytes;
            a_addr = p.wres ? tiles + p.wres_off + (uint32_t)b * w_bytes : w_addr;
            b_addr = w_addr + x_off;
          }
          if (first) {
            // The operands of this issuer's first block have usually landed long ago; looking at them first keeps
            // that check off the path between the epilogue's hand-back and the first MMA.
            if (!mbar_wait(smem_u32(&ctl.tempty[as]), aph ^ 1u, &ctl, p.status, HQ_DEV_TIMEOUT_MMA)) { ok = false; break; }
            if (b != 0 && !mbar_wait(smem_u32(&ctl.tstart[as]), aph, &ctl, p.status, HQ_DEV_TIMEOUT_MMA)) { ok = false; break; }
            tc_fence_after();
            first = false;
          }
          uint64_t adesc = desc_hi | (uint64_t)((a_addr >> 4) & 0x3FFF);
          uint64_t bdesc = desc_hi | (uint64_t)((b_addr >> 4) & 0x3FFF);
          for (int k = 0; k < ksteps; ++k, adesc += 2, bdesc += 2)     // 32 bytes of K per instruction
            mma_i8(d_tmem, adesc, bdesc, idesc, (b | k) ? 1u : 0u);
          if (b == 0 && ni > 1) { tc_fence_before(); mbar_arrive(smem_u32(&ctl.tstart[as])); }   // the overwriting MMA is on its way
          // the accumulator's barrier first on this issuer's last block: the epilogue is the one waiting
          if (b + (int)ni >= p.k_blocks) mma_commit(smem_u32(&ctl.tfull[as]));
          if (ring) {
            mma_commit(smem_u32(&ctl.empty[s]));     // frees the stage when these MMAs have read it
            advance(ni);                             // my next block, in this tile or the next
          }
        }
        if (!ok) break;
        if (p.strip && cur_chunk >= 0) mma_commit(smem_u32(&ctl.pempty[ps]));
        b -= p.k_blocks;                             // the numbering runs on into the next tile
      }
      // Drain: all issued MMAs must have completed before tensor memory is freed.
      if constexpr (DUO) mma_commit_2cta(in_cta(smem_u32(&ctl.drain), 0)); else mma_commit(smem_u32(&ctl.drain));
      const unsigned long long t0 = global_ns();
      while (!mbar_try_wait(smem_u32(&ctl.drain), 0)) {
        if (global_ns() - t0 > kWaitBudgetNs) { atomicCAS(p.status, 0u, (uint32_t)HQ_DEV_TIMEOUT_DRAIN); break; }
      }
    }
  } else if (FRAG && warp == 1 + MMA_WARPS + EPI_WARPS) {
    // ------------------------------------------------------------ store warp (frag): finished tiles leave by TMA
    // The buffer of a tile whose store has read it takes the residual of the tile 2^lg_rbufs later at once (one thread less
    // between the two, and the operand producer, whose own instructions are on the tiles' path, does not see residuals at all).
    if (elect_one()) {
      const uint32_t bufs = 1u << p.lg_rbufs, rmask = bufs - 1u;
      const bool res = p.staged_res != 0;
      const unsigned long long pol_first = policy_evict_first();
      uint32_t tcount = 0, loads = 0;
      int load_tile = p_tile0;
      auto next_residual = [&]() {
        if (load_tile >= p.p_tiles) return;
        const uint32_t rs = loads & rmask, bar = smem_u32(&ctl.rfull[rs]);
        mbar_expect_tx(bar, res_tile_bytes);
        tma_load_2d_hint(res_stage + rs * res_tile_bytes, &map_res, bar, c_tile * kTileC, tile_at(p, load_tile) * kTileC, pol_first);
        load_tile += p_step; ++loads;
      };
      if (res) {
        asm volatile("griddepcontrol.wait;" ::: "memory");              // the residual is the output of an earlier kernel
        for (uint32_t i = 0; i < bufs; ++i) next_residual();
      }
      for (int p_tile = p_tile0; p_tile < p.p_tiles; p_tile += p_step, ++tcount) {
        const uint32_t rs = tcount & rmask, rph = (tcount >> p.lg_rbufs) & 1u;
        if (!mbar_wait(smem_u32(&ctl.ofull[rs]), rph, &ctl, p.status, HQ_DEV_TIMEOUT_EPILOGUE)) break;
        tma_store_2d(&map_out, res_stage + rs * res_tile_bytes, c_tile * kTileC, tile_at(p, p_tile) * kTileC);
        tma_store_commit();
        // the store before this one has read its tile by now; with two buffers only, this one is awaited
        if (bufs < 4u) tma_store_wait_read0();
        else if (tcount > 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
        else continue;
        if (res) next_residual();
        else mbar_arrive(smem_u32(&ctl.rempty[(bufs < 4u ? tcount : tcount - 1u) & rmask]));
      }
      // every copy this thread started must have landed before the CTA may exit (all consumed unless a wait ran out)
      for (uint32_t k = tcount; k < loads; ++k) {
        const unsigned long long t0 = global_ns();
        while (!mbar_try_wait(smem_u32(&ctl.rfull[k & rmask]), (k >> p.lg_rbufs) & 1u)) {
          if (global_ns() - t0 > kWaitBudgetNs) { atomicCAS(p.status, 0u, (uint32_t)HQ_DEV_TIMEOUT_DRAIN); break; }
        }
      }
      tma_store_wait_all();
    }
  } else {
    // ------------------------------------------------------------ epilogue (the last EPI_WARPS warps)
    const int q = warp & 3;                       // the TMEM lane quarter this warp may read: channels 32q..32q+31
    const int ew = warp - (1 + MMA_WARPS);        // 0 .. EPI_WARPS - 1
    const int half = ew >> 2;                     // which share (of p.halves) of its lane quarter's pixel columns this warp owns
    // Channel tiles of at most 64 channels are folded: the weight rows are loaded twice, so accumulator
    // lanes 64-127 repeat lanes 0-63, and lane quarters 2-3 take the second half of the pixel columns
    // of channels 0-63 instead of idling on channels that do not exist.
    const int cq = p.fold ? (q & 1) : q;          // which 32 channels of the tile
    const int slices = p.halves << p.fold;        // pixel-column slices per channel quarter
    const int px_per_warp = p.pt / slices;        // 128 or 64 pixel columns; 32 or 16 with INT32 boxes
    const int col0 = ((p.fold ? (q >> 1) * p.halves : 0) + half) * px_per_warp;
    const int ch = c_tile * kTileC + cq * 32 + lane;         // this thread's output channel
    const bool ch_live = ch < p.C;
    const bool warp_live = (c_tile * kTileC + cq * 32) < p.C; // warp-uniform
    const int lo = p.relu ? (p.qmin > 0 ? p.qmin : 0) : p.qmin, hi = p.qmax;
    if (params_late) asm volatile("griddepcontrol.wait;" ::: "memory");     // (the constants below)

    if constexpr (WIDE) {
      if (half < p.halves) {
        EpiCtx e;
        e.p = &p; e.ctl = &ctl; e.map_out = &map_out; e.smem_raw = smem_raw; e.raw = raw; e.out_stage = out_stage;
        e.tmem_base = tmem_base; e.lane = lane; e.q = q; e.cq = cq; e.ew = ew; e.half = half;
        e.col0 = col0; e.px_per_warp = px_per_warp; e.ch = ch; e.c_tile = c_tile; e.p_tile0 = p_tile0; e.p_step = p_step;
        e.lo = lo; e.hi = hi; e.ch_live = ch_live; e.warp_live = warp_live;
        if constexpr (WIDE == kRaw32) {
          ChanConst k{};
          k.bias = (ch_live && p.bias) ? p.bias[ch] : 0;
          epilogue_loop_wide<3, false>(e, k, &map_res, &map_q);
        } else {
          const ChanConst k = chan_const(p, ch, false);
          const int qc = p.q_out && ch_live ? p.qc[ch] : 32;
          const bool form1 = __all_sync(0xffffffffu, qc >= 32) != 0;
          const bool form0 = form1 && __all_sync(0xffffffffu, k.sh >= 32 && k.rsh >= 32) != 0;
          asm volatile("griddepcontrol.wait;" ::: "memory");           // the residual is the output of an earlier kernel
          if (p.q_out) {
            if (form0) epilogue_loop_wide<0, true>(e, k, &map_res, &map_q);
            else if (form1) epilogue_loop_wide<1, true>(e, k, &map_res, &map_q);
            else epilogue_loop_wide<2, true>(e, k, &map_res, &map_q);
          } else {
            if (form0) epilogue_loop_wide<0, false>(e, k, &map_res, &map_q);
            else epilogue_loop_wide<1, false>(e, k, &map_res, &map_q);
          }
        }
      }
    } else {
    // per-channel constants, once per kernel (spelled out: through chan_const the loops compile worse, ResNet-50 INT8 2.11 -> 2.25 ms)
    ChanConst k{};
    uint32_t fast = (p.out_bits != 32) ? 1u : 0u;
    const int pch = p.pairs ? ch & 63 : ch;       // (pixel pairs: both outputs of a pair have the layer's channels)
    k.bias = (ch_live && p.bias) ? p.bias[pch] : 0;
    if (p.out_bits != 32) {
      k.b = ch_live ? p.b[pch] : 0;
      const int cc = ch_live ? p.c[pch] : 32;
      k.sh = cc;
      k.r0 = (long long)k.bias * (long long)k.b + (1LL << (cc - 1));
      if (p.res) {
        const int rcc = ch_live ? p.rc[ch] : 32;
        if (rcc < 9 || p.res_bits != 8) fast = 0;
        k.rb = ch_live ? p.rb[ch] : 0;
        k.rsh = rcc;
        k.rr0 = 1LL << (rcc - 1);
      }
    }
    fast = epi_bar_and<32 * EPI_WARPS>(fast);                    // every live channel of the CTA allows 32-bit intermediates
    const bool warp_small = __any_sync(0xffffffffu, k.sh < 32) != 0;     // some channel of this warp has c < 32
    // ... and for each of them accumulator and bias stay below 2^(c-2): the pre-shift form of requant_fast is exact
    // and its result below 2^30 in magnitude, so that the residual term still adds without overflow
    const int babs = k.bias < 0 ? ~k.bias : k.bias;
    const bool warp_pre = warp_small &&
        __all_sync(0xffffffffu, k.sh >= 32 || (k.sh - 2 >= p.acc_bits && k.sh >= 3 && babs < (1 << (k.sh - 2)))) != 0;
    if (fast) {
      k.sh1 = k.sh < 32 ? k.sh : 32;
      k.cmin31 = k.sh < 31 ? k.sh : 31;
      k.sh -= k.sh1;
      k.pre = 32 - k.sh1;                        // (r0 is shifted by the loops that use the pre-shift form)
      if (p.res) {
        if (k.rsh >= 40) { k.rb = 0; k.rh = 0; k.rsh = 1; }            // |r*rb| < 2^39: rounds to 0
        else { k.rh = 1 << (k.rsh - 9); k.rsh -= 8; }
      }
    }
    // narrow residual pairs, when the caller prepared them and every channel of this warp has one
    bool warp_narrow = false;
    if (fast && (!warp_small || warp_pre) && p.res && p.res_narrow) {
      if (p.narrow_fresh) asm volatile("griddepcontrol.wait;" ::: "memory");
      const int4 nr = ch_live ? p.res_narrow[ch] : make_int4(0, 0, 0, 1);
      warp_narrow = __all_sync(0xffffffffu, nr.w != 0) != 0;
      if (warp_narrow) { k.rb = nr.x; k.rh = nr.y; k.rsh = nr.z; }
    }

    if (p.res && !p.staged_res) asm volatile("griddepcontrol.wait;" ::: "memory");   // direct residual loads below
    EpiCtx e;
    e.p = &p; e.ctl = &ctl; e.map_out = &map_out; e.smem_raw = smem_raw; e.raw = raw; e.out_stage = out_stage;
    e.res_stage = res_stage; e.res_tile_bytes = res_tile_bytes; e.tmem_base = tmem_base;
    e.warp = warp; e.lane = lane; e.q = q; e.cq = cq; e.ew = ew; e.half = half; e.col0 = col0; e.px_per_warp = px_per_warp; e.ch = ch;
    e.c_tile = c_tile; e.p_tile0 = p_tile0; e.p_step = p_step; e.lo = lo; e.hi = hi;
    e.ch_live = ch_live; e.warp_live = warp_live;
    if constexpr (FRAG) {
        const bool rn = warp_narrow, os = p.out_signed != 0, rs = p.res_signed != 0;
        // (narrow residual pairs only with the plain and the pre-shift form; the funnel-shift form keeps the multiply-high term)
#define HQ_FRAG(S, OS) do { \
          if (!p.res) { if (!warp_small) epilogue_loop_frag<false, false, false, S, OS, false, 0>(e); \
                        else if (warp_pre) epilogue_loop_frag<false, false, false, S, OS, false, 2>(e); \
                        else epilogue_loop_frag<false, false, false, S, OS, false, 1>(e); } \
          else if (warp_small && !warp_pre) { if (rs) epilogue_loop_frag<true, false, true, S, OS, false, 1>(e); else epilogue_loop_frag<true, false, false, S, OS, false, 1>(e); } \
          else if (warp_small) { if (rs) HQ_FRAG_RES(true, S, OS, 2); else HQ_FRAG_RES(false, S, OS, 2); } \
          else { if (rs) HQ_FRAG_RES(true, S, OS, 0); else HQ_FRAG_RES(false, S, OS, 0); } } while (0)
#define HQ_FRAG_RES(RS, S, OS, SM) do { if (rn) epilogue_loop_frag<true, false, RS, S, OS, true, SM>(e); \
                                        else epilogue_loop_frag<true, false, RS, S, OS, false, SM>(e); } while (0)
        if (!fast) {
          if (os) { if (rs) epilogue_loop_frag<true, true, true, false, true, false>(e); else epilogue_loop_frag<true, true, false, false, true, false>(e); }
          else { if (rs) epilogue_loop_frag<true, true, true, false, false, false>(e); else epilogue_loop_frag<true, true, false, false, false, false>(e); }
        } else if (p.sat_pack) { if (os) HQ_FRAG(true, true); else HQ_FRAG(true, false); }
        else { if (os) HQ_FRAG(false, true); else HQ_FRAG(false, false); }
#undef HQ_FRAG_RES
#undef HQ_FRAG
    } else {
    if (half >= p.halves) {
      // the 64-pixel tile has one 64-column slice per lane quarter: this warp only took part in the vote above
    } else if (fast && p.staged_out && p.out_bits == 4 && !p.res && !p.strip && lo >= 0 && hi <= 15) {
      // unsigned 4-bit outputs without a residual (the convs inside a 4-bit block)
      if (warp_pre) epilogue_loop_fast8<false, false, false, false, 2, false, true>(e, k);
      else if (warp_small) epilogue_loop_fast8<false, false, false, false, 1, false, true>(e, k);
      else epilogue_loop_fast8<false, false, false, false, 0, false, true>(e, k);
    } else if (fast && p.staged_out && p.out_bits == 8 && (!p.res || p.staged_res)) {
      const int variant = (p.res ? 4 : 0) | ((p.res && p.res_signed) ? 2 : 0) | (p.sat_pack ? 1 : 0);
      switch (variant) {
#define HQ_FAST8(R, RS, S, OS) do { if (warp_pre && R && warp_narrow) epilogue_loop_fast8<R, RS, S, OS, 2, R>(e, k); \
                                    else if (warp_pre) epilogue_loop_fast8<R, RS, S, OS, 2, false>(e, k); \
                                    else if (warp_small) epilogue_loop_fast8<R, RS, S, OS, 1, false>(e, k); \
                                    else if (R && warp_narrow) epilogue_loop_fast8<R, RS, S, OS, 0, R>(e, k); \
                                    else epilogue_loop_fast8<R, RS, S, OS, 0, false>(e, k); } while (0)
        case 0: HQ_FAST8(false, false, false, false); break;
        case 1: if (p.out_signed) HQ_FAST8(false, false, true, true); else HQ_FAST8(false, false, true, false); break;
        case 4: HQ_FAST8(true, false, false, false); break;
        case 5: if (p.out_signed) HQ_FAST8(true, false, true, true); else HQ_FAST8(true, false, true, false); break;
        case 6: HQ_FAST8(true, true, false, false); break;
        default: if (p.out_signed) HQ_FAST8(true, true, true, true); else HQ_FAST8(true, true, true, false); break;
#undef HQ_FAST8
      }
    } else {
      epilogue_loop_general(e, k, fast);
    }
    }
    }
  }


  tc_fence_before();
  __syncthreads();
  // A pair leaves together: the leading CTA has seen its MMAs complete (they read the partner's shared memory and
  // signal its barriers), the partner has sent its last remote arrival.
  if constexpr (DUO) cluster_sync_all();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    if constexpr (DUO) tmem_dealloc2(tmem_base, p.tmem_cols); else tmem_dealloc(tmem_base, p.tmem_cols);
  }
}

// ---------------------------------------------------------------- narrow residual pairs ------
// The residual term dn(r, rb, rc) = (r*rb + 2^(rc-1)) >> rc (Section 3.3, Appendix G) has only 256 possible
// inputs per channel.  For most (rb, rc) a 23-bit multiplier m ~ rb / 2^8 with s = rc - 8 and a = 2^(s-1)
// gives (r*m + a) >> s == dn(r, rb, rc) for every one of them, and r*m + a fits 32 bits.  One warp per
// channel tries the two neighbouring multipliers and checks all 256 inputs; channels without such a pair
// are marked invalid and keep the wide form.  Run once per layer when a network is built, and ahead of a
// single large element-wise call.
struct NarrowJob { const int32_t* rb; const int32_t* rc; int is_signed; int4* out; };

__global__ void __launch_bounds__(128) residual_narrow_kernel(NarrowJob j0, NarrowJob j1, int n) {
  hq_pdl_entry();
  // one warp per channel: lane l checks the inputs l, l + 32, ... for both candidate multipliers; warps past the
  // first n channels serve the second job (the other operand of an element-wise call), if there is one
  int ch = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const bool second = ch >= n;
  if (second) ch -= n;
  const NarrowJob& j = second ? j1 : j0;
  if (ch >= n || !j.out) return;
  const long long b = j.rb[ch];
  const int c = j.rc[ch];
  int4 res = make_int4(0, 0, 0, 0);
  const int r_lo = j.is_signed ? -128 : 0;
  if (c >= 41 && c <= 62) {
    res = make_int4(0, 0, 0, 1);                       // |r*rb| < 2^39 <= 2^(rc-2): the term is 0 for every r
  } else if (c >= 9 && c <= 38) {
    const int s = c - 8, a = 1 << (s - 1);
    const long long m0 = b >> 8, m1 = m0 + 1;
    bool same0 = m0 <= (1 << 23), same1 = m1 <= (1 << 23);
    for (int k = 0; k < 8; ++k) {
      const int r = r_lo + lane + 32 * k;
      const long long exact = ((long long)r * b + (1LL << (c - 1))) >> c;
      same0 = same0 && exact == (long long)((r * (int)m0 + a) >> s);
      same1 = same1 && exact == (long long)((r * (int)m1 + a) >> s);
    }
    same0 = __all_sync(0xffffffffu, same0);
    same1 = __all_sync(0xffffffffu, same1);
    if (same0) res = make_int4((int)m0, a, s, 1);
    else if (same1) res = make_int4((int)m1, a, s, 1);
  }
  if (lane == 0) j.out[ch] = res;
}

// Pixel tile: the largest of 256 / 128 / 64 that still gives every SM work, at most `cap`.
int pick_pt(long long pixels, int c_tiles, int sm_count, int cap) {
  const int cands[3] = {256, 128, 64};
  for (int i = 0; i < 3; ++i) {
    const int pt = cands[i];
    if (pt > cap) continue;
    const long long tiles = (pixels + pt - 1) / pt * c_tiles;
    if (tiles >= 2LL * sm_count || pt == 64) return pt;
  }
  return 64;
}

}  // namespace

// One-time set-up that must not happen inside a stream capture: driver entry points for the
// tensor-map encoders and the kernel's dynamic shared-memory limit.
bool hq_conv_tc_init() {
  if (!load_driver_entry_points()) return false;
  return cudaFuncSetAttribute(conv_tc_kernel<kSoloEpilogueWarps, 1, kSoloIssuerWarps>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              kSmemAttr) == cudaSuccess &&
         cudaFuncSetAttribute(conv_tc_kernel<kPairEpilogueWarps, 2, kPairIssuerWarps>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              112 * 1024) == cudaSuccess &&
         cudaFuncSetAttribute(conv_tc_kernel<kFragWarps, 1, kFragIssuers, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemAttr) == cudaSuccess &&
         cudaFuncSetAttribute(conv_tc_kernel<kWideWarps, 1, kSoloIssuerWarps, false, false, kRaw32>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              kSmemAttr) == cudaSuccess &&
         cudaFuncSetAttribute(conv_tc_kernel<kWideWarps, 1, kSoloIssuerWarps, false, false, kAdd32>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              kSmemAttr) == cudaSuccess &&
         cudaFuncSetAttribute(conv_tc_kernel<kSoloEpilogueWarps, 1, 1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              kSmemAttr) == cudaSuccess;
}

bool hq_conv_tc_supported(const ConvArgs& a) {
  if (a.in_bits != 8) return false;
  if (a.cin % 16 != 0) return false;
  if (a.kh > 255 || a.kw > 255 || a.pad > 127 || a.stride > 8) return false;
  if ((long long)a.n * a.ho * a.wo >= (1ll << 31) - 256) return false;
  if ((long long)a.kh * a.kw * a.cin >= (1ll << 24)) return false;
  if (a.out_bits == 4 && (a.cout & 1)) return false;
  if (a.res && !(a.res_bits == 8 || a.res_bits == 32)) return false;
  // the corners of an im2col-mode tensor map are 8-bit signed offsets: wider filters are declined here, before any
  // map is encoded (more channel tiles than the GPU has SMs are declined by the launcher, which knows the count)
  const int pad_after = a.pad + a.pad_after_delta;
  if (pad_after - (a.kw - 1) < -128 || pad_after - (a.kh - 1) < -128 || pad_after > 127) return false;
  return true;
}

// im2col-mode tensor maps over activation tensors smaller than 128 KiB returned wrong tiles on the driver this
// library was brought up on (the map encoder marks such tensors in a field of the opaque descriptor).  Instead of
// editing the descriptor, layers that would need such a map are not run by the direct kernel at all: the kernel for small
// problems gathers their activations (conv_small.cu), and what it does not take goes through the patch-matrix form
// (lowering.cu), whose 1x1 convolution uses a plain tiled map.  Inside a network the map is declared large enough instead.
bool hq_conv_tc_small_im2col(const ConvArgs& a) {
  const bool tiled = !a.pitch_w && a.kh == 1 && a.kw == 1 && a.stride == 1 && a.pad == 0;
  if (tiled || a.in_slack) return false;              // (with room behind the tensor the map is declared large enough)
  const long long span = a.pitch_n ? (long long)a.n * a.pitch_n : (long long)a.n * a.h * a.w * a.cin;
  return span < kIm2colMinTensorBytes;
}

// Filters over channel counts that are not a multiple of 32: the direct kernel fetches every tap's short row anew for every
// tile of output channels, the patch matrix pays once for long rows.  In cycles per output pixel and SM, from launches of both
// forms: a direct row costs 5 (up to 64 bytes) or 7, a patch row 7, building the matrix K / 16.  Direct: 5x5 over 48 channels to 64
// 135 us against 161; patches: 3x3 over 48 channels to 1664 66 us against 81.
static bool prefers_patches(const ConvArgs& a) {
  if (a.cin % 32 == 0 || a.kh * a.kw == 1 || a.pitch_w || a.pairs || !hq_conv_lowering_applies(a)) return false;
  const long long K = (long long)a.kh * a.kw * a.cin, tiles = (a.cout + kTileC - 1) / kTileC;
  const int bkb = hq_conv_bkb(a.cin);
  const long long direct_rows = (long long)a.kh * a.kw * ((a.cin + bkb - 1) / bkb), patch_rows = (K + 127) / 128;
  return tiles * (direct_rows * (bkb < 128 ? 5 : 7) - 7 * patch_rows) > K / 16;
}
bool hq_conv_tc_declines(const ConvArgs& a) { return hq_conv_tc_small_im2col(a) || prefers_patches(a); }

bool hq_conv_wide_applies(const ConvArgs& a, int sm_count) {
  // (the smallest tile with its weights in the stages always leaves room for three of them beside the boxes)
  static_assert(kSmemBudget - kWideWarps * (kWideSlots * kWideBox + 2 * kWideQBox) >= 3 * (kTileC + 64) * 128, "stages of the INT32 shape");
  return hq_conv_tc_supported(a) && !hq_conv_tc_declines(a) && a.cout % 16 == 0 && (a.cout + kTileC - 1) / kTileC <= sm_count;
}

namespace {
// Launch shape of a layer and what it needs: host arithmetic on sizes alone (no pointer is looked at but for being NULL).
struct TcPlan {
  TcParams p{};
  bool pair = false, int32_boxes = false;
  int stages = 0, stage_bytes = 0, res_tile_bytes = 0, out_tile_bytes = 0, wres_bytes = 0;
  size_t patch_total = 0, dyn_smem = 0;
};

hq_status plan_conv_tc(const ConvArgs& a, int sm_count, int conv_path, TcPlan& t) {
  TcParams& p = t.p;
  const long long P = (long long)a.n * a.ho * a.wo;
  p.P = (int32_t)P; p.C = a.cout; p.howo = a.ho * a.wo; p.wo = a.wo;
  p.stride = a.stride; p.pad = a.pad; p.kw = a.kw;
  auto set_bkb = [&](int bkb) { p.bkb = bkb; p.cchunks = (a.cin + bkb - 1) / bkb; p.k_blocks = a.kh * a.kw * p.cchunks; };
  p.cin = a.cin;
  set_bkb(hq_conv_bkb(a.cin));
  p.c_tiles = (a.cout + kTileC - 1) / kTileC;
  if (p.c_tiles > sm_count) return HQ_ERR_UNSUPPORTED;
  // outputs and 8-bit residuals whose rows are 16-byte multiples travel through TMA
  const long long out_row_bytes = (long long)a.cout * a.out_bits / 8;
  p.staged_out = (a.out_bits != 32 && out_row_bytes % 16 == 0) ? 1 : 0;
  p.staged_res = (p.staged_out && a.res && a.res_bits == 8 && a.cout % 16 == 0) ? 1 : 0;
  // Launch shape: pair (two CTAs per SM) for short reductions when the tile pipeline fits half an SM.
  const long long k_total = (long long)a.kh * a.kw * a.cin;
  // INT32 results through TMA boxes (epilogue_loop_wide): every residual add, and raw results but for the long reductions
  // that the two-CTA shape serves better (and rows that are not whole 16-byte pieces)
  const bool int32_boxes = a.wide || (a.out_bits == 32 && !a.res && a.cout % 4 == 0 && k_total < 2048);
  t.int32_boxes = int32_boxes;
  const int box_bytes = kWideWarps * (kWideSlots * kWideBox + (a.wide && a.wide->q ? 2 * kWideQBox : 0));
  // (measured: with the weight slab resident the one-CTA shape catches up for K >= 128; the pair shape still
  // wins on the fused-residual expansions with the shortest reduction, and loses where a tile carries little
  // epilogue work, e.g. 64 output channels.  Where the layer is large enough for 256-pixel tiles and its residual
  // travels by TMA, the frag shape below is faster still: 64 -> 256 at 56x56, batch 256: 129 -> 97 us.)
  const bool frag_fits = p.staged_res && a.out_bits == 8 && a.cout > 64 && pick_pt(P, p.c_tiles, sm_count, 256) == 256;
  // Without a residual the frag shape takes over where a CTA's weights stay in shared memory, but for longer reductions whose
  // pixel rows the im2col mode gathers: four blocks of 128 pixels are issued more slowly than two of 256 (256 images, L2 flushed,
  // 256-pixel tiles against frag: 1x1 64 -> 256 at 56x56 90 / 69 us, 512 -> 128 at 28x28 32.7 / 27.7, 256 -> 128 / 2 28.7 / 22.0, 256 -> 512 / 2
  // 55.3 / 54.3, 512 -> 1024 / 2 36.8 / 46.1).
  const bool tiled = !a.pitch_w && a.kh == 1 && a.kw == 1 && a.stride == 1 && a.pad == 0;
  const bool plain_frag = !a.res && !a.pitch_w && !a.pairs && a.cout % 16 == 0 && (tiled || k_total <= 256);
  bool& pair = t.pair;
  pair = !a.wide && k_total <= 64 && a.res != nullptr && a.res_bits == 8 && a.cout >= 128 && !frag_fits;
  int &stages = t.stages, &stage_bytes = t.stage_bytes, &res_tile_bytes = t.res_tile_bytes, &out_tile_bytes = t.out_tile_bytes, &wres_bytes = t.wres_bytes;
  if (pair) {
    // 128-pixel tiles, two accumulator buffers (256 columns), K blocks of at most 64 bytes
    if (p.bkb > 64) set_bkb(64);
    p.pt = pick_pt(P, p.c_tiles, 2 * sm_count, 128);
    wres_bytes = p.k_blocks * kTileC * p.bkb;
    p.wres = wres_bytes <= 16 * 1024 ? 1 : 0;              // short reductions: the weight slab stays resident
    if (!p.wres) wres_bytes = 0;
    stage_bytes = ((p.wres ? 0 : kTileC) + p.pt) * p.bkb;
    p.fold = (a.cout <= 64 && p.pt >= 128) ? 1 : 0;
    p.halves = 1;
    p.lg_bufs = 1;
    p.lg_rbufs = 1;
    out_tile_bytes = p.staged_out ? kPairEpilogueWarps * p.pt * 32 : 0;
    res_tile_bytes = p.staged_res ? p.pt * kTileC : 0;
    stages = (110 * 1024 - out_tile_bytes - 2 * res_tile_bytes - wres_bytes) / stage_bytes;
    if (stages < 3 || p.pt < 128) pair = false;
  }
  if (!pair) {
    set_bkb(hq_conv_bkb(a.cin));
    const int smem_budget = kSmemBudget;                // dynamic bytes after the 1024-byte alignment slack
    // staging: 8 warps x pt/2 pixel rows x 32 bytes (reserved at the 8-bit size), residual 2 or 4 x [pt][128]
    bool chosen = false;
    for (int cap = int32_boxes && a.cout > 64 ? 128 : 256; cap >= 64 && !chosen; cap >>= 1) {   // largest pixel tile that leaves room for >= 3 stages
      p.pt = pick_pt(P, p.c_tiles, sm_count, cap);
      // A weight slab of at most 72 KiB stays resident (the stages then hold activations only): a third less
      // traffic into shared memory per K block.  Where the slab would cost the larger pixel tile its stages, the
      // tile wins and the weights travel with the stages.
      for (int keep_w = 1; keep_w >= 0 && !chosen; --keep_w) {
        wres_bytes = p.k_blocks * kTileC * p.bkb;
        p.wres = (keep_w && wres_bytes <= 72 * 1024) ? 1 : 0;
        if (!p.wres) { if (keep_w) continue; wres_bytes = 0; }
        stage_bytes = ((p.wres ? 0 : kTileC) + p.pt) * p.bkb;
        p.fold = (a.cout <= 64 && p.pt >= 128) ? 1 : 0;
        p.halves = int32_boxes ? 4 : p.pt >= (p.fold ? 256 : 128) ? 2 : 1;
        out_tile_bytes = int32_boxes ? box_bytes : p.staged_out ? 4 * p.pt * 32 : 0;
        p.lg_bufs = p.pt <= 128 ? 2 : 1;
        res_tile_bytes = p.staged_res ? p.pt * kTileC : 0;
        // residual tiles: as many buffers as accumulators, fewer when a long reduction needs the room for stages
        // (its epilogue has slack: a single residual buffer only delays the next tile's prefetch)
        // The frag shape (below) works in place in the residual tiles and needs no staging box; with the
        // weights resident two stages are enough for its short reductions (the epilogue bounds the tile).
        const bool frag_here = p.pt == 256 && !p.fold && p.staged_out && a.out_bits == 8 && (p.staged_res || (plain_frag && p.wres)) && k_total < 1024;
        if (frag_here) out_tile_bytes = 0;
        const int min_stages = (frag_here && p.wres) ? 2 : 3;
        for (p.lg_rbufs = p.lg_bufs; ; --p.lg_rbufs) {
          stages = (smem_budget - out_tile_bytes - (res_tile_bytes << p.lg_rbufs) - wres_bytes) / stage_bytes;
          if (stages >= min_stages || p.lg_rbufs == 0 || !res_tile_bytes || k_total < 1024) break;
        }
        if (stages >= min_stages || (p.pt == 64 && keep_w == 0)) chosen = true;
      }
    }
  }
  p.p_tiles = (int32_t)((P + p.pt - 1) / p.pt);
  // Strip mode for 3x3 / stride 1 / pad 1: one padded input patch per cin chunk serves all nine taps (a tap is a
  // row offset into the patch), so the activations enter shared memory once instead of nine times.  The tile is
  // 256 positions of a raster whose pitch is the next power of two above the padded width; worth it while at
  // least three quarters of a pitch are real columns.
  size_t& patch_total = t.patch_total;
  {
    int lg_wp = 0;
    if (a.w >= 11 && a.w <= 14) lg_wp = 4; else if (a.w >= 23 && a.w <= 30) lg_wp = 5; else if (a.w >= 47 && a.w <= 62) lg_wp = 6;
    const bool shape_ok = !pair && lg_wp && a.kh == 3 && a.kw == 3 && a.stride == 1 && a.pad == 1 && !a.pitch_w && !a.res &&
                          p.staged_out && a.out_bits == 8 && a.cin % 64 == 0 && a.n < 65536;
    if (shape_ok) {
      const int bkb = a.cin % 128 == 0 ? 128 : 64;
      const int cchunks = a.cin / bkb, rows = 256 >> lg_wp, tpi = (a.h + rows - 1) / rows;
      const long long tiles_all = (long long)a.n * tpi * p.c_tiles;
      const size_t patch = (size_t)(rows + 3) * (1u << lg_wp) * bkb, wb = (size_t)kTileC * bkb;
      const size_t slab = (size_t)(a.pairs ? 6 : 9 * cchunks) * wb;
      const bool keep_w = slab <= 72 * 1024 || a.pairs;
      const size_t room = (size_t)kSmemBudget - 32 * 1024 - (keep_w ? slab : 0);
      int npatch = 0, wstages = 0;
      if (keep_w) { npatch = (int)(room / patch); if (npatch > 3) npatch = 3; }
      else if (room >= 2 * patch + 3 * wb) { npatch = 2; wstages = (int)((room - 2 * patch) / wb); }
      // measured: with the weights streaming through the stage ring the strip form is no faster than the plain
      // one (both are bound by what the SM can take in per cycle), so it is used where the weights stay resident
      if (((tiles_all >= 2LL * sm_count && keep_w) || conv_path == 3 || a.pairs) && npatch >= 2) {
        p.strip = 1; p.lg_wp = lg_wp; p.rows = rows; p.tpi = tpi; p.ho = a.h; p.npatch = npatch;
        p.patch_bytes = (uint32_t)patch;
        p.bkb = bkb; p.cchunks = cchunks; p.k_blocks = a.pairs ? 12 : 9 * cchunks;
        p.pairs = a.pairs;
        p.pt = 256; p.lg_bufs = 1; p.lg_rbufs = 1; p.halves = 2;
        p.fold = a.cout <= 64 ? 1 : 0;
        p.wres = keep_w ? 1 : 0;
        wres_bytes = keep_w ? (int)slab : 0;
        stage_bytes = keep_w ? 0 : (int)wb;
        stages = keep_w ? 0 : (wstages > kMaxStages ? kMaxStages : wstages);
        out_tile_bytes = 4 * 256 * 32;
        res_tile_bytes = 0;
        p.p_tiles = a.n * tpi;
        patch_total = (size_t)npatch * patch;
      }
    }
  }
  // The direct kernel fetches activations through an im2col-mode map unless the layer is 1x1 / stride 1 / unpadded
  // (tiled map) or takes the strip form (tiled map over padded patches).  That mode is not used on tensors below
  // 128 KiB (hq_conv_tc_small_im2col); such a layer is declined here.
  if ((!p.strip && hq_conv_tc_declines(a)) || (a.pairs && !p.strip)) return HQ_ERR_UNSUPPORTED;
  p.x_signed = a.in_signed;
  bool frag = false;
  {
    // issuer warps in use: at most one per K block; where the blocks travel through the stage ring, the stage count
    // becomes a multiple of it (every stage then belongs to one issuer)
    // Measured: several issuers pay off where the operands are mostly in shared memory already (strip form,
    // resident weights); where every block waits for 48 KiB from L2 the tile is bound by that stream and the extra
    // issuers only cost a few percent.
    // Third launch shape, *frag*, for the fused 8-bit residual with a short reduction on layers large enough for
    // 256-pixel tiles (the condition it shares with the tile choice above): see epilogue_loop_frag.
    frag = !pair && !p.strip && p.pt == 256 && !p.fold && p.staged_out && a.out_bits == 8 &&
           (p.staged_res || (plain_frag && p.wres)) && k_total < 1024;
    if (frag) {
      // 128-pixel tiles, four accumulators; the residual tiles double as the output boxes
      p.frag = 1; p.halves = 2;
      p.pt = 128; p.lg_bufs = 2; p.lg_rbufs = 1;
      p.p_tiles = (int32_t)((P + p.pt - 1) / p.pt);
      out_tile_bytes = 0;
      res_tile_bytes = p.pt * kTileC;
      wres_bytes = p.k_blocks * kTileC * p.bkb;
      p.wres = wres_bytes <= 72 * 1024 ? 1 : 0;
      if (!p.wres) wres_bytes = 0;
      stage_bytes = ((p.wres ? 0 : kTileC) + p.pt) * p.bkb;
      // Eight residual / output tiles where a tile is one or two K blocks, else four: a tile is held from its load to the end of its
      // store, and the loads of the next tiles must be in flight meanwhile to cover the memory latency (inside ResNet-50 at 256 images,
      // four / eight tiles: 128 -> 512 at 28x28 65 / 55 us, 256 -> 1024 at 14x14 39 / 34; a call of 64 -> 256 at 56x56 134 / 128).  Longer
      // tiles cover it by themselves and need the room for stages: with the three that eight tiles leave, the second issuer has none
      // of its own (calls of 256 images, eight / four tiles: 3x3 64 -> 256 at 28x28 85 / 79 us; 1x1 768 -> 1024 at 14x14, weights streaming,
      // 74 / 68; 384 -> 768 at 28x28, 128 images, 62 / 54).
      // Without a residual the tiles only carry outputs, and what is in flight are the operand stages: as many as there may be.
      for (p.lg_rbufs = p.staged_res && p.k_blocks <= 2 ? 3 : 2; ; --p.lg_rbufs) {
        stages = (kSmemBudget - (res_tile_bytes << p.lg_rbufs) - wres_bytes) / stage_bytes;
        if (p.staged_res || stages >= kMaxStages || p.lg_rbufs == 1) break;
      }
    }
    // Fourth shape, *duo*: clusters of two CTAs on adjacent SMs share every MMA (cta_group::2, M = 256): each CTA
    // fetches its own 128 weight rows and HALF of the tile's pixel rows, 32 KiB per K block and SM instead of
    // 48 KiB for the same MMA time.  For the long reductions whose weights stream, which the operand fetch bounds.
    p.duo = (!pair && !frag && !int32_boxes && !p.strip && !p.wres && !p.fold && p.pt >= 128 && p.bkb == 128 && a.cout % 256 == 0 &&
             k_total >= 2048 && (long long)p.p_tiles * p.c_tiles >= 2LL * sm_count) ? 1 : 0;
    if (p.duo) {
      stage_bytes = (kTileC + p.pt / 2) * p.bkb;
      stages = (kSmemBudget - out_tile_bytes - (res_tile_bytes << p.lg_rbufs)) / stage_bytes;
    }
    // (the dealt loop knows whole K blocks only: channels that do not fill their last block take the single issuer)
    const bool tail = a.cin % p.bkb > 0 && a.cin % p.bkb <= p.bkb - 32;
    const int issuers = pair ? kPairIssuerWarps : (p.strip || (p.wres && !tail)) ? kSoloIssuerWarps : 1;
    p.ni = p.k_blocks < issuers ? p.k_blocks : issuers;
    if (frag) {
      if (stages > kMaxStages) stages = kMaxStages;
      p.ni = kFragIssuers;
      // (a stage has to stay with one issuer, see frag_issue)
      if (stages >= kFragAccs * p.k_blocks) stages -= stages % (kFragIssuers * p.k_blocks);
      else if (stages >= 4 && p.k_blocks > 1) { p.deal = 1; stages -= stages % kFragIssuers; }
      else p.ni = 1;
    } else if (!(p.strip && p.wres)) {
      while (p.ni > 1 && stages < p.ni) --p.ni;
      if (stages > kMaxStages) stages = kMaxStages;
      // every stage counts more than the third issuer: the bytes in flight set the tile rate of the layers that wait
      // on memory latency (first layer: three 32 KiB stages 163 us, four with two issuers 143 us)
      while (p.ni > 1 && stages % p.ni) --p.ni;
      stages -= stages % p.ni;
    }
  }
  p.acc_stride = p.pt;
  p.w_blocks = p.pairs ? 6 : p.k_blocks;
  p.tail_steps = (a.cin - (p.cchunks - 1) * p.bkb + 31) >> 5;
  { const long long bound = k_total * 255 * 128; int bits = 0; while ((1LL << bits) <= bound) ++bits; p.acc_bits = bits; }
  p.tmem_cols = (uint32_t)(p.acc_stride << p.lg_bufs);  // 512 columns, or 256 for the smallest tile
  if (stages > kMaxStages) stages = kMaxStages;
  if (stages < 2 && !p.strip) return HQ_ERR_UNSUPPORTED;
  p.stages = stages;
  p.out_stage_off = (uint32_t)(stages * stage_bytes);             // all pieces are multiples of 1024 bytes
  p.res_stage_off = p.out_stage_off + (uint32_t)out_tile_bytes;
  p.wres_off = p.res_stage_off + ((uint32_t)res_tile_bytes << p.lg_rbufs);
  p.patch_off = p.wres_off + (uint32_t)wres_bytes;
  t.dyn_smem = (size_t)stages * stage_bytes + out_tile_bytes + ((size_t)res_tile_bytes << p.lg_rbufs) + wres_bytes + patch_total + 1024;
  return HQ_OK;
}
}  // namespace

hq_status hq_conv_tc_plan(const ConvArgs& a, int sm_count, hq_conv_plan* out) {
  if (!hq_conv_tc_supported(a)) return HQ_ERR_UNSUPPORTED;
  TcPlan t;
  const hq_status st = plan_conv_tc(a, sm_count, 0, t);
  if (st != HQ_OK) return st;
  const TcParams& p = t.p;
  out->shape = p.frag ? HQ_SHAPE_FRAG : p.duo ? HQ_SHAPE_DUO : t.pair ? HQ_SHAPE_PAIR : t.int32_boxes ? HQ_SHAPE_WIDE : p.strip ? HQ_SHAPE_STRIP : HQ_SHAPE_SOLO;
  out->pixel_tile = p.pt; out->k_blocks = p.k_blocks; out->block_bytes = p.bkb; out->weights_resident = p.wres;
  out->stages = p.stages; out->issuers = p.ni; out->alternate_tiles = p.frag && !p.deal;
  out->residual_tiles = p.frag || p.staged_res ? 1 << p.lg_rbufs : 0;
  out->shared_bytes = (int32_t)t.dyn_smem;
  return HQ_OK;
}

hq_status hq_launch_conv_tc(hq_handle* h, const ConvArgs& a, cudaStream_t stream) {
  if (!hq_conv_tc_supported(a)) return HQ_ERR_UNSUPPORTED;
  if (!load_driver_entry_points()) return HQ_ERR_CUDA;
  const long long P = (long long)a.n * a.ho * a.wo;
  if (P == 0) return HQ_OK;
  TcPlan t;
  const hq_status planned = plan_conv_tc(a, h->sm_count, h->conv_path, t);
  if (planned != HQ_OK) return planned;
  TcParams& p = t.p;
  p.rev = h->tile_order ? 1 : 0;
  p.bias = a.bias; p.b = a.b; p.c = a.c;
  p.res = a.res; p.res_bits = a.res_bits; p.res_signed = a.res_signed; p.rb = a.rb; p.rc = a.rc;
  p.res_narrow = (a.res && a.res_bits == 8) ? (const int4*)a.res_narrow : nullptr;
  p.narrow_fresh = a.res_narrow_fresh;
  p.params_late = a.params_late;
  p.relu = a.relu; p.qmin = a.qmin; p.qmax = a.qmax;
  p.out = a.out; p.out_bits = a.out_bits; p.out_signed = a.out_signed;
  if (a.wide) {
    p.q_out = a.wide->q; p.qb = a.wide->qb; p.qc = a.wide->qc; p.q_hi = a.wide->q_qmax;
    p.q_sat = 0;
    p.q_lo = a.wide->q_relu ? (a.wide->q_qmin > 0 ? a.wide->q_qmin : 0) : a.wide->q_qmin;
    p.q_sat = p.q_lo == 0 && p.q_hi == 255 ? 1 : 0;
  }
  {
    const int lo = a.relu ? (a.qmin > 0 ? a.qmin : 0) : a.qmin;
    p.sat_pack = (a.out_bits == 8 && ((!a.out_signed && lo == 0 && a.qmax == 255) ||
                                      (a.out_signed && lo == -128 && a.qmax == 127))) ? 1 : 0;
  }
  p.status = h->dev_status;

  const CUtensorMapSwizzle swz = swizzle_for(p.bkb);
  alignas(64) CUtensorMap map_x, map_w, map_out, map_res, map_q;
  p.x_tiled = (!a.pitch_w && a.kh == 1 && a.kw == 1 && a.stride == 1 && a.pad == 0) ? 1 : 0;
  if (p.strip) {
    // activations (C, W, H, N), box = one patch: bkb channels x pitch columns x (rows + 3) rows of one image
    const cuuint64_t dims[4] = {(cuuint64_t)a.cin, (cuuint64_t)a.w, (cuuint64_t)a.h, (cuuint64_t)a.n};
    const cuuint64_t strides[3] = {(cuuint64_t)a.cin, (cuuint64_t)a.cin * a.w, (cuuint64_t)a.cin * a.w * a.h};
    const cuuint32_t box[4] = {(cuuint32_t)p.bkb, 1u << p.lg_wp, (cuuint32_t)(p.rows + 3), 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    if (g_encode_tiled(&map_x, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void*>(a.in), dims, strides, box, estr,
                       CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) return HQ_ERR_CUDA;
    p.x_tiled = 0;
  } else if (p.x_tiled) {
    if (!encode_rows_map(&map_x, a.in, P, a.cin, p.bkb, p.pt >> p.duo, swz)) return HQ_ERR_CUDA;
  } else {
    if (!encode_im2col_map(&map_x, a, p.bkb, p.pt >> p.duo)) return HQ_ERR_CUDA;
  }
  if (p.pairs) {
    // weights (filter row of 3 x 64 bytes, 3 rows, 64 channels), box = 128 bytes of one filter row of every channel
    const cuuint64_t dims[3] = {192, 3, 64}, strides[2] = {192, 576};
    const cuuint32_t box[3] = {128, 1, 64}, estr[3] = {1, 1, 1};
    if (g_encode_tiled(&map_w, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<void*>(a.wgt), dims, strides, box, estr,
                       CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) return HQ_ERR_CUDA;
  } else if (p.frag) {
    if (!encode_paired_rows_map(&map_w, a.wgt, a.cout, (long long)a.kh * a.kw * a.cin, p.bkb, swz)) return HQ_ERR_CUDA;
  } else if (!encode_rows_map(&map_w, a.wgt, a.cout, (long long)a.kh * a.kw * a.cin, p.bkb, p.fold ? 64 : kTileC, swz)) return HQ_ERR_CUDA;
  map_out = map_w; map_res = map_w; map_q = map_w;                    // valid placeholders when a path is not staged
  // (with frag the residual tile becomes the output box: 128-byte swizzle both ways)
  const CUtensorMapSwizzle box_swz = p.frag ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE;
  if (p.strip) {
    // output (C, W, H, N), box = 32 positions of the raster: 32 channels x min(pitch, 32) columns x the rows that makes
    const cuuint32_t bw = p.lg_wp >= 5 ? 32u : (1u << p.lg_wp);
    const cuuint64_t dims[4] = {(cuuint64_t)a.cout, (cuuint64_t)a.wo, (cuuint64_t)a.ho, (cuuint64_t)a.n};
    const cuuint64_t strides[3] = {(cuuint64_t)a.cout, (cuuint64_t)a.cout * a.wo, (cuuint64_t)a.cout * a.wo * a.ho};
    const cuuint32_t box[4] = {32, bw, 32u / bw, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    if (g_encode_tiled(&map_out, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, a.out, dims, strides, box, estr,
                       CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) return HQ_ERR_CUDA;
  } else
  if (p.staged_out && !encode_rows_map(&map_out, a.out, P, (long long)a.cout * a.out_bits / 8, p.frag ? kTileC : a.out_bits == 4 ? 16 : 32, p.frag ? p.pt : p.pt / (p.halves << p.fold),
                                       box_swz)) return HQ_ERR_CUDA;
  if (p.staged_res && !encode_rows_map(&map_res, a.res, P, a.cout, kTileC, p.pt, box_swz))
    return HQ_ERR_CUDA;

  if (t.int32_boxes) {
    if (a.out && !encode_rows_map(&map_out, a.out, P, 4ll * a.cout, 128, 16, CU_TENSOR_MAP_SWIZZLE_NONE)) return HQ_ERR_CUDA;
    if (a.res && !encode_rows_map(&map_res, a.res, P, (long long)a.cout * a.res_bits / 8, a.res_bits == 32 ? 128 : 32, 16, CU_TENSOR_MAP_SWIZZLE_NONE)) return HQ_ERR_CUDA;
    if (p.q_out && !encode_rows_map(&map_q, p.q_out, P, a.cout, 32, 16, CU_TENSOR_MAP_SWIZZLE_NONE)) return HQ_ERR_CUDA;
  }

  const size_t dyn_smem = t.dyn_smem;
  const long long total_tiles = (long long)p.p_tiles * p.c_tiles;
  // a multiple of c_tiles, so that every CTA keeps one channel tile
  const int slots = t.pair ? 2 * h->sm_count : h->sm_count;
  const int grid = (int)(total_tiles <= slots ? total_tiles : (slots / p.c_tiles) * p.c_tiles);
  // Launched with programmatic stream serialization: the grid may begin (barrier set-up, tensor-memory
  // allocation) while the previous kernel drains; the kernel waits for it before reading any input.
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;          // duo: consecutive CTAs (channel tiles 2j, 2j+1) pair up
  attr[1].val.clusterDim.x = 2; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid); cfg.stream = stream; cfg.attrs = attr; cfg.numAttrs = p.duo ? 2 : 1;
  cudaError_t err;
  if (p.duo) {
    cfg.blockDim = dim3(32 * (2 + kSoloEpilogueWarps)); cfg.dynamicSmemBytes = dyn_smem < 120 * 1024 ? 120 * 1024 : dyn_smem;
    err = cudaLaunchKernelEx(&cfg, conv_tc_kernel<kSoloEpilogueWarps, 1, 1, true>, map_x, map_w, map_out, map_res, map_q, p);
  } else if (p.frag) {
    cfg.blockDim = dim3(32 * (2 + kFragIssuers + kFragWarps)); cfg.dynamicSmemBytes = dyn_smem < 120 * 1024 ? 120 * 1024 : dyn_smem;
    err = cudaLaunchKernelEx(&cfg, conv_tc_kernel<kFragWarps, 1, kFragIssuers, false, true>, map_x, map_w, map_out, map_res, map_q, p);
  } else if (t.pair) {
    cfg.blockDim = dim3(32 * (1 + kPairIssuerWarps + kPairEpilogueWarps)); cfg.dynamicSmemBytes = dyn_smem;
    err = cudaLaunchKernelEx(&cfg, conv_tc_kernel<kPairEpilogueWarps, 2, kPairIssuerWarps>, map_x, map_w, map_out, map_res, map_q, p);
  } else {
    // one CTA per SM (it may allocate all 512 tensor-memory columns): never request less than 120 KiB
    cfg.blockDim = dim3(32 * (1 + kSoloIssuerWarps + (t.int32_boxes ? kWideWarps : kSoloEpilogueWarps))); cfg.dynamicSmemBytes = dyn_smem < 120 * 1024 ? 120 * 1024 : dyn_smem;
    if (a.wide) err = cudaLaunchKernelEx(&cfg, conv_tc_kernel<kWideWarps, 1, kSoloIssuerWarps, false, false, kAdd32>, map_x, map_w, map_out, map_res, map_q, p);
    else if (t.int32_boxes) err = cudaLaunchKernelEx(&cfg, conv_tc_kernel<kWideWarps, 1, kSoloIssuerWarps, false, false, kRaw32>, map_x, map_w, map_out, map_res, map_q, p);
    else err = cudaLaunchKernelEx(&cfg, conv_tc_kernel<kSoloEpilogueWarps, 1, kSoloIssuerWarps>, map_x, map_w, map_out, map_res, map_q, p);
  }
  return err == cudaSuccess ? HQ_OK : HQ_ERR_CUDA;
}

cudaError_t hq_launch_residual_narrow(const int32_t* rb, const int32_t* rc, int res_signed, int channels, void* out,
                                      cudaStream_t s) {
  return hq_launch_residual_narrow2(rb, rc, res_signed, out, nullptr, nullptr, 0, nullptr, channels, s);
}

cudaError_t hq_launch_residual_narrow2(const int32_t* b0, const int32_t* c0, int signed0, void* out0,
                                       const int32_t* b1, const int32_t* c1, int signed1, void* out1, int channels,
                                       cudaStream_t s) {
  if (channels <= 0) return cudaSuccess;
  const NarrowJob j0{b0, c0, signed0, (int4*)out0}, j1{b1, c1, signed1, (int4*)out1};
  const int warps = out1 ? 2 * channels : channels;
  hq_launch_pdl(residual_narrow_kernel, (warps + 3) / 4, 128, 0, s, j0, j1, channels);
  return cudaGetLastError();
}

namespace {
// The wait of the kernels above, on a barrier that nothing signals: it gives up after the budget and says so in the status word.
__global__ void expire_wait_kernel(uint32_t* status, unsigned long long budget_ns) {
  struct Ctl { unsigned long long bar; volatile uint32_t abort_flag; };
  __shared__ Ctl ctl;
  ctl.abort_flag = 0;
  mbar_init(smem_u32(&ctl.bar), 1);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  mbar_wait(smem_u32(&ctl.bar), 0, &ctl, status, (uint32_t)HQ_DEV_TIMEOUT_EPILOGUE, budget_ns);
}
}  // namespace

cudaError_t hq_launch_expire_wait(uint32_t* status, int budget_ms, cudaStream_t s) {
  expire_wait_kernel<<<1, 1, 0, s>>>(status, (unsigned long long)budget_ms * 1000000ull);
  return cudaGetLastError();
}
