// Convolution for small problems on sm_100a: the same contraction and integer epilogue as conv_tc.cu (Eq. 3 and 4,
// Section 3.3, Appendix D), shaped for latency instead of throughput.
//
// A layer with few output pixels (small batches, late stages, classifiers) is bound by a chain of latencies: launch,
// first operand fetch, MMA, epilogue, store, next launch.  The persistent kernel of conv_tc.cu leaves most SMs idle
// there (one CTA per tile of 64 pixels x 128 channels walks the whole reduction alone) and its im2col fetch does not
// take inputs below 128 KiB.  This kernel computes ONE tile per CTA and is built so that as little as possible
// happens between the end of the previous kernel and the end of this one:
//   - a cluster of S CTAs (1, 2, 4 or 8) shares a tile and splits the reduction; INT32 partial sums meet through
//     distributed shared memory (st.async, counted on the receiver's barrier), each CTA finishing 1/S of the tile's
//     pixels (integer sums: any split is exact);
//   - weights do not depend on the previous kernel, so their TMA copies are issued before griddepcontrol.wait, as are
//     barrier set-up, tensor-memory allocation and the per-channel constants;
//   - activations come by TMA (tiled or im2col); where no tensor map can describe the fetch (packed 4-bit values, tensors
//     below 128 KiB without room behind them) the eight epilogue warps gather
//     them with 16-byte loads into the same swizzled layout: zeros for padding taps, nibbles widened on the way, no patch matrix;
//   - the epilogue turns 4 x 4 bytes round inside lane quads with two shuffles and writes words: no staging box and no
//     store whose completion has to be awaited;
//   - at most 105 KiB of shared memory and 64 tensor-memory columns: two CTAs per SM, so that the next kernel's CTAs are
//     resident, with their weights under way, while this one still runs.
// What bounds it (traced inside ResNet-50 at batch 1, ns from the end of the previous kernel's middle CTA): 1300 until
// griddepcontrol.wait returns, 500 for the first operands, 300-800 for the MMAs, 1300 for the exchange of a split
// reduction and 1000-1500 for the epilogue: a chain of latencies, no throughput.
#include "tc_common.cuh"

namespace {

constexpr int kGatherWarps = 8;
constexpr int kSmallThreads = 32 * (2 + kGatherWarps);   // warp 0: weights by TMA, warp 1: MMA, warps 2-9: gather and epilogue
constexpr int kSmallStages = 8;
constexpr int kGroup = 4;                                // gather: K blocks a thread loads and writes at once (at most the stages)
enum { kXGather = 0, kXTiled = 1, kXIm2col = 2 };        // how the activations reach shared memory

// n / d for 0 <= n < 2^31 by a multiplication: with l = ceil(log2 d) and m = ceil(2^(31 + l) / d) < 2^32 the error of
// n m / 2^(31 + l) stays below 1 / d (Granlund and Montgomery, "Division by invariant integers using multiplication", 1994).
struct FastDiv {
  uint32_t m, shift;
  __device__ __forceinline__ uint32_t div(uint32_t n) const { return (uint32_t)(((unsigned long long)n * m) >> shift); }
};

FastDiv fast_div(uint32_t d) {
  uint32_t l = 0;
  while ((1ull << l) < d) ++l;
  return {(uint32_t)(((1ull << (31 + l)) + d - 1) / d), 31 + l};
}

struct SmallParams {
  FastDiv by_cchunks, by_c_tiles, by_howo, by_wo, by_cin, by_kw;
  const void* x; const void* w4;                 // activations; packed 4-bit weights (NULL: weights by TMA)
  int32_t h, w, cin, wo, howo, stride, pad, kh, kw;
  int32_t P, C, K;                               // output pixels, output channels, reduction length (values)
  int32_t bkb, nkb, lg_split, stages;            // bytes of K per stage (gather: 128); K blocks of the layer; log2 of the cluster size; stages per CTA
  int32_t x_mode, cchunks, tail_steps;           // kXGather / kXTiled / kXIm2col; K blocks per filter tap and MMA steps of its last one (TMA modes)
  int32_t pt, lg_cols, c_tiles, fold;            // pixels per tile (MMA N); log2 of the pixels a CTA finishes; channel tiles; folded rows
  int32_t x_bits, x_signed, params_late;         // params_late: weights and constants may be the previous launch's output
  uint32_t part_off;                             // partial sums of a cluster, from the 1024-aligned base
  uint32_t tmem_cols;
  const int32_t* bias; const int32_t* b; const int32_t* c;
  const void* res; int32_t res_bits, res_signed; const int32_t* rb; const int32_t* rc;
  int32_t acc_bits;                              // |accumulator| < 2^acc_bits for every operand pair of these types
  const int4* res_narrow; int32_t narrow_fresh;  // optional checked narrow residual pairs (see conv_tc.cu)
  int32_t relu, qmin, qmax, sat;                 // sat: 1 / 2 when the clamp bounds equal the range of u8 / s8
  void* out; int32_t out_bits;
  uint32_t* status;
};

struct SmallCtl {
  unsigned long long wfull[kSmallStages];    // weights landed (TMA)
  unsigned long long xfull[kSmallStages];    // activations (and packed weights) written by the gather warps
  unsigned long long empty[kSmallStages];
  unsigned long long tfull;
  unsigned long long pfull;                  // cluster: every partner's sums landed
  uint32_t tmem_base;
  volatile uint32_t abort_flag;
};

__device__ __forceinline__ uint4 widen16(uint2 v, bool is_signed) {
  unsigned o[4];
  const unsigned w[2] = {v.x, v.y};
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    unsigned lo = w[k] & 0x0F0F0F0Fu, hi = (w[k] >> 4) & 0x0F0F0F0Fu;
    if (is_signed) { lo |= (lo & 0x08080808u) * 0x1Eu; hi |= (hi & 0x08080808u) * 0x1Eu; }   // sign-extend each nibble
    o[2 * k] = __byte_perm(lo, hi, 0x5140);
    o[2 * k + 1] = __byte_perm(lo, hi, 0x7362);
  }
  return make_uint4(o[0], o[1], o[2], o[3]);
}

// 4 NG columns x 32 lanes of the accumulator into this lane's registers, one wait for all of them
template <int NG>
__device__ __forceinline__ void load_columns(uint32_t taddr, int (&v)[4 * NG]) {
#pragma unroll
  for (int g = 0; g < NG; ++g)
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v[4 * g]), "=r"(v[4 * g + 1]), "=r"(v[4 * g + 2]), "=r"(v[4 * g + 3]) : "r"(taddr + 4 * g) : "memory");
  tmem_ld_wait();
#pragma unroll
  for (int i = 0; i < 4 * NG; ++i) asm volatile("" : "+r"(v[i]));      // nothing below may move above the wait
}

// What an epilogue warp knows about its part of the tile.
struct SmallEpi {
  const SmallParams* p;
  uint8_t* smem;                // 1024-aligned dynamic base
  uint32_t part, rank;          // shared-memory address of the sums; CTA of the cluster
  int ew, lane, quarter, ch, rows;
  int c_base;                   // first channel of the warp's quarter
  int px_tile, px_base;         // first pixel of the tile; first pixel this CTA finishes
  bool word_live;               // the four channels of this lane's output word exist
};

// This warp's accumulator columns go to the CTAs that finish them: 4 columns of one channel are one 16-byte word, counted
// on the receiver's `pfull` barrier as it lands.  Groups without a live pixel are neither sent nor expected.
template <int NG>
__device__ __forceinline__ void scatter_partials(const SmallEpi& e, uint32_t taddr, int col0, int row, uint32_t pfull) {
  const SmallParams& p = *e.p;
  int v[4 * NG];
  load_columns<NG>(taddr, v);
  const int lg_groups = p.lg_cols - 2, groups = 1 << lg_groups;
#pragma unroll
  for (int g = 0; g < NG; ++g) {
    const int gcol = (col0 >> 2) + g;                         // group of the tile
    if (e.px_tile + 4 * gcol >= p.P) break;
    const uint32_t dest = (uint32_t)(gcol >> lg_groups);
    const uint32_t off = e.part + (uint32_t)((((int)e.rank * groups + (gcol & (groups - 1))) * e.rows + row) << 4);
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
                 ::"r"(in_cta(off, dest)), "r"(v[4 * g]), "r"(v[4 * g + 1]), "r"(v[4 * g + 2]), "r"(v[4 * g + 3]),
                   "r"(in_cta(pfull, dest)) : "memory");
  }
}

// The sums of NF groups of 4 columns of this lane's channel: one term per CTA of the cluster.
template <int NF>
__device__ __forceinline__ void gather_partials(const SmallEpi& e, int lg_quarters, int (&acc)[NF][4]) {
  const int lg_groups = e.p->lg_cols - 2;
  uint32_t at = e.part + (uint32_t)((e.quarter * 32 + e.lane) << 4);
#pragma unroll
  for (int f = 0; f < NF; ++f) acc[f][0] = acc[f][1] = acc[f][2] = acc[f][3] = 0;
  for (int s = 0; s < (1 << e.p->lg_split); ++s, at += (uint32_t)(e.rows << (4 + lg_groups))) {
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      const int gi = (f * kGatherWarps + e.ew) >> lg_quarters;
      int4 a;
      asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w)
                   : "r"(at + (uint32_t)((gi * e.rows) << 4)) : "memory");
      acc[f][0] += a.x; acc[f][1] += a.y; acc[f][2] += a.z; acc[f][3] += a.w;
    }
  }
}

// Residual words of the groups a warp finishes, one per lane and group: four channels of pixel px0 + lane % 4, turned round
// when they are used.  `px(f)` is the first pixel of the warp's f-th group.
template <int NF, class Px>
__device__ __forceinline__ void load_residual_words(const SmallEpi& e, Px px, unsigned (&r)[NF]) {
  const SmallParams& p = *e.p;
  const int ch4 = e.c_base + (e.lane & ~3);
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    const int q = px(f) + (e.lane & 3);
    r[f] = (q < p.P && ch4 < p.C) ? __ldcg((const unsigned*)((const unsigned char*)p.res + (long long)q * p.C + ch4)) : 0u;
  }
}

// Eq. 4 on 4 pixels of this lane's channel in 32-bit steps, 8-bit output, whole words (C a multiple of 4).
// RES: 0 none, 1 / 2 unsigned / signed 8-bit residual, 3 / 4 the same with a checked narrow pair (see requant_fast);
// PRE: some channel of the warp has c < 32 and takes the pre-shift form.
template <int RES, bool PRE>
__device__ __forceinline__ void finish_fast8(const SmallEpi& e, const ChanConst& k, const int* acc, unsigned rword, int px0, unsigned char* dst, int lo, int hi) {
  const SmallParams& p = *e.p;
  constexpr bool SIGNED = RES == 2 || RES == 4;
  if (RES) rword = quad_transpose(rword, e.lane);
  int y[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int r = RES == 0 ? 0 : (int)hq_prmt(rword, 0u, SIGNED ? 0x8880u + 0x1111u * j : 0x4440u + j);
    y[j] = requant_fast<RES != 0, SIGNED, PRE ? 2 : 0, RES >= 3>(acc[j], r, k);
  }
  unsigned w;
  if (p.sat == 1) w = sat_pack4<false>(y[0], y[1], y[2], y[3]);
  else if (p.sat == 2) w = sat_pack4<true>(y[0], y[1], y[2], y[3]);
  else {
#pragma unroll
    for (int j = 0; j < 4; ++j) y[j] = min(max(y[j], lo), hi);
    w = (unsigned)(y[0] & 0xFF) | ((unsigned)(y[1] & 0xFF) << 8) | ((unsigned)(y[2] & 0xFF) << 16) | ((unsigned)(y[3] & 0xFF) << 24);
  }
  w = quad_transpose(w, e.lane);                                        // four channels of pixel px0 + lane % 4
  if (px0 + (e.lane & 3) < p.P && e.word_live) *(unsigned*)dst = w;
}

// Every other type, shift and channel count; 64-bit arithmetic.
__device__ __noinline__ void finish_general(const SmallEpi& e, const ChanConst& k, const int (&acc)[4], int px0) {
  const SmallParams& p = *e.p;
  const bool ch_live = e.ch < p.C, words = (p.C & 3) == 0;
  if (px0 >= p.P) return;
  if (p.out_bits == 32) {
    if (ch_live) {
      int* dst = (int*)p.out + (long long)px0 * p.C + e.ch;
#pragma unroll
      for (int j = 0; j < 4; ++j) if (px0 + j < p.P) dst[(long long)j * p.C] = acc[j] + k.bias;
    }
    return;
  }
  int y[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    long long s = ((long long)acc[j] * (long long)k.b + k.r0) >> k.sh;
    if (p.res && ch_live && px0 + j < p.P)
      s += ((long long)hq_load_elem(p.res, (long long)(px0 + j) * p.C + e.ch, p.res_bits, p.res_signed) * (long long)k.rb + k.rr0) >> k.rsh;
    y[j] = hq_clamp_ll(s, p.relu, p.qmin, p.qmax);
  }
  if (words) {
    const unsigned wv = quad_transpose((unsigned)(y[0] & 0xFF) | ((unsigned)(y[1] & 0xFF) << 8) | ((unsigned)(y[2] & 0xFF) << 16) |
                                       ((unsigned)(y[3] & 0xFF) << 24), e.lane);
    const int px = px0 + (e.lane & 3), ch4 = e.c_base + (e.lane & ~3);
    if (px < p.P && ch4 < p.C) {
      if (p.out_bits == 8) *(unsigned*)((unsigned char*)p.out + (long long)px * p.C + ch4) = wv;
      else {
        const unsigned n = wv & 0x0F0F0F0Fu, two = n | (n >> 4);          // bytes 0 and 2: channel pairs
        *(unsigned short*)((unsigned char*)p.out + (((long long)px * p.C + ch4) >> 1)) = (unsigned short)__byte_perm(two, 0u, 0x4420);
      }
    }
  } else if (p.out_bits == 8) {
    if (ch_live) {
#pragma unroll
      for (int j = 0; j < 4; ++j) if (px0 + j < p.P) ((unsigned char*)p.out)[(long long)(px0 + j) * p.C + e.ch] = (unsigned char)y[j];
    }
  } else {
    // neighbouring channels share a byte (C is even)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int other = __shfl_xor_sync(0xffffffffu, y[j], 1);
      if (ch_live && !(e.lane & 1) && px0 + j < p.P)
        ((unsigned char*)p.out)[((long long)(px0 + j) * p.C + e.ch) >> 1] = (unsigned char)((y[j] & 0xF) | ((other & 0xF) << 4));
    }
  }
}

// One CTA per tile: a warp finishes the columns it reads, NG groups of 4 from tile column col0 on.
template <int NG, int RES, bool PRE>
__device__ __forceinline__ void finish_own(const SmallEpi& e, const ChanConst& k, uint32_t taddr, int col0, const unsigned* r, int lo, int hi) {
  int v[4 * NG];
  load_columns<NG>(taddr, v);
  const int px0 = e.px_base + col0;
  const int step = 4 * e.p->C;
  unsigned char* dst = (unsigned char*)e.p->out + (long long)(px0 + (e.lane & 3)) * e.p->C + e.c_base + (e.lane & ~3);
#pragma unroll
  for (int g = 0; g < NG; ++g, dst += step) finish_fast8<RES, PRE>(e, k, v + 4 * g, RES ? r[g] : 0u, px0 + 4 * g, dst, lo, hi);
}
// A cluster shares the tile: the warp finishes NF (group, quarter) pairs of the CTA's pixels.
template <int NF, int RES, bool PRE>
__device__ __forceinline__ void finish_split(const SmallEpi& e, const ChanConst& k, int lg_quarters, const unsigned* r, int lo, int hi) {
  int acc[NF][4];
  gather_partials<NF>(e, lg_quarters, acc);
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    const int px0 = e.px_base + 4 * ((f * kGatherWarps + e.ew) >> lg_quarters);
    unsigned char* dst = (unsigned char*)e.p->out + (long long)(px0 + (e.lane & 3)) * e.p->C + e.c_base + (e.lane & ~3);
    finish_fast8<RES, PRE>(e, k, acc[f], RES ? r[f] : 0u, px0, dst, lo, hi);
  }
}
template <int NF>
__device__ __forceinline__ void finish_split_general(const SmallEpi& e, const ChanConst& k, int lg_quarters) {
  int acc[NF][4];
  gather_partials<NF>(e, lg_quarters, acc);
#pragma unroll
  for (int f = 0; f < NF; ++f) finish_general(e, k, acc[f], e.px_base + 4 * ((f * kGatherWarps + e.ew) >> lg_quarters));
}
template <int NG>
__device__ __forceinline__ void finish_own_general(const SmallEpi& e, const ChanConst& k, uint32_t taddr, int col0) {
  int v[4 * NG];
  load_columns<NG>(taddr, v);
#pragma unroll
  for (int g = 0; g < NG; ++g) {
    const int acc[4] = {v[4 * g], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3]};
    finish_general(e, k, acc, e.px_base + col0 + 4 * g);
  }
}

// GATHER: the activations are fetched by the epilogue warps (kXGather), else by TMA.
template <bool GATHER>
__global__ void __launch_bounds__(kSmallThreads, 2) conv_small_kernel(const __grid_constant__ CUtensorMap map_w,
                                                                      const __grid_constant__ CUtensorMap map_x,
                                                                      const __grid_constant__ SmallParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ SmallCtl ctl;
  const uint32_t raw = smem_u32(smem_raw), tiles = (raw + 1023u) & ~1023u;
  const uint32_t w_bytes = (uint32_t)(kTileC * p.bkb), x_bytes = (uint32_t)(p.pt * p.bkb), stage_bytes = w_bytes + x_bytes;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = blockIdx.x & ((1u << p.lg_split) - 1u);
  const uint32_t tile = blockIdx.x >> p.lg_split;
  const int p_tile = (int)p.by_c_tiles.div(tile), c_tile = (int)tile - p_tile * p.c_tiles;
  // this CTA's K blocks
  const int kb0 = (p.nkb * (int)rank) >> p.lg_split, L = ((p.nkb * ((int)rank + 1)) >> p.lg_split) - kb0;

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(smem_u32(&ctl.wfull[s]), 1); mbar_init(smem_u32(&ctl.xfull[s]), GATHER ? kGatherWarps : 1); mbar_init(smem_u32(&ctl.empty[s]), 1);
    }
    mbar_init(smem_u32(&ctl.tfull), 1);
    mbar_init(smem_u32(&ctl.pfull), 1);
    ctl.abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (p.lg_split) {
      // groups of 4 pixels this CTA finishes that hold a live pixel, from every CTA of the cluster
      const int left = p.P - (p_tile * p.pt + ((int)rank << p.lg_cols));
      const int live_groups = left <= 0 ? 0 : min((left + 3) >> 2, 1 << (p.lg_cols - 2));
      mbar_expect_tx(smem_u32(&ctl.pfull), (uint32_t)((live_groups * (p.fold ? 64 : kTileC)) << (4 + p.lg_split)));
    }
  }
  if (warp == 1) tmem_alloc(smem_u32(&ctl.tmem_base), p.tmem_cols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (p.lg_split) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");   // waited for before the first remote store
  const uint32_t tmem_base = ctl.tmem_base;
  // A call of its own may follow the kernel that wrote its weights and constants: nothing is read ahead of that one's end.
  if (p.params_late) asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  if (warp == 0) {
    // Weights, before anything of the previous kernel is awaited (see conv_tc.cu: no launch writes weights immediately
    // before the convolution that reads them); activations, in the TMA modes, after it.
    if (elect_one()) {
      const int row = p.fold ? c_tile * 64 : c_tile * kTileC, row2 = p.fold ? row : row + 64;
      // (K blocks are loaded in order: the weight column advances by a block, and by a tap's channels at its end)
      const int wtap = GATHER ? 0 : (int)p.by_cchunks.div((uint32_t)kb0);
      int wchunk = kb0 - wtap * p.cchunks, tap_x = wtap * p.cin, wx = GATHER ? kb0 * 128 : tap_x + wchunk * p.bkb;
      auto load_w = [&](int s) {
        const uint32_t bar = smem_u32(&ctl.wfull[s]), dst = tiles + (uint32_t)s * stage_bytes;
        mbar_expect_tx(bar, w_bytes);
        tma_load_2d(dst, &map_w, bar, wx, row);
        tma_load_2d(dst + w_bytes / 2, &map_w, bar, wx, row2);
        wx += p.bkb;
        if (!GATHER && ++wchunk == p.cchunks) { wchunk = 0; tap_x += p.cin; wx = tap_x; }
      };
      const int px0 = p_tile * p.pt;
      const int img = (int)p.by_howo.div((uint32_t)px0), rem = px0 - img * p.howo, oh = (int)p.by_wo.div((uint32_t)rem), ow = rem - oh * p.wo;
      const int tap0 = p.x_mode == kXIm2col ? (int)p.by_cchunks.div((uint32_t)kb0) : 0;
      int chunk = kb0 - tap0 * p.cchunks, tr = (int)p.by_kw.div((uint32_t)tap0), ts = tap0 - tr * p.kw;
      auto load_x = [&](int s) {
        const uint32_t bar = smem_u32(&ctl.xfull[s]), dst = tiles + (uint32_t)s * stage_bytes + w_bytes;
        mbar_expect_tx(bar, x_bytes);
        if (p.x_mode == kXTiled) tma_load_2d(dst, &map_x, bar, chunk * p.bkb, px0);
        else tma_load_im2col(dst, &map_x, bar, chunk * p.bkb, ow * p.stride - p.pad, oh * p.stride - p.pad, img, (uint16_t)ts, (uint16_t)tr);
        if (++chunk == p.cchunks) { chunk = 0; if (++ts == p.kw) { ts = 0; ++tr; } }
      };
      const int ahead = L < p.stages ? L : p.stages;
      if (!p.w4) for (int i = 0; i < ahead; ++i) load_w(i);
      if constexpr (!GATHER) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        for (int i = 0; i < ahead; ++i) load_x(i);
      }
      int issued = ahead;
      for (int i = ahead, s = 0, ph = 0; i < L && !(p.w4 && GATHER); ++i, ++issued) {
        if (!mbar_wait(smem_u32(&ctl.empty[s]), (uint32_t)ph, &ctl, p.status, HQ_DEV_TIMEOUT_PRODUCER)) break;
        if (!p.w4) load_w(s);
        if (!GATHER) load_x(s);
        if (++s == p.stages) { s = 0; ph ^= 1; }
      }
      // every copy this thread started must have landed before the CTA may exit
      for (int i = issued > p.stages ? issued - p.stages : 0; i < issued; ++i) {
        const uint32_t ph = (uint32_t)(i / p.stages) & 1u;
        for (int which = 0; which < 2; ++which) {
          if (which == 0 ? p.w4 != nullptr : GATHER) continue;
          const uint32_t bar = smem_u32(which == 0 ? &ctl.wfull[i % p.stages] : &ctl.xfull[i % p.stages]);
          if (mbar_try_wait(bar, ph)) continue;
          const unsigned long long t0 = global_ns();
          while (!mbar_try_wait(bar, ph))
            if (global_ns() - t0 > kWaitBudgetNs) { atomicCAS(p.status, 0u, (uint32_t)HQ_DEV_TIMEOUT_DRAIN); break; }
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (elect_one()) {
      // D = S32, A = s8 weights, B = u8/s8 activations, both K-major, N = pt, M = 128
      const uint32_t idesc = (2u << 4) | (1u << 7) | ((uint32_t)(p.x_signed ? 1 : 0) << 10) | ((uint32_t)(p.pt >> 3) << 17) |
                             ((uint32_t)(kTileC >> 4) << 24);
      const uint64_t hi = smem_desc(0, p.bkb);
      const int full_steps = p.bkb >> 5;
      int chunk = GATHER ? 0 : kb0 - (int)p.by_cchunks.div((uint32_t)kb0) * p.cchunks;
      for (int i = 0, s = 0, ph = 0; i < L; ++i) {
        if (!p.w4 && !mbar_wait(smem_u32(&ctl.wfull[s]), (uint32_t)ph, &ctl, p.status, HQ_DEV_TIMEOUT_MMA)) break;
        if (!mbar_wait(smem_u32(&ctl.xfull[s]), (uint32_t)ph, &ctl, p.status, HQ_DEV_TIMEOUT_MMA)) break;
        tc_fence_after();
        const uint32_t a = tiles + (uint32_t)s * stage_bytes;
        uint64_t adesc = hi | (uint64_t)((a >> 4) & 0x3FFF), bdesc = hi | (uint64_t)(((a + w_bytes) >> 4) & 0x3FFF);
        // (a block may reach past the channels: whole 32-byte steps beyond them are left out, a partial step meets zeros)
        int steps;
        if (GATHER) steps = (min(p.K - (kb0 + i) * p.bkb, p.bkb) + 31) >> 5;
        else { steps = full_steps; if (++chunk == p.cchunks) { chunk = 0; steps = p.tail_steps; } }
        for (int q = 0; q < steps; ++q, adesc += 2, bdesc += 2) mma_i8(tmem_base, adesc, bdesc, idesc, (i | q) ? 1u : 0u);
        mma_commit(smem_u32(i + 1 == L ? &ctl.tfull : &ctl.empty[s]));
        if (++s == p.stages) { s = 0; ph ^= 1; }
      }
    }
    __syncwarp();
  }
  if (warp < 2) {
    if (p.lg_split) { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); cluster_sync_all(); }
    __syncthreads();
    if (warp == 1) { tc_fence_after(); tmem_dealloc(tmem_base, p.tmem_cols); }
    return;
  }

  const int ew = warp - 2;
  // what this warp finishes, and its channel's constants (parameters of the layer, never written by the previous launch)
  SmallEpi e;
  e.p = &p; e.smem = smem_raw + (tiles - raw); e.part = tiles + p.part_off; e.rank = rank; e.ew = ew; e.lane = lane;
  e.rows = p.fold ? 64 : kTileC;                              // distinct accumulator rows
  const int q = warp & 3, half = ew >> 2;                     // tensor-memory lane quarter this warp may read
  const int lg_quarters = p.fold ? 1 : 2;
  const int own_quarter = q & ((1 << lg_quarters) - 1);
  // split: (group of 4 columns, quarter) pairs dealt round-robin, so that the quarter is fixed per warp
  e.quarter = p.lg_split ? (ew & ((1 << lg_quarters) - 1)) : own_quarter;
  e.c_base = c_tile * e.rows + e.quarter * 32; e.ch = e.c_base + lane; e.word_live = e.c_base + (lane & ~3) < p.C;
  e.px_tile = p_tile * p.pt; e.px_base = e.px_tile + ((int)rank << p.lg_cols);
  const int lg_slices = p.fold ? 2 : 1, si = p.fold ? (q >> 1) * 2 + half : half;
  const int ncol = max(p.pt >> lg_slices, 4), col0 = si * ncol;
  const bool reads = col0 < p.pt;
  ChanConst k{};
  bool fast = false, pre = false;
  int form = 0;                                               // RES of finish_fast8
  if (p.out_bits == 32) k.bias = (e.ch < p.C && p.bias) ? p.bias[e.ch] : 0;
  else {
    k = chan_const(p, e.ch, false);
    pre = __any_sync(0xffffffffu, k.sh < 32) != 0;
    fast = p.out_bits == 8 && (p.C & 3) == 0 &&
           __all_sync(0xffffffffu, (k.sh >= 32 || (k.sh - 2 >= p.acc_bits && k.sh >= 3 && (k.bias < 0 ? ~k.bias : k.bias) < (1 << (k.sh - 2)))) &&
                                   (!p.res || (p.res_bits == 8 && k.rsh >= 9))) != 0;
    if (fast) {
      k = chan_const(p, e.ch, true, pre);
      if (p.res) {
        form = p.res_signed ? 2 : 1;
        if (p.res_narrow) {
          if (p.narrow_fresh) asm volatile("griddepcontrol.wait;" ::: "memory");
          const int4 nr = e.ch < p.C ? p.res_narrow[e.ch] : make_int4(0, 0, 0, 1);
          if (__all_sync(0xffffffffu, nr.w != 0)) { k.rb = nr.x; k.rh = nr.y; k.rsh = nr.z; form += 2; }
        }
      }
    }
  }
  const int lo = p.relu ? (p.qmin > 0 ? p.qmin : 0) : p.qmin, hi = p.qmax;
  unsigned rw[8];

  // residual words of the groups this warp will finish: they land while the reduction runs
  auto fetch_residual = [&]() {
    if (!p.res || !fast) return;
    if (p.lg_split) load_residual_words<8>(e, [&](int f) { const int gi = (f * kGatherWarps + ew) >> lg_quarters; return gi < (1 << (p.lg_cols - 2)) ? e.px_base + 4 * gi : p.P; }, rw);
    else load_residual_words<8>(e, [&](int f) { return 4 * f < ncol && reads ? e.px_base + col0 + 4 * f : p.P; }, rw);
  };
  if constexpr (!GATHER) {
    if (p.res) {
      asm volatile("griddepcontrol.wait;" ::: "memory");
      fetch_residual();
    }
  } else {
    // ---------------------------------------------------------- gather: [pt pixels][128 bytes] per stage, 128-byte swizzle
    const int t = threadIdx.x - 64;
    const int piece = t & 7, px_lo = t >> 3;                    // 16-byte piece of the row; pixels px_lo and px_lo + 32
    int ih0[2], iw0[2];
    const unsigned char* base[2];
    bool live[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int px = px_lo + 32 * u, g = p_tile * p.pt + px;
      live[u] = px < p.pt && g < p.P;
      const int n = (int)p.by_howo.div((uint32_t)g), r = g - n * p.howo, oh = (int)p.by_wo.div((uint32_t)r), ow = r - oh * p.wo;
      ih0[u] = oh * p.stride - p.pad; iw0[u] = ow * p.stride - p.pad;
      const long long e = (((long long)n * p.h + ih0[u]) * p.w + iw0[u]) * p.cin;      // (may lie before the tensor; only used with a tap inside)
      base[u] = (const unsigned char*)p.x + (p.x_bits == 4 ? e >> 1 : e);
    }
    int ci = kb0 * 128 + piece * 16, fr = 0, fs = 0;        // this thread's position in K: (filter row, column, channel)
    {
      const int tap = (int)p.by_cin.div((uint32_t)ci);
      ci -= tap * p.cin;
      fr = (int)p.by_kw.div((uint32_t)tap); fs = tap - fr * p.kw;
    }
    bool ok = true;
    int s = 0, eph = 1;
    const int group = min(kGroup, p.stages);                  // a group waits for all its stages at once
    for (int i0 = 0; i0 < L && ok; i0 += group) {
      const int nb = min(group, L - i0);
      uint4 v[kGroup][2];
      if (i0 == 0) asm volatile("griddepcontrol.wait;" ::: "memory");    // activations and residual: the previous kernel's output
#pragma unroll
      for (int g = 0; g < kGroup; ++g) {
        if (g >= nb) break;
        const bool kin = fr < p.kh;                             // inside K
        const int off = (fr * p.w + fs) * p.cin + ci;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          v[g][u] = make_uint4(0u, 0u, 0u, 0u);
          if (kin && live[u] && (unsigned)(ih0[u] + fr) < (unsigned)p.h && (unsigned)(iw0[u] + fs) < (unsigned)p.w) {
            if (p.x_bits == 4) { const uint2 x = __ldcg((const uint2*)(base[u] + (off >> 1))); v[g][u].x = x.x; v[g][u].y = x.y; }
            else v[g][u] = __ldcg((const uint4*)(base[u] + off));
          }
        }
        ci += 128;
        while (ci >= p.cin) { ci -= p.cin; if (++fs == p.kw) { fs = 0; ++fr; } }
      }
      if (i0 == 0) fetch_residual();
      // every stage of this group must be free
      if (i0 + nb > p.stages) {
        uint32_t w = 1;
        if (lane == 0)
          for (int g = 0, sg = s, pg = eph; g < nb && w; ++g) {
            if (i0 + g >= p.stages) w = mbar_wait(smem_u32(&ctl.empty[sg]), (uint32_t)pg, &ctl, p.status, HQ_DEV_TIMEOUT_PRODUCER) ? 1u : 0u;
            if (++sg == p.stages) { sg = 0; pg ^= 1; }
          }
        ok = __shfl_sync(0xffffffffu, w, 0) != 0;
        if (!ok) break;
      }
#pragma unroll
      for (int g = 0; g < kGroup; ++g) {
        if (g >= nb) break;
        uint8_t* const stage = e.smem + (uint32_t)s * stage_bytes;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int px = px_lo + 32 * u;
          if (live[u]) {
            const uint4 x = p.x_bits == 4 ? widen16(make_uint2(v[g][u].x, v[g][u].y), p.x_signed != 0) : v[g][u];
            *(uint4*)(stage + w_bytes + px * 128 + ((piece ^ (px & 7)) << 4)) = x;
          }
        }
        if (p.w4) {
          // packed 4-bit weights: 128 rows x 8 pieces, four per thread
          const int kk = (kb0 + i0 + g) * 128 + piece * 16;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int row = px_lo + 32 * j, oc = p.fold ? c_tile * 64 + (row & 63) : c_tile * kTileC + row;
            uint4 x = make_uint4(0u, 0u, 0u, 0u);
            if (oc < p.C && kk < p.K) x = widen16(__ldg((const uint2*)((const unsigned char*)p.w4 + (((long long)oc * p.K + kk) >> 1))), true);
            *(uint4*)(stage + row * 128 + ((piece ^ (row & 7)) << 4)) = x;
          }
        }
        fence_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&ctl.xfull[s]));
        if (++s == p.stages) { s = 0; eph ^= 1; }
      }
    }
  }
  {
    uint32_t w = 1;
    if (lane == 0) w = mbar_wait(smem_u32(&ctl.tfull), 0, &ctl, p.status, HQ_DEV_TIMEOUT_EPILOGUE) ? 1u : 0u;
    __shfl_sync(0xffffffffu, w, 0);
    tc_fence_after();
  }

  const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)col0;
  if (!p.lg_split) {
    // ---------------------------------------------------------- the whole reduction is here: finish the columns this warp reads
    if (reads) {
      // (the form is the same for every chunk: chosen once, the chunks unrolled behind it)
#define HQ_FORMS(CALL) do { \
        if (pre) { if (form == 0) CALL(0, true); else if (form == 1) CALL(1, true); else if (form == 2) CALL(2, true); \
                   else if (form == 3) CALL(3, true); else CALL(4, true); } \
        else { if (form == 0) CALL(0, false); else if (form == 1) CALL(1, false); else if (form == 2) CALL(2, false); \
               else if (form == 3) CALL(3, false); else CALL(4, false); } } while (0)
#define HQ_OWN4(R, PR) do { finish_own<4, R, PR>(e, k, taddr, col0, rw, lo, hi); \
                            if (ncol == 32) finish_own<4, R, PR>(e, k, taddr + 16, col0 + 16, rw + 4, lo, hi); } while (0)
#define HQ_OWN2(R, PR) finish_own<2, R, PR>(e, k, taddr, col0, rw, lo, hi)
#define HQ_OWN1(R, PR) finish_own<1, R, PR>(e, k, taddr, col0, rw, lo, hi)
      if (!fast) {
        for (int c = 0; c < ncol; c += 4) finish_own_general<1>(e, k, taddr + c, col0 + c);
      } else if (ncol >= 16) HQ_FORMS(HQ_OWN4); else if (ncol == 8) HQ_FORMS(HQ_OWN2); else HQ_FORMS(HQ_OWN1);
#undef HQ_OWN4
#undef HQ_OWN2
#undef HQ_OWN1
    }
    tc_fence_before();
    __syncthreads();
    return;
  }
  // ------------------------------------------------------------ sums over the cluster, then 1/S of the pixels each
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");    // every CTA of the cluster runs, its barriers exist
  if (reads) {
    const int row = own_quarter * 32 + lane;
    const uint32_t pfull = smem_u32(&ctl.pfull);
    if (ncol == 32) scatter_partials<8>(e, taddr, col0, row, pfull);
    else if (ncol == 16) scatter_partials<4>(e, taddr, col0, row, pfull);
    else if (ncol == 8) scatter_partials<2>(e, taddr, col0, row, pfull);
    else scatter_partials<1>(e, taddr, col0, row, pfull);
  }
  tc_fence_before();
  {
    uint32_t w = 1;
    if (lane == 0) w = mbar_wait(smem_u32(&ctl.pfull), 0, &ctl, p.status, HQ_DEV_TIMEOUT_EPILOGUE) ? 1u : 0u;
    __shfl_sync(0xffffffffu, w, 0);
  }
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");  // nobody leaves while sums may still be sent to it
  const int npairs = 1 << (p.lg_cols - 2 + lg_quarters);                 // at most 32 columns x 4 quarters over eight warps
  if (ew < npairs) {
#define HQ_SPLIT4(R, PR) finish_split<4, R, PR>(e, k, lg_quarters, rw, lo, hi)
#define HQ_SPLIT2(R, PR) finish_split<2, R, PR>(e, k, lg_quarters, rw, lo, hi)
#define HQ_SPLIT1(R, PR) finish_split<1, R, PR>(e, k, lg_quarters, rw, lo, hi)
    if (!fast) { if (npairs == 32) finish_split_general<4>(e, k, lg_quarters); else if (npairs == 16) finish_split_general<2>(e, k, lg_quarters); else finish_split_general<1>(e, k, lg_quarters); }
    else if (npairs == 32) HQ_FORMS(HQ_SPLIT4); else if (npairs == 16) HQ_FORMS(HQ_SPLIT2); else HQ_FORMS(HQ_SPLIT1);
#undef HQ_SPLIT4
#undef HQ_SPLIT2
#undef HQ_SPLIT1
#undef HQ_FORMS
  }
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  __syncthreads();                                                       // tensor memory has been read: warp 1 frees it
}

// Shape of one launch, as a function of the layer and the device.
struct SmallShape { int x_mode, bkb, pt, lg_split, stages, nkb, c_tiles, fold; long long p_tiles; };
constexpr int kExchangeBlocks = 5;                       // the exchange of a cluster's sums, in K blocks
constexpr int kSmallSmem = 104 * 1024;                   // stages and partial sums: two CTAs per SM

SmallShape small_shape(const ConvArgs& a, int sm_count) {
  SmallShape s{};
  const long long P = (long long)a.n * a.ho * a.wo;
  // TMA where a tensor map can describe the fetch: dense rows, or an im2col walk over a tensor of at least 128 KiB (or one
  // a network allocated with that much room, see ConvArgs::in_slack)
  ConvArgs b8 = a;
  b8.in_bits = 8;
  const bool packed = a.in_bits == 4, rows_map = a.kh == 1 && a.kw == 1 && a.stride == 1 && a.pad == 0;
  s.x_mode = packed || !hq_conv_tc_supported(b8) ? kXGather
           : rows_map ? kXTiled : !hq_conv_tc_small_im2col(a) ? kXIm2col : kXGather;
  s.bkb = s.x_mode == kXGather ? 128 : hq_conv_bkb(a.cin);
  s.nkb = s.x_mode == kXGather ? (int)(((long long)a.kh * a.kw * a.cin + s.bkb - 1) / s.bkb) : a.kh * a.kw * ((a.cin + s.bkb - 1) / s.bkb);
  // Pixel tile and split of the reduction: 64 pixels, fewer while that still doubles the CTAs without exceeding one per SM
  // (the epilogue of a tile is the longest piece of the chain, and half as long on half the pixels).
  for (s.pt = 64; ; s.pt >>= 1) {
    s.p_tiles = (P + s.pt - 1) / s.pt;
    // 64-channel tiles where even a cluster of eight per tile fits: half the epilogue and half the sums to exchange per CTA
    s.fold = a.cout <= 64 || s.p_tiles * ((a.cout + 63) / 64) <= sm_count / 8 ? 1 : 0;
    s.c_tiles = (a.cout + (s.fold ? 63 : kTileC - 1)) / (s.fold ? 64 : kTileC);
    const long long tiles = s.p_tiles * s.c_tiles;
    // Split the reduction where it pays and while the clusters fit the device at once (clusters of up to eight leave some
    // SMs of a GPC over: 7/8 of them).  Measured: a K block costs about 0.3 us, the exchange of the sums 1.3 us whatever the
    // split (1x1 512 -> 128 at 28x28, 4 blocks: one CTA 4.4 us, two 4.6; 1024 -> 256 at 14x14, 8 blocks: 5.6 / 5.1 / four 4.9).
    s.lg_split = 0;
    int best = s.nkb;
    for (int lg = 1; lg <= 3 && (tiles << lg) <= sm_count - sm_count / 8 && (s.nkb >> lg) >= 1 && (s.pt >> lg) >= 4; ++lg) {
      const int cost = ((s.nkb + (1 << lg) - 1) >> lg) + kExchangeBlocks;
      if (cost < best) { best = cost; s.lg_split = lg; }
    }
    if (s.pt == 16 || (P > s.pt / 2 && (tiles << (s.lg_split + 1)) > sm_count)) break;
  }
  const int rows = s.fold ? 64 : kTileC;
  const int per_cta = (s.nkb + (1 << s.lg_split) - 1) >> s.lg_split;
  const int room = (kSmallSmem - (s.lg_split ? s.pt * rows * 4 : 0)) / ((kTileC + s.pt) * s.bkb);
  s.stages = per_cta < room ? per_cta : room;
  if (s.stages > kSmallStages) s.stages = kSmallStages;
  return s;
}

}  // namespace

bool hq_conv_small_init() {
  return load_driver_entry_points() &&
         cudaFuncSetAttribute(conv_small_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 110 * 1024) == cudaSuccess &&
         cudaFuncSetAttribute(conv_small_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 110 * 1024) == cudaSuccess;
}

bool hq_conv_small_supported(const ConvArgs& a, int sm_count) {
  if (!(a.in_bits == 8 || a.in_bits == 4) || a.cin % 16 != 0 || a.pitch_w) return false;
  if ((long long)a.n * a.ho * a.wo >= (1ll << 31) - 64 || (long long)a.kh * a.kw * a.cin >= (1ll << 24)) return false;
  if ((long long)a.kh * a.w * a.cin >= (1ll << 31)) return false;
  if (a.out_bits == 4 && (a.cout & 1)) return false;
  if (a.res && !(a.res_bits == 8 || a.res_bits == 32)) return false;
  if (((uintptr_t)a.in & 15u) || ((uintptr_t)a.wgt & 15u)) return false;
  const SmallShape s = small_shape(a, sm_count);
  return ((s.p_tiles * s.c_tiles) << s.lg_split) < (1ll << 31);
}

hq_status hq_launch_conv_small(hq_handle* h, const ConvArgs& a, cudaStream_t stream) {
  if (!hq_conv_small_supported(a, h->sm_count)) return HQ_ERR_UNSUPPORTED;
  if (!load_driver_entry_points()) return HQ_ERR_CUDA;
  const SmallShape s = small_shape(a, h->sm_count);
  if (s.p_tiles == 0) return HQ_OK;
  SmallParams p{};
  p.by_c_tiles = fast_div((uint32_t)s.c_tiles); p.by_howo = fast_div((uint32_t)(a.ho * a.wo)); p.by_wo = fast_div((uint32_t)a.wo);
  p.by_cchunks = fast_div((uint32_t)((a.cin + s.bkb - 1) / s.bkb));
  p.by_cin = fast_div((uint32_t)a.cin); p.by_kw = fast_div((uint32_t)a.kw);
  p.x = a.in; p.h = a.h; p.w = a.w; p.cin = a.cin; p.wo = a.wo; p.howo = a.ho * a.wo;
  p.stride = a.stride; p.pad = a.pad; p.kh = a.kh; p.kw = a.kw;
  p.P = (int32_t)((long long)a.n * a.ho * a.wo); p.C = a.cout; p.K = a.kh * a.kw * a.cin;
  p.x_mode = s.x_mode; p.bkb = s.bkb; p.cchunks = (a.cin + s.bkb - 1) / s.bkb;
  p.tail_steps = (a.cin - (p.cchunks - 1) * s.bkb + 31) >> 5;
  p.nkb = s.nkb; p.lg_split = s.lg_split; p.stages = s.stages; p.pt = s.pt; p.c_tiles = s.c_tiles;
  while ((1 << p.lg_cols) < (s.pt >> s.lg_split)) ++p.lg_cols;
  p.fold = s.fold;
  p.x_bits = a.in_bits; p.x_signed = a.in_signed; p.params_late = a.params_late;
  const void* wgt = (a.in_bits == 4 && a.wgt_widened) ? a.wgt_widened : a.wgt;
  if (a.in_bits == 4 && !a.wgt_widened) p.w4 = a.wgt;
  const int stage_bytes = (kTileC + s.pt) * s.bkb;
  p.part_off = (uint32_t)(s.stages * stage_bytes);
  const int total = s.stages * stage_bytes + (s.lg_split ? s.pt * (s.fold ? 64 : kTileC) * 4 : 0);
  { const long long bound = (long long)p.K * (a.in_bits == 4 ? 15 * 8 : 255 * 128); while ((1LL << p.acc_bits) <= bound) ++p.acc_bits; }
  p.tmem_cols = s.pt <= 32 ? 32u : 64u;
  p.bias = a.bias; p.b = a.b; p.c = a.c;
  p.res = a.res; p.res_bits = a.res_bits; p.res_signed = a.res_signed; p.rb = a.rb; p.rc = a.rc;
  p.res_narrow = (a.res && a.res_bits == 8) ? (const int4*)a.res_narrow : nullptr; p.narrow_fresh = a.res_narrow_fresh;
  p.relu = a.relu; p.qmin = a.qmin; p.qmax = a.qmax; p.out = a.out; p.out_bits = a.out_bits; p.status = h->dev_status;
  {
    const int lo = a.relu ? (a.qmin > 0 ? a.qmin : 0) : a.qmin;
    p.sat = a.out_bits != 8 ? 0 : (!a.out_signed && lo == 0 && a.qmax == 255) ? 1 : (a.out_signed && lo == -128 && a.qmax == 127) ? 2 : 0;
  }

  alignas(64) CUtensorMap map_w{};
  if (!p.w4 && !encode_rows_map(&map_w, wgt, a.cout, p.K, s.bkb, 64, swizzle_for(s.bkb))) return HQ_ERR_CUDA;
  alignas(64) CUtensorMap map_x = map_w;
  if (s.x_mode == kXTiled && !encode_rows_map(&map_x, a.in, p.P, a.cin, s.bkb, s.pt, swizzle_for(s.bkb))) return HQ_ERR_CUDA;
  if (s.x_mode == kXIm2col && !encode_im2col_map(&map_x, a, s.bkb, s.pt)) return HQ_ERR_CUDA;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 1u << s.lg_split; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)((s.p_tiles * s.c_tiles) << s.lg_split)); cfg.blockDim = dim3(kSmallThreads);
  cfg.dynamicSmemBytes = (size_t)total + 1024; cfg.stream = stream; cfg.attrs = attr; cfg.numAttrs = s.lg_split ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, s.x_mode == kXGather ? conv_small_kernel<true> : conv_small_kernel<false>, map_w, map_x, p) == cudaSuccess ? HQ_OK : HQ_ERR_CUDA;
}

// The automatic path's choice.  Measured against the persistent kernel, both in a chain of dependent launches, us per launch:
//   - spatial filters over inputs below 128 KiB, which the persistent kernel only takes as a patch matrix (three launches):
//     3x3 128 at 28x28 n = 1 13.1 -> 5.8, 256 at 14x14 n = 1 17.1 -> 6.4, 512 at 7x7 n = 4 29.3 -> 8.9.  Four waves of tiles still win;
//   - otherwise while the tiles are resident at once, two CTAs per SM: 1x1 64 -> 64 at 56x56 n = 4 (196 tiles) 4.9 -> 3.5, n = 8
//     (392) 6.0 -> 6.8; 256 -> 1024 with residual at 14x14 n = 8 (200) 6.4 -> 4.8, n = 13 (320) 7.7 -> 8.6; 3x3 128 at 28x28
//     n = 24 (294) 10.1 -> 8.1; 1x1 2048 -> 1000, n = 1..24 11.2..12.1 -> 4.4..4.6;
//   - and while a CTA has few K blocks to walk: 9 blocks 9.1 -> 6.6 (3x3 128 at 28x28, n = 13), 16 blocks 8.1 -> 8.3 (2048 -> 512 at
//     7x7, n = 24), 36 blocks 13.3 -> 14.8 (3x3 512 at 7x7, n = 24).
bool hq_conv_small_wanted(const ConvArgs& a, int sm_count) {
  if (!hq_conv_small_supported(a, sm_count)) return false;
  const SmallShape s = small_shape(a, sm_count);
  const long long ctas = (s.p_tiles * s.c_tiles) << s.lg_split;
  ConvArgs b8 = a;
  b8.in_bits = 8;
  const bool direct = hq_conv_tc_supported(b8) && !hq_conv_tc_small_im2col(b8);
  if (!direct) return ctas <= 4LL * sm_count;
  return ctas <= 2LL * sm_count && (s.nkb >> s.lg_split) <= 12;
}
