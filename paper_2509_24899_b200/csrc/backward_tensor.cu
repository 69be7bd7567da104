// Gradient of the value-distillation loss w.r.t. the feature-map weights ("Attention Distillation"; Algorithm 1
// updates the feature maps only) on the tensor cores, for one-layer maps with d = F = 128 and no bias.  The chain rule
// (formulas in backward_simt.cu) is a handful of products per 128-token tile:
//
//   query side   A  = Q W_q^T                  pre-activations                   [tokens x F]
//                U  = g S^T                     g = sign(y_hat - y) / den         [tokens x F]
//                dS  += (lambda phi_q)^T g      state gradient                    [F x d]
//                dW_q += (dL/da_q)^T Q          dL/da_q = lambda (U + z s) phi'    [F x d]
//   key side     A  = K W_k^T,  T = V dS^T,     dW_k += (dL/da_k)^T K             dL/da_k = (T + dz) phi' on linear tokens
//
// bf16 operands, fp32 accumulation in TMEM.  dz = sum_i lambda phi_q,i s_i is summed in fp32 from the very bf16 values the
// dS product multiplies.  One CTA per (token chunk, batch*head); how each side is laid out stands before its kernel.  The
// chunks' partial results leave in the layout of the CUDA-core version and are added up by its fixed-order reduction
// kernels.  Every wait is bounded (status word, abort flag).
#include "backward_common.h"
#include "tensor_common.cuh"

namespace {

using namespace as_tc;

constexpr int BT_COMPUTE = 512;          // warps 0-15
constexpr int TILE = 128 * 128 * 2;      // bytes of a [128 x 128] bf16 tile

AS_DEV float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
AS_DEV float bf_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
AS_DEV uint32_t sub_bf16x2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("sub.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
// the two halves of a, read as bf16, minus b in fp32 (mixed-precision subtraction of sm_100)
AS_DEV float2 sub_bf16x2_f32(uint32_t a, float2 b) {
  float2 r;
  asm("{\n\t.reg .b16 lo, hi;\n\t"
      "mov.b32 {lo, hi}, %2;\n\t"
      "sub.rn.f32.bf16 %0, lo, %3;\n\t"
      "sub.rn.f32.bf16 %1, hi, %4;\n\t}"
      : "=f"(r.x), "=f"(r.y)
      : "r"(a), "f"(b.x), "f"(b.y));
  return r;
}
// all ones in the halves that differ (or are unordered)
AS_DEV uint32_t ne_bf16x2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("set.neu.u32.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}

// Writes 32 columns of one accumulator row (TMEM lane = feature row) to dst.
AS_DEV void bt_store_acc(uint32_t tacc, float* dst) {
  uint32_t x[32];
  tmem_ld32(tacc, x);
  tmem_ld_wait(x);
#pragma unroll
  for (int i = 0; i < 8; ++i) reinterpret_cast<uint4*>(dst)[i] = make_uint4(x[4 * i], x[4 * i + 1], x[4 * i + 2], x[4 * i + 3]);
}

// ---------------------------------------------------------------------------------------------- query side
// Tiles of 64 tokens.  Everything is laid out feature by feature: A^T and U^T land with TMEM lane = feature and column =
// token, the threads write lambda phi_q and dL/da_q back over them as packed bf16, and both gradient products take their A
// operand from there.  What is per feature (z, the power, dz) stays in a thread's registers, what is per token (lambda, s)
// is read from shared memory; no feature goes through shared memory, which leaves room to load four tiles ahead.  Eight
// warps turn y, y_hat into g (up to two tiles ahead), eight others work on the features, and A^T, U^T are double-buffered:
// the products of one tile, the features of another and the g of a third run side by side.  Headline layer, whole gradient:
// 203 us with everything laid out token by token (features and dL/da through shared memory, one 128-token tile at a time),
// 159 feature by feature but with all sixteen warps on the same phase of the same tile (8300 clk a tile: 2000 for g, 2200
// for the features, 700 to store them, 2400 waiting), 138 like this; N = 7800 81.5 -> 65.  What bounds it now is the issuing
// warp: 24 MMAs a tile at about 67 clk beside the compute warps and three waits of 200.
struct BtqLayout {
  static constexpr int QTILE = 64 * 128 * 2;      // bytes of a [64 tokens x 128] bf16 tile: two boxes of 64 columns
  static constexpr int QBOX = QTILE / 2;
  static constexpr int SLOTS = 4;
  static constexpr int W_OFF = 0;                 // W_q [F][d]
  static constexpr int S_OFF = TILE;              // S in bf16 [F][d]
  static constexpr int QY_OFF = 2 * TILE;         // ring of [q | y, then g in place]
  static constexpr int H_OFF = QY_OFF + SLOTS * 2 * QTILE;   // two tiles of y_hat
  static constexpr int VEC_OFF = H_OFF + 2 * QTILE;          // ring of s and lambda of the tile's tokens
  static constexpr int BAR_OFF = VEC_OFF + SLOTS * 512;
  static constexpr int TOTAL = BAR_OFF + 192;     // (the array is aligned to 1024 bytes)
  static constexpr int RED_OFF = QY_OFF;          // at the end: token groups' shares of dz, then the warps' loss sums
};
enum { Q_WFULL = 0, Q_QY = 1, Q_H = Q_QY + BtqLayout::SLOTS, Q_GRDY = Q_H + 2, Q_AU = Q_GRDY + BtqLayout::SLOTS, Q_PRDY = Q_AU + 2, Q_DONE = Q_PRDY + 2,
       Q_END = Q_DONE + BtqLayout::SLOTS, Q_BARS };
constexpr int BTQ_THREADS = BT_COMPUTE + 96;     // warps 0-7: features; 8-15: g; 16: MMA issue; 17: loads q, y, W, S; 18: loads y_hat
constexpr uint32_t ID_TOK64 = make_idesc(128, 64, 0, 0);    // [F x 64 tokens] = [F x d] [64 tokens x d]^T
constexpr uint32_t ID_TM = make_idesc(128, 128, 0, 1);      // A from tensor memory, B MN-major (token rows are the K index)
// [F x d] (two boxes of 128 rows) times a [64 tokens x d] tile (two boxes of 64 rows), both K-major
AS_DEV void btq_issue_tokens(uint32_t d_tmem, uint32_t mat, uint32_t tile) {
  const uint64_t a0 = kmajor_desc(mat), b0 = kmajor_desc(tile);
#pragma unroll
  for (int kk = 0; kk < 8; ++kk)
    mma_ss(d_tmem, a0 + kstep_kmajor(kk), b0 + (uint64_t)(((kk / 4) * BtqLayout::QBOX + (kk % 4) * 32) >> 4), ID_TOK64, kk > 0 ? 1u : 0u);
}
// [F x d] += [F x 64 tokens, packed bf16 in tensor memory] [64 tokens x d]
AS_DEV void btq_issue_grad(uint32_t d_tmem, uint32_t a_tmem, uint32_t tile, bool acc) {
  const uint64_t b0 = make_sdesc(tile, BtqLayout::QBOX, 1024);
#pragma unroll
  for (int kk = 0; kk < 4; ++kk) mma_ts(d_tmem, a_tmem + kk * 8, b0 + kstep_mnmajor(kk), ID_TM, (acc || kk > 0) ? 1u : 0u);
}

// One feature of 32 tokens: lambda phi_q and dL/da_q = lambda (U + z s) phi' as bf16 pairs; dz from the very bf16 values
// the dS product multiplies.  vec: s of the tokens, lambda 64 floats further on (EXACT; otherwise lambda is 1, and rows past
// the end have q, g and s zero).  Packed fp32x2 arithmetic: the threads' instruction count is what bounds the kernel.
template <int PW, bool EXACT>
AS_DEV void btq_features(const uint32_t (&xa)[32], const uint32_t (&xu)[32], const float* vec, float z, float2& dz, uint32_t (&wp)[16],
                         uint32_t (&wa)[16]) {
  const float2 z2 = make_float2(z, z);
#pragma unroll
  for (int i = 0; i < 16; i += 2) {
    const float4 s4 = *reinterpret_cast<const float4*>(vec + 2 * i);
    float4 l4;
    if (EXACT) l4 = *reinterpret_cast<const float4*>(vec + 64 + 2 * i);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int k = 2 * (i + j);
      const float2 s2 = j == 0 ? make_float2(s4.x, s4.y) : make_float2(s4.z, s4.w);
      const float a0 = __uint_as_float(xa[k]), a1 = __uint_as_float(xa[k + 1]);
      const float2 r = make_float2(fmaxf(a0, 0.f), fmaxf(a1, 0.f));
      const float2 t = __ffma2_rn(z2, s2, make_float2(__uint_as_float(xu[k]), __uint_as_float(xu[k + 1])));
      float2 ph = r, da;
      if (PW == 1) {
        da = __fmul2_rn(t, make_float2(a0 > 0.f ? 1.f : 0.f, a1 > 0.f ? 1.f : 0.f));      // (a product: a NaN reaches every feature)
      } else {
        float2 rp = r;                               // r^(p-1)
#pragma unroll
        for (int e = 2; e < PW; ++e) rp = __fmul2_rn(rp, r);
        ph = __fmul2_rn(rp, r);
        da = __fmul2_rn(__fmul2_rn(t, rp), make_float2((float)PW, (float)PW));
      }
      if (EXACT) {
        const float2 l2 = j == 0 ? make_float2(l4.x, l4.y) : make_float2(l4.z, l4.w);
        ph = __fmul2_rn(ph, l2);
        da = __fmul2_rn(da, l2);
      }
      wp[i + j] = pack_bf16(ph.x, ph.y);
      wa[i + j] = pack_bf16(da.x, da.y);
      dz = __ffma2_rn(make_float2(bf_lo(wp[i + j]), bf_hi(wp[i + j])), s2, dz);
    }
  }
}
template <int PW>
AS_DEV void btq_features(bool exact, const uint32_t (&xa)[32], const uint32_t (&xu)[32], const float* vec, float z, float2& dz,
                         uint32_t (&wp)[16], uint32_t (&wa)[16]) {
  if (exact) btq_features<PW, true>(xa, xu, vec, z, dz, wp, wa);
  else btq_features<PW, false>(xa, xu, vec, z, dz, wp, wa);
}

__global__ void __launch_bounds__(BTQ_THREADS, 1)
btq_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmY, const __grid_constant__ CUtensorMap tmH,
           const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmS, const __grid_constant__ BwParams p) {
  using L = BtqLayout;
  extern __shared__ __align__(1024) uint8_t btq_smem[];
  uint8_t* smem = btq_smem;
  const uint32_t sbase = smem_u32(smem);
  auto bar = [&](int i) { return sbase + L::BAR_OFF + 8 * i; };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::BAR_OFF + 8 * Q_BARS);
  volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem + L::BAR_OFF + 8 * Q_BARS + 4);
  volatile uint32_t* skip = reinterpret_cast<volatile uint32_t*>(smem + L::BAR_OFF + 8 * Q_BARS + 8);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int bh = blockIdx.y, chunk = blockIdx.x, h = bh % p.H;
  const int tok_begin = chunk * p.chunk_tokens;
  const int tok_end = min(p.N, tok_begin + p.chunk_tokens);
  const int nt = (tok_end - tok_begin + 63) / 64;

  if (threadIdx.x == 0) {
    *abort_flag = 0u;
    mbar_init(bar(Q_WFULL), 1); mbar_init(bar(Q_END), 1);
    for (int i = 0; i < L::SLOTS; ++i) { mbar_init(bar(Q_QY + i), 1); mbar_init(bar(Q_GRDY + i), 256); mbar_init(bar(Q_DONE + i), 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(bar(Q_H + i), 1); mbar_init(bar(Q_AU + i), 1); mbar_init(bar(Q_PRDY + i), 256); }
    fence_barrier_init();
    fence_proxy_async();
  }
  if (threadIdx.x == 32) *skip = status_now(p.status);
  if (warp == 16) { tmem_alloc(smem_u32(tmem_slot), 512); tmem_relinquish(); griddep_launch(); }
  if (threadIdx.x == 17 * 32) { tma_prefetch_desc(&tmQ); tma_prefetch_desc(&tmY); tma_prefetch_desc(&tmH); tma_prefetch_desc(&tmW); tma_prefetch_desc(&tmS); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  griddep_wait();                                    // the set-up above ran beside the kernel before this one
  // an earlier launch timed out: do nothing (decided once per CTA)
  if (*skip != 0u) {
    if (warp == 16) tmem_dealloc(*tmem_slot, 512);
    return;
  }
  const uint32_t tmem = *tmem_slot;
  const uint32_t tdS = tmem + 256, tdW = tmem + 384;
  auto tA = [&](int t) { return tmem + (t & 1) * 128u; };
  auto tU = [&](int t) { return tmem + (t & 1) * 128u + 64u; };
  const WaitCtx wc{p.status, abort_flag};
  auto slot_off = [&](int t) { return L::QY_OFF + (t % L::SLOTS) * 2 * L::QTILE; };
  bool ok = true;

  auto load = [&](uint32_t dst, const CUtensorMap* m, uint32_t fb, int t) {
    tma_load_3d(dst, m, fb, 0, tok_begin + t * 64, bh);
    tma_load_3d(dst + L::QBOX, m, fb, 64, tok_begin + t * 64, bh);
  };
  if (warp == 18) {
    if (lane == 0) {
      for (int t = 0; t < nt; ++t) {
        // (g of tile t - 2 is in its place: its y_hat has been read)
        if (t >= 2 && !mbar_wait(bar(Q_GRDY + (t - 2) % L::SLOTS), ((t - 2) / L::SLOTS) & 1, wc)) break;
        mbar_expect_tx(bar(Q_H + (t & 1)), L::QTILE);
        load(sbase + L::H_OFF + (t & 1) * L::QTILE, &tmH, bar(Q_H + (t & 1)), t);
      }
    }
    __syncwarp();
  } else if (warp == 17) {
    if (lane == 0) {
      for (int t = 0; t < nt; ++t) {
        const uint32_t fb = bar(Q_QY + t % L::SLOTS), dst = sbase + slot_off(t);
        // (the products of the tile that had the slot have read it)
        if (t >= L::SLOTS && !mbar_wait(bar(Q_DONE + t % L::SLOTS), (t / L::SLOTS - 1) & 1, wc)) break;
        mbar_expect_tx(fb, 2 * L::QTILE);
        load(dst + L::QTILE, &tmY, fb, t);
        load(dst, &tmQ, fb, t);
        if (t == 0) {
          mbar_expect_tx(bar(Q_WFULL), 2 * TILE);
          load_tile<128>(sbase + L::W_OFF, &tmW, bar(Q_WFULL), 0, h);
          load_tile<128>(sbase + L::S_OFF, &tmS, bar(Q_WFULL), 0, bh);
        }
      }
    }
    __syncwarp();
  } else if (warp == 16) {
    // The whole warp walks the loop, one elected lane issues: converged, the operands of an MMA stay in uniform registers.  (A
    // lane by itself took 110 clk an MMA beside the compute warps: 163 us instead of 138.  Two issuing warps, one for A^T and U^T,
    // one for the gradients: 144.)
    const uint32_t sb = __shfl_sync(0xffffffffu, sbase, 0), tm = __shfl_sync(0xffffffffu, tmem, 0);
    // A^T and U^T of tile t, over columns whose features the products of tile t - 2 read: those were issued before (one
    // thread's products complete in order), and the threads had read the A^T and U^T of that tile
    auto first_products = [&](int t) -> bool {
      const uint32_t sQ = sb + slot_off(t), sY = sQ + L::QTILE, tAU = tm + (t & 1) * 128u;
      if (!mbar_wait_warp(bar(Q_QY + t % L::SLOTS), (t / L::SLOTS) & 1, wc)) return false;
      tc_fence_after();
      if (elect_one()) btq_issue_tokens(tAU, sb + L::W_OFF, sQ);
      if (!mbar_wait_warp(bar(Q_GRDY + t % L::SLOTS), (t / L::SLOTS) & 1, wc)) return false;      // g over y
      tc_fence_after();
      if (elect_one()) {
        btq_issue_tokens(tAU + 64, sb + L::S_OFF, sY);
        tc_commit(bar(Q_AU + (t & 1)));
      }
      return true;
    };
    ok = mbar_wait_warp(bar(Q_WFULL), 0, wc) && first_products(0);
    for (int t = 0; t < nt && ok; ++t) {
      if (t + 1 < nt && !first_products(t + 1)) break;
      if (!mbar_wait_warp(bar(Q_PRDY + (t & 1)), (t >> 1) & 1, wc)) break;
      tc_fence_after();
      if (elect_one()) {
        const uint32_t sQ = sb + slot_off(t), sY = sQ + L::QTILE, tAU = tm + (t & 1) * 128u;
        btq_issue_grad(tm + 256, tAU, sY, t > 0);                       // dS += (lambda phi_q)^T g
        btq_issue_grad(tm + 384, tAU + 64, sQ, t > 0);                  // dW_q += (dL/da_q)^T Q
        tc_commit(bar(Q_DONE + t % L::SLOTS));
        if (t == nt - 1) tc_commit(bar(Q_END));
      }
    }
  } else {
    float* red = reinterpret_cast<float*>(smem + L::RED_OFF);
    const bool exact = p.stab_mode == AS_STAB_EXACT && p.n_s > 0;
    const int r = threadIdx.x & 127, cg = threadIdx.x >> 7;    // TMEM lane; group of columns
    const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
    float2 dz = make_float2(0.f, 0.f);
    float loss = 0.f;
    if (warp >= 8) {
      // ---------------------------------------------------------------- g = sign(y_hat - y) / den over y
      // four lanes share a token row, and take its 16-byte pieces in an order in which a warp's lanes hit different banks
      const int gr = (threadIdx.x - 256) >> 2, gq = threadIdx.x & 3;
      // the row's statistics of the forward pass (c_i, the two parts of the denominator), fetched one tile ahead
      auto row_stats = [&](int t, float (&a)[3]) {
        const int n = tok_begin + t * 64 + gr;
        if (t < nt && n < tok_end) {
          const float* ap = p.aux + ((size_t)bh * p.N + n) * 3;
          a[0] = ap[0]; a[1] = ap[1]; a[2] = ap[2];
        } else {
          a[0] = 0.f; a[1] = 1.f; a[2] = 0.f;
        }
      };
      float st_next[3];
      row_stats(0, st_next);
      for (int t = 0; t < nt; ++t) {
        const float st_c[3] = {st_next[0], st_next[1], st_next[2]};
        row_stats(t + 1, st_next);
        float* vec = reinterpret_cast<float*>(smem + L::VEC_OFF) + (t % L::SLOTS) * 128;
        if (ok) ok = mbar_wait_warp(bar(Q_H + (t & 1)), (t >> 1) & 1, wc);
        if (ok) ok = mbar_wait_warp(bar(Q_QY + t % L::SLOTS), (t / L::SLOTS) & 1, wc);
        if (ok) {
          uint8_t* sY = smem + slot_off(t) + L::QTILE;
          const uint8_t* sH = smem + L::H_OFF + (t & 1) * L::QTILE;
          float lam = 0.f, den = 1.f;
          if (tok_begin + t * 64 + gr < tok_end) {
            lam = exact ? __expf(-st_c[0]) : 1.f;
            den = st_c[1] + lam * st_c[2];
          }
          const float inv_den = 1.f / den;
          const uint32_t inv2 = pack_bf16(inv_den, inv_den);
          float2 hs = make_float2(0.f, 0.f), ls = make_float2(0.f, 0.f);      // sums of G y_hat and of -|y_hat - y|
#pragma unroll
          for (int c4 = 0; c4 < 4; ++c4) {
            const uint32_t off = (gq >> 1) * L::QBOX + swz128_chunk_offset(gr, (gq & 1) * 4 + (c4 ^ ((gq >> 1) << 1)));
            const uint4 yv = *reinterpret_cast<const uint4*>(sY + off), hv = *reinterpret_cast<const uint4*>(sH + off);
            const uint32_t yw[4] = {yv.x, yv.y, yv.z, yv.w}, hw[4] = {hv.x, hv.y, hv.z, hv.w};
            uint32_t gw[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              // on pairs of bf16: the sign of y_hat - y (rounding a difference changes neither its sign nor whether it is zero),
              // none where it is zero - and rows past the end of the sequence arrive as zeros.  (Infinity less infinity is not zero: such
              // an element makes the loss and the row's gradient NaN.)
              const uint32_t diff = sub_bf16x2(hw[i], yw[i]), sign = diff & 0x80008000u, differ = ne_bf16x2(diff, 0u);
              gw[i] = (inv2 ^ sign) & differ;
              const uint32_t Gh = (hw[i] ^ sign) & differ, Gy = (yw[i] ^ sign) & differ;
              const float2 h2 = make_float2(bf_lo(Gh), bf_hi(Gh));
              hs = __fadd2_rn(hs, h2);
              // the differences in fp32 one by one: a difference of two sums would cancel where y_hat is close to y (y_hat one bf16 unit
              // from y, values spread over several decades: 2e-6 to 9e-6 off)
              ls = __fadd2_rn(ls, sub_bf16x2_f32(Gy, h2));
            }
            *reinterpret_cast<uint4*>(sY + off) = make_uint4(gw[0], gw[1], gw[2], gw[3]);
          }
          float sdot = hs.x + hs.y;
          loss -= ls.x + ls.y;                         // sum of |y_hat - y|
          sdot += __shfl_xor_sync(0xffffffffu, sdot, 1);
          sdot += __shfl_xor_sync(0xffffffffu, sdot, 2);
          if (gq == 0) {
            vec[gr] = -sdot * inv_den;                 // s = -(g . y_hat)
            vec[64 + gr] = lam;
          }
        }
        fence_proxy_async();
        mbar_arrive(bar(Q_GRDY + t % L::SLOTS));
      }
    } else {
      // ---------------------------------------------------------------- features: lane = feature, 32 of the tile's tokens
      const int pw = min(((warp & 3) * 32) / (128 / p.P), p.P - 1) + 1;    // power of this warp's features
      const float z = p.z[(size_t)bh * 128 + r];
      for (int t = 0; t < nt; ++t) {
        const float* vec = reinterpret_cast<const float*>(smem + L::VEC_OFF) + (t % L::SLOTS) * 128;
        if (ok) ok = mbar_wait_warp(bar(Q_AU + (t & 1)), (t >> 1) & 1, wc);
        // (U^T is complete only after every g thread has arrived on the tile's g barrier: s and lambda of every token are there)
        uint32_t wp[16], wa[16];
        if (ok) {
          tc_fence_after();
          uint32_t xa[32], xu[32];
          tmem_ld32(tA(t) + lane_off + cg * 32, xa);
          tmem_ld32(tU(t) + lane_off + cg * 32, xu);
          tmem_ld_wait(xa);
          tmem_ld_wait(xu);
          switch (pw) {
            case 1: btq_features<1>(exact, xa, xu, vec + cg * 32, z, dz, wp, wa); break;
            case 2: btq_features<2>(exact, xa, xu, vec + cg * 32, z, dz, wp, wa); break;
            case 3: btq_features<3>(exact, xa, xu, vec + cg * 32, z, dz, wp, wa); break;
            default: btq_features<4>(exact, xa, xu, vec + cg * 32, z, dz, wp, wa); break;
          }
        }
        named_barrier_sync(2 + (warp & 3), 64);        // both token groups of these lanes have read A^T and U^T
        if (ok) {
          tmem_st16(tA(t) + lane_off + cg * 16, wp);
          tmem_st16(tU(t) + lane_off + cg * 16, wa);
          tmem_st_wait();
          tc_fence_before();
        }
        mbar_arrive(bar(Q_PRDY + (t & 1)));
      }
    }
    // ---- the chunk's partial results
    const uint32_t late = status_now(p.status);      // behind the wait, ahead of the first write: not 0, and nothing is written
    if (ok && nt > 0) ok = mbar_wait_warp(bar(Q_END), 0, wc);
    const size_t slot = (size_t)bh * p.chunks + chunk;
    if (ok && late == 0u && nt > 0) {
      tc_fence_after();
      bt_store_acc(tdS + lane_off + cg * 32, p.part_dS + (slot * 128 + r) * 128 + cg * 32);
      bt_store_acc(tdW + lane_off + cg * 32, p.part_dW + (slot * 128 + r) * 128 + cg * 32);
      tc_fence_before();
    }
    // dz of the chunk: the two token groups' shares; the loss: the eight g warps' sums in warp order
    if (cg < 2) red[cg * 128 + r] = dz.x + dz.y;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, off);
    if (lane == 0 && warp >= 8) red[256 + warp - 8] = loss;
    named_barrier_sync(1, BT_COMPUTE);
    if (cg == 0 && late == 0u) p.part_dz[slot * 128 + r] = red[r] + red[128 + r];
    if (threadIdx.x == 128 && late == 0u) {
      float l = 0.f;
      for (int w = 0; w < 8; ++w) l += red[256 + w];
      p.part_loss[slot] = l;
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 16) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// ---------------------------------------------------------------------------------------------- key side
// As the query side: A^T = W_k K^T and T^T = dS V^T with TMEM lane = feature, dL/da_k written back over A^T as packed bf16,
// dW_k += (dL/da_k)^T K with that as the A operand.  Two groups of eight warps take turns at the tiles, each with columns
// of its own.  (Before: 128-token tiles, all sixteen warps on one, dL/da_k through shared memory.  Whole gradient 136.9 -> 130.5
// us at the headline shape, 63.1 -> 61.9 at N = 7800.)
struct BtkLayout {
  static constexpr int QTILE = BtqLayout::QTILE;
  static constexpr int SLOTS = 5;
  static constexpr int W_OFF = 0;                 // W_k [F][d]
  static constexpr int S_OFF = TILE;              // dS in bf16 [F][d]
  static constexpr int KV_OFF = 2 * TILE;         // ring of [k | v]
  static constexpr int BAR_OFF = KV_OFF + SLOTS * 2 * QTILE;
  static constexpr int TOTAL = BAR_OFF + 192;     // (the array is aligned to 1024 bytes)
};
enum { K_WFULL = 0, K_FULL = 1, K_AT = K_FULL + BtkLayout::SLOTS, K_PRDY = K_AT + 2, K_DONE = K_PRDY + 2, K_END = K_DONE + BtkLayout::SLOTS, K_BARS };
constexpr int BTK_THREADS = BT_COMPUTE + 64;      // warps 0-15: features; 16: MMA issue; 17: loads

// One feature of 32 tokens: dL/da_k = (T + dz) phi' on linear tokens (bits of `linear`), zero on the others.
template <int PW>
AS_DEV void btk_features(const uint32_t (&xa)[32], const uint32_t (&xt)[32], float dz, uint32_t linear, uint32_t (&wa)[16]) {
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const float a0 = __uint_as_float(xa[2 * i]), a1 = __uint_as_float(xa[2 * i + 1]);
    float2 t = __fadd2_rn(make_float2(__uint_as_float(xt[2 * i]), __uint_as_float(xt[2 * i + 1])), make_float2(dz, dz));
    if (PW == 1) {
      t = __fmul2_rn(t, make_float2(a0 > 0.f ? 1.f : 0.f, a1 > 0.f ? 1.f : 0.f));
    } else {
      const float2 r = make_float2(fmaxf(a0, 0.f), fmaxf(a1, 0.f));
      float2 rp = r;                                 // r^(p-1)
#pragma unroll
      for (int e = 2; e < PW; ++e) rp = __fmul2_rn(rp, r);
      t = __fmul2_rn(__fmul2_rn(t, rp), make_float2((float)PW, (float)PW));
    }
    wa[i] = pack_bf16((linear >> (2 * i)) & 1u ? t.x : 0.f, (linear >> (2 * i + 1)) & 1u ? t.y : 0.f);
  }
}

__global__ void __launch_bounds__(BTK_THREADS, 1)
btk_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmW,
           const __grid_constant__ CUtensorMap tmS, const __grid_constant__ BwParams p) {
  using L = BtkLayout;
  extern __shared__ __align__(1024) uint8_t btq_smem[];
  uint8_t* smem = btq_smem;
  const uint32_t sbase = smem_u32(smem);
  auto bar = [&](int i) { return sbase + L::BAR_OFF + 8 * i; };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::BAR_OFF + 8 * K_BARS);
  volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem + L::BAR_OFF + 8 * K_BARS + 4);
  volatile uint32_t* skip = reinterpret_cast<volatile uint32_t*>(smem + L::BAR_OFF + 8 * K_BARS + 8);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int bh = blockIdx.y, chunk = blockIdx.x, h = bh % p.H;
  const int tok_begin = chunk * p.chunk_tokens;
  const int tok_end = min(p.N, tok_begin + p.chunk_tokens);
  const int nt = (tok_end - tok_begin + 63) / 64;

  if (threadIdx.x == 0) {
    *abort_flag = 0u;
    mbar_init(bar(K_WFULL), 1); mbar_init(bar(K_END), 1);
    for (int i = 0; i < L::SLOTS; ++i) { mbar_init(bar(K_FULL + i), 1); mbar_init(bar(K_DONE + i), 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(bar(K_AT + i), 1); mbar_init(bar(K_PRDY + i), 256); }
    fence_barrier_init();
    fence_proxy_async();
  }
  if (threadIdx.x == 32) *skip = status_now(p.status);
  if (warp == 16) { tmem_alloc(smem_u32(tmem_slot), 512); tmem_relinquish(); griddep_launch(); }
  if (threadIdx.x == 17 * 32) { tma_prefetch_desc(&tmK); tma_prefetch_desc(&tmV); tma_prefetch_desc(&tmW); tma_prefetch_desc(&tmS); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  griddep_wait();                                    // the set-up above ran beside the kernel before this one
  // an earlier launch timed out: do nothing (decided once per CTA)
  if (*skip != 0u) {
    if (warp == 16) tmem_dealloc(*tmem_slot, 512);
    return;
  }
  const uint32_t tmem = *tmem_slot;
  const WaitCtx wc{p.status, abort_flag};
  auto slot_off = [&](int t) { return L::KV_OFF + (t % L::SLOTS) * 2 * L::QTILE; };
  bool ok = true;

  if (warp == 17) {
    if (lane == 0) {
      auto load = [&](uint32_t dst, const CUtensorMap* m, uint32_t fb, int t) {
        tma_load_3d(dst, m, fb, 0, tok_begin + t * 64, bh);
        tma_load_3d(dst + BtqLayout::QBOX, m, fb, 64, tok_begin + t * 64, bh);
      };
      mbar_expect_tx(bar(K_WFULL), 2 * TILE);
      load_tile<128>(sbase + L::W_OFF, &tmW, bar(K_WFULL), 0, h);
      load_tile<128>(sbase + L::S_OFF, &tmS, bar(K_WFULL), 0, bh);
      for (int t = 0; t < nt; ++t) {
        const uint32_t fb = bar(K_FULL + t % L::SLOTS), dst = sbase + slot_off(t);
        // (the product of the tile that had the slot has read it)
        if (t >= L::SLOTS && !mbar_wait(bar(K_DONE + t % L::SLOTS), (t / L::SLOTS - 1) & 1, wc)) break;
        mbar_expect_tx(fb, 2 * L::QTILE);
        load(dst, &tmK, fb, t);
        load(dst + L::QTILE, &tmV, fb, t);
      }
    }
    __syncwarp();
  } else if (warp == 16) {
    const uint32_t sb = __shfl_sync(0xffffffffu, sbase, 0), tm = __shfl_sync(0xffffffffu, tmem, 0);
    // A^T and T^T of tile t over columns whose features the product of tile t - 2 reads: that was issued before (one
    // thread's products complete in order), and the threads had read the A^T and T^T of that tile
    auto first_products = [&](int t) -> bool {
      const uint32_t sK = sb + slot_off(t), tAT = tm + (t & 1) * 128u;
      if (!mbar_wait_warp(bar(K_FULL + t % L::SLOTS), (t / L::SLOTS) & 1, wc)) return false;
      tc_fence_after();
      if (elect_one()) {
        btq_issue_tokens(tAT, sb + L::W_OFF, sK);
        btq_issue_tokens(tAT + 64, sb + L::S_OFF, sK + L::QTILE);
        tc_commit(bar(K_AT + (t & 1)));
      }
      return true;
    };
    ok = mbar_wait_warp(bar(K_WFULL), 0, wc) && first_products(0) && (nt < 2 || first_products(1));
    for (int t = 0; t < nt && ok; ++t) {
      if (!mbar_wait_warp(bar(K_PRDY + (t & 1)), (t >> 1) & 1, wc)) break;
      tc_fence_after();
      if (elect_one()) {
        btq_issue_grad(tm + 256, tm + (t & 1) * 128u, sb + slot_off(t), t > 0);   // dW_k += (dL/da_k)^T K
        tc_commit(bar(K_DONE + t % L::SLOTS));
        if (t == nt - 1) tc_commit(bar(K_END));
      }
      if (t + 2 < nt && !first_products(t + 2)) break;
    }
  } else {
    const int r = threadIdx.x & 127, cg = threadIdx.x >> 7;    // feature (= TMEM lane); tile group and token group: cg = 2 * group + tokens
    const int grp = cg >> 1, tg = cg & 1;
    const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
    const int pw = min(((warp & 3) * 32) / (128 / p.P), p.P - 1) + 1;    // power of this warp's features
    const uint32_t tA = tmem + grp * 128u, tT = tA + 64;
    const float dz = p.dz[(size_t)bh * 128 + r];
    // which of the tile's 32 tokens are linear tokens, fetched a turn ahead
    auto linear_tokens = [&](int t) {
      const int n = tok_begin + t * 64 + tg * 32 + lane;
      return __ballot_sync(0xffffffffu, t < nt && n < tok_end && p.sm_rank[n] < 0);
    };
    uint32_t lin_next = linear_tokens(grp);
    for (int t = grp; t < nt; t += 2) {
      const uint32_t lin = lin_next;
      lin_next = linear_tokens(t + 2);
      if (ok) ok = mbar_wait_warp(bar(K_AT + grp), (t >> 1) & 1, wc);
      uint32_t wa[16];
      if (ok) {
        tc_fence_after();
        uint32_t xa[32], xt[32];
        tmem_ld32(tA + lane_off + tg * 32, xa);
        tmem_ld32(tT + lane_off + tg * 32, xt);
        tmem_ld_wait(xa);
        tmem_ld_wait(xt);
        switch (pw) {
          case 1: btk_features<1>(xa, xt, dz, lin, wa); break;
          case 2: btk_features<2>(xa, xt, dz, lin, wa); break;
          case 3: btk_features<3>(xa, xt, dz, lin, wa); break;
          default: btk_features<4>(xa, xt, dz, lin, wa); break;
        }
      }
      named_barrier_sync(2 + (warp & 3) + 4 * grp, 64);        // both token groups of these lanes have read A^T
      if (ok) {
        tmem_st16(tA + lane_off + tg * 16, wa);
        tmem_st_wait();
        tc_fence_before();
      }
      mbar_arrive(bar(K_PRDY + grp));
    }
    const uint32_t late = status_now(p.status);      // behind the wait, ahead of the first write: not 0, and nothing is written
    if (ok && nt > 0) ok = mbar_wait_warp(bar(K_END), 0, wc);
    if (ok && late == 0u && nt > 0) {
      tc_fence_after();
      const size_t slot = (size_t)bh * p.chunks + chunk;
      bt_store_acc(tmem + 256 + lane_off + cg * 32, p.part_dW + (slot * 128 + r) * 128 + cg * 32);
      tc_fence_before();
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 16) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

}  // namespace

cudaError_t as_bw_tensor_init() {
  cudaError_t e;
  if ((e = opt_in_smem(btq_kernel, BtqLayout::TOTAL)) != cudaSuccess) return e;
  return opt_in_smem(btk_kernel, BtkLayout::TOTAL);
}

cudaError_t as_bw_tensor_query(const BwParams& p, cudaStream_t st) {
  const int BH = p.B * p.H;
  CUtensorMap tmQ, tmY, tmH, tmW, tmS;
  if (!make_map(&tmQ, p.q, 128, p.N, BH, 64) || !make_map(&tmY, p.y, 128, p.N, BH, 64) ||
      !make_map(&tmH, p.yhat, 128, p.N, BH, 64) || !make_map(&tmW, p.wq, 128, 128, p.H, 128) ||
      !make_map(&tmS, p.Sb, 128, 128, BH, 128))
    return cudaErrorInvalidValue;
  return as_launch_dependent(btq_kernel, dim3(p.chunks, BH), dim3(BTQ_THREADS), BtqLayout::TOTAL, st, tmQ, tmY, tmH, tmW, tmS, p);
}

cudaError_t as_bw_tensor_key(const BwParams& p, cudaStream_t st) {
  const int BH = p.B * p.H;
  CUtensorMap tmK, tmV, tmW, tmS;
  if (!make_map(&tmK, p.k, 128, p.N, BH, 64) || !make_map(&tmV, p.v, 128, p.N, BH, 64) ||
      !make_map(&tmW, p.wk, 128, 128, p.H, 128) || !make_map(&tmS, p.dSb, 128, 128, BH, 128))
    return cudaErrorInvalidValue;
  return as_launch_dependent(btk_kernel, dim3(p.chunks, BH), dim3(BTK_THREADS), BtkLayout::TOTAL, st, tmK, tmV, tmW, tmS, p);
}
