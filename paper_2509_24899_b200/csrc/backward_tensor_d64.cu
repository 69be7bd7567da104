// Gradient of the value-distillation loss w.r.t. the feature-map weights on the tensor cores for one-layer maps with
// d = F = 64, with the precision of the fp32 CUDA-core kernels (formulas in backward_simt.cu).
//
// Every product of the chain rule has one operand that bf16 holds exactly: the inputs q, k, v, W and - once 1 / den is
// moved to the other side - the signs G = sign(y_hat - y).  The other operand (S, dS, the features, dL/da) is an fp32
// value; it is cut into three bf16 pieces of eight significant bits each (x = hi + mid + lo exactly), and the three
// products are added in fp32.  With w = lambda / den and t = -(G . y_hat) of a token:
//
//   query side   A = Q W_q^T,  U = G S^T                       [tokens x F]
//                phi' slope of phi at A:  X = [ w phi | w (U + z t) phi' ]          [tokens x 2F], three pieces
//                X^T [ G | Q ]  holds dS in its upper left and dW_q in its lower right quarter
//                dz = sum of (w phi) t over the tokens, fp32 in registers
//   key side     A = K W_k^T,  T = V dS^T,  X = (T + dz) phi' on linear tokens, three pieces;  dW_k = X^T K
//
// (The two quarters of X^T [G | Q] that nothing reads come for free: an M = 128 product costs the same tensor time as
// the two M = 64 products it replaces.)  One CTA per (token chunk, batch*head), one 128-token tile at a time: sixteen
// compute warps, a token row (= TMEM lane) shared by four threads with 16 features each; lane 0 of warp 16 loads the
// tiles and issues the products.  The chunks' partial results leave in the layout of the CUDA-core version and are
// added up by its fixed-order reduction kernels.  Every wait is bounded (status word, abort flag).
//
// Errors against 64 bits from the same y_hat, aux, S, z, over B * H = 1 .. 180, N = 63 .. 31200, rates 0 .. 32: 0.8 - 2.3e-7
// on dW_q and 0.9 - 4.0e-7 on dW_k, against 1.1 - 5.6e-7 and 1.3 - 7.1e-7 of the CUDA-core kernels.  Time of a step
// (forward and gradient) at B = 2, H = 12, N = 2430: 594 us with the CUDA-core kernels (327 + 237 us of it theirs), 107 us
// with these.  What bounds them is the chain of one tile (load -> G -> U -> features -> final product, about 2 us) and,
// at that size, the set-up and the drain around four tiles a CTA.
#include "backward_common.h"
#include "tensor_common.cuh"

namespace {

using namespace as_tc;

constexpr int BS_COMPUTE = 512;
constexpr int BS_THREADS = BS_COMPUTE + 32;
constexpr int MAT = 64 * 64 * 2;         // bytes of a [64 x 64] bf16 matrix
constexpr int BOX = BOX_BYTES;           // bytes of a [128 tokens x 64] bf16 tile
constexpr uint32_t ID_TOK = make_idesc(128, 64, 0, 0);      // [tokens x 64] = [tokens x d] [64 x d]^T
constexpr uint32_t ID_Q2 = make_idesc(128, 128, 1, 1);      // X^T [G | Q]
constexpr uint32_t ID_K2 = make_idesc(128, 64, 1, 1);       // [two pieces of X]^T K

// x = hi + mid + lo with eight significant bits each, by truncation: exact, and nothing overflows.  A value that is
// not finite is all in hi (the pieces of an infinity would add up to NaN).
AS_DEV void split3(float x0, float x1, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
  const uint32_t u0 = __float_as_uint(x0), u1 = __float_as_uint(x1);
  hi = __byte_perm(u0, u1, 0x7632);
  float r0 = x0 - __uint_as_float(u0 & 0xffff0000u), r1 = x1 - __uint_as_float(u1 & 0xffff0000u);
  const float inf = __uint_as_float(0x7f800000u);
  r0 = fabsf(x0) < inf ? r0 : 0.f;
  r1 = fabsf(x1) < inf ? r1 : 0.f;
  const uint32_t m0 = __float_as_uint(r0), m1 = __float_as_uint(r1);
  mid = __byte_perm(m0, m1, 0x7632);
  const float l0 = r0 - __uint_as_float(m0 & 0xffff0000u), l1 = r1 - __uint_as_float(m1 & 0xffff0000u);
  lo = __byte_perm(__float_as_uint(l0), __float_as_uint(l1), 0x7632);
}
AS_DEV void st_shared4(uint32_t addr, const uint32_t* w) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]) : "memory");
}
// The three pieces of a [64 x 64] fp32 matrix as swizzled K-major tiles, by the 512 compute threads.
AS_DEV void split_matrix(const float* src, uint32_t dst, int tid) {
  const int f = tid >> 3, c = tid & 7;
  const float4 a = *reinterpret_cast<const float4*>(src + f * 64 + c * 8);
  const float4 b = *(reinterpret_cast<const float4*>(src + f * 64 + c * 8) + 1);
  uint32_t w[3][4];
  split3(a.x, a.y, w[0][0], w[1][0], w[2][0]);
  split3(a.z, a.w, w[0][1], w[1][1], w[2][1]);
  split3(b.x, b.y, w[0][2], w[1][2], w[2][2]);
  split3(b.z, b.w, w[0][3], w[1][3], w[2][3]);
  const uint32_t at = dst + swz128_chunk_offset(f, c);
#pragma unroll
  for (int i = 0; i < 3; ++i) st_shared4(at + i * MAT, w[i]);
}
// Sixteen fp32 values of token row r, columns [c0, c0 + 16) of a 64-column box, as three boxes `stride` bytes apart.
AS_DEV void store_split16(uint32_t box, uint32_t stride, uint32_t r, uint32_t c0, const float (&x)[16]) {
  const uint32_t base = box + r * 128u + ((r & 7u) << 4), ch = c0 / 8;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t w[3][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) split3(x[h * 8 + 2 * i], x[h * 8 + 2 * i + 1], w[0][i], w[1][i], w[2][i]);
#pragma unroll
    for (int i = 0; i < 3; ++i) st_shared4((base ^ ((ch + h) << 4)) + i * stride, w[i]);
  }
}
// T = sum over the three pieces, smallest first: [tokens x 64] = X[tokens x 64] (piece)^T
AS_DEV void issue_pieces(uint32_t d_tmem, uint32_t x_box, uint32_t pieces) {
#pragma unroll
  for (int i = 2; i >= 0; --i) issue_kmajor<64>(d_tmem, kmajor_desc(x_box), kmajor_desc(pieces + i * MAT), ID_TOK, i < 2);
}
// acc += 16 columns of one accumulator lane.  The tensor cores round a running sum toward zero at every step of 16
// tokens; summed over a whole chunk that is an error of up to 1.5e-5 in dW_q, against 3e-7 of the fp32 FMA chains this
// replaces.  So an accumulator holds one tile only and the tiles are added here, rounded to nearest.
AS_DEV void add_acc16(uint32_t tacc, float (&acc)[16]) {
  uint32_t x[16];
  tc_fence_after();
  tmem_ld16(tacc, x);
  tmem_ld16_wait(x);
  tc_fence_before();
#pragma unroll
  for (int i = 0; i < 16; ++i) acc[i] += __uint_as_float(x[i]);
}

// ---------------------------------------------------------------------------------------------- query side
struct BsqLayout {
  static constexpr int W_OFF = 0;                           // W_q [64][64]
  static constexpr int S_OFF = MAT;                         // S, three pieces
  static constexpr int IN_OFF = 4 * MAT;                    // two stages of [y, then G in place | q | y_hat]
  static constexpr int STAGE = 3 * BOX;
  static constexpr int X_OFF = IN_OFF + 2 * STAGE;          // three pieces of [w phi | dL/da]
  static constexpr int BAR_OFF = X_OFF + 6 * BOX;
  static constexpr int T_OFF = BAR_OFF + 128;               // 2 x 128 floats: t of the tile's rows, per tile parity
  static constexpr int Z_OFF = T_OFF + 1024;                // 64 floats: z
  static constexpr int TOTAL = Z_OFF + 256 + 1024;          // + slack for the 1024-byte alignment
};
enum { Q_WFULL = 0, Q_FULL = 1, Q_GRDY = 3, Q_AU = 4, Q_XRDY = 5, Q_DONE = 6, Q_BARS = 7 };

template <int PW>
AS_DEV void bsq_features(const uint32_t (&xa)[16], const uint32_t (&xu)[16], const float* zv, float t, float w, float (&ph)[16],
                         float (&da)[16], float (&dz)[16]) {
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const float a = __uint_as_float(xa[i]), r = fmaxf(a, 0.f);
    const float slope = PW == 1 ? (a > 0.f ? 1.f : 0.f) : 2.f * r;
    ph[i] = w * (PW == 1 ? r : r * r);
    da[i] = w * fmaf(zv[i], t, __uint_as_float(xu[i])) * slope;
    dz[i] = fmaf(ph[i], t, dz[i]);
  }
}

__global__ void __launch_bounds__(BS_THREADS, 1)
bsq_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmY, const __grid_constant__ CUtensorMap tmH,
           const __grid_constant__ CUtensorMap tmW, const __grid_constant__ BwParams p) {
  using L = BsqLayout;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t sbase = smem_u32(smem);
  auto bar = [&](int i) { return sbase + L::BAR_OFF + 8 * i; };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::BAR_OFF + 8 * Q_BARS);
  volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem + L::BAR_OFF + 8 * Q_BARS + 4);
  float* tvec = reinterpret_cast<float*>(smem + L::T_OFF);
  float* zvec = reinterpret_cast<float*>(smem + L::Z_OFF);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int bh = blockIdx.y, chunk = blockIdx.x, h = bh % p.H;
  const int tok_begin = chunk * p.chunk_tokens;
  const int tok_end = min(p.N, tok_begin + p.chunk_tokens);
  const int nt = (tok_end - tok_begin + 127) / 128;

  if (threadIdx.x == 0) {
    *abort_flag = 0u;
    mbar_init(bar(Q_WFULL), 1); mbar_init(bar(Q_FULL), 1); mbar_init(bar(Q_FULL + 1), 1); mbar_init(bar(Q_GRDY), BS_COMPUTE);
    mbar_init(bar(Q_AU), 1); mbar_init(bar(Q_XRDY), BS_COMPUTE); mbar_init(bar(Q_DONE), 1);
    fence_barrier_init();
    fence_proxy_async();
  }
  __shared__ uint32_t s_skip;
  if (threadIdx.x == 32) s_skip = status_now(p.status);
  if (warp == 16) { tmem_alloc(smem_u32(tmem_slot), 256); tmem_relinquish(); griddep_launch(); }
  if (threadIdx.x == 15 * 32) { tma_prefetch_desc(&tmQ); tma_prefetch_desc(&tmY); tma_prefetch_desc(&tmH); tma_prefetch_desc(&tmW); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  griddep_wait();                                    // the set-up above ran beside the kernel before this one
  // an earlier launch timed out: do nothing (decided once per CTA)
  if (s_skip != 0u) {
    if (warp == 16) tmem_dealloc(*tmem_slot, 256);
    return;
  }
  const uint32_t tmem = *tmem_slot;
  const uint32_t tA = tmem, tU = tmem + 64, tAcc = tmem + 128;
  const WaitCtx wc{p.status, abort_flag};
  auto stage = [&](int t) { return L::IN_OFF + (t & 1) * L::STAGE; };

  if (warp == 16) {
    if (lane == 0) {
      auto request = [&](int t) {
        const uint32_t fb = bar(Q_FULL + (t & 1)), dst = sbase + stage(t);
        const int row0 = tok_begin + t * 128;
        mbar_expect_tx(fb, 3 * BOX);
        tma_load_3d(dst, &tmY, fb, 0, row0, bh);
        tma_load_3d(dst + 2 * BOX, &tmH, fb, 0, row0, bh);
        tma_load_3d(dst + BOX, &tmQ, fb, 0, row0, bh);
      };
      request(0);
      mbar_expect_tx(bar(Q_WFULL), MAT);
      tma_load_3d(sbase + L::W_OFF, &tmW, bar(Q_WFULL), 0, 0, h);
      if (nt > 1) request(1);
      bool ok = mbar_wait(bar(Q_WFULL), 0, wc);
      for (int t = 0; t < nt && ok; ++t) {
        const uint32_t in = sbase + stage(t);
        // (the threads have read A and U of the tile before: they arrived on the X barrier)
        if (!mbar_wait(bar(Q_FULL + (t & 1)), (t >> 1) & 1, wc)) break;
        tc_fence_after();
        issue_kmajor<64>(tA, kmajor_desc(in + BOX), kmajor_desc(sbase + L::W_OFF), ID_TOK, false);
        if (!mbar_wait(bar(Q_GRDY), t & 1, wc)) break;       // G over y (and, at t = 0, the pieces of S)
        tc_fence_after();
        issue_pieces(tU, in, sbase + L::S_OFF);
        tc_commit(bar(Q_AU));
        if (t > 0 && t + 1 < nt) {
          if (!mbar_wait(bar(Q_DONE), (t - 1) & 1, wc)) break;   // the stage of tile t - 1 is free
          request(t + 1);
        }
        if (!mbar_wait(bar(Q_XRDY), t & 1, wc)) break;
        tc_fence_after();
        const uint64_t b0 = mnmajor_desc(in);                // [G | q]
#pragma unroll
        for (int i = 2; i >= 0; --i) {                       // smallest pieces first: a tile's sum is rounded at its own size 8 times, not 24
          const uint64_t a0 = mnmajor_desc(sbase + L::X_OFF + i * 2 * BOX);
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)
            mma_ss(tAcc, a0 + kstep_mnmajor(kk), b0 + kstep_mnmajor(kk), ID_Q2, (i < 2 || kk > 0) ? 1u : 0u);
        }
        tc_commit(bar(Q_DONE));
      }
    }
    __syncwarp();
  } else {
    const int r = threadIdx.x & 127, cg = threadIdx.x >> 7;    // token row (= TMEM lane) and group of 16 features
    const int gr = threadIdx.x >> 2, gq = threadIdx.x & 3;     // the G pass: row and 16 of its columns
    const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
    const bool square = p.P == 2 && cg >= 2;                   // power of this thread's features (parts are 64 or 32 wide)
    split_matrix(p.S + (size_t)bh * 4096, sbase + L::S_OFF, threadIdx.x);
    if (threadIdx.x < 64) zvec[threadIdx.x] = p.z[(size_t)bh * 64 + threadIdx.x];
    float loss = 0.f, dz[16], acc[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) { dz[i] = 0.f; acc[i] = 0.f; }
    // lanes 0-63: features of dS against the columns of G; lanes 64-127: features of dW_q against the columns of q
    const uint32_t t_own = tAcc + lane_off + (r < 64 ? 0 : 64) + cg * 16;
    bool ok = true;
    // the row's statistics of the forward pass (c_i, the two parts of the denominator), fetched one tile ahead
    auto row_stats = [&](int t, float (&a)[3]) {
      const int n = tok_begin + t * 128 + r;
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
      if (ok) ok = mbar_wait_warp(bar(Q_FULL + (t & 1)), (t >> 1) & 1, wc);
      if (ok) {
        // G = sign(y_hat - y) over y, t = -(G . y_hat) and the loss on the way.  Four lanes share a row of 128 bytes.
        // (rows past the end of the sequence arrive as zeros: no difference, no sign, nothing added)
        uint8_t* sY = smem + stage(t);
        const uint8_t* sH = sY + 2 * BOX;
        float sdot = 0.f;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const uint32_t off = swz128_chunk_offset(gr, 2 * gq + c);
          const uint4 yv = *reinterpret_cast<const uint4*>(sY + off), hv = *reinterpret_cast<const uint4*>(sH + off);
          const uint32_t yw[4] = {yv.x, yv.y, yv.z, yv.w}, hw[4] = {hv.x, hv.y, hv.z, hv.w};
          uint32_t gw[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float h0 = __uint_as_float(hw[i] << 16), h1 = __uint_as_float(hw[i] & 0xffff0000u);
            const float d0 = h0 - __uint_as_float(yw[i] << 16), d1 = h1 - __uint_as_float(yw[i] & 0xffff0000u);
            const float G0 = d0 > 0.f ? 1.f : (d0 < 0.f ? -1.f : 0.f), G1 = d1 > 0.f ? 1.f : (d1 < 0.f ? -1.f : 0.f);
            loss += fabsf(d0) + fabsf(d1);
            sdot = fmaf(G0, h0, fmaf(G1, h1, sdot));
            gw[i] = __byte_perm(__float_as_uint(G0), __float_as_uint(G1), 0x7632);
          }
          *reinterpret_cast<uint4*>(sY + off) = make_uint4(gw[0], gw[1], gw[2], gw[3]);
        }
        sdot += __shfl_xor_sync(0xffffffffu, sdot, 1);
        sdot += __shfl_xor_sync(0xffffffffu, sdot, 2);
        if (gq == 0) tvec[(t & 1) * 128 + gr] = -sdot;
      }
      fence_proxy_async();
      mbar_arrive(bar(Q_GRDY));
      if (ok) ok = mbar_wait_warp(bar(Q_AU), t & 1, wc);
      // (U is complete only after every thread has arrived on the G barrier: t of every row is there, and z)
      if (ok) {
        tc_fence_after();
        uint32_t xa[16], xu[16];
        tmem_ld16(tA + lane_off + cg * 16, xa);
        tmem_ld16(tU + lane_off + cg * 16, xu);
        const float ti = tvec[(t & 1) * 128 + r];
        float w = 0.f;
        if (tok_begin + t * 128 + r < tok_end) {
          const float lam = (p.stab_mode == AS_STAB_EXACT && p.n_s > 0) ? __expf(-st_c[0]) : 1.f;
          w = lam / (st_c[1] + lam * st_c[2]);
        }
        tmem_ld16_wait(xa);
        tmem_ld16_wait(xu);
        tc_fence_before();
        float ph[16], da[16];
        if (square) bsq_features<2>(xa, xu, zvec + cg * 16, ti, w, ph, da, dz);
        else bsq_features<1>(xa, xu, zvec + cg * 16, ti, w, ph, da, dz);
        if (t > 0) ok = mbar_wait_warp(bar(Q_DONE), (t - 1) & 1, wc);        // the products of the tile before have read X
        if (ok) {
          if (t > 0) add_acc16(t_own, acc);
          store_split16(sbase + L::X_OFF, 2 * BOX, r, cg * 16, ph);
          store_split16(sbase + L::X_OFF + BOX, 2 * BOX, r, cg * 16, da);
        }
      }
      fence_proxy_async();
      mbar_arrive(bar(Q_XRDY));
    }
    // ---- the chunk's partial results
    const uint32_t late = status_now(p.status);      // behind the wait, ahead of the first write: not 0, and nothing is written
    if (ok && nt > 0) ok = mbar_wait_warp(bar(Q_DONE), (nt - 1) & 1, wc);
    const size_t slot = (size_t)bh * p.chunks + chunk;
    if (ok && nt > 0) {
      add_acc16(t_own, acc);
      float* dst = (r < 64 ? p.part_dS : p.part_dW) + (slot * 64 + (r & 63)) * 64 + cg * 16;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (late == 0u) reinterpret_cast<float4*>(dst)[i] = make_float4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]);
    }
    // dz: over the warp's 32 rows by shuffles, then the four row blocks in order; the loss: the warps' sums in order
    float* red = reinterpret_cast<float*>(smem + L::X_OFF);       // idle: the last product has read it
#pragma unroll
    for (int i = 0; i < 16; ++i) {
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) dz[i] += __shfl_xor_sync(0xffffffffu, dz[i], off);
      if (lane == i) red[(warp & 3) * 64 + cg * 16 + i] = dz[i];
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, off);
    if (lane == 0) red[256 + warp] = loss;
    named_barrier_sync(1, BS_COMPUTE);
    if (threadIdx.x < 64 && late == 0u)
      p.part_dz[slot * 64 + threadIdx.x] = (red[threadIdx.x] + red[64 + threadIdx.x]) + (red[128 + threadIdx.x] + red[192 + threadIdx.x]);
    if (threadIdx.x == 64 && late == 0u) {
      float l = 0.f;
      for (int i = 0; i < 16; ++i) l += red[256 + i];
      p.part_loss[slot] = l;
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 16) {
    tc_fence_after();
    tmem_dealloc(tmem, 256);
  }
}

// ---------------------------------------------------------------------------------------------- key side
struct BskLayout {
  static constexpr int STAGES = 3;
  static constexpr int W_OFF = 0;                           // W_k [64][64]
  static constexpr int S_OFF = MAT;                         // dS, three pieces
  static constexpr int IN_OFF = 4 * MAT;                    // stages of [k | v]
  static constexpr int STAGE = 2 * BOX;
  static constexpr int X_OFF = IN_OFF + STAGES * STAGE;     // two sets (tile parity) of the three pieces of dL/da_k
  static constexpr int BAR_OFF = X_OFF + 6 * BOX;
  static constexpr int Z_OFF = BAR_OFF + 128;               // 64 floats: dz
  static constexpr int TOTAL = Z_OFF + 256 + 1024;
};
// Who has passed what before a barrier can complete again (a wait that looks after two more phases would not see its own).  The
// compute threads can be a tile ahead of the issuing lane: for tile t + 1 they need AT(t + 1) and DONE(t - 1), both from before
// the lane looks at XRDY(t).  So XRDY is one barrier per tile parity: arriving for tile t + 2 needs AT(t + 2), which the lane
// issues only after it has passed XRDY(t).  AT(t + 2) and DONE(t + 2) come after XRDY(t + 1) and XRDY(t + 2), where every thread
// has passed AT(t) and DONE(t); FULL(t + 3) is requested after DONE(t), whose products the lane issued after FULL(t).
enum { K_WFULL = 0, K_SRDY = 1, K_FULL = 2, K_AT = 5, K_XRDY = 7, K_DONE = 9, K_BARS = 11 };

__global__ void __launch_bounds__(BS_THREADS, 1)
bsk_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmW,
           const __grid_constant__ BwParams p) {
  using L = BskLayout;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t sbase = smem_u32(smem);
  auto bar = [&](int i) { return sbase + L::BAR_OFF + 8 * i; };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::BAR_OFF + 8 * K_BARS);
  volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem + L::BAR_OFF + 8 * K_BARS + 4);
  float* zvec = reinterpret_cast<float*>(smem + L::Z_OFF);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int bh = blockIdx.y, chunk = blockIdx.x, h = bh % p.H;
  const int tok_begin = chunk * p.chunk_tokens;
  const int tok_end = min(p.N, tok_begin + p.chunk_tokens);
  const int nt = (tok_end - tok_begin + 127) / 128;

  if (threadIdx.x == 0) {
    *abort_flag = 0u;
    mbar_init(bar(K_WFULL), 1); mbar_init(bar(K_SRDY), BS_COMPUTE);
    for (int s = 0; s < L::STAGES; ++s) mbar_init(bar(K_FULL + s), 1);
    for (int b = 0; b < 2; ++b) { mbar_init(bar(K_AT + b), 1); mbar_init(bar(K_XRDY + b), BS_COMPUTE); mbar_init(bar(K_DONE + b), 1); }
    fence_barrier_init();
    fence_proxy_async();
  }
  __shared__ uint32_t s_skip;
  if (threadIdx.x == 32) s_skip = status_now(p.status);
  if (warp == 16) { tmem_alloc(smem_u32(tmem_slot), 512); tmem_relinquish(); griddep_launch(); }
  if (threadIdx.x == 15 * 32) { tma_prefetch_desc(&tmK); tma_prefetch_desc(&tmV); tma_prefetch_desc(&tmW); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  griddep_wait();                                    // the set-up above ran beside the kernel before this one
  // an earlier launch timed out: do nothing (decided once per CTA)
  if (s_skip != 0u) {
    if (warp == 16) tmem_dealloc(*tmem_slot, 512);
    return;
  }
  const uint32_t tmem = *tmem_slot;
  // per tile parity: A, T and two accumulators: lanes 0-63 of the first hold the product of the hi pieces, lanes 64-127 of
  // the mid pieces; lanes 64-127 of the second of the lo pieces (its lower half repeats the mid pieces and is not read)
  auto tA = [&](int t) { return tmem + (t & 1) * 128u; };
  auto tT = [&](int t) { return tmem + (t & 1) * 128u + 64u; };
  auto tHM = [&](int t) { return tmem + 256u + (t & 1) * 128u; };
  auto tML = [&](int t) { return tmem + 320u + (t & 1) * 128u; };
  const WaitCtx wc{p.status, abort_flag};

  if (warp == 16) {
    if (lane == 0) {
      auto sK = [&](int t) { return sbase + L::IN_OFF + (t % L::STAGES) * L::STAGE; };
      auto request = [&](int t) {
        const uint32_t fb = bar(K_FULL + t % L::STAGES);
        mbar_expect_tx(fb, 2 * BOX);
        tma_load_3d(sK(t), &tmK, fb, 0, tok_begin + t * 128, bh);
        tma_load_3d(sK(t) + BOX, &tmV, fb, 0, tok_begin + t * 128, bh);
      };
      auto first_products = [&](int t) -> bool {             // A = K W_k^T and T = V dS^T of tile t
        if (!mbar_wait(bar(K_FULL + t % L::STAGES), (t / L::STAGES) & 1, wc)) return false;
        tc_fence_after();
        issue_kmajor<64>(tA(t), kmajor_desc(sK(t)), kmajor_desc(sbase + L::W_OFF), ID_TOK, false);
        issue_pieces(tT(t), sK(t) + BOX, sbase + L::S_OFF);
        tc_commit(bar(K_AT + (t & 1)));
        return true;
      };
      mbar_expect_tx(bar(K_WFULL), MAT);
      tma_load_3d(sbase + L::W_OFF, &tmW, bar(K_WFULL), 0, 0, h);
      for (int t = 0; t < L::STAGES && t < nt; ++t) request(t);
      bool ok = nt > 0 && mbar_wait(bar(K_WFULL), 0, wc) && mbar_wait(bar(K_SRDY), 0, wc) && first_products(0);
      for (int t = 0; t < nt && ok; ++t) {
        // (A and T of tile t - 1, whose columns tile t + 1 takes, were read before the threads arrived on the X barrier)
        if (t + 1 < nt && !first_products(t + 1)) break;
        if (t > 0 && t + 2 < nt) {
          if (!mbar_wait(bar(K_DONE + ((t - 1) & 1)), ((t - 1) >> 1) & 1, wc)) break;      // the stage of tile t - 1 is free
          request(t + 2);
        }
        if (!mbar_wait(bar(K_XRDY + (t & 1)), (t >> 1) & 1, wc)) break;
        tc_fence_after();
        const uint32_t x0 = sbase + L::X_OFF + (t & 1) * 3 * BOX;
        const uint64_t hm = mnmajor_desc(x0), ml = mnmajor_desc(x0 + BOX), bK = mnmajor_desc(sK(t));
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) mma_ss(tHM(t), hm + kstep_mnmajor(kk), bK + kstep_mnmajor(kk), ID_K2, kk > 0 ? 1u : 0u);
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) mma_ss(tML(t), ml + kstep_mnmajor(kk), bK + kstep_mnmajor(kk), ID_K2, kk > 0 ? 1u : 0u);
        tc_commit(bar(K_DONE + (t & 1)));
      }
    }
    __syncwarp();
  } else {
    const int r = threadIdx.x & 127, cg = threadIdx.x >> 7;
    const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
    const bool square = p.P == 2 && cg >= 2;
    split_matrix(p.dS + (size_t)bh * 4096, sbase + L::S_OFF, threadIdx.x);
    if (threadIdx.x < 64) zvec[threadIdx.x] = p.dz[(size_t)bh * 64 + threadIdx.x];
    fence_proxy_async();
    mbar_arrive(bar(K_SRDY));
    named_barrier_sync(1, BS_COMPUTE);
    bool ok = true;
    auto is_linear = [&](int t) { const int n = tok_begin + t * 128 + r; return t < nt && n < tok_end && p.sm_rank[n] < 0; };
    bool lin_next = is_linear(0);                    // fetched one tile ahead
    float acc[16], accl[16];                         // lanes 0-63: hi; lanes 64-127: mid and lo
#pragma unroll
    for (int i = 0; i < 16; ++i) { acc[i] = 0.f; accl[i] = 0.f; }
    auto add_tile = [&](int t) {
      add_acc16(tHM(t) + lane_off + cg * 16, acc);
      if (r >= 64) add_acc16(tML(t) + lane_off + cg * 16, accl);
    };
    for (int t = 0; t < nt; ++t) {
      const bool lin = lin_next;
      lin_next = is_linear(t + 1);
      if (ok) ok = mbar_wait_warp(bar(K_AT + (t & 1)), (t >> 1) & 1, wc);
      if (ok) {
        tc_fence_after();
        uint32_t xa[16], xt[16];
        tmem_ld16(tA(t) + lane_off + cg * 16, xa);
        tmem_ld16(tT(t) + lane_off + cg * 16, xt);
        tmem_ld16_wait(xa);
        tmem_ld16_wait(xt);
        tc_fence_before();
        float da[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const float a = __uint_as_float(xa[i]);
          const float slope = square ? 2.f * fmaxf(a, 0.f) : (a > 0.f ? 1.f : 0.f);
          da[i] = lin ? (__uint_as_float(xt[i]) + zvec[cg * 16 + i]) * slope : 0.f;
        }
        // the products of the tile before the last have read this set and left their sums
        if (t > 1) ok = mbar_wait_warp(bar(K_DONE + (t & 1)), ((t - 2) >> 1) & 1, wc);
        if (ok && t > 1) add_tile(t - 2);
        if (ok) store_split16(sbase + L::X_OFF + (t & 1) * 3 * BOX, BOX, r, cg * 16, da);
      }
      fence_proxy_async();
      mbar_arrive(bar(K_XRDY + (t & 1)));
    }
    const uint32_t late = status_now(p.status);      // behind the wait, ahead of the first write: not 0, and nothing is written
    for (int t = nt > 1 ? nt - 2 : 0; t < nt; ++t) {
      if (ok) ok = mbar_wait_warp(bar(K_DONE + (t & 1)), (t >> 1) & 1, wc);
      if (ok) add_tile(t);
    }
    // hi + mid + lo: the threads of lanes 64-127 hand the mid and lo sums over through shared memory
    float* red = reinterpret_cast<float*>(smem + L::X_OFF);       // idle: the last product has read it
    if (r >= 64) {
#pragma unroll
      for (int i = 0; i < 16; ++i) red[(cg * 16 + i) * 64 + (r - 64)] = acc[i] + accl[i];
    }
    named_barrier_sync(1, BS_COMPUTE);
    if (ok && late == 0u && nt > 0 && r < 64) {
      float* dst = p.part_dW + ((((size_t)bh * p.chunks + chunk) * 64) + r) * 64 + cg * 16;
#pragma unroll
      for (int i = 0; i < 16; ++i) dst[i] = acc[i] + red[(cg * 16 + i) * 64 + r];
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

cudaError_t as_bw_tensor_d64_init() {
  cudaError_t e;
  if ((e = opt_in_smem(bsq_kernel, BsqLayout::TOTAL)) != cudaSuccess) return e;
  return opt_in_smem(bsk_kernel, BskLayout::TOTAL);
}

cudaError_t as_bw_tensor_d64_query(const BwParams& p, cudaStream_t st) {
  const int BH = p.B * p.H;
  CUtensorMap tmQ, tmY, tmH, tmW;
  if (!make_map(&tmQ, p.q, 64, p.N, BH, 128) || !make_map(&tmY, p.y, 64, p.N, BH, 128) ||
      !make_map(&tmH, p.yhat, 64, p.N, BH, 128) || !make_map(&tmW, p.wq, 64, 64, p.H, 64))
    return cudaErrorInvalidValue;
  return as_launch_dependent(bsq_kernel, dim3(p.chunks, BH), dim3(BS_THREADS), BsqLayout::TOTAL, st, tmQ, tmY, tmH, tmW, p);
}

cudaError_t as_bw_tensor_d64_key(const BwParams& p, cudaStream_t st) {
  const int BH = p.B * p.H;
  CUtensorMap tmK, tmV, tmW;
  if (!make_map(&tmK, p.k, 64, p.N, BH, 128) || !make_map(&tmV, p.v, 64, p.N, BH, 128) || !make_map(&tmW, p.wk, 64, 64, p.H, 64))
    return cudaErrorInvalidValue;
  return as_launch_dependent(bsk_kernel, dim3(p.chunks, BH), dim3(BS_THREADS), BskLayout::TOTAL, st, tmK, tmV, tmW, p);
}
