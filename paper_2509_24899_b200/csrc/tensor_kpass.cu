// K pass of the hybrid attention forward on the tensor cores of sm_100a (phi_k projection, linear
// state, softmax gather) and the first layer of a two-layer feature map for the keys.
//
//   One CTA = (chunk of 128-token tiles, batch*head, chunk of 128 features).  Per token tile:
//     Phi^T = W X^T       tcgen05.mma, smem x smem -> TMEM; TMEM lane = feature, column = token.
//                         One layer: W = W_k rows of the feature chunk, X = the K tile.  Two layers:
//                         W = W_k2[feature chunk, :], X = relu(K W_k1^T + b1) as left by phi1_kernel,
//                         one MMA chain per 128-wide slice of the hidden width.
//     phi   = poly(relu(Phi + b)), zero for softmax tokens and past the sequence end, rounded to bf16
//             into spare TMEM columns (eight feature warps, two per lane quadrant)
//     S    += phi^T-tile V   tcgen05.mma, TMEM x smem -> TMEM accumulator that lives across the chunk
//     z    += the bf16 features, summed per feature in registers
//     the tile's softmax-token rows are copied to the compact K_S / V_S (feature chunk 0 only).
//   All tiles travel through one ring of shared-memory slots filled by TMA; every mbarrier wait is bounded.
#include "tensor_common.cuh"

namespace {

using namespace as_tc;

struct KParams {
  int N, n_s, n_chunks, chunk_tiles, P, F, H;
  const int32_t* sm_rank;              // [N (+ padding)]: position in T_S, or -1 for a linear token
  __nv_bfloat16 *ks_w, *vs_w;          // compact softmax K / V (nullptr when nothing is gathered)
  const __nv_bfloat16* bias;           // last-layer bias [H][F], or nullptr
  float *part_s, *part_z;              // the chunk's state
  float *S, *z;                        // [B*H][F][D], [B*H][F]: the chunks' partials added up ...
  __nv_bfloat16* Sb;                   // ... and S once more rounded to bf16 (the query stage's MMA operand)
  uint32_t* counters;                  // [B*H][feature chunks][2]: CTAs that have stored (and, times 2^16, that have given up) / that have left; zero
                                       // between launches
  uint32_t* status;
};

constexpr int K_THREADS = 416;           // warps 0-7: feature warps; 8: TMA; 9: issues Phi^T; 10: issues S; 11-12: gather
constexpr int K_FEATURE_THREADS = 256;
constexpr long long kSumPatience = 400ll * 1000ll;   // clocks, 0.2 ms: the chunks of a head differ by a few us where all CTAs run

// LAYERS == 1: ring items per token tile are (K, V), one resident weight tile.
// LAYERS == 2: ring items are (h1 slice 0 .. NH-1, V), NH resident weight tiles W_2[feature chunk, hidden slice].
// Every tile is [128 rows x D columns] bf16 (a hidden slice is D wide).
template <int D, int LAYERS, int NH>
struct KLayout {
  static constexpr int NX = LAYERS == 1 ? 1 : NH;               // tiles that feed the feature product
  static constexpr int IPT = NX + 1;                            // ring items per token tile
  static constexpr int TILE = 128 * D * 2;
  static constexpr int SLOTS = D == 128 ? 7 - NH : 8;
  static constexpr int W_OFF = 0;
  static constexpr int RING_OFF = NH * TILE;
  static constexpr int BAR_OFF = RING_OFF + SLOTS * TILE;
  static constexpr int N_BARS = 1 + 3 * SLOTS + 7;
  static constexpr int PAIR_OFF = (BAR_OFF + 8 * N_BARS + 8 + 15) / 16 * 16;   // (behind two words) 32 words a feature warp: per token pair, which halves are linear tokens
  static constexpr int Z_OFF = PAIR_OFF + 8 * 32 * 4;           // 128 floats: z of the upper column half
  static constexpr int TOTAL = Z_OFF + 128 * 4 + 1024;          // + slack for the 1024-byte alignment
  // the chunk's partial S leaves through the ring (idle by then): 128 rows of D floats, each row padded by 16
  // bytes so that the 32 lanes of a warp, one row each, write to different banks
  static constexpr int OUT_PITCH = D * 4 + 16;
  static_assert(128 * OUT_PITCH <= SLOTS * TILE, "staging area");
  static_assert(RING_OFF % 1024 == 0 && PAIR_OFF % 16 == 0 && Z_OFF % 16 == 0 && OUT_PITCH % 16 == 0, "tiles, and what is read 16 bytes at a time");
  static_assert(TOTAL <= 232448, "shared memory of a CTA");
};

// Features of 32 token columns of one TMEM lane: bias, ReLU, power, linear-token mask, bf16.
template <int POW>
AS_DEV void k_features(const uint32_t (&x)[32], const uint4* mask4, float bias, uint32_t (&w)[16], float& z0, float& z1) {
#pragma unroll
  for (int g4 = 0; g4 < 4; ++g4) {
    const uint4 m = mask4[g4];
    const uint32_t mm[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int i = 4 * g4 + e;
      float a0 = fmaxf(__uint_as_float(x[2 * i]) + bias, 0.f), a1 = fmaxf(__uint_as_float(x[2 * i + 1]) + bias, 0.f);
      if (POW == 2) { a0 *= a0; a1 *= a1; }
      if (POW == 3) { a0 = a0 * a0 * a0; a1 = a1 * a1 * a1; }
      if (POW == 4) { a0 *= a0; a1 *= a1; a0 *= a0; a1 *= a1; }
      w[i] = pack_bf16(a0, a1) & mm[e];
      // z sums the features as the MMA sees them: the bf16 values
      add_bf16x2(z0, z1, w[i]);
    }
  }
}

template <int D, int LAYERS, int NH>
__global__ void __launch_bounds__(K_THREADS, 1)
kpass_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
             const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmH, const KParams p) {
  using L = KLayout<D, LAYERS, NH>;
  constexpr int SLOTS = L::SLOTS, IPT = L::IPT, NX = L::NX;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t sbase = smem_u32(smem);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::BAR_OFF);
  // Whether a ring slot is full is told on a barrier of its item's kind, XFULL (K, hidden slices) or VFULL: whoever waits looks at every phase of a
  // barrier, in order.  D1: Phi^T has landed; PK: it has been read and the features are packed; SD: the product that reads these has completed.
  enum { B_W = 0, B_XFULL = 1, B_VFULL = B_XFULL + SLOTS, B_EMPTY = B_VFULL + SLOTS, B_D1 = B_EMPTY + SLOTS, B_PK = B_D1 + 2, B_SD = B_PK + 2,
         B_DONE = B_SD + 2, B_COUNT = B_DONE + 1 };
  static_assert(B_COUNT == L::N_BARS, "barrier count");
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::BAR_OFF + 8 * B_COUNT);
  volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem + L::BAR_OFF + 8 * B_COUNT + 4);
  uint32_t* sPair = reinterpret_cast<uint32_t*>(smem + L::PAIR_OFF);
  float* sZ = reinterpret_cast<float*>(smem + L::Z_OFF);
  auto bar = [&](int i) { return smem_u32(bars + i); };

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int bh = blockIdx.y, h = bh % p.H, chunk = blockIdx.x, fc = blockIdx.z;
  const int tiles_total = (p.N + 127) / 128;
  const int t_begin = chunk * p.chunk_tiles;
  const int nt = min(p.chunk_tiles, tiles_total - t_begin);
  const WaitCtx wc{p.status, abort_flag};
  const bool gathers = (p.ks_w != nullptr) && fc == 0;       // this CTA copies the softmax rows out

  auto sW = [&](int j) { return sbase + L::W_OFF + j * L::TILE; };
  auto sSlot = [&](int it) { return sbase + L::RING_OFF + (it % SLOTS) * L::TILE; };
  // one ring item: tile t's K (one layer) or hidden slice i (two layers), or its V tile
  auto load_item = [&](int it) {
    const int st = it % SLOTS, t = it / IPT, i = it % IPT, row = (t_begin + t) * 128;
    const uint32_t full = bar((i == NX ? B_VFULL : B_XFULL) + st);
    mbar_expect_tx(full, L::TILE);
    if (i == NX) load_tile<D>(sSlot(it), &tmV, full, row, bh);
    else if (LAYERS == 1) load_tile<D>(sSlot(it), &tmK, full, row, bh);
    else load_boxes(sSlot(it), &tmH, full, i * D, row, bh, D / 64);
  };
  // `looks`: bit s is the parity of the next phase of the barrier of slot s that the warp has not looked at
  auto wait_full = [&](int first_bar, int it, uint32_t& looks) -> bool {
    const int st = it % SLOTS;
    const uint32_t parity = (looks >> st) & 1u;
    looks ^= 1u << st;
    return mbar_wait_warp(bar(first_bar + st), parity, wc);
  };
  constexpr int FIRST = IPT;                                 // items requested at once, the first tile's

  // ---- Set-up that runs beside the kernel before this one.  The table of softmax ranks is the handle's and does not change; and the status word is asked
  // for here because small loads that come behind the first tiles' wait as long as these do (4 us at N = 7800, 12 heads).
  __shared__ uint32_t s_skip;
  if (threadIdx.x == 32) s_skip = status_now(p.status);
  if (warp == 9) {
    // the query stage's CTAs may then set up as these ones end
    tmem_alloc(smem_u32(tmem_slot), 512); tmem_relinquish(); griddep_launch();
  } else if (threadIdx.x == 0) {
    *abort_flag = 0u;
    mbar_init(bar(B_W), 1);
    // a slot is free again when the MMA that read it has completed and, where rows are gathered, when both gather warps are through with it
    for (int s = 0; s < SLOTS; ++s) { mbar_init(bar(B_XFULL + s), 1); mbar_init(bar(B_VFULL + s), 1); mbar_init(bar(B_EMPTY + s), gathers ? 3 : 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(bar(B_D1 + b), 1); mbar_init(bar(B_PK + b), K_FEATURE_THREADS); mbar_init(bar(B_SD + b), 1); }
    mbar_init(bar(B_DONE), 1);
    fence_barrier_init();
    fence_proxy_async();
  }
  // Feature warps: the ranks of a pair of their 64 tokens of a tile, the first tile's.  Gather warps: those of two of their 64 rows.
  const int my_n0 = t_begin * 128 + (warp < 8 ? (warp >> 2) * 64 + 2 * lane : (warp & 1 ? 0 : 64) + lane);
  auto pair_ranks = [&](int t) -> int2 {                       // (the table is N + 8 long)
    const int n0 = my_n0 + t * 128;
    return t < nt && n0 < p.N ? *reinterpret_cast<const int2*>(p.sm_rank + n0) : make_int2(0, 0);
  };
  auto row_ranks = [&](int t) -> int2 {
    const int n0 = my_n0 + t * 128;
    return make_int2(t < nt && n0 < p.N ? p.sm_rank[n0] : -1, t < nt && n0 + 32 < p.N ? p.sm_rank[n0 + 32] : -1);
  };
  // Four tiles ahead: under the load of the tiles' copies these take longer than a tile.  (A register that waits for its load cannot be moved to another
  // without waiting, hence a branch by t % 4 where they are used.)
  int2 rk0 = make_int2(-1, -1), rk1 = rk0, rk2 = rk0, rk3 = rk0;
  if (warp < 8) { rk0 = pair_ranks(0); rk1 = pair_ranks(1); rk2 = pair_ranks(2); rk3 = pair_ranks(3); }
  else if (warp >= 11 && gathers) { rk0 = row_ranks(0); rk1 = row_ranks(1); rk2 = row_ranks(2); rk3 = row_ranks(3); }
  auto by_turns = [&](int t, auto use) {
    switch (t & 3) {
      case 0: use(rk0); break;
      case 1: use(rk1); break;
      case 2: use(rk2); break;
      default: use(rk3); break;
    }
  };
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (s_skip != 0u) {                                        // an earlier launch timed out: nothing is requested
    griddep_wait();
    if (warp == 9) tmem_dealloc(*tmem_slot, 512);
    return;
  }
  __shared__ volatile uint32_t s_late;                       // the status word behind the wait: not 0, and nothing is written
  if (warp >= 8) griddep_wait();                             // (the feature warps: see their loop)
  const uint32_t tmem = *tmem_slot;
  const uint32_t tD1[2] = {tmem + 0u, tmem + 128u};          // Phi^T of a tile, fp32
  const uint32_t tAcc = tmem + 256u;                         // S of this feature chunk
  const uint32_t tPA[2] = {tmem + 384u, tmem + 448u};        // the tile's features as packed bf16 (A operand)

  if (warp == 8) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      mbar_expect_tx(bar(B_W), NH * L::TILE);
      // rows past F are out of bounds and arrive as zeros
      for (int j = 0; j < NH; ++j) load_boxes(sW(j), &tmW, bar(B_W), j * D, fc * 128, h, D / 64);
      for (int it = 0; it < FIRST; ++it) load_item(it);
    }
    __syncwarp();
    for (int it = FIRST; it < nt * IPT; ++it) {
      // (the first tile has the memory system to itself: with the whole ring asked for at once its latency is that of the ring)
      if (it == FIRST && !mbar_wait_warp(bar(B_XFULL), 0, wc)) break;
      const int st = it % SLOTS;
      if (!mbar_wait_warp(bar(B_EMPTY + st), ((it / SLOTS) & 1) ^ 1, wc)) break;
      if (lane == 0) load_item(it);
      __syncwarp();
    }
  } else if (warp == 9) {
    // ------------------------------------------------------------ issues Phi^T(t) as soon as the tile's X items have landed and the features of tile
    // t - 2, which lay in the same columns, have been read.  Two issuing warps, a lane of each elected from converged code: one thread that took whichever of
    // the two products was ready, by turns of non-blocking looks, needed 1700 - 2000 clk a tile,
    // more than the feature warps.
    constexpr uint32_t ID_PHI = make_idesc(128, 128, 0, 0);    // Phi^T = W X^T : M = features, N = 128 tokens
    uint32_t looks = 0u;
    bool ok = mbar_wait_warp(bar(B_W), 0, wc);
    for (int t = 0; ok && t < nt; ++t) {
      const int b = t & 1;
      if (t >= 2) ok = mbar_wait_warp(bar(B_PK + b), ((t - 2) >> 1) & 1, wc);
#pragma unroll
      for (int j = 0; j < NX; ++j) {
        const int it = t * IPT + j;
        ok = ok && wait_full(B_XFULL, it, looks);
        if (!ok) break;
        tc_fence_after();
        const uint64_t w0 = kmajor_desc(sW(j)), x0 = kmajor_desc(sSlot(it));
        if (elect_one()) {
          issue_kmajor<D>(tD1[b], w0, x0, ID_PHI, j > 0);
          tc_commit(bar(B_EMPTY + it % SLOTS));
          if (j == NX - 1) tc_commit(bar(B_D1 + b));
        }
        __syncwarp();
      }
    }
  } else if (warp == 10) {
    // ------------------------------------------------------------ issues S += phi^T V (t) as soon as the features are packed
    constexpr uint32_t ID_ACC = make_idesc(128, D, 0, 1);      // S += phi^T V  : V is MN-major
    uint32_t looks = 0u;
    bool ok = true;
    for (int t = 0; ok && t < nt; ++t) {
      const int b = t & 1, it = t * IPT + NX;
      ok = wait_full(B_VFULL, it, looks) && mbar_wait_warp(bar(B_PK + b), (t >> 1) & 1, wc);
      if (!ok) break;
      tc_fence_after();
      const uint64_t v0 = mnmajor_desc(sSlot(it));
      if (elect_one()) {
        issue_tmemA_mnB(tAcc, tPA[b], v0, ID_ACC, t > 0);
        tc_commit(bar(B_EMPTY + it % SLOTS));
        tc_commit(bar(B_SD + b));
        if (t == nt - 1) tc_commit(bar(B_DONE));
      }
      __syncwarp();
    }
  } else if (warp >= 11) {
    // ------------------------------------------------------------ gather of softmax-token rows
    const uint32_t late = gathers || warp == 11 ? status_now(p.status) : 0u;
    if (gathers) {
      const int gw = warp & 1 ? 0 : 1;
      // rows handled by this warp: gw*64 .. gw*64+63; two ranks per lane
      uint32_t looks_x = 0u, looks_v = 0u;
      for (int t = 0; t < nt; ++t) {
        int rk[2];
        by_turns(t, [&](int2& r) { rk[0] = r.x; rk[1] = r.y; r = row_ranks(t + 4); });
        bool ok = true;
        for (int i = 0; i < IPT; ++i) {
          const int it = t * IPT + i;
          ok = ok && (i == NX ? wait_full(B_VFULL, it, looks_v) : wait_full(B_XFULL, it, looks_x));
          if (LAYERS == 2 && i < NX && ok && lane == 0) mbar_arrive(bar(B_EMPTY + it % SLOTS));   // a hidden slice: not read here
        }
        if (!ok) break;
        const uint8_t* kt = LAYERS == 1 ? smem + L::RING_OFF + ((t * IPT) % SLOTS) * L::TILE : nullptr;
        const uint8_t* vt = smem + L::RING_OFF + ((t * IPT + NX) % SLOTS) * L::TILE;
        // CH 16-byte pieces a row; a row is LPR lanes wide: its K and its V pieces (two layers: V's alone, phi1_kernel has copied K).
        // AHEAD loads per lane before the first of their stores: one row after the other, each a chain of bit search, shuffle, load and store, the two
        // warps took 3000 - 4000 clk for the 32 rows of a tile at rate 1/4, and held its ring slots meanwhile (N = 8505, 32 heads, d = 64: this
        // kernel 44.7 us against 33.9; rate 1/2 67.6 against 44.8; d = 128, N = 32760, 12 heads, rate 1/2: 73.7 against 59.3).
        constexpr int CH = D / 8, LPR = LAYERS == 1 ? 2 * CH : CH, RPI = 32 / LPR, AHEAD = 4;
        const int c = lane % CH;
        const bool is_v = LAYERS == 2 || lane % LPR >= CH;
        const uint8_t* from = (is_v ? vt : kt) + (c / 8) * BOX_BYTES;
        __nv_bfloat16* to = (is_v ? p.vs_w : p.ks_w) + (size_t)bh * p.n_s * D + c * 8;
        for (int e = 0; e < 2; ++e) {
          const int mine = late != 0u ? -1 : e == 0 ? rk[0] : rk[1];
          uint32_t bits = __ballot_sync(0xffffffffu, mine >= 0);
          while (bits) {
            int src[AHEAD], rank[AHEAD];
            uint4 val[AHEAD];
#pragma unroll
            for (int a = 0; a < AHEAD; ++a) {
              src[a] = -1;
#pragma unroll
              for (int i = 0; i < RPI; ++i) {
                if (lane / LPR == i && bits) src[a] = __ffs(bits) - 1;
                bits &= bits - 1;                          // (0 stays 0)
              }
              rank[a] = __shfl_sync(0xffffffffu, mine, src[a] < 0 ? 0 : src[a]);
              if (src[a] >= 0) val[a] = *reinterpret_cast<const uint4*>(from + swz128_chunk_offset(gw * 64 + e * 32 + src[a], c % 8));
            }
#pragma unroll
            for (int a = 0; a < AHEAD; ++a)
              if (src[a] >= 0) *reinterpret_cast<uint4*>(to + (size_t)rank[a] * D) = val[a];
          }
        }
        __syncwarp();
        if (lane == 0)
          for (int i = LAYERS == 1 ? 0 : NX; i < IPT; ++i) mbar_arrive(bar(B_EMPTY + (t * IPT + i) % SLOTS));
      }
    }
    if (threadIdx.x == 11 * 32) s_late = late;
    named_barrier_arrive(2, K_FEATURE_THREADS + 64);           // the feature warps may reuse the ring for the partial S
  } else {
    // ------------------------------------------------------------ feature warps: lane of TMEM = feature
    // warp w works on TMEM lanes 32 * (w % 4) .. + 31 and on token columns 64 * (w / 4) .. + 63
    const int quad = warp & 3, hf = warp >> 2;
    const int f_local = quad * 32 + lane, f = fc * 128 + f_local;
    const uint32_t lane_off = (uint32_t)(quad * 32) << 16;
    const int part = p.F / p.P;
    const int pw = min(f / part, p.P - 1) + 1;                 // power of this feature's part (the same in a whole warp
                                                               // whenever the part width is a multiple of 32)
    float bias = 0.f;                                          // the caller's: not before the wait for the kernel before this one
    float z0 = 0.f, z1 = 0.f;
    bool ok = true;
    uint32_t x[32];
    // Which tokens of a tile are linear tokens (inside the sequence, not softmax tokens), as one word per
    // token pair that masks the packed bf16 features.  A lane makes the word of one pair of its warp's 64 tokens; the ranks are asked for tiles ahead
    // and not looked at before (a comparison at the load made two warps wait for L2 in every tile and, with masks shared by
    // all eight, the others for these two: 700 - 1900 clk of the 3000 - 3800 that a tile took.  N = 7800, 12 heads, no softmax tokens:
    // 21.4 us before, 19.7 with this).
    uint32_t* pairs = sPair + warp * 32;
    // The loop's first turn is none of a tile: it brings the loop's instructions into the SM beside the kernel before this one.  They come through the
    // same memory system as the first tiles, and behind those they took 2 - 4 us to arrive (N = 7800, N = 32760, 12 heads: first features 1.9 and 4.2 us,
    // each later tile's 0.6).  What it computes from whatever lies in tensor memory goes into operand columns that the tiles overwrite.
    for (int t = -1; t < nt; ++t) {
      const int b = t & 1;
      __syncwarp();                                            // the tile before: every lane has read the words
      if (t >= 0) {
        by_turns(t, [&](int2& r) {
          pairs[lane] = (r.x < 0 ? 0x0000ffffu : 0u) | (r.y < 0 && my_n0 + t * 128 + 1 < p.N ? 0xffff0000u : 0u);
          r = pair_ranks(t + 4);
        });
        __syncwarp();
        ok = mbar_wait_warp(bar(B_D1 + b), (t >> 1) & 1, wc);
        if (!ok) break;
        tc_fence_after();
      }
      // (not unrolled: half the instructions to fetch in the first turn, N = 7800 77.9 -> 77.0 us a call)
#pragma unroll 1
      for (int c = 0; c < 2; ++c) {
        const int col = hf * 64 + c * 32;
        tmem_ld32(tD1[b] + lane_off + col, x);
        tmem_ld_wait(x);
        const uint4* mask4 = reinterpret_cast<const uint4*>(pairs + c * 16);
        uint32_t w[16];
        switch (pw) {
          case 1: k_features<1>(x, mask4, bias, w, z0, z1); break;
          case 2: k_features<2>(x, mask4, bias, w, z0, z1); break;
          case 3: k_features<3>(x, mask4, bias, w, z0, z1); break;
          default: k_features<4>(x, mask4, bias, w, z0, z1); break;
        }
        if (c == 0 && t >= 2) {                                // the product that read tile t - 2's features has completed
          ok = mbar_wait_warp(bar(B_SD + b), ((t - 2) >> 1) & 1, wc);
          if (!ok) break;
          tc_fence_after();
        }
        tmem_st16(tPA[b] + lane_off + col / 2, w);
      }
      if (!ok) break;
      tmem_st_wait();
      tc_fence_before();
      if (t < 0) {
        z0 = 0.f; z1 = 0.f;
        griddep_wait();
        if (p.bias != nullptr && f < p.F) bias = __bfloat162float(p.bias[(size_t)h * p.F + f]);
        continue;
      }
      mbar_arrive(bar(B_PK + b));
    }
    if (ok) ok = mbar_wait_warp(bar(B_DONE), 0, wc);
    // z of the two column halves is added through shared memory.  The partial S leaves through the ring: each
    // thread puts its half row there (rows padded so that a warp's lanes hit different banks), and the warps store whole rows, 512 bytes an instruction - a
    // row written straight from registers would cost one 32-byte sector per lane and instruction; row by row by the copy engine, the CTA waited 2400 clk
    // for the rows to be read.  The ring is idle once the last product has
    // completed and the gather warps (barrier 2) have read their last tile.  Every feature thread takes part in
    // the barriers whatever its waits returned.
    if (hf == 1) sZ[f_local] = z0 + z1;
    named_barrier_sync(2, K_FEATURE_THREADS + 64);
    uint8_t* stage = smem + L::RING_OFF;
    if (ok) {
      tc_fence_after();
      constexpr int HALF = D / 2;                              // accumulator columns per warp
#pragma unroll
      for (int c = 0; c < HALF / 32; ++c) {
        const int col = hf * HALF + c * 32;
        tmem_ld32(tAcc + lane_off + col, x);                   // warp-collective: also lanes beyond F take part
        tmem_ld_wait(x);
#pragma unroll
        for (int i = 0; i < 8; ++i)
          *reinterpret_cast<uint4*>(stage + f_local * L::OUT_PITCH + (col + 4 * i) * 4) = make_uint4(x[4 * i], x[4 * i + 1], x[4 * i + 2], x[4 * i + 3]);
      }
    }
    named_barrier_sync(1, K_FEATURE_THREADS);
    if (ok && s_late == 0u) {
      constexpr int LPR = D / 4, RPW = 32 / LPR;               // lanes a row, rows an instruction
      const size_t slot = ((size_t)bh * p.n_chunks + chunk) * p.F + fc * 128;
      const int nf = min(128, p.F - fc * 128);
      float4* out = reinterpret_cast<float4*>(p.part_s + slot * D);
#pragma unroll 4
      for (int r = warp * RPW + lane / LPR; r < nf; r += 8 * RPW)
        out[(size_t)r * LPR + lane % LPR] = *reinterpret_cast<const float4*>(stage + r * L::OUT_PITCH + lane % LPR * 16);
      if (hf == 0 && f_local < nf) p.part_z[slot + f_local] = (z0 + z1) + sZ[f_local];
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 9) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
  if (s_late != 0u) return;
  // ---- The chunks' partial states are added up here, in chunk order (fixed order, no float atomics): every CTA of
  // a (batch, head, feature chunk) takes a slice of the [F x (D + 1)] entries once all of them have stored theirs.
  // The CTAs of a launch are resident together where nothing else is on the GPU (one per SM at most).  A CTA that has waited for kSumPatience for
  // one that has not even started gives its slice up and leaves its SM: the last to store adds all slices up then (the same sums once more where
  // others do theirs).  So no CTA waits for good, and this is no cooperative launch, which the kernel before it in the stream would have to end for
  // first (N = 1024, 2 heads, d = 64: a call 18.3 -> 15.8 us).  The second counter tells the last CTA to leave that both
  // counters can go back to zero for the next launch.  This is a chain of L2 round trips: the loads of all
  // chunks at once instead of four by four, and no sleep between two looks at the counter, took N = 7800 from 87.5 to 86.3 us
  // and N = 1024 with 2 heads from 19.5 to 18.5 us.  (Added up in the query stage's kernel instead, by its compute warps ahead of their first scores: its loads
  // come behind the first tiles' copies, 9.5 us where it takes 4 here, N = 32760 without softmax tokens 103.7 -> 108.9 us; by
  // one warp beside the key loop: latency after latency, N = 7800 82.6 -> 103.)
  __shared__ uint32_t s_go;                                    // 0: nothing, 1: this CTA's slice, 2: all slices
  uint32_t* cnt = p.counters + 2 * ((size_t)bh * gridDim.z + fc);
  const uint32_t n_ctas = gridDim.x;
  if (threadIdx.x == 0) {
    __threadfence();
    const uint32_t stored = atomicAdd(cnt, 1u);
    uint32_t go = (stored & 0xffffu) + 1u == n_ctas && stored >> 16 != 0u ? 2u : 1u, it = 0;
    long long t0 = 0;
    while ((*reinterpret_cast<volatile uint32_t*>(cnt) & 0xffffu) < n_ctas) {
      if ((++it & 15u) != 0u) continue;                        // a look at the counter is a round trip to L2: no need to sleep between
      const long long now = clock64();
      if (t0 == 0) t0 = now;
      if (now - t0 > kSumPatience) {
        if ((atomicAdd(cnt, 0x10000u) & 0xffffu) < n_ctas) go = 0u;
        break;
      }
    }
    s_go = go;
  }
  __syncthreads();
  const uint32_t go = s_go;
  if (go != 0u) {
    __threadfence();
    const int f0 = fc * 128, nf = min(128, p.F - f0);
    const size_t pitch = (size_t)p.F * D;                      // floats between two chunks' partials
    const float* src = p.part_s + ((size_t)bh * p.n_chunks * p.F + f0) * D;
    float* dS = p.S + ((size_t)bh * p.F + f0) * D;
    __nv_bfloat16* dSb = p.Sb + ((size_t)bh * p.F + f0) * D;
    const int n4 = nf * D / 4, per = (n4 + (int)n_ctas - 1) / (int)n_ctas;       // float4 entries, a CTA's slice
    const int i_end = go == 2u ? n4 : min(n4, (chunk + 1) * per);
    for (int i = (go == 2u ? 0 : chunk * per) + (int)threadIdx.x; i < i_end; i += K_THREADS) {
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
      int c = 0;
      for (; c < p.n_chunks; c += 12) {                        // up to twelve chunks' loads in flight, added in chunk order
        float4 v[12];
#pragma unroll
        for (int j = 0; j < 12; ++j)
          if (c + j < p.n_chunks) v[j] = __ldcg(reinterpret_cast<const float4*>(src + (c + j) * pitch) + i);
#pragma unroll
        for (int j = 0; j < 12; ++j)
          if (c + j < p.n_chunks) { acc.x += v[j].x; acc.y += v[j].y; acc.z += v[j].z; acc.w += v[j].w; }
      }
      reinterpret_cast<float4*>(dS)[i] = acc;
      reinterpret_cast<uint2*>(dSb)[i] = make_uint2(pack_bf16(acc.x, acc.y), pack_bf16(acc.z, acc.w));
    }
    if (chunk == 0 || go == 2u) {
      for (int f = threadIdx.x; f < nf; f += K_THREADS) {
        float acc = 0.f;
        for (int c = 0; c < p.n_chunks; c += 12) {
          float v[12];
#pragma unroll
          for (int j = 0; j < 12; ++j) v[j] = c + j < p.n_chunks ? __ldcg(p.part_z + ((size_t)bh * p.n_chunks + c + j) * p.F + f0 + f) : 0.f;
#pragma unroll
          for (int j = 0; j < 12; ++j)
            if (c + j < p.n_chunks) acc += v[j];
        }
        p.z[(size_t)bh * p.F + f0 + f] = acc;
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const uint32_t left = atomicAdd(cnt + 1, 1u);
    if (left + 1u == n_ctas) { cnt[0] = 0u; cnt[1] = 0u; }     // nobody looks at the first counter any more: ready for the next launch
  }
}

// ======================================================================================
// First layer of a two-layer feature map for the keys ("Characterization of phi": the embedding
// network): h1 = relu(k W_1^T + b_1), [B*H, N, hidden] bf16.  One 128-token tile per CTA.
// The softmax rows of K are copied to K_S here, where the K tile is in shared memory, by the warps that otherwise only wait
// for the product.  (The K pass, which has h1 tiles in its ring instead, fetched them from global memory one row after
// the other and held its slots of the ring meanwhile: the whole key side 338 us against 181 at N = 32760, rate 1/8, hidden =
// F = 256, the layer 1182 against 1071.)
// This one: hidden widths of 64 and 128, several CTAs on an SM; what bounds it is the chain of one (set-up, loads, product, rows, stores), so the rows are
// taken by eight warps, staged over the weights and stored at once, and the CTA ends when its stores have been read.
// ======================================================================================
// A dependent launch: its CTAs set up beside the kernel before it (N = 1144, 2 heads, 128 / 128: a call 28.9 -> 27.8 us; N = 1036, 5 heads, d = 64
// 24.9 -> 22.9).
struct P1Params { int H, hid, N, n_s, tiles, total; const __nv_bfloat16* bias; const int32_t* sm_rank; __nv_bfloat16* ks_w; uint32_t* status; };
constexpr int P1_THREADS = 288;          // warps 0-7: epilogue (two threads per token row, each half of a slice's columns); warp 8: TMA + MMA

template <int D>
struct P1Layout {
  static constexpr int TILE = 128 * D * 2;
  static constexpr int X_OFF = 0, W_OFF = TILE, BAR_OFF = 2 * TILE;
  static constexpr int BIAS_OFF = BAR_OFF + 64;                 // D floats
  static constexpr int TOTAL = BIAS_OFF + D * 4 + 1024;
};

// Copies rows row0 + i of a K tile, i the set bits, to the rows of the compact K_S that their lanes i hold in `rank`.  By a warp, D / 8 lanes a row.
template <int D>
AS_DEV void copy_rows(const uint8_t* tile, int row0, uint32_t bits, int rank, __nv_bfloat16* ks) {
  constexpr int CH = D / 8, RPI = 32 / CH;
  const int lane = threadIdx.x & 31, c = lane % CH;
  while (bits) {
    int src = -1;
#pragma unroll
    for (int i = 0; i < RPI; ++i) {
      if (bits) {
        if (lane / CH == i) src = __ffs(bits) - 1;
        bits &= bits - 1;
      }
    }
    const int to = __shfl_sync(0xffffffffu, rank, src < 0 ? 0 : src);
    if (src >= 0)
      *reinterpret_cast<uint4*>(ks + (size_t)to * D + c * 8) = *reinterpret_cast<const uint4*>(tile + (c / 8) * BOX_BYTES + swz128_chunk_offset(row0 + src, c % 8));
  }
}

template <int D>
__global__ void __launch_bounds__(P1_THREADS)
phi1_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW,
            const __grid_constant__ CUtensorMap tmH, const P1Params p) {
  using L = P1Layout<D>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t sbase = smem_u32(smem);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::BAR_OFF);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::BAR_OFF + 32);
  volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem + L::BAR_OFF + 36);
  float* sBias = reinterpret_cast<float*>(smem + L::BIAS_OFF);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t s_late = sbase + L::BAR_OFF + 48;               // the status word behind the wait: not 0, and nothing is written
  const int bh = blockIdx.y, h = bh % p.H, row0 = blockIdx.x * 128;
  const WaitCtx wc{p.status, abort_flag};
  const uint32_t bar_full = smem_u32(bars);
  const uint32_t bar_done = smem_u32(bars + 1);                  // the product has completed
  const uint32_t bar_late = smem_u32(bars + 2);                  // the status word is there
  constexpr int TM_COLS = 128;

  __shared__ uint32_t s_skip;
  if (threadIdx.x == 32) s_skip = status_now(p.status);
  if (threadIdx.x == 0) {
    *abort_flag = 0u;
    mbar_init(bar_full, 1);
    mbar_init(bar_done, 1);
    mbar_init(bar_late, 1);
    fence_barrier_init();
    fence_proxy_async();
  }
  if (warp == 8) { tmem_alloc(smem_u32(tmem_slot), TM_COLS); tmem_relinquish(); }
  griddep_wait();                                    // the set-up above ran beside the kernel before this one
  if (threadIdx.x == 0) status_again(s_late, p.status, bar_late);   // (the thread that has made the barrier)
  for (int i = threadIdx.x; i < D; i += P1_THREADS)
    sBias[i] = (p.bias != nullptr && i < p.hid) ? __bfloat162float(p.bias[(size_t)h * p.hid + i]) : 0.f;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (s_skip != 0u) {                                // an earlier launch timed out: do nothing
    if (warp == 8) tmem_dealloc(*tmem_slot, TM_COLS);
    return;
  }
  const uint32_t tmem = *tmem_slot;
  const uint32_t sX = sbase + L::X_OFF;
  const uint32_t sW = sbase + L::W_OFF;             // h1 is staged for its store over the weights, which nothing reads once the product has completed

  if (warp == 8) {
    if (lane == 0) {
      mbar_expect_tx(bar_full, 2 * L::TILE);
      load_tile<D>(sX, &tmX, bar_full, row0, bh);
      load_tile<D>(sW, &tmW, bar_full, 0, h);          // W_1[h] (rows past hid: zeros)
    }
    __syncwarp();
    if (mbar_wait_warp(bar_full, 0, wc)) {
      tc_fence_after();
      if (lane == 0) {
        issue_kmajor<D>(tmem, kmajor_desc(sX), kmajor_desc(sW), make_idesc(128, D, 0, 0), false);   // X W_1^T
        tc_commit(bar_done);
      }
      __syncwarp();
    }
  } else {
    const int quad = warp & 3, hf = warp >> 2, r = quad * 32 + lane;
    const uint32_t lane_off = (uint32_t)(quad * 32) << 16;
    const bool live = __all_sync(0xffffffffu, status_clear(bar_late, s_late));
    bool ok = true;
    if (live && p.ks_w != nullptr) {
      const int rank = lane / 16 == hf && row0 + r < p.N ? p.sm_rank[row0 + r] : -1;
      const uint32_t bits = __ballot_sync(0xffffffffu, rank >= 0);
      if (bits) ok = mbar_wait_warp(bar_full, 0, wc);
      if (ok) copy_rows<D>(smem + L::X_OFF, quad * 32, bits, rank, p.ks_w + (size_t)bh * p.n_s * D);
      __syncwarp();
    }
    uint32_t x[32];
    if (ok) ok = mbar_wait_warp(bar_done, 0, wc);
    if (ok) {
      tc_fence_after();
#pragma unroll
      for (int c = 0; c < D / 64; ++c) {
        const int col = hf * (D / 2) + c * 32;
        tmem_ld32(tmem + lane_off + col, x);
        tmem_ld_wait(x);
        const float* bb = sBias + col;
        uint32_t w[16];
#pragma unroll
        for (int i = 0; i < 16; ++i)
          w[i] = pack_bf16(fmaxf(__uint_as_float(x[2 * i]) + bb[2 * i], 0.f), fmaxf(__uint_as_float(x[2 * i + 1]) + bb[2 * i + 1], 0.f));
        store_row_chunk(smem + L::W_OFF, r, col, w);
      }
      fence_proxy_async();
    }
    named_barrier_sync(1, 256);                               // reached by every epilogue thread, also after a failed wait
    if (ok && live && threadIdx.x == 0) {
#pragma unroll
      for (int b = 0; b < D / 64; ++b) tma_store_3d(&tmH, sW + b * BOX_BYTES, b * 64, row0, bh);
      tma_store_commit();
    }
    if (threadIdx.x == 0) tma_store_wait_read();              // (the writes land by the end of the kernel)
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 8) {
    tc_fence_after();
    tmem_dealloc(tmem, TM_COLS);
  }
}

// The same for a hidden width of 256 at d = 128, bound by HBM (k in, h1 out twice as wide): a CTA per SM takes a run of tiles, one after the other.  The
// head's weights stay in shared memory, three tiles of K are in flight, the products of a tile run under the rows of the one before (two sets of
// accumulators), and a slice of h1 is stored while the next one is formed.  Where a run goes on into the next head, its weights come when the last
// product with the old ones has completed; its first tile of K is asked for before that.  N = 32760, 12 heads, no softmax tokens: this stage 65 -> 56 us (floor
// 46), the call 314 -> 304; rate 1/8 990 -> 980, N = 7800 140.5 -> 138.1, 8 heads of N = 1560 38.4 -> 37.7.  Narrower maps keep the kernel above, which has
// several CTAs on an SM there: in runs of tiles, 128 / 128 with 2 heads of N = 1560 27.4 -> 28.2 us, d = 64 with 12 of 7800 78.4 -> 79.5 (24 of 15600 without
// softmax tokens 110.9 -> 107.1).  Tried: softmax rows of K copied behind the slices' rows instead of ahead of them, N = 15600, 16 heads 85.5 -> 87.5.
constexpr int P1R_THREADS = 320;          // warps 0-7: epilogue (two threads per token row, each half of a slice's columns); 8: TMA; 9: MMA
constexpr int P1R_RING = 3;               // tiles of K in shared memory

struct P1RLayout {
  static constexpr int D = 128, NH = 2;
  static constexpr int TILE = 128 * D * 2;
  static constexpr int W_OFF = 0, X_OFF = NH * TILE, OUT_OFF = X_OFF + P1R_RING * TILE, BAR_OFF = OUT_OFF + 2 * TILE;
  static constexpr int BIAS_OFF = BAR_OFF + 192;                // NH * D floats
  static constexpr int TOTAL = BIAS_OFF + NH * D * 4 + 1024;
  static constexpr int COLS = 2 * NH * D;                       // tensor memory: two tiles' products
  static_assert(TOTAL <= 227 * 1024 && COLS == 512);
};

__global__ void __launch_bounds__(P1R_THREADS)
phi1_run_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW,
            const __grid_constant__ CUtensorMap tmH, const P1Params p) {
  using L = P1RLayout;
  constexpr int D = L::D, NH = L::NH;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t sbase = smem_u32(smem);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::BAR_OFF);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::BAR_OFF + 160);
  volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem + L::BAR_OFF + 164);
  __shared__ __align__(16) volatile uint32_t s_late[4];        // the status word behind the wait: not 0, and nothing is written
  float* sBias = reinterpret_cast<float*>(smem + L::BIAS_OFF);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t0 = (int)((long long)blockIdx.x * p.total / gridDim.x), t1 = (int)((long long)(blockIdx.x + 1) * p.total / gridDim.x);
  const WaitCtx wc{p.status, abort_flag};
  auto bar_x = [&](int s) { return smem_u32(bars + s); };                            // ring slot s: its tile has arrived
  auto bar_x_empty = [&](int s) { return smem_u32(bars + P1R_RING + s); };            // read by the products and, for softmax rows, by the eight warps
  auto bar_w = [&](int j) { return smem_u32(bars + 2 * P1R_RING + j); };              // a head's weights of slice j
  const uint32_t bar_w_free = smem_u32(bars + 2 * P1R_RING + 2);                      // the last product with them has completed
  auto bar_done = [&](int b, int j) { return smem_u32(bars + 2 * P1R_RING + 3 + 2 * b + j); };   // accumulators b: slice j's product has completed
  auto bar_free = [&](int b) { return smem_u32(bars + 2 * P1R_RING + 7 + b); };       // accumulators b have been read
  const uint32_t bar_late = smem_u32(bars + 2 * P1R_RING + 9);                        // the status word is there
  static_assert((2 * P1R_RING + 10) * 8 <= 160);

  const int quad = warp & 3, hf = (warp >> 2) & 1, r = quad * 32 + lane;
  auto head_of = [&](int t) { return t / p.tiles % p.H; };
  auto rank_of = [&](int t) {            // of the sixteen rows of tile t whose softmax rows this warp copies
    const int row = t % p.tiles * 128 + r;
    return p.ks_w != nullptr && warp < 8 && lane / 16 == hf && t < t1 && row < p.N ? p.sm_rank[row] : -1;
  };
  auto load_bias = [&](int h) {          // by the eight warps
    for (int i = threadIdx.x; i < NH * D; i += 256)
      sBias[i] = (p.bias != nullptr && i < p.hid) ? __bfloat162float(p.bias[(size_t)h * p.hid + i]) : 0.f;
  };
  __shared__ uint32_t s_skip;
  if (threadIdx.x == 32) s_skip = status_now(p.status);
  if (threadIdx.x == 0) {
    *abort_flag = 0u;
    for (int s = 0; s < P1R_RING; ++s) { mbar_init(bar_x(s), 1); mbar_init(bar_x_empty(s), p.ks_w != nullptr ? 9 : 1); }
    for (int j = 0; j < 2; ++j) {
      mbar_init(bar_w(j), 1);
      mbar_init(bar_free(j), 8);
      for (int b = 0; b < 2; ++b) mbar_init(bar_done(b, j), 1);
    }
    mbar_init(bar_w_free, 1);
    mbar_init(bar_late, 1);
    fence_barrier_init();
    fence_proxy_async();
  }
  if (warp == 8 && lane == 0) { tma_prefetch_desc(&tmX); tma_prefetch_desc(&tmW); tma_prefetch_desc(&tmH); }
  if (warp == 9) { tmem_alloc(smem_u32(tmem_slot), L::COLS); tmem_relinquish(); }   // (dependents let in early gain nothing)
  int rank_now = rank_of(t0), rank_next = rank_of(t0 + 1);     // two tiles ahead: a load behind copies of tiles takes microseconds
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  griddep_wait();                                    // the set-up above ran beside the kernel before this one
  if (s_skip != 0u) {                                // an earlier launch timed out: do nothing
    if (warp == 9) tmem_dealloc(tmem, L::COLS);
    return;
  }

  if (warp == 8) {
    if (lane == 0) {
      uint32_t n_w = 0;
      for (int t = t0, i = 0; t < t1; ++t, ++i) {
        const int bh = t / p.tiles, h = bh % p.H, s = i % P1R_RING;
        if (i >= P1R_RING && !mbar_wait(bar_x_empty(s), (i / P1R_RING - 1) & 1, wc)) break;
        mbar_expect_tx(bar_x(s), L::TILE);
        load_tile<D>(sbase + L::X_OFF + s * L::TILE, &tmX, bar_x(s), (t - bh * p.tiles) * 128, bh);
        if (i > 0 && h == head_of(t - 1)) continue;
        if (i > 0 && !mbar_wait(bar_w_free, (n_w - 1) & 1, wc)) break;
        for (int j = 0; j < NH; ++j) {
          mbar_expect_tx(bar_w(j), L::TILE);
          load_tile<D>(sbase + L::W_OFF + j * L::TILE, &tmW, bar_w(j), j * 128, h);   // W_1[h] rows of slice j (past hid: zeros)
        }
        ++n_w;
      }
    }
    __syncwarp();
  } else if (warp == 9) {
    if (lane == 0) status_again(smem_u32(const_cast<uint32_t*>(s_late)), p.status, bar_late);
    __syncwarp();
    uint32_t n_w = 0;
    bool ok = true;
    for (int t = t0, i = 0; ok && t < t1; ++t, ++i) {
      const int s = i % P1R_RING, b = i & 1;
      const bool first = i == 0 || head_of(t) != head_of(t - 1), last = t + 1 < t1 && head_of(t) != head_of(t + 1);
      if (i >= 2) ok = mbar_wait_warp(bar_free(b), ((i >> 1) - 1) & 1, wc);
      ok = ok && mbar_wait_warp(bar_x(s), (i / P1R_RING) & 1, wc);
      for (int j = 0; j < NH; ++j) {         // X W_1^T: the D hidden units of slice j
        if (first) ok = ok && mbar_wait_warp(bar_w(j), n_w & 1, wc);
        if (!ok) break;
        tc_fence_after();
        if (elect_one()) {
          issue_kmajor<D>(tmem + (b * NH + j) * D, kmajor_desc(sbase + L::X_OFF + s * L::TILE), kmajor_desc(sbase + L::W_OFF + j * L::TILE),
                          make_idesc(128, D, 0, 0), false);
          tc_commit(bar_done(b, j));
          if (j == NH - 1 && t + P1R_RING < t1) tc_commit(bar_x_empty(s));
          if (j == NH - 1 && last) tc_commit(bar_w_free);
        }
        __syncwarp();
      }
      n_w += first ? 1 : 0;
    }
  } else {
    const uint32_t lane_off = (uint32_t)(quad * 32) << 16;
    load_bias(head_of(t0));                                     // (they meet below before the first look at it)
    bool ok = __all_sync(0xffffffffu, status_clear(bar_late, smem_u32(const_cast<uint32_t*>(s_late))));
    if (!ok) status_give_up(wc);                                // the launch before has timed out: nothing is written
    for (int t = t0, i = 0; t < t1; ++t, ++i) {
      const int bh = t / p.tiles, s = i % P1R_RING, b = i & 1, row0 = (t - bh * p.tiles) * 128;
      const int rank = rank_now;
      rank_now = rank_next;
      rank_next = rank_of(t + 2);
      if (i > 0 && p.bias != nullptr && bh % p.H != head_of(t - 1)) {
        load_bias(bh % p.H);                                    // (all have read the old one: they met behind it)
      }
      if (p.ks_w != nullptr) {
        const uint32_t bits = __ballot_sync(0xffffffffu, rank >= 0);
        if (ok) ok = mbar_wait_warp(bar_x(s), (i / P1R_RING) & 1, wc);
        if (ok) copy_rows<D>(smem + L::X_OFF + s * L::TILE, quad * 32, bits, rank, p.ks_w + (size_t)bh * p.n_s * D);
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_x_empty(s));
      }
      uint32_t x[32];
#pragma unroll
      for (int j = 0; j < NH; ++j) {
        const int out = L::OUT_OFF + ((i * NH + j) & 1) * L::TILE;
        if (ok) ok = mbar_wait_warp(bar_done(b, j), (i >> 1) & 1, wc);
        if (threadIdx.x == 0) tma_store_wait_read_but_last();   // the store before the last one has read its tile, which is `out`
        named_barrier_sync(1, 256);                             // these two are reached by every epilogue thread, also after a failed wait
        if (ok) {
          tc_fence_after();
#pragma unroll
          for (int c = 0; c < D / 64; ++c) {
            const int col = hf * (D / 2) + c * 32;
            tmem_ld32(tmem + lane_off + (b * NH + j) * D + col, x);
            tmem_ld_wait(x);
            const float* bb = sBias + j * D + col;
            uint32_t w[16];
#pragma unroll
            for (int i = 0; i < 16; ++i)
              w[i] = pack_bf16(fmaxf(__uint_as_float(x[2 * i]) + bb[2 * i], 0.f), fmaxf(__uint_as_float(x[2 * i + 1]) + bb[2 * i + 1], 0.f));
            store_row_chunk(smem + out, r, col, w);
          }
          fence_proxy_async();
          if (j == NH - 1) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_free(b));
          }
        }
        named_barrier_sync(1, 256);
        if (ok && threadIdx.x == 0) {
#pragma unroll
          for (int q = 0; q < D / 64; ++q) tma_store_3d(&tmH, sbase + out + q * BOX_BYTES, j * D + q * 64, row0, bh);
          tma_store_commit();
        }
      }
    }
    if (threadIdx.x == 0) tma_store_wait_read();              // (the writes land by the end of the kernel)
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 9) {
    tc_fence_after();
    tmem_dealloc(tmem, L::COLS);
  }
}

template <int D, int LAYERS, int NH>
cudaError_t launch_kpass(const CUtensorMap& tmK, const CUtensorMap& tmV, const CUtensorMap& tmW, const CUtensorMap& tmH,
                         const KParams& p, dim3 grid, cudaStream_t st) {
  return as_launch_dependent(kpass_kernel<D, LAYERS, NH>, grid, dim3(K_THREADS), KLayout<D, LAYERS, NH>::TOTAL, st, tmK, tmV, tmW, tmH, p);
}

}  // namespace

cudaError_t as_tensor_init_kpass() {
  cudaError_t e;
  if ((e = opt_in_smem(kpass_kernel<128, 1, 1>, KLayout<128, 1, 1>::TOTAL)) != cudaSuccess) return e;
  if ((e = opt_in_smem(kpass_kernel<64, 1, 1>, KLayout<64, 1, 1>::TOTAL)) != cudaSuccess) return e;
  if ((e = opt_in_smem(kpass_kernel<128, 2, 1>, KLayout<128, 2, 1>::TOTAL)) != cudaSuccess) return e;
  if ((e = opt_in_smem(kpass_kernel<128, 2, 2>, KLayout<128, 2, 2>::TOTAL)) != cudaSuccess) return e;
  if ((e = opt_in_smem(kpass_kernel<64, 2, 1>, KLayout<64, 2, 1>::TOTAL)) != cudaSuccess) return e;
  if ((e = opt_in_smem(phi1_kernel<128>, P1Layout<128>::TOTAL)) != cudaSuccess) return e;
  if ((e = opt_in_smem(phi1_run_kernel, P1RLayout::TOTAL)) != cudaSuccess) return e;
  if ((e = opt_in_smem(phi1_kernel<64>, P1Layout<64>::TOTAL)) != cudaSuccess) return e;
  return cudaSuccess;
}

// First layer of the key feature map: h1k = relu(k W_k1^T + b_k1).
cudaError_t as_tensor_phi1(const as_launch_args& a, cudaStream_t st) {
  const int BH = a.B * a.H;
  CUtensorMap tmX, tmW, tmH;
  if (!make_map(&tmX, a.k, a.d, a.N, BH, 128) || !make_map(&tmW, a.wk, a.d, a.hid, a.H, 128) ||
      !make_map(&tmH, a.h1k, a.hid, a.N, BH, 128))
    return cudaErrorInvalidValue;
  const int tiles = (a.N + 127) / 128;
  P1Params p{a.H, a.hid, a.N, a.n_s, tiles, tiles * BH, a.bk1, a.sm_rank, a.ks_w, a.status};
  if (a.d == 128 && a.hid == 256) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
      return cudaErrorInvalidValue;
    return as_launch_dependent(phi1_run_kernel, dim3(std::min(p.total, sms)), dim3(P1R_THREADS), P1RLayout::TOTAL, st, tmX, tmW, tmH, p);
  }
  dim3 grid(tiles, BH, 1);
  if (a.d == 128) return as_launch_dependent(phi1_kernel<128>, grid, dim3(P1_THREADS), P1Layout<128>::TOTAL, st, tmX, tmW, tmH, p);
  return as_launch_dependent(phi1_kernel<64>, grid, dim3(P1_THREADS), P1Layout<64>::TOTAL, st, tmX, tmW, tmH, p);
}

cudaError_t as_tensor_kpass(const as_launch_args& a, cudaStream_t st) {
  const int BH = a.B * a.H;
  const bool two = a.layers == 2;
  CUtensorMap tmK, tmV, tmW, tmH;
  if (!make_map(&tmK, a.k, a.d, a.N, BH, 128) || !make_map(&tmV, a.v, a.d, a.N, BH, 128)) return cudaErrorInvalidValue;
  // last-layer weights [H][F][width of their input]
  if (!make_map(&tmW, two ? a.wk2 : a.wk, two ? a.hid : a.d, a.F, a.H, 128)) return cudaErrorInvalidValue;
  if (two) { if (!make_map(&tmH, a.h1k, a.hid, a.N, BH, 128)) return cudaErrorInvalidValue; }
  else tmH = tmK;               // never used with a one-layer map
  KParams p{};
  p.N = a.N; p.n_s = a.n_s; p.n_chunks = a.n_chunks; p.chunk_tiles = a.chunk_tiles; p.P = a.P; p.F = a.F;
  p.H = a.H; p.sm_rank = a.sm_rank; p.ks_w = a.ks_w; p.vs_w = a.vs_w;
  p.bias = two ? a.bk2 : a.bk1;
  p.part_s = a.part_s; p.part_z = a.part_z; p.status = a.status;
  p.S = a.S; p.z = a.z; p.Sb = a.Sb; p.counters = a.counters;
  dim3 grid(a.n_chunks, BH, (a.F + 127) / 128);
  if (a.d == 128) {
    if (!two) return launch_kpass<128, 1, 1>(tmK, tmV, tmW, tmH, p, grid, st);
    if (a.hid == 256) return launch_kpass<128, 2, 2>(tmK, tmV, tmW, tmH, p, grid, st);
    return launch_kpass<128, 2, 1>(tmK, tmV, tmW, tmH, p, grid, st);
  }
  if (!two) return launch_kpass<64, 1, 1>(tmK, tmV, tmW, tmH, p, grid, st);
  return launch_kpass<64, 2, 1>(tmK, tmV, tmW, tmH, p, grid, st);
}
