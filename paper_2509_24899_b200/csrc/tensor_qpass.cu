// Q pass of the hybrid attention forward on the tensor cores of sm_100a: softmax branch, phi_q
// projection, linear apply and merge, fused in one persistent kernel.
//
//   persistent, one CTA per SM (what is left over after the full rounds is dealt out in one last round, in
//   units of two 128-row tiles or of one, see as_plan_units, or by key tiles, see as_plan_parts); per unit a flash-style loop over 128-key tiles
//   of K_S / V_S:        S = Q K_S^T -> TMEM; the softmax threads (one or two per row) read their row and
//                        release the score columns at once, so the next product into them runs under the
//                        exponentials; running max / sum per row; P = exp2(.) as bf16 -> TMEM,
//                        O += P V_S (TMEM x smem -> TMEM).  Two issuing warps: one for what writes
//                        the score columns, one for what accumulates into O.
//   tail, per chunk c of 128 features:
//                        Phi_c = Q W_q[c]^T -> TMEM (in the place of a next tile's scores), phi_q scaled per
//                        row as bf16 into shared memory, O += phi_q,c S_c (S in bf16 read like a V tile),
//                        den = l + phi_q.z, y = O / den -> bf16 -> staged where phi_q sat -> TMA store.
//   two-layer feature map: the hidden activations relu(Q W_q1^T + b1) are formed in the same way first
//                        (128 hidden units at a time) and kept as bf16 in the group's phi_q tile and, once nothing reads
//                        Q any more, in the Q tile; Phi_c = sum over the hidden slices of h1_j W_q2[c, j]^T.
// All tiles are staged by TMA with the 128-byte swizzle; every mbarrier wait is bounded.
#include "query_plan.h"
#include "tensor_common.cuh"

namespace {

using namespace as_tc;

// ======================================================================================
// Q pass
// ======================================================================================
struct QParams {
  int N, n_s, nkv, lin, stab_mode, P, H;
  int layers;                // depth of the feature map (1 or 2)
  int F, fc, fcw;            // feature width, its chunks of 128 (ceil), width of a chunk (min(F, 128))
  int nh;                    // two layers: slices of the hidden width (each D wide)
  const __nv_bfloat16* b1;   // two layers: first-layer bias of this launch's first head [H][hidden], or nullptr
  const __nv_bfloat16* b2;   // last-layer bias [H][F], or nullptr
  int nx, n_pairs;           // two-tile units per (batch, head); over all (batch, head) pairs
  int n_single;              // units of a (batch, head)'s last tile alone: one per (batch, head) or none
  int n_rounds;              // rounds in which every CTA has a two-tile unit (n_pairs / gridDim.x)
  int split_last;            // 1: the two-tile units left over after those rounds are cut in two, one tile per CTA
  float scale_log2;          // softmax scale * log2(e)
  const float* z;            // [B*H][F]
  float* aux;                // [B*H][N][3] or nullptr
  uint32_t* status;
  // ---- key loops in parts (cf. as_plan_parts; only the kernels compiled for them look at these)
  int share;                 // key tiles of a CTA in the last round; 0: units are whole
  float* parts;              // [CTAs]: what a CTA leaves of a unit that another one finishes, see QPart
  uint32_t* part_flags;      // [CTAs][compute warps, AS_PART_FLAGS at most]: what the warp leaves is there; zero between launches
  const __nv_bfloat16* v;    // the keys' values [B*H][v_rows][D]
  int v_rows;
  uint32_t* part_ticket;     // which CTA of the last round a CTA is: the order in which they have started; zero between launches
  // of one part (0 / unused in the launch's own parameters): in place of nkv, n_s and lin above those of the part, and
  int part;                  // 1: a part
  int cta;                   // the CTA's index in the last round
  int bh, row0, key0;        // its unit; its first key
  int at_items, at_s, at_p, at_pf, at_tail;   // ring items, phases and tails of the CTA before it
  int leaves, merges;        // 1: leaves what it has to another CTA; number of CTAs right before this one that have left it theirs
};

// How the compute threads share a 128-row tile: T = 1, one thread per row (eight warps), or T = 2, threads t and t + 16 of a warp, each
// with half of the row's columns (sixteen warps; the two share their maxima and sums by one shuffle).  cf. as_threads_per_row.
template <int T>
struct QShape {
  static constexpr int COLS = 128 / T;                     // score columns of a thread
  static constexpr int W_TMA = 8 * T, W_SCORE = W_TMA + 1, W_ACCUM = W_TMA + 2;
  // warps 0 .. 8 * T - 1: compute (quadrant = bits 0-1, group = bit 2, T = 2: half of the quadrant's rows = bit 3)
  static constexpr int THREADS = (W_TMA + 3) * 32, GROUP = 128 * T;
};
// The feature maps that the kernel with a key loop is compiled for: one layer, one layer whose tail is several products at d = 128 (more than 128
// features; not where a CTA has one tile only and there are no groups to take turns), two layers.
constexpr int MAP_ONE = 0, MAP_WIDE = 1, MAP_TWO = 2;
constexpr int KV_STAGES = 3;
constexpr float RESCALE_THRESHOLD = 8.f; // log2 units: rescale O only when the row max grew by > 2^8

// A thread's share of a row (of 32 columns in TMEM; SPLIT: distance of the two threads' shares where two share a row)
template <int T, int SPLIT>
AS_DEV void q_ld32(uint32_t t, uint32_t (&x)[32]) {
  if constexpr (T == 1) tmem_ld32(t, x); else tmem_ldh32<SPLIT>(t, x);
}
template <int T, int SPLIT>
AS_DEV void q_ld16(uint32_t t, uint32_t (&x)[16]) {
  if constexpr (T == 1) tmem_ld16(t, x); else tmem_ldh16<SPLIT>(t, x);
}
template <int T, int SPLIT>
AS_DEV void q_st16(uint32_t t, const uint32_t (&x)[16]) {
  if constexpr (T == 1) tmem_st16(t, x); else tmem_sth16<SPLIT>(t, x);
}

// Two exponentials 2^x, x <= 8, on the FMA pipe: x = n + f with n the nearest integer (added into the last bits of 1.5 * 2^23), 2^f by
// the polynomial of degree 5 with constant term 1 that is closest to it on [-1/2, 1/2] in relative error (1.08e-7 with the coefficients
// rounded, found by reweighted least squares), times 2^n put together from its exponent.  Within 1.72e-7 of 2^x for all x in [-126, 8]
// (ex2.approx: 2.4e-7).  Below that 0, as ex2.approx.ftz gives it: 2^-127 comes out of the exponent as 0, and the product flushes what lies
// between (a key far below its row's maximum weighs nothing in every column, also with a value near the end of the range).  What is no
// number stays none.
AS_DEV float2 ex2_fma(float2 x) {
  auto both = [](float v) { return make_float2(v, v); };
  x = make_float2(fmax_nan(x.x, -127.f), fmax_nan(x.y, -127.f));
  const float2 t = __fadd2_rn(x, both(12582912.f));
  const float2 f = __ffma2_rn(__fadd2_rn(t, both(-12582912.f)), both(-1.f), x);
  float2 y = __ffma2_rn(both(1.326472731307149e-3f), f, both(9.671512991189957e-3f));
  y = __ffma2_rn(y, f, both(5.550733581185341e-2f));
  y = __ffma2_rn(y, f, both(2.4022242426872253e-1f));
  y = __ffma2_rn(y, f, both(6.931470036506653e-1f));
  y = __ffma2_rn(y, f, both(1.f));
  const float2 p = make_float2(__uint_as_float((__float_as_uint(t.x) << 23) + 0x3f800000u), __uint_as_float((__float_as_uint(t.y) << 23) + 0x3f800000u));
  return fmul2_ftz(y, p);
}

// The second two of the i-th group of four exponentials.  Sixteen warps: every fourth such pair on the FMA pipe, one exponential in eight of all (the
// special-function unit, 16 a clock, is what four warps per sub-partition wait for): d = 64, N 8505, 2142 keys 293 -> 279 us; one in
// sixteen 284, one in four 304.  Eight warps: none (81 frames of full softmax 4637 us; one in sixteen 4650, one in eight 4709).
template <int T>
AS_DEV float2 ex2_second_pair(int i, float2 x) { return T == 2 && i % 4 == 3 ? ex2_fma(x) : make_float2(ex2(x.x), ex2(x.y)); }

template <int D>
struct QLayout {
  static constexpr int TILE = 128 * D * 2;                 // bytes of a [128 x D] bf16 tile
  static constexpr int PTILE = 128 * 128 * 2;              // bytes of a [128 rows x 128 features] bf16 tile
  static constexpr int Q_OFF = 0;
  static constexpr int P_OFF = 2 * TILE;                   // per group: phi_q, then the output rows
  static constexpr int KV_OFF = P_OFF + 2 * PTILE;
  static constexpr int BAR_OFF = KV_OFF + KV_STAGES * TILE;
  static constexpr int LATE_OFF = BAR_OFF + 240;           // the status word behind the wait for the kernel before
  static constexpr int TOTAL = BAR_OFF + 256 + 1024;       // + slack for the 1024-byte alignment
};

// Persistent: one CTA per SM walks over units of two 128-row tiles (unit w = blockIdx.x + u * gridDim.x, the last one
// from as_plan_units; the units of one (batch, head) are consecutive, so the CTAs that run at the same time
// share K_S / V_S in L2).
// Barrier phases and the K/V ring run on across units.
//
// Scores and probabilities live in different columns of tensor memory: the softmax threads read their rows of S = Q K^T into
// registers and release the S columns at once; P goes back into columns of its own as bf16 and is the A operand of O += P V.  A
// group waits for the tensor pipe neither with its scores nor with P in the steady state, and V is all that the second product
// reads from shared memory.  (P through shared memory, with score columns for each group at d = 128, before: every key tile cost the
// threads 16-byte stores, a proxy fence and a tile to wait for.  Measured in turn: 81 frames of full softmax 4940 -> 4720 us in short
// runs, 81 frames at rate 1/8 710 -> 690, N = 7800 84.4 -> 82.4.)
//
// d = 128: both groups use the same 128 score columns in the key loop, in turn: Q_1 K(j)^T follows once group 0 has read its tile j, Q_0 K(j+1)^T once
// group 1 has read its tile j.  A product into them takes 512 clk, the groups' reads 150 each and their waits and commits as much, so a
// round is 2100 - 2500 clk where the exponentials of both groups take 2048 at the least: the groups run half a period
// apart and little waits for the columns.  In the long tail of a two-layer map, where a group has little else to do than to wait for its
// next columns, group 1 has the columns of both P's instead (32 key tiles 920 -> 890 us), and in that of a one-layer map with several feature
// chunks (see own_tail).  One warp that issues everything in that fixed order, the second product in halves around
// the next scores, is slower (full softmax 4700 -> 5130 us): issuing blocks it.
//
// The work of one unit is a function per role, kept out of line: each role then gets a register
// allocation of its own (the softmax rows need nearly the whole budget, and the issuing warps must
// not spill).  Everything about a unit is derived from its index u inside the function.
struct QCtx {
  uint32_t sbase;            // shared-memory window address of the 1024-aligned base
  uint32_t tmem;             // TMEM base address
  WaitCtx wc;
};

// Unit u of this CTA: which (batch, head), the row it starts at, and how many of the two 128-row groups work on it.  In
// the rounds every CTA takes part in, CTA c has two-tile unit c + u * gridDim.x.  Last, each CTA takes at most one of what
// is left: two-tile units - cut into their two tiles where CTAs enough are left for that - and the last tiles of heads with
// an odd number of them (see as_plan_units).  A group that has the tensor and XU pipes to itself needs about two thirds of
// the time that the two of a two-tile unit take.
struct QUnit { int bh, row0, ng; };
template <bool KS = false>
AS_DEV QUnit q_unit(const QParams& p, int u) {
  if (KS && p.part) return QUnit{p.bh, p.row0, 2};
  const int c = (int)blockIdx.x, n = (int)gridDim.x;
  int w = c + u * n, half = 0, ng = 2;
  if (u >= p.n_rounds) {
    const int left = p.n_pairs - p.n_rounds * n, cut = p.split_last ? 2 * left : left;
    if (c >= cut) return QUnit{c - cut, p.nx * 256, 1};
    if (p.split_last) { w = p.n_rounds * n + (c >> 1); half = (c & 1) * 128; ng = 1; }
  }
  return QUnit{w / p.nx, (w % p.nx) * 256 + half, ng};
}
// number of units CTA c walks over
AS_DEV int q_units_of_cta(const QParams& p) {
  const int left = p.n_pairs - p.n_rounds * (int)gridDim.x;
  return p.n_rounds + ((int)blockIdx.x < (p.split_last ? 2 * left : left) + p.n_single ? 1 : 0);
}

// Tensor memory, 512 columns: O takes 2 x D, P (bf16 pairs) 2 x 64.  At d = 64 that leaves score columns for each group, at d = 128
// for one: there the groups take turns at them.
template <int D, bool SH = (D == 128)>
struct QRing {
  using L = QLayout<D>;
  // barrier indices; per group: S (scores, hidden activations or Phi landed in the score columns), SF (score
  // columns read out), P (P in tensor memory, phi_q in shared memory), PF (the product that reads it has completed),
  // O (output accumulator final), QF (nothing of the unit reads the Q tile any more), H (two layers: the
  // hidden activations are in shared memory); for both, a tail in columns of their own: PL (nothing reads the unit's P in tensor memory any more); once: LATE (the status word is there, cf. status_again)
  // Whether a ring slot is full is told on a barrier of the warp that will use the item: KFULL for what is multiplied into the score columns (K,
  // weights), VFULL for what is added to O (V, S).  Each warp looks at every phase of its own barriers, in order.  (With one barrier for both a
  // warp would look at some of its phases only, and a wait by parity for a phase two ahead of the last one looked at passes while
  // the one between - a copy still under way for the other warp - is not over.)
  static constexpr int B_Q0 = 0, B_KFULL = 2, B_VFULL = B_KFULL + KV_STAGES, B_EMPTY = B_VFULL + KV_STAGES, B_S = B_EMPTY + KV_STAGES, B_SF = B_S + 2,
                       B_P = B_SF + 2, B_PF = B_P + 2, B_O = B_PF + 2, B_QF = B_O + 2, B_H = B_QF + 2, B_PL = B_H + 2, B_LATE = B_PL + 1, B_COUNT = B_LATE + 1;
  static_assert(8 * B_COUNT + 8 <= L::LATE_OFF - L::BAR_OFF, "two words follow the barriers");
  const QCtx c;              // by value: nothing here is re-read from memory after a barrier or an MMA
  int nkv, lin, two, fc, nh, vl;
  int n_stream, n_items;
  int n_s, n_p, n_pf;        // per unit and group: uses of the score columns, hand-overs of P or phi_q, products that have read one
  // Ring items of one unit, in the order they are consumed: K_0; then K_{j+1}, V_j for j = 0 .. nkv-2; then
  // the linear tail with V_{nkv-1} in second place:
  //   one layer:   W[0], V_last, then W[c], S[c-1] for c = 1 .. fc-1, then S[fc-1]
  //   two layers:  W1[0], V_last, W1[1 .. nh-1], then W2[c, j] (c slow), then S[0 .. fc-1]
  // addresses and waits only (the key loop needs nothing else)
  AS_DEV explicit QRing(const QCtx& c_) : c(c_), nkv(0), lin(0), two(0), fc(0), nh(0), vl(0), n_stream(0), n_items(0), n_s(0), n_p(0), n_pf(0) {}
  // `uniform`: for warps that issue MMAs, addresses that the compiler can see to be the same in all lanes
  AS_DEV QRing(const QParams& p, const QCtx& c_, bool uniform = false)
      : c(uniform ? QCtx{__shfl_sync(0xffffffffu, c_.sbase, 0), __shfl_sync(0xffffffffu, c_.tmem, 0), c_.wc} : c_),
        nkv(p.nkv), lin(p.lin), two(p.lin && p.layers == 2), fc(p.lin ? p.fc : 0), nh(p.nh), vl(p.nkv > 0 ? 1 : 0) {
    n_stream = nkv > 0 ? 2 * nkv - 1 : 0;
    n_items = n_stream + vl + (two ? nh + fc * nh + fc : 2 * fc);
    n_s = nkv + (two ? nh + fc : fc);
    n_p = nkv + fc;
    n_pf = nkv + (two ? 1 : fc);
  }
  AS_DEV int item_k(int j) const { return j == 0 ? 0 : 2 * j - 1; }
  AS_DEV int it_vlast() const { return n_stream + (lin ? 1 : 0); }   // after the tail's first weight tile, if there is a tail
  AS_DEV int item_v(int j) const { return j + 1 < nkv ? 2 * j + 2 : it_vlast(); }
  // one layer: last-layer weights of feature chunk ch; two layers: first-layer weights of hidden slice ch
  AS_DEV int it_w(int ch) const { return ch == 0 ? n_stream : (two ? n_stream + vl + ch : n_stream + vl + 2 * ch - 1); }
  AS_DEV int it_w2(int ch, int j) const { return n_stream + vl + nh + ch * nh + j; }
  AS_DEV int it_st(int ch) const {
    if (two) return n_stream + vl + nh + fc * nh + ch;
    return ch + 1 < fc ? n_stream + vl + 2 * ch + 2 : n_stream + vl + 2 * fc - 1;
  }
  AS_DEV uint32_t bar(int i) const { return c.sbase + L::BAR_OFF + 8 * i; }
  AS_DEV uint32_t sQ(int g) const { return c.sbase + L::Q_OFF + g * L::TILE; }
  AS_DEV uint32_t sP(int g) const { return c.sbase + L::P_OFF + g * L::PTILE; }
  // The K/V ring is indexed by a running item number that does not restart with a unit.
  AS_DEV uint32_t sKV(int item) const { return c.sbase + L::KV_OFF + (item % KV_STAGES) * L::TILE; }
  AS_DEV uint32_t tS(int g) const { return SH ? c.tmem : c.tmem + 128u * g; }
  AS_DEV uint32_t tP(int g) const { return c.tmem + (SH ? 128u : 384u) + 64u * g; }
  AS_DEV uint32_t tO(int g) const { return c.tmem + 256u + (uint32_t)D * g; }
  // At d = 128 a tail of several products lands in columns of each group's own: group 1 has those of both P's for it.  One layer with 256 features,
  // N = 32760, 12 heads, groups in turn -> own columns, two threads per row / one: 1 key tile 118 -> 114 / 134 -> 119 us, 8 tiles 271 -> 265 /
  // 281 -> 268; 512 features, 8 tiles 335 -> 323 / 367 -> 325.  (A tail of one product isn't worth the wait for the last P V of both groups:
  // N = 7800 79.4 -> 82.2 us.)
  template <int MAP>
  static constexpr bool own_tail = SH && MAP != MAP_ONE;
  template <int MAP>
  AS_DEV uint32_t tTail(int g) const { return own_tail<MAP> ? c.tmem + 128u * g : tS(g); }
  // Before product i of the unit into group g's score columns, the ph-th of all: what lay there has been read.  With columns of its own
  // (at d = 64; in a tail as above) by the group itself; else by the groups in turn.
  // (A unit of one group, the CTA's last one, follows a unit of two.)
  template <int MAP>
  AS_DEV bool s_free(int g, int ph, int ng, int i, int u) const {
    constexpr bool OWN = own_tail<MAP>;
    if (!SH || (OWN && (i > nkv || nkv == 0))) return ph == 0 ? true : wait(B_SF + g, ph - 1);
    if (g == 1) return !OWN || i < nkv ? wait(B_SF, ph) : wait(B_PL, u);
    if (ph == 0) return true;
    if (OWN && i == 0 && !wait(B_SF, ph - 1)) return false;   // the unit before: group 0's rows lay here, group 1's where P_0 will go
    return wait(B_SF + (ng == 2 || i == 0 ? 1 : 0), ph - 1);
  }
  AS_DEV bool wait(int b, int phase) const { return mbar_wait_warp(bar(b), phase & 1, c.wc); }
  AS_DEV void release(int item) const { tc_commit(bar(B_EMPTY + item % KV_STAGES)); }
  // `looks`: bit s is the parity of the next phase of the warp's barrier of slot s; it runs on across units
  AS_DEV bool wait_full(int b, int item, uint32_t& looks) const {
    const int slot = item % KV_STAGES, parity = (int)(looks >> slot) & 1;
    looks ^= 1u << slot;
    return wait(b + slot, parity);
  }
};

// ---------------------------------------------------------------- TMA producer
// The first copies of a CTA, by one thread: ring item 0 (the first key tile, else the first weights) and the first unit's Q tiles.  Right behind the wait for the kernel
// before, and a few lines of instructions of their own: as a part of q_produce_unit they went out 2500 - 3500 clk later, which is what its instructions and its
// parameters take to arrive in a CTA that has just started.  (Compiled into the kernel itself it moves q_softmax_unit's registers, N = 7800 + 2 us.)
template <int D, int MAP, bool KS = false>
__device__ __noinline__ void q_first_loads(const QParams& p, const QCtx& c, const QUnit& un, const CUtensorMap* tmQ, const CUtensorMap* tmK, const CUtensorMap* tmW,
                          const CUtensorMap* tmW1) {
  using R = QRing<D>;
  using L = QLayout<D>;
  const R q(c);
  const CUtensorMap* first = p.nkv > 0 ? tmK : MAP == MAP_TWO ? tmW1 : tmW;
  mbar_expect_tx(q.bar(R::B_KFULL), L::TILE);
  load_tile<D>(q.sKV(0), first, q.bar(R::B_KFULL), KS ? p.key0 : 0, p.nkv > 0 ? un.bh : un.bh % p.H);
  for (int g = 0; g < un.ng; ++g) {
    mbar_expect_tx(q.bar(R::B_Q0 + g), L::TILE);
    load_tile<D>(q.sQ(g), tmQ, q.bar(R::B_Q0 + g), un.row0 + g * 128, un.bh);
  }
}
// one unit
template <int D, int MAP, bool GEN, bool KS = false>
__device__ __noinline__ bool q_produce_unit(const QParams& p, const QCtx& c, const CUtensorMap* tmQ, const CUtensorMap* tmK,
                                            const CUtensorMap* tmV, const CUtensorMap* tmW, const CUtensorMap* tmSt,
                                            const CUtensorMap* tmW1, int u) {
  using R = QRing<D>;
  using L = QLayout<D>;
  const int nkv = p.nkv;
  const R q(p, c);
  const int lane = threadIdx.x & 31;
  const QUnit un = q_unit<KS>(p, u);
  const int bh = un.bh, h = bh % p.H, row0 = un.row0;
  const int base = KS && p.part ? p.at_items : u * q.n_items, key0 = KS ? p.key0 : 0;
  const int q_at = nkv > 0 ? 1 : 0;                   // the Q tiles are requested right after the unit's first K tile
  for (int it = 0; it < q.n_items; ++it) {
    if (it == q_at && u > 0) {
      for (int g = 0; g < un.ng; ++g) {
        // the previous unit's last product that reads this Q buffer has completed
        if (!q.wait(R::B_QF + g, u - 1)) return false;
        if (lane == 0) {
          mbar_expect_tx(q.bar(R::B_Q0 + g), L::TILE);
          load_tile<D>(q.sQ(g), tmQ, q.bar(R::B_Q0 + g), row0 + g * 128, bh);
        }
        __syncwarp();
      }
    }
    const int gi = base + it, st = gi % KV_STAGES;
    if (u == 0 && it == 0) continue;                  // (requested with the Q tiles, see q_first_loads)
    if (!q.wait(R::B_EMPTY + st, gi / KV_STAGES + 1)) return false;
    if (lane == 0) {
      const uint32_t dst = q.sKV(gi);
      auto to = [&](int b) { mbar_expect_tx(q.bar(b + st), L::TILE); return q.bar(b + st); };   // the barrier that the item arrives at
      if (it < q.n_stream) {
        if (it == 0 || (it & 1)) load_tile<D>(dst, tmK, to(R::B_KFULL), key0 + ((it + 1) >> 1) * 128, bh);   // K_0 at 0, K_j at 2j-1
        else load_tile<D>(dst, tmV, to(R::B_VFULL), key0 + ((it >> 1) - 1) * 128, bh);                 // V_j at 2j+2
      } else if (q.vl && it == q.it_vlast()) {
        load_tile<D>(dst, tmV, to(R::B_VFULL), key0 + (nkv - 1) * 128, bh);
      } else if (MAP != MAP_TWO) {
        // W[ch] / S[ch] in bf16: [128 feature rows][D]; rows past F arrive as zeros
        const int r = it - q.n_stream - (it > q.n_stream ? q.vl : 0);     // 0: W[0]; 2ch-1: W[ch]; 2ch+2 (and the last): S[ch]
        if (r == 0) load_tile<D>(dst, tmW, to(R::B_KFULL), 0, h);
        else if (r == 2 * q.fc - 1) load_tile<D>(dst, tmSt, to(R::B_VFULL), (q.fc - 1) * 128, bh);
        else if (r & 1) load_tile<D>(dst, tmW, to(R::B_KFULL), ((r + 1) >> 1) * 128, h);
        else load_tile<D>(dst, tmSt, to(R::B_VFULL), ((r >> 1) - 1) * 128, bh);
      } else {
        const int r = it - q.n_stream - (it > q.n_stream ? q.vl : 0);     // W1[0 .. nh-1], W2[c, j], S[c]
        if (r < q.nh) load_tile<D>(dst, tmW1, to(R::B_KFULL), r * 128, h);                                  // hidden rows of slice r
        else if (r < q.nh + q.fc * q.nh) {
          const int e = r - q.nh;
          load_boxes(dst, tmW, to(R::B_KFULL), (e % q.nh) * D, (e / q.nh) * 128, h, D / 64);                // W2[feature chunk, hidden slice]
        } else load_tile<D>(dst, tmSt, to(R::B_VFULL), (r - q.nh - q.fc * q.nh) * 128, bh);
      }
    }
    __syncwarp();
  }
  return true;
}

// ---------------------------------------------------------------- MMA issuers, one unit: what to look for next (see wait_full), or Q_FAILED
constexpr uint32_t Q_FAILED = ~0u;
// Two issuing warps: one issues what writes the score columns (Q K^T per tile, Phi at the end) as soon as
// the softmax threads have read them out, the other what accumulates into O (P V per tile, phi_q S at the end) as soon as
// P is there.  The two streams touch different TMEM columns and release different ring items, so they
// need no ordering between them; each warp's commits cover its own MMAs.  The whole warp walks the loop and one elected
// lane issues: from converged code the operands of an MMA sit in uniform registers.  With a single thread in a branch of
// its own, eight MMAs took 630 - 700 clk to issue beside the softmax warps (N = 64, d = 64: as long, though they execute in
// 380); now 320 - 380 (130 for the four of Q K^T at d = 64).  N = 7800: 96.3 -> 93.7 us, headline layer 838 -> 830 us
// (sustained), two-layer map 1203 -> 1176 us.
template <int D, int MAP, bool GEN, bool SH, bool KS = false>
__device__ __noinline__ uint32_t q_score_unit(const QParams& p, const QCtx& c, int u, uint32_t looks) {
  using R = QRing<D, SH>;
  constexpr uint32_t ID_QK = make_idesc(128, 128, 0, 0);      // S = Q K^T      (N = 128 keys)
  const int nkv = p.nkv, lin = p.lin;
  const R q(p, c, true);
  const uint32_t id_phi = make_idesc(128, D == 128 ? 128 : p.fcw, 0, 0);   // Phi_c = X W^T  (N = features of a chunk; 128 at d = 128)
  constexpr uint32_t ID_HID = make_idesc(128, D, 0, 0);       // hidden slice = Q W_1[j]^T (N = D hidden units)
  const int base = KS && p.part ? p.at_items : u * q.n_items, ps = KS && p.part ? p.at_s : u * q.n_s;   // first ring item / first score-column phase of the unit
  const int tail = KS && p.part ? p.at_tail : u;              // tails before the unit's
  const int ng = q_unit<KS>(p, u).ng;                             // groups at work on this unit (the last one of a group: ng - 1)
  uint64_t dq[2][8];                                          // the Q tiles do not move within a unit
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    const uint64_t q0 = kmajor_desc(q.sQ(g));
#pragma unroll
    for (int kk = 0; kk < 8; ++kk) dq[g][kk] = q0 + kstep_kmajor(kk);
  }
  auto s_free = [&](int g, int i) -> bool { return q.template s_free<MAP>(g, ps + i, ng, i, tail); };

  // ---- first key tile (its product opens the unit)
  if (nkv > 0) {
    for (int g = 0; g < ng; ++g) {
      if (!s_free(g, 0)) return Q_FAILED;
      if (g == 0 && !q.wait_full(R::B_KFULL, base, looks)) return Q_FAILED;
      if (!q.wait(R::B_Q0 + g, u)) return Q_FAILED;
      tc_fence_after();
      const uint64_t k0 = kmajor_desc(q.sKV(base));
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) mma_ss(q.tS(g), dq[g][kk], k0 + kstep_kmajor(kk), ID_QK, kk > 0 ? 1u : 0u);
        tc_commit(q.bar(R::B_S + g));
        if (g == ng - 1) q.release(base);
        if (nkv == 1 && !lin) tc_commit(q.bar(R::B_QF + g));
      }
    }
  }
  // ---- as soon as the groups have read their score rows: the next tile's Q K^T
  for (int j = 0; j + 1 < nkv; ++j) {
    const int ik = base + q.item_k(j + 1);
    const uint64_t k0 = kmajor_desc(q.sKV(ik));
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      if (g >= ng) break;
      if (g == 0 && !q.wait_full(R::B_KFULL, ik, looks)) return Q_FAILED;
      if (!s_free(g, j + 1)) return Q_FAILED;
      tc_fence_after();
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) mma_ss(q.tS(g), dq[g][kk], k0 + kstep_kmajor(kk), ID_QK, kk > 0 ? 1u : 0u);
        tc_commit(q.bar(R::B_S + g));
        if (j + 2 == nkv && !lin) tc_commit(q.bar(R::B_QF + g));   // the unit's last read of the Q tile
      }
    }
    if (elect_one()) q.release(ik);
  }
  if (!lin) return looks;

  // ---- linear tail: what lands in the score columns after the last key tile
  if constexpr (MAP != MAP_TWO) {
    // Phi_c = Q W[c]^T, one chunk of features after the other
    for (int ch = 0; ch < q.fc; ++ch) {
      const int iw = base + q.it_w(ch);
      const uint64_t w0 = kmajor_desc(q.sKV(iw));
      for (int g = 0; g < ng; ++g) {
        if (!s_free(g, nkv + ch)) return Q_FAILED;
        if (nkv == 0 && ch == 0 && !q.wait(R::B_Q0 + g, u)) return Q_FAILED;
        if (g == 0 && !q.wait_full(R::B_KFULL, iw, looks)) return Q_FAILED;
        tc_fence_after();
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk) mma_ss(q.template tTail<MAP>(g), dq[g][kk], w0 + kstep_kmajor(kk), id_phi, kk > 0 ? 1u : 0u);
          tc_commit(q.bar(R::B_S + g));
          if (ch == q.fc - 1) tc_commit(q.bar(R::B_QF + g));     // nothing of this unit reads the group's Q tile any more
        }
      }
      if (elect_one()) q.release(iw);
    }
    return looks;
  } else {
  // two layers: hidden slices first (A = Q), then Phi_c = sum_j h1_j W2[c, j]^T with the hidden slices read from
  // where the threads put them: slice 0 in the group's phi_q tile, slice 1 in its Q tile
  for (int j = 0; j < q.nh; ++j) {
    const int iw = base + q.it_w(j);
    const uint64_t w0 = kmajor_desc(q.sKV(iw));
    for (int g = 0; g < ng; ++g) {
      if (!s_free(g, nkv + j)) return Q_FAILED;
      if (nkv == 0 && j == 0 && !q.wait(R::B_Q0 + g, u)) return Q_FAILED;
      if (g == 0 && !q.wait_full(R::B_KFULL, iw, looks)) return Q_FAILED;
      tc_fence_after();
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) mma_ss(q.template tTail<MAP>(g), dq[g][kk], w0 + kstep_kmajor(kk), ID_HID, kk > 0 ? 1u : 0u);
        tc_commit(q.bar(R::B_S + g));
        if (q.nh == 1 && q.fc == 1) tc_commit(q.bar(R::B_QF + g));   // the Q tile is not reused as a buffer in this shape
      }
    }
    if (elect_one()) q.release(iw);
  }
  for (int ch = 0; ch < q.fc; ++ch) {
    for (int g = 0; g < ng; ++g) {
      if (!s_free(g, nkv + q.nh + ch)) return Q_FAILED;
      if (ch == 0 && !q.wait(R::B_H + g, tail)) return Q_FAILED;       // the group's hidden activations are in shared memory
      for (int j = 0; j < q.nh; ++j) {
        const int iw = base + q.it_w2(ch, j);
        const uint64_t w0 = kmajor_desc(q.sKV(iw));
        if (g == 0 && !q.wait_full(R::B_KFULL, iw, looks)) return Q_FAILED;
        tc_fence_after();
        const uint64_t a0 = kmajor_desc(j == 0 ? q.sP(g) : q.sQ(g));
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk)
            mma_ss(q.template tTail<MAP>(g), a0 + kstep_kmajor(kk), w0 + kstep_kmajor(kk), id_phi, (j > 0 || kk > 0) ? 1u : 0u);
          if (j == q.nh - 1) {
            tc_commit(q.bar(R::B_S + g));
            // two hidden slices, one feature chunk: this was the last read of the Q tile (as a buffer)
            if (q.nh == 2 && q.fc == 1) tc_commit(q.bar(R::B_QF + g));
          }
          if (g == ng - 1) q.release(iw);
        }
      }
    }
  }
  return looks;
  }
}

template <int D, int MAP, bool GEN, bool SH, bool KS = false>
__device__ __noinline__ uint32_t q_accum_unit(const QParams& p, const QCtx& c, int u, uint32_t looks) {
  using R = QRing<D, SH>;
  constexpr uint32_t ID_PV = make_idesc(128, D, 0, 1);        // O += P V and O += phi_q S  (V, S are MN-major)
  const int nkv = p.nkv, lin = p.lin;
  const R q(p, c, true);
  const int base = KS && p.part ? p.at_items : u * q.n_items, pp = KS && p.part ? p.at_p : u * q.n_p;   // first ring item / first P hand-over phase of the unit
  const int ng = q_unit<KS>(p, u).ng;
  for (int j = 0; j < nkv; ++j) {
    const bool last = (j + 1 == nkv);
    // as soon as P is there: O += P V
    const int iv = base + q.item_v(j);
    const uint64_t v0 = mnmajor_desc(q.sKV(iv));
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      if (g >= ng) break;
      if (g == 0 && !q.wait_full(R::B_VFULL, iv, looks)) return Q_FAILED;
      if (!q.wait(R::B_P + g, pp + j)) return Q_FAILED;
      tc_fence_after();
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) mma_ts(q.tO(g), q.tP(g) + kk * 8, v0 + kstep_mnmajor(kk), ID_PV, (j > 0 || kk > 0) ? 1u : 0u);
        tc_commit(q.bar(R::B_PF + g));
        if (last && !lin) tc_commit(q.bar(R::B_O + g));
        if (R::template own_tail<MAP> && last && lin && g == 1) tc_commit(q.bar(R::B_PL));    // (the other group's product was issued before)
      }
    }
    if (elect_one()) q.release(iv);
  }
  if (!lin) return looks;
  // O += phi_q,c S_c per feature chunk: phi_q sits in its tile (two layers, second chunk: in the Q tile),
  // S plays the part of a V tile
  const int ksteps = (D == 128 ? 128 : p.fcw) / 16;           // a constant at d = 128: the chains below unroll
  for (int ch = 0; ch < q.fc; ++ch) {
    const int is = base + q.it_st(ch);
    const uint64_t s0 = mnmajor_desc(q.sKV(is));
    const bool in_q_tile = MAP == MAP_TWO && ch == 1;
    for (int g = 0; g < ng; ++g) {
      if (g == 0 && !q.wait_full(R::B_VFULL, is, looks)) return Q_FAILED;
      if (!q.wait(R::B_P + g, pp + nkv + ch)) return Q_FAILED;
      tc_fence_after();
      const uint64_t a0 = kmajor_desc(in_q_tile ? q.sQ(g) : q.sP(g));
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < 8; ++kk)
          if (kk < ksteps) mma_ss(q.tO(g), a0 + kstep_kmajor(kk), s0 + kstep_mnmajor(kk), ID_PV, (nkv > 0 || ch > 0 || kk > 0) ? 1u : 0u);
        if (!in_q_tile) tc_commit(q.bar(R::B_PF + g));           // a reader of the phi_q tile has completed
        if (ch == q.fc - 1) {
          tc_commit(q.bar(R::B_O + g));
          if (in_q_tile) tc_commit(q.bar(R::B_QF + g));          // ... and the last reader of the Q tile
        }
      }
    }
    if (elect_one()) q.release(is);
  }
  return looks;
}

// ---------------------------------------------------------------- feature rows of the linear tail
// The biases of 32 columns as bf16 pairs, zeros without a bias; their loads (the same address in all lanes, or in half of them) go out together.
AS_DEV void q_ask_bias(const uint32_t* row, uint32_t (&w)[16]) {
#pragma unroll
  for (int i = 0; i < 16; ++i) w[i] = 0u;
  if (row == nullptr) return;
#pragma unroll
  for (int i = 0; i < 16; ++i) w[i] = __ldg(row + i);
}
AS_DEV void q_add_bias(const uint32_t (&w)[16], uint32_t (&x)[32]) {
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const float2 y = __fadd2_rn(make_float2(__uint_as_float(x[2 * i]), __uint_as_float(x[2 * i + 1])),
                                make_float2(__uint_as_float(w[i] << 16), __uint_as_float(w[i] & 0xffff0000u)));
    x[2 * i] = __float_as_uint(y.x);
    x[2 * i + 1] = __float_as_uint(y.y);
  }
}
// 32 columns of a thread's row (of its share, SPLIT as in q_ld32) with their biases added.  One thread per row has the registers to ask for the
// biases ahead of the columns (nothing stands between the columns' load and its wait); with two the other warps cover that latency, and the
// sums are left out where there is no bias.  Each bias behind the test of its pointer, one after the other, before; query stage with biases at
// N = 32760, 12 heads: two layers 128 / 128, no softmax tokens, one thread per row 132 -> 115 us, 8 key tiles 291 -> 277; whole layers at N = 7800,
// rate 1/8, two threads: 256 / 256 162 -> 158, one layer with F = 256 105.0 -> 104.6, with F = 128 and degree 4 87.6 -> 86.4.  (Asked for ahead with
// two threads per row, 8 at a time: the features' registers spill, degree 4 without a bias 1 % slower.)
template <int T, int SPLIT, bool GEN>
AS_DEV void q_ld32_biased(uint32_t t, const uint32_t* row, uint32_t (&x)[32], bool half_split = false) {
  uint32_t w[16];
  if (GEN && T == 1) q_ask_bias(row, w);
  if (half_split) q_ld32<T, SPLIT / 2>(t, x);
  else q_ld32<T, SPLIT>(t, x);
  tmem_ld_wait(x);
  if (GEN && T == 1) q_add_bias(w, x);
  if (GEN && T == 2 && row != nullptr) { q_ask_bias(row, w); q_add_bias(w, x); }
}

// A thread's share of a row of Phi (feature chunk ch) from the score columns -> bf16(lam * poly(relu(Phi + b))) -> row r of `tile` (the A operand
// of the apply product), 32 columns at a time (the loop is not unrolled: the tail runs once per unit, and on a CTA's first
// unit its instructions come from L2 line by line, so its size is its cost).  Arrives on `sf_bar` once the last columns
// are in registers.  Returns the share's part of phi_q.z, formed with the very bf16 values the MMA multiplies with S.
// GEN = false is the common case (no bias, polynomial degree <= 2).
template <int D, int T, bool GEN>
AS_DEV float q_features_from_tmem(const QParams& p, uint32_t tSg, uint32_t sf_bar, uint8_t* tile, int r, int hc, int bh, int ch, float lam) {
  const int fcw = D == 128 ? 128 : p.fcw, half = fcw / T;
  const int part = p.F / p.P;
  const float2* zrow = reinterpret_cast<const float2*>(p.z + (size_t)bh * p.F + ch * 128 + hc * half);
  const uint32_t* brow = nullptr;
  if (GEN && p.b2 != nullptr) brow = reinterpret_cast<const uint32_t*>(p.b2 + (size_t)(bh % p.H) * p.F + ch * 128 + hc * half);
  const float2 lam2 = make_float2(lam, lam);
  float2 dl2 = make_float2(0.f, 0.f);
  uint32_t x[32];
#pragma unroll 1
  for (int cc = 0; cc * 32 < half; ++cc) {
    q_ld32_biased<T, 64, GEN>(tSg + cc * 32, brow == nullptr ? nullptr : brow + cc * 16, x, D == 64 && fcw == 64);
    if (cc * 32 + 32 >= half) {
      tc_fence_before();
      mbar_arrive(sf_bar);                             // the next product into the score columns may follow
    }
    const int pw = min((ch * 128 + hc * half + cc * 32) / part, p.P - 1);     // 0-based part of these 32 features
    uint32_t wd[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const float2 a = make_float2(fmaxf(__uint_as_float(x[2 * i]), 0.f), fmaxf(__uint_as_float(x[2 * i + 1]), 0.f));
      float2 rr = a;
      if (pw >= 1) rr = __fmul2_rn(rr, a);
      if (GEN) {
        if (pw >= 2) rr = __fmul2_rn(rr, a);
        if (pw >= 3) rr = __fmul2_rn(rr, a);
      }
      rr = __fmul2_rn(rr, lam2);
      wd[i] = pack_bf16(rr.x, rr.y);
      const float2 zz = __ldg(zrow + cc * 16 + i);
      dl2 = __ffma2_rn(make_float2(__uint_as_float(wd[i] << 16), __uint_as_float(wd[i] & 0xffff0000u)), zz, dl2);
    }
    store_row_chunk(tile, r, hc * half + cc * 32, wd);
  }
  fence_proxy_async();
  return dl2.x + dl2.y;
}

// One-layer feature map, one unit and group: the feature chunks, one after the other.  Adds this thread's part of phi_q.z to dl;
// false: a wait ran out.
template <int D, int T, bool GEN>
AS_DEV bool q_one_layer_tail(const QParams& p, const QRing<D>& q, int g, uint32_t tSg, uint8_t* sPg, int r, int hc, int bh, int ps, int ppf, float lam,
                             float& dl) {
  using R = QRing<D>;
  const int nkv = p.nkv;
  for (int ch = 0; ch < q.fc; ++ch) {
    if (!q.wait(R::B_S + g, ps + nkv + ch)) return false;
    tc_fence_after();
    // the tile may be written once this warp's previous output store has been read out and the previous chunk's product has read it
    if ((threadIdx.x & 31) == 0) tma_store_wait_read();
    if (ch == 0) __syncwarp();
    else if (!q.wait(R::B_PF + g, ppf + nkv + ch - 1)) return false;
    dl += q_features_from_tmem<D, T, GEN>(p, tSg, q.bar(R::B_SF + g), sPg, r, hc, bh, ch, lam);   // the A operand of the apply product
    // not before every thread of the group has arrived for the last key tile
    if (ch == 0 && ppf + nkv > 0 && !q.wait(R::B_PF + g, ppf + nkv - 1)) return false;
    mbar_arrive(q.bar(R::B_P + g));
  }
  return true;
}

// The same out of line.  With a score row in a thread's registers, and the tail beside it, the key loop spills some of what it needs in every
// tile (81 frames at rate 1/8 717 us, full softmax 4840; with this 697 and 4675).  That is not all of it: q_softmax_unit<128, 1, ., .> still
// reloads 76 bytes (44 with biases) and stores 0 (8), as -Xptxas -v counts them.  With half a row (0 and 20) the call costs more than it gains (d = 64,
// 2142 keys 279 -> 290).
template <int D, int T, bool GEN>
__device__ __noinline__ bool q_one_layer_tail_apart(const QParams& p, const QCtx& c, int g, uint32_t tSg, uint8_t* sPg, int r, int hc, int bh, int ps, int ppf,
                                                    float lam, float& dl) {
  float sum = 0.f;
  const bool ok = q_one_layer_tail<D, T, GEN>(p, QRing<D>(p, c), g, tSg, sPg, r, hc, bh, ps, ppf, lam, sum);
  dl = sum;
  return ok;
}

// Two-layer feature map, one unit and group: hidden slices relu(Q W_1[j]^T + b_1) as bf16 (slice 0 into the phi_q tile,
// slice 1 into the Q tile, free once the product that made slice 1, the last reader of Q, has completed), then the
// feature chunks.  Returns phi_q.z, or -1 when a wait ran out.
template <int D, int T, bool GEN>
__device__ __noinline__ float q_two_layer_tail(const QParams& p, const QRing<D>& q, int g, uint32_t tSg, uint8_t* sPg, uint8_t* sQg, int r, int hc,
                                               int bh, int ps, int ppf, float lam) {
  using R = QRing<D>;
  constexpr int DC = D / T, FC = 128 / T;   // hidden units / features of a slice / chunk per thread
  const int nkv = p.nkv, h = bh % p.H, lane = threadIdx.x & 31;
  const __nv_bfloat16* b1 = (GEN && p.b1) ? p.b1 + (size_t)h * (q.nh * D) : nullptr;
  uint32_t x[32];
  for (int j = 0; j < q.nh; ++j) {
    if (!q.wait(R::B_S + g, ps + nkv + j)) return -1.f;
    tc_fence_after();
    if (j == 0) {                                    // this warp's output store of the previous unit has read its rows
      if (lane == 0) tma_store_wait_read();
      __syncwarp();
    }
    const uint32_t* brow = b1 ? reinterpret_cast<const uint32_t*>(b1 + j * D + hc * DC) : nullptr;
    uint8_t* tile = j == 0 ? sPg : sQg;
#pragma unroll
    for (int cc = 0; cc < DC / 32; ++cc) {
      q_ld32_biased<T, D / 2, GEN>(tSg + cc * 32, brow == nullptr ? nullptr : brow + cc * 16, x);
      uint32_t wd[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        wd[i] = pack_bf16(fmaxf(__uint_as_float(x[2 * i]), 0.f), fmaxf(__uint_as_float(x[2 * i + 1]), 0.f));
      }
      store_row_chunk(tile, r, hc * DC + cc * 32, wd);
    }
    tc_fence_before();
    mbar_arrive(q.bar(R::B_SF + g));
    fence_proxy_async();
    mbar_arrive(q.bar(R::B_H + g));
  }
  // (waits by parity look at every phase in turn)
  if (ppf + nkv > 0 && !q.wait(R::B_PF + g, ppf + nkv - 1)) return -1.f;
  // Feature chunks.  The hidden slices stay in their buffers until the last chunk's product has completed.
  if (!q.wait(R::B_S + g, ps + nkv + q.nh)) return -1.f;
  tc_fence_after();
  if (q.fc == 1) {                                   // Phi_0 is complete: nothing reads the slices any more
    const float dl = q_features_from_tmem<D, T, GEN>(p, tSg, q.bar(R::B_SF + g), sPg, r, hc, bh, 0, lam);
    mbar_arrive(q.bar(R::B_P + g));
    return dl;
  }
  // two chunks: chunk 0 is kept as bf16 pairs in registers until Phi_1 has landed (then the slices are free)
  float dl0 = 0.f, dl1 = 0.f;
  uint32_t pk[FC / 32][16];
  {
    const int part = p.F / p.P;
    const float2* zrow = reinterpret_cast<const float2*>(p.z + (size_t)bh * p.F + hc * FC);
    const uint32_t* brow = (GEN && p.b2) ? reinterpret_cast<const uint32_t*>(p.b2 + (size_t)h * p.F + hc * FC) : nullptr;
#pragma unroll
    for (int cc = 0; cc < FC / 32; ++cc) {
      q_ld32_biased<T, 64, GEN>(tSg + cc * 32, brow == nullptr ? nullptr : brow + cc * 16, x);
      const int pw = min((hc * FC + cc * 32) / part, p.P - 1);
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const float a0 = fmaxf(__uint_as_float(x[2 * i]), 0.f), a1 = fmaxf(__uint_as_float(x[2 * i + 1]), 0.f);
        float r0 = a0, r1 = a1;
        if (pw >= 1) { r0 *= a0; r1 *= a1; }
        if (pw >= 2) { r0 *= a0; r1 *= a1; }
        if (pw >= 3) { r0 *= a0; r1 *= a1; }
        const uint32_t wv = pack_bf16(r0 * lam, r1 * lam);
        pk[cc][i] = wv;
        const float2 zz = __ldg(zrow + cc * 16 + i);
        dl0 = fmaf(__uint_as_float(wv << 16), zz.x, dl0);
        dl1 = fmaf(__uint_as_float(wv & 0xffff0000u), zz.y, dl1);
      }
    }
    tc_fence_before();
    mbar_arrive(q.bar(R::B_SF + g));                 // Phi_1 may overwrite the score columns
  }
  if (!q.wait(R::B_S + g, ps + nkv + q.nh + 1)) return -1.f;     // Phi_1 is there: nothing reads the hidden slices any more
  tc_fence_after();
#pragma unroll
  for (int cc = 0; cc < FC / 32; ++cc) store_row_chunk(sPg, r, hc * FC + cc * 32, pk[cc]);
  fence_proxy_async();
  mbar_arrive(q.bar(R::B_P + g));
  const float dlb = q_features_from_tmem<D, T, GEN>(p, tSg, q.bar(R::B_SF + g), sQg, r, hc, bh, 1, lam);
  // not before every thread of the group has arrived for the first chunk
  if (!q.wait(R::B_PF + g, ppf + nkv)) return -1.f;
  mbar_arrive(q.bar(R::B_P + g));
  return (dl0 + dl1) + dlb;
}

// ---------------------------------------------------------------- key loops in parts
// What a CTA leaves of a unit whose key loop another one finishes: per group O (fp32, unnormalised, [4 columns][row][4]: a warp's lanes are neighbours), then of
// each row the reference maximum, the true one and the sum.
template <int D>
struct QPart {
  static constexpr int O = 128 * D, GROUP = O + 128 * 4, TOTAL = 2 * GROUP;    // floats
  AS_DEV static float4* of(const QParams& p, int cta, int g) { return reinterpret_cast<float4*>(p.parts + (size_t)cta * TOTAL + (size_t)g * GROUP); }
};

// By the threads of a group, whose last product into O has completed.  Every warp has a flag of its own and the warp of that index of the other CTA, with the
// same rows, waits for that alone: where a wait runs out its warp leaves, and no other one is waiting for it at a barrier that has no limit.
template <int D, int T>
__device__ __noinline__ void q_leave_part(const QParams& p, uint32_t tOg, int g, int r, int hc, float m_ref, float m_true, float l) {
  static_assert(8 * T <= AS_PART_FLAGS);
  float4* to = QPart<D>::of(p, p.cta, g);
#pragma unroll 1
  for (int o = 0; o < D / T; o += 16) {
    uint32_t y[16];
    q_ld16<T, D / 2>(tOg + o, y);
    tmem_ld16_wait(y);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      to[((hc * (D / T) + o) / 4 + i) * 128 + r] = make_float4(__uint_as_float(y[4 * i]), __uint_as_float(y[4 * i + 1]), __uint_as_float(y[4 * i + 2]),
                                                                __uint_as_float(y[4 * i + 3]));
  }
  if (hc == 0) to[QPart<D>::O / 4 + r] = make_float4(m_ref, m_true, l, 0.f);
  __syncwarp();
  if ((threadIdx.x & 31) == 0)                                 // (what the warp's lanes have stored goes with it)
    asm volatile("st.release.gpu.global.u32 [%0], 1;" ::"l"(p.part_flags + AS_PART_FLAGS * p.cta + (threadIdx.x >> 5)) : "memory");
}

// Where a part that weighs nothing against another one had a sum that is no number or past the end of the range (`bad`: in this thread's row).  Values near the end of the
// range, many of them, are one cause: their sum is left out, as each of them would be in an unbroken key loop.  The other is a value that is infinite or no
// number itself: 0 times that is no number there, and so it is here, in its column.  By a whole warp; on ordinary input never.
template <int D, int T>
__device__ __noinline__ void q_weightless(const QParams& p, uint32_t tOg, int hc, bool bad) {
  const int lane = threadIdx.x & 31;
  const uint16_t* v = reinterpret_cast<const uint16_t*>(p.v) + (size_t)p.bh * p.v_rows * D;
  uint32_t mine = 0u;                                          // bit i: column lane + 32 i has such a value
  for (int k = 0; k < p.v_rows; ++k)
#pragma unroll
    for (int i = 0; i < D / 32; ++i) mine |= (v[(size_t)k * D + i * 32 + lane] & 0x7f80u) == 0x7f80u ? 1u << i : 0u;
#pragma unroll 1
  for (int o = 0; o < D / T; o += 16) {
    uint32_t y[16];
    q_ld16<T, D / 2>(tOg + o, y);
    tmem_ld16_wait(y);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      bool there[T];
#pragma unroll
      for (int h = 0; h < T; ++h) {                            // (every lane asks for the columns of either share)
        const int col = h * (D / T) + o + i;
        there[h] = (__shfl_sync(0xffffffffu, mine, col & 31) >> (col / 32) & 1u) != 0u;
      }
      if (bad && there[T == 1 ? 0 : hc] && fabsf(__uint_as_float(y[i])) < INFINITY) y[i] = 0x7fc00000u;
    }
    q_st16<T, D / 2>(tOg + o, y);
  }
  tmem_st_wait();
}

// Adds to O, and to the row's maxima and sum, what the p.merges CTAs right before this one have left.  A CTA's index is the order in which it has started (see
// the kernel), so those are running or through, and their parts that are left come first in them and wait for nothing: the wait ends whatever else is on the GPU, in
// whatever order CTAs are started (and is bounded like every other).  Returns (m_ref, m_true, l); the sum is negative when a wait ran out.
template <int D, int T>
__device__ __noinline__ float4 q_merge_parts(const QParams& p, const WaitCtx& wc, uint32_t tOg, int g, int r, int hc, float m_ref, float m_true, float l) {
  constexpr int STEP = 32, N = STEP / 4;                       // columns and loads at once
  for (int n = 1; n <= p.merges; ++n) {
    const int cta = p.cta - n;
    uint32_t* flag = p.part_flags + AS_PART_FLAGS * cta + (threadIdx.x >> 5);
    bool ok = true;
    if ((threadIdx.x & 31) == 0) {
      uint32_t there, it = 0;
      long long t0 = 0;
      while (true) {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(there) : "l"(flag) : "memory");
        if (there != 0u) break;
        if ((++it & 15u) != 0u) continue;
        const long long now = clock64();
        if (t0 == 0) t0 = now;
        if (*wc.abort != 0u || now - t0 > kWaitLimitCycles) { *wc.abort = 1u; atomicOr(wc.status, 1u); ok = false; break; }
      }
    }
    if (!__all_sync(0xffffffffu, ok)) return make_float4(0.f, 0.f, -1.f, 0.f);
    if ((threadIdx.x & 31) == 0) *reinterpret_cast<volatile uint32_t*>(flag) = 0u;   // nobody else looks at it before the next launch
    __syncwarp();                                              // (the lanes' loads come behind lane 0's)
    const float4* from = QPart<D>::of(p, cta, g);
    const float4* mine_from = from + hc * (D / T / 4) * 128 + r;
    const float4 st = __ldcg(from + QPart<D>::O / 4 + r);
    float4 x[N];
#pragma unroll
    for (int i = 0; i < N; ++i) x[i] = __ldcg(mine_from + i * 128);
    const float m = fmaxf(m_ref, st.x), mine = ex2(m_ref - m), theirs = ex2(st.x - m);
    const bool weightless = !(mine > 0.f) || !(theirs > 0.f);
    float odd = 0.f;                                           // no number if a weightless sum is past the end of the range or none
#pragma unroll 1
    for (int o = 0; o < D / T; o += STEP) {
      uint32_t y[32];
      q_ld32<T, D / 2>(tOg + o, y);
      tmem_ld_wait(y);
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const float part[4] = {x[i].x, x[i].y, x[i].z, x[i].w};
        if (weightless)
#pragma unroll
          for (int e = 0; e < 4; ++e) odd = fmaf(part[e], 0.f, fmaf(__uint_as_float(y[4 * i + e]), 0.f, odd));
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          // a sum that weighs nothing is left out, also where it is past the end of the range (cf. q_weightless)
          const float own = mine > 0.f ? __uint_as_float(y[4 * i + e]) * mine : 0.f;
          y[4 * i + e] = __float_as_uint(theirs > 0.f ? fmaf(part[e], theirs, own) : own);
        }
      }
      if (o + STEP < D / T) {
#pragma unroll
        for (int i = 0; i < N; ++i) x[i] = __ldcg(mine_from + ((o + STEP) / 4 + i) * 128);
      }
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        uint32_t z[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) z[i] = y[16 * half + i];
        q_st16<T, D / 2>(tOg + o + 16 * half, z);
      }
    }
    tmem_st_wait();
    if (__any_sync(0xffffffffu, odd != odd)) q_weightless<D, T>(p, tOg, hc, odd != odd);
    l = l * mine + st.z * theirs;
    m_true = fmaxf(m_true, st.y);
    m_ref = m;
  }
  tc_fence_before();
  return make_float4(m_ref, m_true, l, 0.f);
}

// ---------------------------------------------------------------- softmax / merge group, one unit
template <int D, int T, int MAP, bool GEN, bool KS = false>
__device__ __noinline__ bool q_softmax_unit(const QParams& p, const QCtx& c, const CUtensorMap* tmO, uint8_t* smem, int u) {
  using R = QRing<D>;
  using L = QLayout<D>;
  using X = QShape<T>;
  const int nkv = p.nkv, n_s = p.n_s;
  const float scale_log2 = p.scale_log2;
  const R q(p, c);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = (warp >> 2) & 1;                    // group 0 or 1
  const int r0 = (warp & 3) * 32 + (T == 2 ? (warp >> 3) * 16 : 0);   // this warp's rows of the group's 128-row tile
  const int r = r0 + (T == 2 ? lane & 15 : lane), hc = T == 2 ? lane >> 4 : 0;   // this thread's row, its share of the columns
  const uint32_t lane_off = (uint32_t)r0 << 16;
  const uint32_t tSg = q.tS(g) + lane_off, tOg = q.tO(g) + lane_off, tPg = q.tP(g) + lane_off;
  uint8_t* sPg = smem + L::P_OFF + g * L::PTILE;    // this group's phi_q / output staging tile
  const int ps = KS && p.part ? p.at_s : u * q.n_s, ppf = KS && p.part ? p.at_pf : u * q.n_pf;   // first phases of the unit (cf. QRing)
  // (a part behind a unit's first starts from a finite maximum: keys with scores of -infinity weigh nothing, as they do behind others in an unbroken key loop)
  float m_ref = KS ? (p.key0 > 0 ? -3.402823466e38f : -INFINITY) : 0.f, m_true = -INFINITY, l = 0.f;

  for (int j = 0; j < nkv; ++j) {
    if (!q.wait(R::B_S + g, ps + j)) return false;
    tc_fence_after();
    uint32_t sv[X::COLS];                           // this thread's share of its row of the 128 x 128 score tile
    if constexpr (T == 1) tmem_ld128_sync(tSg, sv); else tmem_ldh64_sync<64>(tSg, sv);
    tc_fence_before();
    mbar_arrive(q.bar(R::B_SF + g));                // the score columns may be overwritten
    if (n_s - j * 128 < 128) {
      const int valid = n_s - j * 128 - hc * X::COLS;   // this thread's keys of the tile that exist
#pragma unroll
      for (int i = 0; i < X::COLS; ++i) sv[i] = (i < valid) ? sv[i] : 0xff800000u;   // -inf: exp2 gives 0
    }
    float mx0 = fmax3(__uint_as_float(sv[0]), __uint_as_float(sv[1]), __uint_as_float(sv[2]));
    float mx1 = fmax3(__uint_as_float(sv[3]), __uint_as_float(sv[4]), __uint_as_float(sv[5]));
#pragma unroll
    for (int i = 6; i + 3 < X::COLS; i += 4) {
      mx0 = fmax3(mx0, __uint_as_float(sv[i]), __uint_as_float(sv[i + 1]));
      mx1 = fmax3(mx1, __uint_as_float(sv[i + 2]), __uint_as_float(sv[i + 3]));
    }
    float mx = fmax3(mx0, mx1, fmaxf(__uint_as_float(sv[X::COLS - 2]), __uint_as_float(sv[X::COLS - 1])));
    if (T == 2) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 16));   // the other half of the row
    mx *= scale_log2;
    m_true = fmaxf(m_true, mx);
    // The reference maximum only moves when the row maximum grew by more than 2^8; then O and l
    // are rescaled (once the previous tile's P V has completed, before this tile's P is handed over).
    const bool need = (j > 0) && (mx > m_ref + RESCALE_THRESHOLD);
    const float resc = need ? ex2(m_ref - mx) : 1.f;
    if (j == 0 || need) m_ref = KS ? fmaxf(mx, m_ref) : mx;
    // P = exp2(s * scale_log2 - m_ref) as bf16 into the group's columns of tensor memory
    const float neg_m = -m_ref;
    // packed fp32x2 arithmetic halves the instruction count of the scaling and of the row sum
    const float2 scale2 = make_float2(scale_log2, scale_log2), negm2 = make_float2(neg_m, neg_m);
    float2 la = make_float2(0.f, 0.f), lb = make_float2(0.f, 0.f);
    // Whether the previous tile's P V has completed is asked here and looked at behind the first exponentials (d = 128: a wait for
    // something that is already there costs a round trip; at d = 64 the other warps cover it)
    bool p_free = false;
    if (T == 1 && ppf + j > 0) p_free = mbar_try_wait(q.bar(R::B_PF + g), (ppf + j - 1) & 1);
#pragma unroll
    for (int cc = 0; cc < X::COLS / 32; ++cc) {
      uint32_t pw[16];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int k = cc * 32 + 4 * i;
        const float2 xa = __ffma2_rn(make_float2(__uint_as_float(sv[k]), __uint_as_float(sv[k + 1])), scale2, negm2);
        const float2 xb = __ffma2_rn(make_float2(__uint_as_float(sv[k + 2]), __uint_as_float(sv[k + 3])), scale2, negm2);
        const float2 pa = make_float2(ex2(xa.x), ex2(xa.y));
        const float2 pc = ex2_second_pair<T>(i, xb);
        la = __fadd2_rn(la, pa);
        lb = __fadd2_rn(lb, pc);
        pw[2 * i] = pack_bf16(pa.x, pa.y);
        pw[2 * i + 1] = pack_bf16(pc.x, pc.y);
      }
      if (cc == 0) {                                // the previous tile's P V has read the columns of P
        if (ppf + j > 0 && (T == 2 || !__all_sync(0xffffffffu, p_free)) && !q.wait(R::B_PF + g, ppf + j - 1)) return false;
        tc_fence_after();
        if (__any_sync(0xffffffffu, need)) {        // ... and left its sum in O, which no product touches until this tile's P is handed over
#pragma unroll 1
          for (int o = 0; o < D / T; o += 16) {
            uint32_t y[16];
            q_ld16<T, D / 2>(tOg + o, y);
            tmem_ld16_wait(y);
#pragma unroll
            for (int i = 0; i < 16; ++i) y[i] = __float_as_uint(__uint_as_float(y[i]) * resc);
            q_st16<T, D / 2>(tOg + o, y);
          }
        }
      }
      q_st16<T, 32>(tPg + cc * 16, pw);
    }
    // The sum above adds the unrounded probabilities while the MMA multiplies their bf16 roundings with V.
    // Over many keys the rounding errors average out, but the error of a probability that dominates its
    // row does not, and a result close to one large v_j would be off by up to 2^-9 of its value.  So the
    // sum takes over the rounding error of the tile's largest probability.
    const float p_top = ex2(mx - m_ref);
    const float p_top_err = __uint_as_float(pack_bf16(0.f, p_top) & 0xffff0000u) - p_top;
    l = l * resc + (((la.x + la.y) + (lb.x + lb.y)) + (T == 1 || hc == 0 ? p_top_err : 0.f));
    tmem_st_wait();
    tc_fence_before();
    mbar_arrive(q.bar(R::B_P + g));
  }

  const QUnit un = q_unit<KS>(p, u);
  const int bh = un.bh;
  if (T == 2) l += __shfl_xor_sync(0xffffffffu, l, 16);
  if constexpr (KS) {
    if (p.leaves) {
      if (!q.wait(R::B_O + g, u)) return false;
      tc_fence_after();
      q_leave_part<D, T>(p, tOg, g, r, hc, m_ref, m_true, l);
      tc_fence_before();
      return true;
    }
    if (p.merges > 0) {
      if (!q.wait(R::B_PF + g, ppf + nkv - 1)) return false;   // the last P V has completed (looked at once more in the tail)
      tc_fence_after();
      const float4 sum = q_merge_parts<D, T>(p, c.wc, tOg, g, r, hc, m_ref, m_true, l);
      if (sum.z < 0.f) return false;
      m_ref = sum.x; m_true = sum.y; l = sum.z;
    }
  }
  const int row = un.row0 + g * 128 + r;
  float den = l, den_l_out = 0.f;
  if (p.lin) {
    // per-row factor applied to phi_q so that the linear branch lands on the scale of O and l
    float e = 0.f;
    if (nkv > 0) e = (p.stab_mode == AS_STAB_EXACT) ? -m_ref : (m_true - m_ref);
    e = fminf(fmaxf(e, -100.f), 100.f);
    const float lam = ex2(e);
    float dl = 0.f;
    const uint32_t tTail = q.template tTail<MAP>(g) + lane_off;
    if constexpr (MAP != MAP_TWO) {
      const bool ok = T == 1 ? q_one_layer_tail_apart<D, T, GEN>(p, c, g, tTail, sPg, r, hc, bh, ps, ppf, lam, dl)
                             : q_one_layer_tail<D, T, GEN>(p, q, g, tTail, sPg, r, hc, bh, ps, ppf, lam, dl);
      if (!ok) return false;
    } else {
      uint8_t* sQg = smem + L::Q_OFF + g * L::TILE;    // the group's Q tile: a second buffer once Q is done with
      dl = q_two_layer_tail<D, T, GEN>(p, q, g, tTail, sPg, sQg, r, hc, bh, ps, ppf, lam);
      if (dl < 0.f) return false;                      // a wait ran out (the sum itself is never negative)
    }
    if (T == 2) dl += __shfl_xor_sync(0xffffffffu, dl, 16);
    den = l + dl;
    den_l_out = dl / lam;
  }
  if (!q.wait(R::B_O + g, u)) return false;
  tc_fence_after();
  const float inv = 1.f / den;
  // The output rows are staged in the group's phi_q tile (the product that read it has completed with the O
  // barrier; a layer without linear tokens: this warp's previous output store has been read out); each warp stores its own rows (rows past N are clipped by the tensor map).
  const int wrow0 = un.row0 + g * 128 + r0;
  if (!p.lin) {
    if (lane == 0) tma_store_wait_read();
    __syncwarp();
  }
  uint32_t x[32];
#pragma unroll 1
  for (int cc = 0; cc < D / T / 32; ++cc) {
    q_ld32<T, D / 2>(tOg + cc * 32, x);
    tmem_ld_wait(x);
    uint32_t wd[16];
#pragma unroll
    for (int i = 0; i < 16; ++i)
      wd[i] = pack_bf16(__uint_as_float(x[2 * i]) * inv, __uint_as_float(x[2 * i + 1]) * inv);
    store_row_chunk(sPg, r, hc * (D / T) + cc * 32, wd);
  }
  fence_proxy_async();
  __syncwarp();
  if (lane == 0 && wrow0 < p.N) {
#pragma unroll
    for (int b = 0; b < D / 64; ++b)
      tma_store_3d(tmO, smem_u32(sPg) + b * BOX_BYTES + r0 * 128, b * 64, wrow0, bh);
    tma_store_commit();
  }
  if (p.aux != nullptr && row < p.N && hc == 0) {
    const float ln2 = 0.6931471805599453f;
    float* ap = p.aux + ((size_t)bh * p.N + row) * 3;
    ap[0] = nkv > 0 ? m_true * ln2 : 0.f;
    ap[1] = nkv > 0 ? l * ex2(m_ref - m_true) : 0.f;
    ap[2] = den_l_out;
  }
  // The next unit's first P V overwrites O: every tcgen05.ld above has completed (tmem_ld_wait), and
  // the arrive on the P barrier that releases that MMA follows in program order.
  tc_fence_before();
  return true;
}

// ---------------------------------------------------------------- layers without softmax tokens (rate 0)
// With no key loop a unit is: Phi = Q W^T, phi_q, O = phi_q S, y = O / (phi_q . z), store.  The tensor pipe has
// little to do and the kernel is bound by how fast the threads turn rows around, so this variant of the kernel runs
// SIXTEEN compute warps: each 128-row group is worked on by two warps per TMEM lane quadrant, each taking one half of
// the columns of a row (features on the way in, output columns on the way out).  Producer and issuing warps are the
// ones of the general kernel; a row's two threads add their shares of phi_q . z through shared memory.
constexpr int QL_THREADS = 608;          // warps 0-15: compute (group = bit 2, quadrant = bits 0-1, column half = bit 3);
                                         // warp 16: TMA; warps 17, 18: MMA issuers

template <int D, bool GEN>
__device__ __noinline__ bool q_linear_unit(const QParams& p, const QCtx& c, const CUtensorMap* tmO, uint8_t* smem, float* sDl, int u) {
  using R = QRing<D, false>;
  using L = QLayout<D>;
  const R q(p, c);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = (warp >> 2) & 1, quad = warp & 3, hf = warp >> 3;
  const int r = quad * 32 + lane;                   // row inside the group's 128-row tile
  const uint32_t lane_off = (uint32_t)(quad * 32) << 16;
  const uint32_t tSg = q.tS(g) + lane_off, tOg = q.tO(g) + lane_off;
  uint8_t* sPg = smem + L::P_OFF + g * L::PTILE;    // phi_q, then the output rows
  float* dl_slot = sDl + g * 128 + r;
  const int ps = u * q.n_s, ppf = u * q.n_pf;
  const int fcw = D == 128 ? 128 : p.fcw;           // width of a feature chunk; this thread takes columns [hf, hf + 1) * half
  const int half = fcw / 2;
  const QUnit un = q_unit(p, u);
  const int bh = un.bh, row = un.row0 + g * 128 + r;
  const int part = p.F / p.P;
  uint32_t x[32];
  float dl = 0.f;
  bool ok = true;                                   // a warp whose wait has run out still comes to the group's barriers, which have no limit
  for (int ch = 0; ch < q.fc; ++ch) {
    ok = ok && q.wait(R::B_S + g, ps + ch);
    tc_fence_after();
    // the phi_q tile may be written once the product that read it has completed and the previous unit's output store
    // has been read out (the stores are issued by the warps of column half 0)
    if (hf == 0 && lane == 0) tma_store_wait_read();
    if (ppf + ch > 0) ok = ok && q.wait(R::B_PF + g, ppf + ch - 1);
    named_barrier_sync(1 + g, 256);
    const float2* zrow = reinterpret_cast<const float2*>(p.z + (size_t)bh * p.F + ch * 128 + hf * half);
    const uint32_t* brow = nullptr;
    if (GEN && p.b2 != nullptr) brow = reinterpret_cast<const uint32_t*>(p.b2 + (size_t)(bh % p.H) * p.F + ch * 128 + hf * half);
    float dl0 = 0.f, dl1 = 0.f;
#pragma unroll
    for (int cc = 0; cc < 2; ++cc) {
      if (cc * 32 < half) {
        const int col = hf * half + cc * 32;
        tmem_ld32(tSg + col, x);
        tmem_ld_wait(x);
        const int pw = min((ch * 128 + col) / part, p.P - 1);
        uint32_t wd[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          float a0 = __uint_as_float(x[2 * i]), a1 = __uint_as_float(x[2 * i + 1]);
          if (GEN && brow != nullptr) {
            const uint32_t bb = __ldg(brow + cc * 16 + i);
            a0 += __uint_as_float(bb << 16);
            a1 += __uint_as_float(bb & 0xffff0000u);
          }
          a0 = fmaxf(a0, 0.f); a1 = fmaxf(a1, 0.f);
          float r0 = a0, r1 = a1;
          if (pw >= 1) { r0 *= a0; r1 *= a1; }
          if (GEN) {
            if (pw >= 2) { r0 *= a0; r1 *= a1; }
            if (pw >= 3) { r0 *= a0; r1 *= a1; }
          }
          wd[i] = pack_bf16(r0, r1);
          const float2 zz = __ldg(zrow + cc * 16 + i);
          dl0 = fmaf(__uint_as_float(wd[i] << 16), zz.x, dl0);
          dl1 = fmaf(__uint_as_float(wd[i] & 0xffff0000u), zz.y, dl1);
        }
        store_row_chunk(sPg, r, col, wd);
      }
    }
    dl += dl0 + dl1;
    tc_fence_before();
    mbar_arrive(q.bar(R::B_SF + g));                 // the next product into the score columns may follow
    fence_proxy_async();
    mbar_arrive(q.bar(R::B_P + g));
  }
  // the row's denominator: both column halves' shares of phi_q . z
  if (hf == 1) *dl_slot = dl;
  named_barrier_sync(1 + g, 256);
  if (hf == 0) dl += *dl_slot;
  named_barrier_sync(1 + g, 256);
  if (hf == 0) *dl_slot = dl;
  ok = ok && q.wait(R::B_O + g, u);                  // (the products run meanwhile)
  named_barrier_sync(1 + g, 256);
  const float den = *dl_slot;
  tc_fence_after();
  const float inv = 1.f / den;
  const int ohalf = D / 2;                           // output columns per thread
#pragma unroll
  for (int cc = 0; cc < 2; ++cc) {
    if (cc * 32 < ohalf) {
      const int col = hf * ohalf + cc * 32;
      tmem_ld32(tOg + col, x);
      tmem_ld_wait(x);
      uint32_t wd[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) wd[i] = pack_bf16(__uint_as_float(x[2 * i]) * inv, __uint_as_float(x[2 * i + 1]) * inv);
      store_row_chunk(sPg, r, col, wd);
    }
  }
  fence_proxy_async();
  tc_fence_before();
  named_barrier_sync(1 + g, 256);                    // both halves of every row are staged
  if (!ok) return false;
  const int wrow0 = row - lane;
  if (hf == 0 && lane == 0 && wrow0 < p.N) {
#pragma unroll
    for (int b = 0; b < D / 64; ++b)
      tma_store_3d(tmO, smem_u32(sPg) + b * BOX_BYTES + quad * 32 * 128, b * 64, wrow0, bh);
    tma_store_commit();
  }
  if (hf == 0 && p.aux != nullptr && row < p.N) {
    float* ap = p.aux + ((size_t)bh * p.N + row) * 3;
    ap[0] = 0.f; ap[1] = 0.f; ap[2] = den;
  }
  return true;
}

template <int D, bool GEN>
__global__ void __launch_bounds__(QL_THREADS, 1)
qlin_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmW,
            const __grid_constant__ CUtensorMap tmSt, const __grid_constant__ CUtensorMap tmO, const __grid_constant__ QParams p) {
  using L = QLayout<D>;
  using R = QRing<D>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t sbase = smem_u32(smem);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::BAR_OFF + 8 * R::B_COUNT);
  volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem + L::BAR_OFF + 8 * R::B_COUNT + 4);
  auto bar = [&](int i) { return sbase + L::BAR_OFF + 8 * i; };
  const int warp = threadIdx.x >> 5;
  __shared__ float sDl[2 * 128];                     // per group and row: share of phi_q . z, then the denominator

  if (threadIdx.x == 0) {
    *abort_flag = 0u;
    mbar_init(bar(R::B_Q0), 1); mbar_init(bar(R::B_Q0 + 1), 1); mbar_init(bar(R::B_LATE), 1);
    for (int s = 0; s < KV_STAGES; ++s) { mbar_init(bar(R::B_KFULL + s), 1); mbar_init(bar(R::B_VFULL + s), 1); mbar_init(bar(R::B_EMPTY + s), 1); }
    for (int g = 0; g < 2; ++g) {
      mbar_init(bar(R::B_S + g), 1); mbar_init(bar(R::B_SF + g), 256); mbar_init(bar(R::B_P + g), 256);
      mbar_init(bar(R::B_PF + g), 1); mbar_init(bar(R::B_O + g), 1); mbar_init(bar(R::B_QF + g), 1);
      mbar_init(bar(R::B_H + g), 128);
    }
    fence_barrier_init();
    fence_proxy_async();
  }
  __shared__ uint32_t s_skip;
  if (threadIdx.x == 32) s_skip = status_now(p.status);   // (ahead of the wait: behind the first copies it would wait for these)
  if (warp == 17) { tmem_alloc(smem_u32(tmem_slot), 512); tmem_relinquish(); griddep_launch(); }
  if (warp == 16 && (threadIdx.x & 31) == 0) { tma_prefetch_desc(&tmQ); tma_prefetch_desc(&tmW); tma_prefetch_desc(&tmSt); tma_prefetch_desc(&tmO); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const QCtx c{sbase, *tmem_slot, WaitCtx{p.status, abort_flag}};
  const int n_mine = q_units_of_cta(p);
  griddep_wait();                                    // the set-up above ran beside the kernel before this one
  if (s_skip != 0u) {                                // an earlier launch timed out: do nothing (decided once per CTA)
    if (warp == 17) tmem_dealloc(c.tmem, 512);
    return;
  }

  if (threadIdx.x == 18 * 32) status_again(sbase + L::LATE_OFF, p.status, bar(R::B_LATE));

  if (warp == 16) {
    if ((threadIdx.x & 31) == 0) q_first_loads<D, MAP_ONE>(p, c, q_unit(p, 0), &tmQ, &tmQ, &tmW, &tmW);
    __syncwarp();
    for (int u = 0; u < n_mine; ++u)
      if (!q_produce_unit<D, MAP_ONE, GEN>(p, c, &tmQ, &tmQ, &tmQ, &tmW, &tmSt, &tmW, u)) break;
  } else if (warp == 17) {
    uint32_t looks = 0u;
    for (int u = 0; u < n_mine && looks != Q_FAILED; ++u) looks = q_score_unit<D, MAP_ONE, GEN, false>(p, c, u, looks);
  } else if (warp == 18) {
    uint32_t looks = 0u;
    for (int u = 0; u < n_mine && looks != Q_FAILED; ++u) looks = q_accum_unit<D, MAP_ONE, GEN, false>(p, c, u, looks);
  } else {
    const int g = (warp >> 2) & 1;
    // a unit worked on by one group only is the CTA's last one: group 1 stops before it
    const int n_grp = (n_mine > p.n_rounds && g == 1 && q_unit(p, p.n_rounds).ng == 1) ? p.n_rounds : n_mine;
    // not where the launch before has timed out behind the set-up's look at the status word
    const bool start = __all_sync(0xffffffffu, status_clear(bar(R::B_LATE), sbase + L::LATE_OFF));
    if (!start) status_give_up(c.wc);
    for (int u = 0; start && u < n_grp; ++u)
      if (!q_linear_unit<D, GEN>(p, c, &tmO, smem, sDl, u)) break;
    if ((threadIdx.x & 31) == 0) tma_store_wait_read();
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 17) {
    tc_fence_after();
    tmem_dealloc(c.tmem, 512);
  }
}

// The parts of CTA c in the last round (see as_deal_parts), each as the parameters of a unit.  Written by one thread.
AS_DEV int q_parts(const QParams& p, int c, QParams* to) {
  AsPart part[2];
  const int n = (int)gridDim.x, np = as_deal_parts(p.n_pairs, p.n_rounds, p.share, p.nkv, p.lin, p.fc, p.layers == 2 ? p.nh : 0, n, c, part);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    if (i >= np) break;
    const AsPart& a = part[i];
    QParams& q = to[i];
    const int w = p.n_rounds * n + a.unit;
    q = p;
    q.part = 1; q.cta = c;
    q.bh = w / p.nx; q.row0 = (w % p.nx) * 256; q.key0 = a.k0 * 128;
    q.nkv = a.k1 - a.k0; q.n_s = p.n_s - q.key0;
    q.leaves = a.leaves; q.merges = a.merges;
    q.lin = a.leaves ? 0 : p.lin;
    q.at_items = a.at_items; q.at_s = a.at_s; q.at_p = a.at_p; q.at_pf = a.at_pf; q.at_tail = a.at_tail;
  }
  return np;
}

template <int D, int T, int MAP, bool GEN, bool KS = false>
__global__ void __launch_bounds__(QShape<T>::THREADS, 1)
qpass_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
             const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmW,
             const __grid_constant__ CUtensorMap tmSt, const __grid_constant__ CUtensorMap tmW1,
             const __grid_constant__ CUtensorMap tmO, const __grid_constant__ QParams p) {
  using L = QLayout<D>;
  using R = QRing<D>;
  using X = QShape<T>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t sbase = smem_u32(smem);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::BAR_OFF + 8 * R::B_COUNT);
  volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem + L::BAR_OFF + 8 * R::B_COUNT + 4);
  auto bar = [&](int i) { return sbase + L::BAR_OFF + 8 * i; };
  const int warp = threadIdx.x >> 5;

  if (threadIdx.x == 0) {
    *abort_flag = 0u;
    mbar_init(bar(R::B_Q0), 1); mbar_init(bar(R::B_Q0 + 1), 1); mbar_init(bar(R::B_LATE), 1);
    for (int s = 0; s < KV_STAGES; ++s) { mbar_init(bar(R::B_KFULL + s), 1); mbar_init(bar(R::B_VFULL + s), 1); mbar_init(bar(R::B_EMPTY + s), 1); }
    for (int g = 0; g < 2; ++g) {
      mbar_init(bar(R::B_S + g), 1); mbar_init(bar(R::B_SF + g), X::GROUP); mbar_init(bar(R::B_P + g), X::GROUP);
      mbar_init(bar(R::B_PF + g), 1); mbar_init(bar(R::B_O + g), 1); mbar_init(bar(R::B_QF + g), 1);
      mbar_init(bar(R::B_H + g), X::GROUP * (p.nh > 0 ? p.nh : 1));   // one arrival per thread and hidden slice
    }
    mbar_init(bar(R::B_PL), 1);
    fence_barrier_init();
    fence_proxy_async();
  }
  __shared__ uint32_t s_skip;
  __shared__ QParams s_part[KS ? 2 : 1];
  __shared__ int s_parts;
  if (threadIdx.x == 32) s_skip = status_now(p.status);   // (ahead of the wait: behind the first copies it would wait for these)
  // The CTA's index in the last round is the order in which it has started, by a counter that goes back to 0 with the launch's last CTA.  Ahead of the wait for the kernel
  // before, and of griddep_launch: a later launch starts when all CTAs of this one have come past that, and so have taken theirs.
  if (KS && threadIdx.x == X::W_SCORE * 32) s_parts = q_parts(p, (int)atomicInc(p.part_ticket, gridDim.x - 1u), s_part);
  if (warp == X::W_SCORE) { tmem_alloc(smem_u32(tmem_slot), 512); tmem_relinquish(); griddep_launch(); }
  if (warp == X::W_TMA && (threadIdx.x & 31) == 0) { tma_prefetch_desc(&tmQ); tma_prefetch_desc(&tmK); tma_prefetch_desc(&tmV); tma_prefetch_desc(&tmO); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  griddep_wait();                                    // the set-up above ran beside the kernel before this one
  if (s_skip != 0u) {                                // an earlier launch timed out: do nothing (decided once per CTA)
    if (warp == X::W_SCORE) tmem_dealloc(*tmem_slot, 512);
    return;
  }
  const QCtx c{sbase, *tmem_slot, WaitCtx{p.status, abort_flag}};
  const int n_mine = KS ? p.n_rounds + s_parts : q_units_of_cta(p);   // units of this CTA
  auto of = [&](int u) -> const QParams& { return KS && u >= p.n_rounds ? s_part[KS ? u - p.n_rounds : 0] : p; };

  if (threadIdx.x == X::W_ACCUM * 32) status_again(sbase + L::LATE_OFF, p.status, bar(R::B_LATE));

  if (warp == X::W_TMA) {
    if ((threadIdx.x & 31) == 0) q_first_loads<D, MAP, KS>(of(0), c, q_unit<KS>(of(0), 0), &tmQ, &tmK, &tmW, &tmW1);
    __syncwarp();
    for (int u = 0; u < n_mine; ++u)
      if (!q_produce_unit<D, MAP, GEN, KS>(of(u), c, &tmQ, &tmK, &tmV, &tmW, &tmSt, &tmW1, u)) break;
  } else if (warp == X::W_SCORE) {
    uint32_t looks = 0u;
    for (int u = 0; u < n_mine && looks != Q_FAILED; ++u) looks = q_score_unit<D, MAP, GEN, D == 128, KS>(of(u), c, u, looks);
  } else if (warp == X::W_ACCUM) {
    uint32_t looks = 0u;
    for (int u = 0; u < n_mine && looks != Q_FAILED; ++u) looks = q_accum_unit<D, MAP, GEN, D == 128, KS>(of(u), c, u, looks);
  } else {
    // a unit worked on by one group only is the CTA's last one: group 1 stops before it
    const int n_grp = (!KS && n_mine > p.n_rounds && ((warp >> 2) & 1) == 1 && q_unit(p, p.n_rounds).ng == 1) ? p.n_rounds : n_mine;
    // not where the launch before has timed out behind the set-up's look at the status word
    const bool start = __all_sync(0xffffffffu, status_clear(bar(R::B_LATE), sbase + L::LATE_OFF));
    if (!start) status_give_up(c.wc);
    for (int u = 0; start && u < n_grp; ++u)
      if (!q_softmax_unit<D, T, MAP, GEN, KS>(of(u), c, &tmO, smem, u)) break;
    if ((threadIdx.x & 31) == 0) tma_store_wait_read();  // this warp's output stores have read their rows (the writes land by the end of the kernel)
  }

  // ------------------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  if (warp == X::W_SCORE) {
    tc_fence_after();
    tmem_dealloc(c.tmem, 512);
  }
}

}  // namespace

cudaError_t as_tensor_init_qpass() {
  cudaError_t e;
#define AS_OPT_IN_Q(D_, T_, MAP_) \
  if ((e = opt_in_smem(qpass_kernel<D_, T_, MAP_, false>, QLayout<D_>::TOTAL)) != cudaSuccess) return e; \
  if ((e = opt_in_smem(qpass_kernel<D_, T_, MAP_, true>, QLayout<D_>::TOTAL)) != cudaSuccess) return e
#define AS_OPT_IN_QP(D_, T_, MAP_) \
  if ((e = opt_in_smem(qpass_kernel<D_, T_, MAP_, false, true>, QLayout<D_>::TOTAL)) != cudaSuccess) return e; \
  if ((e = opt_in_smem(qpass_kernel<D_, T_, MAP_, true, true>, QLayout<D_>::TOTAL)) != cudaSuccess) return e
  AS_OPT_IN_Q(128, 1, MAP_ONE); AS_OPT_IN_Q(128, 1, MAP_WIDE); AS_OPT_IN_Q(128, 1, MAP_TWO);
  AS_OPT_IN_Q(128, 2, MAP_ONE); AS_OPT_IN_Q(128, 2, MAP_WIDE); AS_OPT_IN_Q(128, 2, MAP_TWO);
  AS_OPT_IN_Q(64, 2, MAP_ONE); AS_OPT_IN_Q(64, 2, MAP_TWO);
  AS_OPT_IN_QP(128, 1, MAP_ONE); AS_OPT_IN_QP(128, 1, MAP_WIDE); AS_OPT_IN_QP(128, 1, MAP_TWO); AS_OPT_IN_QP(64, 2, MAP_ONE); AS_OPT_IN_QP(64, 2, MAP_TWO);
#undef AS_OPT_IN_Q
#undef AS_OPT_IN_QP
  if ((e = opt_in_smem(qlin_kernel<128, false>, QLayout<128>::TOTAL)) != cudaSuccess) return e;
  if ((e = opt_in_smem(qlin_kernel<128, true>, QLayout<128>::TOTAL)) != cudaSuccess) return e;
  if ((e = opt_in_smem(qlin_kernel<64, false>, QLayout<64>::TOTAL)) != cudaSuccess) return e;
  if ((e = opt_in_smem(qlin_kernel<64, true>, QLayout<64>::TOTAL)) != cudaSuccess) return e;
  return cudaSuccess;
}

size_t as_qpass_parts_bytes(int N, int BH, int d, int sms) {
  AsUnits p;
  as_plan_units(p, N, BH, sms);
  const int pairs = ((N + 127) / 128 + 1) / 2 * BH, rounds = pairs / sms;
  const double now = p.n_rounds + (p.split_last ? (p.n_pairs > p.n_rounds * sms || p.n_single > 0 ? 0.62 : 0.) : p.n_pairs > p.n_rounds * sms ? 1. : 0.);
  if (pairs == rounds * sms || (double)pairs / sms > 0.96 * now) return 0;   // what as_plan_parts says of a key loop without an end
  return sizeof(float) * (size_t)(d == 128 ? QPart<128>::TOTAL : QPart<64>::TOTAL) * sms;
}

cudaError_t as_tensor_qpass(const as_launch_args& a, cudaStream_t st) {
  if (as_tensor_qstream_handles(a)) return as_tensor_qstream(a, st);   // no softmax tokens, the common feature map
  const int BH = a.B * a.H;
  const bool lin = a.n_l > 0;
  CUtensorMap tmQ, tmK, tmV, tmW, tmSt, tmW1, tmO;
  const bool two = lin && a.layers == 2;
  const bool qlin = a.n_s == 0 && lin && !two;         // no softmax tokens, one-layer map: the variant without a key loop
  QParams p{};
  p.layers = lin ? a.layers : 1;
  p.N = a.N; p.n_s = a.n_s; p.nkv = (a.n_s + 127) / 128; p.lin = lin ? 1 : 0; p.stab_mode = a.stab_mode; p.P = a.P;
  p.H = a.H;
  p.F = a.F; p.fc = (a.F + 127) / 128; p.fcw = a.F < 128 ? a.F : 128;
  p.nh = two ? a.hid / a.d : 0;
  p.b1 = two ? a.bq1 : nullptr;
  p.b2 = two ? a.bq2 : a.bq1;
  p.scale_log2 = a.scale * 1.4426950408889634f;
  p.z = a.z; p.aux = a.aux; p.status = a.status;
  // persistent: one CTA per SM (the kernel's shared memory and its 512 TMEM columns allow no second one)
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
    return cudaErrorInvalidValue;
  // the general kernels carry the bias and the powers beyond 2; the common case does without them
  const bool gen = lin && (a.P > 2 || p.b1 != nullptr || p.b2 != nullptr);
  const AsLoop loop{a.d, p.nkv, p.lin, p.fc, p.nh, gen ? 1 : 0};
  AsUnits plan;
  dim3 grid(as_plan_units(plan, a.N, BH, sms), 1, 1);
  const int ctas = a.parts != nullptr && !qlin ? as_plan_parts(plan, loop, a.N, BH, sms) : 0;
  const bool ks = ctas > 0;
  if (ks) grid.x = ctas;
  p.nx = plan.nx; p.n_pairs = plan.n_pairs; p.n_single = plan.n_single; p.n_rounds = plan.n_rounds; p.split_last = plan.split_last; p.share = plan.share;
  p.v = a.vs; p.v_rows = a.n_s;
  p.parts = a.parts; p.part_flags = a.part_flags; p.part_ticket = a.part_flags + AS_PART_FLAGS * sms;
  const int tpr = as_threads_per_row(plan, loop);
  // the output is stored warp by warp: boxes of a warp's rows
  if (!make_map(&tmQ, a.q, a.d, a.N, BH, 128) || !make_map(&tmO, a.out, a.d, a.N, BH, qlin ? 32 : 32 / tpr)) return cudaErrorInvalidValue;
  if (a.n_s > 0) {
    if (!make_map(&tmK, a.ks, a.d, a.n_s, BH, 128) || !make_map(&tmV, a.vs, a.d, a.n_s, BH, 128)) return cudaErrorInvalidValue;
  } else {
    tmK = tmQ; tmV = tmQ;       // never used: the key loop is empty
  }
  if (lin) {
    // boxes are always 128 rows: rows past F (or the hidden width) are out of bounds and arrive as zeros.
    // tmW: last-layer weights [H][F][width of their input]; tmW1: first-layer weights of a two-layer map.
    if (!make_map(&tmW, two ? a.wq2 : a.wq, two ? a.hid : a.d, a.F, a.H, 128) || !make_map(&tmSt, a.Sb, a.d, a.F, BH, 128))
      return cudaErrorInvalidValue;
  } else {
    tmW = tmQ; tmSt = tmQ;      // never used: no linear branch at rate 1
  }
  if (two) { if (!make_map(&tmW1, a.wq, a.d, a.hid, a.H, 128)) return cudaErrorInvalidValue; }
  else tmW1 = tmQ;            // never used with a one-layer map
  if (qlin) {
#define AS_LAUNCH_QL(D_, GEN_) \
  return as_launch_dependent(qlin_kernel<D_, GEN_>, grid, dim3(QL_THREADS), QLayout<D_>::TOTAL, st, tmQ, tmW, tmSt, tmO, p)
    if (a.d == 128) { if (gen) AS_LAUNCH_QL(128, true); else AS_LAUNCH_QL(128, false); }
    if (gen) AS_LAUNCH_QL(64, true); else AS_LAUNCH_QL(64, false);
#undef AS_LAUNCH_QL
  }
#define AS_LAUNCH_Q(...) \
  return as_launch_dependent(qpass_kernel<__VA_ARGS__>, grid, dim3(threads), smem, st, tmQ, tmK, tmV, tmW, tmSt, tmW1, tmO, p)
#define AS_LAUNCH_QG(D_, T_, MAP_) \
  do { \
    const int threads = QShape<T_>::THREADS, smem = QLayout<D_>::TOTAL; \
    if (gen) AS_LAUNCH_Q(D_, T_, MAP_, true); else AS_LAUNCH_Q(D_, T_, MAP_, false); \
  } while (0)
#define AS_LAUNCH_QP(D_, T_, MAP_) \
  do { \
    const int threads = QShape<T_>::THREADS, smem = QLayout<D_>::TOTAL; \
    if (gen) AS_LAUNCH_Q(D_, T_, MAP_, true, true); else AS_LAUNCH_Q(D_, T_, MAP_, false, true); \
  } while (0)
  const int map = two ? MAP_TWO : lin && p.fc > 1 && !as_one_tile_each(plan) ? MAP_WIDE : MAP_ONE;
  if (ks) {
    if (a.d == 64) { if (two) AS_LAUNCH_QP(64, 2, MAP_TWO); else AS_LAUNCH_QP(64, 2, MAP_ONE); }
    if (map == MAP_TWO) AS_LAUNCH_QP(128, 1, MAP_TWO);
    if (map == MAP_WIDE) AS_LAUNCH_QP(128, 1, MAP_WIDE); else AS_LAUNCH_QP(128, 1, MAP_ONE);
  }
#define AS_LAUNCH_QT(T_) \
  do { \
    if (map == MAP_TWO) AS_LAUNCH_QG(128, T_, MAP_TWO); else if (map == MAP_WIDE) AS_LAUNCH_QG(128, T_, MAP_WIDE); else AS_LAUNCH_QG(128, T_, MAP_ONE); \
  } while (0)
  if (a.d == 128) { if (tpr == 2) AS_LAUNCH_QT(2); else AS_LAUNCH_QT(1); }
  if (two) AS_LAUNCH_QG(64, 2, MAP_TWO); else AS_LAUNCH_QG(64, 2, MAP_ONE);
#undef AS_LAUNCH_Q
#undef AS_LAUNCH_QG
#undef AS_LAUNCH_QP
#undef AS_LAUNCH_QT
}
