// k_ascent.cu -- PerformSteepestAscent of Fig. 2, batched: every listed start
// is climbed by 1-bit flips, always taking the flip of largest gain (lowest
// index on ties) while the gain is positive.  Gains are the 1-flip move values
// of Glover et al. (2002) that the Pseudocode section cites,
//     Delta_j = Q_jj + 2 (1 - 2 x_j) y_j,   y = Q x,
// and a flip of bit k (d = 1 - 2 x_k before the flip) changes y by d times
// column k of Q (= row k, Q being symmetric) and negates the sign of x_k.
//
// Design.  A group of T threads owns one start at a time (one warp, or one
// block of several).  Thread g owns E = 16*C elements, in chunks of 16
// consecutive indices: element e lives at j = (e/16)*16T + 16g + e%16, so one
// move loads row k of the int8 Q (= column k, Q being symmetric) with C fully
// coalesced 16-byte loads per thread.  Per element the thread keeps, in
// registers,
//     key_j = 32 Delta_j + (31 - e%32)   and   sel_j = +-64 in j's byte lane,
// the sign of sel_j being (1 - 2 x_j) d for the move at hand.  A move is then,
// per element, one dp4a (key += 64 (1 - 2 x_j) d q_kj) and half a three-way
// max: no y is kept, and no multiply-add forms the key.  When d changes sign
// from one move to the next the selectors are flipped (one XOR each, about
// every other move).  Measured against y, S and C registers with a dp4a, a
// multiply-add and half a max per element (3 registers, 2.5 instructions):
// 2 registers, so more starts fit an SM, and about 2 instructions, the ALU
// pipe (XOR, max) and the FMA pipe (dp4a) sharing them.  The key orders by
// gain, then by lower index inside the thread (up to 32 elements; larger
// threads keep one maximum per 32); across threads the group reduces (gain,
// 2j + x) with warp max/min reductions (redux.sync), so every thread learns k,
// x_k and Delta_k.  The thread owning k resets key_k to -Delta_k, turns sel_k
// and flips its x bit; it takes q_kk from a copy of the diagonal in shared
// memory, so that nothing but the update itself waits for the row (with q_kk
// taken from the row the owner's branches came after the load: n = 7000, 2172
// starts 6.53 -> 5.24 ms, 54 starts 1.70 -> 1.64).  Rows are read from L2 (the
// int8 Q of one instance, e.g. 49 MB at n = 7000, stays resident there); nothing
// per move goes to HBM.
//
// What bounds it.  With few starts the chain of moves is latency-bound: per
// move a dependent L2 row fetch, the update and a block-wide reduction (n =
// 7000, 54 starts: 737 cycles per move, 1.58 ms; 863 and 1.85 with y, S and C
// registers).  The loads of the row are issued before anything else of the
// move, its end test included; the selectors' flip and the owner's branches run
// in their shadow.  Relinking, climbs above n = 8192 and the unpacked batch climb's
// short lists take the fetch off the chain where the move was predicted: every
// move also copies the row of the reduction's runner-up into shared memory, and
// the next move is that row about 40% of the time at n = 7000.  The other climbs
// make no such copies: they cost more per move than the hits save.
// With many starts the issue slots and the latency of 12 to 20 warps bound it
// (n = 1400, 6069 starts: about 185 warp instructions per move, 91 cycles per
// move and SM, 0.63 ms; 199 cycles and 1.38 ms with y, S and C registers).
// launch_ascent_shaped picks the group shape by n and count.
//
// Start-up: y = Q x of every listed start comes from the tensor-core product of
// the ascent workspace when given (exact integers in fp32), else each group
// sums the rows k with x_k = 1 on the CUDA cores.
#include "ascent_core.cuh"

namespace ubqp {

cudaError_t launch_relink(const ubqp_q* h, const uint64_t* X, const int64_t* f, const uint64_t* G,
                          int64_t P, uint64_t* Xb, int64_t* fb, int32_t* dist, uint16_t* trace,
                          int64_t ldt, const float* Y, unsigned long long* next,
                          cudaStream_t st) {
  const int n = h->n;
  if (next) {
    cudaError_t e = cudaMemsetAsync(next, 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
  }
  // P is known here: up to one pair per SM the registers are sized for one
  // block per SM (the shortest chain), above it for two, so that 256 pairs are one
  // wave and not two (n = 4500, 256 pairs 674 us with y, S and C registers and one
  // block per SM, 432 now; 150 pairs 394 and 342)
  const bool wide = P > h->sm_count;
#define UBQP_RL(TT, CC, OCC) \
  return launch_relink_block<TT, CC, OCC>(h, X, f, G, P, Xb, fb, dist, trace, ldt, Y, next, st)
  if (n <= 512) return launch_relink_warp<1>(h, X, f, G, P, Xb, fb, dist, trace, ldt, Y, next, st);
  if (n <= 1024) UBQP_RL(64, 1, 4);
  if (n <= 2048) UBQP_RL(128, 1, 3);
  if (n <= 2560) UBQP_RL(160, 1, 3);
  if (n <= 4096) UBQP_RL(128, 2, 2);
  if (n <= 5120) {
    if (wide) UBQP_RL(160, 2, 2);
    UBQP_RL(160, 2, 1);
  }
  if (n <= 7168) {
    if (wide) UBQP_RL(224, 2, 2);
    UBQP_RL(224, 2, 1);
  }
  if (n <= 8192) {
    if (wide) UBQP_RL(256, 2, 2);
    UBQP_RL(256, 2, 1);
  }
  if (n <= 16384) UBQP_RL(512, 2, 1);
#undef UBQP_RL
  return cudaErrorInvalidValue;
}

bool ascent_batch_supported(int T, int C) {
  return (T == 64 || T == 128 || T == 256 || T == 512) && (C == 1 || C == 2);
}

// The unpacked climb of a batch: one shape for every instance.  Without
// runner-up copies: with them, the threads of a group that is wider than an
// instance's rows copied the same 16 bytes, one request to one L2 slice each (30
// instances n = 64 to 400, 1024 starts, 256 x 1: 14.5 ms per run, 0.67 without
// copies), and a full chip gains from dropping them in any case (the same in 64
// x 1, 0.49 -> 0.25; 8 of n = 3000 in 256 x 1, 4.51 -> 3.36).  Where the rows fill
// three quarters of a group of 128 threads or more (filled) and there is no more
// than one start per SM, the copies still hide part of the row fetch (8 of n =
// 3000, 100 random starts each, about 50 climbed: 757 us with copies, 824 without;
// 2 of n = 8000: 2370, 2515; but one of n = 9000 in 512 x 2, 0.56 filled: 3049,
// 2827): those counts keep a launch with copies.
cudaError_t launch_ascent_batch(const BatchDesc* d, const int2* items, const int64_t* n_items,
                                int T, int C, bool filled, int64_t most, int32_t max_flips,
                                int sm_count, unsigned long long* next, cudaStream_t st) {
  if (next) {
    cudaError_t e = cudaMemsetAsync(next, 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
  }
  auto pair = [&](auto few, auto many) {
    cudaError_t e = filled ? few(0, sm_count) : cudaSuccess;
    if (e == cudaSuccess && (!filled || most > sm_count))
      e = many(filled ? sm_count + 1 : 0, INT64_MAX);
    return e;
  };
#define UBQP_BT(TT, CC, RR, OCC)                                                                \
  [&](int64_t lo, int64_t hi) {                                                                 \
    return launch_batch_shape<TT, CC, RR, OCC>(d, items, n_items, max_flips, next, most, lo,    \
                                               hi, sm_count, st);                               \
  }
#define UBQP_PAIR(TT, CC, OCC) \
  if (T == TT && C == CC) return pair(UBQP_BT(TT, CC, 1, 1), UBQP_BT(TT, CC, 0, OCC));
  if (T == 64 && C == 1) return UBQP_BT(64, 1, 0, 10)(0, INT64_MAX);
  if (T == 64 && C == 2) return UBQP_BT(64, 2, 0, 8)(0, INT64_MAX);
  UBQP_PAIR(128, 1, 5) UBQP_PAIR(128, 2, 4) UBQP_PAIR(256, 1, 3) UBQP_PAIR(256, 2, 2)
  UBQP_PAIR(512, 1, 1) UBQP_PAIR(512, 2, 1)
#undef UBQP_PAIR
#undef UBQP_BT
  return cudaErrorInvalidValue;
}

bool ascent_packed_supported(int T, int C) { return T == 256 && (C == 1 || C == 2); }

// One size class of a packed batch, in the group shapes launch_ascent_shaped
// uses for lists of that length: with at most 10 starts per SM in the whole
// batch the ones with the shorter chains, else the fewest warps that hold n.
// Packed climbs ran before as one launch of 256-thread blocks split into
// sub-groups on named barriers, the classes one after another in each block;
// a kernel per class keeps each class's registers to what its n needs (C = 2:
// 20 warps per SM, C = 4: 12), and the classes' launches share the chip on
// streams of their own (32 instances n ~ U[200, 2500], 1024 starts each:
// 4.38 -> 3.42 ms per run, 6.58 with y, S, C registers; 2.61 now).
cudaError_t launch_ascent_batch_packed(const BatchDesc* d, const int2* items, const int4* ranges,
                                       int cls, const int64_t* n_items, int64_t most,
                                       int64_t batch_most, int32_t max_flips, int sm_count,
                                       unsigned long long* next, cudaStream_t st) {
  const int64_t full = 10ll * sm_count;
  auto both = [&](auto mid, auto all) {
    cudaError_t e = mid(0, full);
    if (e == cudaSuccess && batch_most > full) e = all(full + 1, INT64_MAX);
    return e;
  };
#define UBQP_PK(TT, CC, RR, OCC)                                                              \
  [&](int64_t lo, int64_t hi) {                                                               \
    return launch_class<TT, CC, RR, OCC>(d, items, ranges, cls, n_items, max_flips, next,     \
                                         most, lo, hi, sm_count, st);                         \
  }
  switch (cls) {
    case 0: return both(UBQP_PK(32, 1, 0, 8), UBQP_PK(32, 1, 0, 10));
    case 1: return both(UBQP_PK(64, 1, 0, 8), UBQP_PK(32, 2, 0, 8));
    case 2: return both(UBQP_PK(96, 1, 0, 7), UBQP_PK(32, 3, 0, 6));
    case 3: return both(UBQP_PK(128, 1, 0, 4), UBQP_PK(32, 4, 0, 5));
    case 4: return both(UBQP_PK(96, 2, 0, 4), UBQP_PK(32, 5, 0, 4));
    case 5: return both(UBQP_PK(96, 2, 0, 4), UBQP_PK(64, 3, 0, 7));
    case 6: return both(UBQP_PK(128, 2, 0, 4), UBQP_PK(64, 4, 0, 5));
  }
#undef UBQP_PK
  return cudaErrorInvalidValue;
}

cudaError_t launch_ascent(const ubqp_q* h, uint64_t* X, int64_t* f, const int32_t* idx,
                          const int64_t* count, int64_t S, int32_t max_flips, int32_t* flips,
                          const float* Y, unsigned long long* next, cudaStream_t st,
                          bool next_zeroed) {
  return launch_ascent_shaped<false>(h, X, f, idx, count, S, max_flips, flips, Y, next, nullptr,
                                     0, st, next_zeroed);
}

}  // namespace ubqp
