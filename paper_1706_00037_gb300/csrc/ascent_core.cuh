// ascent_core.cuh -- the move machinery of the batched steepest ascent and of
// path relinking (kernels and launch helpers), shared by k_ascent.cu and
// k_ascent_trace.cu.  Internal to libubqp.  The design is described at the
// top of k_ascent.cu.
#pragma once
#include <algorithm>
#include <climits>

#include "ubqp_internal.cuh"

namespace ubqp {
namespace {

constexpr int64_t kTimeoutNs = 20ll * 1000 * 1000 * 1000;  // per start
// Runner-up rows that relinking copies one move ahead.  One against none, us, with
// the present flip and reduction: one pair n = 1000 149 / 169, n = 4500 397 / 484,
// n = 7500 640 / 793; 100 pairs 125 / 121, 342 / 334, 541 / 516; 256 pairs 128 / 127,
// 432 / 383, 759 / 630.  So the copies pay while few blocks run, and a rule by the
// number of pairs would gain above about one pair per SM.  (Climbs above n = 8192,
// one against none: n = 9000, 11 starts 3245 / 2972, 544 starts 5382 / 4640; n =
// 16384, 21 starts 6355 / 6895, 547 starts 10438 / 10255.)
constexpr int kSpecRows = 1;
// Starts per block of the one-warp kernels.
constexpr int kWarps = 2;
// shared-memory slots (16 bytes each) of a group of T threads: two buffers of
// R rows x C chunks per thread, laid out thread-minor
template <int T, int C, int R>
constexpr int spec_slot_count() {
  return R > 0 ? T * 2 * R * C : 1;
}

__device__ __forceinline__ uint64_t globaltimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// The R best entries (gain r.x, tag r.y) held one per lane across a warp,
// excluding the entry tagged `first`: their tags in decreasing order of gain
// (ties to the lower lane), INT_MAX where fewer entries remain.  One max
// reduction per rank on gain * 32 + (31 - lane) (|gain| < 2^26), then one
// shuffle per rank for the tags.
template <int R>
__device__ __forceinline__ void runners_up(int2 r, int first, int* cand) {
  const int lane = threadIdx.x & 31;
  int key = (r.y == first || r.y == INT_MAX) ? INT_MIN : r.x * 32 + (31 - lane);
  int wl[R];
  bool ok[R];
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int m = __reduce_max_sync(0xffffffffu, key);
    ok[i] = m != INT_MIN;
    wl[i] = 31 - (m & 31);
    if (lane == wl[i]) key = INT_MIN;
  }
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int t = __shfl_sync(0xffffffffu, r.y, wl[i]);
    cand[i] = ok[i] ? t : INT_MAX;
  }
}

// Keys.  Element e of a thread keeps key = 32 gain + (31 - e % 32), so that an
// integer maximum over up to 32 keys orders by gain, then by lower index
// (|gain| < 2^23, so |key| < 2^28).  An element that is no candidate (beyond n,
// or in relinking one that has been flipped or need not be) has kOutKey, and row
// updates move that too, since every element of a thread takes them.  Over any
// number of moves they add up to little: the element's own bit does not change
// and its selector changes sign only with d, so the sum is +-64 times the change
// of y = Q x in the column that it reads (column off + e of every row, for chunks
// beyond the row the same first ones throughout), and y stays within 2^21, so
// the key within 2^28 of kOutKey: it never reaches a real key.
constexpr int kKeyBits = 5;
constexpr int kOutKey = -(1 << 30);
// Below every real key and above every kOutKey: a thread without candidates
// enters the reduction with it, and in the block-wide one, 2^2 times as large,
// it still fits.
constexpr int kFloorKey = -(1 << 28);

// The flip of the owned element ek, found by a binary decision on its local
// index (about log2(E) branches instead of E predicated operations): its key
// becomes that of the gain -gain (relinking: it leaves the candidates) with
// the element's own term of the row update that follows, -2 q_kk, taken off
// beforehand; its selector changes sign and its x bit flips.  q_kk comes from
// shared memory, not from the row, so the flip does not wait for the row.
// The decisions depend on ek alone, which the whole group knows: every lane of
// the owner's warp takes the same path and only the writes are the owner's
// (own).  Taken by the owner alone, each level was a divergent branch of its own:
// climbs of n = 500, 398 starts 79.1 -> 73.5 us; 2500, 3213 starts 1153 -> 1057;
// 4000, 2193 starts 1824 -> 1679.
template <int LO, int HI, int E, bool RL>
__device__ __forceinline__ void flip_tree(int (&key)[E], uint32_t (&sel)[E],
                                          uint32_t (&xm)[(E + 31) / 32], int ek, int v, bool own) {
  if constexpr (HI - LO == 1) {
    if (own) key[LO] = RL ? kOutKey : v + (31 - (LO & 31));
    sel[LO] ^= own ? 0x80u << (8 * (LO & 3)) : 0u;
    xm[LO >> 5] ^= own ? 1u << (LO & 31) : 0u;
  } else {
    constexpr int MID = (LO + HI) / 2;
    if (ek < MID) flip_tree<LO, MID, E, RL>(key, sel, xm, ek, v, own);
    else flip_tree<MID, HI, E, RL>(key, sel, xm, ek, v, own);
  }
}

template <int T>
struct Group;

// One warp per start.
template <>
struct Group<32> {
  __device__ __forceinline__ int rank() const { return threadIdx.x & 31; }
  int2 mine;  // this lane's entry of the last reduction
  // returns {max gain, 2k + x_k} over the group
  template <int CB>
  __device__ __forceinline__ int2 reduce(int rank, int jx) {
    const int gain = rank >> CB;
    const int m = __reduce_max_sync(0xffffffffu, gain);
    const int c = __reduce_min_sync(0xffffffffu, gain == m ? jx : INT_MAX);
    mine = make_int2(gain, jx);
    return make_int2(m, c);
  }
  // runners-up of the last reduction among the lanes' own maxima
  template <int R>
  __device__ __forceinline__ void runners(int first, int* cand) const {
    runners_up<R>(mine, first, cand);
  }
  __device__ __forceinline__ bool any(bool p) { return __any_sync(0xffffffffu, p); }
  __device__ __forceinline__ void sync() { __syncwarp(); }
  __device__ __forceinline__ int sum(int v) { return __reduce_add_sync(0xffffffffu, v); }
};

// One block per start.
template <int T>
struct Group {
  static constexpr int NW = T / 32;
  int2 (*rec)[NW];  // [2][NW] shared
  int parity;
  __device__ __forceinline__ int rank() const { return threadIdx.x; }
  int2 mine;  // warp `lane`'s winner in the last reduction
  // returns {max gain, 2k + x_k} over the group.  rank orders the threads'
  // entries by gain, then by chunk (2^CB gain + the chunks above the entry's),
  // and within a chunk a lower lane has the lower index, so one maximum of
  // {rank, 31 - lane} finds the warp's first winner, which writes its own entry.
  // (With a second reduction for the index, climbs of n = 1025, 510 starts: 136.2
  // -> 132.6 us; 2500, 542: 352.2 -> 348.7; 7000, 641: 2617 -> 2573.)
  template <int CB>
  __device__ __forceinline__ int2 reduce(int rank, int jx) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int key = (rank << 5) | (31 - lane);
    // predicated, not a branch: divergence costs more than the store
    asm volatile(
        "{\n .reg .pred p;\n setp.eq.s32 p, %0, %1;\n @p st.shared.v2.s32 [%2], {%3, %4};\n}\n" ::"r"(
            key),
        "r"(__reduce_max_sync(0xffffffffu, key)),
        "r"((uint32_t)__cvta_generic_to_shared(&rec[parity][warp])), "r"(rank), "r"(jx)
        : "memory");
    __syncthreads();
    const int2 r = lane < NW ? rec[parity][lane] : make_int2(INT_MIN, INT_MAX);
    const int m2 = __reduce_max_sync(0xffffffffu, r.x);
    const int c2 = __reduce_min_sync(0xffffffffu, r.x == m2 ? r.y : INT_MAX);
    parity ^= 1;
    mine = r;
    return make_int2(m2 >> CB, c2);
  }
  // runners-up of the last reduction among the warps' winners
  template <int R>
  __device__ __forceinline__ void runners(int first, int* cand) const {
    runners_up<R>(mine, first, cand);
  }
  __device__ __forceinline__ bool any(bool p) { return __syncthreads_or(p) != 0; }
  __device__ __forceinline__ void sync() { __syncthreads(); }
  __device__ __forceinline__ int sum(int v) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int s = __reduce_add_sync(0xffffffffu, v);
    if (lane == 0) rec[parity][warp] = make_int2(s, 0);
    __syncthreads();
    const int r = lane < NW ? rec[parity][lane].x : 0;
    parity ^= 1;
    return __reduce_add_sync(0xffffffffu, r);
  }
};

// Path relinking of one pair (see relink_block_kernel): the guiding solution,
// the outputs and a trace of the flipped indices (n entries of scratch).
struct RelinkArgs {
  const uint64_t* g;
  uint64_t* x_best;
  int64_t* f_best;
  int32_t* dist;
  uint16_t* trace;
  uint64_t* xs;  // W words of shared memory
};

// RL = false: steepest ascent of x_g in place (f_s updated, flips to flips_s).
// RL = true: path relinking from x_g (read only, value *f_s) toward rl->g --
// the same move machinery, but only variables where x and g differ are
// candidates, every step is taken whatever its gain, a flipped variable leaves
// the candidate set, and the best solution strictly between the endpoints is
// the result.  diag: T C slots of shared memory for the diagonal (RL: unused).
template <int T, int C, int R, bool RL = false, bool TR = false, class G = Group<T>>
__device__ __forceinline__ void ascend_one(const int8_t* __restrict__ Q8, int64_t ldq,
                                           int64_t ldy, int n,
                                           int W, uint64_t* __restrict__ x_g,
                                           int64_t* __restrict__ f_s, int32_t max_flips,
                                           int32_t* __restrict__ flips_s,
                                           unsigned* __restrict__ err, uint4* spec_slots,
                                           uint4* diag,
                                           const float* __restrict__ y_g, G& grp,
                                           const RelinkArgs* rl = nullptr,
                                           uint16_t* __restrict__ trace_row = nullptr,
                                           int64_t trace_cap = 0) {
  constexpr int E = 16 * C;
  constexpr int NG = (E + 31) / 32;  // key groups
  constexpr int CW = 16 * T;         // indices per chunk
  const int g = grp.rank();
  // this thread's column offset in each chunk, 0 where the chunk lies beyond
  // the row: those elements are no candidates, and what they read moves their
  // keys by no more than a real row would.  Row offsets fit 32 bits (n and
  // ldq <= 2^14).
  const uint32_t ld32 = (uint32_t)ldq;
  const int warp = __shfl_sync(0xffffffffu, g >> 5, 0);  // the same register in every lane
  uint32_t off[C];
#pragma unroll
  for (int c = 0; c < C; ++c)
    off[c] = c * CW + 16 * g < ldq ? (uint32_t)(c * CW + 16 * g) : 0u;
  auto row_chunk = [&](int k, int c) {
    return reinterpret_cast<const uint4*>(Q8 + ((uint32_t)k * ld32 + off[c]));
  };

  int key[E];
  uint32_t sel[E];  // +-64 in the element's byte: (1 - 2x) times the sign below
  uint32_t xm[NG];  // x bits of the owned elements
  uint32_t neg = 0;  // 0: sel is oriented for moves with d = +1, else for -1
  int ndiff = 0;    // relinking: owned variables where x and g differ
#pragma unroll
  for (int h = 0; h < NG; ++h) xm[h] = 0;
  // ---- owned bits of x, selectors, and keys from y = Q x of the tensor-core
  // start-up (y_g, exact integers in fp32; without it the rows are added below)
#pragma unroll
  for (int c = 0; c < C; ++c) {
    const int j0 = c * CW + 16 * g;
    uint32_t nib = 0, in = 0;
    if (j0 < n) {
      in = n - j0 < 16 ? (1u << (n - j0)) - 1u : 0xFFFFu;
      nib = (uint32_t)(x_g[j0 >> 6] >> (j0 & 63)) & in;
      if (RL) {
        in &= nib ^ (uint32_t)(rl->g[j0 >> 6] >> (j0 & 63));
        ndiff += __popc(in);
      }
    }
    xm[c >> 1] |= nib << (16 * (c & 1));
    float4 y4[4];
#pragma unroll
    for (int v = 0; v < 4; ++v)
      y4[v] = y_g && j0 < ldy ? reinterpret_cast<const float4*>(y_g + j0)[v]
                              : make_float4(0.f, 0.f, 0.f, 0.f);
    uint32_t dg[4] = {0, 0, 0, 0};
#pragma unroll
    for (int o = 0; o < 16; ++o) {
      const int e = c * 16 + o, j = j0 + o;
      const bool xb = (nib >> o) & 1u, cd = (in >> o) & 1u;
      const float4 yv = y4[o >> 2];
      const float yf = (o & 3) == 0 ? yv.x : (o & 3) == 1 ? yv.y : (o & 3) == 2 ? yv.z : yv.w;
      const int y2 = 2 * __float2int_rn(yf);
      const int qjj = cd ? Q8[(int64_t)j * ldq + j] : 0;
      key[e] = cd ? ((qjj + (xb ? -y2 : y2)) << kKeyBits) + (31 - (e & 31)) : kOutKey;
      sel[e] = (xb ? 0xC0u : 0x40u) << (8 * (o & 3));
      dg[o >> 2] |= (uint32_t)(uint8_t)qjj << (8 * (o & 3));
    }
    if constexpr (!RL) diag[c * T + g] = make_uint4(dg[0], dg[1], dg[2], dg[3]);
  }
  for (int w = 0; w < W && !y_g; ++w) {
    uint64_t word = x_g[w] & valid_mask(n, w);
    while (word) {
      // rows in flight.  Relinking takes as many of the two-chunk rows, its shapes
      // having the registers (128 x 2, n = 2800: one pair 865 us with 2 rows, 524
      // with 8; 16 pairs 631, 447; the ascent's have not)
      constexpr int RF = C == 1 || (RL && C == 2) ? 8 : C == 2 ? 2 : 1;
      int ks[RF];
      int nk = 0;
#pragma unroll
      for (int r = 0; r < RF; ++r) {
        ks[r] = 0;
        if (word) {
          ks[r] = w * 64 + __ffsll((long long)word) - 1;
          word &= word - 1;
          nk = r + 1;
        }
      }
      uint4 q[RF][C];
#pragma unroll
      for (int r = 0; r < RF; ++r)
#pragma unroll
        for (int c = 0; c < C; ++c) {
          q[r][c] = r < nk ? __ldg(row_chunk(ks[r], c)) : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
      for (int r = 0; r < RF; ++r)
#pragma unroll
        for (int c = 0; c < C; ++c) {
          const int wv[4] = {(int)q[r][c].x, (int)q[r][c].y, (int)q[r][c].z, (int)q[r][c].w};
#pragma unroll
          for (int o = 0; o < 16; ++o)
            key[c * 16 + o] = __dp4a(wv[o >> 2], (int)sel[c * 16 + o], key[c * 16 + o]);
        }
    }
  }
  // ---- first argmax
  int km[NG][2];
#pragma unroll
  for (int h = 0; h < NG; ++h) km[h][0] = km[h][1] = kFloorKey;
#pragma unroll
  for (int e = 0; e < E; e += 2)
    km[e >> 5][(e >> 1) & 1] = __vimax3_s32(km[e >> 5][(e >> 1) & 1], key[e], key[e + 1]);
  // the group's {max gain, 2k + x_k} from each thread's best key: the first
  // key group that attains the thread's largest gain (lower groups hold lower
  // indices)
  // bits that count chunks (one warp looks for the lowest index itself)
  constexpr int CB = T == 32 || C == 1 ? 0 : C == 2 ? 1 : C <= 4 ? 2 : 3;
  auto reduce_key = [&]() {
    int bk = max(km[0][0], km[0][1]), e0 = 31;
    uint32_t xw = xm[0];
#pragma unroll
    for (int h = 1; h < NG; ++h) {
      const int k = max(km[h][0], km[h][1]);
      if (k > (bk | 31)) {
        bk = k;
        e0 = 32 * h + 31;
        xw = xm[h];
      }
    }
    const int l = 31 - (bk & 31), e = e0 - (bk & 31);
    const int j = (e >> 4) * CW + 16 * g + (e & 15);
    // 2^CB gain + 2^CB - 1 - chunk
    const int rank = CB == 0   ? bk >> kKeyBits
                     : CB == 1 ? bk >> 4
                               : ((bk >> kKeyBits) << CB) + ((1 << CB) - 1 - (e >> 4));
    return grp.template reduce<CB>(rank, (j << 1) | (int)((xw >> l) & 1u));
  };
  // Speculation: the next move is often the runner-up of the previous
  // reduction (about 40% of moves at n = 7000), so each move copies this
  // thread's chunks of the runner-up rows (prow) into its own shared-memory
  // slots with cp.async; a hit reads them there instead of waiting for a
  // dependent L2 round trip.  Two buffers alternate: the copies of move t go
  // to buffer t % 2 and are read at move t + 1.  Each thread reads only the
  // bytes it copied, so its own cp.async.wait_group orders them.
  constexpr int RR = R > 0 ? R : 1;
  int cand[RR], prow[RR];
#pragma unroll
  for (int i = 0; i < RR; ++i) prow[i] = -1;
  // slot (buffer b, row i, chunk c) of thread g at plane ((b RR + i) C + c):
  // planes of T x 16 bytes, threads side by side, so a warp's copies and
  // reads cover all banks without conflicts
  const uint32_t slot0 =
      R > 0 ? (uint32_t)__cvta_generic_to_shared(spec_slots) + (uint32_t)g * 16 : 0u;
  int buf = 0;
  int2 best = reduce_key();
  // every lane of the owner's warp reads q_kk from diag: a block's reduction orders
  // the writes before it, a warp's holds no barrier.  (Placed here it costs nothing;
  // right behind the writes, or with the read left to the owner, 1 to 6%.)
  if constexpr (!RL && T == 32) grp.sync();

  int64_t fval = *f_s;
  int flips = 0;
  if (max_flips == 0) max_flips = INT_MAX;
  // relinking: path length, best intermediate value and its step
  const int dist = RL ? grp.sum(ndiff) : 0;
  int64_t fbest = fval;
  int tbest = 0;
  const uint64_t t0 = globaltimer();
  const int last = RL ? dist - 1 : max_flips;  // relinking: the last step only reaches g
  int lim = min(last, 1023);                   // the next move count to look at
  for (;;) {
    // the row first: everything up to the update runs in the shadow of its
    // load (a load for the move that is not made reads a valid row)
    const int k = RL ? min(best.y >> 1, n - 1) : best.y >> 1;
    int q[4 * C];
    bool hit = false;
    if constexpr (R > 0) {
      int hi = -1;
#pragma unroll
      for (int i = 0; i < RR; ++i)
        if (prow[i] == k) hi = i;
      if (hi >= 0) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        const uint32_t a = slot0 + (uint32_t)(((buf ^ 1) * RR + hi) * C) * (T * 16);
#pragma unroll
        for (int c = 0; c < C; ++c)
          asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                       : "=r"(q[4 * c]), "=r"(q[4 * c + 1]), "=r"(q[4 * c + 2]),
                         "=r"(q[4 * c + 3])
                       : "r"(a + (uint32_t)(c * T * 16)));
        hit = true;
      }
    }
    if (!hit) {
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const uint4 v = __ldg(row_chunk(k, c));
        q[4 * c] = (int)v.x;
        q[4 * c + 1] = (int)v.y;
        q[4 * c + 2] = (int)v.z;
        q[4 * c + 3] = (int)v.w;
      }
    }
    if ((!RL && best.x <= 0) || flips >= lim) {
      if ((!RL && best.x <= 0) || flips >= last) break;
      const bool late = (int64_t)(globaltimer() - t0) > kTimeoutNs;
      if (grp.any(late)) {
        if (g == 0) atomicOr(err, UBQP_DEVERR_TIMEOUT);
        break;
      }
      lim = min(last, flips + 1024);
    }
    fval += best.x;
    ++flips;
    if (RL) {
      if (flips < dist && (tbest == 0 || fval > fbest)) {
        fbest = fval;
        tbest = flips;
      }
      if (g == 0) rl->trace[flips - 1] = (uint16_t)k;
    }
    if constexpr (TR) {  // the move record: flipped indices in order
      if (g == 0 && flips <= trace_cap) trace_row[flips - 1] = (uint16_t)k;
    }
    if constexpr (R > 0) {  // fetch the runners-up's rows for the next move
      grp.template runners<R>(best.y, cand);
      // the copies into this buffer two moves ago have landed
      asm volatile("cp.async.wait_group 1;" ::: "memory");
#pragma unroll
      for (int i = 0; i < R; ++i) {
        const int r = cand[i] >> 1;
        prow[i] = r < n ? r : -1;
        const int from = r < n ? r : 0;
#pragma unroll
        for (int c = 0; c < C; ++c)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                           slot0 + (uint32_t)((buf * RR + i) * C + c) * (T * 16)),
                       "l"(row_chunk(from, c))
                       : "memory");
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      buf ^= 1;
    }
    // orient the selectors for this move's d = 1 - 2 x_k (they are kept as
    // the last move left them: the signs of successive moves agree about
    // every other time)
    const uint32_t ng = (uint32_t)(best.y & 1);
    if (ng != neg) {
#pragma unroll
      for (int e = 0; e < E; ++e) sel[e] ^= 0x80u << (8 * (e & 3));
      neg = ng;
    }
    // the owner of k flips x_k (when relinking, k leaves the candidates)
    const int kc = k / CW, kr = k - kc * CW;
    if (T == 32 || (kr >> 9) == warp) {
      const int qkk = RL ? 0 : reinterpret_cast<const int8_t*>(diag)[k];
      flip_tree<0, E, E, RL>(key, sel, xm, kc * 16 + (kr & 15),
                             (2 * qkk - best.x) * (1 << kKeyBits), (kr >> 4) == g);
    }
#pragma unroll
    for (int h = 0; h < NG; ++h) km[h][0] = km[h][1] = kFloorKey;
#pragma unroll
    for (int e = 0; e < E; e += 2) {
      key[e] = __dp4a(q[e >> 2], (int)sel[e], key[e]);
      key[e + 1] = __dp4a(q[e >> 2], (int)sel[e + 1], key[e + 1]);
      km[e >> 5][(e >> 1) & 1] = __vimax3_s32(km[e >> 5][(e >> 1) & 1], key[e], key[e + 1]);
    }
    best = reduce_key();
  }
  // copies still in flight must land before the slots serve another start
  if (R > 0) asm volatile("cp.async.wait_group 0;" ::: "memory");
  if constexpr (RL) {
    // ---- the best intermediate: x with the first tbest traced flips applied
    if (g == 0) {
      *rl->f_best = fbest;
      if (rl->dist) *rl->dist = dist;
    }
    uint64_t* xs = rl->xs;
    for (int w = g; w < W; w += T) xs[w] = x_g[w];
    grp.sync();
    for (int t = g; t < tbest; t += T) {
      const int k = rl->trace[t];
      atomicXor(reinterpret_cast<unsigned long long*>(&xs[k >> 6]), 1ull << (k & 63));
    }
    grp.sync();
    for (int w = g; w < W; w += T) rl->x_best[w] = xs[w];
    grp.sync();
    return;
  }
  // ---- write back f, flips and x
  if (g == 0) {
    *f_s = fval;
    if (flips_s) *flips_s = flips;
  }
  grp.sync();  // every thread has read its words of x_g
#pragma unroll
  for (int c = 0; c < C; ++c) {
    const int j0 = c * CW + 16 * g;
    if (j0 < 64 * W)
      reinterpret_cast<uint16_t*>(x_g)[j0 >> 4] =
          (uint16_t)(xm[c >> 1] >> (16 * (c & 1)));
  }
  grp.sync();
}

// The first wave of listed starts goes one per group in launch order (the
// block scheduler spreads them over the SMs); the rest are taken from the
// counter *next (zero at launch) one at a time as groups finish, so the long
// and short climbs even out over the SMs.  next == NULL: round robin.
// TR: also record each start's flipped indices in order, row s of trace (ldt
// entries; moves beyond ldt are made but not recorded).  OCC: blocks per SM
// the registers are sized for.  The kernel climbs only when the number of
// listed starts lies in [cnt_lo, cnt_hi] and returns at once otherwise, so
// that two launches of different OCC can share one list, each taking the
// counts it is faster for, with no host round trip for the count.  Y has S
// rows; the starts of a longer list (which has entries outside [0, S)) sum
// their own start-up.  A programmatic dependent of the kernel before it on the
// stream (pdl_wait).
template <int T, int C, int R, bool TR, int OCC>
__global__ void __launch_bounds__(T, OCC)
ascent_block_kernel(const int8_t* __restrict__ Q8, int64_t ldq, int n, int W,
                    uint64_t* __restrict__ X, int64_t* __restrict__ f,
                    const int32_t* __restrict__ idx, const int64_t* __restrict__ count,
                    int64_t S, int32_t max_flips, int32_t* __restrict__ flips,
                    const float* __restrict__ Y, int64_t ldy, unsigned* __restrict__ err,
                    unsigned long long* __restrict__ next, uint16_t* __restrict__ trace,
                    int64_t ldt, int64_t cnt_lo, int64_t cnt_hi) {
  __shared__ int2 rec[2][T / 32];
  __shared__ uint4 spec_slots[spec_slot_count<T, C, R>()];
  __shared__ uint4 diag[T * C];
  __shared__ unsigned long long ticket;
  Group<T> grp{rec, 0};
  pdl_wait();  // no early release: see pdl_release
  if (err[1] != 0) return;  // Q failed its symmetry check: no climb
  const int64_t cnt = *count;
  if (cnt < cnt_lo || cnt > cnt_hi) return;  // the other launch's counts
  auto take = [&](int64_t t) -> int64_t {  // the block's next start
    if (t < 0) return blockIdx.x;
    if (!next) return t + gridDim.x;
    if (threadIdx.x == 0) ticket = atomicAdd(next, 1ull);
    __syncthreads();
    const int64_t v = (int64_t)gridDim.x + (int64_t)ticket;
    __syncthreads();
    return v;
  };
  for (int64_t t = take(-1); t < cnt; t = take(t)) {
    const int s = idx[t];
    if (s < 0 || s >= S) {
      if (threadIdx.x == 0) atomicOr(err, UBQP_DEVERR_BADIDX);
      continue;
    }
    ascend_one<T, C, R, false, TR>(Q8, ldq, ldy, n, W, X + (int64_t)s * W, f + s, max_flips,
                                   flips ? flips + s : nullptr, err, spec_slots, diag,
                                   Y && cnt <= S ? Y + t * ldy : nullptr, grp, nullptr,
                                   TR ? trace + (int64_t)s * ldt : nullptr, ldt);
  }
}

// All passing starts of a batch of instances in one persistent launch: item
// t = (instance, position in its passing list); every instance has n <= 16 T C.
// Climbs only when the number of items lies in [lo, hi].
template <int T, int C, int R, int OCC>
__global__ void __launch_bounds__(T, OCC)
ascent_batch_kernel(const BatchDesc* __restrict__ d, const int2* __restrict__ items,
                    const int64_t* __restrict__ n_items, int32_t max_flips,
                    unsigned long long* __restrict__ next, int64_t lo, int64_t hi) {
  __shared__ int2 rec[2][T / 32];
  __shared__ uint4 spec_slots[spec_slot_count<T, C, R>()];
  __shared__ uint4 diag[T * C];
  __shared__ unsigned long long ticket;
  Group<T> grp{rec, 0};
  const int64_t cnt = *n_items;
  if (cnt < lo || cnt > hi) return;  // the other launch's counts
  // the first wave one item per block, the rest from the counter (as in
  // ascent_block_kernel)
  auto take = [&](int64_t t) -> int64_t {
    if (t < 0) return blockIdx.x;
    if (!next) return t + gridDim.x;
    if (threadIdx.x == 0) ticket = atomicAdd(next, 1ull);
    __syncthreads();
    const int64_t v = (int64_t)gridDim.x + (int64_t)ticket;
    __syncthreads();
    return v;
  };
  for (int64_t t = take(-1); t < cnt; t = take(t)) {
    const int2 it = items[t];
    const BatchDesc& b = d[it.x];
    if (b.err[1] != 0) continue;  // Q failed its symmetry check: no climb
    const int s = b.idx[it.y];
    if (s < 0 || s >= b.S) {
      if (threadIdx.x == 0) atomicOr(b.err, UBQP_DEVERR_BADIDX);
      continue;
    }
    ascend_one<T, C, R>(b.Q8, b.ldq, b.ldy, b.n, b.W,
                     b.X + (int64_t)s * b.W, b.f + s, max_flips,
                     b.flips ? b.flips + s : nullptr, b.err, spec_slots, diag,
                     b.Y ? b.Y + (int64_t)it.y * b.ldy : nullptr, grp);
  }
}

// Independent warps, one start each (kWarps per block); counts, starts and
// launch as in the block kernel, the first wave one warp per block over the
// whole grid before any block's second warp.  (The test for Y's S rows is per
// entry and in 32 bits here: as in the block kernel it cost the 80-element warps
// four spilled registers and 2%.)
template <int C, int R, bool TR, int OCC>
__global__ void __launch_bounds__(32 * kWarps, OCC)
ascent_warp_kernel(const int8_t* __restrict__ Q8, int64_t ldq, int n, int W,
                   uint64_t* __restrict__ X, int64_t* __restrict__ f,
                   const int32_t* __restrict__ idx, const int64_t* __restrict__ count,
                   int64_t S, int32_t max_flips, int32_t* __restrict__ flips,
                   const float* __restrict__ Y, int64_t ldy, unsigned* __restrict__ err,
                   unsigned long long* __restrict__ next, uint16_t* __restrict__ trace,
                   int64_t ldt, int64_t cnt_lo, int64_t cnt_hi) {
  __shared__ uint4 spec_slots[kWarps * spec_slot_count<32, C, R>()];
  __shared__ uint4 diag[kWarps * 32 * C];
  Group<32> grp;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  pdl_wait();  // no early release: see pdl_release
  if (err[1] != 0) return;  // Q failed its symmetry check: no climb
  const int64_t cnt = *count;
  if (cnt < cnt_lo || cnt > cnt_hi) return;  // another launch's counts
  auto take = [&](int64_t t) -> int64_t {  // the warp's next start (see the block kernel)
    if (t < 0) return (int64_t)warp * gridDim.x + blockIdx.x;
    if (!next) return t + (int64_t)gridDim.x * kWarps;
    unsigned long long v = 0;
    if (lane == 0) v = atomicAdd(next, 1ull);
    return (int64_t)gridDim.x * kWarps + (int64_t)__shfl_sync(0xffffffffu, v, 0);
  };
  for (int64_t t = take(-1); t < cnt; t = take(t)) {
    const int s = idx[t];
    if (s < 0 || s >= S) {
      if (lane == 0) atomicOr(err, UBQP_DEVERR_BADIDX);
      continue;
    }
    ascend_one<32, C, R, false, TR>(Q8, ldq, ldy, n, W, X + (int64_t)s * W, f + s, max_flips,
                                    flips ? flips + s : nullptr, err,
                                    spec_slots + warp * spec_slot_count<32, C, R>(),
                                    diag + warp * (32 * C),
                                    Y && (t >> 31) == 0 && (int)t < (int)S ? Y + t * ldy : nullptr, grp,
                                    nullptr,
                                    TR ? trace + (int64_t)s * ldt : nullptr, ldt);
  }
}

// The passing starts of one size class of a batch (launch_ascent_batch_packed):
// items[ranges[cls].x .. + ranges[cls].y), every instance with n <= 16 T C, T
// threads per start (T = 32: kWarps starts per block).  First wave and counter
// as in the kernels above.  Climbs only when the batch's total number of items
// lies in [lo, hi].
template <int T, int C, int R, int OCC>
__global__ void __launch_bounds__(T == 32 ? 32 * kWarps : T, OCC)
ascent_class_kernel(const BatchDesc* __restrict__ d, const int2* __restrict__ items,
                    const int4* __restrict__ ranges, int cls,
                    const int64_t* __restrict__ n_items, int32_t max_flips,
                    unsigned long long* __restrict__ next, int64_t lo, int64_t hi) {
  constexpr int PER = T == 32 ? kWarps : 1;
  __shared__ int2 rec[2][T / 32];
  __shared__ uint4 spec_slots[PER * spec_slot_count<T, C, R>()];
  __shared__ uint4 diag[PER * T * C];
  __shared__ unsigned long long ticket;
  const int64_t total = *n_items;
  if (total < lo || total > hi) return;
  const int4 range = ranges[cls];
  const int sub = (int)threadIdx.x / T, rank = (int)threadIdx.x % T;
  const int64_t wave = (int64_t)gridDim.x * PER;
  for (int64_t t = (int64_t)sub * gridDim.x + blockIdx.x; t < range.y;) {
    const int2 it = items[range.x + t];
    const BatchDesc& b = d[it.x];
    const int s = b.idx[it.y];
    if (b.err[1] == 0) {  // else Q failed its symmetry check: no climb
      if (s < 0 || s >= b.S) {
        if (rank == 0) atomicOr(b.err, UBQP_DEVERR_BADIDX);
      } else {
        const float* y = b.Y ? b.Y + (int64_t)it.y * b.ldy : nullptr;
        int32_t* fl = b.flips ? b.flips + s : nullptr;
        if constexpr (T == 32) {
          Group<32> grp;
          ascend_one<32, C, R>(b.Q8, b.ldq, b.ldy, b.n, b.W, b.X + (int64_t)s * b.W, b.f + s,
                               max_flips, fl, b.err,
                               spec_slots + sub * spec_slot_count<32, C, R>(),
                               diag + sub * (32 * C), y, grp);
        } else {
          Group<T> grp{rec, 0};
          ascend_one<T, C, R>(
              b.Q8, b.ldq, b.ldy, b.n, b.W, b.X + (int64_t)s * b.W, b.f + s, max_flips, fl, b.err,
              spec_slots, diag, y, grp);
        }
      }
    }
    if (!next) {
      t += wave;
    } else if constexpr (T == 32) {
      unsigned long long v = 0;
      if (rank == 0) v = atomicAdd(&next[cls], 1ull);
      t = wave + (int64_t)__shfl_sync(0xffffffffu, v, 0);
    } else {
      __syncthreads();  // rec is free for the next start; ticket was read
      if (rank == 0) ticket = atomicAdd(&next[cls], 1ull);
      __syncthreads();
      t = wave + (int64_t)ticket;
    }
  }
}

// Path relinking of pairs p < P: from X[p] (value f[p]) toward G[p]; the best
// intermediate solution to Xb[p], its value to fb[p], the distance to dist[p]
// (may be NULL).  trace: P rows of ldt uint16 scratch.  Y: y = Q X[p] rows from
// the tensor-core start-up, or NULL.
template <int T, int C, int R, int OCC>
__global__ void __launch_bounds__(T, OCC)
relink_block_kernel(const int8_t* __restrict__ Q8, int64_t ldq, int n, int W,
                    const uint64_t* __restrict__ X, const int64_t* __restrict__ f,
                    const uint64_t* __restrict__ G, int64_t P, uint64_t* __restrict__ Xb,
                    int64_t* __restrict__ fb, int32_t* __restrict__ dist,
                    uint16_t* __restrict__ trace, int64_t ldt, const float* __restrict__ Y,
                    int64_t ldy, unsigned* __restrict__ err,
                    unsigned long long* __restrict__ next) {
  __shared__ int2 rec[2][T / 32];
  __shared__ uint64_t xs[UBQP_MAX_N / 64];
  __shared__ uint4 spec_slots[spec_slot_count<T, C, R>()];
  __shared__ unsigned long long ticket;
  Group<T> grp{rec, 0};
  if (err[1] != 0) return;  // Q failed its symmetry check: no walk
  // the first wave one pair per block, the rest from the counter (as in
  // ascent_block_kernel)
  auto take = [&](int64_t t) -> int64_t {
    if (t < 0) return blockIdx.x;
    if (!next) return t + gridDim.x;
    if (threadIdx.x == 0) ticket = atomicAdd(next, 1ull);
    __syncthreads();
    const int64_t v = (int64_t)gridDim.x + (int64_t)ticket;
    __syncthreads();
    return v;
  };
  for (int64_t p = take(-1); p < P; p = take(p)) {
    const RelinkArgs a{G + p * W, Xb + p * W, fb + p, dist ? dist + p : nullptr,
                       trace + p * ldt, xs};
    int64_t f0 = f[p];
    ascend_one<T, C, R, true>(Q8, ldq, ldy, n, W, const_cast<uint64_t*>(X + p * W), &f0, 0,
                              nullptr, err, spec_slots, nullptr, Y ? Y + p * ldy : nullptr, grp,
                              &a);
  }
}

template <int C, int R>
__global__ void __launch_bounds__(128)
relink_warp_kernel(const int8_t* __restrict__ Q8, int64_t ldq, int n, int W,
                   const uint64_t* __restrict__ X, const int64_t* __restrict__ f,
                   const uint64_t* __restrict__ G, int64_t P, uint64_t* __restrict__ Xb,
                   int64_t* __restrict__ fb, int32_t* __restrict__ dist,
                   uint16_t* __restrict__ trace, int64_t ldt, const float* __restrict__ Y,
                   int64_t ldy, unsigned* __restrict__ err,
                   unsigned long long* __restrict__ next) {
  __shared__ uint64_t xs_all[4][16];
  __shared__ uint4 spec_slots[4 * spec_slot_count<32, C, R>()];
  Group<32> grp;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (err[1] != 0) return;  // Q failed its symmetry check: no walk
  auto take = [&](int64_t t) -> int64_t {  // the warp's next pair (see the block kernel)
    if (t < 0) return (int64_t)blockIdx.x * 4 + warp;
    if (!next) return t + (int64_t)gridDim.x * 4;
    unsigned long long v = 0;
    if (lane == 0) v = atomicAdd(next, 1ull);
    return (int64_t)gridDim.x * 4 + (int64_t)__shfl_sync(0xffffffffu, v, 0);
  };
  for (int64_t p = take(-1); p < P; p = take(p)) {
    const RelinkArgs a{G + p * W, Xb + p * W, fb + p, dist ? dist + p : nullptr,
                       trace + p * ldt, xs_all[warp]};
    int64_t f0 = f[p];
    ascend_one<32, C, R, true>(Q8, ldq, ldy, n, W, const_cast<uint64_t*>(X + p * W), &f0, 0,
                               nullptr, err,
                               spec_slots + warp * spec_slot_count<32, C, R>(), nullptr,
                               Y ? Y + p * ldy : nullptr, grp, &a);
  }
}

template <class K>
int resident_grid(K kernel, int threads, int sm_count) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0) !=
          cudaSuccess ||
      per_sm < 1) {
    cudaGetLastError();
    per_sm = 1;
  }
  return per_sm * sm_count;
}

// One ascent launch of a group shape: T threads and 16 C elements per thread
// for each start (T = 32: one warp, kWarps to a block), R runner-up rows
// copied ahead, registers sized for OCC blocks per SM.  Climbs only for counts
// in [lo, hi].
struct AscArgs {
  const ubqp_q* h;
  uint64_t* X;
  int64_t* f;
  const int32_t* idx;
  const int64_t* count;
  int64_t S;
  int32_t max_flips;
  int32_t* flips;
  const float* Y;
  unsigned long long* next;
  uint16_t* trace;
  int64_t ldt;
  cudaStream_t st;
};
template <int T, int C, int R, int OCC, bool TR>
struct Climb {
  static constexpr int kBlock = T == 32 ? 32 * kWarps : T;
  static constexpr int kPer = kBlock / T;  // starts per block
  // starts resident on the device at once
  static int64_t capacity(const ubqp_q* h) { return (int64_t)kPer * blocks(h); }
  static int64_t blocks(const ubqp_q* h) {
    if constexpr (T == 32)
      return resident_grid(ascent_warp_kernel<C, R, TR, OCC>, kBlock, h->sm_count);
    else
      return resident_grid(ascent_block_kernel<T, C, R, TR, OCC>, kBlock, h->sm_count);
  }
  static cudaError_t launch(const AscArgs& a, int64_t lo, int64_t hi) {
    const dim3 grid((unsigned)std::min<int64_t>(blocks(a.h), (a.S + kPer - 1) / kPer));
    if constexpr (T == 32)
      return launch_pdl(ascent_warp_kernel<C, R, TR, OCC>, grid, dim3(kBlock), 0, a.st, a.h->Q8,
                        a.h->ldq, a.h->n, a.h->W, a.X, a.f, a.idx, a.count, a.S, a.max_flips,
                        a.flips, a.Y, (int64_t)a.h->n_tc, a.h->err, a.next, a.trace, a.ldt, lo,
                        hi);
    else
      return launch_pdl(ascent_block_kernel<T, C, R, TR, OCC>, grid, dim3(kBlock), 0, a.st,
                        a.h->Q8, a.h->ldq, a.h->n, a.h->W, a.X, a.f, a.idx, a.count, a.S,
                        a.max_flips, a.flips, a.Y, (int64_t)a.h->n_tc, a.h->err, a.next, a.trace,
                        a.ldt, lo, hi);
  }
};

// The ascent launches over the listed starts, by n and by how many of them
// there are.  The count is known only on the device, so for a list that may
// exceed a shape's range several launches are made, each climbing only for its
// own range of counts; the others return at once (about 2 us).
//   few  the shortest chain of moves: mostly 16 elements per thread, registers for
//        as many blocks per SM as that leaves; for lists up to its resident
//        capacity.  (n = 5000, 16 starts: 160 threads of 32 elements 1083, 320 of
//        16 970; 256 starts 1467 -> 1172.)
//   mid  two chunks per thread and several blocks per SM, whose waits cover
//        one another.
// Neither copies the runner-up's row any more (R = 0): with the cheaper flip and
// reduction the runner-up's reductions and copies cost every move more than the
// 40% of moves that hit saved (with and without: n = 1025, 510 starts 131 -> 113; 2500,
// 542 starts 351 -> 270; 7000, 54 starts 1630 -> 1580, 641 starts 2567 -> 2192).
//   all  few warps per start, and elements beyond n in as few threads as the
//        registers allow (one warp up to n = 2560, 80 elements a thread), for lists
//        that keep every SM busy: there the issue slots bound the climb, and the
//        copies cost more than their hits save.
//        (n = 2500, 3213 starts: two warps of 48 elements a thread 1059, one of 80
//        996; n = 5000, 4469 starts: 96 threads of 64 5255, with 1144 elements
//        beyond n, 160 of 32 4659; n = 1400: seven blocks per SM 662, six 634.)
// Measured on 1000 to 12 000 diversified starts, the passing ones climbed (us,
// with y, S, C registers -> now): n = 1025, 510 starts 187 -> 113; 2500, 542
// starts 533 -> 270; 1000, 5638 starts 784 -> 344; 1400, 6069: 1382 -> 634;
// 2000, 4214: 1406 -> 832; 2500, 3213: 2082 -> 996; 4000, 2193: 3046 -> 1675;
// 5000, 4469: 9080 -> 4659; 6000, 2187: 7464 -> 3584; 7000, 54: 1857 -> 1580;
// 7000, 641: 3364 -> 2192; 7000, 2172: 9610 -> 5045.  The boundary between mid
// and all lies near 10 starts per SM, where a list of that n keeps mid's SMs busy
// anyway, and at 2 per SM for 4096 < n <= 6144, where mid fits few blocks.
template <bool TR>
cudaError_t launch_ascent_shaped(const ubqp_q* h, uint64_t* X, int64_t* f, const int32_t* idx,
                                 const int64_t* count, int64_t S, int32_t max_flips,
                                 int32_t* flips, const float* Y, unsigned long long* next,
                                 uint16_t* trace, int64_t ldt, cudaStream_t st,
                                 bool next_zeroed) {
  const int n = h->n;
  if (next && !next_zeroed) {
    cudaError_t e = cudaMemsetAsync(next, 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
  }
  const AscArgs a{h, X, f, idx, count, S, max_flips, flips, Y, next, trace, ldt, st};
  // few: the shortest chain of moves, for lists up to its resident capacity;
  // mid: several blocks per SM, whose waits cover one another; all: few warps
  // per start, for lists that keep the whole chip busy (more than `full` starts)
  // The last launch made also takes every larger count: a list may be longer
  // than S when entries in it lie outside [0, S), which the climb reports.
  auto tiers = [&](auto few, auto mid, auto all, int64_t full) {
    const int64_t cap = std::min(few.capacity(h), full);
    cudaError_t e = few.launch(a, 0, S > cap ? cap : INT64_MAX);
    if (e == cudaSuccess && cap < full && S > cap)
      e = mid.launch(a, cap + 1, S > full ? full : INT64_MAX);
    if (e == cudaSuccess && S > full) e = all.launch(a, full + 1, INT64_MAX);
    return e;
  };
  auto two = [&](auto few, auto all, int64_t full) {
    cudaError_t e = few.launch(a, 0, S > full ? full : INT64_MAX);
    if (e == cudaSuccess && S > full) e = all.launch(a, full + 1, INT64_MAX);
    return e;
  };
  const int64_t full = 10ll * h->sm_count;
#define UBQP_C(TT, CC, RR, OCC) Climb<TT, CC, RR, OCC, TR>{}
  // n <= 128: one launch, the climbs being as short as a launch that returns at once
  // (33, 23 of 1600 starts, a few moves each: 24.2 us with both, 23.0; 100, 28 of
  // 1600 30.3, 28.3; two launches are faster again from n = 200 on, 1380 of 8000
  // starts 65.2 with one, 59.0 with two)
  if (n <= 128)
    return S > full ? UBQP_C(32, 1, 0, 10).launch(a, 0, INT64_MAX)
                    : UBQP_C(32, 1, 0, 8).launch(a, 0, INT64_MAX);
  if (n <= 512) return two(UBQP_C(32, 1, 0, 8), UBQP_C(32, 1, 0, 10), full);
  if (n <= 1024) return two(UBQP_C(64, 1, 0, 8), UBQP_C(32, 2, 0, 8), full);
  if (n <= 1536) return tiers(UBQP_C(96, 1, 0, 7), UBQP_C(64, 2, 0, 8), UBQP_C(32, 3, 0, 6), full);
  if (n <= 2048) return tiers(UBQP_C(128, 1, 0, 4), UBQP_C(64, 2, 0, 8), UBQP_C(32, 4, 0, 5), full);
  if (n <= 2560) return tiers(UBQP_C(160, 1, 0, 4), UBQP_C(96, 2, 0, 4), UBQP_C(32, 5, 0, 4), full);
  if (n <= 3072) return tiers(UBQP_C(192, 1, 0, 2), UBQP_C(96, 2, 0, 4), UBQP_C(64, 3, 0, 7), full);
  if (n <= 4096) return tiers(UBQP_C(256, 1, 0, 2), UBQP_C(128, 2, 0, 4), UBQP_C(64, 4, 0, 5), full);
  if (n <= 5120) return two(UBQP_C(320, 1, 0, 2), UBQP_C(160, 2, 0, 4), 2ll * h->sm_count);
  if (n <= 6144)
    return tiers(UBQP_C(384, 1, 0, 1), UBQP_C(192, 2, 0, 3), UBQP_C(96, 4, 0, 3), 2ll * h->sm_count);
  if (n <= 7168)
    return tiers(UBQP_C(224, 2, 0, 1), UBQP_C(224, 2, 0, 2), UBQP_C(128, 4, 0, 3), full);
  if (n <= 8192)
    return tiers(UBQP_C(256, 2, 0, 1), UBQP_C(256, 2, 0, 2), UBQP_C(128, 4, 0, 3), full);
  return UBQP_C(512, 2, 1, 1).launch(a, 0, INT64_MAX);
#undef UBQP_C
}

template <int T, int C, int R, int OCC>
cudaError_t launch_class(const BatchDesc* d, const int2* items, const int4* ranges, int cls,
                         const int64_t* n_items, int32_t max_flips, unsigned long long* next,
                         int64_t most, int64_t lo, int64_t hi, int sm_count, cudaStream_t st) {
  constexpr int kBlock = T == 32 ? 32 * kWarps : T, kPer = kBlock / T;
  int64_t grid = resident_grid(ascent_class_kernel<T, C, R, OCC>, kBlock, sm_count);
  if (grid > (most + kPer - 1) / kPer) grid = (most + kPer - 1) / kPer;
  ascent_class_kernel<T, C, R, OCC><<<(unsigned)grid, kBlock, 0, st>>>(
      d, items, ranges, cls, n_items, max_flips, next, lo, hi);
  return cudaGetLastError();
}

template <int T, int C, int R, int OCC>
cudaError_t launch_batch_shape(const BatchDesc* d, const int2* items, const int64_t* n_items,
                               int32_t max_flips, unsigned long long* next, int64_t most,
                               int64_t lo, int64_t hi, int sm_count, cudaStream_t st) {
  const int64_t grid = std::min<int64_t>(
      resident_grid(ascent_batch_kernel<T, C, R, OCC>, T, sm_count), most);
  ascent_batch_kernel<T, C, R, OCC>
      <<<(unsigned)grid, T, 0, st>>>(d, items, n_items, max_flips, next, lo, hi);
  return cudaGetLastError();
}

template <int T, int C, int OCC>
cudaError_t launch_relink_block(const ubqp_q* h, const uint64_t* X, const int64_t* f,
                                const uint64_t* G, int64_t P, uint64_t* Xb, int64_t* fb,
                                int32_t* dist, uint16_t* trace, int64_t ldt, const float* Y,
                                unsigned long long* next, cudaStream_t st) {
  int grid = resident_grid(relink_block_kernel<T, C, kSpecRows, OCC>, T, h->sm_count);
  if ((int64_t)grid > P) grid = (int)P;
  relink_block_kernel<T, C, kSpecRows, OCC><<<grid, T, 0, st>>>(
      h->Q8, h->ldq, h->n, h->W, X, f, G, P, Xb, fb, dist, trace, ldt, Y, h->n_tc, h->err,
      next);
  return cudaGetLastError();
}

template <int C>
cudaError_t launch_relink_warp(const ubqp_q* h, const uint64_t* X, const int64_t* f,
                               const uint64_t* G, int64_t P, uint64_t* Xb, int64_t* fb,
                               int32_t* dist, uint16_t* trace, int64_t ldt, const float* Y,
                               unsigned long long* next, cudaStream_t st) {
  int grid = resident_grid(relink_warp_kernel<C, kSpecRows>, 128, h->sm_count);
  const int64_t need = (P + 3) / 4;
  if ((int64_t)grid > need) grid = (int)need;
  relink_warp_kernel<C, kSpecRows><<<grid, 128, 0, st>>>(
      h->Q8, h->ldq, h->n, h->W, X, f, G, P, Xb, fb, dist, trace, ldt, Y, h->n_tc, h->err,
      next);
  return cudaGetLastError();
}

}  // namespace
}  // namespace ubqp
