// k_prepare.cu -- one pass over Q: symmetry check (problem (P) requires a
// symmetric Q), max|Q|, the padded int8 copy read by the ascent, the bf16
// tensor-core operands Q' = 2*tril(Q,-1) + diag(Q) (evaluation) and its
// transpose 2*triu(Q,1) + diag(Q) (with Q', the ascent's y = Q x), and the row
// sums behind the first-derivative start of Fig. 2
// (CalculateFirstDerivativeSolution).
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>

#include "ubqp_internal.cuh"

namespace ubqp {
namespace {

constexpr int PT = 64;        // tile edge
static_assert(UBQP_TC_ALIGN % (4 * PT) == 0, "a multiple of four tiles");
constexpr int PTHREADS = 256;  // 4 threads per tile row, 16 columns each

// Four bytes of row j from column k (zero at or beyond n): one 32-bit load when
// the four are inside the row and W4 (4-byte aligned rows); on other rows the
// two aligned words around them, shifted together, where both words lie inside
// the caller's rows [Q, end); else bytes.
template <bool W4>
__device__ __forceinline__ uint32_t row_word(const int8_t* __restrict__ Q, const int8_t* end,
                                             int64_t ldq_in, int n, int j, int k) {
  if (j >= n) return 0;
  const int8_t* p = Q + (int64_t)j * ldq_in + k;
  if (k + 3 < n) {
    if (W4) return *reinterpret_cast<const uint32_t*>(p);
    const unsigned off = (unsigned)((uintptr_t)p & 3);
    const int8_t* lo = p - off;
    if (lo >= Q && lo + 8 <= end) {
      const uint32_t* q = reinterpret_cast<const uint32_t*>(lo);
      return __funnelshift_r(q[0], q[1], 8 * off);
    }
  }
  uint32_t w = 0;
#pragma unroll
  for (int b = 0; b < 4; ++b)
    if (k + b < n) w |= (uint32_t)(uint8_t)p[b] << (8 * b);
  return w;
}

// Two of a word's four int8 values as packed bf16.  With v = m - 128 s (m the low
// seven bits, s the sign), 0x4300 | m is 128 + m and 0x4300 | 128 s is 128 + 128 s,
// both exact in bf16, and so is their difference v: no conversion instruction
// (they run at a quarter of the rate or less).
__device__ __forceinline__ __nv_bfloat162 bf16_pair(uint32_t w, unsigned bytes) {
  const uint32_t h = __byte_perm(w, 0, bytes);  // {v0, 0, v1, 0}
  const uint32_t a = (h & 0x007F007Fu) | 0x43004300u, c = (h & 0x00800080u) | 0x43004300u;
  __nv_bfloat162 x, y;
  memcpy(&x, &a, 4);
  memcpy(&y, &c, 4);
  return __hsub2(x, y);
}
__device__ __forceinline__ uint32_t bits_of(__nv_bfloat162 v) {
  uint32_t u;
  memcpy(&u, &v, 4);
  return u;
}

// Largest column of Q' that the tensor-core evaluation reads in rows
// j0 .. j0 + PT - 1: an N-block of 256 rows (192 in the tensor-memory
// variant) reads K up to the end of its own block.  Tiles of Q' beyond it are
// never read and are not written.
__device__ __forceinline__ int qt_kmax(int j0) {
  const int jl = j0 + PT - 1;
  return max((jl / 256 + 1) * 256, (jl / 192 + 1) * 192) - 1;
}

// One staged tile (rows rb PT .., columns cb PT ..) to the outputs: 16 columns of
// one row per thread.  SIDE: the tile lies on (0), above (1) or below (-1) the
// diagonal.
template <int SIDE>
__device__ __forceinline__ void emit_tile(const int8_t (*tile)[PT + 4], int rb, int cb, int n,
                                          int8_t* __restrict__ Q8, int64_t ldq,
                                          uint16_t* __restrict__ Qt, uint16_t* __restrict__ Qu,
                                          int n_tc, int32_t* __restrict__ rowsum,
                                          __nv_bfloat162& big) {
  const int t = threadIdx.x, r = t >> 2, c0 = (t & 3) * 16;
  const int j = rb * PT + r, kb = cb * PT, k = kb + c0;
  int sum = 0;
  uint32_t b8[4], ht[8], hu[8];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    b8[q] = *reinterpret_cast<const uint32_t*>(&tile[r][c0 + 4 * q]);
    sum = __dp4a((int)b8[q], 0x01010101, sum);
  }
  const int rel = j - k;  // column rel of the 16 is on the diagonal
#pragma unroll
  for (int p = 0; p < 8; ++p) {
    const __nv_bfloat162 one = bf16_pair(b8[p >> 1], p & 1 ? 0x4342 : 0x4140);
    big = __hmax2(big, __habs2(one));
    const uint32_t two = bits_of(__hadd2(one, one));
    if (SIDE != 0) {
      ht[p] = SIDE < 0 ? two : 0;
      hu[p] = SIDE > 0 ? two : 0;
    } else {
      const uint32_t low = (2 * p < rel ? 0xFFFFu : 0) | (2 * p + 1 < rel ? 0xFFFF0000u : 0);
      const uint32_t dia = (2 * p == rel ? 0xFFFFu : 0) | (2 * p + 1 == rel ? 0xFFFF0000u : 0);
      const uint32_t d = bits_of(one) & dia;
      ht[p] = (two & low) | d;
      hu[p] = (two & ~(low | dia)) | d;
    }
  }
  if (j < n && k < ldq)
    *reinterpret_cast<uint4*>(Q8 + (int64_t)j * ldq + k) = make_uint4(b8[0], b8[1], b8[2], b8[3]);
  if (SIDE <= 0 || kb <= qt_kmax(rb * PT)) {
    uint4* dt = reinterpret_cast<uint4*>(Qt + (int64_t)j * n_tc + k);
    dt[0] = make_uint4(ht[0], ht[1], ht[2], ht[3]);
    dt[1] = make_uint4(ht[4], ht[5], ht[6], ht[7]);
  }
  if (SIDE >= 0 || kb >= rb * PT / 256 * 256) {  // the upper block triangle of 256-row blocks
    uint4* du = reinterpret_cast<uint4*>(Qu + (int64_t)j * n_tc + k);
    du[0] = make_uint4(hu[0], hu[1], hu[2], hu[3]);
    du[1] = make_uint4(hu[4], hu[5], hu[6], hu[7]);
  }
  // the row's partial sum over this tile: the 4 threads of row r are lanes
  // 4m .. 4m+3 of one warp
  sum += __shfl_xor_sync(0xffffffffu, sum, 1);
  sum += __shfl_xor_sync(0xffffffffu, sum, 2);
  if ((t & 3) == 0 && j < n && sum != 0) atomicAdd(&rowsum[j], sum);
}

// One symmetric pair of 64 x 64 tiles per block: T = Q[bi rows][bj cols] and
// U = Q[bj rows][bi cols] (bi <= bj; the diagonal tile pairs with itself), so
// every byte of Q is read once.  Both are staged in shared memory four bytes
// at a time; T is compared with U transposed (the symmetry check of problem
// (P)), one 4 x 4 block per thread with byte permutes; then for each of the two
// tiles every thread takes 16 consecutive columns of one row and writes them as
// 16-byte vectors: the int8 copy (rows < n), Q' = 2 tril(Q,-1) + diag(Q) (tiles
// the evaluation reads) and Q'^t = 2 triu(Q,1) + diag(Q) (the upper block
// triangle, which the start-up reads), both in bf16 and zero outside n (so the
// padded squares need no separate clearing), and adds its row's partial sum.  It
// also tracks max|Q|.
// Bound: HBM (n^2 bytes read, about 3.1 n^2 written).  Converting every element
// twice through int -> float -> bf16 and comparing byte by byte made it
// instruction-bound: 60.1 us at n = 6001 (rows not aligned), 50.4 with the packed
// forms, 41.7 with all of a thread's loads before the first use of one and no
// checks on them inside Q (aligned words and a funnel shift where rows are not).
// What is left is the latency of a load phase and a store phase per block, five
// blocks to an SM (eight, with 32 registers, measured slower).
// Which pair a block takes.  Small squares: along the rows, the triangle folded
// into a rectangle (tiles + 1, tiles / 2).  From DIAG_N on: along the diagonals, 2 x 2
// tiles at a time (super-tiles (a, b), b = a + d mod sn for d = 0 .. sn / 2;
// blockIdx.y = d sn + a, the last diagonal, d = sn / 2, only half as long).  Along a
// row a block's second tile lies 64 rows below the previous block's, so hundreds of
// blocks at once touch addresses a multiple of 64 rows apart, which costs the more
// the longer the rows, most of all where they are a power of two.  Preparing, us, by
// rows / by diagonals: n = 12288 197 / 179, n = 14336 309 / 255, n = 16383 566 / 375, n =
// 16384 485 / 373 (446 and 444 before the packed forms).  The lines meet near n = 8000;
// below, an evaluation right behind the preparation finds more of Q' in the L2 after
// the rows (with 100 starts, n = 7000 136 / 139, n = 8192 161 / 159, n = 10240 223 /
// 217).  The number of tiles is a multiple of four, so sn is even.
// (Two kernels: with the choice made inside, 47 registers instead of 40, n = 16384
// prepared in 525.)
constexpr int DIAG_N = 8192;
template <bool W4, bool DIAG>
__global__ void __launch_bounds__(PTHREADS)
prepare_pairs(const int8_t* __restrict__ Q, int n, int64_t ldq_in, int8_t* __restrict__ Q8,
              int64_t ldq, uint16_t* __restrict__ Qt, uint16_t* __restrict__ Qu, int n_tc,
              int32_t* __restrict__ rowsum, unsigned* __restrict__ flags) {
  pdl_enter();
  const int tiles = n_tc / PT;
  int bi = blockIdx.y, bj = (int)blockIdx.x - 1;
  if (DIAG) {
    const int sn = tiles / 2, a = (int)blockIdx.y % sn, b = (a + (int)blockIdx.y / sn) % sn;
    bi = 2 * min(a, b) + (int)blockIdx.x / 2;
    bj = 2 * max(a, b) + (int)blockIdx.x % 2;
    if (bi > bj) return;
  } else if (bj < bi) {
    bi = tiles - 1 - bi;
    bj = tiles - 1 - (int)blockIdx.x;
  }
  __shared__ __align__(16) int8_t tile[2][PT][PT + 4];  // T, then U
  const int t = threadIdx.x;
  const int nt = bi == bj ? 1 : 2;
  {  // thread t loads column word t % 16 of the rows t / 16 + 16 i of both tiles
    constexpr int LR = PTHREADS * 4 / PT, LN = PT / LR;
    const int lr = t >> 4, lc = (t & 15) * 4;
    uint32_t v[2][LN];
    if (bj * PT + PT + 4 <= n && (W4 || bi > 0 || ((uintptr_t)Q & 3) == 0)) {
      // every word, and the aligned word after it, is inside its row (and the
      // aligned word before the first one inside Q): no checks
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int8_t* p = Q + (int64_t)((u ? bj : bi) * PT + lr) * ldq_in + (u ? bi : bj) * PT + lc;
        const unsigned off = W4 ? 0u : (unsigned)((uintptr_t)p & 3);  // LR rows: a multiple of 4
        p -= off;
        if (u < nt) {
#pragma unroll
          for (int i = 0; i < LN; ++i) {
            const uint32_t* q = reinterpret_cast<const uint32_t*>(p + i * LR * ldq_in);
            v[u][i] = W4 ? __ldg(q) : __funnelshift_r(__ldg(q), __ldg(q + 1), 8 * off);
          }
        }
      }
    } else {
      const int8_t* end = Q + (int64_t)(n - 1) * ldq_in + n;
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int i = 0; i < LN; ++i)
          v[u][i] = row_word<W4>(Q, end, ldq_in, n, (u ? bj : bi) * PT + lr + i * LR,
                                 (u ? bi : bj) * PT + lc);
    }
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (u < nt) {
#pragma unroll
        for (int i = 0; i < LN; ++i)
          *reinterpret_cast<uint32_t*>(&tile[u][lr + i * LR][lc]) = v[u][i];
      }
  }
  __syncthreads();
  unsigned asym = 0;
  {  // rows 4a .. 4a+3, columns 4c .. 4c+3 of T against the same block of U^t
    const int a = t >> 4, c = t & 15;
    uint32_t T[4], U[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      T[i] = *reinterpret_cast<const uint32_t*>(&tile[0][4 * a + i][4 * c]);
      U[i] = *reinterpret_cast<const uint32_t*>(&tile[nt - 1][4 * c + i][4 * a]);
    }
    const uint32_t p0 = __byte_perm(U[0], U[1], 0x5140), p1 = __byte_perm(U[2], U[3], 0x5140);
    const uint32_t p2 = __byte_perm(U[0], U[1], 0x7362), p3 = __byte_perm(U[2], U[3], 0x7362);
    asym = (T[0] ^ __byte_perm(p0, p1, 0x5410)) | (T[1] ^ __byte_perm(p0, p1, 0x7632)) |
           (T[2] ^ __byte_perm(p2, p3, 0x5410)) | (T[3] ^ __byte_perm(p2, p3, 0x7632));
  }
  __nv_bfloat162 big = __floats2bfloat162_rn(0.f, 0.f);
  if (nt == 1) {
    emit_tile<0>(tile[0], bi, bj, n, Q8, ldq, Qt, Qu, n_tc, rowsum, big);
  } else {
    emit_tile<1>(tile[0], bi, bj, n, Q8, ldq, Qt, Qu, n_tc, rowsum, big);
    emit_tile<-1>(tile[1], bj, bi, n, Q8, ldq, Qt, Qu, n_tc, rowsum, big);
  }
  const unsigned any = __ballot_sync(0xffffffffu, asym != 0);
  const int amax = __reduce_max_sync(
      0xffffffffu, (int)fmaxf(__low2float(big), __high2float(big)));
  if ((t & 31) == 0) {
    if (any) atomicAdd(&flags[0], 1u);
    atomicMax(&flags[1], (unsigned)amax);
  }
}

// Zeroes what prepare_pairs adds to or leaves out, in one launch: the row sums,
// the error word and the two flags behind it, and the int8 copy's columns
// n_tc .. ldq (outside the tiles).
__global__ void __launch_bounds__(PTHREADS)
prepare_clear(int32_t* __restrict__ rowsum, unsigned* __restrict__ err, int8_t* __restrict__ Q8,
              int64_t ldq, int n, int n_tc) {
  pdl_release();
  const int64_t i0 = (int64_t)blockIdx.x * PTHREADS + threadIdx.x,
                step = (int64_t)gridDim.x * PTHREADS;
  for (int64_t i = i0; i < n; i += step) rowsum[i] = 0;
  if (i0 < 3) err[i0] = 0;
  const int per = (int)(ldq - n_tc) / 16;  // 16-byte pieces per row, 0 to 48
  for (int64_t i = i0; i < (int64_t)n * per; i += step)
    *reinterpret_cast<uint4*>(Q8 + i / per * ldq + n_tc + i % per * 16) = make_uint4(0, 0, 0, 0);
}

// Bit j of x0 is set when row j's sum is positive: a warp reads 32 sums and
// votes.  (One thread per word read 64 sums one after the other: 8.7 us at
// n = 6001, 2.3 now.)
__global__ void __launch_bounds__(PTHREADS)
first_derivative_bits(const int32_t* __restrict__ rowsum, int n, int W,
                      uint64_t* __restrict__ x0) {
  pdl_enter();
  const int j = blockIdx.x * PTHREADS + threadIdx.x;
  const unsigned bits = __ballot_sync(0xffffffffu, j < n && rowsum[j] > 0);
  if ((threadIdx.x & 31) == 0 && j < W * 64)
    reinterpret_cast<uint32_t*>(x0)[j >> 5] = bits;
}

template <bool W4, bool DIAG>
cudaError_t launch_pairs(const int8_t* Q, int n, int64_t ldq_in, ubqp_q* h, cudaStream_t st) {
  const int tiles = h->n_tc / PT, sn = tiles / 2;
  const dim3 grid = DIAG ? dim3(4, sn * (sn + 1) / 2) : dim3(tiles + 1, sn);
  return launch_pdl(prepare_pairs<W4, DIAG>, grid, dim3(PTHREADS), 0, st, Q, n, ldq_in, h->Q8,
                    h->ldq, h->Qt, h->Qu, h->n_tc, h->rowsum, h->scratch_flags);
}

}  // namespace

cudaError_t launch_prepare(const int8_t* Q, int n, int64_t ldq_in, ubqp_q* h,
                           cudaStream_t st) {
  const int64_t work = std::max<int64_t>(h->n, (int64_t)h->n * (h->ldq - h->n_tc) / 16);
  prepare_clear<<<(unsigned)std::min<int64_t>((work + PTHREADS - 1) / PTHREADS,
                                              8ll * h->sm_count),
                  PTHREADS, 0, st>>>(h->rowsum, h->err, h->Q8, h->ldq, n, h->n_tc);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const bool w4 = ((uintptr_t)Q & 3) == 0 && (ldq_in & 3) == 0;
  if (h->n_tc >= DIAG_N)
    e = w4 ? launch_pairs<true, true>(Q, n, ldq_in, h, st)
           : launch_pairs<false, true>(Q, n, ldq_in, h, st);
  else
    e = w4 ? launch_pairs<true, false>(Q, n, ldq_in, h, st)
           : launch_pairs<false, false>(Q, n, ldq_in, h, st);
  if (e != cudaSuccess) return e;
  return launch_pdl(first_derivative_bits, dim3((unsigned)((h->W * 64 + PTHREADS - 1) / PTHREADS)),
                    dim3(PTHREADS), 0, st, h->rowsum, n, h->W, h->x0);
}

}  // namespace ubqp
