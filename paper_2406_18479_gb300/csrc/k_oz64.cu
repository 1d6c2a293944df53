// FP64-accurate complex GEMM on tcgen05 tensor cores through exact integer digits.
//
// GB300 issues 2 FP64 FMAs per clock and SM (1.25 TFLOP/s), 1/900 of its bf16 tensor rate, so an
// FP64 product is cheaper as a sum of exact bf16 products (the error-free splitting of Ozaki et
// al.). C(m, n) = alpha sum_k A(m, k) B(n, k) over complex k is taken as a real GEMM: one operand
// (P) is embedded as two real rows (re, -im), (im, re) per complex row over 2 K real k, the other
// (Q) as its plain real row (re, im); the product of the two gives (Re C, Im C) in adjacent rows,
// which is the memory order of a complex output.
//
// Each row is scaled by one power of two 2^E above its largest |re|, |im| and rounded to
//   N = round(x 2^(62 - E)) = sum_i d_i 256^(7 - i),   d_i in [-128, 127], i = 0..7
// (residual 2^-63 of the row's scale, 2^10 finer than FP64's own rounding of its largest
// element). Digits are exact in bf16. Products of order o = i + j are summed in their own FP32
// accumulator over at most 128 real k: |sum| <= 8 * 128 * 2^14 = 2^24, exact whatever order the
// tensor core adds in. The 8 accumulators (o = 0..7; higher orders are below 2^-59) are joined
// into a 96-bit integer, summed over the chunks of 128 k without rounding, and brought to FP64 at the
// end. The result does not depend on tiling or batching.
//
// The error of K complex terms is at most K 2^-58 2^Ep 2^Eq: it goes with the largest elements of the two
// rows, an FP64 sum's (at most K 2^-52 sum |p| |q|) with the terms. Where the large elements of one row meet
// the small ones of the other the digits hold too little. So every output has a lower bound
// S <= sum |p| |q| 2^-(Ep + Eq) made for it (oz64_bound_kernel: one bf16 product of the magnitudes), and those
// with S < 2^-6 (but not 0: then every term is exactly 0) are left to the FP64 pipe:
// no output has a larger error bound than an FP64 sum of its terms. Transforms avoid the case through a power of
// two per k that moves the grading of the matrix's columns into the input (ZGemm::kexp).
//
// Bound: the L2 reads of the digit tiles at long K (48 KB per k-step of a 128 x 64 tile, 5.5 TB/s), the
// epilogue's three FP64 operations an output at short K. 27 TFLOP/s of complex products at long K (R of a
// molecule, nao = 45) and 16 where the output is as large as the work (transforms), against 0.7..1.1 on
// the FP64 pipe. P0 of a 2x2x2 solid (nao = 26, naux = 104, 80 nodes): 313 -> 21.9 ms; Sigma of a molecule
// (nao = 45): 76.9 -> 5.3 ms; the two transforms of a 3x3x3 solid (naux = 200, 100 nodes): 198 -> 19 ms with
// their packing. Error against 64-bit references on these: 2e-16 and 4e-16 (FP64 pipe: 3e-15 and 6e-15).
//
// Rows with a non-finite element, or whose scale lies outside 2^+-480 (where the scaled product
// could over- or underflow), carry a NaN scale, and outputs that meet one are left as well, so infinities, NaN and
// extreme ranges behave as in zgemm_fp64. The epilogue leaves an output alone, and the CTA computes it after its last
// tile (plain_tiles): a loop over K in the epilogue itself would keep the CTA's other warps in waits that give up
// after 4 s, reached from K of about 10^6.
//
// Kernels
//   oz64_pack_kernel  FP64 views -> digit tiles, in the order the tensor core reads shared memory
//                     (8-row x 16-byte core matrices, no swizzle): a k-step of a tile is one
//                     contiguous block, moved by one bulk copy, no tensor map
//   oz64_bound_kernel the bound S of every output, one bit for each that is left
//   oz64_gemm_kernel  persistent GEMM, 128 real rows of P x NT rows of Q per tile. The 8 digit
//                     tiles of Q lie behind one another in N, and the accumulator of order o in
//                     TMEM columns [o NT, (o + 1) NT): one MMA of digit i of P against the digits
//                     0..7-i of Q (N = (8 - i) NT, split at 256) adds every product of row i to its
//                     order at once: 8 to 12 wide MMAs per 16 k instead of 36 narrow ones.
#include <algorithm>
#include <cmath>

#include "gw_internal.h"
#include "tc_ptx.cuh"

namespace gwi {

namespace {

constexpr int kDigits = 8;
constexpr int kK = 16;              // real k per MMA
constexpr int kChunkSteps = 8;      // k-steps per exact chunk (128 real k)
constexpr int kPTile = 64;          // complex rows of P per tile (128 TMEM lanes)
constexpr int kScaleMax = 480;      // |E| beyond this has no digit form
constexpr int kEpiWarps = 16;
constexpr int kSegSteps = 8;        // least k-steps of a packing segment
constexpr int kMaxSegs = 32;
constexpr int kSplitTiles = 608;    // tiles of a split-K launch, at most (four waves)
constexpr int kMaxSplit = 16;
constexpr int kMagTile = 128;       // rows of a tile of magnitudes
constexpr int kMagK = 16;           // complex k of one of its steps
constexpr int kMagStep = kMagTile * kMagK * 2;   // bytes of a step
constexpr float kLeastSum = 0.015625f;           // S below which the digits hold too little
constexpr int kMapBits = 1024;      // of a CTA's map of units with outputs that are left (a warp's lanes x 32)

// x / d for x < 2^31: multiply-high (see FastDiv in k_mixed.cu)
struct Div {
  unsigned long long m = 1ull << 31;
  int sh = 31, d = 1 << 30;
};
Div make_div(int d) {
  Div f;
  int l = 0;
  while ((1ll << l) < d) ++l;
  f.d = d;
  f.sh = 31 + l;
  f.m = ((1ull << f.sh) + (unsigned long long)d - 1) / (unsigned long long)d;
  return f;
}
__device__ __forceinline__ int div_by(int x, const Div& f) {
  return (int)(((unsigned long long)(unsigned)x * f.m) >> f.sh);
}

// one operand: element (r, k) of batch (bo, bi) as in ZGemm, and where its digit tiles go
struct Side {
  const double2* src = nullptr;
  ZBatch b;
  long long rs_in = 0, rs_out = 0, ks_in = 0, ks_out = 0;
  Div rdiv, kdiv;
  int row0 = 0, rows = 0, tiles = 0;    // rows [row0, row0 + rows) of this launch
  int dep_o = 0, dep_i = 0;             // whether the operand varies with the outer / inner batch index
  int no = 1, ni = 1;                   // packed batches
  unsigned char* dst = nullptr;
  double* scale = nullptr;              // per packed row: 2^(E - 34), NaN: no digit form
  unsigned long long* pmax = nullptr;   // segs > 1: largest |value| bits of each row and K segment
  // magnitudes max(|re|, |im|) 2^-E, bf16 rounded down: tiles of 128 rows (the last of what is left, in eights), steps of 16 k
  unsigned char* mag = nullptr;
  int mtiles = 0;                       // tiles of a packed batch
  const int* kexp = nullptr;            // element (r, k) counts as x 2^(ksign e) (ZGemm::kexp)
  int ksign = 0, kbatch = 0;
};

struct Job {
  Side p, q;
  int K = 0, nks = 0;                   // complex k; k-steps of 16 real k
  int nms = 0;                          // steps of 16 complex k of the magnitudes
  int segs = 1, seg_steps = 0;          // packing: K segments per row tile, k-steps of one
  int o0 = 0, i0 = 0, no = 1, ni = 1;   // batch range of this launch: bo in [o0, o0 + no), bi likewise
  double2* C = nullptr;
  ZBatch bc;
  // output element of P row a, Q row b: cp(a) + cq(b)
  long long cp_in = 0, cp_out = 0, cq_in = 0, cq_out = 0;
  Div cp_div, cq_div;
  double alpha = 1.0;
  int accumulate = 0;
  int skip0 = 0, skip1 = 0;             // outputs with both indices in [skip0, skip1) are not written
  // split K: ksplit CTAs share a tile, each summing split_chunks chunks; their 96-bit integers meet in
  // part ([tile][split][column][128 lanes], hi and lo apart), and the last to arrive (a counter per
  // tile and epilogue warp) adds them, exactly, and writes the output
  int ksplit = 1, split_chunks = 0;
  long long* part_hi = nullptr;
  uint32_t* part_lo = nullptr;
  unsigned int* counter = nullptr;
  uint32_t* left = nullptr;             // [tile][64 rows of P][NT / 32]: bit c: column c is left to plain_tiles
  int* status = nullptr;
};

// bytes of one step of tile t of the magnitudes; where the tile begins
__device__ __forceinline__ int mag_step(const Side& s, int t) { return min(kMagTile, (s.rows - t * kMagTile + 7) / 8 * 8) * (2 * kMagK); }
__device__ __forceinline__ unsigned char* mag_tile(const Side& s, int nms, int batch, int t) {
  return s.mag + (long long)nms * (2 * kMagK) * ((long long)batch * ((s.rows + 7) / 8 * 8) + (long long)t * kMagTile);
}

__device__ __forceinline__ long long side_row(const Side& s, int r) {
  const int rq = div_by(r, s.rdiv);
  return (long long)rq * s.rs_out + (long long)(r - rq * s.rdiv.d) * s.rs_in;
}
__device__ __forceinline__ long long side_k(const Side& s, int k) {
  const int kq = div_by(k, s.kdiv);
  return (long long)kq * s.ks_out + (long long)(k - kq * s.kdiv.d) * s.ks_in;
}
__device__ __forceinline__ long long batch_in(const ZBatch& b, int bi) {
  return b.tab ? b.tab[bi] : (long long)(b.list ? b.list[bi] : bi) * b.bs_in;
}
__device__ __forceinline__ const double2* side_base(const Side& s, int bo, int bi) {
  return s.src + batch_in(s.b, bi) + (long long)bo * s.b.bs_out;
}

constexpr int kExpMax = 400;          // of ZGemm::kexp: no over- or underflow of ordinary values
template <bool KX>
__device__ __forceinline__ double2 side_elem(const Side& s, const double2* row, const int* kexp, int k) {
  double2 x = row[side_k(s, k)];
  if (KX) {
    const int b = kexp[k], e = b == 0 || b == 2047 ? 0 : max(-kExpMax, min(kExpMax, b - 1022));
    const double f = __longlong_as_double((long long)(1023 + s.ksign * e) << 52);
    x = make_double2(x.x * f, x.y * f);
  }
  return x;
}

// round(x 2^(62 - E)) + 0x80..80 for |x| < 2^E: byte 7 - i of the result is digit i plus 128
__device__ __forceinline__ unsigned long long digits_of(double x, int E) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)((bits >> 52) & 0x7FF);
  const unsigned long long m = ex ? ((bits & 0xFFFFFFFFFFFFFull) | (1ull << 52)) : 0ull;
  const int sh = E + 1013 - ex;                  // x = m 2^(ex - 1075): right shift, >= -9
  unsigned long long n;
  if (sh <= 0) n = m << -sh;
  else n = sh > 54 ? 0ull : (m + (1ull << (sh - 1))) >> sh;
  const unsigned long long neg = (unsigned long long)((long long)bits >> 63);
  return ((n ^ neg) - neg) + 0x8080808080808080ull;
}

// max(|re|, |im|) 2^-E < 1 as bf16, rounded down, from the leading words of digits_of; what is below 2^-22 but not
// zero counts as 2^-60, so that a sum of products is zero only where every product is
__device__ __forceinline__ uint32_t magnitude(double2 x, unsigned long long re, unsigned long long im) {
  const int a = abs((int)((uint32_t)(re >> 32) - 0x80808080u)), b = abs((int)((uint32_t)(im >> 32) - 0x80808080u));
  const float m = __int2float_rz(max(a, b)) * 9.313225746154785e-10f;     // 2^-30
  return max(a, b) >= 256 ? __float_as_uint(m) >> 16 : x.x != 0.0 || x.y != 0.0 ? 67u << 7 : 0u;
}

// digit j (0: leading) of four words as two bf16 pairs
__device__ __forceinline__ float digit_f(unsigned long long u, int j) {
  const uint32_t w = j < 4 ? (uint32_t)(u >> 32) : (uint32_t)u;
  const uint32_t b = (w >> (24 - 8 * (j & 3))) & 0xFFu;
  return __fsub_rn(__uint_as_float(0x4B000000u | b), 8388736.0f);     // 2^23 + b - (2^23 + 128)
}
__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi) {   // both exact in bf16
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

// One block per row tile, packed batch and K segment. A thread owns one row and every
// (256 / RT)-th group of four complex k (8 real k: one 16-byte piece of a core-matrix row per digit).
// The row's scale needs a pass over the row first: within the block where it covers all of K, by
// oz64_scale_kernel (a maximum per segment) where long rows are split so that few row tiles still
// fill the GPU. Bound: memory (16 bytes read twice, 64 (P) or 32 (Q) written per complex element);
// neighbouring lanes hold neighbouring rows, so that a digit's 8 rows make one 128-byte line.
template <int kRows>
struct PackPos {
  int tile, pb, seg, row, grp, k0, k1;   // this block's tile, batch and segment; this thread's row and group
  long long prow;
  bool row_ok;
  const double2* src;
  const int* kexp;
  __device__ PackPos(const Side& s, const Job& j, long long t) {
    seg = (int)(t % j.segs);
    t /= j.segs;
    tile = (int)(t % s.tiles);
    pb = (int)(t / s.tiles);
    row = threadIdx.x % kRows;
    grp = threadIdx.x / kRows;
    const int r = tile * kRows + row;
    row_ok = r < s.rows;
    src = side_base(s, j.o0 + pb / s.ni, j.i0 + pb % s.ni) + (row_ok ? side_row(s, s.row0 + r) : 0);
    kexp = s.kexp + (long long)(j.i0 + pb % s.ni) * s.kbatch;
    prow = ((long long)pb * s.tiles + tile) * kRows + row;
    k0 = seg * j.seg_steps;              // k-steps [k0, k1) of the segment
    k1 = min(j.nks, k0 + j.seg_steps);
  }
};

template <int kRows, bool KX>
__device__ __forceinline__ unsigned long long row_max(const Side& s, const Job& j, const PackPos<kRows>& p) {
  constexpr int kGroups = 256 / kRows;
  unsigned long long mx = 0;
  if (p.row_ok) {
    const int kend = min(j.K, 8 * p.k1);
    for (int k = 8 * p.k0 + p.grp * 4; k < kend; k += kGroups * 4) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (k + u >= kend) break;
        const double2 x = side_elem<KX>(s, p.src, p.kexp, k + u);
        mx = max(mx, max((unsigned long long)__double_as_longlong(x.x) & 0x7FFFFFFFFFFFFFFFull,
                         (unsigned long long)__double_as_longlong(x.y) & 0x7FFFFFFFFFFFFFFFull));
      }
    }
  }
  __shared__ unsigned long long red[256];
  red[threadIdx.x] = mx;
  __syncthreads();
#pragma unroll
  for (int g = 0; g < kGroups; ++g) mx = max(mx, red[g * kRows + p.row]);
  return mx;
}

template <int kRows, bool KX>
__device__ void scale_tile(const Side& s, const Job& j, long long t) {
  const PackPos<kRows> p(s, j, t);
  const unsigned long long mx = row_max<kRows, KX>(s, j, p);
  if (p.grp == 0) s.pmax[p.prow * j.segs + p.seg] = mx;
}

template <int RT, bool PSIDE, bool KX>
__device__ void pack_tile(const Side& s, const Job& j, long long t) {
  constexpr int kRows = PSIDE ? kPTile : RT;      // complex rows of the tile
  constexpr int kReal = PSIDE ? 2 * kPTile : RT;  // real rows of the tile
  constexpr int kGroups = 256 / kRows;
  const PackPos<kRows> p(s, j, t);
  unsigned long long mx = 0;
  if (j.segs == 1) {
    mx = row_max<kRows, KX>(s, j, p);
  } else {
    for (int g = 0; g < j.segs; ++g) mx = max(mx, s.pmax[p.prow * j.segs + g]);
  }
  const int ex = (int)(mx >> 52);
  int E = ex - 1022;
  const bool plain = mx != 0 && (ex == 0x7FF || E > kScaleMax || E < -kScaleMax);
  const bool zero = mx == 0 || plain;
  if (zero) E = 0;
  if (p.grp == 0 && p.seg == 0)
    s.scale[p.prow] = plain ? __longlong_as_double(0x7FF8000000000000ll)
                            : __longlong_as_double((long long)(E - 34 + 1023) << 52);
  unsigned char* base = s.dst + ((long long)p.pb * s.tiles + p.tile) * j.nks * (long long)(kDigits * kReal * 32);
  const int rr = PSIDE ? 2 * p.row : p.row;
  // the padding rows of the last tile stay unwritten: a row of digits meets only its own row of the output
  if (!p.row_ok) return;
  const int mrow = p.tile * kRows + p.row;
  const int mstep = mag_step(s, mrow / kMagTile);
  unsigned char* mag = mag_tile(s, j.nms, p.pb, mrow / kMagTile) + (mrow % kMagTile >> 3) * 256 + (mrow & 7) * 16;
  auto mag_at = [&](int g) { return reinterpret_cast<uint2*>(mag + (long long)(g >> 2) * mstep + (g >> 1 & 1) * 128 + (g & 1) * 8); };
  if (p.k1 == j.nks && (j.nks & 1) && p.grp < 2) *mag_at(2 * j.nks + p.grp) = make_uint2(0u, 0u);   // half a step beyond K
  for (int g = 2 * p.k0 + p.grp; g < 2 * p.k1; g += kGroups) {
    unsigned long long u[8];
    uint32_t m[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int k = 4 * g + c;
      double2 x = make_double2(0.0, 0.0);
      if (!zero && k < j.K) x = side_elem<KX>(s, p.src, p.kexp, k);
      u[2 * c] = digits_of(x.x, E);
      u[2 * c + 1] = digits_of(x.y, E);
      m[c] = magnitude(x, u[2 * c], u[2 * c + 1]);
    }
    *mag_at(g) = make_uint2(m[0] | m[1] << 16, m[2] | m[3] << 16);
    unsigned char* d = base + (long long)(g >> 1) * (kDigits * kReal * 32) + (rr >> 3) * 256 + (g & 1) * 128 +
                       (rr & 7) * 16;
#pragma unroll
    for (int q = 0; q < kDigits; ++q) {
      uint32_t w[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) w[c] = bf16_pair(digit_f(u[2 * c], q), digit_f(u[2 * c + 1], q));
      uint4* o = reinterpret_cast<uint4*>(d + q * (kReal * 32));
      if (PSIDE) {   // rows (re, -im) and (im, re)
        o[0] = make_uint4(w[0] ^ 0x80000000u, w[1] ^ 0x80000000u, w[2] ^ 0x80000000u, w[3] ^ 0x80000000u);
        o[1] = make_uint4(__funnelshift_l(w[0], w[0], 16), __funnelshift_l(w[1], w[1], 16),
                          __funnelshift_l(w[2], w[2], 16), __funnelshift_l(w[3], w[3], 16));
      } else {
        o[0] = make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
  }
}

template <int NT, bool KX>
__global__ void __launch_bounds__(256) oz64_scale_kernel(const __grid_constant__ Job j) {
  const long long np = (long long)j.p.tiles * j.p.no * j.p.ni * j.segs;
  if (blockIdx.x < np) scale_tile<kPTile, KX>(j.p, j, blockIdx.x);
  else scale_tile<NT, KX>(j.q, j, blockIdx.x - np);
}

template <int NT, bool KX>
__global__ void __launch_bounds__(256) oz64_pack_kernel(const __grid_constant__ Job j) {
  asm volatile("griddepcontrol.launch_dependents;");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const long long np = (long long)j.p.tiles * j.p.no * j.p.ni * j.segs;
  if (blockIdx.x < np) pack_tile<2 * kPTile, true, KX>(j.p, j, blockIdx.x);
  else pack_tile<NT, false, KX>(j.q, j, blockIdx.x - np);
}

// bits of the columns c, c + 1, .. (n <= 32) within [skip0, skip1)
__device__ __forceinline__ uint32_t skip_bits(const Job& j, int c, int n) {
  const int lo = min(max(j.skip0 - c, 0), n), hi = min(max(j.skip1 - c, 0), n);
  return (uint32_t)((1ull << hi) - (1ull << lo));
}

// The outputs of this CTA's tiles that are left to the FP64 pipe, every sum in order of k as in zgemm_fp64_kernel.
// Tiles with a few of them (kFew at most) go into one list, a thread per output; a tile of many goes 32 x 32 at a time, a
// group of 256 threads each, staged through shared memory, 2 x 2 outputs a thread (a warp skips those that none of its
// lanes needs). R = P~ V of a molecule (nao = 36, naux = 125), 3e-4 of its outputs left, one in a quarter of the
// 32 x 32 pieces: 153 us a launch with pieces only, 106 with the list, 62 if nothing were left.
// Of CTAs that share a tile's K the first takes it. sm: the stages.
constexpr int kPlainK = 16, kPlainGroups = kEpiWarps / 8;
constexpr int kFew = 128, kListMax = 8192, kUnitsMax = 16384;        // of a tile; entries; tiles looked over at a time
constexpr size_t kPlainStage = 2 * kPlainK * 33 * sizeof(double2) + 256;   // of a group
constexpr size_t kPlainSmem = kPlainGroups * kPlainStage + kListMax * 8 + kUnitsMax * 4 + 16;
template <int NT>
__device__ __noinline__ void plain_tiles(const Job& j, int ksplit, const uint32_t* map, int map_sh, int tid, unsigned char* sm) {
  constexpr int kThreads = 32 * kEpiWarps, kWords = NT / 32;
  const int group = tid >> 8, gid = tid & 255, warp = tid >> 5, lane = tid & 31;
  unsigned char* stage = sm + group * kPlainStage;
  double2(*Ps)[33] = reinterpret_cast<double2(*)[33]>(stage);
  double2(*Qs)[33] = Ps + kPlainK;
  uint32_t* s_left = reinterpret_cast<uint32_t*>(Qs + kPlainK);         // left columns of each row; whether any
  int2* list = reinterpret_cast<int2*>(sm + kPlainGroups * kPlainStage);   // outputs: tile, row * 64 + column
  int* many = reinterpret_cast<int*>(list + kListMax);                  // tiles with many
  int* counts = many + kUnitsMax;                                       // of list and many
  auto sync = [&] { asm volatile("bar.sync %0, 256;" ::"r"(1 + group) : "memory"); };
  auto sync_all = [&] { asm volatile("bar.sync 3, %0;" ::"n"(kThreads) : "memory"); };
  constexpr int kSub = 2 * (NT / 32);                 // 32 x 32 pieces of a GEMM tile
  const int per_batch = j.p.tiles * j.q.tiles, total = per_batch * j.no * j.ni * ksplit;
  const int owned = (total - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
  auto mac = [](double2& s, double2 x, double2 y) {
    s.x = fma(-x.y, y.y, fma(x.x, y.x, s.x));
    s.y = fma(x.y, y.x, fma(x.x, y.y, s.y));
  };
  auto put = [&](int bo, int bi, int a, int c, double2 v) {              // output of P row a, Q row c
    const int aq = div_by(a, j.cp_div), cq = div_by(c, j.cq_div);
    double2* at = j.C + batch_in(j.bc, bi) + (long long)bo * j.bc.bs_out + (long long)aq * j.cp_out +
                  (long long)(a - aq * j.cp_div.d) * j.cp_in + (long long)cq * j.cq_out + (long long)(c - cq * j.cq_div.d) * j.cq_in;
    double2 x = make_double2(j.alpha * v.x, j.alpha * v.y);
    if (j.accumulate) {
      const double2 old = *at;
      x.x += old.x;
      x.y += old.y;
    }
    *at = x;
  };
#pragma unroll 1
  for (int own0 = 0; own0 < owned; own0 += kUnitsMax) {
    if (tid < 2) counts[tid] = 0;
    sync_all();
    // ---- a warp per tile: its outputs into the list, or the tile among those with many
#pragma unroll 1
    for (int own = own0 + warp; own < min(owned, own0 + kUnitsMax); own += kEpiWarps) {
      if (!(map[own >> map_sh >> 5] >> (own >> map_sh & 31) & 1)) continue;
      const int unit = blockIdx.x + own * gridDim.x, tile = unit / ksplit;
      if (unit != tile * ksplit) continue;
      const int pt = tile % per_batch / j.q.tiles;
      uint32_t w[2 * kWords];
      int n = 0;
#pragma unroll
      for (int u = 0; u < 2 * kWords; ++u) {
        const int word = u * 32 + lane;
        w[u] = pt * kPTile + word / kWords < j.p.rows ? j.left[(long long)tile * kPTile * kWords + word] : 0u;
        n += __popc(w[u]);
      }
      int before = n;                      // outputs of the lanes up to this one
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, before, o);
        if (lane >= o) before += x;
      }
      const int all = __shfl_sync(0xffffffffu, before, 31);
      if (all == 0) continue;
      int first = kListMax;
      if (all <= kFew) {
        if (lane == 0) first = atomicAdd(&counts[0], all);
        first = __shfl_sync(0xffffffffu, first, 0);
      }
      if (first + all > kListMax) {        // no room, or many
        if (lane == 0) many[atomicAdd(&counts[1], 1)] = tile;
        for (int e = first + lane; e < kListMax && e < first + all; e += 32) list[e] = make_int2(-1, 0);
        continue;
      }
      int at = first + before - n;
#pragma unroll
      for (int u = 0; u < 2 * kWords; ++u)
        for (uint32_t x = w[u]; x; x &= x - 1) {
          const int word = u * 32 + lane;
          list[at++] = make_int2(tile, word / kWords * 64 + word % kWords * 32 + __ffs(x) - 1);
        }
    }
    sync_all();
    // ---- the list, a thread per output, 4 k in flight
    const int listed = min(counts[0], kListMax);
#pragma unroll 1
    for (int e = tid; e < listed; e += kThreads) {
      const int2 x = list[e];
      if (x.x < 0) continue;
      const int b = x.x / per_batch, w = x.x - b * per_batch, o = b / j.ni, i = b - o * j.ni;
      const int pt = w / j.q.tiles, qt = w - pt * j.q.tiles, bo = j.o0 + o, bi = j.i0 + i;
      const int a = j.p.row0 + pt * kPTile + x.y / 64, c = j.q.row0 + qt * NT + x.y % 64;
      const double2* A = side_base(j.p, bo, bi) + side_row(j.p, a);
      const double2* B = side_base(j.q, bo, bi) + side_row(j.q, c);
      double2 acc = make_double2(0.0, 0.0);
#pragma unroll 1
      for (int k0 = 0; k0 < j.K; k0 += 4) {
        double2 p[4], q[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (k0 + k < j.K) {
            p[k] = A[side_k(j.p, k0 + k)];
            q[k] = B[side_k(j.q, k0 + k)];
          }
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (k0 + k < j.K) mac(acc, p[k], q[k]);
      }
      put(bo, bi, a, c, acc);
    }
    // ---- the tiles with many
    const int tx = gid & 15, ty = gid >> 4, nmany = counts[1];
#pragma unroll 1
    for (int piece = group; piece < nmany * kSub; piece += kPlainGroups) {
      const int tile = many[piece / kSub], sub = piece % kSub;
      const int b = tile / per_batch, w = tile - b * per_batch, o = b / j.ni, i = b - o * j.ni;
      const int pt = w / j.q.tiles, qt = w - pt * j.q.tiles;
      const int p0 = (sub & 1) * 32, q0 = (sub >> 1) * 32;        // of the tile
      const int np = min(32, j.p.rows - pt * kPTile - p0), nq = min(32, j.q.rows - qt * NT - q0);
      if (np <= 0 || nq <= 0) continue;
      sync();
      if (gid < 32) {
        s_left[gid] = gid < np ? j.left[((long long)tile * kPTile + p0 + gid) * kWords + q0 / 32] : 0u;
        const bool any = __any_sync(0xffffffffu, s_left[gid] != 0);
        if (gid == 0) s_left[32] = any;
      }
      sync();
      if (!s_left[32]) continue;
      bool need[2][2];
      double2 acc[2][2];
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          need[u][v] = s_left[2 * tx + u] >> (2 * ty + v) & 1;
          acc[u][v] = make_double2(0.0, 0.0);
        }
      const int bo = j.o0 + o, bi = j.i0 + i;
      const double2* A = side_base(j.p, bo, bi);
      const double2* B = side_base(j.q, bo, bi);
      const int pr = j.p.row0 + pt * kPTile + p0, qr = j.q.row0 + qt * NT + q0;
      const bool pk = j.p.ks_in == 1, qk = j.q.ks_in == 1;         // neighbouring threads on neighbouring elements
#pragma unroll 1
      for (int k0 = 0; k0 < j.K; k0 += kPlainK) {
        sync();
#pragma unroll
        for (int e = gid; e < 32 * kPlainK; e += 256) {
          const int rp = pk ? e / kPlainK : e % 32, kp = pk ? e % kPlainK : e / 32;
          const int rq = qk ? e / kPlainK : e % 32, kq = qk ? e % kPlainK : e / 32;
          Ps[kp][rp] = rp < np && k0 + kp < j.K ? A[side_row(j.p, pr + rp) + side_k(j.p, k0 + kp)] : make_double2(0.0, 0.0);
          Qs[kq][rq] = rq < nq && k0 + kq < j.K ? B[side_row(j.q, qr + rq) + side_k(j.q, k0 + kq)] : make_double2(0.0, 0.0);
        }
        sync();
        const int kn = min(kPlainK, j.K - k0);
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int v = 0; v < 2; ++v) {
            if (!need[u][v]) continue;
            double2 x = acc[u][v];
#pragma unroll 4
            for (int k = 0; k < kn; ++k) mac(x, Ps[k][2 * tx + u], Qs[k][2 * ty + v]);
            acc[u][v] = x;
          }
      }
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int v = 0; v < 2; ++v)
          if (need[u][v]) put(bo, bi, pr + 2 * tx + u, qr + 2 * ty + v, acc[u][v]);
    }
    sync_all();
  }
}

template <int NT>
struct Oz64Shape {
  static constexpr int kABytes = kDigits * 128 * 32;            // one k-step of a P tile
  static constexpr int kBBytes = kDigits * NT * 32;             // and of a Q tile
  static constexpr int kStageBytes = kABytes + kBBytes;
  static constexpr int kStages = NT == 64 ? 4 : 5;
  static constexpr int kBufCols = kDigits * NT;
  static constexpr int kBufs = 512 / kBufCols;                  // accumulator sets in TMEM
  static constexpr int kThreads = 64 + 32 * kEpiWarps;          // producer, MMA, epilogue warps
  static constexpr size_t kSmem = 128 + (size_t)kStages * kStageBytes + 512;
  static_assert(kSmem <= 232448, "stages exceed shared memory");
  static_assert(kPlainSmem <= (size_t)kStages * kStageBytes, "plain_tiles works in the stages");
};

// K-major operand without swizzle: 8 x 16-byte core matrices, 128 bytes between the two k halves
// (leading offset), 256 bytes between 8-row groups (stride offset)
__device__ __forceinline__ uint64_t core_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
  d |= (uint64_t)(128 >> 4) << 16;
  d |= (uint64_t)(256 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// old + alpha 2^e (hi 2^32 + lo) for |hi|, |lo| < 2^51: the integers become FP64 by an addition to the bits
// of 1.5 2^52 (scaled by 2^e) and that is taken off again, exactly; no branch and three FP64 operations,
// so that a thread's outputs overlap (the general form, to_fp64, is 200 instructions in a row)
__device__ __forceinline__ double finish(long long hi, long long lo, int e, double alpha, double old) {
  const long long es = (long long)e << 52;
  const double h = __longlong_as_double(0x4338000000000000ll + hi + es);
  const double l = __longlong_as_double(0x4338000000000000ll + lo + es);
  const double k = __longlong_as_double(0x4538000000180000ll + es);      // 2^e (1.5 2^84 + 1.5 2^52)
  return fma(fma(h, 4294967296.0, -k) + l, alpha, old);
}
constexpr int kFinishSteps = 64 * kChunkSteps;     // k-steps up to which hi stays below 2^51

// the exact integer accumulators a_o of one chunk as hi 2^32 + lo = sum_o a_o 256^(7 - o)
__device__ __forceinline__ void join_chunk(const float (&v)[kDigits][4], int u, long long& hi, long long& lo) {
  int a[kDigits];
#pragma unroll
  for (int o = 0; o < kDigits; ++o) a[o] = __float2int_rn(v[o][u]);
  // leading digits are within 64, so |a0| <= 2^19, |a1| <= 2^21, |a2| <= 2^22: no overflow in 32 bits
  hi = (long long)(a[0] * 256 + a[1]) * 65536 + (a[2] * 256 + a[3]);
  lo = (long long)a[4] * 16777216 + (long long)a[5] * 65536 + (long long)a[6] * 256 + a[7];
}

// the same, added to a running hi 2^32 + lo with 0 <= lo < 2^32
__device__ __forceinline__ void join_orders(const float (&v)[kDigits][4], int u, long long& hi, uint32_t& lo) {
  long long h, l;
  join_chunk(v, u, h, l);
  l += (long long)(unsigned long long)lo;
  hi += h + (l >> 32);
  lo = (uint32_t)l;
}

// (hi 2^32 + lo) 2^e rounded to FP64, in integer arithmetic, for sums of any length
__device__ __forceinline__ double to_fp64(long long hi, uint32_t lo, int e) {
  const long long neg = hi >> 63;
  unsigned long long H = (unsigned long long)(hi ^ neg);
  uint32_t L = lo ^ (uint32_t)neg;
  if (neg) {                                   // two's complement of the 96 bits
    L += 1u;
    H += L == 0u;
  }
  if (H == 0) {
    if (L == 0) return 0.0;
    H = (unsigned long long)L << 32;
    L = 0;
    e -= 64;
  }
  const int lz = __clzll((long long)H);
  H = (H << lz) | (((unsigned long long)L << 32) >> 1 >> (63 - lz));
  const unsigned long long m = (H >> 11) + ((H >> 10) & 1ull);      // 53 bits, rounded half up
  const int E = 52 + 43 - lz + e + 1023;
  if (E < 1 || E > 2045) {                     // beyond the normal range: rare
    const double x = scalbn((double)m, 43 - lz + e);
    return neg ? -x : x;
  }
  return __longlong_as_double((long long)((((unsigned long long)(E - 1) << 52) + m) | ((unsigned long long)neg & (1ull << 63))));
}

// S of every output: magnitudes of 128 rows of P times 128 rows of Q, summed over K in one FP32 accumulator (truncated,
// so from below), two tiles in flight. Long K in two passes: 512 of its k spread evenly, which is enough for every output
// of most tiles, then all of it for the other tiles (P0 of a 2x2x2 solid, 13 tiles of K = 5408: 10 us, 50 for all of it).
// Bound: launch and copy latency; 1/70 of the digit MMAs and 1/30 of their bytes, and one load and compare an output.
// Steps lie behind one another in shared memory as in global memory; where a tile has fewer than 128 rows an MMA reads on
// into the next ones, for rows and columns that are not there.
constexpr int kMagStages = 3, kMagPer = 4;           // stages, steps of a stage
constexpr int kMagFirst = 8;                         // stages of a first pass (512 k)
constexpr int kMagThreads = 192;                     // producer, MMA, four epilogue warps
constexpr size_t kMagSmem = 128 + (size_t)kMagStages * kMagPer * 2 * kMagStep + 384;
template <int NT>
__global__ void __launch_bounds__(kMagThreads) oz64_bound_kernel(const __grid_constant__ Job j) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
  constexpr int kHalf = kMagPer * kMagStep;          // P's part of a stage
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + (size_t)kMagStages * 2 * kHalf);
  uint64_t* empty = full + kMagStages;
  uint64_t* acc_full = empty + kMagStages;           // [2]
  uint64_t* acc_empty = acc_full + 2;
  uint64_t* drain_bar = acc_full + 4;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_full + 5);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  uint32_t* map = tmem_slot + 2;                     // tiles for a second pass, as in oz64_gemm_kernel
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kMagStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], 4);
    }
    mbar_init(drain_bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 2) map[lane] = 0;
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(256));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  asm volatile("griddepcontrol.launch_dependents;");
  asm volatile("griddepcontrol.wait;" ::: "memory");   // the packing
  const int per_batch = j.p.mtiles * j.q.mtiles, total = per_batch * j.no * j.ni;
  auto packed = [](const Side& s, int b, int ni) {
    const int o = b / ni, i = b - o * ni;
    return (s.dep_o ? o : 0) * s.ni + (s.dep_i ? i : 0);
  };
  const int nstages = (j.nms + kMagPer - 1) / kMagPer;
  const int npass = nstages > kMagFirst ? 2 : 1;
  int map_sh = 0;
  while ((total / (int)gridDim.x) >> map_sh >= kMapBits) ++map_sh;
  uint32_t step = 0, n = 0;           // stages and tiles so far (of a role)
  bool ok = true;
#pragma unroll 1
  for (int pass = 0; pass < npass; ++pass) {
    // the stages of this pass: all, or kMagFirst spread over K
    const int ns = npass == 2 && pass == 0 ? kMagFirst : nstages;
    auto stage_at = [&](int s) { return ns == nstages ? s : (int)((long long)s * (nstages - 1) / (kMagFirst - 1)); };
    auto steps_of = [&](int s) { return min(kMagPer, j.nms - s * kMagPer); };
    if (warp == 0) {
      if (lane == 0) {
        int own = 0;
        for (int tile = blockIdx.x; tile < total && !*abort_flag; tile += gridDim.x, ++own) {
          if (pass && !(map[own >> map_sh >> 5] >> (own >> map_sh & 31) & 1)) continue;
          const int b = tile / per_batch, w = tile - b * per_batch, pt = w / j.q.mtiles, qt = w - pt * j.q.mtiles;
          const unsigned char* a = mag_tile(j.p, j.nms, packed(j.p, b, j.ni), pt);
          const unsigned char* q = mag_tile(j.q, j.nms, packed(j.q, b, j.ni), qt);
          const int pb = mag_step(j.p, pt), qb = mag_step(j.q, qt);
          for (int i = 0; i < ns; ++i, ++step) {
            const int st = step % kMagStages, s = stage_at(i), nk = steps_of(s);
            if (!mbar_wait(&empty[st], ((step / kMagStages) & 1) ^ 1, abort_flag, j.status, 25)) break;
            uint8_t* sa = smem + (size_t)st * 2 * kHalf;
            mbar_expect_tx(&full[st], nk * (pb + qb));
            bulk_load(sa, a + (long long)s * kMagPer * pb, nk * pb, &full[st]);
            bulk_load(sa + kHalf, q + (long long)s * kMagPer * qb, nk * qb, &full[st]);
          }
        }
      }
    } else if (warp == 1) {
      if (lane == 0) {
        const uint64_t desc0 = core_desc(smem_u32(smem));
        int own = 0;
        for (int tile = blockIdx.x; tile < total && ok; tile += gridDim.x, ++own) {
          if (pass && !(map[own >> map_sh >> 5] >> (own >> map_sh & 31) & 1)) continue;
          const int w = tile % per_batch, pb = mag_step(j.p, w / j.q.mtiles), qb = mag_step(j.q, w % j.q.mtiles);
          const uint32_t buf = n & 1;
          if (!mbar_wait(&acc_empty[buf], ((n >> 1) & 1) ^ 1, abort_flag, j.status, 26)) { ok = false; break; }
          ++n;
          tc_fence_after();
          for (int i = 0; i < ns; ++i, ++step) {
            const int st = step % kMagStages, nk = steps_of(stage_at(i));
            if (!mbar_wait(&full[st], (step / kMagStages) & 1, abort_flag, j.status, 27)) { ok = false; break; }
            tc_fence_after();
            const uint64_t sa = desc0 + (uint64_t)((st * 2 * kHalf) >> 4);
            for (int k = 0; k < nk; ++k)
              mma_bf16(tmem + buf * kMagTile, sa + (uint64_t)(k * pb >> 4), sa + (uint64_t)((kHalf + k * qb) >> 4),
                       idesc_bf16(kMagTile, false), i == 0 && k == 0 ? 0u : 1u);
            mma_commit(&empty[st]);
          }
          if (ok) mma_commit(&acc_full[buf]);
        }
      }
    } else {
      const int quarter = warp & 3;
      int own = 0;
      for (int tile = blockIdx.x; tile < total && ok; tile += gridDim.x, ++own) {
        if (pass && !(map[own >> map_sh >> 5] >> (own >> map_sh & 31) & 1)) continue;
        const int b = tile / per_batch, w = tile - b * per_batch, pt = w / j.q.mtiles, qt = w - pt * j.q.mtiles;
        const int r = pt * kMagTile + quarter * 32 + lane;
        const bool row_ok = r < j.p.rows;
        const bool row_bad = row_ok && isnan(j.p.scale[(long long)packed(j.p, b, j.ni) * j.p.tiles * kPTile + r]);
        const double* sq = j.q.scale + (long long)packed(j.q, b, j.ni) * j.q.tiles * NT;
        uint32_t* left = j.left + ((long long)(b * j.p.tiles + r / kPTile) * j.q.tiles * kPTile + r % kPTile) * (NT / 32);
        uint32_t bad[kMagTile / 32], in[kMagTile / 32];   // columns without a digit form, columns there are
#pragma unroll
        for (int g = 0; g < kMagTile / 32; ++g) {
          const int c = qt * kMagTile + g * 32 + lane;
          in[g] = __ballot_sync(0xffffffffu, c < j.q.rows);
          bad[g] = __ballot_sync(0xffffffffu, c < j.q.rows && isnan(sq[c]));
        }
        const uint32_t buf = n & 1;
        if (!mbar_wait(&acc_full[buf], (n >> 1) & 1, abort_flag, j.status, 28)) { ok = false; break; }
        ++n;
        tc_fence_after();
        bool again = false;               // below the bound with part of K
#pragma unroll
        for (int g = 0; g < kMagTile / 32; ++g) {
          float v[32];
#pragma unroll
          for (int u = 0; u < 32; u += 8) tmem_ld8(tmem + ((uint32_t)(quarter * 32) << 16) + buf * kMagTile + g * 32 + u, v + u);
          tmem_wait_ld();
          if (g == kMagTile / 32 - 1) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[buf]);
          }
          const int c0 = qt * kMagTile + g * 32;
          uint32_t m = 0, z = 0;
#pragma unroll
          for (int u = 0; u < 32; ++u) {
            m |= (v[u] < kLeastSum ? 1u : 0u) << u;
            z |= (v[u] == 0.0f ? 1u : 0u) << u;
          }
          again |= (row_ok && !row_bad ? m & ~bad[g] & in[g] : 0u) != 0;
          m = (row_bad ? ~0u : (m & ~z) | bad[g]) & in[g];
          if (j.p.row0 + r >= j.skip0 && j.p.row0 + r < j.skip1) m &= ~skip_bits(j, j.q.row0 + c0, 32);
          if (row_ok && c0 < j.q.tiles * NT)
            left[(long long)(c0 / NT) * kPTile * (NT / 32) + (c0 % NT) / 32] = m;
        }
        if (ns < nstages && __any_sync(0xffffffffu, again) && lane == 0) atomicOr(&map[own >> map_sh >> 5], 1u << (own >> map_sh & 31));
      }
    }
    __syncthreads();
  }
  if (warp == 0 && lane == 0 && *abort_flag) {   // let every issued copy land before the CTA exits (bounded)
    const uint64_t t0 = globaltimer();
    for (int k = 0; k < kMagStages && step > (uint32_t)k; ++k) {
      const uint32_t s2 = step - 1 - k;
      while (!mbar_try(&full[s2 % kMagStages], (s2 / kMagStages) & 1) && globaltimer() - t0 < kWaitLimitNs) {
      }
    }
  }
  if (warp == 1 && lane == 0) {
    mma_commit(drain_bar);   // the last MMAs end before TMEM is released
    const uint64_t t0 = globaltimer();
    while (!mbar_try(drain_bar, 0) && globaltimer() - t0 < kWaitLimitNs) {
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256));
}

template <int NT, bool MULTI>
__global__ void __launch_bounds__(64 + 32 * kEpiWarps, 1) oz64_gemm_kernel(const __grid_constant__ Job j) {
  using S = Oz64Shape<NT>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + (size_t)S::kStages * S::kStageBytes);
  uint64_t* empty = full + S::kStages;
  uint64_t* acc_full = empty + S::kStages;      // [kBufs]
  uint64_t* acc_empty = acc_full + 2;
  uint64_t* drain_bar = acc_full + 4;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_full + 5);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  // which of this CTA's units have outputs that are left to plain_tiles: a bit for 2^map_sh units in order
  uint32_t* map = tmem_slot + 2;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < S::kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < S::kBufs; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], kEpiWarps);
    }
    mbar_init(drain_bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 2) map[lane] = 0;
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  asm volatile("griddepcontrol.wait;" ::: "memory");   // the bounds (and the packing, which they wait for)
  const int per_batch = j.p.tiles * j.q.tiles;
  const int ksplit = MULTI ? j.ksplit : 1;
  const int total = per_batch * j.no * j.ni * ksplit;
  int map_sh = 0;
  while ((total / (int)gridDim.x) >> map_sh >= kMapBits) ++map_sh;
  // work unit -> batch, P tile, Q tile (Q fastest: neighbouring CTAs share the larger P tile in L2),
  // and its k-steps [s0, s1)
  auto split = [&](int unit, int& o, int& i, int& pt, int& qt, int& s0, int& s1) {
    const int tile = MULTI ? unit / ksplit : unit;
    s0 = 0;
    s1 = j.nks;
    if (MULTI && ksplit > 1) {
      s0 = (unit - tile * ksplit) * j.split_chunks * kChunkSteps;
      s1 = min(j.nks, s0 + j.split_chunks * kChunkSteps);
    }
    const int b = tile / per_batch, w = tile - b * per_batch;
    o = b / j.ni;
    i = b - o * j.ni;
    pt = w / j.q.tiles;
    qt = w - pt * j.q.tiles;
  };
  auto packed = [](const Side& s, int o, int i) { return (s.dep_o ? o : 0) * s.ni + (s.dep_i ? i : 0); };

  if (warp == 0) {
    if (lane == 0) {
      uint32_t step = 0;
      for (int tile = blockIdx.x; tile < total && !*abort_flag; tile += gridDim.x) {
        int o, i, pt, qt, s0, s1;
        split(tile, o, i, pt, qt, s0, s1);
        const unsigned char* a = j.p.dst + ((long long)packed(j.p, o, i) * j.p.tiles + pt) * j.nks * (long long)S::kABytes;
        const unsigned char* b = j.q.dst + ((long long)packed(j.q, o, i) * j.q.tiles + qt) * j.nks * (long long)S::kBBytes;
        for (int s = s0; s < s1; ++s, ++step) {
          const int st = step % S::kStages;
          if (!mbar_wait(&empty[st], ((step / S::kStages) & 1) ^ 1, abort_flag, j.status, 21)) break;
          mbar_expect_tx(&full[st], S::kStageBytes);
          uint8_t* sa = smem + (size_t)st * S::kStageBytes;
          bulk_load(sa, a + (long long)s * S::kABytes, S::kABytes, &full[st]);
          bulk_load(sa + S::kABytes, b + (long long)s * S::kBBytes, S::kBBytes, &full[st]);
        }
      }
      if (*abort_flag) {   // let every issued copy land before the CTA exits (bounded)
        const uint64_t t0 = globaltimer();
        for (int k = 0; k < S::kStages && step > (uint32_t)k; ++k) {
          const uint32_t s2 = step - 1 - k;
          while (!mbar_try(&full[s2 % S::kStages], (s2 / S::kStages) & 1) && globaltimer() - t0 < kWaitLimitNs) {
          }
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      uint32_t step = 0, chunk = 0;
      const uint64_t desc0 = core_desc(smem_u32(smem));
      bool ok = true;
      for (int tile = blockIdx.x; tile < total && ok; tile += gridDim.x) {
        int o, i, pt, qt, s0, s1;
        split(tile, o, i, pt, qt, s0, s1);
        for (int s = s0; s < s1 && ok; ++s, ++step) {
          const bool start = (s % kChunkSteps) == 0;
          const uint32_t buf = chunk % S::kBufs;
          if (start) {
            if (!mbar_wait(&acc_empty[buf], ((chunk / S::kBufs) & 1) ^ 1, abort_flag, j.status, 22)) { ok = false; break; }
            tc_fence_after();
          }
          const int st = step % S::kStages;
          if (!mbar_wait(&full[st], (step / S::kStages) & 1, abort_flag, j.status, 23)) { ok = false; break; }
          tc_fence_after();
          const uint64_t sa = desc0 + (uint64_t)((st * S::kStageBytes) >> 4);
          const uint64_t sb = sa + (uint64_t)(S::kABytes >> 4);
          const uint32_t d = tmem + buf * S::kBufCols;
#pragma unroll
          for (int i = 0; i < kDigits; ++i) {
            // digits 0..7-i of Q, at most 256 columns per MMA; digit 0 of P opens every order
            constexpr int kPer = 256 / NT;
#pragma unroll
            for (int q = 0; q < kDigits - i; q += kPer) {
              const int nq = kDigits - i - q < kPer ? kDigits - i - q : kPer;
              mma_bf16(d + (uint32_t)((i + q) * NT), sa + (uint64_t)(i * 128 * 32 >> 4),
                       sb + (uint64_t)(q * NT * 32 >> 4), idesc_bf16(nq * NT, false), start && i == 0 ? 0u : 1u);
            }
          }
          mma_commit(&empty[st]);
          if ((s % kChunkSteps) == kChunkSteps - 1 || s == s1 - 1) {
            mma_commit(&acc_full[buf]);
            ++chunk;
          }
        }
      }
      mma_commit(drain_bar);   // the last MMAs end before TMEM is released
      const uint64_t t0 = globaltimer();
      while (!mbar_try(drain_bar, 0) && globaltimer() - t0 < kWaitLimitNs) {
      }
    }
  } else {
    // epilogue: TMEM lane quarter warp % 4, columns [half kCols, (half + 1) kCols). 16 warps: each output
    // is a long chain (8 conversions, the joins, three FP64 operations), and two warps a scheduler
    // left it idle three clocks in four
    const int quarter = warp & 3, half = (warp - 2) >> 2;
    constexpr int kCols = NT * 4 / kEpiWarps;
    const int lrow = quarter * 32 + lane;
    const int part = lrow & 1;
    uint32_t chunk = 0;
    int own = 0;
    // this warp's columns of the row that are left to plain_tiles, read a unit ahead
    auto left_at = [&](int tile) {
      return j.left[((long long)(MULTI ? tile / ksplit : tile) * kPTile + (lrow >> 1)) * (NT / 32) + half * kCols / 32];
    };
    uint32_t left_next = blockIdx.x < total ? left_at(blockIdx.x) : 0u;
    for (int tile = blockIdx.x; tile < total; tile += gridDim.x, ++own) {
      int o, i, pt, qt, s0, s1;
      split(tile, o, i, pt, qt, s0, s1);
      const int nchunks = (s1 - s0 + kChunkSteps - 1) / kChunkSteps;
      const int bo = j.o0 + o, bi = j.i0 + i;
      const int pr = pt * kPTile + (lrow >> 1);
      const bool p_ok = pr < j.p.rows;
      // biased exponents of the scales
      const int ep = __double2hiint(j.p.scale[((long long)packed(j.p, o, i) * j.p.tiles + pt) * kPTile + (lrow >> 1)]) >> 20;
      const double* sq = j.q.scale + ((long long)packed(j.q, o, i) * j.q.tiles + qt) * NT;
      const int ap = j.p.row0 + (p_ok ? pr : 0), apq = div_by(ap, j.cp_div);
      double* C = reinterpret_cast<double*>(j.C + batch_in(j.bc, bi) + (long long)bo * j.bc.bs_out + (long long)apq * j.cp_out +
                                            (long long)(ap - apq * j.cp_div.d) * j.cp_in) + part;
      // output element of tile column col (P row fixed per thread)
      auto at = [&](int col) {
        const int aq = j.q.row0 + qt * NT + col, aqq = div_by(aq, j.cq_div);
        return C + 2 * ((long long)aqq * j.cq_out + (long long)(aq - aqq * j.cq_div.d) * j.cq_in);
      };
      auto col_ok = [&](int col) { return p_ok && qt * NT + col < j.q.rows; };
      uint32_t left = left_next >> (half * kCols % 32) & ((1u << kCols) - 1);
      if (tile + (int)gridDim.x < total) left_next = left_at(tile + gridDim.x);
      const bool mark = p_ok && left;
      if (!MULTI && j.p.row0 + pr >= j.skip0 && j.p.row0 + pr < j.skip1) left |= skip_bits(j, j.q.row0 + qt * NT + half * kCols, kCols);
      const bool quick = j.nks <= kFinishSteps;
      auto put = [&](int col, long long hi, long long lo, double old) {
        const int eq = col_ok(col) ? __double2hiint(sq[col]) >> 20 : 1023;
        const int e = ep + eq - 2046;
        const double x = !MULTI || quick ? finish(hi, lo, e, j.alpha, old)
                                         : fma(to_fp64(hi, (uint32_t)lo, e), j.alpha, old);
        if (col_ok(col) && !(left >> (col - half * kCols) & 1)) *at(col) = x;
      };
      // outputs that are added to are read ahead of the wait for the accumulators (a load behind every
      // store would put 16 memory latencies in a row: 24k clocks a tile instead of 5k)
      constexpr int kAhead = MULTI ? 1 : kCols;
      double old[kAhead];
#pragma unroll
      for (int u = 0; u < kAhead; ++u) old[u] = 0.0;
      if (!MULTI && j.accumulate) {
#pragma unroll
        for (int u = 0; u < kAhead; ++u)
          if (col_ok(half * kCols + u)) old[u] = *at(half * kCols + u);
      }
      long long hi[MULTI ? kCols : 1];
      uint32_t lo[MULTI ? kCols : 1];
      bool ok = true;
      for (int c = 0; c < nchunks; ++c, ++chunk) {
        const uint32_t buf = chunk % S::kBufs;
        if (!mbar_wait(&acc_full[buf], (chunk / S::kBufs) & 1, abort_flag, j.status, 24)) { ok = false; break; }
        tc_fence_after();
        const uint32_t tb = tmem + ((uint32_t)(quarter * 32) << 16) + buf * S::kBufCols + half * kCols;
#pragma unroll
        for (int g = 0; g < kCols / 4; ++g) {
          float v[kDigits][4];
#pragma unroll
          for (int d = 0; d < kDigits; ++d) tmem_ld4(tb + d * NT + 4 * g, v[d]);
          tmem_wait_ld();
          if (g == kCols / 4 - 1) {       // this warp's columns are in registers: release TMEM
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[buf]);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            if constexpr (MULTI) {
              if (c == 0) hi[4 * g + u] = 0, lo[4 * g + u] = 0;
              join_orders(v, u, hi[4 * g + u], lo[4 * g + u]);
            } else {
              long long h, l;
              join_chunk(v, u, h, l);
              put(half * kCols + 4 * g + u, h, l, old[4 * g + u]);
            }
          }
        }
      }
      if (!ok) break;
      if constexpr (MULTI) {
        if (ksplit > 1) {
          const int t = tile / ksplit, me = tile - t * ksplit;
          const long long at = ((long long)t * ksplit + me) * NT * 128 + (long long)half * kCols * 128 + lrow;
#pragma unroll
          for (int u = 0; u < kCols; ++u) {
            j.part_hi[at + u * 128] = hi[u];
            j.part_lo[at + u * 128] = lo[u];
          }
          // every warp meets its counterparts of the other splits on a counter of its own: no wait
          __threadfence();
          __syncwarp();
          unsigned int n = 0;
          if (lane == 0) {
            n = atomicAdd(&j.counter[t * kEpiWarps + warp - 2], 1u);
            if (n == (unsigned)ksplit - 1) j.counter[t * kEpiWarps + warp - 2] = 0;   // ready for the next launch
          }
          if (me == 0 && __any_sync(0xffffffffu, mark) && lane == 0) atomicOr(&map[own >> map_sh >> 5], 1u << (own >> map_sh & 31));
          if (__shfl_sync(0xffffffffu, n, 0) != (unsigned)ksplit - 1) continue;
          __threadfence();
          for (int m = 0; m < ksplit; ++m) {
            if (m == me) continue;
            const long long from = ((long long)t * ksplit + m) * NT * 128 + (long long)half * kCols * 128 + lrow;
#pragma unroll
            for (int u = 0; u < kCols; ++u) {
              const unsigned long long l = (unsigned long long)lo[u] + __ldcg(&j.part_lo[from + u * 128]);
              hi[u] += __ldcg(&j.part_hi[from + u * 128]) + (long long)(l >> 32);
              lo[u] = (uint32_t)l;
            }
          }
        }
#pragma unroll
        for (int u0 = 0; u0 < kCols; u0 += 4) {
          double o4[4] = {0.0, 0.0, 0.0, 0.0};
          if (j.accumulate) {
#pragma unroll
            for (int u = 0; u < 4; ++u)
              if (col_ok(half * kCols + u0 + u)) o4[u] = *at(half * kCols + u0 + u);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) put(half * kCols + u0 + u, hi[u0 + u], lo[u0 + u], o4[u]);
        }
      }
      if (__any_sync(0xffffffffu, mark) && lane == 0) atomicOr(&map[own >> map_sh >> 5], 1u << (own >> map_sh & 31));
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
  if (!*abort_flag && warp >= 2 && __any_sync(0xffffffffu, map[lane] != 0)) plain_tiles<NT>(j, ksplit, map, map_sh, threadIdx.x - 64, smem);
}

int sm_count() {
  static const int n = [] {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return std::max(v, 1);
  }();
  return n;
}

// Launch whose blocks may start while the kernel before it ends (its launch latency, TMEM allocation and barriers
// under that kernel's tail); they wait for it (griddepcontrol.wait) before they touch memory. A small evaluation
// (nao = 8, 8 products): 384 -> 353 us.
template <class... A>
void launch_after(void (*k)(A...), long long grid, int threads, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k, args...);
}

template <int NT, bool KX>
void launch_pack(const Job& j, long long np, long long nq, cudaStream_t st) {
  if (j.segs > 1) {
    prof_begin(SLOT_LIMBS, st);
    oz64_scale_kernel<NT, KX><<<(unsigned)((np + nq) * j.segs), 256, 0, st>>>(j);
    prof_end(SLOT_LIMBS, st, 0.0, ((double)np * kPTile + (double)nq * NT) * 16.0 * j.K);
  }
  prof_begin(SLOT_LIMBS, st);
  oz64_pack_kernel<NT, KX><<<(unsigned)((np + nq) * j.segs), 256, 0, st>>>(j);
  prof_end(SLOT_LIMBS, st, 0.0, ((double)np * kPTile * (32.0 + 64.0) + (double)nq * NT * (32.0 + 32.0)) * 8.0 * j.nks);
}

template <int NT, bool MULTI>
int launch_gemm(const Job& j, int slot, cudaStream_t st) {
  using S = Oz64Shape<NT>;
  static const bool attr = cudaFuncSetAttribute(oz64_gemm_kernel<NT, MULTI>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                (int)S::kSmem) == cudaSuccess &&
                           cudaFuncSetAttribute(oz64_bound_kernel<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                (int)kMagSmem) == cudaSuccess;
  if (!attr) return fail(GW_ECUDA, "oz64_gemm: shared memory attribute refused");
  const long long total = (long long)j.p.tiles * j.q.tiles * j.no * j.ni * j.ksplit;
  const long long np = (long long)j.p.tiles * j.p.no * j.p.ni, nq = (long long)j.q.tiles * j.q.no * j.q.ni;
  if (total > 2147483647LL || (np + nq) * j.segs > 2147483647LL) return fail(GW_EINVAL, "oz64_gemm: too many tiles");
  if (j.p.kexp) launch_pack<NT, true>(j, np, nq, st);
  else launch_pack<NT, false>(j, np, nq, st);
  const long long mags = (long long)j.p.mtiles * j.q.mtiles * j.no * j.ni;
  prof_begin(SLOT_LIMBS, st);
  launch_after(oz64_bound_kernel<NT>, std::min<long long>(mags, 2LL * sm_count()), kMagThreads, kMagSmem, st, j);
  prof_end(SLOT_LIMBS, st, 0.0, (double)mags * j.nms * 2 * kMagStep);
  prof_begin(slot, st);
  launch_after(oz64_gemm_kernel<NT, MULTI>, std::min<long long>(total, sm_count()), S::kThreads, S::kSmem, st, j);
  // algorithmic flops: 8 per complex multiply-add
  prof_end(slot, st, 8.0 * j.p.rows * (double)j.q.rows * j.K * j.no * j.ni,
           (double)total / j.ksplit * j.nks * S::kStageBytes);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? GW_OK : fail(GW_ECUDA, "oz64_gemm launch: %s", cudaGetErrorString(e));
}

Side make_side(const double2* src, const ZView& v, const ZBatch& b, int no, int ni) {
  Side s;
  s.src = src;
  s.b = b;
  s.rs_in = v.rs_in;
  s.rs_out = v.rs_out;
  s.ks_in = v.ks_in;
  s.ks_out = v.ks_out;
  s.rdiv = make_div(v.rin);
  s.kdiv = make_div(v.kin);
  s.dep_o = no > 1 && b.bs_out != 0;
  s.dep_i = ni > 1 && (b.tab || b.bs_in != 0);
  return s;
}

inline long long up(long long x, long long m) { return (x + m - 1) / m * m; }

}  // namespace

size_t oz64_counter_bytes() { return (size_t)kSplitTiles * kEpiWarps * sizeof(unsigned int); }

size_t oz64_bytes(long long p_rows, long long q_rows, int K) {
  const long long nks = (K + 7) / 8;
  // digit tiles (64-row Q tiles bound the padding) and scales; magnitudes; a bit for every output
  const long long extra = 8 + (nks >= 2 * kSegSteps ? 8 * kMaxSegs : 0), mag = (nks + 1) / 2 * 2 * kMagK;
  return (size_t)(up(p_rows, kPTile) * (nks * 512 + extra) + up(q_rows, 64) * (nks * 256 + extra) +
                  (up(p_rows, 8) + up(q_rows, 8)) * mag + up(p_rows, kPTile) * up(q_rows, 64) / 8 + 1024);
}

// Where digits pay: below 8 complex k most of a k-step is padding, and tiny products (under 2^13
// complex multiply-adds per matrix) stay on the FP64 pipe for their single launch. The rule looks
// at one matrix only (g.unit where several share a product), so that batch sizes and tau batches
// never change a result.
bool oz64_takes(const ZGemm& g) {
  return g.ws && g.ws->mem && g.K >= 8 && (g.unit > 0.0 ? g.unit : (double)g.M * g.N * g.K) >= 8192.0;
}

int zgemm_oz64(const ZGemm& g, void* stream, bool* done) {
  *done = false;
  cudaStream_t st = (cudaStream_t)stream;
  const int ni = std::min(g.bin, g.nbatch), no = (g.nbatch + ni - 1) / ni;
  if (no * (long long)ni != g.nbatch) return GW_OK;
  // P, the embedded side, is the one whose output index is contiguous in memory
  const bool p_is_b = g.vc.ks_in == 1 || g.vc.rs_in != 1;
  Job j;
  j.p = p_is_b ? make_side(g.B, g.vb, g.bb, no, ni) : make_side(g.A, g.va, g.ba, no, ni);
  j.q = p_is_b ? make_side(g.A, g.va, g.ba, no, ni) : make_side(g.B, g.vb, g.bb, no, ni);
  if (g.kexp) {
    j.p.kexp = j.q.kexp = g.kexp;
    j.p.kbatch = j.q.kbatch = g.kexp_batch;
    j.p.ksign = p_is_b ? -g.kexp_a : g.kexp_a;
    j.q.ksign = -j.p.ksign;
  }
  const int pr = p_is_b ? g.N : g.M, qr = p_is_b ? g.M : g.N;
  j.K = g.K;
  j.nks = (g.K + 7) / 8;
  j.nms = (j.nks + 1) / 2;
  j.C = g.C;
  j.bc = g.bc;
  j.alpha = g.alpha;
  j.accumulate = g.accumulate;
  j.skip0 = g.skip0;
  j.skip1 = g.skip1;
  if (g.skip1 > g.skip0 && j.nks > kChunkSteps) return fail(GW_EINVAL, "oz64_gemm: a block of outputs is spared in products of one chunk");
  j.status = g.ws->status;
  const Div rd = make_div(g.vc.rin), kd = make_div(g.vc.kin);
  j.cp_div = p_is_b ? kd : rd;
  j.cp_in = p_is_b ? g.vc.ks_in : g.vc.rs_in;
  j.cp_out = p_is_b ? g.vc.ks_out : g.vc.rs_out;
  j.cq_div = p_is_b ? rd : kd;
  j.cq_in = p_is_b ? g.vc.rs_in : g.vc.ks_in;
  j.cq_out = p_is_b ? g.vc.rs_out : g.vc.ks_out;
  // 64-column Q tiles halve the operand traffic per product; 32 where K fits one or two chunks (two
  // accumulator sets: the next tile's MMAs run under this one's epilogue) or 64 would pad more
  const int nt = (j.nks > 2 * kChunkSteps && up(qr, 64) == up(qr, 32)) ? 64 : 32;
  // bytes per packed row: digits, scale, and the segment maxima of long rows
  const long long row_extra = 8 + (j.nks >= 2 * kSegSteps ? 8 * kMaxSegs : 0);
  const long long pb = (long long)j.nks * 512 + row_extra, qb = (long long)j.nks * 256 + row_extra, mb = j.nms * 2LL * kMagK;
  const long long W = (long long)g.ws->bytes - 1024;
  auto p_bytes = [&](long long r) { return up(r, kPTile) * pb + up(r, 8) * mb; };
  auto q_bytes = [&](long long r) { return up(r, nt) * qb + up(r, 8) * mb; };
  auto need = [&](long long prow, long long qrow, long long o, long long i) {
    return p_bytes(prow) * (j.p.dep_o ? o : 1) * (j.p.dep_i ? i : 1) + q_bytes(qrow) * (j.q.dep_o ? o : 1) * (j.q.dep_i ? i : 1) +
           o * i * (up(prow, kPTile) * up(qrow, nt) / 8);
  };
  long long go = no, gi = ni, prc = pr, qrc = qr;
  while (go > 1 && need(pr, qr, go, gi) > W) go = (go + 1) / 2;
  while (gi > 1 && need(pr, qr, go, gi) > W) gi = (gi + 1) / 2;
  if (need(pr, qr, go, gi) > W) {
    qrc = std::min<long long>(qr, (W / 2) / qb / nt * nt);
    while (qrc > 0 && q_bytes(qrc) > W / 2) qrc = (qrc - 1) / nt * nt;
    if (qrc <= 0) return GW_OK;
    prc = std::min<long long>(pr, (W - q_bytes(qrc)) / pb / kPTile * kPTile);
    while (prc > 0 && need(prc, qrc, 1, 1) > W) prc = (prc - 1) / kPTile * kPTile;
    if (prc <= 0) return GW_OK;
  }
  *done = true;
  for (long long o0 = 0; o0 < no; o0 += go)
    for (long long i0 = 0; i0 < ni; i0 += gi)
      for (long long q0 = 0; q0 < qr; q0 += qrc)
        for (long long p0 = 0; p0 < pr; p0 += prc) {
          j.o0 = (int)o0;
          j.i0 = (int)i0;
          j.no = (int)std::min(go, no - o0);
          j.ni = (int)std::min(gi, ni - i0);
          for (Side* s : {&j.p, &j.q}) {
            s->no = s->dep_o ? j.no : 1;
            s->ni = s->dep_i ? j.ni : 1;
          }
          j.p.row0 = (int)p0;
          j.p.rows = (int)std::min(prc, pr - p0);
          j.p.tiles = (j.p.rows + kPTile - 1) / kPTile;
          j.q.row0 = (int)q0;
          j.q.rows = (int)std::min(qrc, qr - q0);
          j.q.tiles = (j.q.rows + nt - 1) / nt;
          j.p.mtiles = (j.p.rows + kMagTile - 1) / kMagTile;
          j.q.mtiles = (j.q.rows + kMagTile - 1) / kMagTile;
          const long long pn = (long long)j.p.no * j.p.ni * j.p.tiles * kPTile;
          const long long qn = (long long)j.q.no * j.q.ni * j.q.tiles * nt;
          unsigned char* m = (unsigned char*)g.ws->mem;
          j.p.dst = m;
          j.q.dst = m + pn * j.nks * 512;
          j.p.mag = j.q.dst + qn * j.nks * 256;
          j.q.mag = j.p.mag + (long long)j.p.no * j.p.ni * up(j.p.rows, 8) * mb;
          j.p.scale = reinterpret_cast<double*>(j.q.mag + (long long)j.q.no * j.q.ni * up(j.q.rows, 8) * mb);
          j.q.scale = j.p.scale + pn;
          // long rows are packed in segments where the row tiles alone leave SMs idle (8 blocks an SM)
          const long long blocks = (long long)j.p.no * j.p.ni * j.p.tiles + (long long)j.q.no * j.q.ni * j.q.tiles;
          const int segs = (int)std::min<long long>(std::min(j.nks / kSegSteps, kMaxSegs), (8LL * sm_count() + blocks - 1) / blocks);
          j.seg_steps = (j.nks + std::max(segs, 1) - 1) / std::max(segs, 1);
          j.segs = (j.nks + j.seg_steps - 1) / j.seg_steps;
          j.p.pmax = reinterpret_cast<unsigned long long*>(j.q.scale + qn);
          j.q.pmax = j.p.pmax + (j.segs > 1 ? pn * j.segs : 0);
          // Tiles that leave the last wave short of work (or never fill one) share their chunks of K among
          // CTAs: the split with the least waves times chunks, a chunk's time for each partial sum that is
          // written and read again. The partial sums take what the digits leave of the workspace. 80 tiles
          // of 85 chunks on 152 SMs (P0 of a 2x2x2 solid): 12.5 -> 7.7 ms (with
          // equal tau batches).
          const long long tiles = (long long)j.p.tiles * j.q.tiles * j.no * j.ni;
          j.left = reinterpret_cast<uint32_t*>(j.q.pmax + (j.segs > 1 ? qn * j.segs : 0));
          const int nchunks = (j.nks + kChunkSteps - 1) / kChunkSteps;
          j.ksplit = 1;
          j.part_hi = reinterpret_cast<long long*>(j.left + tiles * kPTile * (nt / 32));
          const long long room = (m + g.ws->bytes - reinterpret_cast<unsigned char*>(j.part_hi)) / (128 * nt * 12);
          if (g.ws->counters && nchunks > 1 && tiles <= kSplitTiles) {
            long long best = (tiles + sm_count() - 1) / sm_count() * nchunks;
            for (int ks = 2; ks <= std::min(nchunks, kMaxSplit) && tiles * ks <= room; ++ks) {
              const int per = (nchunks + ks - 1) / ks, used = (nchunks + per - 1) / per;
              const long long cost = (tiles * used + sm_count() - 1) / sm_count() * (per + 1);
              if (cost < best) {
                best = cost;
                j.split_chunks = per;
                j.ksplit = used;
              }
            }
            j.counter = reinterpret_cast<unsigned int*>(g.ws->counters);
            j.part_lo = reinterpret_cast<uint32_t*>(j.part_hi + tiles * j.ksplit * 128 * nt);
          }
          int rc;
          if (j.nks <= kChunkSteps)
            rc = nt == 64 ? launch_gemm<64, false>(j, g.slot, st) : launch_gemm<32, false>(j, g.slot, st);
          else
            rc = nt == 64 ? launch_gemm<64, true>(j, g.slot, st) : launch_gemm<32, true>(j, g.slot, st);
          if (rc != GW_OK) return rc;
        }
  return GW_OK;
}

}  // namespace gwi
