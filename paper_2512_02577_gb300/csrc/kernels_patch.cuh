// Cartesian vertex-patch smoother as one matrix product per patch (included
// by inst_k.cuh after kernels.cuh).
//
// On a Cartesian mesh the local solver of every patch -- Algorithm 2 around
// the p-multigrid V-cycle of Algorithm 3, full or half -- is the same linear
// map, up to the factor 1 / h^{d-2}: d_j = B r_j / h^{d-2}.  B is formed once
// per method (patch_columns_kernel: the local solver applied to unit
// vectors) and applied here to a block of patches at a time on the tensor
// cores.  The solver commutes with the reflections of the patch in every
// direction, so in the basis of even and odd combinations of mirrored nodes
// B falls into 2^d independent blocks ("sectors") of K or K - 1 rows per
// direction: (K^2 + (K-1)^2)^d products per patch in place of (2K-1)^{2d}.
//
// Why: sum factorisation spends seven short contractions per vmult and moves
// every intermediate through shared memory; in FP64 it is bound by GB300's
// FP64 pipe (1.25 TFLOP/s, two multiply-adds per clock and SM), in FP32 by
// shared-memory traffic and the barriers between the line passes.
//
// FP64 arithmetic (the Ozaki scheme: Ozaki, Ogita, Oishi, Rump, Numer.
// Algorithms 59, 2012): operands in fixed point (one exponent per matrix row
// and per patch, 60 bits of each value), split into 8 signed digits of 8 bits
// that are exact in FP16; products of digits are summed exactly by the tensor
// cores (integers in the FP32 accumulator) and across digit pairs in 64-bit
// integers, keeping the 36 digit pairs i + j <= 7 (0-based).  The matrices are
// formed in pairs of doubles, their results have one exponent per orbit of
// mirrored nodes.  Windows whose values differ too much for one exponent:
// kUnevenExp below.  No FP64 instruction is executed but for subnormal windows
// and results and for spikes.  Largest error of one local solve of a patch in
// units of 2^-53 |B||r|, N(0,1) residuals, by sum factorisation and now: 3D K = 3 3.1,
// 2.4; K = 4 3.5, 3.5; K = 5 3.7, 1.9; 2D K = 7 5.8, 3.4; K = 8 7.7, 5.6; with one
// value of 1e6 among them 24, 20; 900, 400; 270, 130; 960, 360; 960, 380.  FP32:
// three BF16 parts of each value (8 bits each, exact), the six products of
// weight 2^-16 and above.
//
// Patch launch of one sweep, by sum factorisation and now (GB300): FP64 K = 4
// at 32^3 cells 2.343 and 0.229 ms (tensor pipe 30% of its cycles, issue slots
// 46%: the digit conversions and the 64-bit gather and scatter); FP64 K = 5 at
// 24^3 2.12 and 0.36 ms; FP32 K = 4 at 32^3 0.135 and 0.057 ms (shared-memory
// and L1 wavefronts: 69% of their rate), K = 5 at 40^3 0.473 and 0.316 ms, K =
// 3 at 67^3 0.327 and 0.192 ms, K = 2 at 100^3 0.283 and 0.157 ms.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

namespace pmg {
namespace PMG_KNS {

using TP = std::conditional_t<PMG_PREC == 0, double, float>;  // this part's precision

// Sectors of an operator on a window of M nodes per direction (a patch's
// interior, M = 2K - 1, or a cell, M = K + 1): sector s is odd in direction d
// where bit d of s is set.  Even coefficients 0..E-1 (E - 1: the centre node
// if M is odd), odd ones 0..O-1.  Windows of at most 32 nodes are not split:
// their single matrix fits the same number of 16 x 16 tiles.
template <int DIM, int M_>
struct Sectors {
  static constexpr int M = M_;
  static constexpr int NODES = ipow(M, DIM);
  static constexpr bool SPLIT = NODES > 32;
  static constexpr int NS = SPLIT ? 1 << DIM : 1;
  static constexpr int E = SPLIT ? (M + 1) / 2 : M;  // coefficients per direction of an even sector
  static constexpr int O = SPLIT ? M / 2 : 0;        // and of an odd one
  static constexpr bool CENTRE = SPLIT && E > O;     // coordinate E - 1 is its own mirror image
  static constexpr int ORBITS = ipow(E, DIM);      // nodes up to reflection
  static constexpr int IMAGES = SPLIT ? 1 << DIM : 1;
  __host__ __device__ static constexpr int ext(int s, int d) { return d >= DIM ? 1 : ((s >> d) & 1) ? O : E; }
  __host__ __device__ static constexpr int size(int s) { return ext(s, 0) * ext(s, 1) * ext(s, 2); }
  __host__ __device__ static constexpr int tiles(int s) { return (size(s) + 15) / 16; }  // 16-row tiles per side
  // offsets of sector s: padded rows, rows, 16 x 16 tiles
  __host__ __device__ static constexpr int prow(int s) { int o = 0; for (int t = 0; t < s; ++t) o += 16 * tiles(t); return o; }
  __host__ __device__ static constexpr int row(int s) { int o = 0; for (int t = 0; t < s; ++t) o += size(t); return o; }
  __host__ __device__ static constexpr int tile(int s) { int o = 0; for (int t = 0; t < s; ++t) o += tiles(t) * tiles(t); return o; }
  static constexpr int PROWS = prow(NS), ROWS = row(NS), TILES = tile(NS);
  static_assert(ROWS == NODES, "the sectors hold every node once");
};

// An orbit: a node of the first orthant (coordinates 0..E-1) and its mirror
// images; image b is mirrored in the directions of b's bits.
template <int DIM, int M>
struct Orbit {
  using S = Sectors<DIM, M>;
  int c[3];
  __device__ __forceinline__ explicit Orbit(int o) {
    c[0] = o % S::E;
    c[1] = (o / S::E) % S::E;
    c[2] = DIM == 3 ? o / (S::E * S::E) : 0;
  }
  // image b is a node of its own (the centre has no mirror image); likewise
  // the orbit has a coefficient in sector b
  __device__ __forceinline__ bool has(int b) const {
    bool h = true;
#pragma unroll
    for (int d = 0; d < DIM; ++d) h = h && !(S::CENTRE && ((b >> d) & 1) && c[d] == S::E - 1);
    return h;
  }
  __device__ __forceinline__ int at(int d, int b) const { return ((b >> d) & 1) ? S::M - 1 - c[d] : c[d]; }
  __device__ __forceinline__ int node(int b) const {
    return at(0, b) + S::M * (at(1, b) + S::M * (DIM == 3 ? at(2, b) : 0));
  }
  // directions in which the node is central
  __device__ __forceinline__ int centres() const {
    int n = 0;
#pragma unroll
    for (int d = 0; d < DIM; ++d) n += S::CENTRE && c[d] == S::E - 1;
    return n;
  }
};

// Lines of a window along x up to reflection in the other directions: line L
// holds the nodes (0..M-1, c_1, c_2), c_d < E; image b is mirrored in
// direction d where bit d - 1 of b is set.  A thread takes all images of a
// line, so the offsets of its nodes and coefficients along x are immediates.
template <int DIM, int M>
struct Lines {
  using S = Sectors<DIM, M>;
  static constexpr int N = ipow(S::E, DIM - 1);
  static constexpr int IMAGES = S::SPLIT ? 1 << (DIM - 1) : 1;
  int c[2];
  __device__ __forceinline__ explicit Lines(int L) {
    c[0] = L % S::E;
    c[1] = DIM == 3 ? L / S::E : 0;
  }
  __device__ __forceinline__ bool has(int b) const {
    bool h = true;
#pragma unroll
    for (int d = 0; d < DIM - 1; ++d) h = h && !(S::CENTRE && ((b >> d) & 1) && c[d] == S::E - 1);
    return h;
  }
  // directions in which the line passes through the centre
  __device__ __forceinline__ int centres() const {
    return S::CENTRE ? (c[0] == S::E - 1) + (DIM == 3 && c[1] == S::E - 1) : 0;
  }
  // offset of image b's first node on a grid of N1 nodes per direction
  __device__ __forceinline__ int node(int b, int N1) const {
    const int y = (b & 1) ? S::M - 1 - c[0] : c[0], z = (b & 2) ? S::M - 1 - c[1] : c[1];
    return N1 * (y + (DIM == 3 ? N1 * z : 0));
  }
  // first coefficient of the line in sector s
  __device__ __forceinline__ int coef(int s) const { return S::ext(s, 0) * (c[0] + S::ext(s, 1) * c[1]); }
};

// even / odd combinations of a line's images in every direction: entry i of
// image b becomes the coefficient of parity b in the other directions and,
// along x, even coefficient i for i < E, odd coefficient M - 1 - i beyond.
// (Its own inverse up to the factor 2 per direction, which the matrix absorbs.)
template <int DIM, int M, typename V>
__device__ __forceinline__ void reflect(V (&v)[Lines<DIM, M>::IMAGES][M]) {
  using S = Sectors<DIM, M>;
  if constexpr (S::SPLIT) {
#pragma unroll
    for (int b = 0; b < Lines<DIM, M>::IMAGES; ++b)
#pragma unroll
      for (int i = 0; i < S::O; ++i) {
        const V e = v[b][i] + v[b][M - 1 - i], o = v[b][i] - v[b][M - 1 - i];
        v[b][i] = e;
        v[b][M - 1 - i] = o;
      }
#pragma unroll
    for (int d = 0; d < DIM - 1; ++d)
#pragma unroll
      for (int b = 0; b < Lines<DIM, M>::IMAGES; ++b)
        if (!((b >> d) & 1))
#pragma unroll
          for (int i = 0; i < M; ++i) {
            const V e = v[b][i] + v[b | (1 << d)][i], o = v[b][i] - v[b | (1 << d)][i];
            v[b][i] = e;
            v[b | (1 << d)][i] = o;
          }
  }
}

// f(entry, sector, coefficient along x) for the entries of image b after reflect
template <int DIM, int M, class F>
__device__ __forceinline__ void for_coefs(int b, F&& f) {
  using S = Sectors<DIM, M>;
#pragma unroll
  for (int i = 0; i < M; ++i) {
    if (i < S::E) f(i, S::SPLIT ? 2 * b : 0, i);
    else f(i, 2 * b + 1, M - 1 - i);
  }
}

// ---------------------------------------------------------------- block shape
// P windows per block (the n extent of the products), NW warps: the fastest of
// P = 16, 32 and NW = 2..16 in FP32 (K = 4 at 32^3: 0.055 ms, 0.061 with P =
// 32, 0.067 with 4 or 16 warps; K = 2 at 100^3: 0.157 ms, 0.25 with 8 warps).
// 16 warps where one or two blocks fill an SM's shared memory (K = 5 patches, cells of
// K = 7, 8): a launch of few blocks is one block's latency, half the row tiles per
// warp shorten it (8 and 16 warps: FP32 K = 5 at 8^3 cells, sweep 33.8 and 31.1 us,
// multiplicative 255 and 231; FP64 apply K = 8 71.8 and 67.1), and large
// ones are as fast.  3D FP32 patches of K >= 6 and FP64 ones of K = 8 keep the
// sum-factorised kernel: their operands fill an SM's shared memory with 8-16
// patches, and the matrix is streamed from L2 for so few columns (K = 6 FP32 at
// 33^3 cells: 0.67 ms against 0.49 ms).
template <int DIM, int M, typename T>
struct Dense {
  using S = Sectors<DIM, M>;
  static constexpr bool F64 = sizeof(T) == 8;
  static constexpr int SL = F64 ? 8 : 3;  // parts per value
  static constexpr unsigned long long BIAS = 0x8080808080808080ull;  // digits + 128
  static constexpr int P = 16;
  static constexpr int NT = P / 8;                              // 8-column tiles
  static constexpr int NSUB = 32 / P;                           // lines a warp handles at once
  static constexpr int UNITS = S::PROWS / 16;                   // 16-row tiles of the result
  static constexpr int NW = UNITS >= 32 ? 16 : UNITS >= 16 ? 8 : (UNITS > 2 ? 4 : 2);
  static constexpr int UPW = (UNITS + NW - 1) / NW;             // units per warp
  // Operands: FP64 fixed-point values [row][XP], FP32 the three parts as
  // planes of BF16 [part][row][XP]; the pitch spreads the rows over the banks.
  static constexpr int XP = F64 ? P + 4 : P + 8;
  static constexpr int XBYTES = F64 ? S::PROWS * XP * 8 : SL * S::PROWS * XP * 2;
  // Results [row][YP], nodal results [patch][ZP].  FP64: the results follow
  // the operands (they first hold the gathered values), the nodal results
  // take the operands' place; FP32: both take the operands' place.
  static constexpr int YP = F64 ? P : P + 4;
  static constexpr int YBYTES = (S::ROWS * YP * (int)sizeof(T) + 15) / 16 * 16;
  static constexpr int ZP = S::NODES | 1;
  static constexpr int ZBYTES = P * ZP * (int)sizeof(T);
  static constexpr int max2(int a, int b) { return a > b ? a : b; }
  static constexpr int YOFF = F64 ? (max2(XBYTES, ZBYTES) + 15) / 16 * 16 : 0;
  static constexpr int ZOFF = F64 ? 0 : YBYTES;
  static constexpr int SMEM = F64 ? YOFF + YBYTES : max2(XBYTES, YBYTES + ZBYTES);
  // blocks per SM that the shared memory and 64 K registers (at least 128 a
  // thread in FP64: 7 accumulators and 7 fragments per column tile) allow
  static constexpr int MINB() {
    const int bs = 227 * 1024 / (SMEM + 1536), br = 65536 / (32 * NW * (F64 ? 128 : 64)), b = bs < br ? bs : br;
    return b < 1 ? 1 : (b > 8 ? 8 : b);
  }
  // patches of this part are products; not 2D K = 2 in FP32, whose 9 nodes fill
  // half a tile and are bound by their gather and scatter (700^2 cells: sweep 80
  // us, 66 by sum factorisation; multiplicative 178 and 129)
  static constexpr bool ok() {
    return K >= 2 && M <= (DIM == 2 ? 15 : 9) && SMEM <= kMaxDynSmem && !(DIM == 2 && K == 2 && !F64);
  }
  // table: 16-byte fragments, then (FP64) per row its exponent above its
  // orbit's, and the exponents of the orbits' results (kNoExp in the first: a
  // matrix that is not finite), then the columns of the orbits' first nodes
  // (dense_spikes)
  static constexpr int FRAGS = S::TILES * SL * 32;
  static constexpr int COLUMNS = FRAGS * 16 + (F64 ? (S::ROWS + S::ORBITS + 3) / 4 * 16 : 0);
  static constexpr int64_t TABLE_BYTES = COLUMNS + (int64_t)S::ORBITS * S::NODES * 8;
};

// One 16-row tile of the result: a warp's unit of work.
struct DenseUnit {
  short prow;   // first operand row of the sector
  short kt;     // 16-column tiles
  short row;    // result row of the tile
  short valid;  // its rows that exist
  int frag;     // first fragment (in units of 32 lanes)
};
template <int N>
struct DenseUnits {
  DenseUnit u[N];
};
template <int DIM, int M, typename T>
constexpr DenseUnits<Dense<DIM, M, T>::UNITS> dense_units() {
  using S = Sectors<DIM, M>;
  DenseUnits<Dense<DIM, M, T>::UNITS> r{};
  int n = 0;
  for (int s = 0; s < S::NS; ++s)
    for (int m = 0; m < S::tiles(s); ++m) {
      DenseUnit& u = r.u[n++];
      u.prow = (short)S::prow(s);
      u.kt = (short)S::tiles(s);
      u.row = (short)(S::row(s) + 16 * m);
      u.valid = (short)(S::size(s) - 16 * m < 16 ? S::size(s) - 16 * m : 16);
      u.frag = (S::tile(s) + m * S::tiles(s)) * Dense<DIM, M, T>::SL;
    }
  return r;
}

// Parameters of one level's launch.  FP64: a result is its integer x cmul x
// 2^(vexp + the patch's exponent - its orbit's exponent), cmul in [2^63, 2^64).
template <typename T>
struct DenseJob {
  const T* r;
  T* dst;
  const uint4* table;
  int n, colour;
  T c;                       // omega_AS / scale (additive) or 1 / scale; cells: scale
  unsigned long long cmul;   // FP64: the same as a normalised integer (0: not finite)
  int vexp;                  // and its binary exponent
  uint32_t npatch;
  FastDiv d0, d1;            // patches per direction
};

// ---------------------------------------------------------------- FP64 <-> fixed point
// v 2^(60 - e + 1022) truncated, for |v| < 2^(e - 1022) (e: biased exponent + 1
// bound); mag: its magnitude in units of 2^32
__device__ __forceinline__ long long fixed_of(double v, int e, unsigned& mag) {
  const int hi = __double2hiint(v);
  const unsigned lo = (unsigned)__double2loint(v);
  const int ex = (hi >> 20) & 0x7FF;
  const unsigned mh = ((unsigned)hi & 0xFFFFFu) | (ex ? 0x100000u : 0u);
  const unsigned long long m = (((unsigned long long)mh << 32) | lo) << 7;
  const int sh = min(e - (ex ? ex : 1), 63);
  const long long x = (long long)(m >> sh);
  mag = (unsigned)(x >> 32);
  const long long sg = (long long)(hi >> 31);
  return (x ^ sg) - sg;
}

// Scale of a patch's (or cell's) values for the fixed point: mx the largest
// high word, with its low bit set where only a low word is not zero.  The
// bound e leaves 0.8% to the top digit's range; subnormal windows are scaled
// by 2^100 and bounded by the high word's leading bit.
struct PatchScale {
  int e;
  bool subnormal;  // all values: fixed_of is exact
  bool bad;  // an infinity or NaN, or a matrix that is not finite
  bool tiny, any_tiny;
  __device__ __forceinline__ PatchScale() {}
  __device__ __forceinline__ PatchScale(unsigned mx, bool broken) {
    bad = mx >= 0x7FF00000u || broken;
    tiny = mx < 0x00100000u;
    any_tiny = __any_sync(0xffffffffu, tiny && mx != 0);  // the FP64 products with 2^100 only where needed
    tiny = tiny && any_tiny;
    e = tiny ? 113 - __clz((int)mx) : max((int)((mx + 0x4000u) >> 20), 1);
    subnormal = mx < 0x00100000u;
  }
  // the largest magnitude, in units of 2^40 (normal)
  __device__ __forceinline__ unsigned top(unsigned mx) const {
    return ((mx & 0xFFFFFu) | 0x100000u) >> (e - (int)(mx >> 20) + 1);
  }
  template <int M>
  __device__ __forceinline__ void fixed(double (&r)[M], long long (&v)[M], unsigned (&mag)[M]) const {
    if (any_tiny) {
#pragma unroll
      for (int i = 0; i < M; ++i) r[i] = tiny ? r[i] * 0x1p100 : r[i];
    }
#pragma unroll
    for (int i = 0; i < M; ++i) v[i] = fixed_of(r[i], e, mag[i]);
  }
};

// an even / odd combination of up to 2^(3 - sh) values as operand (63 bits and sign)
__device__ __forceinline__ long long operand_of(long long v, int sh) { return (long long)((unsigned long long)v << sh); }

// The products hold all values of a window to one absolute accuracy (2^-60 of
// its largest in FP64; the even / odd sums in FP32 to 2^-24 of the largest of
// the mirror images).  A result that couples to the largest value through
// small entries only would lose relative accuracy: up to 1e3 (K = 4) and 2e4
// (K = 8) roundings of |A||x| for one value of 1e6 among N(0,1) ones.  The
// products of an uneven window are formed again without its spikes -- the
// values above 2^-10 of the largest --, whose columns are added in FP64
// (dense_spikes).  Uneven is
// - a patch with an octant (a cell; the nodes between cells count for both)
//   whose largest value is below 2^-7 of the patch's: residuals of a solve
//   keep above 2^-4 in every octant, however small their values at most nodes.
//   Largest errors above the line, in roundings of |B||r|: K = 3 26, K = 4 430, K = 5 1,500
//   (N(0,1) values times 1e6 at the outermost corners), the local
//   V-cycle in FP64 24, 900, 270;
// - a cell with a mean magnitude below 1/32 of its largest (N(0,1) values: 1/4, in
//   a corner cell 1/10; x y z 1/8).  Worst found now: K = 3 13, K = 4 42, K = 8 133 roundings of
//   (|K| x |M| x |M| + ...) |x|; line passes 16, 60, 70 (the 1D matrices' own).
// A window whose values above 2^-10 of its largest are more than an eighth of
// its nodes counts as even all the same: they reach every node.  Windows of at
// most 32 nodes are not split, have no such entries, and are not looked at.
constexpr int kUnevenExp = 7, kUnevenCell = 32, kSpikeExp = 10;

// bits of |v| in order of magnitude (FP64: the high word)
__device__ __forceinline__ unsigned magnitude(double v) { return (unsigned)__double2hiint(v) & 0x7FFFFFFFu; }
__device__ __forceinline__ unsigned magnitude(float v) { return __float_as_uint(v) & 0x7FFFFFFFu; }
// above it: a spike of a window whose largest value has the magnitude mx
template <typename T>
__device__ __forceinline__ unsigned spike_bound(unsigned mx) {
  constexpr int MB = sizeof(T) == 8 ? 20 : 23;  // mantissa bits
  return mx > (unsigned)(kSpikeExp + 1) << MB ? mx - ((unsigned)kSpikeExp << MB) : 1u << MB;
}
constexpr unsigned kNoSpikes = 0xFFFFFFFFu;

// The magnitudes of image b of a line into the largest ones of the window's
// octants, s_oct[side along x][image in the other directions][window]
template <int DIM, int M>
constexpr int octants() { return 2 * Lines<DIM, M>::IMAGES; }
template <int DIM, int M, int P, class F>
__device__ __forceinline__ void add_octants(const Lines<DIM, M>& ln, int b, F&& mag, unsigned (*s_oct)[P], int pn) {
  using S = Sectors<DIM, M>;
  constexpr int IM = Lines<DIM, M>::IMAGES;
  unsigned lo = 0, hi = 0;
#pragma unroll
  for (int i = 0; i < M; ++i) {
    if (i < S::E) lo = max(lo, mag(i));
    if (i >= S::O) hi = max(hi, mag(i));
  }
  const bool cy = S::CENTRE && ln.c[0] == S::E - 1, cz = S::CENTRE && DIM == 3 && ln.c[1] == S::E - 1;
#pragma unroll
  for (int o = 0; o < IM; ++o) {  // a central line lies on both sides
    const int x = o ^ b;
    if ((x & 1) && !(cy && !(b & 1))) continue;
    if ((x & 2) && !(cz && !(b & 2))) continue;
    atomicMax(&s_oct[o][pn], lo);
    atomicMax(&s_oct[IM + o][pn], hi);
  }
}

// largest and smallest of a window's octants
template <int N, int P>
__device__ __forceinline__ void octant_range(const unsigned (*s_oct)[P], int pn, unsigned& lo, unsigned& hi) {
  lo = hi = s_oct[0][pn];
#pragma unroll
  for (int o = 1; o < N; ++o) {
    lo = min(lo, s_oct[o][pn]);
    hi = max(hi, s_oct[o][pn]);
  }
}

// y cmul 2^(ve + 64) rounded to nearest (ties away), in integer arithmetic
__device__ __forceinline__ double double_of(long long y, unsigned long long cmul, int ve) {
  const unsigned long long sg = (unsigned long long)(y >> 63);
  const unsigned long long a = ((unsigned long long)y ^ sg) - sg;
  if (a == 0) return 0.0;
  const int z = __clzll((long long)a);
  unsigned long long p = __umul64hi(a << z, cmul);  // >= 2^62
  int ex = ve - z + 64 + 63 + 1023;                 // biased exponent of 2^63 2^(ve + 64 - z)
  if (!(p >> 63)) {
    p <<= 1;
    --ex;
  }
  p += 0x400;                // round at bit 11
  if (p < 0x400) {           // carried out of the top bit
    p = 0x8000000000000000ull;
    ++ex;
  }
  if (ex >= 1 && ex <= 2046) {
    const unsigned long long m = (p >> 11) & 0xFFFFFFFFFFFFFull;
    return __longlong_as_double((long long)(m | ((unsigned long long)ex << 52) | (sg & 0x8000000000000000ull)));
  }
  // overflow or a subnormal result
  const double d = ldexp((double)(p >> 11), ex - 1023 - 52);
  return sg ? -d : d;
}

__device__ __forceinline__ void mma_f16(float (&c)[4], const uint4& a, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint4& a, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm_t(uint32_t (&b)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3])
               : "r"(addr));
}

constexpr int kNoExp = -(1 << 30);          // first orbit's exponent of a matrix that is not finite
constexpr float kMagic = 12582912.0f;       // 1.5 2^23: the accumulator's bits count integers from here
constexpr int kMagicBits = 0x4B400000;

// FP64 products of one unit: result rows of sector coefficients times the
// operand rows, in units of 2^-68 of (table integer x operand integer) at the
// exponent of the row's orbit.  Two k tiles add at most 8 digit pairs of 32
// products below 2^14 to an accumulator (its exact range is 2^22 around kMagic;
// the first digits stay within 127) before it is emptied into Y.
template <class D>
__device__ __forceinline__ void dense_mma(const DenseUnit& u, const uint4* __restrict__ table,
                                          const int* __restrict__ shifts, const long long* X, long long* Y,
                                          int lane) {
  constexpr int SL = D::SL, NT = D::NT, ND = 8;  // ND: digit sums kept, i + j < ND
  const int g = lane >> 2, q = lane & 3;
  const int* shift = shifts + u.row + g;  // row exponent - its orbit's
  const uint4* tp = table + (int64_t)u.frag * 32 + lane;
  const long long* xp = X + (u.prow + 2 * q) * D::XP + g;
  for (int k0 = 0; k0 < u.kt; k0 += 2) {
    float acc[ND][NT][4];
#pragma unroll
    for (int d = 0; d < ND; ++d)
#pragma unroll
      for (int t = 0; t < NT; ++t)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[d][t][i] = kMagic;
    for (int k = k0; k < min(k0 + 2, (int)u.kt); ++k) {
      uint4 a = __ldg(tp + k * SL * 32);
      // digits of the operand values of rows 2q, 2q+1, 2q+8, 2q+9 of the tile
      uint32_t b[SL][NT][2];
#pragma unroll
      for (int t = 0; t < NT; ++t)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const long long* x = xp + (16 * k + 8 * h) * D::XP + 8 * t;
          // biased so that byte SL - 1 - j holds digit j + 128
          const unsigned long long w0 = (unsigned long long)x[0] + D::BIAS, w1 = (unsigned long long)x[D::XP] + D::BIAS;
#pragma unroll
          for (int j = 0; j < SL; ++j) {
            const int byte = SL - 1 - j, bb = byte & 3;
            const uint32_t v0 = (uint32_t)(byte < 4 ? w0 : w0 >> 32), v1 = (uint32_t)(byte < 4 ? w1 : w1 >> 32);
            const uint32_t pr = __byte_perm(v0, v1, bb | (bb << 4) | ((4 + bb) << 8) | ((4 + bb) << 12));
            const uint32_t hb = (pr & 0x00FF00FFu) | 0x64006400u;  // 1024 + digit + 128 as halves
            const __half2 dg = __hsub2(*reinterpret_cast<const __half2*>(&hb), __half2half2(__ushort_as_half(0x6480)));
            b[j][t][h] = *reinterpret_cast<const uint32_t*>(&dg);
          }
        }
#pragma unroll
      for (int i = 0; i < SL; ++i) {
        const uint4 next = i + 1 < SL ? __ldg(tp + (k * SL + i + 1) * 32) : a;
#pragma unroll
        for (int j = 0; j < SL; ++j)
          if (i + j < ND) {
#pragma unroll
            for (int t = 0; t < NT; ++t) mma_f16(acc[i + j][t], a, b[j][t][0], b[j][t][1]);
          }
        a = next;
      }
    }
    // into Y: partial sums at the row's exponent, at the end rounded to the orbit's
    const bool last = k0 + 2 >= u.kt;
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (g + 8 * h < u.valid) {
        const int sh = last ? __ldg(shift + 8 * h) : 0;
        const long long half = (1ll << sh) >> 1;
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            auto pair = [&](int d) {
              return (__float_as_int(acc[d][t][2 * h + i]) - kMagicBits) * 256 +
                     (__float_as_int(acc[d + 1][t][2 * h + i]) - kMagicBits);
            };
            long long* y = Y + (u.row + g + 8 * h) * D::YP + 8 * t + 2 * q + i;
            // rounded, not cut off: a bias would add up over the mirror images
            const long long v = ((long long)pair(0) << 36) + ((long long)pair(2) << 20) + ((long long)pair(4) << 4) +
                                ((pair(6) + 2048) >> 12) + (k0 ? *y : 0);
            *y = (v + half) >> sh;
          }
      }
  }
}

// FP32 products of one unit into y.  The leading products are taken out of
// the accumulator after every k tile and summed with rounding (the tensor
// cores truncate their sums); the five small products share an accumulator.
template <class D>
__device__ __forceinline__ void dense_mma(const DenseUnit& u, const uint4* __restrict__ table, const uint16_t* X,
                                          float (&y)[D::NT][4], int lane) {
  using S = typename D::S;
  constexpr int SL = D::SL, NT = D::NT;
  float lo[NT][4] = {};
#pragma unroll
  for (int t = 0; t < NT; ++t)
#pragma unroll
    for (int i = 0; i < 4; ++i) y[t][i] = 0.f;
  const uint4* tp = table + (int64_t)u.frag * 32 + lane;
  // ldmatrix source row of this lane: (k 0-7 | 8-15) x (n 0-7 | 8-15)
  const uint32_t xa = (uint32_t)__cvta_generic_to_shared(X) +
                      2 * ((u.prow + 8 * ((lane >> 3) & 1) + (lane & 7)) * D::XP + 8 * (lane >> 4));
  for (int k = 0; k < u.kt; ++k) {
    uint4 a[SL];
#pragma unroll
    for (int i = 0; i < SL; ++i) a[i] = __ldg(tp + (k * SL + i) * 32);
#pragma unroll
    for (int t = 0; t < NT; t += 2) {
      uint32_t b[SL][4];
#pragma unroll
      for (int j = 0; j < SL; ++j) ldsm_t(b[j], xa + 2 * ((j * S::PROWS + 16 * k) * D::XP + 8 * t));
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float hi[4] = {};
        mma_bf16(hi, a[0], b[0][2 * h], b[0][2 * h + 1]);
#pragma unroll
        for (int j = 0; j < SL; ++j)
#pragma unroll
          for (int i = 0; i + j < SL; ++i)
            if (i + j > 0) mma_bf16(lo[t + h], a[i], b[j][2 * h], b[j][2 * h + 1]);
#pragma unroll
        for (int i = 0; i < 4; ++i) y[t + h][i] += hi[i];
      }
    }
  }
#pragma unroll
  for (int t = 0; t < NT; ++t)
#pragma unroll
    for (int i = 0; i < 4; ++i) y[t][i] += lo[t][i];
}

// the patch's window and the cell's (FP64 operator apply)
constexpr int kPatchM = mp(K), kCellM = K + 1;
static __constant__ const DenseUnits<Dense<PMG_DIM, kPatchM, TP>::UNITS> c_units = dense_units<PMG_DIM, kPatchM, TP>();
#if PMG_PREC == 0
static __constant__ const DenseUnits<Dense<PMG_DIM, kCellM, double>::UNITS> c_cell_units =
    dense_units<PMG_DIM, kCellM, double>();
#endif

// boundary faces of the grid (bits of edge) at node (x, y, z) of a cell
template <int DIM, int M>
__device__ __forceinline__ bool on_face(unsigned edge, int x, int y, int z) {
  return (x == 0 && (edge & 1)) || (x == M - 1 && (edge & 2)) || (y == 0 && (edge & 4)) || (y == M - 1 && (edge & 8)) ||
         (DIM == 3 && ((z == 0 && (edge & 16)) || (z == M - 1 && (edge & 32))));
}

// Part of a window's result at node i that the spikes contribute, by the
// columns of the orbits' first nodes: the operator commutes with the
// reflections, so the column of a mirror image is the mirrored column.
template <int DIM, int M, typename T>
__device__ __forceinline__ double spikes_at(const double* __restrict__ columns, const T* xw,
                                            const unsigned short* list, int count, int i) {
  using S = Sectors<DIM, M>;
  const int ix = i % M, iy = (i / M) % M, iz = i / (M * M);
  double acc = 0.0;
#pragma unroll 4
  for (int l = 0; l < count; ++l) {
    const int j = list[l], jx = j % M, jy = (j / M) % M, jz = j / (M * M);
    const bool fx = jx >= S::E, fy = jy >= S::E, fz = jz >= S::E;
    const int orbit = (fx ? M - 1 - jx : jx) + S::E * ((fy ? M - 1 - jy : jy) + S::E * (fz ? M - 1 - jz : jz));
    const int node = (fx ? M - 1 - ix : ix) + M * ((fy ? M - 1 - iy : iy) + M * (fz ? M - 1 - iz : iz));
    acc += __ldg(columns + (int64_t)orbit * S::NODES + node) * (double)xw[j];
  }
  return acc;
}

// list of the nodes with a magnitude above bound, in order (whole block; returns after a barrier)
template <int NODES, typename T>
__device__ __forceinline__ int list_spikes(const T* xw, unsigned bound, unsigned short* list, int* s_count) {
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    int count = 0;
    for (int i = 0; i < NODES; i += 32) {
      const bool is = i + lane < NODES && magnitude(xw[min(i + lane, NODES - 1)]) > bound;
      const unsigned mask = __ballot_sync(0xffffffffu, is);
      if (is) list[count + __popc(mask & ((1u << lane) - 1))] = (unsigned short)(i + lane);
      count += __popc(mask);
    }
    if (lane == 0) *s_count = count;
  }
  __syncthreads();
  return *s_count;
}

// The spikes of a batch's uneven windows, one window after the other, added to
// the results (whole block; its dynamic shared memory is free once the block has met).
template <int DIM, typename T, bool CELL>
__device__ __noinline__ void dense_spikes(const DenseJob<T>& J, uint32_t batch, const unsigned* s_spike,
                                          const int64_t* s_base, const int* s_colour, int* s_count) {
  constexpr int M = CELL ? kCellM : kPatchM;
  using S = Sectors<DIM, M>;
  using D = Dense<DIM, M, T>;
  static_assert(D::SMEM >= S::NODES * ((int)sizeof(T) + 2), "a window and its list fit");
  extern __shared__ __align__(16) unsigned char smraw[];
  T* xw = reinterpret_cast<T*>(smraw);
  unsigned short* list = reinterpret_cast<unsigned short*>(xw + S::NODES);
  const int N1 = K * J.n + 1;
  const int64_t N = (int64_t)N1 * N1 * (DIM == 3 ? N1 : 1);
  const double* columns = reinterpret_cast<const double*>(reinterpret_cast<const char*>(J.table) + D::COLUMNS);
#pragma unroll 1
  for (int gp = 0; gp < D::P; ++gp) {
    if (s_spike[gp] == kNoSpikes) continue;
    __syncthreads();
    const int edge = s_colour[gp];
    const T* r = J.r + s_base[gp];
    for (int i = threadIdx.x; i < S::NODES; i += blockDim.x) {
      const int x = i % M, y = (i / M) % M, z = i / (M * M);
      xw[i] = CELL && on_face<DIM, M>(edge, x, y, z) ? T(0) : r[x + N1 * (y + (DIM == 3 ? N1 * z : 0))];
    }
    __syncthreads();
    const int count = list_spikes<S::NODES>(xw, s_spike[gp], list, s_count);
    for (int i = threadIdx.x; i < S::NODES; i += blockDim.x) {
      const int x = i % M, y = (i / M) % M, z = i / (M * M);
      T* d;
      if constexpr (CELL) d = J.dst + ((int64_t)batch * D::P + gp) * S::NODES + i;
      else d = J.dst + (J.colour < 0 ? s_colour[gp] * N : 0) + s_base[gp] + x + N1 * (y + (DIM == 3 ? N1 * z : 0));
      *d = (T)((double)*d + (double)J.c * spikes_at<DIM, M>(columns, xw, list, count, i));
    }
  }
}

// Operands and products of the windows whose first nodes are at `base` (a lane
// holds one window): gather, even / odd combinations, results in Y.  Finds the
// uneven windows (s_spike, s_any); AGAIN: the block's windows without spikes.
template <int DIM, typename T, bool CELL, bool AGAIN, int NOCT>
__device__ __forceinline__ void dense_pass(const DenseJob<T>& J, int64_t base, bool active, unsigned edge,
                                            unsigned* s_max, unsigned (*s_oct)[Dense<DIM, CELL ? kCellM : kPatchM, T>::P],
                                            unsigned* s_spike, int* s_any) {
  constexpr int M = CELL ? kCellM : kPatchM;
  using S = Sectors<DIM, M>;
  using D = Dense<DIM, M, T>;
  using L = Lines<DIM, M>;
  constexpr int P = D::P, NSUB = D::NSUB, NW = D::NW;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int pn = lane % P, item0 = warp * NSUB + lane / P;
  constexpr int STEP = NW * NSUB;
  const int N1 = K * J.n + 1;
  const T* rp = J.r + base;
  using XT = std::conditional_t<D::F64, long long, uint16_t>;
  using YT = std::conditional_t<D::F64, long long, float>;
  XT* X = reinterpret_cast<XT*>(smraw);
  YT* Y = reinterpret_cast<YT*>(smraw + D::YOFF);
  PatchScale sc;  // FP64
  const int* orbitexp = reinterpret_cast<const int*>(J.table + D::FRAGS) + S::ROWS;
  if constexpr (D::F64) {
      double* R = reinterpret_cast<double*>(Y);
    unsigned mx = 0;
    for (int l = item0; l < S::NODES / S::M; l += STEP) {
      const int ly = DIM == 3 ? l % M : l, lz = DIM == 3 ? l / M : 0;
      const double* q = rp + N1 * (ly + N1 * lz);
      const bool in = active && !(CELL && (((edge & 4) && ly == 0) || ((edge & 8) && ly == M - 1) ||
                                           (DIM == 3 && (((edge & 16) && lz == 0) || ((edge & 32) && lz == M - 1)))));
      double v[M];
#pragma unroll
      for (int i = 0; i < M; ++i)
        v[i] = in && !(CELL && ((i == 0 && (edge & 1)) || (i == M - 1 && (edge & 2)))) ? q[i] : 0.0;
      if constexpr (AGAIN) {
#pragma unroll
        for (int i = 0; i < M; ++i) v[i] = magnitude(v[i]) > s_spike[pn] ? 0.0 : v[i];
      }
#pragma unroll
      for (int i = 0; i < S::M; ++i) {
        R[(l * S::M + i) * P + pn] = v[i];
        // the low bit: a value below the high word's range is not zero
        mx = max(mx, magnitude(v[i]) | (__double2loint(v[i]) != 0));
      }
    }
#pragma unroll
    for (int o = P; o < 32; o <<= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane < P) atomicMax(&s_max[pn], mx);
    __syncthreads();
    sc = PatchScale(s_max[pn], J.cmul == 0 || orbitexp[0] == kNoExp);
  }
  // even / odd combinations, stored as operands
  unsigned sum = 0;  // cells: of the magnitudes, in units of 2^40
  for (int l = item0; l < L::N; l += STEP) {
    const L ln(l);
    if constexpr (D::F64) {
      const double* R = reinterpret_cast<const double*>(Y);
      long long v[L::IMAGES][M];
#pragma unroll
      for (int b = 0; b < L::IMAGES; ++b) {
        const double* q = R + ln.node(b, M) * P + pn;
        double r[M];
#pragma unroll
        for (int i = 0; i < M; ++i) r[i] = ln.has(b) || !S::SPLIT ? q[i * P] : 0.0;
        unsigned mag[M];
        sc.template fixed<M>(r, v[b], mag);
        if constexpr (S::SPLIT && CELL) {
#pragma unroll
          for (int i = 0; i < M; ++i) sum += mag[i] >> 8;
        }
        if constexpr (NOCT > 1 && !AGAIN) add_octants(ln, b, [&](int i) { return mag[i]; }, s_oct, pn);
      }
      reflect<DIM, M>(v);
      const int sh0 = (S::SPLIT ? 3 - DIM : 3) + ln.centres();  // 2^(d-c) images were summed
#pragma unroll
      for (int b = 0; b < L::IMAGES; ++b)
        if (ln.has(b) || !S::SPLIT)
          for_coefs<DIM, M>(b, [&](int i, int s, int ox) {
            X[(S::prow(s) + ox + ln.coef(s)) * D::XP + pn] =
                operand_of(v[b][i], S::CENTRE && i == S::E - 1 ? sh0 + 1 : sh0);
          });
    } else {
      float v[L::IMAGES][M];
#pragma unroll
      for (int b = 0; b < L::IMAGES; ++b) {
        const float* q = rp + ln.node(b, N1);
        const bool in = active && (ln.has(b) || !S::SPLIT);
#pragma unroll
        for (int i = 0; i < M; ++i) v[b][i] = in ? q[i] : 0.f;
      }
      if constexpr (NOCT > 1) {
        if constexpr (AGAIN) {
#pragma unroll
          for (int b = 0; b < L::IMAGES; ++b)
#pragma unroll
            for (int i = 0; i < M; ++i) v[b][i] = magnitude(v[b][i]) > s_spike[pn] ? 0.f : v[b][i];
        } else {
#pragma unroll
          for (int b = 0; b < L::IMAGES; ++b)
            add_octants(ln, b, [&](int i) { return magnitude(v[b][i]); }, s_oct, pn);
        }
      }
      reflect<DIM, M>(v);
#pragma unroll
      for (int b = 0; b < L::IMAGES; ++b)
        if (ln.has(b) || !S::SPLIT)
          for_coefs<DIM, M>(b, [&](int i, int s, int ox) {
            XT* x = X + (S::prow(s) + ox + ln.coef(s)) * D::XP + pn;
            const uint32_t b1 = __float_as_uint(v[b][i]);
            const float f2 = v[b][i] - __uint_as_float(b1 & 0xFFFF0000u);
            const uint32_t b2 = __float_as_uint(f2);
            const float f3 = f2 - __uint_as_float(b2 & 0xFFFF0000u);
            x[0] = (uint16_t)(b1 >> 16);
            x[S::PROWS * D::XP] = (uint16_t)(b2 >> 16);
            x[2 * S::PROWS * D::XP] = (uint16_t)(__float_as_uint(f3) >> 16);
          });
    }
  }
  // integers throughout, so that the choice does not depend on the batch
  if constexpr (S::SPLIT && CELL) {
    if constexpr (!AGAIN) {
#pragma unroll
      for (int o = P; o < 32; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      if (lane < P) atomicAdd(&s_oct[0][pn], sum);
    }
  }
  __syncthreads();
  if (S::SPLIT && !AGAIN && threadIdx.x < P) {
    unsigned mx = s_max[pn];
    bool uneven;
    if constexpr (CELL) {
      uneven = !sc.bad && !sc.subnormal &&
               (unsigned long long)s_oct[0][pn] * kUnevenCell < (unsigned long long)sc.top(mx) * S::NODES;
    } else {
      unsigned lo, hi;
      octant_range<NOCT>(s_oct, pn, lo, hi);
      if constexpr (D::F64) {
        uneven = !sc.bad && !sc.subnormal && lo < hi >> kUnevenExp;
      } else {
        mx = hi;
        uneven = hi < 0x7F800000u && hi > (unsigned)(kUnevenExp + 1) << 23 && lo < hi - ((unsigned)kUnevenExp << 23);
      }
    }
    if (uneven) {
      s_spike[pn] = spike_bound<T>(mx);
      *s_any = 1;
    }
  }
  if constexpr (D::F64) {
    for (int u = warp; u < D::UNITS; u += NW) {
#if PMG_PREC == 0
      dense_mma<D>(CELL ? c_cell_units.u[CELL ? u : 0] : c_units.u[CELL ? 0 : u], J.table, orbitexp - S::ROWS, X, Y, lane);
#endif
    }
    __syncthreads();
  } else {
    float y[D::UPW][D::NT][4];
#pragma unroll
    for (int i = 0; i < D::UPW; ++i)
      if (warp + i * NW < D::UNITS) dense_mma<D>(c_units.u[warp + i * NW], J.table, X, y[i], lane);
    __syncthreads();  // the results take the operands' place
    if (S::SPLIT && !AGAIN && *s_any) return;  // not needed
#pragma unroll
    for (int i = 0; i < D::UPW; ++i)
      if (warp + i * NW < D::UNITS) {
        const DenseUnit& u = c_units.u[warp + i * NW];
#pragma unroll
        for (int t = 0; t < D::NT; ++t)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int rr = (lane >> 2) + 8 * h;
            if (rr < u.valid)
              *reinterpret_cast<float2*>(Y + (u.row + rr) * D::YP + 8 * t + 2 * (lane & 3)) =
                  make_float2(y[i][t][2 * h], y[i][t][2 * h + 1]);
          }
      }
    __syncthreads();
  }
}

// The second pass.  A window with more spikes than an eighth of its nodes
// keeps them (kNoSpikes): its large values reach every node.
template <int DIM, typename T, bool CELL, int NOCT>
__device__ __noinline__ void dense_again(const DenseJob<T>& J, const int64_t* s_base, const int* s_colour,
                                         unsigned* s_max,
                                         unsigned (*s_oct)[Dense<DIM, CELL ? kCellM : kPatchM, T>::P],
                                         unsigned* s_spike, int* s_any) {
  constexpr int P = Dense<DIM, CELL ? kCellM : kPatchM, T>::P;
  constexpr int M = CELL ? kCellM : kPatchM, NODES = ipow(M, DIM);
  const int pn = (threadIdx.x & 31) % P, N1 = K * J.n + 1;
  if (threadIdx.x < P) s_oct[0][pn] = 0;
  __syncthreads();
  const int64_t base = s_base[pn];
  const unsigned bound = s_spike[pn];
  if (bound != kNoSpikes) {
    unsigned count = 0;
    for (int i = threadIdx.x / P; i < NODES; i += blockDim.x / P) {
      const int x = i % M, y = (i / M) % M, z = i / (M * M);
      const T v = J.r[base + x + N1 * (y + (DIM == 3 ? N1 * z : 0))];
      count += magnitude(v) > bound && !(CELL && on_face<DIM, M>(s_colour[pn], x, y, z));
    }
    atomicAdd(&s_oct[0][pn], count);
  }
  __syncthreads();
  if (threadIdx.x < P && s_oct[0][pn] > NODES / 8) s_spike[pn] = kNoSpikes;
  __syncthreads();
  if (!__syncthreads_or(s_spike[pn] != kNoSpikes) && sizeof(T) == 8) return;  // the first pass's results stand
  if (threadIdx.x < P) s_max[pn] = 0;
  __syncthreads();
  dense_pass<DIM, T, CELL, true, NOCT>(J, base < 0 ? 0 : base, base >= 0, CELL ? (unsigned)s_colour[pn] : 0, s_max, s_oct,
                                        s_spike, s_any);
}

// The patches of batch `batch` of a level: gather r_j, even / odd
// combinations, products, and back; omega_AS d_j to the colour's vector
// (additive) or d_j added to u (multiplicative).  A lane holds one patch (P
// lanes) and the warps share the nodes, so index arithmetic is uniform and
// shared-memory accesses fall on consecutive patches.
//
// CELL: the windows are cells, the matrix the element stiffness matrix of
// Eq. (3) at unit scale; boundary nodes are read as zero and the results go
// to the cell's block of dst (summed per node by cell_sum).
template <int DIM, typename T, bool CELL>
__device__ __forceinline__ void dense_body(const DenseJob<T>& J, uint32_t batch) {
  constexpr int M = CELL ? kCellM : kPatchM;
  using S = Sectors<DIM, M>;
  using D = Dense<DIM, M, T>;
  constexpr int P = D::P, NSUB = D::NSUB, NW = D::NW;
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int64_t s_base[P];
  __shared__ int s_colour[P];
  constexpr int NOCT = S::SPLIT && !CELL ? octants<DIM, M>() : 1;
  __shared__ unsigned s_max[P], s_oct[NOCT][P];  // magnitudes: largest; octants', or (cells) the sum
  __shared__ unsigned s_spike[P];  // magnitude above which a value is a spike
  __shared__ int s_any, s_count;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int pn = lane % P, item0 = warp * NSUB + lane / P;
  constexpr int STEP = NW * NSUB;
  const int N1 = K * J.n + 1;
  // this lane's patch (patch_meta_init's order)
  const uint32_t pid = batch * P + pn;
  const bool active = pid < J.npatch;
  int64_t base;
  unsigned edge = 0;  // CELL: bits of the grid's boundary faces that the cell touches
  {
    const uint32_t t = active ? pid : 0, r1 = J.d0.div(t), r2 = J.d1.div(r1);
    const int i[3] = {(int)(t - r1 * J.d0.d), (int)(DIM == 3 ? r1 - r2 * J.d1.d : r1), (int)(DIM == 3 ? r2 : 0)};
    int v[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      if constexpr (CELL) {
        v[d] = i[d];
        edge |= (v[d] == 0 ? 1u << (2 * d) : 0u) | (v[d] == J.n - 1 ? 2u << (2 * d) : 0u);
      } else {
        v[d] = J.colour < 0 ? i[d] + 1 : 2 * i[d] + (((J.colour >> d) & 1) ? 1 : 2);
      }
    }
    const int o = CELL ? 0 : 1;  // a window starts at node K (v - o) + o
    base = (int64_t)(K * (v[0] - o) + o) + (int64_t)N1 * (K * (v[1] - o) + o);
    if (DIM == 3) base += (int64_t)N1 * N1 * (K * (v[2] - o) + o);
    if (threadIdx.x < P) {
      s_base[pn] = active ? base : -1;
      s_colour[pn] = CELL ? (int)edge : J.colour < 0 ? (v[0] & 1) | ((v[1] & 1) << 1) | (DIM == 3 ? (v[2] & 1) << 2 : 0) : 0;
      s_max[pn] = 0;
#pragma unroll
      for (int o = 0; o < NOCT; ++o) s_oct[o][pn] = 0;
      s_spike[pn] = kNoSpikes;
    }
    if (threadIdx.x == 0) s_any = 0;
  }
  using L = Lines<DIM, M>;
  using XT = std::conditional_t<D::F64, long long, uint16_t>;
  using YT = std::conditional_t<D::F64, long long, float>;
  XT* X = reinterpret_cast<XT*>(smraw);
  YT* Y = reinterpret_cast<YT*>(smraw + D::YOFF);
  T* Z = reinterpret_cast<T*>(smraw + D::ZOFF);
  // padding rows of the operand: zero
  if constexpr (S::PROWS != S::ROWS) {
#pragma unroll
    for (int s = 0; s < S::NS; ++s) {
      constexpr int PARTS = D::F64 ? 1 : D::SL;
      const int z0 = S::prow(s) + S::size(s), nz = S::prow(s) + 16 * S::tiles(s) - z0;
      if (nz > 0)
        for (int i = threadIdx.x; i < PARTS * nz * P; i += 32 * NW) {
          const int pt = i / (nz > 0 ? nz * P : 1), w = i - pt * nz * P;
          X[(pt * S::PROWS + z0 + w / P) * D::XP + w % P] = 0;
        }
    }
  }
  __syncthreads();  // the shared arrays
  dense_pass<DIM, T, CELL, false, NOCT>(J, base, active, edge, s_max, s_oct, s_spike, &s_any);
  if constexpr (S::SPLIT) {
    if (s_any) dense_again<DIM, T, CELL, NOCT>(J, s_base, s_colour, s_max, s_oct, s_spike, &s_any);
  }
  const int* orbitexp = reinterpret_cast<const int*>(J.table + D::FRAGS) + S::ROWS;
  PatchScale sc;  // FP64
  if constexpr (D::F64) sc = PatchScale(s_max[pn], J.cmul == 0 || orbitexp[0] == kNoExp);
  // back to the nodes
  for (int l = item0; l < L::N; l += STEP) {
    const L ln(l);
    YT v[L::IMAGES][S::M];
#pragma unroll
    for (int b = 0; b < L::IMAGES; ++b) {
      const bool in = ln.has(b) || !S::SPLIT;
      for_coefs<DIM, M>(b, [&](int i, int s, int ox) {
        v[b][i] = in ? Y[(S::row(s) + ox + ln.coef(s)) * D::YP + pn] : YT(0);
      });
    }
    reflect<DIM, M>(v);
#pragma unroll
    for (int b = 0; b < L::IMAGES; ++b)
      if (ln.has(b) || !S::SPLIT) {
        T* z = Z + pn * D::ZP + ln.node(b, S::M);
        const int ve = D::F64 ? J.vexp + sc.e - (sc.tiny ? 100 : 0) : 0;
#pragma unroll
        for (int i = 0; i < S::M; ++i) {
          if constexpr (D::F64)
            z[i] = sc.bad ? __longlong_as_double(0x7FF8000000000000ll)
                          : double_of(v[b][i], J.cmul, ve - __ldg(orbitexp + S::E * l + (i < S::E ? i : M - 1 - i)));
          else
            z[i] = J.c * v[b][i];
        }
      }
  }
  __syncthreads();
  if constexpr (CELL) {  // the block's cells are consecutive, like their results
    T* o = J.dst + (int64_t)batch * P * S::NODES;
    const int cells = min(P, (int)(J.npatch - batch * P));
    for (int i = threadIdx.x; i < cells * S::NODES; i += 32 * NW) {
      const int gp = i / S::NODES;
      o[i] = Z[gp * D::ZP + i - gp * S::NODES];
    }
    if (S::SPLIT && s_any) dense_spikes<DIM, T, true>(J, batch, s_spike, s_base, s_colour, &s_count);
    return;
  }
  // a warp writes a patch; each lane keeps the offsets of its nodes
  constexpr int NO = (S::NODES + 31) / 32;
  int off[NO];
#pragma unroll
  for (int j = 0; j < NO; ++j) {
    const int i = lane + 32 * j, r = i / S::M;
    off[j] = i - r * S::M + N1 * (DIM == 3 ? r % S::M + N1 * (r / S::M) : r);
  }
  const int64_t N = (int64_t)N1 * N1 * (DIM == 3 ? N1 : 1);
  if (J.colour < 0) {
    for (int gp = warp; gp < P; gp += NW) {
      if (s_base[gp] < 0) break;  // past the last patch
      T* o = J.dst + s_colour[gp] * N + s_base[gp];
      const T* z = Z + gp * D::ZP + lane;
#pragma unroll
      for (int j = 0; j < NO; ++j)
        if (lane + 32 * j < S::NODES) o[off[j]] = z[32 * j];
    }
  } else {
    // one patch of the colour per node.  The loads of GB patches precede their
    // stores: one after the other they were most of a launch of few blocks (K =
    // 5 FP32, 8^3 cells: a sweep of 8 colours 342 us, 231 now)
    constexpr int PPW = P / NW, GB = NO >= 8 ? 1 : (8 / NO < PPW ? 8 / NO : PPW);
#pragma unroll 1
    for (int g0 = 0; g0 < PPW; g0 += GB) {
      T u[GB][NO];
      auto patch = [&](int g) { return g0 + g < PPW ? warp + NW * (g0 + g) : P; };
#pragma unroll
      for (int g = 0; g < GB; ++g) {
        const int gp = patch(g);
        if (gp >= P || s_base[gp] < 0) continue;
#pragma unroll
        for (int j = 0; j < NO; ++j)
          if (lane + 32 * j < S::NODES) u[g][j] = J.dst[s_base[gp] + off[j]];
      }
#pragma unroll
      for (int g = 0; g < GB; ++g) {
        const int gp = patch(g);
        if (gp >= P || s_base[gp] < 0) continue;
#pragma unroll
        for (int j = 0; j < NO; ++j)
          if (lane + 32 * j < S::NODES) J.dst[s_base[gp] + off[j]] = u[g][j] + Z[gp * D::ZP + lane + 32 * j];
      }
    }
  }
  if (S::SPLIT && s_any) dense_spikes<DIM, T, false>(J, batch, s_spike, s_base, s_colour, &s_count);
}

template <int DIM, typename T>
using PatchDense = Dense<DIM, kPatchM, T>;
template <int DIM>
using CellDense = Dense<DIM, kCellM, double>;

template <int DIM, typename T>
__global__ void __launch_bounds__(32 * PatchDense<DIM, T>::NW, PatchDense<DIM, T>::MINB())
    patch_dense_kernel(const __grid_constant__ DenseJob<T> J) {
  dense_body<DIM, T, false>(J, blockIdx.x);
}

// Grouped launch: the batches of all jobs, job after job
template <int DIM, typename T>
__global__ void __launch_bounds__(32 * PatchDense<DIM, T>::NW, PatchDense<DIM, T>::MINB())
    patch_dense_group_kernel(const __grid_constant__ GroupOf<DenseJob<T>> G) {
  const int j = group_find(G, blockIdx.x);
  dense_body<DIM, T, false>(G.job[j], blockIdx.x - (uint32_t)G.start[j]);
}

// FP64 operator apply on Cartesian meshes: cell results, one block of dst per
// cell, then cell_sum per node.  The line passes (cart_pass) are bound by the
// FP64 pipe; here it only sums the one to 2^d cells of a node.  One apply,
// by line passes and now: 3D K = 4 at 32^3 cells 0.231 and 0.118 ms, K = 2 at
// 100^3 0.62 and 0.53, K = 3 at 67^3 0.72 and 0.45, K = 6 at 33^3 1.01 and
// 0.36, K = 8 at 25^3 1.23 and 0.53; 2D K = 8 at 300^2 0.51 and 0.19.
template <int DIM>
__global__ void __launch_bounds__(32 * CellDense<DIM>::NW, CellDense<DIM>::MINB())
    cell_dense_kernel(const __grid_constant__ DenseJob<double> J) {
  dense_body<DIM, double, true>(J, blockIdx.x);
}

template <int DIM>
__global__ void __launch_bounds__(32 * CellDense<DIM>::NW, CellDense<DIM>::MINB())
    cell_dense_group_kernel(const __grid_constant__ GroupOf<DenseJob<double>> G) {
  const int j = group_find(G, blockIdx.x);
  dense_body<DIM, double, true>(G.job[j], blockIdx.x - (uint32_t)G.start[j]);
}

// y = sum of the cells' results at each node, or b - that sum; boundary nodes
// of y are 0.  Cells in a fixed order: the node's own, then its lower
// neighbours in x, y and z.
template <int DIM>
struct CellSumJob {
  const double* cells;
  const double* b;
  double* y;
  int n;
  FastDiv dN1;
};

template <int DIM>
__device__ __forceinline__ void cell_sum(const CellSumJob<DIM>& J, int64_t t) {
  constexpr int n1 = K + 1, NP = ipow(n1, DIM);
  const int N1 = K * J.n + 1, n = J.n;
  int g[3];
  const int64_t N = (int64_t)N1 * N1 * (DIM == 3 ? N1 : 1);
  if (N < kFastDivItems) {
    const uint32_t v = (uint32_t)t, r = J.dN1.div(v), z = DIM == 3 ? J.dN1.div(r) : 0;
    g[0] = (int)(v - r * J.dN1.d);
    g[1] = (int)(r - z * J.dN1.d);
    g[2] = (int)z;
  } else {
    g[0] = (int)(t % N1);
    g[1] = (int)((t / N1) % N1);
    g[2] = DIM == 3 ? (int)(t / ((int64_t)N1 * N1)) : 0;
  }
  bool bnd = false;
  int c[3] = {0, 0, 0}, a[3] = {0, 0, 0};
#pragma unroll
  for (int d = 0; d < DIM; ++d) {
    bnd = bnd || g[d] == 0 || g[d] == N1 - 1;
    c[d] = g[d] / K;
    a[d] = g[d] - K * c[d];
  }
  if (bnd) {
    J.y[t] = 0.0;
    return;
  }
  // an interior node with a_d = 0 also lies on cell c_d - 1, at its end
  const double* p = J.cells + (c[0] + (int64_t)n * (c[1] + (DIM == 3 ? (int64_t)n * c[2] : 0))) * NP + a[0] +
                    n1 * (a[1] + (DIM == 3 ? n1 * a[2] : 0));
  double v[1 << DIM];
  bool has[1 << DIM];
#pragma unroll
  for (int s = 0; s < 1 << DIM; ++s) {
    int64_t o = 0;
    has[s] = true;
#pragma unroll
    for (int d = 0; d < DIM; ++d)
      if ((s >> d) & 1) {
        has[s] = has[s] && a[d] == 0;
        o -= (d == 0 ? 1 : (d == 1 ? (int64_t)n : (int64_t)n * n)) * NP - K * (d == 0 ? 1 : (d == 1 ? n1 : n1 * n1));
      }
    v[s] = has[s] ? p[o] : 0.0;
  }
  double r = v[0];
#pragma unroll
  for (int s = 1; s < 1 << DIM; ++s)
    if (__any_sync(__activemask(), has[s])) r = has[s] ? r + v[s] : r;  // FP64 adds only where a lane needs one
  J.y[t] = J.b ? J.b[t] - r : r;
}

template <int DIM>
__global__ void __launch_bounds__(256) cell_sum_kernel(const __grid_constant__ CellSumJob<DIM> J, int64_t N) {
  const int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (t < N) cell_sum<DIM>(J, t);
}

template <int DIM>
__global__ void __launch_bounds__(256) cell_sum_group_kernel(const __grid_constant__ GroupOf<CellSumJob<DIM>> G) {
  const int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (t >= G.start[G.count]) return;
  const int j = group_find(G, t);
  cell_sum<DIM>(G.job[j], t - G.start[j]);
}

// ---------------------------------------------------------------- staged products
// FP64 patches of K = 6, 7 in 3D: the operands of 16 patches (180-290 KB) do
// not fit an SM, so the steps of dense_body run as three launches over a chunk
// of batches, whose operands and results (kStageBatches x 0.35-0.57 MB) stay
// in L2: patch_split (gather to fixed point, even / odd combinations), one
// block per batch and sector for the products, patch_merge (back to the
// nodes), one block per batch and pair of mirrored z planes.  Patch
// launch, sum factorisation before and now: K = 7 at 28^3 cells 11.8 and 3.91
// ms, at 12^3 1.02 and 0.32, at 4^3 0.123 and 0.071; K = 6 at 32^3 9.75 and
// 2.78 ms (the matrix, 4-10 MB, is streamed from L2 for every 16 patches).
constexpr bool kStaged = PMG_PREC == 0 && PMG_DIM == 3 && (K == 6 || K == 7);
constexpr int kStageBatches = 76;  // 8 sectors each: two waves of two blocks per SM

template <int DIM>
struct Stage {
  using D = Dense<DIM, kPatchM, double>;
  using S = Sectors<DIM, kPatchM>;
  static constexpr int P = D::P;
  static constexpr int64_t XWORDS = (int64_t)S::ROWS * P, YWORDS = XWORDS;  // per batch
  static constexpr int64_t BYTES = 8 * (XWORDS + YWORDS) + 8 * P;          // and two words per patch
  static constexpr int MAXT = S::tiles(0);
  static constexpr int XSM = 16 * MAXT * D::XP * 8, YSM = S::size(0) * P * 8;  // products: one sector
  static constexpr int MP2 = kPatchM * kPatchM, ZP = (2 * MP2) | 1, ZSM = P * ZP * 8;  // merge: two planes
  static_assert(ZSM >= 10 * S::NODES, "or a window and its list of spikes");
};

// exponent word of a patch: bits 0-11 the exponent bound, 12 tiny, 13 bad;
// the words are followed by the patches' spike bounds (kNoSpikes: even)
struct PatchOrigin {
  int64_t base;
  int colour;
  bool active;
};
template <int DIM>
__device__ __forceinline__ PatchOrigin patch_origin(const DenseJob<double>& J, uint32_t pid) {
  const int N1 = K * J.n + 1;
  PatchOrigin o;
  o.active = pid < J.npatch;
  const uint32_t t = o.active ? pid : 0, r1 = J.d0.div(t), r2 = J.d1.div(r1);
  const int i[3] = {(int)(t - r1 * J.d0.d), (int)(r1 - r2 * J.d1.d), (int)r2};
  int v[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) v[d] = J.colour < 0 ? i[d] + 1 : 2 * i[d] + (((J.colour >> d) & 1) ? 1 : 2);
  o.base = (int64_t)(K * (v[0] - 1) + 1) + (int64_t)N1 * ((K * (v[1] - 1) + 1) + (int64_t)N1 * (K * (v[2] - 1) + 1));
  o.colour = J.colour < 0 ? (v[0] & 1) | ((v[1] & 1) << 1) | ((v[2] & 1) << 2) : 0;
  return o;
}

// A run of batches of one level: batch first + b of the job in place b of the buffers
struct StageJob {
  DenseJob<double> J;
  uint32_t first;
  long long* X;
  long long* Y;
  int* words;
};

// X [row][P] and the words of batch first + b
template <int DIM>
__device__ __forceinline__ void patch_split(const StageJob& G, uint32_t b) {
  const DenseJob<double>& J = G.J;
  constexpr int M = kPatchM;
  using S = Sectors<DIM, M>;
  using L = Lines<DIM, M>;
  constexpr int P = Stage<DIM>::P;
  constexpr int NOCT = octants<DIM, M>();
  __shared__ unsigned s_max[P], s_oct[NOCT][P], s_spike[P];
  __shared__ int s_any;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, pn = lane % P, item0 = warp * (32 / P) + lane / P;
  constexpr int STEP = 8 * (32 / P);
  const int N1 = K * J.n + 1;
  const PatchOrigin o = patch_origin<DIM>(J, (G.first + b) * P + pn);
  const double* rp = J.r + o.base;
  const int* orbitexp = reinterpret_cast<const int*>(J.table + Stage<DIM>::D::FRAGS) + S::ROWS;
  long long* X = G.X + b * Stage<DIM>::XWORDS;
  int* words = G.words + b * 2 * P;
  if (threadIdx.x < P) {
    s_max[threadIdx.x] = 0;
    for (int i = 0; i < NOCT; ++i) s_oct[i][threadIdx.x] = 0;
    s_spike[threadIdx.x] = kNoSpikes;
  }
  if (threadIdx.x == 0) s_any = 0;
  __syncthreads();
#pragma unroll 1
  for (int pass = 0;; ++pass) {  // as in dense_body
    const unsigned bound = s_spike[pn];
    unsigned mx = 0;
    for (int l = item0; l < M * M; l += STEP) {
      const double* q = rp + N1 * (l % M + N1 * (l / M));
      double v[M];
#pragma unroll
      for (int i = 0; i < M; ++i) v[i] = o.active ? q[i] : 0.0;
#pragma unroll
      for (int i = 0; i < M; ++i) {
        const unsigned m = magnitude(v[i]);
        mx = max(mx, m > bound ? 0 : m | (__double2loint(v[i]) != 0));
      }
    }
#pragma unroll
    for (int w = P; w < 32; w <<= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, w));
    if (lane < P) atomicMax(&s_max[pn], mx);
    __syncthreads();
    mx = s_max[pn];
    const PatchScale sc(mx, J.cmul == 0 || orbitexp[0] == kNoExp);
    for (int l = item0; l < L::N; l += STEP) {
      const L ln(l);
      long long v[L::IMAGES][M];
#pragma unroll
      for (int b = 0; b < L::IMAGES; ++b) {
        const double* q = rp + ln.node(b, N1);
        const bool in = o.active && ln.has(b);
        double r[M];
#pragma unroll
        for (int i = 0; i < M; ++i) r[i] = in ? q[i] : 0.0;
        if (pass) {
#pragma unroll
          for (int i = 0; i < M; ++i) r[i] = magnitude(r[i]) > bound ? 0.0 : r[i];
        }
        unsigned mag[M];
        sc.template fixed<M>(r, v[b], mag);
        if (pass == 0) add_octants(ln, b, [&](int i) { return mag[i]; }, s_oct, pn);
      }
      reflect<DIM, M>(v);
      const int sh0 = 3 - DIM + ln.centres();
#pragma unroll
      for (int b = 0; b < L::IMAGES; ++b)
        if (ln.has(b))
          for_coefs<DIM, M>(b, [&](int i, int s, int ox) {
            X[(S::row(s) + ox + ln.coef(s)) * P + pn] =
                operand_of(v[b][i], S::CENTRE && i == S::E - 1 ? sh0 + 1 : sh0);
          });
    }
    __syncthreads();
    if (threadIdx.x < P) {
      unsigned lo, hi;
      octant_range<NOCT>(s_oct, pn, lo, hi);
      if (pass == 0 && !sc.bad && !sc.subnormal && lo < hi >> kUnevenExp) {
        s_spike[pn] = spike_bound<double>(mx);
        s_any = 1;
      }
      s_max[pn] = s_oct[0][pn] = 0;
      words[pn] = sc.e | (sc.tiny ? 1 << 12 : 0) | (sc.bad ? 1 << 13 : 0);
      words[P + pn] = (int)s_spike[pn];
    }
    __syncthreads();
    if (pass || !s_any) break;
    if (s_spike[pn] != kNoSpikes) {  // as dense_again
      unsigned count = 0;
      for (int i = threadIdx.x / P; i < S::NODES; i += 256 / P)
        count += magnitude(rp[i % M + N1 * (i / M % M + N1 * (i / (M * M)))]) > s_spike[pn];
      atomicAdd(&s_oct[0][pn], count);
    }
    __syncthreads();
    if (threadIdx.x < P) {
      if (s_oct[0][pn] > S::NODES / 8) s_spike[pn] = kNoSpikes;
      words[P + pn] = (int)s_spike[pn];
    }
    __syncthreads();
    if (!__syncthreads_or(s_spike[pn] != kNoSpikes)) break;
  }
}

// products of sector s for batch first + b; the sector's row tiles in
// gridDim.z parts (stage_launch)
template <int DIM>
__device__ __forceinline__ void patch_product(const StageJob& G, uint32_t b, int s) {
  using St = Stage<DIM>;
  using D = typename St::D;
  using S = typename St::S;
  constexpr int P = St::P;
  extern __shared__ __align__(16) unsigned char smraw[];
  long long* xs = reinterpret_cast<long long*>(smraw);
  long long* ys = reinterpret_cast<long long*>(smraw + St::XSM);
  const int size = S::size(s), tiles = S::tiles(s), row = S::row(s);
  const uint4* table = G.J.table;
  const long long* x = G.X + b * St::XWORDS + (int64_t)row * P;
  for (int i = threadIdx.x; i < 16 * tiles * P; i += 256)
    xs[i / P * D::XP + i % P] = i < size * P ? x[i] : 0;
  __syncthreads();
  const int* shifts = reinterpret_cast<const int*>(table + D::FRAGS) + row;
  const int m0 = (int)(blockIdx.z * tiles / gridDim.z), m1 = (int)((blockIdx.z + 1) * tiles / gridDim.z);
  for (int m = m0 + (threadIdx.x >> 5); m < m1; m += 8) {
    DenseUnit u;
    u.prow = 0;
    u.kt = (short)tiles;
    u.row = (short)(16 * m);
    u.valid = (short)min(16, size - 16 * m);
    u.frag = (S::tile(s) + m * tiles) * D::SL;
    dense_mma<D>(u, table, shifts, xs, ys, threadIdx.x & 31);
  }
  __syncthreads();
  long long* y = G.Y + b * St::YWORDS + (int64_t)row * P;
  for (int i = 16 * m0 * P + threadIdx.x; i < min(16 * m1, size) * P; i += 256) y[i] = ys[i];
}

// nodes of the planes z = cz and its mirror image, batch first + b
template <int DIM>
__device__ __forceinline__ void patch_merge(const StageJob& G, uint32_t b, int cz) {
  const DenseJob<double>& J = G.J;
  constexpr int M = kPatchM;
  using St = Stage<DIM>;
  using S = typename St::S;
  using L = Lines<DIM, M>;
  constexpr int P = St::P, MP2 = St::MP2, ZP = St::ZP;
  extern __shared__ __align__(16) unsigned char smraw[];
  double* Z = reinterpret_cast<double*>(smraw);
  const int pn = threadIdx.x % P;
  const int N1 = K * J.n + 1;
  const int* orbitexp = reinterpret_cast<const int*>(J.table + St::D::FRAGS) + S::ROWS;
  __shared__ int s_count;
  const int* words = G.words + b * 2 * P;
  const int word = words[pn];
  const int ve = J.vexp + (word & 0xFFF) - (word & (1 << 12) ? 100 : 0);
  const long long* Y = G.Y + b * St::YWORDS;
  for (int cy = threadIdx.x / P; cy < S::E; cy += 128 / P) {
    const L ln(cy + S::E * cz);
    long long v[L::IMAGES][M];
#pragma unroll
    for (int b = 0; b < L::IMAGES; ++b) {
      const bool in = ln.has(b);
      for_coefs<DIM, M>(b, [&](int i, int s, int ox) {
        v[b][i] = in ? __ldg(Y + (S::row(s) + ox + ln.coef(s)) * P + pn) : 0ll;
      });
    }
    reflect<DIM, M>(v);
    const int* oe = orbitexp + S::E * (cy + S::E * cz);
#pragma unroll
    for (int b = 0; b < L::IMAGES; ++b)
      if (ln.has(b)) {
        double* z = Z + pn * ZP + (b >> 1) * MP2 + M * ((b & 1) ? M - 1 - cy : cy);
#pragma unroll
        for (int i = 0; i < M; ++i)
          z[i] = word & (1 << 13) ? __longlong_as_double(0x7FF8000000000000ll)
                                  : double_of(v[b][i], J.cmul, ve - __ldg(oe + (i < S::E ? i : M - 1 - i)));
      }
  }
  const bool any = __syncthreads_or((unsigned)words[P + pn] != kNoSpikes);
  const int64_t N = (int64_t)N1 * N1 * N1;
  const int planes = cz == S::E - 1 ? 1 : 2;
  for (int gp = threadIdx.x >> 5; gp < P; gp += 4) {
    const PatchOrigin o = patch_origin<DIM>(J, (G.first + b) * P + gp);
    if (!o.active) break;
    constexpr int NO = (2 * MP2 + 31) / 32;
    double u[NO];
    auto node = [&](int i) {
      const int pl = i >= MP2, r = (i - pl * MP2) / M, ix = i - pl * MP2 - r * M, iz = pl ? M - 1 - cz : cz;
      return J.dst + (J.colour < 0 ? o.colour * N : 0) + o.base + ix + N1 * (r + N1 * iz);
    };
    if (J.colour >= 0) {  // one patch of the colour per node; all loads before the first store
#pragma unroll
      for (int j = 0; j < NO; ++j) {
        const int i = (threadIdx.x & 31) + 32 * j;
        if (i < planes * MP2) u[j] = *node(i);
      }
    }
#pragma unroll
    for (int j = 0; j < NO; ++j) {
      const int i = (threadIdx.x & 31) + 32 * j;
      if (i < planes * MP2) *node(i) = J.colour < 0 ? Z[gp * ZP + i] : u[j] + Z[gp * ZP + i];
    }
  }
  if (!any) return;
  // the spikes' part of this block's planes of the uneven patches
  const double* columns = reinterpret_cast<const double*>(reinterpret_cast<const char*>(J.table) + St::D::COLUMNS);
  unsigned short* list = reinterpret_cast<unsigned short*>(Z + S::NODES);
#pragma unroll 1
  for (int gp = 0; gp < P; ++gp) {
    const unsigned bound = (unsigned)words[P + gp];
    if (bound == kNoSpikes) continue;
    const PatchOrigin o = patch_origin<DIM>(J, (G.first + b) * P + gp);
    __syncthreads();
    for (int i = threadIdx.x; i < S::NODES; i += 128) Z[i] = J.r[o.base + i % M + N1 * (i / M % M + N1 * (i / MP2))];
    __syncthreads();
    const int count = list_spikes<S::NODES>(Z, bound, list, &s_count);
    for (int i = threadIdx.x; i < planes * MP2; i += 128) {
      const int pl = i >= MP2, q = i - pl * MP2, iz = pl ? M - 1 - cz : cz;
      J.dst[(J.colour < 0 ? o.colour * N : 0) + o.base + q % M + N1 * (q / M + N1 * iz)] +=
          J.c * spikes_at<DIM, M>(columns, Z, list, count, q + MP2 * iz);
    }
  }
}

// one run, and the runs of several levels (blockIdx.x numbers the batches)
template <int DIM>
__global__ void __launch_bounds__(256) patch_split_kernel(const __grid_constant__ StageJob G) {
  patch_split<DIM>(G, blockIdx.x);
}
template <int DIM>
__global__ void __launch_bounds__(256) patch_split_group_kernel(const __grid_constant__ GroupOf<StageJob> G) {
  const int j = group_find(G, blockIdx.x);
  patch_split<DIM>(G.job[j], blockIdx.x - (uint32_t)G.start[j]);
}
template <int DIM>
__global__ void __launch_bounds__(256, 2) patch_product_kernel(const __grid_constant__ StageJob G) {
  patch_product<DIM>(G, blockIdx.x, blockIdx.y);
}
template <int DIM>
__global__ void __launch_bounds__(256, 2) patch_product_group_kernel(const __grid_constant__ GroupOf<StageJob> G) {
  const int j = group_find(G, blockIdx.x);
  patch_product<DIM>(G.job[j], blockIdx.x - (uint32_t)G.start[j], blockIdx.y);
}
template <int DIM>
__global__ void __launch_bounds__(128) patch_merge_kernel(const __grid_constant__ StageJob G) {
  patch_merge<DIM>(G, blockIdx.x, blockIdx.y);
}
template <int DIM>
__global__ void __launch_bounds__(128) patch_merge_group_kernel(const __grid_constant__ GroupOf<StageJob> G) {
  const int j = group_find(G, blockIdx.x);
  patch_merge<DIM>(G.job[j], blockIdx.x - (uint32_t)G.start[j], blockIdx.y);
}

// K = 1: the patch is its vertex, the local solve one multiplication by
// c = omega_AS / A_{j,1} (additive) or 1 / A_{j,1}.
template <int DIM, typename T>
__device__ __forceinline__ void point_body(const DenseJob<T>& J, uint32_t pid) {
  const uint32_t r1 = J.d0.div(pid), r2 = J.d1.div(r1);
  const int i[3] = {(int)(pid - r1 * J.d0.d), (int)(DIM == 3 ? r1 - r2 * J.d1.d : r1), (int)(DIM == 3 ? r2 : 0)};
  int v[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) v[d] = J.colour < 0 ? i[d] + 1 : 2 * i[d] + (((J.colour >> d) & 1) ? 1 : 2);
  const int64_t N1 = J.n + 1, node = v[0] + N1 * (v[1] + (DIM == 3 ? N1 * v[2] : 0));
  const int64_t N = DIM == 3 ? N1 * N1 * N1 : N1 * N1;
  const int pc = (v[0] & 1) | ((v[1] & 1) << 1) | (DIM == 3 ? (v[2] & 1) << 2 : 0);
  if (J.colour < 0) J.dst[pc * N + node] = J.c * J.r[node];
  else J.dst[node] += J.c * J.r[node];
}

template <int DIM, typename T>
__global__ void __launch_bounds__(256) patch_point_kernel(const __grid_constant__ DenseJob<T> J) {
  const uint32_t t = blockIdx.x * 256u + threadIdx.x;
  if (t < J.npatch) point_body<DIM, T>(J, t);
}

template <int DIM, typename T>
__global__ void __launch_bounds__(256) patch_point_group_kernel(const __grid_constant__ GroupOf<DenseJob<T>> G) {
  const int j = group_find(G, blockIdx.x);
  const uint32_t t = (uint32_t)(blockIdx.x - G.start[j]) * 256u + threadIdx.x;
  if (t < G.job[j].npatch) point_body<DIM, T>(G.job[j], t);
}

// ---------------------------------------------------------------- the matrix
// Columns of B at unit scale (the FP64 part serves both precisions): the local
// solver applied to the unit vectors of the orbits' first nodes, one node per
// patch of the block; column[orbit][node], hi + lo (lo only with V = dd).  A
// further local cycle (Algorithm 2, N_iter > 1) continues from them.  For FP64
// products V = dd: the matrix is rounded once, where the local solver in plain
// FP64 would leave 2-5 times the error of a solve in the products (K = 3:
// 1.1e-15 against 3.3e-16).  orbitexp: set to kNoOrbit for sector_exponents_kernel.
constexpr int kNoOrbit = 1 << 30;

template <int DIM, typename V>
__global__ void __launch_bounds__(256) patch_columns_kernel(double* __restrict__ hi, double* __restrict__ lo,
                                                            int* __restrict__ orbitexp, int np, bool first,
                                                            const double* __restrict__ dinv, PatchParams<double> H) {
  using S = Sectors<DIM, kPatchM>;
  if (sizeof(V) == 16 && blockIdx.x == 0)
    for (int i = threadIdx.x; i < S::ORBITS; i += blockDim.x) orbitexp[i] = kNoOrbit;
  using PS = PatchShape<DIM>;
  constexpr int SZT = PS::SZT, RT = PS::off_r(PS::L - 1), DT = PS::off_d(PS::L - 1);
  extern __shared__ __align__(16) unsigned char smraw[];
  const int c0 = blockIdx.x * np, nc = min(np, S::ORBITS - c0);
  const PBlock<V, 0> pb{reinterpret_cast<V*>(smraw), PS::ELEMS, nc};
  PatchParams<V> P;
  P.scale = H.scale;
  P.omega_as = H.omega_as;
  for (int i = 0; i < 4; ++i) P.omega[i] = H.omega[i];
  P.inv_a0 = H.inv_a0;
  P.inv_scale = H.inv_scale;
  P.half = H.half;
  P.colour = H.colour;
  const CartGeo<DIM, V> geo{dinv, P.scale, P.inv_scale, P.inv_a0};
  auto value = [&](int64_t t) {
    if constexpr (sizeof(V) == 16) return V(hi[t], lo[t]);
    else return V(hi[t]);
  };
  pfor<SZT>(pb, [&](int g, int i) {
    pb.at(g)[RT + i] = V(i == Orbit<DIM, kPatchM>(c0 + g).node(0) ? 1.0 : 0.0);
    if (!first) pb.at(g)[DT + i] = value((int64_t)(c0 + g) * SZT + i);
  });
  __syncthreads();
  if constexpr (PS::L > 1) {
    if (!first) geo.template resid<PS::L - 1>(pb, DT, RT, RT);  // r = e_j - A x
  }
  pvcycle<DIM, PS::L - 1>(pb, geo, P);
  pfor<SZT>(pb, [&](int g, int i) {
    const int64_t t = (int64_t)(c0 + g) * SZT + i;
    V d = pb.at(g)[DT + i];
    if (!first) d = value(t) + d;
    if constexpr (sizeof(V) == 16) {
      const double v = value_of(d);
      lo[t] = (d.hi - v) + d.lo;
      hi[t] = v;
    } else {
      hi[t] = d;
    }
  });
}

// Columns of the element stiffness matrix of Eq. (3) at unit scale, from the
// 1D element matrices; as patch_columns_kernel
template <int DIM>
__global__ void __launch_bounds__(256) cell_columns_kernel(double* __restrict__ hi, double* __restrict__ lo,
                                                           int* __restrict__ orbitexp) {
  constexpr int M = kCellM;
  using S = Sectors<DIM, M>;
  const int t = blockIdx.x * 256 + threadIdx.x;
  if (t < S::ORBITS) orbitexp[t] = kNoOrbit;
  if (t >= S::ORBITS * S::NODES) return;
  const Orbit<DIM, M> o(t / S::NODES);
  const int i = t % S::NODES, c[3] = {i % M, (i / M) % M, i / (M * M)};
  dd acc(0.0);
#pragma unroll
  for (int d = 0; d < DIM; ++d) {
    dd p(1.0);
#pragma unroll
    for (int e = 0; e < DIM; ++e) p = c_tab64[(d == e ? LAY.Ke : LAY.Me) + c[e] * M + o.c[e]] * p;
    acc += p;
  }
  const double v = value_of(acc);
  hi[t] = v;
  lo[t] = (acc.hi - v) + acc.lo;
}

// coefficient k of sector s: its orbit
template <int DIM, int M>
__device__ __forceinline__ Orbit<DIM, M> orbit_of(int s, int k) {
  using S = Sectors<DIM, M>;
  const int e0 = S::ext(s, 0), e1 = S::ext(s, 1);
  return Orbit<DIM, M>(k % e0 + S::E * ((k / e0) % e1 + S::E * (k / (e0 * e1))));
}

// Entry of row om and coefficient oj of sector s: the signed sum over the
// mirror images of om's node of the operator's entry for oj's node, over 2^d
// -- the operand of an orbit with c central coordinates, which has only
// 2^(d-c) images, counts 2^c times.
// V = dd, or double without lo.
template <typename V, int DIM, int M>
__device__ __forceinline__ V sector_entry(const double* __restrict__ hi, const double* __restrict__ lo, int s,
                                          const Orbit<DIM, M>& om, const Orbit<DIM, M>& oj) {
  using S = Sectors<DIM, M>;
  const int64_t col = (int64_t)(oj.c[0] + S::E * (oj.c[1] + S::E * oj.c[2])) * S::NODES;
  V a(0.0);
#pragma unroll
  for (int b = 0; b < S::IMAGES; ++b) {
    if (S::IMAGES > 1 && !oj.has(b)) continue;
    const int64_t t = col + om.node(b);
    const double sg = (__popc(s & b) & 1) ? -1.0 / S::IMAGES : 1.0 / S::IMAGES;
    if constexpr (sizeof(V) == 16) a += V(sg * hi[t], sg * lo[t]);
    else a += sg * hi[t];
  }
  return a;
}

// Exponents of the sector matrices, one warp per row.
// rowexp: the largest exponent x with entry 2^x below 0.98 2^63 (8 signed
// digits reach 127/128 of 2^63) and the row's sum of magnitudes times 2^x
// below 2^65 (results and their even / odd sums stay within 64 bits).  The
// sectors' results for one orbit are summed, so they need a common exponent:
// minexp, the least one of the orbit's rows (kNoExp in the first if an entry is not finite).
template <int DIM, int M>
__global__ void __launch_bounds__(128) sector_exponents_kernel(const double* __restrict__ hi,
                                                               int* __restrict__ rowexp, int* __restrict__ minexp) {
  using S = Sectors<DIM, M>;
  const int row = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= S::ROWS) return;
  int s = 0;
  while (s + 1 < S::NS && row >= S::row(s + 1)) ++s;
  const int m = row - S::row(s), sz = S::size(s);
  const Orbit<DIM, M> om = orbit_of<DIM, M>(s, m);
  double top = 0.0, sum = 0.0;
  for (int k = lane; k < sz; k += 32) {
    const double a = fabs(sector_entry<double, DIM, M>(hi, nullptr, s, om, orbit_of<DIM, M>(s, k)));
    top = fmax(top, a);
    sum += a;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    top = fmax(top, __shfl_xor_sync(0xffffffffu, top, o));
    sum += __shfl_xor_sync(0xffffffffu, sum, o);
  }
  if (lane) return;
  int te = 0, se = 0;
  if (frexp(top, &te) > 0.98) ++te;
  frexp(sum, &se);
  const int x = sum == 0.0 ? 1000 : min(63 - te, 65 - se);
  rowexp[row] = x;
  atomicMin(minexp + om.c[0] + S::E * (om.c[1] + S::E * om.c[2]), x);
  if (!isfinite(sum)) atomicMin(minexp, kNoExp);
}

// Fragments of the first operand of mma.m16n8k16, per 16 x 16 tile and part:
// lane l holds rows l / 4 and l / 4 + 8, columns 2 (l % 4) and + 8.  FP64:
// 8-bit signed digits of entry 2^(the row's exponent, at most 15 above its
// orbit's); FP32: three BF16 parts, rounded.
template <int DIM, typename T, int M>
__global__ void __launch_bounds__(256) sector_table_kernel(const double* __restrict__ hi, const double* __restrict__ lo,
                                                           const int* __restrict__ rowexp,
                                                           const int* __restrict__ minexp,
                                                           uint32_t* __restrict__ table) {
  using S = Sectors<DIM, M>;
  using D = Dense<DIM, M, T>;
  constexpr int SL = D::SL;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int* tail = reinterpret_cast<int*>(table + (int64_t)D::FRAGS * 4);
  if (sizeof(T) == 8 && t < S::ORBITS) tail[S::ROWS + t] = minexp[t];
  if (t >= (int64_t)S::TILES * 32 * 4) return;
  const int reg = (int)(t & 3), lane = (int)(t >> 2) & 31, tile = (int)(t >> 7);
  int s = 0;
  while (s + 1 < S::NS && tile >= S::tile(s + 1)) ++s;
  const int nt = S::tiles(s), sz = S::size(s), mt = (tile - S::tile(s)) / nt, kt = (tile - S::tile(s)) % nt;
  const int m = 16 * mt + (lane >> 2) + 8 * (reg & 1), k0 = 16 * kt + 2 * (lane & 3) + 8 * (reg >> 1);
  const Orbit<DIM, M> om = orbit_of<DIM, M>(s, m < sz ? m : 0);
  int re = 0;
  if (sizeof(T) == 8 && m < sz) {
    const int exp = minexp[om.c[0] + S::E * (om.c[1] + S::E * om.c[2])];
    re = min(rowexp[S::row(s) + m], exp + 15);
    if (kt == 0 && (lane & 3) == 0 && reg < 2) tail[S::row(s) + m] = re - exp;
  }
  uint32_t part[SL] = {};
  for (int h = 0; h < 2; ++h) {
    const int k = k0 + h;
    const Orbit<DIM, M> oj = orbit_of<DIM, M>(s, k < sz ? k : 0);
    using V = std::conditional_t<sizeof(T) == 8, dd, double>;
    const V a = m < sz && k < sz ? sector_entry<V, DIM, M>(hi, lo, s, om, oj) : V(0.0);
    if constexpr (sizeof(T) == 8) {
      const long long w = __double2ll_rn(scalbn(a.hi, re)) + __double2ll_rn(scalbn(a.lo, re));
      const unsigned long long v = (unsigned long long)w + D::BIAS;
      for (int i = 0; i < SL; ++i) {
        const int digit = (int)((v >> (8 * (SL - 1 - i))) & 0xFF) - 128;
        part[i] |= (uint32_t)__half_as_ushort(__int2half_rn(digit)) << (16 * h);
      }
    } else {
      // FP32 operands are plain sums over the images
      double rest = a * (1 << oj.centres());
      for (int i = 0; i < SL; ++i) {
        const __nv_bfloat16 p = __double2bfloat16(rest);
        rest -= (double)__bfloat162float(p);
        part[i] |= (uint32_t)__bfloat16_as_ushort(p) << (16 * h);
      }
    }
  }
  for (int i = 0; i < SL; ++i) table[(((int64_t)tile * SL + i) * 32 + lane) * 4 + reg] = part[i];
}

}  // namespace PMG_KNS
}  // namespace pmg
