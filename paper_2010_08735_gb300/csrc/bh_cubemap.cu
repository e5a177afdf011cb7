// Star cube map build (Sec. 3.3.2 "Emitted light", Sec. 4).
//
// Each texel holds the colour SUM of the stars it contains and their
// luminance-weighted mean position inside the texel; a mip texel sums the
// colours of its 4 children and averages their positions weighted by Y
// (Sec. 3.3.2).  The paper derives the in-texel position from a hash of the
// colour; here it is stored explicitly as two unorm8 (reading C15).
//
// Determinism: colours are accumulated as 64-bit fixed point (2^-20 units)
// with integer atomics, so the sums do not depend on the order in which
// threads arrive; the position averages are those of FP64 arithmetic in one
// fixed child order with round-to-nearest (this file is compiled without
// multiply-add contraction).  The build is therefore bit-for-bit
// reproducible.
//
// Layout: records of 4 x 16 bit -- X, Y, Z (half or bfloat16 of the colour
// sum divided by 4^level, so that coarse levels stay in range) and the
// position word (s in the low byte, t in the high byte) -- level-major, then
// face (+x,-x,+y,-y,+z,-z), row t, column s.
//
// How it runs.  The floor is the write of the records (268 MB for faces of
// 2048^2: 40 us), but GB300 does two FP64 multiply-adds per SM and clock, so
// arithmetic decides: a star's black body was 95 exponentials (8 ms for 1M
// stars), now two polynomials (chroma_kernel).  Stars are sorted by region (32
// x 32 texels of level 0) and one block builds a region's six levels from
// them in shared memory, writing every record once; the last block of 32 x 32
// regions to finish builds the next five levels.  Dense accumulators in global
// memory (64 bytes a texel, cleared, summed and read back level by level)
// moved 4 GB for those 268 MB.  1M stars on 2048^2 faces: fit 18 us, bins 44,
// places 4, colours 74 (FP64 at 86 % of its rate), regions 231, mask of the
// small levels 8 -- 0.38 ms where the kernels took 15.9 ms; 20,000 stars on
// 128^2 faces 46 us instead of 419.
#include <algorithm>
#include <cmath>

#include "bh_colour.cuh"
#include "bh_internal.cuh"

namespace bh {

constexpr double kXyzScale = 1048576.0;  // 2^20

// ---------------------------------------------------------------------------
// Chromaticity of black bodies
//
// A star's colour is its luminosity times (X, Y, Z) / (X + Y + Z) of a black
// body, a smooth function of 1/T alone.  For T in [1024 K, 1e9 K] it is
// read off polynomials of degree 8 in 1/T on 64 equal cells of [0, 1/1024 K]
// (Chebyshev nodes; a cell spans 0.6 in h c / (lambda k T) at 360 nm), fitted on
// the device at each build: 576 black bodies instead of one per star.  Relative
// error over the fitted range against extended precision: at most 1.4e-15 (the
// FP64 sum over the wavelengths itself: 2.2e-15).
// ---------------------------------------------------------------------------
constexpr int kChromaCells = 64, kChromaNodes = 9;
constexpr double kChromaTMin = 1024.0, kChromaTMax = 1e9;
constexpr int kChromaStride = 2 * kChromaNodes + 2;  // X and Z coefficients, minus twice the cell's centre, pad
constexpr int kChromaCoefs = kChromaCells * kChromaStride, kChromaVals = kChromaCells * kChromaNodes * 2;

using ChromaFit = BlackBodyFit<kChromaNodes>;

// One warp (a block of its own: 576 of them spread over the SMs) per node, 45
// FP64 operations per wavelength, whose constants come from the host; the last
// node of a cell to finish fits the cell.  The block past the nodes writes the
// matching functions, for stars outside the fitted range.
__global__ void chroma_kernel(const ChromaFit fit, double *cmf_out, double *val, unsigned *done, double *coef) {
  const int lane = threadIdx.x, cell = blockIdx.x / kChromaNodes, node = blockIdx.x - cell * kChromaNodes;
  if (cell == kChromaCells) {
    for (int k = lane; k < kNLambda; k += 32)
      for (int c = 0; c < 3; ++c) cmf_out[3 * k + c] = fit.cmf[c][k];
    return;
  }
  const double v = (cell + 0.5 * (fit.node[node] + 1.0)) * (1.0 / (kChromaCells * kChromaTMin));  // 1/T
  double s[3] = {0.0, 0.0, 0.0};
  for (int k = lane; k < kNLambda; k += 32) {
    const double b = 1.0 / expm1(fit.x[k] * v);
    for (int c = 0; c < 3; ++c) s[c] = fma(b, fit.w[c][k], s[c]);
  }
  for (int o = 16; o > 0; o >>= 1)
    for (int c = 0; c < 3; ++c) s[c] += __shfl_xor_sync(0xffffffffu, s[c], o);
  unsigned before = 0;
  if (lane == 0) {
    const double sum = 1.0 / (s[0] + s[1] + s[2]);
    val[blockIdx.x * 2] = s[0] * sum;
    val[blockIdx.x * 2 + 1] = s[2] * sum;
    __threadfence();
    before = atomicAdd(done + cell, 1u);
    __threadfence();
  }
  if (__shfl_sync(0xffffffffu, before, 0) != kChromaNodes - 1u) return;
  double *out = coef + cell * kChromaStride;
  if (lane < 2 * kChromaNodes) {
    const int c = lane / kChromaNodes, m = lane - c * kChromaNodes;
    out[lane] = fit_coefficient(fit, m, val + cell * kChromaNodes * 2 + c, 2);
  } else if (lane == 2 * kChromaNodes) {
    out[lane] = -(2.0 * cell + 1.0);
  }
}

// val: kChromaVals doubles of scratch; done: kChromaCells counters, zero.
static void chroma_launch(double *cmf, double *val, unsigned *done, double *coef, cudaStream_t s) {
  chroma_kernel<<<kChromaCells * kChromaNodes + 1, 32, 0, s>>>(black_body_fit<kChromaNodes>(), cmf, val, done, coef);
}

// 1/b by Newton's iteration from the float reciprocal (b a normal float whose
// reciprocal is one): 2^-23, 2^-46, then rounding.
__device__ __forceinline__ double newton_rcp(float bf, double b) {
  double r = (double)__frcp_rn(bf);
  r = fma(r, fma(-b, r, 1.0), r);
  return fma(r, fma(-b, r, 1.0), r);
}

// Emitted XYZ of a star (black body of its temperature scaled to its
// luminosity X+Y+Z, rounded to float) in 2^-20 units.
__device__ __forceinline__ void star_colour(const bh_star &st, const double *cmf, const double *coef, long long *q) {
  const double lum = (double)st.lum;
  float xf[3];
  if (st.temp_K >= (float)kChromaTMin && st.temp_K <= (float)kChromaTMax) {
    // 32 FP64 operations, which bound the kernel (98 us for 1M stars with a
    // divide and 64-bit conversions)
    const double r = newton_rcp(st.temp_K, (double)st.temp_K);
    const int cell = min((int)((float)(kChromaCells * kChromaTMin) * __frcp_rn(st.temp_K)), kChromaCells - 1);
    const double *a = coef + cell * kChromaStride, *b = a + kChromaNodes;
    const double u = fma(2.0 * kChromaCells * kChromaTMin, r, a[2 * kChromaNodes]);
    double x = a[kChromaNodes - 1], z = b[kChromaNodes - 1];
#pragma unroll
    for (int m = kChromaNodes - 2; m >= 0; --m) {
      x = fma(x, u, a[m]);
      z = fma(z, u, b[m]);
    }
    xf[0] = (float)(lum * x);
    xf[1] = (float)(lum * ((1.0 - x) - z));
    xf[2] = (float)(lum * z);
  } else {
    double b[3];
    dblackbody_xyz(cmf, (double)st.temp_K, b);
    const double s = __dadd_rn(__dadd_rn(b[0], b[1]), b[2]);
    for (int c = 0; c < 3; ++c) xf[c] = (float)__ddiv_rn(__dmul_rn(lum, b[c]), s);
  }
  // in units of 2^-20, to the nearest integer: below 2^23 by the 32-bit
  // conversion, above it the float is an integer, its mantissa shifted
  for (int c = 0; c < 3; ++c) {
    const float f = xf[c] * 1048576.f, m = fabsf(f);
    if (m < 8388608.f) q[c] = __float2int_rn(f);
    else if (m < 1.8e19f / 2) {
      const unsigned bits = __float_as_uint(m);
      const long long v = (long long)((bits & 0x7fffffu) | 0x800000u) << ((bits >> 23) - 150);
      q[c] = f < 0.f ? -v : v;
    } else q[c] = __double2ll_rn(__dmul_rn((double)xf[c], kXyzScale));  // out of range or not a number
  }
}

// GL major-axis face and face coordinates (sc, tc, |ma|).
__device__ __forceinline__ int cube_face_f(float x, float y, float z, float &sc, float &tc, float &ma) {
  const float ax = fabsf(x), ay = fabsf(y), az = fabsf(z);
  if (ax >= ay && ax >= az) {
    ma = ax;
    if (x >= 0.f) { sc = -z; tc = -y; return 0; }
    sc = z; tc = -y; return 1;
  }
  if (ay >= az) {
    ma = ay;
    if (y >= 0.f) { sc = x; tc = z; return 2; }
    sc = x; tc = -z; return 3;
  }
  ma = az;
  if (z >= 0.f) { sc = x; tc = -y; return 4; }
  sc = -x; tc = -y; return 5;
}

// Face, texel and 16-bit position inside the texel of a star.
struct StarTexel {
  int face, i, j;
  unsigned s16, t16;
};

__device__ __forceinline__ StarTexel star_texel(const bh_star &st, int N) {
  float sc, tc, ma;
  StarTexel r;
  r.face = cube_face_f(st.dir[0], st.dir[1], st.dir[2], sc, tc, ma);
  // floor(65536 N (sc/ma + 1)/2) holds the column (above 16 bits) and the position
  const double scale = 32768.0 * N;
  long long S, T;
  if (ma >= 1e-30f && ma <= 1e30f) {
    // One reciprocal for both quotients, each put right by its exact remainder
    // (Markstein: the quotient rounds as a division would); the floor is the low
    // word of a sum rounded down onto the integers above 2^52.
    const double b = (double)ma, rb = newton_rcp(ma, b);
    auto place = [&](double a) {
      const double q0 = a * rb, q = fma(fma(-q0, b, a), rb, q0);
      return (long long)(unsigned)__double2loint(__fma_rd(__dadd_rn(q, 1.0), scale, 4503599627370496.0));
    };
    S = place((double)sc);
    T = place((double)tc);
  } else {
    S = __double2ll_rd(__dmul_rn(__dadd_rn(__ddiv_rn((double)sc, (double)ma), 1.0), scale));
    T = __double2ll_rd(__dmul_rn(__dadd_rn(__ddiv_rn((double)tc, (double)ma), 1.0), scale));
  }
  const long long most = (long long)N << 16;
  auto split = [&](long long v, int &cell, unsigned &pos) {
    if (v < 0) { cell = 0; pos = 0; }                          // a direction that is not a number
    else if (v >= most) { cell = N - 1; pos = 65535; }         // the far edge
    else { cell = (int)(v >> 16); pos = (unsigned)v & 65535u; }
  };
  split(S, r.i, r.s16);
  split(T, r.j, r.t16);
  return r;
}

// ---------------------------------------------------------------------------
// Records
// ---------------------------------------------------------------------------

// v / 2^k as half (at most 65504) or bfloat16, one rounding: the sum is first
// rounded to odd in 24 bits (13 or more beyond the result's).  32-bit integer
// work: conversions of 64-bit integers run at the FP64 rate.
__device__ __forceinline__ unsigned short enc16(long long v, int k, int dtype) {
  unsigned long long u = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
  const int lz = u ? __clzll(u) : 0;
  u <<= lz;
  const unsigned m = (unsigned)(u >> 40) | ((u & 0xffffffffffull) ? 1u : 0u);
  float f = __uint2float_rn(m) * __int_as_float((127 + 40 - lz - k) << 23);
  if (v < 0) f = -f;
  if (dtype == BH_BF16) return __bfloat16_as_ushort(__float2bfloat16_rn(f));
  return __half_as_ushort(__float2half_rn(fminf(f, 65504.f)));
}

__device__ __forceinline__ uint2 make_record(long long x, long long y, long long z, unsigned p, int L, int dtype) {
  const int k = 20 + 2 * L;
  return make_uint2((unsigned)enc16(x, k, dtype) | ((unsigned)enc16(y, k, dtype) << 16),
                    (unsigned)enc16(z, k, dtype) | (p << 16));
}

__device__ __forceinline__ float approx_float(long long v) {  // v >= 0, to 2^-23
  return fmaf(__uint2float_rn((unsigned)((unsigned long long)v >> 32)), 4294967296.f, __uint2float_rn((unsigned)v));
}

// floor(num / den) for 0 <= num <= 256 den, den > 0: a float estimate is off by
// one at most and put right in integers.
__device__ __forceinline__ int small_quotient(long long num, long long den) {
  const int p = (int)__fdividef(approx_float(num), approx_float(den));
  const long long r = num - p * den;
  return r < 0 ? p - 1 : r >= den ? p + 1 : p;
}

// Mean position byte at level 0 from y = sum of Y and a = sum of Y * s16:
// floor(256 (a/y + 1/2)/65536).  Rounding FP64 cannot carry the mean over a
// byte boundary while y is below 2^35 (its distance from one is at least 1/(512
// y)), so the quotient is taken in integers there.
__device__ __forceinline__ int mean_byte0(long long a, long long y) {
  if (y < (1LL << 35) && a >= 0 && a <= 65535 * y) return min(small_quotient(2 * a + y, 512 * y), 255);
  const double f = __ddiv_rn(__dadd_rn(__ddiv_rn((double)a, (double)y), 0.5), 65536.0);
  return min((int)floor(__dmul_rn(f, 256.0)), 255);
}

// A texel's sums and mean position (s | t << 8).
struct alignas(16) Node {
  long long x, y, z;
  unsigned p, pad;
};

constexpr unsigned kNoPosition = 128u | (128u << 8);  // of a texel without Y
constexpr uint2 kEmptyRecord = {0u, kNoPosition << 16};

// A mip texel from its children in the order (a,b) = (0,0), (1,0), (0,1),
// (1,1), a the column and b the row offset: sums, and the Y-weighted mean
// position floor(256 sum(cy (a + (p + 1/2)/256)/2) / sum(cy)).  As above,
// integers give the FP64 result while the weights sum to less than 2^40.
__device__ __forceinline__ Node mip_node(const Node *c) {
  Node r = {0, 0, 0, kNoPosition, 0};
  bool plain = true;
  for (int k = 0; k < 4; ++k) {
    r.x += c[k].x;
    r.y += c[k].y;
    r.z += c[k].z;
    plain = plain && c[k].y >= 0 && c[k].y < (1LL << 40);
  }
  if (r.y <= 0) return r;
  int ps, pt;
  if (plain && r.y < (1LL << 40)) {
    long long ns = 0, nt = 0;
    for (int k = 0; k < 4; ++k) {
      ns += c[k].y * (long long)((k & 1) * 512 + 2 * (c[k].p & 255) + 1);
      nt += c[k].y * (long long)((k >> 1) * 512 + 2 * (c[k].p >> 8) + 1);
    }
    ps = min(small_quotient(ns, 4 * r.y), 255);
    pt = min(small_quotient(nt, 4 * r.y), 255);
  } else {
    double ns = 0.0, nt = 0.0;
    for (int k = 0; k < 4; ++k) {
      const double cs = __ddiv_rn((double)(c[k].p & 255) + 0.5, 256.0), ct = __ddiv_rn((double)(c[k].p >> 8) + 0.5, 256.0);
      ns = __dadd_rn(ns, __dmul_rn((double)c[k].y, __dmul_rn(__dadd_rn((double)(k & 1), cs), 0.5)));
      nt = __dadd_rn(nt, __dmul_rn((double)c[k].y, __dmul_rn(__dadd_rn((double)(k >> 1), ct), 0.5)));
    }
    ps = min((int)floor(__dmul_rn(__ddiv_rn(ns, (double)r.y), 256.0)), 255);
    pt = min((int)floor(__dmul_rn(__ddiv_rn(nt, (double)r.y), 256.0)), 255);
  }
  r.p = (unsigned)(ps | (pt << 8)) & 0xffffu;
  return r;
}

// ---------------------------------------------------------------------------
// Stars to regions of 32 x 32 level-0 texels (the whole face below that)
// ---------------------------------------------------------------------------
constexpr int kRegion = 32, kRegionTexels = kRegion * kRegion;

struct alignas(16) StarBin {
  unsigned texel;  // region * 1024 + row * 32 + column
  unsigned pos;    // s16 | t16 << 16
  unsigned long long rank;  // of the star in its region
};

struct alignas(16) StarItem {  // a star in region order
  long long q[3];
  unsigned pos, local;
};

__global__ void star_bin_kernel(const bh_star *stars, long long n, int N, unsigned long long *count, StarBin *bins) {
  const long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const unsigned active = __ballot_sync(0xffffffffu, k < n);
  if (k >= n) return;
  const StarTexel t = star_texel(stars[k], N);
  const int nr = max(N / kRegion, 1);
  const unsigned region = (t.face * nr + t.j / kRegion) * nr + t.i / kRegion;
  // one atomic per region and warp: fields may be clustered
  const unsigned same = __match_any_sync(active, region);
  const int lane = threadIdx.x & 31, leader = __ffs(same) - 1;
  unsigned long long base = 0;
  if (lane == leader) base = atomicAdd(count + region, (unsigned long long)__popc(same));
  base = __shfl_sync(same, base, leader);
  StarBin b;
  b.texel = region * kRegionTexels + (t.j % kRegion) * kRegion + t.i % kRegion;
  b.pos = t.s16 | (t.t16 << 16);
  b.rank = base + __popc(same & ((1u << lane) - 1u));
  bins[k] = b;
}

struct RegionSpan {
  unsigned long long first, count;  // a region's stars in items
};

// A region's block reads its items once per band of rows, alone: 1M stars in one
// region took 22.3 ms, 4M on faces of 32^2 28.0.  A crowded region -- one whose
// items have room for the sums X, Y, Z, Y s16, Y t16 of every texel (5 words
// each) -- holds those sums there instead, added by every star's own thread: 0.70
// and 0.53 ms, 400,000 uniform stars on 128^2 (4,167 a region) 380 -> 180 us.
// Just below the line (1,250 a region) the bands are as fast: 139 against 128 us
// for 120,000 on 128^2.
constexpr unsigned long long kCrowded = 5 * sizeof(unsigned long long) * kRegionTexels / sizeof(StarItem);

// Place of each region's stars, in any order of regions; the sums of crowded
// ones are cleared.  One warp per block.
__global__ void region_span_kernel(const unsigned long long *count, int regions, unsigned long long *cursor,
                                   RegionSpan *span, StarItem *items) {
  const int lane = threadIdx.x, r = blockIdx.x * 32 + lane;
  const unsigned long long c = r < regions ? count[r] : 0;
  unsigned long long s = c;
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long v = __shfl_up_sync(0xffffffffu, s, o);
    if (lane >= o) s += v;
  }
  unsigned long long base = 0;
  if (lane == 31) base = atomicAdd(cursor, s);
  base = __shfl_sync(0xffffffffu, base, 31);
  const unsigned long long first = base + s - c;
  if (r < regions) span[r] = {first, c};
  for (unsigned crowded = __ballot_sync(0xffffffffu, c >= kCrowded); crowded; crowded &= crowded - 1u) {
    uint4 *sums = reinterpret_cast<uint4 *>(items + __shfl_sync(0xffffffffu, first, __ffs(crowded) - 1));
    for (int k = lane; k < (int)(kCrowded * sizeof(StarItem) / sizeof(uint4)); k += 32) sums[k] = make_uint4(0u, 0u, 0u, 0u);
  }
}

// A star's colour and position into the sums of its texel.
__device__ __forceinline__ void star_sum(unsigned long long *a, const long long *q, unsigned s16, unsigned t16) {
  for (int c = 0; c < 3; ++c) atomicAdd(a + c, (unsigned long long)q[c]);
  atomicAdd(a + 3, (unsigned long long)(q[1] * (long long)s16));
  atomicAdd(a + 4, (unsigned long long)(q[1] * (long long)t16));
}

__global__ void star_scatter_kernel(const bh_star *stars, long long n, const StarBin *bins, const RegionSpan *span,
                                    const double *cmf, const double *coef, StarItem *items) {
  const long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (k >= n) return;
  const StarBin b = bins[k];
  const RegionSpan at = span[b.texel / kRegionTexels];
  StarItem it;
  star_colour(stars[k], cmf, coef, it.q);
  it.pos = b.pos;
  it.local = b.texel % kRegionTexels;
  if (at.count < kCrowded) items[at.first + b.rank] = it;
  else star_sum(reinterpret_cast<unsigned long long *>(items + at.first) + it.local * 5, it.q, b.pos & 0xffffu, b.pos >> 16);
}

// Without room for a sorted copy: the sums X, Y, Z, Y s16, Y t16 of every
// level-0 texel in global memory (5 words each, zero at the start).
__global__ void star_accumulate_kernel(const bh_star *stars, long long n, int N, const double *cmf,
                                       const double *coef, unsigned long long *acc) {
  const long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (k >= n) return;
  const bh_star st = stars[k];
  long long q[3];
  star_colour(st, cmf, coef, q);
  const StarTexel t = star_texel(st, N);
  star_sum(acc + (((long long)t.face * N + t.j) * N + t.i) * 5, q, t.s16, t.t16);
}

// ---------------------------------------------------------------------------
// Regions to records
// ---------------------------------------------------------------------------
struct RegionParams {
  const StarItem *items;               // kSortedSlots: stars by region
  const RegionSpan *span;              // nullptr: no stars
  const unsigned long long *acc;       // kDenseSlots: the sums of every texel
  uint2 *rec;
  unsigned char *mask;                 // nullptr: no occupancy mask (or faces below a region)
  Node *nodes;                         // the top texel of every group, stage after stage
  unsigned *arrived;                   // groups finished, per group of the next stage (zero at launch)
  int N, dtype;
  long long level_off[14];             // cube_level_offset
  long long mask_off[3];               // mask_level_offset
};

static void region_levels(RegionParams &P) {
  for (int L = 0; L < 14; ++L) P.level_off[L] = (P.N >> L) ? cube_level_offset(P.N, L) : 0;
  for (int L = 0; L < 3; ++L) P.mask_off[L] = mask_level_offset(P.N, L);
}

// Threads of a region's block, and texels summed at a time: sorted stars and
// dense sums (few regions: all of a region in two bands).
constexpr int kSortedSlots = 128, kDenseSlots = 512;

template <int kSlots>
struct RegionShared {
  unsigned acc[10][kSlots];             // X, Y, Z, Y s16, Y t16 of a texel: low and high halves
  unsigned short p0[kSlots];
  unsigned short slot[kRegionTexels];   // of a texel that a star touches
  unsigned short list0[kSlots], list1[kSlots];  // the texels of levels 0 and 1 that hold sums
  unsigned touched[kRegion];            // texels of level 0 that hold sums, one word per row
  unsigned lit[3][kRegionTexels / 32];  // texels whose record has a colour, levels 0-2
  unsigned full[6][8];                  // texels of levels 1-5 that hold sums
  long long x[341], y[341], z[341];     // their sums: 256 of level 1, 64, 16, 4, 1
  unsigned short p[341];
  unsigned n0, n1;                      // lengths of the lists
  int last;
};

template <typename Shared>
__device__ __forceinline__ long long shared_sum(const Shared &sh, int c, int t) {
  return (long long)(((unsigned long long)sh.acc[2 * c + 1][t] << 32) | sh.acc[2 * c][t]);
}

// 64-bit add by two 32-bit shared atomics (which are native): the low half's
// carry goes into the high half's addend, so the sum is exact in any order.
template <typename Shared>
__device__ __forceinline__ void shared_add(Shared &sh, int c, int t, long long v) {
  const unsigned lo = (unsigned)v, hi = (unsigned)((unsigned long long)v >> 32);
  const unsigned old = atomicAdd(&sh.acc[2 * c][t], lo);
  const unsigned up = hi + (old + lo < lo ? 1u : 0u);
  if (up) atomicAdd(&sh.acc[2 * c + 1][t], up);
}

__device__ __forceinline__ int level_base(int l) { return l == 1 ? 0 : l == 2 ? 256 : l == 3 ? 320 : l == 4 ? 336 : 340; }

// Texel t of level l from its children; false if none holds sums.
template <typename Shared, typename Below>
__device__ __forceinline__ bool build_texel(const RegionParams &P, Shared &sh, int l, int ls, int t, int L,
                                            const Below &below, uint2 &v) {
  const int j = t >> ls, i = t & ((1 << ls) - 1);
  Node c[4];
  bool any = false;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    c[q] = {0, 0, 0, kNoPosition, 0};
    if (below(2 * j + (q >> 1), 2 * i + (q & 1), c[q])) any = true;
  }
  if (!any) return false;
  const Node r = mip_node(c);
  const int k = level_base(l) + t;
  sh.x[k] = r.x;
  sh.y[k] = r.y;
  sh.z[k] = r.z;
  sh.p[k] = (unsigned short)r.p;
  v = make_record(r.x, r.y, r.z, r.p, L, P.dtype);
  return true;
}

__device__ __forceinline__ bool has_colour(uint2 v) { return (v.x | (v.y & 0xffffu)) != 0u; }

// Texels first .. first + n - 1 of level l (side 2^ls texels) of a group whose
// level 0 is level L0 of the map and begins at texel (ox, oy) of it: sums and
// records.  `below` gives a child (row, column) if it holds sums.  Called by
// threads t0, t0 + step, ... in whole warps.
template <typename Shared, typename Below>
__device__ void build_level(const RegionParams &P, Shared &sh, int l, int ls, int first, int n, int L0, int face,
                            int ox, int oy, int t0, int step, const Below &below) {
  const int L = L0 + l, NL = P.N >> L;
  uint2 *rec = P.rec + P.level_off[L] + ((long long)face * NL + (oy >> l)) * NL + (ox >> l);
  for (int k = t0; k < ((n + 31) & ~31); k += step) {
    const int t = first + k;
    uint2 v = kEmptyRecord;
    bool any = false;
    if (k < n) {
      any = build_texel(P, sh, l, ls, t, L, below, v);
      rec[(long long)(t >> ls) * NL + (t & ((1 << ls) - 1))] = v;
    }
    const unsigned full = __ballot_sync(0xffffffffu, any), lit = __ballot_sync(0xffffffffu, has_colour(v));
    if ((threadIdx.x & 31) == 0) {
      sh.full[l][t >> 5] = full;
      if (l <= 2) sh.lit[l][t >> 5] = lit;
    }
  }
}

// A child from the level below in shared memory.
template <typename Shared>
struct FromLevel {
  const Shared &sh;
  int l, ls;  // the child's level and log2 of its side
  __device__ bool operator()(int j, int i, Node &c) const {
    const int t = (j << ls) + i;
    if (!(sh.full[l][t >> 5] >> (t & 31) & 1u)) return false;
    const int k = level_base(l) + t;
    c = {sh.x[k], sh.y[k], sh.z[k], sh.p[k], 0};
    return true;
  }
};

// Levels 2 .. ls of a group (side 2^ls) whose level 1 is in shared memory.
// Level 2 takes the block, the rest (16, 4 and 1 texels) the first warp while
// the others go on; ends without a barrier, the top texel is in shared memory
// for the first warp.
template <typename Shared>
__device__ void build_upper(const RegionParams &P, Shared &sh, int ls, int L0, int face, int ox, int oy) {
  if (ls >= 2) {
    build_level(P, sh, 2, ls - 2, 0, 1 << (2 * (ls - 2)), L0, face, ox, oy, threadIdx.x, blockDim.x,
                FromLevel<Shared>{sh, 1, ls - 1});
    __syncthreads();
  }
  if (threadIdx.x < 32)
    for (int l = 3; l <= ls; ++l) {
      build_level(P, sh, l, ls - l, 0, 1 << (2 * (ls - l)), L0, face, ox, oy, threadIdx.x, 32,
                  FromLevel<Shared>{sh, l - 1, ls - l + 1});
      __syncwarp();
    }
}

template <typename Shared>
__device__ __forceinline__ Node top_node(const Shared &sh, int ls) {
  Node r = {0, 0, 0, kNoPosition, 0};
  FromLevel<Shared>{sh, ls, 0}(0, 0, r);
  return r;
}

// Occupancy blocks (mask_level_offset) of level l <= 2 of a region of 32 x 32
// level-0 texels.  A block's second eight columns belong to its right
// neighbour: within the region they are at hand, past it the neighbour
// writes them (and this region writes its left neighbour's), byte by byte.
template <typename Shared>
__device__ void write_mask(const RegionParams &P, const Shared &sh, int l, int face, int rx, int ry, int t0) {
  const int s = kRegion >> l, lc = 2 - l, nbc = 1 << lc, nbr = s / 4, NL = P.N >> l, nbx = NL / 8, nby = NL / 4;
  for (int b = t0; b < nbc * nbr; b += 32) {
    const int bx = b & (nbc - 1), by = b >> lc, gx = rx * nbc + bx, gy = ry * nbr + by;
    unsigned row[4];
    for (int r = 0; r < 4; ++r) {
      const int bit = (by * 4 + r) * s;
      const unsigned w = (sh.lit[l][bit >> 5] >> (bit & 31)) & (s == 32 ? 0xffffffffu : (1u << s) - 1u);
      row[r] = __brev(w >> (8 * bx)) >> 16;  // columns 8 bx .. 8 bx + 15, the first on top
    }
    unsigned char *m = P.mask + 8 * (P.mask_off[l] + ((long long)face * nby + gy) * nbx + gx);
    if (bx + 1 < nbc || gx + 1 == nbx) {
      *reinterpret_cast<uint2 *>(m) = make_uint2((row[0] << 16) | row[1], (row[2] << 16) | row[3]);
    } else {
      m[3] = (unsigned char)(row[0] >> 8);
      m[1] = (unsigned char)(row[1] >> 8);
      m[7] = (unsigned char)(row[2] >> 8);
      m[5] = (unsigned char)(row[3] >> 8);
    }
    if (bx == 0 && gx > 0) {
      m -= 8;
      m[2] = (unsigned char)(row[0] >> 8);
      m[0] = (unsigned char)(row[1] >> 8);
      m[6] = (unsigned char)(row[2] >> 8);
      m[4] = (unsigned char)(row[3] >> 8);
    }
  }
}

// Bound by instruction issue and by the chain of loads and levels (about 6 us a
// region), so: eight small blocks per SM, and the few texels that hold sums (41
// of 1024 for 1M stars on 2048^2 faces) are listed and computed side by side
// instead of one or two to a warp.
template <int kSlots>
__global__ void __launch_bounds__(kSlots, 1024 / kSlots) region_kernel(const RegionParams P) {
  constexpr bool kSorted = kSlots == kSortedSlots;  // stars by region, else the sums of all texels
  __shared__ __align__(16) RegionShared<kSlots> sh;
  const int N = P.N, ls = min(31 - __clz(N), 5), side = 1 << ls;
  int lp = max(31 - __clz(N) - 5, 0);  // log2 of the groups per face side
  const int region = blockIdx.x, face = region >> (2 * lp);
  int gx = region & ((1 << lp) - 1), gy = region >> lp & ((1 << lp) - 1);
  const int tid = threadIdx.x, lane = tid & 31;
  RegionSpan span = {0, 0};
  if (kSorted && P.span) span = P.span[region];
  const StarItem *items = P.items + span.first;
  const bool listed = kSorted && span.count < kCrowded;
  uint2 *const rec0 = P.rec + ((long long)face * N + gy * side) * N + gx * side;
  if (tid < kRegion) {
    sh.touched[tid] = 0;
    sh.lit[0][tid] = 0;
    sh.lit[1][tid] = 0;
  }
  if (tid < 8) sh.full[1][tid] = 0;
  if (tid == 0) sh.n0 = sh.n1 = 0;
  // ---- sums of the region's texels, and levels 0 and 1
  auto add = [&](const StarItem &st, int k) {
    for (int c = 0; c < 3; ++c) shared_add(sh, c, k, st.q[c]);
    shared_add(sh, 3, k, st.q[1] * (long long)(st.pos & 0xffffu));
    shared_add(sh, 4, k, st.q[1] * (long long)(st.pos >> 16));
  };
  auto level0_record = [&](int q) {  // of the sums in slot q
    const long long x = shared_sum(sh, 0, q), y = shared_sum(sh, 1, q), z = shared_sum(sh, 2, q);
    unsigned p = kNoPosition;
    if (y > 0)
      p = (unsigned)(mean_byte0(shared_sum(sh, 3, q), y) | (mean_byte0(shared_sum(sh, 4, q), y) << 8)) & 0xffffu;
    sh.p0[q] = (unsigned short)p;
    return make_record(x, y, z, p, 0, P.dtype);
  };
  if (listed && span.count <= kSlots) {
    // few stars: a slot for each texel that one touches
    StarItem st;
    const bool has = tid < (int)span.count;
    if (has) st = items[tid];
    __syncthreads();
    if (has) {
      const int j = st.local >> 5, i = st.local & 31;
      if (!(atomicOr(&sh.touched[j], 1u << i) >> i & 1u)) {  // the texel's first star
        const unsigned k = atomicAdd(&sh.n0, 1u);
        sh.slot[st.local] = (unsigned short)k;
        sh.list0[k] = (unsigned short)st.local;
        for (int c = 0; c < 10; ++c) sh.acc[c][k] = 0;
        if (ls > 0) {
          const unsigned t = ((j >> 1) << (ls - 1)) + (i >> 1);
          if (!(atomicOr(&sh.full[1][t >> 5], 1u << (t & 31)) >> (t & 31) & 1u))
            sh.list1[atomicAdd(&sh.n1, 1u)] = (unsigned short)t;
        }
      }
    }
    __syncthreads();
    if (has) add(st, sh.slot[st.local]);
    for (int k = tid; k < side * side; k += blockDim.x) {
      const int j = k >> ls, i = k & (side - 1);
      if (!(sh.touched[j] >> i & 1u)) rec0[(long long)j * N + i] = kEmptyRecord;
    }
    __syncthreads();
    if (tid < (int)sh.n0) {
      const int t = sh.list0[tid], j = t >> 5, i = t & 31;
      const uint2 v = level0_record(tid);
      rec0[(long long)j * N + i] = v;
      if (has_colour(v)) atomicOr(&sh.lit[0][j], 1u << i);
    }
    __syncthreads();
    if (ls > 0) {
      const int l1 = ls - 1, N1 = N >> 1;
      uint2 *rec1 = P.rec + P.level_off[1] + ((long long)face * N1 + (gy << l1)) * N1 + (gx << l1);
      for (int t = tid; t < 1 << (2 * l1); t += blockDim.x)
        if (!(sh.full[1][t >> 5] >> (t & 31) & 1u)) rec1[(long long)(t >> l1) * N1 + (t & ((1 << l1) - 1))] = kEmptyRecord;
      if (tid < (int)sh.n1) {
        const int t = sh.list1[tid];
        uint2 v = kEmptyRecord;
        build_texel(P, sh, 1, l1, t, 1, [&](int j, int i, Node &c) {
          if (!(sh.touched[j] >> i & 1u)) return false;
          const int q = sh.slot[j * kRegion + i];
          c = {shared_sum(sh, 0, q), shared_sum(sh, 1, q), shared_sum(sh, 2, q), sh.p0[q], 0};
          return true;
        }, v);
        rec1[(long long)(t >> l1) * N1 + (t & ((1 << l1) - 1))] = v;
        if (has_colour(v)) atomicOr(&sh.lit[1][t >> 5], 1u << (t & 31));
      }
      __syncthreads();
    }
  } else {
    // many stars, or dense sums: bands of rows, a slot for each texel
    const int rows = min(side, kSlots >> ls), n = rows << ls;
    for (int r0 = 0; r0 < side; r0 += rows) {
      for (int c = 0; c < 10; ++c) sh.acc[c][tid] = 0;
      __syncthreads();
      if (listed) {
        for (unsigned long long s = tid; s < span.count; s += blockDim.x) {
          const int j = (int)(items[s].local >> 5) - r0;
          if (j < 0 || j >= rows) continue;
          const StarItem st = items[s];
          atomicOr(&sh.touched[r0 + j], 1u << (st.local & 31));
          add(st, (j << ls) + (st.local & 31));
        }
      } else if (tid < n) {
        const int j = r0 + (tid >> ls), i = tid & (side - 1);
        const unsigned long long *a =
            kSorted ? reinterpret_cast<const unsigned long long *>(items) + (j * kRegion + i) * 5
                    : P.acc + (((long long)face * N + gy * side + j) * N + gx * side + i) * 5;
        unsigned long long any = 0;
        for (int c = 0; c < 5; ++c) {
          const unsigned long long v = a[c];
          any |= v;
          sh.acc[2 * c][tid] = (unsigned)v;
          sh.acc[2 * c + 1][tid] = (unsigned)(v >> 32);
        }
        if (any) atomicOr(&sh.touched[j], 1u << i);
      }
      __syncthreads();
      if (tid < n) {
        const int j = r0 + (tid >> ls), i = tid & (side - 1);
        uint2 v = kEmptyRecord;
        if (sh.touched[j] >> i & 1u) v = level0_record(tid);
        rec0[(long long)j * N + i] = v;
        if (has_colour(v)) atomicOr(&sh.lit[0][j], 1u << i);
      }
      __syncthreads();
      if (ls > 0)
        build_level(P, sh, 1, ls - 1, (r0 / 2) << (ls - 1), (rows / 2) << (ls - 1), 0, face, gx * side, gy * side, tid,
                    blockDim.x, [&](int j, int i, Node &c) {
                      if (!(sh.touched[j] >> i & 1u)) return false;
                      const int q = ((j - r0) << ls) + i;
                      c = {shared_sum(sh, 0, q), shared_sum(sh, 1, q), shared_sum(sh, 2, q), sh.p0[q], 0};
                      return true;
                    });
      __syncthreads();
    }
  }
  if (ls == 0) return;
  build_upper(P, sh, ls, 0, face, gx * side, gy * side);
  if (P.mask && (tid >> 5) >= 1 && (tid >> 5) <= 3) write_mask(P, sh, (tid >> 5) - 1, face, gx, gy, lane);
  // ---- the groups above: the last of up to 32 x 32 groups to finish builds
  // the next levels from the top texels of them all
  int L0 = ls, lg = ls;
  Node *nodes = P.nodes;
  unsigned *arrived = P.arrived;
  while (lp > 0) {
    const int lm = min(lp, 5), la = lp - lm, ax = gx >> lm, ay = gy >> lm;
    if (tid == 0) {
      nodes[(((face << lp) + gy) << lp) + gx] = top_node(sh, lg);
      __threadfence();
      sh.last = atomicAdd(arrived + (((face << la) + ay) << la) + ax, 1u) == (1u << (2 * lm)) - 1u;
      __threadfence();
    }
    __syncthreads();
    if (!sh.last) return;
    const Node *group = nodes + ((((face << lp) + (ay << lm)) << lp) + (ax << lm));
    build_level(P, sh, 1, lm - 1, 0, 1 << (2 * (lm - 1)), L0, face, ax << lm, ay << lm, tid, blockDim.x,
                [&](int j, int i, Node &c) {
                  const ulonglong2 *g = reinterpret_cast<const ulonglong2 *>(group + ((long long)j << lp) + i);
                  const ulonglong2 a = __ldcg(g), b = __ldcg(g + 1);
                  c = {(long long)a.x, (long long)a.y, (long long)b.x, (unsigned)b.y, 0};
                  return true;
                });
    __syncthreads();
    build_upper(P, sh, lm, L0, face, ax << lm, ay << lm);
    nodes += 6LL << (2 * lp);
    arrived += 6LL << (2 * la);
    L0 += lm;
    lg = lm;
    lp = la;
    gx = ax;
    gy = ay;
  }
}

// Nodes and arrival counters of the stages above the regions.
static void stage_sizes(int N, long long *nodes, long long *counters) {
  *nodes = *counters = 0;
  for (long long per = std::max(N / kRegion, 1); per > 1;) {
    const long long above = per / std::min<long long>(per, kRegion);
    *nodes += 6 * per * per;
    *counters += 6 * above * above;
    per = above;
  }
}

// Occupancy blocks of levels first .. levels - 1 (mask_level_offset) from the
// records, one warp per block; a ballot gives the bits of 8 columns x 4 rows
// (lane = 8 row + column, reversed into bit 31 - lane).  A texel is occupied
// when its colour is not zero: the renderer takes only those of a footprint.
__global__ void occupancy_kernel(const uint2 *rec, int N, int first, int levels, uint2 *mask) {
  long long blk = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  int L = 0, nbx = 0, nby = 0;
  long long in_level = blk, before = 0, texels = 0;  // blocks and records of the levels before L
  for (L = 0; L < levels; texels += 6LL * (N >> L) * (N >> L), ++L) {
    nbx = max((N >> L) >> 3, 1);
    nby = max((N >> L) >> 2, 1);
    const long long here = 6LL * nbx * nby;
    if (L < first) { before += here; continue; }
    if (in_level < here) break;
    in_level -= here;
    before += here;
  }
  if (L == levels) return;  // whole warps leave together
  const int lane = threadIdx.x & 31, NL = N >> L;
  const int bx = (int)(in_level % nbx), by = (int)(in_level / nbx % nby), face = (int)(in_level / ((long long)nbx * nby));
  const int j = by * 4 + (lane >> 3), i = bx * 8 + (lane & 7);
  const uint2 *level = rec + texels;
  auto occupied = [&](const int ii) {
    if (ii >= NL || j >= NL) return false;
    const uint2 v = level[((long long)face * NL + j) * NL + ii];
    return (v.x | (v.y & 0xffffu)) != 0u;
  };
  const unsigned a = __brev(__ballot_sync(0xffffffffu, occupied(i)));
  const unsigned b = __brev(__ballot_sync(0xffffffffu, occupied(i + 8)));
  // bytes of a and b are rows (row 0 on top): interleave them
  if (lane == 0) mask[before + in_level] = make_uint2(__byte_perm(a, b, 0x3726u), __byte_perm(a, b, 0x1504u));
}

// The occupancy mask of levels `first` and up from the records.
void occupancy_launch(bh_ctx *ctx, const bh_cubemap *c, int first, cudaStream_t s) {
  const long long blocks = mask_level_offset(c->n, c->levels) - mask_level_offset(c->n, first);
  if (blocks <= 0) return;
  occupancy_kernel<<<(unsigned)((blocks + 7) / 8), 256, 0, s>>>(c->rec, c->n, first, c->levels, c->mask);
  count_launch(ctx);
}

static unsigned star_blocks(long long n) { return (unsigned)((n + 255) / 256); }

}  // namespace bh

using namespace bh;

extern "C" long long bh_cubemap_records(int N) {
  if (N < 1 || (N & (N - 1))) return 0;
  return cube_level_offset(N, cube_levels(N));
}

extern "C" bh_status bh_build_star_cubemap(bh_ctx *ctx, const bh_star *stars, long long n, int N,
                                           bh_dtype storage, int on_device, void *stream,
                                           bh_cubemap **out) {
  TraceRange trace_("bh_build_star_cubemap");
  if (!ctx || !out || (n > 0 && !stars)) { set_error("bh_build_star_cubemap: NULL argument"); return BH_ERR_INVALID_ARG; }
  *out = nullptr;
  if (n < 0 || N < 1 || N > 8192 || (N & (N - 1))) {
    set_error("bh_build_star_cubemap: n = %lld, face_size = %d (power of two, 1..8192)", n, N);
    return BH_ERR_INVALID_ARG;
  }
  if (storage != BH_F16 && storage != BH_BF16) {
    set_error("bh_build_star_cubemap: storage must be BH_F16 or BH_BF16");
    return BH_ERR_INVALID_ARG;
  }
  BH_CUDA(cudaSetDevice(ctx->device));
  cudaStream_t s = (cudaStream_t)stream;
  bh_cubemap *c = nullptr;
  bh_status st = cubemap_alloc_public(ctx, N, storage, s, &c);
  if (st) return st;
  // Scratch, one allocation: counters (cleared), offsets, colour fit, stage
  // nodes, then the sorted stars -- or, where those would take more than the
  // dense sums of the level-0 texels and 1 GiB, or more than the device has, the
  // sums (cleared).
  const long long per = std::max(N / kRegion, 1), regions = 6 * per * per, texels = 6LL * N * N;
  long long n_nodes, n_counters;
  stage_sizes(N, &n_nodes, &n_counters);
  const size_t sorted = (sizeof(StarBin) + sizeof(StarItem)) * (size_t)n, dense = sizeof(unsigned long long) * 5 * texels;
  auto up16 = [](size_t b) { return (b + 15) / 16 * 16; };
  const size_t b_arrived = up16(sizeof(unsigned) * (kChromaCells + n_counters)), b_count = up16(sizeof(unsigned long long) * (regions + 1));
  const size_t b_span = sizeof(RegionSpan) * regions;
  const size_t b_fit = up16(sizeof(double) * (3 * kNLambda + kChromaCoefs + kChromaVals)), b_nodes = sizeof(Node) * n_nodes;
  const size_t b_copy = n > 0 && !on_device ? up16(sizeof(bh_star) * (size_t)n) : 0;
  bool sort = sorted <= std::max<size_t>(dense, (size_t)1 << 30);
  size_t b_stars, cleared;
  PoolBlock mem;
  cudaError_t e;
  for (;; sort = false) {
    b_stars = sort ? sorted : 0;
    cleared = b_arrived + b_count + (sort ? 0 : dense);
    e = pool_get(*ctx->pool, cleared + b_span + b_fit + b_nodes + b_stars + b_copy, s, &mem, true);
    if (e != cudaErrorMemoryAllocation || !sort || dense >= sorted) break;
    cudaGetLastError();
  }
  unsigned char *scratch = static_cast<unsigned char *>(mem.p);
  if (e != cudaSuccess) {
    bh_cubemap_free(c);
    return cuda_fail(e, "bh_build_star_cubemap");
  }
  RegionParams P;
  unsigned *fitted = reinterpret_cast<unsigned *>(scratch);
  P.arrived = fitted + kChromaCells;
  unsigned long long *count = reinterpret_cast<unsigned long long *>(scratch + b_arrived), *cursor = count + regions;
  unsigned long long *acc = reinterpret_cast<unsigned long long *>(scratch + b_arrived + b_count);
  RegionSpan *span = reinterpret_cast<RegionSpan *>(scratch + cleared);
  double *cmf = reinterpret_cast<double *>(scratch + cleared + b_span), *coef = cmf + 3 * kNLambda, *vals = coef + kChromaCoefs;
  P.nodes = reinterpret_cast<Node *>(scratch + cleared + b_span + b_fit);
  StarItem *items = reinterpret_cast<StarItem *>(scratch + cleared + b_span + b_fit + b_nodes);
  StarBin *bins = reinterpret_cast<StarBin *>(items + n);
  const bh_star *src = stars;
  if (b_copy) {
    bh_star *copy = reinterpret_cast<bh_star *>(scratch + cleared + b_span + b_fit + b_nodes + b_stars);
    e = cudaMemcpyAsync(copy, stars, sizeof(bh_star) * n, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);  // the host list may be freed on return
    src = copy;
  }
  if (e == cudaSuccess) e = cudaMemsetAsync(scratch, 0, cleared, s);
  if (e == cudaSuccess) {
    if (n > 0) {
      chroma_launch(cmf, vals, fitted, coef, s);
      if (sort) {
        star_bin_kernel<<<star_blocks(n), 256, 0, s>>>(src, n, N, count, bins);
        region_span_kernel<<<(unsigned)((regions + 31) / 32), 32, 0, s>>>(count, (int)regions, cursor, span, items);
        star_scatter_kernel<<<star_blocks(n), 256, 0, s>>>(src, n, bins, span, cmf, coef, items);
      } else {
        star_accumulate_kernel<<<star_blocks(n), 256, 0, s>>>(src, n, N, cmf, coef, acc);
      }
      count_launch(ctx, sort ? 4 : 2);
    }
    P.items = sort ? items : nullptr;
    P.span = n > 0 ? span : nullptr;
    P.acc = acc;
    P.rec = c->rec;
    P.mask = N >= kRegion ? reinterpret_cast<unsigned char *>(c->mask) : nullptr;
    P.N = N;
    P.dtype = storage;
    region_levels(P);
    if (sort) region_kernel<kSortedSlots><<<(unsigned)regions, kSortedSlots, 0, s>>>(P);
    else region_kernel<kDenseSlots><<<(unsigned)regions, kDenseSlots, 0, s>>>(P);
    count_launch(ctx);
    occupancy_launch(ctx, c, N >= kRegion ? 3 : 0, s);
    e = cudaGetLastError();
  }
  pool_put(*ctx->pool, mem, s);
  if (e != cudaSuccess) {
    bh_cubemap_free(c);
    return cuda_fail(e, "bh_build_star_cubemap");
  }
  *out = c;
  return BH_OK;
}

extern "C" bh_status bh_cubemap_copy_out(const bh_cubemap *c, uint16_t *h, long long n) {
  if (!c || !h) { set_error("bh_cubemap_copy_out: NULL argument"); return BH_ERR_INVALID_ARG; }
  if (n != c->records) {
    set_error("bh_cubemap_copy_out: %lld records requested, map has %lld", n, c->records);
    return BH_ERR_INVALID_ARG;
  }
  BH_CUDA(cudaSetDevice(c->ctx->device));
  BH_CUDA(cudaDeviceSynchronize());
  BH_CUDA(cudaMemcpy(h, c->rec, sizeof(uint2) * n, cudaMemcpyDeviceToHost));
  return BH_OK;
}

namespace bh {
// An empty map of face size N (all levels and the occupancy mask allocated,
// contents undefined), for loading from a checkpoint.
bh_status cubemap_alloc_public(bh_ctx *ctx, int N, bh_dtype storage, cudaStream_t s, bh_cubemap **out) {
  bh_cubemap *c = new bh_cubemap();
  c->ctx = ctx;
  c->pool = ctx->pool;
  c->n = N;
  c->levels = cube_levels(N);
  c->storage = storage;
  c->records = bh_cubemap_records(N);
  const size_t rec_bytes = (sizeof(uint2) * c->records + 255) / 256 * 256;
  const cudaError_t e = pool_get(*ctx->pool, rec_bytes + sizeof(uint2) * mask_level_offset(N, c->levels), s, &c->mem);
  if (e != cudaSuccess) {
    delete c;
    return cuda_fail(e, "cube map allocation");
  }
  c->rec = static_cast<uint2 *>(c->mem.p);
  c->mask = reinterpret_cast<uint2 *>(static_cast<char *>(c->mem.p) + rec_bytes);
  *out = c;
  return BH_OK;
}
}  // namespace bh

extern "C" void bh_cubemap_free(bh_cubemap *c) {
  if (!c) return;
  cudaSetDevice(c->pool->device);
  pool_put_synced(*c->pool, c->mem);
  delete c;
}

// ---------------------------------------------------------------------------
// Allocation-free cube-map build
//
// For callers that may not allocate device memory themselves: applications
// that hand every byte of device memory to their own pool or arena (engines,
// plug-in hosts with a fixed memory budget), and real-time threads that must
// not call cudaMalloc/cudaFree, which can synchronise the device and take an
// unbounded time.  The scratch lives in one file-scope device array, sized for
// faces of up to kNoAllocMaxFace texels; every GPU that loads this library
// holds it (about 4 MB) until the process exits.
// ---------------------------------------------------------------------------
namespace bh {

constexpr int kNoAllocMaxFace = 128;
constexpr long long kNoAllocTexels0 = 6LL * kNoAllocMaxFace * kNoAllocMaxFace;
// arrival counters of the stage above the regions, the sums of the level-0
// texels (5 x 64 bit each), the top texels of the regions, the matching functions
// and the colour fit
constexpr size_t kNoAllocRegions = 6 * (kNoAllocMaxFace / kRegion) * (kNoAllocMaxFace / kRegion);
constexpr size_t kNoAllocCounters = (kChromaCells + 6 + 1) / 2 / 2 * 2 + 2;  // 32-bit counters: the fit's cells, the faces
constexpr size_t kNoAllocScratchWords =
    kNoAllocCounters + 5 * kNoAllocTexels0 + 4 * kNoAllocRegions + 3 * kNLambda + kChromaCoefs + kChromaVals;
static_assert(kNoAllocMaxFace <= kRegion * kRegion && sizeof(Node) == 32, "one stage above the regions");

static __device__ __align__(256) unsigned long long g_noalloc_scratch[kNoAllocScratchWords];

// Device address of the scratch array on the current device (the host-side
// name of a __device__ array is not a device address).  Looked up on every
// call that is not being captured into a CUDA graph, so that a device or
// primary-context reset between calls cannot leave a stale address behind;
// a call under stream capture uses the address its device's last uncaptured
// call found (cudaGetSymbolAddress may load the module, which capture forbids).
static bh_status noalloc_scratch(int device, bool capturing, unsigned long long **out) {
  static std::mutex mu;
  static unsigned long long *addr[64] = {nullptr};
  if (device < 0 || device >= 64) {
    set_error("bh_build_star_cubemap_noalloc: device %d out of range", device);
    return BH_ERR_INVALID_ARG;
  }
  std::lock_guard<std::mutex> lk(mu);
  if (!capturing) {
    void *p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return cuda_fail(e, "bh_build_star_cubemap_noalloc: cudaGetSymbolAddress");
    addr[device] = static_cast<unsigned long long *>(p);
  } else if (!addr[device]) {
    set_error("bh_build_star_cubemap_noalloc: the first call on device %d is under stream capture; "
              "make one call before capturing", device);
    return BH_ERR_INVALID_ARG;
  }
  *out = addr[device];
  return BH_OK;
}

}  // namespace bh

extern "C" bh_status bh_build_star_cubemap_noalloc(const bh_star *stars_device, long long n,
                                                   int N, bh_dtype storage, uint16_t *records_device,
                                                   void *stream) {
  if ((n > 0 && !stars_device) || !records_device) {
    set_error("bh_build_star_cubemap_noalloc: NULL argument");
    return BH_ERR_INVALID_ARG;
  }
  if (N < 1 || (N & (N - 1)) || N > kNoAllocMaxFace) {
    set_error("bh_build_star_cubemap_noalloc: face_size %d must be a power of two <= %d (the size of "
              "its static scratch)", N, kNoAllocMaxFace);
    return BH_ERR_INVALID_ARG;
  }
  if (n < 0 || (storage != BH_F16 && storage != BH_BF16) || ((uintptr_t)records_device & 7)) {
    set_error("bh_build_star_cubemap_noalloc: n >= 0, storage BH_F16/BH_BF16 and 8-byte aligned records required");
    return BH_ERR_INVALID_ARG;
  }
  int dev = 0;
  BH_CUDA(cudaGetDevice(&dev));
  cudaStream_t s = (cudaStream_t)stream;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  BH_CUDA(cudaStreamIsCapturing(s, &cap));
  unsigned long long *scratch = nullptr;
  bh_status st = noalloc_scratch(dev, cap != cudaStreamCaptureStatusNone, &scratch);
  if (st) return st;
  const long long nt0 = 6LL * N * N, per = std::max(N / kRegion, 1);
  RegionParams P;
  unsigned *fitted = reinterpret_cast<unsigned *>(scratch);
  P.arrived = fitted + kChromaCells;
  unsigned long long *acc = scratch + kNoAllocCounters;
  P.nodes = reinterpret_cast<Node *>(acc + 5 * kNoAllocTexels0);
  double *cmf = reinterpret_cast<double *>(P.nodes + kNoAllocRegions), *coef = cmf + 3 * kNLambda;
  double *vals = coef + kChromaCoefs;
  // the array keeps the previous call's contents: counters and sums must start at zero
  BH_CUDA(cudaMemsetAsync(scratch, 0, sizeof(unsigned long long) * (kNoAllocCounters + 5 * nt0), s));
  if (n > 0) {
    chroma_launch(cmf, vals, fitted, coef, s);
    star_accumulate_kernel<<<star_blocks(n), 256, 0, s>>>(stars_device, n, N, cmf, coef, acc);
  }
  P.items = nullptr;
  P.span = nullptr;
  P.acc = acc;
  P.rec = reinterpret_cast<uint2 *>(records_device);
  P.mask = nullptr;
  P.N = N;
  P.dtype = storage;
  region_levels(P);
  region_kernel<kDenseSlots><<<(unsigned)(6 * per * per), kDenseSlots, 0, s>>>(P);
  BH_CUDA(cudaGetLastError());
  return BH_OK;
}
