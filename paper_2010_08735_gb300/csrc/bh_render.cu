// Per-pixel render (Sec. 3.2-3.4, Algorithm 1 TRACERAY) for sm_103a.
//
// Mapping: one thread per pixel; a warp covers an 8x4 pixel tile made of
// eight 2x2 quads (lane bit 0 = column parity, bit 1 = row parity), so the
// screen-space derivatives of Sec. 3.3.2 are two warp shuffles (xor 1 and
// xor 2) with GLSL "fine" semantics.  Blocks are persistent and walk a tile
// queue that spans every camera of a batch.  The U table (8 KiB) is copied into
// shared memory once per block by the bulk-copy (TMA) engine behind an
// mbarrier; the 512x512 D table (1 MiB), the disc black-body table (16 KiB) and
// the C(xy,D) table stay in L2 and are read through the read-only path; the
// star cube map is gathered from L2/HBM with 8-byte
// records.  Pixels leave as one float4 store each (a warp writes four full
// 128-byte lines).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "bh_internal.cuh"

namespace bh {

constexpr int kMaxLevels = 14;
constexpr int kMaxOrbits = 1024;  // of one bh_render_orbits call

// Per-camera constants, computed on the host in FP64 (Eq. staticbasis,
// Eq. camerabasis, the boost B(v) of Appendix C, Eq. d) and rounded to float.
struct alignas(16) CamConst {
  float M[9];       // R O^T: camera (e_w, e_h, e_d) components -> pseudo-Cartesian components, where
                    // R (static orthonormal -> pseudo-Cartesian) has columns sqrt(1-u) r^, theta^, phi^
  float w[3];       // unit velocity direction on the camera axes (0 if v = 0)
  float rv[3];      // R v^: the unit velocity direction in pseudo-Cartesian components (0 if v = 0)
  float beta, inv_gamma2;
  float x[3];       // e_x' = position direction r^
  float zdeg[3];    // e_z' for radial beams (reading C8)
  float gamma, f, u, inv_sqrt_1mu;
  float half_w, half_h;
  int width, height;
  int tiles_x, tile0;
  float inv_tiles_x;
  float4 *out;      // RGBA float4 per pixel, or packed RGB floats when rgb != 0
  float *dbg;
  int rgb;          // 1: packed linear RGB, 3 floats per pixel (host-bound frames)
  int rgb_vec;      // 1: packed rows start 16-byte aligned (width % 4 == 0, aligned base)
};

struct RenderParams {
  CamConst cam0;            // single-camera launches
  const CamConst *cams;     // batched launches (nullptr: cam0)
  int ncams, total_tiles;   // tiles are 8 x 4 pixel warp tiles, row-major per camera
  const int *total_tiles_dev;  // if set, the tile count computed on the device
  unsigned *sched;          // {next fetch, retired warps}: zero before and after every launch
  unsigned fetch, tail;     // warp tiles taken per fetch, and handed out singly at the end
  unsigned by_place;        // fetches up to which a launch has no counter
  const void *D;
  int d_n;
  const void *U;
  int u_ne, u_nphi, u_bytes;
  float d_n1f, u_ne1f, u_nphi1f;  // d_n - 1, u_ne - 1, u_nphi - 1 as floats (operands, not conversions)
  const float *DTt, *UTt;   // regularised-time channels of D and U (debug and animated disc)
  const double *parts;      // animated disc: 8 doubles per particle (u1, u2, phi0, omega, c, rmin, rmax, 0)
  int n_parts;              // 0: constant disc density
  double time;              // coordinate time of the frame at the camera
  const float4 *C;
  const float4 *disc;
  const uint2 *cube;
  const uint2 *cube_mask;   // occupancy bits by blocks of texels
  int cube_n, cube_levels, cube_bf16;
  long long level_off[kMaxLevels];
  long long mask_off[kMaxLevels];
  float u_ic, u_oc, t_peak, rho;
  float fmax_disc;          // max of u^3 (1 - sqrt(3u)), at u = 12/49
  float lg_t0;              // log2(t_peak) - log2(fmax_disc) / 4: log2 T(u) = lg_t0 + log2(u^3 (1 - sqrt(3u))) / 4
  int disc_on;
  float exp_disc, exp_stars;
  float M[9];               // XYZ -> linear sRGB
  unsigned *status;
  unsigned long long wait_ns;  // bound of the table-load wait
  int inject_wait;          // fault injection: also wait on a barrier nothing arrives at
  unsigned long long inject_wait_ns;
};

__device__ __forceinline__ float ld_tab(const float *p, int i) { return __ldg(p + i); }
__device__ __forceinline__ float ld_tab(const __half *p, int i) { return __half2float(__ldg(p + i)); }
__device__ __forceinline__ float sm_tab(const float *p, int i) { return p[i]; }
__device__ __forceinline__ float sm_tab(const __half *p, int i) { return __half2float(p[i]); }

constexpr float kMuF = 4.0f / 27.0f;

// a / b and 1 / b for b below 2^126 (or a quotient that vanishes): SHORT leaves
// out the range check of the general division, with the same bits (88 frames
// compared).  Frames without the animated disc: 77.5 -> 76.3 M warp instructions
// at 1080p, 84.4 -> 83.2 us, 4K 350 -> 343 us.  The animated variant, at its
// register limit, got slower (67.8 -> 71.8 us) and keeps the general form.
template <bool SHORT>
__device__ __forceinline__ float quot(float a, float b) {
  return SHORT ? __fdividef(a, b) : a / b;
}
template <bool SHORT>
__device__ __forceinline__ float recip(float b) {
  float r;
  if (SHORT) asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(b));
  else r = 1.f / b;
  return r;
}

constexpr int kDbgFloats = 20;  // debug values per pixel (five float4)
constexpr float kPiF = 3.14159265358979f;

// Texel pair (row j, row min(j+1, n-1)) of the row-paired D table.
__device__ __forceinline__ float2 ld_pair(const float *p, int i) {
  return __ldg(reinterpret_cast<const float2 *>(p) + i);
}
__device__ __forceinline__ float2 ld_pair(const __half *p, int i) {
  return __half22float2(__ldg(reinterpret_cast<const __half2 *>(p) + i));
}

// Bilinear lookup in the row-paired D table (texel (j, i) holds D at rows j
// and min(j+1, n-1)): two loads, the x lerps of both rows as one packed f32x2
// step.  Appendix A coordinates; x clamped to its branch (C2).
template <typename DT>
__device__ __forceinline__ float d_bilinear_pair(const DT *D, int n, float fx, float fy, int xlo, int xhi,
                                                 unsigned *chk = nullptr) {
  fx = fminf(fmaxf(fx, (float)xlo), (float)xhi);
  fy = fminf(fmaxf(fy, 0.f), (float)(n - 1));
  const int i0 = (int)fx, j0 = (int)fy;
  const int i1 = min(i0 + 1, xhi);
  if (chk && !(i0 >= 0 && j0 >= 0 && i1 < n && j0 < n && i0 <= i1)) {
    atomicOr(chk, kStatusBadIndex);  // checked (debug) render: record and skip the access
    return 0.f;
  }
  const float tx = fx - i0, ty = fy - j0;
  const float2 p = ld_pair(D, j0 * n + i0), q = ld_pair(D, j0 * n + i1);  // (a, c), (b, d)
  const float2 lh = __ffma2_rn(make_float2(tx, tx), __ffma2_rn(p, make_float2(-1.f, -1.f), q), p);
  return fmaf(ty, lh.y - lh.x, lh.x);
}

// Bilinear D lookup at Appendix A coordinates; x clamped to its branch (C2).
template <typename DT>
__device__ __forceinline__ float d_bilinear(const DT *D, int n, float fx, float fy, int xlo, int xhi,
                                            unsigned *chk = nullptr) {
  fx = fminf(fmaxf(fx, (float)xlo), (float)xhi);
  fy = fminf(fmaxf(fy, 0.f), (float)(n - 1));
  int i0 = (int)fx, j0 = (int)fy;
  int i1 = min(i0 + 1, xhi), j1 = min(j0 + 1, n - 1);
  if (chk && !(i0 >= 0 && j0 >= 0 && i1 < n && j1 < n && i0 <= i1 && j0 <= j1)) {
    atomicOr(chk, kStatusBadIndex);  // checked (debug) render: record and skip the access
    return 0.f;
  }
  float tx = fx - i0, ty = fy - j0;
  float a = ld_tab(D, j0 * n + i0), b = ld_tab(D, j0 * n + i1);
  float c = ld_tab(D, j1 * n + i0), d = ld_tab(D, j1 * n + i1);
  float lo = fmaf(tx, b - a, a), hi = fmaf(tx, d - c, c);
  return fmaf(ty, hi - lo, lo);
}

// x coordinate of D for e^2 (em = e^2 - mu, formed without cancellation).
template <bool SHORT>
__device__ __forceinline__ float d_x(float e2, float em) {
  if (em < 0.f) {
    float r = quot<SHORT>(e2, kMuF);  // 1 - eta
    float lg = r < 0.5f ? log1pf(-r) : logf(quot<SHORT>(-em, kMuF));
    return 0.5f - sqrtf(fmaxf(-lg, 0.f) * 0.02f);
  }
  float r = quot<SHORT>(kMuF, e2);  // 1 - (e^2 - mu)/e^2
  float lg = r < 0.5f ? log1pf(-r) : logf(quot<SHORT>(em, e2));
  return 0.5f + sqrtf(fmaxf(-lg, 0.f) * 0.02f);
}

// Disc density of Appendix B at a hit seen `delay` before the frame's time,
// at radius hr and azimuth hphi: the sum over linear particles of
// (1 - d^2)^2, d^2 = (a/pi - 1)^2 + (hr - 1/u_a)^2, a = (hphi - phi(t)) mod
// 2 pi, times rho, clamped to 1.  Per particle (two float4, sorted by rmin):
// (rmin, rmax, u1, u2 - u1), (omega, c, phi(time) mod 2 pi, c phi(time) mod pi);
// only particles with rmin <= hr <= rmax (|hr - 1/u| < 1 possible) count.
__device__ __forceinline__ float particle_density(const float4 *sp, int n, float rho, float delay, float hr,
                                                  float hphi) {
  const float two_pi = 2.f * kPiF, inv_pi = 1.f / kPiF;
  float sum = 0.f;
  for (int k = 0; k < n; ++k) {
    const float4 A = sp[2 * k];
    if (A.x > hr) break;
    if (hr > A.y) continue;
    const float4 B = sp[2 * k + 1];
    float a = fmaf(B.x, delay, hphi - B.z);  // phi(time - delay) = phi(time) - omega delay
    a = fmaf(-two_pi, floorf(a * (1.f / two_pi)), a);
    float arg = fmaf(-B.y * B.x, delay, fmaf(B.y, a, B.w));
    arg = fmaf(-kPiF, rintf(arg * (1.f / kPiF)), arg);  // sin^2 has period pi: reduce to [-pi/2, pi/2]
    const float sn = __sinf(arg);                       // where the hardware sine is good to ~5e-7
    const float ua = fmaf(A.w, sn * sn, A.z);
    const float x = fmaf(a, inv_pi, -1.f), y = hr - 1.f / ua;
    const float d2 = fmaf(x, x, y * y);
    if (d2 < 1.f) {
      const float f = 1.f - d2;
      sum = fmaf(f, f, sum);
    }
  }
  return fminf(rho * sum, 1.f);
}

#ifndef BH_RENDER_MIN_BLOCKS
#define BH_RENDER_MIN_BLOCKS 4  // resident 256-thread blocks per SM the register budget must allow
#endif

// A footprint window is culled to its parallelogram when it holds more
// occupied texels than this: the cull costs about five takes.  Measured at 2 /
// 4 / 6 / 8 / 12: 88.6 / 88.9 / 89.4 / 89.8 / 90.3 us for a 1080p frame
// (density of 1M stars on 2048^2 faces), 388 / 383 / 379 / 376 / 374 us for
// a 4K one (4M on 4096^2); without it 106 us at 1080p.
constexpr int kCullAbove = 6;

// The camera of a tile past `cam`, by a whole warp: its lanes look at 32 parts of
// the cameras that are left.  Stepping through the cameras one by one took 6.1 ms
// for 20,000 thumbnails and 448 us for 1,000 cameras of 64 x 64; this 1.2 ms (the
// host's part) and 347 us, 300 of them 154 -> 127 us.
__device__ __forceinline__ int camera_of_tile(const CamConst *cams, int ncams, int cam, int tile) {
  const int lane = threadIdx.x & 31;
  for (int left = ncams - 1 - cam; left > 0;) {
    const int part = (left + 31) >> 5, at = min((lane + 1) * part, left);
    const int n = __popc(__ballot_sync(0xffffffffu, __ldg(&cams[cam + at].tile0) <= tile));
    const int go = min(n * part, left);
    cam += go;
    left = n == 32 ? 0 : min(part - 1, left - go);
  }
  return cam;
}

// A warp's next tile is mostly in the same camera, so the search is a function of
// its own (4K 351 -> 346 us); in the animated variant, which lacks registers for
// the call, it is not (64 frames of 640 x 360 with 64 particles 853 -> 831 us).
__device__ __noinline__ int search_camera(const CamConst *cams, int ncams, int cam, int tile) {
  return camera_of_tile(cams, ncams, cam, tile);
}

// Kernel variants: plain, animated disc (Appendix B), debug (any disc, plus
// per-pixel intermediate values).
enum RenderMode { kPlain = 0, kAnimated = 1, kDebug = 2 };

template <typename DT, int MODE>
__global__ void __launch_bounds__(256, BH_RENDER_MIN_BLOCKS) render_kernel(const RenderParams P) {
  constexpr bool DEBUG = MODE == kDebug;
  constexpr bool SHORT = MODE != kAnimated;  // quotients
  // The debug render is also the checked build: every table, cube-map and
  // occupancy index is tested before its access; a bad one sets a status bit
  // (bh_check_status) and the access is skipped -- no trap, no fault.
  unsigned *const chk = DEBUG ? P.status : nullptr;
  auto check = [&](bool ok) {
    if (DEBUG && !ok) atomicOr(P.status, kStatusBadIndex);
    return !DEBUG || ok;
  };
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ __align__(8) unsigned long long mbar;
  __shared__ __align__(8) unsigned long long mbar_never;  // fault injection: nothing arrives
  const float4 *s_disc = P.disc;  // black-body table: read through L1 (16 KiB), not staged
  const DT *s_U = reinterpret_cast<const DT *>(smem);
  // packed-RGB staging of the single-camera host-bound form: 96 floats per warp
  float *s_rgb = reinterpret_cast<float *>(smem + P.u_bytes + 2 * sizeof(float4) * P.n_parts);

  // ---- stage U into shared memory with the bulk-copy engine
  unsigned mb = (unsigned)__cvta_generic_to_shared(&mbar);
  unsigned mb_never = (unsigned)__cvta_generic_to_shared(&mbar_never);
  if (threadIdx.x == 0) {
    unsigned bytes = (unsigned)(P.u_bytes);
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mb));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mb_never));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb), "r"(bytes) : "memory");
    unsigned dst1 = (unsigned)__cvta_generic_to_shared(s_U);
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst1),
        "l"(P.U), "r"((unsigned)P.u_bytes), "r"(mb)
        : "memory");
  }
  // ln Y at the peak temperature, by which the disc's light is divided: its table
  // entries are asked for here, behind the copy above
  float peak_t, peak_a, peak_b;
  {
    float f = (log2f(P.t_peak) - 8.f) / 12.f * kDiscN - 0.5f;
    f = fminf(fmaxf(f, 0.f), (float)(kDiscN - 1));
    int k0 = (int)f, k1 = min(k0 + 1, kDiscN - 1);
    peak_t = f - k0;
    peak_a = s_disc[k0].x;
    peak_b = s_disc[k1].x;
  }
  // animated disc (Appendix B): this frame's particle constants, phases
  // reduced in FP64 so that FP32 keeps them exact to ~1e-7 rad at any time
  float4 *s_part = reinterpret_cast<float4 *>(smem + P.u_bytes);
  for (int k = threadIdx.x; k < P.n_parts; k += blockDim.x) {
    const double *q = P.parts + 8 * k;
    const double Phi = fma(q[3], P.time, q[2]);           // phi(t) = omega t + phi0
    const double Phir = Phi - 2.0 * kPi * floor(Phi / (2.0 * kPi));
    const double cPhi = q[4] * Phi;                       // sin^2 has period pi
    const double S = cPhi - kPi * floor(cPhi / kPi);
    s_part[2 * k] = make_float4((float)q[5], (float)q[6], (float)q[0], (float)(q[1] - q[0]));
    s_part[2 * k + 1] = make_float4((float)q[3], (float)q[4], (float)Phir, (float)S);
  }
  __syncthreads();
  bool table_ok;
  {
    // bounded waits: give up after a limit of global time
    auto bounded_wait = [](unsigned bar, unsigned long long limit_ns) -> bool {
      unsigned done = 0;
      unsigned long long t0, t;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
      for (;;) {
        asm volatile(
            "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0; selp.u32 %0, 1, 0, p; }"
            : "=r"(done)
            : "r"(bar)
            : "memory");
        if (done) return true;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t - t0 > limit_ns) return false;
      }
    };
    bool ok = bounded_wait(mb, P.wait_ns);
    if (!ok) bounded_wait(mb, P.wait_ns);  // let copies still in flight land before leaving
    // fault injection (bh_inject_fault): a barrier nothing arrives at
    if (ok && P.inject_wait) ok = bounded_wait(mb_never, P.inject_wait_ns);
    if (!ok && threadIdx.x == 0) atomicOr(P.status, kStatusMbarTimeout);
    table_ok = ok;
  }

  const int lane = threadIdx.x & 31;
  const int lx = ((lane >> 2) & 3) * 2 + (lane & 1);
  const int ly = ((lane >> 4) & 1) * 2 + ((lane >> 1) & 1);
  const int dn = P.d_n;
  const DT *D = reinterpret_cast<const DT *>(P.D);
  const int n_half = dn / 2;

  // below the table (256 K) the light is not normalised
  const float ln_peak = P.t_peak >= 256.f ? fmaf(peak_t, peak_b - peak_a, peak_a) : 0.f;

  // Dynamic schedule: a warp's first tiles follow from its place in the grid; then
  // it takes the next ones from a global counter until none are left: P.fetch at
  // a time while plenty are left, one at a time for the last P.tail, so that no
  // warp sits on a second tile while others have run out.  A launch with no more
  // to hand out than P.by_place never touches the counter, whose round trips were
  // a fifth of such a frame's time (256 x 256: 13.8 -> 10.5 us).
  // Asking for the next fetch before the current one is rendered measured slower
  // (1080p 86.0 -> 88.9 us: the early claim lengthens the tail by a tile).
  const unsigned total_tiles = P.total_tiles_dev ? *P.total_tiles_dev : P.total_tiles;
  const unsigned n_warps = gridDim.x * (blockDim.x >> 5), fetch = P.fetch;
  const unsigned chunked = total_tiles > P.tail ? (total_tiles - P.tail) / fetch * fetch : 0u;
  const bool counted = chunked / fetch + (total_tiles - chunked) > P.by_place;
  int cam = 0;  // the camera of the warp's last tile: its tiles only ever increase
  for (unsigned g = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); table_ok;) {
    // whole chunks first, then single tiles (g stays below total_tiles + 2 n_warps)
    const unsigned first = g * fetch, single = chunked + (g - chunked / fetch);
    const bool chunk = g < chunked / fetch;
    unsigned tile = chunk ? first : single;
    const unsigned tile_end = tile + (chunk ? fetch : 1u);
    if (tile >= total_tiles) break;
    do {
    // ---- which camera and which tile of it.  A single-camera launch reads
    // its constants straight from the kernel parameters (constant bank); a
    // batch reads them from global memory.  The pixel work is written once.
    auto shade = [&](const CamConst &C, const int t) {
    // tile row by a float reciprocal, corrected by one step (exact: the
    // quotient is at most 4096, so the rounded product is off by < 1)
    int ty = __float2int_rz(__int2float_rn(t) * C.inv_tiles_x), tx = t - ty * C.tiles_x;
    if (tx < 0) { --ty; tx += C.tiles_x; } else if (tx >= C.tiles_x) { ++ty; tx -= C.tiles_x; }
    int px = tx * 8 + lx, py = ty * 4 + ly;

    // ---- beam initialisation (Eq. d, Eq. raybasis, Eq. alpha)
    float qw = (px + 0.5f) - C.half_w, qh = C.half_h - (py + 0.5f), qd = -C.f;
    float qq = fmaf(qw, qw, fmaf(qh, qh, qd * qd));
    float inv = rsqrtf(qq), nq = qq * inv;
    float q0 = qw * inv, q1 = qh * inv, q2 = qd * inv;
    // Aberration (Eq. d): the backward direction -e_tau + n, on the static
    // frame, keeps n's part across v and has gamma (n.v^ - beta) along v^.
    // n.v^ - beta = (|q|^2/gamma^2 - |q x w|^2) / (|q| (q.w + beta |q|)) for
    // forward beams, free of the cancellation of n.v^ - beta near 1 - beta.
    float wq = fmaf(C.w[0], qw, fmaf(C.w[1], qh, C.w[2] * qd));
    float dpar, pxw = 0.f;  // |q x w|^2 (forward beams)
    if (wq > 0.f) {
      float x0_ = fmaf(qh, C.w[2], -qd * C.w[1]), x1_ = fmaf(qd, C.w[0], -qw * C.w[2]),
            x2_ = fmaf(qw, C.w[1], -qh * C.w[0]);
      float c2 = fmaf(x0_, x0_, fmaf(x1_, x1_, x2_ * x2_));
      pxw = c2;
      dpar = C.gamma * quot<SHORT>(fmaf(qq, C.inv_gamma2, -c2), nq * fmaf(C.beta, nq, wq));
    } else {
      dpar = C.gamma * fmaf(wq, inv, -C.beta);
    }
    // the backward direction on the static frame is ds = O^T p + dpar v^ with p
    // (n's part across v) orthogonal to v^, so |ds|^2 = |p|^2 + dpar^2, |p|^2 =
    // |q x w|^2 / |q|^2 (the forward branch has |q x w|^2 already)
    float p0 = fmaf(-wq, C.w[0], qw) * inv, p1 = fmaf(-wq, C.w[1], qh) * inv, p2 = fmaf(-wq, C.w[2], qd) * inv;
    const float wqi = wq * inv;
    const float pp = wq > 0.f ? pxw * (inv * inv) : fmaf(-wqi, wqi, 1.f);
    float dcam = C.gamma * fmaf(C.beta, dpar * rsqrtf(fmaf(dpar, dpar, pp)), 1.f);
    // pseudo-Cartesian beam direction d = R ds = (R O^T) p + dpar (R v^)
    float d0 = fmaf(C.M[0], p0, fmaf(C.M[1], p1, fmaf(C.M[2], p2, dpar * C.rv[0])));
    float d1 = fmaf(C.M[3], p0, fmaf(C.M[4], p1, fmaf(C.M[5], p2, dpar * C.rv[1])));
    float d2 = fmaf(C.M[6], p0, fmaf(C.M[7], p1, fmaf(C.M[8], p2, dpar * C.rv[2])));
    const float x0 = C.x[0], x1 = C.x[1], x2 = C.x[2];
    float c0 = fmaf(x1, d2, -x2 * d1), c1 = fmaf(x2, d0, -x0 * d2), c2 = fmaf(x0, d1, -x1 * d0);
    const float cn2 = fmaf(c0, c0, fmaf(c1, c1, c2 * c2));
    const float icn = rsqrtf(fmaxf(cn2, 1.2e-38f));  // 1/|e_x' ^ d| (guarded for radial beams)
    float cosd = fmaf(x0, d0, fmaf(x1, d1, x2 * d2));
    const float dd2 = fmaf(d0, d0, fmaf(d1, d1, d2 * d2));
    // delta itself is needed only for the debug channels: the disc hits use
    // delta - alpha, one angle (below)
    const float delta = DEBUG ? atan2f(cn2 * icn, cosd) : 0.f;
    float z0, z1, z2;
    if (cn2 < 1e-14f * dd2) {
      z0 = C.zdeg[0]; z1 = C.zdeg[1]; z2 = C.zdeg[2];
    } else {
      z0 = c0 * icn; z1 = c1 * icn; z2 = c2 * icn;
    }
    // e_y' = e_z' ^ e_x' (its z component is not needed below)
    float y0 = fmaf(z1, x2, -z2 * x1), y1 = fmaf(z2, x0, -z0 * x2);
    bool alpha_ok = false;
    float dma = 0.f;             // delta - alpha: the angle from t to the beam in the ray plane
    float tsx = 0.f, tsy = 0.f;  // t in the disc plane (x, y): hits lie at +-t
    {
      // t = +-(e_z ^ e_z')/|.| with t . e_y' >= 0 (Eq. alpha: alpha is the angle
      // from e_x' to t, delta the angle from e_x' to the beam d, both towards
      // e_y'); delta - alpha = atan2((t ^ d) . e_z', t . d), t's length and d's
      // length cancelling
      const float t0 = -z1, t1 = z0;
      const float tn2 = fmaf(t0, t0, t1 * t1);
      if (tn2 > 1e-24f) {
        const float sg = fmaf(t0, y0, t1 * y1) < 0.f ? -1.f : 1.f;
        const float X = fmaf(t1 * d2, z0, fmaf(-t0 * d2, z1, fmaf(t0, d1, -t1 * d0) * z2));
        const float Y = fmaf(t0, d0, t1 * d1);
        dma = atan2f(sg * X, sg * Y);
        if (MODE == kAnimated || DEBUG) {
          const float itn = rsqrtf(tn2);
          tsx = sg * t0 * itn;
          tsy = sg * t1 * itn;
        }
        alpha_ok = true;
      }
    }

    // ---- TRACERAY (Algorithm 1)
    const float u = C.u;
    float udot = -u * cosd * icn;
    float um = u - 2.f / 3.f;
    float em = fmaf(udot, udot, -um * um * (u + 1.f / 3.f));  // e^2 - mu
    float e2 = kMuF + em;
    bool captured = false;
    int nh = 0;
    float hu0 = 0.f, hu1 = 0.f;
    float th0 = 0.f, th1 = 0.f;  // retarded-time delays of the hits (debug render, animated disc)
    bool odd0 = false, odd1 = false;  // hit at -t rather than +t (an odd number of half turns)
    const bool anim = MODE == kAnimated || (DEBUG && P.n_parts > 0);
    float delta_p = 0.f, turn = 0.f;  // delta' = delta + turn
    if (em < 0.f && u > 2.f / 3.f) {
      captured = true;
    } else {
      int s = udot > 0.f ? 1 : -1;
      float xd = d_x<SHORT>(e2, em);
      float fx = xd * P.d_n1f;
      int xlo = em < 0.f ? 0 : n_half, xhi = em < 0.f ? n_half - 1 : dn - 1;
      float ua = 0.f, Dl, Da = 0.f, phia = INFINITY, yv;
      if (em < 0.f) {
        float eta = quot<SHORT>(-em, kMuF);
        float sa = asinf(sqrtf(fminf(eta, 1.f)));
        float th = fmaf(-2.f, sa, 0.5f * kPiF) * (1.f / 3.f);
        ua = fmaf(2.f / 3.f, sinf(th), 1.f / 3.f);
        // 1 - u/u_a = (du/dphi)^2 / (u_a g), g = (f(u_a) - f(u))/(u_a - u), f(x) = x^2 - x^3:
        // no cancellation when the camera is near the apsis (du/dphi -> 0)
        float g = fmaf(-u, u, fmaf(-ua, u, fmaf(-ua, ua, ua + u)));
        float om = g > 0.f ? quot<SHORT>(udot * udot, ua * g) : 1.f - quot<SHORT>(u, ua);
        yv = 1.f - sqrtf(fmaxf(om, 0.f));
        Dl = d_bilinear_pair(D, dn, fx, yv * P.d_n1f, xlo, xhi, chk);
        Da = d_bilinear_pair(D, dn, fx, P.d_n1f, xlo, xhi, chk);
        phia = Da + 0.5f * kPiF;
      } else {
        const float r23 = 0.81649658f, r13 = 0.57735027f;
        float sq = sqrtf(fabsf(um));
        yv = quot<SHORT>(r23 + (um >= 0.f ? sq : -sq), r23 + r13);
        Dl = d_bilinear_pair(D, dn, fx, yv * P.d_n1f, xlo, xhi, chk);
      }
      if (alpha_ok && P.disc_on) {
        // Appendix A coordinates of U: x = 1/(1 + 6e^2), y = phi (1 + 6e^3)/(3 (1 + e^2)),
        // from one reciprocal; y's scale folds in the texel count
        const float e = sqrtf(e2);
        const float a6 = fmaf(6.f, e2, 1.f), a3 = 3.f * (1.f + e2);
        const float iq = recip<SHORT>(a6 * a3);
        const float ux = a3 * iq;
        const float yk = fmaf(6.f * e2, e, 1.f) * (a6 * iq) * P.u_nphi1f;
        float fxu = fminf(fmaxf(ux * P.u_ne1f, 0.f), P.u_ne1f);
        int ui0 = (int)fxu, ui1 = min(ui0 + 1, P.u_ne - 1);
        float utx = fxu - ui0;
        auto ulook = [&](float ph) {
          float fy = fminf(fmaxf(ph * yk, 0.f), P.u_nphi1f);
          int j0 = (int)fy, j1 = min(j0 + 1, P.u_nphi - 1);
          float ty2 = fy - j0;
          if (!check(j0 >= 0 && j1 < P.u_nphi && ui0 >= 0 && ui1 < P.u_ne)) return 0.f;
          const int b0 = j0 * P.u_ne + ui0, du = ui1 - ui0, dv = (j1 - j0) * P.u_ne;
          float a = sm_tab(s_U, b0), b = sm_tab(s_U, b0 + du);
          float c = sm_tab(s_U, b0 + dv), d = sm_tab(s_U, b0 + dv + du);
          float lo = fmaf(utx, b - a, a), hi = fmaf(utx, d - c, c);
          return fmaf(ty2, hi - lo, lo);
        };
        // retarded times (debug render and animated disc): t = R - 1/u +
        // ln(u/(1-u)) of the camera point and of the apsis, from D's time channel
        float tcam = 0.f, tapsis = 0.f;
        auto t_of_R = [](float R, float uu) { return R - recip<SHORT>(uu) + logf(quot<SHORT>(uu, 1.f - uu)); };
        auto ulookT = [&](float ph) {
          float fy = fminf(fmaxf(ph * yk, 0.f), P.u_nphi1f);
          int j0 = (int)fy, j1 = min(j0 + 1, P.u_nphi - 1);
          float ty2 = fy - j0;
          if (!check(j0 >= 0 && j1 < P.u_nphi && ui0 >= 0 && ui1 < P.u_ne)) return 0.f;
          float a = __ldg(P.UTt + j0 * P.u_ne + ui0), b = __ldg(P.UTt + j0 * P.u_ne + ui1);
          float c = __ldg(P.UTt + j1 * P.u_ne + ui0), d = __ldg(P.UTt + j1 * P.u_ne + ui1);
          float lo = fmaf(utx, b - a, a), hi = fmaf(utx, d - c, c);
          return fmaf(ty2, hi - lo, lo);
        };
        if (DEBUG || anim) {
          tcam = t_of_R(d_bilinear(P.DTt, dn, fx, yv * (dn - 1), xlo, xhi, chk), u);
          if (em < 0.f) tapsis = t_of_R(d_bilinear(P.DTt, dn, fx, (float)(dn - 1), xlo, xhi, chk), ua);
        }
        float phi = Dl + (s == 1 ? kPiF - dma : dma);
        float turns0 = floorf(quot<SHORT>(phi, kPiF));
        float phi0 = fmaf(-kPiF, turns0, phi);
        const float u0 = phi0 < phia ? ulook(phi0) : 0.f;
        if (phi0 < phia && P.u_oc <= u0 && u0 <= P.u_ic && ((s == 1 && u0 > u) || (s == -1 && u0 < u))) {
          hu0 = u0;
          nh = 1;
          odd0 = ((int)turns0 & 1) != 0;
          if (DEBUG || anim) th0 = (float)s * (t_of_R(ulookT(phi0), u0) - tcam);
        }
        if (em < 0.f && s == 1) {
          phi = fmaf(2.f, phia, -phi);
          float turns1 = floorf(quot<SHORT>(phi, kPiF));
          float phi1 = fmaf(-kPiF, turns1, phi);
          const float u1 = phi1 < phia ? ulook(phi1) : 0.f;
          if (phi1 < phia && P.u_oc <= u1 && u1 <= P.u_ic) {
            float tk = 0.f;
            if (DEBUG || anim) tk = fmaf(2.f, tapsis, -tcam) - t_of_R(ulookT(phi1), u1);
            const bool odd = ((int)turns1 & 1) != 0;
            if (nh == 0) { hu0 = u1; th0 = tk; odd0 = odd; } else { hu1 = u1; th1 = tk; odd1 = odd; }
            ++nh;
          }
        }
      }
      if (udot > 0.f) {
        if (em < 0.f) turn = fmaf(2.f, Da, -Dl);
        else captured = true;
      } else {
        turn = Dl;
      }
      delta_p = delta + turn;
    }

    // ---- disc hits, front to back (Sec. 3.3.3, 3.4.2)
    float LX = 0.f, LY = 0.f, LZ = 0.f, trans = 1.f;
    float dop0 = 0.f, dop1 = 0.f, dens0 = 0.f, dens1 = 0.f;
    if (nh > 0) {
      // nu/nu' for an emitter on the circular orbit at u' (Eq. Doppler, Eq. k_prime):
      // gamma (1 + beta.d^) / (gamma' (1 + beta'.d^')) sqrt((1-u')/(1-u)) simplifies to
      // dcam sqrt(2 - 3u') / (sqrt(1-u) (sqrt(2) + u'^(3/2) (e_z.e_z') / e)).
      const float ie = rsqrtf(e2);
      const float dpre = dcam * C.inv_sqrt_1mu;
      for (int h = 0; h < nh; ++h) {
        float up = h == 0 ? hu0 : hu1;
        float rho_h = P.rho;
        if (anim) {
          // Appendix B: density at the hit's retarded time, radius and azimuth
          const float sg = (h == 0 ? odd0 : odd1) ? -1.f : 1.f;
          rho_h = particle_density(s_part, P.n_parts, P.rho, h == 0 ? th0 : th1, recip<SHORT>(up),
                                   atan2f(sg * tsy, sg * tsx));
        }
        if (h == 0) dens0 = rho_h; else dens1 = rho_h;
        const float sc = rho_h * P.exp_disc;
        float su = sqrtf(up);
        float Dk = quot<SHORT>(dpre * sqrtf(fmaf(-3.f, up, 2.f)), fmaf(up * su * z2, ie, 1.41421356f));
        if (h == 0) dop0 = Dk; else dop1 = Dk;
        // T^4 ~ u^3 (1 - sqrt(3u)), T = t_peak at the maximum: log2(D T)
        float fu = up * up * up * fmaf(-1.7320508f, su, 1.f);
        if (fu > 0.f) {
          // hardware log2 and exp (errors of a few 1e-6 relative at most
          // here, far below the black-body table's interpolation error)
          float lgT = fmaf(0.25f, __log2f(Dk * Dk * Dk * Dk * fu), P.lg_t0);  // log2(D T)
          if (lgT >= 8.f) {  // D T >= 256 K
            float f = fmaf(lgT - 8.f, kDiscN / 12.f, -0.5f);
            f = fminf(fmaxf(f, 0.f), (float)(kDiscN - 1));
            int k0 = (int)f, k1 = min(k0 + 1, kDiscN - 1);
            float tt = f - k0;
            if (!check(k0 >= 0 && k1 < kDiscN)) k0 = k1 = 0;
            float4 a = s_disc[k0], b = s_disc[k1];
            // (ln Y, X/Y, Z/Y) table.  Y over the peak's by the difference of the
            // logarithms: Y itself leaves the float range below 383 K (at 256 K it is
            // e^-113), the ratio does not, and the exponential of a small number is
            // the more accurate one.
            float wy = trans * sc * __expf(fmaf(tt, b.x - a.x, a.x) - ln_peak);
            LX = fmaf(wy, fmaf(tt, b.y - a.y, a.y), LX);
            LY += wy;
            LZ = fmaf(wy, fmaf(tt, b.z - a.z, a.z), LZ);
          }
        }
        trans *= 1.f - rho_h;
      }
    }

    // ---- escape direction and its screen-space derivatives (quad shuffles)
    // d' = cos(delta') e_x' + sin(delta') e_y', evaluated as the rotation of the
    // unit beam direction by the turn angle (delta' - delta) about e_z': the
    // sum delta + turn is never rounded, which keeps d' to a few 1e-8.
    float st_, ct_;
    sincosf(turn, &st_, &ct_);
    float idd = rsqrtf(dd2);
    float b0 = d0 * idd, b1 = d1 * idd, b2 = d2 * idd;
    float n0 = fmaf(z1, b2, -z2 * b1), n1 = fmaf(z2, b0, -z0 * b2), n2 = fmaf(z0, b1, -z1 * b0);
    float dp0 = captured ? 0.f : fmaf(ct_, b0, st_ * n0);
    float dp1 = captured ? 0.f : fmaf(ct_, b1, st_ * n1);
    float dp2 = captured ? 0.f : fmaf(ct_, b2, st_ * n2);
    unsigned capbits = __ballot_sync(0xffffffffu, captured);
    bool anycap = ((capbits >> (lane & ~3)) & 0xfu) != 0u;
    // Fine derivatives up to sign: the quad neighbour's value subtracted from
    // this pixel's.  The signs (+1 on odd columns, -1 on odd rows) are left
    // out: every use below is even in them -- |cross products| for
    // Omega/Omega', |J| column sums for the half-extents, and the tent weights
    // f(w) f(h), whose (w, h) only change sign with J's columns -- and a sign
    // flip is exact in floating point.
    auto dw = [&](float v) { return v - __shfl_xor_sync(0xffffffffu, v, 1); };
    auto dh = [&](float v) { return v - __shfl_xor_sync(0xffffffffu, v, 2); };
    float dw0 = dw(dp0), dw1 = dw(dp1), dw2 = dw(dp2);
    float dh0 = dh(dp0), dh1 = dh(dp1), dh2 = dh(dp2);
    float qw0 = dw(q0), qw1 = dw(q1), qw2 = dw(q2);
    float qh0 = dh(q0), qh1 = dh(q1), qh2 = dh(q2);

    // ---- star gather over the beam footprint (Sec. 3.3.2) and lensing (Sec. 3.4.1)
    float omega = 0.f, dstar = 0.f, SX = 0.f, SY = 0.f, SZ = 0.f;
    int level = -1, face = -1, visited = 0;
    if (!anycap && P.cube) {
      float cq0 = fmaf(qw1, qh2, -qw2 * qh1), cq1 = fmaf(qw2, qh0, -qw0 * qh2), cq2 = fmaf(qw0, qh1, -qw1 * qh0);
      float cd0 = fmaf(dw1, dh2, -dw2 * dh1), cd1 = fmaf(dw2, dh0, -dw0 * dh2), cd2 = fmaf(dw0, dh1, -dw1 * dh0);
      const float den2 = fmaf(cd0, cd0, fmaf(cd1, cd1, cd2 * cd2));
      if (den2 > 0.f) {
        omega = sqrtf(fmaf(cq0, cq0, fmaf(cq1, cq1, cq2 * cq2))) * rsqrtf(den2);
        float ax = fabsf(dp0), ay = fabsf(dp1), az = fabsf(dp2);
        float sc, tc, ma, dmaw, dmah, dscw, dsch, dtcw, dtch;
        if (ax >= ay && ax >= az) {
          ma = ax;
          if (dp0 >= 0.f) { face = 0; sc = -dp2; tc = -dp1; dmaw = dw0; dmah = dh0; dscw = -dw2; dsch = -dh2; dtcw = -dw1; dtch = -dh1; }
          else { face = 1; sc = dp2; tc = -dp1; dmaw = -dw0; dmah = -dh0; dscw = dw2; dsch = dh2; dtcw = -dw1; dtch = -dh1; }
        } else if (ay >= az) {
          ma = ay;
          if (dp1 >= 0.f) { face = 2; sc = dp0; tc = dp2; dmaw = dw1; dmah = dh1; dscw = dw0; dsch = dh0; dtcw = dw2; dtch = dh2; }
          else { face = 3; sc = dp0; tc = -dp2; dmaw = -dw1; dmah = -dh1; dscw = dw0; dsch = dh0; dtcw = -dw2; dtch = -dh2; }
        } else {
          ma = az;
          if (dp2 >= 0.f) { face = 4; sc = dp0; tc = -dp1; dmaw = dw2; dmah = dh2; dscw = dw0; dsch = dh0; dtcw = -dw1; dtch = -dh1; }
          else { face = 5; sc = -dp0; tc = -dp1; dmaw = -dw2; dmah = -dh2; dscw = -dw0; dsch = -dh0; dtcw = -dw1; dtch = -dh1; }
        }
        const int N = P.cube_n;
        float hN = 0.5f * N, ima = recip<SHORT>(ma), hNi = hN * ima;
        float sr = sc * ima, tr = tc * ima;
        float S = (sr + 1.f) * hN, T = (tr + 1.f) * hN;
        float Jsw = hNi * fmaf(-sr, dmaw, dscw), Jsh = hNi * fmaf(-sr, dmah, dsch);
        float Jtw = hNi * fmaf(-tr, dmaw, dtcw), Jth = hNi * fmaf(-tr, dmah, dtch);
        float hs = fabsf(Jsw) + fabsf(Jsh), ht = fabsf(Jtw) + fabsf(Jth);
        float hm = fmaxf(hs, ht);
        // smallest level L with 2 hm <= 8 * 2^L (at most 9x9 texels, C17): from
        // the exponent of hm/4 (exact: every quantity is a power-of-two scale)
        int L = 0;
        {
          const float t4 = 0.25f * hm;
          if (t4 > 1.f) {
            const unsigned b = __float_as_uint(t4);
            L = (int)(b >> 23) - 127 + ((b & 0x7fffffu) != 0u ? 1 : 0);
          }
          L = min(L, P.cube_levels - 1);
        }
        level = L;
        const float sL = __int_as_float((127 - L) << 23);  // 2^-L
        int NL = N >> L;
        float cS = S * sL, cT = T * sL, hsL = hs * sL, htL = ht * sL;
        float a11 = Jsw * sL, a12 = Jsh * sL, a21 = Jtw * sL, a22 = Jth * sL;
        float det = fmaf(a11, a22, -a12 * a21);
        if (det * det > 1e-12f * (fmaf(a11, a11, a21 * a21) * fmaf(a12, a12, a22 * a22)) &&
            check(L >= 0 && L < P.cube_levels && L < kMaxLevels && face >= 0 && face < 6)) {
          float id = recip<SHORT>(det);
          float i11 = a22 * id, i12 = -a12 * id, i21 = -a21 * id, i22 = a11 * id;
          int i0 = max((int)floorf(cS - hsL), 0), i1 = min((int)floorf(cS + hsL), NL - 1);
          int j0 = max((int)floorf(cT - htL), 0), j1 = min((int)floorf(cT + htL), NL - 1);
          if (DEBUG) visited = max(i1 - i0 + 1, 0) * max(j1 - j0 + 1, 0);
          const uint2 *rec = P.cube + P.level_off[L] + face * NL * NL;
          const float lscale = __int_as_float((127 + 2 * L) << 23);  // 4^L
          // star at (i + (ps + 1/2)/256, j + (pt + 1/2)/256) in level-L texels
          const float q11 = i11 * (1.f / 256.f), q12 = i12 * (1.f / 256.f);
          const float q21 = i21 * (1.f / 256.f), q22 = i22 * (1.f / 256.f);
          const int nbx = max(NL >> 3, 1);  // occupancy blocks per block row
          const uint2 *blk = P.cube_mask + P.mask_off[L] + face * (nbx * max(NL >> 2, 1));
          const float ds0 = (i0 - cS) + 0.5f / 256.f;
          // The gather is bound by instruction issue, and what it issues is set by
          // the warp's busiest lane.  So a lane's stars come from one 64-bit window
          // of occupancy bits and every lane walks its own list, whichever row it is
          // in: 3.3 take iterations per warp tile of the 1080p frame against 8.6 when
          // the lanes moved from row to row together (of 123 occupied texels in a
          // tile's 32 bounding boxes only 15 hold a star with a weight: the rest lie
          // beside thin, slanted footprints; the cull leaves 61).  Every star's weight is rounded in the
          // same steps as in a walk row by row; stars are taken window by window
          // (in row order up to eight columns) and by rows inside one.
          // 1080p frame 98.5 -> 87.3 us, 4K 435 -> 375 us, 256^2 24.7 -> 17.2 us.
          // Occupancy of the 8 x 8 texels from (wi, wj) on, clipped to the
          // footprint: bit 31 - (8 r + c) of x (rows 0-3) or y (rows 4-7) is
          // texel (wi + c, wj + r).  Blocks overlap by half along a row, so the
          // window's columns lie in one block column; its rows in two or three
          // blocks, put together by one funnel shift.
          auto window = [&](const int wi, const int wj) {
            const int c = wi & 7, r = wj & 3;
            const int ncol = min(i1 - wi + 1, 8), nrow = min(j1 - wj + 1, 8);
            const uint2 *p = blk + ((wj >> 2) * nbx + (wi >> 3));
            if (!check(wi >= 0 && wj >= 0 && ncol > 0 && nrow > 0 && wi + ncol <= NL && wj + nrow <= NL))
              return make_uint2(0u, 0u);
            const uint2 zero = make_uint2(0u, 0u);
            const uint2 a = __ldg(p), b = r + nrow > 4 ? __ldg(p + nbx) : zero,
                        d = r + nrow > 8 ? __ldg(p + 2 * nbx) : zero;
            // the eight columns from c on of a block's four 16-bit rows
            auto rows = [&](const uint2 v) { return __byte_perm(v.y << c, v.x << c, 0x7531u); };
            const unsigned wa = rows(a), wb = rows(b), wd = rows(d);
            const unsigned mc = ((0xff00u >> ncol) & 0xffu) * 0x01010101u;
            const unsigned lo = __funnelshift_l(wb, wa, 8 * r), hi = __funnelshift_l(wd, wb, 8 * r);
            return make_uint2(lo & mc & ~__funnelshift_rc(0xffffffffu, 0u, 8 * nrow),
                              hi & mc & ~__funnelshift_rc(0xffffffffu, 0u, max(8 * nrow - 32, 0)));
          };
          // Texels of the window that the footprint can touch: the columns that
          // both of its strips |w| < 1 and |h| < 1 reach anywhere in a row, widened
          // by 0.01 texel and the rounding of the strip's own terms.  A strip along
          // the rows (a slope that is not finite) bounds nothing: fmaxf and fminf
          // drop the NaN.
          auto cull = [&](const uint2 bits, const int wi, const int wj) {
            const float r22 = recip<SHORT>(a22), r21 = recip<SHORT>(a21);
            const float s1 = a12 * r22, s2 = a11 * r21, g1 = fabsf(det * r22), g2 = fabsf(det * r21);
            const float y = wj - cT, x = cS - wi;
            const float e1 = fmaf(1e-5f, fmaf(16.f, fabsf(s1), g1), g1 + 0.01f);
            const float e2 = fmaf(1e-5f, fmaf(16.f, fabsf(s2), g2), g2 + 0.01f);
            const float m1 = fmaf(s1, y, x), m2 = fmaf(s2, y, x);
            const float lo1 = (m1 + fminf(s1, 0.f)) - e1, hi1 = (m1 + fmaxf(s1, 0.f)) + e1 + 1.f;
            const float lo2 = (m2 + fminf(s2, 0.f)) - e2, hi2 = (m2 + fmaxf(s2, 0.f)) + e2 + 1.f;
            auto rows = [&](const int r0) {
              unsigned row[4];
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                const float r = (float)(r0 + k);
                const float lo = fmaxf(fmaxf(fmaf(r, s1, lo1), fmaf(r, s2, lo2)), 0.f);
                const float hi = fminf(fminf(fmaf(r, s1, hi1), fmaf(r, s2, hi2)), 9.f);
                row[k] = __funnelshift_rc(0xffu, 0u, __float2uint_rd(lo)) &
                         ~__funnelshift_rc(0xffu, 0u, __float2uint_rd(hi));
              }
              return __byte_perm(__byte_perm(row[3], row[2], 0x0040u), __byte_perm(row[1], row[0], 0x0040u), 0x5410u);
            };
            return make_uint2(bits.x & rows(0), bits.y ? bits.y & rows(4) : 0u);
          };
          // the loop is compiled once per record format (no format test per star)
          auto gather = [&](auto bf16_tag) {
            for (int wj = j0; wj <= j1; wj += 8)
              for (int wi = i0; wi <= i1; wi += 8) {
                uint2 bits = window(wi, wj);
                if (__popc(bits.x) + __popc(bits.y) > kCullAbove) bits = cull(bits, wi, wj);
                int jw = wj;  // first row of bits.x
                // every lane walks its own stars, whichever row they are in
                while (bits.x | bits.y) {
                  if (bits.x == 0u) {
                    bits = make_uint2(bits.y, 0u);
                    jw = wj + 4;
                  }
                  const int k = __clz(bits.x);
                  bits.x &= ~(0x80000000u >> k);
                  const int ii = wi + (k & 7), jj = jw + (k >> 3);
                  if (!check(ii <= i1 && jj <= j1)) continue;
                  const uint2 r = __ldg(rec + (jj * NL + ii));
                  // small integers as floats: 2^23 + n has the bits 0x4B000000 + n
                  const float kf = __uint_as_float(0x4B000000u + (ii - i0)) - 8388608.f;
                  const float jf = __uint_as_float(0x4B000000u + jj) - 8388608.f;
                  const float dt = (jf - cT) + 0.5f / 256.f;
                  const float wrow = fmaf(i11, ds0, i12 * dt), hrow = fmaf(i21, ds0, i22 * dt);
                  // the star's position bytes (bits 16..23 and 24..31 of r.y) as floats
                  const float ps = __uint_as_float(__byte_perm(r.y, 0x4B000000u, 0x7442u)) - 8388608.f;
                  const float pt = __uint_as_float(__byte_perm(r.y, 0x4B000000u, 0x7443u)) - 8388608.f;
                  const float w = fmaf(q11, ps, fmaf(q12, pt, fmaf(i11, kf, wrow)));
                  const float h = fmaf(q21, ps, fmaf(q22, pt, fmaf(i21, kf, hrow)));
                  // tent weight f(w) f(h), 0 outside the footprint (1 - |w| <= 1: the
                  // saturation clamps at 0 only)
                  const float wt = __saturatef(1.f - fabsf(w)) * __saturatef(1.f - fabsf(h));
                  float X, Y, Z;
                  if constexpr (decltype(bf16_tag)::value) {
                    X = __uint_as_float(r.x << 16);
                    Y = __uint_as_float(r.x & 0xffff0000u);
                    Z = __uint_as_float(r.y << 16);
                  } else {
                    __half2 xy2, zp2;
                    memcpy(&xy2, &r.x, 4);
                    memcpy(&zp2, &r.y, 4);
                    const float2 xy = __half22float2(xy2);
                    X = xy.x;
                    Y = xy.y;
                    Z = __low2float(zp2);
                  }
                  // the level's scale 4^L multiplies the sums once, after the loop
                  // (a power of two: the same result as scaling every weight)
                  SX = fmaf(wt, X, SX);
                  SY = fmaf(wt, Y, SY);
                  SZ = fmaf(wt, Z, SZ);
                }
              }
          };
          if (P.cube_bf16) gather(std::true_type{}); else gather(std::false_type{});
          SX *= lscale;
          SY *= lscale;
          SZ *= lscale;
        }
      }
      dstar = dcam * C.inv_sqrt_1mu;  // static star at infinity: u' = 0
      float Ssum = SX + SY + SZ;
      if (Ssum > 0.f) {
        // C(xy, D): trilinear, texel centres, clamped.  One base texel and
        // constant strides (0 at a clamped edge, where the weight is 0);
        // interpolated along x, then y, then log2 D.
        const float iS = recip<SHORT>(Ssum);
        float fx = fmaf(SX * iS, kCnx / 0.60f, -(0.15f * kCnx / 0.60f + 0.5f));
        float fy = fmaf(SY * iS, kCny / 0.35f, -(0.15f * kCny / 0.35f + 0.5f));
        float fz = fmaf(__log2f(dstar), kCnd / 8.f, 4.f * kCnd / 8.f - 0.5f);
        fx = fminf(fmaxf(fx, 0.f), kCnx - 1.f);
        fy = fminf(fmaxf(fy, 0.f), kCny - 1.f);
        fz = fminf(fmaxf(fz, 0.f), kCnd - 1.f);
        int i0 = (int)fx, j0 = (int)fy, k0 = (int)fz;
        const float tx2 = fx - i0, ty2 = fy - j0, tz2 = fz - k0;
        const int si = i0 < kCnx - 1 ? 1 : 0, sj = j0 < kCny - 1 ? kCnx : 0;
        const int sk = k0 < kCnd - 1 ? kCnx * kCny : 0;
        if (!check(i0 >= 0 && j0 >= 0 && k0 >= 0 && i0 < kCnx && j0 < kCny && k0 < kCnd)) i0 = j0 = k0 = 0;
        const float4 *cb = P.C + ((k0 * kCny + j0) * kCnx + i0);
        const float4 c000 = __ldg(cb), c100 = __ldg(cb + si), c010 = __ldg(cb + sj), c110 = __ldg(cb + sj + si);
        const float4 c001 = __ldg(cb + sk), c101 = __ldg(cb + sk + si), c011 = __ldg(cb + sk + sj),
                     c111 = __ldg(cb + sk + sj + si);
        // packed f32x2 lerps: (x, y) and (z, pad) of each float4 texel at once
        auto lerp3 = [](float t, float4 a, float4 b) {
          const float2 t2 = make_float2(t, t), m1 = make_float2(-1.f, -1.f);
          const float2 axy = make_float2(a.x, a.y), azw = make_float2(a.z, a.w);
          const float2 xy = __ffma2_rn(t2, __ffma2_rn(axy, m1, make_float2(b.x, b.y)), axy);
          const float2 zw = __ffma2_rn(t2, __ffma2_rn(azw, m1, make_float2(b.z, b.w)), azw);
          return make_float4(xy.x, xy.y, zw.x, zw.y);
        };
        const float4 cy0 = lerp3(ty2, lerp3(tx2, c000, c100), lerp3(tx2, c010, c110));
        const float4 cy1 = lerp3(ty2, lerp3(tx2, c001, c101), lerp3(tx2, c011, c111));
        const float4 cc = lerp3(tz2, cy0, cy1);
        const float cx = cc.x, cy = cc.y, cz = cc.z;
        float sc = Ssum * omega * P.exp_stars * trans;
        LX = fmaf(sc, cx, LX);
        LY = fmaf(sc, cy, LY);
        LZ = fmaf(sc, cz, LZ);
      }
    }

    // ---- store
    const float R_ = fmaf(P.M[0], LX, fmaf(P.M[1], LY, P.M[2] * LZ));
    const float G_ = fmaf(P.M[3], LX, fmaf(P.M[4], LY, P.M[5] * LZ));
    const float B_ = fmaf(P.M[6], LX, fmaf(P.M[7], LY, P.M[8] * LZ));
    if (!DEBUG && C.rgb) {
      // packed RGB (12 bytes per pixel), for frames that go to the host
      float *o3 = reinterpret_cast<float *>(C.out);
      const int px0 = px - lx, py0 = py - ly;
      if (C.rgb_vec && px0 + 8 <= C.width) {
        // the warp's four 8-pixel rows are four 96-byte runs: stage them in
        // shared memory, then lanes 0..23 store them as 16-byte chunks
        float *sw = s_rgb + 96 * (threadIdx.x >> 5);
        sw[24 * ly + 3 * lx] = R_;
        sw[24 * ly + 3 * lx + 1] = G_;
        sw[24 * ly + 3 * lx + 2] = B_;
        __syncwarp();
        if (lane < 24) {
          const int r = lane / 6, c = lane - 6 * r;
          if (py0 + r < C.height)
            reinterpret_cast<float4 *>(o3 + 3 * ((long long)(py0 + r) * C.width + px0))[c] =
                reinterpret_cast<const float4 *>(sw + 24 * r)[c];
        }
        __syncwarp();
      } else if (px < C.width && py < C.height) {
        float *q = o3 + 3 * ((long long)py * C.width + px);
        q[0] = R_;
        q[1] = G_;
        q[2] = B_;
      }
    } else if (px < C.width && py < C.height) {
      long long o = (long long)py * C.width + px;
      C.out[o] = make_float4(R_, G_, B_, 1.f);
      if (DEBUG) {
        float *g = C.dbg + o * kDbgFloats;
        float4 *g4 = reinterpret_cast<float4 *>(g);
        g4[0] = make_float4(e2, delta, captured ? INFINITY : delta_p, (float)nh);
        g4[1] = make_float4(hu0, hu1, (float)(anycap ? -1 : level), (float)(anycap ? -1 : face));
        g4[2] = make_float4(omega, dstar, SX, SY);
        g4[3] = make_float4(SZ, dop0, dop1, (float)visited);
        g4[4] = make_float4(th0, th1, dens0, dens1);
      }
    }
    };
    if (P.cams) {
      if (cam + 1 < P.ncams && __ldg(&P.cams[cam + 1].tile0) <= (int)tile)
        cam = MODE == kAnimated ? camera_of_tile(P.cams, P.ncams, cam, (int)tile)
                                : search_camera(P.cams, P.ncams, cam, (int)tile);
      const CamConst &Cb = P.cams[cam];
      const int t = (int)tile - Cb.tile0;
      ++tile;
      shade(Cb, t);
    } else {
      const int t = (int)tile;
      ++tile;
      shade(P.cam0, t);
    }
    } while (tile != tile_end);
    if (!counted) {
      if (MODE == kAnimated) return;
      g += n_warps;
      continue;
    }
    if (lane == 0) g = n_warps + atomicAdd(P.sched, 1u);
    g = __shfl_sync(0xffffffffu, g, 0);
  }
  if (!counted) return;
  // Retire the warp; the last warp of the grid re-arms the counters for the
  // next launch that uses them (every warp has taken its final fetch by then).
  if (lane == 0) {
    __threadfence();
    unsigned nw = gridDim.x * (blockDim.x >> 5);
    if (atomicAdd(P.sched + 1, 1u) == nw - 1u) {
      atomicExch(P.sched, 0u);
      atomicExch(P.sched + 1, 0u);
    }
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------

static bool validate_camera(const bh_camera *c, int idx) {
  if (!c) { set_error("camera %d is NULL", idx); return false; }
  if (!(c->r > 1.0) || !std::isfinite(c->r)) {
    set_error("camera %d: r = %g, must be > 1 (outside the horizon)", idx, c->r);
    return false;
  }
  double v2 = c->v[0] * c->v[0] + c->v[1] * c->v[1] + c->v[2] * c->v[2];
  if (!(v2 < 1.0)) { set_error("camera %d: |v| = %g, must be < 1", idx, sqrt(v2)); return false; }
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      double s = 0.0;
      for (int k = 0; k < 3; ++k) s += c->orient[i * 3 + k] * c->orient[j * 3 + k];
      if (fabs(s - (i == j ? 1.0 : 0.0)) > 1e-6) {
        set_error("camera %d: orientation is not orthonormal", idx);
        return false;
      }
    }
  if (!(c->fov_y > 0.0 && c->fov_y < kPi)) { set_error("camera %d: fov_y out of (0, pi)", idx); return false; }
  if (c->width < 1 || c->height < 1 || c->width > 16384 || c->height > 16384) {
    set_error("camera %d: size %dx%d out of 1..16384", idx, c->width, c->height);
    return false;
  }
  return true;
}

static bool validate_disc(const bh_disc *d) {
  if (!d) { set_error("disc is NULL"); return false; }
  if (!d->enabled) return true;
  if (!(d->r_in >= 3.0) || !(d->r_out > d->r_in) || !std::isfinite(d->r_out)) {
    set_error("disc: need 3 <= r_in < r_out (got %g, %g)", d->r_in, d->r_out);
    return false;
  }
  if (!(d->density >= 0.0 && d->density <= 1.0) || !(d->t_peak_K > 0.0)) {
    set_error("disc: density in [0,1] and t_peak_K > 0 required");
    return false;
  }
  if (d->particles && !std::isfinite(d->time)) {
    set_error("disc: time must be finite");
    return false;
  }
  return true;
}

// Complete elliptic integral of the first kind K(k) by the arithmetic-
// geometric mean: K = pi / (2 AGM(1, sqrt(1 - k^2))).
static double ellipk_agm(double k) {
  double a = 1.0, b = sqrt(1.0 - k * k);
  for (int it = 0; it < 64 && fabs(a - b) > 1e-16 * a; ++it) {
    double an = 0.5 * (a + b);
    b = sqrt(a * b);
    a = an;
  }
  return kPi / (2.0 * a);
}

extern "C" bh_status bh_disc_particles_create(bh_ctx *ctx, const double *ph, int n, bh_particles **out) {
  if (!ctx || !ph || !out) { set_error("bh_disc_particles_create: NULL argument"); return BH_ERR_INVALID_ARG; }
  *out = nullptr;
  if (n < 1 || n > kMaxParticles) {
    set_error("bh_disc_particles_create: n = %d, must be 1..%d", n, kMaxParticles);
    return BH_ERR_INVALID_ARG;
  }
  std::vector<double> rows((size_t)n * 8);
  for (int k = 0; k < n; ++k) {
    const double u1 = ph[3 * k], u2 = ph[3 * k + 1], phi0 = ph[3 * k + 2];
    if (!(u1 > 0.0 && u1 <= u2 && u2 <= 1.0 / 3.0) || !std::isfinite(phi0)) {
      set_error("bh_disc_particles_create: row %d needs 0 < u1 <= u2 <= 1/3 and a finite phase", k);
      return BH_ERR_INVALID_ARG;
    }
    const double u3 = 1.0 - u1 - u2, ub = 0.5 * (u1 + u2);
    const double K = ellipk_agm(sqrt((u2 - u1) / (u3 - u1)));
    double *r = &rows[(size_t)k * 8];
    r[0] = u1;
    r[1] = u2;
    r[2] = phi0;
    r[3] = sqrt(0.5 * ub * ub * ub);          // d phi / dt
    r[4] = kPi * sqrt(u3 - u1) / (4.0 * K);    // sin^2 argument per radian of phi
    r[5] = 1.0 / u2 - 1.0;                     // radii a hit can be within 1 of
    r[6] = 1.0 / u1 + 1.0;
    r[7] = 0.0;
  }
  // sorted by rmin: the density loop stops at the first particle beyond the hit
  std::vector<int> idx(n);
  for (int k = 0; k < n; ++k) idx[k] = k;
  std::stable_sort(idx.begin(), idx.end(), [&](int a, int b) { return rows[a * 8 + 5] < rows[b * 8 + 5]; });
  std::vector<double> sorted((size_t)n * 8);
  for (int k = 0; k < n; ++k)
    for (int j = 0; j < 8; ++j) sorted[(size_t)k * 8 + j] = rows[(size_t)idx[k] * 8 + j];
  BH_CUDA(cudaSetDevice(ctx->device));
  bh_particles *p = new bh_particles();
  p->ctx = ctx;
  p->n = n;
  cudaError_t e = pool_malloc(*ctx->pool, (void **)&p->dev, sorted.size() * sizeof(double));
  if (e == cudaSuccess) e = cudaMemcpy(p->dev, sorted.data(), sorted.size() * sizeof(double), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    cudaFree(p->dev);
    delete p;
    return cuda_fail(e, "bh_disc_particles_create");
  }
  *out = p;
  return BH_OK;
}

extern "C" void bh_disc_particles_free(bh_particles *p) {
  if (!p) return;
  cudaSetDevice(p->ctx->device);
  cudaDeviceSynchronize();
  cudaFree(p->dev);
  delete p;
}

// Camera frame in FP64: static basis (Eq. staticbasis), boost B(v) (the
// camera's 4-velocity is gamma (1, v) on the static frame), user rotation O.
__host__ __device__ static void camera_constants_at(const bh_camera *c, double st, double ct, double sp, double cph,
                                                    CamConst *k) {  // sines and cosines of theta, phi
  double u = 1.0 / c->r;
  double rh[3] = {st * cph, st * sp, ct}, th[3] = {ct * cph, ct * sp, -st}, ph[3] = {-sp, cph, 0.0};
  const double *v = c->v;
  double v2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
  double g = 1.0 / sqrt(1.0 - v2);
  // The boost B(v) keeps the components across v and scales the one along v
  // (the camera's 4-velocity is gamma (1, v) on the static frame); the
  // camera axes e_w, e_h, e_d are O e' (rows of O on the boosted axes).
  double vn = sqrt(v2);
  double vh[3] = {0.0, 0.0, 0.0};
  if (vn > 0.0)
    for (int j = 0; j < 3; ++j) vh[j] = v[j] / vn;
  for (int j = 0; j < 3; ++j) {
    double wc = 0.0;
    for (int m = 0; m < 3; ++m) wc += c->orient[j * 3 + m] * vh[m];
    k->w[j] = (float)wc;
  }
  k->beta = (float)vn;
  k->inv_gamma2 = (float)(1.0 - v2);
  double s1 = sqrt(1.0 - u);
  for (int r = 0; r < 3; ++r) {
    // row r of R: (sqrt(1-u) r^, theta^, phi^) components r; M = R O^T, rv = R v^
    const double Rr[3] = {s1 * rh[r], th[r], ph[r]};
    for (int col = 0; col < 3; ++col)
      k->M[r * 3 + col] = (float)(Rr[0] * c->orient[col * 3 + 0] + Rr[1] * c->orient[col * 3 + 1] +
                                  Rr[2] * c->orient[col * 3 + 2]);
    k->rv[r] = (float)(Rr[0] * vh[0] + Rr[1] * vh[1] + Rr[2] * vh[2]);
    k->x[r] = (float)rh[r];
  }
  // radial beams (reading C8): e_z' = x ^ (least-aligned axis) / |.|
  int m = fabs(rh[0]) <= fabs(rh[1]) ? (fabs(rh[0]) <= fabs(rh[2]) ? 0 : 2) : (fabs(rh[1]) <= fabs(rh[2]) ? 1 : 2);
  double axv[3] = {0, 0, 0};
  axv[m] = 1.0;
  double z[3] = {rh[1] * axv[2] - rh[2] * axv[1], rh[2] * axv[0] - rh[0] * axv[2], rh[0] * axv[1] - rh[1] * axv[0]};
  double zn = sqrt(z[0] * z[0] + z[1] * z[1] + z[2] * z[2]);
  for (int r = 0; r < 3; ++r) k->zdeg[r] = (float)(z[r] / zn);
  k->gamma = (float)g;
  k->f = (float)(0.5 * c->height / tan(0.5 * c->fov_y));
  k->u = (float)u;
  k->inv_sqrt_1mu = (float)(1.0 / s1);
  k->half_w = (float)(0.5 * c->width);
  k->half_h = (float)(0.5 * c->height);
  k->width = c->width;
  k->height = c->height;
  k->rgb = 0;  // RGBA float4 frames unless the host-bound form asks for packed RGB
  k->rgb_vec = 0;
}

__host__ __device__ static void camera_constants(const bh_camera *c, CamConst *k) {
  camera_constants_at(c, sin(c->theta), cos(c->theta), sin(c->phi), cos(c->phi), k);
}

// XYZ -> linear sRGB from the Rec.709 primaries and the D65 white point.
static void xyz_to_srgb(float *M) {
  const double px[3] = {0.64, 0.30, 0.15}, py[3] = {0.33, 0.60, 0.06};
  const double W[3] = {0.3127 / 0.3290, 1.0, (1.0 - 0.3127 - 0.3290) / 0.3290};
  double P[3][3];
  for (int c = 0; c < 3; ++c) {
    P[0][c] = px[c] / py[c];
    P[1][c] = 1.0;
    P[2][c] = (1.0 - px[c] - py[c]) / py[c];
  }
  // inverse by Gauss-Jordan
  double a[3][6];
  for (int r = 0; r < 3; ++r)
    for (int c = 0; c < 6; ++c) a[r][c] = c < 3 ? P[r][c] : (c - 3 == r ? 1.0 : 0.0);
  for (int c = 0; c < 3; ++c) {
    int p = c;
    for (int r = c + 1; r < 3; ++r)
      if (fabs(a[r][c]) > fabs(a[p][c])) p = r;
    for (int k = 0; k < 6; ++k) { double t = a[c][k]; a[c][k] = a[p][k]; a[p][k] = t; }
    double d = a[c][c];
    for (int k = 0; k < 6; ++k) a[c][k] /= d;
    for (int r = 0; r < 3; ++r)
      if (r != c) {
        double f = a[r][c];
        for (int k = 0; k < 6; ++k) a[r][k] -= f * a[c][k];
      }
  }
  double S[3];
  for (int r = 0; r < 3; ++r) S[r] = a[r][3] * W[0] + a[r][4] * W[1] + a[r][5] * W[2];
  for (int r = 0; r < 3; ++r)
    for (int c = 0; c < 3; ++c) M[r * 3 + c] = (float)(a[r][3 + c] / S[r]);
}

static bh_status fill_params(bh_ctx *ctx, const bh_tables *t, const bh_cubemap *cube,
                             const bh_disc *disc, const bh_shading *sh, RenderParams &P) {
  memset(&P, 0, sizeof P);
  P.D = t->D;
  P.d_n = t->desc.d_n;
  P.U = t->U;
  P.u_ne = t->desc.u_ne;
  P.u_nphi = t->desc.u_nphi;
  P.d_n1f = (float)(t->desc.d_n - 1);
  P.u_ne1f = (float)(t->desc.u_ne - 1);
  P.u_nphi1f = (float)(t->desc.u_nphi - 1);
  size_t es = t->desc.storage == BH_F32 ? 4 : 2;
  P.u_bytes = (int)(((size_t)P.u_ne * P.u_nphi * es + 15) / 16 * 16);
  P.DTt = t->DT;
  P.UTt = t->UT;
  P.C = t->C;
  P.disc = t->disc;
  if (cube) {
    P.cube = cube->rec;
    P.cube_n = cube->n;
    P.cube_levels = cube->levels;
    P.cube_bf16 = cube->storage == BH_BF16;
    P.cube_mask = cube->mask;
    for (int L = 0; L < cube->levels && L < kMaxLevels; ++L) {
      P.level_off[L] = cube_level_offset(cube->n, L);
      P.mask_off[L] = mask_level_offset(cube->n, L);
    }
  }
  P.disc_on = disc->enabled ? 1 : 0;
  P.u_ic = disc->enabled ? (float)(1.0 / disc->r_in) : 0.f;
  P.u_oc = disc->enabled ? (float)(1.0 / disc->r_out) : 1.f;
  P.t_peak = (float)(disc->t_peak_K > 0 ? disc->t_peak_K : 1e4);
  P.rho = (float)disc->density;
  if (disc->enabled && disc->particles) {
    P.parts = disc->particles->dev;
    P.n_parts = disc->particles->n;
    P.time = disc->time;
  }
  P.fmax_disc = (float)(pow(12.0 / 49.0, 3) * (1.0 - sqrt(36.0 / 49.0)));
  P.lg_t0 = (float)(log2((double)P.t_peak) - 0.25 * log2(pow(12.0 / 49.0, 3) * (1.0 - sqrt(36.0 / 49.0))));
  P.exp_disc = sh ? sh->exposure_disc : 1.f;
  P.exp_stars = sh ? sh->exposure_stars : 0.01f;
  xyz_to_srgb(P.M);
  P.status = ctx->status_dev;
  P.wait_ns = 200000000ull;  // 0.2 s: the copies take microseconds
  P.inject_wait = 0;
  P.inject_wait_ns = 2000000ull;  // 2 ms
  if (ctx->inject_table_wait) {
    P.inject_wait = 1;
    ctx->inject_table_wait = 0;
  }
  P.sched = ctx->sched_dev + 2 * (ctx->sched_next.fetch_add(1, std::memory_order_relaxed) % kSchedRing);
  return BH_OK;
}

// Warp tiles (8 x 4 pixels) of a w x h image.
__host__ __device__ static inline int tiles_across(int w) { return (w + 7) / 8; }
__host__ __device__ static inline int warp_tiles(int w, int h) { return tiles_across(w) * ((h + 3) / 4); }

// Persistent grid: enough blocks to fill the GPU, no more than the work needs.
static int render_grid(const bh_ctx *ctx, long long tiles) {
  const long long need = (tiles + ctx->tuning.warps_per_block - 1) / ctx->tuning.warps_per_block;
  return (int)std::min<long long>(need, (long long)ctx->sm_count * ctx->tuning.blocks_per_sm);
}

// Tiles of a launch by chunks of two where it has up to kFewTiles per warp, the
// last kFewTail per warp singly; above it by chunks of four, the last kTail singly.
// A chunk in a disc of 256 particles takes four to five times the mean tile's
// time, of which a 1080p frame has 13 per warp: by fours such a chunk was the
// whole frame's time (1080p infall 307 against 229 us, a wide view 276 against 213,
// 4K, with 53 tiles per warp, 323 against 280).  With many tiles per warp the
// counter's round trips are what counts: 64 frames of 1080p (852 per warp) 4072 us
// by fours, 4124 by twos.  kTail measured at 2 / 4 / 6 / 8 / 16 with chunks of four:
// 1080p frame 92.2 / 87.0 / 84.4 / 84.8 / 86.0 us, 4K 353 / 350 / 349 / 349 / 352;
// kFewTail at 3 / 4 / 6 / 8 with chunks of two: 80.0 / 79.8 / 80.0 / 80.1 us, without
// stars 47.5 / 47.5 / 49.5 / 49.5, the infall with 256 particles 231 / 230 / 232 / 190.
// Up to two tiles per warp are taken by place: 640 x 360 23.2 -> 18.7 us, without
// stars 14.6 -> 9.6, all of it in the shadow 14.6 -> 8.6 (counted two at a time 12.6);
// in an animated disc, where two slow tiles of a warp are the frame's time, one (two:
// 64 particles 39 -> 47 us).
constexpr long long kFewTiles = 64, kFewTail = 4, kTail = 6;

static void set_schedule(const bh_ctx *ctx, RenderParams &P, int grid, long long tiles) {
  const long long warps = (long long)grid * ctx->tuning.warps_per_block;
  const bool few = tiles <= kFewTiles * warps;
  P.fetch = ctx->tuning.fetch ? ctx->tuning.fetch : few ? 2 : 4;
  P.by_place = (unsigned)((P.n_parts ? 1 : 2) * warps);
  P.tail = (unsigned)((few ? kFewTail : kTail) * warps);
}

static const void *kernel_ptr(bool half, int mode) {
  if (half)
    return mode == kDebug      ? (const void *)render_kernel<__half, kDebug>
           : mode == kAnimated ? (const void *)render_kernel<__half, kAnimated>
                               : (const void *)render_kernel<__half, kPlain>;
  return mode == kDebug      ? (const void *)render_kernel<float, kDebug>
         : mode == kAnimated ? (const void *)render_kernel<float, kAnimated>
                             : (const void *)render_kernel<float, kPlain>;
}

static bh_status launch(bh_ctx *ctx, const bh_tables *t, RenderParams &P, bool debug, cudaStream_t s) {
  int threads = 32 * ctx->tuning.warps_per_block;
  size_t smem = P.u_bytes + 2 * sizeof(float4) * P.n_parts +
                (P.cams == nullptr && P.cam0.rgb ? sizeof(float) * 96 * ctx->tuning.warps_per_block : 0);
  int grid = render_grid(ctx, P.total_tiles);
  if (grid < 1) return BH_OK;
  set_schedule(ctx, P, grid, P.total_tiles);
  bool half = t->desc.storage == BH_F16;
  const void *f = kernel_ptr(half, debug ? kDebug : (P.n_parts > 0 ? kAnimated : kPlain));
  void *args[] = {&P};
  BH_CUDA(cudaLaunchKernel(f, dim3(grid), dim3(threads), args, smem, s));
  count_launch(ctx);
  BH_CUDA(cudaGetLastError());
  return BH_OK;
}

static bh_status render_one(bh_ctx *ctx, const bh_tables *t, const bh_cubemap *cube,
                            const bh_camera *cam, const bh_disc *disc, const bh_shading *sh,
                            float *out, float *dbg, cudaStream_t s, bool rgb = false) {
  if (!ctx || !t || !out) { set_error("bh_render: NULL argument"); return BH_ERR_INVALID_ARG; }
  if (((uintptr_t)out & 15) || (dbg && ((uintptr_t)dbg & 15))) {
    set_error("bh_render: output buffers must be 16-byte aligned");
    return BH_ERR_INVALID_ARG;
  }
  if (!validate_camera(cam, 0) || !validate_disc(disc)) return BH_ERR_INVALID_ARG;
  BH_CUDA(cudaSetDevice(ctx->device));
  RenderParams P;
  fill_params(ctx, t, cube, disc, sh, P);
  camera_constants(cam, &P.cam0);
  P.cam0.tiles_x = tiles_across(cam->width);
  P.cam0.inv_tiles_x = 1.f / (float)P.cam0.tiles_x;
  P.cam0.tile0 = 0;
  P.cam0.out = reinterpret_cast<float4 *>(out);
  P.cam0.dbg = dbg;
  P.cam0.rgb = rgb ? 1 : 0;
  P.cam0.rgb_vec = rgb && (cam->width % 4) == 0 ? 1 : 0;
  P.cams = nullptr;
  P.ncams = 1;
  P.total_tiles = warp_tiles(cam->width, cam->height);
  return launch(ctx, t, P, dbg != nullptr, s);
}

static bh_status ensure_cam_staging(bh_ctx *ctx, int n) {
  if (n <= ctx->cam_cap) return BH_OK;
  ctx->graph.reset();
  if (ctx->cam_host) cudaFreeHost(ctx->cam_host);
  if (ctx->cam_dev) cudaFree(ctx->cam_dev);
  ctx->cam_host = ctx->cam_dev = nullptr;
  ctx->cam_cap = 0;
  int cap = std::max(n, 64);
  BH_CUDA(cudaMallocHost(&ctx->cam_host, sizeof(CamConst) * cap));
  BH_CUDA(pool_malloc(*ctx->pool, &ctx->cam_dev, sizeof(CamConst) * cap));
  ctx->cam_cap = cap;
  return BH_OK;
}


bh_status render_batch_impl(bh_ctx *ctx, const bh_tables *t, const bh_cubemap *cube, int n,
                            const bh_camera *cams, const bh_disc *disc, const bh_shading *sh,
                            float *const *outs, cudaStream_t s, void *cam_host, void *cam_dev,
                            BatchGraph *bg) {
  RenderParams P;
  fill_params(ctx, t, cube, disc, sh, P);
  CamConst *h = static_cast<CamConst *>(cam_host);
  int tiles = 0;
  for (int k = 0; k < n; ++k) {
    camera_constants(&cams[k], &h[k]);
    h[k].tiles_x = tiles_across(cams[k].width);
    h[k].inv_tiles_x = 1.f / (float)h[k].tiles_x;
    h[k].tile0 = tiles;
    h[k].out = reinterpret_cast<float4 *>(outs[k]);
    h[k].dbg = nullptr;
    tiles += warp_tiles(cams[k].width, cams[k].height);
  }
  P.cams = static_cast<const CamConst *>(cam_dev);
  P.ncams = n;
  P.total_tiles = tiles;
  int threads = 32 * ctx->tuning.warps_per_block;
  size_t smem = P.u_bytes + 2 * sizeof(float4) * P.n_parts;
  int grid = render_grid(ctx, P.total_tiles);
  if (grid < 1) return BH_OK;
  set_schedule(ctx, P, grid, P.total_tiles);
  const void *func = kernel_ptr(t->desc.storage == BH_F16, P.n_parts > 0 ? kAnimated : kPlain);
  void *args[] = {&P};
  cudaKernelNodeParams kp = {};
  kp.func = const_cast<void *>(func);
  kp.gridDim = dim3(grid);
  kp.blockDim = dim3(threads);
  kp.sharedMemBytes = (unsigned)smem;
  kp.kernelParams = args;
  if (!bg->exec || bg->n != n || bg->func != func || bg->cam_dev != cam_dev || bg->block != threads) {
    bg->reset();
    BH_CUDA(cudaGraphCreate(&bg->graph, 0));
    BH_CUDA(cudaGraphAddMemcpyNode1D(&bg->copy, bg->graph, nullptr, 0, cam_dev, cam_host,
                                     sizeof(CamConst) * n, cudaMemcpyHostToDevice));
    BH_CUDA(cudaGraphAddKernelNode(&bg->kern, bg->graph, &bg->copy, 1, &kp));
    BH_CUDA(cudaGraphInstantiate(&bg->exec, bg->graph, 0));
    bg->n = n;
    bg->block = threads;
    bg->func = func;
    bg->cam_dev = cam_dev;
  } else {
    BH_CUDA(cudaGraphExecKernelNodeSetParams(bg->exec, bg->kern, &kp));
  }
  BH_CUDA(cudaGraphLaunch(bg->exec, s));
  count_launch(ctx);
  return BH_OK;
}

size_t cam_const_size() { return sizeof(CamConst); }


// ---------------------------------------------------------------------------
// Free-fall camera orbits (Appendix C), advanced and turned into camera
// constants on the device so that a viewer's trajectory never leaves HBM.
// ---------------------------------------------------------------------------

// Camera of an orbit state: position from r (cos chi cos psi, sin psi,
// sin chi cos psi); velocity wrt the static observer ((dr/dtau)/e, 0,
// l u sqrt(1-u)/e) on (e_r, e_chi, e_psi); e_chi = a e_theta + b e_phi,
// e_psi = -b e_theta + a e_phi with e_chi = e_psi ^ e_r (reading C22).
__host__ __device__ static void orbit_to_camera(const bh_orbit *o, bh_camera *c) {
  double th = acos(cos(o->psi) * sin(o->chi));
  double ph = atan2(sin(o->psi), cos(o->chi) * cos(o->psi));
  double u = 1.0 / o->r;
  double a = sin(o->chi) * cos(th) * cos(ph) + cos(o->chi) * sin(th);
  double b = -sin(o->chi) * sin(ph);
  double vpsi = o->l * u * sqrt(1.0 - u) / o->e;
  c->r = o->r;
  c->theta = th;
  c->phi = ph;
  c->v[0] = o->rdot / o->e;
  c->v[1] = -b * vpsi;
  c->v[2] = a * vpsi;
  for (int i = 0; i < 3; ++i) {
    const double *Or = o->orient + 3 * i;  // on (r', chi', psi')
    c->orient[3 * i + 0] = Or[0];
    c->orient[3 * i + 1] = a * Or[1] - b * Or[2];
    c->orient[3 * i + 2] = b * Or[1] + a * Or[2];
  }
  c->fov_y = o->fov_y;
  c->width = o->width;
  c->height = o->height;
}

// The camera constants of an orbit state on the device, straight from the
// position's direction (cos chi cos psi, sin psi, sin chi cos psi): the chain of
// acos, atan2 and their sines again took half of a set-up that nothing overlaps
// (one thread per orbit, FP64 latency).
__device__ static void orbit_constants(const bh_orbit &o, int width, int height, float *out, CamConst *k) {
  double sp, cp, sc, cc;
  sincos(o.psi, &sp, &cp);
  sincos(o.chi, &sc, &cc);
  const double rx = cc * cp, ry = sp, ct = sc * cp, st = sqrt(fma(rx, rx, ry * ry));
  const double ist = st > 0.0 ? 1.0 / st : 0.0;
  const double cph = st > 0.0 ? rx * ist : 1.0, sph = ry * ist;
  const double u = 1.0 / o.r, a = sc * ct * cph + cc * st, b = -sc * sph;
  const double ie = 1.0 / o.e, vpsi = o.l * u * sqrt(1.0 - u) * ie;
  bh_camera c;
  c.r = o.r;
  c.v[0] = o.rdot * ie;
  c.v[1] = -b * vpsi;
  c.v[2] = a * vpsi;
  for (int i = 0; i < 3; ++i) {
    const double *Or = o.orient + 3 * i;  // on (r', chi', psi')
    c.orient[3 * i + 0] = Or[0];
    c.orient[3 * i + 1] = a * Or[1] - b * Or[2];
    c.orient[3 * i + 2] = b * Or[1] + a * Or[2];
  }
  c.fov_y = o.fov_y;
  c.width = width;
  c.height = height;
  camera_constants_at(&c, st, ct, sph, cph, k);
  k->tiles_x = (width + 7) / 8;  // 8 x 4 pixel warp tiles
  k->inv_tiles_x = 1.f / (float)k->tiles_x;
  k->out = reinterpret_cast<float4 *>(out);
  k->dbg = nullptr;
}

// First tile of every camera from the cameras' tile counts (shared memory), by
// the first warp.
__device__ static void tile_offsets(const int *tiles, int n, CamConst *cams, int *total_tiles) {
  if (threadIdx.x >= 32) return;
  int base = 0;
  for (int k0 = 0; k0 < n; k0 += 32) {
    const int k = k0 + (int)threadIdx.x, t = k < n ? tiles[k] : 0;
    int sum = t;
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, sum, o);
      if ((int)threadIdx.x >= o) sum += v;
    }
    if (k < n) cams[k].tile0 = base + sum - t;
    base += __shfl_sync(0xffffffffu, sum, 31);
  }
  if (threadIdx.x == 0) *total_tiles = base;
}

// d^2r/dtau^2 = (2 l^2 u^3 - 3 l^2 u^4 - u^2)/2, dpsi/dtau = l u^2,
// dt/dtau = e/(1-u): RK4 in proper time, FP64, one thread per orbit.  An orbit
// that would reach r <= 1.05 stops there (no static observer inside the
// horizon, Sec. 5).  Bound by the latency of one chain, 4 x steps evaluations
// long, so each is kept short: reciprocals by Newton's iteration from the
// single-precision one (2^-23, 2^-46, then rounding), u^2 (l^2 u (2 - 3 u) - 1)/2.
__device__ __forceinline__ double orbit_rcp(double x) {
  if (!(fabs(x) > 1e-30 && fabs(x) < 1e30)) return 1.0 / x;
  double r = (double)__frcp_rn((float)x);
  r = fma(r, fma(-x, r, 1.0), r);
  return fma(r, fma(-x, r, 1.0), r);
}

__device__ __forceinline__ static void orbit_rhs(const bh_orbit &o, double l2, const double *y, double *dy) {
  const double u = orbit_rcp(y[1]), u2 = u * u;
  dy[0] = o.e * orbit_rcp(1.0 - u);
  dy[1] = y[3];
  dy[2] = o.l * u2;
  dy[3] = 0.5 * u2 * fma(l2 * u, fma(-3.0, u, 2.0), -1.0);
}

__device__ static void orbit_advance_one(bh_orbit &o, double dtau, int steps) {
  const double h = dtau / steps, l2 = o.l * o.l, h6 = h / 6.0;
  for (int s = 0; s < steps; ++s) {
    double y[4] = {o.t, o.r, o.psi, o.rdot}, k1[4], k2[4], k3[4], k4[4], z[4];
    orbit_rhs(o, l2, y, k1);
    for (int a = 0; a < 4; ++a) z[a] = fma(0.5 * h, k1[a], y[a]);
    orbit_rhs(o, l2, z, k2);
    for (int a = 0; a < 4; ++a) z[a] = fma(0.5 * h, k2[a], y[a]);
    orbit_rhs(o, l2, z, k3);
    for (int a = 0; a < 4; ++a) z[a] = fma(h, k3[a], y[a]);
    orbit_rhs(o, l2, z, k4);
    double next[4];
    for (int a = 0; a < 4; ++a) next[a] = fma(h6, (k1[a] + k4[a]) + 2.0 * (k2[a] + k3[a]), y[a]);
    if (!(next[1] > 1.05)) break;
    o.t = next[0];
    o.r = next[1];
    o.psi = next[2];
    o.rdot = next[3];
  }
}

__global__ void orbit_advance_kernel(bh_orbit *orbits, int n, double dtau, int steps) {
  int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  bh_orbit o = orbits[k];
  orbit_advance_one(o, dtau, steps);
  orbits[k] = o;
}

// Served viewers on device-resident orbits: advance each request's orbit
// (its own, in place), then its camera constants at the request's image size,
// then the tile offsets -- one block, ahead of the render launch.
__global__ void serve_orbit_setup_kernel(const OrbitJob *jobs, int n, CamConst *cams, int *total_tiles) {
  __shared__ int tiles[kMaxOrbits];
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    const OrbitJob j = jobs[k];
    bh_orbit o = *j.orbit;
    if (j.steps > 0) {
      orbit_advance_one(o, j.dtau, j.steps);
      *j.orbit = o;
    }
    orbit_constants(o, j.width, j.height, j.out, &cams[k]);
    tiles[k] = warp_tiles(j.width, j.height);
  }
  __syncthreads();
  tile_offsets(tiles, n, cams, total_tiles);
}

// Camera constants of every orbit (one block), then the tile offsets -- the
// same layout bh_render_batch stages from the host.  The output addresses are a
// kernel parameter: no staging buffer that a call would have to wait for.
template <int N>
struct OrbitOuts {
  float *p[N];
};

template <int N>
__global__ void orbit_camconst_kernel(const bh_orbit *orbits, int n, const OrbitOuts<N> outs, CamConst *cams,
                                      int *total_tiles) {
  __shared__ int tiles[N];
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    const bh_orbit o = orbits[k];
    orbit_constants(o, o.width, o.height, outs.p[k], &cams[k]);
    tiles[k] = warp_tiles(o.width, o.height);
  }
  __syncthreads();
  tile_offsets(tiles, n, cams, total_tiles);
}

// One served batch of orbit requests: jobs staged in pinned memory are
// copied, set up on the device and rendered in one persistent launch.
bh_status render_orbit_jobs(bh_ctx *ctx, const bh_tables *t, const bh_cubemap *cube, int n,
                            const OrbitJob *jobs_host, OrbitJob *jobs_dev, void *cams_dev, int *total_dev,
                            const bh_disc *disc, const bh_shading *sh, cudaStream_t s) {
  BH_CUDA(cudaMemcpyAsync(jobs_dev, jobs_host, sizeof(OrbitJob) * n, cudaMemcpyHostToDevice, s));
  CamConst *cams = static_cast<CamConst *>(cams_dev);
  serve_orbit_setup_kernel<<<1, 256, 0, s>>>(jobs_dev, n, cams, total_dev);
  count_launch(ctx);
  RenderParams P;
  fill_params(ctx, t, cube, disc, sh, P);
  P.cams = cams;
  P.ncams = n;
  P.total_tiles = 0;
  P.total_tiles_dev = total_dev;
  int threads = 32 * ctx->tuning.warps_per_block;
  size_t smem = P.u_bytes + 2 * sizeof(float4) * P.n_parts;
  int grid = ctx->sm_count * ctx->tuning.blocks_per_sm;
  long long tiles = 0;
  for (int k = 0; k < n; ++k) tiles += warp_tiles(jobs_host[k].width, jobs_host[k].height);
  set_schedule(ctx, P, grid, tiles);
  void *args[] = {&P};
  const void *f = kernel_ptr(t->desc.storage == BH_F16, P.n_parts > 0 ? kAnimated : kPlain);
  BH_CUDA(cudaLaunchKernel(f, dim3(grid), dim3(threads), args, smem, s));
  count_launch(ctx);
  BH_CUDA(cudaGetLastError());
  return BH_OK;
}

bool validate_disc_ext(const bh_disc *d) { return validate_disc(d); }

bh_status validate_batch(int n, const bh_camera *cams, const bh_disc *disc, float *const *outs) {
  if (n < 1 || !cams || !outs) { set_error("batch: n >= 1 cameras and outputs required"); return BH_ERR_INVALID_ARG; }
  for (int k = 0; k < n; ++k) {
    if (!validate_camera(&cams[k], k)) return BH_ERR_INVALID_ARG;
    if (!outs[k] || ((uintptr_t)outs[k] & 15)) {
      set_error("batch: output %d is NULL or not 16-byte aligned", k);
      return BH_ERR_INVALID_ARG;
    }
  }
  if (!validate_disc(disc)) return BH_ERR_INVALID_ARG;
  return BH_OK;
}

}  // namespace bh

using namespace bh;

extern "C" bh_status bh_render(bh_ctx *ctx, const bh_tables *t, const bh_cubemap *cube,
                               const bh_camera *cam, const bh_disc *disc, const bh_shading *sh,
                               float *out, void *stream) {
  TraceRange trace_("bh_render");
  return render_one(ctx, t, cube, cam, disc, sh, out, nullptr, (cudaStream_t)stream);
}

extern "C" bh_status bh_render_debug(bh_ctx *ctx, const bh_tables *t, const bh_cubemap *cube,
                                     const bh_camera *cam, const bh_disc *disc,
                                     const bh_shading *sh, float *out, float *dbg, void *stream) {
  TraceRange trace_("bh_render_debug");
  if (!dbg) { set_error("bh_render_debug: dbg is NULL"); return BH_ERR_INVALID_ARG; }
  return render_one(ctx, t, cube, cam, disc, sh, out, dbg, (cudaStream_t)stream);
}

static bh_status render_to_host(bh_ctx *ctx, const bh_tables *t, const bh_cubemap *cube,
                                const bh_camera *cam, const bh_disc *disc, const bh_shading *sh,
                                float *host, void *stream, bool rgb) {
  if (!ctx || !host || !cam) { set_error("bh_render_to_host: NULL argument"); return BH_ERR_INVALID_ARG; }
  if (!validate_camera(cam, 0)) return BH_ERR_INVALID_ARG;
  BH_CUDA(cudaSetDevice(ctx->device));
  cudaStream_t s = (cudaStream_t)stream;
  size_t bytes = (rgb ? 3 * sizeof(float) : sizeof(float4)) * (size_t)cam->width * cam->height;
  // Pinned host memory the device can address (cudaHostAlloc, cudaHostRegister;
  // all pinned memory under unified addressing): the kernel stores the image
  // straight into it over the host link, overlapping the transfer with the
  // rendering.  (Rendering into device memory in row bands, each copied by the
  // copy engine while the next renders, measured slower: 4,497 against 4,816
  // packed-RGB 1080p frames/s.)
  cudaPointerAttributes pa;
  if (cudaPointerGetAttributes(&pa, host) == cudaSuccess && pa.type == cudaMemoryTypeHost && pa.devicePointer &&
      ((uintptr_t)pa.devicePointer & 15) == 0) {
    bh_status st = render_one(ctx, t, cube, cam, disc, sh, static_cast<float *>(pa.devicePointer), nullptr, s, rgb);
    if (st) return st;
    BH_CUDA(cudaStreamSynchronize(s));
    return BH_OK;
  }
  cudaGetLastError();  // pageable memory: cudaPointerGetAttributes may have set an error
  std::lock_guard<std::mutex> lk(ctx->mu);
  if (bytes > ctx->frame_cap) {
    BH_CUDA(cudaStreamSynchronize(s));
    if (ctx->frame_dev) cudaFree(ctx->frame_dev);
    ctx->frame_dev = nullptr;
    ctx->frame_cap = 0;
    BH_CUDA(pool_malloc(*ctx->pool, (void **)&ctx->frame_dev, bytes));
    ctx->frame_cap = bytes;
  }
  bh_status st = render_one(ctx, t, cube, cam, disc, sh, ctx->frame_dev, nullptr, s, rgb);
  if (st) return st;
  BH_CUDA(cudaMemcpyAsync(host, ctx->frame_dev, bytes, cudaMemcpyDeviceToHost, s));
  BH_CUDA(cudaStreamSynchronize(s));
  return BH_OK;
}

// Frames in flight: frame n renders into device slot n % 2 on the caller's
// stream, then the copy engine moves it to the host on the context's copy
// stream while frame n + 1 renders into the other slot.  A slot is rendered
// into again only after its previous copy has finished (the stream waits on
// that copy's event), so at most two frames are in flight and the rendering
// of one overlaps the transfer of the other.
static bh_status render_to_host_async(bh_ctx *ctx, const bh_tables *t, const bh_cubemap *cube,
                                      const bh_camera *cam, const bh_disc *disc, const bh_shading *sh,
                                      float *host, void *stream, bool rgb, unsigned long long *ticket) {
  if (!ctx || !host || !cam || !ticket) {
    set_error("bh_render_to_host_async: NULL argument");
    return BH_ERR_INVALID_ARG;
  }
  if (!validate_camera(cam, 0)) return BH_ERR_INVALID_ARG;
  BH_CUDA(cudaSetDevice(ctx->device));
  cudaStream_t s = (cudaStream_t)stream;
  cudaPointerAttributes pa;
  const bool pinned = cudaPointerGetAttributes(&pa, host) == cudaSuccess && pa.type == cudaMemoryTypeHost;
  cudaGetLastError();  // pageable memory: cudaPointerGetAttributes may have set an error
  if (!pinned) {
    set_error("bh_render_to_host_async: the host buffer must be pinned (cudaHostAlloc or cudaHostRegister)");
    return BH_ERR_INVALID_ARG;
  }
  const size_t bytes = (rgb ? 3 * sizeof(float) : sizeof(float4)) * (size_t)cam->width * cam->height;
  std::lock_guard<std::mutex> lk(ctx->mu);
  if (!ctx->ring_copy) {
    BH_CUDA(cudaStreamCreateWithFlags(&ctx->ring_copy, cudaStreamNonBlocking));
    for (int k = 0; k < 2; ++k) {
      BH_CUDA(cudaEventCreateWithFlags(&ctx->ring_ready[k], cudaEventDisableTiming));
      BH_CUDA(cudaEventCreateWithFlags(&ctx->ring_done[k], cudaEventDisableTiming));
    }
  }
  if (bytes > ctx->ring_cap) {
    // every earlier copy has finished, and with it the render it waited for
    BH_CUDA(cudaStreamSynchronize(ctx->ring_copy));
    for (int k = 0; k < 2; ++k) {
      if (ctx->ring_dev[k]) cudaFree(ctx->ring_dev[k]);
      ctx->ring_dev[k] = nullptr;
    }
    ctx->ring_cap = 0;
    for (int k = 0; k < 2; ++k) BH_CUDA(pool_malloc(*ctx->pool, (void **)&ctx->ring_dev[k], bytes));
    ctx->ring_cap = bytes;
  }
  const int k = (int)(ctx->ring_seq & 1u);
  // the slot's previous frame must have left the device before it is
  // overwritten (a no-op before the slot's first copy)
  BH_CUDA(cudaStreamWaitEvent(s, ctx->ring_done[k], 0));
  bh_status st = render_one(ctx, t, cube, cam, disc, sh, ctx->ring_dev[k], nullptr, s, rgb);
  if (st) return st;
  BH_CUDA(cudaEventRecord(ctx->ring_ready[k], s));
  BH_CUDA(cudaStreamWaitEvent(ctx->ring_copy, ctx->ring_ready[k], 0));
  BH_CUDA(cudaMemcpyAsync(host, ctx->ring_dev[k], bytes, cudaMemcpyDeviceToHost, ctx->ring_copy));
  BH_CUDA(cudaEventRecord(ctx->ring_done[k], ctx->ring_copy));
  *ticket = ctx->ring_seq++;
  return BH_OK;
}

extern "C" bh_status bh_render_to_host_async(bh_ctx *ctx, const bh_tables *t, const bh_cubemap *cube,
                                             const bh_camera *cam, const bh_disc *disc,
                                             const bh_shading *sh, float *host, int rgb, void *stream,
                                             unsigned long long *ticket) {
  TraceRange trace_("bh_render_to_host_async");
  if (rgb != 0 && rgb != 1) {
    set_error("bh_render_to_host_async: rgb = %d, must be 0 (RGBA) or 1 (packed RGB)", rgb);
    return BH_ERR_INVALID_ARG;
  }
  return render_to_host_async(ctx, t, cube, cam, disc, sh, host, stream, rgb == 1, ticket);
}

extern "C" bh_status bh_host_wait(bh_ctx *ctx, unsigned long long ticket) {
  TraceRange trace_("bh_host_wait");
  if (!ctx) { set_error("bh_host_wait: NULL context"); return BH_ERR_INVALID_ARG; }
  cudaEvent_t e;
  {
    std::lock_guard<std::mutex> lk(ctx->mu);
    if (ticket >= ctx->ring_seq) {
      set_error("bh_host_wait: ticket %llu was never issued (%llu issued)", ticket, ctx->ring_seq);
      return BH_ERR_INVALID_ARG;
    }
    // the slot's event belongs to this frame or to a later one; copies run in
    // order on one stream, so either has finished only after this frame's
    e = ctx->ring_done[ticket & 1u];
  }
  BH_CUDA(cudaSetDevice(ctx->device));
  BH_CUDA(cudaEventSynchronize(e));
  return BH_OK;
}

extern "C" bh_status bh_render_to_host(bh_ctx *ctx, const bh_tables *t, const bh_cubemap *cube,
                                       const bh_camera *cam, const bh_disc *disc,
                                       const bh_shading *sh, float *host, void *stream) {
  TraceRange trace_("bh_render_to_host");
  return render_to_host(ctx, t, cube, cam, disc, sh, host, stream, false);
}

extern "C" bh_status bh_render_to_host_rgb(bh_ctx *ctx, const bh_tables *t, const bh_cubemap *cube,
                                           const bh_camera *cam, const bh_disc *disc,
                                           const bh_shading *sh, float *host_rgb, void *stream) {
  TraceRange trace_("bh_render_to_host_rgb");
  return render_to_host(ctx, t, cube, cam, disc, sh, host_rgb, stream, true);
}

extern "C" bh_status bh_render_batch(bh_ctx *ctx, const bh_tables *t, const bh_cubemap *cube, int n,
                                     const bh_camera *cams, const bh_disc *disc,
                                     const bh_shading *sh, float *const *outs, void *stream) {
  TraceRange trace_("bh_render_batch");
  if (!ctx || !t) { set_error("bh_render_batch: NULL argument"); return BH_ERR_INVALID_ARG; }
  bh_status st = validate_batch(n, cams, disc, outs);
  if (st) return st;
  BH_CUDA(cudaSetDevice(ctx->device));
  cudaStream_t s = (cudaStream_t)stream;
  std::lock_guard<std::mutex> lk(ctx->mu);
  // the staging buffer is reused: wait until the previous copy out of it ran
  BH_CUDA(cudaStreamSynchronize(s));
  st = ensure_cam_staging(ctx, n);
  if (st) return st;
  return render_batch_impl(ctx, t, cube, n, cams, disc, sh, outs, s, ctx->cam_host, ctx->cam_dev,
                           &ctx->graph);
}

extern "C" bh_status bh_autotune_batch(bh_ctx *ctx, const bh_tables *t, const bh_cubemap *cube,
                                       int n, const bh_camera *cams, const bh_disc *disc,
                                       const bh_shading *sh, float *const *outs, int *chosen) {
  TraceRange trace_("bh_autotune_batch");
  if (!ctx || !t) { set_error("bh_autotune_batch: NULL argument"); return BH_ERR_INVALID_ARG; }
  bh_status st = validate_batch(n, cams, disc, outs);
  if (st) return st;
  BH_CUDA(cudaSetDevice(ctx->device));
  // Candidates: warps per block, warp tiles per fetch, resident blocks per SM.  All
  // have the 32 warps per SM that fit at 64 registers: of a larger grid the last
  // blocks, whose first tiles are theirs by their place in it, would start when
  // the others leave.
  static const RenderTuning cand[] = {{8, 1, 4}, {8, 2, 4}, {8, 4, 4}, {8, 8, 4},
                                      {4, 1, 8}, {4, 2, 8}, {4, 4, 8}, {8, 16, 4}};
  const int nc = sizeof(cand) / sizeof(cand[0]);
  cudaStream_t s;
  BH_CUDA(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  RenderTuning keep = ctx->tuning;
  int best = -1;
  float best_ms = 1e30f;
  // Each timed run starts from a cold L2, as a frame does after other work:
  // a scratch buffer of twice the L2 size is cleared before it (outside the
  // timed span).  Without the memory for it the runs are timed warm.
  int l2 = 0;
  cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, ctx->device);
  const size_t flush_bytes = 2 * (size_t)std::max(l2, 0);
  void *flush = nullptr;
  if (flush_bytes && pool_malloc(*ctx->pool, &flush, flush_bytes) != cudaSuccess) {
    flush = nullptr;
    cudaGetLastError();
  }
  constexpr int kReps = 7;  // the first run of a candidate builds its graph and is not timed
  std::lock_guard<std::mutex> lk(ctx->mu);
  st = ensure_cam_staging(ctx, n);
  for (int c = 0; c < nc && st == BH_OK; ++c) {
    ctx->tuning = cand[c];
    float ms[kReps - 1];
    for (int rep = 0; rep < kReps && st == BH_OK; ++rep) {
      if (flush) cudaMemsetAsync(flush, rep & 0xff, flush_bytes, s);
      cudaEventRecord(e0, s);
      st = render_batch_impl(ctx, t, cube, n, cams, disc, sh, outs, s, ctx->cam_host, ctx->cam_dev,
                             &ctx->graph);
      cudaEventRecord(e1, s);
      cudaEventSynchronize(e1);
      float m = 0.f;
      cudaEventElapsedTime(&m, e0, e1);
      if (rep > 0) ms[rep - 1] = m;
    }
    if (st != BH_OK) break;
    std::sort(ms, ms + kReps - 1);
    const float med = 0.5f * (ms[(kReps - 1) / 2 - 1] + ms[(kReps - 1) / 2]);
    if (med < best_ms) { best_ms = med; best = c; }
  }
  if (flush) cudaFree(flush);
  ctx->tuning = best >= 0 ? cand[best] : keep;
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaStreamDestroy(s);
  if (chosen) *chosen = best;
  return st;
}

extern "C" bh_status bh_orbit_init(double r0, double delta0, double v0, double chi, const double *orient,
                                   double fov_y, int width, int height, bh_orbit *out) {
  if (!out) { set_error("bh_orbit_init: out is NULL"); return BH_ERR_INVALID_ARG; }
  if (!(r0 > 1.05) || !(v0 >= 0.0 && v0 < 1.0) || !(delta0 > 0.0 && delta0 < kPi)) {
    set_error("bh_orbit_init: need r0 > 1.05, 0 <= v0 < 1, 0 < delta0 < pi");
    return BH_ERR_INVALID_ARG;
  }
  memset(out, 0, sizeof *out);
  double u = 1.0 / r0;
  double e2 = (1.0 - u) / (1.0 - v0 * v0);  // gamma = e / sqrt(1 - u)
  double cot = cos(delta0) / sin(delta0);     // tan(delta) = r dpsi/dr
  double l2 = (e2 + u - 1.0) / (u * u * (1.0 - u + cot * cot));
  out->r = r0;
  out->chi = chi;
  out->e = sqrt(e2);
  out->l = sqrt(l2 > 0.0 ? l2 : 0.0);
  double rd2 = e2 + l2 * u * u * u - l2 * u * u + u - 1.0;
  out->rdot = (delta0 < 0.5 * kPi ? 1.0 : -1.0) * sqrt(rd2 > 0.0 ? rd2 : 0.0);
  const double eye[9] = {1, 0, 0, 0, 1, 0, 0, 0, 1};
  for (int k = 0; k < 9; ++k) out->orient[k] = orient ? orient[k] : eye[k];
  out->fov_y = fov_y;
  out->width = width;
  out->height = height;
  bh_camera c;
  orbit_to_camera(out, &c);
  return validate_camera(&c, 0) ? BH_OK : BH_ERR_INVALID_ARG;
}

extern "C" bh_status bh_orbit_camera(const bh_orbit *o, bh_camera *out) {
  if (!o || !out) { set_error("bh_orbit_camera: NULL argument"); return BH_ERR_INVALID_ARG; }
  orbit_to_camera(o, out);
  return BH_OK;
}

extern "C" bh_status bh_orbits_advance(bh_ctx *ctx, bh_orbit *orbits_device, int n, double dtau, int steps,
                                       void *stream) {
  TraceRange trace_("bh_orbits_advance");
  if (!ctx || (n > 0 && !orbits_device) || n < 0 || steps < 1) {
    set_error("bh_orbits_advance: bad argument");
    return BH_ERR_INVALID_ARG;
  }
  if (n == 0) return BH_OK;
  BH_CUDA(cudaSetDevice(ctx->device));
  orbit_advance_kernel<<<(n + 127) / 128, 128, 0, (cudaStream_t)stream>>>(orbits_device, n, dtau, steps);
  count_launch(ctx);
  BH_CUDA(cudaGetLastError());
  return BH_OK;
}

extern "C" bh_status bh_render_orbits(bh_ctx *ctx, const bh_tables *t, const bh_cubemap *cube, int n,
                                      const bh_orbit *orbits_device, const bh_disc *disc,
                                      const bh_shading *sh, float *const *outs, void *stream) {
  TraceRange trace_("bh_render_orbits");
  if (!ctx || !t || !orbits_device || !outs || n < 1 || n > kMaxOrbits) {
    set_error("bh_render_orbits: bad argument (1 <= n <= 1024)");
    return BH_ERR_INVALID_ARG;
  }
  for (int k = 0; k < n; ++k)
    if (!outs[k] || ((uintptr_t)outs[k] & 15)) {
      set_error("bh_render_orbits: output %d is NULL or not 16-byte aligned", k);
      return BH_ERR_INVALID_ARG;
    }
  if (!validate_disc(disc)) return BH_ERR_INVALID_ARG;
  BH_CUDA(cudaSetDevice(ctx->device));
  cudaStream_t s = (cudaStream_t)stream;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  BH_CUDA(cudaStreamIsCapturing(s, &cap));
  if (cap != cudaStreamCaptureStatusNone) {
    set_error("bh_render_orbits: the stream is being captured");
    return BH_ERR_CUDA;
  }
  std::lock_guard<std::mutex> lk(ctx->mu);
  if (!ctx->orb_done) BH_CUDA(cudaEventCreateWithFlags(&ctx->orb_done, cudaEventDisableTiming));
  if (!ctx->orb_cams_dev) BH_CUDA(pool_malloc(*ctx->pool, &ctx->orb_cams_dev, sizeof(CamConst) * kMaxOrbits + 16));
  // the last call's launch may still read the constants, on another stream
  BH_CUDA(cudaStreamWaitEvent(s, ctx->orb_done, 0));
  RenderParams P;
  fill_params(ctx, t, cube, disc, sh, P);
  CamConst *cams = static_cast<CamConst *>(ctx->orb_cams_dev);
  int *total_dev = reinterpret_cast<int *>(cams + kMaxOrbits);
  const int setup_threads = std::min((n + 31) / 32 * 32, 256);
  if (n <= 64) {
    OrbitOuts<64> o = {};
    for (int k = 0; k < n; ++k) o.p[k] = outs[k];
    orbit_camconst_kernel<64><<<1, setup_threads, 0, s>>>(orbits_device, n, o, cams, total_dev);
  } else {
    OrbitOuts<kMaxOrbits> o = {};
    for (int k = 0; k < n; ++k) o.p[k] = outs[k];
    orbit_camconst_kernel<kMaxOrbits><<<1, setup_threads, 0, s>>>(orbits_device, n, o, cams, total_dev);
  }
  count_launch(ctx);
  P.cams = cams;
  P.ncams = n;
  P.total_tiles = 0;
  P.total_tiles_dev = total_dev;
  int threads = 32 * ctx->tuning.warps_per_block;
  size_t smem = P.u_bytes + 2 * sizeof(float4) * P.n_parts;
  int grid = ctx->sm_count * ctx->tuning.blocks_per_sm;
  // Only the device knows the sizes: taken as 640 x 360.  Chunks of two cost 16 frames
  // of 1080p 1.2 %, chunks of four as many of 640 x 360 2 % and, in an animated
  // disc, one of 1080p a third.
  set_schedule(ctx, P, grid, (long long)n * warp_tiles(640, 360));
  void *args[] = {&P};
  const void *f = kernel_ptr(t->desc.storage == BH_F16, P.n_parts > 0 ? kAnimated : kPlain);
  BH_CUDA(cudaLaunchKernel(f, dim3(grid), dim3(threads), args, smem, s));
  count_launch(ctx);
  BH_CUDA(cudaGetLastError());
  BH_CUDA(cudaEventRecord(ctx->orb_done, s));
  return BH_OK;
}

extern "C" bh_status bh_inject_fault(bh_ctx *ctx, int kind) {
  if (!ctx) { set_error("bh_inject_fault: NULL context"); return BH_ERR_INVALID_ARG; }
  if (kind == BH_FAULT_TABLE_WAIT) ctx->inject_table_wait = 1;
  else if (kind == BH_FAULT_BLOOM_BARRIER) ctx->inject_bloom_barrier = 1;
  else { set_error("bh_inject_fault: unknown kind %d", kind); return BH_ERR_INVALID_ARG; }
  return BH_OK;
}

extern "C" bh_status bh_check_status(bh_ctx *ctx, void *stream) {
  if (!ctx) { set_error("bh_check_status: NULL context"); return BH_ERR_INVALID_ARG; }
  BH_CUDA(cudaSetDevice(ctx->device));
  return check_status(ctx, (cudaStream_t)stream);
}
