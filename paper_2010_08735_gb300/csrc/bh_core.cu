// libbh core: context, errors, and the GPU precompute of the tables.
//
//  * D(e,u) and U(e,phi) (Algorithm 1 PRECOMPUTE, Appendix A): instead of
//    Euler steps along each e row, FP64 quadrature of the ray equation's first
//    integral
//        phi(u) = int_0^u du' / sqrt(P(u')),  P(u) = e^2 - u^2 (1 - u)
//    (Eq. rayequation), in a variable without the apsis singularity and fine
//    enough for the near-double root at the photon sphere:
//      e^2 < mu:  P = (u_a - u) q(u), u = u_a - w^2, q = A + B w^2 - w^4;
//      e^2 > mu:  P = (e^2 - mu) + v^2 (v + 1), v = u - 2/3 = z |z|
//    (D, whose texels are equal steps of w and of z), or w = sqrt(A/B) sinh t and
//    v = sqrt(e^2-mu) sinh t (U, any e).  One block takes an e: every step
//    between texels is one four-node Gauss-Legendre panel, a block scan gives
//    the integrals up to every texel.  Delta = phi - atan2(u, du/dphi)
//    (Algorithm 1) is integrated directly: with u'' = -u + 3/2 u^2 (the ray
//    equation), dDelta/dphi = (3/2) u^3 / (e^2 + u^3).  U inverts phi(u) by
//    Newton steps inside a panel, using the apsis reflection phi -> 2 phi_a - phi
//    past the apsis (Sec. 3.3.1).
//    GB300 does two FP64 multiply-adds per SM and clock, so the number of
//    integrand values decides: one quadrature from infinity per texel took 64 to
//    160 of them twice (6.05 ms for 512 x 512; U by up to 80 Newton steps of
//    whole quadratures 0.99 ms); this takes four per texel: 145 us for both, of
//    which FP64 is busy 120.  Largest errors at 512 x 512 against quadratures
//    with 128 nodes: 1.7e-13 on Delta (before: 2.0e-12), 6e-13 on R (4.4e-12),
//    1.0e-15 on u (1.1e-15), 1.1e-12 on U's R (1.6e-12).
//  * The colour tables (Sec. 3.4.2): C(xy, D) and the disc black-body table.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>

#include "bh_colour.cuh"
#include "bh_internal.cuh"

namespace bh {

static thread_local std::string g_last_error;

void set_error(const char *fmt, ...) {
  char buf[1024];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  g_last_error = buf;
}

bh_status cuda_fail(cudaError_t e, const char *what) {
  set_error("%s: %s", what, cudaGetErrorString(e));
  return e == cudaErrorMemoryAllocation ? BH_ERR_OOM : BH_ERR_CUDA;
}

void count_launch(bh_ctx *ctx, int n) { ctx->launches.fetch_add(n, std::memory_order_relaxed); }

static void pool_release(Pool &pool) {  // pool.mu held
  for (PoolBlock &b : pool.kept) {
    if (b.ready) {
      cudaEventSynchronize(b.ready);
      cudaEventDestroy(b.ready);
    }
    cudaFree(b.p);
    pool.bytes -= b.bytes;
  }
  pool.kept.clear();
  for (HeldBlock &h : pool.held) {
    if (cudaFree(h.b.p) != cudaSuccess) cudaGetLastError();  // waits for the device
    pool.bytes -= h.b.bytes;
  }
  pool.held.clear();
}

// An allocation, made again without the kept memory where it fails.  pool.mu held.
template <typename Allocate>
static cudaError_t pool_allocate(Pool &pool, const Allocate &allocate) {
  cudaError_t e = allocate();
  if (e == cudaErrorMemoryAllocation && !(pool.kept.empty() && pool.held.empty())) {
    cudaGetLastError();
    pool_release(pool);
    // the stream-ordered allocator gives its free memory back at the next
    // synchronisation only
    cudaMemPool_t ordered;
    if (cudaDeviceGetDefaultMemPool(&ordered, pool.device) == cudaSuccess) cudaMemPoolTrimTo(ordered, 0);
    e = allocate();
  }
  return e;
}

cudaError_t pool_malloc(Pool &pool, void **p, size_t bytes) {
  std::lock_guard<std::mutex> lk(pool.mu);
  return pool_allocate(pool, [&] { return cudaMalloc(p, bytes); });
}

cudaError_t pool_get(Pool &pool, size_t bytes, cudaStream_t s, PoolBlock *out, bool scratch) {
  // Under stream capture nothing is taken from the pool (a block's event lies
  // outside the capture) or put into it: a handle's memory is allocated, which
  // only a relaxed capture allows, and scratch belongs to the graph.
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  const cudaError_t ce = cudaStreamIsCapturing(s, &cap);
  if (ce != cudaSuccess) return ce;
  if (cap != cudaStreamCaptureStatusNone) {
    PoolBlock b;
    b.bytes = scratch ? 0 : bytes;  // 0: freed on its stream
    const cudaError_t e = scratch ? cudaMallocAsync(&b.p, bytes, s) : cudaMalloc(&b.p, bytes);
    if (e == cudaSuccess) *out = b;
    return e;
  }
  std::lock_guard<std::mutex> lk(pool.mu);
  int best = -1;  // the smallest that fits and wastes less than its half
  for (int k = 0; k < (int)pool.kept.size(); ++k) {
    const size_t have = pool.kept[k].bytes;
    if (have >= bytes && have / 2 <= bytes && (best < 0 || have < pool.kept[best].bytes)) best = k;
  }
  if (best >= 0) {
    PoolBlock b = pool.kept[best];
    if (b.ready) {
      const cudaError_t e = cudaStreamWaitEvent(s, b.ready, 0);
      if (e != cudaSuccess) return e;
      cudaEventDestroy(b.ready);  // takes effect once the event has completed
      b.ready = nullptr;
    }
    pool.kept.erase(pool.kept.begin() + best);
    pool.bytes -= b.bytes;
    if (scratch) pool.lent += b.bytes;
    *out = b;
    return cudaSuccess;
  }
  // Scratch that there will be room to keep; other scratch is freed behind its
  // stream's work, where a cudaFree would make the caller wait for it.
  const bool keep = scratch && pool.bytes + pool.lent + bytes <= kPoolBytes;
  PoolBlock b;
  b.bytes = scratch && !keep ? 0 : bytes;
  const cudaError_t e = pool_allocate(
      pool, [&] { return scratch && !keep ? cudaMallocAsync(&b.p, bytes, s) : cudaMalloc(&b.p, bytes); });
  if (e != cudaSuccess) return e;
  if (keep) pool.lent += bytes;
  if (scratch && !keep) pool.missed = std::max(pool.missed, bytes);
  *out = b;
  return cudaSuccess;
}

void pool_put(Pool &pool, PoolBlock b, cudaStream_t s) {
  if (!b.p) return;
  if (b.bytes == 0) {
    cudaFreeAsync(b.p, s);
    return;
  }
  b.ready = nullptr;
  const bool ok = cudaEventCreateWithFlags(&b.ready, cudaEventDisableTiming) == cudaSuccess &&
                  cudaEventRecord(b.ready, s) == cudaSuccess;
  std::lock_guard<std::mutex> lk(pool.mu);
  pool.lent -= b.bytes;
  if (ok) {
    pool.kept.push_back(b);
    pool.bytes += b.bytes;
    return;
  }
  if (b.ready) cudaEventDestroy(b.ready);
  cudaFree(b.p);  // waits for the device
}

void pool_put_synced(Pool &pool, PoolBlock b) {
  unsigned long long before;
  {
    std::lock_guard<std::mutex> lk(pool.mu);
    before = pool.holds;
  }
  const bool idle = cudaDeviceSynchronize() == cudaSuccess;
  if (!idle) cudaGetLastError();
  if (!b.p) return;
  b.ready = nullptr;
  std::vector<PoolBlock> out;  // to be freed
  {
    std::lock_guard<std::mutex> lk(pool.mu);
    if (!idle) {
      // The device cannot be synchronised while one of its streams is captured: a
      // launch of another stream may still use the block, which therefore goes to
      // nobody until a synchronisation succeeds.
      if (pool.open && pool.bytes + pool.lent + b.bytes <= kPoolBytes) {
        pool.held.push_back({b, pool.holds++});
        pool.bytes += b.bytes;
      } else {
        out.push_back(b);  // cudaFree waits for the device
      }
    } else {
      // what was held when the synchronisation began is idle too
      size_t left = 0;
      for (const HeldBlock &h : pool.held) {
        if (h.seq < before) pool.kept.push_back(h.b);
        else pool.held[left++] = h;
      }
      pool.held.resize(left);
      if (pool.open && b.bytes + pool.lent <= kPoolBytes) {
        pool.kept.push_back(b);
        pool.bytes += b.bytes;
      } else {
        out.push_back(b);
      }
      // The oldest blocks go where there is no room, also for the scratch that had
      // none lately.
      const size_t room = pool.missed <= kPoolBytes / 2 ? pool.missed : 0;
      pool.missed = 0;
      size_t k = 0;
      while (k < pool.kept.size() && pool.bytes + pool.lent + room > kPoolBytes) {
        pool.bytes -= pool.kept[k].bytes;
        out.push_back(pool.kept[k++]);
      }
      pool.kept.erase(pool.kept.begin(), pool.kept.begin() + k);
    }
  }
  for (PoolBlock &o : out) {
    if (o.ready) {
      cudaEventSynchronize(o.ready);
      cudaEventDestroy(o.ready);
    }
    if (cudaFree(o.p) != cudaSuccess) cudaGetLastError();
  }
}

bh_status check_status(bh_ctx *ctx, cudaStream_t s) {
  unsigned st = 0;
  BH_CUDA(cudaMemcpyAsync(&st, ctx->status_dev, sizeof st, cudaMemcpyDeviceToHost, s));
  BH_CUDA(cudaStreamSynchronize(s));
  if (st) {
    set_error("kernel status word 0x%x (%s%s%s)", st, (st & kStatusMbarTimeout) ? "table load timed out " : "",
              (st & kStatusBarrierTimeout) ? "grid barrier timed out " : "",
              (st & kStatusBadIndex) ? "index out of range" : "");
    BH_CUDA(cudaMemsetAsync(ctx->status_dev, 0, sizeof(unsigned), s));
    return (st & (kStatusMbarTimeout | kStatusBarrierTimeout)) ? BH_ERR_TIMEOUT : BH_ERR_DEVICE_STATUS;
  }
  return BH_OK;
}

// ---------------------------------------------------------------------------
// Gauss-Legendre nodes (4 points) computed once on the host by Newton's method
// on P_4 with its three-term recurrence.
// ---------------------------------------------------------------------------
constexpr int kGL = 4;
__constant__ double cGLx[kGL], cGLw[kGL];

static void gauss_legendre(int n, double *x, double *w) {
  for (int i = 0; i < n; ++i) {
    double z = cos(kPi * (i + 0.75) / (n + 0.5)), dp = 0.0;
    for (int it = 0; it < 100; ++it) {
      double p0 = 1.0, p1 = z;
      for (int k = 2; k <= n; ++k) {
        double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
        p0 = p1;
        p1 = p2;
      }
      dp = n * (z * p1 - p0) / (z * z - 1.0);
      double dz = p1 / dp;
      z -= dz;
      if (fabs(dz) < 1e-16) break;
    }
    x[i] = z;
    w[i] = 2.0 / ((1.0 - z * z) * dp * dp);
  }
}

// ---------------------------------------------------------------------------
// Device quadrature
// ---------------------------------------------------------------------------
struct Apsis {
  double ua, A, B;  // u_a (Eq. uapsis); q(w) = A + B w^2 - w^4
};

// From eta = 1 - e^2/mu in (0,1]: u_a = 1/3 + 2/3 sin(asin(2e^2/mu - 1)/3)
// with asin(1 - 2 eta) = pi/2 - 2 asin(sqrt(eta)), and
// A = u_a (2 - 3u_a) = 4 u_a cos(pi/12 + th/2) sin(asin(sqrt(eta))/3),
// B = 3 u_a - 1 = 2 sin(th), th = asin(2e^2/mu - 1)/3 -- free of cancellation
// near the photon sphere.
__device__ Apsis apsis_of_eta(double eta) {
  double s = asin(sqrt(eta));
  double th = (0.5 * kPi - 2.0 * s) / 3.0;
  Apsis a;
  a.ua = 1.0 / 3.0 + 2.0 / 3.0 * sin(th);
  a.A = 4.0 * a.ua * cos(kPi / 12.0 + 0.5 * th) * sin(s / 3.0);
  a.B = 2.0 * sin(th);
  return a;
}

// The regularised time R = t + 1/u - ln(u/(1-u)) (reading C5) obeys
// dR/dphi = 1/(e + du/dphi), so every angle integral has a time twin whose
// integrand carries the extra factor 1/(e + du/dphi).

// Rays of one e.
struct Ray {
  double e, e2;
  bool low;       // e^2 < mu
  Apsis ap;       // low
  double w1;      // low: w at infinity, sqrt(u_a)
  double c;       // low: scale of w = c sinh t
  double em, se;  // high: e^2 - mu and its root
};

__device__ __forceinline__ Ray low_ray(double eta, double e2) {
  Ray r;
  r.low = true;
  r.e2 = e2;
  r.e = sqrt(e2);
  r.ap = apsis_of_eta(eta);
  r.w1 = sqrt(r.ap.ua);
  r.c = r.ap.B > 0.0 ? sqrt(r.ap.A / r.ap.B) : 1.0;
  r.em = r.se = 0.0;
  return r;
}

__device__ __forceinline__ Ray high_ray(double em, double e2) {
  Ray r;
  r.low = false;
  r.e2 = e2;
  r.e = sqrt(e2);
  r.em = em;
  r.se = sqrt(em);
  r.ap = {0.0, 0.0, 0.0};
  r.w1 = r.c = 0.0;
  return r;
}

// 1/x and 1/sqrt(x) by Newton's iteration from the single-precision value (x a
// normal float whose reciprocal is one): 2^-23, 2^-46, then rounding.  Six and
// ten FP64 operations, a third of the general routines'.
__device__ __forceinline__ double newton_rcp(double x) {
  double r = (double)__frcp_rn((float)x);
  r = fma(r, fma(-x, r, 1.0), r);
  return fma(r, fma(-x, r, 1.0), r);
}

__device__ __forceinline__ double newton_rsqrt(double x) {
  double r = (double)rsqrtf((float)x);
  r = fma(0.5 * r, fma(-x * r, r, 1.0), r);
  return fma(0.5 * r, fma(-x * r, r, 1.0), r);
}

// dphi/ds, u and du/dphi at a point: s = w (low) or z (high), falling and
// rising with phi.
__device__ __forceinline__ double ray_rate(const Ray &r, double s, double &u, double &ud) {
  if (r.low) {
    const double w2 = s * s, q = fma(w2, r.ap.B - w2, r.ap.A), rq = newton_rsqrt(q);
    u = r.ap.ua - w2;
    ud = s * (q * rq);
    return 2.0 * rq;
  }
  const double v = s * fabs(s), P = fma(v * v, v + 1.0, r.em), rp = newton_rsqrt(P);
  u = 2.0 / 3.0 + v;
  ud = P * rp;
  return 2.0 * fabs(s) * rp;
}

// The same in t: w = c sinh t where u_a > 0.6 and v = sqrt(e^2-mu) sinh t, else w
// = t.
__device__ __forceinline__ bool ray_sinh(const Ray &r) { return !r.low || r.ap.ua > 0.6; }

__device__ __forceinline__ double ray_rate_t(const Ray &r, double t, double &u, double &ud) {
  if (!ray_sinh(r)) return ray_rate(r, t, u, ud);
  const double sh = sinh(t), ch = sqrt(fma(sh, sh, 1.0));
  if (r.low) return ray_rate(r, r.c * sh, u, ud) * r.c * ch;
  // P = (e^2 - mu) cosh^2 t (1 + v tanh^2 t)
  const double v = r.se * sh, th = sh / ch, g = fma(v * th, th, 1.0), rg = rsqrt(g);
  u = 2.0 / 3.0 + v;
  ud = r.se * ch * (g * rg);
  return rg;
}

// Inclusive scan of two sums over the block (a multiple of 32 threads, at
// most 1024), plus the totals; buf holds 64 doubles.
__device__ __forceinline__ void block_scan2(double &a, double &b, double *buf, double &ta, double &tb) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  for (int o = 1; o < 32; o <<= 1) {
    const double x = __shfl_up_sync(0xffffffffu, a, o), y = __shfl_up_sync(0xffffffffu, b, o);
    if (lane >= o) { a += x; b += y; }
  }
  __syncthreads();  // buf may still be read from the scan before
  if (lane == 31) { buf[warp] = a; buf[32 + warp] = b; }
  __syncthreads();
  double pa = 0.0, pb = 0.0;
  ta = tb = 0.0;
  for (int w = 0; w < warps; ++w) {
    if (w == warp) { pa = ta; pb = tb; }
    ta += buf[w];
    tb += buf[32 + w];
  }
  a += pa;
  b += pb;
}

template <typename T>
__device__ __forceinline__ T to_storage(double v);
template <>
__device__ __forceinline__ float to_storage<float>(double v) { return (float)v; }
template <>
__device__ __forceinline__ __half to_storage<__half>(double v) { return __double2half(v); }

constexpr int kColumnThreads = 256, kDSteps = 2;

// Column i of D and its time channel: texel (i,j) holds the Appendix A
// coordinates x = i/(n-1), y = j/(n-1) (reading C3).
__device__ void d_column(int n, int i, double *D64, double *DT64, float *DTs, double *buf) {
  // the ray's constants cost as much FP64 as 50 nodes: one thread forms them
  __shared__ Ray ray;
  if (threadIdx.x == 0) {
    // x = 1/2 - sqrt(-log(1 - e^2/mu)/50): eta = 1 - e^2/mu = exp(-50 (1/2 - x)^2);
    // x = 1/2 + sqrt(-log(1 - mu/e^2)/50): 1 - mu/e^2 = exp(-50 (x - 1/2)^2)
    const double x = (double)i / (n - 1), a = fabs(0.5 - x);
    const double eta = exp(-50.0 * a * a), one_eta = -expm1(-50.0 * a * a);
    ray = i < n / 2 ? low_ray(eta, kMu * one_eta) : high_ray(kMu / one_eta * eta, kMu / one_eta);
  }
  __syncthreads();
  const Ray r = ray;
  const double r23 = sqrt(2.0 / 3.0), r13 = sqrt(1.0 / 3.0);
  // y = 1 - sqrt(1 - u/u_a) = 1 - w/w1 (low), equal steps of z (high)
  auto place = [&](double y) { return r.low ? r.w1 * (1.0 - y) : y * (r23 + r13) - r23; };
  // panels between two texels: never wider than 1/511 of the range
  const int parts = (511 + n - 2) / (n - 1), panels = (n - 1) * parts;
  const double dy = 1.0 / panels;
  double base_d = 0.0, base_t = 0.0;
  for (int k0 = 0; k0 < panels; k0 += kDSteps * blockDim.x) {
    const int first = k0 + kDSteps * threadIdx.x;
    double sd[kDSteps], st[kDSteps], all_d = 0.0, all_t = 0.0, p = place(first * dy);
#pragma unroll
    for (int c = 0; c < kDSteps; ++c) {
      sd[c] = st[c] = 0.0;
      if (first + c < panels) {
        // the last panel ends at y = 1 exactly
        const double q = place(first + c + 1 == panels ? 1.0 : (first + c + 1) * dy);
        auto panel = [&](double p, double q) {
          const double m = 0.5 * (p + q), h = 0.5 * fabs(q - p);
          double vd = 0.0, vt = 0.0;
#pragma unroll
          for (int g = 0; g < kGL; ++g) {
            double u, ud;
            const double f = ray_rate(r, fma(h, cGLx[g], m), u, ud) * cGLw[g];
            const double u3 = u * u * u, den = r.e2 + u3, den_t = r.e + ud, inv = newton_rcp(den * den_t);
            vd = fma(f, u3 * (den_t * inv), vd);
            vt = fma(f, den * inv, vt);
          }
          sd[c] = fma(1.5 * h, vd, sd[c]);
          st[c] = fma(h, vt, st[c]);
        };
        if (!r.low && p < 0.0 && q > 0.0) {  // |z| has a corner at 0
          panel(p, 0.0);
          panel(0.0, q);
        } else {
          panel(p, q);
        }
        p = q;
      }
      all_d += sd[c];
      all_t += st[c];
    }
    double up_d = all_d, up_t = all_t, td, tt;
    block_scan2(up_d, up_t, buf, td, tt);
    up_d += base_d - all_d;  // the integrals before this thread's panels
    up_t += base_t - all_t;
#pragma unroll
    for (int c = 0; c < kDSteps; ++c) {
      const int k = first + c + 1;
      up_d += sd[c];
      up_t += st[c];
      if (k <= panels && (parts == 1 || k % parts == 0)) {
        const size_t o = (size_t)(parts == 1 ? k : k / parts) * n + i;
        D64[o] = up_d;
        DT64[o] = up_t;
        DTs[o] = (float)up_t;
      }
    }
    base_d += td;
    base_t += tt;
  }
  if (threadIdx.x == 0) {
    D64[i] = 0.0;
    DT64[i] = 0.0;
    DTs[i] = 0.f;
  }
}

// Column i of U: x = 1/(1 + 6 e^2), y = (phi/3)(1 + 6 e^3)/(1 + e^2).  UT gets
// the regularised time at the same point; past the apsis it follows from the
// time symmetry of the ray about its apsis, t(phi) = 2 t_a - t(2 phi_a - phi).
// The integrals up to kUPanels + 1 points first; then eight lanes per texel
// invert phi inside the panel that holds it.
constexpr int kUPanels = 256;

template <typename T>
__device__ void u_column(int ne, int nphi, int i, double *U64, T *Us, double *UT64, float *UTs, double *buf) {
  __shared__ double phis[kUPanels + 1], times[kUPanels + 1];
  const double x = (double)i / (ne - 1);
  const double e2 = i == 0 ? 0.0 : (1.0 / x - 1.0) / 6.0;
  const bool radial = i == 0, none = !radial && e2 <= 0.0;
  __shared__ Ray ray;
  __shared__ double span[2];  // t at u = 0 and at the apsis (low: 0) or the horizon
  if (threadIdx.x == 0 && !radial && !none) {
    if (e2 < kMu) {
      ray = low_ray(1.0 - e2 / kMu, e2);
      span[0] = ray_sinh(ray) ? asinh(ray.w1 / ray.c) : ray.w1;
      span[1] = 0.0;
    } else {
      ray = high_ray(fmax(e2 - kMu, 1e-24), e2);
      span[0] = asinh(-2.0 / 3.0 / ray.se);
      span[1] = asinh(1.0 / 3.0 / ray.se);
    }
  }
  __syncthreads();
  const Ray r = ray;
  const double t0 = span[0], t1 = span[1];
  if (!radial && !none) {
    const double step = (t1 - t0) / kUPanels;
    static_assert(kUPanels <= kColumnThreads, "one panel per thread");
    const int k = threadIdx.x;
    double sp = 0.0, st = 0.0, tp, tt;
    const double m = fma(k + 0.5, step, t0), h = 0.5 * fabs(step);
    if (k < kUPanels) {
#pragma unroll
      for (int g = 0; g < kGL; ++g) {
        double u, ud;
        const double f = ray_rate_t(r, fma(h, cGLx[g], m), u, ud) * (cGLw[g] * h);
        sp += f;
        st = fma(f, newton_rcp(r.e + ud), st);
      }
    }
    block_scan2(sp, st, buf, tp, tt);
    if (k < kUPanels) {
      phis[k + 1] = sp;
      times[k + 1] = st;
    }
    if (k == 0) phis[0] = times[0] = 0.0;
  }
  __syncthreads();
  const int lane8 = threadIdx.x & 7;
  for (int j0 = 0; j0 < nphi; j0 += blockDim.x / 8) {
    const int j = j0 + (int)(threadIdx.x >> 3);
    const bool real = j < nphi;
    double u = 0.0, R = 0.0;  // R = 0 where there is no ray or it was captured
    const double y = (double)min(j, nphi - 1) / (nphi - 1);
    if (radial) {
      u = j == 0 ? 0.0 : 1.0;  // e -> infinity: radial ray, captured at once
    } else if (!none) {        // the same for the whole block: its lanes stay together
      double phi = 3.0 * y * (1.0 + e2) / (1.0 + 6.0 * e2 * r.e);
      const double last = phis[kUPanels];
      const bool start = phi <= 0.0;
      const bool captured = !r.low && phi >= last;  // reached the horizon before phi (reading C7)
      const bool past = r.low && phi > last;
      if (past) phi = 2.0 * last - phi;  // past the apsis: reflection
      const bool away = phi < 0.0;       // back at infinity: no texel of the mapping gets here
      int k = 0;                         // the panel with phis[k] <= phi < phis[k + 1]
      for (int bit = kUPanels / 2; bit > 0; bit >>= 1)
        if (k + bit < kUPanels && phis[k + bit] <= phi) k += bit;
      const double step = (t1 - t0) / kUPanels, ta = fma((double)k, step, t0);
      const double p0 = phis[k], p1 = phis[k + 1];
      double f = fmin(fmax((phi - p0) / (p1 - p0), 0.0), 1.0);  // place in the panel
      double at, uu, rate = 1.0, rsum = 0.0;
      // three Newton steps from the linear guess (error 1e-4 of the panel, then its
      // square, then rounding), then the time: lanes 0-3 take the nodes, lane 4
      // the end
#pragma unroll 1
      for (int it = 0; it < 4; ++it) {
        at = fma(f, step, ta);
        const double h = 0.5 * fabs(f * step), m = fma(0.5 * f, step, ta);
        const double node = lane8 < kGL ? cGLx[lane8] : 0.0, wt = lane8 < kGL ? cGLw[lane8] * h : 0.0;
        double un, ud;
        const double g = ray_rate_t(r, lane8 < kGL ? fma(h, node, m) : at, un, ud);
        double sum = wt * (it == 3 ? g / (r.e + ud) : g);
        for (int o = 4; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        rate = __shfl_sync(0xffffffffu, g, (threadIdx.x & 24) + 4);
        uu = __shfl_sync(0xffffffffu, un, (threadIdx.x & 24) + 4);
        if (it < 3) f = fmin(fmax(f - (p0 + sum - phi) / (rate * fabs(step)), 0.0), 1.0);
        else rsum = sum;
      }
      u = uu;
      R = times[k] + rsum;
      if (past) {
        const double Ra = times[kUPanels], ua = r.ap.ua;
        R = u > 0.0 ? 2.0 * Ra - 2.0 / ua + 2.0 * log(ua / (1.0 - ua)) - R + 2.0 / u - 2.0 * log(u / (1.0 - u)) : 0.0;
      }
      if (captured) { u = 1.0; R = 0.0; }
      if (start || away) u = R = 0.0;
    }
    if (real && lane8 == 0) {
      const size_t o = (size_t)j * ne + i;
      U64[o] = u;
      Us[o] = to_storage<T>(u);
      UT64[o] = R;
      UTs[o] = (float)R;
    }
  }
}

// One block per column: U's first (they take longest), then D's.
template <typename T>
__global__ void __launch_bounds__(kColumnThreads, 4) precompute_kernel(int n, double *D64, double *DT64, float *DTs, int ne,
                                                                   int nphi, double *U64, T *Us, double *UT64,
                                                                   float *UTs) {
  __shared__ double buf[64];
  if ((int)blockIdx.x < ne) u_column<T>(ne, nphi, blockIdx.x, U64, Us, UT64, UTs, buf);
  else d_column(n, blockIdx.x - ne, D64, DT64, DTs, buf);
}

// The render copy of D, row-paired: texel (j, i) holds D(j, i) and
// D(min(j+1, n-1), i) side by side, so a bilinear lookup is two loads.
template <typename T>
__global__ void pair_d_kernel(int n, const double *D64, T *Dp) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
  if (i >= n || j >= n) return;
  const size_t o = (size_t)j * n + i;
  Dp[2 * o] = to_storage<T>(D64[o]);
  Dp[2 * o + 1] = to_storage<T>(D64[(size_t)min(j + 1, n - 1) * n + i]);
}

template <typename T>
__global__ void convert_kernel(const double *src, T *dst, size_t n) {
  size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (i < n) dst[i] = to_storage<T>(src[i]);
}

// ---------------------------------------------------------------------------
// Colour tables (Sec. 3.4.2, reading C14)
// ---------------------------------------------------------------------------
// A black body's X, Y, Z times exp(c2/(830 nm T)) - 1 is smooth and between 0 and
// O(1) for any T: fitted by polynomials in 1/T, from 0 to 1/960 K on 22 cells (the
// Planckian locus, whose nearest points are decided in FP64: truncation 1e-15)
// and to 1/64 K on 138 cells (C alone, rounded to float: 1e-11).  1,920 black
// bodies replace 400,000 (3.5 ms) for the locus, the disc table and C.
constexpr int kSpecFine = 22, kSpecCells = 160, kSpecNodes = 12;
constexpr double kSpecV0 = 1.0 / 960.0, kSpecV1 = 1.0 / 64.0;  // 1/K
constexpr double kSpecStep0 = kSpecV0 / kSpecFine, kSpecStep1 = (kSpecV1 - kSpecV0) / (kSpecCells - kSpecFine);
constexpr int kSpecCoefs = kSpecCells * 3 * kSpecNodes;
using SpecFit = BlackBodyFit<kSpecNodes>;

// One warp per node; the last node of a cell to finish fits the cell.
__global__ void spectrum_kernel(const SpecFit fit, double *val, unsigned *done, double *coef) {
  const int lane = threadIdx.x, cell = blockIdx.x / kSpecNodes, node = blockIdx.x - cell * kSpecNodes;
  const double at = 0.5 * (fit.node[node] + 1.0);
  const double v = cell < kSpecFine ? (cell + at) * kSpecStep0 : kSpecV0 + (cell - kSpecFine + at) * kSpecStep1;  // 1/T
  const double ref = expm1(fit.x[kNLambda - 1] * v);
  double s[3] = {0.0, 0.0, 0.0};
  for (int k = lane; k < kNLambda; k += 32) {
    const double b = ref / expm1(fit.x[k] * v);
    for (int c = 0; c < 3; ++c) s[c] = fma(b, fit.w[c][k], s[c]);
  }
  for (int o = 16; o > 0; o >>= 1)
    for (int c = 0; c < 3; ++c) s[c] += __shfl_xor_sync(0xffffffffu, s[c], o);
  unsigned before = 0;
  if (lane == 0) {
    for (int c = 0; c < 3; ++c) val[blockIdx.x * 3 + c] = s[c];
    __threadfence();
    before = atomicAdd(done + cell, 1u);
    __threadfence();
  }
  if (__shfl_sync(0xffffffffu, before, 0) != kSpecNodes - 1u) return;
  for (int k = lane; k < 3 * kSpecNodes; k += 32)
    coef[cell * 3 * kSpecNodes + k] = fit_coefficient(fit, k % kSpecNodes, val + cell * kSpecNodes * 3 + k / kSpecNodes, 3);
}

// X, Y, Z of the black body of temperature 1/v, times exp(c2 v / 830 nm) - 1.
__device__ __forceinline__ void spectrum_xyz(const double *coef, double v, double *g) {
  const bool fine = v < kSpecV0;
  const double t = fine ? v * (1.0 / kSpecStep0) : (v - kSpecV0) * (1.0 / kSpecStep1);
  const int k = min((int)t, fine ? kSpecFine - 1 : kSpecCells - kSpecFine - 1), cell = fine ? k : kSpecFine + k;
  const double u = fma(2.0, t - k, -1.0);
  const double *a = coef + cell * 3 * kSpecNodes;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    double s = a[c * kSpecNodes + kSpecNodes - 1];
#pragma unroll
    for (int m = kSpecNodes - 2; m >= 0; --m) s = fma(s, u, a[c * kSpecNodes + m]);
    g[c] = s;
  }
}

constexpr double kRefK = 1.4387769e7 / 830.0;  // c2 / 830 nm

__device__ __forceinline__ void uv1960(const double *xyz, double *uv) {
  double den = __dadd_rn(__dadd_rn(xyz[0], __dmul_rn(15.0, xyz[1])), __dmul_rn(3.0, xyz[2]));
  uv[0] = __ddiv_rn(__dmul_rn(4.0, xyz[0]), den);
  uv[1] = __ddiv_rn(__dmul_rn(6.0, xyz[1]), den);
}

struct Locus {
  double2 uv[kNLocus];     // Planckian locus in CIE 1960 uv, T = 1000 40^(m/4095)
  double2 body[kNLocus];   // 1/T, and (exp(c2/(830 nm T)) - 1) / (X+Y+Z) of the fit
  double shift[kCnd];      // 1/D of C's layers
  float2 uv32[kNLocus];
};

// The locus, and the disc table: ln Y, X/Y, Z/Y of B_T at log2 T = 8 + 12 (k +
// 1/2)/n (one exponential per lookup).
__global__ void locus_disc_kernel(const double *coef, Locus *locus, float4 *disc) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  double g[3];
  if (m < kNLocus) {
    const double v = 1.0 / (1000.0 * pow(40.0, m / 4095.0));
    spectrum_xyz(coef, v, g);
    double uv[2];
    uv1960(g, uv);
    locus->uv[m] = make_double2(uv[0], uv[1]);
    locus->uv32[m] = make_float2((float)uv[0], (float)uv[1]);
    locus->body[m] = make_double2(v, expm1(kRefK * v) / (g[0] + g[1] + g[2]));
    if (m < kCnd) locus->shift[m] = exp2(4.0 - 8.0 * (m + 0.5) / kCnd);
  } else if (m < kNLocus + kDiscN) {
    const int k = m - kNLocus;
    const double v = exp2(-(8.0 + 12.0 * (k + 0.5) / kDiscN));
    spectrum_xyz(coef, v, g);
    // the fit's wavelengths are in units of 560 nm
    disc[k] = make_float4((float)(log(g[1] / expm1(kRefK * v)) - 5.0 * log(560.0)), (float)(g[0] / g[1]),
                          (float)(g[2] / g[1]), 0.f);
  }
}

// C(xy, D) = XYZ(B_{D T}) / (X+Y+Z)(B_T), T the nearest Planckian-locus
// temperature of the cell in CIE 1960 uv (D^5 I(D lambda) of a black body is the
// black body at temperature D T).  One warp per (x, y) cell.  The nearest point
// is searched in FP32; FP64 decides between the points within its error.
__global__ void colour_cell_kernel(const Locus *locus, const double *coef, float4 *C) {
  const int cell = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (cell >= kCnx * kCny) return;  // whole warps leave together
  const int i = cell % kCnx, j = cell / kCnx;
  const double x = 0.15 + 0.60 * (i + 0.5) / kCnx, y = 0.15 + 0.35 * (j + 0.5) / kCny;
  const double c[3] = {__ddiv_rn(x, y), 1.0, __ddiv_rn(__dadd_rn(__dadd_rn(1.0, -x), -y), y)};
  double uv[2];
  uv1960(c, uv);
  const float uf = (float)uv[0], vf = (float)uv[1];
  auto near = [&](int m) {
    const float2 p = locus->uv32[m];
    const float du = uf - p.x, dv = vf - p.y;
    return fmaf(du, du, dv * dv);
  };
  float least = INFINITY;
  for (int m = lane; m < kNLocus; m += 32) least = fminf(least, near(m));
  for (int o = 16; o > 0; o >>= 1) least = fminf(least, __shfl_xor_sync(0xffffffffu, least, o));
  // du and dv are off by at most 1.2e-7 each
  const float bound = fmaf(1e-6f, sqrtf(least) + least, least + 1e-12f);
  double bd = INFINITY;
  int best = kNLocus;
  // the candidates of a lane as bits first: under a condition in this loop, the
  // FP64 of all its steps would be issued, predicated off (146 us)
  for (int m0 = 0; m0 < kNLocus; m0 += 1024) {
    unsigned in = 0;
    for (int k = 0; k < 32; ++k) in |= near(m0 + 32 * k + lane) <= bound ? 1u << k : 0u;
    while (in) {
      const int m = m0 + 32 * (__ffs(in) - 1) + lane;
      in &= in - 1u;
      const double2 p = locus->uv[m];
      const double du = __dadd_rn(uv[0], -p.x), dv = __dadd_rn(uv[1], -p.y);
      const double d = __dadd_rn(__dmul_rn(du, du), __dmul_rn(dv, dv));
      if (d < bd) { bd = d; best = m; }
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    const double d = __shfl_xor_sync(0xffffffffu, bd, o);
    const int m = __shfl_xor_sync(0xffffffffu, best, o);
    if (d < bd || (d == bd && m < best)) { bd = d; best = m; }
  }
  const double2 body = locus->body[best];
  for (int k = lane; k < kCnd; k += 32) {
    const double vk = body.x * locus->shift[k];
    double r[3];
    spectrum_xyz(coef, vk, r);
    const double f = body.y / expm1(kRefK * vk);
    C[((size_t)k * kCny + j) * kCnx + i] = make_float4((float)(r[0] * f), (float)(r[1] * f), (float)(r[2] * f), 0.f);
  }
}

bh_status colour_tables_launch(bh_ctx *ctx, bh_tables *t, cudaStream_t s) {
  struct Scratch {
    Locus locus;
    double coef[kSpecCoefs], val[kSpecCells * kSpecNodes * 3];
    unsigned done[kSpecCells];
  };
  PoolBlock mem;
  BH_CUDA(pool_get(*ctx->pool, sizeof(Scratch), s, &mem, true));
  Scratch *w = static_cast<Scratch *>(mem.p);
  cudaError_t e = cudaMemsetAsync(w->done, 0, sizeof w->done, s);
  spectrum_kernel<<<kSpecCells * kSpecNodes, 32, 0, s>>>(black_body_fit<kSpecNodes>(), w->val, w->done, w->coef);
  locus_disc_kernel<<<(kNLocus + kDiscN) / 64, 64, 0, s>>>(w->coef, &w->locus, t->disc);
  colour_cell_kernel<<<kCnx * kCny / 4, 128, 0, s>>>(&w->locus, w->coef, t->C);
  count_launch(ctx, 3);
  if (e == cudaSuccess) e = cudaGetLastError();
  pool_put(*ctx->pool, mem, s);
  return e == cudaSuccess ? BH_OK : cuda_fail(e, "colour tables");
}

}  // namespace bh

using namespace bh;

// ---------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------
extern "C" const char *bh_last_error(void) { return g_last_error.c_str(); }

extern "C" bh_status bh_create(int device, size_t budget, bh_ctx **out) {
  if (!out) { set_error("bh_create: out is NULL"); return BH_ERR_INVALID_ARG; }
  *out = nullptr;
  int ndev = 0;
  BH_CUDA(cudaGetDeviceCount(&ndev));
  if (device < 0 || device >= ndev) {
    set_error("bh_create: device %d not in [0, %d)", device, ndev);
    return BH_ERR_INVALID_ARG;
  }
  BH_CUDA(cudaSetDevice(device));
  bh_ctx *c = new bh_ctx();
  c->device = c->pool->device = device;
  c->budget = budget;
  cudaError_t e = cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, device);
  if (e == cudaSuccess) e = cudaMalloc((void **)&c->status_dev, sizeof(unsigned));
  if (e == cudaSuccess) e = cudaMemset(c->status_dev, 0, sizeof(unsigned));
  if (e == cudaSuccess) e = cudaMalloc((void **)&c->sched_dev, sizeof(unsigned) * 2 * kSchedRing);
  if (e == cudaSuccess) e = cudaMemset(c->sched_dev, 0, sizeof(unsigned) * 2 * kSchedRing);
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&c->aux, cudaStreamNonBlocking);
  if (e != cudaSuccess) {
    bh_destroy(c);
    return cuda_fail(e, "bh_create");
  }
  static bool gl_ready[64] = {false};
  static std::mutex gl_mu;
  {
    std::lock_guard<std::mutex> lk(gl_mu);
    if (device < 64 && !gl_ready[device]) {
      double x[kGL], w[kGL];
      gauss_legendre(kGL, x, w);
      e = cudaMemcpyToSymbol(cGLx, x, sizeof x);
      if (e == cudaSuccess) e = cudaMemcpyToSymbol(cGLw, w, sizeof w);
      if (e != cudaSuccess) {
        bh_destroy(c);
        return cuda_fail(e, "bh_create: Gauss-Legendre nodes");
      }
      gl_ready[device] = true;
    }
  }
  *out = c;
  return BH_OK;
}

namespace bh {
void serve_destroy(bh_ctx *ctx);
}

extern "C" void bh_destroy(bh_ctx *c) {
  if (!c) return;
  cudaSetDevice(c->device);
  bh::serve_destroy(c);
  cudaDeviceSynchronize();
  c->graph.reset();
  {
    std::lock_guard<std::mutex> lk(c->pool->mu);
    c->pool->open = false;
    bh::pool_release(*c->pool);
  }
  if (c->status_dev) cudaFree(c->status_dev);
  if (c->sched_dev) cudaFree(c->sched_dev);
  if (c->aux) cudaStreamDestroy(c->aux);
  if (c->cam_host) cudaFreeHost(c->cam_host);
  if (c->cam_dev) cudaFree(c->cam_dev);
  if (c->frame_dev) cudaFree(c->frame_dev);
  for (int k = 0; k < 2; ++k) {
    if (c->ring_dev[k]) cudaFree(c->ring_dev[k]);
    if (c->ring_ready[k]) cudaEventDestroy(c->ring_ready[k]);
    if (c->ring_done[k]) cudaEventDestroy(c->ring_done[k]);
  }
  if (c->ring_copy) cudaStreamDestroy(c->ring_copy);
  if (c->bloom_dev) cudaFree(c->bloom_dev);
  if (c->bloom_bar) cudaFree(c->bloom_bar);
  if (c->orb_done) cudaEventDestroy(c->orb_done);
  if (c->orb_cams_dev) cudaFree(c->orb_cams_dev);
  delete c;
}

extern "C" long long bh_kernel_launches(const bh_ctx *ctx) {
  return ctx ? ctx->launches.load() : 0;
}

static bool valid_desc(const bh_table_desc *d) {
  if (!d) { set_error("table desc is NULL"); return false; }
  if (d->d_n < 4 || d->d_n > 4096 || (d->d_n & 1)) {
    set_error("d_n = %d: must be even, 4..4096", d->d_n);
    return false;
  }
  if (d->u_ne < 2 || d->u_nphi < 2 || d->u_ne * d->u_nphi > kMaxUTexels) {
    set_error("U table %d x %d: each >= 2 and at most %d texels", d->u_ne, d->u_nphi, kMaxUTexels);
    return false;
  }
  if (d->storage != BH_F32 && d->storage != BH_F16) {
    set_error("table storage must be BH_F32 or BH_F16");
    return false;
  }
  return true;
}

static bh_status tables_alloc(bh_ctx *ctx, const bh_table_desc *desc, cudaStream_t s,
                              bh_tables **out) {
  bh_tables *t = new bh_tables();
  t->ctx = ctx;
  t->pool = ctx->pool;
  t->desc = *desc;
  size_t nd = (size_t)desc->d_n * desc->d_n, nu = (size_t)desc->u_ne * desc->u_nphi;
  const size_t es = desc->storage == BH_F32 ? 4 : 2;
  // one allocation, every array on a 256-byte line
  size_t bytes = 0;
  auto place = [&](size_t b) {
    const size_t at = bytes;
    bytes += (b + 255) / 256 * 256;
    return at;
  };
  const size_t o_D64 = place(nd * 8), o_U64 = place(nu * 8), o_D = place(2 * nd * es) /* row-paired render copy */,
               o_U = place(nu * es), o_DT64 = place(nd * 8), o_UT64 = place(nu * 8), o_DT = place(nd * 4),
               o_UT = place(nu * 4), o_C = place(sizeof(float4) * kCnx * kCny * kCnd), o_disc = place(sizeof(float4) * kDiscN);
  const cudaError_t e = pool_get(*ctx->pool, bytes, s, &t->mem);
  if (e != cudaSuccess) {
    delete t;
    return cuda_fail(e, "table allocation");
  }
  char *p = static_cast<char *>(t->mem.p);
  t->D64 = reinterpret_cast<double *>(p + o_D64);
  t->U64 = reinterpret_cast<double *>(p + o_U64);
  t->D = p + o_D;
  t->U = p + o_U;
  t->DT64 = reinterpret_cast<double *>(p + o_DT64);
  t->UT64 = reinterpret_cast<double *>(p + o_UT64);
  t->DT = reinterpret_cast<float *>(p + o_DT);
  t->UT = reinterpret_cast<float *>(p + o_UT);
  t->C = reinterpret_cast<float4 *>(p + o_C);
  t->disc = reinterpret_cast<float4 *>(p + o_disc);
  *out = t;
  return BH_OK;
}

extern "C" bh_status bh_precompute_tables(bh_ctx *ctx, const bh_table_desc *desc, void *stream,
                                          bh_tables **out) {
  TraceRange trace_("bh_precompute_tables");
  if (!ctx || !out) { set_error("bh_precompute_tables: NULL argument"); return BH_ERR_INVALID_ARG; }
  *out = nullptr;
  if (!valid_desc(desc)) return BH_ERR_INVALID_ARG;
  BH_CUDA(cudaSetDevice(ctx->device));
  cudaStream_t s = (cudaStream_t)stream;
  bh_tables *t = nullptr;
  bh_status st = tables_alloc(ctx, desc, s, &t);
  if (st) return st;
  const int n = desc->d_n;
  const dim3 gd((n + 127) / 128, n);
  const unsigned columns = (unsigned)(n + desc->u_ne);
  if (desc->storage == BH_F32) {
    precompute_kernel<float><<<columns, kColumnThreads, 0, s>>>(n, t->D64, t->DT64, t->DT, desc->u_ne, desc->u_nphi,
                                                               t->U64, (float *)t->U, t->UT64, t->UT);
    pair_d_kernel<float><<<gd, 128, 0, s>>>(n, t->D64, (float *)t->D);
  } else {
    precompute_kernel<__half><<<columns, kColumnThreads, 0, s>>>(n, t->D64, t->DT64, t->DT, desc->u_ne, desc->u_nphi,
                                                                t->U64, (__half *)t->U, t->UT64, t->UT);
    pair_d_kernel<__half><<<gd, 128, 0, s>>>(n, t->D64, (__half *)t->D);
  }
  count_launch(ctx, 2);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { bh_tables_free(t); return cuda_fail(e, "precompute launch"); }
  st = colour_tables_launch(ctx, t, s);
  if (st) { bh_tables_free(t); return st; }
  *out = t;
  return BH_OK;
}

namespace bh {
bh_status tables_alloc_public(bh_ctx *ctx, const bh_table_desc *desc, cudaStream_t s, bh_tables **out) {
  return tables_alloc(ctx, desc, s, out);
}

// Storage copies of D and U (the table's storage type) and FP32 copies of the
// time channels from the FP64 values already on the device.
bh_status tables_convert_storage(bh_ctx *ctx, bh_tables *t, cudaStream_t s) {
  size_t nd = (size_t)t->desc.d_n * t->desc.d_n, nu = (size_t)t->desc.u_ne * t->desc.u_nphi;
  const int n = t->desc.d_n;
  const dim3 gd((n + 127) / 128, n);
  if (t->desc.storage == BH_F32) {
    pair_d_kernel<float><<<gd, 128, 0, s>>>(n, t->D64, (float *)t->D);
    convert_kernel<float><<<(nu + 255) / 256, 256, 0, s>>>(t->U64, (float *)t->U, nu);
  } else {
    pair_d_kernel<__half><<<gd, 128, 0, s>>>(n, t->D64, (__half *)t->D);
    convert_kernel<__half><<<(nu + 255) / 256, 256, 0, s>>>(t->U64, (__half *)t->U, nu);
  }
  convert_kernel<float><<<(nd + 255) / 256, 256, 0, s>>>(t->DT64, t->DT, nd);
  convert_kernel<float><<<(nu + 255) / 256, 256, 0, s>>>(t->UT64, t->UT, nu);
  count_launch(ctx, 4);
  BH_CUDA(cudaGetLastError());
  return BH_OK;
}
}  // namespace bh

extern "C" bh_status bh_tables_upload(bh_ctx *ctx, const bh_table_desc *desc, const double *Dh,
                                      const double *Uh, void *stream, bh_tables **out) {
  TraceRange trace_("bh_tables_upload");
  if (!ctx || !out || !Dh || !Uh) { set_error("bh_tables_upload: NULL argument"); return BH_ERR_INVALID_ARG; }
  *out = nullptr;
  if (!valid_desc(desc)) return BH_ERR_INVALID_ARG;
  BH_CUDA(cudaSetDevice(ctx->device));
  cudaStream_t s = (cudaStream_t)stream;
  bh_tables *t = nullptr;
  bh_status st = tables_alloc(ctx, desc, s, &t);
  if (st) return st;
  size_t nd = (size_t)desc->d_n * desc->d_n, nu = (size_t)desc->u_ne * desc->u_nphi;
  cudaError_t e = cudaMemcpyAsync(t->D64, Dh, nd * 8, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(t->U64, Uh, nu * 8, cudaMemcpyHostToDevice, s);
  // no time channel until bh_tables_upload_time: all-ones bytes read as NaN
  if (e == cudaSuccess) e = cudaMemsetAsync(t->DT64, 0xff, nd * 8, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(t->UT64, 0xff, nu * 8, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(t->DT, 0xff, nd * 4, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(t->UT, 0xff, nu * 4, s);
  if (e == cudaSuccess) {
    const int n = desc->d_n;
    const dim3 gd((n + 127) / 128, n);
    if (desc->storage == BH_F32) {
      pair_d_kernel<float><<<gd, 128, 0, s>>>(n, t->D64, (float *)t->D);
      convert_kernel<float><<<(nu + 255) / 256, 256, 0, s>>>(t->U64, (float *)t->U, nu);
    } else {
      pair_d_kernel<__half><<<gd, 128, 0, s>>>(n, t->D64, (__half *)t->D);
      convert_kernel<__half><<<(nu + 255) / 256, 256, 0, s>>>(t->U64, (__half *)t->U, nu);
    }
    count_launch(ctx, 2);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) {
    st = colour_tables_launch(ctx, t, s);
    if (st) { bh_tables_free(t); return st; }
    e = cudaStreamSynchronize(s);
  }
  if (e != cudaSuccess) { bh_tables_free(t); return cuda_fail(e, "bh_tables_upload"); }
  *out = t;
  return BH_OK;
}

extern "C" bh_status bh_tables_copy_out(const bh_tables *t, double *Dh, double *Uh) {
  if (!t) { set_error("bh_tables_copy_out: NULL tables"); return BH_ERR_INVALID_ARG; }
  BH_CUDA(cudaSetDevice(t->ctx->device));
  BH_CUDA(cudaDeviceSynchronize());
  if (Dh) BH_CUDA(cudaMemcpy(Dh, t->D64, sizeof(double) * t->desc.d_n * t->desc.d_n, cudaMemcpyDeviceToHost));
  if (Uh) BH_CUDA(cudaMemcpy(Uh, t->U64, sizeof(double) * t->desc.u_ne * t->desc.u_nphi, cudaMemcpyDeviceToHost));
  return BH_OK;
}

extern "C" bh_status bh_tables_upload_time(bh_tables *t, const double *DTh, const double *UTh, void *stream) {
  if (!t || !DTh || !UTh) { set_error("bh_tables_upload_time: NULL argument"); return BH_ERR_INVALID_ARG; }
  BH_CUDA(cudaSetDevice(t->ctx->device));
  cudaStream_t s = (cudaStream_t)stream;
  size_t nd = (size_t)t->desc.d_n * t->desc.d_n, nu = (size_t)t->desc.u_ne * t->desc.u_nphi;
  BH_CUDA(cudaMemcpyAsync(t->DT64, DTh, nd * 8, cudaMemcpyHostToDevice, s));
  BH_CUDA(cudaMemcpyAsync(t->UT64, UTh, nu * 8, cudaMemcpyHostToDevice, s));
  convert_kernel<float><<<(nd + 255) / 256, 256, 0, s>>>(t->DT64, t->DT, nd);
  convert_kernel<float><<<(nu + 255) / 256, 256, 0, s>>>(t->UT64, t->UT, nu);
  count_launch(t->ctx, 2);
  BH_CUDA(cudaGetLastError());
  BH_CUDA(cudaStreamSynchronize(s));
  return BH_OK;
}

extern "C" bh_status bh_tables_copy_time(const bh_tables *t, double *DTh, double *UTh) {
  if (!t) { set_error("bh_tables_copy_time: NULL tables"); return BH_ERR_INVALID_ARG; }
  BH_CUDA(cudaSetDevice(t->ctx->device));
  BH_CUDA(cudaDeviceSynchronize());
  if (DTh) BH_CUDA(cudaMemcpy(DTh, t->DT64, sizeof(double) * t->desc.d_n * t->desc.d_n, cudaMemcpyDeviceToHost));
  if (UTh)
    BH_CUDA(cudaMemcpy(UTh, t->UT64, sizeof(double) * t->desc.u_ne * t->desc.u_nphi, cudaMemcpyDeviceToHost));
  return BH_OK;
}

extern "C" bh_status bh_tables_copy_colour(const bh_tables *t, float *Ch, float *dh) {
  if (!t) { set_error("bh_tables_copy_colour: NULL tables"); return BH_ERR_INVALID_ARG; }
  BH_CUDA(cudaSetDevice(t->ctx->device));
  BH_CUDA(cudaDeviceSynchronize());
  if (Ch) BH_CUDA(cudaMemcpy(Ch, t->C, sizeof(float4) * kCnx * kCny * kCnd, cudaMemcpyDeviceToHost));
  if (dh) BH_CUDA(cudaMemcpy(dh, t->disc, sizeof(float4) * kDiscN, cudaMemcpyDeviceToHost));
  return BH_OK;
}

extern "C" void bh_tables_free(bh_tables *t) {
  if (!t) return;
  cudaSetDevice(t->pool->device);
  pool_put_synced(*t->pool, t->mem);
  delete t;
}
