// Frequency-domain model (Eq. 7): the measurement matrix
//     K(m,n)_i = i c k_n exp(-i k_n |r_i - r_m|) / |r_i - r_m|,   k_n = 2 pi f_n / c,
// at the frequencies f_n = f0 + n df (n < Q), applied to a real image
//     P[m][n] = amp sum_i K(m,n)_i x_i                       (pa_freq_forward)
// and its adjoint for the real inner product Re sum conj(P) Q
//     g_i = amp / d_im sum_{m,n} c k_n Im(exp(i k_n d_im) P[m][n])   (pa_freq_adjoint).
//
// Both run per (pixel tile, sensor) pair.  The phase k_n d is split into the
// tile centre's part k_n d_ref, reduced modulo one cycle in FP64 per (tile,
// sensor, n) (R_n = exp(-i k_n d_ref)), and the pixel's part k_n (d - d_ref),
// whose FP32 error is that of the small difference d - d_ref = (2 e.delta +
// |delta|^2) / (d + d_ref) (e = centre - sensor, delta = pixel - centre): about
// k_n |delta| 2^-24 rad.  Across frequencies the pixel part advances by the
// complex recurrence E_{n+1} = E_n W, W = exp(-i df 2 pi (d - d_ref) / c),
// re-anchored with sincospi every kAnchor steps.
//
// From kMmaForward / kMmaAdjoint frequencies on, reaching phases of kMmaMinSpan
// cycles across a tile, the sums run on the tensor cores (see "tensor-core kernels"
// below); else by the recurrence:
// the adjoint is a gather: each thread accumulates, over the CTA's sensors and
// all frequencies, Im(conj(E_n) B_n) with B_n = c k_n conj(R_n) P[m][n] staged
// in shared memory.  Sensor chunks write partial images summed afterwards in
// chunk order.  The forward sums x_i / d_i E_n over the tile's pixels for
// blocks of kFreqBlock frequencies: each thread keeps its four pixels' sums in
// registers, and the CTA reduces them through shared memory in a fixed order;
// a combine kernel then sums the tiles' spectra R_n S_n in tile order.  No
// atomics: results are bitwise reproducible.
#include <algorithm>
#include <cfloat>
#include <cmath>

#include "pa_internal.cuh"

namespace pa {
namespace {

constexpr int kFreqThreads = 256;    // 4 pixels of a 1024-pixel tile per thread
constexpr int kFreqPPT = kTilePixels / kFreqThreads;
constexpr int kAnchor = 32;          // recurrence steps between exact anchors
constexpr int kFreqBlock = 16;       // frequencies per forward reduction block
constexpr int kFreqSensors = 8;      // sensors per CTA

// Per (tile, sensor) reference of the tensor-core kernels (k_freq_prep).
struct __align__(16) FreqRef {
  float ex, ey, ez, dref;        // tile centre - sensor, and its norm
  unsigned long long ph0, phd;   // f0 d_ref / c and df d_ref / c modulo one cycle, times 2^64
  float dlo;                     // a lower bound of the tile's pixel distances
};

struct FreqParams {
  const double* sensors;  // [S][dim]
  int S, Q, dim;
  int nx, ny, nz, ntx, nty, ntz;
  double dx, dy, dz, ox, oy, oz;
  double c, inv_c, f0, df, amp;
  const float* x;         // forward: [N]
  float2* part;           // forward: [S][ntiles][Q]
  const float2* p;        // adjoint: [S][Q]
  float* gpart;           // adjoint: [n_chunks][N]
  float2* out;            // combine: [S][Q]
  float* gout;            // adjoint sum: [N]
  int n_chunks;
  // tensor-core kernels: work of k_freq_prep and the work split
  FreqRef* refs;          // [ntiles][S]
  float* cks;             // [Q]: c k_n
  int* scales;            // [S]: exponent of the power of two that scales the sensor's spectrum
  int spc;                // adjoint: sensors per CTA
  float inv_cf, f0f, dff, hdx, hdy, hdz;  // in FP32: 1 / c, f0, df, half spacings
};

template <int DIM>
struct TileGeo {
  int tx, ty, tz, nvx, nvy, nvz;
};

template <int DIM>
__device__ __forceinline__ TileGeo<DIM> tile_geo(const FreqParams& P, int tile) {
  constexpr int TX = Tile<DIM>::X, TY = Tile<DIM>::Y, TZ = Tile<DIM>::Z;
  TileGeo<DIM> t;
  t.tx = tile % P.ntx;
  t.ty = (tile / P.ntx) % P.nty;
  t.tz = tile / (P.ntx * P.nty);
  t.nvx = min(TX, P.nx - t.tx * TX);
  t.nvy = min(TY, P.ny - t.ty * TY);
  t.nvz = min(TZ, P.nz - t.tz * TZ);
  return t;
}

// pixel p (row-major within the tile) -> local coordinates
template <int DIM>
__device__ __forceinline__ void local_xyz(int p, int& lx, int& ly, int& lz) {
  constexpr int TX = Tile<DIM>::X, TY = Tile<DIM>::Y;
  lx = p % TX;
  ly = (p / TX) % TY;
  lz = p / (TX * TY);
}

// Per (tile, sensor): e = centre - sensor (FP64) and d_ref = |e|; the centre
// is that of the tile's in-grid pixels.
template <int DIM>
__device__ __forceinline__ void tile_ref(const FreqParams& P, const TileGeo<DIM>& t, int s,
                                         double& ex, double& ey, double& ez, double& dref) {
  constexpr int TX = Tile<DIM>::X, TY = Tile<DIM>::Y, TZ = Tile<DIM>::Z;
  const double cx = P.ox + (t.tx * TX + 0.5 * (t.nvx - 1)) * P.dx;
  const double cy = P.oy + (t.ty * TY + 0.5 * (t.nvy - 1)) * P.dy;
  const double cz = DIM == 3 ? P.oz + (t.tz * TZ + 0.5 * (t.nvz - 1)) * P.dz : 0.0;
  ex = cx - P.sensors[(int64_t)s * P.dim + 0];
  ey = cy - P.sensors[(int64_t)s * P.dim + 1];
  ez = DIM == 3 ? cz - P.sensors[(int64_t)s * P.dim + 2] : 0.0;
  dref = sqrt(ex * ex + ey * ey + ez * ez);
}

// exp(-i 2 pi cycles) for cycles already reduced (|cycles| small)
__device__ __forceinline__ float2 expm2pi(float cycles) {
  float sn, cs;
  sincospif(2.0f * cycles, &sn, &cs);
  return make_float2(cs, -sn);
}

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}

// The pixel part of one (pixel, sensor) pair: 1/d and (d - d_ref) / c.
template <int DIM>
__device__ __forceinline__ void pixel_part(const TileGeo<DIM>& t, int p, float hdx, float hdy,
                                           float hdz, float exf, float eyf, float ezf, float dreff,
                                           float inv_c, float& rinv, float& dt) {
  int lx, ly, lz;
  local_xyz<DIM>(p, lx, ly, lz);
  lx = min(lx, t.nvx - 1);  // ragged edge: a copy of an in-grid pixel (not stored)
  ly = min(ly, t.nvy - 1);
  lz = min(lz, t.nvz - 1);
  const float dx = (float)(2 * lx - (t.nvx - 1)) * hdx;
  const float dy = (float)(2 * ly - (t.nvy - 1)) * hdy;
  const float dz = DIM == 3 ? (float)(2 * lz - (t.nvz - 1)) * hdz : 0.0f;
  const float rx = exf + dx, ry = eyf + dy, rz = ezf + dz;
  const float d2 = fmaf(rx, rx, fmaf(ry, ry, rz * rz));
  rinv = rsqrtf(d2);
  const float d = d2 * rinv;
  const float q = fmaf(2.0f * exf + dx, dx, fmaf(2.0f * eyf + dy, dy, (2.0f * ezf + dz) * dz));
  dt = q / (d + dreff) * inv_c;  // (d - d_ref) / c, seconds
}

constexpr float kHalfMagic = 6291456.0f;  // 1.5 * 2^22: adding it rounds to a multiple of 1/2

__device__ __forceinline__ float2 dup(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }

// cos and sin of 2 pi f d for two (f, d) pairs: the phase is reduced to
// [-1/4, 1/4] cycles by a multiple of 1/2 (subtracted inside the product's FMA,
// so it carries one rounding), then polynomials in r^2 fitted to cos(2 pi r) and
// sin(2 pi r) / r by iteratively reweighted least squares (Lawson 1961);
// absolute error at most 1.5e-7.  |f d| < 2^21.
__device__ __forceinline__ void sincos2(float2 f, float2 d, float2& c, float2& s) {
  const float2 t = fma2(f, d, dup(kHalfMagic));
  const float2 nk = fma2(t, dup(-1.0f), dup(kHalfMagic));
  const float2 r = fma2(f, d, nk);
  const float2 z = mul2(r, r);
  float2 pc = fma2(z, dup(-25.00679588317871f), dup(60.1482048034668f));
  pc = fma2(z, pc, dup(-85.45382690429688f));
  pc = fma2(z, pc, dup(64.9393539428711f));
  pc = fma2(z, pc, dup(-19.739208221435547f));
  pc = fma2(z, pc, dup(1.0f));
  float2 ps = fma2(z, dup(39.76161575317383f), dup(-76.5813980102539f));
  ps = fma2(z, ps, dup(81.60248565673828f));
  ps = fma2(z, ps, dup(-41.34168243408203f));
  ps = fma2(z, ps, dup(6.2831854820251465f));
  ps = mul2(ps, r);
  // an odd multiple of 1/2 flips both signs (the last bit of t)
  const int fx = __float_as_int(t.x) << 31, fy = __float_as_int(t.y) << 31;
  c = make_float2(__int_as_float(__float_as_int(pc.x) ^ fx), __int_as_float(__float_as_int(pc.y) ^ fy));
  s = make_float2(__int_as_float(__float_as_int(ps.x) ^ fx), __int_as_float(__float_as_int(ps.y) ^ fy));
}

// 2^e, e in [-126, 127]
__device__ __forceinline__ float pow2i(int e) { return __int_as_float((e + 127) << 23); }
// The exponent e of a power-of-two scale 2^e that takes values up to mx below
// 2^(top + 1), over the whole range of FP32 (subnormal values, and an mx that
// overflowed, count as the nearest end of it: they still land within FP16's range);
// |e| <= 126, so that 2^e and 2^-e are normal.  0 for mx = 0 or NaN.
__device__ __forceinline__ int scale_exp(float mx, int top) {
  if (!(mx > 0.0f)) return 0;
  const int e = min((__float_as_int(mx) >> 23) & 255, 254) - 127;
  return max(-126, min(126, top - e));
}

// Per (tile, sensor): the geometry that needs FP64 (the FP64 pipe takes 64
// cycles per warp instruction: evaluated by every warp of the gathers it cost
// them 80 us at 256^2 and 256 sensors, whatever the number of frequencies; here
// 3 us), with the tile centre's
// phase per Hz as fractions of a cycle in units of 2^-64: exp(-i k_n d_ref) =
// exp(-2 pi i (ph0 + n phd) 2^-64), exact modulo one cycle in integer arithmetic.
template <int DIM>
__global__ void __launch_bounds__(kFreqThreads) k_freq_prep(const FreqParams P, int nb_ref,
                                                            int nb_ck) {
  const int b = blockIdx.x;
  if (b < nb_ref) {
    const int64_t idx = (int64_t)b * kFreqThreads + threadIdx.x;
    if (idx >= (int64_t)P.ntx * P.nty * P.ntz * P.S) return;
    const int tile = (int)(idx / P.S), s = (int)(idx % P.S);
    const TileGeo<DIM> t = tile_geo<DIM>(P, tile);
    double e[3], dref;
    tile_ref<DIM>(P, t, s, e[0], e[1], e[2], dref);
    const double a = dref * P.inv_c;
    double c0 = P.f0 * a, cd = P.df * a;
    c0 -= floor(c0);
    cd -= floor(cd);
    // distance from the sensor to the box of the tile's pixel centres
    const double hx = 0.5 * (t.nvx - 1) * P.dx, hy = 0.5 * (t.nvy - 1) * P.dy;
    const double hz = DIM == 3 ? 0.5 * (t.nvz - 1) * P.dz : 0.0;
    const double qx = fmax(fabs(e[0]) - hx, 0.0), qy = fmax(fabs(e[1]) - hy, 0.0);
    const double qz = fmax(fabs(e[2]) - hz, 0.0);
    const double hmin = DIM == 3 ? fmin(P.dx, fmin(P.dy, P.dz)) : fmin(P.dx, P.dy);
    FreqRef r;
    r.ex = (float)e[0];
    r.ey = (float)e[1];
    r.ez = (float)e[2];
    r.dref = (float)dref;
    r.ph0 = (unsigned long long)(c0 * 18446744073709551616.0);
    r.phd = (unsigned long long)(cd * 18446744073709551616.0);
    r.dlo = (float)fmax(sqrt(qx * qx + qy * qy + qz * qz), 0.45 * hmin);
    P.refs[idx] = r;
  } else if (b < nb_ref + nb_ck) {
    const int n = (b - nb_ref) * kFreqThreads + threadIdx.x;
    if (n < P.Q) P.cks[n] = (float)(2.0 * M_PI * (P.f0 + n * P.df));  // c k_n
  } else {
    // adjoint: one warp per sensor finds the scale of its spectrum c k_n P[m][n]
    const int s = (b - nb_ref - nb_ck) * (kFreqThreads / 32) + (threadIdx.x >> 5);
    if (s >= P.S) return;
    const float f0 = (float)P.f0, fdf = (float)P.df;
    float mx = 0.0f;
    int bad = 0;
    for (int n = threadIdx.x & 31; n < P.Q; n += 32) {
      const float2 v = P.p[(int64_t)s * P.Q + n];
      const float m = 6.2831855f * fmaf((float)n, fdf, f0) * fmaxf(fabsf(v.x), fabsf(v.y));
      bad |= !(fabsf(v.x) <= FLT_MAX) || !(fabsf(v.y) <= FLT_MAX);
      mx = fmaxf(mx, m);
    }
    mx = __int_as_float(__reduce_max_sync(0xffffffffu, __float_as_int(mx)));
    bad = __any_sync(0xffffffffu, bad);
    if ((threadIdx.x & 31) == 0) P.scales[s] = bad ? 0 : scale_exp(mx, 9);
  }
}

// exp(-2 pi i (ph0 + n phd) 2^-64) as (cos, sin of the reduced phase, positive sign)
__device__ __forceinline__ float2 centre_phase(unsigned long long ph0, unsigned long long phd,
                                               int n) {
  const unsigned long long ph = ph0 + (unsigned long long)n * phd;
  const float r = (float)(int)(unsigned)(ph >> 32) * 2.3283064365386963e-10f;
  const float2 e = expm2pi(r);
  return make_float2(e.x, -e.y);
}

// ------------------------------- adjoint ---------------------------------
template <int DIM>
__global__ void __launch_bounds__(kFreqThreads) k_freq_adjoint(const FreqParams P) {
  extern __shared__ __align__(16) unsigned char smem[];
  float2* sB = reinterpret_cast<float2*>(smem);  // [Q] per sensor
  const int tile = blockIdx.y, chunk = blockIdx.x;
  const TileGeo<DIM> t = tile_geo<DIM>(P, tile);
  const int s0 = chunk * kFreqSensors, s1 = min(P.S, s0 + kFreqSensors);
  const float hdx = P.hdx, hdy = P.hdy, hdz = P.hdz, inv_c = P.inv_cf, f0 = P.f0f, fdf = P.dff;
  float acc[kFreqPPT];
#pragma unroll
  for (int m = 0; m < kFreqPPT; ++m) acc[m] = 0.0f;
  for (int s = s0; s < s1; ++s) {
    const FreqRef r = P.refs[(int64_t)tile * P.S + s];
    __syncthreads();  // the previous sensor's B is consumed
    for (int n = threadIdx.x; n < P.Q; n += kFreqThreads) {
      const float2 pv = P.p[(int64_t)s * P.Q + n];
      const float ck = P.cks[n];
      const float2 b = cmul(centre_phase(r.ph0, r.phd, n), pv);  // conj(R_n) P
      sB[n] = make_float2(ck * b.x, ck * b.y);
    }
    __syncthreads();
    const float exf = r.ex, eyf = r.ey, ezf = r.ez, dreff = r.dref;
#pragma unroll
    for (int m = 0; m < kFreqPPT; ++m) {
      float rinv, dt;
      pixel_part<DIM>(t, threadIdx.x + m * kFreqThreads, hdx, hdy, hdz, exf, eyf, ezf, dreff,
                      inv_c, rinv, dt);
      const float2 W = expm2pi(fdf * dt);
      float v = 0.0f;
      for (int n0 = 0; n0 < P.Q; n0 += kAnchor) {
        float2 E = expm2pi(fmaf((float)n0, fdf, f0) * dt);  // exp(-i 2 pi f_n (d - d_ref) / c)
        const int n1 = min(P.Q, n0 + kAnchor);
        for (int n = n0; n < n1; ++n) {
          const float2 b = sB[n];
          v = fmaf(E.x, b.y, fmaf(-E.y, b.x, v));  // Im(conj(E) B)
          E = cmul(E, W);
        }
      }
      acc[m] = fmaf(v, rinv, acc[m]);
    }
  }
  constexpr int TX = Tile<DIM>::X, TY = Tile<DIM>::Y, TZ = Tile<DIM>::Z;
#pragma unroll
  for (int m = 0; m < kFreqPPT; ++m) {
    int lx, ly, lz;
    local_xyz<DIM>(threadIdx.x + m * kFreqThreads, lx, ly, lz);
    if (lx < t.nvx && ly < t.nvy && lz < t.nvz) {
      const int64_t i = ((int64_t)(t.tz * TZ + lz) * P.ny + (t.ty * TY + ly)) * P.nx + (t.tx * TX + lx);
      P.gpart[(int64_t)chunk * P.nx * P.ny * P.nz + i] = acc[m];
    }
  }
}

__global__ void __launch_bounds__(kFreqThreads) k_freq_adjoint_sum(const FreqParams P,
                                                                   int64_t N) {
  const int64_t i = blockIdx.x * (int64_t)kFreqThreads + threadIdx.x;
  if (i >= N) return;
  float v = 0.0f;
  for (int c = 0; c < P.n_chunks; ++c) v += P.gpart[(int64_t)c * N + i];
  P.gout[i] = (float)P.amp * v;
}

// ------------------------------- forward ---------------------------------
template <int DIM>
__global__ void __launch_bounds__(kFreqThreads) k_freq_forward(const FreqParams P) {
  __shared__ float2 sacc[kFreqBlock][kFreqThreads + 1];
  extern __shared__ __align__(16) unsigned char smem[];
  float2* sR = reinterpret_cast<float2*>(smem);  // [Q]: exp(-i k_n d_ref) of the sensor
  const int tile = blockIdx.y, chunk = blockIdx.x;
  const TileGeo<DIM> t = tile_geo<DIM>(P, tile);
  const int s0 = chunk * kFreqSensors, s1 = min(P.S, s0 + kFreqSensors);
  const float hdx = P.hdx, hdy = P.hdy, hdz = P.hdz, inv_c = P.inv_cf, f0 = P.f0f, fdf = P.dff;
  constexpr int TX = Tile<DIM>::X, TY = Tile<DIM>::Y, TZ = Tile<DIM>::Z;
  float xv[kFreqPPT];
#pragma unroll
  for (int m = 0; m < kFreqPPT; ++m) {
    int lx, ly, lz;
    local_xyz<DIM>(threadIdx.x + m * kFreqThreads, lx, ly, lz);
    xv[m] = 0.0f;
    if (lx < t.nvx && ly < t.nvy && lz < t.nvz)
      xv[m] = P.x[((int64_t)(t.tz * TZ + lz) * P.ny + (t.ty * TY + ly)) * P.nx + (t.tx * TX + lx)];
  }
  for (int s = s0; s < s1; ++s) {
    const FreqRef r = P.refs[(int64_t)tile * P.S + s];
    __syncthreads();  // the previous sensor's sR is consumed
    for (int n = threadIdx.x; n < P.Q; n += kFreqThreads) {
      const float2 R = centre_phase(r.ph0, r.phd, n);
      sR[n] = make_float2(R.x, -R.y);
    }
    __syncthreads();
    const float exf = r.ex, eyf = r.ey, ezf = r.ez, dreff = r.dref;
    float a[kFreqPPT], dt[kFreqPPT];
    float2 W[kFreqPPT];
#pragma unroll
    for (int m = 0; m < kFreqPPT; ++m) {
      float rinv;
      pixel_part<DIM>(t, threadIdx.x + m * kFreqThreads, hdx, hdy, hdz, exf, eyf, ezf, dreff,
                      inv_c, rinv, dt[m]);
      a[m] = xv[m] * rinv;
      W[m] = expm2pi(fdf * dt[m]);
    }
    for (int n0 = 0; n0 < P.Q; n0 += kFreqBlock) {
      // this thread's four pixels, kFreqBlock frequencies from n0 (anchored at
      // n0, which is a multiple of kFreqBlock and so of the anchor spacing)
      float2 sum[kFreqBlock];
#pragma unroll
      for (int j = 0; j < kFreqBlock; ++j) sum[j] = make_float2(0.0f, 0.0f);
#pragma unroll
      for (int m = 0; m < kFreqPPT; ++m) {
        float2 E = expm2pi(fmaf((float)n0, fdf, f0) * dt[m]);
#pragma unroll
        for (int j = 0; j < kFreqBlock; ++j) {
          sum[j].x = fmaf(a[m], E.x, sum[j].x);
          sum[j].y = fmaf(a[m], E.y, sum[j].y);
          E = cmul(E, W[m]);
        }
      }
#pragma unroll
      for (int j = 0; j < kFreqBlock; ++j) sacc[j][threadIdx.x] = sum[j];
      __syncthreads();
      // frequency j = thread / 16 summed by 16 threads (16 values each, lane
      // `part` taking the threads part, part + 16, ...: consecutive lanes read
      // consecutive entries, so a half-warp's loads fill distinct banks), then
      // a fixed xor tree over those 16 lanes
      const int j = threadIdx.x >> 4, part = threadIdx.x & 15;
      float2 v = make_float2(0.0f, 0.0f);
#pragma unroll
      for (int q = 0; q < kFreqThreads / 16; ++q) {
        const float2 w = sacc[j][q * 16 + part];
        v.x += w.x;
        v.y += w.y;
      }
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
      }
      const int n = n0 + j;
      if (part == 0 && n < P.Q)
        P.part[((int64_t)s * (P.ntx * P.nty * P.ntz) + tile) * P.Q + n] = cmul(sR[n], v);
      __syncthreads();  // sacc is reused by the next block
    }
  }
}

// ------------------------ tensor-core kernels ----------------------------
// With n = n0 + 16 a + b (a, b < 16; blocks of 256 frequencies) the pixel part
// of the phase factors, exp(+-2 pi i f_n dt_i) = U_ia V_ib with
//     U_ia = exp(+-2 pi i (f0 + (n0 + 16 a) df) dt_i),  V_ib = exp(+-2 pi i b df dt_i),
// so a (tile, sensor) pair is a matrix product over 32 generated factors per
// pixel instead of a 256-step recurrence:
//   forward  S_ab = sum_i (x_i / d_i U_ia) V_ib        (contraction over pixels),
//   adjoint  v_i  = sum_a Im(U_ia sum_b V_ib B_ab)     (contraction over b).
// Operands go to mma.sync as FP16 pairs hi + lo (22 significant bits of a
// factor of modulus at most 1; x / d and B scaled by a power of two per (tile,
// sensor) and per sensor), three products hi hi + hi lo + lo hi.  An MMA adds to its
// accumulator without rounding to nearest, so the forward's partial sums leave the
// tensor core after every 16 pixels and are added in FP32.  The factors come from
// one sine and cosine of a phase reduced with one rounding and at most three complex
// products (the recurrence multiplies up to 32), so the error against FP64 stays
// that of the FP32 dt: 5.1e-6 at 256 frequencies up to 20 MHz (96 x 75 pixels of
// 0.1 mm) in the forward and 4.9e-6 in the adjoint, against 6.4e-6 and 6.1e-6 with
// the recurrence; at 128 frequencies up to 2 MHz 5.5e-7 and 5.3e-7 against 5.8e-7
// and 6.5e-7; 5.7e-6 against 6.0e-6 for a positive image up to 20 MHz, and 2e-7 in
// its lowest rows with both.  (With sums kept in the tensor core over 128
// pixels, and hi cut in both operands, sums of like terms were off by 2e-6 at any
// frequency.)
//
// What bounds them: issue slots.  Per 16 pixels and sensor a warp issues about
// 200 instructions for the factors, their splits and the dot products (220 with the
// forward's sums), and 24 MMAs, each of which holds the issue port for about 8 cycles
// (a loop of one m16n8k16 with 4 or 8 independent FFMAs takes 11.6 and 15.9 cycles
// per step, 8.1 without them); the two add up to 86-89% of the cycles.  256^2 ring,
// 256 sensors, 256 frequencies: forward 1474 -> 553 us, adjoint 1269 -> 429 us.
struct C2 {  // two complex numbers
  float2 re, im;
};
__device__ __forceinline__ C2 cmul2(C2 a, C2 b, float2 nbi) {  // nbi = -b.im
  return C2{fma2(a.im, nbi, mul2(a.re, b.re)), fma2(a.re, b.im, mul2(a.im, b.re))};
}

__device__ __forceinline__ uint32_t h2_bits(__half2 h) {
  return *reinterpret_cast<uint32_t*>(&h);
}
// v as FP16 pairs hi + lo, v.x in the low half: hi is v cut to 11 significant
// bits (an AND on the ALU pipe: the FMA pipe, which converting hi back would
// use, is the one that limits these kernels), lo = fp16(v - hi), so hi + lo
// holds v to 2^-22 (and to 2^-25 absolutely).
__device__ __forceinline__ float cut(float v) {
  return __int_as_float(__float_as_int(v) & 0xffffe000);
}
__device__ __forceinline__ uint32_t pack_h2(float lo, float hi) {
  return h2_bits(__floats2half2_rn(lo, hi));
}
__device__ __forceinline__ void split(float2 v, uint32_t& hi, uint32_t& lo) {
  const float2 h = make_float2(cut(v.x), cut(v.y));
  const float2 r = fma2(h, dup(-1.0f), v);
  hi = pack_h2(h.x, h.y);
  lo = pack_h2(r.x, r.y);
}
// The same with hi rounded to nearest, so that lo carries no sign of its own: one
// operand of each product is split this way, or the dropped lo lo products, all of
// one sign, would add up in a sum of like terms.
__device__ __forceinline__ void split_rn(float2 v, uint32_t& hi, uint32_t& lo) {
  const __half2 h = __floats2half2_rn(v.x, v.y);
  const float2 r = fma2(__half22float2(h), dup(-1.0f), v);
  hi = h2_bits(h);
  lo = pack_h2(r.x, r.y);
}
// two complex numbers: (re, im) of number x and of number y
__device__ __forceinline__ void split_c2(C2 v, uint32_t& hx, uint32_t& hy, uint32_t& lx,
                                         uint32_t& ly) {
  const float2 hr = make_float2(cut(v.re.x), cut(v.re.y)), hi = make_float2(cut(v.im.x), cut(v.im.y));
  const float2 re = fma2(hr, dup(-1.0f), v.re), im = fma2(hi, dup(-1.0f), v.im);
  hx = pack_h2(hr.x, hi.x);
  hy = pack_h2(hr.y, hi.y);
  lx = pack_h2(re.x, im.x);
  ly = pack_h2(re.y, im.y);
}

__device__ __forceinline__ void mma_f16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                        uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// d - d_ref over c, and 1/d, of two pixels (offsets dx, dy, dz from the tile centre)
template <int DIM>
__device__ __forceinline__ void pixel_part2(float2 dx, float2 dy, float2 dz, const FreqRef& r,
                                            float inv_c, float2& rinv, float2& dt) {
  const float2 rx = add2(dup(r.ex), dx), ry = add2(dup(r.ey), dy);
  const float2 qx = fma2(dup(2.0f), dup(r.ex), dx), qy = fma2(dup(2.0f), dup(r.ey), dy);
  float2 d2 = mul2(ry, ry), q = mul2(qy, dy);
  if (DIM == 3) {
    const float2 rz = add2(dup(r.ez), dz), qz = fma2(dup(2.0f), dup(r.ez), dz);
    d2 = fma2(ry, ry, mul2(rz, rz));
    q = fma2(qy, dy, mul2(qz, dz));
  }
  d2 = fma2(rx, rx, d2);
  q = fma2(qx, dx, q);
  rinv = make_float2(rsqrtf(d2.x), rsqrtf(d2.y));
  const float2 den = fma2(d2, rinv, dup(r.dref));
  dt = mul2(make_float2(__fdiv_rn(q.x, den.x), __fdiv_rn(q.y, den.y)), dup(inv_c));
}

// offsets of pixel p (row-major within the tile) from the tile centre
template <int DIM>
__device__ __forceinline__ void pixel_offsets(const TileGeo<DIM>& t, int p, float hdx, float hdy,
                                              float hdz, float& dx, float& dy, float& dz) {
  int lx, ly, lz;
  local_xyz<DIM>(p, lx, ly, lz);
  lx = min(lx, t.nvx - 1);  // ragged edge: a copy of an in-grid pixel (not stored)
  ly = min(ly, t.nvy - 1);
  lz = min(lz, t.nvz - 1);
  dx = (float)(2 * lx - (t.nvx - 1)) * hdx;
  dy = (float)(2 * ly - (t.nvy - 1)) * hdy;
  dz = DIM == 3 ? (float)(2 * lz - (t.nvz - 1)) * hdz : 0.0f;
}

// Adjoint.  CTA: one tile, P.spc sensors; warp w owns pixels 128 w .. 128 w + 127
// as eight 16-row MMA tiles (rows g and g + 8 of lane 4 g + t).  Lane t of a row
// generates V_ib for b = t, t + 4, t + 8, t + 12 (the A fragment's columns are
// (Re, Im) pairs in b) and U_ia for a = t + 4 j, the columns of its accumulators
// of n-tile j.  B fragments of a (sensor, frequency block) are staged in shared
// memory in fragment order, double-buffered, and held in registers over the
// warp's eight row tiles.  Per pixel and sensor the owner lane evaluates dt, 1/d
// and the two steps exp(2 pi i 4 df dt), exp(2 pi i 64 df dt) once.
constexpr int kFreqFragWords = 32 * 32;
template <int DIM, int NJ>
__global__ void __launch_bounds__(kFreqThreads, 3) k_freq_adjoint_mma(const FreqParams P) {
  extern __shared__ __align__(16) unsigned char smem[];
  uint32_t* sB = reinterpret_cast<uint32_t*>(smem);                       // [2][32 regs][32 lanes]
  float* sP = reinterpret_cast<float*>(sB + 2 * kFreqFragWords);          // [8 warps][6][128]
  float2* sA = reinterpret_cast<float2*>(sP + 8 * 6 * 128);               // [8 groups][256]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t = lane & 3;
  const int tile = blockIdx.y, chunk = blockIdx.x;
  const TileGeo<DIM> tg = tile_geo<DIM>(P, tile);
  const int s0 = chunk * P.spc, s1 = min(P.S, s0 + P.spc);
  const int nblk = (P.Q + 255) / 256, n_it = (s1 - s0) * nblk;
  const float inv_c = P.inv_cf, f0 = P.f0f, fdf = P.dff;
  float2 ox[2], oy[2], oz[2];  // the lane's own pixels 128 w + lane + 32 k, k = 2 m + (0, 1)
  {
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      const int p = warp * 128 + lane + 64 * m;
      pixel_offsets<DIM>(tg, p, P.hdx, P.hdy, P.hdz, ox[m].x, oy[m].x, oz[m].x);
      pixel_offsets<DIM>(tg, p + 32, P.hdx, P.hdy, P.hdz, ox[m].y, oy[m].y, oz[m].y);
    }
  }
#pragma unroll
  for (int gr = 0; gr < 8; ++gr) sA[gr * 256 + tid] = make_float2(0.0f, 0.0f);

  // B_n = 2^scale c k_n conj(R_n) P[m][n] as fragments: element (k = (b, part of
  // V), column (a, part of T)): T.re = Vr Br - Vi Bi, T.im = Vr Bi + Vi Br
  auto stage = [&](int it) {
    const int s = s0 + it / nblk, n = (it % nblk) * 256 + tid;
    float br = 0.0f, bi = 0.0f;
    if (n < P.Q) {
      const FreqRef& r = P.refs[(int64_t)tile * P.S + s];
      const float2 R = centre_phase(r.ph0, r.phd, n);  // conj(R_n) = R.x + i R.y
      const float2 pv = P.p[(int64_t)s * P.Q + n];
      const float ck = P.cks[n], scale = pow2i(P.scales[s]);
      const float2 b = cmul(R, pv);
      br = (ck * b.x) * scale;  // ck scale alone may be too large
      bi = (ck * b.y) * scale;
    }
    const int a = tid >> 4, b = tid & 15;
    const int ks = b >> 3, bk = (b >> 2) & 1, j = a >> 2;
    uint32_t hi0, lo0, hi1, lo1;
    split_rn(make_float2(br, -bi), hi0, lo0);
    split_rn(make_float2(bi, br), hi1, lo1);
    uint32_t* buf = sB + (it & 1) * kFreqFragWords;
    const int idx = ks * 8 + j * 2 + bk, ln = 8 * (a & 3) + (b & 3);  // lanes of columns 2a', 2a'+1
    const int w0 = ((idx >> 2) * 32 + ln) * 4 + (idx & 3);
    buf[w0] = hi0;
    buf[w0 + 16] = hi1;
    buf[w0 + 512] = lo0;
    buf[w0 + 512 + 16] = lo1;
  };
  if (n_it > 0) stage(0);
  float* wp = sP + warp * 6 * 128;
  for (int it = 0; it < n_it; ++it) {
    __syncthreads();  // buffer `it` is staged; buffer it - 1 is consumed
    if (it + 1 < n_it) stage(it + 1);
    const int s = s0 + it / nblk, n0 = (it % nblk) * 256;
    if (n0 == 0) {
      const FreqRef r = P.refs[(int64_t)tile * P.S + s];
      __syncwarp();
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        float2 rinv, dt;
        pixel_part2<DIM>(ox[m], oy[m], oz[m], r, inv_c, rinv, dt);
        float2 vr, vi, ur, ui;
        sincos2(dup(4.0f * fdf), dt, vr, vi);
        sincos2(dup(64.0f * fdf), dt, ur, ui);
        // rows g and g + 8 of a 16-pixel group are neighbours: one 8-byte load
        const int q = lane & 15;
        const int o = ((lane >> 4) + 4 * m) * 16 + 2 * (q & 7) + (q >> 3);
        wp[o] = dt.x, wp[o + 32] = dt.y;
        wp[128 + o] = rinv.x, wp[128 + o + 32] = rinv.y;
        wp[256 + o] = vr.x, wp[256 + o + 32] = vr.y;
        wp[384 + o] = vi.x, wp[384 + o + 32] = vi.y;
        wp[512 + o] = ur.x, wp[512 + o + 32] = ur.y;
        wp[640 + o] = ui.x, wp[640 + o + 32] = ui.y;
      }
      __syncwarp();
    }
    const uint4* sBf = reinterpret_cast<const uint4*>(sB + (it & 1) * kFreqFragWords) + lane;
    const float2 isc = dup(pow2i(-P.scales[s]));
    const float2 fv = dup((float)t * fdf), fu = dup(fmaf((float)(n0 + 16 * t), fdf, f0));
#pragma unroll 1
    for (int gr = 0; gr < 8; ++gr) {
      const int o = gr * 16 + 2 * g;
      auto ld = [&](int k) { return *reinterpret_cast<const float2*>(wp + k * 128 + o); };
      const float2 dt = ld(0);
      C2 V, U;
      uint32_t Ah[2][4], Al[2][4];
      {
        const C2 V4{ld(2), ld(3)};
        const float2 nv = neg2(V4.im);
        sincos2(fv, dt, V.re, V.im);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int ks = q >> 1, bk = 2 * (q & 1);
          split_c2(V, Ah[ks][bk], Ah[ks][bk + 1], Al[ks][bk], Al[ks][bk + 1]);
          if (q < 3) V = cmul2(V, V4, nv);
        }
      }
      float C[NJ][4];
#pragma unroll
      for (int j = 0; j < NJ; ++j) C[j][0] = C[j][1] = C[j][2] = C[j][3] = 0.0f;
#pragma unroll
      for (int ks = 0; ks < 2; ++ks)
#pragma unroll
        for (int jj = 0; jj < (NJ + 1) / 2; ++jj) {  // n-tiles 2 jj and 2 jj + 1
          const uint4 bh = sBf[(2 * ks + jj) * 32], bl = sBf[(4 + 2 * ks + jj) * 32];
          constexpr bool two = NJ > 1;
          float(&c1)[4] = C[two ? 2 * jj + 1 : 0];
          mma_f16(C[2 * jj], Al[ks], bh.x, bh.y);
          if (two) mma_f16(c1, Al[ks], bh.z, bh.w);
          mma_f16(C[2 * jj], Ah[ks], bl.x, bl.y);
          if (two) mma_f16(c1, Ah[ks], bl.z, bl.w);
          mma_f16(C[2 * jj], Ah[ks], bh.x, bh.y);
          if (two) mma_f16(c1, Ah[ks], bh.z, bh.w);
        }
      const C2 U4{ld(4), ld(5)};
      const float2 nu = neg2(U4.im);
      sincos2(fu, dt, U.re, U.im);
      float2 v = make_float2(0.0f, 0.0f);
#pragma unroll
      for (int j = 0; j < NJ; ++j) {  // Im(U T)
        v.x = fmaf(U.re.x, C[j][1], fmaf(U.im.x, C[j][0], v.x));
        v.y = fmaf(U.re.y, C[j][3], fmaf(U.im.y, C[j][2], v.y));
        if (j < NJ - 1) U = cmul2(U, U4, nu);
      }
      sA[gr * 256 + tid] = fma2(mul2(v, ld(1)), isc, sA[gr * 256 + tid]);
    }
  }
  constexpr int TX = Tile<DIM>::X, TY = Tile<DIM>::Y, TZ = Tile<DIM>::Z;
#pragma unroll 1
  for (int gr = 0; gr < 8; ++gr) {  // the four lanes of a row in a fixed tree
    float2 a = sA[gr * 256 + tid];
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
      a.x += __shfl_xor_sync(0xffffffffu, a.x, o);
      a.y += __shfl_xor_sync(0xffffffffu, a.y, o);
    }
    if (t < 2) {  // lane t = 0 stores row g, t = 1 row g + 8
      int lx, ly, lz;
      local_xyz<DIM>(warp * 128 + gr * 16 + g + 8 * t, lx, ly, lz);
      if (lx < tg.nvx && ly < tg.nvy && lz < tg.nvz) {
        const int64_t i =
            ((int64_t)(tg.tz * TZ + lz) * P.ny + (tg.ty * TY + ly)) * P.nx + (tg.tx * TX + lx);
        P.gpart[(int64_t)chunk * P.nx * P.ny * P.nz + i] = t == 0 ? a.x : a.y;
      }
    }
  }
}
constexpr int kFreqAdjSmem = 2 * kFreqFragWords * 4 + 8 * 6 * 128 * 4 + 8 * 256 * 8;

// Forward.  CTA: one (tile, sensor) pair, 128 pixels per warp, the warps' sums added
// in order.  Rows of the A operand are (Re, Im) of x / d U_ia (16-row tile mt: Re of
// a = 8 mt + g in row g, Im in row g + 8), columns of B are (Re, Im) of V_ib, k runs
// over 16 pixels: lane 4 g + t generates a, b = g and g + 8 for pixels 2t, 2t + 1,
// 2t + 8, 2t + 9.  MT = 1 covers up to 128 frequencies per block (a < 8), three CTAs
// per SM (434 -> 419 us at 128 frequencies); MT = 2 up to 256, two (three spill: 564
// against 550 us).
template <int DIM, int MT>
__global__ void __launch_bounds__(kFreqThreads, MT == 1 ? 3 : 2)
    k_freq_forward_mma(const FreqParams P) {
  extern __shared__ __align__(16) unsigned char smem[];
  float* sX = reinterpret_cast<float*>(smem);          // [1024]
  float* sP = sX + kTilePixels;                        // [8 warps][6][32]
  float* sR = sP + 8 * 6 * 32;                         // [8 warps][16 MT regs][32 lanes]
  __shared__ float s_max[kFreqThreads / 32];
  constexpr int TX = Tile<DIM>::X, TY = Tile<DIM>::Y, TZ = Tile<DIM>::Z;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t = lane & 3;
  const int tile = blockIdx.y, ntiles = P.ntx * P.nty * P.ntz;
  const TileGeo<DIM> tg = tile_geo<DIM>(P, tile);
  float mx = 0.0f;
  int bad = 0;
  for (int p = tid; p < kTilePixels; p += kFreqThreads) {
    int lx, ly, lz;
    local_xyz<DIM>(p, lx, ly, lz);
    float v = 0.0f;
    if (lx < tg.nvx && ly < tg.nvy && lz < tg.nvz)
      v = P.x[((int64_t)(tg.tz * TZ + lz) * P.ny + (tg.ty * TY + ly)) * P.nx + (tg.tx * TX + lx)];
    sX[p] = v;
    mx = fmaxf(mx, fabsf(v));
    bad |= !(fabsf(v) <= FLT_MAX);
  }
  mx = __int_as_float(__reduce_max_sync(0xffffffffu, __float_as_int(mx)));
  if (lane == 0) s_max[warp] = mx;
  bad = __syncthreads_or(bad);
#pragma unroll
  for (int w = 0; w < kFreqThreads / 32; ++w) mx = fmaxf(mx, s_max[w]);
  const int s = blockIdx.x;
  const float inv_c = P.inv_cf, f0 = P.f0f, fdf = P.dff;
  const FreqRef r = P.refs[(int64_t)tile * P.S + s];
  const int sc = bad ? 0 : scale_exp(__fdiv_rn(mx, r.dlo), 4);  // |x| / d <= mx / dlo
  const float scale = pow2i(sc), iscale = pow2i(-sc);
  float* wp = sP + warp * 6 * 32;
  constexpr int kBlk = 128 * MT;
  for (int n0 = 0; n0 < P.Q; n0 += kBlk) {
    float2 acc[MT][4][2];
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[m][j][0] = acc[m][j][1] = dup(0.0f);
    const float2 fu = dup(-fmaf((float)(n0 + 16 * g), fdf, f0)), fv = dup(-(float)g * fdf);
    if (mx > 0.0f || bad) {
#pragma unroll 1
      for (int gp = 4 * warp; gp < 4 * warp + 4; ++gp) {
        {  // each lane its own pixel of 32
          const int p = gp * 32 + lane;
          float dx, dy, dz;
          pixel_offsets<DIM>(tg, p, P.hdx, P.hdy, P.hdz, dx, dy, dz);
          float2 rinv, dt;
          pixel_part2<DIM>(dup(dx), dup(dy), dup(dz), r, inv_c, rinv, dt);
          float2 c, sn;  // steps of eight in a and in b
          sincos2(make_float2(-128.0f * fdf, -8.0f * fdf), dt, c, sn);
          __syncwarp();
          wp[lane] = dt.x;
          wp[32 + lane] = (sX[p] * scale) * rinv.x;  // scale alone may be too large
          wp[64 + lane] = c.x;
          wp[96 + lane] = sn.x;
          wp[128 + lane] = c.y;
          wp[160 + lane] = sn.y;
          __syncwarp();
        }
#pragma unroll
        for (int gr = 0; gr < 2; ++gr) {
          uint32_t Ah[MT][4], Al[MT][4];
          C2 V[2], W[2];
          auto ld = [&](int k, int h) {
            return *reinterpret_cast<const float2*>(wp + 32 * k + gr * 16 + 8 * h + 2 * t);
          };
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const float2 dt = ld(0, h), xc = ld(1, h);
            C2 U;
            sincos2(fu, dt, U.re, U.im);
            U.re = mul2(U.re, xc);
            U.im = mul2(U.im, xc);
            split_rn(U.re, Ah[0][2 * h], Al[0][2 * h]);
            split_rn(U.im, Ah[0][2 * h + 1], Al[0][2 * h + 1]);
            if (MT == 2) {
              const C2 U8{ld(2, h), ld(3, h)};
              U = cmul2(U, U8, neg2(U8.im));
              split_rn(U.re, Ah[MT - 1][2 * h], Al[MT - 1][2 * h]);
              split_rn(U.im, Ah[MT - 1][2 * h + 1], Al[MT - 1][2 * h + 1]);
            }
            sincos2(fv, dt, V[h].re, V[h].im);
            const C2 V8{ld(4, h), ld(5, h)};
            W[h] = cmul2(V[h], V8, neg2(V8.im));
          }
          auto col = [&](int j, float2 v0, float2 v1) {
            uint32_t h0, l0, h1, l1;
            split(v0, h0, l0);
            split(v1, h1, l1);
            float d[MT][4] = {};  // the products of these 16 pixels alone
#pragma unroll
            for (int m = 0; m < MT; ++m) mma_f16(d[m], Al[m], h0, h1);
#pragma unroll
            for (int m = 0; m < MT; ++m) mma_f16(d[m], Ah[m], l0, l1);
#pragma unroll
            for (int m = 0; m < MT; ++m) mma_f16(d[m], Ah[m], h0, h1);
#pragma unroll
            for (int m = 0; m < MT; ++m) {
              acc[m][j][0] = add2(acc[m][j][0], make_float2(d[m][0], d[m][1]));
              acc[m][j][1] = add2(acc[m][j][1], make_float2(d[m][2], d[m][3]));
            }
          };
          col(0, V[0].re, V[1].re);
          col(1, V[0].im, V[1].im);
          col(2, W[0].re, W[1].re);
          col(3, W[0].im, W[1].im);
        }
      }
    }
    // the warps' sums in order, one output per thread (warp = (m, bh, e))
    __syncthreads();  // the previous block's sums are read
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e)
          sR[(warp * 16 * MT + (m * 4 + j) * 4 + e) * 32 + lane] =
              e & 1 ? acc[m][j][e >> 1].y : acc[m][j][e >> 1].x;
    __syncthreads();
    if (warp < 4 * MT) {
      const int m = warp >> 2, bh = (warp >> 1) & 1, e = warp & 1;
      const int n = n0 + 16 * (8 * m + g) + 8 * bh + 2 * t + e;
      const float* q = sR + (m * 16 + 8 * bh + e) * 32 + lane;  // Re U Re V; + 2: Im U Re V; ...
      float rr = 0.0f, ir = 0.0f, ri = 0.0f, ii = 0.0f;
#pragma unroll
      for (int w = 0; w < 8; ++w, q += 16 * MT * 32) {
        rr += q[0];
        ir += q[2 * 32];
        ri += q[4 * 32];
        ii += q[6 * 32];
      }
      if (n < P.Q) {
        const float2 R = centre_phase(r.ph0, r.phd, n);
        const float2 v = cmul(make_float2(R.x, -R.y), make_float2(rr - ii, ri + ir));
        P.part[((int64_t)s * ntiles + tile) * P.Q + n] = make_float2(iscale * v.x, iscale * v.y);
      }
    }
  }
}
int freq_fwd_smem(int mt) {
  return (kTilePixels + 8 * 6 * 32 + 8 * 16 * mt * 32) * (int)sizeof(float);
}

// The matrix kernels' cost per (pixel, sensor) pair does not depend on Q up to a
// block of 128 (forward) or 64 (one n-tile of the adjoint); with few frequencies
// the recurrence is cheaper.  256^2 ring, recurrence against matrix kernel:
// forward 382 / 425 us at 64 frequencies, 621 / 425 at 100; adjoint 206 / 261 us
// at 32, 294 / 262 at 48.  (On small grids the matrix kernels win at any count,
// by at most 30%: 64^2, 64 sensors, 32 frequencies: 25 against 37 us.)
constexpr int kMmaForward = 72, kMmaAdjoint = 44;
// They also take over only where the phases of a tile's pixels span a few cycles at
// the highest frequency.  Below, the FP32 dt no longer dominates the error, and with
// few roundings per term the recurrence is up to 1.2x more accurate (96 x 75 pixels
// of 0.1 mm, 128 and 256 frequencies up to 0.1 MHz, 0.15 cycles: forward 8.3e-8 to
// 9.4e-8 against 8.9e-8 to 1.1e-7; 1 MHz, 1.5 cycles: 0.9x to 1.2x; 2 MHz, 2.9
// cycles: 0.97x; adjoint 0.5x to 1.2x, 0.6x to 1.1x and 0.8x).
constexpr double kMmaMinSpan = 2.5;
// And not where sincos2's phases could leave its domain of 2^21 cycles (the blocks
// reach up to twice the highest frequency): such phases mean little in FP32, but the
// recurrence's factors keep their modulus of 1.
constexpr double kMmaMaxSpan = 524288.0;

// cycles from the centre of a tile to its corner at the highest frequency
double freq_span(const pa_plan* p, int Q, double f0, double df) {
  const bool d2 = p->dim == 2;
  const double ex = (std::min(p->grid.nx, d2 ? Tile<2>::X : Tile<3>::X) - 1) * p->grid.dx;
  const double ey = (std::min(p->grid.ny, d2 ? Tile<2>::Y : Tile<3>::Y) - 1) * p->grid.dy;
  const double ez = d2 ? 0.0 : (std::min(p->grid.nz, Tile<3>::Z) - 1) * p->grid.dz;
  return 0.5 * std::sqrt(ex * ex + ey * ey + ez * ez) / p->c * (f0 + (Q - 1) * df);
}
bool use_mma(const pa_plan* p, int Q, double f0, double df, int min_count) {
  const double span = freq_span(p, Q, f0, df);
  return Q >= min_count && span >= kMmaMinSpan && span <= kMmaMaxSpan;
}

__global__ void __launch_bounds__(kFreqThreads) k_freq_combine(const FreqParams P, int ntiles) {
  const int64_t idx = blockIdx.x * (int64_t)kFreqThreads + threadIdx.x;
  if (idx >= (int64_t)P.S * P.Q) return;
  const int s = (int)(idx / P.Q), n = (int)(idx % P.Q);
  float2 v = make_float2(0.0f, 0.0f);
  for (int t = 0; t < ntiles; ++t) {
    const float2 w = P.part[((int64_t)s * ntiles + t) * P.Q + n];
    v.x += w.x;
    v.y += w.y;
  }
  const float ck = (float)(2.0 * M_PI * (P.f0 + n * P.df) * P.amp);  // amp c k_n
  P.out[idx] = make_float2(-ck * v.y, ck * v.x);                      // i c k_n v
}

FreqParams freq_params(const pa_plan* p, int Q, double f0, double df) {
  FreqParams f{};
  f.sensors = p->d_sensors;
  f.S = p->S;
  f.Q = Q;
  f.dim = p->dim;
  f.nx = p->grid.nx;
  f.ny = p->grid.ny;
  f.nz = p->grid.nz;
  f.ntx = p->g.ntx;
  f.nty = p->g.nty;
  f.ntz = p->g.ntz;
  f.dx = p->grid.dx;
  f.dy = p->grid.dy;
  f.dz = p->grid.dz;
  f.ox = p->grid.origin[0];
  f.oy = p->grid.origin[1];
  f.oz = p->grid.origin[2];
  f.c = p->c;
  f.inv_c = 1.0 / p->c;
  f.f0 = f0;
  f.df = df;
  f.amp = p->amp;
  f.n_chunks = (p->S + kFreqSensors - 1) / kFreqSensors;
  f.inv_cf = (float)f.inv_c;
  f.f0f = (float)f0;
  f.dff = (float)df;
  f.hdx = (float)(0.5 * f.dx);
  f.hdy = (float)(0.5 * f.dy);
  f.hdz = (float)(0.5 * f.dz);
  return f;
}

pa_status freq_workspace(pa_plan* p, size_t bytes) {
  if (p->freq_bytes >= bytes) return PA_OK;
  if (p->d_freq) {
    PA_CUDA(cudaDeviceSynchronize());
    cudaFree(p->d_freq);
    p->bytes -= (int64_t)p->freq_bytes;
    p->d_freq = nullptr;
    p->freq_bytes = 0;
  }
  cudaError_t e = cudaMalloc(&p->d_freq, bytes);
  if (e != cudaSuccess) {
    cudaGetLastError();
    set_error("frequency-domain workspace: cudaMalloc of %zu bytes failed", bytes);
    return PA_ERR_OOM;
  }
  p->freq_bytes = bytes;
  p->bytes += (int64_t)bytes;
  return PA_OK;
}

size_t a256(size_t v) { return (v + 255) / 256 * 256; }

// Workspace of a call with `bytes` of partial results: the partials first, then
// the tables of k_freq_prep.
size_t freq_table_bytes(const pa_plan* p, int Q) {
  return a256((size_t)p->ntiles * p->S * sizeof(FreqRef)) + a256((size_t)Q * sizeof(float)) +
         a256((size_t)p->S * sizeof(int));
}
void freq_tables(const pa_plan* p, FreqParams& f, size_t part_bytes) {
  unsigned char* w = static_cast<unsigned char*>(p->d_freq) + a256(part_bytes);
  f.refs = reinterpret_cast<FreqRef*>(w);
  w += a256((size_t)p->ntiles * p->S * sizeof(FreqRef));
  f.cks = reinterpret_cast<float*>(w);
  w += a256((size_t)f.Q * sizeof(float));
  f.scales = reinterpret_cast<int*>(w);
}
cudaError_t freq_prep(const pa_plan* p, const FreqParams& f, cudaStream_t st) {
  const int64_t n_ref = (int64_t)p->ntiles * p->S;
  const int nb_ref = (int)((n_ref + kFreqThreads - 1) / kFreqThreads);
  const int nb_ck = (f.Q + kFreqThreads - 1) / kFreqThreads;
  const int nb_sc = f.p ? (p->S + kFreqThreads / 32 - 1) / (kFreqThreads / 32) : 0;
  auto kernel = p->dim == 2 ? k_freq_prep<2> : k_freq_prep<3>;
  kernel<<<nb_ref + nb_ck + nb_sc, kFreqThreads, 0, st>>>(f, nb_ref, nb_ck);
  return cudaGetLastError();
}
// CTAs that the adjoint's work split aims at: two per SM.  Three are resident, so a
// split that just reaches this leaves a third of their places empty.
int64_t freq_wave() {
  int dev = 0, n = 152;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1)
    n = 152;
  return 2 * (int64_t)n;
}

pa_status check_freq(const pa_plan* p, int Q, double f0, double df, const void* a, const void* b,
                     const char* who) {
  if (!p || !a || !b) {
    set_error("%s: NULL argument", who);
    return PA_ERR_INVALID_ARG;
  }
  if (Q < 1 || Q > 20480 || !std::isfinite(f0) || !std::isfinite(df) || f0 < 0.0 || df < 0.0) {
    set_error("%s: need 1 <= n_freq <= 20480 and finite f0, df >= 0", who);
    return PA_ERR_INVALID_ARG;
  }
  return PA_OK;
}

}  // namespace
}  // namespace pa

using namespace pa;

extern "C" {

pa_status pa_freq_forward(pa_plan* plan, int n_freq, double f0, double df, const float* x_dev,
                          float* p_dev, pa_stream stream) {
  PA_TRY(check_freq(plan, n_freq, f0, df, x_dev, p_dev, "pa_freq_forward"));
  DeviceGuard guard(plan->device);
  const bool mma = use_mma(plan, n_freq, f0, df, kMmaForward);
  const size_t bytes = (size_t)plan->S * plan->ntiles * n_freq * sizeof(float2);
  PA_TRY(freq_workspace(plan, a256(bytes) + freq_table_bytes(plan, n_freq)));
  FreqParams f = freq_params(plan, n_freq, f0, df);
  f.x = x_dev;
  f.part = static_cast<float2*>(plan->d_freq);
  f.out = reinterpret_cast<float2*>(p_dev);
  cudaStream_t st = (cudaStream_t)stream;
  const size_t smem = (size_t)n_freq * sizeof(float2);
  if (smem > 160 * 1024) {
    set_error("pa_freq_forward: n_freq %d needs more shared memory than a CTA has", n_freq);
    return PA_ERR_UNSUPPORTED;
  }
  freq_tables(plan, f, bytes);
  PA_CUDA(freq_prep(plan, f, st));
  if (mma) {
    auto kernel = plan->dim == 2
                      ? (n_freq > 128 ? k_freq_forward_mma<2, 2> : k_freq_forward_mma<2, 1>)
                      : (n_freq > 128 ? k_freq_forward_mma<3, 2> : k_freq_forward_mma<3, 1>);
    kernel<<<dim3(plan->S, plan->ntiles), kFreqThreads, freq_fwd_smem(n_freq > 128 ? 2 : 1), st>>>(
        f);
  } else {
    auto kernel = plan->dim == 2 ? k_freq_forward<2> : k_freq_forward<3>;
    PA_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const dim3 grid(f.n_chunks, plan->ntiles);
    kernel<<<grid, kFreqThreads, smem, st>>>(f);
  }
  PA_CUDA(cudaGetLastError());
  const int64_t n_out = (int64_t)plan->S * n_freq;
  k_freq_combine<<<(unsigned)((n_out + kFreqThreads - 1) / kFreqThreads), kFreqThreads, 0, st>>>(
      f, plan->ntiles);
  PA_CUDA(cudaGetLastError());
  return PA_OK;
}

pa_status pa_freq_adjoint(pa_plan* plan, int n_freq, double f0, double df, const float* p_dev,
                          float* x_dev, pa_stream stream) {
  PA_TRY(check_freq(plan, n_freq, f0, df, p_dev, x_dev, "pa_freq_adjoint"));
  DeviceGuard guard(plan->device);
  FreqParams f = freq_params(plan, n_freq, f0, df);
  const int64_t N = (int64_t)plan->grid.nx * plan->grid.ny * plan->grid.nz;
  const size_t smem = (size_t)n_freq * sizeof(float2);
  if (smem > 200 * 1024) {
    set_error("pa_freq_adjoint: n_freq %d needs more shared memory than a CTA has", n_freq);
    return PA_ERR_UNSUPPORTED;
  }
  const bool mma = use_mma(plan, n_freq, f0, df, kMmaAdjoint);
  if (mma) {
    // fewer sensors per CTA until the grid fills the chip
    f.spc = kFreqSensors;
    while (f.spc > 1 && (int64_t)plan->ntiles * ((plan->S + f.spc - 1) / f.spc) < freq_wave())
      f.spc /= 2;
    f.n_chunks = (plan->S + f.spc - 1) / f.spc;
  }
  const size_t bytes = (size_t)f.n_chunks * N * sizeof(float);
  PA_TRY(freq_workspace(plan, a256(bytes) + freq_table_bytes(plan, n_freq)));
  f.p = reinterpret_cast<const float2*>(p_dev);
  f.gpart = static_cast<float*>(plan->d_freq);
  f.gout = x_dev;
  cudaStream_t st = (cudaStream_t)stream;
  const dim3 grid(f.n_chunks, plan->ntiles);
  freq_tables(plan, f, bytes);
  PA_CUDA(freq_prep(plan, f, st));
  if (mma) {
    // n-tiles of 64 frequencies: 1, 2 or a whole block of 4
    auto kernel = plan->dim == 2 ? (n_freq <= 64    ? k_freq_adjoint_mma<2, 1>
                                    : n_freq <= 128 ? k_freq_adjoint_mma<2, 2>
                                                    : k_freq_adjoint_mma<2, 4>)
                                 : (n_freq <= 64    ? k_freq_adjoint_mma<3, 1>
                                    : n_freq <= 128 ? k_freq_adjoint_mma<3, 2>
                                                    : k_freq_adjoint_mma<3, 4>);
    PA_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kFreqAdjSmem));
    kernel<<<grid, kFreqThreads, kFreqAdjSmem, st>>>(f);
  } else {
    auto kernel = plan->dim == 2 ? k_freq_adjoint<2> : k_freq_adjoint<3>;
    PA_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    kernel<<<grid, kFreqThreads, smem, st>>>(f);
  }
  PA_CUDA(cudaGetLastError());
  k_freq_adjoint_sum<<<(unsigned)((N + kFreqThreads - 1) / kFreqThreads), kFreqThreads, 0, st>>>(
      f, N);
  PA_CUDA(cudaGetLastError());
  return PA_OK;
}

}  // extern "C"
