// Input standardization (Sec. III-A): one scan of floating-point Cartesian
// points -> an H x W range image (rows by altitude, columns by azimuth) and
// attribute images, quantized to unsigned integers, 0 where no valid point.
//
// The paper leaves the arithmetic open; this library fixes it in integers so
// that every decision is exact (no floating-point rounding can move a point
// to another pixel between two implementations):
//   coordinates  X = round-half-even(x * k), the product rounded to float32
//                (k = range units per metre); |x * k| >= 2^31 or NaN drops
//                the point
//   range        R = nearest integer to sqrt(X^2 + Y^2 + Z^2) (exact integer
//                square root)
//   angles       binary angles, 2^32 per turn, by CORDIC vectoring (Volder,
//                1959) in 32-bit integers: 30 micro-rotations of atan(2^-i)
//                on the vector scaled by a power of two (arithmetic shifts)
//                so that its larger component has 29 bits. Azimuth of (X, Y)
//                (counterclockwise from +x, 0 for X = Y = 0); elevation of
//                (rho, Z 2^f), rho = floor(sqrt(X^2 + Y^2) 2^f), f the
//                largest (possibly negative) integer keeping both below 2^29
//   pixel        row = nearest beam (midpoints between the beams' binary
//                altitudes; beyond half a spacing outside the first or last
//                beam the point is dropped), column = floor(((az - az0) mod
//                2^32) W / 2^32)
//   collisions   the nearest point wins (smallest R, then smallest index)
//   attributes   round-half-even(v * scale), the product rounded to float32,
//                clamped to the sample type, NaN and v * scale <= 0 -> 0
//
// Two launches per call of up to 256 scans: k_std_points (one thread per
// point, one grid row per scan: pixel and an atomicMin of the key (R << 32 |
// index in the scan) into a per-pixel word, L2-resident for a few scans) and
// k_std_pixels (a warp per 128 pixels of a scan, four a lane, grid-stride: the
// winning point's range and attributes, and the key word reset for the next
// call).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include <cuda_runtime.h>

#include "jiffy.h"
#include "jiffy_types.h"

namespace jiffy {
namespace {

constexpr int kStdIter = 30;         // CORDIC micro-rotations
constexpr int kNormBits = 29;        // CORDIC inputs scaled to this many bits
constexpr uint32_t kStdMaxAttr = 16;
constexpr uint32_t kStdMaxScans = 256;  // scans per call
constexpr double kPi = 3.14159265358979323846;

struct StdAttr {
  const float* v;
  void* out;
  float scale;
  uint32_t bytes;
};

struct StdParams {
  uint32_t H, W, T, clockwise, range_bytes, rmin, rmax, n_attr;
  float k;
  uint32_t az0;          // binary angle (2^32 per turn)
  int top, bottom;       // elevation limits (H > 1)
  const int* mid;        // [H - 1] midpoints between beams, decreasing
  float el0, row_scale;  // row of elevation el, were the beams evenly spaced: (el0 - el) row_scale
  int atan_t[kStdIter];
  const float* xyz;
  unsigned long long* keys;  // [T][H * W]
  void* range_out;           // [T][H * W]
  StdAttr attr[kStdMaxAttr];
  unsigned long long off[kStdMaxScans + 1];  // scan t's points: [off[t], off[t + 1])
};

__device__ __forceinline__ bool coord(float p, long long& out) {
  if (!(fabsf(p) < 2147483648.0f)) return false;  // also NaN
  out = (long long)rintf(p);                     // round half to even
  return true;
}

// floor(sqrt(n)) for n < 2^63.6 (n < 3 2^62): a float32 estimate (the FP64
// units of this GPU are few), one Newton correction r += (n - r^2) / 2r in
// float32 (leaves r within one of the root), then exact integer corrections.
__device__ __forceinline__ unsigned long long isqrt64(unsigned long long n) {
  if (n == 0ull) return 0ull;
  unsigned long long r = (unsigned long long)__fsqrt_rn(__ull2float_rn(n));
  const long long e = (long long)(n - r * r);  // |e| < 2^42
  r = (unsigned long long)((long long)r + __float2ll_rn(__fdividef((float)e, 2.0f * (float)r)));
  while (r * r > n) r--;
  while ((r + 1) * (r + 1) <= n) r++;
  return r;
}

__device__ __forceinline__ int cordic_vec(int x, int y, const int* t) {
  int ang = 0;
#pragma unroll
  for (int i = 0; i < kStdIter; i++) {
    const int xs = x >> i, ys = y >> i;
    const bool up = y > 0;
    x += up ? ys : -ys;
    y += up ? -xs : xs;
    ang += up ? t[i] : -t[i];
  }
  return ang;
}

__device__ __forceinline__ int bit_length(unsigned long long m) { return 64 - __clzll(m); }

// v 2^s, floor division (arithmetic shift) for s < 0
__device__ __forceinline__ long long scale2(long long v, int s) { return s >= 0 ? v * (1ll << s) : (v >> (-s)); }

__device__ __forceinline__ uint32_t azimuth(long long X, long long Y, const int* t) {
  if (X == 0 && Y == 0) return 0u;
  const unsigned long long m = (unsigned long long)(X < 0 ? -X : X) | (unsigned long long)(Y < 0 ? -Y : Y);
  const int s = kNormBits - bit_length(m);
  int x = (int)scale2(X, s), y = (int)scale2(Y, s);
  uint32_t base = 0u;
  if (x < 0) {  // a half turn first
    x = -x;
    y = -y;
    base = 0x80000000u;
  }
  return base + (uint32_t)cordic_vec(x, y, t);  // modulo 2^32
}

__device__ __forceinline__ int elevation(long long X, long long Y, long long Z, const int* t) {
  const unsigned long long h = (unsigned long long)(X * X) + (unsigned long long)(Y * Y);
  const unsigned long long z2 = (unsigned long long)(Z * Z);
  const unsigned long long m = h > z2 ? h : z2;
  if (m == 0) return 0;
  const int e = bit_length(m);
  const int f = e <= 2 * kNormBits ? (2 * kNormBits - e) / 2 : -((e - 2 * kNormBits + 1) / 2);  // m 4^f < 2^58
  const unsigned long long hs = f >= 0 ? h << (2 * f) : h >> (-2 * f);
  return cordic_vec((int)isqrt64(hs), (int)scale2(Z, f), t);
}

__device__ __forceinline__ void store_sample(void* p, uint32_t bytes, size_t i, uint32_t v) {
  if (bytes == 4) static_cast<uint32_t*>(p)[i] = v;
  else if (bytes == 2) static_cast<uint16_t*>(p)[i] = (uint16_t)v;
  else static_cast<uint8_t*>(p)[i] = (uint8_t)v;
}

__device__ __forceinline__ uint32_t quantize_attr(float v, float scale, uint32_t bytes) {
  const float p = __fmul_rn(v, scale);
  const uint32_t mx = bytes == 4 ? 0xffffffffu : ((1u << (8 * bytes)) - 1u);
  if (!(p > 0.0f)) return 0u;  // also NaN
  if (p >= (float)mx) return mx;
  const float r = rintf(p);
  return r >= (float)mx ? mx : (uint32_t)r;
}

// Square root to 2^-23 relative.
__device__ __forceinline__ float root(float v) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}

// The exact pixel of a point in range (row * W + column; ~0 outside the
// vertical field of view), by CORDIC: the definition, taken for the points
// that quick_pixel leaves open.
__device__ __noinline__ uint32_t exact_pixel(const StdParams& p, long long X, long long Y, long long Z) {
  const int* t = p.atan_t;
  uint32_t row = 0;
  if (p.H > 1) {
    const int el = elevation(X, Y, Z, t);
    if (el > p.top || el < p.bottom) return ~0u;
    uint32_t lo = 0, hi = p.H - 1;  // row = number of midpoints above el
    while (lo < hi) {
      const uint32_t m = (lo + hi) >> 1;
      if (__ldg(p.mid + m) > el) lo = m + 1;
      else hi = m;
    }
    row = lo;
  }
  const uint32_t a = azimuth(X, Y, t) - p.az0;  // modulo 2^32
  return row * p.W + (uint32_t)(((unsigned long long)a * p.W) >> 32);
}

// The same pixel from float32 angles, where they decide it. A CORDIC angle is
// within 1.5e-7 rad of the true one by its error bound (30 truncated steps on
// 28-bit vectors and more, 30 rounded table entries; below 6e-8 where tested),
// a float32 one within 1.2e-6 rad (atan2f: 3 ulp, 7.2e-7 at half a turn;
// inputs and scaling 4e-7): together less than 1000 units of 2^-32 turn. So where the pixel is the same over kMargin units
// either side of the float angle, the CORDIC angle falls into it too. About 1
// point in 300 of a 128 x 2048 image is closer to an edge than that (returns
// false) and goes to exact_pixel. With two CORDICs for every point (935
// instructions) the kernel was bound by issue: 273 us for 40 scans of
// 128 x 2048, 74 us this way.
constexpr int kMargin = 2048;
constexpr float kUnits = 683565275.576f;  // 2^32 / (2 pi)

__device__ __forceinline__ bool quick_pixel(const StdParams& p, float x, float y, float z, uint32_t& px) {
  uint32_t row = 0;
  if (p.H > 1) {
    const int el = __float2int_rn(atan2f(z, root(x * x + y * y)) * kUnits);  // |el| <= 2^30
    if (el - kMargin > p.top || el + kMargin < p.bottom) {
      px = ~0u;
      return true;
    }
    if (el + kMargin > p.top || el - kMargin < p.bottom) return false;
    auto above = [&](uint32_t m) { return __ldg(p.mid + m) > el; };
    // evenly spaced beams: the row directly, else by search
    uint32_t lo = (uint32_t)min(max(__float2int_rn((p.el0 - (float)el) * p.row_scale), 0), (int)p.H - 1);
    if ((lo > 0 && !above(lo - 1u)) || (lo < p.H - 1u && above(lo))) {
      uint32_t hi = p.H - 1;
      lo = 0;
      while (lo < hi) {
        const uint32_t m = (lo + hi) >> 1;
        if (above(m)) lo = m + 1;
        else hi = m;
      }
    }
    if ((lo > 0 && __ldg(p.mid + lo - 1u) <= el + kMargin) || (lo < p.H - 1u && __ldg(p.mid + lo) > el - kMargin))
      return false;
    row = lo;
  }
  const uint32_t a = (uint32_t)__float2int_rn(atan2f(y, x) * kUnits) - p.az0;  // modulo 2^32
  const uint32_t a0 = a - kMargin, a1 = a + kMargin, col = __umulhi(a0, p.W);
  if (a0 > a1 || __umulhi(a1, p.W) != col) return false;
  px = row * p.W + col;
  return true;
}

__global__ void __launch_bounds__(256) k_std_points(const __grid_constant__ StdParams p) {
  const uint32_t scan = blockIdx.y;
  const unsigned long long p0 = p.off[scan], n = p.off[scan + 1] - p0;
  unsigned long long* keys = p.keys + (size_t)scan * p.H * p.W;
  for (unsigned long long ii = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; ii < n;
       ii += (unsigned long long)gridDim.x * blockDim.x) {
    const uint32_t i = (uint32_t)ii;  // index within the scan (< 2^32)
    const float* q = p.xyz + 3ull * (p0 + ii);
    const float fx = __fmul_rn(__ldg(q), p.k), fy = __fmul_rn(__ldg(q + 1), p.k), fz = __fmul_rn(__ldg(q + 2), p.k);
    unsigned long long R;
    uint32_t px;
    if (fmaxf(fmaxf(fabsf(fx), fabsf(fy)), fabsf(fz)) < 1048576.0f && fx == fx && fy == fy && fz == fz) {
      // |X|, |Y|, |Z| <= 2^20, exact in float32: the range from a float32
      // root off by less than 1.5 and one correction against the sum of
      // squares modulo 2^32
      const int X = __float2int_rn(fx), Z = __float2int_rn(fz), Y = p.clockwise ? -__float2int_rn(fy) : __float2int_rn(fy);
      const float x = (float)X, y = (float)Y, z = (float)Z;
      int r = __float2int_rn(root(x * x + y * y + z * z));
      auto sq = [](int v) { return (uint32_t)v * (uint32_t)v; };
      const int e = (int)(sq(X) + sq(Y) + sq(Z) - sq(r));
      if (e > r) r++;
      else if (e <= -r) r--;
      R = (unsigned long long)(uint32_t)r;
      if (r < 1 || (uint32_t)r < p.rmin || (uint32_t)r > p.rmax) continue;
      if (!quick_pixel(p, x, y, z, px)) px = exact_pixel(p, X, Y, Z);
    } else {
      long long X, Y, Z;
      if (!coord(fx, X) || !coord(fy, Y) || !coord(fz, Z)) continue;
      if (p.clockwise) Y = -Y;
      const unsigned long long m = (unsigned long long)(X * X) + (unsigned long long)(Y * Y) +
                                   (unsigned long long)(Z * Z);  // < 3 2^62
      const unsigned long long r = isqrt64(m);
      R = r + ((m - r * r) > r ? 1ull : 0ull);
      if (R < 1 || R < p.rmin || R > p.rmax) continue;
      px = exact_pixel(p, X, Y, Z);
    }
    if (px != ~0u) atomicMin(keys + px, (R << 32) | i);
  }
}

// One pixel of every scan: a warp takes 128 pixels of a scan at a time, each
// lane four of them 32 apart, so that four keys and then four values per
// attribute are in flight and every access of a warp is to neighbouring
// words (40 scans of 128 x 2048 with three attributes: 68 us; one pixel per lane
// took 92, four neighbouring ones as vectors 177). Bound by memory: the keys
// in and out, the winners' attributes, the images.
__global__ void __launch_bounds__(256) k_std_pixels(const __grid_constant__ StdParams p) {
  constexpr uint32_t N = 4;
  const uint32_t HW = p.H * p.W, tiles = (HW + 127u) / 128u;  // HW <= 2^26
  const uint32_t lane = threadIdx.x & 31u, G = gridDim.x * 8u, g0 = blockIdx.x * 8u + (threadIdx.x >> 5);
  const uint32_t dt = G / tiles, dr = G % tiles;  // the stride as (scans, tiles)
  uint32_t t = g0 / tiles, r = g0 % tiles;        // this warp's scan and tile
  while (t < p.T) {
    const uint32_t px = 128u * r + lane;
    const size_t at0 = (size_t)t * HW + px;
    unsigned long long key[N];
#pragma unroll
    for (uint32_t i = 0; i < N; i++) key[i] = px + 32u * i < HW ? p.keys[at0 + 32u * i] : ~0ull;
    const unsigned long long first = p.off[t];
#pragma unroll
    for (uint32_t i = 0; i < N; i++) {
      if (px + 32u * i >= HW) continue;
      const bool hit = key[i] != ~0ull;
      if (hit) p.keys[at0 + 32u * i] = ~0ull;  // ready for the next call
      store_sample(p.range_out, p.range_bytes, at0 + 32u * i, hit ? (uint32_t)(key[i] >> 32) : 0u);
    }
    for (uint32_t a = 0; a < p.n_attr; a++) {
      const StdAttr& at = p.attr[a];
      float f[N];  // the winning points' values
#pragma unroll
      for (uint32_t i = 0; i < N; i++) f[i] = key[i] != ~0ull ? __ldg(at.v + first + (uint32_t)key[i]) : 0.0f;
#pragma unroll
      for (uint32_t i = 0; i < N; i++)
        if (px + 32u * i < HW) store_sample(at.out, at.bytes, at0 + 32u * i, quantize_attr(f[i], at.scale, at.bytes));  // (0 gives 0)
    }
    t += dt;
    r += dr;
    if (r >= tiles) {
      r -= tiles;
      t++;
    }
  }
}

long long binary_angle(double rad) {
  return std::llround(rad / (2.0 * kPi) * 4294967296.0);  // 2^32 per turn
}

}  // namespace
}  // namespace jiffy

struct jiffy_standardizer {
  int device = 0;
  uint32_t H = 0, W = 0;
  jiffy::StdParams base{};
  int* d_mid = nullptr;
  unsigned long long* d_keys = nullptr;  // key_scans x H x W, all ~0 between calls
  uint32_t key_scans = 0;
  int sms = 0;
};

extern "C" {

jiffy_status jiffy_standardizer_create(jiffy_standardizer** out, const jiffy_sensor_desc* sd, int device) {
  using namespace jiffy;
  if (!out || !sd) return JIFFY_ERR_INVALID_ARG;
  *out = nullptr;
  const uint32_t H = sd->H, W = sd->W;
  if (H == 0 || H > kMaxH || W == 0 || W > kMaxW || !sd->beam_altitude || !(sd->units_per_m > 0.0f) ||
      !(sd->range_bytes == 2 || sd->range_bytes == 4) || !std::isfinite(sd->azimuth0))
    return JIFFY_ERR_INVALID_ARG;
  std::vector<long long> alt(H);
  std::vector<int> mid(H > 1 ? H - 1 : 1, 0);
  for (uint32_t b = 0; b < H; b++) {
    if (!std::isfinite(sd->beam_altitude[b])) return JIFFY_ERR_INVALID_ARG;
    alt[b] = binary_angle(sd->beam_altitude[b]);
    if (alt[b] > (1ll << 30) || alt[b] < -(1ll << 30) || (b > 0 && alt[b] >= alt[b - 1]))  // within +-90 deg
      return JIFFY_ERR_INVALID_ARG;
  }
  for (uint32_t b = 0; b + 1 < H; b++) mid[b] = (int)(alt[b + 1] + (alt[b] - alt[b + 1]) / 2);
  int prev = 0, ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) return JIFFY_ERR_CUDA;
  if (cudaGetDevice(&prev) != cudaSuccess || cudaSetDevice(device) != cudaSuccess) return JIFFY_ERR_CUDA;
  jiffy_standardizer* s = new (std::nothrow) jiffy_standardizer();
  jiffy_status st = s ? JIFFY_OK : JIFFY_ERR_NOMEM;
  if (st == JIFFY_OK) {
    s->device = device;
    s->H = H;
    s->W = W;
    StdParams& p = s->base;
    p.H = H;
    p.W = W;
    p.clockwise = sd->clockwise ? 1u : 0u;
    p.range_bytes = sd->range_bytes;
    p.rmin = sd->min_range;
    const uint32_t dmax = sd->range_bytes == 4 ? 0xffffffffu : 0xffffu;
    p.rmax = sd->max_range < dmax ? sd->max_range : dmax;
    p.k = sd->units_per_m;
    p.az0 = (uint32_t)(unsigned long long)binary_angle(sd->azimuth0);  // modulo 2^32
    if (H > 1) {
      p.top = (int)std::min<long long>(alt[0] + (alt[0] - alt[1]) / 2, 0x7fffffffll);
      p.bottom = (int)std::max<long long>(alt[H - 1] - (alt[H - 2] - alt[H - 1]) / 2, -0x7fffffffll - 1);
      p.el0 = (float)alt[0];
      p.row_scale = (float)((double)(H - 1) / (double)(alt[0] - alt[H - 1]));
    }
    for (int i = 0; i < kStdIter; i++)
      p.atan_t[i] = (int)std::llround(std::atan(std::ldexp(1.0, -i)) / (2.0 * kPi) * 4294967296.0);
    if (cudaDeviceGetAttribute(&s->sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess ||
        cudaMalloc(&s->d_mid, sizeof(int) * mid.size()) != cudaSuccess ||
        cudaMalloc(&s->d_keys, sizeof(unsigned long long) * (size_t)H * W) != cudaSuccess ||
        cudaMemcpy(s->d_mid, mid.data(), sizeof(int) * mid.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(s->d_keys, 0xff, sizeof(unsigned long long) * (size_t)H * W) != cudaSuccess ||
        cudaDeviceSynchronize() != cudaSuccess)
      st = JIFFY_ERR_CUDA;
    p.mid = s->d_mid;
    s->key_scans = 1;
  }
  if (st != JIFFY_OK && s) {
    cudaFree(s->d_mid);
    cudaFree(s->d_keys);
    delete s;
    s = nullptr;
  }
  cudaSetDevice(prev);
  *out = s;
  return st;
}

void jiffy_standardizer_destroy(jiffy_standardizer* s) {
  if (!s) return;
  int prev = 0;
  cudaGetDevice(&prev);
  cudaSetDevice(s->device);
  cudaDeviceSynchronize();
  cudaFree(s->d_mid);
  cudaFree(s->d_keys);
  cudaSetDevice(prev);
  delete s;
}

jiffy_status jiffy_standardize_seq(jiffy_standardizer* s, uint32_t n_scans, const float* xyz,
                                   const uint64_t* point_offsets, void* range_out, uint32_t n_attr,
                                   const jiffy_point_attr* attrs, void* cuda_stream) {
  using namespace jiffy;
  if (!s || n_scans == 0 || n_scans > kStdMaxScans || !point_offsets || !range_out || n_attr > kStdMaxAttr ||
      (n_attr && !attrs))
    return JIFFY_ERR_INVALID_ARG;
  StdParams p = s->base;
  unsigned long long max_n = 0;
  for (uint32_t t = 0; t < n_scans; t++) {
    if (point_offsets[t + 1] < point_offsets[t] || point_offsets[t + 1] - point_offsets[t] > 0xffffffffull)
      return JIFFY_ERR_INVALID_ARG;
    max_n = std::max<unsigned long long>(max_n, point_offsets[t + 1] - point_offsets[t]);
  }
  for (uint32_t t = 0; t <= n_scans; t++) p.off[t] = point_offsets[t];
  if (max_n && !xyz) return JIFFY_ERR_INVALID_ARG;
  p.T = n_scans;
  p.xyz = xyz;
  p.range_out = range_out;
  p.n_attr = n_attr;
  for (uint32_t a = 0; a < n_attr; a++) {
    const uint32_t b = attrs[a].dtype_bytes;
    if (!(b == 1 || b == 2 || b == 4) || !attrs[a].out || (max_n && !attrs[a].values)) return JIFFY_ERR_INVALID_ARG;
    p.attr[a] = StdAttr{attrs[a].values, attrs[a].out, attrs[a].scale, b};
  }
  int prev = 0;
  if (cudaGetDevice(&prev) != cudaSuccess || cudaSetDevice(s->device) != cudaSuccess) return JIFFY_ERR_CUDA;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
  const size_t HW = (size_t)s->H * s->W;
  jiffy_status rc = JIFFY_OK;
  if (n_scans > s->key_scans || !s->d_keys) {  // a larger pixel table: wait for the calls using the old one
    if (cudaStreamSynchronize(st) != cudaSuccess) rc = JIFFY_ERR_CUDA;
    cudaFree(s->d_keys);
    s->d_keys = nullptr;
    s->key_scans = 0;
    if (rc == JIFFY_OK) {
      const size_t bytes = sizeof(unsigned long long) * HW * n_scans;
      const cudaError_t me = cudaMalloc(&s->d_keys, bytes);
      if (me != cudaSuccess) rc = me == cudaErrorMemoryAllocation ? JIFFY_ERR_NOMEM : JIFFY_ERR_CUDA;
      else if (cudaMemsetAsync(s->d_keys, 0xff, bytes, st) != cudaSuccess) rc = JIFFY_ERR_CUDA;
      else s->key_scans = n_scans;
    }
  }
  if (rc == JIFFY_OK) {
    p.keys = s->d_keys;
    const uint32_t target = 16u * (uint32_t)s->sms;  // CTAs of 256 threads in flight, grid-stride beyond
    if (max_n) {
      const unsigned long long need = (max_n + 255u) / 256u;
      const uint32_t bx = (uint32_t)std::max<unsigned long long>(
          1ull, std::min<unsigned long long>(need, (target + n_scans - 1) / n_scans));
      k_std_points<<<dim3(bx, n_scans), 256, 0, st>>>(p);
    }
    const size_t tiles = (HW + 127) / 128 * n_scans;
    k_std_pixels<<<(uint32_t)std::min<size_t>(target, (tiles + 7) / 8), 256, 0, st>>>(p);
    if (cudaGetLastError() != cudaSuccess) rc = JIFFY_ERR_CUDA;
  }
  cudaSetDevice(prev);
  return rc;
}

jiffy_status jiffy_standardize(jiffy_standardizer* s, const float* xyz, uint32_t n_points, void* range_out,
                               uint32_t n_attr, const jiffy_point_attr* attrs, void* cuda_stream) {
  const uint64_t off[2] = {0, n_points};
  return jiffy_standardize_seq(s, 1, xyz, off, range_out, n_attr, attrs, cuda_stream);
}

}  // extern "C"
