// PERCH successor evaluation: device kernels for sm_103a.
//
// Arithmetic contract: every floating-point step on the evaluation path is a
// single IEEE binary32 operation rounded to nearest-even (__fadd_rn,
// __fmul_rn, __fmaf_rn, __frcp_rn, __int2float_rn, __float2int_rn); a fused
// multiply-add appears only where written as ffma (one rounding, as IEEE 754
// defines it) and the library is compiled with -fmad=false so nothing else is
// contracted. Coverage and z-buffer resolution are exact integer /
// order-independent min operations, so every count is bit-exact with the CPU
// oracle, which writes out the same arithmetic.
#include <climits>

#include "perch_internal.h"

namespace perch {

// ------------------------------------------------------------------ helpers
__device__ __forceinline__ float fmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float ffma(float a, float b, float c) { return __fmaf_rn(a, b, c); }

__device__ __forceinline__ int ford(float f) {  // order-preserving float -> int
  int i = __float_as_int(f);
  return i >= 0 ? i : i ^ 0x7fffffff;
}

// squared camera-frame distance, d^2 = fma(dz, dz, fma(dy, dy, dx dx))
__device__ __forceinline__ float dist2(float px, float py, float pz, float4 q) {
  const float dx = fsub(px, q.x), dy = fsub(py, q.y), dz = fsub(pz, q.z);
  return ffma(dz, dz, ffma(dy, dy, fmul(dx, dx)));
}

// V(O) of Sec. III-A for mesh m at pose (ox, oy, yaw iyaw): the inscribed
// vertical cylinder (kind 0) or the closed-form solid (kinds 1-3), tested in
// the object frame: x' = fma(s, dy, c dx), y' = fma(c, dy, -(s dx)) with the
// pose table's (c, s); z is the world height.
__device__ __forceinline__ bool in_volume(const Geometry& g, const DevMesh& m, float ox, float oy, int iyaw,
                                          float4 qw) {
  const float dx = fsub(qw.x, ox), dy = fsub(qw.y, oy);
  if (m.vol_kind == 0) {
    const float d2 = ffma(dy, dy, fmul(dx, dx));
    return d2 <= m.vol_r2 && m.vol_zlo <= qw.z && qw.z <= m.vol_zhi;
  }
  const float2 cs = g.cs[iyaw];
  const float xo = ffma(cs.y, dy, fmul(cs.x, dx));
  const float yo = ffma(cs.x, dy, -fmul(cs.y, dx));
  if (m.vol_kind == 1)
    return fabsf(xo) <= m.vol_p[0] && fabsf(yo) <= m.vol_p[1] && m.vol_z0 <= qw.z && qw.z <= m.vol_z1;
  if (m.vol_kind == 2) {
    if (!(m.vol_z0 <= qw.z && qw.z <= m.vol_z1)) return false;
    // every face test passes inside the inscribed circle shrunk by 2^-12 in
    // r^2, and one fails outside the circumscribed circle grown by 2^-12,
    // whatever the binary32 rounding of the face tests (n <= 256 sides);
    // only the thin annulus between them needs the faces
    const float d2 = ffma(yo, yo, fmul(xo, xo));
    if (d2 <= m.vol_p[1]) return true;
    if (d2 >= m.vol_p[2]) return false;
    const float2* nr = g.vol_normals + m.vol_nrm;
    for (int k = 0; k < m.vol_n; ++k)
      if (ffma(nr[k].y, yo, fmul(nr[k].x, xo)) > m.vol_p[0]) return false;
    return true;
  }
  const float X = fmul(xo, m.vol_p[0]), Y = fmul(yo, m.vol_p[1]), Z = fmul(fsub(qw.z, m.vol_p[3]), m.vol_p[2]);
  const float t = ffma(Y, Y, fmul(X, X));
  const float z2 = fmul(Z, Z);
  const float F = m.vol_n == 2 ? ffma(t, t, fmul(z2, z2)) : fadd(t, z2);
  return F <= 1.0f;
}

struct Vtx {
  int X, Y;   // snapped pixel coordinates, 1/16 px (absolute or tile-relative)
  float iz;   // 1 / z_c; negative marks a culled vertex
};

// Camera-frame vertex (table entry M_yaw v plus the pose offset b) -> pixel:
// 1/z = 1/c_z; u = fma(fx, c_x (1/z), cx); X = rint(16 u).
__device__ __forceinline__ Vtx project_vertex(const Camera& c, float4 mv, float4 b) {
  const float xc = fadd(mv.x, b.x), yc = fadd(mv.y, b.y), zc = fadd(mv.z, b.z);
  bool bad = !(zc > kNearZ);
  const float iz = __frcp_rn(zc);
  const float u = ffma(c.fx, fmul(xc, iz), c.cx);
  const float v = ffma(c.fy, fmul(yc, iz), c.cy);
  bad = bad || !(fabsf(u) <= kGuard) || !(fabsf(v) <= kGuard);
  Vtx o;
  if (bad) {
    o.X = 0; o.Y = 0; o.iz = -1.0f;
    return o;
  }
  o.X = __float2int_rn(fmul(16.0f, u));
  o.Y = __float2int_rn(fmul(16.0f, v));
  o.iz = iz;
  return o;
}

__device__ __forceinline__ int floor16(int a) { return a >> 4; }
__device__ __forceinline__ int ceil16(int a) { return -((-a) >> 4); }

// depth at a covered pixel centre: b_i = E_i / A, 1/z = fma(b2, 1/z2,
// fma(b1, 1/z1, b0/z0)), z = 1/(1/z); returned as the float's bits
__device__ __forceinline__ uint32_t pixel_depth_bits(int w0, int w1, int w2, float invA, float iz0, float iz1,
                                                     float iz2) {
  const float b0 = fmul(__int2float_rn(w0), invA);
  const float b1 = fmul(__int2float_rn(w1), invA);
  const float b2 = fmul(__int2float_rn(w2), invA);
  const float iz = ffma(b2, iz2, ffma(b1, iz1, fmul(b0, iz0)));
  return __float_as_uint(__frcp_rn(iz));
}

// edge ownership for the top-left tie rule (front faces in this orientation)
__device__ __forceinline__ bool owns(int dx, int dy) { return dy > 0 || (dy == 0 && dx < 0); }

// Rasterise one triangle (any size) into a tile of tw x th pixels whose
// top-left pixel is at (ox16 / 16, oy16 / 16): exact edge functions, top-left
// tie rule, min-z resolve through `sink`. Used for full-image parent renders.
template <typename Sink>
__device__ __forceinline__ void raster_tri(Vtx a, Vtx b, Vtx c, int ox16, int oy16, int tw, int th,
                                           unsigned& culled, Sink sink) {
  if (a.iz < 0.0f || b.iz < 0.0f || c.iz < 0.0f) {
    culled = 1u;
    return;
  }
  const int X0 = a.X - ox16, Y0 = a.Y - oy16;
  const int X1 = b.X - ox16, Y1 = b.Y - oy16;
  const int X2 = c.X - ox16, Y2 = c.Y - oy16;
  const int xmin = min(X0, min(X1, X2)), xmax = max(X0, max(X1, X2));
  const int ymin = min(Y0, min(Y1, Y2)), ymax = max(Y0, max(Y1, Y2));
  if (xmax - xmin >= kMaxExtent || ymax - ymin >= kMaxExtent) {
    long long A64 = (long long)(Y1 - Y0) * (X2 - X0) - (long long)(X1 - X0) * (Y2 - Y0);
    if (A64 > 0) culled = 1u;
    return;
  }
  const int A = (Y1 - Y0) * (X2 - X0) - (X1 - X0) * (Y2 - Y0);
  if (A <= 0) return;  // back-facing or degenerate
  const int px0 = max(ceil16(xmin), 0), px1 = min(floor16(xmax), tw - 1);
  const int py0 = max(ceil16(ymin), 0), py1 = min(floor16(ymax), th - 1);
  if (px0 > px1 || py0 > py1) return;
  const bool own12 = owns(X2 - X1, Y2 - Y1), own20 = owns(X0 - X2, Y0 - Y2), own01 = owns(X1 - X0, Y1 - Y0);
  const float invA = __frcp_rn(__int2float_rn(A));
  for (int py = py0; py <= py1; ++py) {
    const int Py = 16 * py;
    for (int px = px0; px <= px1; ++px) {
      const int Px = 16 * px;
      const int w0 = (Y2 - Y1) * (Px - X1) - (X2 - X1) * (Py - Y1);
      const int w1 = (Y0 - Y2) * (Px - X2) - (X0 - X2) * (Py - Y2);
      const int w2 = (Y1 - Y0) * (Px - X0) - (X1 - X0) * (Py - Y0);
      const bool in = (w0 > 0 || (w0 == 0 && own12)) && (w1 > 0 || (w1 == 0 && own20)) &&
                      (w2 > 0 || (w2 == 0 && own01));
      if (in) sink(py * tw + px, pixel_depth_bits(w0, w1, w2, invA, a.iz, b.iz, c.iz));
    }
  }
}

// Row k of a cell's 3x3x3 neighbourhood: three cells in x at (y + dy, z + dz);
// the centre row first (the likeliest to hold a match).
__device__ __forceinline__ void near_row(int k, int& dy, int& dz) {
  const int q = (k * 11) >> 5, r = k - 3 * q;  // k / 3, k % 3
  dz = (q & 1) ? -1 : q >> 1;
  dy = (r & 1) ? -1 : r >> 1;
}

// Eq. (1) against the observed cloud: is some observed point within delta of
// p? 3x3x3 neighbourhood of a grid whose cells are at least delta wide; three
// consecutive x-cells are one contiguous range of the bucketed array. Bound
// by the dependent loads of the ranges, so rows3 tells which of the nine rows
// hold any point (mostly none to three near a surface): the others cost
// nothing (640x480 root expansion 3.0 -> 2.7 ms, multi-scene batches, where
// k_cost makes these tests, 2.4 -> 1.9 ms, against one bit for all nine). A
// window of the depth image about p's pixel was slower (root expansion
// 4.2 ms): most tests are of points about a centimetre off the cloud, which
// must see all 49 depths.
__device__ __forceinline__ bool explained_by_obs(const ObsIndex& o, float px, float py, float pz, float d2max) {
  if (o.n == 0) return false;
  const float fx = fmul(fsub(px, o.g3x), o.inv3);
  const float fy = fmul(fsub(py, o.g3y), o.inv3);
  const float fz = fmul(fsub(pz, o.g3z), o.inv3);
  const int ix = (int)floorf(fminf(fmaxf(fx, -2.0f), (float)o.n3x + 1.0f));
  const int iy = (int)floorf(fminf(fmaxf(fy, -2.0f), (float)o.n3y + 1.0f));
  const int iz = (int)floorf(fminf(fmaxf(fz, -2.0f), (float)o.n3z + 1.0f));
  const int x0 = max(ix - 1, 0), x1 = min(ix + 1, o.n3x - 1);
  if (x0 > x1) return false;
  uint32_t rows = 0x1ffu;
  if (ix >= 0 && ix < o.n3x && iy >= 0 && iy < o.n3y && iz >= 0 && iz < o.n3z)
    rows = __ldg(&o.rows3[(iz * o.n3y + iy) * o.n3x + ix]);
  for (; rows; rows &= rows - 1u) {
    int dy, dz;
    near_row(__ffs((int)rows) - 1, dy, dz);
    const int cy = iy + dy, cz = iz + dz;
    if (cy < 0 || cy >= o.n3y || cz < 0 || cz >= o.n3z) continue;
    const int base = (cz * o.n3y + cy) * o.n3x;
    const int s = __ldg(&o.start3[base + x0]), e = __ldg(&o.start3[base + x1 + 1]);
    for (int k = s; k < e; ++k)
      if (dist2(px, py, pz, __ldg(&o.cam3[k])) <= d2max) return true;
  }
  return false;
}

// Half-width in pixels, along an axis of focal length f, of a window about
// the pixel of a point (slope t = x / z or y / z, depth z) that holds the pixel
// of every point within delta of it: for |p - q| <= delta and z > delta,
// |x_p / z_p - x_q / z_q| <= delta sqrt(1 + t^2) / (z - delta). 1 + t^2 / 2
// bounds the square root; both pixels are whole, so the slack only has to
// cover the rounding of the rays, of d^2 and of this bound.
__device__ __forceinline__ int delta_radius(const Camera& cam, float f, float t, float z) {
  const float d = 1.0001f * cam.delta;
  return (int)fminf(f * (1.0f + 0.5f * t * t) * __fdividef(d, z - d) + (0.05f + 1e-6f * (float)(cam.W + cam.H)), 1e6f);
}
__device__ __forceinline__ bool delta_bounded(const Camera& cam, float z) { return z - 1.0001f * cam.delta > 1e-3f; }

// The pixel of observed point q and the window of delta_radius about it.
__device__ __forceinline__ void delta_window(const Camera& cam, float4 q, int& u, int& v, int& u0, int& u1, int& v0,
                                             int& v1) {
  const float tx = __fdividef(q.x, q.z), ty = __fdividef(q.y, q.z);
  if (cam.W <= 16384 && cam.H <= 16384) {  // far less than half a pixel off
    u = __float2int_rn(cam.fx * tx + cam.cx);
    v = __float2int_rn(cam.fy * ty + cam.cy);
  } else {
    const int pix = __float_as_int(q.w);
    u = pix % cam.W;
    v = pix / cam.W;
  }
  if (delta_bounded(cam, q.z)) {
    const int Ru = delta_radius(cam, cam.fx, tx, q.z), Rv = delta_radius(cam, cam.fy, ty, q.z);
    u0 = u - Ru; u1 = u + Ru; v0 = v - Rv; v1 = v + Rv;
  } else {
    u0 = INT_MIN / 2; u1 = INT_MAX / 2; v0 = INT_MIN / 2; v1 = INT_MAX / 2;
  }
}

// The new object's dR over its pose's box (rows of the box width): either a
// z tile with +inf off dR (mask == nullptr), or the staged render (z bits,
// with the explained flag in the sign bit) and a bitmask of dR pixels.
struct DRTile {
  const uint32_t* z;
  const uint32_t* mask;
  __device__ __forceinline__ uint32_t at(int i) const {
    if (!mask) return z[i];
    return ((mask[i >> 5] >> (i & 31)) & 1u) ? (z[i] & 0x7fffffffu) : kInfBits;
  }
};

// Eq. (1) against the new object's dR: is some rendered point within delta
// of the observed point q?
__device__ __forceinline__ bool explained_by_tile(const Camera& cam, float4 q, const DRTile& tile,
                                                  const float* rxs, const float* rys, int4 bb) {
  int u, v, u0, u1, v0, v1;
  delta_window(cam, q, u, v, u0, u1, v0, v1);
  u0 = max(u0 - bb.x, 0); u1 = min(u1 - bb.x, bb.z - 1);
  v0 = max(v0 - bb.y, 0); v1 = min(v1 - bb.y, bb.w - 1);
  auto near = [&](int lx, int ly) {
    const uint32_t zb = tile.at(ly * bb.z + lx);
    if (zb == kInfBits) return false;
    const float z = __uint_as_float(zb);
    return dist2(fmul(rxs[lx], z), fmul(rys[ly], z), z, q) <= cam.delta2;
  };
  u -= bb.x;
  v -= bb.y;
  if (u >= u0 && u <= u1 && v >= v0 && v <= v1 && near(u, v)) return true;  // its own pixel: the likeliest
  for (int ly = v0; ly <= v1; ++ly)
    for (int lx = u0; lx <= u1; ++lx)
      if (near(lx, ly)) return true;
  return false;
}

__device__ __forceinline__ int warp_sum(int v) { return __reduce_add_sync(0xffffffffu, v); }

// ------------------------------------------------------------------ utility
__global__ void k_fill_u32(uint32_t* p, uint32_t v, long long n) {
  long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  long long stride = (long long)gridDim.x * blockDim.x;
  for (; i < n; i += stride) p[i] = v;
}

cudaError_t launch_fill_u32(uint32_t* p, uint32_t v, long long n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  long long blocks = (n + 255) / 256;
  if (blocks > 152 * 32) blocks = 152 * 32;
  k_fill_u32<<<(unsigned)blocks, 256, 0, s>>>(p, v, n);
  return cudaGetLastError();
}

// a batch's buffers in one launch, bound by storing the parents' z-buffers, instead of a
// fill and three memsets: smallest evaluation 134 -> 130 us
__global__ void __launch_bounds__(256) k_prepare(uint32_t* z, long long n, int* a, long long n0, int* b, long long n1) {
  const long long i0 = blockIdx.x * 256LL + threadIdx.x, stride = gridDim.x * 256LL, n4 = n >> 2;
  for (long long i = i0; i < n4; i += stride)
    reinterpret_cast<uint4*>(z)[i] = make_uint4(kInfBits, kInfBits, kInfBits, kInfBits);
  if (i0 < (n & 3)) z[4 * n4 + i0] = kInfBits;
  for (long long i = i0; i < n0; i += stride) a[i] = 0;
  for (long long i = i0; i < n1; i += stride) b[i] = 0;
}

cudaError_t launch_prepare(uint32_t* z, long long n, int* a, long long n0, int* b, long long n1, cudaStream_t s) {
  const long long most = std::max(std::max(n >> 2, n0), std::max(n1, 1LL));
  k_prepare<<<(unsigned)std::min(152LL * 16, (most + 255) / 256), 256, 0, s>>>(z, n, a, n0, b, n1);
  return cudaGetLastError();
}

// Exclusive scans in two launches (one for a single block): the sums of the
// blocks' ranges, then each block adds the sums before its own and scans its
// range. At most 2048 blocks, of 1024 elements or a multiple. F gives the elements
// and takes each with its prefix: f.load(i), f.store(i, prefix, element),
// f.total(sum). A scan of 120k elements takes
// 3 + 4 us; three launches (block scans, their sums, the sums added) took 3 + 3 + 4.
constexpr int kScanBlocks = 2048;

template <typename F>
__device__ __forceinline__ typename F::T scan_thread(const F& f, long long base, int n, typename F::T (&v)[4]) {
  typename F::T s = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    v[k] = base + k < n ? f.load((int)(base + k)) : 0;
    s += v[k];
  }
  return s;
}
// inclusive scan over the block's 256 threads; every thread gets the block's sum
template <typename T>
__device__ __forceinline__ T scan_256(T v, T& sum) {
  __shared__ T warp_tot[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int d = 1; d < 32; d <<= 1) {
    const T t = __shfl_up_sync(0xffffffffu, v, d);
    if (lane >= d) v += t;
  }
  __syncthreads();
  if (lane == 31) warp_tot[warp] = v;
  __syncthreads();
  sum = 0;
  T before = 0;
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    if (w == warp) before = sum;
    sum += warp_tot[w];
  }
  return v + before;
}

template <typename F>
__global__ void __launch_bounds__(256) k_scan_sums(F f, int n, long long per, typename F::T* sums) {
  typename F::T a = 0, v[4], sum;
  for (long long b = blockIdx.x * per; b < (blockIdx.x + 1) * per; b += 1024)
    a += scan_thread(f, b + 4 * threadIdx.x, n, v);
  scan_256(a, sum);
  if (threadIdx.x == 0) sums[blockIdx.x] = sum;
}

template <typename F>
__global__ void __launch_bounds__(256) k_scan_out(F f, int n, long long per, const typename F::T* sums) {
  typename F::T a = 0, v[4], carry, sum;
  for (int k = threadIdx.x; k < (int)blockIdx.x; k += 256) a += sums[k];
  scan_256(a, carry);
  for (long long b = blockIdx.x * per; b < (blockIdx.x + 1) * per; b += 1024) {
    const long long base = b + 4 * threadIdx.x;
    const typename F::T s = scan_thread(f, base, n, v);
    typename F::T run = carry + scan_256(s, sum) - s;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (base + k < n) f.store((int)(base + k), run, v[k]);
      run += v[k];
    }
    carry += sum;
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) f.total(carry);
}

template <typename F>
cudaError_t launch_scan(const F& f, int n, typename F::T* tmp, cudaStream_t s) {
  const int units = std::max(1, (int)(((long long)n + 1023) / 1024));
  const long long per = 1024LL * ((units + kScanBlocks - 1) / kScanBlocks);
  const unsigned nb = (unsigned)std::max(1LL, (n + per - 1) / per);
  if (nb > 1) k_scan_sums<<<nb, 256, 0, s>>>(f, n, per, tmp);
  k_scan_out<<<nb, 256, 0, s>>>(f, n, per, tmp);
  return cudaGetLastError();
}

// out[0..n] with out[n] = total; `copy` (or nullptr) gets out[0..n - 1] as well
struct ScanInts {
  typedef int T;
  const int* in;
  int *out, *copy;
  int n;
  __device__ int load(int i) const { return in[i]; }
  __device__ void store(int i, int prefix, int) const {
    out[i] = prefix;
    if (copy) copy[i] = prefix;
  }
  __device__ void total(int sum) const { out[n] = sum; }
};

cudaError_t launch_exclusive_scan(const int* in, int* out, int n, int* tmp, cudaStream_t s) {
  return launch_scan(ScanInts{in, out, nullptr, n}, n, tmp, s);
}

// ------------------------------------------------------- observation prep
__device__ __forceinline__ bool depth_valid(float d) { return d > 0.0f && isfinite(d); }

__global__ void k_obs_count(const float* depth, int n, int* block_counts) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  const bool ok = i < n && depth_valid(depth[i]);
  int c = __syncthreads_count(ok);
  if (threadIdx.x == 0) block_counts[blockIdx.x] = c;
}

cudaError_t launch_obs_count(const float* depth, int W, int H, int* block_counts, cudaStream_t s) {
  const int n = W * H;
  k_obs_count<<<(n + 255) / 256, 256, 0, s>>>(depth, n, block_counts);
  return cudaGetLastError();
}

// back-project valid pixels (observed cloud I) in pixel order, camera and
// world frames; accumulate bounding boxes for the grids
__global__ void k_obs_write(const float* depth, Camera cam, const float* rx, const float* ry,
                            const int* block_offsets, float4* cam_pts, float4* world_pts, int* bounds) {
  __shared__ int warp_cnt[8];
  const int n = cam.W * cam.H;
  const int i = blockIdx.x * 256 + threadIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float d = i < n ? depth[i] : 0.0f;
  const bool ok = i < n && depth_valid(d);
  const unsigned bal = __ballot_sync(0xffffffffu, ok);
  if (lane == 0) warp_cnt[warp] = __popc(bal);
  __syncthreads();
  int off = block_offsets[blockIdx.x];
  for (int w = 0; w < warp; ++w) off += warp_cnt[w];
  off += __popc(bal & ((1u << lane) - 1u));
  if (!ok) return;
  const int u = i % cam.W, v = i / cam.W;
  const float x = fmul(rx[u], d), y = fmul(ry[v], d), z = d;
  const float xw = fadd(ffma(cam.Rwc[2], z, ffma(cam.Rwc[1], y, fmul(cam.Rwc[0], x))), cam.twc[0]);
  const float yw = fadd(ffma(cam.Rwc[5], z, ffma(cam.Rwc[4], y, fmul(cam.Rwc[3], x))), cam.twc[1]);
  const float zw = fadd(ffma(cam.Rwc[8], z, ffma(cam.Rwc[7], y, fmul(cam.Rwc[6], x))), cam.twc[2]);
  cam_pts[off] = make_float4(x, y, z, __int_as_float(i));
  world_pts[off] = make_float4(xw, yw, zw, 0.0f);
  atomicMin(&bounds[0], ford(x)); atomicMin(&bounds[1], ford(y)); atomicMin(&bounds[2], ford(z));
  atomicMax(&bounds[3], ford(x)); atomicMax(&bounds[4], ford(y)); atomicMax(&bounds[5], ford(z));
  atomicMin(&bounds[6], ford(xw)); atomicMin(&bounds[7], ford(yw));
  atomicMax(&bounds[8], ford(xw)); atomicMax(&bounds[9], ford(yw));
}

cudaError_t launch_obs_write(const float* depth, const Camera& cam, const float* rx, const float* ry,
                             const int* block_offsets, float4* cam_pts, float4* world_pts, int* bounds,
                             cudaStream_t s) {
  const int n = cam.W * cam.H;
  k_obs_write<<<(n + 255) / 256, 256, 0, s>>>(depth, cam, rx, ry, block_offsets, cam_pts, world_pts, bounds);
  return cudaGetLastError();
}

__device__ __forceinline__ int cell_of(float x, float g, float inv, int n) {
  const float f = fmul(fsub(x, g), inv);
  int c = (int)floorf(fminf(fmaxf(f, -2.0f), (float)n + 1.0f));
  return c;
}

__device__ __forceinline__ int sat_sum(const int* S, int cols, int r0, int r1, int c0, int c1) {  // inclusive
  const int w = cols + 1;
  return S[(r1 + 1) * w + c1 + 1] - S[r0 * w + c1 + 1] - S[(r1 + 1) * w + c0] + S[r0 * w + c0];
}

// Could some observed point lie within delta of a point that object o
// renders? No, when the world (x, y) cells around its footprint disk (radius
// fp_r, plus delta, plus 2 cm for the rounding of the back-projected depth,
// plus a cell either side) hold no point: every rendered point lies within
// that disk horizontally, and Eq. (1) bounds the 3D distance, hence the
// horizontal one (the grid covers the whole cloud, so a disk beyond its
// cells holds none).
__device__ __forceinline__ bool obs_near(const Camera& cam, const Geometry& g, const ObsIndex& obs,
                                         const perch_obj& o) {
  if (obs.n == 0) return false;
  const float R = g.meshes[o.mesh].fp_r + cam.delta + 0.02f;
  const float ox = g.xs[o.ix], oy = g.ys[o.iy];
  const int cx0 = max(cell_of(ox - R, obs.g2x, obs.inv2, obs.n2x) - 1, 0);
  const int cx1 = min(cell_of(ox + R, obs.g2x, obs.inv2, obs.n2x) + 1, obs.n2x - 1);
  const int cy0 = max(cell_of(oy - R, obs.g2y, obs.inv2, obs.n2y) - 1, 0);
  const int cy1 = min(cell_of(oy + R, obs.g2y, obs.inv2, obs.n2y) + 1, obs.n2y - 1);
  return cx0 <= cx1 && cy0 <= cy1 && sat_sum(obs.sat2, obs.n2x, cy0, cy1, cx0, cx1) != 0;
}

__global__ void k_grid3_keys(const float4* pts, int n, float gx, float gy, float gz, float inv, int nx, int ny,
                             int nz, int* keys, int* counts) {
  const int k = blockIdx.x * 256 + threadIdx.x;
  if (k >= n) return;
  const float4 p = pts[k];
  const int ix = min(max(cell_of(p.x, gx, inv, nx), 0), nx - 1);
  const int iy = min(max(cell_of(p.y, gy, inv, ny), 0), ny - 1);
  const int iz = min(max(cell_of(p.z, gz, inv, nz), 0), nz - 1);
  const int key = (iz * ny + iy) * nx + ix;
  keys[k] = key;
  atomicAdd(&counts[key], 1);
}

cudaError_t launch_grid3_keys(const float4* cam_pts, int n, float g3x, float g3y, float g3z, float inv3, int n3x,
                              int n3y, int n3z, int* keys, int* counts, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  k_grid3_keys<<<(n + 255) / 256, 256, 0, s>>>(cam_pts, n, g3x, g3y, g3z, inv3, n3x, n3y, n3z, keys, counts);
  return cudaGetLastError();
}

__global__ void k_grid2_keys(const float4* pts, int n, float gx, float gy, float inv, int nx, int ny, int* keys,
                             int* counts) {
  const int k = blockIdx.x * 256 + threadIdx.x;
  if (k >= n) return;
  const float4 p = pts[k];
  const int ix = min(max(cell_of(p.x, gx, inv, nx), 0), nx - 1);
  const int iy = min(max(cell_of(p.y, gy, inv, ny), 0), ny - 1);
  const int key = iy * nx + ix;
  keys[k] = key;
  atomicAdd(&counts[key], 1);
}

cudaError_t launch_grid2_keys(const float4* world_pts, int n, float g2x, float g2y, float inv2, int n2x, int n2y,
                              int* keys, int* counts, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  k_grid2_keys<<<(n + 255) / 256, 256, 0, s>>>(world_pts, n, g2x, g2y, inv2, n2x, n2y, keys, counts);
  return cudaGetLastError();
}

__global__ void k_scatter(const int* keys, int n, int* cursor, const float4* a_in, float4* a_out,
                          const float4* b_in, float4* b_out) {
  const int k = blockIdx.x * 256 + threadIdx.x;
  if (k >= n) return;
  const int pos = atomicAdd(&cursor[keys[k]], 1);
  a_out[pos] = a_in[k];
  if (b_in) b_out[pos] = b_in[k];
}

cudaError_t launch_scatter(const int* keys, int n, int* cursor, const float4* a_in, float4* a_out,
                           const float4* b_in, float4* b_out, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  k_scatter<<<(n + 255) / 256, 256, 0, s>>>(keys, n, cursor, a_in, a_out, b_in, b_out);
  return cudaGetLastError();
}

// ray slopes rx[u] = (u - cx) / fx, ry[v] = (v - cy) / fy in double, rounded once
__global__ void k_rays(Camera cam, float* rx, float* ry) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i < cam.W) rx[i] = (float)__ddiv_rn(__dsub_rn((double)i, (double)cam.cx), (double)cam.fx);
  if (i < cam.H) ry[i] = (float)__ddiv_rn(__dsub_rn((double)i, (double)cam.cy), (double)cam.fy);
}

cudaError_t launch_rays(const Camera& cam, float* rx, float* ry, cudaStream_t s) {
  const int n = cam.W > cam.H ? cam.W : cam.H;
  k_rays<<<(n + 255) / 256, 256, 0, s>>>(cam, rx, ry);
  return cudaGetLastError();
}

// per cell of the 3D grid, which rows of its neighbourhood (near_row) hold a point
__global__ void k_near_rows(const int* start3, int nx, int ny, int nz, uint16_t* rows3) {
  const long long c = blockIdx.x * 256LL + threadIdx.x;
  const long long n = (long long)nx * ny * nz;
  if (c >= n) return;
  const int ix = (int)(c % nx), iy = (int)((c / nx) % ny), iz = (int)(c / ((long long)nx * ny));
  const int x0 = max(ix - 1, 0), x1 = min(ix + 1, nx - 1);
  unsigned rows = 0;
  for (int k = 0; k < 9; ++k) {
    int dy, dz;
    near_row(k, dy, dz);
    const int y = iy + dy, z = iz + dz;
    if (y < 0 || y >= ny || z < 0 || z >= nz) continue;
    const int base = (z * ny + y) * nx;
    if (start3[base + x1 + 1] > start3[base + x0]) rows |= 1u << k;
  }
  rows3[c] = (uint16_t)rows;
}

cudaError_t launch_near_rows(const int* start3, int n3x, int n3y, int n3z, uint16_t* rows3, cudaStream_t s) {
  const long long n = (long long)n3x * n3y * n3z;
  if (n == 0) return cudaSuccess;
  k_near_rows<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(start3, n3x, n3y, n3z, rows3);
  return cudaGetLastError();
}
// Camera-frame pose tables: per yaw M = R_cw Rz(yaw), per (ix, iy)
// b = R_cw (x, y, 0) + t_cw, in double from the binary32 inputs (products of
// two floats are exact in double), rounded once.
__global__ void k_pose_tables(Camera cam, Geometry g, float* yaw_mats, float4* pose_off) {
  const int t = blockIdx.x * 256 + threadIdx.x;
  if (t < g.n_yaw) {
    const double cs = g.cs[t].x, sn = g.cs[t].y;
    for (int r = 0; r < 3; ++r) {
      const double r0 = cam.Rcw[r * 3 + 0], r1 = cam.Rcw[r * 3 + 1];
      yaw_mats[t * 9 + r * 3 + 0] = __double2float_rn(__dadd_rn(__dmul_rn(r0, cs), __dmul_rn(r1, sn)));
      yaw_mats[t * 9 + r * 3 + 1] = __double2float_rn(__dsub_rn(__dmul_rn(r1, cs), __dmul_rn(r0, sn)));
      yaw_mats[t * 9 + r * 3 + 2] = cam.Rcw[r * 3 + 2];
    }
  }
  if (t < g.nx * g.ny) {
    const double x = g.xs[t / g.ny], y = g.ys[t % g.ny];
    float b[3];
    for (int r = 0; r < 3; ++r) {
      const double r0 = cam.Rcw[r * 3 + 0], r1 = cam.Rcw[r * 3 + 1];
      b[r] = __double2float_rn(__dadd_rn(__dadd_rn(__dmul_rn(r0, x), __dmul_rn(r1, y)), (double)cam.tcw[r]));
    }
    pose_off[t] = make_float4(b[0], b[1], b[2], 0.0f);
  }
}

// per (yaw, chunk vertex): M v = fma(M_r2, vz, fma(M_r1, vy, M_r0 vx)) per row
__global__ void k_vertex_table(Geometry g, const float* yaw_mats, float* vtab) {
  const long long t = blockIdx.x * 256LL + threadIdx.x;
  if (t >= (long long)g.n_yaw * g.n_cverts) return;
  const int k = (int)(t / g.n_cverts), j = (int)(t % g.n_cverts);
  const float* M = yaw_mats + 9 * k;
  const float4 v = g.chunk_verts[j];
  for (int r = 0; r < 3; ++r)
    vtab[3 * t + r] = ffma(M[r * 3 + 2], v.z, ffma(M[r * 3 + 1], v.y, fmul(M[r * 3 + 0], v.x)));
}

cudaError_t launch_pose_tables(const Camera& cam, const Geometry& g, float* yaw_mats, float4* pose_off,
                               float* vtab, cudaStream_t s) {
  const int n = g.n_yaw > g.nx * g.ny ? g.n_yaw : g.nx * g.ny;
  k_pose_tables<<<(n + 255) / 256, 256, 0, s>>>(cam, g, yaw_mats, pose_off);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const long long nv = (long long)g.n_yaw * g.n_cverts;
  if (nv == 0) return cudaSuccess;
  k_vertex_table<<<(unsigned)((nv + 255) / 256), 256, 0, s>>>(g, yaw_mats, vtab);
  return cudaGetLastError();
}

// conservative screen box of every (mesh, pose) from the 8 corners of the
// mesh's bounding box (a convex hull of its vertices), plus one pixel;
// bad: 1 = a corner at or behind the near plane or far off-screen,
// 2 = the unclipped box is wider or taller than kMaxObjectPixels
__global__ void k_pose_bbox(Camera cam, Geometry g, const float* yaw_mats, int4* bbox, int* max_wh, int* bad_any,
                            uint8_t* general) {
  const long long n = (long long)g.n_mesh * g.nx * g.ny * g.n_yaw;
  const long long t = blockIdx.x * 256LL + threadIdx.x;
  if (t >= n) return;
  const int iyaw = (int)(t % g.n_yaw);
  const int iy = (int)((t / g.n_yaw) % g.ny);
  const int ix = (int)((t / ((long long)g.n_yaw * g.ny)) % g.nx);
  const int m = (int)(t / ((long long)g.n_yaw * g.ny * g.nx));
  const DevMesh dm = g.meshes[m];
  const float* M = yaw_mats + 9 * iyaw;
  const float4 b = g.pose_off[ix * g.ny + iy];
  float umin = 1e30f, umax = -1e30f, vmin = 1e30f, vmax = -1e30f, zmin = 1e30f, slope = 0.0f;
  bool bad = false;
  for (int k = 0; k < 8; ++k) {
    const float vx = (k & 1) ? dm.hi[0] : dm.lo[0];
    const float vy = (k & 2) ? dm.hi[1] : dm.lo[1];
    const float vz = (k & 4) ? dm.hi[2] : dm.lo[2];
    const float xc = M[0] * vx + M[1] * vy + M[2] * vz + b.x;
    const float yc = M[3] * vx + M[4] * vy + M[5] * vz + b.y;
    const float zc = M[6] * vx + M[7] * vy + M[8] * vz + b.z;
    if (!(zc > kNearZ)) { bad = true; break; }
    const float u = cam.fx * (xc / zc) + cam.cx, v = cam.fy * (yc / zc) + cam.cy;
    umin = fminf(umin, u); umax = fmaxf(umax, u);
    vmin = fminf(vmin, v); vmax = fmaxf(vmax, v);
    zmin = fminf(zmin, zc);
    slope = fmaxf(slope, fmaxf(fabsf(xc / zc), fabsf(yc / zc)));
  }
  // The tile renders' quick path needs triangles of at most kSmallPixels and
  // no vertex that could be culled. Points at distance <= L and depths >= zmin
  // project at most f (|dx| + |x_q / z_q| |dz|) / z_p <= f L (1 + slope) / zmin
  // pixels apart in u or v; two pixels for the snap and the rounding.
  const float ext = fmaxf(cam.fx, cam.fy) * dm.edge * (1.0f + slope) / zmin + 2.0f;
  general[t] = bad || !(ext <= (float)kSmallPixels) || !(zmin > 1.2f * kNearZ) ||
               !(fmaxf(fmaxf(fabsf(umin), fabsf(umax)), fmaxf(fabsf(vmin), fabsf(vmax))) <= kGuard - 48.0f);
  int4 r;
  if (bad || !(umax - umin < 4096.0f) || !(vmax - vmin < 4096.0f)) {
    r = make_int4(0, 0, cam.W, cam.H);
    atomicOr(bad_any, 1);
  } else {
    if (umax - umin > (float)(kMaxObjectPixels - 4) || vmax - vmin > (float)(kMaxObjectPixels - 4))
      atomicOr(bad_any, 2);
    int x0 = (int)floorf(fmaxf(umin, -8.0f)) - 1, x1 = (int)ceilf(fminf(umax, (float)cam.W + 8.0f)) + 1;
    int y0 = (int)floorf(fmaxf(vmin, -8.0f)) - 1, y1 = (int)ceilf(fminf(vmax, (float)cam.H + 8.0f)) + 1;
    x0 = max(x0, 0); y0 = max(y0, 0);
    x1 = min(x1, cam.W - 1); y1 = min(y1, cam.H - 1);
    if (x0 > x1 || y0 > y1) r = make_int4(0, 0, 0, 0);
    else r = make_int4(x0, y0, x1 - x0 + 1, y1 - y0 + 1);
  }
  bbox[t] = r;
  atomicMax(&max_wh[2 * m], r.z);  // per-mesh tile
  atomicMax(&max_wh[2 * m + 1], r.w);
}

cudaError_t launch_pose_bbox(const Camera& cam, const Geometry& g, const float* yaw_mats, int4* bbox, int* max_wh,
                             int* bad, uint8_t* general, cudaStream_t s) {
  const long long n = (long long)g.n_mesh * g.nx * g.ny * g.n_yaw;
  if (n == 0) return cudaSuccess;
  k_pose_bbox<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(cam, g, yaw_mats, bbox, max_wh, bad, general);
  return cudaGetLastError();
}

// ------------------------------------------------------------ parent prep
struct GlobalSink {
  uint32_t* z;
  __device__ __forceinline__ void operator()(int idx, uint32_t zbits) const { atomicMin(&z[idx], zbits); }
};

__device__ __forceinline__ bool obj_ok(const Geometry& g, const perch_obj& o) {
  return o.mesh < g.n_mesh && o.ix >= 0 && o.ix < g.nx && o.iy >= 0 && o.iy < g.ny && o.iyaw < g.n_yaw;
}

// z-buffer render of every parent's objects (R_j) into its own full image.
// Block = one chunk of one (parent, object) pair.
__global__ void __launch_bounds__(256) k_render_parents(Camera cam, Geometry g, Batch b,
                                                        unsigned long long* culled_total) {
  __shared__ int2 sXY[kChunkMaxVerts];
  __shared__ float sIZ[kChunkMaxVerts];
  const int item = blockIdx.y;
  const int p = item / b.parent_stride, k = item % b.parent_stride;
  if (p >= b.n_par) return;
  const int plen = b.parent_len[p];
  if (k >= plen || plen > b.parent_stride) return;
  const perch_obj o = b.parents[(long long)p * b.parent_stride + k];
  if (!obj_ok(g, o)) return;
  const DevMesh m = g.meshes[o.mesh];
  if ((int)blockIdx.x >= m.chunk_count) return;
  const int4 ci = g.chunk_info[m.chunk_begin + blockIdx.x];
  const float4 bo = g.pose_off[o.ix * g.ny + o.iy];
  const float* V = g.vtab + 3 * ((size_t)o.iyaw * g.n_cverts + ci.x);
  for (int v = threadIdx.x; v < ci.y; v += 256) {
    const Vtx r = project_vertex(cam, make_float4(V[3 * v], V[3 * v + 1], V[3 * v + 2], 0.0f), bo);
    sXY[v] = make_int2(r.X, r.Y);
    sIZ[v] = r.iz;
  }
  __syncthreads();
  unsigned culled = 0;
  uint32_t* z = reinterpret_cast<uint32_t*>(b.parent_z) + (size_t)p * cam.W * cam.H;
  for (int t = threadIdx.x; t < ci.w; t += 256) {
    const uint32_t pk = g.chunk_tris[ci.z + t];
    const int i0 = pk & 1023, i1 = (pk >> 10) & 1023, i2 = (pk >> 20) & 1023;
    raster_tri(Vtx{sXY[i0].x, sXY[i0].y, sIZ[i0]}, Vtx{sXY[i1].x, sXY[i1].y, sIZ[i1]},
               Vtx{sXY[i2].x, sXY[i2].y, sIZ[i2]}, 0, 0, cam.W, cam.H, culled, GlobalSink{z});
  }
  if (culled_total) {
    const int c = __syncthreads_count(culled != 0);
    if (threadIdx.x == 0 && c) atomicAdd(culled_total, (unsigned long long)c);
  }
}

cudaError_t launch_render_parents(const Camera& cam, const Geometry& g, const Batch& b, int max_chunks,
                                  unsigned long long* culled, cudaStream_t s) {
  if (b.n_par == 0 || b.parent_stride == 0 || max_chunks == 0) return cudaSuccess;
  const long long items = (long long)b.n_par * b.parent_stride;
  if (items > 65535) return cudaErrorInvalidValue;
  dim3 grid(max_chunks, (unsigned)items);
  k_render_parents<<<grid, 256, 0, s>>>(cam, g, b, culled);
  return cudaGetLastError();
}

// U set of a parent one object short of a complete scene:
// U = {q in I - V_{K-1} : q unexplained by R_{K-1}}; then for the last object
// O_K, residual(K) = #{q in U : q not in V(O_K), q unexplained by dR_K}. U is
// kept as a bit per point of the 2D-sorted cloud, and its size.
__global__ void k_uset(Camera cam, Geometry g, ObsIndex obs0, Batch b) {
  const int p = blockIdx.y;
  const int plen = b.parent_len[p];
  const int K_total = b.parent_K ? b.parent_K[p] : b.K_total;
  if (plen + 1 != K_total || plen > b.parent_stride) return;
  const int scene = b.parent_scene ? b.parent_scene[p] : 0;
  if (b.parent_scene && (scene < 0 || scene >= b.n_scenes)) return;
  const ObsIndex& obs = b.parent_scene ? b.scenes[scene] : obs0;
  const int k = blockIdx.x * 256 + threadIdx.x;
  bool in = k < obs.n;
  if (in) {
    const float4 qw = obs.world2[k];
    for (int j = 0; j < plen && in; ++j) {
      const perch_obj o = b.parents[(long long)p * b.parent_stride + j];
      in = obj_ok(g, o) && !in_volume(g, g.meshes[o.mesh], g.xs[o.ix], g.ys[o.iy], o.iyaw, qw);
    }
  }
  if (in && plen > 0) {
    const float4 q = obs.cam2[k];
    const float* zp = b.parent_z + (size_t)p * cam.W * cam.H;
    int u, v, u0, u1, v0, v1;
    delta_window(cam, q, u, v, u0, u1, v0, v1);
    u0 = max(u0, 0); u1 = min(u1, cam.W - 1);
    v0 = max(v0, 0); v1 = min(v1, cam.H - 1);
    for (int vp = v0; vp <= v1 && in; ++vp) {
      const float ry = g.ry[vp];
      for (int up = u0; up <= u1 && in; ++up) {
        const float z = zp[(size_t)vp * cam.W + up];
        in = __float_as_uint(z) == kInfBits || !(dist2(fmul(g.rx[up], z), fmul(ry, z), z, q) <= cam.delta2);
      }
    }
  }
  const unsigned bits = __ballot_sync(0xffffffffu, in);
  if ((threadIdx.x & 31) == 0 && k < obs.n) {
    b.uset[(size_t)p * b.uset_stride + (k >> 5)] = bits;
    if (bits) atomicAdd(&b.uset_count[p], __popc(bits));
  }
}

cudaError_t launch_uset(const Camera& cam, const Geometry& g, const ObsIndex& obs, const Batch& b,
                        cudaStream_t s) {
  const int n_max = b.parent_scene ? b.uset_stride : obs.n;  // the largest cloud of the batch's scenes
  if (b.n_par == 0 || n_max == 0) return cudaSuccess;
  if (b.n_par > 65535) return cudaErrorInvalidValue;
  dim3 grid((n_max + 255) / 256, b.n_par);
  k_uset<<<grid, 256, 0, s>>>(cam, g, obs, b);
  return cudaGetLastError();
}

// ------------------------------------------------------------- evaluation
// ---- bulk asynchronous copies (TMA, 1D) into shared memory, with mbarriers
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_barrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// one thread: announce `bytes` of transfer and start the copy gmem -> smem
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
               : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_addr(dst)),
               "l"(src), "r"(bytes), "r"(smem_addr(bar))
               : "memory");
}

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Wait for the phase with the given parity. Each poll may suspend the thread
// in hardware (up to 0.1 ms) instead of spinning; the wait gives up after
// `polls` polls or 2 s, whichever comes first, and then returns false.
__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(smem_addr(bar)), "r"(parity), "r"(100000u)
      : "memory");
  return done != 0;
}
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int polls = kWaitSpins) {
  if (polls > 0 && mbar_try(bar, parity)) return true;  // the usual case reads no clock
  const uint64_t t0 = global_ns();
  for (int i = 1; i < polls; ++i) {
    if (mbar_try(bar, parity)) return true;
    if (global_ns() - t0 > 2000000000ull) break;
  }
  return false;
}

// One projected vertex of a tile render: the snapped position in pixels
// relative to the tile's corner (ox, oy) and 1/z (negative: culled). x and y
// are multiples of 1/16: adding 1.5 2^23 to 16 u rounds it to the nearest
// integer, ties to even, as rint does, and every later step is exact.
constexpr float kRoundMagic = 12582912.0f;
template <bool CULL>  // false: the pose has no vertex near the near plane or the guard band
__device__ __forceinline__ float3 project_pixel(const Camera& c, float mx, float my, float mz, float4 b, float ox,
                                                float oy) {
  const float xc = fadd(mx, b.x), yc = fadd(my, b.y), zc = fadd(mz, b.z);
  const float iz = __frcp_rn(zc);
  const float u = ffma(c.fx, fmul(xc, iz), c.cx);
  const float v = ffma(c.fy, fmul(yc, iz), c.cy);
  if (CULL && (!(zc > kNearZ) || !(fabsf(u) <= kGuard) || !(fabsf(v) <= kGuard))) return make_float3(0.0f, 0.0f, -1.0f);
  return make_float3(ffma(fsub(ffma(u, 16.0f, kRoundMagic), kRoundMagic), 0.0625f, -ox),
                     ffma(fsub(ffma(v, 16.0f, kRoundMagic), kRoundMagic), 0.0625f, -oy), iz);
}
__device__ __forceinline__ float min3(float a, float b, float c) {
  float r;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
// a position in pixels (a multiple of 1/16) in units of 1/16 px
__device__ __forceinline__ int2 units16(float2 p) {
  return make_int2(__float2int_rn(fmul(p.x, 16.0f)), __float2int_rn(fmul(p.y, 16.0f)));
}

// Is the pixel centre with edge values (w0, w1, w2) inside the triangle
// under the top-left rule? Exact zeros (rare) look at the edge directions.
__device__ __forceinline__ bool covers(int w0, int w1, int w2, int2 a, int2 b, int2 c) {
  if ((w0 | w1 | w2) < 0) return false;  // strictly outside some edge
  if (w0 == 0 && !owns(c.x - b.x, c.y - b.y)) return false;
  if (w1 == 0 && !owns(a.x - c.x, a.y - c.y)) return false;
  if (w2 == 0 && !owns(b.x - a.x, b.y - a.y)) return false;
  return true;
}

// 1/z at a covered pixel centre: b_i = E_i (1/A), 1/z = fma(b2, 1/z2,
// fma(b1, 1/z1, b0/z0)). The tile keeps the largest 1/z (the nearest
// surface; z = 1/(1/z) is taken once per pixel afterwards).
__device__ __forceinline__ uint32_t pixel_iz_bits(int w0, int w1, int w2, float invA, float iz0, float iz1, float iz2) {
  const float b0 = fmul(__int2float_rn(w0), invA);
  const float b1 = fmul(__int2float_rn(w1), invA);
  const float b2 = fmul(__int2float_rn(w2), invA);
  return __float_as_uint(ffma(b2, iz2, ffma(b1, iz1, fmul(b0, iz0))));
}

// Test the candidate pixel centres [px0, px1] x [py0, py1] of a front-facing
// triangle (tile-relative 1/16-px vertices) and max its 1/z into the tile.
__device__ __forceinline__ void raster_box(int2 a, int2 b, int2 c, int A, int px0, int px1, int py0, int py1,
                                           const float* sIZ, int i0, int i1, int i2, uint32_t* tile, int tw) {
  // edge functions at the first candidate, then stepped by their exact
  // integer increments per pixel (16 sub-pixel units)
  const float invA = __frcp_rn(__int2float_rn(A));
  const int d0x = 16 * (c.y - b.y), d0y = -16 * (c.x - b.x);
  const int d1x = 16 * (a.y - c.y), d1y = -16 * (a.x - c.x);
  const int d2x = 16 * (b.y - a.y), d2y = -16 * (b.x - a.x);
  int r0 = (c.y - b.y) * (16 * px0 - b.x) - (c.x - b.x) * (16 * py0 - b.y);
  int r1 = (a.y - c.y) * (16 * px0 - c.x) - (a.x - c.x) * (16 * py0 - c.y);
  int r2 = (b.y - a.y) * (16 * px0 - a.x) - (b.x - a.x) * (16 * py0 - a.y);
  const float z0 = sIZ[i0], z1 = sIZ[i1], z2 = sIZ[i2];
  for (int py = py0; py <= py1; ++py) {
    int w0 = r0, w1 = r1, w2 = r2;
    for (int px = px0; px <= px1; ++px) {
      if (covers(w0, w1, w2, a, b, c))
        atomicMax(&tile[py * tw + px], pixel_iz_bits(w0, w1, w2, invA, z0, z1, z2));
      w0 += d0x;
      w1 += d1x;
      w2 += d2x;
    }
    r0 += d0y;
    r1 += d1y;
    r2 += d2y;
  }
}

#define kNoCover make_float4(1e6f, -1.0f, 1e6f, -1.0f)

struct EvalShared {
  uint64_t* bar;   // the vertex slice's bulk copy
  int* cnt;        // viol, n_new, culled, djr, djo, resid, n_vol
  int* qn;         // [2]: queued larger triangles of even and odd chunks
  unsigned char* dyn;
  uint32_t pv;     // parity of the barrier's next phase
  struct EvalHyp* hyp;  // k_eval: the hypothesis at work
};

// Outcome of one render or evaluation: done; a bounded wait gave up but
// every copy it was waiting for has landed since (the record carries
// kFlagTimeout and the CTA may go on); or a copy may still be in flight (the
// CTA must stop).
enum EvalStatus { kEvalDone = 0, kEvalTimedOut = 1, kEvalStop = 2 };

// Dynamic shared memory of a render: the chunk buffers (vertex-table slice,
// projected vertices, queue of larger triangles), then the tile (rows of the
// pose's box width). Only vbuf receives bulk copies; threads never write it.
struct RenderSmem {
  float* vbuf;  // x, y, z per vertex
  float2* sXY;  // pixels, relative to the tile's corner
  float* sIZ;
  uint32_t* queue;  // (triangle, box) pairs
  uint32_t* tile;
};

__device__ __forceinline__ RenderSmem render_smem(unsigned char* smem) {
  RenderSmem s;
  s.vbuf = reinterpret_cast<float*>(smem);
  s.sXY = reinterpret_cast<float2*>(s.vbuf + 3 * kChunkMaxVerts);
  s.sIZ = reinterpret_cast<float*>(s.sXY + kChunkMaxVerts);
  s.queue = reinterpret_cast<uint32_t*>(s.sIZ + kChunkMaxVerts);
  s.tile = s.queue + 2 * kBigQueue;
  return s;
}

constexpr size_t kChunkSmem = (size_t)kChunkMaxVerts * (12 + 8 + 4) + (size_t)kBigQueue * 8;

size_t render_smem_bytes(int tile_w, int tile_h) { return kChunkSmem + (size_t)tile_w * tile_h * 4; }

size_t eval_smem_bytes(int tile_w, int tile_h) {
  return render_smem_bytes(tile_w, tile_h) + (size_t)(tile_w + tile_h) * 4;
}

bool eval_tile_fits(int device, int tile_w, int tile_h) {
  int optin = 0;
  if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device) != cudaSuccess) return false;
  return eval_smem_bytes(tile_w, tile_h) + 256 <= (size_t)optin;  // 256: static shared memory of k_eval
}

constexpr int kNearList = 512;  // observed points per round of finish_phase's list

size_t cost_smem_bytes(int tile_w, int tile_h, int stages) {  // stages, dR bitmask (16-byte multiples), rays, list
  return (size_t)stages * ((tile_w * tile_h + 3) & ~3) * 4 + (size_t)(((tile_w * tile_h + 31) / 32 + 3) & ~3) * 4 +
         (size_t)(tile_w + tile_h) * 4 + (size_t)(kNearList + 1) * 4;
}

// thread 0: start the bulk copy of n vertices from entry v of yaw iyaw's
// table (whole 16-byte units: every chunk starts at a multiple of 4)
__device__ __forceinline__ void load_slice(const Geometry& g, int iyaw, int v, int n, const RenderSmem& s,
                                           uint64_t* bar) {
  bulk_load(s.vbuf, g.vtab + 3 * ((size_t)iyaw * g.n_cverts + v), ((uint32_t)n * 12u + 15u) & ~15u, bar);
}
// thread 0: start the copy of the first chunk of mesh m at yaw iyaw
__device__ __forceinline__ void render_start(const Geometry& g, const DevMesh& m, int iyaw, const RenderSmem& s,
                                             uint64_t* bar) {
  const int4 ci = g.chunk_info[m.chunk_begin];
  load_slice(g, iyaw, ci.x, ci.y, s, bar);
}

// The sign bit of three edge values together: set where one of them is negative.
__device__ __forceinline__ uint32_t outside(float w0, float w1, float w2) {
  return __float_as_uint(w0) | __float_as_uint(w1) | __float_as_uint(w2);
}
// An edge value is a multiple of 2^-8 px^2, so adding +-2^-10 leaves the sign
// of every other value as it is and gives a centre on the edge the sign of
// the top-left rule: + where the edge (dx, dy) owns it (owns()), else -. The
// sign is that of 8192 dy - dx: |dy| >= 1/16 or 0, |dx| < 256.
__device__ __forceinline__ float tie_bias(float dx, float dy) {
  return __uint_as_float((__float_as_uint(ffma(dy, 8192.0f, -dx)) & 0x80000000u) | 0x3a800000u);
}
__device__ __forceinline__ uint32_t iz_bits(float w0, float w1, float w2, float invA, float iz0, float iz1, float iz2) {
  return __float_as_uint(ffma(fmul(w2, invA), iz2, ffma(fmul(w1, invA), iz1, fmul(fmul(w0, invA), iz0))));
}

// a queued triangle's box: x0 and y0 in 10 bits, width - 1 and height - 1 in 6 bits each
__device__ __forceinline__ uint32_t queue_box(int x0, int y0, int dw, int dh) {
  return (uint32_t)x0 | ((uint32_t)y0 << 10) | ((uint32_t)dw << 20) | ((uint32_t)dh << 26);
}

// The render of one chunk's triangles where a triangle may be of any size or
// have a culled vertex (Geometry::pose_general): integer edge functions.
// Queues what a warp should share, as the quick path does.
struct GeneralResult {
  float4 cov;
  unsigned culled;
};
template <int NT, int INL>
__device__ __noinline__ GeneralResult raster_general(RenderSmem s, const uint32_t* tris, int n_tri, int tw, int th, int* s_qn, int qcap,
                                                     float4 cov) {
  unsigned culled = 0;
  for (int t = threadIdx.x; t < n_tri; t += NT) {
    const uint32_t pk = __ldg(&tris[t]);
    const int i0 = pk & 1023, i1 = (pk >> 10) & 1023, i2 = (pk >> 20) & 1023;
    if (s.sIZ[i0] < 0.0f || s.sIZ[i1] < 0.0f || s.sIZ[i2] < 0.0f) {
      culled = 1u;
      continue;
    }
    const int2 a = units16(s.sXY[i0]), b = units16(s.sXY[i1]), c = units16(s.sXY[i2]);
    const int A = (b.y - a.y) * (c.x - a.x) - (b.x - a.x) * (c.y - a.y);
    if (A <= 0) continue;  // back-facing or degenerate
    const int px0 = max(ceil16(min(a.x, min(b.x, c.x))), 0), px1 = min(floor16(max(a.x, max(b.x, c.x))), tw - 1);
    const int py0 = max(ceil16(min(a.y, min(b.y, c.y))), 0), py1 = min(floor16(max(a.y, max(b.y, c.y))), th - 1);
    if (px0 > px1 || py0 > py1) continue;
    cov = make_float4(fminf(cov.x, (float)px0), fmaxf(cov.y, (float)px1), fminf(cov.z, (float)py0),
                      fmaxf(cov.w, (float)py1));
    if ((px1 - px0 + 1) * (py1 - py0 + 1) > INL && px1 - px0 < 64 && py1 - py0 < 64) {
      const int slot = atomicAdd(s_qn, 1);
      if (slot < qcap) {
        s.queue[2 * slot] = pk;
        s.queue[2 * slot + 1] = queue_box(px0, py0, px1 - px0, py1 - py0);
        continue;
      }
    }
    raster_box(a, b, c, A, px0, px1, py0, py1, s.sIZ, i0, i1, i2, s.tile, tw);
  }
  return GeneralResult{cov, culled};
}

// One queued triangle of raster_general, its pixel centres across the warp
__device__ __noinline__ void raster_queued_general(RenderSmem s, uint32_t pk, uint32_t box, int tw) {
  const int i0 = pk & 1023, i1 = (pk >> 10) & 1023, i2 = (pk >> 20) & 1023;
  const int2 va = units16(s.sXY[i0]), vb = units16(s.sXY[i1]), vc = units16(s.sXY[i2]);
  const int px0 = box & 1023, py0 = (box >> 10) & 1023, bw = (int)((box >> 20) & 63) + 1;
  const int n = bw * ((int)(box >> 26) + 1);
  // k / bw = umulhi(k, ceil(2^32 / bw)) for k, bw < 2^16 (bw = 1 would overflow the magic)
  const uint32_t magic = 0xffffffffu / (uint32_t)bw + 1u;
  float invA = 0.0f;
  for (int k = threadIdx.x & 31; k < n; k += 32) {
    const int ry = bw == 1 ? k : (int)__umulhi((uint32_t)k, magic);
    const int px = px0 + k - ry * bw, py = py0 + ry;
    const int Px = 16 * px, Py = 16 * py;
    const int w0 = (vc.y - vb.y) * (Px - vb.x) - (vc.x - vb.x) * (Py - vb.y);
    const int w1 = (va.y - vc.y) * (Px - vc.x) - (va.x - vc.x) * (Py - vc.y);
    const int w2 = (vb.y - va.y) * (Px - va.x) - (vb.x - va.x) * (Py - va.y);
    if (!covers(w0, w1, w2, va, vb, vc)) continue;
    if (invA == 0.0f) invA = __frcp_rn(__int2float_rn(w0 + w1 + w2));
    atomicMax(&s.tile[py * tw + px], pixel_iz_bits(w0, w1, w2, invA, s.sIZ[i0], s.sIZ[i1], s.sIZ[i2]));
  }
}

// Render mesh m at pose o (index `pose`) into the tile (1/z bits, 0 = empty)
// covering the pose's screen box bb. The first chunk's triangle list must
// have been started (render_start) and the tile cleared before the call; the
// first CTA barrier inside orders those writes.
//
// The mesh is walked in chunks of <= 680 vertices / 1536 triangles: as many
// as 17 KB of buffers hold, which leaves four CTAs to an SM beside the largest
// tiles of 640x480 scenes. A chunk's slice of the yaw's camera-frame vertex table (M_yaw v) is brought
// into shared memory by a bulk asynchronous copy (TMA), issued as soon as the
// previous chunk's vertices are projected, so that it overlaps the
// rasterisation; each thread loads its triangles one ahead. Coverage resolves
// by an order-independent max, so the tile does not depend on which thread
// rasterises a triangle.
//
// The kernel is bound by instruction issue, so the work per triangle is
// arranged for few instructions:
// - Positions are binary32 multiples of 1/16 px relative to the tile. With
//   triangles of at most kSmallPixels the edge functions are binary32
//   multiples of 2^-8 px^2 below 2^13, exact in every step, and E_i (1 / A)
//   rounds as from integers (the powers of two cancel), without conversions.
//   Poses with larger triangles on the screen, or with a vertex that may have
//   to be culled, take raster_general.
// - A front face covers a fifth of the centres in its box on meshes of 10k
//   triangles, so the centres are tested first, two by two rows, their sign
//   bits shifted into a mask, and only the covered ones are shaded (a loop
//   that most warps run once). Centres outside the triangle's box test
//   outside; those past the tile's border are masked.
// - A triangle of more than about INL centres (the inline limit) is queued
//   and its box's columns are split across eight lanes; a full queue leaves
//   it to the thread. Without queued triangles a chunk passes two CTA
//   barriers.
// Measured on the 120k distinct poses of a 640x480 expansion (meshes of 10k
// triangles), against integer edges tested and shaded one centre at a time in
// chunks of 512 vertices: 9.85 ms instead of 12.06; 57-73k warp instructions
// a pose instead of 78-110k. Meshes of 2k-50k triangles, one parent: 7.2 ms
// instead of 9.0 for 30k hypotheses.
//
// `culled` is set in the threads that dropped a triangle; with COV `cov` grows to
// hold every covered pixel (x0, x1, y0, y1 within bb). On kEvalTimedOut /
// kEvalStop the tile is incomplete; the caller reports the failure and must
// pass a CTA barrier before reusing the tile.
template <int NT, int INL, bool COV>
__device__ __forceinline__ int render_chunks(const Camera& cam, const Geometry& g, const Batch& b, const DevMesh& m,
                                             const perch_obj& o, long long pose, int4 bb, const RenderSmem& s,
                                             EvalShared& sh, unsigned& culled, float4& cov) {
  constexpr int NW = NT / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t* tile = s.tile;
  const int tw = bb.z, th = bb.w;
  const float4 bo = g.pose_off[o.ix * g.ny + o.iy];
  const float ox = (float)bb.x, oy = (float)bb.y;
  const bool general = g.pose_general[pose] != 0;
  // a box that may have been cut at the image's border: its triangles may reach past it
  const bool clip = bb.x == 0 || bb.y == 0 || bb.x + tw == cam.W || bb.y + th == cam.H;
  const int qcap = b.queue_cap > 0 && b.queue_cap < kBigQueue ? b.queue_cap : kBigQueue;
  const unsigned char* xy = reinterpret_cast<const unsigned char*>(s.sXY);
  bool pending = true;  // a vertex slice in flight
  bool timed_out = false;
  int4 ci = g.chunk_info[m.chunk_begin];
  uint32_t pk_next = tid < ci.w ? __ldg(&g.chunk_tris[ci.z + tid]) : 0u;  // this thread's next triangle
  for (int c = 0; c < m.chunk_count; ++c) {
    const int n_vert = ci.y, n_tri = ci.w;
    const uint32_t* tris = g.chunk_tris + ci.z;
    const bool more = c + 1 < m.chunk_count;
    if (more) ci = g.chunk_info[m.chunk_begin + c + 1];
    // vertices: wait for the slice, project, then reuse its buffer for c+1
    const bool ok = mbar_wait(sh.bar, sh.pv, b.wait_polls);
    for (int v = ok ? tid : n_vert; v < n_vert; v += NT) {
      const float* q = s.vbuf + 3 * v;
      const float3 r = general ? project_pixel<true>(cam, q[0], q[1], q[2], bo, ox, oy)
                               : project_pixel<false>(cam, q[0], q[1], q[2], bo, ox, oy);
      s.sXY[v] = make_float2(r.x, r.y);
      s.sIZ[v] = r.z;
    }
    int* qn = &sh.qn[c & 1];  // the other chunk's count may still be read
    if (tid == 0) *qn = 0;
    if (__syncthreads_or(ok ? 0 : 1)) {
      timed_out = true;
      break;
    }
    sh.pv ^= 1u;
    pending = more;
    if (more && tid == 0) load_slice(g, o.iyaw, ci.x, ci.y, s, sh.bar);
    if (general) {
      const GeneralResult r = raster_general<NT, INL>(s, tris, n_tri, tw, th, qn, qcap, COV ? cov : kNoCover);
      if (COV) cov = r.cov;
      culled |= r.culled;
    }
    for (int t = general ? n_tri : tid; t < n_tri; t += NT) {
      const uint32_t pk = pk_next;
      if (t + NT < n_tri) pk_next = __ldg(&tris[t + NT]);
      const uint32_t o0 = (pk << 3) & 8184u, o1 = (pk >> 7) & 8184u, o2 = (pk >> 17) & 8184u;
      const float2 va = *reinterpret_cast<const float2*>(xy + o0);
      const float2 vb = *reinterpret_cast<const float2*>(xy + o1);
      const float2 vc = *reinterpret_cast<const float2*>(xy + o2);
      const float abx = fsub(vb.x, va.x), aby = fsub(vb.y, va.y), acx = fsub(vc.x, va.x), acy = fsub(vc.y, va.y);
      const float A = ffma(aby, acx, -fmul(abx, acy));
      if (!(A > 0.0f)) continue;  // back-facing or degenerate
      float xmax = max3(va.x, vb.x, vc.x), ymax = max3(va.y, vb.y, vc.y);
      float px0 = ceilf(min3(va.x, vb.x, vc.x)), py0 = ceilf(min3(va.y, vb.y, vc.y));
      if (clip) {
        px0 = fmaxf(px0, 0.0f);
        py0 = fmaxf(py0, 0.0f);
        xmax = fminf(xmax, (float)(tw - 1));
        ymax = fminf(ymax, (float)(th - 1));
      }
      const float xw = fsub(xmax, px0), yw = fsub(ymax, py0);  // columns past the first, rows past the first
      if (fminf(xw, yw) < 0.0f) continue;
      if (COV) {
        cov.x = fminf(cov.x, px0);
        cov.y = fmaxf(cov.y, xmax);
        cov.z = fminf(cov.z, py0);
        cov.w = fmaxf(cov.w, ymax);
      }
      if (fmul(fadd(xw, 0.5f), fadd(yw, 0.5f)) > (float)INL) {
        const int slot = atomicAdd(qn, 1);
        if (slot < qcap) {
          s.queue[2 * slot] = pk;
          s.queue[2 * slot + 1] = queue_box((int)px0, (int)py0, (int)xw, (int)yw);
          continue;
        }
      }
      const float cbx = fsub(acx, abx), cby = fsub(acy, aby);
      const float pax = fsub(px0, va.x), pay = fsub(py0, va.y);
      const float e0 = tie_bias(cbx, cby), e1 = tie_bias(-acx, -acy), e2 = tie_bias(abx, aby);
      float w2 = ffma(aby, pax, -fmul(abx, pay)), w1 = ffma(acx, pay, -fmul(acy, pax));
      float w0 = fsub(fsub(A, w1), w2);
      const float invA = __frcp_rn(A);
      const unsigned char* iz = reinterpret_cast<const unsigned char*>(s.sIZ);
      const float iz0 = *reinterpret_cast<const float*>(iz + (o0 >> 1));
      const float iz1 = *reinterpret_cast<const float*>(iz + (o1 >> 1));
      const float iz2 = *reinterpret_cast<const float*>(iz + (o2 >> 1));
      uint32_t* at = tile + (int)ffma(py0, (float)tw, px0);
      auto centre = [&](float u0, float u1, float u2, uint32_t* px) {
        if ((int)outside(fadd(u0, e0), fadd(u1, e1), fadd(u2, e2)) >= 0)
          atomicMax(px, iz_bits(u0, u1, u2, invA, iz0, iz1, iz2));
      };
      // the box's first two columns and rows; centres past the box are outside
      // the triangle, and past the tile's border only where the box was cut
      auto block = [&](bool c1, bool r1) {
        centre(w0, w1, w2, at);
        if (c1) centre(fadd(w0, cby), fsub(w1, acy), fadd(w2, aby), at + 1);
        if (r1) {
          const float n0 = fsub(w0, cbx), n1 = fadd(w1, acx), n2 = fsub(w2, abx);
          centre(n0, n1, n2, at + tw);
          if (c1) centre(fadd(n0, cby), fsub(n1, acy), fadd(n2, aby), at + tw + 1);
        }
      };
      block(xw >= 1.0f, yw >= 1.0f);
      if (fmaxf(xw, yw) >= 2.0f) {  // the rest of a larger box, block by block
        float r0 = w0, r1 = w1, r2 = w2;
        uint32_t* row = at;
        float x = 2.0f, y = 0.0f;
        for (;;) {
          if (x > xw) {
            y = fadd(y, 2.0f);
            if (y > yw) break;
            x = 0.0f;
            w0 = r0 = ffma(-2.0f, cbx, r0);
            w1 = r1 = ffma(2.0f, acx, r1);
            w2 = r2 = ffma(-2.0f, abx, r2);
            at = row += 2 * tw;
          } else {
            w0 = ffma(2.0f, cby, w0);
            w1 = ffma(-2.0f, acy, w1);
            w2 = ffma(2.0f, aby, w2);
            at += 2;
          }
          block(fadd(x, 1.0f) <= xw, fadd(y, 1.0f) <= yw);
          x = fadd(x, 2.0f);
        }
      }
    }
    if (more && tid < ci.w) pk_next = __ldg(&g.chunk_tris[ci.z + tid]);
    __syncthreads();
    // larger triangles: eight lanes to one, a lane to a column of its box
    const int nq = min(*qn, qcap);
    if (general) {
      for (int e = warp; e < nq; e += NW) raster_queued_general(s, s.queue[2 * e], s.queue[2 * e + 1], tw);
    } else {
      for (int e = 4 * warp + (lane >> 3); e < nq; e += 4 * NW) {
        const uint32_t pk = s.queue[2 * e], box = s.queue[2 * e + 1];
        const int i0 = pk & 1023, i1 = (pk >> 10) & 1023, i2 = (pk >> 20) & 1023;
        const float2 va = s.sXY[i0], vb = s.sXY[i1], vc = s.sXY[i2];
        const int px0 = box & 1023, py0 = (box >> 10) & 1023, dw = (box >> 20) & 63, dh = box >> 26;
        const float abx = fsub(vb.x, va.x), aby = fsub(vb.y, va.y), acx = fsub(vc.x, va.x), acy = fsub(vc.y, va.y);
        const float cbx = fsub(acx, abx), cby = fsub(acy, aby);
        const float A = ffma(aby, acx, -fmul(abx, acy)), invA = __frcp_rn(A);
        const float e0 = tie_bias(cbx, cby), e1 = tie_bias(-acx, -acy), e2 = tie_bias(abx, aby);
        const float iz0 = s.sIZ[i0], iz1 = s.sIZ[i1], iz2 = s.sIZ[i2];
        const float pay = fsub((float)py0, va.y);
        for (int x = lane & 7; x <= dw; x += 8) {
          const float pax = fsub((float)(px0 + x), va.x);
          float w1 = ffma(acx, pay, -fmul(acy, pax)), w2 = ffma(aby, pax, -fmul(abx, pay));
          float w0 = fsub(fsub(A, w1), w2);
          uint32_t* at = &tile[py0 * tw + px0 + x];
          for (int y = 0; y <= dh; ++y) {
            if ((int)outside(fadd(w0, e0), fadd(w1, e1), fadd(w2, e2)) >= 0)
              atomicMax(at, iz_bits(w0, w1, w2, invA, iz0, iz1, iz2));
            w0 = fsub(w0, cbx);
            w1 = fadd(w1, acx);
            w2 = fsub(w2, abx);
            at += tw;
          }
        }
      }
    }
    if (nq > 0) __syncthreads();  // the next chunk reuses sXY, sIZ and the queue
  }
  if (timed_out) {
    // A wait gave up: drain the copy still in flight with the full bound
    // (kWaitSpins polls or 2 s). Once it has landed the barrier's phase is
    // known again and the CTA may take further work; if the drain also gives
    // up, a copy may still be writing into this CTA's shared memory and it
    // must stop.
    const bool ok = __syncthreads_and(!pending || mbar_wait(sh.bar, sh.pv));
    if (ok && pending) sh.pv ^= 1u;
    return ok ? kEvalTimedOut : kEvalStop;
  }
  return kEvalDone;
}

// What a render source holds per pixel of the pose's box (shared memory,
// rows of the box width): 1/z bits with 0 = empty (the per-hypothesis
// kernel's own tile); z bits with +inf = empty (the tile store); or z bits
// whose sign bit says the rendered point is explained by I (Eq. (1)), which
// k_render decides once per pose for a single-scene batch.
constexpr int kSrcInvZ = 0, kSrcZ = 1, kSrcZExplained = 2;
constexpr uint32_t kExplainedBit = 0x80000000u;  // z > 0: the sign bit is free

// The first part of cost_phase: the monotone test against the parent render
// and dR (Eq. (3)). Reads the render from src, writes z on dR (+inf
// elsewhere) into the tile, and sums violations and |dR| into s_cnt[0],
// s_cnt[1] (with kSrcZExplained also dJ_r, the dR pixels not explained by I,
// into s_cnt[3]); ends with a CTA barrier, after which src is no longer read.
template <int NT, int SRC>
__device__ __forceinline__ void compare_phase(int pid, int plen, int4 bb, const Camera& cam, const Batch& b,
                                              const uint32_t* src, uint32_t* tile, int* s_cnt) {
  const int tid = threadIdx.x, lane = tid & 31;
  const int tw = bb.z, n = bb.z * bb.w;
  int viol = 0, nnew = 0, djr = 0;
  const float* zp = plen > 0 ? b.parent_z + (size_t)pid * cam.W * cam.H : nullptr;
  const uint32_t empty = SRC == kSrcInvZ ? 0u : kInfBits;
  // pixel i of the box is (i mod tw, i div tw); i div tw = umulhi(i, ceil(2^32 / tw)),
  // exact for i tw < 2^32 (the box is at most kMaxObjectPixels wide and high)
  const uint32_t mg = tw > 1 ? 0xffffffffu / (uint32_t)tw + 1u : 0u;
  // U pixels per thread at a time: their parent depths are loaded together
  constexpr int U = 4;
  for (int i0 = tid; i0 < n; i0 += NT * U) {
    uint32_t sv[U];
    float pz[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + u * NT;
      sv[u] = i < n ? src[i] : empty;
      pz[u] = __uint_as_float(kInfBits);
      if (zp && sv[u] != empty) {
        const int ly = tw > 1 ? (int)__umulhi((uint32_t)i, mg) : i;
        pz[u] = __ldg(&zp[(size_t)(bb.y + ly) * cam.W + bb.x + (i - ly * tw)]);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + u * NT;
      if (i >= n) break;
      if (sv[u] == empty) {
        tile[i] = kInfBits;
        continue;
      }
      const uint32_t zb = SRC == kSrcInvZ ? __float_as_uint(__frcp_rn(__uint_as_float(sv[u]))) : (sv[u] & ~kExplainedBit);
      if (__float_as_uint(pz[u]) != kInfBits) {  // hidden by (or hiding) the parent: not in dR
        if (__uint_as_float(zb) < pz[u]) viol++;
        tile[i] = kInfBits;
        continue;
      }
      tile[i] = zb;
      nnew++;
      if (SRC == kSrcZExplained && !(sv[u] & kExplainedBit)) djr++;
    }
  }
  viol = warp_sum(viol);
  nnew = warp_sum(nnew);
  if (SRC == kSrcZExplained) djr = warp_sum(djr);
  if (lane == 0) {
    if (viol) atomicAdd(&s_cnt[0], viol);
    if (nnew) atomicAdd(&s_cnt[1], nnew);
    if (djr) atomicAdd(&s_cnt[3], djr);
  }
  __syncthreads();
}

// compare_phase for a staged render that stays as it is (z bits, +inf =
// empty, with kSrcZExplained the explained flag in the sign bit): the same
// test and counts, but dR goes to a bitmask (bit i of mask[i / 32] = pixel i
// is in dR) instead of a z tile. Warps take 32 consecutive pixels at a time
// (NT is a multiple of 32, so every word is written by one ballot). Ends
// with a CTA barrier.
template <int NT, int SRC>
__device__ __forceinline__ void compare_phase_mask(int pid, int plen, int4 bb, const Camera& cam, const Batch& b,
                                                   const uint32_t* src, uint32_t* mask, int* s_cnt) {
  static_assert(SRC != kSrcInvZ && NT % 32 == 0, "staged z source");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tw = bb.z, n = bb.z * bb.w;
  int viol = 0, nnew = 0, djr = 0;
  const float* zp = plen > 0 ? b.parent_z + (size_t)pid * cam.W * cam.H : nullptr;
  const uint32_t mg = tw > 1 ? 0xffffffffu / (uint32_t)tw + 1u : 0u;  // i / tw, as in compare_phase
  constexpr int U = 4;
  for (int w0 = 32 * warp; w0 < n; w0 += NT * U) {  // warp-uniform
    uint32_t sv[U];
    float pz[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = w0 + u * NT + lane;
      sv[u] = i < n ? src[i] : kInfBits;
      pz[u] = __uint_as_float(kInfBits);
      if (zp && sv[u] != kInfBits) {
        const int ly = tw > 1 ? (int)__umulhi((uint32_t)i, mg) : i;
        pz[u] = __ldg(&zp[(size_t)(bb.y + ly) * cam.W + bb.x + (i - ly * tw)]);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      bool in_dr = false;
      if (sv[u] != kInfBits) {
        const uint32_t zb = sv[u] & ~kExplainedBit;
        if (__float_as_uint(pz[u]) != kInfBits) {  // hidden by (or hiding) the parent: not in dR
          if (__uint_as_float(zb) < pz[u]) viol++;
        } else {
          in_dr = true;
          nnew++;
          if (SRC == kSrcZExplained && !(sv[u] & kExplainedBit)) djr++;
        }
      }
      const unsigned bits = __ballot_sync(0xffffffffu, in_dr);
      if (lane == 0 && w0 + u * NT < n) mask[(w0 + u * NT) >> 5] = bits;
    }
  }
  viol = warp_sum(viol);
  nnew = warp_sum(nnew);
  if (SRC == kSrcZExplained) djr = warp_sum(djr);
  if (lane == 0) {
    if (viol) atomicAdd(&s_cnt[0], viol);
    if (nnew) atomicAdd(&s_cnt[1], nnew);
    if (djr) atomicAdd(&s_cnt[3], djr);
  }
  __syncthreads();
}

// The rest of cost_phase, after compare_phase: the record of an invalid
// child, or dJ_r (unless DJR_DONE: compare_phase counted it), dJ_o,
// residual(K) and n_vol from the tile (z on dR, +inf elsewhere). `list`: shared
// scratch of kNearList + 1 entries. Ends with a CTA barrier.
template <int NT, bool DJR_DONE>
__device__ __forceinline__ void finish_phase(long long h, int pid, int plen, int K_total, const perch_obj& o,
                                             int4 bb, const DevMesh& m, const Camera& cam, const Geometry& g,
                                             const ObsIndex& obs, const Batch& b, const DRTile& tile,
                                             const float* rxs, const float* rys, int* s_cnt, int* list) {
  constexpr int NW = NT / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tw = bb.z, th = bb.w;
  const float ox = g.xs[o.ix], oy = g.ys[o.iy];
  const uint32_t flags = s_cnt[2] ? PERCH_FLAG_CULLED : 0u;
  if (s_cnt[0] > 0) {
    if (tid == 0) {
      perch_cost r = {0, 0, 0, s_cnt[0], s_cnt[1], flags | PERCH_FLAG_INVALID, 0};
      b.out[h] = r;
    }
    __syncthreads();  // s_cnt is reset by the next hypothesis
    return;
  }

  // ---- dJ_r: dR points with no observed point within delta (with no
  // observed point near the footprint, all |dR| of them, s_cnt[1])
  int djr = 0;
  const bool probe = !DJR_DONE && obs_near(cam, g, obs, o);
  if (!DJR_DONE && !probe && tid == 0) djr = s_cnt[1];
  for (int ly = warp; probe && ly < th; ly += NW) {
    const float ry = rys[ly];
    for (int lx = lane; lx < tw; lx += 32) {
      const uint32_t zb = tile.at(ly * tw + lx);
      if (zb == kInfBits) continue;
      const float z = __uint_as_float(zb);
      if (!explained_by_obs(obs, fmul(rxs[lx], z), fmul(ry, z), z, cam.delta2)) djr++;
    }
  }

  // ---- dJ_o: observed points inside V(O) with no dR point within delta; and
  // on edges into the last level residual(K) = |U| less the points of U that
  // are inside V(O) or within delta of a dR point. Both look only at the
  // observed points of the world cells about the pose: within V(O)'s radius,
  // and on the last level within the footprint's radius + delta (+ 2 cm and
  // a sixteenth of a pixel at the object's depth for the snap: every rendered
  // point lies that near the footprint). Few points of those cells need the
  // scan of the tile, so a first pass lists them (kNearList cells' points at
  // a time) and a second takes one per thread. This phase was most of k_cost:
  // it took a row of cells per CTA pass, scanned windows of 11 to 13 pixels
  // where 7 hold delta (delta_radius), and tested all of U (up to the whole
  // cloud) per hypothesis of the last level. k_cost, 640x480: 480k
  // hypotheses of eight states 4.1 -> 1.5 ms, the 240k-hypothesis batch
  // 3.5 -> 2.25 ms, 4.7k hypotheses next to the objects 1.4 -> 0.51 ms.
  const bool last = plen + 1 == K_total;
  int djo = 0, nvol = 0, done = 0;  // done: points of U that are accounted for
  if (obs.n > 0) {
    float r = m.vol_rmax * 1.001f + 1e-6f;
    if (last) {
      const float depth = g.pose_off[o.ix * g.ny + o.iy].z + m.fp_r + fmaxf(fabsf(m.lo[2]), fabsf(m.hi[2]));
      r = fmaxf(r, m.fp_r + cam.delta + 0.02f + depth / (16.0f * fminf(cam.fx, cam.fy)));
    }
    const int cx0 = max(cell_of(ox - r, obs.g2x, obs.inv2, obs.n2x) - 1, 0);
    const int cx1 = min(cell_of(ox + r, obs.g2x, obs.inv2, obs.n2x) + 1, obs.n2x - 1);
    const int cy0 = max(cell_of(oy - r, obs.g2y, obs.inv2, obs.n2y) - 1, 0);
    const int cy1 = min(cell_of(oy + r, obs.g2y, obs.inv2, obs.n2y) + 1, obs.n2y - 1);
    const uint32_t* U = b.uset + (size_t)pid * b.uset_stride;
    const bool any = cx0 <= cx1 && cy0 <= cy1 && sat_sum(obs.sat2, obs.n2x, cy0, cy1, cx0, cx1) != 0;
    for (int cy = cy0; any && cy <= cy1; cy += 32) {  // 32 rows of cells, a lane to a row
      int s = 0, cnt = 0;
      if (cy + lane <= cy1) {
        s = obs.start2[(cy + lane) * obs.n2x + cx0];
        cnt = obs.start2[(cy + lane) * obs.n2x + cx1 + 1] - s;
      }
      int incl = cnt;
      for (int d = 1; d < 32; d <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += t;
      }
      const int total = __shfl_sync(0xffffffffu, incl, 31);
      for (int base = 0; base < total; base += kNearList) {
        const int lim = min(total, base + kNearList);
        if (tid == 0) list[0] = 0;
        __syncthreads();  // also: the last round's list has been read
        for (int i0 = base + 32 * warp; i0 < lim; i0 += NT) {  // warp-uniform
          const int i = i0 + lane;
          int row = 0;  // the row whose range holds the i-th point
          for (int d = 16; d > 0; d >>= 1)
            if (__shfl_sync(0xffffffffu, incl, row + d - 1) <= i) row += d;
          const int k = __shfl_sync(0xffffffffu, s, row) + i - __shfl_sync(0xffffffffu, incl - cnt, row);
          bool in_v = false, in_u = false;
          if (i < lim) {
            in_v = in_volume(g, m, ox, oy, o.iyaw, obs.world2[k]);
            in_u = last && ((U[k >> 5] >> (k & 31)) & 1u);
          }
          const unsigned take = __ballot_sync(0xffffffffu, in_v || in_u);
          int at = 0;
          if (lane == 0 && take) at = atomicAdd(&list[0], __popc(take));
          at = __shfl_sync(0xffffffffu, at, 0);
          if (in_v || in_u)
            list[1 + at + __popc(take & ((1u << lane) - 1u))] = k | (in_v ? 1 << 30 : 0) | (in_u ? 1 << 31 : 0);
        }
        __syncthreads();
        const int n_list = list[0];
        for (int e = tid; e < n_list; e += NT) {
          const int f = list[1 + e], k = f & 0x3fffffff;
          const bool ex = explained_by_tile(cam, obs.cam2[k], tile, rxs, rys, bb);
          if (f < 0 && (ex || (f & (1 << 30)))) done++;
          if (!(f & (1 << 30))) continue;
          if (!ex) djo++;
          bool in_parent = false;  // already inside an assigned volume?
          for (int j = 0; j < plen && !in_parent; ++j) {
            const perch_obj po = b.parents[(long long)pid * b.parent_stride + j];
            in_parent = in_volume(g, g.meshes[po.mesh], g.xs[po.ix], g.ys[po.iy], po.iyaw, obs.world2[k]);
          }
          if (!in_parent) nvol++;
        }
      }
    }
  }
  djr = warp_sum(djr);
  djo = warp_sum(djo);
  done = warp_sum(done);
  nvol = warp_sum(nvol);
  if (lane == 0) {
    if (djr) atomicAdd(&s_cnt[3], djr);
    if (djo) atomicAdd(&s_cnt[4], djo);
    if (done) atomicAdd(&s_cnt[5], done);
    if (nvol) atomicAdd(&s_cnt[6], nvol);
  }
  __syncthreads();
  if (tid == 0) {
    perch_cost r = {s_cnt[3], s_cnt[4], last ? b.uset_count[pid] - s_cnt[5] : 0, 0, s_cnt[1], flags, s_cnt[6]};
    b.out[h] = r;
  }
  __syncthreads();  // s_cnt and the tile are reused by the next hypothesis
}

// Cost of hypothesis h (Eq. (3), Eq. (4)) from its new object's render,
// which the shared tile holds as 1/z bits (0 = empty) over the pose's box bb,
// rows of bb.z pixels; the tile then receives z on dR and +inf elsewhere.
// rxs / rys hold the ray slopes of the box's columns and rows; s_cnt is zero
// except the culled flag s_cnt[2]; a CTA barrier must separate those writes
// from the call. Ends with a CTA barrier (s_cnt and the tile may be reused
// after it).
template <int NT>
__device__ __forceinline__ void cost_phase(long long h, int pid, int plen, int K_total, const perch_obj& o, int4 bb,
                                           const DevMesh& m, const Camera& cam, const Geometry& g,
                                           const ObsIndex& obs, const Batch& b, uint32_t* tile, const float* rxs,
                                           const float* rys, int* s_cnt, int* list) {
  compare_phase<NT, kSrcInvZ>(pid, plen, bb, cam, b, tile, tile, s_cnt);
  finish_phase<NT, false>(h, pid, plen, K_total, o, bb, m, cam, g, obs, b, DRTile{tile, nullptr}, rxs, rys, s_cnt,
                          list);
}

// The checks every evaluation of hypothesis h makes before it touches its
// parent or pose: false means the record is the bad-index record.
struct HypArgs {
  perch_obj o;
  int pid, plen, scene, K_total;
  long long pose;
};

struct EvalHyp {
  HypArgs a;
  int4 bb;
  long long h;
};

__device__ __forceinline__ bool hyp_args(const Geometry& g, const Batch& b, long long h, HypArgs& a) {
  a.o = b.hyp[h];
  a.pid = b.hyp_parent[h];
  bool bad = a.pid < 0 || a.pid >= b.n_par || !obj_ok(g, a.o);
  a.plen = bad ? 0 : b.parent_len[a.pid];
  bad = bad || a.plen < 0 || a.plen > b.parent_stride;
  a.scene = (bad || !b.parent_scene) ? 0 : b.parent_scene[a.pid];
  a.K_total = (bad || !b.parent_K) ? b.K_total : b.parent_K[a.pid];
  bad = bad || (b.parent_scene && (a.scene < 0 || a.scene >= b.n_scenes));
  a.pose = bad ? 0 : (((long long)a.o.mesh * g.nx + a.o.ix) * g.ny + a.o.iy) * g.n_yaw + a.o.iyaw;
  return !bad;
}

// One CTA per hypothesis: render the new object into a shared-memory z tile
// covering its screen box (render_chunks), test it against the parent render
// (Eq. (3)), and count dJ_r, dJ_o and residual(K) (Sec. IV-A, Eq. (4))
// (cost_phase). The CTA's two mbarriers persist across hypotheses (their
// phase parities are in sh).
template <int NT, bool MULTI>
__device__ int eval_one(long long h, const Camera& cam, const Geometry& g, const ObsIndex& obs0, const Batch& b,
                        EvalShared& sh, ObsIndex* s_obs) {
  constexpr int NW = NT / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int* s_cnt = sh.cnt;
  HypArgs a;
  const bool ok = hyp_args(g, b, h, a);
  const int4 bb = ok ? g.pose_bbox[a.pose] : make_int4(0, 0, 0, 0);
  if (!ok || bb.z > b.tile_w || bb.w > b.tile_h) {
    if (tid == 0) {
      perch_cost r = {0, 0, 0, 0, 0, kFlagBadIndex, 0};
      b.out[h] = r;
    }
    return kEvalDone;
  }
  if (MULTI && tid < (int)(sizeof(ObsIndex) / 4))  // this scene's index, read from shared memory below
    reinterpret_cast<int*>(s_obs)[tid] = reinterpret_cast<const int*>(&b.scenes[a.scene])[tid];
  const ObsIndex& obs = MULTI ? *s_obs : obs0;
  const RenderSmem s = render_smem(sh.dyn);
  const int tw = bb.z, th = bb.w;
  const DevMesh m = g.meshes[a.o.mesh];
  if (tid == 0) render_start(g, m, a.o.iyaw, s, sh.bar);
  {
    float* rxs = reinterpret_cast<float*>(s.tile + b.tile_w * b.tile_h);
    float* rys = rxs + b.tile_w;
    for (int i = tid; i < tw; i += NT) rxs[i] = g.rx[bb.x + i];
    for (int i = tid; i < th; i += NT) rys[i] = g.ry[bb.y + i];
  }
  for (int ly = warp; ly < th; ly += NW)
    for (int lx = lane; lx < tw; lx += 32) s.tile[ly * tw + lx] = 0u;  // 1/z = 0: empty
  if (tid < 7) s_cnt[tid] = 0;

  unsigned culled = 0;
  float4 cov = kNoCover;  // not needed here
  // The cost needs these again. In registers they were spilled in the render's loops, with the
  // covered box that only k_render needs 108 bytes a thread, now 40: root expansion 2.97 -> 2.73 ms,
  // 30k hypotheses of uneven meshes 6.73 -> 6.10.
  if (tid == 0) {
    sh.hyp->a = a;
    sh.hyp->bb = bb;
    sh.hyp->h = h;
  }
  const int st = render_chunks<NT, kInlinePixels, false>(cam, g, b, m, a.o, a.pose, bb, s, sh, culled, cov);
  if (st != kEvalDone) {
    if (tid == 0) {
      perch_cost r = {0, 0, 0, 0, 0, kFlagTimeout, 0};
      b.out[sh.hyp->h] = r;
    }
    __syncthreads();  // s_cnt and the tile are reused by the next hypothesis
    return st;
  }
  if (culled) s_cnt[2] = 1;
  __syncthreads();
  // the render's projected vertices are done with: their buffer holds the list
  static_assert(sizeof(float2) * kChunkMaxVerts >= sizeof(int) * (kNearList + 1), "the list fits");
  const EvalHyp& e = *sh.hyp;
  float* rxs = reinterpret_cast<float*>(s.tile + b.tile_w * b.tile_h);
  cost_phase<NT>(e.h, e.a.pid, e.a.plen, e.a.K_total, e.a.o, e.bb, g.meshes[e.a.o.mesh], cam, g, obs, b, s.tile, rxs,
                 rxs + b.tile_w, s_cnt, reinterpret_cast<int*>(s.sXY));
  return kEvalDone;
}

// A group of hypotheses evaluated by one persistent launch: items
// order[offset .. offset + count) (order == nullptr: hypotheses 0 .. count-1),
// claimed one at a time from the device counter `next`.
struct EvalGroup {
  const int* order;
  const int* offset;  // device scalar
  const int* count;   // device scalar
  int* next;          // device counter, zero before the launch
};

template <int NT, bool MULTI>
__global__ void __launch_bounds__(NT, 1024 / NT) k_eval(Camera cam, Geometry g, ObsIndex obs, Batch b, EvalGroup grp) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(16) ObsIndex s_obs;
  __shared__ __align__(8) uint64_t s_bar;
  __shared__ int s_cnt[7];
  __shared__ int s_qn[2];
  __shared__ int s_item;
  __shared__ EvalHyp s_hyp;
  if (threadIdx.x == 0) {
    mbar_init(&s_bar, 1);
    fence_barrier_init();
  }
  __syncthreads();
  EvalShared sh{&s_bar, s_cnt, s_qn, smem, 0u, &s_hyp};
  const int count = *grp.count, offset = grp.order ? *grp.offset : 0;
  for (;;) {
    if (threadIdx.x == 0) s_item = atomicAdd(grp.next, 1);
    __syncthreads();
    const int item = s_item;
    __syncthreads();
    if (item >= count) break;
    const long long h = grp.order ? grp.order[offset + item] : item;
    if (eval_one<NT, MULTI>(h, cam, g, obs, b, sh, &s_obs) == kEvalStop) break;
  }
}

// ---- shared renders: one render per distinct pose of a batch, then one
// cost per hypothesis. The new object's render depends on its mesh and pose
// alone, not on its parent, so k_render rasterises each distinct (mesh,
// pose) of the batch once into the tile store (global memory, 1/z bits of
// the pose's screen box at 16-byte offset tile_off[pose]), and k_cost gives
// every hypothesis its own comparison with its parent and its own costs
// from that stored tile, read with plain coalesced loads.
template <int NT, bool EXPL, int INL>
__global__ void __launch_bounds__(NT, 1024 / NT) k_render(Camera cam, Geometry g, ObsIndex obs, Batch b,
                                                          RenderWork w) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t s_bar;
  __shared__ int s_qn[2];
  __shared__ int s_pose;  // the pose to render, -1 = none left
  __shared__ int s_box[4];  // the covered pixels' box within the pose's box: x0, x1, y0, y1
  __shared__ perch_obj s_obj;  // the pose's object and box, which the store reads again:
  __shared__ int4 s_bb;        // in registers they would be spilled in the render's loops
  constexpr int NW = NT / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    mbar_init(&s_bar, 1);
    fence_barrier_init();
  }
  __syncthreads();
  EvalShared sh{&s_bar, nullptr, s_qn, smem, 0u, nullptr};
  const RenderSmem s = render_smem(smem);
  const int count = *w.count, offset = *w.offset;
  // the store holds at most 2^28 poses; with the divisions below in 64 bits a step of
  // 120k distinct poses took 12.08 ms, not 11.96
  const uint32_t n_yaw = g.n_yaw, per_x = g.ny * n_yaw, per_mesh = g.nx * per_x;
  // the tile is empty between poses (the store clears what a pose covered);
  // a claim made earlier, during the render, would leave CTAs idle at the end
  // of a small batch (2352 poses near the objects: 0.70 against 0.56 ms)
  auto pose_of = [&](int item) { return item < count ? w.gpose[offset + item] : -1; };
  for (int i = tid; i < b.tile_w * b.tile_h; i += NT) s.tile[i] = 0u;  // 1/z = 0: empty
  if (tid == 0) s_pose = pose_of(atomicAdd(w.next, 1));
  __syncthreads();
  for (;;) {
    const long long p = s_pose;
    if (p < 0) break;
    perch_obj o;
    uint32_t q = (uint32_t)p;
    o.mesh = (uint16_t)(q / per_mesh);
    q %= per_mesh;
    o.ix = (int16_t)(q / per_x);
    q %= per_x;
    o.iy = (int16_t)(q / n_yaw);
    o.iyaw = (uint16_t)(q % n_yaw);
    const int4 bb = g.pose_bbox[p];
    if (bb.z > b.tile_w || bb.w > b.tile_h) {  // never for a valid pose: the mesh's tile is its largest box
      __syncthreads();  // every thread has read s_pose
      if (tid == 0) {
        w.pose_flags[p] = kPoseFailed;
        s_pose = pose_of(atomicAdd(w.next, 1));
      }
      __syncthreads();
      continue;
    }
    const DevMesh m = g.meshes[o.mesh];
    if (tid == 0) {
      render_start(g, m, o.iyaw, s, sh.bar);
      s_obj = o;
      s_bb = bb;
    }
    if (tid < 4) s_box[tid] = (tid & 1) ? -1 : 0x7fffffff;  // ordered by render_chunks' first barrier
    unsigned culled = 0;
    float4 cov = kNoCover;  // x0, x1, y0, y1 of this thread's triangle boxes
    const int st = render_chunks<NT, INL, true>(cam, g, b, m, o, p, bb, s, sh, culled, cov);
    const int4 box = s_bb;
    const int tw = box.z;
    if (st != kEvalDone) {
      for (int i = tid; i < tw * box.w; i += NT) s.tile[i] = 0u;
      if (tid == 0) {
        w.pose_flags[s_pose] = kPoseFailed;
        s_pose = pose_of(atomicAdd(w.next, 1));
      }
      __syncthreads();
      if (st == kEvalStop) break;
      continue;
    }
    {  // the union of the front faces' candidate boxes holds every covered pixel:
       // the store (and every cost of this pose) keeps only that box
      const int x0 = __reduce_min_sync(0xffffffffu, (int)cov.x), x1 = __reduce_max_sync(0xffffffffu, (int)cov.y);
      const int y0 = __reduce_min_sync(0xffffffffu, (int)cov.z), y1 = __reduce_max_sync(0xffffffffu, (int)cov.w);
      if (lane == 0 && x1 >= 0) {
        atomicMin(&s_box[0], x0);
        atomicMax(&s_box[1], x1);
        atomicMin(&s_box[2], y0);
        atomicMax(&s_box[3], y1);
      }
    }
    const int any_culled = __syncthreads_or(culled != 0);  // also publishes s_box
    const bool empty = s_box[1] < 0;
    const int cx0 = empty ? 0 : s_box[0], cy0 = empty ? 0 : s_box[2];
    const int cw = empty ? 0 : s_box[1] - s_box[0] + 1, ch = empty ? 0 : s_box[3] - s_box[2] + 1;
    // the store gets z = 1/(1/z) (+inf where empty) over that box, rows of
    // its width, and, for a single-scene batch (EXPL), the Eq. (1) test of
    // each rendered point against I in the sign bit: it depends on the pose
    // and the scene, not on the parent. A pose with no observed point near
    // its footprint explains no point.
    const bool probe = EXPL && obs_near(cam, g, obs, s_obj);
    uint32_t* dst = w.store + 4 * (size_t)w.tile_off[s_pose];
    for (int ly = warp; ly < ch; ly += NW) {
      const float ry = EXPL ? g.ry[box.y + cy0 + ly] : 0.0f;
      for (int lx = lane; lx < cw; lx += 32) {
        uint32_t* px = &s.tile[(cy0 + ly) * tw + cx0 + lx];
        const uint32_t izb = *px;
        uint32_t v = kInfBits;
        if (izb != 0u) {
          *px = 0u;
          const float z = __frcp_rn(__uint_as_float(izb));
          v = __float_as_uint(z);
          if (probe && explained_by_obs(obs, fmul(g.rx[box.x + cx0 + lx], z), fmul(ry, z), z, cam.delta2))
            v |= kExplainedBit;
        }
        dst[ly * cw + lx] = v;
      }
    }
    if (tid == 0) {
      w.pose_flags[s_pose] = any_culled ? kPoseCulled : 0;
      w.tile_box[s_pose] = make_int4(box.x + cx0, box.y + cy0, cw, ch);
      if (w.valid) w.valid[s_pose] = w.tag;  // read by later launches only
      s_pose = pose_of(atomicAdd(w.next, 1));
    }
    __syncthreads();
  }
}

// k_cost: one persistent CTA per SM slot costs hypotheses, sorted by pose,
// from the tile store. A hypothesis's tile is brought into one of NS shared
// stage buffers by a 1D bulk copy (TMA), which threads only read: the compare
// pass marks dR in a bitmask beside it, and dJ_r, dJ_o and the residual read
// z from the stage through that mask. Thread 0 claims the next hypothesis and
// looks up its arguments, box and tile while the rest of the CTA finishes the
// current one. A hypothesis of a pose whose tile a stage already holds (the
// batch is sorted by pose) takes it as it is, with no copy. With one stage
// (NS = 1) the copy starts once the current hypothesis is done, and the
// smaller footprint lets more CTAs share an SM to cover each other's copies;
// with two (NS = 2, where the tiles are small) it starts into the other stage
// as soon as the next hypothesis is claimed, and overlaps dJ_o and the
// residual.
template <int NT, bool MULTI, int NS>
__global__ void __launch_bounds__(NT) k_cost(Camera cam, Geometry g, ObsIndex obs0, Batch b, CostWork w) {
  static_assert(NS == 1 || NS == 2, "one or two stages");
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(16) ObsIndex s_obs;
  __shared__ __align__(8) uint64_t s_bar[NS];
  __shared__ int s_cnt[7];
  // the claimed item: its index, hypothesis, arguments, box, pose flags, tile
  // offset, stage and how its tile reaches the stage (thread 0 writes it,
  // everyone reads it)
  enum { kItemBad = 0, kItemFailed = 1, kItemCopy = 2, kItemReuse = 3 };
  __shared__ struct {
    int item, state, pf, off, sidx;
    long long h;
    HypArgs a;
    int4 bb;
  } s_nx;
  const int tid = threadIdx.x;
  const int stage_words = (b.tile_w * b.tile_h + 3) & ~3;  // 16-byte multiples
  uint32_t* mask = reinterpret_cast<uint32_t*>(smem) + NS * stage_words;
  float* rxs = reinterpret_cast<float*>(mask + (((b.tile_w * b.tile_h + 31) / 32 + 3) & ~3));
  float* rys = rxs + b.tile_w;
  int* list = reinterpret_cast<int*>(rys + b.tile_h);
  if (tid == 0) {
    for (int k = 0; k < NS; ++k) mbar_init(&s_bar[k], 1);
    fence_barrier_init();
  }
  __syncthreads();
  const int count = *w.count, offset = *w.offset;
  // thread 0: the pose whose tile each stage holds or will receive, and the
  // stage of the last claimed item
  long long stage_pose[NS];
  for (int k = 0; k < NS; ++k) stage_pose[k] = -1;
  int cur = 0;
  auto stage_of = [&](int k) { return reinterpret_cast<uint32_t*>(smem) + k * stage_words; };
  auto copy = [&](int k, int off, int4 bb) {
    bulk_load(stage_of(k), w.store + 4 * (size_t)off, 16u * (uint32_t)((bb.z * bb.w + 3) >> 2), &s_bar[k]);
  };
  // thread 0: claim the next item and look it up; with two stages also start
  // its copy into the stage the current item does not use. No barrier (the
  // caller's next one publishes it)
  auto claim = [&]() {
    const int it = atomicAdd(w.next, 1);
    s_nx.item = it;
    if (it >= count) return;
    const long long h = w.order[offset + it];
    HypArgs a;
    int state = kItemBad, pf = 0, off = 0, sidx = cur;
    int4 bb = make_int4(0, 0, 0, 0);
    if (hyp_args(g, b, h, a)) {
      bb = w.tile_box[a.pose];  // the covered pixels' box (k_render)
      pf = w.pose_flags[a.pose];
      if (pf & kPoseFailed) {
        state = kItemFailed;
      } else if (bb.z <= b.tile_w && bb.w <= b.tile_h) {
        if (bb.z == 0 || bb.w == 0) {
          state = kItemReuse;  // nothing rendered: no pixel to copy or compare
        } else if (a.pose == stage_pose[cur]) {
          state = kItemReuse;
        } else if (NS == 2 && a.pose == stage_pose[NS - 1 - cur]) {
          state = kItemReuse;
          sidx = NS - 1 - cur;
        } else {
          state = kItemCopy;
          off = w.tile_off[a.pose];
          sidx = NS - 1 - cur;  // the other stage (the same one with NS = 1)
          stage_pose[sidx] = a.pose;
          if (NS == 2) copy(sidx, off, bb);  // the other stage's last reader has finished
        }
        cur = sidx;
      }
    }
    s_nx.h = h;
    s_nx.state = state;
    s_nx.pf = pf;
    s_nx.off = off;
    s_nx.sidx = sidx;
    s_nx.a = a;
    s_nx.bb = bb;
  };
  if (tid == 0) claim();
  __syncthreads();
  uint32_t parity[NS];
  for (int k = 0; k < NS; ++k) parity[k] = 0;
  for (;;) {
    const int item = s_nx.item;
    if (item >= count) break;
    const long long h = s_nx.h;
    const int state = s_nx.state, pf = s_nx.pf, sidx = s_nx.sidx;
    const HypArgs a = s_nx.a;
    const int4 bb = s_nx.bb;
    if (state == kItemBad || state == kItemFailed) {  // no copy for it
      __syncthreads();  // every thread has read s_nx
      if (tid == 0) {
        perch_cost r = {0, 0, 0, 0, 0, state == kItemFailed ? kFlagTimeout : kFlagBadIndex, 0};
        b.out[h] = r;
        claim();
      }
      __syncthreads();
      continue;
    }
    // one stage: the previous hypothesis's last barrier has passed, the stage is free
    if (NS == 1 && state == kItemCopy && tid == 0) copy(0, s_nx.off, bb);
    if (MULTI && tid < (int)(sizeof(ObsIndex) / 4))
      reinterpret_cast<int*>(&s_obs)[tid] = reinterpret_cast<const int*>(&b.scenes[a.scene])[tid];
    const ObsIndex& obs = MULTI ? s_obs : obs0;
    for (int i = tid; i < bb.z; i += NT) rxs[i] = g.rx[bb.x + i];
    for (int i = tid; i < bb.w; i += NT) rys[i] = g.ry[bb.y + i];
    if (tid < 7) s_cnt[tid] = tid == 2 ? (pf & kPoseCulled) : 0;
    if (state == kItemCopy) {
      // wait for the stage (bounded); on give-up drain the copy with the
      // full bound, report the hypothesis and go on, or stop if it is still
      // in flight
      if (!__syncthreads_and(mbar_wait(&s_bar[sidx], parity[sidx], b.wait_polls))) {
        const bool drained = __syncthreads_and(mbar_wait(&s_bar[sidx], parity[sidx]));
        if (tid == 0) {
          perch_cost r = {0, 0, 0, 0, 0, kFlagTimeout, 0};
          b.out[h] = r;
          for (int k = 0; k < NS; ++k) stage_pose[k] = -1;
          if (drained) claim();
        }
        if (!drained) break;
        parity[sidx] ^= 1u;
        __syncthreads();
        continue;
      }
      parity[sidx] ^= 1u;
    } else {
      __syncthreads();  // a stage holds this pose's tile already; rays and counters are written
    }
    const uint32_t* stage = stage_of(sidx);
    // a single-scene store holds z with the explained flag (k_render); a
    // multi-scene one plain z, and dJ_r is counted here against the scene
    compare_phase_mask<NT, MULTI ? kSrcZ : kSrcZExplained>(a.pid, a.plen, bb, cam, b, stage, mask, s_cnt);
    if (tid == 0) claim();  // look the next one up (and with two stages start its copy)
    const DevMesh m = g.meshes[a.o.mesh];
    finish_phase<NT, !MULTI>(h, a.pid, a.plen, a.K_total, a.o, bb, m, cam, g, obs, b, DRTile{stage, mask}, rxs, rys,
                             s_cnt, list);
  }
}

cudaError_t preload_eval_kernels() {
  cudaFuncAttributes a;
  cudaError_t e;
  if ((e = cudaFuncGetAttributes(&a, k_fill_u32)) != cudaSuccess) return e;
  if ((e = cudaFuncGetAttributes(&a, k_render_parents)) != cudaSuccess) return e;
  if ((e = cudaFuncGetAttributes(&a, k_uset)) != cudaSuccess) return e;
  return cudaFuncGetAttributes(&a, k_eval<256, false>);
}

// group hypotheses by mesh: hist -> offsets (exclusive scan) -> order;
// hypotheses whose record the shortcut already wrote (skip[h] = 1) are left out
// counts (and below places) a warp's hypotheses of one mesh with one atomic:
// on a counter each they took 37 + 38 us for 120k hypotheses of three meshes, now 3.7 + 3.8
__device__ __forceinline__ int group_key(const perch_obj* hyp, long long h, long long n, int n_mesh, const uint8_t* skip) {
  return h >= n || (skip && skip[h]) ? -1 : min((int)hyp[h].mesh, n_mesh - 1);
}

__global__ void k_group_hist(const perch_obj* hyp, long long n, int n_mesh, int* hist, const uint8_t* skip) {
  const int m = group_key(hyp, blockIdx.x * 256LL + threadIdx.x, n, n_mesh, skip), lane = threadIdx.x & 31;
  const unsigned peers = __match_any_sync(0xffffffffu, m);
  if (m >= 0 && lane == __ffs(peers) - 1) atomicAdd(&hist[m], __popc(peers));
}

__global__ void k_group_scatter(const perch_obj* hyp, long long n, int n_mesh, int* cursor, int* order,
                                const uint8_t* skip) {
  const long long h = blockIdx.x * 256LL + threadIdx.x;
  const int m = group_key(hyp, h, n, n_mesh, skip), lane = threadIdx.x & 31;
  const unsigned peers = __match_any_sync(0xffffffffu, m);
  const int lead = __ffs(peers) - 1;
  int at = 0;
  if (m >= 0 && lane == lead) at = atomicAdd(&cursor[m], __popc(peers));
  at = __shfl_sync(0xffffffffu, at, lead) + __popc(peers & ((1u << lane) - 1));
  if (m >= 0) order[at] = (int)h;
}

cudaError_t launch_group_by_mesh(const perch_obj* hyp, long long n, int n_mesh, int* hist, int* offsets,
                                 int* cursor, int* order, int* scan_tmp, cudaStream_t s, const uint8_t* skip) {
  if (n == 0) return cudaSuccess;
  cudaError_t e;
  const unsigned blocks = (unsigned)((n + 255) / 256);
  k_group_hist<<<blocks, 256, 0, s>>>(hyp, n, n_mesh, hist, skip);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if ((e = launch_scan(ScanInts{hist, offsets, cursor, n_mesh}, n_mesh, scan_tmp, s)) != cudaSuccess) return e;
  k_group_scatter<<<blocks, 256, 0, s>>>(hyp, n, n_mesh, cursor, order, skip);
  return cudaGetLastError();
}

// ---- hypotheses grouped by pose, for shared renders: counts per pose, one
// scan of the counts and of the distinct poses together, hypotheses placed in
// their pose's range. Five launches; with separate scans, flags, list and ranges
// it was eleven (120k poses: 45 us in all, now 19).
__global__ void k_pose_count(Geometry g, Batch b, int* cnt) {
  const long long h = blockIdx.x * 256LL + threadIdx.x;
  if (h >= b.n_hyp || (b.skip && b.skip[h])) return;
  HypArgs a;
  if (!hyp_args(g, b, h, a)) {  // the record k_eval would write; joins no group
    perch_cost r = {0, 0, 0, 0, 0, kFlagBadIndex, 0};
    b.out[h] = r;
    return;
  }
  atomicAdd(&cnt[a.pose], 1);
}

// Per pose the hypotheses before it (low word) and the poses to render before it
// (high word). A pose is rendered when some hypothesis has it and (with the
// render cache) the store does not hold its render under this batch's tag already.
// Mesh m owns poses [m per_mesh, (m + 1) per_mesh): its ranges of order and of
// gpose begin at ranges[4 m] and ranges[4 m + 2] (n_mesh + 1 entries: the last
// has the totals).
struct ScanPoses {
  typedef unsigned long long T;
  const int* cnt;
  const uint32_t* valid;
  uint32_t tag;
  int *start, *gpose, *ranges;
  int per_mesh, n_mesh;
  __device__ T load(int i) const {
    const int c = cnt[i];
    return (T)(uint32_t)c | (T)(c > 0 && !(valid && valid[i] == tag)) << 32;
  }
  __device__ void store(int i, T prefix, T v) const {
    start[i] = (int)(uint32_t)prefix;
    if (v >> 32) gpose[prefix >> 32] = i;
    if (i % per_mesh == 0) range(i / per_mesh, prefix);
  }
  __device__ void range(int m, T prefix) const {
    ranges[4 * m] = (int)(uint32_t)prefix;
    ranges[4 * m + 2] = (int)(prefix >> 32);
  }
  __device__ void total(T sum) const { range(n_mesh, sum); }
};

// also the meshes' counts, from the beginnings of their ranges
__global__ void k_pose_place(Geometry g, Batch b, const int* start, int* cnt, int* order, int* ranges) {
  const long long h = blockIdx.x * 256LL + threadIdx.x;
  if (blockIdx.x == 0)
    for (int m = threadIdx.x; m < g.n_mesh; m += 256) {
      ranges[4 * m + 1] = ranges[4 * m + 4] - ranges[4 * m];
      ranges[4 * m + 3] = ranges[4 * m + 6] - ranges[4 * m + 2];
    }
  if (h >= b.n_hyp || (b.skip && b.skip[h])) return;
  HypArgs a;
  if (!hyp_args(g, b, h, a)) return;
  order[start[a.pose] + atomicSub(&cnt[a.pose], 1) - 1] = (int)h;
}

cudaError_t launch_group_by_pose(const Geometry& g, const Batch& b, const PoseGroups& pg, const uint32_t* valid,
                                 uint32_t tag, cudaStream_t s) {
  const int per_mesh = g.nx * g.ny * g.n_yaw, P = g.n_mesh * per_mesh;
  const unsigned hb = (unsigned)std::max(1LL, (b.n_hyp + 255) / 256);
  cudaError_t e;
  if (b.n_hyp > 0) k_pose_count<<<hb, 256, 0, s>>>(g, b, pg.cnt);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const ScanPoses f{pg.cnt, valid, tag, pg.start, pg.gpose, pg.ranges, per_mesh, g.n_mesh};
  if ((e = launch_scan(f, P, pg.tmp, s)) != cudaSuccess) return e;
  k_pose_place<<<hb, 256, 0, s>>>(g, b, pg.start, pg.cnt, pg.order, pg.ranges);
  return cudaGetLastError();
}

__global__ void k_tile_sizes(Geometry g, int P, int* sizes) {
  const int p = blockIdx.x * 256 + threadIdx.x;
  if (p >= P) return;
  const int4 bb = g.pose_bbox[p];
  sizes[p] = (bb.z * bb.w + 3) >> 2;  // 16-byte units: every tile starts 16-byte aligned
}

cudaError_t launch_tile_offsets(const Geometry& g, int* sizes, int* tile_off, int* tmp, cudaStream_t s) {
  const int P = g.n_mesh * g.nx * g.ny * g.n_yaw;
  k_tile_sizes<<<(unsigned)((P + 255) / 256), 256, 0, s>>>(g, P, sizes);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_exclusive_scan(sizes, tile_off, P, tmp, s);
}

// ------------------------------------------------------------ exact shortcut
// A hypothesis whose parent render is empty over its screen box and which has
// no observed point within (footprint radius + delta + 2 cm) of its (x, y)
// in the world plane has a record fixed by its solo render alone: every
// rendered pixel is new (dR = R(O)) and in no conflict with the parent
// (viol = 0); no observed point is within delta of a rendered point (all of
// dR unexplained: dJ_r = |dR|); none lies in V(O) (dJ_o = 0, n_vol = 0); and on
// a last-level edge every q of U is outside V(O) and unexplained (residual =
// |U|). |dR| and the cull flag come from the same rasteriser run once per
// (mesh, pose) against an empty parent and an empty observation.

// summed-area table S[(r + 1) (cols + 1) + c + 1] = sum of counts[0..r][0..c]
// of `mats` matrices (one block of 512 threads each); S's first row and column
// are zero. Warps scan rows, threads then add down columns, 16 rows read at a
// time: bound by those round trips to L2 (60 x 80 cells, 4 matrices: 12 -> 7.5 us).
__global__ void __launch_bounds__(512) k_sat(const int* counts, int rows, int cols, int* sat) {
  const int* cnt = counts + (size_t)blockIdx.x * rows * cols;
  const int ld = cols + 1, lane = threadIdx.x & 31;
  int* S = sat + (size_t)blockIdx.x * (rows + 1) * ld;
  for (int c = threadIdx.x; c <= cols; c += blockDim.x) S[c] = 0;
  for (int r = threadIdx.x >> 5; r < rows; r += blockDim.x >> 5) {
    int* row = S + (size_t)(r + 1) * ld;
    if (lane == 0) row[0] = 0;
    int carry = 0;
    for (int c0 = 0; c0 < cols; c0 += 128) {
      int v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int c = c0 + 32 * k + lane;
        v[k] = c < cols ? cnt[(size_t)r * cols + c] : 0;
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        for (int d = 1; d < 32; d <<= 1) {
          const int t = __shfl_up_sync(0xffffffffu, v[k], d);
          if (lane >= d) v[k] += t;
        }
        v[k] += carry;
        carry = __shfl_sync(0xffffffffu, v[k], 31);
        const int c = c0 + 32 * k + lane;
        if (c < cols) row[c + 1] = v[k];
      }
    }
  }
  __syncthreads();
  for (int c = 1 + threadIdx.x; c <= cols; c += blockDim.x) {
    int a = 0;
    for (int r0 = 1; r0 <= rows; r0 += 16) {
      int v[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) v[k] = r0 + k <= rows ? S[(size_t)(r0 + k) * ld + c] : 0;
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        a += v[k];
        if (r0 + k <= rows) S[(size_t)(r0 + k) * ld + c] = a;
      }
    }
  }
}

__global__ void k_cell_counts(const int* start2, int n, int* counts) {
  const int c = blockIdx.x * 256 + threadIdx.x;
  if (c < n) counts[c] = start2[c + 1] - start2[c];
}

cudaError_t launch_grid2_sat(const int* start2, int n2x, int n2y, int* counts, int* sat, cudaStream_t s) {
  const int n = n2x * n2y;
  k_cell_counts<<<(n + 255) / 256, 256, 0, s>>>(start2, n, counts);
  k_sat<<<1, 512, 0, s>>>(counts, n2y, n2x, sat);
  return cudaGetLastError();
}

// occupied pixels of each parent render per 8x8 tile
// (a warp: the eight rows of four tiles, eight pixels a lane)
__global__ void __launch_bounds__(256) k_parent_tile_counts(Camera cam, Batch b, int* counts) {
  const int p = blockIdx.y, lane = threadIdx.x & 31, quads = (b.tiles_w + 3) >> 2;
  const int w = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (w >= quads * b.tiles_h) return;
  const int ty = w / quads, tx = 4 * (w % quads) + (lane & 3), v = 8 * ty + (lane >> 2), u0 = 8 * tx;
  const float* z = b.parent_z + (size_t)p * cam.W * cam.H + (size_t)v * cam.W;
  int c = 0;
  if (v < cam.H && (cam.W & 3) == 0 && u0 + 8 <= cam.W) {  // rows start on 16 bytes
    const uint4* q = reinterpret_cast<const uint4*>(z + u0);
    const uint4 a = __ldg(q), d = __ldg(q + 1);
    c = (a.x != kInfBits) + (a.y != kInfBits) + (a.z != kInfBits) + (a.w != kInfBits) + (d.x != kInfBits) +
        (d.y != kInfBits) + (d.z != kInfBits) + (d.w != kInfBits);
  } else if (v < cam.H) {
    for (int u = u0; u < min(u0 + 8, cam.W); ++u) c += __float_as_uint(z[u]) != kInfBits;
  }
  for (int d = 4; d < 32; d <<= 1) c += __shfl_xor_sync(0xffffffffu, c, d);
  if (lane < 4 && tx < b.tiles_w) counts[((size_t)p * b.tiles_h + ty) * b.tiles_w + tx] = c;
}

cudaError_t launch_parent_tiles(const Camera& cam, const Batch& b, int* counts, int* sat, cudaStream_t s) {
  if (b.n_par > 65535) return cudaErrorInvalidValue;
  dim3 grid((((b.tiles_w + 3) >> 2) * b.tiles_h + 7) / 8, b.n_par);
  k_parent_tile_counts<<<grid, 256, 0, s>>>(cam, b, counts);
  k_sat<<<b.n_par, 512, 0, s>>>(counts, b.tiles_h, b.tiles_w, sat);
  return cudaGetLastError();
}

__global__ void k_shortcut(Camera cam, Geometry g, ObsIndex obs0, Batch b) {
  const long long h = blockIdx.x * 256LL + threadIdx.x;
  int fast = 0;
  if (h < b.n_hyp) {
    const perch_obj o = b.hyp[h];
    const int pid = b.hyp_parent[h];
    bool ok = pid >= 0 && pid < b.n_par && obj_ok(g, o);
    const int plen = ok ? b.parent_len[pid] : 0;
    ok = ok && plen >= 0 && plen <= b.parent_stride;
    const int scene = (ok && b.parent_scene) ? b.parent_scene[pid] : 0;
    ok = ok && (!b.parent_scene || (scene >= 0 && scene < b.n_scenes));
    const long long pose = (((long long)o.mesh * g.nx + o.ix) * g.ny + o.iy) * g.n_yaw + o.iyaw;
    const int4 bb = ok ? g.pose_bbox[pose] : make_int4(0, 0, 0, 0);
    ok = ok && bb.z <= b.tile_w && bb.w <= b.tile_h;
    if (ok && plen > 0 && bb.z > 0 && bb.w > 0) {  // parent render empty over the screen box?
      const int tx0 = max(bb.x, 0) >> 3, tx1 = min(bb.x + bb.z - 1, cam.W - 1) >> 3;
      const int ty0 = max(bb.y, 0) >> 3, ty1 = min(bb.y + bb.w - 1, cam.H - 1) >> 3;
      if (tx0 <= tx1 && ty0 <= ty1) {
        const int* S = b.parent_sat + (size_t)pid * (b.tiles_h + 1) * (b.tiles_w + 1);
        ok = sat_sum(S, b.tiles_w, ty0, ty1, tx0, tx1) == 0;
      }
    }
    if (ok) ok = !obs_near(cam, g, b.parent_scene ? b.scenes[scene] : obs0, o);  // no observed point near (x, y)
    if (ok) {
      const int K_total = b.parent_K ? b.parent_K[pid] : b.K_total;
      const int2 so = b.solo[pose];
      perch_cost r;
      r.djr = so.x;
      r.djo = 0;
      r.resid = plen + 1 == K_total ? b.uset_count[pid] : 0;
      r.viol = 0;
      r.n_new = so.x;
      r.flags = (uint32_t)so.y;
      r.n_vol = 0;
      b.out[h] = r;
      fast = 1;
    }
    b.skip[h] = (uint8_t)fast;
  }
  const int n_fast = __syncthreads_count(fast);
  if (threadIdx.x == 0 && n_fast && b.n_short) atomicAdd(b.n_short, (unsigned long long)n_fast);
}

cudaError_t launch_shortcut(const Camera& cam, const Geometry& g, const ObsIndex& obs, const Batch& b,
                            cudaStream_t s) {
  if (b.n_hyp == 0) return cudaSuccess;
  k_shortcut<<<(unsigned)((b.n_hyp + 255) / 256), 256, 0, s>>>(cam, g, obs, b);
  return cudaGetLastError();
}

// solo table entry from a record evaluated against an empty parent and an
// empty observation: (|dR| = pixels covered, cull flag)
__global__ void k_solo_pack(const perch_cost* rec, long long n, int2* solo) {
  const long long h = blockIdx.x * 256LL + threadIdx.x;
  if (h < n) solo[h] = make_int2(rec[h].n_new, (int)(rec[h].flags & 1u));
}

// *flags = the flags of all records together
__global__ void k_any_flags(const perch_cost* rec, long long n, uint32_t* flags) {
  uint32_t a = 0;
  for (long long h = blockIdx.x * 256LL + threadIdx.x; h < n; h += gridDim.x * 256LL) a |= (uint32_t)rec[h].flags;
  a = __reduce_or_sync(0xffffffffu, a);
  if ((threadIdx.x & 31) == 0 && a) atomicOr(flags, a);
}

cudaError_t launch_any_flags(const perch_cost* rec, long long n, uint32_t* flags, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(flags, 0, 4, s);
  if (e != cudaSuccess) return e;
  k_any_flags<<<(unsigned)std::min<long long>((n + 255) / 256, 152 * 8), 256, 0, s>>>(rec, n, flags);
  return cudaGetLastError();
}

cudaError_t launch_solo_pack(const perch_cost* rec, long long n, int2* solo, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  k_solo_pack<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(rec, n, solo);
  return cudaGetLastError();
}

template <int NT, bool MULTI>
static cudaError_t launch_group_t(const Camera& cam, const Geometry& g, const ObsIndex& obs, const Batch& b,
                                  const EvalGroup& grp, long long max_items, int sm_count, cudaStream_t s) {
  const size_t smem = eval_smem_bytes(b.tile_w, b.tile_h);
  auto kern = k_eval<NT, MULTI>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NT, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  long long grid = (long long)per_sm * sm_count;
  if (grid > max_items) grid = max_items;
  if (grid < 1) grid = 1;
  kern<<<(unsigned)grid, NT, smem, s>>>(cam, g, obs, b, grp);
  return cudaGetLastError();
}

template <int NT, bool EXPL, int INL>
static cudaError_t launch_render_t(const Camera& cam, const Geometry& g, const ObsIndex& obs, const Batch& b,
                                   const RenderWork& w, long long max_items, int sm_count, cudaStream_t s) {
  const size_t smem = render_smem_bytes(b.tile_w, b.tile_h);
  auto kern = k_render<NT, EXPL, INL>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NT, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  long long grid = (long long)per_sm * sm_count;
  if (grid > max_items) grid = max_items;
  if (grid < 1) grid = 1;
  kern<<<(unsigned)grid, NT, smem, s>>>(cam, g, obs, b, w);
  return cudaGetLastError();
}

template <int NT, bool EXPL>
static cudaError_t launch_render_i(const Camera& cam, const Geometry& g, const ObsIndex& obs, const Batch& b,
                                   const RenderWork& w, long long max_items, int inline_px, int sm_count,
                                   cudaStream_t s) {
  switch (inline_px) {
    case 8: return launch_render_t<NT, EXPL, 8>(cam, g, obs, b, w, max_items, sm_count, s);
    case 32: return launch_render_t<NT, EXPL, 32>(cam, g, obs, b, w, max_items, sm_count, s);
    default: return launch_render_t<NT, EXPL, 16>(cam, g, obs, b, w, max_items, sm_count, s);
  }
}

// One persistent launch rendering one mesh's distinct poses of a batch into
// the tile store, with CTAs of `threads` (128, 256 or 512), the inline limit
// `inline_px` (8, 16 or 32 candidate pixel centres) and the mesh's tile
// (b.tile_w x b.tile_h). A single-scene batch also stores each rendered
// point's Eq. (1) test against `obs`.
cudaError_t launch_render_group(const Camera& cam, const Geometry& g, const ObsIndex& obs, const Batch& b,
                                const RenderWork& w, long long max_items, int threads, int inline_px,
                                int sm_count, cudaStream_t s) {
  if (max_items <= 0) return cudaSuccess;
  const bool expl = b.parent_scene == nullptr;
  switch (threads) {
    case 128: return expl ? launch_render_i<128, true>(cam, g, obs, b, w, max_items, inline_px, sm_count, s)
                          : launch_render_i<128, false>(cam, g, obs, b, w, max_items, inline_px, sm_count, s);
    case 512: return expl ? launch_render_i<512, true>(cam, g, obs, b, w, max_items, inline_px, sm_count, s)
                          : launch_render_i<512, false>(cam, g, obs, b, w, max_items, inline_px, sm_count, s);
    default: return expl ? launch_render_i<256, true>(cam, g, obs, b, w, max_items, inline_px, sm_count, s)
                         : launch_render_i<256, false>(cam, g, obs, b, w, max_items, inline_px, sm_count, s);
  }
}

template <int NT, bool MULTI, int NS>
static cudaError_t launch_cost_t(const Camera& cam, const Geometry& g, const ObsIndex& obs, const Batch& b,
                                 const CostWork& w, long long max_items, int sm_count, cudaStream_t s) {
  const size_t smem = cost_smem_bytes(b.tile_w, b.tile_h, NS);
  auto kern = k_cost<NT, MULTI, NS>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NT, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  long long grid = (long long)per_sm * sm_count;
  if (grid > max_items) grid = max_items;
  if (grid < 1) grid = 1;
  kern<<<(unsigned)grid, NT, smem, s>>>(cam, g, obs, b, w);
  return cudaGetLastError();
}

template <int NS>
static cudaError_t launch_cost_s(const Camera& cam, const Geometry& g, const ObsIndex& obs, const Batch& b,
                                 const CostWork& w, long long max_items, int threads, int sm_count, cudaStream_t s) {
  const bool multi = b.parent_scene != nullptr;
  if (threads == 256)
    return multi ? launch_cost_t<256, true, NS>(cam, g, obs, b, w, max_items, sm_count, s)
                 : launch_cost_t<256, false, NS>(cam, g, obs, b, w, max_items, sm_count, s);
  return multi ? launch_cost_t<128, true, NS>(cam, g, obs, b, w, max_items, sm_count, s)
               : launch_cost_t<128, false, NS>(cam, g, obs, b, w, max_items, sm_count, s);
}

// One persistent launch costing one mesh's hypotheses of a batch from the
// tile store, with CTAs of `threads` (128 or 256) and `stages` (1 or 2) stage
// buffers; two stages fall back to one where they do not fit.
bool cost_stages_fit(int device, int tile_w, int tile_h, int stages) {
  int optin = 0;
  if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device) != cudaSuccess) return false;
  return cost_smem_bytes(tile_w, tile_h, stages) + 1024 <= (size_t)optin;  // 1024: static shared memory
}

cudaError_t launch_cost_group(const Camera& cam, const Geometry& g, const ObsIndex& obs, const Batch& b,
                              const CostWork& w, long long max_items, int threads, int stages, int sm_count,
                              cudaStream_t s) {
  if (max_items <= 0) return cudaSuccess;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (stages == 2 && cost_stages_fit(dev, b.tile_w, b.tile_h, 2))
    return launch_cost_s<2>(cam, g, obs, b, w, max_items, threads, sm_count, s);
  return launch_cost_s<1>(cam, g, obs, b, w, max_items, threads, sm_count, s);
}

// One persistent launch for one group of hypotheses with CTAs of `threads`
// (128, 256 or 512) and the group's tile (b.tile_w x b.tile_h).
cudaError_t launch_eval_group(const Camera& cam, const Geometry& g, const ObsIndex& obs, const Batch& b,
                              const int* order, const int* offset, const int* count, int* next, long long max_items,
                              int threads, int sm_count, cudaStream_t s) {
  if (max_items <= 0) return cudaSuccess;
  EvalGroup grp{order, offset, count, next};
  const bool multi = b.parent_scene != nullptr;
  switch (threads) {
    case 128: return multi ? launch_group_t<128, true>(cam, g, obs, b, grp, max_items, sm_count, s)
                           : launch_group_t<128, false>(cam, g, obs, b, grp, max_items, sm_count, s);
    case 512: return multi ? launch_group_t<512, true>(cam, g, obs, b, grp, max_items, sm_count, s)
                           : launch_group_t<512, false>(cam, g, obs, b, grp, max_items, sm_count, s);
    default: return multi ? launch_group_t<256, true>(cam, g, obs, b, grp, max_items, sm_count, s)
                          : launch_group_t<256, false>(cam, g, obs, b, grp, max_items, sm_count, s);
  }
}

// -------------------------------------------------------------------- ICP
// Local alignment of each successor's new object with the observed cloud
// (Sec. IV-E-1: the object's non-occluded portion, aligned by ICP; Sec. V-B:
// correspondences only within 2 cm), step by step as the public header
// states it. The render, the model set and every distance are the binary32
// arithmetic of the evaluation path; the pairs' sums are exact 64-bit
// integers (coordinates in units of 2^-16 m), so the order in which the
// warps add them does not matter; the fit from those sums is double
// arithmetic in a fixed order, made by one thread.

// the observed world points with their index in I, and their bounds
__global__ void k_icp_points(const float4* world2, const float4* cam2, int n, float4* pts, int* bounds) {
  const int k = blockIdx.x * 256 + threadIdx.x;
  const bool ok = k < n;
  const float4 w = ok ? world2[k] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  if (ok) pts[k] = make_float4(w.x, w.y, w.z, cam2[k].w);
  const int lo[3] = {ok ? ford(w.x) : INT_MAX, ok ? ford(w.y) : INT_MAX, ok ? ford(w.z) : INT_MAX};
  const int hi[3] = {ok ? ford(w.x) : INT_MIN, ok ? ford(w.y) : INT_MIN, ok ? ford(w.z) : INT_MIN};
  for (int d = 0; d < 3; ++d) {
    const int a = __reduce_min_sync(0xffffffffu, lo[d]), b = __reduce_max_sync(0xffffffffu, hi[d]);
    if ((threadIdx.x & 31) == 0 && a <= b) {
      atomicMin(&bounds[d], a);
      atomicMax(&bounds[3 + d], b);
    }
  }
}

cudaError_t launch_icp_points(const float4* world2, const float4* cam2, int n, float4* pts, int* bounds,
                              cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_icp_points<<<(n + 255) / 256, 256, 0, s>>>(world2, cam2, n, pts, bounds);
  return cudaGetLastError();
}

__device__ __forceinline__ int icp_fixed(float v) { return __float2int_rn(fmul(v, 65536.0f)); }  // |v| < 32: 21 bits

// hi 2^64 + lo: each part rounded to double, then one rounded addition
__device__ __forceinline__ double icp_i128_to_double(__int128 v) {
  const long long hi = (long long)(v >> 64);
  const unsigned long long lo = (unsigned long long)v;
  return __dadd_rn(__dmul_rn(__ll2double_rn(hi), 18446744073709551616.0), __ull2double_rn(lo));
}

// one pair's terms: n, sum X_m, sum Y_m, sum X_q, sum Y_q, sum X_m X_q,
// sum Y_m Y_q, sum X_m Y_q, sum Y_m X_q (|x|, |y| < 32 m: |X|, |Y| < 2^21)
__device__ __forceinline__ void icp_add_pair(long long* L, float mx, float my, float qx, float qy) {
  if (!(fabsf(mx) < 32.0f && fabsf(my) < 32.0f && fabsf(qx) < 32.0f && fabsf(qy) < 32.0f)) return;
  const int X = icp_fixed(mx), Y = icp_fixed(my), QX = icp_fixed(qx), QY = icp_fixed(qy);
  L[0] += 1;
  L[1] += X;
  L[2] += Y;
  L[3] += QX;
  L[4] += QY;
  L[5] += (long long)X * QX;
  L[6] += (long long)Y * QY;
  L[7] += (long long)X * QY;
  L[8] += (long long)Y * QX;
}

// Planar Procrustes from the sums: C = n sum(m . q) - sum m . sum q and
// S = n sum(m x q) - sum m x sum q (exact), (c, s) = (C, S) / |(C, S)|,
// t = (sum q - R sum m) / n. False when C = S = 0.
__device__ bool icp_solve(const long long* S, double* T) {
  const __int128 n = S[0];
  const __int128 C = n * ((__int128)S[5] + S[6]) - ((__int128)S[1] * S[3] + (__int128)S[2] * S[4]);
  const __int128 X = n * ((__int128)S[7] - S[8]) - ((__int128)S[1] * S[4] - (__int128)S[2] * S[3]);
  if (C == 0 && X == 0) return false;
  const double Cd = icp_i128_to_double(C), Xd = icp_i128_to_double(X);
  const double h = __dsqrt_rn(__dadd_rn(__dmul_rn(Cd, Cd), __dmul_rn(Xd, Xd)));
  const double c = __ddiv_rn(Cd, h), s = __ddiv_rn(Xd, h);
  const double nd = __ll2double_rn(S[0]), sx = __ll2double_rn(S[1]), sy = __ll2double_rn(S[2]);
  T[0] = c;
  T[1] = s;
  T[2] = __dmul_rn(__ddiv_rn(__dsub_rn(__ll2double_rn(S[3]), __dsub_rn(__dmul_rn(c, sx), __dmul_rn(s, sy))), nd),
                   1.0 / 65536.0);
  T[3] = __dmul_rn(__ddiv_rn(__dsub_rn(__ll2double_rn(S[4]), __dadd_rn(__dmul_rn(s, sx), __dmul_rn(c, sy))), nd),
                   1.0 / 65536.0);
  return true;
}

// World points of scene 0 by pixel, rows of q.stride pixels and q.blocks_y
// 4 rows (NaN where nothing was observed: no distance to it passes a test),
// and the box of each 4 x 4 block's points (lo = +inf: none). A thread takes a
// block.
__global__ void k_icp_image(const float* depth, Camera cam, const float* rx, const float* ry, IcpImage q, float4* pts,
                            float4* lo, float4* hi) {
  const int k = blockIdx.x * 256 + threadIdx.x, nbx = q.stride / 4;
  if (k >= nbx * q.blocks_y) return;
  const int bu = 4 * (k % nbx), bv = 4 * (k / nbx);
  const float inf = __uint_as_float(kInfBits), nan = __uint_as_float(0x7fc00000u);
  float4 a = make_float4(inf, inf, inf, 0.0f), b = make_float4(-inf, -inf, -inf, 0.0f);
  for (int i = 0; i < 16; ++i) {
    const int u = bu + (i & 3), v = bv + (i >> 2);
    float4 o = make_float4(nan, nan, nan, nan);
    const float z = u < cam.W && v < cam.H ? depth[v * cam.W + u] : 0.0f;
    if (depth_valid(z)) {
      const float x = fmul(rx[u], z), y = fmul(ry[v], z);
      o.x = fadd(ffma(cam.Rwc[2], z, ffma(cam.Rwc[1], y, fmul(cam.Rwc[0], x))), cam.twc[0]);
      o.y = fadd(ffma(cam.Rwc[5], z, ffma(cam.Rwc[4], y, fmul(cam.Rwc[3], x))), cam.twc[1]);
      o.z = fadd(ffma(cam.Rwc[8], z, ffma(cam.Rwc[7], y, fmul(cam.Rwc[6], x))), cam.twc[2]);
      a = make_float4(fminf(a.x, o.x), fminf(a.y, o.y), fminf(a.z, o.z), 0.0f);
      b = make_float4(fmaxf(b.x, o.x), fmaxf(b.y, o.y), fmaxf(b.z, o.z), 0.0f);
    }
    pts[v * q.stride + u] = o;
  }
  lo[k] = a;
  hi[k] = b;
}

cudaError_t launch_icp_image(const float* depth, const Camera& cam, const float* rx, const float* ry,
                             const IcpImage& q, float4* pts, float4* lo, float4* hi, cudaStream_t s) {
  const int n = q.stride / 4 * q.blocks_y;
  k_icp_image<<<(n + 255) / 256, 256, 0, s>>>(depth, cam, rx, ry, q, pts, lo, hi);
  return cudaGetLastError();
}

// The nearest observed point of a model point within the radius (ties: the
// smaller pixel, which is the smaller index in I). Starts from no point and the
// radius squared, or from a point within the radius (the last matching's).
struct IcpBest {
  float d;  // squared distance
  int j;    // place in the image (or the grid's points); -1: none
  int tie;  // pixel order
  float x, y;
};

// In the image: a point within rho of p lies within f rho sqrt(1 + t^2) /
// (z - rho) pixels of p's projection (slope t, depth z), as in delta_radius;
// q.ortho pads rho by what the camera's matrix differs from a rotation. A
// small window is scanned; in a larger one (most model points of a wrong pose
// are many millimetres from the cloud, or have no pair) the boxes of its
// 4 x 4 blocks are tested first, all lanes at a time, and then the blocks whose box
// is nearer than the best point, the nearest one first. Bound by the issue of
// those tests: two 640x480 scenes, 120k successors each, 35 and 48 ms
// (renders 11.5 ms of it). The points' grid (cells of half a radius, as many
// points in reach but in as many places as lanes) took 52 and 82; smaller
// cells, masks of the rows that hold points, or keeping a pair while the second
// nearest point stays farther (ICP's steps are longer than that) 51 to 126.
__device__ __forceinline__ void icp_nearest(const Camera& cam, const IcpImage& q, float px, float py, float pz,
                                            IcpBest& b) {
  const float xc = cam.Rcw[0] * px + cam.Rcw[1] * py + cam.Rcw[2] * pz + cam.tcw[0];
  const float yc = cam.Rcw[3] * px + cam.Rcw[4] * py + cam.Rcw[5] * pz + cam.tcw[1];
  const float zc = cam.Rcw[6] * px + cam.Rcw[7] * py + cam.Rcw[8] * pz + cam.tcw[2];
  const float rho = __fsqrt_rn(b.d) * 1.001f + 1e-6f + q.ortho * (fabsf(xc) + fabsf(yc) + fabsf(zc));
  int u0 = 0, u1 = cam.W - 1, v0 = 0, v1 = cam.H - 1;
  if (zc - rho > 1e-3f) {
    const float slack = 0.05f + 1e-6f * (float)(cam.W + cam.H);
    const float inv = __fdividef(1.0f, zc), tx = xc * inv, ty = yc * inv, f = __fdividef(rho, zc - rho);
    const float uc = cam.fx * tx + cam.cx, ru = cam.fx * (1.0f + 0.5f * tx * tx) * f + slack;
    const float vc = cam.fy * ty + cam.cy, rv = cam.fy * (1.0f + 0.5f * ty * ty) * f + slack;
    u0 = max((int)ceilf(fmaxf(uc - ru, -1e6f)), u0);
    u1 = min((int)floorf(fminf(uc + ru, 1e6f)), u1);
    v0 = max((int)ceilf(fmaxf(vc - rv, -1e6f)), v0);
    v1 = min((int)floorf(fminf(vc + rv, 1e6f)), v1);
  }
  if (u0 > u1 || v0 > v1) return;
  // the loops below are unrolled for loads in flight: bound by their latency (120k
  // successors: 34.9 -> 32.9 ms; two boxes at a time, four took 33.9)
  auto test = [&](int i) {
    const float4 o = __ldg(&q.pts[i]);
    const float d = dist2(px, py, pz, o);
    if (d <= b.d && (d < b.d || i < b.tie)) b = IcpBest{d, i, i, o.x, o.y};
  };
  if ((u1 - u0 + 1) * (v1 - v0 + 1) <= kIcpDirect) {
    for (int v = v0; v <= v1; ++v)
#pragma unroll 2
      for (int u = u0; u <= u1; ++u) test(v * q.stride + u);
    return;
  }
  auto gap2 = [&](int at) {  // squared distance to a block's box
    const float4 lo = __ldg(&q.lo[at]), hi = __ldg(&q.hi[at]);
    const float gx = max3(lo.x - px, px - hi.x, 0.0f), gy = max3(lo.y - py, py - hi.y, 0.0f),
                gz = max3(lo.z - pz, pz - hi.z, 0.0f);
    return gx * gx + gy * gy + gz * gz;
  };
  const int pitch = q.stride >> 2, bx1 = u1 >> 2, by1 = v1 >> 2;
  for (int x0 = u0 >> 2; x0 <= bx1; x0 += 8)  // at most 8 x 4 blocks at a time
    for (int y0 = v0 >> 2; y0 <= by1; y0 += 4) {
      const int nx = min(bx1 - x0, 7), ny = min(by1 - y0, 3);
      uint32_t mask = 0;
      int first = -1;
      float nearest = b.d * 1.00001f;
      for (int y = 0; y <= ny; ++y)
#pragma unroll 2
        for (int x = 0; x <= nx; ++x) {
          const float g = gap2((y0 + y) * pitch + x0 + x);
          if (g > b.d * 1.00001f) continue;
          mask |= 1u << (8 * y + x);
          if (g < nearest) {
            nearest = g;
            first = 8 * y + x;
          }
        }
      while (mask) {
        const int k = first >= 0 ? first : __ffs((int)mask) - 1, y = y0 + (k >> 3), x = x0 + (k & 7);
        mask &= ~(1u << k);
        if (first < 0 && gap2(y * pitch + x) > b.d * 1.00001f) continue;
        first = -1;
        const int at = 4 * (y * q.stride + x);
#pragma unroll
        for (int i = 0; i < 16; ++i) test(at + (i >> 2) * q.stride + (i & 3));
      }
    }
}

// In the grid of the points, where the camera's matrix is no rotation: the
// cells that meet a cube about p.
__device__ __noinline__ IcpBest icp_nearest_grid(IcpGrid q, float px, float py, float pz, IcpBest b) {
  const float rho = __fsqrt_rn(b.d) * 1.01f + 1e-6f;
  const int x0 = max(cell_of(px - rho, q.gx, q.inv, q.nx), 0), x1 = min(cell_of(px + rho, q.gx, q.inv, q.nx), q.nx - 1);
  const int y0 = max(cell_of(py - rho, q.gy, q.inv, q.ny), 0), y1 = min(cell_of(py + rho, q.gy, q.inv, q.ny), q.ny - 1);
  const int z0 = max(cell_of(pz - rho, q.gz, q.inv, q.nz), 0), z1 = min(cell_of(pz + rho, q.gz, q.inv, q.nz), q.nz - 1);
  if (x0 > x1) return b;
  for (int iz = z0; iz <= z1; ++iz)
    for (int iy = y0; iy <= y1; ++iy) {
      const int row = (iz * q.ny + iy) * q.nx;
      const int end = q.start[row + x1 + 1];
      for (int t = q.start[row + x0]; t < end; ++t) {
        const float4 o = q.pts[t];
        const float d = dist2(px, py, pz, o);
        const int j = __float_as_int(o.w);
        if (d <= b.d && (d < b.d || j < b.tie)) b = IcpBest{d, t, j, o.x, o.y};
      }
    }
  return b;
}

struct IcpClaim {
  int* next;  // device counter, zero before the launch
};

// One CTA per hypothesis at a time (claimed from a counter): render the new
// object into the shared-memory tile over its screen box (render_chunks),
// keep the pixels in front of the parent's render as the model set, as a
// list of world points, then iterate. In each matching a thread takes one
// model point, moves it and finds its nearest observed point, starting
// from the one it was paired with last time when that is still within the
// radius. It adds the pair to its own sums, and the warps reduce
// those to one set each. Thread 0 then decides and fits. A
// successor with no observed point within the radius of its footprint has no
// pair: it is done with the model set.
template <int NT>
__global__ void __launch_bounds__(NT, NT == 256 ? 3 : 1) k_icp(Camera cam, Geometry g, Batch b, IcpGrid q, IcpWork w, IcpClaim cl) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t s_bar;
  __shared__ long long s_sum[9][NT / 32];
  __shared__ double s_T[4];
  __shared__ int s_qn[2], s_item, s_stop, s_nm;
  constexpr int NW = NT / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    mbar_init(&s_bar, 1);
    fence_barrier_init();
  }
  __syncthreads();
  EvalShared sh{&s_bar, nullptr, s_qn, smem, 0u, nullptr};
  const RenderSmem s = render_smem(smem);
  uint32_t* tile = s.tile;
  for (;;) {
    if (tid == 0) s_item = atomicAdd(cl.next, 1);
    __syncthreads();
    const long long h = s_item;
    __syncthreads();
    if (h >= b.n_hyp) break;
    HypArgs a;
    const bool ok = hyp_args(g, b, h, a);
    const int4 bb = ok ? g.pose_bbox[a.pose] : make_int4(0, 0, 0, 0);
    if (!ok || bb.z > b.tile_w || bb.w > b.tile_h) {
      if (tid == 0) w.out[h] = perch_icp{0.0, 0.0, 0.0, 0.0, 0, 0, 0, (int32_t)kFlagBadIndex};
      continue;
    }
    const int tw = bb.z, area = bb.z * bb.w;
    const DevMesh m = g.meshes[a.o.mesh];
    if (tid == 0) render_start(g, m, a.o.iyaw, s, sh.bar);
    for (int i = tid; i < area; i += NT) tile[i] = 0u;  // 1/z = 0: empty
    if (tid == 0) {
      s_nm = 0;
      s_T[0] = 1.0;
      s_T[1] = s_T[2] = s_T[3] = 0.0;
    }
    unsigned culled = 0;
    float4 cov = kNoCover;  // not needed here
    const int st = render_chunks<NT, kInlinePixels, false>(cam, g, b, m, a.o, a.pose, bb, s, sh, culled, cov);
    if (st != kEvalDone) {
      if (tid == 0) w.out[h] = perch_icp{0.0, 0.0, 0.0, 0.0, 0, 0, 0, (int32_t)kFlagTimeout};
      __syncthreads();  // the tile is cleared by the next hypothesis
      if (st == kEvalStop) break;
      continue;
    }
    // model set: z where the object lies strictly in front of the parent,
    // and the list of those pixels (in any order: every sum is order-free)
    const float* zp = b.parent_z + (size_t)a.pid * cam.W * cam.H;
    const size_t cap = (size_t)b.tile_w * b.tile_h;
    float4* list = w.model + cap * blockIdx.x;  // this CTA's slice: model points, and each one's last pair
    // a warp takes 8 x 4 pixels: its points then search alike
    const int wx = (tw + 7) >> 3, n_win = wx * ((bb.w + 3) >> 2);
    for (int k = warp; k < n_win; k += NW) {
      const int lx = 8 * (k % wx) + (lane & 7), ly = 4 * (k / wx) + (lane >> 3);
      uint32_t v = 0u;
      if (lx < tw && ly < bb.w) {
        const uint32_t izb = tile[ly * tw + lx];
        if (izb != 0u) {
          const float z = __frcp_rn(__uint_as_float(izb));
          if (z < zp[(size_t)(bb.y + ly) * cam.W + bb.x + lx]) v = __float_as_uint(z);
        }
      }
      const unsigned mask = __ballot_sync(0xffffffffu, v != 0u);
      int base = 0;
      if (lane == 0 && mask) base = atomicAdd(&s_nm, __popc(mask));
      base = __shfl_sync(0xffffffffu, base, 0);
      if (v != 0u) {  // its world point (R7)
        const float z = __uint_as_float(v), xc = fmul(g.rx[bb.x + lx], z), yc = fmul(g.ry[bb.y + ly], z);
        const float mx = fadd(ffma(cam.Rwc[2], z, ffma(cam.Rwc[1], yc, fmul(cam.Rwc[0], xc))), cam.twc[0]);
        const float my = fadd(ffma(cam.Rwc[5], z, ffma(cam.Rwc[4], yc, fmul(cam.Rwc[3], xc))), cam.twc[1]);
        const float mz = fadd(ffma(cam.Rwc[8], z, ffma(cam.Rwc[7], yc, fmul(cam.Rwc[6], xc))), cam.twc[2]);
        list[base + __popc(mask & ((1u << lane) - 1u))] = make_float4(mx, my, mz, __int_as_float(-1));
      }
    }
    __syncthreads();  // |M| and the list are complete
    const int nm = s_nm;
    long long prev[9];  // thread 0: the previous matching's sums
    bool have_prev = false;
    int iters = 0, n_corr = 0, status = PERCH_ICP_CAP;
    // every model point lies within the footprint's radius of (x, y) (+ 2 cm
    // and a sixteenth of a pixel at the object's depth for the snap)
    const float depth = g.pose_off[a.o.ix * g.ny + a.o.iy].z + m.fp_r + fmaxf(fabsf(m.lo[2]), fabsf(m.hi[2]));
    const float reach_m = m.fp_r + 0.02f + depth / (16.0f * fminf(cam.fx, cam.fy));
    const float ox = g.xs[a.o.ix], oy = g.ys[a.o.iy];
    bool met = nm > 0 && w.obs.n > 0;
    {
      const float R = reach_m + w.rwin;
      if (met) {
        const int cx0 = max(cell_of(ox - R, w.obs.g2x, w.obs.inv2, w.obs.n2x) - 1, 0);
        const int cx1 = min(cell_of(ox + R, w.obs.g2x, w.obs.inv2, w.obs.n2x) + 1, w.obs.n2x - 1);
        const int cy0 = max(cell_of(oy - R, w.obs.g2y, w.obs.inv2, w.obs.n2y) - 1, 0);
        const int cy1 = min(cell_of(oy + R, w.obs.g2y, w.obs.inv2, w.obs.n2y) + 1, w.obs.n2y - 1);
        met = cx0 <= cx1 && cy0 <= cy1 && sat_sum(w.obs.sat2, w.obs.n2x, cy0, cy1, cx0, cx1) != 0;
      }
    }
    if (!met && w.max_iter > 0) status = PERCH_ICP_FEW;
    for (int k = 1; met && k <= w.max_iter; ++k) {
      __syncthreads();  // publishes s_T; the last sums have been read
      const float cf = __double2float_rn(s_T[0]), sf = __double2float_rn(s_T[1]);
      const float txf = __double2float_rn(s_T[2]), tyf = __double2float_rn(s_T[3]);
      long long L[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
      for (int e = tid; e < nm; e += NT) {
        const float4 m4 = list[e];
        const float px = fadd(fsub(fmul(cf, m4.x), fmul(sf, m4.y)), txf);
        const float py = fadd(fadd(fmul(sf, m4.x), fmul(cf, m4.y)), tyf);
        IcpBest best{w.r2, -1, INT_MAX, 0.0f, 0.0f};
        const int j0 = __float_as_int(m4.w);  // the last matching's point: a bound, if still within the radius
        if (j0 >= 0) {
          const float4 o = __ldg(&(w.img.pts ? w.img.pts : q.pts)[j0]);
          const float d = dist2(px, py, m4.z, o);
          if (d <= w.r2) best = IcpBest{d, j0, w.img.pts ? j0 : __float_as_int(o.w), o.x, o.y};
        }
        if (w.img.pts)
          icp_nearest(cam, w.img, px, py, m4.z, best);
        else
          best = icp_nearest_grid(q, px, py, m4.z, best);
        if (best.j != j0) list[e].w = __int_as_float(best.j);
        if (best.j >= 0) icp_add_pair(L, m4.x, m4.y, best.x, best.y);
      }
      for (int t = 0; t < 9; ++t) {
        long long v = L[t];
        for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
        if (lane == 0) s_sum[t][warp] = v;
      }
      __syncthreads();
      if (tid == 0) {
        long long S[9];
        for (int t = 0; t < 9; ++t) {
          S[t] = 0;
          for (int k = 0; k < NW; ++k) S[t] += s_sum[t][k];
        }
        n_corr = (int)S[0];
        int stop = 0;
        bool same = have_prev;
        for (int t = 0; t < 9 && same; ++t) same = S[t] == prev[t];
        if (S[0] < 3) {
          status = PERCH_ICP_FEW;
          stop = 1;
        } else if (same) {
          status = PERCH_ICP_CONVERGED;
          stop = 1;
        } else {
          double T[4];
          if (!icp_solve(S, T)) {
            status = PERCH_ICP_DEGENERATE;
            stop = 1;
          } else {
            for (int t = 0; t < 4; ++t) s_T[t] = T[t];
            for (int t = 0; t < 9; ++t) prev[t] = S[t];
            have_prev = true;
            iters = k;
          }
        }
        s_stop = stop;
      }
      __syncthreads();
      if (s_stop) break;
    }
    if (tid == 0) w.out[h] = perch_icp{s_T[0], s_T[1], s_T[2], s_T[3], s_nm, n_corr, iters, status};
    __syncthreads();  // the tile, s_T and s_nm are reused by the next hypothesis
  }
}

cudaError_t launch_icp(const Camera& cam, const Geometry& g, const Batch& b, const IcpGrid& q, const IcpWork& w,
                       long long model_elems, int* next, int sm_count, cudaStream_t s) {
  if (b.n_hyp <= 0) return cudaSuccess;
  const size_t smem = render_smem_bytes(b.tile_w, b.tile_h);
  // no more hypotheses than SMs: a CTA has its SM to itself, and twice the
  // threads halve the rounds of each matching (the five objects of a scene,
  // 640x480: 1.18 -> 0.62 ms)
  const int nt = b.n_hyp <= sm_count ? 512 : 256;
  auto kern = nt == 512 ? k_icp<512> : k_icp<256>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, nt, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  long long grid = (long long)per_sm * sm_count;
  if (grid > b.n_hyp) grid = b.n_hyp;
  const long long cap = (long long)b.tile_w * b.tile_h;  // each CTA's slice of w.model
  if (cap > 0 && grid > model_elems / cap) grid = model_elems / cap;
  if (grid < 1) return cudaErrorInvalidValue;
  kern<<<(unsigned)grid, nt, smem, s>>>(cam, g, b, q, w, IcpClaim{next});
  return cudaGetLastError();
}

}  // namespace perch
