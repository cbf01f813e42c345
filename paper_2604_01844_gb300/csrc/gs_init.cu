// Initialisation of the Gaussians (Sec. 3.1): an FDK reconstruction (Feldkamp, Davis and Kress
// 1984) of the projections, then means sampled with probability proportional to the gradient
// magnitude of that volume above a background threshold, densities k * V(p) with k = 0.15,
// identity rotations and isotropic scales equal to the nearest-neighbour distance.  The same
// sampler initialises the volume fit from a ground-truth volume (Sec. 3.6).
//
// FDK (circular cone beam, each view's own frame; u, v scaled to the plane through the
// rotation axis perpendicular to the central ray, D_so = source-to-axis distance):
//   1. weight   p(u, v) * D_so / sqrt(D_so^2 + u^2 + v^2)
//   2. filter   rows convolved with the Ram-Lak kernel h(0) = 1/(4 tau^2),
//               h(n odd) = -1/(n pi tau)^2, h(n even) = 0 (tau: scaled pitch), times tau
//   3. back-project  f(x) = (pi / V) sum_k D_so^2 / U_k(x)^2 q_k(u_k(x), v_k(x)), U = depth of x
//               along the central ray, bilinear interpolation on the detector.
#include <cmath>

#include "gs_internal.cuh"

namespace gs {
namespace {

constexpr int kThreads = 256;
constexpr double kPi = 3.14159265358979323846;

struct FdkView {
  float s[3];       // source
  float eu[3], ev[3], n[3];
  float Dso, Dsd;   // source-to-axis-plane and source-to-detector distances
  float pu, pv;     // detector pitch
  float su, sv;     // Dsd / pu, Dsd / pv
  float Dso2;
};

__global__ void k_fdk_setup(const gs_view* __restrict__ views, int nv, FdkView* __restrict__ out) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nv) return;
  const gs_view v = views[k];
  FdkView f;
  f.pu = sqrtf(v.u[0] * v.u[0] + v.u[1] * v.u[1] + v.u[2] * v.u[2]);
  f.pv = sqrtf(v.v[0] * v.v[0] + v.v[1] * v.v[1] + v.v[2] * v.v[2]);
  float d[3];
  for (int a = 0; a < 3; ++a) {
    f.s[a] = v.src[a];
    f.eu[a] = v.u[a] / f.pu;
    f.ev[a] = v.v[a] / f.pv;
    d[a] = v.det_center[a] - v.src[a];
  }
  f.Dsd = sqrtf(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
  for (int a = 0; a < 3; ++a) f.n[a] = d[a] / f.Dsd;
  // distance from the source to the plane through the origin perpendicular to the central ray
  f.Dso = -(f.s[0] * f.n[0] + f.s[1] * f.n[1] + f.s[2] * f.n[2]);
  f.su = f.Dsd / f.pu;
  f.sv = f.Dsd / f.pv;
  f.Dso2 = f.Dso * f.Dso;
  out[k] = f;
}

// Filtered projections live in a padded layout: rows of `pitch` floats, kPadL zero columns left
// of the detector and at least two right of it, two zero rows above and below, so that the
// back-projection reads all four bilinear neighbours of a clamped position without a test.
constexpr int kPadL = 4;
int fdk_pitch(int W) { return (W + kPadL + 2 + 3) / 4 * 4; }  // rows stay 16-byte aligned
size_t fdk_padded(int n_views, int W, int H) {
  return (size_t)n_views * ((size_t)H + 4) * fdk_pitch(W);
}

// Weight and ramp-filter.  The Ram-Lak kernel vanishes at even distances, so the outputs of one
// parity are a convolution of the inputs of the other parity with the weights h(2 d + 1): a
// dense FP32 contraction (W^2 / 2 FMAs per row), bound by the FMA pipes once it is blocked.  A
// CTA filters 2 RP rows; a thread computes 16 consecutive outputs (8 of each parity) of a row
// pair in packed FP32x2 arithmetic and walks the inputs four per parity at a time, the sliding
// window of 12 weights per parity in registers (four new ones per chunk): 64 packed FMAs for
// six 16-byte shared-memory loads.  75 x 512^2: 3.19 -> 0.22 ms (the first version walked one
// output per thread with two scalar loads and a division per tap).  RP = 4 while the rows fit
// beside a second CTA, RP = 1 for wider detectors.
constexpr int kFilterThreads = 128;
struct FilterShape {
  int Wp, plane, G, nT;
  size_t smem;
};
__host__ __device__ inline FilterShape filter_shape(int W, int RP) {
  FilterShape s;
  const int Wh = (W + 1) / 2;
  s.Wp = (Wh + 11) / 12 * 12;  // inputs per parity, zero-padded to whole weight rotations
  // plane = float2 per (row pair, parity), 2 mod 8: the row pairs' 16-byte loads hit other banks
  s.plane = s.Wp + (s.Wp % 8 == 0 ? 2 : 6);
  s.G = (W + 15) / 16;
  s.nT = s.Wp + 8 * s.G;       // weights of distances -Wp .. 8 G - 1
  s.smem = sizeof(float) * (4 * (size_t)RP * s.plane + 2 * (size_t)s.nT);
  return s;
}
// 2 d + 1 (parity 1 outputs) and 2 d - 1 (parity 0): the odd distance of weight index d
__device__ __forceinline__ float ramlak_odd(float hk, int m) { return hk / (float)(m * m); }

// One chunk: inputs b0 .. b0 + 3 of the other parity into the eight outputs a0 .. a0 + 7, the
// weights of distances a0 - b0 - 4 .. a0 - b0 + 7 in A, B, C.
__device__ __forceinline__ void filter_chunk(const float4 A, const float4 B, const float4 C,
                                             const float2* __restrict__ in, float2 (&acc)[8]) {
  const float4 p = *reinterpret_cast<const float4*>(in), q = *reinterpret_cast<const float4*>(in + 2);
  const float2 x[4] = {make_float2(p.x, p.y), make_float2(p.z, p.w), make_float2(q.x, q.y),
                       make_float2(q.z, q.w)};
  const float w[12] = {A.x, A.y, A.z, A.w, B.x, B.y, B.z, B.w, C.x, C.y, C.z, C.w};
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int o = 0; o < 8; ++o) {
      const float wt = w[o - c + 4];
      acc[o] = __ffma2_rn(make_float2(wt, wt), x[c], acc[o]);
    }
}

template <int RP>
__global__ void __launch_bounds__(kFilterThreads)
    k_fdk_filter(const float* __restrict__ proj, const FdkView* __restrict__ fv, int W, int H,
                 int pitch, float* __restrict__ out) {
  extern __shared__ float4 sm_f4[];
  const FilterShape S = filter_shape(W, RP);
  float2* s_in = reinterpret_cast<float2*>(sm_f4);               // [RP][parity][plane]
  float* s_w = reinterpret_cast<float*>(s_in + 2 * RP * S.plane);  // [parity][nT]
  const int v = blockIdx.y, row0 = blockIdx.x * 2 * RP;
  const FdkView f = fv[v];
  const float scale = f.Dso / f.Dsd;
  const float tau = f.pu * scale;
  const float h0 = 0.25f / (tau * tau);
  const float hk = -1.f / (float)(kPi * kPi) / (tau * tau);
  const float* p = proj + (size_t)v * H * W;
  float* ov = out + (size_t)v * ((size_t)H + 4) * pitch;
  // padding: the columns beside this CTA's rows, the rows above the first and below the last
  for (int r = 0; r < 2 * RP; ++r) {
    if (row0 + r >= H) break;
    float* o = ov + (size_t)(row0 + r + 2) * pitch;
    for (int c = threadIdx.x; c < pitch - W; c += kFilterThreads) o[c < kPadL ? c : W + c] = 0.f;
  }
  for (int c = threadIdx.x; c < 2 * pitch; c += kFilterThreads) {
    if (blockIdx.x == 0) ov[c] = 0.f;
    if (blockIdx.x == gridDim.x - 1) ov[(size_t)(H + 2) * pitch + c] = 0.f;
  }
  // weights and weighted inputs (positions past the row are zero)
  for (int k = threadIdx.x; k < S.nT; k += kFilterThreads) {
    const int d = k - S.Wp;
    s_w[k] = ramlak_odd(hk, 2 * d - 1);
    s_w[S.nT + k] = ramlak_odd(hk, 2 * d + 1);
  }
  for (int r = 0; r < 2 * RP; ++r) {
    const int row = row0 + r;
    const float vs = ((float)row + 0.5f - 0.5f * H) * f.pv * scale;
    for (int i = threadIdx.x; i < 2 * S.Wp; i += kFilterThreads) {
      const float us = ((float)i + 0.5f - 0.5f * W) * tau;
      const float x = row < H && i < W ? p[(size_t)row * W + i] * f.Dso *
                                             rsqrtf(f.Dso * f.Dso + us * us + vs * vs)
                                       : 0.f;
      float* d = reinterpret_cast<float*>(s_in + ((r >> 1) * 2 + (i & 1)) * S.plane + (i >> 1));
      d[r & 1] = x;
    }
  }
  __syncthreads();
  for (int item = threadIdx.x; item < S.G * RP; item += kFilterThreads) {
    const int rp = item % RP, a0 = (item / RP) * 8;
    const float2* in0 = s_in + (rp * 2) * S.plane;  // even positions
    const float2* in1 = in0 + S.plane;              // odd positions
    float2 e[8], o[8];                              // outputs 2 (a0 + k) and 2 (a0 + k) + 1
#pragma unroll
    for (int k = 0; k < 8; ++k) e[k] = o[k] = make_float2(0.f, 0.f);
    // weight index of distance d: d + Wp; a chunk at b0 adds distances a0 - b0 - 4 .. - 1
    const float* w0 = s_w + S.Wp + a0;
    const float* w1 = w0 + S.nT;
    float4 B0 = *reinterpret_cast<const float4*>(w0), C0 = *reinterpret_cast<const float4*>(w0 + 4);
    float4 B1 = *reinterpret_cast<const float4*>(w1), C1 = *reinterpret_cast<const float4*>(w1 + 4);
    for (int b0 = 0; b0 < S.Wp; b0 += 12) {  // three chunks: the window's registers rotate once
      if (a0 >= b0 && a0 < b0 + 12) {
        // the centre tap joins between the left and the right neighbours: the partial sums
        // then stay as small as the result's own terms (the ramp's taps cancel), which keeps
        // the rounding error at that of a sum taken outward from the centre
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          if (a0 + k >= S.Wp) break;
          const float2 x0 = in0[a0 + k], x1 = in1[a0 + k];
          e[k] = __ffma2_rn(make_float2(h0, h0), x0, e[k]);
          o[k] = __ffma2_rn(make_float2(h0, h0), x1, o[k]);
        }
      }
      float4 A0 = *reinterpret_cast<const float4*>(w0 - b0 - 4);
      float4 A1 = *reinterpret_cast<const float4*>(w1 - b0 - 4);
      filter_chunk(A0, B0, C0, in1 + b0, e);
      filter_chunk(A1, B1, C1, in0 + b0, o);
      C0 = *reinterpret_cast<const float4*>(w0 - b0 - 8);
      C1 = *reinterpret_cast<const float4*>(w1 - b0 - 8);
      filter_chunk(C0, A0, B0, in1 + b0 + 4, e);
      filter_chunk(C1, A1, B1, in0 + b0 + 4, o);
      B0 = *reinterpret_cast<const float4*>(w0 - b0 - 12);
      B1 = *reinterpret_cast<const float4*>(w1 - b0 - 12);
      filter_chunk(B0, C0, A0, in1 + b0 + 8, e);
      filter_chunk(B1, C1, A1, in0 + b0 + 8, o);
      // the next chunk's window is (new, B0, C0)
    }
    const int i0 = 2 * a0;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int row = row0 + 2 * rp + r;
      if (row >= H) break;
      float* q = ov + (size_t)(row + 2) * pitch + kPadL + i0;
      float t[16];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        t[2 * k] = (r ? e[k].y : e[k].x) * tau;
        t[2 * k + 1] = (r ? o[k].y : o[k].x) * tau;
      }
      if (i0 + 16 <= W) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
          reinterpret_cast<float4*>(q)[k] = make_float4(t[4 * k], t[4 * k + 1], t[4 * k + 2], t[4 * k + 3]);
      } else {
#pragma unroll
        for (int k = 0; k < 16; ++k)
          if (i0 + k < W) q[k] = t[k];
      }
    }
  }
}

// Back-projection: one thread per (x, y) column of ZT voxels, a CTA per 16 x 16 x ZT block and a
// warp per 8 x 4 patch of its columns, so that a warp's bilinear reads of one view span few
// cache lines and the CTA's footprint stays in L1 (93 % hits).  Where a view's frame has no z component in its depth and u axes (every circular
// trajectory about z with an upright detector) the depth, the u position and both weights are
// the column's and only v advances along z; other views take the general form.  Positions are
// clamped into the padded image, whose border is zero, so the four reads need no test.  Bound
// by the L1 reads (four per sample; ncu: L1 77 % busy, DRAM 1 %).  256^3 from 75 x 512^2:
// 5.16 -> 1.56 ms (one voxel per thread, general geometry and four tested reads per sample
// before; warps of 16 x 2 columns 1.69, of 32 x 1 2.2 ms).
__device__ __forceinline__ float fdk_bilinear(const float* __restrict__ q, int pitch, int ix,
                                              float ax, float cy, float ymax) {
  cy = fminf(fmaxf(cy, -2.f), ymax);
  const float fy = floorf(cy);
  const float ay = cy - fy;
  const float* r0 = q + (int64_t)((int)fy + 2) * pitch + ix;
  const float* r1 = r0 + pitch;
  const float a = __ldg(r0), b = __ldg(r0 + 1), c = __ldg(r1), d = __ldg(r1 + 1);
  const float top = fmaf(ax, b - a, a), bot = fmaf(ax, d - c, c);
  return fmaf(ay, bot - top, top);
}

constexpr int kBackX = 16, kBackY = kThreads / kBackX;  // columns of a CTA
constexpr int kPatchX = 8, kPatchY = 4;                   // and of a warp
template <int ZT>
__global__ void __launch_bounds__(kThreads)
    k_fdk_backproject(const float* __restrict__ q, const FdkView* __restrict__ fv, int nv, int W,
                      int H, int pitch, int64_t view, int nx, int ny, int nz, float ox, float oy,
                      float oz, float hx, float hy, float hz, float* __restrict__ vol) {
  __shared__ FdkView s_v[64];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int bx = (nx - 1) / kBackX + 1, by = (ny - 1) / kBackY + 1;  // up to 2^31 - 1 voxels a side
  const int x = (int)(blockIdx.x % bx) * kBackX + w % (kBackX / kPatchX) * kPatchX + lane % kPatchX;
  const int y = (int)(blockIdx.x / bx % by) * kBackY + w / (kBackX / kPatchX) * kPatchY + lane / kPatchX;
  const int z0 = (int)(blockIdx.x / bx / by) * ZT;
  const bool live = x < nx && y < ny;
  const float px = ox + ((float)x + 0.5f) * hx, py = oy + ((float)y + 0.5f) * hy;
  const float xmax = (float)W, ymax = (float)H;  // clamped positions lie in the zero border
  float pz[ZT], acc[ZT];
#pragma unroll
  for (int k = 0; k < ZT; ++k) {
    pz[k] = oz + ((float)(z0 + k) + 0.5f) * hz;
    acc[k] = 0.f;
  }
  for (int base = 0; base < nv; base += 64) {
    const int m = min(64, nv - base);
    __syncthreads();
    for (int k = threadIdx.x; k < m; k += kThreads) s_v[k] = fv[base + k];
    __syncthreads();
    if (!live) continue;
    const float* qv = q + base * view + kPadL;
    for (int k = 0; k < m; ++k, qv += view) {
      const FdkView& f = s_v[k];
      const float rx = px - f.s[0], ry = py - f.s[1];
      const float Ub = rx * f.n[0] + ry * f.n[1];
      const float ub = rx * f.eu[0] + ry * f.eu[1], vb = rx * f.ev[0] + ry * f.ev[1];
      if (f.n[2] == 0.f && f.eu[2] == 0.f) {
        if (!(Ub > 0.f)) continue;
        const float iU = 1.f / Ub;
        const float cx = fminf(fmaxf(fmaf(ub * iU, f.su, 0.5f * W - 0.5f), -2.f), xmax);
        const float fx = floorf(cx);
        const float ax = cx - fx, g = iU * f.sv, wt = f.Dso2 * iU * iU;
#pragma unroll
        for (int j = 0; j < ZT; ++j) {
          const float cy = fmaf(fmaf(pz[j] - f.s[2], f.ev[2], vb), g, 0.5f * H - 0.5f);
          acc[j] = fmaf(wt, fdk_bilinear(qv, pitch, (int)fx, ax, cy, ymax), acc[j]);
        }
      } else {
#pragma unroll
        for (int j = 0; j < ZT; ++j) {
          const float rz = pz[j] - f.s[2];
          const float U = fmaf(rz, f.n[2], Ub);
          if (!(U > 0.f)) continue;
          const float iU = 1.f / U;
          const float cx =
              fminf(fmaxf(fmaf(fmaf(rz, f.eu[2], ub) * iU, f.su, 0.5f * W - 0.5f), -2.f), xmax);
          const float cy = fmaf(fmaf(rz, f.ev[2], vb), iU * f.sv, 0.5f * H - 0.5f);
          const float fx = floorf(cx);
          acc[j] = fmaf(f.Dso2 * iU * iU,
                        fdk_bilinear(qv, pitch, (int)fx, cx - fx, cy, ymax), acc[j]);
        }
      }
    }
  }
  if (!live) return;
#pragma unroll
  for (int k = 0; k < ZT; ++k)
    if (z0 + k < nz) vol[((size_t)(z0 + k) * ny + y) * nx + x] = acc[k] * (float)(kPi / nv);
}

// ------------------------------------------------------------------------------------------
// Gradient-magnitude sampling
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ unsigned ordered(float f) {
  const unsigned u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float unordered(unsigned u) {
  return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

__global__ void k_vmax_init(unsigned* vmax) { *vmax = 0u; }

__global__ void __launch_bounds__(kThreads)
    k_vmax(const float* __restrict__ v, int64_t total, unsigned* __restrict__ vmax) {
  float m = -INFINITY;
  for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * kThreads)
    m = fmaxf(m, v[i]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(vmax, ordered(m));
}

// w = |grad V| (central differences, one-sided at the border) where V > frac * max(V), else 0;
// per-block FP64 sums of w for the scan.
__global__ void __launch_bounds__(kThreads)
    k_grad_weight(const float* __restrict__ V, int nx, int ny, int nz, float hx, float hy,
                  float hz, const unsigned* __restrict__ vmax, float frac,
                  double* __restrict__ w, double* __restrict__ block_sums) {
  __shared__ double part[kThreads / 32];
  const int64_t total = (int64_t)nx * ny * nz;
  const int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  double val = 0.0;
  if (i < total) {
    const int x = (int)(i % nx), y = (int)((i / nx) % ny), z = (int)(i / ((int64_t)nx * ny));
    const float thr = __fmul_rn(frac, unordered(*vmax));
    const float c = V[i];
    if (c > thr) {
      const int64_t sy = nx, sz = (int64_t)nx * ny;
      const int xa = max(x - 1, 0), xb = min(x + 1, nx - 1);
      const int ya = max(y - 1, 0), yb = min(y + 1, ny - 1);
      const int za = max(z - 1, 0), zb = min(z + 1, nz - 1);
      // plain IEEE single-precision operations without contraction, so that the weights (and
      // with them the sampled voxel indices) can be reproduced exactly off the device
      const float gx = xb > xa ? __fdiv_rn(__fsub_rn(V[i + (xb - x)], V[i - (x - xa)]),
                                           __fmul_rn((float)(xb - xa), hx)) : 0.f;
      const float gy = yb > ya ? __fdiv_rn(__fsub_rn(V[i + (yb - y) * sy], V[i - (y - ya) * sy]),
                                           __fmul_rn((float)(yb - ya), hy)) : 0.f;
      const float gz = zb > za ? __fdiv_rn(__fsub_rn(V[i + (zb - z) * sz], V[i - (z - za) * sz]),
                                           __fmul_rn((float)(zb - za), hz)) : 0.f;
      val = (double)__fsqrt_rn(__fadd_rn(__fadd_rn(__fmul_rn(gx, gx), __fmul_rn(gy, gy)),
                                         __fmul_rn(gz, gz)));
    }
    w[i] = val;
  }
  double s = val;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double b = 0.0;
    for (int k = 0; k < kThreads / 32; ++k) b += part[k];
    block_sums[blockIdx.x] = b;
  }
}

// exclusive scan of the block sums in one CTA (FP64)
__global__ void __launch_bounds__(1024) k_scan_f64(double* __restrict__ sums, int nb) {
  __shared__ double warp_tot[32];
  const int t = threadIdx.x, lane = t & 31, wi = t >> 5;
  const int per = (nb + 1023) / 1024;
  const int b0 = min(nb, t * per), b1 = min(nb, b0 + per);
  double local = 0.0;
  for (int b = b0; b < b1; ++b) local += sums[b];
  double incl = local;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double u = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += u;
  }
  if (lane == 31) warp_tot[wi] = incl;
  __syncthreads();
  if (wi == 0) {
    double v = warp_tot[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double u = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += u;
    }
    warp_tot[lane] = v;
  }
  __syncthreads();
  double run = incl - local + (wi > 0 ? warp_tot[wi - 1] : 0.0);
  for (int b = b0; b < b1; ++b) {
    const double x = sums[b];
    sums[b] = run;
    run += x;
  }
  if (t == 1023) sums[nb] = warp_tot[31];  // grand total
}

// inclusive prefix of w inside each block, plus the block's offset: w becomes the CDF
__global__ void __launch_bounds__(kThreads)
    k_cdf(double* __restrict__ w, int64_t total, const double* __restrict__ offs) {
  __shared__ double warp_tot[kThreads / 32];
  const int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
  double v = i < total ? w[i] : 0.0;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double u = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += u;
  }
  if (lane == 31) warp_tot[wi] = v;
  __syncthreads();
  double pre = offs[blockIdx.x];
  for (int k = 0; k < wi; ++k) pre += warp_tot[k];
  if (i < total) w[i] = pre + v;
}

__device__ __forceinline__ float trilinear(const float* V, int nx, int ny, int nz, float cx,
                                           float cy, float cz) {
  cx = fminf(fmaxf(cx, 0.f), (float)(nx - 1));
  cy = fminf(fmaxf(cy, 0.f), (float)(ny - 1));
  cz = fminf(fmaxf(cz, 0.f), (float)(nz - 1));
  const int x0 = min((int)floorf(cx), nx - 1), y0 = min((int)floorf(cy), ny - 1),
            z0 = min((int)floorf(cz), nz - 1);
  const int x1 = min(x0 + 1, nx - 1), y1 = min(y0 + 1, ny - 1), z1 = min(z0 + 1, nz - 1);
  const float ax = cx - x0, ay = cy - y0, az = cz - z0;
  auto at = [&](int x, int y, int z) { return V[((size_t)z * ny + y) * nx + x]; };
  const float c00 = at(x0, y0, z0) * (1 - ax) + at(x1, y0, z0) * ax;
  const float c10 = at(x0, y1, z0) * (1 - ax) + at(x1, y1, z0) * ax;
  const float c01 = at(x0, y0, z1) * (1 - ax) + at(x1, y0, z1) * ax;
  const float c11 = at(x0, y1, z1) * (1 - ax) + at(x1, y1, z1) * ax;
  return (c00 * (1 - ay) + c10 * ay) * (1 - az) + (c01 * (1 - ay) + c11 * ay) * az;
}

// thread per Gaussian: voxel chosen by inverse CDF, jittered inside the voxel
__global__ void __launch_bounds__(kThreads)
    k_sample(const double* __restrict__ cdf, int64_t total, const double* __restrict__ grand,
             const float* __restrict__ V, int nx, int ny, int nz, float ox, float oy, float oz,
             float hx, float hy, float hz, const float* __restrict__ uni, int n, float k_density,
             float4* __restrict__ mean_rho, float4* __restrict__ quat,
             int32_t* __restrict__ voxel_out) {
  const int j = blockIdx.x * kThreads + threadIdx.x;
  if (j >= n) return;
  const double target = (double)uni[4 * j] * grand[0];
  // first index with cdf > target
  int64_t lo = 0, hi = total - 1;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (cdf[mid] > target) hi = mid; else lo = mid + 1;
  }
  const int x = (int)(lo % nx), y = (int)((lo / nx) % ny), z = (int)(lo / ((int64_t)nx * ny));
  const float cx = (float)x + uni[4 * j + 1], cy = (float)y + uni[4 * j + 2],
              cz = (float)z + uni[4 * j + 3];  // index-space position (voxel centre at +0.5)
  const float px = ox + cx * hx, py = oy + cy * hy, pz = oz + cz * hz;
  const float rho = k_density * trilinear(V, nx, ny, nz, cx - 0.5f, cy - 0.5f, cz - 0.5f);
  mean_rho[j] = make_float4(px, py, pz, rho);
  quat[j] = make_float4(1.f, 0.f, 0.f, 0.f);
  if (voxel_out) voxel_out[j] = (int32_t)lo;
}

// ------------------------------------------------------------------------------------------
// Nearest-neighbour distance on a uniform hash grid (counting sort by cell, then an expanding
// search over shells of cells)
// ------------------------------------------------------------------------------------------
struct HashGrid {
  float lo[3];
  float cell;
  int dim[3];
};

__device__ __forceinline__ int cell_of(const HashGrid& g, float p, int a) {
  return min(g.dim[a] - 1, max(0, (int)floorf((p - g.lo[a]) / g.cell)));
}

__global__ void __launch_bounds__(kThreads)
    k_hash_count(const float4* __restrict__ pts, int n, HashGrid g, uint32_t* __restrict__ cnt,
                 uint32_t* __restrict__ cell_id) {
  const int j = blockIdx.x * kThreads + threadIdx.x;
  if (j >= n) return;
  const float4 p = pts[j];
  const int c = (cell_of(g, p.z, 2) * g.dim[1] + cell_of(g, p.y, 1)) * g.dim[0] + cell_of(g, p.x, 0);
  cell_id[j] = (uint32_t)c;
  atomicAdd(&cnt[c], 1u);
}

__global__ void __launch_bounds__(1024) k_scan_u32_single(uint32_t* __restrict__ a, int n) {
  __shared__ uint32_t warp_tot[32];
  const int t = threadIdx.x, lane = t & 31, wi = t >> 5;
  const int per = (n + 1023) / 1024;
  const int b0 = min(n, t * per), b1 = min(n, b0 + per);
  uint32_t local = 0;
  for (int b = b0; b < b1; ++b) local += a[b];
  uint32_t incl = gsd::warp_inclusive_scan(local);
  if (lane == 31) warp_tot[wi] = incl;
  __syncthreads();
  if (wi == 0) warp_tot[lane] = gsd::warp_inclusive_scan(warp_tot[lane]);
  __syncthreads();
  uint32_t run = incl - local + (wi > 0 ? warp_tot[wi - 1] : 0u);
  for (int b = b0; b < b1; ++b) {
    const uint32_t x = a[b];
    a[b] = run;
    run += x;
  }
  if (t == 1023) a[n] = warp_tot[31];
}

__global__ void __launch_bounds__(kThreads)
    k_hash_fill(const uint32_t* __restrict__ cell_id, int n, uint32_t* __restrict__ cursor,
                uint32_t* __restrict__ sorted) {
  const int j = blockIdx.x * kThreads + threadIdx.x;
  if (j >= n) return;
  sorted[atomicAdd(&cursor[cell_id[j]], 1u)] = (uint32_t)j;
}

__global__ void __launch_bounds__(kThreads)
    k_nn(const float4* __restrict__ pts, int n, HashGrid g, const uint32_t* __restrict__ start,
         const uint32_t* __restrict__ sorted, float min_scale, float4* __restrict__ scale) {
  const int j = blockIdx.x * kThreads + threadIdx.x;
  if (j >= n) return;
  const float4 p = pts[j];
  const int cx = cell_of(g, p.x, 0), cy = cell_of(g, p.y, 1), cz = cell_of(g, p.z, 2);
  float best = INFINITY;  // squared distance
  const int rmax = max(g.dim[0], max(g.dim[1], g.dim[2]));
  for (int r = 0; r <= rmax; ++r) {
    // a point in a cell r shells away is at least (r - 1) cells from p
    const float inner = (float)(r - 1) * g.cell;
    if (r >= 1 && best <= inner * inner) break;
    for (int z = cz - r; z <= cz + r; ++z) {
      if (z < 0 || z >= g.dim[2]) continue;
      for (int y = cy - r; y <= cy + r; ++y) {
        if (y < 0 || y >= g.dim[1]) continue;
        const bool edge_zy = (z == cz - r || z == cz + r || y == cy - r || y == cy + r);
        for (int x = cx - r; x <= cx + r; x += (edge_zy || r == 0) ? 1 : 2 * r) {
          if (x < 0 || x >= g.dim[0]) continue;
          const int c = (z * g.dim[1] + y) * g.dim[0] + x;
          for (uint32_t k = start[c]; k < start[c + 1]; ++k) {
            const uint32_t o = sorted[k];
            if ((int)o == j) continue;
            const float4 q = pts[o];
            const float dx = q.x - p.x, dy = q.y - p.y, dz = q.z - p.z;
            best = fminf(best, dx * dx + dy * dy + dz * dz);
          }
        }
      }
    }
  }
  const float d = best < INFINITY ? sqrtf(best) : min_scale;
  const float s = fmaxf(d, min_scale);
  scale[j] = make_float4(s, s, s, 0.f);
}

bool al16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

struct InitLayout {
  double* w = nullptr;         // total: weights, then CDF
  double* bsums = nullptr;     // nblocks + 1
  unsigned* vmax = nullptr;
  uint32_t* cnt = nullptr;     // cells + 1
  uint32_t* cell_id = nullptr; // n
  uint32_t* sorted = nullptr;  // n
  uint32_t* cursor = nullptr;  // cells
  size_t bytes = 0;
};

HashGrid make_hash(const gs_grid* g, int n) {
  HashGrid h;
  float ext[3];
  for (int a = 0; a < 3; ++a) {
    h.lo[a] = g->origin[a];
    ext[a] = g->dims[a] * g->voxel[a];
  }
  // about two points per cell on average, never smaller than a voxel
  const double vol = (double)ext[0] * ext[1] * ext[2];
  float c = (float)cbrt(vol * 2.0 / std::max(n, 1));
  c = std::max(c, std::max(g->voxel[0], std::max(g->voxel[1], g->voxel[2])));
  h.cell = c;
  for (int a = 0; a < 3; ++a) h.dim[a] = std::max(1, std::min(256, (int)ceilf(ext[a] / c)));
  // cells are clamped to 256 per axis; enlarge the cell so that they still cover the extent
  for (int a = 0; a < 3; ++a) h.cell = std::max(h.cell, ext[a] / h.dim[a]);
  return h;
}

InitLayout carve_init(void* ws, const gs_grid* g, int n) {
  const int64_t total = (int64_t)g->dims[0] * g->dims[1] * g->dims[2];
  const int64_t nb = (total + kThreads - 1) / kThreads;
  const HashGrid h = make_hash(g, n);
  const int64_t cells = (int64_t)h.dim[0] * h.dim[1] * h.dim[2];
  Carve c(ws);
  InitLayout L;
  L.w = c.take<double>(total);
  L.bsums = c.take<double>(nb + 1);
  L.vmax = c.take<unsigned>(1);
  L.cnt = c.take<uint32_t>(cells + 1);
  L.cursor = c.take<uint32_t>(cells + 1);
  L.cell_id = c.take<uint32_t>(n);
  L.sorted = c.take<uint32_t>(n);
  L.bytes = align_up(c.off, 256);
  return L;
}

}  // namespace

// Shared with the volume fit: sampling of n Gaussians from a volume.
int grad_init(const float* d_vol, const gs_grid* g, int n, float frac, float k_density,
              float min_scale, const float* d_uniforms, float* d_mean_rho, float* d_scale,
              float* d_quat, int32_t* d_voxel, void* d_ws, size_t ws_bytes, cudaStream_t s) {
  InitLayout L = carve_init(d_ws, g, n);
  if (ws_bytes < L.bytes) return GS_ERR_CAPACITY;
  const int nx = g->dims[0], ny = g->dims[1], nz = g->dims[2];
  const int64_t total = (int64_t)nx * ny * nz;
  const int64_t nb = (total + kThreads - 1) / kThreads;
  if (nb > ((int64_t)1 << 31) - 1) return GS_ERR_ARG;
  GS_TRY(launch("vmax_init", k_vmax_init, dim3(1), dim3(1), 0, s, L.vmax));
  GS_TRY(launch("vmax", k_vmax, dim3((unsigned)std::min<int64_t>(nb, 8 * num_sms())),
                dim3(kThreads), 0, s, d_vol, total, L.vmax));
  GS_TRY(launch("grad_weight", k_grad_weight, dim3((unsigned)nb), dim3(kThreads), 0, s, d_vol,
                nx, ny, nz, g->voxel[0], g->voxel[1], g->voxel[2], (const unsigned*)L.vmax,
                frac, L.w, L.bsums));
  GS_TRY(launch("scan_f64", k_scan_f64, dim3(1), dim3(1024), 0, s, L.bsums, (int)nb));
  GS_TRY(launch("cdf", k_cdf, dim3((unsigned)nb), dim3(kThreads), 0, s, L.w, total,
                (const double*)L.bsums));
  const int gb = (n + kThreads - 1) / kThreads;
  GS_TRY(launch("sample", k_sample, dim3(gb), dim3(kThreads), 0, s, (const double*)L.w, total,
                (const double*)(L.bsums + nb), d_vol, nx, ny, nz, g->origin[0], g->origin[1],
                g->origin[2], g->voxel[0], g->voxel[1], g->voxel[2], d_uniforms, n, k_density,
                (float4*)d_mean_rho, (float4*)d_quat, d_voxel));
  const HashGrid h = make_hash(g, n);
  const int64_t cells = (int64_t)h.dim[0] * h.dim[1] * h.dim[2];
  GS_CUDA(cudaMemsetAsync(L.cnt, 0, (cells + 1) * sizeof(uint32_t), s));
  GS_TRY(launch("hash_count", k_hash_count, dim3(gb), dim3(kThreads), 0, s,
                (const float4*)d_mean_rho, n, h, L.cnt, L.cell_id));
  GS_TRY(launch("scan_u32", k_scan_u32_single, dim3(1), dim3(1024), 0, s, L.cnt, (int)cells));
  GS_CUDA(cudaMemcpyAsync(L.cursor, L.cnt, (cells + 1) * sizeof(uint32_t),
                          cudaMemcpyDeviceToDevice, s));
  GS_TRY(launch("hash_fill", k_hash_fill, dim3(gb), dim3(kThreads), 0, s,
                (const uint32_t*)L.cell_id, n, L.cursor, L.sorted));
  return launch("nn", k_nn, dim3(gb), dim3(kThreads), 0, s, (const float4*)d_mean_rho, n, h,
                (const uint32_t*)L.cnt, (const uint32_t*)L.sorted, min_scale,
                (float4*)d_scale);
}

size_t grad_init_workspace(const gs_grid* g, int n) { return carve_init(nullptr, g, n).bytes; }

}  // namespace gs

using namespace gs;

extern "C" {

size_t gs_fdk_workspace_size(int n_views, int W, int H) {
  if (n_views < 1 || W < 1 || H < 1) return 0;
  return align_up(fdk_padded(n_views, W, H) * sizeof(float), 256) +
         align_up((size_t)n_views * sizeof(FdkView), 256) + 16;  // the workspace may start anywhere
}

}  // extern "C"

namespace gs {
namespace {
template <int RP>
int fdk_filter(const float* proj, const FdkView* fv, int nv, int W, int H, float* q,
               cudaStream_t s) {
  const size_t smem = filter_shape(W, RP).smem;
  if (smem > 48 * 1024)  // host-side state of the current device, set on every call
    GS_CUDA(cudaFuncSetAttribute(k_fdk_filter<RP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem));
  return launch("fdk_filter", k_fdk_filter<RP>, dim3((H + 2 * RP - 1) / (2 * RP), nv),
                dim3(kFilterThreads), smem, s, proj, fv, W, H, fdk_pitch(W), q);
}

// 16 x 16 blocks of columns of the back-projection.
int64_t fdk_columns(const gs_grid* g) {
  return (((int64_t)g->dims[0] + kBackX - 1) / kBackX) * (((int64_t)g->dims[1] + kBackY - 1) / kBackY);
}

template <int ZT>
int fdk_backproject(const float* q, const FdkView* fv, int nv, int W, int H, const gs_grid* g,
                    float* vol, cudaStream_t s) {
  const int nx = g->dims[0], ny = g->dims[1], nz = g->dims[2];
  const int64_t blocks = fdk_columns(g) * (((int64_t)nz + ZT - 1) / ZT);
  if (blocks > ((int64_t)1 << 31) - 1) return GS_ERR_ARG;
  return launch("fdk_backproject", k_fdk_backproject<ZT>, dim3((unsigned)blocks), dim3(kThreads),
                0, s, q, fv, nv, W, H, fdk_pitch(W), (int64_t)fdk_padded(1, W, H), nx, ny, nz,
                g->origin[0], g->origin[1], g->origin[2], g->voxel[0], g->voxel[1], g->voxel[2],
                vol);
}
}  // namespace
}  // namespace gs

extern "C" {

int gs_fdk(const float* d_proj, const gs_view* d_views, int n_views, int W, int H,
           const gs_grid* grid, float* d_vol, void* d_ws, size_t ws_bytes, void* stream) {
  if (!d_proj || !d_views || !grid || !d_vol || !d_ws || n_views < 1 || n_views > 65535 ||
      W < 1 || H < 1 || W > 12288)
    return GS_ERR_ARG;
  for (int k = 0; k < 3; ++k)
    if (grid->dims[k] < 1 || !(grid->voxel[k] > 0.f)) return GS_ERR_ARG;
  if (ws_bytes < gs_fdk_workspace_size(n_views, W, H)) return GS_ERR_CAPACITY;
  cudaStream_t s = (cudaStream_t)stream;
  Carve c((void*)(((uintptr_t)d_ws + 15) & ~(uintptr_t)15));
  float* q = c.take<float>(fdk_padded(n_views, W, H));
  FdkView* fv = c.take<FdkView>(n_views);
  GS_TRY(launch("fdk_setup", k_fdk_setup, dim3((n_views + 63) / 64), dim3(64), 0, s, d_views,
                n_views, fv));
  if (filter_shape(W, 4).smem <= 110 * 1024)
    GS_TRY(fdk_filter<4>(d_proj, fv, n_views, W, H, q, s));
  else
    GS_TRY(fdk_filter<1>(d_proj, fv, n_views, W, H, q, s));
  // more voxels per thread share more of a column's geometry; fewer while the grid would leave
  // SMs idle (four CTAs each).  256^3 from 75 x 512^2: 1.56 ms with 16, 1.83 with 8, 2.1 with 4;
  // 32 spills the block's rows out of L1 (2.9 ms)
  const int64_t cols = fdk_columns(grid), nz = grid->dims[2];
  const int64_t want = 4 * (int64_t)num_sms();
  if (cols * ((nz + 15) / 16) >= want)
    return fdk_backproject<16>(q, fv, n_views, W, H, grid, d_vol, s);
  if (cols * ((nz + 3) / 4) >= want)
    return fdk_backproject<4>(q, fv, n_views, W, H, grid, d_vol, s);
  return fdk_backproject<1>(q, fv, n_views, W, H, grid, d_vol, s);
}

size_t gs_grad_init_workspace_size(const gs_grid* grid, int n) {
  if (!grid || n < 1) return 0;
  return grad_init_workspace(grid, n);
}

int gs_grad_init(const float* d_vol, const gs_grid* grid, int n, float threshold_frac,
                 float density_k, float min_scale, const float* d_uniforms, float* d_mean_rho,
                 float* d_scale, float* d_quat, int32_t* d_voxel, void* d_ws, size_t ws_bytes,
                 void* stream) {
  if (!d_vol || !grid || n < 1 || !d_uniforms || !d_mean_rho || !d_scale || !d_quat || !d_ws)
    return GS_ERR_ARG;
  if (!al16(d_mean_rho) || !al16(d_scale) || !al16(d_quat)) return GS_ERR_ARG;
  for (int k = 0; k < 3; ++k)
    if (grid->dims[k] < 1 || !(grid->voxel[k] > 0.f)) return GS_ERR_ARG;
  return grad_init(d_vol, grid, n, threshold_frac, density_k, min_scale, d_uniforms, d_mean_rho,
                   d_scale, d_quat, d_voxel, d_ws, ws_bytes, (cudaStream_t)stream);
}

}  // extern "C"
