// warp_kernels.cu -- the trilinear warp I_k o Phi_ki^i with the flow-to-image
// upsample fused in (Sec. Background; flows on the 2x coarser grid of Sec.
// Implementation Details), and its adjoint fused with the transposed upsample.
//
// The image voxels 2m + d, d in {0,1}^3, form the block of flow node m. With voxel-centre alignment
// q = (p + 1/2)/2 - 1/2 and clamp-to-edge sampling, the upsampled displacement
// of image voxel 2m is 0.25 U(m-1) + 0.75 U(m) and of 2m+1 is
// 0.75 U(m) + 0.25 U(m+1) along each axis, with node indices clamped into the
// grid: an exact separable stencil on the 3x3x3 nodes around m. The forward also stores grad I_k at the sample
// point (12 B per voxel), which spares the adjoint the upsample and the 8-corner
// gathers. The adjoint applies the transpose of the stencil, reduced along W with
// warp shuffles, along H in shared memory and along D in registers while
// streaming over D; every flow node is written once. When the image width is a
// multiple of 4 the adjoint's inputs (dL/dW and the three components of grad I_k) are
// staged plane pair by plane pair by the tensor memory accelerator, two stages ahead.
#include <string.h>

#include <mutex>

#include "kernels.h"
#include "tma.cuh"

namespace muster {

namespace {

constexpr int BX = 32, BY = 8;             // forward: threads per CTA (image columns x node rows)
constexpr int kWarpCtas = 4;               // CTAs per SM its registers are cut for
constexpr int RX = 32, RY = 8;             // adjoint: threads per CTA (W lanes x H)
constexpr int OX = RX - 2, OY = RY - 2;    // adjoint: flow nodes written per CTA
// the staged adjoint's box starts at x = 2 (OX blockIdx.x - 1) - 2, a multiple of 4 floats
// (a tensor copy must start on a 16-byte boundary) only while OX is even
static_assert(OX % 2 == 0, "the staged warp-adjoint box must start at a multiple of 4 floats");


// The stencil's passes with weights 0.25 / 0.75, scaled by 4 (a power of two commutes with every
// rounding): a + 3 b with the product rounded first, and 3 b + c in one rounding, as the unscaled
// fma(0.25, a, 0.75 b) and fma(0.75, b, 0.25 c) round.
__device__ __forceinline__ float3 lower(float3 a, float3 b) {
  return make_float3(__fadd_rn(a.x, __fmul_rn(3.f, b.x)), __fadd_rn(a.y, __fmul_rn(3.f, b.y)),
                     __fadd_rn(a.z, __fmul_rn(3.f, b.z)));
}
__device__ __forceinline__ float3 upper(float3 b, float3 c) {
  return make_float3(fmaf(3.f, b.x, c.x), fmaf(3.f, b.y, c.y), fmaf(3.f, b.z, c.z));
}

// A moving image as cells along W: cell (z, y, x) holds I(x) and I(x + 1) - I(x), which every
// trilinear sample starts with, for -1 <= z, y, x < n and the coordinates clamped into the grid
// (k_image_cells). One 8-byte load replaces two 4-byte ones and a subtraction. The sampling operator
// clamps each coordinate into the grid; on the extended volume a coordinate clamped to
// [-1/2, n - 1/2] samples the same values, and its derivative is 0 outside [0, n - 1] by itself,
// because the two nodes of a border cell are equal. So no corner needs its own offset or a test.
struct Cells {
  const float2* p00;  // cell (-1, -1, -1); the three others one row, one plane, both further
  const float2 *p01, *p10, *p11;
  unsigned n1, n2, k;  // rows per plane, row pitch, offset of the magic numbers below
  float hz, hy, hx;    // upper clamps
  __device__ __forceinline__ Cells(const float2* p, Dims n) {
    n1 = n.n1 + 2, n2 = n.n2 + 1;
    k = 0x4B000000u * ((n1 + 1u) * n2 + 1u);
    p00 = p, p01 = p + n2, p10 = p + (size_t)n1 * n2, p11 = p10 + n2;
    hz = n.n0 - 0.5f, hy = n.n1 - 0.5f, hx = n.n2 - 0.5f;
  }
  // the cells of rows (y, y + 1) of planes (z, z + 1) at the positions b of cell_axis
  __device__ __forceinline__ void load(unsigned bz, unsigned by, unsigned bx, float2 (&v)[2][2]) const {
    const unsigned o = (bz * n1 + by) * n2 + bx - k;
    v[0][0] = __ldg(p00 + o), v[0][1] = __ldg(p01 + o), v[1][0] = __ldg(p10 + o), v[1][1] = __ldg(p11 + o);
  }
};
// The same cells made on the way from the image itself, for a context whose device has no room for them
// (8 bytes per voxel): two loads and a subtraction per cell (an evaluation of 8 x 160^3 takes 6039 us, with
// cells 5936).
struct Voxels {
  const float* p;
  int n1, n2, mz, my, mx;  // rows per plane, row pitch, last index per axis
  float hz, hy, hx;
  __device__ __forceinline__ Voxels(const float* image, Dims n) {
    p = image, n1 = n.n1, n2 = n.n2, mz = n.n0 - 1, my = n.n1 - 1, mx = n.n2 - 1;
    hz = n.n0 - 0.5f, hy = n.n1 - 0.5f, hx = n.n2 - 0.5f;
  }
  __device__ __forceinline__ void load(unsigned bz, unsigned by, unsigned bx, float2 (&v)[2][2]) const {
    const int z = (int)(bz - 0x4B000001u), y = (int)(by - 0x4B000001u), x = (int)(bx - 0x4B000001u);  // -1 .. n - 1
    const int zs[2] = {max(z, 0), min(z + 1, mz)}, ys[2] = {max(y, 0), min(y + 1, my)};
    const int x0 = max(x, 0), x1 = min(x + 1, mx);
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const float* row = p + (zs[a] * n1 + ys[b]) * n2;
        const float l = __ldg(row + x0), r = __ldg(row + x1);
        v[a][b] = make_float2(l, __fsub_rn(r, l));
      }
  }
};
// one axis: c = q clamped (a NaN to -1/2), bits of floor(c) + 1 + 2^23 (adding 2^23 + 1 rounded
// down leaves floor(c) + 1 in the last bits: full-rate adds instead of FRND and F2I), t = c - floor(c)
__device__ __forceinline__ unsigned cell_axis(float q, float hi, float& t) {
  const float c = fminf(fmaxf(q, -0.5f), hi);
  const float r = __fadd_rd(c, 8388609.f);
  t = c - (r - 8388609.f);
  return __float_as_uint(r);
}
// S[I](q), with GRAD its derivative in g; I: Cells or Voxels
template <bool GRAD, class Source>
__device__ __forceinline__ float cell_sample(const Source& I, float qz, float qy, float qx, float3& g) {
  float tz, ty, tx;
  const unsigned bz = cell_axis(qz, I.hz, tz), by = cell_axis(qy, I.hy, ty), bx = cell_axis(qx, I.hx, tx);
  float2 v[2][2];
  I.load(bz, by, bx, v);
  const float2 v00 = v[0][0], v01 = v[0][1], v10 = v[1][0], v11 = v[1][1];
  const float c00 = fmaf(tx, v00.y, v00.x), c01 = fmaf(tx, v01.y, v01.x);
  const float c10 = fmaf(tx, v10.y, v10.x), c11 = fmaf(tx, v11.y, v11.x);
  const float y0 = c01 - c00, y1 = c11 - c10;
  const float c0 = fmaf(ty, y0, c00), c1 = fmaf(ty, y1, c10), z0 = c1 - c0;
  if (GRAD) {
    g.x = z0;
    g.y = lerpf(y0, y1, tz);
    g.z = lerpf(lerpf(v00.y, v01.y, ty), lerpf(v10.y, v11.y, ty), tz);
  }
  return fmaf(tz, z0, c0);
}

// The cells of image volumes (grid y over images), a warp per row, 4 cells under way per thread; bad (nullable) is
// set if a voxel is not finite. DRAM bounds it (12 bytes per voxel). 10 x 160 x 192 x 160 in four levels: 130 us
// with the check; a thread per cell that found its place by three integer divisions took 269 us, and
// the check as a pass of its own 84 us more.
constexpr int kCellRows = 8, kCellRun = 4;
__global__ void __launch_bounds__(32 * kCellRows) k_image_cells(const float* __restrict__ in, Dims n, float2* __restrict__ out,
                                                                int* __restrict__ bad) {
  grid_begin();
  const int rows = (n.n0 + 2) * (n.n1 + 2), r = blockIdx.x * kCellRows + threadIdx.y;
  if (r >= rows) return;
  const int z = r / (n.n1 + 2), y = r - z * (n.n1 + 2);
  const int yi = min(max(y - 1, 0), n.n1 - 1), zi = min(max(z - 1, 0), n.n0 - 1);
  const float* row = in + blockIdx.y * vox(n) + ((size_t)zi * n.n1 + yi) * n.n2;
  float2* o = out + ((size_t)blockIdx.y * rows + r) * (n.n2 + 1);
  bool fine = true;
  for (int x0 = (int)threadIdx.x; x0 <= n.n2; x0 += 32 * kCellRun) {  // cell x0 is that of voxel x0 - 1
    float a[kCellRun], b[kCellRun];
#pragma unroll
    for (int k = 0; k < kCellRun; ++k) {
      const int x = min(x0 + 32 * k, n.n2) - 1;
      a[k] = __ldg(row + max(x, 0)), b[k] = __ldg(row + min(x + 1, n.n2 - 1));
    }
#pragma unroll
    for (int k = 0; k < kCellRun; ++k) {
      fine = fine && isfinite(a[k]);
      if (x0 + 32 * k <= n.n2) o[x0 + 32 * k] = make_float2(a[k], __fsub_rn(b[k], a[k]));
    }
  }
  if (bad && !fine) atomicOr(bad, 1);
}

// ---- W(p) = S[I_k](p + U~(p)) for every image voxel of the pair batch; with GRAD the
// gradient of the sampled image at the same point (needed by the adjoint) is
// written too, as three planes gI[c * stride + v].
// A warp covers 32 neighbouring voxels of a row, a thread one x, the two rows of a node row and
// nz node planes of D, which it walks with the stencil's D neighbours in registers (6 vector loads
// of U per 4 voxels). What bounds it: the line look-ups of the gathers in L1 and their latency (L1
// 67 to 79 % busy, DRAM 50 to 60 %). 32 neighbouring voxels touch half the lines that the even or the
// odd voxels of 16 nodes do, and the cells halve the gathers. Measured (90 pairs of 160 x 192 x 160 /
// 20 of 91 x 109 x 91 / 240 of 256^3 / 30 of 128^3 with rigid motion): 2170 us / 107 us / 22.2 ms /
// 331 us; a 2 x 2 x 2 block per thread with eight 4-byte gathers per voxel took 2714 us / 141 us /
// 24.1 ms / 366 us. Streaming stores keep the images in L2 (5 % of the first two). Staging U in
// shared memory, 48 registers for 5 CTAs and 8 warps' rows per CTA instead of 4 or 16 were within 3 %.
template <bool GRAD, bool RIGID, bool CELLS>
__global__ void __launch_bounds__(BX* BY, kWarpCtas) k_warp(const PairDesc* __restrict__ pd, int n_pairs, Dims ni, Dims nf, int nz,
                                                 float* __restrict__ W, float* __restrict__ gI, size_t stride,
                                                 const float* __restrict__ rig) {
  grid_begin();
  // the pairs of the launch run beside each other on a tile, so that a moving image's region is read
  // from L2 by all pairs but the first
  unsigned id = blockIdx.x;
  const int pair = (int)(id % (unsigned)n_pairs);
  id /= (unsigned)n_pairs;
  const unsigned gx = (ni.n2 + BX - 1) / BX, gy = (nf.n1 + BY - 1) / BY;
  const int x = (int)(id % gx) * BX + threadIdx.x;
  id /= gx;
  const int my = (int)(id % gy) * BY + threadIdx.y, m0 = (int)(id / gy) * nz;
  if (x >= ni.n2 || my >= nf.n1) return;
  const PairDesc d = pd[pair];
  const auto I = [&] {
    if constexpr (CELLS)
      return Cells(d.Ic, ni);
    else
      return Voxels(d.Ik, ni);
  }();
  const int fp = nf.n1 * nf.n2, plane = ni.n1 * ni.n2;
  // along W voxel x takes 3 parts of node x / 2 and one of the node on its side; the product is
  // rounded before the sum for even voxels (lower) and in it for odd ones (upper): fma(ca, cb P, Q)
  const bool odd = x & 1;
  const int mx = x >> 1, mq = odd ? min(mx + 1, nf.n2 - 1) : max(mx - 1, 0);
  const float ca = odd ? 3.f : 1.f, cb = odd ? 1.f : 3.f;
  const int r0 = max(my - 1, 0) * nf.n2, r1 = my * nf.n2, r2 = min(my + 1, nf.n1 - 1) * nf.n2;
  auto along_w = [&](const float4* row) {
    const float4 P = __ldg(row + mx), Q = __ldg(row + mq);
    return make_float3(__fmaf_rn(ca, __fmul_rn(cb, P.x), Q.x), __fmaf_rn(ca, __fmul_rn(cb, P.y), Q.y),
                       __fmaf_rn(ca, __fmul_rn(cb, P.z), Q.z));
  };
  // the W and H passes of one node plane: s[dy] for the two rows of this thread
  auto node_plane = [&](int mz, float3 (&s)[2]) {
    const float4* U = d.U + (size_t)mz * fp;
    const float3 a = along_w(U + r0), b = along_w(U + r1), c = along_w(U + r2);
    s[0] = lower(a, b);
    s[1] = upper(b, c);
  };
  const float* t = RIGID ? rig + 12 * d.fi : nullptr;
  const float px = (float)x;
  const bool two = 2 * my + 1 < ni.n1;
  float* out = W + (size_t)pair * stride + (size_t)(2 * m0) * plane + (2 * my) * ni.n2 + x;
  float* go = GRAD ? gI + (size_t)pair * 3 * stride + (size_t)(2 * m0) * plane + (2 * my) * ni.n2 + x : nullptr;
  // the two voxels of image plane z, whose displacements, scaled by 32, are u
  auto emit = [&](int z, const float3 (&u)[2]) {
    const float pz = (float)z;
#pragma unroll
    for (int dy = 0; dy < 2; ++dy) {
      const float py = (float)(2 * my + dy);
      float qz, qy, qx;
      if (RIGID) {  // Sec. Rigid Registration: the rigid displacement A p + b of the fixed session's grid
        qz = pz + fmaf(u[dy].x, 0.03125f, fmaf(t[0], pz, fmaf(t[1], py, fmaf(t[2], px, t[9]))));
        qy = py + fmaf(u[dy].y, 0.03125f, fmaf(t[3], pz, fmaf(t[4], py, fmaf(t[5], px, t[10]))));
        qx = px + fmaf(u[dy].z, 0.03125f, fmaf(t[6], pz, fmaf(t[7], py, fmaf(t[8], px, t[11]))));
      } else {
        qz = fmaf(u[dy].x, 0.03125f, pz), qy = fmaf(u[dy].y, 0.03125f, py), qx = fmaf(u[dy].z, 0.03125f, px);
      }
      float3 g;
      const float w = cell_sample<GRAD>(I, qz, qy, qx, g);
      if (dy == 0 || two) {
        const int v = dy * ni.n2;
        __stcs(out + v, w);
        if (GRAD) {
          __stcs(go + v, g.x);
          __stcs(go + stride + v, g.y);
          __stcs(go + 2 * stride + v, g.z);
        }
      }
    }
    out += plane;
    if (GRAD) go += plane;
  };
  float3 s0[2], s1[2], s2[2], u[2];
  node_plane(max(m0 - 1, 0), s0);
  node_plane(m0, s1);
  const int m1 = min(m0 + nz, nf.n0);
  for (int mz = m0; mz < m1; ++mz) {
    node_plane(min(mz + 1, nf.n0 - 1), s2);
    // along D, and the factor 2 from flow to image voxel units: u is 32 times the displacement
    u[0] = lower(s0[0], s1[0]), u[1] = lower(s0[1], s1[1]);
    emit(2 * mz, u);
    if (2 * mz + 1 >= ni.n0) break;
    u[0] = upper(s1[0], s2[0]), u[1] = upper(s1[1], s2[1]);
    emit(2 * mz + 1, u);
#pragma unroll
    for (int dy = 0; dy < 2; ++dy) s0[dy] = s1[dy], s1[dy] = s2[dy];
  }
}

// racc += sums of dL/dq and dL/dq p^T over the block of node (mz, my, mx), g = 2 dL/dq: with p = 2 m + d
// the products reduce to 2 m sum g + sum over d_a = 1 of g, per axis a
template <int NR>
__device__ __forceinline__ void rigid_sums(const float3 (&g)[2][2][2], int mz, int my, int mx, float (&racc)[NR]) {
  if constexpr (NR == 12) {
    const float m2[3] = {(float)(2 * mz), (float)(2 * my), (float)(2 * mx)};
    auto add = [](float3 a, float3 b) { return make_float3(a.x + b.x, a.y + b.y, a.z + b.z); };
    const float3 z0y0 = add(g[0][0][0], g[0][0][1]), z0y1 = add(g[0][1][0], g[0][1][1]);
    const float3 z1y0 = add(g[1][0][0], g[1][0][1]), z1y1 = add(g[1][1][0], g[1][1][1]);
    const float3 hi[3] = {add(z1y0, z1y1), add(z0y1, z1y1),
                          add(add(g[0][0][1], g[0][1][1]), add(g[1][0][1], g[1][1][1]))};
    const float3 all = add(add(z0y0, z0y1), hi[0]);
    const float s[3] = {0.5f * all.x, 0.5f * all.y, 0.5f * all.z};
#pragma unroll
    for (int q = 0; q < 3; ++q) racc[q] += s[q];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      racc[3 + a] += fmaf(m2[a], s[0], 0.5f * hi[a].x);
      racc[6 + a] += fmaf(m2[a], s[1], 0.5f * hi[a].y);
      racc[9 + a] += fmaf(m2[a], s[2], 0.5f * hi[a].z);
    }
  }
}

// ---- adjoint: g(p) = 2 dL/dW(p) grad S[I_k](p + U~(p)) at every image voxel (the image
// gradient at the sample point was stored by the forward warp), then
// dL/dU(node) = sum over the image voxels of the node's stencil with the same
// 0.25 / 0.75 weights (contributions to clamped node indices fold onto the edge node).
template <bool RIGID>
__global__ void __launch_bounds__(RX* RY) k_warp_bwd2(const PairDesc* __restrict__ pd, const float* __restrict__ dLdWb,
                                                      const float* __restrict__ gIb, size_t stride, Dims ni, Dims nf,
                                                      int fz, int nzc, float* __restrict__ rpart,
                                                      unsigned* __restrict__ gmax) {
  grid_begin();
  __shared__ float sh[RY][RX][12];
  float gm = 0.f;  // largest |component| of the nodes this thread writes
  // with rpart: sums of dL/dq and dL/dq p^T over the image voxels of the nodes this CTA
  // writes (the rigid gradient, Sec. Rigid Registration), 12 per CTA
  float racc[RIGID ? 12 : 1];
#pragma unroll
  for (int k = 0; k < (RIGID ? 12 : 1); ++k) racc[k] = 0.f;
  const int pair = blockIdx.z / nzc, zc = blockIdx.z - pair * nzc;
  const PairDesc d = pd[pair];
  const float* __restrict__ dW = dLdWb + (size_t)pair * stride;
  const float* __restrict__ gI = gIb + (size_t)pair * 3 * stride;
  const int lane = threadIdx.x, ty = threadIdx.y;
  const int mx = blockIdx.x * OX - 1 + lane, my = blockIdx.y * OY - 1 + ty;
  const bool active = mx >= 0 && mx < nf.n2 && my >= 0 && my < nf.n1;
  const bool writer = lane >= 1 && lane <= OX && ty >= 1 && ty <= OY && active;
  const int Z0 = zc * fz, Z1 = min(Z0 + fz, nf.n0);
  // even widths with 8-byte aligned inputs: the two voxels of a W pair start on an
  // 8-byte boundary in every row, pair and plane
  const bool pair_load = (ni.n2 & 1) == 0 && (reinterpret_cast<uintptr_t>(dW) & 7) == 0 &&
                         (reinterpret_cast<uintptr_t>(gI) & 7) == 0 && (stride & 1) == 0;
  float3 pend = make_float3(0.f, 0.f, 0.f), carry = pend;
  for (int mz = max(Z0 - 1, 0); mz <= min(Z1, nf.n0 - 1); ++mz) {
    // per-voxel gradient of the 8 image voxels of block (mz, my, mx)
    float3 g[2][2][2];
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int c = 0; c < 2; ++c) g[a][b][c] = make_float3(0.f, 0.f, 0.f);
    if (active && pair_load) {
      // the two voxels of a W pair with 8-byte loads
#pragma unroll
      for (int dz = 0; dz < 2; ++dz)
#pragma unroll
        for (int dy = 0; dy < 2; ++dy) {
          const int z = 2 * mz + dz, y = 2 * my + dy;
          if (z < ni.n0 && y < ni.n1) {
            const int o = (z * ni.n1 + y) * ni.n2 + 2 * mx;
            const float2 s = *reinterpret_cast<const float2*>(dW + o);
            const float2 a = *reinterpret_cast<const float2*>(gI + o);
            const float2 b = *reinterpret_cast<const float2*>(gI + stride + o);
            const float2 c = *reinterpret_cast<const float2*>(gI + 2 * stride + o);
            g[dz][dy][0] = make_float3(2.f * s.x * a.x, 2.f * s.x * b.x, 2.f * s.x * c.x);
            g[dz][dy][1] = make_float3(2.f * s.y * a.y, 2.f * s.y * b.y, 2.f * s.y * c.y);
          }
        }
    } else if (active) {
#pragma unroll
      for (int dz = 0; dz < 2; ++dz)
#pragma unroll
        for (int dy = 0; dy < 2; ++dy)
#pragma unroll
          for (int dx = 0; dx < 2; ++dx) {
            const int z = 2 * mz + dz, y = 2 * my + dy, x = 2 * mx + dx;
            if (z < ni.n0 && y < ni.n1 && x < ni.n2) {
              const int o = (z * ni.n1 + y) * ni.n2 + x;
              const float s = 2.f * dW[o];
              g[dz][dy][dx] = make_float3(s * gI[o], s * gI[stride + o], s * gI[2 * stride + o]);
            }
          }
    }
    if (RIGID && writer && mz >= Z0 && mz < Z1) {
      // g holds 2 dL/dq (the 2 of the flow-to-image scale); image voxels outside the
      // grid were left at 0
      rigid_sums(g, mz, my, mx, racc);
    }
    // transpose along W: node mx gets 0.75 (g0 + g1) of its block, 0.25 g1 of block mx-1
    // and 0.25 g0 of block mx+1 (neighbouring lanes); edge nodes keep their folded share
    float hx[2][2][3];
#pragma unroll
    for (int dz = 0; dz < 2; ++dz)
#pragma unroll
      for (int dy = 0; dy < 2; ++dy) {
        const float3 g0 = g[dz][dy][0], g1 = g[dz][dy][1];
        const float e0 = (mx == 0) ? 0.25f : 0.f, e1 = (mx == nf.n2 - 1) ? 0.25f : 0.f;
        const float a0[3] = {g0.x, g0.y, g0.z}, a1[3] = {g1.x, g1.y, g1.z};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const float left = __shfl_up_sync(0xffffffffu, a1[c], 1);
          const float right = __shfl_down_sync(0xffffffffu, a0[c], 1);
          hx[dz][dy][c] = 0.75f * (a0[c] + a1[c]) + 0.25f * (left + right) + e0 * a0[c] + e1 * a1[c];
        }
      }
#pragma unroll
    for (int dz = 0; dz < 2; ++dz)
#pragma unroll
      for (int dy = 0; dy < 2; ++dy)
#pragma unroll
        for (int c = 0; c < 3; ++c) sh[ty][lane][(dz * 2 + dy) * 3 + c] = hx[dz][dy][c];
    __syncthreads();
    // transpose along H (neighbouring rows in shared memory)
    float k[2][3];
    {
      const int up = max(ty - 1, 0), dn = min(ty + 1, RY - 1);
      const float e0 = (my == 0) ? 0.25f : 0.f, e1 = (my == nf.n1 - 1) ? 0.25f : 0.f;
#pragma unroll
      for (int dz = 0; dz < 2; ++dz)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const float h0 = hx[dz][0][c], h1 = hx[dz][1][c];
          const float l = ty > 0 ? sh[up][lane][(dz * 2 + 1) * 3 + c] : 0.f;
          const float r = ty < RY - 1 ? sh[dn][lane][(dz * 2 + 0) * 3 + c] : 0.f;
          k[dz][c] = 0.75f * (h0 + h1) + 0.25f * (l + r) + e0 * h0 + e1 * h1;
        }
    }
    __syncthreads();
    // transpose along D, streaming: node mz-1 is complete once block mz added its 0.25 k0
    const float3 k0 = make_float3(k[0][0], k[0][1], k[0][2]), k1 = make_float3(k[1][0], k[1][1], k[1][2]);
    if (mz - 1 >= Z0 && mz - 1 < Z1 && writer)
    {
      const float4 gv = make_float4(pend.x + 0.25f * k0.x, pend.y + 0.25f * k0.y, pend.z + 0.25f * k0.z, 0.f);
      d.G[((mz - 1) * nf.n1 + my) * nf.n2 + mx] = gv;
      gm = fmaxf(gm, fmaxf(fabsf(gv.x), fmaxf(fabsf(gv.y), fabsf(gv.z))));
    }
    const float e0 = (mz == 0) ? 0.25f : 0.f, e1 = (mz == nf.n0 - 1) ? 0.25f : 0.f;
    pend.x = 0.75f * (k0.x + k1.x) + carry.x + e0 * k0.x + e1 * k1.x;
    pend.y = 0.75f * (k0.y + k1.y) + carry.y + e0 * k0.y + e1 * k1.y;
    pend.z = 0.75f * (k0.z + k1.z) + carry.z + e0 * k0.z + e1 * k1.z;
    carry = make_float3(0.25f * k1.x, 0.25f * k1.y, 0.25f * k1.z);
  }
  // the last node of the volume has no block after it
  if (Z1 == nf.n0 && writer) {
    d.G[((nf.n0 - 1) * nf.n1 + my) * nf.n2 + mx] = make_float4(pend.x, pend.y, pend.z, 0.f);
    gm = fmaxf(gm, fmaxf(fabsf(pend.x), fmaxf(fabsf(pend.y), fabsf(pend.z))));
  }
  if (gmax) {  // the scale of the deterministic adjoint's fixed-point sums
    const unsigned b = __reduce_max_sync(0xffffffffu, __float_as_uint(gm));
    if ((threadIdx.x & 31) == 0 && b) atomicMax(gmax, b);
  }
  if (RIGID) {
    // CTA sums in a fixed order: warp shuffles, then the warps in order (through sh)
    __syncthreads();
    float* red = &sh[0][0][0];
    const int tid = ty * RX + lane, w = tid >> 5;
#pragma unroll
    for (int k = 0; k < (RIGID ? 12 : 1); ++k) {
      float v = racc[k];
      for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
      if (lane == 0) red[w * 12 + k] = v;
    }
    __syncthreads();
    if (tid < 12) {
      float t = 0.f;
      for (int i = 0; i < RX * RY / 32; ++i) t += red[i * 12 + tid];
      const int per_pair = gridDim.x * gridDim.y * nzc;
      const int cta = (zc * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
      rpart[((size_t)pair * per_pair + cta) * 12 + tid] = t;
    }
  }
}

// ---- the same adjoint with its inputs staged by the tensor memory accelerator. Per flow
// plane mz one thread copies the 2 image planes 2mz, 2mz+1 of the CTA's region (16 rows,
// 68 columns from a 16-byte aligned start: the 64 columns of the 32 node columns and 4 of
// alignment) of dL/dW and of each component of grad I_k into one of two stages; the copy
// of plane mz+2 is issued once every thread has read plane mz. Voxels outside the image
// arrive as zeros, as the plain loads of k_warp_bwd2 leave them. A wait that runs out sets
// *err and the CTA carries on without waiting (its results are reported as invalid).
constexpr int SXW = 2 * RX + 4, SYH = 2 * RY, SZD = 2;  // staged box: columns, rows, planes
constexpr int SARR = SZD * SYH * SXW;                    // floats of one array in one stage

template <bool RIGID>
__global__ void __launch_bounds__(RX* RY) k_warp_bwd3t(const __grid_constant__ WarpBwdMaps maps,
                                                       const PairDesc* __restrict__ pd, Dims ni, Dims nf, int fz,
                                                       int nzc, float* __restrict__ rpart, int* __restrict__ err,
                                                       unsigned* __restrict__ gmax) {
  grid_begin();
  float gm = 0.f;  // largest |component| of the nodes this thread writes
  __shared__ __align__(8) uint64_t bar[2];
  extern __shared__ __align__(128) float smem_raw[];
  float* stage = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
  // the H transpose's exchange buffer [RY][RX][12] lives in the stage just read (its next
  // copy is issued once the exchange is done), which leaves room for 3 CTAs per SM
  typedef float ShRow[RX][12];
  static_assert(RY * RX * 12 <= 4 * SARR, "exchange buffer larger than a stage");
  float racc[RIGID ? 12 : 1];
#pragma unroll
  for (int k = 0; k < (RIGID ? 12 : 1); ++k) racc[k] = 0.f;
  const int pair = blockIdx.z / nzc, zc = blockIdx.z - pair * nzc;
  const PairDesc d = pd[pair];
  const int lane = threadIdx.x, ty = threadIdx.y, tid = ty * RX + lane;
  const int mx = blockIdx.x * OX - 1 + lane, my = blockIdx.y * OY - 1 + ty;
  const bool writer = lane >= 1 && lane <= OX && ty >= 1 && ty <= OY && mx >= 0 && mx < nf.n2 && my >= 0 &&
                      my < nf.n1;
  const int Z0 = zc * fz, Z1 = min(Z0 + fz, nf.n0);
  const int m0 = max(Z0 - 1, 0), m1 = min(Z1, nf.n0 - 1), niter = m1 - m0 + 1;
  const int xs = 2 * (blockIdx.x * OX - 1) - 2, ys = 2 * (blockIdx.y * OY - 1);  // xs: multiple of 4
  if (tid == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    mbar_fence_init();
  }
  __syncthreads();
  auto issue = [&](int k) {  // one thread: flow plane m0 + k into stage k & 1
    const int st = k & 1, zs = 2 * (m0 + k);
    float* dst = stage + st * 4 * SARR;
    mbar_expect_tx(&bar[st], 4u * SARR * 4u);
    tma_load4(dst, &maps.dW, xs, ys, zs, pair, &bar[st]);
#pragma unroll
    for (int c = 0; c < 3; ++c) tma_load4(dst + (1 + c) * SARR, &maps.gI, xs, ys, zs, 3 * pair + c, &bar[st]);
  };
  if (tid == 0) {
    issue(0);
    if (niter > 1) issue(1);
  }
  float3 pend = make_float3(0.f, 0.f, 0.f), carry = pend;
  bool ok = true;
  for (int k = 0; k < niter; ++k) {
    const int mz = m0 + k, st = k & 1;
    ok = ok && mbar_wait(&bar[st], (unsigned)(k >> 1) & 1u);  // after a failure, stop waiting
    const float* sd = stage + st * 4 * SARR;
    ShRow* sh = reinterpret_cast<ShRow*>(stage + st * 4 * SARR);
    // per-voxel gradient of the 8 image voxels of block (mz, my, mx)
    float3 g[2][2][2];
#pragma unroll
    for (int dz = 0; dz < 2; ++dz)
#pragma unroll
      for (int dy = 0; dy < 2; ++dy) {
        const int o = (dz * SYH + 2 * ty + dy) * SXW + 2 + 2 * lane;
        const float2 sv = *reinterpret_cast<const float2*>(sd + o);
        const float2 a = *reinterpret_cast<const float2*>(sd + SARR + o);
        const float2 b = *reinterpret_cast<const float2*>(sd + 2 * SARR + o);
        const float2 c = *reinterpret_cast<const float2*>(sd + 3 * SARR + o);
        g[dz][dy][0] = make_float3(2.f * sv.x * a.x, 2.f * sv.x * b.x, 2.f * sv.x * c.x);
        g[dz][dy][1] = make_float3(2.f * sv.y * a.y, 2.f * sv.y * b.y, 2.f * sv.y * c.y);
      }
    if (RIGID && writer && mz >= Z0 && mz < Z1) {
      // g holds 2 dL/dq (the 2 of the flow-to-image scale); image voxels outside the
      // grid arrived as 0
      rigid_sums(g, mz, my, mx, racc);
    }
    // transpose along W (neighbouring lanes), as in k_warp_bwd2
    float hx[2][2][3];
#pragma unroll
    for (int dz = 0; dz < 2; ++dz)
#pragma unroll
      for (int dy = 0; dy < 2; ++dy) {
        const float3 g0 = g[dz][dy][0], g1 = g[dz][dy][1];
        const float e0 = (mx == 0) ? 0.25f : 0.f, e1 = (mx == nf.n2 - 1) ? 0.25f : 0.f;
        const float a0[3] = {g0.x, g0.y, g0.z}, a1[3] = {g1.x, g1.y, g1.z};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const float left = __shfl_up_sync(0xffffffffu, a1[c], 1);
          const float right = __shfl_down_sync(0xffffffffu, a0[c], 1);
          hx[dz][dy][c] = 0.75f * (a0[c] + a1[c]) + 0.25f * (left + right) + e0 * a0[c] + e1 * a1[c];
        }
      }
    __syncthreads();  // every thread is past its reads of stage st, which now takes the exchange
#pragma unroll
    for (int dz = 0; dz < 2; ++dz)
#pragma unroll
      for (int dy = 0; dy < 2; ++dy)
#pragma unroll
        for (int c = 0; c < 3; ++c) sh[ty][lane][(dz * 2 + dy) * 3 + c] = hx[dz][dy][c];
    __syncthreads();
    // transpose along H (neighbouring rows in shared memory)
    float kk[2][3];
    {
      const int up = max(ty - 1, 0), dn = min(ty + 1, RY - 1);
      const float e0 = (my == 0) ? 0.25f : 0.f, e1 = (my == nf.n1 - 1) ? 0.25f : 0.f;
#pragma unroll
      for (int dz = 0; dz < 2; ++dz)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const float h0 = hx[dz][0][c], h1 = hx[dz][1][c];
          const float l = ty > 0 ? sh[up][lane][(dz * 2 + 1) * 3 + c] : 0.f;
          const float r = ty < RY - 1 ? sh[dn][lane][(dz * 2 + 0) * 3 + c] : 0.f;
          kk[dz][c] = 0.75f * (h0 + h1) + 0.25f * (l + r) + e0 * h0 + e1 * h1;
        }
    }
    // the exchange is read: refill stage st with plane k + 2 (every thread orders its generic
    // accesses of the stage before the copy engine's writes)
    fence_proxy_async();
    __syncthreads();
    if (tid == 0 && k + 2 < niter) issue(k + 2);
    // transpose along D, streaming: node mz-1 is complete once block mz added its 0.25 k0
    const float3 k0 = make_float3(kk[0][0], kk[0][1], kk[0][2]), k1 = make_float3(kk[1][0], kk[1][1], kk[1][2]);
    if (mz - 1 >= Z0 && mz - 1 < Z1 && writer)
    {
      const float4 gv = make_float4(pend.x + 0.25f * k0.x, pend.y + 0.25f * k0.y, pend.z + 0.25f * k0.z, 0.f);
      d.G[((mz - 1) * nf.n1 + my) * nf.n2 + mx] = gv;
      gm = fmaxf(gm, fmaxf(fabsf(gv.x), fmaxf(fabsf(gv.y), fabsf(gv.z))));
    }
    const float e0 = (mz == 0) ? 0.25f : 0.f, e1 = (mz == nf.n0 - 1) ? 0.25f : 0.f;
    pend.x = 0.75f * (k0.x + k1.x) + carry.x + e0 * k0.x + e1 * k1.x;
    pend.y = 0.75f * (k0.y + k1.y) + carry.y + e0 * k0.y + e1 * k1.y;
    pend.z = 0.75f * (k0.z + k1.z) + carry.z + e0 * k0.z + e1 * k1.z;
    carry = make_float3(0.25f * k1.x, 0.25f * k1.y, 0.25f * k1.z);
  }
  if (Z1 == nf.n0 && writer) {
    d.G[((nf.n0 - 1) * nf.n1 + my) * nf.n2 + mx] = make_float4(pend.x, pend.y, pend.z, 0.f);
    gm = fmaxf(gm, fmaxf(fabsf(pend.x), fmaxf(fabsf(pend.y), fabsf(pend.z))));
  }
  if (gmax) {  // the scale of the deterministic adjoint's fixed-point sums
    const unsigned b = __reduce_max_sync(0xffffffffu, __float_as_uint(gm));
    if ((threadIdx.x & 31) == 0 && b) atomicMax(gmax, b);
  }
  if (!ok) {
    // report, then give the copies still in flight into this CTA's stages one more bounded
    // wait (the last use of each stage) before the CTA's shared memory is released
    if (err) atomicOr(err, 1);
    for (int st = 0; st < 2 && st < niter; ++st) {
      const int last = niter - 1 - ((niter - 1 - st) & 1);
      mbar_wait(&bar[st], (unsigned)(last >> 1) & 1u);
    }
  }
  if (RIGID) {
    __syncthreads();
    float* red = stage;  // every copy into the stages has been waited for
    const int w = tid >> 5;
#pragma unroll
    for (int k = 0; k < (RIGID ? 12 : 1); ++k) {
      float v = racc[k];
      for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
      if (lane == 0) red[w * 12 + k] = v;
    }
    __syncthreads();
    if (tid < 12) {
      float t = 0.f;
      for (int i = 0; i < RX * RY / 32; ++i) t += red[i * 12 + tid];
      const int per_pair = gridDim.x * gridDim.y * nzc;
      const int cta = (zc * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
      rpart[((size_t)pair * per_pair + cta) * 12 + tid] = t;
    }
  }
}
constexpr size_t kWarpBwd3tBytes = 128 + sizeof(float) * 2 * 4 * SARR;

// flow planes per D chunk of the adjoint: every chunk streams two planes more than it
// writes, so chunks are split only until a launch of `batch` pairs has about four waves of
// four CTAs on each of 152 SMs (2432 CTAs), and halved only while above 2 planes
// (6 pairs of 48^3: 7.5 us at 2 planes, 8.5 at 3)
int chunk_nodes(int ntiles, int depth, int batch) {
  int fz = depth;
  while (fz > 2 && (long)batch * ntiles * ((depth + fz - 1) / fz) < 2432) fz = (fz + 1) / 2;
  return fz < 1 ? 1 : fz;
}
}  // namespace

// node planes a thread of the forward walks: every walk loads two planes more than it emits, so it
// is as long as leaves the launch about four waves of four CTAs on every SM, 32 planes at most
// (90 pairs of 160 x 192 x 160: 2286 us at 8 planes, 2211 at 16, 2170 at 32). Walks of one plane only
// where they fit one wave (6 pairs of 48^3, 1.4 waves of them: 7.2 us at 1, 6.2 at 2 and 3, 7.2 at 4)
static int warp_planes(long tiles, int depth) {
  const int least = tiles * depth <= (long)kWarpCtas * device_sm_count() ? 1 : 2;
  int nz = 32;
  while (nz > least && tiles * ((depth + nz - 1) / nz) < 16L * device_sm_count()) nz /= 2;
  return nz;
}
void launch_warp(const PairDesc* pd, int n_pairs, bool cells, Dims ni, Dims nf, float* W, float* gI, size_t Wstride,
                 const float* rigid, cudaStream_t s) {
  const int gx = (ni.n2 + BX - 1) / BX, gy = (nf.n1 + BY - 1) / BY;
  const int nz = warp_planes((long)gx * gy * n_pairs, nf.n0);
  const unsigned grid = (unsigned)gx * gy * ((nf.n0 + nz - 1) / nz) * n_pairs;
  auto go = [&](auto kernel) {
    launch(kernel, grid, dim3(BX, BY), 0, s, false)(pd, n_pairs, ni, nf, nz, W, gI, Wstride, rigid);
  };
  if (cells) {
    if (gI)
      rigid ? go(k_warp<true, true, true>) : go(k_warp<true, false, true>);
    else
      rigid ? go(k_warp<false, true, true>) : go(k_warp<false, false, true>);
  } else {
    if (gI)
      rigid ? go(k_warp<true, true, false>) : go(k_warp<true, false, false>);
    else
      rigid ? go(k_warp<false, true, false>) : go(k_warp<false, false, false>);
  }
}

size_t image_cells(Dims n) { return vox(Dims{n.n0 + 2, n.n1 + 2, n.n2 + 1}); }
void launch_image_cells(const float* in, int n_images, Dims n, float2* out, int* bad, cudaStream_t s) {
  const unsigned rows = (unsigned)(n.n0 + 2) * (n.n1 + 2);
  launch(k_image_cells, dim3((rows + kCellRows - 1) / kCellRows, n_images), dim3(32, kCellRows), 0, s)(in, n, out, bad);
}

int warp_bwd_ctas_per_pair(Dims nf, int batch) {
  const int gx = (nf.n2 + OX - 1) / OX, gy = (nf.n1 + OY - 1) / OY;
  const int fz = chunk_nodes(gx * gy, nf.n0, batch);
  return gx * gy * ((nf.n0 + fz - 1) / fz);
}
int warp_bwd_zchunks(Dims nf, int batch) {
  const int gx = (nf.n2 + OX - 1) / OX, gy = (nf.n1 + OY - 1) / OY;
  const int fz = chunk_nodes(gx * gy, nf.n0, batch);
  return (nf.n0 + fz - 1) / fz;
}

void make_warp_bwd_maps(WarpBwdMaps* m, const float* dLdW, const float* gI, int batch, Dims ni) {
  memset(m, 0, sizeof(*m));
  m->ok = encode_volumes(&m->dW, dLdW, ni, batch, SXW, SYH, SZD) &&
          encode_volumes(&m->gI, gI, ni, 3 * batch, SXW, SYH, SZD);
}

cudaError_t prepare_warp_kernels() {
  static std::mutex mu;
  static bool done[kMaxDevices] = {};
  return once_per_device(done, mu, [] {
    const cudaError_t a =
        cudaFuncSetAttribute(k_warp_bwd3t<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWarpBwd3tBytes);
    const cudaError_t b =
        cudaFuncSetAttribute(k_warp_bwd3t<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWarpBwd3tBytes);
    return a != cudaSuccess ? a : b;
  });
}

void launch_warp_bwd(const PairDesc* pd, int n_pairs, int batch, const float* dLdW, const float* gI, size_t stride,
                     Dims ni, Dims nf, float* rigid_part, const WarpBwdMaps* maps, int* err, unsigned* gmax,
                     cudaStream_t s) {
  const int gx = (nf.n2 + OX - 1) / OX, gy = (nf.n1 + OY - 1) / OY;
  const int fz = chunk_nodes(gx * gy, nf.n0, batch);
  const int nzc = (nf.n0 + fz - 1) / fz;
  const dim3 g(gx, gy, nzc * n_pairs), b(RX, RY);
  if (maps && maps->ok && stride == vox(ni)) {
    if (rigid_part)
      launch(k_warp_bwd3t<true>, g, b, kWarpBwd3tBytes, s)(*maps, pd, ni, nf, fz, nzc, rigid_part, err, gmax);
    else
      launch(k_warp_bwd3t<false>, g, b, kWarpBwd3tBytes, s)(*maps, pd, ni, nf, fz, nzc, nullptr, err, gmax);
    return;
  }
  if (rigid_part)
    launch(k_warp_bwd2<true>, g, b, 0, s)(pd, dLdW, gI, stride, ni, nf, fz, nzc, rigid_part, gmax);
  else
    launch(k_warp_bwd2<false>, g, b, 0, s)(pd, dLdW, gI, stride, ni, nf, fz, nzc, nullptr, gmax);
}

}  // namespace muster
