// metrics_kernels.cu -- determinant maps of the spatial Jacobian of x -> x + u(x) (the maps
// of Sec. Sensitivity to clinical outcomes, Fig. 1c) and the deformation metrics of Sec.
// Evaluation Metrics: mean Euclidean distance Eu, vector Pearson correlation PCC of the
// centred fields and the slope B = trace(A)/3 of the least-squares fit u_est = A u_true + b.
//
// The determinant uses central differences, one-sided on the first and last plane of an
// axis and 0 along an axis of one plane. The metrics take two passes over the fields
// (means, then centred second moments) and a final single-CTA kernel that adds the partial
// sums in a fixed order and solves the 3x3 normal equations: the results are the same on
// every run. GB300 runs FP64 arithmetic far slower than FP32, so the per-voxel terms and each thread's
// running sums are double-float values (an unevaluated sum hi + lo of two floats, about 48
// significant bits) built from error-free transformations: Knuth's TwoSum for sums and the
// FMA form of Dekker's product (Ogita, Rump and Oishi, "Accurate sum and dot product", 2005)
// for products. The sums over a CTA's threads carry three floats, then FP64; the final sums are FP64.
#include <algorithm>

#include "kernels.h"

namespace muster {

namespace {
constexpr int kJT = 256;                 // Jacobian: threads per CTA
// metrics: threads per CTA, and the most CTAs of the grid-stride passes (3 per SM of the
// device; kMCtas bounds the scratch of the per-CTA partial sums)
constexpr int kMT = 256, kMCtas = 3 * 256, kMCtasPerSM = 3;
constexpr int kP1 = 8, kP2 = 16;         // partial sums per CTA of pass 1 and pass 2

// one derivative from the values below (lo) and above (hi) index p of an axis of m planes:
// central inside, one-sided on the first and last plane, 0 on an axis of one plane
__device__ __forceinline__ float dstep(float lo, float mid, float hi, int p, int m) {
  if (m == 1) return 0.f;
  if (p == 0) return hi - mid;
  if (p == m - 1) return mid - lo;
  return 0.5f * (hi - lo);
}

// A thread owns NX neighbouring voxels of each of NY rows and walks a chunk of D with the planes z-1, z,
// z+1 of the three components in registers: 4 or 2 of one row with 16- or 8-byte loads where the width is
// a multiple and the fields are aligned, else one of two rows, which read the row between them once. The
// rows beside the run are loads that hit the L1 or L2 lines of the neighbouring threads' own rows; x-1 and
// x+NX come from the neighbouring lanes, or from memory at a row's or warp's end. DRAM is the floor (16 bytes
// per voxel, 12 us at 160 x 192 x 160); the latency of a plane's loads bounds it, so 3 or 4 CTAs share an SM and
// the walk is short. 160 x 192 x 160: 28 us with runs of 4 (36 us with 2 CTAs per SM, 29 us with runs of 2), 160 x
// 192 x 161 41 us (46 us with one voxel of one or four rows); staging every plane of a 32 x 8 tile in shared
// memory behind two barriers took 41 and 47 us.
template <int NX>
struct Run {
  float v[NX];
};
template <int NX>
__device__ __forceinline__ Run<NX> load_run(const float* __restrict__ p) {
  Run<NX> r;
  if constexpr (NX == 4) {
    const float4 t = __ldg(reinterpret_cast<const float4*>(p));
    r.v[0] = t.x, r.v[1] = t.y, r.v[2] = t.z, r.v[3] = t.w;
  } else if constexpr (NX == 2) {
    const float2 t = __ldg(reinterpret_cast<const float2*>(p));
    r.v[0] = t.x, r.v[1] = t.y;
  } else {
    r.v[0] = __ldg(p);
  }
  return r;
}
template <int NX, int NY>
__global__ void __launch_bounds__(kJT, NX == 4 ? 3 : 4) k_jacobian_det(const float* __restrict__ u, Dims n,
                                                                       float* __restrict__ J, int zchunk) {
  grid_begin();
  const int runs = n.n2 / NX, i = blockIdx.x * kJT + threadIdx.x, lane = threadIdx.x & 31;
  const bool in = i < runs * ((n.n1 + NY - 1) / NY);
  const int y = in ? i / runs * NY : 0, x = in ? i % runs * NX : 0;
  const int z0 = blockIdx.y * zchunk, z1 = min(z0 + zchunk, n.n0);
  const size_t V = vox(n);
  const ptrdiff_t plane = (ptrdiff_t)n.n1 * n.n2;
  int row[NY];  // rows of the run from its first one, the volume's last row repeated
#pragma unroll
  for (int r = 0; r < NY; ++r) row[r] = min(r, n.n1 - 1 - y) * n.n2;
  const int below = y > 0 ? -n.n2 : 0, above = min(NY, n.n1 - 1 - y) * n.n2;
  const bool left = x > 0, right = x + NX < n.n2;  // x-1 and x+NX exist
  const float* f = u + (size_t)y * n.n2 + x + z0 * plane;
  Run<NX> prv[3][NY], cur[3][NY], nxt[3][NY];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int r = 0; r < NY; ++r) {
      cur[c][r] = load_run<NX>(f + c * V + row[r]);
      prv[c][r] = z0 > 0 ? load_run<NX>(f + c * V + row[r] - plane) : cur[c][r];
    }
  for (int z = z0; z < z1; ++z, f += plane) {
    Run<NX> lo[3], hi[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
#pragma unroll
      for (int r = 0; r < NY; ++r) nxt[c][r] = z + 1 < n.n0 ? load_run<NX>(f + c * V + row[r] + plane) : cur[c][r];
      lo[c] = load_run<NX>(f + c * V + below);
      hi[c] = load_run<NX>(f + c * V + above);
    }
#pragma unroll
    for (int r = 0; r < NY; ++r) {
      float M[NX][3][3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const Run<NX>& me = cur[c][r];
        // the voxels beside the run: a run of the same row in the next lane, else memory
        float l = __shfl_up_sync(0xffffffffu, me.v[NX - 1], 1), g = __shfl_down_sync(0xffffffffu, me.v[0], 1);
        if (lane == 0 && left) l = __ldg(f + c * V + row[r] - 1);
        if (lane == 31 && right) g = __ldg(f + c * V + row[r] + NX);
#pragma unroll
        for (int k = 0; k < NX; ++k) {
          const float mid = me.v[k];
          M[k][c][0] = (c == 0 ? 1.f : 0.f) + dstep(prv[c][r].v[k], mid, nxt[c][r].v[k], z, n.n0);
          M[k][c][1] = (c == 1 ? 1.f : 0.f) + dstep(r > 0 ? cur[c][r > 0 ? r - 1 : 0].v[k] : lo[c].v[k], mid,
                                                    r < NY - 1 ? cur[c][r < NY - 1 ? r + 1 : r].v[k] : hi[c].v[k], y + r, n.n1);
          M[k][c][2] = (c == 2 ? 1.f : 0.f) + dstep(k > 0 ? me.v[k > 0 ? k - 1 : 0] : l, mid,
                                                    k < NX - 1 ? me.v[k < NX - 1 ? k + 1 : k] : g, x + k, n.n2);
        }
      }
      float det[NX];
#pragma unroll
      for (int k = 0; k < NX; ++k) {
        const float(*A)[3] = M[k];
        det[k] = A[0][0] * (A[1][1] * A[2][2] - A[1][2] * A[2][1]) - A[0][1] * (A[1][0] * A[2][2] - A[1][2] * A[2][0]) +
                 A[0][2] * (A[1][0] * A[2][1] - A[1][1] * A[2][0]);
      }
      if (in && y + r < n.n1) {
        float* o = J + (size_t)z * plane + (size_t)y * n.n2 + row[r] + x;
        if constexpr (NX == 4)
          *reinterpret_cast<float4*>(o) = make_float4(det[0], det[1], det[2], det[3]);
        else if constexpr (NX == 2)
          *reinterpret_cast<float2*>(o) = make_float2(det[0], det[1]);
        else
          o[0] = det[0];
      }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int r = 0; r < NY; ++r) {
        prv[c][r] = cur[c][r];
        cur[c][r] = nxt[c][r];
      }
  }
}

// ---- double-float arithmetic. The _rn intrinsics keep the compiler from fusing a product
// into a later addition, which would break the error-free transformations.
struct DF {
  float hi, lo;
};
// a + b = s + e exactly (Knuth)
__device__ __forceinline__ DF two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return DF{s, e};
}
// s + e with |e| <= ulp(s) / 2 (requires |a| >= |b| or a == 0)
__device__ __forceinline__ DF fast_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return DF{s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ DF df_add(DF x, DF y) {
  const DF s = two_sum(x.hi, y.hi);
  return fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(x.lo, y.lo)));
}
// a - (m_hi + m_lo) for a float a and a split double m
__device__ __forceinline__ DF df_sub_split(float a, float m_hi, float m_lo) {
  const DF s = two_sum(a, -m_hi);
  return fast_two_sum(s.hi, __fsub_rn(s.lo, m_lo));
}
// square root of x >= 0: r = sqrt(hi), then one Newton correction (x - r^2) / (2 r)
__device__ __forceinline__ DF df_sqrt(DF x) {
  if (!(x.hi > 0.f)) return DF{0.f, 0.f};
  const float r = sqrtf(x.hi);
  const float res = __fadd_rn(fmaf(-r, r, x.hi), x.lo);
  return fast_two_sum(r, res * (0.5f / r));
}

// acc += x. The sum is renormalised at every term: a thread adds 42 terms at 160 x 192 x 160 but 18,000 at the
// largest volume, and a low part that only collects the errors loses a bit with every fourfold count.
__device__ __forceinline__ void df_accumulate(DF& acc, DF x) { acc = df_add(acc, x); }
// acc += x y
__device__ __forceinline__ void df_accumulate_product(DF& acc, DF x, DF y) {
  const float p = __fmul_rn(x.hi, y.hi);
  const float e = __fmaf_rn(x.hi, y.hi, -p);
  df_accumulate(acc, DF{p, __fmaf_rn(x.hi, y.lo, __fmaf_rn(x.lo, y.hi, e))});
}

// the CTA's sums of NK double-float values per thread, written as doubles to part[0 .. NK) by the
// first NK threads, in a fixed order: each value's kMT entries are added in 16 runs of 16 threads'
// entries, then the runs in double. A run's sum is kept in three floats (every addition of the first two is
// exact), so it is as good as one in double, without a conversion and an FP64 addition per thread and value
// (48^3: 70 us with this, 81 us with runs in double)
template <int NK>
__device__ __forceinline__ void cta_sums(const DF (&acc)[NK], double* __restrict__ part) {
  constexpr int kRuns = 16;
  static_assert(NK <= kMT / kRuns, "one run per thread");
  __shared__ DF sh[NK][kMT + 1];
  __shared__ double run[NK][kRuns];
#pragma unroll
  for (int k = 0; k < NK; ++k) sh[k][threadIdx.x] = acc[k];
  __syncthreads();
  const int k = threadIdx.x / kRuns, r = threadIdx.x % kRuns;
  if (k < NK) {
    float a = 0.f, b = 0.f, c = 0.f;
    for (int i = 0; i < kMT / kRuns; ++i) {
      const DF x = sh[k][i * kRuns + r], s = two_sum(a, x.hi), t = two_sum(b, x.lo), q = two_sum(t.hi, s.lo);
      a = s.hi, b = q.hi, c = __fadd_rn(c, __fadd_rn(t.lo, q.lo));
    }
    run[k][r] = (double)a + ((double)b + (double)c);
  }
  __syncthreads();
  if (threadIdx.x < NK) {
    double s = 0.0;
    for (int i = 0; i < kRuns; ++i) s += run[threadIdx.x][i];
    part[threadIdx.x] = s;
  }
}

// out[0 .. nk) = sums over the nparts rows of nk doubles, in a fixed order (one CTA; sh: kMT doubles)
__device__ __forceinline__ void part_sums(const double* __restrict__ part, int nparts, int nk, double* sh,
                                          double* out) {
  const int lanes = kMT / nk, k = threadIdx.x % nk, l = threadIdx.x / nk;
  double a = 0.0;
  for (int i = l; i < nparts; i += lanes) a += part[(size_t)i * nk + k];
  sh[threadIdx.x] = a;
  __syncthreads();
  if (threadIdx.x < nk) {
    double s = 0.0;
    for (int i = 0; i < lanes; ++i) s += sh[i * nk + threadIdx.x];
    out[threadIdx.x] = s;
  }
  __syncthreads();
}

// pass 1: count, sum |ut - ue|, sum ut, sum ue
__global__ void __launch_bounds__(kMT) k_metrics_pass1(const float* __restrict__ ut, const float* __restrict__ ue,
                                                       const unsigned char* __restrict__ roi, size_t V,
                                                       double* __restrict__ part) {
  grid_begin();
  int count = 0;
  DF acc[kP1];  // count, sum |d|, sum ut (3), sum ue (3)
#pragma unroll
  for (int k = 0; k < kP1; ++k) acc[k] = DF{0.f, 0.f};
  for (size_t v = (size_t)blockIdx.x * kMT + threadIdx.x; v < V; v += (size_t)gridDim.x * kMT) {
    if (roi && !roi[v]) continue;
    DF d2{0.f, 0.f};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float a = ut[(size_t)c * V + v], b = ue[(size_t)c * V + v];
      const DF d = two_sum(a, -b);  // a - b exactly
      df_accumulate_product(d2, d, d);
      df_accumulate(acc[2 + c], DF{a, 0.f});
      df_accumulate(acc[5 + c], DF{b, 0.f});
    }
    ++count;
    df_accumulate(acc[1], df_sqrt(d2));
  }
  // a thread's count (below 2^31 voxels over the grid) as a float pair: 24 low bits and the rest
  acc[0] = DF{(float)(count & ~0xffffff), (float)(count & 0xffffff)};
  cta_sums<kP1>(acc, part + (size_t)blockIdx.x * kP1);
}

// means from the pass-1 partials: stats = {count, sum |d|, mt[3], me[3]} with means in place
__global__ void __launch_bounds__(kMT) k_metrics_means(const double* __restrict__ part, int nparts,
                                                       double* __restrict__ stats) {
  grid_begin();
  __shared__ double sh[kMT];
  __shared__ double S[kP1];
  part_sums(part, nparts, kP1, sh, S);
  if (threadIdx.x < kP1) stats[threadIdx.x] = threadIdx.x >= 2 && S[0] > 0.0 ? S[threadIdx.x] / S[0] : S[threadIdx.x];
}

// pass 2: centred moments Ctt (6 unique), Cet (9), see
__global__ void __launch_bounds__(kMT) k_metrics_pass2(const float* __restrict__ ut, const float* __restrict__ ue,
                                                       const unsigned char* __restrict__ roi, size_t V,
                                                       const double* __restrict__ stats, double* __restrict__ part) {
  grid_begin();
  // the means as double-float pairs (hi = nearest float, lo = the float of the remainder)
  float mh[6], ml[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const double m = stats[2 + k];
    mh[k] = (float)m;
    ml[k] = (float)(m - (double)mh[k]);
  }
  DF acc[kP2];
#pragma unroll
  for (int k = 0; k < kP2; ++k) acc[k] = DF{0.f, 0.f};
  for (size_t v = (size_t)blockIdx.x * kMT + threadIdx.x; v < V; v += (size_t)gridDim.x * kMT) {
    if (roi && !roi[v]) continue;
    DF a[3], b[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      a[c] = df_sub_split(ut[(size_t)c * V + v], mh[c], ml[c]);
      b[c] = df_sub_split(ue[(size_t)c * V + v], mh[3 + c], ml[3 + c]);
    }
    df_accumulate_product(acc[0], a[0], a[0]);
    df_accumulate_product(acc[1], a[0], a[1]);
    df_accumulate_product(acc[2], a[0], a[2]);
    df_accumulate_product(acc[3], a[1], a[1]);
    df_accumulate_product(acc[4], a[1], a[2]);
    df_accumulate_product(acc[5], a[2], a[2]);
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int c = 0; c < 3; ++c) df_accumulate_product(acc[6 + 3 * r + c], b[r], a[c]);
#pragma unroll
    for (int c = 0; c < 3; ++c) df_accumulate_product(acc[15], b[c], b[c]);
  }
  cta_sums<kP2>(acc, part + (size_t)blockIdx.x * kP2);
}

// final: fixed-order sums of the pass-2 partials, then Eu, PCC, A = Cet Ctt^-1, b, B
__global__ void __launch_bounds__(kMT) k_metrics_final(const double* __restrict__ part, int nparts,
                                                       const double* __restrict__ stats, double* __restrict__ out) {
  grid_begin();
  __shared__ double sh[kMT];
  __shared__ double S[kP2];
  part_sums(part, nparts, kP2, sh, S);
  if (threadIdx.x != 0) return;
  for (int k = 0; k < 16; ++k) out[k] = 0.0;
  const double cnt = stats[0];
  out[15] = cnt;
  if (cnt == 0.0) return;
  const double C[3][3] = {{S[0], S[1], S[2]}, {S[1], S[3], S[4]}, {S[2], S[4], S[5]}};
  const double E[3][3] = {{S[6], S[7], S[8]}, {S[9], S[10], S[11]}, {S[12], S[13], S[14]}};
  const double stt = C[0][0] + C[1][1] + C[2][2], ste = E[0][0] + E[1][1] + E[2][2];
  out[0] = stats[1] / cnt;
  out[1] = ste / (sqrt(stt) * sqrt(S[15]));
  const double det = C[0][0] * (C[1][1] * C[2][2] - C[1][2] * C[2][1]) -
                     C[0][1] * (C[1][0] * C[2][2] - C[1][2] * C[2][0]) +
                     C[0][2] * (C[1][0] * C[2][1] - C[1][1] * C[2][0]);
  const double rdet = 1.0 / det;
  double inv[3][3];
  inv[0][0] = (C[1][1] * C[2][2] - C[1][2] * C[2][1]) * rdet;
  inv[0][1] = (C[0][2] * C[2][1] - C[0][1] * C[2][2]) * rdet;
  inv[0][2] = (C[0][1] * C[1][2] - C[0][2] * C[1][1]) * rdet;
  inv[1][0] = (C[1][2] * C[2][0] - C[1][0] * C[2][2]) * rdet;
  inv[1][1] = (C[0][0] * C[2][2] - C[0][2] * C[2][0]) * rdet;
  inv[1][2] = (C[0][2] * C[1][0] - C[0][0] * C[1][2]) * rdet;
  inv[2][0] = (C[1][0] * C[2][1] - C[1][1] * C[2][0]) * rdet;
  inv[2][1] = (C[0][1] * C[2][0] - C[0][0] * C[2][1]) * rdet;
  inv[2][2] = (C[0][0] * C[1][1] - C[0][1] * C[1][0]) * rdet;
  double tr = 0.0;
  for (int r = 0; r < 3; ++r) {
    double Ar[3];
    for (int c = 0; c < 3; ++c) Ar[c] = E[r][0] * inv[0][c] + E[r][1] * inv[1][c] + E[r][2] * inv[2][c];
    for (int c = 0; c < 3; ++c) out[3 + 3 * r + c] = Ar[c];
    out[12 + r] = stats[5 + r] - (Ar[0] * stats[2] + Ar[1] * stats[3] + Ar[2] * stats[4]);
    tr += Ar[r];
  }
  out[2] = tr / 3.0;
}
}  // namespace

void launch_jacobian_det(const float* u, Dims n, float* J, cudaStream_t s) {
  const uintptr_t at = reinterpret_cast<uintptr_t>(u) | reinterpret_cast<uintptr_t>(J);
  const int nx = n.n2 % 4 == 0 && at % 16 == 0 ? 4 : n.n2 % 2 == 0 && at % 8 == 0 ? 2 : 1;
  // D chunks so that the grid has at least 8 CTAs per SM of the device (5: 30 us, 8 to 30: 28 us)
  const size_t runs = (size_t)(nx > 1 ? n.n1 : (n.n1 + 1) / 2) * (n.n2 / nx);
  const unsigned gx = (unsigned)((runs + kJT - 1) / kJT);
  const long want = 8L * device_sm_count();
  int zc = n.n0;
  while (zc > 4 && (long)gx * ((n.n0 + zc - 1) / zc) < want) zc = (zc + 1) / 2;
  const dim3 g(gx, (n.n0 + zc - 1) / zc);
  if (nx == 4)
    launch(k_jacobian_det<4, 1>, g, kJT, 0, s)(u, n, J, zc);
  else if (nx == 2)
    launch(k_jacobian_det<2, 1>, g, kJT, 0, s)(u, n, J, zc);
  else
    launch(k_jacobian_det<1, 2>, g, kJT, 0, s)(u, n, J, zc);
}

size_t metrics_scratch_doubles() { return (size_t)kMCtas * (kP1 + kP2) + kP1; }

void launch_deformation_metrics(const float* ut, const float* ue, const unsigned char* roi, Dims n, double* scratch,
                                double* out, cudaStream_t s) {
  const size_t V = vox(n);
  const size_t per_device = (size_t)std::min(kMCtas, kMCtasPerSM * device_sm_count());
  const int ctas = (int)std::max<size_t>(1, std::min<size_t>(per_device, (V + kMT - 1) / kMT));
  double* p1 = scratch;
  double* p2 = scratch + (size_t)kMCtas * kP1;
  double* stats = p2 + (size_t)kMCtas * kP2;
  launch(k_metrics_pass1, ctas, kMT, 0, s)(ut, ue, roi, V, p1);
  launch(k_metrics_means, 1, kMT, 0, s)(p1, ctas, stats);
  launch(k_metrics_pass2, ctas, kMT, 0, s)(ut, ue, roi, V, stats, p2);
  launch(k_metrics_final, 1, kMT, 0, s)(p2, ctas, stats, out);
}

}  // namespace muster
