// sim_kernels.cu -- the windowed similarity of Eq. LNCC / the SiLNCC equation,
// averaged over the valid windows (Eq. sum_lncc, Eq. sim_loss), and its adjoint.
//
// Window R has lower corner c (centre c + R); the valid corners are
// 0 <= c_a <= n_a - w. Forward and adjoint are streamed separable box sums: a CTA owns a
// 32 (W) x 16 (H) tile of windows (forward) or voxels (adjoint) and a chunk of D, and walks D
// plane by plane, in two roles that run beside each other:
//  - W warps, a thread per 8 neighbouring sums of one halo row: box sums along W from 16-byte
//    loads of the staged plane into one of two buffers of W sums;
//  - H/D warps, a thread per column and 4 rows: box sums along H, then along D through a
//    shared-memory ring of the last 2R+1 plane sums with a running total that is re-summed
//    exactly every 2R+1 planes (bounded FP32 drift), and the outputs of the plane.
// The roles hand the buffers over by named barriers (full / empty), so the W pass of one plane
// overlaps the H and D passes of the one before, and no barrier holds all warps of the CTA.
//
// What bounds them: the shared-memory pipe (bytes moved through L1 per output), then instruction
// issue. The layout is chosen for both: 8 sums per W task read 14 inputs (w = 7) instead of 10 for
// every 4, four rows per H/D thread read 10 W sums instead of 16, the ring moves 16 bytes per
// access, and the pitch of the staged rows (4 modulo 8 floats) and the order of the W sums in theirs (sx_col) keep
// the W task's accesses free of bank conflicts.
// Measured on 90 pairs of 160 x 192 x 160, w = 7, SiLNCC: forward 1729 us, adjoint 1451 us (L1 data
// pipe 76 and 81 % busy, DRAM 39 and 57 %); one role per thread with a barrier per plane, W sums in
// runs of 4 and two rows per thread took 2605 and 1802 us. 4 CTAs of 7 warps run on an SM; larger windows and
// LNCC's third moment leave room for 3 or 2 (Box::min_ctas). 56 pairs of 160^3, forward / adjoint: SiLNCC w = 7 965 /
// 775 us, w = 11 1202 / 1007 us; LNCC w = 7 1492 / 1283 us, w = 11 1981 / 1378 us.
//
// The order of the additions is part of the results, and the layout keeps it: along W runs of 4
// sums (a pairwise tree, then a running sum), along H runs of 2, along D the ring. An optimiser
// amplifies the last bits of the gradient (the 20-step registration of three 48^3 volumes moves
// its velocities by 6e-5 when they change), and LNCC, which divides by sqrt(S_FF S_WW), has
// gradients that follow the rounding of the sums in flat regions.
//
// Inputs are staged two planes ahead, by the tensor memory accelerator (mbarrier completion, zero
// fill outside the volume) when the width is a multiple of 4 and the bases are 16-byte aligned,
// otherwise by 4-byte asynchronous copies.
//
// The fixed image's window statistics (mu_F, S_FF) depend on the session only and
// are computed once per level (k_fixed_stats); the forward per pair then needs
// the box sums of W' and F'W' (and of W'^2 for LNCC) only.
// Forward: for every corner of the image grid it writes the coefficients of
//   dSim_R/dW(p) = A_R W(p) - B_R F(p) - C_R   (zero for invalid corners)
//   SiLNCC: A = 1 (implicit; 2/|R| is applied by the adjoint), B = beta = S_FW/(S_FF+eps),
//           C = mu_W - beta mu_F;
//   LNCC:   A = S_FW S_FF / Q^{3/2}, B = 1/sqrt(Q), C = A mu_W - B mu_F, Q = S_FF S_WW + eps,
// and adds Sim_R to a per-CTA partial sum. Sums are taken on values shifted by
// one voxel of the tile (variance is shift invariant) to limit cancellation.
// SiLNCC needs S_WW only in the loss, where sum_R S_WW = sum_p cnt(p) W'(p)^2 - sum_R (sum W')^2/|R|
// with cnt(p) the number of the CTA's windows that hold voxel p: the W pass adds the first term
// once per voxel, which spares a third box sum (a third of the ring and of the arithmetic: 2570 us
// instead of 1729). Both sums are larger than their difference and are carried without rounding
// (FSum), so that the loss stays as smooth in the images as the sum over windows: central
// differences of it with step 1e-3 agree with the gradient to a median of 1.0 to 1.4 % (three draws of
// 128 entries, 6 sessions of 128^3), with a third box sum and Kahan sums to 1.3 to 1.4 %.
// Adjoint: dL/dW(p) = scale * (W(p) sum A - F(p) sum B - sum C) over the
// windows containing p (corners p - 2R .. p).
#include <cudaTypedefs.h>
#include <string.h>

#include <algorithm>
#include <mutex>

#include "kernels.h"
#include "tma.cuh"

namespace muster {

namespace {
constexpr int TX = 32;  // k_fixed_stats

// Statistics of the fixed image of every window, once per session and level:
// out[0][c] = mu_F and out[1][c] = S_FF (centred sum of squares) at corner c, or for SiLNCC
// (KIND 0, which needs S_FF only in beta = S_FW / (S_FF + eps)) out[1][c] = 1 / (S_FF + eps).
// A CTA walks the planes of a 32 x 8 tile: a W task forms 4 neighbouring sums from one read of their
// inputs, a thread of the H and D sums has 1 or 2 rows of a column, and a plane's loads are under way while
// the plane before is summed. Every sum adds its terms one after the other, whatever the threads.
// Shared memory and, in small launches, latency bound it; which number of threads and register budget serves
// both best was measured for each instantiation, over 1 to 10 images of 48^3 to 256^3 (StatCut). w = 7, us, on
// 10, 4 and 2 images of 160 x 192 x 160 and one in the chunks of a stateless call: SiLNCC 275, 131, 69, 32 (128
// threads uncapped 352, 171, 87, 35), LNCC 322, 152, 77, 59 (564, 280, 148, 115); one sum per thread and pass with
// its loads between two barriers took 401, 194, 95, 84 and 378, 181, 88, 78.
template <int R, int KIND>
struct StatCut {
  static constexpr int kCut[2][5][2] = {{{128, 8}, {128, 8}, {256, 4}, {128, 0}, {256, 4}},
                                        {{256, 0}, {256, 6}, {256, 0}, {256, 4}, {256, 4}}};
  static constexpr int threads = kCut[KIND][R - 1][0], ctas = kCut[KIND][R - 1][1];  // CTAs per SM at least (0: no cap)
};
template <int R, int KIND>
__global__ void __launch_bounds__(StatCut<R, KIND>::threads, StatCut<R, KIND>::ctas)
    k_fixed_stats(const float* __restrict__ imgs, float* __restrict__ stats, Dims n, int tz, int nzc, float eps,
                  OpHead* __restrict__ head, PairDesc pd) {
  grid_wait();
  constexpr int NT = StatCut<R, KIND>::threads;
  if (head && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0) *head = OpHead{{}, {}, pd};
  constexpr int WW = 2 * R + 1, TY = 8, RX = TX + 2 * R, RY = TY + 2 * R, PF = (RX + 3) / 4 * 4;
  constexpr int NE = RY * RX, NSLOT = (NE + NT - 1) / NT;
  constexpr int NO = 4, NI = NO + 2 * R, NV = (NI + 3) / 4, NR = TY * TX / NT;
  __shared__ float4 sF[RY][PF / 4];
  __shared__ float4 sx[2][RY][TX / 4];
  const int img = blockIdx.z / nzc, zc = blockIdx.z - img * nzc;
  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY, z0 = zc * tz;
  const int tid = threadIdx.x, tx = tid & 31, row = tid / 32 * NR;
  const int plane = n.n1 * n.n2;
  const size_t V = (size_t)plane * n.n0;
  const float* __restrict__ F = imgs + (size_t)img * V;
  float* __restrict__ out = stats + (size_t)img * 2 * V;
  int goff[NSLOT], soff[NSLOT];  // global (-1: outside) and shared position of a thread's inputs
#pragma unroll
  for (int k = 0; k < NSLOT; ++k) {
    const int e = tid + NT * k;
    const int ry = e / RX, rx = e - ry * RX;
    const int gy = y0 + ry, gx = x0 + rx;
    goff[k] = e < NE && gy < n.n1 && gx < n.n2 ? gy * n.n2 + gx : -1;
    soff[k] = e < NE ? ry * PF + rx : -1;
  }
  const float shF = F[min(z0 + R, n.n0 - 1) * plane + min(y0 + R, n.n1 - 1) * n.n2 + min(x0 + R, n.n2 - 1)];
  const float inv_nw = 1.f / (float)(WW * WW * WW);
  float ring[NR][2][WW] = {}, S[NR][2] = {};
  const int zend = min(z0 + tz, n.n0);
  const int niter = (zend - z0) + 2 * R;
  float next[NSLOT];
  auto load = [&](int z) {
#pragma unroll
    for (int k = 0; k < NSLOT; ++k) next[k] = z < n.n0 && goff[k] >= 0 ? F[z * plane + goff[k]] - shF : 0.f;
  };
  load(z0);
  for (int base = 0; base < niter; base += WW) {
#pragma unroll
    for (int j = 0; j < WW; ++j) {
      const int it = base + j;
      if (it >= niter) break;
#pragma unroll
      for (int k = 0; k < NSLOT; ++k)
        if (soff[k] >= 0) reinterpret_cast<float*>(sF)[soff[k]] = next[k];
      __syncthreads();
      load(z0 + it + 1);
      for (int t = tid; t < RY * (TX / NO); t += NT) {
        const int ry = t / (TX / NO), run = t % (TX / NO);
        float v[4 * NV], a0[NO] = {}, a1[NO] = {};
#pragma unroll
        for (int q = 0; q < NV; ++q) {
          const float4 f = sF[ry][run + q];
          v[4 * q] = f.x, v[4 * q + 1] = f.y, v[4 * q + 2] = f.z, v[4 * q + 3] = f.w;
        }
#pragma unroll
        for (int o = 0; o < NO; ++o)
#pragma unroll
          for (int k = 0; k < WW; ++k) {
            a0[o] += v[o + k];
            a1[o] = fmaf(v[o + k], v[o + k], a1[o]);
          }
        sx[0][ry][run] = make_float4(a0[0], a0[1], a0[2], a0[3]);
        sx[1][ry][run] = make_float4(a1[0], a1[1], a1[2], a1[3]);
      }
      __syncthreads();
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        float h[NR + 2 * R];
#pragma unroll
        for (int k = 0; k < NR + 2 * R; ++k) h[k] = reinterpret_cast<const float*>(sx[m][row + k])[tx];
#pragma unroll
        for (int i = 0; i < NR; ++i) {
          float v = 0.f;
#pragma unroll
          for (int k = 0; k < WW; ++k) v += h[i + k];
          S[i][m] += v - ring[i][m][j];
          ring[i][m][j] = v;
          if (j == WW - 1) {
            float t = 0.f;
#pragma unroll
            for (int k = 0; k < WW; ++k) t += ring[i][m][k];
            S[i][m] = t;
          }
        }
      }
      if (it >= 2 * R) {
        const int cz = z0 + it - 2 * R, cx = x0 + tx;
#pragma unroll
        for (int i = 0; i < NR; ++i) {
          const int cy = y0 + row + i;
          if (cx < n.n2 && cy < n.n1) {
            const int o = cz * plane + cy * n.n2 + cx;
            out[o] = S[i][0] * inv_nw + shF;
            const float sff = fmaxf(S[i][1] - S[i][0] * S[i][0] * inv_nw, 0.f);
            out[V + o] = KIND == 0 ? 1.f / (sff + eps) : sff;
          }
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
constexpr int kTX = 32, kTY = 16;   // outputs of a CTA's tile along W and H
constexpr int kXO = 8;              // sums of one W task
constexpr int kYO = 4;              // rows of one H/D thread
constexpr int kHD = kTX * kTY / kYO;  // H/D threads
// a tensor copy must start on a 16-byte boundary: the forward's box starts at x0 = 32 * tile
static_assert(kTX % 4 == 0, "the staged forward box must start at a multiple of 4 floats");

// tile shapes for window radius R
template <int R>
struct Box {
  static constexpr int WW = 2 * R + 1;
  static constexpr int RX = kTX + 2 * R, RY = kTY + 2 * R;  // halo columns and rows of a plane
  static constexpr int NI = kXO + 2 * R;                    // inputs of a W task
  static constexpr int NV = (NI + (2 * R & 3) + 3) / 4;     // its float4 loads at most (bwd_xoff columns early)
  static constexpr int NTASK = RY * (kTX / kXO);            // W tasks of a plane
  static constexpr int WT = (NTASK + 31) / 32 * 32;         // W threads
  static constexpr int NT = kHD + WT;
  static constexpr int PX = R <= 2 ? 36 : 44;               // row pitch of a staged plane
  static constexpr int TS = (RY * PX + 31) & ~31;           // floats of one staged plane (128-byte multiple)
  static_assert(PX >= kTX - kXO + 4 * NV && PX % 8 == 4, "pitch");
  __host__ __device__ static constexpr int sx_floats(int nm) { return nm * RY * kTX; }
  __host__ __device__ static constexpr int ring_floats(int nm) { return WW * nm * kTX * kTY; }
  // dynamic shared memory: [2 stages][nin][TS] without the last one's padding, [2 planes][nm] W sums, D
  // ring, two mbarriers
  __host__ __device__ static constexpr int sx_at(int nin) { return (2 * nin - 1) * TS + RY * PX; }
  __host__ __device__ static constexpr int bar_at(int nin, int nm) {
    return sx_at(nin) + 2 * sx_floats(nm) + ring_floats(nm);
  }
  static_assert(RY * PX % 4 == 0, "the W sums and the ring are moved by 16 bytes");
  __host__ __device__ static constexpr size_t bytes(int nin, int nm) {
    return sizeof(float) * (size_t)bar_at(nin, nm) + 2 * sizeof(uint64_t);
  }
  // CTAs that an SM's 228 KB hold (1 KB of each CTA's share is the system's, shares are multiples of
  // 128 bytes), 4 at most: the register budget is cut for these. Cut for 3, the SiLNCC forward of w = 7 takes 12 %
  // longer; cut for 4 where only 2 fit, the kernels of w = 11 spilled 76 to 92 bytes.
  static constexpr int min_ctas(int nin, int nm) {
    const size_t fit = (228 << 10) / ((bytes(nin, nm) + 1024 + 127) / 128 * 128);
    return fit > 4 ? 4 : (int)fit;
  }
};
// position of W sum x of row r, without its row's base: odd rows swap neighbouring runs of 4, so that the two rows
// that 8 lanes of a W warp write with 16-byte stores take all banks once
__device__ __forceinline__ int sx_col(int x, int r) { return x ^ (4 * (r & 1)); }

// x offset of the adjoint's staged box: its first column x0 - 2R is rounded down to a
// multiple of 4 (16-byte aligned tile coordinate), so the box starts XOFF columns early
template <int R>
__host__ __device__ constexpr int bwd_xoff() {
  return (2 * R) & 3;
}

// the launch's tiles: a one-dimensional grid over groups of `grp` pairs, then D chunks, tiles
// and, fastest, the pairs of the group
struct Tiles {
  int np, grp, gx, gy, nzc, tz;
};
struct Tile {
  int pair, x0, y0, z0, part;  // part: index of the CTA's partial sum
};
// Pairs that share a fixed image (the engine orders them by fixed image) run beside each other
// on the same tile, so that its F, mu_F and S_FF planes are read from L2 by all but the first
// (10 sessions of 160 x 192 x 160: forward 1678 us, in pair order 1763 us, before the loss sums were widened).
__device__ __forceinline__ Tile tile_of(const Tiles& g) {
  const unsigned per = (unsigned)g.gx * g.gy * g.nzc;
  unsigned id = blockIdx.x;
  const unsigned span = g.grp * per, first = id / span * g.grp;
  id -= id / span * span;
  const unsigned in = min((unsigned)g.grp, (unsigned)g.np - first);
  Tile t;
  t.pair = (int)(first + id % in);
  id /= in;
  t.part = (int)(t.pair * per + id);
  t.x0 = (int)(id % g.gx) * kTX;
  id /= g.gx;
  t.y0 = (int)(id % g.gy) * kTY;
  t.z0 = (int)(id / g.gy) * g.tz;
  return t;
}

// The CTA's sum of the per-thread float-float sums, valid in thread 0: float-float
// sums within each warp, then the warp sums in double.
template <int NT>
__device__ __forceinline__ double block_sum(FF x, float* sh) {
  x = warp_sum_ff(x);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) {
    sh[2 * w] = x.hi;
    sh[2 * w + 1] = x.lo;
  }
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < NT / 32; ++i) r += (double)sh[2 * i] + (double)sh[2 * i + 1];
  return r;
}

// a + b = s exactly, with the rounding error of s in e (Knuth)
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
  const float s = __fadd_rn(a, b), v = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, v)), __fsub_rn(b, v));
  return s;
}

// running sum without rounding: hi + lo carries every term (Knuth's two-sum). A term changes nothing
// but the sum, so a change in one window leaves the rounding of all others as it was.
struct FSum {
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(float x) {
    float e;
    hi = two_sum(hi, x, e);
    lo += e;
  }
};

// pairwise sum of v[0..N-1]: a dependency chain of depth log2(N) instead of N - 1
template <int N>
struct TreeSum {
  __device__ __forceinline__ static float of(const float* v) {
    return TreeSum<N / 2>::of(v) + TreeSum<N - N / 2>::of(v + N / 2);
  }
};
template <>
struct TreeSum<1> {
  __device__ __forceinline__ static float of(const float* v) { return v[0]; }
};

// running box sum of one run: out[i] = sum_{k<WW} v[i + k], i < NO
template <int WW, int NO>
__device__ __forceinline__ void runsum(const float* v, float* out) {
  float s = TreeSum<WW>::of(v);
  out[0] = s;
#pragma unroll
  for (int i = 1; i < NO; ++i) {
    s += v[i + WW - 1] - v[i - 1];
    out[i] = s;
  }
}

// The same for products v[k] = a[k] b[k]: a product that enters one addition only is fused into
// it, the others are rounded first (p). In a run of 4 those are the products past the first sum's
// window and, within it, all but the first three, which leave the running sum again.
template <int N>
struct ProdTree {
  template <int K>  // sum of the products K .. K + N - 1
  __device__ __forceinline__ static float of(const float* a, const float* b, const float* p) {
    if constexpr (N == 1) {
      return p[K];
    } else {
      constexpr int NL = N / 2;
      if constexpr (NL == 1 && K >= 3)
        return __fmaf_rn(a[K], b[K], ProdTree<N - NL>::template of<K + NL>(a, b, p));
      else if constexpr (N - NL == 1 && K + NL >= 3)
        return __fmaf_rn(a[K + NL], b[K + NL], ProdTree<NL>::template of<K>(a, b, p));
      else
        return __fadd_rn(ProdTree<NL>::template of<K>(a, b, p), ProdTree<N - NL>::template of<K + NL>(a, b, p));
    }
  }
};
template <int WW>
__device__ __forceinline__ void runsum4(const float* a, const float* b, float* out) {
  float p[WW];
#pragma unroll
  for (int k = 0; k < WW; ++k) p[k] = __fmul_rn(a[k], b[k]);
  out[0] = ProdTree<WW>::template of<0>(a, b, p);
#pragma unroll
  for (int i = 1; i < 4; ++i)
    out[i] = __fadd_rn(out[i - 1], __fmaf_rn(a[i + WW - 1], b[i + WW - 1], -p[i - 1]));
}

// ---- hand-over of the two buffers of W sums between the roles (named barriers; 0 is
// __syncthreads). Whole warps take part, converged first: bar.sync / bar.arrive are aligned.
enum { kBarFull = 1, kBarEmpty = 3, kBarStage = 5 };  // full, empty: one per buffer
__device__ __forceinline__ void bar_sync(int id, int threads) {
  __syncwarp();
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
  __syncwarp();
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// ---- staged input planes of the W warps, two stages of NIN arrays. TMA: one thread issues a
// 4-D tile copy (x, y, z, volume) per array and plane, an mbarrier per stage tracks completion.
// Waits are bounded: a wait that runs out sets *err and the kernel carries on without waiting (its
// results are then reported as invalid by the host), so no CTA can hang. Otherwise every W thread
// copies its share of a plane with 4-byte asynchronous copies, zeros outside the volume.
__device__ __forceinline__ void copy4(float* dst, const float* src, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(bytes)
               : "memory");
}
template <int R, int NIN, bool TMA>
struct Stages {
  float* stage;
  uint64_t* bar;
  const CUtensorMap* map[NIN];
  int vol[NIN];
  const float* src[NIN];  // the volumes of the unstaged path
  int x0, y0, z0, niter, wt;
  Dims n;
  bool ok;
  __device__ __forceinline__ void load(int it) {  // plane z0 + it into stage it & 1
    using B = Box<R>;
    float* dst = stage + (it & 1) * NIN * B::TS;
    if (TMA) {
      if (wt == 0) {
        mbar_expect_tx(&bar[it & 1], (unsigned)(NIN * B::RY * B::PX * 4));
#pragma unroll
        for (int a = 0; a < NIN; ++a) tma_load4(dst + a * B::TS, map[a], x0, y0, z0 + it, vol[a], &bar[it & 1]);
      }
    } else {
      // a warp per row, columns lane and lane + 32; outside the volume the copy reads nothing
      const int z = z0 + it, lane = wt & 31, xa = x0 + lane, xb = xa + 32;
      const bool zin = z >= 0 && z < n.n0;
      const int ina = zin && xa >= 0 && xa < n.n2 ? 4 : 0, inb = zin && xb >= 0 && xb < n.n2 ? 4 : 0;
      const int ca = ina ? xa : 0, cb = inb ? xb : 0, zo = zin ? z * n.n1 : 0;
      for (int row = wt >> 5; row < B::RY; row += B::WT / 32) {
        const int y = y0 + row;
        const bool yin = y >= 0 && y < n.n1;
        const int o = (zo + (yin ? y : 0)) * n.n2;
#pragma unroll
        for (int a = 0; a < NIN; ++a) {
          float* to = dst + a * B::TS + row * B::PX + lane;
          copy4(to, src[a] + (o + ca), yin ? ina : 0);
          if (lane < 2 * R) copy4(to + 32, src[a] + (o + cb), yin ? inb : 0);
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
  }
  __device__ __forceinline__ void start() {
    ok = true;
    load(0);
    if (niter > 1)
      load(1);
    else if (!TMA)
      asm volatile("cp.async.commit_group;" ::: "memory");
  }
  __device__ __forceinline__ void wait(int it) {  // plane it is in its stage
    if (TMA) {
      ok = ok && mbar_wait(&bar[it & 1], (unsigned)(it >> 1) & 1u);  // after a failure, stop waiting
    } else {
      asm volatile("cp.async.wait_group 1;" ::: "memory");
      bar_sync(kBarStage, Box<R>::WT);
    }
  }
  __device__ __forceinline__ void next(int it) {  // every W thread is past plane it: refill its stage
    bar_sync(kBarStage, Box<R>::WT);
    if (TMA) {
      if (it + 2 < niter) {
        if (wt == 0) fence_proxy_async();
        load(it + 2);
      }
    } else if (it + 2 < niter) {
      load(it + 2);
    } else {
      asm volatile("cp.async.commit_group;" ::: "memory");  // keeps the group count of wait()
    }
  }
  // report a failed wait, then give the copies still in flight into this CTA's stages one more
  // bounded wait (the last use of each stage) before the CTA's shared memory is released
  __device__ __forceinline__ void finish(int* err) {
    if (!TMA || ok) return;
    if (err) atomicOr(err, 1);
    for (int st = 0; st < 2 && st < niter; ++st) {
      const int last = niter - 1 - ((niter - 1 - st) & 1);  // last iteration that used stage st
      mbar_wait(&bar[st], (unsigned)(last >> 1) & 1u);
    }
  }
};

// the 8 sums of one moment of a W task, of values or of products, into the W sums: the first 4 to
// d0, the others to d1
template <int R>
__device__ __forceinline__ void w_sums(const float* v, float* __restrict__ d0, float* __restrict__ d1) {
  float o[kXO];
  runsum<Box<R>::WW, 4>(v, o);
  runsum<Box<R>::WW, 4>(v + 4, o + 4);
  *reinterpret_cast<float4*>(d0) = make_float4(o[0], o[1], o[2], o[3]);
  *reinterpret_cast<float4*>(d1) = make_float4(o[4], o[5], o[6], o[7]);
}
template <int R>
__device__ __forceinline__ void w_sums(const float* a, const float* b, float* __restrict__ d0, float* __restrict__ d1) {
  float o[kXO];
  runsum4<Box<R>::WW>(a, b, o);
  runsum4<Box<R>::WW>(a + 4, b + 4, o + 4);
  *reinterpret_cast<float4*>(d0) = make_float4(o[0], o[1], o[2], o[3]);
  *reinterpret_cast<float4*>(d1) = make_float4(o[4], o[5], o[6], o[7]);
}

// H and D passes of one plane for a thread's column and rows: S += newest - oldest plane sum,
// re-summed from the ring when its last slot was written (as a tree, or with SEQ one after the other)
template <int R, int NM, bool SEQ = false>
struct Ring {
  static constexpr int kSlot = kHD;  // float4 (the thread's rows) of one moment of one plane
  float4* mem;
  float S[NM][kYO];
  int j;
  __device__ __forceinline__ void init(float* base) {
    mem = reinterpret_cast<float4*>(base) + threadIdx.x;
    j = 0;
#pragma unroll
    for (int m = 0; m < NM; ++m)
#pragma unroll
      for (int i = 0; i < kYO; ++i) S[m][i] = 0.f;
#pragma unroll
    for (int q = 0; q < NM * Box<R>::WW; ++q) mem[q * kSlot] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  // plane h of niter from its buffer of W sums: waits for it and hands it back once read
  __device__ __forceinline__ void plane(const float* sx2, int h, int niter, int col, int row) {
    using B = Box<R>;
    bar_sync(kBarFull + (h & 1), B::NT);
    static_assert(kYO % 2 == 0, "a thread's first row is even");
    const float* sx = sx2 + (h & 1) * B::sx_floats(NM) + row * kTX;
    const float* sxk[2] = {sx + sx_col(col, 0), sx + sx_col(col, 1)};
    float a[NM][kYO];
#pragma unroll
    for (int m = 0; m < NM; ++m) {
      float v[kYO + 2 * R];
#pragma unroll
      for (int k = 0; k < kYO + 2 * R; ++k) v[k] = sxk[k & 1][(m * B::RY + k) * kTX];
#pragma unroll
      for (int i = 0; i < kYO; i += 2) runsum<B::WW, 2>(v + i, a[m] + i);
    }
    if (h + 2 < niter) bar_arrive(kBarEmpty + (h & 1), B::NT);
#pragma unroll
    for (int m = 0; m < NM; ++m) {
      float4* rp = mem + (j * NM + m) * kSlot;
      const float4 old = *rp;
      S[m][0] += a[m][0] - old.x;
      S[m][1] += a[m][1] - old.y;
      S[m][2] += a[m][2] - old.z;
      S[m][3] += a[m][3] - old.w;
      *rp = make_float4(a[m][0], a[m][1], a[m][2], a[m][3]);
    }
    if (++j == B::WW) {  // exact re-sum bounds the drift of the running sums
      j = 0;
#pragma unroll
      for (int m = 0; m < NM; ++m) {
        float t[kYO][B::WW];
#pragma unroll
        for (int q = 0; q < B::WW; ++q) {
          const float4 r = mem[(q * NM + m) * kSlot];
          t[0][q] = r.x, t[1][q] = r.y, t[2][q] = r.z, t[3][q] = r.w;
        }
#pragma unroll
        for (int i = 0; i < kYO; ++i) {
          if (SEQ) {
            S[m][i] = t[i][0];
#pragma unroll
            for (int q = 1; q < B::WW; ++q) S[m][i] += t[i][q];
          } else {
            S[m][i] = TreeSum<B::WW>::of(t[i]);
          }
        }
      }
    }
  }
};

// number of window corners in [0, last] that hold offset k (0 when last < 0)
__device__ __forceinline__ int corners_holding(int k, int last, int reach) {
  return max(0, min(k, last) - max(0, k - reach) + 1);
}

// Forward of one pair (see the head of the file).
template <int R, int KIND, bool TMA>
__global__ void __launch_bounds__(Box<R>::NT, Box<R>::min_ctas(2, KIND == 0 ? 2 : 3))
    k_sim_fwd(const __grid_constant__ SimMaps maps, const PairDesc* __restrict__ pd, const float* __restrict__ Wb,
              size_t Wstride, float* __restrict__ coef, size_t cstride, double* __restrict__ part, Dims n, Tiles g,
              float eps, int* __restrict__ err) {
  grid_wait();
  using B = Box<R>;
  constexpr int NM = KIND == 0 ? 2 : 3, NC = KIND == 0 ? 2 : 3;
  extern __shared__ __align__(128) float smem[];
  float* sx2 = smem + B::sx_at(2);  // stages: [2][F, W][TS]
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + B::bar_at(2, NM));
  const Tile t = tile_of(g);
  const int plane = n.n1 * n.n2;
  const PairDesc d = pd[t.pair];
  const float* __restrict__ F = d.Ii;
  const float* __restrict__ W = Wb + (size_t)t.pair * Wstride;
  const int zend = min(t.z0 + g.tz, n.n0), niter = (zend - t.z0) + 2 * R;
  const int mx = n.n2 - B::WW, my = n.n1 - B::WW, mz = n.n0 - B::WW;
  const int so = min(t.z0 + R, n.n0 - 1) * plane + min(t.y0 + R, n.n1 - 1) * n.n2 + min(t.x0 + R, n.n2 - 1);
  const float shF = F[so], shW = W[so];
  const int wt = (int)threadIdx.x - kHD;  // W thread, or an H/D thread when negative
  if (TMA && wt == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    mbar_fence_init();
  }
  __syncthreads();
  // SiLNCC: W threads sum_p cnt(p) W'(p)^2, H/D threads sum_R ((sum W')^2/|R| + beta S_FW);
  // LNCC: H/D threads sum_R Sim_R
  FSum acc;
  if (wt >= 0) {
    Stages<R, 2, TMA> st{smem, bar, {&maps.F, &maps.W}, {d.fi, t.pair}, {F, W}, t.x0, t.y0, t.z0, niter, wt, n, true};
    st.start();
    const bool on = wt < B::NTASK;
    const int row = wt >> 2, xs = kXO * (wt & 3);
    // how many of the tile's windows hold a voxel of this row, per axis (along W: valid corners
    // of this task, all kXO of them except at the volume's end)
    const int cnt_y = on ? corners_holding(row, min(kTY - 1, my - t.y0), 2 * R) : 0;
    const int last_x = min(kXO - 1, mx - t.x0 - xs), last_z = min(zend - 1, mz) - t.z0;
    for (int it = 0; it < niter; ++it) {
      if (it >= 2) bar_sync(kBarEmpty + (it & 1), B::NT);
      st.wait(it);
      float f[4 * B::NV], w[4 * B::NV];
      if (on) {
        const float4* pF = reinterpret_cast<const float4*>(smem + 2 * (it & 1) * B::TS + row * B::PX + xs);
        const float4* pW = pF + B::TS / 4;
#pragma unroll
        for (int q = 0; q < (B::NI + 3) / 4; ++q) {
          const float4 a = pF[q], b = pW[q];
          f[4 * q] = a.x - shF, f[4 * q + 1] = a.y - shF, f[4 * q + 2] = a.z - shF, f[4 * q + 3] = a.w - shF;
          w[4 * q] = b.x - shW, w[4 * q + 1] = b.y - shW, w[4 * q + 2] = b.z - shW, w[4 * q + 3] = b.w - shW;
        }
        float* sx = sx2 + (it & 1) * B::sx_floats(NM) + row * kTX;
        float *d0 = sx + sx_col(xs, row), *d1 = sx + sx_col(xs + 4, row);
        constexpr int M = B::RY * kTX;
        w_sums<R>(w, d0, d1);
        w_sums<R>(f, w, d0 + (NM - 1) * M, d1 + (NM - 1) * M);
        if (KIND == 1) w_sums<R>(w, w, d0 + M, d1 + M);
      }
      bar_arrive(kBarFull + (it & 1), B::NT);
      if (KIND == 0) {
        // a voxel that no window holds adds nothing, whatever it is (0 * Inf)
        const int c = cnt_y * corners_holding(it, last_z, 2 * R);
        if (c > 0 && last_x >= 0) {
          float sq[B::NI];
          if (last_x == kXO - 1) {
#pragma unroll
            for (int k = 0; k < B::NI; ++k)
              sq[k] = (float)((k < kXO - 1 ? k : kXO - 1) - (k > 2 * R ? k - 2 * R : 0) + 1) * w[k] * w[k];
          } else {
#pragma unroll
            for (int k = 0; k < B::NI; ++k) sq[k] = (float)corners_holding(k, last_x, 2 * R) * w[k] * w[k];
          }
          // the two upper levels of the pairwise sum and the product with c, with their errors
          constexpr int N1 = B::NI / 2, N2 = B::NI - N1;
          float e0, e1, e2;
          const float lo = two_sum(TreeSum<N1 / 2>::of(sq), TreeSum<N1 - N1 / 2>::of(sq + N1 / 2), e0);
          const float hi = two_sum(TreeSum<N2 / 2>::of(sq + N1), TreeSum<N2 - N2 / 2>::of(sq + N1 + N2 / 2), e1);
          const float a = two_sum(lo, hi, e2), ca = __fmul_rn((float)c, a);
          acc.add(ca);
          acc.lo += __fmaf_rn((float)c, e2 + (e0 + e1), __fmaf_rn((float)c, a, -ca));
        }
      }
      st.next(it);
    }
    st.finish(err);
  } else {
    const float inv_nw = 1.f / (float)(B::WW * B::WW * B::WW);
    const int col = threadIdx.x & 31, row = (threadIdx.x >> 5) * kYO;
    const int cx = t.x0 + col, cy = t.y0 + row;
    const int rows = cx < n.n2 ? min(kYO, n.n1 - cy) : 0;            // rows inside the volume
    const int live_rows = cx <= mx ? min(rows, my - cy + 1) : 0;     // rows whose window is inside (H and W)
    const ptrdiff_t o0 = (ptrdiff_t)t.z0 * plane + (ptrdiff_t)cy * n.n2 + cx;
    const float* __restrict__ mu_p = d.Fs + o0;
    const float* __restrict__ sf_p = mu_p + (size_t)plane * n.n0;
    float* __restrict__ c_p = coef + (size_t)t.pair * NC * cstride + o0;
    Ring<R, NM, !TMA> ring;
    ring.init(sx2 + 2 * B::sx_floats(NM));
    // coefficients of row i's window and its term of the loss
    auto window = [&](int i, float muF, float Sff, float& c0, float& c1, float& c2) -> float {
      const float s0 = ring.S[0][i];
      const float Sfw = ring.S[NM - 1][i] - (muF - shF) * s0;
      const float muW = __fmaf_rn(s0, inv_nw, shW);  // s0 * inv_nw is used again below: fused all the same
      if (KIND == 0) {
        const float beta = Sfw * Sff;  // Sff holds 1 / (S_FF + eps) for SiLNCC
        c0 = beta;
        c1 = muW - beta * muF;
        return fmaf(s0, s0 * inv_nw, Sfw * beta);
      }
      const float Sww = fmaxf(ring.S[1][i] - s0 * s0 * inv_nw, 0.f);
      const float Q = Sff * Sww + eps;
      const float rq = 1.f / sqrtf(Q);
      c0 = Sfw * Sff * rq * rq * rq;
      c1 = rq;
      c2 = c0 * muW - c1 * muF;
      return 1.f - Sfw * rq;
    };
    for (int h = 0; h < niter; ++h) {
      // mu_F and S_FF of this thread's windows of the output plane (corner plane h - 2R), loaded
      // now and used after the passes
      const bool outp = h >= 2 * R;
      const int nl = outp && t.z0 + h - 2 * R <= mz ? live_rows : 0;
      float mu[kYO], sf[kYO];
      if (nl == kYO) {
#pragma unroll
        for (int i = 0; i < kYO; ++i) {
          mu[i] = __ldg(mu_p + i * n.n2);
          sf[i] = __ldg(sf_p + i * n.n2);
        }
      } else {
#pragma unroll
        for (int i = 0; i < kYO; ++i)
          if (i < nl) {
            mu[i] = __ldg(mu_p + i * n.n2);
            sf[i] = __ldg(sf_p + i * n.n2);
          }
      }
      ring.plane(sx2, h, niter, col, row);
      if (outp) {
        if (nl == kYO) {
          float val[kYO];
#pragma unroll
          for (int i = 0; i < kYO; ++i) {
            float c0, c1, c2;
            val[i] = window(i, mu[i], sf[i], c0, c1, c2);
            c_p[i * n.n2] = c0;
            c_p[cstride + i * n.n2] = c1;
            if (KIND == 1) c_p[2 * cstride + i * n.n2] = c2;
          }
          acc.add((val[0] + val[1]) + (val[2] + val[3]));
        } else {
#pragma unroll
          for (int i = 0; i < kYO; ++i)
            if (i < rows) {
              float c0 = 0.f, c1 = 0.f, c2 = 0.f;
              if (i < nl) acc.add(window(i, mu[i], sf[i], c0, c1, c2));
              c_p[i * n.n2] = c0;
              c_p[cstride + i * n.n2] = c1;
              if (KIND == 1) c_p[2 * cstride + i * n.n2] = c2;
            }
        }
        mu_p += plane, sf_p += plane, c_p += plane;
      }
    }
  }
  const float sgn = KIND == 0 && wt < 0 ? -1.f : 1.f;
  // the warp sums take the place of the W sums, which no thread reads any more past the barrier
  const double sum = block_sum<B::NT>(FF{sgn * acc.hi, sgn * acc.lo}, sx2);
  if (threadIdx.x == 0) part[t.part] = KIND == 0 ? sum / (double)(B::WW * B::WW * B::WW) : sum;
}

template <int R, int KIND, bool TMA>
__global__ void __launch_bounds__(Box<R>::NT, Box<R>::min_ctas(KIND == 0 ? 2 : 3, KIND == 0 ? 2 : 3))
    k_sim_bwd(const __grid_constant__ SimMaps maps, const PairDesc* __restrict__ pd, const float* __restrict__ Wb,
              size_t Wstride, const float* __restrict__ coef, size_t cstride, float* __restrict__ dLdW, Dims n, Tiles g,
              float scale, int* __restrict__ err) {
  grid_wait();
  using B = Box<R>;
  constexpr int NC = KIND == 0 ? 2 : 3, XOFF = TMA ? bwd_xoff<R>() : 0;
  static_assert(!TMA || (2 * R + XOFF) % 4 == 0, "the staged adjoint box must start at a multiple of 4 floats");
  extern __shared__ __align__(128) float smem[];
  float* sx2 = smem + B::sx_at(NC);  // stages: [2][NC][TS]
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + B::bar_at(NC, NC));
  const Tile t = tile_of(g);
  const int plane = n.n1 * n.n2;
  const int zend = min(t.z0 + g.tz, n.n0), niter = (zend - t.z0) + 2 * R;
  const int wt = (int)threadIdx.x - kHD;  // W thread, or an H/D thread when negative
  if (TMA && wt == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    mbar_fence_init();
  }
  __syncthreads();
  if (wt >= 0) {
    Stages<R, NC, TMA> st;
    st.stage = smem, st.bar = bar, st.niter = niter, st.wt = wt, st.n = n;
    st.x0 = t.x0 - 2 * R - XOFF, st.y0 = t.y0 - 2 * R, st.z0 = t.z0 - 2 * R;
#pragma unroll
    for (int m = 0; m < NC; ++m) {
      st.map[m] = &maps.C;
      st.vol[m] = t.pair * NC + m;
      st.src[m] = coef + ((size_t)t.pair * NC + m) * cstride;
    }
    st.start();
    const bool on = wt < B::NTASK;
    const int row = wt >> 2, xs = kXO * (wt & 3);
    for (int it = 0; it < niter; ++it) {
      if (it >= 2) bar_sync(kBarEmpty + (it & 1), B::NT);
      st.wait(it);
      if (on) {
        float* sx = sx2 + (it & 1) * B::sx_floats(NC) + row * kTX;
        float *d0 = sx + sx_col(xs, row), *d1 = sx + sx_col(xs + 4, row);
#pragma unroll
        for (int m = 0; m < NC; ++m) {
          float v[4 * B::NV];
          const float4* src = reinterpret_cast<const float4*>(smem + (NC * (it & 1) + m) * B::TS + row * B::PX + xs);
#pragma unroll
          for (int q = 0; q < (B::NI + XOFF + 3) / 4; ++q) {
            const float4 a = src[q];
            v[4 * q] = a.x, v[4 * q + 1] = a.y, v[4 * q + 2] = a.z, v[4 * q + 3] = a.w;
          }
          w_sums<R>(v + XOFF, d0 + m * B::RY * kTX, d1 + m * B::RY * kTX);
        }
      }
      bar_arrive(kBarFull + (it & 1), B::NT);
      st.next(it);
    }
    st.finish(err);
    return;
  }
  const int mx = n.n2 - B::WW, my = n.n1 - B::WW, mz = n.n0 - B::WW;
  const int col = threadIdx.x & 31, row = (threadIdx.x >> 5) * kYO;
  const int px = t.x0 + col, py = t.y0 + row;
  const int rows = px < n.n2 ? min(kYO, n.n1 - py) : 0;
  float cnt_xy[kYO];  // valid windows that hold the voxel, in the plane
#pragma unroll
  for (int i = 0; i < kYO; ++i)
    cnt_xy[i] = (float)(corners_holding(px, mx, 2 * R) * corners_holding(py + i, my, 2 * R));
  const ptrdiff_t o0 = (ptrdiff_t)t.z0 * plane + (ptrdiff_t)py * n.n2 + px;
  const float* __restrict__ F_p = pd[t.pair].Ii + o0;
  const float* __restrict__ W_p = Wb + (size_t)t.pair * Wstride + o0;
  float* __restrict__ out = dLdW + (size_t)t.pair * Wstride + o0;
  Ring<R, NC> ring;
  ring.init(sx2 + 2 * B::sx_floats(NC));
  auto gradient = [&](int i, float czn, float wv, float fv) {
    if (KIND == 0) return scale * (cnt_xy[i] * czn * wv - fv * ring.S[0][i] - ring.S[1][i]);
    return scale * (wv * ring.S[0][i] - fv * ring.S[1][i] - ring.S[NC - 1][i]);
  };
  for (int h = 0; h < niter; ++h) {
    // W and F at this thread's voxels of the output plane, loaded now, used after the passes
    const int nr = h >= 2 * R ? rows : 0;
    float wv[kYO], fv[kYO];
    if (nr == kYO) {
#pragma unroll
      for (int i = 0; i < kYO; ++i) {
        wv[i] = __ldg(W_p + i * n.n2);
        fv[i] = __ldg(F_p + i * n.n2);
      }
    } else {
#pragma unroll
      for (int i = 0; i < kYO; ++i)
        if (i < nr) {
          wv[i] = __ldg(W_p + i * n.n2);
          fv[i] = __ldg(F_p + i * n.n2);
        }
    }
    ring.plane(sx2, h, niter, col, row);
    if (h >= 2 * R) {
      const float czn = (float)corners_holding(t.z0 - 2 * R + h, mz, 2 * R);
      if (nr == kYO) {
#pragma unroll
        for (int i = 0; i < kYO; ++i) out[i * n.n2] = gradient(i, czn, wv[i], fv[i]);
      } else {
#pragma unroll
        for (int i = 0; i < kYO; ++i)
          if (i < nr) out[i * n.n2] = gradient(i, czn, wv[i], fv[i]);
      }
      W_p += plane, F_p += plane, out += plane;
    }
  }
}

template <typename Kern>
cudaError_t set_smem(Kern k, size_t bytes) {
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}
template <int R, int KIND, bool TMA>
cudaError_t prepare_one() {
  constexpr int NC = KIND == 0 ? 2 : 3;
  const cudaError_t a = set_smem(k_sim_fwd<R, KIND, TMA>, Box<R>::bytes(2, NC)),
                    b = set_smem(k_sim_bwd<R, KIND, TMA>, Box<R>::bytes(NC, NC));
  return a != cudaSuccess ? a : b;
}
template <int R>
cudaError_t prepare_r() {
  const cudaError_t e[4] = {prepare_one<R, 0, false>(), prepare_one<R, 0, true>(), prepare_one<R, 1, false>(),
                            prepare_one<R, 1, true>()};
  for (cudaError_t x : e)
    if (x != cudaSuccess) return x;
  return cudaSuccess;
}

// f(radius, kind, tma) with the three as compile-time constants
template <class Fn>
void dispatch(int R, int kind, bool tma, Fn f) {
  auto with_r = [&](auto r) {
    using std::integral_constant;
    if (kind == 0)
      tma ? f(r, integral_constant<int, 0>{}, std::true_type{}) : f(r, integral_constant<int, 0>{}, std::false_type{});
    else
      tma ? f(r, integral_constant<int, 1>{}, std::true_type{}) : f(r, integral_constant<int, 1>{}, std::false_type{});
  };
  switch (R) {
    case 1: with_r(std::integral_constant<int, 1>{}); break;
    case 2: with_r(std::integral_constant<int, 2>{}); break;
    case 3: with_r(std::integral_constant<int, 3>{}); break;
    case 4: with_r(std::integral_constant<int, 4>{}); break;
    case 5: with_r(std::integral_constant<int, 5>{}); break;
    default: break;
  }
}

}  // namespace

// ---- tensor maps (host): the encoder comes from the driver through the runtime's entry
// point query, so the library needs no link against the driver library
static PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    else
      cudaGetLastError();
  });
  return fn;
}

bool encode_volumes(CUtensorMap* m, const float* base, Dims n, int n_vol, int box_x, int box_y, int box_z) {
  const PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
  if (!enc || !base || n_vol < 1 || box_x > 256 || box_y > 256 || box_z < 1 || box_z > 256 || (box_x & 3))
    return false;
  if ((n.n2 & 3) || (reinterpret_cast<uintptr_t>(base) & 15)) return false;
  const cuuint64_t dims[4] = {(cuuint64_t)n.n2, (cuuint64_t)n.n1, (cuuint64_t)n.n0, (cuuint64_t)n_vol};
  const cuuint64_t row = (cuuint64_t)n.n2 * 4;
  const cuuint64_t strides[3] = {row, row * n.n1, row * n.n1 * n.n0};
  const cuuint32_t box[4] = {(cuuint32_t)box_x, (cuuint32_t)box_y, (cuuint32_t)box_z, 1};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  const CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<float*>(base), dims, strides, box, estr,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

namespace {
int staged_row(int R) {  // row pitch of the staged planes, Box<R>::PX
  switch (R) {
    case 1: return Box<1>::PX;
    case 2: return Box<2>::PX;
    case 3: return Box<3>::PX;
    case 4: return Box<4>::PX;
    case 5: return Box<5>::PX;
    default: return 0;
  }
}

// D chunk of one CTA: every chunk streams 2R planes more than it covers, so D is split only
// while one pair has fewer than 16384 threads and the launch (batch pairs) fewer than 1824
// CTAs (four waves of three CTAs on each of 152 SMs), and halved only while above min_chunk planes.
// The chunks are where the D sums restart, so this rule is part of the results.
int chunk_for(int ntiles, int depth, int min_chunk, int threads, int batch) {
  int tz = depth;
  for (;;) {
    const long chunks = (depth + tz - 1) / tz;
    if (tz <= min_chunk || (long)ntiles * chunks * threads >= 16384 || (long)batch * ntiles * chunks >= 1824) break;
    tz = (tz + 1) / 2;
  }
  return tz < 1 ? 1 : tz;
}

// D chunks of a launch of `tiles` tiles that should fill the device on its own (one pair of a
// stateless call). Every chunk streams 2R planes more than it covers, so fewer chunks do less work;
// more chunks fill more SMs. The cost of a chunking is its planes per CTA times the time of a plane at
// its CTAs per SM: c <= 4 resident CTAs take about 0.55 + 0.21 c us per plane (one 160 x 192 x 160
// pair, w = 7, forward: 0.97 us at 2, 1.39 us at 4), and more than 4 follow one another. That pair runs
// in 10 chunks (forward and adjoint 57 us), where the rule above takes 2 (148 us). The figures of w = 7
// serve every window and the statistics too: chunks are part of the results.
int filling_chunks(long tiles, int depth, int reach) {
  const long sms = device_sm_count();
  auto wave = [](long c) { return c ? 26 + 10 * c : 0; };
  int best = 1;
  long cost = 0;
  for (int c = 1; c <= depth && (c == 1 || tiles * c <= 8 * sms); ++c) {
    const long tz = (depth + c - 1) / c, per_sm = (tiles * c + sms - 1) / sms;
    const long k = (tz + reach + 1) * (per_sm / 4 * wave(4) + wave(per_sm % 4));
    if (c == 1 || k < cost) best = c, cost = k;
  }
  return best;
}

// batch 0: a stateless call. Its chunks may lie elsewhere than the engine's, for SiLNCC: LNCC's
// gradient follows the rounding of the window sums in flat regions, so it keeps the one rule.
int chunk_planes(int ntiles, Dims ni, int window, int kind, int min_chunk, int threads, int batch) {
  if (batch > 0 || kind != 0) return chunk_for(ntiles, ni.n0, min_chunk, threads, std::max(batch, 1));
  const int c = filling_chunks(ntiles, ni.n0, window - 1);
  return (ni.n0 + c - 1) / c;
}

Tiles sim_tiles(Dims ni, int window, int kind, int n_pairs, int batch, int group) {
  Tiles g;
  g.np = n_pairs;
  g.grp = std::max(1, std::min(group, n_pairs));
  g.gx = (ni.n2 + kTX - 1) / kTX;
  g.gy = (ni.n1 + kTY - 1) / kTY;
  g.tz = chunk_planes(g.gx * g.gy, ni, window, kind, 8, 256, batch);
  g.nzc = (ni.n0 + g.tz - 1) / g.tz;
  return g;
}
unsigned ctas(const Tiles& g) { return (unsigned)g.gx * g.gy * g.nzc * g.np; }
template <int R, int KIND>
void fixed_stats(dim3 g, const float* imgs, Dims ni, float eps, float* stats, int tz, int nzc, OpHead* head,
                 const PairDesc& pd, cudaStream_t s) {
  launch(k_fixed_stats<R, KIND>, g, StatCut<R, KIND>::threads, 0, s)(imgs, stats, ni, tz, nzc, eps, head, pd);
}
}  // namespace

void launch_fixed_stats(const float* imgs, int n_images, int batch, Dims ni, int window, int kind, float eps,
                        float* stats, cudaStream_t s, OpHead* head, const PairDesc& pd) {
  const int gx = (ni.n2 + TX - 1) / TX, gy = (ni.n1 + 7) / 8;
  const int tz = chunk_planes(gx * gy, ni, window, kind, 16, 128, batch), nzc = (ni.n0 + tz - 1) / tz;
  const dim3 g(gx, gy, nzc * n_images);
  dispatch(window / 2, kind, false, [&](auto r, auto k, auto) {
    fixed_stats<r(), k()>(g, imgs, ni, eps, stats, tz, nzc, head, pd, s);
  });
}

cudaError_t prepare_kernels() {
  // dynamic shared memory limits of the similarity kernels, once per device
  static std::mutex mu;
  static bool done[kMaxDevices] = {};
  return once_per_device(done, mu, [] {
    const cudaError_t e[5] = {prepare_r<1>(), prepare_r<2>(), prepare_r<3>(), prepare_r<4>(), prepare_r<5>()};
    for (cudaError_t x : e)
      if (x != cudaSuccess) return x;
    return cudaSuccess;
  });
}

SimGeom sim_geom(Dims ni, int window, int batch, int kind) {
  const Tiles g = sim_tiles(ni, window, kind, 1, batch, 1);
  return SimGeom{g.nzc, g.tz, (int)ctas(g)};
}
int sim_ncoef(int kind) { return kind == 0 ? 2 : 3; }

void make_sim_maps(SimMaps* m, const float* W, int n_pairs, const float* imgs, int n_images, const float* coef,
                   Dims ni, int window, int kind) {
  memset(m, 0, sizeof(*m));
  const int R = window / 2, px = staged_row(R), ry = kTY + 2 * R;
  if (!px) return;
  m->fwd_ok =
      encode_volumes(&m->W, W, ni, n_pairs, px, ry, 1) && encode_volumes(&m->F, imgs, ni, n_images, px, ry, 1);
  m->bwd_ok = encode_volumes(&m->C, coef, ni, n_pairs * sim_ncoef(kind), px, ry, 1);
}

void launch_sim_fwd(const PairDesc* pd, int n_pairs, int batch, int group, const float* W, size_t Wstride, float* coef,
                    size_t cs, double* partials, Dims ni, int window, int kind, float eps, const SimMaps* maps,
                    int* err, cudaStream_t s) {
  const Tiles g = sim_tiles(ni, window, kind, n_pairs, batch, group);
  dispatch(window / 2, kind, maps && maps->fwd_ok, [&](auto r, auto k, auto t) {
    launch(k_sim_fwd<r(), k(), t()>, ctas(g), Box<r()>::NT, Box<r()>::bytes(2, k() == 0 ? 2 : 3), s)(
        maps ? *maps : SimMaps{}, pd, W, Wstride, coef, cs, partials, ni, g, eps, err);
  });
}
void launch_sim_bwd(const PairDesc* pd, int n_pairs, int batch, int group, const float* W, size_t Wstride,
                    const float* coef, size_t cs, float* dLdW, Dims ni, int window, int kind, float scale,
                    const SimMaps* maps, int* err, cudaStream_t s) {
  const Tiles g = sim_tiles(ni, window, kind, n_pairs, batch, group);
  dispatch(window / 2, kind, maps && maps->bwd_ok, [&](auto r, auto k, auto t) {
    constexpr int nc = k() == 0 ? 2 : 3;
    launch(k_sim_bwd<r(), k(), t()>, ctas(g), Box<r()>::NT, Box<r()>::bytes(nc, nc), s)(
        maps ? *maps : SimMaps{}, pd, W, Wstride, coef, cs, dLdW, ni, g, scale, err);
  });
}

}  // namespace muster
