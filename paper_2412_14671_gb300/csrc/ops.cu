// ops.cu -- stateless entry points of include/muster_ops.h: single steps of the
// registration loop on caller-owned device buffers, running the engine's kernels.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <mutex>
#include <string>

#include "kernels.h"
#include "muster.h"
#include "muster_ops.h"

using namespace muster;

namespace {
thread_local std::string g_err;

int op_fail(int code, const std::string& m) {
  g_err = m;
  return code;
}
int op_cuda(cudaError_t e, const char* what) {
  return op_fail(MUSTER_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
}
#define OK_(call)                                    \
  do {                                               \
    cudaError_t e_ = (call);                         \
    if (e_ != cudaSuccess) return op_cuda(e_, #call); \
  } while (0)

bool dims_ok(int64_t D, int64_t H, int64_t W) {
  return D >= 1 && H >= 1 && W >= 1 && D <= 4096 && H <= 4096 && W <= 4096 && (double)D * H * W < 2147483647.0;
}
}  // namespace

// ---- scratch of the stateless calls: a memory pool of the library per device. The default pool gives
// everything back at each synchronisation, so a call that returns a number to the host paid for
// mapping its scratch again every time (about 200 us of the 290 us of a 48^3 similarity). This one
// keeps at most kPoolKeep bytes of unused scratch; after a failed allocation, of a call here or of a
// context (by cudaMalloc or its own callback), what the device has released goes back and the
// allocation is tried once more. Allocation and release are ordered by the caller's stream.
namespace {
constexpr uint64_t kPoolKeep = (uint64_t)256 << 20;
std::mutex g_pool_mu;
cudaMemPool_t g_pool[kMaxDevices] = {};

cudaMemPool_t op_pool() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
  std::lock_guard<std::mutex> lock(g_pool_mu);
  if (!g_pool[dev]) {
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.handleTypes = cudaMemHandleTypeNone;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t p = nullptr;
    uint64_t keep = kPoolKeep;
    if (cudaMemPoolCreate(&p, &props) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
    g_pool[dev] = p;
  }
  return g_pool[dev];
}
cudaError_t op_alloc(void** out, size_t bytes, cudaStream_t s) {
  // in a capture the graph owns the scratch, as an allocation node of the default pool
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) cudaGetLastError();
  const cudaMemPool_t pool = cap == cudaStreamCaptureStatusNone ? op_pool() : nullptr;
  if (!pool) return cudaMallocAsync(out, bytes, s);
  cudaError_t e = cudaMallocFromPoolAsync(out, bytes, pool, s);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    muster::trim_op_pools();
    e = cudaMallocFromPoolAsync(out, bytes, pool, s);
  }
  return e;
}
}  // namespace

namespace muster {
void trim_op_pools() {
  std::lock_guard<std::mutex> lock(g_pool_mu);
  for (cudaMemPool_t p : g_pool)
    if (p) cudaMemPoolTrimTo(p, 0);
}
void set_ops_error(const std::string& m) { g_err = m; }
}  // namespace muster

extern "C" {

const char* muster_ops_last_error(void) { return g_err.c_str(); }

int muster_op_downsample(const float* in, int n_images, int64_t D, int64_t H, int64_t W, float* out, void* stream) {
  if (!in || !out || n_images < 1) return op_fail(MUSTER_EINVAL, "bad arguments");
  if (!dims_ok(D, H, W)) return op_fail(MUSTER_EINVAL, "bad shape");
  const Dims n{(int)D, (int)H, (int)W}, m{(int)(D + 1) / 2, (int)(H + 1) / 2, (int)(W + 1) / 2};
  launch_down2(in, n, out, m, n_images, (cudaStream_t)stream);
  OK_(cudaGetLastError());
  return MUSTER_OK;
}

int muster_op_exp(const float* phi, int64_t D, int64_t H, int64_t W, int K, float sign, float* u, void* stream) {
  if (!phi || !u) return op_fail(MUSTER_EINVAL, "NULL pointer");
  if (!dims_ok(D, H, W)) return op_fail(MUSTER_EINVAL, "bad shape");
  if (K < 0 || K > 20) return op_fail(MUSTER_EINVAL, "K must be 0..20");
  if (sign != 1.f && sign != -1.f) return op_fail(MUSTER_EINVAL, "sign must be +1 or -1");
  cudaStream_t s = (cudaStream_t)stream;
  const Dims n{(int)D, (int)H, (int)W};
  const size_t V = vox(n);
  // u_0 = sign phi / 2^K, then K squarings, the last one into the caller's planar field
  float4* buf = nullptr;
  OK_(op_alloc((void**)&buf, sizeof(float4) * 2 * V, s));
  float4 *a = buf, *b = buf + V;
  launch_planar_to_f4(phi, a, 1, V, s, sign * ldexpf(1.f, -K));
  for (int t = 0; t + 1 < K; ++t) {
    launch_squaring(a, b, 1, n, s, 1);
    std::swap(a, b);
  }
  if (K > 0)
    launch_squaring_planar(a, u, n, s);
  else
    launch_f4_to_planar(a, u, 1, V, s);
  cudaError_t e = cudaGetLastError();
  cudaFreeAsync(buf, s);
  if (e != cudaSuccess) return op_cuda(e, "exp launches");
  return MUSTER_OK;
}

int muster_op_similarity(const float* F, const float* W, int64_t D, int64_t H, int64_t Wd, int window, int kind,
                         float eps, double* loss, float* dLdW, void* stream) {
  if (!F || !W) return op_fail(MUSTER_EINVAL, "NULL image");
  if (!dims_ok(D, H, Wd)) return op_fail(MUSTER_EINVAL, "bad shape");
  if (window < 3 || window > 11 || window % 2 == 0) return op_fail(MUSTER_EINVAL, "window must be odd, 3..11");
  if (kind != MUSTER_SILNCC && kind != MUSTER_LNCC) return op_fail(MUSTER_EINVAL, "unknown similarity");
  if (!(eps >= 0.f)) return op_fail(MUSTER_EINVAL, "eps must be >= 0");
  cudaStream_t s = (cudaStream_t)stream;
  const Dims n{(int)D, (int)H, (int)Wd};
  const size_t V = vox(n);
  const int64_t NR = (D - window + 1) < 1 || (H - window + 1) < 1 || (Wd - window + 1) < 1
                         ? 0
                         : (D - window + 1) * (H - window + 1) * (Wd - window + 1);
  if (NR == 0) {
    if (dLdW) OK_(cudaMemsetAsync(dLdW, 0, sizeof(float) * V, s));
    if (loss) {
      OK_(cudaStreamSynchronize(s));
      *loss = 0.0;
    }
    return MUSTER_OK;
  }
  const int NC = sim_ncoef(kind);
  const SimGeom g = sim_geom(n, window, 0, kind);
  // scratch: [head | partials | coefficients | F statistics]
  const size_t off_part = (sizeof(OpHead) + 255) / 256 * 256;
  const size_t off_coef = (off_part + sizeof(double) * (size_t)g.ctas + 255) / 256 * 256;
  const size_t off_stat = off_coef + sizeof(float) * NC * V;
  const size_t bytes = off_stat + sizeof(float) * 2 * V;
  char* buf = nullptr;
  OK_(op_alloc((void**)&buf, bytes, s));
  OpHead* d = (OpHead*)buf;
  double* part = (double*)(buf + off_part);
  float* coef = (float*)(buf + off_coef);
  float* stat = (float*)(buf + off_stat);
  OpHead h{};
  h.pd.Ii = F;
  h.pd.Fs = stat;
  SimMaps maps;
  make_sim_maps(&maps, W, 1, F, 1, coef, n, window, kind);
  cudaError_t e = prepare_kernels();
  if (e == cudaSuccess) {
    launch_fixed_stats(F, 1, 0, n, window, kind, eps, stat, s, d, h.pd);
    launch_sim_fwd(&d->pd, 1, 0, 1, W, V, coef, V, part, n, window, kind, eps, &maps, d->ints + 2, s);
    if (dLdW) {
      const int nw = window * window * window;
      const float scale = kind == MUSTER_SILNCC ? (float)(2.0 / ((double)nw * (double)NR)) : (float)(1.0 / (double)NR);
      launch_sim_bwd(&d->pd, 1, 0, 1, W, V, coef, V, dLdW, n, window, kind, scale, &maps, d->ints + 2, s);
    }
    launch_loss_reduce(part, g.ctas, nullptr, 0, 1.0 / (double)NR, 0.0, 0.0, 0.f, 0.f, 0.f, d->out, nullptr, d->ints,
                       d->ints + 1, 0, s);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && loss) e = cudaMemcpyAsync(&h, d, offsetof(OpHead, pd), cudaMemcpyDeviceToHost, s);
  cudaFreeAsync(buf, s);
  if (e != cudaSuccess) return op_cuda(e, "similarity launches");
  if (loss) {
    OK_(cudaStreamSynchronize(s));
    if (h.ints[2]) return op_fail(MUSTER_ETIMEOUT, "a bounded wait for an input copy ran out");
    *loss = h.out[1];
  }
  return MUSTER_OK;
}

int muster_op_jacobian_det(const float* u, int64_t D, int64_t H, int64_t Wd, float* J, void* stream) {
  if (!u || !J) return op_fail(MUSTER_EINVAL, "NULL field");
  if (!dims_ok(D, H, Wd)) return op_fail(MUSTER_EINVAL, "bad shape");
  launch_jacobian_det(u, Dims{(int)D, (int)H, (int)Wd}, J, (cudaStream_t)stream);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return op_cuda(e, "jacobian launch");
  return MUSTER_OK;
}

int muster_op_deformation_metrics(const float* u_true, const float* u_est, const uint8_t* roi, int64_t D, int64_t H,
                                  int64_t Wd, double out[16], void* stream) {
  if (!u_true || !u_est || !out) return op_fail(MUSTER_EINVAL, "NULL argument");
  if (!dims_ok(D, H, Wd)) return op_fail(MUSTER_EINVAL, "bad shape");
  cudaStream_t s = (cudaStream_t)stream;
  const size_t nd = metrics_scratch_doubles();
  double* buf = nullptr;
  OK_(op_alloc((void**)&buf, sizeof(double) * (nd + 16), s));
  launch_deformation_metrics(u_true, u_est, roi, Dims{(int)D, (int)H, (int)Wd}, buf, buf + nd, s);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpyAsync(out, buf + nd, sizeof(double) * 16, cudaMemcpyDeviceToHost, s);
  cudaFreeAsync(buf, s);
  if (e != cudaSuccess) return op_cuda(e, "metrics launches");
  OK_(cudaStreamSynchronize(s));
  return MUSTER_OK;
}

}  // extern "C"
