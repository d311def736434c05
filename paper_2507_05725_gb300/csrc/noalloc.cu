// fthms_assemble_self_noalloc: the self-matrix assembly of fthms_assemble_self without any device
// allocation.  Its temporary device data (node coordinates, the log weights' cosine sums, the tile and system
// descriptors) live in one file-scope device array that every GPU loading the library holds until the
// process exits.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>

#include "fthms.h"
#include "kernels.h"
#include "self_one.h"

namespace {

using namespace fthms;

constexpr int kNoallocMaxN = 256;                       // largest N accepted
constexpr size_t kScratchBytes = self_one_bytes(kNoallocMaxN);   // ~13 KB

static __device__ __align__(256) unsigned char g_scratch[kScratchBytes];

std::mutex g_mu;
unsigned char* g_scratch_dev[64] = {};   // device address of g_scratch per device (set-up once)

fthms_status fail_msg(fthms_status s, const char* msg) {
  set_last_error(msg);
  return s;
}

fthms_status cuda_msg(cudaError_t e, const char* what) {
  char buf[256];
  std::snprintf(buf, sizeof buf, "%s: %s", what, cudaGetErrorString(e));
  set_last_error(buf);
  return FTHMS_ECUDA;
}

// Per-device set-up, done by the first call on each device with that device current: the device
// address of g_scratch (host code only has a host-side stand-in for the symbol) and the Bessel tables.
fthms_status scratch_address(int dev, unsigned char** out) {
  std::lock_guard<std::mutex> lk(g_mu);
  if (dev < 0 || dev >= 64) return fail_msg(FTHMS_EINVAL, "fthms_assemble_self_noalloc: device index >= 64");
  if (!g_scratch_dev[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_scratch);
    if (e != cudaSuccess) return cuda_msg(e, "cudaGetSymbolAddress(no-alloc scratch)");
    e = init_constants(dev);
    if (e != cudaSuccess) return cuda_msg(e, "init_constants");
    g_scratch_dev[dev] = static_cast<unsigned char*>(p);
  }
  *out = g_scratch_dev[dev];
  return FTHMS_OK;
}

void curve_eval(const fthms_curve* c, double th, double& x, double& y, double& dx, double& dy) {
  x = y = dx = dy = 0.0;
  for (int k = 0; k <= c->degree; ++k) {
    const double cs = std::cos(k * th), sn = std::sin(k * th);
    x += c->ax[k] * cs + c->bx[k] * sn;
    y += c->ay[k] * cs + c->by[k] * sn;
    dx += k * (-c->ax[k] * sn + c->bx[k] * cs);
    dy += k * (-c->ay[k] * sn + c->by[k] * cs);
  }
}

}  // namespace

extern "C" fthms_status fthms_assemble_self_noalloc(const fthms_curve* curve, const fthms_arc* arc, int N,
                                                    double kappa, double* A_dev, void* cuda_stream) {
  if (!curve || !arc || !A_dev || !curve->ax || !curve->bx || !curve->ay || !curve->by || curve->degree < 1 ||
      !(kappa > 0) || !(arc->theta_b > arc->theta_a))
    return fail_msg(FTHMS_EINVAL, "fthms_assemble_self_noalloc: bad arguments");
  if (N < 2 || N > kNoallocMaxN)
    return fail_msg(FTHMS_EINVAL, "fthms_assemble_self_noalloc: N must be in [2, 256] (size of the static scratch)");
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_msg(e, "cudaGetDevice");
  unsigned char* base = nullptr;
  fthms_status s = scratch_address(dev, &base);
  if (s != FTHMS_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);

  // Host-side tables on the stack (no heap, no device allocation).  A copy from pageable host memory
  // has been staged by the time cudaMemcpyAsync returns, so this buffer may go out of scope; the kernels stay
  // queued on the stream.  Every byte that the kernels read is overwritten here or by k_rlog and every
  // entry of A is written, so nothing carried over from an earlier call is used and nothing needs clearing.
  alignas(16) unsigned char host[self_one_copy_bytes(kNoallocMaxN)];
  self_one_pack(host, N, kappa);
  double* nodes = reinterpret_cast<double*>(host + kSelfOneNodes);
  const double tc = 0.5 * (arc->theta_a + arc->theta_b), half = 0.5 * (arc->theta_b - arc->theta_a);
  for (int i = 0; i < N; ++i) {
    const double t = std::cos((2.0 * i + 1.0) * 3.14159265358979323846 / (2.0 * N));
    double x, y, dx, dy;
    curve_eval(curve, tc + half * t, x, y, dx, dy);
    nodes[i] = t;
    nodes[N + i] = x;
    nodes[2 * N + i] = y;
    nodes[3 * N + i] = std::hypot(dx, dy) * half;
  }
  e = cudaMemcpyAsync(base, host, self_one_copy_bytes(N), cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return cuda_msg(e, "cudaMemcpyAsync(no-alloc scratch)");
  DevJob J{};
  self_one_bind(J, base, N, kappa, A_dev);
  int nl = 0;
  e = launch_tables_rlog_only(J, st, &nl);
  if (e == cudaSuccess) e = launch_assemble_self(J, st, &nl);
  if (e != cudaSuccess) return cuda_msg(e, "fthms_assemble_self_noalloc launch");
  return FTHMS_OK;
}
