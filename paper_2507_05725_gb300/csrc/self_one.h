// One arc's self matrix outside a job: the tables its kernels read, packed into one block so that a call
// makes one host-to-device copy (six to nine small copies took longer than the assembly itself).
#pragma once
#include <cstring>

#include "kernels.h"

namespace fthms {

// Block layout (byte offsets): descriptors, 4 N node doubles (t, x, y, |x'|), then the tiles; the cosine sums of
// the log weights (N + 1 doubles, written on the device) follow the copied part.
constexpr size_t kSelfOneNodes = 256;
constexpr int self_one_edge(int N) { return (N + kSelfTile - 1) / kSelfTile; }
constexpr int self_one_tiles(int N) { return self_one_edge(N) * (self_one_edge(N) + 1) / 2; }
constexpr size_t self_one_tile_off(int N) { return kSelfOneNodes + 4 * (size_t)N * sizeof(double); }
constexpr size_t self_one_copy_bytes(int N) { return self_one_tile_off(N) + self_one_tiles(N) * sizeof(SelfTile); }
constexpr size_t self_one_rlog_off(int N) { return (self_one_copy_bytes(N) + 15) / 16 * 16; }
constexpr size_t self_one_bytes(int N) { return self_one_rlog_off(N) + ((size_t)N + 1) * sizeof(double); }

struct SelfOneHead {
  SysDesc sys;
  Panel panel;
  long long rlog_off;
  int rlogN;
};
static_assert(sizeof(SelfOneHead) <= kSelfOneNodes, "descriptors outgrow their slot");

// Descriptors and tiles into `host` (self_one_copy_bytes(N) bytes; the caller fills the 4 N node doubles).  One
// system in a band of length 1 at frequency index 1 with step h = kappa: the band kernel's kappa = l h,
// ln l = 0 and the recurrence step h R all refer to this kappa.
inline void self_one_pack(unsigned char* host, int N, double kappa) {
  SelfOneHead h{};
  h.sys.l = 1;
  h.sys.N = N;
  h.sys.kappa = kappa;
  h.panel = Panel{0, N, 0};
  h.rlogN = N;
  std::memcpy(host, &h, sizeof h);
  unsigned char* t = host + self_one_tile_off(N);
  const int nt = self_one_edge(N);
  for (int a = 0; a < nt; ++a)
    for (int b = a; b < nt; ++b, t += sizeof(SelfTile)) {
      const SelfTile tile{0, 1, a, b};
      std::memcpy(t, &tile, sizeof tile);
    }
}

// The kernels' view of a block at device address `base` (16-byte aligned).
inline void self_one_bind(DevJob& J, unsigned char* base, int N, double kappa, double* A_dev) {
  const SelfOneHead* h = reinterpret_cast<const SelfOneHead*>(base);
  const double* nd = reinterpret_cast<const double*>(base + kSelfOneNodes);
  J.node_t = nd;
  J.node_x = nd + N;
  J.node_y = nd + 2 * N;
  J.node_sp = nd + 3 * N;
  J.sys = &h->sys;
  J.panels = &h->panel;
  J.rlogN = &h->rlogN;
  J.rlog_off_N = &h->rlog_off;
  J.tiles = reinterpret_cast<const SelfTile*>(base + self_one_tile_off(N));
  J.rlog = reinterpret_cast<double*>(base + self_one_rlog_off(N));
  J.A = reinterpret_cast<double2*>(A_dev);
  J.h = kappa;
  J.n_rlogN = 1;
  J.n_tiles = self_one_tiles(N);
  J.max_n = N;
  J.K = 16;   // unused FFT tables are not launched
}

}  // namespace fthms
