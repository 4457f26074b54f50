// m2l_keys.cu -- the distinct M2L translations of a plan.
//
// Expansion centres are octree box centres, so the translation of a pair is
// fixed by the level difference dl = l_T - l_S and an integer lattice offset I:
//   v = (c_T - c_S) / s_T = I 2^-(max(0, -dl) + 1),
//   I = (2 k_T + 1) - (2 k_S + 1) 2^dl  (dl >= 0),  (2 k_T + 1) 2^-dl - (2 k_S + 1)  otherwise
// (k = integer box coordinates).  A ball of 224k tets has ~8k distinct keys for
// ~870k pairs: operators and derivative tables are built once per key.
//
// Each pair's key is packed into 64 bits (dl + 32 in 6 bits, each offset + 2^18
// in 19), sorted, made unique and searched, all on the device.  Offsets beyond
// 19 bits (very small theta on deep trees) take the host map instead.
#include <algorithm>
#include <array>
#include <unordered_map>
#include <vector>

#include <cub/cub.cuh>

#include "common.cuh"

namespace demag {

namespace {

constexpr int KEY_OFF_BITS = 19;
constexpr int64_t KEY_OFF_HALF = 1ll << (KEY_OFF_BITS - 1);

__host__ __device__ inline void cell_coords(uint64_t prefix, int level, int64_t* k) {  // x bit at 3b
  k[0] = k[1] = k[2] = 0;
  for (int b = 0; b < level; b++)
    for (int a = 0; a < 3; a++) k[a] |= (int64_t)((prefix >> (3 * b + a)) & 1ull) << b;
}

__host__ __device__ inline void key_offset(const int64_t* kT, const int64_t* kS, int dl, int64_t* off) {
  for (int a = 0; a < 3; a++)
    off[a] = dl >= 0 ? (2 * kT[a] + 1) - ((2 * kS[a] + 1) << dl) : ((2 * kT[a] + 1) << (-dl)) - (2 * kS[a] + 1);
}

// block per target: the packed key of each of its pairs; *wide counts offsets beyond the packing
__global__ void k_pair_keys(const int32_t* __restrict__ targets, const int64_t* __restrict__ m2l_off,
                            const int32_t* __restrict__ m2l_src, const uint64_t* __restrict__ prefix,
                            const int32_t* __restrict__ level, uint64_t* keys, unsigned long long* wide) {
  const int32_t T = targets[blockIdx.x];
  int64_t kT[3];
  cell_coords(prefix[T], level[T], kT);
  for (int64_t e = m2l_off[T] + threadIdx.x; e < m2l_off[T + 1]; e += blockDim.x) {
    const int32_t S = m2l_src[e];
    const int dl = level[T] - level[S];
    int64_t kS[3], off[3];
    cell_coords(prefix[S], level[S], kS);
    key_offset(kT, kS, dl, off);
    uint64_t key = (uint64_t)(dl + 32);
    bool ok = true;
    for (int a = 0; a < 3; a++) {
      ok = ok && off[a] >= -KEY_OFF_HALF && off[a] < KEY_OFF_HALF;
      key = (key << KEY_OFF_BITS) | (uint64_t)((off[a] + KEY_OFF_HALF) & ((1ll << KEY_OFF_BITS) - 1));
    }
    keys[e] = key;
    if (!ok) atomicAdd(wide, 1ull);
  }
}

// position of every pair's key in the sorted distinct keys
__global__ void k_key_index(int64_t n, const uint64_t* __restrict__ keys, const uint64_t* __restrict__ uniq, int nu,
                            int32_t* op) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= n) return;
  const uint64_t k = keys[e];
  int lo = 0, hi = nu - 1;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (uniq[mid] < k)
      lo = mid + 1;
    else
      hi = mid;
  }
  op[e] = lo;
}

template <class T>
struct Buf {
  T* p = nullptr;
  explicit Buf(size_t n) {
    if (cudaMalloc(&p, std::max<size_t>(n, 1) * sizeof(T)) != cudaSuccess) {
      cudaGetLastError();
      fail(DEMAG_ERR_OUT_OF_MEMORY, "M2L key buffers");
    }
  }
  Buf(const Buf&) = delete;
  ~Buf() {
    if (p) cudaFree(p);
  }
};

struct KeyHash {
  size_t operator()(const std::array<int64_t, 4>& k) const {
    uint64_t h = 1469598103934665603ull;
    for (int64_t v : k) h = (h ^ (uint64_t)v) * 1099511628211ull;
    return (size_t)h;
  }
};

// the general form on the host: offsets of any size up to 32 bits
M2lKeys host_keys(Plan& P) {
  M2lKeys K;
  cudaStream_t s = P.stream;
  const int64_t nc = P.ncells;
  std::vector<uint64_t> prefix(nc);
  std::vector<int32_t> lev(nc), src(P.n_m2l), op(P.n_m2l);
  std::vector<int64_t> off(nc + 1);
  DM_CUDA(cudaMemcpyAsync(prefix.data(), P.cell_prefix, nc * sizeof(uint64_t), cudaMemcpyDeviceToHost, s));
  DM_CUDA(cudaMemcpyAsync(lev.data(), P.cell_level, nc * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  DM_CUDA(cudaMemcpyAsync(off.data(), P.m2l_off, (nc + 1) * sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  DM_CUDA(cudaMemcpyAsync(src.data(), P.m2l_src, P.n_m2l * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  DM_CUDA(cudaStreamSynchronize(s));
  std::vector<std::array<int64_t, 3>> kc(nc);
  for (int64_t c = 0; c < nc; c++) cell_coords(prefix[c], lev[c], kc[c].data());
  std::unordered_map<std::array<int64_t, 4>, int32_t, KeyHash> index;
  for (int64_t T = 0; T < nc; T++)
    for (int64_t e = off[T]; e < off[T + 1]; e++) {
      const int dl = lev[T] - lev[src[e]];
      std::array<int64_t, 4> key{dl, 0, 0, 0};
      key_offset(kc[T].data(), kc[src[e]].data(), dl, key.data() + 1);
      auto f = index.find(key);
      if (f == index.end()) {
        for (int a = 1; a < 4; a++)
          if (key[a] > INT32_MAX || key[a] < INT32_MIN) return M2lKeys{};  // beyond the table's key range
        f = index.emplace(key, (int32_t)K.keys.size()).first;
        K.keys.push_back(make_int4(dl, (int)key[1], (int)key[2], (int)key[3]));
      }
      op[e] = f->second;
    }
  P.m2l_op = dalloc<int32_t>(P, P.n_m2l);
  DM_CUDA(cudaMemcpyAsync(P.m2l_op, op.data(), P.n_m2l * sizeof(int32_t), cudaMemcpyHostToDevice, s));
  DM_CUDA(cudaStreamSynchronize(s));
  K.ok = true;
  return K;
}

}  // namespace

M2lKeys build_m2l_keys(Plan& P) {
  M2lKeys K;
  if (P.n_m2l == 0 || P.h_m2l_targets.empty()) return K;
  cudaStream_t s = P.stream;
  const int64_t n = P.n_m2l;
  std::vector<uint64_t> hk;
  {
    // one allocation: keys, sorted and distinct keys, two counters, sort workspace
    struct Counters {
      unsigned long long wide;  // offsets beyond the packing
      long long nu;             // distinct keys
    };
    const int bits = 6 + 3 * KEY_OFF_BITS;
    size_t b1 = 0, b2 = 0;
    uint64_t* none = nullptr;
    DM_CUDA(cub::DeviceRadixSort::SortKeys(nullptr, b1, none, none, n, 0, bits, s));
    DM_CUDA(cub::DeviceSelect::Unique(nullptr, b2, none, none, (long long*)nullptr, n, s));
    const size_t list = ((size_t)n * sizeof(uint64_t) + 255) / 256 * 256;
    Buf<unsigned char> buf(3 * list + 256 + std::max(b1, b2));
    uint64_t *keys = (uint64_t*)buf.p, *sorted = (uint64_t*)(buf.p + list), *uniq = (uint64_t*)(buf.p + 2 * list);
    Counters* cnt = (Counters*)(buf.p + 3 * list);
    unsigned char* tmp = buf.p + 3 * list + 256;
    DM_CUDA(cudaMemsetAsync(cnt, 0, sizeof(Counters), s));
    k_pair_keys<<<(unsigned)P.h_m2l_targets.size(), 128, 0, s>>>(P.m2l_targets, P.m2l_off, P.m2l_src, P.cell_prefix,
                                                                 P.cell_level, keys, &cnt->wide);
    DM_LAUNCH("k_pair_keys");
    DM_CUDA(cub::DeviceRadixSort::SortKeys(tmp, b1, keys, sorted, n, 0, bits, s));
    DM_CUDA(cub::DeviceSelect::Unique(tmp, b2, sorted, uniq, &cnt->nu, n, s));
    Counters h{};
    DM_CUDA(cudaMemcpyAsync(&h, cnt, sizeof h, cudaMemcpyDeviceToHost, s));
    DM_CUDA(cudaStreamSynchronize(s));
    if (h.wide == 0) {
      hk.resize(h.nu);
      DM_CUDA(cudaMemcpyAsync(hk.data(), uniq, h.nu * sizeof(uint64_t), cudaMemcpyDeviceToHost, s));
      P.m2l_op = dalloc<int32_t>(P, n);
      k_key_index<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, keys, uniq, (int)h.nu, P.m2l_op);
      DM_LAUNCH("k_key_index");
      DM_CUDA(cudaStreamSynchronize(s));
    }
  }
  if (hk.empty()) {
    K = host_keys(P);
  } else {
    for (uint64_t k : hk) {
      auto o = [&](int a) {
        return (int)((int64_t)((k >> (KEY_OFF_BITS * (2 - a))) & ((1ull << KEY_OFF_BITS) - 1)) - KEY_OFF_HALF);
      };
      K.keys.push_back(make_int4((int)(k >> (3 * KEY_OFF_BITS)) - 32, o(0), o(1), o(2)));
    }
    K.ok = true;
  }
  P.n_m2l_keys = K.ok ? (int64_t)K.keys.size() : 0;
  return K;
}

}  // namespace demag
