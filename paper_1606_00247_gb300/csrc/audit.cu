// audit.cu -- bounds audit of the plan's index lists, on the device.
//
// Every list that an evaluation kernel follows into another array (node and
// tet permutations, cell links and ranges, the CSR interaction lists of
// Sec. 3.3, support nodes, near-field columns and tile rows, M2L operator
// indices and groups, gradient-operator columns, the parts of the integrated near
// field's clusters, translation entries) is written once, while the plan is built,
// and only read afterwards.  Checking each entry once here is
// therefore the same guarantee as a bounds check at every read, at no cost to
// an evaluation, and without a device assert (which would end the context).
// Each list's count is first checked against the size of the allocation it
// lives in (a list whose count runs past it is reported, not read).
// A failed check is a planner bug: the plan is not returned and
// demag_last_error() names the list, the first bad position and its value.
#include <climits>
#include <cstring>
#include <string>
#include <vector>

#include "common.cuh"

namespace demag {

namespace {

struct AuditOut {
  unsigned long long bad;    // entries that failed
  unsigned long long first;  // first failing position (ULLONG_MAX: none)
};

__device__ __forceinline__ void audit_fail(AuditOut* o, int64_t i) {
  atomicAdd(&o->bad, 1ull);
  atomicMin(&o->first, (unsigned long long)i);
}

// lo <= (a[i] & mask) < hi for every i < n (mask = -1: the value itself)
template <class T>
__global__ void k_audit_values(const T* __restrict__ a, int64_t n, int64_t mask, int64_t lo, int64_t hi, AuditOut* o) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = (int64_t)a[i] & mask;
    if (v < lo || v >= hi) audit_fail(o, i);
  }
}

// n + 1 non-decreasing offsets within [lo, hi]; first = off[0] and last = off[n] when >= 0
__global__ void k_audit_offsets(const int64_t* __restrict__ off, int64_t n, int64_t lo, int64_t hi, int64_t first,
                                int64_t last, AuditOut* o) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i <= n; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = off[i];
    bool ok = v >= lo && v <= hi;
    if (i < n) ok = ok && v <= off[i + 1];
    if (i == 0 && first >= 0) ok = ok && v == first;
    if (i == n && last >= 0) ok = ok && v == last;
    if (!ok) audit_fail(o, i);
  }
}

// cell ranges: 0 <= tet begin <= tet end <= nt, 0 <= node begin <= node end <= nn
__global__ void k_audit_ranges(const int4* __restrict__ r, int64_t n, int64_t nt, int64_t nn, AuditOut* o) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int4 v = r[i];
    if (!(0 <= v.x && v.x <= v.y && v.y <= nt && 0 <= v.z && v.z <= v.w && v.w <= nn)) audit_fail(o, i);
  }
}

// child links: 0 <= nchild <= 8; children of a parent lie after it and inside the cell array
__global__ void k_audit_children(const int32_t* __restrict__ child0, const int32_t* __restrict__ nchild, int64_t n,
                                 AuditOut* o) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int k = nchild[i];
    if (k < 0 || k > 8 || (k > 0 && (child0[i] <= i || (int64_t)child0[i] + k > n))) audit_fail(o, i);
  }
}

// blocks of the integrated near field: a target, 1 .. PF_G of its leaf's nodes
__global__ void k_audit_blocks(const int4* __restrict__ blk, int64_t n, const int32_t* __restrict__ targets, int64_t nT,
                               const int4* __restrict__ range, AuditOut* o) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int4 b = blk[i];
    bool ok = b.x >= 0 && b.x < nT && b.z >= 1 && b.z <= PF_G;
    if (ok) {
      const int4 r = range[targets[b.x]];
      ok = b.y >= r.z && (int64_t)b.y + b.z <= r.w;
    }
    if (!ok) audit_fail(o, i);
  }
}

// clusters: 1 .. CL_V vertices, CL_E edges, CL_F faces, boundary faces among them, each part inside its array
__global__ void k_audit_clusters(const int4* __restrict__ cnt, const int4* __restrict__ pos, int64_t n, int64_t nv,
                                 int64_t ne, int64_t nf, int64_t nb, AuditOut* o) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int4 c = cnt[i], p = pos[i];
    const bool ok = c.x >= 1 && c.x <= CL_V && c.y >= 1 && c.y <= CL_E && c.z >= 1 && c.z <= CL_F && c.w >= 0 &&
                    c.w <= c.z && p.x >= 0 && (int64_t)p.x + c.x <= nv && p.y >= 0 && (int64_t)p.y + c.y <= ne &&
                    p.z >= 0 && (int64_t)p.z + c.z <= nf && p.w >= 0 && (int64_t)p.w + c.w <= nb;
    if (!ok) audit_fail(o, i);
  }
}

// packed positions of a cluster's edges (two vertices) and faces (three vertices, three edges) below its
// counts; the failing position is that of the edge or face.  One block per cluster (checked before).
__global__ void k_audit_cluster_edges(const int4* __restrict__ cnt, const int4* __restrict__ pos,
                                      const uint32_t* __restrict__ edge, int64_t ne, AuditOut* o) {
  const int4 c = cnt[blockIdx.x], p = pos[blockIdx.x];
  for (int t = threadIdx.x; t < c.y && t < CL_E; t += blockDim.x) {
    const int64_t q = (int64_t)p.y + t;
    if (q < 0 || q >= ne) continue;  // reported by k_audit_clusters
    if ((int)(edge[q] & 0xFFFFu) >= c.x || (int)(edge[q] >> 16) >= c.x) audit_fail(o, q);
  }
}
__global__ void k_audit_cluster_faces(const int4* __restrict__ cnt, const int4* __restrict__ pos,
                                      const uint2* __restrict__ fidx, int64_t nf, AuditOut* o) {
  const int4 c = cnt[blockIdx.x], p = pos[blockIdx.x];
  for (int t = threadIdx.x; t < c.z && t < CL_F; t += blockDim.x) {
    const int64_t q = (int64_t)p.z + t;
    if (q < 0 || q >= nf) continue;
    bool ok = true;
    for (int k = 0; k < 3; k++)
      ok = ok && (int)((fidx[q].x >> (8 * k)) & 255u) < c.x && (int)((fidx[q].y >> (9 * k)) & 511u) < c.y;
    if (!ok) audit_fail(o, q);
  }
}

// entries of an octree translation: position below hi
template <class T>
__global__ void k_audit_entries(const TEnt<T>* __restrict__ ent, int64_t n, int hi, AuditOut* o) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    if (ent[i].k >= hi) audit_fail(o, i);
}

// items of the table M2L: table positions up to the zero at nc, the chunk's moments within the padded block
__global__ void k_audit_items(const TabItem* __restrict__ it, int64_t n, int nc, int nchunk, AuditOut* o) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    bool ok = it[i].chunk >= 0 && it[i].chunk < nchunk;
    for (int k = 0; k < TAB_TR * TAB_TC; k++) ok = ok && it[i].idx[k] <= nc;
    if (!ok) audit_fail(o, i);
  }
}

// ranges [x, y) within [0, hi]
__global__ void k_audit_spans(const int2* __restrict__ r, int64_t n, int hi, AuditOut* o) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    if (!(0 <= r[i].x && r[i].x <= r[i].y && r[i].y <= hi)) audit_fail(o, i);
}

// a scratch copy of a device list with one entry replaced, freed on scope exit (test hook)
template <class T>
struct Planted {
  T* p = nullptr;
  Planted(const T* list, int64_t n, int64_t at, T value, cudaStream_t s) {
    if (cudaMalloc(&p, sizeof(T) * (size_t)n) != cudaSuccess) {
      cudaGetLastError();
      fail(DEMAG_ERR_OUT_OF_MEMORY, "plan audit scratch");
    }
    DM_CUDA(cudaMemcpyAsync(p, list, sizeof(T) * n, cudaMemcpyDeviceToDevice, s));
    DM_CUDA(cudaMemcpyAsync(p + at, &value, sizeof value, cudaMemcpyHostToDevice, s));
    DM_CUDA(cudaStreamSynchronize(s));
  }
  Planted(const Planted&) = delete;
  ~Planted() {
    if (p) cudaFree(p);
  }
};

template <class T>
T entry(const T* list, int64_t at) {
  T v{};
  DM_CUDA(cudaMemcpy(&v, list + at, sizeof v, cudaMemcpyDeviceToHost));
  return v;
}

struct Check {
  std::string name;
  const void* ptr;
  int esize;  // bytes of one entry (its value is read back for the message), 0 = none
};

class Auditor {
 public:
  explicit Auditor(Plan& P) : P_(P), s_(P.stream) {}

  template <class T>
  void values(const char* name, const T* a, int64_t n, int64_t lo, int64_t hi, int64_t mask = -1) {
    if (!begin(name, a, n, sizeof(T), n * (int64_t)sizeof(T))) return;
    k_audit_values<T><<<grid(n), 256, 0, s_>>>(a, n, mask, lo, hi, out(name));
    DM_LAUNCH("k_audit_values");
  }
  void offsets(const char* name, const int64_t* off, int64_t n, int64_t lo, int64_t hi, int64_t first, int64_t last) {
    if (!begin(name, off, n + 1, sizeof(int64_t), (n + 1) * (int64_t)sizeof(int64_t))) return;
    k_audit_offsets<<<grid(n + 1), 256, 0, s_>>>(off, n, lo, hi, first, last, out(name));
    DM_LAUNCH("k_audit_offsets");
  }
  void ranges(const char* name, const int4* r, int64_t n) {
    if (!begin(name, r, n, 0, n * (int64_t)sizeof(int4))) return;
    k_audit_ranges<<<grid(n), 256, 0, s_>>>(r, n, P_.nt, P_.nn, out(name));
    DM_LAUNCH("k_audit_ranges");
  }
  void children(const char* name, const int32_t* child0, const int32_t* nchild, int64_t n) {
    if (!begin(name, child0, n, 0, n * (int64_t)sizeof(int32_t))) return;
    k_audit_children<<<grid(n), 256, 0, s_>>>(child0, nchild, n, out(name));
    DM_LAUNCH("k_audit_children");
  }
  void blocks(const char* name, const int4* blk, int64_t n) {
    if (!begin(name, blk, n, 0, n * (int64_t)sizeof(int4))) return;
    k_audit_blocks<<<grid(n), 256, 0, s_>>>(blk, n, P_.p2p_targets, (int64_t)P_.h_p2p_targets.size(), P_.cell_range,
                                            out(name));
    DM_LAUNCH("k_audit_blocks");
  }
  void clusters(const char* name, const int4* cnt, const int4* pos, int64_t n) {
    if (!begin(name, cnt, n, 0, n * (int64_t)sizeof(int4))) return;
    k_audit_clusters<<<grid(n), 256, 0, s_>>>(cnt, pos, n, P_.n_cl_v, P_.n_cl_e, P_.n_cl_f, P_.n_cl_b, out(name));
    DM_LAUNCH("k_audit_clusters");
  }
  void cluster_edges(const char* name, const uint32_t* edge, int64_t n) {
    if (!begin(name, edge, n, 0, n * (int64_t)sizeof(uint32_t))) return;
    k_audit_cluster_edges<<<(unsigned)P_.n_clusters, 128, 0, s_>>>(P_.cl_cnt, P_.cl_pos, edge, n, out(name));
    DM_LAUNCH("k_audit_cluster_edges");
  }
  void cluster_faces(const char* name, const uint2* fidx, int64_t n) {
    if (!begin(name, fidx, n, 0, n * (int64_t)sizeof(uint2))) return;
    k_audit_cluster_faces<<<(unsigned)P_.n_clusters, 128, 0, s_>>>(P_.cl_cnt, P_.cl_pos, fidx, n, out(name));
    DM_LAUNCH("k_audit_cluster_faces");
  }
  template <class T>
  void entries(const char* name, const TEnt<T>* ent, int64_t n, int hi) {
    if (!begin(name, ent, n, 0, n * (int64_t)sizeof(TEnt<T>))) return;
    k_audit_entries<T><<<grid(n), 256, 0, s_>>>(ent, n, hi, out(name));
    DM_LAUNCH("k_audit_entries");
  }
  void items(const char* name, const TabItem* it, int64_t n) {
    if (!begin(name, it, n, 0, n * (int64_t)sizeof(TabItem))) return;
    k_audit_items<<<grid(n), 256, 0, s_>>>(it, n, P_.nc, (P_.nq + TAB_TC - 1) / TAB_TC, out(name));
    DM_LAUNCH("k_audit_items");
  }
  void spans(const char* name, const int2* r, int64_t n, int hi) {
    if (!begin(name, r, n, 0, n * (int64_t)sizeof(int2))) return;
    k_audit_spans<<<grid(n), 256, 0, s_>>>(r, n, hi, out(name));
    DM_LAUNCH("k_audit_spans");
  }
  // the last of n + 1 device offsets (the length of the list they index)
  int64_t last(const int64_t* off, int64_t n) {
    int64_t v = 0;
    if (!off) return 0;
    DM_CUDA(cudaMemcpyAsync(&v, off + n, sizeof v, cudaMemcpyDeviceToHost, s_));
    DM_CUDA(cudaStreamSynchronize(s_));
    return v;
  }

  // the first failed check ("": none); ends this auditor's checks
  std::string report() {
    std::string msg;
    if (!checks_.empty()) {
      std::vector<AuditOut> h(checks_.size());
      DM_CUDA(cudaMemcpyAsync(h.data(), dout_, sizeof(AuditOut) * h.size(), cudaMemcpyDeviceToHost, s_));
      DM_CUDA(cudaStreamSynchronize(s_));
      for (size_t k = 0; k < h.size() && msg.empty(); k++) {
        if (h[k].bad == 0) continue;
        const Check& c = checks_[k];
        msg = "plan audit: " + c.name + "[" + std::to_string(h[k].first) + "]";
        if (c.esize == 4 || c.esize == 8) {
          int64_t v = 0;
          int32_t v32 = 0;
          const char* src = (const char*)c.ptr + h[k].first * (unsigned long long)c.esize;
          DM_CUDA(cudaMemcpy(c.esize == 4 ? (void*)&v32 : (void*)&v, src, c.esize, cudaMemcpyDeviceToHost));
          msg += " = " + std::to_string(c.esize == 4 ? (int64_t)v32 : v);
        }
        msg += " out of range (" + std::to_string(h[k].bad) + " entries)";
      }
    }
    if (msg.empty()) msg = error_;
    release();
    return msg;
  }
  void finish() {
    const std::string msg = report();
    if (!msg.empty()) fail(DEMAG_ERR_INTERNAL, msg);
  }
  ~Auditor() { release(); }

 private:
  static unsigned grid(int64_t n) { return (unsigned)std::min<int64_t>(std::max<int64_t>((n + 255) / 256, 1), 4096); }

  // size of the plan allocation that starts at p (0: not a plan allocation)
  size_t alloc_bytes(const void* p) const {
    for (const DevBuf& b : P_.bufs)
      if (b.ptr == p) return b.bytes;
    return 0;
  }

  bool begin(const char* name, const void* p, int64_t n, int esize, int64_t bytes) {
    if (n <= 0) return false;
    if (!p) {
      if (error_.empty()) error_ = std::string("plan audit: ") + name + " is missing (" + std::to_string(n) + " entries)";
      return false;
    }
    const size_t cap = alloc_bytes(p);
    if (cap && (size_t)bytes > cap) {  // the list's own count runs past its allocation: not read
      if (error_.empty())
        error_ = std::string("plan audit: ") + name + " counts " + std::to_string(n) + " entries, its allocation " +
                 std::to_string(cap) + " bytes";
      return false;
    }
    checks_.push_back(Check{name, p, esize});
    return true;
  }

  AuditOut* out(const char*) {
    const size_t k = checks_.size() - 1;
    if (k >= cap_) {  // grow the result array (results of earlier checks are still in flight)
      const size_t nc = std::max<size_t>(64, 2 * cap_);
      AuditOut* d = nullptr;
      if (cudaMalloc(&d, sizeof(AuditOut) * nc) != cudaSuccess) {
        cudaGetLastError();
        fail(DEMAG_ERR_OUT_OF_MEMORY, "plan audit buffers");
      }
      const std::vector<AuditOut> init(nc, AuditOut{0ull, ULLONG_MAX});
      DM_CUDA(cudaMemcpyAsync(d, init.data(), sizeof(AuditOut) * nc, cudaMemcpyHostToDevice, s_));
      if (dout_) DM_CUDA(cudaMemcpyAsync(d, dout_, sizeof(AuditOut) * cap_, cudaMemcpyDeviceToDevice, s_));
      DM_CUDA(cudaStreamSynchronize(s_));
      if (dout_) cudaFree(dout_);
      dout_ = d;
      cap_ = nc;
    }
    return dout_ + k;
  }

  void release() {
    if (dout_) cudaFree(dout_);
    dout_ = nullptr;
    cap_ = 0;
    checks_.clear();
    error_.clear();
  }

  Plan& P_;
  cudaStream_t s_;
  std::vector<Check> checks_;
  AuditOut* dout_ = nullptr;
  size_t cap_ = 0;
  std::string error_;
};

template <class T>
void audit_translations(Plan& P, Auditor& A) {
  A.entries("m2m_ent", (const TEnt<T>*)P.m2m_ent, (int64_t)P.m2m_width * P.nq, 8 * P.nq);
  A.entries("l2l_ent", (const TEnt<T>*)P.l2l_ent, P.l2l_nent, P.nl);
}

// test hook: lists of every kind as scratch copies with one entry out of range (read by the audit only, the
// plan's own lists are untouched); the reports of all of them
std::string planted(Plan& P, Auditor& A) {
  std::string all = A.report();
  cudaStream_t s = P.stream;
  auto add = [&] {
    const std::string m = A.report();
    all += (all.empty() || m.empty() ? "" : "; ") + m;
  };
  if (P.n_clusters > 0 && P.n_pc_blk > 0) {
    const int64_t c = P.n_clusters - 1;
    const int4 cnt = entry(P.cl_cnt, c), pos = entry(P.cl_pos, c);
    Planted<int4> n(P.cl_cnt, P.n_clusters, c, make_int4(cnt.x, cnt.y, CL_F + 1, cnt.w), s);
    A.clusters("cl_cnt (planted copy)", n.p, P.cl_pos, P.n_clusters);
    add();
    Planted<uint32_t> e(P.cl_edge, P.n_cl_e, pos.y, entry(P.cl_edge, pos.y) | (uint32_t)cnt.x << 16, s);
    A.cluster_edges("cl_edge (planted copy)", e.p, P.n_cl_e);
    add();
    Planted<uint2> f(P.cl_fidx, P.n_cl_f, pos.z, make_uint2(entry(P.cl_fidx, pos.z).x, 511u << 18), s);
    A.cluster_faces("cl_fidx (planted copy)", f.p, P.n_cl_f);
    add();
    const int4 b = entry(P.pc_blk, P.n_pc_blk - 1);
    Planted<int4> k(P.pc_blk, P.n_pc_blk, P.n_pc_blk - 1, make_int4(b.x, b.y, PF_G + 1, 0), s);
    A.blocks("pc_blk (planted copy)", k.p, P.n_pc_blk);
    add();
  }
  if (P.l2l_nent > 0) {
    Planted<int2> r(P.l2l_cls, 8 * P.nl, 0, make_int2(0, P.l2l_nent + 1), s);
    A.spans("l2l_cls (planted copy)", r.p, 8 * P.nl, P.l2l_nent);
    add();
  }
  if (P.m2l_tab_nitems > 0) {
    TabItem it = entry(P.m2l_tab_items, 0);
    it.idx[0] = (uint16_t)(P.nc + 1);
    Planted<TabItem> t(P.m2l_tab_items, P.m2l_tab_nitems, 0, it, s);
    A.items("m2l_tab_items (planted copy)", t.p, P.m2l_tab_nitems);
    add();
  }
  if (P.n_m2l > 0) {
    Planted<int32_t> m(P.m2l_src, P.n_m2l, P.n_m2l - 1, (int32_t)P.ncells, s);
    A.values("m2l_src (planted copy)", m.p, P.n_m2l, 0, P.ncells);
    add();
  }
  return all;
}

}  // namespace

void audit_plan(Plan& P, bool plant) {
  Auditor A(P);
  const int64_t nn = P.nn, nt = P.nt, nc = P.ncells;
  // sorted geometry and the octree (Sec. 3.1)
  A.values("node_perm", P.node_perm, nn, 0, nn);
  A.values("tet_perm", P.tet_perm, nt, 0, nt);
  A.values("tets_s", P.tets_s, 4 * nt, 0, nn);
  A.values("cell_level", P.cell_level, nc, 0, MAX_LEVEL + 1);
  A.values("cell_parent", P.cell_parent, nc, -1, nc);
  A.ranges("cell_range", P.cell_range, nc);
  A.children("cell_child0", P.cell_child0, P.cell_nchild, nc);
  A.values("node_leaf", P.node_leaf, nn, 0, nc);
  A.values("node_leaves", P.node_leaves, P.n_node_leaves, 0, nc);
  A.values("src_leaves", P.src_leaves, (int64_t)P.h_src_leaves.size(), 0, nc);
  A.offsets("nt_off", P.nt_off, nn, 0, 4 * nt, 0, 4 * nt);
  A.values("nt_tet", P.nt_tet, 4 * nt, 0, nt);
  // interaction lists (Sec. 3.3)
  A.offsets("m2l_off", P.m2l_off, nc, 0, P.n_m2l, 0, P.n_m2l);
  A.values("m2l_src", P.m2l_src, P.n_m2l, 0, nc);
  A.offsets("p2p_off", P.p2p_off, nc, 0, P.n_p2p, 0, P.n_p2p);
  A.values("p2p_src", P.p2p_src, P.n_p2p, 0, nc);
  A.values("m2l_targets", P.m2l_targets, (int64_t)P.h_m2l_targets.size(), 0, nc);
  A.values("p2p_targets", P.p2p_targets, (int64_t)P.h_p2p_targets.size(), 0, nc);
  // source-leaf supports (P2M)
  A.offsets("sup_off", P.sup_off, nc, 0, P.n_sup, 0, P.n_sup);
  A.values("sup_node", P.sup_node, P.n_sup, 0, nn);
  // stored near field
  if (P.opt.near_mode == 1) {
    const int64_t nT = (int64_t)P.h_p2p_targets.size();
    A.offsets("w_coloff", P.w_coloff, nT, 0, P.n_wcols, 0, P.n_wcols);
    A.offsets("w_off", P.w_off, nT, 0, P.n_wentries, 0, P.n_wentries);
    if (P.nf_ntiles > 0) {
      const int64_t nq = P.nf_ntiles;
      A.values("nf_cols", P.nf_cols, P.nf_ncols, 0, nn);
      A.values("nf_rownode", P.nf_rownode, nq * NF_ROWS, -1, nn);
      A.values("nf_order", P.nf_order, nq, 0, nq);
      A.values("nf_coff", P.nf_coff, nq, 0, P.nf_ncols + 1);
      A.values("nf_woff", P.nf_woff, nq, 0, P.nf_wbytes + 1);
      A.values("nf_ng", P.nf_ng, nq, 0, P.nf_ncols / 16 + 1);
      A.values("nf_npad", P.nf_npad, nq, 0, NF_ROWS + 1);
    } else {
      A.values("w_cols", P.w_cols, P.n_wcols, 0, nn);
      if (P.w_off32) A.offsets("w_off32", P.w_off32, nT, 0, P.n_wentries / 3 * 4, 0, P.n_wentries / 3 * 4);
    }
  }
  // integrated near field: clusters and their parts
  if (P.n_clusters > 0) {
    const int64_t nT = (int64_t)P.h_p2p_targets.size();
    A.values("cl_off", P.cl_off, nc + 1, 0, P.n_clusters + 1);
    A.values("cl_vnode", P.cl_vnode, P.n_cl_v, 0, nn);
    A.values("cl_ftet", (const int32_t*)P.cl_ftet, 2 * P.n_cl_f, -1, nt);
    A.clusters("cl_cnt", P.cl_cnt, P.cl_pos, P.n_clusters);
    A.cluster_edges("cl_edge", P.cl_edge, P.n_cl_e);
    A.cluster_faces("cl_fidx", P.cl_fidx, P.n_cl_f);
    A.blocks("pc_blk", P.pc_blk, P.n_pc_blk);
    if (P.pc_off) {
      A.offsets("pc_off", P.pc_off, nT, 0, P.n_pc, 0, P.n_pc);
      A.values("pc_src", P.pc_src, P.n_pc, 0, P.n_clusters);
    }
  }
  // far field: parent lists, M2L operator indices
  A.values("par_list", P.par_list, P.par_start.empty() ? 0 : P.par_start.back(), 0, nc);
  A.values("m2m_cnt", P.m2m_cnt, P.nq, 0, P.m2m_width + 1);
  A.spans("l2l_cls", P.l2l_cls, 8 * P.nl, P.l2l_nent);
  if (P.opt.precision == DEMAG_FP64)
    audit_translations<double>(P, A);
  else
    audit_translations<float>(P, A);
  if (P.m2l_op) A.values("m2l_op", P.m2l_op, P.n_m2l, 0, P.n_m2l_keys);
  if (P.m2l_tab_opdl) A.values("m2l_tab_opdl", P.m2l_tab_opdl, P.n_m2l, 0, P.n_m2l_keys, 0x00ffffff);
  A.items("m2l_tab_items", P.m2l_tab_items, P.m2l_tab_nitems);
  // mixed path: gradient operator, M2L groups
  if (P.opt.precision != DEMAG_FP64) {
    A.values("node_iperm", P.node_iperm, nn, 0, nn);
    const int64_t nh = A.last(P.hg_off, nn);
    A.offsets("hg_off", P.hg_off, nn, 0, nh, 0, nh);
    A.values("hg_col", P.hg_col, nh, 0, nn);
    if (P.tc_g1_off)
      A.offsets("tc_g1_off", P.tc_g1_off, (int64_t)P.h_m2l_targets.size(), 0, P.n_m2l, -1, -1);
    if (P.tc_n_g2 > 0) {
      const int64_t ne = A.last(P.tc_g2_off, P.tc_n_g2);
      A.values("tc_g2_tgt", P.tc_g2_tgt, 2 * P.tc_n_g2, -1, nc);
      A.offsets("tc_g2_off", P.tc_g2_off, P.tc_n_g2, 0, ne, 0, ne);
      A.values("tc_g2_src", P.tc_g2_src, ne, 0, nc);
      A.values("tc_g2_op", P.tc_g2_op, 2 * ne, -1, P.n_m2l_keys);
    }
  }
  if (plant) {
    const std::string found = planted(P, A);
    if (!found.empty()) fail(DEMAG_ERR_INTERNAL, found);
    return;
  }
  A.finish();
}

}  // namespace demag
