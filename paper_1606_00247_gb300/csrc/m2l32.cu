// m2l32.cu -- M2L on CUDA cores, FP64 or FP32: the table-driven kernel of every
// plan whose translations have a table (below), and k_m2l_rows for the others
// (m2l_table_batch < 0, or more than 2^24 distinct translations).
//
//   Lt^T_m = (-1)^|m| / (4 pi s_T) sum_S sum_{|n| <= p - |m|} b_{n+m}(v_S) f_S^|n| Qt^S_n
// (v_S = (c_T - c_S)/s_T, f_S = s_S/s_T, notation of far.cu; n and m run over
// the trace-free indices of common.cuh, 1 <= |n|, |m| < p).
//
// k_m2l_rows: one block per (target cell, slice of 32 states).  Thread = one
// output row m and SPT = 16 states held in registers, so every operator value
// b_{n+m} read from shared memory feeds 16 FMAs and the 16 moments of a given n
// are read with 16-byte shared-memory broadcasts.  Sources are staged CHUNK at
// a time (their moments for the slice and their operator vectors b_k(v),
// computed in the block by the Taylor-coefficient recurrence of 1/|x|).
#include <algorithm>
#include <vector>

#include "common.cuh"

namespace demag {

namespace {

constexpr int SPT = 16;    // states per thread
constexpr int SLICE = 32;  // states per block

__device__ __forceinline__ int idx3(int a, int b, int c) {
  const int t = a + b + c, j = b + c;
  return t * (t + 1) * (t + 2) / 6 + j * (j + 1) / 2 + c;
}

template <class T>
__global__ void __launch_bounds__(1024) k_m2l_rows(const int32_t* __restrict__ targets,
                                                    const int64_t* __restrict__ m2l_off,
                                                    const int32_t* __restrict__ m2l_src,
                                                    const double* __restrict__ centre,
                                                    const int32_t* __restrict__ level, double side, int p, int nc,
                                                    int B, int CHUNK, const T* __restrict__ Q, T* L) {
  extern __shared__ __align__(16) unsigned char rows_smem[];
  T* smem = (T*)rows_smem;
  const int nq = nq_of(p), nl = nl_of(p);
  T* Qs = smem;                              // CHUNK x nq x SLICE
  T* bks = Qs + CHUNK * nq * SLICE;          // CHUNK x nc
  T* fps = bks + CHUNK * nc;                 // CHUNK x 16
  T* geo = fps + CHUNK * 16;                 // CHUNK x 4
  int* mi = (int*)(geo + CHUNK * 4);             // nc packed (a | b<<8 | c<<16 | t<<24)
  const int32_t Tc = targets[blockIdx.x];
  const int b0 = blockIdx.y * SLICE;
  const double sT = ldexp(side, -level[Tc]);
  const double cx = centre[3 * Tc], cy = centre[3 * Tc + 1], cz = centre[3 * Tc + 2];
  for (int i = threadIdx.x; i < nc; i += blockDim.x) {
    int a, b, c;
    mi_decode(i, a, b, c);
    mi[i] = a | (b << 8) | (c << 16) | ((a + b + c) << 24);
  }
  // thread -> (row m, half of the slice)
  const int m = threadIdx.x % nl, half = threadIdx.x / nl;
  const bool active = threadIdx.x < 2 * nl;
  T acc[SPT];
#pragma unroll
  for (int r = 0; r < SPT; r++) acc[r] = (T)0;
  __syncthreads();
  int ma, mb, mz;
  h_decode(active ? m : 0, ma, mb, mz);
  const int tm = ma + mb + mz;
  const int64_t e0 = m2l_off[Tc], e1 = m2l_off[Tc + 1];
  for (int64_t ec = e0; ec < e1; ec += CHUNK) {
    const int ns = (e1 - ec < CHUNK) ? (int)(e1 - ec) : CHUNK;
    __syncthreads();  // the previous chunk is consumed
    for (int q = threadIdx.x; q < ns * nq * SLICE; q += blockDim.x) {
      const int s = q / (nq * SLICE), r = q - s * nq * SLICE, n = r / SLICE, l = r - n * SLICE;
      const int32_t S = m2l_src[ec + s];
      Qs[q] = (b0 + l < B) ? Q[((int64_t)S * nq + n) * B + b0 + l] : (T)0;
    }
    if (threadIdx.x < ns) {
      const int32_t S = m2l_src[ec + threadIdx.x];
      const T x = (T)((cx - centre[3 * S]) / sT), y = (T)((cy - centre[3 * S + 1]) / sT),
                  z = (T)((cz - centre[3 * S + 2]) / sT);
      T* g = geo + 4 * threadIdx.x;
      g[0] = x;
      g[1] = y;
      g[2] = z;
      g[3] = x * x + y * y + z * z;
      bks[threadIdx.x * nc] = (T)(1.0 / sqrt((double)g[3]));
      const int dl = level[Tc] - level[S];
      for (int t = 0; t <= p; t++) fps[threadIdx.x * 16 + t] = (T)ldexp(1.0, dl * t);
    }
    __syncthreads();
    for (int t = 1; t <= p; t++) {
      const int o = t * (t + 1) * (t + 2) / 6, cnt = (t + 1) * (t + 2) / 2;
      for (int q = threadIdx.x; q < ns * cnt; q += blockDim.x) {
        const int s = q / cnt, k = o + (q - s * cnt);
        const int kk = mi[k], ka = kk & 255, kb = (kk >> 8) & 255, kz = (kk >> 16) & 255;
        const T* g = geo + 4 * s;
        const T* bb = bks + s * nc;
        T s1 = (T)0, s2 = (T)0;
        if (ka) s1 += ka * g[0] * bb[idx3(ka - 1, kb, kz)];
        if (kb) s1 += kb * g[1] * bb[idx3(ka, kb - 1, kz)];
        if (kz) s1 += kz * g[2] * bb[idx3(ka, kb, kz - 1)];
        if (ka > 1) s2 += ka * (ka - 1) * bb[idx3(ka - 2, kb, kz)];
        if (kb > 1) s2 += kb * (kb - 1) * bb[idx3(ka, kb - 2, kz)];
        if (kz > 1) s2 += kz * (kz - 1) * bb[idx3(ka, kb, kz - 2)];
        bks[s * nc + k] = ((2 * t - 1) * s1 - (t - 1) * s2) / (t * g[3]);
      }
      __syncthreads();
    }
    if (active) {
      for (int s = 0; s < ns; s++) {
        const T* bk = bks + s * nc;
        const T* fp = fps + s * 16;
        const T* qs = Qs + s * nq * SLICE + half * SPT;
        int n = 0;  // moment position: degree t, then n_x = 0, 1 by ascending n_z
        for (int t = 1; t <= p - tm; t++) {
          const T f = fp[t];
          for (int na = 0; na < 2; na++) {
            for (int c = 0; c <= t - na; c++, n++) {
              const T w = bk[idx3(na + ma, t - na - c + mb, c + mz)] * f;
              T q[SPT];
              load_q<T, SPT>(qs + n * SLICE, q);
#pragma unroll
              for (int r = 0; r < SPT; r++) acc[r] += w * q[r];
            }
          }
        }
      }
    }
  }
  if (!active) return;
  const T inv = (T)(1.0 / (4.0 * M_PI * sT));
  const T sg = (tm & 1) ? -inv : inv;
#pragma unroll
  for (int r = 0; r < SPT; r++) {
    const int b = b0 + half * SPT + r;
    if (b < B) L[((int64_t)Tc * nl + m) * B + b] = sg * acc[r];
  }
}

}  // namespace

template <class T>
void launch_m2l_rows(Plan& P, int B, const T* Q, T* L, cudaStream_t s) {
  if (P.h_m2l_targets.empty()) return;
  const int nc = P.nc;
  const int threads = ((2 * P.nl + 31) / 32) * 32;
  constexpr int chunk = 4;  // at most 4 sources x (168 moments x 32 states + 455): 187 KB in FP64
  const size_t smem = sizeof(T) * (chunk * P.nq * SLICE + chunk * nc + chunk * 16 + chunk * 4) + sizeof(int) * nc;
  smem_opt_in((const void*)k_m2l_rows<T>, smem);
  dim3 grid((unsigned)P.h_m2l_targets.size(), (unsigned)((B + SLICE - 1) / SLICE));
  k_m2l_rows<T><<<grid, threads, smem, s>>>(P.m2l_targets, P.m2l_off, P.m2l_src, P.cell_centre, P.cell_level, P.side,
                                            P.p, nc, B, chunk, Q, L);
  DM_LAUNCH("k_m2l_rows");
}
template void launch_m2l_rows<float>(Plan&, int, const float*, float*, cudaStream_t);
template void launch_m2l_rows<double>(Plan&, int, const double*, double*, cudaStream_t);

// ---------------------------------------------------------------------------
// Table-driven M2L on CUDA cores (k_m2l_tab): the FP64 path, the FP32 precision
// and the small batches of the tensor-core precisions.
//
// The same sum, with b_k(v_S) read from a per-plan table: one row of nc values
// per distinct translation key (dl, lattice offset; m2l_keys.cu), so a pair
// costs a table row (L2-resident: ~8k rows) instead of the recurrence.
//
// Work: an item is a group of TR consecutive rows m and a chunk of TC
// consecutive moments n; a thread is (item, source subgroup k0) and keeps the
// TR x SB sums of its rows for the SB <= 8 states of its slice, over the sources
// k0, k0 + kg, ... of every step.  Per moment it reads SB moments (16-byte
// shared-memory broadcasts: the items are chunk-major, so the lanes of a warp
// share the chunk) and TR table values for TR SB FMAs.  The TR x TC table
// positions of b_{m+n} are read once from a per-order list and held in
// registers (positions as compile-time constants made the code too long for the
// instruction cache); a term beyond |n| + |m| <= p points at a zero behind the
// table row.  ks sources are staged per step by eight warps (cp.async, two
// buffers); f_S^|n|, a power of two, is applied to what is read from sources on
// another level.  The parts of a row (chunks, then subgroups) are added in a fixed
// order at the end, so results do not depend on timing.
namespace tab {

constexpr int TR = TAB_TR, TC = TAB_TC, THREADS = 256, WARPS = THREADS / 32;
constexpr int MAX_CHUNKS = (MAX_P + 1) * (MAX_P + 1) / TC + 1;
constexpr int KS_MAX = 32;  // sources per step, at most KS_MAX / WARPS per staging warp

struct Shape {
  int ks, kg;                    // sources per step, source subgroups
  int nchunk, nitems;
  int16_t off[MAX_CHUNKS + 1];   // first item of every chunk: row group g is item off[c] + g
};

// items of order p: chunk c of row group g exists when the group's lowest row takes moments of it
Shape shape(int p, size_t elem) {
  Shape S{};
  S.nchunk = (nq_of(p) + TC - 1) / TC;
  for (int c = 0; c < S.nchunk; c++) {
    int g = 0;
    while (TR * g < nl_of(p) && c * TC < nq_of(p - h_degree(TR * g))) g++;
    S.off[c + 1] = (int16_t)(S.off[c] + g);
  }
  S.nitems = S.off[S.nchunk];
  // as many subgroups as fit the block, whole rounds of them per step of at
  // least one source per staging warp; FP64 stops at four (p = 8: two blocks'
  // buffers fit an SM)
  const int par = std::max(1, THREADS / S.nitems);
  S.kg = std::min(par, elem == 8 ? (S.nitems > 24 ? 4 : 16) : KS_MAX);
  S.ks = S.kg * ((WARPS + S.kg - 1) / S.kg);
  return S;
}

// table rows: nc values, then zeros up to a multiple of four (at least one)
__host__ __device__ constexpr int row_len(int nc) { return nc / 4 * 4 + 4; }
// moment rows staged per source: padded to whole chunks (the padding stays zero)
__host__ __device__ constexpr int mom_rows(int nq) { return (nq + TC - 1) / TC * TC; }
// one buffer: ks table rows, ks moment blocks, ks level differences
template <int SB>
__host__ __device__ constexpr size_t buf_len(int ks, int nc, int nq) {
  return (size_t)ks * (row_len(nc) + mom_rows(nq) * SB) + (ks + 3) / 4 * 4;
}

template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(d), "l"(src), "n"(BYTES) : "memory");
}

// v 2^e; one multiplication where 2^e is a normal number
__device__ __forceinline__ float scale_pow2(float v, int e) {
  return abs(e) <= 126 ? v * __int_as_float((127 + e) << 23) : ldexpf(v, e);
}
__device__ __forceinline__ double scale_pow2(double v, int e) {
  return abs(e) <= 1022 ? v * __longlong_as_double((long long)(1023 + e) << 52) : ldexp(v, e);
}

template <class T, int SB>
__global__ void __launch_bounds__(THREADS, 2) k_m2l_tab(const int32_t* __restrict__ targets,
                                                     const int64_t* __restrict__ m2l_off,
                                                     const int32_t* __restrict__ m2l_src,
                                                     const int32_t* __restrict__ m2l_opdl, const T* __restrict__ tab,
                                                     const TabItem* __restrict__ items, const Shape S, const int32_t* __restrict__ level, double side,
                                                     int p, int nc, int B, const T* __restrict__ Q, T* L) {
  extern __shared__ __align__(16) unsigned char tab_smem[];
  T* sm = (T*)tab_smem;
  constexpr int V = 16 / (int)sizeof(T);
  const int nq = nq_of(p), nl = nl_of(p), rl = row_len(nc), mr = mom_rows(nq), ks = S.ks;
  const size_t bufsz = buf_len<SB>(ks, nc, nq), qoff = (size_t)ks * rl, doff = qoff + (size_t)ks * mr * SB;
  const int32_t Tc = targets[blockIdx.x];
  const int b0 = blockIdx.y * SB, nlive = min(SB, B - b0);
  const int64_t e0 = m2l_off[Tc], nsrc = m2l_off[Tc + 1] - e0;
  const int nsteps = (int)((nsrc + ks - 1) / ks);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // the whole block of moments is contiguous when one slice holds the batch
  const bool lin = B == SB && (nq * SB) % V == 0;
  const bool vec = SB % V == 0 && nlive == SB && B % V == 0;
  for (int i = tid; i < 2 * ks * (mr - nq) * SB; i += THREADS) {  // padding rows of the moment blocks
    const int per = (mr - nq) * SB, blk = i / per;
    sm[(size_t)(blk / ks) * bufsz + qoff + (size_t)(blk % ks) * mr * SB + nq * SB + i % per] = (T)0;
  }
  // this thread's item
  const int k0 = tid / S.nitems;
  const bool has = k0 < S.kg;
  const TabItem* it = items + (tid - k0 * S.nitems);
  const int c = it->chunk;
  // table positions; FP64 (bound by its arithmetic, short of registers) keeps two per word
  constexpr int IP = sizeof(T) == 8 ? 2 : 1;
  uint32_t idx[TR][TC / IP];
#pragma unroll
  for (int r = 0; r < TR; r++)
#pragma unroll
    for (int j = 0; j < TC / IP; j++)
      idx[r][j] = IP == 2 ? ((const uint32_t*)it->idx)[(r * TC) / 2 + j] : it->idx[r * TC + j];
  auto pos = [&](int r, int j) { return IP == 2 ? (j & 1 ? idx[r][j / IP] >> 16 : idx[r][j / IP] & 0xFFFFu) : idx[r][j / IP]; };
  const uint2 degs = *(const uint2*)it->deg;
  T acc[TR][SB];
#pragma unroll
  for (int r = 0; r < TR; r++)
#pragma unroll
    for (int b = 0; b < SB; b++) acc[r][b] = (T)0;
  // staging: warp w takes the sources w, w + 8, ... of every step; their list
  // entries are read one step ahead by lanes 0 .. ks / 8 - 1
  int32_t mS = -1, mO = 0;
  auto meta = [&](int s) {
    const int64_t e = (int64_t)s * ks + warp + WARPS * lane;
    const bool v = WARPS * lane + warp < ks && s < nsteps && e < nsrc;
    mS = v ? m2l_src[e0 + e] : -1;
    mO = v ? m2l_opdl[e0 + e] : 0;
  };
  auto stage = [&](T* buf) {
    for (int j = 0; WARPS * j + warp < ks; j++) {
      const int k = WARPS * j + warp;
      const int32_t So = __shfl_sync(0xffffffffu, mS, j), od = __shfl_sync(0xffffffffu, mO, j);
      T* brow = buf + (size_t)k * rl;
      T* qblk = buf + qoff + (size_t)k * mr * SB;
      if (lane == 0) ((int*)(buf + doff))[k] = So < 0 ? 0 : od >> 24;  // level difference
      if (So < 0) {  // beyond the list: a zero row and zero moments
        for (int i = lane; i < rl; i += 32) brow[i] = (T)0;
        for (int i = lane; i < nq * SB; i += 32) qblk[i] = (T)0;
        continue;
      }
      const T* trow = tab + (int64_t)(od & 0xFFFFFF) * rl;
      for (int i = lane; i < rl / V; i += 32) cp_async<16>(brow + V * i, trow + V * i);
      const T* q = Q + (int64_t)So * nq * B + b0;
      if (lin) {
        for (int i = lane; i < nq * SB / V; i += 32) cp_async<16>(qblk + V * i, q + V * i);
        continue;
      }
      if constexpr (SB % V == 0) {
        if (vec) {
          constexpr int NV = SB / V;
          for (int i = lane; i < nq * NV; i += 32) {
            const int n = i / NV, v = i - n * NV;
            cp_async<16>(qblk + n * SB + V * v, q + (int64_t)n * B + V * v);
          }
          continue;
        }
      }
      for (int i = lane; i < nq * SB; i += 32) {
        const int n = i / SB, b = i - n * SB;
        if (b < nlive)
          cp_async<sizeof(T)>(qblk + i, q + (int64_t)n * B + b);
        else
          qblk[i] = (T)0;
      }
    }
  };
  meta(0);
  stage(sm);
  meta(1);
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  for (int s = 0; s < nsteps; s++) {
    T* buf = sm + (size_t)(s & 1) * bufsz;
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();  // step s staged; step s - 1 consumed
    if (s + 1 < nsteps) {
      stage(sm + (size_t)((s + 1) & 1) * bufsz);
      meta(s + 2);
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    if (has) {
#pragma unroll 1
      for (int k = k0; k < ks; k += S.kg) {
        const T* bs = buf + (size_t)k * rl;
        const T* qs = buf + qoff + ((size_t)k * mr + c * TC) * SB;
        const int dl = ((const int*)(buf + doff))[k];
#pragma unroll
        for (int j = 0; j < TC; j++) {
          T q[SB];
          load_q<T, SB>(qs + j * SB, q);
          T w[TR];
#pragma unroll
          for (int r = 0; r < TR; r++) w[r] = bs[pos(r, j)];
          if (dl != 0) {  // f_S^|n| = 2^(dl |n|), on the fewer factors
            const int e = dl * (int)(((j < 4 ? degs.x : degs.y) >> (8 * (j & 3))) & 255u);
            if constexpr (SB < TR) {
#pragma unroll
              for (int b = 0; b < SB; b++) q[b] = scale_pow2(q[b], e);
            } else {
#pragma unroll
              for (int r = 0; r < TR; r++) w[r] = scale_pow2(w[r], e);
            }
          }
#pragma unroll
          for (int r = 0; r < TR; r++)
#pragma unroll
            for (int b = 0; b < SB; b++) acc[r][b] += w[r] * q[b];
        }
      }
    }
  }
  // add the parts of each row: chunks in order, subgroups in order
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  __syncthreads();
  T* part = sm;  // [thread][TR][SB]
  if (has)
#pragma unroll
    for (int r = 0; r < TR; r++)
#pragma unroll
      for (int b = 0; b < SB; b++) part[(tid * TR + r) * SB + b] = acc[r][b];
  __syncthreads();
  const T inv = (T)(1.0 / (4.0 * M_PI * ldexp(side, -level[Tc])));
  for (int q = tid; q < nl * SB; q += THREADS) {
    const int m = q / SB, b = q - m * SB, gr = m / TR, r = m - TR * gr;
    if (b >= nlive) continue;
    T v = (T)0;
    for (int cc = 0; cc < S.nchunk; cc++) {
      if (gr >= S.off[cc + 1] - S.off[cc]) break;
      for (int k = 0; k < S.kg; k++) v += part[((k * S.nitems + S.off[cc] + gr) * TR + r) * SB + b];
    }
    L[((int64_t)Tc * nl + m) * B + b0 + b] = (h_degree(m) & 1) ? -inv * v : inv * v;
  }
}

template <class T, int SB>
void launch_sb(Plan& P, int B, const T* Q, T* L, cudaStream_t s) {
  const Shape S = shape(P.p, sizeof(T));
  if constexpr (SB == 8)  // FP64 at p = 12: two buffers of 8 sources x 8 states exceed the shared memory
    if (sizeof(T) * 2 * buf_len<SB>(S.ks, P.nc, P.nq) > 227 * 1024) return launch_sb<T, 4>(P, B, Q, L, s);
  const size_t smem = sizeof(T) * std::max(2 * buf_len<SB>(S.ks, P.nc, P.nq), (size_t)THREADS * TR * SB);
  smem_opt_in((const void*)k_m2l_tab<T, SB>, smem);
  const dim3 grid((unsigned)P.h_m2l_targets.size(), (unsigned)((B + SB - 1) / SB));
  k_m2l_tab<T, SB><<<grid, THREADS, smem, s>>>(P.m2l_targets, P.m2l_off, P.m2l_src, P.m2l_tab_opdl,
                                               (const T*)P.m2l_tab, P.m2l_tab_items, S,
                                               P.cell_level, P.side, P.p, P.nc, B, Q, L);
  DM_LAUNCH("k_m2l_tab");
}

// b_k(v) for one key per block, FP64 recurrence, rounded to T
template <class T>
__global__ void __launch_bounds__(128) k_m2l_tab_ops(const int4* __restrict__ keys, int p, int nc, T* tab) {
  __shared__ double b[MAX_NCOEF];
  const int4 key = keys[blockIdx.x];
  const int dl = key.x;
  const double sc = ldexp(1.0, -((dl < 0 ? -dl : 0) + 1));
  const double vx = key.y * sc, vy = key.z * sc, vz = key.w * sc, r2 = vx * vx + vy * vy + vz * vz;
  if (threadIdx.x == 0) b[0] = 1.0 / sqrt(r2);
  __syncthreads();
  // b_k = (-1)^|k| d^k (1/|x|) at v:  |k| r^2 b_k = (2|k|-1) sum k_i v_i b_{k-e_i} - (|k|-1) sum k_i (k_i-1) b_{k-2e_i}
  for (int t = 1; t <= p; t++) {
    for (int k = ncoef_of(t - 1) + threadIdx.x; k < ncoef_of(t); k += blockDim.x) {
      int ka, kb, kz;
      mi_decode(k, ka, kb, kz);
      double s1 = 0.0, s2 = 0.0;
      if (ka) s1 += ka * vx * b[mi_index(ka - 1, kb, kz)];
      if (kb) s1 += kb * vy * b[mi_index(ka, kb - 1, kz)];
      if (kz) s1 += kz * vz * b[mi_index(ka, kb, kz - 1)];
      if (ka > 1) s2 += ka * (ka - 1) * b[mi_index(ka - 2, kb, kz)];
      if (kb > 1) s2 += kb * (kb - 1) * b[mi_index(ka, kb - 2, kz)];
      if (kz > 1) s2 += kz * (kz - 1) * b[mi_index(ka, kb, kz - 2)];
      b[k] = ((2 * t - 1) * s1 - (t - 1) * s2) / (t * r2);
    }
    __syncthreads();
  }
  const int rl = row_len(nc);
  for (int k = threadIdx.x; k < rl; k += blockDim.x) tab[(int64_t)blockIdx.x * rl + k] = k < nc ? (T)b[k] : (T)0;
}

// key index and level difference of every pair in one word
__global__ void k_opdl(int64_t n, const int32_t* __restrict__ op, const int4* __restrict__ keys, int32_t* opdl) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e < n) opdl[e] = op[e] | (int32_t)((uint32_t)(keys[op[e]].x & 255) << 24);
}

}  // namespace tab

void build_m2l_tab(Plan& P, const M2lKeys& K) {
  if (!K.ok || K.keys.empty() || K.keys.size() >= (1u << 24)) return;
  cudaStream_t s = P.stream;
  const size_t nk = K.keys.size();
  const bool fp64 = P.opt.precision == DEMAG_FP64;
  const tab::Shape S = tab::shape(P.p, fp64 ? 8 : 4);
  std::vector<TabItem> items(S.nitems);
  for (int c = 0; c < S.nchunk; c++)
    for (int i = S.off[c]; i < S.off[c + 1]; i++) {
      TabItem& it = items[i];
      it.chunk = c;
      it.pad = 0;
      for (int j = 0; j < tab::TC; j++) {
        const int n = c * tab::TC + j;
        int na, nb, nz;
        h_decode(n + 1, na, nb, nz);
        it.deg[j] = (uint8_t)(na + nb + nz);
        for (int r = 0; r < tab::TR; r++) {
          const int m = tab::TR * (i - S.off[c]) + r;
          int ma, mb, mz;
          h_decode(m, ma, mb, mz);
          const bool term = m < P.nl && n < nq_of(P.p - ma - mb - mz);
          it.idx[r * tab::TC + j] = (uint16_t)(term ? mi_index(ma + na, mb + nb, mz + nz) : P.nc);
        }
      }
    }
  P.m2l_tab_nitems = S.nitems;
  P.m2l_tab_items = dalloc<TabItem>(P, items.size());
  DM_CUDA(cudaMemcpyAsync(P.m2l_tab_items, items.data(), items.size() * sizeof(TabItem), cudaMemcpyHostToDevice, s));
  P.m2l_tab_opdl = dalloc<int32_t>(P, P.n_m2l);
  P.m2l_tab = dalloc<unsigned char>(P, nk * (size_t)tab::row_len(P.nc) * (fp64 ? sizeof(double) : sizeof(float)));
  int4* dkeys = nullptr;
  if (cudaMalloc(&dkeys, nk * sizeof(int4)) != cudaSuccess) {
    cudaGetLastError();
    fail(DEMAG_ERR_OUT_OF_MEMORY, "M2L table temporary allocation failed");
  }
  cudaError_t e = cudaMemcpyAsync(dkeys, K.keys.data(), nk * sizeof(int4), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) {
    if (fp64)
      tab::k_m2l_tab_ops<double><<<(unsigned)nk, 128, 0, s>>>(dkeys, P.p, P.nc, (double*)P.m2l_tab);
    else
      tab::k_m2l_tab_ops<float><<<(unsigned)nk, 128, 0, s>>>(dkeys, P.p, P.nc, (float*)P.m2l_tab);
    tab::k_opdl<<<(unsigned)((P.n_m2l + 255) / 256), 256, 0, s>>>(P.n_m2l, P.m2l_op, dkeys, P.m2l_tab_opdl);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaFree(dkeys);
  if (e != cudaSuccess) fail(DEMAG_ERR_CUDA, std::string("M2L table build: ") + cudaGetErrorString(e));
}

template <class T>
bool launch_m2l_tab(Plan& P, int B, const T* Q, T* L, cudaStream_t s) {
  if (P.m2l_tab == nullptr) return false;
  if (P.h_m2l_targets.empty()) return true;
  if (B == 1)
    tab::launch_sb<T, 1>(P, B, Q, L, s);
  else if (B == 2)
    tab::launch_sb<T, 2>(P, B, Q, L, s);
  else if (B <= 4)
    tab::launch_sb<T, 4>(P, B, Q, L, s);
  else
    tab::launch_sb<T, 8>(P, B, Q, L, s);
  return true;
}
template bool launch_m2l_tab<float>(Plan&, int, const float*, float*, cudaStream_t);
template bool launch_m2l_tab<double>(Plan&, int, const double*, double*, cudaStream_t);

}  // namespace demag
