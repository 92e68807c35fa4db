// uf_embed.cu -- per-branch embeddings (emb of Figs. 1-3; in the paper a CPU
// producer prepares them buffer by buffer, Sec. 3), built level by level on the GPU.
//
// A node's count row is the sum of its children's count rows (postorder:
// children first); a tip's row is its column of the count table.  The
// embedding row of a branch is then f(count[k] / total[k]) for every sample
// k, written over a padded width so that the stripe kernel can read the
// partner column k + d without a modulo.
#include <algorithm>
#include <type_traits>

#include "uf_device.cuh"
#include "uf_embed.h"

namespace ufg {

// One CTA per tip: zero the table's part of the tip's count row, then
// scatter its CSC column (counts points at the table's first column; the row
// of node v is slot v).
__global__ void k_tip_counts(const int32_t *__restrict__ tip_nodes,
                             const int32_t *__restrict__ tip_of_node,
                             const int64_t *__restrict__ col_ptr,
                             const int32_t *__restrict__ col_row,
                             const double *__restrict__ col_val, double *__restrict__ counts,
                             int64_t ld, int n) {
  const int v = tip_nodes[blockIdx.x];
  double *row = counts + (int64_t)v * ld;
  for (int k = threadIdx.x; k < n; k += blockDim.x) row[k] = 0.0;
  __syncthreads();
  const int f = tip_of_node[v];
  const int64_t q1 = col_ptr[f + 1];
  for (int64_t q = col_ptr[f] + threadIdx.x; q < q1; q += blockDim.x) row[col_row[q]] = col_val[q];
}

// One group of G threads per node of a list (and table, blockIdx.y): zero the
// table's part of the node's count slot, then add the CSC columns of its tips [tip_lo, tip_hi)
// one after the other (within one tip's column the samples are distinct, so its
// entries scatter without conflicts).  Serves tips and the nodes whose own
// subtree is not walked level by level (a branch scattered by the sparse-row
// path whose parent runs through the dense kernels).  G = 32: the tips of such a
// node come one after the other, each a trip to memory and a barrier, so with
// columns that a warp takes in a step or two a warp per node has eight times the
// nodes in flight (8 tables of 203 to 1,000 samples: 0.43 ms with 256 threads).
template <int G>
__global__ void __launch_bounds__(256) k_slice_counts(const int32_t *__restrict__ nodes, int n_list,
                                                      const int32_t *__restrict__ tip_lo,
                                                      const int32_t *__restrict__ tip_hi,
                                                      const int32_t *__restrict__ slot_of_node,
                                                      const SliceTab *__restrict__ tabs, double *__restrict__ counts,
                                                      int64_t ld) {
  const int i = blockIdx.x * (256 / G) + threadIdx.x / G, t = threadIdx.x % G;
  if (i >= n_list) return;  // whole groups
  auto sync = [] {
    if constexpr (G == 32) __syncwarp();
    else __syncthreads();
  };
  const int v = nodes[i];
  const SliceTab tb = tabs[blockIdx.y];
  double *row = counts + (int64_t)slot_of_node[v] * ld + tb.off;
  for (int k = t; k < tb.n; k += G) row[k] = 0.0;
  sync();
  const int f1 = tip_hi[v];
  int64_t q0 = tb.col_ptr[tip_lo[v]];
  for (int f = tip_lo[v]; f < f1; f++) {
    const int64_t q1 = tb.col_ptr[f + 1];
    for (int64_t q = q0 + t; q < q1; q += G) row[tb.col_row[q]] += tb.col_val[q];
    if (q1 > q0) sync();
    q0 = q1;
  }
}

// Presence bits of the same nodes, one warp per node: bit k of its row (word
// k / 32) is 1 where combined sample k has a count below the node.  The rows of
// all tables are one: `words` words of 32 samples.
__global__ void k_slice_bits(const int32_t *__restrict__ nodes, int n_list, const int32_t *__restrict__ tip_lo,
                             const int32_t *__restrict__ tip_hi, const int32_t *__restrict__ slot_of_node,
                             const SliceTab *__restrict__ tabs, int n_tabs, uint32_t *__restrict__ bits, int64_t words) {
  const int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= n_list) return;
  const int v = nodes[i];
  uint32_t *row = bits + (int64_t)slot_of_node[v] * words;
  for (int64_t w = lane; w < words; w += 32) row[w] = 0u;
  __syncwarp();
  for (int t = 0; t < n_tabs; t++) {
    const SliceTab &tb = tabs[t];
    const int64_t q1 = tb.col_ptr[tip_hi[v]];
    for (int64_t q = tb.col_ptr[tip_lo[v]] + lane; q < q1; q += 32) {
      const int k = tb.off + tb.col_row[q];
      atomicOr(row + (k >> 5), 1u << (k & 31));
    }
  }
}

// Table whose row segment holds column j (segments are contiguous, in order).
__device__ __forceinline__ int segment_of(const TabDesc *tabs, int n_tabs, int64_t j) {
  int lo = 0, hi = n_tabs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (tabs[mid].x_col <= j) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// One CTA per branch row r (node nodes[r], or b0 + r without a list): in
// table t's segment, X[r][x_col + j] = f(count[off + (j mod n)]) for j < the
// segment's width.
template <typename T, int KIND>
__global__ void k_emb_rows(int64_t b0, const int32_t *__restrict__ nodes,
                           const int32_t *__restrict__ slot_of_node,
                           const double *__restrict__ counts, int64_t ld,
                           const double *__restrict__ length, const double *__restrict__ total,
                           const float *__restrict__ inv_total_f, T *__restrict__ X, int64_t pitch,
                           const TabDesc *__restrict__ tabs, int n_tabs, double row_scale) {
  const int64_t v = nodes ? (int64_t)nodes[blockIdx.x] : b0 + blockIdx.x;
  const double *c = counts + (slot_of_node ? (int64_t)slot_of_node[v] : v) * ld;
  const double l = length[v];
  T *x = X + (int64_t)blockIdx.x * pitch;
  for (int64_t j = threadIdx.x; j < pitch; j += blockDim.x) {
    const TabDesc &tb = tabs[n_tabs == 1 ? 0 : segment_of(tabs, n_tabs, j)];
    int64_t k = j - tb.x_col;
    while (k >= tb.n) k -= tb.n;
    k += tb.off;
    if constexpr (std::is_same_v<T, unsigned long long>)
      x[j] = __double2ull_rn(emb_value<double, KIND>(c[k], l, total[k], 0.f) * row_scale);
    else x[j] = emb_value<T, KIND>(c[k], l, total[k], inv_total_f[k]);
  }
}

// Variance-adjusted rows: three planes per row r, each `pitch` elements:
// l p = l c / T (the branch length folded in, as it multiplies both sums),
// the count c below the branch and T - c, with the same wrap-padded columns
// as k_emb_rows.
template <typename T>
__global__ void k_emb_rows_vaw(const int32_t *__restrict__ nodes, const int32_t *__restrict__ slot_of_node,
                               const double *__restrict__ counts, int64_t ld, const double *__restrict__ length,
                               const double *__restrict__ total, const float *__restrict__ inv_total_f,
                               T *__restrict__ X, int64_t pitch, const TabDesc *__restrict__ tabs, int n_tabs) {
  const int64_t v = nodes[blockIdx.x];
  const double *c = counts + (int64_t)slot_of_node[v] * ld;
  const double l = length[v];
  T *x = X + (int64_t)blockIdx.x * 3 * pitch;
  for (int64_t j = threadIdx.x; j < pitch; j += blockDim.x) {
    const TabDesc &tb = tabs[n_tabs == 1 ? 0 : segment_of(tabs, n_tabs, j)];
    int64_t k = j - tb.x_col;
    while (k >= tb.n) k -= tb.n;
    k += tb.off;
    const double ck = c[k], tk = total[k];
    // FP32 rows use the FP32 reciprocal of the total (an FP64 division per
    // value costs more than the whole FP32 kernel saves)
    if constexpr (sizeof(T) == 4) x[j] = (float)l * ((float)ck * inv_total_f[k]);
    else x[j] = l * (ck / tk);
    x[pitch + j] = (T)ck;
    x[2 * pitch + j] = (T)(tk - ck);
  }
}

// ---- count rows level by level, with the embedding rows ----
// A thread keeps one column: its total, its reciprocal and where its value goes
// in a row (a row repeats its own head, so a value has several places) are
// read once for all the nodes it visits, and a node's value is written when its
// count is summed (a second pass over the counts before).  Levels of many
// elements are a launch each over whole rows: bound by the counts' traffic.
// The narrow levels, most of them and bound by launching, share one launch: a
// sample's counts depend on no other sample's, so a CTA owns a slab of `w`
// columns and walks the levels with a block barrier between them.  2,048
// samples, 19,331 dense branches, 36 levels: 0.48 ms (0.57 with a launch per
// level and the rows apart; 0.62 with every level in slabs, whose 32-byte pieces
// of rows leave L2 apart); FP64 rows of 1,531 samples 0.57 ms (1.70); 64
// samples, one launch instead of 22.
template <typename T, int KIND>
struct RowValue;  // one column's value of an embedding row from its count c and the branch length l
template <int KIND>
struct RowValue<float, KIND> {
  double t;
  float it;
  __device__ RowValue(double total, float inv, double) : t(total), it(inv) {}
  __device__ float operator()(double c, double l) const { return emb_value<float, KIND>(c, l, t, it); }
};
// c / t by the reciprocal and one correction of the remainder (Markstein):
// 3 FP64 instructions per value instead of a division's dozen, on a GPU with
// 2 FP64 lanes per clock per SM (totals outside plain_total() do not come here:
// a test per value for them took 4 us of a 158 us call)
struct Quotient {
  double t, rt;
  __device__ Quotient(double total) : t(total), rt(1.0 / total) {}
  __device__ double operator()(double c) const {
    const double q = c * rt;
    return fma(fma(-q, t, c), rt, q);
  }
};
template <int KIND>
struct RowValue<double, KIND> {
  Quotient q;
  __device__ RowValue(double total, float, double) : q(total) {}
  __device__ double operator()(double c, double l) const {
    if (KIND == EMB_PRESENCE) return c > 0.0 ? l : 0.0;
    return KIND == EMB_SCALED ? l * q(c) : q(c);
  }
};
template <int KIND>
struct RowValue<unsigned long long, KIND> {
  Quotient q;
  double scale;
  __device__ RowValue(double total, float, double row_scale) : q(total), scale(row_scale) {}
  __device__ unsigned long long operator()(double c, double l) const {
    const double ls = l * scale;  // exact, and finite for every branch (grid_fits)
    if (KIND == EMB_PRESENCE) return c > 0.0 ? __double2ull_rn(ls) : 0ull;
    return __double2ull_rn(ls * q(c));
  }
};

// Table holding combined sample column k (tables in order of off).
__device__ __forceinline__ int embed_table_of(const TabDesc *tabs, int n_tabs, int k) {
  int lo = 0, hi = n_tabs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (tabs[mid].off <= k) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// What the slab kernel needs of list position p in one 16-byte load: the
// node's slot, its first and second child's (-1: none; two or more levels of
// indirection per node otherwise, each a trip to L2), its row of X; more than
// two children: -2 - node in .z.
__global__ void k_embed_steps(const EmbedArgs a, int4 *__restrict__ steps, double *__restrict__ len) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.n_nodes) return;
  const int p = a.levels[0] + i, v = a.list[p];
  const bool built = a.n_levels < 2 || p < a.levels[a.level_step];
  const int c0 = a.child_ptr[v], nc = built ? 0 : a.child_ptr[v + 1] - c0;
  int4 q;
  q.x = a.slot_of_node[v];
  q.y = nc > 0 ? a.slot_of_node[a.child_idx[c0]] : -1;
  q.z = nc == 2 ? a.slot_of_node[a.child_idx[c0 + 1]] : nc > 2 ? -2 - v : -1;
  q.w = a.xrow ? a.xrow[p] : -1;
  steps[i] = q;
  if (len) len[i] = a.length[v];
}

// STEPS: from k_embed_steps' records; else from the tree's arrays (the
// allocation-free call, which has no room for records)
template <typename T, int KIND, bool STEPS>
__global__ void __launch_bounds__(512) k_embed_slab(const EmbedArgs a) {
  constexpr int U = 4;  // nodes per thread in flight
  const int per = blockDim.x / a.w, g = threadIdx.x / a.w;  // nodes at a time, this thread's
  const int k = blockIdx.x * a.w + (threadIdx.x - g * a.w);
  const bool on = k < a.n_cols;
  const int kc = on ? k : 0;
  const int ti = a.n_tabs == 1 ? 0 : embed_table_of(a.tabs, a.n_tabs, kc);
  const int n = a.tabs[ti].n;
  const int64_t j0 = a.tabs[ti].x_col + (kc - a.tabs[ti].off);
  const int64_t j1 = ti + 1 < a.n_tabs ? a.tabs[ti + 1].x_col : a.pitch;
  const double total = a.total[kc];
  const float inv = a.inv_total_f[kc];
  const RowValue<T, KIND == EMB_VAW ? EMB_PROP : KIND> value(total, inv, a.row_scale);
  T *X = (T *)a.X;
  double *counts = a.counts + kc;
  auto put = [&](int row, double l, double c) {
    if constexpr (KIND == EMB_VAW) {
      // three planes: l p, the count below and the rest of the total (FP32
      // rows use the FP32 reciprocal of the total)
      T *x = X + (int64_t)row * 3 * a.pitch;
      T y;
      if constexpr (sizeof(T) == 4) y = (float)l * ((float)c * inv);
      else y = l * value(c, l);
      for (int64_t j = j0; j < j1; j += n) {
        x[j] = y;
        x[a.pitch + j] = (T)c;
        x[2 * a.pitch + j] = (T)(total - c);
      }
    } else {
      T *x = X + (int64_t)row * a.pitch;
      const T y = value(c, l);
      for (int64_t j = j0; j < j1; j += n) x[j] = y;
    }
  };
  auto more = [&](int v, int c0) {  // the sum over a node's children from c0 on, in index order
    double s = 0.0;
    for (int c = c0; c < a.child_ptr[v + 1]; c++) {
      const int ch = a.child_idx[c];
      s += counts[(int64_t)(a.slot_of_node ? a.slot_of_node[ch] : ch) * a.ld];
    }
    return s;
  };
  const int p_first = a.levels[0];
  for (int lv = a.first ? 0 : a.lv0; lv < a.lv1; lv = max(lv + 1, a.lv0)) {
    const int pb = a.levels[a.level_step * lv], p1 = a.levels[a.level_step * lv + 1];
    if (on && (lv > 0 || X)) {
      if constexpr (STEPS) {
        for (int p = pb + blockIdx.y * (U * per) + g; p < p1; p += gridDim.y * (U * per)) {
          int4 q[U];
          double l[U], s[U];
#pragma unroll
          for (int u = 0; u < U; u++) {
            const int pu = p + u * per;
            q[u] = pu < p1 ? a.steps[pu - p_first] : make_int4(-1, -1, -1, -1);
            l[u] = pu < p1 ? a.steps_len[pu - p_first] : 0.0;
          }
#pragma unroll
          for (int u = 0; u < U; u++) {
            // a built row is read (if it has an embedding row), others summed
            const int c0 = lv == 0 ? (q[u].w >= 0 ? q[u].x : -1) : q[u].y;
            s[u] = c0 >= 0 ? counts[(int64_t)c0 * a.ld] : 0.0;
            if (q[u].z >= 0) s[u] += counts[(int64_t)q[u].z * a.ld];
          }
#pragma unroll
          for (int u = 0; u < U; u++) {
            if (q[u].z < -1) {
              const int v = -2 - q[u].z;
              s[u] = more(v, a.child_ptr[v]);
            }
            if (lv > 0 && q[u].x >= 0) counts[(int64_t)q[u].x * a.ld] = s[u];
            if (X && q[u].w >= 0) put(q[u].w, l[u], s[u]);
          }
        }
      } else {
        for (int p = pb + g; p < p1; p += per) {
          const int v = a.list[p];
          double *at = counts + (int64_t)v * a.ld;
          const double s = lv == 0 ? *at : more(v, a.child_ptr[v]);
          if (lv > 0) *at = s;
          if (X) put(v, a.length[v], s);
        }
      }
    }
    __syncthreads();  // the level's counts, before its parents read them
  }
}

// The same walk for presence bits: a node's words are the OR of its children's.
__global__ void __launch_bounds__(512) k_bits_slab(const EmbedArgs a) {
  constexpr int U = 4;
  const int per = blockDim.x / a.w, g = threadIdx.x / a.w;
  const int k = blockIdx.x * a.w + (threadIdx.x - g * a.w);
  uint32_t *bits = a.bits + k;
  const int p_first = a.levels[0];
  for (int lv = a.lv0; lv < a.lv1; lv++) {
    const int p1 = a.levels[a.level_step * lv + 1];
    if (k < a.n_cols)
      for (int p = a.levels[a.level_step * lv] + blockIdx.y * (U * per) + g; p < p1; p += gridDim.y * (U * per)) {
        int4 q[U];
        uint32_t s[U];
#pragma unroll
        for (int u = 0; u < U; u++)
          q[u] = p + u * per < p1 ? a.steps[p + u * per - p_first] : make_int4(-1, -1, -1, -1);
#pragma unroll
        for (int u = 0; u < U; u++) {
          s[u] = q[u].y >= 0 ? bits[(int64_t)q[u].y * a.ld] : 0u;
          if (q[u].z >= 0) s[u] |= bits[(int64_t)q[u].z * a.ld];
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
          if (q[u].z < -1)
            for (int v = -2 - q[u].z, c = a.child_ptr[v]; c < a.child_ptr[v + 1]; c++)
              s[u] |= bits[(int64_t)a.slot_of_node[a.child_idx[c]] * a.ld];
          if (q[u].x >= 0) bits[(int64_t)q[u].x * a.ld] = s[u];
        }
      }
    __syncthreads();
  }
}

namespace {
// elements of a level from which it gets a launch of its own
constexpr int64_t EMBED_WIDE = 1 << 18;

cudaError_t embed_launch(int kind, bool fp32, const EmbedArgs &a, dim3 grid, int nt, cudaStream_t st) {
  const bool steps = a.steps != nullptr;
  if (a.bits) return launch_k(k_bits_slab, grid, dim3(nt), 0, st, a);
#define UF_SLAB(T, K)                                                                    \
  return launch_k(steps ? k_embed_slab<T, K, true> : k_embed_slab<T, K, false>, grid, dim3(nt), 0, st, a)
  if (kind == EMB_VAW) {
    if (fp32) UF_SLAB(float, EMB_VAW);
    UF_SLAB(double, EMB_VAW);
  }
  if (fp32) {
    if (kind == EMB_SCALED) UF_SLAB(float, EMB_SCALED);
    if (kind == EMB_PRESENCE) UF_SLAB(float, EMB_PRESENCE);
    UF_SLAB(float, EMB_PROP);
  }
  if (a.row_scale != 0.0) {
    if (kind == EMB_SCALED) UF_SLAB(unsigned long long, EMB_SCALED);
    if (kind == EMB_PRESENCE) UF_SLAB(unsigned long long, EMB_PRESENCE);
  }
  if (kind == EMB_SCALED) UF_SLAB(double, EMB_SCALED);
  if (kind == EMB_PRESENCE) UF_SLAB(double, EMB_PRESENCE);
  UF_SLAB(double, EMB_PROP);
#undef UF_SLAB
}

}  // namespace

cudaError_t launch_embed(int kind, bool fp32, const EmbedArgs &a0, const int *level_nodes, cudaStream_t st,
                         int64_t *launches) {
  if (a0.n_nodes <= 0 || a0.n_cols <= 0) return cudaSuccess;
  EmbedArgs a = a0;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const bool steps = a.steps != nullptr;
  if (steps) {
    e = launch_k(k_embed_steps, dim3((unsigned)((a.n_nodes + 255) / 256)), dim3(256), 0, st, a, a.steps, a.steps_len);
    if (e != cudaSuccess) return e;
    (*launches)++;
  }
  // levels of at least EMBED_WIDE elements: CTAs of 256 columns, enough of
  // them for eight per SM, each with its share of the level's nodes
  auto wide = [&](int lv) -> cudaError_t {
    EmbedArgs w = a;
    w.lv0 = lv;
    w.lv1 = lv + 1;
    w.first = 0;
    w.w = 256;
    const int64_t gx = (a.n_cols + 255) / 256;
    const int64_t gy = std::max<int64_t>(1, std::min<int64_t>((level_nodes[lv] + 3) / 4, 8 * (int64_t)sms / gx + 1));
    (*launches)++;
    return embed_launch(kind, fp32, w, dim3((unsigned)gx, (unsigned)gy), 256, st);
  };
  auto is_wide = [&](int lv) { return steps && (int64_t)level_nodes[lv] * a.n_cols >= EMBED_WIDE; };
  // runs of other levels in slabs: the widest (whole 128-byte lines at 16) that
  // still give every SM one
  auto slab = [&](int lv0, int lv1, int first) -> cudaError_t {
    EmbedArgs s = a;
    s.lv0 = lv0;
    s.lv1 = lv1;
    s.first = first;
    s.w = 16;
    while (s.w > (a.bits ? 1 : 2) && (a.n_cols + s.w - 1) / s.w < sms) s.w /= 2;
    int most = first ? level_nodes[0] : 1;
    for (int l = lv0; l < lv1; l++) most = std::max(most, level_nodes[l]);
    const int nt = (int64_t)most * s.w >= 2048 ? 512 : 128;
    (*launches)++;
    return embed_launch(kind, fp32, s, dim3((unsigned)((a.n_cols + s.w - 1) / s.w)), nt, st);
  };
  int first = a.X != nullptr && level_nodes[0] > 0;  // level 0 still to do
  if (first && is_wide(0)) {
    first = 0;
    if ((e = wide(0)) != cudaSuccess) return e;
  }
  for (int l = 1; l < a.n_levels;) {
    if (is_wide(l)) {
      if ((e = wide(l++)) != cudaSuccess) return e;
      continue;
    }
    int m = l + 1;
    while (m < a.n_levels && !is_wide(m)) m++;
    if ((e = slab(l, m, first)) != cudaSuccess) return e;
    first = 0;
    l = m;
  }
  return first ? slab(a.n_levels, a.n_levels, 1) : cudaSuccess;
}

cudaError_t launch_tip_counts(const int32_t *tip_nodes, int n_list, const int32_t *tip_of_node, const int64_t *col_ptr,
                              const int32_t *col_row, const double *col_val, double *counts,
                              int64_t ld, int n, cudaStream_t st) {
  if (n_list <= 0) return cudaSuccess;
  k_tip_counts<<<n_list, 256, 0, st>>>(tip_nodes, tip_of_node, col_ptr, col_row, col_val, counts, ld, n);
  return cudaGetLastError();
}

cudaError_t launch_slice_counts(const int32_t *nodes, int n_list, const int32_t *tip_lo, const int32_t *tip_hi,
                                const int32_t *slot_of_node, const SliceTab *tabs, int n_tabs, double *counts,
                                int64_t ld, cudaStream_t st) {
  // a warp per node up to 8,192 columns in all, else a CTA; tables along grid.y,
  // at most 65,535 of them at a time
  const bool warp = ld <= 8192;
  for (int t = 0; n_list > 0 && t < n_tabs; t += 65535) {
    const cudaError_t e =
        launch_k(warp ? k_slice_counts<32> : k_slice_counts<256>,
                 dim3(warp ? (n_list + 7) / 8 : n_list, std::min(n_tabs - t, 65535)), dim3(256), 0, st, nodes, n_list,
                 tip_lo, tip_hi, slot_of_node, tabs + t, counts, ld);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_slice_bits(const int32_t *nodes, int n_list, const int32_t *tip_lo, const int32_t *tip_hi,
                              const int32_t *slot_of_node, const SliceTab *tabs, int n_tabs, uint32_t *bits,
                              int64_t words, cudaStream_t st) {
  if (n_list <= 0) return cudaSuccess;
  return launch_k(k_slice_bits, dim3((n_list + 7) / 8), dim3(256), 0, st, nodes, n_list, tip_lo, tip_hi, slot_of_node,
                  tabs, n_tabs, bits, words);
}

cudaError_t launch_emb_rows(int kind, bool fp32, int64_t b0, int rows,
                            const int32_t *slot_of_node, const double *counts, int64_t ld,
                            const double *length, const double *total, const float *inv_total_f,
                            void *X, int64_t pitch, const TabDesc *tabs, int n_tabs, cudaStream_t st,
                            const int32_t *nodes, double row_scale) {
  if (rows <= 0) return cudaSuccess;
  if (kind == EMB_VAW) {
    if (!nodes) return cudaErrorInvalidValue;
    if (fp32)
      return launch_k(k_emb_rows_vaw<float>, dim3(rows), dim3(256), 0, st, nodes, slot_of_node, counts, ld, length,
                      total, inv_total_f, (float *)X, pitch, tabs, n_tabs);
    return launch_k(k_emb_rows_vaw<double>, dim3(rows), dim3(256), 0, st, nodes, slot_of_node, counts, ld, length,
                    total, inv_total_f, (double *)X, pitch, tabs, n_tabs);
  }
#define UF_EMB(T, K)                                                                                 \
  return launch_k(k_emb_rows<T, K>, dim3(rows), dim3(256), 0, st, b0, nodes, slot_of_node, counts, ld, length, \
                  total, inv_total_f, (T *)X, pitch, tabs, n_tabs, row_scale)
  if (fp32) {
    if (kind == EMB_SCALED) UF_EMB(float, EMB_SCALED);
    if (kind == EMB_PRESENCE) UF_EMB(float, EMB_PRESENCE);
    UF_EMB(float, EMB_PROP);
  }
  if (row_scale != 0.0) {
    if (kind == EMB_SCALED) UF_EMB(unsigned long long, EMB_SCALED);
    if (kind == EMB_PRESENCE) UF_EMB(unsigned long long, EMB_PRESENCE);
  }
  if (kind == EMB_SCALED) UF_EMB(double, EMB_SCALED);
  if (kind == EMB_PRESENCE) UF_EMB(double, EMB_PRESENCE);
  UF_EMB(double, EMB_PROP);
#undef UF_EMB
}

}  // namespace ufg
