// uf_embed.h -- count rows and embedding rows (uf_embed.cu).
#pragma once
#include "uf_internal.h"

namespace ufg {

// ---- embed (uf_embed.cu) ----
// Count rows live in slots of `ld` doubles (the combined sample axis).
cudaError_t launch_tip_counts(const int32_t *tip_nodes, int n_list, const int32_t *tip_of_node,
                              const int64_t *col_ptr,
                              const int32_t *col_row, const double *col_val, double *counts,
                              int64_t ld, int n, cudaStream_t st);
// One table's CSC arrays and its columns on the combined axis.
struct SliceTab {
  const int64_t *col_ptr;
  const int32_t *col_row;
  const double *col_val;
  int n, off;
};
// Count rows of listed nodes straight from the CSC columns of their tips
// (tip numbers [tip_lo[v], tip_hi[v]), in order), for every table.
cudaError_t launch_slice_counts(const int32_t *nodes, int n_list, const int32_t *tip_lo, const int32_t *tip_hi,
                                const int32_t *slot_of_node, const SliceTab *tabs, int n_tabs, double *counts,
                                int64_t ld, cudaStream_t st);
// Presence bits (`words` words of 32 combined samples a row) instead of counts.
cudaError_t launch_slice_bits(const int32_t *nodes, int n_list, const int32_t *tip_lo, const int32_t *tip_hi,
                              const int32_t *slot_of_node, const SliceTab *tabs, int n_tabs, uint32_t *bits,
                              int64_t words, cudaStream_t st);
// Count rows of a block's internal nodes, level by level, and the embedding
// rows of its dense branches.
struct EmbedArgs {
  // the block's nodes: positions [levels[0], levels[1]) of list hold dense
  // branches whose count rows are built already, [levels[s l], levels[s l + 1])
  // internal nodes whose children are in earlier levels or blocks, s = level_step
  // (1: consecutive levels, each ending where the next starts)
  const int32_t *list, *levels;
  int level_step;
  int n_levels, n_nodes;        // levels (>= 1), list positions from levels[0] to the last level's end
  const int32_t *xrow;          // per list position its row of X, or -1
  const int32_t *child_ptr, *child_idx;
  const int32_t *slot_of_node;
  double *counts;               // rows of ld values, one column per combined sample, or:
  uint32_t *bits;               // rows of ld presence words, n_cols of them used (no X then)
  int64_t ld;
  int n_cols;
  const double *length;         // by node
  const double *total;          // by combined sample
  const float *inv_total_f;
  void *X;                      // null: counts only
  int64_t pitch;
  const TabDesc *tabs;
  int n_tabs;
  double row_scale;             // != 0: 64-bit fixed-point rows (FP64, EMB_SCALED and EMB_PRESENCE)
  int4 *steps;                  // scratch of n_nodes records each, or both null (with xrow and
  double *steps_len;            // slot_of_node null: row and slot v for node v)
  int w, lv0, lv1, first;       // set by launch_embed: columns per CTA, levels of the launch, 1: level 0 too
};
// level_nodes[l]: nodes of level l; *launches grows by the kernels launched
cudaError_t launch_embed(int kind, bool fp32, const EmbedArgs &a, const int *level_nodes, cudaStream_t st,
                         int64_t *launches);
// Fewest samples of a table for which launch_embed writes the rows itself: a
// row of fewer repeats its head so often that a launch over rows
// (launch_emb_rows) is faster than a thread per column.
constexpr int EMBED_MIN_SAMPLES = 32;
// It forms FP64 quotients from a total's reciprocal, which has to be a normal
// number; a table with another total takes launch_emb_rows, which divides.
inline bool plain_total(double t) { return t > 1e-290 && t < 1e290; }
// Embedding rows of branches nodes[0 .. rows) (b0 .. b0 + rows - 1 when
// nodes is null) for every table segment; EMB_VAW rows hold three planes of
// `pitch` elements each, l p, c and T - c (a node list is required).  With
// row_scale != 0 (FP64, EMB_SCALED and EMB_PRESENCE) the rows are 64-bit
// integers, the FP64 values times row_scale rounded to nearest.
cudaError_t launch_emb_rows(int kind, bool fp32, int64_t b0, int rows,
                            const int32_t *slot_of_node, const double *counts, int64_t ld,
                            const double *length, const double *total, const float *inv_total_f,
                            void *X, int64_t pitch, const TabDesc *tabs, int n_tabs, cudaStream_t st,
                            const int32_t *nodes = nullptr, double row_scale = 0.0);

}  // namespace ufg
