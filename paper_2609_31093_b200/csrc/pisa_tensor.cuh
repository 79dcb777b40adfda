// Tensor-core (tcgen05 / TMEM) path: key-block-major leaf scoring and block-sparse attention.
#pragma once

#include "pisa_common.cuh"

namespace pisa {

bool tensor_path_supported(const Geometry& g, int dtype);
size_t tensor_route_workspace_bytes(const Geometry& g);
size_t tensor_bsa_workspace_bytes(const Geometry& g);
// ws points past the status word; status is the workspace's status word
// lse_out (nullable): softmax denominators of the kept leaves, float [B,Hq,N]
// sel_lse (nullable): per-head denominators of the kept leaves, float [B,Hq,N,K]
int tensor_route(const Geometry& g, int dtype, const void* q, const void* k, const void* pyramid, int32_t* idx,
                 float* sel_lse, float* margin, float* lse_out, void* ws, int32_t* status, cudaStream_t s);
// lse_ready: `lse` already holds the denominators of exactly these idx (as tensor_route writes them)
// sel_lse (nullable): per-block denominators of exactly these idx (as tensor_route writes them); used when
// lse_ready is false to skip the block-LSE pass
// forced_present: idx comes from the routing, i.e. every row holds its forced leaves (0, c-1, c), each leaf once: what
// neighbouring rows share is then served query-major (shared_attend.cu) instead of by the lists
int tensor_bsa(const Geometry& g, int dtype, const void* q, const void* k, const void* v, const int32_t* idx,
               const float* sel_lse, void* out, float* lse, bool lse_ready, bool forced_present, void* ws,
               int32_t* status, cudaStream_t s);

// query-major path (query_major.cuh): dense scoring, one-thread-per-token selection, masked dense attention
namespace qm { struct Args; }
bool qm_supported(const Geometry& g, int dtype);
// shapes for which the whole forward is cheaper query-major than through the lists
bool qm_dense_preferred(const Geometry& g, int dtype);
size_t qm_workspace_bytes(const Geometry& g);
int qm_route(const Geometry& g, const void* q, const void* k, const void* pyramid, int32_t* idx, float* sel_lse,
             float* margin, float* lse_out, void* ws, int32_t* status, cudaStream_t s);
int qm_attend(const Geometry& g, const void* q, const void* k, const void* v, void* out, const float* lse, void* ws,
              int32_t* status, cudaStream_t s);
int qm_tiles_per_item(const Geometry& g, long long unit_tokens);
// packed batches: workspace one sequence needs, and the forward of the sequences ids[0..n) (qm_packed.cu)
size_t qm_packed_bytes(const Geometry& g, int len);
int qm_forward_packed(const Geometry& g, const int32_t* cu, const int* ids, int n, long long total, const void* q, const void* k,
                      const void* v, int32_t* idx, void* out, float* lse, void* ws, size_t ws_bytes, int32_t* status,
                      cudaStream_t s);
// levels L..2 for the list-driven path: scores of the nodes that can prune and the selection among them, a range of
// tokens at a time through `scratch`
bool qm_stage1_preferred(const Geometry& g, int dtype, size_t scratch_bytes);
int qm_stage1(const Geometry& g, const void* q, const void* pyramid, int32_t* par, float* margin, float* scratch,
              size_t scratch_bytes, int32_t* status, cudaStream_t s);
// leaf level of the list-driven path: Select_K among the children of `par` by their scores `blk` (any score mode)
int qm_select_final(const Geometry& g, const int32_t* par, const float* blk, int32_t* idx, float* margin, float* lse_out,
                    float* sel_lse, int32_t* status, cudaStream_t s);
bool tma_strides(const long long* st);
bool qm_map_rows(void* map, const void* base, int d, int H, long long tokens, int B, const long long* st, int heads, int rows);
int launch_qm_score(const Geometry& g, const qm::Args& a, const void* q, const void* k, long long tokens, const void* pyramid,
                    long long pyr_rows, cudaStream_t s);
int launch_qm_select_full(const Geometry& g, const qm::Args& a, long long rows, int32_t* idx, float* margin, float* lse,
                          float* sel_lse, cudaStream_t s);
int launch_qm_select_stage1(const Geometry& g, const qm::Args& a, long long rows, int32_t* par, float* margin, cudaStream_t s);
int launch_qm_select_final(const Geometry& g, const qm::Args& a, long long rows, const int32_t* par, const float* blk,
                           int32_t* idx, float* margin, float* lse, float* sel_lse, cudaStream_t s);
int launch_qm_attend(const Geometry& g, const qm::Args& a, const void* q, const void* k, const void* v, long long tokens,
                     const float* row_lse, void* out, bool one_leaf, bool two_terms, cudaStream_t s);

// dense masked backward (qm_bwd.cuh).  gate (nullable): the choice is left to the data; receives what the list-driven kernels
// have to look at; stat: where the preparation leaves the rows' (-lse * log2 e, -delta), [B, Hkv, N, G], for them too
bool qm_bwd_supported(const Geometry& g, int dtype);
size_t qm_bwd_workspace_bytes(const Geometry& g);
int qm_bwd(const Geometry& g, const void* q, const void* k, const void* v, const int32_t* idx, const void* out, const float* lse,
           const void* dout, void* dq, void* dk, void* dv, void* ws, int32_t* status, Gate* gate, const float2** stat, cudaStream_t s);
// length up to which the dense backward is the better one whatever the rows selected
int qm_bwd_always(const Geometry& g);
int qm_bwd_packed_longest(const Geometry& g);
// packed batches: workspace one sequence needs, and the backward of the sequences ids[0..n)
size_t qm_bwd_packed_bytes(const Geometry& g, int len);
int qm_bwd_packed(const Geometry& g, const int32_t* cu, const int* ids, int n, long long total, const void* q, const void* k,
                  const void* v, const int32_t* idx, const void* out, const float* lse, const void* dout, void* dq, void* dk,
                  void* dv, void* ws, size_t ws_bytes, int32_t* status, cudaStream_t s);
namespace qm { struct Seq; struct SeqOrder; }
// a packed launch's table -> device, as kernel parameters
int qm_write_table(const qm::Seq* seqs, const qm::SeqOrder* order, int n, qm::Seq* d_seqs, qm::SeqOrder* d_order, cudaStream_t s);


// backward of the block-sparse attention with frozen indices; dq [B,N,Hq,d], dk, dv [B,N,Hkv,d] dense
bool tensor_bwd_supported(const Geometry& g, int dtype);
size_t tensor_bwd_workspace_bytes(const Geometry& g);
// dq_strides: element strides (b, n, h) of dq; dkv_pitch: elements between consecutive tokens of dk / dv
// (both describe the caller's dense tensors, of which a chunk of units writes its part)
int tensor_bsa_bwd(const Geometry& g, const void* q, const void* k, const void* v, const int32_t* idx,
                   const void* out, const float* lse, const void* dout, void* dq, void* dk, void* dv,
                   const long long* dq_strides, long long dkv_pitch, void* ws, int32_t* status, const Gate& gate, const float2* stat,
                   cudaStream_t s);

}  // namespace pisa
