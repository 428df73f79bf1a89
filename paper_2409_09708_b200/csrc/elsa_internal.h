// Internal declarations shared by the translation units of libelsa (not installed).
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "elsa.h"

namespace elsa {

// log2(M) for the supported group sizes, -1 otherwise.
inline int index_bits(int M) { return M == 4 ? 2 : M == 8 ? 3 : M == 16 ? 4 : -1; }
inline size_t values_per_row(int in, int N, int M) { return (size_t)(in / M) * (size_t)N; }
inline size_t index_words_per_row(int in, int N, int M)
{
    if (N == M) return 0;
    return ((size_t)(in / M) * (size_t)N * (size_t)index_bits(M) + 31) / 32;
}
inline size_t round_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// Records a message for elsa_last_error() and returns `st`.
elsa_status fail(elsa_status st, const char* fmt, ...);
// Counts one kernel launch and converts the launch's cudaError_t.
elsa_status launched(const char* what);

// Brackets one kernel launch with CUDA events while profiling is on (see elsa_profile_start).
class ProfileScope {
public:
    ProfileScope(int kernel, cudaStream_t stream);
    ~ProfileScope();
private:
    int slot_;
    cudaStream_t stream_;
};
// Layer index attached to the records of the calling thread (-1 outside a table).
void set_profile_layer(int layer);

#ifdef __CUDACC__
// Programmatic dependent launch.  Every kernel of the library is launched with the attribute that
// lets it start while its predecessor on the stream is still draining; in exchange each kernel calls
// pdl_wait_for_predecessors() before its first access to global memory (it returns once the
// predecessor grid has completed and its writes are visible) and pdl_release_successors() as soon as
// its own successor may begin its set-up.  With a predecessor launched the ordinary way both are no-ops.
__device__ __forceinline__ void pdl_wait_for_predecessors() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release_successors() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                       unsigned cluster_x, Args&&... args)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    int n = 0;
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
    if (cluster_x > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = cluster_x;
        attr[n].val.clusterDim.y = 1;
        attr[n].val.clusterDim.z = 1;
        ++n;
    }
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = (unsigned)n;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Args&&>(args)...);
}
#endif

struct DeviceInfo {
    int device;
    int sm_count;
    int cc_major;
    size_t smem_optin;
};
// Properties of the current device (cached per device).
elsa_status device_info(DeviceInfo* info);

// --- kernels (each enqueues on `stream` and returns the launch status) ---
elsa_status launch_compress(const uint16_t* W, int out, int in, int N, int M, uint16_t* vals,
                            uint32_t* idx, cudaStream_t stream);
elsa_status launch_unpack(const uint16_t* vals, const uint32_t* idx, int out, int in, int N, int M,
                          uint16_t* Wm, cudaStream_t stream);
elsa_status launch_linear_simt(const uint16_t* X, int rows, const uint16_t* vals,
                               const uint32_t* idx, const uint16_t* bias, int out, int in, int N,
                               int M, elsa_dtype dtype, uint16_t* Y, cudaStream_t stream);
// Dense tensor-core GEMM Y = X Wd^T + bias with Wd a dense [out][in] image (tcgen05 / TMEM / TMA).
elsa_status launch_linear_tc_dense(const uint16_t* X, int rows, const uint16_t* Wd,
                                   const uint16_t* bias, int out, int in, elsa_dtype dtype,
                                   uint16_t* Y, uint32_t* dev_status, cudaStream_t stream);

// Few token rows: the product straight from the packed weight (or the dense shared weight projected on the fly), one
// launch for up to linear_small_group_max() independent layers.  early: the weights are older than the call's first
// kernel, so their expansion may start before the predecessor kernel has ended.
struct SmallJob {
    const uint16_t* X;
    const uint16_t* w;        // packed values (N == M: the weight itself); masked: the dense shared weight
    const uint32_t* idx;
    const uint16_t* bias;
    uint16_t* Y;
    int rows, in, out, N, M;
    bool masked = false;
    int act = 0;                          // 0 none, 1 GELU
    const uint16_t* residual = nullptr;   // [rows][out], added after the activation, before the one rounding
    const void* ahead = nullptr;          // launches of one job: the next linear's weight, brought into L2 meanwhile (16-byte
    size_t ahead_bytes = 0;               // aligned; nothing reads it here, so it may still be written)
    bool chained = false;                 // one of a chain of linears with other kernels between them
    bool after_image = false;             // of a call that has just made this weight with another kernel
};
int linear_small_group_max();
// Ranges the reductions of these jobs are cut into when they run together.  A result depends on it in its last bits.
int linear_small_splits(const SmallJob* jobs, int n, int sm_count);
elsa_status launch_linear_small_group(const SmallJob* jobs, int n, int splits, bool early, elsa_dtype dtype, uint32_t* dev_status,
                                      cudaStream_t stream);

// The same GEMM on CTA pairs (cluster of two, tcgen05 cta_group::2); for large row counts.
elsa_status launch_linear_tc_pair(const uint16_t* X, int rows, const uint16_t* Wd, const uint16_t* bias,
                                  int out, int in, elsa_dtype dtype, uint16_t* Y, uint32_t* dev_status,
                                  cudaStream_t stream);
// Y [m][n] = A^T B on the same kernel with both operands stored reduction-outermost, A [k][m] and B [k][n]
// (m, n multiples of 8): the weight-gradient product dY^T X without transposed copies.
// shape: columns of a tile (256 or 128) and ranges the reduction is cut into, by linear_tc_pair_tn_shape with at most splits_most
// ranges, and with at most sums_parts rows of sums (0: none are asked for); with several ranges their fp32 sums go to
// partial [splits][m][n] (Y is then not written).  Where sums_a is not NULL, there are no more tiles than SM pairs and no part has
// too many rows for the running sums, *sums_parts rows of m floats that add up to the sums of A over the reduction go there, one
// a range and tile column; else *sums_parts is 0.
struct TnShape {
    int columns, splits;
};
TnShape linear_tc_pair_tn_shape(int m, int n, int k, int splits_most, int sums_parts, int sm_count);
elsa_status launch_linear_tc_pair_tn(const uint16_t* A, const uint16_t* B, int m, int n, int k, elsa_dtype dtype,
                                     uint16_t* Y, const TnShape& shape, float* partial, float* sums_a, int* sums_parts,
                                     uint32_t* dev_status, cudaStream_t stream);
// Levels with N <= 2 on the hardware 2:4 sparse MMA: re-encodes the packed weight into `workspace`
// (2-of-4 values + metadata), then runs the sparse GEMM.
elsa_status launch_linear_tc_sparse(const uint16_t* X, int rows, const uint16_t* vals, const uint32_t* idx,
                                    const uint16_t* bias, int out, int in, int N, int M, elsa_dtype dtype,
                                    uint16_t* Y, void* workspace, uint32_t* dev_status, cudaStream_t stream);
// Forms of the 2-of-4 image (its rows are rounded up to 32, rows past `out` are zero):
//   SP24_ROWS      [row][in/2], row r holds feature r                       (TMA-fed kernels)
//   SP24_PERMUTED  [row][in/2], row r of every block of 32 holds feature 8 * (r % 4) + r / 4 of the block: the
//                  lane order of the kernels whose epilogue transposes with stmatrix (weight-stationary)
//   SP24_TILED     permuted rows, and per (block of 32 rows, 256 k) the 16-byte units of all rows interleaved,
//                  [unit][row][16 bytes], so that a warp reads one unit of 32 rows as one contiguous run
//                  (streaming kernel); needs in % 128 == 0
enum Sp24Layout { SP24_ROWS = 0, SP24_PERMUTED = 1, SP24_TILED = 2 };
// packed weight -> 2-of-4 image + metadata blocks of 2 KB per (128 features, block_k of K), block_k = 64 or 128.
elsa_status launch_nm_to_sp24(const uint16_t* vals, const uint32_t* idx, int out, int in, int N, int M, int block_k,
                              int layout, uint16_t* a_img, uint8_t* meta, cudaStream_t stream);
// Any number of weight images, one launch per 256: the dense masked weight or its 2-of-4 form, from the packed weight
// or from the dense shared weight projected onto its level (src then holds the dense weight, idx is unused).
enum ImageKind { IMAGE_UNPACK = 0, IMAGE_SP24 = 1, IMAGE_MASK = 2, IMAGE_MASK_SP24 = 3 };
struct ImageJob {
    int kind = IMAGE_UNPACK;
    const uint16_t* src = nullptr;
    const uint32_t* idx = nullptr;
    uint16_t* dst = nullptr;
    uint8_t* meta = nullptr;      // 2-of-4 forms
    int out = 0, in = 0, N = 0, M = 0;
    int layout = SP24_ROWS, block_k = 128;
};
elsa_status launch_images(const ImageJob* jobs, int n, cudaStream_t stream);
// Where the metadata blocks start in a layer's scratch: after the image, whose rows are rounded up to 32.
inline size_t sp24_meta_offset(int out, int in) { return round_up((size_t)((out + 31) / 32 * 32) * (size_t)in, 256); }
// The same on CTA pairs (256 features x 224 rows per pair, K blocks of 128).
elsa_status launch_linear_tc_sparse_pair(const uint16_t* X, int rows, const uint16_t* vals, const uint32_t* idx,
                                         const uint16_t* bias, int out, int in, int N, int M, elsa_dtype dtype,
                                         uint16_t* Y, void* workspace, uint32_t* dev_status, cudaStream_t stream);
// Several N <= 2 layers in one persistent launch of the sparse pair kernel; each job's workspace must
// already hold its re-encoded weight (launch_linear_tc_sparse_pair_prepare).
struct SparseJob {
    const uint16_t* X;
    const uint16_t* bias;
    uint16_t* Y;
    const void* workspace;
    int rows, in, out;
    int act = 0;      // epilogue activation: 0 none, 1 GELU (weight-stationary and streaming kernels only)
    // weight-stationary kernel: the packed weight (kept values, index words, level), from which it makes its weight block
    // itself; without it (one plain layer) the block comes from the image in `workspace`
    const uint16_t* w = nullptr;
    const uint32_t* idx = nullptr;
    int N = 0, M = 0;
    // weight-stationary and streaming kernels, without an activation: [rows][out] added before the one rounding
    const uint16_t* residual = nullptr;
};
int linear_tc_sparse_pair_group_max();
elsa_status launch_linear_tc_sparse_pair_prepare(const uint16_t* vals, const uint32_t* idx, int out, int in, int N, int M,
                                                 int layout, void* workspace, cudaStream_t stream);
elsa_status launch_linear_tc_sparse_pair_group(const SparseJob* jobs, int n, elsa_dtype dtype, uint32_t* dev_status,
                                               cudaStream_t stream);
bool linear_tc_sparse_suits(int in, int N);
// The same product with the 256-feature weight block of each CTA pair resident in tensor memory for a
// whole layer (in % 128 == 0, in <= 1024); the weight as it is packed, or re-encoded as for the pair kernel (SP24_PERMUTED).
int linear_tc_sparse_ws_group_max();
bool linear_tc_sparse_ws_suits(int in, int out, int N, int sm_count);
elsa_status launch_linear_tc_sparse_ws_group(const SparseJob* jobs, int n, elsa_dtype dtype, uint32_t* dev_status,
                                             cudaStream_t stream);
size_t linear_tc_sparse_workspace(int out, int in);
// The same product with the weight block streaming through tensor memory in K chunks of 256 (in % 128 == 0,
// any length); jobs as for the pair kernel, weight image in the SP24_TILED form.
int linear_tc_sparse_st_group_max();
bool linear_tc_sparse_st_suits(int in, int N);
elsa_status launch_linear_tc_sparse_st_group(const SparseJob* jobs, int n, elsa_dtype dtype, uint32_t* dev_status,
                                             cudaStream_t stream);
elsa_status launch_linear_tc_sparse_st(const uint16_t* X, int rows, const uint16_t* vals, const uint32_t* idx,
                                       const uint16_t* bias, int out, int in, int N, int M, elsa_dtype dtype, uint16_t* Y,
                                       void* workspace, uint32_t* dev_status, cudaStream_t stream);
// Row-wise and elementwise kernels of the chained block (16-bit tensors, fp32 arithmetic, one rounding).
// R == NULL: Yn = LayerNorm(A).  R != NULL: S = A + R, and Yn = LayerNorm(S) unless Yn is NULL.  dim % 8 == 0.
// row_map (or NULL): Swin's window order of the token rows (grid H x W, windows of ws x ws, roll by shift), applied
// to where A is read (on_input) or where Yn is written (on_output).
struct RowMap {
    int H, W, ws, shift;
    int on_input, on_output;
};
elsa_status launch_layer_norm(const uint16_t* A, const uint16_t* R, uint16_t* S, const uint16_t* gain,
                              const uint16_t* beta, uint16_t* Yn, int rows, int dim, float eps, elsa_dtype dtype,
                              cudaStream_t stream, const RowMap* row_map = nullptr);
// Y = act(Y) over `count` values (count % 8 == 0); act as in the GEMM epilogues.
elsa_status launch_act_inplace(uint16_t* Y, long long count, int act, elsa_dtype dtype, cudaStream_t stream);
// dst[r][0 .. cols) = src[r][col0 .. col0 + cols); src rows of src_ld values; all multiples of 8.
elsa_status launch_copy_columns(const uint16_t* src, uint16_t* dst, int rows, int src_ld, int col0, int cols,
                                cudaStream_t stream);
// Multi-head self-attention a = softmax(q k^T / sqrt d + bias + mask) v per image and head on tcgen05 (tokens <= 256,
// head dimension 64 or 32): qkv [images * tokens][3 * dim] -> out [images * tokens][dim].  bias (or NULL):
// fp32 [heads][tokens][bias_pitch]; mask (or NULL): fp32 [n_masks][tokens][bias_pitch], image i takes table i % n_masks.
bool attention_suits(int tokens, int heads, int dim);
elsa_status launch_attention(const uint16_t* qkv, int images, int tokens, int heads, int dim, elsa_dtype dtype,
                             uint16_t* out, uint32_t* dev_status, cudaStream_t stream, const float* bias = nullptr,
                             const float* mask = nullptr, int n_masks = 0, int bias_pitch = 0);
// The same without tables for calls of few items, sixteen query rows a CTA; arguments as checked by launch_attention, which
// calls it.
bool attention_rows_suits(int images, int tokens, int heads, int head_dim, int sm_count);
elsa_status launch_attention_rows(const uint16_t* qkv, int images, int tokens, int heads, int dim, elsa_dtype dtype, uint16_t* out,
                                  uint32_t* dev_status, cudaStream_t stream, const DeviceInfo& dev);
// The same for windows that fit a warp's registers (head dimension 32, at most 64 tokens); arguments as checked by
// launch_attention, which calls it.
bool window_attention_suits(int tokens, int heads, int dim);
elsa_status launch_window_attention(const uint16_t* qkv, int windows, int tokens, int heads, int dim, elsa_dtype dtype, uint16_t* out,
                                    uint32_t* dev_status, cudaStream_t stream, const float* bias, const float* mask, int n_masks,
                                    int bias_pitch, const DeviceInfo& dev);
// Operand forms of the backward pass.  transpose_packed: dst [in][out] (out a multiple of 8) = the transposed masked weight,
// positions that were not kept zero.  colsum: db [C] = column sums of src [R][C], through ceil(R / 512) * C floats of scratch.
elsa_status launch_transpose_packed(const uint16_t* vals, const uint32_t* idx, uint16_t* dst, int out, int in, int N, int M, cudaStream_t stream);
elsa_status launch_colsum(const uint16_t* src, int R, int C, float* partial, uint16_t* db, elsa_dtype dtype, cudaStream_t stream);
// db[c] = round16(sum over parts of partial[part][c]).
elsa_status launch_colsum_finish(const float* partial, int parts, int C, uint16_t* db, elsa_dtype dtype, cudaStream_t stream);
// Zeroes the pruned positions of a dense [out][in] tensor in place.
elsa_status launch_mask_apply(uint16_t* dW, const uint32_t* idx, int out, int in, int N, int M, cudaStream_t stream);
// dW [out][in] = mask .* round16(sum over ranges of partial [splits][out][in]); idx NULL (N == M) keeps everything.  With
// db_parts > 0 also db as colsum_finish makes it.
elsa_status launch_wgrad_finish(const float* partial, int splits, const uint32_t* idx, int out, int in, int N, int M,
                                elsa_dtype dtype, uint16_t* dW, const float* db_sums, int db_parts, uint16_t* db, cudaStream_t stream);
// Any number of (weight, level) pairs, one launch per 256.
struct CompressJob {
    const uint16_t* W;
    uint16_t* vals;
    uint32_t* idx;
    int out, in, N, M;
};
elsa_status launch_compress_jobs(const CompressJob* jobs, int n, cudaStream_t stream);
constexpr int kMaxLevels = 16;

// Several dense-rate layers in one persistent launch of the CTA-pair kernel (at most
// linear_tc_pair_group_max() of them): their tiles form one sequence.
struct PairJob {
    const uint16_t* X;
    const uint16_t* Wd;     // dense weight image [out][in]
    const uint16_t* bias;
    uint16_t* Y;
    int rows, in, out;
    const float* w_scale = nullptr;   // INT8 form only
    float x_scale = 0.f;
    int act = 0;                          // epilogue activation: 0 none, 1 GELU (applied to acc + bias)
    const uint16_t* residual = nullptr;   // [rows][out], added after the activation, before the one rounding
    int splits = 1;                       // Tn form: ranges the reduction is cut into; > 1 writes fp32 sums to `partial`
    int tn_columns = 256;                 // Tn form: columns of a tile
    float* partial = nullptr;             // [splits][rows][out]
    float* sums_a = nullptr;              // Tn form: see launch_linear_tc_pair_tn
    int* sums_parts = nullptr;
};
int linear_tc_pair_group_max();
elsa_status launch_linear_tc_pair_group(const PairJob* jobs, int n, elsa_dtype dtype, uint32_t* dev_status,
                                        cudaStream_t stream);
// INT8 form of the same GEMM: X [rows][in] and the dense weight image Wd [out][in] hold signed 8-bit integers,
// accumulation is int32, Y[r][o] = round16(float(acc) * (x_scale * w_scale[o]) + bias[o]).
elsa_status launch_linear_tc_pair_i8(const int8_t* X, int rows, const int8_t* Wd, const float* w_scale, float x_scale,
                                     const uint16_t* bias, int out, int in, elsa_dtype dtype, uint16_t* Y,
                                     uint32_t* dev_status, cudaStream_t stream);
// Whether the problem has enough 256-row tiles to occupy every SM pair.
bool linear_tc_pair_suits(int rows, int out, int sm_count);

}  // namespace elsa
