// The tensor-core passes of csrc/knn_tc.cu with a chosen one left out, as after an expired pipeline wait: its
// error word is set, and its outputs hold 0x7f bytes, which no kernel may take for indices.  Linked with the
// library's other objects in place of knn_tc.o (tests/test_gpu_failed_passes.py).
#define knn_candidates_bf16 real_candidates_bf16
#define knn_candidates_bf16_shares real_candidates_bf16_shares
#define knn_lists_bf16 real_lists_bf16
#define knn_collect_bf16 real_collect_bf16
#include "../paper_2408_05459_gb300/csrc/knn_tc.cu"
#undef knn_candidates_bf16
#undef knn_candidates_bf16_shares
#undef knn_lists_bf16
#undef knn_collect_bf16

namespace ancka {

namespace {
int g_countdown = 0;
bool fails() { return g_countdown > 0 && --g_countdown == 0; }

ancka_status fail(float* cand_val, int32_t* cand_idx, size_t entries, int32_t* err, cudaStream_t s) {
  ANCKA_CUDA(cudaMemsetAsync(cand_val, 0x7f, entries * sizeof(float), s));
  ANCKA_CUDA(cudaMemsetAsync(cand_idx, 0x7f, entries * sizeof(int32_t), s));
  ANCKA_CUDA(cudaMemsetAsync(err, 5, 1, s));  // the low byte of a zeroed word
  return ANCKA_OK;
}
}  // namespace

ancka_status knn_candidates_bf16(Workspace& ws, const PrepOut& pr, int64_t n, float* cand_val, int32_t* cand_idx,
                                 int32_t* err, cudaStream_t s) {
  if (fails()) return fail(cand_val, cand_idx, (size_t)n * kCandC, err, s);
  return real_candidates_bf16(ws, pr, n, cand_val, cand_idx, err, s);
}

ancka_status knn_candidates_bf16_shares(Workspace& ws, const PrepOut& pr, int64_t n, int shares, float* cand_val,
                                        int32_t* cand_idx, int32_t* err, cudaStream_t s) {
  if (fails()) return fail(cand_val, cand_idx, (size_t)n * shares * kCandC, err, s);
  return real_candidates_bf16_shares(ws, pr, n, shares, cand_val, cand_idx, err, s);
}

// the buffers hold n_rows lists at least
ancka_status knn_lists_bf16(Workspace& ws, const __nv_bfloat16* a, int64_t a_rows_total, const int32_t* rows,
                            int64_t n_rows, const __nv_bfloat16* keys, int64_t n_keys, int64_t keys_pad, int dp, int d,
                            const int64_t* blk_ptr, const int32_t* blk_tiles, int64_t blk_work, bool no_self,
                            float* cand_val, int32_t* cand_idx, int32_t* err, cudaStream_t s) {
  if (fails()) return fail(cand_val, cand_idx, (size_t)n_rows * kCandC, err, s);
  return real_lists_bf16(ws, a, a_rows_total, rows, n_rows, keys, n_keys, keys_pad, dp, d, blk_ptr, blk_tiles,
                         blk_work, no_self, cand_val, cand_idx, err, s);
}

ancka_status knn_collect_bf16(Workspace& ws, const PrepOut& pr, int64_t n, const int32_t* rows, int64_t n_a,
                              const float* thr, int32_t* cnt, int32_t* buf, int cap, int32_t* err, cudaStream_t s) {
  if (!fails()) return real_collect_bf16(ws, pr, n, rows, n_a, thr, cnt, buf, cap, err, s);
  ANCKA_CUDA(cudaMemset2DAsync(cnt, sizeof(int32_t), 100, 1, (size_t)n_a, s));  // 100 keys a row
  ANCKA_CUDA(cudaMemsetAsync(buf, 0x7f, (size_t)n_a * cap * sizeof(int32_t), s));
  ANCKA_CUDA(cudaMemsetAsync(err, 5, 1, s));
  return ANCKA_OK;
}

}  // namespace ancka

// the nth pass from now fails (0: none)
extern "C" void set_failing_pass(int nth) { ancka::g_countdown = nth; }
