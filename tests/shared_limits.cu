// The dynamic shared memory limits of the kernels whose need depends on the call (KNN: knn_tc.cu, else warm.cu),
// as the calls so far have left them.  Linked in place of that file's object (tests/test_gpu_shared_limits.py).
#ifdef KNN
#include "../paper_2408_05459_gb300/csrc/knn_tc.cu"
#else
#include "../paper_2408_05459_gb300/csrc/warm.cu"
#endif

template <class F>
static int limit_of(F* kernel) {
  cudaFuncAttributes a{};
  return cudaFuncGetAttributes(&a, kernel) == cudaSuccess ? a.maxDynamicSharedSizeBytes : -1;
}

#ifdef KNN
extern "C" void knn_limits(int* out) {
  using namespace ancka;
  out[0] = limit_of(k_knn_pair<false, false>);
  out[1] = limit_of(k_knn_pair<false, true>);
  out[2] = limit_of(k_knn_pair<true, false>);
  out[3] = limit_of(k_knn_tc<false>);
  out[4] = limit_of(k_knn_tc<true>);
  out[5] = limit_of(k_knn_sym);
}
#else
extern "C" void warm_limits(int* out) {
  using namespace ancka;
  out[0] = limit_of(k_mlp_out);
  out[1] = limit_of(k_warm_coeffs);
}
#endif
