// One epoch of a made-up task list through the library's launcher: `tasks`
// tasks of one rating each, item t by user t mod users, all of them waiting for
// the given versions except the first, which waits for nothing.
#include <vector>

#include "kernels.h"

using namespace bsvd;

namespace {
template <typename T>
T *put(const T *h, size_t n) {
  T *d = nullptr;
  if (cudaMalloc(&d, n * sizeof(T)) != cudaSuccess) return nullptr;
  cudaMemcpy(d, h, n * sizeof(T), cudaMemcpyHostToDevice);
  return d;
}
}  // namespace

// out: the error word, the epoch's control words. Returns the CUDA status.
extern "C" int give_up(int f32, int k, int tasks, int users, unsigned other_ver,
                       unsigned own_ver, unsigned idle_polls,
                       unsigned long long *out) {
  std::vector<unsigned> first(tasks + 1), ov(tasks, other_ver), wv(tasks, own_ver);
  std::vector<int32_t> own(tasks), other(tasks);
  std::vector<float> x(tasks, 3.f);
  ov[0] = wv[0] = 0;
  for (int t = 0; t <= tasks; ++t) first[t] = t;
  for (int t = 0; t < tasks; ++t) {
    own[t] = t;
    other[t] = t % users;
  }
  const std::vector<double> zero((size_t)(tasks + users) * (k + 1), 0.0);
  const std::vector<unsigned long long> rows(zero.size() * 2, 0), ctl(3, 0);
  const int64_t ntasks = tasks;
  const int32_t none = 0;
  double *P = put(zero.data(), zero.size()), *Q = put(zero.data(), zero.size());
  double *bu = put(zero.data(), zero.size()), *bi = put(zero.data(), zero.size());
  SgdEpoch e;
  e.task_first = put(first.data(), first.size());
  e.ntasks = put(&ntasks, 1);
  e.own = put(own.data(), own.size());
  e.other = put(other.data(), other.size());
  e.x = put(x.data(), x.size());
  e.other_ver = put(ov.data(), ov.size());
  e.own_ver = put(wv.data(), wv.size());
  e.own_rows = put(rows.data(), rows.size());
  e.other_rows = put(rows.data(), rows.size());
  e.r = SgdRates{0.01, 0.01, 0.01, 0.01, 0.01, 0.01, 0.01, 0.01};
  e.own_items = 1;
  e.k = k;
  e.ctl = put(ctl.data(), ctl.size());
  e.err = put(&none, 1);
  e.idle_polls = idle_polls;
  cudaError_t s = launch_sgd_rows(1, f32, users, tasks, k, P, Q, bu, bi,
                                  e.other_rows, e.own_rows, e.ctl, nullptr);
  if (s == cudaSuccess) s = launch_sgd_epoch(e, tasks, f32, 152, nullptr);
  if (s == cudaSuccess) s = cudaDeviceSynchronize();
  int32_t err = 0;
  if (s == cudaSuccess) {
    cudaMemcpy(&err, e.err, sizeof err, cudaMemcpyDeviceToHost);
    s = cudaMemcpy(out + 1, e.ctl, 3 * sizeof *out, cudaMemcpyDeviceToHost);
  }
  out[0] = (unsigned long long)err;
  const void *all[] = {P, Q, bu, bi, e.task_first, e.ntasks, e.own, e.other,
                       e.x, e.other_ver, e.own_ver, e.own_rows, e.other_rows,
                       e.ctl, e.err};
  for (const void *p : all) cudaFree(const_cast<void *>(p));
  return (int)s;
}
