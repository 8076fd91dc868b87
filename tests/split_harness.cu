// One FP64 job list with operands of the caller's choice, by the digit split on the
// tensor cores or (chain = 1) by multiply-adds on the CUDA cores:
//   split_harness < in > out
// in (little-endian): int32 project, chain, d0, d1, d2, d3, n, max_split, leg[n]; then complex doubles:
//   project = 0: n operators M_i (d x d of leg[i]) and X: out = sum_i M_i x_leg[i] X
//   project = 1: U and W: out[x', x] = sum conj(U) W over the legs other than leg[0]
// out: int32 launched, CUDA status; then the result.
#include <cstdio>
#include <vector>

#include "kernels.cuh"
#include "plan.hpp"

using namespace ttn;

namespace {

constexpr int64_t kPlanes = 1 << 20;

bool read(void* p, size_t n) { return fread(p, 1, n, stdin) == n; }

double2* upload(const std::vector<double2>& v) {
  double2* d = nullptr;
  if (cudaMalloc(&d, v.size() * sizeof(double2)) != cudaSuccess) return nullptr;
  return cudaMemcpy(d, v.data(), v.size() * sizeof(double2), cudaMemcpyHostToDevice) == cudaSuccess ? d : nullptr;
}

}  // namespace

int main() {
  int32_t hd[8];
  if (!read(hd, sizeof(hd))) return 2;
  const int dd[4] = {hd[2], hd[3], hd[4], hd[5]}, n = hd[6], max_split = hd[7];
  const bool chain = hd[1] != 0;
  const int64_t P = (int64_t)dd[0] * dd[1] * dd[2] * dd[3];
  std::vector<int32_t> leg(n);
  if (!read(leg.data(), n * sizeof(int32_t))) return 2;
  std::vector<double2*> bufs, mats;
  auto take = [&](int64_t elems, std::vector<double2*>& to) {
    std::vector<double2> v(elems);
    if (!read(v.data(), elems * sizeof(double2))) return false;
    to.push_back(upload(v));
    return to.back() != nullptr;
  };
  const int64_t n_res = hd[0] ? (int64_t)dd[leg[0]] * dd[leg[0]] : P;
  double flops = 0.0;
  std::vector<ApTerm> terms;
  if (hd[0] == 0) {
    for (int i = 0; i < n; ++i) {
      if (!take((int64_t)dd[leg[i]] * dd[leg[i]], mats)) return 3;
      terms.push_back(ApTerm{i, leg[i], 0, 0});
      flops += 8.0 * P * dd[leg[i]];
    }
    if (!take(P, bufs)) return 3;
  } else {
    if (!take(P, bufs) || !take(P, bufs)) return 3;
    flops = 8.0 * P * dd[leg[0]];
  }
  double2* res = upload(std::vector<double2>(n_res, make_double2(0.0, 0.0)));
  double2* planes = upload(std::vector<double2>(std::max(kPlanes, 4 * P), make_double2(0.0, 0.0)));
  if (!res || !planes) return 3;
  int32_t st[2] = {0, 0};
  if (hd[0] == 0) {
    bufs.push_back(res);
    const ApOut out{dd[0], dd[1], dd[2], 0, n, 1, 0, dd[3]};
    ApList L{0, 1, (int)((P + 31) / 32)};
    L.flops = flops;
    const Epi store{EPI_STORE, nullptr, nullptr, nullptr, nullptr, 0.0};
    if (chain) {
      launch_apply(PREC_F64, DevTables{}, HostTables{(void* const*)bufs.data(), (void* const*)mats.data(), &out, terms.data(), nullptr},
                   L, store, nullptr);
      st[0] = n <= 12;  // the tables fit the launch's parameters
    } else {
      st[0] = xs_applicable(L, &out, terms.data(), max_split) &&
              launch_apply_xs(bufs.data(), mats.data(), L, store, &out, terms.data(), planes, std::max(kPlanes, 4 * P),
                              max_split, nullptr);
    }
  } else {
    mats.push_back(res);
    const PjOut out{dd[0], dd[1], dd[2], leg[0], 0, 1, 0, 0};
    PjList L{0, 1, (int)((n_res + 31) / 32)};
    L.flops = flops;
    if (chain) {
      launch_project(PREC_F64, DevTables{}, HostTables{(void* const*)bufs.data(), (void* const*)mats.data(), nullptr, nullptr, &out},
                     L, nullptr);
      st[0] = 1;
    } else {
      st[0] = launch_project_xs(bufs.data(), mats.data(), L, &out, max_split, nullptr);
    }
  }
  std::vector<double2> back(n_res);
  st[1] = (int32_t)cudaMemcpy(back.data(), res, n_res * sizeof(double2), cudaMemcpyDeviceToHost);
  fwrite(st, sizeof(st), 1, stdout);
  fwrite(back.data(), sizeof(double2), n_res, stdout);
  return 0;
}
