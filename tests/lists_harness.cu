// Host access to the library's job lists for the tests: builds the plan of a
// model and hands every FP64 contraction list to the tensor-core launcher, as
// the executor does.
//
//   lists < model        one line per list: applicable launched n_outs n_terms d0 d1 d2 d3
//
// model (numbers separated by white space): n_nodes parent[] n_legs leg_node[]
// leg_dims[] ranks[] n_ops op_leg[] n_data op_offset[] op_data[] n_terms
// term_offsets[] n_fac term_ops[] coef[] coef_drive[] max_split
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <iostream>
#include <vector>

#include "kernels.cuh"
#include "plan.hpp"

using namespace ttn;

namespace {

template <typename T>
std::vector<T> read(size_t n) {
  std::vector<T> v(n);
  for (T& x : v) std::cin >> x;
  return v;
}
int read1() {
  int v = 0;
  std::cin >> v;
  return v;
}

int lists() {
  const int n = read1();
  const auto parent = read<int32_t>(n);
  const int nl = read1();
  const auto leg_node = read<int32_t>(nl), leg_dims = read<int32_t>(nl), ranks = read<int32_t>(n);
  const int n_ops = read1();
  const auto op_leg = read<int32_t>(n_ops);
  const int nd = read1();
  const auto op_offset = read<int64_t>(n_ops);
  const auto op_data = read<double>(nd);
  const int n_terms = read1();
  const auto term_offsets = read<int32_t>(n_terms + 1);
  const auto term_ops = read<int32_t>(read1());
  const auto coef = read<double>(2 * n_terms);
  const auto coef_drive = read<int32_t>(n_terms);
  const int max_split = read1();
  Plan p;
  std::string e = p.build(n, parent.data(), nl, leg_node.data(), leg_dims.data(), ranks.data());
  if (e.empty())
    e = p.load_sop(n_ops, op_leg.data(), op_offset.data(), op_data.data(), n_terms, term_offsets.data(),
                   term_ops.data(), coef.data(), coef_drive.data());
  if (e.empty()) {
    p.set_caps(32);
    e = p.rebuild_classes();
  }
  if (!e.empty()) {
    std::fprintf(stderr, "%s\n", e.c_str());
    return 2;
  }
  std::vector<double2*> bufs(p.buf.n_bufs, nullptr), mats(p.mats.size(), nullptr);
  const int64_t planes = std::max<int64_t>(4 * std::max(p.P_cap_max, p.theta_cap), std::min<int64_t>(24 * p.P_cap_max, 1 << 20));
  for (const ApList& L : p.ap_lists) {
    const ApOut& f = p.ap_outs[L.out_begin];
    const bool ok = xs_applicable(L, p.ap_outs.data(), p.ap_terms.data(), 1);  // the lower line claims the most lists
    const Epi store{EPI_STORE, nullptr, nullptr, nullptr, nullptr, 0.0};
    const bool done = ok && launch_apply_xs(bufs.data(), mats.data(), L, store, p.ap_outs.data(), p.ap_terms.data(),
                                            nullptr, planes, max_split, nullptr);
    std::printf("%d %d %d %d %d %d %d %d\n", (int)ok, (int)done, L.out_end - L.out_begin,
                p.ap_outs[L.out_end - 1].term_end - f.term_begin, f.d0, f.d1, f.d2, f.d3);
  }
  return 0;
}

}  // namespace

int main(int argc, char** argv) {
  if (argc == 2 && !std::strcmp(argv[1], "lists")) return lists();
  std::fprintf(stderr, "usage: lists_harness lists\n");
  return 2;
}
