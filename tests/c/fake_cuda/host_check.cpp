// The library's host side on the stand-in runtime (fake_cuda.cpp): prints what
// went wrong, one line each.
#include <varlingam_gb300.h>

#include <cstdio>
#include <cstring>

#include "fake_cuda.h"

#include <cuda_runtime_api.h>

namespace {

double* const X = reinterpret_cast<double*>(uintptr_t(1) << 44);  // never read
int32_t* const ORDER = reinterpret_cast<int32_t*>(uintptr_t(1) << 45);

void report(const char* call, int device, int m, vl_status s) {
  for (const fake::Launch& l : fake::launches)
    if (l.refused)
      std::printf("%s m=%d device %d: refused %s with %zu bytes\n", call, m, device,
                  l.name.c_str(), l.smem);
  if (s != VL_OK) std::printf("%s m=%d device %d: status %d\n", call, m, device, (int)s);
  fake::launches.clear();
}

// Every call on the first device, then on the second.
void two_devices() {
  for (int d = 0; d < 2; ++d) {
    cudaSetDevice(d);
    vl_handle h;
    if (vl_create(&h, d, nullptr, 0) != VL_OK) std::printf("vl_create\n");
    for (int m : {20, 40, 64, 78, 79, 100, 160, 161, 300, 448, 449, 512, 600}) {
      const int n = 3 * m + 50;
      report("vl_causal_order", d, m, vl_causal_order(h, X, m, ORDER, X));
      report("vl_causal_order_certified", d, m,
             vl_causal_order_certified(h, X, X, n, m, n, ORDER, X, nullptr));
      if (m <= VL_NOALLOC_MAX_M)
        report("vl_causal_order_noalloc", d, m,
               vl_causal_order_noalloc(nullptr, X, m, ORDER, X));
      for (vl_precision prec : {VL_PREC_MIXED, VL_PREC_FP64}) {
        report("vl_pairwise_measure", d, m,
               vl_pairwise_measure(h, X, n, m, n, prec, X, X, X));
        report("vl_var_fit", d, m, vl_var_fit(h, X, n, m, n, 2, prec, X, X));
        report("vl_fit_b", d, m, vl_fit_b(h, X, n, m, n, ORDER, X, 1, prec, X, X));
      }
      vl_instance I[2] = {{X, n, m, n, 1, ORDER, X, X, X, X}, {X, n, m, n, 1, ORDER, X, X, X, X}};
      vl_status st[2];
      report("vl_fit_batched", d, m, vl_fit_batched(h, I, 2, VL_PREC_MIXED, st));
    }
    vl_destroy(h);
  }
}

// A search that cannot be launched: another takes its place; without any, the
// call fails and nothing that would use the order as an index is launched.
void no_search() {
  vl_handle h;
  if (vl_create(&h, 0, nullptr, 0) != VL_OK) std::printf("vl_create\n");
  for (int m : {50, 160, 300}) {
    const int n = 3 * m + 50;
    const vl_instance I{X, n, m, n, 1, ORDER, X, X, X, X};
    fake::refuse = {"order_local_kernel", "order_cluster_kernel"};
    vl_status s = vl_causal_order(h, X, m, ORDER, X);
    if (s != VL_OK || !fake::launched("order_kernel")) std::printf("m=%d: no other search\n", m);
    s = vl_causal_order_noalloc(nullptr, X, m, ORDER, X);
    if (s != VL_OK) std::printf("m=%d: no other search without allocation\n", m);
    fake::refuse.push_back("order_kernel");
    for (int call = 0; call < 5; ++call) {
      fake::launches.clear();
      vl_status st = VL_OK;
      if (call == 0) s = vl_causal_order(h, X, m, ORDER, X);
      if (call == 1) s = vl_causal_order_noalloc(nullptr, X, m, ORDER, X);
      if (call == 2) s = vl_causal_order_certified(h, X, X, n, m, n, ORDER, X, nullptr);
      if (call == 3) s = vl_fit(h, X, n, m, n, 1, VL_PREC_MIXED, X, ORDER, X, X, X);
      if (call == 4) s = vl_fit_batched(h, &I, 1, VL_PREC_MIXED_CERTIFIED, &st);
      if (s != VL_ERR_CUDA) std::printf("m=%d call %d: status %d\n", m, call, (int)s);
      for (const char* k : {"gap_scores_kernel", "cert_", "permute_cov_kernel"})
        if (fake::launched(k)) std::printf("m=%d call %d: %s without an order\n", m, call, k);
    }
    fake::refuse.clear();
  }
  vl_destroy(h);
}

// Which calls' launches overlap: those up to m n = 2^18, but never a batch's or an
// FP64 product's.
void overlap() {
  vl_handle h;
  if (vl_create(&h, 0, nullptr, 0) != VL_OK) std::printf("vl_create\n");
  const struct {
    int m, n;
    bool overlap;
  } sizes[] = {{10, 1000, true}, {64, 4096, true}, {64, 4097, false}, {400, 2500, false}};
  for (const auto& z : sizes)
    for (vl_precision prec : {VL_PREC_MIXED, VL_PREC_FP64})
      for (int call = 0; call < 7; ++call) {
        const vl_instance I{X, z.n, z.m, z.n, 1, ORDER, X, X, X, X};
        vl_status st;
        fake::launches.clear();
        if (call == 0) vl_var_fit(h, X, z.n, z.m, z.n, 1, prec, X, X);
        if (call == 1) vl_pairwise_measure(h, X, z.n, z.m, z.n, prec, X, X, X);
        if (call == 2) vl_causal_order_standard(h, X, z.n, z.m, z.n, prec, ORDER, X);
        if (call == 3) vl_fit_b(h, X, z.n, z.m, z.n, ORDER, X, 1, prec, X, X);
        if (call == 4) vl_fit(h, X, z.n, z.m, z.n, 1, prec, X, ORDER, X, X, X);
        if (call == 5) vl_var_select(h, X, z.n, z.m, z.n, 2, VL_IC_BIC, prec, X, ORDER);
        if (call == 6) vl_fit_batched(h, &I, 1, prec, &st);
        bool any = false, product = false;
        for (const fake::Launch& l : fake::launches) {
          any |= l.overlap;
          product |= l.overlap && l.name.find("gemm_kernelIdd") != std::string::npos;
        }
        if (any != (z.overlap && call != 6) || product)
          std::printf("call %d m=%d n=%d precision %d: overlap %d, FP64 product %d\n", call, z.m,
                      z.n, (int)prec, any, product);
      }
  vl_destroy(h);
}

}  // namespace

int main(int argc, char** argv) {
  if (argc == 2 && !std::strcmp(argv[1], "two_devices")) two_devices();
  if (argc == 2 && !std::strcmp(argv[1], "no_search")) no_search();
  if (argc == 2 && !std::strcmp(argv[1], "overlap")) overlap();
  return 0;
}
