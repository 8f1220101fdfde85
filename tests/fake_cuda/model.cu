// The few kernels that the runtime without a device models: the end of a block of iterations
// (k_true_residual; in three dimensions k3_finish<3>), which counts fake_model's iterations and decides;
// the 3-D iteration's decisions on a given run of residuals; the 3-D set-up's counts and norm; and the transform products, which raise the time-out flag on demand.
#include "model.h"

#include <vector>

#include "../../paper_1704_08897_gb300/csrc/common.cuh"

static struct Model {
  int its = 1;           // iterations a block makes
  int ok_after = 0;      // blocks until convergence (0: never)
  int err_after = 0;     // transform products until one raises the time-out flag (0: none)
  int blocks = 0, products = 0;
} model;

static std::vector<double> residuals;   // 3-D: ||r||^2 / ||b||^2 after each iteration
static std::vector<int> replaced;       // the iterations at which the residual was replaced

// what the kernel does, with its arguments read now
std::function<void()> body(const std::string& k, void** a) {
  using bx::SlotScalars;
  auto block_end = [](SlotScalars* sc) {
    if (sc->status != bx::ST_RUNNING) return;
    ++model.blocks;
    sc->it += model.its;
    sc->rr = sc->rr_true = sc->bb * 1e-4 / model.blocks;
    if (model.ok_after && model.blocks >= model.ok_after) sc->status = bx::ST_OK;
    else if (sc->it >= sc->maxit) sc->status = bx::ST_ENOTCONV;
  };
  if (k.find("PKNS_8SlotDescEPKNS_8WorkItemEPKi") != std::string::npos)  // descriptors, work list, its length
    for (int i = 0; i < 3; ++i)
      if (!in_device_memory(*(const void**)a[i])) {
        fault(k + ": argument outside a live allocation");
        return [] {};
      }
  if (k.find("k_true_residual") != std::string::npos) {
    auto slots = *(const bx::SlotDesc**)a[0];
    auto items = *(const bx::WorkItem**)a[1];
    auto n = *(const int**)a[2];
    return [=] {
      for (int i = 0; i < *n; ++i)
        if (items[i].tile == 0) block_end(slots[items[i].slot].sc);
    };
  }
  if (k.find("k3_finishILi1E") != std::string::npos && !residuals.empty()) {
    auto sc = *(SlotScalars**)a[0];
    return [=] {
      if (sc->active) bx::decide_update3(sc, sc->bb * residuals.at(sc->it));
    };
  }
  if (k.find("k3_finishILi3E") != std::string::npos) {
    auto sc = *(SlotScalars**)a[0];
    return [=] {
      if (residuals.empty()) return block_end(sc);
      if (!sc->fold) return;
      replaced.push_back(sc->it);
      bx::decide_true(sc, sc->bb * residuals.at(sc->it - 1) * 1.0001);
    };
  }
  if (k.find("k3_setup") != std::string::npos) {
    const size_t n = *(size_t*)a[0];
    auto c = *(unsigned long long**)a[6];
    return [=] { c[0] = n / 2, c[1] = n - n / 2; };
  }
  if (k.find("k3_sum") != std::string::npos) {
    auto out = *(double**)a[2];
    return [=] { *out = 1.0; };
  }
  if (k.find("k_prec_tc") != std::string::npos) {
    auto err = *(int**)a[4];
    return [=] {
      if (++model.products == model.err_after) *err = 1;
    };
  }
  return [] {};
}

extern "C" {
void fake_model(int its, int ok_after, int err_after) { model = Model{its, ok_after, err_after, 0, 0}; }
void fake_residuals(const double* r, int n) {
  residuals.assign(r, r + n);
  replaced.clear();
}
int fake_replaced(int* its, int n) {
  for (int i = 0; i < n && i < (int)replaced.size(); ++i) its[i] = replaced[i];
  return (int)replaced.size();
}
int fake_blocks() { return model.blocks; }
int fake_products() { return model.products; }
}
