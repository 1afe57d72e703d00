// What the launches of the step kernels are given, checked by the fake runtime (fake_runtime.cpp):
// every pointer has to be a live allocation.
#include <string>

#include "lbw_march.cuh"
#include "lbw_resident.h"

void fake_want_live(const void* p, const char* what);

namespace {

// a step kernel's arguments for one lattice
template <typename S>
void check_args(const lbw::dev::StepArgs<S>& a) {
  fake_want_live(a.fin, "populations read");
  fake_want_live(a.fout, "populations written");
  fake_want_live(a.tab, "coefficient table");
  fake_want_live(a.counters, "counters");
  if (a.nprobe > 0) {
    fake_want_live(a.probe_q, "probe nodes");
    fake_want_live(a.series, "probe series");
  }
}

template <typename S>
void check_ensemble(void** args, int items) {
  const auto* members = *static_cast<const lbw::dev::StepArgs<S>**>(args[0]);
  fake_want_live(members, "members");
  fake_want_live(*static_cast<void**>(args[items]), "work list");
  if (members) check_args(members[0]);
}

}  // namespace

void fake_check_launch(const std::string& name, void** args) {
  auto has = [&](const char* part) { return name.find(part) != std::string::npos; };
  const bool tiled = has("batch_tma_kernel") || has("batch_row_kernel");
  if (!tiled && !has("batch_step_kernel")) return;
  const int items = tiled ? 3 : 1;
  if (has("kernelId")) check_ensemble<double>(args, items);
  else if (has("kernelIf")) check_ensemble<float>(args, items);
  else if (has("bfloat16")) check_ensemble<__nv_bfloat16>(args, items);
  else check_ensemble<__half>(args, items);
}

// The multi-step kernel's plan as it is when a launch reads it (linked with --wrap): ranges of sources
// only where the lists that they index are alive.
cudaError_t real_resident_run(const lbw::Resident* r, const lbw::Grid* one, const void* members,
                              const lbw::ResState& st, int steps)
    asm("__real__ZN3lbw12resident_runEPKNS_8ResidentEPKNS_4GridEPKvRKNS_8ResStateEi");
cudaError_t wrap_resident_run(const lbw::Resident* r, const lbw::Grid* one, const void* members,
                              const lbw::ResState& st, int steps)
    asm("__wrap__ZN3lbw12resident_runEPKNS_8ResidentEPKNS_4GridEPKvRKNS_8ResStateEi");
cudaError_t wrap_resident_run(const lbw::Resident* r, const lbw::Grid* one, const void* members,
                              const lbw::ResState& st, int steps) {
  fake_want_live(r->items, "boxes");
  fake_want_live(r->bars, "barriers");
  for (size_t k = 0; k < r->host_items.size(); ++k)
    if (r->items[k].src_hi > r->items[k].src_lo) {
      fake_want_live(st.src, "source list");
      fake_want_live(r->src_order, "source order");
      break;
    }
  if (one && one->nprobe > 0) {
    fake_want_live(one->probe_q, "probe nodes");
    fake_want_live(one->series, "probe series");
  }
  if (members) {
    void* list = const_cast<void*>(members);
    void* args[] = {&list, &list};  // no work list: the members stand in for it
    if (r->prec == LBW_F64) check_ensemble<double>(args, 1);
    else if (r->prec == LBW_F32) check_ensemble<float>(args, 1);
    else if (r->prec == LBW_F16S) check_ensemble<__half>(args, 1);
    else check_ensemble<__nv_bfloat16>(args, 1);
  }
  return real_resident_run(r, one, members, st, steps);
}
