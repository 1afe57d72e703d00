// lbw_resident.h -- host interface of the multi-step kernel for small lattices
// (lbw_resident.cu).
#pragma once

#include <vector>

#include "lbw_internal.h"

namespace lbw {

constexpr int kResChunk = 256;  // time steps per launch at most

// One box of one lattice, owned by one CTA during a launch: the CTAs of a lattice share a
// barrier (group); src_lo .. src_hi - 1 are its harmonic sources in Resident::src_order.
struct ResItem {
  int member, x0, y0, z0, bx, by, bz, group, group_size, src_lo, src_hi, pad;
};

struct Resident {
  struct Launch {
    int first = 0, count = 0, groups = 0;  // items [first, first + count), one CTA each
    int own = 0, threads = 0, smem = 0;  // nodes of the largest box, launch shape
  };
  std::vector<Launch> launches;  // an ensemble's lattices in turns of what the SMs hold
  std::vector<ResItem> host_items;
  int prec = 0;
  bool tile = false;             // operations of the tile kernels (see lbw_resident.cu)
  bool x13 = false;              // some lattice's metric couples q1 and q3
  long long nodes = 0;           // of all lattices
  int most = 0;                  // sources of the box that holds the most
  ResItem* items = nullptr;
  unsigned* bars = nullptr;
  int* src_order = nullptr;
};

// What a run needs of the lattice or ensemble that it advances.
struct ResState {
  void* f[2];
  int cur;
  unsigned long long* counters;
  const unsigned long long* stall;  // injected-timeout request, or nullptr
  int nprobe;
  long long cap;
  const SourceEntry* src;
  int src_kind;
  double src_amp;
  cudaStream_t stream;
};

// Plans the launches for n lattices of one storage type; *out stays nullptr when they do not
// fit (a lattice of more nodes than the SMs hold, more than max_nodes in all) or ask for
// another source of the geometry than AUTO.
lbw_status resident_create(const Grid* const* lattices, int n, int prec, bool tile, long long max_nodes,
                           cudaStream_t stream, Resident** out);
void resident_destroy(Resident* r, cudaStream_t stream);
// Assigns the sources (per_lattice nodes of each lattice, in SourceEntry order) to the boxes; none
// (0) before their list is freed, which needs no memory.
lbw_status resident_sources(Resident* r, const int32_t* host_q, int per_lattice, cudaStream_t stream);
// Whether it is ahead of a launch per step with the sources that it has (a box's sources are served
// by one SM, which a plate of several planes keeps busy).
bool resident_pays(const Resident* r, int src_kind);
// `steps` <= kResChunk time steps from buffer st.cur: of the lattice `one`, or of an ensemble
// with StepArgs array `members` (source buffer 0).
cudaError_t resident_run(const Resident* r, const Grid* one, const void* members, const ResState& st, int steps);

}  // namespace lbw
