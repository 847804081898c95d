// The inner BiCGStab of small systems in one launch (internal).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "krylov.h"

namespace ddps {

// Up to kInnerRows consecutive rows of G^ held by one CTA (they share the block).
constexpr int kInnerRows = 8;
struct InnerGroup {
  int64_t gsrc;    // offset of the first row in G^
  int32_t goff;    // offset of the first row in the CTA's copy
  int32_t row;     // first row within the CTA's slice of the vectors
  int32_t nrows;
  int32_t xoff;    // offset of the block's gathered vector
  int32_t nc, ld;  // coupling columns, row stride
};
// One CTA: a slice of one system's reduced rows.
struct InnerCta {
  int32_t sys, q0;             // system, its first reduced row
  int32_t row0, nrows;         // the slice, within the system
  int32_t grp0, ngrp;          // groups
  int32_t col0, ncol;          // gathered columns of all blocks of the slice
};
// Systems launched together: CTAs [cta0, cta0 + ncta), and the sizes of the
// shared-memory arrays (the largest of the class).
struct InnerClass {
  int32_t cs;       // CTAs per system (cluster size)
  bool held;        // rows of G^ in shared memory, else streamed
  int32_t cta0, ncta;
  int32_t g_elems, cols, rows, groups;
  size_t smem;
};

struct InnerPlan {
  bool ok = false;  // every system fits a cluster
  std::vector<InnerClass> classes;
  std::vector<InnerCta> h_ctas;
  std::vector<InnerGroup> h_groups;
  std::vector<int32_t> h_cols;
  const InnerCta* ctas = nullptr;
  const InnerGroup* groups = nullptr;
  const int32_t* cols = nullptr;
};

struct InnerInput {
  int32_t nsys;
  const int64_t *sys_c_ptr;            // nsys + 1
  const int32_t *sys_block_ptr;        // nsys + 1
  const int64_t *gq0, *gq1, *gcol_ptr, *ghat_off, *gld;
  const int32_t* gcols_panel;          // coupling columns in G^ column order (reduced indices)
  int32_t size_g, size_acc, size_i;    // bytes of a stored entry, an accumulator, a vector entry
  int32_t nsm;                         // SMs of the device
};
// Plans the launch; P.ok stays false when some system needs more shared
// memory than a cluster has.
void plan_inner_cluster(const InnerInput& in, InnerPlan& P);

// z = G^-1 g for every system, from z0 (may be null); sc[s] receives system
// s's scalars: iters, active (0), flag = 1 when its guess was used.  Systems that the
// outer iteration has finished (outer[s].active = 0; outer may be null) get z = 0.  Returns the
// number of launches.
template <typename TG, typename TI>
int launch_inner_cluster(const InnerPlan& P, const TG* ghat, const double* g64, const double* z064,
                         double* z64, KScal* sc, const KScal* outer, double tol, int maxit,
                         cudaStream_t s);

}  // namespace ddps
