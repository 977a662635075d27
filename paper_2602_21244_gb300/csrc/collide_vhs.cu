// VHS isotropic scatter with the centre-of-mass update (Sec. 2.1, 2.3).
//
// One persistent launch walks the pairs of the step in round-major order:
// each warp claims 32 pairs of one round at a time from a global cursor and
// each lane waits (bounded) until the previous pairs of its two particles
// are done, then updates its pair and stamps both particles done.  The
// pairs of a round are disjoint, so no two lanes of a unit touch the same
// particle.  Velocities are read and written through L2 (ld/st .cg).
#include "internal.cuh"
#include "pair.cuh"

namespace dsmc {

struct VhsArgs {
  uint64_t seed, step;
  const uint64_t* step_dev;
  const int4* pairs;
  const uint32_t* deps;
  const int32_t* ro;
  const dsmc_select_info_t* info;
  double *vx, *vy, *vz;
  unsigned* done;
  unsigned* bar;   // [2] abort word, [3] unit cursor
  int* status;
};

__global__ void __launch_bounds__(256) k_collide_vhs(VhsArgs a) {
  dep_wait();
  if (a.step_dev) a.step = *a.step_dev;
  const int R = a.info->n_rounds;
  const int lane = threadIdx.x & 31;
  int r = 0;
  int64_t base = 0;
  // the next unit claimed and its pair records loading while the current
  // one updates (as in k_collide_table)
  auto claim = [&](int32_t* u0, int32_t* u1, int* ur) {
    unsigned unit = 0;
    if (lane == 0) unit = atomicAdd(a.bar + 3, 1u);
    unit = __shfl_sync(0xffffffffu, unit, 0);
    const bool got = unit_range(a.ro, R, 32, r, base, unit, u0, u1);
    *ur = r;
    return got;
  };
  int32_t p0 = 0, p1 = 0;
  int rc = 0;
  bool have = claim(&p0, &p1, &rc);
  int4 q = make_int4(0, 0, 0, 0);
  uint32_t dep = 0u;
  if (have && p0 + lane < p1) { q = a.pairs[p0 + lane]; dep = a.deps[p0 + lane]; }
  while (have) {
    int32_t n0 = 0, n1 = 0;
    int rn = 0;
    const bool next = claim(&n0, &n1, &rn);
    int4 qn = make_int4(0, 0, 0, 0);
    uint32_t depn = 0u;
    if (next && n0 + lane < n1) { qn = a.pairs[n0 + lane]; depn = a.deps[n0 + lane]; }
    const bool valid = p0 + lane < p1;
    bool ok = true;
    if (valid) ok = wait_deps(a.done, q.x, q.y, dep, a.bar + 2, a.status);
    const bool live = valid && ok;
    double v[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    if (live) {
      v[0] = __ldcg(a.vx + q.x); v[1] = __ldcg(a.vy + q.x); v[2] = __ldcg(a.vz + q.x);
      v[3] = __ldcg(a.vx + q.y); v[4] = __ldcg(a.vy + q.y); v[5] = __ldcg(a.vz + q.y);
    }
    // the lanes leave their dependency waits at different times: every lane
    // runs the pair update together after the warp reconverges (a lane
    // without a pair on zero velocities, its result not stored), since
    // GB300's FP64 pipe costs a warp instruction however few lanes are active
    __syncwarp();
    vhs_pair(a.seed, a.step, (uint32_t)q.w, (uint32_t)q.z, v);
    if (live) {
      __stcg(a.vx + q.x, v[0]); __stcg(a.vy + q.x, v[1]); __stcg(a.vz + q.x, v[2]);
      __stcg(a.vx + q.y, v[3]); __stcg(a.vy + q.y, v[4]); __stcg(a.vz + q.y, v[5]);
      release_pair(a.done, q.x, q.y, (unsigned)(rc + 1));
    }
    if (!__all_sync(0xffffffffu, ok)) break;
    have = next; p0 = n0; p1 = n1; rc = rn; q = qn; dep = depn;
  }
}


// resident blocks per SM of the VHS collide at a block size (0 on failure)
int occupancy_collide_vhs(int threads) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (const void*)k_collide_vhs, threads, 0) != cudaSuccess)
    return 0;
  return per_sm;
}

// The done stamps and the barrier words (abort, unit cursor) of a collide call
// start at zero: one launch for both.
__global__ void k_clear_stamps(unsigned* __restrict__ done, int32_t n, unsigned* bar) {
  dep_wait();
  if (blockIdx.x == 0 && threadIdx.x < 4) bar[threadIdx.x] = 0u;
  const int64_t first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
  // 16 bytes at a time from an aligned workspace, word by word otherwise and at the end
  const int64_t n4 = ((uintptr_t)done & 15u) ? 0 : n / 4;
  for (int64_t q = first; q < n4; q += stride) ((uint4*)done)[q] = make_uint4(0u, 0u, 0u, 0u);
  for (int64_t q = 4 * n4 + first; q < n; q += stride) done[q] = 0u;
}

int launch_clear_stamps(Ctx* c, unsigned* done, int32_t n, unsigned* bar, cudaStream_t s) {
  int64_t b = ((int64_t)n + 4095) / 4096;
  if (b < 1) b = 1;
  if (b > 8 * sm_count(c)) b = 8 * sm_count(c);
  launch_dep(k_clear_stamps, (unsigned)b, 256, 0, s, done, n, bar);
  count_launches(c, 1);
  return cudaGetLastError() == cudaSuccess ? 0 : DSMC_ERR_CUDA;
}

size_t collide_ws(int32_t n) { return align256(sizeof(unsigned) * (size_t)(n > 0 ? n : 1)); }

int launch_collide_vhs(Ctx* c, const dsmc_gas_t& gas, uint64_t step, int32_t n, const int32_t* pairs,
                       const uint32_t* deps, const int32_t* ro, const dsmc_select_info_t* info, double* vx,
                       double* vy, double* vz, void* ws, size_t ws_bytes, cudaStream_t s) {
  if (ws_bytes < collide_ws(n)) return record(c, DSMC_ERR_ARG, "collide_vhs: workspace too small");
  const Shape sh = shape_or_default(c, DSMC_TUNE_COLLIDE_VHS);
  const int occ = occupancy_collide_vhs(sh.threads);
  if (occ < 1) return record(c, DSMC_ERR_CUDA, "collide_vhs: occupancy query failed");
  const int blocks = sm_count(c) * (sh.blocks_per_sm > 0 && sh.blocks_per_sm < occ ? sh.blocks_per_sm : occ);
  VhsArgs a{gas.seed, step, graph_step_ptr(c), (const int4*)pairs, deps, ro, info, vx, vy, vz,
            (unsigned*)ws, barrier_ptr(c), status_ptr(c)};
  if (int rc = launch_clear_stamps(c, a.done, n, a.bar, s)) return rc;
  launch_dep(k_collide_vhs, blocks, sh.threads, 0, s, a);
  count_launches(c, 1);
  return cudaGetLastError() == cudaSuccess ? 0 : record(c, DSMC_ERR_CUDA, "collide_vhs: launch failed");
}

// ---------------------------------------------------------------- pair updates of the step
// In a step the pair list is the selection's own: inside a round the pairs are
// in cell order, and a cell's pairs touch that cell's particles only.  So a warp
// can take a group of consecutive cells through all rounds by itself, 32 pairs at a
// time, with a __syncwarp between rounds where the collide calls (which take
// any list) wait on done stamps, release fences and a claim per 32 pairs.  Lane r
// finds the group's pairs of round r by two binary searches on the cell index.
// A group has about kGroupPairs pairs (fewer cells than that to a group leave a
// round's lanes empty, and the FP64 pipe costs a warp instruction however few
// lanes are active; more make the chain of one warp long), at most kGroupCells cells,
// and there are a thousand groups if there are as many cells.  Step of 2,867 cells
// and 47,580 pairs on the look-up path 152 -> 120 us.  Blocks of one warp, so that few
// groups spread evenly over the SMs' four sub-partitions, each with an FP64 pipe of its
// own: 105 us where blocks of four took 110 (of two: 106).  Larger gases fill the
// chip without this, and the groups' partly filled warps and searches cost more than
// the waits they save, as does the one warp that takes a dense cell's pairs: see groups_suit.
struct GroupArgs {
  uint64_t seed, step;
  const uint64_t* step_dev;
  const int4* pairs;
  const int32_t* ro;
  const dsmc_select_info_t* info;
  double *vx, *vy, *vz;
  unsigned* work;   // groups claimed, finished blocks (zero between launches)
  int32_t n_cells;
};

struct VhsUpdate {
  __device__ __forceinline__ void operator()(const GroupArgs& a, int4 q, double* v) const {
    vhs_pair(a.seed, a.step, (uint32_t)q.w, (uint32_t)q.z, v);
  }
};
struct TableUpdate {
  TableLook look;
  __device__ __forceinline__ void operator()(const GroupArgs& a, int4 q, double* v) const {
    table_pair(look, a.seed, a.step, (uint32_t)q.w, (uint32_t)q.z, v);
  }
};

constexpr int kGroupThreads = 32;   // a warp: see above
constexpr int kGroupBlocks = 32;    // per SM
constexpr int kGroupPairs = 128, kGroupCells = 8;

template <class Update>
__global__ void __launch_bounds__(kGroupThreads, kGroupBlocks) k_collide_groups(GroupArgs a, Update update) {
  dep_wait();
  if (a.step_dev) a.step = *a.step_dev;
  const int R = a.info->n_rounds;
  const int64_t pairs = a.info->n_pairs;
  // cells per group
  const int cells = (int)min((int64_t)(a.n_cells / 1024 + 1),
                             max((int64_t)1, pairs > 0 ? min((int64_t)kGroupCells, kGroupPairs * (int64_t)a.n_cells / pairs)
                                                       : (int64_t)kGroupCells));
  const int lane = threadIdx.x & 31;
  // every warp's first group is its own index; further ones, if there are more groups
  // than warps, are claimed (dense cells lie together: 37,500 cells of the
  // hypersonic gas 577 us, by stride 685; claims from one counter by warps that have
  // only one group to take cost 20 us)
  const unsigned warps = gridDim.x * (kGroupThreads / 32);
  const bool claims = (int64_t)warps * cells < a.n_cells;
  unsigned g = blockIdx.x * (kGroupThreads / 32) + (threadIdx.x >> 5);
  for (int64_t first; (first = (int64_t)g * cells) < a.n_cells;) {
    const int32_t k0 = (int32_t)first, k1 = (int32_t)min((int64_t)a.n_cells, first + cells);
    for (int rb = 0; rb < R; rb += 32) {
      // the pairs of cells [k0, k1) in round rb + lane: [lo, hi)
      int32_t lo = 0, hi = 0;
      if (rb + lane < R) {
        int32_t l0 = a.ro[rb + lane], l1 = a.ro[rb + lane + 1], h0 = l0, h1 = l1;
        while (l0 < l1 || h0 < h1) {
          const int32_t ml = (l0 + l1) >> 1, mh = (h0 + h1) >> 1;
          const int32_t zl = l0 < l1 ? a.pairs[ml].z : k0, zh = h0 < h1 ? a.pairs[mh].z : k1;
          if (l0 < l1) { if (zl < k0) l0 = ml + 1; else l1 = ml; }
          if (h0 < h1) { if (zh < k1) h0 = mh + 1; else h1 = mh; }
        }
        lo = l0; hi = h0;
      }
      __syncwarp();
      const int nr = min(32, R - rb);
      int r = -1;
      int32_t p0 = 0, end = 0;
      auto next = [&]() {
        p0 += 32;
        while (p0 >= end) {
          if (++r >= nr) return false;
          p0 = __shfl_sync(0xffffffffu, lo, r);
          end = __shfl_sync(0xffffffffu, hi, r);
        }
        return true;
      };
      bool have = next();
      int4 qn = make_int4(0, 0, 0, 0);
      bool actn = have && p0 + lane < end;
      if (actn) qn = a.pairs[p0 + lane];
      while (have) {
        const int4 q = qn;
        const bool act = actn;
        // the next pairs' records load while these update
        have = next();
        actn = have && p0 + lane < end;
        if (actn) qn = a.pairs[p0 + lane];
        double v[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        if (act) {
          v[0] = a.vx[q.x]; v[1] = a.vy[q.x]; v[2] = a.vz[q.x];
          v[3] = a.vx[q.y]; v[4] = a.vy[q.y]; v[5] = a.vz[q.y];
        }
        update(a, q, v);
        if (act) {
          a.vx[q.x] = v[0]; a.vy[q.x] = v[1]; a.vz[q.x] = v[2];
          a.vx[q.y] = v[3]; a.vy[q.y] = v[4]; a.vz[q.y] = v[5];
        }
        __syncwarp();   // the next round's loads see these stores
      }
    }
    if (!claims) break;
    if (lane == 0) g = warps + atomicAdd(a.work, 1u);
    g = __shfl_sync(0xffffffffu, g, 0);
  }
  // the last block to finish leaves the counters zero for the next launch
  if (claims) {
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      if (atomicAdd(a.work + 1, 1u) == gridDim.x - 1) {
        __threadfence();
        a.work[0] = 0u;
        a.work[1] = 0u;
      }
    }
  }
}

template <class Update>
static int launch_groups(Ctx* c, const Update& u, const dsmc_gas_t& gas, uint64_t step, int32_t n_cells,
                         const int32_t* pairs, const int32_t* ro, const dsmc_select_info_t* info, double* vx,
                         double* vy, double* vz, cudaStream_t s) {
  GroupArgs a{gas.seed, step, graph_step_ptr(c), (const int4*)pairs, ro, info, vx, vy, vz, work_ptr(c), n_cells};
  const int warps = kGroupThreads / 32;
  const int64_t want = ((int64_t)n_cells + warps - 1) / warps, most = (int64_t)sm_count(c) * kGroupBlocks;
  launch_dep(k_collide_groups<Update>, (unsigned)(want < most ? want : most), kGroupThreads, 0, s, a, u);
  count_launches(c, 1);
  return cudaGetLastError() == cudaSuccess ? 0 : record(c, DSMC_ERR_CUDA, "step: pair update launch failed");
}

int launch_groups_vhs(Ctx* c, const dsmc_gas_t& gas, uint64_t step, int32_t n_cells, const int32_t* pairs,
                    const int32_t* ro, const dsmc_select_info_t* info, double* vx, double* vy, double* vz,
                    cudaStream_t s) {
  return launch_groups(c, VhsUpdate{}, gas, step, n_cells, pairs, ro, info, vx, vy, vz, s);
}
int launch_groups_table(Ctx* c, const dsmc_gas_t& gas, const dsmc_chi_table_t& tab, uint64_t step, int32_t n_cells,
                      const int32_t* pairs, const int32_t* ro, const dsmc_select_info_t* info, double* vx, double* vy,
                      double* vz, cudaStream_t s) {
  return launch_groups(c, TableUpdate{table_look(gas, tab)}, gas, step, n_cells, pairs, ro, info, vx, vy, vz, s);
}

// Failure-detection self test: every block but block 0 enters the grid
// barrier; block 0 never arrives, so the others' bounded waits run out and
// record DSMC_ERR_TIMEOUT.  No trap, no unbounded spin.
__global__ void k_selftest_barrier(unsigned* bar, int* status, uint64_t limit_ns) {
  if (blockIdx.x == 0) return;
  grid_barrier(bar, status, limit_ns);
}

// Failure-detection self test of the pair-dependency wait: one thread waits
// for a done stamp that nothing ever sets (word 0 of the zeroed barrier
// words); the bounded wait must record DSMC_ERR_TIMEOUT and return.
__global__ void k_selftest_deps(unsigned* bar, int* status, uint64_t limit_ns) {
  if (threadIdx.x == 0) wait_deps(bar, 0, 0, 1u, bar + 2, status, limit_ns);
}

int launch_selftest_deps(Ctx* c, uint64_t limit_ns, cudaStream_t s) {
  unsigned* bar = barrier_ptr(c);
  if (cudaMemsetAsync(bar, 0, 4 * sizeof(unsigned), s) != cudaSuccess) return DSMC_ERR_CUDA;
  k_selftest_deps<<<1, 32, 0, s>>>(bar, status_ptr(c), limit_ns);
  count_launches(c, 1);
  return cudaGetLastError() == cudaSuccess ? 0 : record(c, DSMC_ERR_CUDA, "selftest_deps: launch failed");
}

int launch_selftest_barrier(Ctx* c, uint64_t limit_ns, cudaStream_t s) {
  if (cudaMemsetAsync(barrier_ptr(c), 0, 4 * sizeof(unsigned), s) != cudaSuccess) return DSMC_ERR_CUDA;
  unsigned* bar = barrier_ptr(c);
  int* st = status_ptr(c);
  void* args[] = {&bar, &st, &limit_ns};
  if (cudaLaunchCooperativeKernel((const void*)k_selftest_barrier, dim3(4), dim3(32), args, 0, s) != cudaSuccess)
    return record(c, DSMC_ERR_CUDA, "selftest_barrier: launch failed");
  count_launches(c, 1);
  return 0;
}

}  // namespace dsmc
