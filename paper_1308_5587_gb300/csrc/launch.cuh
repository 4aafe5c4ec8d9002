// launch.cuh -- host-side launchers of the libgbmd kernels (one per kernel family).
// Every launcher enqueues on `st` and returns the launch status; none allocates.
// Grids are tile counts: each block handles one Tile of its table.
#pragma once
#include "gbmd_internal.cuh"

namespace gbmd {

constexpr int TILE_P = 256;     // particles per block of the streaming kernels
// particles per FP64 energy/virial partial sum (a block of the energy launches), by the
// system's size, so the sums depend on the lanes per particle (a warp's 32 / TPP particles
// are summed first; wide tiles hold TPP / 32 as many) but not on the force block.  Up to EV_SMALL_N particles a
// block of 128 leaves SMs idle or unevenly loaded (FP64, N = 4,000: 32 blocks of 512
// threads, 120 us; the whole readout 177 us with them, 68 with tiles of 32)
constexpr int EV_TILE_P = 128, EV_TILE_SMALL = 32, EV_SMALL_N = 131072;
inline int ev_tile(int n) { return n <= EV_SMALL_N ? EV_TILE_SMALL : EV_TILE_P; }
constexpr int CELLS_PER_TILE = 8;   // warps (= cells) per block of the cell kernels
constexpr int SCAN_THREADS = 1024;

// kernel-node description for graph building: function + grid + argument values.
// Copyable: the pointer array that cudaLaunchKernel / kernel nodes want is built
// from `store` at the point of use (args_of), never kept inside the object.
struct KernelCall {
  void* func;
  dim3 grid, block;
  size_t smem;
  bool cooperative;
  int nargs;
  alignas(16) unsigned char store[10][16];
};

inline void args_of(const KernelCall& k, void** a) {
  for (int i = 0; i < k.nargs; ++i) a[i] = const_cast<unsigned char*>(k.store[i]);
}

// cell list + sort + neighbour list (each a no-op for systems not rebuilding); the
// sort bins are cells, or (type, cell) pairs for systems on the tree list
KernelCall bin_call(const SysDev* d, const Tile* tiles_p, int ntiles, GroupCtl* ctl);
KernelCall scan_call(const SysDev* d, const Tile* tiles_s, int nsys, GroupCtl* ctl);
KernelCall scatter_call(const SysDev* d, const Tile* tiles_p, int ntiles, GroupCtl* ctl);
KernelCall cellsort_call(const SysDev* d, const Tile* tiles_c, int ntiles, GroupCtl* ctl);
KernelCall permute_call(const SysDev* d, const Tile* tiles_p, int ntiles, GroupCtl* ctl);
KernelCall copyback_call(const SysDev* d, const Tile* tiles_p, int ntiles, GroupCtl* ctl);
// window table of every staged 2x2x2 block (8 blocks per kernel block of 256)
KernelCall blocks_call(const SysDev* d, const Tile* tiles_b, int ntiles, GroupCtl* ctl);
KernelCall nlist_call(const SysDev* d, const Tile* tiles_c, int ntiles, GroupCtl* ctl, bool rel,
                      bool multi, bool staged);
// all of the above for the single system d[0], tree lists included, by the grid of a
// cooperative launch (no staged window); returns at once when the step asked for no rebuild
void* rebuild_func(bool multi);
KernelCall rebuild_call(const SysDev* d, int blocks, GroupCtl* ctl, bool multi);
// the same rows built by four warps per cell (tiles over (cell, part) items)
KernelCall nlist_split_call(const SysDev* d, const Tile* tiles_n, int ntiles, GroupCtl* ctl, bool multi);
// tree neighbour list (k_tree.cu): the boxes of every type's tree (one thread per
// leaf; tiles over the system's leaves), then the list (one warp per group of particles;
// tiles over groups)
constexpr int TREE_WARPS = 8;   // groups a block
constexpr int TREE_G = 8;       // particles of a group: TREE_G x 4 lanes
KernelCall tree_build_call(const SysDev* d, const Tile* tiles_l, int ntiles, GroupCtl* ctl);
KernelCall tree_nlist_call(const SysDev* d, const Tile* tiles_g, int ntiles, GroupCtl* ctl);
// pair force kernels.  MODE_FORCE: forces at the current positions; MODE_READ: also a
// readout's rows (sa.readout); MODE_EV: also energy / virial / v.v partial sums (+
// per-particle arrays when the descriptor has them); MODE_STEP: the step kernel -- forces, the velocity Verlet
// update of every particle into the next shadow buffer, and the end-of-step
// decisions by the last of sa.total_blocks blocks over the step's force launches.
// MODE_NVT_A: the first half of an NVT step -- forces, the closing half kick and
// thermostat scaling of the previous step, v.v partial sums; a system's last block
// updates its thermostat.  nvt_b_call: the second half (opening scaling and kick, drift,
// shadow, rebuild check, end-of-step decisions).
enum { MODE_FORCE = 0, MODE_EV = 1, MODE_STEP = 2, MODE_NVT_A = 3, MODE_READ = 4 };
// which step configurations take wide tiles, a warp a particle (all modes of one do, so
// that a readout's forces are the step's): not the register-capped step kernel of one
// lane a particle
__host__ __device__ constexpr bool has_wide(int prec, int tpp) { return prec == GBMD_FP64 || tpp > 1; }
enum { READ_FORCE = 1, READ_VEL = 2, READ_POS = 4, READ_IMAGE = 8 };   // rows of a readout
struct StepArgs {
  int nsys = 0;             // systems of the group (decisions of the last block)
  int total_blocks = 0;     // blocks of all the step's force launches
  cudaGraphConditionalHandle cond = 0;   // the rebuild conditional of the step graph
  int use_cond = 0;
  int readout = 0;          // MODE_READ: the READ_ bits of what to write out
};
// eval: the PairEval of every system of the launch
KernelCall force_call(int prec, int multi, int mode, int tpp, int block, const SysDev* d,
                      const Tile* tiles_f, int ntiles, GroupCtl* ctl, const StepArgs& sa,
                      int eval);
// staged pair force: one kernel block per 2x2x2 cell block, window in shared memory
// (mixed precision, LJ evaluator); part_base = first partial-sum slot of these tiles
KernelCall force_staged_call(int multi, int mode, const SysDev* d, const Tile* tiles_s, int ntiles,
                             GroupCtl* ctl, int part_base, int window_cap, const StepArgs& sa);
KernelCall nvt_b_call(int prec, const SysDev* d, const Tile* tiles_p, int ntiles, GroupCtl* ctl,
                      const StepArgs& sa);
constexpr int STAGED_BLOCK = 256;
// thermo reduction (K7), one block per system
KernelCall thermo_call(const SysDev* d, const Tile* tiles_s, int nsys, GroupCtl* ctl);
// import row-major tag-order staging -> internal arrays; export the reverse
KernelCall prep_state_call(const SysDev* d, const Tile* tiles_p, int ntiles, const double* pos,
                           const double* vel, int* type_by_tag, int* bad);
KernelCall import_call(const SysDev* d, const Tile* tiles_p, int ntiles, const double* pos,
                       const double* vel, const int* type, const int* image, const int* bad);
// the flags of a state being loaded into system *d, and the Snapshot of *d; with `bad`
// (may be null) set the load changes nothing
KernelCall load_flags_call(const SysDev* d, const int* bad, long long step, long long limit);
KernelCall snapshot_call(const SysDev* d);
KernelCall export_call(const SysDev* d, const Tile* tiles_p, int ntiles, double* pos,
                       double* vel, int* image, double* force, double* pp_u, double* pp_w);
// domain decomposition (one system, d pointing at its descriptor): ghost positions
// (row-major, real units) into the current step's state; wrapped positions of listed
// tags out
KernelCall ghost_set_call(const SysDev* d, int n_ghost, const double* pos);
KernelCall gather_pos_call(const SysDev* d, const int* tags, int m, double* out);
// neighbour rows -> tag-order rows sorted ascending (test readout)
KernelCall nlist_export_call(const SysDev* d, const Tile* tiles_p, int ntiles, int* counts,
                             int* idx, int cap_out, int* too_many);

cudaError_t launch(const KernelCall& k, cudaStream_t st);

// the team kernel (k_team.cuh): many steps of one or more systems in one launch
// one block an SM, 128 registers a thread, and the warps a small system fills (spilled, by
// -Xptxas -v: 40 to 110 bytes in the mixed LJ instances, 200 to 220 in the FP64 ones);
// the rest of the SM's 256 KB stays L1 for the force phase's gathers
constexpr int TEAM_T = 512;
constexpr size_t TEAM_SMEM = 112 * 1024;
// the rebuild alone: more warps, 80 registers each
constexpr int REBUILD_T = 768;
constexpr size_t REBUILD_SMEM = 220 * 1024;
constexpr int TEAM_MAX_CLUSTER = 16;
struct TeamArgs {
  const SysDev* desc;
  const int* list;   // the systems of the launch (positions in desc), the largest first
  GroupCtl* ctl;
  int nsteps;
  int cluster;       // blocks of a team; 0: the grid is one team, or several by `share`
  // per block of the grid, or null: (position in list, rank in its team, the team's
  // blocks, its barrier in sync)
  const int4* share;
  TeamSync* sync;
};
// two_in_one: mixed with two lanes a particle, one lane doing the work of both
void* k_team_variant(int eval, int prec, int tpp, int mt, bool two_in_one);

// arithmetic throughput probe (k_probe.cu): one timed launch over every SM
cudaError_t probe_run(int kind, cudaStream_t st, int iters, double* ops, float* ms);

// force-kernel variants available (threads per particle)
bool tpp_supported(int tpp);

}  // namespace gbmd
