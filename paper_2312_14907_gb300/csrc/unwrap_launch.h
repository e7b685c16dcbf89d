// unwrap_launch.h -- the phase unwrapper and the projector Pi_U (mpbp_unwrap.cu).
#pragma once
#include "mpbp_internal.h"

namespace mpbp {

// D maps of n1 x n2 pixels (nodes = D * npix)
struct UnwrapArgs {
  const float* wrapped;   // [nodes] wrapped phases in [-pi, pi)
  const float* mask;      // [npix] nonzero = inside, or nullptr
  float* out;             // [nodes] unwrapped phases
  float* rel;             // [nodes] pixel reliabilities
  int* parent;            // forest, double-buffered
  int* off;               //   multiple of 2 pi relative to the parent
  int* parent2;
  int* off2;
  int* hook_parent;       // [nodes] the current Boruvka round's hooks of the roots
  int* hook_off;
  int* minnode;           // [nodes] lowest node of each group (at its root)
  unsigned long long* best;   // [nodes] heaviest incident edge of each root
  unsigned long long* ekey;   // [2 nodes] key of edge e = 2 v + dir (0: no edge)
  int* flags;             // [3] rotating "something changed" flags, zeroed before launch
  unsigned* bar_count;    // grid barrier, zeroed before launch
  unsigned* bar_gen;
  int* lists;             // [2 D] components and edges listed per map, zero between calls
  int* map_flags;         // [3 D] the map kernel's "something changed" flags
  int* comps;             // [6 D comp_cap] the map kernel's components
  int2* edge_ends;        // [D spill_cap] labels of the listed edges past its registers
  long long comp_cap, spill_cap;   // per map (unwrap_comp_cap, unwrap_spill_cap)
  int* err;               // kErrTimeout if a barrier wait runs out
  long long npix, nodes;
  int n1, n2;
  int max_rounds;
  int max_blocks;         // largest cluster the map kernel may use (unwrap_map_blocks)
  int test_stall;         // != 0: block 0 never arrives at a grid barrier (test
                          // of the bounded waits; the result is meaningless)
};

struct ProjectArgs {
  float* u;               // [C][npix], corrected in place
  const float* mask;      // [npix] or nullptr
  float* phi;             // [D][npix] phase_scale G_m . u
  float* wrapped;         // [D][npix] W(phi)
  const float* unwrapped; // [D][npix]
  float g_scaled[kMaxPeaks * kMaxComp];      // phase_scale G[m][c]
  float pinv_scaled[kMaxComp * kMaxPeaks];   // pinv(G)[c][m] / phase_scale
  long long npix;
  int C, D;
};

bool unwrap_prepare(int num_sms, int* grid);
int unwrap_map_blocks();
// The cooperative path, on the given grid; flags and barrier zeroed before.
cudaError_t unwrap_launch(const UnwrapArgs& a, int grid, cudaStream_t s);
// Whether the path by tiles and maps serves these maps (its lists hold every
// map of such a size); its two kernels; and the one that writes out
// (project_correct does without).
bool unwrap_by_tiles(const UnwrapArgs& a);
long long unwrap_comp_cap(int n1, int n2);
long long unwrap_spill_cap(int n1, int n2);
cudaError_t unwrap_tiles_launch(const UnwrapArgs& a, cudaStream_t s);
cudaError_t unwrap_close_launch(const UnwrapArgs& a, int num_sms, cudaStream_t s);
cudaError_t project_phase_launch(const ProjectArgs& a, int num_sms, cudaStream_t s);
// tiles: the unwrapped phases from uw's offsets (unwrap_tiles_launch without
// unwrap_close_launch), else from a.unwrapped
cudaError_t project_correct_launch(const ProjectArgs& a, const UnwrapArgs& uw, bool tiles, int num_sms,
                                   cudaStream_t s);

}  // namespace mpbp
