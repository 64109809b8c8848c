// hd_analysis.h -- launchers of the positional-order analysis (Sec. IV.C,
// Eqs. 10-12): the structure factor S[R][nq] at box-periodic wave vectors
// hk[R][nq] (best[R] = index of the largest), the q_0 candidate window around
// the first reciprocal shell, chi_j = exp(i q_0 . x_j), and the positional
// correlation C[R][nr] at r_k = (k + 1) dr.
#pragma once

#include <vector>

#include "hd_kernels.h"

namespace hd {

int sq_disk_blocks(const std::vector<int64_t>& N);
cudaError_t launch_sq(const LaunchCfg& c, int nq, const int2* hk, const double* xy, int nbx, double2* part, double* S,
                      int* best);
// The same for wave vectors given by components: comp[R][nh + nk] the distinct
// h, then k, of each replica, pair[R][nq] the indices of every wave vector's
// (sq_pairs_fit: whether that is the cheaper way); grid: the components of
// every replica are nh and nk consecutive integers and sq_grid_fit.  part: R x
// nbx x max(nq, nh nk) with nbx = sq_pair_blocks.  best is nullable in both.
bool sq_pairs_fit(int nh, int nk, int nq);
bool sq_grid_fit(int nh, int nk, int nq);
int sq_pair_blocks(int R, int nq, const std::vector<int64_t>& N);
cudaError_t launch_sq_pairs(const LaunchCfg& c, int nq, int nh, int nk, bool grid, const int* comp, const ushort2* pair,
                            const double* xy, int nbx, double2* part, double* S, int* best);
// The window's wave vectors into hk[R][nq], and its components and pairs.
cudaError_t launch_q0_window(const LaunchCfg& c, int hw, const double* psi, int2* hk, int* comp, ushort2* pair);
cudaError_t launch_chi(const LaunchCfg& c, int64_t Ntot, const int2* hk0, const double* xy, double2* chi);
cudaError_t launch_poscorr(const LaunchCfg& c, CellBufs cells, const double* xy, const double2* chi, int nr, double dr,
                           int reach, double* acc, double2* out);

// The same from unordered pairs, for the windows whose sums fit shared memory
// (corr_pairs_fit) and a reach that holds the largest window with a cell to
// spare.  most_cells: of one
// replica; gpos, chi, off: one entry per slot of the cell arrays; acc:
// corr_pairs_acc doubles.
bool corr_pairs_fit(int nr);
size_t corr_pairs_acc(int R, int nr);
cudaError_t launch_corr_pairs(const LaunchCfg& c, int64_t most_cells, const Frame* cur, CellBufs cells, const int2* hk0,
                              double2* gpos, double2* chi, float2* off, int nr, double dr, int reach, double* acc,
                              double2* out);

}  // namespace hd
