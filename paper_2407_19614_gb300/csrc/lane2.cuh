// Two-centre and one-electron integrals with one lane, or a few, per shell pair
// (spherical bases): eri2_lane.cu, one_lane.cu.
#pragma once
#include "eri3_lane.cuh"

namespace rihf {

// Shell pairs by class on the device; chunks of at most one warp's tasks.
struct Lane2Tasks {
  const int2* tasks = nullptr;
  const LaneChunk* chunks = nullptr;
  long long nchunk = 0;
};

// (P|Q): auxiliary shell pairs, the lower l first; cls = la | lc << 8.
void build_lane2_tasks(const std::vector<int>& l, const std::vector<int>& atom, std::vector<int2>& tasks,
                       std::vector<LaneChunk>& chunks);
// A[P][Q] = (P|Q), both triangles.
void launch_lane_eri2(const IntegralCtx& ic, const DevShells& aux, const Lane2Tasks& t, const KetTable* ket, double* A);
// grad[atom] += -1/2 sum_PQ Z_PQ d(P|Q).
void launch_lane_grad_eri2(const IntegralCtx& ic, const DevShells& aux, const Lane2Tasks& t, const KetTable* ket,
                           const double* Z, double* grad);

// One-electron: primary shell pairs (a, b), la >= lb, in chunks of at most kOneChunk;
// cls = la | lb << 4.  A launch gives every pair 4 to 32 lanes, which share out the nuclei.
constexpr int kOneChunk = 8;
void build_one_tasks(const std::vector<int>& l, std::vector<int2>& tasks, std::vector<LaneChunk>& chunks);
// The lanes of a pair when `share` contexts launch at the same time.
int one_lanes(int nshell, int natoms, int sms, int share);
// S and h = T + V, both triangles.
void launch_lane_one(const IntegralCtx& ic, const DevShells& prim, const Lane2Tasks& t, int lanes, int natoms, const int* Z,
                     const double* axyz, double* S, double* H);
// grad_one += sum D d(T + V), grad_ovl += -sum W dS.
void launch_lane_grad_one(const IntegralCtx& ic, const DevShells& prim, const Lane2Tasks& t, int lanes, int natoms,
                          const int* Z, const double* axyz, const double* D, const double* W, double* grad_one, double* grad_ovl);

}  // namespace rihf
