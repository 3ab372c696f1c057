// Resident solves: a whole linear solve (refinement sweeps, Krylov iterations and
// multigrid cycles) as one cooperative launch, for systems small enough that the
// blocks' shared memory holds the matrix and the vectors (resident.cu).
#pragma once

#include "amg.cuh"
#include "solver.cuh"

namespace oasis {

constexpr int kResValues = 16;           // values of one grid-wide sum at most
constexpr int kResBlocks = 1024;         // blocks of one launch at most
// Rows up to which a solve may run resident (where a block's vectors fit its shared
// memory: with three components about 440,000 rows mixed, 200,000 float64).  Resident
// against separate kernels, us per step: 14x13x12 dofs float64 Jacobi eager 1160 / 4130;
// 41^3 Jacobi mixed 1810 / 5690; 85^3 Jacobi mixed 16460 / 23330; velocity solve alone
// changed: 73^3 mixed 2890 / 3140, 621^2 mixed 2070 / 2320.
constexpr int64_t kResidentRows = 650000;

// Device memory in which the blocks of a launch meet (zero between launches).
struct ResidentSync {
    uint32_t *count, *ticket;            // arrivals; blocks that have left
    void* partial;                       // [2][kResValues][blocks] 8-byte sums
    void* pub;                           // three vectors of n dofs that neighbours gather
};
size_t resident_sync_bytes(int64_t n, size_t value_bytes);
ResidentSync resident_sync(void* mem);
// Limit of the waits of launches that meet there, in SM clock cycles (0: the usual one).
void resident_set_wait(void* mem, int64_t cycles, cudaStream_t s);

// Plans for the solve of NR of D components, the mass solve of D and the pressure solve
// on a pattern (host row pointers), for the current device; blocks = 0 where a block's
// share does not fit, or where the device does not take the launch (no cooperative
// launches, or fewer blocks resident than the plan needs).
template <class P, int D, int NR>
ResidentPlan resident_plan_bicg(const std::vector<int32_t>& row_ptr, int64_t n);
template <class P, int D>
ResidentPlan resident_plan_mass(const std::vector<int32_t>& row_ptr, int64_t n);
template <class P>
ResidentPlan resident_plan_cg(const std::vector<int32_t>& row_ptr, int64_t n, bool amg);
// Likewise for the tail of a V-cycle whose finest level has n rows.  The tail runs inside
// conditional graph bodies, where cooperative launches are allowed without MPS only.
template <class V>
ResidentPlan resident_plan_tail(int64_t n);

// One operator level of the multigrid cycle as a resident solve reads it.
template <class V>
struct ResidentLevel {
    using AV = typename std::conditional<sizeof(V) == 8, double, uint16_t>::type;
    int32_t n;
    V w;
    const V* d;
    const int32_t *a_rp, *a_ci, *s_rp, *s_ci, *t_rp, *t_ci;
    const AV *a, *s, *t;                 // the level's matrix, S and S^T (level 0: a is null, its matrix is K)
    V *r, *y, *x;                        // the level's input, smoothed part and result
    int32_t ga, gs, gt;                  // lanes per row of a, s and t
};
constexpr int kResLevels = 12;
template <class V>
struct ResidentAmg {
    int32_t levels = 0, nc = 0, ld = 0;
    const V* inv = nullptr;
    V *rc = nullptr, *xc = nullptr;      // input and result of the dense coarsest level
    ResidentLevel<V> lv[kResLevels];
};

// The hierarchy from level `first` on, and a solver's cycle vectors, for a launch of
// the given shape.
template <class V>
ResidentAmg<V> resident_amg(const AmgHierarchy& h, AmgWork& w, int first, int blocks, int threads);

// D components per dof, NR of them (from k0) solved together.
template <class P, int D, int NR>
void resident_bicg(const StepData<P>& q, int k0, const Ctl& c, const ResidentPlan& pl, const ResidentSync& sy,
                   cudaStream_t s);
// Pressure CG; m.levels = 0: Jacobi.
template <class P>
void resident_cg(const StepData<P>& q, const Ctl& c, const ResidentAmg<typename P::V>& m, const ResidentPlan& pl,
                 const ResidentSync& sy, cudaStream_t s);

// Consistent-mass update: the increment into q.mx.
template <class P, int D>
void resident_mass(const StepData<P>& q, double dt, const Ctl& c, const ResidentPlan& pl, const ResidentSync& sy,
                   cudaStream_t s);

}  // namespace oasis
