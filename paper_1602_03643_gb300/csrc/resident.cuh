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
// memory: three components to about 440,000 rows mixed; float64 one component to
// 500,000, the mass solve of three to 240,000), and the d components of a float64
// velocity solve together.  Resident against separate kernels, us per step, the named
// solves alone changed.  Mixed: velocity 439,000 rows 5859 / 5920 (triangles 386,000: 1562
// / 1796); one component at a time 636,000: 3520 / 5017; with two scalars 636,000: 4367 /
// 4885; with the mass solve 493,000: 3365 / 3757; Jacobi pressure 636,000: 10009 / 12343.
// Float64: velocity 132,700 rows 3683 / 3802, 148,900: 3905 / 3947, 185,200: 4736 / 4760,
// 205,400: 5074 / 4913; triangles 90,600: 1513 / 1599, 160,800: 2287 / 2264; one component
// at a time 357,900: 8427 / 9881; two scalars 357,900: 10116 / 10557; mass 205,400: 6840 /
// 7217; Jacobi pressure 68,900: 4856 / 9233.
constexpr int64_t kResidentRows = 650000, kResidentRows64 = 150000;

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
