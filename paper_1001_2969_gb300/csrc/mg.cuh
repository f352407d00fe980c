// mg.cuh -- workspace and control block of the multigrid solve in mg.cu.
#pragma once

#include <vector>

#include "pic_internal.cuh"

namespace pic {

// device-side control of one solve (the one-launch V-cycles)
struct MGCtl {
    int converged, zero_rhs, cycles, timeout;
    int skip, pad;  // the step had halted when the solve was set up: its blocks do nothing
    double last_res, bnorm;
};

// a timestep's solve reports to the step control instead of the host: V-cycle
// count, residual, an unconverged flag, and a halt on a timed-out wait (one
// thread calls it).  `cont`: a second solve with the previous one's operator
// (the external circuit's charge-free part) adds its cycles to the step's last
// report and keeps the larger residual
__device__ __forceinline__ void solve_report(const MGCtl *c, StepCtl *s, int cont) {
    if (s->halt) return;
    if (c->timeout) {
        s->halt = 1;
        s->halt_status = ST_TIMEOUT;
        s->halt_step = s->step;
        return;
    }
    const int cyc = c->zero_rhs ? 0 : c->cycles;
    s->mg_cycles += (unsigned long long)cyc;
    const double res = (c->zero_rhs || !(c->bnorm > 0.0)) ? 0.0 : c->last_res / c->bnorm;
    if (cont) {
        s->mg_last_cycles += cyc;
        s->mg_last_res = fmax(s->mg_last_res, res);
    } else {
        s->mg_last_cycles = cyc;
        s->mg_last_res = res;
    }
    if (!c->zero_rhs && !c->converged) s->mg_flags |= 1;
}

// returned by mg_fast_solve when a bounded device wait gave up, and when
// the one-launch solve cannot be launched (shared memory, co-residency)
constexpr int kSolveTimeout = -1000000;
constexpr int kSolveNoLaunch = -1000001;

constexpr int kMaxLevels = 16;

struct MGFast;
struct MGFast {
    int nlev;
    int nz[kMaxLevels];
    double dz[kMaxLevels];
    double *chi[kMaxLevels];
    // face coefficients: in z per level (mixed path: FP64 on the fine level
    // alone, FP32 on all), in r of the fine level (the line factors hold the rest)
    double *cz[kMaxLevels], *cr;
    float *cz32[kMaxLevels];
    // face geometry per level, by column j (filled once by mg_fast_geometry):
    // gz = pi (r_{j+1/2}^2 - r_{j-1/2}^2) / dz_l, gr = 2 pi r_{j+1/2} dz_l / dr;
    // ga = pi (r_{j+1/2}^2 - r_{j-1/2}^2) dz / eps0 (level 0's right-hand side)
    double *gz[kMaxLevels], *gr[kMaxLevels];
    double *ga;
    // V-cycle correction and right-hand side per level (level 0: the
    // correction of phi and the residual) in flagged words, [nz_l][nr]:
    // Flag<float>::W on the mixed path, Flag<double>::W on the FP64 path
    void *lu[kMaxLevels], *lf[kMaxLevels];
    double *fac64[kMaxLevels];                  // line factors, FP64 path
    float *fac32[kMaxLevels];                   // line factors, FP32 V-cycle
    double *facc;                               // coarsest level's line factors (FP64)
    float *facc32;                              // coarsest level's line factors, FP32 V-cycle
    double *f0;                                 // fine right-hand side
    double *dg0;                                // fine operator's diagonal
    // per residual tile, node by node (mg_tile_elems): flexible GCR(1) of the
    // mixed path -- the FP64 residual, A z of the last correction z, the
    // previous direction and its A-image; FP64 path: phi of the tile and its
    // two neighbour columns
    double *kr, *kw, *kzp, *kwp, *ps;
    // what the blocks tell one another each cycle, in flagged words: the
    // norms {max |r|, max |b|} and the GCR step's four partial dot products
    ulonglong2 *xr, *xd;
    unsigned *epoch;  // the last solve's tags end below it
    MGCtl *ctl;
    MGFast *self;  // device copy of this struct (kernels read it through a pointer)
};

// Where a solve's charge and susceptibility come from: computed by the set-up
// from the species' deposits (Ne, Ni) and the node volumes' inverses (rho and chi
// are then written), or given (Ne null).
struct FieldSource {
    const double *Ne, *Ni;
    const double2 *iV;
    double q0, q1, c0, c1;
    double *rho, *chi;
};

// Shared-memory layout of the one-launch solve (byte offsets), set on the host.
struct SolveLayout {
    // from 0 in the line phases: three line buffers (line_buffer values each)
    int offT;   // from 0 in the residual phase: the tile with its neighbour columns; at offT: two restriction buffers
    int offF;   // factor slots: each two red lines and the black line
    int offC;   // factors of the coarsest row
    int slots;  // factor slots
    int tw;     // columns per residual tile
    int tw_max; // the most there is room for (0: tw stands)
};
constexpr int kMaxSlots = 4;

// One reactor's one-launch solve, as the kernel takes it (a table of these
// drives the solves of several reactors in one cooperative launch), with its
// launch shape on the host.
struct SolveJob {
    const MGFast *mp;
    double *phi;
    int nz, nr;
    SolveLayout lay;
    double tol;
    int max_cycles;
    int block0, nblocks;  // this job's blocks in the launch
    int most;             // what it can use of a GPU with room to spare
    // host side
    int M, mixed;
    size_t smem;
    void *fn;
};

// line-factor elements of one r-line of a mesh with nr nodes per row
// (in FP64 65 to 512 unknowns are solved by more lanes: f64)
size_t mg_line_factor_elems(int nr, bool f64);
// doubles of each tile-wise array (kr, kw, kzp, kwp; ps has the neighbour columns), and the most blocks
// a solve takes (entries of xr and xd)
size_t mg_tile_elems(int nz, int nr, bool with_neighbours);
constexpr int kMaxSolveBlocks = 512;
// copies of them, so that not every block reads the same few lines of L2
constexpr int kCopies = 8;

// copy the level table to the device (once: its pointers do not change)
void mg_fast_upload(MGFast &m, cudaStream_t st);
// host values of gz, gr (every level) and ga, laid out [gz_0 gr_0 gz_1 gr_1 ... ga]
// with nr entries each; the caller copies them to one device array
void mg_fast_geometry(const MGFast &m, int nr, double dr, std::vector<double> &out);

// Solve into phi.  Alone (sctl null): returns the cycles (>= 0, converged)
// or -cycles-1, after a host synchronisation.  Inside a timestep (sctl set):
// enqueues the work only, takes the voltage from sctl->V (v_from_ctl), skips everything
// once sctl->halt is set, reports cycles, residual and failures to sctl, and
// returns 0 (or kSolveNoLaunch).  at_solve (optional) is recorded on st just
// before the one-launch solve, after the set-up: work that waits for it runs
// beside the solve.  wide: a block per SM, as many as there are line units or
// residual tiles (a reactor alone on the GPU); else one per two rows (many
// reactors solving side by side).
// defer (narrow solves of a batch): the set-up is enqueued, the solve itself
// is described in *defer and left to mg_multi_launch; the report to sctl is
// then the caller's.
// report false: the report to sctl is left to the caller (launch_efield).
// after (optional): what the voltage waits for (the set-up's first launch does not).
// pinned (optional): host memory for the read-back of a solve alone.
// phi_prev (warm solves only, optional): the potential of the step before
// phi's; the V-cycles then start from 2 phi - phi_prev on the interior, and
// phi_prev takes phi's values (the starting value w_0 of Algorithm 1,
// extrapolated linearly in time).
int mg_fast_solve(const FieldDims &fd, MGFast &m, const FieldSource &src, double V,
                  const double *phi_zL, double *phi, bool warm, bool mixed, double tol,
                  int max_cycles, double *rel_res, int *launches, StepCtl *sctl, cudaStream_t st,
                  bool v_from_ctl = true, bool setup = true, cudaEvent_t at_solve = nullptr,
                  bool wide = true, SolveJob *defer = nullptr, double *phi_prev = nullptr, bool report = true,
                  cudaEvent_t after = nullptr, MGCtl *pinned = nullptr);

// the launch shape of one reactor's solve (host only); false: not launchable
bool solve_job(const FieldDims &fd, MGFast &m, double *phi, bool mixed, double tol, int max_cycles, bool wide,
               SolveJob &job);

// Plan deferred solves for shared cooperative launches: jobs of one (precision,
// line chunk) kind share a launch; each kind gets SMs in proportion to the
// blocks its jobs would take alone, and each job's blocks are cut in
// proportion so that the launches of all kinds fit the GPU together (at
// least one block per job; a kind with more jobs than its share takes
// several launches).  concurrent (out): the kinds' launches fit side by side;
// else each takes the whole GPU and they run one after another.
// Returns the launches as [first job, end job) ranges of `jobs`, which it
// reorders by kind and fills with block0 / nblocks.  Host only.
std::vector<std::pair<int, int>> mg_multi_plan(std::vector<SolveJob> &jobs, bool &concurrent);
// launch the planned range [j0, j1) of the device copy of the table
int mg_multi_launch(const std::vector<SolveJob> &jobs, int j0, int j1, const SolveJob *jobs_dev,
                    cudaStream_t st);
}  // namespace pic
