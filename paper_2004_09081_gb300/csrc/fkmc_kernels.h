// fkmc_kernels.h -- host-side launchers of the kernels in fkmc_kernels.cu.
#pragma once
#include <cuda_runtime.h>

#include "fkmc_device.cuh"

namespace fkmc {

// sets the thread-local message of kmc_last_error() and returns `code`
int set_error(int code, const char* msg);

cudaError_t upload_neighbours(const NbEntry* host24);
cudaError_t launch_init(const RepDesc& D, int b_bits, int64_t n_vac, int64_t n_total, uint32_t* occ,
                        VacRec* recs, int32_t* counts, int cap, uint32_t* status, cudaStream_t st);
size_t phase_smem_bytes(int cap, bool site);
cudaError_t phase_prepare(int cap);
cudaError_t run_pass_blocks(int prec, int cap, bool site, bool grain, int* blocks);
cudaError_t small_pass_blocks(int prec, bool grain, int lane, int* blocks);
constexpr int64_t SPLIT_MIN_ITEMS = 32768;  // fragments per phase from which the small-fragment pass runs
constexpr int ACT_COUNTERS = 32;  // act_count: 3 active lists x 8 phases, 8 window tickets
constexpr int LANE_MAX_V = 8;      // vacancies per fragment of the persistent one-thread-per-fragment pass
constexpr int LANE_REG_MAX_V = 4;  // ... of its register form
constexpr int64_t LANE_PERSIST_ITEMS = 1 << 19;  // fragments per phase from which the persistent form runs
constexpr int LANE_NONE = 0, LANE_REGISTERS = 1, LANE_PERSISTENT = 2;
// mode: kmc_opts.small_pass (0 auto, 1 always, 2 always and grouped, -1 never)
bool window_split(bool site, int64_t total_items, int mode);
// form of the one-thread-per-fragment pass (mixed form only; LANE_NONE: the
// grouped pass); form: kmc_opts.lane_form (0 auto, 1 registers, 2 persistent)
int window_lane(int prec, int mode, int form, int64_t total_items);
// act: 3 lists of total_items entries (general, one vacancy, two vacancies);
// act_count: ACT_COUNTERS counters (list l, phase p at 8 l + p; the window
// ticket of phase p of the one-thread-per-fragment pass at 24 + p)
// cls: total_items bytes (the screen's class of each item for the register form)
cudaError_t launch_window(int prec, const RepDesc* d_descs, int nrep, int64_t total_items,
                          unsigned long long* wctl, uint32_t* perms, ActEntry* act, int32_t* act_count,
                          uint8_t* cls, uint32_t* occ, VacRec* recs, int32_t* counts, int32_t* tracer,
                          unsigned long long* stats, uint32_t* status, int cap, int run_blocks,
                          int small_blocks, bool split, int lane_form, const SiteArgs& sa, cudaStream_t st,
                          cudaStream_t side, cudaEvent_t fork, cudaEvent_t join);
cudaError_t launch_grains(const RepDesc* d_descs, int nrep, int64_t ncell_total, int n_grains, int width, int64_t* X,
                          int32_t* grain, uint8_t* gb, cudaStream_t st);
cudaError_t launch_init_dopants(const RepDesc& D, int b_bits, int64_t n_fe, uint8_t* fe, cudaStream_t st);
cudaError_t launch_site_field(const RepDesc* d_descs, int nrep, const VacRec* recs, const int32_t* counts,
                              int64_t nfrag_total, int cap, int64_t nsite_total, const uint8_t* fe,
                              const SiteOff* bo, int n_bo, const SiteArgs& sa, cudaStream_t st);
// atom-based fragment kMC with null events (fkmc_null.cu)
cudaError_t launch_null_gather(const RepDesc* d_descs, int nrep, const VacRec* recs, const int32_t* counts,
                               int64_t nfrag_total, int cap, VacRec* vac, uint32_t* status, cudaStream_t st);
cudaError_t launch_null_scatter(const RepDesc* d_descs, int nrep, int64_t total_vac, const VacRec* vac,
                                VacRec* recs, int32_t* counts, int64_t nfrag_total, int cap, uint32_t* status,
                                cudaStream_t st);
cudaError_t null_upload_neighbours(const NbEntry* host24);
cudaError_t launch_null_step(const RepDesc* d_descs, int nrep, int64_t total_vac, int64_t total_picks, VacRec* vac,
                             uint32_t* occ, const uint8_t* gb, unsigned long long* acc,
                             NullProp* props,
                             unsigned long long* claims, int32_t* tracer, double* theta, double* nE,
                             unsigned long long* stats, unsigned long long* nctl, cudaStream_t st);
// the same steps by one cooperative launch for up to NULL_LOG_STEPS of them (where the plan holds)
constexpr int NULL_LOG_STEPS = 4096;
struct NullStepsPlan {
    int ctas, per;  // CTAs per replica, vacancies and picks per thread
};
size_t null_log_bytes(int nrep, int steps);  // their log, `steps` of them at most per launch
bool null_steps_plan(int nrep, int64_t max_vac, int64_t max_sites, NullStepsPlan* out);
cudaError_t launch_null_steps(const NullStepsPlan& p, const RepDesc* d_descs, int nrep, uint64_t k0, int steps,
                              VacRec* vac, uint32_t* types, uint32_t* occ, const uint8_t* gb,
                              unsigned long long* claims, int32_t* tracer, void* log_mem, double* theta,
                              unsigned long long* stats, uint32_t* status, uint32_t stuck_wait_us, cudaStream_t st);
// read-outs: species codes of rows of the (t, z, y) order; record rows with their
// offsets per fragment (offsets: fragments + 1 entries, the last the total)
cudaError_t launch_unpack_state(const RepDesc& D, const uint32_t* occ, int64_t row0, int64_t rows, uint8_t* out,
                                cudaStream_t st);
cudaError_t launch_rows(const RepDesc& D, const VacRec* recs, const int32_t* counts, int cap, int64_t* offsets,
                        int64_t max_rows, int64_t* rows, cudaStream_t st);
cudaError_t launch_moments(const RepDesc& D, int species, const uint32_t* occ, const VacRec* recs,
                           const int32_t* counts, const int32_t* tracer, int cap,
                           unsigned long long* out, cudaStream_t st);

cudaError_t launch_moments_all(const RepDesc* d_descs, int nrep, const VacRec* recs, const int32_t* counts,
                               int64_t max_frag_per_replica, int cap, unsigned long long* out, cudaStream_t st);

// electrostatics of the mu-scale model (fkmc_poisson.cu): multigrid on the B-site grid
constexpr int MG_MAX_LEVELS = 16;
constexpr int MG_PARTIALS = 256;  // blocks of the deterministic reductions
struct MgPlan {
    int levels;
    int dim[MG_MAX_LEVELS][3];
    int64_t off[MG_MAX_LEVELS];  // first node of each level in the level-stacked buffers
    int64_t total;
};
struct MgBuffers {
    double* phi;     // [level-0 nodes] the potential (FP64)
    double* f;       // [level-0 nodes] right-hand side (FP64)
    double* r;       // [level-0 nodes] residual of the final check
    float* e;        // [total] FP32 correction per level
    float* g;        // [total] FP32 right-hand side per level (level 0: the FP64 defect, rounded)
    float* s;        // [total] FP32 residual (and the Jacobi scratch of an odd level)
    int32_t* cnt;    // [level-0 nodes] half-charge counts
    double* part;    // [MG_PARTIALS]
    double* scalar;  // [2]
};
MgPlan mg_plan(int nx, int ny, int nz);
int64_t mg_cycle_kernels(const MgPlan& p);  // kernel launches of one V-cycle
cudaError_t elec_solve(const RepDesc& D, const VacRec* recs, const int32_t* counts, int cap, int64_t n_vac,
                       double q, double scale, int cycles, const MgPlan& p, const MgBuffers& b, double* resid_rel,
                       const double* init, double* save, cudaStream_t st);
cudaError_t elec_solve_unit(const RepDesc& D, int t, double scale, int cycles, const MgPlan& p, const MgBuffers& b,
                            cudaStream_t st);
cudaError_t elec_update(const RepDesc& D, const double* phi, double q, int32_t* u, int32_t* field, unsigned* umax,
                        cudaStream_t st);
cudaError_t elec_add(int32_t* field, const int32_t* u, int64_t n, cudaStream_t st);

// Per fragment (batch-wide index) the screen's limit that the resident kernels
// leave at the end of a launch, and per replica whether they are still valid: the
// host clears `valid` whenever anything but a resident run changes a replica's
// state or rates, and the next launch then starts from every fragment unknown.
struct ResCache {
    uint64_t* lim;
    uint8_t* valid;
};

// resident kernels (fkmc_resident.cu): a replica's occupancy in the shared memory
// of one CTA, or of a thread-block cluster, CTA c holding the z-slab of fragment
// layers [fz0[c], fz0[c+1])
constexpr int RESIDENT_MAX_SLOTS = 64;            // vacancy slots per fragment (kmc_opts.cap_v) they take
constexpr size_t RESIDENT_MAX_SMEM = 220 * 1024;  // dynamic shared memory per CTA
constexpr int CLUSTER_MAX_CTAS = 16;
constexpr int CLUSTER_THREADS = 512;
struct ClusterPlan {
    int32_t rep;                          // replica index in the batch
    int32_t ncta;                         // CTAs of the cluster
    int32_t fz0[CLUSTER_MAX_CTAS + 1];    // fragment layers of CTA c: [fz0[c], fz0[c + 1])
    int32_t zs;                           // cells in z of the thickest slab (the common layout)
    int32_t nfl;                          // fragments of the thickest slab
};
struct ResidentArgs {  // fixed for a batch and its plan
    const RepDesc* descs;
    uint32_t* occ;
    VacRec* recs;
    VacRec* tmp;       // stage-out copies of the records, by RepDesc.tmp_off
    uint32_t* vmap;    // record index of every vacancy's site, by RepDesc.vmap_off
    int32_t* counts;
    int32_t* tracer;
    unsigned long long* stats;
    uint32_t* status;
    int cap;
    NbTable nbt;
    int64_t frag_tot;  // fragments of all resident replicas (stride of the plain form's draws)
    int draw_ev;       // events per fragment in the plain form's draws
    SiteArgs sa;       // plain form with site energies
    uint32_t stuck_wait_us;
    ResCache rc;
};
size_t resident_smem_bytes(const RepDesc& D, int cap, int threads, int pre_g, int pre_ev, int prec);
size_t cluster_smem_bytes(const RepDesc& D, const ClusterPlan& p, int cap, int pre_ev, int prec);
// the plan with the most CTAs in [min_ctas, max_ctas] whose slabs fit one SM's shared memory
bool make_cluster_plan(const RepDesc& D, int cap, int pre_ev, int prec, int min_ctas, int max_ctas, ClusterPlan* out);
int cluster_fits(int form, int ncta, size_t smem);  // clusters of this shape the GPU can hold at once
cudaError_t resident_prepare();
// first draws of `windows` windows from w0 on, of every resident replica (plain form)
cudaError_t launch_gate(cudaStream_t st);  // an empty kernel
cudaError_t launch_draws(const RepDesc* d_descs, int nrep, int64_t max_frag, uint64_t w0, int windows, int ev_per,
                         int64_t frag_tot, Draw* draws, cudaStream_t st);
// form: 0 plain, 1 mixed, 2 plain with site energies, 3 mixed with lists of sixteen vacancies
cudaError_t launch_resident(int form, const ResidentArgs& a, const int32_t* d_reps, int nreps, size_t smem, int threads,
                            uint64_t w0, uint64_t windows, const Draw* draws, cudaStream_t st);
cudaError_t launch_cluster(int form, const ResidentArgs& a, const ClusterPlan* d_plans, int nplans, int ncta,
                           size_t smem, uint64_t w0, uint64_t windows, const Draw* draws, cudaStream_t st);

}  // namespace fkmc
