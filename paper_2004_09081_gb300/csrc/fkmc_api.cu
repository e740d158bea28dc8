// fkmc_api.cu -- host side of the C ABI declared in include/fkmc.h:
// validation, partition of the lattice into fragments, device buffers,
// rate tables (Eq. RateCnst1 of arXiv:2004.09081 with the ESP shift of
// Sec. III), the window loop and the read-outs.
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <iterator>
#include <string>
#include <type_traits>
#include <vector>

#include "fkmc.h"
#include "fkmc_check.h"
#include "fkmc_kernels.h"

namespace {
// NVTX range over one ABI call, named after it (shown by Nsight tools; without
// a tool attached the header-only NVTX calls do nothing)
struct NvtxRange {
    explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange&) = delete;
    NvtxRange& operator=(const NvtxRange&) = delete;
};
}  // namespace

using namespace fkmc;

namespace {

thread_local std::string g_err;

int fail(int code, const std::string& msg)
{
    g_err = msg;
    return code;
}

int cuda_fail(cudaError_t e, const char* what)
{
    return fail(FKMC_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

#define CK(call, what)                                  \
    do {                                                \
        cudaError_t e_ = (call);                        \
        if (e_ != cudaSuccess) return cuda_fail(e_, what); \
    } while (0)

const double KB_EV = 8.617333262e-5;  // Boltzmann constant, eV/K (R of Eq. RateCnst1)

// Neighbour table built from the geometry: a site of type t sits at a/2 e_t
// from its cell corner; its 8 nearest O neighbours are at a/2 (s_t e_t + s_u e_u)
// for the two other axes u and signs s_t, s_u = +-1.  The neighbour has type u
// and lies in the cell offset (d + e_t - e_u)/2.  Listed in ascending (dx,dy,dz).
void build_nb_table(NbEntry tab[3][8])
{
    for (int t = 0; t < 3; ++t) {
        struct Row { int d[3]; int u; };
        std::vector<Row> rows;
        for (int u = 0; u < 3; ++u) {
            if (u == t) continue;
            for (int st = -1; st <= 1; st += 2)
                for (int su = -1; su <= 1; su += 2) {
                    Row r{};
                    r.d[t] = st;
                    r.d[u] = su;
                    r.u = u;
                    rows.push_back(r);
                }
        }
        std::sort(rows.begin(), rows.end(), [](const Row& a, const Row& b) {
            return std::lexicographical_compare(a.d, a.d + 3, b.d, b.d + 3);
        });
        for (int n = 0; n < 8; ++n) {
            NbEntry& e = tab[t][n];
            e.t2 = (int8_t)rows[n].u;
            for (int k = 0; k < 3; ++k) {
                e.d[k] = (int8_t)rows[n].d[k];
                e.dc[k] = (int8_t)((rows[n].d[k] + (k == t) - (k == rows[n].u)) / 2);
            }
            e.pad = 0;
        }
    }
}

int partition_count(int L, int edge)
{
    int nf = 2 * (int)std::floor((double)L / (2.0 * edge) + 0.5);
    if (nf < 2) nf = L >= 4 ? 2 : 1;
    while (nf > 1 && L / nf < 2) nf -= 2;
    if (nf < 1) nf = 1;
    return nf;
}

bool partition_ok(int L, int nf)
{
    if (nf < 1 || nf > L) return false;
    if (nf == 1) return true;
    return (nf % 2 == 0) && (L / nf >= 2);
}

int ceil_log2(int64_t v)
{
    int lg = 0;
    while (((int64_t)1 << lg) < v) ++lg;
    return lg;
}

}  // namespace

namespace fkmc {
// error reporting shared with the other translation units of the library
int set_error(int code, const char* msg)
{
    return fail(code, msg);
}
}  // namespace fkmc

struct kmc_batch {
    int n = 0;
    kmc_opts opts{};
    cudaStream_t st = nullptr;
    int cap = 0;
    std::vector<RepDesc> desc;
    std::vector<int64_t> n_vac, n_H;
    std::vector<int> b_bits;
    std::vector<double> a_ang;
    std::vector<unsigned long long> stats_host;  // hops, handoffs per replica
    int64_t nfrag_total = 0, occ_words = 0, nsite_total = 0, total_items = 0;
    bool rates_set = false;
    // device buffers
    uint32_t* occ = nullptr;
    VacRec* recs = nullptr;
    int32_t* counts = nullptr;
    int32_t* tracer = nullptr;
    RepDesc* d_desc = nullptr;
    unsigned long long* stats = nullptr;
    uint32_t* status = nullptr;
    unsigned long long* scratch = nullptr;  // 7 moments
    unsigned long long* scratch_all = nullptr;  // 7 moments per replica
    unsigned long long* check_buf = nullptr;    // CHECK_WORDS sums of kmc_check_invariants
    void* read_buf = nullptr;                   // read-outs: expanded codes or record rows (READ_BUF_MAX at most)
    size_t read_bytes = 0;
    bool records_match = true;                  // every replica holds one record per vacancy, as far as the host knows
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    std::vector<void*> owned;
    // replica-resident kernel: replicas grouped by shared-memory size class
    NbTable nbt{};
    int32_t* d_reps = nullptr;   // resident replica ids, class by class
    ClusterPlan* d_plans = nullptr;  // cluster-resident replicas' slab plans, grouped by CTA count
    ResCache rcache{};               // fragment totals the resident kernels carry from call to call
    uint32_t* vmap = nullptr;        // resident replicas: record index of every vacancy's site
    VacRec* rec_tmp = nullptr;       // and the stage-out copies of their records
    Draw* draws = nullptr;           // plain form: first draws of draw_windows windows, two buffers
    size_t vmap_bytes = 0, tmp_bytes = 0, draws_bytes = 0;
    int64_t res_frags = 0, res_max_frag = 0;
    int res_ev = 4, draw_windows = 0;
    cudaStream_t draw_st = nullptr;
    cudaEvent_t draw_done[2] = {nullptr, nullptr}, draw_free[2] = {nullptr, nullptr};
    // a launch of the resident kernel: one CTA per replica (start/count index d_reps)
    // or, with slabs, one cluster of `cluster` CTAs per replica (index d_plans)
    struct RClass {
        int start, count;
        size_t smem;
        int threads;
        int cluster;
        cudaStream_t st;
        cudaEvent_t done;
        bool slabs;
        bool long_lists;  // a replica of the class has lists of sixteen vacancies
    };
    std::vector<RClass> rclass;
    cudaEvent_t fork = nullptr;
    cudaGraphExec_t res_exec = nullptr;  // one call's class launches (fork, launches, join), captured
    uint64_t res_exec_windows = 0;
    cudaStream_t res_st = nullptr;       // the graph's stream, beside the colour-phase launches
    cudaEvent_t res_fork = nullptr, res_join = nullptr;
    cudaStream_t side_st = nullptr;       // the small-fragment run pass, beside the general one
    cudaEvent_t side_fork = nullptr, side_join = nullptr;
    bool any_global = true;
    int cluster_top = 0;  // how many of the largest replicas run as 2-CTA clusters (kmc_opts)
    std::vector<int32_t> run_kernel, run_ctas;  // per replica: kmc_replica_info.kernel and .ctas
    // colour-phase path: per-window set-up, screen and run, captured once in a graph
    unsigned long long* wctl = nullptr;  // [0] windows of this call so far, [1] current offset
    uint32_t* perms = nullptr;           // colour order of every replica, this window
    ActEntry* act = nullptr;             // screened fragments of a phase
    int32_t* act_count = nullptr;        // per list and phase
    uint8_t* cls = nullptr;              // per work item: the screen's class for the register lane pass
    int run_blocks = 0;
    cudaStream_t cap_st = nullptr;
    cudaGraphExec_t window_exec = nullptr;
    // site-energy interactions (plain form, colour-phase kernels)
    bool site_on = false;
    bool field_valid = false;
    std::vector<int64_t> n_fe;
    std::vector<double> T;           // temperature of every replica (kmc_set_barriers)
    int n_vv = 0, n_bo = 0, e_self = 0;
    int reach_vv = 0;                // largest cell offset of the V-V shells
    int64_t e_bound = 0;             // bound on |E_site|, 1e-4 eV units
    int64_t ncell_total = 0;
    uint8_t* fe = nullptr;           // one byte per cell, batch-wide cell index
    int32_t* field = nullptr;        // E_site per O site
    SiteOff* d_vv = nullptr;
    SiteOff* d_bo = nullptr;
    double* btab = nullptr;          // Boltzmann tables of every replica
    size_t btab_bytes = 0;
    // electrostatics (mu-scale model): potential of the vacancy charges, frozen between refreshes
    bool elec_on = false;
    kmc_electrostatics elec{};
    int32_t* elec_u = nullptr;          // q phi per O site, 1e-4 eV units (batch-wide site index)
    int32_t* d_elec_g = nullptr;        // [replica][3][8] own-potential share of a hop
    std::vector<int32_t> elec_g;        // host copy
    unsigned* d_umax = nullptr;         // max |u| of the last refresh
    int64_t elec_umax = 0;
    uint64_t elec_age = 0;              // windows since the last refresh
    MgPlan mg{};
    MgBuffers mgb{};
    int64_t mg_total = -1, mg_nodes = -1;
    double* phi_prev = nullptr;         // each replica's last potential (warm start of the next solve)
    struct ElecGraph {                  // one refresh solve + update of replica r, captured
        int r, cycles;
        bool warm, field;
        cudaGraphExec_t exec;
    };
    std::vector<ElecGraph> elec_graphs;
    bool phi_prev_valid = false;
    // grains (mu-scale model): boundary cells raise the barrier of hops touching them
    bool grains_on = false;
    kmc_grains grains{};
    int32_t* grain = nullptr;              // grain of every cell
    uint8_t* gbound = nullptr;             // boundary flag of every cell
    int64_t* gX = nullptr;                 // seed positions
    int64_t gX_len = 0;
    std::vector<kmc_barrier_table> tables; // of the last kmc_set_barriers
    std::vector<double> Ez;
    // atom-based fragment kMC with null events (Sec. II.B)
    VacRec* vac = nullptr;                 // vacancies by id, replica after replica
    int64_t vac_cap = 0;
    unsigned long long* claims = nullptr;  // per site: (step tag, pick) of the earliest claim
    NullProp* props = nullptr;
    int64_t props_cap = 0;
    unsigned long long* nacc = nullptr;    // R_tot, R_max, N_updated per replica
    double* theta = nullptr;               // null-event clock per replica (1/k32max units)
    double* nE = nullptr;                  // the current step's clock variate per replica
    unsigned long long* nctl = nullptr;    // [0] steps of this call so far, [1] current step, [2] blocks done
    std::vector<double> theta_host;
    uint32_t* null_types = nullptr;        // one launch for many steps: packed event types per vacancy
    void* null_log = nullptr;              // and each replica's barrier and sums per step
    size_t null_types_bytes = 0, null_log_size = 0;
    cudaGraphExec_t null_exec = nullptr;
    int64_t null_exec_picks = -1, null_exec_vac = -1;
    bool null_exec_grains = false;

    void* dalloc(size_t bytes)
    {
        bytes = (bytes + 255) & ~(size_t)255;
        if (bytes == 0) bytes = 256;
        void* p = nullptr;
        if (opts.alloc) {
            p = opts.alloc(opts.alloc_ctx, bytes);
        } else if (cudaMalloc(&p, bytes) != cudaSuccess) {
            cudaGetLastError();
            p = nullptr;
        }
        if (p) owned.push_back(p);
        return p;
    }

    void dfree(void* p)
    {
        if (!p) return;
        auto it = std::find(owned.begin(), owned.end(), p);
        if (it == owned.end()) return;
        owned.erase(it);
        if (opts.alloc) {
            if (opts.free) opts.free(opts.alloc_ctx, p);
        } else {
            cudaFree(p);
        }
    }

    void release()
    {
        for (void* p : owned) {
            if (opts.alloc) {
                if (opts.free) opts.free(opts.alloc_ctx, p);
            } else {
                cudaFree(p);
            }
        }
        owned.clear();
        if (ev0) cudaEventDestroy(ev0);
        if (ev1) cudaEventDestroy(ev1);
        if (fork) cudaEventDestroy(fork);
        ev0 = ev1 = fork = nullptr;
        if (side_fork) cudaEventDestroy(side_fork);
        if (side_join) cudaEventDestroy(side_join);
        if (side_st) cudaStreamDestroy(side_st);
        side_fork = side_join = nullptr;
        side_st = nullptr;
        for (auto& c : rclass) {
            if (c.st) cudaStreamDestroy(c.st);
            if (c.done) cudaEventDestroy(c.done);
        }
        rclass.clear();
        if (window_exec) cudaGraphExecDestroy(window_exec);
        if (res_exec) cudaGraphExecDestroy(res_exec);
        res_exec = nullptr;
        if (res_st) cudaStreamDestroy(res_st);
        if (res_fork) cudaEventDestroy(res_fork);
        if (res_join) cudaEventDestroy(res_join);
        res_st = nullptr;
        res_fork = res_join = nullptr;
        if (draw_st) cudaStreamDestroy(draw_st);
        draw_st = nullptr;
        for (int k = 0; k < 2; ++k) {
            if (draw_done[k]) cudaEventDestroy(draw_done[k]);
            if (draw_free[k]) cudaEventDestroy(draw_free[k]);
            draw_done[k] = draw_free[k] = nullptr;
        }
        if (null_exec) cudaGraphExecDestroy(null_exec);
        null_exec = nullptr;
        for (auto& g : elec_graphs) cudaGraphExecDestroy(g.exec);
        elec_graphs.clear();
        if (cap_st) cudaStreamDestroy(cap_st);
        window_exec = nullptr;
        cap_st = nullptr;
    }
};

namespace {

// the site-energy run pass is on: shells, dopant energies or electrostatics
bool site_path(const kmc_batch* b) { return b->site_on || b->elec_on; }

// anything but a resident run changed a replica's state or rates: the resident
// kernels' fragment totals from the last call no longer hold
int drop_resident_cache(kmc_batch* b)
{
    if (b->rcache.valid) CK(cudaMemsetAsync(b->rcache.valid, 0, (size_t)b->n, b->st), "memset");
    return FKMC_OK;
}

// kernel launches of one window of the colour-phase path: set-up, then per phase
// screen + run, + the grouped small pass where it runs, or the one-thread-per-
// fragment pass + run
uint64_t window_launches(const kmc_batch* b)
{
    const bool split = window_split(site_path(b), b->total_items, b->opts.small_pass);
    return split && window_lane(b->opts.precision, b->opts.small_pass, b->opts.lane_form, b->total_items) !=
                        LANE_PERSISTENT
               ? 25
               : 17;
}

int check_status(kmc_batch* b, uint32_t* word = nullptr)
{
    uint32_t s = 0;
    CK(cudaMemcpyAsync(&s, b->status, sizeof s, cudaMemcpyDeviceToHost, b->st), "status copy");
    CK(cudaStreamSynchronize(b->st), "synchronize");
    if (word) *word = s;
    if (s) b->records_match = false;
    if (s & STATUS_OVERFLOW)
        return fail(FKMC_EOVERFLOW, "a fragment received more vacancies than cap_v slots");
    if (s & STATUS_TIMEOUT) return fail(FKMC_ETIMEOUT, "a device-side wait ran out of time");
    if (s & STATUS_EVENT_LIMIT)
        return fail(FKMC_ETIMEOUT, "a fragment reached the per-phase event limit (window too long)");
    if (s & STATUS_ENERGY_RANGE)
        return fail(FKMC_ESTATE, "a site-energy difference fell outside the Boltzmann tables' bound");
    return FKMC_OK;
}

int upload_desc(kmc_batch* b)
{
    CK(cudaMemcpyAsync(b->d_desc, b->desc.data(), sizeof(RepDesc) * b->n, cudaMemcpyHostToDevice, b->st),
       "descriptor upload");
    CK(cudaStreamSynchronize(b->st), "synchronize");
    return FKMC_OK;
}

int rate_table_impl(const kmc_barrier_table* t, double T_K, double Ez, double a_ang, int cap_v,
                    double k64[6], float k32[6], uint64_t q[6], int32_t* F_out)
{
    if (!t || !(T_K > 0.0) || !std::isfinite(T_K) || !std::isfinite(Ez) || !(a_ang > 0.0) ||
        !std::isfinite(t->Ea_O_eV) || !std::isfinite(t->Ea_H_eV) || !(t->prefactor > 0.0) ||
        !std::isfinite(t->q_O) || !std::isfinite(t->q_H) || cap_v < 1)
        return fail(FKMC_EINVAL, "rate table: T must be > 0, inputs finite, prefactor > 0");
    const double Ea[2] = {t->Ea_O_eV, t->Ea_H_eV};
    const double qc[2] = {t->q_O, t->q_H};
    const double half_a_m = 0.5 * a_ang * 1e-10;
    for (int h = 0; h < 2; ++h)
        for (int dz = -1; dz <= 1; ++dz) {
            // Eq. (RateCnst1) with the vacancy's z step dz a/2 shifting the barrier by dU/2
            const double dz_m = (double)dz * half_a_m;
            const double dU = -(qc[h] * Ez) * dz_m;
            const double barrier = Ea[h] + 0.5 * dU;
            k64[3 * h + dz + 1] = t->prefactor * std::exp(-(barrier / (KB_EV * T_K)));
        }
    float kmax = 0.0f;
    for (int i = 0; i < 6; ++i) {
        k32[i] = (float)k64[i];
        kmax = std::max(kmax, k32[i]);
    }
    if (!(kmax > 0.0f) || !std::isfinite(kmax))
        return fail(FKMC_EINVAL, "rate table: rates underflow or overflow in fp32");
    const int F = 63 - ceil_log2(8 * (int64_t)cap_v);
    for (int i = 0; i < 6; ++i) q[i] = (uint64_t)std::llrint(std::ldexp((double)k32[i] / (double)kmax, F));
    *F_out = F;
    return FKMC_OK;
}

bool valid_replica(const kmc_batch* b, int32_t r) { return b && r >= 0 && r < b->n; }

// Forgets the launch classes and the captured launches that hold them.
void drop_classes(kmc_batch* b)
{
    if (b->res_exec) cudaGraphExecDestroy(b->res_exec);
    b->res_exec = nullptr;
    for (auto& c : b->rclass) {
        if (c.st) cudaStreamDestroy(c.st);
        if (c.done) cudaEventDestroy(c.done);
    }
    b->rclass.clear();
}

// Every replica on the colour-phase passes, which need no memory of their own.
void plan_passes(kmc_batch* b)
{
    drop_classes(b);
    for (RepDesc& D : b->desc) D.resident = 0;
    b->run_kernel.assign(b->n, 0);
    b->run_ctas.assign(b->n, 0);
    b->any_global = true;
    b->res_frags = b->res_max_frag = 0;
}

// Device buffers of the resident replicas: site -> record maps, stage-out copies,
// first draws (plain form).  False where the allocator has no room.
bool resident_buffers(kmc_batch* b, int prec, int plain_ev)
{
    int64_t sites = 0, frags = 0;
    b->res_max_frag = 0;
    for (RepDesc& D : b->desc) {
        D.vmap_off = sites;
        D.tmp_off = D.draw_off = frags;
        if (!D.resident) continue;
        const int64_t nf = (int64_t)D.nf[0] * D.nf[1] * D.nf[2];
        sites += 48 * (int64_t)D.L[2] * D.L[1] * D.row_words;  // sixteen sites per occupancy word
        frags += nf;
        b->res_max_frag = std::max(b->res_max_frag, nf);
    }
    b->res_frags = frags;
    b->res_ev = plain_ev;
    auto grow = [&](void** p, size_t* have, size_t want) -> bool {
        if (want <= *have) return true;
        b->dfree(*p);
        *p = b->dalloc(want);
        *have = *p ? want : 0;
        return *p != nullptr;
    };
    b->draw_windows = 0;
    if (frags == 0) return true;
    if (prec == 0) {  // two buffers of up to 64 windows, 64 MB together where one window fits
        const int64_t per = frags * plain_ev * (int64_t)sizeof(Draw);
        b->draw_windows = (int)std::max<int64_t>(1, std::min<int64_t>(64, ((int64_t)32 << 20) / per));
        if (!grow((void**)&b->draws, &b->draws_bytes, 2 * (size_t)per * b->draw_windows)) return false;
    }
    return grow((void**)&b->vmap, &b->vmap_bytes, sizeof(uint32_t) * (size_t)sites) &&
           grow((void**)&b->rec_tmp, &b->tmp_bytes, sizeof(VacRec) * (size_t)frags * b->cap);
}

// Decide which replicas run in the replica-resident kernel and group them
// into shared-memory size classes (one launch per class, on forked streams).
int plan_residency(kmc_batch* b)
{
    if (int rc0 = drop_resident_cache(b)) return rc0;
    drop_classes(b);
    const int prec = b->opts.precision == FKMC_MIXED ? 1 : 0;
    const bool allowed = b->opts.schedule != 1 && (prec == 1 || b->opts.schedule == 0) &&
                         b->cap <= RESIDENT_MAX_SLOTS && !b->grains_on;
    const int form = prec ? 1 : (site_path(b) ? 2 : 0);
    int sms = 0, dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        sms = 1;
    // launch classes: (shared-memory bound, threads); a replica takes the first
    // class its state fits, so small replicas pack several CTAs per SM and the
    // largest get the most warps.
    const size_t bounds[4] = {24 * 1024, 48 * 1024, 96 * 1024, RESIDENT_MAX_SMEM};
    const int threads[4] = {128, 128, 256, 512};
    // events per fragment drawn ahead in the plain form (k_draws): about twice
    // the expected number of a visit
    double mean = 0.0;
    for (int r = 0; r < b->n; ++r)
        mean = std::max(mean, (double)b->n_vac[r] / ((double)b->desc[r].nf[0] * b->desc[r].nf[1] * b->desc[r].nf[2]));
    const int plain_ev = mean * b->opts.n_tau <= 0.5 ? 4 : 8;
    std::vector<std::vector<int>> cls(4);
    std::vector<size_t> cmax(4, 0), need_of(b->n, 0);
    std::vector<ClusterPlan> plans;
    std::vector<int> pairs;  // replicas that may run on two CTAs (kmc_opts.cluster_top)
    b->run_kernel.assign(b->n, 0);
    b->run_ctas.assign(b->n, 0);
    const int force = b->opts.cluster_ctas;
    // clusters of nc CTAs that the GPU holds at once (one CTA of these kernels fills an
    // SM's registers, whatever its shared memory)
    int fit_count[CLUSTER_MAX_CTAS + 1];
    std::fill(fit_count, fit_count + CLUSTER_MAX_CTAS + 1, -1);
    auto fits = [&](int nc) -> int {
        if (fit_count[nc] < 0) fit_count[nc] = cluster_fits(form, nc, RESIDENT_MAX_SMEM);
        return fit_count[nc];
    };
    // lists of sixteen vacancies where a fragment often holds more than eight and is so
    // large that scanning it is slow (more than 31 cells per lane), mixed form: 96^3 cells
    // in 12^3-cell fragments at 0.001 vacancies per site (5.2 a fragment) 85.7 -> 76.3 us
    // per window; fragments of 8^3 cells gain less than the longer code costs the rest
    auto long_lists = [&](int r) {
        const RepDesc& D = b->desc[r];
        int e[3];
        for (int d = 0; d < 3; ++d) e[d] = D.base[d] + (D.rem[d] > 0 ? 1 : 0);
        return prec == 1 && (double)b->n_vac[r] > 4.0 * D.nf[0] * D.nf[1] * D.nf[2] &&
               (int64_t)((e[1] * e[2] + 31) / 32) * e[0] > 31;
    };
    // replica r on the most of lo..hi CTAs that hold it and that the GPU can place
    struct Placed {
        RepDesc D;
        ClusterPlan pl;
    };
    auto slabs_of = [&](int r, int lo, int hi, Placed* out) -> bool {
        // (events drawn ahead, list entries), the next where the slabs do not fit
        const int ev = prec ? 4 : plain_ev;
        const int want[5][2] = {{ev, 16}, {ev, 8}, {ev, 4}, {4, 4}, {2, 4}};
        for (int nc = std::min(hi, (int)b->desc[r].nf[2]); nc >= lo; --nc) {
            if (fits(nc) <= 0) continue;
            for (int q = long_lists(r) ? 0 : 1; q < (form == 2 ? 10 : 5); ++q) {
                if (q == 5 && !long_lists(r)) continue;
                out->D = b->desc[r];
                out->D.btab_smem = form == 2 && q < 5;
                out->D.kslots = want[q % 5][1];
                out->D.pre_ev = want[q % 5][0];
                out->pl = ClusterPlan{};
                if (!make_cluster_plan(out->D, b->cap, out->D.pre_ev, prec, nc, nc, &out->pl)) continue;
                out->pl.rep = r;
                out->D.resident = 1;
                return true;
            }
        }
        return false;
    };
    auto put_on_cluster = [&](const Placed& c) {
        const int r = c.pl.rep;
        b->desc[r] = c.D;
        plans.push_back(c.pl);
        b->run_kernel[r] = 2;
        b->run_ctas[r] = c.pl.ncta;
    };
    // fragments and vacancies per colour phase
    auto phase_frags = [&](int r) {
        const int32_t* nf = b->desc[r].nf;
        return (int64_t)((nf[0] + 1) / 2) * ((nf[1] + 1) / 2) * ((nf[2] + 1) / 2);
    };
    auto phase_vacs = [&](int r) {
        const int32_t* nf = b->desc[r].nf;
        return (double)b->n_vac[r] / ((nf[0] > 1 ? 2 : 1) * (nf[1] > 1 ? 2 : 1) * (nf[2] > 1 ? 2 : 1));
    };
    std::vector<int> wide;  // replicas that only a cluster can hold
    for (int r = 0; r < b->n; ++r) {
        RepDesc& D = b->desc[r];
        int c = -1;
        size_t need = 0;
        // (Boltzmann tables in shared memory, list entries), the next where the state does not fit
        const int lay[6][2] = {{form == 2, 16}, {0, 16}, {form == 2, 8}, {0, 8}, {form == 2, 4}, {0, 4}};
        for (int q = long_lists(r) ? 0 : 2; q < 6 && allowed && c < 0; ++q) {
            D.btab_smem = lay[q][0];
            D.kslots = lay[q][1];
            for (int k = 0; k < 4 && c < 0; ++k) {
                need = resident_smem_bytes(D, b->cap, threads[k], 1, prec ? 2 : plain_ev, prec);
                if (need <= bounds[k]) c = k;
            }
        }
        // the first draws of as many colour phases per batch as the class's shared
        // memory allows beside the state (8: one batch per window): four events per
        // fragment where 2 or more phases of them fit, else two
        D.pre_g = 1;
        D.pre_ev = prec ? 2 : plain_ev;
        static const int pick[6][2] = {{8, 4}, {4, 4}, {2, 4}, {8, 2}, {4, 2}, {2, 2}};  // (phases, events)
        for (int k = 0; c >= 0 && k < 6; ++k) {
            const int ev = prec ? pick[k][1] : plain_ev;
            const size_t ng = resident_smem_bytes(D, b->cap, threads[c], pick[k][0], ev, prec);
            if (ng <= bounds[c]) {
                D.pre_g = pick[k][0];
                D.pre_ev = ev;
                need = ng;
                break;
            }
        }
        // a cluster: a replica too large for one SM, below, or, with cluster_ctas
        // forced, every replica with exactly so many CTAs
        Placed forced;
        if (allowed && force >= 2 && slabs_of(r, force, force, &forced)) {
            put_on_cluster(forced);
            continue;
        }
        if (c < 0 && allowed && force == 0) wide.push_back(r);
        D.resident = c >= 0 ? 1 : 0;
        if (c < 0) continue;
        cls[c].push_back(r);
        need_of[r] = need;
        b->run_kernel[r] = 1;
        b->run_ctas[r] = 1;
    }
    // how many SMs the classes take (a class's CTAs per SM, by registers: 4, 4, 2, 1)
    const double share[4] = {0.25, 0.25, 0.5, 1.0};
    auto singles_sms = [&]() {
        double used = 0.0;
        for (int c = 0; c < 4; ++c) used += share[c] * (double)cls[c].size();
        return used;
    };
    auto sms_used = [&]() {
        double used = singles_sms();
        for (const ClusterPlan& pl : plans) used += pl.ncta;
        return used;
    };
    // Estimate of a resident replica's window, us: the longest of a phase's visits (on one
    // CTA it grows with their number), each visit per warp, each vacancy of a fragment, and
    // the screen and draws per fragment and CTA.  Fitted to 70 timings on one GB300 of 8^3
    // .. 128^3 cells at 0.001 to 0.02 vacancies per site, on one CTA and on 2 to 16 (within
    // 30%); the lines below need no better.
    auto window_us = [&](int r, int nc, double warps) {
        static const double c1[3] = {6.5, 5.5, 11.0}, cn[3] = {41.0, 36.0, 63.0}, per_visit[3] = {4.6, 3.7, 8.0},
                            per_vac[3] = {7.0, 4.0, 7.0}, per_frag[3] = {0.04, 0.04, 0.08};
        const int32_t* nf = b->desc[r].nf;
        const int busy = nc > 1 ? std::min(nc, std::max(1, nf[2] / 2)) : 1;  // a phase takes every other layer
        return (nc > 1 ? cn[form] : c1[form] * std::log(1.0 + phase_vacs(r))) + per_visit[form] * phase_vacs(r) / (warps * busy) +
               per_vac[form] * (double)b->n_vac[r] / ((double)nf[0] * nf[1] * nf[2]) +
               per_frag[form] * (double)phase_frags(r) / busy;
    };
    // a set of replicas on clusters of at most hi CTAs: their share of the GPU (1: it is
    // full, as the GPU can place no more of them at once) and the longest window
    struct Group {
        std::vector<Placed> on;
        double load = 0.0, us = 0.0;
        int most = 0;  // CTAs of the largest
    };
    auto group = [&](const std::vector<int>& list, int lo, int hi, auto limit) {
        Group g;
        Placed p;
        for (int r : list)
            if (slabs_of(r, lo, std::min(hi, limit(r)), &p)) {
                g.load += 1.0 / fits(p.pl.ncta);
                g.us = std::max(g.us, window_us(r, p.pl.ncta, CLUSTER_THREADS / 32));
                g.most = std::max(g.most, p.pl.ncta);
                g.on.push_back(p);
            }
        return g;
    };
    // Replicas that only a cluster can hold: the most CTAs at which all run at once, and
    // where no size does, the one with the shortest estimate (waves times window).  64^3
    // cells in 16^3 fragments at 0.001 vacancies per site, mixed: 39 us per window on 16
    // CTAs, 49 on 3, but the GPU holds 7 clusters of 16 and 46 of 3, so that 32 replicas
    // take 190 us on 16 CTAs and 45 on 4.
    double load = singles_sms() / sms, cluster_load = 0.0, slowest = 0.0;
    if (!wide.empty()) {
        Group best;
        double best_us = 0.0;
        for (int hi = CLUSTER_MAX_CTAS; hi >= 2;) {
            Group g = group(wide, 2, hi, [](int) { return CLUSTER_MAX_CTAS; });
            if (g.on.size() < best.on.size() || g.most == 0) break;  // too few CTAs for some
            const double us = std::ceil(load + g.load - 1e-9) * g.us;
            hi = g.most - 1;
            if (best.on.empty() || us < best_us) {
                best = std::move(g);
                best_us = us;
                if (load + best.load <= 1.0) break;
            }
        }
        for (const Placed& p : best.on) put_on_cluster(p);
        load += best.load;
        cluster_load = best.load;
        slowest = best.us;
    }
    // Replicas with four visits or more per warp and phase, or 128 fragments or more to
    // look at, on clusters instead of one CTA each where the GPU can place all of them at
    // once: of 48^3 cells in 12^3 fragments, 0.02 vacancies per site, plain 289 -> 117 us
    // per window (mixed 137 -> 85), in 8^3 fragments 510 -> 277 (mixed 197 -> 158). Fewer
    // visits are not worth the cluster's barriers: 32^3 cells in 8^3 fragments at 0.001
    // take 26 us on one CTA, 31 on four (mixed 23 and 29), and at 0.005 44 and 45 (36 and
    // 40). Half as many CTAs as layers of fragments: a phase takes every other layer (48^3
    // cells at 0.02 take the same on four CTAs as on eight); four at least (64 x 64 x 16
    // cells in 16 x 16 x 4 fragments at 0.001: 38 us on two, 35 on four). All or none: a
    // batch waits for its slowest replica, and with some on clusters the rest have fewer
    // SMs (152 replicas of 32^3 cells at 0.01, 19 on clusters: mixed 52 -> 83, plain 142 ->
    // 203 us).
    if (force == 0 && allowed && b->opts.test_stuck_wait_us == 0) {
        std::vector<int> dense;
        double freed = 0.0;
        for (int c = 0; c < 4; ++c)
            for (int r : cls[c]) {
                const int64_t F = phase_frags(r);
                if (b->desc[r].nf[2] >= 4 && (F >= 128 || (F >= 64 && phase_vacs(r) >= 64.0))) {
                    dense.push_back(r);
                    freed += share[c];
                }
            }
        std::sort(dense.begin(), dense.end(), [&](int a, int q) {
            return b->n_vac[a] != b->n_vac[q] ? b->n_vac[a] > b->n_vac[q] : a < q;
        });
        for (int hi = CLUSTER_MAX_CTAS; hi >= 4 && !dense.empty();) {
            Group g = group(dense, 4, hi, [&](int r) { return std::max(4, b->desc[r].nf[2] / 2); });
            if (g.on.size() < dense.size()) break;
            if (load - freed / sms + g.load > 0.9) {
                hi = g.most - 1;
                continue;
            }
            for (const Placed& p : g.on) put_on_cluster(p);
            for (int c = 0; c < 4; ++c)
                cls[c].erase(std::remove_if(cls[c].begin(), cls[c].end(), [&](int r) { return b->run_kernel[r] == 2; }),
                             cls[c].end());
            load += g.load - freed / sms;
            cluster_load += g.load;
            slowest = std::max(slowest, g.us);
            break;
        }
    }
    // Many replicas on the colour-phase passes, which take the batch as one: where the
    // resident kernels need several waves, or the plain form's first draws (for empty
    // fragments too; 0.125 ns each beside CTAs of one replica, 0.25 ns beside clusters,
    // which leave fewer SMs) longer than the windows they are for.
    // Both sides are estimates; T_pass is fitted to 8 to 1216 replicas of the shapes above.
    // 64 replicas of 96^3 cells in 24^3 fragments at 0.001: plain 1778 us per window on
    // clusters, 450 in passes (mixed 507 and 227); 608 of 48^3: plain 617 and 533 (mixed
    // 156 and 272), 304 of them 307 and 367.
    if (force == 0 && allowed && b->opts.schedule == 0) {
        int64_t frags = 0, res_vac = 0;
        double mean_vac = 0.0;
        for (int r = 0; r < b->n; ++r) {
            if (!b->desc[r].resident) continue;
            const int64_t nf = (int64_t)b->desc[r].nf[0] * b->desc[r].nf[1] * b->desc[r].nf[2];
            frags += nf;
            res_vac += b->n_vac[r];
            mean_vac = std::max(mean_vac, (double)b->n_vac[r] / (double)nf);
        }
        // one CTA each: a replica takes its share of an SM for its window's time
        double work = std::ceil(cluster_load - 1e-9) * slowest;
        for (int c = 0; c < 4; ++c)
            for (int r : cls[c]) {
                const double us = window_us(r, 1, threads[c] / 32);
                work += us * share[c] / sms;
                slowest = std::max(slowest, us);
            }
        const bool beside = cluster_load > 0.0;
        const double draws_us = prec ? 0.0 : (beside ? 0.25e-3 : 0.125e-3) * (double)frags * plain_ev;
        // (mixed replicas on one CTA each are faster there in any number)
        if ((prec ? cluster_load : load) > 1.0 || draws_us > slowest) {
            static const double base[3] = {175.0, 98.0, 205.0}, per_vac[3] = {20.0, 12.0, 20.0},
                                per_frag[3] = {1.6e-4, 0.7e-4, 1.8e-4}, per_v[3] = {7.5e-4, 3.6e-4, 16e-4};
            const double waves_us = std::max(work, slowest);
            const double resident_us = std::max(waves_us, draws_us) + (beside ? 0.4 : 0.7) * std::min(waves_us, draws_us);
            const double passes_us = base[form] + per_vac[form] * mean_vac + per_frag[form] * (double)frags +
                                     per_v[form] * (double)res_vac;
            // (waves of clusters disturb each other more than the estimate has it, with site
            // energies most; a batch that runs at once is the safer choice)
            static const double bias[3] = {1.0, 0.95, 0.9};
            if (passes_us * (load <= 1.0 ? 1.12 : (cluster_load > 1.0 ? bias[form] : 1.02)) < resident_us) {
                for (RepDesc& D : b->desc) D.resident = 0;
                b->run_kernel.assign(b->n, 0);
                b->run_ctas.assign(b->n, 0);
                plans.clear();
                for (int c = 0; c < 4; ++c) cls[c].clear();
            }
        }
    }
    // a dense replica alone on the colour-phase passes, which spread over every SM:
    // 128^3 cells in 32^3 fragments at 0.02 (61 vacancies per warp and phase) take 498 us
    // per window on 16 CTAs and 344 in passes (mixed 350 and 191), 96^3 cells in 24^3
    // fragments at 0.02 (35) 265 and 296 (mixed 203 and 168), 128^3 cells in 32^3 at 0.005
    // (15) 175 and 233 (mixed 113 and 127). With several replicas the clusters fill the
    // SMs that one leaves idle, so the line holds up to a quarter of them.
    if (force == 0 && b->opts.schedule == 0 && sms_used() <= 0.25 * sms) {
        const double line = prec ? 24.0 : 40.0;
        auto to_passes = [&](int r, int ncta) {
            const int busy = std::min(ncta, std::max(1, b->desc[r].nf[2] / 2));
            if (phase_vacs(r) <= line * busy * (CLUSTER_THREADS / 32)) return false;
            b->desc[r].resident = 0;
            b->run_kernel[r] = b->run_ctas[r] = 0;
            return true;
        };
        for (int c = 0; c < 4; ++c)
            cls[c].erase(std::remove_if(cls[c].begin(), cls[c].end(), [&](int r) { return to_passes(r, 1); }),
                         cls[c].end());
        plans.erase(std::remove_if(plans.begin(), plans.end(),
                                   [&](const ClusterPlan& pl) { return to_passes(pl.rep, pl.ncta); }),
                    plans.end());
    }
    // largest replicas (by vacancies, the work per phase) first in every class: the
    // longest-running CTAs start earliest, which shortens the tail of the launch
    for (int c = 0; c < 4; ++c)
        std::sort(cls[c].begin(), cls[c].end(), [&](int a, int q) {
            return b->n_vac[a] != b->n_vac[q] ? b->n_vac[a] > b->n_vac[q] : a < q;
        });
    // the largest of the last class on two CTAs each (kmc_opts.cluster_top)
    for (int k = 0; prec == 1 && k < std::min<int>((int)cls[3].size(), b->cluster_top);) {
        const int r = cls[3][k];
        ClusterPlan pl{};
        if (!make_cluster_plan(b->desc[r], b->cap, 4, prec, 2, 2, &pl) ||
            cluster_fits(form, 2, cluster_smem_bytes(b->desc[r], pl, b->cap, 4, prec)) <= 0) {
            ++k;
            continue;
        }
        pl.rep = r;
        plans.push_back(pl);
        b->desc[r].pre_ev = 4;
        b->run_ctas[r] = 2;
        pairs.push_back(r);
        if ((int)pairs.size() >= b->cluster_top) break;
        ++k;
    }
    for (int r : pairs) cls[3].erase(std::find(cls[3].begin(), cls[3].end(), r));
    // more warps for the replicas with the most vacancies while every CTA still has
    // its share of an SM: a phase takes as long as its slowest visit, so a visit
    // should not wait for a warp.  First to 256 threads, then to 512, and where not all
    // can have them, only those with a quarter more vacancies than the largest left
    // behind, for which the batch would wait all the same: 300 replicas of 24^3 cells
    // took 40 us per window (mixed) with 100 of them on 512 threads, and 22 with none.
    // The plain form leaves half the SMs to k_draws (100 of 32^3: 73 -> 60 us).
    const double most_sms = (prec ? 1.0 : 0.5) * sms;
    for (int to = 2; to <= 3; ++to) {
        std::vector<std::pair<int64_t, int>> want;  // (vacancies, replica)
        for (int c = to - 2; c < to; ++c)
            for (int r : cls[c]) {
                const int warps = threads[c] / 32;  // one visit per warp, at most phase_frags of them
                if ((to == 2 || c == 2) && phase_frags(r) > warps && b->n_vac[r] > 4 * warps) want.push_back({b->n_vac[r], r});
            }
        std::sort(want.rbegin(), want.rend());
        std::vector<int> class_of(b->n, 0), moved(b->n, 0);
        for (int c = 0; c < 4; ++c)
            for (int r : cls[c]) class_of[r] = c;
        double used = sms_used();
        size_t k = 0;
        for (; k < want.size(); ++k) {
            const double more = share[to] - share[class_of[want[k].second]];
            if (used + more > most_sms) break;
            used += more;
        }
        if (k < want.size()) {
            const double left = 1.25 * (double)want[k].first;
            while (k > 0 && (double)want[k - 1].first < left) --k;
        }
        for (size_t i = 0; i < k; ++i) {
            const int r = want[i].second;
            const RepDesc& D = b->desc[r];
            const size_t nd = resident_smem_bytes(D, b->cap, threads[to], D.pre_g, D.pre_ev, prec);
            if (nd > bounds[to]) continue;
            moved[r] = 1;
            cls[to].push_back(r);
            need_of[r] = nd;
        }
        for (int c = to - 2; c < to; ++c)
            cls[c].erase(std::remove_if(cls[c].begin(), cls[c].end(), [&](int r) { return moved[r] != 0; }), cls[c].end());
    }
    for (int c = 0; c < 4; ++c)
        std::sort(cls[c].begin(), cls[c].end(), [&](int a, int q) {
            return b->n_vac[a] != b->n_vac[q] ? b->n_vac[a] > b->n_vac[q] : a < q;
        });
    for (int c = 0; c < 4; ++c)
        for (int r : cls[c]) cmax[c] = std::max(cmax[c], need_of[r]);
    b->any_global = std::any_of(b->desc.begin(), b->desc.end(), [](const RepDesc& D) { return !D.resident; });
    if (b->opts.schedule == 2 && b->any_global)
        return fail(FKMC_EINVAL, "schedule 2 needs every replica to fit the resident kernel (mixed form)");
    std::vector<int32_t> order;
    for (int c = 0; c < 4; ++c) {
        if (cls[c].empty()) continue;
        kmc_batch::RClass rc{(int)order.size(), (int)cls[c].size(), cmax[c], threads[c], 1, nullptr, nullptr, false, false};
        for (int r : cls[c]) {
            order.push_back(r);
            rc.long_lists = rc.long_lists || b->desc[r].kslots == 16;
        }
        CK(cudaStreamCreateWithFlags(&rc.st, cudaStreamNonBlocking), "stream");
        CK(cudaEventCreateWithFlags(&rc.done, cudaEventDisableTiming), "event");
        b->rclass.push_back(rc);
    }
    if (!order.empty())
        CK(cudaMemcpyAsync(b->d_reps, order.data(), sizeof(int32_t) * order.size(), cudaMemcpyHostToDevice,
                           b->st),
           "replica list upload");
    // replicas on clusters: one launch per CTA count (a launch has one cluster shape)
    std::stable_sort(plans.begin(), plans.end(),
                     [](const ClusterPlan& x, const ClusterPlan& y) { return x.ncta < y.ncta; });
    for (size_t k = 0; k < plans.size();) {
        size_t e = k, smem = 0;
        while (e < plans.size() && plans[e].ncta == plans[k].ncta) {
            const RepDesc& D = b->desc[plans[e].rep];
            smem = std::max(smem, cluster_smem_bytes(D, plans[e], b->cap, D.pre_ev, prec));
            ++e;
        }
        kmc_batch::RClass rc{(int)k, (int)(e - k), smem, CLUSTER_THREADS, plans[k].ncta, nullptr, nullptr, true, false};
        for (size_t i = k; i < e; ++i) rc.long_lists = rc.long_lists || b->desc[plans[i].rep].kslots == 16;
        CK(cudaStreamCreateWithFlags(&rc.st, cudaStreamNonBlocking), "stream");
        CK(cudaEventCreateWithFlags(&rc.done, cudaEventDisableTiming), "event");
        b->rclass.push_back(rc);  // launched last-first: a cluster takes its SMs before single CTAs spread out
        k = e;
    }
    if (!plans.empty())
        CK(cudaMemcpyAsync(b->d_plans, plans.data(), sizeof(ClusterPlan) * plans.size(), cudaMemcpyHostToDevice,
                           b->st),
           "cluster plan upload");
    if (!resident_buffers(b, prec, plain_ev)) {
        if (b->opts.schedule == 2) return fail(FKMC_ENOMEM, "device allocation failed (resident replicas)");
        plan_passes(b);
    }
    return FKMC_OK;
}

// ---------------------------------------------------------------- site energies
// Partners of a site by displacement: a vector d (units a/2) from a site at p0
// lands on an O site when exactly one coordinate of p0 + d is odd (that axis is
// the O site's type), on a B site (cell corner) when all are even.
struct Landing { int kind; int t2; int dc[3]; };  // kind 0: O site, 1: B site, -1: neither

Landing land(const int p0[3], const int d[3])
{
    Landing L{-1, -1, {0, 0, 0}};
    int p[3], odd = 0, axis = -1;
    for (int k = 0; k < 3; ++k) {
        p[k] = p0[k] + d[k];
        if (p[k] & 1) { ++odd; axis = k; }
    }
    if (odd == 1) {
        L.kind = 0;
        L.t2 = axis;
        for (int k = 0; k < 3; ++k) L.dc[k] = (p[k] - (k == axis)) / 2;
    } else if (odd == 0) {
        L.kind = 1;
        for (int k = 0; k < 3; ++k) L.dc[k] = p[k] / 2;
    }
    return L;
}

int32_t energy_units(double eV) { return (int32_t)std::llrint(eV * 1e4); }

// Partner tables of a shell set: V-V partners of each O site type, the O
// sites around a B site (dopant scatter), the B sites around each O site type,
// the reaches in cells, the bound on |E_site| and the a/sqrt2 shell energy.
struct ShellTables {
    std::vector<SiteOff> vv = std::vector<SiteOff>((size_t)3 * SITE_MAX_VV);
    int nvv = 0;
    std::vector<SiteOff> bo;
    std::vector<SiteOff> ob[3];
    int reach_vv = 0, reach_all = 0;
    int64_t bound = 0;
    int32_t e_self = 0;
};

int make_shells(const kmc_site_energy* e, ShellTables* out)
{
    if (e->n_vv < 0 || e->n_vv > FKMC_MAX_SHELLS || e->n_fe < 0 || e->n_fe > FKMC_MAX_SHELLS)
        return fail(FKMC_EINVAL, "0 to 8 shells of each kind");
    const int ns = e->n_vv + e->n_fe;
    auto d2_of = [&](int k) { return k < e->n_vv ? e->vv_d2[k] : e->fe_d2[k - e->n_vv]; };
    auto en_of = [&](int k) { return k < e->n_vv ? e->vv_eV[k] : e->fe_eV[k - e->n_vv]; };
    for (int k = 0; k < ns; ++k) {
        if (d2_of(k) < 1 || d2_of(k) > 36 || !std::isfinite(en_of(k)) || std::fabs(en_of(k)) > 10.0)
            return fail(FKMC_EINVAL, "shell squared distances must be in [1, 36], energies finite within 10 eV");
        for (int q = 0; q < k; ++q)
            if ((q < e->n_vv) == (k < e->n_vv) && d2_of(q) == d2_of(k))
                return fail(FKMC_EINVAL, "a shell is listed twice");
    }
    ShellTables& sh = *out;
    int nvv[3] = {0, 0, 0};
    std::vector<int> hit(ns, 0);
    // centre = an O site of type t (t = 0..2) or a B site (t = 3); |d| <= 6
    // half-units per axis covers every squared distance up to 36
    for (int t = 0; t < 4; ++t) {
        const int p0[3] = {t == 0, t == 1, t == 2};
        int64_t sum = 0;
        for (int dz = -6; dz <= 6; ++dz)
            for (int dy = -6; dy <= 6; ++dy)
                for (int dx = -6; dx <= 6; ++dx) {
                    const int d[3] = {dx, dy, dz};
                    const int d2 = dx * dx + dy * dy + dz * dz;
                    const Landing L = land(p0, d);
                    if (L.kind < 0) continue;
                    // O centre: O partners in V-V shells, B partners in dopant shells;
                    // B centre: O partners in dopant shells
                    const bool want_vv = t < 3 && L.kind == 0;
                    if (!want_vv && (L.kind == 0) == (t < 3)) continue;
                    for (int k = want_vv ? 0 : e->n_vv; k < (want_vv ? e->n_vv : ns); ++k) {
                        if (d2_of(k) != d2) continue;
                        hit[k] = 1;
                        SiteOff o;
                        o.t2 = (int8_t)(L.kind == 0 ? L.t2 : -1);
                        for (int a = 0; a < 3; ++a) o.dc[a] = (int8_t)L.dc[a];
                        o.e = energy_units(en_of(k));
                        int reach = 0;
                        for (int a = 0; a < 3; ++a) reach = std::max(reach, std::abs(L.dc[a]));
                        sh.reach_all = std::max(sh.reach_all, reach);
                        if (t == 3) {
                            if ((int)sh.bo.size() == SITE_MAX_BO) return fail(FKMC_EINVAL, "too many dopant partners");
                            sh.bo.push_back(o);
                            continue;
                        }
                        sum += o.e < 0 ? -(int64_t)o.e : o.e;
                        if (want_vv) {
                            sh.reach_vv = std::max(sh.reach_vv, reach);
                            if (nvv[t] == SITE_MAX_VV) return fail(FKMC_EINVAL, "too many V-V partners per site");
                            sh.vv[(size_t)t * SITE_MAX_VV + nvv[t]++] = o;
                        } else {
                            sh.ob[t].push_back(o);
                        }
                    }
                }
        if (t < 3) sh.bound = std::max(sh.bound, sum);
    }
    for (int k = 0; k < ns; ++k)
        if (!hit[k]) return fail(FKMC_EINVAL, "a squared distance is not a shell of this lattice");
    sh.nvv = nvv[0];
    for (int k = 0; k < e->n_vv; ++k)
        if (e->vv_d2[k] == 2) sh.e_self = energy_units(e->vv_eV[k]);
    return FKMC_OK;
}

// bound on |E_site| over every site: shells plus the electrostatic term
int64_t energy_bound(const kmc_batch* b)
{
    int64_t g = 0;
    for (int32_t v : b->elec_g) g = std::max<int64_t>(g, v < 0 ? -(int64_t)v : v);
    return b->e_bound + (b->elec_on ? b->elec_umax + g : 0);
}

// Boltzmann tables of every replica: lo[m0] = exp(-m0 c), hi[i] = exp(-512 (i - mid) c),
// c = 1e-4 / (2 kB T); |m| <= 2 e_bound, so m >> 9 stays within [-mid, mid].
int build_btab(kmc_batch* b)
{
    const int mid = (int)((2 * energy_bound(b) + 511) / 512) + 1;
    const int len = 2 * mid + 1;
    const size_t per = (size_t)BOLTZ_LO + len;
    std::vector<double> h(per * b->n);
    for (int r = 0; r < b->n; ++r) {
        const double c = 1e-4 / (2.0 * (KB_EV * b->T[r]));
        double* lo = h.data() + per * r;
        for (int m0 = 0; m0 < BOLTZ_LO; ++m0) lo[m0] = std::exp(-((double)m0 * c));
        for (int i = 0; i < len; ++i) lo[BOLTZ_LO + i] = std::exp(-((double)(512 * (int64_t)(i - mid)) * c));
        b->desc[r].btab_off = (int64_t)(per * r);
        b->desc[r].bhi_mid = mid;
        b->desc[r].bhi_len = len;
    }
    const size_t bytes = sizeof(double) * h.size();
    if (bytes > b->btab_bytes) {
        b->dfree(b->btab);
        b->btab = (double*)b->dalloc(bytes);
        b->btab_bytes = b->btab ? bytes : 0;
        if (!b->btab) return fail(FKMC_ENOMEM, "device allocation failed (Boltzmann tables)");
    }
    CK(cudaMemcpyAsync(b->btab, h.data(), bytes, cudaMemcpyHostToDevice, b->st), "table upload");
    CK(cudaStreamSynchronize(b->st), "synchronize");
    return FKMC_OK;
}

SiteArgs site_args(const kmc_batch* b)
{
    SiteArgs a{};
    a.vv = b->d_vv;
    a.btab = b->btab;
    a.field = b->field;
    a.n_vv = b->n_vv;
    a.e_self = b->e_self;
    a.reach = b->n_vv > 0 ? b->reach_vv + 1 : 0;
    a.gbound = b->grains_on ? b->gbound : nullptr;
    a.g_elec = b->elec_on ? b->d_elec_g : nullptr;
    return a;
}

// Rate tables of boundary hops: barriers raised by the grains' barrier, the
// mixed form quantised against the bulk table's k32max (same F).
int grain_tables(kmc_batch* b, int r)
{
    RepDesc& D = b->desc[r];
    if (!b->grains_on) {
        for (int i = 0; i < 6; ++i) {
            D.k64g[i] = D.k64[i];
            D.qg[i] = D.q[i];
        }
        return FKMC_OK;
    }
    kmc_barrier_table t = b->tables[r];
    t.Ea_O_eV += b->grains.barrier_eV;
    t.Ea_H_eV += b->grains.barrier_eV;
    float k32g[6], kmax = 0.0f;
    uint64_t qtmp[6];
    int32_t F;
    int rc = rate_table_impl(&t, b->T[r], b->Ez[r], b->a_ang[r], b->cap, D.k64g, k32g, qtmp, &F);
    if (rc) return rc;
    for (int i = 0; i < 6; ++i) kmax = std::max(kmax, (float)D.k64[i]);
    for (int i = 0; i < 6; ++i) D.qg[i] = (uint64_t)std::llrint(std::ldexp((double)k32g[i] / (double)kmax, D.F));
    return FKMC_OK;
}

int rebuild_field(kmc_batch* b)
{
    const SiteArgs a = site_args(b);
    CK(launch_site_field(b->d_desc, b->n, b->recs, b->counts, b->nfrag_total, b->cap, b->nsite_total, b->fe, b->d_bo,
                         b->n_bo, a, b->st),
       "energy field");
    if (b->elec_on) CK(elec_add(b->field, b->elec_u, b->nsite_total, b->st), "energy field");
    b->field_valid = true;
    return FKMC_OK;
}

void drop_window_graph(kmc_batch* b);

// What a change of rates, options or composition needs before the next run: the
// Boltzmann tables (`tables`, where site energies are on), the plan that their size
// enters, and the descriptors.  On an error nothing runs until kmc_set_barriers
// succeeds: the plan, the buffers and the device's descriptors need not agree.
int apply_rates(kmc_batch* b, bool tables)
{
    b->rates_set = false;
    const double* before = b->btab;
    int rc = tables && site_path(b) ? build_btab(b) : FKMC_OK;
    if (b->btab != before) drop_window_graph(b);  // it holds the old tables
    if (!rc) rc = plan_residency(b);
    if (!rc) rc = upload_desc(b);
    if (rc) {
        drop_classes(b);
        return rc;
    }
    b->rates_set = true;
    return FKMC_OK;
}

// the Boltzmann tables must cover electrostatic energies up to |u| = um
int elec_cover(kmc_batch* b, int64_t um)
{
    if (um <= b->elec_umax) return FKMC_OK;
    b->elec_umax = 2 * um + 1024;
    if (!b->rates_set) return FKMC_OK;  // kmc_set_barriers builds the tables
    return apply_rates(b, true);
}

// V-cycles of the next automatic refresh
static int refresh_cycles(const kmc_batch* b)
{
    return b->phi_prev_valid && b->elec.warm_cycles > 0 ? b->elec.warm_cycles : b->elec.cycles;
}

// kernels of one refresh: per replica the solve (deposit, right-hand side,
// V-cycles, mean) and the update
uint64_t elec_launches(const kmc_batch* b)
{
    uint64_t k = 0;
    for (int r = 0; r < b->n; ++r) {
        const MgPlan p = mg_plan(b->desc[r].L[0], b->desc[r].L[1], b->desc[r].L[2]);
        k += 2 + (uint64_t)refresh_cycles(b) * mg_cycle_kernels(p) + 3 + 1;
    }
    return k;
}

// Potential of every replica's vacancy charges (multigrid), then u and the
// energy field moved to it; the Boltzmann tables grow if the bound does.
int elec_refresh(kmc_batch* b)
{
    CK(cudaMemsetAsync(b->d_umax, 0, sizeof(unsigned), b->st), "memset");
    const int cycles = refresh_cycles(b);
    const bool warm = b->phi_prev_valid, with_field = b->field_valid;
    if (!b->cap_st) CK(cudaStreamCreateWithFlags(&b->cap_st, cudaStreamNonBlocking), "stream");
    for (int r = 0; r < b->n; ++r) {
        // each replica's solve is one graph (some 40 launches per V-cycle); every
        // argument is fixed until the window graph is dropped, which drops these too
        cudaGraphExec_t exec = nullptr;
        for (auto& g : b->elec_graphs)
            if (g.r == r && g.cycles == cycles && g.warm == warm && g.field == with_field) exec = g.exec;
        if (!exec) {
            const RepDesc& D = b->desc[r];
            const MgPlan p = mg_plan(D.L[0], D.L[1], D.L[2]);
            const double scale = 1.602176634e-19 / (8.8541878128e-12 * b->elec.eps_r * b->a_ang[r] * 1e-10);
            double* prev = b->phi_prev + D.site_off / 3;
            cudaGraph_t graph = nullptr;
            CK(cudaStreamBeginCapture(b->cap_st, cudaStreamCaptureModeThreadLocal), "graph capture");
            cudaError_t le = elec_solve(D, b->recs, b->counts, b->cap, b->n_vac[r], b->elec.q_vac, scale, cycles, p,
                                        b->mgb, nullptr, warm ? prev : nullptr, prev, b->cap_st);
            if (le == cudaSuccess)
                le = elec_update(D, b->mgb.phi, b->elec.q_vac, b->elec_u, with_field ? b->field : nullptr, b->d_umax,
                                 b->cap_st);
            cudaError_t ce = cudaStreamEndCapture(b->cap_st, &graph);
            if (le != cudaSuccess) return cuda_fail(le, "potential solve capture");
            if (ce != cudaSuccess) return cuda_fail(ce, "potential solve capture");
            cudaError_t ie = cudaGraphInstantiate(&exec, graph, 0);
            cudaGraphDestroy(graph);
            if (ie != cudaSuccess) return cuda_fail(ie, "graph instantiate");
            b->elec_graphs.push_back({r, cycles, warm, with_field, exec});
        }
        CK(cudaGraphLaunch(exec, b->st), "graph launch");
    }
    unsigned um = 0;
    CK(cudaMemcpyAsync(&um, b->d_umax, sizeof um, cudaMemcpyDeviceToHost, b->st), "copy");
    CK(cudaStreamSynchronize(b->st), "synchronize");
    b->elec_age = 0;
    b->phi_prev_valid = true;
    return elec_cover(b, (int64_t)um);
}

// simulated time of the null-event form of replica r (s): its clock counts in 1/k32max
double null_time(const kmc_batch* b, int r)
{
    float kmax = 0.0f;
    for (int i = 0; i < 6; ++i) kmax = std::max(kmax, (float)b->desc[r].k64[i]);
    return kmax > 0.0f ? b->theta_host[r] / (double)kmax : 0.0;
}

void drop_window_graph(kmc_batch* b)
{
    if (b->window_exec) cudaGraphExecDestroy(b->window_exec);
    b->window_exec = nullptr;
    for (auto& g : b->elec_graphs) cudaGraphExecDestroy(g.exec);
    b->elec_graphs.clear();
}

}  // namespace

extern "C" {

const char* kmc_last_error(void) { return g_err.c_str(); }

void kmc_default_opts(kmc_opts* o)
{
    if (!o) return;
    std::memset(o, 0, sizeof *o);
    o->edge = 4;
    o->precision = FKMC_PLAIN;
    o->n_tau = 1.0;
    o->cluster_top = -1;
}

int32_t kmc_partition_count(int32_t L, int32_t edge)
{
    if (L < 1 || edge < 1) return 0;
    return partition_count(L, edge);
}

void kmc_neighbour_table(int32_t out[168])
{
    NbEntry tab[3][8];
    build_nb_table(tab);
    for (int t = 0; t < 3; ++t)
        for (int n = 0; n < 8; ++n) {
            int32_t* o = out + (t * 8 + n) * 7;
            o[0] = tab[t][n].t2;
            for (int k = 0; k < 3; ++k) {
                o[1 + k] = tab[t][n].dc[k];
                o[4 + k] = tab[t][n].d[k];
            }
        }
}

int kmc_rate_table(const kmc_barrier_table* t, double T_K, double field_z_Vpm, double a_angstrom,
                   int32_t cap_v, double k64[6], float k32[6], uint64_t q[6], int32_t* F)
{
    if (!k64 || !k32 || !q || !F) return fail(FKMC_EINVAL, "null output");
    return rate_table_impl(t, T_K, field_z_Vpm, a_angstrom, cap_v, k64, k32, q, F);
}

int kmc_create_batch(int32_t n, const kmc_cells* cells, const kmc_composition* comp, uint64_t seed,
                     const kmc_opts* opts_in, kmc_batch** out)
{
    if (!out) return fail(FKMC_EINVAL, "out is NULL");
    *out = nullptr;
    if (n < 1 || !cells || !comp) return fail(FKMC_EINVAL, "need n >= 1 replicas with cells and composition");
    kmc_opts o;
    kmc_default_opts(&o);
    if (opts_in) o = *opts_in;
    if (o.edge <= 0) o.edge = 4;
    if (!(o.n_tau > 0.0) || !(o.n_tau <= 64.0)) return fail(FKMC_EINVAL, "n_tau must be in (0, 64]");
    if (o.precision != FKMC_PLAIN && o.precision != FKMC_MIXED) return fail(FKMC_EINVAL, "bad precision");
    if (o.cap_v != 0 && (o.cap_v < 8 || o.cap_v > 256 || o.cap_v % 8))
        return fail(FKMC_EINVAL, "cap_v must be 0 or a multiple of 8 in [8, 256]");
    if (o.schedule < 0 || o.schedule > 2) return fail(FKMC_EINVAL, "schedule must be 0, 1 or 2");
    if (o.small_pass < -1 || o.small_pass > 2) return fail(FKMC_EINVAL, "small_pass must be -1, 0, 1 or 2");
    if (o.lane_form < 0 || o.lane_form > 2) return fail(FKMC_EINVAL, "lane_form must be 0, 1 or 2");
    if (o.cluster_ctas < -1 || o.cluster_ctas == 1 || o.cluster_ctas > CLUSTER_MAX_CTAS)
        return fail(FKMC_EINVAL, "cluster_ctas must be -1, 0 or 2..16");
    if (o.test_stuck_wait_us < 0 || o.test_stuck_wait_us > 2000000)
        return fail(FKMC_EINVAL, "test_stuck_wait_us must be in [0, 2e6]");

    kmc_batch* b = new kmc_batch();
    b->n = n;
    b->opts = o;
    b->st = (cudaStream_t)o.stream;
    b->desc.resize(n);
    b->n_vac.resize(n);
    b->n_H.resize(n);
    b->n_fe.assign(n, 0);
    b->T.assign(n, 0.0);
    b->theta_host.assign(n, 0.0);
    b->b_bits.resize(n);
    b->a_ang.resize(n);
    b->stats_host.assign(2 * (size_t)n, 0ull);
    double worst_mean = 0.0;
    for (int r = 0; r < n; ++r) {
        const kmc_cells& c = cells[r];
        const int L[3] = {c.nx, c.ny, c.nz};
        RepDesc& D = b->desc[r];
        std::memset(&D, 0, sizeof D);
        for (int d = 0; d < 3; ++d) {
            if (L[d] < 1 || L[d] > 65535) {
                delete b;
                return fail(FKMC_EINVAL, "cells per dimension must be in [1, 65535]");
            }
            D.L[d] = L[d];
            D.nf[d] = o.nfrag[d] > 0 ? o.nfrag[d] : partition_count(L[d], o.edge);
            if (!partition_ok(L[d], D.nf[d])) {
                delete b;
                return fail(FKMC_EINVAL, "fragments per dimension must be 1, or even with every edge >= 2");
            }
            D.base[d] = L[d] / D.nf[d];
            D.rem[d] = L[d] % D.nf[d];
        }
        if (!(c.a_angstrom > 0.0)) {
            delete b;
            return fail(FKMC_EINVAL, "lattice constant must be > 0");
        }
        D.nsite = 3 * (int64_t)L[0] * L[1] * L[2];
        if (comp[r].n_vac < 0 || comp[r].n_H < 0 || comp[r].n_vac + comp[r].n_H > D.nsite ||
            comp[r].n_vac > 0xffffffffll) {
            delete b;
            return fail(FKMC_EINVAL, "composition does not fit the lattice");
        }
        if (comp[r].n_Fe < 0 || comp[r].n_Fe > (int64_t)L[0] * L[1] * L[2]) {
            delete b;
            return fail(FKMC_EINVAL, "dopant count must be in [0, nx ny nz]");
        }
        b->n_vac[r] = comp[r].n_vac;
        b->n_H[r] = comp[r].n_H;
        b->n_fe[r] = comp[r].n_Fe;
        b->a_ang[r] = c.a_angstrom;
        D.replica = (uint32_t)r;
        D.seed = seed;
        D.row_words = (int32_t)(((L[0] + 63) / 64) * 4);  // 16 sites per word, rows padded to 16 bytes
        D.items = ((D.nf[0] + 1) / 2) * ((D.nf[1] + 1) / 2) * ((D.nf[2] + 1) / 2);
        D.items_off = b->total_items;
        b->total_items += D.items;
        const int64_t nfrag = (int64_t)D.nf[0] * D.nf[1] * D.nf[2];
        D.frag_base = b->nfrag_total;
        b->nfrag_total += nfrag;
        D.occ_word_off = b->occ_words;
        b->occ_words += 3 * (int64_t)L[2] * L[1] * D.row_words;
        D.site_off = b->nsite_total;
        b->nsite_total += D.nsite;
        int bb = 1;
        while (((int64_t)1 << (2 * bb)) < D.nsite) ++bb;
        b->b_bits[r] = bb;
        worst_mean = std::max(worst_mean, (double)comp[r].n_vac / (double)nfrag);
    }
    if (o.cap_v == 0) {
        int cap = (int)std::ceil(worst_mean + 10.0 * std::sqrt(worst_mean + 1.0) + 8.0);
        cap = ((cap + 7) / 8) * 8;
        b->cap = std::min(256, std::max(8, cap));
    } else {
        b->cap = o.cap_v;
    }
    b->opts.cap_v = b->cap;
    if (o.cluster_top >= 0) {
        b->cluster_top = o.cluster_top;
    } else {  // auto: the largest replicas take an extra SM each, about one SM in eight
        int dev = 0, sms = 0;
        if (cudaGetDevice(&dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess)
            b->cluster_top = sms / 8;
        else
            b->cluster_top = 0;
    }

    b->occ = (uint32_t*)b->dalloc(sizeof(uint32_t) * b->occ_words);
    b->recs = (VacRec*)b->dalloc(sizeof(VacRec) * b->nfrag_total * b->cap);
    b->counts = (int32_t*)b->dalloc(sizeof(int32_t) * b->nfrag_total);
    if (o.tracer) b->tracer = (int32_t*)b->dalloc(sizeof(int32_t) * 3 * b->nsite_total);
    b->d_desc = (RepDesc*)b->dalloc(sizeof(RepDesc) * n);
    b->stats = (unsigned long long*)b->dalloc(sizeof(unsigned long long) * 2 * n);
    b->status = (uint32_t*)b->dalloc(sizeof(uint32_t));
    b->scratch = (unsigned long long*)b->dalloc(sizeof(unsigned long long) * 8);
    b->scratch_all = (unsigned long long*)b->dalloc(sizeof(unsigned long long) * 7 * n);
    b->d_reps = (int32_t*)b->dalloc(sizeof(int32_t) * n);
    b->d_plans = (ClusterPlan*)b->dalloc(sizeof(ClusterPlan) * n);
    b->rcache.lim = (uint64_t*)b->dalloc(sizeof(uint64_t) * std::max<int64_t>(b->nfrag_total, 1));
    b->rcache.valid = (uint8_t*)b->dalloc((size_t)n);
    b->wctl = (unsigned long long*)b->dalloc(sizeof(unsigned long long) * 2);
    b->perms = (uint32_t*)b->dalloc(sizeof(uint32_t) * n);
    b->act = (ActEntry*)b->dalloc(sizeof(ActEntry) * 3 * std::max<int64_t>(b->total_items, 1));
    b->act_count = (int32_t*)b->dalloc(sizeof(int32_t) * ACT_COUNTERS);
    b->cls = (uint8_t*)b->dalloc((size_t)std::max<int64_t>(b->total_items, 1));
    b->ncell_total = b->nsite_total / 3;
    bool any_fe = false;
    for (int r = 0; r < n; ++r) any_fe = any_fe || b->n_fe[r] > 0;
    if (any_fe) {
        b->fe = (uint8_t*)b->dalloc((size_t)b->ncell_total);
        if (!b->fe) {
            b->release();
            delete b;
            return fail(FKMC_ENOMEM, "device allocation failed");
        }
    }
    if (!b->occ || !b->recs || !b->counts || (o.tracer && !b->tracer) || !b->d_desc || !b->stats ||
        !b->status || !b->scratch || !b->scratch_all || !b->d_reps || !b->d_plans || !b->rcache.lim ||
        !b->rcache.valid || !b->wctl ||
        !b->perms ||
        !b->act || !b->act_count || !b->cls) {
        b->release();
        delete b;
        return fail(FKMC_ENOMEM, "device allocation failed");
    }
    int rc = FKMC_OK;
    auto step = [&](cudaError_t e, const char* what) {
        if (rc == FKMC_OK && e != cudaSuccess) rc = cuda_fail(e, what);
    };
    build_nb_table(b->nbt.e);
    step(upload_neighbours(&b->nbt.e[0][0]), "neighbour table upload");
    step(null_upload_neighbours(&b->nbt.e[0][0]), "neighbour table upload");
    step(phase_prepare(b->cap), "kernel attributes");
    step(run_pass_blocks(b->opts.precision, b->cap, false, false, &b->run_blocks), "occupancy query");
    step(resident_prepare(), "kernel attributes");
    step(cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming), "event");
    step(cudaEventCreate(&b->ev0), "event");
    step(cudaEventCreate(&b->ev1), "event");
    step(cudaMemsetAsync(b->occ, 0, sizeof(uint32_t) * b->occ_words, b->st), "memset");
    step(cudaMemsetAsync(b->counts, 0, sizeof(int32_t) * b->nfrag_total, b->st), "memset");
    if (o.tracer) step(cudaMemsetAsync(b->tracer, 0, sizeof(int32_t) * 3 * b->nsite_total, b->st), "memset");
    step(cudaMemsetAsync(b->stats, 0, sizeof(unsigned long long) * 2 * n, b->st), "memset");
    step(cudaMemsetAsync(b->rcache.valid, 0, (size_t)n, b->st), "memset");
    step(cudaMemsetAsync(b->status, 0, sizeof(uint32_t), b->st), "memset");
    for (int r = 0; r < n && rc == FKMC_OK; ++r)
        step(launch_init(b->desc[r], b->b_bits[r], b->n_vac[r], b->n_vac[r] + b->n_H[r], b->occ, b->recs,
                         b->counts, b->cap, b->status, b->st),
             "init kernel");
    if (b->fe) {
        step(cudaMemsetAsync(b->fe, 0, (size_t)b->ncell_total, b->st), "memset");
        for (int r = 0; r < n && rc == FKMC_OK; ++r) {
            int bb = 1;
            while (((int64_t)1 << (2 * bb)) < b->desc[r].nsite / 3) ++bb;
            step(launch_init_dopants(b->desc[r], bb, b->n_fe[r], b->fe, b->st), "dopant kernel");
        }
    }
    if (rc == FKMC_OK) rc = upload_desc(b);
    if (rc == FKMC_OK) rc = check_status(b);
    if (rc != FKMC_OK) {
        std::string keep = g_err;
        b->release();
        delete b;
        g_err = keep;
        return rc;
    }
    *out = b;
    return FKMC_OK;
}

int kmc_create_lattice(const kmc_cells* cells, const kmc_composition* comp, uint64_t seed,
                       const kmc_opts* opts, kmc_batch** out)
{
    return kmc_create_batch(1, cells, comp, seed, opts, out);
}

int kmc_set_barriers(kmc_batch* b, const kmc_barrier_table* tables, const double* T_K,
                     const double* field_z_Vpm)
{
    if (!b || !tables || !T_K) return fail(FKMC_EINVAL, "null argument");
    std::vector<RepDesc> nd = b->desc;
    for (int r = 0; r < b->n; ++r) {
        RepDesc& D = nd[r];
        float k32[6];
        int32_t F;
        const double Ez = field_z_Vpm ? field_z_Vpm[r] : 0.0;
        int rc = rate_table_impl(&tables[r], T_K[r], Ez, b->a_ang[r], b->cap, D.k64, k32, D.q, &F);
        if (rc) return rc;
        double kmax = 0.0;
        float kmax32 = 0.0f;
        for (int i = 0; i < 6; ++i) {
            if ((i < 3 || b->n_H[r] > 0) && D.k64[i] > kmax) kmax = D.k64[i];
            kmax32 = std::max(kmax32, k32[i]);
        }
        D.F = F;
        D.tau = b->opts.n_tau / (8.0 * kmax);
        D.theta_tau = D.tau * (double)kmax32;
    }
    b->desc = nd;
    b->tables.assign(tables, tables + b->n);
    b->Ez.assign(b->n, 0.0);
    for (int r = 0; r < b->n; ++r) {
        b->T[r] = T_K[r];
        b->Ez[r] = field_z_Vpm ? field_z_Vpm[r] : 0.0;
    }
    int rc = FKMC_OK;
    for (int r = 0; r < b->n && rc == FKMC_OK; ++r) rc = grain_tables(b, r);
    if (rc) return rc;
    return apply_rates(b, true);
}

}  // extern "C"

namespace {

ResidentArgs resident_args(const kmc_batch* b)
{
    ResidentArgs a;
    a.descs = b->d_desc;
    a.occ = b->occ;
    a.recs = b->recs;
    a.tmp = b->rec_tmp;
    a.vmap = b->vmap;
    a.counts = b->counts;
    a.tracer = b->tracer;
    a.stats = b->stats;
    a.status = b->status;
    a.cap = b->cap;
    a.nbt = b->nbt;
    a.frag_tot = b->res_frags;
    a.draw_ev = b->res_ev;
    a.sa = site_args(b);
    a.stuck_wait_us = (uint32_t)b->opts.test_stuck_wait_us;
    a.rc = b->rcache;
    return a;
}

// one launch per class on the classes' streams, after `from` and before `to`
// (largest classes first: their CTAs run longest and should take SMs first)
cudaError_t launch_classes(kmc_batch* b, int form, uint64_t w0, uint64_t windows, const Draw* draws, cudaEvent_t from,
                           cudaStream_t to)
{
    const ResidentArgs args = resident_args(b);
    cudaError_t le = cudaSuccess;
    // Each class but the first (the largest CTAs) starts behind an empty kernel, and
    // these form a chain: started together, the classes' CTAs reach the SMs in any
    // order, and a small CTA on every SM keeps the last large ones waiting until it
    // ends (256 uneven replicas, 1024 windows behind another kernel: 69 -> 54.5 ms).
    // The empty kernels are not in the call's launch count.
    for (auto it = b->rclass.rbegin(); it != b->rclass.rend() && le == cudaSuccess; ++it) {
        auto& c = *it;
        const bool first = it == b->rclass.rbegin();
        if (first) le = cudaStreamWaitEvent(c.st, from, 0);
        if (le == cudaSuccess && !first) le = launch_gate(c.st);
        if (le == cudaSuccess && std::next(it) != b->rclass.rend()) {
            if (!first) le = cudaEventRecord(c.done, c.st);
            if (le == cudaSuccess) le = cudaStreamWaitEvent(std::next(it)->st, first ? from : c.done, 0);
        }
        const int f = c.long_lists ? 3 : form;
        if (le == cudaSuccess && c.slabs)
            le = launch_cluster(f, args, b->d_plans + c.start, c.count, c.cluster, c.smem, w0, windows, draws, c.st);
        else if (le == cudaSuccess)
            le = launch_resident(f, args, b->d_reps + c.start, c.count, c.smem, c.threads, w0, windows, draws, c.st);
        if (le == cudaSuccess) le = cudaEventRecord(c.done, c.st);
        if (le == cudaSuccess) le = cudaStreamWaitEvent(to, c.done, 0);
    }
    return le;
}

// The resident replicas' windows (the call's windows [w_first, w_first + windows)) on a stream beside the caller's (res_st, after
// res_fork, ended by res_join).  Mixed form: the class launches captured once
// per window count into a graph (fork, one launch per class, join).  Plain
// form: the first draws of draw_windows windows at a time by k_draws on a
// stream of their own, the next chunk's beside the current chunk's windows
// (two buffers).
int launch_resident_classes(kmc_batch* b, uint64_t w_first, uint64_t windows, uint64_t* launches)
{
    if (!b->cap_st) CK(cudaStreamCreateWithFlags(&b->cap_st, cudaStreamNonBlocking), "stream");
    if (!b->res_st) {
        CK(cudaStreamCreateWithFlags(&b->res_st, cudaStreamNonBlocking), "stream");
        CK(cudaEventCreateWithFlags(&b->res_fork, cudaEventDisableTiming), "event");
        CK(cudaEventCreateWithFlags(&b->res_join, cudaEventDisableTiming), "event");
    }
    if (b->opts.precision == FKMC_MIXED) {
        if (!b->res_exec || b->res_exec_windows != windows) {
            if (b->res_exec) cudaGraphExecDestroy(b->res_exec);
            b->res_exec = nullptr;
            cudaGraph_t graph = nullptr;
            CK(cudaStreamBeginCapture(b->cap_st, cudaStreamCaptureModeThreadLocal), "graph capture");
            cudaError_t le = cudaEventRecord(b->fork, b->cap_st);
            if (le == cudaSuccess) le = launch_classes(b, 1, 0, windows, nullptr, b->fork, b->cap_st);
            cudaError_t ce = cudaStreamEndCapture(b->cap_st, &graph);
            if (le != cudaSuccess) return cuda_fail(le, "resident capture");
            if (ce != cudaSuccess) return cuda_fail(ce, "resident capture");
            cudaError_t ie = cudaGraphInstantiate(&b->res_exec, graph, 0);
            cudaGraphDestroy(graph);
            if (ie != cudaSuccess) {
                b->res_exec = nullptr;
                return cuda_fail(ie, "graph instantiate");
            }
            b->res_exec_windows = windows;
        }
        CK(cudaEventRecord(b->res_fork, b->st), "event record");
        CK(cudaStreamWaitEvent(b->res_st, b->res_fork, 0), "stream wait");
        CK(cudaGraphLaunch(b->res_exec, b->res_st), "graph launch");
        CK(cudaEventRecord(b->res_join, b->res_st), "event record");
        *launches += b->rclass.size();
        return FKMC_OK;
    }
    if (!b->draw_st) {
        CK(cudaStreamCreateWithFlags(&b->draw_st, cudaStreamNonBlocking), "stream");
        for (int k = 0; k < 2; ++k) {
            CK(cudaEventCreateWithFlags(&b->draw_done[k], cudaEventDisableTiming), "event");
            CK(cudaEventCreateWithFlags(&b->draw_free[k], cudaEventDisableTiming), "event");
        }
    }
    CK(cudaEventRecord(b->res_fork, b->st), "event record");
    CK(cudaStreamWaitEvent(b->res_st, b->res_fork, 0), "stream wait");
    CK(cudaStreamWaitEvent(b->draw_st, b->res_fork, 0), "stream wait");
    const uint64_t step = (uint64_t)b->draw_windows;
    uint64_t done = 0;
    const int form = site_path(b) ? 2 : 0;
    for (uint64_t w0 = w_first; w0 < w_first + windows; w0 += step, ++done) {
        const int k = (int)(done & 1);
        const uint64_t nw = std::min(step, w_first + windows - w0);
        Draw* buf = b->draws + (size_t)k * b->res_frags * b->res_ev * step;
        if (done >= 2) CK(cudaStreamWaitEvent(b->draw_st, b->draw_free[k], 0), "stream wait");
        CK(launch_draws(b->d_desc, b->n, b->res_max_frag, w0, (int)nw, b->res_ev, b->res_frags, buf, b->draw_st),
           "draws kernel");
        CK(cudaEventRecord(b->draw_done[k], b->draw_st), "event record");
        CK(cudaStreamWaitEvent(b->res_st, b->draw_done[k], 0), "stream wait");
        CK(cudaEventRecord(b->draw_free[k], b->res_st), "event record");  // the windows before have ended
        CK(launch_classes(b, form, w0, nw, buf, b->draw_free[k], b->res_st), "resident launch");
        CK(cudaEventRecord(b->draw_free[k], b->res_st), "event record");
        *launches += 1 + b->rclass.size();
    }
    CK(cudaEventRecord(b->res_join, b->res_st), "event record");
    return FKMC_OK;
}

}  // namespace

extern "C" {

int kmc_run(kmc_batch* b, uint64_t windows, kmc_run_stats* stats)
{
    NvtxRange nvtx_range("kmc_run");
    if (!b) return fail(FKMC_EINVAL, "null batch");
    if (!b->rates_set) return fail(FKMC_ESTATE, "kmc_set_barriers must come before kmc_run");
    std::vector<unsigned long long> before = b->stats_host;
    CK(cudaEventRecord(b->ev0, b->st), "event record");
    uint64_t res_launches = 0;
    uint64_t extra_launches = 0;
    if (site_path(b) && !b->field_valid) {
        int rc0 = rebuild_field(b);
        if (rc0) return rc0;
        extra_launches = (b->n_vv > 0) + (b->n_bo > 0);
    }
    // capture one window (set-up + 8 x (screen, run)); every argument is fixed until
    // the tables are rebuilt, which drops the graph
    auto ensure_graph = [&]() -> int {
        if (b->window_exec) return FKMC_OK;
        if (!b->cap_st) CK(cudaStreamCreateWithFlags(&b->cap_st, cudaStreamNonBlocking), "stream");
        cudaGraph_t graph = nullptr;
        int small_blocks = 1;
        const bool split = window_split(site_path(b), b->total_items, b->opts.small_pass);
        const int lane = window_lane(b->opts.precision, b->opts.small_pass, b->opts.lane_form, b->total_items);
        if (split) CK(small_pass_blocks(b->opts.precision, b->grains_on, lane, &small_blocks), "occupancy query");
        if (!b->side_st) {
            CK(cudaStreamCreateWithFlags(&b->side_st, cudaStreamNonBlocking), "stream");
            CK(cudaEventCreateWithFlags(&b->side_fork, cudaEventDisableTiming), "event");
            CK(cudaEventCreateWithFlags(&b->side_join, cudaEventDisableTiming), "event");
        }
        CK(cudaStreamBeginCapture(b->cap_st, cudaStreamCaptureModeThreadLocal), "graph capture");
        SiteArgs wa = site_args(b);
        if (!site_path(b)) wa.field = nullptr;  // the table-rate run pass
        cudaError_t le = launch_window(b->opts.precision, b->d_desc, b->n, b->total_items, b->wctl, b->perms, b->act,
                                       b->act_count, b->cls, b->occ, b->recs, b->counts, b->tracer, b->stats, b->status, b->cap,
                                       b->run_blocks, small_blocks, split, lane, wa, b->cap_st, b->side_st,
                                       b->side_fork, b->side_join);
        cudaError_t ce = cudaStreamEndCapture(b->cap_st, &graph);
        if (le != cudaSuccess) return cuda_fail(le, "window capture");
        if (ce != cudaSuccess) return cuda_fail(ce, "window capture");
        cudaError_t ie = cudaGraphInstantiate(&b->window_exec, graph, 0);
        cudaGraphDestroy(graph);
        if (ie != cudaSuccess) {
            b->window_exec = nullptr;
            return cuda_fail(ie, "graph instantiate");
        }
        return FKMC_OK;
    };
    uint64_t passes_at = UINT64_MAX, pass_windows = 0;  // the passes' window counter; windows they ran
    const uint64_t every = b->elec_on ? (uint64_t)b->elec.refresh_windows : 0;
    for (uint64_t wk = 0; wk < windows;) {
        if (every > 0 && b->elec_age >= every) {  // the potential follows the vacancies
            int rc1 = elec_refresh(b);
            if (rc1) return rc1;
            extra_launches += elec_launches(b);
            rc1 = drop_resident_cache(b);  // the rates of every fragment changed
            if (rc1) return rc1;
        }
        const uint64_t nw = every > 0 ? std::min(windows - wk, every - b->elec_age) : windows - wk;
        if (!b->rclass.empty()) {
            int rc2 = launch_resident_classes(b, wk, nw, &res_launches);
            if (rc2) return rc2;
        }
        if (b->any_global) {
            int rc2 = ensure_graph();
            if (rc2) return rc2;
            if (passes_at != wk) {  // the first, or the first after a refresh that changed the plan
                const unsigned long long at[2] = {wk, 0};
                CK(wk == 0 ? cudaMemsetAsync(b->wctl, 0, sizeof at, b->st)
                           : cudaMemcpyAsync(b->wctl, at, sizeof at, cudaMemcpyHostToDevice, b->st),
                   "window counter");
            }
            for (uint64_t k = 0; k < nw; ++k) CK(cudaGraphLaunch(b->window_exec, b->st), "graph launch");
            passes_at = wk + nw;
            pass_windows += nw;
        }
        if (!b->rclass.empty()) CK(cudaStreamWaitEvent(b->st, b->res_join, 0), "stream wait");
        wk += nw;
        b->elec_age += nw;
    }
    CK(cudaEventRecord(b->ev1, b->st), "event record");
    for (int r = 0; r < b->n; ++r) b->desc[r].window += windows;
    int rc = upload_desc(b);
    if (rc) return rc;
    CK(cudaMemcpyAsync(b->stats_host.data(), b->stats, sizeof(unsigned long long) * 2 * b->n,
                       cudaMemcpyDeviceToHost, b->st),
       "stats copy");
    rc = check_status(b);
    if (stats) {
        std::memset(stats, 0, sizeof *stats);
        for (int r = 0; r < b->n; ++r) {
            stats->hops += b->stats_host[2 * r] - before[2 * r];
            stats->handoffs += b->stats_host[2 * r + 1] - before[2 * r + 1];
        }
        stats->windows = windows;
        stats->launches =
            res_launches +
            window_launches(b) * pass_windows +
            extra_launches;
        float ms = 0.f;
        cudaEventElapsedTime(&ms, b->ev0, b->ev1);
        stats->gpu_ms = ms;
    }
    return rc;
}

int kmc_run_null(kmc_batch* b, uint64_t steps, int64_t n_frg, kmc_run_stats* stats)
{
    NvtxRange nvtx_range("kmc_run_null");
    if (!b) return fail(FKMC_EINVAL, "null batch");
    if (!b->rates_set) return fail(FKMC_ESTATE, "kmc_set_barriers must come before kmc_run_null");
    if (site_path(b)) return fail(FKMC_EINVAL, "the null-event form has no site energies or electrostatics");
    if (n_frg < 1) return fail(FKMC_EINVAL, "n_frg must be >= 1");
    if (steps > 0xFFFFFFF0ull) return fail(FKMC_EINVAL, "at most 2^32 - 16 steps per call");
    // per-replica tables and offsets
    int64_t total_vac = 0, total_picks = 0;
    for (int r = 0; r < b->n; ++r) {
        RepDesc& D = b->desc[r];
        float k32[6], kmax = 0.0f;
        for (int i = 0; i < 6; ++i) {
            k32[i] = (float)D.k64[i];
            kmax = std::max(kmax, k32[i]);
        }
        const int64_t nv = b->n_vac[r];
        const int F = 63 - ceil_log2(8 * std::max<int64_t>(nv, 1));
        for (int i = 0; i < 6; ++i) D.qn[i] = (uint64_t)std::llrint(std::ldexp((double)k32[i] / (double)kmax, F));
        for (int i = 0; i < 6; ++i)
            D.qng[i] = b->grains_on ? (uint64_t)std::llrint(std::ldexp((double)(float)D.k64g[i] / (double)kmax, F))
                                    : D.qn[i];
        D.two_pow_Fn = std::ldexp(1.0, F);
        D.vac_off = total_vac;
        D.null_nv = nv;
        D.null_nfrg = std::min<int64_t>(n_frg, nv);
        D.pick_off = total_picks;
        total_vac += nv;
        total_picks += D.null_nfrg;
    }
    if (total_vac > b->vac_cap) {
        b->dfree(b->vac);
        b->vac = (VacRec*)b->dalloc(sizeof(VacRec) * total_vac);
        b->vac_cap = b->vac ? total_vac : 0;
        if (!b->vac) return fail(FKMC_ENOMEM, "device allocation failed (null-event vacancies)");
        if (b->null_exec) cudaGraphExecDestroy(b->null_exec);
        b->null_exec = nullptr;
    }
    if (!b->theta) {  // the last of the five: all of them are there once it is
        auto have = [&](auto*& p, size_t bytes) {
            if (!p) p = static_cast<std::remove_reference_t<decltype(p)>>(b->dalloc(bytes));
            return p != nullptr;
        };
        if (!have(b->claims, sizeof(unsigned long long) * b->nsite_total) ||
            !have(b->nacc, sizeof(unsigned long long) * 3 * b->n) || !have(b->nE, sizeof(double) * b->n) ||
            !have(b->nctl, sizeof(unsigned long long) * 3) || !have(b->theta, sizeof(double) * b->n))
            return fail(FKMC_ENOMEM, "device allocation failed (null-event buffers)");
        CK(cudaMemcpyAsync(b->theta, b->theta_host.data(), sizeof(double) * b->n, cudaMemcpyHostToDevice, b->st),
           "clock upload");
    }
    // one launch for many steps: where its grid holds the vacancies and its two buffers
    // can be had, else the launches of each step.  (One step alone is cheaper in its own
    // launches: a call on 64^3 cells 92 us, 97 with the barriers and the clock's launch;
    // two steps 115 and 106.)
    NullStepsPlan plan;
    int64_t max_vac = 0, max_sites = 0;
    for (int r = 0; r < b->n; ++r) {
        max_vac = std::max(max_vac, b->n_vac[r]);
        max_sites = std::max(max_sites, b->desc[r].nsite);
    }
    auto grow = [&](void** p, size_t* have, size_t want) -> bool {
        if (want <= *have) return true;
        b->dfree(*p);
        *p = b->dalloc(want);
        *have = *p ? want : 0;
        return *p != nullptr;
    };
    const int log_steps = (int)std::min<uint64_t>(NULL_LOG_STEPS, steps);
    const bool one_launch = steps > 1 && null_steps_plan(b->n, max_vac, max_sites, &plan) &&
                            grow((void**)&b->null_types, &b->null_types_bytes, sizeof(uint32_t) * (size_t)total_vac) &&
                            grow(&b->null_log, &b->null_log_size, null_log_bytes(b->n, log_steps));
    if (total_picks > b->props_cap) {
        if (b->null_exec) cudaGraphExecDestroy(b->null_exec);
        b->null_exec = nullptr;
        b->dfree(b->props);
        b->props = (NullProp*)b->dalloc(sizeof(NullProp) * total_picks);
        if (!b->props) {
            b->props_cap = 0;
            return fail(FKMC_ENOMEM, "device allocation failed (null-event picks)");
        }
        b->props_cap = total_picks;
    }
    int rc = upload_desc(b);
    if (rc) return rc;
    std::vector<unsigned long long> before = b->stats_host;
    CK(cudaEventRecord(b->ev0, b->st), "event record");
    uint64_t launches = 0;
    CK(cudaMemsetAsync(b->claims, 0xFF, sizeof(unsigned long long) * b->nsite_total, b->st), "memset");
    CK(cudaMemsetAsync(b->nacc, 0, sizeof(unsigned long long) * 3 * b->n, b->st), "memset");
    CK(cudaMemsetAsync(b->nctl, 0, sizeof(unsigned long long) * 3, b->st), "memset");
    CK(launch_null_gather(b->d_desc, b->n, b->recs, b->counts, b->nfrag_total, b->cap, b->vac, b->status, b->st),
       "null gather");
    ++launches;
    if (one_launch) {
        const uint64_t run = b->opts.test_stuck_wait_us ? std::min<uint64_t>(steps, NULL_LOG_STEPS) : steps;
        for (uint64_t k = 0; k < run; k += NULL_LOG_STEPS) {
            CK(launch_null_steps(plan, b->d_desc, b->n, k, (int)std::min<uint64_t>(NULL_LOG_STEPS, steps - k), b->vac,
                                 b->null_types, b->occ, b->grains_on ? b->gbound : nullptr, b->claims, b->tracer,
                                 b->null_log, b->theta, b->stats, b->status, (uint32_t)b->opts.test_stuck_wait_us,
                                 b->st),
               "null-event steps");
            launches += 2;
        }
    } else if (steps > 0 && total_vac > 0) {
        if (!b->null_exec || b->null_exec_picks != total_picks || b->null_exec_vac != total_vac ||
            b->null_exec_grains != b->grains_on) {
            if (b->null_exec) cudaGraphExecDestroy(b->null_exec);
            b->null_exec = nullptr;
            if (!b->cap_st) CK(cudaStreamCreateWithFlags(&b->cap_st, cudaStreamNonBlocking), "stream");
            cudaGraph_t graph = nullptr;
            CK(cudaStreamBeginCapture(b->cap_st, cudaStreamCaptureModeThreadLocal), "graph capture");
            cudaError_t le = launch_null_step(b->d_desc, b->n, total_vac, total_picks, b->vac, b->occ,
                                              b->grains_on ? b->gbound : nullptr, b->nacc, b->props, b->claims,
                                              b->tracer, b->theta, b->nE, b->stats, b->nctl, b->cap_st);
            cudaError_t ce = cudaStreamEndCapture(b->cap_st, &graph);
            if (le != cudaSuccess) return cuda_fail(le, "null step capture");
            if (ce != cudaSuccess) return cuda_fail(ce, "null step capture");
            cudaError_t ie = cudaGraphInstantiate(&b->null_exec, graph, 0);
            cudaGraphDestroy(graph);
            if (ie != cudaSuccess) {
                b->null_exec = nullptr;
                return cuda_fail(ie, "graph instantiate");
            }
            b->null_exec_picks = total_picks;
            b->null_exec_vac = total_vac;
            b->null_exec_grains = b->grains_on;
        }
        for (uint64_t k = 0; k < steps; ++k) CK(cudaGraphLaunch(b->null_exec, b->st), "graph launch");
        launches += 3 * steps;
    }
    CK(launch_null_scatter(b->d_desc, b->n, total_vac, b->vac, b->recs, b->counts, b->nfrag_total, b->cap, b->status,
                           b->st),
       "null scatter");
    ++launches;
    CK(cudaEventRecord(b->ev1, b->st), "event record");
    for (int r = 0; r < b->n; ++r) b->desc[r].null_step += steps;
    rc = upload_desc(b);  // ahead of the copies: its wait is for the kernels anyway
    if (rc) return rc;
    CK(cudaMemcpyAsync(b->stats_host.data(), b->stats, sizeof(unsigned long long) * 2 * b->n, cudaMemcpyDeviceToHost,
                       b->st),
       "stats copy");
    CK(cudaMemcpyAsync(b->theta_host.data(), b->theta, sizeof(double) * b->n, cudaMemcpyDeviceToHost, b->st),
       "clock copy");
    uint32_t word = 0;
    rc = check_status(b, &word);
    if (word & STATUS_TIMEOUT) {  // a wait ran out: the steps are incomplete and do not count
        for (int r = 0; r < b->n; ++r) b->desc[r].null_step -= steps;
        if (const int rc_ = upload_desc(b)) return rc_;
    }
    b->field_valid = false;
    {
        const int rc_ = drop_resident_cache(b);
        if (rc_) return rc_;
    }
    if (stats) {
        std::memset(stats, 0, sizeof *stats);
        for (int r = 0; r < b->n; ++r) stats->hops += b->stats_host[2 * r] - before[2 * r];
        stats->windows = 0;
        stats->launches = launches;
        float ms = 0.f;
        cudaEventElapsedTime(&ms, b->ev0, b->ev1);
        stats->gpu_ms = ms;
    }
    return rc;
}

int kmc_read_moments(kmc_batch* b, int32_t r, int32_t species, int64_t out[7])
{
    if (!valid_replica(b, r) || !out) return fail(FKMC_EINVAL, "bad replica or output");
    if (species != FKMC_O && species != FKMC_H && species != FKMC_V) return fail(FKMC_EINVAL, "bad species");
    if (species != FKMC_V && !b->tracer) return fail(FKMC_ESTATE, "ion moments need tracer mode");
    CK(launch_moments(b->desc[r], species, b->occ, b->recs, b->counts, b->tracer, b->cap, b->scratch, b->st),
       "moments kernel");
    unsigned long long h[7];
    CK(cudaMemcpyAsync(h, b->scratch, sizeof h, cudaMemcpyDeviceToHost, b->st), "moments copy");
    CK(cudaStreamSynchronize(b->st), "synchronize");
    for (int k = 0; k < 7; ++k) out[k] = (int64_t)h[k];
    return FKMC_OK;
}

int kmc_read_moments_all(kmc_batch* b, int64_t* out, size_t n_out)
{
    if (!b || !out) return fail(FKMC_EINVAL, "null argument");
    if (n_out != 7 * (size_t)b->n) return fail(FKMC_EINVAL, "n_out must be 7 x replicas");
    int64_t max_frag = 0;
    for (const RepDesc& D : b->desc) max_frag = std::max<int64_t>(max_frag, (int64_t)D.nf[0] * D.nf[1] * D.nf[2]);
    CK(launch_moments_all(b->d_desc, b->n, b->recs, b->counts, max_frag, b->cap, b->scratch_all, b->st),
       "moments kernel");
    CK(cudaMemcpyAsync(out, b->scratch_all, sizeof(int64_t) * n_out, cudaMemcpyDeviceToHost, b->st),
       "moments copy");
    CK(cudaStreamSynchronize(b->st), "synchronize");
    return FKMC_OK;
}

int kmc_read_msd(kmc_batch* b, int32_t r, int32_t species, double msd_xyz[3], double mean_xyz[3],
                 double* t_s)
{
    int64_t m[7];
    int rc = kmc_read_moments(b, r, species, m);
    if (rc) return rc;
    const double h = 0.5 * b->a_ang[r] * 1e-10;
    const double n = m[0] > 0 ? (double)m[0] : 1.0;
    for (int k = 0; k < 3; ++k) {
        if (msd_xyz) msd_xyz[k] = (double)m[4 + k] / n * h * h;
        if (mean_xyz) mean_xyz[k] = (double)m[1 + k] / n * h;
    }
    if (t_s) *t_s = (double)b->desc[r].window * b->desc[r].tau + null_time(b, r);
    return FKMC_OK;
}

int kmc_read_D(kmc_batch* b, int32_t r, int32_t species, double D_xyz[3], double* D, double* D_xy,
               double v_drift[3])
{
    double msd[3], mean[3], t;
    int rc = kmc_read_msd(b, r, species, msd, mean, &t);
    if (rc) return rc;
    if (!(t > 0.0)) return fail(FKMC_ESTATE, "no simulated time yet");
    for (int k = 0; k < 3; ++k) {
        // the variance of the displacement along each axis: the drift is removed
        if (D_xyz) D_xyz[k] = (msd[k] - mean[k] * mean[k]) / (2.0 * t);
        if (v_drift) v_drift[k] = mean[k] / t;
    }
    if (D) *D = (msd[0] + msd[1] + msd[2]) / (6.0 * t);
    if (D_xy) *D_xy = (msd[0] + msd[1]) / (4.0 * t);
    return FKMC_OK;
}

}  // extern "C"

namespace {

constexpr size_t READ_BUF_MAX = (size_t)128 << 20;

// the batch's read-out buffer with at least `bytes` (at most READ_BUF_MAX), or null
void* read_buffer(kmc_batch* b, size_t bytes)
{
    if (bytes > b->read_bytes) {
        b->dfree(b->read_buf);
        b->read_buf = b->dalloc(bytes);
        b->read_bytes = b->read_buf ? bytes : 0;
    }
    return b->read_buf;
}

// Writes one byte per page of a host buffer that a device copy is about to fill
// whole: a page the process has not touched yet is mapped here in under a
// microsecond, by the copy's own page fault in some fifty.
void touch_pages(void* host, size_t bytes)
{
    volatile char* p = static_cast<volatile char*>(host);
    for (size_t k = 0; k < bytes; k += 4096) p[k] = 0;
}

// The state without a device buffer: the packed words, expanded here.
int unpack_on_host(kmc_batch* b, const RepDesc& D, uint8_t* host_occ)
{
    std::vector<uint32_t> w((size_t)3 * D.L[2] * D.L[1] * D.row_words);
    CK(cudaMemcpyAsync(w.data(), b->occ + D.occ_word_off, sizeof(uint32_t) * w.size(), cudaMemcpyDeviceToHost, b->st),
       "state copy");
    CK(cudaStreamSynchronize(b->st), "synchronize");
    int64_t s = 0;
    for (int t = 0; t < 3; ++t)
        for (int z = 0; z < D.L[2]; ++z)
            for (int y = 0; y < D.L[1]; ++y)
                for (int x = 0; x < D.L[0]; ++x)
                    host_occ[s++] = (uint8_t)((w[occ_index(D.row_words, D.L[1], t, x, y, z)] >> ((x & 15) * 2)) & 3u);
    return FKMC_OK;
}

}  // namespace

extern "C" {

int kmc_read_state(kmc_batch* b, int32_t r, uint8_t* host_occ, size_t n)
{
    if (!valid_replica(b, r) || !host_occ) return fail(FKMC_EINVAL, "bad replica or output");
    const RepDesc& D = b->desc[r];
    if ((int64_t)n != D.nsite) return fail(FKMC_EINVAL, "n must equal 3 nx ny nz");
    // (a small state is sooner expanded here: 8^3 cells 15 us against 20)
    if (D.nsite <= 4096) return unpack_on_host(b, D, host_occ);
    const int64_t rows = 3 * (int64_t)D.L[2] * D.L[1];
    const int64_t chunk = std::min<int64_t>(rows, std::max<int64_t>(1, (int64_t)READ_BUF_MAX / D.L[0]));
    uint8_t* buf = (uint8_t*)read_buffer(b, (size_t)(chunk * D.L[0]));
    if (!buf) return unpack_on_host(b, D, host_occ);
    touch_pages(host_occ, n);
    for (int64_t r0 = 0; r0 < rows; r0 += chunk) {
        const int64_t nr = std::min(chunk, rows - r0);
        CK(launch_unpack_state(D, b->occ, r0, nr, buf, b->st), "state kernel");
        CK(cudaMemcpyAsync(host_occ + r0 * D.L[0], buf, (size_t)(nr * D.L[0]), cudaMemcpyDeviceToHost, b->st),
           "state copy");
    }
    CK(cudaStreamSynchronize(b->st), "synchronize");
    return FKMC_OK;
}

int kmc_write_state(kmc_batch* b, int32_t r, const uint8_t* host_occ, size_t n)
{
    if (!valid_replica(b, r) || !host_occ) return fail(FKMC_EINVAL, "bad replica or input");
    const RepDesc& D = b->desc[r];
    if ((int64_t)n != D.nsite) return fail(FKMC_EINVAL, "n must equal 3 nx ny nz");
    const int64_t words = 3 * (int64_t)D.L[2] * D.L[1] * D.row_words;
    const int64_t nfrag = (int64_t)D.nf[0] * D.nf[1] * D.nf[2];
    std::vector<uint32_t> w(words, 0u);
    std::vector<int32_t> cnt(nfrag, 0);
    std::vector<VacRec> rec((size_t)nfrag * b->cap);
    int64_t s = 0, nv = 0, nh = 0;
    for (int t = 0; t < 3; ++t)
        for (int z = 0; z < D.L[2]; ++z)
            for (int y = 0; y < D.L[1]; ++y) {
                for (int x = 0; x < D.L[0]; ++x, ++s) {
                    const uint8_t c = host_occ[s];
                    if (c > 2) return fail(FKMC_EINVAL, "species codes must be 0, 1 or 2");
                    w[occ_index(D.row_words, D.L[1], t, x, y, z)] |= (uint32_t)c << ((x & 15) * 2);
                    if (c == FKMC_H) ++nh;
                    if (c != FKMC_V) continue;
                    int f[3];
                    const int cc[3] = {x, y, z};
                    for (int d = 0; d < 3; ++d) {
                        const int big = D.rem[d] * (D.base[d] + 1);
                        f[d] = cc[d] < big ? cc[d] / (D.base[d] + 1) : D.rem[d] + (cc[d] - big) / D.base[d];
                    }
                    const int64_t g = ((int64_t)f[2] * D.nf[1] + f[1]) * D.nf[0] + f[0];
                    if (cnt[g] >= b->cap) return fail(FKMC_EOVERFLOW, "a fragment would exceed cap_v vacancies");
                    VacRec& v = rec[g * b->cap + cnt[g]++];
                    v.key = ((uint64_t)t << 48) | ((uint64_t)z << 32) | ((uint64_t)y << 16) | (uint64_t)x;
                    v.d[0] = v.d[1] = v.d[2] = 0;
                    v.id = (uint32_t)nv++;
                }
            }
    CK(cudaMemcpyAsync(b->occ + D.occ_word_off, w.data(), sizeof(uint32_t) * words, cudaMemcpyHostToDevice,
                       b->st),
       "state upload");
    CK(cudaMemcpyAsync(b->counts + D.frag_base, cnt.data(), sizeof(int32_t) * nfrag, cudaMemcpyHostToDevice,
                       b->st),
       "count upload");
    CK(cudaMemcpyAsync(b->recs + D.frag_base * b->cap, rec.data(), sizeof(VacRec) * rec.size(),
                       cudaMemcpyHostToDevice, b->st),
       "record upload");
    if (b->tracer)
        CK(cudaMemsetAsync(b->tracer + 3 * D.site_off, 0, sizeof(int32_t) * 3 * D.nsite, b->st), "memset");
    CK(cudaStreamSynchronize(b->st), "synchronize");
    b->n_vac[r] = nv;
    b->n_H[r] = nh;
    b->field_valid = false;
    {
        const int rc_ = drop_resident_cache(b);
        if (rc_) return rc_;
    }
    b->elec_age = UINT64_MAX / 2;  // the potential is solved again at the next refresh point
    b->phi_prev_valid = false;  // and from zero: the vacancies may have moved anywhere
    drop_window_graph(b);       // the captured solves hold the vacancy count
    return b->rates_set ? apply_rates(b, false) : FKMC_OK;
}

int kmc_read_records(kmc_batch* b, int32_t r, int64_t* rows, int64_t max_rows, int64_t* n_rows)
{
    if (!valid_replica(b, r) || (!rows && max_rows > 0)) return fail(FKMC_EINVAL, "bad replica or output");
    const RepDesc& D = b->desc[r];
    const int64_t nfrag = (int64_t)D.nf[0] * D.nf[1] * D.nf[2];
    // rows ordered on the device, as many as the replica has vacancies (a state that
    // was uploaded with more records than that takes the host path below, as does a
    // read-out that finds no room for the buffer)
    const int64_t want = std::min(std::max<int64_t>(max_rows, 0), b->n_vac[r]);
    const size_t off_bytes = (sizeof(int64_t) * (size_t)(nfrag + 1) + 255) & ~(size_t)255;
    const size_t need = off_bytes + sizeof(int64_t) * 6 * (size_t)want;
    char* const buf = need <= READ_BUF_MAX ? (char*)read_buffer(b, need) : nullptr;
    if (buf) {
        int64_t* off = (int64_t*)buf;
        int64_t* d_rows = (int64_t*)(buf + off_bytes);
        CK(launch_rows(D, b->recs, b->counts, b->cap, off, want, d_rows, b->st), "records kernel");
        int64_t total = want;
        auto read_total = [&]() -> int {
            CK(cudaMemcpyAsync(&total, off + nfrag, sizeof total, cudaMemcpyDeviceToHost, b->st), "record copy");
            CK(cudaStreamSynchronize(b->st), "synchronize");
            return FKMC_OK;
        };
        // a state that may hold fewer records than the replica has vacancies: rows beyond
        // the last are not the call's to write, so the total comes first
        if (!b->records_match)
            if (int rc = read_total()) return rc;
        const int64_t n = std::min(total, want);
        if (n > 0) {
            touch_pages(rows, sizeof(int64_t) * 6 * (size_t)n);
            CK(cudaMemcpyAsync(rows, d_rows, sizeof(int64_t) * 6 * (size_t)n, cudaMemcpyDeviceToHost, b->st),
               "record copy");
        }
        if (int rc = read_total()) return rc;
        if (total <= want || want == max_rows || max_rows <= 0) {
            if (n_rows) *n_rows = total;
            return FKMC_OK;
        }
    }
    std::vector<int32_t> cnt(nfrag);
    std::vector<VacRec> rec((size_t)nfrag * b->cap);
    CK(cudaMemcpyAsync(cnt.data(), b->counts + D.frag_base, sizeof(int32_t) * nfrag, cudaMemcpyDeviceToHost,
                       b->st),
       "count copy");
    CK(cudaMemcpyAsync(rec.data(), b->recs + D.frag_base * b->cap, sizeof(VacRec) * rec.size(),
                       cudaMemcpyDeviceToHost, b->st),
       "record copy");
    CK(cudaStreamSynchronize(b->st), "synchronize");
    int64_t k = 0, total = 0;
    for (int64_t f = 0; f < nfrag; ++f) {
        const int c = std::min(cnt[f], b->cap);
        total += c;
        std::vector<std::pair<int64_t, int>> lst;
        for (int m = 0; m < c; ++m) {
            const VacRec& v = rec[f * b->cap + m];
            const int64_t x = v.key & 0xffff, y = (v.key >> 16) & 0xffff, z = (v.key >> 32) & 0xffff,
                          t = (int64_t)(v.key >> 48);
            lst.push_back({((t * D.L[2] + z) * D.L[1] + y) * D.L[0] + x, m});
        }
        std::sort(lst.begin(), lst.end());
        for (auto& pr : lst) {
            if (k >= max_rows) break;
            const VacRec& v = rec[f * b->cap + pr.second];
            int64_t* o = rows + 6 * k++;
            o[0] = f;
            o[1] = pr.first;
            o[2] = v.d[0];
            o[3] = v.d[1];
            o[4] = v.d[2];
            o[5] = v.id;
        }
    }
    if (n_rows) *n_rows = total;
    return FKMC_OK;
}

int kmc_read_tracer(kmc_batch* b, int32_t r, int32_t* host_disp, size_t n_sites)
{
    if (!valid_replica(b, r) || !host_disp) return fail(FKMC_EINVAL, "bad replica or output");
    if (!b->tracer) return fail(FKMC_ESTATE, "tracer mode is off");
    const RepDesc& D = b->desc[r];
    if ((int64_t)n_sites != D.nsite) return fail(FKMC_EINVAL, "n_sites must equal 3 nx ny nz");
    touch_pages(host_disp, sizeof(int32_t) * 3 * (size_t)D.nsite);
    CK(cudaMemcpyAsync(host_disp, b->tracer + 3 * D.site_off, sizeof(int32_t) * 3 * D.nsite,
                       cudaMemcpyDeviceToHost, b->st),
       "tracer copy");
    CK(cudaStreamSynchronize(b->st), "synchronize");
    return FKMC_OK;
}

}  // extern "C"

namespace {

// The state blob: a header, one row of counters per replica, then every
// mutable device array of the batch (each part starts on an 8-byte boundary).
constexpr uint64_t BLOB_MAGIC = 0x31415453434d4b46ull;  // "FKMCSTA1"
enum : uint32_t { BLOB_TRACER = 1u, BLOB_DOPANTS = 2u, BLOB_ELEC = 4u };
struct BlobHeader {
    uint64_t magic;
    uint32_t n, flags;
    uint64_t occ_words, nfrag_total, cap, nsite_total;
    uint64_t elec_age, phi_prev_valid;
};
struct BlobReplica {
    uint64_t window, null_step, hops, handoffs;
    double null_theta;
    int64_t n_vac, n_H;
};
static_assert(sizeof(BlobHeader) == 64 && sizeof(BlobReplica) == 56, "blob layout");

uint32_t blob_flags(const kmc_batch* b)
{
    return (b->tracer ? BLOB_TRACER : 0u) | (b->fe ? BLOB_DOPANTS : 0u) | (b->elec_on ? BLOB_ELEC : 0u);
}

struct BlobPart {
    void* dev;
    size_t bytes;
};

// the device arrays of the blob in order, and the header + rows size
size_t blob_parts(const kmc_batch* b, std::vector<BlobPart>* parts)
{
    const uint32_t f = blob_flags(b);
    parts->clear();
    parts->push_back({b->occ, sizeof(uint32_t) * b->occ_words});
    parts->push_back({b->recs, sizeof(VacRec) * b->nfrag_total * b->cap});
    parts->push_back({b->counts, sizeof(int32_t) * b->nfrag_total});
    if (f & BLOB_TRACER) parts->push_back({b->tracer, sizeof(int32_t) * 3 * b->nsite_total});
    if (f & BLOB_DOPANTS) parts->push_back({b->fe, (size_t)b->ncell_total});
    if (f & BLOB_ELEC) {
        parts->push_back({b->elec_u, sizeof(int32_t) * b->nsite_total});
        parts->push_back({b->phi_prev, sizeof(double) * b->ncell_total});
    }
    return sizeof(BlobHeader) + sizeof(BlobReplica) * (size_t)b->n;
}

size_t align8(size_t v) { return (v + 7) & ~(size_t)7; }

}  // namespace

extern "C" {

int kmc_state_bytes(kmc_batch* b, size_t* bytes)
{
    if (!b || !bytes) return fail(FKMC_EINVAL, "null argument");
    std::vector<BlobPart> parts;
    size_t total = blob_parts(b, &parts);
    for (const BlobPart& p : parts) total = align8(total) + p.bytes;
    *bytes = align8(total);
    return FKMC_OK;
}

int kmc_download_state(kmc_batch* b, void* host, size_t bytes)
{
    size_t need = 0;
    int rc = kmc_state_bytes(b, &need);
    if (rc) return rc;
    if (!host || bytes != need) return fail(FKMC_EINVAL, "buffer size must equal kmc_state_bytes");
    char* h = (char*)host;
    std::vector<BlobPart> parts;
    size_t off = blob_parts(b, &parts);
    BlobHeader hd{};
    hd.magic = BLOB_MAGIC;
    hd.n = (uint32_t)b->n;
    hd.flags = blob_flags(b);
    hd.occ_words = (uint64_t)b->occ_words;
    hd.nfrag_total = (uint64_t)b->nfrag_total;
    hd.cap = (uint64_t)b->cap;
    hd.nsite_total = (uint64_t)b->nsite_total;
    hd.elec_age = b->elec_age;
    hd.phi_prev_valid = b->phi_prev_valid ? 1u : 0u;
    std::memcpy(h, &hd, sizeof hd);
    for (int r = 0; r < b->n; ++r) {
        BlobReplica row{b->desc[r].window, b->desc[r].null_step, b->stats_host[2 * r], b->stats_host[2 * r + 1],
                        b->theta_host[r], b->n_vac[r], b->n_H[r]};
        std::memcpy(h + sizeof hd + sizeof row * r, &row, sizeof row);
    }
    for (const BlobPart& p : parts) {
        off = align8(off);
        CK(cudaMemcpyAsync(h + off, p.dev, p.bytes, cudaMemcpyDeviceToHost, b->st), "state copy");
        off += p.bytes;
    }
    CK(cudaStreamSynchronize(b->st), "synchronize");
    return FKMC_OK;
}

int kmc_upload_state(kmc_batch* b, const void* host, size_t bytes)
{
    size_t need = 0;
    int rc = kmc_state_bytes(b, &need);
    if (rc) return rc;
    if (!host || bytes != need) return fail(FKMC_EINVAL, "buffer size must equal kmc_state_bytes");
    const char* h = (const char*)host;
    BlobHeader hd;
    std::memcpy(&hd, h, sizeof hd);
    if (hd.magic != BLOB_MAGIC || hd.n != (uint32_t)b->n || hd.flags != blob_flags(b) ||
        hd.occ_words != (uint64_t)b->occ_words || hd.nfrag_total != (uint64_t)b->nfrag_total ||
        hd.cap != (uint64_t)b->cap || hd.nsite_total != (uint64_t)b->nsite_total)
        return fail(FKMC_EINVAL, "state blob of another batch shape (replicas, sizes, cap_v, tracer, dopants, "
                                 "electrostatics)");
    std::vector<BlobReplica> rows(b->n);
    for (int r = 0; r < b->n; ++r) {
        std::memcpy(&rows[r], h + sizeof hd + sizeof(BlobReplica) * r, sizeof(BlobReplica));
        if (rows[r].n_vac < 0 || rows[r].n_H < 0 || rows[r].n_vac + rows[r].n_H > b->desc[r].nsite)
            return fail(FKMC_EINVAL, "state blob: bad composition");
    }
    b->records_match = false;  // the blob's counts are the caller's
    std::vector<BlobPart> parts;
    size_t off = blob_parts(b, &parts);
    for (const BlobPart& p : parts) {
        off = align8(off);
        CK(cudaMemcpyAsync(p.dev, h + off, p.bytes, cudaMemcpyHostToDevice, b->st), "state upload");
        off += p.bytes;
    }
    for (int r = 0; r < b->n; ++r) {
        b->desc[r].window = rows[r].window;
        b->desc[r].null_step = rows[r].null_step;
        b->stats_host[2 * r] = rows[r].hops;
        b->stats_host[2 * r + 1] = rows[r].handoffs;
        b->theta_host[r] = rows[r].null_theta;
        b->n_vac[r] = rows[r].n_vac;
        b->n_H[r] = rows[r].n_H;
    }
    CK(cudaMemcpyAsync(b->stats, b->stats_host.data(), sizeof(unsigned long long) * 2 * b->n, cudaMemcpyHostToDevice,
                       b->st),
       "counter upload");
    if (b->theta)
        CK(cudaMemcpyAsync(b->theta, b->theta_host.data(), sizeof(double) * b->n, cudaMemcpyHostToDevice, b->st),
           "clock upload");
    CK(cudaStreamSynchronize(b->st), "synchronize");
    b->field_valid = false;  // the site-energy field is rebuilt from the restored vacancies, dopants and u
    {
        const int rc_ = drop_resident_cache(b);
        if (rc_) return rc_;
    }
    if (blob_flags(b) & BLOB_ELEC) {
        b->elec_age = hd.elec_age;
        b->phi_prev_valid = hd.phi_prev_valid != 0;
    } else {
        b->elec_age = UINT64_MAX / 2;
        b->phi_prev_valid = false;
    }
    drop_window_graph(b);  // the captured solves hold the vacancy counts
    return b->rates_set ? apply_rates(b, false) : upload_desc(b);
}

int kmc_set_site_energy(kmc_batch* b, const kmc_site_energy* e)
{
    if (!b) return fail(FKMC_EINVAL, "null batch");
    if (!e || (e->n_vv == 0 && e->n_fe == 0)) {
        if (b->site_on) {
            b->site_on = false;
            b->n_vv = b->n_bo = b->e_self = 0;  // electrostatics may keep the site-energy pass
            b->e_bound = 0;
            b->field_valid = false;
            {
                const int rc_ = drop_resident_cache(b);
                if (rc_) return rc_;
            }
            drop_window_graph(b);
            CK(run_pass_blocks(site_path(b) ? FKMC_PLAIN : b->opts.precision, b->cap, site_path(b), b->grains_on,
                               &b->run_blocks),
               "occupancy query");
            if (b->rates_set) return apply_rates(b, false);
        }
        return FKMC_OK;
    }
    if (b->opts.precision != FKMC_PLAIN) return fail(FKMC_EINVAL, "site energies need the plain form");
    ShellTables sh;
    int rc0 = make_shells(e, &sh);
    if (rc0) return rc0;
    const int reach_all = sh.reach_all, reach_vv = sh.reach_vv;
    const std::vector<SiteOff>& vv = sh.vv;
    const std::vector<SiteOff>& bo = sh.bo;
    for (int r = 0; r < b->n; ++r)
        for (int d = 0; d < 3; ++d) {
            const RepDesc& D = b->desc[r];
            if (D.L[d] < 2 * reach_all + 1)
                return fail(FKMC_EINVAL, "a dimension is shorter than twice the interaction reach plus one cell");
            if (D.nf[d] > 1 && D.base[d] < 2 + reach_vv)
                return fail(FKMC_EINVAL, "fragment edges must be at least 2 + the V-V reach (cells)");
        }
    const int32_t eself = sh.e_self;

    if (!b->field) b->field = (int32_t*)b->dalloc(sizeof(int32_t) * b->nsite_total);
    if (!b->d_vv) b->d_vv = (SiteOff*)b->dalloc(sizeof(SiteOff) * 3 * SITE_MAX_VV);
    if (!b->d_bo) b->d_bo = (SiteOff*)b->dalloc(sizeof(SiteOff) * SITE_MAX_BO);
    if (!b->fe) {
        b->fe = (uint8_t*)b->dalloc((size_t)b->ncell_total);
        if (b->fe) CK(cudaMemsetAsync(b->fe, 0, (size_t)b->ncell_total, b->st), "memset");
    }
    if (!b->field || !b->d_vv || !b->d_bo || !b->fe) return fail(FKMC_ENOMEM, "device allocation failed");
    b->n_vv = sh.nvv;
    b->reach_vv = reach_vv;
    b->n_bo = (int)bo.size();
    b->e_self = eself;
    b->e_bound = sh.bound;
    CK(cudaMemcpyAsync(b->d_vv, vv.data(), sizeof(SiteOff) * vv.size(), cudaMemcpyHostToDevice, b->st),
       "table upload");
    if (!bo.empty())
        CK(cudaMemcpyAsync(b->d_bo, bo.data(), sizeof(SiteOff) * bo.size(), cudaMemcpyHostToDevice, b->st),
           "table upload");
    b->site_on = true;
    b->field_valid = false;
    {
        const int rc_ = drop_resident_cache(b);
        if (rc_) return rc_;
    }
    drop_window_graph(b);
    CK(run_pass_blocks(FKMC_PLAIN, b->cap, true, b->grains_on, &b->run_blocks), "occupancy query");
    if (b->rates_set)
        if (int rc = apply_rates(b, true)) return rc;
    CK(cudaStreamSynchronize(b->st), "synchronize");
    return FKMC_OK;
}

int kmc_site_shells(const kmc_site_energy* e, int32_t t, int32_t* rows, int32_t max_rows, int32_t* n_rows)
{
    if (!e || t < 0 || t > 2 || (!rows && max_rows > 0)) return fail(FKMC_EINVAL, "bad argument");
    ShellTables sh;
    int rc = make_shells(e, &sh);
    if (rc) return rc;
    int k = 0;
    auto put = [&](const SiteOff& o) {
        if (k < max_rows) {
            int32_t* w = rows + 5 * k;
            w[0] = o.t2;
            for (int a = 0; a < 3; ++a) w[1 + a] = o.dc[a];
            w[4] = o.e;
        }
        ++k;
    };
    for (int i = 0; i < sh.nvv; ++i) put(sh.vv[(size_t)t * SITE_MAX_VV + i]);
    for (const SiteOff& o : sh.ob[t]) put(o);
    if (n_rows) *n_rows = k;
    return FKMC_OK;
}

int kmc_set_electrostatics(kmc_batch* b, const kmc_electrostatics* e)
{
    if (!b) return fail(FKMC_EINVAL, "null batch");
    if (!e) {
        if (!b->elec_on) return FKMC_OK;
        b->elec_on = false;
        b->elec_g.clear();
        b->elec_umax = 0;
        b->field_valid = false;
        {
            const int rc_ = drop_resident_cache(b);
            if (rc_) return rc_;
        }
        drop_window_graph(b);
        CK(run_pass_blocks(site_path(b) ? FKMC_PLAIN : b->opts.precision, b->cap, site_path(b), b->grains_on,
                           &b->run_blocks),
           "occupancy query");
        return b->rates_set ? apply_rates(b, true) : FKMC_OK;
    }
    if (b->opts.precision != FKMC_PLAIN) return fail(FKMC_EINVAL, "electrostatics need the plain form");
    if (!(e->eps_r > 0.0) || !(e->eps_r <= 1e6) || !std::isfinite(e->q_vac) || std::fabs(e->q_vac) > 8.0 ||
        e->cycles < 1 || e->cycles > 200 || e->warm_cycles < 0 || e->warm_cycles > 200 || e->refresh_windows < 0)
        return fail(FKMC_EINVAL,
                    "electrostatics: eps_r in (0, 1e6], |q| <= 8, 1..200 cycles, 0..200 warm cycles, refresh >= 0");
    for (int r = 0; r < b->n; ++r)
        if (b->desc[r].nsite / 3 > INT32_MAX)
            return fail(FKMC_EINVAL, "electrostatics: at most 2^31 - 1 cells per replica");
    // buffers: u per site, tables, the multigrid levels of the largest replica
    int64_t total = 0, nodes = 0;
    for (int r = 0; r < b->n; ++r) {
        const MgPlan p = mg_plan(b->desc[r].L[0], b->desc[r].L[1], b->desc[r].L[2]);
        total = std::max(total, p.total);
        nodes = std::max<int64_t>(nodes, b->desc[r].nsite / 3);
    }
    if (!b->elec_u) b->elec_u = (int32_t*)b->dalloc(sizeof(int32_t) * b->nsite_total);
    if (!b->d_elec_g) b->d_elec_g = (int32_t*)b->dalloc(sizeof(int32_t) * 24 * b->n);
    if (!b->d_umax) b->d_umax = (unsigned*)b->dalloc(sizeof(unsigned));
    if (!b->field) b->field = (int32_t*)b->dalloc(sizeof(int32_t) * b->nsite_total);
    if (total > b->mg_total || nodes > b->mg_nodes) {
        for (void* q : {(void*)b->mgb.phi, (void*)b->mgb.f, (void*)b->mgb.r, (void*)b->mgb.e, (void*)b->mgb.g,
                        (void*)b->mgb.s, (void*)b->mgb.cnt})
            b->dfree(q);
        b->mgb.phi = (double*)b->dalloc(sizeof(double) * nodes);
        b->mgb.f = (double*)b->dalloc(sizeof(double) * nodes);
        b->mgb.r = (double*)b->dalloc(sizeof(double) * nodes);
        b->mgb.e = (float*)b->dalloc(sizeof(float) * total);
        b->mgb.g = (float*)b->dalloc(sizeof(float) * total);
        b->mgb.s = (float*)b->dalloc(sizeof(float) * total);
        b->mgb.cnt = (int32_t*)b->dalloc(sizeof(int32_t) * nodes);
        b->mg_total = total;
        b->mg_nodes = nodes;
    }
    if (!b->phi_prev) b->phi_prev = (double*)b->dalloc(sizeof(double) * b->ncell_total);
    if (!b->mgb.part) b->mgb.part = (double*)b->dalloc(sizeof(double) * MG_PARTIALS);
    if (!b->mgb.scalar) b->mgb.scalar = (double*)b->dalloc(sizeof(double) * 2);
    if (!b->elec_u || !b->d_elec_g || !b->d_umax || !b->field || !b->phi_prev || !b->mgb.phi || !b->mgb.f || !b->mgb.r ||
        !b->mgb.e || !b->mgb.g || !b->mgb.s || !b->mgb.cnt || !b->mgb.part || !b->mgb.scalar)
        return fail(FKMC_ENOMEM, "device allocation failed (electrostatics)");
    b->elec = *e;
    b->phi_prev_valid = false;  // the first solve starts from zero
    // own-potential tables: a unit charge on a site of each type, its 8 neighbours
    b->elec_g.assign(24 * (size_t)b->n, 0);
    for (int r = 0; r < b->n; ++r) {
        const RepDesc& D = b->desc[r];
        const MgPlan p = mg_plan(D.L[0], D.L[1], D.L[2]);
        const double scale = 1.602176634e-19 / (8.8541878128e-12 * e->eps_r * b->a_ang[r] * 1e-10);
        const int nx = D.L[0], ny = D.L[1], nz = D.L[2];
        std::vector<double> phi((size_t)nx * ny * nz);
        auto node = [&](int x, int y, int z) {
            x = ((x % nx) + nx) % nx;
            y = ((y % ny) + ny) % ny;
            z = ((z % nz) + nz) % nz;
            return phi[((size_t)z * ny + y) * nx + x];
        };
        auto site_phi = [&](int t, int x, int y, int z) {
            return 0.5 * (node(x, y, z) + node(x + (t == 0), y + (t == 1), z + (t == 2)));
        };
        for (int t = 0; t < 3; ++t) {
            CK(elec_solve_unit(D, t, scale, e->cycles, p, b->mgb, b->st), "unit-charge solve");
            CK(cudaMemcpyAsync(phi.data(), b->mgb.phi, sizeof(double) * phi.size(), cudaMemcpyDeviceToHost, b->st),
               "copy");
            CK(cudaStreamSynchronize(b->st), "synchronize");
            const int x = nx / 2, y = ny / 2, z = nz / 2;
            const double ps = site_phi(t, x, y, z);
            for (int n = 0; n < 8; ++n) {
                const NbEntry& nb = b->nbt.e[t][n];
                const double pj = site_phi(nb.t2, x + nb.dc[0], y + nb.dc[1], z + nb.dc[2]);
                b->elec_g[24 * (size_t)r + 8 * t + n] = (int32_t)std::llrint(e->q_vac * e->q_vac * (pj - ps) * 1e4);
            }
        }
    }
    CK(cudaMemcpyAsync(b->d_elec_g, b->elec_g.data(), sizeof(int32_t) * b->elec_g.size(), cudaMemcpyHostToDevice,
                       b->st),
       "table upload");
    b->elec_on = true;
    b->elec_umax = 0;
    b->field_valid = false;  // rebuilt with u at the next run
    {
        const int rc_ = drop_resident_cache(b);
        if (rc_) return rc_;
    }
    int rc = elec_refresh(b);
    if (rc) return rc;
    drop_window_graph(b);
    CK(run_pass_blocks(FKMC_PLAIN, b->cap, true, b->grains_on, &b->run_blocks), "occupancy query");
    if (b->rates_set) {
        rc = apply_rates(b, true);
        if (rc) return rc;
    }
    CK(cudaStreamSynchronize(b->st), "synchronize");
    return FKMC_OK;
}

int kmc_solve_potential(kmc_batch* b, int32_t r, double* phi, size_t n, double* resid_rel)
{
    NvtxRange nvtx_range("kmc_solve_potential");
    if (!valid_replica(b, r) || !phi) return fail(FKMC_EINVAL, "bad replica or output");
    if (!b->elec_on) return fail(FKMC_ESTATE, "electrostatics are off");
    const RepDesc& D = b->desc[r];
    if ((int64_t)n != D.nsite / 3) return fail(FKMC_EINVAL, "n must equal nx ny nz");
    const MgPlan p = mg_plan(D.L[0], D.L[1], D.L[2]);
    const double scale = 1.602176634e-19 / (8.8541878128e-12 * b->elec.eps_r * b->a_ang[r] * 1e-10);
    double res = 0.0;
    CK(elec_solve(D, b->recs, b->counts, b->cap, b->n_vac[r], b->elec.q_vac, scale, b->elec.cycles, p, b->mgb, &res,
                  nullptr, nullptr, b->st),
       "potential solve");
    CK(cudaMemcpyAsync(phi, b->mgb.phi, sizeof(double) * n, cudaMemcpyDeviceToHost, b->st), "copy");
    CK(cudaStreamSynchronize(b->st), "synchronize");
    if (resid_rel) *resid_rel = res;
    return FKMC_OK;
}

int kmc_read_potential_energy(kmc_batch* b, int32_t r, int32_t* u, size_t n, int32_t* g)
{
    if (!valid_replica(b, r) || !u) return fail(FKMC_EINVAL, "bad replica or output");
    if (!b->elec_on) return fail(FKMC_ESTATE, "electrostatics are off");
    const RepDesc& D = b->desc[r];
    if ((int64_t)n != D.nsite) return fail(FKMC_EINVAL, "n must equal 3 nx ny nz");
    CK(cudaMemcpyAsync(u, b->elec_u + D.site_off, sizeof(int32_t) * n, cudaMemcpyDeviceToHost, b->st), "copy");
    CK(cudaStreamSynchronize(b->st), "synchronize");
    if (g) std::memcpy(g, b->elec_g.data() + 24 * (size_t)r, sizeof(int32_t) * 24);
    return FKMC_OK;
}

int kmc_write_potential_energy(kmc_batch* b, int32_t r, const int32_t* u, size_t n, const int32_t* g)
{
    if (!valid_replica(b, r) || !u) return fail(FKMC_EINVAL, "bad replica or input");
    if (!b->elec_on) return fail(FKMC_ESTATE, "electrostatics are off");
    const RepDesc& D = b->desc[r];
    if ((int64_t)n != D.nsite) return fail(FKMC_EINVAL, "n must equal 3 nx ny nz");
    int64_t um = 0;
    for (size_t i = 0; i < n; ++i) um = std::max<int64_t>(um, u[i] < 0 ? -(int64_t)u[i] : u[i]);
    CK(cudaMemcpyAsync(b->elec_u + D.site_off, u, sizeof(int32_t) * n, cudaMemcpyHostToDevice, b->st), "upload");
    if (g) {
        std::memcpy(b->elec_g.data() + 24 * (size_t)r, g, sizeof(int32_t) * 24);
        CK(cudaMemcpyAsync(b->d_elec_g + 24 * (size_t)r, g, sizeof(int32_t) * 24, cudaMemcpyHostToDevice, b->st),
           "upload");
    }
    CK(cudaStreamSynchronize(b->st), "synchronize");
    b->field_valid = false;
    {
        const int rc_ = drop_resident_cache(b);
        if (rc_) return rc_;
    }
    b->elec_age = 0;
    // the tables' range follows what was written, u and g both (g enters energy_bound
    // by itself, so that an all-zero u can need larger tables too)
    b->elec_umax = um > 0 ? 2 * um + 1024 : 0;
    drop_window_graph(b);
    return b->rates_set ? apply_rates(b, true) : FKMC_OK;
}

int kmc_set_grains(kmc_batch* b, const kmc_grains* g)
{
    if (!b) return fail(FKMC_EINVAL, "null batch");
    const bool on = g && g->n_grains > 1;
    if (on && b->opts.schedule == 2)
        return fail(FKMC_EINVAL, "grains need the colour-phase kernels (schedule 0 or 1)");
    if (on) {
        if (g->n_grains > 4096 || g->width < 1 || !(g->barrier_eV >= 0.0) || !(g->barrier_eV <= 10.0))
            return fail(FKMC_EINVAL, "grains: 2..4096 seeds, width >= 1, barrier in [0, 10] eV");
        for (int r = 0; r < b->n; ++r)
            for (int d = 0; d < 3; ++d)
                if (b->desc[r].L[d] < 2 * g->width + 1)
                    return fail(FKMC_EINVAL, "grains: every dimension must be >= 2 width + 1 cells");
        if (!b->grain) {
            b->grain = (int32_t*)b->dalloc(sizeof(int32_t) * b->ncell_total);
            b->gbound = (uint8_t*)b->dalloc((size_t)b->ncell_total);
            if (!b->grain || !b->gbound) return fail(FKMC_ENOMEM, "device allocation failed (grains)");
        }
        const int64_t need = 3 * (int64_t)b->n * g->n_grains;
        if (need > b->gX_len) {
            b->dfree(b->gX);
            b->gX = (int64_t*)b->dalloc(sizeof(int64_t) * need);
            b->gX_len = b->gX ? need : 0;
            if (!b->gX) return fail(FKMC_ENOMEM, "device allocation failed (grain seeds)");
        }
        CK(launch_grains(b->d_desc, b->n, b->ncell_total, g->n_grains, g->width, b->gX, b->grain, b->gbound, b->st),
           "grain kernels");
        b->grains = *g;
    }
    if (!on && !b->grains_on) return FKMC_OK;
    b->grains_on = on;
    drop_window_graph(b);
    CK(run_pass_blocks(site_path(b) ? FKMC_PLAIN : b->opts.precision, b->cap, site_path(b), on, &b->run_blocks),
       "occupancy query");
    if (b->rates_set) {
        for (int r = 0; r < b->n; ++r) {
            int rc = grain_tables(b, r);
            if (rc) return rc;
        }
        if (int rc = apply_rates(b, false)) return rc;
    }
    CK(cudaStreamSynchronize(b->st), "synchronize");
    return FKMC_OK;
}

int kmc_read_grains(kmc_batch* b, int32_t r, int32_t* grain, uint8_t* boundary, size_t n)
{
    if (!valid_replica(b, r) || !grain || !boundary) return fail(FKMC_EINVAL, "bad replica or output");
    if (!b->grains_on) return fail(FKMC_ESTATE, "grains are off");
    const RepDesc& D = b->desc[r];
    if ((int64_t)n != D.nsite / 3) return fail(FKMC_EINVAL, "n must equal nx ny nz");
    CK(cudaMemcpyAsync(grain, b->grain + D.site_off / 3, sizeof(int32_t) * n, cudaMemcpyDeviceToHost, b->st),
       "grain copy");
    CK(cudaMemcpyAsync(boundary, b->gbound + D.site_off / 3, n, cudaMemcpyDeviceToHost, b->st), "grain copy");
    CK(cudaStreamSynchronize(b->st), "synchronize");
    return FKMC_OK;
}

int kmc_read_dopants(kmc_batch* b, int32_t r, uint8_t* host_cells, size_t n)
{
    if (!valid_replica(b, r) || !host_cells) return fail(FKMC_EINVAL, "bad replica or output");
    const RepDesc& D = b->desc[r];
    if ((int64_t)n != D.nsite / 3) return fail(FKMC_EINVAL, "n must equal nx ny nz");
    if (!b->fe) {
        std::memset(host_cells, 0, n);
        return FKMC_OK;
    }
    CK(cudaMemcpyAsync(host_cells, b->fe + D.site_off / 3, n, cudaMemcpyDeviceToHost, b->st), "dopant copy");
    CK(cudaStreamSynchronize(b->st), "synchronize");
    return FKMC_OK;
}

int kmc_write_dopants(kmc_batch* b, int32_t r, const uint8_t* host_cells, size_t n)
{
    if (!valid_replica(b, r) || !host_cells) return fail(FKMC_EINVAL, "bad replica or input");
    const RepDesc& D = b->desc[r];
    if ((int64_t)n != D.nsite / 3) return fail(FKMC_EINVAL, "n must equal nx ny nz");
    if (!b->fe) {
        b->fe = (uint8_t*)b->dalloc((size_t)b->ncell_total);
        if (!b->fe) return fail(FKMC_ENOMEM, "device allocation failed");
        CK(cudaMemsetAsync(b->fe, 0, (size_t)b->ncell_total, b->st), "memset");
    }
    std::vector<uint8_t> h(n);
    int64_t cnt = 0;
    for (size_t c = 0; c < n; ++c) {
        h[c] = host_cells[c] ? 1 : 0;
        cnt += h[c];
    }
    CK(cudaMemcpyAsync(b->fe + D.site_off / 3, h.data(), n, cudaMemcpyHostToDevice, b->st), "dopant upload");
    CK(cudaStreamSynchronize(b->st), "synchronize");
    b->n_fe[r] = cnt;
    b->field_valid = false;
    {
        const int rc_ = drop_resident_cache(b);
        if (rc_) return rc_;
    }
    return FKMC_OK;
}

int kmc_read_site_field(kmc_batch* b, int32_t r, int32_t* host_field, size_t n)
{
    if (!valid_replica(b, r) || !host_field) return fail(FKMC_EINVAL, "bad replica or output");
    if (!site_path(b)) return fail(FKMC_ESTATE, "site energies are off");
    const RepDesc& D = b->desc[r];
    if ((int64_t)n != D.nsite) return fail(FKMC_EINVAL, "n must equal 3 nx ny nz");
    if (!b->field_valid) {
        int rc = rebuild_field(b);
        if (rc) return rc;
    }
    CK(cudaMemcpyAsync(host_field, b->field + D.site_off, sizeof(int32_t) * n, cudaMemcpyDeviceToHost, b->st),
       "field copy");
    CK(cudaStreamSynchronize(b->st), "synchronize");
    return FKMC_OK;
}

int kmc_check_invariants(kmc_batch* b, int32_t r, kmc_invariants* out)
{
    NvtxRange nvtx_range("kmc_check_invariants");
    if (!valid_replica(b, r) || !out) return fail(FKMC_EINVAL, "bad replica or output");
    if (!b->check_buf) {
        b->check_buf = (unsigned long long*)b->dalloc(sizeof(unsigned long long) * CHECK_WORDS);
        if (!b->check_buf) return fail(FKMC_ENOMEM, "device allocation failed");
    }
    CK(launch_check(b->desc[r], b->occ, b->recs, b->counts, b->cap, b->check_buf, b->st), "check kernels");
    unsigned long long h[CHECK_WORDS];
    CK(cudaMemcpyAsync(h, b->check_buf, sizeof h, cudaMemcpyDeviceToHost, b->st), "check copy");
    CK(cudaStreamSynchronize(b->st), "synchronize");
    std::memset(out, 0, sizeof *out);
    for (int c = 0; c < 4; ++c) out->sites[c] = (int64_t)h[CHK_SITES + c];
    out->records = (int64_t)h[CHK_RECORDS];
    out->rec_not_vacancy = (int64_t)h[CHK_NOT_VAC];
    out->rec_wrong_fragment = (int64_t)h[CHK_WRONG_FRAG];
    out->rec_outside = (int64_t)h[CHK_BAD_SITE];
    out->frag_bad_count = (int64_t)h[CHK_BAD_COUNT];
    out->hash_vac_sites = h[CHK_HASH_VAC];
    out->hash_rec_sites = h[CHK_HASH_REC];
    out->hash_rec_ids = h[CHK_HASH_ID];
    uint64_t ids = 0;  // every id 0 .. n_vac-1 once
    for (int64_t i = 0; i < b->n_vac[r]; ++i) ids += check_mix64((uint64_t)i);
    out->hash_ids_expected = ids;
    out->ok = out->sites[FKMC_V] == b->n_vac[r] && out->sites[FKMC_H] == b->n_H[r] && out->sites[3] == 0 &&
              out->records == b->n_vac[r] && out->rec_not_vacancy == 0 && out->rec_wrong_fragment == 0 &&
              out->rec_outside == 0 && out->frag_bad_count == 0 && out->hash_vac_sites == out->hash_rec_sites &&
              out->hash_rec_ids == ids;
    return FKMC_OK;
}

int kmc_get_replica_info(kmc_batch* b, int32_t r, kmc_replica_info* out)
{
    if (!valid_replica(b, r) || !out) return fail(FKMC_EINVAL, "bad replica or output");
    const RepDesc& D = b->desc[r];
    std::memset(out, 0, sizeof *out);
    for (int d = 0; d < 3; ++d) out->nfrag[d] = D.nf[d];
    out->cap_v = b->cap;
    out->F = D.F;
    out->precision = b->opts.precision;
    out->tau = D.tau;
    out->theta_tau = D.theta_tau;
    for (int i = 0; i < 6; ++i) {
        out->k64[i] = D.k64[i];
        out->q[i] = D.q[i];
    }
    out->window = D.window;
    out->hops = b->stats_host[2 * r];
    out->handoffs = b->stats_host[2 * r + 1];
    out->nsite = D.nsite;
    out->n_vac = b->n_vac[r];
    out->n_H = b->n_H[r];
    out->null_steps = D.null_step;
    out->null_theta = b->theta_host[r];
    out->null_time_s = null_time(b, r);
    out->n_Fe = b->n_fe[r];
    if ((int)b->run_kernel.size() == b->n) {
        out->kernel = b->run_kernel[r];
        out->ctas = b->run_ctas[r];
        out->draw_phases = b->run_kernel[r] == 1 ? D.pre_g : 0;
        out->draw_events = b->run_kernel[r] == 1 ? D.pre_ev : 0;
    }
    return FKMC_OK;
}

int32_t kmc_num_replicas(const kmc_batch* b) { return b ? b->n : 0; }

int kmc_destroy(kmc_batch* b)
{
    if (!b) return FKMC_OK;
    if (b->st) cudaStreamSynchronize(b->st);
    else cudaDeviceSynchronize();
    b->release();
    delete b;
    return FKMC_OK;
}

}  // extern "C"
