// fkmc_null.cu -- the atom-based fragment kMC with null events of
// arXiv:2004.09081 Sec. II.B (Eqs. AtomP, TimeStepFrg), the atoms being the
// vacancies.  One step over every replica of the batch, three parts:
//
//   k_null_rates    R_I of every vacancy; R_tot = sum, R_max = max (exact u64)
//   k_null_propose  N_frg picks (keyed bijection of the vacancy ids: an
//                   alternating Feistel network with hash rounds); each
//                   takes event i with probability q_i / R_max or the null
//                   event, and claims the two sites of its exchange with an
//                   atomic minimum of (step tag, pick index)
//   k_null_apply    a pick that holds both its claims applies its exchange
//                   (an earlier non-null pick sharing a site wins); the
//                   updated exchanges are disjoint and commute.  The last
//                   block to finish advances every replica's clock,
//                   clock += -ln(r') / R_tot * N_updated (Eq. TimeStepFrg)
//
// The parts run in one launch for many steps (k_null_steps, below), or, for more
// vacancies than the GPU holds threads for, as three launches per step in a graph.
//
// Rates are the mixed form's fixed point with F_null = 63 - ceil(log2(8 N_V)),
// so every sum is an exact integer and no reduction order enters the result.
#include <cuda_runtime.h>

#include <cstring>

#include <algorithm>

#include "fkmc_device.cuh"
#include "fkmc_kernels.h"

namespace fkmc {

namespace {

// replica of a vacancy (by = 0) or of a pick (by = 1)
__device__ __forceinline__ int null_replica(const RepDesc* descs, int nrep, int64_t v, int by)
{
    int lo = 0, hi = nrep - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        const int64_t start = by == 0 ? descs[mid].vac_off : descs[mid].pick_off;
        if (start <= v) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// MurmurHash3's 64-bit finaliser (Appleby): three xor-shifts by 33 around its
// two published odd multipliers.
__device__ __forceinline__ uint64_t fmix64(uint64_t h)
{
    h ^= h >> 33;
    h *= 0xff51afd7ed558ccdull;
    h ^= h >> 33;
    h *= 0xc4ceb9fe1a85ec53ull;
    h ^= h >> 33;
    return h;
}

// Pick p of a step: the image of p under an alternating Feistel bijection of
// [0, 2^m), m = max(2, ceil(log2 n)), high part m - m/2 bits, low part m/2,
// twelve rounds (high, low, high, ...) of x ^= fmix64(other ^ k_r), walked back
// into [0, n).  k[4j + i] = word i of the step's Philox block (step, j) under
// (seed, replica, PICK), j = 0, 1, 2.
constexpr int NULL_PICK_ROUNDS = 12;
struct PickKeys {
    uint64_t k[NULL_PICK_ROUNDS];
};

__device__ __forceinline__ PickKeys pick_keys(uint64_t step, uint64_t seed, uint32_t replica)
{
    PickKeys pk;
#pragma unroll
    for (int j = 0; j < NULL_PICK_ROUNDS / 4; ++j) {
        const U64x4 b = philox4x64(step, (uint64_t)j, 0, 0, seed, key_word(replica, PURPOSE_PICK));
#pragma unroll
        for (int i = 0; i < 4; ++i) pk.k[4 * j + i] = b.x[i];
    }
    return pk;
}

__device__ __forceinline__ uint64_t null_pick(uint64_t p, uint64_t n, const PickKeys& pk)
{
    int m = 2;
    while ((1ull << m) < n) ++m;
    const int bl = m / 2, bh = m - bl;
    const uint64_t ml = (1ull << bl) - 1ull, mh = (1ull << bh) - 1ull;
    uint64_t v = p;
    do {
        uint64_t hi = v >> bl, lo = v & ml;
#pragma unroll
        for (int r = 0; r < NULL_PICK_ROUNDS; r += 2) {
            hi ^= fmix64(lo ^ pk.k[r]) & mh;
            lo ^= fmix64(hi ^ pk.k[r + 1]) & ml;
        }
        v = (hi << bl) | lo;
    } while (v >= n);
    return v;
}

__device__ __forceinline__ int64_t lin(const RepDesc& D, int t, int x, int y, int z)
{
    return (((int64_t)t * D.L[2] + z) * D.L[1] + y) * D.L[0] + x;
}

// fixed-point rate of neighbour n of a vacancy at (t, x, y, z); 0 for a
// vacancy; the raised table for a hop touching a grain-boundary cell (gb)
// The neighbour table in global memory: threads of a warp index it with
// different site types, which a kernel-parameter (constant bank) table would
// serve one distinct entry at a time.
__device__ __align__(8) NbEntry g_nbn[3][8];

__device__ __forceinline__ NbEntry null_nb(int t, int n)
{
    const uint2 v = __ldg(reinterpret_cast<const uint2*>(&g_nbn[0][0]) + 8 * t + n);
    NbEntry e;
    memcpy(&e, &v, sizeof e);
    return e;
}

__device__ __forceinline__ uint64_t null_rate(const RepDesc& D, const uint32_t* occ, const uint8_t* gb, int t, int x,
                                              int y, int z, int n)
{
    const NbEntry nb = null_nb(t, n);
    const int jx = wrapc(x + nb.dc[0], D.L[0]);
    const int jy = wrapc(y + nb.dc[1], D.L[1]);
    const int jz = wrapc(z + nb.dc[2], D.L[2]);
    const uint32_t w = __ldcg(occ + occ_word(D, nb.t2, jx, jy, jz));
    const int code = (int)((w >> occ_shift(jx)) & 3u);
    if (code == SP_V) return 0ull;
    const int ty = code * 3 + nb.d[2] + 1;
    if (gb && (gb[cell_index(D, x, y, z)] | gb[cell_index(D, jx, jy, jz)])) return D.qng[ty];
    return D.qn[ty];
}

// step tag of step k of a call: later steps have smaller tags, so a claim left
// by an earlier step never beats a claim of the current one
__device__ __forceinline__ uint64_t claim_of(uint64_t k, int64_t p)
{
    return ((uint64_t)(0xFFFFFFFEu - (uint32_t)k) << 32) | (uint64_t)(uint32_t)p;
}

__global__ void k_null_gather(const RepDesc* __restrict__ descs, int nrep, const VacRec* recs, const int32_t* counts,
                              int64_t nfrag_total, int cap, VacRec* vac, uint32_t* status)
{
    const int64_t total = nfrag_total * cap;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < total;
         k += (int64_t)gridDim.x * blockDim.x) {
        const int64_t g = k / cap;
        const int slot = (int)(k % cap);
        if (slot >= counts[g]) continue;
        int lo = 0, hi = nrep - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (descs[mid].frag_base <= g) lo = mid; else hi = mid - 1;
        }
        const RepDesc& D = descs[lo];
        const VacRec r = recs[g * cap + slot];
        if ((int64_t)r.id < D.null_nv) vac[D.vac_off + r.id] = r;
        else atomicOr(status, STATUS_OVERFLOW);  // ids are 0 .. N_V-1 in a consistent state
    }
}

__global__ void k_null_scatter(const RepDesc* __restrict__ descs, int nrep, int64_t total_vac, const VacRec* vac,
                               VacRec* recs, int32_t* counts, int cap, uint32_t* status)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total_vac;
         i += (int64_t)gridDim.x * blockDim.x) {
        const RepDesc& D = descs[null_replica(descs, nrep, i, 0)];
        const VacRec r = vac[i];
        int t, x, y, z;
        split_key(r.key, t, x, y, z);
        const int64_t g = D.frag_base + ((int64_t)frag_of(z, D.base[2], D.rem[2]) * D.nf[1] +
                                         frag_of(y, D.base[1], D.rem[1])) * D.nf[0] + frag_of(x, D.base[0], D.rem[0]);
        const int slot = atomicAdd(counts + g, 1);
        if (slot < cap) recs[g * cap + slot] = r;
        else atomicOr(status, STATUS_OVERFLOW);
    }
}

// acc[3 r + 0] = R_tot, acc[3 r + 1] = R_max, acc[3 r + 2] = N_updated
__global__ void __launch_bounds__(256) k_null_rates(const RepDesc* __restrict__ descs, int nrep, int64_t total_vac,
                                                    const VacRec* __restrict__ vac, const uint32_t* occ,
                                                    const uint8_t* __restrict__ gb, unsigned long long* acc,
                                                    unsigned long long* nctl)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) {  // nothing else in this launch reads nctl
        nctl[1] = nctl[0];
        nctl[0] = nctl[0] + 1;
    }
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = i < total_vac;
    const int r = valid ? null_replica(descs, nrep, i, 0) : -1;
    unsigned long long R = 0ull;
    if (valid) {
        const RepDesc& D = descs[r];
        int t, x, y, z;
        split_key(vac[i].key, t, x, y, z);
#pragma unroll
        for (int n = 0; n < 8; ++n) R += null_rate(D, occ, gb, t, x, y, z, n);
    }
    const int r0 = __shfl_sync(0xffffffffu, r, 0);
    if (__all_sync(0xffffffffu, valid && r == r0)) {  // one replica: reduce in the warp first
        unsigned long long s = R, m = R;
#pragma unroll
        for (int off = 16; off; off >>= 1) {
            s += __shfl_xor_sync(0xffffffffu, s, off);
            m = max(m, __shfl_xor_sync(0xffffffffu, m, off));
        }
        if ((threadIdx.x & 31) == 0) {
            atomicAdd(acc + 3 * r0, s);
            atomicMax(acc + 3 * r0 + 1, m);
        }
    } else if (valid) {
        atomicAdd(acc + 3 * r, R);
        atomicMax(acc + 3 * r + 1, R);
    }
}

__global__ void __launch_bounds__(256) k_null_propose(const RepDesc* __restrict__ descs, int nrep, int64_t total_picks,
                                                      const VacRec* __restrict__ vac, const uint32_t* occ,
                                                      const uint8_t* __restrict__ gb, const unsigned long long* acc,
                                                      NullProp* props,
                                                      unsigned long long* claims, double* nE,
                                                      const unsigned long long* nctl)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total_picks) return;
    const int r = null_replica(descs, nrep, i, 1);
    const RepDesc& D = descs[r];
    const int64_t p = i - D.pick_off;
    const uint64_t k = nctl[1];
    const uint64_t step = D.null_step + k;
    const PickKeys rk = pick_keys(step, D.seed, D.replica);
    const int64_t id = (int64_t)null_pick((uint64_t)p, (uint64_t)D.null_nv, rk);
    int t, x, y, z;
    split_key(vac[D.vac_off + id].key, t, x, y, z);
    const U64x4 blk = philox4x64(step, (uint64_t)p, 0, 0, D.seed, key_word(D.replica, PURPOSE_NULL));
    const unsigned long long target = __umul64hi(blk.x[0], acc[3 * r + 1]);
    unsigned long long q[8];
#pragma unroll
    for (int n = 0; n < 8; ++n) q[n] = null_rate(D, occ, gb, t, x, y, z, n);  // 8 independent loads
    unsigned long long P = 0ull;
    int sel = -1;
#pragma unroll
    for (int n = 0; n < 8; ++n) {
        P += q[n];
        if (sel < 0 && P > target) sel = n;
    }
    if (p == 0) {  // the step's clock variate, off the critical path of the last apply block
        const U64x4 tb = philox4x64(step, ~0ull, 0, 0, D.seed, key_word(D.replica, PURPOSE_NULL));
        nE[r] = neglog64(tb.x[0]);
    }
    NullProp pr;
    pr.v = id;
    pr.n = sel;
    pr.pad = 0;
    props[i] = pr;
    if (sel < 0) return;
    const NbEntry nb = null_nb(t, sel);
    const unsigned long long mine = claim_of(k, p);
    atomicMin(claims + D.site_off + lin(D, t, x, y, z), mine);
    atomicMin(claims + D.site_off +
                  lin(D, nb.t2, wrapc(x + nb.dc[0], D.L[0]), wrapc(y + nb.dc[1], D.L[1]), wrapc(z + nb.dc[2], D.L[2])),
              mine);
}

// clock of replica r after a step: + -ln(r') / R_tot * N_updated, in units of
// 1/k32max (E = -ln(r'), r' from Philox (step, 2^64-1), drawn by the propose
// pass); hop counter; accumulators cleared
__device__ __forceinline__ void null_time(const RepDesc& D, int r, unsigned long long* acc, double* theta,
                                          unsigned long long* stats, const double* nE)
{
    const unsigned long long Rtot = __ldcg(acc + 3 * r), n = __ldcg(acc + 3 * r + 2);
    if (Rtot > 0ull) {
        const double E = __ldcg(nE + r);
        const double dth = __dmul_rn(__dmul_rn(__ddiv_rn(E, __ull2double_rn(Rtot)), D.two_pow_Fn), __ull2double_rn(n));
        theta[r] = __dadd_rn(theta[r], dth);
    }
    stats[2 * r] += n;
    acc[3 * r] = acc[3 * r + 1] = acc[3 * r + 2] = 0ull;
}

// nctl[2] counts the blocks of this launch that have finished
__global__ void __launch_bounds__(256) k_null_apply(const RepDesc* __restrict__ descs, int nrep, int64_t total_picks,
                                                    VacRec* vac, uint32_t* occ,
                                                    const NullProp* __restrict__ props,
                                                    const unsigned long long* claims, int32_t* tracer,
                                                    unsigned long long* acc, double* theta,
                                                    unsigned long long* stats, const double* nE,
                                                    unsigned long long* nctl)
{
    __shared__ bool last;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t k = nctl[1];
    bool did = false;
    int r = -1;
    if (i < total_picks) {
        r = null_replica(descs, nrep, i, 1);
        const RepDesc& D = descs[r];
        const NullProp pr = props[i];
        if (pr.n >= 0) {
            const int64_t p = i - D.pick_off;
            VacRec& v = vac[D.vac_off + pr.v];
            int t, x, y, z;
            split_key(v.key, t, x, y, z);
            const NbEntry nb = null_nb(t, pr.n);
            const int jx = wrapc(x + nb.dc[0], D.L[0]);
            const int jy = wrapc(y + nb.dc[1], D.L[1]);
            const int jz = wrapc(z + nb.dc[2], D.L[2]);
            const int64_t s_lin = lin(D, t, x, y, z), j_lin = lin(D, nb.t2, jx, jy, jz);
            const unsigned long long mine = claim_of(k, p);
            if (claims[D.site_off + s_lin] == mine && claims[D.site_off + j_lin] == mine) {
                const uint32_t w = __ldcg(occ + occ_word(D, nb.t2, jx, jy, jz));
                const uint32_t ion = (w >> occ_shift(jx)) & 3u;
                atomicXor(occ + occ_word(D, t, x, y, z), ((uint32_t)SP_V ^ ion) << occ_shift(x));
                atomicXor(occ + occ_word(D, nb.t2, jx, jy, jz), (ion ^ (uint32_t)SP_V) << occ_shift(jx));
                v.d[0] += nb.d[0];
                v.d[1] += nb.d[1];
                v.d[2] += nb.d[2];
                v.key = make_key(nb.t2, jx, jy, jz);
                if (tracer) {
                    int32_t* ts = tracer + 3 * (D.site_off + s_lin);
                    int32_t* tj = tracer + 3 * (D.site_off + j_lin);
                    ts[0] = tj[0] - nb.d[0];
                    ts[1] = tj[1] - nb.d[1];
                    ts[2] = tj[2] - nb.d[2];
                    tj[0] = tj[1] = tj[2] = 0;
                }
                did = true;
            }
        }
    }
    const int r0 = __shfl_sync(0xffffffffu, r, 0);
    if (__all_sync(0xffffffffu, r == r0)) {
        const unsigned n = __popc(__ballot_sync(0xffffffffu, did));
        if ((threadIdx.x & 31) == 0 && n) atomicAdd(acc + 3 * r0 + 2, (unsigned long long)n);
    } else if (did) {
        atomicAdd(acc + 3 * r + 2, 1ull);
    }
    // the last block to finish closes the step (threadFenceReduction pattern)
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(nctl + 2, 1ull) == (unsigned long long)(gridDim.x - 1);
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int q = threadIdx.x; q < nrep; q += blockDim.x) null_time(descs[q], q, acc, theta, stats, nE);
    if (threadIdx.x == 0) nctl[2] = 0ull;
}

// ---------------------------------------------------------------- one launch for many steps
// The same steps by one cooperative launch for a whole range of steps, `ctas`
// CTAs per replica: a step's three parts are separated by barriers among a
// replica's CTAs instead of kernel launches: 24.7 -> 12.8 us per step on the 128^3
// lattice's 18,874 vacancies (148 CTAs).  What bounds a step is its chain
// of dependent L2 round trips: about 0.4 us each for a vacancy's key, its
// neighbour words, a pick's key and types, its claims, and some 1 us per barrier.
// The picks' hashes and draws, which depend on no state, are computed while the
// rates' reads are in flight; the rates pass leaves the eight events' types packed
// in a word, so that a pick reads one word instead of eight.  A thread-block
// cluster of 16 CTAs with hardware barriers took 40 us per step: the uncoalesced
// reads of 16 SMs are what bounds it then, so the work is spread over every SM.
constexpr int CT = 128;  // threads per CTA

// One step's sums of a replica.
struct NullStep {
    unsigned long long tot, max, updated, pad;
};
// A replica's barrier: arrivals since the launch, and whether a wait ran out.
struct NullBarrier {
    unsigned int count, stop;
};

constexpr unsigned long long NULL_WAIT_NS = 2000000000ull;  // bound on one barrier wait

// Barrier number `target / ctas` of the replica's CTAs; false when a wait of
// `limit` ns ran out (here or elsewhere), after which every CTA leaves.
__device__ __forceinline__ bool null_barrier(NullBarrier* bar, unsigned target, unsigned long long limit)
{
    __shared__ int stop;
    __threadfence();  // this thread's writes before the arrival
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned c;
        asm volatile("atom.add.release.gpu.global.u32 %0, [%1], 1;" : "=r"(c) : "l"(&bar->count) : "memory");
        unsigned long long t0, t;
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
        int out = 0;
        ++c;
        while ((int)(c - target) < 0) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(&bar->count) : "memory");
            asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
            if (t - t0 > limit) {
                atomicExch(&bar->stop, 1u);
                out = 1;
                break;
            }
        }
        stop = out || *reinterpret_cast<volatile unsigned*>(&bar->stop) != 0u;
    }
    __syncthreads();
    return stop == 0;
}

// Sum and maximum over a warp of values below 2^63, by 32-bit warp reductions.
__device__ __forceinline__ void warp_sum_max(unsigned long long v, unsigned long long& sum, unsigned long long& mx)
{
    constexpr unsigned FULL = 0xffffffffu;
    const unsigned a = __reduce_add_sync(FULL, (unsigned)v & 0x1fffffu);
    const unsigned b = __reduce_add_sync(FULL, (unsigned)(v >> 21) & 0x1fffffu);
    const unsigned c = __reduce_add_sync(FULL, (unsigned)(v >> 42));
    sum = (unsigned long long)a + ((unsigned long long)b << 21) + ((unsigned long long)c << 42);
    const unsigned hi = __reduce_max_sync(FULL, (unsigned)(v >> 32));
    const unsigned lo = __reduce_max_sync(FULL, (unsigned)(v >> 32) == hi ? (unsigned)v : 0u);
    mx = ((unsigned long long)hi << 32) | lo;
}

// Steps k0 .. k0 + steps - 1 of every replica (CTAs [r ctas, (r + 1) ctas): replica
// r).  types: one word per vacancy, nibble n = rate type of event n + 1 (0: no
// event).  log: per replica and step, cleared by the caller, as are the barriers.
// A launch behind one whose wait ran out makes no step.
template <int PER>
__global__ void __launch_bounds__(CT)
    k_null_steps(const RepDesc* __restrict__ descs, int ctas, uint64_t k0, int steps, VacRec* vac, uint32_t* types,
                 uint32_t* occ, const uint8_t* __restrict__ gb, unsigned long long* claims, int32_t* tracer,
                 NullStep* log, int log_stride, NullBarrier* bars, uint32_t* status)
{
    __shared__ RepDesc D;
    __shared__ PickKeys pk[2];           // by step parity
    __shared__ unsigned long long q[16]; // rate of type t at t + 1, 0 for no event
    __shared__ unsigned long long part[2][CT / 32];
    __shared__ unsigned long long rmax;
    constexpr unsigned FULL = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rep = (int)(blockIdx.x / ctas), me = (int)(blockIdx.x - rep * ctas);
    NullBarrier* const bar = bars + rep;
    unsigned target = 0;
    __shared__ bool late;
    if (tid == 0) {
        D = descs[rep];
        late = (*reinterpret_cast<volatile uint32_t*>(status) & STATUS_TIMEOUT) != 0u;
    }
    __syncthreads();
    if (late) return;
    if (tid < 16) q[tid] = tid == 0 || tid > 12 ? 0ull : (tid <= 6 ? D.qn[tid - 1] : D.qng[tid - 7]);
    const int nv = (int)D.null_nv, np = (int)D.null_nfrg;
    VacRec* const vr = vac + D.vac_off;
    uint32_t* const ty_r = types + D.vac_off;
    uint32_t* const occ_r = occ + D.occ_word_off;
    unsigned long long* const cl = claims + D.site_off;
    const uint64_t key_null = key_word(D.replica, PURPOSE_NULL);
    const int first = me * CT + tid, stride = ctas * CT;
    auto keys_of = [&](uint64_t step) {  // one Philox block per thread of lanes 0 .. 2 of the last warp
        if (warp == CT / 32 - 1 && lane < NULL_PICK_ROUNDS / 4) {
            const U64x4 b = philox4x64(step, (uint64_t)lane, 0, 0, D.seed, key_word(D.replica, PURPOSE_PICK));
            for (int i = 0; i < 4; ++i) pk[step & 1].k[4 * lane + i] = b.x[i];
        }
    };
    keys_of(D.null_step + k0);
    __syncthreads();
    for (int s = 0; s < steps; ++s) {
        const uint64_t k = k0 + s, step = D.null_step + k;
        NullStep* const st = log + (int64_t)rep * log_stride + s;
        // ---- rates
        unsigned long long sum = 0ull, mx = 0ull;
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int i = first + u * stride;
            unsigned long long R = 0ull;
            if (i < nv) {
                int t, x, y, z;
                split_key(__ldcg(&vr[i].key), t, x, y, z);
                uint32_t w[8];
                int sh[8], base[8];
                bool bnd[8];
#pragma unroll
                for (int n = 0; n < 8; ++n) {
                    const NbEntry nb = null_nb(t, n);
                    const int jx = wrapc(x + nb.dc[0], D.L[0]);
                    const int jy = wrapc(y + nb.dc[1], D.L[1]);
                    const int jz = wrapc(z + nb.dc[2], D.L[2]);
                    w[n] = __ldcg(occ_r + occ_index(D.row_words, D.L[1], nb.t2, jx, jy, jz));
                    sh[n] = occ_shift(jx);
                    base[n] = nb.d[2] + 2;
                    bnd[n] = gb && gb[cell_index(D, jx, jy, jz)];
                }
                const bool own = gb && gb[cell_index(D, x, y, z)];
                uint32_t packed = 0;
#pragma unroll
                for (int n = 0; n < 8; ++n) {
                    const int code = (int)((w[n] >> sh[n]) & 3u);
                    const int e = code == SP_V ? 0 : code * 3 + base[n] + ((own || bnd[n]) ? 6 : 0);
                    packed |= (uint32_t)e << (4 * n);
                    R += q[e];
                }
                ty_r[i] = packed;
            }
            unsigned long long ws, wm;
            warp_sum_max(R, ws, wm);
            sum += ws;
            mx = max(mx, wm);
        }
        if (lane == 0) {
            part[0][warp] = sum;
            part[1][warp] = mx;
        }
        // this thread's picks and their draws: they depend on no state
        int id[PER];
        uint64_t xs[PER];
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int p = first + u * stride;
            id[u] = -1;
            xs[u] = 0;
            if (p < np) {
                id[u] = (int)null_pick((uint64_t)p, (uint64_t)nv, pk[step & 1]);
                xs[u] = philox4x64(step, (uint64_t)p, 0, 0, D.seed, key_null).x[0];
            }
        }
        __syncthreads();
        if (tid == 0) {
            unsigned long long t2 = 0ull, m2 = 0ull;
            for (int w = 0; w < CT / 32; ++w) {
                t2 += part[0][w];
                m2 = max(m2, part[1][w]);
            }
            atomicAdd(&st->tot, t2);
            atomicMax(&st->max, m2);
        }
        keys_of(step + 1);
        if (!null_barrier(bar, target += ctas, NULL_WAIT_NS)) break;
        // ---- picks: event or null event, claims
        if (tid == 0) rmax = __ldcg(&st->max);
        uint64_t key[PER];
        uint32_t pt[PER];
        int sel[PER], ls[PER], lj[PER];
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            key[u] = 0;
            pt[u] = 0;
            if (id[u] >= 0) {
                key[u] = __ldcg(&vr[id[u]].key);
                pt[u] = __ldcg(ty_r + id[u]);
            }
        }
        __syncthreads();
        const unsigned long long Rmax = rmax;
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            sel[u] = -1;
            ls[u] = lj[u] = 0;
            if (id[u] < 0) continue;
            const unsigned long long target = __umul64hi(xs[u], Rmax);
            unsigned long long P = 0ull;
#pragma unroll
            for (int n = 0; n < 8; ++n) {
                P += q[(pt[u] >> (4 * n)) & 15u];
                if (sel[u] < 0 && P > target) sel[u] = n;
            }
            if (sel[u] < 0) continue;
            int t, x, y, z;
            split_key(key[u], t, x, y, z);
            const NbEntry nb = null_nb(t, sel[u]);
            ls[u] = (int)lin(D, t, x, y, z);
            lj[u] = (int)lin(D, nb.t2, wrapc(x + nb.dc[0], D.L[0]), wrapc(y + nb.dc[1], D.L[1]),
                             wrapc(z + nb.dc[2], D.L[2]));
            const unsigned long long mine = claim_of(k, first + u * stride);
            atomicMin(cl + ls[u], mine);
            atomicMin(cl + lj[u], mine);
        }
        if (!null_barrier(bar, target += ctas, NULL_WAIT_NS)) break;
        // ---- exchanges of the picks that hold both their claims
        unsigned done = 0;
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            bool did = false;
            if (sel[u] >= 0) {
                const unsigned long long mine = claim_of(k, first + u * stride);
                const unsigned long long c0 = __ldcg(cl + ls[u]), c1 = __ldcg(cl + lj[u]);
                if (c0 == mine && c1 == mine) {
                    did = true;
                    int t, x, y, z;
                    split_key(key[u], t, x, y, z);
                    const NbEntry nb = null_nb(t, sel[u]);
                    const int jx = wrapc(x + nb.dc[0], D.L[0]);
                    const int jy = wrapc(y + nb.dc[1], D.L[1]);
                    const int jz = wrapc(z + nb.dc[2], D.L[2]);
                    const uint32_t ion = ((((pt[u] >> (4 * sel[u])) & 15u) - 1u) % 6u) / 3u;
                    atomicXor(occ_r + occ_index(D.row_words, D.L[1], t, x, y, z), ((uint32_t)SP_V ^ ion) << occ_shift(x));
                    atomicXor(occ_r + occ_index(D.row_words, D.L[1], nb.t2, jx, jy, jz),
                              (ion ^ (uint32_t)SP_V) << occ_shift(jx));
                    VacRec* v = vr + id[u];
                    v->key = make_key(nb.t2, jx, jy, jz);
#pragma unroll
                    for (int d = 0; d < 3; ++d)
                        if (nb.d[d]) atomicAdd(&v->d[d], (int)nb.d[d]);
                    if (tracer) {
                        int32_t* ts = tracer + 3 * (D.site_off + ls[u]);
                        int32_t* tj = tracer + 3 * (D.site_off + lj[u]);
#pragma unroll
                        for (int d = 0; d < 3; ++d) {
                            ts[d] = __ldcg(tj + d) - nb.d[d];
                            tj[d] = 0;
                        }
                    }
                }
            }
            done += __popc(__ballot_sync(FULL, did));
        }
        if (lane == 0 && done) atomicAdd(&st->updated, (unsigned long long)done);
        if (!null_barrier(bar, target += ctas, NULL_WAIT_NS)) break;
    }
    if (tid == 0 && *reinterpret_cast<volatile unsigned*>(&bar->stop) != 0u) atomicOr(status, STATUS_TIMEOUT);
}

// The test of the barrier's bounded wait: the replica's CTAs wait for one arrival more
// than there are of them.
__global__ void __launch_bounds__(CT) k_null_stuck(int ctas, NullBarrier* bars, uint32_t* status,
                                                   unsigned long long limit)
{
    if (!null_barrier(bars + blockIdx.x / ctas, (unsigned)ctas + 1u, limit) && threadIdx.x == 0)
        atomicOr(status, STATUS_TIMEOUT);
}

// The clocks and hop counters of `steps` steps from their log, one block per
// replica: clock += -ln(r') / R_tot * N_updated step by step (Eq. TimeStepFrg),
// the terms computed side by side, the sum in order.
__global__ void __launch_bounds__(256) k_null_clock(const RepDesc* __restrict__ descs, uint64_t k0, int steps,
                                                    const NullStep* __restrict__ log, int log_stride, double* theta,
                                                    unsigned long long* stats)
{
    __shared__ double term[256];
    __shared__ unsigned long long hops;
    const int r = blockIdx.x, tid = threadIdx.x;
    const RepDesc& D = descs[r];
    if (tid == 0) hops = 0ull;
    double th = theta[r];
    for (int s0 = 0; s0 < steps; s0 += 256) {
        const int s = s0 + tid;
        double dth = 0.0;
        __syncthreads();
        if (s < steps) {
            const NullStep l = log[(int64_t)r * log_stride + s];
            if (l.tot > 0ull) {
                const U64x4 b = philox4x64(D.null_step + k0 + s, ~0ull, 0, 0, D.seed, key_word(D.replica, PURPOSE_NULL));
                dth = __dmul_rn(__dmul_rn(__ddiv_rn(neglog64(b.x[0]), __ull2double_rn(l.tot)), D.two_pow_Fn),
                                __ull2double_rn(l.updated));
            }
            if (l.updated) atomicAdd(&hops, l.updated);
        }
        term[tid] = dth;
        __syncthreads();
        if (tid == 0)
            for (int q = 0; q < min(256, steps - s0); ++q) th = __dadd_rn(th, term[q]);
    }
    __syncthreads();
    if (tid == 0) {
        theta[r] = th;
        stats[2 * r] += hops;
    }
}

constexpr int NT = 256;

unsigned grid_of(int64_t n)
{
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + NT - 1) / NT, 1 << 30));
}

}  // namespace

cudaError_t launch_null_gather(const RepDesc* d_descs, int nrep, const VacRec* recs, const int32_t* counts,
                               int64_t nfrag_total, int cap, VacRec* vac, uint32_t* status, cudaStream_t st)
{
    const unsigned blocks = (unsigned)std::min<int64_t>(65536, std::max<int64_t>(1, (nfrag_total * cap + NT - 1) / NT));
    k_null_gather<<<blocks, NT, 0, st>>>(d_descs, nrep, recs, counts, nfrag_total, cap, vac, status);
    return cudaGetLastError();
}

cudaError_t launch_null_scatter(const RepDesc* d_descs, int nrep, int64_t total_vac, const VacRec* vac,
                                VacRec* recs, int32_t* counts, int64_t nfrag_total, int cap, uint32_t* status,
                                cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(counts, 0, sizeof(int32_t) * nfrag_total, st);
    if (e != cudaSuccess || total_vac == 0) return e;
    const unsigned blocks = (unsigned)std::min<int64_t>(65536, (total_vac + NT - 1) / NT);
    k_null_scatter<<<blocks, NT, 0, st>>>(d_descs, nrep, total_vac, vac, recs, counts, cap, status);
    return cudaGetLastError();
}

cudaError_t null_upload_neighbours(const NbEntry* host24)
{
    return cudaMemcpyToSymbol(g_nbn, host24, sizeof(NbEntry) * 24);
}

// One step of every replica (three launches; fixed arguments, so a graph can
// hold it).  nctl[2] must be 0 before the first step.
cudaError_t launch_null_step(const RepDesc* d_descs, int nrep, int64_t total_vac, int64_t total_picks, VacRec* vac,
                             uint32_t* occ, const uint8_t* gb, unsigned long long* acc,
                             NullProp* props,
                             unsigned long long* claims, int32_t* tracer, double* theta, double* nE,
                             unsigned long long* stats, unsigned long long* nctl, cudaStream_t st)
{
    k_null_rates<<<grid_of(total_vac), NT, 0, st>>>(d_descs, nrep, total_vac, vac, occ, gb, acc, nctl);
    k_null_propose<<<grid_of(total_picks), NT, 0, st>>>(d_descs, nrep, total_picks, vac, occ, gb, acc, props,
                                                        claims, nE, nctl);
    k_null_apply<<<grid_of(total_picks), NT, 0, st>>>(d_descs, nrep, total_picks, vac, occ, props, claims, tracer,
                                                      acc, theta, stats, nE, nctl);
    return cudaGetLastError();
}

using NullStepsFn = void (*)(const RepDesc*, int, uint64_t, int, VacRec*, uint32_t*, uint32_t*, const uint8_t*,
                             unsigned long long*, int32_t*, NullStep*, int, NullBarrier*, uint32_t*);

static NullStepsFn null_steps_kernel(int per)
{
    return per == 1 ? k_null_steps<1> : (per == 2 ? k_null_steps<2> : k_null_steps<4>);
}

size_t null_log_bytes(int nrep, int steps)
{
    return (sizeof(NullStep) * steps + sizeof(NullBarrier)) * (size_t)nrep + 32;
}

// One launch for many steps: the CTAs that hold the largest replica at the
// fewest vacancies and picks per thread (1, 2 or 4), all replicas' CTAs resident
// at once, and 32-bit site indices.  Beyond that (several hundred thousand
// vacancies) a step is bound by its reads, and the launches are as good.
bool null_steps_plan(int nrep, int64_t max_vac, int64_t max_sites, NullStepsPlan* out)
{
    if (max_vac < 1 || max_vac > (1 << 22) || max_sites > 0x7fffffffll) return false;
    int dev = 0, sms = 0, coop = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) {
        cudaGetLastError();
        return false;
    }
    for (int per = 1; per <= 4; per *= 2) {
        int per_sm = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, null_steps_kernel(per), CT, 0) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        const int64_t ctas = (max_vac + (int64_t)CT * per - 1) / ((int64_t)CT * per);
        if (ctas * nrep > (int64_t)sms * per_sm) continue;
        out->ctas = (int)ctas;
        out->per = per;
        return true;
    }
    return false;
}

cudaError_t launch_null_steps(const NullStepsPlan& p, const RepDesc* d_descs, int nrep, uint64_t k0, int steps,
                              VacRec* vac, uint32_t* types, uint32_t* occ, const uint8_t* gb,
                              unsigned long long* claims, int32_t* tracer, void* log_mem, double* theta,
                              unsigned long long* stats, uint32_t* status, uint32_t stuck_wait_us, cudaStream_t st)
{
    NullBarrier* bars = reinterpret_cast<NullBarrier*>(log_mem);
    NullStep* log = reinterpret_cast<NullStep*>(reinterpret_cast<char*>(log_mem) + ((sizeof(NullBarrier) * nrep + 31) & ~(size_t)31));
    int stride = steps;
    cudaError_t e = cudaMemsetAsync(log_mem, 0, (((sizeof(NullBarrier) * nrep + 31) & ~(size_t)31) +
                                                 sizeof(NullStep) * (size_t)nrep * stride), st);
    if (e != cudaSuccess) return e;
    int ctas = p.ctas;
    if (stuck_wait_us) {  // the steps' launch then finds the status set
        unsigned long long limit = 1000ull * stuck_wait_us;
        void* stuck[] = {&ctas, &bars, &status, &limit};
        e = cudaLaunchCooperativeKernel((const void*)k_null_stuck, dim3((unsigned)(ctas * nrep)), dim3(CT), stuck, 0, st);
        if (e != cudaSuccess) return e;
    }
    void* args[] = {(void*)&d_descs, &ctas, &k0, &steps, &vac, &types, &occ, (void*)&gb, &claims, &tracer, &log,
                    &stride, &bars, &status};
    e = cudaLaunchCooperativeKernel((const void*)null_steps_kernel(p.per), dim3((unsigned)(ctas * nrep)), dim3(CT), args,
                                    0, st);
    if (e != cudaSuccess) return e;
    k_null_clock<<<nrep, 256, 0, st>>>(d_descs, k0, steps, log, stride, theta, stats);
    return cudaGetLastError();
}

}  // namespace fkmc
