// fkmc_resident.cu -- replica-resident window kernels (both arithmetic forms).
//
// One CTA (k_resident<..., false>) or one thread-block cluster of up to 16 CTAs
// (k_resident<..., true>, CTA c holding the z-slab of fragment layers
// [P.fz0[c], P.fz0[c+1])) owns one replica for a whole launch: the packed
// occupancy lives in shared memory and every window and colour phase runs with
// CTA or cluster barriers only, because replicas are independent.  The fragment
// BKL is that of arXiv:2004.09081 Sec. II.A (Eqs. RateCnst1, eventSelection,
// TimeStep) with fragment-local selection (Sec. II.B, Eq. AtomP); the mixed
// form's sums are exact u64 integers, the plain form sums FP64 rates in the
// canonical order of the colour-phase kernels, so both reproduce them (and the
// oracle) bit for bit.
//
// The occupancy is the only copy of the vacancies' positions.  A visit finds
// its fragment's vacancies by scanning the fragment's rows for the vacancy
// code, which yields them in site order (the slots' order) without a list to
// walk, sort, relink or hand over: a vacancy that hops into another fragment
// (or another CTA's slab) belongs to it by lying there.  A record is reached
// only when its vacancy hops, through vmap, one word per site in global memory
// with the index of the vacancy's record; the word is loaded when a visit
// starts and arrives long before the first exchange needs it, and the
// displacement goes to the record with fire-and-forget reductions.  At the end
// of a launch the records move to the lists of the fragments that hold them.
//
// Each colour phase has two passes:
//   screen  one thread per fragment of the colour.  A fragment whose
//           neighbourhood did not change since its last visit keeps its exact
//           event total; with the first draw of the phase, a first event past
//           the window proves that nothing happens, and the fragment is skipped.
//           Everything else goes to a compact list.
//   run     one warp per listed fragment (lane = 4 slots x 8 directions per
//           32-event chunk): total, clock, selection by warp scan, exchange, and
//           "dirty" marks on the owners of every vacancy next to one of the two
//           changed sites -- exactly the fragments whose total changed.
//           Fragments of one colour never touch each other's sites (edges >= 2).
//
// What bounds it: dependent instructions.  A running warp issues one every 6 to
// 8 cycles (2.2 to 2.6 of them fixed latency, 1.0 to 1.1 shared memory, 0.3 to
// 1.0 L2, 0.5 to 1.3 instruction fetch; 256 uneven replicas and one of 128^3
// cells, calls of 8 and 16 windows), a phase lasts as long as its slowest visit
// (one to three events, some 900 instructions), and no pipe is near its rate: a
// quarter SM issues in 7 to 23% of its cycles.  So a visit does
// as little as it can in sequence: totals by warp reductions with the prefix
// scan only for events that happen, no FP64 instruction in the mixed form and
// few in the plain one, records and tracer written an exchange late.
// Measured (one GB300, whole calls with read-out, against linked per-fragment
// lists for the mixed form and per-phase launches for the plain form): 256
// uneven replicas mixed 60.5 -> 52.2 us per window, 24 traced 32^3 replicas
// mixed 22.7 -> 18.4, 128^3 mixed 54.9 -> 47.7; plain: five 32^3 replicas 154 ->
// 27.4, 8^3 112 -> 28.0, 128^3 195 -> 69.2.
//
// With site energies (plain form) a visit's chain is some 8,000 cycles per event
// instead of 3,500: the rates wait for the energy field's words in L2, after an
// exchange behind the 116 atomics that move the vacancy's share.  Five doped 96^3
// replicas 302 -> 156 us per window (182 in the first pass on a new state), 128^3
// in its own potential 482 -> 313 with the solves.  Holding a visit's moves back
// and correcting the rates by pair energies instead was slower (190 -> 200): the
// pair energies cost as many instructions as the wait.
//
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstddef>

#include "fkmc_device.cuh"
#include "fkmc_kernels.h"

namespace fkmc {

namespace {

__device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ uint64_t globaltimer()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait: gives up after `ns` nanoseconds and reports it.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, uint64_t ns)
{
    const uint64_t t0 = globaltimer();
    while (!mbar_try_wait(bar, parity))
        if (globaltimer() - t0 > ns) return false;
    return true;
}

__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void bulk_s2g(void* dst, const void* src, uint32_t bytes)
{
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)),
                 "r"(bytes)
                 : "memory");
}

// ---- thread-block cluster and distributed shared memory
__device__ __forceinline__ uint32_t cluster_ctarank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ uint32_t cluster_nctas()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}

// every thread of every CTA of the cluster; release / acquire of shared memory
__device__ __forceinline__ void cluster_sync()
{
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// the two halves of cluster_sync: work that reads and writes nothing a peer
// touches may run between them
__device__ __forceinline__ void cluster_arrive()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait()
{
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// address in CTA `peer`'s shared memory of the same variable as `p`
__device__ __forceinline__ uint32_t peer_addr(const void* p, uint32_t peer)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(peer));
    return r;
}

__device__ __forceinline__ void st_peer8(uint32_t a, uint8_t v)
{
    asm volatile("st.shared::cluster.u8 [%0], %1;" ::"r"(a), "h"((unsigned short)v) : "memory");
}
__device__ __forceinline__ void st_peer(uint32_t a, uint32_t v)
{
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void st_peer64(uint32_t a, unsigned long long v)
{
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}
__device__ __forceinline__ void red_peer_xor(uint32_t a, uint32_t v)
{
    asm volatile("red.shared::cluster.xor.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ int32_t ld_peer(uint32_t a)
{
    int32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}

constexpr uint32_t BULK_CHUNK = 32768;        // bytes per bulk copy instruction
constexpr uint64_t WAIT_NS = 2000000000ull;   // 2 s bound on any device-side wait
constexpr uint32_t DEAD = 0xffffffffu;        // slot key of a vacancy that left the fragment, or of no vacancy

// compact site key: t<<30 | z<<20 | y<<10 | x (cells < 1024), ordered like the
// linear site index
__device__ __forceinline__ uint32_t key32(int t, int x, int y, int z)
{
    return ((uint32_t)t << 30) | ((uint32_t)z << 20) | ((uint32_t)y << 10) | (uint32_t)x;
}

__device__ __forceinline__ void split32(uint32_t k, int& t, int& x, int& y, int& z)
{
    x = (int)(k & 1023u);
    y = (int)((k >> 10) & 1023u);
    z = (int)((k >> 20) & 1023u);
    t = (int)(k >> 30);
}

// rate types of an event: species * 3 + dz + 1; a vacancy neighbour (species 2)
// gives 6..8, which the rate table holds as zeros
constexpr int NO_EVENT = 6;

struct Shared {
    RepDesc D;
    ClusterPlan P;
    uint64_t rate[9];    // mixed: fixed-point rates, plain: bits of the FP64 rates
    uint64_t bar;
    uint64_t bar_test;   // the wait test's barrier, which nothing completes
    uint32_t perms[64];  // colour orders of 64 consecutive windows (nibble p = colour of phase p)
    int coff[9];         // first entry of each colour in the fragment list
    int zbeg[CLUSTER_MAX_CTAS + 1];  // first z cell of CTA c's slab
    int nact[2];         // screened fragments, by phase parity
    int next_act[2];     // tickets beyond each warp's first
    int ndraw;           // fragments of the current batch of first draws
    unsigned long long hops, hand;
    int abort;
    int cached;          // the fragment totals of the last launch are valid
};

// What the screen compares a fragment's first variate E with (see `limit_of`):
// active where E <= limit.  Mixed: FP32 bits, plain: FP64 bits.
template <int PREC>
struct Limit;
template <>
struct Limit<1> {
    using T = uint32_t;
    static constexpr T DIRTY = 0x7f800000u;  // +inf: the total is not known
    static constexpr T EMPTY = 0u;           // no event
};
template <>
struct Limit<0> {
    using T = uint64_t;
    static constexpr T DIRTY = 0x7ff0000000000000ull;
    static constexpr T EMPTY = 0ull;
};

struct Layout {
    uint32_t* occ;         // [zs][L1][RW][3], the global layout of the slab's z cells
    void* lim;             // Limit<PREC>::T by local fragment
    uint8_t* stale;        // 1: a vacancy came in since `slots` was written
    uint64_t* wlog;        // plain, per warp: E and R of events whose clock division is put off
    double* btab;          // site energies: the Boltzmann tables lo[BOLTZ_LO], hi[bhi_len]
    uint32_t* slots;       // site keys of each local fragment's vacancies in site order (DEAD: none), or
                           // UNLISTED where it holds more than KSLOTS
    uint2* box;            // first cell and extent of each local fragment, 10 bits per dimension
    uint16_t* flist;       // this CTA's fragments by colour
    uint32_t* act;         // screened fragments: local fragment | index in its colour << 16
    uint64_t* pre_xs;      // first draws by (row, event): selection words
    void* pre_E;           // and exponential variates (mixed: floats; plain: doubles)
    uint16_t* pre_row;     // one CTA: row of each fragment's first draws, NO_ROW: none
    uint16_t* dlist;       // one CTA: the fragments of the current batch of first draws
    uint16_t* frag_of_c;   // cell -> fragment coordinate: x cells, then y, then z
    uint32_t* zmap;        // cluster: z cell -> CTA | z within its slab << 8 | fragment layer within it << 18
    uint32_t* wkey;        // per warp: site key of each slot
    uint32_t* wvac;        // per warp: record index of each slot (fragments of more than 32 vacancies)
    int8_t* wtype;         // per warp: rate type of each event (more than two chunks)
};
constexpr unsigned NO_ROW = 0xffffu;      // a fragment's row of first draws: none,
constexpr unsigned ROW_FULL = 0x8000u;    // or row | ROW_FULL where every event of the row was drawn (else two)
constexpr int KSLOTS = 8;                  // entries of a fragment's list (or 4 or 16: RepDesc.kslots)
constexpr int LONG_SLOTS = 16;
constexpr int CLOCK_LOG = 8;  // events whose clock division the plain form puts off
constexpr uint32_t UNLISTED = 0xfffffffeu;

// Shared-memory arrays of one CTA: `zs` cells in z, `nfl` fragments, `maxc`
// fragments of one colour at most.
struct Sizes {
    int64_t words;
    int nfl, maxc, cap, nwarps, ltot, lz, rows, pre_ev, prec, kslots, btab;
};

constexpr int NARR = 18;

__host__ __device__ inline size_t layout_bytes(const Sizes& z, size_t* off /* NARR offsets or null */)
{
    // every array starts on a 16-byte boundary, whatever the sizes before it
    const size_t draws = (size_t)z.rows * z.maxc * z.pre_ev;
    const size_t sz[NARR] = {
        (size_t)z.words * 4,             // 0 occupancy (bulk-copied)
        (size_t)z.nfl * (z.prec ? 4 : 8),  // 1 limits
        (size_t)z.nfl * 8,               // 2 boxes
        (size_t)z.nfl * 2,               // 3 fragment list
        (size_t)z.maxc * 4,              // 4 screened list
        draws * 8,                       // 5 first draws: selection words
        draws * (z.prec ? 4 : 8),        // 6 and variates
        z.lz ? 0 : (size_t)z.nfl * 2,    // 7 their rows
        z.lz ? 0 : (size_t)z.rows * z.maxc * 2,  // 8 the batch's fragments
        (size_t)z.ltot * 2,              // 9 cell -> fragment tables
        (size_t)z.lz * 4,                // 10 z cell -> CTA, slab z, slab layer
        (size_t)z.nwarps * z.cap * 4,    // 11 per-warp slot keys
        (size_t)z.nwarps * z.cap * 4,    // 12 per-warp record indices
        (size_t)z.nwarps * z.cap * 8,    // 13 per-warp event types
        (size_t)z.nfl,                   // 14 stale flags
        (size_t)z.nfl * z.kslots * 4,    // 15 vacancies by fragment
        z.prec ? 0 : (size_t)z.nwarps * CLOCK_LOG * 16,  // 16 per-warp clock log (plain)
        (size_t)z.btab * 8,              // 17 Boltzmann tables (site energies, where they fit)
    };
    size_t b = 0;
    for (int k = 0; k < NARR; ++k) {
        if (off) off[k] = b;
        b += (sz[k] + 15) & ~(size_t)15;
    }
    return (b + 127) & ~(size_t)127;
}

__host__ __device__ inline int half_up(int n) { return (n + 1) / 2; }

// one CTA holding the whole replica: `rows` = colour phases whose first draws are made in one batch
__host__ __device__ inline Sizes sizes_single(const RepDesc& D, int cap, int nwarps, int rows, int pre_ev, int prec)
{
    Sizes z;
    z.words = 3 * (int64_t)D.L[2] * D.L[1] * D.row_words;
    z.nfl = D.nf[0] * D.nf[1] * D.nf[2];
    z.maxc = half_up(D.nf[0]) * half_up(D.nf[1]) * half_up(D.nf[2]);
    z.cap = cap;
    z.nwarps = nwarps;
    z.ltot = D.L[0] + D.L[1] + D.L[2];
    z.lz = 0;
    z.rows = rows;
    z.pre_ev = pre_ev;
    z.prec = prec;
    z.kslots = D.kslots == 4 ? 4 : (D.kslots == LONG_SLOTS ? LONG_SLOTS : KSLOTS);
    z.btab = D.btab_smem ? BOLTZ_LO + D.bhi_len : 0;
    return z;
}

// one CTA of a cluster: rows = 2 (the phase's first draws and the next phase's)
__host__ __device__ inline Sizes sizes_cluster(const RepDesc& D, const ClusterPlan& P, int cap, int nwarps, int pre_ev,
                                               int prec)
{
    Sizes z;
    z.words = (int64_t)3 * P.zs * D.L[1] * D.row_words;
    z.nfl = P.nfl;
    z.maxc = half_up(D.nf[0]) * half_up(D.nf[1]) * half_up(P.nfl / (D.nf[0] * D.nf[1]));
    z.cap = cap;
    z.nwarps = nwarps;
    z.ltot = D.L[0] + D.L[1] + D.L[2];
    z.lz = D.L[2];
    z.rows = 2;
    z.pre_ev = pre_ev;
    z.prec = prec;
    z.kslots = D.kslots == 4 ? 4 : (D.kslots == LONG_SLOTS ? LONG_SLOTS : KSLOTS);
    z.btab = D.btab_smem ? BOLTZ_LO + D.bhi_len : 0;
    return z;
}

__device__ __forceinline__ Layout carve(unsigned char* dyn, const Sizes& z)
{
    size_t o[NARR];
    layout_bytes(z, o);
    Layout L;
    L.occ = reinterpret_cast<uint32_t*>(dyn + o[0]);
    L.lim = dyn + o[1];
    L.box = reinterpret_cast<uint2*>(dyn + o[2]);
    L.flist = reinterpret_cast<uint16_t*>(dyn + o[3]);
    L.act = reinterpret_cast<uint32_t*>(dyn + o[4]);
    L.pre_xs = reinterpret_cast<uint64_t*>(dyn + o[5]);
    L.pre_E = dyn + o[6];
    L.pre_row = reinterpret_cast<uint16_t*>(dyn + o[7]);
    L.dlist = reinterpret_cast<uint16_t*>(dyn + o[8]);
    L.frag_of_c = reinterpret_cast<uint16_t*>(dyn + o[9]);
    L.zmap = reinterpret_cast<uint32_t*>(dyn + o[10]);
    L.wkey = reinterpret_cast<uint32_t*>(dyn + o[11]);
    L.wvac = reinterpret_cast<uint32_t*>(dyn + o[12]);
    L.wtype = reinterpret_cast<int8_t*>(dyn + o[13]);
    L.wlog = reinterpret_cast<uint64_t*>(dyn + o[16]);
    L.btab = reinterpret_cast<double*>(dyn + o[17]);
    L.stale = dyn + o[14];
    L.slots = reinterpret_cast<uint32_t*>(dyn + o[15]);
    return L;
}

// lattice and slab sizes, in registers
struct Geo {
    int L0, L1, L2, RW, nf0, nf1;
    int zb, zl;   // this CTA's z cells: [zb, zb + zl)
    int fzb;      // its first fragment layer
    uint32_t me;  // its rank
};

// a neighbour of a site: coordinates, site type, dz + 1
struct NbSite {
    int t2, x, y, z, dz1;
};

// This lane's direction q = lane & 7 for the three site types: 10 bits each,
// t2 | (dc_x+1) << 2 | (dc_y+1) << 4 | (dc_z+1) << 6 | (d_z+1) << 8.
__device__ __forceinline__ uint32_t pack_direction(const NbTable& nbt, int q)
{
    uint32_t p = 0;
#pragma unroll
    for (int t = 0; t < 3; ++t) {
        const NbEntry e = nbt.e[t][q];
        p |= ((uint32_t)e.t2 | (uint32_t)(e.dc[0] + 1) << 2 | (uint32_t)(e.dc[1] + 1) << 4 |
              (uint32_t)(e.dc[2] + 1) << 6 | (uint32_t)(e.d[2] + 1) << 8)
             << (10 * t);
    }
    return p;
}

// c in [-1, L] to [0, L): the least of c, c + L and c - L as unsigned numbers
__device__ __forceinline__ int wrap1(int c, int L)
{
    return (int)min(min((unsigned)c, (unsigned)(c + L)), (unsigned)(c - L));
}

__device__ __forceinline__ NbSite nb_site(const Geo& g, uint32_t dirs, uint32_t key)
{
    int t, x, y, z;
    split32(key, t, x, y, z);
    const uint32_t e = dirs >> (10 * t);
    NbSite s;
    s.t2 = (int)(e & 3u);
    s.x = wrap1(x + (int)((e >> 2) & 3u) - 1, g.L0);
    s.y = wrap1(y + (int)((e >> 4) & 3u) - 1, g.L1);
    s.z = wrap1(z + (int)((e >> 6) & 3u) - 1, g.L2);
    s.dz1 = (int)((e >> 8) & 3u);
    return s;
}

// word of a site in its CTA's slab: index for a slab-local z
__device__ __forceinline__ int word_of(const Geo& g, int t, int x, int y, int zr)
{
    return ((zr * g.L1 + y) * g.RW + (x >> 4)) * 3 + t;
}

// species code of a site; a site in another CTA's slab is read through
// distributed shared memory
template <bool CL>
__device__ __forceinline__ int site_code(const Layout& S, const Geo& g, int t, int x, int y, int z)
{
    uint32_t w;
    const int zr = CL ? z - g.zb : z;
    if (!CL || (unsigned)zr < (unsigned)g.zl) {
        w = S.occ[word_of(g, t, x, y, zr)];
    } else {
        const uint32_t zm = S.zmap[z];
        w = (uint32_t)ld_peer(peer_addr(S.occ + word_of(g, t, x, y, (int)((zm >> 8) & 1023u)), zm & 255u));
    }
    return (int)((w >> occ_shift(x)) & 3u);
}

// marks the fragment owning a site as changed, unless it is this CTA's fragment
// `own`; `came`: a vacancy came to that site
template <int PREC, bool CL>
__device__ __forceinline__ void mark_owner(const Layout& S, const Geo& g, int x, int y, int z, int own, bool came)
{
    using Lim = Limit<PREC>;
    typename Lim::T* lim = reinterpret_cast<typename Lim::T*>(S.lim);
    const int fx = S.frag_of_c[x], fy = S.frag_of_c[g.L0 + y];
    if constexpr (!CL) {
        const int f = ((int)S.frag_of_c[g.L0 + g.L1 + z] * g.nf1 + fy) * g.nf0 + fx;
        if (f != own) {
            lim[f] = Lim::DIRTY;
            if (came) S.stale[f] = 1;
        }
    } else {
        const uint32_t zm = S.zmap[z];
        const int f = ((int)(zm >> 18) * g.nf1 + fy) * g.nf0 + fx;
        if ((zm & 255u) == g.me) {
            if (f != own) {
                lim[f] = Lim::DIRTY;
                if (came) S.stale[f] = 1;
            }
        } else {
            if constexpr (PREC == 1) st_peer(peer_addr(lim + f, zm & 255u), Lim::DIRTY);
            else st_peer64(peer_addr(lim + f, zm & 255u), Lim::DIRTY);
            if (came) st_peer8(peer_addr(S.stale + f, zm & 255u), 1);
        }
    }
}

// site index (within the replica) of a shell partner: packed SiteOff {t2, dc[3]} of a cell
__device__ __forceinline__ int shell_lin(const Geo& g, int off, int x, int y, int z)
{
    const int t2 = (int)(int8_t)off;
    const int px = wrapc(x + (int)(int8_t)(off >> 8), g.L0), py = wrapc(y + (int)(int8_t)(off >> 16), g.L1),
              pz = wrapc(z + (int)(int8_t)(off >> 24), g.L2);
    return ((t2 * g.L2 + pz) * g.L1 + py) * g.L0 + px;
}

// a cell of the interval [c - r, c + 1 + r] or [c - 1 - r, c + r] around the cells c and j of a
// hop (j = c or a neighbour, periodic): its lower end (p = 0), c (1) or its upper end (2)
__device__ __forceinline__ int box_cell(int c, int j, int p, int r, int L)
{
    if (p == 1) return c;
    int d = j - c;
    d = d > 1 ? -1 : (d < -1 ? 1 : d);
    int v = p == 0 ? c + min(d, 0) - r : c + max(d, 0) + r;
    while (v < 0) v += L;
    while (v >= L) v -= L;
    return v;
}

// index of a site in the site -> record map: sixteen entries per occupancy word
__device__ __forceinline__ uint32_t map_index(const Geo& g, uint32_t key)
{
    int t, x, y, z;
    split32(key, t, x, y, z);
    return (uint32_t)word_of(g, t, x, y, z) * 16u + (uint32_t)(x & 15);
}

// The vacancies of a box (first cell lo, extents ex, ey, ez) in site order: their
// keys to wkey[0 .. min(n, cap)), the number n returned.  Lane l scans rows
// [RPL l, RPL (l + 1)) of the box, three words (site types) per row; with at
// most one vacancy per lane and type the slots follow from three ballots,
// else from a scan of the packed counts.
template <typename M>
__device__ __forceinline__ int gather_rows(const Layout& S, const Geo& g, uint32_t* wkey, int cap, int lane, int lo0,
                                           int lo1, int lo2, int ex, int ey, int rows, int rpl)
{
    constexpr unsigned FULL = 0xffffffffu;
    const unsigned below = (1u << lane) - 1u;
    // masks of up to 16 or 32 cells, bit 2 c for cell c: row c / ex of this lane's rows, x = lo0 + c % ex
    const int r = rpl * lane;
    int z = (int)(((float)r + 0.5f) * __fdividef(1.0f, (float)ey));  // r / ey, exact for r < 2^19
    int y = r - z * ey;
    const int dy = y, dz = z;
    const M emask = ex == 16 ? (M)0xffffffffu : (M)((1u << (2 * ex)) - 1u);
    const int off = (lo0 & 15) * 2;
    const bool two = off + 2 * ex > 32;
    M m[3] = {0, 0, 0};
    for (int k = 0; k < rpl; ++k) {
        if (r + k < rows) {
            const uint32_t* w = S.occ + word_of(g, 0, lo0, lo1 + y, lo2 - g.zb + z);
#pragma unroll
            for (int t = 0; t < 3; ++t) {
                const uint32_t v = two ? __funnelshift_r(w[t], w[3 + t], off) : w[t] >> off;
                m[t] |= ((M)((v >> 1) & ~v & 0x55555555u) & emask) << (2 * ex * k);
            }
        }
        if (++y == ey) {
            y = 0;
            ++z;
        }
    }
    auto count = [](M v) { return sizeof(M) == 8 ? __popcll(v) : __popc((unsigned)v); };
    int s0, s1, s2, n;
    if (!__any_sync(FULL, ((m[0] & (m[0] - 1)) | (m[1] & (m[1] - 1)) | (m[2] & (m[2] - 1))) != 0)) {
        const unsigned b0 = __ballot_sync(FULL, m[0] != 0), b1 = __ballot_sync(FULL, m[1] != 0),
                       b2 = __ballot_sync(FULL, m[2] != 0);
        const int n0 = __popc(b0), n1 = __popc(b1);
        s0 = __popc(b0 & below);
        s1 = n0 + __popc(b1 & below);
        s2 = n0 + n1 + __popc(b2 & below);
        n = n0 + n1 + __popc(b2);
    } else {
        const uint32_t mine = (uint32_t)count(m[0]) | (uint32_t)count(m[1]) << 10 | (uint32_t)count(m[2]) << 20;
        uint32_t c = mine;  // at most 32 lanes x 16 (or 31) cells per field: the last may carry out unused
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t u = __shfl_up_sync(FULL, c, o);
            if (lane >= o) c += u;
        }
        const uint32_t tot = __shfl_sync(FULL, c, 31);
        c -= mine;
        const int n0 = (int)(tot & 1023u), n1 = (int)((tot >> 10) & 1023u);
        s0 = (int)(c & 1023u);
        s1 = n0 + (int)((c >> 10) & 1023u);
        s2 = n0 + n1 + (int)(c >> 20);
        n = n0 + n1 + (int)(tot >> 20);
    }
    // one vacancy per turn and lane, over the three masks
    int t = 0;
    while (true) {
        while (t < 3 && m[0] == 0) {  // the next type with a vacancy left
            m[0] = m[1];
            m[1] = m[2];
            m[2] = 0;
            s0 = s1;
            s1 = s2;
            ++t;
        }
        if (t >= 3) break;
        const int c = (sizeof(M) == 8 ? __ffsll((long long)m[0]) - 1 : __ffs((int)m[0]) - 1) >> 1;
        m[0] &= m[0] - 1;
        int yy = dy, zz = dz, xx = c;
        while (xx >= ex) {
            xx -= ex;
            if (++yy == ey) {
                yy = 0;
                ++zz;
            }
        }
        if (s0 < cap) wkey[s0] = key32(t, lo0 + xx, lo1 + yy, lo2 + zz);
        ++s0;
    }
    __syncwarp();
    return n;
}

__device__ __forceinline__ int gather(const Layout& S, const Geo& g, uint32_t* wkey, int cap, int lane, int lo0, int lo1,
                                      int lo2, int ex, int ey, int ez)
{
    constexpr unsigned FULL = 0xffffffffu;
    const int rows = ey * ez, rpl = (rows + 31) >> 5;
    // (at most 31 cells per lane keep every count of the packed scan below 1024)
    if (rpl * ex <= 16) return gather_rows<uint32_t>(S, g, wkey, cap, lane, lo0, lo1, lo2, ex, ey, rows, rpl);
    if (rpl * ex <= 31 && ex <= 16)
        return gather_rows<uint64_t>(S, g, wkey, cap, lane, lo0, lo1, lo2, ex, ey, rows, rpl);
    // larger boxes: a lane takes 16-cell pieces of rows, all three site types at once; the
    // keys go to wkey as they are found and are put into site order by rank.  (One type
    // after the other, in order: 96^3 cells in 12^3-cell fragments at 0.001 vacancies per
    // site, most of whose visits scan, 102 us per window, now 86.)
    const int pieces = (ex + 15) >> 4, items = rows * pieces;
    int n = 0;
    for (int base = 0; base < items; base += 32) {
        const int it = base + lane;
        uint32_t m[3] = {0, 0, 0};
        int x0 = 0, y = 0, z = 0;
        if (it < items) {
            const int r = pieces == 1 ? it : it / pieces, p = it - r * pieces;
            z = (int)(((float)r + 0.5f) * __fdividef(1.0f, (float)ey));  // r / ey, exact for r < 2^19
            y = lo1 + r - z * ey;
            z += lo2;
            x0 = lo0 + 16 * p;
            const int len = min(16, lo0 + ex - x0), off = (x0 & 15) * 2;
            const uint32_t* w = S.occ + word_of(g, 0, x0, y, z - g.zb);
            const bool two = off + 2 * len > 32;
            const uint32_t mask = 0x55555555u & (uint32_t)((1ull << (2 * len)) - 1ull);
#pragma unroll
            for (int t = 0; t < 3; ++t) {
                const uint32_t v = __funnelshift_r(w[t], two ? w[3 + t] : 0u, off);
                m[t] = (v >> 1) & ~v & mask;
            }
        }
        const int c = __popc(m[0]) + __popc(m[1]) + __popc(m[2]);
        const unsigned some = __ballot_sync(FULL, c != 0);
        if (!some) continue;
        int slot;
        if (!__any_sync(FULL, c > 1)) {
            slot = n + __popc(some & ((1u << lane) - 1u));
            n += __popc(some);
        } else {
            int s = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(FULL, s, o);
                if (lane >= o) s += u;
            }
            slot = n + s - c;
            n += __shfl_sync(FULL, s, 31);
        }
#pragma unroll
        for (int t = 0; t < 3; ++t)
            while (m[t]) {
                const int b = (__ffs(m[t]) - 1) >> 1;
                m[t] &= m[t] - 1;
                if (slot < cap) wkey[slot] = key32(t, x0 + b, y, z);
                ++slot;
            }
    }
    __syncwarp();
    const int have = min(n, cap);  // at most RESIDENT_MAX_SLOTS = 64: two keys per lane
    const uint32_t k0 = lane < have ? wkey[lane] : DEAD, k1 = lane + 32 < have ? wkey[lane + 32] : DEAD;
    int r0 = 0, r1 = 0;
    for (int q = 0; q < have; ++q) {
        const uint32_t v = wkey[q];
        r0 += v < k0 ? 1 : 0;
        r1 += v < k1 ? 1 : 0;
    }
    __syncwarp();
    if (k0 != DEAD) wkey[r0] = k0;
    if (k1 != DEAD) wkey[r1] = k1;
    __syncwarp();
    return n;
}

// u = floor(x / 2^11) 2^-53, exact, from integer instructions
__device__ __forceinline__ double uniform53(uint64_t x)
{
    const uint64_t u = x >> 11;
    if (u == 0) return 0.0;
    const int n = 63 - __clzll((long long)u);
    return __longlong_as_double((long long)(((u << (52 - n)) & 0x000fffffffffffffull) | ((uint64_t)(n + 970) << 52)));
}

// A positive double as a float, truncated, from integer instructions; exponents
// in [-100, 100] only.
__device__ __forceinline__ bool float_range(long long b) { return (unsigned)((int)(b >> 52) - 923) <= 200u; }
__device__ __forceinline__ float to_float(long long b)
{
    return __uint_as_float((uint32_t)((b - (896ll << 52)) >> 29));
}

// The screen's limit for a fragment of event total `tot` (> 0): no less than any
// first variate E that does not put the first event past the window.  Mixed:
// fl(E / S32) > theta' whenever E > S32 theta' (1 + 2^-20), lim32 the factor
// theta' (1 + 2^-20) rounded up; plain: fl(E / R) > tau whenever E exceeds
// fl(tau R) by 2^-40.
template <int PREC>
__device__ __forceinline__ typename Limit<PREC>::T limit_of(uint64_t tot, float lim32, double tau)
{
    if constexpr (PREC == 1) return __float_as_uint(__fmul_ru(u64_to_float_rn(tot), lim32));
    else return (uint64_t)__double_as_longlong(__dmul_rn(tau, __longlong_as_double((long long)tot))) + 4096ull;
}

// warp total of u64 values below 2^63 / 32: three 21-bit limbs by warp reductions
__device__ __forceinline__ unsigned long long warp_total(unsigned long long v)
{
    constexpr unsigned FULL = 0xffffffffu;
    const unsigned a = __reduce_add_sync(FULL, (unsigned)v & 0x1fffffu);
    const unsigned b = __reduce_add_sync(FULL, (unsigned)(v >> 21) & 0x1fffffu);
    const unsigned c = __reduce_add_sync(FULL, (unsigned)(v >> 42));
    return (unsigned long long)a + ((unsigned long long)b << 21) + ((unsigned long long)c << 42);
}

}  // namespace

size_t resident_smem_bytes(const RepDesc& D, int cap, int threads, int pre_g, int pre_ev, int prec)
{
    const Sizes z = sizes_single(D, cap, threads / 32, 1, 2, prec);
    if (D.L[0] > 1024 || D.L[1] > 1024 || D.L[2] > 1024 || z.nfl > 65535 || 8 * z.maxc > 32767)
        return ~(size_t)0;  // compact keys, 16-bit fragment and row indices
    if (pre_g < 1 || pre_g > 8 || (8 % pre_g) != 0 || (pre_ev != 2 && pre_ev != 4 && pre_ev != 8)) return ~(size_t)0;
    return layout_bytes(sizes_single(D, cap, threads / 32, pre_g, pre_ev, prec), nullptr);
}

size_t cluster_smem_bytes(const RepDesc& D, const ClusterPlan& p, int cap, int pre_ev, int prec)
{
    return layout_bytes(sizes_cluster(D, p, cap, CLUSTER_THREADS / 32, pre_ev, prec), nullptr);
}

// Put before a launch to let another one take its SMs first.
__global__ void k_gate() {}

// First draws of the plain form, one window after the other: event ev of
// fragment f of window w0 + z at ((z frag_tot + draw_off + f) ev_per + ev).
// The FP64 logarithm (some 45 FP64 instructions at 64 cycles of an SM quarter's
// FP64 pipe each) would keep the few SMs that hold a plain replica busy for
// longer than the events themselves; here the whole GPU computes it, beside
// the windows before.
__global__ void __launch_bounds__(64) k_draws(const RepDesc* __restrict__ descs, int nrep, uint64_t w0, int ev_per,
                                              int64_t frag_tot, Draw* draws)
{
    const int nbk = ev_per >> 1;
    for (int r = blockIdx.y; r < nrep; r += gridDim.y) {
        const RepDesc& D = descs[r];
        if (!D.resident) continue;
        const int64_t n = (int64_t)D.nf[0] * D.nf[1] * D.nf[2] * nbk;
        const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
        if (i >= n) continue;
        const int64_t fid = i / nbk;
        const int bk = (int)(i - fid * nbk);
        const U64x4 b = philox4x64((uint64_t)fid, D.window + w0 + blockIdx.z, (uint64_t)bk, 0, D.seed,
                                   key_word(D.replica, PURPOSE_HOP));
        Draw* o = draws + ((int64_t)blockIdx.z * frag_tot + D.draw_off + fid) * ev_per + 2 * bk;
        o[0].E = neglog64(b.x[0]);
        o[0].xs = b.x[1];
        o[1].E = neglog64(b.x[2]);
        o[1].xs = b.x[3];
    }
}

// LONG: replicas of the launch may have lists of LONG_SLOTS (kept out of the others' code:
// the branch alone costs them 2%)
template <int PREC, int NT, bool CL, bool SITE, bool LONG>
__global__ void __launch_bounds__(NT, (NT <= 128 ? 4 : (NT <= 256 ? 2 : 1)))
    k_resident(const RepDesc* __restrict__ descs, const int32_t* __restrict__ reps,
               const ClusterPlan* __restrict__ plans, uint64_t w0, uint64_t windows, uint32_t* occ, VacRec* recs,
               VacRec* tmp, uint32_t* vmap, int32_t* counts, int32_t* tracer, unsigned long long* stats,
               uint32_t* status, int cap, NbTable nbt, const Draw* __restrict__ draws, int64_t frag_tot, int draw_ev,
               uint32_t stuck_wait_us, ResCache rc, SiteArgs sa)
{
    static_assert(!SITE || PREC == 0, "site energies use the plain form");
    extern __shared__ __align__(128) unsigned char dyn[];
    __shared__ Shared sh;
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t me = CL ? cluster_ctarank() : 0u;

    if (tid == 0) {
        int r;
        if constexpr (CL) {
            sh.P = plans[blockIdx.x / cluster_nctas()];
            r = sh.P.rep;
        } else {
            r = reps[blockIdx.x];
        }
        sh.D = descs[r];
        if constexpr (!CL) {
            sh.P.rep = r;
            sh.P.ncta = 1;
            sh.P.fz0[0] = 0;
            sh.P.fz0[1] = sh.D.nf[2];
        }
        for (int c = 0; c <= sh.P.ncta; ++c) sh.zbeg[c] = frag_start(sh.P.fz0[c], sh.D.base[2], sh.D.rem[2]);
        for (int k = 0; k < 9; ++k) {
            if constexpr (PREC == 1) sh.rate[k] = k < 6 ? sh.D.q[k] : 0ull;
            else sh.rate[k] = k < 6 ? (uint64_t)__double_as_longlong(sh.D.k64[k]) : 0ull;
        }
        sh.nact[0] = sh.nact[1] = 0;
        sh.ndraw = 0;
        sh.next_act[0] = sh.next_act[1] = NW;  // each warp's first fragment is its own index
        sh.hops = 0;
        sh.hand = 0;
        sh.abort = 0;
        sh.cached = rc.valid[r];
    }
    __syncthreads();
    const RepDesc& D = sh.D;
    const ClusterPlan& P = sh.P;
    const int rep = P.rep;
    const int pre_ev = D.pre_ev == 8 ? 8 : (D.pre_ev == 4 ? 4 : 2);
    const int pre_g = CL ? 2 : ((D.pre_g == 2 || D.pre_g == 4 || D.pre_g == 8) ? D.pre_g : 1);
    const Sizes sz = CL ? sizes_cluster(D, P, cap, NW, pre_ev, PREC) : sizes_single(D, cap, NW, pre_g, pre_ev, PREC);
    const Layout S = carve(dyn, sz);
    using Lim = Limit<PREC>;
    typename Lim::T* const lim = reinterpret_cast<typename Lim::T*>(S.lim);
    const int maxc = sz.maxc, ks = sz.kslots;
    const int fzb = P.fz0[me], fze = P.fz0[me + 1];
    const Geo geo{D.L[0], D.L[1], D.L[2], D.row_words, D.nf[0], D.nf[1], sh.zbeg[me], sh.zbeg[me + 1] - sh.zbeg[me],
                  fzb, me};
    const int nfl = (fze - fzb) * D.nf[0] * D.nf[1];
    const int64_t frag0 = D.frag_base + (int64_t)fzb * D.nf[1] * D.nf[0];  // layers are contiguous in the global order

    // ---- stage in: this CTA's occupancy (its z cells are contiguous in the global
    // layout) by TMA bulk copies, the record index of every vacancy's site
    const int slab_words = geo.zl * D.L[1] * D.row_words * 3;
    const int slab_word0 = geo.zb * D.L[1] * D.row_words * 3;
    uint32_t* const occ_g = occ + D.occ_word_off + (int64_t)geo.zb * D.L[1] * D.row_words * 3;
    const uint32_t occ_bytes = (uint32_t)slab_words * 4u;  // rows are multiples of 16 bytes
    if (tid == 0) {
        mbar_init(&sh.bar, 1);
        mbar_arrive_expect_tx(&sh.bar, occ_bytes);
        const char* src = reinterpret_cast<const char*>(occ_g);
        for (uint32_t off = 0; off < occ_bytes; off += BULK_CHUNK)
            bulk_g2s(S.occ + off / 4, src + off, min(BULK_CHUNK, occ_bytes - off), &sh.bar);
    }
    for (int k = tid; k < D.L[0] + D.L[1] + D.L[2]; k += NT) {
        const int d = k < D.L[0] ? 0 : (k < D.L[0] + D.L[1] ? 1 : 2);
        const int c = d == 0 ? k : (d == 1 ? k - D.L[0] : k - D.L[0] - D.L[1]);
        S.frag_of_c[k] = (uint16_t)frag_of(c, D.base[d], D.rem[d]);
    }
    if constexpr (CL) {
        for (int z = tid; z < D.L[2]; z += NT) {
            const int fz = frag_of(z, D.base[2], D.rem[2]);
            int c = 0;
            while (c + 1 < P.ncta && P.fz0[c + 1] <= fz) ++c;
            S.zmap[z] = (uint32_t)c | ((uint32_t)(z - sh.zbeg[c]) << 8) | ((uint32_t)(fz - P.fz0[c]) << 18);
        }
    }
    // this CTA's fragments by colour
    auto colour_count = [&](int colour, int cnt[2], int& lz0) -> int {
        const int b0 = colour & 1, b1 = (colour >> 1) & 1, b2 = colour >> 2;
        cnt[0] = D.nf[0] == 1 ? (b0 == 0 ? 1 : 0) : D.nf[0] / 2;
        cnt[1] = D.nf[1] == 1 ? (b1 == 0 ? 1 : 0) : D.nf[1] / 2;
        lz0 = D.nf[2] == 1 ? 0 : (fzb + ((fzb & 1) != b2 ? 1 : 0));
        const int nlz = D.nf[2] == 1 ? (b2 == 0 ? 1 : 0) : (fze > lz0 ? (fze - lz0 + 1) / 2 : 0);
        return cnt[0] * cnt[1] * nlz;
    };
    if (tid == 0) {
        int s = 0;
        for (int c = 0; c < 8; ++c) {
            int cnt[2], lz0;
            sh.coff[c] = s;
            s += colour_count(c, cnt, lz0);
        }
        sh.coff[8] = s;
    }
    __syncthreads();
    if constexpr (SITE) {
        for (int k = tid; k < sz.btab; k += NT) S.btab[k] = sa.btab[D.btab_off + k];
    }
    for (int lf = tid; lf < nfl; lf += NT) {
        const int q = lf / D.nf[0], f0 = lf - q * D.nf[0], lz = q / D.nf[1], f1 = q - lz * D.nf[1], f2 = fzb + lz;
        const int c = (f0 & 1) | (f1 & 1) << 1 | (f2 & 1) << 2;
        // its place in its colour: this CTA's first layer of the colour is fzb or the next one
        const int l = ((f2 - fzb) / 2 * half_up(D.nf[1] - (c >> 1 & 1)) + f1 / 2) * half_up(D.nf[0] - (c & 1)) + f0 / 2;
        S.flist[sh.coff[c] + l] = (uint16_t)lf;
        const int o0 = frag_start(f0, D.base[0], D.rem[0]), e0 = frag_start(f0 + 1, D.base[0], D.rem[0]) - o0;
        const int o1 = frag_start(f1, D.base[1], D.rem[1]), e1 = frag_start(f1 + 1, D.base[1], D.rem[1]) - o1;
        const int o2 = frag_start(f2, D.base[2], D.rem[2]), e2 = frag_start(f2 + 1, D.base[2], D.rem[2]) - o2;
        S.box[lf] = make_uint2((uint32_t)o0 | (uint32_t)o1 << 10 | (uint32_t)o2 << 20,
                               (uint32_t)(e0 - 1) | (uint32_t)(e1 - 1) << 10 | (uint32_t)(e2 - 1) << 20);
    }
    // sites of this slab count from vmap_s, sites of the replica from vmap_r
    uint32_t* const vmap_r = vmap + D.vmap_off;
    uint32_t* const vmap_s = vmap_r + (int64_t)geo.zb * D.L[1] * D.row_words * 48;
    VacRec* const recs_r = recs + D.frag_base * cap;  // record indices count from here
    const uint32_t rec_lim = (uint32_t)(D.nf[0] * D.nf[1] * D.nf[2] * cap);
    // one thread per fragment, its next count on the way while it is staged and four records at a time
    int c_next = tid < nfl ? counts[frag0 + tid] : 0;
    for (int f = tid; f < nfl; f += NT) {
        const int64_t g = frag0 + f;
        const int c = c_next;
        if (f + NT < nfl) c_next = counts[g + NT];
        if (c > cap) atomicOr(status, STATUS_OVERFLOW);
        uint32_t* const sl = S.slots + f * ks;
        for (int k = 0; k < ks; ++k) sl[k] = DEAD;
        const uint32_t at = (uint32_t)((g - D.frag_base) * cap);
        for (int k0 = 0; k0 < c && k0 < cap; k0 += 4) {
            uint64_t k64[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (k0 + u < c) k64[u] = recs[g * cap + k0 + u].key;  // (cap is a multiple of 8)
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (k0 + u < c) {
                    int t, x, y, z;
                    split_key(k64[u], t, x, y, z);
                    vmap_s[map_index(geo, key32(t, x, y, z - geo.zb))] = at + k0 + u;
                    if (k0 + u < ks) sl[k0 + u] = key32(t, x, y, z);  // the first visit sorts them
                }
        }
        if (c > ks) sl[0] = UNLISTED;
        S.stale[f] = 0;
        // the limit the last launch left, where nothing changed the replica since
        lim[f] = sh.cached ? (typename Lim::T)rc.lim[g] : (c > 0 ? Lim::DIRTY : Lim::EMPTY);
    }
    if (!mbar_wait_bounded(&sh.bar, 0, WAIT_NS)) {
        if (tid == 0) {
            atomicOr(status, STATUS_TIMEOUT);
            sh.abort = 1;
        }
        mbar_wait_bounded(&sh.bar, 0, WAIT_NS);  // let copies in flight land before leaving
    }
    __syncthreads();
    if (!CL && stuck_wait_us && !sh.abort) {
        // test of the bounded wait: no copy is in flight here, and the barrier
        // below is never completed, so the wait must give up after
        // stuck_wait_us, report FKMC_ETIMEOUT and leave the state untouched
        if (tid == 0) mbar_init(&sh.bar_test, 1);
        __syncthreads();
        const bool done = mbar_wait_bounded(&sh.bar_test, 0, (uint64_t)stuck_wait_us * 1000ull);
        if (!done && tid == 0) {
            atomicOr(status, STATUS_TIMEOUT);
            sh.abort = 1;
        }
        __syncthreads();
    }
    if constexpr (CL) {
        // every slab is in place before any CTA reads a peer's; the CTAs of a cluster
        // stop together: a CTA whose stage-in timed out tells all
        const bool bad = sh.abort != 0;
        cluster_sync();
        if (bad && tid < P.ncta) st_peer8(peer_addr(&sh.abort, (uint32_t)tid), 1);
        cluster_sync();
    }
    if (sh.abort) return;

    const uint64_t hop_k1 = key_word(D.replica, PURPOSE_HOP);
    const uint64_t th = window_bits(D.theta_tau, D.F);  // mixed form
    const double tau = D.tau;                           // plain form
    const float lim32 = __double2float_ru(__dmul_ru(__longlong_as_double((long long)th), 1.0 + 0x1p-20));
    const uint32_t dirs = pack_direction(nbt, lane & 7);
    uint32_t* const wkey = S.wkey + warp * cap;
    uint32_t* const wvac = S.wvac + warp * cap;
    int8_t* const wtype = S.wtype + warp * cap * 8;
    uint64_t* const wlog = S.wlog + warp * 2 * CLOCK_LOG;
    unsigned long long my_hops = 0, my_hand = 0;

    const uint32_t key0 = key32(0, 0, 0, geo.zb);  // a site of this slab
    const int frag_off = fzb * geo.nf1 * geo.nf0;  // fragment index of local fragment 0
    // first draws of local fragment lf, events 0 .. pre_ev - 1, at offset o: part k, one
    // Philox block (mixed) or one event (plain: a copy of what k_draws computed);
    // they depend on no fragment's state
    const int per = PREC == 1 ? pre_ev >> 1 : pre_ev;
    const int sh_per = per == 8 ? 3 : (per == 4 ? 2 : (per == 2 ? 1 : 0));
    auto draw = [&](int lf, uint64_t wk, int o, int k) {
        const int fid = frag_off + lf;
        if constexpr (PREC == 1) {
            const U64x4 b = philox4x64((uint64_t)fid, D.window + w0 + wk, (uint64_t)k, 0, D.seed, hop_k1);
            float* E = reinterpret_cast<float*>(S.pre_E);
            E[o + 2 * k] = neglog32(b.x[0]);
            E[o + 2 * k + 1] = neglog32(b.x[2]);
            S.pre_xs[o + 2 * k] = b.x[1];
            S.pre_xs[o + 2 * k + 1] = b.x[3];
        } else {
            const int4 d = __ldg(
                reinterpret_cast<const int4*>(draws + ((int64_t)wk * frag_tot + D.draw_off + fid) * draw_ev + k));
            reinterpret_cast<uint64_t*>(S.pre_E)[o + k] = (uint64_t)(uint32_t)d.x | (uint64_t)(uint32_t)d.y << 32;
            S.pre_xs[o + k] = (uint64_t)(uint32_t)d.z | (uint64_t)(uint32_t)d.w << 32;
        }
    };
    // cluster: of every fragment of a colour, to row `row`
    auto draw_colour = [&](int colour, uint64_t wk, int row) {
        const int c0 = sh.coff[colour], n = sh.coff[colour + 1] - c0;
        for (int it = tid; it < n << sh_per; it += NT)
            draw(S.flist[c0 + (it >> sh_per)], wk, (row * maxc + (it >> sh_per)) * pre_ev, it & (per - 1));
    };
    // rate type and neighbour key of this lane's direction (no event for a dead slot, without a branch)
    auto type_of = [&](uint32_t key, uint32_t& nkey) -> int {
        const bool dead = key == DEAD;
        const NbSite s = nb_site(geo, dirs, dead ? key0 : key);
        nkey = key32(s.t2, s.x, s.y, s.z);
        const int ty = site_code<CL>(S, geo, s.t2, s.x, s.y, s.z) * 3 + s.dz1;
        return dead ? NO_EVENT : ty;
    };
    auto rate_of = [&](int ty) -> uint64_t { return sh.rate[ty]; };
    // site energies: FP64 rate of the event of type ty from the site of key k to that of key nk in this
    // lane's direction: the table rate times the two Boltzmann factors of the energy difference, in the
    // order of the colour-phase kernel.  Field words come from L2: the exchanges update them by atomics.
    const int32_t* const field_r = SITE ? sa.field + D.site_off : nullptr;
    const double* const blo = SITE ? (sz.btab ? S.btab : sa.btab + D.btab_off) : nullptr;
    auto site_rate = [&](int& ty, uint32_t k, uint32_t nk) -> uint64_t {
        if (ty >= NO_EVENT) return 0ull;
        int t, x, y, z, t2, jx, jy, jz;
        split32(k, t, x, y, z);
        split32(nk, t2, jx, jy, jz);
        const int32_t Es = __ldcg(field_r + ((t * geo.L2 + z) * geo.L1 + y) * geo.L0 + x);
        const int32_t Ej = __ldcg(field_r + ((t2 * geo.L2 + jz) * geo.L1 + jy) * geo.L0 + jx);
        int32_t dm = Ej - sa.e_self - Es;
        if (sa.g_elec) dm -= __ldg(sa.g_elec + 24 * D.replica + 8 * t + (lane & 7));
        const int h = D.bhi_mid + (dm >> 9);
        if (h < 0 || h >= D.bhi_len) {  // outside the bound the tables were built for: report, no event
            atomicOr(status, STATUS_ENERGY_RANGE);
            ty = NO_EVENT;
            return 0ull;
        }
        return (uint64_t)__double_as_longlong(
            __dmul_rn(__dmul_rn(__longlong_as_double((long long)sh.rate[ty]), blo[BOLTZ_LO + h]), blo[dm & 511]));
    };
    // moves a vacancy's share of the energy field from the site of key k to that of key nk (every lane a
    // part); integer atomics: fragments of one colour may touch the same word
    auto move_share = [&](uint32_t k, uint32_t nk) {
        int t, x, y, z, t2, jx, jy, jz;
        split32(k, t, x, y, z);
        split32(nk, t2, jx, jy, jz);
        int32_t* const fw = sa.field + D.site_off;
        for (int o = lane; o < sa.n_vv; o += 32) {
            const int2 a = __ldg(reinterpret_cast<const int2*>(sa.vv + t * SITE_MAX_VV + o));
            const int2 c = __ldg(reinterpret_cast<const int2*>(sa.vv + t2 * SITE_MAX_VV + o));
            atomicAdd(fw + shell_lin(geo, a.x, x, y, z), -a.y);
            atomicAdd(fw + shell_lin(geo, c.x, jx, jy, jz), c.y);
        }
    };
    // inclusive prefix over the lanes, strides 1, 2, .. 16; with values in the first `len` lanes only
    // the strides below len (the others add zeros to those lanes)
    auto scan64 = [&](uint64_t v, int len = 32) -> uint64_t {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            if (o >= 8 && o >= len) break;
            const uint64_t u = __shfl_up_sync(FULL, (unsigned long long)v, o);
            if (lane >= o) {
                if constexpr (PREC == 1) v += u;
                else v = (uint64_t)__double_as_longlong(
                         __dadd_rn(__longlong_as_double((long long)v), __longlong_as_double((long long)u)));
            }
        }
        return v;
    };
    auto add = [&](uint64_t a, uint64_t b) -> uint64_t {
        if constexpr (PREC == 1) return a + b;
        else return (uint64_t)__double_as_longlong(
                 __dadd_rn(__longlong_as_double((long long)a), __longlong_as_double((long long)b)));
    };

    uint32_t ph = 0;  // phases of this launch so far
    for (uint64_t wk = 0; wk < windows; ++wk) {
        const uint64_t w = D.window + w0 + wk;
        if ((wk & 63) == 0) {  // colour orders of the next 64 windows, one thread each
            if (tid < 64 && wk + tid < windows) sh.perms[tid] = colour_perm_packed(D.seed, D.replica, w + tid);
            __syncthreads();
        }
        const uint32_t wperm = sh.perms[wk & 63];
        for (int p = 0; p < 8; ++p, ++ph) {
            const int colour = (int)((wperm >> (4 * p)) & 15u);
            const int par = (int)(ph & 1u);
            if constexpr (CL) {
                if (p == 0 && (wk & 63) == 0) {  // otherwise drawn at the end of the phase before
                    draw_colour(colour, wk, par);
                    __syncthreads();
                }
            } else if ((p & (pre_g - 1)) == 0) {
                // of the next pre_g phases at once, for the fragments that hold an event now: a
                // list of them, then one thread per part of their draws (an empty fragment that
                // receives a vacancy meanwhile draws for itself)
                for (int it = tid; it < pre_g * maxc; it += NT) {
                    const int pp = it / maxc, l = it - pp * maxc;
                    const int col = (int)((wperm >> (4 * (p + pp))) & 15u);
                    if (l >= sh.coff[col + 1] - sh.coff[col]) continue;
                    const int lf = S.flist[sh.coff[col] + l];
                    unsigned r = NO_ROW;
                    const typename Lim::T m = lim[lf];
                    if (m != Lim::EMPTY) {
                        r = (unsigned)atomicAdd(&sh.ndraw, 1);
                        // the limit is about the expected number of events: below 1/4 a third is rare
                        if (PREC == 0 || m >= 0x3e800000u) r |= ROW_FULL;
                        S.dlist[r & ~ROW_FULL] = (uint16_t)lf;
                    }
                    S.pre_row[lf] = (uint16_t)r;
                }
                __syncthreads();
                const int nd = sh.ndraw << sh_per;
                for (int it = tid; it < nd; it += NT) {
                    const int lf = S.dlist[it >> sh_per], k = it & (per - 1);
                    if (PREC == 1 && k > 0 && !(S.pre_row[lf] & ROW_FULL)) continue;
                    draw(lf, wk, (it >> sh_per) * pre_ev, k);
                }
                __syncthreads();
                if (tid == 0) sh.ndraw = 0;
            }
            // ---- screen: one thread per fragment of the colour
            const int c0 = sh.coff[colour], ncol = sh.coff[colour + 1] - c0;
            for (int l = tid; l < ncol; l += NT) {
                const int lf = S.flist[c0 + l];
                const typename Lim::T m = lim[lf];
                bool active = m == Lim::DIRTY;
                if (active && S.stale[lf] == 0) {  // marked, but without a vacancy?
                    bool none = true;
                    for (int q = 0; q < ks; ++q) none = none && S.slots[lf * ks + q] == DEAD;
                    if (none) {
                        lim[lf] = Lim::EMPTY;
                        active = false;
                    }
                }
                if (!active && m != Lim::EMPTY && m != Lim::DIRTY) {
                    const int o = (CL ? par * maxc + l : (int)(S.pre_row[lf] & (ROW_FULL - 1u))) * pre_ev;
                    if constexpr (PREC == 1) active = reinterpret_cast<const float*>(S.pre_E)[o] <= __uint_as_float(m);
                    else active = reinterpret_cast<const uint64_t*>(S.pre_E)[o] <= m;  // positive doubles
                }
                if (active) S.act[atomicAdd(&sh.nact[par], 1)] = (uint32_t)lf | (uint32_t)l << 16;
            }
            __syncthreads();
            if (tid == 0) {  // the next phase's counters
                sh.nact[par ^ 1] = 0;
                sh.next_act[par ^ 1] = NW;
            }
            // ---- run: one warp per listed fragment; each warp's first by its index, then as they become free
            const int nact = sh.nact[par];
            for (int a = warp; a < nact;) {
                const uint32_t ent = S.act[a];
                const int lf = (int)(ent & 0xffffu);
                const unsigned prow = CL ? (unsigned)(par * maxc) + (ent >> 16) : (unsigned)S.pre_row[lf];
                const int o0 = (int)(CL ? prow : prow & (ROW_FULL - 1u)) * pre_ev;
                // events drawn ahead
                const int n_pre = CL || (prow & ROW_FULL) ? (!CL && prow == NO_ROW ? 0 : pre_ev) : 2;
                const uint2 bx = S.box[lf];
                const int lo0 = (int)(bx.x & 1023u), lo1 = (int)((bx.x >> 10) & 1023u), lo2 = (int)(bx.x >> 20);
                const int ex = (int)(bx.y & 1023u) + 1, ey = (int)((bx.y >> 10) & 1023u) + 1, ez = (int)(bx.y >> 20) + 1;
                // the fragment's vacancies: its list, or, where it changed from outside or is too long
                // for one, a scan of its rows.  Up to two chunks (8 vacancies) each lane keeps the site
                // keys of its two events' slots, their rate types and their targets' keys in registers
                uint32_t* const sl = S.slots + lf * ks;
                uint32_t kc0 = sl[lane >> 3], kc1 = ks > 4 ? sl[4 + (lane >> 3)] : DEAD;
                const bool scan = S.stale[lf] != 0 || __shfl_sync(FULL, kc0, 0) == UNLISTED;
                // key of slot lane & 7 (up to two chunks)
                auto slot_key = [&]() -> uint32_t {
                    const uint32_t u = __shfl_sync(FULL, kc0, (lane & 3) * 8), v = __shfl_sync(FULL, kc1, (lane & 3) * 8);
                    return lane & 4 ? v : u;
                };
                int n = 0;
                bool sorted = false;
                if (LONG && !scan && ks == LONG_SLOTS) {  // with more than eight entries: by rank to wkey
                    const uint32_t k = lane < LONG_SLOTS ? sl[lane] : DEAD;
                    const unsigned held = __ballot_sync(FULL, k != DEAD);
                    if (held >> KSLOTS) {
                        int r = 0;
#pragma unroll
                        for (int q = 0; q < LONG_SLOTS; ++q) r += __shfl_sync(FULL, k, q) < k ? 1 : 0;
                        if (k != DEAD) wkey[r] = k;
                        __syncwarp();
                        n = __popc(held);
                        sorted = true;
                    }
                }
                if (!scan && !sorted) {
                    n = __popc(__ballot_sync(FULL, kc0 != DEAD) & 0x01010101u) +
                        __popc(__ballot_sync(FULL, kc1 != DEAD) & 0x01010101u);
                    // the last visit left its slots' order: into site order where its exchanges changed it
                    const uint32_t k = slot_key();
                    const uint32_t up = __shfl_up_sync(FULL, k, 1);
                    if (__any_sync(FULL, (lane & 7) > 0 && up > k)) {
                        int r = 0;
#pragma unroll
                        for (int q = 0; q < KSLOTS; ++q) r += __shfl_sync(FULL, k, q) < k ? 1 : 0;
                        if (lane < KSLOTS && k != DEAD) wkey[r] = k;
                        __syncwarp();
                        const int m = lane >> 3;
                        kc0 = m < n ? wkey[m] : DEAD;
                        kc1 = m + 4 < n ? wkey[m + 4] : DEAD;
                    }
                } else {
                    if (scan) n = gather(S, geo, wkey, cap, lane, lo0, lo1, lo2, ex, ey, ez);
                    if (n > cap) {
                        if (lane == 0) atomicOr(status, STATUS_OVERFLOW);
                        n = cap;
                    }
                    const int m = lane >> 3;
                    kc0 = m < n ? wkey[m] : DEAD;
                    kc1 = m + 4 < n ? wkey[m + 4] : DEAD;
                }
                const int nch = (n + 3) >> 2;
                // record index of slot `lane` (beyond 32 slots: through wvac); used at the first exchange
                uint32_t vrec = 0;
                if (nch <= 2) {
                    const uint32_t k = slot_key();
                    if (lane < n) vrec = __ldcg(vmap_r + map_index(geo, k));
                } else {
                    if (lane < n) vrec = __ldcg(vmap_r + map_index(geo, wkey[lane]));
                    if (n > 32)
                        for (int k = lane; k < n; k += 32) wvac[k] = __ldcg(vmap_r + map_index(geo, wkey[k]));
                }
                uint32_t nk0 = 0, nk1 = 0;
                int ty0 = NO_EVENT, ty1 = NO_EVENT;
                uint64_t sr0 = 0, sr1 = 0;  // site energies: the rates
                auto compute_types = [&]() {
                    if (nch <= 2) {
                        ty0 = type_of(kc0, nk0);
                        if (nch == 2) ty1 = type_of(kc1, nk1);
                        if constexpr (SITE) {
                            sr0 = site_rate(ty0, kc0, nk0);
                            if (nch == 2) sr1 = site_rate(ty1, kc1, nk1);
                        }
                    } else {
                        for (int c = 0; c < nch; ++c) {
                            const int e = c * 32 + lane, m = e >> 3;
                            int ty = NO_EVENT;
                            uint32_t nk;
                            if (m < n && wkey[m] != DEAD) ty = type_of(wkey[m], nk);
                            wtype[e] = (int8_t)ty;
                        }
                        __syncwarp();
                    }
                };
                // rate of event c * 32 + lane beyond two chunks (site energies: computed again)
                auto rate_at = [&](int c) -> uint64_t {
                    int ty = wtype[c * 32 + lane];
                    if constexpr (SITE) {
                        const int m = (c * 32 + lane) >> 3;
                        uint32_t nk = 0;
                        if (ty < NO_EVENT) type_of(wkey[m], nk);
                        return site_rate(ty, ty < NO_EVENT ? wkey[m] : key0, nk);
                    } else {
                        return rate_of(ty);
                    }
                };
                compute_types();

                // mixed: mixed_clock's; plain: FP64 bits, of the events before `logged0`, those from
                // there on in the log (E, R), and an FP32 estimate of the whole in units of tau
                uint64_t clock = 0;
                bool fp = false;
                int logged0 = 0;
                float xclock = 0.0f;
                uint64_t i = 0, batch = ~0ull;
                uint64_t xs_even = 0, xs_odd = 0, E_even = 0, E_odd = 0;
                uint64_t tot = 0;
                // the last exchange's record: its slot (-1: none), the target's entry of the map
                // (lane 1), the displacement (lanes 0..2), and the exchanged ion's displacement
                // (lanes 8..10).  Written at the next exchange or at the end of the visit, when the
                // record index and the ion's displacement have long arrived.
                int pend_m = -1, pend_at = 0, pend_d = 0;
                int trv = 0;
                int64_t trs = 0, trj = 0;
                auto flush = [&]() {
                    if (pend_m < 0) return;
                    const uint32_t v = n <= 32 ? __shfl_sync(FULL, vrec, pend_m & 31) : wvac[pend_m];
                    if (v >= rec_lim) {  // a vacancy without a record: not a state this library wrote
                        if (lane == 0) atomicOr(status, STATUS_OVERFLOW);
                    } else {
                        if (lane == 1) vmap_r[pend_at] = v;
                        if (lane < 3 && pend_d != 0) atomicAdd(&recs_r[v].d[lane], pend_d);
                    }
                    if (tracer && lane >= 8 && lane < 11) {
                        tracer[trs] = trv;
                        tracer[trj] = 0;
                    }
                };
                for (;;) {
                    // the total of the fragment's events; the plain form's scans, in the canonical
                    // order, give the inclusive prefixes that the selection needs besides
                    uint64_t inc0 = 0, inc1 = 0;
                    bool nz0 = false, nz1 = false;  // plain: this lane's events have a rate
                    if (nch <= 2) {
                        inc0 = SITE ? sr0 : rate_of(ty0);
                        inc1 = nch == 2 ? (SITE ? sr1 : rate_of(ty1)) : 0ull;
                        if constexpr (PREC == 1) {
                            tot = warp_total(inc0 + inc1);
                        } else {
                            nz0 = inc0 != 0ull;
                            nz1 = inc1 != 0ull;
                            const int len = n <= 2 ? 8 * max(n, 1) : 32;
                            inc0 = scan64(inc0, len);
                            tot = __shfl_sync(FULL, inc0, len - 1);
                            if (nch == 2) {
                                inc1 = add(tot, scan64(inc1));
                                tot = __shfl_sync(FULL, inc1, 31);
                            }
                        }
                    } else if constexpr (PREC == 1) {
                        unsigned long long part = 0;
                        for (int c = 0; c < nch; ++c) part += rate_at(c);
                        tot = warp_total(part);
                    } else {
                        tot = 0;
                        for (int c = 0; c < nch; ++c)
                            tot = __shfl_sync(FULL, add(tot, scan64(rate_at(c))), 31);
                    }
                    if (tot == 0ull) break;
                    if (i >= MAX_EVENTS_PER_PHASE) {
                        if (lane == 0) atomicOr(status, STATUS_EVENT_LIMIT);
                        break;
                    }
                    uint64_t xs, Eb;
                    if (i < (uint64_t)n_pre) {  // drawn ahead
                        xs = S.pre_xs[o0 + (int)i];
                        if constexpr (PREC == 1) Eb = reinterpret_cast<const uint32_t*>(S.pre_E)[o0 + (int)i];
                        else Eb = reinterpret_cast<const uint64_t*>(S.pre_E)[o0 + (int)i];
                    } else {
                        // events [64 b, 64 b + 64) come from blocks 32 b + lane (those drawn ahead
                        // are computed again, unused)
                        const uint64_t k = i;
                        if ((k >> 6) != batch) {
                            batch = k >> 6;
                            const U64x4 blk =
                                philox4x64((uint64_t)(frag_off + lf), w, 32 * batch + lane, 0, D.seed, hop_k1);
                            xs_even = blk.x[1];
                            xs_odd = blk.x[3];
                            if constexpr (PREC == 1) {
                                E_even = __float_as_uint(neglog32(blk.x[0]));
                                E_odd = __float_as_uint(neglog32(blk.x[2]));
                            } else {
                                E_even = (uint64_t)__double_as_longlong(neglog64(blk.x[0]));
                                E_odd = (uint64_t)__double_as_longlong(neglog64(blk.x[2]));
                            }
                        }
                        const int src = (int)((k >> 1) & 31);
                        const bool odd = (k & 1) != 0;
                        xs = __shfl_sync(FULL, odd ? xs_odd : xs_even, src);
                        Eb = __shfl_sync(FULL, odd ? E_odd : E_even, src);
                    }
                    // the window test, and the selection (no side effects) beside it
                    uint64_t nclock = 0;
                    bool past;
                    uint64_t target;
                    if constexpr (PREC == 1) {
                        past = mixed_clock(clock, fp, __fdiv_rn(__uint_as_float((uint32_t)Eb), u64_to_float_rn(tot)), th,
                                           nclock);
                        target = __umul64hi(xs, tot);
                    } else {
                        // clock + fl(E / R) > tau, the clock the rounded sum of the events before.  An
                        // estimate of clock / tau in FP32 (each term E / fl(tau R) to 2^-20, 2^12 of them
                        // at most) decides unless it comes within 2^-10 of 1; then the divisions are done,
                        // those of the events before from the log.  (A division is some ten FP64
                        // instructions, each 64 cycles of the SM quarter's FP64 pipe.)
                        const double R = __longlong_as_double((long long)tot);
                        const long long pb = __double_as_longlong(__dmul_rn(tau, R));
                        float est = 2.0f;  // out of the estimate's range: exact
                        bool sure = float_range((long long)Eb) && float_range(pb) && i < 4096;
                        if (sure) {
                            est = xclock + __fdividef(to_float((long long)Eb), to_float(pb));
                            sure = fabsf(est - 1.0f) > 0x1p-10f;
                            past = est > 1.0f;
                        }
                        const int left = (int)i - logged0;
                        if (!sure || left == CLOCK_LOG) {
                            double c = __longlong_as_double((long long)clock);
                            for (int q = 0; q < left; ++q)
                                c = __dadd_rn(c, __ddiv_rn(__longlong_as_double((long long)wlog[2 * q]),
                                                           __longlong_as_double((long long)wlog[2 * q + 1])));
                            clock = (uint64_t)__double_as_longlong(c);
                            logged0 = (int)i;
                            if (!sure) {
                                c = __dadd_rn(c, __ddiv_rn(__longlong_as_double((long long)Eb), R));
                                past = c > tau;
                                if (!past) {
                                    clock = (uint64_t)__double_as_longlong(c);
                                    logged0 = (int)i + 1;
                                    xclock = __double2float_rn(__ddiv_rn(c, tau));
                                }
                            }
                            __syncwarp();
                        }
                        if (sure && !past) {
                            if (lane == 0) {
                                wlog[2 * ((int)i - logged0)] = Eb;
                                wlog[2 * ((int)i - logged0) + 1] = tot;
                            }
                            __syncwarp();
                            xclock = est;
                        }
                        nclock = clock;
                        // doubles >= 0 compare as their bits
                        target = (uint64_t)__double_as_longlong(__dmul_rn(uniform53(xs), R));
                    }
                    if (past) break;
                    if constexpr (PREC == 1) {  // the prefixes, only for an event that happens
                        if (nch <= 2) {
                            inc0 = scan64(inc0, n <= 2 ? 8 * n : 32);
                            if (nch == 2) inc1 = __shfl_sync(FULL, inc0, 31) + scan64(inc1);
                        }
                    }
                    // first event whose inclusive prefix exceeds the target (plain: among the events of
                    // nonzero rate, and the last of those where rounding left no prefix above it)
                    int e_sel = -1;
                    if (nch <= 2) {
                        const bool h0 = inc0 > target && (PREC == 1 || nz0);
                        const bool h1 = nch == 2 && inc1 > target && (PREC == 1 || nz1);
                        const unsigned b0 = __ballot_sync(FULL, h0), b1 = __ballot_sync(FULL, h1);
                        e_sel = b0 ? __ffs(b0) - 1 : (b1 ? 32 + __ffs(b1) - 1 : -1);
                        if (PREC == 0 && e_sel < 0) {
                            const unsigned l0 = __ballot_sync(FULL, nz0), l1 = __ballot_sync(FULL, nz1);
                            e_sel = l1 ? 63 - __clz(l1) : 31 - __clz(l0);
                        }
                    } else {
                        uint64_t carry = 0;
                        for (int c = 0; c < nch && e_sel < 0; ++c) {
                            const uint64_t v = rate_at(c);
                            const uint64_t inc = add(carry, scan64(v));
                            const unsigned bal = __ballot_sync(FULL, inc > target && (PREC == 1 || v != 0ull));
                            if (bal) e_sel = c * 32 + __ffs(bal) - 1;
                            carry = __shfl_sync(FULL, inc, 31);
                        }
                        if (PREC == 0) {
                            for (int c = nch - 1; c >= 0 && e_sel < 0; --c) {
                                const unsigned bal = __ballot_sync(FULL, rate_at(c) != 0ull);
                                if (bal) e_sel = c * 32 + 31 - __clz(bal);
                            }
                        }
                    }
                    if (e_sel < 0) {  // cannot happen: the target lies below the total
                        if (lane == 0) atomicOr(status, STATUS_OVERFLOW);
                        break;
                    }
                    // the exchange: site s, its target j, the ion
                    const int m = e_sel >> 3;
                    uint32_t ks_, kj;
                    int ty;
                    if (nch <= 2) {
                        const bool c1 = e_sel >= 32;
                        ks_ = __shfl_sync(FULL, c1 ? kc1 : kc0, e_sel & 31);
                        kj = __shfl_sync(FULL, c1 ? nk1 : nk0, e_sel & 31);
                        ty = __shfl_sync(FULL, c1 ? ty1 : ty0, e_sel & 31);
                    } else {
                        ks_ = wkey[m];
                        uint32_t nk;
                        type_of(ks_, nk);
                        kj = __shfl_sync(FULL, nk, e_sel & 7);
                        ty = wtype[e_sel];
                    }
                    // even lanes compute s's addresses, odd lanes j's
                    int tk, xk, yk, zk;
                    split32((lane & 1) ? kj : ks_, tk, xk, yk, zk);
                    const int wg = word_of(geo, tk, xk, yk, zk);  // word within the replica
                    if (lane < 2) {
                        const uint32_t flip = ((uint32_t)SP_V ^ (ty >= 3 ? (uint32_t)SP_H : (uint32_t)SP_O))
                                              << occ_shift(xk);
                        const int wl = CL ? wg - slab_word0 : wg;
                        if (!CL || (unsigned)wl < (unsigned)slab_words) {
                            atomicXor(S.occ + wl, flip);
                        } else {
                            const uint32_t zm = S.zmap[zk];
                            red_peer_xor(peer_addr(S.occ + word_of(geo, tk, xk, yk, (int)((zm >> 8) & 1023u)), zm & 255u),
                                         flip);
                        }
                    }
                    const bool own_lane = (unsigned)(xk - lo0) < (unsigned)ex && (unsigned)(yk - lo1) < (unsigned)ey &&
                                          (unsigned)(zk - lo2) < (unsigned)ez;
                    const bool owned = __shfl_sync(FULL, (int)own_lane, 1) != 0;
                    flush();  // the exchange before
                    {
                        // displacement in units of a/2 along this lane's axis
                        const int ts = (int)(ks_ >> 30), tj = (int)(kj >> 30);
                        const uint32_t e = __shfl_sync(FULL, dirs, e_sel & 7) >> (10 * ts);
                        const int ax = lane & 3;  // 0..2
                        pend_m = m;
                        pend_at = wg * 16 + (xk & 15);
                        pend_d = 2 * ((int)((e >> (2 + 2 * ax)) & 3u) - 1) + (tj == ax) - (ts == ax);
                        if (tracer) {
                            const int lin = ((tk * geo.L2 + zk) * geo.L1 + yk) * geo.L0 + xk;
                            const int ls = __shfl_sync(FULL, lin, 0), lj = __shfl_sync(FULL, lin, 1);
                            if (lane >= 8 && lane < 11) {
                                trj = 3 * (D.site_off + lj) + ax;
                                trs = 3 * (D.site_off + ls) + ax;
                                trv = __ldcg(tracer + trj) - pend_d;
                            }
                        }
                    }
                    if constexpr (SITE) {
                        if (sa.n_vv > 0) {
                            move_share(ks_, kj);
                            __threadfence_block();  // before the rate reads
                        }
                    }
                    __syncwarp();  // the exchanged codes are in place
                    const uint32_t nk = owned ? kj : DEAD;
                    if (nch <= 2) {  // the moved vacancy's lanes follow it (or drop a handed-off slot)
                        if ((lane >> 3) == m) kc0 = nk;
                        if ((lane >> 3) + 4 == m) kc1 = nk;
                    } else {
                        if (lane == 0) wkey[m] = nk;
                        __syncwarp();
                    }
                    my_hand += !owned;
                    {
                        // the fragments whose totals changed: owners of the vacancies next to the two
                        // changed sites (lanes 0-7 look around s, 8-15 around j; 16-31 repeat them
                        // without marking, so that no branch splits the warp)
                        // (with up to two vacancies lanes 16-31, which hold no event, do it beside the
                        // rate types of lanes 0-15)
                        const uint32_t pk = (lane & 8) ? kj : ks_;
                        NbSite c;
                        int code;
                        if (!SITE && n <= 2) {
                            const bool dead = kc0 == DEAD;
                            const uint32_t k = lane < 16 ? (dead ? key0 : kc0) : pk;
                            c = nb_site(geo, dirs, k);
                            nk0 = key32(c.t2, c.x, c.y, c.z);
                            code = site_code<CL>(S, geo, c.t2, c.x, c.y, c.z);
                            ty0 = lane < 16 && !dead ? code * 3 + c.dz1 : NO_EVENT;
                            if (lane < 16) code = SP_O;
                        } else {
                            c = nb_site(geo, dirs, pk);
                            code = site_code<CL>(S, geo, c.t2, c.x, c.y, c.z);
                            if (lane >= 16) code = SP_O;
                            compute_types();
                        }
                        if (code == SP_V)
                            mark_owner<PREC, CL>(S, geo, c.x, c.y, c.z, lf, key32(c.t2, c.x, c.y, c.z) == kj);
                        if constexpr (SITE) {
                            // the energy field changed within the shells' reach of s and j, so every rate of
                            // a vacancy one cell further did: the owners of the cells at -r, 0 and +r around
                            // the two sites (fragment edges exceed r, so no fragment lies between those)
                            if (sa.reach > 0 && lane < 27) {
                                int t, x, y, z, t2, jx, jy, jz;
                                split32(ks_, t, x, y, z);
                                split32(kj, t2, jx, jy, jz);
                                const int px = lane % 3, py = (lane / 3) % 3, pz = lane / 9;
                                mark_owner<PREC, CL>(S, geo, box_cell(x, jx, px, sa.reach, geo.L0),
                                                     box_cell(y, jy, py, sa.reach, geo.L1),
                                                     box_cell(z, jz, pz, sa.reach, geo.L2), lf, false);
                            }
                        }
                    }
                    clock = nclock;
                    ++i;
                }
                flush();
                if (lane == 0) {
                    lim[lf] = tot == 0ull ? Lim::EMPTY : limit_of<PREC>(tot, lim32, tau);
                    my_hops += i;
                    if (scan) S.stale[lf] = 0;
                }
                if (i > 0 || scan) {  // the fragment's list, in slot order
                    if (LONG && n > KSLOTS && n <= ks) {
                        if (lane < ks) sl[lane] = lane < n ? wkey[lane] : DEAD;
                    } else if (n <= ks) {
                        const uint32_t k = slot_key();
                        if (lane < ks) sl[lane] = !LONG || lane < KSLOTS ? k : DEAD;
                    } else if (lane == 0) {
                        sl[0] = UNLISTED;
                    }
                }
                if (nact <= NW) break;  // every listed fragment has its warp
                if (lane == 0) a = atomicAdd(&sh.next_act[par], 1);
                a = __shfl_sync(FULL, a, 0);
            }
            if constexpr (CL) {
                // every write of the phase, local and remote, is visible after the wait; between
                // arrival and wait the next phase's first draws
                __syncwarp();
                cluster_arrive();
                if (p < 7)
                    draw_colour((int)((wperm >> (4 * (p + 1))) & 15u), wk, par ^ 1);
                else if (wk + 1 < windows && ((wk + 1) & 63) != 0)  // the next window's order is known
                    draw_colour((int)(sh.perms[(wk + 1) & 63] & 15u), wk + 1, par ^ 1);
                __syncwarp();
                cluster_wait();
                __syncthreads();  // the draws of this CTA's other threads, made after their arrival
            } else {
                __syncthreads();
            }
        }
    }

    // ---- stage out: occupancy by TMA bulk stores; each fragment's records from
    // where they lay to tmp, and back to its list once every CTA has read its own
    if (tid == 0) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        char* dst = reinterpret_cast<char*>(occ_g);
        for (uint32_t off = 0; off < occ_bytes; off += BULK_CHUNK)
            bulk_s2g(dst + off, S.occ + off / 4, min(BULK_CHUNK, occ_bytes - off));
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    }
    VacRec* const tmp_r = tmp + (D.tmp_off + (int64_t)fzb * D.nf[1] * D.nf[0]) * cap;
    // a record: key and id | displacement, as three words
    auto index_of = [&](uint32_t key) -> uint32_t { return min(__ldcg(vmap_r + map_index(geo, key)), rec_lim - 1); };
    auto put_copy = [&](int f, int slot, uint32_t key, int2 d01, int2 d2id) {
        int t, x, y, z;
        split32(key, t, x, y, z);
        VacRec& o = tmp_r[(int64_t)f * cap + slot];
        o.key = make_key(t, x, y, z);
        *reinterpret_cast<int2*>(&o.d[0]) = d01;
        *reinterpret_cast<int2*>(&o.d[2]) = d2id;
    };
    static_assert(sizeof(VacRec) == 24 && offsetof(VacRec, d) == 8 && offsetof(VacRec, id) == 20, "copied as words");
    // A valid list gives a fragment's vacancies; a fragment without one is scanned for it
    // first, or, where a list cannot hold them, copied at once.  (A scan of every fragment,
    // and the chain vmap - record - copy for one fragment of a warp after the other, made a
    // call of one window take 166 us on 64^3 cells in 2^3-cell fragments and 68 on 32^3 in
    // 4^3-cell ones, now 65 and 41 at 0.001 vacancies per site.)
    for (int f0 = warp; f0 < nfl; f0 += 32 * NW) {
        const int f = f0 + NW * lane;
        bool todo = f < nfl && (S.stale[f] != 0 || S.slots[f * ks] == UNLISTED);
        if (LONG && f < nfl)
            for (int q = KSLOTS; q < ks; ++q) todo = todo || S.slots[f * ks + q] != DEAD;  // more than the copies below take
        for (unsigned td = __ballot_sync(FULL, todo); td; td &= td - 1) {
            const int fs = f0 + NW * (__ffs(td) - 1);
            const uint2 bx = S.box[fs];
            int n = gather(S, geo, wkey, cap, lane, (int)(bx.x & 1023u), (int)((bx.x >> 10) & 1023u), (int)(bx.x >> 20),
                           (int)(bx.y & 1023u) + 1, (int)((bx.y >> 10) & 1023u) + 1, (int)(bx.y >> 20) + 1);
            if (n > cap) {
                if (lane == 0) atomicOr(status, STATUS_OVERFLOW);
                n = cap;
            }
            const bool listed = n <= KSLOTS && n <= ks;
            if (listed) {
                if (lane < ks) S.slots[fs * ks + lane] = lane < n ? wkey[lane] : DEAD;
            } else {
                for (int m = lane; m < n; m += 32) {
                    const VacRec* src = recs_r + index_of(wkey[m]);
                    put_copy(fs, m, wkey[m], __ldcg(reinterpret_cast<const int2*>(&src->d[0])),
                             __ldcg(reinterpret_cast<const int2*>(&src->d[2])));
                }
                if (lane == 0) S.stale[fs] = (uint8_t)n;  // more than a list holds: copied
            }
            __syncwarp();
            if (listed && lane == 0) S.stale[fs] = 0;
            __syncwarp();
        }
    }
    __syncthreads();
    for (int f = tid; f < nfl; f += NT) {  // one thread per fragment, the reads of four records in flight
        int n = S.stale[f];
        if (n == 0) {
            uint32_t key[KSLOTS];
#pragma unroll
            for (int q = 0; q < KSLOTS; ++q) {
                key[q] = q < ks ? S.slots[f * ks + q] : DEAD;
                n += key[q] != DEAD ? 1 : 0;
            }
            if (n > 0) {
#pragma unroll
                for (int q0 = 0; q0 < KSLOTS; q0 += 4) {
                    uint32_t at[4];
                    int2 d01[4], d2id[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) at[u] = key[q0 + u] != DEAD ? index_of(key[q0 + u]) : 0u;
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (key[q0 + u] != DEAD) {
                            d01[u] = __ldcg(reinterpret_cast<const int2*>(&recs_r[at[u]].d[0]));
                            d2id[u] = __ldcg(reinterpret_cast<const int2*>(&recs_r[at[u]].d[2]));
                        }
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (key[q0 + u] != DEAD) {
                            int r = 0;  // its place in site order
#pragma unroll
                            for (int q = 0; q < KSLOTS; ++q) r += key[q] < key[q0 + u] ? 1 : 0;
                            put_copy(f, r, key[q0 + u], d01[u], d2id[u]);
                        }
                }
            }
        }
        counts[frag0 + f] = n;
        S.stale[f] = (uint8_t)n;  // for the move back
        rc.lim[frag0 + f] = (uint64_t)lim[f];
    }
    if (my_hand && lane == 0) atomicAdd(&sh.hand, my_hand);
    if (my_hops) atomicAdd(&sh.hops, my_hops);
    if constexpr (CL) cluster_sync();
    else __syncthreads();
    for (int f = tid; f < nfl; f += NT) {
        const int n = S.stale[f];
        const VacRec* const from = tmp_r + (int64_t)f * cap;
        VacRec* const to = recs + (frag0 + f) * cap;
        for (int k0 = 0; k0 < n; k0 += 4) {  // (cap is a multiple of 8)
            VacRec r[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (k0 + u < n) r[u] = from[k0 + u];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (k0 + u < n) to[k0 + u] = r[u];
        }
    }
    if (tid == 0) {
        if (sh.hops) atomicAdd(stats + 2 * rep, sh.hops);
        if (sh.hand) atomicAdd(stats + 2 * rep + 1, sh.hand);
        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
    if constexpr (CL) cluster_sync();  // no CTA leaves while a peer may still address it
    if (tid == 0 && me == 0) rc.valid[rep] = 1;
}

// `nc` CTAs of one z-slab of fragment layers each, or false where they do not fit
static bool cluster_plan_for(const RepDesc& D, int cap, int pre_ev, int prec, int nc, ClusterPlan* out)
{
    const int nf2 = D.nf[2];
    if (D.L[0] > 1024 || D.L[1] > 1024 || D.L[2] > 1024 || nc < 2 || nc > CLUSTER_MAX_CTAS || nc > nf2) return false;
    ClusterPlan p{};
    p.ncta = nc;
    int zs = 0, layers = 0;
    for (int c = 0; c <= nc; ++c) p.fz0[c] = (int)((int64_t)c * nf2 / nc);
    for (int c = 0; c < nc; ++c) {
        const int z0 = p.fz0[c] * D.base[2] + std::min(p.fz0[c], D.rem[2]);
        const int z1 = p.fz0[c + 1] * D.base[2] + std::min(p.fz0[c + 1], D.rem[2]);
        zs = std::max(zs, z1 - z0);
        layers = std::max(layers, p.fz0[c + 1] - p.fz0[c]);
    }
    p.zs = zs;
    p.nfl = layers * D.nf[0] * D.nf[1];
    if (p.nfl > 65535) return false;  // 16-bit fragment indices
    if (cluster_smem_bytes(D, p, cap, pre_ev, prec) > RESIDENT_MAX_SMEM) return false;
    *out = p;
    return true;
}

bool make_cluster_plan(const RepDesc& D, int cap, int pre_ev, int prec, int min_ctas, int max_ctas, ClusterPlan* out)
{
    for (int nc = std::min(max_ctas, CLUSTER_MAX_CTAS); nc >= std::max(2, min_ctas); --nc)
        if (cluster_plan_for(D, cap, pre_ev, prec, nc, out)) return true;
    return false;
}

using ResidentFn = void (*)(const RepDesc*, const int32_t*, const ClusterPlan*, uint64_t, uint64_t, uint32_t*, VacRec*,
                            VacRec*, uint32_t*, int32_t*, int32_t*, unsigned long long*, uint32_t*, int, NbTable,
                            const Draw*, int64_t, int, uint32_t, ResCache, SiteArgs);

template <int PREC, bool SITE, bool LONG = false>
static ResidentFn resident_variant(int threads, bool cluster)
{
    if (cluster) return k_resident<PREC, CLUSTER_THREADS, true, SITE, LONG>;
    if (threads == 128) return k_resident<PREC, 128, false, SITE, LONG>;
    if (threads == 256) return k_resident<PREC, 256, false, SITE, LONG>;
    return k_resident<PREC, 512, false, SITE, LONG>;
}

// form: 0 plain, 1 mixed, 2 plain with site energies, 3 mixed with long lists
static ResidentFn resident_kernel(int form, int threads, bool cluster)
{
    if (form == 1) return resident_variant<1, false>(threads, cluster);
    if (form == 3) return resident_variant<1, false, true>(threads, cluster);
    return form == 2 ? resident_variant<0, true>(threads, cluster) : resident_variant<0, false>(threads, cluster);
}

cudaError_t resident_prepare()
{
    cudaError_t e = cudaSuccess;
    for (int form = 0; form < 4; ++form) {
        for (int threads : {128, 256, 512})
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(resident_kernel(form, threads, false),
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RESIDENT_MAX_SMEM);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(resident_kernel(form, 0, true), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)RESIDENT_MAX_SMEM);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(resident_kernel(form, 0, true), cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    }
    return e;
}

static cudaLaunchConfig_t cluster_config(int nclusters, int ncta, size_t smem, cudaStream_t st,
                                         cudaLaunchAttribute* attr)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(nclusters * ncta));
    cfg.blockDim = dim3(CLUSTER_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = (unsigned)ncta;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

int cluster_fits(int form, int ncta, size_t smem)
{
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = cluster_config(1, ncta, smem, nullptr, attr);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, resident_kernel(form, 0, true), &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

cudaError_t launch_gate(cudaStream_t st)
{
    k_gate<<<1, 32, 0, st>>>();
    return cudaGetLastError();
}

cudaError_t launch_draws(const RepDesc* d_descs, int nrep, int64_t max_frag, uint64_t w0, int windows, int ev_per,
                         int64_t frag_tot, Draw* draws, cudaStream_t st)
{
    const int64_t n = max_frag * (ev_per / 2);
    const dim3 grid((unsigned)((n + 63) / 64), (unsigned)std::min(nrep, 65535), (unsigned)windows);
    k_draws<<<grid, 64, 0, st>>>(d_descs, nrep, w0, ev_per, frag_tot, draws);
    return cudaGetLastError();
}

cudaError_t launch_resident(int form, const ResidentArgs& a, const int32_t* d_reps, int nreps, size_t smem, int threads,
                            uint64_t w0, uint64_t windows, const Draw* draws, cudaStream_t st)
{
    if (nreps <= 0) return cudaSuccess;
    resident_kernel(form, threads, false)<<<nreps, threads, smem, st>>>(
        a.descs, d_reps, nullptr, w0, windows, a.occ, a.recs, a.tmp, a.vmap, a.counts, a.tracer, a.stats, a.status,
        a.cap, a.nbt, draws, a.frag_tot, a.draw_ev, a.stuck_wait_us, a.rc, a.sa);
    return cudaGetLastError();
}

cudaError_t launch_cluster(int form, const ResidentArgs& a, const ClusterPlan* d_plans, int nplans, int ncta,
                           size_t smem, uint64_t w0, uint64_t windows, const Draw* draws, cudaStream_t st)
{
    if (nplans <= 0) return cudaSuccess;
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = cluster_config(nplans, ncta, smem, st, attr);
    return cudaLaunchKernelEx(&cfg, resident_kernel(form, 0, true), a.descs, (const int32_t*)nullptr, d_plans, w0,
                              windows, a.occ, a.recs, a.tmp, a.vmap, a.counts, a.tracer, a.stats, a.status, a.cap,
                              a.nbt, draws, a.frag_tot, a.draw_ev, a.stuck_wait_us, a.rc, a.sa);
}

}  // namespace fkmc
