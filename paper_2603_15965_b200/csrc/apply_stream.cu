// Grouped LoRA shrink -> expand for calls below the tcgen05 crossover (Eq. 2, Section 3.3 step 4), bf16, one launch.
//
// A work item is (projection, tile of <= 16 or 32 positions of one segment) and belongs to a cluster of S CTAs (S = 1, 2, 4
// or 8).  Each CTA streams its share of the tile's x columns and of A_c through a ring of shared-memory stages into a
// partial t[ROWS, R]; the partials are exchanged through distributed shared memory (bulk copies into the peers, counted
// on their mbarriers) and summed in rank order by every CTA; each CTA then streams its share of the y columns and of B_c
// through the same ring, updates y in shared memory and stores it back.  There is no workspace and no second launch.
//
// Chunks are walked in a skewed order -- shrink of item 0, shrink of item 1, expand of item 0, shrink of item 2, expand of
// item 1, ... -- so that the exchange of an item's t runs behind the next item's shrink and never leaves the ring idle.
//
//   warps 8-11 (copy)    walk the chunk jobs of the CTA in that order -- shrink chunks (CH columns of the x rows + the
//                        matching rows of A_c), expand chunks (CH columns of the y rows + B_c) -- and keep the ring
//                        full: one bulk request per row of x and y (each warp a quarter of them; the SM accepts a
//                        request every ~25 cycles whatever its size and a warp's lanes issue theirs one after the other,
//                        so requests are what a small chunk costs), one TMA box for the chunk of A_c and one for the
//                        chunk of B_c, completion counted in bytes on the stage's "full" mbarrier.  The weights arrive
//                        swizzled in lines of 128 bytes (a line of A_c holds 64 / rank of its rows; boxes of shorter
//                        rows are slower to fetch): read as they lie in memory, the eight rows of a transposed ldmatrix hit one bank
//                        2, 4 or 8 times over.  Before a warp refills a stage it waits for the stage's "done"
//                        mbarrier and, if the job in it was an expand chunk (ranks 16 and 32), issues the bulk stores of
//                        its updated y rows and waits until they have been read out.
//   warps 0-7 (compute)  shrink chunk: interleaved 32-wide k blocks, ldmatrix + mma.sync.m16n8k16, fp32 partial
//                        t per warp in registers (rank 64: four warps share the k blocks, two halves the columns of t).
//                        After the CTA's last shrink chunk of an item the partials are summed in warp order
//                        through that stage's memory (it has been consumed) and pushed to the peers.
//                        Before an item's first expand chunk the CTAs' partials are summed in rank order, scaled
//                        (and multiplied by the token's routing weight, if given) and split into bf16 hi + lo A-fragments.
//                        expand chunk: 32-column groups, y += t B_c in shared memory (fp32 add, one rounding), then
//                        the warp arrives on "done".  At rank 64 the warp that updated a group also stores it (a layer of a wide
//                        model at 93 tokens: 54 us against 60; at ranks 16 and 32 the bulk stores are faster, 17.6 against 20.4).
//
// Variants: GROUP starts from the routing decisions r and groups on chip (group_inline.cuh) instead of loading offsets
// and perm; SHORT uses 16-row tiles for small calls; see FsVariant.
//
// What bounds it: small calls the launch, the grouping and the first round trip (~6 us); rank 64 the weights (a chunk of 42 KB
// takes ~1 us on an SM, against 0.8 us at the rate of the copy bandwidth); layers of a few hundred tokens the uneven
// numbers of chunk jobs per SM.  Measured with one CTA per item, linear weights and full-width rank-64 chunks (before) and
// as it is (after), us per layer of seven projections, grouping included:
//   rank 64, hidden 4096, 16 adapters, 20 / 93 / 250 tokens   84 / 91 / 92 -> 29 / 43 / 52
//   rank 64, hidden 2048,  8 adapters,  8 / 60 tokens         42 / 49 -> 15.5 / 20.5
//   rank 32, hidden 2048,  8 adapters,  8 / 256 / 777 tokens  21.7 / 25.8 / 43 -> 12.3 / 20.1 / 28
//   rank 16, hidden 2048,  8 adapters,  8 / 256 tokens        11.0 / 14.8 -> 10.9 / 14.1;  hidden 4096, 256: 24.5 -> 22.5
//   rank 16, four projections, 256 adapters, 3001 tokens      48.6 -> 37.0
//
// mma.sync is the legacy tensor path on sm_100a; a 32-row tile is far below the 128-row tcgen05 tile, and this path
// is bound by the bytes it moves, not by its flops.  Every wait is bounded; after a time-out the CTA stops issuing
// copies, lets the ones in flight land (bounded again) and returns with MOLORA_DEV_TIMEOUT set.
#include <cuda.h>
#include <stdlib.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "common.cuh"
#include "group_inline.cuh"
#include "pipeline.cuh"
#include "sm100_ptx.cuh"
#include "stream_slices.cuh"
#include "tensor_map.cuh"

namespace molora {

using namespace ptx;

constexpr int kFsWarps = 8;               // compute warps
constexpr int kFsCopyWarps = 4;           // each moves a quarter of the rows of the tile
constexpr int kFsThreads = (kFsWarps + kFsCopyWarps) * 32;
constexpr long long kFsLandingCycles = 1000000;    // ~0.5 ms; a copy between CTAs takes ~1 us
constexpr int kFsPermCache = 4096;        // calls with at most this many tokens keep perm in shared memory

// Weight boxes of the launch's projections (the kernels that use none are launched without them).
struct StreamMaps {
    CUtensorMap tm_a[MOLORA_MAX_PROJECTIONS];        // the stack as lines of 64 elements, whatever the rank; a box is a chunk of one adapter
    CUtensorMap tm_b[MOLORA_MAX_PROJECTIONS];        // [d_out / block][adapters x rank][block] views, block = bcols columns
    int32_t bcols[MOLORA_MAX_PROJECTIONS];           // 64, or 32 where d_out is no multiple of 64
};
struct NoMaps {
};
struct StreamParams {
    molora_proj_desc_t p[MOLORA_MAX_PROJECTIONS];     // the projections of the launch's rank, heaviest first
    const int32_t* offsets;
    const int32_t* perm;
    uint32_t* dev_status;
    // A projection's output may be cut into slices, each an item of its own that repeats the shrink (its bytes come from L2):
    // projection p owns units [ustart[p], ustart[p + 1]) of och[p] chunks of d_out each.
    int32_t ustart[MOLORA_MAX_PROJECTIONS + 1], och[MOLORA_MAX_PROJECTIONS];
    int32_t N, P, C, max_rows;                // segments with at least max_rows rows belong to the tcgen05 kernel
    // Top-k routing in one pass (Eq. 8): a segment is a SET of `parts` adapters (set_table[4 * segment + j] names them, in
    // ascending order), the launch's rank R is parts x the adapters' rank, A_c and B_c are gathered from the
    // parts' adapters, and row_scale holds the routing weights [parts][N].  parts == 1: plain top-1 routing.
    int32_t parts, n_adapters;
    const uint8_t* set_table;
    // grouping variant only: the routing decisions and where counts / offsets / perm are written (as by molora_group)
    const int32_t* r;
    int32_t* counts_out;
    int32_t* offsets_out;
    int32_t* perm_out;
};
// adapter of part j of segment `seg`
// (set_tab: the kernel's shared-memory copy of prm.set_table)
__device__ __forceinline__ int fs_part_adapter(const StreamParams& prm, const uint8_t* set_tab, int seg, int j)
{
    return prm.parts == 1 ? seg : (int)set_tab[seg * 4 + j];
}
// SHORT: 16-row tiles (rank 16: with chunks of 1024 columns, since a chunk costs a fixed ~0.5 us besides its bytes).
// Variants are kernels of their own: the code that a variant does not need is fetched all the same when it is there, and cost
// the launches of ~10 us about 0.6 us.
enum FsVariant : int {
    kFsOne = 0,        // one CTA per item
    kFsLinear = 1,     // ... and no tensor maps, whose first use costs ~0.5 us (rank 16, short tiles, items of at most seven jobs)
    kFsCluster = 2,    // 2 to 8 CTAs per item (ranks 32 and 64, short tiles)
};
template <int R, bool SHORT, int V>
struct FsCfg {
    static_assert(V == kFsOne || (V == kFsLinear && R == 16 && SHORT) || (V == kFsCluster && R >= 32 && SHORT), "variants that exist");
    static constexpr int ROWS = SHORT ? 16 : 32;                 // positions per tile
    static constexpr int MT = ROWS / 16;                         // 16-row MMA tiles
    static constexpr int RPW = ROWS / kFsCopyWarps;              // rows of the tile a copy warp moves
    static constexpr int CH = R == 64 ? 256 : R == 16 && SHORT ? 1024 : 512;     // columns of a chunk (of d_in or of d_out)
    static constexpr int NSTAGE = R == 16 ? (SHORT ? (CH == 1024 ? 3 : 5) : 4) : R == 32 ? 3 : (SHORT ? 4 : 3);
    static constexpr int NH = R == 64 ? 2 : 1;                   // column parts of t in the shrink
    static constexpr int KW = kFsWarps / NH;                     // warps that share the k blocks
    static constexpr int GPW = CH / 32 / kFsWarps;               // 32-column groups of an expand chunk per warp
    static constexpr bool DIRECT = R >= 64;                      // the compute warps store y
    static constexpr int RP = CH * 2 + 16;                       // pitch of a staged x / y / B_c row: 16 bytes of padding
    static constexpr int ROWBYTES = ROWS * RP;                //   keep the 8 rows of an ldmatrix in distinct banks
    static constexpr int ABYTES = CH * R * 2;                    // the chunk's rows of A_c, one [CH][rank] block per part
    static constexpr bool BOX = V != kFsLinear;                  // weights by TMA box, in swizzled lines
    static constexpr int WBYTES = BOX || R * RP < ABYTES ? ABYTES : R * RP;    // a stage: weights, then the rows
    static constexpr int STAGE = (WBYTES + ROWBYTES + 1023) / 1024 * 1024;
    static constexpr int TFLOATS = ROWS * R;                  // one fp32 copy of t
    static constexpr int MAXS = V != kFsCluster ? 1 : R == 32 ? 8 : 4;         // largest cluster
    static constexpr int RECV = 2 * MAXS * TFLOATS * 4;        // the CTAs' partials of two items
    static constexpr int SMEM = NSTAGE * STAGE + RECV + 1024;  // (the stages start at a 1024-byte boundary)
    static_assert(SMEM + 20992 <= 232448, "with the static tables a CTA fits an SM");
    static_assert(KW * TFLOATS * 4 <= STAGE, "the per-warp partials are summed through one stage");
    static_assert(kGroupInCtaScratch<kFsThreads> <= NSTAGE * STAGE, "the grouping scratch is the ring");
};
template <int R, bool SHORT, int V>
struct FsArgs : std::conditional_t<FsCfg<R, SHORT, V>::BOX, StreamMaps, NoMaps>, StreamParams {
};

namespace {

__device__ __forceinline__ void fs_mma(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void fs_ldsm(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void fs_ldsm_t(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
// barrier of the compute warps only (the copy warp never joins it)
__device__ __forceinline__ void fs_compute_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kFsWarps * 32) : "memory"); }

// One work item, decoded the same way by the copy warps and the compute warps.
struct FsItem {
    int proj, seg, row0, rows;
    int nks;        // shrink chunks (CTA c of the cluster takes c, c + S, ...)
    int ne;         // expand chunks
    int col0;       // first output column
};
__device__ __forceinline__ FsItem fs_item(const StreamParams& prm, const int32_t* offs_s, const int32_t* tstart_s, int T, int item,
                                          int CH, int ROWS)
{
    FsItem it;
    const int unit = item / T;
    it.proj = 0;
#pragma unroll
    for (int p = 1; p < MOLORA_MAX_PROJECTIONS; ++p)
        if (p < prm.P && unit >= prm.ustart[p]) it.proj = p;
    it.seg = 0;
    it.row0 = 0;
    it.rows = 1;
    find_tile_bisect(offs_s, tstart_s, prm.C, ROWS, item - unit * T, it.seg, it.row0, it.rows);
    const molora_proj_desc_t& pd = prm.p[it.proj];
    it.nks = (pd.d_in + CH - 1) / CH;
    it.col0 = (unit - prm.ustart[it.proj]) * prm.och[it.proj] * CH;
    it.ne = min(prm.och[it.proj], (pd.d_out - it.col0 + CH - 1) / CH);
    return it;
}
__device__ __forceinline__ int fs_token(const StreamParams& prm, const int32_t* perm_s, int pos)
{
    return prm.N <= kFsPermCache ? perm_s[pos] : ptx::ld_dependent(prm.perm + pos);
}

}  // namespace

// GROUP: the call starts from the routing decisions r instead of offsets / perm (at most kFsPermCache tokens).  Every
// CTA then runs the whole grouping (Section 3.3 steps 1-3: histogram, exclusive scan, stable permutation -- the
// algorithm of group_cluster_kernel on one CTA) into its own shared memory before its first copy request, which
// replaces the table load and saves the grouping launch; the CTAs also write counts, offsets and perm out, bit-equal
// to molora_group's, each a slice of perm.
template <int R, bool GROUP, bool SHORT, int V>
__global__ void __launch_bounds__(kFsThreads, 1) apply_stream_kernel(const __grid_constant__ FsArgs<R, SHORT, V> args)
{
    using Cfg = FsCfg<R, SHORT, V>;
    const StreamParams& prm = args;
    constexpr int NS = Cfg::NSTAGE;
    __shared__ int32_t offs_s[MOLORA_MAX_ADAPTERS + 1];
    __shared__ int32_t tstart_s[MOLORA_MAX_ADAPTERS + 1];
    __shared__ int32_t perm_s[kFsPermCache];
    __shared__ __align__(8) uint64_t full_s[NS], done_s[NS];
    __shared__ __align__(8) uint64_t tfull_s[2], tfree_s[2];    // partials of an item have arrived / have been read by every peer
    __shared__ unsigned long long st_dst[NS][Cfg::ROWS];   // expand job in the stage: where its y rows go back to
    __shared__ uint32_t st_bytes[kFsCopyWarps][NS];      // bytes per row to store (0: nothing to store)
    __shared__ int st_rows[kFsCopyWarps][NS];
    __shared__ int abort_s;
    __shared__ __align__(16) uint8_t set_tab_s[MOLORA_MAX_ADAPTERS * 4];   // adapter sets of top-k routing: set -> adapters
    extern __shared__ unsigned char dsm_raw[];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // (a constant where there are no clusters: those kernels carry none of the exchange)
    const int S = Cfg::MAXS == 1 ? 1 : (int)cluster_nctarank(), crank = Cfg::MAXS == 1 ? 0 : (int)cluster_ctarank();
    const int cid = (int)blockIdx.x / S, ncl = (int)gridDim.x / S;
    unsigned char* dsm = dsm_raw + ((1024u - (smem_u32(dsm_raw) & 1023u)) & 1023u);
    float* recv = reinterpret_cast<float*>(dsm + NS * Cfg::STAGE);         // [slot][rank][TFLOATS]
    if (tid == kFsThreads - 32) {              // (not of the first warps: the tokens of a small call are theirs)
        for (int s = 0; s < NS; ++s) {
            mbar_init(smem_u32(&full_s[s]), kFsCopyWarps);
            mbar_init(smem_u32(&done_s[s]), kFsWarps);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(smem_u32(&tfull_s[s]), 1);
            mbar_init(smem_u32(&tfree_s[s]), S > 1 ? (S - 1) * kFsWarps : 1);
        }
        abort_s = 0;
        fence_mbar_init();
        if constexpr (Cfg::BOX)
            for (int p = 0; p < prm.P; ++p) {
                prefetch_tensormap(&args.tm_a[p]);
                prefetch_tensormap(&args.tm_b[p]);
            }
    }
    grid_dependency_sync();                    // (launched under its predecessor, whatever that is)
    if (prm.parts > 1)                         // (visible after the block-wide barriers of the prologue below)
        for (int i = tid; i < prm.C; i += kFsThreads)
            reinterpret_cast<uint32_t*>(set_tab_s)[i] = (uint32_t)ld_dependent(reinterpret_cast<const int32_t*>(prm.set_table) + i);
    if constexpr (GROUP) {
        // the grouping itself, on this CTA, while the ring is idle (its memory is the scratch)
        group_in_cta<kFsThreads, kFsPermCache>(prm.r, prm.N, prm.C, offs_s, tstart_s, perm_s, dsm, Cfg::ROWS, true, prm.counts_out,
                                               prm.offsets_out, prm.dev_status);
    } else {
        // segment table and (small calls) the permutation on chip in one memory round trip
        for (int i = tid; i <= prm.C; i += kFsThreads) offs_s[i] = ld_dependent(prm.offsets + i);
        if (prm.N <= kFsPermCache)
            for (int i = tid; i < prm.N; i += kFsThreads) perm_s[i] = ld_dependent(prm.perm + i);
        __syncthreads();
    }
    // tiles of the segments before each segment (those with 1 <= rows < max_rows own tiles here), so that an item finds
    // its tile by bisection instead of a walk over all segments
    // (the grouping variant has done that)
    if constexpr (!GROUP) {
        if (warp == 0) tile_starts(offs_s, prm.C, Cfg::ROWS, 1, prm.max_rows, tstart_s);
        __syncthreads();
    }
    const int T = tstart_s[prm.C];
    const int nitems = T * prm.ustart[prm.P];
    // Items of my cluster: one of every ncl consecutive ones, from the front and from the back in turn.  Items are numbered
    // heaviest projection first, so the clusters that took the heaviest of one round take the lightest of the next, or none.
    // (Always from the front, the clusters with a gate or up projection also got the second item: 93 tokens of a wide rank-64
    // layer 48.7 us, so 42.7; rank 32, 777 tokens 36.0 / 28.3; rank 16, 1500 tokens 44.6 / 39.3.)
    auto item_of = [&](int i) { return i * ncl + ((i & 1) ? ncl - 1 - cid : cid); };
    const int rounds = nitems / ncl;
    const int mine = rounds + (item_of(rounds) < nitems ? 1 : 0);
    const uint32_t stage0 = smem_u32(dsm);
    if (S > 1) cluster_sync_all();             // every peer's barriers are initialised

    if (warp >= kFsWarps) {
        // ------------------------------------------------------------------------------------------ copy warps
        // Copy warp w owns RPW consecutive rows of the tile (its first RPW lanes, one bulk request each); warp 0 also requests
        // the weights (the lanes after them, one per adapter of the segment).  The four warps run the same job list without
        // talking to one another -- each arrives once per job on the stage's "full" barrier with the bytes it requested.
        const int cw = warp - kFsWarps;
        constexpr int RPW = Cfg::RPW;
        const int myrow = cw * RPW + (lane % RPW);
        const int parts = prm.parts, pr = R / parts;            // adapters per segment, rank of each
        // the stage's previous job is finished: write back my y rows if it was an expand chunk
        auto retire = [&](uint32_t k) {
            const uint32_t s = k % NS;
            wait_bar(smem_u32(&done_s[s]), (k / NS) & 1u, &abort_s, prm.dev_status);
            if constexpr (!Cfg::DIRECT) {
                const uint32_t nb = st_bytes[cw][s];
                if (nb != 0 && !abort_s) {
                    if (lane < RPW && myrow < st_rows[cw][s])
                        bulk_store(reinterpret_cast<void*>(st_dst[s][myrow]), stage0 + s * Cfg::STAGE + Cfg::WBYTES + myrow * Cfg::RP, nb);
                    bulk_commit_group();
                    bulk_wait_group_read<0>(); // the stage may be overwritten
                }
                __syncwarp();                  // every lane has read the stage's record before lane 0 rewrites it
            }
        };
        uint32_t g = 0;                        // jobs issued so far; job k lives in stage k % NS
        auto token_of = [&](const FsItem& it) -> int64_t {
            return lane < RPW && myrow < it.rows ? fs_token(prm, perm_s, it.row0 + myrow) : 0;
        };
        auto issue_shrink = [&](const FsItem& it, int64_t tok) {
            const molora_proj_desc_t& pd = prm.p[it.proj];
            const bool rowlane = lane < RPW && myrow < it.rows;
            const char* xrow = static_cast<const char*>(pd.x) + tok * pd.ldx * 2;
            const int myrows = max(0, min(RPW, it.rows - cw * RPW));
            for (int j = crank; j < it.nks; j += S, ++g) {
                const uint32_t s = g % NS;
                if (g >= (uint32_t)NS) retire(g - NS);
                if (abort_s) return;
                const uint32_t sb = stage0 + s * Cfg::STAGE, bar = smem_u32(&full_s[s]);
                fence_proxy_async_smem();      // earlier accesses to the stage are ordered before the copies
                const int k0 = j * Cfg::CH, kc = min(Cfg::CH, pd.d_in - k0);
                const uint32_t xbytes = (uint32_t)kc * 2u;
                if (lane == 0) {
                    st_bytes[cw][s] = 0;
                    mbar_arrive_expect_tx(bar, (uint32_t)myrows * xbytes +
                                                   (!Cfg::BOX ? (uint32_t)(kc * R * 2 / kFsCopyWarps) : cw == 0 ? (uint32_t)Cfg::ABYTES : 0u));
                }
                __syncwarp();
                if (rowlane) bulk_load(sb + Cfg::WBYTES + myrow * Cfg::RP, xrow + (int64_t)k0 * 2, xbytes, bar);
                if constexpr (!Cfg::BOX) {
                    // my quarter of the chunk's rows of A_c (kc is a multiple of 32: a quarter is a multiple of 16 bytes)
                    const int part = lane - RPW;
                    const uint32_t aq = (uint32_t)(kc * pr * 2 / kFsCopyWarps);
                    if (part >= 0 && part < parts)
                        bulk_load(sb + part * (Cfg::CH * pr * 2) + cw * aq,
                                  static_cast<const char*>(pd.A) +
                                      ((int64_t)fs_part_adapter(prm, set_tab_s, it.seg, part) * pd.d_in + k0) * pr * 2 + cw * aq, aq, bar);
                } else if (cw == 0 && lane >= RPW && lane < RPW + parts) {
                    const int part = lane - RPW;
                    const int line = (int)(((int64_t)fs_part_adapter(prm, set_tab_s, it.seg, part) * pd.d_in + k0) * pr / 64);
                    tma_load_2d(sb + part * (Cfg::CH * pr * 2), &args.tm_a[it.proj], 0, line, bar);    // (what lies past d_in is never read)
                }
            }
        };
        auto issue_expand = [&](const FsItem& it, int64_t tok) {
            const molora_proj_desc_t& pd = prm.p[it.proj];
            const bool rowlane = lane < RPW && myrow < it.rows;
            char* yrow = static_cast<char*>(pd.y) + tok * pd.ldy * 2;
            [[maybe_unused]] int bsh = 6;
            if constexpr (Cfg::BOX) bsh = args.bcols[it.proj] == 64 ? 6 : 5;
            const int myrows = max(0, min(RPW, it.rows - cw * RPW));
            for (int j = crank; j < it.ne; j += S, ++g) {
                const uint32_t s = g % NS;
                if (g >= (uint32_t)NS) retire(g - NS);
                if (abort_s) return;
                const uint32_t sb = stage0 + s * Cfg::STAGE, bar = smem_u32(&full_s[s]);
                fence_proxy_async_smem();
                const int c0 = it.col0 + j * Cfg::CH, nc = min(Cfg::CH, pd.d_out - c0);
                const uint32_t rowbytes = (uint32_t)nc * 2u;
                if (!Cfg::DIRECT && rowlane) st_dst[s][myrow] = reinterpret_cast<unsigned long long>(yrow + (int64_t)c0 * 2);
                if (lane == 0) {
                    st_bytes[cw][s] = rowbytes;
                    st_rows[cw][s] = it.rows;
                    mbar_arrive_expect_tx(bar, (uint32_t)(myrows + (Cfg::BOX ? 0 : R / kFsCopyWarps)) * rowbytes +
                                                   (Cfg::BOX && cw == 0 ? (uint32_t)Cfg::ABYTES : 0u));
                }
                __syncwarp();
                if (rowlane) bulk_load(sb + Cfg::WBYTES + myrow * Cfg::RP, yrow + (int64_t)c0 * 2, rowbytes, bar);
                if constexpr (!Cfg::BOX) {
                    const int brow = cw * (R / kFsCopyWarps) + lane - RPW;       // my row of the stacked B
                    if (lane >= RPW && lane < RPW + R / kFsCopyWarps)
                        bulk_load(sb + brow * Cfg::RP,
                                  static_cast<const char*>(pd.B) +
                                      (((int64_t)fs_part_adapter(prm, set_tab_s, it.seg, brow / pr) * pr + brow % pr) * pd.d_out + c0) * 2, rowbytes, bar);
                } else if (cw == 0 && lane >= RPW && lane < RPW + parts) {     // (blocks past d_out arrive as zeros)
                    tma_load_3d(sb + (lane - RPW) * (Cfg::CH * pr * 2), &args.tm_b[it.proj], 0,
                                fs_part_adapter(prm, set_tab_s, it.seg, lane - RPW) * pr, c0 >> bsh, bar);
                }
            }
        };
        FsItem cur = {}, next = {};
        int64_t ctok = 0, ntok = 0;
        for (int i = -1; i < mine && !abort_s; ++i) {       // (one copy of either body: code that is fetched once)
            cur = next;
            ctok = ntok;
            if (i + 1 < mine) {
                next = fs_item(prm, offs_s, tstart_s, T, item_of(i + 1), Cfg::CH, Cfg::ROWS);
                ntok = token_of(next);
                issue_shrink(next, ntok);
                if (abort_s) break;
            }
            if (i >= 0) issue_expand(cur, ctok);
        }
        // the jobs still in the ring
        const uint32_t first = g > (uint32_t)NS ? g - NS : 0;
        if (!Cfg::DIRECT && !abort_s)
            for (uint32_t k = first; k < g; ++k) retire(k);
        if (abort_s) {
            // stopped early: give the copies in flight into this CTA's shared memory a bounded chance to land
            for (uint32_t k = first; k < g; ++k) {
                const long long t0 = clock64();
                while (!mbar_try_wait(smem_u32(&full_s[k % NS]), (k / NS) & 1u) && clock64() - t0 < kTimeoutCycles) {
                }
            }
        }
        bulk_wait_group<0>();                  // my stores have completed
    } else {
        // ---------------------------------------------------------------------------------------------- compute warps
        constexpr int NT = R / 8 / Cfg::NH;        // n8 tiles of t that a warp computes
        constexpr int KB = R / 16;                 // k16 blocks of the expand
        constexpr int MT = Cfg::MT;
        const int g4 = lane >> 2, q = lane & 3;
        const int kw = warp % Cfg::KW, n0 = warp / Cfg::KW * (NT * 8);        // my share of the k blocks, my columns of t
        uint32_t g = 0;
        if constexpr (GROUP) group_write_perm(perm_s, offs_s[prm.C], prm.perm_out, tid, kFsWarps * 32);
        auto slot_of = [&](int i, int rank) { return recv + ((i & 1) * S + rank) * Cfg::TFLOATS; };
        // LoRA scale x the token's routing weight (top-k in one pass: the weight of the part the column belongs to) of the pieces of t
        // that this thread finishes.  With one CTA per item it is asked for before the item's chunks: in front of the sum the two loads in a
        // row cost every item of a top-2 call ~0.5 us (a layer of 2048 tokens 72.5 us, so 70.9).
        constexpr int PIECES = (Cfg::TFLOATS / 4 + kFsWarps * 32 - 1) / (kFsWarps * 32);
        auto scale_of = [&](const FsItem& it, const molora_proj_desc_t& pd, int e4) {
            const int row = e4 * 4 / R;
            float sc = pd.scale;
            if (pd.row_scale != nullptr && row < it.rows)
                sc *= ld_dependent(pd.row_scale + (int64_t)((e4 * 4 % R) / (R / prm.parts)) * prm.N + fs_token(prm, perm_s, it.row0 + row));
            return sc;
        };
        auto scaled = [&](float sc, bool live, float4 v) {          // rows past the tile hold stale shared memory
            return live ? make_float4(v.x * sc, v.y * sc, v.z * sc, v.w * sc) : make_float4(0.f, 0.f, 0.f, 0.f);
        };

        // ---- shrink: this CTA's partial of t = x A_c, item i of the cluster
        auto shrink = [&](const FsItem& it, int i) {
            const molora_proj_desc_t& pd = prm.p[it.proj];
            const bool two = MT == 2 && it.rows > 16;   // the second 16-row MMA tile holds valid rows
            const int pr = R / prm.parts, wbytes = pr * 2;
            [[maybe_unused]] float sc[PIECES];
            if constexpr (Cfg::MAXS == 1) {
#pragma unroll
                for (int k = 0; k < PIECES; ++k) sc[k] = scale_of(it, pd, tid + k * kFsWarps * 32);
            }
            float acc[MT][NT][4];
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int n = 0; n < NT; ++n)
#pragma unroll
                    for (int k = 0; k < 4; ++k) acc[mt][n][k] = 0.f;
            for (int j = crank; j < it.nks; j += S, ++g) {
                const uint32_t s = g % NS;
                const uint32_t as = stage0 + s * Cfg::STAGE, xs = as + Cfg::WBYTES;
                wait_bar(smem_u32(&full_s[s]), (g / NS) & 1u, &abort_s, prm.dev_status);
                const int nb = min(Cfg::CH, pd.d_in - j * Cfg::CH) / 32;
                for (int b = kw; b < nb; b += Cfg::KW) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {                           // two k16 steps per block
                        uint32_t bf[NT / 2][4];
                        const int m = lane >> 3;                            // matrix of the x4 load this lane addresses
#pragma unroll
                        for (int n16 = 0; n16 < NT / 2; ++n16) {
                            // the chunk's rows of A: one [k][pr] block per part (pr >= 16: an n16 tile lies in one part)
                            const int col = n0 + n16 * 16, part = col / pr;
                            const uint32_t addr = as + part * (Cfg::CH * wbytes) + (b * 32 + h * 16 + (m & 1) * 8 + (lane & 7)) * wbytes +
                                                  (col - part * pr + (m >> 1) * 8) * 2;
                            fs_ldsm_t(bf[n16], Cfg::BOX ? addr ^ (((addr >> 7) & 7u) << 4) : addr);
                        }
#pragma unroll
                        for (int mt = 0; mt < MT; ++mt) {
                            if (mt == 0 || two) {
                                uint32_t a[4];
                                fs_ldsm(a, xs + (mt * 16 + (lane & 15)) * Cfg::RP + (b * 32 + h * 16 + (lane >> 4) * 8) * 2);
#pragma unroll
                                for (int n16 = 0; n16 < NT / 2; ++n16) {
                                    fs_mma(acc[mt][2 * n16], a, bf[n16][0], bf[n16][1]);
                                    fs_mma(acc[mt][2 * n16 + 1], a, bf[n16][2], bf[n16][3]);
                                }
                            }
                        }
                    }
                }
                if (j + S < it.nks) {
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&done_s[s]));
                } else {
                    // last chunk: sum the per-warp partials in warp order through this stage, then release it
                    float* tparts = reinterpret_cast<float*>(dsm + s * Cfg::STAGE);
                    float* tpart = tparts + kw * Cfg::TFLOATS + n0;
                    // My slot still feeds the copies of item i - 2 to the peers until every peer has read what arrived; no warp
                    // writes to it before that (the barriers order them behind warp 0's wait; waiting after the sums have been laid
                    // out instead costs the layer of a wide rank-64 model at 93 tokens 48 us, not 41).
                    if (S > 1 && warp == 0 && i >= 2)
                        wait_bar_cluster(smem_u32(&tfree_s[i & 1]), (uint32_t)((i >> 1) - 1) & 1u, &abort_s, prm.dev_status);
                    fs_compute_sync();                 // every warp has finished reading the stage
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                        for (int n = 0; n < NT; ++n) {
                            const int c = n * 8 + 2 * q;
                            *reinterpret_cast<float2*>(&tpart[(mt * 16 + g4) * R + c]) = make_float2(acc[mt][n][0], acc[mt][n][1]);
                            *reinterpret_cast<float2*>(&tpart[(mt * 16 + g4 + 8) * R + c]) = make_float2(acc[mt][n][2], acc[mt][n][3]);
                        }
                    fs_compute_sync();
                    float* out = slot_of(i, crank);
#pragma unroll
                    for (int k = 0; k < PIECES; ++k) {
                        const int e4 = tid + k * kFsWarps * 32;
                        if (e4 >= Cfg::TFLOATS / 4) break;
                        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                        for (int w = 0; w < Cfg::KW; ++w) {
                            const float4 u = *reinterpret_cast<const float4*>(&tparts[w * Cfg::TFLOATS + e4 * 4]);
                            v.x += u.x;
                            v.y += u.y;
                            v.z += u.z;
                            v.w += u.w;
                        }
                        if constexpr (Cfg::MAXS == 1) v = scaled(sc[k], e4 * 4 / R < it.rows, v);
                        *reinterpret_cast<float4*>(&out[e4 * 4]) = v;
                    }
                    fence_proxy_async_smem();          // my writes are ordered before the copies that refill the stage or read the slot
                    fs_compute_sync();                 // the partial is complete; the stage is free
                    if (lane == 0) mbar_arrive(smem_u32(&done_s[s]));
                    if (S > 1 && warp == 0) {          // push it to the peers, who have read what their slots held before (waited for above)
                        if (lane == 0) mbar_arrive_expect_tx(smem_u32(&tfull_s[i & 1]), (uint32_t)(S - 1) * Cfg::TFLOATS * 4u);
                        if (lane < S && lane != crank && !abort_s)
                            bulk_copy_to_peer(map_to_cta(smem_u32(out), lane), smem_u32(out), Cfg::TFLOATS * 4u,
                                              map_to_cta(smem_u32(&tfull_s[i & 1]), lane));
                    }
                    __syncwarp();
                }
            }
        };

        // ---- expand: y += t B_c for this CTA's chunks, in shared memory
        auto expand = [&](const FsItem& it, int i) {
            const molora_proj_desc_t& pd = prm.p[it.proj];
            const bool two = MT == 2 && it.rows > 16;
            // t of the item: with S > 1 the sum of the CTAs' partials in rank order, formed in the slot of the next rank (its
            // content is read by the same thread that overwrites it)
            float* tfin = slot_of(i, S == 1 ? 0 : (crank + 1) % S);
            if (S > 1) {
                wait_bar_cluster(smem_u32(&tfull_s[i & 1]), (uint32_t)(i >> 1) & 1u, &abort_s, prm.dev_status);
                for (int e4 = tid; e4 < Cfg::TFLOATS / 4; e4 += kFsWarps * 32) {
                    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
                    for (int k = 0; k < S; ++k) {
                        const float4 u = *reinterpret_cast<const float4*>(&slot_of(i, k)[e4 * 4]);
                        v.x += u.x;
                        v.y += u.y;
                        v.z += u.z;
                        v.w += u.w;
                    }
                    *reinterpret_cast<float4*>(&tfin[e4 * 4]) = scaled(scale_of(it, pd, e4), e4 * 4 / R < it.rows, v);
                }
                fs_compute_sync();
            }
            // A fragments of t: bf16 hi and lo parts
            uint32_t thi[MT][KB][4], tlo[MT][KB][4];
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int kb = 0; kb < KB; ++kb)
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int r = mt * 16 + g4 + 8 * (k & 1);
                        const int c = kb * 16 + 2 * q + 8 * (k >> 1);
                        const float2 tv = *reinterpret_cast<const float2*>(&tfin[r * R + c]);
                        const float h0 = __bfloat162float(__float2bfloat16_rn(tv.x)), h1 = __bfloat162float(__float2bfloat16_rn(tv.y));
                        thi[mt][kb][k] = f32x2_to_bf16x2(h0, h1);
                        tlo[mt][kb][k] = f32x2_to_bf16x2(tv.x - h0, tv.y - h1);
                    }
            if (S > 1) {                               // the peers may overwrite this slot
                fence_proxy_async_smem();
                __syncwarp();
                if (lane < S && lane != crank) mbar_arrive_remote(map_to_cta(smem_u32(&tfree_s[i & 1]), lane));
            }
            // DIRECT: finished y leaves through the warp that computed it: 16-byte pieces, 64 bytes of eight rows per store
            char* yrow[MT][2];
            if constexpr (Cfg::DIRECT) {
                const bool live = *static_cast<volatile int*>(&abort_s) == 0;      // no wait has run out: t is what it should be
#pragma unroll
                for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int row = mt * 16 + h * 8 + (lane & 7);
                        yrow[mt][h] = live && row < it.rows ? static_cast<char*>(pd.y) + (int64_t)fs_token(prm, perm_s, it.row0 + row) * pd.ldy * 2 : nullptr;
                    }
            }

            // B_c in shared memory: per part [block of bcols columns][rank][bcols], rows swizzled over 128 or 64 bytes
            const int pr = R / prm.parts;
            int bsh = 6;
            if constexpr (Cfg::BOX) bsh = args.bcols[it.proj] == 64 ? 6 : 5;
            const uint32_t bmask = bsh == 6 ? 7u : 3u;
            for (int j = crank; j < it.ne; j += S, ++g) {
                const uint32_t s = g % NS;
                const uint32_t bs = stage0 + s * Cfg::STAGE;
                unsigned char* ysp = dsm + s * Cfg::STAGE + Cfg::WBYTES;
                const bool arrived = wait_bar(smem_u32(&full_s[s]), (g / NS) & 1u, &abort_s, prm.dev_status);
                if (Cfg::DIRECT && !arrived) break;        // a wait ran out: the stage may hold anything, y keeps what it has
                const int ngroups = min(Cfg::CH, pd.d_out - it.col0 - j * Cfg::CH) / 32;
                // my 32-column groups: y words first, then the MMAs, then add, round once and write back.
                // Rows past the tile hold stale shared memory; they are updated like the others and never stored.
                for (int grp = warp; grp < ngroups; grp += kFsWarps) {
                    uint32_t yv[MT][2][4];
                    float d[MT][4][4];
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                        for (int h = 0; h < 2; ++h)
#pragma unroll
                            for (int nt = 0; nt < 4; ++nt)
                                yv[mt][h][nt] = *reinterpret_cast<const uint32_t*>(ysp + (mt * 16 + g4 + 8 * h) * Cfg::RP +
                                                                                   (grp * 32 + nt * 8 + 2 * q) * 2);
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                            for (int k = 0; k < 4; ++k) d[mt][nt][k] = 0.f;
#pragma unroll
                    for (int kb = 0; kb < KB; ++kb) {
                        uint32_t bf[2][4];                              // [n16 pair][b0,b1 of tile 2p, b0,b1 of tile 2p+1]
                        const int m = lane >> 3;
#pragma unroll
                        for (int p2 = 0; p2 < 2; ++p2)
                        {
                            const int part = kb * 16 / pr, row = kb * 16 - part * pr + (m & 1) * 8 + (lane & 7);
                            const int col = grp * 32 + p2 * 16 + (m >> 1) * 8;
                            const uint32_t addr = bs + part * (Cfg::CH * pr * 2) + ((((col >> bsh) * pr + row) << bsh) + (col & ((1 << bsh) - 1))) * 2;
                            fs_ldsm_t(bf[p2], Cfg::BOX ? addr ^ (((addr >> 7) & bmask) << 4) : bs + (kb * 16 + (m & 1) * 8 + (lane & 7)) * Cfg::RP + col * 2);
                        }
#pragma unroll
                        for (int mt = 0; mt < MT; ++mt) {
                            if (mt == 0 || two) {
#pragma unroll
                                for (int p2 = 0; p2 < 2; ++p2) {
                                    fs_mma(d[mt][2 * p2], thi[mt][kb], bf[p2][0], bf[p2][1]);
                                    fs_mma(d[mt][2 * p2 + 1], thi[mt][kb], bf[p2][2], bf[p2][3]);
                                }
#pragma unroll
                                for (int p2 = 0; p2 < 2; ++p2) {
                                    fs_mma(d[mt][2 * p2], tlo[mt][kb], bf[p2][0], bf[p2][1]);
                                    fs_mma(d[mt][2 * p2 + 1], tlo[mt][kb], bf[p2][2], bf[p2][3]);
                                }
                            }
                        }
                    }
                    // accumulator element (row g4 + 8h, columns 2q, 2q+1 of n8 tile nt)
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                        for (int h = 0; h < 2; ++h)
#pragma unroll
                            for (int nt = 0; nt < 4; ++nt) {
                                const uint32_t v = yv[mt][h][nt];
                                *reinterpret_cast<uint32_t*>(ysp + (mt * 16 + g4 + 8 * h) * Cfg::RP + (grp * 32 + nt * 8 + 2 * q) * 2) =
                                    f32x2_to_bf16x2(bf16lo_to_f32(v) + d[mt][nt][2 * h], bf16hi_to_f32(v) + d[mt][nt][2 * h + 1]);
                            }
                    if constexpr (Cfg::DIRECT) {
                        __syncwarp();
                        const int piece = grp * 64 + (lane >> 3) * 16;
#pragma unroll
                        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                            for (int h = 0; h < 2; ++h)
                                if (yrow[mt][h] != nullptr)
                                    stg128(yrow[mt][h] + (int64_t)(it.col0 + j * Cfg::CH) * 2 + piece,
                                           *reinterpret_cast<const uint4*>(ysp + (mt * 16 + h * 8 + (lane & 7)) * Cfg::RP + piece));
                    }
                }
                if constexpr (!Cfg::DIRECT) fence_proxy_async_smem();   // my updates of y are visible to the bulk stores
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&done_s[s]));
            }
        };

        FsItem cur = {}, next = {};
        for (int i = -1; i < mine; ++i) {
            cur = next;
            if (i + 1 < mine) {
                next = fs_item(prm, offs_s, tstart_s, T, item_of(i + 1), Cfg::CH, Cfg::ROWS);
                shrink(next, i + 1);
            }
            if (i >= 0) expand(cur, i);
        }
    }
    // No CTA leaves while a peer may still write into its shared memory or read from it.  Every wait above is bounded, so all get here.
    if (S > 1) {
        // After a time-out copies between the CTAs may be in flight that nobody has waited for: all of them learn of it, stop
        // issuing (the first barrier) and give the copies, of a few KB each, a bounded time to land.
        volatile int* aborted = &abort_s;
        if (*aborted && lane < S) st_cluster_u32(map_to_cta(smem_u32(&abort_s), lane), 1u);
        __syncwarp();
        cluster_sync_all();
        if (*aborted) {
            const long long t0 = clock64();
            while (clock64() - t0 < kFsLandingCycles) {
            }
            __syncwarp();
            cluster_sync_all();
        }
    }
}

// ------------------------------------------------------------------------------------------------ host side
bool stream_eligible(const molora_proj_desc_t& p, molora_dtype_t dt)
{
    return dt == MOLORA_BF16 && (p.rank == 16 || p.rank == 32 || p.rank == 64) && (p.d_in % 32) == 0 && (p.d_out % 32) == 0;
}

static SliceShapes slice_shapes(const StreamParams& prm, int CH)
{
    SliceShapes sh;
    sh.P = prm.P;
    for (int i = 0; i < prm.P; ++i) {
        sh.in[i] = ceil_div(prm.p[i].d_in, CH);
        sh.out[i] = ceil_div(prm.p[i].d_out, CH);
    }
    return sh;
}

// most tiles that `rows` rows in C segments can give (every segment that has rows adds at most one partial tile)
static int64_t tiles_bound(int64_t rows, int64_t C, int tile_rows) { return std::min(rows, ceil_div64(rows, tile_rows) + std::min(C, rows)); }

// Segments that may have rows: of the adapter sets of top-k routing only those of different adapters are met; the others are there for
// callers that repeat one.
static double segments_met(const StreamParams& prm)
{
    return (double)(prm.parts > 1 && prm.n_adapters >= prm.parts ? binom_small(prm.n_adapters, prm.parts) : prm.C);
}

// Tiles that `rows` rows are expected to give.
static double expected_tiles(const StreamParams& prm, int64_t rows, int tile_rows)
{
    // Tiles of segments of about equal size: one each while that is well below a tile's height, half a tile lost per segment from there
    // on.  Of the segments as many are counted as three quarters of the rows, spread at random, meet: adapters are not equally popular
    // (rank 64, 4096 wide, 20 tokens of 16 adapters by popularity: clusters of four 26 us, of two, as for all 16, 32).
    const double met = segments_met(prm);
    const double segments = std::min((double)rows, std::max(1.0, met * (1.0 - std::pow(1.0 - 1.0 / met, 0.75 * (double)rows))));
    const double fill = (double)rows / segments / tile_rows;
    return segments * (fill <= 0.75 ? 1.0 : fill <= 1.0 ? 1.0 + 2.0 * (fill - 0.75) : fill + 0.5);
}

// Tiles of as many rows spread evenly.
static int equal_tiles(const StreamParams& prm, int64_t rows, int tile_rows)
{
    const int64_t segments = std::max<int64_t>(1, std::min(rows, (int64_t)segments_met(prm)));
    return (int)(segments * ceil_div64(ceil_div64(rows, segments), tile_rows));
}

template <int R, bool GROUP, bool SHORT, int V>
static cudaError_t stream_launch(StreamParams prm, [[maybe_unused]] const StreamMaps& maps, int64_t rows, int S, cudaStream_t s)
{
    using Cfg = FsCfg<R, SHORT, V>;
    static int clusters_dev[kMaxDevices][4] = {};  // resident clusters of 1, 2, 4, 8 CTAs per device: the size of a wave
    int& clusters = clusters_dev[device_slot()][S == 1 ? 0 : S == 2 ? 1 : S == 4 ? 2 : 3];
    if (clusters == 0) {
        cudaError_t e = cudaFuncSetAttribute(apply_stream_kernel<R, GROUP, SHORT, V>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::SMEM);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        cfg.gridDim = dim3((unsigned)(S * sm_count()));
        cfg.blockDim = dim3(kFsThreads);
        cfg.dynamicSmemBytes = Cfg::SMEM;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)S;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int n = 0;
        e = cudaOccupancyMaxActiveClusters(&n, apply_stream_kernel<R, GROUP, SHORT, V>, &cfg);
        if (e != cudaSuccess) return e;
        clusters = std::max(1, n);
    }
    const int64_t tiles_max = tiles_bound(rows, prm.C, Cfg::ROWS);
    const SliceShapes shapes = slice_shapes(prm, Cfg::CH);
    const int tiles = S == 1 && prm.P > 2 && tiles_max * prm.P > clusters && tiles_max * prm.P <= 3 * clusters && clusters <= kSliceMaxClusters
                          ? (int)std::lround(expected_tiles(prm, rows, Cfg::ROWS)) : 0;
    if (tiles > 0) prm.ustart[prm.P] = balanced_units(shapes, clusters, tiles, equal_tiles(prm, rows, Cfg::ROWS), prm.och, prm.ustart);
    else prm.ustart[prm.P] = slice_outputs(shapes, S == 1 ? clusters / tiles_max : 0, prm.och, prm.ustart);
    const unsigned grid = (unsigned)(std::max<int64_t>(1, std::min<int64_t>(tiles_max * prm.ustart[prm.P], clusters)) * S);
    FsArgs<R, SHORT, V> args;
    static_cast<StreamParams&>(args) = prm;
    if constexpr (Cfg::BOX) static_cast<StreamMaps&>(args) = maps;
    return launch_kernel(apply_stream_kernel<R, GROUP, SHORT, V>, dim3(grid), dim3(kFsThreads), Cfg::SMEM, s, (unsigned)S, true, args);
}

// Estimated time of a launch (us, without its fixed part) and the CTAs per item that give it.  A launch lasts as long as its
// busiest cluster: `tiles` items per projection (and slice), each of nks + ne chunk jobs spread over S CTAs, on sms / S clusters (a few
// SMs are lost to S = 4 and 8: clusters do not straddle a GPC).  The exchange of t costs an item about 3 jobs.  A chunk job
// costs 1.30 us with 16 x 1024 and 1.19 us with 32 x 512 elements of x or y (rank 16), 1.17 / 1.72 us (rank 32, 512 columns),
// 0.90 / 1.67 us (rank 64, 256 columns), fitted to one projection of 300 - 8000 tokens and layers of 8 - 1000 tokens; a third of it
// does not depend on the chunk's width.  Against an estimate that knew neither slices nor partial chunks and counted half a tile
// for every segment, us: rank 16, 512 wide, 200 tokens, four projections 8.2 -> 7.2; rank 32, 1536 wide, 1 token, two projections
// 13.6 -> 11.0; rank 32, 2048 wide, 2500 tokens, one projection 19.5 -> 17.0.
template <int R, bool SHORT>
static double stream_estimate(const StreamParams& prm, int64_t rows, int& split)
{
    using Cfg = FsCfg<R, SHORT, (SHORT && R >= 32 ? kFsCluster : kFsOne)>;
    const double job_us = R == 16 ? (SHORT ? 1.30 : 1.19) : R == 32 ? (SHORT ? 1.17 : 1.72) : (SHORT ? 0.90 : 1.67);
    const double tiles = expected_tiles(prm, rows, Cfg::ROWS);
    auto jobs = [](int width) {            // jobs that `width` columns cost
        const int full = width / Cfg::CH, rest = width % Cfg::CH;
        return full + (rest > 0 ? 0.35 + 0.65 * rest / Cfg::CH : 0.0);
    };
    int most = Cfg::MAXS;
    for (int i = 0; i < prm.P; ++i) most = std::min(most, ceil_div(prm.p[i].d_in, Cfg::CH));      // every CTA shrinks something
    const int64_t forced = tune(kTuneStreamSplit);
    const int sms = sm_count();
    const SliceShapes shapes = slice_shapes(prm, Cfg::CH);
    double best = 1e30;
    for (int S = 1; S <= most; S *= 2) {
        const double clusters = S <= 2 ? sms / S : S == 4 ? sms * 0.9 / 4 : sms * 0.86 / 8;
        int32_t och[MOLORA_MAX_PROJECTIONS], ustart[MOLORA_MAX_PROJECTIONS + 1];
        const int units = slice_outputs(shapes, S == 1 ? sms / tiles_bound(rows, prm.C, Cfg::ROWS) : 0, och, ustart);
        double sum = 0.0, longest = 0.0;
        for (int i = 0; i < prm.P; ++i) {
            // (the CTAs of a cluster take whole chunks: the first one has the most)
            const int in = S == 1 ? prm.p[i].d_in : std::min(prm.p[i].d_in, ceil_div(ceil_div(prm.p[i].d_in, Cfg::CH), S) * Cfg::CH);
            const int out = std::min(prm.p[i].d_out, ceil_div(och[i], S) * Cfg::CH);
            const double each = jobs(in) + jobs(out) + (S > 1 ? 3.0 : 0.0);
            sum += each * (ustart[i + 1] - ustart[i]);
            longest = std::max(longest, each);
        }
        double t = longest;
        // equal items are dealt in whole rounds (a margin where the number of resident clusters is an estimate)
        if (units == 1) t = longest * std::ceil((S >= 4 ? 1.05 : 1.0) * tiles / clusters);
        else if (tiles * units > clusters) t = std::max(longest, sum * tiles / clusters + 0.15 * sum / units);
        t += S == 1 ? 0.0 : S == 2 ? 1.5 : S == 4 ? 2.25 : 3.0;
        if (forced > 0 ? S <= forced : t < best) {
            best = t;
            split = S;
        }
    }
    return best * job_us;
}

template <int R>
static cudaError_t stream_rank(const molora_proj_desc_t* projs, int32_t P, int64_t N, StreamParams& prm, bool group, cudaStream_t s)
{
    int idx[MOLORA_MAX_PROJECTIONS], n = 0;
    for (int i = 0; i < P; ++i)
        if (projs[i].rank == R) idx[n++] = i;
    if (n == 0) return cudaSuccess;
    std::stable_sort(idx, idx + n, [&](int a, int b) {
        return (int64_t)projs[a].d_in + projs[a].d_out > (int64_t)projs[b].d_in + projs[b].d_out;
    });
    prm.P = n;
    for (int i = 0; i < MOLORA_MAX_PROJECTIONS; ++i) prm.p[i] = i < n ? projs[idx[i]] : molora_proj_desc_t{};
    // every segment adds at most one partial tile; with a row cap only min(N, C * cap) rows can come here
    const int64_t cap_rows = prm.max_rows == INT32_MAX ? N : std::min<int64_t>(N, (int64_t)prm.C * prm.max_rows);
    int split16 = 1, split32 = 1;
    const double t16 = stream_estimate<R, true>(prm, cap_rows, split16), t32 = stream_estimate<R, false>(prm, cap_rows, split32);
    bool small = t16 <= t32;
    if (const int64_t forced = tune(kTuneStreamTile)) small = forced == 16;
    using Short = FsCfg<R, true, kFsOne>;
    const int pr = R / prm.parts, ch = small ? Short::CH : FsCfg<R, false, kFsOne>::CH;
    StreamMaps maps;
    // linear weights while no item has more than seven chunk jobs (us, linear / boxes; 256 tokens, 8 adapters, a layer: hidden 512 (3 jobs)
    // 7.8 / 8.4, 2048 (8 jobs) 14.9 / 14.4, 4096 (16 jobs) 24.5 / 22.4; 1536 wide, two projections (7 jobs) 7.2 / 7.7 at 1 token, 8.2 / 8.7
    // at 200)
    int jobs = 0;
    for (int i = 0; i < n; ++i) jobs = std::max(jobs, ceil_div(prm.p[i].d_in, ch) + ceil_div(prm.p[i].d_out, ch));
    const bool box = !(R == 16 && small && jobs <= 7);
    for (int i = 0; i < n && box; ++i) {
        if (!make_tensor_map_bf16_2d(&maps.tm_a[i], prm.p[i].A, 64, (uint64_t)prm.n_adapters * prm.p[i].d_in * pr / 64, 64, 64,
                                     (uint32_t)(ch * pr / 64), CU_TENSOR_MAP_SWIZZLE_128B))
            return cudaErrorInvalidValue;
        const int bc = prm.p[i].d_out % 64 == 0 ? 64 : 32;
        maps.bcols[i] = bc;
        if (!make_tensor_map_bf16_blocks(&maps.tm_b[i], prm.p[i].B, (uint64_t)prm.n_adapters * pr, (uint64_t)prm.p[i].d_out, (uint32_t)bc,
                                         (uint32_t)pr, (uint32_t)(ch / bc), bc == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B))
            return cudaErrorInvalidValue;
    }
    const int S = small ? split16 : split32;
    auto launch = [&](auto tile, auto variant) {
        constexpr bool SHORT = decltype(tile)::value;
        constexpr int V = decltype(variant)::value;
        return group ? stream_launch<R, true, SHORT, V>(prm, maps, cap_rows, S, s) : stream_launch<R, false, SHORT, V>(prm, maps, cap_rows, S, s);
    };
    using One = std::integral_constant<int, kFsOne>;
    if (!small) return launch(std::false_type{}, One{});
    if constexpr (R == 16) {
        if (!box) return launch(std::true_type{}, std::integral_constant<int, kFsLinear>{});
    } else {
        if (S > 1) return launch(std::true_type{}, std::integral_constant<int, kFsCluster>{});
    }
    return launch(std::true_type{}, One{});
}

static molora_status_t stream_enqueue(const molora_proj_desc_t* projs, int32_t P, int64_t N, int32_t C, StreamParams& prm,
                                      bool group, cudaStream_t s)
{
    prm.C = C;
    prm.N = (int32_t)N;
    // grouping: one rank only (checked by the caller), one launch does it all
    cudaError_t e = stream_rank<16>(projs, P, N, prm, group, s);
    if (e == cudaSuccess) e = stream_rank<32>(projs, P, N, prm, group, s);
    if (e == cudaSuccess) e = stream_rank<64>(projs, P, N, prm, group, s);
    return cuda_ok(e);
}

molora_status_t launch_apply_stream(const molora_proj_desc_t* projs, int32_t P, int64_t N, int32_t C,
                                    const int32_t* offsets, const int32_t* perm, int32_t max_rows, uint32_t* dev_status,
                                    cudaStream_t s)
{
    if (N == 0 || P == 0) return MOLORA_OK;
    StreamParams prm;
    prm.offsets = offsets;
    prm.perm = perm;
    prm.dev_status = dev_status;
    prm.max_rows = max_rows;
    prm.r = nullptr;
    prm.counts_out = prm.offsets_out = prm.perm_out = nullptr;
    prm.parts = 1;
    prm.n_adapters = C;
    prm.set_table = nullptr;
    return stream_enqueue(projs, P, N, C, prm, false, s);
}

// Top-k routing in one pass: `projs` carry the STACKED rank (parts x the adapters' rank) and row_scale = weights
// [parts][N]; offsets / perm group the tokens by adapter set, C_sets = cbase^parts segments.
molora_status_t launch_apply_stream_sets(const molora_proj_desc_t* projs, int32_t P, int64_t N, int32_t n_sets, int32_t parts,
                                         int32_t n_adapters, const uint8_t* set_table, const int32_t* offsets, const int32_t* perm,
                                         uint32_t* dev_status, cudaStream_t s)
{
    if (N == 0 || P == 0) return MOLORA_OK;
    StreamParams prm;
    prm.offsets = offsets;
    prm.perm = perm;
    prm.dev_status = dev_status;
    prm.max_rows = INT32_MAX;
    prm.r = nullptr;
    prm.counts_out = prm.offsets_out = prm.perm_out = nullptr;
    prm.parts = parts;
    prm.n_adapters = n_adapters;
    prm.set_table = set_table;
    return stream_enqueue(projs, P, N, n_sets, prm, false, s);
}

// ... and started from the set indices (at most 4096 tokens): grouping by set and apply in one launch.  (Forming the sets
// inside this kernel as well was measured and lost: every CTA repeats the sort, 23.2 against 21.5 us at 4096 tokens.)
molora_status_t launch_group_apply_stream_sets(const int32_t* sets, const molora_proj_desc_t* projs, int32_t P, int64_t N,
                                               int32_t n_sets, int32_t parts, int32_t n_adapters, const uint8_t* set_table, int32_t* counts,
                                               int32_t* offsets, int32_t* perm, uint32_t* dev_status, cudaStream_t s)
{
    if (N == 0 || P == 0) return MOLORA_OK;
    StreamParams prm;
    prm.offsets = nullptr;
    prm.perm = nullptr;
    prm.dev_status = dev_status;
    prm.max_rows = INT32_MAX;
    prm.r = sets;
    prm.counts_out = counts;
    prm.offsets_out = offsets;
    prm.perm_out = perm;
    prm.parts = parts;
    prm.n_adapters = n_adapters;
    prm.set_table = set_table;
    return stream_enqueue(projs, P, N, n_sets, prm, true, s);
}

bool group_apply_stream_eligible(int64_t N) { return N >= 1 && N <= kFsPermCache; }

molora_status_t launch_group_apply_stream(const int32_t* r, const molora_proj_desc_t* projs, int32_t P, int64_t N,
                                          int32_t C, int32_t* counts, int32_t* offsets, int32_t* perm,
                                          uint32_t* dev_status, cudaStream_t s)
{
    StreamParams prm;
    prm.offsets = nullptr;
    prm.perm = nullptr;
    prm.dev_status = dev_status;
    prm.max_rows = INT32_MAX;
    prm.r = r;
    prm.counts_out = counts;
    prm.offsets_out = offsets;
    prm.perm_out = perm;
    prm.parts = 1;
    prm.n_adapters = C;
    prm.set_table = nullptr;
    return stream_enqueue(projs, P, N, C, prm, true, s);
}

}  // namespace molora
