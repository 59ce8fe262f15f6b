// Section 3.3 steps 1-3 (histogram, exclusive scan, stable permutation) done by ONE CTA in its own shared memory, for
// kernels that start from the routing decisions r instead of offsets / perm: every CTA of such a kernel runs this
// before its first copy request, which replaces the table load and saves the grouping launch.  At most MAXN tokens.
// Results: offs_s[0..C], perm_s[0..offs_s[C]) and, with tile_rows > 0, tstart_s[0..C] (tiles of tile_rows rows before each segment);
// with write_out CTA 0 also writes counts and offsets to global memory and the CTAs are to write perm with group_write_perm, a slice
// each, whenever it suits them -- bit-equal to what molora_group writes.
//   scratch   shared memory that is idle at this point: kGroupInCtaScratch<NT> bytes
//   tstart_s  MOLORA_MAX_ADAPTERS + 1 ints (temporary storage where no tiles are asked for)
// Ends with a block-wide barrier.  All NT threads of the CTA must call it.
#pragma once
#include "common.cuh"
#include "sm100_ptx.cuh"

namespace molora {

constexpr int kGroupInCtaTableMaxC = 32;       // adapters handled by lanes and by the per-thread count table (ballots / match above)
template <int NT>
constexpr int kGroupInCtaScratch = kGroupInCtaTableMaxC * NT * 4 + 4 * kGroupInCtaTableMaxC;      // (covers the histograms of the ballots)

template <int NT, int MAXN>
__device__ __forceinline__ void group_in_cta(const int32_t* __restrict__ r, int N_, int C_, int32_t* offs_s, int32_t* tstart_s,
                                             int32_t* perm_s, unsigned char* scratch, int tile_rows, bool write_out, int32_t* counts_out,
                                             int32_t* offsets_out, uint32_t* dev_status)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
        constexpr int NW = NT / 32;
        static_assert(NW * MOLORA_MAX_ADAPTERS * 4 <= kGroupInCtaScratch<NT>, "histograms of the ballots");
      if (C_ <= kGroupInCtaTableMaxC && N_ <= NT) {
        // A token per thread, lane c counts adapter c: one ballot per bit of the adapter index, from which every lane takes the tokens
        // of its adapter (for the count) and the tokens that share its own token's (for the rank); the warps meet once.  What bounds it
        // is the code that a CTA meets for the first time, fetched at about ten cycles an instruction: the loops stay rolled.  With the
        // table below a decode call of 8 tokens was grouped after 4900 cycles, so after 3500; with more steps a warp it is the slower one.
        int* hist = reinterpret_cast<int*>(scratch);                               // [warp][32]
        const int C = C_, N = N_;
        const int raw = tid < N ? ptx::ld_dependent(r + tid) : -1;
        const int v = raw < C ? raw : -1;
        unsigned own = __ballot_sync(0xFFFFFFFFu, v >= 0), same = own;
        const int bits = 32 - __clz(C - 1);
#pragma unroll 1
        for (int b = 0; b < bits; ++b) {
            const unsigned m = __ballot_sync(0xFFFFFFFFu, (v >> b) & 1);
            own &= m ^ (((unsigned)lane >> b & 1u) - 1u);                          // (m where my bit is set, ~m where it is not)
            same &= m ^ (((unsigned)v >> b & 1u) - 1u);
        }
        hist[warp * 32 + lane] = __popc(own);            // (lanes past C repeat others' counts and are never read)
        __syncthreads();
        int before = 0, total = 0;
        const int warps = (N + 31) >> 5;
#pragma unroll 4
        for (int w = 0; w < warps; ++w) {
            const int t = hist[w * 32 + lane];
            if (w < warp) before += t;
            total += t;
        }
        if (lane >= C) total = 0;
        int incl = total, tiles = tile_rows > 0 ? (total + tile_rows - 1) / tile_rows : 0, tincl = tiles;
#pragma unroll 1
        for (int off = 1; off < 32; off <<= 1) {
            const int up = __shfl_up_sync(0xFFFFFFFFu, incl, off), tup = __shfl_up_sync(0xFFFFFFFFu, tincl, off);
            if (lane >= off) {
                incl += up;
                tincl += tup;
            }
        }
        const int at = __shfl_sync(0xFFFFFFFFu, incl - total + before, v & 31) + __popc(same & ((1u << lane) - 1u));
        if (v >= 0) perm_s[at] = tid;
        if (warp == 0 && lane < C) {
            offs_s[lane] = incl - total;
            if (lane == C - 1) offs_s[C] = incl;
            if (tile_rows > 0) {
                tstart_s[lane] = tincl - tiles;
                if (lane == C - 1) tstart_s[C] = tincl;
            }
            if (write_out && blockIdx.x == 0) {
                counts_out[lane] = total;
                offsets_out[lane] = incl - total;
                if (lane == C - 1) offsets_out[C] = incl;
            }
        }
        if ((write_out && blockIdx.x == 0) && dev_status != nullptr && __any_sync(0xFFFFFFFFu, raw < -1 || raw >= C) && lane == 0)
            atomicOr(dev_status, MOLORA_DEV_BAD_ROUTE);
        __syncthreads();
        return;
      }
      if (C_ <= kGroupInCtaTableMaxC) {
        // Up to 32 adapters: every thread owns a contiguous run of tokens and counts it into its own column of a
        // [adapter][thread] table in shared memory (consecutive threads hit consecutive banks); a warp
        // per adapter turns the table into exclusive prefixes over the threads, and every thread then writes its run
        // out in token order -- stable by construction, no atomics.
        constexpr int TPT = (MAXN + NT - 1) / NT;      // tokens per thread
        constexpr int LPT = NT / 32;                                   // table entries per lane in the scan
        int* cnt_s = reinterpret_cast<int*>(scratch);                              // [C][NT]
        int* tot_s = cnt_s + kGroupInCtaTableMaxC * NT;                    // [C] adapter totals
        const int C = C_, N = N_;
        const int per = (N + NT - 1) / NT;
        const int b0 = min(tid * per, N), e0 = min(b0 + per, N);
        int v[TPT];
        bool bad = false;
#pragma unroll
        for (int j = 0; j < TPT; ++j) {
            const int raw = b0 + j < e0 ? ptx::ld_dependent(r + b0 + j) : -1;
            bad |= (raw < -1) || (raw >= C);
            v[j] = (raw >= 0 && raw < C) ? raw : -1;
        }
        for (int c = 0; c < C; ++c) cnt_s[c * NT + tid] = 0;
#pragma unroll
        for (int j = 0; j < TPT; ++j)
            if (v[j] >= 0) cnt_s[v[j] * NT + tid] += 1;
        __syncthreads();
        for (int c = warp; c < C; c += NW) {           // exclusive prefix over the threads, lane = LPT consecutive threads
            int* row = cnt_s + c * NT + lane * LPT;
            int loc[LPT], sum = 0;
#pragma unroll
            for (int k = 0; k < LPT; ++k) {
                loc[k] = row[k];
                sum += loc[k];
            }
            int incl = sum;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int up = __shfl_up_sync(0xFFFFFFFFu, incl, off);
                if (lane >= off) incl += up;
            }
            int run = incl - sum;
#pragma unroll
            for (int k = 0; k < LPT; ++k) {
                row[k] = run;
                run += loc[k];
            }
            if (lane == 31) tot_s[c] = incl;
        }
        __syncthreads();
        if (warp == 0) {                               // offsets: exclusive prefix of the totals (C <= 32: one per lane)
            const int mine = lane < C ? tot_s[lane] : 0;
            int incl = mine;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int up = __shfl_up_sync(0xFFFFFFFFu, incl, off);
                if (lane >= off) incl += up;
            }
            if (lane < C) offs_s[lane] = incl - mine;
            if (lane == C - 1) offs_s[C] = incl;
            if ((write_out && blockIdx.x == 0) && lane < C) counts_out[lane] = mine;
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < TPT; ++j)
            if (v[j] >= 0) {
                int* slot = cnt_s + v[j] * NT + tid;
                const int k = *slot;
                *slot = k + 1;
                perm_s[offs_s[v[j]] + k] = b0 + j;
            }
        if ((write_out && blockIdx.x == 0) && dev_status != nullptr && __any_sync(0xFFFFFFFFu, bad) && lane == 0)
            atomicOr(dev_status, MOLORA_DEV_BAD_ROUTE);
        __syncthreads();
        if ((write_out && blockIdx.x == 0))
            for (int c = tid; c <= C; c += NT) offsets_out[c] = offs_s[c];
      } else {
        constexpr int STEPS = (MAXN + NW * 32 - 1) / (NW * 32);      // 32-token steps of a warp
        int(*hist)[MOLORA_MAX_ADAPTERS] = reinterpret_cast<int(*)[MOLORA_MAX_ADAPTERS]>(scratch);   // [warp][adapter]
        const int C = C_, N = N_;
        const unsigned lt_mask = (1u << lane) - 1u;
        const int chunk = ((N + NW - 1) / NW + 31) / 32 * 32;                // tokens of a warp: ascending token order
        const int begin = min(warp * chunk, N), end = min(begin + chunk, N);
        int vreg[STEPS];
#pragma unroll
        for (int j = 0; j < STEPS; ++j) {
            const int i = begin + j * 32 + lane;
            vreg[j] = i < end ? ptx::ld_dependent(r + i) : -1;
        }
        for (int c = lane; c < C; c += 32) hist[warp][c] = 0;
        __syncwarp();
        // A token's rank among its adapter's in the warp's range comes from the first walk: tokens of the steps before (the histogram so far)
        // and of the lanes before (one ballot per bit of the adapter index; bits above the highest change nothing).  With a match per
        // step and the same again for the scatter, 2048 tokens of 36 sets took 9800 cycles (four projections, 3001 tokens spread over 256 adapters
        // 47.8 us, so 43.7; a top-2 layer of 600 tokens 31.3 / 30.5).
        bool bad = false;
        int pos[STEPS];
#pragma unroll
        for (int j = 0; j < STEPS; ++j) {
            if (begin + j * 32 < end) {
                bad |= (vreg[j] < -1) || (vreg[j] >= C);
                if (vreg[j] >= C) vreg[j] = -1;
                const int v = vreg[j];
                unsigned same = __ballot_sync(0xFFFFFFFFu, v >= 0);
#pragma unroll
                for (int b = 0; b < 8; ++b) {
                    const unsigned m = __ballot_sync(0xFFFFFFFFu, (v >> b) & 1);
                    same &= m ^ (((unsigned)v >> b & 1u) - 1u);            // (m where my bit is set, ~m where it is not)
                }
                const int before = v >= 0 ? hist[warp][v] : 0, mine = __popc(same & lt_mask);
                pos[j] = before + mine;
                __syncwarp();
                if (v >= 0 && mine == 0) hist[warp][v] = before + __popc(same);
                __syncwarp();
            }
        }
        __syncthreads();
        // exclusive prefix over the warps, per adapter; the totals are the histogram
        for (int c = tid; c < C; c += NT) {
            int run = 0;
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                const int t = hist[w][c];
                hist[w][c] = run;
                run += t;
            }
            tstart_s[c] = run;                 // counts, until the tile prefix replaces them below
        }
        __syncthreads();
        if (warp == 0) {                       // exclusive prefix over adapters, eight consecutive adapters per lane
            int local[8], sum = 0;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int c = lane * 8 + j;
                local[j] = c < C ? tstart_s[c] : 0;
                sum += local[j];
            }
            if ((write_out && blockIdx.x == 0)) {
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (lane * 8 + j < C) counts_out[lane * 8 + j] = local[j];
            }
            int incl = sum;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int up = __shfl_up_sync(0xFFFFFFFFu, incl, off);
                if (lane >= off) incl += up;
            }
            int run = incl - sum;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int c = lane * 8 + j;
                if (c <= C) offs_s[c] = run;
                run += local[j];
            }
            if (lane == 31 && C == MOLORA_MAX_ADAPTERS) offs_s[MOLORA_MAX_ADAPTERS] = run;
        }
        __syncthreads();
        // stable scatter into the CTA's copy of perm
#pragma unroll
        for (int j = 0; j < STEPS; ++j)
            if (vreg[j] >= 0 && begin + j * 32 < end) perm_s[offs_s[vreg[j]] + hist[warp][vreg[j]] + pos[j]] = begin + j * 32 + lane;
        if ((write_out && blockIdx.x == 0)) {
            for (int c = tid; c <= C; c += NT) offsets_out[c] = offs_s[c];
            if (dev_status != nullptr && __any_sync(0xFFFFFFFFu, bad) && lane == 0) atomicOr(dev_status, MOLORA_DEV_BAD_ROUTE);
        }
        __syncthreads();
      }
        if (tile_rows > 0) {
            if (warp == 0) tile_starts(offs_s, C_, tile_rows, 1, INT32_MAX, tstart_s);
            __syncthreads();
        }
}

// Writes the CTA's slice of perm out, with `threads` threads numbered from `tid`.
__device__ __forceinline__ void group_write_perm(const int32_t* perm_s, int total, int32_t* perm_out, int tid, int threads)
{
    const int per = (total + (int)gridDim.x - 1) / (int)gridDim.x;
    const int lo = (int)blockIdx.x * per, hi = min(lo + per, total);
#pragma unroll 1
    for (int i = lo + tid; i < hi; i += threads) perm_out[i] = perm_s[i];
}

}  // namespace molora
