// Grouped LoRA shrink -> expand on CUDA cores (Eq. 2 evaluated segment by segment, Figure 2 right).
//
// This is the path for small segments (decode-sized batches) and for fp32 storage.  One CTA owns a
// tile of TM = 128 / rank consecutive positions of one segment (all rows of a tile share adapter c):
//
//   shrink  t[m][n] = sum_k x[row_m][k] * A_c[k][n]
//           the 256 threads split d_in in 16-byte vectors; thread-local partial sums for the whole
//           TM x rank tile (128 fp32 registers) are finished by one butterfly reduce-scatter per warp
//           and a cross-warp add through shared memory.  x is streamed once with 128-bit loads;
//           A_c rows (rank elements, contiguous) come through L1/L2.
//   expand  y[row_m][o] += scale * sum_n t[m][n] * B_c[n][o]
//           the threads split d_out in 16-byte vectors; t is broadcast from shared memory, B_c rows
//           are read with coalesced 128-bit loads, y is read, updated in fp32 and stored once (one
//           rounding to the storage type) at the token's original row.
//
// The intermediate t never leaves the chip.  Tiles are located on the device from `offsets`
// (no host read of the histogram), so the grid is sized for the worst case and surplus CTAs exit.
#include "common.cuh"
#include "group_inline.cuh"
#include "sm100_ptx.cuh"
#include "warp_reduce.cuh"

namespace molora {

struct ApplyBatchParams {
    molora_proj_desc_t p[MOLORA_MAX_PROJECTIONS];
    const int32_t* offsets;
    const int32_t* perm;
    int32_t P;
    int32_t C;
    int32_t max_rows;     // segments with at least this many rows belong to the tensor-core kernel
    // grouping variant only: the routing decisions and where counts / offsets / perm are written (as by molora_group)
    const int32_t* r;
    int32_t* counts_out;
    int32_t* offsets_out;
    int32_t* perm_out;
    uint32_t* dev_status;
    int32_t N;
};

constexpr int kRowTileThreads = 256;
constexpr int kRowTileGroupMaxN = 2048;
// what group_in_cta needs, all of it static: offsets, temporary words, perm and its scratch
struct RowTileGroup {
    int32_t offs[MOLORA_MAX_ADAPTERS + 1], tmp[MOLORA_MAX_ADAPTERS + 1], perm[kRowTileGroupMaxN];
    alignas(16) unsigned char scratch[kGroupInCtaScratch<kRowTileThreads>];
};

// GROUP: the call starts from the routing decisions r (at most kRowTileGroupMaxN tokens); every CTA groups them on chip, which costs
// it ~1 us against a grouping launch of 3.4 us and the gap behind it (256 fp32 tokens 512 wide, vocabulary routing included: 15.4 us
// in three launches, 12.3 in two).
template <typename T, int R, bool GROUP>
__global__ void __launch_bounds__(kRowTileThreads, 1) apply_rowtile_kernel(const __grid_constant__ ApplyBatchParams prm)
{
    constexpr int VEC = VecTraits<T>::kElems;
    constexpr int TM = 128 / R;              // rows per tile: TM * R = 128 partial sums per thread
    constexpr int WARPS = kRowTileThreads / 32;
    constexpr int RV = R / VEC;              // 16-byte vectors per row of A_c

    ptx::grid_dependency_sync();             // (launched under its predecessor, whatever that is)
    const molora_proj_desc_t& pd = prm.p[blockIdx.y];
    if (pd.rank != R) return;                // a launch of this instantiation serves the projections of rank R

    int seg, row0, rows;
    const int32_t* perm_s = nullptr;
    if constexpr (GROUP) {
        __shared__ RowTileGroup grp;
        group_in_cta<kRowTileThreads, kRowTileGroupMaxN>(prm.r, prm.N, prm.C, grp.offs, grp.tmp, grp.perm, grp.scratch, 0, blockIdx.y == 0,
                                                         prm.counts_out, prm.offsets_out, prm.dev_status);
        if (blockIdx.y == 0) group_write_perm(grp.perm, grp.offs[prm.C], prm.perm_out, threadIdx.x, kRowTileThreads);
        if (!find_tile_smem(grp.offs, prm.C, TM, blockIdx.x, 1, INT32_MAX, seg, row0, rows)) return;
        perm_s = grp.perm;
    } else {
        if (!find_tile(prm.offsets, prm.C, TM, blockIdx.x, 1, prm.max_rows, seg, row0, rows)) return;
    }

    __shared__ __align__(16) float partial[WARPS][128];
    __shared__ __align__(16) float t_s[128];   // [TM][R]
    __shared__ int32_t row_s[TM];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid < TM) {
        const int pos = row0 + (tid < rows ? tid : rows - 1);                              // pad with the last row
        row_s[tid] = GROUP ? perm_s[pos] : ptx::ld_dependent(prm.perm + pos);
    }
    __syncthreads();

    const int d_in = pd.d_in, d_out = pd.d_out;
    const T* __restrict__ x = static_cast<const T*>(pd.x);
    T* __restrict__ y = static_cast<T*>(pd.y);
    const T* __restrict__ Ac = static_cast<const T*>(pd.A) + (int64_t)seg * d_in * R;
    const T* __restrict__ Bc = static_cast<const T*>(pd.B) + (int64_t)seg * R * d_out;

    // ---------------- shrink ----------------
    float acc[TM * R];
#pragma unroll
    for (int i = 0; i < TM * R; ++i) acc[i] = 0.f;

    for (int k0 = tid * VEC; k0 < d_in; k0 += kRowTileThreads * VEC) {
        uint4 xp[TM];
#pragma unroll
        for (int m = 0; m < TM; ++m) xp[m] = ld128_rw_stream(x + (int64_t)row_s[m] * pd.ldx + k0);
#pragma unroll
        for (int j = 0; j < VEC; ++j) {
            float af[R];
#pragma unroll
            for (int v = 0; v < RV; ++v) unpack<T>(ptx::ld_dependent(reinterpret_cast<const uint4*>(Ac + (int64_t)(k0 + j) * R + v * VEC)), af + v * VEC);
#pragma unroll
            for (int m = 0; m < TM; ++m) {
                float xv[VEC];
                unpack<T>(xp[m], xv);
#pragma unroll
                for (int n = 0; n < R; ++n) acc[m * R + n] = fmaf(xv[j], af[n], acc[m * R + n]);
            }
        }
    }

    warp_reduce_scatter<128>(acc, lane);
    {
        const int base = reduce_scatter_base<128>(lane);
        *reinterpret_cast<float4*>(&partial[warp][base]) = make_float4(acc[0], acc[1], acc[2], acc[3]);
    }
    __syncthreads();
    if (tid < 128) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < WARPS; ++w) s += partial[w][tid];
        // fold the LoRA scale (and the token's routing weight, if given) into t once: t_s is [TM][R], row m = tid / R
        const float rs = pd.row_scale != nullptr ? ptx::ld_dependent(pd.row_scale + row_s[tid / R]) : 1.f;
        t_s[tid] = s * pd.scale * rs;
    }
    __syncthreads();

    // ---------------- expand ----------------
    for (int o0 = tid * VEC; o0 < d_out; o0 += kRowTileThreads * VEC) {
        uint4 yp[TM];
#pragma unroll
        for (int m = 0; m < TM; ++m) yp[m] = ld128_rw_stream(y + (int64_t)row_s[m] * pd.ldy + o0);
        float out[TM][VEC];
#pragma unroll
        for (int m = 0; m < TM; ++m)
#pragma unroll
            for (int j = 0; j < VEC; ++j) out[m][j] = 0.f;
#pragma unroll
        for (int n4 = 0; n4 < R; n4 += 4) {
            float bf[4][VEC];
#pragma unroll
            for (int q = 0; q < 4; ++q) unpack<T>(ptx::ld_dependent(reinterpret_cast<const uint4*>(Bc + (int64_t)(n4 + q) * d_out + o0)), bf[q]);
#pragma unroll
            for (int m = 0; m < TM; ++m) {
                const float4 tv = *reinterpret_cast<const float4*>(&t_s[m * R + n4]);
#pragma unroll
                for (int j = 0; j < VEC; ++j) {
                    out[m][j] = fmaf(tv.x, bf[0][j], out[m][j]);
                    out[m][j] = fmaf(tv.y, bf[1][j], out[m][j]);
                    out[m][j] = fmaf(tv.z, bf[2][j], out[m][j]);
                    out[m][j] = fmaf(tv.w, bf[3][j], out[m][j]);
                }
            }
        }
#pragma unroll
        for (int m = 0; m < TM; ++m) {
            if (m < rows) {
                float yv[VEC];
                unpack<T>(yp[m], yv);
#pragma unroll
                for (int j = 0; j < VEC; ++j) yv[j] += out[m][j];
                stg128(y + (int64_t)row_s[m] * pd.ldy + o0, pack<T>(yv));
            }
        }
    }
}

template <typename T, int R, bool GROUP>
static cudaError_t rowtile_launch(const ApplyBatchParams& prm, int64_t N, cudaStream_t s)
{
    constexpr int TM = 128 / R;
    // every segment adds at most one partial tile; with a row cap only min(N, C * cap) rows can come here
    const int64_t cap_rows = prm.max_rows == INT32_MAX ? N : (N < (int64_t)prm.C * prm.max_rows ? N : (int64_t)prm.C * prm.max_rows);
    const int64_t tiles = ceil_div64(cap_rows, TM) + prm.C;
    dim3 grid((unsigned)tiles, (unsigned)prm.P);
    return launch_kernel(apply_rowtile_kernel<T, R, GROUP>, grid, dim3(kRowTileThreads), 0, s, 1, true, prm);
}

template <typename T, bool GROUP>
static cudaError_t rowtile_dispatch(const ApplyBatchParams& prm, int64_t N, cudaStream_t s)
{
    bool has[4] = {false, false, false, false};
    for (int i = 0; i < prm.P; ++i) {
        const int r = prm.p[i].rank;
        has[r == 8 ? 0 : r == 16 ? 1 : r == 32 ? 2 : 3] = true;
    }
    cudaError_t e = cudaSuccess;
    if (has[0] && e == cudaSuccess) e = rowtile_launch<T, 8, GROUP>(prm, N, s);
    if (has[1] && e == cudaSuccess) e = rowtile_launch<T, 16, GROUP>(prm, N, s);
    if (has[2] && e == cudaSuccess) e = rowtile_launch<T, 32, GROUP>(prm, N, s);
    if (has[3] && e == cudaSuccess) e = rowtile_launch<T, 64, GROUP>(prm, N, s);
    return e;
}

static ApplyBatchParams rowtile_params(const molora_proj_desc_t* projs, int32_t P, int32_t C, int32_t max_rows)
{
    ApplyBatchParams prm{};
    for (int i = 0; i < P; ++i) prm.p[i] = projs[i];
    prm.P = P;
    prm.C = C;
    prm.max_rows = max_rows;
    return prm;
}

molora_status_t launch_apply_rowtile(const molora_proj_desc_t* projs, int32_t P, molora_dtype_t dt, int64_t N,
                                     int32_t C, const int32_t* offsets, const int32_t* perm, int32_t max_rows,
                                     cudaStream_t s)
{
    if (N == 0 || P == 0) return MOLORA_OK;
    ApplyBatchParams prm = rowtile_params(projs, P, C, max_rows);
    prm.offsets = offsets;
    prm.perm = perm;
    return cuda_ok(dt == MOLORA_BF16 ? rowtile_dispatch<__nv_bfloat16, false>(prm, N, s) : rowtile_dispatch<float, false>(prm, N, s));
}

// Grouping and apply in one launch: calls that go to this kernel with one rank (fp32 storage, or rank 8) while every tile has an SM
// of its own -- a second wave would group again.  The launch-count queries ask this of descriptors that nobody has checked: what
// molora_group_apply_batched refuses is no launch of this kernel.
bool group_apply_rowtile_eligible(const molora_proj_desc_t* projs, int32_t P, molora_dtype_t dt, int64_t N, int32_t C)
{
    const int32_t rank = projs[0].rank;
    if (rank != 8 && rank != 16 && rank != 32 && rank != 64) return false;
    if (dt != MOLORA_F32 && (dt != MOLORA_BF16 || rank != 8)) return false;
    if (N < 1 || N > kRowTileGroupMaxN || C < 1 || C > MOLORA_MAX_ADAPTERS) return false;
    for (int i = 0; i < P; ++i) {
        const molora_proj_desc_t& p = projs[i];
        if (p.rank != rank || p.d_in <= 0 || p.d_out <= 0 || (p.d_in % 8) != 0 || (p.d_out % 8) != 0 || decode_eligible(p, dt)) return false;
    }
    return (ceil_div64(N, 128 / rank) + C) * P <= sm_count();
}

molora_status_t launch_group_apply_rowtile(const int32_t* r, const molora_proj_desc_t* projs, int32_t P, molora_dtype_t dt, int64_t N,
                                           int32_t C, int32_t* counts, int32_t* offsets, int32_t* perm, uint32_t* dev_status,
                                           cudaStream_t s)
{
    ApplyBatchParams prm = rowtile_params(projs, P, C, INT32_MAX);
    prm.r = r;
    prm.counts_out = counts;
    prm.offsets_out = offsets;
    prm.perm_out = perm;
    prm.dev_status = dev_status;
    prm.N = (int32_t)N;
    return cuda_ok(dt == MOLORA_BF16 ? rowtile_dispatch<__nv_bfloat16, true>(prm, N, s) : rowtile_dispatch<float, true>(prm, N, s));
}

}  // namespace molora
