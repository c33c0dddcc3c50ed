// kinetic_impl.cuh -- the plasma-row kernel template and its launch for one
// (lanes per row, vectors per lane) shape; instantiated per storage type in
// kinetic.cu (FP32), kinetic_bf16.cu and kinetic_f64.cu.
#pragma once

#include "kinetic_row.cuh"

namespace fp {

template <typename TS, typename TA, int VPL, int L, int VS = VPL>   // VS: vectors a partial sum (row_update_to)
__global__ void __launch_bounds__(256) k_kinetic(KinArgs<TA> a)
{
    // What no kernel before this one writes is fetched before the grid dependency: the tables, and of the first
    // row group the cell index and the delta-f vectors.  Within a sequence of steps only this kernel writes delta f,
    // and between two of its launches lies a stencil launch that waits for the first one before it lets the next
    // start, so the rows are final; the loads then overlap the stencil's last wave (5 k rows of 1024 nodes on a
    // 192 x 160 grid: 14.6 -> 12.3 us a step).  The second half of a split step may follow a write of delta f
    // instead, so it is launched without the overlap (a.after_stencil).
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TA *s_tab = reinterpret_cast<TA *>(smem_raw);
    for (int t = threadIdx.x; t < 3 * a.pitch; t += blockDim.x) s_tab[t] = a.tab[t];
    const TA *s_al = s_tab, *s_be = s_tab + a.pitch, *s_w = s_tab + 2 * a.pitch;

    using V = typename Vec<TS>::type;
    constexpr int VEC = Vec<TS>::n;
    constexpr int R = 32 / L;   // rows per warp
    const int lane = threadIdx.x & 31;
    const int sub = lane / L, l = lane % L;
    const int64_t wg = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const uint2 key = make_uint2((uint32_t)a.seed, (uint32_t)(a.seed >> 32));

    // the slot -> cell index of the next row group is fetched one iteration
    // ahead, so the E gather of a row issues together with its delta-f loads
    int64_t row = wg * R + sub;
    int32_t cell_next = row < a.nslots ? __ldg(a.slot_cell + row) : 0;
    // (not the shortest BF16 rows: one more condition in their loop costs them a CTA a SM and 10 %)
    constexpr bool kEarly = !(std::is_same<TS, __nv_bfloat16>::value && VPL * L <= 8);
    // Rows a lane each: consecutive vectors share a 32-byte sector, so the lines stay in L1 by the plain policy until
    // the row is loaded (streaming loads give them up early: 2.1 GB of 32-node BF16 rows 808 -> 772 us, of 16-node
    // FP32 rows 892 -> 840, of 16-node BF16 rows 864 -> 847).  Two-vector FP32 rows and longer ones are no faster with
    // it, or hardly (8-node FP32 840 -> 860, 64-node BF16 760 both, 32-node FP32 700 -> 694), and keep the streaming
    // hint (profiles/probes_rows_fp64_lines.md).
    constexpr bool kShared = L == 1 && !std::is_same<TS, double>::value &&
                             (VPL == 4 || (VPL == 2 && std::is_same<TS, __nv_bfloat16>::value));
    V v[VPL];
    if (kEarly && row < a.nslots) {
        const V *rp = reinterpret_cast<const V *>(a.df) + row * (a.pitch / VEC);
#pragma unroll
        for (int q = 0; q < VPL; ++q) v[q] = __ldcg(rp + q * L + l);   // (from L2, where the writes are)
    }
    __syncthreads();
    pdl_enter();
    const int64_t step = *a.d_step + a.kstep;
    bool loaded = kEarly;   // v holds the first group's rows
    for (int64_t base = wg * R; base < a.nslots; base += nw * R) {
        row = base + sub;
        const bool valid = row < a.nslots;
        const int32_t cell = cell_next;
        TA E = TA(0), nE = TA(0);
        V *rp = reinterpret_cast<V *>(a.df) + (valid ? row : 0) * (a.pitch / VEC);
        if (valid) {
            if (!kEarly || !loaded) {
#pragma unroll
                for (int q = 0; q < VPL; ++q) v[q] = kShared ? rp[q * L + l] : __ldcs(rp + q * L + l);
            }
            E = a.E[cell];
            nE = __ldg(a.dens + row) * E;
        }
        loaded = false;
        const int64_t row_next = row + nw * R;
        cell_next = row_next < a.nslots ? __ldg(a.slot_cell + row_next) : 0;
        TA s = TA(0), c = TA(0);
        if (valid) row_update<TS, TA, VPL, L, VS>(rp, v, s_al, s_be, s_w, nE, l, (uint32_t)(row + a.slot_base), step, key, s, c);
        const TA J = row_reduce<TA, L>(s, c);
        if (valid && l == 0) {
            if (a.store_j) a.jslot[row] = J;
            a.E[cell] = E - a.cj * J;
        }
    }
}

template <typename TS, typename TA, int VPL, int L, int VS = VPL>
cudaError_t run_kinetic(cudaStream_t st, const KinArgs<TA> &a, int num_sms, int blocks_per_sm)
{
    auto kern = k_kinetic<TS, TA, VPL, L, VS>;
    const size_t smem = 3 * (size_t)a.pitch * sizeof(TA);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 256, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    if (blocks_per_sm > 0 && blocks_per_sm < per_sm) per_sm = blocks_per_sm;
    const int64_t rows_per_block = (256 / 32) * (32 / L);
    int64_t blocks = (a.nslots + rows_per_block - 1) / rows_per_block;
    const int64_t cap = (int64_t)num_sms * per_sm;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    if (a.after_stencil) launch_pdl(kern, dim3((unsigned)blocks), dim3(256), smem, st, a);
    else launch_plain(kern, dim3((unsigned)blocks), dim3(256), smem, st, a);
    return cudaGetLastError();
}

// Shape candidates (VPL, L) for V vectors per row.  The first keeps >= 4 sixteen-byte loads a lane in flight when the
// row allows it; kinetic_default_shape takes it except where another measured faster.
inline int kinetic_shape_candidates(int V, int (*out)[2])
{
    static const int tab[][2] = {{1, 1},
                                 {2, 1}, {1, 2},
                                 {4, 1}, {2, 2}, {1, 4},
                                 {4, 2}, {8, 1}, {2, 4}, {1, 8},
                                 {4, 4}, {8, 2}, {2, 8}, {1, 16},
                                 {4, 8}, {8, 4}, {2, 16}, {1, 32},
                                 {4, 16}, {8, 8}, {2, 32},
                                 {4, 32}, {8, 16}, {16, 8},
                                 {8, 32}, {16, 16},
                                 {16, 32}};
    int n = 0;
    for (const auto &p : tab)
        if (p[0] * p[1] == V) { out[n][0] = p[0]; out[n][1] = p[1]; ++n; }
    return n;
}

template <typename TS, typename TA>
cudaError_t dispatch_kinetic(cudaStream_t st, const KinArgs<TA> &a, int num_sms, int vpl, int l, int bps)
{
    switch (vpl * 64 + l) {
#define FP_KCASE(V_, L_) \
    case V_ * 64 + L_: return run_kinetic<TS, TA, V_, L_>(st, a, num_sms, bps);
    FP_KCASE(1, 1) FP_KCASE(2, 1) FP_KCASE(1, 2) FP_KCASE(4, 1) FP_KCASE(2, 2) FP_KCASE(1, 4)
    FP_KCASE(4, 2) FP_KCASE(8, 1) FP_KCASE(2, 4) FP_KCASE(1, 8) FP_KCASE(4, 4) FP_KCASE(8, 2) FP_KCASE(2, 8)
    FP_KCASE(1, 16) FP_KCASE(4, 8) FP_KCASE(8, 4) FP_KCASE(2, 16) FP_KCASE(1, 32) FP_KCASE(4, 16) FP_KCASE(8, 8)
    FP_KCASE(2, 32) FP_KCASE(4, 32) FP_KCASE(8, 16) FP_KCASE(16, 8) FP_KCASE(8, 32) FP_KCASE(16, 16)
    FP_KCASE(16, 32)
#undef FP_KCASE
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace fp
