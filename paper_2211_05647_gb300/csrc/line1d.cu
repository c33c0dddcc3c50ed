// line1d.cu -- many steps of one 1-D grid in one cooperative launch: the H
// update, the Sec. 5.2 row update with its J moment, the E update with the soft
// source and the Mur ends (the step of Sec. 2 and Sec. 5.2), the whole state
// held in shared memory from the first step to the last.
//
// A 1-D step is a fraction of a microsecond of work; as three dependent launches
// it costs their latencies (10.3 us a step in FP64, 6 us in FP32, at 2000 cells).
// Here the line is cut into one contiguous range of nodes per CTA (equal cost,
// rows counted), a CTA keeps E, H and the delta-f rows of its range in shared
// memory, and neighbouring CTAs exchange one E value each way per step:
//   phase A: rows (J from E^n, df updated) and H^{n+1/2} of the range, while one
//            warp a side waits for the neighbour's E^n and forms the H node that
//            needs it (H at the lower cut is formed by both neighbours, from the
//            same values by the same operations)
//   phase B: E^{n+1} of the range, the edge values sent to the neighbours
// with a block barrier after each, so the exchange's L2 round trip hides behind
// the rows.  A mailbox word carries 32 bits of the value and the step's 32-bit
// tag in one 64-bit access (a double takes two words), so no fence or separate
// flag is needed; boxes alternate by step parity, and a neighbour can be at most
// one step ahead, since it needs this CTA's value of the step before.  Tags grow
// across launches.  Range ends are read before anything is sent and written back
// after the neighbours' first message, so no CTA reads what another has already
// overwritten.  Waits are bounded (1 s of wall-clock time): a CTA that gives up
// sets bit 4 of the error word and returns, and its neighbours follow.
//
// Bound by the exchange and barrier latencies while a CTA has few rows (2000 cells,
// 500 rows of 64 nodes: 0.97 us a step against 6.0 for the three launches), by
// shared memory when it has many (110 k cells, 100 k BF16 rows of 64 nodes: 6.3
// against 11.5), in FP64 by the FP64 pipe on the rows (the 500 rows 2.3 against
// 13.1 us; 100 k rows of 16 nodes 28 against 54).
#include "async.cuh"
#include "kinetic_row.cuh"
#include "line1d.cuh"
#include "stencil_common.cuh"

namespace fp {

namespace {

constexpr int kLineWarps = kLineThreads / 32;
constexpr int kRowWarps = kLineWarps - 2;          // the last two warps take the neighbours' messages
constexpr int kSrcChunk = 64;                      // source values formed at a time, one a thread
constexpr uint64_t kLineWaitNs = 1000000000ull;

template <typename T>
__device__ __forceinline__ void mail_put(uint64_t *box, T v, uint32_t tag)
{
    const uint64_t t = (uint64_t)tag << 32;
    if constexpr (sizeof(T) == 4) {
        asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(box), "l"(t | __float_as_uint(v)) : "memory");
    } else {
        const uint64_t b = (uint64_t)__double_as_longlong(v);
        asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(box), "l"(t | (b & 0xffffffffu)),
                     "l"(t | (b >> 32))
                     : "memory");
    }
}

// wait for the message tagged `tag`; false if it did not come in time.  The neighbour runs: a cooperative grid
// starts when all of its CTAs can be resident, and none of them before (beside a launch of another stream that
// held 32 SMs for 3.6 s, all 152 started at its end), so it answers within microseconds.
template <typename T>
__device__ __forceinline__ bool mail_get(const uint64_t *box, T &v, uint32_t tag, uint64_t limit_ns = kLineWaitNs)
{
    uint64_t t0 = 0;
    for (uint32_t it = 1;; ++it) {
        if constexpr (sizeof(T) == 4) {
            uint64_t w;
            asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(box) : "memory");
            if ((uint32_t)(w >> 32) == tag) {
                v = __uint_as_float((uint32_t)w);
                return true;
            }
        } else {
            uint64_t w0, w1;
            asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(w0), "=l"(w1) : "l"(box) : "memory");
            if ((uint32_t)(w0 >> 32) == tag && (uint32_t)(w1 >> 32) == tag) {
                v = __longlong_as_double((long long)((w1 << 32) | (w0 & 0xffffffffu)));
                return true;
            }
        }
        if ((it & 127u) == 0) {
            const uint64_t t = globaltimer_ns();
            if (!t0) t0 = t;
            else if (t - t0 > limit_ns) return false;
        }
    }
}

// dynamic shared memory: w' / alpha / beta tables, rows, E, H and J of the range (a node of halo on either
// side), densities, source values, row -> node
template <typename TS, typename TA>
struct LineSmem {
    size_t tab, df, e, h, j, dn, g, node, total;
    __host__ __device__ LineSmem(int pitch, int rows, int nodes)
    {
        auto up = [](size_t b) { return (b + 15) & ~(size_t)15; };
        tab = 0;
        df = up(3 * (size_t)pitch * sizeof(TA));
        e = df + up((size_t)rows * pitch * sizeof(TS));
        h = e + up((size_t)(nodes + 2) * sizeof(TA));
        j = h + up((size_t)(nodes + 2) * sizeof(TA));
        dn = j + up((size_t)(nodes + 2) * sizeof(TA));
        g = dn + up((size_t)rows * sizeof(TA));
        node = g + up(kSrcChunk * sizeof(TA));
        total = node + up((size_t)rows * sizeof(int));
    }
};

template <typename TS, typename TA, int VPL, int L>
__global__ void __launch_bounds__(kLineThreads, 1) k_line1d(LineArgs<TA> a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_dead;
    using V = typename Vec<TS>::type;
    constexpr int VEC = Vec<TS>::n, R = 32 / L;
    const LineSmem<TS, TA> lay(a.pitch, a.rows_max, a.nodes_max);
    TA *s_al = reinterpret_cast<TA *>(smem_raw + lay.tab), *s_be = s_al + a.pitch, *s_w = s_be + a.pitch;
    V *s_df = reinterpret_cast<V *>(smem_raw + lay.df);
    TA *sE = reinterpret_cast<TA *>(smem_raw + lay.e), *sH = reinterpret_cast<TA *>(smem_raw + lay.h);
    TA *sJ = reinterpret_cast<TA *>(smem_raw + lay.j), *s_dn = reinterpret_cast<TA *>(smem_raw + lay.dn);
    TA *s_g = reinterpret_cast<TA *>(smem_raw + lay.g);
    int *s_node = reinterpret_cast<int *>(smem_raw + lay.node);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int sub = lane / L, l = lane % L;
    const int b = blockIdx.x, nb = gridDim.x, nz = a.nz;
    const int k0 = a.cut[b], nk = a.cut[b + 1] - k0;               // nodes [k0, k0 + nk): index i = k - k0 + 1
    const int s0 = a.slot_cut[b], nr = a.slot_cut[b + 1] - s0;     // their plasma slots
    const int vpr = a.pitch / VEC;
    const uint2 key = make_uint2((uint32_t)a.seed, (uint32_t)(a.seed >> 32));
    const bool src_here = a.src.kind && a.src.k >= k0 && a.src.k < k0 + nk;

    V *df = reinterpret_cast<V *>(a.df) + (int64_t)s0 * vpr;
    for (int t = tid; t < nr * vpr; t += kLineThreads) s_df[t] = __ldcs(df + t);
    for (int t = tid; t < 3 * a.pitch; t += kLineThreads) s_al[t] = a.tab[t];
    for (int r = tid; r < nr; r += kLineThreads) {
        s_node[r] = a.slot_cell[s0 + r] - k0 + 1;
        s_dn[r] = a.dens[s0 + r];
    }
    for (int i = tid; i < nk + 2; i += kLineThreads) {
        const int k = k0 - 1 + i;
        sE[i] = i >= 1 && i <= nk ? a.E[k] : TA(0);
        sH[i] = i <= nk && k >= 0 && k < nz ? a.H[k] : TA(0);
        sJ[i] = TA(0);
    }
    if (tid == 0) s_dead = 0;
    __syncthreads();
    // the boxes of this CTA: [side (0 from below, 1 from above)][parity][2 words]
    const uint64_t *box = a.mail + (size_t)b * 8;
    auto send = [&](int side, TA v, uint32_t tag) {   // side 0: to the CTA above (its box from below)
        uint64_t *to = a.mail + (size_t)(side ? b - 1 : b + 1) * 8 + side * 4 + (tag & 1u) * 2;
        mail_put<TA>(to, v, tag);
    };
    if (tid == 0) {
        __threadfence();
        if (b > 0) send(1, sE[1], a.seq);
        if (b < nb - 1) send(0, sE[nk], a.seq);
    }

    for (int s = 0; s < a.nsteps; ++s) {
        const uint32_t tag = a.seq + (uint32_t)s;
        const int64_t step = a.step0 + s;
        // ---- phase A: J and the rows from E^n, H^{n+1/2}
        if (warp >= kRowWarps) {
            if (lane == 0) {
                const int side = warp - kRowWarps;     // 0: the CTA below, 1: the CTA above
                if (side ? b < nb - 1 : b > 0) {
                    TA v = TA(0);
                    if (!mail_get<TA>(box + side * 4 + (tag & 1u) * 2, v, tag)) {
                        atomicOr(a.err, 4);
                        s_dead = 1;
                    }
                    if (side) sH[nk] -= a.ch * (v - sE[nk]);
                    else sH[0] -= a.ch * (sE[1] - v);
                }
            }
        } else {
            if (src_here && s % kSrcChunk == 0 && tid < kSrcChunk && s + tid < a.nsteps)
                s_g[tid] = (TA)source_value(a.src, (double)(step + tid + 1) * a.src.dt);
            for (int i = 1 + tid; i < nk; i += kRowWarps * 32) sH[i] -= a.ch * (sE[i + 1] - sE[i]);
            // few FP32 rows are spread over the warps; FP64 rows fill warps (see dispatch_line)
            for (int r0 = 0; r0 < nr; r0 += kRowWarps * R) {
                const int r = r0 + (sizeof(TA) == 8 ? warp * R + sub : sub * kRowWarps + warp);
                if (r0 + (sizeof(TA) == 8 ? warp * R : warp) >= nr) break;   // none of the warp's rows
                const bool valid = r < nr;
                TA sm = TA(0), cm = TA(0);
                int node = 0;
                if (valid) {
                    V *rp = s_df + r * vpr, v[VPL];
#pragma unroll
                    for (int q = 0; q < VPL; ++q) v[q] = rp[q * L + l];
                    node = s_node[r];
                    const TA nE = s_dn[r] * sE[node];
                    row_update_to<TS, TA, VPL, L, VPL>(v, s_al, s_be, s_w, nE, l, (uint32_t)(s0 + r), step, key, sm, cm,
                                                  [&](int vi, const V &x) { rp[vi] = x; });
                }
                const TA J = row_reduce<TA, L>(sm, cm);
                if (valid && l == 0) sJ[node] = J;
            }
        }
        __syncthreads();
        if (s_dead) return;
        // ---- phase B: E^{n+1}, the source, the Mur ends; the edges to the neighbours
        const bool last = s + 1 == a.nsteps;
        for (int i = 1 + tid; i <= nk; i += kLineThreads) {
            const int k = k0 - 1 + i;
            if (k < 1 || k >= nz) continue;
            const TA e = sE[i];                       // E^n
            TA v = nr > 0 ? e - a.cj * sJ[i] : e;     // E^n - dt/eps0 J (J = 0 outside the plasma)
            v = v - a.ce * (sH[i] - sH[i - 1]);
            if (src_here && k == (int)a.src.k) v += s_g[s % kSrcChunk];
            sE[i] = v;
            if (a.mur) {
                if (k == 1) sE[i - 1] = e + a.m * (v - sE[i - 1]);
                if (k == nz - 1) sE[i + 1] = e + a.m * (v - sE[i + 1]);
                if (last && k == 1) a.mur[0] = e;
                if (last && k == nz - 1) a.mur[1] = e;
            }
            if (!last) {
                if (i == 1 && b > 0) send(1, v, tag + 1u);
                if (i == nk && b < nb - 1) send(0, v, tag + 1u);
            }
        }
        __syncthreads();
    }

    for (int t = tid; t < nr * vpr; t += kLineThreads) __stcs(df + t, s_df[t]);
    for (int r = tid; r < nr; r += kLineThreads) a.jslot[s0 + r] = sJ[s_node[r]];
    for (int i = 1 + tid; i <= nk; i += kLineThreads) {
        const int k = k0 - 1 + i;
        a.E[k] = sE[i];
        if (k < nz) a.H[k] = sH[i];
    }
    if (b == 0 && tid == 0) *a.d_step = a.step0 + a.nsteps;
}

template <typename TS, typename TA, int VPL, int L>
cudaError_t run_line(cudaStream_t st, const LineArgs<TA> &a, int ctas)
{
    auto kern = k_line1d<TS, TA, VPL, L>;
    const size_t smem = LineSmem<TS, TA>(a.pitch, a.rows_max, a.nodes_max).total;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3(kLineThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;   // the CTAs wait for one another: all resident at once
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, a);
}

// FP32 and BF16 rows take the shape launch_kinetic picks by default, so J's sums are formed in the same order.
template <typename TS, typename TA>
cudaError_t dispatch_line(cudaStream_t st, const LineArgs<TA> &a, int ctas)
{
    int vpl = 1, l = 1;   // no plasma
    if (a.pitch) kinetic_default_shape(a.pitch, std::is_same<TS, float>::value ? FDTD_DF_F32 : FDTD_DF_BF16, &vpl, &l);
    switch (vpl * 64 + l) {
#define FP_LINE(VPL_, L_) \
    case VPL_ * 64 + L_: return run_line<TS, TA, VPL_, L_>(st, a, ctas);
    FP_LINE(1, 1) FP_LINE(2, 1) FP_LINE(4, 1) FP_LINE(4, 4) FP_LINE(4, 8)
    default: break;
    }
    if constexpr (std::is_same<TS, float>::value) {
        switch (vpl * 64 + l) {
            FP_LINE(2, 4) FP_LINE(8, 8) FP_LINE(8, 16)
        default: return cudaErrorInvalidValue;
        }
    } else {
        switch (vpl * 64 + l) {
            FP_LINE(4, 2) FP_LINE(4, 16) FP_LINE(4, 32)
        default: return cudaErrorInvalidValue;
        }
    }
#undef FP_LINE
}

// FP64 rows: the shape with the fewest FP64 instructions on the busiest sub-core, each of which takes 64 cycles
// whether one lane of the warp or all are active.  A lane's n = 2 V / L nodes take 3 n for the update and the
// product and 4 (n - 1) to sum, a level of the reduction over the row's lanes 5; the warps of a CTA's rows are
// spread over four sub-cores.  2000 cells, 500 rows of 64 nodes, three or four a CTA: 4 x 8 takes 3.4 us a
// step, 1 x 32 2.3.
template <>
cudaError_t dispatch_line<double, double>(cudaStream_t st, const LineArgs<double> &a, int ctas)
{
    const int V = a.pitch / 2;
    if (V > 128) return cudaErrorInvalidValue;
    const int ldef = std::max(V / 4, 1), lmax = std::min(std::max(V, 1), 32);
    int best = ldef, least = 0;
    for (int L = ldef, lg = 0; L <= lmax; L <<= 1) {
        while ((1 << lg) < L) ++lg;
        const int n = 2 * V / L, warps = (a.rows_max * L + 31) / 32;
        const int ops = ((warps + 3) / 4) * (7 * n - 4 + 5 * lg);
        if (L == ldef || ops < least) {
            best = L;
            least = ops;
        }
    }
    switch (std::max(V, 1) / best * 64 + best) {
#define FP_LINE64(VPL_, L_) \
    case VPL_ * 64 + L_: return run_line<double, double, VPL_, L_>(st, a, ctas);
    FP_LINE64(1, 1) FP_LINE64(2, 1) FP_LINE64(1, 2) FP_LINE64(4, 1) FP_LINE64(2, 2) FP_LINE64(1, 4)
    FP_LINE64(4, 2) FP_LINE64(2, 4) FP_LINE64(1, 8) FP_LINE64(4, 4) FP_LINE64(2, 8) FP_LINE64(1, 16)
    FP_LINE64(4, 8) FP_LINE64(2, 16) FP_LINE64(1, 32) FP_LINE64(4, 16) FP_LINE64(2, 32) FP_LINE64(4, 32)
#undef FP_LINE64
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

template <>
cudaError_t launch_line1d<float>(cudaStream_t st, const LineArgs<float> &a, int f_dtype, int ctas)
{
    return f_dtype == FDTD_DF_BF16 ? dispatch_line<__nv_bfloat16, float>(st, a, ctas)
                                   : dispatch_line<float, float>(st, a, ctas);
}
template <>
cudaError_t launch_line1d<double>(cudaStream_t st, const LineArgs<double> &a, int, int ctas)
{
    return dispatch_line<double, double>(st, a, ctas);
}

// one thread waits for a message that never comes
__global__ void k_line_wait_selftest(const uint64_t *box, uint64_t limit_ns, int *gave_up)
{
    float v = 0.0f;
    *gave_up = mail_get<float>(box, v, 1u, limit_ns) ? 0 : 1;
}

size_t line1d_smem_bytes(int f_dtype, int pitch, int rows, int nodes)
{
    if (f_dtype == FDTD_DF_F64) return LineSmem<double, double>(pitch, rows, nodes).total;
    if (f_dtype == FDTD_DF_BF16) return LineSmem<__nv_bfloat16, float>(pitch, rows, nodes).total;
    return LineSmem<float, float>(pitch, rows, nodes).total;
}

}  // namespace fp

using namespace fp;

extern "C" int fdtd_selftest_line_wait(uint32_t limit_us, int32_t *gave_up)
{
    if (!gave_up || limit_us == 0 || limit_us > 1000000u)
        return fp_set_global_error(FDTD_ERR_INVAL, "fdtd_selftest_line_wait: gave_up NULL or limit_us not in 1..10^6");
    uint64_t *d = nullptr;   // the message box and the result
    if (cudaMalloc(&d, 2 * sizeof(uint64_t)) != cudaSuccess)
        return fp_set_global_error(FDTD_ERR_NOMEM, "cudaMalloc failed");
    int h = -1;
    cudaError_t e = cudaMemset(d, 0, 2 * sizeof(uint64_t));
    if (e == cudaSuccess) {
        k_line_wait_selftest<<<1, 1>>>(d, (uint64_t)limit_us * 1000u, reinterpret_cast<int *>(d + 1));
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(&h, d + 1, sizeof(int), cudaMemcpyDeviceToHost);
    cudaFree(d);
    if (e != cudaSuccess) return fp_set_global_error(FDTD_ERR_CUDA, cudaGetErrorString(e));
    *gave_up = h;
    return FDTD_OK;
}
