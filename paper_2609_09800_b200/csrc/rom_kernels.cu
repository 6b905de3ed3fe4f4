// Reduced-order thermal model at run time (Eq. 2): x' = A x + B p + b, T = C x + D p + d, x the state before the
// update.  A few hundred states: one thread block steps the model, a warp per row of the matrices, in double
// (the matrices come from a fit in double; at this size the arithmetic is not what a step costs).
#include <cooperative_groups.h>

#include "device_utils.cuh"

namespace cg = cooperative_groups;

namespace hbf {

constexpr int kRomThreads = 512;

__global__ void __launch_bounds__(kRomThreads)
k_rom_steps(uint32_t n, uint32_t m, uint32_t o, const double *__restrict__ A, const double *__restrict__ B,
            const double *__restrict__ b, const double *__restrict__ C, const double *__restrict__ D,
            const double *__restrict__ d, double *x, const double *__restrict__ power, uint32_t n_steps,
            double *__restrict__ temps_out) {
    extern __shared__ double rom_smem[];                     // x [n], x' [n], p [m]
    double *xs = rom_smem, *xn = rom_smem + n, *ps = rom_smem + 2 * n;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n_warps = kRomThreads / 32;
    for (uint32_t i = tid; i < n; i += kRomThreads) xs[i] = x[i];
    __syncthreads();
    for (uint32_t k = 0; k < n_steps; ++k) {
        for (uint32_t j = tid; j < m; j += kRomThreads) ps[j] = power[(size_t)k * m + j];
        __syncthreads();
        for (uint32_t row = warp; row < n + o; row += n_warps) {          // rows of [A B] first, then rows of [C D]
            const bool out_row = row >= n;
            const uint32_t r = out_row ? row - n : row;
            const double *mx = out_row ? C + (size_t)r * n : A + (size_t)r * n;
            const double *mp = out_row ? D + (size_t)r * m : B + (size_t)r * m;
            double acc = 0.0;
            for (uint32_t j = lane; j < n; j += 32) acc += mx[j] * xs[j];
            for (uint32_t j = lane; j < m; j += 32) acc += mp[j] * ps[j];
#pragma unroll
            for (int s = 16; s > 0; s >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, s);
            if (lane == 0) {
                if (out_row) temps_out[(size_t)k * o + r] = acc + d[r];
                else xn[r] = acc + b[r];
            }
        }
        __syncthreads();
        for (uint32_t i = tid; i < n; i += kRomThreads) xs[i] = xn[i];
        __syncthreads();
    }
    for (uint32_t i = tid; i < n; i += kRomThreads) x[i] = xs[i];
}

// The same steps on a cluster of eight blocks: block c keeps rows [c * rpc, (c + 1) * rpc) of [A B; C D] in its shared
// memory for the whole launch, computes those rows every step and writes its part of x' into the next-state buffer of
// all eight blocks through distributed shared memory; one cluster barrier per step.  Each row is summed in the same
// order as in the single-block kernel, so both give the same bits.
constexpr int kRomClusterBlocks = 8;
constexpr int kRomClusterThreads = 256;

__global__ void __cluster_dims__(kRomClusterBlocks, 1, 1) __launch_bounds__(kRomClusterThreads)
k_rom_steps_cluster(uint32_t n, uint32_t m, uint32_t o, uint32_t rpc, const double *__restrict__ A, const double *__restrict__ B,
                    const double *__restrict__ b, const double *__restrict__ C, const double *__restrict__ D,
                    const double *__restrict__ d, double *x, const double *__restrict__ power, uint32_t n_steps,
                    double *__restrict__ temps_out) {
    extern __shared__ double rom_smem[];
    cg::cluster_group cluster = cg::this_cluster();
    const uint32_t rank = cluster.block_rank();
    const uint32_t width = n + m;
    double *rows = rom_smem;                                 // [rpc][n + m]: this block's rows of [A B] then [C D]
    double *bias = rows + (size_t)rpc * width;               // [rpc]
    double *xb0 = bias + rpc, *xb1 = xb0 + n, *ps = xb1 + n; // state, next state, this step's power
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n_warps = kRomClusterThreads / 32;
    const uint32_t row0 = rank * rpc, row1 = min(n + o, row0 + rpc);
    for (uint32_t r = row0 + warp; r < row1; r += n_warps) {
        const bool out_row = r >= n;
        const uint32_t rr = out_row ? r - n : r;
        const double *mx = out_row ? C + (size_t)rr * n : A + (size_t)rr * n;
        const double *mp = out_row ? D + (size_t)rr * m : B + (size_t)rr * m;
        double *dst = rows + (size_t)(r - row0) * width;
        for (uint32_t j = lane; j < n; j += 32) dst[j] = mx[j];
        for (uint32_t j = lane; j < m; j += 32) dst[n + j] = mp[j];
        if (lane == 0) bias[r - row0] = out_row ? d[rr] : b[rr];
    }
    for (uint32_t i = tid; i < n; i += kRomClusterThreads) xb0[i] = x[i];
    double *cur = xb0, *nxt = xb1;
    cluster.sync();
    for (uint32_t k = 0; k < n_steps; ++k) {
        for (uint32_t j = tid; j < m; j += kRomClusterThreads) ps[j] = power[(size_t)k * m + j];
        __syncthreads();
        for (uint32_t r = row0 + warp; r < row1; r += n_warps) {
            const double *mr = rows + (size_t)(r - row0) * width;
            double acc = 0.0;
            for (uint32_t j = lane; j < n; j += 32) acc += mr[j] * cur[j];
            for (uint32_t j = lane; j < m; j += 32) acc += mr[n + j] * ps[j];
#pragma unroll
            for (int s = 16; s > 0; s >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, s);
            const double v = acc + bias[r - row0];
            if (r >= n) { if (lane == 0) temps_out[(size_t)k * o + (r - n)] = v; }
            else if (lane < kRomClusterBlocks) cluster.map_shared_rank(nxt, lane)[r] = v;    // every block's copy of x'
        }
        cluster.sync();                                      // x' is complete everywhere; nobody reads x any more
        double *t = cur; cur = nxt; nxt = t;
    }
    if (rank == 0)
        for (uint32_t i = tid; i < n; i += kRomClusterThreads) x[i] = cur[i];
}

// ---- the thermal step of a context on a reduced-order model: power vector, one model step, controller --------
__device__ __forceinline__ int rom_next_mode(const ThermalDev &t, int mode, long long mk) {
    if (mode == HBF_MODE_SHUTDOWN || mk >= t.shut_mk) return HBF_MODE_SHUTDOWN;
    if (mode == HBF_MODE_NORMAL) return mk >= t.stt_mk ? HBF_MODE_SEVERE : mk >= t.ltt_mk ? HBF_MODE_LIGHT : HBF_MODE_NORMAL;
    if (mode == HBF_MODE_LIGHT) return mk >= t.stt_mk ? HBF_MODE_SEVERE : mk <= t.rtt_mk ? HBF_MODE_NORMAL : HBF_MODE_LIGHT;
    return mk <= t.rtt_mk ? HBF_MODE_NORMAL : mk <= t.ltt_mk ? HBF_MODE_LIGHT : HBF_MODE_SEVERE;
}

// One launch: a warp per row of [A B; C D] (within one step the rows do not wait for one another), the row's first 256 + 128
// entries on their way before the batch before has ended; every block works out the power vector for itself, as the grid's power
// map does (one thread per region walks its dies in a fixed order); the block that is done last takes the new state over, consumes
// the window's energy, finds the hottest output of each medium and makes the controller's transition on the HBF one (quantised to
// integer mK).  Each row is summed in the order of the kernels above.  224 states, 63 inputs: as three launches (power, the cluster
// kernel, one thread for the controller) 29 us and
// three launch gaps; a window served from host memory, with its results on the way: 101 -> 66 us.
constexpr int kRomRowThreads = 128;
__global__ void __launch_bounds__(kRomRowThreads)
k_rom_window(uint32_t n, uint32_t m, uint32_t o, const double *__restrict__ A, const double *__restrict__ B, const double *__restrict__ b,
             const double *__restrict__ C, const double *__restrict__ D, const double *__restrict__ d, double *x, double *x_next, double *temps,
             uint32_t *done, const __grid_constant__ ThermalDev t, int64_t *pending, int64_t dt_ns, int has_ext, const int32_t *__restrict__ kind, DevState *state) {
    extern __shared__ double rom_smem[];                     // p [m]
    __shared__ uint32_t s_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t row = blockIdx.x * (kRomRowThreads / 32) + warp, r = row < n ? row : row - n;
    const double *mx = row < n ? A + (size_t)r * n : C + (size_t)r * n, *mp = row < n ? B + (size_t)r * m : D + (size_t)r * m;
    const bool mine = row < n + o;
    constexpr int kN = 8, kM = 4;
    double an[kN], am[kM], bias = 0.0;
    if (mine) {
#pragma unroll
        for (int k = 0; k < kN; ++k) { const uint32_t j = k * 32u + lane; an[k] = j < n ? mx[j] : 0.0; }
#pragma unroll
        for (int k = 0; k < kM; ++k) { const uint32_t j = k * 32u + lane; am[k] = j < m ? mp[j] : 0.0; }
        bias = row < n ? b[r] : d[r];
    }
    pdl_wait();
    pdl_trigger();
    for (uint32_t g = tid; g < m; g += kRomRowThreads) {
        double p = 0.0;
        for (int32_t k = t.region_die_ptr[g]; k < t.region_die_ptr[g + 1]; ++k)
            p += ((double)pending[t.region_die_list[k]] * 1e-12) / ((double)dt_ns * 1e-9);
        p += (double)t.region_idle_w[g];
        if (has_ext) p += (double)t.ext_power[g];
        rom_smem[g] = p;
    }
    double xn[kN];
#pragma unroll
    for (int k = 0; k < kN; ++k) { const uint32_t j = k * 32u + lane; xn[k] = j < n ? x[j] : 0.0; }
    __syncthreads();
    if (mine) {
        double acc = 0.0;
#pragma unroll
        for (int k = 0; k < kN; ++k) if (k * 32u + lane < n) acc += an[k] * xn[k];
        for (uint32_t j = kN * 32u + lane; j < n; j += 32) acc += mx[j] * x[j];
#pragma unroll
        for (int k = 0; k < kM; ++k) if (k * 32u + lane < m) acc += am[k] * rom_smem[k * 32u + lane];
        for (uint32_t j = kM * 32u + lane; j < m; j += 32) acc += mp[j] * rom_smem[j];
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, s);
        if (lane == 0) { if (row < n) x_next[r] = acc + bias; else temps[r] = acc + bias; }
    }
    __syncthreads();
    if (tid == 0) { __threadfence(); s_last = atomicAdd(done, 1u) == gridDim.x - 1u ? 1u : 0u; }
    __syncthreads();
    if (!s_last) return;
    // every block has read the state and the energy, and written its rows
    __threadfence();
    for (uint32_t i = tid; i < n; i += kRomRowThreads) x[i] = __ldcg(x_next + i);
    for (uint32_t e = tid; e < t.n_dies; e += kRomRowThreads) pending[e] = 0;
    if (warp != 0) return;
    double hot[3] = {-1e300, -1e300, -1e300};
    for (uint32_t i = lane; i < o; i += 32) {
        const double v = __ldcg(temps + i);
        const int slot = kind[i] == HBF_KIND_HBF ? 0 : kind[i] == HBF_KIND_HBM ? 1 : kind[i] == HBF_KIND_GPU ? 2 : -1;
#pragma unroll
        for (int k = 0; k < 3; ++k) if (slot == k && v > hot[k]) hot[k] = v;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) { const double v = __shfl_xor_sync(0xffffffffu, hot[k], s); if (v > hot[k]) hot[k] = v; }
        if (hot[k] == -1e300) hot[k] = (double)t.ambient_c;
    }
    if (lane != 0) return;
    for (int k = 0; k < 3; ++k) t.hot[k] = (float)hot[k];
    const int mode = rom_next_mode(t, state->mode, (long long)floor(hot[0] * 1000.0 + 0.5));
    state->mode = mode;
    if (mode == HBF_MODE_NORMAL) state->q_ppm = 1000000;
    else if (mode == HBF_MODE_LIGHT) state->q_ppm = t.q_light_ppm;
    *done = 0u;
}

cudaError_t launch_rom_window(uint32_t n, uint32_t m, uint32_t o, const double *A, const double *B, const double *b, const double *C, const double *D, const double *d,
                              double *x, double *x_next, double *temps, uint32_t *done, const ThermalDev &t, int64_t *pending, int64_t dt_ns, int has_ext, const int32_t *kind,
                              DevState *state, bool *plain_next, cudaStream_t st) {
    const unsigned rows = kRomRowThreads / 32;
    g_kernel_launches += 1;
    return launch_first(plain_next, k_rom_window, (n + o + rows - 1) / rows, kRomRowThreads, m * sizeof(double), st, n, m, o, A, B, b, C, D, d, x, x_next, temps, done, t,
                        pending, dt_ns, has_ext, kind, state);
}

static size_t rom_cluster_smem(uint32_t n, uint32_t m, uint32_t o, uint32_t *rpc_out) {
    const uint32_t rpc = (n + o + kRomClusterBlocks - 1) / kRomClusterBlocks;
    *rpc_out = rpc;
    return ((size_t)rpc * (n + m) + rpc + 2 * (size_t)n + m) * sizeof(double);
}

cudaError_t launch_rom_steps(uint32_t n, uint32_t m, uint32_t o, const double *A, const double *B, const double *b,
                             const double *C, const double *D, const double *d, double *x, const double *power,
                             uint32_t n_steps, double *temps_out, cudaStream_t st) {
    uint32_t rpc = 0;
    const size_t csmem = rom_cluster_smem(n, m, o, &rpc);
    if (csmem <= 200u * 1024u) {                             // the rows fit the shared memory of eight blocks
        { cudaError_t e = ensure_dyn_smem((const void *)k_rom_steps_cluster, csmem); if (e != cudaSuccess) return e; }
        k_rom_steps_cluster<<<kRomClusterBlocks, kRomClusterThreads, csmem, st>>>(n, m, o, rpc, A, B, b, C, D, d, x, power, n_steps, temps_out);
        g_kernel_launches += 1;
        return cudaGetLastError();
    }
    const size_t smem = (size_t)(2 * n + m) * sizeof(double);
    k_rom_steps<<<1, kRomThreads, smem, st>>>(n, m, o, A, B, b, C, D, d, x, power, n_steps, temps_out);
    g_kernel_launches += 1;
    return cudaGetLastError();
}

}  // namespace hbf
