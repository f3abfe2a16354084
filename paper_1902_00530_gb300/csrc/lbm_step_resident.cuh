// lbm_step_resident.cuh -- many steps of small lattices held on chip.
//
// The paper's own boxes (90 x 30, 180 x 60, App. C) and parity-sized lattices
// hold 10^3 to 5 10^4 sites.  A step of one of them is a launch that cannot
// fill the GPU, so a launch per step is bound by its latency: the launch gap
// and a few warps walking their rows one after the other.  Here one
// thread-block cluster owns a whole lattice for `nsteps` consecutive steps (none of
// them a sample step): block r of the C in the cluster holds the row band
// [r ny/C, (r+1) ny/C) of both population buffers in its shared memory, in the
// storage type, with a halo of rows and columns; HBM is read once before the first
// step and written once by the last.  A thread takes one site at a time, so a
// band of a few hundred sites is one pass of all its threads.
//
// Exchange.  A site's new populations go to the block's own buffer (and, on
// the first and last column, to the periodic halo column), and those that
// stream out of the band also straight into the halo rows of the neighbouring
// block's buffer (stores to distributed shared memory: nothing waits for
// them).  One cluster barrier per step then orders the step's stores before
// the next step's reads, and the step's reads before the next step's stores to
// the same buffer.  MIPS needs the post-stream density one row beyond the band, so
// its halo is two rows deep and the densities of rows -1 .. R are formed in
// shared memory before the update.
//
// The per-site arithmetic is that of the per-step kernels (collide_v /
// collide7, the noise and the negative correction), every operation rounded
// explicitly, and 16-bit populations are rounded at every step by the same
// Store: states are bitwise those of one launch per step.
//
// Measured (FP32, us per step, one launch per step before and this): 90 x 30
// D2Q7 MIPS 12.4 and 1.3, 64 x 64 D2Q9 MIPS 13 and about 1, 32 boxes of 180 x 60
// D2Q7 CIL 11.9 and 4.4.  What bounds it: the small boxes by the dependent chain of about
// 500 instructions of one warp per scheduler; the 32 boxes by issue (297
// instructions per site, 66 % issue active in 22 warps per SM, the rest the ramp and
// drain of four passes of sites per step).  Not faster: populations of a site
// adjacent, bulk copies or asynchronous stores between the blocks in place of the
// cluster barrier (within 2 % of this, and 1.05 to 1.9 times as long on 90 x 30),
// 512 or 1024 threads per block.
//
// Clusters do not wait on one another, so any number of lattices may be
// queued; the blocks of a cluster are co-scheduled by the hardware.
#pragma once

#include "lbm_step_q7.cuh"

namespace lbm {

__device__ __forceinline__ uint32_t map_to_rank(uint32_t smem, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, float v)
{
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void st_cluster(uint32_t addr, __half v)
{
    asm volatile("st.shared::cluster.u16 [%0], %1;" ::"r"(addr), "h"(__half_as_ushort(v)) : "memory");
}
__device__ __forceinline__ void st_cluster(uint32_t addr, __nv_bfloat16 v)
{
    asm volatile("st.shared::cluster.u16 [%0], %1;" ::"r"(addr), "h"(__bfloat16_as_ushort(v)) : "memory");
}
// All threads of every block of the cluster; orders their stores before (shared,
// distributed shared) ahead of the others' loads after.
__device__ __forceinline__ void cluster_barrier()
{
    __syncwarp();  // the aligned forms need whole warps
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// What differs between the lattices: where population i of a site is pulled
// from (column and row offsets; P: the row's parity, D2Q7 only), and the update.
template <int Q> struct ResidentLattice;
template <> struct ResidentLattice<9> {
    static __host__ __device__ constexpr int dy(int i) { return -vy(i); }
    static __device__ __forceinline__ int dx(int i, int) { return -vx(i); }
    static __device__ __forceinline__ float shift(const Shift3 &s, int i) { return s.q9(i); }
    static __device__ __forceinline__ float rho_of(const float f[9]) { return vdensity(f); }
    // the update of one site; r points at its density in rows of `pitch` values (MIPS)
    template <int MODEL, bool NOISE>
    static __device__ __forceinline__ void update(float f[9], const float *r, int pitch, int, const SiteParams &d,
                                                  uint32_t x, uint32_t y, uint32_t t, uint32_t id, const uint32_t *rk)
    {
        float u[9], gx[1] = {0.f}, gy[1] = {0.f}, rho0 = 0.f;
        if constexpr (NOISE) noise_u(x, y, t, id, rk, u);
        if constexpr (MODEL == MODEL_MIPS) {
            const float rm[3] = {r[-pitch - 1], r[-pitch], r[-pitch + 1]}, rc[3] = {r[-1], r[0], r[1]},
                        rn[3] = {r[pitch - 1], r[pitch], r[pitch + 1]};
            mips_gradients<1>(rm, rc, rn, gx, gy);
            rho0 = rc[1];
        }
        const float rho = collide_v<MODEL, float>(f, gx[0], gy[0], d, NOISE, u, MODEL == MODEL_MIPS ? &rho0 : nullptr);
        negative_correction(f, rho);
    }
};
template <> struct ResidentLattice<7> {
    static __host__ __device__ constexpr int dy(int i) { return q7_src_dy(i); }
    static __device__ __forceinline__ int dx(int i, int P)
    {
        return i == 1 ? -1 : i == 4 ? 1 : (i == 2 || i == 6) ? P - 1 : (i == 3 || i == 5) ? P : 0;
    }
    static __device__ __forceinline__ float shift(const Shift3 &s, int i) { return s.q7(i); }
    static __device__ __forceinline__ float rho_of(const float f[7]) { return density7(f); }
    template <int MODEL, bool NOISE>
    static __device__ __forceinline__ void update(float f[7], const float *r, int pitch, int P, const SiteParams &d,
                                                  uint32_t x, uint32_t y, uint32_t t, uint32_t id, const uint32_t *rk)
    {
        float u[7], gx[1] = {0.f}, gy[1] = {0.f}, rho0 = 0.f;
        if constexpr (NOISE) noise_u7(x, y, t, id, rk, u);
        if constexpr (MODEL == MODEL_MIPS) {
            // the rows above and below enter at columns x + P - 1 and x + P: the windows of
            // mips_gradients7<1, 0> taken P columns further right
            const float *a = r + P;
            const float rm[3] = {a[-pitch - 1], a[-pitch], 0.f}, rc[3] = {r[-1], r[0], r[1]},
                        rn[3] = {a[pitch - 1], a[pitch], 0.f};
            mips_gradients7<1, 0>(rm, rc, rn, gx, gy);
            rho0 = rc[1];
        }
        const float rho = collide7<MODEL>(f, gx[0], gy[0], d, NOISE, u, MODEL == MODEL_MIPS ? &rho0 : nullptr);
        negative_correction7(f, rho);
    }
};

template <int Q, int MODEL, int ST, bool NOISE>
__device__ __forceinline__ void resident_steps(const StepArgs &a, const ResidentArgs &p, const LatDesc *dp)
{
    using T = typename Store<ST>::T;
    using L = ResidentLattice<Q>;
    constexpr bool MIPS = MODEL == MODEL_MIPS;
    constexpr int H = resident_halo(MODEL);
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int rank = (int)cluster_rank(), C = p.cluster;
    const int nx = dp->nx, ny = dp->ny, pitch = dp->pitch;
    auto band = [&](int r) { return (int)((long long)ny * r / C); };
    const int y0 = band(rank), R = band(rank + 1) - y0;
    const int up = rank + 1 < C ? rank + 1 : 0, dn = rank > 0 ? rank - 1 : C - 1;
    const int Rdn = band(dn + 1) - band(dn);
    const int np = nx + 2, plane = ((ny + C - 1) / C + 2 * H) * np;  // the tallest band's plane, the same in every block
    T *const buf0 = reinterpret_cast<T *>(smem_raw);
    float *const rho_s = reinterpret_cast<float *>(smem_raw + resident_rho_offset(Q, (int)sizeof(T), plane));
    auto at = [&](int row, int col) { return (row + H) * np + col + 1; };
    const Shift3 sh = load_shift(dp);
    const SiteParams d = load_params(dp);
    const uint32_t id = (uint32_t)dp->id, t0 = *a.t_ptr + a.k;
    const size_t gplane = (size_t)ny * pitch;
    const T *const src = reinterpret_cast<const T *>(dp->f[a.src]);
    T *const dst = reinterpret_cast<T *>(dp->f[p.dst]);

    // the band and its halo, rows -H .. R-1+H and columns -1 .. nx, from HBM
    for (int e = threadIdx.x; e < (R + 2 * H) * np; e += blockDim.x) {
        const int row = e / np, col = e - row * np;
        int y = y0 + row - H, x = col - 1;
        y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
        x = x < 0 ? nx - 1 : (x >= nx ? 0 : x);
#pragma unroll
        for (int i = 0; i < Q; ++i) buf0[i * plane + e] = src[i * gplane + (size_t)y * pitch + x];
    }
    cluster_barrier();  // every block of the cluster has started and holds its band

    // the walk over sites tid, tid + blockDim.x, ... as (row, column) without divisions
    const int row_first = (int)threadIdx.x / nx, col_first = (int)threadIdx.x - row_first * nx;
    const int row_inc = (int)blockDim.x / nx, col_inc = (int)blockDim.x - row_inc * nx;
    auto next_site = [&](int &row, int &col) {
        row += row_inc;
        col += col_inc;
        if (col >= nx) {
            col -= nx;
            ++row;
        }
    };

    for (int j = 0; j < p.nsteps; ++j) {
        const T *const A = buf0 + (j & 1) * Q * plane;
        T *const B = buf0 + (1 - (j & 1)) * Q * plane;
        const uint32_t b_addr = smem_addr(B);
        const uint32_t b_up = map_to_rank(b_addr, (uint32_t)up), b_dn = map_to_rank(b_addr, (uint32_t)dn);
        const bool last = j + 1 == p.nsteps;
        if constexpr (MIPS) {
            // post-stream densities of rows -1 .. R (rho_s row k holds row k - 1), with the halo columns
            for (int row = row_first - 1, col = col_first; row < R + 1; next_site(row, col)) {
                const int P = Q == 7 ? (y0 + row) & 1 : 0, c = at(row, col);
                float f[Q];
#pragma unroll
                for (int i = 0; i < Q; ++i)
                    f[i] = Store<ST>::get(A[i * plane + c + L::dy(i) * np + L::dx(i, P)], L::shift(sh, i));
                const float r = L::rho_of(f);
                float *const o = rho_s + (row + 1) * np + col + 1;
                *o = r;
                if (col == 0) o[nx] = r;
                if (col == nx - 1) o[-nx] = r;
            }
            __syncthreads();
        }
        for (int row = row_first, col = col_first; row < R; next_site(row, col)) {
            const int y = y0 + row, P = Q == 7 ? y & 1 : 0, c = at(row, col);
            float f[Q];
#pragma unroll
            for (int i = 0; i < Q; ++i)
                f[i] = Store<ST>::get(A[i * plane + c + L::dy(i) * np + L::dx(i, P)], L::shift(sh, i));
            L::template update<MODEL, NOISE>(f, rho_s + (row + 1) * np + col + 1, np, P, d, (uint32_t)col, (uint32_t)y,
                                             t0 + (uint32_t)j, id, a.rk);
            if (last) {
                T *const o = dst + (size_t)y * pitch + col;
#pragma unroll
                for (int i = 0; i < Q; ++i) o[i * gplane] = Store<ST>::put(f[i], L::shift(sh, i));
                continue;
            }
            T v[Q];
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                v[i] = Store<ST>::put(f[i], L::shift(sh, i));
                B[i * plane + c] = v[i];
            }
            const int wrap = col == 0 ? nx : (col == nx - 1 ? -nx : 0);  // its periodic halo column
            if (wrap != 0) {
#pragma unroll
                for (int i = 0; i < Q; ++i) B[i * plane + c + wrap] = v[i];
                if (nx == 1) {
#pragma unroll
                    for (int i = 0; i < Q; ++i) B[i * plane + c - 1] = v[i];
                }
            }
            // the populations that cross into the bands above and below (with
            // MIPS also those a halo row's density needs), into their halo rows
            auto push = [&](uint32_t base, int to_row, int cross, bool same_row) {
                const int to = at(to_row, col);
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    if (L::dy(i) == cross || (MIPS && same_row && L::dy(i) == 0)) {
                        const uint32_t o = base + (uint32_t)(i * plane + to) * (uint32_t)sizeof(T);
                        st_cluster(o, v[i]);
                        if (wrap != 0) st_cluster(o + (uint32_t)(wrap * (int)sizeof(T)), v[i]);
                        if (nx == 1) st_cluster(o - (uint32_t)sizeof(T), v[i]);
                    }
                }
            };
            if (row >= R - H) push(b_up, row - R, -1, row == R - 1);
            if (row < H) push(b_dn, Rdn + row, 1, row == 0);
        }
        if (!last) cluster_barrier();
    }
}

template <int Q, int MODEL, int ST>
__global__ void __launch_bounds__(RESIDENT_THREADS, 1) step_resident_kernel(const StepArgs a, const ResidentArgs p)
{
    const LatDesc *dp = a.desc + blockIdx.x / p.cluster;
    if (dp->sigma_q > 0.f) resident_steps<Q, MODEL, ST, true>(a, p, dp);
    else resident_steps<Q, MODEL, ST, false>(a, p, dp);
}

// Launch (or, with `clusters`, only report how many clusters of this shape
// the GPU holds at once).
template <int Q, int MODEL, int ST>
static cudaError_t launch_resident_one(const StepArgs &a, const ResidentArgs &p, int *clusters, cudaStream_t stream)
{
    auto kern = step_resident_kernel<Q, MODEL, ST>;
    cudaError_t e = allow_all_smem(kern);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(p.cluster * a.nlat));
    cfg.blockDim = dim3((unsigned)p.threads);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)p.cluster;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (clusters) return cudaOccupancyMaxActiveClusters(clusters, kern, &cfg);
    return cudaLaunchKernelEx(&cfg, kern, a, p);
}

template <int Q, int ST>
static cudaError_t launch_resident_m(int model, const StepArgs &a, const ResidentArgs &p, int *clusters,
                                     cudaStream_t stream)
{
    switch (model) {
    case MODEL_PASSIVE: return launch_resident_one<Q, MODEL_PASSIVE, ST>(a, p, clusters, stream);
    case MODEL_MIPS: return launch_resident_one<Q, MODEL_MIPS, ST>(a, p, clusters, stream);
    case MODEL_CIL: return launch_resident_one<Q, MODEL_CIL, ST>(a, p, clusters, stream);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace lbm

#define LBM_INSTANTIATE_RESIDENT(ST, SUFFIX)                                                                 \
    namespace lbm {                                                                                          \
    cudaError_t launch_resident_##SUFFIX(int q, int model, const StepArgs &a, const ResidentArgs &p,           \
                                         int *clusters, cudaStream_t stream)                                 \
    {                                                                                                        \
        return q == 7 ? launch_resident_m<7, ST>(model, a, p, clusters, stream)                              \
                      : launch_resident_m<9, ST>(model, a, p, clusters, stream);                             \
    }                                                                                                        \
    }
