// lbm_aux.cu -- initialisation, moment output, state exchange and the
// observable finaliser.  Small kernels around the fused step.
#include <type_traits>

#include "lbm_internal.h"
#include "lbm_step_staged.cuh"  // the bounded barrier wait of the staged kernels

namespace lbm {

// ---------------------------------------------------------------------------
// Initial state (App. C.2): per site two Philox words give rho and the
// direction of u; populations are f^SS(rho, u) evaluated in FP64 and rounded
// once to the storage type.  Counter purpose 1, t = 0, call 0.
// ---------------------------------------------------------------------------
struct InitSpecDev {
    double rho_mean, rho_amp, u_amp, ux0, uy0, A, B;
    int u_kind, pad;
};

template <int ST>
__global__ void init_kernel(const LatDesc *desc, const InitSpecDev *specs, int dst,
                            uint32_t key0, uint32_t key1)
{
    using T = typename Store<ST>::T;
    const LatDesc d = desc[blockIdx.y];
    const Shift3 shf = load_shift(&d);
    const InitSpecDev sp = specs[blockIdx.y];
    const long long n = (long long)d.nx * d.ny;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n;
         c += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(c % d.nx), y = (int)(c / d.nx);
        const uint4 w = philox4x32_10(
            make_uint4((uint32_t)x, (uint32_t)y, 0u, ((uint32_t)d.id & 0xFFFFFFu) | (1u << 24)), key0, key1);
        const double U0v = ((double)(w.x >> 8) + 0.5) * (1.0 / 16777216.0);
        const double U1v = ((double)(w.y >> 8) + 0.5) * (1.0 / 16777216.0);
        const double U2v = ((double)(w.z >> 8) + 0.5) * (1.0 / 16777216.0);
        const double rho = sp.rho_mean * (1.0 + sp.rho_amp * (2.0 * U0v - 1.0));
        double ux, uy;
        if (sp.u_kind == 0) {
            ux = sp.ux0 + sp.u_amp * (2.0 * U1v - 1.0);
            uy = sp.uy0 + sp.u_amp * (2.0 * U2v - 1.0);
        } else {
            double sn, cs;
            sincospi(2.0 * U1v, &sn, &cs);
            double mag = sp.u_amp;
            if (sp.u_kind == 2) {
                const double ar2 = sp.A * rho * rho;
                mag = sp.B >= ar2 ? sp.B - ar2 : 0.0;
                ux = mag * cs;
                uy = mag * sn;
            } else {
                ux = sp.ux0 + mag * cs;
                uy = sp.uy0 + mag * sn;
            }
        }
        const double usq = ux * ux + uy * uy;
        T *base = reinterpret_cast<T *>(d.f[dst]);
        const size_t plane = (size_t)d.ny * d.pitch;
        auto put = [&](int i, double feq, float shift) {
            T v;
            if constexpr (ST == ST_F32) v = (float)feq;
            else if constexpr (ST == ST_F16) v = __double2half(feq - (double)shift);
            else v = __double2bfloat16(feq - (double)shift);
            base[i * plane + (size_t)y * d.pitch + x] = v;
        };
        if (d.q == 7) {
            // Eq. (fssD2Q7): w_i rho [1 + 4 e.u + 8 (e.u)^2 - 2 u^2], e_i at (i-1) pi/3
            const double hs3 = 0.86602540378443864676;
            const double ex[7] = {0.0, 1.0, 0.5, -0.5, -1.0, -0.5, 0.5};
            const double ey[7] = {0.0, 0.0, hs3, hs3, 0.0, -hs3, -hs3};
#pragma unroll
            for (int i = 0; i < 7; ++i) {
                const double eu = ex[i] * ux + ey[i] * uy;
                put(i, wq7_d(i) * rho * (1.0 + 4.0 * eu + 8.0 * eu * eu - 2.0 * usq), shf.q7(i));
            }
        } else {
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const double eu = vx(i) * ux + vy(i) * uy;
                put(i, wq_d(i) * rho * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * usq), shf.q9(i));
            }
        }
    }
}

// ---------------------------------------------------------------------------
// State exchange.  These kernels only move bytes, so they are laid out for that:
// a thread takes VEC adjacent sites of a row (16 bytes of storage where nx and
// the caller's pointer allow it), a block covers whole row segments of several rows
// (threadIdx.y), and each thread holds the loads of EXCHANGE_ROWS rows in
// flight.  No index is divided: a site's row and plane come from the grid.  (With
// one element per thread and 64-bit divisions for its plane, row and column,
// 4096^2 BF16 took 620 us out, 736 us in, 603 us for a density step and 161 us
// for the moments; the bytes take 134, 134, 89 and 74 us.  FP32 went through
// cudaMemcpy2D: 608 us against 178.  Whole calls of these kernels now: BF16 181 us
// out, 155 in, 115 for a density step, 106 for the moments; FP32 186 out, 201 in.)
// ---------------------------------------------------------------------------
constexpr int EXCHANGE_ROWS = 4;

// f(row) for this thread's rows of a plane, EXCHANGE_ROWS apart by the grid's height
struct RowWalk {
    int x, y0, dy;
    __device__ RowWalk(int vec)
        : x((int)(blockIdx.x * blockDim.x + threadIdx.x) * vec), y0((int)(blockIdx.y * blockDim.y + threadIdx.y)),
          dy((int)(gridDim.y * blockDim.y))
    {
    }
};

// VEC dense FP32 values (16-byte aligned where VEC >= 4)
template <int VEC> __device__ __forceinline__ void put_dense(float *p, const float v[VEC])
{
    if constexpr (VEC % 4 == 0) {
#pragma unroll
        for (int k = 0; k < VEC / 4; ++k)
            reinterpret_cast<float4 *>(p)[k] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
    } else {
#pragma unroll
        for (int k = 0; k < VEC; ++k) p[k] = v[k];
    }
}
template <int VEC> __device__ __forceinline__ void get_dense(const float *p, float v[VEC])
{
    if constexpr (VEC % 4 == 0) {
#pragma unroll
        for (int k = 0; k < VEC / 4; ++k) {
            const float4 w = __ldg(reinterpret_cast<const float4 *>(p) + k);
            v[4 * k] = w.x;
            v[4 * k + 1] = w.y;
            v[4 * k + 2] = w.z;
            v[4 * k + 3] = w.w;
        }
    } else {
#pragma unroll
        for (int k = 0; k < VEC; ++k) v[k] = __ldg(p + k);
    }
}

// Stored state -> dense FP32 moments (rho, ux, uy) [ny][nx].
template <int ST, int VEC, int Q>
__global__ void __launch_bounds__(256) moments_kernel(const LatDesc *desc, int lat, int src, float *rho, float *ux,
                                                      float *uy)
{
    using T = typename Store<ST>::T;
    const LatDesc *d = desc + lat;
    const int nx = d->nx, ny = d->ny, pitch = d->pitch;
    const Shift3 shf = load_shift(d);
    const T *base = reinterpret_cast<const T *>(d->f[src]);
    const size_t plane = (size_t)ny * pitch;
    const RowWalk w(VEC);
    if (w.x >= nx) return;
    for (int y = w.y0; y < ny; y += w.dy) {
        RawVec<ST, VEC> raw[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) raw[i] = load_raw<ST, VEC>(base + i * plane + (size_t)y * pitch + w.x);
        float f[Q][VEC], r[VEC], vx_[VEC], vy_[VEC];
#pragma unroll
        for (int i = 0; i < Q; ++i) expand_raw<ST, VEC>(raw[i], shf.of(Q, i), f[i]);
#pragma unroll
        for (int j = 0; j < VEC; ++j) {
            float jx, jy;
            if constexpr (Q == 7) {
                r[j] = ((f[0][j] + f[1][j]) + (f[2][j] + f[3][j])) + ((f[4][j] + f[5][j]) + f[6][j]);
                jx = (f[1][j] - f[4][j]) + 0.5f * ((f[2][j] + f[6][j]) - (f[3][j] + f[5][j]));
                jy = 0.86602540378443865f * ((f[2][j] + f[3][j]) - (f[5][j] + f[6][j]));
            } else {
                r[j] = ((f[0][j] + f[1][j]) + (f[2][j] + f[3][j])) + ((f[4][j] + f[5][j]) + (f[6][j] + f[7][j])) +
                       f[8][j];
                jx = (f[1][j] + f[5][j] + f[8][j]) - (f[3][j] + f[6][j] + f[7][j]);
                jy = (f[2][j] + f[5][j] + f[6][j]) - (f[4][j] + f[7][j] + f[8][j]);
            }
            vx_[j] = r[j] > 0.f ? jx / r[j] : 0.f;
            vy_[j] = r[j] > 0.f ? jy / r[j] : 0.f;
        }
        const size_t o = (size_t)y * nx + w.x;
        put_dense<VEC>(rho + o, r);
        put_dense<VEC>(ux + o, vx_);
        put_dense<VEC>(uy + o, vy_);
    }
}

// Stored populations i0 .. i0 + gridDim.z - 1 -> dense FP32 [gridDim.z][ny][nx].
template <int ST, int VEC>
__global__ void __launch_bounds__(256) export_kernel(const LatDesc *desc, int lat, int src, int i0, float *out)
{
    using T = typename Store<ST>::T;
    const LatDesc *d = desc + lat;
    const int nx = d->nx, ny = d->ny, pitch = d->pitch, i = i0 + (int)blockIdx.z;
    const float shift = load_shift(d).of(d->q, i);
    const RowWalk w(VEC);
    if (w.x >= nx) return;
    const T *base = reinterpret_cast<const T *>(d->f[src]) + (size_t)i * ny * pitch + w.x;
    out += (size_t)blockIdx.z * ny * nx + w.x;
    for (int y = w.y0; y < ny; y += EXCHANGE_ROWS * w.dy) {
        RawVec<ST, VEC> raw[EXCHANGE_ROWS];
#pragma unroll
        for (int k = 0; k < EXCHANGE_ROWS; ++k)
            if (y + k * w.dy < ny) raw[k] = load_raw<ST, VEC>(base + (size_t)(y + k * w.dy) * pitch);
#pragma unroll
        for (int k = 0; k < EXCHANGE_ROWS; ++k)
            if (y + k * w.dy < ny) {
                float v[VEC];
                expand_raw<ST, VEC>(raw[k], shift, v);
                put_dense<VEC>(out + (size_t)(y + k * w.dy) * nx, v);
            }
    }
}

// ... and back.
template <int ST, int VEC>
__global__ void __launch_bounds__(256) import_kernel(const LatDesc *desc, int lat, int dst, int i0, const float *in)
{
    using T = typename Store<ST>::T;
    const LatDesc *d = desc + lat;
    const int nx = d->nx, ny = d->ny, pitch = d->pitch, i = i0 + (int)blockIdx.z;
    const float shift = load_shift(d).of(d->q, i);
    const RowWalk w(VEC);
    if (w.x >= nx) return;
    T *base = reinterpret_cast<T *>(d->f[dst]) + (size_t)i * ny * pitch + w.x;
    in += (size_t)blockIdx.z * ny * nx + w.x;
    for (int y = w.y0; y < ny; y += EXCHANGE_ROWS * w.dy) {
        float v[EXCHANGE_ROWS][VEC];
#pragma unroll
        for (int k = 0; k < EXCHANGE_ROWS; ++k)
            if (y + k * w.dy < ny) get_dense<VEC>(in + (size_t)(y + k * w.dy) * nx, v[k]);
#pragma unroll
        for (int k = 0; k < EXCHANGE_ROWS; ++k)
            if (y + k * w.dy < ny) store_vec<ST, VEC>(base + (size_t)(y + k * w.dy) * pitch, shift, v[k]);
    }
}

// Add a constant to every population of one lattice (App. C.2 density step).
template <int ST, int VEC>
__global__ void __launch_bounds__(256) add_density_kernel(const LatDesc *desc, int lat, int buf, float per_population)
{
    using T = typename Store<ST>::T;
    const LatDesc *d = desc + lat;
    const int nx = d->nx, ny = d->ny, pitch = d->pitch, i = (int)blockIdx.z;
    const float shift = load_shift(d).of(d->q, i);
    const RowWalk w(VEC);
    if (w.x >= nx) return;
    T *base = reinterpret_cast<T *>(d->f[buf]) + (size_t)i * ny * pitch + w.x;
    for (int y = w.y0; y < ny; y += EXCHANGE_ROWS * w.dy) {
        float v[EXCHANGE_ROWS][VEC];
#pragma unroll
        for (int k = 0; k < EXCHANGE_ROWS; ++k)
            if (y + k * w.dy < ny) load_vec_plain<ST, VEC>(base + (size_t)(y + k * w.dy) * pitch, shift, v[k]);
#pragma unroll
        for (int k = 0; k < EXCHANGE_ROWS; ++k)
            if (y + k * w.dy < ny) {
#pragma unroll
                for (int j = 0; j < VEC; ++j) v[k][j] = __fadd_rn(v[k][j], per_population);
                store_vec<ST, VEC>(base + (size_t)(y + k * w.dy) * pitch, shift, v[k]);
            }
    }
}

// ---------------------------------------------------------------------------
// Observable finaliser.  Grid (nchunk, nlat): block (c, l) sums, in a fixed
// order, chunk c of lattice l's column partials (over strip rows), row
// partials (over strip columns) and per-strip scalars, and writes nine chunk
// sums.  The last block to arrive for a lattice combines the chunks and
// writes one record: deterministic whatever the arrival order.
//
// Bound by latency: dependent loads and FP64 chains.  So a chunk is 32 columns (one
// per lane) whose strip rows are split over the block's warps (8192^2 in 8-row
// strips: 128 loads a lane, not 1024 in a row), the sums of each kind are
// reduced by their own warps at the same time (an FP64 addition takes a
// warp's scheduler 64 cycles), and the record's divisions and square roots are
// formed by eight lanes at once.  (ncu, cold caches: 4096^2 44 -> 19 us; 32 lattices
// of 180 x 60 20.5 -> 15.6 us.)
//
// An on-demand call (to_ring 0) wants one lattice's record on the host, and
// the error word after every lattice's sums: the last lattice to finish writes
// both to `host`, pinned memory the kernel reaches itself, which saves the
// two copies that would follow.
// ---------------------------------------------------------------------------
constexpr int FIN_THREADS = 256, FIN_WARPS = FIN_THREADS / 32;

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    return v;
}

__global__ void __launch_bounds__(FIN_THREADS) finalize_kernel(const LatDesc *desc, int nlat,
                                                               const uint32_t *t_ptr, uint32_t k,
                                                               int to_ring, unsigned *err, int want, double *host)
{
    __shared__ double part[FIN_WARPS][32], S[9];
    __shared__ bool am_last;
    wait_for_previous();
    allow_dependents();
    const int l = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (l >= nlat) return;
    const LatDesc *dp = desc + l;
    const int c = blockIdx.x, nchunk = dp->nchunk;
    if (c >= nchunk) return;
    const int nx = dp->nx, ny = dp->ny, nsx = dp->nsx, nsy = dp->nsy, nstrip = nsx * nsy;
    // this chunk's share of n items
    auto first = [&](int n, int cc) { return (int)((long long)n * cc / nchunk); };
    double v[2] = {0, 0};  // warp 0: sums over columns and their squares; warp 1: the same over rows
    // line sums: partial p of line i at base[p * n + i], np partials each
    auto lines = [&](const double *base, int n, int np, int owner) {
        for (int i0 = first(n, c); i0 < first(n, c + 1); i0 += 32) {
            const int i = i0 + lane;
            const bool in = i < first(n, c + 1);
            double s = 0.0;
            if (in) {
#pragma unroll 4
                for (int p = warp; p < np; p += FIN_WARPS) s += base[(size_t)p * n + i];
            }
            part[warp][lane] = s;
            __syncthreads();
            if (warp == owner && in) {
                s = 0.0;
#pragma unroll
                for (int w = 0; w < FIN_WARPS; ++w) s += part[w][lane];
                v[0] += s;
                v[1] += s * s;
            }
            __syncthreads();
        }
    };
    lines(dp->colp, nx, nsy, 0);
    lines(dp->rowp, ny, nsx, 1);
    double *const out_c = dp->finp + (size_t)c * 9;
    if (warp < 2) {
        const double a = warp_sum(v[0]), b = warp_sum(v[1]);
        if (lane == 0) {
            out_c[5 + 2 * warp] = a;
            out_c[6 + 2 * warp] = b;
        }
    } else if (warp < 7) {
        const int q = warp - 2, s1 = first(nstrip, c + 1);
        double s = 0.0;
        for (int i = first(nstrip, c) + lane; i < s1; i += 32) s += dp->scal[(size_t)i * 5 + q];
        s = warp_sum(s);
        if (lane == 0) out_c[q] = s;
    }
    if (lane == 0) __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned ticket = atomicAdd(&dp->counters[1], 1u);
        am_last = (ticket == (unsigned)nchunk - 1);
    }
    __syncthreads();
    if (!am_last) return;
    __threadfence();
    for (int q = warp; q < 9; q += FIN_WARPS) {
        double s = 0.0;
        for (int cc = lane; cc < nchunk; cc += 32) s += ((volatile double *)dp->finp)[(size_t)cc * 9 + q];
        s = warp_sum(s);
        if (lane == 0) S[q] = s;
    }
    __syncthreads();
    if (warp != 0) return;
    // lane k: quotient k = a / b, then the square roots of lanes 3 and 4
    const double dx = (double)nx, dy = (double)ny, n = dx * dy, mass = S[0];
    double a = mass, b = n;                          // 0: mean
    if (lane == 1) a = sqrt(S[1] * S[1] + S[2] * S[2]), b = mass;  // phi
    if (lane == 2) a = S[4], b = mass;               // sum |j| / mass
    if (lane == 3) a = S[6], b = dy * dy * dx;       // <rho_y^2>: column means rho_y(x) = colsum / ny
    if (lane == 4) a = S[8], b = dx * dx * dy;       // <rho_x^2>
    if (lane == 5) a = S[3], b = n;                  // <rho^2>
    if (lane == 6) a = S[5], b = dy * dx;            // mean of rho_y
    if (lane == 7) a = S[7], b = dx * dy;            // mean of rho_x
    const double quo = a / b;
    const double mcol = __shfl_sync(FULL, quo, 6), mrow = __shfl_sync(FULL, quo, 7), mean = __shfl_sync(FULL, quo, 0);
    const double m = lane == 3 ? mcol : (lane == 4 ? mrow : mean);
    const double var = quo - m * m;  // lanes 3, 4, 5: population variances over x, over y, over sites
    const double dev = sqrt(fmax(var, 0.0));
    const double zeta = (double)dp->B - quo;  // lane 2
    const bool finite = lane == 0 ? isfinite(mass) : lane == 1 ? isfinite(quo) : lane == 2 ? isfinite(zeta)
                        : (lane >= 3 && lane <= 5) ? isfinite(var) : true;
    const bool all_finite = __all_sync(FULL, finite);
    double rec = 0.0;
    if (lane == 0) rec = __longlong_as_double((long long)(uint32_t)(*t_ptr + k + (to_ring ? 1u : 0u)));
    const double r1 = mass, r2 = __shfl_sync(FULL, quo, 1), r3 = __shfl_sync(FULL, dev, 3),
                 r4 = __shfl_sync(FULL, dev, 4), r5 = __shfl_sync(FULL, fmax(var, 0.0), 5),
                 r6 = __shfl_sync(FULL, zeta, 2);
    if (lane == 1) rec = r1;
    if (lane == 2) rec = r2;
    if (lane == 3) rec = r3;
    if (lane == 4) rec = r4;
    if (lane == 5) rec = r5;
    if (lane == 6) rec = r6;
    unsigned idx = 0;
    if (lane == 0) {
        if (!all_finite) atomicOr(err, (unsigned)DEVERR_NUMERIC);
        dp->counters[1] = 0;
        if (to_ring) {
            idx = dp->counters[0];
            dp->counters[0] = idx + 1;
        }
    }
    idx = __shfl_sync(FULL, idx, 0);
    double *out = to_ring ? dp->ring + (size_t)(idx % (unsigned)dp->ring_cap) * 8 : dp->now;
    if (lane < 8) out[lane] = rec;
    if (to_ring) return;
    unsigned *const done = err + 1;  // lattices finished in this call
    __threadfence();
    __syncwarp();
    unsigned ticket = 0;
    if (lane == 0) ticket = atomicAdd(done, 1u);
    if (__shfl_sync(FULL, ticket, 0) != (unsigned)nlat - 1) return;
    __threadfence();
    if (lane < 8) host[lane] = ((volatile double *)desc[want].now)[lane];
    if (lane == 8) host[8] = (double)*(volatile unsigned *)err;
    if (lane == 0) *done = 0;
    __threadfence_system();
}

__global__ void advance_time_kernel(uint32_t *t_ptr, uint32_t n)
{
    wait_for_previous();
    *t_ptr += n;
}

__global__ void set_time_kernel(uint32_t *t_ptr, uint32_t t) { *t_ptr = t; }

// The failure path of the staged kernels' waits, exercised on purpose: one
// warp waits, with the same bounded wait, on a barrier phase that nothing
// completes; the wait gives up after its limit (about 1 s) and the warp raises
// the timeout flag, as a step kernel does when a staged row never arrives.
__global__ void wait_timeout_kernel(unsigned *err)
{
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        mbar_init_fence();
    }
    __syncwarp();
    if (!stage_wait(&bar, 0u) && threadIdx.x == 0) atomicOr(err, (unsigned)DEVERR_TIMEOUT);
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
static int grid_for(long long n, int threads)
{
    long long b = (n + threads - 1) / threads;
    if (b > 152LL * 64) b = 152LL * 64;
    return (int)(b < 1 ? 1 : b);
}

cudaError_t launch_init(int storage, const LatDesc *desc, const void *specs, int nlat, long long max_cells,
                        int dst, uint64_t seed, cudaStream_t s)
{
    dim3 g(grid_for(max_cells, 256), nlat);
    const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    const InitSpecDev *sp = reinterpret_cast<const InitSpecDev *>(specs);
    if (storage == ST_F32) init_kernel<ST_F32><<<g, 256, 0, s>>>(desc, sp, dst, k0, k1);
    else if (storage == ST_F16) init_kernel<ST_F16><<<g, 256, 0, s>>>(desc, sp, dst, k0, k1);
    else init_kernel<ST_BF16><<<g, 256, 0, s>>>(desc, sp, dst, k0, k1);
    return cudaGetLastError();
}

size_t init_spec_bytes() { return sizeof(InitSpecDev); }

void pack_init_spec(void *dst, double rho_mean, double rho_amp, int u_kind, double u_amp, double ux0,
                    double uy0, double A, double B)
{
    InitSpecDev s;
    s.rho_mean = rho_mean;
    s.rho_amp = rho_amp;
    s.u_amp = u_amp;
    s.ux0 = ux0;
    s.uy0 = uy0;
    s.A = A;
    s.B = B;
    s.u_kind = u_kind;
    s.pad = 0;
    *reinterpret_cast<InitSpecDev *>(dst) = s;
}

// Sites per thread of an exchange kernel: 16 bytes of storage (or, in 16-bit
// storage, 8) where nx is a multiple of them and the caller's dense arrays
// are 16-byte aligned; else one.
static int exchange_vec(int storage, int nx, const void *dense)
{
    if (reinterpret_cast<uintptr_t>(dense) & 15) return 1;
    if (storage != ST_F32 && nx % 8 == 0) return 8;
    return nx % 4 == 0 ? 4 : 1;
}

// Blocks of 256 threads, as wide as the row needs (a power of two from a warp
// on) and the rest in rows; enough of them for every SM, each thread walking
// several rows.
static void exchange_grid(int nx, int ny, int planes, int vec, int rows_per_pass, dim3 &grid, dim3 &block)
{
    const int nv = nx / vec;
    unsigned bx = 32;
    while (bx < 256 && bx < (unsigned)nv) bx *= 2;
    block = dim3(bx, 256 / bx);
    grid.x = (unsigned)((nv + bx - 1) / bx);
    grid.z = (unsigned)planes;
    const long long want = (ny + (long long)block.y * rows_per_pass - 1) / ((long long)block.y * rows_per_pass);
    grid.y = (unsigned)(want > 65535 ? 65535 : want);
}

// Run `launch` with the storage type and vector width as template arguments.
template <int ST, typename F> static void with_vec(int vec, F launch)
{
    if (vec == 8) {
        if constexpr (ST != ST_F32) launch(std::integral_constant<int, ST>{}, std::integral_constant<int, 8>{});
    } else if (vec == 4) {
        launch(std::integral_constant<int, ST>{}, std::integral_constant<int, 4>{});
    } else {
        launch(std::integral_constant<int, ST>{}, std::integral_constant<int, 1>{});
    }
}
template <typename F> static cudaError_t with_storage(int storage, int vec, F launch)
{
    if (storage == ST_F32) with_vec<ST_F32>(vec, launch);
    else if (storage == ST_F16) with_vec<ST_F16>(vec, launch);
    else with_vec<ST_BF16>(vec, launch);
    return cudaGetLastError();
}

cudaError_t launch_moments(int storage, const LatDesc *desc, int lat, int q, int nx, int ny, int src, float *rho,
                           float *ux, float *uy, cudaStream_t s)
{
    const uintptr_t all = reinterpret_cast<uintptr_t>(rho) | reinterpret_cast<uintptr_t>(ux) | reinterpret_cast<uintptr_t>(uy);
    int vec = exchange_vec(storage, nx, reinterpret_cast<const void *>(all));
    if (vec == 8) vec = 4;  // eight sites of nine populations would spill
    dim3 g, b;
    exchange_grid(nx, ny, 1, vec, 1, g, b);
    return with_storage(storage, vec, [&](auto st, auto v) {
        constexpr int ST = decltype(st)::value, VEC = decltype(v)::value > 4 ? 4 : decltype(v)::value;
        if (q == 7) moments_kernel<ST, VEC, 7><<<g, b, 0, s>>>(desc, lat, src, rho, ux, uy);
        else moments_kernel<ST, VEC, 9><<<g, b, 0, s>>>(desc, lat, src, rho, ux, uy);
    });
}

cudaError_t launch_export(int storage, const LatDesc *desc, int lat, int i0, int planes, int nx, int ny, int src,
                          float *out, cudaStream_t s)
{
    const int vec = exchange_vec(storage, nx, out);
    dim3 g, b;
    exchange_grid(nx, ny, planes, vec, EXCHANGE_ROWS, g, b);
    return with_storage(storage, vec, [&](auto st, auto v) {
        export_kernel<decltype(st)::value, decltype(v)::value><<<g, b, 0, s>>>(desc, lat, src, i0, out);
    });
}

cudaError_t launch_import(int storage, const LatDesc *desc, int lat, int i0, int planes, int nx, int ny, int dst,
                          const float *in, cudaStream_t s)
{
    const int vec = exchange_vec(storage, nx, in);
    dim3 g, b;
    exchange_grid(nx, ny, planes, vec, EXCHANGE_ROWS, g, b);
    return with_storage(storage, vec, [&](auto st, auto v) {
        import_kernel<decltype(st)::value, decltype(v)::value><<<g, b, 0, s>>>(desc, lat, dst, i0, in);
    });
}

cudaError_t launch_add_density(int storage, const LatDesc *desc, int lat, int q, int nx, int ny, int buf, float per_pop,
                               cudaStream_t s)
{
    const int vec = exchange_vec(storage, nx, nullptr);
    dim3 g, b;
    exchange_grid(nx, ny, q, vec, EXCHANGE_ROWS, g, b);
    return with_storage(storage, vec, [&](auto st, auto v) {
        add_density_kernel<decltype(st)::value, decltype(v)::value><<<g, b, 0, s>>>(desc, lat, buf, per_pop);
    });
}

cudaError_t launch_finalize(const LatDesc *desc, int nlat, int max_chunk, const uint32_t *t_ptr, uint32_t k,
                            int to_ring, unsigned *err, int want, double *host, cudaStream_t s)
{
    dim3 g(max_chunk, nlat);
    return launch_dependent(finalize_kernel, g, dim3(FIN_THREADS), 0, s, desc, nlat, t_ptr, k, to_ring, err, want, host);
}

cudaError_t launch_advance_time(uint32_t *t_ptr, uint32_t n, cudaStream_t s)
{
    return launch_dependent(advance_time_kernel, dim3(1), dim3(1), 0, s, t_ptr, n);
}

cudaError_t launch_wait_timeout(unsigned *err, cudaStream_t s)
{
    wait_timeout_kernel<<<1, 32, 0, s>>>(err);
    return cudaGetLastError();
}

cudaError_t launch_set_time(uint32_t *t_ptr, uint32_t t, cudaStream_t s)
{
    set_time_kernel<<<1, 1, 0, s>>>(t_ptr, t);
    return cudaGetLastError();
}

}  // namespace lbm
