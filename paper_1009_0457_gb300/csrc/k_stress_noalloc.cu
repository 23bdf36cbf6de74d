// Allocation-free stress pass: hmc_stress_noalloc (declared in include/hmc.h).
//
// Some callers cannot allocate device memory at the point where they need the
// stress field: code running inside another framework's memory pool or a
// fixed-budget arena, or code that may not call cudaMalloc/cudaFree at that
// point because those calls synchronise the device.  For them this entry point
// computes the same quantities as hmc_compute_stress + hmc_get_stress
// (FP32 stress of every point, FP64 mean stress and elastic energy) from
// caller-owned device buffers, and keeps its only scratch -- the per-CTA
// partial sums of the fixed-order reduction -- in a file-scope device array.
//
// Limits and sharing: the array holds NOALLOC_MAX_CTAS partial-sum slots of
// 8 doubles (512 KiB, resident on every GPU that loads the library until the
// process exits); one CTA covers 256 cells of 2x2x2 points, so grids of up to
// 2,097,152 cells (16,777,216 points) are served -- 256^3 is the largest cube
// accepted -- and larger ones are rejected.  Every call uses the same array and
// leaves its partial sums there; each call overwrites every slot it reads, so
// nothing has to start at zero, but two calls whose work overlaps on the GPU
// (different streams, no ordering) race on the array.  The array's device
// address is looked up once per device and kept for the life of the process,
// which assumes the device's primary context and no cudaDeviceReset after the
// first call.
#include <cooperative_groups.h>

#include <cmath>
#include <mutex>
#include <string>

#include "hmc.h"
#include "hmc_device.cuh"

namespace hmc {
void set_unbound_error(const std::string &msg);  // message for hmc_last_error(NULL)
}

namespace {

constexpr int NOALLOC_MAX_CTAS = 8192;
constexpr int NOALLOC_THREADS = 256;   // cells of a CTA (and its threads, over CELLS)
constexpr int NOALLOC_SPREAD = 304;    // CTAs (two per SM) from which a thread takes four cells

static __device__ __align__(256) double g_noalloc_partials[NOALLOC_MAX_CTAS * 8];

struct NoallocArgs {
    const uint16_t *spins;  // natural order
    const float *u;         // nnodes x 3
    const float *ctab;      // Q x 36, full Voigt C'(q), row-major
    float *sigma;           // N x 6, natural order
    double *partials;       // device address of g_noalloc_partials
    double *mean;           // 6
    double *energy;         // 1
    float eb[6];
    int nx, ny, nz, nbx, nby, nbz;
    long long nblk, n_sites;
};

// Knuth's TwoSum: hi + x = s + its error exactly, whatever the signs and sizes (Kahan's sum, three additions
// shorter, loses bits where terms cancel: 1e-9 of them instead of 1e-15).
__device__ __forceinline__ void two_sum_add(float &hi, float &lo, float x) {
    const float s = hi + x;
    const float bb = s - hi;
    lo += (hi - (s - bb)) + (x - bb);
    hi = s;
}

// a point's full 6x6 stiffness, 16-byte loads where the table allows them
template <bool VEC>
__device__ __forceinline__ void load_c36(const float *p, float (&c)[36]) {
    if constexpr (VEC) {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const float4 t = __ldg(reinterpret_cast<const float4 *>(p) + i);
            c[4 * i] = t.x;
            c[4 * i + 1] = t.y;
            c[4 * i + 2] = t.z;
            c[4 * i + 3] = t.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < 36; ++i) c[i] = __ldg(p + i);
    }
}

// One thread per 2x2x2 cell: strain of its eight points from the trilinear
// nodal field, Hooke's law with the point's rotated stiffness, natural-order
// stress out, and per-CTA FP64 partial sums of sigma and 1/2 sigma.eps.
//
// The 24 bytes a point writes are most of the traffic (403 of 461 MB at 256^3).
// Written by the thread that formed them they were 4-byte stores 48 bytes apart;
// a lane's two x-neighbours are 48 contiguous bytes instead, which a warp passes
// through shared memory (16-byte units 3 lane + j: free of bank conflicts) and
// stores in order of address, 16 bytes a lane.  The stiffness row is kept in
// registers while consecutive points share an orientation.  VEC: every pointer
// allows the wide accesses (4 bytes for the spins, 16 for ctab and sigma); the
// other form takes 4-byte loads and stores in the same order.
//
// What bounds it: the L1 data pipe (76 % of its wavefronts), most of it the divergent
// reloads of the 144-byte rows in cells that a grain boundary cuts.  Measured at 256^3, 419
// voxels a grain: 440 us a call before, 266 us with the coalesced stores, 165 us with four
// cells a thread and the Gray-code order (floor of its bytes: 68 us).
//
// CELLS: blocks of a CTA's 256 that a thread takes in turn.  Four on large grids: the
// warp's TwoSum reduction (about 350 of 1900 instructions when every cell paid it) is then paid
// once for four cells.  One on grids of fewer CTAs than NOALLOC_SPREAD, where the chain of four cells would
// be longer than the whole pass.
template <bool VEC, int CELLS>
__global__ void __launch_bounds__(NOALLOC_THREADS / CELLS, 2 * CELLS) k_stress_noalloc(NoallocArgs a) {
    constexpr int THREADS = NOALLOC_THREADS / CELLS;
    __shared__ double red[THREADS / 32][7];
    __shared__ float4 stage[THREADS / 32][96];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    float hi[7], lo[7];
#pragma unroll
    for (int i = 0; i < 7; ++i) hi[i] = lo[i] = 0.f;
    // a cell's first point (the caller's arrays), corner displacements and spins (two x neighbours a word)
    auto load_cell = [&](unsigned blk, unsigned &p0, float (&u)[8][3], unsigned (&sp)[4]) {
        const unsigned rr = blk / (unsigned)a.nbx;
        const int bx = (int)(blk - rr * (unsigned)a.nbx), by = (int)(rr % (unsigned)a.nby), bz = (int)(rr / (unsigned)a.nby);
        p0 = 2u * bx + (unsigned)a.nx * (2u * by + (unsigned)a.ny * 2u * bz);
#pragma unroll
        for (int K = 0; K < 2; ++K)
#pragma unroll
            for (int J = 0; J < 2; ++J)
#pragma unroll
                for (int I = 0; I < 2; ++I) {
                    const int gi = bx + I == a.nbx ? 0 : bx + I;
                    const int gj = by + J == a.nby ? 0 : by + J;
                    const int gk = bz + K == a.nbz ? 0 : bz + K;
                    const unsigned n = 3u * (gi + (unsigned)a.nbx * (gj + (unsigned)a.nby * gk));
#pragma unroll
                    for (int d = 0; d < 3; ++d) u[hmc::corner(I, J, K)][d] = __ldg(a.u + n + d);
                }
#pragma unroll
        for (int row = 0; row < 4; ++row) {
            const unsigned p = p0 + (unsigned)a.nx * ((row & 1) + (unsigned)a.ny * (row >> 1));
            if constexpr (VEC)
                sp[row] = __ldg(reinterpret_cast<const unsigned *>(a.spins + p));
            else
                sp[row] = __ldg(a.spins + p) | (unsigned)__ldg(a.spins + p + 1) << 16;
        }
    };
#pragma unroll 1
    for (int cell = 0; cell < CELLS; ++cell) {
        const unsigned blk = blockIdx.x * NOALLOC_THREADS + cell * THREADS + threadIdx.x;   // < 2^21 + 256
        const bool live = blk < (unsigned)a.nblk;
        if (!__any_sync(0xffffffffu, live)) break;
        unsigned p0 = 0, sp[4] = {0, 0, 0, 0};
        hmc::CellGrad<float> g;
        if (live) {
            float u[8][3];
            load_cell(blk, p0, u, sp);
            hmc::cell_gradients<float>(u, g);
        }
        // place of the cell's first point in sigma in 16-byte units (6 floats a point, even points)
        const unsigned base4 = live ? p0 / 2u * 3u : 0xffffffffu;
        float c[36];
        unsigned qprev = 0xffffffffu;
        // rows and the two points of each in a Gray-code order of the eight points, so that a boundary
        // through the cell reloads the stiffness row least often
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            const int row = n == 2 ? 3 : n == 3 ? 2 : n, ly = row & 1, lz = row >> 1;
            __syncwarp();
            if (live) {
                float out[12];
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    const int lx = m ^ (n & 1);
                    float e[6];
                    hmc::point_strain<float>(g, a.eb, lx, ly, lz, e);
                    const unsigned q = lx ? sp[row] >> 16 : sp[row] & 0xffffu;
                    if (q != qprev) {
                        load_c36<VEC>(a.ctab + 36ll * q, c);
                        qprev = q;
                    }
                    float w = 0.f;
#pragma unroll
                    for (int i = 0; i < 6; ++i) {
                        float acc = 0.f;
#pragma unroll
                        for (int j = 0; j < 6; ++j) acc += c[6 * i + j] * e[j];
                        out[6 * lx + i] = acc;
                        w += acc * e[i];
                        two_sum_add(hi[i], lo[i], acc);
                    }
                    two_sum_add(hi[6], lo[6], 0.5f * w);
                }
#pragma unroll
                for (int j = 0; j < 3; ++j)
                    stage[warp][3 * lane + j] = make_float4(out[4 * j], out[4 * j + 1], out[4 * j + 2], out[4 * j + 3]);
            }
            __syncwarp();
            const unsigned row4 = (unsigned)a.nx * (ly + (unsigned)a.ny * lz) / 2u * 3u;
            if constexpr (VEC) {
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const unsigned t = 32u * k + lane;
                    const unsigned to = __shfl_sync(0xffffffffu, base4, t / 3);
                    if (to != 0xffffffffu)
                        __stcs(reinterpret_cast<float4 *>(a.sigma) + (size_t)(to + row4 + t % 3), stage[warp][t]);
                }
            } else {
#pragma unroll
                for (int k = 0; k < 12; ++k) {
                    const unsigned t = 32u * k + lane;
                    const unsigned to = __shfl_sync(0xffffffffu, base4, t / 12);
                    if (to != 0xffffffffu)
                        a.sigma[4 * (size_t)(to + row4) + t % 12] = reinterpret_cast<const float *>(stage[warp])[t];
                }
            }
        }
    }
#pragma unroll
    for (int off = 16; off; off >>= 1)
#pragma unroll
        for (int i = 0; i < 7; ++i) {
            const float oh = __shfl_down_sync(0xffffffffu, hi[i], off);
            const float ol = __shfl_down_sync(0xffffffffu, lo[i], off);
            two_sum_add(hi[i], lo[i], oh);
            lo[i] += ol;
        }
    if (lane == 0)
        for (int i = 0; i < 7; ++i) red[warp][i] = (double)hi[i] + (double)lo[i];
    __syncthreads();
    if (threadIdx.x < 7) {
        double s = 0.0;
        for (int w = 0; w < THREADS / 32; ++w) s += red[w][threadIdx.x];
        a.partials[8ll * blockIdx.x + threadIdx.x] = s;  // every slot this call reads is written here
    }
}

// Fixed-order FP64 sum of the partials of all CTAs by one cluster of FINISH_CTAS CTAs: CTA k
// takes the slots k, k + FINISH_CTAS, ... with one warp per quantity, and CTA 0 adds the CTAs'
// sums.  (One CTA alone was bound by the FP64 rate of its SM: 31 us for the 8192 x 7 values of
// 256^3.)  Launched with programmatic serialisation, so that its launch overlaps the pass.
constexpr int FINISH_CTAS = 8;
__global__ void __cluster_dims__(FINISH_CTAS, 1, 1) __launch_bounds__(224) k_noalloc_finish(NoallocArgs a, int nparts) {
    __shared__ double sum[7];
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int i = threadIdx.x >> 5, lane = threadIdx.x & 31;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    double s = 0.0;
    for (int p = blockIdx.x + FINISH_CTAS * lane; p < nparts; p += FINISH_CTAS * 32) s += a.partials[8ll * p + i];
#pragma unroll
    for (int off = 16; off; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
    if (lane == 0) sum[i] = s;
    cl.sync();
    if (blockIdx.x == 0 && threadIdx.x < 7) {
        double t = 0.0;
        for (int k = 0; k < FINISH_CTAS; ++k) t += *cl.map_shared_rank(&sum[threadIdx.x], k);
        if (threadIdx.x < 6)
            a.mean[threadIdx.x] = t / (double)a.n_sites;
        else
            *a.energy = t;
    }
    cl.sync();   // the others' shared memory stays until it has been read
}


// Device address of the scratch array, looked up once per device.
std::mutex g_setup_mutex;
double *g_partials_addr[64] = {nullptr};

}  // namespace

extern "C" hmc_status hmc_stress_noalloc(const uint16_t *d_spins, const float *d_u, const float *d_ctab,
                                         const double *strain_bar, int32_t nx, int32_t ny, int32_t nz,
                                         float *d_sigma, double *d_mean, double *d_energy, void *stream) {
    if (!d_spins || !d_u || !d_ctab || !strain_bar || !d_sigma || !d_mean || !d_energy) {
        hmc::set_unbound_error("hmc_stress_noalloc: NULL pointer argument");
        return HMC_ERR_ARG;
    }
    if (nx < 4 || ny < 4 || nz < 4 || nx % 2 || ny % 2 || nz % 2) {
        hmc::set_unbound_error("hmc_stress_noalloc: grid edges must be even and >= 4");
        return HMC_ERR_ARG;
    }
    const long long nblk = (long long)(nx / 2) * (ny / 2) * (nz / 2);
    const long long nparts = (nblk + NOALLOC_THREADS - 1) / NOALLOC_THREADS;
    if (nparts > NOALLOC_MAX_CTAS) {
        hmc::set_unbound_error("hmc_stress_noalloc: " + std::to_string(8 * nblk) +
                               " points exceed the limit of " +
                               std::to_string(8ll * NOALLOC_THREADS * NOALLOC_MAX_CTAS) +
                               " points of its fixed scratch array");
        return HMC_ERR_ARG;
    }
    for (int i = 0; i < 6; ++i)
        if (!std::isfinite(strain_bar[i])) {
            hmc::set_unbound_error("hmc_stress_noalloc: non-finite strain_bar");
            return HMC_ERR_ARG;
        }
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= 64) {
        hmc::set_unbound_error(std::string("hmc_stress_noalloc: cudaGetDevice: ") + cudaGetErrorString(e));
        return HMC_ERR_CUDA;
    }
    double *partials = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_setup_mutex);
        if (!g_partials_addr[dev]) {
            void *p = nullptr;
            e = cudaGetSymbolAddress(&p, g_noalloc_partials);
            if (e != cudaSuccess) {
                hmc::set_unbound_error(std::string("hmc_stress_noalloc: cudaGetSymbolAddress: ") +
                                       cudaGetErrorString(e));
                return HMC_ERR_CUDA;
            }
            g_partials_addr[dev] = static_cast<double *>(p);
        }
        partials = g_partials_addr[dev];
    }
    NoallocArgs a;
    a.spins = d_spins;
    a.u = d_u;
    a.ctab = d_ctab;
    a.sigma = d_sigma;
    a.partials = partials;
    a.mean = d_mean;
    a.energy = d_energy;
    for (int i = 0; i < 6; ++i) a.eb[i] = (float)strain_bar[i];
    a.nx = nx; a.ny = ny; a.nz = nz;
    a.nbx = nx / 2; a.nby = ny / 2; a.nbz = nz / 2;
    a.nblk = nblk;
    a.n_sites = 8 * nblk;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    auto addr = [](const void *p) { return reinterpret_cast<uintptr_t>(p); };
    const bool vec = (addr(d_ctab) | addr(d_sigma)) % 16 == 0 && addr(d_spins) % 4 == 0;
    const unsigned grid = (unsigned)nparts;
    if (nparts < NOALLOC_SPREAD) {
        if (vec)
            k_stress_noalloc<true, 1><<<grid, NOALLOC_THREADS, 0, s>>>(a);
        else
            k_stress_noalloc<false, 1><<<grid, NOALLOC_THREADS, 0, s>>>(a);
    } else if (vec) {
        k_stress_noalloc<true, 4><<<grid, NOALLOC_THREADS / 4, 0, s>>>(a);
    } else {
        k_stress_noalloc<false, 4><<<grid, NOALLOC_THREADS / 4, 0, s>>>(a);
    }
    e = cudaGetLastError();
    if (e == cudaSuccess) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(FINISH_CTAS);
        cfg.blockDim = dim3(224);
        cfg.stream = s;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        e = cudaLaunchKernelEx(&cfg, k_noalloc_finish, a, (int)nparts);
    }
    if (e != cudaSuccess) {
        hmc::set_unbound_error(std::string("hmc_stress_noalloc: launch: ") + cudaGetErrorString(e));
        return HMC_ERR_CUDA;
    }
    return HMC_OK;
}
