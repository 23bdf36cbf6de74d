// Stress of every material point (for the sweeps), the end-of-step reductions
// and loading control, statistics (unlike bonds, orientation volumes, texture
// bins) and the spin layout conversions.
#include <cooperative_groups.h>

#include "hmc_device.cuh"

namespace hmc {

namespace {

// Error-free sum of two floats (Knuth's TwoSum): a + b = s + e exactly.
struct FSum {
    float hi, lo;
    __device__ __forceinline__ void add(float x) {
        const float s = hi + x;
        const float bb = s - hi;
        const float e = (hi - (s - bb)) + (x - bb);
        hi = s;
        lo += e;
    }
    __device__ __forceinline__ void add(const FSum &o) {
        add(o.hi);
        lo += o.lo;
    }
};

// Per-thread accumulators of the seven reduced quantities.
template <typename T>
struct Acc7;
template <>
struct Acc7<float> {
    FSum v[7];
    __device__ __forceinline__ void zero() {
        for (int i = 0; i < 7; ++i) v[i].hi = v[i].lo = 0.f;
    }
    __device__ __forceinline__ void add(int i, float x) { v[i].add(x); }
    __device__ __forceinline__ void warp_reduce() {
#pragma unroll
        for (int off = 16; off; off >>= 1)
#pragma unroll
            for (int i = 0; i < 7; ++i) {
                FSum o;
                o.hi = __shfl_down_sync(0xffffffffu, v[i].hi, off);
                o.lo = __shfl_down_sync(0xffffffffu, v[i].lo, off);
                v[i].add(o);
            }
    }
    __device__ __forceinline__ double get(int i) const { return (double)v[i].hi + (double)v[i].lo; }
};
template <>
struct Acc7<double> {
    double v[7];
    __device__ __forceinline__ void zero() {
        for (int i = 0; i < 7; ++i) v[i] = 0.0;
    }
    __device__ __forceinline__ void add(int i, double x) { v[i] += x; }
    __device__ __forceinline__ void warp_reduce() {
#pragma unroll
        for (int off = 16; off; off >>= 1)
#pragma unroll
            for (int i = 0; i < 7; ++i) v[i] += __shfl_down_sync(0xffffffffu, v[i], off);
    }
    __device__ __forceinline__ double get(int i) const { return v[i]; }
};

// Stores of one colour's component of a block's stress: streaming (evict-first), so that the
// 403 MB written per pass do not push the spin field out of L2.  (Storing the red stress with
// the normal priority, for the red half sweep that reads it next, measured no faster.)
template <typename T>
__device__ __forceinline__ void store4(T *p, const T (&v)[4]);
template <>
__device__ __forceinline__ void store4<float>(float *p, const float (&v)[4]) {
    __stcs(reinterpret_cast<float4 *>(p), make_float4(v[0], v[1], v[2], v[3]));
}
template <>
__device__ __forceinline__ void store4<double>(double *p, const double (&v)[4]) {
    __stcs(reinterpret_cast<double2 *>(p), make_double2(v[0], v[1]));
    __stcs(reinterpret_cast<double2 *>(p) + 1, make_double2(v[2], v[3]));
}

// Stress of the eight points of each cell from the current displacement; the
// colour-packed stress array is what the half sweeps read.  Each CTA covers the
// 256 blocks of one replica's tile with STRESS_THREADS threads, each taking
// STRESS_CELLS blocks in turn (the warp reduction below is then paid once per
// STRESS_CELLS cells), and writes its partial sums of sigma and of 1/2 sigma.eps
// (a cell's eight points summed plainly, then FP32 TwoSum pairs or FP64 within a
// thread and a warp, by T, and FP64 across warps) for a fixed-order final
// reduction.
// threads of a stress CTA (measured on the 256^3 workload: 256 threads, one block each, 0.244 ms;
// 128 threads 0.180 ms; 64 threads 0.156 ms; 32 threads 0.156 ms).  Each thread loads its next
// block's corners and spins while it works on the current one (0.156 -> 0.150 ms), held to
// 128 registers in FP32 (eight CTAs per SM).
// WIDE: 256 threads with one block each, for grids of few CTAs, where the chain of four blocks is
// longer than the pass; the blocks' sums go through shared memory and are added in the order
// of the other form, so both give the same bits.  The line is one wave of its CTAs (profiler,
// cold: FP32 106 CTAs 11.3 -> 7.8 us, 489 CTAs 14.2 -> 15.5 us; FP64 16 CTAs 91 -> 51 us).
constexpr int STRESS_THREADS = 64;
constexpr int STRESS_CELLS = BLOCK_THREADS / STRESS_THREADS;
static_assert(BLOCK_THREADS % STRESS_THREADS == 0, "a tile splits evenly over the threads");

// one wave of the wide form's CTAs on 152 SMs: two per SM in FP32, one in FP64
template <typename T>
constexpr int stress_wide() { return sizeof(T) == 4 ? 304 : 152; }

// A tile's partial sums from the accumulators of its first STRESS_THREADS threads.
template <typename T>
__device__ __forceinline__ void tile_sums(Acc7<T> &acc, double (&red)[STRESS_THREADS / 32][7], double *out) {
    acc.warp_reduce();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0)
        for (int i = 0; i < 7; ++i) red[warp][i] = acc.get(i);
    asm volatile("bar.sync 1, %0;" ::"n"(STRESS_THREADS) : "memory");   // the two warps that sum
    if (threadIdx.x < 7) {
        double s = 0.0;
        for (int w = 0; w < STRESS_THREADS / 32; ++w) s += red[w][threadIdx.x];
        out[threadIdx.x] = s;
    }
}
// ... from the sums of its n <= BLOCK_THREADS blocks, added in the order of the form without them
template <typename T>
__device__ __forceinline__ void tile_sums(const T (*cells)[7], int n, double (&red)[STRESS_THREADS / 32][7], double *out) {
    Acc7<T> acc;
    acc.zero();
    for (int t = threadIdx.x; t < n; t += STRESS_THREADS)
#pragma unroll
        for (int k = 0; k < 7; ++k) acc.add(k, cells[t][k]);
    tile_sums<T>(acc, red, out);
}

template <typename T, bool STORE, bool WIDE>
__global__ void __launch_bounds__(WIDE ? BLOCK_THREADS : STRESS_THREADS, sizeof(T) == 4 ? (WIDE ? 2 : 8) : 1)
    k_stress(StressArgs<T> a) {
    __shared__ double red[STRESS_THREADS / 32][7];
    __shared__ T cells[WIDE ? BLOCK_THREADS : 1][7];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int rep = __ldg(a.cta_rep + blockIdx.x);
    const Replica &R = a.reps[rep];
    const int t0 = (blockIdx.x - R.cta_off) * BLOCK_THREADS;
    Acc7<T> acc;
    acc.zero();
    const DevState *st = R.st;
    const int nbx = R.nbx, nby = R.nby, nbz = R.nbz;
    const T *u = a.u + 3 * R.blk_off;
    T *sig = a.sig + 48ll * R.blk_off;
    // a cell's corner displacements and spins, loaded one cell ahead of its arithmetic
    auto load_cell = [&](int blk, T (&uc)[8][3], uint4 &sp) {
        const int bx = blk % nbx, rr = blk / nbx;
        const int by = rr % nby, bz = rr / nby;
#pragma unroll
        for (int K = 0; K < 2; ++K)
#pragma unroll
            for (int J = 0; J < 2; ++J)
#pragma unroll
                for (int I = 0; I < 2; ++I) {
                    const int gi = bx + I == nbx ? 0 : bx + I;
                    const int gj = by + J == nby ? 0 : by + J;
                    const int gk = bz + K == nbz ? 0 : bz + K;
                    const int n = 3 * (gi + nbx * (gj + nby * gk));
#pragma unroll
                    for (int d = 0; d < 3; ++d) uc[corner(I, J, K)][d] = u[n + d];
                }
        sp = a.spins[R.blk_off + blk];
    };
    T un[8][3];
    uint4 spn = make_uint4(0, 0, 0, 0);
    int blk = t0 + threadIdx.x;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    T eb[6];
    load_ebar<T>(st, eb);
    if (blk < R.nblk) load_cell(blk, un, spn);
#pragma unroll 1
    for (int c8 = 0; c8 < (WIDE ? 1 : STRESS_CELLS); ++c8) {
        if (blk >= R.nblk) break;
        T uc[8][3];
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int d = 0; d < 3; ++d) uc[i][d] = un[i][d];
        const uint4 sp = spn;
        const int blk_next = blk + STRESS_THREADS;
        if (!WIDE && c8 + 1 < STRESS_CELLS && blk_next < R.nblk) load_cell(blk_next, un, spn);
        CellGrad<T> g;
        cell_gradients<T>(uc, g);
        T csum[7] = {T(0), T(0), T(0), T(0), T(0), T(0), T(0)};   // this cell's eight points, plain sums
        Row24<T> row;
        uint32_t qprev = 0xffffffffu;
        // red slots 0..3, then black 4..7: each colour's stress is stored as soon as it is formed
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            T out[6][4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int slot = 4 * c + j, L = slot_local(slot);
                T e[6], st[6];
                point_strain<T>(g, eb, L & 1, (L >> 1) & 1, L >> 2, e);
                const uint32_t q = spin_of(sp, slot);  // points of a cell mostly share one orientation
                if (q != qprev) {
                    row.load(a.ctab + 24ll * q);
                    qprev = q;
                }
                hooke21<T>(row.v, e, st);
                T w = T(0);
#pragma unroll
                for (int k = 0; k < 6; ++k) {
                    out[k][j] = st[k];
                    csum[k] += st[k];
                    w += st[k] * e[k];
                }
                csum[6] += T(0.5) * w;
            }
            if (STORE) {
#pragma unroll
                for (int k = 0; k < 6; ++k) store4<T>(sig + 4ll * ((long long)(c * 6 + k) * R.nblk + blk), out[k]);
            }
        }
#pragma unroll
        for (int k = 0; k < 7; ++k) {
            if (WIDE)
                cells[threadIdx.x][k] = csum[k];
            else
                acc.add(k, csum[k]);
        }
        blk = blk_next;
    }
    double *out = a.partials + 7ll * blockIdx.x;
    if constexpr (WIDE) {
        __syncthreads();
        if (threadIdx.x < STRESS_THREADS) tile_sums<T>(cells, min(BLOCK_THREADS, R.nblk - t0), red, out);
    } else {
        tile_sums<T>(acc, red, out);
    }
}

// The FP64 pass on small grids: a cluster of SPLIT CTAs to a tile and four threads to a cell, two points
// each.  An SM retires two FP64 lanes a clock, so what counts is over how many SMs the points are
// spread: a call at 32^3 took 70 us with its 16 tiles on 16 SMs and takes 45 us (24^3: 70 and 36),
// although a cell costs 1.5 times the operations (gradients formed once per thread).  16 clusters do not
// quite fit one CTA to an SM; asking for an SM each did not help.  The line: see launch_stress.
// The same products and sums in the same order as the other forms (a cell's points are summed in
// slot order, then tile_sums), so the bits are the same.
constexpr int SPLIT = 8, SPLIT_CELLS = BLOCK_THREADS / SPLIT;
template <bool STORE>
__global__ void __cluster_dims__(SPLIT, 1, 1) __launch_bounds__(4 * SPLIT_CELLS) k_stress_split(StressArgs<double> a) {
    namespace cg = cooperative_groups;
    __shared__ double red[STRESS_THREADS / 32][7];
    __shared__ double pts[8][7][SPLIT_CELLS + 1];      // by slot: stress, energy
    __shared__ double cells[BLOCK_THREADS][7];         // of the tile, in its first CTA
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    cg::cluster_group cl = cg::this_cluster();
    const int part = blockIdx.x % SPLIT, tile = blockIdx.x / SPLIT;
    const Replica &R = a.reps[__ldg(a.cta_rep + tile)];
    const int nblk = R.nblk, tile0 = (tile - R.cta_off) * BLOCK_THREADS, t0 = tile0 + part * SPLIT_CELLS;
    const int nbx = R.nbx, nby = R.nby, nbz = R.nbz;
    const double *u = a.u + 3 * R.blk_off;
    const DevState *st = R.st;
    const int tid = threadIdx.x, cell = tid >> 2, b = tid & 1, c = tid >> 1 & 1, blk = t0 + cell;
    const bool live = blk < nblk;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (live) {
        double eb[6];
        load_ebar<double>(st, eb);
        const uint4 sp = a.spins[R.blk_off + blk];
        double uc[8][3];
        const int bx = blk % nbx, rr = blk / nbx, by = rr % nby, bz = rr / nby;
#pragma unroll
        for (int n = 0; n < 8; ++n) {
            const int gi = (n & 1) && bx + 1 == nbx ? 0 : bx + (n & 1), gj = (n & 2) && by + 1 == nby ? 0 : by + (n >> 1 & 1);
            const int gk = (n & 4) && bz + 1 == nbz ? 0 : bz + (n >> 2);
#pragma unroll
            for (int d = 0; d < 3; ++d) uc[n][d] = u[3 * (gi + nbx * (gj + nby * gk)) + d];
        }
        // interp2's two stages at one point: x d0 + y d1
        auto mix = [](double x, double d0, double y, double d1) { return rfma(x, d0, rmul(y, d1)); };
        const double b0 = b ? 0.25 : 0.75, b1 = b ? 0.75 : 0.25;   // first stage, weights in y
        const double hb0 = b ? 0.125 : 0.375, hb1 = b ? 0.375 : 0.125, hc0 = c ? 0.125 : 0.375, hc1 = c ? 0.375 : 0.125;
        double gx[3], gy[2][3], gz[2][3];   // [d], [a][d]
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            gx[d] = mix(hc0, mix(b0, uc[1][d] - uc[0][d], b1, uc[3][d] - uc[2][d]), hc1,
                        mix(b0, uc[5][d] - uc[4][d], b1, uc[7][d] - uc[6][d]));
            const double y00 = uc[2][d] - uc[0][d], y10 = uc[3][d] - uc[1][d], y01 = uc[6][d] - uc[4][d], y11 = uc[7][d] - uc[5][d];
            const double z00 = uc[4][d] - uc[0][d], z10 = uc[5][d] - uc[1][d], z01 = uc[6][d] - uc[2][d], z11 = uc[7][d] - uc[3][d];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const double p = i ? 0.25 : 0.75, q = i ? 0.75 : 0.25;
                gy[i][d] = mix(hc0, mix(p, y00, q, y10), hc1, mix(p, y01, q, y11));
                gz[i][d] = mix(hb0, mix(p, z00, q, z10), hb1, mix(p, z01, q, z11));
            }
        }
        Row24<double> row;
        uint32_t qprev = 0xffffffffu;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const uint32_t q0 = b ? spin_of(sp, local_slot(i + 2)) : spin_of(sp, local_slot(i));
            const uint32_t q1 = b ? spin_of(sp, local_slot(i + 6)) : spin_of(sp, local_slot(i + 4));
            const uint32_t q = c ? q1 : q0;
            if (q != qprev) {
                row.load(a.ctab + 24ll * q);
                qprev = q;
            }
            const double e[6] = {eb[0] + gx[0], eb[1] + gy[i][1], eb[2] + gz[i][2], eb[3] + (gz[i][1] + gy[i][2]),
                                 eb[4] + (gz[i][0] + gx[2]), eb[5] + (gy[i][0] + gx[1])};
            double sg[6], w = 0.0;
            hooke21<double>(row.v, e, sg);
            double(&out)[7][SPLIT_CELLS + 1] = pts[local_slot(i + 2 * b + 4 * c)];
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                out[k][cell] = sg[k];
                w = rfma(sg[k], e[k], w);
            }
            out[6][cell] = 0.5 * w;
        }
    }
    cl.sync();   // the points are there, and the tile's first CTA runs
    double(*to)[7] = cl.map_shared_rank(cells, 0) + part * SPLIT_CELLS;
    for (int i = tid; i < 7 * SPLIT_CELLS; i += 4 * SPLIT_CELLS) {
        const int k = i / SPLIT_CELLS, n = i % SPLIT_CELLS;
        double s = 0.0;
#pragma unroll
        for (int slot = 0; slot < 8; ++slot) s += pts[slot][k][n];
        if (t0 + n < nblk) to[n][k] = s;
    }
    if (STORE && live) {
        double *sig = a.sig + 48ll * R.blk_off + 4ll * t0 + tid;
#pragma unroll
        for (int i = 0; i < 12; ++i) __stcs(sig + 4ll * i * nblk, pts[i / 6 * 4 + (tid & 3)][i % 6][cell]);
    }
    cl.sync();   // the tile's sums are there
    if (part == 0 && tid < STRESS_THREADS)
        tile_sums<double>(cells, min(BLOCK_THREADS, nblk - tile0), red, a.partials + 7ll * tile);
}

// sum over the lanes of a warp (a butterfly: every lane has it)
__device__ __forceinline__ double lanes_sum(double x) {
#pragma unroll
    for (int off = 16; off; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
    return x;
}

// End of a step: fixed-order FP64 reduction of each replica's stress partials (one set of seven
// per stress CTA), uniaxial control update of its mean strain, and its Monte Carlo step counter.
// Group g of G takes the CTAs g, g + G, ..., one warp per quantity; the last group to arrive sums the
// group sums the same way and finishes with one lane per strain component.  A warp instruction of
// the FP64 pipe takes 64 cycles however many lanes it serves, so what counts is the length of the
// chain: 20 instead of about 150 of them (the 250-thread tree and the update by one thread took
// 15 us; 4 us).
// after_sweeps: the kernel before this one is the black half sweep, which lets this one start only
// when the stress pass has finished: all but the results' stores runs beside it.  What it reads ahead of
// its wait comes from kernels that were over before the black half sweep passed its own: the stress
// pass and the end of the step before, never the kernel that it overlaps.
__global__ void __launch_bounds__(224) k_end_mcs(const Replica *reps, int nrep, int gmax, double *partials, int nctas,
                                                  int update_strain, int advance, int after_sweeps) {
    __shared__ double tot[7];
    __shared__ int last;
    const int r = blockIdx.x / gmax, grp = blockIdx.x % gmax;
    const Replica &R = reps[r];
    const int G = end_groups(R.ncta);
    const int i = threadIdx.x >> 5, lane = threadIdx.x & 31;   // quantity
    if (!after_sweeps) asm volatile("griddepcontrol.wait;" ::: "memory");
    if (grp >= G) return;
    DevState *st = R.st;
    double *gsum = partials + 7ll * nctas + 7ll * END_GROUPS * r;   // this replica's group sums
    unsigned *arrive = reinterpret_cast<unsigned *>(partials + 7ll * nctas + 7ll * END_GROUPS * nrep) + r;
    // the update's operands, loaded while the sums are formed (lane c: component c)
    const int c = lane < 6 ? lane : 0;
    double sr[6], axN = 0, axNs = 0, axB = 0, axNB = 1, eps0 = 0, sig0 = 0, ebar = 0;
    if (i == 0) {   // (from L2: the SM's L1 may hold a line from before the last end of a step)
#pragma unroll
        for (int j = 0; j < 6; ++j) sr[j] = __ldcg(st->sr + 6 * c + j);
        axN = __ldcg(st->axN + c);
        axNs = __ldcg(st->axNs + c);
        axB = __ldcg(st->axB + c);
        axNB = __ldcg(&st->axNB);
        eps0 = __ldcg(&st->eps0);
        sig0 = __ldcg(&st->sig0);
        ebar = __ldcg(st->ebar + c);
    }
    double s = 0.0;
    for (int p = grp + G * lane; p < R.ncta; p += 32 * G) s += __ldcg(partials + 7ll * (R.cta_off + p) + i);
    s = lanes_sum(s);
    if (G == 1) {
        if (lane == 0) tot[i] = s;
        __syncthreads();
    } else {
        if (lane == 0) {
            gsum[7 * grp + i] = s;
            __threadfence();
        }
        __syncthreads();
        if (threadIdx.x == 0) last = atomicAdd(arrive, 1u) == (unsigned)G - 1u;
        __syncthreads();
        if (!last) return;
        __threadfence();
        double t = lane < G ? __ldcg(gsum + 7 * lane + i) : 0.0;
        t = lanes_sum(t);
        if (lane == 0) tot[i] = t;
        __syncthreads();
    }
    if (i != 0) return;
    const bool comp = lane < 6;
    const double n_sites = 8.0 * (double)R.nblk;
    const double mean = tot[c] / n_sites, energy = tot[6];
    const bool bad = __any_sync(0xffffffffu, !isfinite(mean) || !isfinite(energy));
    const int bc = update_strain && !bad ? st->bc : -1;
    if (bc == 0) {
        // remove the lateral mean stress with the Reuss compliance, then restore
        // the axial strain along the uniaxial-stress direction S_R (n(x)n)
        const double nsn = lanes_sum(comp ? axNs * mean : 0.0);
        const double q = mean - nsn * axN;
        double d = 0.0;
#pragma unroll
        for (int j = 0; j < 6; ++j) d += sr[j] * __shfl_sync(0xffffffffu, q, j);
        const double e = ebar - d;
        const double beta = (eps0 - lanes_sum(comp ? axN * e : 0.0)) / axNB;
        ebar = e + beta * axB;
    } else if (bc == 2) {
        // stress control: Ebar += S_R (sig0 n(x)n - <sigma>)
        const double q = sig0 * axN - mean;
        double d = 0.0;
#pragma unroll
        for (int j = 0; j < 6; ++j) d += sr[j] * __shfl_sync(0xffffffffu, q, j);
        ebar += d;
    }
    // the black half sweep reads the step counter and the mean strain
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (comp) {
        st->mean_sigma[lane] = mean;
        if (bc == 0 || bc == 2) {
            st->ebar[lane] = ebar;
            st->ebar_f[lane] = (float)ebar;
        }
    }
    if (lane == 0) {
        st->energy = energy;
        if (bad) st->nonfinite = 1;
        if (advance) st->mcs += 1;
        *arrive = 0u;   // ready for the next launch
    }
}

// Upload check: flag any orientation index >= Q (8 indices per thread, 16 B loads).
__global__ void k_check_spins(const uint16_t *__restrict__ nat, long long n, int nq, DevState *st) {
    const long long n8 = n >> 3;
    int bad = 0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n8; i += (long long)gridDim.x * blockDim.x) {
        const uint4 v = __ldg(reinterpret_cast<const uint4 *>(nat) + i);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) bad |= ((w[k] & 0xffffu) >= (uint32_t)nq) | ((w[k] >> 16) >= (uint32_t)nq);
    }
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(&st->bad_spin, 1);
}

// natural uint16 field <-> 2x2x2 blocks in slot order; a field that the check flagged stays out
__global__ void k_pack_spins(const uint16_t *__restrict__ nat, uint4 *__restrict__ blk, int nx, int ny, int nz,
                             const int32_t *bad) {
    if (*bad) return;
    const int nbx = nx >> 1, nby = ny >> 1, nbz = nz >> 1;
    const long long nblk = (long long)nbx * nby * nbz;
    for (long long b = (long long)blockIdx.x * blockDim.x + threadIdx.x; b < nblk; b += (long long)gridDim.x * blockDim.x) {
        const int bx = (int)(b % nbx);
        const long long r = b / nbx;
        const int by = (int)(r % nby), bz = (int)(r / nby);
        uint32_t w[4] = {0, 0, 0, 0};
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            const int L = slot_local(s);
            const long long x = 2 * bx + (L & 1), y = 2 * by + ((L >> 1) & 1), z = 2 * bz + (L >> 2);
            const uint32_t q = nat[x + nx * (y + (long long)ny * z)];
            w[s >> 1] |= (s & 1) ? (q << 16) : q;
        }
        blk[b] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

__global__ void k_unpack_spins(const uint4 *__restrict__ blk, uint16_t *__restrict__ nat, int nx, int ny, int nz) {
    const int nbx = nx >> 1, nby = ny >> 1, nbz = nz >> 1;
    const long long nblk = (long long)nbx * nby * nbz;
    for (long long b = (long long)blockIdx.x * blockDim.x + threadIdx.x; b < nblk; b += (long long)gridDim.x * blockDim.x) {
        const int bx = (int)(b % nbx);
        const long long r = b / nbx;
        const int by = (int)(r % nby), bz = (int)(r / nby);
        const uint4 v = blk[b];
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            const int L = slot_local(s);
            const long long x = 2 * bx + (L & 1), y = 2 * by + ((L >> 1) & 1), z = 2 * bz + (L >> 2);
            nat[x + nx * (y + (long long)ny * z)] = spin_of(v, s);
        }
    }
}

// Unlike +x/+y/+z bonds of every site (each bond once) and the volume of
// every orientation, one thread per block.
__global__ void __launch_bounds__(256) k_bonds_counts(const uint4 *__restrict__ spins, int nbx, int nby, int nbz,
                                                      int nq, int smem_bins, unsigned long long *counts,
                                                      DevState *st) {
    extern __shared__ unsigned int hist[];
    if (smem_bins)
        for (int i = threadIdx.x; i < nq; i += blockDim.x) hist[i] = 0;
    __syncthreads();
    const long long nblk = (long long)nbx * nby * nbz;
    unsigned long long unlike = 0;
    for (long long b = (long long)blockIdx.x * blockDim.x + threadIdx.x; b < nblk; b += (long long)gridDim.x * blockDim.x) {
        const int bx = (int)(b % nbx);
        const long long r = b / nbx;
        const int by = (int)(r % nby), bz = (int)(r / nby);
        const uint4 me = __ldg(spins + b);
        const uint4 px = __ldg(spins + (b + (bx == nbx - 1 ? 1 - nbx : 1)));
        const uint4 py = __ldg(spins + (b + (by == nby - 1 ? -(long long)(nby - 1) * nbx : nbx)));
        const uint4 pz = __ldg(spins + (b + (bz == nbz - 1 ? -(long long)(nbz - 1) * nbx * nby : (long long)nbx * nby)));
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            const int L = slot_local(s);
            const int lx = L & 1, ly = (L >> 1) & 1, lz = L >> 2;
            const uint16_t q = spin_of(me, s);
            const uint16_t qx = lx ? spin_of(px, local_slot(L ^ 1)) : spin_of(me, local_slot(L ^ 1));
            const uint16_t qy = ly ? spin_of(py, local_slot(L ^ 2)) : spin_of(me, local_slot(L ^ 2));
            const uint16_t qz = lz ? spin_of(pz, local_slot(L ^ 4)) : spin_of(me, local_slot(L ^ 4));
            unlike += (q != qx) + (q != qy) + (q != qz);
            if (smem_bins)
                atomicAdd(&hist[q], 1u);
            else
                atomicAdd(&counts[q], 1ull);
        }
    }
    for (int off = 16; off; off >>= 1) unlike += __shfl_down_sync(0xffffffffu, unlike, off);
    if ((threadIdx.x & 31) == 0 && unlike) atomicAdd(&st->unlike, unlike);
    __syncthreads();
    if (smem_bins)
        for (int i = threadIdx.x; i < nq; i += blockDim.x)
            if (hist[i]) atomicAdd(&counts[i], (unsigned long long)hist[i]);
}

__global__ void k_bins(const unsigned long long *counts, const int32_t *binmap, int nq, int nbins,
                       unsigned long long *bins, double *fractions, long long n_sites) {
    for (int q = threadIdx.x; q < nq; q += blockDim.x) atomicAdd(&bins[binmap[q]], counts[q]);
    __syncthreads();
    for (int b = threadIdx.x; b < nbins; b += blockDim.x) fractions[b] = (double)bins[b] / (double)n_sites;
}

}  // namespace

// FP64 tiles up to which the pass is spread over clusters: three CTAs to an SM (a call at 40^3, 32
// tiles, takes 46 us against 70; at 48^3, 54 tiles, 69 against 71; at 56^3, 86 tiles, 82 against 71)
constexpr int STRESS_SPLIT = 57;

template <typename T>
cudaError_t launch_stress(const StressArgs<T> &a, bool store, cudaStream_t s) {
    if constexpr (sizeof(T) == 8)
        if (a.nctas <= STRESS_SPLIT)
            return launch_pdl(store ? k_stress_split<true> : k_stress_split<false>, a.nctas * SPLIT, 4 * SPLIT_CELLS, 0, s, a);
    if (a.nctas <= stress_wide<T>())
        return launch_pdl(store ? k_stress<T, true, true> : k_stress<T, false, true>, a.nctas, BLOCK_THREADS, 0, s, a);
    return launch_pdl(store ? k_stress<T, true, false> : k_stress<T, false, false>, a.nctas, STRESS_THREADS, 0, s, a);
}
template cudaError_t launch_stress<float>(const StressArgs<float> &, bool, cudaStream_t);
template cudaError_t launch_stress<double>(const StressArgs<double> &, bool, cudaStream_t);

cudaError_t launch_end_mcs(const Replica *reps, int nrep, int max_ncta, double *partials, int nctas, int update_strain,
                           int advance, int after_sweeps, cudaStream_t s) {
    const int gmax = end_groups(max_ncta);
    return launch_pdl(k_end_mcs, (unsigned)(nrep * gmax), 224u, 0, s, reps, nrep, gmax, partials, nctas, update_strain,
                      advance, after_sweeps);
}

static int grid_for(long long n) {
    long long g = (n + 255) / 256;
    if (g > 65535ll * 8) g = 65535ll * 8;
    if (g < 1) g = 1;
    return (int)g;
}

cudaError_t launch_check_spins(const uint16_t *nat, long long n, int nq, DevState *st, cudaStream_t s) {
    k_check_spins<<<grid_for(n >> 3), 256, 0, s>>>(nat, n, nq, st);
    return cudaGetLastError();
}

cudaError_t launch_pack_spins(const uint16_t *nat, uint4 *blk, int nx, int ny, int nz, const int32_t *bad,
                              cudaStream_t s) {
    const long long nblk = (long long)(nx / 2) * (ny / 2) * (nz / 2);
    k_pack_spins<<<grid_for(nblk), 256, 0, s>>>(nat, blk, nx, ny, nz, bad);
    return cudaGetLastError();
}

cudaError_t launch_unpack_spins(const uint4 *blk, uint16_t *nat, int nx, int ny, int nz, cudaStream_t s) {
    const long long nblk = (long long)(nx / 2) * (ny / 2) * (nz / 2);
    k_unpack_spins<<<grid_for(nblk), 256, 0, s>>>(blk, nat, nx, ny, nz);
    return cudaGetLastError();
}

cudaError_t launch_bonds_counts(const uint4 *blk, int nbx, int nby, int nbz, int nq, unsigned long long *counts,
                                DevState *st, cudaStream_t s) {
    const long long nblk = (long long)nbx * nby * nbz;
    const int smem_bins = nq <= 12288;
    long long g = (nblk + 255) / 256;
    if (g > 4096) g = 4096;  // grid-stride: fewer, longer CTAs amortise the shared histogram flush
    k_bonds_counts<<<(int)g, 256, smem_bins ? nq * sizeof(unsigned int) : 0, s>>>(blk, nbx, nby, nbz, nq, smem_bins,
                                                                                counts, st);
    return cudaGetLastError();
}

cudaError_t launch_bins(const unsigned long long *counts, const int32_t *binmap, int nq, int nbins,
                        unsigned long long *bins, double *fractions, long long n_sites, cudaStream_t s) {
    k_bins<<<1, 1024, 0, s>>>(counts, binmap, nq, nbins, bins, fractions, n_sites);
    return cudaGetLastError();
}

}  // namespace hmc
