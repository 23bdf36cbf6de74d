// Fused explicit MPM step in FP32 (Sec. "Elastic Deformation"): for every material
// point strain from the nodal displacement, Hooke's law (Eq. 1) with the
// point's rotated stiffness, internal nodal force, then the damped
// velocity / displacement update of every node -- one kernel, one pass over
// the spins and the nodal state.
//
// Two forms, chosen per batch by the autotuner; both give the same bits.
//
// March (k_mpm_step): 256 or 128 threads compute a patch of W x H <= 256 or 128 cells per cell
// plane (one thread per cell, all eight points of the cell) and owns the (W-1) x (H-1) nodes
// whose four lower and four upper cells all lie in the patch.  It marches up a chunk of planes
// in z: each cell writes its eight nodal force contributions to shared memory, and a node's
// force is the sum of its four cells below (carried in registers from the previous plane) and
// four above.  Node planes are triple-buffered in shared memory and the next plane's spins and
// the owned node's velocity are fetched one plane ahead.  Displacements are read from one
// buffer and written to the other, so CTAs never race on the halo.  The (replica, tile, plane)
// space of the batch is cut into one contiguous range per resident CTA, over replicas of any
// size; a range costs its planes and one more per tile that it enters (the restart plane below
// its first), and the cuts are laid so that the costliest range is as short as possible.
// W and H are not fixed: a patch of 16 x 16 covers 15 x 15 nodes, which leaves edges of 64 or 50
// nodes with slivers of tiles; the fitted patch divides each replica's edges evenly.
//
// Block (k_mpm_block): for grids whose nodes fit the GPU in one go.  A CTA computes a block of
// W x H x D <= 256 cells at once, one thread each, and owns its (W-1)(H-1)(D-1) inner nodes:
// twice the cells of the march, but one load, one cell, one barrier and one store long.
//
// Scaling: the interpolation weights 3/4 and 1/4 of the trilinear shape
// functions at the points 1/4 and 3/4 of the cell are applied as 3 and 1; the
// factors 1/16 and 1/h are folded into the displacements held in shared memory
// (u/32) and into the force constant of the node update (-dt/(32 m)) -- both
// exact powers of two.
#include "hmc_device.cuh"

namespace hmc {

namespace {

// A node's or a cell corner's three components and a pad: one 16-byte shared-memory access
// in FP32 (eight consecutive lanes read 128 contiguous bytes, free of bank conflicts)
// instead of three 4-byte ones.
struct alignas(16) Vec4 {
    float x, y, z, p;
};

template <int GT>
struct MarchSmem {
    static constexpr int NODES = GT == MPM_THREADS ? MPM_NODES : MPM_HALF_NODES;
    Vec4 us[3][NODES];             // node planes, row-major with a patch's nodes a row, held as u/32
    Vec4 fb[4][GT];                // cell contributions to their lower corner nodes (corner I+2J)
    Vec4 ft[4][GT];                // ... to their upper corner nodes
};
template <int THREADS>
struct BlockSmem {
    Vec4 us[2 * THREADS];
    Vec4 f[8][THREADS];            // cell contributions to corner I + 2J + 4K
};

// Node plane k of a patch with origin node (i0-1, j0-1) and P nodes a row, read from global
// memory into registers / written to shared memory.
template <int GT>
struct PlaneLoad {
    static constexpr int PER = (MarchSmem<GT>::NODES + GT - 1) / GT;
    float r[PER][3];
    int col[PER];   // this thread's nodes as (i + nbx j) in the replica's node plane, -1 beyond the patch
    // once per tile: the periodic (i, j) of each node this thread loads
    __device__ __forceinline__ void prepare(int i0, int j0, int P, int n, int nbx, int nby) {
#pragma unroll
        for (int m = 0; m < PER; ++m) {
            const int t = threadIdx.x % GT + m * GT;
            col[m] = t < n ? wrapi(i0 - 1 + t % P, nbx) + nbx * wrapi(j0 - 1 + t / P, nby) : -1;
        }
    }
    // node plane k, -1 <= k <= nbz (periodic in z)
    __device__ __forceinline__ void fetch(const float *u, long long node0, int k, int nbz, int plane) {
        const int gk = k < 0 ? k + nbz : (k >= nbz ? k - nbz : k);
        const float *base = u + 3 * (node0 + (long long)plane * gk);
#pragma unroll
        for (int m = 0; m < PER; ++m)
            if (col[m] >= 0) {
                const float *p = base + 3 * col[m];
                r[m][0] = p[0];
                r[m][1] = p[1];
                r[m][2] = p[2];
            }
    }
    __device__ __forceinline__ void store(Vec4 *us) const {
#pragma unroll
        for (int m = 0; m < PER; ++m)
            if (col[m] >= 0)
                us[threadIdx.x % GT + m * GT] =
                    Vec4{r[m][0] * 0.03125f, r[m][1] * 0.03125f, r[m][2] * 0.03125f, 0.f};
    }
};

// Hooke's law for the MPM step: the cubic form of one rotated cubic material,
//   sigma = (C12 tr + Ad p2) I + 2 C44 eps + Ad (p0 - p2) a0 a0 + Ad (p1 - p2) a1 a1,
//   p_m = a_m.eps.a_m = W_m.e,  p2 = tr - p0 - p1,  Ad = C11 - C12 - 2 C44,
// with e the Voigt strain (engineering shear), sigma in tensor shear and W_m the Voigt
// weights (x^2, y^2, z^2, yz, xz, xy) of crystal axis a_m = (x, y, z); the third axis
// drops out because the axes are orthonormal.  12 values per orientation instead of
// 21, so the table of up to MPM_STAB_MAX orientations sits in shared memory (STAB) and
// a cell whose points change orientation reloads from there.  Every operation is
// explicitly rounded, in one order, so that both forms of the step give the same bits.
__device__ __forceinline__ void cubic_hooke(const float (&w)[12], const float (&cub)[4], const float (&e)[6],
                                            float (&s)[6]) {
    float p0 = __fmul_rn(w[0], e[0]), p1 = __fmul_rn(w[6], e[0]);
#pragma unroll
    for (int k = 1; k < 6; ++k) {
        p0 = __fmaf_rn(w[k], e[k], p0);
        p1 = __fmaf_rn(w[6 + k], e[k], p1);
    }
    const float tr = __fadd_rn(__fadd_rn(e[0], e[1]), e[2]);
    const float p2 = __fsub_rn(__fsub_rn(tr, p0), p1);
    // A = Ad p2; c = C12 tr + A; d_m = Ad p_m - A (one fused operation each)
    const float A = __fmul_rn(cub[3], p2);
    const float c = __fmaf_rn(cub[0], tr, A);
    const float d0 = __fmaf_rn(cub[3], p0, -A), d1 = __fmaf_rn(cub[3], p1, -A);
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const float base = k < 3 ? __fmaf_rn(cub[1], e[k], c) : __fmul_rn(cub[2], e[k]);
        s[k] = __fmaf_rn(d1, w[6 + k], __fmaf_rn(d0, w[k], base));
    }
}

template <bool STAB>
struct HookeRow {
    float w[12];
    // cw: the table in shared memory (STAB) or in global memory
    __device__ __forceinline__ void load(const float *cw, uint32_t q) {
        const float4 *p = reinterpret_cast<const float4 *>(cw + 12 * q);
        float4 v[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) v[i] = STAB ? p[i] : __ldg(p + i);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            w[4 * i] = v[i].x; w[4 * i + 1] = v[i].y; w[4 * i + 2] = v[i].z; w[4 * i + 3] = v[i].w;
        }
    }
    __device__ __forceinline__ void apply(const float (&e)[6], float (&s)[6], const float (&cub)[4]) const {
        cubic_hooke(w, cub, e, s);
    }
};

// 2x2 -> 2x2 transform with weights 3 (same side) and 1 (other side) in both
// indices: o[b][c] = sum_J sum_K W(J,b) W(K,c) d[J][K], eight FMAs.
__device__ __forceinline__ void interp31(float d00, float d10, float d01, float d11, float (&o)[2][2]) {
    const float e00 = fma(3.f, d00, d10), e10 = fma(3.f, d10, d00);  // (b, K=0)
    const float e01 = fma(3.f, d01, d11), e11 = fma(3.f, d11, d01);  // (b, K=1)
    o[0][0] = fma(3.f, e00, e01);
    o[0][1] = fma(3.f, e01, e00);
    o[1][0] = fma(3.f, e10, e11);
    o[1][1] = fma(3.f, e11, e10);
}

// Displacement gradients of the cell's points from corner displacements held
// as u/32: the 3/1 weights then give (1/h) sum w w (difference) exactly.
__device__ __forceinline__ void cell_gradients31(const float (&u)[8][3], CellGrad<float> &g) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        float o[2][2];
        interp31(u[corner(1, 0, 0)][d] - u[corner(0, 0, 0)][d], u[corner(1, 1, 0)][d] - u[corner(0, 1, 0)][d],
                    u[corner(1, 0, 1)][d] - u[corner(0, 0, 1)][d], u[corner(1, 1, 1)][d] - u[corner(0, 1, 1)][d], o);
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int c = 0; c < 2; ++c) g.gx[b][c][d] = o[b][c];
        interp31(u[corner(0, 1, 0)][d] - u[corner(0, 0, 0)][d], u[corner(1, 1, 0)][d] - u[corner(1, 0, 0)][d],
                    u[corner(0, 1, 1)][d] - u[corner(0, 0, 1)][d], u[corner(1, 1, 1)][d] - u[corner(1, 0, 1)][d], o);
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int c = 0; c < 2; ++c) g.gy[a][c][d] = o[a][c];
        interp31(u[corner(0, 0, 1)][d] - u[corner(0, 0, 0)][d], u[corner(1, 0, 1)][d] - u[corner(1, 0, 0)][d],
                    u[corner(0, 1, 1)][d] - u[corner(0, 1, 0)][d], u[corner(1, 1, 1)][d] - u[corner(1, 1, 0)][d], o);
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 2; ++b) g.gz[a][b][d] = o[a][b];
    }
}

// The point visited n-th in a cell: the corners in a Gray-code order, one coordinate
// changing per step.  A cell split by a grain boundary reloads its stiffness row
// whenever the orientation changes from one point to the next: 4, 2 and 1 times for a
// boundary plane normal to x, y and z (7, 3 and 1 in plain corner order).  Every MPM
// variant visits the points in this order, so their results stay bit-identical.
__host__ __device__ constexpr int gray_point(int n) {
    return n == 0 ? 0 : n == 1 ? 1 : n == 2 ? 3 : n == 3 ? 2 : n == 4 ? 6 : n == 5 ? 7 : n == 6 ? 5 : 4;
}

// Eight points of one cell: F[corner] = (2I-1) X'[J][K] + (2J-1) Y'[I][K] +
// (2K-1) Z'[I][J] with X', Y', Z' the 3/1-weighted sums of the traction
// columns of sigma; the nodal force is -(V/h)/16 F = -F/32 (V = 1 voxel, h = 2).
template <bool STAB>
__device__ __forceinline__ void cell_forces(const float (&u)[8][3], const uint4 &sp,
                                            const float *cw, const float (&cub)[4], const float (&eb)[6],
                                            float (&f)[8][3]) {
    // the first point's stiffness row is requested before the gradients are formed, so that
    // its load latency overlaps them
    HookeRow<STAB> row;
    uint32_t qprev = spin_of(sp, local_slot(0));
    row.load(cw, qprev);
    CellGrad<float> g;
    cell_gradients31(u, g);
    // each strain component of a point is eb_k plus gradient entries that two points share:
    // add eb_k once to the one entry of each component that only that component uses (the
    // normal entries, and one of the two entries of each shear)
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            g.gx[i][j][0] = eb[0] + g.gx[i][j][0];
            g.gy[i][j][1] = eb[1] + g.gy[i][j][1];
            g.gz[i][j][2] = eb[2] + g.gz[i][j][2];
            g.gz[i][j][1] = eb[3] + g.gz[i][j][1];
            g.gz[i][j][0] = eb[4] + g.gz[i][j][0];
            g.gy[i][j][0] = eb[5] + g.gy[i][j][0];
        }
    float tx[2][2][3], ty[2][2][3], tz[2][2][3];  // traction sums over a, b, c respectively
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int d = 0; d < 3; ++d) tx[i][j][d] = ty[i][j][d] = tz[i][j][d] = 0.f;
#pragma unroll
    for (int n = 0; n < 8; ++n) {
        const int L = gray_point(n);
        const int a = L & 1, b = (L >> 1) & 1, c = L >> 2;
        float e[6], s[6];
        e[0] = g.gx[b][c][0];
        e[1] = g.gy[a][c][1];
        e[2] = g.gz[a][b][2];
        e[3] = g.gz[a][b][1] + g.gy[a][c][2];
        e[4] = g.gz[a][b][0] + g.gx[b][c][2];
        e[5] = g.gy[a][c][0] + g.gx[b][c][1];
        // points of one cell mostly share one orientation: fetch the row only when it changes
        const uint32_t q = spin_of(sp, local_slot(L));
        if (q != qprev) {
            row.load(cw, q);
            qprev = q;
        }
        row.apply(e, s, cub);
        // columns of sigma: x = (s0,s5,s4), y = (s5,s1,s3), z = (s4,s3,s2)
        tx[b][c][0] += s[0]; tx[b][c][1] += s[5]; tx[b][c][2] += s[4];
        ty[a][c][0] += s[5]; ty[a][c][1] += s[1]; ty[a][c][2] += s[3];
        tz[a][b][0] += s[4]; tz[a][b][1] += s[3]; tz[a][b][2] += s[2];
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        float X[2][2], Y[2][2], Z[2][2];
        interp31(tx[0][0][d], tx[1][0][d], tx[0][1][d], tx[1][1][d], X);  // X[J][K]
        interp31(ty[0][0][d], ty[1][0][d], ty[0][1][d], ty[1][1][d], Y);  // Y[I][K]
        interp31(tz[0][0][d], tz[1][0][d], tz[0][1][d], tz[1][1][d], Z);  // Z[I][J]
#pragma unroll
        for (int K = 0; K < 2; ++K)
#pragma unroll
            for (int J = 0; J < 2; ++J)
#pragma unroll
                for (int I = 0; I < 2; ++I) {
                    const float fx = I ? X[J][K] : -X[J][K];
                    const float fy = J ? Y[I][K] : -Y[I][K];
                    const float fz = K ? Z[I][J] : -Z[I][J];
                    f[corner(I, J, K)][d] = fx + fy + fz;
                }
    }
}

// the FP32 orientation table of the cubic form, staged in shared memory behind a kernel's tiles
template <bool STAB>
__device__ __forceinline__ const float *stage_table(const MpmArgs<float> &a, unsigned char *behind) {
    if constexpr (!STAB) return a.cubw;
    float *ts = reinterpret_cast<float *>(behind);
    for (int i = threadIdx.x; i < 3 * a.nq; i += blockDim.x)
        reinterpret_cast<float4 *>(ts)[i] = __ldg(reinterpret_cast<const float4 *>(a.cubw) + i);
    __syncthreads();
    return ts;
}

__device__ __forceinline__ void take(float (&u)[3], const Vec4 &n) {
    u[0] = n.x;
    u[1] = n.y;
    u[2] = n.z;
}

// barrier of one march (barrier 0 is the CTA's own)
template <int GT, int GROUPS>
__device__ __forceinline__ void march_sync() {
    if constexpr (GROUPS == 1)
        __syncthreads();
    else
        asm volatile("bar.sync %0, %1;" ::"r"((int)(threadIdx.x / GT) + 1), "n"(GT) : "memory");
}

// PITCH: nodes a row of the patch, 0 for W + 1 (the 16x16 patch's constant 17 saves 1 % at 256^3)
// GT: threads of a march, GROUPS: marches to a CTA, which share its orientation table and run on
// their own behind barriers of their own.  A march of 128 threads computes 8 % more halo than one of
// 256, but four of them per SM are out of step with each other, so that one's barriers and node
// updates lie under the others' cells: at 200^3 (256 orientations) 50.0 -> 48.8 us a step.  At 256^3
// (1024 orientations, a table of 48 KB) four tables would not fit; with one for four marches, which
// also leaves L1 43 KB more than two CTAs of 256 do, 96.7 -> 88.1 us.
template <int GT, int GROUPS, bool STAB, int PITCH>
__global__ void __launch_bounds__(GT *GROUPS, 512 / (GT * GROUPS)) k_mpm_step(MpmArgs<float> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x % GT;
    MarchSmem<GT> &sm = reinterpret_cast<MarchSmem<GT> *>(smem_raw)[threadIdx.x / GT];
    const float fscale = -a.dt_over_m * 0.03125f;          // -dt / (32 m)
    // the next step may be launched now: its CTAs take the SM slots this grid's CTAs free
    // and stage their table while this grid finishes
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const float *cw = stage_table<STAB>(a, smem_raw + GROUPS * sizeof(MarchSmem<GT>));
    float cub[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) cub[i] = a.cub[i];
    // this march's contiguous range of the linear (replica, tile, plane) index; those of a CTA lie far
    // apart, so that fewer ranges than there is room for load the SMs evenly
    const int range = GROUPS == 1 ? (int)blockIdx.x : (int)(threadIdx.x / GT * gridDim.x + blockIdx.x);
    if (GROUPS > 1 && range >= a.ranges) return;
    long long w = a.cuts[range];
    const long long wend = a.cuts[range + 1];
    int r = 0;
    while (w < wend) {
        while (a.sched[r + 1].off <= w) ++r;              // replica of work item w (ranges are ascending)
        const Replica &R = a.reps[r];
        const MpmSched &SC = a.sched[r];
        // in a register: read through the table it is loaded again in every plane, because the stores of
        // u and v might alias it (at 256^3 97 -> 88 us with four marches a CTA, 99.6 -> 96.7 with one)
        const long long node0 = R.blk_off;
        const int nbx = R.nbx, nby = R.nby, nbz = R.nbz;
        const long long lw = w - SC.off;
        const int tile = (int)(lw / nbz);
        const int k0 = (int)(lw - (long long)tile * nbz);
        const long long rem = min(wend, a.sched[r + 1].off) - w;
        const int kend = (int)min((long long)nbz, (long long)k0 + rem);
        w += kend - k0;
        const int i0 = (tile % SC.tiles_x) * SC.ox, j0 = (tile / SC.tiles_x) * SC.oy;
        // cells needed by the tile's owned nodes: W x H (fewer at the high edges of the replica),
        // numbered W-wide so that the active threads fill whole warps
        const int W = min(SC.ox, nbx - i0) + 1, H = min(SC.oy, nby - j0) + 1;
        const int P = PITCH ? PITCH : W + 1;
        const int lci = tid % W, lcj = tid / W;               // this thread's cell in the patch
        const bool need = tid < W * H;
        const bool own = need && lci >= 1 && lcj >= 1;        // it owns the node at its cell's lower corner
        const int plane = nbx * nby;
        const long long col = node0 + wrapi(i0 - 1 + lci, nbx) + nbx * wrapi(j0 - 1 + lcj, nby);
        const int nd = lci + P * lcj;                         // that node in the patch
        PlaneLoad<GT> pl;
        int b0 = 0, b1 = 1, b2 = 2;
        pl.prepare(i0, j0, P, P * (H + 1), nbx, nby);
        // u, v and the spins come from the kernels before this one; everything above reads only tables
        // (from the second tile on there is nothing left to wait for).  With the wait ahead of the
        // range's look-ups, a chain of dependent loads, a step took 1.35 us more (128^3 19.0 -> 17.65
        // us); with the two first planes loaded one after the other, 0.25 us more
        asm volatile("griddepcontrol.wait;" ::: "memory");
        float eb[6];
        load_ebar<float>(R.st, eb);
        PlaneLoad<GT> pl0 = pl;
        pl0.fetch(a.u_in, node0, k0 - 1, nbz, plane);
        pl.fetch(a.u_in, node0, k0, nbz, plane);
        uint4 sp = need ? a.spins[col + (long long)plane * wrapi(k0 - 1, nbz)] : make_uint4(0, 0, 0, 0);
        pl0.store(sm.us[b0]);
        pl.store(sm.us[b1]);
        march_sync<GT, GROUPS>();

        float acc[3] = {0.f, 0.f, 0.f};
        // this column's spins of the next plane, and its node's velocity and new displacement in
        // the current plane, advanced by one plane per iteration
        const uint4 *spn = a.spins + col + (long long)plane * k0;
        float *vp = a.v + 3 * (col + (long long)plane * k0);
        float *up = a.u_out + 3 * (col + (long long)plane * k0);
        const long long pstride = 3ll * plane;
        for (int kk = k0 - 1; kk < kend; ++kk) {
            // one plane ahead: next plane's spins and u, this plane's owned velocity
            uint4 sp_next = make_uint4(0, 0, 0, 0);
            if (need && kk + 1 < kend) sp_next = *spn;
            spn += plane;
            float vold[3] = {0.f, 0.f, 0.f};
            if (own && kk >= k0) {
#pragma unroll
                for (int d = 0; d < 3; ++d) vold[d] = vp[d];
            }
            const bool more = kk + 1 < kend;
            if (more) pl.fetch(a.u_in, node0, kk + 2, nbz, plane);
            float uc[3] = {0.f, 0.f, 0.f};   // the owned node's u/32: corner 0 of this thread's cell
            if (need) {
                float u[8][3];
                const Vec4 *n0 = sm.us[b0] + nd, *n1 = sm.us[b1] + nd;
#pragma unroll
                for (int c = 0; c < 8; ++c) take(u[c], (c & 4 ? n1 : n0)[(c & 1) + (c & 2 ? P : 0)]);
                float f[8][3];
#pragma unroll
                for (int d = 0; d < 3; ++d) uc[d] = u[0][d];
                cell_forces<STAB>(u, sp, cw, cub, eb, f);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    sm.fb[c][tid] = Vec4{f[c][0], f[c][1], f[c][2], 0.f};
                    sm.ft[c][tid] = Vec4{f[c + 4][0], f[c + 4][1], f[c + 4][2], 0.f};
                }
            }
            if (more) pl.store(sm.us[b2]);   // buffer b2 was last read before the previous barrier
            march_sync<GT, GROUPS>();
            if (own) {
                // cells (lci-1, lcj-1), (lci, lcj-1), (lci-1, lcj), (lci, lcj) see this node as corner 3, 2, 1, 0
                if (kk >= k0) {
                    const Vec4 c3 = sm.fb[3][tid - W - 1], c2 = sm.fb[2][tid - W];
                    const Vec4 c1 = sm.fb[1][tid - 1], c0 = sm.fb[0][tid];
                    const float F[3] = {acc[0] + c3.x + c2.x + c1.x + c0.x, acc[1] + c3.y + c2.y + c1.y + c0.y,
                                        acc[2] + c3.z + c2.z + c1.z + c0.z};
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        const float vn = rfma(fscale, F[d], rmul(a.keep, vold[d]));
                        vp[d] = vn;
                        up[d] = rfma(a.dt, vn, rmul(a.ukeep, uc[d] * 32.f));
                    }
                    vp += pstride;
                    up += pstride;
                }
                const Vec4 c3 = sm.ft[3][tid - W - 1], c2 = sm.ft[2][tid - W];
                const Vec4 c1 = sm.ft[1][tid - 1], c0 = sm.ft[0][tid];
                acc[0] = c3.x + c2.x + c1.x + c0.x;
                acc[1] = c3.y + c2.y + c1.y + c0.y;
                acc[2] = c3.z + c2.z + c1.z + c0.z;
            }
            march_sync<GT, GROUPS>();
            const int t = b0;
            b0 = b1;
            b1 = b2;
            b2 = t;
            sp = sp_next;
        }
    }
}

// One block per CTA, every cell at once.  What bounds it: the chain of one load, one cell, one
// barrier and one store (see the dispatch in hmc_api.cu for the sizes where it is the faster form).
template <int THREADS, bool STAB>
__global__ void __launch_bounds__(THREADS, 512 / THREADS) k_mpm_block(MpmArgs<float> a) {
    constexpr int PER = 2;   // nodes a thread loads: the blocks are laid with at most two a cell
    using Smem = BlockSmem<THREADS>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Smem &sm = *reinterpret_cast<Smem *>(smem_raw);
    const int tid = threadIdx.x;
    const float fscale = -a.dt_over_m * 0.03125f;          // -dt / (32 m)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const float *cw = stage_table<STAB>(a, smem_raw + sizeof(Smem));
    float cub[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) cub[i] = a.cub[i];
    int r = 0;
    while (a.sched[r + 1].off <= blockIdx.x) ++r;
    const Replica &R = a.reps[r];
    const MpmSched &SC = a.sched[r];
    const BlockPlace B(SC, R, blockIdx.x - (int)SC.off);
    const int nbx = R.nbx, nby = R.nby, nbz = R.nbz;
    const int W = B.W, H = B.H, P = W + 1, PP = P * (H + 1);
    const int lci = tid % W, lcj = tid / W % H, lck = tid / (W * H);
    const bool need = lck < B.D;
    const bool own = need && lci >= 1 && lcj >= 1 && lck >= 1;
    const long long at = R.blk_off + wrapi(B.i0 - 1 + lci, nbx) +
                         (long long)nbx * (wrapi(B.j0 - 1 + lcj, nby) + (long long)nby * wrapi(B.k0 - 1 + lck, nbz));
    long long node[PER];
#pragma unroll
    for (int m = 0; m < PER; ++m) node[m] = B.node(R, tid + m * THREADS);
    float eb[6], un[3] = {0.f, 0.f, 0.f}, vold[3] = {0.f, 0.f, 0.f};
    const DevState *st = R.st;   // (looked up behind the wait, the mean strain came last: 32^3 3.7 -> 3.5 us)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    load_ebar<float>(st, eb);
    const uint4 sp = need ? a.spins[at] : make_uint4(0, 0, 0, 0);
    if (own) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            vold[d] = a.v[3 * at + d];
            un[d] = a.u_in[3 * at + d];
        }
    }
#pragma unroll
    for (int m = 0; m < PER; ++m)
        if (node[m] >= 0) {
            const float *p = a.u_in + 3 * node[m];
            sm.us[tid + m * THREADS] = Vec4{p[0] * 0.03125f, p[1] * 0.03125f, p[2] * 0.03125f, 0.f};
        }
    __syncthreads();
    if (need) {
        float u[8][3], f[8][3];
        const Vec4 *n0 = sm.us + lci + P * lcj + PP * lck;
#pragma unroll
        for (int c = 0; c < 8; ++c) take(u[c], n0[(c & 1) + (c & 2 ? P : 0) + (c & 4 ? PP : 0)]);
        cell_forces<STAB>(u, sp, cw, cub, eb, f);
#pragma unroll
        for (int c = 0; c < 8; ++c) sm.f[c][tid] = Vec4{f[c][0], f[c][1], f[c][2], 0.f};
    }
    __syncthreads();
    if (own) {
        // the march's order: the four cells below, then the four above
        const int dn = tid - W * H;
        const Vec4 l3 = sm.f[7][dn - W - 1], l2 = sm.f[6][dn - W], l1 = sm.f[5][dn - 1], l0 = sm.f[4][dn];
        const Vec4 c3 = sm.f[3][tid - W - 1], c2 = sm.f[2][tid - W], c1 = sm.f[1][tid - 1], c0 = sm.f[0][tid];
        const float F[3] = {(l3.x + l2.x + l1.x + l0.x) + c3.x + c2.x + c1.x + c0.x,
                            (l3.y + l2.y + l1.y + l0.y) + c3.y + c2.y + c1.y + c0.y,
                            (l3.z + l2.z + l1.z + l0.z) + c3.z + c2.z + c1.z + c0.z};
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const float vn = rfma(fscale, F[d], rmul(a.keep, vold[d]));
            a.v[3 * at + d] = vn;
            a.u_out[3 * at + d] = rfma(a.dt, vn, rmul(a.ukeep, (un[d] * 0.03125f) * 32.f));
        }
    }
}

// one launch form: kernel, threads, shared memory
struct Form {
    void (*kernel)(MpmArgs<float>);
    int threads;
    size_t smem;
};
template <int GT, int GROUPS, bool STAB, int PITCH>
Form march(size_t table) {
    return Form{k_mpm_step<GT, GROUPS, STAB, PITCH>, GT * GROUPS, GROUPS * sizeof(MarchSmem<GT>) + (STAB ? table : 0)};
}
template <int THREADS, bool STAB>
Form block(size_t table) {
    return Form{k_mpm_block<THREADS, STAB>, THREADS, sizeof(BlockSmem<THREADS>) + (STAB ? table : 0)};
}
Form form_of(int variant, int nq) {
    constexpr int T = MPM_THREADS, H = MPM_HALF_THREADS, S = MPM_SMALL_BLOCK;
    const size_t table = sizeof(float) * 12 * (size_t)nq;
    const bool st = nq <= MPM_STAB_MAX;
    const bool stb = nq <= MPM_STAB_BLOCK;   // a block stages the table only while it is small beside its loads
    switch (variant) {
        case 0: return st ? march<T, 1, true, 17>(table) : march<T, 1, false, 0>(0);
        case MPM_BLOCK: return stb ? block<T, true>(table) : block<T, false>(0);
        case MPM_BLOCK + 1: return stb ? block<S, true>(table) : block<S, false>(0);
        case MPM_QUAD: return st ? march<H, 4, true, 17>(table) : march<H, 4, false, 17>(0);
        case MPM_HALF + 1: return st ? march<H, 1, true, 17>(table) : march<H, 1, false, 0>(0);
        case MPM_HALF + 2: return st ? march<H, 1, true, 0>(table) : march<H, 1, false, 0>(0);
        default: return st ? march<T, 1, true, 0>(table) : march<T, 1, false, 0>(0);
    }
}

}  // namespace

// The limit of a kernel is the process's, so it is only ever set to the most that the kernel is launched with,
// each time to the same value: a launch of another thread's handle may come at any moment.
cudaError_t mpm_prepare() {
    for (int v = 0; v < mpm_nvariants(true); ++v) {
        const int most = mpm_is_block(v) ? MPM_STAB_BLOCK : MPM_STAB_MAX;   // orientations staged; beyond: none
        for (int nq : {most, MPM_STAB_MAX + 1}) {
            const Form f = form_of(v, nq);
            const cudaError_t e = cudaFuncSetAttribute(f.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)f.smem);
            if (e != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

template <>
int mpm_per_sm<float>(int variant, int nq) {
    const Form f = form_of(variant, nq);
    int n = 1;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, f.kernel, f.threads, f.smem);
    return mpm_groups(variant) * ((e != cudaSuccess || n < 1) ? 1 : n);
}

// launched with programmatic stream serialisation: the kernel waits for the grid before it
// (griddepcontrol.wait) only after its prologue
template <>
cudaError_t launch_mpm_step<float>(const MpmArgs<float> &a, int variant, cudaStream_t s) {
    const Form f = form_of(variant, a.nq);
    return launch_pdl(f.kernel, (unsigned)a.grid, (unsigned)f.threads, f.smem, s, a);
}

}  // namespace hmc
