// Grain count of one replica: grains are the face-connected sets of sites of
// one orientation on the periodic lattice (a grain's volume is the number of
// sites it holds, Sec. "Microstructural Evolution"; the mean grain volume is the
// site count over the grain count).  Union-find over the sites with labels in
// block-slot order (8 block + slot): every union hooks the larger root under the
// smaller one with one compare-and-swap, so a parent is always smaller than its
// child and the forest stays acyclic under any interleaving; finds halve paths
// (writing an ancestor is always a valid parent).  The count is the number of
// roots, independent of the order in which the unions ran.  Every loop is capped;
// a capped-out loop sets the error word instead of spinning.
#include <algorithm>

#include "hmc_device.cuh"

namespace hmc {

namespace {

constexpr int CC_CAP = 1 << 22;

__device__ __forceinline__ unsigned cc_load(const unsigned *p) { return *reinterpret_cast<const volatile unsigned *>(p); }

__device__ __forceinline__ unsigned cc_find(unsigned *parent, unsigned x, int *err) {
    for (int it = 0; it < CC_CAP; ++it) {
        const unsigned p = cc_load(parent + x);
        if (p == x) return x;
        const unsigned gp = cc_load(parent + p);
        if (gp != p) parent[x] = gp;
        x = gp;
    }
    *err = 1;
    return x;
}

__device__ __forceinline__ void cc_unite(unsigned *parent, unsigned a, unsigned b, int *err) {
    for (int it = 0; it < CC_CAP; ++it) {
        a = cc_find(parent, a, err);
        b = cc_find(parent, b, err);
        if (a == b) return;
        const unsigned lo = min(a, b), hi = max(a, b);
        if (atomicCAS(parent + hi, hi, lo) == hi) return;
    }
    *err = 1;
}

// Labels inside every 2x2x2 block (one thread each, no memory traffic but the result): a site's
// parent is the lowest slot of its orientation that it reaches within the block.
__global__ void k_cc_init(const uint4 *__restrict__ spins, long long nblk, unsigned *parent) {
    for (long long b = (long long)blockIdx.x * blockDim.x + threadIdx.x; b < nblk; b += (long long)gridDim.x * blockDim.x) {
        const uint4 me = __ldg(spins + b);
        unsigned lab[8];
#pragma unroll
        for (int s = 0; s < 8; ++s) lab[s] = s;
#pragma unroll
        for (int L = 0; L < 8; ++L)
#pragma unroll
            for (int bit = 1; bit < 8; bit <<= 1) {
                if (L & bit) continue;
                const int s = local_slot(L), t = local_slot(L | bit);
                if (spin_of(me, s) != spin_of(me, t)) continue;
                const unsigned lo = min(lab[s], lab[t]), hi = max(lab[s], lab[t]);
#pragma unroll
                for (int k = 0; k < 8; ++k) lab[k] = lab[k] == hi ? lo : lab[k];
            }
        uint4 *out = reinterpret_cast<uint4 *>(parent + 8 * b);
        const unsigned o = (unsigned)(8 * b);
        out[0] = make_uint4(o + lab[0], o + lab[1], o + lab[2], o + lab[3]);
        out[1] = make_uint4(o + lab[4], o + lab[5], o + lab[6], o + lab[7]);
    }
}

// Unions across the +x, +y and +z face of every block, one thread per block and axis.  Of the face's
// four pairs, one whose neighbour pair in the face has the same orientation is already connected
// through it (inside both blocks), so a face within a grain takes one union.  The unions of a thread
// are a chain of dependent memory accesses: 24 per thread, as every site was joined to its three
// neighbours, took 83 us on 60^3 sites and 1.0 ms on 256^3.
__global__ void k_cc_union(const uint4 *__restrict__ spins, int nbx, int nby, int nbz, unsigned *parent, int *err) {
    const long long nblk = (long long)nbx * nby * nbz;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < 3 * nblk; i += (long long)gridDim.x * blockDim.x) {
        const int axis = (int)(i / nblk), bit = 1 << axis;
        const long long b = i - axis * nblk;
        const int bx = (int)(b % nbx);
        const long long r = b / nbx;
        const int by = (int)(r % nby), bz = (int)(r / nby);
        const long long next = axis == 0   ? b + (bx == nbx - 1 ? 1 - nbx : 1)
                               : axis == 1 ? b + (by == nby - 1 ? -(long long)(nby - 1) * nbx : nbx)
                                           : b + (bz == nbz - 1 ? -(long long)(nbz - 1) * nbx * nby : (long long)nbx * nby);
        const uint16_t *me = reinterpret_cast<const uint16_t *>(spins + b);   // slot s of a block at s
        const uint16_t *to = reinterpret_cast<const uint16_t *>(spins + next);
        int q[4];   // orientation of a matching pair, -1 for the others
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            // corner of this block on the face: the two bits of p in the other two axes
            const int low = p & (bit - 1), L = low | bit | (p & ~(bit - 1)) << 1;
            const int s = local_slot(L), t = local_slot(L ^ bit);
            q[p] = __ldg(me + s) == __ldg(to + t) ? (int)__ldg(me + s) : -1;
            const bool known = (p & 1 && q[p ^ 1] == q[p]) || (p & 2 && q[p ^ 2] == q[p]);
            if (q[p] >= 0 && !known) cc_unite(parent, (unsigned)(8 * b + s), (unsigned)(8 * next + t), err);
        }
    }
}

__global__ void k_cc_roots(const unsigned *parent, long long n, unsigned long long *count) {
    unsigned long long c = 0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        c += parent[i] == (unsigned)i;
    for (int off = 16; off; off >>= 1) c += __shfl_down_sync(0xffffffffu, c, off);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(count, c);
}

}  // namespace

cudaError_t launch_grain_count(const uint4 *spins, int nbx, int nby, int nbz, unsigned *parent,
                               unsigned long long *count, int *err, cudaStream_t s) {
    const long long nblk = (long long)nbx * nby * nbz, n = 8 * nblk;
    const int g0 = (int)std::min<long long>((nblk + 255) / 256, 65536), g1 = (int)std::min<long long>((n + 255) / 256, 8192);
    const int g2 = (int)std::min<long long>((3 * nblk + 127) / 128, 131072);
    cudaError_t e;
    if ((e = cudaMemsetAsync(count, 0, sizeof(unsigned long long), s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(err, 0, sizeof(int), s)) != cudaSuccess) return e;
    k_cc_init<<<g0, 256, 0, s>>>(spins, nblk, parent);
    k_cc_union<<<g2, 128, 0, s>>>(spins, nbx, nby, nbz, parent, err);
    k_cc_roots<<<g1, 256, 0, s>>>(parent, n, count);
    return cudaGetLastError();
}

}  // namespace hmc
