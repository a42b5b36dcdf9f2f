// Largest-droplet measurement (Sec. 3): cluster labelling of every walker's
// configuration on the device.
//
// A droplet is a set of occupied sites connected through nearest-neighbour
// bonds of the periodic lattice.  One block labels one walker at a time
// (grid-stride over the walkers of a system) with a concurrent union-find:
// roots are linked larger index -> smaller index by compare-and-swap, so every
// parent pointer points to a smaller index and the pointer chains cannot form
// cycles; finds halve their paths.  V_D is the largest number of particles
// with one root; thread 0 stores it and adds (1, V_D, V_D^2) to the system's
// accumulators at the walker's energy bin.
//
// droplet_rank_kernel (where its tables fit into shared memory) numbers the
// particles by the rank of their site's bit in the occupation bitset, so its
// tables have one entry per particle:
//   1. the bitset goes to shared memory and its words' popcounts are summed;
//   2. every particle's site, and as its parent the particle on the site
//      before it in its row, if there is one: the bonds along the rows are
//      united without any search;
//   3. the bonds along the other axes, and those around the rows' ends, are
//      united by compare-and-swap; a neighbour's rank is a table word and a
//      popcount.  Of two rows that run on beside each other only the first
//      bond is taken;
//   4. every particle adds one to its root's counter (read-only finds), and
//      the counters' maximum is V_D.
// What bounds it: the latency of the searches and of the block barriers, so
// the blocks that share an SM decide.  One parent word per lattice site (the
// other kernel) is 128 KB on 3D L = 32, one block per SM; the tables here are
// 26 KB.  8192 walkers of 3D L = 32, N = 3277: 1531 -> 527 us; 4096
// walkers of 2D L = 64, N = 410: 33 -> 28 us.
//
// droplet_kernel (dense or large lattices) keeps one parent word per lattice
// site, in shared memory when 4 V bytes fit into one block, else in a global
// scratch slice per block (at most 512 MiB for all blocks):
//   1. parent[s] = s for every particle site s;
//   2. every occupied forward neighbour is united;
//   3. parent[s] = root(s) for every particle (full compression; these
//      finds only read, so that no stale ancestor overwrites a root);
//   4. each root's entry becomes a counter, marked by the top bit, and every
//      particle adds one to the counter of its root.
//
// Every compare-and-swap loop has an iteration limit; hitting it (which a
// correct run never does: every failed swap means another thread linked a
// root) sets an error flag that the host reads.

#include <cstdint>

#include "mucal_internal.h"

namespace mucal {
namespace {

constexpr int kDropThreads = 256;
constexpr uint32_t kRootMark = 0x80000000u;
constexpr int kUniteLimit = 1 << 22;
constexpr size_t kDropScratchBytes = size_t(512) << 20;

__device__ __forceinline__ uint32_t particle_site(const SysParams &p, int w, int i)
{
    if (p.idx16) return static_cast<const uint16_t *>(p.S)[(size_t)w * p.V + i];
    return static_cast<const uint32_t *>(p.S)[(size_t)w * p.V + i];
}

// Forward neighbour of site s along axis k (periodic).
__device__ __forceinline__ uint32_t forward(const SysParams &p, uint32_t s, int k)
{
    const uint32_t L = (uint32_t)p.L;
    if (k == 0) return (s % L == L - 1) ? s + 1 - L : s + 1;
    if (k == 1) return ((s / L) % L == L - 1) ? s + L - (uint32_t)p.L2 : s + L;
    const uint32_t L2 = (uint32_t)p.L2;
    return (s / L2 == L - 1) ? s + L2 - (uint32_t)p.V : s + L2;
}

__device__ __forceinline__ uint32_t find_root(volatile uint32_t *P, uint32_t x)
{
    uint32_t px = P[x];
    while (px != x) {
        const uint32_t gp = P[px];
        if (gp != px) P[x] = gp;   // path halving: gp is still an ancestor of x
        x = px;
        px = gp;
    }
    return x;
}

// Root without writes.  The compression pass uses this: a path-halving write
// there could overwrite another thread's final "parent = root" with a mere
// ancestor, and the counting pass relies on every particle pointing at its root.
__device__ __forceinline__ uint32_t find_root_ro(volatile uint32_t *P, uint32_t x)
{
    uint32_t px = P[x];
    while (px != x) {
        x = px;
        px = P[x];
    }
    return x;
}

__device__ __forceinline__ bool unite(volatile uint32_t *P, uint32_t a, uint32_t b)
{
    for (int it = 0; it < kUniteLimit; ++it) {
        a = find_root(P, a);
        b = find_root(P, b);
        if (a == b) return true;
        if (a < b) {
            const uint32_t t = a;
            a = b;
            b = t;
        }
        const uint32_t old = atomicCAS(const_cast<uint32_t *>(P + a), a, b);
        if (old == a) return true;
        a = old;   // a was linked meanwhile: continue from its new parent
    }
    return false;
}

// Walker w's largest droplet into its slot and its energy's accumulators.
__device__ __forceinline__ void record(const SysParams &p, const DropletOut &o, int w, uint32_t size)
{
    o.last[w] = (int32_t)size;
    const int b = p.E[w] - p.e_lo;
    if (b >= 0 && b < p.n_bins) {
        atomicAdd(o.acc + b, 1ull);
        atomicAdd(o.acc + p.n_bins + b, (unsigned long long)size);
        atomicAdd(o.acc + 2 * (size_t)p.n_bins + b, (unsigned long long)size * size);
    } else {
        atomicExch(o.err, 2);
    }
}

template <bool SHARED>
__global__ void __launch_bounds__(kDropThreads)
droplet_kernel(SysParams p, DropletOut o, uint32_t *scratch)
{
    extern __shared__ uint32_t dyn_smem[];
    __shared__ uint32_t red[kDropThreads / 32];
    volatile uint32_t *P = SHARED ? dyn_smem : scratch + (size_t)blockIdx.x * (size_t)p.V;
    const int tid = threadIdx.x;
    bool ok = true;
    for (int w = blockIdx.x; w < p.n_walkers; w += gridDim.x) {
        const uint32_t *bits = p.bits + (size_t)w * p.words;
        for (int i = tid; i < p.N; i += kDropThreads) {
            const uint32_t s = particle_site(p, w, i);
            P[s] = s;
        }
        __syncthreads();
        for (int i = tid; i < p.N; i += kDropThreads) {
            const uint32_t s = particle_site(p, w, i);
            for (int k = 0; k < p.d; ++k) {
                const uint32_t t = forward(p, s, k);
                if ((bits[t >> 5] >> (t & 31u)) & 1u) ok &= unite(P, s, t);
            }
        }
        __syncthreads();
        for (int i = tid; i < p.N; i += kDropThreads) {
            const uint32_t s = particle_site(p, w, i);
            P[s] = find_root_ro(P, s);
        }
        __syncthreads();
        for (int i = tid; i < p.N; i += kDropThreads) {
            const uint32_t s = particle_site(p, w, i);
            if (P[s] == s) P[s] = kRootMark;
        }
        __syncthreads();
        for (int i = tid; i < p.N; i += kDropThreads) {
            const uint32_t s = particle_site(p, w, i);
            const uint32_t v = P[s];
            const uint32_t r = (v & kRootMark) ? s : v;
            atomicAdd(const_cast<uint32_t *>(P + r), 1u);
        }
        __syncthreads();
        uint32_t m = 0;
        for (int i = tid; i < p.N; i += kDropThreads) {
            const uint32_t v = P[particle_site(p, w, i)];
            if (v & kRootMark) m = max(m, v & ~kRootMark);
        }
        for (int off = 16; off > 0; off >>= 1) m = max(m, __shfl_xor_sync(0xFFFFFFFFu, m, off));
        if ((tid & 31) == 0) red[tid >> 5] = m;
        __syncthreads();
        if (tid == 0) {
            uint32_t D = 0;
            for (int j = 0; j < kDropThreads / 32; ++j) D = max(D, red[j]);
            record(p, o, w, D);
        }
        __syncthreads();   // P and red are reused by the next walker
    }
    if (!ok) atomicExch(o.err, 1);
}

// Shared memory of droplet_rank_kernel: bitset, parents (uint32 per particle),
// sites and later counters (IdxT per particle), ranks of the words (IdxT).
__host__ __device__ __forceinline__ size_t rank_smem(const SysParams &p)
{
    const size_t ib = p.idx16 ? 2 : 4;
    const size_t words = (size_t)p.words, n = (size_t)p.N;
    return 4 * words + 4 * n + (((ib * n) + 3) & ~(size_t)3) + ib * words;
}

template <int D, typename IdxT>
__global__ void __launch_bounds__(kDropThreads, 6)
droplet_rank_kernel(SysParams p, DropletOut o)
{
    extern __shared__ __align__(16) uint32_t dyn_smem[];
    __shared__ uint32_t red[kDropThreads / 32];
    const int words = p.words, T = blockDim.x, tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5, warps = T >> 5;
    const uint32_t N = (uint32_t)p.N, L = (uint32_t)p.L, V = (uint32_t)p.V;
    uint32_t *bits = dyn_smem;
    volatile uint32_t *parent = bits + words;
    uint32_t *tail = bits + words + N;                 // sites, then counters
    IdxT *site = reinterpret_cast<IdxT *>(tail);
    IdxT *base = reinterpret_cast<IdxT *>(reinterpret_cast<char *>(tail) + ((sizeof(IdxT) * N + 3) & ~(size_t)3));
    auto occupied_at = [&](uint32_t t) { return (bits[t >> 5] >> (t & 31u)) & 1u; };
    auto rank_of = [&](uint32_t t) {
        return (uint32_t)base[t >> 5] + (uint32_t)__popc(bits[t >> 5] & ((1u << (t & 31u)) - 1u));
    };
    const int chunk = (words + T - 1) / T;
    bool ok = true;
    for (int w = blockIdx.x; w < p.n_walkers; w += gridDim.x) {
        const uint32_t *src = p.bits + (size_t)w * words;
        for (int i = tid; i < words; i += T) bits[i] = src[i];
        __syncthreads();
        // ranks of this thread's words, then its particles' sites and parents
        const int c0 = min(tid * chunk, words), c1 = min(c0 + chunk, words);
        uint32_t sum = 0;
        for (int i = c0; i < c1; ++i) sum += (uint32_t)__popc(bits[i]);
        uint32_t incl = sum;
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, off);
            if (lane >= off) incl += y;
        }
        if (lane == 31) red[warp] = incl;
        __syncthreads();
        uint32_t r = incl - sum, n = 0;
        for (int i = 0; i < warps; ++i) {
            r += i < warp ? red[i] : 0u;
            n += red[i];
        }
        n = min(n, N);     // particles with tables: N, or fewer bits of a bitset that lacks some
        for (int i = c0; i < c1; ++i) {
            const uint32_t word = bits[i];
            base[i] = (IdxT)r;
            // bit b set if the site before site 32 i + b (in any row) is occupied
            const uint32_t left = (word << 1) | (i > 0 ? bits[i - 1] >> 31 : 0u);
            for (uint32_t x = word; x; x &= x - 1u, ++r) {
                const uint32_t b = (uint32_t)__ffs(x) - 1u, s = 32u * (uint32_t)i + b;
                const bool row_start = s - __umulhi(s, p.magL) * L == 0u;
                if (r < n) {
                    site[r] = (IdxT)s;
                    parent[r] = ((left >> b) & 1u) && !row_start ? r - 1u : r;
                }
            }
        }
        __syncthreads();
        for (uint32_t i = tid; i < n; i += T) {
            const uint32_t s = site[i];
            const uint32_t q = __umulhi(s, p.magL), x = s - q * L;
            uint32_t t[D];
            bool bond[D];
            t[0] = s - (L - 1u);                         // around the row's end
            if constexpr (D == 2) {
                t[1] = s >= V - L ? s - (V - L) : s + L;
            } else {
                const uint32_t L2 = (uint32_t)p.L2;
                const uint32_t y = q - __umulhi(q, p.magL) * L;
                t[1] = y == L - 1u ? s - (L2 - L) : s + L;
                t[2] = s >= V - L2 ? s - (V - L2) : s + L2;
            }
            bond[0] = x == L - 1u && occupied_at(t[0]);
            // (a pair of rows is united once where both have a run on: the
            // sites before these two, if occupied, are bonded too)
            const bool left = x != 0u && occupied_at(s - 1u);
#pragma unroll
            for (int k = 1; k < D; ++k) bond[k] = occupied_at(t[k]) && !(left && occupied_at(t[k] - 1u));
#pragma unroll
            for (int k = 0; k < D; ++k)
                if (bond[k]) {
                    const uint32_t rt = rank_of(t[k]);
                    if (rt < n) ok &= unite(parent, i, rt);
                }
        }
        __syncthreads();
        // the sites' words become counters
        const uint32_t tail_words = (uint32_t)((sizeof(IdxT) * N + 3) / 4);
        for (uint32_t i = tid; i < tail_words; i += T) tail[i] = 0u;
        __syncthreads();
        for (uint32_t i = tid; i < n; i += T) {
            const uint32_t root = find_root_ro(parent, i);
            // (two 16-bit counters per word; a count is below 65536)
            if constexpr (sizeof(IdxT) == 2) atomicAdd(tail + (root >> 1), 1u << ((root & 1u) << 4));
            else atomicAdd(tail + root, 1u);
        }
        __syncthreads();
        uint32_t m = 0;
        for (uint32_t i = tid; i < tail_words; i += T) {
            if constexpr (sizeof(IdxT) == 2) m = max(m, max(tail[i] & 0xFFFFu, tail[i] >> 16));
            else m = max(m, tail[i]);
        }
        m = __reduce_max_sync(0xFFFFFFFFu, m);
        if (lane == 0) red[warp] = m;
        __syncthreads();
        if (tid == 0) {
            uint32_t size = 0;
            for (int j = 0; j < warps; ++j) size = max(size, red[j]);
            record(p, o, w, size);
        }
        __syncthreads();   // the tables and red are reused by the next walker
    }
    if (!ok) atomicExch(o.err, 1);
}

template <int D, typename IdxT>
cudaError_t rank_plan(const SysParams &p, int sms, int optin, DropletPlan *plan)
{
    cudaFuncAttributes attr{};
    cudaError_t e = cudaFuncGetAttributes(&attr, droplet_rank_kernel<D, IdxT>);
    if (e != cudaSuccess) return e;
    const size_t need = rank_smem(p);
    if (need + attr.sharedSizeBytes > (size_t)optin) return cudaSuccess;
    // two to eight words of the bitset per thread: wide enough to share the
    // searches, small enough that blocks overlap each other's barriers
    plan->threads = p.words >= 512 ? 256 : (p.words >= 128 ? 128 : 64);
    plan->smem = need;
    e = cudaFuncSetAttribute(droplet_rank_kernel<D, IdxT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             optin - (int)attr.sharedSizeBytes);
    int per_sm = 0;
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, droplet_rank_kernel<D, IdxT>, plan->threads,
                                                          need);
    if (e != cudaSuccess) return e;
    const long long blocks = (long long)sms * (per_sm > 0 ? per_sm : 1);
    plan->grid = (int)(p.n_walkers < blocks ? p.n_walkers : blocks);
    plan->rank = true;
    return cudaSuccess;
}

}  // namespace

cudaError_t droplet_plan(const SysParams &p, DropletPlan *plan)
{
    int dev = 0, sms = 0, optin = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    *plan = DropletPlan{};
    if (p.d == 2)
        e = p.idx16 ? rank_plan<2, uint16_t>(p, sms, optin, plan) : rank_plan<2, uint32_t>(p, sms, optin, plan);
    else
        e = p.idx16 ? rank_plan<3, uint16_t>(p, sms, optin, plan) : rank_plan<3, uint32_t>(p, sms, optin, plan);
    if (e != cudaSuccess || plan->rank) return e;
    const size_t need = (size_t)p.V * sizeof(uint32_t);
    const size_t static_bytes = (kDropThreads / 32) * sizeof(uint32_t);
    plan->shared = need + static_bytes <= (size_t)optin;
    if (plan->shared) {
        plan->smem = need;
        // (as much as there is, not this lattice's need: plans of other lattices are kept)
        e = cudaFuncSetAttribute(droplet_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 optin - (int)static_bytes);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, droplet_kernel<true>,
                                                              kDropThreads, need);
        if (e != cudaSuccess) return e;
        plan->scratch_words = 0;
    } else {
        plan->smem = 0;
        per_sm = 2;
    }
    if (per_sm < 1) per_sm = 1;
    long long blocks = (long long)sms * per_sm;
    if (!plan->shared) {
        // global parent arrays: at most kDropScratchBytes in total
        const long long fit = (long long)(kDropScratchBytes / need);
        blocks = fit < 1 ? 1 : (fit < blocks ? fit : blocks);
    }
    plan->grid = (int)(p.n_walkers < blocks ? p.n_walkers : blocks);
    if (plan->grid < 1) plan->grid = 1;
    if (!plan->shared) plan->scratch_words = (size_t)plan->grid * (size_t)p.V;
    return cudaSuccess;
}

cudaError_t launch_droplets(const SysParams &p, const DropletOut &o, const DropletPlan &plan,
                            uint32_t *scratch, cudaStream_t stream)
{
    if (plan.rank) {
        if (p.d == 2 && p.idx16)
            droplet_rank_kernel<2, uint16_t><<<plan.grid, plan.threads, plan.smem, stream>>>(p, o);
        else if (p.d == 2)
            droplet_rank_kernel<2, uint32_t><<<plan.grid, plan.threads, plan.smem, stream>>>(p, o);
        else if (p.idx16)
            droplet_rank_kernel<3, uint16_t><<<plan.grid, plan.threads, plan.smem, stream>>>(p, o);
        else
            droplet_rank_kernel<3, uint32_t><<<plan.grid, plan.threads, plan.smem, stream>>>(p, o);
    } else if (plan.shared)
        droplet_kernel<true><<<plan.grid, kDropThreads, plan.smem, stream>>>(p, o, nullptr);
    else
        droplet_kernel<false><<<plan.grid, kDropThreads, 0, stream>>>(p, o, scratch);
    return cudaGetLastError();
}

}  // namespace mucal
