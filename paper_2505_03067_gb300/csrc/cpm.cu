// cpm.cu -- the growth driver coupled to the fields: tumour growth into the
// pleural space and mitosis on the device (the CPM and its Steppables of
// Sec. 2.1 / 2.4; the paper gives no Hamiltonian, so this is one simple
// rule, stated in the C header).
//
// Five launches per step (four on a small lattice), all stream-ordered, no host round trip.  The lattice
// is read once: one bit per voxel (tumour or not) stands in for it afterwards,
// so that only the words of the tumour and of its front are touched again.
//   k_cpm_scan     lattice -> tumour bits; per-cell volume and coordinate sums
//                  (exact integer atomics, aggregated over the lanes of a warp
//                  that hold one id);
//   k_cpm_front    the medium voxels of the mask next to a tumour cell;
//   k_cpm_grow     each of them is taken over with p = p_grow * c_O/(K_O+c_O) * c_n/(K_n+c_n)
//                  (0 below o2_min) by one of its tumour neighbours, in place;
//   k_cpm_plan     one CTA: cells of at least v_div voxels get daughter ids in
//                  increasing id order while the rate tables have room, an
//                  axis each, and their parent's rates;
//   k_cpm_apply    voxels strictly above the parent's centroid along its axis
//                  move to the daughter (tumour words only; nothing to do when
//                  no cell divides).
// The growth is synchronous (every voxel reads the lattice as it was) although
// it writes in place: whether a neighbour is tumour is read from the bits of
// the old lattice, an id is read only at a voxel whose bit is set, and growth
// writes only voxels whose bit is clear, each by the thread that decides it.
// On the 512x384x384 lattice (75 M voxels, 302 MB of ids): a step took 917 us
// with a full-lattice pass per launch (grow 495, stats 196, plan 28, apply
// 149 us) and takes 152 us now (scan 63, front 27, grow 9, plan 13, apply 3, or
// 21 us when cells divide), against 56 us for one reading of ids and mask.
// Small lattices (kSmallWords) are a chain of short launches, each as long as
// its slowest warp's loads: there the scan gives a warp one word at a time, and
// the front kernel takes 32 words a CTA and decides the growth itself.  A step
// on 64^3 takes 28 us so and 32 us in the other form (27 us with a full-lattice
// pass per launch), on 128^3 29 against 33, on 192^3 48 against 41; around 160^3
// it depends on the tumour's surface (37 against 39, 42 against 39.5).
// Randomness: SplitMix64's output function on a counter (seed, step, stream,
// index), so the decisions do not depend on the launch shape.
#include <cmath>
#include <cstring>

#include "mpm_internal.cuh"

namespace mpm {

constexpr uint64_t kGamma = 0x9E3779B97F4A7C15ull;
constexpr int kPlanThreads = 1024;

__device__ __forceinline__ uint64_t splitmix_out(uint64_t z)
{
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__device__ __forceinline__ uint64_t cpm_draw(uint64_t seed, int64_t step, int stream, uint64_t idx)
{
    const uint64_t c = ((uint64_t)((4 * step + stream) & ((1 << 24) - 1)) << 40) | idx;
    return splitmix_out(seed + (c + 1ull) * kGamma);
}

constexpr uint32_t kSmallWords = 1u << 16;   // 2 M voxels: the line between the two forms

struct CpmArgs {
    int32_t *cell;               // lattice cell ids (in: before the step, out: after)
    uint32_t *bits, *grown;      // per voxel: id > 0 before growth; and after it
    uint32_t nwords;             // 32-voxel words of the lattice
    uint32_t *front, *nfront;    // medium voxels of the mask next to the tumour, and how many
    const uint8_t *mask;
    const double *o2, *nut;
    int32_t Lx, Ly, Lz;
    int64_t L;
    double p_grow, K_o2, K_nut, o2_min;
    int32_t v_div;
    int32_t cap;                 // rate-table entries per species
    int32_t nspecies;
    double *k_cell, *q_cell;     // [nspecies][cap]
    int32_t *ncell;              // ids in use (device)
    unsigned long long *vol, *sum;   // [cap], [3][cap]
    int32_t *daughter, *axis;    // [cap + 1] (daughter[cap]: the ids in use before the step),
                                 // [cap + 1] (axis[cap]: divisions of this step)
    unsigned long long *stats;   // grown, divisions, ids outside the tables
    uint64_t seed;
    int64_t step;
};

// Adds the voxels of the calling lanes (all holding valid ids; lane l's voxel is
// lattice index v) to their cells' volumes and coordinate sums.
__device__ __forceinline__ void cpm_count(const CpmArgs &A, unsigned lanes, int32_t id, uint32_t v)
{
    const uint32_t Lx = A.Lx, Ly = A.Ly;
    const uint32_t row = v / Lx, x = v - row * Lx, z = row / Ly, y = row - z * Ly;
    const unsigned peers = __match_any_sync(lanes, id);
    const unsigned n = __popc(peers);
    const unsigned sx = __reduce_add_sync(peers, x), sy = __reduce_add_sync(peers, y), sz = __reduce_add_sync(peers, z);
    if ((int)(threadIdx.x & 31) == __ffs(peers) - 1) {
        atomicAdd(A.vol + id, (unsigned long long)n);
        atomicAdd(A.sum + id, (unsigned long long)sx);
        atomicAdd(A.sum + A.cap + id, (unsigned long long)sy);
        atomicAdd(A.sum + 2 * (int64_t)A.cap + id, (unsigned long long)sz);
    }
}

// The same for 32 consecutive voxels of one lattice row, v0 the first: the sums
// follow from the bits of the lanes that hold one id.
__device__ __forceinline__ void cpm_count_row(const CpmArgs &A, unsigned lanes, int32_t id, uint32_t x0, uint32_t y,
                                              uint32_t z)
{
    const unsigned peers = __match_any_sync(lanes, id);
    if ((int)(threadIdx.x & 31) != __ffs(peers) - 1) return;
    const unsigned n = __popc(peers);
    const unsigned pos = __popc(peers & 0xaaaaaaaau) + 2 * __popc(peers & 0xccccccccu) +
                         4 * __popc(peers & 0xf0f0f0f0u) + 8 * __popc(peers & 0xff00ff00u) +
                         16 * __popc(peers & 0xffff0000u);
    atomicAdd(A.vol + id, (unsigned long long)n);
    atomicAdd(A.sum + id, (unsigned long long)n * x0 + pos);
    atomicAdd(A.sum + A.cap + id, (unsigned long long)n * y);
    atomicAdd(A.sum + 2 * (int64_t)A.cap + id, (unsigned long long)n * z);
}

// Bound by HBM: 4 bytes read and an eighth of a byte written per voxel.  A warp
// takes kScanWords (8; small lattices 1) consecutive words at a time, loads the next ones (coalesced
// 128-byte loads) before it works on these, keeps word k in lane k and stores
// them together; a word without any id is done after its vote.  63 us on the
// 512x384x384 lattice (4.8 TB/s); 81 us with 16 words a warp, no load ahead and
// the sums by warp reductions.
template <int kScanWords>
__global__ void __launch_bounds__(256, 6) k_cpm_scan(const __grid_constant__ CpmArgs A)
{
    const int lane = threadIdx.x & 31;
    const uint32_t nw = gridDim.x * (blockDim.x >> 5), L = (uint32_t)A.L;
    const uint32_t ngroups = (A.nwords + kScanWords - 1) / kScanWords;
    uint32_t grp = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    int32_t next[kScanWords];
    auto load = [&](uint32_t g) {
#pragma unroll
        for (int k = 0; k < kScanWords; ++k) {
            const uint32_t v = (g * kScanWords + k) * 32 + lane;
            next[k] = g < ngroups && v < L ? __ldcs(A.cell + v) : 0;
        }
    };
    load(grp);
    for (; grp < ngroups; grp += nw) {
        const uint32_t w0 = grp * kScanWords;
        int32_t id[kScanWords];
#pragma unroll
        for (int k = 0; k < kScanWords; ++k) id[k] = next[k];
        load(grp + nw);
        uint32_t mine = 0u;
#pragma unroll
        for (int k = 0; k < kScanWords; ++k) {
            if (!__any_sync(0xffffffffu, id[k] != 0)) continue;
            const unsigned tum = __ballot_sync(0xffffffffu, id[k] > 0);
            if (lane == k) mine = tum;
            const unsigned okm = __ballot_sync(0xffffffffu, id[k] > 0 && id[k] < A.cap);
            const unsigned badm = __ballot_sync(0xffffffffu, id[k] < 0 || id[k] >= A.cap);
            if (lane == 0 && badm) atomicAdd(A.stats + 2, (unsigned long long)__popc(badm));
            const uint32_t v0 = (w0 + k) * 32, row = v0 / A.Lx, x0 = v0 - row * A.Lx;
            if ((okm >> lane) & 1u) {
                if (x0 + 32 <= (uint32_t)A.Lx) {
                    const uint32_t z = row / A.Ly;
                    cpm_count_row(A, okm, id[k], x0, row - z * A.Ly, z);
                } else {
                    cpm_count(A, okm, id[k], v0 + lane);
                }
            }
        }
        if (lane < kScanWords && w0 + lane < A.nwords) A.bits[w0 + lane] = mine;
    }
}

// The 32 tumour bits from lattice index p on (p may lie outside the lattice).
__device__ __forceinline__ uint32_t cpm_bits(const CpmArgs &A, int64_t p)
{
    const int64_t w = p >> 5;
    const uint32_t lo = w >= 0 && w < A.nwords ? A.bits[w] : 0u;
    const uint32_t sh = (uint32_t)(p & 31);
    if (!sh) return lo;
    const uint32_t hi = w + 1 >= 0 && w + 1 < A.nwords ? A.bits[w + 1] : 0u;
    return __funnelshift_r(lo, hi, sh);
}

__device__ __forceinline__ bool cpm_tumour(const CpmArgs &A, uint32_t v) { return (A.bits[v >> 5] >> (v & 31)) & 1u; }

// The growth of front voxel v: the id that takes it over (written), or 0.
__device__ __forceinline__ int32_t cpm_take(const CpmArgs &A, uint32_t v)
{
    const uint32_t Lx = A.Lx, Ly = A.Ly, Lz = A.Lz, Lxy = Lx * Ly;
    const double c0 = A.o2[v], c1 = A.nut[v];
    const uint32_t row = v / Lx, x = v - row * Lx, z = row / Ly, y = row - z * Ly;
    uint32_t tm = 0;   // tumour neighbours -x, +x, -y, +y, -z, +z
    if (x > 0 && cpm_tumour(A, v - 1)) tm |= 1u;
    if (x + 1 < Lx && cpm_tumour(A, v + 1)) tm |= 2u;
    if (y > 0 && cpm_tumour(A, v - Lx)) tm |= 4u;
    if (y + 1 < Ly && cpm_tumour(A, v + Lx)) tm |= 8u;
    if (z > 0 && cpm_tumour(A, v - Lxy)) tm |= 16u;
    if (z + 1 < Lz && cpm_tumour(A, v + Lxy)) tm |= 32u;
    if (!tm || c0 < A.o2_min) return 0;
    // same operations, same order as the rule's statement (no contraction possible)
    const double p = A.p_grow * (c0 / (A.K_o2 + c0)) * (c1 / (A.K_nut + c1));
    const double u = (double)(cpm_draw(A.seed, A.step, 0, (uint64_t)v) >> 11) * 0x1.0p-53;
    if (!(u < p)) return 0;
    const uint64_t h = cpm_draw(A.seed, A.step, 1, (uint64_t)v) >> 32;
    const uint32_t j = (uint32_t)((h * (uint32_t)__popc(tm)) >> 32);
    uint32_t t = tm;   // the j-th tumour neighbour
    for (uint32_t r = 0; r < j; ++r) t &= t - 1;
    const uint32_t d = __ffs(t) - 1;
    const uint32_t o = d < 2 ? 1u : d < 4 ? Lx : Lxy;
    const int32_t out = A.cell[(d & 1) ? v + o : v - o];
    A.cell[v] = out;
    atomicOr(A.grown + (v >> 5), 1u << (v & 31));
    return out;
}

// Counts a warp's growth (out: what cpm_take gave, 0 at lanes without a voxel).
__device__ __forceinline__ void cpm_count_growth(const CpmArgs &A, int32_t out, uint32_t v)
{
    const int lane = threadIdx.x & 31;
    const unsigned g = __ballot_sync(0xffffffffu, out > 0);
    const unsigned okm = __ballot_sync(0xffffffffu, out > 0 && out < A.cap);
    if (lane == 0 && g) {
        atomicAdd(A.stats + 0, (unsigned long long)__popc(g));
        if (g != okm) atomicAdd(A.stats + 2, (unsigned long long)__popc(g & ~okm));
    }
    if ((okm >> lane) & 1u) cpm_count(A, okm, out, v);
}

// The medium voxels of the mask next to a tumour voxel, to a list.  A CTA takes
// kWords (256: 8192 voxels; small lattices 32) words: a thread dilates one word of the bits (six shifted
// words, all in L2), the voxels of the dilation that are no tumour go to a list
// in shared memory, and the CTA's threads look at the mask and the id of the
// list's voxels.  The dilation ignores the lattice's faces; k_cpm_grow looks at
// them.  Bound by latency, hence the small kernel with eight CTAs on an SM.
// kGrow: the growth is decided here as well, without the list.  That saves a
// launch; on the 512x384x384 lattice (two FP64 divisions a voxel, few lanes of a
// warp) it took 51 us against 27 + 9 us.
constexpr int kFrontThreads = 256;
template <int kWords, bool kGrow>
__global__ void __launch_bounds__(kFrontThreads, 8) k_cpm_front(const __grid_constant__ CpmArgs A)
{
    __shared__ uint16_t s_list[kWords * 32];
    __shared__ int s_n;
    const uint32_t Lx = A.Lx, Lxy = Lx * (uint32_t)A.Ly;
    const uint32_t w = blockIdx.x * kWords + threadIdx.x;
    const int64_t v0 = (int64_t)w * 32;
    uint32_t cand = 0u;
    if (threadIdx.x == 0) s_n = 0;
    if (threadIdx.x < kWords && w < A.nwords) {
        const uint32_t own = A.bits[w];
        cand = (cpm_bits(A, v0 - 1) | cpm_bits(A, v0 + 1) | cpm_bits(A, v0 - Lx) | cpm_bits(A, v0 + Lx) |
                cpm_bits(A, v0 - Lxy) | cpm_bits(A, v0 + Lxy)) & ~own;
        if (v0 + 32 > A.L) cand &= 0xffffffffu >> (32 - (int)(A.L - v0));
        A.grown[w] = own;
    }
    if (!__syncthreads_or(cand != 0u)) return;
    if (cand) {
        int at = atomicAdd(&s_n, __popc(cand));
        for (uint32_t c = cand; c; c &= c - 1) s_list[at++] = (uint16_t)(threadIdx.x * 32 + __ffs(c) - 1);
    }
    __syncthreads();
    const int n = s_n, lane = threadIdx.x & 31;
    for (int i0 = threadIdx.x & ~31; i0 < n; i0 += kFrontThreads) {   // warp-uniform: the vote is legal inside
        const int i = i0 + lane;
        const uint32_t v = blockIdx.x * (kWords * 32u) + (i < n ? s_list[i] : 0);
        const bool front = i < n && A.mask[v] != 0 && A.cell[v] == 0;
        if (kGrow) {
            cpm_count_growth(A, front ? cpm_take(A, v) : 0, v);
            continue;
        }
        const unsigned f = __ballot_sync(0xffffffffu, front);
        if (!f) continue;
        uint32_t at = 0;
        if (lane == 0) at = atomicAdd(A.nfront, (uint32_t)__popc(f));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (front) A.front[at + __popc(f & ((1u << lane) - 1u))] = v;
    }
}

// The growth of the listed voxels, spread evenly over the GPU.
__global__ void __launch_bounds__(256) k_cpm_grow(const __grid_constant__ CpmArgs A)
{
    const uint32_t n = *A.nfront, lane = threadIdx.x & 31;
    for (uint32_t i0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); i0 < n; i0 += gridDim.x * blockDim.x) {
        const uint32_t v = i0 + lane < n ? A.front[i0 + lane] : 0u;
        cpm_count_growth(A, i0 + lane < n ? cpm_take(A, v) : 0, v);
    }
}
// One CTA: daughters in increasing parent id order while the tables have room.
// Bound by the latency of its loads: a round takes kPlanRun ids per thread (ids
// 1024 apart, so that all accesses are coalesced, with all volumes in flight),
// one scan of the votes of its warps orders them, and the daughters' rates are
// copied afterwards, one thread per id.  13 us for 15 600 ids; 31 us with runs
// of consecutive ids per thread.
constexpr int kPlanRun = 8;
__global__ void __launch_bounds__(kPlanThreads) k_cpm_plan(const __grid_constant__ CpmArgs A)
{
    constexpr int kVotes = kPlanRun * kPlanThreads / 32;
    __shared__ int32_t s_vote[kVotes], s_total;
    const int nc0 = *A.ncell;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int n = max(0, min(nc0, A.cap));
    int64_t carry = nc0;                // the next daughter's id, were there room
    for (int64_t base = 0; base < n; base += kPlanThreads * kPlanRun) {
        unsigned long long vol[kPlanRun];
        unsigned votes[kPlanRun];
#pragma unroll
        for (int k = 0; k < kPlanRun; ++k) {
            const int64_t id = base + k * kPlanThreads + threadIdx.x;
            vol[k] = id < n ? A.vol[id] : 0ull;
        }
#pragma unroll
        for (int k = 0; k < kPlanRun; ++k) {
            const int64_t id = base + k * kPlanThreads + threadIdx.x;
            votes[k] = __ballot_sync(0xffffffffu, id >= 1 && id < n && vol[k] >= (unsigned long long)A.v_div);
            if (lane == 0) s_vote[k * (kPlanThreads / 32) + wid] = __popc(votes[k]);
        }
        __syncthreads();
        if (wid == 0) {                 // exclusive scan, eight votes a lane
            int32_t c[kVotes / 32], sum = 0;
#pragma unroll
            for (int i = 0; i < kVotes / 32; ++i) {
                c[i] = s_vote[lane * (kVotes / 32) + i];
                sum += c[i];
            }
            int32_t incl = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            int32_t at = incl - sum;
#pragma unroll
            for (int i = 0; i < kVotes / 32; ++i) {
                s_vote[lane * (kVotes / 32) + i] = at;
                at += c[i];
            }
            if (lane == 31) s_total = incl;
        }
        __syncthreads();
        const int32_t total = s_total;
#pragma unroll
        for (int k = 0; k < kPlanRun; ++k) {
            const int64_t id = base + k * kPlanThreads + threadIdx.x;
            if (id >= n) break;
            int32_t d = -1, ax = 0;
            if ((votes[k] >> lane) & 1u) {
                const int64_t next =
                    carry + s_vote[k * (kPlanThreads / 32) + wid] + __popc(votes[k] & ((1u << lane) - 1u));
                if (next < A.cap) {
                    d = (int32_t)next;
                    const uint64_t h = cpm_draw(A.seed, A.step, 2, (uint64_t)id) >> 32;
                    ax = (int32_t)((h * 3ull) >> 32);
                }
            }
            A.daughter[id] = d;
            A.axis[id] = ax;
        }
        carry += total;
        __syncthreads();
    }
    if (carry > nc0 && nc0 < A.cap) {   // daughters were assigned
        for (int id = threadIdx.x; id < n; id += kPlanThreads) {
            const int32_t d = A.daughter[id];
            if (d < 0) continue;
            double k[kMaxSpecies], q[kMaxSpecies];
#pragma unroll
            for (int s = 0; s < kMaxSpecies; ++s) {
                k[s] = s < A.nspecies ? A.k_cell[(int64_t)s * A.cap + id] : 0.0;
                q[s] = s < A.nspecies ? A.q_cell[(int64_t)s * A.cap + id] : 0.0;
            }
#pragma unroll
            for (int s = 0; s < kMaxSpecies; ++s) {
                if (s >= A.nspecies) break;
                A.k_cell[(int64_t)s * A.cap + d] = k[s];
                A.q_cell[(int64_t)s * A.cap + d] = q[s];
            }
        }
    }
    if (threadIdx.x == 0) {
        const int32_t end = n > 0 ? (int32_t)min((int64_t)A.cap, carry) : nc0;
        A.daughter[A.cap] = nc0;      // the ids the apply pass may meet
        A.axis[A.cap] = end - nc0;
        A.stats[1] += (unsigned long long)(int64_t)(end - nc0);
        *A.ncell = end;
    }
}

// A warp reads 32 words of the bits after growth and works through those that
// hold tumour voxels, kApplyWords at a time (an id and then its daughter: two
// dependent loads each); their ids are all that is read of the lattice.  The
// whole step went from 169 to 152 us with four words instead of one.
constexpr int kApplyWords = 4;
__global__ void __launch_bounds__(256) k_cpm_apply(const __grid_constant__ CpmArgs A)
{
    if (A.axis[A.cap] <= 0) return;
    const uint32_t Lx = A.Lx, Ly = A.Ly;
    const int32_t nc0 = A.daughter[A.cap];
    const int lane = threadIdx.x & 31;
    const uint32_t nw = gridDim.x * (blockDim.x >> 5), ngroups = (A.nwords + 31) / 32;
    for (uint32_t grp = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); grp < ngroups; grp += nw) {
        const uint32_t w = grp * 32 + lane;
        const uint32_t mine = w < A.nwords ? A.grown[w] : 0u;
        unsigned todo = __ballot_sync(0xffffffffu, mine != 0u);
        while (todo) {
            uint32_t v[kApplyWords];
            int32_t id[kApplyWords], d[kApplyWords];
#pragma unroll
            for (int i = 0; i < kApplyWords; ++i) {
                const int k = todo ? __ffs(todo) - 1 : 0;
                const uint32_t word = __shfl_sync(0xffffffffu, mine, k);
                v[i] = (grp * 32 + k) * 32 + lane;
                id[i] = todo && ((word >> lane) & 1u) ? A.cell[v[i]] : 0;
                todo &= todo - 1;   // 0 stays 0
            }
#pragma unroll
            for (int i = 0; i < kApplyWords; ++i)
                d[i] = id[i] > 0 && id[i] < nc0 && id[i] < A.cap ? A.daughter[id[i]] : -1;
#pragma unroll
            for (int i = 0; i < kApplyWords; ++i) {
                if (d[i] < 0) continue;
                const int a = A.axis[id[i]];
                const uint32_t row = v[i] / Lx, z = row / Ly;
                const uint64_t c = a == 0 ? v[i] - row * Lx : a == 1 ? row - z * Ly : z;
                if (c * A.vol[id[i]] > A.sum[(int64_t)a * A.cap + id[i]]) A.cell[v[i]] = d[i];
            }
        }
    }
}

}  // namespace mpm

using namespace mpm;

extern "C" mpm_status mpm_cpm_step(mpm_ctx *ctx, const mpm_lattice *lat, const mpm_params *prm,
                                   const mpm_cpm_params *cp, uint64_t seed, int64_t step, int32_t *ncell_dev,
                                   int64_t *stats_dev, void *stream)
{
    if (!ctx) return MPM_ERR_ARG;
    ctx->err.clear();
    if (!lat || !prm || !cp || !ncell_dev || !stats_dev) return mpm_fail(ctx, MPM_ERR_ARG, "cpm_step: null argument");
    if (!lat->cell_id || !lat->mask || prm->nspecies < 2 || !lat->field[0] || !lat->field[1])
        return mpm_fail(ctx, MPM_ERR_ARG, "cpm_step: needs cell ids, the mask and species 0 (O2) and 1 (nutrient)");
    if (!prm->k_cell || !prm->q_cell || prm->ncell < 1 || prm->nspecies > MPM_MAX_SPECIES)
        return mpm_fail(ctx, MPM_ERR_ARG, "cpm_step: rate tables missing");
    const int64_t L = (int64_t)lat->dims[0] * lat->dims[1] * lat->dims[2];
    if (lat->dims[0] < 1 || lat->dims[1] < 1 || lat->dims[2] < 1 || L >= ((int64_t)1 << 31))
        return mpm_fail(ctx, MPM_ERR_ARG, "cpm_step: lattice dims out of range");
    if (!(cp->p_grow >= 0.0) || !(cp->K_o2 >= 0.0) || !(cp->K_nut >= 0.0) || !std::isfinite(cp->o2_min) ||
        cp->v_div < 2 || step < 0)
        return mpm_fail(ctx, MPM_ERR_ARG, "cpm_step: bad growth parameters");
    cudaStream_t st = (cudaStream_t)stream;
    const int cap = prm->ncell;
    auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
    // a front voxel has a tumour neighbour, and a tumour voxel at most six of them: at most 6 L / 7.
    // Bits, front and its count lie close together (the bits on 128-byte boundaries
    // where there is room): for every L they take no more than 4 L bytes rounded up
    // to 256, which small contexts are made for.
    const size_t nwords = (size_t)((L + 31) / 32), nfront = (size_t)(L - L / 7);
    const size_t bits = L < 4096 ? nwords : (nwords + 31) & ~(size_t)31;
    const size_t b_lat = al((2 * bits + nfront + 1) * 4), b_vol = al((size_t)cap * 8), b_sum = al((size_t)cap * 24),
                 b_i = al((size_t)(cap + 1) * 4);
    mpm_status r = mpm_grow(ctx, (void **)&ctx->d_cpm, &ctx->cpm_cap, b_lat + b_vol + b_sum + 2 * b_i,
                            "growth driver scratch");
    if (r != MPM_OK) return r;
    char *p = (char *)ctx->d_cpm;
    CpmArgs A;
    memset(&A, 0, sizeof(A));
    A.cell = const_cast<int32_t *>(lat->cell_id);   // updated in place (documented)
    A.bits = (uint32_t *)p;
    A.grown = A.bits + bits;
    A.nwords = (uint32_t)nwords;
    A.front = A.grown + bits;
    p += b_lat;
    A.nfront = (uint32_t *)p - 1;   // just before the sums: zeroed with them
    A.vol = (unsigned long long *)p;
    A.sum = (unsigned long long *)(p + b_vol);
    A.daughter = (int32_t *)(p + b_vol + b_sum);
    A.axis = (int32_t *)(p + b_vol + b_sum + b_i);
    A.mask = lat->mask;
    A.o2 = lat->field[0];
    A.nut = lat->field[1];
    A.Lx = lat->dims[0];
    A.Ly = lat->dims[1];
    A.Lz = lat->dims[2];
    A.L = L;
    A.p_grow = cp->p_grow;
    A.K_o2 = cp->K_o2;
    A.K_nut = cp->K_nut;
    A.o2_min = cp->o2_min;
    A.v_div = cp->v_div;
    A.cap = cap;
    A.nspecies = prm->nspecies;
    A.k_cell = const_cast<double *>(prm->k_cell);
    A.q_cell = const_cast<double *>(prm->q_cell);
    A.ncell = ncell_dev;
    A.stats = (unsigned long long *)stats_dev;
    A.seed = seed;
    A.step = step;
    // from a 256-byte boundary on (an unaligned fill cost 1 us): what lies there before the count is written later
    MPM_CU(cudaMemsetAsync(p - 256, 0, 256 + b_vol + b_sum, st));
    const bool small = A.nwords <= kSmallWords;
    if (small) {
        k_cpm_scan<1><<<ctx->num_sms * 6, 256, 0, st>>>(A);
        k_cpm_front<32, true><<<(A.nwords + 31) / 32, kFrontThreads, 0, st>>>(A);
    } else {
        k_cpm_scan<8><<<ctx->num_sms * 6, 256, 0, st>>>(A);
        k_cpm_front<256, false><<<(A.nwords + 255) / 256, kFrontThreads, 0, st>>>(A);
        k_cpm_grow<<<ctx->num_sms * 4, 256, 0, st>>>(A);
    }
    k_cpm_plan<<<1, kPlanThreads, 0, st>>>(A);
    k_cpm_apply<<<ctx->num_sms * 8, 256, 0, st>>>(A);
    ctx->launches += small ? 4 : 5;
    return mpm_cuda_check(ctx, cudaGetLastError(), "cpm_step");
}
