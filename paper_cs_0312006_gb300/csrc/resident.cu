// resident.cu -- many sweeps of one small lattice in one launch, its spins in
// the shared memory of a thread-block cluster.
//
// A pass of a lattice of up to a few hundred thousand sites takes less than its
// launch (1.6 us of host time, ~2 us from one dependent pass to the next), so n
// sweeps run as one launch: the cluster's CTAs each hold a slab of units (2D:
// half rows; 3D: planes of half rows) of both colours as int8 spins, with a copy
// of the unit before and behind (halo).  A pass updates its colour from local
// shared memory only; the words of a slab's first and last unit are also stored
// into the neighbours' halos (distributed shared memory), and the passes are
// separated by the cluster barrier (one CTA: __syncthreads).  A thread's first
// draws of the next pass are made between arriving at that barrier and waiting
// at it: what is left behind the barrier is the neighbour sum and the store.
//
// Rows are kept in whole words (four sites, one Philox call) at a fixed pitch,
// with the row's last site once more before its first byte and its first behind
// its last, so that no word needs a wrap in x.  Rows that start inside a Philox
// group (W % 4 != 0) test the group that holds their word's first draw, take the
// rest from the next lane's and shift by bytes (as packed_draws does with bits).
//
// Same rule, draws and results as the pass kernels.  E and M are summed per
// warp and added to the sweep's record by one reduction each, which nothing
// waits for.
#include <cooperative_groups.h>

#include <cstdint>

#include "engine_internal.h"
#include "ising_device.cuh"
#include "pass_bodies.cuh"

namespace cg = cooperative_groups;

namespace ising {

namespace {

struct ResidentArgs {
    PassArgs a;              // own / other: the colour arrays 0 / 1; t: the first sweep
    unsigned long long* obs; // the records' zeroed slots
    int nsweeps, every;
    uint32_t words;          // words per half row
    uint32_t pitch;          // words of shared memory per half row
    FastDiv by_words, by_L;
};

// Unit u of rank's slab lies at [first_unit(rank), first_unit(rank + 1)).
__host__ __device__ __forceinline__ uint32_t first_unit(uint32_t rank, uint32_t L,
                                                        uint32_t ranks) {
    return rank * L / ranks;
}

// Four spins of half row r from half column 4 q on, as bytes +1 / -1 (past the
// row's end: anything).
template <int LAYOUT>
__device__ __forceinline__ uint32_t spins_in(const void* col, uint32_t r, uint32_t q, uint32_t W) {
    if constexpr (LAYOUT == ISING_BITPACK) {
        const uint32_t nq = (W + 31u) >> 5;
        const uint32_t w = static_cast<const uint32_t*>(col)[r * nq + (q >> 3)];
        const uint32_t four = (w >> (4u * (q & 7u))) & 0xFu;
        return 0xFFFFFFFFu - 0xFEu * ((four * 0x00204081u) & kByteOnes);
    } else {
        const uint8_t* p = static_cast<const uint8_t*>(col) + (size_t)r * W + 4u * q;
        if ((W & 3u) == 0u) return *reinterpret_cast<const uint32_t*>(p);
        uint32_t v = 0u;
        for (uint32_t j = 0; j < 4u && 4u * q + j < W; ++j) v |= (uint32_t)p[j] << (8u * j);
        return v;
    }
}

// One word (index q of a row; `at` points to it) into shared memory, with the
// copies beyond the row's ends: the row's first site once more at byte W, its
// last at byte -1.  In a ragged row the copy of the first site shares the last
// word, so that one is stored by bytes.
template <bool RAGGED>
__device__ __forceinline__ void put_word(uint32_t* at, uint32_t q, uint32_t words, uint32_t W,
                                         uint32_t v) {
    uint8_t* bytes = reinterpret_cast<uint8_t*>(at - q);
    const bool last = q + 1u == words;
    const uint32_t n = RAGGED && last ? W - 4u * q : 4u;  // the word's sites
    if (!RAGGED || n == 4u) {
        *at = v;
    } else {
        bytes[4u * q] = (uint8_t)v;
        if (n > 1u) bytes[4u * q + 1u] = (uint8_t)(v >> 8);
        if (n > 2u) bytes[4u * q + 2u] = (uint8_t)(v >> 16);
    }
    if (q == 0u) bytes[W] = (uint8_t)v;
    if (last) bytes[-1] = (uint8_t)(v >> (8u * (n - 1u)));
}

template <int DIMS, int RULE, int LAYOUT, bool RAGGED>
__global__ void __launch_bounds__(512) resident_kernel(ResidentArgs k) {
    extern __shared__ uint32_t smem[];
    cg::cluster_group cl = cg::this_cluster();
    const uint32_t ranks = cl.num_blocks(), rank = cl.block_rank();
    const uint32_t L = (uint32_t)k.a.L, W = (uint32_t)k.a.W, words = k.words, P = k.pitch;
    const uint32_t unit_rows = DIMS == 3 ? L : 1u;
    const uint32_t u0 = first_unit(rank, L, ranks), u1 = first_unit(rank + 1u, L, ranks);
    const uint32_t rows = (u1 - u0) * unit_rows;           // own half rows
    const uint32_t all_rows = rows + 2u * unit_rows;       // with the halos
    const uint32_t row0 = u0 * unit_rows;                  // the first own row in the lattice
    const uint32_t lattice_rows = L * unit_rows;
    uint32_t* const S0 = smem;                             // colour 0, then colour 1
    // the neighbours' slabs: the unit before goes to the end of theirs
    const uint32_t before = rank == 0u ? ranks - 1u : rank - 1u;
    const uint32_t behind = rank + 1u == ranks ? 0u : rank + 1u;
    const uint32_t before_units =
        first_unit(before + 1u, L, ranks) - first_unit(before, L, ranks);
    const uint32_t behind_units =
        first_unit(behind + 1u, L, ranks) - first_unit(behind, L, ranks);
    uint32_t* const before_smem = cl.map_shared_rank(smem, before);
    uint32_t* const behind_smem = cl.map_shared_rank(smem, behind);

    // the slab and its halos
    for (uint32_t i = threadIdx.x; i < 2u * all_rows * words; i += blockDim.x) {
        const uint32_t row = k.by_words.quot(i), q = i - row * words;
        const uint32_t c = row >= all_rows ? 1u : 0u, lr = row - c * all_rows;
        uint32_t r = row0 + lattice_rows - unit_rows + lr;
        r -= r >= lattice_rows ? lattice_rows : 0u;
        r -= r >= lattice_rows ? lattice_rows : 0u;
        put_word<RAGGED>(S0 + row * P + 1u + q, q, words, W,
                         spins_in<LAYOUT>(c == 0u ? k.a.own : k.a.other, r, q, W));
    }

    constexpr uint32_t step = RAGGED ? 31u : 32u;
    const uint32_t items = rows * words;
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t stride = (blockDim.x >> 5) * step;
    const uint32_t first0 = (threadIdx.x >> 5) * step;
    // the stride of a thread's items in rows and words
    const uint32_t stride_rows = k.by_words.quot(stride), stride_words = stride - stride_rows * words;
    struct Place {
        uint32_t row, q;      // own row of the slab, word of the row
        uint32_t at;          // word index of (row, q) in a colour's slab
        uint32_t h;           // the half index of the word's first site
        int32_t up, down;     // word offsets of the rows next to it
        uint32_t parity;
        bool mine;
        bool first_unit, last_unit;
    };
    auto fill = [&](Place& p, bool in) {
        p.mine = in && lane < step;
        p.h = (row0 + p.row) * W + 4u * p.q;
        const uint32_t own_row = in ? p.row : 0u;
        uint32_t y = row0 + own_row, z = 0u;
        if (DIMS == 3) {
            z = k.by_L.quot(y);
            y -= z * L;
        }
        p.parity = (y + z) & 1u;
        p.at = (unit_rows + own_row) * P + 1u + p.q;
        p.up = -(int32_t)P;
        p.down = (int32_t)P;
        if (DIMS == 3) {  // planes are whole: y wraps inside them
            if (y == 0u) p.up = (int32_t)((L - 1u) * P);
            if (y + 1u == L) p.down = -(int32_t)((L - 1u) * P);
        }
        p.first_unit = own_row < unit_rows;
        p.last_unit = own_row + unit_rows >= rows;
    };
    auto place = [&](uint32_t first) {
        Place p;
        p.row = k.by_words.quot(first + lane);
        p.q = first + lane - p.row * words;
        fill(p, first + lane < items);
        return p;
    };
    auto next_place = [&](const Place& p0, uint32_t first) {
        Place p = p0;
        p.row += stride_rows;
        p.q += stride_words;
        if (p.q >= words) {
            p.q -= words;
            ++p.row;
        }
        fill(p, first + lane < items);
        return p;
    };
    // where a slab's first (last) unit goes in the CTA before (behind): word
    // offsets from p.at, per colour
    const uint32_t own_colour = all_rows * P;
    const uint32_t before_colour = (before_units + 2u) * unit_rows * P;
    const uint32_t behind_colour = (behind_units + 2u) * unit_rows * P;
    const uint32_t to_before = before_units * unit_rows * P;  // unit 1 -> unit before_units + 1
    const uint32_t to_behind = rows * P;                      // unit n -> unit 0 (subtracted)
    PassArgs a = k.a;
    auto tests = [&](uint32_t h, uint32_t t, uint32_t c) {
        const Philox4 u = philox4x32_10(h >> 2, t, c, kTagSweep, a.key0, a.key1);
        uint32_t n = count_word<DIMS, RULE>(u, a);
        if (RAGGED) {
            const uint32_t next = __shfl_down_sync(0xffffffffu, n, 1);
            n = __funnelshift_r(n, next, 8u * (h & 3u));
        }
        return n;
    };
    auto update = [&](const Place& p, uint32_t count, uint32_t c, int& e, int& m) {
        uint32_t* own = S0 + (c == 0u ? 0u : own_colour) + p.at;
        const uint32_t* other = S0 + (c == 0u ? own_colour : 0u) + p.at;
        const uint32_t s = own[0];
        const uint32_t nx = other[0], nl = other[-1], nr = other[1];
        const uint32_t nym = other[p.up], nyp = other[p.down];
        uint32_t nzm = 0u, nzp = 0u;
        if (DIMS == 3) {
            nzm = other[-(int32_t)(L * P)];
            nzp = other[(int32_t)(L * P)];
        }
        const uint32_t nxs = ((c + p.parity) & 1u) == 0u ? __funnelshift_l(nl, nx, 8)
                                                         : __funnelshift_r(nx, nr, 8);
        const uint32_t D = disagreements<DIMS>(s, nx, nxs, nym, nyp, nzm, nzp);
        const uint32_t X = flip_mask(D, count);
        const uint32_t v = s ^ (X & kByteFlip);
        if (!p.mine) return;
        put_word<RAGGED>(own, p.q, words, W, v);
        if (p.first_unit)
            put_word<RAGGED>(before_smem + (c == 0u ? 0u : before_colour) + p.at + to_before, p.q,
                             words, W, v);
        if (p.last_unit)
            put_word<RAGGED>(behind_smem + (c == 0u ? 0u : behind_colour) + p.at - to_behind, p.q,
                             words, W, v);
        uint32_t valid = 0xFFFFFFFFu;
        int n = 4;
        if (RAGGED && p.q + 1u == words) {
            n = (int)(W - 4u * p.q);
            valid = n == 4 ? 0xFFFFFFFFu : (1u << (8 * n)) - 1u;
        }
        m = add_bytes(v & valid, m);
        if (c == 1u) {
            constexpr uint32_t q2 = 4u * DIMS * kByteOnes;
            e = add_bytes(((D & ~X) | ((q2 - D) & X)) & valid, e - n * 2 * DIMS);
        }
    };
    const bool works = first0 < items;  // the same for the whole warp
    const Place p0 = place(first0);
    auto arrive = [&] {
        __syncwarp();
        if (ranks > 1u) cl.barrier_arrive();
    };
    auto wait = [&] {
        __syncwarp();
        if (ranks > 1u)
            cl.barrier_wait();
        else
            __syncthreads();
    };
    arrive();
    uint32_t count = works ? tests(p0.h, a.t, 0u) : 0u;
    int64_t rec = 0;
    uint32_t until = (uint32_t)k.every - (uint32_t)((uint64_t)a.t % (uint32_t)k.every);
    for (int s = 0; s < k.nsweeps; ++s) {
        const uint32_t t = a.t + (uint32_t)s;
        int e = 0, m = 0;
        for (uint32_t c = 0; c < 2u; ++c) {
            wait();
            if (works) {
                update(p0, count, c, e, m);
                Place p = p0;
                for (uint32_t first = first0 + stride; first < items; first += stride) {
                    p = next_place(p, first);
                    update(p, tests(p.h, t, c), c, e, m);
                }
            }
            arrive();
            if (works) count = tests(p0.h, c == 0u ? t : t + 1u, c ^ 1u);
        }
        if (--until == 0u) {  // sweep t is recorded
            until = (uint32_t)k.every;
            e = __reduce_add_sync(0xffffffffu, e);
            m = __reduce_add_sync(0xffffffffu, m);
            if (works && lane == 0u) {
                if (e != 0) atomicAdd(&k.obs[2 * rec], (unsigned long long)(long long)e);
                if (m != 0) atomicAdd(&k.obs[2 * rec + 1], (unsigned long long)(long long)m);
            }
            ++rec;
        }
    }
    wait();

    // the slab back to the lattice's layout
    if constexpr (LAYOUT == ISING_BITPACK) {
        const uint32_t nq = (W + 31u) >> 5;
        for (uint32_t i = threadIdx.x; i < 2u * rows * nq; i += blockDim.x) {
            const uint32_t row = i / nq, q = i - row * nq;
            const uint32_t c = row >= rows ? 1u : 0u, r = row - c * rows;
            const uint32_t* in = S0 + (c * all_rows + unit_rows + r) * P + 1u + 8u * q;
            uint32_t bits = 0u;
            for (uint32_t j = 0; j < 8u && 8u * q + j < words; ++j) {
                const uint32_t up = (~in[j] >> 7) & kByteOnes;
                bits |= ((up * 0x01020408u >> 24) & 0xFu) << (4u * j);
            }
            const uint32_t nb = W - 32u * q;
            if (nb < 32u) bits &= (1u << nb) - 1u;
            static_cast<uint32_t*>(c == 0u ? k.a.own : const_cast<void*>(k.a.other))
                [(row0 + r) * nq + q] = bits;
        }
    } else {
        for (uint32_t i = threadIdx.x; i < 2u * rows * words; i += blockDim.x) {
            const uint32_t row = k.by_words.quot(i), q = i - row * words;
            const uint32_t c = row >= rows ? 1u : 0u, r = row - c * rows;
            const uint32_t v = S0[(c * all_rows + unit_rows + r) * P + 1u + q];
            uint8_t* out = static_cast<uint8_t*>(c == 0u ? k.a.own : const_cast<void*>(k.a.other)) +
                           (size_t)(row0 + r) * W + 4u * q;
            if ((W & 3u) == 0u)
                *reinterpret_cast<uint32_t*>(out) = v;
            else
                for (uint32_t j = 0; j < 4u && 4u * q + j < W; ++j) out[j] = (uint8_t)(v >> (8u * j));
        }
    }
    // no CTA leaves while another may still store into its halos: the last wait
    // above was behind the last of those stores
}

template <int DIMS, int RULE, int LAYOUT, bool RAGGED>
cudaError_t launch_resident(const ResidentArgs& k, unsigned ranks, unsigned threads, size_t smem,
                            cudaStream_t st) {
    auto kernel = resident_kernel<DIMS, RULE, LAYOUT, RAGGED>;
    cudaError_t e = cudaSuccess;
    if (smem > 48 * 1024)
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess && ranks > 8u)  // beyond the portable size
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ranks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = ranks;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, k);
}

template <int DIMS, int RULE>
cudaError_t launch_resident_layout(const ResidentArgs& k, int layout, unsigned ranks,
                                   unsigned threads, size_t smem, cudaStream_t st) {
    const bool ragged = k.a.W % 4 != 0;
    if (layout == ISING_BITPACK)
        return ragged ? launch_resident<DIMS, RULE, ISING_BITPACK, true>(k, ranks, threads, smem, st)
                      : launch_resident<DIMS, RULE, ISING_BITPACK, false>(k, ranks, threads, smem,
                                                                          st);
    return ragged ? launch_resident<DIMS, RULE, ISING_INT8, true>(k, ranks, threads, smem, st)
                  : launch_resident<DIMS, RULE, ISING_INT8, false>(k, ranks, threads, smem, st);
}

}  // namespace

// Where one launch beats 2 n passes of the layout.  Measured, us a pass in runs
// of 50 sweeps (here / pass kernels; the single CTA that took the smallest
// lattices before in brackets): 2D L = 64 0.7 / 2.7 [1.1], L = 128 0.75 / 2.7
// [10.9 int8, 1.6 packed], L = 256 0.9 - 1.0 / 2.8 int8 and 1.85 packed, L = 384
// 1.65, L = 512 2.15; ragged L = 100 1.05, L = 510 3.1; 3D L = 32 0.96, L = 64
// 2.4, ragged L = 26 1.4, L = 62 3.3.  A pass grows with the words, ragged ones
// costing 1.6 times as much, so the line is where it meets the pass kernels': 2.7
// us for int8 and 1.85 for packed.  The launch, the load and the store take 3 to
// 6 us, by size, which two int8 sweeps' passes outlast; packed ones, in us a call
// of back-to-back calls (here / pass kernels): two sweeps 2D L = 16 5.2 / 7.3, L =
// 128 6.2 / 7.2, but ragged L = 50 8.2 / 7.3 and L = 256 8.2 / 7.2; three L = 50
// 10.3 / 10.6, L = 256 9.3 / 10.6, but L = 250 14.1 / 10.7; one sweep L = 64 6.2 /
// 4.0 in either layout.  Rows of less than a vector go word by word in the int8
// pass kernels (4 us a pass and more), so those always come here.  (Unless the
// caller names an int8 kernel, by ising_set_kernel or a registered configuration:
// ising_sweep then runs that one's passes.)
bool resident_ok(const ising_lattice* h, int64_t n) {
    if (h->rule != ISING_RULE_METROPOLIS && h->rule != ISING_RULE_HEATBATH) return false;
    if (n > 0x7FFFFFFF) return false;
    const bool packed = h->layout == ISING_BITPACK;
    const int64_t words = h->rows * ((h->W + 3) / 4);
    const int64_t cost = h->W % 4 == 0 ? words : words * 8 / 5;
    if (!packed) return cost <= 42000 && n >= (h->W < 16 ? 1 : 2);
    return cost <= 22000 && n >= (h->W % 4 == 0 && words <= 2048 ? 2 : cost <= 8192 ? 3 : 4);
}

cudaError_t resident_sweep(ising_lattice* h, const PassArgs& args, int64_t n, int every,
                           unsigned long long* slots) {
    ResidentArgs k;
    k.a = args;
    k.obs = slots;
    k.nsweeps = (int)n;
    k.every = every;
    k.words = ((uint32_t)h->W + 3u) / 4u;
    k.pitch = k.words + 2u;
    k.by_words = FastDiv(k.words);
    k.by_L = FastDiv((uint32_t)h->L);
    // as many CTAs as give every thread about one word of a colour, at most 16
    // and at most one per unit
    const uint32_t unit_rows = h->dims == 3 ? (uint32_t)h->L : 1u;
    const uint64_t items = (uint64_t)h->rows * k.words;
    unsigned ranks = 1;
    while (ranks < 16u && items > (uint64_t)ranks * 256u && 2u * ranks <= (unsigned)h->L)
        ranks *= 2u;
    const uint64_t per_rank = (items + ranks - 1) / ranks;
    unsigned threads = (unsigned)((per_rank + 30) / 31 * 32);
    if (threads > 512u) threads = 512u;
    const uint32_t units = ((uint32_t)h->L + ranks - 1u) / ranks;
    const size_t smem = (size_t)2 * (units + 2u) * unit_rows * k.pitch * sizeof(uint32_t);
    if (h->dims == 2)
        return h->rule == ISING_RULE_HEATBATH
                   ? launch_resident_layout<2, kRuleHeatBath>(k, h->layout, ranks, threads, smem,
                                                              h->stream)
                   : launch_resident_layout<2, kRuleMetropolis>(k, h->layout, ranks, threads, smem,
                                                                h->stream);
    return h->rule == ISING_RULE_HEATBATH
               ? launch_resident_layout<3, kRuleHeatBath>(k, h->layout, ranks, threads, smem,
                                                          h->stream)
               : launch_resident_layout<3, kRuleMetropolis>(k, h->layout, ranks, threads, smem,
                                                            h->stream);
}

}  // namespace ising
