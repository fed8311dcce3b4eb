// sweep_bitpack.cu -- colour pass of the checkerboard Metropolis sweep on the
// bit-packed ("multispin") layout, with the E and M reductions fused in.
//
// Layout: each half row r of colour c (its W = L/2 sites, half column
// xh = 0..W-1, half index h = r*W + xh) takes nq = ceil(W/32) uint32 words;
// site xh is bit (xh mod 32) of word r*nq + xh/32, bit 1 meaning spin +1.  The
// bits past W in a row's last word are padding: zero, never read as spins,
// never flipped.  Row r's word q of the other colour lines up with the site
// word bit for bit (same half column), the second x-neighbour is one bit to
// the right (p = 0: xh - 1) or left (p = 1: xh + 1), p = (c + y + z) & 1, and
// the y- and z-neighbour words are the same word of the neighbouring rows.
//
// The Metropolis rule (Sec. 2.2) is evaluated for 32 sites at once: the
// per-site count d of disagreeing neighbours is formed by bit-sliced adders
// over the xor of the site word with its 2*dims neighbour words, which yields
// the mask of sites with dE <= 0 (d >= dims; they flip) and, for the others,
// the mask of sites with each d < dims, selecting the threshold
// floor(exp(-2 beta k) 2^32), k = 2(dims - d).  Draws are identical to the
// int8 layout: site h uses word h & 3 of Philox(seed; h >> 2, t, c, 0).
#include <cstdint>

#include "engine_internal.h"
#include "ising_device.cuh"
#include "pass_bodies.cuh"

namespace ising {

namespace {

// How a lattice's words are walked.
//   kWordsFull: lattices whose words are all full (W % 32 == 0) and whose word
//     count per half row nq = 2^nq_shift is a power of two (then so is
//     L = 64 nq; in 3D l_shift = log2 L): an item's row, word and neighbours come
//     from shifts and masks, and every row starts on a Philox group.
//   kWordsAligned: rows that start on a Philox group (W % 4 == 0).
//   kWordsRagged: any other even L.
// In the last two a warp takes its words together (packed_place).
//
// The first item's draws need only counters: they are made before the wait for
// the previous pass, so that a pass placed on the SMs while the previous one
// drains has them ready.  The next pass is let in only behind the wait: a lattice
// that leaves SMs free would otherwise have three passes or more on the GPU at
// once.  Later items load first and draw while the loads are under way.
// Per pass, in us, against waiting first: 2D L = 512 2.6 -> 1.8 (the host's
// launches then set the pace), L = 2048 4.4 -> 3.0, L = 4096 8.4 -> 6.5, L = 8192
// 24.4 -> 23.6; 3D L = 128 3.0 -> 2.2, L = 202 8.7 -> 6.4.  (The int8 passes
// gained nothing by it: 2D L = 500 2.75 -> 2.77, L = 1000 2.75 -> 3.64.)
constexpr int kWordsFull = 0, kWordsAligned = 1, kWordsRagged = 2;

// Multi-hit: the first item's later trials drawn ahead too, up to this many, kept
// in shared memory (three hits, us a pass: 2D L = 512 3.6 -> 3.3, L = 2048 7.6 ->
// 5.8, L = 8192 66 either way).
constexpr int kLaterTrials = 3;

template <int DIMS, bool MEASURE, int RULE, int WORDS>
__global__ void __launch_bounds__(256, 3) pass_packed(PassArgs a, PackedGeom geom,
                                                      uint32_t nq_shift, uint32_t l_shift) {
    constexpr int draw = WORDS == kWordsRagged ? kDrawRagged : kDrawAligned;
    constexpr uint32_t step = kWarpWords<draw>;
    const uint32_t items = geom.items, L = (uint32_t)a.L, W = (uint32_t)a.W;
    const uint32_t stride = ((gridDim.x * blockDim.x) >> 5) * step;
    const int second = WORDS == kWordsFull ? 4 : packed_second(a);
    auto place = [&](uint32_t first) {
        if constexpr (WORDS != kWordsFull) {
            return packed_place<draw>(geom, W, first);
        } else {  // items is a multiple of 32
            const uint32_t item = first + (threadIdx.x & 31u);
            PackedPlace p;
            p.r = item >> nq_shift;
            p.q = item & ((1u << nq_shift) - 1u);
            p.hbase = p.r * W + 32u * p.q;
            p.mine = true;
            return p;
        }
    };
    auto load = [&](const PackedPlace& pl) {
        if constexpr (WORDS != kWordsFull) {
            return packed_load<DIMS>(a, geom, pl);
        } else {
            const uint32_t nq = 1u << nq_shift, r = pl.r, q = pl.q;
            const uint32_t* other = static_cast<const uint32_t*>(a.other);
            const uint32_t z = DIMS == 3 ? r >> l_shift : 0u, y = r & (L - 1u);
            const uint32_t row = r * nq, plane = z * L;
            PackedWord w;
            w.p = (a.c + (int)y + (int)z) & 1;
            // x-neighbour word: the one before (p = 0) or after (p = 1), wrapping in the row
            const uint32_t xq = (w.p == 0 ? q - 1u : q + 1u) & (nq - 1u);
            w.at = row + q;
            w.o = other[w.at];
            w.x = other[row + xq];
            w.ym = other[(plane + ((y - 1u) & (L - 1u))) * nq + q];
            w.yp = other[(plane + ((y + 1u) & (L - 1u))) * nq + q];
            w.zm = w.zp = 0u;
            if (DIMS == 3) {
                w.zm = other[(((z - 1u) & (L - 1u)) * L + y) * nq + q];
                w.zp = other[(((z + 1u) & (L - 1u)) * L + y) * nq + q];
            }
            w.s = static_cast<const uint32_t*>(a.own)[w.at];
            w.valid = 0xFFFFFFFFu;
            w.hbase = pl.hbase;
            w.edge = 0u;
            w.mine = true;
            return w;
        }
    };
    int e_acc = 0, m_acc = 0;
    uint32_t first = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * step;
    if (first < items) {
        uint32_t A[kThresholds<DIMS, RULE>];
        PackedPlace pl = place(first);
        packed_draws<DIMS, RULE, draw>(pl.hbase, second, a, (uint32_t)a.c, A);
#pragma unroll
        for (uint32_t& v : A) pin_here(v);
        constexpr int N = kThresholds<DIMS, RULE>;
        __shared__ uint32_t s_later[RULE == kRuleMultiHit ? kLaterTrials * N * 256 : 1];
        uint32_t* later = s_later + (RULE == kRuleMultiHit ? threadIdx.x : 0u);
        int n_later = 0;
        if constexpr (RULE == kRuleMultiHit) {
            n_later = a.hits - 1 < kLaterTrials ? a.hits - 1 : kLaterTrials;
#pragma unroll 1
            for (int m = 0; m < n_later; ++m) {
                uint32_t B[N];
                packed_draws<DIMS, RULE, draw>(pl.hbase, second, a,
                                               (uint32_t)a.c + 2u * (uint32_t)(m + 1), B);
#pragma unroll
                for (int n = 0; n < N; ++n) later[(m * N + n) * 256] = B[n];
            }
        }
        grid_dependency_wait();
        launch_dependents();
        PackedWord w = load(pl);
        for (;;) {
            __syncwarp();
            packed_update<DIMS, MEASURE, RULE, draw>(a, w, A, second, e_acc, m_acc, later, n_later);
            first += stride;
            n_later = 0;
            if (first >= items) break;
            pl = place(first);
            w = load(pl);
            packed_draws<DIMS, RULE, draw>(pl.hbase, second, a, (uint32_t)a.c, A);
        }
    } else {
        grid_dependency_wait();
        launch_dependents();
    }
    if (MEASURE) block_reduce_add(e_acc, m_acc, a.obs, a.c == 1);
}

// Initial state written straight into the packed layout: one thread per word
// of one colour; bit b of word (r, q) is half column xh = 32q + b, i.e. the
// canonical site i = L*r + 2*xh + p.
__global__ void init_packed(uint32_t* col0, uint32_t* col1, int L, int dims, int64_t rows,
                            int start, uint32_t key0, uint32_t key1) {
    const int W = L / 2, nq = (W + 31) / 32;
    const int64_t words = rows * nq;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t w2 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w2 < 2 * words;
         w2 += stride) {
        const int c = (int)(w2 / words);
        const int64_t w = w2 - (int64_t)c * words;
        const int64_t r = w / nq;
        const int q = (int)(w - r * nq);
        const int nb = W - 32 * q < 32 ? W - 32 * q : 32;
        uint32_t bits = 0u;
        if (start == 0) {
            const int64_t y = r % L, z = dims == 3 ? r / L : 0;
            const int p = (int)((c + y + z) & 1);
            for (int b = 0; b < nb; ++b) {
                const int64_t i = (int64_t)L * r + 2 * (32 * q + b) + p;
                const Philox4 u = philox4x32_10((uint32_t)(i >> 2), 0u, 0u, kTagInit, key0, key1);
                const uint32_t wd[4] = {u.w0, u.w1, u.w2, u.w3};
                if (wd[i & 3] < 0x80000000u) bits |= 1u << b;
            }
        } else if (start == 1) {
            bits = nb == 32 ? 0xFFFFFFFFu : ((1u << nb) - 1u);
        }
        (c == 0 ? col0 : col1)[w] = bits;
    }
}

__global__ void export_packed(const uint32_t* col0, const uint32_t* col1, int8_t* out, int L,
                              int dims, int64_t sites) {
    const int nq = (L / 2 + 31) / 32;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < sites; i += stride) {
        const int64_t x = i % L, r = i / L;
        const int64_t y = r % L, z = dims == 3 ? r / L : 0;
        const int64_t xh = x >> 1;
        const uint32_t word = (((x + y + z) & 1) == 0 ? col0 : col1)[r * nq + (xh >> 5)];
        out[i] = ((word >> (xh & 31)) & 1u) ? (int8_t)1 : (int8_t)-1;
    }
}

// One thread per packed word: gather its canonical bytes.
__global__ void import_packed(uint32_t* col0, uint32_t* col1, const int8_t* in, int L, int dims,
                              int64_t rows) {
    const int W = L / 2, nq = (W + 31) / 32;
    const int64_t words = rows * nq;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t w2 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w2 < 2 * words;
         w2 += stride) {
        const int c = (int)(w2 / words);
        const int64_t w = w2 - (int64_t)c * words;
        const int64_t r = w / nq;
        const int q = (int)(w - r * nq);
        const int64_t y = r % L, z = dims == 3 ? r / L : 0;
        const int p = (int)((c + y + z) & 1);
        const int nb = W - 32 * q < 32 ? W - 32 * q : 32;
        uint32_t bits = 0u;
        for (int b = 0; b < nb; ++b)
            if (in[(int64_t)L * r + 2 * (32 * q + b) + p] > 0) bits |= 1u << b;
        (c == 0 ? col0 : col1)[w] = bits;
    }
}

unsigned grid_for(int64_t n, const DeviceProps& dp) {
    int64_t b = (n + 255) / 256;
    const int64_t cap = (int64_t)dp.sm_count * 16;
    if (b > cap) b = cap;
    return (unsigned)(b < 1 ? 1 : b);
}

bool is_pow2(int x) { return x > 0 && (x & (x - 1)) == 0; }

template <int DIMS, bool MEASURE, int RULE>
cudaError_t launch_packed_t(const PassArgs& a, const DeviceProps& dp, cudaStream_t st) {
    const int nq = (a.W + 31) >> 5;
    const int64_t items = a.rows * nq;
    const int words = a.W % 32 == 0 && is_pow2(nq) ? kWordsFull
                      : a.W % 4 == 0               ? kWordsAligned
                                                   : kWordsRagged;
    const int64_t per_block =
        8 * (words == kWordsRagged ? kWarpWords<kDrawRagged> : kWarpWords<kDrawAligned>);
    int64_t blocks = (items + per_block - 1) / per_block;
    const int64_t cap =
        (int64_t)dp.sm_count * dp.blocks_per_sm_packed[RULE][DIMS - 2][MEASURE][words];
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    const PackedGeom geom((uint32_t)a.W, (uint32_t)a.L, (uint32_t)a.rows);
    if (words == kWordsFull) {
        const uint32_t nq_shift = (uint32_t)__builtin_ctz((unsigned)nq);
        const uint32_t l_shift = DIMS == 3 ? (uint32_t)__builtin_ctz((unsigned)a.L) : 0u;
        return launch_chained(pass_packed<DIMS, MEASURE, RULE, kWordsFull>, (unsigned)blocks,
                              256u, 0, st, a, geom, nq_shift, l_shift);
    }
    if (words == kWordsAligned)
        return launch_chained(pass_packed<DIMS, MEASURE, RULE, kWordsAligned>, (unsigned)blocks,
                              256u, 0, st, a, geom, 0u, 0u);
    return launch_chained(pass_packed<DIMS, MEASURE, RULE, kWordsRagged>, (unsigned)blocks, 256u,
                          0, st, a, geom, 0u, 0u);
}

}  // namespace

cudaError_t packed_query_occupancy(DeviceProps& dp) {
    cudaError_t e;
#define ISING_OCC1(R, D, M, F)                                                                \
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&dp.blocks_per_sm_packed[R][D - 2][M][F],\
                                                      pass_packed<D, M, R, F>, 256, 0);       \
    if (e != cudaSuccess) return e;
#define ISING_OCC(R, D, M)                                                        \
    ISING_OCC1(R, D, M, kWordsFull) ISING_OCC1(R, D, M, kWordsAligned)            \
        ISING_OCC1(R, D, M, kWordsRagged)
    ISING_OCC(kRuleMetropolis, 2, false)
    ISING_OCC(kRuleMetropolis, 2, true)
    ISING_OCC(kRuleMetropolis, 3, false)
    ISING_OCC(kRuleMetropolis, 3, true)
    ISING_OCC(kRuleHeatBath, 2, false)
    ISING_OCC(kRuleHeatBath, 2, true)
    ISING_OCC(kRuleHeatBath, 3, false)
    ISING_OCC(kRuleHeatBath, 3, true)
    ISING_OCC(kRuleMultiHit, 2, false)
    ISING_OCC(kRuleMultiHit, 2, true)
    ISING_OCC(kRuleMultiHit, 3, false)
    ISING_OCC(kRuleMultiHit, 3, true)
#undef ISING_OCC
#undef ISING_OCC1
    return cudaSuccess;
}

template <int RULE>
static cudaError_t packed_pass_rule(const PassArgs& a, int dims, bool measure,
                                    const DeviceProps& dp, cudaStream_t st) {
    if (dims == 2)
        return measure ? launch_packed_t<2, true, RULE>(a, dp, st)
                       : launch_packed_t<2, false, RULE>(a, dp, st);
    return measure ? launch_packed_t<3, true, RULE>(a, dp, st)
                   : launch_packed_t<3, false, RULE>(a, dp, st);
}

cudaError_t packed_pass(const PassArgs& a, int dims, bool measure, int rule,
                        const DeviceProps& dp, cudaStream_t st) {
    if (rule == kRuleHeatBath) return packed_pass_rule<kRuleHeatBath>(a, dims, measure, dp, st);
    if (rule == kRuleMultiHit) return packed_pass_rule<kRuleMultiHit>(a, dims, measure, dp, st);
    return packed_pass_rule<kRuleMetropolis>(a, dims, measure, dp, st);
}

cudaError_t packed_init(uint32_t* col0, uint32_t* col1, int L, int dims, int64_t rows, int start,
                        uint32_t key0, uint32_t key1, const DeviceProps& dp, cudaStream_t st) {
    init_packed<<<grid_for(2 * rows * ((L / 2 + 31) / 32), dp), 256, 0, st>>>(
        col0, col1, L, dims, rows, start, key0, key1);
    return cudaGetLastError();
}

cudaError_t packed_export(const uint32_t* col0, const uint32_t* col1, int8_t* out, int L,
                          int dims, int64_t sites, const DeviceProps& dp, cudaStream_t st) {
    export_packed<<<grid_for(sites, dp), 256, 0, st>>>(col0, col1, out, L, dims, sites);
    return cudaGetLastError();
}

cudaError_t packed_import(uint32_t* col0, uint32_t* col1, const int8_t* in, int L, int dims,
                          int64_t rows, const DeviceProps& dp, cudaStream_t st) {
    import_packed<<<grid_for(2 * rows * ((L / 2 + 31) / 32), dp), 256, 0, st>>>(col0, col1, in,
                                                                                 L, dims, rows);
    return cudaGetLastError();
}

}  // namespace ising
