// pass_bodies.cuh -- per-word and per-vector bodies of a colour pass, shared by
// the per-lattice kernels (sweep_int8.cu, sweep_int8_tma.cu, sweep_bitpack.cu),
// the small lattices' cluster kernel (resident.cu) and the batched kernels
// (batch.cu).
//
// The int8 word body (int8_word, rows of less than a 16-site vector; longer rows
// take int8_vec) works for any even L: a word of the colour array holds the
// four half indices h = 4w..4w+3 (one Philox group), whatever rows they fall
// in.  A word that lies inside one half row, away from the x-wrap and from
// the first and last row (and plane) of the lattice, takes the byte-sliced
// path: its neighbour words are 4-byte windows of the other colour at byte
// offsets h - 1 / h + 1 (x), h -+ W (y) and h -+ L*W (z), read as two aligned
// words and a funnel shift.  Every other word (rows shorter than a word, row
// ends, wrap rows and planes, the ragged tail) takes the per-site path, which
// finds each neighbour from the site's coordinates.  Both paths apply the
// same rule and the same draw (word h & 3 of Philox(seed; h >> 2, t, c, 0)).
//
// The other colour is read with ordinary loads throughout: a chained pass lives
// while the pass before it still writes that colour, and the batched kernel runs
// both colours' passes in one launch (see grid_dependency_wait()).
#pragma once

#include <cstdint>

#include "ising_device.cuh"

namespace ising {

constexpr uint32_t kByteBit1 = 0x02020202u;
constexpr uint32_t kByteBit7 = 0x80808080u;
constexpr uint32_t kByteOnes = 0x01010101u;

// 0xFF per site whose flip is decided without a draw: byte j of D is 2 d_j, and
// bit 7 of D + bias is set iff d_j >= dims (dE <= 0).
template <int DIMS>
__device__ __forceinline__ uint32_t downhill_mask(uint32_t D) {
    return byte_signs(D + (0x80u - 2u * DIMS) * kByteOnes);
}

// The tests of a word's four sites, from their draws alone: byte j of count_word
// is bias + 2 cnt_j; and the sites that flip, 0xFF per byte, once D (byte j is
// 2 d_j) is known.  With cnt_j the number of the rule's thresholds that
// u_j lies below (they are nested) -- Metropolis: the thresholds fall with k, so
// a site with d < dims flips iff cnt + d >= dims, and one with d >= dims always
// does: bit 7 of D + 2 cnt + bias (at most 0x80 + 4 dims: no carry).  Heat bath
// (every site draws; it flips iff u < thr[d], the thresholds rising with d): iff
// cnt + d >= 2 dims + 1 (at most 4 (2 dims) + 2 + bias < 256).
//
// A compare and a predicated add per threshold: with the generator, E and M in
// registers 106 issue slots a word (2D; 83 the generator alone).  The sum of
// selects took 119 as compiled, toggling the bits of the count 127: the ALU pipe
// takes one instruction in two cycles, and adds (and the byte sums of E and M)
// need not go there.
template <int DIMS, int RULE>
__device__ __forceinline__ uint32_t count_word(const Philox4& u, const PassArgs& a,
                                               uint32_t D = 0u) {
    constexpr int N = RULE == kRuleHeatBath ? 2 * DIMS + 1 : DIMS;
    constexpr uint32_t need = RULE == kRuleHeatBath ? 2u * DIMS + 1u : (uint32_t)DIMS;
    uint32_t acc = D + (0x80u - 2u * need) * kByteOnes;
    static_for<4>([&](auto site) {
        constexpr int j = decltype(site)::value;
        const uint32_t w = j == 0 ? u.w0 : j == 1 ? u.w1 : j == 2 ? u.w2 : u.w3;
#pragma unroll
        for (int n = 0; n < N; ++n) add_below<(2u << (8 * j))>(acc, w, a.thr[n]);
    });
    return acc;
}
__device__ __forceinline__ uint32_t flip_mask(uint32_t D, uint32_t count) {
    return byte_signs(D + count);
}
// Both where D is known by then (an add less).
template <int DIMS, int RULE>
__device__ __forceinline__ uint32_t flip_mask(uint32_t D, const Philox4& u, const PassArgs& a) {
    return byte_signs(count_word<DIMS, RULE>(u, a, D));
}

// Sum of a word's four spins (bytes +1 / -1) or counts, added to acc.
__device__ __forceinline__ int add_bytes(uint32_t w, int acc) {
    return __dp4a((int)w, (int)kByteOnes, acc);
}

constexpr uint32_t kByteFlip = 0xFEFEFEFEu;  // 0x01 <-> 0xFF

// thr[d] by selects (d = 0..2*dims), for code that holds PassArgs in registers.
template <int DIMS>
__device__ __forceinline__ uint32_t heatbath_threshold(int d, const PassArgs& a) {
    uint32_t t = a.thr[0];
#pragma unroll
    for (int m = 1; m <= 2 * DIMS; ++m) t = d == m ? a.thr[m] : t;
    return t;
}

// Multi-hit Metropolis on one 4-site word: a.hits successive trials, the
// neighbours fixed; after a trial the flipped sites' D becomes 2(2 dims - d).
// Trial m draws Philox(seed; group, t, c + 2m, 0).  Returns the net flip mask.
template <int DIMS>
__device__ __forceinline__ uint32_t multihit_word(uint32_t D, uint32_t group, const PassArgs& a) {
    constexpr uint32_t q2 = 4u * DIMS * kByteOnes;
    uint32_t net = 0u;
#pragma unroll 1
    for (int m = 0; m < a.hits; ++m) {
        uint32_t X = downhill_mask<DIMS>(D);
        if (X != 0xFFFFFFFFu) {
            const Philox4 u = philox4x32_10(group, a.t, (uint32_t)a.c + 2u * (uint32_t)m,
                                            kTagSweep, a.key0, a.key1);
            X = flip_mask<DIMS, kRuleMetropolis>(D, u, a);
        }
        D = (D & ~X) | ((q2 - D) & X);
        net ^= X;
    }
    return net;
}

template <int DIMS>
__device__ __forceinline__ uint32_t disagreements(uint32_t s, uint32_t n0, uint32_t n1,
                                                  uint32_t n2, uint32_t n3, uint32_t n4,
                                                  uint32_t n5) {
    uint32_t D = ((s ^ n0) & kByteBit1) + ((s ^ n1) & kByteBit1) + ((s ^ n2) & kByteBit1) +
                 ((s ^ n3) & kByteBit1);
    if (DIMS == 3) D += ((s ^ n4) & kByteBit1) + ((s ^ n5) & kByteBit1);
    return D;
}

// Four bytes of the other colour starting at byte offset o (o >= 0; the array
// is padded so that the word after the last one may be read).
__device__ __forceinline__ uint32_t window4(const uint32_t* other, uint32_t o) {
    const uint32_t lo = other[o >> 2];
    if ((o & 3u) == 0u) return lo;
    const uint32_t hi = other[(o >> 2) + 1];
    return __funnelshift_r(lo, hi, 8u * (o & 3u));
}

// Quotients by a fixed divisor d >= 1 of n < 2^31: with 2^s <= d < 2^(s+1) and
// m = ceil(2^(32+s) / d), n m / 2^(32+s) exceeds n / d by less than
// n / 2^31 / d, too little to reach the next integer.  Powers of two take
// half of both, and d = 1 the last term.  Six issue slots instead of the twenty
// or so of a division, of which a packed word of ragged rows needs four.
struct FastDiv {
    uint32_t d, m, s, one;
    FastDiv() = default;
    __host__ __device__ __forceinline__ explicit FastDiv(uint32_t div) : d(div), s(0), one(0) {
        while ((2u << s) <= d && s < 31u) ++s;
        if (d == 1u) {
            m = 0u;
            one = 0xFFFFFFFFu;
        } else if ((d & (d - 1u)) == 0u) {
            m = 0x80000000u;
            --s;
        } else {
            m = (uint32_t)(((1ull << (32u + s)) + d - 1u) / d);
        }
    }
    __device__ __forceinline__ uint32_t quot(uint32_t n) const {
        return (__umulhi(n, m) >> s) + (n & one);
    }
};

struct WordGeom {
    uint32_t W;       // sites per half row
    uint32_t L;
    uint32_t rows;    // L^(dims-1)
    uint32_t half;    // sites per colour
    FastDiv by_W, by_L;
    WordGeom() = default;
    __host__ __device__ __forceinline__ WordGeom(uint32_t W_, uint32_t L_, uint32_t rows_)
        : W(W_), L(L_), rows(rows_), half(W_ * rows_), by_W(W_), by_L(L_) {}
};

// Update word w of the int8 colour array `own` (colour a.c).  Accumulates the
// sum of the spins written (m_sum) and, in the white pass,
// sum (2 d_new - 2 dims) over them (e_acc).
template <int DIMS, bool MEASURE, int RULE>
__device__ __forceinline__ void int8_word(const PassArgs& a, const WordGeom& g, uint32_t w,
                                          int& e_acc, int& m_sum) {
    uint32_t* own = static_cast<uint32_t*>(a.own);
    const uint32_t* other = static_cast<const uint32_t*>(a.other);
    const int8_t* other_b = static_cast<const int8_t*>(a.other);
    const uint32_t h0 = 4u * w;
    const uint32_t r0 = g.by_W.quot(h0);
    const uint32_t xh0 = h0 - r0 * g.W;
    uint32_t y0 = r0, z0 = 0;
    if (DIMS == 3) {
        z0 = g.by_L.quot(r0);
        y0 = r0 - z0 * g.L;
    }
    const int p = (a.c + (int)y0 + (int)z0) & 1;
    bool fast = (xh0 + 3u < g.W) && (h0 + 3u < g.half) && y0 != 0u && y0 + 1u != g.L;
    if (DIMS == 3) fast = fast && z0 != 0u && z0 + 1u != g.L;
    fast = fast && (p == 0 ? xh0 != 0u : xh0 + 4u != g.W);
    if (fast) {
        const uint32_t s = own[w];
        const uint32_t nx = other[w];
        const uint32_t nxs = p == 0 ? window4(other, h0 - 1u) : window4(other, h0 + 1u);
        const uint32_t nym = window4(other, h0 - g.W);
        const uint32_t nyp = window4(other, h0 + g.W);
        uint32_t nzm = 0u, nzp = 0u;
        if (DIMS == 3) {
            nzm = window4(other, h0 - g.L * g.W);
            nzp = window4(other, h0 + g.L * g.W);
        }
        const uint32_t D = disagreements<DIMS>(s, nx, nxs, nym, nyp, nzm, nzp);
        uint32_t X;
        if (RULE == kRuleMultiHit) {
            X = multihit_word<DIMS>(D, w, a);
        } else {
            const Philox4 u = philox4x32_10(w, a.t, (uint32_t)a.c, kTagSweep, a.key0, a.key1);
            X = flip_mask<DIMS, RULE>(D, u, a);
        }
        const uint32_t snew = s ^ (X & kByteFlip);
        own[w] = snew;
        if (MEASURE) {
            m_sum = add_bytes(snew, m_sum);
            if (a.c == 1) {
                constexpr uint32_t q2 = 4u * DIMS * kByteOnes;
                const uint32_t Dn = (D & ~X) | ((q2 - D) & X);
                e_acc = add_bytes(Dn, e_acc - 4 * 2 * DIMS);
            }
        }
        return;
    }
    // per-site path
    int8_t* own_b = static_cast<int8_t*>(a.own);
    int s_val[4], d_val[4];
    bool valid[4], need = false;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint32_t h = h0 + (uint32_t)j;
        valid[j] = h < g.half;
        s_val[j] = 1;
        d_val[j] = DIMS;
        if (!valid[j]) continue;
        const uint32_t r = g.by_W.quot(h);
        const uint32_t xh = h - r * g.W;
        uint32_t y = r, z = 0;
        if (DIMS == 3) {
            z = g.by_L.quot(r);
            y = r - z * g.L;
        }
        const int pp = (a.c + (int)y + (int)z) & 1;
        const uint32_t x = 2u * xh + (uint32_t)pp;
        const uint32_t xm = (x == 0u ? g.L - 1u : x - 1u) >> 1;
        const uint32_t xp = (x + 1u == g.L ? 0u : x + 1u) >> 1;
        const uint32_t plane = z * g.L;
        const uint32_t rym = plane + (y == 0u ? g.L - 1u : y - 1u);
        const uint32_t ryp = plane + (y + 1u == g.L ? 0u : y + 1u);
        const int s = own_b[h];
        int hsum = other_b[r * g.W + xm] + other_b[r * g.W + xp] + other_b[rym * g.W + xh] +
                   other_b[ryp * g.W + xh];
        if (DIMS == 3) {
            const uint32_t rzm = (z == 0u ? g.L - 1u : z - 1u) * g.L + y;
            const uint32_t rzp = (z + 1u == g.L ? 0u : z + 1u) * g.L + y;
            hsum += other_b[rzm * g.W + xh] + other_b[rzp * g.W + xh];
        }
        s_val[j] = s;
        d_val[j] = (2 * DIMS - s * hsum) >> 1;  // k = s*h = 2*(dims - d)
        if (d_val[j] < DIMS || RULE == kRuleHeatBath) need = true;
    }
    if (RULE == kRuleMultiHit) {
        int d_cur[4], flips[4] = {0, 0, 0, 0};
#pragma unroll
        for (int j = 0; j < 4; ++j) d_cur[j] = d_val[j];
#pragma unroll 1
        for (int m = 0; m < a.hits; ++m) {
            bool any = false;
#pragma unroll
            for (int j = 0; j < 4; ++j) any |= valid[j] && d_cur[j] < DIMS;
            uint32_t uu[4] = {0u, 0u, 0u, 0u};
            if (any) {
                const Philox4 q = philox4x32_10(w, a.t, (uint32_t)a.c + 2u * (uint32_t)m,
                                                kTagSweep, a.key0, a.key1);
                uu[0] = q.w0;
                uu[1] = q.w1;
                uu[2] = q.w2;
                uu[3] = q.w3;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                bool f = d_cur[j] >= DIMS;
                if (!f) {
                    const int dj = d_cur[j];
                    const uint32_t t = DIMS == 2 ? (dj == 0 ? a.thr[1] : a.thr[0])
                                                 : (dj == 0 ? a.thr[2] : (dj == 1 ? a.thr[1] : a.thr[0]));
                    f = uu[j] < t;
                }
                if (f) {
                    d_cur[j] = 2 * DIMS - d_cur[j];
                    flips[j] ^= 1;
                }
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (!valid[j]) continue;
            const int sn = flips[j] ? -s_val[j] : s_val[j];
            if (flips[j]) own_b[h0 + j] = (int8_t)sn;
            if (MEASURE) {
                m_sum += sn;
                if (a.c == 1) e_acc += 2 * d_cur[j] - 2 * DIMS;
            }
        }
        return;
    }
    uint32_t u[4] = {0u, 0u, 0u, 0u};
    if (need) {
        const Philox4 q = philox4x32_10(w, a.t, (uint32_t)a.c, kTagSweep, a.key0, a.key1);
        u[0] = q.w0;
        u[1] = q.w1;
        u[2] = q.w2;
        u[3] = q.w3;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (!valid[j]) continue;
        bool flip;
        if (RULE == kRuleHeatBath) {
            flip = u[j] < heatbath_threshold<DIMS>(d_val[j], a);
        } else {
            flip = d_val[j] >= DIMS;
            if (!flip) {
                const uint32_t t = DIMS == 2 ? (d_val[j] == 0 ? a.thr[1] : a.thr[0])
                                             : (d_val[j] == 0 ? a.thr[2] : (d_val[j] == 1 ? a.thr[1] : a.thr[0]));
                flip = u[j] < t;
            }
        }
        const int sn = flip ? -s_val[j] : s_val[j];
        if (flip) own_b[h0 + j] = (int8_t)sn;
        if (MEASURE) {
            m_sum += sn;
            if (a.c == 1) {
                const int dn = flip ? 2 * DIMS - d_val[j] : d_val[j];
                e_acc += 2 * dn - 2 * DIMS;
            }
        }
    }
}

// The draws of the four Philox groups g0 .. g0 + 3 (one 16-byte vector) ...
__device__ __forceinline__ void vec_draws(uint32_t g0, const PassArgs& a, uint32_t c2,
                                          PhiloxRuns<1>& ps) {
    const uint32_t base[1] = {g0};
    ps.first_round(base, a.t, c2, kTagSweep, a.key0, a.key1);
#pragma unroll
    for (int r = 1; r < 10; ++r) ps.next_round();
}
// ... and their tests (count_word).
template <int DIMS, int RULE>
__device__ __forceinline__ void vec_counts(uint32_t g0, const PassArgs& a, uint32_t c2,
                                           uint32_t (&cnt)[4]) {
    PhiloxRuns<1> ps;
    vec_draws(g0, a, c2, ps);
#pragma unroll
    for (int w = 0; w < 4; ++w) cnt[w] = count_word<DIMS, RULE>(ps.result(w), a);
}

// Update the 16 sites of one 16-byte vector (Philox groups g0..g0+3); flips(w, D)
// is the flip mask of word w in the first trial.  Accumulates the sum of the new spins (m_sum) and,
// in the white pass, sum_j 2*d_new_j (e_acc), over the bytes set in `counted`.
template <int DIMS, bool MEASURE, int RULE, typename F>
__device__ __forceinline__ uint4 update_vec(const uint4& s, const uint4& x, const uint4& xs,
                                            const uint4& ym, const uint4& yp, const uint4& zm,
                                            const uint4& zp, uint32_t g0, F&& flips,
                                            const uint4& counted, const PassArgs& a, int& e_acc,
                                            int& m_sum) {
    const uint32_t cv[4] = {counted.x, counted.y, counted.z, counted.w};
    const uint32_t sv[4] = {s.x, s.y, s.z, s.w};
    uint32_t D[4], X[4];
    D[0] = disagreements<DIMS>(s.x, x.x, xs.x, ym.x, yp.x, zm.x, zp.x);
    D[1] = disagreements<DIMS>(s.y, x.y, xs.y, ym.y, yp.y, zm.y, zp.y);
    D[2] = disagreements<DIMS>(s.z, x.z, xs.z, ym.z, yp.z, zm.z, zp.z);
    D[3] = disagreements<DIMS>(s.w, x.w, xs.w, ym.w, yp.w, zm.w, zp.w);
    // one trial, or a.hits in a row with the neighbours fixed
    const int hits = RULE == kRuleMultiHit ? a.hits : 1;
    uint32_t Dc[4];
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        X[w] = flips(w, D[w]);
        constexpr uint32_t q2 = 4u * DIMS * kByteOnes;
        if (RULE == kRuleMultiHit) Dc[w] = (D[w] & ~X[w]) | ((q2 - D[w]) & X[w]);
    }
    if (RULE == kRuleMultiHit) {
#pragma unroll 1
        for (int m = 1; m < hits; ++m) {
            uint32_t cnt[4];
            vec_counts<DIMS, RULE>(g0, a, (uint32_t)a.c + 2u * (uint32_t)m, cnt);
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                constexpr uint32_t q2 = 4u * DIMS * kByteOnes;
                const uint32_t Y = flip_mask(Dc[w], cnt[w]);
                Dc[w] = (Dc[w] & ~Y) | ((q2 - Dc[w]) & Y);
                X[w] ^= Y;
            }
        }
    }
    uint32_t out[4];
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        out[w] = sv[w] ^ (X[w] & kByteFlip);
        if (MEASURE) {
            m_sum = add_bytes(out[w] & cv[w], m_sum);
            if (a.c == 1) {
                // 2*d_new = 2*(2 dims) - 2*d where flipped
                constexpr uint32_t q2 = 4u * DIMS * kByteOnes;
                const uint32_t Dn = (D[w] & ~X[w]) | ((q2 - D[w]) & X[w]);
                e_acc = add_bytes(Dn & cv[w], e_acc);
            }
        }
    }
    return make_uint4(out[0], out[1], out[2], out[3]);
}


// 16 bytes of the other colour at byte offset o (any alignment), in two steps:
// the two aligned 16-byte loads (the same one twice where o is aligned), so that
// all of a vector's loads are under way before the first is used, and the byte
// shift.  The shift o mod 16 is the same for a whole lattice and direction (it
// depends only on W, L and the direction), so the switch does not diverge.
// FROM_BEFORE: o may be -15 .. -1 (as unsigned), a window that starts before the
// array; the bytes before it are whatever the array starts with.
struct Window16 {
    uint4 lo, hi;
    uint32_t r;
    __device__ __forceinline__ uint4 get() const {
        if (r == 0u) return lo;
        const uint32_t b = 8u * (r & 3u);
        uint32_t w0, w1, w2, w3, w4;
        switch (r >> 2) {
            case 0: w0 = lo.x; w1 = lo.y; w2 = lo.z; w3 = lo.w; w4 = hi.x; break;
            case 1: w0 = lo.y; w1 = lo.z; w2 = lo.w; w3 = hi.x; w4 = hi.y; break;
            case 2: w0 = lo.z; w1 = lo.w; w2 = hi.x; w3 = hi.y; w4 = hi.z; break;
            default: w0 = lo.w; w1 = hi.x; w2 = hi.y; w3 = hi.z; w4 = hi.w; break;
        }
        return make_uint4(__funnelshift_r(w0, w1, b), __funnelshift_r(w1, w2, b),
                          __funnelshift_r(w2, w3, b), __funnelshift_r(w3, w4, b));
    }
};
template <bool FROM_BEFORE = false>
__device__ __forceinline__ Window16 load_window(const uint4* other16, uint32_t o) {
    Window16 w;
    w.r = o & 15u;
    const bool before = FROM_BEFORE && o >= 0xFFFFFFF0u;
    const uint32_t b = before ? 0u : o >> 4;
    w.lo = other16[b];
    w.hi = other16[before || w.r == 0u ? b : b + 1u];
    return w;
}

// Byte j of word i of the mask is 0xFF iff 4 i + j >= n (n = 0..16 or more).
__device__ __forceinline__ uint4 bytes_from(int n) {
    const int s = 8 * n;
    return make_uint4(__funnelshift_lc(0u, 0xFFFFFFFFu, (uint32_t)s),
                      __funnelshift_lc(0u, 0xFFFFFFFFu, (uint32_t)max(s - 32, 0)),
                      __funnelshift_lc(0u, 0xFFFFFFFFu, (uint32_t)max(s - 64, 0)),
                      __funnelshift_lc(0u, 0xFFFFFFFFu, (uint32_t)max(s - 96, 0)));
}
__device__ __forceinline__ uint4 select4(const uint4& m, const uint4& t, const uint4& f) {
    return make_uint4((m.x & t.x) | (~m.x & f.x), (m.y & t.y) | (~m.y & f.y),
                      (m.z & t.z) | (~m.z & f.z), (m.w & t.w) | (~m.w & f.w));
}

// Update the 16 sites of vector v (half indices 16v..16v+15, Philox groups
// 4v..4v+3) of the int8 colour array.  With W >= 16 a vector holds sites of one
// row, or the end of one (part A) and the start of the next (part B; none behind
// the last row); shorter rows go word by word.  Its y- and z-neighbours are
// 16-byte windows of the other colour at an offset that is the same for both parts but
// where one of them wraps; its x-neighbours are the bytes before or behind, by
// each part's parity, with the bytes that wrap at a row's ends put in singly.
// Every vector takes this one path, and all its loads come first: word by word
// (int8_word) the few at the row ends and edges held the whole pass up, alone
// (2D L = 1000 7.6 -> 2.7, 3D L = 202 32.4 -> 9.2 us a pass).  Accumulates
// m_sum and, in the white pass, e_acc as int8_word does.
template <int DIMS, bool MEASURE, int RULE>
__device__ __forceinline__ void int8_vec(const PassArgs& a, const WordGeom& g, uint32_t v,
                                         int& e_acc, int& m_sum) {
    const uint32_t h0 = 16u * v, W = g.W;
    if (W < 16u) {  // short rows: word by word
#pragma unroll 1
        for (uint32_t w = 4u * v; w < 4u * v + 4u; ++w)
            if (4u * w < g.half) int8_word<DIMS, MEASURE, RULE>(a, g, w, e_acc, m_sum);
        return;
    }
    const uint32_t r0 = g.by_W.quot(h0);
    const uint32_t xh0 = h0 - r0 * W;
    uint32_t y0 = r0, z0 = 0;
    if (DIMS == 3) {
        z0 = g.by_L.quot(r0);
        y0 = r0 - z0 * g.L;
    }
    const uint32_t left = W - xh0;  // sites of row r0 from here on
    const bool ends = left < 16u;   // the row ends inside the vector
    const bool two = ends && r0 + 1u < g.rows;
    // part B's row
    uint32_t yb = y0 + 1u, zb = z0;
    if (yb == g.L) {
        yb = 0u;
        ++zb;
    }
    const bool edge = two && (y0 == 0u || yb == 0u || yb + 1u == g.L);  // one part wraps
    const uint4* other16 = static_cast<const uint4*>(a.other);
    const uint32_t* other32 = static_cast<const uint32_t*>(a.other);
    const uint8_t* other8 = static_cast<const uint8_t*>(a.other);
    uint4* own16 = static_cast<uint4*>(a.own);
    const uint32_t row = r0 * W;
    const uint32_t plane = g.L * W, y_wrap = plane - W, z_wrap = (g.L - 1u) * plane;
    const uint4 zero4 = make_uint4(0u, 0u, 0u, 0u), ones4 = make_uint4(~0u, ~0u, ~0u, ~0u);
    const uint4 s = own16[v];
    const uint4 nx = other16[v];
    const Window16 wym = load_window(other16, y0 == 0u ? h0 + y_wrap : h0 - W);
    const Window16 wyp = load_window(other16, y0 + 1u == g.L ? h0 - y_wrap : h0 + W);
    Window16 wzm{zero4, zero4, 0u}, wzp{zero4, zero4, 0u};
    if (DIMS == 3) {
        wzm = load_window(other16, z0 == 0u ? h0 + z_wrap : h0 - plane);
        wzp = load_window(other16, z0 + 1u == g.L ? h0 - z_wrap : h0 + plane);
    }
    const uint32_t word_before = other32[v == 0u ? 0u : 4u * v - 1u];
    const uint32_t word_behind = other32[4u * v + 4u];
    const uint32_t row_first = other8[row];
    const uint32_t row_last = other8[row + W - 1u];
    const uint32_t next_last = other8[row + (two ? 2u * W : W) - 1u];
    // the draws while the loads are under way
    uint32_t cnt[4];
    vec_counts<DIMS, RULE>(4u * v, a, (uint32_t)a.c, cnt);
    const uint4 part_b = ends ? bytes_from((int)left) : zero4;
    uint4 nym = wym.get(), nyp = wyp.get(), nzm = zero4, nzp = zero4;
    if (DIMS == 3) {
        nzm = wzm.get();
        nzp = wzp.get();
    }
    if (edge) {  // part B's own windows (they may start up to 15 bytes before the first row)
        const Window16 bym = load_window<true>(other16, h0 + (yb == 0u ? y_wrap : 0u - W));
        const Window16 byp =
            load_window<true>(other16, h0 + (yb + 1u == g.L ? 0u - y_wrap : W));
        Window16 bzm = wzm, bzp = wzp;
        if (DIMS == 3) {
            bzm = load_window<true>(other16, h0 + (zb == 0u ? z_wrap : 0u - plane));
            bzp = load_window<true>(other16, h0 + (zb + 1u == g.L ? 0u - z_wrap : plane));
        }
        nym = select4(part_b, bym.get(), nym);
        nyp = select4(part_b, byp.get(), nyp);
        if (DIMS == 3) {
            nzm = select4(part_b, bzm.get(), nzm);
            nzp = select4(part_b, bzp.get(), nzp);
        }
    }
    const int pa = (a.c + (int)y0 + (int)z0) & 1, pb = (a.c + (int)yb + (int)zb) & 1;
    // part A's x-neighbours, and part B's where there is one: the bytes before
    // (byte j <- byte j - 1) or behind (byte j <- byte j + 1)
    const uint32_t prev = xh0 == 0u ? row_last << 24 : word_before;
    const uint32_t next = left == 16u ? row_first : word_behind;
    const uint4 before =
        make_uint4(__funnelshift_l(prev, nx.x, 8), __funnelshift_l(nx.x, nx.y, 8),
                   __funnelshift_l(nx.y, nx.z, 8), __funnelshift_l(nx.z, nx.w, 8));
    const uint4 behind =
        make_uint4(__funnelshift_r(nx.x, nx.y, 8), __funnelshift_r(nx.y, nx.z, 8),
                   __funnelshift_r(nx.z, nx.w, 8), __funnelshift_r(nx.w, next, 8));
    uint4 nxs = pa ? behind : before;
    if (ends) {
        if (pa == 1) {  // part A's last site wraps to its row's first
            const uint32_t f = row_first * kByteOnes;
            nxs = select4(bytes_from((int)left - 1), make_uint4(f, f, f, f), nxs);
        }
        nxs = select4(part_b, pb ? behind : before, nxs);
        if (pb == 0) {  // part B's first site wraps to its row's last
            const uint32_t l = next_last * kByteOnes;
            const uint4 m = bytes_from((int)left + 1);
            nxs = select4(make_uint4(part_b.x & ~m.x, part_b.y & ~m.y, part_b.z & ~m.z,
                                     part_b.w & ~m.w),
                          make_uint4(l, l, l, l), nxs);
        }
    }
    // past the last row's end: the array's padding, which counts for nothing
    uint4 counted = ones4;
    int n_sites = 16;
    if (MEASURE && ends && !two) {
        counted = make_uint4(~part_b.x, ~part_b.y, ~part_b.z, ~part_b.w);
        n_sites = (int)left;
    }
    int e_vec = 0;
    auto flips = [&](int w, uint32_t D) { return flip_mask(D, cnt[w]); };
    own16[v] = update_vec<DIMS, MEASURE, RULE>(s, nx, nxs, nym, nyp, nzm, nzp, 4u * v, flips,
                                               counted, a, e_vec, m_sum);
    if (MEASURE && a.c == 1) e_acc += e_vec - n_sites * 2 * DIMS;
}

// ----------------------------------------------------------------------------
// Bit-packed body: one 32-site word per call; see sweep_bitpack.cu for the
// layout.
// ----------------------------------------------------------------------------
struct Counts {
    uint32_t always, eq0, eq1, eq2;
};

__device__ __forceinline__ Counts count2(uint32_t a, uint32_t b, uint32_t c, uint32_t e) {
    const uint32_t s1 = a ^ b, c1 = a & b;
    const uint32_t s2 = c ^ e, c2 = c & e;
    const uint32_t b0 = s1 ^ s2, c3 = s1 & s2;
    const uint32_t always = c1 | c2 | c3;  // d = b0 + 2 (c1 + c2 + c3) >= 2
    return Counts{always, ~(b0 | always), b0 & ~always, 0u};
}

__device__ __forceinline__ Counts count3(uint32_t a, uint32_t b, uint32_t c, uint32_t d,
                                         uint32_t e, uint32_t f) {
    const uint32_t s1 = a ^ b ^ c, k1 = (a & b) | (c & (a ^ b));
    const uint32_t s2 = d ^ e ^ f, k2 = (d & e) | (f & (d ^ e));
    const uint32_t bit0 = s1 ^ s2, k0 = s1 & s2;
    const uint32_t bit1 = k1 ^ k2 ^ k0, bit2 = (k1 & k2) | (k0 & (k1 ^ k2));
    const uint32_t always = bit2 | (bit1 & bit0);  // d = bit0 + 2 bit1 + 4 bit2 >= 3
    const uint32_t low = ~(bit2 | bit1);
    return Counts{always, low & ~bit0, low & bit0, bit1 & ~bit0 & ~bit2};
}

// Bit-sliced number of disagreeing neighbours d = d0 + 2 d1 + 4 d2 of each
// of the 32 sites (the heat-bath rule needs every value of d).
struct Digits {
    uint32_t d0, d1, d2;
};

__device__ __forceinline__ Digits digits2(uint32_t a, uint32_t b, uint32_t c, uint32_t e) {
    const uint32_t s1 = a ^ b, c1 = a & b;
    const uint32_t s2 = c ^ e, c2 = c & e;
    const uint32_t c3 = s1 & s2;  // d = (s1 ^ s2) + 2 (c1 + c2 + c3)
    return Digits{s1 ^ s2, c1 ^ c2 ^ c3, (c1 & c2) | (c3 & (c1 ^ c2))};
}

__device__ __forceinline__ Digits digits3(uint32_t a, uint32_t b, uint32_t c, uint32_t d,
                                          uint32_t e, uint32_t f) {
    const uint32_t s1 = a ^ b ^ c, k1 = (a & b) | (c & (a ^ b));
    const uint32_t s2 = d ^ e ^ f, k2 = (d & e) | (f & (d ^ e));
    const uint32_t k0 = s1 & s2;  // d = (s1 ^ s2) + 2 (k1 + k2 + k0)
    return Digits{s1 ^ s2, k1 ^ k2 ^ k0, (k1 & k2) | (k0 & (k1 ^ k2))};
}

// Thresholds of a rule: the Metropolis dims, or the heat bath's 2 dims + 1.
template <int DIMS, int RULE>
constexpr int kThresholds = RULE == kRuleHeatBath ? 2 * DIMS + 1 : DIMS;

// What bounds the drawing passes is instructions issued.  Measured on the
// generator and these tests alone (cycles per scheduler and Philox call, any
// occupancy from two to eight CTAs per SM): a 32x32 -> 64-bit product holds the
// issue port ~3.6 cycles, a 32-bit multiply-add 2 and everything else 1,
// whichever pipe it runs on.  Ten rounds cost 82.5.  Selecting each site's
// threshold and comparing took 33 more (as compiled); every draw against every
// threshold with mark_below takes 15 (2D), and choose_answer picks for 32 sites
// at once.  2D L = 8192: 29.1 -> 24.6 us per pass (1.36e12 site updates/s).
// Tests as saturating fp32 multiply-adds, off the integer pipes, took 26: a
// multiply-add costs an issue slot like a compare.
//
// The draws of the Philox groups g0 .. g0 + 7 against all N thresholds: bit b of
// A[n] is set iff draw b (word b & 3 of group g0 + (b >> 2)) lies below
// threshold n.  Four calls at a time; of the second four only as many as `second`
// says (0, 1 or 4), the other bits stay clear.
template <int N>
__device__ __forceinline__ void word_tests(uint32_t g0, const PassArgs& a, uint32_t c2, int second,
                                           uint32_t (&A)[N]) {
#pragma unroll
    for (int n = 0; n < N; ++n) A[n] = 0u;
    static_for<2>([&](auto half) {
        constexpr int h = decltype(half)::value;
        if (h == 1 && second < 4) return;
        PhiloxRuns<1> ps;
        const uint32_t base[1] = {g0 + 4u * h};
        ps.first_round(base, a.t, c2, kTagSweep, a.key0, a.key1);
#pragma unroll
        for (int r = 1; r < 10; ++r) ps.next_round();
        static_for<16>([&](auto bit) {
            constexpr int b = decltype(bit)::value, j = b & 3;
            const Philox4 u = ps.result(b >> 2);
            const uint32_t w = j == 0 ? u.w0 : j == 1 ? u.w1 : j == 2 ? u.w2 : u.w3;
#pragma unroll
            for (int n = 0; n < N; ++n) mark_below<(1u << (16 * h + b))>(A[n], w, a.thr[n]);
        });
    });
    if (second == 1) {
        const Philox4 u = philox4x32_10(g0 + 4u, a.t, c2, kTagSweep, a.key0, a.key1);
        static_for<4>([&](auto bit) {
            constexpr int j = decltype(bit)::value;
            const uint32_t w = j == 0 ? u.w0 : j == 1 ? u.w1 : j == 2 ? u.w2 : u.w3;
#pragma unroll
            for (int n = 0; n < N; ++n) mark_below<(1u << (16 + j))>(A[n], w, a.thr[n]);
        });
    }
}

// Each site's answer for the threshold of its own number of disagreeing
// neighbours, from the answers A[n] for every threshold, 32 sites at once.
template <int DIMS>
__device__ __forceinline__ uint32_t choose_answer(const Counts& k, const uint32_t (&A)[DIMS]) {
    if constexpr (DIMS == 2) return (k.eq0 & A[1]) | (k.eq1 & A[0]);
    else return (k.eq0 & A[2]) | (k.eq1 & A[1]) | (k.eq2 & A[0]);
}
template <int DIMS>
__device__ __forceinline__ uint32_t choose_answer(const Digits& k,
                                                  const uint32_t (&A)[2 * DIMS + 1]) {
    const uint32_t a01 = (k.d0 & A[1]) | (~k.d0 & A[0]), a23 = (k.d0 & A[3]) | (~k.d0 & A[2]);
    const uint32_t lo = (k.d1 & a23) | (~k.d1 & a01);
    uint32_t hi = A[4];
    if constexpr (DIMS == 3) {
        const uint32_t a45 = (k.d0 & A[5]) | (~k.d0 & A[4]);
        hi = (k.d1 & A[6]) | (~k.d1 & a45);
    }
    return (k.d2 & hi) | (~k.d2 & lo);
}

// How the words of a lattice draw (the whole warp takes part in a word's
// tests, each lane for its own word).
constexpr int kDrawAligned = 0;  // every row starts on a Philox group
constexpr int kDrawRagged = 1;   // rows start anywhere in a group
// Words a warp takes at a time.
template <int DRAW>
constexpr uint32_t kWarpWords = DRAW == kDrawRagged ? 31u : 32u;

// The tests of a packed word whose 32 bits are the half indices hbase + b: bit b
// of A[n] says whether site b's draw, word (hb & 3) of Philox group hb >> 2, lies
// below threshold n.  A row that starts
// inside a group (hbase & 3 = M != 0) needs nine groups' draws 0..35 and uses
// draws M .. M + 31: the tests stay at draw positions, the same code for every
// M, the last four positions are the next lane's first four (its word starts
// with the ninth group: words follow one another in h, and where a row's last
// word is shorter than 32 - M sites the ninth group is not needed), and one
// funnel shift per threshold moves the answers to their sites.  So a ragged
// word costs eight calls like an aligned one; the last lane of the warp only
// lends its draws (packed_words).  Against five calls per half, with the code
// compiled per M and the rows grouped by M, and with divisions for an item's
// place: 3D L = 202 11.0 -> 8.6 us per pass; a joint pass of 256 mixed lattices
// 47 -> 39 us.
template <int DIMS, int RULE, int DRAW>
__device__ __forceinline__ void packed_draws(uint32_t hbase, int second, const PassArgs& a,
                                             uint32_t c2,
                                             uint32_t (&A)[kThresholds<DIMS, RULE>]) {
    constexpr int N = kThresholds<DIMS, RULE>;
    word_tests<N>(hbase >> 2, a, c2, second, A);
    if constexpr (DRAW == kDrawRagged) {
#pragma unroll
        for (int n = 0; n < N; ++n) {
            const uint32_t next = __shfl_down_sync(0xffffffffu, A[n], 1);
            A[n] = __funnelshift_r(A[n], next, hbase & 3u);
        }
    }
}

// The geometry of a packed lattice's words.
struct PackedGeom {
    uint32_t items;    // words per colour
    FastDiv words, L;  // words per half row, L
    PackedGeom() = default;
    __host__ __device__ __forceinline__ PackedGeom(uint32_t W, uint32_t L_, uint32_t rows)
        : words((W + 31u) >> 5), L(L_) {
        items = rows * words.d;
    }
};

// One packed word and its neighbours, as loaded.
struct PackedWord {
    uint32_t at;              // its index in the colour array
    uint32_t s, o, x, ym, yp, zm, zp;  // x: the word that holds the outer x-neighbour
    uint32_t valid;           // the word's sites
    uint32_t hbase;           // the half index of bit 0
    uint32_t edge;            // how x joins: 0 inside the row, else it wraps (see x_neighbours)
    int p;                    // 0: bit b <- neighbour xh - 1, 1: xh + 1
    bool mine;                // this lane stores the word
};

// The word of x-neighbours: o shifted by one site, the site that enters taken
// from x: inside a row its bit 31 (p = 0) or bit 0 (p = 1); where the row wraps,
// the row's last valid bit (p = 0, edge - 1 the shift that brings it to bit 31)
// or its first, entering at the word's last valid bit (p = 1).
__device__ __forceinline__ uint32_t x_neighbours(const PackedWord& w) {
    if (w.p == 0) return __funnelshift_l(w.edge ? w.x << (w.edge - 1u) : w.x, w.o, 1);
    if (w.edge == 0u) return __funnelshift_r(w.o, w.x, 1);
    const uint32_t top = w.valid ^ (w.valid >> 1);
    return ((w.o >> 1) & ~top) | ((w.x & 1u) ? top : 0u);
}

// The rule applied to one packed word, given its tests (of the first trial; in
// `later`, if set, those of trials 1 .. n_later, one word a thread of the block
// per trial and threshold), then the store and the word's share of E and M.  With
// ragged draws the whole warp takes part.
template <int DIMS, bool MEASURE, int RULE, int DRAW>
__device__ __forceinline__ void packed_update(const PassArgs& a, const PackedWord& w,
                                              uint32_t (&A)[kThresholds<DIMS, RULE>], int second,
                                              int& e_acc, int& m_acc,
                                              const uint32_t* later = nullptr, int n_later = 0) {
    const uint32_t s = w.s, sh = x_neighbours(w);
    uint32_t flip;
    if constexpr (RULE == kRuleHeatBath) {
        const Digits k = DIMS == 2 ? digits2(s ^ w.o, s ^ sh, s ^ w.ym, s ^ w.yp)
                                   : digits3(s ^ w.o, s ^ sh, s ^ w.ym, s ^ w.yp, s ^ w.zm,
                                             s ^ w.zp);
        flip = choose_answer<DIMS>(k, A);
    } else {
        // one Metropolis trial, or a.hits in a row with the neighbours fixed
        const int hits = RULE == kRuleMultiHit ? a.hits : 1;
        uint32_t cur = s;
#pragma unroll 1
        for (int m = 0;;) {
            Counts k;
            if (DIMS == 2) {
                k = count2(cur ^ w.o, cur ^ sh, cur ^ w.ym, cur ^ w.yp);
            } else {
                k = count3(cur ^ w.o, cur ^ sh, cur ^ w.ym, cur ^ w.yp, cur ^ w.zm, cur ^ w.zp);
            }
            cur ^= k.always | choose_answer<DIMS>(k, A);
            if (++m >= hits) break;
            if (RULE == kRuleMultiHit && m <= n_later) {
#pragma unroll
                for (int n = 0; n < kThresholds<DIMS, RULE>; ++n)
                    A[n] = later[((m - 1) * kThresholds<DIMS, RULE> + n) * (int)blockDim.x];
                continue;
            }
            packed_draws<DIMS, RULE, DRAW>(w.hbase, second, a, (uint32_t)a.c + 2u * (uint32_t)m, A);
        }
        flip = cur ^ s;
    }
    const uint32_t snew = s ^ (flip & w.valid);
    if (!w.mine) return;
    static_cast<uint32_t*>(a.own)[w.at] = snew;
    if (MEASURE) {
        const int nb = __popc(w.valid);
        m_acc += 2 * __popc(snew & w.valid) - nb;
        if (a.c == 1) {
            int dsum = __popc((snew ^ w.o) & w.valid) + __popc((snew ^ sh) & w.valid) +
                       __popc((snew ^ w.ym) & w.valid) + __popc((snew ^ w.yp) & w.valid);
            if (DIMS == 3)
                dsum += __popc((snew ^ w.zm) & w.valid) + __popc((snew ^ w.zp) & w.valid);
            e_acc += 2 * dsum - nb * 2 * DIMS;
        }
    }
}

// A warp's words of the packed colour array: items first .. first + 31, the
// lane's own at first + lane.  A half row of W sites takes nq = ceil(W / 32)
// words; bit b of word q is half column xh = 32q + b (valid when xh < W; the
// other bits of a row's last word stay 0 and never flip).  With ragged draws
// lane 31 only lends its draws, for lane 30's last sites, and its word is the
// first of the next step; a lane past the end draws for the row after the last.
struct PackedPlace {
    uint32_t r, q;
    uint32_t hbase;
    bool mine;
};

template <int DRAW>
__device__ __forceinline__ PackedPlace packed_place(const PackedGeom& g, uint32_t W,
                                                    uint32_t first) {
    const uint32_t lane = threadIdx.x & 31u, item = first + lane;
    PackedPlace p;
    p.r = g.words.quot(item);
    p.q = item - p.r * g.words.d;
    p.hbase = p.r * W + 32u * p.q;
    p.mine = item < g.items && lane < kWarpWords<DRAW>;
    if (item >= g.items) {  // loads something, keeps nothing
        p.r = 0u;
        p.q = 0u;
    }
    return p;
}

template <int DIMS>
__device__ __forceinline__ PackedWord packed_load(const PassArgs& a, const PackedGeom& g,
                                                  const PackedPlace& pl) {
    const uint32_t W = (uint32_t)a.W, L = (uint32_t)a.L, nq = g.words.d;
    const uint32_t r = pl.r, q = pl.q;
    uint32_t y = r, z = 0;
    if (DIMS == 3) {
        z = g.L.quot(r);
        y = r - z * L;
    }
    PackedWord w;
    w.at = r * nq + q;
    w.mine = pl.mine;
    w.hbase = pl.hbase;
    w.p = (a.c + (int)y + (int)z) & 1;
    const uint32_t nb = W - 32u * q < 32u ? W - 32u * q : 32u;  // valid bits
    w.valid = nb == 32u ? 0xFFFFFFFFu : ((1u << nb) - 1u);
    const uint32_t* at = static_cast<const uint32_t*>(a.other) + w.at;
    // the word with the outer x-neighbour, and the rows (and planes) next to
    // this one, as offsets
    int32_t dx;
    if (w.p == 0) {
        dx = q == 0u ? (int32_t)nq - 1 : -1;
        w.edge = q == 0u ? 32u - ((W - 1u) & 31u) : 0u;
    } else {
        dx = q + 1u == nq ? -(int32_t)q : 1;
        w.edge = q + 1u == nq ? 1u : 0u;
    }
    const int32_t up = y == 0u ? (int32_t)((L - 1u) * nq) : -(int32_t)nq;
    const int32_t down = y + 1u == L ? -(int32_t)((L - 1u) * nq) : (int32_t)nq;
    w.o = *at;
    w.x = at[dx];
    w.ym = at[up];
    w.yp = at[down];
    w.zm = w.zp = 0u;
    if (DIMS == 3) {
        const int32_t plane = (int32_t)(L * nq), wrap = (int32_t)((L - 1u) * L * nq);
        w.zm = at[z == 0u ? wrap : -plane];
        w.zp = at[z + 1u == L ? -wrap : plane];
    }
    w.s = static_cast<const uint32_t*>(a.own)[w.at];
    return w;
}

// How many of a word's second four calls any of its sites needs: rows of one word
// that start at most 3 draws into a group (2 where W is even, 0 where W % 4 == 0).
// (64 of 3D L = 30 in a CTA each: 14.1 us a pass with eight calls, 10.0 with five.)
__device__ __forceinline__ int packed_second(const PassArgs& a) {
    const int last = a.W + (a.W % 4 == 0 ? 0 : a.W % 2 == 0 ? 2 : 3);
    return last <= 16 ? 0 : last <= 20 ? 1 : 4;
}

// One step of a warp, loads first: their latency hides behind the draws.
template <int DIMS, bool MEASURE, int RULE, int DRAW>
__device__ __forceinline__ void packed_words(const PassArgs& a, const PackedGeom& g,
                                             uint32_t first, int& e_acc, int& m_acc) {
    const PackedWord w =
        packed_load<DIMS>(a, g, packed_place<DRAW>(g, (uint32_t)a.W, first));
    uint32_t A[kThresholds<DIMS, RULE>];
    __syncwarp();
    packed_draws<DIMS, RULE, DRAW>(w.hbase, packed_second(a), a, (uint32_t)a.c, A);
    packed_update<DIMS, MEASURE, RULE, DRAW>(a, w, A, packed_second(a), e_acc, m_acc);
}

}  // namespace ising
