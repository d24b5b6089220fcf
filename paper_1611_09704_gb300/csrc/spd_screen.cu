// spd_screen.cu -- the screen of the candidate search (Sec. 2.3-2.4).
//
// On a plane with few pulses almost no start can reach the threshold, and the
// search kernel (spd_search_kernel.cuh) spends its time on what it does for
// every tile: centred samples, prefixes and window sums in shared memory, the
// table of prefix maxima, a bound per width group.  The screen does only what
// is needed to know which units of 16 starts can hold a candidate at all: it
// reads every sample once, through a ring of each warp's own, keeps five numbers per
// block of 16, and makes one test per class of widths.  Tiles with many units
// that pass are listed whole for the search kernel, the units of the others
// one by one for its half-warps (spd_live.cuh).
#include "spd_device.cuh"

namespace spd {

namespace {

constexpr int kScrThreads = 128;
constexpr int kScrWarps = kScrThreads / 32;
constexpr int kScrBufs = 3;         // rounds of samples in shared memory per warp

struct ScreenRange {
    const void *data;
    int64_t stride, n_samp;
    int64_t n_emit;             // starts that can become candidates
    const float *scale, *offset;
    const float2 *mu_tab;
    const int32_t *flags;
    const float *scr_tab;
    uint32_t tile0;             // first launch-wide tile
    int32_t tiles_per_row;
    int32_t vec_ok, per_row;
    uint32_t classes;           // bit c: class c holds an evaluated width
    int32_t reach;              // blocks past a unit that its tests read
    int32_t dense;              // live units up to which a tile is not searched whole
    float threshold;
};

struct ScreenArgs {
    ScreenRange rng[kMaxRanges];
    ScreenLists lists;
    int32_t n_ranges;
    uint32_t n_tiles;
    int32_t units;              // units per search tile
    int32_t ring, mirror;       // rounds of block data kept per warp (a power
                                // of two), and how many of them twice
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const void *src, int bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(dst), "l"(src), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
    asm volatile("cp.async.commit_group;\n" ::: "memory");
}
template <int N> __device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

__device__ __forceinline__ uint4 lds128(uint32_t addr) {
    uint4 r;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];\n"
                 : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
                 : "r"(addr)
                 : "memory");
    return r;
}

// x plus the value O lanes below, where there is such a lane.
template <int O> __device__ __forceinline__ float add_up(float x) {
    asm volatile(
        "{\n .reg .f32 t;\n .reg .pred p;\n"
        " shfl.sync.up.b32 t|p, %0, %1, 0, 0xffffffff;\n @p add.rn.f32 %0, %0, t;\n}\n"
        : "+f"(x)
        : "n"(O));
    return x;
}

// Four 32-bit words of stored samples as 2 (FP32) or 4 pairs.
template <int DT> __device__ __forceinline__ void to_pairs(uint4 r, float2 *v) {
    const uint32_t w[4] = {r.x, r.y, r.z, r.w};
    if constexpr (DT == SPD_F32) {
        v[0] = make_float2(__uint_as_float(w[0]), __uint_as_float(w[1]));
        v[1] = make_float2(__uint_as_float(w[2]), __uint_as_float(w[3]));
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if constexpr (DT == SPD_F16)
                v[e] = __half22float2(*reinterpret_cast<const __half2 *>(&w[e]));
            else
                v[e] = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&w[e]));
        }
    }
}

// Shared bytes of one warp: the samples' buffers, then per block of the ring
// and its mirror the largest and smallest C and two energies, and per 4 and
// per 8 blocks the largest C.
__host__ __device__ inline int screen_warp_bytes(int esz, int rows) {
    return (kScrBufs * 512 * esz + rows * 32 * 16 + rows * 8 * 4 + rows * 4 * 4 + 127) & ~127;
}

// One warp per search tile, with no barrier wider than the warp.  The warp
// walks its tile and the blocks past it that the tests reach in rounds of 32
// blocks of 16 samples.  The samples of a round arrive by asynchronous copies
// two rounds ahead, coalesced, with the 16-byte pieces of a block rotated so
// that the 128-bit reads of a block by its lane meet no bank conflict.  Each
// lane reduces its block to
//   its sum, the largest and smallest of its prefixes (at its 16 starts), and
//   the energy of its two halves;
// a warp scan and the running total turn the prefixes into prefixes C of the
// tile.  A ring in shared memory keeps, per block, the largest and the
// smallest C and the energies, and the largest C per 4 (and 8) blocks.  Its
// first rounds are stored twice, so that a unit and the blocks it reaches lie
// in one piece.
//
// Once the blocks that a unit's windows reach are in the ring the unit (block
// t) is tested, per class of widths:
//   classes 0, 1 (widths 1..8, 9..16): a window starting in the first half of
//     the block lies in 2 (3) half blocks from it, one starting in the second
//     half in as many from there; SNR^2 <= energy x the largest w / sigma_w^2
//     (Cauchy-Schwarz);
//   classes 1 ..: B <= max C over the blocks the windows end in (for classes
//     4 .. the whole groups of 4 or 8 blocks around them) - min C over the
//     starts; SNR <= that (plus the margin for FP32 rounding) x the largest
//     1 / sigma_w.
// A unit is live when some class's bound is not below the threshold (with a
// NaN bound, too).  Windows past the row end do not exist for it.
//
// kTop: the widest class of the launch (3, 5, 6 or 9).  Widths up to 512 have
// their own forms, with fixed reads and, as they reach 32 blocks at most, a lag
// of one round and a ring of two.  kScaled: some range of the launch has a
// scale (a range without one then takes 1 and 0).  Both are arguments of the
// template because a branch between the scaled and the plain samples moved all
// of them at its end: 4096 x 524288 FP32 1.33 ms with the branch and the ring's
// sizes read, 1.20 with these fixed, 1.17 without the branch; the four ranges
// of a batched search (to 64, 128, 256 and 512) 1.17, 1.06 and 1.03 ms; 2048 x
// 524288 FP16 with a scale 0.69, 0.63 and 0.62 ms.
//
// Bound by the plane's one read in FP32: 4096 x 524288 samples (8.6 GB) in
// 1.17 ms, 7.3 TB/s (a plain copy, half of it writes, reaches 6.8); in FP16 by
// instruction issue (3.5 TB/s).  Before, the search kernel took 10.3 and 4.9 ms
// over every tile of the same planes.  A first form of the
// screen, with a CTA over four tiles, a lane's 64 bytes loaded to registers
// and CTA barriers between the prefix passes, took 2.14 ms (the loads touch 16
// lines each); the copies here, with a test written class by class, 1.75 ms
// (407 instructions per warp and round).  72
// registers and 7.9 KB leave 7 CTAs of 4 warps per SM, two rounds in flight in
// each warp: 112 KB per SM.
template <int DT, int kTop, bool kScaled>
__global__ void __launch_bounds__(kScrThreads, 7)
    screen_kernel(const __grid_constant__ ScreenArgs A) {
    using T = typename Elem<DT>::T;
    constexpr int kEsz = sizeof(T);
    constexpr int kPer = 16 / kEsz;             // samples per 16-byte piece
    constexpr int kPieces = 16 / kPer;          // pieces per block
    constexpr int kBuf = 512 * kEsz;            // bytes of a round
    constexpr float kInf = INFINITY;
    extern __shared__ __align__(128) unsigned char s_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t tile = blockIdx.x * kScrWarps + warp;
    if (tile >= A.n_tiles) return;              // the whole warp; no barrier spans warps
    // widths up to 512 reach 32 blocks at most: a lag of one round, a ring of two
    const int ring = kTop > 6 ? A.ring : 2, mirror = kTop > 6 ? A.mirror : 1;
    const int rows = ring + mirror;             // rounds stored, the mirrored ones included
    unsigned char *buf = s_raw + warp * screen_warp_bytes(kEsz, rows);
    float2 *s_e = reinterpret_cast<float2 *>(buf + kScrBufs * kBuf);   // half-block energies
    float *s_x = reinterpret_cast<float *>(s_e + rows * 32);           // largest C
    float *s_n = s_x + rows * 32;                                      // smallest C
    float *s_q4 = s_n + rows * 32;                                     // largest C of 4 blocks
    float *s_q8 = s_q4 + rows * 8;                                     // and of 8

    int ri = 0;
    while (ri + 1 < A.n_ranges && tile >= A.rng[ri + 1].tile0) ++ri;
    const ScreenRange &rd = A.rng[ri];
    const uint32_t lt = tile - rd.tile0;
    const uint32_t row = lt / (uint32_t)rd.tiles_per_row;
    const int64_t t0 = (int64_t)(lt - row * (uint32_t)rd.tiles_per_row) * A.units * kX;
    const int entry = rd.per_row ? (int)row : 0;
    const int64_t emit = min(rd.n_emit - t0, (int64_t)A.units * kX);
    if (emit <= 0 || rd.flags[entry]) return;
    // the tile's limit of live units, not held in a register through the walk (2048
    // x 524288 FP16 with a scale, 46 widths: 619 us with a constant limit, 627 with
    // the launch's read at the end); widths to 256 all have the same
    __shared__ int s_dense[kScrWarps];
    if (kTop > 5 && lane == 0) s_dense[warp] = rd.dense;
    const int nu = (int)((emit + kX - 1) / kX);
    const int reach = rd.reach;
    const int nb = nu + reach;
    const int rounds = (nb + 31) >> 5;
    const int have = (int)min((int64_t)rounds * 512, rd.n_samp - t0);   // positions inside the row
    const T *rowp = static_cast<const T *>(rd.data) + (int64_t)row * rd.stride + t0;
    const bool has_sc = kScaled && rd.scale != nullptr;
    const float sc = has_sc ? rd.scale[row] : 1.f;
    const float of = (has_sc && rd.offset) ? rd.offset[row] : 0.f;
    const float2 mu = rd.mu_tab[entry];
    const float2 mh = make_float2(-mu.x, -mu.x), ml = make_float2(-mu.y, -mu.y);
    const bool vec = rd.vec_ok != 0;

    // piece q of block b of a round lies at 16 (b kPieces + (q ^ s)), where
    // s = (b >> 1) & 3 (FP32: 4 pieces) or (b >> 2) & 1 (2 pieces).  Copies:
    // lane l takes pieces l + 32 j, whose s is the same for all j
    const uint32_t buf0 = saddr(buf);
    const uint32_t put = buf0 + 16u * (uint32_t)((lane & ~(kPieces - 1)) |
                                                 ((lane & (kPieces - 1)) ^
                                                  ((lane >> 3) & (kPieces - 1))));
    // reads: piece q of the lane's own block at get ^ 16 q (blocks of a
    // buffer are 64 or 32 bytes apart, buffers aligned to 128)
    const uint32_t get = buf0 + 16u * (uint32_t)(lane * kPieces +
                                                 (kPieces == 4 ? (lane >> 1) & 3 : (lane >> 2) & 1));
    const T *src = rowp + lane * kPer;
    auto stage = [&](int r, uint32_t at) {   // round r into the buffer at byte `at`; one copy group
        if (r < rounds) {
            const int base = 512 * r;
            if (vec) {
                if (base + 512 <= have) {
#pragma unroll
                    for (int j = 0; j < kPieces; ++j)
                        cp_async16(put + at + 512u * j, src + base + 32 * kPer * j, 16);
                } else {
#pragma unroll
                    for (int j = 0; j < kPieces; ++j) {
                        const int p = base + (lane + 32 * j) * kPer;
                        const int left = (have - p) * kEsz;      // bytes inside the row
                        const int n = left >= 16 ? 16 : (left > 0 ? left : 0);
                        cp_async16(put + at + 512u * j, n ? rowp + p : rowp, n);
                    }
                }
            } else if constexpr (DT == SPD_F32) {   // rows at any 4-byte step
#pragma unroll
                for (int j = 0; j < 16; ++j) {      // block (lane >> 4) + 2 j: s = j & 3
                    const int e = lane + 32 * j;
                    const bool ok = base + e < have;
                    cp_async4(buf0 + at + 16u * (uint32_t)((e >> 4) * 4 + (((e >> 2) & 3) ^ (j & 3))) +
                                  4u * (uint32_t)(e & 3),
                              ok ? rowp + base + e : rowp, ok ? 4 : 0);
                }
            } else {
                T *d = reinterpret_cast<T *>(buf + at);
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const int e = lane + 32 * j, b = e >> 4;
                    if (base + e < have)
                        d[8 * (b * 2 + (((e >> 3) & 1) ^ ((b >> 2) & 1))) + (e & 7)] = rowp[base + e];
                }
            }
        }
        cp_async_commit();
    };

    // ---- the bars of the tests
    const float *tab = rd.scr_tab + (int64_t)entry * kScrTab;
    const float thr = rd.threshold;
    const float lim = thr - 1e-5f * fabsf(thr);
    const bool all = !(lim > 0.f);   // then no bound rules anything out
    // class c is live where m - min C + slack >= g_c, m the largest C its
    // windows end in, g_c = lim / (largest 1 / sigma_w): +inf without widths
    auto bar = [&](int c) { return lim * 0.999999f / __ldg(tab + c); };
    const float g1 = bar(1), g2 = bar(2), g3 = bar(3);
    const float g4 = kTop > 3 ? bar(4) : kInf, g5 = kTop > 3 ? bar(5) : kInf;
    const float g6 = kTop > 5 ? bar(6) : kInf;
    float gw[3];
#pragma unroll
    for (int c = 7; c < kScrClasses; ++c) gw[c - 7] = kTop > 6 ? bar(c) : kInf;
    // energies: live where e >= h = lim^2 / (largest w / sigma_w^2)
    const float h0 = lim * lim * 0.99999f / __ldg(tab + kScrClasses);
    const float h1 = lim * lim * 0.99999f / __ldg(tab + kScrClasses + 1);
    float slack = 1e-30f;
    uint32_t words = 0u;      // lane r: the live units of round r
    int total = 0;
    // the units of round rt, whose blocks are in the ring from `slot` on
    auto test = [&](int rt, int slot) {
        const int t = slot + lane;
        const float2 ea = s_e[t], eb = s_e[t + 1];
        const float base = slack - s_n[t];
        const float x0 = s_x[t], x1 = s_x[t + 1], x2 = s_x[t + 2], x3 = s_x[t + 3], x4 = s_x[t + 4];
        const float ha = ea.x + ea.y, hb = ea.y + eb.x, hc = eb.x + eb.y;
        float m = fmaxf(fmaxf(x1, x2) - g2, fmax3(x2, x3, x4) - g3);
        if (kTop > 3) {
            const float *q = s_q4 + (slot >> 2) + (lane >> 2);
            const float y2 = q[2];
            m = fmax3(m, fmaxf(q[1], y2) - g4, fmax3(y2, q[3], q[4]) - g5);
        }
        if (kTop > 5) {   // widths up to 512: ends in blocks t + 16 .. t + 32
            const float *q = s_q8 + (slot >> 3) + (lane >> 3);
            m = fmaxf(m, fmax3(q[2], q[3], q[4]) - g6);
        }
        if (kTop > 6) {   // above: blocks t + a .. t + 2 a
#pragma unroll
            for (int c = 7; c < kScrClasses; ++c) {
                if (!((rd.classes >> c) & 1u)) continue;
                const int a0 = 1 << (c - 2);
                float mc = -kInf;
                for (int j = (t + a0) >> 3; j <= (t + 2 * a0) >> 3; ++j) mc = fmaxf(mc, s_q8[j]);
                m = fmaxf(m, mc - gw[c - 7]);
            }
        }
        // a prefix that is not finite (a sample before the unit that is not)
        // rules nothing out, nor does an energy
        bool live = all | !(fabsf(base) < kInf) | !(m + base < 0.f);
        live |= !(fmax_nan(ha, hb) < h0);
        live |= !(fmaxf(x0, x1) - g1 + base < 0.f) & !(fmax_nan(ha + eb.x, ea.y + hc) < h1);
        live &= 32 * rt + lane < nu;
        const uint32_t bal = __ballot_sync(0xffffffffu, live);
        if (lane == rt) words = bal;
        total += __popc(bal);
    };

    // rounds from a unit to the last block it reads
    const int lag = kTop > 6 ? (reach + 31) >> 5 : 1;
    float run = 0.f, mag = 0.f;
    uint32_t at = 0;                     // the buffer of round r, and of round r + 2
    uint32_t at2 = 2 * kBuf;
    stage(0, 0);
    stage(1, kBuf);
    for (int r = 0; r < rounds; ++r) {
        cp_async_wait<1>();   // this lane's copies of round r have landed
        __syncwarp();         // every lane's; the buffer of round r - 1 is read
        float2 v[8];
#pragma unroll
        for (int q = 0; q < kPieces; ++q)
            to_pairs<DT>(lds128((get + at) ^ (16u * q)), v + (kPer / 2) * q);
        stage(r + 2, at2);
        at = at == 2 * kBuf ? 0 : at + kBuf;
        at2 = at2 == 2 * kBuf ? 0 : at2 + kBuf;
        if constexpr (kScaled) {
            const float2 s2 = make_float2(sc, sc), o2 = make_float2(of, of);
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = add2(add2(fma2(s2, v[q], o2), mh), ml);
        } else {
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = add2(add2(v[q], mh), ml);
        }
        float sum = 0.f, hi = 0.f, lo = 0.f;
        float2 e0 = make_float2(0.f, 0.f), e1 = e0;
        if (512 * r + 512 <= have) {          // warp-uniform
            float cp[17];                     // prefixes: cp[q] = y[0] + ... + y[q-1]
            cp[0] = 0.f;
            e0 = mul2(v[0], v[0]);
            e1 = mul2(v[4], v[4]);
#pragma unroll
            for (int q = 1; q < 4; ++q) {
                e0 = fma2(v[q], v[q], e0);
                e1 = fma2(v[4 + q], v[4 + q], e1);
            }
            cp[1] = v[0].x;
            cp[2] = cp[1] + v[0].y;
#pragma unroll
            for (int q = 1; q < 8; ++q) {
                cp[2 * q + 1] = cp[2 * q] + v[q].x;
                cp[2 * q + 2] = cp[2 * q + 1] + v[q].y;
            }
            hi = fmax3(cp[0], cp[1], cp[2]);
            lo = fmin3(cp[0], cp[1], cp[2]);
#pragma unroll
            for (int q = 3; q < 15; q += 2) {
                hi = fmax3(hi, cp[q], cp[q + 1]);
                lo = fmin3(lo, cp[q], cp[q + 1]);
            }
            hi = fmaxf(hi, cp[15]);
            lo = fminf(lo, cp[15]);
            sum = cp[16];
        } else {   // the row ends here: no window may end past it, no start lies past it
            const int left = have - 512 * r - 16 * lane;
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                const float y = (q & 1) ? v[q >> 1].y : v[q >> 1].x;
                if (q < left) {
                    lo = fminf(lo, sum);
                    sum += y;
                    if (q < 15) hi = fmaxf(hi, sum);
                    if (q < 8) e0.x = fmaf(y, y, e0.x); else e1.x = fmaf(y, y, e1.x);
                }
            }
            if (left < 16) sum = -kInf;
        }
        // inclusive scan of the round's sums
        const float xs = add_up<16>(add_up<8>(add_up<4>(add_up<2>(add_up<1>(sum)))));
        float ex = __shfl_up_sync(0xffffffffu, xs, 1);
        ex = run + (lane ? ex : 0.f);
        run += __shfl_sync(0xffffffffu, xs, 31);
        const float mx = ex + hi, mn = ex + lo;
        const float2 en = make_float2(e0.x + e0.y, e1.x + e1.y);
        float m4 = mx, m8 = mx;
        if (kTop > 3) {
            m4 = fmaxf(m4, __shfl_xor_sync(0xffffffffu, m4, 1));
            m4 = fmaxf(m4, __shfl_xor_sync(0xffffffffu, m4, 2));
            if (kTop > 5) m8 = fmaxf(m4, __shfl_xor_sync(0xffffffffu, m4, 4));
        }
        const int rr = r & (ring - 1);
        auto keep = [&](int k) {
            const int slot = 32 * k + lane;
            s_x[slot] = mx;
            s_n[slot] = mn;
            s_e[slot] = en;
            if (kTop > 3) s_q4[slot >> 2] = m4;   // the same value from each of the lanes
            if (kTop > 5) s_q8[slot >> 3] = m8;
        };
        keep(rr);
        if (rr < mirror) keep(rr + ring);
        // margin for the rounding of the prefixes: 200 unit roundoffs of the
        // tile's largest partial sum so far.  The same additions restated on the
        // host beside FP64 put a difference of two prefixes off by 9 at most on
        // noise, offsets of 0.6 and 100 sigma, drifts and spikes of 10^4 and 10^5
        // sigma.  It is no bound of the worst case: a constant with spikes of
        // +-10^5 in every block, whose additions all round the same way, is off
        // by 940 (and the SNRs' own sums with it)
        const float big = fmaxf(fabsf(mx), fabsf(mn));
        const uint32_t top = __reduce_max_sync(0xffffffffu, big < kInf ? __float_as_uint(big) : 0u);
        mag = fmaxf(mag, __uint_as_float(top));
        slack = fmaf(1.2e-5f, mag, 1e-30f);
        __syncwarp();
        if (r >= lag) test(r - lag, 32 * ((r - lag) & (ring - 1)));
    }
    cp_async_wait<0>();
    for (int rt = max(0, rounds - lag); 32 * rt < nu; ++rt) test(rt, 32 * (rt & (ring - 1)));
    if (!total) return;

    // ---- the lists: a tile with many live units whole, else its units
    if (total > (kTop > 5 ? s_dense[warp] : kScrDense)) {
        if (lane == 0) A.lists.tiles[atomicAdd(&A.lists.ctl->dense, 1u)] = tile;
        return;
    }
    uint32_t base = 0u;
    if (lane == 0) base = atomicAdd(&A.lists.ctl->live, (uint32_t)total);
    base = __shfl_sync(0xffffffffu, base, 0);
    for (int q = 0; 32 * q < nu; ++q) {
        const uint32_t w = __shfl_sync(0xffffffffu, words, q);
        if ((w >> lane) & 1u)
            A.lists.units[base + __popc(w & ((1u << lane) - 1u))] =
                tile << 8 | (uint32_t)(32 * q + lane);
        base += __popc(w);
    }
}

template <int DT, bool kScaled> void (*screen_of(int top))(const ScreenArgs) {
    return top <= 3   ? screen_kernel<DT, 3, kScaled>
           : top <= 5 ? screen_kernel<DT, 5, kScaled>
           : top <= 6 ? screen_kernel<DT, 6, kScaled> : screen_kernel<DT, 9, kScaled>;
}
template <bool kScaled> void (*screen_of(int dtype, int top))(const ScreenArgs) {
    return dtype == SPD_F32 ? screen_of<SPD_F32, kScaled>(top)
           : dtype == SPD_F16 ? screen_of<SPD_F16, kScaled>(top) : screen_of<SPD_BF16, kScaled>(top);
}

}  // namespace

cudaError_t launch_screen(const Launch &L, const ScreenLists &S, int dtype, cudaStream_t s) {
    static thread_local ScreenArgs A;
    int lag = 1, widest = 0;
    bool scaled = false;
    for (int r = 0; r < L.n_ranges; ++r) {
        const RangeDesc &rd = L.rng[r];
        ScreenRange &q = A.rng[r];
        q.data = rd.data;
        q.stride = rd.stride;
        q.n_samp = rd.n_samp;
        q.n_emit = rd.n_emit;
        q.scale = rd.scale;
        scaled |= rd.scale != nullptr;
        q.offset = rd.offset;
        q.mu_tab = rd.mu_tab;
        q.flags = rd.flags;
        q.scr_tab = rd.scr_tab;
        q.tiles_per_row = (int32_t)rd.tiles_per_row;
        q.vec_ok = rd.vec_ok;
        q.per_row = rd.per_row;
        q.tile0 = (uint32_t)rd.tile0;
        q.threshold = rd.threshold;
        q.dense = screen_dense(rd.prog.wmax);
        q.classes = 0;
        int top = 0;
        for (int g = 0; g < rd.prog.n_groups; ++g) {
            const Group &gr = rd.prog.groups[g];
            const int d = (gr.flags & kGroupCoarse) ? rd.prog.G : 1;
            for (int c = 0; c < gr.count; ++c) {
                const int k = screen_class(gr.off + (c + 1) * d);
                q.classes |= 1u << k;
                top = k > top ? k : top;
            }
        }
        // the last block the widest class's windows end in: 2^(top-1) past
        // the unit's own.  (A group of 4 or 8 blocks read for it lies in that
        // block's round; what it holds past the reach only loosens a bound.)
        q.reach = top < 2 ? 1 : 1 << (top - 1);
        const int l = (q.reach + 31) / 32;
        lag = l > lag ? l : lag;
        widest = top > widest ? top : widest;
    }
    A.lists = S;
    A.n_ranges = L.n_ranges;
    A.n_tiles = (uint32_t)L.n_tiles;
    A.units = L.units;
    A.ring = 2;
    while (A.ring < lag + 1) A.ring *= 2;
    A.mirror = lag;
    if (L.n_tiles <= 0) return cudaSuccess;
    const size_t smem =
        (size_t)kScrWarps * screen_warp_bytes((int)elem_bytes(dtype), A.ring + A.mirror);
    auto k = scaled ? screen_of<true>(dtype, widest) : screen_of<false>(dtype, widest);
    if (smem > 48 * 1024) {   // wide lists
        const cudaError_t e =
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    k<<<(unsigned)((L.n_tiles + kScrWarps - 1) / kScrWarps), kScrThreads, smem, s>>>(A);
    return cudaGetLastError();
}

}  // namespace spd
