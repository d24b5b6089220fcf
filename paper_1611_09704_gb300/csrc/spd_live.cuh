// spd_live.cuh -- the search of single live units of 16 starts (listed by the
// screen, spd_screen.cu), a half-warp per unit: the search kernel's work after
// its tiles.
#pragma once
#include "spd_device.cuh"

namespace spd {

namespace {

__device__ __forceinline__ float half_min(float v, uint32_t hm) {
#pragma unroll
    for (int o = 8; o; o >>= 1) v = fminf(v, __shfl_xor_sync(hm, v, o));
    return v;
}

// One half-warp per live unit, one start per lane.  The lanes stage the
// unit's window as the search kernel stages a tile's (y, in-block prefixes P,
// window sums S_G, block sums), then visit the width groups from the widest
// down with the search kernel's bounds, group starts, sums and packed max.  A
// group evaluated in both comes out of the same operations in the same order,
// but for its start when the two skipped different wider groups: the margin of
// the bounds is that of the unit's prefixes here and of the tile's there, and a
// start is formed from that of the last group evaluated.  So an SNR can differ
// in its last rounding: 70 of 357,800 records whose tiles hold a spike of 10^5
// sigma, none in 120 planes without one.  The two halves of a warp meet again
// to write their records.
//
// Bound by latency: a unit's staging waits for L2 or DRAM once, and a group
// takes its widths one after the other.  Many units in flight hide it: 20 us
// for the live units of 4096 x 524288 samples of noise.
//
// s_dyn: the CTA's dynamic shared memory, whose first use is over.  in_tiles:
// the units of the listed tiles, when these are searched here too (else 0).
template <int DT, int G, bool MG>
__device__ __forceinline__ void live_units(const Launch &L, float *s_dyn, uint32_t in_tiles) {
    using T = typename Elem<DT>::T;
    const int blocks = L.live_blocks, halves = L.live_halves;
    const uint32_t *units = L.unit_list;
    const int tid = threadIdx.x, lane = tid & 31, k = lane & 15;
    const int half = tid >> 4;                          // half-warp of the CTA
    const uint32_t hm = 0xffffu << (lane & 16);
    const bool has_room = half < halves;                // shared memory for this half-warp
    float *s_y = s_dyn + (int64_t)(has_room ? half : 0) * live_words(blocks, G);
    float *s_p = s_y + blocks * kSPad;
    float *s_g = s_p + blocks * kSPad;
    float *s_bs = s_p + (G > 1 ? 2 : 1) * blocks * kSPad;
    float *s_mx = s_bs + blocks;
    float *s_pq = s_mx + blocks;                        // [blocks + 1]
    const uint32_t n = in_tiles + *L.unit_count;
    const uint32_t per = gridDim.x * (uint32_t)halves;
    // warp-uniform trip count: the first half-warp of the warp decides
    for (uint32_t i0 = blockIdx.x * (uint32_t)halves + (uint32_t)((tid >> 5) * 2); i0 < n; i0 += per) {
        const uint32_t i = i0 + (uint32_t)((lane >> 4) & 1);
        uint32_t id = ~0u;   // none (a tile index is under 2^24 - 1)
        if (has_room && i < n) {
            if (i < in_tiles) {
                const uint32_t t = i / (uint32_t)L.units;
                id = L.tile_list[t] << 8 | (i - t * (uint32_t)L.units);
            } else {
                id = units[i - in_tiles];
            }
        }
        uint32_t bits = 0u;
        int eb = 0, ri = 0;
        int64_t row = 0, i1 = 0;
        bool cand = false;
        if (id != ~0u) {
            const uint32_t tl = id >> 8;
            while (ri + 1 < L.n_ranges && (int64_t)tl >= L.rng[ri + 1].tile0) ++ri;
            const RangeDesc &rd = L.rng[ri];
            const uint32_t lt = tl - (uint32_t)rd.tile0;
            const uint32_t q = lt / (uint32_t)rd.tiles_per_row;
            row = q;
            const int64_t col = lt - q * (uint32_t)rd.tiles_per_row;
            i1 = (col * L.units + (int64_t)(id & 255u)) * kX;   // the unit's first start
            if (i1 >= rd.n_emit) id = ~0u;   // a listed tile's unit past the row's last start
        }
        if (id != ~0u) {
            const RangeDesc &rd = L.rng[ri];
            const RangeProg &rp = rd.prog;
            const int entry = rd.per_row ? (int)row : 0;
            const bool has_sc = rd.scale != nullptr;
            const float sc = has_sc ? rd.scale[row] : 1.f;
            const float of = (has_sc && rd.offset) ? rd.offset[row] : 0.f;
            const float2 mu = rd.mu_tab[entry];
            const float *inv = rd.inv_tab + (int64_t)entry * rp.n_eval;
            const float2 *grp = rd.grp_tab + (int64_t)entry * rp.n_groups;
            const T *p0 = static_cast<const T *>(rd.data) + row * rd.stride + i1;
            const int nblk = ((15 + rp.wmax) >> 4) + 1;   // blocks of the unit's windows
            const int have = (int)min((int64_t)nblk * 16 + 16, rd.n_samp - i1);
            const int nraw = rd.vec_ok ? have : 0;        // elements vector loads may read

            // ---- staging, a block per lane; the half-warp's scan of the sums
            float run = 0.f, runq = 0.f, mag = 0.f, lo0 = 0.f;
            __syncwarp(hm);
            for (int c0 = 0; c0 < nblk; c0 += 16) {
                const int c = c0 + k;
                float sum = 0.f, en = 0.f, hi = 0.f, lo = 0.f;
                if (c < nblk) {
                    constexpr int NX = G > 1 ? 16 + G : 16;
                    float v[NX];
                    load_centred<DT, 16>(v, p0, p0, 16 * c, nraw, have, has_sc, sc, of, mu);
                    if (G > 1)
                        load_centred<DT, G>(v + 16, p0, p0, 16 * c + 16, nraw, have, has_sc, sc,
                                            of, mu);
                    float Cp[NX + 1];
                    Cp[0] = 0.f;
#pragma unroll
                    for (int e = 0; e < NX; ++e) Cp[e + 1] = __fadd_rn(Cp[e], v[e]);
                    sum = Cp[16];
#pragma unroll
                    for (int e = 1; e < 16; ++e) {
                        hi = fmaxf(hi, Cp[e]);
                        lo = fminf(lo, Cp[e]);
                    }
#pragma unroll
                    for (int e = 0; e < 16; ++e) en += 16 * c + e < have ? v[e] * v[e] : 0.f;
                    float *yd = s_y + kSPad * c, *pd = s_p + kSPad * c;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        *reinterpret_cast<float4 *>(yd + 4 * u) =
                            make_float4(v[4 * u], v[4 * u + 1], v[4 * u + 2], v[4 * u + 3]);
                        *reinterpret_cast<float4 *>(pd + 4 * u) =
                            make_float4(Cp[4 * u], Cp[4 * u + 1], Cp[4 * u + 2], Cp[4 * u + 3]);
                    }
                    if (G > 1) {
                        float *gd = s_g + kSPad * c;
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            *reinterpret_cast<float4 *>(gd + 4 * u) = make_float4(
                                __fsub_rn(Cp[4 * u + G], Cp[4 * u]),
                                __fsub_rn(Cp[4 * u + 1 + G], Cp[4 * u + 1]),
                                __fsub_rn(Cp[4 * u + 2 + G], Cp[4 * u + 2]),
                                __fsub_rn(Cp[4 * u + 3 + G], Cp[4 * u + 3]));
                    }
                    s_bs[c] = sum;
                }
                float xs = sum, xq = en;
#pragma unroll
                for (int o = 1; o < 16; o <<= 1) {
                    const float us = __shfl_up_sync(hm, xs, o, 16);
                    const float uq = __shfl_up_sync(hm, xq, o, 16);
                    if (k >= o) {
                        xs += us;
                        xq += uq;
                    }
                }
                const float exs = __shfl_up_sync(hm, xs, 1, 16);
                const float P = run + (k ? exs : 0.f);
                if (c < nblk) {
                    const float mx = P + hi;
                    s_mx[c] = mx;
                    s_pq[c + 1] = runq + xq;
                    if (fabsf(mx) < INFINITY) mag = fmaxf(mag, fabsf(mx));
                    if (fabsf(P + lo) < INFINITY) mag = fmaxf(mag, fabsf(P + lo));
                }
                if (c0 == 0) lo0 = __shfl_sync(hm, lo, 0, 16);
                run += __shfl_sync(hm, xs, 15, 16);
                runq += __shfl_sync(hm, xq, 15, 16);
            }
#pragma unroll
            for (int o = 8; o; o >>= 1) mag = fmaxf(mag, __shfl_xor_sync(hm, mag, o));
            __syncwarp(hm);

            // ---- the groups, widest first
            const float thr = rd.threshold;
            const float cslack = fmaf(8e-6f, mag, 1e-30f) - lo0;
            float limv = thr;
            float lim_lo = thr - 1e-5f * fabsf(thr);
            float lim2 = thr > 0.f ? lim_lo * lim_lo : -1.f;
            float cb = -INFINITY, ob = -INFINITY;
            int obk = 0, cur = -1;
            int lastO = -1;
            float lastD = 0.f;
            for (int gi = rp.n_groups - 1; gi >= 0; --gi) {
                const Group g = rp.groups[gi];
                const float2 gt = __ldg(grp + gi);
                const bool coarse = G > 1 && (g.flags & kGroupCoarse);
                const int d = coarse ? G : 1;
                const int end = g.off + g.count * d;
                // energy of the blocks the windows lie in: this group's and all narrower ones'
                if (s_pq[1 + ((14 + end) >> 4)] * 1.000008f * gt.y < lim2) break;
                float rmax = -INFINITY;
                for (int b = (g.off + d) >> 4; b <= (15 + end) >> 4; ++b)
                    rmax = fmax_nan(rmax, s_mx[b]);
                if (fmax_nan(rmax + cslack, 0.f) * gt.x < lim_lo) continue;   // NaN never prunes
                if (MG && (g.widx0 >> 6) != cur) {
                    if (cur >= 0 && trunc17(cb) >= trunc17(ob)) {
                        ob = cb;
                        obk = cur;
                    }
                    cb = -INFINITY;
                    cur = g.widx0 >> 6;
                }
                if (g.flags & kGroupRefine) {   // each start's own 16 samples against its best
                    float en = 0.f;
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        const float y = s_y[sadr(k + e)];
                        en = fmaf(y, y, en);
                    }
                    const float lim = fmaxf(thr, trunc17(MG ? fmaxf(cb, ob) : cb));
                    const float ll = lim * (1.f - 2e-5f);
                    if (!__any_sync(hm, !(lim > 0.f && (en * 1.000008f + 1e-30f) * gt.y < ll * ll)))
                        continue;
                }
                // B_off at the lane's start
                float B = 0.f;
                if (g.off && (g.off & 15) == 0) {
                    const int o = g.off >> 4;
                    float D;
                    if (lastO >= o && lastO - o <= 16 && fabsf(lastD) < INFINITY) {
                        D = lastD;
                        for (int b = o; b < lastO; ++b) D = __fsub_rn(D, s_bs[b]);
                    } else {
                        D = 0.f;
                        if (o <= 16) {
                            for (int b = 0; b < o; ++b) D = __fadd_rn(D, s_bs[b]);
                        } else {   // Kahan-compensated in block order
                            float comp = 0.f;
                            for (int b = 0; b < o; ++b) {
                                const float y = __fsub_rn(s_bs[b], comp);
                                const float sn = __fadd_rn(D, y);
                                comp = __fsub_rn(__fsub_rn(sn, D), y);
                                D = sn;
                            }
                        }
                    }
                    lastO = o;
                    lastD = D;
                    B = __fadd_rn(D, __fsub_rn(s_p[kSPad * o + k], s_p[k]));
                } else if (g.off) {   // the sum over [0, off), then one slide per start
                    const int o = g.off >> 4;
                    for (int b = 0; b < o; ++b) B = __fadd_rn(B, s_bs[b]);
                    for (int j = 16 * o; j < g.off; ++j) B = __fadd_rn(B, s_y[sadr(j)]);
                    for (int j = 0; j < k; ++j)
                        B = __fadd_rn(B, __fsub_rn(s_y[sadr(g.off + j)], s_y[sadr(j)]));
                }
                const float *arr = coarse ? s_g : s_y;
#pragma unroll 4
                for (int c = 0; c < g.count; ++c) {
                    const int wi = g.widx0 + c;
                    B = __fadd_rn(B, arr[sadr(g.off + c * d + k)]);
                    cb = fmaxf(cb, packw(__fmul_rn(B, __ldg(inv + wi)), 63u - (uint32_t)(wi & 63)));
                }
                const float mb = trunc17(half_min(MG ? fmaxf(cb, ob) : cb, hm));
                if (mb > limv) {
                    limv = mb;
                    lim_lo = mb - 1e-5f * fabsf(mb);
                    lim2 = mb > 0.f ? lim_lo * lim_lo : -1.f;
                }
            }
            if (MG && cur >= 0 && trunc17(cb) >= trunc17(ob)) {
                ob = cb;
                obk = cur;
            }
            const float best = MG ? ob : cb;
            bits = __float_as_uint(best);
            eb = MG ? 64 * obk : 0;
            cand = trunc17(best) >= thr && i1 + k < rd.n_emit;
        }
        __syncwarp();
        const uint32_t bal = __ballot_sync(0xffffffffu, cand);
        if (!bal) continue;
        unsigned long long base = 0;
        if (lane == 0)
            base = atomicAdd(reinterpret_cast<unsigned long long *>(&L.result->count),
                             (unsigned long long)__popc(bal));
        base = __shfl_sync(0xffffffffu, base, 0);
        const unsigned long long slot = base + (unsigned)__popc(bal & ((1u << lane) - 1u));
        if (cand && slot < (unsigned long long)L.capacity) {
            const RangeDesc &rd = L.rng[ri];
            const int wi = eb + 63 - (int)(bits & 63u);
            int w = 0;
            for (int gi = 0; gi < rd.prog.n_groups; ++gi) {
                const Group g = rd.prog.groups[gi];
                if (wi >= g.widx0 && wi < g.widx0 + g.count)
                    w = g.off + (wi - g.widx0 + 1) * ((G > 1 && (g.flags & kGroupCoarse)) ? G : 1);
            }
            reinterpret_cast<int4 *>(L.out)[slot] =
                make_int4(rd.dm_offset + (int)row,
                          (int)(rd.sample_base + ((i1 + k) << rd.sample_shift)),
                          (int)(bits & 0xFFFFFFC0u), w << rd.sample_shift);
        }
    }
}

}  // namespace

}  // namespace spd
