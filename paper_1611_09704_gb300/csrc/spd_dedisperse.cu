// spd_dedisperse.cu -- incoherent de-dispersion: the DM x time plane the
// detector searches (Sec. 1), made from a filterbank of channel rows by
// summing each channel shifted by its dispersion delay for every DM trial.
// A producer for the streaming search: it can write DM trials straight into
// a push workspace's chunk view, so the search reads them in place (the
// coupling Sec. 3 names as future work).
#include "spd_internal.cuh"

namespace spd {
void note_cuda_error(int e);
}

using namespace spd;

namespace {

constexpr int kDdThreads = 256;
constexpr int kDdChunk = 128;       // channels whose delays are staged at once (even)
constexpr int kDdSpread = 1024;     // delay spread of a DM block held in shared memory
constexpr int kDdRing = 3;          // channel pairs staged or in flight
constexpr int kDdSlack = 16;        // window elements lost to 16-byte alignment, at most

// Shape of a CTA: kPer outputs per thread (256 apart) of kDms DM trials.
template <int PER, int DMS> struct DdShape {
    static constexpr int kSpan = kDdThreads * PER;                 // output samples per CTA
    static constexpr int kWin = kSpan + kDdSpread + kDdSlack;      // raw window of a channel
    static constexpr int kPat = DMS / 4;                           // sums of a pair, at most
    static constexpr int kOne = kSpan + kDdSpread;                 // decoded window of a channel
    static constexpr int kSums = kPat * kSpan + kDdSpread > 2 * kOne ? kPat * kSpan + kDdSpread
                                                                     : 2 * kOne;
    static constexpr size_t smem(size_t esz) {
        return (size_t)kDdChunk * (DMS + 6) * 4 + (size_t)kDdRing * 2 * kWin * esz +
               2 * (size_t)kSums * 4;
    }
};

template <int DT>
__device__ __forceinline__ float fb_value(const typename Elem<DT>::T *p, bool has_sc, float sc,
                                          float of) {
    const float x = Elem<DT>::cvt(*p);
    return has_sc ? fmaf(sc, x, of) : x;
}

__device__ __forceinline__ void store_out(void *out, int dt, int64_t idx, float v) {
    if (dt == SPD_F32) static_cast<float *>(out)[idx] = v;
    else if (dt == SPD_F16) static_cast<__half *>(out)[idx] = __float2half_rn(v);
    else static_cast<__nv_bfloat16 *>(out)[idx] = __float2bfloat16_rn(v);
}

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}
// The float at a shared-memory address plus a constant.
template <int OFF> __device__ __forceinline__ float lds_at(uint32_t addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1 + %2];\n" : "=f"(v) : "r"(addr), "n"(OFF) : "memory");
    return v;
}
__device__ __forceinline__ void cp_async_commit() {
    asm volatile("cp.async.commit_group;\n" ::: "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

// One CTA: 256 PER consecutive outputs t0 .. of DMS consecutive DM trials
// d0 ...  For every channel c the trials of the block read the one window
// x[c][t0 + lo_c, t0 + 256 PER + hi_c) (lo_c, hi_c: the smallest and largest
// delay of the block at c).  Channels go in pairs.  A pair's windows arrive by
// 16-byte asynchronous copies two pairs ahead, from the 16-byte boundary at or
// before their first sample; thread t sums outputs t0 + t + 256 j, j < PER, of
// every trial.
//
// Pairs whose trials share few delay differences: the sum a trial needs,
// x[c][t + delay] + x[c + 1][t + delay + difference], depends on the
// difference alone, so it is formed once per distinct difference (at most
// DMS / 4 of them; two or three are usual in a block of neighbouring trials)
// over the samples its trials read, and each trial adds the sum: one
// shared-memory word per output, trial and pair instead of two.  Otherwise the
// channels are added one by one, FP32 straight from the staged window, FP16 /
// BF16 from a decoded one (decoding is part of forming the sums).  A channel
// whose spread exceeds kDdSpread is read from global memory.  Either way a
// trial's channels are added in the order 0, 1, ..., the two of a pair as one
// sum.  A delay outside [0, n_samp - n_out] makes its trial's outputs NaN and
// sets the status (no read outside the row).
//
// Bound by the shared-memory pipe (71 % of its rate), with 16 warps per SM (64
// registers of sums per thread).  256 channels x 256 trials x 2^18 outputs
// FP32: 3.40 ms with one word per output, trial and channel, 4-byte copies and
// 2 outputs per thread (5.9 instructions per add); 2.97 ms with sums of pairs
// and 4 outputs; 2.44 ms with the copies' addresses prepared once per channel
// and whole blocks of the sums formed without bound checks (2.8 per add).  200
// x 117 x 60001 FP16: 583 -> 300 us (16-bit windows staged as they are).
// Trials too far apart to share a window, 200 x 32 x 16000: 0.51 -> 0.14 ms
// (the loads of four trials in flight).  The small shape fits four CTAs per SM in
// shared memory, and is held to the registers for that: 512 x 16 x 30000 FP32 (472
// CTAs) 363 us with three of 68 registers, 230 so.
template <int DT, int PER, int DMS>
__global__ void __launch_bounds__(kDdThreads, PER == 1 ? 4 : 2) dedisperse_kernel(
    const typename Elem<DT>::T *fb, int64_t n_chan, int64_t n_samp, int64_t fb_stride,
    const float *scale, const float *offset, const int32_t *delays, int64_t n_dm, void *out,
    int out_dt, int64_t n_out, int64_t out_stride, spd_result *status) {
    using T = typename Elem<DT>::T;
    using S = DdShape<PER, DMS>;
    constexpr int kSpan = S::kSpan;
    constexpr int kPiece = 16 / (int)sizeof(T);      // elements per 16-byte piece
    extern __shared__ __align__(16) unsigned char smem[];
    // per channel: the trials' delays as byte offsets into what they read; for a
    // pair summed by differences the second channel's row holds the sums
    int32_t(*s_dl)[DMS] = reinterpret_cast<int32_t(*)[DMS]>(smem);
    int32_t *s_lo = reinterpret_cast<int32_t *>(s_dl + kDdChunk);   // smallest delay
    int32_t *s_sp = s_lo + kDdChunk;                                // spread
    int32_t *s_md = s_sp + kDdChunk;                                // pair: its sums, 0 = none
    int32_t *s_nd = s_md + kDdChunk;                                // elements to stage, see below
    const T **s_src = reinterpret_cast<const T **>(s_nd + kDdChunk);   // and from where
    T *s_x = reinterpret_cast<T *>(s_src + kDdChunk);               // [ring][2][kWin]
    float *s_w = reinterpret_cast<float *>(s_x + kDdRing * 2 * S::kWin);   // [2][kSums]
    __shared__ uint32_t s_bad;                   // bit d: trial d0 + d has a bad delay
    const int tid = threadIdx.x;
    // block b: DM block b % n_dmb of time tile b / n_dmb, so the DM blocks of
    // one time tile run side by side and read its channel windows from L2
    const int64_t n_dmb = (n_dm + DMS - 1) / DMS;
    const int64_t b = blockIdx.x;
    const int64_t t0 = (b / n_dmb) * kSpan;
    const int64_t d0 = (b % n_dmb) * DMS;
    const int nd = (int)min((int64_t)DMS, n_dm - d0);
    const int64_t max_delay = n_samp - n_out;
    const bool has_sc = scale != nullptr;
    const T *fb_end = fb + (n_chan - 1) * fb_stride + n_samp;
    // outputs 2 j and 2 j + 1 of a trial as one packed pair (two IEEE adds per
    // packed add); PER 1: the first of the pair alone
    constexpr int kPair = (PER + 1) / 2;
    float2 acc[DMS][kPair];
#pragma unroll
    for (int d = 0; d < DMS; ++d)
#pragma unroll
        for (int j = 0; j < kPair; ++j) acc[d][j] = make_float2(0.f, 0.f);
    if (tid == 0) s_bad = 0u;
    for (int64_t c0 = 0; c0 < n_chan; c0 += kDdChunk) {
        const int nc = (int)min((int64_t)kDdChunk, n_chan - c0);
        const int npair = (nc + 1) / 2;
        // elements from the 16-byte boundary before it to channel c's window
        auto shift = [&](int c) { return abs(s_nd[c]) - kSpan - s_sp[c]; };
        __syncthreads();   // the last chunk's delays and windows are no longer read
        for (int i = tid; i < nc * DMS; i += kDdThreads) {
            const int c = i / DMS, d = i - c * DMS;
            int32_t v = -1;
            if (d < nd) {
                v = __ldg(delays + (d0 + d) * n_chan + c0 + c);
                if (v < 0 || (int64_t)v > max_delay) {
                    atomicOr(&s_bad, 1u << d);
                    v = -1;
                }
            }
            s_dl[c][d] = v;
        }
        __syncthreads();
        for (int c = tid; c < nc; c += kDdThreads) {
            int lo = INT32_MAX, hi = -1;
            for (int d = 0; d < nd; ++d) {
                const int v = s_dl[c][d];
                if (v >= 0) {
                    lo = min(lo, v);
                    hi = max(hi, v);
                }
            }
            if (hi < 0) lo = hi = 0;
            // delays relative to the channel's smallest; a bad delay and the
            // trials past the block's last read offset 0 (their sums are
            // never stored)
            for (int d = 0; d < DMS; ++d) {
                const int v = s_dl[c][d];
                s_dl[c][d] = v >= 0 ? v - lo : 0;
            }
            s_lo[c] = lo;
            s_sp[c] = hi - lo;
            // the window from the 16-byte boundary at or before it; nothing
            // for one read from global memory, and with a minus sign the
            // length of one that sticks out of the filterbank by a piece
            const T *src = fb + (c0 + c) * fb_stride + t0 + lo;
            const int sh = (int)((reinterpret_cast<uintptr_t>(src) & 15) / sizeof(T));
            src -= sh;
            int need = hi - lo <= kDdSpread ? kSpan + hi - lo + sh : 0;
            if (need && (src < fb || src + (need + kPiece - 1) / kPiece * kPiece > fb_end))
                need = -need;
            s_src[c] = src;
            s_nd[c] = need;
        }
        __syncthreads();
        for (int q = tid; q < npair; q += kDdThreads) {
            const int c = 2 * q;
            // the distinct differences, and the offsets their trials read
            int np = 0, df[S::kPat], mn[S::kPat], mx[S::kPat];
            bool ok = c + 1 < nc && s_sp[c] <= kDdSpread && s_sp[c + 1] <= kDdSpread;
            for (int d = 0; d < DMS && ok; ++d) {
                const int o = s_dl[c][d], f = s_dl[c + 1][d] - o;
                bool hit = false;
#pragma unroll
                for (int p = 0; p < S::kPat; ++p) {
                    if (p < np && !hit && df[p] == f) {
                        mn[p] = min(mn[p], o);
                        mx[p] = max(mx[p], o);
                        hit = true;
                    }
                }
                if (!hit) {
                    if (np == S::kPat) ok = false;
#pragma unroll
                    for (int p = 0; p < S::kPat; ++p) {
                        if (p == np && ok) {
                            df[p] = f;
                            mn[p] = mx[p] = o;
                        }
                    }
                    ++np;
                }
            }
            int room = 0;
#pragma unroll
            for (int p = 0; p < S::kPat; ++p)
                if (p < np) room += kSpan + mx[p] - mn[p];
            ok = ok && room <= S::kSums;
            s_md[q] = ok ? np : 0;
            if (ok) {
                int at[S::kPat], next = 0;
#pragma unroll
                for (int p = 0; p < S::kPat; ++p) {
                    at[p] = next;
                    if (p < np) next += kSpan + mx[p] - mn[p];
                }
                for (int d = 0; d < DMS; ++d) {
                    const int o = s_dl[c][d], f = s_dl[c + 1][d] - o;
#pragma unroll
                    for (int p = 0; p < S::kPat; ++p)
                        if (p < np && df[p] == f) s_dl[c][d] = 4 * (at[p] + o - mn[p]);
                }
                const int sa = shift(c), sb = shift(c + 1);
#pragma unroll
                for (int p = 0; p < S::kPat; ++p) {
                    if (p < np) {   // first element in each window, length
                        s_dl[c + 1][4 * p] = mn[p] + sa;
                        s_dl[c + 1][4 * p + 1] = mn[p] + df[p] + sb;
                        s_dl[c + 1][4 * p + 2] = kSpan + mx[p] - mn[p];
                        s_dl[c + 1][4 * p + 3] = at[p];
                    }
                }
            } else {   // the decoded windows side by side, or the staged ones themselves
                const bool raw = DT == SPD_F32 && !has_sc;
                for (int e = c; e < min(c + 2, nc); ++e) {
                    if (s_sp[e] > kDdSpread) continue;   // stays as it is: see add_global
                    const int first = raw ? (e - c) * S::kWin + shift(e) : (e - c) * S::kOne;
                    for (int d = 0; d < DMS; ++d) s_dl[e][d] = 4 * (s_dl[e][d] + first);
                }
            }
        }
        __syncthreads();

        // pair q's windows into their slot of the ring (one copy group, also
        // an empty one); none for a channel read from global memory
        auto stage = [&](int q) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int c = 2 * q + e;
                if (c < nc) {
                    const int need = s_nd[c];
                    const T *src = s_src[c];
                    T *dst = s_x + ((q % kDdRing) * 2 + e) * S::kWin;
                    if (need >= 0) {
#pragma unroll
                        for (int k = 0; k < (S::kWin + kDdThreads * kPiece - 1) / (kDdThreads * kPiece); ++k) {
                            const int i = (tid + k * kDdThreads) * kPiece;
                            if (i < need) cp_async16(dst + i, src + i);
                        }
                    } else {
                        for (int i = tid; i < -need; i += kDdThreads)
                            dst[i] = src + i >= fb && src + i < fb_end ? src[i] : T(0.f);
                    }
                }
            }
            cp_async_commit();
        };
        // n >= kSpan elements of w from f(i)
        auto fill = [&](float *w, int n, auto f) {
#pragma unroll
            for (int j = 0; j < PER; ++j) w[tid + j * kDdThreads] = f(tid + j * kDdThreads);
            for (int i = kSpan + tid; i < n; i += kDdThreads) w[i] = f(i);
        };
        // pair q's sums, or its decoded windows
        auto form = [&](int q) {
            if (q >= npair) return;
            const int c = 2 * q, np = s_md[q];
            if (DT == SPD_F32 && !np && !has_sc) return;
            const T *xa = s_x + (q % kDdRing) * 2 * S::kWin, *xb = xa + S::kWin;
            float *w = s_w + (q & 1) * S::kSums;
            float sa = 1.f, oa = 0.f, sb = 1.f, ob = 0.f;
            if (has_sc) {
                sa = __ldg(scale + c0 + c);
                if (offset) oa = __ldg(offset + c0 + c);
                if (c + 1 < nc) {
                    sb = __ldg(scale + c0 + c + 1);
                    if (offset) ob = __ldg(offset + c0 + c + 1);
                }
            }
            if (np) {
                const int4 *pat = reinterpret_cast<const int4 *>(s_dl[c + 1]);
                for (int p = 0; p < np; ++p) {
                    const int4 g = pat[p];
                    const T *pa = xa + g.x, *pb = xb + g.y;
                    fill(w + g.w, g.z, [&](int i) {
                        return __fadd_rn(fb_value<DT>(pa + i, has_sc, sa, oa),
                                         fb_value<DT>(pb + i, has_sc, sb, ob));
                    });
                }
            } else {
                for (int e = c; e < min(c + 2, nc); ++e) {
                    if (s_sp[e] > kDdSpread) continue;
                    const T *px = (e == c ? xa : xb) + shift(e);
                    const float se = e == c ? sa : sb, oe = e == c ? oa : ob;
                    fill(w + (e - c) * S::kOne, kSpan + s_sp[e],
                         [&](int i) { return fb_value<DT>(px + i, has_sc, se, oe); });
                }
            }
        };
        // every trial's outputs of one row of offsets (bytes), read from the
        // floats at shared-memory address w
        auto add = [&](uint32_t w, const int32_t *dl) {
            const int4 *dv = reinterpret_cast<const int4 *>(dl);
            w += 4u * tid;
#pragma unroll
            for (int q = 0; q < DMS / 4; ++q) {
                const int4 d4 = dv[q];   // four trials' offsets, one broadcast load
                const int o[4] = {d4.x, d4.y, d4.z, d4.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const uint32_t p = w + (uint32_t)o[e];
                    float2 *a = acc[4 * q + e];
                    constexpr int kStep = 4 * kDdThreads;
                    if constexpr (PER == 1) {
                        a[0].x = __fadd_rn(a[0].x, lds_at<0>(p));
                    } else {
                        a[0] = __fadd2_rn(a[0], make_float2(lds_at<0>(p), lds_at<kStep>(p)));
                        if constexpr (PER == 4)
                            a[1] = __fadd2_rn(a[1], make_float2(lds_at<2 * kStep>(p),
                                                                lds_at<3 * kStep>(p)));
                    }
                }
            }
        };
        // a wide spread: channel c straight from global memory, the loads of all
        // trials in flight together
        auto add_global = [&](int c) {
            const T *row = fb + (c0 + c) * fb_stride + s_lo[c] + t0 + tid;
            const float sc = has_sc ? __ldg(scale + c0 + c) : 1.f;
            const float of = (has_sc && offset) ? __ldg(offset + c0 + c) : 0.f;
            const int left = (int)min(n_out - t0 - tid, (int64_t)kSpan);   // outputs from the first
            const int4 *dv = reinterpret_cast<const int4 *>(s_dl[c]);
#pragma unroll
            for (int q = 0; q < DMS / 4; ++q) {
                const int4 d4 = dv[q];   // trials past the block's last read offset 0
                const int o[4] = {d4.x, d4.y, d4.z, d4.w};
                T v[4][PER];
#pragma unroll
                for (int e = 0; e < 4; ++e)
#pragma unroll
                    for (int j = 0; j < PER; ++j)
                        v[e][j] = j * kDdThreads < left ? row[o[e] + j * kDdThreads] : T(0.f);
#pragma unroll
                for (int e = 0; e < 4; ++e)
#pragma unroll
                    for (int j = 0; j < PER; ++j) {
                        float &a = (j & 1) ? acc[4 * q + e][j / 2].y : acc[4 * q + e][j / 2].x;
                        a = __fadd_rn(a, fb_value<DT>(&v[e][j], has_sc, sc, of));
                    }
            }
        };
        const uint32_t w0 = (uint32_t)__cvta_generic_to_shared(s_w);
        const uint32_t x0 = (uint32_t)__cvta_generic_to_shared(s_x);
        stage(0);
        cp_async_wait_all();
        __syncthreads();
        stage(1);
        form(0);
        for (int q = 0; q < npair; ++q) {
            cp_async_wait_all();   // this thread's copies of pair q + 1 have landed
            __syncthreads();       // everyone's; pair q's sums are formed, pair q - 1 is added
            stage(q + 2);          // into the slot that pair q - 1 used
            form(q + 1);
            const int c = 2 * q;
            uint32_t w = w0 + (uint32_t)((q & 1) * S::kSums * 4);
            if (s_md[q]) {
                add(w, s_dl[c]);
            } else {
                if (DT == SPD_F32 && !has_sc) w = x0 + (uint32_t)((q % kDdRing) * 2 * S::kWin * 4);
                for (int e = c; e < min(c + 2, nc); ++e) {
                    if (s_sp[e] <= kDdSpread) add(w, s_dl[e]);
                    else add_global(e);
                }
            }
        }
        cp_async_wait_all();
    }
    __syncthreads();
    const uint32_t bad = s_bad;
    if (bad && status && tid == 0) atomicExch(&status->status, (int)SPD_ERR_INVALID_ARG);
#pragma unroll
    for (int d = 0; d < DMS; ++d) {
        if (d >= nd) break;
        const float nan = __int_as_float(0x7fc00000);
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int64_t t = t0 + tid + j * kDdThreads;
            if (t < n_out)
                store_out(out, out_dt, (d0 + d) * out_stride + t,
                          ((bad >> d) & 1u) ? nan : (j & 1) ? acc[d][j / 2].y : acc[d][j / 2].x);
        }
    }
}

template <int DT, int PER, int DMS>
cudaError_t launch_dd(const spd_plane *fb, const int32_t *delays, int64_t n_dm, void *out,
                      int out_dt, int64_t n_out, int64_t out_stride, spd_result *status,
                      cudaStream_t s) {
    using T = typename Elem<DT>::T;
    using S = DdShape<PER, DMS>;
    const int64_t ctas = (n_out + S::kSpan - 1) / S::kSpan * ((n_dm + DMS - 1) / DMS);
    const size_t smem = S::smem(sizeof(T));
    auto k = dedisperse_kernel<DT, PER, DMS>;
    const cudaError_t e =
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k<<<(unsigned)ctas, kDdThreads, smem, s>>>(
        static_cast<const T *>(fb->data), fb->n_dm, fb->n_samp, fb->row_stride, fb->row_scale,
        fb->row_offset, delays, n_dm, out, out_dt, n_out, out_stride, status);
    return cudaGetLastError();
}

// The middle shape, 2 outputs of 16 trials per thread, where its CTAs all fit the
// chip at once (two per SM) but are not few.  Beyond that 4 outputs: 256 channels
// FP32, 48 trials x 60000 (354 CTAs of the middle shape) 260 us in the middle
// shape, 227 in the large one; 100 x 30000 (413) 263 and 212; but 256 x 8192
// (256) 140 and 154, 48 x 30000 (177) 157 and 177.  With few, CTAs of an eighth
// of the middle shape, which form each window for 4 trials only: FP32 48 x 16384
// (96) 126 in the middle shape and 170 in the small one, 256 x 2000 (64) 112 and
// 118, 100 x 4000 (56) 117 and 99, 16 x 30000 (59) 140 and 118; FP16 113 and 144 at
// 64, 122 and 126 at 56.  Planes of up to 4 trials that would take the large shape
// have it in blocks of 4 (one of 16 adds, and where a spread is wide reads, all
// 16): 128 x 3 x 262144 FP32 147 and 85 us, with delays to 1000 pc/cm3 283 and 140.
template <int DT>
cudaError_t launch_dd_dt(const spd_plane *fb, const int32_t *delays, int64_t n_dm, void *out,
                         int out_dt, int64_t n_out, int64_t out_stride, spd_result *status,
                         cudaStream_t s) {
    const int64_t b16 = (n_dm + 15) / 16;
    const int64_t ctas = (n_out + 511) / 512 * b16;
    if (ctas > 304 && n_dm <= 4)
        return launch_dd<DT, 4, 4>(fb, delays, n_dm, out, out_dt, n_out, out_stride, status, s);
    if (ctas > 304)
        return launch_dd<DT, 4, 16>(fb, delays, n_dm, out, out_dt, n_out, out_stride, status, s);
    if (ctas >= 64)
        return launch_dd<DT, 2, 16>(fb, delays, n_dm, out, out_dt, n_out, out_stride, status, s);
    return launch_dd<DT, 1, 4>(fb, delays, n_dm, out, out_dt, n_out, out_stride, status, s);
}

}  // namespace

extern "C" spd_status spd_dedisperse(const spd_plane *fb, const int32_t *delays, int64_t n_dm,
                                     void *out, int32_t out_dtype, int64_t n_out,
                                     int64_t out_stride, spd_result *status_dev, void *stream) {
    if (!fb || fb->dtype < SPD_F32 || fb->dtype > SPD_BF16) return SPD_ERR_INVALID_ARG;
    if (out_dtype < SPD_F32 || out_dtype > SPD_BF16) return SPD_ERR_INVALID_ARG;
    const int64_t n_chan = fb->n_dm, n_samp = fb->n_samp;
    if (n_chan < 0 || n_samp < 0 || n_dm < 0 || n_out < 0 || n_out > n_samp) return SPD_ERR_INVALID_ARG;
    if (n_dm == 0 || n_out == 0) return SPD_OK;
    if (n_chan == 0 || !fb->data || fb->row_stride < n_samp || !delays || !out ||
        out_stride < n_out)
        return SPD_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(fb->data) % elem_bytes(fb->dtype) ||
        reinterpret_cast<uintptr_t>(out) % elem_bytes(out_dtype) ||
        reinterpret_cast<uintptr_t>(delays) % 4)
        return SPD_ERR_INVALID_ARG;
    if (fb->row_offset && !fb->row_scale) return SPD_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // CTAs: fewer than this in the largest shape, and few in the smaller ones
    if ((n_out + 511) / 512 > INT32_MAX / ((n_dm + 15) / 16)) return SPD_ERR_INVALID_ARG;
    const cudaError_t e =
        fb->dtype == SPD_F32   ? launch_dd_dt<SPD_F32>(fb, delays, n_dm, out, out_dtype, n_out, out_stride, status_dev, st)
        : fb->dtype == SPD_F16 ? launch_dd_dt<SPD_F16>(fb, delays, n_dm, out, out_dtype, n_out, out_stride, status_dev, st)
                               : launch_dd_dt<SPD_BF16>(fb, delays, n_dm, out, out_dtype, n_out, out_stride, status_dev, st);
    if (e != cudaSuccess) {
        note_cuda_error((int)e);
        return SPD_ERR_CUDA;
    }
    return SPD_OK;
}
