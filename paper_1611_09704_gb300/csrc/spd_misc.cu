// spd_misc.cu -- step (d) on a stored SNR plane (Sec. 2.4), the per-DM
// clustering of its candidates, and the raw boxcar sums test aid.
#include "spd_internal.cuh"

#include <math.h>

namespace spd {

namespace {

constexpr int kThrThreads = 256;
constexpr int kThrPer = 8;                        // samples per thread
constexpr int kThrTile = kThrThreads * kThrPer;   // samples per CTA

// Every (dm, t) with snr >= thr becomes a record.  One atomicAdd per CTA on
// the global count (block-aggregated); records past `capacity` are counted
// but not written.
__global__ void __launch_bounds__(kThrThreads) threshold_kernel(
    const float *snr, const uint16_t *width, int64_t n_samp, int64_t stride,
    int64_t tiles_per_row, float thr, spd_candidate *out, int64_t capacity,
    spd_result *result) {
    __shared__ int s_wsum[kThrThreads / 32];
    __shared__ unsigned long long s_base;
    const int tid = threadIdx.x;
    const int64_t row = blockIdx.x / tiles_per_row;
    const int64_t t0 = (blockIdx.x - row * tiles_per_row) * (int64_t)kThrTile;
    const int64_t i0 = t0 + (int64_t)tid * kThrPer;
    const float *sp = snr + row * stride;
    const uint16_t *wp = width + row * stride;

    float v[kThrPer];
    int w[kThrPer];
    const bool vec = i0 + kThrPer <= n_samp &&
                     ((reinterpret_cast<uintptr_t>(sp + i0) & 15) == 0) &&
                     ((reinterpret_cast<uintptr_t>(wp + i0) & 15) == 0);
    if (vec) {
        const float4 a = __ldcs(reinterpret_cast<const float4 *>(sp + i0));
        const float4 b = __ldcs(reinterpret_cast<const float4 *>(sp + i0) + 1);
        const uint4 u = __ldcs(reinterpret_cast<const uint4 *>(wp + i0));
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
        v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
        w[0] = u.x & 0xffff; w[1] = u.x >> 16; w[2] = u.y & 0xffff; w[3] = u.y >> 16;
        w[4] = u.z & 0xffff; w[5] = u.z >> 16; w[6] = u.w & 0xffff; w[7] = u.w >> 16;
    } else {
#pragma unroll
        for (int k = 0; k < kThrPer; ++k) {
            const bool ok = i0 + k < n_samp;
            v[k] = ok ? sp[i0 + k] : -INFINITY;
            w[k] = ok ? wp[i0 + k] : 0;
        }
    }
    uint32_t mask = 0;
#pragma unroll
    for (int k = 0; k < kThrPer; ++k)
        if (i0 + k < n_samp && v[k] >= thr) mask |= 1u << k;
    const int cnt = __popc(mask);
    const int lane = tid & 31, warp = tid >> 5;
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
    }
    if (lane == 31) s_wsum[warp] = incl;
    __syncthreads();
    if (tid < 32) {
        const int wv = (lane < kThrThreads / 32) ? s_wsum[lane] : 0;
        int wi = wv;
#pragma unroll
        for (int o = 1; o < kThrThreads / 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += x;
        }
        if (lane < kThrThreads / 32) s_wsum[lane] = wi - wv;
        const int total = __shfl_sync(0xffffffffu, wi, kThrThreads / 32 - 1);
        if (lane == 0)
            s_base = total ? atomicAdd(reinterpret_cast<unsigned long long *>(&result->count),
                                       (unsigned long long)total)
                           : 0ull;
    }
    __syncthreads();
    if (cnt) {
        unsigned long long idx = s_base + (unsigned long long)(s_wsum[warp] + incl - cnt);
#pragma unroll
        for (int k = 0; k < kThrPer; ++k) {
            if (mask & (1u << k)) {
                if (idx < (unsigned long long)capacity) {
                    int4 rec;
                    rec.x = (int)row;
                    rec.y = (int)(i0 + k);
                    rec.z = __float_as_int(v[k]);
                    rec.w = w[k];
                    reinterpret_cast<int4 *>(out)[idx] = rec;
                }
                ++idx;
            }
        }
    }
}

// Raw boxcar sum of one width per output sample, compensated FP32 summation.
template <int DT>
__global__ void boxcar_sums_kernel(const spd_plane p, int w, float *out, int64_t out_stride) {
    using T = typename Elem<DT>::T;
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t r = blockIdx.y;
    if (i >= p.n_samp) return;
    float *o = out + r * out_stride + i;
    if (i + w > p.n_samp) {
        *o = __int_as_float(0x7fc00000);
        return;
    }
    const T *x = static_cast<const T *>(p.data) + r * p.row_stride + i;
    const bool has_sc = p.row_scale != nullptr;
    const float sc = has_sc ? p.row_scale[r] : 1.f;
    const float of = (has_sc && p.row_offset) ? p.row_offset[r] : 0.f;
    float s = 0.f, c = 0.f;
    for (int k = 0; k < w; ++k) {
        float v = Elem<DT>::cvt(x[k]);
        if (has_sc) v = fmaf(sc, v, of);
        const float y = v - c;
        const float t = s + y;
        c = (t - s) - y;
        s = t;
    }
    *o = s;
}

// Per-DM clustering of the candidates of an SNR plane.  A row is cut into
// segments, a warp each; a cluster belongs to the segment of its first
// candidate.  Its warp follows it past the segment's end; a warp whose
// segment begins inside a cluster (a candidate at most `gap` before its first
// one, found by looking back) passes over the rest of that one.  So the
// records are those of one walk along the whole row.
//
// A step is 32 consecutive samples, one per lane; 16 steps are loaded at once,
// and with no candidate among them are done with one vote.  In a step the
// candidates are a ballot mask, the lanes that start a cluster (more than
// `gap` past the last candidate before them: the previous set bit, else the
// open cluster's last) form a second mask, and each segment between starts is
// absorbed with a popcount and its highest set bit.  Every lane holds the same
// cluster state but for the peak, of which it keeps its own over order-
// preserving keys; one warp max when the cluster ends finds the lane that writes
// the record and reads the peak's width: the width plane is not streamed.
//
// Bound by the SNR plane's one read where candidates are few.  1024 x 262144
// samples: a warp per row left 7 warps per SM and streamed the widths too, 815
// us; now 169 us, 6.3 TB/s.  A cluster that runs through a row is one warp's
// walk, while the other segments' warps pass over their parts of it.  With a
// warp max for every step, and no way to take a load at once, such rows took
// longer than with a warp per row: gap 32, every sample a candidate 3.54 ms (a
// warp per row 1.95), now 1.85; gap 8 3.56 (1.95) and 2.28.
constexpr int kClusterWarps = 8;    // segments per CTA
constexpr int kClusterSteps = 16;   // 32-sample steps loaded at once per warp

// The open cluster: the same in every lane, but for the peak, of which a lane
// holds the highest of the members it has seen (the earliest among equals).
struct ClusterState {
    int first, last, members;
    unsigned key;
    float peak;
    int peak_t;
};

// Monotone map of a non-NaN float to an unsigned key (larger float, larger
// key; -0.0 and +0.0 compare equal, so they share one key); every key is
// > 0, so 0 stands for "no member".
__device__ __forceinline__ unsigned order_key(float f) {
    unsigned u = __float_as_uint(f);
    if (u == 0x80000000u) u = 0u;
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// The whole warp: the peak over its lanes; the lane that saw it writes the record.
__device__ __forceinline__ void emit_cluster(const ClusterState &c, int64_t row,
                                             const uint16_t *wp, spd_cluster *out,
                                             int64_t capacity, spd_result *result) {
    const unsigned top = __reduce_max_sync(0xffffffffu, c.key);
    const unsigned at = __reduce_min_sync(0xffffffffu, c.key == top ? (unsigned)c.peak_t : ~0u);
    if (c.key != top || (unsigned)c.peak_t != at) return;
    const int w = wp[c.peak_t];   // beside the atomic, not after it
    const unsigned long long idx =
        atomicAdd(reinterpret_cast<unsigned long long *>(&result->count), 1ull);
    if (idx < (unsigned long long)capacity) {
        spd_cluster r;
        r.dm = (int32_t)row;
        r.first = c.first;
        r.last = c.last;
        r.peak_sample = c.peak_t;
        r.peak_snr = c.peak;
        r.peak_width = w;
        r.members = c.members;
        r.reserved0 = 0;
        out[idx] = r;
    }
}

// The members M (a lane mask of this step, starting at sample t0) join the open
// cluster: count, last sample, and each lane's own peak (key: 0 where the lane's
// sample is no candidate).
__device__ __forceinline__ void absorb(ClusterState &c, unsigned M, int t0, unsigned key, float v,
                                       int lane) {
    c.members += __popc(M);
    c.last = t0 + (31 - __clz(M));
    const unsigned mine = ((M >> lane) & 1u) ? key : 0u;
    const bool up = mine > c.key;
    c.key = up ? mine : c.key;
    c.peak = up ? v : c.peak;
    c.peak_t = up ? t0 + lane : c.peak_t;
}

// All the candidates of a load's steps (samples from t0 on) join the open cluster
// when none of them starts one; else nothing changes and the result is false.
// One vote for all steps, where the walk below has one or two a step.
__device__ __forceinline__ bool join_steps(ClusterState &c, bool foreign,
                                           const float (&v)[kClusterSteps], float thr, int t0,
                                           int gap, int lane) {
    int last = c.last, members = 0;
    bool far = false;
#pragma unroll
    for (int k = 0; k < kClusterSteps; ++k) {
        const unsigned m = __ballot_sync(0xffffffffu, v[k] >= thr);
        if (m) {
            far |= t0 + 32 * k + __ffs(m) - 1 - last > gap;
            if (gap < 31) {   // more than gap samples between two of the step
                const unsigned below = m & ((1u << lane) - 1u);
                far |= ((m >> lane) & 1u) && below && lane - (31 - __clz(below)) > gap;
            }
            last = t0 + 32 * k + (31 - __clz(m));
            members += __popc(m);
        }
    }
    if (__any_sync(0xffffffffu, far)) return false;
    c.last = last;
    if (foreign) return true;
    c.members += members;
#pragma unroll
    for (int k = 0; k < kClusterSteps; ++k) {
        const unsigned key = v[k] >= thr ? order_key(v[k]) : 0u;
        if (key > c.key) {
            c.key = key;
            c.peak = v[k];
            c.peak_t = t0 + 32 * k + lane;
        }
    }
    return true;
}

__global__ void __launch_bounds__(32 * kClusterWarps) cluster_kernel(
    const float *snr, const uint16_t *width, int n_dm, int n, int64_t stride, float thr, int gap,
    int seg_len, int segs_per_row, spd_cluster *out, int64_t capacity, spd_result *result) {
    const int lane = threadIdx.x & 31;
    const int64_t sg = (int64_t)blockIdx.x * kClusterWarps + (threadIdx.x >> 5);
    const int64_t row = sg / segs_per_row;
    if (row >= n_dm) return;   // the whole warp
    const int a = (int)(sg - row * segs_per_row) * seg_len;
    const int b = n - a < seg_len ? n : a + seg_len;
    const float *sp = snr + row * stride;
    const uint16_t *wp = width + row * stride;
    bool open = false, foreign = false, looked = a == 0;
    int quiet = 0;   // loads since one in which a cluster started
    ClusterState c{0, 0, 0, 0u, 0.f, 0};
    // the segment, then on past its end while an own cluster is open
    for (int64_t base = a; base < n; base += 32 * kClusterSteps) {
        if (base >= b && (!open || foreign || base - c.last > gap)) break;
        float v[kClusterSteps];
        bool any = false;
#pragma unroll
        for (int k = 0; k < kClusterSteps; ++k) {
            const int64_t t = base + 32 * k + lane;
            v[k] = t < n ? __ldcs(sp + t) : __int_as_float(0x7fc00000);   // NaN: not a candidate
        }
#pragma unroll
        for (int k = 0; k < kClusterSteps; ++k) any |= v[k] >= thr;
        if (!__any_sync(0xffffffffu, any)) continue;
        // worth trying after some loads without a start: a load that has one is
        // gone over twice (gap 8, clusters of 500 samples: 1.13 ms never tried,
        // 1.20 after four such loads, 1.48 after two)
        if (quiet >= 4 && join_steps(c, foreign, v, thr, (int)base, gap, lane)) continue;
        ++quiet;
#pragma unroll
        for (int k = 0; k < kClusterSteps; ++k) {
            const bool cand = v[k] >= thr;
            const unsigned m = __ballot_sync(0xffffffffu, cand);
            if (!m) continue;
            const int t0 = (int)(base + 32 * k);
            if (!looked) {   // the segment's first candidate: in a cluster from before it?
                looked = true;
                const int t1 = t0 + __ffs(m) - 1;
                for (int q = a; q > 0 && t1 - (q - 1) <= gap && !foreign; q -= 32) {
                    const int p = q - 32 + lane;
                    const bool hit = p >= 0 && t1 - p <= gap && sp[p] >= thr;
                    foreign = __any_sync(0xffffffffu, hit);
                }
                if (foreign) {
                    open = true;
                    c.last = t1 - 1;   // any sample at most gap before it
                }
            }
            const unsigned key = cand ? order_key(v[k]) : 0u;
            // a gap of 31 or more spans what lies between two set bits: all join
            if (gap >= 31 && open && t0 + __ffs(m) - 1 - c.last <= gap) {
                absorb(c, m, t0, key, v[k], lane);
                continue;
            }
            // does this lane's candidate start a cluster?
            const unsigned below = m & ((1u << lane) - 1u);
            const bool has_prev = below != 0u || open;
            const int prev = below ? t0 + (31 - __clz(below)) : c.last;
            const bool start = cand && (!has_prev || (t0 + lane) - prev > gap);
            unsigned S = __ballot_sync(0xffffffffu, start);
            // members before the first start continue the open cluster
            const int fs = S ? __ffs(S) - 1 : 32;
            const unsigned cont = fs == 32 ? m : (m & ((1u << fs) - 1u));
            if (cont) absorb(c, cont, t0, key, v[k], lane);   // a foreign one's is never written
            if (S) quiet = 0;
            while (S) {
                const int s0 = __ffs(S) - 1;
                S &= S - 1u;
                const int e = S ? __ffs(S) - 1 : 32;
                const unsigned seg = m & (0xffffffffu << s0) & (e == 32 ? 0xffffffffu : ((1u << e) - 1u));
                if (open && !foreign) emit_cluster(c, row, wp, out, capacity, result);
                open = t0 + s0 < b;   // one that starts past the segment is the next one's
                foreign = false;
                if (!open) return;
                c.first = t0 + s0;
                c.members = 0;
                c.key = 0u;
                absorb(c, seg, t0, key, v[k], lane);
            }
        }
    }
    if (open && !foreign) emit_cluster(c, row, wp, out, capacity, result);
}

}  // namespace

// Thresholding of Sec. 2.4 on the plane, in place: 8 samples per thread,
// 128-bit accesses where the row allows.  Only what changes is written, and a
// width is read only where some of its 8 neighbours stay: 10 bytes a sample
// below the threshold and 4 above it, where reading and writing both planes
// took 12 (512 x 262144 with 38 % kept: 228 -> 149 us).
__global__ void __launch_bounds__(256) threshold_plane_kernel(float *snr, uint16_t *width,
                                                              int64_t n_samp, int64_t stride,
                                                              float thr) {
    const int64_t row = blockIdx.y;
    const int64_t i0 = ((int64_t)blockIdx.x * 256 + threadIdx.x) * 8;
    if (i0 >= n_samp) return;
    float *sp = snr + row * stride;
    uint16_t *wp = width ? width + row * stride : nullptr;
    const bool vec = i0 + 8 <= n_samp && ((reinterpret_cast<uintptr_t>(sp + i0) & 15) == 0) &&
                     (!wp || (reinterpret_cast<uintptr_t>(wp + i0) & 15) == 0);
    if (vec) {
        float4 a = reinterpret_cast<float4 *>(sp + i0)[0];
        float4 b = reinterpret_cast<float4 *>(sp + i0)[1];
        const bool k[8] = {a.x >= thr, a.y >= thr, a.z >= thr, a.w >= thr,
                           b.x >= thr, b.y >= thr, b.z >= thr, b.w >= thr};
        const bool ka = k[0] & k[1] & k[2] & k[3], kb = k[4] & k[5] & k[6] & k[7];
        if (ka && kb) return;   // all stay
        a.x = k[0] ? a.x : 0.f; a.y = k[1] ? a.y : 0.f; a.z = k[2] ? a.z : 0.f;
        a.w = k[3] ? a.w : 0.f; b.x = k[4] ? b.x : 0.f; b.y = k[5] ? b.y : 0.f;
        b.z = k[6] ? b.z : 0.f; b.w = k[7] ? b.w : 0.f;
        if (!ka) reinterpret_cast<float4 *>(sp + i0)[0] = a;
        if (!kb) reinterpret_cast<float4 *>(sp + i0)[1] = b;
        if (wp) {
            uint4 u = make_uint4(0u, 0u, 0u, 0u);
            if (k[0] | k[1] | k[2] | k[3] | k[4] | k[5] | k[6] | k[7]) {
                u = reinterpret_cast<uint4 *>(wp + i0)[0];
                uint32_t *uw = reinterpret_cast<uint32_t *>(&u);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t lo = k[2 * q] ? (uw[q] & 0xffffu) : 0u;
                    const uint32_t hi = k[2 * q + 1] ? (uw[q] & 0xffff0000u) : 0u;
                    uw[q] = lo | hi;
                }
            }
            reinterpret_cast<uint4 *>(wp + i0)[0] = u;
        }
        return;
    }
    for (int q = 0; q < 8 && i0 + q < n_samp; ++q) {
        const bool keep = sp[i0 + q] >= thr;
        if (!keep) {
            sp[i0 + q] = 0.f;
            if (wp) wp[i0 + q] = 0;
        }
    }
}

cudaError_t launch_threshold_plane(float *snr, uint16_t *width, int64_t n_dm, int64_t n_samp,
                                   int64_t stride, float thr, cudaStream_t s) {
    if (n_dm <= 0 || n_samp <= 0) return cudaSuccess;
    const int64_t per = 256 * 8;
    int64_t y = n_dm;
    for (int64_t r0 = 0; r0 < n_dm; r0 += 65535) {   // grid.y limit
        y = n_dm - r0 < 65535 ? n_dm - r0 : 65535;
        const dim3 grid((unsigned)((n_samp + per - 1) / per), (unsigned)y);
        threshold_plane_kernel<<<grid, 256, 0, s>>>(snr + r0 * stride,
                                                    width ? width + r0 * stride : nullptr,
                                                    n_samp, stride, thr);
    }
    return cudaGetLastError();
}

// Rows of a halo or a chunk from one pitch to another, where the two may lie
// differently to 16-byte boundaries (a stream's halo is wmax - 1 samples long,
// so its chunk follows at any element step).  One 16-byte piece of the
// destination per thread: from one piece of the source or, shifted, from the
// two it lies in; the pieces at a row's ends, and those whose source pieces
// stick out of the source, element by element.  2048 x 32768 FP16 at an odd
// step: a 2-D copy by the runtime took 0.1 ms, this 0.04.
template <typename T>
__global__ void __launch_bounds__(256) copy_rows_kernel(char *dst, int64_t dst_stride,
                                                        const char *src, int64_t src_stride,
                                                        int64_t width, int64_t pieces,
                                                        int64_t n_rows) {
    const int64_t idx = (int64_t)blockIdx.x * 256 + threadIdx.x;
    const int64_t row = gridDim.x < (1u << 24) ? (uint32_t)idx / (uint32_t)pieces : idx / pieces;
    if (row >= n_rows) return;
    char *d0 = dst + row * dst_stride;
    const char *s0 = src + row * src_stride;
    const char *end = src + (n_rows - 1) * src_stride + width;
    // the piece's first byte, from the row's start (negative: before it)
    const int64_t o = (idx - row * pieces) * 16 - (int64_t)(reinterpret_cast<uintptr_t>(d0) & 15);
    if (o >= width) return;
    const char *p = s0 + o;
    const uint32_t m = (uint32_t)(reinterpret_cast<uintptr_t>(p) & 15);
    if (o >= 0 && o + 16 <= width && p - m >= src && p - m + (m ? 32 : 16) <= end) {
        uint4 a = __ldg(reinterpret_cast<const uint4 *>(p - m));
        if (m) {
            const uint4 b = __ldg(reinterpret_cast<const uint4 *>(p - m) + 1);
            uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
            const uint32_t k = m >> 2, half = (m & 2) * 8u;
#pragma unroll
            for (int i = 0; i < 7; ++i) w[i] = (k & 1) ? w[i + 1] : w[i];
#pragma unroll
            for (int i = 0; i < 6; ++i) w[i] = (k & 2) ? w[i + 2] : w[i];
            a = make_uint4(__funnelshift_r(w[0], w[1], half), __funnelshift_r(w[1], w[2], half),
                           __funnelshift_r(w[2], w[3], half), __funnelshift_r(w[3], w[4], half));
        }
        *reinterpret_cast<uint4 *>(d0 + o) = a;
        return;
    }
    for (int64_t e = o < 0 ? 0 : o; e < o + 16 && e < width; e += (int64_t)sizeof(T))
        *reinterpret_cast<T *>(d0 + e) = *reinterpret_cast<const T *>(s0 + e);
}

cudaError_t launch_copy_rows(void *dst, int64_t dst_stride, const void *src, int64_t src_stride,
                             int64_t width, int64_t n_rows, int esz, cudaStream_t s) {
    if (width <= 0 || n_rows <= 0) return cudaSuccess;
    const int64_t pieces = width / 16 + 2;   // a row may begin and end inside one
    const int64_t blocks = (n_rows * pieces + 255) / 256;
    if (blocks > INT32_MAX) return cudaErrorInvalidValue;
    char *d = static_cast<char *>(dst);
    const char *p = static_cast<const char *>(src);
    if (esz == 2)
        copy_rows_kernel<uint16_t><<<(unsigned)blocks, 256, 0, s>>>(d, dst_stride, p, src_stride,
                                                                    width, pieces, n_rows);
    else
        copy_rows_kernel<uint32_t><<<(unsigned)blocks, 256, 0, s>>>(d, dst_stride, p, src_stride,
                                                                    width, pieces, n_rows);
    return cudaGetLastError();
}

// Decimation in time: up to four levels of a plane in one pass, level k + 1
// from level k: dst_k[r][j] = dst_{k-1}[r][2j] + dst_{k-1}[r][2j+1] in FP32
// (dst_-1: the dequantised source).  A thread sums 16 consecutive source
// samples to 8, 4, 2 and 1 outputs.  Level by level, 1024 x 262144 FP32 down
// to 1/16 read 2.0 GB and took 492 us; this reads the source once.
struct DecimateArgs {
    const void *src;
    int64_t src_stride, n_src;
    const float *scale, *offset;
    float *dst[4];              // null: not wanted
    int64_t stride[4], n[4];    // n[k] = n_src >> (k + 1)
    int vec_ok;                 // 16-byte aligned rows
};

template <int DT>
__global__ void __launch_bounds__(256) decimate_kernel(const __grid_constant__ DecimateArgs a) {
    using T = typename Elem<DT>::T;
    const int64_t row = blockIdx.y;
    const int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x;
    const int64_t i0 = 16 * t;
    if (i0 >= a.n_src) return;
    const T *sp = static_cast<const T *>(a.src) + row * a.src_stride + i0;
    float v[16];
    if (a.vec_ok && i0 + 16 <= a.n_src) {
        constexpr int kVec = DT == SPD_F32 ? 4 : 2;
#pragma unroll
        for (int q = 0; q < kVec; ++q) {
            const uint4 u = __ldg(reinterpret_cast<const uint4 *>(sp) + q);
            const T *e = reinterpret_cast<const T *>(&u);
#pragma unroll
            for (int k = 0; k < 16 / kVec; ++k) v[16 / kVec * q + k] = Elem<DT>::cvt(e[k]);
        }
    } else {
#pragma unroll
        for (int q = 0; q < 16; ++q) v[q] = i0 + q < a.n_src ? Elem<DT>::cvt(sp[q]) : 0.f;
    }
    if (a.scale) {
        const float sc = a.scale[row], of = a.offset ? a.offset[row] : 0.f;
#pragma unroll
        for (int q = 0; q < 16; ++q) v[q] = fmaf(sc, v[q], of);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int m = 8 >> k;              // outputs of this level
#pragma unroll
        for (int q = 0; q < m; ++q) v[q] = __fadd_rn(v[2 * q], v[2 * q + 1]);
        if (!a.dst[k]) continue;
        const int64_t j0 = t * m;
        float *d = a.dst[k] + row * a.stride[k] + j0;
        if (j0 + m <= a.n[k]) {
            if (m >= 4) {
#pragma unroll
                for (int q = 0; q < m; q += 4)
                    *reinterpret_cast<float4 *>(d + q) = make_float4(v[q], v[q + 1], v[q + 2], v[q + 3]);
            } else if (m == 2) {
                *reinterpret_cast<float2 *>(d) = make_float2(v[0], v[1]);
            } else {
                *d = v[0];
            }
        } else {
#pragma unroll
            for (int q = 0; q < m; ++q)
                if (j0 + q < a.n[k]) d[q] = v[q];
        }
    }
}

cudaError_t launch_decimate(const spd_plane &p, float *const *dst, const int64_t *stride, int levels,
                            cudaStream_t s) {
    if (p.n_dm <= 0 || p.n_samp < 2) return cudaSuccess;
    for (int64_t r0 = 0; r0 < p.n_dm; r0 += 65535) {   // grid.y limit
        const int64_t y = p.n_dm - r0 < 65535 ? p.n_dm - r0 : 65535;
        const size_t eb = elem_bytes(p.dtype);
        DecimateArgs a;
        a.src = static_cast<const char *>(p.data) + r0 * p.row_stride * (int64_t)eb;
        a.src_stride = p.row_stride;
        a.n_src = p.n_samp;
        a.scale = p.row_scale ? p.row_scale + r0 : nullptr;
        a.offset = p.row_offset ? p.row_offset + r0 : nullptr;
        for (int k = 0; k < 4; ++k) {
            a.dst[k] = k < levels && dst[k] ? dst[k] + r0 * stride[k] : nullptr;
            a.stride[k] = k < levels ? stride[k] : 0;
            a.n[k] = p.n_samp >> (k + 1);
        }
        a.vec_ok = reinterpret_cast<uintptr_t>(a.src) % 16 == 0 && (p.row_stride * (int64_t)eb) % 16 == 0;
        const dim3 grid((unsigned)((p.n_samp + 4095) / 4096), (unsigned)y);
        switch (p.dtype) {
            case SPD_F32: decimate_kernel<SPD_F32><<<grid, 256, 0, s>>>(a); break;
            case SPD_F16: decimate_kernel<SPD_F16><<<grid, 256, 0, s>>>(a); break;
            default: decimate_kernel<SPD_BF16><<<grid, 256, 0, s>>>(a); break;
        }
    }
    return cudaGetLastError();
}

cudaError_t launch_threshold(const float *snr, const uint16_t *width, int64_t n_dm,
                             int64_t n_samp, int64_t stride, float thr, spd_candidate *out,
                             int64_t capacity, spd_result *result, cudaStream_t s) {
    const int64_t tpr = (n_samp + kThrTile - 1) / kThrTile;
    const int64_t tiles = n_dm * tpr;
    if (tiles <= 0) return cudaSuccess;
    threshold_kernel<<<(unsigned)tiles, kThrThreads, 0, s>>>(snr, width, n_samp, stride, tpr,
                                                             thr, out, capacity, result);
    return cudaGetLastError();
}

cudaError_t launch_cluster(const float *snr, const uint16_t *width, int64_t n_dm,
                           int64_t n_samp, int64_t stride, float thr, int64_t gap,
                           spd_cluster *out, int64_t capacity, spd_result *result,
                           cudaStream_t s) {
    if (n_dm <= 0 || n_samp <= 0) return cudaSuccess;
    // segments: about 32768 (200 per SM), of at least 4096 samples (a warp's
    // fixed work is that of some 512) and at least 4 gaps (looking back reads
    // one)
    const int64_t step = 32 * kClusterSteps;
    if (gap > n_samp) gap = n_samp;
    int64_t len = (n_dm * n_samp / 32768 + step - 1) / step * step;
    if (len < 4096) len = 4096;
    if (len < 4 * gap) len = (4 * gap + step - 1) / step * step;
    if (len > n_samp) len = n_samp;
    const int64_t per_row = (n_samp + len - 1) / len;
    const int64_t blocks = (n_dm * per_row + kClusterWarps - 1) / kClusterWarps;
    cluster_kernel<<<(unsigned)blocks, 32 * kClusterWarps, 0, s>>>(
        snr, width, (int)n_dm, (int)n_samp, stride, thr, (int)gap, (int)len, (int)per_row, out,
        capacity, result);
    return cudaGetLastError();
}

cudaError_t launch_boxcar_sums(const spd_plane &p, int w, float *out, int64_t out_stride,
                               cudaStream_t s) {
    if (p.n_dm <= 0 || p.n_samp <= 0) return cudaSuccess;
    const dim3 grid((unsigned)((p.n_samp + 255) / 256), (unsigned)p.n_dm);
    switch (p.dtype) {
        case SPD_F32: boxcar_sums_kernel<SPD_F32><<<grid, 256, 0, s>>>(p, w, out, out_stride); break;
        case SPD_F16: boxcar_sums_kernel<SPD_F16><<<grid, 256, 0, s>>>(p, w, out, out_stride); break;
        default: boxcar_sums_kernel<SPD_BF16><<<grid, 256, 0, s>>>(p, w, out, out_stride); break;
    }
    return cudaGetLastError();
}

}  // namespace spd
