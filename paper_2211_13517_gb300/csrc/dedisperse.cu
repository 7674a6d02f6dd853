// Incoherent dedispersion: the stage that turns a filterbank into the
// DM-trial series the search runs on (the paper's workload is 5925 DM trials,
// §3; the paper does not describe this stage, so the textbook definition is
// used).
//
// Channel c has centre frequency f_c = f_top - c df (MHz, descending).  At
// DM_d = dm_lo + d dm_step the cold-plasma delay of channel c relative to the
// top of the band, in samples, is
//
//     Delta(c, d) = floor(K_DM DM_d (f_c^-2 - f_top^-2) / tsamp + 1/2),
//     K_DM = 4.148808e3 MHz^2 pc^-1 cm^3 s,
//
// and the dedispersed series is out[d][t] = sum_c in[c][t + Delta(c, d)],
// samples at or past n_t counted as 0.  The delays are computed once per plan
// in FP64 with every operation rounded separately (no contraction), so they
// are exactly those of the same formula evaluated in IEEE FP64 elsewhere.
//
// Plain kernel (by channel groups: further down): a CTA owns 32 DM trials x 512
// output samples.  Per batch of channels it stages, for each channel, the window
// of input samples its 32 DMs read (512 + the spread of their delays) in shared
// memory by asynchronous 4-byte copies (cp.async, zero-filled past n_t), double
// buffered so that the copies of the next batch run during the sums of this
// one.  Warp w accumulates DMs 4w..4w+3, lane l the samples l + 32k (k < 16),
// reading shared memory with consecutive lanes on consecutive words; where
// two DMs of a pair have the same delay for a channel (common at high
// frequency and small DM steps) one load feeds both.  FP32 sums over the
// channels in channel order; the bound is shared-memory bandwidth (one 4-byte
// word per lane per addition, less with shared delays).
#include <algorithm>
#include <cmath>
#include <new>
#include <string>
#include <vector>

#include "fdas_internal.cuh"

namespace fdas {
namespace {

constexpr int kDdT = 512;        // output samples per tile
constexpr int kDdD = 32;         // DM trials per tile
constexpr int kDdThreads = 256;  // 8 warps x 4 DM trials
constexpr int kDdPer = kDdT / 32;
constexpr double kDm = 4.148808e3;
constexpr size_t kDdSmemCap = 200 * 1024;   // both buffers
constexpr size_t kGrSmem = 222 * 1024;      // by groups: all CTAs of an SM

__global__ void dm_delay_kernel(int32_t *__restrict__ out, int n_chan, int n_dm, double f_top,
                                double df, double tsamp, double dm_lo, double dm_step) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)n_chan * n_dm) return;
    const int d = (int)(i / n_chan), c = (int)(i % n_chan);
    const double f = __dsub_rn(f_top, __dmul_rn((double)c, df));
    const double a = __ddiv_rn(1.0, __dmul_rn(f, f));
    const double b = __ddiv_rn(1.0, __dmul_rn(f_top, f_top));
    const double dm = __dadd_rn(dm_lo, __dmul_rn((double)d, dm_step));
    const double x = __ddiv_rn(__dmul_rn(__dmul_rn(kDm, dm), __dsub_rn(a, b)), tsamp);
    out[i] = (int32_t)floor(__dadd_rn(x, 0.5));
}

// 4-byte global -> shared copy, zero-filled when `valid` is false
__device__ __forceinline__ void cp_async4(float *dst, const float *src, bool valid) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src),
                 "r"(valid ? 4 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// 16-byte global -> shared copy of the first `valid` bytes (the rest zero)
__device__ __forceinline__ void cp_async16(void *dst, const void *src, int valid) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(valid)
                 : "memory");
}

// acc_a += w[oa + 32k], acc_b += w[ob + 32k]; one load when oa == ob
template <class T, class A>
__device__ __forceinline__ void add_pair(const T *w, int oa, int ob, A (&acc_a)[kDdPer],
                                         A (&acc_b)[kDdPer]) {
    if (oa == ob) {
#pragma unroll
        for (int k = 0; k < kDdPer; ++k) {
            const A v = (A)w[oa + 32 * k];
            acc_a[k] += v;
            acc_b[k] += v;
        }
    } else {
#pragma unroll
        for (int k = 0; k < kDdPer; ++k) {
            acc_a[k] += (A)w[oa + 32 * k];
            acc_b[k] += (A)w[ob + 32 * k];
        }
    }
}

// Input sample type T: FP32 samples sum in FP32 (4-byte asynchronous copies
// of each window, `pitch` = win elements per channel); 8-bit samples sum in
// int32, exactly (16-byte copies of the window rounded out to 16-byte
// boundaries, `pitch` = win + 16 bytes per channel, rows 16-byte aligned).
template <class T>
struct DdIn;
template <>
struct DdIn<float> {
    using Acc = float;
    static constexpr int kPad = 0;
};
template <>
struct DdIn<uint8_t> {
    using Acc = int;
    static constexpr int kPad = 16;
};

template <class T>
__global__ void __launch_bounds__(kDdThreads, 2)
    dedisperse_kernel(const T *__restrict__ fb, const int32_t *__restrict__ delays,
                      float *__restrict__ out, int n_chan, int64_t n_t, int n_dm, int64_t n_out,
                      int win, int chan_batch) {
    using Acc = typename DdIn<T>::Acc;
    extern __shared__ __align__(16) unsigned char dd_smem[];   // [2][chan_batch][pitch] of T
    T *sw = reinterpret_cast<T *>(dd_smem);
    const int pitch = win + DdIn<T>::kPad;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t t0 = (int64_t)blockIdx.x * kDdT;
    const int d_lo = blockIdx.y * kDdD;
    const int32_t *dl = delays + (int64_t)d_lo * n_chan;
    // this warp's four DM trials (clamped: rows past n_dm are not stored)
    const int32_t *dw[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) dw[q] = delays + (int64_t)min(d_lo + 4 * warp + q, n_dm - 1) * n_chan;
    Acc acc[4][kDdPer];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int k = 0; k < kDdPer; ++k) acc[q][k] = 0;

    const size_t buf_elems = (size_t)chan_batch * pitch;
    auto stage = [&](int cb, int slot) {
        const int nc = min(chan_batch, n_chan - cb);
        T *dst0 = sw + slot * buf_elems;
        for (int j = 0; j < nc; ++j) {
            const int64_t base = t0 + __ldg(dl + cb + j);
            const T *src = fb + (int64_t)(cb + j) * n_t;
            T *dst = dst0 + (size_t)j * pitch;
            if constexpr (sizeof(T) == 4) {
                for (int i = threadIdx.x; i < win; i += kDdThreads) {
                    const int64_t s = base + i;
                    const bool ok = s < n_t;
                    cp_async4(dst + i, src + (ok ? s : 0), ok);
                }
            } else {
                const int64_t b16 = base & ~(int64_t)15;
                for (int i = threadIdx.x; i < pitch / 16; i += kDdThreads) {
                    const int64_t s = b16 + 16 * (int64_t)i;
                    const int64_t left = n_t - s;
                    const int valid = left <= 0 ? 0 : (left >= 16 ? 16 : (int)left);
                    cp_async16(dst + 16 * i, src + (valid > 0 ? s : 0), valid);
                }
            }
        }
        cp_async_commit();
    };

    stage(0, 0);
    int slot = 0;
    for (int cb = 0; cb < n_chan; cb += chan_batch, slot ^= 1) {
        const int nc = min(chan_batch, n_chan - cb);
        if (cb + chan_batch < n_chan) {
            stage(cb + chan_batch, slot ^ 1);
            cp_async_wait<1>();   // this batch has landed (the next may be in flight)
        } else {
            cp_async_wait<0>();
        }
        __syncthreads();
        const T *buf = sw + slot * buf_elems + lane;
        for (int j = 0; j < nc; ++j) {
            const int c = cb + j;
            const int lo = __ldg(dl + c);
            // 8-bit windows start at the 16-byte boundary below the first sample
            const int shift = sizeof(T) == 1 ? (int)((t0 + lo) & 15) : 0;
            const T *w = buf + (size_t)j * pitch + shift;
            add_pair(w, __ldg(dw[0] + c) - lo, __ldg(dw[1] + c) - lo, acc[0], acc[1]);
            add_pair(w, __ldg(dw[2] + c) - lo, __ldg(dw[3] + c) - lo, acc[2], acc[3]);
        }
        __syncthreads();   // every warp is done with this slot before it is refilled
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int d = d_lo + 4 * warp + q;
        if (d >= n_dm) continue;
        float *row = out + (int64_t)d * n_out;
#pragma unroll
        for (int k = 0; k < kDdPer; ++k) {
            const int64_t t = t0 + lane + 32 * k;
            if (t < n_out) row[t] = (float)acc[q][k];
        }
    }
}

// ---------------------------------------------------------------------------
// Dedispersion by channel groups.
//
// The delays of up to 4 neighbouring channels differ by a few samples, and
// over the 32 DM trials of a tile they do so in only a few ways: a "pattern"
// is the tuple of the channels' shifts relative to the first one (3.7 patterns
// per group of 4 on average for 1024 channels of 0.25 MHz below 1670 MHz and 32
// trials 0.25 pc cm^-3 apart).  So the channels of a group are summed once per
// pattern into shared memory, and every DM trial adds one value per group
// instead of one per channel: the plain kernel's bound, one shared-memory load
// per addition, falls by nearly the group's size.
//
// A CTA owns 32 DM trials x 512 output samples, as the plain kernel does.  Per
// batch of groups: the windows of the batch's channels arrive by asynchronous
// copies (the next batch's are in flight meanwhile); the warps form the
// pattern sums, sorted so that a pattern keeps the partial sums of the leading
// channels it shares with the one before; then warp w adds to the DM trials
// 4w .. 4w+3 at each trial's offset.  FP32: sums of a group's channels in
// channel order, groups in order.  8-bit: sums as pairs of 16-bit integers (two
// samples per word and addition), stored twice, the second time one sample
// further on, so that odd offsets find aligned words too; 32-bit totals every
// 64 groups (64 * 4 * 255 < 2^16).  Exact.
//
// Bound: instruction issue (2.4 a cycle) and the two barriers per batch.  With 8-bit
// samples the pattern sums take 43 % of the time, the trials' additions 26 %,
// staging and barriers the rest (each part left out in turn).  So a batch takes
// the groups whose pattern sums fill the 8 warps best (8-bit: 2 pieces of 372
// samples for 32 trials 71 samples apart, 4 groups; with 3 pieces of 248 samples
// 6.63 ms below), its sums lie packed in shared memory (a place for the most
// patterns of any group left room for 2 groups only: 7.04), and what a piece
// reads again for each pattern stays in registers (7.35 without).
// Measured: 1024 channels of 8-bit samples, 128 trials, 2^20 outputs 5.90 ms
// (plain kernel 18.7); 300 FP32 channels, 75 trials, 262181 outputs 0.60 ms
// (1.32).
// ---------------------------------------------------------------------------
constexpr int kGrMax = 4;         // channels per group
constexpr int kGrPat = 8;         // patterns per group
constexpr int kGrBatchMax = 8;    // groups per batch
constexpr int kGrFlush = 64;      // groups between 32-bit totals (8-bit samples)
// samples of a pattern sum that a warp forms at a time
template <class T>
constexpr int kGrCtas = sizeof(T) == 4 ? 2 : 3;   // CTAs per SM
template <class T>
constexpr int kGrChunk = sizeof(T) == 4 ? 160 : 372;
constexpr int kGrPer = 5;         // FP32 samples of a chunk per lane

// one group of a DM tile as the kernel reads it (whole 16-byte copies)
struct GrRec {
    int32_t c0, nk;               // first channel, channels
    int16_t np, y0[2], pad;       // patterns; patterns of the batch's groups before (FP32, 8-bit)
    int32_t first[kGrMax];        // delay of channel k in the tile's first trial
    int16_t pat[kGrPat + 2][4];   // [0]: first channel that differs from the pattern
                                  // before; [k]: shift of channel k (one is read ahead)
    // per DM the first word of its samples among the batch's pattern sums, of
    // FP32 and of 8-bit samples (words of two; odd offsets in the second copy)
    int32_t off[2][kDdD];
};
static_assert(sizeof(GrRec) % 16 == 0, "whole 16-byte copies");

// 12 samples (six 16-bit pairs) of an 8-bit window from byte `at` + 12 lane on
__device__ __forceinline__ void add12_u8(const uint8_t *x, int at, int lane, uint32_t (&v)[6]) {
    const uint32_t *w = reinterpret_cast<const uint32_t *>(x) + (at >> 2) + 3 * lane;
    const uint32_t a[4] = {w[0], w[1], w[2], w[3]};
    const unsigned sh = 8u * (unsigned)(at & 3);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const uint32_t b = __funnelshift_r(a[i], a[i + 1], sh);
        v[2 * i] += __byte_perm(b, 0u, 0x4140u);
        v[2 * i + 1] += __byte_perm(b, 0u, 0x4342u);
    }
}

// shared-memory geometry: per slot the channel windows (xpitch bytes each) and
// the batch's records; then the pattern sums (ypitch words each)
template <class T>
__global__ void __launch_bounds__(kDdThreads, kGrCtas<T>)
    dedisperse_group_kernel(const T *__restrict__ fb, const GrRec *__restrict__ recs,
                            const int32_t *__restrict__ n_groups, int max_groups,
                            float *__restrict__ out, int64_t n_t, int n_dm, int64_t n_out, int chunks,
                            int lead, int xpitch, int ypitch, int batch) {
    constexpr bool kU8 = sizeof(T) == 1;
    extern __shared__ __align__(16) unsigned char dd_smem[];
    const int slot_bytes = batch * (kGrMax * xpitch + (int)sizeof(GrRec));
    uint32_t *const Y = reinterpret_cast<uint32_t *>(dd_smem + 2 * slot_bytes);
    __shared__ __align__(16) int32_t shift[2][kGrBatchMax * kGrMax];   // of each window's first sample
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t t0 = (int64_t)blockIdx.x * kDdT;
    const int d_lo = blockIdx.y * kDdD;
    const GrRec *rec = recs + (int64_t)blockIdx.y * max_groups;
    const int ng = n_groups[blockIdx.y];
    auto slot_rec = [&](int slot) {
        return reinterpret_cast<const GrRec *>(dd_smem + slot * slot_bytes +
                                               batch * kGrMax * xpitch);
    };
    auto stage = [&](int g0, int slot) {
        const int n = min(batch, ng - g0);
        unsigned char *base = dd_smem + slot * slot_bytes;
        unsigned char *rd = base + batch * kGrMax * xpitch;
        for (int i = threadIdx.x; i < n * (int)(sizeof(GrRec) / 16); i += kDdThreads)
            cp_async16(rd + 16 * i, reinterpret_cast<const unsigned char *>(rec + g0) + 16 * i, 16);
        // one warp per channel
        for (int i = warp; i < n * kGrMax; i += kDdThreads / 32) {
            const int g = i / kGrMax, k = i % kGrMax;
            const int2 head = __ldg(reinterpret_cast<const int2 *>(rec + g0 + g));   // c0, nk
            const int delay = __ldg(&rec[g0 + g].first[k]);
            if (k >= head.y) continue;
            const int c = head.x + k;
            // the window starts `lead` samples early (shifts may be negative),
            // rounded down to an address of a multiple of 16 bytes
            const int64_t first = t0 + delay - lead;
            const T *src = fb + (int64_t)c * n_t;
            constexpr int kV = 16 / (int)sizeof(T);
            const int a = (int)((reinterpret_cast<uintptr_t>(src + first) / sizeof(T)) % kV);
            T *dst = reinterpret_cast<T *>(base + i * xpitch);
            if (lane == 0) shift[slot][i] = lead + a;
            if (first - a >= 0 && first - a + xpitch / (int)sizeof(T) <= n_t) {
                const T *from = src + (first - a);
                for (int j = lane; j < xpitch / 16; j += 32)
                    cp_async16(dst + kV * j, from + kV * j, 16);
                continue;
            }
            for (int j = lane; j < xpitch / 16; j += 32) {
                const int64_t s = first - a + kV * j;
                if (s >= n_t) {
                    // past the last sample: no copy, whose address would have to be
                    // inside the row and aligned (rows start anywhere on 4 bytes)
                    *reinterpret_cast<uint4 *>(dst + kV * j) = make_uint4(0u, 0u, 0u, 0u);
                } else if (s >= 0) {
                    const int64_t left = n_t - s;
                    cp_async16(dst + kV * j, src + s, left >= kV ? 16 : (int)left * (int)sizeof(T));
                } else {
                    // before the first sample: zeros, then element by element
#pragma unroll
                    for (int x = 0; x < kV; ++x)
                        dst[kV * j + x] = s + x >= 0 && s + x < n_t ? src[s + x] : (T)0;
                }
            }
        }
        cp_async_commit();
    };

    // 8-bit: the 32-bit totals, touched every 64 groups only, stay in local
    // memory (reached through a pointer the compiler cannot see through), which
    // leaves the registers for a third CTA per SM
    using Acc = typename DdIn<T>::Acc;
    Acc acc[4][kDdPer];
    Acc *total = &acc[0][0];
    if constexpr (kU8) asm volatile("" : "+l"(total) : : "memory");
    uint32_t part[4][kU8 ? kDdPer / 2 : 1];   // 8-bit: pairs of 16-bit partial sums
#pragma unroll
    for (int q = 0; q < 4; ++q) {
#pragma unroll
        for (int k = 0; k < kDdPer; ++k) {
            if constexpr (kU8) total[q * kDdPer + k] = 0;
            else acc[q][k] = 0;
        }
#pragma unroll
        for (int k = 0; k < (kU8 ? kDdPer / 2 : 1); ++k) part[q][k] = 0u;
    }
    const bool warp_on = d_lo + 4 * warp < n_dm;
    int since = 0;   // groups in `part`
    auto flush = [&] {
        if constexpr (kU8) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int k = 0; k < kDdPer / 2; ++k) {
                    total[q * kDdPer + 2 * k] += (int)(part[q][k] & 0xffffu);
                    total[q * kDdPer + 2 * k + 1] += (int)(part[q][k] >> 16);
                    part[q][k] = 0u;
                }
            since = 0;
        }
    };

    // the warp's first piece of pattern sums and the step to its next one
    const int g_first = warp / chunks, ch_first = warp - g_first * chunks;
    const int g_step = (kDdThreads / 32) / chunks, ch_step = kDdThreads / 32 - g_step * chunks;
    stage(0, 0);
    int slot = 0;
    for (int g0 = 0; g0 < ng; g0 += batch, slot ^= 1) {
        const int n = min(batch, ng - g0);
        cp_async_wait<0>();
        __syncthreads();   // this batch has landed; every warp is done with the sums before
        if (g0 + batch < ng) stage(g0 + batch, slot ^ 1);
        const GrRec *r = slot_rec(slot);
        // pattern sums: one warp per group and kGrChunk samples
        for (int g = g_first, ch = ch_first; g < n;) {
            const int np = r[g].np, nk = r[g].nk;
            const unsigned char *xs = dd_smem + slot * slot_bytes + g * kGrMax * xpitch;
            // where each channel's samples start (kept in registers: the stores
            // of the sums would have them read again for every pattern)
            const int4 sh = *reinterpret_cast<const int4 *>(shift[slot] + g * kGrMax);
            short4 next = *reinterpret_cast<const short4 *>(r[g].pat[0]);
            if constexpr (!kU8) {
                // lane: samples chunk start + lane + 32 j
                const int at_y = kGrChunk<T> * ch + lane;   // (past ypitch nothing is read)
                const float *xw = reinterpret_cast<const float *>(xs) + at_y;
                float *y = reinterpret_cast<float *>(Y) + r[g].y0[0] * ypitch + at_y;
                float p0[kGrPer], p1[kGrPer], p2[kGrPer];
                {
                    const float *w = xw + sh.x;
#pragma unroll
                    for (int j = 0; j < kGrPer; ++j) p0[j] = w[32 * j];
                }
                // v = u + channel k at shift s (u itself past the group's channels)
                const int at[kGrMax] = {0, xpitch / 4 + sh.y, 2 * (xpitch / 4) + sh.z,
                                        3 * (xpitch / 4) + sh.w};
                auto x = [&](int k, int s, const float (&u)[kGrPer], float (&v)[kGrPer]) {
                    if (k < nk) {
                        const float *w = xw + at[k] + s;
#pragma unroll
                        for (int j = 0; j < kGrPer; ++j) v[j] = u[j] + w[32 * j];
                    } else {
#pragma unroll
                        for (int j = 0; j < kGrPer; ++j) v[j] = u[j];
                    }
                };
                for (int p = 0; p < np; ++p, y += ypitch) {
                    const short4 pt = next;
                    next = *reinterpret_cast<const short4 *>(r[g].pat[p + 1]);
                    if (pt.x <= 1) x(1, pt.y, p0, p1);
                    if (pt.x <= 2) x(2, pt.z, p1, p2);
                    float v[kGrPer];
                    x(3, pt.w, p2, v);
#pragma unroll
                    for (int j = 0; j < kGrPer; ++j)
                        if (at_y + 32 * j < ypitch) y[32 * j] = v[j];
                }
            } else {
                // lane: samples 372 ch + 12 lane .. + 11 as six pairs (an odd number
                // of words per lane: no bank conflicts); lane 31 only hands its
                // first sample to lane 30
                constexpr int kC = kGrChunk<T>;
                const bool store = lane < 31 && kC / 2 * ch + 6 * lane < ypitch;
                uint32_t *y = Y + r[g].y0[1] * 2 * ypitch + kC / 2 * ch + 6 * lane;
                uint32_t p0[6] = {0u, 0u, 0u, 0u, 0u, 0u}, p1[6], p2[6];
                // (windows start on multiples of 16 bytes, so a window's place can
                // go into the byte offset)
                const int at[kGrMax] = {sh.x + kC * ch, xpitch + sh.y + kC * ch,
                                        2 * xpitch + sh.z + kC * ch, 3 * xpitch + sh.w + kC * ch};
                add12_u8(xs, at[0], lane, p0);
                auto x = [&](int k, int s, const uint32_t (&u)[6], uint32_t (&v)[6]) {
#pragma unroll
                    for (int j = 0; j < 6; ++j) v[j] = u[j];
                    if (k < nk) add12_u8(xs, at[k] + s, lane, v);
                };
                for (int p = 0; p < np; ++p, y += 2 * ypitch) {
                    const short4 pt = next;
                    next = *reinterpret_cast<const short4 *>(r[g].pat[p + 1]);
                    if (pt.x <= 1) x(1, pt.y, p0, p1);
                    if (pt.x <= 2) x(2, pt.z, p1, p2);
                    uint32_t v[6];
                    x(3, pt.w, p2, v);
                    const uint32_t nx = __shfl_down_sync(0xffffffffu, v[0], 1);
                    if (store) {
#pragma unroll
                        for (int j = 0; j < 6; j += 2) {
                            const uint32_t after = j == 4 ? nx : v[j + 2];
                            *reinterpret_cast<uint2 *>(y + j) = make_uint2(v[j], v[j + 1]);
                            // and one sample further on
                            *reinterpret_cast<uint2 *>(y + ypitch + j) =
                                make_uint2(__byte_perm(v[j], v[j + 1], 0x5432u),
                                           __byte_perm(v[j + 1], after, 0x5432u));
                        }
                    }
                }
            }
            ch += ch_step;
            g += g_step;
            if (ch >= chunks) {
                ch -= chunks;
                ++g;
            }
        }
        __syncthreads();
        if (!warp_on) continue;
        if constexpr (!kU8) {
            for (int g = 0; g < n; ++g) {
                const int4 o = *reinterpret_cast<const int4 *>(r[g].off[0] + 4 * warp);
                const float *y = reinterpret_cast<const float *>(Y) + lane;
                add_pair(y, o.x, o.y, acc[0], acc[1]);
                add_pair(y, o.z, o.w, acc[2], acc[3]);
            }
        } else {
            // two groups per addition
            const uint32_t *y = Y + lane;
            int g = 0;
            for (; g + 1 < n; g += 2) {
                const int4 oa = *reinterpret_cast<const int4 *>(r[g].off[1] + 4 * warp);
                const int4 ob = *reinterpret_cast<const int4 *>(r[g + 1].off[1] + 4 * warp);
                const int wa[4] = {oa.x, oa.y, oa.z, oa.w}, wb[4] = {ob.x, ob.y, ob.z, ob.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t *a = y + wa[q], *b = y + wb[q];
#pragma unroll
                    for (int k = 0; k < kDdPer / 2; ++k) part[q][k] += a[32 * k] + b[32 * k];
                }
            }
            if (g < n) {
                const int4 oa = *reinterpret_cast<const int4 *>(r[g].off[1] + 4 * warp);
                const int wa[4] = {oa.x, oa.y, oa.z, oa.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t *a = y + wa[q];
#pragma unroll
                    for (int k = 0; k < kDdPer / 2; ++k) part[q][k] += a[32 * k];
                }
            }
            since += n;
            if (since > kGrFlush - kGrBatchMax) flush();
        }
    }
    flush();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int d = d_lo + 4 * warp + q;
        if (d >= n_dm) continue;
        float *row = out + (int64_t)d * n_out;
#pragma unroll
        for (int k = 0; k < kDdPer; ++k) {
            const int64_t t = kU8 ? t0 + 2 * (lane + 32 * (k >> 1)) + (k & 1) : t0 + lane + 32 * k;
            if (t < n_out) row[t] = (float)(kU8 ? total[q * kDdPer + k] : acc[q][k]);
        }
    }
}

// The groups of one DM tile (rows d0 .. d1 - 1 of the delay table): runs of up
// to 4 channels, halved until their trials' shifts form at most kGrPat
// patterns.
struct GrShape {
    int lo = 0, hi = 0;   // smallest and largest shift
    double cost = 0.0;    // shared-memory accesses per 32 samples
};
void group_tile(const int32_t *delays, int n_chan, int d0, int d1, int chunks, std::vector<GrRec> &out,
                GrShape &shape) {
    for (int c = 0; c < n_chan;) {
        int nk = std::min(kGrMax, n_chan - c);
        for (;; nk = nk / 2) {
            struct Pat {
                int s[kGrMax];
            };
            std::vector<Pat> pats;
            const int nd = d1 - d0;
            std::vector<Pat> of(nd);
            const int32_t *base = delays + (size_t)d0 * n_chan + c;
            for (int d = 0; d < nd; ++d) {
                const int32_t *row = delays + (size_t)(d0 + d) * n_chan + c;
                for (int k = 0; k < kGrMax; ++k)
                    of[d].s[k] = k < nk ? (row[k] - base[k]) - (row[0] - base[0]) : 0;
            }
            pats = of;
            auto less = [](const Pat &a, const Pat &b) {
                return std::lexicographical_compare(a.s, a.s + kGrMax, b.s, b.s + kGrMax);
            };
            auto same = [](const Pat &a, const Pat &b) { return std::equal(a.s, a.s + kGrMax, b.s); };
            std::sort(pats.begin(), pats.end(), less);
            pats.erase(std::unique(pats.begin(), pats.end(), same), pats.end());
            bool fits = (int)pats.size() <= kGrPat;
            for (const Pat &q : pats)
                for (int k = 1; k < nk; ++k) fits = fits && q.s[k] >= -64 && q.s[k] <= 64;
            if (!fits && nk > 1) continue;
            GrRec r{};
            r.c0 = c;
            r.nk = nk;
            r.np = (int16_t)pats.size();
            int nodes = 1;
            for (int k = 0; k < nk; ++k) r.first[k] = base[k];
            for (int p = 0; p < r.np; ++p) {
                int first = 1;
                if (p > 0)
                    while (first < kGrMax && pats[p].s[first] == pats[p - 1].s[first]) ++first;
                r.pat[p][0] = (int16_t)first;
                for (int k = 1; k < kGrMax; ++k) r.pat[p][k] = (int16_t)pats[p].s[k];
                nodes += std::max(0, nk - first);
                for (int k = 1; k < nk; ++k) {
                    shape.lo = std::min(shape.lo, pats[p].s[k]);
                    shape.hi = std::max(shape.hi, pats[p].s[k]);
                }
            }
            for (int d = 0; d < kDdD; ++d) {
                const int dd = std::min(d, nd - 1);
                const int p = (int)(std::lower_bound(pats.begin(), pats.end(), of[dd], less) -
                                    pats.begin());
                const int off = delays[(size_t)(d0 + dd) * n_chan + c] - base[0];
                r.off[0][d] = p;     // (turned into words once the layout is known)
                r.off[1][d] = off;
            }
            shape.cost += 4.0 * chunks * (nodes + r.np) + 16.0 * nd;
            out.push_back(r);
            break;
        }
        c += out.back().nk;
    }
}

}  // namespace

struct DedispPlan {
    int32_t n_chan = 0, n_dm = 0;
    int64_t n_t = 0, n_out = 0;
    double f_top = 0, df = 0, tsamp = 0, dm_lo = 0, dm_step = 0;
    int32_t *delays = nullptr;   // device [n_dm][n_chan]
    std::vector<int32_t> host_delays;
    int32_t max_delay = 0, span = 0, win = 0, chan_batch = 0, chan_batch_u8 = 0;
    int device = 0;
    // channel groups: used when they need fewer shared-memory accesses than
    // the plain kernel's one per addition (few channels with widely different
    // delays leave groups of one channel)
    bool grouped = false;
    GrRec *recs = nullptr;          // device [tiles][max_groups]
    int32_t *n_groups = nullptr;    // device [tiles]
    int32_t max_groups = 0, lead = 0, tail = 0;
    int32_t batch[2] = {0, 0}, batch_pat[2] = {0, 0};   // FP32, 8-bit: groups and most patterns of a batch
    int64_t table_bytes = 0;
};

// pieces of a pattern sum, bytes of a channel window, words of a pattern sum,
// and the shared memory of `batch` groups with `pats` patterns
template <class T>
static size_t group_layout(const DedispPlan &p, int batch, int pats, int *chunks, int *xpitch,
                           int *ypitch) {
    const int len = kDdT + p.span;   // samples that the DM trials read
    *chunks = (len + kGrChunk<T> - 1) / kGrChunk<T>;
    // (from up to 15 bytes past a 16-byte boundary.  Lanes past `len` read on into
    // what follows, at most a chunk, and store nothing: the records and sums
    // behind the last window are longer)
    *xpitch = ((int)sizeof(T) * (len + p.lead + p.tail) + 15 + 15) / 16 * 16;
    *ypitch = sizeof(T) == 4 ? len : (len + 11) / 12 * 6;   // (whole lanes)
    return 2 * (size_t)batch * (kGrMax * (size_t)*xpitch + sizeof(GrRec)) +
           4 * (size_t)pats * *ypitch * (sizeof(T) == 4 ? 1 : 2);
}

// groups per batch: as many as fill the warps of the pattern sums best, in the
// shared memory of the fullest batch
template <class T>
static void choose_batch(DedispPlan &p, const std::vector<std::vector<GrRec>> &tiles) {
    constexpr int kIdx = sizeof(T) == 4 ? 0 : 1;
    const int warps = kDdThreads / 32;
    double best = 0.0;
    for (int b = 1; b <= kGrBatchMax; ++b) {
        int pats = 0;
        for (const std::vector<GrRec> &recs : tiles)
            for (size_t g = 0; g < recs.size(); g += b) {
                int n = 0;
                for (size_t i = g; i < std::min(recs.size(), g + b); ++i) n += recs[i].np;
                pats = std::max(pats, n);
            }
        int chunks, xp, yp;
        if (group_layout<T>(p, b, pats, &chunks, &xp, &yp) > kGrSmem / kGrCtas<T>) break;
        const double fill = (double)b * chunks / (warps * ((b * chunks + warps - 1) / warps));
        if (fill >= best) {
            best = fill;
            p.batch[kIdx] = b;
            p.batch_pat[kIdx] = pats;
        }
    }
}

template <class T>
fdas_status launch_dedisperse(DedispPlan &p, const T *filterbank, float *out, cudaStream_t s) {
    int cur = 0;
    cudaGetDevice(&cur);
    if (cur != p.device) cudaSetDevice(p.device);
    dim3 grid((unsigned)((p.n_out + kDdT - 1) / kDdT), (unsigned)((p.n_dm + kDdD - 1) / kDdD));
    cudaError_t e;
    if (p.grouped) {
        constexpr int kIdx = sizeof(T) == 4 ? 0 : 1;
        const int batch = p.batch[kIdx];
        int chunks, xpitch, ypitch;
        const size_t smem = group_layout<T>(p, batch, p.batch_pat[kIdx], &chunks, &xpitch, &ypitch);
        e = cudaFuncSetAttribute(dedisperse_group_kernel<T>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess) {
            dedisperse_group_kernel<T><<<grid, kDdThreads, smem, s>>>(
                filterbank, p.recs, p.n_groups, p.max_groups, out, p.n_t, p.n_dm,
                p.n_out, chunks, p.lead, xpitch, ypitch, batch);
            e = cudaGetLastError();
        }
        if (cur != p.device) cudaSetDevice(cur);
        return e == cudaSuccess ? FDAS_OK : cuda_status(e, "dedisperse_group_kernel");
    }
    const int pitch = p.win + DdIn<T>::kPad;
    const int cb = sizeof(T) == 4 ? p.chan_batch : p.chan_batch_u8;
    const size_t smem = 2 * sizeof(T) * (size_t)pitch * cb;
    e = cudaFuncSetAttribute(dedisperse_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem);
    if (e == cudaSuccess) {
        dedisperse_kernel<T><<<grid, kDdThreads, smem, s>>>(filterbank, p.delays, out, p.n_chan,
                                                            p.n_t, p.n_dm, p.n_out, p.win, cb);
        e = cudaGetLastError();
    }
    if (cur != p.device) cudaSetDevice(cur);
    return e == cudaSuccess ? FDAS_OK : cuda_status(e, "dedisperse_kernel");
}

}  // namespace fdas

using fdas::DedispPlan;

namespace {

fdas_status dd_arg(const std::string &m) {
    fdas::set_error(m);
    return FDAS_ERR_ARG;
}

}  // namespace

extern "C" {

fdas_status fdas_dedisp_plan_create(fdas_dedisp_plan **out, int32_t n_chan, int64_t n_t,
                                    double f_top_mhz, double df_mhz, double tsamp, double dm_lo,
                                    double dm_step, int32_t n_dm, int64_t n_out) {
    try {
        if (!out) return dd_arg("out is NULL");
        *out = nullptr;
        if (n_chan < 1 || n_chan > 65536) return dd_arg("n_chan must be in [1, 65536]");
        if (n_dm < 1 || n_dm > 65536) return dd_arg("n_dm must be in [1, 65536]");
        if (n_t < 1 || n_t > (int64_t(1) << 34)) return dd_arg("n_t must be in [1, 2^34]");
        if (n_out < 1 || n_out > n_t) return dd_arg("n_out must be in [1, n_t]");
        if ((int64_t)n_chan * n_t > (int64_t(1) << 36)) return dd_arg("filterbank larger than 2^36 samples");
        if (!(tsamp > 0.0) || !std::isfinite(tsamp)) return dd_arg("tsamp must be > 0");
        if (!(f_top_mhz > 0.0) || !(df_mhz > 0.0) || !std::isfinite(f_top_mhz) || !std::isfinite(df_mhz))
            return dd_arg("need f_top_mhz > 0 and df_mhz > 0");
        const double f_bot = f_top_mhz - (double)(n_chan - 1) * df_mhz;
        if (!(f_bot > 0.0)) return dd_arg("the lowest channel frequency must be > 0");
        if (!(dm_lo >= 0.0) || !(dm_step >= 0.0) || !std::isfinite(dm_lo) || !std::isfinite(dm_step))
            return dd_arg("need dm_lo >= 0 and dm_step >= 0");
        const double dm_hi = dm_lo + (double)(n_dm - 1) * dm_step;
        const double x_max = fdas::kDm * dm_hi * (1.0 / (f_bot * f_bot) - 1.0 / (f_top_mhz * f_top_mhz)) / tsamp;
        if (!(x_max < 1.0e9)) return dd_arg("delays beyond 1e9 samples");

        DedispPlan *p = new (std::nothrow) DedispPlan();
        if (!p) return dd_arg("out of host memory");
        p->n_chan = n_chan;
        p->n_dm = n_dm;
        p->n_t = n_t;
        p->n_out = n_out;
        p->f_top = f_top_mhz;
        p->df = df_mhz;
        p->tsamp = tsamp;
        p->dm_lo = dm_lo;
        p->dm_step = dm_step;
        auto fail = [&](fdas_status s) {
            cudaFree(p->delays);
            cudaFree(p->recs);
            cudaFree(p->n_groups);
            delete p;
            return s;
        };
        cudaError_t e = cudaGetDevice(&p->device);
        if (e != cudaSuccess) return fail(fdas::cuda_status(e, "cudaGetDevice"));
        const size_t n = (size_t)n_chan * n_dm;
        e = cudaMalloc(&p->delays, sizeof(int32_t) * n);
        if (e != cudaSuccess) {
            cudaGetLastError();
            fdas::set_error("dedispersion: out of device memory for the delay table");
            return fail(FDAS_ERR_OOM);
        }
        fdas::dm_delay_kernel<<<(unsigned)((n + 255) / 256), 256>>>(p->delays, n_chan, n_dm, f_top_mhz,
                                                                    df_mhz, tsamp, dm_lo, dm_step);
        if ((e = cudaGetLastError()) != cudaSuccess) return fail(fdas::cuda_status(e, "dm_delay_kernel"));
        p->host_delays.resize(n);
        e = cudaMemcpy(p->host_delays.data(), p->delays, sizeof(int32_t) * n, cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) return fail(fdas::cuda_status(e, "cudaMemcpy"));
        // the widest window a 16-DM tile reads (per channel) and the largest delay
        int32_t span = 0, mx = 0;
        for (int d0 = 0; d0 < n_dm; d0 += fdas::kDdD) {
            const int d1 = std::min(n_dm - 1, d0 + fdas::kDdD - 1);
            for (int c = 0; c < n_chan; ++c) {
                const int32_t lo = p->host_delays[(size_t)d0 * n_chan + c];
                const int32_t hi = p->host_delays[(size_t)d1 * n_chan + c];
                span = std::max(span, hi - lo);
                mx = std::max(mx, hi);
            }
        }
        p->span = span;
        p->max_delay = mx;
        p->win = (fdas::kDdT + span + 31) / 32 * 32;
        const size_t per_chan = 2 * sizeof(float) * (size_t)p->win;   // double buffered
        if (per_chan > fdas::kDdSmemCap) {
            fdas::set_error("dedispersion: the delays of 32 consecutive DM trials spread over more "
                            "than " + std::to_string(fdas::kDdSmemCap / 8 - fdas::kDdT) +
                            " samples; use a smaller dm_step");
            return fail(FDAS_ERR_UNSUPPORTED);
        }
        p->chan_batch = (int)std::max<size_t>(1, std::min<size_t>(8, (96 * 1024) / per_chan));
        // 8-bit windows: a quarter of the bytes, so more channels per batch
        const size_t per_chan_u8 = 2 * (size_t)(p->win + 16);
        p->chan_batch_u8 = (int)std::max<size_t>(1, std::min<size_t>(16, (96 * 1024) / per_chan_u8));
        // channel groups per DM tile
        {
            const int tiles = (n_dm + fdas::kDdD - 1) / fdas::kDdD;
            const int chunks = (fdas::kDdT + span + 127) / 128;
            std::vector<std::vector<fdas::GrRec>> per(tiles);
            std::vector<int32_t> counts(tiles);
            fdas::GrShape shape;
            double plain = 0.0;
            size_t most = 0;
            for (int t = 0; t < tiles; ++t) {
                const int d0 = t * fdas::kDdD, d1 = std::min(n_dm, d0 + fdas::kDdD);
                fdas::group_tile(p->host_delays.data(), n_chan, d0, d1, chunks, per[t], shape);
                plain += 16.0 * (d1 - d0) * n_chan;
                counts[t] = (int32_t)per[t].size();
                most = std::max(most, per[t].size());
            }
            p->lead = -shape.lo;
            p->tail = shape.hi;
            fdas::choose_batch<float>(*p, per);
            fdas::choose_batch<uint8_t>(*p, per);
            const int bf = p->batch[0], bu = p->batch[1];
            int nc, xp, ypf, ypu;
            fdas::group_layout<float>(*p, bf, p->batch_pat[0], &nc, &xp, &ypf);
            fdas::group_layout<uint8_t>(*p, bu, p->batch_pat[1], &nc, &xp, &ypu);
            // (accesses of the pattern sums and of the trials against the plain
            // kernel's one per addition; at equal counts the extra barriers and
            // table reads make groups slower)
            if (shape.cost < 0.75 * plain && bf >= 1 && bu >= 1 && span < (1 << 24)) {
                std::vector<fdas::GrRec> flat(most * (size_t)tiles);
                for (int t = 0; t < tiles; ++t) {
                    int y0[2] = {0, 0};   // patterns of the batch so far
                    for (size_t g = 0; g < per[t].size(); ++g) {
                        fdas::GrRec &r = flat[(size_t)t * most + g] = per[t][g];
                        for (int i = 0; i < 2; ++i) {
                            if (g % (size_t)p->batch[i] == 0) y0[i] = 0;
                            r.y0[i] = (int16_t)y0[i];
                        }
                        for (int d = 0; d < fdas::kDdD; ++d) {
                            const int pat = r.off[0][d], off = r.off[1][d];
                            r.off[0][d] = (y0[0] + pat) * ypf + off;
                            r.off[1][d] = (2 * (y0[1] + pat) + (off & 1)) * ypu + off / 2;
                        }
                        for (int &y : y0) y += r.np;
                    }
                }
                p->table_bytes = (int64_t)(sizeof(fdas::GrRec) * flat.size() + sizeof(int32_t) * tiles);
                e = cudaMalloc(&p->recs, sizeof(fdas::GrRec) * flat.size());
                if (e == cudaSuccess) e = cudaMalloc(&p->n_groups, sizeof(int32_t) * tiles);
                if (e != cudaSuccess) {
                    cudaGetLastError();
                    fdas::set_error("dedispersion: out of device memory for the channel groups");
                    return fail(FDAS_ERR_OOM);
                }
                e = cudaMemcpy(p->recs, flat.data(), sizeof(fdas::GrRec) * flat.size(),
                               cudaMemcpyHostToDevice);
                if (e == cudaSuccess)
                    e = cudaMemcpy(p->n_groups, counts.data(), sizeof(int32_t) * tiles,
                                   cudaMemcpyHostToDevice);
                if (e != cudaSuccess) return fail(fdas::cuda_status(e, "cudaMemcpy"));
                p->max_groups = (int32_t)most;
                p->grouped = true;
            }
        }
        *out = reinterpret_cast<fdas_dedisp_plan *>(p);
        return FDAS_OK;
    } catch (...) {
        fdas::set_error("unexpected C++ exception in fdas_dedisp_plan_create");
        return FDAS_ERR_CUDA;
    }
}

void fdas_dedisp_plan_destroy(fdas_dedisp_plan *plan) {
    if (!plan) return;
    DedispPlan *p = reinterpret_cast<DedispPlan *>(plan);
    cudaFree(p->delays);
    cudaFree(p->recs);
    cudaFree(p->n_groups);
    delete p;
}

fdas_status fdas_dedisp_get_info(const fdas_dedisp_plan *plan, fdas_dedisp_info *info) {
    if (!plan || !info) return dd_arg("NULL argument");
    const DedispPlan &p = *reinterpret_cast<const DedispPlan *>(plan);
    info->n_chan = p.n_chan;
    info->n_dm = p.n_dm;
    info->n_t = p.n_t;
    info->n_out = p.n_out;
    info->f_top_mhz = p.f_top;
    info->df_mhz = p.df;
    info->tsamp = p.tsamp;
    info->dm_lo = p.dm_lo;
    info->dm_step = p.dm_step;
    info->max_delay = p.max_delay;
    info->tile_span = p.span;
    info->workspace_bytes = (int64_t)sizeof(int32_t) * p.n_chan * p.n_dm + p.table_bytes;
    return FDAS_OK;
}

fdas_status fdas_dedisp_delays(const fdas_dedisp_plan *plan, int32_t *delays_out) {
    if (!plan || !delays_out) return dd_arg("NULL argument");
    const DedispPlan &p = *reinterpret_cast<const DedispPlan *>(plan);
    std::copy(p.host_delays.begin(), p.host_delays.end(), delays_out);
    return FDAS_OK;
}

fdas_status fdas_dedisperse(fdas_dedisp_plan *plan, const float *filterbank, float *out,
                            void *stream) {
    if (!plan || !filterbank || !out) return dd_arg("NULL argument");
    return fdas::launch_dedisperse(*reinterpret_cast<DedispPlan *>(plan), filterbank, out,
                                   (cudaStream_t)stream);
}

fdas_status fdas_dedisperse_u8(fdas_dedisp_plan *plan, const uint8_t *filterbank, float *out,
                               void *stream) {
    if (!plan || !filterbank || !out) return dd_arg("NULL argument");
    DedispPlan &p = *reinterpret_cast<DedispPlan *>(plan);
    if (p.n_t % 16 != 0 || ((uintptr_t)filterbank & 15u) != 0)
        return dd_arg("8-bit filterbanks need n_t a multiple of 16 and a 16-byte aligned pointer");
    return fdas::launch_dedisperse(p, filterbank, out, (cudaStream_t)stream);
}

}  // extern "C"
