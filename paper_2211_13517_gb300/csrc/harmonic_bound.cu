// Harmonic sum + threshold by bounds: the same crossings as
// harmonic_dedup_kernel (harmonic.cu), from the sums of far fewer cells.
//
// A 6-sigma crossing is rare (about one cell in 10^9 of noise), so almost
// every sum only has to be shown not to cross.  The plane is reduced to its
// maxima over boxes of 2 bins x one row block (at most kPoolMaxRows = 4 template
// rows), A[block][r/2], and a box of the top plane is compared through the maxima of
// the boxes its harmonics read:
//
//   for every cell of the box and every stage,  S_h <= sum_j max(boxes of j).
//
// A box whose bound stays below every stage threshold holds no crossing.  The
// cells of the others (about 7 in 10^4 boxes of noise at 6 sigma, 16 harmonics,
// z_step 1; more at coarser steps, see bounds_pay in plan.cu) are summed
// exactly, in the same stage order and FP32 rounding as harmonic_dedup_kernel, and
// compared exactly, so the records are identical.
// Neighbouring templates are strongly correlated, neighbouring bins are not:
// pooling 2 bins x 4 rows passes 7e-4 of noise boxes, 4 bins x 2 rows 1.3e-2
// (measured on a noise plane, 193 templates, 16 harmonics, 6 sigma).
//
// The bound is summed in FP16 pairs (two boxes per instruction).  A is the
// plane's cells rounded to FP16 (exact for 16-bit planes in range; beyond its
// range +inf, which only sends a box to the exact sums), and each of at most
// 17 roundings loses at most 2^-11 of the sum, so the FP16 sum is at least
// 0.9917 of the true one: thresholds are lowered by 1 % before the
// comparison.  A threshold outside [0.5, 30000] (a plane far from unit mean)
// is replaced by 0: every box is then summed exactly.  Cells are powers (>= 0).
// A cell that is NaN never crosses, and neither does a sum that reads it, but the
// sums beside it may, so no maximum of a caller's plane is NaN: where pool_kernel
// compares 16-bit cells as integers a NaN would be the largest, and it becomes
// +inf there, which sends its box to the exact sums (FP32 maxima drop it).  A plane
// of the search with a NaN cell has a NaN mean and thresholds that nothing
// crosses, so the tensor-core epilogue's maxima are left as they are.
//
// Bound of the kernel: instruction issue and the latency of the span copies
// (the gathers move 1/8 of the cells' bytes).
#include "check.cuh"
#include "fdas_internal.cuh"
#include "harmonic_index.cuh"
#include "tma.cuh"

#include <algorithm>
#include <cstring>

namespace fdas {
namespace {

// ---------------------------------------------------------------------------
// maxima of 2 bins x one row block, from a plane (of the overlap-save
// correlator, or a caller's; the tensor-core correlation writes its own).  A
// thread reduces 8
// consecutive bins of the block's rows (at most kPoolMaxRows; 16-byte loads,
// all of them in flight).  Reads the plane once: HBM bound.
// ---------------------------------------------------------------------------
template <class P>
__global__ void __launch_bounds__(256) pool_kernel(const typename P::real *__restrict__ plane,
                                                   uint16_t *__restrict__ A,
                                                   const int32_t *__restrict__ blk, int64_t n_r) {
    const int64_t c = ((int64_t)blockIdx.x * 256 + threadIdx.x) * 8;
    if (c >= n_r) return;
    const int kb = blockIdx.y;
    const int r0 = blk[kb], nr = blk[kb + 1] - r0;
    const typename P::real *src = plane + (int64_t)r0 * n_r + c;
    float e[4];
    if constexpr (sizeof(typename P::real) == 2) {
        uint4 w[kPoolMaxRows];
#pragma unroll
        for (int r = 0; r < kPoolMaxRows; ++r)
            w[r] = r < nr ? __ldg(reinterpret_cast<const uint4 *>(src + (int64_t)r * n_r))
                          : make_uint4(0u, 0u, 0u, 0u);
        // 16-bit patterns of values >= 0 order as signed integers
        uint4 m = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int r = 0; r < kPoolMaxRows; ++r) {
            m.x = __vmaxs2(m.x, w[r].x);
            m.y = __vmaxs2(m.y, w[r].y);
            m.z = __vmaxs2(m.z, w[r].z);
            m.w = __vmaxs2(m.w, w[r].w);
        }
        const uint32_t mm[4] = {m.x, m.y, m.z, m.w};
        constexpr uint32_t inf = P::id == FDAS_BF16 ? 0x7f80u : 0x7c00u;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const unsigned short h =
                (unsigned short)min(max(mm[k] & 0xffffu, mm[k] >> 16), inf);   // NaN: +inf
            typename P::real v;
            memcpy(&v, &h, 2);
            e[k] = P::ldr(v) * (1.0f / P::plane_scale);
        }
    } else {
        float4 w[kPoolMaxRows][2];
#pragma unroll
        for (int r = 0; r < kPoolMaxRows; ++r)
#pragma unroll
            for (int q = 0; q < 2; ++q)
                w[r][q] = r < nr ? __ldg(reinterpret_cast<const float4 *>(src + (int64_t)r * n_r) + q)
                                 : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int k = 0; k < 4; ++k) e[k] = 0.f;
#pragma unroll
        for (int r = 0; r < kPoolMaxRows; ++r)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                e[2 * q] = fmaxf(e[2 * q], fmaxf(w[r][q].x, w[r][q].y));
                e[2 * q + 1] = fmaxf(e[2 * q + 1], fmaxf(w[r][q].z, w[r][q].w));
            }
    }
    const __half2 lo = __floats2half2_rn(e[0], e[1]), hi = __floats2half2_rn(e[2], e[3]);
    uint2 o;
    memcpy(&o.x, &lo, 4);
    memcpy(&o.y, &hi, 4);
    *reinterpret_cast<uint2 *>(A + (int64_t)kb * (n_r / 2) + c / 2) = o;
}

// ---------------------------------------------------------------------------
// geometry of the bound sums.  A CTA of W = 8 warps walks down a column of 1024
// boxes, 8 block rows at a time, one per warp; lane t owns G = 32 consecutive
// boxes (64 bins) of the warp's row.  Harmonic J of its
// box i reads the bins from floor((2 i J + H/2)/H) to
// floor(((2 i + 1) J + H/2)/H) past 64 J t/H, that is one or two consecutive
// boxes of A at compile-time places past 32 J t/H.  With 32 boxes per lane
// every window starts on an even box (H <= 16), so pairs of boxes are picked
// out of whole words with constant selectors.
// ---------------------------------------------------------------------------
constexpr int kBoundW = 8;   // warps of a CTA = block rows of a step

template <int H>
struct Bound {
    static constexpr int G = 32;
    static constexpr int BOXES = 32 * G;       // per warp
    static constexpr int NS = ilog2h(H) + 1;   // stages; also barriers (0 unused)
    static constexpr int e0(int J, int i) { return ((2 * i * J + H / 2) / H) >> 1; }
    static constexpr int e1(int J, int i) { return (((2 * i + 1) * J + H / 2) / H) >> 1; }
    static constexpr int step(int J) { return G * J / H; }     // boxes per lane
    static constexpr int ne(int J) { return e1(J, G - 1) + 1; }
    // widest load (boxes) that every lane's start is aligned to
    static constexpr int width(int J) {
        int w = 1;
        while (w < 8 && step(J) % (2 * w) == 0) w *= 2;
        return w;
    }
    static constexpr int words(int J) { return (ne(J) + width(J) - 1) / width(J) * (width(J) / 2); }
    // boxes the warp reads of harmonic J, in whole 16-byte vectors
    static constexpr int len(int J) { return (step(J) * 31 + 2 * words(J) + 7) / 8 * 8; }
    // source blocks held at a time: those of 8 consecutive block rows (their
    // rows advance J / H as fast; pool_sources checks the number)
    static constexpr int slots(int J) { return kBoundW * J / H + 2; }
    static constexpr int off(int J) { return J <= 1 ? 0 : off(J - 1) + slots(J - 1) * len(J - 1); }
    static constexpr int SMEM_ELEMS = off(H) + 8;   // the top row (J = H) is not staged
};

__device__ __forceinline__ uint32_t hmax2_u32(uint32_t a, uint32_t b) {
    __half2 x, y;
    memcpy(&x, &a, 4);
    memcpy(&y, &b, 4);
    const __half2 m = __hmax2(x, y);
    uint32_t r;
    memcpy(&r, &m, 4);
    return r;
}
__device__ __forceinline__ __half2 as_half2(uint32_t a) {
    __half2 x;
    memcpy(&x, &a, 4);
    return x;
}

template <int H>
struct BoundSteps {
    using D = Bound<H>;

    // lane t's window of harmonic J out of the warp's boxes in shared memory
    template <int J>
    __device__ __forceinline__ static void load_window(const uint16_t *sp, int t,
                                                       uint32_t (&w)[D::words(J)]) {
        constexpr int W = D::width(J);
        static_assert(W >= 2, "windows start on even boxes");
        if constexpr (W == 2) {
            const uint32_t *pw = reinterpret_cast<const uint32_t *>(sp + D::step(J) * t);
#pragma unroll
            for (int k = 0; k < D::words(J); ++k) w[k] = pw[k];
        } else if constexpr (W == 4) {
            const uint2 *pw = reinterpret_cast<const uint2 *>(sp + D::step(J) * t);
#pragma unroll
            for (int k = 0; k < D::words(J) / 2; ++k) {
                const uint2 u = pw[k];
                w[2 * k] = u.x;
                w[2 * k + 1] = u.y;
            }
        } else {
            const uint4 *pw = reinterpret_cast<const uint4 *>(sp + D::step(J) * t);
#pragma unroll
            for (int k = 0; k < D::words(J) / 4; ++k) {
                const uint4 u = pw[k];
                w[4 * k] = u.x;
                w[4 * k + 1] = u.y;
                w[4 * k + 2] = u.z;
                w[4 * k + 3] = u.w;
            }
        }
    }

    // boxes (X, Y), Y - X in {0, 1}, of the window as one pair
    template <int J, int X, int Y>
    __device__ __forceinline__ static uint32_t pick(const uint32_t (&w)[D::words(J)]) {
        static_assert(Y == X || Y == X + 1, "consecutive boxes");
        constexpr int k = X >> 1, k1 = k + 1 < D::words(J) ? k + 1 : k;
        if constexpr ((X & 1) == 0 && Y == X + 1) return w[k];
        constexpr uint32_t sel = (X & 1) == 0 ? 0x1010u : (Y == X ? 0x3232u : 0x5432u);
        return __byte_perm(w[k], w[k1], sel);
    }

    template <int J, int PAIR>
    __device__ __forceinline__ static void add_pairs(const uint32_t (&w)[D::words(J)],
                                                     __half2 (&S)[D::G / 2]) {
        if constexpr (PAIR < D::G / 2) {
            constexpr int a0 = D::e0(J, 2 * PAIR), a1 = D::e0(J, 2 * PAIR + 1);
            constexpr int b0 = D::e1(J, 2 * PAIR), b1 = D::e1(J, 2 * PAIR + 1);
            uint32_t m = pick<J, a0, a1>(w);
            if constexpr (b0 != a0 || b1 != a1) m = hmax2_u32(m, pick<J, b0, b1>(w));
            S[PAIR] = __hadd2(S[PAIR], as_half2(m));
            add_pairs<J, PAIR + 1>(w, S);
        }
    }

    // harmonics j_at(H, IDX), ... in stage order; stage(s, S) after each
    // stage.  msk: 4 bits per harmonic (from .x on) with the slot of its (first)
    // source block, and in .z a bit per harmonic whose sources span two blocks.
    template <int IDX, class F>
    __device__ __forceinline__ static bool sums(const uint16_t *sm, uint64_t *bars, unsigned parity,
                                                int t, uint4 msk, __half2 (&S)[D::G / 2], F &&stage) {
        if constexpr (IDX < H) {
            constexpr int J = j_at(H, IDX);
            if constexpr ((IDX & (IDX - 1)) == 0)
                if (!mbar_wait(&bars[ilog2h(IDX) + 1], parity)) return false;
            const uint16_t *base = sm + D::off(J);
            const int slot = (int)(((J <= 8 ? msk.x : msk.y) >> (4 * ((J - 1) & 7))) & 15u);
            uint32_t w[D::words(J)];
            load_window<J>(base + slot * D::len(J), t, w);
            if ((msk.z >> (J - 1)) & 1u) {
                uint32_t w2[D::words(J)];
                load_window<J>(base + (slot + 1 == D::slots(J) ? 0 : slot + 1) * D::len(J), t, w2);
#pragma unroll
                for (int k = 0; k < D::words(J); ++k) w[k] = hmax2_u32(w[k], w2[k]);
            }
            add_pairs<J, 0>(w, S);
            if constexpr (((IDX + 1) & IDX) == 0) stage(ilog2h(IDX + 1), S);
            return sums<IDX + 1>(sm, bars, parity, t, msk, S, stage);
        } else {
            return true;
        }
    }

    // the span lane IDX of warp 0 copies (J = 0: none)
    struct Lane {
        int J = 0, g = 0, off = 0, len = 0, slots = 1;
    };
    template <int IDX>
    __device__ __forceinline__ static void lane_span(int lane, Lane &L) {
        if constexpr (IDX < H) {
            constexpr int J = j_at(H, IDX), OFF = D::off(J), LEN = D::len(J), SLOTS = D::slots(J);
            if (lane == IDX) {
                L.J = J;
                L.g = ilog2h(IDX) + 1;
                L.off = OFF;
                L.len = LEN;
                L.slots = SLOTS;
            }
            lane_span<IDX + 1>(lane, L);
        }
    }
};

// Lane IDX of warp 0 brings harmonic j_at(H, IDX)'s boxes (consecutive: 64 J of
// a source block at H = 16) to shared memory by a bulk copy when the walk first
// reaches their source block, into slot (block mod slots) of the harmonic, so a
// source block is copied once per walk.  The copies of a stage complete on the
// stage's own barrier, one phase per step.  The 8 block rows of a step share the
// staged blocks: 107 KB for 8 warps at H = 16, two CTAs per SM.
//
// A box that reaches a threshold is listed with its last-stage bound (+inf
// when an earlier stage reached its threshold, which is very rare); `listed`
// counts them, also beyond the list's capacity.
//
// Measured at 2^22 bins x 193 rows, H = 16 (56 block rows): 301 us, 1.6
// instructions per cycle.  One warp per CTA, with two slots per harmonic of its
// own (31 KB, 7 warps per SM): 312 us, and half again as slow at H = 8; 16 boxes
// per lane: a third more instructions, the same time.  A copying warp and 8
// summing ones that take the next row as soon as the row 8 before it is done
// (no CTA barrier): 309 us; 2048 boxes per CTA, half the copies: 346 us; the
// same with 16-byte asynchronous copies instead of bulk ones: 1.2 ms.  Windows
// exchanged through a small buffer per harmonic from coalesced global loads
// instead of staged (20 warps per SM): bound by the L1, 419 us.
template <int H>
__global__ void __launch_bounds__(32 * kBoundW, 2)
    harmonic_bound_kernel(const uint16_t *__restrict__ A, int64_t n_r, int nb, int walk,
                          const uint32_t *__restrict__ src, const uint4 *__restrict__ masks,
                          const TrialStats *__restrict__ st, unsigned long long *__restrict__ list,
                          unsigned int list_cap, unsigned int *__restrict__ listed,
                          unsigned int *__restrict__ flags) {
    using D = Bound<H>;
    using Steps = BoundSteps<H>;
    constexpr int NS = D::NS;
    extern __shared__ __align__(16) unsigned char hb_smem[];
    uint16_t *sm = reinterpret_cast<uint16_t *>(hb_smem);
    __shared__ __align__(8) uint64_t bars[NS + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t pitch = n_r / 2;
    const int64_t box0 = (int64_t)blockIdx.x * D::BOXES;   // rows hold whole columns of boxes
    const int kb_begin = blockIdx.y * walk, kb_end = min(kb_begin + walk, nb);
    if (threadIdx.x == 0) {
        for (int g = 0; g <= NS; ++g) mbar_init(&bars[g], 1);
        mbar_fence_init();
    }
    __half2 T16[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        const float th = st->thr[s];
        T16[s] = __half2half2(th >= 0.5f && th <= 30000.f ? __float2half_rd(0.99f * th) : __half(0.f));
    }
    typename Steps::Lane sp;
    if (warp == 0) Steps::template lane_span<1>(lane, sp);
    const int64_t c0 = sp.J * box0 / H;
    const unsigned bytes = 2u * (unsigned)sp.len;
    int have = -1;   // last source block this lane copied
    bool failed = false;
    int step = 0;
    // the lane's boxes of the top row and the row's slots, one step ahead
    uint4 top[D::G / 8];
    uint4 msk = make_uint4(0u, 0u, 0u, 0u);
    auto load_top = [&](int kb) {
        const int64_t at = kb * pitch + box0 + D::G * lane;
        if (kb < kb_end && FDAS_IN_BOUNDS(at, D::G, nb * pitch, kSiteHsTopLoad)) {
#pragma unroll
            for (int k = 0; k < D::G / 8; ++k) top[k] = __ldg(reinterpret_cast<const uint4 *>(A + at) + k);
            msk = __ldg(masks + kb);
        }
    };
    load_top(kb_begin + warp);

    for (int kb0 = kb_begin; kb0 < kb_end; kb0 += kBoundW, ++step) {
        // every warp is done with the last step's boxes (and the barriers are
        // initialised); stop together after a wait that gave up
        if (__syncthreads_or(failed)) {
            failed = true;
            break;
        }
        if (warp == 0) {
            if (sp.J != 0) {
                const int sb0 = (int)(__ldg(src + kb0 * H + sp.J - 1) & 0xffffu);
                const int sb1 = (int)(__ldg(src + min(kb0 + kBoundW, kb_end) * H - H + sp.J - 1) >> 16);
                for (int x = max(sb0, have + 1); x <= sb1; ++x) {
                    if (!FDAS_IN_BOUNDS(x, 1, nb, kSiteHsSpanRow) ||
                        !FDAS_IN_BOUNDS(c0, sp.len, pitch, kSiteHsSpanRange))
                        continue;
                    fence_proxy_async_smem();
                    mbar_expect_tx(&bars[sp.g], bytes);
                    bulk_copy_g2s(sm + sp.off + (x % sp.slots) * sp.len, A + (int64_t)x * pitch + c0,
                                  bytes, &bars[sp.g]);
                }
                have = sb1;
            }
            __syncwarp();
            if (lane >= 1 && lane < NS) mbar_arrive(&bars[lane]);
        }
        const int kb = kb0 + warp;
        if (kb >= kb_end) continue;
        __half2 S[D::G / 2];
#pragma unroll
        for (int k = 0; k < D::G / 8; ++k) {
            S[4 * k] = as_half2(top[k].x);
            S[4 * k + 1] = as_half2(top[k].y);
            S[4 * k + 2] = as_half2(top[k].z);
            S[4 * k + 3] = as_half2(top[k].w);
        }
        const uint4 m_now = msk;
        load_top(kb + kBoundW);
        uint32_t mask = 0u;    // boxes of this lane that need their exact sums
        uint32_t bound = 0u;   // the largest last-stage bound among them
        auto stage = [&](int s, __half2 (&Sv)[D::G / 2]) {
            __half2 m = Sv[0];
#pragma unroll
            for (int p = 1; p < D::G / 2; ++p) m = __hmax2(m, Sv[p]);
            if (__hge2_mask(m, T16[s]) != 0u) {
#pragma unroll
                for (int p = 0; p < D::G / 2; ++p) {
                    const uint32_t ge = __hge2_mask(Sv[p], T16[s]);
                    mask |= ((ge & 1u) | ((ge >> 16) & 2u)) << (2 * p);
                }
                bound = s < NS - 1 ? 0x7c00u
                                   : max(bound, (uint32_t)__half_as_ushort(
                                                    __hmax(__low2half(m), __high2half(m))));
            }
        };
        stage(0, S);
        if (!Steps::template sums<1>(sm, bars, (unsigned)(step & 1), lane, m_now, S, stage))
            failed = true;
        if (__any_sync(0xffffffffu, mask != 0u)) {
            int n = __popc(mask), before = n;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, before, off);
                if (lane >= off) before += v;
            }
            unsigned int first = 0u;
            if (lane == 31) first = atomicAdd(listed, (unsigned int)before);
            first = __shfl_sync(0xffffffffu, first, 31) + (unsigned int)(before - n);
            while (mask != 0u) {
                const int i = __ffs((int)mask) - 1;
                mask &= mask - 1u;
                if (first < list_cap)
                    list[first] = ((unsigned long long)bound << 48) |
                                  ((unsigned long long)kb << 32) |
                                  (unsigned long long)(box0 + D::G * lane + i);
                ++first;
            }
        }
    }
    if (__syncthreads_or(failed)) {
        if (threadIdx.x == 0) atomicOr(flags, 2u);
        // copies still in flight land before shared memory is released (bounded):
        // those of the last step issued
        if (threadIdx.x == 0 && step > 0)
            for (int g = 1; g < NS; ++g) (void)mbar_wait(&bars[g], (unsigned)((step - 1) & 1));
    }
}

// The exact sums of the listed boxes: a warp sums four at a time, one lane
// per cell (2 bins x up to 4 rows).  Nothing is done when the list overflowed
// (harmonic_dedup_kernel then sums the whole plane).
//
// The gathers are what costs (a 32-byte sector per row, harmonic and box,
// mostly from DRAM), and most bounds exceed the threshold by little.  So a box
// that only the last stage marked is gathered four harmonics at a time: with
// g_j the largest of the values its lanes read for harmonic j, every cell's
// sum is at most bound - sum_j (g_j - v_j) over the harmonics read so far, and
// a cell that falls below the threshold is dropped (FP16 slack: the bound is
// raised by 1 %).  A cell that stays is summed in the stage order of
// harmonic_dedup_kernel, with its roundings.
constexpr int kExactThreads = 128;
constexpr int kExactCtas = 8;      // per SM

template <class P, int H>
__global__ void __launch_bounds__(kExactThreads, kExactCtas)
    harmonic_exact_kernel(const unsigned long long *__restrict__ list, unsigned int list_cap,
                          const unsigned int *__restrict__ listed,
                          const typename P::real *__restrict__ plane, int64_t n_r, int n_z, int iz0,
                          const int32_t *__restrict__ blk, const TrialStats *__restrict__ st,
                          uint32_t rank, CandRec *__restrict__ cand,
                          unsigned long long *__restrict__ count, int64_t cap) {
    constexpr int NS = Bound<H>::NS;
    constexpr int kStep = H < 4 ? H : 4;
    const int lane = threadIdx.x & 31;
    const unsigned int n = *listed;
    if (n > list_cap) return;
    const float inv = 1.0f / P::plane_scale;
    float thr[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) thr[s] = st->thr[s];
    const unsigned int warps = gridDim.x * (kExactThreads / 32);
    for (unsigned int i0 = 4 * (blockIdx.x * (kExactThreads / 32) + (threadIdx.x >> 5)); i0 < n;
         i0 += 4 * warps) {
        const unsigned int i = i0 + (lane >> 3);
        const unsigned long long e = list[min(i, n - 1u)];
        const int kb = (int)((e >> 32) & 0xffffu);
        const int iz = blk[kb] + ((lane >> 1) & 3), o = iz - iz0;
        const uint32_t ir = 2u * (uint32_t)e + (uint32_t)(lane & 1);
        bool alive = i < n && iz < blk[kb + 1];   // the lane has a cell
        // the last stage's bound of the cell, as read so far
        float bound = 1.01f * __half2float(__ushort_as_half((unsigned short)(e >> 48)));
        float v[H];
#pragma unroll
        for (int k = 0; k < H; ++k) v[k] = 0.f;
        unsigned any = 0xffffffffu;
#pragma unroll
        for (int k0 = 0; k0 < H; k0 += kStep) {
            if (any != 0u) {
#pragma unroll
                for (int k = k0; k < k0 + kStep; ++k) {
                    const int J = j_at(H, k);
                    const int row = iz0 + src_off(H, o, J);
                    const uint32_t c = (ir * (uint32_t)J + H / 2) / H;
                    if (alive && FDAS_IN_BOUNDS(row, 1, n_z, kSiteHsSpanRow) &&
                        FDAS_IN_BOUNDS(c, 1, n_r, kSiteHsSpanRange))
                        v[k] = P::ldr(__ldg(plane + (int64_t)row * n_r + c));
                }
#pragma unroll
                for (int k = k0; k < k0 + kStep; ++k) {
                    float g = v[k];
                    g = fmaxf(g, __shfl_xor_sync(0xffffffffu, g, 1));
                    g = fmaxf(g, __shfl_xor_sync(0xffffffffu, g, 2));
                    g = fmaxf(g, __shfl_xor_sync(0xffffffffu, g, 4));
                    bound -= (g - v[k]) * inv;
                }
                if (bound < thr[NS - 1]) alive = false;
                any = __ballot_sync(0xffffffffu, alive);
            }
        }
        if (alive) {
            float S = 0.f;
            int s = 0;   // stage
#pragma unroll
            for (int k = 0; k < H; ++k) {
                S += v[k];
                if (((k + 1) & k) == 0) {
                    const float val = S * inv;
                    if (val > thr[s]) {
                        const unsigned long long x = atomicAdd(count, 1ull);
                        if ((int64_t)x < cap) {
                            CandRec rec;
                            rec.key = cand_key(rank, s, iz, ir);
                            rec.power = val;
                            rec.pad = 0.f;
                            cand[x] = rec;
                        }
                    }
                    ++s;
                }
            }
        }
    }
}

template <class P, int H>
fdas_status launch_bound(Plan &p, const void *plane, int buf, const TrialStats *st, uint32_t rank,
                         cudaStream_t s) {
    using D = Bound<H>;
    const size_t smem = sizeof(uint16_t) * (size_t)D::SMEM_ELEMS;
    auto k = harmonic_bound_kernel<H>;
    FDAS_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const unsigned cols = (unsigned)(p.n_r / 2 / D::BOXES);
    // block rows per walk, in whole steps: long walks copy each source block
    // once, but the grid should fill the GPU (2 CTAs per SM) a few times
    const int steps = (p.pool_nb + kBoundW - 1) / kBoundW;
    const int64_t want = 8 * (int64_t)p.n_sms;
    const int walks = (int)std::max<int64_t>(1, std::min<int64_t>(steps, (want + cols - 1) / cols));
    const int walk = (steps + walks - 1) / walks * kBoundW;
    dim3 grid(cols, (unsigned)((p.pool_nb + walk - 1) / walk));
    k<<<grid, 32 * kBoundW, smem, s>>>(p.pool[buf], p.n_r, p.pool_nb, walk, p.pool_src, p.pool_masks, st,
                             p.pool_list, p.pool_list_cap, p.pool_listed, p.flags);
    FDAS_CUDA_TRY(cudaGetLastError());
    const unsigned exact_ctas = std::min(kExactCtas * (unsigned)p.n_sms, p.pool_list_cap / 16);
    harmonic_exact_kernel<P, H><<<exact_ctas, kExactThreads, 0, s>>>(
        p.pool_list, p.pool_list_cap, p.pool_listed, (const typename P::real *)plane, p.n_r, p.n_z,
        p.iz0, p.pool_blk, st, rank, p.cand, p.cand_count, p.store_cap);
    FDAS_CUDA_TRY(cudaGetLastError());
    return FDAS_OK;
}

template <class P>
fdas_status launch_bound_P(Plan &p, const void *plane, int buf, bool pooled, const TrialStats *st,
                           uint32_t rank, cudaStream_t s) {
    if (!pooled) {
        dim3 grid((unsigned)((p.n_r / 8 + 255) / 256), (unsigned)p.pool_nb);
        pool_kernel<P><<<grid, 256, 0, s>>>((const typename P::real *)plane, p.pool[buf], p.pool_blk,
                                            p.n_r);
        FDAS_CUDA_TRY(cudaGetLastError());
    }
    switch (p.H) {
        case 2: return launch_bound<P, 2>(p, plane, buf, st, rank, s);
        case 4: return launch_bound<P, 4>(p, plane, buf, st, rank, s);
        case 8: return launch_bound<P, 8>(p, plane, buf, st, rank, s);
        default: return launch_bound<P, 16>(p, plane, buf, st, rank, s);
    }
}

}  // namespace

// first rows of the row blocks (and n_z at the end): runs of 3 or 4 rows (of 1 or 2
// for the smallest n_z)
std::vector<int32_t> pool_blocks(int n_z) {
    std::vector<int32_t> out;
    const int nb = (n_z + 3) / 4;
    for (int i = 0; i <= nb; ++i) out.push_back((int32_t)((int64_t)n_z * i / nb));
    return out;
}

// per block and harmonic j = 1..H the first and last source block (16 bits
// each), and per block the slots of the first ones (4 bits per harmonic) and
// which harmonics have two; false when the sources do not fit the kernel's
// slots (two blocks per block row, slots() per step of kBoundW of them)
bool pool_sources(const std::vector<int32_t> &blk, int n_z, int iz0, int H,
                  std::vector<uint32_t> *src, std::vector<uint4> *masks) {
    const int nb = (int)blk.size() - 1;
    std::vector<int32_t> of(n_z);
    for (int i = 0; i < nb; ++i) {
        if (blk[i + 1] - blk[i] > kPoolMaxRows) return false;
        for (int r = blk[i]; r < blk[i + 1]; ++r) of[r] = i;
    }
    src->assign((size_t)nb * H, 0u);
    masks->assign((size_t)nb, make_uint4(0u, 0u, 0u, 0u));
    for (int i = 0; i < nb; ++i)
        for (int j = 1; j <= H; ++j) {
            const int lo = of[iz0 + src_off(H, blk[i] - iz0, j)];
            const int hi = of[iz0 + src_off(H, blk[i + 1] - 1 - iz0, j)];
            if (hi < lo || hi > lo + 1 || (j == H && (lo != i || hi != i))) return false;
            (*src)[(size_t)i * H + j - 1] = (uint32_t)lo | ((uint32_t)hi << 16);
            if (j == H) continue;
            const int slots = kBoundW * j / H + 2, e = std::min(i + kBoundW, nb) - 1;
            if (of[iz0 + src_off(H, blk[e + 1] - 1 - iz0, j)] - lo + 1 > slots) return false;
            uint4 &m = (*masks)[i];
            (j <= 8 ? m.x : m.y) |= (uint32_t)(lo % slots) << (4 * ((j - 1) & 7));
            m.z |= (uint32_t)(hi != lo) << (j - 1);
        }
    return true;
}

fdas_status launch_harmonic_bound(Plan &p, const void *plane, int buf, bool pooled,
                                  const TrialStats *st, uint32_t rank, cudaStream_t s) {
    switch (p.prec) {
        case FDAS_FP32: return launch_bound_P<PrecF32>(p, plane, buf, pooled, st, rank, s);
        case FDAS_BF16: return launch_bound_P<PrecBF16>(p, plane, buf, pooled, st, rank, s);
        default: return launch_bound_P<PrecF16>(p, plane, buf, pooled, st, rank, s);
    }
}

FDAS_BOUNDS_LOG_TU(harmonic_bound)

}  // namespace fdas
