// Fourier slice stage on bins-fastest spectra (X[q][theta][bin], Y[trace][bin]
// per cube): the lanes of a warp are consecutive frequency bins.
//
// The arithmetic is that of slice_kernels.cu (the same taps, kernel weights,
// phases and deapodisation, see slice_math.cuh); the layout of the work is
// not.  A block owns a tile of TB bins and a range of azimuth slices of one
// cube.  It keeps the q grids of two neighbouring slices in shared memory as
// [grid point][bin], walks its slices in order, and in each interval
// [theta_j, theta_j+1) handles the traces whose first slice is j.  A trace's
// grid position differs from bin to bin, but a bin stays in its own bank, so in
// tiles of 32 and 16 bins neither the forward's reads nor the adjoint's integer
// atomics conflict, whatever the positions (with a bin per block and 32 traces
// per warp they hit random banks: 3.7 wavefronts per atomic, measured); in
// tiles of 8 bins (512-point grids) two of a warp's four traces do, half the
// time.  Every global access is a run of TB consecutive bins.
//
// The nos-point DFT of a grid column stays inside the lanes of its bin:
// nos = 16 R, n = n1 R + n2, p = p1 + 16 p2,
//   G[p] = sum_n2 w_R^(n2 p2) w_nos^(n2 p1) sum_n1 w_16^(n1 p1) x[n1 R + n2],
// a radix-16 step (fed from global memory), one layer of twiddles, and a
// radix-R step, in place in rows p1 + 16 n2.  Rows nos .. nos + W - 2 repeat
// rows 0 .. W - 2, so a trace's taps are consecutive rows (forward); the
// adjoint spreads into them and its first step folds them back.
//
// Bound: issue (68-71 % of the slots) with the L1 / shared-memory pipe at
// 57-71 %; the bin-per-block kernels had that pipe at 87-91 %, half of it
// conflicts.  Per launch on 16 cubes of 200-3000 traces, 64 q x 24 azimuths,
// 2048 bins (nos 128, W 7), bin per block -> these kernels: forward 823 -> 440
// us, adjoint 1108 -> 618; one 2000-trace gather, 100 q x 36 azimuths (nos 256,
// W 6) 99 -> 71 and 125 -> 92; one 8000-trace gather, 200 q x 72 azimuths (nos
// 512, W 6) 929 -> 595 and 1400 -> 756.
#pragma once

#include "fft.cuh"
#include "internal.cuh"
#include "slice_math.cuh"

namespace aahrt {

struct TileArgs {
    const TraceGeo *__restrict__ geo;      // by slice, then r^2
    const SliceGroup *__restrict__ groups;
    const int *__restrict__ slice_start;
    const float *__restrict__ dec;
    const float2 *__restrict__ tw;
    int *counter;
    long long total;                       // groups x tiles
    int nbins, ntiles, nq, ntheta, cq;
    float scale;
    float phicap;                          // bound on one kernel weight
    unsigned *ymax;
    const float *__restrict__ wsum;
    int ncube, nychunk, ychunk_log;
    EsPoly poly;
};

__host__ __device__ constexpr int tile_rows(int nos, int W) { return nos + W - 1; }

// Dynamic shared memory: two grids of nos + W - 1 rows of TB complex values,
// the nos twiddles and the deapodisation factor of every grid point.
inline size_t tile_smem(int nos, int W, int TB) {
    return ((size_t)2 * tile_rows(nos, W) * TB + nos) * sizeof(float2) + nos * sizeof(float);
}

// The sizes of one kernel instance: spreading width W, nos = 16 << LR grid
// points, TB bins per tile, THREADS threads.
template <int W_, int LR_, int TB_, int THREADS_>
struct Tile {
    static constexpr int W = W_, LR = LR_, R = 1 << LR_, NOS = 16 << LR_, TB = TB_;
    static constexpr int THREADS = THREADS_, NSUB = THREADS_ / TB_;
    static constexpr int MINB = 3;
    static constexpr int ROWS = NOS + W_ - 1;
};

// s_tw[16 n2 + p1] = exp(-2 pi i n2 p1 / nos), the twiddles between the two
// steps; s_dec[u] = factor of curvature l = (u + cq) mod nos (0 beyond nq),
// with the operator's 1/Nfft (a power of two, so it changes no rounding).
template <class T>
__device__ __forceinline__ void tile_tables(const TileArgs &a, float2 *s_tw, float *s_dec) {
    for (int i = threadIdx.x; i < T::NOS; i += T::THREADS) {
        s_tw[i] = __ldg(a.tw + (i >> 4) * (i & 15));
        const int l = (i + a.cq) & (T::NOS - 1);
        s_dec[i] = l < a.nq ? a.scale * __ldg(a.dec + l) : 0.f;
    }
}

// The block's work is done (thread 0 has drawn its last item): the last block
// of the grid returns true in every thread and clears the work counter, so the
// next launch finds it cleared without a memset between the kernels.
__device__ __forceinline__ bool tile_last_block(int *counter) {
    __shared__ int s_last;
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(counter + kDoneSlot, 1) == (int)gridDim.x - 1;
        if (s_last) counter[0] = counter[kDoneSlot] = 0;
    }
    __syncthreads();
    return s_last != 0;
}

// acc + w * g
__device__ __forceinline__ float2 axpy2(float w, float2 g, float2 acc) {
    return make_float2(fmaf(w, g.x, acc.x), fmaf(w, g.y, acc.y));
}

// The radix-16 DIF network on inputs of which only m < 4 and m >= 12 are
// nonzero (a column of nq <= nos / 2 curvatures centred on the grid): the
// first stage has one nonzero operand per butterfly.
template <bool INV>
__device__ __forceinline__ void dif16_centred(float2 *v) {
#pragma unroll
    for (int m = 0; m < 4; ++m) v[m + 8] = kappa_mul<INV>(v[m], 3, m);
#pragma unroll
    for (int m = 4; m < 8; ++m) {
        v[m] = v[m + 8];
        v[m + 8] = kappa_mul<INV>(make_float2(-v[m].x, -v[m].y), 3, m);
    }
    dif_network<3, INV, true>(v);
    dif_network<3, INV, true>(v + 8);
}

// Half of a radix-32 DFT (nos = 512): v[n] = (x[n] +- x[n + 16]) w_32^(n b),
// whose radix-16 DFT is the outputs of parity b; x(n) reads input n.
template <bool INV, class Read>
__device__ __forceinline__ void half_of_32(float2 *v, int b, const float2 *s_tw, Read x) {
#pragma unroll
    for (int n = 0; n < 16; ++n) {
        const float2 p = x(n), q = x(n + 16);
        if (b == 0) {
            v[n] = cadd2(p, q);
        } else {
            const float2 w = s_tw[16 * 16 + n];
            v[n] = cmul(csub2(p, q), make_float2(w.x, INV ? -w.y : w.y));
        }
    }
}

// Forward, second step: rows p1 + 16 n2 -> rows p1 + 16 p2, n2, p2 < R, and
// the wrapped copies of the first W - 1 rows.  R = 32 is done by two threads,
// one for each parity of p2 (16 values each in registers), which both read
// all 32 rows before either writes.
template <class T>
__device__ __forceinline__ void tile_fwd_step2(float2 *G, const float2 *s_tw, int sub, int bin) {
    constexpr int TB = T::TB, R = T::R;
    if constexpr (T::LR == 5) {
        static_assert(T::LR != 5 || T::NSUB == 32, "two threads per column of 32 rows");
        const int p1 = sub & 15, b = sub >> 4;
        float2 *col = G + p1 * TB + bin;
        float2 v[16];
        half_of_32<false>(v, b, s_tw, [&](int n) { return col[n * 16 * TB]; });
        dif_network<4, false, true>(v);
        __syncthreads();
#pragma unroll
        for (int m = 0; m < 16; ++m) col[(2 * rev_bits_c<4>(m) + b) * 16 * TB] = v[m];
        if (b == 0 && p1 < T::W - 1) col[T::NOS * TB] = v[0];
    } else {
#pragma unroll
        for (int p0 = 0; p0 < 16; p0 += T::NSUB) {
            const int p1 = p0 + sub;
            float2 *col = G + p1 * TB + bin;
            float2 v[R];
#pragma unroll
            for (int n = 0; n < R; ++n) v[n] = col[n * 16 * TB];
            dif_network<T::LR, false, true>(v);
#pragma unroll
            for (int m = 0; m < R; ++m) col[rev_bits_c<T::LR>(m) * 16 * TB] = v[m];
            if (p1 < T::W - 1) col[T::NOS * TB] = v[0];
        }
    }
}

// Slice j of the lane's bin into the grid G: deapodised column, DFT along q.
// Grid point u = m R + n2 holds curvature l = u + cq (u < nq - cq) or
// u + cq - nos (u >= nos - cq), else zero.
template <class T>
__device__ __forceinline__ void tile_fwd_grid(const TileArgs &a, const float2 *__restrict__ Xc,
                                              int j, float2 *G, const float2 *s_tw,
                                              const float *s_dec, int bin, int sub, bool live) {
    constexpr int TB = T::TB, R = T::R;
    const long long sl = (long long)a.ntheta * a.nbins;      // from a curvature to the next
    const bool centred = a.nq <= T::NOS / 2;                 // only m < 4 and m >= 12 nonzero
    for (int n2 = sub; n2 < R; n2 += T::NSUB) {
        const float2 *p = Xc + (long long)j * a.nbins + (n2 + a.cq) * sl;
        const int hi = live ? a.nq - a.cq - n2 : 0;
        const int lo = live ? T::NOS - a.cq - n2 : T::NOS;
        float2 v[16];
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            v[m] = make_float2(0.f, 0.f);
            if (m >= 4 && m < 12 && centred) continue;
            // (past L1, which keeps the trace records)
            if (m < 8 ? m * R < hi : m * R >= lo)
                v[m] = __ldcg(p + (m < 8 ? m * R : m * R - T::NOS) * sl);
        }
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            if (m >= 4 && m < 12 && centred) continue;
            const float d = s_dec[m * R + n2];
            v[m].x *= d;
            v[m].y *= d;
        }
        if (centred) dif16_centred<false>(v);
        else dif_network<4, false, true>(v);
        float2 *col = G + (n2 << 4) * TB + bin;
        const float2 *tw = s_tw + (n2 << 4);
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            const int p1 = rev_bits_c<4>(m);
            col[p1 * TB] = p1 == 0 ? v[m] : cmul(v[m], tw[p1]);
        }
    }
    __syncthreads();
    tile_fwd_step2<T>(G, s_tw, sub, bin);
}

template <class T>
__global__ void __launch_bounds__(T::THREADS, T::MINB)
tile_fwd_kernel(const TileArgs a, const float2 *__restrict__ X, float2 *__restrict__ Y) {
    extern __shared__ float4 smem_f4[];
    constexpr int W = T::W, TB = T::TB, NSUB = T::NSUB, GRID = T::ROWS * TB;
    __shared__ long long s_item;
    float2 *buf = reinterpret_cast<float2 *>(smem_f4);
    float2 *s_tw = buf + 2 * GRID;
    float *s_dec = reinterpret_cast<float *>(s_tw + T::NOS);
    tile_tables<T>(a, s_tw, s_dec);
    const int bin = threadIdx.x & (TB - 1);
    const int sub = threadIdx.x / TB;
    for (;;) {
        if (threadIdx.x == 0) s_item = (long long)atomicAdd(a.counter, 1);
        __syncthreads();
        const long long item = s_item;
        if (item >= a.total) break;
        const int gi = (int)(item / a.ntiles);
        const int kb = (int)(item - (long long)gi * a.ntiles) * TB + bin;
        const SliceGroup g = a.groups[gi];
        const bool live = kb < a.nbins;
        const float2 *Xc = X + g.x_off + kb;
        float2 *Yc = Y + g.y_off + kb;
        const TraceGeo *geo = a.geo + g.geo_off;
        const int *ss = a.slice_start + g.ss_off;
        int have = -1;               // slice whose grid is in buffer `cur`
        int cur = 0;
        for (int jj = 0; jj < g.nj; ++jj) {
            const int j = g.ja + jj;
            const int t0 = ss[j], t1 = ss[j + 1];
            if (t0 == t1) continue;              // no trace reads this interval
            const int jn = j + 1 == a.ntheta ? 0 : j + 1;
            if (have != j)
                tile_fwd_grid<T>(a, Xc, j, buf + cur * GRID, s_tw, s_dec, bin, sub, live);
            tile_fwd_grid<T>(a, Xc, jn, buf + (cur ^ 1) * GRID, s_tw, s_dec, bin, sub, live);
            // a trace's record is loaded one trace ahead
            TraceGeo nxt{};
            if (t0 + sub < t1) nxt = geo[t0 + sub];
            __syncthreads();
            const float2 *G0 = buf + cur * GRID + bin;
            const float2 *G1 = buf + (cur ^ 1) * GRID + bin;
            for (int t = t0 + sub; t < t1; t += NSUB) {
                const TraceGeo tr = nxt;
                if (t + NSUB < t1) nxt = geo[t + NSUB];
                const TapSet ts = trace_taps<W>(tr.A, tr.B, (unsigned)kb, T::LR + 4);
                float phi[W];
                es_weights<W>(a.poly, ts.g, phi);
                const int row = (ts.u0 & (T::NOS - 1)) * TB;
                float2 p = make_float2(0.f, 0.f), q = p;
#pragma unroll
                for (int i = 0; i < W; ++i) {
                    p = axpy2(phi[i], G0[row + i * TB], p);
                    q = axpy2(phi[i], G1[row + i * TB], q);
                }
                const float ar = fmaf(tr.w0, p.x, tr.w1 * q.x);
                const float ai = fmaf(tr.w0, p.y, tr.w1 * q.y);
                float sn, cs;
                phase_cs(ts.ph, &sn, &cs);
                // times exp(-2 pi i ph) = cs - i sn
                if (live)
                    Yc[(long long)tr.col * a.nbins] =
                        make_float2(ar * cs + ai * sn, ai * cs - ar * sn);
            }
            __syncthreads();
            cur ^= 1;
            have = jn;
        }
        __syncthreads();             // s_item is rewritten next
    }
    tile_last_block(a.counter);
}

// ------------------------------------------------------------- adjoint
// A grid row holds TB real parts, then TB imaginary parts in 32-bit fixed point
// while spreading, and TB complex floats between the two DFT steps (every row
// is read, rewritten and cleared by the lanes of one warp).  With TB = 16 a
// warp spreads two traces: its halves take the real and the imaginary plane in
// opposite order, so their rows never share a bank (with TB = 8, four traces:
// pairs of them do, half the time).
template <int TB>
struct PlanePair {
    const int *first, *second;   // the plane this half warp takes first, and the other
    bool swap;
    __device__ __forceinline__ explicit PlanePair(const int *p)
        : first(p), second(p + TB), swap(TB < 32 && (threadIdx.x & 16)) {
        if (swap) {
            first = p + TB;
            second = p;
        }
    }
    __device__ __forceinline__ int2 load(int off) const {
        const int x = first[off], y = second[off];
        return swap ? make_int2(y, x) : make_int2(x, y);
    }
};

template <int TB, int W>
__device__ __forceinline__ void tile_spread(int *G, const float *phi, int row, float vr, float vi,
                                            int bin) {
    const bool swap = TB < 32 && (threadIdx.x & 16);
    const float x0 = swap ? vi : vr, x1 = swap ? vr : vi;
    int *p0 = G + row * 2 * TB + bin + (swap ? TB : 0);
    int *p1 = G + row * 2 * TB + bin + (swap ? 0 : TB);
#pragma unroll
    for (int i = 0; i < W; ++i) {
        atomicAdd(p0 + i * 2 * TB, __float2int_rn(phi[i] * x0));
        atomicAdd(p1 + i * 2 * TB, __float2int_rn(phi[i] * x1));
    }
}

// Adjoint, first step: rows p1 + 16 p2 (fixed point; wrapped rows folded in
// and cleared) -> inverse radix-R, conjugate twiddles, floats in rows
// p1 + 16 n2.  R = 32 by two threads, one for each parity of n2.
template <class T>
__device__ __forceinline__ void tile_adj_step1(float2 *G, int sub, int bin, const float2 *s_tw,
                                               float ifx) {
    constexpr int TB = T::TB, R = T::R;
    // row n of the column in fixed point
    auto fixed = [&](const PlanePair<TB> &pl, int p1, int n) {
        int2 v = pl.load(n * 32 * TB);
        if (n == 0 && p1 < T::W - 1) {
            const int2 u = pl.load(T::NOS * 2 * TB);
            v.x += u.x;
            v.y += u.y;
        }
        return make_float2((float)v.x * ifx, (float)v.y * ifx);
    };
    auto twiddled = [&](float2 v, int n2, int p1) {
        const float2 w = s_tw[(n2 << 4) + p1];
        return cmul(v, make_float2(w.x, -w.y));
    };
    if constexpr (T::LR == 5) {
        const int p1 = sub & 15, b = sub >> 4;           // NSUB = 32
        const PlanePair<TB> pl(reinterpret_cast<const int *>(G + p1 * TB) + bin);
        float2 v[16];
        half_of_32<true>(v, b, s_tw, [&](int n) { return fixed(pl, p1, n); });
        dif_network<4, true, true>(v);
        __syncthreads();
        float2 *col = G + p1 * TB + bin;
        if (b == 0 && p1 < T::W - 1) col[T::NOS * TB] = make_float2(0.f, 0.f);
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            const int n2 = 2 * rev_bits_c<4>(m) + b;
            col[n2 * 16 * TB] = twiddled(v[m], n2, p1);
        }
    } else {
#pragma unroll
        for (int p0 = 0; p0 < 16; p0 += T::NSUB) {
            const int p1 = p0 + sub;
            const PlanePair<TB> pl(reinterpret_cast<const int *>(G + p1 * TB) + bin);
            float2 v[R];
#pragma unroll
            for (int n = 0; n < R; ++n) v[n] = fixed(pl, p1, n);
            dif_network<T::LR, true, true>(v);
            float2 *col = G + p1 * TB + bin;
            __syncwarp();        // the row's lanes have read it
            if (p1 < T::W - 1) col[T::NOS * TB] = make_float2(0.f, 0.f);
#pragma unroll
            for (int m = 0; m < R; ++m) {
                const int n2 = rev_bits_c<T::LR>(m);
                col[n2 * 16 * TB] = n2 == 0 ? v[m] : twiddled(v[m], n2, p1);
            }
        }
    }
}

// Adjoint, second step: rows p1 + 16 n2 (cleared once read) -> inverse radix-16,
// deapodised curvatures of slice j.
template <class T>
__device__ __forceinline__ void tile_adj_step2(const TileArgs &a, float2 *G, int sub, int bin,
                                               const float *s_dec, float2 *__restrict__ Xc, int j,
                                               bool live) {
    constexpr int TB = T::TB, R = T::R;
    const long long sl = (long long)a.ntheta * a.nbins;
    const bool centred = a.nq <= T::NOS / 2;
    for (int n2 = sub; n2 < R; n2 += T::NSUB) {
        float2 *col = G + (n2 << 4) * TB + bin;
        float2 v[16];
#pragma unroll
        for (int p1 = 0; p1 < 16; ++p1) {
            v[p1] = col[p1 * TB];
            col[p1 * TB] = make_float2(0.f, 0.f);
        }
        dif_network<4, true, true>(v);
        float2 *p = Xc + (long long)j * a.nbins + (n2 + a.cq) * sl;
        const int hi = live ? a.nq - a.cq - n2 : 0;
        const int lo = live ? T::NOS - a.cq - n2 : T::NOS;
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            const int n1 = rev_bits_c<4>(m);
            if (n1 >= 4 && n1 < 12 && centred) continue;
            if (n1 < 8 ? n1 * R < hi : n1 * R >= lo) {
                const float d = s_dec[n1 * R + n2];
                p[(n1 < 8 ? n1 * R : n1 * R - T::NOS) * sl] = make_float2(v[m].x * d, v[m].y * d);
            }
        }
    }
}

template <class T>
__global__ void __launch_bounds__(T::THREADS, T::MINB)
tile_adj_kernel(const TileArgs a, const float2 *__restrict__ Y, float2 *__restrict__ X) {
    extern __shared__ float4 smem_f4[];
    constexpr int W = T::W, TB = T::TB, NSUB = T::NSUB, GRID = T::ROWS * TB;
    __shared__ long long s_item;
    float2 *buf = reinterpret_cast<float2 *>(smem_f4);
    float2 *s_tw = buf + 2 * GRID;
    float *s_dec = reinterpret_cast<float *>(s_tw + T::NOS);
    tile_tables<T>(a, s_tw, s_dec);
    // the grids start cleared, and the last reader of a row clears it
    for (int i = threadIdx.x; i < 2 * GRID; i += T::THREADS) buf[i] = make_float2(0.f, 0.f);
    const int bin = threadIdx.x & (TB - 1);
    const int sub = threadIdx.x / TB;
    for (;;) {
        if (threadIdx.x == 0) s_item = (long long)atomicAdd(a.counter, 1);
        __syncthreads();
        const long long item = s_item;
        if (item >= a.total) break;
        const int gi = (int)(item / a.ntiles);
        const int kb = (int)(item - (long long)gi * a.ntiles) * TB + bin;
        const SliceGroup g = a.groups[gi];
        const bool live = kb < a.nbins;
        const float2 *Yc = Y + g.y_off + kb;
        float2 *Xc = X + g.x_off + kb;
        const TraceGeo *geo = a.geo + g.geo_off;
        const int *ss = a.slice_start + g.ss_off;
        // fixed-point scale of a slice: 2^30 over the largest value a grid
        // point can reach (every trace of the slice at most phicap there)
        const float M = live ? __uint_as_float(__ldcg(a.ymax + (long long)g.cube * a.nychunk +
                                                      (kb >> a.ychunk_log)))
                             : 0.f;
        const float *ws = a.wsum + (long long)g.cube * a.ntheta;
        int cur = 0;
        // interval jj spreads into slice jj (weights w0) and jj + 1 (w1);
        // interval -1 holds the traces before the first owned slice
        float bound1 = 0.f;          // of slice j + 1
        for (int jj = -1; jj < g.nj; ++jj) {
            int j = g.ja + jj;
            if (j < 0) j += a.ntheta;
            const int jn = j + 1 == a.ntheta ? 0 : j + 1;
            const int t0 = ss[j], t1 = ss[j + 1];
            const float bound0 = bound1;
            bound1 = M * __ldg(ws + jn) * a.phicap;
            const float fx0 = bound0 > 0.f ? 1073741824.0f / bound0 : 0.f;   // 2^30 / bound
            const float fx1 = bound1 > 0.f ? 1073741824.0f / bound1 : 0.f;
            const bool own0 = jj >= 0, own1 = jj + 1 < g.nj;
            int *G0 = reinterpret_cast<int *>(buf + cur * GRID);
            int *G1 = reinterpret_cast<int *>(buf + (cur ^ 1) * GRID);
            if (live && t0 + sub < t1) {
                // a trace's record is loaded two traces ahead of its use, its y
                // (found by the record) one ahead
                TraceGeo nxt = geo[t0 + sub], far{};
                if (t0 + sub + NSUB < t1) far = geo[t0 + sub + NSUB];
                float2 ynxt = __ldcg(Yc + (long long)nxt.col * a.nbins);
                for (int t = t0 + sub; t < t1; t += NSUB) {
                    const TraceGeo tr = nxt;
                    const float2 y = ynxt;
                    nxt = far;
                    if (t + NSUB < t1) ynxt = __ldcg(Yc + (long long)nxt.col * a.nbins);
                    if (t + 2 * NSUB < t1) far = geo[t + 2 * NSUB];
                    const TapSet ts = trace_taps<W>(tr.A, tr.B, (unsigned)kb, T::LR + 4);
                    float phi[W];
                    es_weights<W>(a.poly, ts.g, phi);
                    float sn, cs;
                    phase_cs(ts.ph, &sn, &cs);
                    // y * exp(+2 pi i ph)
                    const float vr = y.x * cs - y.y * sn;
                    const float vi = y.x * sn + y.y * cs;
                    const int row = ts.u0 & (T::NOS - 1);
                    const float f0 = tr.w0 * fx0, f1 = tr.w1 * fx1;
                    if (own0) tile_spread<TB, W>(G0, phi, row, f0 * vr, f0 * vi, bin);
                    if (own1) tile_spread<TB, W>(G1, phi, row, f1 * vr, f1 * vi, bin);
                }
            }
            __syncthreads();
            if (own0 && !(__ldg(ws + j) > 0.f)) {
                // no trace reaches the slice: its grid is untouched
                if (live)
                    for (int l = sub; l < a.nq; l += NSUB)
                        Xc[((long long)l * a.ntheta + j) * a.nbins] = make_float2(0.f, 0.f);
            } else if (own0) {
                float2 *G = buf + cur * GRID;
                const float ifx = bound0 > 0.f ? bound0 * 9.3132257461547852e-10f : 0.f;   // 1/fx0
                tile_adj_step1<T>(G, sub, bin, s_tw, ifx);
                __syncthreads();
                tile_adj_step2<T>(a, G, sub, bin, s_dec, Xc, j, live);
                __syncthreads();
            }
            cur ^= 1;
        }
        __syncthreads();             // s_item is rewritten next
    }
    // the bound table is read: clear it for the analysis that writes the next Y
    if (tile_last_block(a.counter))
        for (int i = threadIdx.x; i < a.ncube * a.nychunk; i += T::THREADS) a.ymax[i] = 0u;
}

}  // namespace aahrt
