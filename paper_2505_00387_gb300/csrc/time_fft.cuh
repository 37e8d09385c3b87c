// Time-axis stages on bins-fastest spectra X[q][theta][bin], Y[trace][bin]:
// the arithmetic of time_kernels.cu (stretch and unstretch resamplers, two
// real columns per complex FFT, FISTA epilogues) with the FFT held in
// registers.
//
// A column pair's frame of N = 256 C samples (C = 2 .. 32) belongs to
// T = 16 C threads of 16 values each; index n = t + T a on one side,
// p0 + 16 p1 + 256 p2 on the other:
//   y[p] = sum_c w_C^(c p2) w_T^(c p1) sum_b w_16^(b p1) w_N^(t p0)
//          sum_a w_16^(a p0) x[t + T a],            t = C b + c,
// three register steps (radix 16, 16, C) and two exchanges through shared
// memory.  The first crosses the block (one barrier); the second stays inside
// the C threads of one p0, which lie in one warp, so it needs none.  Spectra
// arrive in the frame by cp.async past L1 and the radix steps work in
// registers: a frame passes through shared memory 5-6 times a transform,
// against 8 with every radix step working there (time_kernels.cu).
//
// Bound: the L1 / shared-memory pipe (85 %) and issue (60-66 % of the slots),
// at 64 registers (four blocks of 256 threads an SM; 80 and three in the
// analysis alone) instead of 128 and two.  Per launch on 16 cubes of 1001
// samples and 200-3000 traces (4096-sample frames), shared-memory FFT ->
// these kernels: data half 839 -> 442 us, model half 734 -> 477; of 32 such
// cubes analysis 661 -> 431 (model) and 1064 -> 638 (data), synthesis 699 -> 469
// (data) and 977 -> 685 (model).
//
// Shared-memory layout of an exchange: element (p0, i) of group p0 at
// p0 (T + C) + i (the skew spreads the groups a half warp touches over the
// banks), in the second one (p1, c) at p1 C + (c ^ (p1 mod C)).  A frame in
// natural order holds sample n at n + (n >> 4).
#pragma once

#include "fft.cuh"
#include "internal.cuh"
#include "resample.cuh"

namespace aahrt {

template <int C_>
struct Frame {
    static constexpr int C = C_, T = 16 * C_, N = 256 * C_;
    static constexpr int LC = C_ == 2 ? 1 : C_ == 4 ? 2 : C_ == 8 ? 3 : C_ == 16 ? 4 : 5;
    static constexpr int L = 8 + LC;
    static constexpr int GS = T + C_;                  // group stride of an exchange
    // exchange or natural frame with one zero sample either side
    static constexpr int LEN = N + N / 16 + 4;
    static constexpr int THREADS = T > 256 ? T : 256;  // most threads of a block
    // blocks an SM holds: four (two of 512 threads) at 64 registers; the
    // analysis alone keeps 80, which its table entries and rows in flight need
    // (431 against 535 us for the model columns of 32 cubes; at 80 the model
    // analyses of 2048 samples and fewer still spill 32 to 36 words, the other
    // kernels 7 or fewer)
    static constexpr int MINB = T > 256 ? 2 : 4, MINB_ANA = T > 256 ? 1 : 3;
};

__device__ __forceinline__ int frame_at(int n) { return 2 + n + (n >> 4); }

// Shared memory of one block: tables, the source fractions of a transposed
// resampler, and per pair the frame and the staged rows (one zero row before,
// four after).
struct FrameMem {
    float2 *s_tw;       // [p1][c] = exp(-2 pi i c p1 / T)
    float *sfr;
    float2 *sm;         // this pair's frame
    float2 *stg;        // this pair's staged rows, row 0 at stg
};
// (seq > 1: the block takes that many pairs in turn and stages all their rows.)
// (The strides put neighbouring pairs four banks apart modulo 16: LEN is 4
// modulo 16, so rows are a multiple of 16 beside a frame, 4 more without one.)
__host__ __device__ constexpr int staged_rows(int nrows) { return (nrows + 5 + 15) & ~15; }
__host__ __device__ constexpr int turn_rows(int nrows) { return staged_rows(nrows) + 4; }
template <class F>
__host__ __device__ constexpr size_t frame_smem(int pairs, int seq, int nrows, int nfrac) {
    return (size_t)F::T * sizeof(float2) + (size_t)((nfrac + 3) & ~3) * sizeof(float) +
           (size_t)pairs * (F::LEN + (seq > 1 ? seq * turn_rows(nrows) : staged_rows(nrows))) *
               sizeof(float2);
}
template <class F>
__device__ __forceinline__ FrameMem frame_mem(float4 *base, int pair, int nrows, int nfrac) {
    FrameMem m;
    m.s_tw = reinterpret_cast<float2 *>(base);
    m.sfr = reinterpret_cast<float *>(m.s_tw + F::T);
    float2 *p = reinterpret_cast<float2 *>(m.sfr + ((nfrac + 3) & ~3));
    m.sm = p + (size_t)pair * (F::LEN + staged_rows(nrows));
    m.stg = m.sm + F::LEN + 1;
    return m;
}

template <class F>
__device__ __forceinline__ void frame_tables(float2 *s_tw, const float2 *__restrict__ tw) {
    for (int i = threadIdx.x; i < F::T; i += blockDim.x)
        s_tw[i] = __ldg(tw + 16 * (i / F::C) * (i & (F::C - 1)));
}

// The four table values (powers 1, 2, 4, 8 of exp(-2 pi i t / N)) the first
// step's twiddles are built from, loaded ahead of their use.
struct FrameTwiddle {
    float2 w[4];
};
template <class F>
__device__ __forceinline__ FrameTwiddle frame_twiddle(const float2 *__restrict__ tw, int t) {
    FrameTwiddle r;
#pragma unroll
    for (int b = 0; b < 4; ++b) r.w[b] = __ldg(tw + ((t << b) & (F::N - 1)));
    return r;
}

// The transform of one pair; v[a] = x[t + T a] in, v[m] = y[frame_out(m)] out.
// Ends without a barrier: sm may be rewritten outside the thread's own group
// only after one.
template <class F, bool INV>
__device__ __forceinline__ void frame_fft(float2 *v, float2 *sm, const FrameTwiddle &ft,
                                          const float2 *s_tw, int t) {
    constexpr int C = F::C;
    dif_network<4, INV, true>(v);
    {
        float2 w[16];
#pragma unroll
        for (int b = 0; b < 4; ++b) w[1 << b] = make_float2(ft.w[b].x, INV ? -ft.w[b].y : ft.w[b].y);
#pragma unroll
        for (int r = 3; r < 16; ++r) {
            if ((r & (r - 1)) == 0) continue;
            int hi = r;
            while (hi & (hi - 1)) hi &= hi - 1;      // highest set bit
            w[r] = cmul(w[hi], w[r - hi]);
        }
#pragma unroll
        for (int m = 1; m < 16; ++m) v[m] = cmul(v[m], w[rev_bits_c<4>(m)]);
    }
#pragma unroll
    for (int m = 0; m < 16; ++m) sm[rev_bits_c<4>(m) * F::GS + t] = v[m];
    __syncthreads();
    const int c = t & (C - 1);
    float2 *grp = sm + (t / C) * F::GS;
#pragma unroll
    for (int b = 0; b < 16; ++b) v[b] = grp[C * b + c];
    dif_network<4, INV, true>(v);
#pragma unroll
    for (int m = 1; m < 16; ++m) {
        float2 w = s_tw[rev_bits_c<4>(m) * C + c];
        if (INV) w.y = -w.y;
        v[m] = cmul(v[m], w);
    }
    __syncwarp();
#pragma unroll
    for (int m = 0; m < 16; ++m) {
        const int p1 = rev_bits_c<4>(m);
        grp[p1 * C + (c ^ (p1 & (C - 1)))] = v[m];
    }
    __syncwarp();
    if constexpr (C == 32) {
        // half of a radix-32 step: outputs p2 of the thread's parity
        const int p1 = c & 15;
        const bool odd = c >> 4;
#pragma unroll
        for (int n = 0; n < 16; ++n) {
            const float2 x = grp[p1 * C + (n ^ p1)], y = grp[p1 * C + ((n + 16) ^ p1)];
            float2 w = s_tw[n * C + 16];               // exp(-2 pi i n / 32)
            if (INV) w.y = -w.y;
            v[n] = odd ? cmul(csub2(x, y), w) : cadd2(x, y);
        }
        dif_network<4, INV, true>(v);
    } else {
#pragma unroll
        for (int j = 0; j < 16 / C; ++j) {
            const int p1 = c + C * j;
#pragma unroll
            for (int i = 0; i < C; ++i) v[j * C + i] = grp[p1 * C + (i ^ (p1 & (C - 1)))];
            dif_network<F::LC, INV, true>(v + j * C);
        }
    }
}

// index of frame_fft's output v[m]
template <class F>
__device__ __forceinline__ int frame_out(int m, int t) {
    const int g = t & (F::C - 1), p0 = t / F::C;
    if constexpr (F::C == 32) return p0 + 16 * (g & 15) + 256 * (2 * rev_bits_c<4>(m) + (g >> 4));
    else return p0 + 16 * (g + F::C * (m / F::C)) + 256 * rev_bits_c<F::LC>(m % F::C);
}

template <int BYTES>
__device__ __forceinline__ void frame_cp(void *smem, const void *gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    if (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem));
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(sa), "l"(gmem), "n"(BYTES));
}
__device__ __forceinline__ void frame_cp_wait() {
    asm volatile("cp.async.commit_group;\n");
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}
// the transposed resampler's fractions (the array is padded to whole float4)
__device__ __forceinline__ void copy_fractions(float *sfr, const float *__restrict__ frac, int n) {
    for (int i = threadIdx.x; 4 * i < n; i += blockDim.x) frame_cp<16>(sfr + 4 * i, frac + 4 * i);
}
// Where U^T changes from gathering to scattering (see frame_unstretch_t).
struct FrameScatter {
    int i0, n0;
};

struct FrameBound {      // amplitude bound table of the data spectrum, or max == null
    unsigned *max;
    int nchunk, chunk_log;
};

// The stretch S onto the frame, one frame row per register.
template <class F, int INTERP>
__device__ __forceinline__ void frame_stretch(const FrameMem &mem, const DevResampler &rs,
                                              int nrows, int t, float2 *v) {
    constexpr int T = F::T, AHEAD = 4;
    // row table entries are loaded AHEAD rows early
    int2 e[AHEAD];
#pragma unroll
    for (int a = 0; a < AHEAD; ++a) {
        const int n = min(t + T * a, rs.nrows - 1);
        e[a] = __ldg(reinterpret_cast<const int2 *>(rs.pos + n));
    }
#pragma unroll
    for (int a = 0; a < 16; ++a) {
        const int2 cur = e[a % AHEAD];
        if (a + AHEAD < 16) {
            const int n = min(t + T * (a + AHEAD), rs.nrows - 1);
            e[a % AHEAD] = __ldg(reinterpret_cast<const int2 *>(rs.pos + n));
        }
        float2 s = make_float2(0.f, 0.f);
        if (t + T * a < rs.nrows) {
            const float fr = __int_as_float(cur.y);
            // positions past the last row (a model axis shorter than the
            // data's) read the zero rows there
            const float2 *row = mem.stg + min(cur.x, nrows + 1);
#pragma unroll
            for (int q = 0; q < Taps<INTERP>::n; ++q) {
                const int k = Taps<INTERP>::t0 + q;
                const float w = tap_weight<INTERP>(k, fr);
                const float2 x = row[k];
                s.x = fmaf(w, x.x, s.x);
                s.y = fmaf(w, x.y, s.y);
            }
        }
        v[a] = s;
    }
}

// U^T onto the frame.  Source row i adds to the frame rows of its taps; the
// frame rows grow as i^2, so all but the first rows have few or no sources and
// a gather would mostly run empty loops.  Rows i >= sc.i0 (from there every
// row starts at a new frame row) are scattered, rows of equal i mod 4 in one
// pass (their taps are disjoint), in four passes; frame rows below sc.n0 (all
// that the first i0 rows reach) are gathered, four lanes to a row, one for
// each tap.  The order of every sum is fixed.
template <class F, int INTERP>
__device__ __forceinline__ void frame_unstretch_t(const FrameMem &mem, const DevResampler &rs,
                                                  const FrameScatter &sc, int nrows, int t,
                                                  float2 *v) {
    constexpr int T = F::T, NT = Taps<INTERP>::n, T0 = Taps<INTERP>::t0;
    float2 *z = mem.sm;
    // first block of scattered rows' entries, ahead of the gather
    int2 e[4];
#pragma unroll
    for (int c = 0; c < 4; ++c)
        e[c] = __ldg(reinterpret_cast<const int2 *>(rs.pos + min(sc.i0 + 4 * t + c, nrows - 1)));
#pragma unroll
    for (int a = 0; a < 16; ++a)
        if (t + T * a >= sc.n0) z[t + T * a] = make_float2(0.f, 0.f);
    const int q = t & 3;
    for (int r0 = 0; r0 < sc.n0; r0 += T / 4) {
        const int n = r0 + (t >> 2);
        float2 s = make_float2(0.f, 0.f);
        if (n < sc.n0 && q < NT) {
            const int2 g = __ldg(reinterpret_cast<const int2 *>(rs.rng + n));
            int r = g.x;
            for (int p = NT - 1; p > q; --p) r += (g.y >> (8 * p)) & 255;
            const int end = r + ((g.y >> (8 * q)) & 255);
            for (; r < end; ++r) {
                const float fr = mem.sfr[r];
                float w = 0.f;
#pragma unroll
                for (int p = 0; p < NT; ++p)
                    if (q == p) w = tap_weight<INTERP>(T0 + p, fr);
                const float2 x = mem.stg[r];
                s.x = fmaf(w, x.x, s.x);
                s.y = fmaf(w, x.y, s.y);
            }
        }
#pragma unroll
        for (int sh = 1; sh < 4; sh *= 2) {
            s.x += __shfl_xor_sync(0xffffffffu, s.x, sh);
            s.y += __shfl_xor_sync(0xffffffffu, s.y, sh);
        }
        if (n < sc.n0 && q == 0) z[n] = s;
    }
    __syncthreads();
    for (int b = sc.i0; b < nrows; b += 4 * T) {
        if (b > sc.i0) {
#pragma unroll
            for (int c = 0; c < 4; ++c)
                e[c] = __ldg(reinterpret_cast<const int2 *>(rs.pos + min(b + 4 * t + c, nrows - 1)));
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int i = b + 4 * t + c;
            if (i < nrows) {
                const float fr = __int_as_float(e[c].y);
                const float2 x = mem.stg[i];
                const int n = e[c].x + T0;
#pragma unroll
                for (int p = 0; p < NT; ++p) {
                    const float w = tap_weight<INTERP>(T0 + p, fr);
                    if (n + p >= sc.n0 && n + p < rs.nrows) {
                        float2 s = z[n + p];
                        s.x = fmaf(w, x.x, s.x);
                        s.y = fmaf(w, x.y, s.y);
                        z[n + p] = s;
                    }
                }
            }
            __syncthreads();
        }
    }
#pragma unroll
    for (int a = 0; a < 16; ++a) v[a] = z[t + T * a];
    __syncthreads();
}

// Analysis of the staged rows up to the pair's spectrum Z (natural order, in
// the frame): resample onto the frame, FFT; before_barrier() runs ahead of the
// last barrier.
template <class F, int INTERP, bool TRANS, class Fn>
__device__ __forceinline__ void frame_spectrum(const FrameMem &mem, const DevResampler &rs,
                                               const FrameScatter &sc, int nrows,
                                               const float2 *__restrict__ tw, int t,
                                               Fn before_barrier) {
    const FrameTwiddle ft = frame_twiddle<F>(tw, t);
    float2 v[16];
    if (TRANS) frame_unstretch_t<F, INTERP>(mem, rs, sc, nrows, t, v);
    else frame_stretch<F, INTERP>(mem, rs, nrows, t, v);
    frame_fft<F, false>(v, mem.sm, ft, mem.s_tw, t);
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 16; ++m) mem.sm[frame_at(frame_out<F>(m, t))] = v[m];
    before_barrier();
    __syncthreads();
}

// Bin k of the two real columns whose spectrum A + iB the frame holds:
// A = (Z_k + conj Z_{N-k})/2, B = (Z_k - conj Z_{N-k})/(2i).
template <class F>
__device__ __forceinline__ float4 frame_bin(const float2 *sm, int k) {
    const float2 zk = sm[frame_at(k)];
    const float2 zn = sm[frame_at((F::N - k) & (F::N - 1))];
    return make_float4(0.5f * (zk.x + zn.x), 0.5f * (zk.y - zn.y), 0.5f * (zk.y + zn.y),
                       -0.5f * (zk.x - zn.x));
}

// Analysis of the staged rows: their spectrum, unpacked to bins [0, nbins) of
// the pair's columns.
template <class F, int INTERP, bool TRANS>
__device__ __forceinline__ void frame_analyse(const FrameMem &mem, const ColGroup &cg, bool on,
                                              const DevResampler &rs, const FrameScatter &sc,
                                              int nrows, const float2 *__restrict__ tw, int nbins,
                                              int t, float2 *__restrict__ out,
                                              const FrameBound &ybd) {
    constexpr int T = F::T;
    // (a block of several pairs has few chunks: pairs x chunks <= 128)
    __shared__ unsigned s_ymax[128];
    const bool bound = TRANS && ybd.max != nullptr;
    unsigned *ym = s_ymax + (threadIdx.x / T) * ybd.nchunk;
    frame_spectrum<F, INTERP, TRANS>(mem, rs, sc, nrows, tw, t, [&] {
        if (bound)
            for (int i = t; i < ybd.nchunk; i += T) ym[i] = 0u;
    });
    const bool two = cg.ncol > 1;
    float2 *d0 = out + cg.bins_off, *d1 = d0 + nbins;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
        const int k = t + T * m;
        float amax = 0.f;
        if (on && k < nbins) {
            const float4 v = frame_bin<F>(mem.sm, k);
            const float2 A = make_float2(v.x, v.y), B = make_float2(v.z, v.w);
            d0[k] = A;
            amax = fabsf(A.x) + fabsf(A.y);
            if (two) {
                d1[k] = B;
                amax = fmaxf(amax, fabsf(B.x) + fabsf(B.y));
            }
        }
        if (bound) {
            // a warp's 32 bins lie in one chunk (chunks of 64 bins or more)
            const unsigned w = __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(amax, 0.f)));
            if ((threadIdx.x & 31) == 0 && w > 0u) atomicMax(ym + (k >> ybd.chunk_log), w);
        }
    }
    if (bound) {
        __syncthreads();
        // the table only grows within a launch, so a block whose maximum does
        // not exceed the value it reads needs no atomic
        if (on) {
            unsigned *row = ybd.max + (long long)cg.cube * ybd.nchunk;
            for (int i = t; i < ybd.nchunk; i += T) {
                const unsigned w = ym[i];
                if (w > *(volatile unsigned *)(row + i)) atomicMax(row + i, w);
            }
        }
    }
}

// Start the copies of the pair's two spectra into its frame (column A at 0, B
// at N/2), past L1 and without registers, so all of them are in flight at
// once; and fetch into L2 what the block `ahead` of this one will read.
template <class F>
__device__ __forceinline__ void frame_fetch(const FrameMem &mem, const ColGroup &cg, bool on,
                                            const float2 *in, int nbins, int t) {
    if (!on) return;
    const float2 *src = in + cg.bins_off;
    const int cols = min(cg.ncol, 2);
    if (((cg.bins_off | nbins) & 1) == 0) {
        for (int c = 0; c < cols; ++c)
            for (int i = t; 2 * i < nbins; i += F::T)
                frame_cp<16>(mem.sm + c * (F::N / 2) + 2 * i, src + (long long)c * nbins + 2 * i);
    } else {
        for (int c = 0; c < cols; ++c)
            for (int i = t; i < nbins; i += F::T)
                frame_cp<8>(mem.sm + c * (F::N / 2) + i, src + (long long)c * nbins + i);
    }
}
__device__ __forceinline__ void prefetch_l2(const void *p, long long bytes) {
    const unsigned long long a = ((unsigned long long)p + 15) & ~15ull;
    const long long n = (bytes - (long long)(a - (unsigned long long)p)) & ~15ll;
    if (n > 0)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(a), "r"((unsigned)n));
}

// Synthesis: fetched bins of the pair's columns -> frame in shared memory
// (natural order, zero beyond the ns resampled samples and either side of
// them).  Thread t's step-1 inputs are bins t + T a and, as
// Z_{N-k} = conj A + i conj B, bins T a - t.
// INTER: the fetched bins of the two columns lie side by side (A at 2k, B at 2k + 1).
template <class F, bool INTER = false>
__device__ __forceinline__ void frame_synthesise(const FrameMem &mem, const ColGroup &cg,
                                                 const float2 *__restrict__ tw, int nbins, int ns,
                                                 int t) {
    constexpr int N = F::N, T = F::T;
    const bool two = cg.ncol > 1;
    const FrameTwiddle ft = frame_twiddle<F>(tw, t);
    frame_cp_wait();             // the spectra, and whatever else the caller staged
    __syncthreads();
    float2 v[16];
#pragma unroll
    for (int a = 0; a < 16; ++a) {
        const int k = a < 8 ? t + T * a : N - t - T * a;       // 0 < k <= N/2 for a >= 8
        float2 A = make_float2(0.f, 0.f), B = A;
        if (k < nbins) {
            A = mem.sm[INTER ? 2 * k : k];
            if (two) B = mem.sm[INTER ? 2 * k + 1 : N / 2 + k];
        }
        if (a == 0 && t == 0) A.y = B.y = 0.f;
        v[a] = a < 8 ? make_float2(A.x - B.y, A.y + B.x) : make_float2(A.x + B.y, B.x - A.y);
    }
    __syncthreads();
    frame_fft<F, true>(v, mem.sm, ft, mem.s_tw, t);
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 16; ++m) {
        const int n = frame_out<F>(m, t);
        mem.sm[frame_at(n)] = n < ns ? v[m] : make_float2(0.f, 0.f);
    }
    if (t < 2) mem.sm[t == 0 ? frame_at(-1) : frame_at(N)] = make_float2(0.f, 0.f);
    __syncthreads();
}

// One resampled row of the synthesised frame.
template <bool TRANS>
__device__ __forceinline__ int2 frame_entry(const DevResampler &rs, int i) {
    return __ldg(reinterpret_cast<const int2 *>(TRANS ? (const void *)(rs.rng + i)
                                                      : (const void *)(rs.pos + i)));
}
template <int INTERP, bool TRANS>
__device__ __forceinline__ float2 frame_row(const FrameMem &mem, const float *__restrict__ frac,
                                            int2 e) {
    float2 s = make_float2(0.f, 0.f);
    if (!TRANS) {
        const float fr = __int_as_float(e.y);
#pragma unroll
        for (int q = 0; q < Taps<INTERP>::n; ++q) {
            const int k = Taps<INTERP>::t0 + q;
            const float w = tap_weight<INTERP>(k, fr);
            const float2 x = mem.sm[frame_at(e.x + k)];
            s.x = fmaf(w, x.x, s.x);
            s.y = fmaf(w, x.y, s.y);
        }
    } else {
        int r = e.x;
#pragma unroll
        for (int q = Taps<INTERP>::n - 1; q >= 0; --q) {
            const int cnt = (e.y >> (8 * q)) & 255;
            for (int j = 0; j < cnt; ++j, ++r) {
                const float w = tap_weight<INTERP>(Taps<INTERP>::t0 + q, __ldg(frac + r));
                const float2 x = mem.sm[frame_at(r)];
                s.x = fmaf(w, x.x, s.x);
                s.y = fmaf(w, x.y, s.y);
            }
        }
    }
    return s;
}

// x = (first column, second column) of a row; a group of one column leaves
// the second alone (its slab or matrix may hold another column there).
__device__ __forceinline__ float2 row_load(const float *p, bool two, bool vec) {
    if (vec && two) return *reinterpret_cast<const float2 *>(p);
    return make_float2(p[0], two ? p[1] : 0.f);
}
__device__ __forceinline__ void row_store(float *p, float2 x, bool two, bool vec) {
    if (vec && two) {
        *reinterpret_cast<float2 *>(p) = x;
        return;
    }
    p[0] = x.x;
    if (two) p[1] = x.y;
}

struct FrameArgs {
    const ColGroup *__restrict__ groups;
    int ngroups;
    DevResampler syn, ana;       // resamplers of the synthesis and the analysis
    int nrows;                   // staged rows (analysis input, or fused middle)
    int nfrac;                   // fractions of the transposed resampler (0: none)
    int ns;                      // stretched samples
    int nbins;
    const float2 *__restrict__ tw;
    const float *__restrict__ frac;   // those fractions
    FrameScatter sc;
    int ahead;                   // blocks resident at once (0: no fetch ahead)
    int seq;                     // pairs an analysis block takes in turn
    FistaArgs fa;
    FrameBound ybd;
};

__device__ __forceinline__ void zero_pads(const FrameMem &mem, int nrows, int t) {
    if (t < 5) mem.stg[t == 0 ? -1 : nrows + t - 1] = make_float2(0.f, 0.f);
}

// FISTA update of one row: m+ = soft(z + gamma g, gamma lambda),
// z+ = m+ + beta (m+ - m).
__device__ __forceinline__ float2 fista_row(const FistaArgs &fa, float2 gt, float2 g, float2 m,
                                            float2 z, float2 *mn) {
    mn->x = soft_threshold(fmaf(gt.x, g.x, z.x), gt.y);
    mn->y = soft_threshold(fmaf(gt.x, g.y, z.y), gt.y);
    return make_float2(fmaf(fa.beta, mn->x - m.x, mn->x), fmaf(fa.beta, mn->y - m.y, mn->y));
}

template <class F>
struct BlockPair {
    int t, pair;
    bool on;
    ColGroup cg;
    __device__ __forceinline__ explicit BlockPair(const FrameArgs &a)
        : t(threadIdx.x % F::T), pair(threadIdx.x / F::T) {
        const int g = blockIdx.x * (blockDim.x / F::T) + pair;
        on = g < a.ngroups;
        cg = a.groups[on ? g : 0];
    }
};

// Resample + FFT (the model's stretch S, or U^T on the data side).  A pair
// is 8 bytes of a row of the row-major input, a quarter of the sector that
// comes with it, so a block of one pair stages the rows of a.seq neighbouring
// pairs together (neighbouring lanes read neighbouring pairs) and transforms
// them in turn.
template <class F, int INTERP, bool TRANS>
__global__ void __launch_bounds__(F::THREADS, F::MINB_ANA)
frame_r2c_kernel(const FrameArgs a, const float *__restrict__ in, float2 *__restrict__ out) {
    extern __shared__ float4 smem_f4[];
    const int t = threadIdx.x % F::T, pair = threadIdx.x / F::T;
    FrameMem mem = frame_mem<F>(smem_f4, pair, a.nrows, a.nfrac);
    const int rows = turn_rows(a.nrows);
    const int g0 = (blockIdx.x * (blockDim.x / F::T) + pair) * a.seq;
    const int lseq = a.seq == 4 ? 2 : a.seq == 2 ? 1 : 0;
    {
        // the pair this thread stages: one of a.seq, the same in every round
        // (T is a multiple of 4)
        const int q = t & (a.seq - 1);
        if (g0 + q < a.ngroups) {
            const ColGroup cg = a.groups[g0 + q];
            const float *src = in + cg.real_off;
            float2 *stg = mem.stg + q * rows;
            const bool two = cg.ncol > 1, vec = ((cg.real_off | cg.ld_real) & 1) == 0;
            if (two && vec)
                for (int r = t >> lseq; r < a.nrows; r += F::T >> lseq)
                    frame_cp<8>(stg + r, src + (long long)r * cg.ld_real);
            else               // odd row length or offset: 4-byte aligned only
                for (int r = t >> lseq; r < a.nrows; r += F::T >> lseq) {
                    const float *x = src + (long long)r * cg.ld_real;
                    frame_cp<4>(&stg[r].x, x);
                    if (two) frame_cp<4>(&stg[r].y, x + 1);
                    else stg[r].y = 0.f;
                }
        }
    }
    for (int q = 0; q < a.seq; ++q) {
        const FrameMem m{mem.s_tw, mem.sfr, mem.sm, mem.stg + q * rows};
        zero_pads(m, a.nrows, t);
    }
    frame_tables<F>(mem.s_tw, a.tw);
    if (TRANS) copy_fractions(mem.sfr, a.frac, a.nfrac);
    frame_cp_wait();
    for (int q = 0; q < a.seq; ++q) {
        __syncthreads();         // rows staged, and the last pair's frame read
        const bool on = g0 + q < a.ngroups;
        const ColGroup cg = a.groups[on ? g0 + q : 0];
        frame_analyse<F, INTERP, TRANS>(mem, cg, on, a.ana, a.sc, a.nrows, a.tw, a.nbins, t, out,
                                        a.ybd);
        mem.stg += rows;
    }
}

// Synthesis + resample with its epilogue: plain store, residual aux - out, or
// the FISTA update.
template <class F, int INTERP, bool TRANS, int EPI>
__global__ void __launch_bounds__(F::THREADS, F::MINB)
frame_c2r_kernel(const FrameArgs a, const float2 *__restrict__ in, float *__restrict__ out,
                 const float *__restrict__ aux) {
    extern __shared__ float4 smem_f4[];
    const BlockPair<F> b(a);
    const FrameMem mem = frame_mem<F>(smem_f4, b.pair, 0, a.nfrac);
    frame_fetch<F>(mem, b.cg, b.on, in, a.nbins, b.t);
    frame_tables<F>(mem.s_tw, a.tw);
    if (threadIdx.x == 0 && a.ahead > 0 && blockIdx.x + a.ahead < gridDim.x)
        prefetch_l2(in + a.groups[blockIdx.x + a.ahead].bins_off,
                    8ll * a.groups[blockIdx.x + a.ahead].ncol * a.nbins);
    frame_synthesise<F>(mem, b.cg, a.tw, a.nbins, a.ns, b.t);
    if (!b.on) return;
    const bool two = b.cg.ncol > 1, vec = ((b.cg.real_off | b.cg.ld_real) & 1) == 0;
    float2 gt = make_float2(a.fa.gamma, a.fa.thresh);
    if (EPI == EPI_FISTA && a.fa.cube_gt) gt = __ldg(a.fa.cube_gt + b.cg.cube);
    // the next row's table entry is loaded while this one is resampled
    int2 nxt = frame_entry<TRANS>(a.syn, min(b.t, a.syn.nrows - 1));
    for (int i = b.t; i < a.syn.nrows; i += F::T) {
        const long long o = b.cg.real_off + (long long)i * b.cg.ld_real;
        const int2 e = nxt;
        nxt = frame_entry<TRANS>(a.syn, min(i + F::T, a.syn.nrows - 1));
        float2 x, z;
        if (EPI == EPI_RESIDUAL) x = row_load(aux + o, two, vec);
        if (EPI == EPI_FISTA) {
            x = row_load(a.fa.m + o, two, vec);
            z = row_load(a.fa.z + o, two, vec);
        }
        const float2 g = frame_row<INTERP, TRANS>(mem, a.frac, e);
        if (EPI == EPI_STORE) {
            row_store(out + o, g, two, vec);
        } else if (EPI == EPI_RESIDUAL) {
            row_store(out + o, make_float2(x.x - g.x, x.y - g.y), two, vec);
        } else {
            float2 mn;
            const float2 zn = fista_row(a.fa, gt, g, x, z, &mn);
            row_store(a.fa.m + o, mn, two, vec);
            row_store(a.fa.z + o, zn, two, vec);
        }
    }
}

// One FISTA half-iteration's two time stages, fused (data side: U H, residual,
// U^T F; model side: S^T H, update, S F of the new z), in place on the
// spectrum; the real rows are the solver's column-blocked state (a pair's
// rows are one slab of float2).
template <class F, int INTERP, bool SYN_TRANS, int EPI>
__global__ void __launch_bounds__(F::THREADS, F::MINB)
frame_fused_kernel(const FrameArgs a, float2 *spec, const float *__restrict__ aux) {
    extern __shared__ float4 smem_f4[];
    const BlockPair<F> b(a);
    const FrameMem mem = frame_mem<F>(smem_f4, b.pair, a.nrows, a.nfrac);
    const bool two = b.cg.ncol > 1;
    frame_fetch<F>(mem, b.cg, b.on, spec, a.nbins, b.t);
    // the epilogue's state rows (d, or z) arrive while the spectrum is transformed
    const float2 *state =
        reinterpret_cast<const float2 *>((EPI == EPI_RESIDUAL ? aux : a.fa.z) + b.cg.real_off);
    if (b.on)
        for (int i = b.t; i < a.nrows; i += F::T) frame_cp<8>(mem.stg + i, state + i);
    if (!SYN_TRANS) copy_fractions(mem.sfr, a.frac, a.nfrac);
    frame_tables<F>(mem.s_tw, a.tw);
    zero_pads(mem, a.nrows, b.t);
    if (threadIdx.x < 3 && a.ahead > 0 && blockIdx.x + a.ahead < gridDim.x) {
        const ColGroup n = a.groups[blockIdx.x + a.ahead];
        if (threadIdx.x == 0) prefetch_l2(spec + n.bins_off, 8ll * n.ncol * a.nbins);
        else if (threadIdx.x == 1)
            prefetch_l2((EPI == EPI_RESIDUAL ? aux : a.fa.z) + n.real_off, 8ll * a.nrows);
        else if (EPI == EPI_FISTA) prefetch_l2(a.fa.m + n.real_off, 8ll * a.nrows);
    }
    frame_synthesise<F>(mem, b.cg, a.tw, a.nbins, a.ns, b.t);
    // each thread rewrites the rows it copied itself
    float2 gt = make_float2(a.fa.gamma, a.fa.thresh);
    if (EPI == EPI_FISTA && a.fa.cube_gt) gt = __ldg(a.fa.cube_gt + b.cg.cube);
    float2 *mrow = reinterpret_cast<float2 *>(a.fa.m + b.cg.real_off);
    float2 *zrow = reinterpret_cast<float2 *>(a.fa.z + b.cg.real_off);
    // the next row's table entry and m are loaded while this one is resampled
    const int last = a.nrows - 1;
    int2 nxt = frame_entry<SYN_TRANS>(a.syn, min(b.t, last));
    float2 mnxt = make_float2(0.f, 0.f);
    if (EPI == EPI_FISTA) mnxt = mrow[min(b.t, last)];
    for (int i = b.t; i < a.nrows; i += F::T) {
        const int2 e = nxt;
        const float2 m = mnxt;
        nxt = frame_entry<SYN_TRANS>(a.syn, min(i + F::T, last));
        if (EPI == EPI_FISTA) mnxt = mrow[min(i + F::T, last)];
        const float2 g = frame_row<INTERP, SYN_TRANS>(mem, a.frac, e);
        const float2 s = mem.stg[i];
        float2 x;
        if (EPI == EPI_RESIDUAL) {
            x = make_float2(s.x - g.x, s.y - g.y);
        } else {
            float2 mn;
            x = fista_row(a.fa, gt, g, m, s, &mn);
            if (b.on) {
                row_store(reinterpret_cast<float *>(mrow + i), mn, two, true);
                row_store(reinterpret_cast<float *>(zrow + i), x, two, true);
            }
        }
        if (!two) x.y = 0.f;
        mem.stg[i] = x;
    }
    __syncthreads();
    frame_analyse<F, INTERP, !SYN_TRANS>(mem, b.cg, b.on, a.ana, a.sc, a.nrows, a.tw, a.nbins,
                                          b.t, spec, a.ybd);
}

// ---------------------------------------------------- gathers fastest
// Plans whose spectra and rows hold the gathers fastest (the tensor-core
// plans): a row, or a bin, of neighbouring pairs is contiguous.  A block owns
// 256 / T neighbouring pairs, at least two (a bin of two pairs is a whole
// sector); they are transformed each by its own T threads, and moved by all
// threads with the pair fastest, so every access is a run of the block's pairs.
template <class F>
struct GatherBlock {
    static constexpr int PB = F::T >= 256 ? 2 : 256 / F::T;
    static constexpr int THREADS = PB * F::T;
    static constexpr int MINB = THREADS == 256 ? 4 : THREADS == 512 ? 2 : 1;
    static constexpr int MINB_ANA = THREADS == 256 ? 3 : THREADS == 512 ? 2 : 1;
    int t, pair;             // this thread's transform
    int io, row0;            // the pair it moves, and its first row or bin (steps of T)
    bool on, io_on;
    ColGroup cg, iog;
    FrameMem mem, iom;
    __device__ __forceinline__ GatherBlock(const FrameArgs &a, float4 *base, int nrows)
        : t(threadIdx.x % F::T), pair(threadIdx.x / F::T), io(threadIdx.x % PB),
          row0(threadIdx.x / PB) {
        const int g = blockIdx.x * PB;
        on = g + pair < a.ngroups;
        io_on = g + io < a.ngroups;
        cg = a.groups[on ? g + pair : 0];
        iog = a.groups[io_on ? g + io : 0];
        mem = frame_mem<F>(base, pair, nrows, a.nfrac);
        iom = frame_mem<F>(base, io, nrows, a.nfrac);
    }
};

template <class F, int INTERP, bool TRANS>
__global__ void __launch_bounds__(GatherBlock<F>::THREADS, GatherBlock<F>::MINB_ANA)
gather_r2c_kernel(const FrameArgs a, const float *__restrict__ in, float2 *__restrict__ out) {
    extern __shared__ float4 smem_f4[];
    const GatherBlock<F> b(a, smem_f4, a.nrows);
    const ColGroup &cg = b.iog;
    const bool two = cg.ncol > 1;
    if (b.io_on) {
        const float *src = in + cg.real_off;
        const bool vec = two && ((cg.real_off | cg.ld_real) & 1) == 0;
        for (int r = b.row0; r < a.nrows; r += F::T) {
            const float *x = src + (long long)r * cg.ld_real;
            float2 *dst = b.iom.stg + r;
            if (vec) {
                frame_cp<8>(dst, x);
            } else {
                frame_cp<4>(&dst->x, x);
                if (two) frame_cp<4>(&dst->y, x + 1);
                else dst->y = 0.f;
            }
        }
    }
    zero_pads(b.mem, a.nrows, b.t);
    frame_tables<F>(b.mem.s_tw, a.tw);
    if (TRANS) copy_fractions(b.mem.sfr, a.frac, a.nfrac);
    frame_cp_wait();
    __syncthreads();
    frame_spectrum<F, INTERP, TRANS>(b.mem, a.ana, a.sc, a.nrows, a.tw, b.t, [] {});
    if (!b.io_on) return;
    float2 *dst = out + cg.spec_off;
    const bool vec = two && ((cg.spec_off | cg.ld_spec) & 1) == 0;
    for (int k = b.row0; k < a.nbins; k += F::T) {
        const float4 v = frame_bin<F>(b.iom.sm, k);
        float2 *d = dst + (long long)k * cg.ld_spec;
        if (vec) {
            *reinterpret_cast<float4 *>(d) = v;
        } else {
            d[0] = make_float2(v.x, v.y);
            if (two) d[1] = make_float2(v.z, v.w);
        }
    }
}

template <class F, int INTERP, bool TRANS, int EPI>
__global__ void __launch_bounds__(GatherBlock<F>::THREADS, GatherBlock<F>::MINB)
gather_c2r_kernel(const FrameArgs a, const float2 *__restrict__ in, float *__restrict__ out,
                  const float *__restrict__ aux) {
    extern __shared__ float4 smem_f4[];
    const GatherBlock<F> b(a, smem_f4, 0);
    const ColGroup &cg = b.iog;
    const bool two = cg.ncol > 1;
    if (b.io_on) {
        const float2 *src = in + cg.spec_off;
        const bool vec = two && ((cg.spec_off | cg.ld_spec) & 1) == 0;
        for (int k = b.row0; k < a.nbins; k += F::T) {
            const float2 *x = src + (long long)k * cg.ld_spec;
            float2 *dst = b.iom.sm + 2 * k;
            if (vec) {
                frame_cp<16>(dst, x);
            } else {
                frame_cp<8>(dst, x);
                if (two) frame_cp<8>(dst + 1, x + 1);
            }
        }
    }
    frame_tables<F>(b.mem.s_tw, a.tw);
    frame_synthesise<F, true>(b.mem, b.cg, a.tw, a.nbins, a.ns, b.t);
    if (!b.io_on) return;
    const bool vec = ((cg.real_off | cg.ld_real) & 1) == 0;
    const int last = a.syn.nrows - 1;
    int2 nxt = frame_entry<TRANS>(a.syn, min(b.row0, last));
    for (int i = b.row0; i < a.syn.nrows; i += F::T) {
        const long long o = cg.real_off + (long long)i * cg.ld_real;
        const int2 e = nxt;
        nxt = frame_entry<TRANS>(a.syn, min(i + F::T, last));
        float2 x;
        if (EPI == EPI_RESIDUAL) x = row_load(aux + o, two, vec);
        float2 g = frame_row<INTERP, TRANS>(b.iom, a.frac, e);
        if (EPI == EPI_RESIDUAL) g = make_float2(x.x - g.x, x.y - g.y);
        row_store(out + o, g, two, vec);
    }
}

}  // namespace aahrt
