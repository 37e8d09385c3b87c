// Curvature-range tools of Sec. 3.5 (eqs. q1-q3): the uniform-slowness
// curvature axis, the sample-count bound of eq. q3, and the partial NMO of
// the data by a reference curvature.
//
// Partial NMO.  In stretched time s = t^2 a hyperbola t^2 = tau^2 + q r^2 is
// the line s = tau^2 + q r^2; shifting the stretched trace by -q_ref r^2
// moves it to curvature q - q_ref.  On the time axis that is one resampling:
//   out(t_i, h) = sum_taps c(u - n) in(t_n, h),  u^2 = i^2 + q_ref r_h^2/dt^2,
// zero where u^2 < 0.  u is evaluated in float-float arithmetic: i^2 and
// c_h = q_ref r_h^2/dt^2 are exact (hi, lo) pairs, the sum is a two-sum, and
// one Newton step on the FP32 root recovers the fraction of a sample to about
// 1e-7 (a plain FP32 u of 1000 samples would lose 6e-5 of a sample).  The
// transpose gathers, for every input sample n, the outputs i whose taps reach
// n (recomputing their positions and weights bit-identically), so it needs no
// atomics and is deterministic.
#include <algorithm>
#include <cmath>

#include "internal.cuh"
#include "resample.cuh"

namespace aahrt {

struct PnArgs {
    const PnBlock *__restrict__ blk;
    const double *__restrict__ rho;   // per trace r^2 / dt^2
    double q_ref;
    int nt;
};

constexpr int kPnRows = 8;            // rows a thread takes of its column
constexpr int kPnCols = 8;            // columns of a block of the transpose

// Forward: one thread owns kPnRows neighbouring rows of a column, so the
// column's coefficient q_ref r^2/dt^2, as (hi, lo), is formed once and no index
// is divided (a flat index cost a 64-bit division a sample, and the
// coefficients a launch of their own: 29 us a call of a 2000-trace, 1001-sample
// gather, 21 now).  The transpose evaluates five or six positions a sample, so
// the coefficient is a small part and the serial chain is what counts: one row
// a thread, in blocks of kPnCols columns x 16 rows.  Per call, flat index /
// eight rows a thread / 32 columns / 16 / 8: 256 traces x 256 samples 23 / 100 /
// 19 / 20 / 19 us, the gather 103 / 183 / 89 / 85 / 80, 16 cubes of 200-3000
// traces 1002 / 1054 / 1014 / 958 / 906, 256 cubes of 33 traces x 100 samples
// 33 / 62 / 39 / 35 / 33, 8000 traces x 2048 samples 928 / 764 / 764 / 694 / 633.
__device__ __forceinline__ float2 pn_coef(const PnArgs &a, const PnBlock &b, int col) {
    const double v = a.q_ref * __ldg(a.rho + b.r0 + col / b.rep);
    const float hi = (float)v;
    return make_float2(hi, (float)(v - (double)hi));
}

// Position u = sqrt(i^2 + c) of output row i as base + frac, frac in [0, 1);
// false where i^2 + c < 0 (the output is muted), or where u is beyond every
// record (nt < 46341) or not a number (c past the float range), so that base
// stays far from the ends of the integers.
__device__ __forceinline__ bool pn_position(int i, float2 c, int *base, float *frac) {
    const int ii = i * i;
    const float a_hi = __int2float_rn(ii);
    const float a_lo = __int2float_rn(ii - __float2int_rn(a_hi));
    const float s = __fadd_rn(a_hi, c.x);                 // two-sum of a_hi + c.x
    const float bb = __fsub_rn(s, a_hi);
    const float err = __fadd_rn(__fsub_rn(a_hi, __fsub_rn(s, bb)), __fsub_rn(c.x, bb));
    const float t = __fadd_rn(__fadd_rn(err, a_lo), c.y);
    const float u2 = __fadd_rn(s, t);
    if (!(u2 >= 0.f && u2 < 4294967296.f)) return false;
    const float u0 = sqrtf(fmaxf(s, 0.f));
    float corr = 0.f;
    if (u0 > 0.f) corr = __fadd_rn(__fmaf_rn(-u0, u0, s), t) / __fmul_rn(2.f, u0);
    const float fb = floorf(u0);
    float fr = __fadd_rn(__fsub_rn(u0, fb), corr);
    int b = (int)fb;
    if (fr < 0.f) {
        fr = __fadd_rn(fr, 1.f);
        --b;
    } else if (fr >= 1.f) {
        fr = __fsub_rn(fr, 1.f);
        ++b;
    }
    if (fr >= 1.f) fr = 0.99999994f;
    *base = b;
    *frac = fr;
    return true;
}

template <int INTERP>
__global__ void __launch_bounds__(128)
pnmo_kernel(const PnArgs a, const float *__restrict__ in, float *__restrict__ out) {
    const PnBlock b = a.blk[blockIdx.z];
    const int col = blockIdx.x * blockDim.x + threadIdx.x;
    if (col >= b.ld) return;
    const float2 c = pn_coef(a, b, col);
    const int i1 = min(a.nt, kPnRows * (int)(blockIdx.y + 1));
    for (int i = kPnRows * blockIdx.y; i < i1; ++i) {
        int base;
        float fr;
        float v = 0.f;
        if (pn_position(i, c, &base, &fr)) {
#pragma unroll
            for (int q = 0; q < Taps<INTERP>::n; ++q) {
                const int t = Taps<INTERP>::t0 + q;
                const int r = base + t;
                if (r >= 0 && r < a.nt)
                    v = fmaf(tap_weight<INTERP>(t, fr),
                             __ldg(in + b.off + (long long)r * b.ld + col), v);
            }
        }
        out[b.off + (long long)i * b.ld + col] = v;
    }
}

// largest i >= 0 with i^2 <= x (x may be negative: -1), by a float root and
// integer corrections; beyond 46341^2 (nt is below 46341) some i > nt, since a
// root past the 32-bit range would leave the corrections without an end
__device__ __forceinline__ int isqrt_floor(float x) {
    if (x < 0.f) return -1;
    x = fminf(x, 2147580964.f);          // 46342^2
    int r = (int)sqrtf(x);
    while ((float)r * r > x) --r;
    while ((float)(r + 1) * (r + 1) <= x) ++r;
    return r;
}

template <int INTERP>
__global__ void __launch_bounds__(128)
pnmo_t_kernel(const PnArgs a, const float *__restrict__ in, float *__restrict__ out) {
    constexpr int T0 = Taps<INTERP>::t0, TN = Taps<INTERP>::n;
    const PnBlock b = a.blk[blockIdx.z];
    const int col = blockIdx.x * kPnCols + threadIdx.x % kPnCols;
    const int r = blockIdx.y * (128 / kPnCols) + threadIdx.x / kPnCols;   // sample receiving
    if (col >= b.ld || r >= a.nt) return;
    const float2 c = pn_coef(a, b, col);
    const float cc = c.x + c.y;
    // outputs i read sample r when base_i + t = r for a tap t, i.e.
    // u_i in [r - T0 - TN + 1, r - T0 + 1); one sample of margin each side
    const float ulo = fmaxf((float)(r - T0 - TN), 0.f);
    const float uhi = (float)(r - T0 + 2);
    int ilo = isqrt_floor(ulo * ulo - cc) - 1;
    int ihi = isqrt_floor(uhi * uhi - cc) + 1;
    if (ilo < 0) ilo = 0;
    if (ihi > a.nt - 1) ihi = a.nt - 1;
    float v = 0.f;
    for (int i = ilo; i <= ihi; ++i) {
        int base;
        float fr;
        if (!pn_position(i, c, &base, &fr)) continue;
        const int t = r - base;
        if (t < T0 || t >= T0 + TN) continue;
        v = fmaf(tap_weight<INTERP>(t, fr), __ldg(in + b.off + (long long)i * b.ld + col), v);
    }
    out[b.off + (long long)r * b.ld + col] = v;
}

}  // namespace aahrt

using namespace aahrt;

extern "C" int aahrt_q_axis_slowness(double pmin, double pmax, int nq, double *q) {
    if (!q) return set_error(AAHRT_ERR_INVALID_ARG, "q is NULL");
    if (nq < 1) return set_error(AAHRT_ERR_INVALID_ARG, "nq must be >= 1");
    if (!std::isfinite(pmin) || !std::isfinite(pmax))
        return set_error(AAHRT_ERR_NONFINITE, "pmin and pmax must be finite");
    const double step = nq > 1 ? (pmax - pmin) / (nq - 1) : 0.0;
    for (int l = 0; l < nq; ++l) {
        const double p = (nq > 1 && l == nq - 1) ? pmax : pmin + l * step;
        q[l] = p * p;
    }
    return AAHRT_OK;
}

extern "C" int aahrt_nq_required(double span, double fmax, double r2max, int *nq) {
    if (!nq) return set_error(AAHRT_ERR_INVALID_ARG, "nq is NULL");
    if (!std::isfinite(span) || !std::isfinite(fmax) || !std::isfinite(r2max))
        return set_error(AAHRT_ERR_NONFINITE, "span, fmax and r2max must be finite");
    if (span < 0.0 || fmax < 0.0 || r2max < 0.0)
        return set_error(AAHRT_ERR_INVALID_ARG, "span, fmax and r2max must be >= 0");
    const double n = std::ceil(span * fmax * r2max - 1e-12);
    if (!(n < 2147483647.0)) return set_error(AAHRT_ERR_INVALID_ARG, "sample count overflows");
    *nq = n < 1.0 ? 1 : (int)n;
    return AAHRT_OK;
}

extern "C" int aahrt_partial_nmo(aahrt_plan *plan, const float *in, float *out, double q_ref,
                                 int transpose, void *stream) {
    if (!plan) return set_error(AAHRT_ERR_INVALID_ARG, "plan is NULL");
    Plan &p = *plan->p;
    DeviceGuard g(p.device);
    int rc;
    if ((rc = check_dev_ptr(in, "in")) || (rc = check_dev_ptr(out, "out"))) return rc;
    if (transpose != 0 && transpose != 1)
        return set_error(AAHRT_ERR_INVALID_ARG, "transpose must be 0 or 1");
    if (!std::isfinite(q_ref)) return set_error(AAHRT_ERR_NONFINITE, "q_ref must be finite");
    const char *a0 = reinterpret_cast<const char *>(in), *b0 = reinterpret_cast<const char *>(out);
    const long long bytes = p.data_len * (long long)sizeof(float);
    if (a0 < b0 + bytes && b0 < a0 + bytes)
        return set_error(AAHRT_ERR_INVALID_ARG, "in and out overlap");
    if (p.nt >= 46341)
        return set_error(AAHRT_ERR_UNSUPPORTED, "nt too large for the partial NMO");
    cudaStream_t st = (cudaStream_t)stream;
    const PnArgs a{p.pn_blk, p.pn_rho, q_ref, p.nt};
    // (eight rows a thread pay for its coefficient and still give 2000 blocks
    // from one 2000-trace gather; the transpose takes one row a thread)
    const int cols = transpose ? kPnCols : 128, rows = transpose ? 128 / kPnCols : kPnRows;
    const dim3 grid((unsigned)((p.pn_ldmax + cols - 1) / cols),
                    (unsigned)((p.nt + rows - 1) / rows), (unsigned)p.pn_nblk);
    const bool keys = p.interp == AAHRT_INTERP_KEYS;
    if (transpose) {
        if (keys) pnmo_t_kernel<AAHRT_INTERP_KEYS><<<grid, 128, 0, st>>>(a, in, out);
        else pnmo_t_kernel<AAHRT_INTERP_LINEAR><<<grid, 128, 0, st>>>(a, in, out);
    } else {
        if (keys) pnmo_kernel<AAHRT_INTERP_KEYS><<<grid, 128, 0, st>>>(a, in, out);
        else pnmo_kernel<AAHRT_INTERP_LINEAR><<<grid, 128, 0, st>>>(a, in, out);
    }
    p.launches[6] += 1;
    const cudaError_t e = cudaGetLastError();
    return e ? cuda_fail(e, "partial NMO launch") : AAHRT_OK;
}
