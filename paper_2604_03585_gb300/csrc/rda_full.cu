// Full Range-Doppler processing with range cell migration correction
// (Sec. IV-A steps 2-4 of the paper: azimuth FFT, RCMC by sinc
// interpolation, azimuth compression with the range-dependent filter
// H_a(f_a, R0), azimuth IFFT).
//
// Geometry (normalised, see sar_plan_set_geometry): a target of closest range
// r0 (in range samples) appears in the range-Doppler domain at r0 / D(f),
// D(f) = sqrt(1 - (f / (kappa v_s))^2), with spectrum phase
// exp(-2 pi i kappa r0 D(f)).  RCMC reads output bin n at frequency f from
// the input at n + (r_near + n)(1/D(f) - 1) through a 16-tap Hann-windowed
// sinc; azimuth compression multiplies by exp(+2 pi i kappa r D(f)),
// r = r_near + n, and applies the inverse FFT (1/N).
//
// Per azimuth frequency index j the plan keeps, computed in FP64 on the host
// and rounded: kappa D(f_j) and 1/D(f_j) - 1, each as an unevaluated float sum
// (hi + lo).  The phase kappa r D of a sample (up to ~1e5 cycles) and the
// migration r (1/D - 1) (up to ~1e2 samples) are then formed in FP32 with an
// exact two-product, so only their fractional parts are rounded; the integer
// range bin n never enters a rounded sum (at n ~ 8000 the FP32 spacing is
// 1e-3 samples, which would cost ~1e-3 relative error on a half-band signal).
#include <type_traits>

#include "../../include/sar.h"
#include "launch_behind.h"
#include "streamed.cuh"
#include "registry.h"
#include "tables.h"

namespace sar {

struct RdColumn {
    float a_hi, a_lo;       // kappa D(f_j) = a_hi + a_lo
    float mig_hi, mig_lo;   // 1 / D(f_j) - 1 = mig_hi + mig_lo
};

// The interpolation weights h(x) = sinc(x) (1 + cos(2 pi x / 16)) / 2 at the 16
// taps t = -7 ... 8 of a source position k0 + frac, as polynomials in u = frac -
// 1/2.  h is even, so taps t and 1 - t are h(u + 1/2 - t) = E_t(u^2) + u
// O_t(u^2) and E_t(u^2) - u O_t(u^2): ten fused multiply-adds give both.  E_t
// and O_t are interpolated in v = u^2 at five Chebyshev points of [0, 1/4]
// (Newton's divided differences, expanded), at compile time in FP64: the
// largest error of a weight is 1.2e-9, and 9e-8 in FP32 arithmetic, all of it
// rounding, with an RMS of 2.5e-8 at the central taps and below 1e-8 beyond.
namespace rcw {
// a * b + c, two-wide: one packed instruction, each half rounded as fmaf
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(f2_pack(a)), "l"(f2_pack(b)), "l"(f2_pack(c)));
    return f2_unpack(r);
}
constexpr int K = 5;
__host__ __device__ constexpr double weight(double x) {
    const double ax = x < 0 ? -x : x;
    const double turns = ax * 0.5 - (double)(long long)(ax * 0.5);   // of pi x
    const double sinc = ax == 0 ? 1.0 : ct::sin2pi_f(turns) / (ct::kPi * ax);
    return sinc * 0.5 * (1.0 + ct::cos2pi_f(ax / 16.0));
}
struct Poly {
    double c[K];   // of v^0 ... v^4
};
// ODD: O_t, else E_t
__host__ __device__ constexpr Poly fit(int t, bool odd) {
    double v[K] = {}, d[K] = {};
    for (int i = 0; i < K; ++i) {
        const double u = 0.5 * ct::cos2pi_f((2 * i + 1) / (8.0 * K));
        const double p = weight(u + 0.5 - t), m = weight(-u + 0.5 - t);
        v[i] = u * u;
        d[i] = odd ? (p - m) / (2.0 * u) : (p + m) * 0.5;
    }
    for (int k = 1; k < K; ++k)
        for (int i = K - 1; i >= k; --i) d[i] = (d[i] - d[i - 1]) / (v[i] - v[i - k]);
    Poly r = {};
    for (int k = K - 1; k >= 0; --k) {   // r <- r (x - v[k]) + d[k]
        for (int i = K - 1; i > 0; --i) r.c[i] = r.c[i - 1] - v[k] * r.c[i];
        r.c[0] = d[k] - v[k] * r.c[0];
    }
    return r;
}
// the polynomial at two v by Horner's rule
template <int T, bool ODD>
__device__ __forceinline__ float2 at(float2 v) {
    constexpr Poly p = fit(T, ODD);
    float2 r = make_float2((float)p.c[K - 1], (float)p.c[K - 1]);
#pragma unroll
    for (int i = K - 2; i >= 0; --i) r = fma2(r, v, make_float2((float)p.c[i], (float)p.c[i]));
    return r;
}
}  // namespace rcw

// RCMC tiles: 32 frequency columns (one per lane) x 128 range bins per block of
// 8 warps.  A block stages the input rows its outputs touch in shared memory
// (rows n0 + min shift - 7 ... n0 + 127 + max shift + 8, zero outside the
// scene); the host sizes that span from the geometry, and a block whose span
// does not fit reads global memory directly.
// Bound by ALU issue: 177 thread instructions per output (223 with the weights
// from reciprocals and sines; the floor of the 4096 x 4096 scene's 268 MB is 40
// us, of its instructions 74).  102.8 us at 4096 x 4096, from 122.5: polynomial
// weights for two outputs at once 105.0 (one at a time 123.5, four 108.8, with
// the coefficients in constant memory 144), rows staged by asynchronous copies
// 102.8.  Tiles of 64 and 256 bins: 107.9 and 106.6.
constexpr int kRcCols = 32;
constexpr int kRcRows = 128;
constexpr int kRcWarps = 8;
constexpr int kRcMaxStaged = 384;   // 96 KB of staged rows per block

// Source position of output bin n in column c: k0 + frac, frac in [0, 1), for
// r = r_near + n with r_near = rn_hi + rn_lo.  r is formed by a two-sum and the
// shift r (1/D - 1) by a two-product, so only the fractional part is rounded.
__device__ __forceinline__ void rc_locate(int n, const RdColumn& c, float rn_hi, float rn_lo, int& k0, float& frac) {
    const float nf = (float)n;
    const float r_hi = rn_hi + nf;                       // two-sum of rn_hi and n
    const float bb = r_hi - rn_hi;
    const float r_lo = ((rn_hi - (r_hi - bb)) + (nf - bb)) + rn_lo;
    const float p = __fmul_rn(r_hi, c.mig_hi);            // never contracted into the next subtraction
    const float e = fmaf(r_hi, c.mig_hi, -p);             // exact error of the product
    const float fl = floorf(p);
    frac = (p - fl) + (e + fmaf(r_hi, c.mig_lo, r_lo * c.mig_hi));   // p - fl is exact
    k0 = n + (int)fl;
    if (frac < 0.f) { frac += 1.f; k0 -= 1; }
    if (frac >= 1.f) { frac -= 1.f; k0 += 1; }
}

// The 16 taps at kRcWide source positions k0 + frac[j], rows of position j read
// through row(j, t) for t = -7 ... 8, outer pairs first.  Positions go through
// the polynomials together, two to a packed instruction, because every
// coefficient costs a move into a register pair whatever uses it.
constexpr int kRcWide = 2;
template <int T, class Row>
__device__ __forceinline__ void rc_pairs(const float2 (&u)[kRcWide / 2], const float2 (&v)[kRcWide / 2],
                                         float2 (&acc)[kRcWide], Row& row) {
    float2 h[kRcWide / 2][2];
#pragma unroll
    for (int i = 0; i < kRcWide / 2; ++i) {
        const float2 e = rcw::at<T, false>(v[i]), o = rcw::at<T, true>(v[i]);
        h[i][0] = rcw::fma2(u[i], o, e);
        h[i][1] = rcw::fma2(make_float2(-u[i].x, -u[i].y), o, e);
    }
#pragma unroll
    for (int j = 0; j < kRcWide; ++j) {
        const float h1 = j & 1 ? h[j / 2][0].y : h[j / 2][0].x, h2 = j & 1 ? h[j / 2][1].y : h[j / 2][1].x;
        const float2 v1 = row(j, T), v2 = row(j, 1 - T);
        acc[j].x = fmaf(h1, v1.x, acc[j].x);
        acc[j].y = fmaf(h1, v1.y, acc[j].y);
        acc[j].x = fmaf(h2, v2.x, acc[j].x);
        acc[j].y = fmaf(h2, v2.y, acc[j].y);
    }
    if constexpr (T < 0) rc_pairs<T + 1>(u, v, acc, row);
}
template <class Row>
__device__ __forceinline__ void rc_interp(const float (&frac)[kRcWide], float2 (&acc)[kRcWide], Row row) {
    float2 u[kRcWide / 2], v[kRcWide / 2];
#pragma unroll
    for (int i = 0; i < kRcWide / 2; ++i) {
        u[i] = make_float2(frac[2 * i] - 0.5f, frac[2 * i + 1] - 0.5f);
        v[i] = make_float2(u[i].x * u[i].x, u[i].y * u[i].y);
    }
#pragma unroll
    for (int j = 0; j < kRcWide; ++j) acc[j] = make_float2(0.f, 0.f);
    rc_pairs<-7>(u, v, acc, row);
#pragma unroll
    for (int j = 0; j < kRcWide; ++j)
        if (frac[j] == 0.f) acc[j] = row(j, 0);   // h_0 = 1, every other tap sits on a zero of the sinc
}

__global__ void __launch_bounds__(kRcCols * kRcWarps)
rcmc_tile_kernel(const float2* in, float2* __restrict__ out, int n_range, int n_f,
                 const RdColumn* __restrict__ cols, float rn_hi, float rn_lo, int staged_rows) {
    extern __shared__ float2 tile[];   // [staged_rows][32]
    grid_wait_predecessor();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // tiles of one range of bins are neighbours, as their rows are
    const int tiles_f = (n_f + kRcCols - 1) / kRcCols;
    const int j = (int)(blockIdx.x % tiles_f) * kRcCols + lane;
    const int n0 = (int)(blockIdx.x / tiles_f) * kRcRows;
    const int n1 = min(n0 + kRcRows, n_range) - 1;
    const bool jok = j < n_f;
    const RdColumn c = cols[jok ? j : n_f - 1];
    // the rows this block reads: the same positions every output computes, so
    // every warp finds the same span
    int k_first, k_last;
    float f_unused;
    rc_locate(n0, c, rn_hi, rn_lo, k_first, f_unused);
    rc_locate(n1, c, rn_hi, rn_lo, k_last, f_unused);
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        k_first = min(k_first, __shfl_xor_sync(0xffffffffu, k_first, o));
        k_last = max(k_last, __shfl_xor_sync(0xffffffffu, k_last, o));
    }
    const int lo = k_first - 7, hi = k_last + 8;
    const int span = hi - lo + 1;
    const bool staged = span <= staged_rows;
    if (staged) {
        // copied without a stop in registers, all of a thread's rows in flight
        // (src size 0: zeros outside the scene)
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(tile) + lane * 8;
#pragma unroll 4
        for (int rr = warp; rr < span; rr += kRcWarps) {
            const int k = lo + rr;
            const bool inside = jok && k >= 0 && k < n_range;
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst + rr * (kRcCols * 8)),
                         "l"(in + (inside ? (int64_t)k * n_f + j : 0)), "r"(inside ? 8 : 0)
                         : "memory");
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
    }
    if (!jok) return;
    for (int n = n0 + warp; n <= n1; n += kRcWide * kRcWarps) {
        int k0[kRcWide];
        float frac[kRcWide];
        float2 y[kRcWide];
#pragma unroll
        for (int i = 0; i < kRcWide; ++i) rc_locate(min(n + i * kRcWarps, n1), c, rn_hi, rn_lo, k0[i], frac[i]);
        if (staged) {
            const float2* b[kRcWide];
#pragma unroll
            for (int i = 0; i < kRcWide; ++i)   // already within; keeps every read inside the tile
                b[i] = tile + (min(max(k0[i], lo + 7), hi - 8) - lo) * kRcCols + lane;
            rc_interp(frac, y, [&](int i, int t) { return b[i][t * kRcCols]; });
        } else {
            rc_interp(frac, y, [&](int i, int t) {
                const int k = k0[i] + t;
                return (k >= 0 && k < n_range) ? in[(int64_t)k * n_f + j] : make_float2(0.f, 0.f);
            });
        }
#pragma unroll
        for (int i = 0; i < kRcWide; ++i)
            if (n + i * kRcWarps <= n1) __stcs(out + (int64_t)(n + i * kRcWarps) * n_f + j, y[i]);
    }
}

// The azimuth kernels of the full processor in group-streamed form: the passes
// before the last run one radix group at a time (R values live, the next
// group's loads in flight during the current group's arithmetic); the last
// pass keeps the line in registers for the scatter to natural order through
// shared memory and the coalesced store.  COMPRESS (range bin `line`,
// r = r_near + line): every sample j is first multiplied by
// exp(+2 pi i frac(kappa r D(f_j))) -- the phase of up to ~1e5 cycles formed
// by an FP32 two-product of r with kappa D(f_j) held as hi + lo, so that only
// its fractional part is rounded -- and conjugated, and the store conjugates
// and scales by 1/N: the inverse FFT of the filtered line through
// conj(FFT(conj .)) (Sec. II-C).  Otherwise the forward FFT of the line (the
// Range-Doppler domain, Sec. IV-A step 2).
// 16384 samples run their passes over the whole line: warp-local the two kernels
// spill under the 128 registers of a 512-thread block (16384 azimuth lines of 512 /
// 2048 range bins, whole processor: 204 / 746 us against 229 / 826).
template <class SC_, bool COMPRESS>
__global__ void __launch_bounds__(SC_::T, SC_::T >= 256 ? min_blocks_128<SC_, 1>() : 0)
az_streamed_kernel(const float2* in, float2* out, int64_t n_lines, const float2* tw, const RdColumn* cols,
                   double r_near) {
    using SC = std::conditional_t<SC_::N == 16384, LineWide<SC_>, SC_>;
    extern __shared__ float2 smem_dyn[];
    grid_wait_predecessor();
    const int t = threadIdx.x;
    const int64_t line = blockIdx.x;
    if (line >= n_lines) return;
    float2* sm = smem_dyn;
    constexpr int R1 = SC::R1, S1 = SC::S1, G1 = SC::E / R1, RL = SC::RL, GL = SC::E / RL;
    const float2* src = in + line * SC::N;
    float r_hi = 0.f, r_lo = 0.f;
    if constexpr (COMPRESS) {
        const double rd = r_near + (double)line;
        r_hi = (float)rd;
        r_lo = (float)(rd - (double)r_hi);
    }
    auto sample = [&](int j) -> float2 {
        float2 x = __ldcs(src + j);
        if constexpr (COMPRESS) {
            const RdColumn c = cols[j];
            const float p = __fmul_rn(r_hi, c.a_hi);   // never contracted into p - rint(p)
            const float e = fmaf(r_hi, c.a_hi, -p);    // exact error of the product
            const float frac = (p - rintf(p)) + (e + fmaf(r_hi, c.a_lo, r_lo * c.a_hi));
            float sn, cs;
            sincospif(2.f * frac, &sn, &cs);
            x = cconj(make_float2(fmaf(x.x, cs, -x.y * sn), fmaf(x.x, sn, x.y * cs)));
        }
        return x;
    };
    // pass 1: HBM -> (phase) -> DFT -> twiddle -> shared memory
    float2 cur[R1];
#pragma unroll
    for (int r = 0; r < R1; ++r) cur[r] = sample(t + r * S1);
#pragma unroll
    for (int s = 0; s < G1; ++s) {
        const int lo = t + SC::T * s;
        float2 nxt[R1];
        if (s + 1 < G1) {
#pragma unroll
            for (int r = 0; r < R1; ++r) nxt[r] = sample(lo + SC::T + r * S1);
        }
        dft_reg<R1, false>(cur);
        grp_twiddle<R1, S1, false>(tw, lo, cur);
        grp_smem_store<R1, S1>(sm, lo, SC::PADSH, cur);
        if (s + 1 < G1) {
#pragma unroll
            for (int r = 0; r < R1; ++r) cur[r] = nxt[r];
        }
    }
    __syncthreads();
    if constexpr (SC::P == 3) {
        streamed_mid_pass<SC, 1, SC::R2, SC::S2, false, true, true>(sm, tw + R1 * S1, t, 0);
        sub_sync<SC, 1>(0);
    }
    // last pass into registers, then natural order through shared memory
    float2 v[SC::E];
#pragma unroll
    for (int s = 0; s < GL; ++s) {
        float2 x[RL];
        grp_smem_load<RL, 1>(sm, pass_group<SC, RL, 1>(t, s) * RL, SC::PADSH, x);
        dft_reg<RL, false>(x);
#pragma unroll
        for (int r = 0; r < RL; ++r) v[s * RL + r] = x[r];
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < GL; ++s) {
#pragma unroll
        for (int r = 0; r < RL; ++r) sm[smem_pos(natural_index<SC>(pass_group<SC, RL, 1>(t, s), r), SC::PADSH)] = v[s * RL + r];
    }
    __syncthreads();
    grid_release_dependents();
    constexpr float inv_n = 1.0f / SC::N;
    float2* dst = out + line * SC::N;
#pragma unroll
    for (int i = 0; i < SC::E; ++i) {
        const int k = t + SC::T * i;
        const float2 x = sm[smem_pos(k, SC::PADSH)];
        __stcs(dst + k, COMPRESS ? make_float2(x.x * inv_n, -x.y * inv_n) : x);
    }
}

namespace {
using A256 = Sched<256, 16, 16, 16>;
using A512 = Sched<512, 32, 16, 32>;
using A1024 = Sched<1024, 32, 32, 32>;
using A2048 = Sched<2048, 16, 16, 8, 16>;
using A4096 = Sched<4096, 32, 16, 16, 16>;
using A8192 = Sched<8192, 32, 16, 16, 32>;
using A16384 = Sched<16384, 32, 16, 32, 32>;

template <class SC, bool COMPRESS>
cudaError_t launch_az(const float2* in, float2* out, int64_t n_lines, const float2* tw, const RdColumn* cols,
                      double r_near, cudaStream_t st) {
    constexpr int smem = SC::SMEM_ELEMS * 8;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(az_streamed_kernel<SC, COMPRESS>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
    }
    return launch_behind(az_streamed_kernel<SC, COMPRESS>, n_lines, SC::T, smem, 1, st, in, out, n_lines, tw, cols,
                         r_near);
}

template <bool COMPRESS>
cudaError_t launch_az_n(int n, const float2* in, float2* out, int64_t n_lines, const float2* tw, const RdColumn* c,
                        double r_near, cudaStream_t st) {
    switch (n) {
        case 256: return launch_az<A256, COMPRESS>(in, out, n_lines, tw, c, r_near, st);
        case 512: return launch_az<A512, COMPRESS>(in, out, n_lines, tw, c, r_near, st);
        case 1024: return launch_az<A1024, COMPRESS>(in, out, n_lines, tw, c, r_near, st);
        case 2048: return launch_az<A2048, COMPRESS>(in, out, n_lines, tw, c, r_near, st);
        case 4096: return launch_az<A4096, COMPRESS>(in, out, n_lines, tw, c, r_near, st);
        case 8192: return launch_az<A8192, COMPRESS>(in, out, n_lines, tw, c, r_near, st);
        case 16384: return launch_az<A16384, COMPRESS>(in, out, n_lines, tw, c, r_near, st);
    }
    return cudaErrorInvalidValue;
}
}  // namespace

// The schedule whose twiddle tables the azimuth kernel of length n uses.
const char* rd_az_schedule(int n) {
    switch (n) {
        case 256: return "n256_e16_r16x16_l8";
        case 512: return "n512_e32_r16x32_l8";
        case 1024: return "n1024_e32_r32x32_l4";
        case 2048: return "n2048_e16_r16x8x16_l1";
        case 4096: return "n4096_e32_r16x16x16_l1";
        case 8192: return "n8192_e32_r16x16x32_l1";
        case 16384: return "n16384_e32_r16x32x32_l1";
    }
    return nullptr;
}

cudaError_t launch_az_compress_rd(int n, const float2* in, float2* out, int64_t n_lines, const float2* tw,
                                  const void* cols, double r_near, cudaStream_t st) {
    return launch_az_n<true>(n, in, out, n_lines, tw, (const RdColumn*)cols, r_near, st);
}

// Forward FFT of n_lines lines of n (natural order in and out, in place
// allowed) with the twiddles of rd_az_schedule(n).
cudaError_t launch_az_fft_rd(int n, const float2* in, float2* out, int64_t n_lines, const float2* tw,
                             cudaStream_t st) {
    return launch_az_n<false>(n, in, out, n_lines, tw, nullptr, 0.0, st);
}

cudaError_t launch_rcmc(int taps, const float2* in, float2* out, int n_range, int n_f, const void* cols,
                        double r_near, int staged_rows, cudaStream_t st) {
    if (taps != 16 || n_range <= 0 || n_f <= 0) return cudaErrorInvalidValue;
    if (staged_rows > kRcMaxStaged) staged_rows = 0;   // too wide: every block reads global memory
    const size_t smem = (size_t)staged_rows * kRcCols * sizeof(float2);
    if (smem > 48 * 1024) {
        cudaError_t e =
            cudaFuncSetAttribute(rcmc_tile_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    const float rn_hi = (float)r_near, rn_lo = (float)(r_near - (double)rn_hi);
    const int tiles_f = (n_f + kRcCols - 1) / kRcCols, tiles_r = (n_range + kRcRows - 1) / kRcRows;
    return launch_behind(rcmc_tile_kernel, (int64_t)tiles_f * tiles_r, kRcCols * kRcWarps, (int)smem, 1, st, in, out,
                         n_range, n_f, (const RdColumn*)cols, rn_hi, rn_lo, staged_rows);
}

// Host: rows a tile must stage, the largest over every tile of the scene:
// 128 bins + 15 taps + the spread of the shift r (1/D - 1) over the tile's
// 32 columns and 128 bins, plus 4 rows of margin for rounding.
int rcmc_staged_rows(int n_range, int n_f, double r_near, const void* host_cols) {
    const RdColumn* c = (const RdColumn*)host_cols;
    double spread = 0;
    for (int g = 0; g < n_f; g += kRcCols) {
        double mn = 1e300, mx = -1e300;
        for (int j = g; j < g + kRcCols && j < n_f; ++j) {
            const double m = (double)c[j].mig_hi + (double)c[j].mig_lo;
            mn = m < mn ? m : mn;
            mx = m > mx ? m : mx;
        }
        for (int n0 = 0; n0 < n_range; n0 += kRcRows) {
            const int n1 = (n0 + kRcRows < n_range ? n0 + kRcRows : n_range) - 1;
            const double d = (r_near + n1) * mx - (r_near + n0) * mn;
            spread = d > spread ? d : spread;
        }
    }
    const double rows = kRcRows + 15 + ceil(spread) + 4;
    return rows > kRcMaxStaged ? kRcMaxStaged + 1 : (int)rows;
}

// Host: the per-frequency columns of a geometry, FP64 then rounded.
void rd_columns(int n_f, double kappa, double vs, void* host_cols) {
    RdColumn* c = (RdColumn*)host_cols;
    for (int j = 0; j < n_f; ++j) {
        const double f = (j < n_f / 2 ? (double)j : (double)(j - n_f)) / (double)n_f;
        const double q = f / (kappa * vs);
        const double d = sqrt(1.0 - q * q);
        const double a = kappa * d;
        c[j].a_hi = (float)a;
        c[j].a_lo = (float)(a - (double)c[j].a_hi);
        const double mig = q * q / (d * (1.0 + d));   // 1/D - 1 without cancellation
        c[j].mig_hi = (float)mig;
        c[j].mig_lo = (float)(mig - (double)c[j].mig_hi);
    }
}

size_t rd_column_bytes() { return sizeof(RdColumn); }

}  // namespace sar
