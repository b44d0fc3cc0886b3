// common.cuh -- device helpers shared by the 1d1v and 1d3v kernels: marker
// position storage, periodic cloud-in-cell neighbours, compensated FP32
// sums, and the marker generator (SplitMix64 jitter, analytic f0).
#pragma once
#include <math.h>

#include "avl_internal.cuh"
#include "fixed.cuh"

namespace avl {

// Raise a kernel's dynamic shared-memory limit to at least `bytes`.  The
// limit is a property of the function for the whole process, shared by every
// context, so it only ever grows (a smaller context created later must not
// lower the limit another one relies on).  Host only; call outside captures.
template <typename K>
static cudaError_t raise_smem_limit(K* kernel, int bytes)
{
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, kernel);
    if (e) return e;
    if (fa.maxDynamicSharedSizeBytes >= bytes) return cudaSuccess;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

// periodic neighbours of a lower CIC cell i0 in [-1, nx-1]; clamped so that a
// non-finite position can never index outside the grid
__device__ __forceinline__ void wrap_pair(int i0, int nx, int& ia, int& ib)
{
    ia = i0 < 0 ? i0 + nx : i0;
    ib = (i0 + 1 >= nx) ? i0 + 1 - nx : i0 + 1;
    ia = min(max(ia, 0), nx - 1);
    ib = min(max(ib, 0), nx - 1);
}

// ---------------------------------------------------------------------------
// marker storage access
// ---------------------------------------------------------------------------
template <typename T>
struct Pos;

// FP32: position = int cell + FP32 offset in [0, 1)
template <>
struct Pos<float> {
    int c;
    float o;
    __device__ __forceinline__ void load(const SpDev& sp, int cb, int k)
    {
        c = reinterpret_cast<const int*>(sp.mx[cb])[k];
        o = sp.moff[cb][k];
    }
    __device__ __forceinline__ void store(const SpDev& sp, int cb, int k) const
    {
        reinterpret_cast<int*>(sp.mx[cb])[k] = c;
        sp.moff[cb][k] = o;
    }
    // cloud-in-cell: lower cell i0 (may be -1) and weight w of cell i0 + 1
    __device__ __forceinline__ void cic(int& i0, float& w) const
    {
        if (o >= 0.5f) {
            i0 = c;
            w = o - 0.5f;
        } else {
            i0 = c - 1;
            w = o + 0.5f;
        }
    }
    __device__ __forceinline__ void drift(float disp, int nx)
    {
        o += disp;
        const float fo = floorf(o);
        c += static_cast<int>(fo);
        o -= fo;
        if (o >= 1.0f) {
            o -= 1.0f;
            c += 1;
        }
        if (c < 0 || c >= nx) {
            c %= nx;
            if (c < 0) c += nx;
        }
    }
    __device__ __forceinline__ double cells() const { return (double)c + (double)o; }
};

// FP64 marker position (step kernels and adjoint engine): a 64-bit
// fixed-point count of 2^-52 cells, x = X 2^-52 cells with
// 0 <= X < nx 2^52 < 2^63 (FP64 grids have nx < 2048).  It resolves 2^-52
// cells everywhere (a double of the same x resolves 2^-52 x), and the
// cloud-in-cell reads the weight straight from the bits: the 52 low bits of
// X - 2^51 are the mantissa of 1 + w, so that w and the lower cell cost one
// FP64 operation instead of four, and none where the weights stay integers
// (k_pd1x, k_pd3x, k_ad_depx).  The drift converts the displacement once.
struct PosX {
    long long X;
    static constexpr double ONE = 4503599627370496.0;   // 2^52: one cell
    __device__ __forceinline__ void load(const SpDev& sp, int cb, int k)
    {
        X = reinterpret_cast<const long long*>(sp.mx[cb])[k];
    }
    __device__ __forceinline__ void store(const SpDev& sp, int cb, int k) const
    {
        reinterpret_cast<long long*>(sp.mx[cb])[k] = X;
    }
    // cloud-in-cell: lower cell i0 (may be -1) and weight w of cell i0 + 1
    __device__ __forceinline__ void cic(int& i0, double& w) const
    {
        const long long U = X - (1ll << 51);   // x - 1/2
        i0 = (int)(U >> 52);                   // floor (arithmetic shift)
        w = __longlong_as_double(0x3FF0000000000000ll | (U & 0x000FFFFFFFFFFFFFll)) - 1.0;
    }
    // x into [0, nx) (periodic); Y computed modulo 2^64 so that no
    // displacement overflows
    __device__ __forceinline__ void wrap(long long Y, int nx)
    {
        const long long N = (long long)nx << 52;
        if ((unsigned long long)Y >= (unsigned long long)N) {
            Y %= N;
            if (Y < 0) Y += N;
        }
        X = Y;
    }
    // displacement of `scaled` 2^-52 cells (a double, rounded to the nearest
    // count; the conversion saturates and maps NaN to 0)
    __device__ __forceinline__ void drift_scaled(double scaled, int nx)
    {
        wrap((long long)((unsigned long long)X + (unsigned long long)__double2ll_rn(scaled)), nx);
    }
    __device__ __forceinline__ void drift(double disp, int nx) { drift_scaled(disp * ONE, nx); }
    __device__ __forceinline__ double cells() const { return (double)X * (1.0 / ONE); }
    __device__ __forceinline__ static PosX from_cells(double xi, int nx)
    {
        PosX p;
        p.X = 0;
        p.drift(xi, nx);
        return p;
    }
};

template <typename T>
struct PosSel;
template <>
struct PosSel<float> {
    using type = Pos<float>;
};
template <>
struct PosSel<double> {
    using type = PosX;
};
// marker position type: FP32 int cell + FP32 offset, FP64 PosX
template <typename T>
using PosM = typename PosSel<T>::type;

// position from a value in cells (FP64) given by a caller or the generator
template <typename T>
__device__ __forceinline__ PosM<T> posm_from_cells(double xi, int nx)
{
    if constexpr (sizeof(T) == 8) {
        return PosX::from_cells(xi, nx);
    } else {
        Pos<float> p;
        const double c = floor(xi);
        int ci = (int)c;
        const double o = xi - c;
        if (ci >= nx) ci -= nx;
        if (ci < 0) ci += nx;
        p.c = min(max(ci, 0), nx - 1);
        p.o = (float)o;
        if (p.o >= 1.0f) {
            p.o = 0.0f;
            p.c = (p.c + 1) % nx;
        }
        return p;
    }
}

// ---------------------------------------------------------------------------
// compensated accumulation
// ---------------------------------------------------------------------------
__device__ __forceinline__ void two_sum_add(float& hi, float& lo, float x)
{
    const float s = __fadd_rn(hi, x);
    const float bp = __fsub_rn(s, hi);
    const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(x, bp));
    hi = s;
    lo = __fadd_rn(lo, e);
}


// FP32 path: float-float arithmetic (an unevaluated sum hi + lo) for the sum
// of the chunks' window partials, the cell values and the column sums,
// without per-cell FP64 work.
struct ff {
    float hi, lo;
};

__device__ __forceinline__ void ff_add(ff& a, float x) { two_sum_add(a.hi, a.lo, x); }

// Sums of a finalize block in FP64.  An FP64 addition or conversion costs a
// warp 64 clocks, so the three sums share their tree, v^2 of a row comes from a
// table and the float-float accumulators of FP32 are widened in integers: nine
// per warp of a block (FP64 accumulators six) where the trees of N, W_kin and
// S, the conversions before them and v^2 took 31 per warp and row pair: k_fin1
// at 512 x 1024 FP32 48 -> 35 us, 512 x 6600 FP64 114 -> 95, 64 small runs
// 423 -> 352, k_fin3 at 100 x 24 x 20 x 18 FP64 53 -> 37.  (Block sums in
// float-float take 33 and 340 us, and 48 bits.)
//
// sum over eight neighbouring lanes
__device__ __forceinline__ double sum8(double v)
{
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// the warp's sums of a, b and c, in lanes 0, 8 and 16: half the lanes go on
// with c, a quarter with b, so that three sums take six additions, not 15
__device__ __forceinline__ double warp_sum3(double a, double b, double c)
{
    const int lane = threadIdx.x & 31;
    const bool h = lane & 16, q = lane & 8;
    double x = h ? c : a, y = h ? 0.0 : b;
    x += __shfl_xor_sync(0xffffffffu, h ? a : c, 16);
    y += __shfl_xor_sync(0xffffffffu, h ? b : 0.0, 16);
    double z = q ? y : x;
    z += __shfl_xor_sync(0xffffffffu, q ? x : y, 8);
    return sum8(z);
}
__device__ __forceinline__ double acc_value(ff a) { return fx_widen(a.hi) + fx_widen(a.lo); }
__device__ __forceinline__ double acc_value(double a) { return a; }

template <typename T>
struct ColAcc;

template <>
struct ColAcc<float> {
    ff rho{0.f, 0.f}, w{0.f, 0.f}, ent{0.f, 0.f};
    __device__ __forceinline__ void add(float fh, float fl, float v2)
    {
        ff_add(rho, fh);
        rho.lo = __fadd_rn(rho.lo, fl);
        ff_add(w, __fmul_rn(v2, fh));
        if (fh > 0.f) ff_add(ent, __fmul_rn(fh, logf(fh)));
    }
    using Sum = ff;
};

template <>
struct ColAcc<double> {
    using Sum = double;
    double rho = 0.0, w = 0.0, ent = 0.0;
    const longlong2* logtab = nullptr;
    __device__ __forceinline__ void add(double fh, double, double v2)
    {
        rho += fh;
        w += v2 * fh;
        if (__double_as_longlong(fh) > 0) ent += fh * fx_log(fh, logtab);   // fh > 0 (fh is not a NaN)
    }
};

// SplitMix64 (Steele, Lea & Flood 2014): output n of the generator seeded
// with `seed`.
__device__ __forceinline__ unsigned long long splitmix64(unsigned long long seed, unsigned long long n)
{
    unsigned long long z = seed + (n + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__device__ __forceinline__ double jitter_u01(unsigned long long seed, int s, long long m, int d)
{
    const unsigned long long n = ((unsigned long long)(unsigned)s << 48) | ((unsigned long long)m * 4ull + d);
    return (double)(splitmix64(seed, n) >> 11) * (1.0 / 9007199254740992.0);
}

__device__ __forceinline__ double f0_value(const avl_f0* p, int nvdim, double L, double x, const double* v)
{
    double pert = 1.0;
    for (int m = 0; m < p->nmode; ++m)
        pert += p->amp[m] * cos(2.0 * M_PI * (double)p->mode[m] / L * x + p->phase[m]);
    double sum = 0.0;
    for (int b = 0; b < p->nbeam; ++b) {
        double gb = p->beam_n[b];
        for (int d = 0; d < nvdim; ++d) {
            const double sd = p->beam_vth[b][d];
            const double t = (v[d] - p->beam_u[b][d]) / sd;
            gb *= exp(-0.5 * t * t) / (sqrt(2.0 * M_PI) * sd);
        }
        sum += gb;
    }
    return sum * pert;
}
}  // namespace avl
