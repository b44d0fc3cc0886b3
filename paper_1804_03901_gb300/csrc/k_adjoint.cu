// k_adjoint.cu -- discrete adjoint of the 1d1v time step on the GPU.
//
// Objective: J = 1/2 sum_i E_i(T)^2 dx after nsteps steps (the field energy
// of Eq. 12 with the factor 1/2 and no 1/cP).  Parameters: the mode
// amplitudes and beam x-drifts of the initial distribution f0 of one species
// (Sec. 3.3 / Eq. 17 form); they enter only through the marker values
// f_l = f0(x_l, v_l), so dJ/dtheta = sum_l mu_l df0_l/dtheta with
// mu_l = dJ/df_l, the total derivative through every later reconstruction
// (Eq. 4), moment (Eq. 14), Poisson solve (Eq. 6) and push (Sec. 2).
//
// The engine keeps its own markers in the fixed lattice order (marker m =
// cell * ppc + sub, as created), so that the adjoint variables of a marker
// stay aligned across steps.  Per step n the forward pass deposits with
// global atomics, forms F = N / D and the charge, solves for E (the circulant
// product up to GREEN_MAX cells, beyond that the FFT) and pushes.  E of every
// state is kept, (x, v) every K steps; the backward pass recomputes each
// segment of K states from its checkpoint in the stored fields (the order of
// the deposit's reductions changes E's last bits, and a marker near a cell's
// edge then takes the other one-sided derivative: with E solved again the
// FP32 gradient spread 1.6 times as far from run to run), storing positions,
// velocities and the grids D and F of every state, then walks it backwards:
//   e^n   = sum_l lt_l (q/m) dt G(X^n_l),  lt = lambda_V + dt lambda_X
//           (e^N = dx E^N at the final state)
//   psi   = q dv P^T e^n = -q dv P e^n   (the multiplier of Eq. 6 is odd and
//           purely imaginary)
//   A = psi / D, B = psi F / D per cell (0 where D = 0)
//   mu   += sum_cells A alpha;  g = sum_cells (A f - B) d alpha / d(X, V)
//   lambda_X = lambda_X + lt (q/m) dt dE/dx(X^n) + g_X;  lambda_V = lt + g_V
// The cloud-in-cell derivatives are the one-sided ones of the floor() rule.
// Per-marker and per-cell arithmetic runs in the storage precision (FP64 is a
// small fraction of the FP32 rate on this GPU); mu, the charge and E stay FP64.
#include <math.h>

#include <algorithm>
#include <vector>

#include "avl_internal.cuh"
#include "common.cuh"

namespace avl {

constexpr int AD_E_THREADS = 512;        // adjoint deposit block
constexpr int AD_E_SMEM = 64 * 1024;     // and its copies of the grid
constexpr int AD_PUSH_NX = 2048;         // largest field an FP32 push stages (8 KB)

// a species' constants in the storage precision, computed once on the host:
// an FP64 operation or conversion takes an SM's pipe as long as 64 FP32
// instructions, and every thread would run a dozen of them for its few
// markers
template <typename T>
struct AdjC {
    T va, vb;        // velocity row: v va + vb
    T qm_dt, dt_dx;
    T lt;            // dt dv / dx: lambda_X dx to lambda_V dv
    double c0;       // (q/m) dt / dv: deposit of lambda_V dv
};

// device-side view of the engine's buffers
struct AdjSp {
    long long n;
    int nv, mobile;
    int lat[2];
    unsigned long long seed;
    double jitter;
    void* hx;          // [K + 1][n] positions per slot (FP32: int cell; FP64: int64 2^-52 cells, PosX)
    float* hoff;       // [K + 1][n] FP32 offsets
    void* hv;          // [K + 1][n] velocities
    void* cx;          // [C][n] checkpoints
    float* coff;
    void* cv;
    void* f;           // [n] marker values
    void* lx;          // [n] lambda_X dx
    void* lv;          // [n] lambda_V dv
    double* mu;        // [n] dJ / df_l
    void* num;         // [nx][nv][2] deposit accumulator: (numerator, denominator) pairs
    float* fref;       // FP32: [nx][nv] F of the initial state; numerators hold deviations from it
    void* hF;          // [K + 1][nx][nv] F = N / D per slot
    void* hD;          // [K + 1][nx][nv] D per slot
    void* AB;          // [nx][nv][2] grid adjoint (A, B) of the state being walked back
    void* dE;          // [nx] (q/m) dt dE / dv, dE from cell i to i + 1, of that state
    AdjC<float> cf;
    AdjC<double> cd;
};
__device__ __forceinline__ const AdjC<float>& adj_c(const AdjSp& a, float) { return a.cf; }
__device__ __forceinline__ const AdjC<double>& adj_c(const AdjSp& a, double) { return a.cd; }

struct AdjDev {
    int ns, theta_s, K;
    int nact, act[MAXS];   // species stepped each time: mobile ones and theta_s
    int nstat, stat[MAXS]; // the others (immobile): their charge is deposited once
    AdjSp sp[MAXS];
    double* rho;       // [nx]
    double* rho_static;   // [nx] charge of the other (immobile) species, deposited once
    double* e;         // [nx] adjoint deposit
    double* tmp;       // [nx] P e
    double* hE;        // [K + 1][nx]
    double* allE;      // [nsteps + 1][nx]: E of every state of the forward pass
    double* grad;      // [nmode + nbeam] of the theta species
    const avl_f0* f0;  // [ns] (theta for theta_s)
};

template <typename T>
struct APos;
template <>
struct APos<float> {
    __device__ static Pos<float> load(const AdjSp& a, int slot, long long k)
    {
        Pos<float> p;
        p.c = reinterpret_cast<const int*>(a.hx)[(size_t)slot * a.n + k];
        p.o = a.hoff[(size_t)slot * a.n + k];
        return p;
    }
    __device__ static void store(const AdjSp& a, int slot, long long k, const Pos<float>& p)
    {
        reinterpret_cast<int*>(a.hx)[(size_t)slot * a.n + k] = p.c;
        a.hoff[(size_t)slot * a.n + k] = p.o;
    }
};
template <>
struct APos<double> {
    __device__ static PosX load(const AdjSp& a, int slot, long long k)
    {
        PosX p;
        p.X = reinterpret_cast<const long long*>(a.hx)[(size_t)slot * a.n + k];
        return p;
    }
    __device__ static void store(const AdjSp& a, int slot, long long k, const PosX& p)
    {
        reinterpret_cast<long long*>(a.hx)[(size_t)slot * a.n + k] = p.X;
    }
};

// velocity dual row j0 and weight w of row j0 + 1 (t = (v - vmin)/dv - 1/2),
// in the storage precision with one explicit fused multiply-add, so that
// the deposit and the gather find the same row and weight
__device__ __forceinline__ int vrow(float v, const AdjC<float>& c, int nv, float& w)
{
    const float t = __fmaf_rn(v, c.va, c.vb);
    if (!(t > -2.f && t < (float)(nv + 1))) {
        w = 0.f;
        return t > 0.f ? nv + 1 : -2;
    }
    const float fl = floorf(t);
    w = t - fl;
    return (int)fl;
}
// FP64: the weight as a count of 2^-52, from t as a 64-bit count of 2^-52
// rows (rows beyond 1023, which that does not hold, from the floor)
__device__ __forceinline__ int vrow52(double v, const AdjC<double>& c, int nv, long long& w)
{
    const double t = __fma_rn(v, c.va, c.vb);
    int j;
    if (((__double2hiint(t) >> 20) & 0x7ff) < 1033) {   // |t| < 1024
        const long long n = fx_count(t);
        w = n & (FX_ONE - 1);
        j = (int)(n >> 52);
    } else {
        const double fl = floor(t);
        w = fx_count(t - fl);
        j = t > 0.0 ? (int)fmin(fl, 1.0e9) : -2;
    }
    if (j < -1 || j > nv) {
        w = 0;
        return j < 0 ? -2 : nv + 1;
    }
    return j;
}
__device__ __forceinline__ int vrow(double v, const AdjC<double>& c, int nv, double& w)
{
    long long w52;
    const int j = vrow52(v, c, nv, w52);
    w = __longlong_as_double(0x3FF0000000000000ll | w52) - 1.0;
    return j;
}

template <typename T>
struct Pair2;
template <>
struct Pair2<float> {
    using type = float2;
};
template <>
struct Pair2<double> {
    using type = double2;
};

// (numerator, denominator) of one cell in one reduction: a v2 FP32
// reduction in the FP32 path, two FP64 ones in the FP64 path
__device__ __forceinline__ void pair_add(float* p, float n, float d)
{
    asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(n), "f"(d) : "memory");
}
__device__ __forceinline__ void pair_add(double* p, double n, double d)
{
    atomicAdd(p, n);
    atomicAdd(p + 1, d);
}

// lattice marker m (order m = (i nv + j) ppc + a pv + b) of species s
template <typename T>
__global__ void k_ad_init(const StepArgs* __restrict__ A, const AdjDev* __restrict__ D, int s)
{
    const SpDev& sp = A->sp[s];
    const AdjSp& a = D->sp[s];
    const avl_f0* f0 = D->f0 + s;
    const int px = a.lat[0], pv = a.lat[1], ppc = px * pv;
    for (long long m = (long long)blockIdx.x * blockDim.x + threadIdx.x; m < a.n; m += (long long)gridDim.x * blockDim.x) {
        const long long cell = m / ppc;
        const int sub = (int)(m - cell * ppc);
        const int i = (int)(cell / sp.nv[0]), j = (int)(cell - (long long)i * sp.nv[0]);
        const int ia = sub / pv, ib = sub - ia * pv;
        const double J0 = (jitter_u01(a.seed, s, m, 0) - 0.5) * a.jitter;
        const double J1 = (jitter_u01(a.seed, s, m, 1) - 0.5) * a.jitter;
        const double xi = (double)i + ((double)ia + 0.5 + J0) / px;
        const double v[3] = {sp.vmin[0] + ((double)j + ((double)ib + 0.5 + J1) / pv) * sp.dv[0], 0.0, 0.0};
        APos<T>::store(a, 0, m, posm_from_cells<T>(xi, sp.nx));
        reinterpret_cast<T*>(a.hv)[m] = (T)v[0];
        reinterpret_cast<T*>(a.f)[m] = (T)f0_value(f0, 1, sp.nx * sp.dx, xi * sp.dx, v);
        reinterpret_cast<T*>(a.lx)[m] = (T)0;
        reinterpret_cast<T*>(a.lv)[m] = (T)0;
        a.mu[m] = 0.0;
    }
}

// Deposit of the markers of slot `slot` (numerator and denominator of Eq. 4).
// The 32 markers of a warp are neighbours on the creation lattice (a few
// velocity rows of one column) and stay together, so with the grid stored
// column by column their reductions fall into a few sectors.  Bound by L2's
// reductions: 1 M markers 18.5 us (27.5 with the grid stored by rows; with
// both rows of a column in one 16-byte reduction where it is aligned 25, with
// a warp's sums formed in shared memory first 36), 19.7 with the numerators as
// deviations from F_0 (k_ad_fin).
__global__ void __launch_bounds__(256) k_ad_dep(const AdjDev* __restrict__ D, int nx, int slot, int all)   // all: the static list
{
    const int s = all ? D->stat[blockIdx.y] : D->act[blockIdx.y];
    const AdjSp& a = D->sp[s];
    const AdjC<float> C = a.cf;
    const int nv = a.nv;
    float* acc = reinterpret_cast<float*>(a.num);
    const float* f = reinterpret_cast<const float*>(a.f);
    const float* __restrict__ fref = a.fref;
    const float* vv = reinterpret_cast<const float*>(a.hv) + (size_t)slot * a.n;
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < a.n; k += (long long)gridDim.x * blockDim.x) {
        int i0, ia, ib;
        float wx, wv;
        APos<float>::load(a, slot, k).cic(i0, wx);
        wrap_pair(i0, nx, ia, ib);
        const int j0 = vrow(vv[k], C, nv, wv);
        const float fl = f[k];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int j = j0 + (q >> 1);
            if (j < 0 || j >= nv) continue;
            const float w = (q & 1 ? wx : 1.f - wx) * (q >> 1 ? wv : 1.f - wv);
            const size_t o = (size_t)(q & 1 ? ib : ia) * nv + j;
            pair_add(acc + 2 * o, w * (fl - fref[o]), w);
        }
    }
}

// FP64: a warp sums its contributions in a patch of shared memory (columns x
// rows around its markers' footprints), weights and sums in integers
// (fixed.cuh), and adds every cell of the patch to the grid: 20 to 60
// reductions of (numerator, denominator) where the markers have 128 corners.
// Lattice neighbours share footprints in fours; four copies of the patch by
// lane keep them off one another's words.  g of a marker (k_ad_gather) has
// the factor (f - F) / D, so F = N / D must not lose what a small D leaves of
// it: the numerator takes the denominator's rounded weights, each product
// whole in two words (2^-57 and 2^-83 of the value's unit), and every cell has
// its own unit, of the largest value that reaches it.  A marker with a corner
// below SMALL_AD = 2^-16 (0.07 % of them), with a value beyond the sums' range
// or in a warp whose patch does not fit adds its corners to the grid in FP64.
// 1 M markers: 75 -> 39 us (34 with the products rounded to 2^-57 of the warp's
// largest value; one copy 54; five blocks per SM, 51 registers, 46).
constexpr int AD_PATCH = 160;   // words of a warp's patch and its copies
constexpr int AD_LO = 26;       // bits of the low words: 32 of them stay below 2^31
constexpr float SMALL_AD = 1.0f / (1 << 16);
__global__ void __launch_bounds__(256, 4) k_ad_depx(const AdjDev* __restrict__ D, int nx, int slot, int all)
{
    __shared__ unsigned long long patch_s[8][2 * AD_PATCH];
    __shared__ unsigned low_s[8][2 * AD_PATCH];
    const int s = all ? D->stat[blockIdx.y] : D->act[blockIdx.y];
    const AdjSp& a = D->sp[s];
    const AdjC<double> C = a.cd;
    const int nv = a.nv, lane = threadIdx.x & 31;
    unsigned long long* Pn = patch_s[threadIdx.x >> 5];   // numerators, denominators
    unsigned long long* Pd = Pn + AD_PATCH;
    unsigned* Pl = low_s[threadIdx.x >> 5];               // low words of the numerators
    int* Pe = reinterpret_cast<int*>(Pl + AD_PATCH);      // exponents of the units
    double* acc = reinterpret_cast<double*>(a.num);
    const double* f = reinterpret_cast<const double*>(a.f);
    const double* vv = reinterpret_cast<const double*>(a.hv) + (size_t)slot * a.n;
    const long long n_pad = (a.n + 31) / 32 * 32;   // whole warps iterate together
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n_pad; k += (long long)gridDim.x * blockDim.x) {
        bool ok = k < a.n;
        int i0 = 0, j0 = -2;
        long long u = 0, w = 0;   // weights, 2^-52
        double fl = 0.0;
        if (ok) {
            const long long U = APos<double>::load(a, slot, k).X - (FX_ONE >> 1);
            i0 = (int)(U >> 52);
            u = U & (FX_ONE - 1);
            j0 = vrow52(vv[k], C, nv, w);
            fl = f[k];
        }
        ok = ok && j0 >= -1 && j0 < nv;   // a corner on the grid
        int e;
        const long long mant = fx_value(fl, e);
        bool pat = ok && lesser_weight(u) * lesser_weight(w) >= SMALL_AD && (fx_in_range(e) || mant == 0);
        const unsigned any = __ballot_sync(0xffffffffu, pat);
        if (any) {
            // the patch: columns relative to the first marker's (periodic), rows
            const int ir = __shfl_sync(0xffffffffu, i0, __ffs(any) - 1);
            int di = i0 - ir;
            if (2 * di > nx) di -= nx;
            if (2 * di < -nx) di += nx;
            const int d0 = __reduce_min_sync(0xffffffffu, pat ? di : 0x3fffffff);
            const int d1 = __reduce_max_sync(0xffffffffu, pat ? di : -0x3fffffff);
            const int r0 = __reduce_min_sync(0xffffffffu, pat ? j0 : 0x3fffffff);
            const int r1 = __reduce_max_sync(0xffffffffu, pat ? j0 : -0x3fffffff);
            const int W = d1 - d0 + 2, H = r1 - r0 + 2;
            if (W <= nx && H <= AD_PATCH && W * H <= AD_PATCH) {
                const int cs = W * H * 4 <= AD_PATCH ? 2 : 0;   // copies: 1 << cs
                for (int q = lane; q < (W * H) << cs; q += 32) {
                    Pn[q] = Pd[q] = 0;
                    Pl[q] = 0;
                    Pe[q] = FX_EMIN;
                }
                __syncwarp();
                const int at = (di - d0) * H + j0 - r0, lc = lane & ((1 << cs) - 1);
                const int cell[4] = {at, at + H, at + 1, at + H + 1};
                if (pat) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) atomicMax(Pe + cell[q], e);
                }
                __syncwarp();
                if (pat) {
                    long long c[4];   // weights of the corners, 2^-57
                    c[3] = fx_mul(fx_split(u << 5), fx_split(w << 4));
                    c[2] = (w << 5) - c[3];
                    c[1] = (u << 5) - c[3];
                    c[0] = (FX_ONE << 5) - (u << 5) - c[2];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int o = (cell[q] << cs) + lc;
                        const Limbs A = fx_split(c[q]), v = fx_split(mant >> min(Pe[cell[q]] - e, 63));
                        long long m = ((long long)A.l * v.l) >> FX_LIMB;
                        mad_wide(m, A.h, v.l);
                        mad_wide(m, A.l, v.h);
                        long long h = m >> FX_LIMB;
                        mad_wide(h, A.h, v.h);
                        atomicAdd(Pn + o, (unsigned long long)h);
                        atomicAdd(Pl + o, ((unsigned)m & ((1u << FX_LIMB) - 1)) >> (FX_LIMB - AD_LO));
                        atomicAdd(Pd + o, (unsigned long long)c[q]);
                    }
                }
                __syncwarp();
                for (int q = lane; q < W * H; q += 32) {
                    long long sn = 0, sd = 0, sl = 0;
                    for (int t = 0; t < 1 << cs; ++t) {
                        sn += (long long)Pn[(q << cs) + t];
                        sd += (long long)Pd[(q << cs) + t];
                        sl += Pl[(q << cs) + t];
                    }
                    sn += sl >> AD_LO;
                    // as many of the low bits as there is room for
                    const int z = min(__clzll(sn < 0 ? ~sn : sn) - 1, AD_LO);
                    sn = sn * (1ll << z) + ((sl & ((1 << AD_LO) - 1)) >> (AD_LO - z));
                    const int col = q / H, j = r0 + q - col * H;
                    int x = ir + d0 + col;
                    x = x < 0 ? x + nx : (x >= nx ? x - nx : x);
                    if (sd != 0 && j >= 0 && j < nv)
                        pair_add(acc + 2 * ((size_t)x * nv + j), fx_scale(fx_double(sn), Pe[q] - 1079 - z),
                                 fx_scale(fx_double(sd), -57));
                }
                __syncwarp();
                ok = ok && !pat;
            }
        }
        if (ok) {
            int ia, ib;
            wrap_pair(i0, nx, ia, ib);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int j = j0 + (q >> 1);
                if (j < 0 || j >= nv) continue;
                const double cd = fx_scale(weight_of(u, q & 1) * weight_of(w, q & 2), -104);
                pair_add(acc + 2 * ((size_t)(q & 1 ? ib : ia) * nv + j), cd * fl, cd);
            }
        }
    }
}

// F = N / D and D into slot `slot`, accumulators cleared; charge per column
// (Eq. 14) added into rho.  One warp per column and group of rows.  FP32:
// N holds sum alpha (f_l - F_0), F_0 the initial state's F, so F = F_0 + N / D
// (Eq. 4 for any F_0) carries the rounding of f's change and of its spread in
// a cell only; the charge is summed in float-float before F is rounded.
template <typename T>
__global__ void __launch_bounds__(256) k_ad_fin(const StepArgs* __restrict__ A, const AdjDev* __restrict__ D, int slot,
                                                int all)
{
    using P = typename Pair2<T>::type;
    const int s = all ? D->stat[blockIdx.y] : D->act[blockIdx.y];
    const SpDev& sp = A->sp[s];
    const AdjSp& a = D->sp[s];
    const int nx = sp.nx, nv = sp.nv[0], lane = threadIdx.x & 31;
    const int x = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (x >= nx) return;
    const size_t cells = (size_t)nx * nv;
    P* acc = reinterpret_cast<P*>(a.num);
    T* F = reinterpret_cast<T*>(a.hF) + (size_t)slot * cells;
    T* Dg = reinterpret_cast<T*>(a.hD) + (size_t)slot * cells;
    using Sum = typename ColAcc<T>::Sum;
    Sum rs{};
    for (int j = blockIdx.z * 32 + lane; j < nv; j += 32 * gridDim.z) {
        const size_t o = (size_t)x * nv + j;
        const P nd = acc[o];
        T fv = (T)0;
        if constexpr (sizeof(T) == 8) {
            if (nd.y > 0.0) fv = fx_div(nd.x, nd.y);
            rs += fv;
        } else {
            if (nd.y > 0.f) {
                const float f0 = a.fref[o], q = nd.x / nd.y;
                ff_add(rs, f0);
                ff_add(rs, q);
                fv = f0 + q;
            }
        }
        F[o] = fv;
        Dg[o] = nd.y;
        acc[o] = P{};
    }
    double r = acc_value(rs);
    for (int q = 16; q; q >>= 1) r += __shfl_down_sync(0xffffffffu, r, q);
    if (lane == 0) atomicAdd(D->rho + x, sp.q * sp.dv[0] * r);
}

// push (Sec. 2) from slot to slot + 1 with the field of slot (`staged`: FP32
// grids whose field fits a block's shared memory convert it once, not two
// values per marker); immobile species are copied
template <typename T>
__global__ void __launch_bounds__(256) k_ad_push(const AdjDev* __restrict__ D, int nx, int slot, bool staged)
{
    extern __shared__ float Es[];
    const int s = D->act[blockIdx.y];
    const AdjSp& a = D->sp[s];
    const AdjC<T> C = adj_c(a, (T)0);
    const bool mobile = a.mobile;
    const double* E = D->hE + (size_t)slot * nx;
    if (staged) {
        for (int i = threadIdx.x; i < nx; i += blockDim.x) Es[i] = (float)E[i];
        __syncthreads();
    }
    auto field = [&](int i) { return staged ? (T)Es[i] : (T)E[i]; };
    const T* v0 = reinterpret_cast<const T*>(a.hv) + (size_t)slot * a.n;
    T* v1 = reinterpret_cast<T*>(a.hv) + (size_t)(slot + 1) * a.n;
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < a.n; k += (long long)gridDim.x * blockDim.x) {
        PosM<T> p = APos<T>::load(a, slot, k);
        T v = v0[k];
        if (mobile) {
            int i0;
            T w;
            p.cic(i0, w);
            int ia, ib;
            wrap_pair(i0, nx, ia, ib);
            const T Ea = field(ia);
            v = fma(C.qm_dt, fma(w, field(ib) - Ea, Ea), v);
            if constexpr (sizeof(T) == 8)
                p.wrap((long long)((unsigned long long)p.X + (unsigned long long)fx_count(v * C.dt_dx)), nx);
            else
                p.drift(v * C.dt_dx, nx);
        }
        APos<T>::store(a, slot + 1, k, p);
        v1[k] = v;
    }
}

// Partial sums in the storage precision, in copies of the grid by lane (the
// 32 markers of a warp are lattice neighbours and meet in one or two cells;
// with one copy per warp their reductions ran one after the other: 1 M
// markers FP64 124 -> 22 us, FP32 36 -> 11), es[i copies + lane mod copies], which also keeps the lanes'
// banks apart.  The copies are summed in FP64 (FP32: float-float).
template <typename T>
__global__ void __launch_bounds__(AD_E_THREADS) k_ad_e(const AdjDev* __restrict__ D, int nx, double dx, int slot,
                                                       int terminal, int copies)
{
    extern __shared__ __align__(16) unsigned char es_raw[];
    T* es = reinterpret_cast<T*>(es_raw);   // [nx][copies]
    const int s = D->act[blockIdx.y];
    const AdjSp& a = D->sp[s];
    if (terminal) {
        if (blockIdx.y == 0 && blockIdx.x == 0)
            for (int i = threadIdx.x; i < nx; i += blockDim.x) D->e[i] = dx * D->hE[(size_t)slot * nx + i];
        return;
    }
    if (!a.mobile) return;
    for (int i = threadIdx.x; i < copies * nx; i += blockDim.x) es[i] = (T)0;
    __syncthreads();
    const int lc = copies ? (threadIdx.x & (copies - 1)) : 0;
    const T* lx = reinterpret_cast<const T*>(a.lx);
    const T* lv = reinterpret_cast<const T*>(a.lv);
    const T clt = adj_c(a, (T)0).lt;
    const double c0 = adj_c(a, (T)0).c0;
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < a.n; k += (long long)gridDim.x * blockDim.x) {
        const PosM<T> p = APos<T>::load(a, slot, k);
        int i0;
        T w;
        p.cic(i0, w);
        int ia, ib;
        wrap_pair(i0, nx, ia, ib);
        const T c = fma(clt, lx[k], lv[k]);
        const T cb = c * w, ca = c - cb;
        if (copies) {
            atomicAdd(es + ia * copies + lc, ca);
            atomicAdd(es + ib * copies + lc, cb);
        } else {   // grid too large for shared copies
            atomicAdd(D->e + ia, c0 * (double)ca);
            atomicAdd(D->e + ib, c0 * (double)cb);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nx && copies; i += blockDim.x) {
        double t;
        if constexpr (sizeof(T) == 4) {
            ff sum{0.f, 0.f};
            for (int q = 0; q < copies; ++q) ff_add(sum, es[i * copies + ((q + i) & (copies - 1))]);
            t = (double)sum.hi + (double)sum.lo;
        } else {
            t = 0.0;
            for (int q = 0; q < copies; ++q) t += es[i * copies + ((q + i) & (copies - 1))];
        }
        if (t != 0.0) atomicAdd(D->e + i, c0 * t);
    }
}

// grid adjoint of slot: A = psi / D, B = psi F / D (0 where D = 0) with
// psi = q dv P^T e = -q dv (P e) = -q dv tmp
template <typename T>
__global__ void k_ad_grid(const StepArgs* __restrict__ A, const AdjDev* __restrict__ D, int slot)
{
    const int s = D->act[blockIdx.y];
    const SpDev& sp = A->sp[s];
    const AdjSp& a = D->sp[s];
    const int nx = sp.nx, nv = sp.nv[0];
    const size_t cells = (size_t)nx * nv;
    if (blockIdx.x == 0) {
        const double* E = D->hE + (size_t)slot * nx;
        const double c = adj_c(a, (T)0).c0;
        for (int i = threadIdx.x; i < nx; i += blockDim.x)
            reinterpret_cast<T*>(a.dE)[i] = (T)(c * (E[i + 1 == nx ? 0 : i + 1] - E[i]));
    }
    const T* F = reinterpret_cast<const T*>(a.hF) + (size_t)slot * cells;
    const T* Dg = reinterpret_cast<const T*>(a.hD) + (size_t)slot * cells;
    T* ab = reinterpret_cast<T*>(a.AB);
    const double psi_c = -sp.q * sp.dv[0];
    for (size_t o = (size_t)blockIdx.x * blockDim.x + threadIdx.x; o < cells; o += (size_t)gridDim.x * blockDim.x) {
        const T d = Dg[o];
        const T ps = (T)(psi_c * D->tmp[cells >> 32 ? o / nv : (unsigned)o / (unsigned)nv]);
        T A_;
        if constexpr (sizeof(T) == 8)
            A_ = d > (T)0 ? fx_div(ps, d) : (T)0;
        else
            A_ = d > (T)0 ? ps / d : (T)0;
        ab[2 * o] = A_;
        ab[2 * o + 1] = A_ * F[o];
    }
}

// per marker: mu += sum A alpha, lambda update (see the file head; lambda_X
// times dx and lambda_V times dv, so that no derivative is scaled).  A and
// A f - B at the four corners (0 off the grid), the weights of rows and
// columns in turn: 28 operations where the corners one by one took about 50,
// on the FP64 pipe in the FP64 path.  Weighted sums, not interpolation by
// differences: A = psi / D is largest where a corner's weight is smallest.
// 1 M markers: FP64 102 -> 62 us, FP32 26 -> 16.
template <typename T>
__global__ void __launch_bounds__(256) k_ad_gather(const AdjDev* __restrict__ D, int nx, int slot, int terminal)
{
    using P = typename Pair2<T>::type;
    const int s = D->act[blockIdx.y];
    const AdjSp& a = D->sp[s];
    const AdjC<T> C = adj_c(a, (T)0);
    const int nv = a.nv;
    const bool mobile = a.mobile;
    const P* ab = reinterpret_cast<const P*>(a.AB);
    const T* dE = reinterpret_cast<const T*>(a.dE);
    const T* vv = reinterpret_cast<const T*>(a.hv) + (size_t)slot * a.n;
    const T* f = reinterpret_cast<const T*>(a.f);
    T* lx = reinterpret_cast<T*>(a.lx);
    T* lv = reinterpret_cast<T*>(a.lv);
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < a.n; k += (long long)gridDim.x * blockDim.x) {
        const PosM<T> p = APos<T>::load(a, slot, k);
        int i0, ia, ib;
        T wx, wv;
        p.cic(i0, wx);
        wrap_pair(i0, nx, ia, ib);
        const int j0 = vrow(vv[k], C, nv, wv);
        const T fl = f[k];
        P p00{}, p01{}, p10{}, p11{};   // (row, column)
        if (j0 >= 0 && j0 < nv) {
            p00 = ab[(size_t)ia * nv + j0];
            p01 = ab[(size_t)ib * nv + j0];
        }
        if (j0 + 1 >= 0 && j0 + 1 < nv) {
            p10 = ab[(size_t)ia * nv + j0 + 1];
            p11 = ab[(size_t)ib * nv + j0 + 1];
        }
        const T ux = (T)1 - wx, uv = (T)1 - wv;
        const T m = uv * fma(wx, p01.x, ux * p00.x) + wv * fma(wx, p11.x, ux * p10.x);
        const T c00 = fma(p00.x, fl, -p00.y), c01 = fma(p01.x, fl, -p01.y);
        const T c10 = fma(p10.x, fl, -p10.y), c11 = fma(p11.x, fl, -p11.y);
        const T gx = fma(wv, c11 - c10, uv * (c01 - c00));
        const T gv = fma(wx, c11 - c01, ux * (c10 - c00));
        a.mu[k] += (double)m;
        if (terminal) {
            lx[k] = gx;
            lv[k] = gv;
        } else if (mobile) {
            const T lxk = lx[k];
            const T lt = fma(C.lt, lxk, lv[k]);
            lx[k] = fma(lt, dE[ia], lxk) + gx;
            lv[k] = lt + gv;
        }
    }
}

// dJ/dtheta = sum_l mu_l df0_l/dtheta for the theta species: df0/d amp_m =
// B(v) cos(k_m x + phase_m), df0/d u_b = P(x) n_b M_b(v) (v - u_b) / vth_b^2
template <typename T>
__global__ void __launch_bounds__(256) k_ad_theta(const StepArgs* __restrict__ A, const AdjDev* __restrict__ D)
{
    const int s = D->theta_s;
    const SpDev& sp = A->sp[s];
    const AdjSp& a = D->sp[s];
    const avl_f0* f0 = D->f0 + s;
    const int nm = f0->nmode, nb = f0->nbeam, nt = nm + nb;
    __shared__ double red[64 + 4][8];
    double acc[64 + 4];
    for (int t = 0; t < nt; ++t) acc[t] = 0.0;
    const int px = a.lat[0], pv = a.lat[1], ppc = px * pv;
    const double L = sp.nx * sp.dx;
    for (long long m = (long long)blockIdx.x * blockDim.x + threadIdx.x; m < a.n; m += (long long)gridDim.x * blockDim.x) {
        const long long cell = m / ppc;
        const int sub = (int)(m - cell * ppc);
        const int i = (int)(cell / sp.nv[0]), j = (int)(cell - (long long)i * sp.nv[0]);
        const int ia = sub / pv, ib = sub - ia * pv;
        const double J0 = (jitter_u01(a.seed, s, m, 0) - 0.5) * a.jitter;
        const double J1 = (jitter_u01(a.seed, s, m, 1) - 0.5) * a.jitter;
        const double x = ((double)i + ((double)ia + 0.5 + J0) / px) * sp.dx;
        const double v = sp.vmin[0] + ((double)j + ((double)ib + 0.5 + J1) / pv) * sp.dv[0];
        const double mu = a.mu[m];
        double B = 0.0, Mb[4], tb[4];
        for (int b = 0; b < nb; ++b) {
            const double sd = f0->beam_vth[b][0];
            tb[b] = (v - f0->beam_u[b][0]) / sd;
            Mb[b] = f0->beam_n[b] * exp(-0.5 * tb[b] * tb[b]) / (sqrt(2.0 * M_PI) * sd);
            B += Mb[b];
        }
        double pert = 1.0;
        for (int q = 0; q < nm; ++q) {
            const double c = cos(2.0 * M_PI * f0->mode[q] * x / L + f0->phase[q]);
            pert += f0->amp[q] * c;
            acc[q] += mu * B * c;
        }
        for (int b = 0; b < nb; ++b) acc[nm + b] += mu * pert * Mb[b] * tb[b] / f0->beam_vth[b][0];
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int t = 0; t < nt; ++t) {
        double v = acc[t];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) red[t][warp] = v;
    }
    __syncthreads();
    if (threadIdx.x < nt) {
        double v = 0.0;
        for (int w = 0; w < 8; ++w) v += red[threadIdx.x][w];
        atomicAdd(D->grad + threadIdx.x, v);
    }
}

// ---------------------------------------------------------------------------
// host: buffers and the passes
// ---------------------------------------------------------------------------
struct AdjEngine {
    int prec = -1, ns = 0, K = 0, C = 0, nx = 0;
    long long n[MAXS] = {};
    std::vector<void*> mem;
    AdjDev h{};
    AdjDev* d = nullptr;
    avl_f0* d_f0 = nullptr;
    // one full segment of K steps, forward (with pushes) and backward,
    // recorded once and replayed for every full segment
    cudaGraphExec_t g_fwd = nullptr, g_rec = nullptr, g_bwd = nullptr;
    int g_K = 0, g_nact = -1;
};

static cudaError_t grab(AdjEngine* E, void** p, size_t bytes)
{
    cudaError_t e = cudaMalloc(p, std::max<size_t>(bytes, 16));
    if (e == cudaSuccess) E->mem.push_back(*p);
    return e;
}

static void drop_graphs(AdjEngine* E)
{
    if (E->g_fwd) cudaGraphExecDestroy(E->g_fwd);
    if (E->g_rec) cudaGraphExecDestroy(E->g_rec);
    if (E->g_bwd) cudaGraphExecDestroy(E->g_bwd);
    E->g_fwd = E->g_rec = E->g_bwd = nullptr;
}

void adjoint_free(AdjEngine* E)
{
    if (!E) return;
    drop_graphs(E);
    for (void* p : E->mem) cudaFree(p);
    delete E;
}

static int grid_for(long long n) { return (int)std::max<long long>(1, std::min<long long>((n + 255) / 256, 152ll * 8)); }

// blocks of the finalize: eight columns and a group of rows each
static dim3 fin_grid(const AdjEngine* E, int species)
{
    const int xb = (E->nx + 7) / 8;
    return dim3(xb, species, std::max(1, std::min(64, (4 * 152 + xb - 1) / xb)));
}

static long long nmax_active(const AdjEngine* E)
{
    long long nmax = 0;
    for (int k = 0; k < E->h.nact; ++k) nmax = std::max(nmax, E->n[E->h.act[k]]);
    return nmax;
}

template <typename T>
static void launch_dep(const AdjEngine* E, long long nmax, int species, int slot, int all, cudaStream_t st)
{
    const dim3 g(grid_for(nmax), species);
    if constexpr (sizeof(T) == 8)
        k_ad_depx<<<g, 256, 0, st>>>(E->d, E->nx, slot, all);
    else
        k_ad_dep<<<g, 256, 0, st>>>(E->d, E->nx, slot, all);
}

// the Poisson solve of Eq. 6 (P rho; the backward pass applies it to e):
// the circulant product with the Green's function on many blocks where the
// context has the table, else the single-block FFT
static cudaError_t solve(const StepArgs& h, const double* in, double* out, int nx, cudaStream_t st)
{
    if (h.fd.green) return launch_poisson_dense(in, out, nx, h.fd.green, st);
    return launch_poisson(in, out, nx, h.fd.tw, h.fd.gmul, st);
}

// reconstruction of the stepped species at slot, rho = static + theirs, E
template <typename T>
static cudaError_t recon_and_field(const StepArgs& h, const StepArgs* dA, AdjEngine* E, int slot, cudaStream_t st)
{
    cudaError_t e = cudaMemcpyAsync(E->h.rho, E->h.rho_static, (size_t)E->nx * 8, cudaMemcpyDeviceToDevice, st);
    if (e) return e;
    launch_dep<T>(E, nmax_active(E), E->h.nact, slot, 0, st);
    k_ad_fin<T><<<fin_grid(E, E->h.nact), 256, 0, st>>>(dA, E->d, slot, 0);
    if ((e = cudaGetLastError())) return e;
    return solve(h, E->h.rho, E->h.hE + (size_t)slot * E->nx, E->nx, st);
}

// FP32: F of slot 0 becomes the reference of the numerators of species s
static cudaError_t keep_reference(const StepArgs& h, AdjEngine* E, int s, cudaStream_t st)
{
    return cudaMemcpyAsync(E->h.sp[s].fref, E->h.sp[s].hF, (size_t)E->nx * h.sp[s].nv[0] * 4, cudaMemcpyDeviceToDevice, st);
}

// charge of the species that are not stepped (immobile, not theta): once
template <typename T>
static cudaError_t static_charge(const StepArgs& h, AdjEngine* E, const StepArgs* dA, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(E->h.rho_static, 0, (size_t)E->nx * 8, st);
    if (e || E->h.nstat == 0) return e;
    long long nmax = 0;
    for (int k = 0; k < E->h.nstat; ++k) nmax = std::max(nmax, E->n[E->h.stat[k]]);
    std::swap(E->h.rho, E->h.rho_static);   // k_ad_fin adds into D->rho
    if ((e = cudaMemcpyAsync(E->d, &E->h, sizeof(AdjDev), cudaMemcpyHostToDevice, st))) return e;
    for (int pass = sizeof(T) == 4 ? 0 : 1; pass < 2; ++pass) {   // FP32: the reference first
        launch_dep<T>(E, nmax, E->h.nstat, 0, 1, st);
        k_ad_fin<T><<<fin_grid(E, E->h.nstat), 256, 0, st>>>(dA, E->d, 0, 1);
        if ((e = cudaGetLastError())) return e;
        if (pass) break;
        for (int k = 0; k < E->h.nstat; ++k)
            if ((e = keep_reference(h, E, E->h.stat[k], st))) return e;
        if ((e = cudaMemsetAsync(E->h.rho, 0, (size_t)E->nx * 8, st))) return e;
    }
    std::swap(E->h.rho, E->h.rho_static);
    return cudaMemcpyAsync(E->d, &E->h, sizeof(AdjDev), cudaMemcpyHostToDevice, st);
}

template <typename T>
static cudaError_t push_slot(AdjEngine* E, int slot, cudaStream_t st)
{
    const bool staged = sizeof(T) == 4 && E->nx <= AD_PUSH_NX;
    k_ad_push<T><<<dim3(grid_for(nmax_active(E)), E->h.nact), 256, staged ? E->nx * 4 : 0, st>>>(E->d, E->nx, slot, staged);
    return cudaGetLastError();
}

template <typename T>
static cudaError_t back_step(const StepArgs& h, const StepArgs* dA, AdjEngine* E, int slot, int terminal, cudaStream_t st)
{
    const long long nmax = nmax_active(E);
    cudaError_t e = cudaMemsetAsync(E->h.e, 0, (size_t)E->nx * 8, st);
    if (e) return e;
    const size_t copy_bytes = (size_t)E->nx * sizeof(T);
    int copies = 32;
    while (copies && copies * copy_bytes > AD_E_SMEM) copies >>= 1;
    if ((e = raise_smem_limit(k_ad_e<T>, (int)(copies * copy_bytes)))) return e;
    const int blocks = (int)std::min<long long>((nmax + AD_E_THREADS - 1) / AD_E_THREADS, sizeof(T) == 4 ? 304 : 152);
    k_ad_e<T><<<dim3(blocks, E->h.nact), AD_E_THREADS, copies * copy_bytes, st>>>(E->d, E->nx, h.fd.dx, slot, terminal,
                                                                                     copies);
    if ((e = cudaGetLastError())) return e;
    if ((e = solve(h, E->h.e, E->h.tmp, E->nx, st))) return e;
    k_ad_grid<T><<<dim3(152 * 2, E->h.nact), 256, 0, st>>>(dA, E->d, slot);
    k_ad_gather<T><<<dim3(grid_for(nmax), E->h.nact), 256, 0, st>>>(E->d, E->nx, slot, terminal);
    return cudaGetLastError();
}

template <typename T>
static cudaError_t fwd_segment(const StepArgs& h, const StepArgs* dA, AdjEngine* E, int len, bool push_last,
                               cudaStream_t st)
{
    cudaError_t e = cudaSuccess;
    for (int j = 0; j < len && !e; ++j) {
        e = recon_and_field<T>(h, dA, E, j, st);
        if (!e && (push_last || j + 1 < len)) e = push_slot<T>(E, j, st);
    }
    return e;
}

template <typename T>
static cudaError_t bwd_segment(const StepArgs& h, const StepArgs* dA, AdjEngine* E, int len, cudaStream_t st)
{
    cudaError_t e = cudaSuccess;
    for (int j = len - 1; j >= 0 && !e; --j) e = back_step<T>(h, dA, E, j, 0, st);
    return e;
}

// record `body` (launches on st) as a graph and instantiate it
template <typename F>
static cudaError_t record(cudaStream_t st, cudaGraphExec_t* out, F body)
{
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal);
    if (e) return e;
    cudaError_t eb = body();
    e = cudaStreamEndCapture(st, &g);
    if (eb || e) {
        if (g) cudaGraphDestroy(g);
        return eb ? eb : e;
    }
    e = cudaGraphInstantiate(out, g, 0);
    cudaGraphDestroy(g);
    return e;
}

// full segments replay the recorded graphs (kernel attributes are set by a
// first direct launch before any recording)
template <typename T>
static cudaError_t full_fwd(const StepArgs& h, const StepArgs* dA, AdjEngine* E, bool push_last, cudaStream_t st)
{
    const int K = E->K;
    if (!push_last) return fwd_segment<T>(h, dA, E, K, false, st);
    if (!E->g_fwd) {
        cudaError_t e = record(st, &E->g_fwd, [&] { return fwd_segment<T>(h, dA, E, K, true, st); });
        if (e) return e;
    }
    return cudaGraphLaunch(E->g_fwd, st);
}

// a full segment again from its checkpoint, in the fields of the forward pass
// (hE): the same trajectories to the bit
template <typename T>
static cudaError_t recompute(const StepArgs& h, const StepArgs* dA, AdjEngine* E, cudaStream_t st)
{
    if (!E->g_rec) {
        cudaError_t e = record(st, &E->g_rec, [&] {
            cudaError_t r = cudaSuccess;
            for (int j = 0; j < E->K && !r; ++j) {
                launch_dep<T>(E, nmax_active(E), E->h.nact, j, 0, st);
                k_ad_fin<T><<<fin_grid(E, E->h.nact), 256, 0, st>>>(dA, E->d, j, 0);
                r = cudaGetLastError();
                if (!r && j + 1 < E->K) r = push_slot<T>(E, j, st);
            }
            return r;
        });
        if (e) return e;
    }
    return cudaGraphLaunch(E->g_rec, st);
}

template <typename T>
static cudaError_t full_bwd(const StepArgs& h, const StepArgs* dA, AdjEngine* E, cudaStream_t st)
{
    if (!E->g_bwd) {
        cudaError_t e = record(st, &E->g_bwd, [&] { return bwd_segment<T>(h, dA, E, E->K, st); });
        if (e) return e;
    }
    return cudaGraphLaunch(E->g_bwd, st);
}

// copy the state of slot a (positions, velocities) of every species into the
// checkpoint c (to_ckpt) or back from it into slot a
static cudaError_t ckpt_copy(AdjEngine* E, int c, int a, bool to_ckpt, cudaStream_t st)
{
    const size_t pb = E->prec == AVL_FP32 ? 4 : 8;
    for (int s = 0; s < E->ns; ++s) {
        const AdjSp& q = E->h.sp[s];
        const size_t n = (size_t)q.n;
        auto cp = [&](void* ck, void* hs, size_t eb) {
            char* cptr = static_cast<char*>(ck) + (size_t)c * n * eb;
            char* hptr = static_cast<char*>(hs) + (size_t)a * n * eb;
            return to_ckpt ? cudaMemcpyAsync(cptr, hptr, n * eb, cudaMemcpyDeviceToDevice, st)
                           : cudaMemcpyAsync(hptr, cptr, n * eb, cudaMemcpyDeviceToDevice, st);
        };
        cudaError_t e = cp(q.cx, q.hx, pb);
        if (!e && E->prec == AVL_FP32) e = cp(q.coff, q.hoff, 4);
        if (!e) e = cp(q.cv, q.hv, pb);
        if (e) return e;
    }
    return cudaSuccess;
}

template <typename T>
static cudaError_t run(const StepArgs& h, const StepArgs* dA, AdjEngine* E, int nsteps, cudaStream_t st,
                       double* grad_host, int ngrad, double* J)
{
    cudaError_t e;
    const int K = E->K;
    if (E->g_K != K || E->g_nact != E->h.nact) {
        drop_graphs(E);
        E->g_K = K;
        E->g_nact = E->h.nact;
    }
    // initial state into slot 0
    for (int s = 0; s < E->ns; ++s) {
        k_ad_init<T><<<grid_for(E->n[s]), 256, 0, st>>>(dA, E->d, s);
        if ((e = cudaGetLastError())) return e;
    }
    if constexpr (sizeof(T) == 4)
        for (int s = 0; s < E->ns; ++s)
            if ((e = cudaMemsetAsync(E->h.sp[s].fref, 0, (size_t)E->nx * h.sp[s].nv[0] * 4, st))) return e;
    if ((e = static_charge<T>(h, E, dA, st))) return e;
    if constexpr (sizeof(T) == 4) {
        if ((e = recon_and_field<T>(h, dA, E, 0, st))) return e;
        for (int k = 0; k < E->h.nact; ++k)
            if ((e = keep_reference(h, E, E->h.act[k], st))) return e;
    }
    if ((e = cudaMemsetAsync(E->h.grad, 0, 8 * (64 + 4), st))) return e;
    // forward: segments of K steps; checkpoint c = state c K
    const int nseg = std::max(1, (nsteps + K - 1) / K);
    int last_len = nsteps;
    for (int c = 0; c < nseg; ++c) {
        const int len = std::min(K, nsteps - c * K);
        if ((e = ckpt_copy(E, c, 0, true, st))) return e;
        if (len == K && c > 0) {
            if ((e = full_fwd<T>(h, dA, E, true, st))) return e;
        } else if ((e = fwd_segment<T>(h, dA, E, len, true, st))) {
            return e;
        }
        last_len = len;
        if ((e = cudaMemcpyAsync(E->h.allE + (size_t)c * K * E->nx, E->h.hE, (size_t)len * E->nx * 8,
                                 cudaMemcpyDeviceToDevice, st)))
            return e;
        if (c + 1 < nseg && (e = ckpt_copy(E, c + 1, len, true, st))) return e;
        if (c + 1 < nseg && (e = ckpt_copy(E, c + 1, 0, false, st))) return e;
    }
    if (nsteps == 0) last_len = 0;
    // final state: its field and J, then the backward walk of the last segment
    if ((e = recon_and_field<T>(h, dA, E, last_len, st))) return e;
    std::vector<double> Ef(E->nx);
    if ((e = cudaMemcpyAsync(Ef.data(), E->h.hE + (size_t)last_len * E->nx, E->nx * 8, cudaMemcpyDeviceToHost, st)))
        return e;
    if ((e = back_step<T>(h, dA, E, last_len, 1, st))) return e;
    if ((e = bwd_segment<T>(h, dA, E, last_len, st))) return e;
    // earlier segments: recompute from the checkpoint, then walk back
    for (int c = nseg - 2; c >= 0; --c) {
        if ((e = ckpt_copy(E, c, 0, false, st))) return e;
        if ((e = cudaMemcpyAsync(E->h.hE, E->h.allE + (size_t)c * K * E->nx, (size_t)K * E->nx * 8,
                                 cudaMemcpyDeviceToDevice, st)))
            return e;
        if ((e = recompute<T>(h, dA, E, st))) return e;
        if ((e = full_bwd<T>(h, dA, E, st))) return e;
    }
    k_ad_theta<T><<<grid_for(E->n[E->h.theta_s]), 256, 0, st>>>(dA, E->d);
    if ((e = cudaGetLastError())) return e;
    if ((e = cudaMemcpyAsync(grad_host, E->h.grad, ngrad * 8, cudaMemcpyDeviceToHost, st))) return e;
    if ((e = cudaStreamSynchronize(st))) return e;
    double s2 = 0.0;
    for (int i = 0; i < E->nx; ++i) s2 += Ef[i] * Ef[i];
    *J = 0.5 * s2 * h.fd.dx;
    return cudaSuccess;
}

cudaError_t adjoint_run(AdjEngine** eng, const StepArgs& h, const StepArgs* dA, const AdjSpec& spec, cudaStream_t st,
                        double* dJ_amp, double* dJ_u, double* J)
{
    const int ns = h.ns, nx = h.fd.nx;
    const int K = std::max(1, std::min(spec.ckpt_every, std::max(1, spec.nsteps)));
    const int C = std::max(1, (spec.nsteps + K - 1) / K);
    const size_t pb = h.prec == AVL_FP32 ? 4 : 8;
    AdjEngine* E = *eng;
    bool fits = E && E->prec == h.prec && E->ns == ns && E->K >= K && E->C >= C && E->nx == nx;
    for (int s = 0; fits && s < ns; ++s) fits = E->n[s] == spec.n[s];
    if (!fits) {
        adjoint_free(E);
        *eng = nullptr;
        E = new AdjEngine();
        E->prec = h.prec;
        E->ns = ns;
        E->K = K;
        E->C = C;
        E->nx = nx;
        cudaError_t e = cudaSuccess;
        auto g = [&](void** p, size_t b) {
            if (!e) e = grab(E, p, b);
        };
        for (int s = 0; s < ns; ++s) {
            AdjSp& q = E->h.sp[s];
            const size_t n = (size_t)spec.n[s];
            const size_t cells = (size_t)nx * h.sp[s].nv[0];
            E->n[s] = spec.n[s];
            q.n = spec.n[s];
            g(&q.hx, (K + 1) * n * pb);
            q.hoff = nullptr;
            if (h.prec == AVL_FP32) g((void**)&q.hoff, (K + 1) * n * 4);
            g(&q.hv, (K + 1) * n * pb);
            g(&q.cx, C * n * pb);
            q.coff = nullptr;
            if (h.prec == AVL_FP32) g((void**)&q.coff, C * n * 4);
            g(&q.cv, C * n * pb);
            g(&q.f, n * pb);
            g(&q.lx, n * pb);
            g(&q.lv, n * pb);
            g((void**)&q.mu, n * 8);
            g(&q.num, 2 * cells * pb);
            g(&q.AB, 2 * cells * pb);
            g(&q.dE, nx * pb);
            q.fref = nullptr;
            if (h.prec == AVL_FP32) g((void**)&q.fref, cells * 4);
            g(&q.hF, (K + 1) * cells * pb);
            g(&q.hD, (K + 1) * cells * pb);
            if (!e) e = cudaMemsetAsync(q.num, 0, 2 * cells * pb, st);
        }
        g((void**)&E->h.rho, nx * 8);
        g((void**)&E->h.rho_static, nx * 8);
        g((void**)&E->h.e, nx * 8);
        g((void**)&E->h.tmp, nx * 8);
        g((void**)&E->h.hE, (size_t)(K + 1) * nx * 8);
        g((void**)&E->h.allE, ((size_t)C * K + 1) * nx * 8);
        g((void**)&E->h.grad, 8 * (64 + 4));
        g((void**)&E->d_f0, sizeof(avl_f0) * ns);
        g((void**)&E->d, sizeof(AdjDev));
        if (e) {
            adjoint_free(E);
            return e;
        }
        *eng = E;
    }
    E->h.ns = ns;
    E->h.theta_s = spec.theta_s;
    E->h.nact = 0;
    E->h.nstat = 0;
    for (int s = 0; s < ns; ++s) {
        if (h.sp[s].mobile || s == spec.theta_s)
            E->h.act[E->h.nact++] = s;
        else
            E->h.stat[E->h.nstat++] = s;
    }
    E->h.K = K;
    E->h.f0 = E->d_f0;
    for (int s = 0; s < ns; ++s) {
        AdjSp& q = E->h.sp[s];
        q.lat[0] = spec.lat[s][0];
        q.lat[1] = spec.lat[s][1];
        q.seed = spec.seed[s];
        q.jitter = spec.jitter[s];
        const SpDev& sp = h.sp[s];
        q.nv = sp.nv[0];
        q.mobile = sp.mobile;
        auto consts = [&](auto& c) {
            using T = decltype(c.va + c.va);
            c.va = (T)sp.inv_dv[0];
            c.vb = (T)(-sp.vmin[0] * sp.inv_dv[0] - 0.5);
            c.qm_dt = (T)sp.qm_dt;
            c.dt_dx = (T)sp.dt_dx;
            c.lt = (T)(sp.dt_dx * sp.dv[0]);
            c.c0 = sp.qm_dt / sp.dv[0];
        };
        consts(q.cf);
        consts(q.cd);
    }
    const int saveK = E->K;
    E->K = K;
    cudaError_t e = cudaMemcpyAsync(E->d_f0, spec.f0, sizeof(avl_f0) * ns, cudaMemcpyHostToDevice, st);
    if (!e) e = cudaMemcpyAsync(E->d, &E->h, sizeof(AdjDev), cudaMemcpyHostToDevice, st);
    if (!e) e = cudaStreamSynchronize(st);
    double grad[64 + 4] = {};
    const int nm = spec.f0[spec.theta_s].nmode, nb = spec.f0[spec.theta_s].nbeam;
    if (!e)
        e = h.prec == AVL_FP32 ? run<float>(h, dA, E, spec.nsteps, st, grad, nm + nb, J)
                               : run<double>(h, dA, E, spec.nsteps, st, grad, nm + nb, J);
    E->K = saveK;
    if (e) return e;
    for (int i = 0; i < nm; ++i) dJ_amp[i] = grad[i];
    for (int b = 0; b < nb; ++b) dJ_u[b] = grad[nm + b];
    return cudaSuccess;
}

}  // namespace avl
