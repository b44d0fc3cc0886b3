// k_vhs3.cu -- 1d3v kernels of the Vlasov-Hybrid time step (Fig. 2; Sec. 2
// with three velocity dimensions).
//
// Without a magnetic field the field changes v_x only and v_y, v_z ride
// along unchanged.  Layout: markers sorted by pencil (the dual rows of v_y and
// v_z, fixed for the life of a marker) and inside a pencil by key (dual row
// of v_x + 1).  One CTA owns one pencil and walks its keys in order; per
// segment (the markers stored under one key):
//   push    gather E (cloud-in-cell, Sec. 2), v_x += (q/m) E dt, x += v_x dt,
//           written back in place
//   sort    the markers whose new key is still the segment's key ("stays")
//           are counting-sorted by their x dual cell in shared memory
//   gather  one thread per x column adds the 16 cloud-in-cell weights (Eq. 4
//           numerator alpha f and denominator alpha) of the markers of its
//           two dual cells into registers: rows j, j+1 of v_x times the
//           pencil's four (v_y, v_z) cells -- no atomics.  FP64 (k_pd3x):
//           the sums in 64-bit integers (fixed.cuh), since an FP64 warp
//           instruction costs its SM sub-partition 64 clocks
//   flush   a finished v_x row is added into the global accumulators; each
//           cell receives the sums of the four pencils that reach it
// Markers whose key moved since the last re-sort deposit their 16
// contributions through global reductions, one thread per contribution;
// their counts decide the next re-sort (k_sort3, per pencil, into the other
// buffer).  k_fin3 forms f = num / den, the moment (Eq. 14) and the
// diagnostics (Sec. 3.4.1) and clears the other accumulator.
//
// With a static background magnetic field (Sec. 3.2: the Boris push of the
// 1d3v version) every velocity component turns, so a marker's pencil changes
// from step to step.  The step is then: Boris push in place with the count of
// every marker's new (pencil, key) bucket (k_bpush3), a global counting sort
// into the other buffer (k_src3_tsum, k_src3_scan, k_rs3_scatter,
// k_src3_flip), and the pencil deposit above without a push (k_pd3 mode 2),
// in which no marker is off its segment.
#include <math.h>

#include <algorithm>

#include "avl_internal.cuh"
#include "common.cuh"
#include "ptx.cuh"

namespace avl {

// position type of the 1d3v kernels (common.cuh): FP32 int cell + FP32
// offset, FP64 PosX
template <typename T>
using Pos3 = PosM<T>;

template <typename T>
__device__ __forceinline__ Pos3<T> pos3_from_cells(double xi, int nx)
{
    return posm_from_cells<T>(xi, nx);
}


__device__ __forceinline__ int species_of_pen(const StepArgs* A, int g)
{
    int s = 0;
    while (s + 1 < A->ns && g >= A->sp[s + 1].pen_base) ++s;
    return s;
}

__device__ __forceinline__ int species_of_fin3(const StepArgs* A, int g)
{
    int s = 0;
    while (s + 1 < A->ns && g >= A->sp[s + 1].fin_base) ++s;
    return s;
}

// Dual row of a velocity component on a grid of n cells: t = v a + b with
// a = 1/dv and b = -vmin/dv - 1/2 (the cloud-in-cell rule of Fig. 1 on a
// cell-centred grid).  Returns floor(t) limited to [-2, n] (-2 and n: the
// footprint misses the grid) and the weight w = t - floor(t) of row j + 1.
// One explicit fused multiply-add, so that every kernel finds the same row.
__device__ __forceinline__ int dual3(float v, float a, float b, int n, float& w)
{
    const float t = __fmaf_rn(v, a, b);
    if (!(t > -2.0f && t < (float)n)) {
        w = 0.0f;
        return t > 0.0f ? n : -2;
    }
    const float fl = floorf(t);
    w = t - fl;
    return (int)fl;
}
// FP64: a and b come scaled by 2^52, so that t 2^52 rounds to a
// 64-bit count of 2^-52 rows in one saturating conversion (NaN gives 0); the
// row is its high bits and the weight its low 52 bits
__device__ __forceinline__ int dual3(double v, double a52, double b52, int n, long long& w)
{
    const long long t = __double2ll_rn(__fma_rn(v, a52, b52));
    const int fl = (int)(t >> 52);
    if (fl < -2 || fl >= n) {
        w = 0;
        return fl < 0 ? -2 : n;
    }
    w = t & (FX_ONE - 1);
    return fl;
}
// type of dual3's weight: a float, or a count of 2^-52
template <typename T>
struct DualW {
    using type = float;
};
template <>
struct DualW<double> {
    using type = long long;
};

// coefficients a, b of dual3 and cell counts of a species' velocity grid
template <typename T>
struct VCoef {
    T a[3], b[3];
    int n[3];
    __device__ __forceinline__ void init(const SpDev& sp)
    {
        const SpConst<T>& k = sp_const<T>(sp);
        for (int d = 0; d < 3; ++d) {
            a[d] = k.a[d];
            b[d] = k.b[d];
            n[d] = sp.nv[d];
        }
    }
};

__device__ __forceinline__ int key_of(int j, int n) { return clampi(j, -1, n - 1) + 1; }

// warp-aggregated slot: lanes with equal keys take consecutive slots of
// cur[key] (one atomic per distinct key in the warp); lanes with ok = false
// take part but get no slot
__device__ __forceinline__ int warp_slot(int* cur, int key, bool ok)
{
    const int kk = ok ? key : -1;
    const unsigned grp = __match_any_sync(0xffffffffu, kk);
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(grp) - 1;
    int base = 0;
    if (ok && lane == leader) base = atomicAdd(&cur[key], __popc(grp));
    base = __shfl_sync(0xffffffffu, base, leader);
    return base + __popc(grp & ((1u << lane) - 1u));
}

// exclusive scan of in[0, n) into out[0, n], out[n] = total, by a block of
// P3_THREADS threads; each thread takes `items` consecutive entries
// (items * P3_THREADS >= n); in may alias out
__device__ void block_exscan(const int* in, int* out, int n, int items, int* wsum)
{
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int i0 = t * items;
    int loc = 0;
    for (int i = 0; i < items; ++i)
        if (i0 + i < n) loc += in[i0 + i];
    int x = loc;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int w = lane < P3_THREADS / 32 ? wsum[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        if (lane < P3_THREADS / 32) wsum[lane] = w;
    }
    __syncthreads();
    int run = x - loc + (warp > 0 ? wsum[warp - 1] : 0);
    for (int i = 0; i < items; ++i)
        if (i0 + i < n) {
            const int v = in[i0 + i];
            out[i0 + i] = run;
            run += v;
        }
    if (t == P3_THREADS - 1) out[n] = run;
    __syncthreads();
}

// ---------------------------------------------------------------------------
// push + deposit
// ---------------------------------------------------------------------------
// A pencil's markers are walked in chunks of at most NB markers, each inside
// one segment; the marker fields of the next chunk are staged into shared
// memory by bulk copies (TMA) while the current one is processed.
// FP32: the fields are cell, offset, v_x, v_y, v_z, f.
struct Stage3 {
    // more than a segment of two markers per cell at nx = 256 (512, give or
    // take its square root), so that few segments take a second chunk
    static constexpr int NB = 640;
    static constexpr int MPT = (NB + P3_THREADS - 1) / P3_THREADS;
    // movers of a chunk kept in shared memory (the others are deposited by their
    // own threads; 16.8 M markers, steps of 0.2 and 0.5: 1.16 and 1.58 ms with 64
    // and one corner at a time, 0.86 and 1.18 ms; 192 cost the third CTA's L1)
    static constexpr int NM = 128;
    static constexpr int NF = 6;
    static constexpr int AL = 4;                             // markers per 16 bytes
    static constexpr int SLEN = NB + 2 * AL;                 // staged entries per field
};

// FP64 (k_pd3x), markers per chunk: more than a segment of two markers per
// cell at nx = 256 (512, give or take its square root), so that few segments
// take a second chunk (longer ones, as of larger nx or more markers per cell,
// walk two or more), and two CTAs per SM with the shared memory it needs
// (98 KB).  64^3 bump-on-tail: 8.29 ms with 640 or 576, 8.40 with 544.
constexpr int NB3X = 640;
constexpr int MPT3X = (NB3X + P3_THREADS - 1) / P3_THREADS;

// x columns per thread of a pencil's block
static int cpt_of(int nx) { return nx <= P3_THREADS ? 1 : (nx <= 2 * P3_THREADS ? 2 : 4); }

size_t pd3_smem_bytes(int nx, int nkey, int prec)
{
    size_t b;
    if (prec == AVL_FP32) {
        using S = Stage3;
        b = 2 * (size_t)S::NF * S::SLEN * 4;                   // two staging buffers
        b += 32 * (size_t)S::NB + 4 * ((size_t)nx + 2) + 64 * (size_t)S::NM;   // sorted payload, E, movers
        b += 8 * (size_t)(P3_THREADS * cpt_of(nx) - nx);       // bins beyond nx
    } else {
        b = 5 * (NB3X + 4) * 8 + 96 * NB3X + 32;                  // staging (w_y, w_z, X, v_x, f), sorted payload
        b += 16 * (size_t)nx;                                  // kick
        b += 16 * (size_t)nx + 8 * (size_t)P3_THREADS;         // exponents, bins beyond nx
    }
    b += 4 * (2 * (size_t)nx + 1) + 4 * ((size_t)nkey + 2) + 64;   // histogram, bin starts, segment row
    return (b + 15) / 16 * 16;
}

// largest key count (nv[0] + 1) over the species of a context
static int nkey_max(const StepArgs& h)
{
    int m = 2;
    for (int s = 0; s < h.ns; ++s) m = std::max(m, h.sp[s].nv[0] + 1);
    return m;
}

// weights of the pencil's four (v_y, v_z) cells: (jy, jz), (jy+1, jz),
// (jy, jz+1), (jy+1, jz+1)
template <typename T>
__device__ __forceinline__ void plane_weights(T wy, T wz, T (&q)[4])
{
    const T ya = (T)1 - wy, za = (T)1 - wz;
    q[0] = ya * za;
    q[1] = wy * za;
    q[2] = ya * wz;
    q[3] = wy * wz;
}

// FP64: the (v_y, v_z) weights of a marker as counts of 2^-52, stored beside
// it (they change only when a magnetic field turns v); -1 when its footprint
// misses the grid in v_y or v_z (such a marker sits in a clamped pencil and
// deposits nothing)
__device__ __forceinline__ longlong2 marker_wyz(const VCoef<double>& vc, double vy, double vz)
{
    long long wy, wz;
    const int jy = dual3(vy, vc.a[1], vc.b[1], vc.n[1], wy);
    const int jz = dual3(vz, vc.a[2], vc.b[2], vc.n[2], wz);
    if (jy < -1 || jy >= vc.n[1] || jz < -1 || jz >= vc.n[2]) return make_longlong2(-1, -1);
    return make_longlong2(wy, wz);
}

// FP64: the weights of the pencil's four (v_y, v_z) cells in units of 2^-56
// from the marker's (v_y, v_z) weights: one product, the others by
// difference (none negative, sum exactly one)
__device__ __forceinline__ void plane_weights(longlong2 w, long long (&q)[4])
{
    if (w.x < 0) {
        q[0] = q[1] = q[2] = q[3] = 0;
        return;
    }
    const long long y = w.x << 4, z = w.y << 4;
    const long long yz = (long long)((__umul64hi((unsigned long long)w.x << 8, (unsigned long long)w.y << 9) + 1) >> 1);
    q[0] = (FX_ONE << 4) - y - z + yz;
    q[1] = y - yz;
    q[2] = z - yz;
    q[3] = yz;
}

// the pencil's four (v_y, v_z) planes: first grid offset of each (row 0,
// column 0) and whether it lies on the grid
struct Planes {
    int base[4];
    bool ok[4];
};

// A marker whose v_x dual row j is not its segment's deposits its 16
// cloud-in-cell contributions apart from the gather, straight into the
// global accumulator.  This is one of them: corner bits x (bit 0), v_x row
// (bit 1), (v_y, v_z) plane (bits 2-3).
__device__ __forceinline__ void deposit_corner(float* gacc, int cells, const Planes& pl, int nx, int nvx, int bin,
                                               float u, int j, float w, float wy, float wz, float f, int corner)
{
    const int cx = corner & 1, cv = (corner >> 1) & 1, q = corner >> 2;
    const bool okq = q == 0 ? pl.ok[0] : q == 1 ? pl.ok[1] : q == 2 ? pl.ok[2] : pl.ok[3];
    const int row = j + cv;
    if (!okq || row < 0 || row >= nvx) return;
    const float ay = (q & 1) ? wy : 1.f - wy, az = (q & 2) ? wz : 1.f - wz;
    const int x = cx ? (bin + 1 == nx ? 0 : bin + 1) : bin;
    const float ax = cx ? u : 1.f - u;
    const float a = ax * (cv ? w : 1.f - w) * (ay * az);
    if (a == 0.f) return;
    const int base = q == 0 ? pl.base[0] : q == 1 ? pl.base[1] : q == 2 ? pl.base[2] : pl.base[3];
    const int o = base + row * nx + x;
    atomicAdd(gacc + o, a * f);
    atomicAdd(gacc + cells + o, a);
}

// exclusive scan of hist[0, 256 CPT) into start[0, 256 CPT]: every warp sums
// the bins in registers (8 CPT per lane) and writes its share, so that the
// scan takes no barrier of its own
template <int CPT>
__device__ __forceinline__ void bin_scan(const int* hist, int* start)
{
    constexpr int PER = 8 * CPT;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int v[PER], sum = 0;
#pragma unroll
    for (int i = 0; i < PER; i += 4) {
        const int4 h = reinterpret_cast<const int4*>(hist)[(lane * PER + i) / 4];
        v[i] = h.x;
        v[i + 1] = h.y;
        v[i + 2] = h.z;
        v[i + 3] = h.w;
        sum += h.x + h.y + h.z + h.w;
    }
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if ((lane >> 2) == warp) {   // a warp's share: 32 CPT bins of four lanes
        int run = incl - sum;
#pragma unroll
        for (int i = 0; i < PER; i += 4) {
            const int4 b = make_int4(run, run + v[i], run + v[i] + v[i + 1], run + v[i] + v[i + 1] + v[i + 2]);
            reinterpret_cast<int4*>(start)[(lane * PER + i) / 4] = b;
            run = b.w + v[i + 3];
        }
        if (lane == 31) start[P3_THREADS * CPT] = run;
    }
}

// two FP32 values in one register pair: one packed instruction for both lanes
// of a product or sum, each rounded as by itself
using F2 = unsigned long long;
__device__ __forceinline__ F2 f2_dup(float v)
{
    F2 r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float2 f2_get(F2 v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ void f2_fma(F2& c, F2 a, F2 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b)); }

// mode 0: deposit of the current markers of every species (refresh);
// mode 1: push of the mobile species, then deposit of the new state;
// mode 2: deposit of the mobile species (pushed and re-sorted before).
// PUSH (mode 1) is a template parameter so that the deposit-only instances
// keep their own registers (one column per thread: three CTAs per SM; four
// without the push took 2.25 ms against 2.20, at 64 registers).
//
// Bound by the latency of its phases: 24 warps per SM, issue slots 46 % busy,
// three barriers and 400 warp instructions per 32 markers, a quarter of them in
// the gather, whose warps run as long as their fullest column (8 markers where
// the mean is 4).  So: a chunk takes a whole segment (640 markers; at 512 half
// of them took a second chunk), the bins are scanned by every warp without a
// barrier of its own, the row of a finished segment leaves from the registers
// of the gather, a marker's payload is two 16-byte words, the sums are packed
// FP32 pairs (one instruction for two planes) and the pencil of a marker is
// checked by comparing, not by taking the floor.  134 M markers, 256 x 64^3:
// with the push 3.48 -> 2.70 ms, without 2.57 -> 2.11 ms.  Left out: the loop
// over a column's markers run to the warp's longest with weights of zero
// (2.80 ms; unrolled by two 2.82, by four 2.92), two markers at a time (2.87),
// four CTAs per SM with the push (3.17, at 64 registers it spills).
template <int CPT, bool PUSH>
__global__ void __launch_bounds__(P3_THREADS, CPT == 1 ? 3 : (CPT == 2 ? 2 : 1))
    k_pd3(const StepArgs* __restrict__ A, int mode)
{
    using T = float;
    using S = Stage3;
    constexpr int MPT = S::MPT, NB = S::NB, NF = S::NF, AL = S::AL, SLEN = S::SLEN;
    constexpr int FVX = 2, FF = 5;            // staged fields of v_x and f (v_y, v_z between)
    constexpr int BINS = P3_THREADS * CPT;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint64_t bar[2];
    __shared__ unsigned long long mov_s, far_s;
    __shared__ int flag_s;
    __shared__ int nmv_s[2];
    __shared__ const void* src_s[6];

    const int g = blockIdx.x;
    const int s = species_of_pen(A, g);
    const SpDev& sp = A->sp[s];
    constexpr bool push = PUSH;   // mode == 1
    if (mode != 0 && !sp.mobile) return;
    Ctl* ctl = A->ctl;
    const long long wait_first = ctl->wait_limit;
    const int p = g - sp.pen_base;
    const int nx = sp.nx, nvx = sp.nv[0], nvy = sp.nv[1], nvz = sp.nv[2], nkey = sp.nkey;
    const int pjy = p % (nvy + 1) - 1, pjz = p / (nvy + 1) - 1;
    const int cb = ctl->cur[s];
    const int cells = sp.nvflat * nx;
    T* const gacc = reinterpret_cast<T*>(sp.acc[ctl->asel[s]]);
    const int* segg = sp.seg[cb] + (size_t)p * (nkey + 1);

    // shared memory: staging | payload (2 x 16 bytes x NB) | movers | hist | start | segment row | E
    T* stage = reinterpret_cast<T*>(smem);
    float4* pa = reinterpret_cast<float4*>(stage + 2 * NF * SLEN);   // u, f, w
    float4* pq = pa + NB;                                            // weights of the four planes
    float4* moved = pq + NB;                                         // movers by chunk parity, 2 x NM x (u, f, w, bin | w_y, w_z, j)
    int* hist = reinterpret_cast<int*>(moved + 4 * S::NM);
    int* start = hist + BINS;
    int* segs = start + BINS + 1;
    T* Es = reinterpret_cast<T*>(segs + nkey + 1);   // E of cells -1 .. nx

    if (threadIdx.x == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        fence_mbar_init();
        mov_s = 0;
        far_s = 0;
        flag_s = 0;
        nmv_s[0] = nmv_s[1] = 0;
        src_s[0] = sp.mx[cb];
        src_s[1] = sp.moff[cb];
        src_s[FVX] = sp.mv[cb][0];
        src_s[FVX + 1] = sp.mv[cb][1];
        src_s[FVX + 2] = sp.mv[cb][2];
        src_s[FF] = sp.mf[cb];
    }
    for (int i = threadIdx.x; i < BINS; i += P3_THREADS) hist[i] = 0;
    if (push)
        for (int i = threadIdx.x; i < nx + 2; i += P3_THREADS) Es[i] = A->fd.E32[i == 0 ? nx - 1 : (i > nx ? 0 : i - 1)];
    for (int i = threadIdx.x; i <= nkey; i += P3_THREADS) segs[i] = segg[i];
    __syncthreads();

    // bulk copy of the chunk [b, b + cnt) of every staged field into buffer bf
    auto issue = [&](int bf, int b, int cnt) {
        const int a0 = b & ~(AL - 1);
        const int a1 = (b + cnt + AL - 1) & ~(AL - 1);
        const unsigned bytes = (unsigned)(a1 - a0) * (unsigned)sizeof(T);
        mbar_arrive_expect_tx(&bar[bf], bytes * NF);
        for (int f = 0; f < NF; ++f)
            bulk_g2s(stage + (bf * NF + f) * SLEN, reinterpret_cast<const T*>(src_s[f]) + a0, bytes, &bar[bf]);
    };
    // first chunk at or after key k whose segment is not empty
    auto first_from = [&](int k, int& kb) {
        for (; k < nkey; ++k)
            if (segs[k] < segs[k + 1]) break;
        kb = k < nkey ? segs[k] : 0;
        return k;
    };
    if (threadIdx.x == 0) {
        int b;
        const int k0 = first_from(0, b);
        if (k0 < nkey) issue(0, b, min(NB, segs[k0 + 1] - b));
    }

    // cached marker pointers (in-place write back)
    T* const gvx = reinterpret_cast<T*>(sp.mv[cb][0]);
    void* const gx = sp.mx[cb];
    float* const goff = sp.moff[cb];
    VCoef<T> vc;
    vc.init(sp);
    const T qm_dt = sp.cf.qm_dt, dt_dx = sp.cf.dt_dx;
    Planes pl;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int ky = pjy + (q & 1), kz = pjz + (q >> 1);
        pl.ok[q] = ky >= 0 && ky < nvy && kz >= 0 && kz < nvz;
        pl.base[q] = pl.ok[q] ? (kz * nvy + ky) * nvx * nx : 0;
    }

    // register rows: R0 = row jseg, R1 = row jseg + 1; pair h: numerators of
    // planes 2h and 2h + 1, pair 2 + h: their denominators
    F2 R0[CPT][4], R1[CPT][4];
#pragma unroll
    for (int c = 0; c < CPT; ++c)
#pragma unroll
        for (int e = 0; e < 4; ++e) R0[c][e] = R1[c][e] = 0;
    unsigned long long nmov = 0, nfar = 0;
    int buf = 0;
    unsigned ph0 = 0, ph1 = 0;

    for (int k = 0; k < nkey; ++k) {
        const int jseg = k - 1;
        const int send = segs[k + 1];
        for (int b0 = segs[k]; b0 < send; b0 += NB) {
            const int cnt = min(NB, send - b0);
            const unsigned ph = buf ? ph1 : ph0;
            if (!mbar_wait_or_drain(&bar[buf], ph, wait_first, WAIT_LIMIT)) flag_s = 1;
            if (buf) ph1 ^= 1u; else ph0 ^= 1u;
            const T* st = stage + buf * NF * SLEN;
            float4* const mv = moved + 2 * buf * S::NM;
            const int o0 = b0 & (AL - 1);

            T pu[MPT], pw[MPT], py[MPT], pz[MPT];
            int pslot[MPT];   // x dual cell | place among its markers << 16
#pragma unroll
            for (int m = 0; m < MPT; ++m) {
                pslot[m] = -1;
                const int i = m * P3_THREADS + threadIdx.x;
                if (i >= cnt) continue;
                const int si = o0 + i;
                const int idx = b0 + i;
                Pos3<T> pos;
                pos.c = reinterpret_cast<const int*>(st)[si];
                pos.o = st[SLEN + si];
                T vx = st[FVX * SLEN + si];
                if (push) {
                    int i0;
                    T wx;
                    pos.cic(i0, wx);
                    i0 = min(max(i0 + 1, 0), nx);
                    const T El = ((T)1 - wx) * Es[i0] + wx * Es[i0 + 1];
                    vx = vx + qm_dt * El;
                    pos.drift(vx * dt_dx, nx);
                    reinterpret_cast<int*>(gx)[idx] = pos.c;
                    goff[idx] = pos.o;
                    gvx[idx] = vx;
                }
                // the (v_y, v_z) dual cells, checked against the pencil
                const T vy = st[(FVX + 1) * SLEN + si], vz = st[(FVX + 2) * SLEN + si];
                const T ty = __fmaf_rn(vy, vc.a[1], vc.b[1]), tz = __fmaf_rn(vz, vc.a[2], vc.b[2]);
                const T tx = __fmaf_rn(vx, vc.a[0], vc.b[0]);
                const T wy = ty - (T)pjy, wz = tz - (T)pjz;
                T w = tx - (T)jseg;
                if (!(ty >= (T)pjy && ty < (T)(pjy + 1) && tz >= (T)pjz && tz < (T)(pjz + 1))) {
                    // outside the pencil only when the footprint misses the grid
                    T d;
                    const int jy = dual3(vy, vc.a[1], vc.b[1], vc.n[1], d), jz = dual3(vz, vc.a[2], vc.b[2], vc.n[2], d);
                    if (jy >= -1 && jy < nvy && jz >= -1 && jz < nvz) flag_s |= 2;
                    continue;
                }
                const bool stays = tx >= (T)jseg && tx < (T)(jseg + 1);
                int jx = jseg;
                if (!stays) {
                    jx = dual3(vx, vc.a[0], vc.b[0], nvx, w);
                    if (jx < -1 || jx >= nvx) continue;
                }
                int i0;
                T u;
                pos.cic(i0, u);
                int bin = i0 < 0 ? i0 + nx : i0;
                bin = min(max(bin, 0), nx - 1);
                if (stays) {
                    pslot[m] = bin | (atomicAdd(&hist[bin], 1) << 16);
                } else {
                    // off its segment's row: kept for the whole block, which
                    // deposits the chunk's few such markers after the sort
                    ++nmov;
                    if (jx > jseg + 1 || jx < jseg - 1) ++nfar;
                    const T f = st[FF * SLEN + si];
                    const int o = atomicAdd(&nmv_s[buf], 1);
                    if (o < S::NM) {
                        mv[2 * o] = make_float4(u, f, w, __int_as_float(bin));
                        mv[2 * o + 1] = make_float4(wy, wz, __int_as_float(jx), 0.f);
                    } else if constexpr (PUSH) {
                        const int x1 = bin + 1 == nx ? 0 : bin + 1;
#pragma unroll 1
                        for (int q = 0; q < 4; ++q) {
                            const bool okq = q == 0 ? pl.ok[0] : q == 1 ? pl.ok[1] : q == 2 ? pl.ok[2] : pl.ok[3];
                            if (!okq) continue;
                            const int base = q == 0 ? pl.base[0] : q == 1 ? pl.base[1] : q == 2 ? pl.base[2] : pl.base[3];
                            const float p = ((q & 1) ? wy : 1.f - wy) * ((q & 2) ? wz : 1.f - wz);
                            float* g = gacc + base + jx * nx;
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const float al = (k & 1 ? u : 1.f - u) * (k & 2 ? w : 1.f - w) * p;
                                const int row = jx + (k >> 1);
                                if (al == 0.f || row < 0 || row >= nvx) continue;
                                float* const gg = g + (k >> 1) * nx + (k & 1 ? x1 : bin);
                                atomicAdd(gg, al * f);
                                atomicAdd(gg + cells, al);
                            }
                        }
                    } else {   // (the instance without the push has hardly any; its registers)
#pragma unroll 1
                        for (int c = 0; c < 16; ++c)
                            deposit_corner(gacc, cells, pl, nx, nvx, bin, u, jx, w, wy, wz, f, c);
                    }
                }
                pu[m] = u;
                pw[m] = w;
                py[m] = wy;
                pz[m] = wz;
            }
            __syncthreads();
            // stage the next chunk into the other buffer (every thread is past
            // the previous chunk's sort, which read it)
            if (threadIdx.x == P3_THREADS - 32) {
                nmv_s[buf ^ 1] = 0;
                int nk = k, nb = b0 + NB;
                if (nb >= send) nk = first_from(k + 1, nb);
                if (nk < nkey) issue(buf ^ 1, nb, min(NB, segs[nk + 1] - nb));
            }
            const int nmv = min(nmv_s[buf], S::NM);
            bin_scan<CPT>(hist, start);
            __syncthreads();   // every warp has read the bins
#pragma unroll
            for (int c = 0; c < CPT; ++c) hist[threadIdx.x + c * P3_THREADS] = 0;
            // stays into x-sorted order
#pragma unroll
            for (int m = 0; m < MPT; ++m) {
                if (pslot[m] < 0) continue;
                const int o = start[pslot[m] & 0xffff] + (pslot[m] >> 16);
                const T f = st[FF * SLEN + o0 + m * P3_THREADS + threadIdx.x];
                T wq[4];
                plane_weights(py[m], pz[m], wq);
                pa[o] = make_float4(pu[m], f, pw[m], 0.f);
                pq[o] = make_float4(wq[0], wq[1], wq[2], wq[3]);
            }
            __syncthreads();
            // the movers: one thread per (marker, corner) into the global
            // accumulator, so that they do not hold one warp behind the others
            for (int t = threadIdx.x ^ (P3_THREADS / 2); t < nmv * 16; t += P3_THREADS) {
                const float4 a = mv[(t >> 4) * 2], b = mv[(t >> 4) * 2 + 1];
                deposit_corner(gacc, cells, pl, nx, nvx, __float_as_int(a.w), a.x, __float_as_int(b.z), a.z, b.x, b.y, a.y,
                               t & 15);
            }
            // gather: column x takes weight u from the markers of dual cell
            // x - 1 and 1 - u from those of dual cell x
#pragma unroll
            for (int c = 0; c < CPT; ++c) {
                const int x = threadIdx.x + c * P3_THREADS;
                int nup = 0, n = 0, up = 0, lo = 0;   // markers of x - 1, of both; k + up / k + lo their places
                if (x < nx) {
                    const int xm = x == 0 ? nx - 1 : x - 1, mid = start[x];
                    up = start[xm];
                    nup = start[xm + 1] - up;
                    lo = mid - nup;
                    n = nup + start[x + 1] - mid;
                }
#pragma unroll 1   // (unrolled, a warp's lanes part in the remainder: twice the iterations)
                for (int k = 0; k < n; ++k) {
                    const int i = k + (k < nup ? up : lo);
                    const float4 m = pa[i];
                    const ulonglong2 wq = *reinterpret_cast<const ulonglong2*>(pq + i);
                    const float ax = k < nup ? m.x : 1.f - m.x;
                    const float b1 = ax * m.z, b0 = ax - b1;
                    const F2 a0 = f2_dup(b0), a1 = f2_dup(b1), f0 = f2_dup(b0 * m.y), f1 = f2_dup(b1 * m.y);
                    f2_fma(R0[c][0], f0, wq.x);
                    f2_fma(R0[c][1], f0, wq.y);
                    f2_fma(R0[c][2], a0, wq.x);
                    f2_fma(R0[c][3], a0, wq.y);
                    f2_fma(R1[c][0], f1, wq.x);
                    f2_fma(R1[c][1], f1, wq.y);
                    f2_fma(R1[c][2], a1, wq.x);
                    f2_fma(R1[c][3], a1, wq.y);
                }
            }
            buf ^= 1;
        }
        // row jseg is complete (no later segment reaches it): registers into
        // the global accumulator; then rotate the rows
        if (jseg >= 0) {
#pragma unroll
            for (int c = 0; c < CPT; ++c) {
                const int x = threadIdx.x + c * P3_THREADS;
                if (x >= nx) continue;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float2 vn = f2_get(R0[c][h]), vd = f2_get(R0[c][2 + h]);
                    T* const g0 = gacc + pl.base[2 * h] + jseg * nx + x;
                    T* const g1 = gacc + pl.base[2 * h + 1] + jseg * nx + x;
                    if (pl.ok[2 * h] && vd.x != 0.f) {
                        atomicAdd(g0, vn.x);
                        atomicAdd(g0 + cells, vd.x);
                    }
                    if (pl.ok[2 * h + 1] && vd.y != 0.f) {
                        atomicAdd(g1, vn.y);
                        atomicAdd(g1 + cells, vd.y);
                    }
                }
            }
        }
#pragma unroll
        for (int c = 0; c < CPT; ++c)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                R0[c][e] = R1[c][e];
                R1[c][e] = 0;
            }
    }

    if (nmov) atomicAdd(&mov_s, nmov);
    if (nfar) atomicAdd(&far_s, nfar);
    __syncthreads();
    if (threadIdx.x == 0) {
        if (mov_s) atomicAdd(&ctl->movers[s], mov_s);
        if (far_s) atomicAdd(&ctl->far_movers[s], far_s);
        if (flag_s & 2) atomicOr(&ctl->err, ERR_CAPACITY);
        if (flag_s & 1) atomicOr(&ctl->err, ERR_TIMEOUT);
    }
}

// FP64 form of the same walk.  The FP64 pipe takes a warp instruction per 64
// clocks and sub-partition, so only the kick, the drift and the v_x row of a
// marker and the conversion of the finished sums run there (6.3 operations
// per marker); every weight and sum is a 64-bit integer (fixed.cuh).  What a
// marker gives to its two columns is worked out once, by the thread that
// sorts it into x order; the gather then is three multiply-adds per sum.  One
// thread per x column keeps the sums of its two v_x rows in registers for the
// length of a segment, in the gather as h and m (64 registers), between the
// chunks as whole units (32; two CTAs per SM at 128 registers).
//
// Bound by the latency of its phases (16 warps per SM, four barriers per
// chunk; issue slots 34 % busy, multiply-add pipe 45 %, shared memory 37 %,
// FP64 pipe 23 %).  134 M markers, 256 x 64^3: 16.95 -> 8.29 ms against the
// same sums in FP64, 8.76 ms with what keeps small cells right (SMALL3 below);
// measured and left out: balanced columns with the sums in
// shared memory (10.3 ms, its random payload reads fill the shared-memory
// pipe), two threads per column (9.5 ms), the push of the next chunk beside
// the gather (9.5 ms, its second staging buffer and tables cost more
// instructions than the barriers they save), the conversions in integers
// (8.6 ms).
//
// A weight carries an error of about a unit of 2^-57 whatever its size, once in
// the denominator of Eq. 4 and once, apart from it, in the numerator, so a
// cell that one weight a reaches would have f (1 +- 2^-57 / a).  A marker with
// a corner below SMALL3 = 2^-20 (0.5 % of markers at random places) is
// deposited corner by corner with FP64 products instead, like a mover but not
// counted as one, which leaves f and n within a few 2^-37 of those sums in
// every cell (134 M markers, 256 x 64^3: the step 9.47 -> 9.71 ms).  For the
// same reason a row's values have a unit of its own, that of the largest value
// that reaches the row in the column (one unit for both rows lost a row that
// followed a much larger one: k_pd3x 8.54 -> 8.79 ms), and a value whose
// exponent the sums do not hold goes with the small corners.
constexpr float SMALL3 = 1.0f / (1 << 20);
// Up to so many of them in a chunk take a thread per corner (8.76 ms at 134 M
// markers; a thread per marker 11.7), more a thread per marker (16.8 M markers
// on an unjittered lattice: 2.52 -> 1.96 ms)
constexpr int PARK_FEW = 48;

struct FxCol {
    long long d0[4], v0[4];   // row jseg: weights, weighted values of the four planes
    long long d1[4], v1[4];   // row jseg + 1
    int c0, c1;               // products in the sums of each row

    __device__ __forceinline__ void clear0()
    {
#pragma unroll
        for (int q = 0; q < 4; ++q) d0[q] = v0[q] = 0;
        c0 = 0;
    }
    __device__ __forceinline__ void clear1()
    {
#pragma unroll
        for (int q = 0; q < 4; ++q) d1[q] = v1[q] = 0;
        c1 = 0;
    }
    // row jseg + 1 becomes row jseg
    __device__ __forceinline__ void next_row()
    {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            d0[q] = d1[q];
            v0[q] = v1[q];
        }
        c0 = c1;
        clear1();
    }
};

__device__ __forceinline__ int4 limbs2(long long a, long long b)
{
    const Limbs A = fx_split(a), B = fx_split(b);
    return make_int4(A.h, A.l, B.h, B.l);
}

// finished sums of a cell into the global accumulator, in units of 2^-57 and
// 2^(el - 1079)
__device__ __forceinline__ void add_sums(long long d, long long v, int el, double* gacc, int cells, bool ok, int o)
{
    if (!ok || d == 0) return;
    atomicAdd(gacc + o, fx_scale((double)v, el - 1079));
    atomicAdd(gacc + cells + o, fx_scale((double)d, -57));
}

template <int CPT, bool PUSH>
__global__ void __launch_bounds__(P3_THREADS, CPT == 1 ? 2 : 1) k_pd3x(const StepArgs* __restrict__ A, int mode)
{
    constexpr int AL = 2, NB = NB3X, SLEN = NB + 2 * AL, NT = P3_THREADS;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint64_t bar;
    __shared__ unsigned long long mov_s, far_s;
    __shared__ int flag_s;
    __shared__ int nmv_s;

    const int g = blockIdx.x;
    const int s = species_of_pen(A, g);
    const SpDev& sp = A->sp[s];
    if (mode != 0 && !sp.mobile) return;
    Ctl* ctl = A->ctl;
    const long long wait_first = ctl->wait_limit;
    const int p = g - sp.pen_base;
    const int nx = sp.nx, nvx = sp.nv[0], nvy = sp.nv[1], nvz = sp.nv[2], nkey = sp.nkey;
    const int pjy = p % (nvy + 1) - 1, pjz = p / (nvy + 1) - 1;
    const int cb = ctl->cur[s];
    const int cells = sp.nvflat * nx;
    double* const gacc = reinterpret_cast<double*>(sp.acc[ctl->asel[s]]);
    const int* segg = sp.seg[cb] + (size_t)p * (nkey + 1);
    const longlong2* const wyz = sp.mwyz[cb];
    const double* const gf = reinterpret_cast<const double*>(sp.mf[cb]);

    // shared memory: staging (v_y and v_z weights, X, v_x, f) | payload
    // (arrays of limb pairs) | kick | hist | start | exponents | segment row
    longlong2* const st_w = reinterpret_cast<longlong2*>(smem);
    long long* const st_x = reinterpret_cast<long long*>(st_w + SLEN);
    double* const st_v = reinterpret_cast<double*>(st_x + SLEN);
    double* const st_f = st_v + SLEN;
    int4* pqa = reinterpret_cast<int4*>(st_f + SLEN);             // weights of planes 0 and 1
    int4* pqb = pqa + NB;                                         //            planes 2 and 3
    int4* pa = pqb + NB;       // weights of rows jseg and jseg + 1: [0, NB) in the marker's dual cell, [NB, 2 NB) in
                               // the next
    int4* pg = pa + 2 * NB + 1;    // the same times the value
    double2* kick = reinterpret_cast<double2*>(pg + 2 * NB + 1);
    int* hist = reinterpret_cast<int*>(kick + nx);   // [256 CPT]
    int* start = hist + NT * CPT;                    // [256 CPT + 1]
    int* ebin = start + NT * CPT + 1;   // [2][nx] largest exponent field of a dual cell's values, by chunk parity
    int* elc = ebin + 2 * nx;           // [nx] exponents el of a column's rows jseg (high half) and jseg + 1: their
                                        // value sums are in units of 2^(el - 1078); [nx] what this chunk adds to them
    int* segs = elc + 2 * nx;

    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
        mov_s = 0;
        far_s = 0;
        flag_s = 0;
        nmv_s = 0;
        pa[2 * NB] = pg[2 * NB] = make_int4(0, 0, 0, 0);
    }
    for (int i = threadIdx.x; i < nx; i += NT) {
        ebin[i] = ebin[nx + i] = 0;
        elc[i] = FX_EMIN << 16 | FX_EMIN;
        // kick of a marker between the centres of cells i and i + 1 with
        // weight w of cell i + 1, as c + (1 + w) d (1 + w: the bits of the
        // position): E_i + w (E_i+1 - E_i), times (q/m) dt
        if (PUSH) {
            const double Ea = A->fd.E64[i], dE = A->fd.E64[i + 1 == nx ? 0 : i + 1] - Ea;
            kick[i] = make_double2(sp.qm_dt * (Ea - dE), sp.qm_dt * dE);
        }
    }
    for (int i = threadIdx.x; i <= nkey; i += NT) segs[i] = segg[i];
    for (int i = threadIdx.x; i < NT * CPT; i += NT) hist[i] = 0;
    __syncthreads();

    double* const gvx = reinterpret_cast<double*>(sp.mv[cb][0]);
    long long* const gx = reinterpret_cast<long long*>(sp.mx[cb]);
    // bulk copy of the chunk [b, b + cnt) of every staged field
    auto issue = [&](int b, int cnt) {
        const int a0 = b & ~(AL - 1);
        const int a1 = (b + cnt + AL - 1) & ~(AL - 1);
        const unsigned bytes = (unsigned)(a1 - a0) * 8u;
        mbar_arrive_expect_tx(&bar, bytes * 5);
        bulk_g2s(st_w, wyz + a0, 2 * bytes, &bar);
        bulk_g2s(st_x, gx + a0, bytes, &bar);
        bulk_g2s(st_v, gvx + a0, bytes, &bar);
        bulk_g2s(st_f, gf + a0, bytes, &bar);
    };
    // first chunk at or after key k whose segment is not empty
    auto first_from = [&](int k, int& kb) {
        for (; k < nkey; ++k)
            if (segs[k] < segs[k + 1]) break;
        kb = k < nkey ? segs[k] : 0;
        return k;
    };
    if (threadIdx.x == 0) {
        int b;
        const int k0 = first_from(0, b);
        if (k0 < nkey) issue(b, min(NB, segs[k0 + 1] - b));
    }

    const double av = sp.cd.a[0], bv = sp.cd.b[0];
    const double dt_dx52 = sp.dt_dx * PosX::ONE;   // dt / dx in 2^-52 cells
    Planes pl;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int ky = pjy + (q & 1), kz = pjz + (q >> 1);
        pl.ok[q] = ky >= 0 && ky < nvy && kz >= 0 && kz < nvz;
        pl.base[q] = pl.ok[q] ? (kz * nvy + ky) * nvx * nx : 0;
    }

    unsigned nmov = 0, nfar = 0;
    unsigned ph = 0;   // phase of the staging barrier
    int par = 0;       // parity of the chunk
    FxCol col[CPT];
#pragma unroll
    for (int c = 0; c < CPT; ++c) {
        col[c].clear0();
        col[c].clear1();
    }

    for (int k = 0; k < nkey; ++k) {
        const int jseg = k - 1;
        const int send = segs[k + 1];
        for (int b0 = segs[k]; b0 < send; b0 += NB) {
            const int cnt = min(NB, send - b0);
            if (!mbar_wait_or_drain(&bar, ph, wait_first, WAIT_LIMIT)) flag_s = 1;
            ph ^= 1u;
            const int o0 = b0 & (AL - 1);

            long long mu[MPT3X], mw[MPT3X];
            int pbin[MPT3X], prank[MPT3X];
#pragma unroll
            for (int m = 0; m < MPT3X; ++m) {
                prank[m] = -1;
                const int i = m * NT + threadIdx.x;
                if (i >= cnt) continue;
                const int si = o0 + i;
                PosX pos;
                pos.X = st_x[si];
                double vx = st_v[si];
                if (PUSH) {
                    const long long U = pos.X - (FX_ONE >> 1);
                    int ia = (int)(U >> 52);   // -1 .. nx - 1
                    ia = min(max(ia < 0 ? ia + nx : ia, 0), nx - 1);
                    const double2 kc = kick[ia];
                    vx += __fma_rn(__longlong_as_double(0x3FF0000000000000ll | (U & (FX_ONE - 1))), kc.y, kc.x);
                    pos.drift_scaled(vx * dt_dx52, nx);
                    gx[b0 + i] = pos.X;
                    gvx[b0 + i] = vx;
                }
                const longlong2 wyz = st_w[si];
                if (wyz.x < 0) continue;   // footprint off the grid in v_y or v_z
                long long w;
                const int jx = dual3(vx, av, bv, nvx, w);
                if (jx < -1 || jx >= nvx) continue;
                const long long U = pos.X - (FX_ONE >> 1);
                int bin = (int)(U >> 52);
                bin = min(max(bin < 0 ? bin + nx : bin, 0), nx - 1);
                mu[m] = U & (FX_ONE - 1);
                mw[m] = w;
                pbin[m] = bin;
                const double f = st_f[si];
                const int ef = __double2hiint(f) >> 20 & 0x7ff;
                const int d = jx - jseg;
                const bool small =
                    lesser_weight(mu[m]) * lesser_weight(w) * (lesser_weight(wyz.x) * lesser_weight(wyz.y)) < SMALL3;
                if (d == 0 && !small && (fx_in_range(ef) | (((__double2hiint(f) & 0x7fffffff) | __double2loint(f)) == 0))) {
                    prank[m] = atomicAdd(&hist[bin], 1);
                    atomicMax(&ebin[par * nx + bin], ef);
                } else {
                    // off its segment's row, a small corner or a value beyond
                    // the sums' range: parked at the tail of the payload
                    // arrays (the stays fill them from the front) and
                    // deposited by the whole block after the sort
                    if (d != 0) ++nmov;
                    if (d > 1 || d < -1) ++nfar;
                    const int o = NB - 1 - atomicAdd(&nmv_s, 1);
                    reinterpret_cast<longlong2*>(pa)[o] = wyz;
                    reinterpret_cast<longlong2*>(pqb)[o] = make_longlong2(mu[m], w);
                    pqa[o] = make_int4(bin, jx, __double2loint(f), __double2hiint(f));
                }
            }
            __syncthreads();
            const int nmv = nmv_s;
            bin_scan<CPT>(hist, start);
            // the columns' units: those of their rows before, or of the
            // largest value of their two dual cells
#pragma unroll
            for (int c = 0; c < CPT; ++c) {
                const int x = threadIdx.x + c * NT;
                if (x >= nx) continue;
                const int et = max(ebin[par * nx + (x == 0 ? nx - 1 : x - 1)], ebin[par * nx + x]);
                const int el0 = elc[x] >> 16, el1 = elc[x] & 0xffff;
                ebin[(par ^ 1) * nx + x] = 0;   // the next chunk's
                elc[nx + x] = min(max(et - el0, 0), 63) << 16 | min(max(et - el1, 0), 63);
                elc[x] = max(el0, et) << 16 | max(el1, et);
            }
            __syncthreads();
            if (threadIdx.x == 0) nmv_s = 0;
            // the bins are counted into afresh after the next barrier
#pragma unroll
            for (int c = 0; c < CPT; ++c) hist[threadIdx.x + c * NT] = 0;
            // stays into x-sorted order
#pragma unroll
            for (int m = 0; m < MPT3X; ++m) {
                if (prank[m] < 0) continue;
                const int bin = pbin[m], o = start[bin] + prank[m], si = o0 + m * NT + threadIdx.x;
                long long q[4];
                plane_weights(st_w[si], q);
                pqa[o] = limbs2(q[0], q[1]);
                pqb[o] = limbs2(q[2], q[3]);
                // value in the unit of row jseg + 1 of the two columns; that of
                // row jseg, which holds the segment before too, is at least it
                const int bp = bin + 1 == nx ? 0 : bin + 1;
                int e;
                const long long mant = fx_value(st_f[si], e);
                const int u0 = elc[bin], u1 = elc[bp];
                const int l0 = u0 & 0xffff, l1 = u1 & 0xffff, s0 = min((u0 >> 16) - l0, 63), s1 = min((u1 >> 16) - l1, 63);
                const Limbs f0 = fx_split(mant >> min(l0 - e, 63)), f1 = fx_split(mant >> min(l1 - e, 63));
                // weights in x and v_x: one product, the others by difference
                // (none negative)
                const long long u = mu[m] << 5, w = mw[m] << 5;
                const long long a11 = fx_mul(fx_split(u), fx_split(mw[m] << 4));
                const long long a01 = w - a11;
                const long long a00 = (FX_ONE << 5) - u - a01, a10 = u - a11;
                const Limbs A00 = fx_split(a00), A01 = fx_split(a01), A10 = fx_split(a10), A11 = fx_split(a11);
                pa[o] = make_int4(A00.h, A00.l, A01.h, A01.l);
                pa[NB + o] = make_int4(A10.h, A10.l, A11.h, A11.l);
                pg[o] = limbs2(fx_mul(A00, f0) >> s0, fx_mul(A01, f0));
                pg[NB + o] = limbs2(fx_mul(A10, f1) >> s1, fx_mul(A11, f1));
            }
            __syncthreads();
            // the staging buffer is free: the next chunk into it
            if (threadIdx.x == 0) {
                int nk = k, nb = b0 + NB;
                if (nb >= send) nk = first_from(k + 1, nb);
                if (nk < nkey) issue(nb, min(NB, segs[nk + 1] - nb));
            }
            // the parked markers: one thread per (marker, corner) into the
            // global accumulator, so that a chunk's few movers do not hold one
            // warp behind the others at the chunk's barrier
            // (many of them: a thread per marker, whose neighbours in the warp
            // are near it on the grid)
            for (int t = threadIdx.x; t < nmv && nmv > PARK_FEW; t += NT) {
                const int o = NB - 1 - t;
                const int4 id = pqa[o];
                const longlong2 uw = reinterpret_cast<const longlong2*>(pqb)[o];
                const longlong2 wyz = reinterpret_cast<const longlong2*>(pa)[o];
                const double f = __hiloint2double(id.w, id.z);
                const int x1 = id.x + 1 == nx ? 0 : id.x + 1;
                double a[4];
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    a[k] = fx_scale(weight_of(uw.x, k & 1) * weight_of(uw.y, k & 2), -104);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const double q = fx_scale(weight_of(wyz.x, c & 1) * weight_of(wyz.y, c & 2), -104);
                    if (!pl.ok[c] || __double_as_longlong(q) == 0) continue;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int row = id.y + (k >> 1);
                        if (__double_as_longlong(a[k]) == 0 || row < 0 || row >= nvx) continue;
                        const double alpha = a[k] * q;
                        const int at = pl.base[c] + row * nx + (k & 1 ? x1 : id.x);
                        atomicAdd(gacc + at, alpha * f);
                        atomicAdd(gacc + cells + at, alpha);
                    }
                }
            }
            for (int t = threadIdx.x; t < nmv * 16 && nmv <= PARK_FEW; t += NT) {
                const int o = NB - 1 - (t >> 4);
                const int4 id = pqa[o];
                const longlong2 uw = reinterpret_cast<const longlong2*>(pqb)[o];
                const longlong2 wyz = reinterpret_cast<const longlong2*>(pa)[o];
                const int c = (t & 15) >> 2, row = id.y + ((t >> 1) & 1);
                const bool ok = (c == 0 ? pl.ok[0] : c == 1 ? pl.ok[1] : c == 2 ? pl.ok[2] : pl.ok[3]) && row >= 0 &&
                                row < nvx;
                const int base = c == 0 ? pl.base[0] : c == 1 ? pl.base[1] : c == 2 ? pl.base[2] : pl.base[3];
                const int x = t & 1 ? (id.x + 1 == nx ? 0 : id.x + 1) : id.x;
                const double al = (weight_of(uw.x, t & 1) * weight_of(uw.y, t & 2)) *
                                  (weight_of(wyz.x, c & 1) * weight_of(wyz.y, c & 2));
                if (!ok || __double_as_longlong(al) == 0) continue;
                const double alpha = fx_scale(al, -208);
                const int at = base + row * nx + x;
                atomicAdd(gacc + at, alpha * __hiloint2double(id.w, id.z));
                atomicAdd(gacc + cells + at, alpha);
            }
            // gather: column x takes weight u from the markers of dual cell
            // x - 1 and 1 - u from those of dual cell x
#pragma unroll
            for (int c = 0; c < CPT; ++c) {
                const int x = threadIdx.x + c * NT;
                if (x >= nx) continue;
                FxCol& C = col[c];
                const int xm = x == 0 ? nx - 1 : x - 1;
                const int lo = start[xm], nup = start[xm + 1] - lo;
                const int blo = start[x] - nup, n = nup + start[x + 1] - start[x];
                if (n == 0) continue;
                const int sh0 = elc[nx + x] >> 16, sh1 = elc[nx + x] & 0xffff;
                FxSum d0[4], v0[4], d1[4], v1[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    d0[q].h = C.d0[q];
                    v0[q].h = C.v0[q] >> sh0;
                    d1[q].h = C.d1[q];
                    v1[q].h = C.v1[q] >> sh1;
                    d0[q].m = v0[q].m = d1[q].m = v1[q].m = 0;
                }
                for (int r = 0; r < n;) {
                    const int re = min(n, r + FX_PAIRS);
                    if (C.c0 + re - r > FX_PAIRS) {   // many markers per column: the sums start again
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const int o = pl.base[q] + jseg * nx + x;
                            add_sums(d0[q].units(), v0[q].units(), elc[x] >> 16, gacc, cells, pl.ok[q] && jseg >= 0, o);
                            add_sums(d1[q].units(), v1[q].units(), elc[x] & 0xffff, gacc, cells, pl.ok[q] && jseg + 1 < nvx, o + nx);
                            d0[q].clear();
                            v0[q].clear();
                            d1[q].clear();
                            v1[q].clear();
                        }
                        C.c0 = C.c1 = 0;
                    }
                    C.c0 += re - r;
                    C.c1 += re - r;
                    // an even number of turns, the last of an odd list with
                    // weights of zero (slot Z)
                    const int re2 = re + ((re - r) & 1);
#pragma unroll 2
                    for (; r < re2; ++r) {
                        const bool upper = r < nup, in = r < n;
                        const int i = in ? r + (upper ? lo : blo) : 0;
                        const int ia = upper ? i + NB : (in ? i : 2 * NB);
                        const int4 a = pa[ia], v = pg[ia], qa = pqa[i], qb = pqb[i];
                        const Limbs Q[4] = {{qa.x, qa.y}, {qa.z, qa.w}, {qb.x, qb.y}, {qb.z, qb.w}};
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            d0[q].add({a.x, a.y}, Q[q]);
                            v0[q].add({v.x, v.y}, Q[q]);
                            d1[q].add({a.z, a.w}, Q[q]);
                            v1[q].add({v.z, v.w}, Q[q]);
                        }
                    }
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    C.d0[q] = d0[q].units();
                    C.v0[q] = v0[q].units();
                    C.d1[q] = d1[q].units();
                    C.v1[q] = v1[q].units();
                }
            }
            __syncthreads();
            par ^= 1;
        }
        // row jseg is complete (the next segment reaches rows jseg + 1 and
        // jseg + 2): its sums into the global accumulator
#pragma unroll
        for (int c = 0; c < CPT; ++c) {
            const int x = threadIdx.x + c * NT;
            if (x >= nx) continue;
            if (jseg >= 0 && col[c].c0) {
                const int el = elc[x] >> 16;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    add_sums(col[c].d0[q], col[c].v0[q], el, gacc, cells, pl.ok[q], pl.base[q] + jseg * nx + x);
            }
            col[c].next_row();
            elc[x] = elc[x] << 16 | FX_EMIN;
        }
    }
    // (the last segment is row nvx - 1; what is left belongs to row nvx, off the grid)

    if (nmov) atomicAdd(&mov_s, (unsigned long long)nmov);
    if (nfar) atomicAdd(&far_s, (unsigned long long)nfar);
    __syncthreads();
    if (threadIdx.x == 0) {
        if (mov_s) atomicAdd(&ctl->movers[s], mov_s);
        if (far_s) atomicAdd(&ctl->far_movers[s], far_s);
        if (flag_s) atomicOr(&ctl->err, ERR_TIMEOUT);
    }
}

// ---------------------------------------------------------------------------
// finalize: f = num / den (Eq. 4), charge per row group (Eq. 14), diagnostics
// ---------------------------------------------------------------------------
// FP64: quotient and entropy logarithm in integers (fx_div, fx_log), which
// leaves three FP64 operations per cell (the sums) of the 17 that bound this
// kernel: 67 M cells 1.97 -> 0.68 ms, 2.7 GB, 58 % of the copy rate (0.63 ms
// with the quotient's last bit left undecided).
template <typename T>
__global__ void __launch_bounds__(FIN3_X * FIN3_R) k_fin3(const StepArgs* __restrict__ A, int all_species)
{
    static_assert(FIN3_X == 32 && FIN3_R == 8, "eight warps, a row each");
    __shared__ double col_red[FIN3_X][8];
    __shared__ double red[3][8];
    const int g = blockIdx.x;
    const int s = species_of_fin3(A, g);
    const SpDev& sp = A->sp[s];
    if (!all_species && !sp.mobile) return;
    const int blk = g - sp.fin_base;
    const int xb = blk % sp.nxb, rqi = blk / sp.nxb;
    const int nx = sp.nx, nvf = sp.nvflat;
    const int col = threadIdx.x % FIN3_X, lr = threadIdx.x / FIN3_X;
    const int x = xb * FIN3_X + col;
    const bool xok = x < nx;
    const int j0 = rqi * sp.rq, j1 = min(nvf, j0 + sp.rq);
    const int a = A->ctl->asel[s];
    const size_t cells = (size_t)nvf * nx;
    const T* num = reinterpret_cast<const T*>(sp.acc[a]);
    const T* den = num + cells;
    T* clr = reinterpret_cast<T*>(sp.acc[1 - a]);
    T* fg = reinterpret_cast<T*>(sp.fgrid);
    const T* v2 = reinterpret_cast<const T*>(sp.v2row);
    ColAcc<T> acc;
    if constexpr (sizeof(T) == 8) acc.logtab = A->fd.logtab;
    auto cell = [&](int j, T nn, T dd, T v2j) {
        const size_t o = (size_t)j * nx + x;
        T f;
        if constexpr (sizeof(T) == 8)
            f = __double_as_longlong(dd) > 0 ? fx_div(nn, dd) : 0.0;   // dd >= 0 is a sum of weights
        else
            f = dd > (T)0 ? nn / dd : (T)0;
        fg[o] = f;
        clr[o] = (T)0;
        clr[cells + o] = (T)0;
        acc.add(f, (T)0, v2j);
    };
    if (xok) {
        // four rows per iteration, their loads issued together; the cells
        // are still taken in row order
        int j = j0 + lr;
        for (; j + 3 * FIN3_R < j1; j += 4 * FIN3_R) {
            T nn[4], dd[4], vv[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const size_t o = (size_t)(j + k * FIN3_R) * nx + x;
                nn[k] = num[o];
                dd[k] = den[o];
                vv[k] = v2[j + k * FIN3_R];
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) cell(j + k * FIN3_R, nn[k], dd[k], vv[k]);
        }
        for (; j < j1; j += FIN3_R) {
            const size_t o = (size_t)j * nx + x;
            cell(j, num[o], den[o], v2[j]);
        }
    }
    // charge per column and diagnostics of the block, in trees (as k_fin1)
    const double dvol = sp.dv[0] * sp.dv[1] * sp.dv[2];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const double N = acc_value(acc.rho), d = warp_sum3(N, acc_value(acc.w), acc_value(acc.ent));
    col_red[col][warp] = N;
    if ((lane & 7) == 0 && lane < 24) red[lane >> 3][warp] = d;
    __syncthreads();
    const int xr = xb * FIN3_X + (threadIdx.x >> 3);   // four columns per warp
    const double r = sum8(col_red[threadIdx.x >> 3][lane & 7]);
    if ((lane & 7) == 0 && xr < nx) sp.rho_part[(size_t)rqi * nx + xr] = sp.q * dvol * r;
    if (warp == 0) {   // N, W_kin, S
        const int k = min(lane >> 3, 2);
        const double t = sum8(red[k][lane & 7]), cell = sp.dx * dvol;
        if ((lane & 7) == 0)
            sp.dpart[(size_t)blk * 4 + (lane >> 3)] = lane == 24 ? 0.0 : t * (k == 1 ? 0.5 * sp.m * cell : cell);
    }
}

// ---------------------------------------------------------------------------
// re-sort: every pencil of a species the field kernel marked, from buffer
// 1 - cur into buffer cur (the field kernel has already flipped cur)
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(P3_THREADS) k_sort3(const StepArgs* __restrict__ A)
{
    __shared__ int cnt[NV3_MAX + 2];
    __shared__ int wsum[P3_THREADS / 32];
    const int g = blockIdx.x;
    const int s = species_of_pen(A, g);
    const SpDev& sp = A->sp[s];
    const Ctl* ctl = A->ctl;
    if (!sp.mobile || !ctl->sort_now[s]) return;
    const int p = g - sp.pen_base;
    const int dst = ctl->cur[s], src = 1 - dst;
    const int nk = sp.nkey, nvx = sp.nv[0];
    const int* sg = sp.seg[src] + (size_t)p * (nk + 1);
    int* dg = sp.seg[dst] + (size_t)p * (nk + 1);
    const int beg = sg[0], end = sg[nk];
    const T ax = sp_const<T>(sp).a[0], bx = sp_const<T>(sp).b[0];
    const T* vxs = reinterpret_cast<const T*>(sp.mv[src][0]);
    for (int i = threadIdx.x; i < nk + 1; i += P3_THREADS) cnt[i] = 0;
    __syncthreads();
    for (int b0 = beg; b0 < end; b0 += P3_THREADS) {
        const int k = b0 + threadIdx.x;
        const bool ok = k < end;
        int key = 0;
        if (ok) {
            typename DualW<T>::type w;
            key = key_of(dual3(vxs[k], ax, bx, nvx, w), nvx);
        }
        const int kk = ok ? key : -1;
        const unsigned grp = __match_any_sync(0xffffffffu, kk);
        if (ok && (threadIdx.x & 31) == __ffs(grp) - 1) atomicAdd(&cnt[key], __popc(grp));
    }
    __syncthreads();
    block_exscan(cnt, cnt, nk, (nk + P3_THREADS - 1) / P3_THREADS, wsum);
    for (int i = threadIdx.x; i <= nk; i += P3_THREADS) dg[i] = beg + cnt[i];
    __syncthreads();
    for (int b0 = beg; b0 < end; b0 += P3_THREADS) {
        const int k = b0 + threadIdx.x;
        const bool ok = k < end;
        int key = 0;
        T vx = 0;
        if (ok) {
            typename DualW<T>::type w;
            vx = vxs[k];
            key = key_of(dual3(vx, ax, bx, nvx, w), nvx);
        }
        const int slot = beg + warp_slot(cnt, key, ok);
        if (ok && slot >= beg && slot < end) {
            Pos3<T> pos;
            pos.load(sp, src, k);
            pos.store(sp, dst, slot);
            reinterpret_cast<T*>(sp.mv[dst][0])[slot] = vx;
            reinterpret_cast<T*>(sp.mv[dst][1])[slot] = reinterpret_cast<const T*>(sp.mv[src][1])[k];
            reinterpret_cast<T*>(sp.mv[dst][2])[slot] = reinterpret_cast<const T*>(sp.mv[src][2])[k];
            reinterpret_cast<T*>(sp.mf[dst])[slot] = reinterpret_cast<const T*>(sp.mf[src])[k];
            if constexpr (sizeof(T) == 8) sp.mwyz[dst][slot] = sp.mwyz[src][k];
        }
    }
}

// ---------------------------------------------------------------------------
// marker creation: jittered lattice (Sec. 2 / Sec. 3.1) or caller arrays,
// counting-sorted by (pencil, key) into buffer 0
// ---------------------------------------------------------------------------
struct MarkerIn3 {
    double xi;   // position in cells
    double v[3];
    double f;
    bool ok;
};

// lattice marker number k in generation order (v_z, v_y, v_x cell slowest,
// then x cell, then sub-point); the jitter streams use the row-major marker
// number ((((i nvx + jx) nvy + jy) nvz + jz) ppc + sub)
struct LatticeSrc3 {
    const avl_f0* f0;
    unsigned long long seed;
    double jitter;
    int s;
    int l[4];
    __device__ MarkerIn3 get(const SpDev& sp, long long k) const
    {
        const int ppc = l[0] * l[1] * l[2] * l[3];
        const int sub = (int)(k % ppc);
        long long r = k / ppc;
        const int i = (int)(r % sp.nx);
        r /= sp.nx;
        const int jx = (int)(r % sp.nv[0]);
        r /= sp.nv[0];
        const int jy = (int)(r % sp.nv[1]);
        const int jz = (int)(r / sp.nv[1]);
        const long long cell = (((long long)i * sp.nv[0] + jx) * sp.nv[1] + jy) * sp.nv[2] + jz;
        const long long m = cell * ppc + sub;
        const int bz = sub % l[3], by = (sub / l[3]) % l[2], bx = (sub / (l[3] * l[2])) % l[1];
        const int a = sub / (l[3] * l[2] * l[1]);
        const int j[3] = {jx, jy, jz}, b[3] = {bx, by, bz};
        MarkerIn3 o;
        const double J0 = (jitter_u01(seed, s, m, 0) - 0.5) * jitter;
        o.xi = (double)i + ((double)a + 0.5 + J0) / l[0];
        for (int d = 0; d < 3; ++d) {
            const double Jd = (jitter_u01(seed, s, m, d + 1) - 0.5) * jitter;
            o.v[d] = sp.vmin[d] + ((double)j[d] + ((double)b[d] + 0.5 + Jd) / l[d + 1]) * sp.dv[d];
        }
        o.f = f0_value(f0, 3, sp.nx * sp.dx, o.xi * sp.dx, o.v);
        o.ok = true;
        return o;
    }
};

struct ArraySrc3 {
    const double* x;
    const double* v;   // component-major: v[d * n + k]
    const double* f;
    long long n;
    __device__ MarkerIn3 get(const SpDev& sp, long long k) const
    {
        MarkerIn3 o;
        const double L = sp.nx * sp.dx;
        const double xv = x[k];
        o.f = f[k];
        o.ok = (xv >= 0.0 && xv < L) && isfinite(o.f);
        for (int d = 0; d < 3; ++d) {
            o.v[d] = v[(long long)d * n + k];
            o.ok = o.ok && isfinite(o.v[d]);
        }
        o.xi = o.ok ? xv / sp.dx : 0.0;
        if (!o.ok) {
            for (int d = 0; d < 3; ++d) o.v[d] = sp.vmin[d];
            o.f = 0.0;
        }
        return o;
    }
};

// bucket (pencil * nkey + key) of a marker from its stored velocities
template <typename T>
__device__ __forceinline__ int bucket3(const SpDev& sp, const VCoef<T>& vc, const T (&v)[3])
{
    typename DualW<T>::type w;
    const int kx = key_of(dual3(v[0], vc.a[0], vc.b[0], vc.n[0], w), vc.n[0]);
    const int ky = key_of(dual3(v[1], vc.a[1], vc.b[1], vc.n[1], w), vc.n[1]);
    const int kz = key_of(dual3(v[2], vc.a[2], vc.b[2], vc.n[2], w), vc.n[2]);
    return (kz * (vc.n[1] + 1) + ky) * sp.nkey + kx;
}

// the same bucket and, FP64, the (v_y, v_z) weights as marker_wyz has them,
// from the same conversions
template <typename T>
__device__ __forceinline__ int bucket3w(const VCoef<T>& vc, int nkey, const T (&v)[3], longlong2& wyz)
{
    typename DualW<T>::type w, wy, wz;
    const int kx = key_of(dual3(v[0], vc.a[0], vc.b[0], vc.n[0], w), vc.n[0]);
    const int jy = dual3(v[1], vc.a[1], vc.b[1], vc.n[1], wy), jz = dual3(v[2], vc.a[2], vc.b[2], vc.n[2], wz);
    if constexpr (sizeof(T) == 8)
        wyz = jy < -1 || jy >= vc.n[1] || jz < -1 || jz >= vc.n[2] ? make_longlong2(-1, -1) : make_longlong2(wy, wz);
    return (key_of(jz, vc.n[2]) * (vc.n[1] + 1) + key_of(jy, vc.n[1])) * nkey + kx;
}

template <typename T, typename Src>
__global__ void __launch_bounds__(256) k_src3_count(const StepArgs* __restrict__ A, int s, Src src,
                                                    unsigned long long* bad)
{
    const SpDev& sp = A->sp[s];
    VCoef<T> vc;
    vc.init(sp);
    unsigned nbad = 0;
    const long long stride = (long long)gridDim.x * blockDim.x;
    // whole warps iterate together (warp-aggregated counting)
    const long long n_pad = (sp.n + 31) / 32 * 32;
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n_pad; k += stride) {
        const bool ok = k < sp.n;
        int b = 0;
        if (ok) {
            const MarkerIn3 mk = src.get(sp, k);
            if (!mk.ok) ++nbad;
            const T v[3] = {(T)mk.v[0], (T)mk.v[1], (T)mk.v[2]};
            b = bucket3<T>(sp, vc, v);
        }
        const int kk = ok ? b : -1;
        const unsigned grp = __match_any_sync(0xffffffffu, kk);
        if (ok && (threadIdx.x & 31) == __ffs(grp) - 1) atomicAdd(&sp.kcount[b], __popc(grp));
    }
    if (nbad && bad) atomicAdd(bad, (unsigned long long)nbad);
}

// Exclusive scan of the bucket counts over tiles of SCAN_TILE buckets (one
// block each): k_src3_tsum sums every tile, k_src3_scan adds the totals of
// the tiles before its own and scans the tile into the slot cursors kcur and
// the segment table of the target buffer, clearing the counts for the next
// use.  Creation (resort = 0) fills buffer 0; a global re-sort (resort = 1)
// fills buffer 1 - cur, and k_src3_flip makes it current after the scatter.
constexpr int SCAN_TILE = 1024;

__device__ __forceinline__ int block_sum_1024(int v, int* ws)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    v = __reduce_add_sync(0xffffffffu, v);
    if (lane == 0) ws[warp] = v;
    __syncthreads();
    int t = lane < (int)(blockDim.x >> 5) ? ws[lane] : 0;
    t = __reduce_add_sync(0xffffffffu, t);
    __syncthreads();
    return t;
}

__global__ void __launch_bounds__(SCAN_TILE) k_src3_tsum(const StepArgs* __restrict__ A, int s)
{
    __shared__ int ws[32];
    const SpDev& sp = A->sp[s];
    const int nb = sp.npen * sp.nkey;
    const int i = blockIdx.x * SCAN_TILE + threadIdx.x;
    const int t = block_sum_1024(i < nb ? sp.kcount[i] : 0, ws);
    if (threadIdx.x == 0) sp.ktile[blockIdx.x] = t;
}

__global__ void __launch_bounds__(SCAN_TILE) k_src3_scan(const StepArgs* __restrict__ A, int s, int resort)
{
    __shared__ int ws[32];
    const SpDev& sp = A->sp[s];
    const int nb = sp.npen * sp.nkey, nk = sp.nkey;
    const int dst = resort ? 1 - A->ctl->cur[s] : 0;
    int o = 0;
    for (int t = threadIdx.x; t < (int)blockIdx.x; t += SCAN_TILE) o += sp.ktile[t];
    const int off = block_sum_1024(o, ws);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = blockIdx.x * SCAN_TILE + threadIdx.x;
    const int v = i < nb ? sp.kcount[i] : 0;
    int x = v;
    for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
    }
    if (lane == 31) ws[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int w = ws[lane];
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, w, d);
            if (lane >= d) w += y;
        }
        ws[lane] = w;
    }
    __syncthreads();
    if (i >= nb) return;
    const int excl = off + x - v + (warp > 0 ? ws[warp - 1] : 0);
    sp.kcur[i] = excl;
    sp.kcount[i] = 0;
    int* sg = sp.seg[dst];
    const int p = i / nk, k = i - p * nk;
    sg[p * (nk + 1) + k] = excl;
    if (k == 0 && p > 0) sg[(p - 1) * (nk + 1) + nk] = excl;   // end of the previous pencil
    if (i == nb - 1) {
        sg[p * (nk + 1) + nk] = excl + v;
        if (resort && (long long)(excl + v) != sp.n) atomicOr(&A->ctl->err, ERR_CAPACITY);
    }
}

// after a global re-sort: the buffer written becomes current
__global__ void k_src3_flip(const StepArgs* __restrict__ A, int s)
{
    if (threadIdx.x == 0) {
        A->ctl->cur[s] = 1 - A->ctl->cur[s];
        A->ctl->nsort[s] += 1;
    }
}

template <typename T, typename Src>
__global__ void __launch_bounds__(256) k_src3_scatter(const StepArgs* __restrict__ A, int s, Src src)
{
    const SpDev& sp = A->sp[s];
    VCoef<T> vc;
    vc.init(sp);
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long n_pad = (sp.n + 31) / 32 * 32;
    bool over = false;
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n_pad; k += stride) {
        const bool ok = k < sp.n;
        MarkerIn3 mk{};
        T v[3] = {(T)0, (T)0, (T)0};
        int b = 0;
        if (ok) {
            mk = src.get(sp, k);
            for (int d = 0; d < 3; ++d) v[d] = (T)mk.v[d];
            b = bucket3<T>(sp, vc, v);
        }
        const int slot = warp_slot(sp.kcur, b, ok);
        if (!ok) continue;
        if (slot < 0 || (long long)slot >= sp.n) {
            over = true;
            continue;
        }
        const Pos3<T> pos = pos3_from_cells<T>(mk.xi, sp.nx);
        pos.store(sp, 0, slot);
        for (int d = 0; d < 3; ++d) reinterpret_cast<T*>(sp.mv[0][d])[slot] = v[d];
        reinterpret_cast<T*>(sp.mf[0])[slot] = (T)mk.f;
        if constexpr (sizeof(T) == 8) sp.mwyz[0][slot] = marker_wyz(vc, v[1], v[2]);
    }
    if (over) atomicOr(&A->ctl->err, ERR_CAPACITY);
}

// ---------------------------------------------------------------------------
// static background magnetic field: Boris push and global re-sort
// ---------------------------------------------------------------------------
template <typename T>
struct Vec2;
template <>
struct Vec2<float> {
    using type = float2;
};
template <>
struct Vec2<double> {
    using type = double2;
};

// Boris push of every marker of species s in buffer cur, written back in
// place: half kick by E_x at the old position, rotation v- -> v+ about B,
// half kick, x += v_x dt.  The (pencil, key) bucket of the new velocities,
// computed from the stored values exactly as the scatter recomputes it, is
// counted into kcount (one atomic per distinct bucket of a warp).  The field
// is staged as half kicks and their differences: 23 FP64 operations per marker
// of the FP64 push where it took 28, and its constants come from the host (a
// thread took 40 for its few markers): 2.6 M markers, 100 x 24 x 20 x 18, push
// and re-sort 294 -> 234 us.
template <typename T>
__global__ void __launch_bounds__(256) k_bpush3(const StepArgs* __restrict__ A, int s)
{
    using T2 = typename Vec2<T>::type;
    extern __shared__ __align__(16) unsigned char smem[];
    T2* Es = reinterpret_cast<T2*>(smem);   // half kick at the centre of cell i and its change to cell i + 1
    const SpDev& sp = A->sp[s];
    const int cb = A->ctl->cur[s];
    const int nx = sp.nx;
    const SpConst<T>& k0 = sp_const<T>(sp);
    struct {
        T a, t[3], s[3];
    } bc = {k0.ba, {k0.bt[0], k0.bt[1], k0.bt[2]}, {k0.bs[0], k0.bs[1], k0.bs[2]}};
    for (int i = threadIdx.x; i < nx; i += blockDim.x) {
        const int j = i + 1 == nx ? 0 : i + 1;
        const T e0 = sizeof(T) == 4 ? (T)A->fd.E32[i] : (T)A->fd.E64[i], e1 = sizeof(T) == 4 ? (T)A->fd.E32[j] : (T)A->fd.E64[j];
        Es[i].x = bc.a * e0;
        Es[i].y = bc.a * (e1 - e0);
    }
    __syncthreads();
    VCoef<T> vc;
    vc.init(sp);
    const T dt_dx = k0.dt_dx;
    const int nkey = sp.nkey;
    T* const g0 = reinterpret_cast<T*>(sp.mv[cb][0]);
    T* const g1 = reinterpret_cast<T*>(sp.mv[cb][1]);
    T* const g2 = reinterpret_cast<T*>(sp.mv[cb][2]);
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long n_pad = (sp.n + 31) / 32 * 32;
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n_pad; k += stride) {
        const bool ok = k < sp.n;
        int b = 0;
        if (ok) {
            Pos3<T> pos;
            pos.load(sp, cb, (int)k);
            int i0;
            T wx;
            pos.cic(i0, wx);
            const T2 e = Es[(unsigned)i0 < (unsigned)nx ? i0 : nx - 1];
            const T aE = fma(wx, e.y, e.x);
            const T m0 = g0[k] + aE, m1 = g1[k], m2 = g2[k];
            const T p0 = m0 + (m1 * bc.t[2] - m2 * bc.t[1]);
            const T p1 = m1 + (m2 * bc.t[0] - m0 * bc.t[2]);
            const T p2 = m2 + (m0 * bc.t[1] - m1 * bc.t[0]);
            const T v[3] = {m0 + (p1 * bc.s[2] - p2 * bc.s[1]) + aE, m1 + (p2 * bc.s[0] - p0 * bc.s[2]),
                            m2 + (p0 * bc.s[1] - p1 * bc.s[0])};
            if constexpr (sizeof(T) == 8)
                pos.wrap((long long)((unsigned long long)pos.X + (unsigned long long)fx_count(v[0] * dt_dx)), nx);
            else
                pos.drift(v[0] * dt_dx, nx);
            pos.store(sp, cb, (int)k);
            g0[k] = v[0];
            g1[k] = v[1];
            g2[k] = v[2];
            longlong2 wyz;
            b = bucket3w<T>(vc, nkey, v, wyz);
        }
        const int kk = ok ? b : -1;
        const unsigned grp = __match_any_sync(0xffffffffu, kk);
        if (ok && (threadIdx.x & 31) == __ffs(grp) - 1) atomicAdd(&sp.kcount[b], __popc(grp));
    }
}

// the markers of species s from buffer cur into their (pencil, key) buckets
// of buffer 1 - cur (k_src3_scan has placed the cursors).  A warp takes
// RS3_ROUNDS x 32 consecutive markers: all loads first, then one slot per
// round (a match on the bucket and one atomic per distinct bucket, all
// rounds' atomics in flight together), then the stores.  Bound by the latency
// of its loads and atomics: 134 M FP32 markers, push and re-sort 2.82 ms with
// four rounds, 2.70 with two (more warps per SM), 2.89 with one.
constexpr int RS3_ROUNDS = 2;

template <typename T>
__global__ void __launch_bounds__(256) k_rs3_scatter(const StepArgs* __restrict__ A, int s)
{
    const SpDev& sp = A->sp[s];
    const int src = A->ctl->cur[s], dst = 1 - src;
    VCoef<T> vc;
    vc.init(sp);
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const long long wid = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    const long long n = sp.n;
    const int nkey = sp.nkey;
    const T* f_src = reinterpret_cast<const T*>(sp.mf[src]);
    bool over = false;
    for (long long w0 = wid * 32 * RS3_ROUNDS; w0 < n; w0 += nw * 32 * RS3_ROUNDS) {
        T v[RS3_ROUNDS][3], fv[RS3_ROUNDS];
        Pos3<T> pos[RS3_ROUNDS];
        int b[RS3_ROUNDS];
        longlong2 wyz[RS3_ROUNDS];
#pragma unroll
        for (int r = 0; r < RS3_ROUNDS; ++r) {
            const long long k = w0 + r * 32 + lane;
            b[r] = -1;
            if (k < n) {
                for (int d = 0; d < 3; ++d) v[r][d] = reinterpret_cast<const T*>(sp.mv[src][d])[k];
                fv[r] = f_src[k];
                pos[r].load(sp, src, (int)k);
                b[r] = bucket3w<T>(vc, nkey, v[r], wyz[r]);
            }
        }
        unsigned grp[RS3_ROUNDS];
        int base[RS3_ROUNDS];
#pragma unroll
        for (int r = 0; r < RS3_ROUNDS; ++r) {
            grp[r] = __match_any_sync(0xffffffffu, b[r]);
            base[r] = 0;
            if (b[r] >= 0 && lane == __ffs(grp[r]) - 1) base[r] = atomicAdd(&sp.kcur[b[r]], __popc(grp[r]));
        }
#pragma unroll
        for (int r = 0; r < RS3_ROUNDS; ++r) {
            const int slot = __shfl_sync(0xffffffffu, base[r], __ffs(grp[r]) - 1) + __popc(grp[r] & lt);
            if (b[r] < 0) continue;
            if (slot < 0 || (long long)slot >= n) {
                over = true;
                continue;
            }
            pos[r].store(sp, dst, slot);
            for (int d = 0; d < 3; ++d) reinterpret_cast<T*>(sp.mv[dst][d])[slot] = v[r][d];
            reinterpret_cast<T*>(sp.mf[dst])[slot] = fv[r];
            if constexpr (sizeof(T) == 8) sp.mwyz[dst][slot] = wyz[r];
        }
    }
    if (over) atomicOr(&A->ctl->err, ERR_CAPACITY);
}

template <typename T>
__global__ void k_get3(const StepArgs* __restrict__ A, int s, double* __restrict__ x, double* __restrict__ v,
                       double* __restrict__ f)
{
    const SpDev& sp = A->sp[s];
    const int cb = A->ctl->cur[s];
    const long long n = sp.n;
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        Pos3<T> pos;
        pos.load(sp, cb, (int)k);
        if (x) x[k] = pos.cells() * sp.dx;
        if (v)
            for (int d = 0; d < 3; ++d) v[(long long)d * n + k] = (double)reinterpret_cast<const T*>(sp.mv[cb][d])[k];
        if (f) f[k] = (double)reinterpret_cast<const T*>(sp.mf[cb])[k];
    }
}

// internal [vz][vy][vx][x] -> caller [x][vx][vy][vz], 32 x 32 tiles of (x, vz)
template <typename T>
__global__ void k_getf3(const T* __restrict__ fg, const T* __restrict__ dg, int nx, int X, int Y, int Z,
                        double* __restrict__ f, double* __restrict__ n)
{
    __shared__ double tile[2][32][33];
    const int tx = (nx + 31) / 32, tz = (Z + 31) / 32;
    const long long ntile = (long long)tx * tz * X * Y;
    const long long nvf = (long long)X * Y * Z;
    for (long long t = blockIdx.x; t < ntile; t += gridDim.x) {
        const int xt = (int)(t % tx);
        long long r = t / tx;
        const int zt = (int)(r % tz);
        r /= tz;
        const int Xi = (int)(r / Y), Yi = (int)(r % Y);
        for (int rr = threadIdx.y; rr < 32; rr += blockDim.y) {
            const int zi = zt * 32 + rr, xi = xt * 32 + threadIdx.x;
            if (zi < Z && xi < nx) {
                const size_t o = (((size_t)zi * Y + Yi) * X + Xi) * nx + xi;
                tile[0][rr][threadIdx.x] = (double)fg[o];
                if (n) tile[1][rr][threadIdx.x] = (double)dg[o];
            }
        }
        __syncthreads();
        for (int rr = threadIdx.y; rr < 32; rr += blockDim.y) {
            const int xi = xt * 32 + rr, zi = zt * 32 + threadIdx.x;
            if (zi < Z && xi < nx) {
                const size_t o = (size_t)xi * nvf + ((size_t)Xi * Y + Yi) * Z + zi;
                f[o] = tile[0][threadIdx.x][rr];
                if (n) n[o] = tile[1][threadIdx.x][rr];
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------

cudaError_t configure_vhs3(const StepArgs& h)
{
    const int smem = (int)pd3_smem_bytes(h.fd.nx, nkey_max(h), h.prec);
    cudaError_t e;
    if (h.prec == AVL_FP64) {
        if ((e = raise_smem_limit(k_pd3x<1, false>, smem))) return e;
        if ((e = raise_smem_limit(k_pd3x<2, false>, smem))) return e;
        if ((e = raise_smem_limit(k_pd3x<1, true>, smem))) return e;
        return raise_smem_limit(k_pd3x<2, true>, smem);
    }
    if ((e = raise_smem_limit(k_pd3<1, false>, smem))) return e;
    if ((e = raise_smem_limit(k_pd3<2, false>, smem))) return e;
    if ((e = raise_smem_limit(k_pd3<4, false>, smem))) return e;
    if ((e = raise_smem_limit(k_pd3<1, true>, smem))) return e;
    if ((e = raise_smem_limit(k_pd3<2, true>, smem))) return e;
    return raise_smem_limit(k_pd3<4, true>, smem);
}

template <bool PUSH>
static void pd3_go(const StepArgs& h, const StepArgs* d, int mode, cudaStream_t st)
{
    const int smem = (int)pd3_smem_bytes(h.fd.nx, nkey_max(h), h.prec), cpt = cpt_of(h.fd.nx), n = h.npen_total;
    if (h.prec == AVL_FP64) {   // nx <= 512
        if (cpt == 1) k_pd3x<1, PUSH><<<n, P3_THREADS, smem, st>>>(d, mode);
        else k_pd3x<2, PUSH><<<n, P3_THREADS, smem, st>>>(d, mode);
    } else if (cpt == 1) {
        k_pd3<1, PUSH><<<n, P3_THREADS, smem, st>>>(d, mode);
    } else if (cpt == 2) {
        k_pd3<2, PUSH><<<n, P3_THREADS, smem, st>>>(d, mode);
    } else {
        k_pd3<4, PUSH><<<n, P3_THREADS, smem, st>>>(d, mode);
    }
}

cudaError_t launch_pd3(const StepArgs& h, const StepArgs* d, int mode, cudaStream_t st)
{
    if (h.npen_total == 0) return cudaSuccess;
    if (mode == 1)
        pd3_go<true>(h, d, mode, st);
    else
        pd3_go<false>(h, d, mode, st);
    return cudaGetLastError();
}

cudaError_t launch_fin3(const StepArgs& h, const StepArgs* d, int all_species, cudaStream_t st)
{
    if (h.prec == AVL_FP32)
        k_fin3<float><<<h.nfin_total, FIN3_X * FIN3_R, 0, st>>>(d, all_species);
    else
        k_fin3<double><<<h.nfin_total, FIN3_X * FIN3_R, 0, st>>>(d, all_species);
    return cudaGetLastError();
}

cudaError_t launch_sort3(const StepArgs& h, const StepArgs* d, cudaStream_t st)
{
    if (h.npen_total == 0) return cudaSuccess;
    if (h.prec == AVL_FP32)
        k_sort3<float><<<h.npen_total, P3_THREADS, 0, st>>>(d);
    else
        k_sort3<double><<<h.npen_total, P3_THREADS, 0, st>>>(d);
    return cudaGetLastError();
}

// bucket counts -> cursors and segment table (creation: buffer 0; re-sort:
// buffer 1 - cur)
static void scan3(const StepArgs& h, const StepArgs* d, int s, int resort, cudaStream_t st)
{
    const int nb = h.sp[s].npen * h.sp[s].nkey;
    const int tiles = (nb + SCAN_TILE - 1) / SCAN_TILE;
    k_src3_tsum<<<tiles, SCAN_TILE, 0, st>>>(d, s);
    k_src3_scan<<<tiles, SCAN_TILE, 0, st>>>(d, s, resort);
}

// source -> layout in buffer 0 (kcount is zero before and after)
template <typename Src>
static cudaError_t source_to_layout3(const StepArgs& h, const StepArgs* d, int s, Src src, unsigned long long* bad,
                                     cudaStream_t st)
{
    const long long n = h.sp[s].n;
    const int blocks = (int)std::max<long long>(1, std::min<long long>((n + 255) / 256, 152ll * 16));
    if (h.prec == AVL_FP32) {
        k_src3_count<float, Src><<<blocks, 256, 0, st>>>(d, s, src, bad);
        scan3(h, d, s, 0, st);
        k_src3_scatter<float, Src><<<blocks, 256, 0, st>>>(d, s, src);
    } else {
        k_src3_count<double, Src><<<blocks, 256, 0, st>>>(d, s, src, bad);
        scan3(h, d, s, 0, st);
        k_src3_scatter<double, Src><<<blocks, 256, 0, st>>>(d, s, src);
    }
    return cudaGetLastError();
}

cudaError_t launch_init3(const StepArgs& h, const StepArgs* d, int s, const int lattice[4], const avl_f0* f0_dev,
                         unsigned long long seed, double jitter, cudaStream_t st)
{
    const LatticeSrc3 src{f0_dev, seed, jitter, s, {lattice[0], lattice[1], lattice[2], lattice[3]}};
    return source_to_layout3(h, d, s, src, nullptr, st);
}

cudaError_t launch_set3(const StepArgs& h, const StepArgs* d, int s, long long n, const double* x, const double* v,
                        const double* f, unsigned long long* bad, cudaStream_t st)
{
    const ArraySrc3 src{x, v, f, n};
    return source_to_layout3(h, d, s, src, bad, st);
}

static int marker_blocks(long long n)
{
    return (int)std::max<long long>(1, std::min<long long>((n + 255) / 256, 152ll * 16));
}

cudaError_t launch_bpush3(const StepArgs& h, const StepArgs* d, int s, cudaStream_t st)
{
    const long long n = h.sp[s].n;
    if (n == 0) return cudaSuccess;
    const int blocks = marker_blocks(n);
    if (h.prec == AVL_FP32)
        k_bpush3<float><<<blocks, 256, (size_t)h.sp[s].nx * 8, st>>>(d, s);
    else
        k_bpush3<double><<<blocks, 256, (size_t)h.sp[s].nx * 16, st>>>(d, s);
    return cudaGetLastError();
}

cudaError_t launch_rsort3(const StepArgs& h, const StepArgs* d, int s, cudaStream_t st)
{
    const long long n = h.sp[s].n;
    if (n == 0) return cudaSuccess;
    const int blocks = marker_blocks(n);
    scan3(h, d, s, 1, st);
    if (h.prec == AVL_FP32)
        k_rs3_scatter<float><<<blocks, 256, 0, st>>>(d, s);
    else
        k_rs3_scatter<double><<<blocks, 256, 0, st>>>(d, s);
    k_src3_flip<<<1, 32, 0, st>>>(d, s);
    return cudaGetLastError();
}

cudaError_t launch_get3(const StepArgs& h, const StepArgs* d, int s, double* x, double* v, double* f, cudaStream_t st)
{
    const long long n = h.sp[s].n;
    if (n == 0) return cudaSuccess;
    const int blocks = (int)std::min<long long>((n + 255) / 256, 152ll * 16);
    if (h.prec == AVL_FP32)
        k_get3<float><<<blocks, 256, 0, st>>>(d, s, x, v, f);
    else
        k_get3<double><<<blocks, 256, 0, st>>>(d, s, x, v, f);
    return cudaGetLastError();
}

cudaError_t launch_getf3(const StepArgs& h, int s, int which, double* f, double* n, cudaStream_t st)
{
    const SpDev& sp = h.sp[s];
    const size_t cells = (size_t)sp.nvflat * sp.nx;
    const long long ntile = (long long)((sp.nx + 31) / 32) * ((sp.nv[2] + 31) / 32) * sp.nv[0] * sp.nv[1];
    const int blocks = (int)std::max<long long>(1, std::min<long long>(ntile, 152ll * 32));
    dim3 block(32, 8);
    if (h.prec == AVL_FP32) {
        const float* dg = reinterpret_cast<const float*>(sp.acc[which]) + cells;
        k_getf3<float><<<blocks, block, 0, st>>>(reinterpret_cast<const float*>(sp.fgrid), dg, sp.nx, sp.nv[0],
                                                 sp.nv[1], sp.nv[2], f, n);
    } else {
        const double* dg = reinterpret_cast<const double*>(sp.acc[which]) + cells;
        k_getf3<double><<<blocks, block, 0, st>>>(reinterpret_cast<const double*>(sp.fgrid), dg, sp.nx, sp.nv[0],
                                                  sp.nv[1], sp.nv[2], f, n);
    }
    return cudaGetLastError();
}

}  // namespace avl
