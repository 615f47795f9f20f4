// fftfx.cuh -- the passes of the FP64 and compensated plans in 64-bit block
// fixed point (sg_fx.cuh): FP64 fields and FP64 half spectra in memory, the
// transforms and the products with the kernel spectra on the integer pipes.
// Included by one translation unit per transform length (fftfx_lg<LG>.cu).
//
// The passes and their buffers are those of the run-time-length FP64 kernels
// (fftconv.cu), element for element, so each may be replaced on its own and
// the edge and wedge updates between them stay as they are.  A transform of N
// points is held by N / 8 threads, 8 points each (32 registers); exchanges go
// through 16-byte elements in shared memory, padded as sg_pad.  Each thread's
// twiddles come from tables laid out by pass (fx_tw_base), read through L1:
// their 62 bits would cost more to form by products.
//
// What bounds them: the integer pipes (a complex product is twelve wide
// multiply-adds and some fifteen additions and moves), and before that the
// instruction cache: unrolled passes are long, and with
// 16 points per thread, every pass unrolled and the inverse transforms apart
// (140 KB of code in the column kernel) half of the cycles waited for
// instructions.  Here the radix-8 passes of a kernel are one loop, and the
// column kernels' three transforms share it (inverses as conj FFT conj).
// Measured at 1024 x 2048, the FP64 pipe's kernels -> these, us: R2C rows 105
// -> 32, columns 486 -> 98, C2R rows 195 -> 51; a forward call 781 -> 169.
// Products that shifted their sums into place, and whose digits' products the
// compiler widened to 64 x 64 bits, took 32, 111, 55 and 188.
// Error of F_phi on a smooth disk of 256 x 512 against an 80-bit evaluation:
// 1.6e-15 -> 1.6e-16 (F_r 4.4e-16 -> 2.2e-16).
#pragma once
#include "sg_internal.cuh"
#include "sg_fx.cuh"

namespace sg {

template <int LG>
struct FxShape {
    static constexpr int N = 1 << LG, NT = N / 8;
    static constexpr int SL = NT >= 128 ? 1 : 128 / NT;  // transforms per block: R2C rows, columns
    static constexpr int RB = NT >= 64 ? 2 : 128 / NT;  // rows per block where 32-byte sectors need two (one of the tensor maps' two)
    static constexpr size_t EX = (size_t)(N + N / 16 + 1) * sizeof(fx2);  // one exchange area
    static constexpr size_t PARK = (size_t)N * sizeof(fx2);               // one parked spectrum
};
// blocks per SM the registers are bounded for: 768 threads' worth (80
// registers); 512-thread blocks two (64 registers) where shared memory holds two
constexpr int fx_minb(int threads, size_t smem) { return threads > 512 || 2 * smem > 220 * 1024 ? 1 : threads == 512 ? 2 : 768 / threads; }

// twiddles of a pass loaded before its second barrier, of seven (1024 x 2048
// forward call, us: none 173.5, 2: 171.5, 3: 171.6, 4: 170.7; more spill)
constexpr int FX_AHEAD = 4;

// OR / maximum over one transform's NT threads (whole warps, or 8 or 16 lanes) into a shared word, zero before
template <int NT>
__device__ __forceinline__ void fx_or_into(unsigned f, unsigned* word)
{
    if constexpr (NT >= 32) {
        f = __reduce_or_sync(0xffffffffu, f);
    } else {
#pragma unroll
        for (int o = NT / 2; o > 0; o >>= 1) f |= __shfl_xor_sync(0xffffffffu, f, o);
    }
    if ((threadIdx.x & (NT < 32 ? NT - 1 : 31)) == 0) atomicOr(word, f);
}
template <int NT>
__device__ __forceinline__ void fx_max_into(unsigned f, unsigned* word)
{
    if constexpr (NT >= 32) {
        f = __reduce_max_sync(0xffffffffu, f);
    } else {
#pragma unroll
        for (int o = NT / 2; o > 0; o >>= 1) f = max(f, __shfl_xor_sync(0xffffffffu, f, o));
    }
    if ((threadIdx.x & (NT < 32 ? NT - 1 : 31)) == 0) atomicMax(word, f);
}

// the same of two values into two words, by two lanes at once
struct FxOr {
    static __device__ __forceinline__ unsigned warp(unsigned a) { return __reduce_or_sync(0xffffffffu, a); }
    static __device__ __forceinline__ unsigned of(unsigned a, unsigned b) { return a | b; }
    static __device__ __forceinline__ void into(unsigned* w, unsigned a) { atomicOr(w, a); }
};
struct FxMax {
    static __device__ __forceinline__ unsigned warp(unsigned a) { return __reduce_max_sync(0xffffffffu, a); }
    static __device__ __forceinline__ unsigned of(unsigned a, unsigned b) { return max(a, b); }
    static __device__ __forceinline__ void into(unsigned* w, unsigned a) { atomicMax(w, a); }
};
struct FxSum {
    static __device__ __forceinline__ unsigned warp(unsigned a) { return __reduce_add_sync(0xffffffffu, a); }
    static __device__ __forceinline__ unsigned of(unsigned a, unsigned b) { return a + b; }
    static __device__ __forceinline__ void into(unsigned* w, unsigned a) { atomicAdd(w, a); }
};
template <int NT, typename Op>
__device__ __forceinline__ void fx_both_into(unsigned a, unsigned b, unsigned* words)
{
    if constexpr (NT >= 32) {
        a = Op::warp(a);
        b = Op::warp(b);
    } else {
#pragma unroll
        for (int o = NT / 2; o > 0; o >>= 1) {
            a = Op::of(a, __shfl_xor_sync(0xffffffffu, a, o));
            b = Op::of(b, __shfl_xor_sync(0xffffffffu, b, o));
        }
    }
    const int lane = threadIdx.x & (NT < 32 ? NT - 1 : 31);
    if (lane < 2) Op::into(words + lane, lane ? b : a);
}

__device__ __forceinline__ fx2 fx_ldg(const fx2* p)
{
    const longlong2 v = __ldg(reinterpret_cast<const longlong2*>(p));
    return fx2{v.x, v.y};
}
// loaded where it stands (ahead of a barrier)
__device__ __forceinline__ fxw fx_ldg_here(const fxw* p)
{
    fxw v;
    asm volatile("ld.global.nc.v4.s32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.rh), "=r"(v.rl), "=r"(v.ih), "=r"(v.il)
                 : "l"(p));
    return v;
}
__device__ __forceinline__ fxw fx_ldg(const fxw* p)
{
    const int4 v = __ldg(reinterpret_cast<const int4*>(p));
    return fxw{v.x, v.y, v.z, v.w};
}

// One transform of 2^LG points, thread t of 2^LG / 8 holding v[e] = x[t + e
// NT] (components up to 2^59) on entry and X[t + e NT] (up to 2^62.5) on
// return, natural order; the value is v 2^E throughout.  nrm: three zeroed
// shared words of this transform.  sm is free on entry and on return.  Every
// thread of the block calls.
template <int LG, int DIR>
__device__ __forceinline__ void fx_fft(fx2 (&v)[8], fx2* sm, unsigned* nrm, int t, const fxw* __restrict__ tw, int& E)
{
    constexpr int N = 1 << LG, NT = N / 8, R1 = 1 << fx_first_lg(LG), NP = fx_passes(LG);
#pragma unroll
    for (int s = 0; s < 8 / R1; s++) {
        fx2 a[8];
#pragma unroll
        for (int r = 0; r < R1; r++) a[r] = v[s + r * (8 / R1)];
        fx_dft<R1, DIR>(a);
#pragma unroll
        for (int r = 0; r < R1; r++) v[s + r * (8 / R1)] = a[r];
    }
    // butterfly t + s NT writes R1 neighbours
#pragma unroll
    for (int s = 0; s < 8 / R1; s++) {
        fx2* q = sm + sg_pad((t + s * NT) * R1);
#pragma unroll
        for (int r = 0; r < R1; r++) q[r] = v[s + r * (8 / R1)];
    }
    int Ns = R1;  // length of the sub-transforms done so far
    const fxw* w = tw + fx_tw_base(LG, 0);
#pragma unroll 1
    for (int p = 0; p < NP; p++) {
        fx_or_into<NT>(fx_fold(v), nrm + p);
        if (p > 0) {
            // base's low digits are k < Np: the padding of r Np adds to base's
            const int Np = Ns >> 3, k = t & (Np - 1);
            fx2* const q = sm + sg_pad((t - k) * 8 + k);
#pragma unroll
            for (int r = 0; r < 8; r++) q[sg_pad(r * Np)] = v[r];
        }
        __syncthreads();
        int s = max(fx_bits(nrm[p]) - FX_T, 0);
#pragma unroll
        for (int r = 0; r < 8; r++) v[r] = sm[sg_pad(t) + sg_pad(r * NT)];
        // the table for a shift of s, and the first twiddles ahead of the barrier
        const fxw* q = w + (max(s, FX_SMIN) - FX_SMIN) * fx_tw_entries() + (t & (Ns - 1));
        fxw ahead[FX_AHEAD];
#pragma unroll
        for (int r = 0; r < FX_AHEAD; r++) ahead[r] = fx_ldg_here(q + r * Ns);
        __syncthreads();
        E += s;
        if (s < FX_SMIN) {
            const int up = FX_SMIN - s;
#pragma unroll
            for (int r = 0; r < 8; r++) v[r] = fx2{v[r].x << up, v[r].y << up};
            s = FX_SMIN;
        }
        const long long h = 1ll << (s - 1);
        v[0] = fx2{(v[0].x + h) >> s, (v[0].y + h) >> s};
#pragma unroll
        for (int r = 1; r <= FX_AHEAD; r++) v[r] = fx_cmul<DIR>(v[r], ahead[r - 1]);
#pragma unroll
        for (int r = FX_AHEAD + 1; r < 8; r++) v[r] = fx_cmul<DIR>(v[r], fx_ldg(q + (r - 1) * Ns));
        fx_dft<8, DIR>(v);
        w += 7 * Ns;
        Ns <<= 3;
    }
}

// a block's exponent from the largest high word; FX_BAD marks infinities and NaN
__device__ __forceinline__ int fx_block_exp(unsigned abshi, int F) { return abshi >= 0x7ff00000u ? FX_BAD : fx_exp_of_field(F); }
// conversions of a whole block: the exponent is the same for all, so the test is uniform
__device__ __forceinline__ double2 fx_out(fx2 a, int E, bool safe)
{
    if (safe) return double2{fx_to_double(a.x, E), fx_to_double(a.y, E)};
    return double2{fx_to_double_any(a.x, E), fx_to_double_any(a.y, E)};
}
__device__ __forceinline__ double fx_weight(const void* w, int i, int wdf)
{
    return wdf ? df_to_double(reinterpret_cast<const dfloat*>(w)[i]) : reinterpret_cast<const double*>(w)[i];
}
// whether a warp's rows are weighted (at p = 0 every weight is 1): an integer
// comparison and a uniform branch around the products, which the FP64 pipe
// would otherwise take 16 cycles a warp instruction for
__device__ __forceinline__ bool fx_weighted(double w0, double w1)
{
    const long long one = 0x3ff0000000000000ll;
    return __any_sync(0xffffffffu, __double_as_longlong(w0) != one || __double_as_longlong(w1) != one);
}
// 32 bytes (a whole L2 sector): two complex values of one mode
__device__ __forceinline__ void fx_st256(double2* p, double2 a, double2 b, uint64_t pol)
{
    asm volatile("st.global.L2::cache_hint.v4.f64 [%0], {%1, %2, %3, %4}, %5;" ::"l"(p), "d"(a.x), "d"(a.y), "d"(b.x),
                 "d"(b.y), "l"(pol)
                 : "memory");
}

// The means of a pair of rows, each at the exponent of its row's largest value:
// 31 bits, 2^29 sum, or the first value where that is within 2^-20 of it, so
// that a constant row leaves nothing.
struct FxLevel {
    unsigned sum[2];
    fx2 first;
    static __device__ __forceinline__ long long pick(unsigned sum, long long first)
    {
        const long long m = (long long)(int)sum << 29;
        return fx_fold(first - m) < 1u << (FX_T - 20 - 32) ? first : m;
    }
    __device__ __forceinline__ fx2 mean() const { return fx2{pick(sum[0], first.x), pick(sum[1], first.y)}; }
};
// the exponent above the rest that a row leaves (folded), -FX_BAD for none
__device__ __forceinline__ int fx_rest_top(int E, unsigned folded)
{
    return folded || E == FX_BAD ? E + min(fx_bits(folded), FX_T) : -FX_BAD;
}
// a row's DC mode with the mean c that was taken off; largest, rest: its nrm words
template <int LG>
__device__ __forceinline__ double fx_with_mean(double dc, long long c, unsigned largest, unsigned rest)
{
    if (fx_bits(rest) > FX_T) return dc;
    const int E = fx_block_exp(largest, fx_field(largest)) + LG;
    const long long hi = c & ~((1ll << 29) - 1);  // exact as a double
    return dc + fx_to_double_any(c - hi, E) + fx_to_double_any(hi, E);
}

// ---------------------------------------------------------------------------
// P1 / P1b: one complex transform of two real sequences per slot, split into
// their half spectra.  Forward: rows 2p, 2p + 1 of sigma (x0), both halves to
// A[m][2p], A[m][2p + 1] as one 32-byte store.  Adjoint: row i of gF_r (x0)
// and gF_phi (x1), the halves to A and C, staged as S[m RB + row] and stored
// by tensor copies of RB rows.
// ---------------------------------------------------------------------------
template <int LG, bool BWD>
struct FxR2C {
    typedef FxShape<LG> S;
    static constexpr int SL = BWD ? S::RB : S::SL, THREADS = SL * S::NT;
    static constexpr size_t SMEM = SL * S::EX + 128;
    static constexpr int MINB = fx_minb(THREADS, SMEM);
};
template <int LG, bool BWD>
__global__ void __launch_bounds__(FxR2C<LG, BWD>::THREADS, FxR2C<LG, BWD>::MINB)
    k_fx_r2c(const double* __restrict__ x0, const double* __restrict__ x1, const void* __restrict__ wrow, int wdf,
             double2* __restrict__ A, int nu, const fxw* __restrict__ tw, int* err,
             const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapC)
{
    constexpr int N = 1 << LG, NT = N / 8, SL = FxR2C<LG, BWD>::SL;
    extern __shared__ __align__(128) unsigned char smraw[];
    __shared__ unsigned nrm[SL][7];  // the transform's three, the rows' largest values and those of their rests
    __shared__ FxLevel level[SL];
    unsigned char* const area = smraw + ((128 - (sg_smem_u32(smraw) & 127)) & 127);
    const int slot = threadIdx.x / NT, t = threadIdx.x % NT;
    fx2* const sm = reinterpret_cast<fx2*>(area) + (size_t)slot * (N + N / 16 + 1);
    if (t < 7) nrm[slot][t] = 0;
    if (t < 2) level[slot].sum[t] = 0;
    __syncthreads();
    const int u = blockIdx.x * SL + slot, rows = BWD ? nu : nu / 2;
    const bool live = u < rows;
    const int i0 = BWD ? (live ? u : 0) : 2 * (live ? u : 0);
    const double w0 = fx_weight(wrow, i0, wdf), w1 = BWD ? w0 : fx_weight(wrow, i0 + 1, wdf);
    sg_grid_dep_launch();
    sg_grid_dep_wait();  // the inputs may come from the previous kernel on the stream
    const double* const r0 = x0 + (size_t)i0 * N + t;
    const double* const r1 = BWD ? x1 + (size_t)i0 * N + t : r0 + N;
    double2 z[8];
#pragma unroll
    for (int e = 0; e < 8; e++) z[e] = double2{sg_ld_dep(r0 + e * NT), sg_ld_dep(r1 + e * NT)};
    if (fx_weighted(w0, w1)) {
        asm volatile("" ::: "memory");  // stays a branch
#pragma unroll
        for (int e = 0; e < 8; e++) z[e] = double2{z[e].x * w0, z[e].y * w1};
    }
    unsigned h0 = 0, h1 = 0;
#pragma unroll
    for (int e = 0; e < 8; e++) {
        h0 = max(h0, fx_abshi(z[e].x));
        h1 = max(h1, fx_abshi(z[e].y));
    }
    fx_both_into<NT, FxMax>(h0, h1, &nrm[slot][3]);
    __syncthreads();
    // Each row less its mean, and both at the exponent of what is left: a
    // disk's axisymmetric part would otherwise set the exponent that its other
    // modes are rounded at, and an axisymmetric row that of the weaker row that
    // shares its transform (1e-12 of a row of 1e-6 beside a constant 1).  The
    // mean is taken off exactly and added to the DC mode below, which holds
    // next to nothing else: whatever the row, its sum takes one rounding.
    // (Taking off the first value left the DC mode of a row with a peak there
    // as the difference of two numbers N times as large: 1e-13 of it, and 1e-15
    // of the row in all other modes, at 4096 points.)
    const int F0 = fx_field(nrm[slot][3]), F1 = fx_field(nrm[slot][4]);
    fx2 v[8];
    int m0 = 0, m1 = 0;
#pragma unroll
    for (int e = 0; e < 8; e++) {
        v[e] = fx2{fx_from_double(z[e].x, F0), fx_from_double(z[e].y, F1)};
        m0 += (int)(v[e].x >> 32);
        m1 += (int)(v[e].y >> 32);
    }
    constexpr int MS = LG - 3;  // the sum of the threads' eighths: 8 high words of the mean, below 2^31
    fx_both_into<NT, FxSum>((m0 + (1 << MS >> 1)) >> MS, (m1 + (1 << MS >> 1)) >> MS, level[slot].sum);
    if (t == 0) level[slot].first = v[0];
    __syncthreads();
    const fx2 c = level[slot].mean();
    unsigned g0 = 0, g1 = 0;
#pragma unroll
    for (int e = 0; e < 8; e++) {
        v[e] = fx_sub(v[e], c);
        g0 |= fx_fold(v[e].x);
        g1 |= fx_fold(v[e].y);
    }
    fx_both_into<NT, FxOr>(g0, g1, &nrm[slot][5]);
    __syncthreads();
    g0 = nrm[slot][5];
    g1 = nrm[slot][6];
    if (fx_bits(g0 | g1) > FX_T) {  // a rest that needs a bit more than its row had keeps the mean
        const fx2 k{fx_bits(g0) > FX_T ? c.x : 0, fx_bits(g1) > FX_T ? c.y : 0};
#pragma unroll
        for (int e = 0; e < 8; e++) v[e] = fx_add(v[e], k);
    }
    const int E0 = fx_block_exp(nrm[slot][3], F0), E1 = fx_block_exp(nrm[slot][4], F1);
    const int top = max(fx_rest_top(E0, g0), fx_rest_top(E1, g1));
    int E = top == -FX_BAD ? E0 : top - FX_T;
    const int l0 = min(max(E0 - E, 0), 63), l1 = min(max(E1 - E, 0), 63);
#pragma unroll
    for (int e = 0; e < 8; e++) v[e] = fx2{v[e].x << l0, v[e].y << l1};
    if (E > min(E0, E1)) {  // the weaker row gives way
#pragma unroll
        for (int e = 0; e < 8; e++) v[e] = fx2{fx_shift(v[e].x, max(E - E0, 0)), fx_shift(v[e].y, max(E - E1, 0))};
    }
    fx_fft<LG, -1>(v, sm, nrm[slot], t, tw, E);
    // X_a = (Z + conj Z[N - m]) / 2, X_b = (Z - conj Z[N - m]) / 2i, the halves of
    // a sum one down, one up (fx_half_sum): both down, half a unit off in every
    // mode's real part would add up at azimuth 0 (F_phi beside it, 4096 points:
    // 2.6e-15 of its rms, where FP64 sums leave 5e-16)
#pragma unroll
    for (int e = 0; e < 8; e++) sm[sg_pad(t + e * NT)] = v[e];
    __syncthreads();
    double2 xa[4], xb[4];
    const bool safe = fx_exp_safe(E);
#pragma unroll
    for (int e = 0; e < 4; e++) {
        const int m = t + e * NT;
        const fx2 a = v[e], b = sm[sg_pad((N - m) & (N - 1))];
        fx2 p{fx_half_sum(a.x, b.x), fx_half_diff(a.y, b.y)}, q{fx_half_sum(a.y, b.y), fx_half_diff(b.x, a.x)};
        if (e == 0 && t == 0) {  // (DC, Nyquist) of both
            const fx2 n = sm[sg_pad(N / 2)];
            p = fx2{v[0].x, n.x};
            q = fx2{v[0].y, n.y};
        }
        xa[e] = fx_out(p, E, safe);
        xb[e] = fx_out(q, E, safe);
        if (e == 0 && t == 0) {
            const fx2 c = level[slot].mean();
            xa[0].x = fx_with_mean<LG>(xa[0].x, c.x, nrm[slot][3], nrm[slot][5]);
            xb[0].x = fx_with_mean<LG>(xb[0].x, c.y, nrm[slot][4], nrm[slot][6]);
        }
    }
    const uint64_t keep = sg_policy_evict_last();  // the column pass reads the spectra from L2
    if constexpr (!BWD) {
        if (live) {
#pragma unroll
            for (int e = 0; e < 4; e++) {
                const size_t at = (size_t)(t + e * NT) * nu + i0;
                SG_IF_OK(sg_in((long long)at, 2, (long long)(N / 2) * nu), err, 901)
                fx_st256(A + at, xa[e], xb[e], keep);
            }
        }
    } else {
        __syncthreads();  // the stages span the exchange areas
        double2* const Sa = reinterpret_cast<double2*>(area);
        double2* const Sc = Sa + (size_t)SL * (N / 2);
#pragma unroll
        for (int e = 0; e < 4; e++) {
            Sa[(t + e * NT) * SL + slot] = xa[e];
            Sc[(t + e * NT) * SL + slot] = xb[e];
        }
        sg_fence_proxy_async();
        __syncthreads();
        if (threadIdx.x < 32) {
            const int ib = blockIdx.x * SL;
            constexpr int MB = N / 2 < 256 ? N / 2 : 256, NBOX = N / 2 / MB;
            for (int j = threadIdx.x; j < 2 * NBOX; j += 32) {
                const double2* src = (j < NBOX ? Sa : Sc) + (size_t)(j % NBOX) * MB * SL;
                SG_IF_OK(ib + SL <= nu && sg_smem_in(smraw, src, MB * SL * sizeof(double2)), err, 902)
                sg_tma_store_2d(j < NBOX ? &mapA : &mapC, 2 * ib, (j % NBOX) * MB, src, keep);
            }
            sg_bulk_commit();
            sg_bulk_wait_read();
        }
    }
}

// ---------------------------------------------------------------------------
// The products with the kernel spectra.  k1, k2: the two spectrum rows
// (columns m > 0: Khat_r, Khat_phi of mode m; mode 0 packs DC and Nyquist:
// Khat_r of both).  An entry's own exponent differs from its row's by dE
// (0..63); the products wait unaligned until the block's largest is known,
// and the entries' dE are then read again.
// ---------------------------------------------------------------------------
struct FxSpecRows {
    const fx2 *k1, *k2;
    bool z;  // mode 0
};
// kappa's entry for the frequency t + e NT, mirrored above N_u: Khat_r is
// Hermitian, Khat_phi anti-Hermitian
template <int NT>
__device__ __forceinline__ int fx_spec_index(int t, int e) { return e < 4 ? t + e * NT : (8 - e) * NT - t; }
template <int NT, bool SECOND>
__device__ __forceinline__ fx2 fx_spec_at(const FxSpecRows& K, int t, int e, int& dE)
{
    fx2 w = fx_ldg((SECOND ? K.k2 : K.k1) + fx_spec_index<NT>(t, e));
    dE = fx_spec_drop(w);
    w = fx_spec_mant(w);
    if (e > 4 || (e == 4 && t != 0)) {
        if (SECOND && !K.z)
            w.x = -w.x;
        else
            w.y = -w.y;
    }
    return w;
}
// the operand of the first (second) product at frequency k: the column's
// spectrum, or for mode 0 the spectrum of its DC (Nyquist) part, from Z and
// its mirror in sm
template <int LG, bool SECOND>
__device__ __forceinline__ fx2 fx_operand(fx2 a, const fx2* sm, int k, bool z)
{
    if (!z) return a;
    const fx2 b = sm[sg_pad(((1 << LG) - k) & ((1 << LG) - 1))];
    if (!SECOND) return fx2{fx_half_sum(a.x, b.x), fx_half_diff(a.y, b.y)};
    return fx2{fx_half_sum(a.y, b.y), fx_half_diff(b.x, a.x)};
}
// DIR < 0: a K, DIR > 0: a conj K; at 2^-64 of the factors' scale
template <int DIR>
__device__ __forceinline__ fx2 fx_product(fx2 a, fx2 w, int dE, unsigned& top)
{
    const fx2 p = fx_cmul<DIR>(a, fx_digits(w.x, w.y));
    top = max(top, (unsigned)(fx_bits(fx_fold(p)) + 64 - dE));
    return p;
}
// a product at the block's exponent: shift = bits above FX_T of the largest.
// Ties (one product in four at a shift of 1) go up at even frequencies and down
// at odd ones (t's parity: N / 8 is even): the bias of one sign that all going up
// leaves would add up in row 0 (2.5e-15 of F_r's rms at 2048 rows), this one's
// sum lies N_u rows on, where the column is cropped.
template <int NT, bool SECOND>
__device__ __forceinline__ fx2 fx_align(fx2 p, const FxSpecRows& K, int t, int e, int shift)
{
    const int2* w = reinterpret_cast<const int2*>((SECOND ? K.k2 : K.k1) + fx_spec_index<NT>(t, e));
    const int d = ((__ldg(&w[0].x) & 7) | (__ldg(&w[1].x) & 7) << 3) + shift;
    return fx2{fx_shift(p.x, d, t & 1), fx_shift(p.y, d, t & 1)};
}

template <int LG>
struct FxCols {
    typedef FxShape<LG> S;
    static constexpr int THREADS = S::SL * S::NT;
    static constexpr size_t SMEM = S::SL * (S::EX + S::PARK);
    static constexpr int MINB = fx_minb(THREADS, SMEM);
};

// the N_u values of a column as the first half of a zero-padded transform;
// top: a zeroed shared word.  Every thread of the block calls.
template <int NT>
__device__ __forceinline__ void fx_load_column(fx2 (&v)[8], const double2* __restrict__ in, unsigned* top, int& E)
{
    double2 a[4];
    unsigned h = 0;
#pragma unroll
    for (int e = 0; e < 4; e++) a[e] = sg_ld_dep(in + e * NT);
#pragma unroll
    for (int e = 0; e < 4; e++) h = max(h, max(fx_abshi(a[e].x), fx_abshi(a[e].y)));
    fx_max_into<NT>(h, top);
    __syncthreads();
    h = *top;
    const int F = fx_field(h);
    E = fx_block_exp(h, F);
#pragma unroll
    for (int e = 0; e < 4; e++) v[e] = fx2{fx_from_double(a[e].x, F), fx_from_double(a[e].y, F)};
#pragma unroll
    for (int e = 4; e < 8; e++) v[e] = fx2{0, 0};
}
__device__ __forceinline__ fx2 fx_conj(fx2 a) { return fx2{a.x, -a.y}; }
// a column's first N_u values, conjugated, to memory
template <int NT>
__device__ __forceinline__ void fx_store_column(const fx2 (&v)[8], double2* out, int E, bool live, long long at,
                                                long long extent, int* err, int site)
{
    const bool safe = fx_exp_safe(E);
    const uint64_t keep = sg_policy_evict_last();  // the row pass reads it from L2
    if (live)
#pragma unroll
        for (int e = 0; e < 4; e++)
            SG_IF_OK(sg_in(at + e * NT, 1, extent), err, site)
            sg_st_hint(out + e * NT, fx_out(fx_conj(v[e]), E, safe), keep);
}

// P2: column m of A, zero-padded transform, times both spectra, two inverse
// transforms cropped to N_u rows: B and C.
template <int LG>
__global__ void __launch_bounds__(FxCols<LG>::THREADS, FxCols<LG>::MINB)
    k_fx_fwd_cols(const double2* __restrict__ A, const fx2* __restrict__ Kr, const fx2* __restrict__ Kp,
                  double2* __restrict__ B, double2* __restrict__ C, int half, const fxw* __restrict__ tw, int* err)
{
    constexpr int L = 1 << LG, NT = L / 8, SL = FxShape<LG>::SL, nu = L / 2, KS = nu + 2;
    extern __shared__ __align__(128) unsigned char smraw[];
    __shared__ unsigned nrm[SL][12];  // three per transform, then the column's and the products' maxima
    const int slot = threadIdx.x / NT, t = threadIdx.x % NT;
    fx2* const sm = reinterpret_cast<fx2*>(smraw) + (size_t)slot * (L + L / 16 + 1);
    fx2* const park = reinterpret_cast<fx2*>(smraw + SL * FxShape<LG>::EX) + (size_t)slot * L;
    for (int j = t; j < 12; j += NT) nrm[slot][j] = 0;
    const int m0 = blockIdx.x * SL + slot;
    const bool live = m0 < half;
    const int m = live ? m0 : half - 1;
    const FxSpecRows K{Kr + (size_t)m * KS, m == 0 ? Kr + (size_t)half * KS : Kp + (size_t)m * KS, m == 0};
    __syncthreads();
    sg_grid_dep_launch();
    sg_grid_dep_wait();  // A is the previous pass's result
    fx2 v[8];
    int E, E2 = 0, shift2 = 0;
    fx_load_column<NT>(v, A + (size_t)m * nu + t, &nrm[slot][9], E);
#pragma unroll 1
    for (int pass = 0; pass < 3; pass++) {
        fx_fft<LG, -1>(v, sm, &nrm[slot][3 * pass], t, tw, E);
        if (pass > 0) {
            fx_store_column<NT>(v, (pass == 1 ? B : C) + (size_t)m * nu + t, E, live, (long long)m * nu + t,
                                (long long)half * nu, err, 903);
            if (pass == 1) {
#pragma unroll
                for (int e = 0; e < 8; e++)
                    v[e] = fx_conj(fx_align<NT, true>(park[t + e * NT], K, t, e, shift2));
                E = E2;
            }
            continue;
        }
        if (blockIdx.x == 0) {  // holds mode 0: the mirror of every frequency
#pragma unroll
            for (int e = 0; e < 8; e++) sm[sg_pad(t + e * NT)] = v[e];
            __syncthreads();
        }
        unsigned top1 = 0, top2 = 0;
#pragma unroll
        for (int e = 0; e < 8; e++) {
            const int k = t + e * NT;
            int d1, d2;
            const fx2 w2 = fx_spec_at<NT, true>(K, t, e, d2);
            park[k] = fx_product<-1>(fx_operand<LG, true>(v[e], sm, k, K.z), w2, d2, top2);
            const fx2 w1 = fx_spec_at<NT, false>(K, t, e, d1);
            v[e] = fx_product<-1>(fx_operand<LG, false>(v[e], sm, k, K.z), w1, d1, top1);
        }
        fx_max_into<NT>(top1, &nrm[slot][10]);
        fx_max_into<NT>(top2, &nrm[slot][11]);
        __syncthreads();
        const int q1 = (int)nrm[slot][10] - 64, q2 = (int)nrm[slot][11] - 64;
        const int EK1 = (int)fx_ldg(K.k1 + nu + 1).x, EK2 = (int)fx_ldg(K.k2 + nu + 1).x;
        if (K.z) {  // Y_r = Y_DC + i Y_Nyquist at one exponent; the azimuthal force of both modes vanishes
            const int EK = max(EK1, EK2), o1 = EK - EK1, o2 = EK - EK2, q = max(q1 - o1, q2 - o2) + 1;
#pragma unroll
            for (int e = 0; e < 8; e++) {
                const fx2 a = fx_align<NT, false>(v[e], K, t, e, o1 + q - FX_T);
                const fx2 b = fx_align<NT, true>(park[t + e * NT], K, t, e, o2 + q - FX_T);
                v[e] = fx_conj(fx2{a.x - b.y, a.y + b.x});
                park[t + e * NT] = fx2{0, 0};
            }
            E2 = E = E + EK + q + FX_PROD - FX_T;
        } else {
#pragma unroll
            for (int e = 0; e < 8; e++) v[e] = fx_conj(fx_align<NT, false>(v[e], K, t, e, q1 - FX_T));
            E2 = E + EK2 + q2 + FX_PROD - FX_T;
            shift2 = q2 - FX_T;
            E = E + EK1 + q1 + FX_PROD - FX_T;
        }
    }
}

// P2b: the columns of A and C, transforms, times conj Khat, summed, one
// inverse transform cropped to N_u rows: B.  Mode 0 takes both its operands
// (DC, Nyquist) from A: the azimuthal kernel vanishes there.
template <int LG>
__global__ void __launch_bounds__(FxCols<LG>::THREADS, FxCols<LG>::MINB)
    k_fx_bwd_cols(const double2* __restrict__ A, const double2* __restrict__ C, const fx2* __restrict__ Kr,
                  const fx2* __restrict__ Kp, double2* __restrict__ B, int half, const fxw* __restrict__ tw, int* err)
{
    constexpr int L = 1 << LG, NT = L / 8, SL = FxShape<LG>::SL, nu = L / 2, KS = nu + 2;
    extern __shared__ __align__(128) unsigned char smraw[];
    __shared__ unsigned nrm[SL][13];  // three per transform, the columns' maxima, the products' maxima
    const int slot = threadIdx.x / NT, t = threadIdx.x % NT;
    fx2* const sm = reinterpret_cast<fx2*>(smraw) + (size_t)slot * (L + L / 16 + 1);
    fx2* const park = reinterpret_cast<fx2*>(smraw + SL * FxShape<LG>::EX) + (size_t)slot * L;
    for (int j = t; j < 13; j += NT) nrm[slot][j] = 0;
    const int m0 = blockIdx.x * SL + slot;
    const bool live = m0 < half;
    const int m = live ? m0 : half - 1;
    const FxSpecRows K{Kr + (size_t)m * KS, m == 0 ? Kr + (size_t)half * KS : Kp + (size_t)m * KS, m == 0};
    __syncthreads();
    sg_grid_dep_launch();
    sg_grid_dep_wait();  // A and C are the previous pass's results
    fx2 v[8];
    int E, Ep0 = 0;
    fx_load_column<NT>(v, A + (size_t)m * nu + t, &nrm[slot][9], E);
#pragma unroll 1
    for (int pass = 0; pass < 3; pass++) {
        fx_fft<LG, -1>(v, sm, &nrm[slot][3 * pass], t, tw, E);
        if (pass == 2) {
            fx_store_column<NT>(v, B + (size_t)m * nu + t, E, live, (long long)m * nu + t, (long long)half * nu, err,
                                904);
            break;
        }
        if (blockIdx.x == 0) {
#pragma unroll
            for (int e = 0; e < 8; e++) sm[sg_pad(t + e * NT)] = v[e];
            __syncthreads();
        }
        unsigned top = 0;
        if (pass == 0) {
#pragma unroll
            for (int e = 0; e < 8; e++) {
                const int k = t + e * NT;
                int d;
                const fx2 w = fx_spec_at<NT, false>(K, t, e, d);
                park[k] = fx_product<+1>(fx_operand<LG, false>(v[e], sm, k, K.z), w, d, top);
            }
            fx_max_into<NT>(top, &nrm[slot][11]);
            Ep0 = E + (int)fx_ldg(K.k1 + nu + 1).x + FX_PROD - FX_T;
            __syncthreads();  // every mirror read is done
            fx_load_column<NT>(v, (K.z ? A : C) + (size_t)m * nu + t, &nrm[slot][10], E);
        } else {
#pragma unroll
            for (int e = 0; e < 8; e++) {
                int d;
                const fx2 w = fx_spec_at<NT, true>(K, t, e, d);
                v[e] = fx_product<+1>(fx_operand<LG, true>(v[e], sm, t + e * NT, K.z), w, d, top);
            }
            fx_max_into<NT>(top, &nrm[slot][12]);
            __syncthreads();  // every mirror read is done; the largest products are known
            // both products at the larger one's exponent, one bit of room for their sum
            const int q1 = (int)nrm[slot][11] - 64, q2 = (int)nrm[slot][12] - 64;
            const int Ep1 = E + (int)fx_ldg(K.k2 + nu + 1).x + FX_PROD - FX_T;
            E = max(Ep0 + q1, Ep1 + q2) + 1;
            const int s1 = E - Ep0 - FX_T, s2 = E - Ep1 - FX_T;
#pragma unroll
            for (int e = 0; e < 8; e++) {
                const fx2 a = fx_align<NT, false>(park[t + e * NT], K, t, e, s1);
                const fx2 b = fx_align<NT, true>(v[e], K, t, e, s2);
                v[e] = fx_conj(K.z ? fx2{a.x - b.y, a.y + b.x} : fx_add(a, b));
            }
        }
    }
}

// ---------------------------------------------------------------------------
// P3 / P3b: RB rows per block.  Forward: per row Z = B + i C (Hermitian halves
// expanded), inverse transform, F_r, F_phi = Re, Im.  Adjoint: per pair of
// rows Z = S_i0 + i S_i1, gsigma of i0, i0 + 1 = Re, Im.  The rows' modes
// arrive by 2-D tensor copies as S[m RB + r] (B, then C), each slot turns its
// own modes into fixed point in place (once, not once per use), and the
// exchange areas then lie over the stage.  The DC and Nyquist terms stay out of
// the transform and are added to its rows: a disk's axisymmetric part, and what
// the column pass's rounding of it leaves in the Nyquist mode that it is packed
// with, would otherwise set the exponent that its other modes are rounded at.
// ---------------------------------------------------------------------------
template <int LG, bool BWD>
struct FxC2R {
    typedef FxShape<LG> S;
    static constexpr int SL = BWD ? S::RB / 2 : S::RB, THREADS = SL * S::NT;
    static constexpr size_t STAGE = (size_t)S::RB * (S::N / 2) * sizeof(double2) * (BWD ? 1 : 2);
    static constexpr size_t SMEM = (SL * S::EX > STAGE ? SL * S::EX : STAGE) + 128;
    static constexpr int MINB = fx_minb(THREADS, SMEM);
};
template <int LG, bool BWD>
__global__ void __launch_bounds__(FxC2R<LG, BWD>::THREADS, FxC2R<LG, BWD>::MINB)
    k_fx_c2r(const void* __restrict__ wrow, int wdf, double* __restrict__ y0, double* __restrict__ y1, int nu,
             const fxw* __restrict__ tw, int* err, const __grid_constant__ CUtensorMap mapB,
             const __grid_constant__ CUtensorMap mapC)
{
    constexpr int N = 1 << LG, NT = N / 8, half = N / 2, RB = FxShape<LG>::RB, SL = FxC2R<LG, BWD>::SL;
    const unsigned long long wlim = sg_wait_budget(err);  // read once, early
    extern __shared__ __align__(128) unsigned char smraw[];
    __shared__ __align__(8) uint64_t bar;
    __shared__ unsigned nrm[SL][4];
    __shared__ double2 ends[SL][2];
    unsigned char* const area = smraw + ((128 - (sg_smem_u32(smraw) & 127)) & 127);
    const int slot = threadIdx.x / NT, t = threadIdx.x % NT;
    fx2* const sm = reinterpret_cast<fx2*>(area) + (size_t)slot * (N + N / 16 + 1);
    if (t < 4) nrm[slot][t] = 0;
    const int ib = blockIdx.x * RB, i0 = ib + (BWD ? 2 * slot : slot);
    const double w0 = fx_weight(wrow, i0, wdf), w1 = BWD ? fx_weight(wrow, i0 + 1, wdf) : w0;
    if (threadIdx.x == 0) sg_mbar_init(&bar, 1);
    __syncthreads();
    sg_grid_dep_launch();
    sg_grid_dep_wait();  // the spectra are the previous pass's results
    if (threadIdx.x < 32) {
        constexpr int MB = half < 256 ? half : 256, NBOX = half / MB, NB = (BWD ? 1 : 2) * NBOX;
        if (threadIdx.x == 0) sg_mbar_expect_tx(&bar, (uint32_t)(FxC2R<LG, BWD>::STAGE));
        __syncwarp();
        const uint64_t drop = sg_policy_evict_first();  // consumed here
        for (int j = threadIdx.x; j < NB; j += 32) {
            double2* dst = reinterpret_cast<double2*>(area) + (size_t)j * MB * RB;
            SG_IF_OK(ib + RB <= nu && sg_smem_in(smraw, dst, MB * RB * sizeof(double2)), err, 905)
            sg_tma_load_2d(dst, j < NBOX ? &mapB : &mapC, 2 * ib, (j % NBOX) * MB, &bar, drop);
        }
    }
    if (__syncthreads_or(!sg_mbar_wait_bounded(&bar, 0, err, 1, wlim))) return;  // inputs never arrived
    // this slot's two half spectra: element m at S0[m RB], S1[m RB]
    double2* const S0 = reinterpret_cast<double2*>(area) + (BWD ? 2 * slot : slot);
    double2* const S1 = BWD ? S0 + 1 : S0 + (size_t)half * RB;
    if (t < 2) {  // DC +- Nyquist, which even and odd places take as one number (the azimuthal force has neither)
        const double2 a = S0[0], b = BWD ? S1[0] : double2{0.0, 0.0};
        ends[slot][t] = t ? double2{a.x - a.y, b.x - b.y} : double2{a.x + a.y, b.x + b.y};
    }
    int E;
    {
        double2 a[4], b[4];
        unsigned h = 0;
#pragma unroll
        for (int e = 0; e < 4; e++) {
            a[e] = S0[(t + e * NT) * RB];
            b[e] = S1[(t + e * NT) * RB];
            if (e == 0 && t == 0) a[0] = b[0] = double2{0.0, 0.0};
            h = max(h, max(max(fx_abshi(a[e].x), fx_abshi(a[e].y)), max(fx_abshi(b[e].x), fx_abshi(b[e].y))));
        }
        fx_max_into<NT>(h, &nrm[slot][3]);
        __syncthreads();
        h = nrm[slot][3];
        const int F = fx_field(h) + 1;  // one bit of room: Z adds two of them
        E = fx_block_exp(h, F);
#pragma unroll
        for (int e = 0; e < 4; e++) {
            reinterpret_cast<fx2*>(S0)[(t + e * NT) * RB] = fx2{fx_from_double(a[e].x, F), fx_from_double(a[e].y, F)};
            reinterpret_cast<fx2*>(S1)[(t + e * NT) * RB] = fx2{fx_from_double(b[e].x, F), fx_from_double(b[e].y, F)};
        }
    }
    __syncthreads();
    fx2 v[8];
#pragma unroll
    for (int e = 0; e < 8; e++) {
        const int n = t + e * NT, mo = e < 4 ? n : (n == half ? 0 : N - n);
        const fx2 a = reinterpret_cast<const fx2*>(S0)[mo * RB], b = reinterpret_cast<const fx2*>(S1)[mo * RB];
        v[e] = e < 4 ? fx2{a.x - b.y, a.y + b.x}   // a + i b
                     : fx2{a.x + b.y, b.x - a.y};  // conj a + i conj b
    }
    __syncthreads();  // the exchange areas lie over the stage
    fx_fft<LG, +1>(v, sm, nrm[slot], t, tw, E);
    const bool safe = fx_exp_safe(E);
    double* const o0 = y0 + (size_t)i0 * N + t;
    double* const o1 = BWD ? y0 + (size_t)(i0 + 1) * N + t : y1 + (size_t)i0 * N + t;
    const double2 end = ends[slot][t & 1];  // N / 8 is even: the parity of all its places
    double2 z[8];
#pragma unroll
    for (int e = 0; e < 8; e++) {
        z[e] = fx_out(v[e], E, safe);
        z[e].x += end.x;
        if (BWD) z[e].y += end.y;
    }
    if (fx_weighted(w0, w1)) {
        asm volatile("" ::: "memory");  // stays a branch
#pragma unroll
        for (int e = 0; e < 8; e++) z[e] = double2{z[e].x * w0, z[e].y * w1};
    }
    SG_IF_OK(i0 + (BWD ? 2 : 1) <= nu, err, 906)
#pragma unroll
    for (int e = 0; e < 8; e++) {
        o0[e * NT] = z[e].x;
        o1[e * NT] = z[e].y;
    }
}

// ---------------------------------------------------------------------------
// one length's kernels, reached through fx_kernels()
// ---------------------------------------------------------------------------
typedef void (*FxR2CFn)(const double*, const double*, const void*, int, double2*, int, const fxw*, int*, CUtensorMap,
                        CUtensorMap);
typedef void (*FxFwdColsFn)(const double2*, const fx2*, const fx2*, double2*, double2*, int, const fxw*, int*);
typedef void (*FxBwdColsFn)(const double2*, const double2*, const fx2*, const fx2*, double2*, int, const fxw*, int*);
typedef void (*FxC2RFn)(const void*, int, double*, double*, int, const fxw*, int*, CUtensorMap, CUtensorMap);
struct FxKernels {
    FxR2CFn r2c[2];  // forward, adjoint
    FxC2RFn c2r[2];
    FxFwdColsFn fwd_cols;
    FxBwdColsFn bwd_cols;
    int r2c_threads[2], c2r_threads[2], cols_threads;
    size_t r2c_smem[2], c2r_smem[2], cols_smem;
    int r2c_slots, cols_slots, rows;  // row pairs per forward R2C block, modes per column block, rows per other block
};
template <int LG>
FxKernels make_fx_kernels()
{
    return FxKernels{{k_fx_r2c<LG, false>, k_fx_r2c<LG, true>},
                     {k_fx_c2r<LG, false>, k_fx_c2r<LG, true>},
                     k_fx_fwd_cols<LG>,
                     k_fx_bwd_cols<LG>,
                     {FxR2C<LG, false>::THREADS, FxR2C<LG, true>::THREADS},
                     {FxC2R<LG, false>::THREADS, FxC2R<LG, true>::THREADS},
                     FxCols<LG>::THREADS,
                     {FxR2C<LG, false>::SMEM, FxR2C<LG, true>::SMEM},
                     {FxC2R<LG, false>::SMEM, FxC2R<LG, true>::SMEM},
                     FxCols<LG>::SMEM,
                     FxShape<LG>::SL,
                     FxShape<LG>::SL,
                     FxShape<LG>::RB};
}
FxKernels fx_kernels_lg6();
FxKernels fx_kernels_lg7();
FxKernels fx_kernels_lg8();
FxKernels fx_kernels_lg9();
FxKernels fx_kernels_lg10();
FxKernels fx_kernels_lg11();
FxKernels fx_kernels_lg12();

}  // namespace sg
