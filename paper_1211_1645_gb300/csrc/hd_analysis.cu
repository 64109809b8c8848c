// hd_analysis.cu -- analysis of the measured chain (Engel et al.,
// arXiv:1211.1645): the autocorrelation of the global orientational order
// Psi_6 over the recorded measurement series and the correlation time of its
// exponential part (Sec. III, Eq. 9, Table II), and the coarse-grained psi_6
// field, the mean of psi_j over square sampling areas (Sec. IV, Figs. 5-6);
// the structure factor, the choice of q_0 at its maximum, the positional
// order chi_j and the positional correlation function (Sec. IV.C, Eqs. 10-12).
#include <math_constants.h>

#include <algorithm>
#include <vector>

#include "hd_kernels.h"
#include "hd_analysis.h"
#include "hd_cell.cuh"

namespace hd {

// Series row layout: series[(t * R + r) * 4 + {0: beta P / rho, 1: g(2 sigma+), 2: Re Psi_6, 3: Im Psi_6}].
//
// S[r][d] = sum_{t < T - d} Psi(t) conj(Psi(t + d)).  A block takes 128 lags
// (one per thread) and kAcfChunk times, staged with the entries the lags reach;
// the partial sums of the chunks are added in order by k_acf_norm.  What bounds
// it is FP64: four fused multiply-adds per term at two lanes per clock and SM.
// One thread per lag over all T instead ran a serial chain of loads and adds
// (T = 4000, 401 lags, four replicas: 2.31 ms, here 0.07).
constexpr int kAcfLags = 128, kAcfChunk = 128;

__global__ void __launch_bounds__(kAcfLags)
k_acf_sums(const double* __restrict__ series, int R, int64_t T, int64_t max_lag, int64_t len, double2* __restrict__ part) {
    pdl_begin(series);
    __shared__ double2 s_a[kAcfChunk], s_c[kAcfChunk + kAcfLags];
    const int r = blockIdx.y;
    const int64_t d0 = int64_t(blockIdx.x) * kAcfLags, d = d0 + threadIdx.x;
    const int64_t t1 = min(T, int64_t(blockIdx.z + 1) * len);
    auto entry = [&](int64_t t) {
        const double* row = series + (size_t(t) * R + r) * 4;
        return t < T ? make_double2(row[2], row[3]) : make_double2(0.0, 0.0);
    };
    double sr = 0.0, si = 0.0, ur = 0.0, ui = 0.0;  // two chains per part
    for (int64_t t0 = int64_t(blockIdx.z) * len; t0 < t1; t0 += kAcfChunk) {
        for (int i = threadIdx.x; i < kAcfChunk + kAcfLags; i += kAcfLags) {
            s_c[i] = entry(t0 + d0 + i);
            if (i < kAcfChunk) s_a[i] = entry(t0 + i);
        }
        __syncthreads();
        // a pair whose later entry is beyond the series is not part of the
        // sum, also where the series holds an infinity or NaN
        const int n = d > max_lag ? 0 : int(max(int64_t(0), min(min(int64_t(kAcfChunk), t1 - t0), T - d - t0)));
        for (int i = 0; i < n; ++i) {
            const double2 a = s_a[i], c = s_c[i + int(threadIdx.x)];
            // (a.x + i a.y)(c.x - i c.y) = (a.x c.x + a.y c.y) + i (a.y c.x - a.x c.y)
            sr = __fma_rn(a.x, c.x, sr);
            ur = __fma_rn(a.y, c.y, ur);
            si = __fma_rn(a.y, c.x, si);
            ui = __fma_rn(a.x, c.y, ui);
        }
        __syncthreads();
    }
    if (d <= max_lag)
        part[(size_t(blockIdx.z) * R + r) * size_t(max_lag + 1) + size_t(d)] = make_double2(__dadd_rn(sr, ur), __dsub_rn(si, ui));
}

// Eq. 9: C(d) = (S(d) / (T - d)) / (S(0) / T), S from the chunks' partial sums
// in order; blockIdx.y = replica.  Every block adds up S(0) itself.
__global__ void __launch_bounds__(128)
k_acf_norm(int R, int64_t T, int64_t max_lag, int chunks, const double2* __restrict__ part, double2* __restrict__ C) {
    pdl_begin(part);
    __shared__ double s_zero[128];
    const int r = blockIdx.y;
    const size_t row = size_t(max_lag + 1), step = size_t(R) * row;
    const double2* p = part + size_t(r) * row;
    double z = 0.0;
    for (int c = threadIdx.x; c < chunks; c += 128) z = __dadd_rn(z, p[size_t(c) * step].x);
    s_zero[threadIdx.x] = z;
    __syncthreads();
    for (int o = 64; o > 0; o >>= 1) {
        if (int(threadIdx.x) < o) s_zero[threadIdx.x] = __dadd_rn(s_zero[threadIdx.x], s_zero[threadIdx.x + o]);
        __syncthreads();
    }
    const int64_t d = int64_t(blockIdx.x) * 128 + threadIdx.x;
    if (d > max_lag) return;
    const double den = __ddiv_rn(s_zero[0], double(T));
    double a = 0.0, b = 0.0;
    for (int c = 0; c < chunks; ++c) {
        const double2 v = p[size_t(c) * step + size_t(d)];
        a = __dadd_rn(a, v.x);
        b = __dadd_rn(b, v.y);
    }
    const double n = double(T - d);
    // S(0) as the denominator has it, so that C(0) = 1
    if (d == 0) a = s_zero[0];
    C[size_t(r) * row + size_t(d)] = make_double2(__ddiv_rn(__ddiv_rn(a, n), den), __ddiv_rn(__ddiv_rn(b, n), den));
}

__device__ __forceinline__ double lane_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = __dadd_rn(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Correlation time of the exponential part: least-squares line through
// (d, ln Re C(d)) over lag_lo <= d <= lag_hi with Re C > 0, tau = -1 / slope
// (NaN with fewer than two such lags or a slope >= 0).  One warp per replica.
__global__ void __launch_bounds__(32)
k_acf_tau(int64_t max_lag, int64_t lag_lo, int64_t lag_hi, const double2* __restrict__ C, double* __restrict__ tau) {
    pdl_begin(C);
    const double2* row = C + size_t(blockIdx.x) * size_t(max_lag + 1);
    const int lane = int(threadIdx.x);
    double sx = 0.0, sy = 0.0, cnt = 0.0;
    for (int64_t d = lag_lo + lane; d <= lag_hi; d += 32) {
        if (row[d].x > 0.0) {
            sx = __dadd_rn(sx, double(d));
            sy = __dadd_rn(sy, log(row[d].x));
            cnt += 1.0;
        }
    }
    sx = lane_sum(sx);
    sy = lane_sum(sy);
    cnt = lane_sum(cnt);
    double out = CUDART_NAN;
    if (cnt >= 2.0) {
        const double mx = __ddiv_rn(sx, cnt), my = __ddiv_rn(sy, cnt);
        double sxy = 0.0, sxx = 0.0;
        for (int64_t d = lag_lo + lane; d <= lag_hi; d += 32) {
            if (row[d].x > 0.0) {
                const double dx = __dsub_rn(double(d), mx);
                sxy = __dadd_rn(sxy, __dmul_rn(dx, __dsub_rn(log(row[d].x), my)));
                sxx = __dadd_rn(sxx, __dmul_rn(dx, dx));
            }
        }
        const double slope = __ddiv_rn(lane_sum(sxy), lane_sum(sxx));
        if (slope < 0.0) out = __ddiv_rn(-1.0, slope);
    }
    if (lane == 0) tau[blockIdx.x] = out;
}

// Coarse field, accumulation: one thread per disk (global id order), from
// the global positions and the local psi_6 of the same state.  Area index
// floor(x bins / L) per axis (FP64), or floor(X bins / LF) of the exact
// integer coordinate X = x 2^24 (fixed form); acc[r][area] = (sum Re, sum Im, count).
__global__ void __launch_bounds__(256)
k_field_accum(const Rep* __restrict__ reps, int R, int64_t Ntot, bool fixed, int bins, const double* __restrict__ xy,
              const double2* __restrict__ psi, double* __restrict__ acc) {
    pdl_begin(xy, psi);
    const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= Ntot) return;
    int lo = 0, hi = R - 1;  // replica of global id i: last one with id_off <= i
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (reps[mid].id_off <= i) lo = mid; else hi = mid - 1;
    }
    const Rep& rep = reps[lo];
    // xy holds caller units (sigma times the internal ones)
    const double x = __ddiv_rn(xy[2 * i], rep.sigma), y = __ddiv_rn(xy[2 * i + 1], rep.sigma);
    int64_t ix, iy;
    if (fixed) {
        const int64_t X = llrint(__dmul_rn(x, 16777216.0)), Y = llrint(__dmul_rn(y, 16777216.0));
        ix = (X * bins) / rep.LF;
        iy = (Y * bins) / rep.LF;
    } else {
        ix = int64_t(floor(__ddiv_rn(__dmul_rn(x, double(bins)), rep.L)));
        iy = int64_t(floor(__ddiv_rn(__dmul_rn(y, double(bins)), rep.L)));
    }
    ix = ix < bins ? ix : bins - 1;
    iy = iy < bins ? iy : bins - 1;
    double* a = acc + (size_t(lo) * size_t(bins) * size_t(bins) + size_t(iy) * bins + size_t(ix)) * 3;
    const double2 v = psi[i];
    atomicAdd(a + 0, v.x);
    atomicAdd(a + 1, v.y);
    atomicAdd(a + 2, 1.0);
}

// Coarse field, means: out[r][iy][ix] = (sum Re, sum Im) / count, NaN if empty.
__global__ void __launch_bounds__(256)
k_field_norm(int64_t cells, const double* __restrict__ acc, double2* __restrict__ out) {
    pdl_begin(acc);
    const int64_t c = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (c >= cells) return;
    const double n = acc[3 * c + 2];
    out[c] = n > 0.0 ? make_double2(__ddiv_rn(acc[3 * c], n), __ddiv_rn(acc[3 * c + 1], n))
                     : make_double2(CUDART_NAN, CUDART_NAN);
}

// ---------------------------------------------------------------------------
// Positional order.  Wave vectors are the box-periodic q = 2 pi (h, k) / L;
// the phase q . x is taken as the turn fraction t = (h x + k y) / L mod 1 --
// exact in the fixed-point form, where x = X 2^-24 and L = LF 2^-24 -- and
// exp(i q . x) = (cospi(2t), sinpi(2t)).
// ---------------------------------------------------------------------------
__device__ __forceinline__ double2 plane_wave(const Rep& rep, bool fixed, int h, int k, double x, double y) {
    double t;
    if (fixed) {
        const int64_t X = llrint(__dmul_rn(x, 16777216.0)), Y = llrint(__dmul_rn(y, 16777216.0));
        int64_t a = (int64_t(h) * X + int64_t(k) * Y) % rep.LF;  // |h X| < 2^17 2^38
        if (a < 0) a += rep.LF;
        t = __ddiv_rn(double(a), double(rep.LF));
    } else {
        t = __ddiv_rn(__dadd_rn(__dmul_rn(double(h), x), __dmul_rn(double(k), y)), rep.Lm);
        t = __dsub_rn(t, floor(t));
    }
    double s, c;
    sincospi(__dmul_rn(2.0, t), &s, &c);
    return make_double2(c, s);
}

// Replica of global disk id i: the last one with id_off <= i.
__device__ __forceinline__ int rep_of_id(const Rep* __restrict__ reps, int R, int64_t i) {
    int lo = 0, hi = R - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (reps[mid].id_off <= i) lo = mid; else hi = mid - 1;
    }
    return lo;
}

constexpr int kSqChunk = 16;  // wave vectors per block of the amplitude kernel

// Amplitudes A_r(q) = sum_n exp(i q . x_n): blockIdx.z = replica, blockIdx.y =
// chunk of wave vectors, blockIdx.x = block of the replica's disks; one
// partial sum per (replica, disk block, q), reduced in a fixed order later.
__global__ void __launch_bounds__(256)
k_sq_amp(const Rep* __restrict__ reps, bool fixed, int nq, const int2* __restrict__ hk, const double* __restrict__ xy,
         int nbx, double2* __restrict__ part) {
    pdl_begin(hk, xy);
    const int r = blockIdx.z;
    const Rep& rep = reps[r];
    const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    const bool live = i < rep.N;
    const double x = live ? __ddiv_rn(xy[2 * (rep.id_off + i)], rep.sigma) : 0.0;
    const double y = live ? __ddiv_rn(xy[2 * (rep.id_off + i) + 1], rep.sigma) : 0.0;
    __shared__ double s_re[kSqChunk][8], s_im[kSqChunk][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int q0 = blockIdx.y * kSqChunk;
    for (int j = 0; j < kSqChunk; ++j) {
        const int q = q0 + j;
        double2 v = make_double2(0.0, 0.0);
        if (live && q < nq) {
            const int2 m = hk[size_t(r) * nq + q];
            v = plane_wave(rep, fixed, m.x, m.y, x, y);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            v.x += __shfl_down_sync(0xffffffffu, v.x, o);
            v.y += __shfl_down_sync(0xffffffffu, v.y, o);
        }
        if (lane == 0) {
            s_re[j][warp] = v.x;
            s_im[j][warp] = v.y;
        }
    }
    __syncthreads();
    if (threadIdx.x < kSqChunk && q0 + int(threadIdx.x) < nq) {
        double a = 0.0, b = 0.0;
        for (int w = 0; w < int(blockDim.x >> 5); ++w) {
            a += s_re[threadIdx.x][w];
            b += s_im[threadIdx.x][w];
        }
        part[(size_t(r) * nbx + blockIdx.x) * nq + q0 + threadIdx.x] = make_double2(a, b);
    }
}

// ---------------------------------------------------------------------------
// The same amplitudes for wave vectors that share their components, as a map
// or a window of them does: with U_n(h) = exp(2 pi i h x_n / L) and V_n(k)
// likewise, A(h, k) = sum_n U_n(h) V_n(k), so a disk needs one plane wave per
// distinct h and k (15 FP64 operations each here) and four fused
// multiply-adds per (h, k), against ~100 FP64-pipe operations for the division
// and the sine and cosine of every (h, k) itself.  FP64 rate is the bound:
// N = 65,536 and 441 wave vectors of 21 x 21 components 2.88 ms before, 0.33
// here.  The turn x / L is kept to 96 bits, so that h x / L mod 1 is exact to
// 2^-64 for every 32-bit h (the division in double loses h 2^-53 of a turn).
// ---------------------------------------------------------------------------
constexpr int kPairDisks = 32;      // disks staged at a time
constexpr int kPairThreads = 256;
constexpr int kPairMax = 160;       // distinct h plus distinct k of a replica
constexpr int kPairQ = 2;           // wave vectors per thread
constexpr int kTurnTable = 128;

struct Turn {
    unsigned long long hi;  // x / L mod 1 in units of 2^-64 ...
    uint32_t lo;            // ... and the next 32 bits
};

// X / LF for 0 <= X < LF < 2^42, digit by digit (22 bits at a time).
__device__ __forceinline__ Turn turn_fixed(uint64_t X, uint64_t LF) {
    uint64_t digit[5], rem = X;
#pragma unroll
    for (int k = 0; k < 5; ++k) {  // 110 bits
        rem <<= 22;
        digit[k] = rem / LF;
        rem -= digit[k] * LF;
    }
    Turn t;
    t.hi = digit[0] << 42 | digit[1] << 20 | digit[2] >> 2;
    t.lo = uint32_t((digit[2] & 3u) << 30 | digit[3] << 8 | digit[4] >> 14);
    return t;
}

// x / L mod 1 for finite x >= 0: the rounded quotient and the quotient of the
// exact remainder.
__device__ __forceinline__ Turn turn_fp64(double x, double L) {
    const double q = __ddiv_rn(x, L), q2 = __ddiv_rn(__fma_rn(-q, L, x), L);
    const double f = __dsub_rn(q, floor(q)), a = __dmul_rn(f, 281474976710656.0), ai = floor(a);  // 2^48
    const uint64_t top = uint64_t(ai), mid = uint64_t(__dmul_rn(__dsub_rn(a, ai), 281474976710656.0));
    // top 2^-48 + mid 2^-96, plus q2 (|q2| < 2^-52) in units of 2^-96
    const int64_t low = llrint(__dmul_rn(q2, 79228162514264337593543950336.0));
    const uint64_t m = mid + uint64_t(low);  // 48 bits, and a carry or borrow
    const int64_t carry = int64_t(m) >> 48;
    const uint64_t t48 = top + uint64_t(carry), m48 = m & ((uint64_t(1) << 48) - 1u);
    return Turn{t48 << 16 | m48 >> 32, uint32_t(m48)};
}

// exp(2 pi i h t): the nearest of 128 table angles and a Taylor polynomial of
// the remainder (|r| <= pi / 128: r^9 / 9! < 10^-20, r^8 / 8! < 10^-17).
__device__ __forceinline__ double2 turn_wave(const Turn& t, int h, const double2* table) {
    const uint64_t p = t.hi * uint64_t(int64_t(h)) + uint64_t((int64_t(t.lo) * int64_t(h)) >> 32);
    const uint64_t near = p + (uint64_t(1) << 56);
    const int64_t rem = int64_t(p - (near >> 57 << 57));  // in [-2^56, 2^56)
    // rem / 2^5 is an integer of 52 bits: exact through the exponent trick
    const double v = __dsub_rn(__longlong_as_double(0x4338000000000000ll + (rem >> 5)), 6755399441055744.0);  // 1.5 2^52
    const double r = __dmul_rn(v, 1.0899589056276974e-17);  // 2 pi 2^-59
    const double z = __dmul_rn(r, r);
    double s = __fma_rn(z, -1.0 / 5040.0, 1.0 / 120.0);
    s = __fma_rn(z, s, -1.0 / 6.0);
    s = __fma_rn(__dmul_rn(z, s), r, r);
    double c = __fma_rn(z, -1.0 / 720.0, 1.0 / 24.0);
    c = __fma_rn(z, c, -0.5);
    c = __dmul_rn(z, c);  // cos r - 1
    const double2 e = table[near >> 57];
    return make_double2(__dadd_rn(e.x, __fma_rn(e.x, c, -__dmul_rn(e.y, s))),
                        __dadd_rn(e.y, __fma_rn(e.y, c, __dmul_rn(e.x, s))));
}

// blockIdx.x: share of the replica's disks (32 at a time), blockIdx.y: 512 of
// its wave vectors, blockIdx.z: replica.  comp[r]: its nh distinct h, then its
// nk distinct k; pair[r][q]: indices of q's components.  With few wave vectors
// the threads split into groups that take every groups-th disk.
__global__ void __launch_bounds__(kPairThreads)
k_sq_pairs(const Rep* __restrict__ reps, bool fixed, int nq, int nh, int nk, const int* __restrict__ comp,
           const ushort2* __restrict__ pair, const double* __restrict__ xy, double2* __restrict__ part) {
    pdl_begin(comp, pair, xy);
    extern __shared__ double2 s_wave[];  // [kPairDisks][nh + nk], then the table
    __shared__ Turn s_turn[kPairDisks][2];
    const int r = blockIdx.z, nc = nh + nk, tid = int(threadIdx.x);
    const Rep& rep = reps[r];
    double2* table = s_wave + kPairDisks * nc;
    for (int j = tid; j < kTurnTable; j += kPairThreads) {
        double s, c;
        sincospi(double(j) * (2.0 / kTurnTable), &s, &c);
        table[j] = make_double2(c, s);
    }
    const int q0 = blockIdx.y * (kPairThreads * kPairQ), here = min(nq - q0, kPairThreads * kPairQ);
    int groups = 1;
    while (groups < 8 && 2 * groups * here <= kPairThreads) groups *= 2;
    const int width = kPairThreads / groups, group = tid / width, lane = tid - group * width;
    int ih[kPairQ], ik[kPairQ];
    bool mine[kPairQ];
    double re[kPairQ], im[kPairQ];
#pragma unroll
    for (int j = 0; j < kPairQ; ++j) {
        const int q = lane + j * width;
        mine[j] = q < here;
        const ushort2 p = mine[j] ? pair[size_t(r) * nq + q0 + q] : make_ushort2(0, 0);
        ih[j] = p.x;
        ik[j] = nh + p.y;
        re[j] = im[j] = 0.0;
    }
    const bool second = width < here;  // the second wave vector of a thread is in use
    const int* cr = comp + size_t(r) * nc;
    for (int64_t base = int64_t(blockIdx.x) * kPairDisks; base < rep.N; base += int64_t(gridDim.x) * kPairDisks) {
        __syncthreads();
        if (tid < 2 * kPairDisks) {
            const int64_t i = base + (tid >> 1);
            Turn t{0ull, 0u};
            if (i < rep.N) {
                double x = xy[2 * (rep.id_off + i) + (tid & 1)];
                if (rep.sigma != 1.0) x = __ddiv_rn(x, rep.sigma);
                t = fixed ? turn_fixed(uint64_t(llrint(__dmul_rn(x, 16777216.0))) % uint64_t(rep.LF), uint64_t(rep.LF))
                          : turn_fp64(x, rep.Lm);
            }
            s_turn[tid >> 1][tid & 1] = t;
        }
        __syncthreads();
        for (int e = tid; e < kPairDisks * nc; e += kPairThreads) {
            const int n = e / nc, j = e - n * nc;
            s_wave[e] = base + n < rep.N ? turn_wave(s_turn[n][j >= nh], cr[j], table) : make_double2(0.0, 0.0);
        }
        __syncthreads();
        for (int n = group; n < kPairDisks; n += groups) {
            const double2* w = s_wave + n * nc;
#pragma unroll
            for (int j = 0; j < kPairQ; ++j) {
                if (j == 1 && !second) break;
                const double2 u = w[ih[j]], v = w[ik[j]];
                re[j] = __fma_rn(u.x, v.x, re[j]);
                im[j] = __fma_rn(u.x, v.y, im[j]);
                re[j] = __fma_rn(-u.y, v.y, re[j]);
                im[j] = __fma_rn(u.y, v.x, im[j]);
            }
        }
    }
    // the groups' sums in order (the waves' space is free: 2 KB at least)
    __syncthreads();
    double2* s_sum = s_wave;
    for (int g = 1; g < groups; ++g) {
        if (group == g && mine[0]) s_sum[lane] = make_double2(re[0], im[0]);
        __syncthreads();
        if (group == 0 && mine[0]) {
            re[0] = __dadd_rn(re[0], s_sum[lane].x);
            im[0] = __dadd_rn(im[0], s_sum[lane].y);
        }
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < kPairQ; ++j)
        if (group == 0 && mine[j])
            part[(size_t(r) * gridDim.x + blockIdx.x) * nq + q0 + lane + j * width] = make_double2(re[j], im[j]);
}

// The same for wave vectors on a full grid of consecutive components, h = hc - j
// .. hc + j and k: with alpha = 2 pi x_n / L and B_n(k) = U_n(hc) V_n(k),
// A(hc +- j, k) = sum_n B_n(k) cos(j alpha_n) +- i sum_n B_n(k) sin(j alpha_n),
// so the two wave vectors of a sign share two sums of a complex times a real:
// two fused multiply-adds each instead of four (326 -> 275 us for 21 x 21 and
// 65,536 disks).  Unit (j, k) of a thread holds both sums.  comp[r] as above,
// each part ascending without gaps; part: [r][block][nh nk].
__global__ void __launch_bounds__(kPairThreads)
k_sq_grid(const Rep* __restrict__ reps, bool fixed, int nh, int nk, const int* __restrict__ comp,
          const double* __restrict__ xy, double2* __restrict__ part) {
    pdl_begin(comp, xy);
    extern __shared__ double2 s_wave[];  // [kPairDisks][nk + 1 + J], then the table
    __shared__ Turn s_turn[kPairDisks][2];
    const int r = blockIdx.z, tid = int(threadIdx.x);
    const int J = nh / 2, nw = nk + 1 + J, units = (J + 1) * nk;  // centre h: entry J of the nh
    const Rep& rep = reps[r];
    double2* table = s_wave + kPairDisks * nw;
    for (int j = tid; j < kTurnTable; j += kPairThreads) {
        double s, c;
        sincospi(double(j) * (2.0 / kTurnTable), &s, &c);
        table[j] = make_double2(c, s);
    }
    int groups = 1;
    while (groups < 8 && 2 * groups * units <= kPairThreads) groups *= 2;
    const int width = kPairThreads / groups, group = tid / width, lane = tid - group * width;
    int uj[kPairQ], uk[kPairQ];
    bool mine[kPairQ];
    double cr[kPairQ], ci[kPairQ], sr[kPairQ], si[kPairQ];
#pragma unroll
    for (int q = 0; q < kPairQ; ++q) {
        const int u = lane + q * width;
        mine[q] = u < units;
        uj[q] = mine[q] ? u / nk : 0;
        uk[q] = mine[q] ? u - uj[q] * nk : 0;
        cr[q] = ci[q] = sr[q] = si[q] = 0.0;
    }
    const bool second = width < units;
    const int* co = comp + size_t(r) * (nh + nk);
    const int hc = co[J];
    for (int64_t base = int64_t(blockIdx.x) * kPairDisks; base < rep.N; base += int64_t(gridDim.x) * kPairDisks) {
        __syncthreads();
        if (tid < 2 * kPairDisks) {
            const int64_t i = base + (tid >> 1);
            Turn t{0ull, 0u};
            if (i < rep.N) {
                double x = xy[2 * (rep.id_off + i) + (tid & 1)];
                if (rep.sigma != 1.0) x = __ddiv_rn(x, rep.sigma);
                t = fixed ? turn_fixed(uint64_t(llrint(__dmul_rn(x, 16777216.0))) % uint64_t(rep.LF), uint64_t(rep.LF))
                          : turn_fp64(x, rep.Lm);
            }
            s_turn[tid >> 1][tid & 1] = t;
        }
        __syncthreads();
        // V(k), then U(hc), then (cos, sin) of j alpha for j = 1 .. J
        for (int e = tid; e < kPairDisks * nw; e += kPairThreads) {
            const int n = e / nw, j = e - n * nw;
            const int h = j < nk ? co[nh + j] : (j == nk ? hc : j - nk);
            s_wave[e] = base + n < rep.N ? turn_wave(s_turn[n][j < nk], h, table) : make_double2(0.0, 0.0);
        }
        __syncthreads();
        for (int e = tid; e < kPairDisks * nk; e += kPairThreads) {  // B(k) = U(hc) V(k)
            const int n = e / nk, k = e - n * nk;
            const double2 u = s_wave[n * nw + nk], v = s_wave[n * nw + k];
            s_wave[n * nw + k] = make_double2(__fma_rn(u.x, v.x, -__dmul_rn(u.y, v.y)), __fma_rn(u.x, v.y, __dmul_rn(u.y, v.x)));
        }
        __syncthreads();
        for (int n = group; n < kPairDisks; n += groups) {
            const double2* w = s_wave + n * nw;
#pragma unroll
            for (int q = 0; q < kPairQ; ++q) {
                if (q == 1 && !second) break;
                const double2 b = w[uk[q]];
                if (uj[q] == 0) {
                    cr[q] = __dadd_rn(cr[q], b.x);
                    ci[q] = __dadd_rn(ci[q], b.y);
                } else {
                    const double2 e = w[nk + uj[q]];
                    cr[q] = __fma_rn(b.x, e.x, cr[q]);
                    ci[q] = __fma_rn(b.y, e.x, ci[q]);
                    sr[q] = __fma_rn(b.x, e.y, sr[q]);
                    si[q] = __fma_rn(b.y, e.y, si[q]);
                }
            }
        }
    }
    // the groups' sums in order
    __syncthreads();
    double2* s_sum = s_wave;  // 2 width entries: at most 256 of at least 32 x 3 + 128
    for (int g = 1; g < groups; ++g) {
        if (group == g && mine[0]) {
            s_sum[2 * lane] = make_double2(cr[0], ci[0]);
            s_sum[2 * lane + 1] = make_double2(sr[0], si[0]);
        }
        __syncthreads();
        if (group == 0 && mine[0]) {
            cr[0] = __dadd_rn(cr[0], s_sum[2 * lane].x);
            ci[0] = __dadd_rn(ci[0], s_sum[2 * lane].y);
            sr[0] = __dadd_rn(sr[0], s_sum[2 * lane + 1].x);
            si[0] = __dadd_rn(si[0], s_sum[2 * lane + 1].y);
        }
        __syncthreads();
    }
    double2* out = part + (size_t(r) * gridDim.x + blockIdx.x) * size_t(nh) * size_t(nk);
#pragma unroll
    for (int q = 0; q < kPairQ; ++q) {
        if (group != 0 || !mine[q]) continue;
        if (J + uj[q] < nh) out[(J + uj[q]) * nk + uk[q]] = make_double2(__dsub_rn(cr[q], si[q]), __dadd_rn(ci[q], sr[q]));
        if (uj[q] > 0) out[(J - uj[q]) * nk + uk[q]] = make_double2(__dadd_rn(cr[q], si[q]), __dsub_rn(ci[q], sr[q]));
    }
}

// S_r(q) = |A_r(q)|^2 / N_r (Eq. 10) from the partial sums: blockIdx.y =
// replica, 32 wave vectors per block, eight threads to each, whose sums are
// added in order (one thread per wave vector over all partial sums ran a
// serial chain: 134 us for 256 partial sums of 441 wave vectors, 6 here).
__global__ void __launch_bounds__(256)
k_sq_sum(const Rep* __restrict__ reps, int nq, int nbx, bool by_disks, const double2* __restrict__ part, int row_len, int nk,
         const ushort2* __restrict__ pair, double* __restrict__ S) {
    pdl_begin(part, pair);
    __shared__ double2 s_v[8][32];
    const int r = blockIdx.y, lane = int(threadIdx.x & 31u), row = int(threadIdx.x >> 5);
    const int q = blockIdx.x * 32 + lane;
    const int nb = by_disks ? int((reps[r].N + 255) / 256) : nbx;  // blocks that hold disks of this replica
    double a = 0.0, b = 0.0;
    if (q < nq) {
        // a row of partial sums holds the wave vectors themselves, or with
        // pair the grid of their components
        size_t at = size_t(q);
        if (pair) {
            const ushort2 c = pair[size_t(r) * nq + q];
            at = size_t(c.x) * nk + c.y;
        }
        for (int x = row; x < nb; x += 8) {
            const double2 p = part[(size_t(r) * nbx + x) * row_len + at];
            a = __dadd_rn(a, p.x);
            b = __dadd_rn(b, p.y);
        }
    }
    s_v[row][lane] = make_double2(a, b);
    __syncthreads();
    if (row == 0 && q < nq) {
        for (int w = 1; w < 8; ++w) {
            a = __dadd_rn(a, s_v[w][lane].x);
            b = __dadd_rn(b, s_v[w][lane].y);
        }
        S[size_t(r) * nq + q] = __ddiv_rn(__dadd_rn(__dmul_rn(a, a), __dmul_rn(b, b)), double(reps[r].N));
    }
}

// best[r] = first q of largest S_r(q).  One block per replica.
__global__ void __launch_bounds__(256)
k_sq_best(int nq, const double* __restrict__ S, int* __restrict__ best) {
    pdl_begin(S);
    const int r = blockIdx.x;
    __shared__ double s_v[256];
    __shared__ int s_i[256];
    double bv = -1.0;
    int bi = 0;
    for (int q = threadIdx.x; q < nq; q += blockDim.x) {
        const double v = S[size_t(r) * nq + q];
        if (v > bv) {
            bv = v;
            bi = q;
        }
    }
    s_v[threadIdx.x] = bv;
    s_i[threadIdx.x] = bi;
    __syncthreads();
    for (int st = blockDim.x / 2; st > 0; st >>= 1) {
        if (int(threadIdx.x) < st) {
            const double ov = s_v[threadIdx.x + st];
            const int oi = s_i[threadIdx.x + st];
            if (ov > s_v[threadIdx.x] || (ov == s_v[threadIdx.x] && oi < s_i[threadIdx.x])) {
                s_v[threadIdx.x] = ov;
                s_i[threadIdx.x] = oi;
            }
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) best[r] = s_i[0];
}

// Candidate window for q_0 per replica: the (2 hw + 1)^2 box-grid points
// around the first-shell reciprocal vector of a triangular lattice of the
// same density (|q| = 4 pi / (a sqrt 3), area per disk sqrt(3) a^2 / 2) at
// the angle arg(Psi_6) / 6 + 30 degrees.  psi[2r], psi[2r + 1] = Psi_6.
// One block per replica; comp and pair as k_sq_pairs takes them (nullable).
__global__ void __launch_bounds__(128)
k_q0_window(const Rep* __restrict__ reps, int hw, const double* __restrict__ psi, int2* __restrict__ hk,
            int* __restrict__ comp, ushort2* __restrict__ pair) {
    pdl_begin(psi);
    const int r = blockIdx.x;
    const Rep& rep = reps[r];
    const double L = rep.Lm;
    const double eta = __ddiv_rn(__dmul_rn(double(rep.N), CUDART_PI), __dmul_rn(L, L));
    const double rho = __ddiv_rn(eta, CUDART_PI);
    const double a = sqrt(__ddiv_rn(2.0, __dmul_rn(sqrt(3.0), rho)));
    const double qmag = __ddiv_rn(__dmul_rn(4.0, CUDART_PI), __dmul_rn(a, sqrt(3.0)));
    const double th = __dadd_rn(__ddiv_rn(atan2(psi[2 * r + 1], psi[2 * r]), 6.0), __ddiv_rn(CUDART_PI, 6.0));
    const double scale = __ddiv_rn(L, __dmul_rn(2.0, CUDART_PI));
    const int hc = int(rint(__dmul_rn(__dmul_rn(qmag, cos(th)), scale)));
    const int kc = int(rint(__dmul_rn(__dmul_rn(qmag, sin(th)), scale)));
    const int w = 2 * hw + 1;
    for (int q = threadIdx.x; q < w * w; q += blockDim.x) {
        const int dh = q / w, dk = q - dh * w;
        hk[size_t(r) * w * w + q] = make_int2(hc - hw + dh, kc - hw + dk);
        if (pair) pair[size_t(r) * w * w + q] = make_ushort2((unsigned short)dh, (unsigned short)dk);
    }
    if (comp)
        for (int j = threadIdx.x; j < 2 * w; j += blockDim.x) comp[size_t(r) * 2 * w + j] = j < w ? hc - hw + j : kc - hw + j - w;
}

// chi_j = exp(i q_0 . x_j) (Eq. 11), by global disk id.
__global__ void __launch_bounds__(256)
k_chi(const Rep* __restrict__ reps, int R, int64_t Ntot, bool fixed, const int2* __restrict__ hk0,
      const double* __restrict__ xy, double2* __restrict__ chi) {
    pdl_begin(hk0, xy);
    const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= Ntot) return;
    const int r = rep_of_id(reps, R, i);
    chi[i] = plane_wave(reps[r], fixed, hk0[r].x, hk0[r].y, __ddiv_rn(xy[2 * i], reps[r].sigma),
                        __ddiv_rn(xy[2 * i + 1], reps[r].sigma));
}

// Positional correlation (Eq. 12): for each ordered pair n != m found through
// the cell grid within reach, with d = x_m - x_n - L rint((x_m - x_n) / L)
// from the global positions and d^2 = dx dx + dy dy, add chi_n conj(chi_m)
// to every window k (r_k = (k + 1) dr) with max(r_k - 1, 0)^2 <= d^2 <=
// (r_k + 1)^2.  acc[r][k] = (sum Re, sum Im, pairs), accumulated per block in
// shared memory (nr <= kMaxCorrWindows).
constexpr int kMaxCorrWindows = 1024;

template <int CAP>
__global__ void __launch_bounds__(256)
k_poscorr(const Rep* __restrict__ reps, int R, const uint8_t* __restrict__ cnt, const int32_t* __restrict__ pid,
          const double* __restrict__ xy, const double2* __restrict__ chi, int nr, double dr, int reach,
          double* __restrict__ acc) {
    extern __shared__ double s_acc[];  // [nr][3]
    pdl_begin(cnt, pid, xy, chi);
    for (int k = threadIdx.x; k < 3 * nr; k += blockDim.x) s_acc[k] = 0.0;
    __syncthreads();
    const int r = find_rep<kGridCell>(reps, R, blockIdx.x);
    const Rep& rep = reps[r];
    const int m = rep.m;
    const int64_t a = int64_t(blockIdx.x - rep.blk_cell) * blockDim.x + threadIdx.x;
    if (a < int64_t(m) * m) {
        int cx, cy;
        cell_coords(rep, a, cx, cy);
        const uint32_t cell = rep.coff + uint32_t(a);
        const int n = min(int(cnt[cell]), CAP);
        const double L = rep.Lm;
        for (int s = 0; s < n; ++s) {
            const int64_t in = rep.id_off + pid[size_t(s) * rep.stride32 + cell];
            const double xn = __ddiv_rn(xy[2 * in], rep.sigma), yn = __ddiv_rn(xy[2 * in + 1], rep.sigma);
            const double2 cn = chi[in];
            for (int dcy = -reach; dcy <= reach; ++dcy) {
                for (int dcx = -reach; dcx <= reach; ++dcx) {
                    const uint32_t nc = rep.coff + row_part(rep, wrap_cell(cy + dcy, m)) + col_part(rep, wrap_cell(cx + dcx, m));
                    const int nn = min(int(cnt[nc]), CAP);
                    for (int q = 0; q < nn; ++q) {
                        const int64_t im = rep.id_off + pid[size_t(q) * rep.stride32 + nc];
                        if (im == in) continue;
                        double dx = __dsub_rn(__ddiv_rn(xy[2 * im], rep.sigma), xn);
                        double dy = __dsub_rn(__ddiv_rn(xy[2 * im + 1], rep.sigma), yn);
                        dx = __dsub_rn(dx, __dmul_rn(L, rint(__ddiv_rn(dx, L))));
                        dy = __dsub_rn(dy, __dmul_rn(L, rint(__ddiv_rn(dy, L))));
                        const double d2 = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
                        const double d = sqrt(d2);
                        const int klo = max(0, int(floor(__ddiv_rn(__dsub_rn(d, 1.0), dr))) - 2);
                        const int khi = min(nr - 1, int(floor(__ddiv_rn(__dadd_rn(d, 1.0), dr))) + 1);
                        if (klo > khi) continue;
                        const double2 cm = chi[im];
                        // chi_n conj(chi_m)
                        const double pr = __dadd_rn(__dmul_rn(cn.x, cm.x), __dmul_rn(cn.y, cm.y));
                        const double pi_ = __dsub_rn(__dmul_rn(cn.y, cm.x), __dmul_rn(cn.x, cm.y));
                        for (int k = klo; k <= khi; ++k) {
                            const double rk = __dmul_rn(double(k + 1), dr);
                            const double lo = rk > 1.0 ? __dsub_rn(rk, 1.0) : 0.0;
                            const double hi = __dadd_rn(rk, 1.0);
                            if (d2 >= __dmul_rn(lo, lo) && d2 <= __dmul_rn(hi, hi)) {
                                atomicAdd(&s_acc[3 * k], pr);
                                atomicAdd(&s_acc[3 * k + 1], pi_);
                                atomicAdd(&s_acc[3 * k + 2], 1.0);
                            }
                        }
                    }
                }
            }
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < 3 * nr; k += blockDim.x)
        if (s_acc[k] != 0.0) atomicAdd(&acc[size_t(r) * 3 * nr + k], s_acc[k]);
}

// ---------------------------------------------------------------------------
// The same correlation from unordered pairs, one disk per thread.  A pair is in
// the windows k with b <= k < a, where a counts the windows whose lower bound
// is at most d^2 and b those whose upper bound is below it, so one addition to
// the elementary interval a + b stands for all its windows; the imaginary
// parts of a pair's two orders cancel exactly.  Every thread keeps its own sums
// per interval in shared memory (interval-major: no two lanes share a bank), so
// nothing is atomic until a block's sums are added up.  a and b come from a
// float estimate of the distance in the cell frame; a pair whose estimate lies
// within its error bound of a window's edge takes the FP64 comparisons of
// k_poscorr on the global positions.  Three FP64 operations per pair remain.
// N = 16,384, 40 windows of 0.5 out to 20 sigma: 13.3 ms with a division, two
// square roots' worth of FP64 and a dozen shared FP64 atomics per ordered pair,
// 0.18 here.
// ---------------------------------------------------------------------------
constexpr size_t kCorrSmem = 112 * 1024;  // two blocks per SM at least
constexpr size_t kCorrBytes = 12;         // a thread's sum and count of one interval

// Threads per block whose interval sums fit, 0 if not even a warp's do.
__host__ __device__ constexpr int corr_threads(int nr) {
    return size_t(2 * nr + 1) * kCorrBytes * 128 <= kCorrSmem ? 128
           : size_t(2 * nr + 1) * kCorrBytes * 64 <= kCorrSmem ? 64
           : size_t(2 * nr + 1) * kCorrBytes * 32 <= kCorrSmem ? 32 : 0;
}

// Per slot and cell: the disk's global position (as k_poscorr reads it), its
// float offset in the cell, and chi.
template <bool FIX, int CAP>
__global__ void __launch_bounds__(256)
k_corr_stage(const Rep* __restrict__ reps, const Frame* __restrict__ cur, const uint8_t* __restrict__ cnt,
             const P2<FIX>* __restrict__ pos, const int2* __restrict__ hk0, double2* __restrict__ gpos,
             double2* __restrict__ chi, float2* __restrict__ off) {
    pdl_begin(cur, cnt, pos, hk0);
    const int r = blockIdx.y;
    const Rep& rep = reps[r];
    const int m = rep.m;
    const uint32_t a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= uint32_t(m) * uint32_t(m)) return;
    int cx, cy;
    cell_coords(rep, a, cx, cy);
    const Frame f = cur[r];
    const uint32_t cell = rep.coff + a;
    const int n = min(int(cnt[cell]), CAP);
    for (int k = 0; k < n; ++k) {
        const size_t at = size_t(k) * rep.stride32 + cell;
        const P2<FIX> q = pos[at];
        double X, Y;
        global_position<FIX>(rep, f, cx, cy, q, X, Y);
        if (rep.sigma != 1.0) {
            X = __ddiv_rn(__dmul_rn(X, rep.sigma), rep.sigma);
            Y = __ddiv_rn(__dmul_rn(Y, rep.sigma), rep.sigma);
        }
        gpos[at] = make_double2(X, Y);
        chi[at] = plane_wave(rep, FIX, hk0[r].x, hk0[r].y, X, Y);
        if constexpr (FIX) off[at] = make_float2(__fmul_rn(__int2float_rn(q.x), 0x1p-24f), __fmul_rn(__int2float_rn(q.y), 0x1p-24f));
        else off[at] = make_float2(__double2float_rn(q.x), __double2float_rn(q.y));
    }
}

// Bounds of window k squared, as k_poscorr compares them.
__device__ __forceinline__ double corr_lo2(int k, double dr) {
    const double rk = __dmul_rn(double(k + 1), dr), lo = rk > 1.0 ? __dsub_rn(rk, 1.0) : 0.0;
    return __dmul_rn(lo, lo);
}
__device__ __forceinline__ double corr_hi2(int k, double dr) {
    const double hi = __dadd_rn(__dmul_rn(double(k + 1), dr), 1.0);
    return __dmul_rn(hi, hi);
}

// a and b of a pair by the FP64 comparisons, from a guess.
static __device__ __noinline__ int2 corr_exact(double2 pn, double2 pm, double L, int nr, double dr, int a, int b) {
    double dx = __dsub_rn(pm.x, pn.x), dy = __dsub_rn(pm.y, pn.y);
    dx = __dsub_rn(dx, __dmul_rn(L, rint(__ddiv_rn(dx, L))));
    dy = __dsub_rn(dy, __dmul_rn(L, rint(__ddiv_rn(dy, L))));
    const double d2 = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
    while (a < nr && corr_lo2(a, dr) <= d2) ++a;
    while (a > 0 && corr_lo2(a - 1, dr) > d2) --a;
    while (b < nr && corr_hi2(b, dr) < d2) ++b;
    while (b > 0 && corr_hi2(b - 1, dr) >= d2) --b;
    return make_int2(a, b);
}

// blockIdx.y: replica, blockIdx.x: cells_per_block of its cells (planar order),
// blockIdx.z: every gridDim.z-th row of the stencil (a small system's blocks
// alone leave the GPU idle).  acc[r][interval] = (sum of Re, pairs).  What
// bounds it is the latency of a neighbour cell's loads, so four cells' are in
// flight at a time.
template <int CAP, int NT>
__global__ void __launch_bounds__(NT)
k_corr_pairs(const Rep* __restrict__ reps, const uint8_t* __restrict__ cnt, const double2* __restrict__ gpos,
             const double2* __restrict__ chi, const float2* __restrict__ off, int nr, double dr, int reach,
             int cells_per_block, double2* __restrict__ acc) {
    extern __shared__ double s_sum[];  // [2 nr + 1][NT], then the counts
    const int bins = 2 * nr + 1;
    uint32_t* s_cnt = reinterpret_cast<uint32_t*>(s_sum + size_t(bins) * NT);
    __shared__ uint16_t s_list[NT * CAP];
    __shared__ int s_n;
    pdl_begin(cnt, gpos, chi, off);
    const int r = blockIdx.y, tid = int(threadIdx.x);
    const Rep& rep = reps[r];
    const int m = rep.m;
    const uint32_t mm = uint32_t(m) * uint32_t(m), a0 = blockIdx.x * uint32_t(cells_per_block);
    if (a0 >= mm) return;
    for (int k = tid; k < bins * NT; k += NT) {
        s_sum[k] = 0.0;
        s_cnt[k] = 0;
    }
    if (tid == 0) s_n = 0;
    __syncthreads();
    // the block's disks, a warp's cells in order
    for (int c0 = 0; c0 < cells_per_block; c0 += NT) {
        const uint32_t a = a0 + uint32_t(c0 + tid);
        const int n = (c0 + tid < cells_per_block && a < mm) ? min(int(cnt[rep.coff + a]), CAP) : 0;
        int v = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, v, o);
            if ((tid & 31) >= o) v += u;
        }
        int base = 0;
        if ((tid & 31) == 31) base = atomicAdd(&s_n, v);
        base = __shfl_sync(0xffffffffu, base, 31) + v - n;
        for (int k = 0; k < n; ++k) s_list[base + k] = uint16_t((c0 + tid) << 4 | k);
    }
    __syncthreads();
    const int disks = s_n;
    const float wf = float(rep.w), inv = __fdiv_rn(1.0f, float(dr)), rmax = float(nr) * float(dr) + 1.0f;
    // error of the float distance: the offsets, the cell offset and the
    // difference each round by at most 2^-24 of the reach, in both components;
    // four times that, and the roundings of the scaled distance
    const float eps = (float(reach + 2) * wf * 0x1p-20f + (rmax + 1.0f) * 0x1p-20f) * inv;
    const double L = rep.Lm;
    for (int d = tid; d < disks; d += NT) {
        const uint32_t a = a0 + (s_list[d] >> 4);
        const int slot = int(s_list[d] & 15u);
        int cx, cy;
        cell_coords(rep, a, cx, cy);
        const size_t me = size_t(slot) * rep.stride32 + rep.coff + a;
        const float2 un = off[me];
        const double2 cn = chi[me];
        auto pair = [&](size_t at, const float2& um, const double2& cm, float bx, float by) {
            const float sx = __fadd_rn(um.x, bx), sy = __fadd_rn(um.y, by);
            const float dist = sqrtf(__fadd_rn(__fmul_rn(sx, sx), __fmul_rn(sy, sy)));
            const float fu = __fmul_rn(__fadd_rn(dist, 1.0f), inv), fv = __fmul_rn(__fsub_rn(dist, 1.0f), inv);
            int wa = int(fminf(floorf(fu), float(nr))), wb = int(fminf(fmaxf(ceilf(fv) - 1.0f, 0.0f), float(nr)));
            // (false also where a window width out of float's range made the estimate infinite)
            const bool sure = eps < 0.25f && fabsf(fu - rintf(fu)) >= eps && fabsf(fv - rintf(fv)) >= eps;
            if (!sure) {
                const int2 e = corr_exact(gpos[me], gpos[at], L, nr, dr, wa, wb);
                wa = e.x;
                wb = e.y;
            }
            if (wa <= wb) return;
            const int s = (wa + wb) * NT + tid;
            s_sum[s] = __dadd_rn(s_sum[s], __fma_rn(cn.x, cm.x, __dmul_rn(cn.y, cm.y)));
            s_cnt[s] += 1u;
        };
        for (int dcy = int(blockIdx.z); dcy <= reach; dcy += int(gridDim.z)) {
            const int y = cy + dcy >= m ? cy + dcy - m : cy + dcy;
            const uint32_t row = rep.coff + row_part(rep, y);
            const float gy = fmaxf(float(dcy - 1), 0.0f) * wf;
            const float by = __fsub_rn(__fmul_rn(float(dcy), wf), un.y);
            // cells of the row with a point in reach
            const float gx2 = (rmax + 0.01f) * (rmax + 0.01f) - gy * gy;
            const int half = gx2 < 0.0f ? -1 : min(reach, int(sqrtf(gx2) / wf) + 2);
            for (int x0 = dcy == 0 ? 0 : -half; x0 <= half; x0 += 4) {
                uint32_t c[4];
                int n[4];
                float2 um[4];
                double2 cm[4];
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    n[h] = 0;
                    if (x0 + h <= half) {
                        c[h] = row + col_part(rep, wrap_cell(cx + x0 + h, m));
                        n[h] = min(int(cnt[c[h]]), CAP);
                        um[h] = off[c[h]];
                        cm[h] = chi[c[h]];
                    }
                }
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const bool same = dcy == 0 && x0 + h == 0;
                    const float bx = __fsub_rn(__fmul_rn(float(x0 + h), wf), un.x);
                    if (n[h] > 0 && !same) pair(c[h], um[h], cm[h], bx, by);
                    for (int q = same ? slot + 1 : 1; q < n[h]; ++q) {
                        const size_t at = size_t(q) * rep.stride32 + c[h];
                        pair(at, off[at], chi[at], bx, by);
                    }
                }
            }
        }
    }
    __syncthreads();
    for (int b = tid >> 5; b < bins; b += NT / 32) {
        double v = 0.0;
        uint32_t c = 0u;
        for (int t = tid & 31; t < NT; t += 32) {
            v = __dadd_rn(v, s_sum[b * NT + t]);
            c += s_cnt[b * NT + t];
        }
        c = __reduce_add_sync(0xffffffffu, c);
        v = lane_sum(v);
        if ((tid & 31) == 0 && c > 0u) {
            double2* o = acc + size_t(r) * bins + b;
            atomicAdd(&o->x, v);
            atomicAdd(&o->y, double(c));
        }
    }
}

// C(r_k): the intervals with b <= k < a.  The pair (a, b) of interval s follows
// from merging the windows' lower and upper bounds (at a tie the lower one
// first: d^2 on both is above the lower and not above the upper).
__global__ void __launch_bounds__(128)
k_corr_windows(int nr, double dr, const double2* __restrict__ acc, double2* __restrict__ out) {
    extern __shared__ double2 s_acc2[];  // [2 nr + 1] sums, then [2 nr] bounds
    pdl_begin(acc);
    const int r = blockIdx.y, bins = 2 * nr + 1, k = int(blockIdx.x * blockDim.x + threadIdx.x);
    double* lo2 = reinterpret_cast<double*>(s_acc2 + bins);
    double* hi2 = lo2 + nr;
    for (int i = threadIdx.x; i < bins; i += blockDim.x) {
        s_acc2[i] = acc[size_t(r) * bins + i];
        if (i < nr) {
            lo2[i] = corr_lo2(i, dr);
            hi2[i] = corr_hi2(i, dr);
        }
    }
    __syncthreads();
    if (k >= nr) return;
    // window k begins with the interval after its lower bound in the merged
    // order and ends with the one before its upper bound comes
    int a = k + 1, b = 0;
    for (int hi = nr; b < hi;) {  // upper bounds before lower bound k: those below it (a tie: after)
        const int mid = (b + hi) >> 1;
        if (hi2[mid] < lo2[k]) b = mid + 1; else hi = mid;
    }
    const int first = a + b;
    a = 0;
    for (int hi = nr; a < hi;) {  // lower bounds before upper bound k: those not above it
        const int mid = (a + hi) >> 1;
        if (lo2[mid] <= hi2[k]) a = mid + 1; else hi = mid;
    }
    const int last = a + k;
    double s = 0.0, c = 0.0;
    for (int i = first; i <= last; ++i) {
        s = __dadd_rn(s, s_acc2[i].x);
        c = __dadd_rn(c, s_acc2[i].y);
    }
    out[size_t(r) * nr + k] = c > 0.0 ? make_double2(__ddiv_rn(s, c), 0.0) : make_double2(CUDART_NAN, CUDART_NAN);
}

__global__ void __launch_bounds__(256)
k_corr_norm(int64_t n, const double* __restrict__ acc, double2* __restrict__ out) {
    pdl_begin(acc);
    const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double c = acc[3 * i + 2];
    out[i] = c > 0.0 ? make_double2(__ddiv_rn(acc[3 * i], c), __ddiv_rn(acc[3 * i + 1], c))
                     : make_double2(CUDART_NAN, CUDART_NAN);
}

// Chunks of times: enough blocks to fill the GPU, no more than the series has
// pieces of kAcfChunk entries, so that the partial sums stay small where the
// lags and replicas are many.
int acf_chunks(int R, int64_t T, int64_t max_lag) {
    const int64_t tiles = int64_t(R) * ((max_lag + kAcfLags) / kAcfLags);
    return int(std::max<int64_t>(1, std::min<int64_t>({64, (1200 + tiles - 1) / tiles, (T + kAcfChunk - 1) / kAcfChunk})));
}

cudaError_t launch_acf(const LaunchCfg& c, const double* series, int64_t T, int64_t max_lag, double2* part, double2* C) {
    const int chunks = acf_chunks(c.R, T, max_lag);
    const int64_t pieces = (T + kAcfChunk - 1) / kAcfChunk, len = (pieces + chunks - 1) / chunks * kAcfChunk;
    const unsigned tiles = unsigned((max_lag + kAcfLags) / kAcfLags);
    const cudaError_t e = launch_k(k_acf_sums, dim3(tiles, unsigned(c.R), unsigned(chunks)), dim3(kAcfLags), 0, c.stream,
                                   series, c.R, T, max_lag, len, part);
    if (e != cudaSuccess) return e;
    return launch_k(k_acf_norm, dim3(unsigned((max_lag + 128) / 128), unsigned(c.R)), dim3(128), 0, c.stream, c.R, T,
                    max_lag, chunks, (const double2*)part, C);
}

cudaError_t launch_acf_tau(const LaunchCfg& c, int64_t max_lag, int64_t lag_lo, int64_t lag_hi, const double2* C,
                           double* tau) {
    return launch_k(k_acf_tau, dim3(unsigned(c.R)), dim3(32), 0, c.stream, max_lag, lag_lo, lag_hi, C, tau);
}

cudaError_t launch_field(const LaunchCfg& c, int64_t Ntot, int bins, const double* xy, const double2* psi,
                         double* acc, double2* out) {
    const int64_t cells = int64_t(c.R) * bins * bins;
    cudaError_t e = cudaMemsetAsync(acc, 0, size_t(cells) * 3 * sizeof(double), c.stream);
    if (e != cudaSuccess) return e;
    e = launch_k(k_field_accum, dim3(unsigned((Ntot + 255) / 256)), dim3(256), 0, c.stream, c.reps, c.R, Ntot,
                 c.fixed, bins, xy, psi, acc);
    if (e != cudaSuccess) return e;
    return launch_k(k_field_norm, dim3(unsigned((cells + 255) / 256)), dim3(256), 0, c.stream, cells,
                    (const double*)acc, out);
}

int sq_disk_blocks(const std::vector<int64_t>& N) {
    int64_t b = 1;
    for (int64_t n : N) b = std::max<int64_t>(b, (n + 255) / 256);
    return int(b);
}

bool sq_pairs_fit(int nh, int nk, int nq) {
    // fewer FP64 operations than a plane wave per wave vector and disk
    return nh + nk <= kPairMax && 15 * (nh + nk) + 4 * nq < 60 * nq;
}

bool sq_grid_fit(int nh, int nk, int nq) {
    const int64_t units = int64_t(nh / 2 + 1) * nk;
    return units <= kPairThreads * kPairQ && units < nq;
}

int sq_pair_blocks(int R, int nq, const std::vector<int64_t>& N) {
    // two blocks per SM (152) over all replicas and tiles of wave vectors
    const int64_t tiles = int64_t(R) * ((nq + kPairThreads * kPairQ - 1) / (kPairThreads * kPairQ));
    int64_t most = 1;
    for (int64_t n : N) most = std::max<int64_t>(most, (n + kPairDisks - 1) / kPairDisks);
    return int(std::max<int64_t>(1, std::min<int64_t>(most, (304 + tiles - 1) / tiles)));
}

cudaError_t launch_sq(const LaunchCfg& c, int nq, const int2* hk, const double* xy, int nbx, double2* part, double* S,
                      int* best) {
    const dim3 grid(unsigned(nbx), unsigned((nq + kSqChunk - 1) / kSqChunk), unsigned(c.R));
    cudaError_t e = launch_k(k_sq_amp, grid, dim3(256), 0, c.stream, c.reps, c.fixed, nq, hk, xy, nbx, part);
    if (e == cudaSuccess)
        e = launch_k(k_sq_sum, dim3(unsigned((nq + 31) / 32), unsigned(c.R)), dim3(256), 0, c.stream, c.reps, nq, nbx, true,
                     (const double2*)part, nq, 0, (const ushort2*)nullptr, S);
    if (e == cudaSuccess && best) e = launch_k(k_sq_best, dim3(unsigned(c.R)), dim3(256), 0, c.stream, nq, (const double*)S, best);
    return e;
}

cudaError_t launch_sq_pairs(const LaunchCfg& c, int nq, int nh, int nk, bool grid, const int* comp, const ushort2* pair,
                            const double* xy, int nbx, double2* part, double* S, int* best) {
    static OncePerDevice once;
    cudaError_t e = allow_smem(once, (kPairDisks * (kPairMax + 1) + kTurnTable) * sizeof(double2), k_sq_pairs, k_sq_grid);
    if (e != cudaSuccess) return e;
    if (grid)
        e = launch_k(k_sq_grid, dim3(unsigned(nbx), 1, unsigned(c.R)), dim3(kPairThreads),
                     size_t(kPairDisks * (nk + 1 + nh / 2) + kTurnTable) * sizeof(double2), c.stream, c.reps, c.fixed, nh, nk,
                     comp, xy, part);
    else
        e = launch_k(k_sq_pairs, dim3(unsigned(nbx), unsigned((nq + kPairThreads * kPairQ - 1) / (kPairThreads * kPairQ)), unsigned(c.R)),
                     dim3(kPairThreads), size_t(kPairDisks * (nh + nk) + kTurnTable) * sizeof(double2), c.stream, c.reps,
                     c.fixed, nq, nh, nk, comp, pair, xy, part);
    if (e == cudaSuccess)
        e = launch_k(k_sq_sum, dim3(unsigned((nq + 31) / 32), unsigned(c.R)), dim3(256), 0, c.stream, c.reps, nq, nbx, false,
                     (const double2*)part, grid ? nh * nk : nq, nk, grid ? pair : (const ushort2*)nullptr, S);
    if (e == cudaSuccess && best) e = launch_k(k_sq_best, dim3(unsigned(c.R)), dim3(256), 0, c.stream, nq, (const double*)S, best);
    return e;
}

cudaError_t launch_q0_window(const LaunchCfg& c, int hw, const double* psi, int2* hk, int* comp, ushort2* pair) {
    return launch_k(k_q0_window, dim3(unsigned(c.R)), dim3(128), 0, c.stream, c.reps, hw, psi, hk, comp, pair);
}

cudaError_t launch_chi(const LaunchCfg& c, int64_t Ntot, const int2* hk0, const double* xy, double2* chi) {
    return launch_k(k_chi, dim3(unsigned((Ntot + 255) / 256)), dim3(256), 0, c.stream, c.reps, c.R, Ntot, c.fixed, hk0,
                    xy, chi);
}

template <int CAP>
static cudaError_t poscorr_t(const LaunchCfg& c, CellBufs cells, const double* xy, const double2* chi, int nr,
                             double dr, int reach, double* acc) {
    static OncePerDevice once;
    const cudaError_t e = allow_smem(once, 3 * kMaxCorrWindows * sizeof(double), k_poscorr<CAP>);
    if (e != cudaSuccess) return e;
    return launch_k(k_poscorr<CAP>, dim3(c.blocks_cell), dim3(c.threads), size_t(3 * nr) * sizeof(double), c.stream,
                    c.reps, c.R, (const uint8_t*)cells.cnt, (const int32_t*)cells.pid, xy, chi, nr, dr, reach, acc);
}

bool corr_pairs_fit(int nr) { return corr_threads(nr) > 0; }
size_t corr_pairs_acc(int R, int nr) { return size_t(R) * size_t(2 * nr + 1) * 2; }

template <bool FIX, int CAP>
static cudaError_t corr_stage_t(const LaunchCfg& c, unsigned cells, const Frame* cur, CellBufs b, const int2* hk0, double2* gpos,
                                double2* chi, float2* off) {
    return launch_k(k_corr_stage<FIX, CAP>, dim3((cells + 255) / 256, unsigned(c.R)), dim3(256), 0, c.stream, c.reps, cur,
                    (const uint8_t*)b.cnt, (const P2<FIX>*)b.pos, hk0, gpos, chi, off);
}

template <int CAP, int NT>
static cudaError_t corr_pairs_t(const LaunchCfg& c, unsigned cells, CellBufs b, const double2* gpos, const double2* chi,
                                const float2* off, int nr, double dr, int reach, double2* acc) {
    static OncePerDevice once;
    const cudaError_t e = allow_smem(once, kCorrSmem, k_corr_pairs<CAP, NT>);
    if (e != cudaSuccess) return e;
    // a little under one cell per thread: at liquid densities a block's disks
    // are then a single round of its threads
    const int cells_per_block = NT * 7 / 8;
    const unsigned blocks = (cells + cells_per_block - 1) / cells_per_block;
    // rows of the stencil split over blocks while there are fewer than ~12 per SM
    const unsigned split = unsigned(std::max<int64_t>(1, std::min<int64_t>({reach + 1, 8, 1824 / (int64_t(blocks) * c.R)})));
    return launch_k(k_corr_pairs<CAP, NT>, dim3(blocks, unsigned(c.R), split), dim3(NT),
                    size_t(2 * nr + 1) * kCorrBytes * NT, c.stream, c.reps, (const uint8_t*)b.cnt, gpos, chi, off, nr, dr, reach,
                    cells_per_block, acc);
}

template <int CAP>
static cudaError_t corr_pairs_nt(const LaunchCfg& c, unsigned cells, CellBufs b, const double2* gpos, const double2* chi,
                                 const float2* off, int nr, double dr, int reach, double2* acc) {
    switch (corr_threads(nr)) {
        case 128: return corr_pairs_t<CAP, 128>(c, cells, b, gpos, chi, off, nr, dr, reach, acc);
        case 64: return corr_pairs_t<CAP, 64>(c, cells, b, gpos, chi, off, nr, dr, reach, acc);
        case 32: return corr_pairs_t<CAP, 32>(c, cells, b, gpos, chi, off, nr, dr, reach, acc);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_corr_pairs(const LaunchCfg& c, int64_t most_cells, const Frame* cur, CellBufs cells, const int2* hk0,
                              double2* gpos, double2* chi, float2* off, int nr, double dr, int reach, double* acc,
                              double2* out) {
    const unsigned n = unsigned(most_cells);
    double2* sums = reinterpret_cast<double2*>(acc);
    cudaError_t e = cudaMemsetAsync(acc, 0, corr_pairs_acc(c.R, nr) * sizeof(double), c.stream);
    if (e == cudaSuccess)
        e = c.fixed ? (c.cap == 4 ? corr_stage_t<true, 4>(c, n, cur, cells, hk0, gpos, chi, off)
                                  : corr_stage_t<true, 9>(c, n, cur, cells, hk0, gpos, chi, off))
                    : (c.cap == 4 ? corr_stage_t<false, 4>(c, n, cur, cells, hk0, gpos, chi, off)
                                  : corr_stage_t<false, 9>(c, n, cur, cells, hk0, gpos, chi, off));
    if (e == cudaSuccess)
        e = c.cap == 4 ? corr_pairs_nt<4>(c, n, cells, gpos, chi, off, nr, dr, reach, sums)
                       : corr_pairs_nt<9>(c, n, cells, gpos, chi, off, nr, dr, reach, sums);
    if (e != cudaSuccess) return e;
    return launch_k(k_corr_windows, dim3(unsigned((nr + 127) / 128), unsigned(c.R)), dim3(128),
                    size_t(2 * nr + 1) * sizeof(double2) + size_t(2 * nr) * sizeof(double), c.stream, nr, dr,
                    (const double2*)sums, out);
}

cudaError_t launch_poscorr(const LaunchCfg& c, CellBufs cells, const double* xy, const double2* chi, int nr, double dr,
                           int reach, double* acc, double2* out) {
    cudaError_t e = cudaMemsetAsync(acc, 0, size_t(c.R) * 3 * nr * sizeof(double), c.stream);
    if (e != cudaSuccess) return e;
    e = c.cap == 4 ? poscorr_t<4>(c, cells, xy, chi, nr, dr, reach, acc) : poscorr_t<9>(c, cells, xy, chi, nr, dr, reach, acc);
    if (e != cudaSuccess) return e;
    const int64_t n = int64_t(c.R) * nr;
    return launch_k(k_corr_norm, dim3(unsigned((n + 255) / 256)), dim3(256), 0, c.stream, n, (const double*)acc, out);
}

}  // namespace hd
