// hd_measure.cu -- measurements on the MPMC cell frame (Engel et al.,
// arXiv:1211.1645): the contact-shell pair histogram and the contact-value
// pressure (Sec. II.C.1, Eqs. 2 and 4), and the local / global
// bond-orientational order psi_6 (Sec. III, Eq. 8).
//
// Pair vectors are formed in the cell frame: for disks i and j whose cells
// differ by (dcx, dcy), r = (u_j + dcx * w) - u_i, which is exact in the
// fixed-point form and has one fixed rounding order in FP64.
#include <type_traits>

#include "hd_kernels.h"

namespace hd {

template <bool FIX>
using P2 = std::conditional_t<FIX, int2, double2>;

constexpr int kMaxFitBins = 512;

// ---------------------------------------------------------------------------
// Contact-shell histogram: unordered pairs with 2 <= r < 2 + K dr, binned by
// comparing r^2 with squared bin edges; each pair is counted once, from its
// lower id (k_hist_global; the FP64 form of k_hist_tile) or, in the fixed
// form of k_hist_tile, from the upper half of the stencil (the same exact
// squared distance from either side, so the same counts).
// One thread per cell scans the (2R+1)^2 stencil; counts gather in a shared
// histogram and are flushed with one atomic per non-empty bin and block.
// k_hist_global reads the stencil from global memory (any reach R);
// k_hist_tile (reach up to kHistMaxHalo) first stages the block's
// tile of cells and a halo of R cells in shared memory, like k_psi6.
// ---------------------------------------------------------------------------
template <bool FIX, int CAP>
__global__ void __launch_bounds__(256)
k_hist_global(const Rep* __restrict__ reps, int R, int K, const double* __restrict__ edges,
       const long long* __restrict__ edgesF, const uint8_t* __restrict__ cnt, const P2<FIX>* __restrict__ pos,
       const int32_t* __restrict__ pid, unsigned long long* __restrict__ hist) {
    extern __shared__ unsigned int s_bins[];
    pdl_begin(cnt, pos, pid);
    for (int b = threadIdx.x; b < K; b += blockDim.x) s_bins[b] = 0u;
    __syncthreads();
    const int r = find_rep<kGridCell>(reps, R, blockIdx.x);
    const Rep& rep = reps[r];
    const int m = rep.m;
    const int64_t a = int64_t(blockIdx.x - rep.blk_cell) * blockDim.x + threadIdx.x;
    if (a < int64_t(m) * m) {
        int cx, cy;
        cell_coords(rep, a, cx, cy);
        const int64_t cell = rep.cell_off + a;
        const int n = min(int(cnt[cell]), CAP);
        const int RR = rep.hist_R;
        const double e0 = edges[0], eK = edges[K];
        const long long f0 = edgesF[0], fK = edgesF[K];
        for (int k = 0; k < n; ++k) {
            const P2<FIX> me = pos[k * rep.stride + cell];
            const int32_t idme = pid[k * rep.stride + cell];
            for (int dcy = -RR; dcy <= RR; ++dcy) {
                for (int dcx = -RR; dcx <= RR; ++dcx) {
                    const int64_t nc = cell_index(rep, wrap_cell(cx + dcx, m), wrap_cell(cy + dcy, m));
                    const int nn = min(int(cnt[nc]), CAP);
                    for (int q = 0; q < nn; ++q) {
                        const int32_t idq = pid[q * rep.stride + nc];
                        if (idq <= idme) continue;
                        const P2<FIX> o = pos[q * rep.stride + nc];
                        int bin;
                        if constexpr (FIX) {
                            const long long rx = (static_cast<long long>(o.x) + static_cast<long long>(dcx) * rep.W) - me.x;
                            const long long ry = (static_cast<long long>(o.y) + static_cast<long long>(dcy) * rep.W) - me.y;
                            const long long r2 = rx * rx + ry * ry;
                            if (r2 < f0 || r2 >= fK) continue;
                            int lo = 0, hi = K - 1;  // largest k with edgesF[k] <= r2
                            while (lo < hi) {
                                const int mid = (lo + hi + 1) >> 1;
                                if (__ldg(&edgesF[mid]) <= r2) lo = mid; else hi = mid - 1;
                            }
                            bin = lo;
                        } else {
                            const double rx = __dsub_rn(__dadd_rn(o.x, __dmul_rn(double(dcx), rep.w)), me.x);
                            const double ry = __dsub_rn(__dadd_rn(o.y, __dmul_rn(double(dcy), rep.w)), me.y);
                            const double r2 = __dadd_rn(__dmul_rn(rx, rx), __dmul_rn(ry, ry));
                            if (r2 < e0 || r2 >= eK) continue;
                            int lo = 0, hi = K - 1;
                            while (lo < hi) {
                                const int mid = (lo + hi + 1) >> 1;
                                if (__ldg(&edges[mid]) <= r2) lo = mid; else hi = mid - 1;
                            }
                            bin = lo;
                        }
                        atomicAdd(&s_bins[bin], 1u);
                    }
                }
            }
        }
    }
    __syncthreads();
    for (int b = threadIdx.x; b < K; b += blockDim.x)
        if (s_bins[b]) atomicAdd(&hist[size_t(r) * K + b], (unsigned long long)s_bins[b]);
}


constexpr int kHistMaxHalo = 4;

// The disks of a block's 32 x rows tile of cells as one list, so that every
// lane works on one disk (a lane per cell would make a warp repeat its scan
// as many times as its most crowded cell holds disks).  Entry: staged cell
// index << 4 | slot, in tile-cell order.  s_list holds blockDim * CAP
// entries, s_warp one int per warp.  Returns the number of disks; every
// thread of the block must call it, after the staging barrier.
__device__ __forceinline__ int tile_disk_list(const uint8_t* s_n, int SX, int halo, int X0, int Y0, int m,
                                              uint16_t* s_list, int* s_warp) {
    const int lx = int(threadIdx.x & 31u), ly = int(threadIdx.x >> 5);
    const int own = (ly + halo) * SX + lx + halo;
    const int n = (X0 + lx < m && Y0 + ly < m) ? int(s_n[own]) : 0;
    int v = n;  // inclusive warp scan of the occupancies
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, v, o);
        if (lx >= o) v += u;
    }
    if (lx == 31) s_warp[ly] = v;
    __syncthreads();
    int base = 0, total = 0;
    for (int w = 0; w < int(blockDim.x >> 5); ++w) {
        const int t = s_warp[w];
        base += w < ly ? t : 0;
        total += t;
    }
    const int off = base + v - n;
    for (int q = 0; q < n; ++q) s_list[off + q] = uint16_t((own << 4) | q);
    __syncthreads();
    return total;
}

// A tile of 32 x 8 cells, one thread per cell; 32 x 4 in the FP64 form where cells
// hold up to nine disks: about two each, so that an SM's FP64 work is that of its
// few blocks (psi_6, one call at cells of 2.9 sigma: N = 16,384 165 us with eight
// rows, 149 with four; N = 2^20 1186 and 1279; the fixed form 99 and 99, 332 and 396).
template <bool FIX, int CAP>
constexpr int kTileThreads = FIX || CAP == 4 ? 256 : 128;

template <bool FIX, int CAP>
__host__ __device__ constexpr size_t hist_stage_bytes(int halo, int K) {
    return size_t(32 + 2 * halo) * size_t(kTileThreads<FIX, CAP> / 32 + 2 * halo) *
               (CAP * (sizeof(P2<FIX>) + (FIX ? 0 : sizeof(float2) + sizeof(int32_t))) + 1) +
           16 + size_t(K + 1) * 8 + size_t(K) * 4;
}

// FP64 bin of a pair (o at cell offset (dcx, dcy) from me) among the K bins
// of squared edges edge[0..K], or -1 outside [edge_0, edge_K); the non-negative
// squared distance is compared through its bit pattern, which orders as the
// value does.
__device__ __forceinline__ int hist_bin_fp64(const double2& o, const double2& me, int dcx, int dcy, double w, const double* edge,
                                             int K) {
    const double rx = __dsub_rn(__dadd_rn(o.x, __dmul_rn(double(dcx), w)), me.x);
    const double ry = __dsub_rn(__dadd_rn(o.y, __dmul_rn(double(dcy), w)), me.y);
    const long long b = __double_as_longlong(__dadd_rn(__dmul_rn(rx, rx), __dmul_rn(ry, ry)));
    if (b < __double_as_longlong(edge[0]) || b >= __double_as_longlong(edge[K])) return -1;
    int lo = 0, hi = K - 1;  // largest k with edge[k] <= r^2
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__double_as_longlong(edge[mid]) <= b) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Each unordered pair is seen once, from the cell whose offset to the other is
// in the upper half of the stencil, or within a cell from the lower slot.
// Fixed form: binned where it is found, by its exact integer distance.
// FP64 form: a pair whose float estimate of r^2 lies within the binned range
// widened by its error bound (set_hist_f32_bounds) is queued, and a warp bins
// its queue 32 pairs at a time by their exact squared distances in the lower
// id's view, whose rounding the oracle follows: about one candidate in forty is
// in the contact shell, so binning each where it was found ran its FP64
// arithmetic once per such pair with one lane in it (57% of the FP64 pipe).
// N = 2^20: FP64 133 -> 78 us; the fixed form 52, with the queue 59.
template <bool FIX, int CAP>
__global__ void __launch_bounds__(kTileThreads<FIX, CAP>)
k_hist_tile(const Rep* __restrict__ reps, int R, int K, const double* __restrict__ edges,
            const long long* __restrict__ edgesF, const uint8_t* __restrict__ cnt, const P2<FIX>* __restrict__ pos,
            const int32_t* __restrict__ pid, unsigned long long* __restrict__ hist, int H) {
    extern __shared__ __align__(16) unsigned char s_raw[];
    pdl_begin(cnt, pos, pid);
    const int r = find_rep<kGridT32>(reps, R, blockIdx.x);
    const Rep& rep = reps[r];
    const int m = rep.m;
    constexpr int rows = kTileThreads<FIX, CAP> / 32;
    int X0, Y0;
    tile32_origin(rep, uint32_t(blockIdx.x - rep.blk_t32), rows, X0, Y0);
    const int SX = 32 + 2 * H, nS = SX * (rows + 2 * H);
    P2<FIX>* s_pos = reinterpret_cast<P2<FIX>*>(s_raw);                      // [CAP][nS]
    // FP64 form: float offsets and ids
    float2* s_img = reinterpret_cast<float2*>(s_pos + size_t(CAP) * nS);                // [CAP][nS]
    int32_t* s_id = reinterpret_cast<int32_t*>(s_img + (FIX ? 0 : size_t(CAP) * nS));   // [CAP][nS]
    uint8_t* s_n = reinterpret_cast<uint8_t*>(s_id + (FIX ? 0 : size_t(CAP) * nS));     // [nS]
    using E = std::conditional_t<FIX, long long, double>;
    E* s_edge = reinterpret_cast<E*>(s_raw + ((size_t(CAP) * nS * (sizeof(P2<FIX>) + (FIX ? 0 : sizeof(float2) + 4)) + nS + 15) & ~size_t(15)));
    unsigned int* s_bins = reinterpret_cast<unsigned int*>(s_edge + (K + 1));
    for (int b = threadIdx.x; b <= K; b += kTileThreads<FIX, CAP>) {
        if constexpr (FIX) s_edge[b] = edgesF[b];
        else s_edge[b] = edges[b];
        if (b < K) s_bins[b] = 0u;
    }
    for (int t = threadIdx.x; t < nS; t += kTileThreads<FIX, CAP>) {
        const int sy = t / SX, sx = t - sy * SX;
        const uint32_t c = uint32_t(rep.coff) + row_part(rep, wrap_cell(Y0 - H + sy, m)) +
                           col_part(rep, wrap_cell(X0 - H + sx, m));
        const int n = min(int(cnt[c]), CAP);
        s_n[t] = uint8_t(n);
        for (int q = 0; q < n; ++q) {
            const P2<FIX> o = pos[size_t(q) * rep.stride32 + c];
            s_pos[q * nS + t] = o;
            if constexpr (!FIX) {
                s_img[q * nS + t] = make_float2(approx_f32(o.x), approx_f32(o.y));
                s_id[q * nS + t] = pid[size_t(q) * rep.stride32 + c];
            }
        }
        if (!FIX && n == 0) s_img[t] = make_float2(__uint_as_float(0x7F800000u), 0.0f);  // slot 0 is tested in any case
    }
    __syncthreads();
    __shared__ uint16_t s_list[kTileThreads<FIX, CAP> * CAP];
    __shared__ int s_warp[8];
    const int D = tile_disk_list(s_n, SX, H, X0, Y0, m, s_list, s_warp);
    const int RR = rep.hist_R;
    if constexpr (FIX) {
        const long long lo_edge = s_edge[0], hi_edge = s_edge[K];
        for (int d = threadIdx.x; d < D; d += kTileThreads<FIX, CAP>) {
            const int own = int(s_list[d] >> 4), k = int(s_list[d] & 15u);
            const int2 me = s_pos[k * nS + own];
            for (int dcy = 0; dcy <= RR; ++dcy) {
                for (int dcx = dcy == 0 ? 0 : -RR; dcx <= RR; ++dcx) {
                    const int sc = own + dcy * SX + dcx;
                    const int nn = s_n[sc];
                    for (int q = (dcy == 0 && dcx == 0) ? k + 1 : 0; q < nn; ++q) {
                        const int2 o = s_pos[q * nS + sc];
                        // |offset| < (RR + 1) W <= 5 W < 2^31
                        const int32_t rx = (o.x + dcx * rep.W) - me.x, ry = (o.y + dcy * rep.W) - me.y;
                        const long long r2 = int64_t(rx) * rx + int64_t(ry) * ry;
                        if (r2 < lo_edge || r2 >= hi_edge) continue;
                        int lo = 0, hi = K - 1;  // largest k with edge[k] <= r2
                        while (lo < hi) {
                            const int mid = (lo + hi + 1) >> 1;
                            if (s_edge[mid] <= r2) lo = mid; else hi = mid - 1;
                        }
                        atomicAdd(&s_bins[lo], 1u);
                    }
                }
            }
        }
    } else {
        __shared__ uint32_t s_queue[kTileThreads<FIX, CAP> / 32][64];  // own entry | other entry << 16
        const int lane = int(threadIdx.x & 31u), warp = int(threadIdx.x >> 5);
        uint32_t* queue = s_queue[warp];
        int queued = 0;  // the same in every lane
        auto bin_queued = [&](int count) {
            if (lane < count) {
                const uint32_t v = queue[lane];
                const int a = int(v & 0xFFFFu), b = int(v >> 16);  // entries slot * nS + cell
                const int ca = a % nS, cb = b % nS;
                const int dcy = cb / SX - ca / SX, dcx = cb % SX - ca % SX;
                const double2 pa = s_pos[a], pb = s_pos[b];
                const int bin = s_id[a] < s_id[b] ? hist_bin_fp64(pb, pa, dcx, dcy, rep.w, s_edge, K)
                                                  : hist_bin_fp64(pa, pb, -dcx, -dcy, rep.w, s_edge, K);
                if (bin >= 0) atomicAdd(&s_bins[bin], 1u);
            }
        };
        for (int base = warp * 32; base < D; base += kTileThreads<FIX, CAP>) {
            const int d = base + lane;
            const bool live = d < D;
            const int own = live ? int(s_list[d] >> 4) : 0, k = live ? int(s_list[d] & 15u) : 0;
            const int mine = k * nS + own;
            const float2 me = s_img[mine];
            for (int dcy = 0; dcy <= RR; ++dcy) {
                const float by = __fmul_rn(float(dcy), rep.wf_sigma);
                for (int dcx = dcy == 0 ? 0 : -RR; dcx <= RR; ++dcx) {
                    const float bx = __fmul_rn(float(dcx), rep.wf_sigma);
                    const bool same = dcx == 0 && dcy == 0;
                    const int sc = live ? own + dcy * SX + dcx : 0;
                    const int nn = s_n[sc];
                    // slot 0 without a look at the occupancy, the others while any lane has one
                    for (int q = 0;; ++q) {
                        const float2 f = s_img[q * nS + sc];
                        const float sx = __fsub_rn(__fadd_rn(f.x, bx), me.x), sy = __fsub_rn(__fadd_rn(f.y, by), me.y);
                        const float d2f = __fadd_rn(__fmul_rn(sx, sx), __fmul_rn(sy, sy));
                        const bool in = live && (q == 0 || q < nn) && (!same || q > k) && d2f >= rep.h_lo && d2f < rep.h_hi;
                        const uint32_t who = __ballot_sync(0xffffffffu, in);
                        if (who) {
                            if (in) queue[queued + __popc(who & ((1u << lane) - 1u))] = uint32_t(mine) | uint32_t(q * nS + sc) << 16;
                            queued += __popc(who);
                            __syncwarp();
                            if (queued >= 32) {
                                bin_queued(32);
                                __syncwarp();
                                const uint32_t v = lane < queued - 32 ? queue[32 + lane] : 0u;
                                __syncwarp();
                                if (lane < queued - 32) queue[lane] = v;
                                queued -= 32;
                            }
                        }
                        if (q + 1 == CAP || !__any_sync(0xffffffffu, q + 1 < nn)) break;
                    }
                }
            }
        }
        __syncwarp();
        bin_queued(queued);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < K; b += kTileThreads<FIX, CAP>)
        if (s_bins[b]) atomicAdd(&hist[size_t(r) * K + b], (unsigned long long)s_bins[b]);
}

// ---------------------------------------------------------------------------
// g(r) normalisation (Eq. 2, p = N^2 / 2), least-squares quartic in
// t = (r - 2 sigma) / (K dr) by Householder QR, value at contact, and the
// contact-value pressure (Eq. 4).  The design matrix A = Q R depends on K
// alone, and the value at contact is linear in g(r): g(2 sigma+) = sum_k c_k
// g(r_k) with c = Q (R^-T e_0).  k_fit_factor works c out once per context;
// k_fit then takes one product sum per measurement, where applying the
// reflectors and solving took a chain of five dot products (18 -> 5 us).
// One warp: the K rows are spread over the lanes and every column norm and dot
// product is a warp sum.
// res[4r + 0..3] = beta P / rho, g(2 sigma+), P* = beta P (2 sigma)^2, eta.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v = __dadd_rn(v, __shfl_xor_sync(0xffffffffu, v, off));
    return v;
}

__global__ void __launch_bounds__(32) k_fit_factor(int K, double* __restrict__ weight) {
    __shared__ double A[kMaxFitBins * 5], c[kMaxFitBins];
    __shared__ double v0s[5], vtvs[5];
    const int lane = threadIdx.x;
    for (int k = lane; k < K; k += 32) {
        const double t = __ddiv_rn(__dadd_rn(double(k), 0.5), double(K));
        double tp = 1.0;
        for (int q = 0; q < 5; ++q) {
            A[k * 5 + q] = tp;
            tp = __dmul_rn(tp, t);
        }
    }
    __syncwarp();
    for (int j = 0; j < 5; ++j) {
        double part = 0.0;
        for (int i = j + lane; i < K; i += 32) part = __dadd_rn(part, __dmul_rn(A[i * 5 + j], A[i * 5 + j]));
        const double nrm2 = warp_sum(part);
        const double nrm = sqrt(nrm2);  // positive: the columns are independent for K >= 5
        const double ajj = A[j * 5 + j];
        const double alpha = ajj > 0.0 ? -nrm : nrm;
        const double v0 = __dsub_rn(ajj, alpha);
        const double vtv = __dadd_rn(__dsub_rn(nrm2, __dmul_rn(ajj, ajj)), __dmul_rn(v0, v0));
        __syncwarp();
        if (lane == 0) A[j * 5 + j] = v0;  // v = (v0, A[j+1.., j])
        __syncwarp();
        for (int q = j + 1; q < 5; ++q) {
            double dp = 0.0;
            for (int i = j + lane; i < K; i += 32) dp = __dadd_rn(dp, __dmul_rn(A[i * 5 + j], A[i * 5 + q]));
            const double sc = __ddiv_rn(__dmul_rn(2.0, warp_sum(dp)), vtv);
            for (int i = j + lane; i < K; i += 32) A[i * 5 + q] = __dsub_rn(A[i * 5 + q], __dmul_rn(sc, A[i * 5 + j]));
            __syncwarp();
        }
        if (lane == 0) {
            A[j * 5 + j] = alpha;  // R diagonal
            v0s[j] = v0;
            vtvs[j] = vtv;
        }
        __syncwarp();
    }
    // y = R^-T e_0, then c = H_0 H_1 .. H_4 (y, 0)
    for (int k = lane; k < K; k += 32) c[k] = 0.0;
    __syncwarp();
    if (lane == 0)
        for (int i = 0; i < 5; ++i) {
            double acc = i == 0 ? 1.0 : 0.0;
            for (int q = 0; q < i; ++q) acc = __dsub_rn(acc, __dmul_rn(A[q * 5 + i], c[q]));
            c[i] = __ddiv_rn(acc, A[i * 5 + i]);
        }
    __syncwarp();
    for (int j = 4; j >= 0; --j) {
        double dp = 0.0;
        for (int i = j + lane; i < K; i += 32) dp = __dadd_rn(dp, __dmul_rn(i == j ? v0s[j] : A[i * 5 + j], c[i]));
        const double sc = __ddiv_rn(__dmul_rn(2.0, warp_sum(dp)), vtvs[j]);
        for (int i = j + lane; i < K; i += 32) c[i] = __dsub_rn(c[i], __dmul_rn(sc, i == j ? v0s[j] : A[i * 5 + j]));
        __syncwarp();
    }
    for (int k = lane; k < K; k += 32) weight[k] = c[k];
}

__global__ void __launch_bounds__(32) k_fit(const Rep* __restrict__ reps, int K, const double* __restrict__ weight,
                                            const unsigned long long* __restrict__ hist, double* __restrict__ res) {
    pdl_begin(hist);
    const int r = blockIdx.x, lane = threadIdx.x;
    const Rep& rep = reps[r];
    const double PI = 3.14159265358979323846;
    const double V = __dmul_rn(rep.Lm, rep.Lm);
    const double p = __dmul_rn(__dmul_rn(double(rep.N), double(rep.N)), 0.5);
    const double dr = rep.dr;
    double part = 0.0;
    for (int k = lane; k < K; k += 32) {
        const double rk = __dadd_rn(2.0, __dmul_rn(__dadd_rn(double(k), 0.5), dr));
        const double shell = __ddiv_rn(__dmul_rn(__dmul_rn(__dmul_rn(2.0, PI), rk), dr), V);
        const double g = __ddiv_rn(__ddiv_rn(double(hist[size_t(r) * K + k]), p), shell);
        part = __dadd_rn(part, __dmul_rn(weight[k], g));
    }
    const double g0 = warp_sum(part);
    if (lane != 0) return;
    const double eta = __ddiv_rn(__dmul_rn(double(rep.N), PI), V);
    const double bp = __dadd_rn(1.0, __dmul_rn(__dmul_rn(2.0, eta), g0));
    res[4 * r + 0] = bp;
    res[4 * r + 1] = g0;
    res[4 * r + 2] = __dmul_rn(__dmul_rn(bp, 4.0), __ddiv_rn(double(rep.N), V));
    res[4 * r + 3] = eta;
}

// ---------------------------------------------------------------------------
// psi_6: six nearest neighbours by (r^2, id) from an expanding ring of cells
// (first the 5 x 5 stencil, then one ring more while the sixth neighbour is
// not strictly closer than the nearest point outside the scanned cells).
// exp(6 i phi) = z^6 / |z|^6, z = rx + i ry, summed in ascending (r^2, id).
// ---------------------------------------------------------------------------
template <bool FIX>
struct Nbr {
    // squared distances: exact integers (fixed form), or the bit patterns of
    // the non-negative FP64 values, which order as the values do (so the
    // list needs no FP64 comparison)
    using Key = long long;
    // pair offsets: 32-bit in the fixed form (the ring search never reaches
    // (RR + 1) W >= 2^31, so |r| < 2^31)
    using Off = std::conditional_t<FIX, int32_t, double>;
    Key key[6];
    int32_t id[6];
    Off rx[6], ry[6];
    int n;

    __device__ __forceinline__ void insert(Key k, int32_t i, Off x, Off y) {
        if (n == 6 && !(k < key[5] || (k == key[5] && i < id[5]))) return;
        bool done = false;
        const int top = n < 6 ? n : 5;
#pragma unroll
        for (int s = 5; s >= 0; --s) {
            if (!done && s <= top) {
                if (s > 0 && (k < key[s - 1] || (k == key[s - 1] && i < id[s - 1]))) {
                    key[s] = key[s - 1];
                    id[s] = id[s - 1];
                    rx[s] = rx[s - 1];
                    ry[s] = ry[s - 1];
                } else {
                    key[s] = k;
                    id[s] = i;
                    rx[s] = x;
                    ry[s] = y;
                    done = true;
                }
            }
        }
        if (n < 6) ++n;
    }
};

template <bool FIX, int CAP>
__device__ __forceinline__ void scan_cell(const Rep& rep, const uint8_t* __restrict__ cnt, const P2<FIX>* __restrict__ pos,
                                          const int32_t* __restrict__ pid, int cx, int cy, int dcx, int dcy,
                                          const P2<FIX>& me, int32_t idme, Nbr<FIX>& nb) {
    const int m = rep.m;
    const int64_t nc = cell_index(rep, wrap_cell(cx + dcx, m), wrap_cell(cy + dcy, m));
    const int nn = min(int(cnt[nc]), CAP);
    for (int q = 0; q < nn; ++q) {
        const int32_t idq = pid[q * rep.stride + nc];
        if (idq == idme) continue;
        const P2<FIX> o = pos[q * rep.stride + nc];
        if constexpr (FIX) {
            const int32_t rx = (o.x + dcx * rep.W) - me.x;
            const int32_t ry = (o.y + dcy * rep.W) - me.y;
            nb.insert(int64_t(rx) * rx + int64_t(ry) * ry, idq, rx, ry);
        } else {
            const double rx = __dsub_rn(__dadd_rn(o.x, __dmul_rn(double(dcx), rep.w)), me.x);
            const double ry = __dsub_rn(__dadd_rn(o.y, __dmul_rn(double(dcy), rep.w)), me.y);
            nb.insert(__double_as_longlong(__dadd_rn(__dmul_rn(rx, rx), __dmul_rn(ry, ry))), idq, rx, ry);
        }
    }
}

// Cover test of the ring search: the sixth neighbour is strictly closer than
// any point outside the (2 RR + 1)^2 cells around the disk's cell.
template <bool FIX>
__device__ __forceinline__ bool ring_covers(const Rep& rep, const Nbr<FIX>& nb, const P2<FIX>& me, int RR) {
    if (nb.n < 6) return false;
    if constexpr (FIX) {
        long long cv = static_cast<long long>(me.x) + static_cast<long long>(RR) * rep.W;
        const long long c2 = static_cast<long long>(RR + 1) * rep.W - me.x;
        const long long c3 = static_cast<long long>(me.y) + static_cast<long long>(RR) * rep.W;
        const long long c4 = static_cast<long long>(RR + 1) * rep.W - me.y;
        cv = c2 < cv ? c2 : cv;
        cv = c3 < cv ? c3 : cv;
        cv = c4 < cv ? c4 : cv;
        return nb.key[5] < cv * cv;
    } else {
        double cv = __dadd_rn(me.x, __dmul_rn(double(RR), rep.w));
        const double c2 = __dsub_rn(__dmul_rn(double(RR + 1), rep.w), me.x);
        const double c3 = __dadd_rn(me.y, __dmul_rn(double(RR), rep.w));
        const double c4 = __dsub_rn(__dmul_rn(double(RR + 1), rep.w), me.y);
        cv = c2 < cv ? c2 : cv;
        cv = c3 < cv ? c3 : cv;
        cv = c4 < cv ? c4 : cv;
        return nb.key[5] < __double_as_longlong(__dmul_rn(cv, cv));
    }
}

// Shared-memory copy of the cells a psi_6 block reads: its 32 x rows tile of
// cells plus a halo of two cells (the 5 x 5 stencil of every tile cell).
constexpr int kPsiHalo = 2;
constexpr int kPsiSX = 32 + 2 * kPsiHalo;

template <bool FIX, int CAP>
__host__ __device__ constexpr size_t psi6_stage_bytes(int rows) {
    return size_t(kPsiSX) * size_t(rows + 2 * kPsiHalo) * (2 * sizeof(float2) + CAP * (sizeof(P2<FIX>) + sizeof(int32_t)) + 1);
}

// What a disk of a tile sees.
template <bool FIX>
struct PsiStage {
    const float2* img;   // [2][nS] float offsets of slots 0 and 1, infinite where unoccupied
    const P2<FIX>* pos;  // [CAP][nS]
    const int32_t* id;   // [CAP][nS]
    const uint8_t* n;    // [nS]
    int nS;
};

// The general search of a disk's six nearest: ordered insertion of every
// candidate by (r^2, id) from the staged rings 0, 1, 2, then rings in global
// memory until the sixth is certified.  Where cells hold up to four disks the
// float search below leaves it about one disk in a thousand, so it is called out
// of line (nearest_general); the disks of wider cells all take it, in line (FP64,
// N = 16,384 at cells of 2.9 sigma, one call with eight rows of cells per block: out of line 183 us, in line 165).  In the FP64 form a candidate whose float estimate of
// r^2 exceeds the sixth key by more than the estimate's error bound is farther
// in FP64 too and is left out before its FP64 arithmetic.
template <bool FIX, int CAP>
__device__ __forceinline__ bool nearest_inserted(const Rep& rep, const PsiStage<FIX>& st, const uint8_t* cnt,
                                                 const P2<FIX>* pos, const int32_t* pid, int own, int cx, int cy,
                                                 const P2<FIX>& me, int32_t idme, int rmax,
                                                 typename Nbr<FIX>::Off (&ox)[6], typename Nbr<FIX>::Off (&oy)[6]) {
    Nbr<FIX> nb;
    nb.n = 0;
    bool ok = false;
    float mfx = 0.0f, mfy = 0.0f;  // FP64 form: float images of the disk's offsets
    if constexpr (!FIX) {
        mfx = approx_f32(me.x);
        mfy = approx_f32(me.y);
    }
    if (rmax >= 2) {
#pragma unroll 1
        for (int ring = 0; ring <= 2; ++ring) {
            for (int dcy = -ring; dcy <= ring; ++dcy) {
                for (int dcx = -ring; dcx <= ring; ++dcx) {
                    if (max(abs(dcx), abs(dcy)) != ring) continue;
                    const int sc = own + dcy * kPsiSX + dcx;
                    const int nn = st.n[sc];
                    for (int q = 0; q < nn; ++q) {
                        const int32_t idq = st.id[q * st.nS + sc];
                        if (idq == idme) continue;
                        const P2<FIX> o = st.pos[q * st.nS + sc];
                        if constexpr (FIX) {
                            const int32_t rx = (o.x + dcx * rep.W) - me.x;
                            const int32_t ry = (o.y + dcy * rep.W) - me.y;
                            nb.insert(int64_t(rx) * rx + int64_t(ry) * ry, idq, rx, ry);
                        } else {
                            if (nb.n == 6) {  // (approx_f32 truncates; the product rounds up past the key itself)
                                const float sx = __fsub_rn(__fadd_rn(approx_f32(o.x), __fmul_rn(float(dcx), rep.wf)), mfx);
                                const float sy = __fsub_rn(__fadd_rn(approx_f32(o.y), __fmul_rn(float(dcy), rep.wf)), mfy);
                                const float d2f = __fadd_rn(__fmul_rn(sx, sx), __fmul_rn(sy, sy));
                                const float k5 = __fmul_ru(approx_f32(__longlong_as_double(nb.key[5])), 1.0f + 0x1p-19f);
                                if (d2f > __fadd_ru(k5, rep.psi_m)) continue;
                            }
                            const double rx = __dsub_rn(__dadd_rn(o.x, __dmul_rn(double(dcx), rep.w)), me.x);
                            const double ry = __dsub_rn(__dadd_rn(o.y, __dmul_rn(double(dcy), rep.w)), me.y);
                            nb.insert(__double_as_longlong(__dadd_rn(__dmul_rn(rx, rx), __dmul_rn(ry, ry))), idq, rx, ry);
                        }
                    }
                }
            }
        }
        ok = ring_covers<FIX>(rep, nb, me, 2);
    }
    for (int RR = 3; RR <= rmax && !ok; ++RR) {
        for (int e = -RR; e <= RR; ++e) {
            scan_cell<FIX, CAP>(rep, cnt, pos, pid, cx, cy, e, -RR, me, idme, nb);
            scan_cell<FIX, CAP>(rep, cnt, pos, pid, cx, cy, e, RR, me, idme, nb);
        }
        for (int e = -RR + 1; e <= RR - 1; ++e) {
            scan_cell<FIX, CAP>(rep, cnt, pos, pid, cx, cy, -RR, e, me, idme, nb);
            scan_cell<FIX, CAP>(rep, cnt, pos, pid, cx, cy, RR, e, me, idme, nb);
        }
        ok = ring_covers<FIX>(rep, nb, me, RR);
    }
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        ox[q] = nb.rx[q];
        oy[q] = nb.ry[q];
    }
    return ok;
}

template <bool FIX, int CAP>
static __device__ __noinline__ bool nearest_general(const Rep& rep, const PsiStage<FIX>& st, const uint8_t* cnt,
                                                    const P2<FIX>* pos, const int32_t* pid, int own, int cx, int cy,
                                                    P2<FIX> me, int32_t idme, int rmax, typename Nbr<FIX>::Off* ox,
                                                    typename Nbr<FIX>::Off* oy) {
    typename Nbr<FIX>::Off x[6], y[6];
    const bool ok = nearest_inserted<FIX, CAP>(rep, st, cnt, pos, pid, own, cx, cy, me, idme, rmax, x, y);
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        ox[q] = x[q];
        oy[q] = y[q];
    }
    return ok;
}

// The six nearest of a disk (slot k of staged cell own) from its 5 x 5 stencil
// by float distances: every candidate's d^2 + 64 has its 23 mantissa bits as a
// fixed-point d^2 (quantum 2^-17) above seven bits of candidate number, and
// the seven smallest of these words are kept by min / max (fourteen
// instructions per candidate, no branch).  For d^2 < 64 the float value errs by
// less than 5.2 quanta: offsets and cell side rounded to 2^-23, two sums below
// 16, the square sum and the addition of 64.  So words 16 quanta apart are in
// the order of the exact distances: a sixth and seventh closer than that, or a
// sixth at 64 or beyond, go to nearest_general (returns 0); closer words among
// the six are put in order by their exact (r^2, id).  Returns 1 when the six
// are certified by the stencil, else 0.
constexpr uint32_t kPsiMargin = 16u << 7;

template <bool FIX, int CAP>
__device__ __forceinline__ bool nearest_float(const Rep& rep, const PsiStage<FIX>& st, int own, int k, const P2<FIX>& me,
                                              typename Nbr<FIX>::Off (&ox)[6], typename Nbr<FIX>::Off (&oy)[6]) {
    const float wf = FIX ? __fmul_rn(__int2float_rn(rep.W), 0x1p-24f) : float(rep.w);
    float2 um;
    if constexpr (FIX) um = make_float2(__fmul_rn(__int2float_rn(me.x), 0x1p-24f), __fmul_rn(__int2float_rn(me.y), 0x1p-24f));
    else um = make_float2(__double2float_rn(me.x), __double2float_rn(me.y));
    uint32_t key[7];
#pragma unroll
    for (int s = 0; s < 7; ++s) key[s] = ~0u;
    auto take = [&](const float2& f, float bx, float by, uint32_t number, bool self) {
        const float sx = __fadd_rn(f.x, bx), sy = __fadd_rn(f.y, by);
        const float d = __fadd_rn(__fmaf_rn(sx, sx, __fmul_rn(sy, sy)), 64.0f);
        uint32_t x = (__float_as_uint(d) << 7) + number;
        if (self) x = ~0u;
#pragma unroll
        for (int s = 0; s < 7; ++s) {
            const uint32_t lo = min(key[s], x);
            x = max(key[s], x);
            key[s] = lo;
        }
    };
#pragma unroll 1
    for (int dcy = -2; dcy <= 2; ++dcy) {
        const float by = __fsub_rn(__fmul_rn(float(dcy), wf), um.y);
        const int row = own + dcy * kPsiSX;
        const uint32_t number = uint32_t(dcy + 2) * 20u;
#pragma unroll
        for (int dcx = -2; dcx <= 2; ++dcx) {
            const float bx = __fsub_rn(__fmul_rn(float(dcx), wf), um.x);
            const bool here = dcx == 0 && dcy == 0;
            take(st.img[row + dcx], bx, by, number + uint32_t(dcx + 2) * 4u, here && k == 0);
            take(st.img[st.nS + row + dcx], bx, by, number + uint32_t(dcx + 2) * 4u + 1u, here && k == 1);
            const int n = st.n[row + dcx];
            for (int q = 2; q < n; ++q) {  // rare
                const P2<FIX> o = st.pos[q * st.nS + row + dcx];
                float2 f;
                if constexpr (FIX) f = make_float2(__fmul_rn(__int2float_rn(o.x), 0x1p-24f), __fmul_rn(__int2float_rn(o.y), 0x1p-24f));
                else f = make_float2(__double2float_rn(o.x), __double2float_rn(o.y));
                take(f, bx, by, number + uint32_t(dcx + 2) * 4u + uint32_t(q), here && k == q);
            }
        }
    }
    if (key[5] >= 0x80000000u || key[6] - key[5] < kPsiMargin) return false;
    Nbr<FIX> nb;
    bool close = false;
#pragma unroll
    for (int s = 0; s < 6; ++s) {
        if (s > 0) close |= key[s] - key[s - 1] < kPsiMargin;
        const uint32_t number = key[s] & 127u, c = number >> 2, dy = (c * 13u) >> 6;  // c / 5 for c < 25
        const int dcx = int(c - dy * 5u) - 2, dcy = int(dy) - 2;
        const int at = int(number & 3u) * st.nS + own + dcy * kPsiSX + dcx;
        const P2<FIX> o = st.pos[at];
        if constexpr (FIX) {
            nb.rx[s] = (o.x + dcx * rep.W) - me.x;
            nb.ry[s] = (o.y + dcy * rep.W) - me.y;
        } else {
            nb.rx[s] = __dsub_rn(__dadd_rn(o.x, __dmul_rn(double(dcx), rep.w)), me.x);
            nb.ry[s] = __dsub_rn(__dadd_rn(o.y, __dmul_rn(double(dcy), rep.w)), me.y);
        }
    }
    auto square = [&](int s) -> long long {
        if constexpr (FIX) return int64_t(nb.rx[s]) * nb.rx[s] + int64_t(nb.ry[s]) * nb.ry[s];
        else return __double_as_longlong(__dadd_rn(__dmul_rn(nb.rx[s], nb.rx[s]), __dmul_rn(nb.ry[s], nb.ry[s])));
    };
    if (close) {  // rare: the exact order of the six
        Nbr<FIX> in;
        in.n = 0;
#pragma unroll
        for (int s = 0; s < 6; ++s) {
            const uint32_t number = key[s] & 127u, c = number >> 2, dy = (c * 13u) >> 6;
            const int at = int(number & 3u) * st.nS + own + (int(dy) - 2) * kPsiSX + int(c - dy * 5u) - 2;
            in.insert(square(s), st.id[at], nb.rx[s], nb.ry[s]);
        }
#pragma unroll
        for (int s = 0; s < 6; ++s) {
            nb.rx[s] = in.rx[s];
            nb.ry[s] = in.ry[s];
        }
    }
    nb.n = 6;
    nb.key[5] = square(5);
#pragma unroll
    for (int s = 0; s < 6; ++s) {
        ox[s] = nb.rx[s];
        oy[s] = nb.ry[s];
    }
    return ring_covers<FIX>(rep, nb, me, 2);
}

// Global sums of psi_j of each replica while k_psi6 runs: the 192-bit sums of
// its blocks added as 32-bit limbs in 64-bit words (Re six, Im six), so that
// blocks add atomically without carries; word 12 is set by a sum marked bad.
// k_psi6_reduce reads them and leaves them zero (one block over a partial sum
// per tile took 27 us at N = 2^20 after the last block; this takes 6).
constexpr int kPsiWords = 16;

// psi_6 of every disk.  A block stages its tile and halo in shared memory in
// one cooperative round of loads; each disk then finds its six nearest there
// (nearest_float, or nearest_general: a stencil that does not certify them, as
// at low density, continues in global memory).
// Instruction-bound in the fixed form (ordered insertion of 25 candidates by
// 64-bit keys took ~4800 instructions per disk, this ~3050): 182 -> 138 us at N
// = 2^20, 58 -> 47 at 262,144.  The FP64 form is bound by the FP64 pipe (84%
// busy, mostly the fourteen correctly rounded divisions per disk): 952 -> 668.
template <bool FIX, int CAP>
__global__ void __launch_bounds__(kTileThreads<FIX, CAP>, (FIX ? 1024 : 512) / kTileThreads<FIX, CAP>)
k_psi6(const Rep* __restrict__ reps, int R, const uint8_t* __restrict__ cnt, const P2<FIX>* __restrict__ pos,
       const int32_t* __restrict__ pid, double2* __restrict__ local, unsigned long long* __restrict__ total,
       int* __restrict__ err) {
    extern __shared__ __align__(16) unsigned char s_raw[];
    pdl_begin(cnt, pos, pid);
    const int r = find_rep<kGridT32>(reps, R, blockIdx.x);
    const Rep& rep = reps[r];
    const int m = rep.m;
    constexpr int rows = kTileThreads<FIX, CAP> / 32;
    int X0, Y0;
    tile32_origin(rep, uint32_t(blockIdx.x - rep.blk_t32), rows, X0, Y0);
    constexpr int nS = kPsiSX * (rows + 2 * kPsiHalo);
    P2<FIX>* s_pos = reinterpret_cast<P2<FIX>*>(s_raw);                    // [CAP][nS]
    float2* s_img = reinterpret_cast<float2*>(s_pos + size_t(CAP) * nS);   // [2][nS]
    int32_t* s_id = reinterpret_cast<int32_t*>(s_img + size_t(2) * nS);    // [CAP][nS]
    uint8_t* s_n = reinterpret_cast<uint8_t*>(s_id + size_t(CAP) * nS);    // [nS]
    for (int t = threadIdx.x; t < nS; t += kTileThreads<FIX, CAP>) {
        const int sy = t / kPsiSX, sx = t - sy * kPsiSX;
        const uint32_t c = uint32_t(rep.coff) + row_part(rep, wrap_cell(Y0 - kPsiHalo + sy, m)) +
                           col_part(rep, wrap_cell(X0 - kPsiHalo + sx, m));
        const int n = min(int(cnt[c]), CAP);
        s_n[t] = uint8_t(n);
        float2 f[2];
        f[0] = f[1] = make_float2(__uint_as_float(0x7F800000u), __uint_as_float(0x7F800000u));
        for (int q = 0; q < n; ++q) {
            const P2<FIX> o = pos[size_t(q) * rep.stride32 + c];
            s_pos[q * nS + t] = o;
            s_id[q * nS + t] = pid[size_t(q) * rep.stride32 + c];
            if (q < 2) {
                if constexpr (FIX) f[q] = make_float2(__fmul_rn(__int2float_rn(o.x), 0x1p-24f), __fmul_rn(__int2float_rn(o.y), 0x1p-24f));
                else f[q] = make_float2(__double2float_rn(o.x), __double2float_rn(o.y));
            }
        }
        s_img[t] = f[0];
        s_img[nS + t] = f[1];
    }
    __syncthreads();

    __shared__ uint16_t s_list[kTileThreads<FIX, CAP> * CAP];
    __shared__ int s_warp[8];
    const int D = tile_disk_list(s_n, kPsiSX, kPsiHalo, X0, Y0, m, s_list, s_warp);
    const PsiStage<FIX> st{s_img, s_pos, s_id, s_n, nS};
    Exact192 sr = exact_zero(), si = exact_zero();  // exact sums of this thread's psi_j
    int rmax = (m - 1) / 2;
    if constexpr (FIX) {
        const int lim = int((int64_t(1) << 31) / rep.W) - 1;
        if (lim < rmax) rmax = lim;
    }
    for (int d = threadIdx.x; d < D; d += kTileThreads<FIX, CAP>) {
        const int own = int(s_list[d] >> 4), k = int(s_list[d] & 15u);
        const P2<FIX> me = s_pos[k * nS + own];
        const int32_t idme = s_id[k * nS + own];
        typename Nbr<FIX>::Off rx[6], ry[6];
        bool ok = false;
        const int sy = own / kPsiSX;
        const int cx = X0 + (own - sy * kPsiSX) - kPsiHalo, cy = Y0 + sy - kPsiHalo;
        if constexpr (CAP == 4) {
            if (rmax >= 2) ok = nearest_float<FIX, CAP>(rep, st, own, k, me, rx, ry);
            if (!ok) {
                typename Nbr<FIX>::Off gx[6], gy[6];
                ok = nearest_general<FIX, CAP>(rep, st, cnt, pos, pid, own, cx, cy, me, idme, rmax, gx, gy);
#pragma unroll
                for (int q = 0; q < 6; ++q) {
                    rx[q] = gx[q];
                    ry[q] = gy[q];
                }
            }
        } else {
            ok = nearest_inserted<FIX, CAP>(rep, st, cnt, pos, pid, own, cx, cy, me, idme, rmax, rx, ry);
        }
        double pre, pim;
        if (!ok) {
            atomicOr(err, 2);
            pre = pim = 0.0;
        } else if constexpr (FIX) {
            float fr = 0.0f, fi = 0.0f;
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                const float x = __fmul_rn(__int2float_rn(rx[q]), 0x1p-24f);
                const float y = __fmul_rn(__int2float_rn(ry[q]), 0x1p-24f);
                const float xx = __fmul_rn(x, x), yy = __fmul_rn(y, y);
                const float r2 = __fadd_rn(xx, yy);
                const float c2 = __fsub_rn(xx, yy), s2 = __fmul_rn(__fmul_rn(x, y), 2.0f);
                const float c4 = __fsub_rn(__fmul_rn(c2, c2), __fmul_rn(s2, s2));
                const float s4 = __fmul_rn(__fmul_rn(c2, s2), 2.0f);
                const float c6 = __fsub_rn(__fmul_rn(c4, c2), __fmul_rn(s4, s2));
                const float s6 = __fadd_rn(__fmul_rn(c4, s2), __fmul_rn(s4, c2));
                const float r6 = __fmul_rn(__fmul_rn(r2, r2), r2);
                fr = __fadd_rn(fr, __fdiv_rn(c6, r6));
                fi = __fadd_rn(fi, __fdiv_rn(s6, r6));
            }
            pre = double(__fdiv_rn(fr, 6.0f));
            pim = double(__fdiv_rn(fi, 6.0f));
        } else {
            double dr_ = 0.0, di = 0.0;
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                const double x = rx[q], y = ry[q];
                const double xx = __dmul_rn(x, x), yy = __dmul_rn(y, y);
                const double r2 = __dadd_rn(xx, yy);
                const double c2 = __dsub_rn(xx, yy), s2 = __dmul_rn(__dmul_rn(x, y), 2.0);
                const double c4 = __dsub_rn(__dmul_rn(c2, c2), __dmul_rn(s2, s2));
                const double s4 = __dmul_rn(__dmul_rn(c2, s2), 2.0);
                const double c6 = __dsub_rn(__dmul_rn(c4, c2), __dmul_rn(s4, s2));
                const double s6 = __dadd_rn(__dmul_rn(c4, s2), __dmul_rn(s4, c2));
                const double r6 = __dmul_rn(__dmul_rn(r2, r2), r2);
                dr_ = __dadd_rn(dr_, __ddiv_rn(c6, r6));
                di = __dadd_rn(di, __ddiv_rn(s6, r6));
            }
            pre = __ddiv_rn(dr_, 6.0);
            pim = __ddiv_rn(di, 6.0);
        }
        if (local) local[rep.id_off + idme] = make_double2(pre, pim);
        exact_add(sr, pre);
        exact_add(si, pim);
    }
    // block sum: exact, so its value does not depend on the order of the disks
    const ExactPair t = exact_block_sum(sr, si);
    if (threadIdx.x == 0) {
        unsigned long long* w = total + size_t(r) * kPsiWords;
        const unsigned long long v[6] = {t.re.w0, t.re.w1, t.re.w2, t.im.w0, t.im.w1, t.im.w2};
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            atomicAdd(&w[2 * q], v[q] & 0xFFFFFFFFull);
            atomicAdd(&w[2 * q + 1], v[q] >> 32);
        }
        if (t.re.bad) atomicOr(&w[12], 1ull);
        if (t.im.bad) atomicOr(&w[12], 2ull);
    }
}

// Psi_6 of each replica: its exact sum rounded once to double, then divided by
// N (the oracle's order of operations).  One block of one warp per replica.
__global__ void __launch_bounds__(32)
k_psi6_reduce(const Rep* __restrict__ reps, unsigned long long* __restrict__ total, double* __restrict__ res) {
    pdl_begin(total);
    const int r = blockIdx.x, lane = int(threadIdx.x);
    unsigned long long* w = total + size_t(r) * kPsiWords;
    __shared__ unsigned long long s_w[kPsiWords];
    if (lane < 13) {
        s_w[lane] = w[lane];
        w[lane] = 0ull;
    }
    __syncwarp();
    if (lane < 2) {
        const unsigned long long* p = s_w + 6 * lane;
        unsigned long long limb[6], carry = 0ull;
#pragma unroll
        for (int q = 0; q < 6; ++q) {  // fewer than 2^31 blocks: no overflow
            const unsigned long long v = p[q] + carry;
            limb[q] = v & 0xFFFFFFFFull;
            carry = v >> 32;
        }
        const Exact192 sum{limb[0] | limb[1] << 32, limb[2] | limb[3] << 32, limb[4] | limb[5] << 32,
                           (unsigned int)(s_w[12] >> lane) & 1u};
        res[2 * r + lane] = __ddiv_rn(exact_round(sum), double(reps[r].N));
    }
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
template <bool FIX, int CAP>
static cudaError_t hist_t(const LaunchCfg& c, const HistCfg& h, CellBufs cells, unsigned long long* hist) {
    if (h.halo <= kHistMaxHalo) {
        static OncePerDevice once;
        const cudaError_t e = allow_smem(once, hist_stage_bytes<FIX, CAP>(kHistMaxHalo, kMaxFitBins), k_hist_tile<FIX, CAP>);
        if (e != cudaSuccess) return e;
        return launch_k(k_hist_tile<FIX, CAP>, dim3(c.blocks_t32), dim3(kTileThreads<FIX, CAP>),
                        hist_stage_bytes<FIX, CAP>(h.halo, h.K), c.stream, c.reps, c.R, h.K, h.edges,
                        h.edgesF, (const uint8_t*)cells.cnt, (const P2<FIX>*)cells.pos, (const int32_t*)cells.pid,
                        hist, h.halo);
    }
    return launch_k(k_hist_global<FIX, CAP>, dim3(c.blocks_cell), dim3(c.threads), size_t(h.K) * sizeof(unsigned int),
                    c.stream, c.reps, c.R, h.K, h.edges, h.edgesF, (const uint8_t*)cells.cnt,
                    (const P2<FIX>*)cells.pos, (const int32_t*)cells.pid, hist);
}

cudaError_t launch_hist(const LaunchCfg& c, const HistCfg& h, CellBufs cells, unsigned long long* hist) {
    if (c.fixed) return c.cap == 4 ? hist_t<true, 4>(c, h, cells, hist) : hist_t<true, 9>(c, h, cells, hist);
    return c.cap == 4 ? hist_t<false, 4>(c, h, cells, hist) : hist_t<false, 9>(c, h, cells, hist);
}

size_t fit_factor_len(int K) { return size_t(K); }

cudaError_t launch_fit_factor(cudaStream_t s, int K, double* qr) {
    if (K < 5 || K > kMaxFitBins) return cudaErrorInvalidValue;
    k_fit_factor<<<1, 32, 0, s>>>(K, qr);
    return cudaGetLastError();
}

cudaError_t launch_fit(const LaunchCfg& c, int K, const double* qr, const unsigned long long* hist, double* res) {
    if (K < 5 || K > kMaxFitBins) return cudaErrorInvalidValue;
    return launch_k(k_fit, dim3(c.R), dim3(32), 0, c.stream, c.reps, K, qr, hist, res);
}

size_t psi6_total_words(int R) { return size_t(R) * kPsiWords; }
int psi6_rows(bool fixed, int cap) { return (fixed || cap == 4 ? kTileThreads<true, 4> : kTileThreads<false, 9>) / 32; }

template <bool FIX, int CAP>
static cudaError_t psi6_t(const LaunchCfg& c, CellBufs cells, double2* local, unsigned long long* total, int* err) {
    constexpr size_t smem = psi6_stage_bytes<FIX, CAP>(kTileThreads<FIX, CAP> / 32);
    static OncePerDevice once;
    const cudaError_t e = allow_smem(once, smem, k_psi6<FIX, CAP>);
    if (e != cudaSuccess) return e;
    return launch_k(k_psi6<FIX, CAP>, dim3(c.blocks_t32), dim3(kTileThreads<FIX, CAP>), smem, c.stream, c.reps, c.R,
                    (const uint8_t*)cells.cnt, (const P2<FIX>*)cells.pos, (const int32_t*)cells.pid, local, total,
                    err);
}

cudaError_t launch_psi6(const LaunchCfg& c, CellBufs cells, double2* local, unsigned long long* total, int* err) {
    if (c.fixed) return c.cap == 4 ? psi6_t<true, 4>(c, cells, local, total, err) : psi6_t<true, 9>(c, cells, local, total, err);
    return c.cap == 4 ? psi6_t<false, 4>(c, cells, local, total, err) : psi6_t<false, 9>(c, cells, local, total, err);
}

__global__ void k_record(int R, const double* __restrict__ fit, const double* __restrict__ psi,
                         double* __restrict__ series, int64_t* __restrict__ len, int64_t cap, int* __restrict__ err) {
    pdl_begin(fit, psi, len);
    const int64_t idx = *len;
    const int r = threadIdx.x;
    if (r < R && idx < cap) {
        double* row = series + (size_t(idx) * R + r) * 4;
        row[0] = fit[4 * r];
        row[1] = fit[4 * r + 1];
        row[2] = psi[2 * r];
        row[3] = psi[2 * r + 1];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (idx < cap) *len = idx + 1;
        else atomicOr(err, 4);
    }
}

cudaError_t launch_record(const LaunchCfg& c, const double* fit, const double* psi, double* series, int64_t* len,
                          int64_t cap, int* err) {
    return launch_k(k_record, dim3(1), dim3(((c.R + 31) / 32) * 32), 0, c.stream, c.R, fit, psi, series, len, cap, err);
}

cudaError_t launch_psi6_reduce(const LaunchCfg& c, unsigned long long* total, double* res) {
    return launch_k(k_psi6_reduce, dim3(c.R), dim3(32), 0, c.stream, c.reps, total, res);
}

}  // namespace hd
