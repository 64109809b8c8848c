// hd_bin.cu -- positions given by the caller (hd_set_positions) binned into
// the unshifted cell frame on the device (Engel et al., arXiv:1211.1645,
// Sec. II.B: cell-relative coordinates).
#include "hd_cell.cuh"
#include "hd_kernels.h"
#include "hd_bin.h"

namespace hd {

// ---------------------------------------------------------------------------
// Binning of caller positions into the unshifted cell frame (hd_set_positions):
// one thread per disk, the same arithmetic as the host binning of the
// initial lattice and as the oracle, slots claimed with byte-lane atomics
// (the colour pass orders a cell by id).  Input errors set err bits
// kErrBinOverflow / kErrBinInput and leave the disk out.
// ---------------------------------------------------------------------------
static __device__ __noinline__ double2 bin_fp64_exact(double t, double w, double w_below, int m) {
    int cc = int(__ddiv_rn(t, w));
    if (cc > m - 1) cc = m - 1;
    if (cc < 0) cc = 0;
    double uu = __dsub_rn(t, __dmul_rn(double(cc), w));
    if (uu < 0.0 && cc > 0) {
        cc -= 1;
        uu = __dsub_rn(t, __dmul_rn(double(cc), w));
    }
    if (uu >= w && cc < m - 1) {
        cc += 1;
        uu = __dsub_rn(t, __dmul_rn(double(cc), w));
    }
    if (uu < 0.0) uu = 0.0;
    if (uu >= w) uu = w_below;
    return make_double2(double(cc), uu);
}

// The same without its division where the quotient t / w is not within 2^-30
// of an integer: the product with 1 / w errs by less than 2^-35 (quotients
// below 2^15), so its integer part is that of the rounded quotient, and the
// offset t - cc w is inside (0, w) with room for its roundings.  FP64 is the
// bound of the binning (N = 2^20: 114 -> 39 us).
__device__ __forceinline__ void bin_fp64_dev(double t, const Rep& r, int& c, double& u) {
    const double q = __dmul_rn(t, r.w_inv);
    const int cc = __double2int_rd(q);
    const double whole = double(cc);
    const double f = __dsub_rn(q, whole);
    if (cc >= 0 && cc < r.m && cc < (1 << 15) && !nonneg_bits(__dsub_rn(0x1p-30, f)) && below_pos_bits(f, 1.0 - 0x1p-30)) {
        c = cc;
        u = __dsub_rn(t, __dmul_rn(whole, r.w));
    } else {
        const double2 e = bin_fp64_exact(t, r.w, r.w_below, r.m);
        c = int(e.x);
        u = e.y;
    }
}

// floor(X / W) for 0 <= X < 2^53 and 0 < W < 2^31 with a quotient below 2^31:
// a float estimate (relative error below 2^-21, so within one of the
// quotient for quotients below 2^20, and corrected step by step otherwise)
// made exact with integer arithmetic, instead of a 64-bit integer division.
__device__ __forceinline__ int64_t floor_div_pos(int64_t X, int32_t W) {
    int64_t q = int64_t(__fmul_rn(__ll2float_rn(X), __frcp_rn(float(W))));
    int64_t r = X - q * int64_t(W);
    while (r < 0) {
        --q;
        r += W;
    }
    while (r >= int64_t(W)) {
        ++q;
        r -= W;
    }
    return q;
}

template <bool FIX, int CAP>
__global__ void __launch_bounds__(256)
k_bin(const Rep* __restrict__ reps, int R, int64_t Ntot, double sigma, const double* __restrict__ xy,
      uint8_t* __restrict__ cnt, P2<FIX>* __restrict__ pos, int32_t* __restrict__ pid, int* __restrict__ err) {
    pdl_begin(xy, cnt);
    const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= Ntot) return;
    int lo = 0, hi = R - 1;  // replica of global id i: last one with id_off <= i
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (reps[mid].id_off <= i) lo = mid; else hi = mid - 1;
    }
    const Rep& rep = reps[lo];
    // a division by 1 is exact: skip it (the FP64 pipe is narrow)
    const double px = sigma == 1.0 ? xy[2 * i] : __ddiv_rn(xy[2 * i], sigma);
    const double py = sigma == 1.0 ? xy[2 * i + 1] : __ddiv_rn(xy[2 * i + 1], sigma);
    if (!isfinite(px) || !isfinite(py)) {
        atomicOr(err, kErrBinInput);
        return;
    }
    int cx, cy;
    P2<FIX> q;
    if constexpr (FIX) {
        int64_t X = llround(__dmul_rn(px, 16777216.0));
        int64_t Y = llround(__dmul_rn(py, 16777216.0));
        // wrapped into [0, LF); a coordinate already inside needs no division
        if (X < 0 || X >= rep.LF) {
            X %= rep.LF;
            if (X < 0) X += rep.LF;
        }
        if (Y < 0 || Y >= rep.LF) {
            Y %= rep.LF;
            if (Y < 0) Y += rep.LF;
        }
        cx = int(floor_div_pos(X, rep.W));
        cy = int(floor_div_pos(Y, rep.W));
        q.x = int32_t(X - int64_t(cx) * rep.W);
        q.y = int32_t(Y - int64_t(cy) * rep.W);
    } else {
        // fmod returns a coordinate already in [0, L) unchanged
        auto into_box = [&](double v) {
            if (nonneg_bits(v) && below_pos_bits(v, rep.L)) return v;
            v = fmod(v, rep.L);
            if (v < 0.0) v = __dadd_rn(v, rep.L);
            return v >= rep.L ? 0.0 : v;
        };
        const double x = into_box(px), y = into_box(py);
        bin_fp64_dev(x, rep, cx, q.x);
        bin_fp64_dev(y, rep, cy, q.y);
    }
    const uint32_t c = rep.coff + row_part(rep, cy) + col_part(rep, cx);
    const int s = claim_slot(cnt, c);
    if (s >= CAP) {
        atomicOr(err, kErrBinOverflow);
        return;
    }
    pos[size_t(s) * rep.stride32 + c] = q;
    pid[size_t(s) * rep.stride32 + c] = int32_t(i - rep.id_off);
}

template <bool FIX, int CAP>
static cudaError_t bin_t(const LaunchCfg& c, int64_t Ntot, double sigma, const double* xy, CellBufs to, int* err) {
    return launch_k(k_bin<FIX, CAP>, dim3(unsigned((Ntot + 255) / 256)), dim3(256), 0, c.stream, c.reps, c.R, Ntot,
                    sigma, xy, to.cnt, (P2<FIX>*)to.pos, to.pid, err);
}

cudaError_t launch_bin(const LaunchCfg& c, int64_t Ntot, double sigma, const double* xy, CellBufs to, int* err) {
    if (c.fixed) return c.cap == 4 ? bin_t<true, 4>(c, Ntot, sigma, xy, to, err) : bin_t<true, 9>(c, Ntot, sigma, xy, to, err);
    return c.cap == 4 ? bin_t<false, 4>(c, Ntot, sigma, xy, to, err) : bin_t<false, 9>(c, Ntot, sigma, xy, to, err);
}

}  // namespace hd
