// hd_tile_cell.cuh -- a staged tile of cells in shared memory and the
// per-cell bodies of a sweep on it (Engel et al., arXiv:1211.1645, Sec.
// II.B): the scatter of a disk into its new cell, and one active cell's
// shuffle and trial moves against its staged neighbours.
//
// Layout.  The staged region is a rectangle of cells in unwrapped local
// coordinates (lx, ly), stored in four colour planes (parities of lx, ly) of
// HR rows and HP columns.  A pass reads the eight neighbours of its cell at
// three computed entries (row, column and diagonal plane) and compile-time
// offsets from them.  Per cell: float images of the positions in slots 0 and
// 1 side by side, so that one 16-byte load brings both of a neighbour's disks;
// what the images leave out of the exact positions; the ids; and one word.  A pair is decided in float
// unless the estimate lies within its error bound of contact (hd_bounds.h),
// which about one trial in 10^4 sees: five full-rate instructions per slot.
// The integer test of the fixed form takes two 32 x 32 -> 64 multiplications
// instead, which issue at a quarter of the rate (measured: 16 slots in 114
// cycles per warp and scheduler, against 69 in float).  An unoccupied slot
// holds an image so far away that no test rejects, so a test needs no
// occupancy.
//   word: bits 0..3 occupancy; bits 4..11 which of the eight neighbours hold
//   more than two disks; bits 12..21 and 22..31 where slots 2 and 3 are kept:
//   entry e of the block's pool as e + 1, or kFar for the block's global
//   spill area.
// Cells of three disks are rare unless cells are clearly wider than 2 sigma (counted
// over random frames of relaxed chains: 4e-6 of the cells at 2.001 sigma, eta = 0.716;
// 2e-5 at 2.024, 0.70; 4e-4 at 2.094, N = 1000; 1e-3 at 2.119, N = 256), so the pool is
// small; the spill area keeps any accepted configuration correct.
#pragma once

#include "hd_cell.cuh"

namespace hd {

constexpr int kTileHalo = 4;            // staged cells around a tile: one per colour pass
constexpr int kCrowdShift = 4;
constexpr uint32_t kFar = 0x3FFu;
constexpr float kFarFloat = 1e18f;      // it and its square are above any contact distance squared, and finite

template <bool FIX>
struct PoolEntry {
    P2<FIX> p;
    int32_t id;
    int32_t cell;  // lx | ly << 16 of a slot 2, -1 of a slot 3
};

// Float image of a coordinate, as the pair tests use it.  Fixed form: its
// integer (below 2^26) without the two lowest bits, in units of 2^-22 sigma;
// those bits are kept beside it, so image and bits are the exact position and
// a staged cell takes 30 bytes.
template <bool FIX, class T>
__device__ __forceinline__ float image(T v) {
    if constexpr (FIX) return __int2float_rn(v >> 2);
    else return approx_f32(v);
}

template <bool FIX, int HP_, int HR_, int POOL_>
struct Stage {
    static constexpr int HP = HP_, HR = HR_, NP = HP_ * HR_, NC = 4 * NP, POOL = POOL_;
    float4* quad;         // [NC] images of slots 0 and 1
    double2* p0;          // FP64 form: [NC] slot 0, [NC] slot 1
    uint8_t* low;         // fixed form: [2 NC] lowest bits of x | y << 2 of slots 0 and 1
    int2* id;             // [NC]
    uint32_t* word;       // [NC]
    PoolEntry<FIX>* pool; // [POOL]
    PoolEntry<FIX>* spill;  // global, [2 NC]
    uint32_t* pool_n;
    // The hard cells of each colour plane: those that hold more than two disks
    // or have a neighbour that does (3e-5 of the cells at 2.001 sigma, 0.7% at N = 256,
    // most where cells are wide).  A pass gives them warps of their own, so that
    // the others do not walk the rare paths with them.  hard_n[4] is set when a list or the
    // pool overflowed; the passes then look at every cell for them.
    uint16_t* hard;       // [4][HARD] hy * HP + hx
    uint32_t* hard_n;     // [5]
    static constexpr int HARD = 160;

    static constexpr size_t kBytes = (size_t(NC) * (16 + (FIX ? 2 : 32) + 8 + 4) + size_t(POOL) * sizeof(PoolEntry<FIX>) +
                                      size_t(4 * HARD) * 2 + 32 + 15) & ~size_t(15);
    __device__ __forceinline__ Stage(unsigned char* s, PoolEntry<FIX>* g) {
        quad = reinterpret_cast<float4*>(s);
        s += size_t(NC) * 16;
        p0 = reinterpret_cast<double2*>(s);
        if constexpr (!FIX) s += size_t(NC) * 32;
        pool = reinterpret_cast<PoolEntry<FIX>*>(s);
        s += size_t(POOL) * sizeof(PoolEntry<FIX>);
        id = reinterpret_cast<int2*>(s);
        s += size_t(NC) * 8;
        word = reinterpret_cast<uint32_t*>(s);
        s += size_t(NC) * 4;
        hard = reinterpret_cast<uint16_t*>(s);
        s += size_t(4 * HARD) * 2;
        pool_n = reinterpret_cast<uint32_t*>(s);
        hard_n = pool_n + 1;
        s += 32;
        low = s;
        spill = g;
    }
    static __device__ __forceinline__ int index(int lx, int ly) {
        return (((ly & 1) << 1) | (lx & 1)) * NP + (ly >> 1) * HP + (lx >> 1);
    }
    // where slot k (2 or 3) of cell e with word w is kept
    __device__ __forceinline__ PoolEntry<FIX>* extra(uint32_t w, int e, int k) const {
        const uint32_t f = (w >> (k == 2 ? 12 : 22)) & 0x3FFu;
        return f == kFar ? spill + (k - 2) * NC + e : pool + (f - 1u);
    }
    __device__ __forceinline__ void clear(int e) const {
        word[e] = 0u;
        quad[e] = make_float4(kFarFloat, kFarFloat, kFarFloat, kFarFloat);
    }
    // The exact position in slot k (0 or 1) of entry e, and its replacement.
    __device__ __forceinline__ P2<FIX> exact(float fx, float fy, uint32_t bits) const {
        return make_int2((__float2int_rn(fx) << 2) | int(bits & 3u), (__float2int_rn(fy) << 2) | int((bits >> 2) & 3u));
    }
    __device__ __forceinline__ P2<FIX> get(int e, int k) const {
        if constexpr (FIX) {
            const float2 f = reinterpret_cast<const float2*>(quad)[2 * e + k];
            return exact(f.x, f.y, low[2 * e + k]);
        } else {
            return p0[k * NC + e];
        }
    }
    __device__ __forceinline__ void set(int e, int k, const P2<FIX>& p) const {
        reinterpret_cast<float2*>(quad)[2 * e + k] = make_float2(image<FIX>(p.x), image<FIX>(p.y));
        if constexpr (FIX) low[2 * e + k] = uint8_t((p.x & 3) | (p.y & 3) << 2);
        else p0[k * NC + e] = p;
    }
    // The same in several entries: what is stored of a position, made once.
    struct Stored {
        float2 f;
        P2<FIX> p;
    };
    __device__ __forceinline__ Stored stored(const P2<FIX>& p) const {
        return Stored{make_float2(image<FIX>(p.x), image<FIX>(p.y)), p};
    }
    __device__ __forceinline__ void set(int e, int k, const Stored& v) const {
        reinterpret_cast<float2*>(quad)[2 * e + k] = v.f;
        if constexpr (FIX) low[2 * e + k] = uint8_t((v.p.x & 3) | (v.p.y & 3) << 2);
        else p0[k * NC + e] = v.p;
    }
    // Claim a slot of local cell (lx, ly), entry e, for disk (p, i); false if the cell is full.
    __device__ __forceinline__ bool place(int lx, int ly, int e, const P2<FIX>& p, int32_t i) const {
        const uint32_t s = atomicAdd(&word[e], 1u) & 0xFu;
        if (s < 2u) {
            set(e, int(s), p);
            reinterpret_cast<int32_t*>(id)[2 * e + s] = i;
            return true;
        }
        return place_extra(lx, ly, e, s, p, i);
    }
    // A third or fourth disk (rare).
    __device__ __noinline__ bool place_extra(int lx, int ly, int e, uint32_t s, P2<FIX> p, int32_t i) const {
        if (s >= 4u) return false;
        const uint32_t q = atomicAdd(pool_n, 1u);
        const bool near = q < uint32_t(POOL);
        PoolEntry<FIX>* x = near ? pool + q : spill + (s - 2u) * NC + e;
        x->p = p;
        x->id = i;
        x->cell = s == 2u ? (lx | ly << 16) : -1;
        atomicAdd(&word[e], (near ? q + 1u : kFar) << (s == 2u ? 12 : 22));
        if (!near) {
            hard_n[4] = 1u;
            if (s == 2u)
                for (int d = 0; d < 8; ++d) mark_crowded(lx, ly, d);
        }
        return true;
    }
    // Tell the neighbour of crowded cell (lx, ly) in direction 7 - d (the
    // eight offsets in row order) that its neighbour in direction d is
    // crowded; returns its word before, or a word of no disks if it is not staged.
    __device__ __forceinline__ uint32_t mark_crowded(int lx, int ly, int d, int* nx = nullptr, int* ny = nullptr) const {
        const int k = 7 - d, i = k + (k >= 4 ? 1 : 0);
        const int x = lx + i % 3 - 1, y = ly + i / 3 - 1;
        if (nx) *nx = x;
        if (ny) *ny = y;
        if (x < 0 || x >= 2 * HP || y < 0 || y >= 2 * HR) return 0u;
        return atomicOr(&word[index(x, y)], 1u << (kCrowdShift + d));
    }
    __device__ __forceinline__ void list_hard(int lx, int ly) const {
        const int col = ((ly & 1) << 1) | (lx & 1);
        const uint32_t k = atomicAdd(&hard_n[col], 1u);
        if (k < uint32_t(HARD)) hard[col * HARD + k] = uint16_t((ly >> 1) * HP + (lx >> 1));
        else hard_n[4] = 1u;
    }
    // Once every disk is placed: pool entry x's cell and its neighbours in
    // direction d are marked and listed.
    __device__ __forceinline__ void mark_entry(uint32_t x, int d) const {
        const int32_t at = pool[x].cell;
        if (at < 0) return;
        const int lx = at & 0xFFFF, ly = at >> 16;
        int nx, ny;
        const uint32_t old = mark_crowded(lx, ly, d, &nx, &ny), n = old & 0xFu;
        if (n >= 1u && n <= 2u && ((old >> kCrowdShift) & 0xFFu) == 0u) list_hard(nx, ny);
        if (d == 0) list_hard(lx, ly);
    }
};

__device__ __forceinline__ bool is_hard(uint32_t w) {
    const uint32_t n = w & 0xFu;
    return n > 2u || (n > 0u && ((w >> kCrowdShift) & 0xFFu) != 0u);
}

// Constants of a replica that the tile bodies use.
template <bool FIX>
struct TileRep {
    int32_t W, D, m, nt;
    uint32_t key0, key1;
    double w, w_below, delta;
    float wf, d2_lo, d2_hi;
    __device__ __forceinline__ explicit TileRep(const Rep& r)
        : W(r.W), D(r.D), m(r.m), nt(r.nt), key0(r.key0), key1(r.key1), w(r.w), w_below(r.w_below), delta(r.delta),
          wf(r.wf), d2_lo(r.d2_lo), d2_hi(r.d2_hi) {}
};

// The eight neighbours of local cell e = (plane col, half-row hy, half-column
// hx): entry of neighbour (ox, oy).
template <class S>
struct NbrBase {
    int h, v, d;  // left neighbour; upper neighbour; upper-left neighbour
    __device__ __forceinline__ NbrBase(int px, int py, int hx, int hy) {
        const int row = hy * S::HP, up = (hy - 1 + py) * S::HP, left = hx - 1 + px;
        h = ((py << 1) | (1 - px)) * S::NP + row + left;
        v = (((1 - py) << 1) | px) * S::NP + up + hx;
        d = (((1 - py) << 1) | (1 - px)) * S::NP + up + left;
    }
    __device__ __forceinline__ int at(int ox, int oy) const {
        if (oy == 0) return ox < 0 ? h : h + 1;
        if (ox == 0) return oy < 0 ? v : v + S::HP;
        return d + (ox < 0 ? 0 : 1) + (oy < 0 ? 0 : S::HP);
    }
};

// One pair by its exact test (rare cases).
template <bool FIX>
__device__ __forceinline__ bool pair_clear_at(const P2<FIX>& q, int ox, int oy, const P2<FIX>& np, const TileRep<FIX>& rep) {
    if constexpr (FIX) {
        const int32_t rx = (q.x + ox * rep.W) - np.x, ry = (q.y + oy * rep.W) - np.y;
        return uint32_t((uint64_t(int64_t(rx) * rx) + uint64_t(int64_t(ry) * ry)) >> 32) >= (1u << 18);
    } else {
        return pair_clear_fp64_exact(q.x, q.y, ox, oy, np.x, np.y, rep.w);
    }
}

// True when np (a proposed position in the local cell nb belongs to, inside
// the cell) is at least 2 sigma from every disk of the eight neighbours and,
// where has_other, from `other` (the second disk of its own cell).  crowd:
// which of the eight neighbours hold more than two disks.
template <bool FIX, class S>
__device__ __forceinline__ bool tile_clear(const S& st, const TileRep<FIX>& rep, const NbrBase<S>& nb, const P2<FIX>& np,
                                           const P2<FIX>& other, bool has_other, uint32_t crowd, int lx, int ly) {
    const float fx = image<FIX>(np.x), fy = image<FIX>(np.y);
    const float ax[3] = {__fadd_rn(fx, rep.wf), fx, __fsub_rn(fx, rep.wf)};
    const float ay[3] = {__fadd_rn(fy, rep.wf), fy, __fsub_rn(fy, rep.wf)};
    auto d2f = [](float rx, float ry) { return __fmaf_rn(rx, rx, __fmul_rn(ry, ry)); };
    const float own = has_other ? d2f(__fsub_rn(image<FIX>(other.x), fx), __fsub_rn(image<FIX>(other.y), fy)) : kFarFloat;
    float least = own;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        if (i == 4) continue;
        const float4 q = st.quad[nb.at(i % 3 - 1, i / 3 - 1)];
        const float bx = ax[i % 3], by = ay[i / 3];
        least = fminf(least, d2f(__fsub_rn(q.x, bx), __fsub_rn(q.y, by)));
        least = fminf(least, d2f(__fsub_rn(q.z, bx), __fsub_rn(q.w, by)));
    }
    bool ok = least >= rep.d2_hi;
    if (!ok && least >= rep.d2_lo) {  // rare: some pair is within the band
        ok = !(own < rep.d2_hi) || pair_clear_at<FIX>(other, 0, 0, np, rep);
#pragma unroll 1
        for (int i = 0; i < 9; ++i) {
            if (i == 4) continue;
            const int ox = i % 3 - 1, oy = i / 3 - 1, e = S::index(lx + ox, ly + oy);
            const float4 q = st.quad[e];
            const float bx = ox < 0 ? ax[0] : (ox > 0 ? ax[2] : ax[1]), by = oy < 0 ? ay[0] : (oy > 0 ? ay[2] : ay[1]);
            if (d2f(__fsub_rn(q.x, bx), __fsub_rn(q.y, by)) < rep.d2_hi) ok = ok && pair_clear_at<FIX>(st.get(e, 0), ox, oy, np, rep);
            if (d2f(__fsub_rn(q.z, bx), __fsub_rn(q.w, by)) < rep.d2_hi) ok = ok && pair_clear_at<FIX>(st.get(e, 1), ox, oy, np, rep);
        }
    }
    // crowded neighbours: only the marked ones
    for (uint32_t c = ok ? crowd : 0u; c != 0u; c &= c - 1u) {
        const int q = __ffs(int(c)) - 1, i = q + (q >= 4 ? 1 : 0);
        const int ox = int((0x24924u >> (2 * i)) & 3u) - 1;  // i % 3 - 1
        const int oy = int((0x2A540u >> (2 * i)) & 3u) - 1;  // i / 3 - 1
        const int e = S::index(lx + ox, ly + oy);
        const uint32_t w = st.word[e];
        const int n = min(int(w & 15u), 4);
        for (int k = 2; k < n; ++k) ok = ok && pair_clear_at<FIX>(st.extra(w, e, k)->p, ox, oy, np, rep);
    }
    return ok;
}

// Order of three or four occupants after the shuffle, one nibble per position
// (Fisher-Yates as try_cell_in: swap k uses word n - 1 - k of the stream).
// Fixed form: the first two words come from trial 0's block.
template <bool FIX>
static __device__ __noinline__ uint32_t shuffle_many(int n, uint32_t sweep, uint32_t cl, uint32_t key0, uint32_t key1,
                                                     uint32_t z, uint32_t w) {
    uint32_t word[3] = {z, w, 0u};
    if (!FIX || n > 3) {
        const uint4 a = philox(sweep, 0u, cl, kTagShuffle, key0, key1);
        if constexpr (FIX) {
            word[2] = a.x;
        } else {
            word[0] = a.x;
            word[1] = a.y;
            word[2] = a.z;
        }
    }
    uint32_t order = 0x3210u;
#pragma unroll
    for (int k = 3; k >= 1; --k) {
        if (k < n) {
            const uint32_t j = bounded(n - 1 - k == 0 ? word[0] : (n - 1 - k == 1 ? word[1] : word[2]), uint32_t(k + 1));
            const uint32_t vk = (order >> (4 * k)) & 0xFu, vj = (order >> (4 * j)) & 0xFu;
            order &= ~((0xFu << (4 * k)) | (0xFu << (4 * j)));
            order |= (vj << (4 * k)) | (vk << (4 * j));
        }
    }
    return order;
}

// The occupants of crowded cell e (word w) in ascending id.
template <bool FIX, class S>
static __device__ __noinline__ void gather_many(const S& st, int e, uint32_t w, int n, P2<FIX>* P, int32_t* I) {
    for (int k = 0; k < n; ++k) {
        P2<FIX> p;
        int32_t i;
        if (k < 2) {
            p = st.get(e, k);
            i = reinterpret_cast<const int32_t*>(st.id)[2 * e + k];
        } else {
            const PoolEntry<FIX>* x = st.extra(w, e, k);
            p = x->p;
            i = x->id;
        }
        int s = k;
        for (; s > 0 && I[s - 1] > i; --s) {
            P[s] = P[s - 1];
            I[s] = I[s - 1];
        }
        P[s] = p;
        I[s] = i;
    }
}

// ... and back after their moves.
template <bool FIX, class S>
static __device__ __noinline__ void put_many(const S& st, int e, uint32_t w, int n, const P2<FIX>* P) {
    for (int k = 0; k < n; ++k) {
        if (k < 2) {
            st.set(e, k, P[k]);
        } else {
            st.extra(w, e, k)->p = P[k];
        }
    }
}

// The draws of a cell's first trial, made ahead: the step, and the word that
// decides the shuffle of two occupants.
template <bool FIX>
__device__ __forceinline__ P2<FIX> trial_step(const TileRep<FIX>& rep, const uint4& u) {
    if constexpr (FIX) {
        const uint32_t span = uint32_t(2 * rep.D + 1);
        return make_int2(int32_t(bounded(u.x, span)) - rep.D, int32_t(bounded(u.y, span)) - rep.D);
    } else {
        return make_double2(step_fp64(u.x, u.y, rep.delta), step_fp64(u.z, u.w, rep.delta));
    }
}
template <bool FIX>
struct Drawn {
    P2<FIX> step;
    uint32_t swap;
    uint32_t swap2 = 0u;  // the second word of the shuffle (hard_cell_ahead)
};

// One active cell: plane (px, py), half-row hy, half-column hx, word w, Philox
// cell counter cl.  Its occupants are ordered by id, shuffled and make rep.nt
// serial trial moves, as try_cell_in defines.  Cells of one or two disks keep
// them in registers; the few with more take their moving disk from per-thread
// memory.  HARD = false: the cell is known not to be hard.  PRE: the first
// trial's draws are given; the caller's emit stores the positions of slots 0
// and 1 in the stage.  emit(k, position, id) is called for every occupant
// afterwards.  Returns the accepted moves.
template <bool FIX, int NTC, bool HARD, bool PRE, class S, class Emit>
__device__ __forceinline__ uint32_t tile_cell(const S& st, const TileRep<FIX>& rep, uint32_t sweep, int px, int py, int hx,
                                              int hy, uint32_t w, uint32_t cl, Emit&& emit,
                                              const Drawn<FIX>& pre = Drawn<FIX>{}) {
    const int e = ((py << 1) | px) * S::NP + hy * S::HP + hx;
    const int n = min(int(w & 15u), 4);
    const bool two = n == 2, many = HARD && n > 2;
    const NbrBase<S> nb(px, py, hx, hy);
    const uint32_t crowd = HARD ? (w >> kCrowdShift) & 0xFFu : 0u;
    P2<FIX> q0, q1;
    if constexpr (FIX) {
        const float4 f = st.quad[e];
        const uint32_t bits = reinterpret_cast<const uint16_t*>(st.low)[e];
        q0 = st.exact(f.x, f.y, bits);
        q1 = st.exact(f.z, f.w, bits >> 8);  // not a disk's unless two
    } else {
        q0 = q1 = st.get(e, 0);
        if (two) q1 = st.get(e, 1);
    }
    int2 ids = st.id[e];
    if (two && ids.y < ids.x) {  // ascending id: the base order of the shuffle
        const P2<FIX> t = q0;
        q0 = q1;
        q1 = t;
        ids = make_int2(ids.y, ids.x);
    }
    // Fisher-Yates of two: position 0 takes slot 1 when the swap word's bound is 0
    uint4 u0 = make_uint4(0u, 0u, 0u, 0u);
    bool flip = false;
    if constexpr (PRE) {
        flip = two && (pre.swap >> 31) == 0u;
        if (FIX && many) u0 = philox(sweep, 0u, cl, kTagTrial, rep.key0, rep.key1);
    } else if constexpr (FIX) {
        u0 = philox(sweep, 0u, cl, kTagTrial, rep.key0, rep.key1);
        flip = two && (u0.z >> 31) == 0u;
    } else if (two) {
        flip = (philox(sweep, 0u, cl, kTagShuffle, rep.key0, rep.key1).x >> 31) == 0u;
    }
    P2<FIX> P[4];
    int32_t I[4];
    uint32_t order = 0u;
    if (many) {
        gather_many<FIX, S>(st, e, w, n, P, I);
        order = shuffle_many<FIX>(n, sweep, cl, rep.key0, rep.key1, u0.z, u0.w);
    }
    uint32_t acc = 0;
    const int nt = NTC > 0 ? NTC : rep.nt;
    for (int t = 0; t < nt; ++t) {
        P2<FIX> step;
        if (PRE && t == 0) step = pre.step;
        else step = trial_step<FIX>(rep, (FIX && !PRE && t == 0) ? u0 : philox(sweep, uint32_t(t), cl, kTagTrial, rep.key0, rep.key1));
        const bool second = two && (((t & 1) != 0) != flip);
        P2<FIX> me = second ? q1 : q0, other = second ? q0 : q1;
        int slot = 0;
        if (many) {
            slot = int((order >> (4 * (t % n))) & 0xFu);
            me = P[slot];
        }
        P2<FIX> np;
        bool ok;
        if constexpr (FIX) {
            np.x = me.x + step.x;
            np.y = me.y + step.y;
            ok = uint32_t(np.x) < uint32_t(rep.W) && uint32_t(np.y) < uint32_t(rep.W);
        } else {
            np.x = __dadd_rn(me.x, step.x);
            np.y = __dadd_rn(me.y, step.y);
            ok = nonneg_bits(np.x) && below_pos_bits(np.x, rep.w) && nonneg_bits(np.y) && below_pos_bits(np.y, rep.w);
        }
        if (ok) ok = tile_clear<FIX, S>(st, rep, nb, np, other, two, crowd, 2 * hx + px, 2 * hy + py);
        if (many && ok)
            for (int k = 0; k < n; ++k) ok = ok && (k == slot || pair_clear_at<FIX>(P[k], 0, 0, np, rep));
        if (ok) {
            if (many) P[slot] = np;
            else if (second) q1 = np;
            else q0 = np;
            ++acc;
        }
    }
    if (many) {
        if (acc) put_many<FIX, S>(st, e, w, n, P);
        for (int k = 0; k < n; ++k) emit(k, P[k], I[k]);
        return acc;
    }
    if (!PRE && acc) {
        st.set(e, 0, q0);
        if (two) st.set(e, 1, q1);
    }
    emit(0, q0, ids.x);
    if (two) emit(1, q1, ids.y);
    return acc;
}

// A hard cell whose first trial's draws were made ahead, all of its occupants in
// registers: one path for one to four disks, so that the few threads of a pass
// that have such cells run it together.  Arguments and results as of tile_cell.
template <bool FIX, int NTC, class S, class Emit>
__device__ __forceinline__ uint32_t hard_cell_ahead(const S& st, const TileRep<FIX>& rep, uint32_t sweep, int px, int py,
                                                    int hx, int hy, uint32_t w, uint32_t cl, Emit&& emit,
                                                    const Drawn<FIX>& pre) {
    const int e = ((py << 1) | px) * S::NP + hy * S::HP + hx;
    const int n = min(int(w & 15u), 4);
    const NbrBase<S> nb(px, py, hx, hy);
    const int2 ids = st.id[e];
    P2<FIX> P[4] = {st.get(e, 0), st.get(e, 1)};  // slots at or beyond n are no disks
    int32_t I[4] = {ids.x, ids.y, 0, 0};
    P[2] = P[3] = P[0];
    uint32_t order = 0x3210u;  // position -> slot, Fisher-Yates as try_cell_in
    if (n > 2) {
#pragma unroll
        for (int k = 2; k < 4; ++k) {
            if (k >= n) continue;
            const PoolEntry<FIX>* x = st.extra(w, e, k);
            P[k] = x->p;
            I[k] = x->id;
        }
        sort_by_id<FIX, 4>(P, I, n);
        uint32_t third = 0u;
        if (n > 3) {
            const uint4 a = philox(sweep, 0u, cl, kTagShuffle, rep.key0, rep.key1);
            third = FIX ? a.x : a.z;
        }
#pragma unroll
        for (int k = 3; k >= 1; --k) {
            if (k >= n) continue;
            const int i = n - 1 - k;
            const uint32_t j = bounded(i == 0 ? pre.swap : (i == 1 ? pre.swap2 : third), uint32_t(k + 1));
            const uint32_t vk = (order >> (4 * k)) & 0xFu, vj = (order >> (4 * j)) & 0xFu;
            order &= ~((0xFu << (4 * k)) | (0xFu << (4 * j)));
            order |= (vj << (4 * k)) | (vk << (4 * j));
        }
    } else if (n == 2) {
        if (ids.y < ids.x) {
            const P2<FIX> t = P[0];
            P[0] = P[1];
            P[1] = t;
            I[0] = ids.y;
            I[1] = ids.x;
        }
        if ((pre.swap >> 31) == 0u) order = 0x3201u;
    }
    const RegCell<FIX, 4> cell{P};
    uint32_t acc = 0;
    const int nt = NTC > 0 ? NTC : rep.nt;
    for (int t = 0; t < nt; ++t) {
        const P2<FIX> step =
            t == 0 ? pre.step : trial_step<FIX>(rep, philox(sweep, uint32_t(t), cl, kTagTrial, rep.key0, rep.key1));
        const int slot = int((order >> (4 * (t == 0 ? 0 : t % n))) & 0xFu);
        const P2<FIX> me = cell.pick(slot);
        P2<FIX> np;
        bool ok;
        if constexpr (FIX) {
            np.x = me.x + step.x;
            np.y = me.y + step.y;
            ok = uint32_t(np.x) < uint32_t(rep.W) && uint32_t(np.y) < uint32_t(rep.W);
            auto own = [&](int q) { ok &= pair_clear_at<FIX>(P[q], 0, 0, np, rep) | (q >= n) | (q == slot); };
            own(0);
            own(1);
            if (n > 2) {
                own(2);
                own(3);
            }
        } else {
            np.x = __dadd_rn(me.x, step.x);
            np.y = __dadd_rn(me.y, step.y);
            ok = nonneg_bits(np.x) && below_pos_bits(np.x, rep.w) && nonneg_bits(np.y) && below_pos_bits(np.y, rep.w);
            const float fx = image<FIX>(np.x), fy = image<FIX>(np.y);
            float least = kFarFloat;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float rx = __fsub_rn(image<FIX>(P[q].x), fx), ry = __fsub_rn(image<FIX>(P[q].y), fy);
                if (q < n && q != slot) least = fminf(least, __fmaf_rn(rx, rx, __fmul_rn(ry, ry)));
            }
            ok = ok && least >= rep.d2_lo;
            if (ok && least < rep.d2_hi) {  // rare: some pair is within the band
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (q < n && q != slot) ok = ok && pair_clear_at<FIX>(P[q], 0, 0, np, rep);
            }
        }
        if (ok) ok = tile_clear<FIX, S>(st, rep, nb, np, np, false, (w >> kCrowdShift) & 0xFFu, 2 * hx + px, 2 * hy + py);
        if (ok) {
            cell.put(slot, np);
            ++acc;
        }
    }
    emit(0, P[0], I[0]);
    if (n > 1) emit(1, P[1], I[1]);
    if (n > 2) {
        emit(2, P[2], I[2]);
        if (n > 3) emit(3, P[3], I[3]);
    }
    return acc;
}

}  // namespace hd
