// hd_tile.cu -- many checkerboard sweeps in one launch, a whole sweep of a
// tile of cells at a time in shared memory (Engel et al., arXiv:1211.1645,
// Sec. II.B).
//
// Work items.  Item (sweep i, tile t) of a launch reads the cells of tile t
// and a few cells around it as they stood after sweep i - 1, moves their
// disks into the sweep's shifted frame in shared memory, makes the four
// colour passes there, and writes the tile's own cells.  Pass p needs the
// neighbours of its active cells as they stood after pass p - 1, so earlier
// passes also update the surrounding cells the later ones read: their draws
// are keyed by the global cell index, so every copy of a cell evolves
// identically and the owner's copy is the one written.  How far a pass
// reaches follows from the colour order of the sweep (active_range): two to
// three cells on average, four at most.  A cell's final state is known after
// its own colour's pass, and the thread that made it writes it out.
//
// Dependencies.  Item (i, t) needs sweep i - 1 of tile t and of the eight
// tiles around it (periodically).  That also makes overwriting the other
// generation safe: its last readers were sweep i - 1 of the same tiles.
// progress[tile] counts the tile's finished sweeps; a block publishes with a
// release add after all its threads are done, and one warp polls the nine
// words with acquire loads.  Blocks take items in ticket order and an item
// depends on lower tickets only, so no co-residency is assumed.  Each sweep
// starts one row of tiles further on than the one before, so that its first
// items depend on the first items of the previous sweep.  A wait that gives
// up after `polls` polls sets bit 16 of err and an abort word, and every
// block leaves.
#include <algorithm>

#include "hd_kernels.h"
#include "hd_tile.h"
#include "hd_tile_cell.cuh"

namespace hd {
namespace {

constexpr int kErrPersist = 16;
constexpr int kLookAhead = 3;  // pass of an item at which the block takes its next ticket
constexpr uint32_t kTilePolls = 1u << 22;

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_release_add(uint32_t* p, uint32_t v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;\n" ::"l"(p), "r"(v) : "memory");
}

// Staging capacity and launch shape of one form: one block per SM with as large
// a staged region as its shared memory holds, since the cells around a tile
// are worked on twice (fixed form: 104 x 68 cells, tiles of up to 96 x 60; over the
// 24 colour orders, the 12 x 18 tiles of N = 2^20 load 1.14 cells and update 1.06 for
// each they own).  Measured at N = 2^20, fixed form, us per sweep:
// 768 threads at 80 registers 29.0, 640 31.3, 992 at 64 registers 32.0 (spills);
// two blocks of 384 threads and half the region each 29.7, three of 256 39.7.
template <bool FIX>
struct TileShape;
template <>
struct TileShape<true> {
    static constexpr int HP = 52, HR = 34, POOL = 384, NT = 768;
};
template <>
struct TileShape<false> {
    static constexpr int HP = 39, HR = 23, POOL = 160, NT = 768;
};
template <bool FIX>
using TileStage = Stage<FIX, TileShape<FIX>::HP, TileShape<FIX>::HR, TileShape<FIX>::POOL>;

__device__ __forceinline__ int wrap1(int c, int m) { return c < 0 ? c + m : (c >= m ? c - m : c); }

// e / n for e < 2^13, 1 <= n <= 128: mul = ceil(2^20 / n)
__device__ __forceinline__ uint32_t small_mul(uint32_t n) { return ((1u << 20) + n - 1u) / n; }
__device__ __forceinline__ uint32_t small_div(uint32_t e, uint32_t mul) { return (e * mul) >> 20; }

// v mod n for v < 2 n, or with twice for v < 3 n
__device__ __forceinline__ uint32_t wrap_half(uint32_t v, uint32_t n, bool twice = false) {
    v = min(v, v - n);
    return twice ? min(v, v - n) : v;
}

// What a block's threads need to know of an item, worked out by one warp
// while the others are in the passes of the item before (every thread doing
// so itself took a third of the kernel's instructions, mostly divisions).
struct TileItem {
    int32_t r, tw, th;          // replica; the tile's cells per axis
    uint32_t hx, hy;            // half-column and half-row of the cell 6 cells before its first, in [0, m / 2)
    int32_t tx, ty, ntx, nty, first;
    int32_t twice;              // staged cells reach over the box more than once (one tile on an axis)
    int32_t go;                 // 0: no item is left (or a wait gave up)
    uint32_t i, sweep, perm;    // sweep of the launch; of the chain (Philox word); colour order
    int32_t fx, fy, ox, oy;     // ShiftDelta
    double dx, dy;
    int32_t lo0x, hi0x, lo0y, hi0y;  // local cells needed before the first pass
    int32_t lhx, lhy;                // half-cell range of the old cells that feed them
    uint32_t lnx, lcells, lmul;
    CellBufs from, to;               // the generations read and written
    uint32_t stride, coff, hh, hm;   // of the replica
    struct {
        int32_t col, hx, hy;  // colour, first half-column and half-row
        uint32_t nx, ny, cells, mul;
    } pass[4];
};

// The range of cells of one axis, of a tile [kTileHalo, kTileHalo + t), whose
// state after pass p is needed, from the last pass back to `upto`: a pass
// reads one cell beyond an active first or last cell.
__device__ __forceinline__ void active_range(uint32_t perm, int axis, int t, int upto, int& lo, int& hi) {
    lo = kTileHalo;
    hi = kTileHalo + t;
    for (int p = 3; p > upto; --p) {
        const int q = int(perm >> (2 * p + axis)) & 1;
        lo -= ((lo ^ q) & 1) == 0 ? 1 : 0;
        hi += (((hi - 1) ^ q) & 1) == 0 ? 1 : 0;
    }
}

// Add a warp's trials and acceptances to the counters of replica r.
__device__ __forceinline__ void warp_count(uint32_t att, uint32_t acc, unsigned long long* counters, int r) {
    att = __reduce_add_sync(0xffffffffu, att);
    acc = __reduce_add_sync(0xffffffffu, acc);
    const int lane = int(threadIdx.x & 31u);
    if (lane == 0 && att) atomicAdd(&counters[2 * r], (unsigned long long)att);
    if (lane == 1 && acc) atomicAdd(&counters[2 * r + 1], (unsigned long long)acc);
}

// Fill *t for item `item` (one warp).
template <bool FIX, bool ONE>
__device__ void make_item(TileItem* t, uint32_t item, uint32_t NI, const TileGrid* __restrict__ grids, int R,
                          const TileGrid& grid1, const Rep* __restrict__ reps, const Rep& rep1,
                          const Frame* __restrict__ table, const CellBufs& g0, const CellBufs& g1) {
    const int lane = int(threadIdx.x & 31u);
    const uint32_t i = item / NI, at = item - i * NI;
    int r = 0;
    if (!ONE) {  // last replica whose first tile is at or before `at`
        int hi = R - 1;
        while (r < hi) {
            const int mid = (r + hi + 1) >> 1;
            if (grids[mid].first <= int(at)) r = mid; else hi = mid - 1;
        }
    }
    const TileGrid g = ONE ? grid1 : grids[r];
    const uint32_t hm = uint32_t(ONE ? rep1.hm : reps[r].hm);
    const uint32_t loc = at - uint32_t(g.first), ntx = uint32_t(g.ntx), nty = uint32_t(g.nty);
    const uint32_t row = loc / ntx, tx = loc - row * ntx, ty = (row + i) % nty;
    const int X0 = 2 * int(hm * tx / ntx), Y0 = 2 * int(hm * ty / nty);
    const int tw = 2 * int(hm * (tx + 1u) / ntx) - X0, th = 2 * int(hm * (ty + 1u) / nty) - Y0;
    const Frame* tab = table + size_t(r) * (kMaxChunk + 1);
    const Frame fn = tab[i + 1u];
    const ShiftDelta<FIX> sd(tab[i], fn);
    int xlo, xhi, ylo, yhi;
    if (lane < 4) {
        const int col = int(fn.perm >> (2 * lane)) & 3, px = col & 1, py = col >> 1;
        active_range(fn.perm, 0, tw, lane, xlo, xhi);
        active_range(fn.perm, 1, th, lane, ylo, yhi);
        const int hx = (xlo - px + 1) >> 1, hy = (ylo - py + 1) >> 1;
        const uint32_t nx = uint32_t(((xhi - px + 1) >> 1) - hx), ny = uint32_t(((yhi - py + 1) >> 1) - hy);
        t->pass[lane].col = col;
        t->pass[lane].hx = hx;
        t->pass[lane].hy = hy;
        t->pass[lane].nx = nx;
        t->pass[lane].ny = ny;
        t->pass[lane].cells = nx * ny;
        t->pass[lane].mul = small_mul(nx);
    } else if (lane == 4) {
        active_range(fn.perm, 0, tw, -1, xlo, xhi);
        active_range(fn.perm, 1, th, -1, ylo, yhi);
        t->lo0x = xlo;
        t->hi0x = xhi;
        t->lo0y = ylo;
        t->hi0y = yhi;
        const int hx0 = (xlo + min(sd.ox, 0)) >> 1, hx1 = (xhi + max(sd.ox, 0) + 1) >> 1;
        const int hy0 = (ylo + min(sd.oy, 0)) >> 1, hy1 = (yhi + max(sd.oy, 0) + 1) >> 1;
        t->lhx = hx0;
        t->lhy = hy0;
        t->lnx = uint32_t(hx1 - hx0);
        t->lcells = 4u * uint32_t(hx1 - hx0) * uint32_t(hy1 - hy0);
        t->lmul = small_mul(uint32_t(hx1 - hx0));
    } else if (lane == 6) {
        const Rep& rep = ONE ? rep1 : reps[r];
        t->from = (i & 1u) == 0u ? g0 : g1;
        t->to = (i & 1u) == 0u ? g1 : g0;
        t->stride = rep.stride32;
        t->coff = rep.coff;
        t->hh = uint32_t(rep.hh);
        t->hm = hm;
    } else if (lane == 5) {
        t->r = r;
        t->hx = (uint32_t(X0) / 2u + hm - 3u) % hm;
        t->hy = (uint32_t(Y0) / 2u + hm - 3u) % hm;
        t->tw = tw;
        t->th = th;
        t->twice = g.ntx == 1 || g.nty == 1;
        t->tx = int(tx);
        t->ty = int(ty);
        t->ntx = g.ntx;
        t->nty = g.nty;
        t->first = g.first;
        t->i = i;
        t->sweep = fn.sweep;
        t->perm = fn.perm;
        t->fx = sd.fx;
        t->fy = sd.fy;
        t->ox = sd.ox;
        t->oy = sd.oy;
        t->dx = sd.dx;
        t->dy = sd.dy;
    }
}

// Empty the first `rows` half-rows of every plane of a stage (nt threads).
template <class S>
__device__ __forceinline__ void clear_stage(const S& st, int rows, int tid, int nt) {
#pragma unroll
    for (int pl = 0; pl < 4; ++pl)
        for (int e = tid; e < rows * S::HP; e += nt) st.clear(pl * S::NP + e);
    if (tid < 6) st.pool_n[tid] = 0u;  // and the hard lists' counts
}

// Pass p of item `it` on local half-column hx and half-row hy: skipped unless
// the cell is hard (HARD) or not (!HARD).  The cell's final occupants go to
// the written generation if the tile owns it.
template <bool FIX, int NTC, bool HARD, class S>
__device__ __forceinline__ void visit_cell(const S& st, const TileRep<FIX>& rep, const TileItem& it, int col, int hx, int hy,
                                           uint32_t& att, uint32_t& acc) {
    const int px = col & 1, py = col >> 1;
    const uint32_t w = st.word[col * S::NP + hy * S::HP + hx];
    if (is_hard(w) != HARD) return;
    const uint32_t hm = it.hm;
    const uint32_t gx = wrap_half(it.hx + 1u + uint32_t(hx), hm, it.twice), gy = wrap_half(it.hy + 1u + uint32_t(hy), hm, it.twice);
    const bool own = uint32_t(2 * hx + px - kTileHalo) < uint32_t(it.tw) && uint32_t(2 * hy + py - kTileHalo) < uint32_t(it.th);
    const uint32_t cell = it.coff + uint32_t(col) * it.hh + gy * hm + gx;
    if (own) it.to.cnt[cell] = uint8_t(min(w & 15u, 4u));
    if ((w & 15u) == 0u) return;
    const uint32_t cl = (2u * gy + uint32_t(py)) * (2u * hm) + 2u * gx + uint32_t(px);
    P2<FIX>* pos = static_cast<P2<FIX>*>(it.to.pos);
    const uint32_t got = tile_cell<FIX, NTC, HARD, false, S>(st, rep, it.sweep, px, py, hx, hy, w, cl,
                                                      [&](int k, const P2<FIX>& q, int32_t id) {
                                                          if (own) {
                                                              pos[size_t(k) * it.stride + cell] = q;
                                                              it.to.pid[size_t(k) * it.stride + cell] = id;
                                                          }
                                                      });
    if (own) {
        att += uint32_t(rep.nt);
        acc += got;
    }
}

// The hard cells of pass p, for threads tid < the number of them (out of line:
// the registers of the rare paths stay out of the ordinary cells' loop).
// Returns trials and acceptances.
template <bool FIX, int NTC, class S>
__device__ __forceinline__ uint2 hard_cells(const S& st, const TileRep<FIX>& rep, const TileItem& it, int p, int tid, int nt) {
    const bool every = st.hard_n[4] != 0u;
    const int col = it.pass[p].col, hx0 = it.pass[p].hx, hy0 = it.pass[p].hy;
    const uint32_t nx = it.pass[p].nx, ny = it.pass[p].ny, n = every ? nx * ny : st.hard_n[col];
    uint32_t att = 0, acc = 0;
    for (uint32_t e = uint32_t(tid); e < n; e += uint32_t(nt)) {
        int hx, hy;
        if (every) {
            hy = int(e / nx);
            hx = hx0 + int(e - uint32_t(hy) * nx);
            hy += hy0;
        } else {
            const uint32_t h = st.hard[col * S::HARD + e];
            hy = int(h / uint32_t(S::HP));
            hx = int(h - uint32_t(hy * S::HP));
            // staged but beyond the cells this pass updates
            if (uint32_t(hx - hx0) >= nx || uint32_t(hy - hy0) >= ny) continue;
        }
        visit_cell<FIX, NTC, true, S>(st, rep, it, col, hx, hy, att, acc);
    }
    return make_uint2(att, acc);
}

}  // namespace

template <bool FIX, int NTC, bool ONE>
__global__ void __launch_bounds__(TileShape<FIX>::NT, 1)
k_sweep_tile(const Rep* __restrict__ reps, const TileGrid* __restrict__ grids, int R, const Rep rep1, const TileGrid grid1,
             const Frame* __restrict__ table, int nsweeps, uint32_t NI, CellBufs g0, CellBufs g1,
             unsigned long long* __restrict__ counters, int* __restrict__ err, uint32_t* sync, void* spill,
             uint32_t polls) {
    using Sh = TileShape<FIX>;
    using S = TileStage<FIX>;
    constexpr int NT = Sh::NT - 32;  // threads that sweep; the last warp looks ahead
    pdl_wait(table);
    extern __shared__ __align__(16) unsigned char s_raw[];
    const S st(s_raw, static_cast<PoolEntry<FIX>*>(spill) + size_t(blockIdx.x) * 2 * S::NC);
    __shared__ TileItem s_item[2];
    __shared__ uint32_t s_queue[NT / 32][64];
    const int tid = int(threadIdx.x);
    const uint32_t total = uint32_t(nsweeps) * NI;
    if (tid >= NT) {
        // The look-ahead warp: while the others sweep an item, it takes the
        // next ticket, works out that item and waits for its dependencies.
        const int lane = tid - NT;
        for (int buf = 0;; buf ^= 1) {
            TileItem& it = s_item[buf];
            uint32_t item = 0u;
            if (lane == 0) item = atomicAdd(sync, 1u);
            item = __shfl_sync(0xffffffffu, item, 0);
            bool go = item < total;
            if (go) {
                make_item<FIX, ONE>(&it, item, NI, grids, R, grid1, reps, rep1, table, g0, g1);
                __syncwarp();
                bool ready = lane >= 9 || it.i == 0u;
                const int nx = it.tx + lane % 3 - 1, ny = it.ty + lane / 3 - 1;
                const uint32_t* p = sync + 2 + it.first + wrap1(ny, it.nty) * it.ntx + wrap1(nx, it.ntx);
                for (uint32_t k = 0;; ++k) {
                    if (!ready) ready = ld_acquire(p) >= it.i;
                    if (__all_sync(0xffffffffu, ready)) break;
                    if ((k & 63u) == 63u) {
                        const bool gone = ld_acquire(sync + 1) != 0u;
                        if (k >= polls && lane == 0) {
                            atomicOr(err, kErrPersist);
                            atomicExch(sync + 1, 1u);
                        }
                        if (__any_sync(0xffffffffu, gone) || k >= polls) {
                            go = false;
                            break;
                        }
                    }
                    if (k > 8u) __nanosleep(20);
                }
            }
            if (lane == 0) it.go = go ? 1 : 0;
            __syncthreads();  // the item is ready, and the one before it done
            if (!go) break;
            asm volatile("bar.sync 2, %0;" ::"n"(Sh::NT) : "memory");  // it has reached kLookAhead
        }
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        return;
    }
    clear_stage(st, S::HR, tid, NT);
    auto sync_sweepers = [] { asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory"); };
    uint32_t att = 0, acc = 0;
    int cur_r = -1;
    bool over = false;
    for (int buf = 0;; buf ^= 1) {
        const TileItem& it = s_item[buf];
        __syncthreads();
        if (it.go == 0) break;
        const int r = ONE ? 0 : it.r;
        if (!ONE && r != cur_r) {  // the trial counts go to the replica of the items that made them
            if (cur_r >= 0) warp_count(att, acc, counters, cur_r);
            att = acc = 0;
            cur_r = r;
        }
        const TileRep<FIX> rep(ONE ? rep1 : reps[r]);


        // ---- move the old cells' disks into the new frame --------------------
        {
            const uint8_t* cnt_o = it.from.cnt;
            const P2<FIX>* pos_o = static_cast<const P2<FIX>*>(it.from.pos);
            const int32_t* pid_o = it.from.pid;
            const uint32_t stride = it.stride, coff = it.coff, hh = it.hh, hm = it.hm;
            const bool twice = it.twice != 0;
            // global half-column and half-row of local ones (at least -1), below
            // 2 hm with two tiles or more per axis (hm >= 12), else below 3 hm (hm >= 6)
            const uint32_t gx0 = it.hx + 1u, gy0 = it.hy + 1u;
            const int lhx = it.lhx, lhy = it.lhy;
            const uint32_t lnx = it.lnx, mul = it.lmul;
            const int32_t fx = it.fx, fy = it.fy;
            const int lo0x = it.lo0x, lo0y = it.lo0y;
            const uint32_t nx0 = uint32_t(it.hi0x - lo0x), ny0 = uint32_t(it.hi0y - lo0y);
            // entry e of the old cells: rows of lnx half-columns, the four colours of a half-row in turn
            auto coords = [&](uint32_t e, int& lx, int& ly) {
                const uint32_t row = small_div(e, mul), pl = row & 3u;
                const int hx = lhx + int(e - row * lnx), hy = lhy + int(row >> 2);
                lx = 2 * hx + int(pl & 1u);
                ly = 2 * hy + int(pl >> 1);
                return coff + pl * hh + wrap_half(gy0 + uint32_t(hy), hm, twice) * hm + wrap_half(gx0 + uint32_t(hx), hm, twice);
            };
            const int sx = fx >= 0 ? 1 : -1, sy = fy >= 0 ? 1 : -1;  // the way a disk can leave its cell (fixed form)
            auto put = [&](const P2<FIX>& q, int32_t id, int lx, int ly) {
                P2<FIX> p;
                if constexpr (FIX) {
                    const int32_t ux = q.x + fx, uy = q.y + fy;
                    const bool ox = uint32_t(ux) >= uint32_t(rep.W), oy = uint32_t(uy) >= uint32_t(rep.W);
                    p.x = ox ? ux - sx * rep.W : ux;
                    p.y = oy ? uy - sy * rep.W : uy;
                    lx += ox ? sx : 0;
                    ly += oy ? sy : 0;
                } else {
                    int cx, cy;
                    frame_change_fp64(it.dx, rep.w, rep.w_below, 1 << 20, lx + 8, q.x, cx, p.x);
                    frame_change_fp64(it.dy, rep.w, rep.w_below, 1 << 20, ly + 8, q.y, cy, p.y);
                    lx = cx - 8;
                    ly = cy - 8;
                }
                if (uint32_t(lx - lo0x) < nx0 && uint32_t(ly - lo0y) < ny0)
                    over |= !st.place(lx, ly, S::index(lx, ly), p, id);
            };
            // Slot 0 of every old cell first; a cell of more disks (4 to 5% of
            // those of 2.00 to 2.02 sigma at eta = 0.70 to 0.716, 9% at N = 256) is
            // queued, and the warp takes its further slots 32 cells at a time,
            // so that its lanes stay together.
            const uint32_t cells = it.lcells;
            const int lane = tid & 31;
            uint32_t* queue = s_queue[tid >> 5];
            int queued = 0;  // the same in every lane
            auto take = [&](int count) {
                if (lane < count) {
                    const uint32_t v = queue[lane], e = v >> 3;
                    const int n = int(v & 7u);
                    int lx, ly;
                    const uint32_t c = coords(e, lx, ly);
                    for (int k = 1; k < n; ++k)
                        put(ld_cell<true>(pos_o + size_t(k) * stride + c), ld_cell<true>(pid_o + size_t(k) * stride + c),
                            lx, ly);
                }
            };
            for (uint32_t b = uint32_t(tid & ~31); b < cells; b += 2u * NT) {
                uint32_t c[2];
                int lx[2], ly[2], n[2];
                P2<FIX> q0[2];
                int32_t id0[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint32_t e = b + uint32_t(lane) + uint32_t(h) * NT;
                    n[h] = 0;
                    if (e < cells) {
                        c[h] = coords(e, lx[h], ly[h]);
                        n[h] = occupancy<4, true>(cnt_o, c[h]);
                        q0[h] = ld_cell<true>(pos_o + c[h]);
                        id0[h] = ld_cell<true>(pid_o + c[h]);
                    }
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (n[h] > 0) put(q0[h], id0[h], lx[h], ly[h]);
                    const uint32_t more = __ballot_sync(0xffffffffu, n[h] > 1);
                    if (n[h] > 1)
                        queue[queued + __popc(more & ((1u << lane) - 1u))] =
                            ((b + uint32_t(lane) + uint32_t(h) * NT) << 3) | uint32_t(n[h]);
                    queued += __popc(more);
                    if (queued >= 32) {
                        __syncwarp();
                        take(32);
                        __syncwarp();
                        const uint32_t v = lane < queued - 32 ? queue[32 + lane] : 0u;
                        __syncwarp();
                        if (lane < queued - 32) queue[lane] = v;
                        queued -= 32;
                    }
                }
            }
            __syncwarp();
            take(queued);
        }
        sync_sweepers();
        // ---- tell the neighbours of crowded cells ------------------------------
        {
            const uint32_t marks = 8u * min(*st.pool_n, uint32_t(S::POOL));
            for (uint32_t x = uint32_t(tid); x < marks; x += NT) st.mark_entry(x >> 3, int(x & 7u));
        }
        sync_sweepers();

        // ---- the four colour passes ------------------------------------------
#pragma unroll 1
        for (int p = 0; p < 4; ++p) {
            if (p == kLookAhead) asm volatile("bar.arrive 2, %0;" ::"n"(Sh::NT) : "memory");
            const int col = it.pass[p].col, hx0 = it.pass[p].hx, hy0 = it.pass[p].hy;
            const uint32_t nx = it.pass[p].nx, cells = it.pass[p].cells, mul = it.pass[p].mul;
            const uint32_t nhard = st.hard_n[4] != 0u ? cells : st.hard_n[col];
            if (uint32_t(tid & ~31) < nhard) {
                const uint2 c = hard_cells<FIX, NTC, S>(st, rep, it, p, tid, NT);
                att += c.x;
                acc += c.y;
            }
            // the warps that had no hard cells begin with the others
            const uint32_t skip = min((nhard + 31u) & ~31u, uint32_t(NT));
            for (uint32_t e = uint32_t(tid) + (uint32_t(tid) < skip ? NT : 0u) - skip; e < cells; e += NT) {
                const uint32_t row = small_div(e, mul);
                visit_cell<FIX, NTC, false, S>(st, rep, it, col, hx0 + int(e - row * nx), hy0 + int(row), att, acc);
            }
            sync_sweepers();
        }
        if (tid == 0) red_release_add(sync + 2 + it.first + it.ty * it.ntx + it.tx, 1u);
        // the rows it placed disks in, and one more that marks of crowded cells reach
        clear_stage(st, min(it.th / 2 + kTileHalo + 1, S::HR), tid, NT);
    }
    if (over) atomicOr(err, 1);
    if (ONE) warp_count(att, acc, counters, 0);
    else if (cur_r >= 0) warp_count(att, acc, counters, cur_r);
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ---------------------------------------------------------------------------
// Small boxes: one block per replica keeps the whole box in shared memory
// over all sweeps of the launch, in two stages that a rebuild moves the disks
// between.  Cell (cx, cy) is local cell (cx + 2, cy + 2), so that parities
// agree; the ring of cells around the box holds copies of the cells of the
// opposite sides, filled after a rebuild and kept up by the thread that moves
// a disk of an edge cell, so that the passes are those of the tiles.  A
// launch boundary between phases costs 2 to 4 us, here a phase is one block
// barrier: what bounds a sweep is the latency of five dependent phases.  The
// draws of the next sweep's trials (generator, step, swap word: a third of a
// pass's chain) are therefore made by warps of their own while the others
// sweep.
// ---------------------------------------------------------------------------
template <bool FIX, int HB>
using BoxStage = Stage<FIX, HB, HB, HB <= 12 ? 64 : (FIX ? 256 : 160)>;

// Hard cells from registers (hard_cell_ahead), but for small fixed-point boxes
// (N <= 400), whose few crowded cells cost less as tile_cell takes them: per
// sweep at N = 256 4.6 us against 4.8; FP64 6.4 -> 6.0, boxes of N = 1024 7.8 -> 7.4
// fixed and 11.5 -> 11.0 FP64.
template <bool FIX, int HB>
constexpr bool kHardRegs = !FIX || HB > 12;

// A cell of the ring around the box, or its source, is (x, y): copy the
// occupants of entry `from` to entry `to`.
template <bool FIX, class S>
__device__ __forceinline__ void copy_cell(const S& st, int from, int to) {
    st.quad[to] = st.quad[from];
    if constexpr (FIX) {
        reinterpret_cast<uint16_t*>(st.low)[to] = reinterpret_cast<const uint16_t*>(st.low)[from];
    } else {
        st.p0[to] = st.p0[from];
        st.p0[S::NC + to] = st.p0[S::NC + from];
    }
    const uint32_t w = st.word[from];
    if ((w & 15u) > 2u)
        for (int k = 2; k < min(int(w & 15u), 4); ++k)
            if (((w >> (k == 2 ? 12 : 22)) & 0x3FFu) == kFar) *st.extra(w, to, k) = *st.extra(w, from, k);
}

template <bool FIX, int HB>
constexpr size_t box_smem() {
    return 2 * BoxStage<FIX, HB>::kBytes + size_t(2) * BoxStage<FIX, HB>::NC * (sizeof(P2<FIX>) + (kHardRegs<FIX, HB> ? 8 : 4));
}

template <bool FIX, int NTC, int HB, int NT, int ND>
__global__ void __launch_bounds__(NT + ND)
k_sweep_box(const Rep* __restrict__ reps, const Frame* __restrict__ table, int nsweeps, CellBufs g0, CellBufs g1,
            unsigned long long* __restrict__ counters, int* __restrict__ err, void* spill) {
    using S = BoxStage<FIX, HB>;
    pdl_wait(table);
    extern __shared__ __align__(16) unsigned char s_raw[];
    PoolEntry<FIX>* far = static_cast<PoolEntry<FIX>*>(spill) + size_t(blockIdx.x) * 4 * S::NC;
    const int tid = int(threadIdx.x), r = int(blockIdx.x);
    const Rep& full = reps[r];
    const TileRep<FIX> rep(full);
    const int m = full.m, hm = full.hm;
    const uint32_t stride = full.stride32, coff = full.coff, hh = uint32_t(full.hh), uhm = uint32_t(hm);
    const uint32_t hm_mul = full.hm_mul;
    const int hm_sh = full.hm_sh;
    const Frame* tab = table + size_t(r) * (kMaxChunk + 1);
    bool over = false;
    uint32_t att = 0, acc = 0;
    // entry e of the box's cells in colour-planar order: local coordinates
    auto local = [&](uint32_t e, int& lx, int& ly) {
        const uint32_t pl = uint32_t(e >= hh) + uint32_t(e >= 2u * hh) + uint32_t(e >= 3u * hh), q = e - pl * hh;
        const uint32_t row = div_by(q, hm_mul, hm_sh);
        lx = 2 * int(q - row * uhm) + int(pl & 1u) + 2;
        ly = 2 * int(row) + int(pl >> 1) + 2;
    };
    auto wrap_local = [m](int v) { return v < 2 ? v + m : (v >= m + 2 ? v - m : v); };
    // [2][NC] steps, then first and (kHardRegs) second swap words, by entry of the stage
    P2<FIX>* s_step = reinterpret_cast<P2<FIX>*>(s_raw + 2 * S::kBytes);
    uint32_t* s_swap = reinterpret_cast<uint32_t*>(s_step + 2 * S::NC);
    uint32_t* s_swap2 = s_swap + 2 * S::NC;
    // frame changes of two sweeps, read ahead
    struct Change {
        double dx, dy;
        int32_t fx, fy;
        uint32_t sweep, perm;
    };
    __shared__ Change s_change[2];
    auto read_change = [&](int i) {
        const Frame fn = tab[i + 1];
        const ShiftDelta<FIX> sd(tab[i], fn);
        s_change[i & 1] = Change{sd.dx, sd.dy, sd.fx, sd.fy, fn.sweep, fn.perm};
    };
    if (tid >= NT) {  // the draws of sweep i and the frame change of sweep i + 1 are ready at barrier i
        if (tid == NT) read_change(0);
        __syncthreads();
        for (int i = 0; i < nsweeps; ++i) {
            const uint32_t sweep = s_change[i & 1].sweep;
            if (tid == NT && i + 1 < nsweeps) read_change(i + 1);
            for (uint32_t e = uint32_t(tid - NT); e < 4u * hh; e += ND) {
                int lx, ly;
                local(e, lx, ly);
                const uint32_t cl = uint32_t(ly - 2) * uint32_t(m) + uint32_t(lx - 2);
                const int at = (i & 1) * S::NC + S::index(lx, ly);
                const uint4 u = philox(sweep, 0u, cl, kTagTrial, rep.key0, rep.key1);
                s_step[at] = trial_step<FIX>(rep, u);
                const uint4 v = FIX ? make_uint4(u.z, u.w, 0u, 0u) : philox(sweep, 0u, cl, kTagShuffle, rep.key0, rep.key1);
                s_swap[at] = v.x;
                if constexpr (kHardRegs<FIX, HB>) s_swap2[at] = v.y;
            }
            __syncthreads();
        }
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        return;
    }
    auto sync_sweepers = [] { asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory"); };
    {
        const S st(s_raw, far);
        clear_stage(st, hm + 2, tid, NT);
        sync_sweepers();
        for (uint32_t e = uint32_t(tid); e < 4u * hh; e += NT) {
            int lx, ly;
            local(e, lx, ly);
            const uint32_t c = coff + e;
            const int n = min(int(g0.cnt[c]), 4);
            for (int k = 0; k < n; ++k)
                st.place(lx, ly, S::index(lx, ly), static_cast<const P2<FIX>*>(g0.pos)[size_t(k) * stride + c],
                         g0.pid[size_t(k) * stride + c]);
        }
    }
    __syncthreads();
    for (int i = 0; i < nsweeps; ++i) {
        const S old(s_raw + (i & 1 ? S::kBytes : 0), far + (i & 1 ? 2 * S::NC : 0));
        const S st(s_raw + (i & 1 ? 0 : S::kBytes), far + (i & 1 ? 0 : 2 * S::NC));
        const Change sd = s_change[i & 1];
        clear_stage(st, hm + 2, tid, NT);
        sync_sweepers();
        // ---- move every disk into the new frame -------------------------------
        for (uint32_t e = uint32_t(tid); e < 4u * hh; e += NT) {
            int lx, ly;
            local(e, lx, ly);
            const int c = S::index(lx, ly);
            const uint32_t w = old.word[c];
            const int n = min(int(w & 15u), 4);
            for (int k = 0; k < n; ++k) {
                P2<FIX> q, p;
                int32_t id;
                if (k < 2) {
                    q = old.get(c, k);
                    id = reinterpret_cast<const int32_t*>(old.id)[2 * c + k];
                } else {
                    q = old.extra(w, c, k)->p;
                    id = old.extra(w, c, k)->id;
                }
                int x, y;
                if constexpr (FIX) {
                    frame_change_fixed(sd.fx, rep.W, 1 << 20, lx, q.x, x, p.x);
                    frame_change_fixed(sd.fy, rep.W, 1 << 20, ly, q.y, y, p.y);
                } else {
                    frame_change_fp64(sd.dx, rep.w, rep.w_below, 1 << 20, lx, q.x, x, p.x);
                    frame_change_fp64(sd.dy, rep.w, rep.w_below, 1 << 20, ly, q.y, y, p.y);
                }
                x = wrap_local(x);
                y = wrap_local(y);
                over |= !st.place(x, y, S::index(x, y), p, id);
            }
        }
        sync_sweepers();
        // ---- the neighbours of crowded cells, and the hard cells ---------------
        const uint32_t pooled = *st.pool_n;
        if (pooled != 0u) {
            for (uint32_t t = uint32_t(tid); t < 8u * min(pooled, uint32_t(S::POOL)); t += NT) {
                const int32_t at = st.pool[t >> 3].cell;
                if (at < 0) continue;
                const int d = int(t & 7u), k = 7 - d, j = k + (k >= 4 ? 1 : 0);
                const int x = wrap_local((at & 0xFFFF) + j % 3 - 1), y = wrap_local((at >> 16) + j / 3 - 1);
                const uint32_t was = atomicOr(&st.word[S::index(x, y)], 1u << (kCrowdShift + d)), n = was & 15u;
                if (n >= 1u && n <= 2u && ((was >> kCrowdShift) & 0xFFu) == 0u) st.list_hard(x, y);
                if (d == 0) st.list_hard(at & 0xFFFF, at >> 16);
            }
            // a pool that overflowed: every cell looks at its neighbours itself
            if (pooled > uint32_t(S::POOL)) {
                sync_sweepers();
                for (uint32_t e = uint32_t(tid); e < 4u * hh; e += NT) {
                    int lx, ly;
                    local(e, lx, ly);
                    uint32_t bits = 0u;
                    for (int d = 0; d < 8; ++d) {
                        const int j = d + (d >= 4 ? 1 : 0);
                        const uint32_t w = st.word[S::index(wrap_local(lx + j % 3 - 1), wrap_local(ly + j / 3 - 1))];
                        if ((w & 15u) > 2u) bits |= 1u << (kCrowdShift + d);
                    }
                    if (bits) atomicOr(&st.word[S::index(lx, ly)], bits);
                }
            }
            sync_sweepers();
        }
        // ---- the ring around the box -------------------------------------------
        for (int t = tid; t < 4 * (m + 1); t += NT) {
            const int side = t / (m + 1), j = t - side * (m + 1) + 1;  // 1 .. m + 1
            const int x = side == 0 ? j : (side == 1 ? m + 2 : (side == 2 ? j + 1 : 1));
            const int y = side == 0 ? 1 : (side == 1 ? j : (side == 2 ? m + 2 : j + 1));
            const int from = S::index(wrap_local(x), wrap_local(y)), to = S::index(x, y);
            st.word[to] = st.word[from];
            copy_cell<FIX, S>(st, from, to);
        }
        __syncthreads();  // and this sweep's draws are made
        // ---- the four colour passes --------------------------------------------
        const bool every = st.hard_n[4] != 0u;
#pragma unroll 1
        for (int p = 0; p < 4; ++p) {
            const int col = int(sd.perm >> (2 * p)) & 3, px = col & 1, py = col >> 1;
            auto visit = [&](auto hard, int hx, int hy) {
                const int e = col * S::NP + hy * S::HP + hx;
                const uint32_t w = st.word[e];
                if (is_hard(w) != hard.value || (w & 15u) == 0u) return;
                const uint32_t cx = uint32_t(2 * hx + px - 2), cy = uint32_t(2 * hy + py - 2);
                // an edge cell's copies in the ring
                const int gx = cx == 0u ? m + 2 : (cx == uint32_t(m - 1) ? 1 : 0);
                const int gy = cy == 0u ? m + 2 : (cy == uint32_t(m - 1) ? 1 : 0);
                const int lx = int(cx) + 2, ly = int(cy) + 2;
                const int at = (i & 1) * S::NC + e;
                const Drawn<FIX> pre{s_step[at], s_swap[at], kHardRegs<FIX, HB> ? s_swap2[at] : 0u};
                auto emit = [&](int k, const P2<FIX>& q, int32_t id) {
                    // in id order, ids and positions together
                    if (k < 2) {
                        const typename S::Stored v = st.stored(q);
                        st.set(e, k, v);
                        reinterpret_cast<int32_t*>(st.id)[2 * e + k] = id;
                        if (gx) st.set(S::index(gx, ly), k, v);
                        if (gy) st.set(S::index(lx, gy), k, v);
                        if (gx && gy) st.set(S::index(gx, gy), k, v);
                    } else {
                        PoolEntry<FIX>* x = st.extra(w, e, k);
                        x->p = q;
                        x->id = id;
                        if (x >= st.spill && x < st.spill + 2 * S::NC) {  // the copies share a pool entry, not the spill area's
                            if (gx) st.extra(w, S::index(gx, ly), k)->p = q;
                            if (gy) st.extra(w, S::index(lx, gy), k)->p = q;
                            if (gx && gy) st.extra(w, S::index(gx, gy), k)->p = q;
                        }
                    }
                };
                const uint32_t cl = cy * uint32_t(m) + cx;
                uint32_t got;
                if constexpr (hard.value && kHardRegs<FIX, HB>)
                    got = hard_cell_ahead<FIX, NTC, S>(st, rep, sd.sweep, px, py, hx, hy, w, cl, emit, pre);
                else
                    got = tile_cell<FIX, NTC, hard.value, true, S>(st, rep, sd.sweep, px, py, hx, hy, w, cl, emit, pre);
                att += uint32_t(rep.nt);
                acc += got;
            };
            const uint32_t nhard = every ? hh : st.hard_n[col];
            for (uint32_t h = uint32_t(tid); h < nhard; h += NT) {
                if (every) {
                    const uint32_t row = div_by(h, hm_mul, hm_sh);
                    visit(std::true_type{}, int(h - row * uhm) + 1, int(row) + 1);
                } else {
                    const uint32_t v = st.hard[col * S::HARD + h];
                    visit(std::true_type{}, int(v % uint32_t(S::HP)), int(v / uint32_t(S::HP)));
                }
            }
            // the warps that had no hard cells begin with the others
            const uint32_t skip = min((nhard + 31u) & ~31u, uint32_t(NT));
            for (uint32_t h = uint32_t(tid) + (uint32_t(tid) < skip ? NT : 0u) - skip; h < hh; h += NT) {
                const uint32_t row = div_by(h, hm_mul, hm_sh);
                visit(std::false_type{}, int(h - row * uhm) + 1, int(row) + 1);
            }
            sync_sweepers();
        }
    }
    // ---- the final state into the generation of the last sweep ------------------
    {
        const S st(s_raw + (nsweeps & 1 ? S::kBytes : 0), far + (nsweeps & 1 ? 2 * S::NC : 0));
        const CellBufs out = nsweeps & 1 ? g1 : g0;
        for (uint32_t e = uint32_t(tid); e < 4u * hh; e += NT) {
            int lx, ly;
            local(e, lx, ly);
            const int c = S::index(lx, ly);
            const uint32_t w = st.word[c];
            const int n = min(int(w & 15u), 4);
            out.cnt[coff + e] = uint8_t(n);
            for (int k = 0; k < n; ++k) {
                const size_t to = size_t(k) * stride + coff + e;
                static_cast<P2<FIX>*>(out.pos)[to] = k < 2 ? st.get(c, k) : st.extra(w, c, k)->p;
                out.pid[to] = k < 2 ? reinterpret_cast<const int32_t*>(st.id)[2 * c + k] : st.extra(w, c, k)->id;
            }
        }
    }
    if (over) atomicOr(err, 1);
    warp_count(att, acc, counters, r);
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Half-cells per axis staged (hm + 2 used), sweeping threads and drawing threads.
// The large shape holds N = 1024 (m = 32) in 130 KB (FP64 228 KB) of shared memory: one block
// per SM, so as many threads as its passes have cells, twice.
struct SmallBox { static constexpr int HB = 12, NT = 256, ND = 128; };
struct LargeBox { static constexpr int HB = 18, NT = 512, ND = 256; };

namespace {

template <bool FIX, int NTC>
cudaError_t tile_allow() {
    static OncePerDevice once;
    return allow_smem(once, TileStage<FIX>::kBytes, k_sweep_tile<FIX, NTC, true>, k_sweep_tile<FIX, NTC, false>);
}

template <bool FIX, int NTC>
auto tile_kernel(bool one) {
    return one ? k_sweep_tile<FIX, NTC, true> : k_sweep_tile<FIX, NTC, false>;
}

template <bool FIX, int NTC>
cudaError_t tile_blocks_t(bool one, int* blocks) {
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = tile_allow<FIX, NTC>();
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, tile_kernel<FIX, NTC>(one), TileShape<FIX>::NT,
                                                          TileStage<FIX>::kBytes);
    *blocks = sms * per_sm;
    return e;
}

template <bool FIX, int NTC>
cudaError_t tile_t(const LaunchCfg& c, const TileCfg& t, const Frame* table, int nsweeps, CellBufs a, CellBufs b,
                   unsigned long long* counters, int* err) {
    const int blocks = int(std::min<int64_t>(t.blocks, t.total));
    const cudaError_t e = tile_allow<FIX, NTC>();
    if (e != cudaSuccess) return e;
    return launch_k(tile_kernel<FIX, NTC>(c.R == 1), dim3(blocks), dim3(TileShape<FIX>::NT), TileStage<FIX>::kBytes,
                    c.stream, c.reps, (const TileGrid*)t.grids, c.R, c.R == 1 ? *c.rep0 : Rep{}, t.grid0, table, nsweeps,
                    uint32_t(t.total), a, b, counters, err, t.sync, t.spill, t.stall ? 1u << 12 : kTilePolls);
}

template <class B, bool FIX, int NTC>
cudaError_t box_t(const LaunchCfg& c, void* spill, const Frame* table, int nsweeps, CellBufs a, CellBufs b,
                  unsigned long long* counters, int* err) {
    constexpr size_t smem = box_smem<FIX, B::HB>();
    constexpr auto kernel = k_sweep_box<FIX, NTC, B::HB, B::NT, B::ND>;
    static OncePerDevice once;
    const cudaError_t e = allow_smem(once, smem, kernel);
    if (e != cudaSuccess) return e;
    return launch_k(kernel, dim3(c.R), dim3(B::NT + B::ND), smem, c.stream, c.reps, table, nsweeps, a, b, counters, err, spill);
}

template <class B>
cudaError_t boxes(const LaunchCfg& c, void* spill, const Frame* table, int nsweeps, CellBufs a, CellBufs b,
                  unsigned long long* counters, int* err) {
    if (c.fixed)
        return c.ntc == 1 ? box_t<B, true, 1>(c, spill, table, nsweeps, a, b, counters, err)
                          : box_t<B, true, 0>(c, spill, table, nsweeps, a, b, counters, err);
    return c.ntc == 1 ? box_t<B, false, 1>(c, spill, table, nsweeps, a, b, counters, err)
                      : box_t<B, false, 0>(c, spill, table, nsweeps, a, b, counters, err);
}

template <class B>
size_t spill_of(bool fixed) {
    return fixed ? size_t(4) * BoxStage<true, B::HB>::NC * sizeof(PoolEntry<true>)
                 : size_t(4) * BoxStage<false, B::HB>::NC * sizeof(PoolEntry<false>);
}

}  // namespace

// One replica beyond the small box: a block's latency against that of several
// tiles.  Fixed form, per sweep as a box and as tiles: N = 600 9.6 and 11.3 us,
// 700 6.1 and 6.6, 900 7.3 and 7.8, 1024 7.4 and 7.6.  FP64: 500 12.8 and 15.0, 600 14.9
// and 16.2, 800 15.9 and 16.4, 900 10.6 and 10.6, 1024 11.0 and 10.3.  Several replicas
// share the GPU, and a block each is less work than four tiles each: 32 of
// N = 1024 7.7 and 9.8 us (FP64 11.5 and 13.5), 152 of them 7.7 and 35.6, 700 37 and 170.
int box_max_hm(bool fixed, int R) { return fixed || R > 1 ? LargeBox::HB - 2 : LargeBox::HB - 4; }

size_t box_spill(bool fixed, int hm) { return hm <= SmallBox::HB - 2 ? spill_of<SmallBox>(fixed) : spill_of<LargeBox>(fixed); }

cudaError_t launch_sweeps_box(const LaunchCfg& c, int hm, void* spill, const Frame* table, int nsweeps, CellBufs from,
                              CellBufs to, unsigned long long* counters, int* err) {
    if (nsweeps < 1 || nsweeps > kMaxChunk || c.cap != 4 || hm > LargeBox::HB - 2) return cudaErrorInvalidValue;
    return hm <= SmallBox::HB - 2 ? boxes<SmallBox>(c, spill, table, nsweeps, from, to, counters, err)
                                  : boxes<LargeBox>(c, spill, table, nsweeps, from, to, counters, err);
}

TileLimits tile_limits(bool fixed) {
    using F = TileShape<true>;
    using D = TileShape<false>;
    return fixed ? TileLimits{2 * F::HP - 2 * kTileHalo, 2 * F::HR - 2 * kTileHalo,
                              size_t(2) * TileStage<true>::NC * sizeof(PoolEntry<true>)}
                 : TileLimits{2 * D::HP - 2 * kTileHalo, 2 * D::HR - 2 * kTileHalo,
                              size_t(2) * TileStage<false>::NC * sizeof(PoolEntry<false>)};
}

cudaError_t tile_blocks(const LaunchCfg& c, int* blocks) {
    if (c.fixed) return c.ntc == 1 ? tile_blocks_t<true, 1>(c.R == 1, blocks) : tile_blocks_t<true, 0>(c.R == 1, blocks);
    return c.ntc == 1 ? tile_blocks_t<false, 1>(c.R == 1, blocks) : tile_blocks_t<false, 0>(c.R == 1, blocks);
}

size_t tile_sync_words(int64_t total) { return size_t(2 + total); }

cudaError_t launch_sweeps_tile(const LaunchCfg& c, const TileCfg& t, const Frame* table, int nsweeps, CellBufs from,
                               CellBufs to, unsigned long long* counters, int* err) {
    if (nsweeps < 1 || nsweeps > kMaxChunk || c.cap != 4) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemsetAsync(t.sync, 0, tile_sync_words(t.total) * sizeof(uint32_t), c.stream);
    if (e == cudaSuccess && t.stall) e = cudaMemsetAsync(t.sync, 1, 1, c.stream);  // the next ticket is 1
    if (e != cudaSuccess) return e;
    if (c.fixed)
        return c.ntc == 1 ? tile_t<true, 1>(c, t, table, nsweeps, from, to, counters, err)
                          : tile_t<true, 0>(c, t, table, nsweeps, from, to, counters, err);
    return c.ntc == 1 ? tile_t<false, 1>(c, t, table, nsweeps, from, to, counters, err)
                      : tile_t<false, 0>(c, t, table, nsweeps, from, to, counters, err);
}

}  // namespace hd
