// Several time steps of a small channel in one launch (GB300, sm_103a).
//
// A channel of some ten thousand nodes is a megabyte: its steps are bound by
// the latency of one sweep (read the neighbours from L2, collide, write, end
// the launch: 2.6 to 3 us), not by any bandwidth.  Here each block takes `w` columns of the
// channel over its whole height, plus a halo of one column per step on either
// side, into shared memory, advances them `nsteps` steps with one block
// barrier each, and writes its own columns back: the global round trip and the
// launch are paid once per `nsteps` steps, the halo columns are computed by
// two blocks.  The blocks of a launch need nothing from one another.  A channel
// that fits one block (TilePlan::whole) needs no halo and takes any number of
// steps per launch.
//
// The arithmetic per node is that of sweep.cu, bit for bit: the stored format
// is kept in shared memory between the steps.
//
// Layout: [9][columns][ny] per copy, columns `cs` (odd, at least ny) elements
// apart, so that both the row-wise global copy and the column-wise steps are
// free of bank conflicts; two copies, alternating from step to step.  Threads
// run along y, then along x, `cpp` whole columns per pass, so a pressure
// channel's end columns sit in few warps and each thread stays in one row.
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "clb_device.cuh"
#include "clb_internal.h"

namespace clb {
namespace {

constexpr int kTileThreads = 512;  // threads that step columns
constexpr int kEndThreads = 128;   // and, at most, that step the end columns of a pressure channel

// Elements of one population plane of a block's copy: a constant, so that
// every shared-memory access is one base register and an immediate offset.
// The small one for blocks of few nodes, the large one for what shared memory
// holds.
constexpr int kPlaneSmall = 1024, kPlaneBytes = 12800;
size_t plane_of(size_t elem, bool big) { return big ? kPlaneBytes / elem : kPlaneSmall; }

// Shared memory of one block: two copies of its columns and the centreline
// densities (two steps x two rows per column).
size_t tile_smem(bool big, int cols, size_t elem, size_t relem) {
    return 2 * 9 * plane_of(elem, big) * elem + 4 * (size_t)cols * relem;
}

template <class T, int MODE, bool PACK, bool BIG>
__global__ void __launch_bounds__(kTileThreads + kEndThreads, 1)
    tile_kernel(const SweepArgs a, const TilePlan p, int nsteps) {
    using R = typename Codec<T>::R;
    constexpr bool kShift = (MODE == MODE_PRESSURE) && !std::is_same<T, double>::value;  // R(x) != 0
    extern __shared__ __align__(16) unsigned char smem[];
    const KC<R>& c = kc<R>(a);
    const int nx = a.nx, ny = a.ny, cs = p.cs;
    // own columns [xa, xb), held columns [lo, hi); an end at which the tile
    // holds the channel's own end column (or a whole period) does not shrink
    const int halo = p.whole ? 0 : nsteps;
    const int xa = (int)((long long)blockIdx.x * nx / gridDim.x), xb = (int)((blockIdx.x + 1LL) * nx / gridDim.x);
    const int lo = MODE == MODE_PRESSURE ? max(0, xa - halo) : xa - halo;
    const int hi = MODE == MODE_PRESSURE ? min(nx, xb + halo) : xb + halo;
    const bool fixl = p.whole || (MODE == MODE_PRESSURE && lo == 0);
    const bool fixr = p.whole || (MODE == MODE_PRESSURE && hi == nx);
    const int cols = hi - lo;
    constexpr int n = BIG ? kPlaneBytes / (int)sizeof(T) : kPlaneSmall;
    T* const s = reinterpret_cast<T*>(smem);
    int cur = 0;  // element offset of the current copy (0 or 9 n)
    R* rcs = reinterpret_cast<R*>(smem + 2 * 9 * n * sizeof(T));  // [step parity][row][cols]
    const bool centre_kn = MODE == MODE_PRESSURE && a.kn_mode == 1;

    // The next launch may start now; nothing global is touched before the
    // previous one has ended.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");

    // No __restrict__ on the input: the previous launch may still write it when this
    // one starts, so it must not be read through the read-only path.
    const T* fin = static_cast<const T*>(a.fin);
    T* __restrict__ fout = static_cast<T*>(a.fout);
    // Global <-> shared copies: a thread moves four columns of a row at once
    // (16 bytes of FP32), a warp 8 such vectors of 4 rows, which keeps both the
    // global segments whole and, with the odd column stride, the shared
    // accesses free of bank conflicts.  The 9 ny rows are spread over the
    // warps, kBatch of them in flight per thread.
    struct alignas(4 * sizeof(T)) Quad {
        T v[4];
    };
    constexpr int kBatch = sizeof(T) == 8 ? 4 : 9;
    const int rows = 9 * ny, rstep = blockDim.x >> 3, di = rstep / ny, dy = rstep - di * ny;
    struct Row {  // row = i ny + y
        int row, i, y;
    };
    auto next_row = [&](Row& q) {
        q.row += rstep;
        q.i += di;
        q.y += dy;
        if (q.y >= ny) {
            q.y -= ny;
            ++q.i;
        }
    };
    Row first{(int)threadIdx.x >> 3, 0, 0};
    first.i = first.row / ny;
    first.y = first.row - first.i * ny;
    const int xv = 4 * (threadIdx.x & 7);
    for (int x = (lo & ~3) + xv; x < hi; x += 32) {
        // the columns' places in the row (periodic: wrapped; a halo may be
        // several periods wide), one vector unless it crosses an end
        const bool vec = MODE == MODE_PRESSURE ? true : x >= 0 && x + 4 <= nx;
        int g[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            g[k] = x + k;
            if (MODE == MODE_PERIODIC && !vec) {
                while (g[k] < 0) g[k] += nx;
                while (g[k] >= nx) g[k] -= nx;
            }
        }
        const T* src = fin + a.xoff;
        for (Row q = first; q.row < rows;) {
            Quad v[kBatch];
            int to[kBatch];
            unsigned live = 0;  // bit b: row b exists
#pragma unroll
            for (int b = 0; b < kBatch; ++b) {
                if (q.row < rows) {
                    const T* r = src + q.i * a.plane + (long long)q.y * a.pitch;
                    to[b] = q.i * n + (x - lo) * cs + q.y;
                    live |= 1u << b;
                    if (vec)
                        v[b] = *reinterpret_cast<const Quad*>(r + x);
                    else
#pragma unroll
                        for (int k = 0; k < 4; ++k) v[b].v[k] = r[g[k]];
                    next_row(q);
                }
            }
#pragma unroll
            for (int b = 0; b < kBatch; ++b)
                if (live >> b & 1)
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (x + k >= lo && x + k < hi) s[to[b] + k * cs] = v[b].v[k];
        }
    }
    if (centre_kn) {
        const R* rc0 = static_cast<const R*>(a.rc_in);
        for (int e = threadIdx.x; e < 2 * cols; e += blockDim.x) {
            const int row = e / cols, x = e - row * cols;
            rcs[e] = rc0[row * a.rc_stride + lo + x];
        }
    }
    __syncthreads();

    // The end columns of a pressure channel take two gathers and a rebuild
    // before their collision: threads of their own step them beside the others
    // (in the warps of the other columns that chain would double the step).
    const bool end_thread = (int)threadIdx.x >= p.main;
    // this thread's row, and its first column (PACK: pair of columns) of every pass
    const int x0 = threadIdx.x / ny, y = threadIdx.x - x0 * ny;
    const bool mine = x0 < p.cpp && !end_thread;
    const bool bottom = y == 0, top = y == ny - 1;
    // where the populations that may come off a wall are read, from the node
    // (a wall) or from the node, its left or its right neighbour
    const int o2 = bottom ? 4 * n : 2 * n - 1, o5 = bottom ? 7 * n : 5 * n - 1, o6 = bottom ? 8 * n : 6 * n - 1;
    const int o4 = top ? 2 * n : 4 * n + 1, o7 = top ? 5 * n : 7 * n + 1, o8 = top ? 6 * n : 8 * n + 1;
    const R sh_b = bottom ? R(0) : c.shd, sh_t = top ? R(0) : c.shd;

    auto dec = [&](int e) { return Codec<T>::dec(s[e], c.isc); };
    // pre-collision populations of column x (Eq. 5, walls Eq. 20)
    auto gather = [&](int x, R (&f)[9]) {
        const int m = cur + x * cs + y;
        // the columns to the left and right (a whole periodic channel wraps)
        int l = m - cs, r = m + cs;
        if (MODE == MODE_PERIODIC && p.whole) {
            if (x == 0) l = m + (cols - 1) * cs;
            if (x == cols - 1) r = m - (cols - 1) * cs;
        }
        f[0] = dec(m);
        f[1] = dec(l + n);
        f[3] = dec(r + 3 * n);
        f[2] = dec(m + o2);
        f[5] = dec((bottom ? m : l) + o5);
        f[6] = dec((bottom ? m : r) + o6);
        f[4] = dec(m + o4);
        f[7] = dec((top ? m : r) + o7);
        f[8] = dec((top ? m : l) + o8);
        if (kShift) {
            f[1] += c.sha;
            f[3] -= c.sha;
            f[5] += sh_b;
            f[6] -= sh_b;
            f[7] -= sh_t;
            f[8] += sh_t;
        }
        if (bottom) {
            R s8 = dec(l + 8 * n), s7 = dec(r + 7 * n);
            if (kShift) {
                s8 += c.shd;
                s7 -= c.shd;
            }
            f[5] = ln::fma(c.r, f[5], ln::mul(c.rc, s8));
            f[6] = ln::fma(c.r, f[6], ln::mul(c.rc, s7));
        }
        if (top) {
            R s6 = dec(r + 6 * n), s5 = dec(l + 5 * n);
            if (kShift) {
                s6 -= c.shd;
                s5 += c.shd;
            }
            f[7] = ln::fma(c.r, f[7], ln::mul(c.rc, s6));
            f[8] = ln::fma(c.r, f[8], ln::mul(c.rc, s5));
        }
    };
    auto ref_of = [&](int x) {
        if (std::is_same<T, double>::value) return R(0);
        return MODE == MODE_PRESSURE ? ln::fma(c.slope, R(lo + x), c.ref0) : c.ref0;
    };
    // the density that sets the column's Knudsen number, and this step's own
    // at the centre rows
    auto centre_in = [&](int x, int par) {
        const R* rc0 = rcs + par * 2 * cols;
        return a.yc0 == a.yc1 ? rc0[x] : R(0.5) * (rc0[x] + rc0[cols + x]);
    };
    auto centre_out = [&](int x, int row, int par, R ref, const R (&f)[9]) {
        if (row != a.yc0 && row != a.yc1) return;
        R dr = f[0];
#pragma unroll
        for (int i = 1; i < 9; ++i) dr += f[i];
        rcs[(par ^ 1) * 2 * cols + (row == a.yc0 ? 0 : cols) + x] = ref + dr;
    };
    auto put = [&](int x, int row, const R (&f)[9]) {
        const int m = (cur ^ (9 * n)) + x * cs + row;
#pragma unroll
        for (int i = 0; i < 9; ++i) s[m + i * n] = Codec<T>::enc(f[i], c.sc);
    };
    auto finish = [&](int x, int row, int par, R (&f)[9]) {
        const R ref = ref_of(x);
        R rk = R(0);
        if (centre_kn) {
            rk = centre_in(x, par);
            centre_out(x, row, par, ref, f);
        }
        if constexpr (std::is_same<T, double>::value)
            collide64<MODE>(f, c, a.kp, centre_kn ? &rk : nullptr);
        else
            collide<R, MODE>(f, ref, c, centre_kn ? &rk : nullptr);
        put(x, row, f);
    };
    constexpr bool kEnds = MODE == MODE_PRESSURE;
    // Item e of the end columns: two lanes per node.  Lane 0 gathers the first
    // interior neighbour and keeps its non-equilibrium part, lane 1 the second,
    // for the velocity, and then the imposed equilibrium (rebuild_nodes, with
    // its two halves side by side).  Whole warps call it; true in lane 0 of a node
    // of this tile.
    auto rebuild_end = [&](int e, int& xe, int& row, R (&f)[9]) {
        constexpr unsigned kAll = 0xffffffffu;
        __syncwarp();
        const int half = e & 1, q = e >> 1;
        const bool right = q >= ny;
        const bool on = e < 4 * ny && (right ? fixr : fixl);
        row = !on ? 0 : right ? q - ny : q;
        const int dir = right ? -1 : 1;
        xe = right ? cols - 1 : 0;
        const int xs = on ? xe + (half ? 2 : 1) * dir : min(1, cols - 1);
        const int m = cur + xs * cs + row;
        R v[9];
        if (on)
            gather_node_at<R>(c, row_kind(row, ny), [&](int i, int dy, int dx) { return dec(m + i * n + dx * cs + dy); }, v);
        else
#pragma unroll
            for (int i = 0; i < 9; ++i) v[i] = R(1);
        if constexpr (std::is_same<T, double>::value) {
            Macro64 mac;
            const bool fine = macro64(v, mac);
            const double rho_b = right ? c.drho_out : c.drho_in;
            // (every lane takes part in every shuffle: none behind a condition)
            const int fine2 = __shfl_xor_sync(kAll, (int)fine, 1);
            const bool both = fine && fine2 && end_fine64(mac, rho_b);  // of lane 0
            const pr::P u2x{__shfl_xor_sync(kAll, mac.ux.h, 1), __shfl_xor_sync(kAll, mac.ux.l, 1)};
            const pr::P u2y{__shfl_xor_sync(kAll, mac.uy.h, 1), __shfl_xor_sync(kAll, mac.uy.l, 1)};
            double n2[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) n2[i] = __shfl_xor_sync(kAll, v[i], 1);
            if (on && !half) {
                if (both) {
                    end_column64(v, mac, u2x, u2y, rho_b, f);
                } else {
                    double n1[9], t[9];
#pragma unroll
                    for (int i = 0; i < 9; ++i) n1[i] = v[i];
                    rebuild_plain64(&c, lo + xe, !right, n1, n2, t);
#pragma unroll
                    for (int i = 0; i < 9; ++i) f[i] = t[i];
                }
            }
            return on && !half;
        } else {
            R dr, jx, jy;
            macro_dev(v, dr, jx, jy);
            const R rho = c.ref0 + c.slope * R(lo + xs) + dr;
            const R ux = jx / rho, uy = jy / rho;
            const R vx = __shfl_xor_sync(kAll, ux, 1), vy = __shfl_xor_sync(kAll, uy, 1);
            const R drb = right ? c.drho_out : c.drho_in;
            const R rb = c.ref0 + c.slope * R(lo + xe) + drb;
            R eq[9];
            feq_dev(half ? drb : dr, half ? rb : rho, half ? R(2) * vx - ux : ux, half ? R(2) * vy - uy : uy, eq);
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const R eb = __shfl_xor_sync(kAll, eq[i], 1);
                f[i] = eb + (v[i] - eq[i]);
            }
            return on && !half;
        }
    };

    const int end_items = (4 * ny + 31) / 32 * 32;  // whole warps
    for (int t = 0; t < nsteps; ++t) {
        // columns whose neighbours are still exact after t steps
        const int al = fixl ? (kEnds ? 1 : 0) : t + 1, ar = fixr ? cols - (kEnds ? 1 : 0) : cols - t - 1;
        const int par = t & 1;
        if constexpr (PACK) {
            if (kEnds && end_thread && (fixl || fixr))
                for (int e = threadIdx.x - p.main; e < end_items; e += blockDim.x - p.main) {
                    int x, row;
                    R f[9];
                    if (rebuild_end(e, x, row, f)) finish(x, row, par, f);
                }
            for (int k = x0; mine && 2 * k < ar; k += p.cpp) {
                // columns 2k and 2k + 1 in packed FP32 instructions (bit for bit the one-node
                // collision); one outside the range steps a copy of the other, for nothing
                const int x = 2 * k, x2 = x + 1;
                const bool in = x >= al, in2 = x2 >= al && x2 < ar;
                if (!in && !in2) continue;
                const int xk = in ? x : x2, xk2 = in2 ? x2 : x;
                R f[9], g[9];
                gather(xk, f);
                gather(xk2, g);
                float2 d[9];
#pragma unroll
                for (int i = 0; i < 9; ++i) d[i] = make_float2(f[i], g[i]);
                const float2 ref = make_float2(ref_of(xk), ref_of(xk2));
                float2 rk = make_float2(0.0f, 0.0f);
                if (centre_kn) {
                    rk = make_float2(centre_in(xk, par), centre_in(xk2, par));
                    centre_out(xk, y, par, ref.x, f);
                    centre_out(xk2, y, par, ref.y, g);
                }
                collide<R, MODE, float2>(d, ref, c, centre_kn ? &rk : nullptr);
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    f[i] = d[i].x;
                    g[i] = d[i].y;
                }
                put(xk, y, f);  // a copy writes what the other writes
                put(xk2, y, g);
            }
        } else {
            // one loop and one copy of the collision's code for both kinds of thread
            const bool ends = kEnds && end_thread;
            const int step = ends ? blockDim.x - p.main : p.cpp;
            const int until = ends ? (fixl || fixr ? end_items : 0) : mine ? ar : 0;
            for (int k = ends ? threadIdx.x - p.main : x0; k < until; k += step) {
                int x = k, row = y;
                R f[9];
                bool on = k >= al;
                if (ends)
                    on = rebuild_end(k, x, row, f);
                else if (on)
                    gather(k, f);
                if (on) finish(x, row, par, f);
            }
        }
        __syncthreads();
        cur ^= 9 * n;
    }

    // the block's own columns back, with the periodic images the sweeps read
    const int own = xb - xa, off = xa - lo;
    for (int x = (xa & ~3) + xv; x < xb; x += 32) {
        const bool vec = x >= xa && x + 4 <= xb;
#pragma unroll 2
        for (Row q = first; q.row < rows; next_row(q)) {
            const int from = cur + q.i * n + (x - lo) * cs + q.y;
            T* r = fout + q.i * a.plane + (long long)q.y * a.pitch + a.xoff;
            Quad v;
            if (vec) {
#pragma unroll
                for (int k = 0; k < 4; ++k) v.v[k] = s[from + k * cs];
                *reinterpret_cast<Quad*>(r + x) = v;
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (x + k >= xa && x + k < xb) r[x + k] = s[from + k * cs];
            }
        }
    }
    if (MODE == MODE_PERIODIC)
        for (int e = threadIdx.x; e < 3 * ny; e += blockDim.x) {
            const int k = e / ny, yy = e - k * ny;
            const int il = k == 0 ? 3 : 5 + k, ir = k == 0 ? 1 : k == 1 ? 5 : 8;  // 3 6 7 to column nx, 1 5 8 to column -1
            T* row = fout + (long long)yy * a.pitch + a.xoff;
            if (xa == 0) row[il * a.plane + nx] = s[cur + il * n + off * cs + yy];
            if (xb == nx) row[ir * a.plane - 1] = s[cur + ir * n + (off + own - 1) * cs + yy];
        }
    if (centre_kn) {
        R* rc0 = static_cast<R*>(a.rc_out);
        for (int e = threadIdx.x; e < 2 * own; e += blockDim.x) {
            const int row = e / own, x = e - row * own;
            if (row == 0 || a.yc1 != a.yc0) rc0[row * a.rc_stride + xa + x] = rcs[(nsteps & 1) * 2 * cols + row * cols + off + x];
        }
    }
}

// Launch fn(kernel) for the kernel of a storage, mode and plan.
template <class T, bool PACK, bool BIG, class F> cudaError_t with_mode(int mode, F&& fn) {
    return mode == MODE_PRESSURE ? fn(tile_kernel<T, MODE_PRESSURE, PACK, BIG>) : fn(tile_kernel<T, MODE_PERIODIC, PACK, BIG>);
}
template <class T, class F> cudaError_t with_shape(int mode, const TilePlan& p, F&& fn) {
    if constexpr (!std::is_same<T, double>::value)
        if (p.pack) return p.big ? with_mode<T, true, true>(mode, fn) : with_mode<T, true, false>(mode, fn);
    return p.big ? with_mode<T, false, true>(mode, fn) : with_mode<T, false, false>(mode, fn);
}
template <class F> cudaError_t with_tile(int storage, int mode, const TilePlan& p, F&& fn) {
    switch (storage) {
        case 0: return with_shape<double>(mode, p, fn);
        case 1: return with_shape<float>(mode, p, fn);
        case 2: return with_shape<__half>(mode, p, fn);
        case 3: return with_shape<__nv_bfloat16>(mode, p, fn);
    }
    return cudaErrorInvalidValue;
}

}  // namespace

// The plan with the least expected time per step, or none (h = 0) where the
// direct sweep is expected to be as fast.  Nanoseconds, from timed runs on
// GB300 (periodic and pressure channels of 128 to 410,000 nodes):
// - a launch costs 2.5 us (launch, one pass over its columns from L2 and back)
//   and 0.04 ns per byte its block moves, spread over its steps;
// - a step costs 0.2 us and 1.5 ns per node of the block (mean over the
//   shrinking halo), and where the block holds the end of a pressure channel
//   at least 1.05 us, the latency of rebuilding its end column;
// - the direct sweep costs 2.5 us per step and 0.01 ns per node of the channel.
// 1601 x 16 pressure FP32: w 11, h 24, expected 1.22, measured 1.36 us per step,
// against 2.9 us; 801 x 8 periodic 0.68 against 2.6; 4 x 32 in one block 0.33
// against 2.8; 6401 x 64 stays with the direct sweep (7.2 against 6.3 us).
// FP64 (pair.cuh), in the same way: a step costs 1.2 us, 3.2 us with the end of
// a pressure channel, and 10 ns per node; the direct sweep 3.7 or 8.2 us and
// 0.048 ns per node.  801 x 8 pressure: 5.3 us per step, against 8.1; periodic
// 2.8 against 3.8; 4 x 32 in one block 2.0 against 4.7; 2101 x 33 stays with the
// direct sweep (9.0 against 7.7).
//
// That model ranks the step counts; it is short on tall narrow tiles, whose
// copies and passes cost more.  So the plan found is kept only where a second
// estimate, fitted to 194 timed plans of 8 to 300 rows and 15,000 to 320,000
// nodes (within 8 % in the mean, 26 % at most), is below the direct sweep's by
// 5 %.  us per step, tiles and direct: 3026 x 76 BF16 periodic 5.45 / 3.28, 1428 x
// 49 3.12 / 2.60, 7187 x 32 3.89 / 3.78, 5882 x 17 2.49 / 2.83; pressure 909 x 110
// 4.49 / 4.04, 3026 x 76 4.40 / 4.48, 3061 x 49 3.16 / 4.08.
struct Fit {  // us, thousands of nodes
    double step, node, launch, copy;   // a step, each node of the block; a launch, each node its block moves
    double flat, direct, direct_node;  // the direct sweep: at least flat
};
constexpr Fit kFit[2][2] = {  // [16 bits][pressure]
    {{0.234, 0.835, 3.465, 3.475, 2.36, 1.843, 0.0083}, {0.802, 0.718, 4.381, 1.945, 2.96, 2.069, 0.0108}},
    {{0.095, 0.958, 6.911, 4.113, 2.73, 2.006, 0.0071}, {1.023, 0.260, 2.841, 4.272, 3.99, 3.409, 0.0056}}};

TilePlan plan_tiles(int storage, int mode, int nx, int ny, int sms, size_t smem_cap) {
    TilePlan best;
    if (ny > kTileThreads || sms < 1) return best;
    const size_t elem = storage == 0 ? 8 : storage == 1 ? 4 : 2, relem = storage == 0 ? 8 : 4;
    const int cs = ny | 1;
    const bool f64 = storage == 0, press = mode == MODE_PRESSURE;
    double best_t = 0.9 * (f64 ? (press ? 8200.0 : 3700.0) + 0.048 * nx * ny : 2500.0 + 0.01 * nx * ny);
    auto consider = [&](int blocks, int h, bool whole) {
        const int w = (nx + blocks - 1) / blocks, cols = whole ? nx : w + 2 * h;
        const bool big = (size_t)cols * cs > plane_of(elem, false);
        const size_t smem = tile_smem(big, cols, elem, relem);
        if (smem > smem_cap || (size_t)cols * cs > plane_of(elem, big)) return;
        const double nodes = (double)ny * (whole ? nx : w + h);
        double step = f64 ? (press ? 3200.0 : 1200.0) + 10.0 * nodes : 200.0 + 1.5 * nodes;
        if (press && !f64) step = std::max(step, 1050.0);
        const double ns = step + (whole ? 0.0 : (2500.0 + 0.04 * 9 * elem * ny * (cols + w)) / h);
        if (ns >= best_t) return;
        best_t = ns;
        TilePlan t;
        t.h = h;
        t.whole = whole;
        t.cs = cs;
        t.big = big;
        // one column per thread and pass, or a pair in packed FP32 where the
        // columns are more than one pass
        const int fit = kTileThreads / ny;  // columns (or pairs) that the threads cover
        t.pack = !f64 && cols > fit;
        const int units = t.pack ? (cols + 1) / 2 : cols, passes = (units + fit - 1) / fit;
        t.cpp = (units + passes - 1) / passes;
        t.main = (t.cpp * ny + 31) / 32 * 32;
        t.threads = t.main + (press ? std::min(kEndThreads, (4 * ny + 31) / 32 * 32) : 0);
        t.blocks = blocks;
        t.smem = smem;
        best = t;
    };
    consider(1, kTileMaxSteps, true);
    // a block that holds an end of a pressure channel needs the three columns
    // beside it to stay exact (the end is rebuilt from columns 1 and 2, which
    // pull from 0 to 3): every block has at least 3 of its own
    const int blocks = std::max(1, std::min(sms, nx / 3));
    if (nx / blocks >= 3)
        for (int h = 1; h <= 32; ++h) consider(blocks, h, false);
    // One step alone is faster as a direct sweep (us per call, tiles and sweep: 801
    // x 8 FP32 3.6 / 2.6, pressure 3.8 / 3.1; 2101 x 33 6.9 / 2.9; FP64 457 x 33
    // pressure 9.6 / 8.2), but for low 16-bit pressure channels (801 x 8 FP16 3.9 /
    // 4.3, 1601 x 16 4.3 / 4.3, 2101 x 21 4.9 / 4.4).  So are two where one block
    // copies the channel in more than one round of rows in flight (4 x 32 FP32 6.8 /
    // 5.3, FP16 10.7 / 6.0, FP64 11.5 / 9.6; 16 x 16, in one round, 4.2 / 4.6).
    best.few = elem == 2 && press && !best.whole && ny <= 16 ? 1 : 2;
    if (best.whole && 9 * ny > 9 * (best.threads / 8)) best.few = 3;  // 9 rows of 8 threads each in flight
    if (best.h > 0 && !best.whole && !f64) {
        const int w = (nx + best.blocks - 1) / best.blocks;
        const Fit& f = kFit[elem == 2][press];
        const double tall = 1e-3 * ny, nodes = 1e-3 * nx * ny;
        const double tiles = f.step + f.node * tall * (w + best.h) + (f.launch + f.copy * tall * (2 * w + 2 * best.h)) / best.h;
        if (tiles > 0.95 * std::max(f.flat, f.direct + f.direct_node * nodes)) return TilePlan{};
    }
    return best;
}

// The limit belongs to the kernel, not to a channel: it is always the cap that
// plans are made under, so that no channel's plan lowers it below another's.
cudaError_t tile_opt_in(int storage, int mode, const TilePlan& p, size_t smem_cap) {
    return with_tile(storage, mode, p, [&](auto kern) {
        return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_cap);
    });
}

cudaError_t launch_tiles(int storage, int mode, const TilePlan& p, const SweepArgs& a, int nsteps, cudaStream_t st) {
    return with_tile(storage, mode, p, [&](auto kern) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(p.blocks);
        cfg.blockDim = dim3(p.threads);
        cfg.dynamicSmemBytes = p.smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, kern, a, p, nsteps);
    });
}

}  // namespace clb
