// Two time steps of a large pressure channel per launch, FP32 storage (GB300,
// sm_103a).
//
// A sweep of a large FP32 channel is bound by reading and writing its
// populations once per step.  Here each warp takes a strip of 120 columns (4
// per lane, the outer two lanes a halo) and marches up its rows: the
// populations of row r at time t come from global memory into registers, step
// t+1 of row r is computed from them, and step t+2 of row r-1 from step t+1 of
// rows r-2 to r, which stay in registers (columns are exchanged between lanes by
// shuffles).  Only step t+2 is written, so the populations cross HBM once per
// two steps.  Nothing is shared between warps: no barrier, no shared memory but
// each lane's own prefetch slots, filled kAhead rows ahead by asynchronous
// copies.
//
// A block's four warps take four strips side by side; the rows are split so
// that one wave of blocks fills the GPU (Plan).  A segment recomputes the row
// below and the row above its own at t+1, the outer lanes recompute their
// neighbours' columns: 11 % of the collisions at 51 rows per segment.
//
// What bounds it: the fixed latencies of the collision's dependent chain, with
// two warps per scheduler (issue slots 45 % busy; 1.17 waiting warps per issued
// instruction, 0.08 of them for loads).  HBM carries the 36 algorithmic bytes per
// node and step at 0.73 of the copy peak.  8 warps per SM, not more: with 12 the
// same bytes move more slowly, the more streams of 480 bytes the worse, and at 16
// the registers spill.  25601 x 256: 47.8 us per step, against 71.6 us of the
// TMA-staged sweep.  16-bit storage gains nothing (47.5 us with 12 warps, against
// 40.8: as many instructions, half the bytes to save), nor do periodic channels
// (71 against 72 us: a third more instructions for the body force).
//
// The arithmetic per node is that of sweep.cu, bit for bit.
#include <algorithm>
#include <cstdint>

#include "clb_device.cuh"
#include "clb_internal.h"
#include "tma_common.cuh"

namespace clb {
namespace {

using tma::seg_dy;
using tma::seg_plane;

constexpr int kV = 4;                 // columns per lane
constexpr int kOwn = 30 * kV;         // columns a warp writes
constexpr int kAhead = 4;             // rows in flight, and prefetch slots
constexpr int kWarps = 4;             // strips, and warps, per block
constexpr int kBlocks = 2;            // per SM
constexpr int kEdge = 2;              // what a row of a group with an end column costs, in plain rows
constexpr int kSmem = kWarps * kAhead * 9 * 32 * (int)sizeof(float4);

// Who marches what.  The strips that hold an end column (the first, the last
// and the one before it, whose halo may) take about twice as long per row:
// each of the first edge_blocks blocks' warps has one of the edge_segs segments
// of one of them.  The other blocks have the other strips in groups of kWarps:
// one of the `segs` segments of a group's rows each, or, segs = 0, equal shares
// of all the groups' rows laid end to end.
struct Plan {
    int strips, edges, edge_segs, edge_blocks;
    int groups, segs;
};

__global__ void __launch_bounds__(32 * kWarps, kBlocks) march_kernel(const SweepArgs a, const Plan p) {
    using R = float;
    constexpr unsigned kAll = 0xffffffffu;
    extern __shared__ __align__(16) unsigned char smem[];
    const KC<R>& c = a.kf;
    const int nx = a.nx, ny = a.ny;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // no __restrict__: the previous launch may still write the input when this one starts
    const float* fin = static_cast<const float*>(a.fin);
    float* fout = static_cast<float*>(a.fout);
    float4* const slot = reinterpret_cast<float4*>(smem) + warp * kAhead * 9 * 32 + lane;  // [stage][population][lane]

    const bool edge = (int)blockIdx.x < p.edge_blocks;
    long long pos = 0, end = 1;  // shares: from row pos to row end of the groups laid end to end
    if (!edge && p.segs == 0) {
        const long long total = (long long)p.groups * ny, blocks = gridDim.x - p.edge_blocks, b = blockIdx.x - p.edge_blocks;
        pos = b * total / blocks;
        end = (b + 1) * total / blocks;
    }
    while (pos < end) {
        int strip, ya, yb;  // rows [ya, yb) are written
        if (edge || p.segs > 0) {
            const int job = edge ? blockIdx.x * kWarps + warp : blockIdx.x - p.edge_blocks;
            const int wide = edge ? p.edges : p.groups, n = edge ? p.edge_segs : p.segs;
            const int seg = job / wide, q = job - seg * wide;
            if (seg >= n) return;
            strip = !edge ? 1 + q * kWarps + warp : q == 0 ? 0 : p.strips - q;
            ya = (int)((long long)seg * ny / n);
            yb = (int)((seg + 1LL) * ny / n);
            pos = end;
        } else {
            const int group = (int)(pos / ny);
            const long long start = (long long)group * ny, stop = min(end, start + ny);
            strip = 1 + group * kWarps + warp;
            ya = (int)(pos - start);
            yb = (int)(stop - start);
            pos = stop;
        }
        if (ya == yb || (!edge && strip > p.strips - p.edges)) continue;

        const int x0 = strip * kOwn - kV + lane * kV;  // this lane's columns
        const bool writes = lane >= 1 && lane <= 30 && x0 < nx;
        // past the row's ends the lane reads its padding
        const int xl = max(-kV, min(x0, (nx + kV - 1) / kV * kV));
        auto fetch = [&](int r, int stage) {
            const int rt = row_kind(r, ny);
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const float* row = fin + seg_plane(i, rt) * a.plane + (long long)(r + seg_dy(i, rt)) * a.pitch + a.xoff;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                                 (uint32_t)__cvta_generic_to_shared(slot + (stage * 9 + i) * 32)),
                             "l"(row + xl)
                             : "memory");
            }
        };
        auto commit = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };

        auto from_left = [&](const R (&v)[kV], R s, R (&o)[kV]) {  // columns x0-1 .. x0+2, plus s
            const R p = __shfl_up_sync(kAll, v[kV - 1], 1);
            o[0] = p + s;
#pragma unroll
            for (int k = 1; k < kV; ++k) o[k] = v[k - 1] + s;
        };
        auto from_right = [&](const R (&v)[kV], R s, R (&o)[kV]) {  // columns x0+1 .. x0+4, minus s
            const R n = __shfl_down_sync(kAll, v[0], 1);
            o[kV - 1] = n - s;
#pragma unroll
            for (int k = 0; k < kV - 1; ++k) o[k] = v[k + 1] - s;
        };
        // Eq. 20: the bounce-back part a, the specular part b
        auto wall = [&](const R (&a_)[kV], const R (&b)[kV], R (&o)[kV]) {
#pragma unroll
            for (int k = 0; k < kV; ++k) o[k] = ln::fma(c.r, a_[k], ln::mul(c.rc, b[k]));
        };
        // the end columns of a pressure channel, rebuilt from the two beside them (Sec. 3.2)
        const int kfirst = -x0, klast = nx - 1 - x0;  // the lane's index of column 0, of column nx - 1
        const bool has_first = strip == 0;
        const bool has_last = __any_sync(kAll, klast >= 0 && klast < kV);
        auto ends = [&](R (&f)[9][kV]) {
            if (has_first && kfirst == 0) {
                R n1[9], n2[9], t[9];
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    n1[i] = f[i][1];
                    n2[i] = f[i][2];
                }
                rebuild_nodes<R>(c, 0, true, n1, n2, t);
#pragma unroll
                for (int i = 0; i < 9; ++i) f[i][0] = t[i];
            }
            if (has_last) {
                R p1[9], p2[9];  // the last two columns of the lane to the left
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    p1[i] = __shfl_up_sync(kAll, f[i][kV - 1], 1);
                    p2[i] = __shfl_up_sync(kAll, f[i][kV - 2], 1);
                }
                if (klast >= 0 && klast < kV) {
                    R n1[9], n2[9], t[9];
#pragma unroll
                    for (int i = 0; i < 9; ++i) {
                        n1[i] = klast == 0 ? p1[i] : klast == 1 ? f[i][0] : klast == 2 ? f[i][1] : f[i][2];
                        n2[i] = klast == 0 ? p2[i] : klast == 1 ? p1[i] : klast == 2 ? f[i][0] : f[i][1];
                    }
                    rebuild_nodes<R>(c, nx - 1, false, n1, n2, t);
#pragma unroll
                    for (int k = 0; k < kV; ++k)
                        if (k == klast)
#pragma unroll
                            for (int i = 0; i < 9; ++i) f[i][k] = t[i];
                }
            }
        };
        auto step = [&](R (&f)[9][kV]) {
#pragma unroll
            for (int k = 0; k < kV; k += 2) {
                float2 d[9];
#pragma unroll
                for (int i = 0; i < 9; ++i) d[i] = make_float2(f[i][k], f[i][k + 1]);
                const float2 ref = ln::fma(ln::bc<float2>(c.slope), make_float2(float(x0 + k), float(x0 + k + 1)),
                                           ln::bc<float2>(c.ref0));
                collide<R, MODE_PRESSURE, float2>(d, ref, c);
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    f[i][k] = d[i].x;
                    f[i][k + 1] = d[i].y;
                }
            }
        };
        // Step t+1 of the rows, as step t+2 pulls it: m0, m1, m3 of the last row,
        // b2, b5, b6 of the last row and of the one before it, all moved along x.
        R m0[kV], m1[kV], m3[kV], b2[kV], b5[kV], b6[kV], c2[kV], c5[kV], c6[kV];
        const int first = max(ya - 1, 0), last = min(yb, ny - 1);  // rows at t+1
#pragma unroll
        for (int q = 0; q < kAhead; ++q) {
            if (first + q <= last) fetch(first + q, q);
            commit();
        }
        int stage = 0;
        for (int r = first; r <= yb; ++r) {
            // at r = ny there is no row; the top wall sends row ny-1's own back
            R f[9][kV];
            R w4[kV], w7[kV], w8[kV];  // what step t+2 of row r-1 pulls from row r
            const bool row = r <= last;
            if (row) {
                asm volatile("cp.async.wait_group %0;" ::"n"(kAhead - 1) : "memory");
                R v[9][kV];
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    const float4 q = slot[(stage * 9 + i) * 32];
                    v[i][0] = q.x;
                    v[i][1] = q.y;
                    v[i][2] = q.z;
                    v[i][3] = q.w;
                }
                const bool bottom = r == 0, top = r == ny - 1;
#pragma unroll
                for (int k = 0; k < kV; ++k) {
                    f[0][k] = v[0][k];
                    f[2][k] = v[2][k];
                    f[4][k] = v[4][k];
                }
                from_left(v[1], c.sha, f[1]);
                from_right(v[3], c.sha, f[3]);
                if (bottom) {
                    R s[kV];
                    from_left(v[6], c.shd, s);
                    wall(v[5], s, f[5]);
                    from_right(v[5], c.shd, s);
                    wall(v[6], s, f[6]);
                } else {
                    from_left(v[5], c.shd, f[5]);
                    from_right(v[6], c.shd, f[6]);
                }
                if (top) {
                    R s[kV];
                    from_right(v[8], c.shd, s);
                    wall(v[7], s, f[7]);
                    from_left(v[7], c.shd, s);
                    wall(v[8], s, f[8]);
                } else {
                    from_right(v[7], c.shd, f[7]);
                    from_left(v[8], c.shd, f[8]);
                }
                ends(f);
                step(f);
                // the slots' values have been used: they can take the row kAhead on
                if (r + kAhead <= last) fetch(r + kAhead, stage);
                commit();
                stage = stage + 1 == kAhead ? 0 : stage + 1;
#pragma unroll
                for (int k = 0; k < kV; ++k) w4[k] = f[4][k];
                from_right(f[7], c.shd, w7);
                from_left(f[8], c.shd, w8);
            } else {  // row ny - 1's c-parts were left as the top wall returns them
#pragma unroll
                for (int k = 0; k < kV; ++k) {
                    w4[k] = c2[k];
                    w7[k] = c5[k];
                    w8[k] = c6[k];
                }
            }
            if (r > ya) {  // step t+2 of row r - 1
                R g[9][kV];
#pragma unroll
                for (int k = 0; k < kV; ++k) {
                    g[0][k] = m0[k];
                    g[1][k] = m1[k];
                    g[3][k] = m3[k];
                    g[2][k] = b2[k];
                    g[5][k] = b5[k];
                    g[6][k] = b6[k];
                    g[4][k] = w4[k];
                    g[7][k] = w7[k];
                    g[8][k] = w8[k];
                }
                ends(g);
                step(g);
                if (writes) {
                    float* out = fout + (long long)(r - 1) * a.pitch + a.xoff + x0;
                    if (x0 + kV <= nx) {
#pragma unroll
                        for (int i = 0; i < 9; ++i) *reinterpret_cast<float4*>(out + i * a.plane) =
                                make_float4(g[i][0], g[i][1], g[i][2], g[i][3]);
                    } else {
#pragma unroll
                        for (int k = 0; k < kV; ++k)
                            if (x0 + k < nx)
#pragma unroll
                                for (int i = 0; i < 9; ++i) out[i * a.plane + k] = g[i][k];
                    }
                }
            }
            if (!row) break;
            // carry row r: what rows r (m) and r + 1 (b) pull from it at t+2
            if (r == 0) {  // row 0 pulls its own from the bottom wall
#pragma unroll
                for (int k = 0; k < kV; ++k) b2[k] = f[4][k];
                wall(f[7], w8, b5);
                wall(f[8], w7, b6);
            } else {
#pragma unroll
                for (int k = 0; k < kV; ++k) {
                    b2[k] = c2[k];
                    b5[k] = c5[k];
                    b6[k] = c6[k];
                }
            }
#pragma unroll
            for (int k = 0; k < kV; ++k) {
                m0[k] = f[0][k];
                c2[k] = f[2][k];
            }
            from_left(f[1], c.sha, m1);
            from_right(f[3], c.sha, m3);
            from_left(f[5], c.shd, c5);
            from_right(f[6], c.shd, c6);
            if (r == ny - 1) {  // the top wall returns them to row ny - 1
                R t5[kV], t6[kV];
                wall(f[5], c6, t5);
                wall(f[6], c5, t6);
#pragma unroll
                for (int k = 0; k < kV; ++k) {
                    c5[k] = t5[k];
                    c6[k] = t6[k];
                }
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    }
}

}  // namespace

cudaError_t march_opt_in() {
    return cudaFuncSetAttribute(march_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
}

cudaError_t launch_march(int sms, const SweepArgs& a, cudaStream_t st) {
    Plan p;
    const int slots = kBlocks * sms, ny = a.ny;
    p.strips = (a.nx + kOwn - 1) / kOwn;
    p.edges = std::min(p.strips, 3);
    p.groups = (p.strips - p.edges + kWarps - 1) / kWarps;
    // a wave of segments of one length, the edge strips' half as long, keeps
    // neighbouring strips at the same rows, which HBM likes (25601 x 256: with
    // equal shares 1.05 times as long); shares where whole segments would
    // leave more than a fifth of the wave empty (80000 x 40: 35.6 and 24.8 us).
    // At least 4 rows each: every segment recomputes two.
    p.segs = (int)std::min(slots / (p.groups + 2.0 * p.edges / kWarps), std::max(1.0, ny / 4.0));
    p.edge_segs = std::max(1, std::min(std::max(2 * p.segs, 1), ny / 2));
    p.edge_blocks = (p.edges * p.edge_segs + kWarps - 1) / kWarps;
    int blocks = p.groups * p.segs;
    if (p.groups > 0 && (p.segs < 1 || (blocks + p.edge_blocks < slots * 4 / 5 && p.segs < ny / 4))) {
        p.segs = 0;
        p.edge_segs = std::max(1, std::min((int)(2LL * slots / p.groups) + 2, ny / 2));
        p.edge_blocks = (p.edges * p.edge_segs + kWarps - 1) / kWarps;
        blocks = (int)std::max(1LL, std::min<long long>(slots - p.edge_blocks, (long long)p.groups * ny / 4));
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks + p.edge_blocks);
    cfg.blockDim = dim3(32 * kWarps);
    cfg.dynamicSmemBytes = kSmem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, march_kernel, a, p);
}

}  // namespace clb
