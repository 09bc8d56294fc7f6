// Discrete adjoint of the body-force channel (Sec. 3.1 of Liu & He,
// arXiv:1603.01955): gradient of the flow sum J = mean_x sum_y u_x after N
// steps with respect to the CBBSR bounce-back fraction r_b (Eq. 20), the
// Bosanquet factor a (Eq. 16-18, 21, through s_v and s_q) and the body force G
// (Eq. 9, 13).
//
// One step is f_{t+1} = C(P(f_t)): P pulls the post-collision populations
// (Eq. 5, periodic x, walls Eq. 20), C collides every node (Eq. 4, 6-13).  The
// adjoint runs backwards: mu = J_C(P f_t)^T lambda_{t+1} per node, then
// lambda_t = P^T mu, while r_b, a and G collect lambda_{t+1}^T dC/dtheta and
// mu^T dP/dr.  J_C^T lambda is the collision's reverse, written out by hand
// (reverse_collide): the moments and kernels of the forward step, then their
// adjoints in the opposite order, which also yield the terms of s_v, s_q and G.
// P^T is a gather (each post-collision population is pulled by one node, or by
// two wall nodes).  The forward keeps a checkpoint every C steps (C ~
// sqrt(N)) and recomputes each segment before walking it backwards.
// Parameter sums are FP64, or FP32 pairs of 48 bits; states and adjoints are FP32
// or FP64.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <type_traits>
#include <vector>

#include "../../include/clb.h"
#include "clb_device.cuh"
#include "clb_internal.h"

using namespace clb;

namespace {

// Constants of one adjoint run in compute type R.
template <class R> struct AdjConst {
    KC<R> c;       // collision constants (body-force channel)
    R dsv4_da;     // d(s_v/4)/da
    R dsq4_da;     // d(s_q/4)/da
    R r, rc;       // r_b, 1 - r_b
    R ref;         // reference density of the stored deviations
    int nx, ny;
};

template <class R>
__global__ void adj_forward_kernel(const R* fin, R* fout, AdjConst<R> k) {
    const int nn = k.nx * k.ny;
    for (int node = blockIdx.x * blockDim.x + threadIdx.x; node < nn; node += gridDim.x * blockDim.x) {
        R d[9];
        gather_at(fin, pull_of(k.nx, k.ny, node % k.nx, node / k.nx), k.r, k.rc, d);
        collide<R, MODE_PERIODIC>(d, k.ref, k.c);
        for (int i = 0; i < 9; ++i) fout[i * nn + node] = d[i];
    }
}

// A sum over many steps: FP64 as it is, FP32 terms in a pair of FP32 numbers
// (the rounding errors of the running sum, exact by Knuth's two-sum, go to the
// second), 48 bits without the FP64 pipe.
template <class R> struct Acc {
    R s = 0;
    __device__ __forceinline__ void add(R v) { s += v; }
    __device__ __forceinline__ void add(R a, R b) { s += a * b; }  // a b
    __device__ __forceinline__ double value() const { return (double)s; }
};
template <> struct Acc<float> {
    float s = 0, e = 0;
    __device__ __forceinline__ void add(float v) {
        const float t = __fadd_rn(s, v), z = __fsub_rn(t, s);
        e = __fadd_rn(e, __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(v, z)));
        s = t;
    }
    __device__ __forceinline__ void add(float a, float b) {
        const float v = __fmul_rn(a, b);
        e = __fadd_rn(e, __fmaf_rn(a, b, -v));
        add(v);
    }
    __device__ __forceinline__ double value() const { return (double)s + (double)e; }
};

// The sums of one thread: l . dC/d(s_v/4), dC/d(s_q/4), dC/dG, and mu . dP/dr.
template <class R> struct ParamSums {
    Acc<R> sv, sq, g, r;
};

// What the reverse of a node's collision needs of its forward step (collide,
// MODE_PERIODIC): velocity, moments, braces and kernels.  It does not depend on
// the adjoint, so a walk can form it one step ahead.
template <class R> struct Forward {
    R rho, irho, jx, jy, ux, uy, ux2, uy2, uxy, kx, ky, nkxy, kxxy, kxyy, rf;
    R t5u, t4, t5, t6, t7, g5, g6, g7, hp, hm;
};
template <class R>
__device__ __forceinline__ Forward<R> forward_of(const R (&d)[9], R ref, const KC<R>& c) {
    const R h = R(0.5), two = R(2), third = R(1.0 / 3.0);
    const R a57 = d[5] + d[7], a68 = d[6] + d[8], p57 = d[5] - d[7], p86 = d[8] - d[6];
    const R nkxy = a68 - a57, kxxyy = a57 + a68, kxxy = p57 - p86, kxyy = p57 + p86;
    const R s13 = d[1] + d[3], s24 = d[2] + d[4];
    const R kxx = s13 + kxxyy, kyy = s24 + kxxyy, drho = d[0] + s13 + s24 + kxxyy;
    const R jx = d[1] - d[3] + kxyy, jy = d[2] - d[4] + kxxy;
    const R rho = ref + drho, irho = rcp(rho), fx = c.fx;
    const R ux = jx * irho + c.hfx, uy = jy * irho;
    const R kx = kxx + third * ref, ky = kyy + third * ref;
    const R ux2 = ux * ux, uy2 = uy * uy, uxy = ux * uy, rf = rho * fx;
    const R t5u = rho * uxy + nkxy;
    const R t3 = rho * (ux2 + uy2) + R(2.0 / 3.0) * drho - (kxx + kyy) - rf * ux;
    const R t4 = rho * (ux2 - uy2) + (kyy - kxx) - rf * ux;
    const R t5 = t5u - h * rf * uy;
    const R t6 = two * ux * t5u - uy * kx + kxxy - rf * uxy;
    const R t7 = two * uy * t5u - ux * ky + kxyy - h * rf * uy2;
    const R g3 = c.s3_12 * t3, g4 = c.sv_4 * t4, g5 = c.sv_4 * t5;
    const R hp = R(1.5) * g3 + h * g4, hm = R(1.5) * g3 - h * g4;
    const R g6 = c.sq_4 * t6 - uy * hp - two * ux * g5;
    const R g7 = c.sq_4 * t7 - ux * hm - two * uy * g5;
    return {rho, irho, jx, jy, ux, uy, ux2, uy2, uxy, kx, ky, nkxy, kxxy, kxyy, rf,
            t5u, t4, t5, t6, t7, g5, g6, g7, hp, hm};
}

// m = J_C(d)^T l for one node of a body-force channel, from its forward_of(d),
// and the node's parameter terms.  Capital names are adjoints.
template <class R>
__device__ __forceinline__ void reverse_collide(const Forward<R>& v, const R (&l)[9], const KC<R>& c, R (&m)[9],
                                                ParamSums<R>& sum) {
    const R h = R(0.5), q = R(0.25), two = R(2), fx = c.fx;
    const auto [rho, irho, jx, jy, ux, uy, ux2, uy2, uxy, kx, ky, nkxy, kxxy, kxyy, rf,
                t5u, t4, t5, t6, t7, g5, g6, g7, hp, hm] = v;
    // reverse of Eq. 6 and of the source (Eq. 9-10)
    const R A1 = l[1] + l[3], A2 = l[2] + l[4], D1 = l[1] - l[3], D2 = l[2] - l[4];
    const R S5 = l[5] + l[7], S6 = l[6] + l[8], E5 = l[7] - l[5], E6 = l[8] - l[6];
    const R A = A1 + A2, S = S5 + S6;
    const R G8 = R(4) * l[0] - two * A + S;
    const R M1 = h * D1, M3 = h * A1 - l[0], M5 = q * (S5 - S6), M6 = -(h * D2 + q * (E5 + E6));
    const R M7 = q * (E6 - E5) - h * D1, M8 = l[0] - h * A + q * S;
    // g8 .. g3
    const R G7 = two * D1 + E5 - E6 - two * ux * G8;
    const R G6 = two * D2 + E5 + E6 - two * uy * G8;
    const R HP = -(uy2 * G8 + uy * G6), HM = -(ux2 * G8 + ux * G7);
    const R G5 = S5 - S6 - R(4) * uxy * G8 - two * (uy * G7 + ux * G6);
    const R G4 = A1 - A2 + h * (HP - HM);
    const R G3 = two * S - R(4) * l[0] - A - two * G8 + R(1.5) * (HP + HM);
    R UXY = R(-4) * g5 * G8;
    R UX = -(two * (ux * hm + g7) * G8 + hm * G7 + two * g5 * G6);
    R UY = -(two * (uy * hp + g6) * G8 + hp * G6 + two * g5 * G7);
    const R T8 = c.s8_4 * G8, T7 = c.sq_4 * G7, T6 = c.sq_4 * G6, T5 = c.sv_4 * G5, T4 = c.sv_4 * G4, T3 = c.s3_12 * G3;
    sum.sv.add(t4, G4);
    sum.sv.add(t5, G5);
    sum.sq.add(t6, G6);
    sum.sq.add(t7, G7);
    // the braces of Eq. 7 and the source's moments: the force terms first, as
    // one factor of rho G and its own adjoint
    const R uxy2 = ux * uy2;
    const R T34 = T3 + T4;
    // d/d(rho fx) of every force term
    const R RF = -(T34 * ux + h * T5 * uy + T6 * uxy + h * T7 * uy2 + T8 * uxy2) + M1 + two * M3 * ux + M5 * uy +
                 two * M6 * uxy + M7 * uy2 + two * M8 * uxy2;
    const R FU = -T34 + two * M3 + (two * M8 - T8) * uy2;              // rf * d/dux (but uxy)
    const R FV = M5 - h * T5 + (two * M7 - T7) * uy + (R(4) * M8 - two * T8) * uxy;  // rf * d/duy (but uxy)
    const R T5U = T5 + two * (uy * T7 + ux * T6) + R(3) * uxy * T8;
    UXY += (R(3) * t5u + nkxy) * T8 + rho * T5U + rf * (two * M6 - T6);
    UX += two * (kxyy - ux * ky) * T8 - ky * T7 + two * t5u * T6 + two * rho * ux * T34 + rf * FU + uy * UXY;
    UY += two * (kxxy - uy * kx) * T8 + two * t5u * T7 - kx * T6 + two * rho * uy * (T3 - T4) + rf * FV + ux * UXY;
    sum.g.add(rho * RF + h * UX);  // u_x holds G/2 as well
    R DR = fx * RF + (ux2 + uy2) * T3 + (ux2 - uy2) * T4 + uxy * T5U;  // through rho
    const R JX = irho * UX, JY = irho * UY;
    DR -= irho * (jx * JX + jy * JY);
    DR += R(2.0 / 3.0) * T3 + R(1.0 / 9.0) * T8;
    const R KXX = -(uy2 * T8 + uy * T6 + T4 + T3), KYY = T4 - T3 - ux2 * T8 - ux * T7;
    const R NKXY = uxy * T8 + T5U;
    const R KXXY = two * uy * T8 + T6 + JY, KXYY = two * ux * T8 + T7 + JX;
    const R X13 = KXX + DR, X24 = KYY + DR, KT = KXX + KYY + DR - T8;
    m[0] = l[0] + DR;
    m[1] = l[1] + (X13 + JX);
    m[3] = l[3] + (X13 - JX);
    m[2] = l[2] + (X24 + JY);
    m[4] = l[4] + (X24 - JY);
    const R K57 = KT - NKXY, K68 = KT + NKXY, P57 = KXXY + KXYY, P86 = KXYY - KXXY;
    m[5] = l[5] + (K57 + P57);
    m[7] = l[7] + (K57 - P57);
    m[6] = l[6] + (K68 - P86);
    m[8] = l[8] + (K68 + P86);
}

// mu . dP/dr of a wall node: f5, f6 (bottom) or f7, f8 (top) of the pull
// r A + (1 - r) B collect mu (A - B) (Eq. 20).
template <class R> __device__ __forceinline__ void wall_term(R mu, R a, R b, Acc<R>& s) {
    if constexpr (std::is_same<R, float>::value) {
        const float v = __fsub_rn(a, b), z = __fsub_rn(v, a);  // a - b and its rounding error
        const float e = __fsub_rn(__fsub_rn(a, __fsub_rn(v, z)), __fadd_rn(b, z));
        s.add(mu, v);
        s.add(mu, e);
    } else {
        s.add(mu, a - b);
    }
}

__device__ __forceinline__ double block_sum(double v, double* sh) {
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    const double s = sh[0];
    __syncthreads();
    return s;
}

constexpr int kAdjThreads = 128;

// lambda_t(node) = (P^T mu)(node): each post-collision population of step t is
// pulled by the node it streams to, or, at a wall, by the bounce-back and the
// specular terms of Eq. 20 (two nodes of the wall row).  The offsets and
// weights for one node, as Pull for the forward direction.
template <class At> __device__ __forceinline__ Pull push_with(int nx, int ny, int x, int y, At at) {
    Pull p;
    const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
    p.top = y == ny - 1;
    p.bottom = y == 0;
    p.wb[0] = p.wb[1] = p.wt[0] = p.wt[1] = 0;
    p.o[0] = at(0, y, x);
    p.o[1] = at(1, y, xp);  // f1 at x is pulled by x+1
    p.o[3] = at(3, y, xm);
    // moving up (2, 5, 6): pulled by row y+1, or by the top-wall terms
    p.o[2] = p.top ? at(4, y, x) : at(2, y + 1, x);
    p.o[5] = p.top ? at(7, y, x) : at(5, y + 1, xp);
    p.o[6] = p.top ? at(8, y, x) : at(6, y + 1, xm);
    if (p.top) {
        p.wt[0] = at(8, y, xp);
        p.wt[1] = at(7, y, xm);
    }
    // moving down (4, 7, 8): pulled by row y-1, or by the bottom-wall terms
    p.o[4] = p.bottom ? at(2, y, x) : at(4, y - 1, x);
    p.o[7] = p.bottom ? at(5, y, x) : at(7, y - 1, xm);
    p.o[8] = p.bottom ? at(6, y, x) : at(8, y - 1, xp);
    if (p.bottom) {
        p.wb[0] = at(6, y, xm);
        p.wb[1] = at(5, y, xp);
    }
    return p;
}
__device__ __forceinline__ Pull push_of(int nx, int ny, int x, int y) {
    return push_with(nx, ny, x, y, [&](int i, int yy, int xx) { return (i * ny + yy) * nx + xx; });
}
template <class R>
__device__ __forceinline__ void transpose_at(const R* mu, const Pull& p, R r, R rc, R (&o)[9]) {
#pragma unroll
    for (int i = 0; i < 9; ++i) o[i] = mu[p.o[i]];
    if (p.top) {
        o[5] = r * o[5] + rc * mu[p.wt[0]];
        o[6] = r * o[6] + rc * mu[p.wt[1]];
    }
    if (p.bottom) {
        o[7] = r * o[7] + rc * mu[p.wb[0]];
        o[8] = r * o[8] + rc * mu[p.wb[1]];
    }
}

// One node's share of backward step t: lambda_{t+1} from mu_{t+1} (or given,
// at the last step), mu_t = J_C^T lambda, the parameter terms.  f: the state
// at t; all [9][ny][nx].
template <class R>
__device__ __forceinline__ void back_node(const R* f, const R* mu_next, const R* lam, R* mu, int node, int x, int y,
                                          const AdjConst<R>& k, ParamSums<R>& sum) {
    const int nn = k.nx * k.ny;
    const Pull p = pull_of(k.nx, k.ny, x, y);
    R fb[9], l[9], m[9];
    gather_at(f, p, k.r, k.rc, fb);
    if (mu_next)
        transpose_at(mu_next, push_of(k.nx, k.ny, x, y), k.r, k.rc, l);
    else
        for (int i = 0; i < 9; ++i) l[i] = lam[i * nn + node];
    reverse_collide(forward_of(fb, k.ref, k.c), l, k.c, m, sum);
    for (int i = 0; i < 9; ++i) mu[i * nn + node] = m[i];
    if (p.bottom) {
        wall_term(m[5], f[p.o[5]], f[p.wb[0]], sum.r);
        wall_term(m[6], f[p.o[6]], f[p.wb[1]], sum.r);
    }
    if (p.top) {
        wall_term(m[7], f[p.o[7]], f[p.wt[0]], sum.r);
        wall_term(m[8], f[p.o[8]], f[p.wt[1]], sum.r);
    }
}

// mu_t at every node from mu_{t+1}, and the parameter terms of step t added to
// this block's slots acc[k * gridDim.x + blockIdx.x], k = 0, 1, 2 (r, a, G).
// Each slot has one writer and the launches run in stream order, so every slot
// is summed in a fixed order and the gradient is the same bit for bit on every
// run.
template <class R>
__global__ void __launch_bounds__(kAdjThreads)
    adj_back_kernel(const R* f_t, const R* mu_next, const R* lam, R* mu, double* acc, AdjConst<R> k) {
    __shared__ double sh[kAdjThreads];
    const int nn = k.nx * k.ny;
    ParamSums<R> sum;
    for (int node = blockIdx.x * blockDim.x + threadIdx.x; node < nn; node += gridDim.x * blockDim.x)
        back_node(f_t, mu_next, lam, mu, node, node % k.nx, node / k.nx, k, sum);
    const double gr = block_sum(sum.r.value(), sh);
    const double ga = block_sum(sum.sv.value() * (double)k.dsv4_da + sum.sq.value() * (double)k.dsq4_da, sh);
    const double gg = block_sum(sum.g.value(), sh);
    if (threadIdx.x == 0) {
        acc[0 * gridDim.x + blockIdx.x] += gr;
        acc[1 * gridDim.x + blockIdx.x] += ga;
        acc[2 * gridDim.x + blockIdx.x] += gg;
    }
}

// One node's term of J = (1/nx) sum u_x of the final post-collision state (its
// populations at f[at + i stride]), and
// its lambda_N = dJ/df_N: u_x = sum_i e_ix f_i / rho - G/2, so
// dJ/df_i = (e_ix - u_x - G/2) / (nx rho).
template <class R>
__device__ __forceinline__ double flow_term(const R* f, int stride, int at, R* lam, int node, const AdjConst<R>& k) {
    const int nn = k.nx * k.ny;
    const int ex[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1};
    double rho = (double)k.ref, jx = 0;
    for (int i = 0; i < 9; ++i) {
        const double v = (double)f[i * stride + at];
        rho += v;
        jx += ex[i] * v;
    }
    const double ux = jx / rho - 0.5 * (double)k.c.fx;
    for (int i = 0; i < 9; ++i) lam[i * nn + node] = R((ex[i] - ux - 0.5 * (double)k.c.fx) / (k.nx * rho));
    return ux / k.nx;
}

template <class R>
__global__ void __launch_bounds__(kAdjThreads) adj_final_kernel(const R* f, R* lam, double* acc, AdjConst<R> k) {
    __shared__ double sh[kAdjThreads];
    const int nn = k.nx * k.ny;
    double js = 0;
    for (int node = blockIdx.x * blockDim.x + threadIdx.x; node < nn; node += gridDim.x * blockDim.x)
        js += flow_term(f, nn, node, lam, node, k);
    js = block_sum(js, sh);
    if (threadIdx.x == 0) acc[3 * gridDim.x + blockIdx.x] = js;
}

// ------------------------------------------------------ resident engine
//
// The whole checkpointed forward pass is one launch, of one block with block
// barriers between the steps for the smallest grids (block_nodes), else of a
// thread-block cluster with cluster barriers; the backward walk
// over every segment is one launch of a cluster.  The parameter sums stay per thread (in step
// order) and are added by fixed trees at the end, so the gradient is the same
// bit for bit on every run.
//
// Backward, FP32 grids of at most one node per thread of a block: a pair of
// blocks (adj_pair_backward_kernel).  One recomputes a segment's steps while
// the other walks the segment after it backwards, each with its state in shared
// memory and block barriers only; the cluster barrier separates segments.
// Other grids: every block of the cluster takes its share of the nodes of each
// step, with a cluster barrier between steps: the states in the blocks' shared
// memory where each thread has one node (adj_share_*_kernel), in L2 where there
// are more (adj_cl_*_kernel).
// 4 x 64 nodes, FP32, per step: forward 0.32 us, backward 0.79 us (0.63 and
// 6.46 us with the pulls worked out every step and J_C^T lambda formed by eleven
// forward-mode columns over 16 blocks); both are bound by issue and latency in
// their one block.  A backward step of one warp per scheduler takes 0.58 us
// (4 x 32), so its latency, not its issue, comes first: the forward part of
// the next step, which does not wait for the adjoint, is formed beside the
// reverse of this one (4 x 64 0.94 us and 4 x 32 0.72 us one after the other).
// 20 x 128 nodes, by a cluster: forward 1.16, backward 2.2 us (31.4 us).
constexpr int kResThreads = 512;

__device__ __forceinline__ double res_block_sum(double v, double* sh) {
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int w = kResThreads / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w && threadIdx.x + w < blockDim.x) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    const double r = sh[0];
    __syncthreads();
    return r;
}

// Steps of the whole grid in shared memory, from copy s to copy o (then the
// other way round), with the block's barrier after each; a node per thread, at
// most, whose pull is worked out once.  Before each collision, visit(step,
// pulled populations, pull, state) sees the node.
template <class R, class V>
__device__ __forceinline__ void res_steps(R*& s, R*& o, long long nsteps, const AdjConst<R>& k, V&& visit) {
    const int nn = k.nx * k.ny, node = threadIdx.x;
    Pull p{};
    if (node < nn) p = pull_of(k.nx, k.ny, node % k.nx, node / k.nx);
    for (long long t = 0; t < nsteps; ++t) {
        if (node < nn) {
            R d[9];
            gather_at(s, p, k.r, k.rc, d);
            visit(t, d, p, s);
            collide<R, MODE_PERIODIC>(d, k.ref, k.c);
#pragma unroll
            for (int i = 0; i < 9; ++i) o[i * nn + node] = d[i];
        }
        __syncthreads();
        R* q = s;
        s = o;
        o = q;
    }
}

// Forward pass from f^eq(rho_out, 0): checkpoint s (the state at step s C)
// into ckpt + s state_elems, then J and lambda_N (as adj_final_kernel).
template <class R>
__global__ void __launch_bounds__(kResThreads)
    adj_res_forward_kernel(R* ckpt, size_t state_elems, int every, long long nsteps, R* lam_final, double* J,
                           AdjConst<R> k) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    const int nn = k.nx * k.ny, n9 = 9 * nn;
    R* a = reinterpret_cast<R*>(sm_raw);
    R* b = a + n9;
    double* red = reinterpret_cast<double*>(sm_raw + ((2 * n9 * sizeof(R) + 15) / 16) * 16);
    for (int e = threadIdx.x; e < n9; e += blockDim.x) a[e] = R(0);  // zero deviations
    __syncthreads();
    for (long long t = 0; t < nsteps; t += every) {
        R* c = ckpt + (size_t)(t / every) * state_elems;
        for (int e = threadIdx.x; e < n9; e += blockDim.x) c[e] = a[e];
        res_steps(a, b, min((long long)every, nsteps - t), k, [](long long, const R*, const Pull&, const R*) {});
    }
    double js = 0;
    for (int node = threadIdx.x; node < nn; node += blockDim.x) js += flow_term(a, nn, node, lam_final, node, k);
    js = res_block_sum(js, red);
    if (threadIdx.x == 0) *J = js;
}

constexpr int kClusterMax = 16;

__device__ __forceinline__ void cluster_barrier() {
    __threadfence();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ int cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return (int)r;
}

template <class R>
__device__ __forceinline__ void write_sums(const ParamSums<R>& sum, const AdjConst<R>& k, double* red, double* out) {
    const double gr = res_block_sum(sum.r.value(), red);
    const double ga = res_block_sum(sum.sv.value() * (double)k.dsv4_da + sum.sq.value() * (double)k.dsq4_da, red);
    const double gg = res_block_sum(sum.g.value(), red);
    if (threadIdx.x == 0) {
        out[0] = gr;
        out[1] = ga;
        out[2] = gg;
    }
}

// The backward walk by a pair of blocks (see above): per step of a segment,
// `seg` holds the pulled populations of every node, coalesced, and the eight
// values each column's wall terms differ by (pair_elems elements).  bufs: the
// segments it holds, 2 (recomputation of one beside the walk over the other) or
// 1 (in turn).  Nodes <= threads of a block.
__host__ __device__ constexpr size_t pair_elems(int nx, int ny) { return 9 * (size_t)nx * ny + 8 * (size_t)nx; }

template <class R>
__global__ void __launch_bounds__(kResThreads)
    adj_pair_backward_kernel(const R* ckpt, R* seg, size_t state_elems, int every, long long nsteps, int bufs,
                             const R* lam_final, double* part, AdjConst<R> k) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    __shared__ double red[kResThreads];
    const int nx = k.nx, ny = k.ny, nn = nx * ny, n9 = 9 * nn;
    R* a = reinterpret_cast<R*>(sm_raw);
    R* b = a + n9;
    const int rank = cluster_rank();
    const int node = threadIdx.x;
    const bool live = node < nn;
    const int x = live ? node % nx : 0, y = live ? node / nx : 0;
    const bool bottom = live && y == 0, top = live && y == ny - 1;
    const long long nseg = (nsteps + every - 1) / every;
    const size_t step_elems = pair_elems(nx, ny), seg_elems = step_elems * every;
    auto length = [&](long long s) { return (int)min((long long)every, nsteps - s * every); };

    auto recompute = [&](long long s) {
        const R* c = ckpt + (size_t)s * state_elems;
        for (int e = threadIdx.x; e < n9; e += blockDim.x) a[e] = c[e];
        __syncthreads();
        R* out = seg + (size_t)(s % bufs) * seg_elems;
        res_steps(a, b, length(s), k, [&](long long t, const R* d, const Pull& p, const R* f) {
            R* w = out + (size_t)t * step_elems;
#pragma unroll
            for (int i = 0; i < 9; ++i) w[i * nn + node] = d[i];
            R* e = w + n9 + x;
            if (bottom) {
                e[0] = f[p.o[5]];
                e[nx] = f[p.wb[0]];
                e[2 * nx] = f[p.o[6]];
                e[3 * nx] = f[p.wb[1]];
            }
            if (top) {
                e[4 * nx] = f[p.o[7]];
                e[5 * nx] = f[p.wt[0]];
                e[6 * nx] = f[p.o[8]];
                e[7 * nx] = f[p.wt[1]];
            }
        });
    };

    ParamSums<R> sum;
    Pull p{};
    if (live) p = push_of(nx, ny, x, y);
    auto walk = [&](long long s) {
        const R* in = seg + (size_t)(s % bufs) * seg_elems;
        const int len = length(s);
        struct Step {
            R fb[9], w[8];
        };
        auto load = [&](int j, Step& v) {
            const R* q = in + (size_t)j * step_elems;
#pragma unroll
            for (int i = 0; i < 9; ++i) v.fb[i] = q[i * nn + node];
            const R* e = q + n9 + x;
            if (bottom)
#pragma unroll
                for (int i = 0; i < 4; ++i) v.w[i] = e[i * nx];
            if (top)
#pragma unroll
                for (int i = 4; i < 8; ++i) v.w[i] = e[i * nx];
        };
        // one step's forward part is formed, and the next but one's values
        // arrive, beside the reverse of this one
        Step cur, nxt;
        Forward<R> v{};
        if (live) {
            load(len - 1, cur);
            v = forward_of(cur.fb, k.ref, k.c);
            load(max(len - 2, 0), nxt);
        }
        for (int j = len - 1; j >= 0; --j) {
            if (live) {
                R l[9], m[9];
                if (s == nseg - 1 && j == len - 1)
                    for (int i = 0; i < 9; ++i) l[i] = lam_final[i * nn + node];
                else
                    transpose_at(a, p, k.r, k.rc, l);
                Step far;
                load(max(j - 2, 0), far);
                const Forward<R> next = forward_of(nxt.fb, k.ref, k.c);
                reverse_collide(v, l, k.c, m, sum);
#pragma unroll
                for (int i = 0; i < 9; ++i) b[i * nn + node] = m[i];
                if (bottom) {
                    wall_term(m[5], cur.w[0], cur.w[1], sum.r);
                    wall_term(m[6], cur.w[2], cur.w[3], sum.r);
                }
                if (top) {
                    wall_term(m[7], cur.w[4], cur.w[5], sum.r);
                    wall_term(m[8], cur.w[6], cur.w[7], sum.r);
                }
                cur = nxt;
                nxt = far;
                v = next;
            }
            __syncthreads();
            R* q = a;
            a = b;
            b = q;
        }
    };

    // block 1 recomputes, block 0 walks; every barrier is reached by both
    if (bufs == 2) {
        if (rank == 1) recompute(nseg - 1);
        cluster_barrier();
        for (long long s = nseg - 1; s >= 0; --s) {
            if (rank == 1) {
                if (s > 0) recompute(s - 1);
            } else {
                walk(s);
            }
            cluster_barrier();
        }
    } else {
        for (long long s = nseg - 1; s >= 0; --s) {
            if (rank == 1) recompute(s);
            cluster_barrier();
            if (rank == 0) walk(s);
            cluster_barrier();
        }
    }
    if (rank == 0) write_sums(sum, k, red, part);
}

// One block's nodes of a cluster, dealt out by whole warps, one to each block
// in turn.  each(node, x, y);
// a block's threads cover its share in one round (ONE) or several.
struct ClusterNodes {
    int first, step, nx, x, y;
    __device__ ClusterNodes(int rank, int nx_) : nx(nx_) {
        first = (((int)threadIdx.x >> 5) * (int)gridDim.x + rank) * 32 + ((int)threadIdx.x & 31);
        step = (int)(gridDim.x * blockDim.x);
        y = first / nx;
        x = first - y * nx;
    }
    template <class F> __device__ __forceinline__ void each(int nn, F&& f) const {
        if (first < nn) f(first, x, y);
        for (int node = first + step; node < nn; node += step) f(node, node % nx, node / nx);
    }
};

// The forward pass by a cluster, states (two, in `work`) in global memory: a
// few hundred KB, resident in L2.  J's sums per block go to part[rank].
template <class R>
__global__ void __launch_bounds__(kResThreads)
    adj_cl_forward_kernel(R* ckpt, R* work, size_t state_elems, int every, long long nsteps, R* lam_final,
                          double* part, AdjConst<R> k) {
    __shared__ double red[kResThreads];
    const int nn = k.nx * k.ny, rank = cluster_rank();
    const ClusterNodes mine(rank, k.nx);
    R* a = work;
    R* b = work + state_elems;
    mine.each(nn, [&](int node, int, int) {  // zero deviations
        for (int i = 0; i < 9; ++i) a[i * nn + node] = ckpt[i * nn + node] = R(0);
    });
    cluster_barrier();
    for (long long t = 0; t < nsteps; ++t) {
        R* c = (t + 1) % every == 0 && t + 1 < nsteps ? ckpt + (size_t)((t + 1) / every) * state_elems : nullptr;
        mine.each(nn, [&](int node, int x, int y) {
            R d[9];
            gather_at(a, pull_of(k.nx, k.ny, x, y), k.r, k.rc, d);
            collide<R, MODE_PERIODIC>(d, k.ref, k.c);
            for (int i = 0; i < 9; ++i) {
                b[i * nn + node] = d[i];
                if (c) c[i * nn + node] = d[i];
            }
        });
        cluster_barrier();
        R* q = a;
        a = b;
        b = q;
    }
    double js = 0;
    mine.each(nn, [&](int node, int, int) { js += flow_term(a, nn, node, lam_final, node, k); });
    js = res_block_sum(js, red);
    if (threadIdx.x == 0) part[rank] = js;
}

// The backward walk by a cluster of `gridDim.x` blocks: recompute the
// segment's states from its checkpoint, then per step mu_t = J_C^T lambda_{t+1}
// with lambda_{t+1} = P^T mu_{t+1} gathered on the fly from the previous
// step's mu (lambda_N itself for the first step), so one cluster barrier
// separates the steps.  mu (two buffers) and the segment states are in global
// memory (resident in L2); the cluster barrier (release / acquire at cluster
// scope) orders them.  Every block runs
// the same loop counts, so every barrier is reached by all of them.  Each
// block's parameter sums go to part[rank * 3 + 0..2], added on the host in rank
// order.
template <class R>
__global__ void __launch_bounds__(kResThreads)
    adj_cl_backward_kernel(const R* ckpt, R* seg, size_t state_elems, int every, long long nsteps,
                           const R* lam_final, R* mu0, R* mu1, double* part, AdjConst<R> k) {
    __shared__ double red[kResThreads];
    const int nn = k.nx * k.ny, n9 = 9 * nn;
    const int rank = cluster_rank();
    const int e0 = rank * (int)blockDim.x + (int)threadIdx.x, es = (int)(gridDim.x * blockDim.x);
    const ClusterNodes mine(rank, k.nx);
    ParamSums<R> sum;
    const R* mu_next = nullptr;  // mu of step t + 1 (none before the first backward step)
    R* mu_cur = mu0;
    const long long nseg = (nsteps + every - 1) / every;
    for (long long s = nseg - 1; s >= 0; --s) {
        const long long t0 = s * every;
        const int len = (int)min((long long)every, nsteps - t0);
        const R* c = ckpt + (size_t)s * state_elems;
        for (int e = e0; e < n9; e += es) seg[e] = c[e];
        cluster_barrier();
        for (int j = 1; j < len; ++j) {  // recompute the segment's states
            const R* a = seg + (size_t)(j - 1) * state_elems;
            R* b = seg + (size_t)j * state_elems;
            mine.each(nn, [&](int node, int x, int y) {
                R d[9];
                gather_at(a, pull_of(k.nx, k.ny, x, y), k.r, k.rc, d);
                collide<R, MODE_PERIODIC>(d, k.ref, k.c);
                for (int i = 0; i < 9; ++i) b[i * nn + node] = d[i];
            });
            cluster_barrier();
        }
        for (int j = len - 1; j >= 0; --j) {
            const R* ft = seg + (size_t)j * state_elems;
            mine.each(nn, [&](int node, int x, int y) {
                back_node(ft, mu_next, lam_final, mu_cur, node, x, y, k, sum);
            });
            cluster_barrier();
            mu_next = mu_cur;
            mu_cur = mu_cur == mu0 ? mu1 : mu0;
        }
    }
    write_sums(sum, k, red, part + rank * 3);
}

// Grids of a node per thread of a cluster: each block holds its share in shared
// memory, the columns (or the rows) from rank W (rank H) on, W x H nodes of
// every block but the last as [9][H][W], and reads the others' where they are,
// through the cluster's shared memory.  A step's round trip through L2, with
// the fence that must precede its barrier, is gone.
struct Share {
    int nx, ny, W, H, rank, x0, y0, w, h, lastx;
    bool live;         // this thread has a node:
    int at, x, y, node;  // its place in the block's state, and in the grid
    __device__ Share(int rank_, int nx_, int ny_, int W_, int H_) : nx(nx_), ny(ny_), W(W_), H(H_), rank(rank_) {
        x0 = W < nx ? rank * W : 0;
        y0 = H < ny ? rank * H : 0;
        const bool any = rank == 0 || W < nx || H < ny;
        w = any ? max(0, min(W, nx - x0)) : 0;
        h = any ? max(0, min(H, ny - y0)) : 0;
        lastx = (nx - 1) / W;
        live = (int)threadIdx.x < w * h;
        const int ly = live ? (int)threadIdx.x / w : 0, lx = live ? (int)threadIdx.x - ly * w : 0;
        at = ly * W + lx;
        x = x0 + lx;
        y = y0 + ly;
        node = y * nx + x;
    }
    // byte address, in the cluster's shared memory, of population i at (xx, yy),
    // a neighbour of one of this block's nodes, in the buffers that start at base
    template <class R> __device__ __forceinline__ int address(unsigned base, int i, int yy, int xx) const {
        int r = rank, lx = xx - x0, ly = yy - y0;
        if (lx < 0 || lx >= w) {  // columns: the next block, or around the end
            r = xx == x0 + w && xx != nx ? rank + 1 : xx == x0 - 1 ? rank - 1 : xx == 0 ? 0 : lastx;
            lx = xx - r * W;
        }
        if (ly < 0 || ly >= h) {  // rows
            r = ly < 0 ? rank - 1 : rank + 1;
            ly = yy - r * H;
        }
        unsigned to;
        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"(base), "r"(r));
        return (int)(to + (unsigned)(((i * H + ly) * W + lx) * (int)sizeof(R)));
    }
};

__device__ __forceinline__ float ld_cluster(int a, float) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ double ld_cluster(int a, double) {
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a));
    return v;
}
// The two halves of cluster_barrier, for what is in shared memory.
__device__ __forceinline__ void cluster_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// pull_of and gather_at, transpose_at, through addresses of the cluster's
// shared memory (of buffer 0; off: of another).
template <class At> __device__ __forceinline__ Pull pull_with(int nx, int ny, int x, int y, At at) {
    Pull p;
    const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
    p.bottom = y == 0;
    p.top = y == ny - 1;
    p.wb[0] = p.wb[1] = p.wt[0] = p.wt[1] = 0;
    p.o[0] = at(0, y, x);
    p.o[1] = at(1, y, xm);
    p.o[3] = at(3, y, xp);
    p.o[2] = p.bottom ? at(4, y, x) : at(2, y - 1, x);
    p.o[5] = p.bottom ? at(7, y, x) : at(5, y - 1, xm);
    p.o[6] = p.bottom ? at(8, y, x) : at(6, y - 1, xp);
    if (p.bottom) {
        p.wb[0] = at(8, y, xm);
        p.wb[1] = at(7, y, xp);
    }
    p.o[4] = p.top ? at(2, y, x) : at(4, y + 1, x);
    p.o[7] = p.top ? at(5, y, x) : at(7, y + 1, xp);
    p.o[8] = p.top ? at(6, y, x) : at(8, y + 1, xm);
    if (p.top) {
        p.wt[0] = at(6, y, xp);
        p.wt[1] = at(5, y, xm);
    }
    return p;
}
template <class R> __device__ __forceinline__ void gather_cluster(const Pull& p, int off, R r, R rc, R (&f)[9]) {
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = ld_cluster(p.o[i] + off, R());
    if (p.bottom) {
        f[5] = ln::fma(r, f[5], ln::mul(rc, ld_cluster(p.wb[0] + off, R())));
        f[6] = ln::fma(r, f[6], ln::mul(rc, ld_cluster(p.wb[1] + off, R())));
    }
    if (p.top) {
        f[7] = ln::fma(r, f[7], ln::mul(rc, ld_cluster(p.wt[0] + off, R())));
        f[8] = ln::fma(r, f[8], ln::mul(rc, ld_cluster(p.wt[1] + off, R())));
    }
}
template <class R> __device__ __forceinline__ void transpose_cluster(const Pull& p, int off, R r, R rc, R (&o)[9]) {
#pragma unroll
    for (int i = 0; i < 9; ++i) o[i] = ld_cluster(p.o[i] + off, R());
    if (p.top) {
        o[5] = r * o[5] + rc * ld_cluster(p.wt[0] + off, R());
        o[6] = r * o[6] + rc * ld_cluster(p.wt[1] + off, R());
    }
    if (p.bottom) {
        o[7] = r * o[7] + rc * ld_cluster(p.wb[0] + off, R());
        o[8] = r * o[8] + rc * ld_cluster(p.wb[1] + off, R());
    }
}

// Threads of a block.  168 registers hold what the walk keeps from step to step;
// with 448 threads and 128 registers it spills (20 x 128 2.52 us per backward
// step against 2.19).  us per step forward + backward, against the round trip
// through L2: 20 x 128 1.16 + 2.19, 1.93 + 3.22; 100 x 50 1.39 + 3.63, 2.17 +
// 3.77; 75 x 80 1.22 + 3.22, 2.33 + 4.18; FP64 4 x 64 5.71 + 15.2, 6.07 + 15.8.
// With several nodes per thread the addresses cost more than the round trip
// (128 x 192 6.0 + 13.4 in shared memory; L2 see kClusterNodes).
constexpr int kShareThreads = 384;

// The forward pass, two copies of each block's share.  J's sums per block go to
// part[rank].
template <class R>
__global__ void __launch_bounds__(kShareThreads)
    adj_share_forward_kernel(R* ckpt, size_t state_elems, int every, long long nsteps, R* lam_final, double* part, int W,
                             int H, AdjConst<R> k) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    __shared__ double red[kResThreads];
    const int nx = k.nx, ny = k.ny, nn = nx * ny, ws = W * H, bytes = 9 * ws * (int)sizeof(R);
    const Share q(cluster_rank(), nx, ny, W, H);
    const unsigned base = (unsigned)__cvta_generic_to_shared(sm_raw);
    R* const s = reinterpret_cast<R*>(sm_raw);
    Pull p{};
    if (q.live) {  // zero deviations
        for (int i = 0; i < 9; ++i) s[i * ws + q.at] = ckpt[i * nn + q.node] = R(0);
        p = pull_with(nx, ny, q.x, q.y, [&](int i, int yy, int xx) { return q.template address<R>(base, i, yy, xx); });
    }
    int cur = 0;  // the copy that holds the state
    cluster_arrive();
    cluster_wait();
    for (long long t = 0; t < nsteps; ++t) {
        R d[9];
        if (q.live) {
            gather_cluster(p, cur * bytes, k.r, k.rc, d);
            collide<R, MODE_PERIODIC>(d, k.ref, k.c);
#pragma unroll
            for (int i = 0; i < 9; ++i) s[((cur ^ 1) * 9 + i) * ws + q.at] = d[i];
        }
        cluster_arrive();
        if (q.live && (t + 1) % every == 0 && t + 1 < nsteps) {
            R* c = ckpt + (size_t)((t + 1) / every) * state_elems;
#pragma unroll
            for (int i = 0; i < 9; ++i) c[i * nn + q.node] = d[i];
        }
        cluster_wait();
        cur ^= 1;
    }
    const double js = q.live ? flow_term(s + cur * 9 * ws, ws, q.at, lam_final, q.node, k) : 0.0;
    const double sum = res_block_sum(js, red);
    if (threadIdx.x == 0) part[q.rank] = sum;
}

// The backward walk: recompute the segment's states from its checkpoint, which
// is its state 0, every later one also written to `seg`; then per step mu_t =
// J_C^T lambda_{t+1} with lambda_{t+1} = P^T mu_{t+1} gathered from the blocks'
// shared memory (lambda_N itself for the first step), one cluster barrier per
// step.  The state at t comes from L2: its pulls are loaded a step ahead, and in
// FP32 the collision's forward part is formed while the barrier is on its way.
// The wall terms read it after the barrier's arrival, when another thread may
// already be in the next segment: state 0 is therefore read where nothing writes
// it (the checkpoint), and a later one is rewritten only beyond a further barrier
// (that of a later step of the walk), which its readers arrive at first.  Three
// buffers: mu of the last step, and the two that the recomputation, then the
// walk, alternate with.  Every block runs the same loop counts, so every
// barrier is reached by all of them.  Each block's parameter sums go to
// part[rank * 3 + 0..2], added on the host in rank order.
template <class R>
__global__ void __launch_bounds__(kShareThreads)
    adj_share_backward_kernel(const R* ckpt, R* seg, size_t state_elems, int every, long long nsteps, const R* lam_final,
                              double* part, int W, int H, AdjConst<R> k) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    __shared__ double red[kResThreads];
    constexpr bool kEarly = std::is_same<R, float>::value;
    const int nx = k.nx, ny = k.ny, nn = nx * ny, ws = W * H, bytes = 9 * ws * (int)sizeof(R);
    const Share q(cluster_rank(), nx, ny, W, H);
    const unsigned base = (unsigned)__cvta_generic_to_shared(sm_raw);
    R* const s = reinterpret_cast<R*>(sm_raw);
    auto addr = [&](int i, int yy, int xx) { return q.template address<R>(base, i, yy, xx); };
    ParamSums<R> sum;
    int last = 0, u = 1, v = 2;  // buffers: mu_{t+1}, and two to work in
    const long long nseg = (nsteps + every - 1) / every;
    for (long long sg = nseg - 1; sg >= 0; --sg) {
        const int len = (int)min((long long)every, nsteps - sg * every);
        const R* c = ckpt + (size_t)sg * state_elems;
        if (q.live)
            for (int i = 0; i < 9; ++i) s[(u * 9 + i) * ws + q.at] = c[i * nn + q.node];
        auto state = [&](int j) { return j > 0 ? seg + (size_t)j * state_elems : c; };
        {
            Pull p{};
            if (q.live) p = pull_with(nx, ny, q.x, q.y, addr);
            for (int j = 1; j < len; ++j) {
                cluster_arrive();
                cluster_wait();
                if (q.live) {
                    R* to = seg + (size_t)j * state_elems;
                    R d[9];
                    gather_cluster(p, u * bytes, k.r, k.rc, d);
                    collide<R, MODE_PERIODIC>(d, k.ref, k.c);
#pragma unroll
                    for (int i = 0; i < 9; ++i) s[(v * 9 + i) * ws + q.at] = to[i * nn + q.node] = d[i];
                }
                const int o = u;
                u = v;
                v = o;
            }
        }
        cluster_barrier();  // the segment's states are in global memory
        Pull pf{}, pm{};  // pulls of the state, of mu
        Forward<R> fw{};
        if (q.live) {
            pf = pull_of(nx, ny, q.x, q.y);
            pm = push_with(nx, ny, q.x, q.y, addr);
            if (kEarly) {
                R fb[9];
                gather_at(state(len - 1), pf, k.r, k.rc, fb);
                fw = forward_of(fb, k.ref, k.c);
            }
        }
        for (int j = len - 1; j >= 0; --j) {
            const R* f = state(j);
            R next[9], m[9];  // the pulls of step j - 1; mu_t
            if (q.live) {
                if (kEarly) {
                    gather_at(state(max(j - 1, 0)), pf, k.r, k.rc, next);
                } else {
                    gather_at(f, pf, k.r, k.rc, next);
                    fw = forward_of(next, k.ref, k.c);
                }
                R l[9];
                if (sg == nseg - 1 && j == len - 1)
                    for (int i = 0; i < 9; ++i) l[i] = lam_final[i * nn + q.node];
                else
                    transpose_cluster(pm, last * bytes, k.r, k.rc, l);
                reverse_collide(fw, l, k.c, m, sum);
#pragma unroll
                for (int i = 0; i < 9; ++i) s[(u * 9 + i) * ws + q.at] = m[i];
            }
            cluster_arrive();
            if (q.live) {
                if (pf.bottom) {
                    wall_term(m[5], f[pf.o[5]], f[pf.wb[0]], sum.r);
                    wall_term(m[6], f[pf.o[6]], f[pf.wb[1]], sum.r);
                }
                if (pf.top) {
                    wall_term(m[7], f[pf.o[7]], f[pf.wt[0]], sum.r);
                    wall_term(m[8], f[pf.o[8]], f[pf.wt[1]], sum.r);
                }
                if (kEarly) fw = forward_of(next, k.ref, k.c);
            }
            cluster_wait();
            const int o = last;
            last = u;
            u = o;
        }
    }
    write_sums(sum, k, red, part + q.rank * 3);
}

// Shared memory of the resident forward kernel: two states and the block sum.
size_t res_smem(int nx, int ny, size_t elem) {
    return ((2 * 9 * (size_t)nx * ny * elem + 15) / 16) * 16 + kResThreads * sizeof(double);
}
// Threads of a resident block: one node each, by whole warps.
int res_threads(int nx, int ny) { return std::min(kResThreads, (nx * ny + 31) / 32 * 32); }
constexpr size_t kResSmemCap = 200 * 1024;
// Largest FP32 grid of the cluster kernels (with the states in L2, as below),
// whose 16 blocks cost 0.3 us per thousand nodes and step beyond 8192; one launch per step costs 5 us forward
// and 12 us backward whatever the grid.  Measured, us per step forward +
// backward, cluster / launches: 100 x 50 2.3 + 3.8 / 4.8 + 12.3; 160 x 100
// 3.9 + 7.0 / 5.2 + 12.4; 200 x 160 6.1 + 11.6 / 6.1 + 12.6; 320 x 200
// 9.6 + 20.9 / 5.8 + 14.6.
constexpr int kClusterNodes = 24576;
// Nodes up to which the forward pass of a resident grid stays in one block.
// FP32, one node per thread: 20 x 25 0.63 us per step there (cluster 25 x 41 0.91);
// with two, 10 x 100 1.42.
// FP64, bound by the FP64 pipe: 4 x 64 12.4 us there, 6.5 us in a cluster (one
// warp per SM), where 4 x 32 takes as long.
int block_nodes(size_t elem) { return elem == 8 ? 128 : kResThreads; }

}  // namespace

struct clb_adjoint {
    int nx = 0, ny = 0, storage = 0;
    int64_t nsteps = 0;
    int every = 0;
    size_t elem = 0, state_elems = 0;
    void* ckpt = nullptr;  // checkpoints: state at steps 0, C, 2C, ...
    int nckpt = 0;
    void* seg = nullptr;   // one recomputed segment: C + 1 states
    void* mu0 = nullptr;   // mu of one backward step, mu of the next
    void* lam_final = nullptr;  // lambda_N = dJ/df_N, kept for every backward call
    void* mu = nullptr;
    double* acc = nullptr; // per-block partial sums [4][nb]: r, a, G and J
    int nb = 0;            // blocks of every adjoint launch
    bool resident = false; // resident engine: the forward pass in one block, the backward in one cluster
    bool pair = false;     // ... the backward in a pair of blocks; seg then holds seg_bufs segments of pulled steps
    int seg_bufs = 1;
    int cluster = 0;       // blocks of the backward cluster otherwise (0: not yet launched)
    AdjConst<float> kf;
    AdjConst<double> kd;
    double J = 0;
    double g = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    void* (*alloc)(size_t, void*) = nullptr;
    void (*dealloc)(void*, void*) = nullptr;
    void* alloc_ctx = nullptr;

    void* dalloc(size_t bytes) {
        if (alloc) return alloc(bytes ? bytes : 256, alloc_ctx);
        void* p = nullptr;
        if (cudaMalloc(&p, bytes ? bytes : 256) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        return p;
    }
    void dfree(void* p) {
        if (!p) return;
        if (dealloc)
            dealloc(p, alloc_ctx);
        else
            cudaFree(p);
    }
};

namespace {

template <class R> AdjConst<R>& kconst(clb_adjoint* h);
template <> AdjConst<float>& kconst<float>(clb_adjoint* h) { return h->kf; }
template <> AdjConst<double>& kconst<double>(clb_adjoint* h) { return h->kd; }

int blocks_for(size_t n, int t) { return (int)std::min<size_t>((n + t - 1) / t, 1024); }

template <class R> R* state_at(void* base, size_t state_elems, int64_t k) {
    return static_cast<R*>(base) + (size_t)k * state_elems;
}

// Copy the [4][nb] partial sums to the host and add each row in block order.
cudaError_t sum_partials(clb_adjoint* h, int rows, double* out) {
    std::vector<double> part((size_t)rows * h->nb);
    cudaError_t e = cudaMemcpyAsync(part.data(), h->acc, part.size() * sizeof(double), cudaMemcpyDeviceToHost,
                                    h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return e;
    for (int k = 0; k < rows; ++k) {
        double v = 0;
        for (int b = 0; b < h->nb; ++b) v += part[(size_t)k * h->nb + b];
        out[k] = v;
    }
    return cudaSuccess;
}

// Allow a kernel the shared memory of the largest resident grid.  The limit
// belongs to the kernel for the whole process: one value for every grid, so that
// no other handle (or thread) lowers it between this and the launch.
template <class K> cudaError_t opt_in(K kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResSmemCap);
}

// Launch fn's kernel with its arguments as one cluster of `cl` blocks (more
// than 8 need the non-portable cluster size, which the device may refuse).
template <class K, class... A>
cudaError_t launch_cluster(K kern, int cl, int threads, size_t smem, cudaStream_t st, A... args) {
    if (cl > 8) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cl);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cl;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

// Threads per block of a cluster of cl blocks: a node each, as far as they go.
int cl_threads(const clb_adjoint* h, int cl) {
    const int warps = (h->nx * h->ny + 31) / 32;
    return std::min(kResThreads, 32 * std::max(1, (warps + cl - 1) / cl));
}

// How a cluster of cl blocks shares a grid of a node per thread (one false:
// there are more): by rows, whose nodes are next to each other in global
// memory, or by columns where that makes a node per thread of it, or leaves a
// share smaller by a fifth or more.  us per step forward + backward, by rows and
// by columns: 64 x 64 1.20 + 2.62, 1.42 + 3.66; 100 x 50 (400 nodes by rows, two
// per thread) 2.11 + 4.24, 1.60 + 3.95.
struct Shares {
    int W, H, threads;
    bool one;
    size_t state_bytes;
};
Shares shares_of(const clb_adjoint* h, int cl) {
    const int w = (h->nx + cl - 1) / cl, r = (h->ny + cl - 1) / cl;
    const long long by_columns = (long long)w * h->ny, by_rows = (long long)r * h->nx;
    const bool columns = by_columns < by_rows && (by_rows > kShareThreads || 5 * by_columns <= 4 * by_rows);
    Shares q;
    q.W = columns ? w : h->nx;
    q.H = columns ? h->ny : r;
    const long long nodes = columns ? by_columns : by_rows;
    q.one = nodes <= kShareThreads;
    q.threads = (int)std::min<long long>(kShareThreads, (nodes + 31) / 32 * 32);
    q.state_bytes = (size_t)9 * nodes * h->elem;
    return q;
}
template <class K, class... A>
cudaError_t launch_shares(K kern, int cl, const Shares& q, int copies, cudaStream_t st, A... args) {
    cudaError_t e = opt_in(kern);
    if (e != cudaSuccess) return e;
    return launch_cluster(kern, cl, q.threads, copies * q.state_bytes, st, args...);
}

// Run launch(cl) with the largest cluster the device takes (16 blocks, else
// the portable 8).
template <class F> cudaError_t with_cluster(clb_adjoint* h, F&& launch) {
    if (h->cluster) return launch(h->cluster);
    h->cluster = kClusterMax;
    cudaError_t e = launch(h->cluster);
    if (e != cudaSuccess) {
        cudaGetLastError();
        h->cluster = 8;
        e = launch(h->cluster);
    }
    if (e != cudaSuccess) h->cluster = 0;
    return e;
}

// The forward pass in one block, or in one cluster (resident engine).
template <class R> cudaError_t forward_resident(clb_adjoint* h) {
    int sums = 1;
    cudaError_t e;
    if (h->nx * h->ny <= block_nodes(sizeof(R))) {
        const size_t smem = res_smem(h->nx, h->ny, sizeof(R));
        e = opt_in(adj_res_forward_kernel<R>);
        if (e != cudaSuccess) return e;
        adj_res_forward_kernel<R><<<1, res_threads(h->nx, h->ny), smem, h->stream>>>(
            static_cast<R*>(h->ckpt), h->state_elems, h->every, (long long)h->nsteps, static_cast<R*>(h->lam_final),
            h->acc, kconst<R>(h));
        e = cudaGetLastError();
    } else {
        e = with_cluster(h, [&](int cl) {
            const Shares q = shares_of(h, cl);
            if (q.one)
                return launch_shares(adj_share_forward_kernel<R>, cl, q, 2, h->stream, static_cast<R*>(h->ckpt),
                                     h->state_elems, h->every, (long long)h->nsteps, static_cast<R*>(h->lam_final),
                                     h->acc, q.W, q.H, kconst<R>(h));
            if constexpr (std::is_same<R, double>::value)
                return cudaErrorInvalidValue;  // resident FP64 grids have a node per thread of 8 blocks
            else
                return launch_cluster(adj_cl_forward_kernel<R>, cl, cl_threads(h, cl), 0, h->stream,
                                  static_cast<R*>(h->ckpt), static_cast<R*>(h->seg), h->state_elems, h->every,
                                  (long long)h->nsteps, static_cast<R*>(h->lam_final), h->acc, kconst<R>(h));
        });
        sums = h->cluster;
    }
    double part[kClusterMax] = {};
    if (e == cudaSuccess) e = cudaMemcpyAsync(part, h->acc, sums * sizeof(double), cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return e;
    h->J = 0;
    for (int r = 0; r < sums; ++r) h->J += part[r];  // rank order
    return cudaSuccess;
}

template <class R> cudaError_t launch_cl_backward(clb_adjoint* h, int cl) {
    const Shares q = shares_of(h, cl);
    if (q.one)
        return launch_shares(adj_share_backward_kernel<R>, cl, q, 3, h->stream, static_cast<const R*>(h->ckpt),
                             static_cast<R*>(h->seg), h->state_elems, h->every, (long long)h->nsteps,
                             static_cast<const R*>(h->lam_final), h->acc, q.W, q.H, kconst<R>(h));
    if constexpr (std::is_same<R, double>::value)
        return cudaErrorInvalidValue;  // as in forward_resident
    else
        return launch_cluster(adj_cl_backward_kernel<R>, cl, cl_threads(h, cl), 0, h->stream, static_cast<const R*>(h->ckpt),
                          static_cast<R*>(h->seg), h->state_elems, h->every, (long long)h->nsteps,
                          static_cast<const R*>(h->lam_final), static_cast<R*>(h->mu0), static_cast<R*>(h->mu),
                          h->acc, kconst<R>(h));
}

cudaError_t launch_pair_backward(clb_adjoint* h) {
    using R = float;
    cudaError_t e = opt_in(adj_pair_backward_kernel<R>);
    if (e != cudaSuccess) return e;
    return launch_cluster(adj_pair_backward_kernel<R>, 2, res_threads(h->nx, h->ny), 2 * h->state_elems * sizeof(R), h->stream,
                          static_cast<const R*>(h->ckpt), static_cast<R*>(h->seg), h->state_elems, h->every,
                          (long long)h->nsteps, h->seg_bufs, static_cast<const R*>(h->lam_final), h->acc, kconst<R>(h));
}

template <class R> cudaError_t backward_resident(clb_adjoint* h, double* out3) {
    cudaError_t e = h->pair ? launch_pair_backward(h)
                            : with_cluster(h, [&](int cl) { return launch_cl_backward<R>(h, cl); });
    const int cl = h->pair ? 1 : h->cluster;  // blocks with sums
    double part[3 * kClusterMax];
    if (e == cudaSuccess) e = cudaMemcpyAsync(part, h->acc, 3 * cl * sizeof(double), cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return e;
    for (int q = 0; q < 3; ++q) {
        double v = 0;
        for (int r = 0; r < cl; ++r) v += part[r * 3 + q];  // rank order
        out3[q] = v;
    }
    return cudaSuccess;
}

template <class R> cudaError_t forward_run(clb_adjoint* h) {
    if (h->resident) return forward_resident<R>(h);
    const AdjConst<R>& k = kconst<R>(h);
    const int nb = h->nb;
    R* cur = state_at<R>(h->seg, h->state_elems, 0);
    R* nxt = state_at<R>(h->seg, h->state_elems, 1);
    cudaError_t e = cudaMemsetAsync(cur, 0, h->state_elems * sizeof(R), h->stream);  // f^eq(rho_out, 0)
    for (int64_t t = 0; t < h->nsteps && e == cudaSuccess; ++t) {
        if (t % h->every == 0)
            e = cudaMemcpyAsync(state_at<R>(h->ckpt, h->state_elems, t / h->every), cur, h->state_elems * sizeof(R),
                                cudaMemcpyDeviceToDevice, h->stream);
        if (e != cudaSuccess) break;
        adj_forward_kernel<R><<<nb, kAdjThreads, 0, h->stream>>>(cur, nxt, k);
        e = cudaGetLastError();
        std::swap(cur, nxt);
    }
    if (e != cudaSuccess) return e;
    // final state and J, lambda_N (into lam_final)
    e = cudaMemsetAsync(h->acc, 0, (size_t)4 * nb * sizeof(double), h->stream);
    if (e == cudaSuccess) {
        adj_final_kernel<R><<<nb, kAdjThreads, 0, h->stream>>>(cur, static_cast<R*>(h->lam_final), h->acc, k);
        e = cudaGetLastError();
    }
    double hacc[4];
    if (e == cudaSuccess) e = sum_partials(h, 4, hacc);
    if (e == cudaSuccess) h->J = hacc[3];
    return e;
}

template <class R> cudaError_t backward_run(clb_adjoint* h, double seed, double grad[3]) {
    if (h->resident) {
        double hacc[3];
        cudaError_t e = backward_resident<R>(h, hacc);
        if (e != cudaSuccess) return e;
        grad[0] = seed * hacc[0];
        grad[1] = seed * hacc[1];
        grad[2] = seed * (hacc[2] - 0.5 * h->ny);
        return cudaSuccess;
    }
    const AdjConst<R>& k = kconst<R>(h);
    const int nb = h->nb;
    cudaError_t e = cudaMemsetAsync(h->acc, 0, (size_t)3 * nb * sizeof(double), h->stream);
    const R* mu_next = nullptr;
    R* mu = static_cast<R*>(h->mu0);
    for (int64_t s = (h->nsteps - 1) / h->every; s >= 0 && e == cudaSuccess; --s) {
        const int64_t t0 = s * h->every;
        const int64_t len = std::min<int64_t>(h->every, h->nsteps - t0);
        // recompute the segment's states t0 .. t0+len-1
        e = cudaMemcpyAsync(state_at<R>(h->seg, h->state_elems, 0), state_at<R>(h->ckpt, h->state_elems, s),
                            h->state_elems * sizeof(R), cudaMemcpyDeviceToDevice, h->stream);
        for (int64_t j = 1; j < len && e == cudaSuccess; ++j) {
            adj_forward_kernel<R><<<nb, kAdjThreads, 0, h->stream>>>(state_at<R>(h->seg, h->state_elems, j - 1),
                                                                     state_at<R>(h->seg, h->state_elems, j), k);
            e = cudaGetLastError();
        }
        for (int64_t j = len - 1; j >= 0 && e == cudaSuccess; --j) {
            adj_back_kernel<R><<<nb, kAdjThreads, 0, h->stream>>>(state_at<R>(h->seg, h->state_elems, j), mu_next,
                                                                  static_cast<const R*>(h->lam_final), mu, h->acc, k);
            e = cudaGetLastError();
            mu_next = mu;
            mu = static_cast<R*>(mu == h->mu0 ? h->mu : h->mu0);
        }
    }
    double hacc[3];
    if (e == cudaSuccess) e = sum_partials(h, 3, hacc);
    if (e != cudaSuccess) return e;
    // explicit dependence of J on G: u_x = sum e f / rho - G/2, summed over y
    grad[0] = seed * hacc[0];
    grad[1] = seed * hacc[1];
    grad[2] = seed * (hacc[2] - 0.5 * h->ny);
    return cudaSuccess;
}

template <class R> void fill_consts(AdjConst<R>& k, const SweepArgs& sa, const KC<R>& c, double dsv_da, double dsq_da,
                                    int nx, int ny) {
    k.c = c;
    k.dsv4_da = R(dsv_da / 4.0);
    k.dsq4_da = R(dsq_da / 4.0);
    k.r = R(sa.r);
    k.rc = R(1.0 - sa.r);
    k.ref = R(sa.ref0);
    k.nx = nx;
    k.ny = ny;
}

}  // namespace

extern "C" {

clb_status clb_adjoint_destroy(clb_adjoint* h) {
    if (!h) return CLB_OK;
    if (h->stream) cudaStreamSynchronize(h->stream);
    h->dfree(h->ckpt);
    h->dfree(h->seg);
    h->dfree(h->mu0);
    h->dfree(h->lam_final);
    h->dfree(h->mu);
    h->dfree(h->acc);
    if (h->own_stream && h->stream) cudaStreamDestroy(h->stream);
    delete h;
    return CLB_OK;
}

clb_status clb_adjoint_forward(int nx, int ny, double kn, double a, double r, double g, int64_t nsteps,
                               int checkpoint_every, const clb_opts* opts, clb_adjoint** out, double* J) {
    clb::TraceRange trace_("clb_adjoint_forward");
    if (!out) return (clb_status)set_error(CLB_EINVAL, "clb_adjoint_forward: out is NULL");
    *out = nullptr;
    clb_opts o;
    clb_opts_default(&o);
    if (opts) o = *opts;
    if (nx < 1 || ny < 1 || (long long)nx * ny > (1 << 22) || nsteps < 1 || !(kn > 0) || !(a >= 0) || r > 1 ||
        !std::isfinite(g) || !(o.rho_out > 0))
        return (clb_status)set_error(CLB_EINVAL, "clb_adjoint_forward: argument out of range");
    if (o.storage != CLB_FP64 && o.storage != CLB_FP32_SHIFTED)
        return (clb_status)set_error(CLB_EINVAL, "clb_adjoint_forward: storage must be FP64 or FP32-shifted");
    if ((o.alloc == nullptr) != (o.free == nullptr))
        return (clb_status)set_error(CLB_EINVAL, "clb_adjoint_forward: alloc and free hooks must be given together");
    clb_adjoint* h = new (std::nothrow) clb_adjoint;
    if (!h) return (clb_status)set_error(CLB_ENOMEM, "clb_adjoint_forward: host allocation failed");
    h->nx = nx;
    h->ny = ny;
    h->storage = o.storage;
    h->nsteps = nsteps;
    h->every = checkpoint_every > 0 ? checkpoint_every : (int)std::ceil(std::sqrt((double)nsteps));
    h->elem = o.storage == CLB_FP64 ? 8 : 4;
    h->state_elems = (size_t)9 * nx * ny;
    h->nckpt = (int)((nsteps + h->every - 1) / h->every);
    h->g = g;
    h->alloc = o.alloc;
    h->dealloc = o.free;
    h->alloc_ctx = o.alloc_ctx;
    // constants: s_v, s_q (Eq. 18, 21) and their derivatives with respect to a
    SweepArgs sa{};
    sa.s3 = o.s3;
    sa.s8 = o.s8;
    rates_at(kn, ny, a, o.b2, &sa.sv, &sa.sq);
    sa.rate_A = 1.0;
    sa.r = r >= 0 ? r : r_from_sigma(o.sigma);
    sa.gx = g;
    sa.ref0 = o.rho_out;  // stored values are deviations from w_i rho_out in both precisions
    sa.store_scale = 1.0;
    derive_constants(sa);
    const double c6 = std::sqrt(6.0 / 3.14159265358979323846) * ny;
    const double tau = c6 * kn / (1.0 + a * kn);
    const double dtau_da = -c6 * kn * kn / ((1.0 + a * kn) * (1.0 + a * kn));
    const double dsv_da = -sa.sv * sa.sv * dtau_da;
    const double dinvsq_dtau = -3.0 / (16.0 * tau * tau) + 3.14159265358979323846 * o.b2 / 4.0;
    const double dsq_da = -sa.sq * sa.sq * dinvsq_dtau * dtau_da;
    fill_consts(h->kf, sa, sa.kf, dsv_da, dsq_da, nx, ny);
    fill_consts(h->kd, sa, sa.kd, dsv_da, dsq_da, nx, ny);
    if (o.stream) {
        h->stream = static_cast<cudaStream_t>(o.stream);
    } else if (cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking) == cudaSuccess) {
        h->own_stream = true;
    } else {
        cudaError_t e = cudaGetLastError();
        delete h;
        return (clb_status)set_error(CLB_ECUDA, "clb_adjoint_forward: stream: %s", cudaGetErrorString(e));
    }
    const size_t sb = h->state_elems * h->elem;
    h->ckpt = h->dalloc(sb * h->nckpt);
    h->mu0 = h->dalloc(sb);
    h->lam_final = h->dalloc(sb);
    h->mu = h->dalloc(sb);
    h->nb = blocks_for((size_t)nx * ny, kAdjThreads);
    h->acc = static_cast<double*>(h->dalloc(std::max<size_t>(4 * (size_t)h->nb, 3 * kClusterMax) * sizeof(double)));
    // (the segment comes last: it may take less where memory is short)
    // one launch per pass, unless opts->pipeline asks for one launch per step
    // (1), while that is faster than filling the GPU in each of two or three
    // launches per step: see the rule's figures at kClusterNodes
    h->resident = o.pipeline != 1 && (res_smem(nx, ny, h->elem) <= kResSmemCap ||
                                      (h->storage == CLB_FP32_SHIFTED && (long long)nx * ny <= kClusterNodes));
    // a pair of blocks for FP32 grids of one node per thread, with two
    // segments in memory, or one where the allocator refuses the second; a
    // cluster, whose segment is plain states, where it refuses that too
    h->pair = h->resident && h->storage == CLB_FP32_SHIFTED && nx * ny <= kResThreads;
    if (h->pair) {
        const size_t one = pair_elems(nx, ny) * h->elem * h->every;
        h->seg_bufs = h->nckpt > 1 ? 2 : 1;
        h->seg = h->dalloc(one * h->seg_bufs);
        if (!h->seg && h->seg_bufs == 2) {
            h->seg_bufs = 1;
            h->seg = h->dalloc(one);
        }
        h->pair = h->seg != nullptr;
    }
    if (!h->seg) h->seg = h->dalloc(sb * (h->every + 1));
    if (!h->ckpt || !h->seg || !h->mu0 || !h->lam_final || !h->mu || !h->acc) {
        clb_adjoint_destroy(h);
        return (clb_status)set_error(CLB_ENOMEM, "clb_adjoint_forward: device allocation failed");
    }
    cudaError_t e = h->storage == CLB_FP64 ? forward_run<double>(h) : forward_run<float>(h);
    if (e != cudaSuccess) {
        clb_adjoint_destroy(h);
        return (clb_status)set_error(CLB_ECUDA, "clb_adjoint_forward: %s", cudaGetErrorString(e));
    }
    if (J) *J = h->J;
    *out = h;
    return CLB_OK;
}

clb_status clb_adjoint_backward(clb_adjoint* h, double seed, double grad[3]) {
    clb::TraceRange trace_("clb_adjoint_backward");
    if (!h || !grad) return (clb_status)set_error(CLB_EINVAL, "clb_adjoint_backward: NULL argument");
    cudaError_t e = h->storage == CLB_FP64 ? backward_run<double>(h, seed, grad) : backward_run<float>(h, seed, grad);
    if (e != cudaSuccess) return (clb_status)set_error(CLB_ECUDA, "clb_adjoint_backward: %s", cudaGetErrorString(e));
    return CLB_OK;
}

// Q = J / (3 G ny^2 sqrt(1/6)): the normalised flow rate of Sec. 3.1 with
// RT = 1/3, p = rho0 RT and F = rho0 G.
static double q_norm_of(const clb_adjoint* h) { return 3.0 * h->g * (double)h->ny * h->ny * std::sqrt(1.0 / 6.0); }

clb_status clb_adjoint_q(const clb_adjoint* h, double* q) {
    if (!h || !q) return (clb_status)set_error(CLB_EINVAL, "clb_adjoint_q: NULL argument");
    if (h->g == 0) return (clb_status)set_error(CLB_EINVAL, "clb_adjoint_q: Q is undefined for G = 0");
    *q = h->J / q_norm_of(h);
    return CLB_OK;
}

clb_status clb_adjoint_q_backward(clb_adjoint* h, double seed, double grad[3]) {
    clb::TraceRange trace_("clb_adjoint_q_backward");
    if (!h || !grad) return (clb_status)set_error(CLB_EINVAL, "clb_adjoint_q_backward: NULL argument");
    if (h->g == 0) return (clb_status)set_error(CLB_EINVAL, "clb_adjoint_q_backward: Q is undefined for G = 0");
    double dj[3];
    cudaError_t e = h->storage == CLB_FP64 ? backward_run<double>(h, 1.0, dj) : backward_run<float>(h, 1.0, dj);
    if (e != cudaSuccess) return (clb_status)set_error(CLB_ECUDA, "clb_adjoint_q_backward: %s", cudaGetErrorString(e));
    // dQ/dtheta = (dJ/dtheta) / norm, and for G also the normalisation's own -Q/G
    const double norm = q_norm_of(h), q = h->J / norm;
    grad[0] = seed * (dj[0] / norm);
    grad[1] = seed * (dj[1] / norm);
    grad[2] = seed * (dj[2] / norm - q / h->g);
    return CLB_OK;
}

}  // extern "C"
