// The adjoint of slr_alpha.cu with one warp per box, for networks of few inputs.
//
// With Q = d + 1 columns per equation a lane holds whole rows of the symbolic
// state in registers (row p = lane + 32 j), so that a layer's product, its
// concrete bounds and its relaxation (forward), or its product and the
// relaxation's adjoint (backward), are one pass without exchange: only the
// product's inputs, n rows of 2 QP floats, go through shared memory, where
// every lane reads the same row (a broadcast of QP / 2 16-byte loads for
// 2 QP RPL FMAs).  Boxes never wait for one another: the phases of a box are
// separated by warp barriers.  The hidden layers' pre-activation equations are
// kept in global memory (coalesced 512-byte accesses; the boxes in flight,
// some ten MB, stay in L2) and read once by the backward sweep.  The weights
// are staged once per CTA, row stride odd, so that both directions read them
// without bank conflicts.
//
// What bounds it: issue slots (65 % active at 27 warps per SM; the packed FMAs
// are a quarter of the instructions, the rest are the loads, the repeated and
// absolute weights and the relaxation's arithmetic).  The block form spends its
// time on scalar shared-memory loads (two per FMA pair) and on barriers between
// phases of a few boxes.  5-6x50-5 network, block form -> this one: 8,192 boxes
// with weight gradients 1.65 -> 0.55 ms, 1,000 boxes at supplied slopes 261 -> 101 us,
// one box 131 -> 87 us, 4,096 boxes' slopes over 20 Adam steps (the sound bounds of
// every step included) 13.9 -> 4.95 ms; 2-3x32-1, 12,000 boxes 467 -> 216 us.  No
// shape of its range was slower (one box to 12,000, widths 8 to 128), so the
// block form serves only networks outside it: more inputs (a row no longer fits
// a lane's registers), wider layers, or weights beyond shared memory.
//
// One block per SM, whose warps share one copy of the weights, and as few of
// them take boxes as keep the number of rounds: the rounds are full, whatever
// the number of boxes.  (Three blocks of eight warps per SM, filled one after
// another, left 4,096 boxes a second round of 448 boxes on a third of the SMs:
// 196 -> 166 us a pass without that; 100 boxes ran on 13 SMs: 114 -> 93 us, with
// weight gradients, seven blocks of 16, 250 -> 169 us; 8,192 boxes with weight
// gradients on 18 warps in three rounds instead of 16 in four 606 -> 550 us.)
//
// Weight gradients are sums over boxes: the warps of a CTA meet at each layer
// and the block adds all its boxes' outer products into accumulators in
// shared memory, each element owned by one thread; one global atomic per
// element and CTA at the end.
//
// Every row bound, slope, slope gradient and box gradient is the sum of
// slr_alpha.cu in the same order, bit for bit.
#include <cstdint>

#include "slr_adj_common.cuh"
#include "slr_eval.cuh"
#include "slr_kernels.h"

namespace slr {

namespace {

// The thread's rows of one layer: equations U, L in columns 0..d-1 and, last, QP - 1.
template <int QP, int RPL>
struct AdjRows {
    float u[RPL][QP], l[RPL][QP];
};

struct RowScal {
    float ll, ul, lu, uu;
};

// Concrete bounds of both equations of one row (column order as stored; the
// columns between d and QP - 1 are zeros).
template <int QP>
__device__ __forceinline__ RowScal row_scal(const float (&u)[QP], const float (&l)[QP]) {
    float su = 0.f, sl = 0.f;
#pragma unroll
    for (int c = 0; c + 1 < QP; ++c) {
        su = __fadd_rn(su, fabsf(u[c]));
        sl = __fadd_rn(sl, fabsf(l[c]));
    }
    RowScal s;
    s.ll = __fsub_rn(l[QP - 1], sl);
    s.ul = __fadd_rn(l[QP - 1], sl);
    s.lu = __fsub_rn(u[QP - 1], su);
    s.uu = __fadd_rn(u[QP - 1], su);
    return s;
}

__device__ __forceinline__ float default_slope(const RowScal &s) {
    return s.ll < 0.f && s.uu > 0.f && s.ul > 0.f ? s.ul / (s.ul - s.ll) : 0.f;
}

// Relaxed row (Eq. 1) as centre x[0..QP) and radius x[QP..2QP).
template <int QP>
__device__ __forceinline__ void relax_to(const float (&u)[QP], const float (&l)[QP], const RowScal &s, float al,
                                         float (&x)[2 * QP]) {
    const bool on = s.ll >= 0.f, off = !on && s.uu <= 0.f;
    const bool chord = !on && !off && !(s.lu >= 0.f);
    const float sg = chord ? s.uu / (s.uu - s.lu) : 1.f;
#pragma unroll
    for (int c = 0; c < QP; ++c) {
        float uh = u[c], lh = l[c];
        if (chord) uh = __fmul_rn(sg, c == QP - 1 ? __fsub_rn(u[c], s.lu) : u[c]);
        if (!on) lh = s.ul > 0.f ? __fmul_rn(al, l[c]) : 0.f;
        if (off) uh = lh = 0.f;
        x[c] = __fmul_rn(0.5f, __fadd_rn(uh, lh));
        x[QP + c] = __fmul_rn(0.5f, __fsub_rn(uh, lh));
    }
}

template <int QP>
__device__ __forceinline__ void put_row(float *to, const float (&x)[2 * QP]) {
#pragma unroll
    for (int q = 0; q < QP / 2; ++q)
        reinterpret_cast<float4 *>(to)[q] = make_float4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]);
}

// Sums over the rows k < n of X: a += w C, b += |w| R, w the weight of row k
// for the thread's row j at w0[j] + k * step.
template <int QP, int RPL>
__device__ __forceinline__ void row_products(const float *X, int n, const float *const (&w0)[RPL], int step,
                                             float (&a)[RPL][QP], float (&b)[RPL][QP]) {
    f32x2 pa[RPL][QP / 2], pb[RPL][QP / 2];
#pragma unroll
    for (int j = 0; j < RPL; ++j)
#pragma unroll
        for (int c = 0; c < QP / 2; ++c) pa[j][c] = pb[j][c] = 0ull;
    const uint32_t x0 = (uint32_t)__cvta_generic_to_shared(X);
#pragma unroll(QP <= 8 ? 2 : 1)
    for (int k = 0; k < n; ++k) {
        f32x2 x[QP];
#pragma unroll
        for (int q = 0; q < QP / 2; ++q) {
            f32x2 v[2];
            lds2x2(x0 + (uint32_t)(k * 2 * QP + 4 * q) * 4u, v);
            x[2 * q] = v[0];
            x[2 * q + 1] = v[1];
        }
#pragma unroll
        for (int j = 0; j < RPL; ++j) {
            const float w = w0[j][k * step];
            const f32x2 ww = pack2(w, w), wa = ww & 0x7fffffff7fffffffull;
#pragma unroll
            for (int c = 0; c < QP / 2; ++c) {
                pa[j][c] = fma2(ww, x[c], pa[j][c]);
                pb[j][c] = fma2(wa, x[QP / 2 + c], pb[j][c]);
            }
        }
    }
#pragma unroll
    for (int j = 0; j < RPL; ++j)
#pragma unroll
        for (int c = 0; c < QP / 2; ++c) {
            unpack2(pa[j][c], a[j][2 * c], a[j][2 * c + 1]);
            unpack2(pb[j][c], b[j][2 * c], b[j][2 * c + 1]);
        }
}

// Adds to acc[i * ld + p] (i < n_in, p < n_out) the boxes' products
// sum_c gC[p] C[i] + sgn(w) gR[p] R[i] and to accb[p] the sums of gC's
// constants: G and X hold the boxes' rows, `stride` floats apart.
template <int QP>
__device__ __forceinline__ void weight_products(const float *X, const float *G, int stride, int nbox, const float *W,
                                                float *acc, float *accb, int ld, int n_in, int n_out) {
    constexpr int TI = QP <= 12 ? 4 : 2, TP = 2;
    const int gp = (n_out + TP - 1) / TP, gi = (n_in + TI - 1) / TI;
    for (int t = threadIdx.x; t < gp * gi; t += blockDim.x) {
        const int ti = t / gp;
        const int i0 = ti * TI, p0 = (t - ti * gp) * TP;
        float s1[TI][TP], s2[TI][TP];
#pragma unroll
        for (int i = 0; i < TI; ++i)
#pragma unroll
            for (int p = 0; p < TP; ++p) s1[i][p] = s2[i][p] = 0.f;
        for (int b = 0; b < nbox; ++b) {
            // (rows past the end read the last row: their sums are not kept)
#pragma unroll
            for (int q = 0; q < QP / 2; ++q) {
                float4 g[TP], x[TI];
#pragma unroll
                for (int p = 0; p < TP; ++p)
                    g[p] = reinterpret_cast<const float4 *>(G + b * stride + min(p0 + p, n_out - 1) * 2 * QP)[q];
#pragma unroll
                for (int i = 0; i < TI; ++i)
                    x[i] = reinterpret_cast<const float4 *>(X + b * stride + min(i0 + i, n_in - 1) * 2 * QP)[q];
#pragma unroll
                for (int i = 0; i < TI; ++i)
#pragma unroll
                    for (int p = 0; p < TP; ++p) {
                        const float gv[4] = {g[p].x, g[p].y, g[p].z, g[p].w};
                        const float xv[4] = {x[i].x, x[i].y, x[i].z, x[i].w};
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            if (4 * q + e < QP) s1[i][p] = fmaf(gv[e], xv[e], s1[i][p]);
                            else s2[i][p] = fmaf(gv[e], xv[e], s2[i][p]);
                        }
                    }
            }
        }
#pragma unroll
        for (int i = 0; i < TI; ++i)
#pragma unroll
            for (int p = 0; p < TP; ++p)
                if (i0 + i < n_in && p0 + p < n_out) {
                    const int o = (i0 + i) * ld + p0 + p;
                    acc[o] += fmaf(sgnf(W[o]), s2[i][p], s1[i][p]);
                }
    }
    for (int p = threadIdx.x; p < n_out; p += blockDim.x) {
        float s = 0.f;
        for (int b = 0; b < nbox; ++b) s += G[b * stride + p * 2 * QP + QP - 1];
        accb[p] += s;
    }
}

// Most threads of a block (one block per SM): as many warps as the registers
// allow with little spilling (5-6x50-5, 20,000 boxes: 28 warps at 72 registers
// 590 us, 24 at 80 637 us).
constexpr int adj_threads(int QP, int RPL, bool w) {
    return w ? (RPL > 2 || QP == 4 ? 512 : 640) : (RPL > 2 ? 256 : (QP <= 6 ? 896 : 768));
}

template <int QP, int RPL, bool kW>
__global__ void __launch_bounds__(adj_threads(QP, RPL, kW), 1)
adj_warp_kernel(const AdjArgs a, const AdjWarpPlan pl, float *chk) {
    extern __shared__ __align__(16) float smem_aw[];
    const NetParams<float> &net = a.net;
    const int K = net.K, d = net.d, R = net.R;
    const int H = (int)a.H;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    float *const sw = smem_aw;                      // weights and biases (pl.w_off, pl.b_off)
    float *const sacc = smem_aw + pl.head;          // kW: their gradients, laid out alike
    float *const boxes = smem_aw + (kW ? 2 : 1) * pl.head;
    const int stride = pl.box[kW ? 1 : 0];
    float *const mine = boxes + warp * stride;
    float *const X = mine;                          // rows of the product's inputs
    float *const G = kW ? mine + pl.rows : mine;    // adjoint rows (X's place where X is not kept)
    float *const sm = mine + (kW ? 2 : 1) * pl.rows, *const sr = sm + QP;
    float *const lo = sr + QP, *const hi = lo + R, *const glo = hi + R, *const ghi = glo + R;
    float4 *const ck = reinterpret_cast<float4 *>(chk) +
                       ((size_t)blockIdx.x * pl.act + warp) * (K - 1) * RPL * (QP / 2) * 32 + lane;

    for (int k = 0; k < K; ++k) {
        const int n_in = net.n[k], n_out = net.n[k + 1], ld = pl.w_ld[k];
        float *w = sw + pl.w_off[k];
        if (k == 0) {
            for (int t = threadIdx.x; t < n_in * n_out; t += blockDim.x) w[t] = net.W0[t];   // n1 x d, row-major
        } else {
            for (int i = warp; i < n_in; i += nw)
                for (int p = lane; p < n_out; p += 32) w[i * ld + p] = net.Wt[k][i * n_out + p];
        }
        for (int p = threadIdx.x; p < n_out; p += blockDim.x) sw[pl.b_off[k] + p] = net.b[k][p];
    }
    if (kW)
        for (int t = threadIdx.x; t < pl.head; t += blockDim.x) sacc[t] = 0.f;
    __syncthreads();

    int64_t n = a.n;
    if (a.count != nullptr) {
        const int64_t c = (int64_t)*a.count;
        n = c < n ? c : n;
    }
    // kW: neighbouring boxes to a block; else boxes go to the blocks first, then to
    // their warps, so that few boxes (a.count) and the last round's spread over the SMs
    const int64_t first = kW ? (int64_t)blockIdx.x * pl.act : blockIdx.x;
    for (int64_t pos0 = first; pos0 < n; pos0 += (int64_t)gridDim.x * pl.act) {
        const int64_t pos = kW ? pos0 + warp : pos0 + (int64_t)warp * gridDim.x;
        const bool live = warp < pl.act && pos < n;
        const int nbox = n - pos0 < pl.act ? (int)(n - pos0) : pl.act;   // kW: the block's boxes
        if (!kW && !live) continue;
        AdjRows<QP, RPL> rw;
        if (live) {
            // ---- the box: centre and radius (Sec. 2.2 bisection for path codes) ----
            const BoxSource &src = a.src;
            if (lane < d) {
                const int64_t idx = src.index != nullptr ? src.index[pos] : pos;
                double m64, r64;
                if (src.mode == 0) {
                    unsigned long long kk;
                    int c;
                    code_dim(src, src.codes[idx], lane, kk, c);
                    const double w = src.root_w[lane];
                    r64 = w * pow2_neg(c + 1);
                    m64 = src.root_lo[lane] + w * ((double)(2 * kk + 1) * pow2_neg(c + 1));
                } else {
                    const double blo = (double)src.lo[idx * d + lane];
                    const double bhi = (double)src.hi[idx * d + lane];
                    m64 = 0.5 * (blo + bhi);
                    r64 = 0.5 * (bhi - blo);
                }
                sm[lane] = (float)m64;
                sr[lane] = (float)r64;
            }
            __syncwarp();

            // ---- layer 1: U = L = [W_1 diag(r) | W_1 m + b_1] ----
#pragma unroll
            for (int j = 0; j < RPL; ++j) {
                const int p = lane + 32 * j;
                const bool in = p < net.n[1];
                const float *w = sw + pl.w_off[0] + (in ? p : 0) * d;
                float v = sw[pl.b_off[0] + (in ? p : 0)];
#pragma unroll
                for (int c = 0; c + 1 < QP; ++c) {
                    float t = 0.f;
                    if (c < d) {
                        t = __fmul_rn(w[c], sr[c]);
                        v = fmaf(w[c], sm[c], v);
                    }
                    rw.u[j][c] = rw.l[j][c] = t;
                }
                rw.u[j][QP - 1] = rw.l[j][QP - 1] = v;
            }
            // ---- hidden layers: bounds, slopes, relaxation, product ----
            int off = 0;
            for (int k = 1; k < K; ++k) {
                const int n_in = net.n[k], n_out = net.n[k + 1];
                if (k > 1) __syncwarp();            // the previous product has read X
#pragma unroll
                for (int j = 0; j < RPL; ++j) {
                    const int p = lane + 32 * j;
                    const RowScal s = row_scal<QP>(rw.u[j], rw.l[j]);
                    float al = default_slope(s);
                    if (p < n_in) {
                        if (a.alpha_mode == kAlphaFree) al = fminf(fmaxf(a.alpha[pos * H + off + p], 0.f), 1.f);
                        else if (a.alpha_mode == kAlphaInit) a.alpha[pos * H + off + p] = al;
                        float4 *c4 = ck + (size_t)((k - 1) * RPL + j) * (QP / 2) * 32;
                        float t[2 * QP];
#pragma unroll
                        for (int c = 0; c < QP; ++c) {
                            t[c] = rw.u[j][c];
                            t[QP + c] = rw.l[j][c];
                        }
#pragma unroll
                        for (int q = 0; q < QP / 2; ++q)
                            c4[q * 32] = make_float4(t[4 * q], t[4 * q + 1], t[4 * q + 2], t[4 * q + 3]);
                        relax_to<QP>(rw.u[j], rw.l[j], s, al, t);
                        put_row<QP>(X + p * 2 * QP, t);
                    }
                }
                off += n_in;
                __syncwarp();
                const float *w0[RPL];
#pragma unroll
                for (int j = 0; j < RPL; ++j) w0[j] = sw + pl.w_off[k] + (lane + 32 * j < n_out ? lane + 32 * j : 0);
                float cc[RPL][QP], rr[RPL][QP];
                row_products<QP, RPL>(X, n_in, w0, pl.w_ld[k], cc, rr);
#pragma unroll
                for (int j = 0; j < RPL; ++j) {
                    const float bp = sw[pl.b_off[k] + (lane + 32 * j < n_out ? lane + 32 * j : 0)];
#pragma unroll
                    for (int c = 0; c < QP; ++c) {
                        const float cv = c == QP - 1 ? __fadd_rn(cc[j][c], bp) : cc[j][c];
                        rw.u[j][c] = __fadd_rn(cv, rr[j][c]);
                        rw.l[j][c] = __fsub_rn(cv, rr[j][c]);
                    }
                }
            }
            // ---- the property rows' bounds and their upstream adjoints ----
            __syncwarp();                           // the last product has read X (G's place)
#pragma unroll
            for (int j = 0; j < RPL; ++j) {
                const int r = lane + 32 * j;
                const RowScal s = row_scal<QP>(rw.u[j], rw.l[j]);
                if (r < R) {
                    lo[r] = s.ll;
                    hi[r] = s.uu;
                    if (a.row_lo != nullptr) {
                        a.row_lo[pos * R + r] = s.ll;
                        a.row_hi[pos * R + r] = s.uu;
                    }
                    if (a.g_lo != nullptr) {
                        glo[r] = a.g_lo[pos * R + r];
                        ghi[r] = a.g_hi[pos * R + r];
                    }
                }
            }
            __syncwarp();
            if (a.g_lo == nullptr && lane == 0) {
                const int8_t dir = (a.alpha_mode == kAlphaInit || a.dir == nullptr) ? 0 : a.dir[pos];
                const int8_t got = decision_grad(net, lo, hi, glo, ghi, dir);
                if (dir == 0 && a.dir != nullptr) a.dir[pos] = got;
            }
            __syncwarp();
            // d lo = d (L_d - sum |L_c|), d hi = d (U_d + sum |U_c|), as (gU + gL, gU - gL)
#pragma unroll
            for (int j = 0; j < RPL; ++j) {
                const int r = lane + 32 * j;
                if (r < R) {
                    const float gl = glo[r], gh = ghi[r];
                    float t[2 * QP];
#pragma unroll
                    for (int c = 0; c < QP; ++c) {
                        const float u = c == QP - 1 ? gh : __fmul_rn(gh, sgnf(rw.u[j][c]));
                        const float l = c == QP - 1 ? gl : __fmul_rn(-gl, sgnf(rw.l[j][c]));
                        t[c] = __fadd_rn(u, l);
                        t[QP + c] = __fsub_rn(u, l);
                    }
                    put_row<QP>(G + r * 2 * QP, t);
                }
            }
            __syncwarp();
        }

        // ---- backward sweep: product k maps hidden layer k to layer k + 1 ----
        int off = H;
        for (int k = K - 1; k >= 1; --k) {
            const int n_in = net.n[k], n_out = net.n[k + 1];
            off -= n_in;
            if (live) {
                // the layer's equations
#pragma unroll
                for (int j = 0; j < RPL; ++j) {
                    const float4 *c4 = ck + (size_t)((k - 1) * RPL + j) * (QP / 2) * 32;
                    float t[2 * QP];
#pragma unroll
                    for (int q = 0; q < QP / 2; ++q) {
                        const float4 v = lane + 32 * j < n_in ? c4[q * 32] : make_float4(0.f, 0.f, 0.f, 0.f);
                        t[4 * q] = v.x;
                        t[4 * q + 1] = v.y;
                        t[4 * q + 2] = v.z;
                        t[4 * q + 3] = v.w;
                    }
#pragma unroll
                    for (int c = 0; c < QP; ++c) {
                        rw.u[j][c] = t[c];
                        rw.l[j][c] = t[QP + c];
                    }
                }
            }
            if (kW) {
                if (live) {
#pragma unroll
                    for (int j = 0; j < RPL; ++j) {
                        const int p = lane + 32 * j;
                        if (p < n_in) {
                            const RowScal s = row_scal<QP>(rw.u[j], rw.l[j]);
                            const float al = a.alpha_mode == kAlphaDefault
                                                 ? default_slope(s)
                                                 : fminf(fmaxf(a.alpha[pos * H + off + p], 0.f), 1.f);
                            float t[2 * QP];
                            relax_to<QP>(rw.u[j], rw.l[j], s, al, t);
                            put_row<QP>(X + p * 2 * QP, t);
                        }
                    }
                }
                __syncthreads();
                weight_products<QP>(boxes, boxes + pl.rows, stride, nbox, sw + pl.w_off[k], sacc + pl.w_off[k],
                                    sacc + pl.b_off[k], pl.w_ld[k], n_in, n_out);
                __syncthreads();
            }
            if (live) {
                // (W^T gC', |W|^T gR')
                const float *w0[RPL];
#pragma unroll
                for (int j = 0; j < RPL; ++j)
                    w0[j] = sw + pl.w_off[k] + (lane + 32 * j < n_in ? lane + 32 * j : 0) * pl.w_ld[k];
                float gx[RPL][QP], gy[RPL][QP];
                row_products<QP, RPL>(G, n_out, w0, 1, gx, gy);
                __syncwarp();
                // through the relaxation (Eq. 1)
#pragma unroll
                for (int j = 0; j < RPL; ++j) {
                    const int p = lane + 32 * j;
                    if (p < n_in) {
                        const float(&u)[QP] = rw.u[j];
                        const float(&l)[QP] = rw.l[j];
                        const RowScal s = row_scal<QP>(u, l);
                        const float ll = s.ll, ul = s.ul, lu = s.lu, uu = s.uu;
                        const int64_t ai = pos * H + off + p;
                        const float al = a.alpha_mode == kAlphaFree ? fminf(fmaxf(a.alpha[ai], 0.f), 1.f)
                                                                    : default_slope(s);
                        float gu[QP], gl[QP], oU[QP], oL[QP];
#pragma unroll
                        for (int c = 0; c < QP; ++c) {
                            gu[c] = __fmul_rn(0.5f, __fadd_rn(gx[j][c], gy[j][c]));
                            gl[c] = __fmul_rn(0.5f, __fsub_rn(gx[j][c], gy[j][c]));
                            oU[c] = gu[c];
                            oL[c] = gl[c];
                        }
                        float g_alpha = 0.f;
                        if (!(ll >= 0.f)) {
                            if (uu <= 0.f) {
#pragma unroll
                                for (int c = 0; c < QP; ++c) oU[c] = oL[c] = 0.f;
                            } else {
                                // upper: identity (lu >= 0) or chord sg (U - lu), sg = uu / (uu - lu)
                                if (!(lu >= 0.f)) {
                                    const float den = uu - lu;
                                    const float sg = uu / den;
                                    float g_s = -lu * gu[QP - 1];
#pragma unroll
                                    for (int c = 0; c < QP; ++c) g_s = fmaf(gu[c], u[c], g_s);
                                    const float g_uu = g_s * (-lu) / (den * den);
                                    const float g_lu = g_s * uu / (den * den) - sg * gu[QP - 1];
#pragma unroll
                                    for (int c = 0; c + 1 < QP; ++c)
                                        oU[c] = sg * gu[c] + (g_uu - g_lu) * sgnf(u[c]);
                                    oU[QP - 1] = sg * gu[QP - 1] + g_uu + g_lu;
                                }
                                // lower: slope * L (ul > 0) or 0
                                if (ul > 0.f) {
#pragma unroll
                                    for (int c = 0; c < QP; ++c) g_alpha = fmaf(gl[c], l[c], g_alpha);
#pragma unroll
                                    for (int c = 0; c < QP; ++c) oL[c] = __fmul_rn(al, gl[c]);
                                    if (a.alpha_mode == kAlphaDefault) {
                                        // slope ul / (ul - ll) depends on the box through (ll, ul)
                                        const float den = ul - ll;
                                        const float g_ul = g_alpha * (-ll) / (den * den);
                                        const float g_ll = g_alpha * ul / (den * den);
#pragma unroll
                                        for (int c = 0; c + 1 < QP; ++c) oL[c] += (g_ul - g_ll) * sgnf(l[c]);
                                        oL[QP - 1] += g_ul + g_ll;
                                    }
                                } else {
#pragma unroll
                                    for (int c = 0; c < QP; ++c) oL[c] = 0.f;
                                }
                            }
                        }
                        if (a.d_alpha != nullptr) a.d_alpha[ai] = g_alpha;
                        if (a.adam_t > 0 && a.alpha_mode != kAlphaDefault) a.alpha[ai] = adam_slope(a, ai, al, g_alpha);
                        float t[2 * QP];
#pragma unroll
                        for (int c = 0; c < QP; ++c) {
                            t[c] = __fadd_rn(oU[c], oL[c]);
                            t[QP + c] = __fsub_rn(oU[c], oL[c]);
                        }
                        put_row<QP>(G + p * 2 * QP, t);
                    }
                }
                __syncwarp();
            }
        }

        // ---- layer 1: G holds gU + gL in its first QP columns ----
        const int n1 = net.n[1];
        const float *W0 = sw + pl.w_off[0];
        if (live) {
            if (lane < d && (a.d_lo != nullptr || a.d_r != nullptr)) {
                float gr = 0.f, gm = 0.f;
#pragma unroll 4
                for (int p = 0; p < n1; ++p) {
                    const float w = W0[p * d + lane];
                    gr = fmaf(G[p * 2 * QP + lane], w, gr);
                    gm = fmaf(G[p * 2 * QP + QP - 1], w, gm);
                }
                if (a.d_lo != nullptr) {
                    // m = (lo + hi) / 2, r = (hi - lo) / 2
                    a.d_lo[pos * d + lane] = 0.5f * (gm - gr);
                    a.d_hi[pos * d + lane] = 0.5f * (gm + gr);
                }
                if (a.d_r != nullptr) a.d_r[pos * d + lane] = gr;
            }
            if (a.split_codes != nullptr) {
                // the dimension of the split set with the largest |dM/dr_i| r_i, the first on ties
                const int64_t idx = a.src.index != nullptr ? a.src.index[pos] : pos;
                if (a.split_cls[idx] == kUndecided) {
                    float score = 0.f;
                    if (lane < a.n_split) {
                        const int i = a.split_dims[lane];
                        float gr = 0.f;
                        for (int p = 0; p < n1; ++p) gr = fmaf(G[p * 2 * QP + i], W0[p * d + i], gr);
                        score = fabsf(gr) * sr[i];
                    }
                    int sel = 0;
                    float best = -1.f;
                    for (int j = 0; j < a.n_split; ++j) {
                        const float v = __shfl_sync(0xffffffffu, score, j);
                        if (v > best) {
                            best = v;
                            sel = j;
                        }
                    }
                    if (lane == 0) a.split_codes[idx] |= (unsigned long long)sel << (kSplitPathBits + 4 * a.src.t);
                }
            }
        }
        if (kW) {
            __syncthreads();
            float *acc = sacc + pl.w_off[0], *accb = sacc + pl.b_off[0];
            for (int t = threadIdx.x; t < n1 * d; t += blockDim.x) {
                const int p = t / d, i = t - p * d;
                float s = 0.f;
                for (int b = 0; b < nbox; ++b) {
                    const float *g = boxes + b * stride + pl.rows + p * 2 * QP;
                    const float *m = boxes + b * stride + 2 * pl.rows;
                    s += fmaf(g[i], m[QP + i], g[QP - 1] * m[i]);
                }
                acc[t] += s;
            }
            for (int p = threadIdx.x; p < n1; p += blockDim.x) {
                float s = 0.f;
                for (int b = 0; b < nbox; ++b) s += boxes[b * stride + pl.rows + p * 2 * QP + QP - 1];
                accb[p] += s;
            }
            __syncthreads();
        } else {
            __syncwarp();
        }
    }

    if (kW) {
        // the block's sums; the folded last layer unfolded with the property rows
        for (int k = 0; k < K; ++k) {
            const int n_in = net.n[k], n_out = k == K - 1 ? a.n_out : net.n[k + 1], ld = pl.w_ld[k];
            const float *acc = sacc + pl.w_off[k], *accb = sacc + pl.b_off[k];
            for (int t = threadIdx.x; t < n_out * n_in; t += blockDim.x) {
                const int p = t / n_in, i = t - p * n_in;
                float v;
                if (k < K - 1) {
                    v = k == 0 ? acc[t] : acc[i * ld + p];
                } else {
                    v = 0.f;
                    for (int r = 0; r < R; ++r) v = fmaf(__ldg(a.Cprop + r * n_out + p), acc[i * ld + r], v);
                }
                atomicAdd(a.dW[k] + t, v);
            }
            for (int p = threadIdx.x; p < n_out; p += blockDim.x) {
                float v;
                if (k < K - 1) {
                    v = accb[p];
                } else {
                    v = 0.f;
                    for (int r = 0; r < R; ++r) v = fmaf(__ldg(a.Cprop + r * n_out + p), accb[r], v);
                }
                atomicAdd(a.db[k] + p, v);
            }
        }
    }
}

typedef void (*AdjWarpKernel)(const AdjArgs, const AdjWarpPlan, float *);

template <bool kW>
AdjWarpKernel pick(int QP, int RPL) {
    switch (QP * 10 + RPL) {
        case 41: return adj_warp_kernel<4, 1, kW>;
        case 42: return adj_warp_kernel<4, 2, kW>;
        case 44: return adj_warp_kernel<4, 4, kW>;
        case 61: return adj_warp_kernel<6, 1, kW>;
        case 62: return adj_warp_kernel<6, 2, kW>;
        case 64: return adj_warp_kernel<6, 4, kW>;
        case 81: return adj_warp_kernel<8, 1, kW>;
        case 82: return adj_warp_kernel<8, 2, kW>;
        case 84: return adj_warp_kernel<8, 4, kW>;
        default: return nullptr;
    }
}

AdjWarpKernel pick(const AdjWarpPlan &p, bool w) { return w ? pick<true>(p.QP, p.RPL) : pick<false>(p.QP, p.RPL); }

size_t smem_of(const AdjWarpPlan &p, bool w) {
    return sizeof(float) * ((size_t)p.head * (w ? 2 : 1) + (size_t)p.box[w ? 1 : 0] * (p.threads[w ? 1 : 0] / 32));
}

}  // namespace

size_t adj_warp_scratch_bytes(const AdjWarpPlan &p, int K, bool w) {
    return (size_t)p.grid[w ? 1 : 0] * (p.threads[w ? 1 : 0] / 32) * (K - 1) * p.RPL * 2 * p.QP * 32 * sizeof(float);
}

// The launch shape for a network, or grid 0 where the warp form does not hold
// it: at least one hidden layer, at most 7 inputs (whole rows in registers),
// layers and property at most 128 wide (4 rows a lane), and the weights (with
// weight gradients: and their sums) beside the warps' rows in shared memory.
void adj_warp_plan(const NetParams<float> &net, int sms, size_t smem_max, AdjWarpPlan &p) {
    p = AdjWarpPlan{};
    int widest = 1;
    for (int k = 1; k <= net.K; ++k) widest = net.n[k] > widest ? net.n[k] : widest;
    if (net.K < 2 || net.d > 7 || widest > 128) return;
    p.QP = net.d <= 3 ? 4 : (net.d <= 5 ? 6 : 8);
    p.RPL = widest <= 32 ? 1 : (widest <= 64 ? 2 : 4);
    int at = 0;
    for (int k = 0; k < net.K; ++k) {
        p.w_off[k] = at;
        p.w_ld[k] = k == 0 ? net.d : (net.n[k + 1] | 1);
        at += k == 0 ? net.n[1] * net.d : net.n[k] * p.w_ld[k];
        p.b_off[k] = at;
        at += net.n[k + 1];
    }
    p.head = (at + 3) & ~3;
    p.rows = widest * 2 * p.QP;
    for (int w = 0; w < 2; ++w) {
        p.box[w] = ((w ? 2 : 1) * p.rows + 2 * p.QP + 4 * net.R + 3) & ~3;
        for (int nt = adj_threads(p.QP, p.RPL, w != 0); nt >= 64; nt -= 32) {
            p.threads[w] = nt;
            const size_t smem = smem_of(p, w != 0);
            if (smem > smem_max) continue;
            AdjWarpKernel k = pick(p, w != 0);
            int nb = 0;
            if (allow_smem(k) != cudaSuccess ||
                cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, nt, smem) != cudaSuccess) {
                (void)cudaGetLastError();
                nb = 0;
            }
            p.grid[w] = nb * sms;
            if (nb > 0) break;
        }
    }
}

cudaError_t launch_adj_warp(const AdjArgs &a, const AdjWarpPlan &p, bool w, float *chk, cudaStream_t s) {
    AdjWarpKernel k = pick(p, w);
    if (k == nullptr || p.grid[w ? 1 : 0] <= 0) return cudaErrorInvalidValue;
    const int nt = p.threads[w ? 1 : 0];
    const size_t smem = smem_of(p, w);
    cudaError_t e = allow_smem(k);
    if (e != cudaSuccess) return e;
    const int64_t most = p.grid[w ? 1 : 0];
    const int64_t grid = a.n < most ? (a.n < 1 ? 1 : a.n) : most;
    // the warps that take boxes: as few as keep the rounds, so that the rounds are full
    AdjWarpPlan pl = p;
    const int64_t n = a.n < 1 ? 1 : a.n;
    const int64_t rounds = (n + grid * (nt / 32) - 1) / (grid * (nt / 32));
    pl.act = (int)((n + grid * rounds - 1) / (grid * rounds));
    k<<<(int)grid, nt, smem, s>>>(a, pl, chk);
    return cudaGetLastError();
}

}  // namespace slr
