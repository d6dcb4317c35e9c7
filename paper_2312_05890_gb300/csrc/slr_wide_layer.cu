// Wide networks with many inputs: one kernel per hidden layer.
//
// The state between two layers is kept as the contraction left it (the raw
// equations C', R' of the pre-activations), with the ReLU relaxation (Eq. 1)
// as two numbers per row, (c, r) -> (pp c + qq r, qq c + pp r).  The next
// layer's product applies them while it loads its operands, and its epilogue
// sums the coefficients for the concrete bounds (Sec. 2.2) while it stores
// them, so each layer's state is written once and read once.  The first
// layer's equations W_1 diag(r) are never stored: the loader forms them.
// Per row only small arrays remain: the partial bound sums, the radius
// constant, N and E (three columns with a product of their own) and the
// constants.
//
// wide_layer_kernel is persistent, one CTA per SM, and warp-specialised:
//   warps 0-7    epilogue: tensor memory -> bound sums and stores
//   warps 8-15   operand producers: global -> relaxation -> TF32 pieces -> shared
//   warp 16      one lane issues the products (tcgen05, kind::tf32)
//   warp 17      one lane copies the weight pieces (bulk copies, laid out in
//                global memory as the stages of the shared-memory ring)
// over a ring of kStages stages of 8 inputs.  A tile is 128 output rows by NC
// input coefficients of one box, both equations: C' = W C and R' = |W| R into
// 2 x 256 columns of tensor memory, three split products each (x = hi + lo,
// lo hi + hi lo + hi hi), in the order of wide_gemm_kernel, so that the sums
// are the same bit for bit.  While the epilogue drains a tile the producers
// fill the ring for the next one.
#include <algorithm>

#include "slr_eval.cuh"
#include "slr_kernels.h"
#include "slr_tc_util.cuh"

namespace slr {

using namespace tc;

namespace {

using WTile = EvalTile<float, 1, 1>;   // only its static row helpers are used

constexpr int kLStages = 4;
constexpr int kLK = 8;                            // inputs per stage (one MMA K step)
constexpr int kLRows = 128;                       // output rows of a tile
constexpr int kLCols = 256;                       // most columns of a tile and equation
constexpr int kLLbo = 128, kLSbo = 256;           // core matrices: 8 rows x 16 bytes, dense
constexpr int kLAImg = kLRows * kLK * 4;          // one piece of the weights of a stage
constexpr int kLA = 4 * kLAImg;                   // [W hi | W lo | |W| hi | |W| lo]
constexpr int kLBImg = kLCols * kLK * 4;          // one piece of one equation's operand
constexpr int kLStage = kLA + 4 * kLBImg;         // ... [C hi | C lo | R hi | R lo]
constexpr int kLEpi = 8, kLProd = 8;              // warps
constexpr int kLThreads = 32 * (kLEpi + kLProd + 2);
constexpr int kLSmem = kLStages * kLStage + 256;
constexpr int kLWait = 1 << 24;

// What a producer thread holds of one stage between its loads and its stores:
// two columns, four inputs each.
struct Raw {
    float4 c[2], r[2], pp, qq;
};

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void split4(const float (&v)[4], unsigned char *hi, unsigned char *lo) {
    float4 h, l;
    h.x = tf32_rna(v[0]);
    h.y = tf32_rna(v[1]);
    h.z = tf32_rna(v[2]);
    h.w = tf32_rna(v[3]);
    l.x = tf32_rna(v[0] - h.x);
    l.y = tf32_rna(v[1] - h.y);
    l.z = tf32_rna(v[2] - h.z);
    l.w = tf32_rna(v[3] - h.w);
    *reinterpret_cast<float4 *>(hi) = h;
    *reinterpret_cast<float4 *>(lo) = l;
}

// A relaxed row is all zeros when pp = qq = 0: its stored equations are not
// looked at (beyond a layer's width the state holds no values).
__device__ __forceinline__ void relax_pair(float pp, float qq, float c0, float r0, float &c, float &r) {
    const bool zero = pp == 0.f && qq == 0.f;
    c = zero ? 0.f : __fmaf_rn(pp, c0, __fmul_rn(qq, r0));
    r = zero ? 0.f : __fmaf_rn(qq, c0, __fmul_rn(pp, r0));
}

}  // namespace

__global__ void __launch_bounds__(kLThreads, 1) wide_layer_kernel(const WideLayer G) {
    extern __shared__ __align__(1024) unsigned char smem_l[];
    uint64_t *full = reinterpret_cast<uint64_t *>(smem_l + kLStages * kLStage);
    uint64_t *empty = full + kLStages, *tfull = empty + kLStages, *tempty = tfull + 1;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(tempty + 1);
    volatile int *sAbort = reinterpret_cast<volatile int *>(tslot + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int s = 0; s < kLStages; ++s) {
            // a stage is full when the producer warps have stored and the bulk copy has landed
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&full[s])), "r"(kLProd + 1));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&empty[s])));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(tfull)));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(tempty)), "r"(kLEpi));
        asm volatile("fence.mbarrier_init.release.cluster;");
        *sAbort = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tslot)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = *tslot;

    const int nst = G.nst, NC = G.NC;
    const int per_box = G.ntile * G.mt;
    const int items = G.nb * per_box;             // item = (box, column tile, row tile), row tile fastest
    bool ok = true;

    if (warp < kLEpi) {
        // ---- epilogue ----
        const int quad = warp & 3, half = warp >> 2;
        const int nch = NC / 16, ch0 = half ? (nch + 1) / 2 : 0, ch1 = half ? nch : (nch + 1) / 2;
        int use = 0;
        for (int item = blockIdx.x; item < items; item += gridDim.x, ++use) {
            const int b = item / per_box, rest = item - b * per_box;
            const int t = rest / G.mt, m = rest - t * G.mt;
            const int p = m * kLRows + quad * 32 + lane;
            if (!mbar_wait(smem_u32(tfull), (uint32_t)(use & 1), kLWait)) ok = false;
            if (__any_sync(0xffffffffu, !ok || *sAbort != 0)) {
                *sAbort = 1;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;");
            RowBounds<float> bd;
            bd.reset();
            for (int ch = ch0; ch < ch1; ++ch) {
                uint32_t c[16], r[16];
                __syncwarp();
                const uint32_t ta = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(16 * ch);
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
                    "[%16];"
                    : "=r"(c[0]), "=r"(c[1]), "=r"(c[2]), "=r"(c[3]), "=r"(c[4]), "=r"(c[5]), "=r"(c[6]), "=r"(c[7]),
                      "=r"(c[8]), "=r"(c[9]), "=r"(c[10]), "=r"(c[11]), "=r"(c[12]), "=r"(c[13]), "=r"(c[14]),
                      "=r"(c[15])
                    : "r"(ta));
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
                    "[%16];"
                    : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                      "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                      "=r"(r[15])
                    : "r"(ta + kLCols));
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (ch + 1 == ch1) {
                    // the last read of this tile: tensor memory is free for the next one
                    asm volatile("tcgen05.fence::before_thread_sync;");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(tempty));
                }
                const int j0 = t * NC + 16 * ch;
                if (p < G.n_out) {
                    const size_t o = ((size_t)b * G.d + j0) * G.NP + p;
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        if (j0 + e < G.d) {
                            const float cv = __uint_as_float(c[e]), rv = __uint_as_float(r[e]);
                            bd.add(cv, rv);
                            G.Cout[o + (size_t)e * G.NP] = cv;
                            G.Rout[o + (size_t)e * G.NP] = rv;
                        }
                    }
                }
            }
            if (ch0 >= ch1) {
                asm volatile("tcgen05.fence::before_thread_sync;");
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(tempty));
            }
            if (p < G.n_out) {
                float *q = G.part + (((size_t)b * G.ntile + t) * 2 + half) * 4 * G.NP + p;
                q[0] = bd.SU;
                q[G.NP] = bd.SL;
                q[2 * G.NP] = bd.NC;
                q[3 * G.NP] = bd.NR;
            }
        }
    } else if (warp < kLEpi + kLProd) {
        // ---- producers: lanes 0-15 the first four inputs of 16 columns, lanes 16-31 the other four ----
        const int q = lane >> 4, col = (warp - kLEpi) * 16 + (lane & 15);
        const bool gen = G.Cin == nullptr;
        // the stage after the last loaded one
        int litem = blockIdx.x, lst = 0;
        const float *cp[2] = {nullptr, nullptr}, *rp[2] = {nullptr, nullptr}, *plan = nullptr;
        float rj[2] = {0.f, 0.f};
        bool in[2] = {false, false};
        auto load = [&](Raw &v) {
            if (litem >= items) return;
            if (lst == 0) {
                const int b = litem / per_box, t = (litem - b * per_box) / G.mt;
                plan = G.plan + (size_t)b * 2 * G.NP + 4 * q;
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int cc = col + 128 * u, j = t * NC + cc;
                    in[u] = cc < NC && j < G.d;
                    if (!in[u]) continue;
                    if (gen) {
                        cp[u] = G.W0p + (size_t)j * G.NP + 4 * q;
                        rj[u] = G.rr[(size_t)b * G.d + j];
                    } else {
                        const size_t o = ((size_t)b * G.d + j) * G.NP + 4 * q;
                        cp[u] = G.Cin + o;
                        rp[u] = G.Rin + o;
                    }
                }
            }
            v.pp = *reinterpret_cast<const float4 *>(plan + lst * kLK);
            v.qq = *reinterpret_cast<const float4 *>(plan + G.NP + lst * kLK);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                v.c[u] = v.r[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (!in[u]) continue;
                v.c[u] = *reinterpret_cast<const float4 *>(cp[u] + lst * kLK);
                if (gen) {
                    v.c[u].x = __fmul_rn(v.c[u].x, rj[u]);
                    v.c[u].y = __fmul_rn(v.c[u].y, rj[u]);
                    v.c[u].z = __fmul_rn(v.c[u].z, rj[u]);
                    v.c[u].w = __fmul_rn(v.c[u].w, rj[u]);
                } else {
                    v.r[u] = *reinterpret_cast<const float4 *>(rp[u] + lst * kLK);
                }
            }
            if (++lst == nst) {
                lst = 0;
                litem += gridDim.x;
            }
        };
        const int mine = blockIdx.x < items ? (items - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
        const int total = mine * nst;
        int s = 0, round = 0;
        auto store = [&](const Raw &v) -> bool {
            if (round > 0 && !mbar_wait(smem_u32(&empty[s]), (uint32_t)((round - 1) & 1), kLWait)) ok = false;
            if (__any_sync(0xffffffffu, !ok || *sAbort != 0)) {
                *sAbort = 1;
                return false;
            }
            unsigned char *st = smem_l + s * kLStage + kLA;
            const float pp[4] = {v.pp.x, v.pp.y, v.pp.z, v.pp.w}, qq[4] = {v.qq.x, v.qq.y, v.qq.z, v.qq.w};
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int cc = col + 128 * u;
                if (cc >= NC) continue;
                const float c0[4] = {v.c[u].x, v.c[u].y, v.c[u].z, v.c[u].w};
                const float r0[4] = {v.r[u].x, v.r[u].y, v.r[u].z, v.r[u].w};
                float c[4], r[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) relax_pair(pp[e], qq[e], c0[e], r0[e], c[e], r[e]);
                unsigned char *o = st + (cc >> 3) * kLSbo + q * kLLbo + (cc & 7) * 16;
                split4(c, o, o + kLBImg);
                split4(r, o + 2 * kLBImg, o + 3 * kLBImg);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&full[s]));
            if (++s == kLStages) {
                s = 0;
                ++round;
            }
            return true;
        };
        // two stages of loads in flight
        Raw v0, v1;
        load(v0);
        load(v1);
        for (int g = 0; g < total; g += 2) {
            if (!store(v0)) break;
            load(v0);
            if (g + 1 < total) {
                if (!store(v1)) break;
                load(v1);
            }
        }
    } else if (warp == kLEpi + kLProd) {
        // ---- products ----
        if (lane == 0) {
            // kind::tf32, FP32 accumulate, both operands K-major, N = NC, M = 128
            const uint32_t idesc = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(NC >> 3) << 17) |
                                   ((uint32_t)(kLRows >> 4) << 24);
            int s = 0, round = 0, use = 0;
            for (int item = blockIdx.x; item < items && ok; item += gridDim.x, ++use) {
                if (use > 0 && !mbar_wait(smem_u32(tempty), (uint32_t)((use - 1) & 1), kLWait)) ok = false;
                asm volatile("tcgen05.fence::after_thread_sync;");
                for (int st = 0; st < nst && ok; ++st) {
                    if (!mbar_wait(smem_u32(&full[s]), (uint32_t)(round & 1), kLWait)) ok = false;
                    if (!ok || *sAbort) {
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;");
                    const uint32_t a0 = smem_u32(smem_l + s * kLStage), b0 = a0 + kLA;
#pragma unroll
                    for (int eq = 0; eq < 2; ++eq) {
                        const uint32_t ah = a0 + 2 * eq * kLAImg, al = ah + kLAImg;
                        const uint32_t bh = b0 + 2 * eq * kLBImg, bl = bh + kLBImg;
                        const uint32_t pa[3] = {ah, al, ah}, pb[3] = {bl, bh, bh};
#pragma unroll
                        for (int ps = 0; ps < 3; ++ps) {
                            const uint64_t da = umma_desc(pa[ps], kLLbo, kLSbo), db = umma_desc(pb[ps], kLLbo, kLSbo);
                            const uint32_t acc = (st > 0 || ps > 0) ? 1u : 0u;
                            asm volatile(
                                "{ .reg .pred p; setp.ne.b32 p, %4, 0; "
                                "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p; }" ::"r"(tmem + eq * kLCols),
                                "l"(da), "l"(db), "r"(idesc), "r"(acc));
                        }
                    }
                    asm volatile(
                        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                            smem_u32(&empty[s]))
                        : "memory");
                    if (++s == kLStages) {
                        s = 0;
                        ++round;
                    }
                }
                // (also after a timeout: what was issued completes and is waited for below)
                asm volatile(
                    "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                        smem_u32(tfull))
                    : "memory");
            }
            if (!ok) {
                *sAbort = 1;
                mbar_wait(smem_u32(tfull), (uint32_t)((use - 1) & 1), kLWait);
            }
        }
    } else {
        // ---- weight pieces ----
        if (lane == 0) {
            int s = 0, round = 0;
            for (int item = blockIdx.x; item < items && ok; item += gridDim.x) {
                const int m = item % G.mt;
                const unsigned char *src = G.Aimg + (size_t)m * nst * kLA;
                for (int st = 0; st < nst; ++st) {
                    if (round > 0 && !mbar_wait(smem_u32(&empty[s]), (uint32_t)((round - 1) & 1), kLWait)) ok = false;
                    if (!ok || *sAbort) {
                        ok = false;
                        break;
                    }
                    const uint32_t bar = smem_u32(&full[s]);
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(kLA)
                                 : "memory");
                    asm volatile(
                        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                            smem_u32(smem_l + s * kLStage)),
                        "l"(src + (size_t)st * kLA), "r"(kLA), "r"(bar)
                        : "memory");
                    if (++s == kLStages) {
                        s = 0;
                        ++round;
                    }
                }
            }
            if (!ok) {
                *sAbort = 1;
                // copies in flight land (their barriers may not complete: the wait is bounded)
                for (int k = 0; k < kLStages; ++k) mbar_wait(smem_u32(&full[k]), (uint32_t)(round & 1), 1 << 16);
            }
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (tid == 0 && *sAbort) atomicOr(G.status, kStatusTimeout);
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

// Weight pieces of one layer as the ring's stages: row tile m, stage s at
// out + (m nst + s) kLA bytes, each [W hi | W lo | |W| hi | |W| lo] of 128 rows
// by 8 inputs in core matrices.  The row-major pieces are zero padded to
// multiples of 128 rows and 32 inputs (ld floats).
__global__ void wide_pack_kernel(const float *hi, const float *lo, const float *ahi, const float *alo, int ld, int mt,
                                 int nst, float *out) {
    const int total = mt * nst * 4 * kLRows * kLK;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
        const int w = t % (kLRows * kLK), img = t / (kLRows * kLK) % 4, ms = t / (4 * kLRows * kLK);
        const int k = w % kLK, r = w / kLK;
        const float *src = img == 0 ? hi : (img == 1 ? lo : (img == 2 ? ahi : alo));
        const float v = src[(size_t)(ms / nst * kLRows + r) * ld + ms % nst * kLK + k];
        out[(size_t)ms * (kLA / 4) + img * (kLAImg / 4) + ((r >> 3) * kLSbo + (k >> 2) * kLLbo + (r & 7) * 16) / 4 +
            (k & 3)] = v;
    }
}

namespace {

// The relaxation of one row into the arrays the next product reads.
__device__ __forceinline__ void store_plan(const RelaxPlan<float> &pl, float *plan, float *S3, float *Ch, float *Cl,
                                           int64_t b, int NP, int p) {
    plan[(size_t)b * 2 * NP + p] = pl.kind == 1 ? 0.f : pl.pp;
    plan[((size_t)b * 2 + 1) * NP + p] = pl.kind == 1 ? 0.f : pl.qq;
    float *s = S3 + (size_t)b * 3 * NP + p;
    s[0] = pl.rd;
    s[NP] = pl.N;
    s[2 * NP] = pl.E;
    Ch[(size_t)b * NP + p] = pl.nh;
    Cl[(size_t)b * NP + p] = pl.nl;
}

}  // namespace

// Layer 1 (R = 0): its concrete bounds, constant and relaxation, without its
// coefficients W_1[p][j] r_j, which the next product forms.  A block is 32
// rows of one box, the d coefficients of a row in 16 slices merged in shared
// memory; sums, constant and error as in wide_init_kernel.
constexpr int kP1X = 32, kP1Y = 16;

__global__ void __launch_bounds__(kP1X * kP1Y)
wide_plan1_kernel(const NetParams<float> net, const float *W0p, int NP, const float *mh, const float *ml,
                  const float *rr, float *plan, float *S3, float *Ch, float *Cl, const float *alpha, int64_t alpha_ld,
                  int64_t base) {
    using A = Arith<float>;
    __shared__ float part[4][kP1Y][kP1X];
    const int d = net.d, n1 = net.n[1];
    const int lane = threadIdx.x, sl = threadIdx.y;
    const int p = blockIdx.x * kP1X + lane;
    const int64_t b = blockIdx.y;
    const float *rb = rr + b * d, *mb = mh + b * d, *lb = ml + b * d;
    float S = 0.f, s = 0.f, e = 0.f, sabs = 0.f;
    if (p < n1) {
        if (sl == 0) {
            s = net.b[0][p];
            sabs = fabsf(s);
        }
#pragma unroll 4
        for (int j = sl; j < d; j += kP1Y) {
            const float wj = W0p[(size_t)j * NP + p];
            S = A::add_up(S, fabsf(A::mul_rn(wj, rb[j])));
            float p1, pe, tt, se;
            two_prod<float>(wj, mb[j], p1, pe);
            two_sum<float>(s, p1, tt, se);
            s = tt;
            e = A::fma_rn(wj, lb[j], e + (pe + se));
            sabs = sabs + fabsf(p1);
        }
    }
    part[0][sl][lane] = S;
    part[1][sl][lane] = s;
    part[2][sl][lane] = e;
    part[3][sl][lane] = sabs;
    __syncthreads();
    if (sl != 0 || p >= NP) return;
    RelaxPlan<float> pl;
    pl.kind = 1;
    pl.pp = pl.qq = pl.nh = pl.nl = pl.rd = pl.N = pl.E = 0.f;
    if (p < n1) {
        for (int y = 1; y < kP1Y; ++y) {
            S = A::add_up(S, part[0][y][lane]);
            float tt, se;
            two_sum<float>(s, part[1][y][lane], tt, se);
            s = tt;
            e = e + (part[2][y][lane] + se);
            sabs = sabs + part[3][y][lane];
        }
        float chi, clo;
        two_sum<float>(s, e, chi, clo);
        const float g = gam<float>(d + 2);
        float E = A::add_up(uerr<float>(S), A::mul_up(A::mul_up(2.f * g, g), A::mul_up(sabs, 1.f + gam<float>(d))));
        E = A::add_up(E, (float)(d + 4) * A::tiny);
        RowBounds<float> t;
        t.reset();
        t.SU = t.SL = t.NC = S;
        t.finish(chi, clo, 0.f);
        const float *a_ptr = alpha != nullptr ? alpha + (base + b) * alpha_ld + p : nullptr;
        pl = WTile::plan_row(t, d, net.relax_mode, chi, clo, 0.f, E, a_ptr, net.act[0]);
    }
    store_plan(pl, plan, S3, Ch, Cl, b, NP, p);
}

// Hidden layer `layer` after its product: the bound sums of its tiles, the
// products of the radius constant, N and E columns (T3), the constants
// (Kh, Kl, Ke) -> error, bounds, relaxation.  One thread per row.
__global__ void __launch_bounds__(128)
wide_plan_kernel(const NetParams<float> net, int layer, int NP, float gcoef, const float *part, int nparts,
                 const float *T3, const float *Kh, const float *Kl, const float *Ke, float *plan, float *S3, float *Ch,
                 float *Cl, const float *alpha, int64_t alpha_ld, int64_t base) {
    using A = Arith<float>;
    const int p = blockIdx.x * 128 + threadIdx.x;
    const int64_t b = blockIdx.y;
    if (p >= NP) return;
    RelaxPlan<float> pl;
    pl.kind = 1;
    pl.pp = pl.qq = pl.nh = pl.nl = pl.rd = pl.N = pl.E = 0.f;
    if (p < net.n[layer]) {
        const int n_in = net.n[layer - 1];
        RowBounds<float> t, o;
        t.reset();
        o.reset();
        const float *q = part + (size_t)b * nparts * 4 * NP + p;
        for (int k = 0; k < nparts; ++k) {
            o.SU = q[(size_t)(4 * k) * NP];
            o.SL = q[(size_t)(4 * k + 1) * NP];
            o.NC = q[(size_t)(4 * k + 2) * NP];
            o.NR = q[(size_t)(4 * k + 3) * NP];
            t.merge(o);
        }
        const float *t3 = T3 + (size_t)b * 3 * NP + p;
        const float rd = t3[0], wN = t3[NP], wE = t3[2 * NP];
        const float chi = Kh[(size_t)b * NP + p], clo = Kl[(size_t)b * NP + p];
        // E' = |W| E (1 + 2 g) + g |W| N (1 + g) + the constant's error
        float eps = A::mul_up(gcoef, A::mul_up(wN, 1.f + gcoef));
        eps = A::add_up(A::add_up(eps, Ke[(size_t)b * NP + p]), (float)(n_in + 4) * A::tiny);
        const float E = A::add_up(A::mul_up(wE, 1.f + 2.f * gcoef), eps);
        t.finish(chi, clo, rd);
        const float *a_ptr = nullptr;
        if (alpha != nullptr) {
            int off = 0;
            for (int j = 1; j < layer; ++j) off += net.n[j];
            a_ptr = alpha + (base + b) * alpha_ld + off + p;
        }
        pl = WTile::plan_row(t, net.d, net.relax_mode, chi, clo, rd, E, a_ptr, net.act[layer - 1]);
    }
    store_plan(pl, plan, S3, Ch, Cl, b, NP, p);
}

// The property layer: relaxation of the last hidden layer and the products of
// its few rows, one input coefficient (column of both equations) per thread,
// FP32 FMA chains over the inputs in order (rounding within gamma_{n_in} of
// sum |W| |x|).  Row r of column j of box b goes to out[((b d + j) 2 + eq) RM + r].
template <int RM>
__global__ void __launch_bounds__(128)
wide_rows_kernel(const NetParams<float> net, int NP, const float *Cin, const float *Rin, const float *W0p,
                 const float *rr, const float *plan, int64_t ncols, float *out) {
    extern __shared__ float sWr[];   // n_in x RM, zero beyond R
    const int K = net.K, n_in = net.n[K - 1], R = net.R, d = net.d;
    const int n4 = (n_in + 3) & ~3;
    for (int q = threadIdx.x; q < n4 * RM; q += blockDim.x) {
        const int i = q / RM, r = q - i * RM;
        sWr[q] = r < R && i < n_in ? net.Wt[K - 1][(size_t)i * R + r] : 0.f;
    }
    __syncthreads();
    for (int64_t col = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; col < ncols;
         col += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = col / d;
        const float *pl = plan + (size_t)b * 2 * NP;
        const bool gen = Cin == nullptr;
        const float *cp = gen ? W0p + (size_t)(col - b * d) * NP : Cin + (size_t)col * NP;
        const float *rp = gen ? nullptr : Rin + (size_t)col * NP;
        const float rj = gen ? rr[col] : 0.f;
        float ac[RM], ar[RM];
#pragma unroll
        for (int r = 0; r < RM; ++r) ac[r] = ar[r] = 0.f;
#pragma unroll 2
        for (int i = 0; i < n4; i += 4) {
            const float4 c4 = *reinterpret_cast<const float4 *>(cp + i);
            const float4 r4 = gen ? make_float4(0.f, 0.f, 0.f, 0.f) : *reinterpret_cast<const float4 *>(rp + i);
            const float4 p4 = *reinterpret_cast<const float4 *>(pl + i);
            const float4 q4 = *reinterpret_cast<const float4 *>(pl + NP + i);
            const float c0[4] = {c4.x, c4.y, c4.z, c4.w}, r0[4] = {r4.x, r4.y, r4.z, r4.w};
            const float pv[4] = {p4.x, p4.y, p4.z, p4.w}, qv[4] = {q4.x, q4.y, q4.z, q4.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float c, x;
                relax_pair(pv[u], qv[u], gen ? __fmul_rn(c0[u], rj) : c0[u], r0[u], c, x);
#pragma unroll
                for (int r = 0; r < RM; ++r) {
                    const float w = sWr[(i + u) * RM + r];
                    ac[r] = fmaf(w, c, ac[r]);
                    ar[r] = fmaf(fabsf(w), x, ar[r]);
                }
            }
        }
        float *o = out + (size_t)col * 2 * RM;
#pragma unroll
        for (int r = 0; r < RM; r += 4) {
            *reinterpret_cast<float4 *>(o + r) = make_float4(ac[r], ac[r + 1], ac[r + 2], ac[r + 3]);
            *reinterpret_cast<float4 *>(o + RM + r) = make_float4(ar[r], ar[r + 1], ar[r + 2], ar[r + 3]);
        }
    }
}

// Property rows of one box per block: sound bounds lo = min L' - E, hi = max U' + E
// (Sec. 3 check) from the columns of wide_rows_kernel, T3 the products of the
// radius constant, N and E.  blockDim.x = 32 RM: warp w sums row w.
__global__ void wide_rows_final_kernel(const NetParams<float> net, int NP, int RM, float gcoef, const float *cols,
                                       const float *T3, const float *Kh, const float *Kl, const float *Ke, float *lo,
                                       float *hi, float *err) {
    using A = Arith<float>;
    const int d = net.d, R = net.R, n_in = net.n[net.K - 1];
    const int r = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t b = blockIdx.x;
    if (r >= R) return;
    RowBounds<float> t;
    t.reset();
#pragma unroll 4
    for (int j = lane; j < d; j += 32) {
        const float *o = cols + ((size_t)b * d + j) * 2 * RM + r;
        t.add(o[0], o[RM]);
    }
    for (int o = 16; o > 0; o >>= 1) {
        RowBounds<float> u;
        u.SU = __shfl_xor_sync(0xffffffffu, t.SU, o);
        u.SL = __shfl_xor_sync(0xffffffffu, t.SL, o);
        u.SUn = __shfl_xor_sync(0xffffffffu, t.SUn, o);
        u.SLn = __shfl_xor_sync(0xffffffffu, t.SLn, o);
        u.NC = __shfl_xor_sync(0xffffffffu, t.NC, o);
        u.NR = __shfl_xor_sync(0xffffffffu, t.NR, o);
        t.merge(u);
    }
    if (lane != 0) return;
    const float *t3 = T3 + (size_t)b * 3 * NP + r;
    float eps = A::mul_up(gcoef, A::mul_up(t3[NP], 1.f + gcoef));
    eps = A::add_up(A::add_up(eps, Ke[(size_t)b * NP + r]), (float)(n_in + 4) * A::tiny);
    const float E = A::add_up(A::mul_up(t3[2 * NP], 1.f + 2.f * gcoef), eps);
    t.finish(Kh[(size_t)b * NP + r], Kl[(size_t)b * NP + r], t3[0]);
    lo[b * R + r] = A::add_dn(t.ll, -E);
    hi[b * R + r] = A::add_up(t.uu, E);
    err[b * R + r] = A::add_up(E, t.delta);
}

// ---------------------------------------------------------------------------
// launch wrappers
// ---------------------------------------------------------------------------

// Column tiles of a box: the fewest of at most 256 columns, each a multiple of 16.
void wide_layer_tiles(int d, int &ntile, int &NC) {
    ntile = (d + kLCols - 1) / kLCols;
    NC = ((d + ntile - 1) / ntile + 15) & ~15;
}

size_t wide_layer_img_bytes(int n_in, int n_out) {
    return (size_t)((n_out + kLRows - 1) / kLRows) * ((n_in + kLK - 1) / kLK) * kLA;
}

cudaError_t launch_wide_pack(const float *hi, const float *lo, const float *ahi, const float *alo, int ld, int n_in,
                             int n_out, void *out, cudaStream_t s) {
    const int mt = (n_out + kLRows - 1) / kLRows, nst = (n_in + kLK - 1) / kLK;
    const int total = mt * nst * 4 * kLRows * kLK;
    wide_pack_kernel<<<std::min(1024, (total + 255) / 256), 256, 0, s>>>(hi, lo, ahi, alo, ld, mt, nst, (float *)out);
    return cudaGetLastError();
}

cudaError_t launch_wide_layer(WideLayer G, int sms, cudaStream_t s) {
    G.mt = (G.n_out + kLRows - 1) / kLRows;
    G.nst = (G.n_in + kLK - 1) / kLK;
    wide_layer_tiles(G.d, G.ntile, G.NC);
    const int64_t items = (int64_t)G.nb * G.ntile * G.mt;
    if (items <= 0) return cudaSuccess;
    if (items > INT32_MAX) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(wide_layer_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kLSmem);
    if (e != cudaSuccess) return e;
    wide_layer_kernel<<<(int)std::min<int64_t>(items, sms), kLThreads, kLSmem, s>>>(G);
    return cudaGetLastError();
}

cudaError_t launch_wide_plan1(const NetParams<float> &net, const float *W0p, int nb, int NP, const float *mh,
                              const float *ml, const float *rr, float *plan, float *S3, float *Ch, float *Cl,
                              const float *alpha, int64_t alpha_ld, int64_t base, cudaStream_t s) {
    wide_plan1_kernel<<<dim3(NP / kP1X, nb), dim3(kP1X, kP1Y), 0, s>>>(net, W0p, NP, mh, ml, rr, plan, S3, Ch, Cl,
                                                                       alpha, alpha_ld, base);
    return cudaGetLastError();
}

cudaError_t launch_wide_plan(const NetParams<float> &net, int layer, int nb, int NP, float gcoef, const float *part,
                             const float *T3, const float *Kh, const float *Kl, const float *Ke, float *plan,
                             float *S3, float *Ch, float *Cl, const float *alpha, int64_t alpha_ld, int64_t base,
                             cudaStream_t s) {
    int ntile, NC;
    wide_layer_tiles(net.d, ntile, NC);
    wide_plan_kernel<<<dim3((NP + 127) / 128, nb), 128, 0, s>>>(net, layer, NP, gcoef, part, 2 * ntile, T3, Kh, Kl, Ke,
                                                                plan, S3, Ch, Cl, alpha, alpha_ld, base);
    return cudaGetLastError();
}

// Rows of a column's record, R rounded up to a multiple of 4 (R <= 16).
int wide_rows_stride(int R) { return (R + 3) & ~3; }

cudaError_t launch_wide_rows(const NetParams<float> &net, int nb, int NP, const float *Cin, const float *Rin,
                             const float *W0p, const float *rr, const float *plan, float *out, int sms,
                             cudaStream_t s) {
    const int64_t ncols = (int64_t)nb * net.d;
    const int grid = (int)std::min<int64_t>((ncols + 127) / 128, (int64_t)sms * 16);
    const int RM = wide_rows_stride(net.R);
    const size_t smem = (size_t)((net.n[net.K - 1] + 3) & ~3) * RM * sizeof(float);
    auto run = [&](auto k) -> cudaError_t {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k<<<grid, 128, smem, s>>>(net, NP, Cin, Rin, W0p, rr, plan, ncols, out);
        return cudaGetLastError();
    };
    switch (RM) {
        case 4: return run(wide_rows_kernel<4>);
        case 8: return run(wide_rows_kernel<8>);
        case 12: return run(wide_rows_kernel<12>);
        case 16: return run(wide_rows_kernel<16>);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_wide_rows_final(const NetParams<float> &net, int nb, int NP, float gcoef, const float *cols,
                                   const float *T3, const float *Kh, const float *Kl, const float *Ke, float *lo,
                                   float *hi, float *err, cudaStream_t s) {
    wide_rows_final_kernel<<<nb, 32 * net.R, 0, s>>>(net, NP, wide_rows_stride(net.R), gcoef, cols, T3, Kh, Kl, Ke, lo,
                                                     hi, err);
    return cudaGetLastError();
}

}  // namespace slr
