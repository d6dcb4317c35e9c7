// Wide networks with many inputs: one kernel per hidden layer.
//
// The state between two layers is kept as the contraction left it (the raw
// equations C', R' of the pre-activations), with the ReLU relaxation (Eq. 1)
// as two numbers per row, (c, r) -> (pp c + qq r, qq c + pp r).  The next
// layer's product applies them while it loads its operands, and its epilogue
// sums the coefficients for the concrete bounds (Sec. 2.2) while it stores
// them, so each layer's state is written once and read once.  The first
// layer's equations W_1 diag(r) are never stored: the loader forms them.
// The state is laid out by the tiles of that kernel: the coefficients of
// neurons 16 k .. 16 k + 15 for the columns (inputs of the network) of one tile
// are one contiguous run, [box][tile][k][column][16], so that what a stage
// reads is contiguous.  (Neurons fastest within a column, the layout of the
// general wide path, has a stage read 64 bytes of every kilobyte: the products
// then wait for DRAM at a sixth of its bandwidth.)
// Per row only small arrays remain: the partial bound sums, and the radius
// constant, N, E and the constant, whose products one thread per row forms
// together (wide_plan_kernel).
//
// wide_layer_kernel is persistent, one CTA per SM, and warp-specialised:
//   warps 0-13   operand producers: global -> relaxation -> TF32 pieces ->
//                shared (64 bytes of a column a stage), and between two tiles
//                (warps 0-11) the epilogue: tensor memory -> bound sums and stores
//   warp 14      one lane issues the products (tcgen05, kind::tf32)
//   warp 15      one lane copies the weight pieces (bulk copies, laid out in
//                global memory as the stages of their shared-memory ring)
// over a ring of kBStages operand stages and one of up to kAMax weight stages
// of 16 inputs.  (One thread issues every product: with stages of 8 inputs its
// waits and descriptors took twice the tensor core's time.)  A tile is 128
// output rows by NC input coefficients of one box, both equations: C' = W C
// and R' = |W| R into 2 x 256 columns of tensor memory, three split products
// each (x = hi + lo, lo hi + hi lo + hi hi), in the order of wide_gemm_kernel,
// so that the sums are the same bit for bit.  The producers fill the ring for
// the next tile before they drain the last one.
//
// Measured on 784-3x256-10, 1,000 boxes (two layers of 1.6 GB read and written):
// 1.29 ms a layer, tensor pipe 45 % busy, 2.5 TB/s; the rest of a tile's 27 us
// is the drain (the product waits for its tensor memory, about 5 us) and the
// producers' loads.  The whole bounds 8.83 -> 3.66 ms, a depth-12 count
// 76.0 -> 31.0 ms against one product kernel and one relaxation kernel in place
// per layer (slr_wide.cu), which still serves fewer than kWideLayerMinD inputs
// (a column tile of one box would be mostly padding: 70 inputs 1.53 -> 1.17 ms
// for 3,000 boxes of a 70-2x200-10 network) and more than 16 property rows.
#include <algorithm>

#include "slr_eval.cuh"
#include "slr_kernels.h"
#include "slr_tc_util.cuh"

namespace slr {

using namespace tc;

namespace {

using WTile = EvalTile<float, 1, 1>;   // only its static row helpers are used

constexpr int kBStages = 2, kAMax = 4;            // ring stages: operands, most of weights
constexpr int kLK = 16;                           // inputs per stage: two MMA K steps
constexpr int kLStep = 8;                         // inputs of a step
constexpr int kLRows = 128;                       // output rows of a tile
// Core matrices are 8 rows x 16 bytes: the weights' dense (bulk copies), the
// state's with a step's two 160 bytes apart and its steps 64 bytes off a
// multiple of 128, so that eight lanes that store two columns' sixteen inputs
// fall in distinct banks.
constexpr int kLLboA = 128, kLSboA = 256;
constexpr int kLLboB = 160, kLSboB = 320;
constexpr int kLAImg = kLRows * kLStep * 4;       // one piece of the weights of a step
constexpr int kLAStep = 4 * kLAImg;               // [W hi | W lo | |W| hi | |W| lo]
constexpr int kLA = kLK / kLStep * kLAStep;       // a stage's weights
// Sixteen warps leave 128 registers a thread: the producers' loads in flight
// must not spill (a spill waits for its load).
constexpr int kLWork = 14, kLEpi = 12;            // producer warps; those that drain tiles too
constexpr int kLThreads = 32 * (kLWork + 2);
constexpr int kLCols = 2 * 8 * kLWork;            // most columns of a tile: two groups of eight per producer warp
constexpr int kLTmemR = 256;                      // tensor memory column of R'
constexpr int kLBar = 256;                        // bytes of the barriers
constexpr int kLWait = 1 << 24;

// Bytes of one piece of one equation's operand of a step, and of a whole step
// [C hi | C lo | R hi | R lo], for NC columns (the 64: see above; a multiple
// of 128 plus 64 in all for NC a multiple of 16).
__host__ __device__ inline int b_img(int NC) { return NC / 8 * kLSboB; }
__host__ __device__ inline int b_step(int NC) { return 4 * b_img(NC) + 64; }
__host__ __device__ inline int b_stage(int NC) { return kLK / kLStep * b_step(NC); }
inline int a_stages(int NC) { return std::min(kAMax, (kCtaSmem - kLBar - kBStages * b_stage(NC)) / kLA); }

// What a producer thread holds between its loads and its stores: four
// neighbouring inputs of two columns.
struct Raw {
    float4 c[2], r[2];
    float rj[2];                  // layer 1: the columns' radii
};

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// A finite x as TF32 hi + lo, rounded to nearest, ties away from zero (as
// cvt.rna.tf32.f32, in fewer instructions: half a unit is added to the bits).
// For the sound bounds only: a NaN may come out as a zero (0x7fffffff, the NaN
// that FP32 arithmetic gives, carries into the sign).  They do not need it,
// since a row that holds one has a NaN or an infinity in its N, which reaches
// every later row's error bound through the products of the N and E columns
// (small_row).  The adjoint has no such columns and keeps the conversion: a
// NaN of the caller's or of a state that overflowed is one in what depends on it.
__device__ __forceinline__ float tf32_bits(float x) {
    return __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xffffe000u);
}

template <bool kPlain>
__device__ __forceinline__ float tf32_piece(float x) {
    return kPlain ? tf32_rna(x) : tf32_bits(x);
}

template <bool kPlain>
__device__ __forceinline__ void split4(const float (&v)[4], unsigned char *hi, unsigned char *lo) {
    float4 h, l;
    h.x = tf32_piece<kPlain>(v[0]);
    h.y = tf32_piece<kPlain>(v[1]);
    h.z = tf32_piece<kPlain>(v[2]);
    h.w = tf32_piece<kPlain>(v[3]);
    l.x = tf32_piece<kPlain>(v[0] - h.x);
    l.y = tf32_piece<kPlain>(v[1] - h.y);
    l.z = tf32_piece<kPlain>(v[2] - h.z);
    l.w = tf32_piece<kPlain>(v[3] - h.w);
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

// kPlain: the two products alone, D_C = W C, D_R = |W| R on states [box][column][NP]
// (the wide adjoint): no relaxation, no bound sums.
template <bool kPlain>
__global__ void __launch_bounds__(kLThreads, 1) wide_layer_kernel(const WideLayer G) {
    extern __shared__ __align__(1024) unsigned char smem_l[];
    const int NA = G.na, NC = G.NC, bimg = b_img(NC), bstep = b_step(NC), bstage = b_stage(NC);
    unsigned char *const sA = smem_l, *const sB = smem_l + NA * kLA;
    uint64_t *afull = reinterpret_cast<uint64_t *>(sB + kBStages * bstage), *aempty = afull + kAMax;
    uint64_t *bfull = aempty + kAMax, *bempty = bfull + kBStages, *tfull = bempty + kBStages, *tempty = tfull + 1;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(tempty + 1);
    volatile int *sAbort = reinterpret_cast<volatile int *>(tslot + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    auto init = [](uint64_t *bar, int count) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
    };
    if (tid == 0) {
        for (int s = 0; s < kAMax; ++s) {
            init(&afull[s], 1);
            init(&aempty[s], 1);
        }
        for (int s = 0; s < kBStages; ++s) {
            init(&bfull[s], kLWork);
            init(&bempty[s], 1);
        }
        init(tfull, 1);
        init(tempty, kLEpi);
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

    const int nst = G.nst;
    // the state of column cc of tile t of box b, inputs or rows 16 k ..: from
    // ((b boxes) + t tiles) + cc cs + k ks
    const size_t tile = (size_t)NC * G.NP;
    const size_t boxs = kPlain ? (size_t)G.d * G.NP : G.ntile * tile;
    const int cs = kPlain ? G.NP : kLK, ks = kPlain ? kLK : NC * kLK;
    const int per_box = G.ntile * G.mt;
    const int items = G.nb * per_box;             // item = (box, column tile, row tile), row tile fastest
    const int mine = (items - 1 - (int)blockIdx.x) / (int)gridDim.x + 1;   // (the grid has at most `items` CTAs)
    bool ok = true;

    if (warp < kLWork) {
        // ---- epilogue of this CTA's item `use`: rows of the warp's quarter of
        // tensor memory, a third of the columns ----
        const int quad = warp & 3, slice = warp >> 2;
        const int nch = NC / 16, ch0 = nch * slice / 3, ch1 = nch * (slice + 1) / 3;
        auto epilogue = [&](int use) -> bool {
            const int item = blockIdx.x + use * gridDim.x;
            const int b = item / per_box, rest = item - b * per_box;
            const int t = rest / G.mt, m = rest - t * G.mt;
            const int p = m * kLRows + quad * 32 + lane;
            if (!mbar_wait(smem_u32(tfull), (uint32_t)(use & 1), kLWait)) ok = false;
            if (__any_sync(0xffffffffu, !ok)) {
                ok = false;
                return false;
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
                    : "r"(ta + kLTmemR));
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (ch + 1 == ch1) {
                    // the warp's last read of this tile: its tensor memory is free
                    asm volatile("tcgen05.fence::before_thread_sync;");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(tempty));
                }
                const int j0 = t * NC + 16 * ch;
                if (p < G.n_out) {
                    const size_t o = b * boxs + t * tile + (size_t)(p / kLK) * ks + (size_t)(16 * ch) * cs + p % kLK;
                    float *co = G.Cout + o, *ro = G.Rout + o;
                    if (j0 + 16 <= G.d) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) {
                            const float cv = __uint_as_float(c[e]), rv = __uint_as_float(r[e]);
                            if (!kPlain) bd.add(cv, rv);
                            co[e * cs] = cv;
                            ro[e * cs] = rv;
                        }
                    } else {
#pragma unroll
                        for (int e = 0; e < 16; ++e) {
                            if (j0 + e < G.d) {
                                const float cv = __uint_as_float(c[e]), rv = __uint_as_float(r[e]);
                                if (!kPlain) bd.add(cv, rv);
                                co[e * cs] = cv;
                                ro[e * cs] = rv;
                            }
                        }
                    }
                }
            }
            if (ch0 >= ch1) {
                asm volatile("tcgen05.fence::before_thread_sync;");
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(tempty));
            }
            if (!kPlain && p < G.n_out) {
                float *q = G.part + (((size_t)b * G.ntile + t) * 3 + slice) * 4 * G.NP + p;
                q[0] = bd.SU;
                q[G.NP] = bd.SL;
                q[2 * G.NP] = bd.NC;
                q[3 * G.NP] = bd.NR;
            }
            return true;
        };

        // ---- producers: four lanes take a stage's 16 inputs of a column, so
        // that a load of a warp reads 64-byte runs of eight columns ----
        const int q = lane & 3;
        const int col = warp * 8 + (lane >> 2);
        const bool gen = !kPlain && G.Cin == nullptr;
        // The loads are unconditional (columns past the tile's end and stages past
        // the last one repeat valid addresses and are not used): a load under a
        // condition is merged with the value it replaces, which waits for it.
        int luse = 0, lst = 0;                    // the next stage to load
        const float *cp[2], *rp[2];
        float rj[2];
        auto start_item = [&]() {
            const int item = blockIdx.x + luse * gridDim.x;
            const int b = item / per_box, t = (item - b * per_box) / G.mt;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int cc = min(col + 8 * kLWork * u, NC - 1), j = min(t * NC + cc, G.d - 1);
                const size_t o = t * tile + (size_t)(j - t * NC) * cs + 4 * q;
                cp[u] = gen ? G.W0b + o : G.Cin + b * boxs + o;
                rp[u] = gen ? cp[u] : G.Rin + b * boxs + o;
                rj[u] = gen ? G.rr[(size_t)b * G.d + j] : 0.f;
            }
        };
        start_item();
        auto load = [&](Raw &v) {
            // (inputs from n_in to the end of the last stage lie within the tile
            // and their plan is zero)
            const size_t o = (size_t)lst * ks;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                v.c[u] = *reinterpret_cast<const float4 *>(cp[u] + o);
                v.r[u] = *reinterpret_cast<const float4 *>(rp[u] + o);
                v.rj[u] = rj[u];
            }
            if (++lst == nst) {
                lst = 0;
                if (luse + 1 < mine) ++luse;
                start_item();
            }
        };
        // the relaxation of the stage to produce: the same few lines for every
        // warp, so one stage ahead is enough
        float4 pp, qq;
        auto load_plan = [&](int use, int st) {
            if (kPlain) return;
            const float *pl = G.plan + (size_t)((blockIdx.x + min(use, mine - 1) * gridDim.x) / per_box) * 2 * G.NP + st * kLK + 4 * q;
            pp = *reinterpret_cast<const float4 *>(pl);
            qq = *reinterpret_cast<const float4 *>(pl + G.NP);
        };
        int use = 0, st = 0, done = 0;            // item and stage to produce, items drained
        int s = 0, round = 0;                     // ring position
        auto produce = [&](Raw &v) -> bool {
            // the ring holds kBStages stages: a tile is drained once the next one's are in it
            while (done < use - (st >= kBStages ? 0 : 1))
                if (++done, warp < kLEpi && !epilogue(done - 1)) return false;
            if (round > 0 && !mbar_wait(smem_u32(&bempty[s]), (uint32_t)((round - 1) & 1), kLWait)) ok = false;
            if (__any_sync(0xffffffffu, !ok)) {
                ok = false;
                return false;
            }
            unsigned char *to = sB + s * bstage + (q >> 1) * bstep + (q & 1) * kLLboB;
            const float pv[4] = {pp.x, pp.y, pp.z, pp.w}, qv[4] = {qq.x, qq.y, qq.z, qq.w};
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int cc = col + 8 * kLWork * u;
                const float c0[4] = {v.c[u].x, v.c[u].y, v.c[u].z, v.c[u].w};
                const float r0[4] = {v.r[u].x, v.r[u].y, v.r[u].z, v.r[u].w};
                float c[4], r[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (kPlain) {
                        const bool in = st * kLK + 4 * q + e < G.n_in;
                        c[e] = in ? c0[e] : 0.f;
                        r[e] = in ? r0[e] : 0.f;
                    } else {
                        relax_pair(pv[e], qv[e], gen ? __fmul_rn(c0[e], v.rj[u]) : c0[e], gen ? 0.f : r0[e], c[e], r[e]);
                    }
                }
                if (cc < NC) {
                    unsigned char *o = to + (cc >> 3) * kLSboB + (cc & 7) * 16;
                    split4<kPlain>(c, o, o + bimg);
                    split4<kPlain>(r, o + 2 * bimg, o + 3 * bimg);
                }
            }
            if (++st == nst) {
                st = 0;
                ++use;
            }
            load(v);                              // two stages ahead
            load_plan(use, st);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bfull[s]));
            if (++s == kBStages) {
                s = 0;
                ++round;
            }
            return true;
        };
        Raw v0, v1;
        load(v0);
        load(v1);
        load_plan(0, 0);
        const int stages = mine * nst;
        for (int g = 0; g < stages; g += 2) {
            if (!produce(v0)) break;
            if (g + 1 < stages && !produce(v1)) break;
        }
        while (ok && done < mine)
            if (++done, warp < kLEpi && !epilogue(done - 1)) break;
        if (!ok) *sAbort = 1;
    } else if (warp == kLWork) {
        // ---- products ----
        if (lane == 0) {
            // kind::tf32, FP32 accumulate, both operands K-major, N = NC, M = 128
            const uint32_t idesc = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(NC >> 3) << 17) |
                                   ((uint32_t)(kLRows >> 4) << 24);
            auto commit = [](uint64_t *bar) {
                asm volatile(
                    "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                    : "memory");
            };
            const uint64_t da0 = umma_desc(smem_u32(sA), kLLboA, kLSboA), db0 = umma_desc(smem_u32(sB), kLLboB, kLSboB);
            int sa = 0, ra = 0, sb = 0, rb = 0, use = 0;
            for (; use < mine && ok; ++use) {
                if (use > 0 && !mbar_wait(smem_u32(tempty), (uint32_t)((use - 1) & 1), kLWait)) ok = false;
                asm volatile("tcgen05.fence::after_thread_sync;");
                for (int st = 0; st < nst && ok; ++st) {
                    if (!mbar_wait(smem_u32(&afull[sa]), (uint32_t)(ra & 1), kLWait) ||
                        !mbar_wait(smem_u32(&bfull[sb]), (uint32_t)(rb & 1), kLWait)) {
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;");
                    // (an address in a descriptor is in units of 16 bytes; the ring stays within its field)
                    const uint64_t da1 = da0 + (uint32_t)(sa * kLA >> 4), db1 = db0 + (uint32_t)(sb * bstage >> 4);
#pragma unroll
                    for (int k = 0; k < kLK / kLStep; ++k) {
#pragma unroll
                        for (int eq = 0; eq < 2; ++eq) {
                            const uint64_t ah = da1 + (uint32_t)((k * kLAStep + 2 * eq * kLAImg) >> 4);
                            const uint64_t al = ah + (uint32_t)(kLAImg >> 4);
                            const uint64_t bh = db1 + (uint32_t)((k * bstep + 2 * eq * bimg) >> 4);
                            const uint64_t bl = bh + (uint32_t)(bimg >> 4);
                            const uint64_t pa[3] = {ah, al, ah}, pb[3] = {bl, bh, bh};
#pragma unroll
                            for (int ps = 0; ps < 3; ++ps) {
                                const uint32_t acc = (st > 0 || k > 0 || ps > 0) ? 1u : 0u;
                                asm volatile(
                                    "{ .reg .pred p; setp.ne.b32 p, %4, 0; "
                                    "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p; }" ::"r"(
                                        tmem + eq * kLTmemR),
                                    "l"(pa[ps]), "l"(pb[ps]), "r"(idesc), "r"(acc));
                            }
                        }
                    }
                    commit(&aempty[sa]);
                    commit(&bempty[sb]);
                    if (++sa == NA) {
                        sa = 0;
                        ++ra;
                    }
                    if (++sb == kBStages) {
                        sb = 0;
                        ++rb;
                    }
                }
                // (also after a timeout: what was issued completes and is waited for below)
                commit(tfull);
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
                const unsigned char *src = G.Aimg + (size_t)(item % G.mt) * nst * kLA;
                for (int st = 0; st < nst; ++st) {
                    if (round > 0 && !mbar_wait(smem_u32(&aempty[s]), (uint32_t)((round - 1) & 1), kLWait)) ok = false;
                    if (!ok) break;
                    const uint32_t bar = smem_u32(&afull[s]);
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(kLA)
                                 : "memory");
                    asm volatile(
                        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                            smem_u32(sA + s * kLA)),
                        "l"(src + (size_t)st * kLA), "r"(kLA), "r"(bar)
                        : "memory");
                    if (++s == NA) {
                        s = 0;
                        ++round;
                    }
                }
            }
            if (!ok) {
                *sAbort = 1;
                // the copies in flight land: the last one of each stage completes its barrier's phase
                for (int k = 0; k < NA; ++k) {
                    const int uses = round + (k < s ? 1 : 0);
                    if (uses > 0) mbar_wait(smem_u32(&afull[k]), (uint32_t)((uses - 1) & 1), kLWait);
                }
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

// Weight pieces of one layer as the ring's stages: row tile m, step k at
// out + (m steps + k) kLAStep bytes, each [W hi | W lo | |W| hi | |W| lo] of
// 128 rows by 8 inputs in core matrices.  The row-major pieces are zero padded
// to multiples of 128 rows and 32 inputs (ld floats).
__global__ void wide_pack_kernel(const float *hi, const float *lo, const float *ahi, const float *alo, int ld, int mt,
                                 int steps, float *out) {
    const int total = mt * steps * 4 * kLRows * kLStep;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
        const int w = t % (kLRows * kLStep), img = t / (kLRows * kLStep) % 4, ms = t / (4 * kLRows * kLStep);
        const int k = w % kLStep, r = w / kLStep;
        const float *src = img == 0 ? hi : (img == 1 ? lo : (img == 2 ? ahi : alo));
        const float v = src[(size_t)(ms / steps * kLRows + r) * ld + ms % steps * kLStep + k];
        out[(size_t)ms * (kLAStep / 4) + img * (kLAImg / 4) +
            ((r >> 3) * kLSboA + (k >> 2) * kLLboA + (r & 7) * 16) / 4 + (k & 3)] = v;
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
// rows of one box, the d coefficients of a row in 16 runs of neighbouring
// inputs (the box in shared memory, read four inputs at a time: one scalar
// load of each of m, l and r per term took twice as long), merged in shared
// memory; constant and error as in wide_init_kernel.
constexpr int kP1X = 32, kP1Y = 16;

__host__ __device__ inline int plan1_run(int d) { return ((d + kP1Y - 1) / kP1Y + 3) & ~3; }

__global__ void __launch_bounds__(kP1X * kP1Y, 2)
wide_plan1_kernel(const NetParams<float> net, const float *W0t, int NP, const float *mh, const float *ml,
                  const float *rr, float *plan, float *S3, float *Ch, float *Cl, const float *alpha, int64_t alpha_ld,
                  int64_t base) {
    using A = Arith<float>;
    extern __shared__ __align__(16) float sbox[];   // m hi, m lo, r: zero past d
    __shared__ float part[4][kP1Y][kP1X];
    const int d = net.d, n1 = net.n[1];
    const int lane = threadIdx.x, sl = threadIdx.y;
    const int p = blockIdx.x * kP1X + lane;
    const int64_t b = blockIdx.y;
    const int run = plan1_run(d), dp = run * kP1Y;
    for (int j = sl * kP1X + lane; j < dp; j += kP1X * kP1Y) {
        sbox[j] = j < d ? mh[b * d + j] : 0.f;
        sbox[dp + j] = j < d ? ml[b * d + j] : 0.f;
        sbox[2 * dp + j] = j < d ? rr[b * d + j] : 0.f;
    }
    __syncthreads();
    float S = 0.f, s = 0.f, e = 0.f, sabs = 0.f;
    if (p < n1) {
        if (sl == 0) {
            s = net.b[0][p];
            sabs = fabsf(s);
        }
        const int j1 = min(d, (sl + 1) * run);
#pragma unroll 2
        for (int j = sl * run; j < j1; j += 4) {
            float m[4], l[4], r[4], w[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) w[u] = W0t[(size_t)min(j + u, d - 1) * n1 + p];
            const float4 m4 = *reinterpret_cast<const float4 *>(sbox + j);
            const float4 l4 = *reinterpret_cast<const float4 *>(sbox + dp + j);
            const float4 r4 = *reinterpret_cast<const float4 *>(sbox + 2 * dp + j);
            m[0] = m4.x; m[1] = m4.y; m[2] = m4.z; m[3] = m4.w;
            l[0] = l4.x; l[1] = l4.y; l[2] = l4.z; l[3] = l4.w;
            r[0] = r4.x; r[1] = r4.y; r[2] = r4.z; r[3] = r4.w;
            // (terms past d are zeros)
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                S = A::add_up(S, fabsf(A::mul_rn(w[u], r[u])));
                float p1, pe, tt, se;
                two_prod<float>(w[u], m[u], p1, pe);
                two_sum<float>(s, p1, tt, se);
                s = tt;
                e = A::fma_rn(w[u], l[u], e + (pe + se));
                sabs = sabs + fabsf(p1);
            }
        }
    }
    part[0][sl][lane] = S;
    part[1][sl][lane] = s;
    part[2][sl][lane] = e;
    part[3][sl][lane] = sabs;
    __syncthreads();
    if (sl != 0) return;
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

namespace {

// Four neighbouring inputs of one box, as the affine step of the small columns
// reads them: constant (float-float), radius constant, N, E.
struct Small4 {
    float h[4], l[4], rd[4], N[4], E[4];
};
__device__ __forceinline__ void ld4(const float *p, float (&v)[4]) {
    const float4 t = *reinterpret_cast<const float4 *>(p);
    v[0] = t.x;
    v[1] = t.y;
    v[2] = t.z;
    v[3] = t.w;
}

// The affine step of one output row's small columns: the constant
// sum_i w_i (h_i + l_i) + b (error-free products, compensated sums) with its
// error bound (on the property layer the fold's too), and |w| times the radius
// constant, N and E (FP32 FMA chains, rounding within gamma_{n_in}).
struct SmallRow {
    float chi, clo, cerr, rd, N, E;
};
__device__ __forceinline__ SmallRow small_row(const NetParams<float> &net, int k, int NP, int64_t b, int p,
                                              const float *S3, const float *Ch, const float *Cl) {
    using A = Arith<float>;
    const int n_in = net.n[k], n_out = net.n[k + 1];
    const bool last = k + 1 == net.K;
    const float *Wt = net.Wt[k] + p;
    const float *s3 = S3 + (size_t)b * 3 * NP, *ch = Ch + (size_t)b * NP, *cl = Cl + (size_t)b * NP;
    float s = net.b[k][p], e = 0.f, a = fabsf(s), f = 0.f;
    SmallRow o{0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 2
    for (int i0 = 0; i0 < n_in; i0 += 4) {
        // (the arrays hold NP entries a box, zeros past the layer's width)
        Small4 v;
        ld4(ch + i0, v.h);
        ld4(cl + i0, v.l);
        ld4(s3 + i0, v.rd);
        ld4(s3 + NP + i0, v.N);
        ld4(s3 + 2 * NP + i0, v.E);
        float w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) w[u] = Wt[(size_t)min(i0 + u, n_in - 1) * n_out];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (i0 + u >= n_in) continue;
            float p1, pe, t, se;
            two_prod<float>(w[u], v.h[u], p1, pe);
            two_sum<float>(s, p1, t, se);
            s = t;
            e = A::fma_rn(w[u], v.l[u], e + (pe + se));
            a = a + fabsf(p1);
            const float aw = fabsf(w[u]);
            o.rd = A::fma_rn(aw, v.rd[u], o.rd);
            o.N = A::fma_rn(aw, v.N[u], o.N);
            o.E = A::fma_rn(aw, v.E[u], o.E);
            if (last) {
                const float z = A::add_up(A::add_up(fabsf(v.N[u]), fabsf(v.h[u])),
                                          A::add_up(fabsf(v.l[u]), fabsf(v.E[u])));
                f = A::add_up(f, A::mul_up(net.fold_err[p * n_in + i0 + u], z));
            }
        }
    }
    const float g = gam<float>(n_in + 2);
    two_sum<float>(s, e, o.chi, o.clo);
    o.cerr = A::mul_up(A::mul_up(2.f * g, g), A::mul_up(a, 1.f + gam<float>(n_in)));
    if (last) o.cerr = A::add_up(o.cerr, A::add_up(f, net.fold_berr[p]));
    return o;
}

// E' = |W| E (1 + 2 g) + g |W| N (1 + g) + the constant's error
__device__ __forceinline__ float small_error(const SmallRow &o, float g, int n_in) {
    using A = Arith<float>;
    float eps = A::mul_up(g, A::mul_up(o.N, 1.f + g));
    eps = A::add_up(A::add_up(eps, o.cerr), (float)(n_in + 4) * A::tiny);
    return A::add_up(A::mul_up(o.E, 1.f + 2.f * g), eps);
}

}  // namespace

// Hidden layer `layer` after its product: the small columns (radius constant,
// N, E, constant) from the previous layer's (S3, Ch, Cl), the bound sums of the
// product's tiles -> error, bounds, relaxation, into plan and (S3o, Cho, Clo).
// One thread per row.
__global__ void __launch_bounds__(128)
wide_plan_kernel(const NetParams<float> net, int layer, int NP, float gcoef, const float *part, int nparts,
                 const float *S3, const float *Ch, const float *Cl, float *plan, float *S3o, float *Cho, float *Clo,
                 const float *alpha, int64_t alpha_ld, int64_t base) {
    const int p = blockIdx.x * 128 + threadIdx.x;
    const int64_t b = blockIdx.y;
    if (p >= NP) return;
    RelaxPlan<float> pl;
    pl.kind = 1;
    pl.pp = pl.qq = pl.nh = pl.nl = pl.rd = pl.N = pl.E = 0.f;
    if (p < net.n[layer]) {
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
        const SmallRow sr = small_row(net, layer - 1, NP, b, p, S3, Ch, Cl);
        const float E = small_error(sr, gcoef, net.n[layer - 1]);
        t.finish(sr.chi, sr.clo, sr.rd);
        const float *a_ptr = nullptr;
        if (alpha != nullptr) {
            int off = 0;
            for (int j = 1; j < layer; ++j) off += net.n[j];
            a_ptr = alpha + (base + b) * alpha_ld + off + p;
        }
        pl = WTile::plan_row(t, net.d, net.relax_mode, sr.chi, sr.clo, sr.rd, E, a_ptr, net.act[layer - 1]);
    }
    store_plan(pl, plan, S3o, Cho, Clo, b, NP, p);
}

// The property layer: relaxation of the last hidden layer and the products of
// its few rows.  Eight lanes share a column (one input coefficient of both
// equations): each takes four neighbouring inputs of every 32, so that a load
// of a warp reads 256-byte runs, and the weights, stored by row, come
// without bank conflicts; every lane group takes kRowsCols columns at a time.
// The lanes' partial sums are added by shuffles (rounding within
// gamma_{n_in} of sum |W| |x| in any order).  Row r of column j of box b goes
// to out[((b d + j) 2 + eq) RM + r].
constexpr int kRowsCols = 2;

template <int RM>
__global__ void __launch_bounds__(256, 2)
wide_rows_kernel(const NetParams<float> net, int NP, int ntile, int NC, const float *Cin, const float *Rin,
                 const float *W0b, const float *rr, const float *plan, int64_t ncols, float *out) {
    extern __shared__ __align__(16) float sWr[];   // RM x n32, zero beyond R and n_in
    const int K = net.K, n_in = net.n[K - 1], R = net.R, d = net.d;
    const int n32 = (n_in + 31) & ~31;             // at most the state's row stride NP
    for (int q = threadIdx.x; q < n32 * RM; q += blockDim.x) {
        const int r = q / n32, i = q - r * n32;
        sWr[q] = r < R && i < n_in ? net.Wt[K - 1][(size_t)i * R + r] : 0.f;
    }
    __syncthreads();
    const bool gen = Cin == nullptr;
    const int g8 = threadIdx.x >> 3, l8 = threadIdx.x & 7;
    const int64_t step = (int64_t)gridDim.x * 32 * kRowsCols;
    // (a warp's lanes make the same trips: its 4 groups take 4 kRowsCols columns together)
    for (int64_t c0 = (int64_t)blockIdx.x * 32 * kRowsCols; c0 < ncols; c0 += step) {
        float ac[kRowsCols][RM], ar[kRowsCols][RM];
        const float *cp[kRowsCols], *rp[kRowsCols], *pl[kRowsCols];
        float rj[kRowsCols];
#pragma unroll
        for (int u = 0; u < kRowsCols; ++u) {
#pragma unroll
            for (int r = 0; r < RM; ++r) ac[u][r] = ar[u][r] = 0.f;
            // columns past the end repeat the last one and are not stored
            const int64_t col = min(c0 + u * 32 + g8, ncols - 1), b = col / d;
            pl[u] = plan + (size_t)b * 2 * NP + 4 * l8;
            const int j = (int)(col - b * d), t = j / NC;
            const size_t o = (size_t)(l8 >> 2) * NC * kLK + (size_t)(j - t * NC) * kLK + 4 * (l8 & 3);
            cp[u] = (gen ? W0b + (size_t)t * NC * NP : Cin + ((size_t)b * ntile + t) * NC * NP) + o;
            rp[u] = gen ? cp[u] : Rin + ((size_t)b * ntile + t) * NC * NP + o;
            rj[u] = gen ? rr[col] : 0.f;
        }
#pragma unroll 1
        for (int i = 0; i < n32; i += 32) {
            float c[kRowsCols][4], x[kRowsCols][4];
#pragma unroll
            for (int u = 0; u < kRowsCols; ++u) {
                const float4 c4 = *reinterpret_cast<const float4 *>(cp[u] + (size_t)i * NC);
                const float4 r4 =
                    gen ? make_float4(0.f, 0.f, 0.f, 0.f) : *reinterpret_cast<const float4 *>(rp[u] + (size_t)i * NC);
                const float4 p4 = *reinterpret_cast<const float4 *>(pl[u] + i);
                const float4 q4 = *reinterpret_cast<const float4 *>(pl[u] + NP + i);
                const float cv[4] = {c4.x, c4.y, c4.z, c4.w}, rv[4] = {r4.x, r4.y, r4.z, r4.w};
                const float pv[4] = {p4.x, p4.y, p4.z, p4.w}, qv[4] = {q4.x, q4.y, q4.z, q4.w};
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    relax_pair(pv[e], qv[e], gen ? __fmul_rn(cv[e], rj[u]) : cv[e], rv[e], c[u][e], x[u][e]);
            }
#pragma unroll
            for (int r = 0; r < RM; ++r) {
                const float4 w4 = *reinterpret_cast<const float4 *>(sWr + r * n32 + i + 4 * l8);
                const float w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
                for (int u = 0; u < kRowsCols; ++u)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        ac[u][r] = fmaf(w[e], c[u][e], ac[u][r]);
                        ar[u][r] = fmaf(fabsf(w[e]), x[u][e], ar[u][r]);
                    }
            }
        }
#pragma unroll
        for (int u = 0; u < kRowsCols; ++u) {
#pragma unroll
            for (int r = 0; r < RM; ++r)
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) {
                    ac[u][r] += __shfl_xor_sync(0xffffffffu, ac[u][r], o);
                    ar[u][r] += __shfl_xor_sync(0xffffffffu, ar[u][r], o);
                }
            const int64_t col = c0 + u * 32 + g8;
            if (col < ncols && l8 < RM / 4) {
                float *o = out + (size_t)col * 2 * RM + 4 * l8;
#pragma unroll
                for (int k = 0; k < RM / 4; ++k)
                    if (k == l8) {
                        *reinterpret_cast<float4 *>(o) =
                            make_float4(ac[u][4 * k], ac[u][4 * k + 1], ac[u][4 * k + 2], ac[u][4 * k + 3]);
                        *reinterpret_cast<float4 *>(o + RM) =
                            make_float4(ar[u][4 * k], ar[u][4 * k + 1], ar[u][4 * k + 2], ar[u][4 * k + 3]);
                    }
            }
        }
    }
}

// Property rows of one box per block: sound bounds lo = min L' - E, hi = max U' + E
// (Sec. 3 check) from the columns of wide_rows_kernel and the small columns.
// blockDim.x = 32 R: warp w sums row w; the first R threads take the small columns.
__global__ void wide_rows_final_kernel(const NetParams<float> net, int NP, int RM, float gcoef, const float *cols,
                                       const float *S3, const float *Ch, const float *Cl, float *lo, float *hi,
                                       float *err) {
    using A = Arith<float>;
    __shared__ RowBounds<float> sums[16];
    const int d = net.d, R = net.R, K = net.K;
    const int r = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t b = blockIdx.x;
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
    if (lane == 0) sums[r] = t;
    __syncthreads();
    if (threadIdx.x >= R) return;
    const int p = threadIdx.x;
    t = sums[p];
    const SmallRow sr = small_row(net, K - 1, NP, b, p, S3, Ch, Cl);
    const float E = small_error(sr, gcoef, net.n[K - 1]);
    t.finish(sr.chi, sr.clo, sr.rd);
    lo[b * R + p] = A::add_dn(t.ll, -E);
    hi[b * R + p] = A::add_up(t.uu, E);
    err[b * R + p] = A::add_up(E, t.delta);
}

// ---------------------------------------------------------------------------
// launch wrappers
// ---------------------------------------------------------------------------

// Column tiles of a box: the fewest of at most kLCols columns, each a multiple of 16.
void wide_layer_tiles(int d, int &ntile, int &NC) {
    ntile = (d + kLCols - 1) / kLCols;
    NC = ((d + ntile - 1) / ntile + 15) & ~15;
}

size_t wide_layer_img_bytes(int n_in, int n_out) {
    return (size_t)((n_out + kLRows - 1) / kLRows) * ((n_in + kLK - 1) / kLK) * kLA;
}

cudaError_t launch_wide_pack(const float *hi, const float *lo, const float *ahi, const float *alo, int ld, int n_in,
                             int n_out, void *out, cudaStream_t s) {
    const int mt = (n_out + kLRows - 1) / kLRows, steps = (n_in + kLK - 1) / kLK * (kLK / kLStep);
    const int total = mt * steps * 4 * kLRows * kLStep;
    wide_pack_kernel<<<std::min(1024, (total + 255) / 256), 256, 0, s>>>(hi, lo, ahi, alo, ld, mt, steps,
                                                                         (float *)out);
    return cudaGetLastError();
}

template <bool kPlain>
static cudaError_t launch_layer(WideLayer G, int sms, cudaStream_t s) {
    G.mt = (G.n_out + kLRows - 1) / kLRows;
    G.nst = (G.n_in + kLK - 1) / kLK;
    wide_layer_tiles(G.d, G.ntile, G.NC);
    const int64_t items = (int64_t)G.nb * G.ntile * G.mt;
    if (items <= 0) return cudaSuccess;
    if (items > INT32_MAX) return cudaErrorInvalidValue;
    G.na = a_stages(G.NC);
    const int smem = G.na * kLA + kBStages * b_stage(G.NC) + kLBar;
    cudaError_t e = allow_smem(wide_layer_kernel<kPlain>);
    if (e != cudaSuccess) return e;
    wide_layer_kernel<kPlain><<<(int)std::min<int64_t>(items, sms), kLThreads, smem, s>>>(G);
    return cudaGetLastError();
}

cudaError_t launch_wide_layer(const WideLayer &G, int sms, cudaStream_t s) { return launch_layer<false>(G, sms, s); }

cudaError_t launch_wide_product(const WideLayer &G, int sms, cudaStream_t s) { return launch_layer<true>(G, sms, s); }

cudaError_t launch_wide_plan1(const NetParams<float> &net, const float *W0t, int nb, int NP, const float *mh,
                              const float *ml, const float *rr, float *plan, float *S3, float *Ch, float *Cl,
                              const float *alpha, int64_t alpha_ld, int64_t base, cudaStream_t s) {
    // (12 KB at most: no need to ask for it)
    const int smem = 3 * plan1_run(net.d) * kP1Y * (int)sizeof(float);
    wide_plan1_kernel<<<dim3(NP / kP1X, nb), dim3(kP1X, kP1Y), smem, s>>>(net, W0t, NP, mh, ml, rr, plan, S3, Ch, Cl,
                                                                          alpha, alpha_ld, base);
    return cudaGetLastError();
}

cudaError_t launch_wide_plan(const NetParams<float> &net, int layer, int nb, int NP, float gcoef, const float *part,
                             const float *S3, const float *Ch, const float *Cl, float *plan, float *S3o, float *Cho,
                             float *Clo, const float *alpha, int64_t alpha_ld, int64_t base, cudaStream_t s) {
    int ntile, NC;
    wide_layer_tiles(net.d, ntile, NC);
    wide_plan_kernel<<<dim3((NP + 127) / 128, nb), 128, 0, s>>>(net, layer, NP, gcoef, part, 3 * ntile, S3, Ch, Cl, plan,
                                                                S3o, Cho, Clo, alpha, alpha_ld, base);
    return cudaGetLastError();
}

// Rows of a column's record, R rounded up to a multiple of 4 (R <= 16).
int wide_rows_stride(int R) { return (R + 3) & ~3; }

cudaError_t launch_wide_rows(const NetParams<float> &net, int nb, int NP, const float *Cin, const float *Rin,
                             const float *W0b, const float *rr, const float *plan, float *out, int sms,
                             cudaStream_t s) {
    const int64_t ncols = (int64_t)nb * net.d;
    int ntile, NC;
    wide_layer_tiles(net.d, ntile, NC);
    const int grid = (int)std::min<int64_t>((ncols + 32 * kRowsCols - 1) / (32 * kRowsCols), (int64_t)sms * 8);
    const int RM = wide_rows_stride(net.R);
    const size_t smem = (size_t)((net.n[net.K - 1] + 31) & ~31) * RM * sizeof(float);
    auto run = [&](auto k) -> cudaError_t {
        cudaError_t e = allow_smem(k);
        if (e != cudaSuccess) return e;
        k<<<grid, 256, smem, s>>>(net, NP, ntile, NC, Cin, Rin, W0b, rr, plan, ncols, out);
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
                                   const float *S3, const float *Ch, const float *Cl, float *lo, float *hi, float *err,
                                   cudaStream_t s) {
    wide_rows_final_kernel<<<nb, 32 * net.R, 0, s>>>(net, NP, wide_rows_stride(net.R), gcoef, cols, S3, Ch, Cl, lo, hi,
                                                     err);
    return cudaGetLastError();
}

}  // namespace slr
