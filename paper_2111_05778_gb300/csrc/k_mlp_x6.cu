// Neural SDB on the tensor cores at FP32 accuracy: split-BF16 products.  This
// is the FP32 evaluator of networks up to x6_max_mid() hidden layers (deeper
// ones run on the FFMA engine, k_mlp_fp32.cu): FP32 hopping, vertex values,
// the refinement of the BF16 path, point lists, the enumeration lattice and
// the adjoint's forward pass and delta chain.
//
// Every FP32 operand x of a hidden layer is split exactly into three BF16
// parts, x = x_h + x_m + x_l (x_h = bf16(x), x_m = bf16(x - x_h), x_l =
// bf16(x - x_h - x_m)); each difference is exact in FP32 and the three parts
// carry 24 significant bits.  Of the nine part products of a * w the six
// whose size is at least 2^-16 |a w| are formed on the tensor core (hh, hm,
// mh, hl, lh, mm) with FP32 accumulation in tensor memory; the three dropped
// (ml, lm, ll) are below 2^-23 |a w| together, the size of one FP32 rounding.
// The accumulator adds the products from the smallest to the largest in four
// passes over the layer's inputs: x_h w_l; x_m w_m and x_h w_m; x_l w_h and
// x_m w_h; x_h w_h.  Only the last pass's W/16 updates are at the size of the
// result.  The accumulator is truncated toward zero; the epilogue adds back what
// that loses on average, by the width and, where an output has few weights, by
// their number (gh_internal.cuh: kappa_row; a selection loses nothing and gets
// nothing).  On dense layers what remains is below the error of a chain of FP32
// FMAs (deviation 0.3 / 0.4 / 0.6 units in the last place at width 64 / 128 / 256
// for terms of one sign, the chain's 1.2 / 1.6 / 2.2).  Dense weights of which
// few see a nonzero activation are corrected too much, by at most the constant.
// The last two passes share the high part's stages in the ring.  Layer 0
// (3 -> W) and the output layer (W -> 1) run on CUDA cores in FP32.
//
// Persistent CTAs, one 128-row tile at a time each, 64 + 2 W threads:
//   warp 0       bulk-copy producer: K-blocks (64 inputs x W outputs) of one
//                weight part per stage, stored pre-swizzled in global
//                memory, into a 4-stage shared-memory ring.
//   warp 1       allocates TMEM (2W columns); one lane issues tcgen05.mma
//                (M = 128, N = W, K = 16): A = x_h or x_m from tensor memory,
//                or x_l from shared memory.
//   warps 2..    epilogue, W/64 threads per row, 64 columns (one K-block of
//                the next layer) each: layer 0, TMEM -> registers -> bias,
//                ReLU, the exact three-way split -> x_h and x_m into tensor
//                memory, x_l into 128B-swizzled shared memory (the next
//                layer's A operands); the output dot product; the hop step of
//                Algorithm 1 or the store of f.
// A thread holds its 64 columns in registers, so the accumulator is free and
// the next layer's first pass (x_h only) starts as soon as x_h is stored; the
// middle and low parts are computed under it (barriers a_h and a_ml).
// x_l, which only one of the six products reads, is the part in shared memory:
// its port carries the weights' copies and the B operands already, and runs
// of products with A in shared memory took 183 cycles each at width 256,
// with A in tensor memory 122.
// TMEM columns: [0, W) accumulator, [W, 3W/2) x_h, [3W/2, 2W) x_m (two BF16
// per 32-bit column, K ascending).  Every wait is bounded as in the BF16
// engine; a timeout sets the error flag, every role leaves, copies in flight
// land and MMAs complete before TMEM is freed.
#include <stdint.h>

#include "gh_internal.cuh"
#include "tc_ptx.cuh"

namespace gh {

namespace {

using namespace tc;

constexpr int TM = 128;   // rows per tile
constexpr int NPASS = 4;  // weight passes per layer: low, middle, high (with x_l, x_m), high (with x_h)
constexpr int EPI_T0 = 64;  // first epilogue thread (warp 2)
constexpr int MAXMID = 8;
constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr uint32_t NONE = 0xFFFFFFFFu;
constexpr int BAR_EPI = 1;  // named barrier of the epilogue threads

enum { XM_HOP = 0, XM_VERTS = 1, XM_REFINE = 2, XM_POINTS = 3, XM_LATTICE = 4, XM_ADJ = 5 };

// Resident CTAs per SM the registers are budgeted for: TMEM (2W of 512
// columns) and shared memory (217 / 105 / 53 KB) allow 1, 2 and 4; at width
// 64 three CTAs leave the threads the registers that four would spill.
template <int W>
constexpr int ctas_of() {
    return W == 256 ? 1 : (W == 128 ? 2 : 3);
}

// Weight ring stages: a divisor of the 3 W/64 stages of a layer, so that the
// K-blocks of every layer fall on the same stages and the issuing thread's
// loop over a layer is straight-line code with constant stage addresses and
// barriers.  (Computing them per stage cost that thread about 400 cycles: 728
// cycles for a stage of four products instead of the 512 of the products.)
template <int W>
constexpr int nst_of() {
    return W == 256 ? 4 : 3;
}

__device__ __forceinline__ float pow2_of(float v) { return __uint_as_float(__float_as_uint(v) & 0xFF800000u); }

template <int W>
struct SmemX {
    static constexpr int NST = nst_of<W>();
    uint8_t al[W / 64][TM * 128];  // x_l: K-blocks of 128 rows x 128 B (1024-aligned)
    uint8_t w[NST][W * 128];       // weight ring: one K-block of one part per stage
    float4 w0b[W];                 // layer-0 rows and biases by output pairs
    float bmid[MAXMID * W];        // hidden-layer biases
    float wout[W];                 // output-layer weights
    float4 pt[TM];                 // the tile's points
    float red[3][W / 64][TM];      // per column group: output dot products (adjoint: grad_x g)
    unsigned long long full[NST], empty[NST], acc_full, a_h, a_ml, item_ready, drain;
    const uint16_t *cur_w;         // split weights of the current item
    uint32_t kbits[2];             // layers and column groups whose outputs have their own correction (MlpDev::kbits)
    int done;
    uint32_t tmem_base;
    int ctl;
};

// BF16 parts of two values, packed (x0 in the low half): the high part ...
__device__ __forceinline__ uint32_t part_h(float x0, float x1) {
    uint32_t h;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(h) : "f"(x1), "f"(x0));
    return h;
}
// ... and the middle and low ones: x = h + m + l, every difference exact.
__device__ __forceinline__ void parts_ml(float x0, float x1, uint32_t &m, uint32_t &l) {
    const uint32_t h = part_h(x0, x1);
    const float r0 = x0 - __uint_as_float(h << 16), r1 = x1 - __uint_as_float(h & 0xFFFF0000u);
    m = part_h(r0, r1);
    l = part_h(r0 - __uint_as_float(m << 16), r1 - __uint_as_float(m & 0xFFFF0000u));
}

__device__ __forceinline__ float outer_f(const MlpDev &m, float x, float y, float z, float g) {
    const float r = sqrtf(fmaf(x, x, fmaf(y, y, z * z)));
    return (fmaf(m.alpha, g, m.radial * r - m.r0) / m.beta) * m.inv_lam;
}

// Loads an item's layer-0 rows, biases and output weights (epilogue threads).
template <int W, bool OWN>
__device__ __forceinline__ void load_params(SmemX<W> &sm, const MlpDev &mm, int e) {
    for (int o = e; o < W; o += 2 * W) {
        float *q = reinterpret_cast<float *>(&sm.w0b[o & ~1]) + (o & 1);
        q[0] = mm.w0[3 * o];
        q[2] = mm.w0[3 * o + 1];
        q[4] = mm.w0[3 * o + 2];
        q[6] = mm.b0[o];
        sm.wout[o] = mm.wout[o];
    }
    for (int i = e; i < mm.n_mid * W; i += 2 * W) sm.bmid[i] = mm.bm[i];
    if (OWN && e < 2) sm.kbits[e] = mm.kbits[e];
}

// x[64] (this thread's row, columns 64 grp .., ReLU'd when RELU) -> x_h into
// tensor memory (32 columns of two inputs each).  The ReLU is the conversion's,
// so that x_h, which the next layer's first products wait for, takes as few
// instructions as can be.
template <bool RELU>
__device__ __forceinline__ void put_h(const float (&x)[64], uint32_t th) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        uint32_t h[8];
#pragma unroll
        for (int p = 0; p < 8; ++p)
            h[p] = RELU ? pack_relu_bf16(x[16 * c + 2 * p], x[16 * c + 2 * p + 1])
                        : part_h(x[16 * c + 2 * p], x[16 * c + 2 * p + 1]);
        tmem_st8(th + 8 * c, h);
    }
    tmem_wait_st();
}

// x_m into tensor memory, x_l into K-block grp of the shared-memory operand
template <bool RELU>
__device__ __forceinline__ void put_ml(const float (&x)[64], uint32_t tm, uint32_t lrow, int sw) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        uint32_t m[8], l[8];
#pragma unroll
        for (int p = 0; p < 8; ++p) {
            const float x0 = x[16 * c + 2 * p], x1 = x[16 * c + 2 * p + 1];
            parts_ml(RELU ? relu_nan(x0) : x0, RELU ? relu_nan(x1) : x1, m[p], l[p]);
        }
        tmem_st8(tm + 8 * c, m);
        sts128(lrow + (uint32_t)(((2 * c) ^ sw) << 4), l[0], l[1], l[2], l[3]);
        sts128(lrow + (uint32_t)(((2 * c + 1) ^ sw) << 4), l[4], l[5], l[6], l[7]);
    }
    tmem_wait_st();
}

// bit c set where x[c] > 0
__device__ __forceinline__ uint2 relu_bits(const float (&x)[64]) {
    uint2 b = make_uint2(0u, 0u);
#pragma unroll
    for (int c = 0; c < 32; ++c) {
        b.x |= (x[c] > 0.f ? 1u : 0u) << c;
        b.y |= (x[c + 32] > 0.f ? 1u : 0u) << c;
    }
    return b;
}

// 64 floats of a row to global memory (16-byte aligned)
__device__ __forceinline__ void store_row(float *dst, const float (&x)[64]) {
#pragma unroll
    for (int c = 0; c < 16; ++c)
        reinterpret_cast<float4 *>(dst)[c] = make_float4(x[4 * c], x[4 * c + 1], x[4 * c + 2], x[4 * c + 3]);
}

// The adjoint's buffers (XM_ADJ): activations relu(z_l) into A + l*ldl and
// deltas delta_l into D + l*ldl (row-major [vertex][W]), ReLU masks, s_v.
struct AdjOut {
    const float *dL;
    float *A, *D, *s;
    uint2 *mask;  // [(l * rows + row) * (W/64) + group], rows = tiles * 128
    long long ldl;
    const uint16_t *wt6;  // split transposed weights, last layer first
};

// A CTA's end after a wait ran out: no item's lists may be read any more ...
__device__ __noinline__ void give_up_items(const Item *items, int n_items) {
    if (threadIdx.x == 0)
        for (int b = 0; b < n_items; ++b) atomicOr(&items[b].s.ctr->flags, FLAG_TIMEOUT);
}
// ... and the calls without a status get NaN in every row of the CTA
__device__ __noinline__ void give_up_rows(float *dst, long long n, Counters *ctr) {
    if (threadIdx.x == 0) atomicOr(&ctr->flags, FLAG_TIMEOUT);
    if (threadIdx.x < TM)
        for (long long i = (long long)blockIdx.x * TM + threadIdx.x; i < n; i += (long long)gridDim.x * TM)
            dst[i] = __int_as_float(0x7FC00000);
}

// OWN: some layer of some item has outputs with corrections of their own
// (MlpDev::kbits).  Dense networks run the form without: deciding it per layer
// cost them 5 % (2^20 points at width 256 2.37 -> 2.48 ms: registers).
template <int W, int MODE, bool OWN>
__global__ void __launch_bounds__(64 + 2 * W, ctas_of<W>())
    k_mlp_x6(const Item *__restrict__ items_in, int n_items, const __grid_constant__ Item single,
             const float *__restrict__ pts, long long npts, float *__restrict__ outv, AdjOut adj,
             unsigned long long wait_ns) {
    // point lists and the adjoint: the one descriptor comes with the launch
    const Item *items = MODE == XM_POINTS || MODE == XM_ADJ ? &single : items_in;
    extern __shared__ uint8_t smem_raw[];
    constexpr int G = W / 64;                  // K-blocks per layer = column groups
    constexpr int NST = nst_of<W>();
    constexpr int EPI = 2 * W;                 // epilogue threads
    constexpr uint32_t STAGE_BYTES = W * 128;  // one K-block of one part
    constexpr uint32_t TMEM_COLS = 2 * W;      // 128, 256 or 512
    constexpr uint32_t AH = W, AM = W + W / 2; // TMEM columns of x_h and x_m
    constexpr uint32_t IDESC = idesc_bf16(TM, W);
    SmemX<W> &sm = *reinterpret_cast<SmemX<W> *>(smem_raw + ((1024 - (su32(smem_raw) & 1023)) & 1023));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    volatile int *ctl = &sm.ctl;
    Counters *ctr0 = items[0].s.ctr;  // a timeout is flagged here at once, in every item at the end
    const int n_mid = items[0].m.n_mid;
    const int n_gemm = MODE == XM_ADJ ? 2 * n_mid : n_mid;  // products per tile (adjoint: there and back)

    if (tid >= EPI_T0) load_params<W, OWN>(sm, items[0].m, tid - EPI_T0);
    if (tid == 0) {
        for (int i = 0; i < NST; ++i) {
            mbar_init(&sm.full[i], 1);
            mbar_init(&sm.empty[i], 1);
        }
        mbar_init(&sm.acc_full, 1);
        mbar_init(&sm.a_h, EPI);
        mbar_init(&sm.a_ml, EPI);
        mbar_init(&sm.item_ready, 1);
        mbar_init(&sm.drain, 1);
        sm.cur_w = items[0].m.wx6;
        sm.done = 0;
        sm.ctl = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&sm.tmem_base)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sm.tmem_base;
    volatile int *vdone = &sm.done;

    if (warp == 0) {
        // ---- producer: per tile, n_gemm layers x 3 parts x G K-blocks ----------
        if (lane == 0) {
            uint32_t issued = 0;
            uint32_t pir = 0;
            bool go = true;
            while (go) {
                if (!wait_bar(&sm.item_ready, pir, ctl, CTL_ABORT, ctr0, wait_ns)) break;
                pir ^= 1u;
                if (*vdone) break;
                const uint8_t *wf = reinterpret_cast<const uint8_t *>(*(const uint16_t *volatile *)&sm.cur_w);
                for (int l = 0; l < n_gemm && go; ++l) {
                    const uint8_t *src = MODE == XM_ADJ && l >= n_mid ? reinterpret_cast<const uint8_t *>(adj.wt6) : wf;
                    src += (size_t)(MODE == XM_ADJ && l >= n_mid ? l - n_mid : l) * 3 * G * STAGE_BYTES;
                    for (int s = 0; s < 3 * G; ++s) {  // parts low, middle, high; the last pass finds high in the ring
                        const uint32_t st = issued % NST, par = ((issued / NST) & 1) ^ 1;
                        if (!wait_bar(&sm.empty[st], par, ctl, CTL_ABORT, ctr0, wait_ns)) {
                            go = false;
                            break;
                        }
                        mbar_expect_tx(&sm.full[st], STAGE_BYTES);
                        bulk_g2s(sm.w[st], src + (size_t)s * STAGE_BYTES, STAGE_BYTES, &sm.full[st]);
                        ++issued;
                    }
                }
            }
            // the copies still in flight land before the CTA may exit
            for (uint32_t i = issued < NST ? 0 : issued - NST; i < issued; ++i)
                wait_bar(&sm.full[i % NST], (i / NST) & 1, ctl, 0, ctr0);
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---- MMA issuer ---------------------------------------------------------
        // (lean issue loop: descriptors built once and advanced by fixed steps,
        // a stage that has landed taken without a call; k_mlp_bf16.cu)
        if (lane == 0) {
            uint32_t pa = 0, pf = 0;  // phases: of the operand barriers, of the ring at the layer's first stage
            bool go = true;
            constexpr unsigned long long A_KB = (TM * 128) >> 4, W_ST = STAGE_BYTES >> 4;
            const unsigned long long ald = sdesc(su32(&sm.al[0][0])), wd0 = sdesc(su32(sm.w[0]));
            while (go) {
                for (int l = 0; l < n_gemm && go; ++l) {
                    // x_h is stored and the accumulator has been read
                    if (!mbar_try(&sm.a_h, pa) && !wait_bar(&sm.a_h, pa, ctl, CTL_ABORT, ctr0, wait_ns)) {
                        go = false;
                        break;
                    }
                    if (l == 0 && *vdone) {
                        go = false;
                        break;
                    }
                    tc_fence_after();
#pragma unroll
                    for (int pass = 0; pass < NPASS; ++pass) {
                        if (pass == 1 && go) {  // from here on x_m and x_l are read too
                            if (!mbar_try(&sm.a_ml, pa) && !wait_bar(&sm.a_ml, pa, ctl, CTL_ABORT, ctr0, wait_ns))
                                go = false;
                            tc_fence_after();
                        }
#pragma unroll
                        for (int kb = 0; kb < G; ++kb) {
                            // the layer's stages in order; the last pass takes the high part's again
                            constexpr int S3 = 2 * G;
                            const int s = (pass == 3 ? S3 : pass * G) + kb, st = s % NST;
                            if (pass != 3 && go && !mbar_try(&sm.full[st], pf ^ ((s / NST) & 1)) &&
                                !wait_bar(&sm.full[st], pf ^ ((s / NST) & 1), ctl, CTL_ABORT, ctr0, wait_ns))
                                go = false;
                            if (!go) continue;
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const unsigned long long bd = wd0 + (st * W_ST + 2 * k);
                                const uint32_t acol = (uint32_t)(kb * 32 + k * 8);
                                if (pass == 2) umma(tmem, ald + (kb * A_KB + 2 * k), bd, IDESC, 1u);  // x_l w_h
                                if (pass == 1 || pass == 2)  // x_m w_m, x_m w_h
                                    umma_ta(tmem, tmem + AM + acol, bd, IDESC, 1u);
                                if (pass != 2)  // x_h w_l (the layer's first op), x_h w_m, and last x_h w_h
                                    umma_ta(tmem, tmem + AH + acol, bd, IDESC, (pass | kb | k) != 0);
                            }
                            if (pass != 2) umma_commit(&sm.empty[st]);
                        }
                    }
                    pa ^= 1u;
                    pf ^= (3 * G / NST) & 1;
                    if (go) umma_commit(&sm.acc_full);
                }
            }
            // every MMA issued above has completed before TMEM is released
            umma_commit(&sm.drain);
            wait_bar(&sm.drain, 0, ctl, 0, ctr0);
        }
        __syncwarp();
    } else {
        // ---- epilogue: G threads per row, 64 columns each ------------------------
        const int e = tid - EPI_T0, grp = e >> 7, q = warp & 3;  // a warp reads TMEM lanes 32 (warp % 4) ..
        const int row = 32 * q + lane;
        const uint32_t tlane = tmem + ((uint32_t)(32 * q) << 16);
        const uint32_t tacc = tlane + 64u * grp, th = tlane + AH + 32u * grp, tm = tlane + AM + 32u * grp;
        const uint32_t lrow = su32(&sm.al[grp][0]) + (uint32_t)((row >> 3) * 1024 + (row & 7) * 128);
        const int sw = row & 7;
        const int c0 = 64 * grp;  // this thread's first column
        const unsigned lt = (1u << lane) - 1u;
        int cur = 0;
        const Item *it = &items[0];
        uint32_t pacc = 0;
        // hopping state of the row (group 0's thread)
        uint32_t col = NONE, rank = 0;
        int k = 0;
        bool done = false;
        float hx = 0.f, hy = 0.f;
        unsigned long long evals = 0;
        for (long long tile = blockIdx.x;; tile += gridDim.x) {
            // 1. the rows' work, from item cur: group 0 decides and shares the points
            unsigned long long idx = 0;
            uint32_t vslot = 0;
            bool live = false;
            const GridP &g = it->g;
            const Scratch &s = it->s;
            const int N = g.N;
            if (grp == 0) {
                float px = 0.f, py = 0.f, pz = 0.f;
                if (MODE == XM_HOP) {
                    const uint32_t ncols = (uint32_t)N * (uint32_t)N;
                    const bool need = col == NONE && !done;
                    const unsigned needm = __ballot_sync(FULL, need);
                    if (needm) {
                        const int leader = __ffs(needm) - 1;
                        unsigned long long base = 0;
                        if (lane == leader) base = atomicAdd(&s.ctr->next_col, (unsigned long long)__popc(needm));
                        base = __shfl_sync(FULL, base, leader);
                        if (need) {
                            const unsigned long long c = base + __popc(needm & lt);
                            if (c < ncols) {
                                col = column_of_claim((uint32_t)c, N);
                                k = 0;
                                rank = 0;
                                const int i = (int)(col / (uint32_t)N), j = (int)(col - (uint32_t)i * N);
                                hx = fmaf((float)i + 0.5f, g.h, g.lo[0]);
                                hy = fmaf((float)j + 0.5f, g.h, g.lo[1]);
                            } else {
                                done = true;
                            }
                        }
                    }
                    live = col != NONE;
                    if (live) {
                        px = hx;
                        py = hy;
                        pz = fmaf((float)k + 0.5f, g.h, g.lo[2]);
                    }
                } else {
                    unsigned long long total = (unsigned long long)npts;
                    if (MODE == XM_LATTICE) total = (unsigned long long)(N + 1) * (N + 1) * (N + 1);
                    if (MODE == XM_VERTS || MODE == XM_REFINE)
                        total = (s.ctr->flags & STOP_FLAGS) ? 0ull : (MODE == XM_VERTS ? s.ctr->verts : s.ctr->refine);
                    unsigned long long base = total;
                    if (MODE == XM_POINTS || MODE == XM_ADJ) {  // equal tiles dealt out in turn
                        base = (unsigned long long)tile * TM + 32 * q;
                    } else {
                        if (lane == 0 && !done)
                            base = atomicAdd(MODE == XM_REFINE ? &s.ctr->next_tile2 : &s.ctr->next_tile, 32ull);
                        base = __shfl_sync(FULL, base, 0);
                    }
                    idx = base + lane;
                    live = idx < total;
                    if (base >= total) done = true;
                    if (live) {
                        if (MODE == XM_POINTS || MODE == XM_ADJ) {
                            px = pts[3 * idx];
                            py = pts[3 * idx + 1];
                            pz = pts[3 * idx + 2];
                        } else if (MODE == XM_LATTICE) {
                            const unsigned long long N1 = N + 1;
                            const unsigned long long a = idx % N1, b = (idx / N1) % N1, c = idx / (N1 * N1);
                            px = fmaf((float)a, g.h, g.lo[0]);
                            py = fmaf((float)b, g.h, g.lo[1]);
                            pz = fmaf((float)c, g.h, g.lo[2]);
                        } else {
                            vslot = MODE == XM_REFINE ? s.rlist[idx] : (uint32_t)idx;
                            const unsigned long long key = s.vkey[vslot];
                            const int N1 = N + 1;
                            const uint32_t line = (uint32_t)(key & 0xFFFFFFFFull), c = (uint32_t)(key >> 32);
                            const uint32_t a = line / (uint32_t)N1, b = line - a * (uint32_t)N1;
                            px = fmaf((float)a, g.h, g.lo[0]);
                            py = fmaf((float)b, g.h, g.lo[1]);
                            pz = fmaf((float)c, g.h, g.lo[2]);
                        }
                    }
                }
                sm.pt[row] = make_float4(px, py, pz, live ? 1.f : 0.f);
            }
            const bool any = bar_any(BAR_EPI, EPI, live);
            // the abort decision goes through the barrier so that it is uniform
            const bool abort = bar_any(BAR_EPI, EPI, (*ctl & CTL_ABORT) != 0);
            if (abort || !any) {
                if (MODE == XM_HOP && grp == 0) {
                    for (int o = 16; o > 0; o >>= 1) evals += __shfl_xor_sync(FULL, evals, o);
                    if (lane == 0 && evals) atomicAdd(&s.ctr->hop_evals, evals);
                    evals = 0;
                }
                if (!abort && cur + 1 < n_items) {
                    // item cur has no rows left for this CTA: the next item
                    ++cur;
                    it = &items[cur];
                    col = NONE;
                    done = false;
                    load_params<W, OWN>(sm, it->m, e);
                    bar_sync(BAR_EPI, EPI);
                    continue;
                }
                if (e == 0) {
                    *vdone = 1;
                    __threadfence_block();
                    mbar_arrive(&sm.item_ready);
                }
                mbar_arrive(&sm.a_h);  // the final phase: the MMA sees done
                break;
            }
            if (e == 0) {
                sm.cur_w = it->m.wx6;
                mbar_arrive(&sm.item_ready);
                if (MODE == XM_HOP) atomicAdd(&s.ctr->row_slots, (unsigned long long)TM);
            }
            const MlpDev &m = it->m;
            const float4 pt = sm.pt[row];
            const bool rlive = pt.w != 0.f;
            // adjoint: this thread's piece of row tile * 128 + row of the chunk's arrays
            const long long arows = (npts + TM - 1) / TM * TM, arow_i = tile * TM + row;
            const size_t aoff = MODE == XM_ADJ ? (size_t)arow_i * W + c0 : 0;
            const size_t moff = MODE == XM_ADJ ? (size_t)arow_i * G + grp : 0;
            constexpr bool RELU_CVT = MODE != XM_ADJ;  // x holds z; the adjoint keeps relu(z), which it also stores
            float x[64];
            // 2. layer 0 in FP32 (the FP32 engine's operation order), split -> A operands
            {
                const unsigned long long ppx = pack2(pt.x, pt.x), ppy = pack2(pt.y, pt.y), ppz = pack2(pt.z, pt.z);
#pragma unroll
                for (int p = 0; p < 32; ++p) {
                    const float4 wa = sm.w0b[c0 + 2 * p], wb = sm.w0b[c0 + 2 * p + 1];
                    const unsigned long long z = ffma2(pack2(wa.x, wa.y), ppx,
                                                       ffma2(pack2(wa.z, wa.w), ppy,
                                                             ffma2(pack2(wb.x, wb.y), ppz, pack2(wb.z, wb.w))));
                    x[2 * p] = RELU_CVT ? lo2(z) : fmaxf(lo2(z), 0.f);
                    x[2 * p + 1] = RELU_CVT ? hi2(z) : fmaxf(hi2(z), 0.f);
                }
            }
            __syncwarp();  // tcgen05.st below needs the whole warp converged
            if (MODE == XM_ADJ) {
                if (rlive) store_row(adj.A + aoff, x);
                adj.mask[moff] = relu_bits(x);
            }
            put_h<RELU_CVT>(x, th);
            tc_fence_before();
            mbar_arrive(&sm.a_h);
            put_ml<RELU_CVT>(x, tm, lrow, sw);
            tc_fence_before();
            fence_async_smem();
            mbar_arrive(&sm.a_ml);
            // 3. the products' results, layer by layer -> the next A operands, and at
            //    the end the output dot product (adjoint: grad_x g)
            constexpr float KAPPA = kappa_units(W);
            const unsigned long long KK = pack2(KAPPA, KAPPA);
            float gs[3] = {0.f, 0.f, 0.f};
            for (int l = 0; l < n_gemm; ++l) {
                const bool back = MODE == XM_ADJ && l >= n_mid;
                uint2 mk = make_uint2(0u, 0u);
                if (back) mk = adj.mask[(size_t)(2 * n_mid - 1 - l) * arows * G + moff];
                wait_bar(&sm.acc_full, pacc, ctl, CTL_ABORT, ctr0, wait_ns);
                pacc ^= 1u;
                __syncwarp();  // tcgen05.ld below needs the whole warp converged
                tc_fence_after();
                {
                    uint32_t lo[32], hi[32];
                    tmem_ld32_async(tacc, lo);
                    tmem_ld32_async(tacc + 32, hi);
                    tmem_wait_ld();
#pragma unroll
                    for (int c = 0; c < 32; ++c) {
                        x[c] = __uint_as_float(lo[c]);
                        x[32 + c] = __uint_as_float(hi[c]);
                    }
                }
                const bool own = OWN && (sm.kbits[back ? 1 : 0] >> ((back ? l - n_mid : l) * G + grp)) & 1u;
                if (!back) {
                    const float4 *bl = reinterpret_cast<const float4 *>(sm.bmid + l * W + c0);
                    // z = acc + (b + kappa 2^e(acc)): one rounding at the size of z
                    auto put = [&](int c, const float4 &b, unsigned long long k0, unsigned long long k1) {
                        const unsigned long long z0 =
                            fadd2(pack2(x[4 * c], x[4 * c + 1]),
                                  ffma2(pack2(pow2_of(x[4 * c]), pow2_of(x[4 * c + 1])), k0, pack2(b.x, b.y)));
                        const unsigned long long z1 =
                            fadd2(pack2(x[4 * c + 2], x[4 * c + 3]),
                                  ffma2(pack2(pow2_of(x[4 * c + 2]), pow2_of(x[4 * c + 3])), k1, pack2(b.z, b.w)));
                        x[4 * c] = RELU_CVT ? lo2(z0) : fmaxf(lo2(z0), 0.f);
                        x[4 * c + 1] = RELU_CVT ? hi2(z0) : fmaxf(hi2(z0), 0.f);
                        x[4 * c + 2] = RELU_CVT ? lo2(z1) : fmaxf(lo2(z1), 0.f);
                        x[4 * c + 3] = RELU_CVT ? hi2(z1) : fmaxf(hi2(z1), 0.f);
                    };
                    if (!own) {
#pragma unroll
                        for (int c = 0; c < 16; ++c) put(c, bl[c], KK, KK);
                    } else {
#pragma unroll
                        for (int c = 0; c < 16; ++c) {
                            const float4 k = __ldg(reinterpret_cast<const float4 *>(m.kap + l * W + c0) + c);
                            put(c, bl[c], pack2(k.x, k.y), pack2(k.z, k.w));
                        }
                    }
                    if (MODE == XM_ADJ) {
                        if (rlive) store_row(adj.A + (size_t)(l + 1) * adj.ldl + aoff, x);
                        const uint2 bits = relu_bits(x);
                        if (l + 1 < n_mid) {
                            adj.mask[(size_t)(l + 1) * arows * G + moff] = bits;
                        } else {  // the top: delta_L = w_out [z_L > 0]
#pragma unroll
                            for (int c = 0; c < 64; ++c)
                                x[c] = ((c < 32 ? bits.x : bits.y) >> (c & 31)) & 1u ? sm.wout[c0 + c] : 0.f;
                            if (rlive) store_row(adj.D + (size_t)n_mid * adj.ldl + aoff, x);
                        }
                    }
                } else {  // delta_{l'} = (W^T delta) [z_{l'} > 0], l' = 2 n_mid - 1 - l
                    if (!own) {
#pragma unroll
                        for (int c = 0; c < 64; ++c) x[c] = fmaf(pow2_of(x[c]), KAPPA, x[c]);
                    } else {
#pragma unroll
                        for (int c = 0; c < 16; ++c) {
                            const float4 k = __ldg(reinterpret_cast<const float4 *>(m.kap + l * W + c0) + c);
                            x[4 * c] = fmaf(pow2_of(x[4 * c]), k.x, x[4 * c]);
                            x[4 * c + 1] = fmaf(pow2_of(x[4 * c + 1]), k.y, x[4 * c + 1]);
                            x[4 * c + 2] = fmaf(pow2_of(x[4 * c + 2]), k.z, x[4 * c + 2]);
                            x[4 * c + 3] = fmaf(pow2_of(x[4 * c + 3]), k.w, x[4 * c + 3]);
                        }
                    }
#pragma unroll
                    for (int c = 0; c < 64; ++c) x[c] = ((c < 32 ? mk.x : mk.y) >> (c & 31)) & 1u ? x[c] : 0.f;
                    if (rlive) store_row(adj.D + (size_t)(2 * n_mid - 1 - l) * adj.ldl + aoff, x);
                }
                if (l + 1 < n_gemm) {
                    put_h<RELU_CVT>(x, th);
                    tc_fence_before();
                    mbar_arrive(&sm.a_h);
                    put_ml<RELU_CVT>(x, tm, lrow, sw);
                    tc_fence_before();
                    fence_async_smem();
                    mbar_arrive(&sm.a_ml);
                } else {
                    tc_fence_before();
                    if (MODE == XM_ADJ) {
#pragma unroll
                        for (int p = 0; p < 32; ++p) {
                            const float4 wa = sm.w0b[c0 + 2 * p], wb = sm.w0b[c0 + 2 * p + 1];
                            gs[0] = fmaf(wa.y, x[2 * p + 1], fmaf(wa.x, x[2 * p], gs[0]));
                            gs[1] = fmaf(wa.w, x[2 * p + 1], fmaf(wa.z, x[2 * p], gs[1]));
                            gs[2] = fmaf(wb.y, x[2 * p + 1], fmaf(wb.x, x[2 * p], gs[2]));
                        }
                    } else {
                        // eight sums of every eighth column: eight fused multiply-adds in a
                        // row instead of 64.  (With four, 9 of 8,640 vertices of the
                        // paper-form network at N = 77 lie beyond 1e-4 h of the FP64 mesh
                        // instead of 8; an exact evaluator at the FP32 lattice has 9.)
                        const float4 *wp = reinterpret_cast<const float4 *>(sm.wout + c0);
                        float d[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
                        for (int c = 0; c < 16; ++c) {
                            const float4 w = wp[c];
                            d[4 * (c & 1)] = fmaf(w.x, relu_nan(x[4 * c]), d[4 * (c & 1)]);
                            d[4 * (c & 1) + 1] = fmaf(w.y, relu_nan(x[4 * c + 1]), d[4 * (c & 1) + 1]);
                            d[4 * (c & 1) + 2] = fmaf(w.z, relu_nan(x[4 * c + 2]), d[4 * (c & 1) + 2]);
                            d[4 * (c & 1) + 3] = fmaf(w.w, relu_nan(x[4 * c + 3]), d[4 * (c & 1) + 3]);
                        }
                        gs[0] = ((d[0] + d[1]) + (d[2] + d[3])) + ((d[4] + d[5]) + (d[6] + d[7]));
                    }
                }
            }
            // 4. the groups' sums in order, then f and the hop step or the store
            for (int a = 0; a < (MODE == XM_ADJ ? 3 : 1); ++a) sm.red[a][grp][row] = gs[a];
            bar_sync(BAR_EPI, EPI);
            if (grp != 0) continue;
            float tot[3] = {0.f, 0.f, 0.f};
            for (int a = 0; a < (MODE == XM_ADJ ? 3 : 1); ++a) {
                tot[a] = sm.red[a][0][row];
                for (int u = 1; u < G; ++u) tot[a] += sm.red[a][u][row];
            }
            if (MODE == XM_ADJ) {
                if (rlive) {
                    // s_v = -(dL/dv . grad_x f) / |grad_x f|^2
                    const float r = sqrtf(pt.x * pt.x + pt.y * pt.y + pt.z * pt.z);
                    const float ir = r > 0.f ? m.radial / r : 0.f, ibl = 1.f / m.beta * m.inv_lam;
                    const float fx = (pt.x * ir + m.alpha * tot[0]) * ibl;
                    const float fy = (pt.y * ir + m.alpha * tot[1]) * ibl;
                    const float fz = (pt.z * ir + m.alpha * tot[2]) * ibl;
                    const float n2 = fx * fx + fy * fy + fz * fz;
                    const float dot = adj.dL[3 * arow_i] * fx + adj.dL[3 * arow_i + 1] * fy + adj.dL[3 * arow_i + 2] * fz;
                    adj.s[arow_i] = n2 > 0.f ? -dot / n2 : 0.f;
                }
                continue;
            }
            const float f = outer_f(m, pt.x, pt.y, pt.z, tot[0] + m.bout);
            if (MODE == XM_HOP) {
                bool mark = false, empty = false;
                int step = 1;
                if (live) {
                    ++evals;
                    float d = fabsf(f) - g.eps;
                    if (!isfinite(f)) {
                        atomicOr(&s.ctr->flags, FLAG_NONFINITE);
                        d = 0.f;
                    }
                    if (d <= g.tau) {
                        mark = true;
                        empty = cell_is_empty(g, d, pt.x, pt.y, pt.z);
                    } else {
                        const float stp = floorf(d * g.inv_h);
                        step = stp < 1.f ? 1 : (stp > (float)N ? N : (int)stp);
                    }
                }
                const unsigned mm = __ballot_sync(FULL, mark);
                if (mm) {
                    const int leader = __ffs(mm) - 1;
                    unsigned long long base = 0;
                    if (lane == leader) base = atomicAdd(&s.ctr->marks, (unsigned long long)__popc(mm));
                    base = __shfl_sync(FULL, base, leader);
                    if (mark) {
                        const unsigned long long mi = base + __popc(mm & lt);
                        if (mi < (unsigned long long)s.cap_marks)
                            s.marks_raw[mi] = pack_mark(col, (uint32_t)k, rank, empty);
                        else
                            atomicOr(&s.ctr->flags, FLAG_MARK_OVERFLOW);
                    }
                }
                if (live) {
                    if (mark) {
                        ++rank;
                        ++k;
                    } else {
                        k += step;
                    }
                    if (k >= N) {
                        s.colcount[col] = rank;
                        col = NONE;
                    }
                }
            } else if (live) {
                if (MODE == XM_POINTS) {
                    outv[idx] = f;
                } else {
                    if (!isfinite(f)) atomicOr(&s.ctr->flags, FLAG_NONFINITE);
                    if (MODE == XM_LATTICE) s.lat[idx] = f;
                    else s.vval[vslot] = f;
                }
            }
        }
    }
    // ---- tear-down ---------------------------------------------------------
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (sm.ctl & CTL_ABORT) {
        if (MODE == XM_POINTS) give_up_rows(outv, npts, ctr0);
        else if (MODE == XM_ADJ) give_up_rows(adj.s, npts, ctr0);  // s_v multiplies every term of the gradient's sums
        else give_up_items(items_in, n_items);
    }
    if (threadIdx.x >> 5 == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
}

template <int W, int MODE, bool OWN>
void launch_x6_as(const Item *items, int n_items, const Item &single, const float *p, long long n, float *out,
               const AdjOut &adj, int nsm, cudaStream_t st) {
    const size_t smem = sizeof(SmemX<W>) + 1024;
    cudaFuncSetAttribute(k_mlp_x6<W, MODE, OWN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int grid = nsm * ctas_of<W>();
    if (MODE == XM_POINTS || MODE == XM_ADJ) {
        const long long tiles = (n + TM - 1) / TM;
        if (grid > tiles) grid = (int)(tiles < 1 ? 1 : tiles);
    }
    k_mlp_x6<W, MODE, OWN><<<grid, EPI_T0 + 2 * W, smem, st>>>(items, n_items, single, p, n, out, adj, wait_limit_ns());
}

template <int W, int MODE>
void launch_x6(bool own, const Item *items, int n_items, const Item &single, const float *p, long long n, float *out,
               const AdjOut &adj, int nsm, cudaStream_t st) {
    if (own) launch_x6_as<W, MODE, true>(items, n_items, single, p, n, out, adj, nsm, st);
    else launch_x6_as<W, MODE, false>(items, n_items, single, p, n, out, adj, nsm, st);
}

}  // namespace

#define GH_X6_W(W, ...)                                       \
    switch (W) {                                              \
    case 64: { constexpr int WW = 64; __VA_ARGS__; } break;   \
    case 128: { constexpr int WW = 128; __VA_ARGS__; } break; \
    default: { constexpr int WW = 256; __VA_ARGS__; } break;  \
    }

int x6_max_mid() { return MAXMID; }

void launch_hop_mlp_x6(const Item *items, int n_items, int width, bool own, int nsm, cudaStream_t st) {
    GH_X6_W(width, (launch_x6<WW, XM_HOP>(own, items, n_items, Item{}, nullptr, 0, nullptr, AdjOut{}, nsm, st)))
}

void launch_eval_vertices_mlp_x6(const Item *items, int n_items, int width, bool own, int nsm, bool refine_list,
                                 cudaStream_t st) {
    if (refine_list) {
        GH_X6_W(width, (launch_x6<WW, XM_REFINE>(own, items, n_items, Item{}, nullptr, 0, nullptr, AdjOut{}, nsm, st)))
    } else {
        GH_X6_W(width, (launch_x6<WW, XM_VERTS>(own, items, n_items, Item{}, nullptr, 0, nullptr, AdjOut{}, nsm, st)))
    }
}

void launch_lattice_mlp_x6(const Item *items, int width, bool own, int nsm, cudaStream_t st) {
    GH_X6_W(width, (launch_x6<WW, XM_LATTICE>(own, items, 1, Item{}, nullptr, 0, nullptr, AdjOut{}, nsm, st)))
}

// A network's descriptor for the kernels that take points instead of an item
// (its counters only carry the error flag of a timeout).
static Item points_item(const MlpDev &m) {
    Item h{};
    h.m = m;
    h.s.ctr = m.err;
    h.kind = 1;
    return h;
}

void launch_eval_points_mlp_x6(const MlpDev &m, const float *p, long long n, float *out, int nsm, cudaStream_t st) {
    const Item it = points_item(m);
    GH_X6_W(m.width, (launch_x6<WW, XM_POINTS>(m.own[0] != 0, nullptr, 1, it, p, n, out, AdjOut{}, nsm, st)))
}

void launch_adj_mlp_x6(const MlpDev &m, const float *P, const float *dL, long long V, float *A, float *D, float *s,
                       uint32_t *mask, long long ldl, int nsm, cudaStream_t st) {
    const Item it = points_item(m);
    const AdjOut a{dL, A, D, s, reinterpret_cast<uint2 *>(mask), ldl, m.wx6t};
    GH_X6_W(m.width, (launch_x6<WW, XM_ADJ>((m.own[0] | m.own[1]) != 0, nullptr, 1, it, P, V, nullptr, a, nsm, st)))
}

}  // namespace gh
