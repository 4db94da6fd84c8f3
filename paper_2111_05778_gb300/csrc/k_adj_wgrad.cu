// Weight gradients of the adjoint's hidden layers on the tensor cores:
//   dL/dW_l[o][i] = sum_v s_v delta_l[v][o] relu(z_{l-1})[v][i],  dL/db_l[o] = sum_v s_v delta_l[v][o]
// for all layers in one launch, as products with K = vertices of split-BF16
// operands (k_mlp_x6.cu: x = x_h + x_m + x_l exactly, six part products).
//
// What bounds it: per 16 vertices and 128 x W outputs six products (N = W, 128
// cycles each at width 256) against 24 KB of FP32 operands read and split, so
// the tensor pipe and the splitting threads are about even (1,536 and 1,350
// cycles per 32 vertices); 1.1 GB of activations and deltas are read at 111 k
// vertices, 0.2 ms of HBM time.
//
// A CTA owns one 128 x W block of one layer's gradient and a range of the
// vertices.  16 warps read 32 vertices' deltas and activations (consecutive
// lanes on consecutive units, so that the loads are coalesced and each thread
// packs eight vertices of one unit into a 16-byte chunk of the K-major
// operand), the next 32 being fetched while these are split; one thread issues
// the products.  The large products (h h) and the five small ones have an
// accumulator each, so that only the former's roundings count, and every 512
// vertices both are added into the CTA's FP32 partial in global memory (which
// stays in L2): the tensor core's accumulator is truncated toward zero, and
// its shortfall grows with the number of updates.  The partials are summed
// over the ranges in a fixed order.
#include <stdint.h>

#include "gh_internal.cuh"
#include "tc_ptx.cuh"

namespace gh {

namespace {

using namespace tc;

constexpr int KV = 32;       // vertices per stage
constexpr int FLUSH = 16;    // stages between additions into the partial
constexpr int NLD = 512;     // loading (and flushing) threads
constexpr int BMR = 128;     // gradient rows (outputs o) per CTA

template <int W>
constexpr int nst_of() {
    return W == 256 ? 3 : 4;
}

template <int W>
struct SmemG {
    static constexpr int NST = nst_of<W>();
    uint8_t a[NST][3][BMR * 2 * KV];  // parts low, middle, high of s_v delta: rows o, 32 vertices (64-byte swizzle)
    uint8_t b[NST][3][W * 2 * KV];    // parts of the activations: rows i
    float bsum[4][BMR];               // bias gradients of the four vertex groups
    unsigned long long full[NST], empty[NST], acc_full, acc_free, drain;
    uint32_t tmem_base;
    int ctl;
};

// eight FP32 values -> three 16-byte chunks (x = h + m + l, every difference exact)
__device__ __forceinline__ void put8(const float (&x)[8], uint32_t pl, uint32_t pm, uint32_t ph) {
    uint32_t h[4], m[4], l[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const float x0 = x[2 * p], x1 = x[2 * p + 1];
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(h[p]) : "f"(x1), "f"(x0));
        const float r0 = x0 - __uint_as_float(h[p] << 16), r1 = x1 - __uint_as_float(h[p] & 0xFFFF0000u);
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(m[p]) : "f"(r1), "f"(r0));
        const float s0 = r0 - __uint_as_float(m[p] << 16), s1 = r1 - __uint_as_float(m[p] & 0xFFFF0000u);
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(l[p]) : "f"(s1), "f"(s0));
    }
    sts128(pl, l[0], l[1], l[2], l[3]);
    sts128(pm, m[0], m[1], m[2], m[3]);
    sts128(ph, h[0], h[1], h[2], h[3]);
}

// x[q] = p[(v0 + q) ld], zero beyond V
__device__ __forceinline__ void get8(float (&x)[8], const float *__restrict__ p, long long v0, long long V, int ld) {
    if (v0 + 8 <= V) {
#pragma unroll
        for (int q = 0; q < 8; ++q) x[q] = __ldg(p + (v0 + q) * ld);
    } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) x[q] = v0 + q < V ? __ldg(p + (v0 + q) * ld) : 0.f;
    }
}

// part: [unit][BMR][W] partial sums, bpart: [unit][BMR], unit = ((l - 1) H + h) S + z
// with H = row blocks of a layer, S = vertex ranges; rows_per: vertices per range.
template <int W>
__global__ void __launch_bounds__(NLD + 32, 1)
    k_adj_wgrad(const float *__restrict__ A, const float *__restrict__ D, const float *__restrict__ s, long long V,
                long long ldl, int S, long long rows_per, float *__restrict__ part, float *__restrict__ bpart,
                Counters *ctr, unsigned long long wait_ns) {
    extern __shared__ uint8_t smem_raw[];
    constexpr int NST = nst_of<W>();
    constexpr int H = W > BMR ? W / BMR : 1;
    constexpr int ROWS = W < BMR ? W : BMR;         // gradient rows of a block
    constexpr uint32_t TMEM_COLS = 2 * W;           // main and small accumulators
    constexpr uint32_t IDESC = idesc_bf16(BMR, W);
    constexpr int NB = W * 4 / NLD > 0 ? W * 4 / NLD : 1;  // activation chunks per thread and stage
    SmemG<W> &sm = *reinterpret_cast<SmemG<W> *>(smem_raw + ((1024 - (su32(smem_raw) & 1023)) & 1023));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    volatile int *ctl = &sm.ctl;
    const int unit = blockIdx.x, lh = unit / S, z = unit - lh * S, l = lh / H + 1, h = lh % H;
    const long long vb = (long long)z * rows_per, ve = vb + rows_per < V ? vb + rows_per : V;
    const int nst = ve > vb ? (int)((ve - vb + KV - 1) / KV) : 0;

    if (tid == 0) {
        for (int i = 0; i < NST; ++i) {
            mbar_init(&sm.full[i], NLD);
            mbar_init(&sm.empty[i], 1);
        }
        mbar_init(&sm.acc_full, 1);
        mbar_init(&sm.acc_free, NLD);
        mbar_init(&sm.drain, 1);
        sm.ctl = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (ROWS < BMR) {  // rows without a unit: their products are discarded, zero keeps them finite
        uint32_t *p = reinterpret_cast<uint32_t *>(&sm.a[0][0][0]);
        for (int i = tid; i < (int)(sizeof(sm.a) / 4); i += blockDim.x) p[i] = 0u;
        fence_async_smem();
    }
    if (warp == NLD / 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&sm.tmem_base)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sm.tmem_base;

    if (warp == NLD / 32) {
        // ---- MMA issuer ---------------------------------------------------------
        if (lane == 0) {
            const unsigned long long ad0 = sdesc64(su32(&sm.a[0][0][0])), bd0 = sdesc64(su32(&sm.b[0][0][0]));
            constexpr unsigned long long A_P = (BMR * 2 * KV) >> 4, B_P = (W * 2 * KV) >> 4;
            bool go = true;
            uint32_t pfree = 1u;  // the accumulators start free
            for (int c = 0; c < nst && go; ++c) {
                const int st = c % NST;
                const bool first = c % FLUSH == 0;
                if (first) {
                    if (!wait_bar(&sm.acc_free, pfree, ctl, CTL_ABORT, ctr, wait_ns)) break;
                    pfree ^= 1u;
                }
                if (!mbar_try(&sm.full[st], (uint32_t)(c / NST) & 1u) &&
                    !wait_bar(&sm.full[st], (uint32_t)(c / NST) & 1u, ctl, CTL_ABORT, ctr, wait_ns)) {
                    go = false;
                    break;
                }
                tc_fence_after();
                const unsigned long long a = ad0 + (unsigned long long)st * 3 * A_P, b = bd0 + (unsigned long long)st * 3 * B_P;
#pragma unroll
                for (int k = 0; k < KV / 16; ++k) {
                    const unsigned long long al = a + 2 * k, am = al + A_P, ah = am + A_P;
                    const unsigned long long bl = b + 2 * k, bm = bl + B_P, bh = bm + B_P;
                    const uint32_t acc = first && k == 0 ? 0u : 1u;
                    umma(tmem + W, ah, bl, IDESC, acc);
                    umma(tmem + W, al, bh, IDESC, 1u);
                    umma(tmem + W, am, bm, IDESC, 1u);
                    umma(tmem + W, ah, bm, IDESC, 1u);
                    umma(tmem + W, am, bh, IDESC, 1u);
                    umma(tmem, ah, bh, IDESC, acc);
                }
                umma_commit(&sm.empty[st]);
                if (c % FLUSH == FLUSH - 1 || c == nst - 1) umma_commit(&sm.acc_full);
            }
            // every MMA issued above has completed before TMEM is released
            umma_commit(&sm.drain);
            wait_bar(&sm.drain, 0, ctl, 0, ctr);
        }
        __syncwarp();
    } else {
        // ---- loading and splitting, and every FLUSH stages the addition ----------
        const int o = tid & (BMR - 1), vg = tid >> 7;  // this thread's delta chunk: row o, vertices 8 vg ..
        const bool has_a = o < ROWS;
        const float *dp = D + (size_t)l * ldl + h * BMR + o;
        const float *ap = A + (size_t)(l - 1) * ldl;
        const uint32_t arow = (uint32_t)((o >> 3) * 512 + (o & 7) * 64 + ((vg ^ ((o >> 1) & 3)) << 4));
        int bi[NB], bg[NB];
        uint32_t brow[NB];
        bool has_b = true;
#pragma unroll
        for (int n = 0; n < NB; ++n) {
            const int u = tid + n * NLD;
            bi[n] = u & (W - 1);
            bg[n] = u / W;
            brow[n] = (uint32_t)((bi[n] >> 3) * 512 + (bi[n] & 7) * 64 + ((bg[n] ^ ((bi[n] >> 1) & 3)) << 4));
            if (bg[n] >= 4) has_b = false;  // width 64: half of the threads
        }
        const int q = warp & 3, cg = warp >> 2, row = 32 * q + lane;  // this thread's piece of the accumulators
        constexpr int CW = W / 4;                                      // columns of it
        float *mypart = part + ((size_t)unit * BMR + row) * W + cg * CW;
        float bs = 0.f, bs_run = 0.f;  // bias gradient: per FLUSH stages, and their sum
        float xa[8], sv[8], xb[NB][8];
        auto fetch = [&](int c) {
            const long long v0 = vb + (long long)c * KV;
            if (has_a) {
                get8(xa, dp, v0 + 8 * vg, ve, W);
                get8(sv, s, v0 + 8 * vg, ve, 1);
            }
            if (has_b) {
#pragma unroll
                for (int n = 0; n < NB; ++n) get8(xb[n], ap + bi[n], v0 + 8 * bg[n], ve, W);
            }
        };
        uint32_t pacc = 0u;
        bool wrote = false;
        if (nst > 0) fetch(0);
        for (int c = 0; c < nst; ++c) {
            const int st = c % NST;
            wait_bar(&sm.empty[st], ((uint32_t)(c / NST) & 1u) ^ 1u, ctl, CTL_ABORT, ctr, wait_ns);
            const uint32_t ab = su32(&sm.a[st][0][0]) + arow;
            if (has_a) {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    xa[k] *= sv[k];
                    bs += xa[k];
                }
                put8(xa, ab, ab + BMR * 2 * KV, ab + 2 * BMR * 2 * KV);
            }
            if (has_b) {
#pragma unroll
                for (int n = 0; n < NB; ++n) {
                    const uint32_t bb = su32(&sm.b[st][0][0]) + brow[n];
                    put8(xb[n], bb, bb + W * 2 * KV, bb + 2 * W * 2 * KV);
                }
            }
            fence_async_smem();
            mbar_arrive(&sm.full[st]);
            if (c + 1 < nst) fetch(c + 1);
            if (c % FLUSH == FLUSH - 1 || c == nst - 1) {
                bs_run += bs;
                bs = 0.f;
                wait_bar(&sm.acc_full, pacc, ctl, CTL_ABORT, ctr, wait_ns);
                pacc ^= 1u;
                __syncwarp();  // tcgen05.ld below needs the whole warp converged
                tc_fence_after();
#pragma unroll 1
                for (int j = 0; j < CW; j += 16) {
                    uint32_t u[16], w[16];
                    tmem_ld16_async(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(cg * CW + j), u);
                    tmem_ld16_async(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(W + cg * CW + j), w);
                    tmem_wait_ld();
                    if (row < ROWS) {
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            float4 *p = reinterpret_cast<float4 *>(mypart + j) + k;
                            float4 a = wrote ? *p : make_float4(0.f, 0.f, 0.f, 0.f);
                            a.x += __uint_as_float(u[4 * k]) + __uint_as_float(w[4 * k]);
                            a.y += __uint_as_float(u[4 * k + 1]) + __uint_as_float(w[4 * k + 1]);
                            a.z += __uint_as_float(u[4 * k + 2]) + __uint_as_float(w[4 * k + 2]);
                            a.w += __uint_as_float(u[4 * k + 3]) + __uint_as_float(w[4 * k + 3]);
                            *p = a;
                        }
                    }
                }
                wrote = true;
                tc_fence_before();
                mbar_arrive(&sm.acc_free);
            }
        }
        if (nst == 0 && row < ROWS)  // a range without vertices
            for (int j = 0; j < CW; ++j) mypart[j] = 0.f;
        sm.bsum[vg][o] = bs_run;
    }
    // ---- tear-down ---------------------------------------------------------
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (*ctl & CTL_ABORT) {  // a wait ran out: no sum of this CTA is one, which NaN says
        const float nan = __int_as_float(0x7FC00000);
        for (int i = tid; i < ROWS * W; i += blockDim.x) part[(size_t)unit * BMR * W + i] = nan;
        if (tid < ROWS) bpart[(size_t)unit * BMR + tid] = nan;
    } else if (tid < ROWS) {
        bpart[(size_t)unit * BMR + tid] = (sm.bsum[0][tid] + sm.bsum[1][tid]) + (sm.bsum[2][tid] + sm.bsum[3][tid]);
    }
    if (warp == NLD / 32)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
}

// dst(W_l)[o][i], dst(b_l)[o] (+)= c * sum over the ranges in order; dst packs { W_l b_l } per layer
template <int W>
__global__ void __launch_bounds__(256) k_adj_wreduce(const float *__restrict__ part, const float *__restrict__ bpart,
                                                     int L, int S, float c, float *__restrict__ dst, int accumulate) {
    constexpr int H = W > BMR ? W / BMR : 1, ROWS = W < BMR ? W : BMR;
    constexpr int PER = W * W + W;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < (long long)L * PER;
         e += (long long)gridDim.x * blockDim.x) {
        const int l = (int)(e / PER), r = (int)(e - (long long)l * PER);
        const bool bias = r >= W * W;
        const int o = bias ? r - W * W : r / W, i = r - o * W;
        const int unit0 = (l * H + o / ROWS) * S, oo = o % ROWS;
        float acc = 0.f;
        if (bias)
            for (int z = 0; z < S; ++z) acc += bpart[(size_t)(unit0 + z) * BMR + oo];
        else
            for (int z = 0; z < S; ++z) acc += part[((size_t)(unit0 + z) * BMR + oo) * W + i];
        dst[e] = accumulate ? __fadd_rn(dst[e], __fmul_rn(c, acc)) : __fmul_rn(c, acc);
    }
}

// Vertex ranges per 128-row block: one CTA per SM over all blocks, none below
// two additions' worth of vertices.
int ranges(int W, int L, long long V, int nsm) {
    const int blocks = L * (W > BMR ? W / BMR : 1);
    long long S = nsm / blocks;
    const long long most = (V + 2 * FLUSH * KV - 1) / (2 * FLUSH * KV);
    if (S > most) S = most;
    return S < 1 ? 1 : (int)S;
}

template <int W>
void wgrad(int L, const float *A, const float *D, const float *s, long long V, long long ldl, float *part, float c,
           float *dst, bool accumulate, Counters *ctr, int nsm, cudaStream_t st) {
    constexpr int H = W > BMR ? W / BMR : 1;
    const int S = ranges(W, L, V, nsm), units = L * H * S;
    const long long rows = ((V + S - 1) / S + KV - 1) / KV * KV;
    const size_t smem = sizeof(SmemG<W>) + 1024;
    cudaFuncSetAttribute(k_adj_wgrad<W>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    float *bpart = part + (size_t)units * BMR * W;
    k_adj_wgrad<W><<<units, NLD + 32, smem, st>>>(A, D, s, V, ldl, S, rows, part, bpart, ctr, wait_limit_ns());
    k_adj_wreduce<W><<<512, 256, 0, st>>>(part, bpart, L, S, c, dst, accumulate ? 1 : 0);
}

}  // namespace

size_t adj_wgrad_floats(int W, int n_mid, int nsm) {
    const int blocks = n_mid * (W > BMR ? W / BMR : 1), units = blocks > nsm ? blocks : nsm;
    return (size_t)units * BMR * (W + 1);
}

void launch_adj_wgrad(const MlpDev &m, const float *A, const float *D, const float *s, long long V, long long ldl,
                      float *part, float c, float *dst, bool accumulate, int nsm, cudaStream_t st) {
    Counters *const ctr = m.err;
    switch (m.width) {
    case 64: wgrad<64>(m.n_mid, A, D, s, V, ldl, part, c, dst, accumulate, ctr, nsm, st); break;
    case 128: wgrad<128>(m.n_mid, A, D, s, V, ldl, part, c, dst, accumulate, ctr, nsm, st); break;
    default: wgrad<256>(m.n_mid, A, D, s, V, ldl, part, c, dst, accumulate, ctr, nsm, st); break;
    }
}

}  // namespace gh
