// Derived layouts of a neural SDB's weights, built on the device from the
// packed parameter block W0[W][3] b0[W] { W_l[W][W] b_l[W] } x n_mid w_out[W]
// b_out, so that creating an SDB costs one upload and one launch.
// Networks of more than 8 hidden layers run on the FFMA engine and get wt and
// wtb (wt != NULL), the others the rest:
//   wt  (FFMA engine): per layer [input i][output o], the outputs
//       of a row permuted so that position q*64 + og*4 + e holds output
//       og + 16(4q + e);
//   wtb (adjoint delta chain): per layer [output o][input i], the inputs
//       permuted the same way;
//   wbf (tensor-core engine): per layer, K-blocks of 64 inputs x W outputs in
//       the 128-byte swizzled K-major layout the MMA reads from shared memory
//       (row n, 16-byte chunk c of inputs [8c, 8c+8) at
//       (n/8)*1024 + (n%8)*128 + ((c ^ n%8) * 16)), BF16 rounded to nearest
//       even; at width 256 K-blocks of 32 inputs with the 64-byte swizzle
//       ((n/8)*512 + (n%8)*64 + ((c ^ (n/2)%4) * 16));
//   wx6 (split-BF16 engine): per layer three BF16 parts of every weight,
//       w = w_h + w_m + w_l exactly (w_h = bf16(w), w_m = bf16(w - w_h),
//       w_l = bf16(w - w_h - w_m)), stored part by part (low, middle, high),
//       each part in K-blocks of 64 inputs with the 128-byte swizzle;
//   wx6t the same of the transposed weights (rows = inputs of the layer, K =
//       its outputs), layer n_mid first (the adjoint walks down);
//   bm  hidden biases, n_mid x [W];
//   kap, kbits  (8 layers of W/64 groups at most fit a word) what the split-BF16 engine's epilogue adds back (gh_internal.cuh:
//       kappa_row, from the number of nonzero weights of each output).
#include "gh_internal.cuh"

namespace gh {

namespace {

__device__ __forceinline__ int perm_pos(int o) {
    const int og = o & 15, m = o >> 4;
    return (m >> 2) * 64 + og * 4 + (m & 3);
}

// BF16 of an FP32 value, rounded to nearest even (finite values)
__device__ __forceinline__ uint16_t bf16_rne(float v) {
    const uint32_t u = __float_as_uint(v);
    return (uint16_t)((u + 0x7FFFu + ((u >> 16) & 1u)) >> 16);
}
__device__ __forceinline__ float bf16_val(uint16_t b) { return __uint_as_float((uint32_t)b << 16); }

__global__ void __launch_bounds__(256) k_prep_mlp(const float *__restrict__ params, int W, int n_mid,
                                                  float *__restrict__ wt, float *__restrict__ wtb,
                                                  uint16_t *__restrict__ wbf, uint16_t *__restrict__ wx6,
                                                  uint16_t *__restrict__ wx6t, float *__restrict__ bm,
                                                  float *__restrict__ kap, uint32_t *__restrict__ kbits) {
    const long long WW = (long long)W * W, total = (long long)n_mid * WW;
    const long long mid0 = 4LL * W;  // W0 and b0 come first
    const int KB = W / 64;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int l = (int)(e / WW);
        const long long r = e - l * WW;
        const int o = (int)(r / W), i = (int)(r - (long long)o * W);  // W_l[o][i]
        const float v = params[mid0 + l * (WW + W) + r];
        if (wt) {  // a network for the FFMA engine
            wt[l * WW + (long long)i * W + perm_pos(o)] = v;
            wtb[l * WW + (long long)o * W + perm_pos(i)] = v;
            continue;
        }
        const int kb = i >> 6, kk = i & 63;
        const int byte = (o >> 3) * 1024 + (o & 7) * 128 + (((kk >> 3) ^ (o & 7)) << 4) + (kk & 7) * 2;
        const uint16_t hi = bf16_rne(v);
        if (W == 256) {
            const int kc = (i >> 3) & 3;
            wbf[((long long)l * 2 * KB + (i >> 5)) * W * 32 +
                ((o >> 3) * 512 + (o & 7) * 64 + ((kc ^ ((o >> 1) & 3)) << 4) + (i & 7) * 2) / 2] = hi;
        } else {
            wbf[((long long)l * KB + kb) * W * 64 + byte / 2] = hi;
        }
        const float rem = v - bf16_val(hi);  // exact
        const uint16_t mid = bf16_rne(rem);
        const uint16_t low = bf16_rne(rem - bf16_val(mid));
        const uint16_t parts[3] = {low, mid, hi};
        const int kt = o >> 6, ko = o & 63;
        const int bytet = (i >> 3) * 1024 + (i & 7) * 128 + (((ko >> 3) ^ (i & 7)) << 4) + (ko & 7) * 2;
        for (int p = 0; p < 3; ++p) {
            wx6[(((long long)l * 3 + p) * KB + kb) * W * 64 + byte / 2] = parts[p];
            wx6t[(((long long)(n_mid - 1 - l) * 3 + p) * KB + kt) * W * 64 + bytet / 2] = parts[p];
        }
    }
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < (long long)n_mid * W;
         e += (long long)gridDim.x * blockDim.x) {
        const int l = (int)(e / W), o = (int)(e - (long long)l * W);
        bm[e] = params[mid0 + l * (WW + W) + WW + o];
    }
    if (wt) return;
    // one warp per output: d = 0 forward, 1 transposed (its layers last first)
    const int lane = threadIdx.x & 31, nwarp = (int)(gridDim.x * blockDim.x) >> 5;
    for (int e = (int)(blockIdx.x * blockDim.x + threadIdx.x) >> 5; e < 2 * n_mid * W; e += nwarp) {
        const int d = e / (n_mid * W), r = e - d * n_mid * W, l = r / W, o = r - l * W;
        const float *w = params + mid0 + (d ? n_mid - 1 - l : l) * (WW + W);
        int n = 0;
        bool pow2 = true;
        for (int i = lane; i < W; i += 32) {
            const float v = d ? w[(long long)i * W + o] : w[(long long)o * W + i];
            n += v != 0.f;
            pow2 = pow2 && (__float_as_uint(v) & 0x7FFFFFu) == 0u;
        }
        n = __reduce_add_sync(0xFFFFFFFFu, n);
        pow2 = __all_sync(0xFFFFFFFFu, pow2);
        if (lane == 0) {
            const float k = kappa_row(W, n, pow2);
            kap[e] = k;
            if (k != kappa_units(W)) atomicOr(kbits + d, 1u << (l * KB + (o >> 6)));
        }
    }
}

}  // namespace

void launch_prep_mlp(const float *params, int W, int n_mid, float *wt, float *wtb, uint16_t *wbf, uint16_t *wx6,
                     uint16_t *wx6t, float *bm, float *kap, uint32_t *kbits, cudaStream_t st) {
    k_prep_mlp<<<1024, 256, 0, st>>>(params, W, n_mid, wt, wtb, wbf, wx6, wx6t, bm, kap, kbits);
}

}  // namespace gh
