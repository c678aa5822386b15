// HBM-bound kernels of the AlexNet training step: preprocessing gather, LRN,
// max-pool, split-K reductions with fused bias/ReLU/dropout, softmax
// cross-entropy, bias gradients, momentum update, replica average, layout
// permutations.  Activations are bf16 in a zero-padded flat NHWC grid
// [B][Hp][Wp][C] whose valid region is the top-left H x W of every image; pad
// positions always hold zero.  All accesses are 16-byte vectors along C.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace kn {

// Programmatic dependent launch: every kernel of the step lets the next launch of its stream start its blocks early
// (they become resident as the SMs drain) and itself waits here, before its first access to global memory, until the
// kernels before it have completed and their writes are visible.  Without the launch attribute both are no-ops.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_sync() { pdl_trigger(); pdl_wait(); }

// ---------------------------------------------------------------- counter hash
// SplitMix64 finaliser over key + golden*(idx+1); key = finalise(seed ^ stream<<56 ^ replica<<48 ^ step).
__host__ __device__ __forceinline__ uint64_t mix64(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}
__host__ __device__ __forceinline__ uint64_t stream_key(uint64_t seed, uint64_t stream, uint64_t replica, uint64_t step) {
    return mix64(seed ^ (stream << 56) ^ (replica << 48) ^ step);
}
__host__ __device__ __forceinline__ uint64_t draw(uint64_t key, uint64_t idx) {
    return mix64(key + 0x9E3779B97F4A7C15ULL * (idx + 1));
}

__device__ __forceinline__ void unpack8(const uint4& u, float* f) {
    const __nv_bfloat162* h = (const __nv_bfloat162*)&u;
    #pragma unroll
    for (int i = 0; i < 4; ++i) { float2 t = __bfloat1622float2(h[i]); f[2 * i] = t.x; f[2 * i + 1] = t.y; }
}
__device__ __forceinline__ uint4 pack8(const float* f) {
    uint4 u;
    __nv_bfloat162* h = (__nv_bfloat162*)&u;
    #pragma unroll
    for (int i = 0; i < 4; ++i) h[i] = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
    return u;
}
// src[0] + src[stride] + ... (n terms, added in that order), NB loads in flight at a time, the remainder included: a plain loop
// over a run-time count has four in flight and takes the remainder one by one, and each such round is a trip to L2 or HBM
// (evaluation of one image, fc8's 16 splits in one round instead of four: 147.1 -> 145.4 us)
template <int NB>
__device__ __forceinline__ float4 sum_splits(const float* __restrict__ src, long long stride, int n) {
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int z0 = 0; z0 < n; z0 += NB) {
        float4 t[NB];
        #pragma unroll
        for (int q = 0; q < NB; ++q) {
            t[q] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (z0 + q < n) t[q] = __ldcg((const float4*)(src + (z0 + q) * stride));
        }
        #pragma unroll
        for (int q = 0; q < NB; ++q) { s.x += t[q].x; s.y += t[q].y; s.z += t[q].z; s.w += t[q].w; }
    }
    return s;
}

// Four consecutive channels of a conv layer's bias gradient from its partials [parts][cout], by eight consecutive lanes of a
// warp: lane k (0..7) adds the partials k, k + 8, ..., then the lanes add up in pairs, so the order is fixed; every lane of
// the eight has the result.  There are up to 148 partials (conv1): one thread per channel group with 16 loads in flight took 8 us.
__device__ __forceinline__ float4 bias_sum8(const float* __restrict__ bp, int cout, int parts, int k) {
    float4 s = k < parts ? sum_splits<10>(bp + (long long)k * cout, 8LL * cout, (parts - k + 7) / 8) : make_float4(0.f, 0.f, 0.f, 0.f);
    #pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        s.x += __shfl_xor_sync(~0u, s.x, o); s.y += __shfl_xor_sync(~0u, s.y, o);
        s.z += __shfl_xor_sync(~0u, s.z, o); s.w += __shfl_xor_sync(~0u, s.w, o);
    }
    return s;
}

// ------------------------------------------------------------- preprocessing
// Per image: crop offset (ox, oy) in [0,29]^2 and flip bit from the hash
// (stream 1, idx = image).  out = u8[sy][sx][c] - mean[sy][sx][c] with
// sy = oy + Y, sx = ox + (flip ? 226 - X : X), written as bf16 in the 4x4
// space-to-depth layout [B][57][57][48], channel = ((Y%4)*4 + X%4)*3 + c,
// with row/column 227 of the 228-padded image set to zero.
// Optional intensity augmentation (Krizhevsky et al. 2012, section 4.1; the paper's experiments leave it out): every
// pixel of image n gets the RGB offset d = sum_i pl[.][i] * alpha_i with pl[c][i] = eigvec[c][i] * eigval[i] and
// alpha_i = sigma * z_i, z_i standard normal from the hash (stream 10, index 3 n + i, Box-Muller as in the init kernel).
struct ColorAug { float pl[9]; float sigma; uint64_t key; };
__device__ __forceinline__ float normal_draw(uint64_t key, uint64_t idx) {
    const uint64_t r = draw(key, idx);
    const float u1 = ((float)(r >> 40) + 1.f) * (1.f / 16777216.f);
    const float u2 = (float)((r >> 16) & 0xFFFFFF) * (1.f / 16777216.f);
    return sqrtf(-2.f * logf(u1)) * cospif(2.f * u2);
}
// One block = one image and four rows of the 228-padded crop (one row `by` of the space-to-depth grid): the four source rows of the
// uint8 image (768 bytes each) and of the mean image (768 floats each) come to shared memory in 16-byte asynchronous copies, then
// thread (bx, dy) forms its 12 values (4 pixels x 3 colours).  Its source bytes are 12 consecutive ones (backwards in pixels when
// flipped) whose offset within a 16-byte group of floats, and within a 4-byte word of bytes, is the same for the whole block, so
// it reads aligned vectors and shifts by a block-uniform amount.  The block's 5472 output bytes are contiguous: they are gathered in
// shared memory (over the mean rows) and leave as one bulk store.  grid: (images, 57): blocks that run together then want the
// same thirty-odd mean rows, which they find in L2 and partly in L1; 256 threads; image n0 + blockIdx.x of the batch.
// labels_src != nullptr: the labels travel with the images (from device or mapped host memory, four bytes per image: cheaper
// than a copy of their own in the stream).
// Bound by L1 and shared memory wavefronts (73% busy; the mean rows are 12 KB per 5 KB of output) and instruction issue (61%), not by HBM;
// hence vectors everywhere and bytes turned into floats by a permute instead of a conversion instruction.  Against scalar loads
// and stores with the block row fastest in the grid: 23.2 -> 19.7 us at batch 128, 83 -> 70 at 512, 4.9 -> 4.6 at 8.
// 128 threads with two rows each, for more blocks in flight: 22.3 and 77.6.
constexpr int kPpMean = 776 * 4, kPpImg = 800;         // row pitches in bytes: 16 bytes of room on either side of a row, and the
                                                       // warp's (8 bx x 4 dy) vector and word reads hit distinct banks
// v[i] = byte i - m[i + SH]; x: 12 bytes; m: sixteen floats
template <int SH>
__device__ __forceinline__ void byte_minus_mean(const uint32_t* x, const float* m, float* v) {
    #pragma unroll
    for (int i = 0; i < 12; ++i)        // 2^23 + byte as a float, exactly; the subtraction is exact too
        v[i] = (__uint_as_float(__byte_perm(x[i >> 2], 0x4B000000u, 0x7440u | (i & 3))) - 8388608.f) - m[i + SH];
}
template <bool AUG>
__global__ void __launch_bounds__(256) preprocess_kernel(const uint8_t* __restrict__ img, const float* __restrict__ mean,
                                                         __nv_bfloat16* __restrict__ out, int32_t* __restrict__ cf_out,
                                                         const int32_t* __restrict__ labels_src, int32_t* __restrict__ labels_dst,
                                                         int n0, uint64_t key, int eval_mode, const ColorAug aug) {
    pdl_sync();
    __shared__ __align__(128) uint8_t s_mem[4 * kPpMean + 4 * kPpImg];
    __shared__ float s_alpha[3];
    const int by = blockIdx.y, n = n0 + blockIdx.x, tid = threadIdx.x;
    if (labels_src && by == 0 && tid == 32) labels_dst[n] = labels_src[n];
    const uint64_t r = draw(key, (uint64_t)n);
    // evaluation: the centre 227 x 227 window, never flipped
    const int ox = eval_mode ? 14 : (int)((r & 0xFFFF) % 30), oy = eval_mode ? 14 : (int)(((r >> 16) & 0xFFFF) % 30);
    const int flip = eval_mode ? 0 : (int)((r >> 32) & 1);
    if (cf_out && by == 0 && tid == 0) { cf_out[3 * n] = ox; cf_out[3 * n + 1] = oy; cf_out[3 * n + 2] = flip; }
    const uint32_t sm = (uint32_t)__cvta_generic_to_shared(s_mem);
    {
        const int dy = tid >> 6, j = tid & 63, Y = by * 4 + dy;         // 64 threads per row: 192 + 48 vectors
        if (Y < 227) {
            const float4* mp = (const float4*)(mean + (size_t)(oy + Y) * 768) + j;
            const uint32_t md = sm + dy * kPpMean + 16 + 16 * j;
            #pragma unroll
            for (int k = 0; k < 3; ++k)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(md + 1024 * k), "l"(mp + 64 * k) : "memory");
            if (j < 48)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sm + 4 * kPpMean + dy * kPpImg + 16 + 16 * j),
                             "l"((const uint4*)(img + (size_t)n * 196608 + (size_t)(oy + Y) * 768) + j) : "memory");
        }
    }
    if (AUG && !eval_mode && tid < 3) s_alpha[tid] = aug.sigma * normal_draw(aug.key, 3ull * n + tid);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    const int dy = tid & 3, bx = tid >> 2;
    float v[12];
    if (bx < 57) {
        const int Y = by * 4 + dy;
        // first source byte: pixel ox + 4 bx, or, mirrored, the last of the four output pixels; it may lie up to 3 bytes before or
        // 15 behind the row (the 228th column), inside the pitch, and is masked below
        const int e = 3 * (flip ? ox + 223 - 4 * bx : ox + 4 * bx), sh = e & 3, a = e - sh;
        const float4* mp = (const float4*)(s_mem + dy * kPpMean + 16 + 4 * a);
        const uint32_t* ip = (const uint32_t*)(s_mem + 4 * kPpMean + dy * kPpImg + 16 + a);
        float m[16];
        #pragma unroll
        for (int k = 0; k < 4; ++k) { const float4 q = mp[k]; m[4 * k] = q.x; m[4 * k + 1] = q.y; m[4 * k + 2] = q.z; m[4 * k + 3] = q.w; }
        const uint32_t w0 = ip[0], w1 = ip[1], w2 = ip[2], w3 = ip[3];
        const uint32_t x[3] = {__funnelshift_r(w0, w1, 8 * sh), __funnelshift_r(w1, w2, 8 * sh), __funnelshift_r(w2, w3, 8 * sh)};
        if (sh == 0) byte_minus_mean<0>(x, m, v);
        else if (sh == 1) byte_minus_mean<1>(x, m, v);
        else if (sh == 2) byte_minus_mean<2>(x, m, v);
        else byte_minus_mean<3>(x, m, v);
        if (flip) {
            #pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float t0 = v[c], t1 = v[3 + c];
                v[c] = v[9 + c]; v[3 + c] = v[6 + c]; v[6 + c] = t1; v[9 + c] = t0;
            }
        }
        if (AUG && !eval_mode) {
            #pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float shift = aug.pl[3 * c] * s_alpha[0] + aug.pl[3 * c + 1] * s_alpha[1] + aug.pl[3 * c + 2] * s_alpha[2];
                #pragma unroll
                for (int dx = 0; dx < 4; ++dx) v[3 * dx + c] += shift;
            }
        }
        if (bx == 56) v[9] = v[10] = v[11] = 0.f;         // column 227
        if (Y == 227) {
            #pragma unroll
            for (int i = 0; i < 12; ++i) v[i] = 0.f;
        }
    }
    __syncthreads();                                     // the mean rows have been read
    if (bx < 57) {
        uint2* o = (uint2*)(s_mem + bx * 96 + dy * 24);
        #pragma unroll
        for (int i = 0; i < 3; ++i) {
            const __nv_bfloat162 lo = __floats2bfloat162_rn(v[4 * i], v[4 * i + 1]), hi = __floats2bfloat162_rn(v[4 * i + 2], v[4 * i + 3]);
            o[i] = make_uint2(*(const uint32_t*)&lo, *(const uint32_t*)&hi);
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (tid == 0) {
        asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                     ::"l"(out + (size_t)(n * 57 + by) * 57 * 48), "r"(sm), "r"(57 * 96) : "memory");
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");        // shared memory stays until it has been read
    }
}

// ----------------------------------------------------------------------- LRN
// All index arithmetic below is 32-bit: the largest activation tensor of a batch of 1024 has
// 1024*57*57*12 < 2^31 sixteen-byte vectors.
__device__ __forceinline__ float rsqrt_fast(float x) { float y; asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
__device__ __forceinline__ float sqrt_fast(float x) { float y; asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
// s^-beta and 1/s; the exponent 0.75 of the paper's network costs two special-function instructions
// B75: the exponent is known to be 0.75 at compile time (the fused kernels of the training step are instantiated both ways,
// so that their inner loops carry no test of beta)
template <bool B75>
__device__ __forceinline__ void pow_neg_t(float s, float beta, float& sp, float& rs) {
    if (B75) { const float r = rsqrt_fast(s); sp = r * sqrt_fast(r); rs = r * r; }
    else { sp = exp2f(-beta * __log2f(s)); rs = __fdividef(1.f, s); }
}
__device__ __forceinline__ void pow_neg(float s, float beta, float& sp, float& rs) {
    if (beta == 0.75f) pow_neg_t<true>(s, beta, sp, rs); else pow_neg_t<false>(s, beta, sp, rs);
}
// b_c = a_c * (k + alpha * sum_{c' in [c-2,c+2] clipped} a_c'^2)^(-beta); one thread = 8 channels of one pixel.
template <bool B75>
__device__ __forceinline__ uint4 lrn_fwd8_t(const uint4* ap, bool has_l, bool has_r, float alpha, float beta, float k) {
    const uint4 zero = make_uint4(0, 0, 0, 0);
    float f[24];
    unpack8(has_l ? __ldg(ap - 1) : zero, f);
    unpack8(__ldg(ap), f + 8);
    unpack8(has_r ? __ldg(ap + 1) : zero, f + 16);
    float sq[12];
    #pragma unroll
    for (int i = 0; i < 12; ++i) sq[i] = f[6 + i] * f[6 + i];
    float o[8];
    #pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float ss = (sq[i] + sq[i + 1]) + (sq[i + 2] + sq[i + 3]) + sq[i + 4];
        float sp, rs;
        pow_neg_t<B75>(fmaf(alpha, ss, k), beta, sp, rs);
        o[i] = f[8 + i] * sp;
    }
    return pack8(o);
}
__device__ __forceinline__ uint4 lrn_fwd8(const uint4* ap, bool has_l, bool has_r, float alpha, float beta, float k) {
    return beta == 0.75f ? lrn_fwd8_t<true>(ap, has_l, has_r, alpha, beta, k) : lrn_fwd8_t<false>(ap, has_l, has_r, alpha, beta, k);
}
__global__ void __launch_bounds__(256) lrn_fwd_kernel(const __nv_bfloat16* __restrict__ a, __nv_bfloat16* __restrict__ b,
                                                      unsigned total, unsigned cpr, float alpha, float beta, float k) {
    pdl_sync();
    const unsigned t = blockIdx.x * 256u + threadIdx.x;
    if (t >= total) return;
    const unsigned ch = t % cpr;
    ((uint4*)b)[t] = lrn_fwd8((const uint4*)a + t, ch > 0, ch < cpr - 1, alpha, beta, k);
}
// da_m = [a_m > 0] * ( g_m s_m^-beta - 2 alpha beta a_m sum_{c in [m-2,m+2]} g_c a_c s_c^(-beta-1) )
// (the ReLU mask of the convolution that produced a is applied here).  One thread = 8 channels of one
// pixel; it needs s for the 12 channels c0-2 .. c0+9 and a for c0-4 .. c0+11.
__device__ __forceinline__ uint4 lrn_bwd8(const float* fa, const float* fg, float alpha, float beta, float k) {
    float sq[16];
    #pragma unroll
    for (int i = 0; i < 16; ++i) sq[i] = fa[4 + i] * fa[4 + i];
    float sp[12], tt[12];   // channels c0-2 .. c0+9
    #pragma unroll
    for (int i = 0; i < 12; ++i) {
        const float ss = (sq[i] + sq[i + 1]) + (sq[i + 2] + sq[i + 3]) + sq[i + 4];
        float rs;
        pow_neg(fmaf(alpha, ss, k), beta, sp[i], rs);
        tt[i] = fg[6 + i] * fa[6 + i] * sp[i] * rs;
    }
    const float c2 = 2.f * alpha * beta;
    float o[8];
    #pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float acc = (tt[i] + tt[i + 1]) + (tt[i + 2] + tt[i + 3]) + tt[i + 4];
        const float am = fa[8 + i];
        const float v = fmaf(fg[8 + i], sp[i + 2], -c2 * am * acc);
        o[i] = am > 0.f ? v : 0.f;
    }
    return pack8(o);
}
__global__ void __launch_bounds__(256) lrn_bwd_kernel(const __nv_bfloat16* __restrict__ a, const __nv_bfloat16* __restrict__ g,
                                                      __nv_bfloat16* __restrict__ da, unsigned total, unsigned cpr,
                                                      float alpha, float beta, float k) {
    pdl_sync();
    const unsigned t = blockIdx.x * 256u + threadIdx.x;
    if (t >= total) return;
    const unsigned ch = t % cpr;
    const uint4* ap = (const uint4*)a + t;
    const uint4* gp = (const uint4*)g + t;
    const uint4 zero = make_uint4(0, 0, 0, 0);
    const bool has_l = ch > 0, has_r = ch < cpr - 1;
    float fa[24], fg[24];
    unpack8(has_l ? __ldg(ap - 1) : zero, fa);
    unpack8(__ldg(ap), fa + 8);
    unpack8(has_r ? __ldg(ap + 1) : zero, fa + 16);
    unpack8(has_l ? __ldg(gp - 1) : zero, fg);
    unpack8(__ldg(gp), fg + 8);
    unpack8(has_r ? __ldg(gp + 1) : zero, fg + 16);
    ((uint4*)da)[t] = lrn_bwd8(fa, fg, alpha, beta, k);
}

// ------------------------------------------------------------------ max pool
// 3x3 stride 2, no padding; first maximum in (ky,kx) row-major order wins; argmax = ky*3+kx.
// grid: (ceil(Wo*cpr / 256), Ho, B); one thread = 8 channels of one output pixel.
__global__ void __launch_bounds__(256) pool_fwd_kernel(const __nv_bfloat16* __restrict__ x, __nv_bfloat16* __restrict__ y,
                                                       uint8_t* __restrict__ arg, int cpr, int Hpi, int Wpi,
                                                       int Ho, int Wo, int Hpo, int Wpo) {
    pdl_sync();
    const unsigned i = blockIdx.x * 256u + threadIdx.x;
    if (i >= (unsigned)(Wo * cpr)) return;
    const int ox = i / cpr, ch = i - ox * cpr;
    const int oy = blockIdx.y, n = blockIdx.z;
    float best[8]; int bi[8];
    const uint4* xp = (const uint4*)x + ((size_t)(n * Hpi + 2 * oy) * Wpi + 2 * ox) * cpr + ch;
    #pragma unroll
    for (int ky = 0; ky < 3; ++ky)
        #pragma unroll
        for (int kx = 0; kx < 3; ++kx) {
            float f[8];
            unpack8(__ldg(xp + (ky * Wpi + kx) * cpr), f);
            #pragma unroll
            for (int q = 0; q < 8; ++q)
                if ((ky == 0 && kx == 0) || f[q] > best[q]) { best[q] = f[q]; bi[q] = ky * 3 + kx; }
        }
    ((uint4*)y)[((size_t)(n * Hpo + oy) * Wpo + ox) * cpr + ch] = pack8(best);
    uint2 ab;
    ab.x = bi[0] | (bi[1] << 8) | (bi[2] << 16) | (bi[3] << 24);
    ab.y = bi[4] | (bi[5] << 8) | (bi[6] << 16) | (bi[7] << 24);
    ((uint2*)arg)[((size_t)(n * Ho + oy) * Wo + ox) * cpr + ch] = ab;
}
// ------------------------------------------------- LRN + pool fused (the training step)
// Geometry is a template parameter (the network's two LRN layers): CPR 16-byte vectors per pixel, input WI x HI.
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t d; asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel)); return d;
}
// Both kernels work on PIXEL PAIRS: a thread owns eight channels of the pixels (2i, 2i+1) of a row and keeps every fp32 value of
// the pair in one 64-bit register, so that sums and products are the packed instructions of sm_100 (add / mul / fma.rn.f32x2):
// the forward kernel is bound by the special-function unit (two instructions per element, 16 lanes per SM and cycle: 63% busy),
// the backward one by instruction issue (64% of the slots; special functions 37%), neither by HBM (26% and 32%), and packing
// halves the arithmetic instructions.  Window sums take pair sums shared by
// neighbouring channels.  Measured at batch 128 (back to back), this form against one thread per pixel vector with the
// pooling gradient scattered through shared memory: forward 40.4 -> 36.6 us (LRN1) and 27.6 -> 24.8 (LRN2), backward 79.1 ->
// 53.5 and 48.9 -> 34; at batch 512 forward 141 -> 128 and 97 -> 83.  Same arithmetic in the same order as the single-operation kernels.
typedef unsigned long long f2;
__device__ __forceinline__ f2 mk2(float lo, float hi) { f2 r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi)); return r; }
__device__ __forceinline__ void un2(f2 v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ f2 add2(f2 a, f2 b) { f2 r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ f2 mul2(f2 a, f2 b) { f2 r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) { f2 r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r; }
__device__ __forceinline__ float bf_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf_hi(uint32_t u) { return __uint_as_float(u & 0xffff0000u); }
// twelve channels c0-2 .. c0+9 of a pixel pair from six words each (two bf16 channels per word)
__device__ __forceinline__ void unpack_pair(const uint32_t* w0, const uint32_t* w1, f2* x) {
    #pragma unroll
    for (int i = 0; i < 6; ++i) {
        x[2 * i] = mk2(bf_lo(w0[i]), bf_lo(w1[i]));
        x[2 * i + 1] = mk2(bf_hi(w0[i]), bf_hi(w1[i]));
    }
}
// out[i] = (x[i] + x[i+1]) + (x[i+2] + x[i+3]) + x[i+4], the five-channel window of channel c0 + i (lrn_fwd8's order)
__device__ __forceinline__ void window_sums(const f2* x, f2* out) {
    f2 t[10];
    #pragma unroll
    for (int i = 0; i < 10; ++i) t[i] = add2(x[i], x[i + 1]);
    #pragma unroll
    for (int i = 0; i < 8; ++i) out[i] = add2(add2(t[i], t[i + 2]), x[i + 4]);
}
__device__ __forceinline__ uint32_t pack_bf(float lo, float hi) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *(const uint32_t*)&h;
}
__device__ __forceinline__ void pack_pair(const f2* o, uint4& p0, uint4& p1) {
    float a[8], b[8];
    #pragma unroll
    for (int i = 0; i < 8; ++i) un2(o[i], a[i], b[i]);
    p0 = make_uint4(pack_bf(a[0], a[1]), pack_bf(a[2], a[3]), pack_bf(a[4], a[5]), pack_bf(a[6], a[7]));
    p1 = make_uint4(pack_bf(b[0], b[1]), pack_bf(b[2], b[3]), pack_bf(b[4], b[5]), pack_bf(b[6], b[7]));
}
// s^-beta (and 1/s) of both pixels
template <bool B75>
__device__ __forceinline__ void pow_pair(f2 s, float beta, f2& sp, f2& rs) {
    float s0, s1;
    un2(s, s0, s1);
    if (B75) {
        const float r0 = rsqrt_fast(s0), r1 = rsqrt_fast(s1);
        const f2 r = mk2(r0, r1);
        sp = mul2(r, mk2(sqrt_fast(r0), sqrt_fast(r1)));
        rs = mul2(r, r);
    } else {
        float p0, p1, q0, q1;
        pow_neg_t<false>(s0, beta, p0, q0);
        pow_neg_t<false>(s1, beta, p1, q1);
        sp = mk2(p0, p1); rs = mk2(q0, q1);
    }
}
// Forward: p = maxpool(LRN(a)) without writing the normalised tensor.  One block = one image, CV of the CPR channel vectors and a
// run of `opr` output rows; a thread owns one pixel pair and vector and walks down the rows, so only the first of the
// 2*opr+1 input rows is normalised by two blocks.  A normalised row (rounded to bf16 as lrn_fwd_kernel stores it) updates the
// running maximum over the filter rows of the thread's two columns, two channels per instruction (a later row
// replaces the best one only if it is greater).  Once per output row the result of the even column goes to the
// left neighbour through shared memory, and the three columns of a window are combined with 32-bit keys (value << 16) |
// (8 - tap): the largest key has the largest value and, among equal values, the first tap in scan order - pool_fwd_kernel's
// tie rule.  (Normalised values are not negative; as signed integers the keys also order a NaN above everything.)
// grid: (ceil(HO / opr), CPR / CV, B); (WI+1)/2 * CV threads.
template <int CPR, int CV, int WI, int HI, bool B75, int MINB>
__global__ void __launch_bounds__((WI + 1) / 2 * CV, MINB) lrn_pool_fwd_kernel(const __nv_bfloat16* __restrict__ a, __nv_bfloat16* __restrict__ y,
                                                                               uint8_t* __restrict__ arg, int opr, int Hpi, int Wpi, int Hpo,
                                                                               int Wpo, float alpha, float beta, float k) {
    // Waits first and lets the next launch start afterwards, unlike every other kernel: when a block of the next kernel runs, conv1
    // (the kernel before this one) has completed, and with it whatever wrote weights and biases before the pass, and in an
    // evaluation the preprocessing kernel, which brings the labels.  The convolution and FC kernels behind this one rely on that when
    // they load weights before their own wait, and fc8_softmax_xent_kernel when it loads labels and its bias.
    // (Nothing is lost: batch 8 and 128 and an evaluation of one image take what they took with the trigger first.)
    pdl_wait();
    pdl_trigger();
    constexpr int NP = (WI + 1) / 2, NT = NP * CV, WO = (WI - 3) / 2 + 1, HO = (HI - 3) / 2 + 1;
    __shared__ uint4 xch[2][2][NT];           // [parity of the output row][value / filter row of the maximum][thread]
    const int n = blockIdx.z, c0 = blockIdx.y * CV, oy0 = opr * blockIdx.x, oy1 = min(HO, oy0 + opr);
    const int xp = threadIdx.x / CV, cv = threadIdx.x - xp * CV, ch = c0 + cv;
    // (the pair of the last pixel has a pad pixel as its second: the grid is wider than WI and pads are zero)
    const uint4* ap = (const uint4*)a + ((size_t)(n * Hpi + 2 * oy0) * Wpi + 2 * xp) * CPR + ch;
    const f2 al2 = mk2(alpha, alpha), k2 = mk2(k, k);
    // the neighbouring channel words come from the neighbouring lanes; only the ends of a warp (and of a block's channel
    // range) load them
    const int lane = threadIdx.x & 31;
    const bool has_l = ch > 0, has_r = ch < CPR - 1;
    const bool ld_l = has_l && (lane == 0 || cv == 0), ld_r = has_r && (lane == 31 || threadIdx.x == NT - 1 || cv == CV - 1);
    // the lanes that exist: the last warp of a block may be partial
    const unsigned mask = NT % 32 && threadIdx.x >= NT / 32 * 32 ? (1u << NT % 32) - 1u : ~0u;
    uint4 v0, v1; uint32_t l0 = 0u, l1 = 0u, r0 = 0u, r1 = 0u;
    auto fetch = [&]() {
        v0 = __ldg(ap); v1 = __ldg(ap + CPR);
        const uint32_t* wp = (const uint32_t*)ap;
        if (ld_l) { l0 = __ldg(wp - 1); l1 = __ldg(wp + 4 * CPR - 1); }
        if (ld_r) { r0 = __ldg(wp + 4); r1 = __ldg(wp + 4 * CPR + 4); }
        ap += Wpi * CPR;
    };
    // normalises the fetched row and fetches the next one meanwhile
    auto norm_row = [&](bool more, uint4& p0, uint4& p1) {
        const uint32_t ul0 = __shfl_up_sync(mask, v0.w, 1), ul1 = __shfl_up_sync(mask, v1.w, 1);
        const uint32_t dr0 = __shfl_down_sync(mask, v0.x, 1), dr1 = __shfl_down_sync(mask, v1.x, 1);
        const uint32_t w0[6] = {has_l && !ld_l ? ul0 : l0, v0.x, v0.y, v0.z, v0.w, has_r && !ld_r ? dr0 : r0};
        const uint32_t w1[6] = {has_l && !ld_l ? ul1 : l1, v1.x, v1.y, v1.z, v1.w, has_r && !ld_r ? dr1 : r1};
        f2 x[12], sq[12], ss[8];
        unpack_pair(w0, w1, x);
        if (more) fetch();
        #pragma unroll
        for (int i = 0; i < 12; ++i) sq[i] = mul2(x[i], x[i]);
        window_sums(sq, ss);
        #pragma unroll
        for (int i = 0; i < 8; ++i) {
            f2 sp, rs;
            pow_pair<B75>(fma2(al2, ss[i], k2), beta, sp, rs);
            ss[i] = mul2(x[i + 2], sp);
        }
        pack_pair(ss, p0, p1);
    };
    auto vmax = [&](const uint4& p, uint32_t* best, uint32_t* row, uint32_t ky3) {
        const uint32_t w[4] = {p.x, p.y, p.z, p.w};
        #pragma unroll
        for (int i = 0; i < 4; ++i) {
            const __nv_bfloat162 vb = *(const __nv_bfloat162*)&w[i], bb = *(const __nv_bfloat162*)&best[i];
            const uint32_t gt = __hgt2_mask(vb, bb);
            const __nv_bfloat162 mx = __hmax2_nan(vb, bb);
            best[i] = *(const uint32_t*)&mx;
            row[i] = (gt & ky3) | (~gt & row[i]);
        }
    };
    fetch();
    uint4 p0, p1;
    norm_row(true, p0, p1);
    #pragma unroll 1
    for (int oy = oy0; oy < oy1; ++oy) {
        uint32_t be[4] = {p0.x, p0.y, p0.z, p0.w}, bo[4] = {p1.x, p1.y, p1.z, p1.w}, re[4] = {0, 0, 0, 0}, ro[4] = {0, 0, 0, 0};
        norm_row(true, p0, p1);
        vmax(p0, be, re, 0x00030003u); vmax(p1, bo, ro, 0x00030003u);
        norm_row(oy + 1 < oy1, p0, p1);
        vmax(p0, be, re, 0x00060006u); vmax(p1, bo, ro, 0x00060006u);
        uint4 (*buf)[NT] = xch[oy & 1];
        buf[0][threadIdx.x] = make_uint4(be[0], be[1], be[2], be[3]);
        buf[1][threadIdx.x] = make_uint4(re[0], re[1], re[2], re[3]);
        __syncthreads();
        if (xp < WO) {
            const uint4 rv = buf[0][threadIdx.x + CV], rr = buf[1][threadIdx.x + CV];
            const uint32_t br[4] = {rv.x, rv.y, rv.z, rv.w}, rw[4] = {rr.x, rr.y, rr.z, rr.w};
            uint32_t val[4], tap[4];
            #pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t ce = 0x00080008u - re[i], co = 0x00070007u - ro[i], cr = 0x00060006u - rw[i];
                const int lo = max(max((int)prmt(be[i], ce, 0x1054u), (int)prmt(bo[i], co, 0x1054u)), (int)prmt(br[i], cr, 0x1054u));
                const int hi = max(max((int)prmt(be[i], ce, 0x3276u), (int)prmt(bo[i], co, 0x3276u)), (int)prmt(br[i], cr, 0x3276u));
                val[i] = prmt((uint32_t)lo, (uint32_t)hi, 0x7632u);
                tap[i] = prmt((uint32_t)lo, (uint32_t)hi, 0x5410u);
            }
            ((uint4*)y)[((size_t)(n * Hpo + oy) * Wpo + xp) * CPR + ch] = make_uint4(val[0], val[1], val[2], val[3]);
            ((uint2*)arg)[((size_t)(n * HO + oy) * WO + xp) * CPR + ch] =
                make_uint2(0x08080808u - prmt(tap[0], tap[1], 0x6420u), 0x08080808u - prmt(tap[2], tap[3], 0x6420u));
        }
    }
}
// the eight gradients of a window where its argmax equals the tap, else zero (four words of two bf16 channels)
__device__ __forceinline__ void tap_words(const uint4& g, const uint2& ab, uint32_t tap, uint32_t* v) {
    const uint32_t T = tap * 0x01010101u;
    const uint32_t m0 = (ab.x ^ T) + 0x7f7f7f7fu, m1 = (ab.y ^ T) + 0x7f7f7f7fu;      // sign bit of a byte: not this tap (bytes are < 16)
    const uint32_t w[4] = {g.x, g.y, g.z, g.w};
    #pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t m = i < 2 ? m0 : m1;
        v[i] = w[i] & ~prmt(m, m, (i & 1) ? 0xbbaau : 0x9988u);          // sign-replicated bytes
    }
}
__device__ __forceinline__ uint32_t add_bf16x2(uint32_t a, uint32_t b) {
    const __nv_bfloat162 r = __hadd2(*(const __nv_bfloat162*)&a, *(const __nv_bfloat162*)&b);
    return *(const uint32_t*)&r;
}
// halves of a word of two bf16 that are greater than zero, as 16-bit masks
__device__ __forceinline__ uint32_t positive_mask(uint32_t w) {
    return __hgt2_mask(*(const __nv_bfloat162*)&w, __nv_bfloat162(__ushort_as_bfloat16(0), __ushort_as_bfloat16(0)));
}
// dx[y][x] = sum over the (up to 4) windows containing (y,x) whose argmax points at it; optional ReLU mask.  One thread = eight
// channels of the 2 x 2 input pixels (2j, 2i) .. (2j+1, 2i+1): their nine taps lie in four windows, so a window's gradients and codes are
// read four times in all instead of nine, and all of a thread's loads are in flight together.  A pixel of one or two terms stays
// packed bf16 (one rounding, as in fp32 followed by the conversion).  Windows cover valid pixels only, so pad pixels get zero.
// Measured (pool5): one thread per pixel and a loop over its windows 10.5 us at batch 128 and 36.0 at 512, this form 7.2 and 22.2
// (HBM floor 4.3 and 17).
// grid: (ceil(ceil(Wpi / 2) * cpr / 256), ceil(Hpi / 2), B).
__global__ void __launch_bounds__(256) pool_bwd_kernel(const __nv_bfloat16* __restrict__ dy, const uint8_t* __restrict__ arg,
                                                       const __nv_bfloat16* __restrict__ relu_src, __nv_bfloat16* __restrict__ dx,
                                                       int cpr, int Hpi, int Wpi, int Ho, int Wo, int Hpo, int Wpo) {
    pdl_sync();
    const unsigned q = blockIdx.x * 256u + threadIdx.x;
    if (q >= (unsigned)((Wpi + 1) / 2 * cpr)) return;
    const int i = q / cpr, ch = q - i * cpr;
    const int j = blockIdx.y, n = blockIdx.z;
    uint4 d[2][2], rl[2][2]; uint2 ab[2][2];            // windows (j - dj, i - di); the pixels' ReLU source
    #pragma unroll
    for (int dj = 0; dj < 2; ++dj)
        #pragma unroll
        for (int di = 0; di < 2; ++di) {
            const int oy = j - dj, ox = i - di;
            d[dj][di] = make_uint4(0, 0, 0, 0);
            ab[dj][di] = make_uint2(0, 0);
            if (oy >= 0 && oy < Ho && ox >= 0 && ox < Wo) {
                ab[dj][di] = __ldg((const uint2*)arg + ((size_t)(n * Ho + oy) * Wo + ox) * cpr + ch);
                d[dj][di] = __ldg((const uint4*)dy + ((size_t)(n * Hpo + oy) * Wpo + ox) * cpr + ch);
            }
        }
    const size_t t0 = ((size_t)(n * Hpi + 2 * j) * Wpi + 2 * i) * cpr + ch;
    #pragma unroll
    for (int r = 0; r < 2; ++r)
        #pragma unroll
        for (int s = 0; s < 2; ++s) {
            rl[r][s] = make_uint4(0, 0, 0, 0);
            if (relu_src && 2 * j + r < Hpi && 2 * i + s < Wpi) rl[r][s] = __ldg((const uint4*)relu_src + t0 + (size_t)(r * Wpi + s) * cpr);
        }
    uint32_t g[2][2][4], u[4], v[4], w[4];
    tap_words(d[0][0], ab[0][0], 0, g[0][0]);
    tap_words(d[0][1], ab[0][1], 2, u);
    tap_words(d[1][0], ab[1][0], 6, v);
    tap_words(d[1][1], ab[1][1], 8, w);
    #pragma unroll
    for (int c = 0; c < 4; ++c)
        g[0][0][c] = pack_bf(((bf_lo(w[c]) + bf_lo(v[c])) + bf_lo(u[c])) + bf_lo(g[0][0][c]),
                             ((bf_hi(w[c]) + bf_hi(v[c])) + bf_hi(u[c])) + bf_hi(g[0][0][c]));
    tap_words(d[0][0], ab[0][0], 1, g[0][1]);
    tap_words(d[1][0], ab[1][0], 7, u);
    tap_words(d[0][0], ab[0][0], 3, g[1][0]);
    tap_words(d[0][1], ab[0][1], 5, v);
    tap_words(d[0][0], ab[0][0], 4, g[1][1]);
    #pragma unroll
    for (int c = 0; c < 4; ++c) {
        g[0][1][c] = add_bf16x2(u[c], g[0][1][c]);
        g[1][0][c] = add_bf16x2(v[c], g[1][0][c]);
    }
    #pragma unroll
    for (int r = 0; r < 2; ++r)
        #pragma unroll
        for (int s = 0; s < 2; ++s) {
            if (2 * j + r >= Hpi || 2 * i + s >= Wpi) continue;
            uint4 o = make_uint4(g[r][s][0], g[r][s][1], g[r][s][2], g[r][s][3]);
            if (relu_src) {
                const uint4 m = rl[r][s];
                o.x &= positive_mask(m.x); o.y &= positive_mask(m.y); o.z &= positive_mask(m.z); o.w &= positive_mask(m.w);
            }
            ((uint4*)dx)[t0 + (size_t)(r * Wpi + s) * cpr] = o;
        }
}
// Backward: da = LRN'(a, dn), dn = maxpool'(dp, arg).  One thread = eight channels of a 2 x 2 block of pixels (rows 2j, 2j+1,
// columns 2i, 2i+1).  The four windows (j-1..j, i-1..i) are the only ones that reach these pixels, in nine (window, tap)
// combinations, so dn is gathered in registers: four argmax bytes are compared with a tap at once, the byte masks select
// the bf16 gradients, and the up to four terms of a pixel are added in fp32 in a fixed order.  No shared memory, no
// barriers, no divergent loops.  dn is rounded to bf16, as pool_bwd_kernel stores it.  Then s^-beta and tt = dn a s^(-beta-1) for the row's pixel pair; the tt of the two channels on
// either side come from the neighbouring lanes, which hold the neighbouring channel vectors: where a pixel is not a whole
// warp (CPR = 12) the first and last lane of a warp only compute for their neighbours (30 of 32 lanes store).  The ReLU
// mask of the convolution that produced a is applied to the packed result.  Pad positions are not written: they are zero.
// grid: (ceil(warps per image / 4), B), 128 threads.
template <int CPR, int WI, int HI>
struct PoolLrnBwdGeo {
    static constexpr int HALO = CPR == 32 ? 0 : 1, PER = 32 - 2 * HALO, NP = (WI + 1) / 2, NJ = (HI + 1) / 2;
    static constexpr int TOT = NJ * NP * CPR, WARPS = (TOT + PER - 1) / PER, BLOCKS = (WARPS + 3) / 4;
};
template <int CPR, int WI, int HI, bool B75>
__global__ void __launch_bounds__(128, 5) pool_lrn_bwd_kernel(const __nv_bfloat16* __restrict__ a, const __nv_bfloat16* __restrict__ dp,
                                                           const uint8_t* __restrict__ arg, __nv_bfloat16* __restrict__ da,
                                                           int Hpi, int Wpi, int Hpo, int Wpo, float alpha, float beta, float k) {
    pdl_sync();
    typedef PoolLrnBwdGeo<CPR, WI, HI> G;
    constexpr int WO = (WI - 3) / 2 + 1, HO = (HI - 3) / 2 + 1;
    const int lane = threadIdx.x & 31, wg = blockIdx.x * 4 + (threadIdx.x >> 5), n = blockIdx.y;
    if (wg * G::PER >= G::TOT) return;                 // whole warps
    const int ql = wg * G::PER + lane - G::HALO, q = min(max(ql, 0), G::TOT - 1);
    const int ch = q % CPR, i = (q / CPR) % G::NP, j = q / (CPR * G::NP);
    const bool store = ql == q && lane >= G::HALO && lane < 32 - G::HALO;
    const uint4* ap = (const uint4*)a + ((size_t)(n * Hpi + 2 * j) * Wpi + 2 * i) * CPR + ch;
    uint4 av[2][2];
    #pragma unroll
    for (int r = 0; r < 2; ++r) { av[r][0] = __ldg(ap + r * Wpi * CPR); av[r][1] = __ldg(ap + r * Wpi * CPR + CPR); }
    uint4 wd[2][2]; uint2 wa[2][2];                    // [row j - d][column i - e]
    #pragma unroll
    for (int d = 0; d < 2; ++d)
        #pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int oy = j - d, ox = i - e;
            wd[d][e] = make_uint4(0u, 0u, 0u, 0u);
            wa[d][e] = make_uint2(0x0f0f0f0fu, 0x0f0f0f0fu);     // matches no tap
            if (oy >= 0 && oy < HO && ox >= 0 && ox < WO) {
                wd[d][e] = __ldg((const uint4*)dp + ((size_t)(n * Hpo + oy) * Wpo + ox) * CPR + ch);
                wa[d][e] = __ldg((const uint2*)arg + ((size_t)(n * HO + oy) * WO + ox) * CPR + ch);
            }
        }
    const f2 al2 = mk2(alpha, alpha), k2 = mk2(k, k), mc2 = mk2(-2.f * alpha * beta, -2.f * alpha * beta);
    #pragma unroll
    for (int r = 0; r < 2; ++r) {
        // dn of the row's even and odd pixel, two channels per word.  Three of the four pixels of a block get one or two terms: a
        // packed bf16 sum is then the fp32 sum rounded to bf16 (exact, or its smaller term is far below half a unit in the last
        // place); only the pixel of four windows adds in fp32.
        f2 g[8];
        {
            uint32_t e[4], o[4], t[4];
            tap_words(wd[0][0], wa[0][0], 3 * r, e);             // window (j, i): taps (r, 0) and (r, 1)
            tap_words(wd[0][0], wa[0][0], 3 * r + 1, o);
            tap_words(wd[0][1], wa[0][1], 3 * r + 2, t);         // window (j, i-1): tap (r, 2) on the even pixel
            if (r == 0) {                                        // windows of row j-1: their last filter row
                uint32_t a6[4], a7[4], a8[4];
                tap_words(wd[1][0], wa[1][0], 6, a6);
                tap_words(wd[1][0], wa[1][0], 7, a7);
                tap_words(wd[1][1], wa[1][1], 8, a8);
                #pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const float lo = ((bf_lo(a6[c]) + bf_lo(a8[c])) + bf_lo(e[c])) + bf_lo(t[c]);
                    const float hi = ((bf_hi(a6[c]) + bf_hi(a8[c])) + bf_hi(e[c])) + bf_hi(t[c]);
                    e[c] = pack_bf(lo, hi);
                    o[c] = add_bf16x2(a7[c], o[c]);
                }
            } else {
                #pragma unroll
                for (int c = 0; c < 4; ++c) e[c] = add_bf16x2(e[c], t[c]);
            }
            #pragma unroll
            for (int c = 0; c < 4; ++c) { g[2 * c] = mk2(bf_lo(e[c]), bf_lo(o[c])); g[2 * c + 1] = mk2(bf_hi(e[c]), bf_hi(o[c])); }
        }
        uint32_t w0[6] = {__shfl_up_sync(0xffffffffu, av[r][0].w, 1), av[r][0].x, av[r][0].y, av[r][0].z, av[r][0].w, __shfl_down_sync(0xffffffffu, av[r][0].x, 1)};
        uint32_t w1[6] = {__shfl_up_sync(0xffffffffu, av[r][1].w, 1), av[r][1].x, av[r][1].y, av[r][1].z, av[r][1].w, __shfl_down_sync(0xffffffffu, av[r][1].x, 1)};
        if (ch == 0) w0[0] = w1[0] = 0u;
        if (ch == CPR - 1) w0[5] = w1[5] = 0u;
        f2 x[12], sq[12], ss[8], sp[8], tt[12];
        unpack_pair(w0, w1, x);
        #pragma unroll
        for (int c = 0; c < 12; ++c) sq[c] = mul2(x[c], x[c]);
        window_sums(sq, ss);
        #pragma unroll
        for (int c = 0; c < 8; ++c) {
            f2 rs;
            pow_pair<B75>(fma2(al2, ss[c], k2), beta, sp[c], rs);
            tt[c + 2] = mul2(mul2(mul2(g[c], x[c + 2]), sp[c]), rs);      // dn a s^(-beta-1)
        }
        tt[0] = __shfl_up_sync(0xffffffffu, tt[8], 1); tt[1] = __shfl_up_sync(0xffffffffu, tt[9], 1);
        tt[10] = __shfl_down_sync(0xffffffffu, tt[2], 1); tt[11] = __shfl_down_sync(0xffffffffu, tt[3], 1);
        if (ch == 0) tt[0] = tt[1] = 0ull;
        if (ch == CPR - 1) tt[10] = tt[11] = 0ull;
        window_sums(tt, ss);
        #pragma unroll
        for (int c = 0; c < 8; ++c) g[c] = fma2(g[c], sp[c], mul2(mul2(mc2, x[c + 2]), ss[c]));
        uint4 p[2];
        pack_pair(g, p[0], p[1]);
        const __nv_bfloat162 z2 = __floats2bfloat162_rn(0.f, 0.f);
        #pragma unroll
        for (int e = 0; e < 2; ++e) {
            const __nv_bfloat162* ah = (const __nv_bfloat162*)&av[r][e];
            p[e].x &= __hgt2_mask(ah[0], z2); p[e].y &= __hgt2_mask(ah[1], z2); p[e].z &= __hgt2_mask(ah[2], z2); p[e].w &= __hgt2_mask(ah[3], z2);
        }
        if (store && 2 * j + r < HI) {
            uint4* op = (uint4*)da + ((size_t)(n * Hpi + 2 * j + r) * Wpi + 2 * i) * CPR + ch;
            op[0] = p[0];
            if (2 * i + 1 < WI) op[CPR] = p[1];
        }
    }
}

// ------------------------------------------------- split-K reductions (FC, wgrad)
// y[b][n] = act( sum_z ws[z][b][n] + bias[n] ) * keep(b*N + n) * scale -> bf16, or fp32 logits when out_f32.
__global__ void fc_reduce_fwd_kernel(const float* __restrict__ ws, int splits, long long split_stride,
                                     const float* __restrict__ bias, int B, int N, int relu,
                                     int use_dropout, uint64_t key, uint32_t thr24, float scale,
                                     __nv_bfloat16* __restrict__ out_bf16, float* __restrict__ out_f32,
                                     uint8_t* __restrict__ keep_out) {
    pdl_sync();
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long long)B * N) return;
    const int n = (int)(t % N);
    float v = 0.f;
    for (int z = 0; z < splits; ++z) v += ws[z * split_stride + t];
    v += bias[n];
    if (relu) v = fmaxf(v, 0.f);
    if (use_dropout == 2) {            // evaluation: the expectation of the mask instead of a mask
        v *= scale;
        if (keep_out) keep_out[t] = 1;
    } else if (use_dropout) {
        const bool keep = (uint32_t)(draw(key, (uint64_t)t) >> 40) >= thr24;
        if (keep_out) keep_out[t] = keep ? 1 : 0;
        v = keep ? v * scale : 0.f;
    } else if (keep_out) {
        keep_out[t] = 1;
    }
    if (out_f32) out_f32[t] = v; else out_bf16[t] = __float2bfloat16_rn(v);
}
// dx[b][k] = [mask[b][k] > 0] * scale * sum_z ws[z][b][k] -> bf16 (mask = the layer input, post ReLU and dropout);
// db[k] = sum_b dx[b][k] (of the bf16-rounded values: the bias gradient of the layer below), when db != nullptr.
// grid: K/32 blocks of 256 threads = 8 column quads x 32 row lanes; a thread owns four columns of the rows rl, rl + 32, ...
// (batch <= 128: at most four) and has all its loads in flight together.  K is a multiple of 4; larger batches take the
// rows in rounds of 128.
__global__ void __launch_bounds__(256) fc_reduce_bwd_kernel(const float* __restrict__ ws, int splits, long long split_stride,
                                                            const __nv_bfloat16* __restrict__ mask, float scale, int B, int K,
                                                            __nv_bfloat16* __restrict__ out, float* __restrict__ db) {
    pdl_sync();
    __shared__ float red[32][33];
    const int cq = threadIdx.x & 7, rl = threadIdx.x >> 3;
    const int c = blockIdx.x * 32 + 4 * cq;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    if (c < K) {
        for (int b0 = 0; b0 < B; b0 += 128) {
            float4 v[4];
            uint2 mk[4];
            #pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int b = b0 + rl + 32 * i;
                v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                mk[i] = make_uint2(0u, 0u);
                if (b < B) {
                    const size_t t = (size_t)b * K + c;
                    if (mask) mk[i] = __ldg((const uint2*)(mask + t));
                    for (int z = 0; z < splits; ++z) {
                        const float4 w = __ldg((const float4*)(ws + z * split_stride + t));
                        v[i].x += w.x; v[i].y += w.y; v[i].z += w.z; v[i].w += w.w;
                    }
                }
            }
            #pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int b = b0 + rl + 32 * i;
                if (b >= B) continue;
                float f[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
                if (mask) {
                    const __nv_bfloat162* m2 = (const __nv_bfloat162*)&mk[i];
                    const float2 ma = __bfloat1622float2(m2[0]), mb = __bfloat1622float2(m2[1]);
                    f[0] = ma.x > 0.f ? f[0] * scale : 0.f; f[1] = ma.y > 0.f ? f[1] * scale : 0.f;
                    f[2] = mb.x > 0.f ? f[2] * scale : 0.f; f[3] = mb.y > 0.f ? f[3] * scale : 0.f;
                }
                const __nv_bfloat162 lo = __floats2bfloat162_rn(f[0], f[1]), hi = __floats2bfloat162_rn(f[2], f[3]);
                *(uint2*)(out + (size_t)b * K + c) = make_uint2(*(const uint32_t*)&lo, *(const uint32_t*)&hi);
                const float2 ra = __bfloat1622float2(lo), rb = __bfloat1622float2(hi);
                acc[0] += ra.x; acc[1] += ra.y; acc[2] += rb.x; acc[3] += rb.y;
            }
        }
    }
    if (!db) return;
    #pragma unroll
    for (int k = 0; k < 4; ++k) red[rl][4 * cq + k] = acc[k];
    __syncthreads();
    if (threadIdx.x < 32 && blockIdx.x * 32 + threadIdx.x < K) {
        float s = 0.f;
        #pragma unroll
        for (int q = 0; q < 32; ++q) s += red[q][threadIdx.x];
        db[blockIdx.x * 32 + threadIdx.x] = s;
    }
}
// g[i] = sum_z ws[z][i]; conv1: entries of the 12x12 zero-padded filter outside 11x11 stay zero.
// The blocks from bias_block0 on add the bias-gradient partials, 32 groups of four channels each (cout is a multiple of 4).
// One entry per thread: with four entries per thread and 8 or 16 vectors in flight conv1, whose 41472 entries have up to 49 splits,
// has a quarter of the threads and takes 10 us more (weight gradient and reduction 51.5 -> 61.8 us at batch 128, 14.6 -> 22.8 at 8;
// conv2 59.1 -> 60.7; conv3 and conv4, hidden beside the data gradients, 41 -> 40).
__global__ void wgrad_reduce_kernel(const float* __restrict__ ws, int splits, long long split_stride,
                                    long long total, float* __restrict__ g, int conv1_pad_mask,
                                    const float* __restrict__ bias_partial, int bias_parts, int cout, float* __restrict__ db,
                                    int bias_block0) {
    pdl_sync();
    if ((int)blockIdx.x >= bias_block0) {
        const int c4 = ((int)blockIdx.x - bias_block0) * 32 + (threadIdx.x >> 3), k = threadIdx.x & 7;
        const bool in = 4 * c4 < cout;
        const float4 b = bias_sum8(bias_partial + (in ? 4 * c4 : 0), cout, bias_parts, k);
        if (in && k == 0) *(float4*)(db + 4 * c4) = b;
        return;
    }
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= total) return;
    float v = 0.f;
    for (int z = 0; z < splits; ++z) v += ws[z * split_stride + t];
    if (conv1_pad_mask) {
        const int ch = (int)(t % 48), tap = (int)(t / (48 * 96));
        const int ky = (tap / 3) * 4 + (ch / 3) / 4, kx = (tap % 3) * 4 + (ch / 3) % 4;
        if (ky > 10 || kx > 10) v = 0.f;
    }
    g[t] = v;
}

// db[c] = sum over rows of dy[row][c] (bf16 in, fp32 out), two stages: grid (ceil(C/64), row_splits)
// writes partial[split][C]; colsum_final_kernel adds the splits in a fixed order.
__global__ void colsum_kernel(const __nv_bfloat16* __restrict__ dy, long long rows, int C, float* __restrict__ partial) {
    pdl_sync();
    // block: 256 threads = 32 row-lanes x 8 column-chunks (8 channels each) -> 64 columns per block
    __shared__ float red[32][65];
    const int cc = threadIdx.x & 7, rl = threadIdx.x >> 3;
    const int c0 = blockIdx.x * 64 + cc * 8;
    const long long per = (rows + gridDim.y - 1) / gridDim.y;
    const long long r0 = (long long)blockIdx.y * per, r1 = min(rows, r0 + per);
    float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (c0 < C) {
        for (long long r = r0 + rl; r < r1; r += 32) {
            float f[8];
            unpack8(*(const uint4*)(dy + r * C + c0), f);
            #pragma unroll
            for (int i = 0; i < 8; ++i) acc[i] += f[i];
        }
    }
    #pragma unroll
    for (int i = 0; i < 8; ++i) red[rl][cc * 8 + i] = acc[i];
    __syncthreads();
    if (threadIdx.x < 64) {
        float s = 0.f;
        for (int r = 0; r < 32; ++r) s += red[r][threadIdx.x];
        const int c = blockIdx.x * 64 + threadIdx.x;
        if (c < C) partial[(size_t)blockIdx.y * C + c] = s;
    }
}
__global__ void colsum_final_kernel(const float* __restrict__ partial, int splits, int C, float* __restrict__ db) {
    pdl_sync();
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    float s = 0.f;
    for (int z = 0; z < splits; ++z) s += partial[(size_t)z * C + c];
    db[c] = s;
}
// same for a row pitch that is not a multiple of 8 elements (the 1000-wide logits gradient)
__global__ void colsum_scalar_kernel(const __nv_bfloat16* __restrict__ dy, int rows, int C, float* __restrict__ db) {
    pdl_sync();
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    float s = 0.f;
    for (int r = 0; r < rows; ++r) s += __bfloat162float(dy[(size_t)r * C + c]);
    db[c] = s;
}

// The same column sums in one launch, for the allocation-free entry point: grid (ceil(C/64), row splits), a block sums 64 columns of
// its rows (eight 16-byte loads of a thread in flight), and the block of a column group that finishes last adds the
// group's partials in a fixed order, so the result does not depend on which block that is.  A group counts its finished
// blocks in the low 16 bits of a word whose upper bits are the number of the launch: the first block of a launch sets the
// word to its number and a count of zero (a maximum: every later block of the launch leaves the count alone), so a launch
// owes nothing to what an earlier one left there, be it one that overlapped another or one that died.  HBM-bound (L2-bound
// where dy fits); what it spends beside that is the launch and the tail of the last block, whose loads of up to 160 partials go in one
// round.  Blocks of 256 threads and 64 registers, four to an SM, fit beside the tensor kernels of a training step, where this
// call belongs; one block of 1024 per SM waits for an SM to be empty.  Per call alone, 256 / 1024: 25088 x 384 5.97 / 6.27 us (several dy in turn 7.5 /
// 8.4), 60000 x 2048 40.5 / 40.9, 8000 x 104 5.5 / 5.5; beside a training handle of batch 32: 8000 x 104 23.5 / 38.2, 3000 x 384 24.1 / 37.1,
// 25088 x 384 34.2 / 38.1, 60000 x 2048 81 / 93, and the step beside them 0.5 to 1% shorter.
__global__ void __launch_bounds__(256, 4) bias_grad_kernel(const __nv_bfloat16* __restrict__ dy, long long rows, int C, float* __restrict__ partial,
                                                           unsigned long long* __restrict__ counters, unsigned long long launch,
                                                           float* __restrict__ db) {
    pdl_sync();
    constexpr int RL = 32, WARPS = 8, ZL = 16;       // lanes over the rows; over the splits in the tail
    __shared__ __align__(16) float red[WARPS][68];
    __shared__ bool last;
    const int tid = threadIdx.x, cc = tid & 7, rl = tid >> 3;
    const int c0 = blockIdx.x * 64 + cc * 8;
    const long long per = (rows + gridDim.y - 1) / gridDim.y;
    const long long r0 = (long long)blockIdx.y * per, r1 = min(rows, r0 + per);
    float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (c0 < C) {
        for (long long r = r0 + rl; r < r1; r += RL * 8) {
            uint4 u[8];
            #pragma unroll
            for (int q = 0; q < 8; ++q) {
                u[q] = make_uint4(0u, 0u, 0u, 0u);
                if (r + RL * q < r1) u[q] = __ldg((const uint4*)(dy + (r + RL * q) * C + c0));
            }
            #pragma unroll
            for (int q = 0; q < 8; ++q) {
                float f[8];
                unpack8(u[q], f);
                #pragma unroll
                for (int i = 0; i < 8; ++i) acc[i] += f[i];
            }
        }
    }
    #pragma unroll
    for (int i = 0; i < 8; ++i) {                // the four row lanes of a warp
        acc[i] += __shfl_xor_sync(~0u, acc[i], 8);
        acc[i] += __shfl_xor_sync(~0u, acc[i], 16);
    }
    if ((tid & 31) < 8) {
        #pragma unroll
        for (int i = 0; i < 8; ++i) red[tid >> 5][cc * 8 + i] = acc[i];
    }
    __syncthreads();
    const int splits = gridDim.y, c = blockIdx.x * 64 + tid;
    if (tid < 64 && c < C) {
        float s = 0.f;
        #pragma unroll
        for (int w = 0; w < WARPS; ++w) s += red[w][tid];
        if (splits == 1) db[c] = s;
        else partial[(size_t)blockIdx.y * C + c] = s;
    }
    if (splits == 1) return;
    __threadfence();
    __syncthreads();
    if (tid == 0) {
        atomicMax(counters + blockIdx.x, launch << 16);
        last = atomicAdd(counters + blockIdx.x, 1ull) == (launch << 16) + (unsigned)splits - 1u;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int q4 = tid & 15, zl = tid >> 4, cq = blockIdx.x * 64 + 4 * q4;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    if (cq < C && zl < splits) a = sum_splits<10>(partial + (size_t)zl * C + cq, (long long)ZL * C, (splits - zl + ZL - 1) / ZL);
    a.x += __shfl_xor_sync(~0u, a.x, 16); a.y += __shfl_xor_sync(~0u, a.y, 16);
    a.z += __shfl_xor_sync(~0u, a.z, 16); a.w += __shfl_xor_sync(~0u, a.w, 16);
    if ((tid & 31) < 16) *(float4*)&red[tid >> 5][4 * q4] = a;
    __syncthreads();
    if (tid < 64 && c < C) {
        float s = 0.f;
        #pragma unroll
        for (int w = 0; w < WARPS; ++w) s += red[w][tid];
        db[c] = s;
    }
}

// ------------------------------------------------------ softmax cross-entropy
// one block per sample: p = softmax(z), loss_n = -log p[label], dz = (p - onehot)/B as bf16
__global__ void softmax_xent_kernel(const float* __restrict__ z, const int32_t* __restrict__ labels,
                                    __nv_bfloat16* __restrict__ dz, float* __restrict__ loss_n, int B, int N) {
    pdl_sync();
    __shared__ float red[32];
    const int n = blockIdx.x, tid = threadIdx.x;
    const float* zr = z + (size_t)n * N;
    float mx = -INFINITY;
    for (int j = tid; j < N; j += blockDim.x) mx = fmaxf(mx, zr[j]);
    for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(~0u, mx, o));
    if ((tid & 31) == 0) red[tid >> 5] = mx;
    __syncthreads();
    mx = red[0];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) mx = fmaxf(mx, red[w]);
    __syncthreads();
    float sum = 0.f;
    for (int j = tid; j < N; j += blockDim.x) sum += expf(zr[j] - mx);
    for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(~0u, sum, o);
    if ((tid & 31) == 0) red[tid >> 5] = sum;
    __syncthreads();
    sum = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) sum += red[w];
    const int lab = labels[n];
    const float inv = 1.f / sum, invB = 1.f / (float)B;
    for (int j = tid; j < N; j += blockDim.x) {
        const float pj = expf(zr[j] - mx) * inv;
        dz[(size_t)n * N + j] = __float2bfloat16_rn((pj - (j == lab ? 1.f : 0.f)) * invB);
    }
    if (tid == 0) loss_n[n] = -(zr[lab] - mx - logf(sum));
}
// What a call that waits for the GPU reads: written by the last kernel of the call to mapped host memory, seq last, so that the
// host polls one word instead of queueing copies behind the kernels (two copies, a synchronisation and a third
// copy of the status word took 60 us of the 205 us of a one-image evaluation).
struct HostResult { int32_t top1, top5; float loss; int32_t status; uint32_t seq; };
__device__ __forceinline__ void publish_result(volatile HostResult* out, int top1, int top5, float loss, int status, uint32_t seq) {
    out->top1 = top1; out->top5 = top5; out->loss = loss; out->status = status;
    __threadfence_system();
    out->seq = seq;
}
__global__ void store_result_kernel(const float* __restrict__ loss, const int* __restrict__ status, HostResult* out, uint32_t seq) {
    pdl_sync();
    publish_result(out, 0, 0, *loss, *(volatile const int*)status, seq);
}
// The training step's form of the three kernels fc_reduce_fwd (fc8), softmax_xent and mean in one launch: block n adds the
// split-K partials of its row of logits in split order, adds the bias, stores z (fp32 logits), then softmax, loss_n and dz as
// above; the block that finishes last (a counter in global memory, reset for the next launch) averages loss_n in index order,
// so the result does not depend on which block that is.  Same arithmetic as the separate kernels.
// EVAL: also counts the samples whose label is among the top 1 / top 5 logits (rank of the label = logits strictly greater than
// it plus equal logits with a smaller class index; integer atomics, so the order does not matter) and the last block
// publishes the counts, the loss and the status word.
template <bool EVAL>
__global__ void __launch_bounds__(256) fc8_softmax_xent_kernel(const float* __restrict__ ws, int splits, long long split_stride,
                                                               const float* __restrict__ bias, float* __restrict__ z,
                                                               const int32_t* __restrict__ labels, __nv_bfloat16* __restrict__ dz,
                                                               float* __restrict__ loss_n, float* __restrict__ loss_mean,
                                                               int* __restrict__ done_counter, int B, int N,
                                                               int32_t* __restrict__ counts, const int* __restrict__ status,
                                                               HostResult* host_out, uint32_t seq) {
    pdl_trigger();
    // the bias and the labels are fetched while the predecessor runs: whatever wrote them (the update of the step before; the loader,
    // or in an evaluation the preprocessing kernel of this very stream and pass) has completed, because lrn_pool_fwd_kernel, between it
    // and this kernel, lets no later launch start before it has itself waited
    const int lab = labels[blockIdx.x];
    float4 b4 = make_float4(0.f, 0.f, 0.f, 0.f);
    if ((N & 3) == 0 && 4 * (int)threadIdx.x < N) b4 = __ldg((const float4*)bias + threadIdx.x);
    pdl_wait();
    __shared__ float red[32];
    __shared__ __align__(16) float zs[1024];
    __shared__ int last;
    const int n = blockIdx.x, tid = threadIdx.x;
    float mx = -INFINITY;
    if ((N & 3) == 0) {
        // four columns per thread, the loads of all splits in flight together (the maximum does not depend on which thread
        // sees which column; the sums below keep the column -> thread mapping of softmax_xent_kernel)
        for (int j = 4 * tid; j < N; j += 1024) {
            const long long t = (long long)n * N + j;
            if (j >= 1024) b4 = __ldg((const float4*)(bias + j));
            float4 v = sum_splits<16>(ws + t, split_stride, splits);
            v.x += b4.x; v.y += b4.y; v.z += b4.z; v.w += b4.w;
            *(float4*)(z + t) = v;
            *(float4*)(zs + j) = v;
            mx = fmaxf(fmaxf(mx, fmaxf(v.x, v.y)), fmaxf(v.z, v.w));
        }
    } else {
        for (int j = tid; j < N; j += 256) {
            const long long t = (long long)n * N + j;
            float v = 0.f;
            for (int q = 0; q < splits; ++q) v += ws[q * split_stride + t];
            v += bias[j];
            z[t] = v;
            zs[j] = v;
            mx = fmaxf(mx, v);
        }
    }
    for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(~0u, mx, o));
    if ((tid & 31) == 0) red[tid >> 5] = mx;
    __syncthreads();
    mx = red[0];
    for (int w = 1; w < 8; ++w) mx = fmaxf(mx, red[w]);
    __syncthreads();
    float sum = 0.f;
    for (int j = tid; j < N; j += 256) sum += expf(zs[j] - mx);
    for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(~0u, sum, o);
    if ((tid & 31) == 0) red[tid >> 5] = sum;
    __syncthreads();
    sum = 0.f;
    for (int w = 0; w < 8; ++w) sum += red[w];
    const float inv = 1.f / sum, invB = 1.f / (float)B;
    for (int j = tid; j < N; j += 256) {
        const float pj = expf(zs[j] - mx) * inv;
        dz[(size_t)n * N + j] = __float2bfloat16_rn((pj - (j == lab ? 1.f : 0.f)) * invB);
    }
    int top1 = 0, top5 = 0;
    if (EVAL) {
        const float zl = zs[lab];
        int c = 0;
        for (int j = tid; j < N; j += 256) c += (zs[j] > zl) || (zs[j] == zl && j < lab);
        const int rank = __reduce_add_sync(~0u, c);
        __syncthreads();
        if ((tid & 31) == 0) red[tid >> 5] = __int_as_float(rank);
        __syncthreads();
        if (tid == 0) {
            int k = 0;
            for (int w = 0; w < 8; ++w) k += __float_as_int(red[w]);
            if (B == 1) {         // nobody to wait for: no counters
                top1 = k < 1; top5 = k < 5;
            } else {
                if (k < 1) atomicAdd(counts, 1);
                if (k < 5) atomicAdd(counts + 1, 1);
            }
        }
    }
    if (B == 1) {
        if (tid == 0) {
            const float t = -(zs[lab] - mx - logf(sum));
            loss_n[0] = t;
            *loss_mean = t;
            if (EVAL) publish_result(host_out, top1, top5, t, *(volatile const int*)status, seq);
        }
        return;
    }
    if (tid == 0) {
        loss_n[n] = -(zs[lab] - mx - logf(sum));
        __threadfence();
        last = atomicAdd(done_counter, 1) == B - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    float s = 0.f;
    for (int i = tid; i < B; i += 256) s += __ldcg(loss_n + i);
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(~0u, s, o);
    __syncthreads();
    if ((tid & 31) == 0) red[tid >> 5] = s;
    __syncthreads();
    if (tid == 0) {
        float t = 0.f;
        for (int w = 0; w < 8; ++w) t += red[w];
        *loss_mean = t / (float)B;
        *done_counter = 0;
        if (EVAL) {
            const int t1 = atomicExch(counts, 0), t5 = atomicExch(counts + 1, 0);      // zero again for the next call
            publish_result(host_out, t1, t5, t / (float)B, *(volatile const int*)status, seq);
        }
    }
}
// one float to wherever dst points (device memory, or pinned host memory mapped into the device's address space): the
// loss read-back without a copy engine, whose queue a batch upload of 25 MB may occupy; NaN once a bounded wait has expired, since a
// loop that reads nothing but its losses has no other sign that the values behind them are wrong
__global__ void store_value_kernel(const float* __restrict__ src, const int* __restrict__ status, float* __restrict__ dst) {
    pdl_sync();
    *dst = *(volatile const int*)status ? __int_as_float(0x7fc00000) : *src;
}
__global__ void mean_kernel(const float* __restrict__ v, int n, float* __restrict__ out) {
    pdl_sync();
    __shared__ float red[32];
    float s = 0.f;
    for (int i = threadIdx.x; i < n; i += blockDim.x) s += v[i];
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(~0u, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
        *out = t / (float)n;
    }
}

// ------------------------------------------------ momentum update and average
// transposed bf16 copies of the grouped conv filters for the backward-data pass:
// wt[tap][g*cig + ci][co'] = wf[tap][g*cog + co'][ci]
struct TransposeJob { long long src_off, dst_off; int taps, cout, cig, groups; long long count; };
struct TransposeJobs { TransposeJob j[5]; int n; int tile0[6]; };   // tile0: first 32 x 32 tile of each job in sgd_update_conv_kernel's grid
// one parameter of the momentum update: v <- mu v - d w - lr g (d = lr * weight decay, or 0); w <- w + v.
// Used by the update kernels and by fc_update_kernel, which applies the update to the FC weights in place, so that both
// give bit-identical results.
__device__ __forceinline__ void sgd_step(float& w, float& v, float g, float d, float lr, float mu) {
    v = fmaf(mu, v, fmaf(-d, w, -lr * g));
    w += v;
}
// v <- mu v - lr wd w [i < n_decay] - lr g ; w <- w + v ; bf16 shadow of w.  22 bytes per parameter.
// Updates the 16-byte vectors [begin4, n4) of the internal order: everything after the conv filters (which
// sgd_update_conv_kernel takes), or only the biases when the FC weight-gradient kernel has already updated the FC weights.
// gscale multiplies the gradient first (1 for a single replica: exact; 1/R for a gradient summed over R replicas).
__global__ void sgd_update_kernel(float* __restrict__ w, float* __restrict__ v, const float* __restrict__ g,
                                  __nv_bfloat16* __restrict__ shadow, long long begin4, long long n4, long long n_decay4,
                                  float lr, float mu, float wd, float gscale) {
    pdl_sync();
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = begin4 + (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += stride) {
        float4 wv = ((float4*)w)[i], vv = ((float4*)v)[i];
        const float4 gv = ((const float4*)g)[i];
        const float d = i < n_decay4 ? lr * wd : 0.f;
        sgd_step(wv.x, vv.x, gscale * gv.x, d, lr, mu);
        sgd_step(wv.y, vv.y, gscale * gv.y, d, lr, mu);
        sgd_step(wv.z, vv.z, gscale * gv.z, d, lr, mu);
        sgd_step(wv.w, vv.w, gscale * gv.w, d, lr, mu);
        ((float4*)w)[i] = wv;
        ((float4*)v)[i] = vv;
        __nv_bfloat162 lo2 = __floats2bfloat162_rn(wv.x, wv.y), hi2 = __floats2bfloat162_rn(wv.z, wv.w);
        ((uint2*)shadow)[i] = make_uint2(*(uint32_t*)&lo2, *(uint32_t*)&hi2);
    }
}
// The same update for the conv filters, tiled so that the transposed bf16 copies are written in runs: one block = one tap,
// 32 output channels and 32 input channels of one layer.  Thread (r, c4) updates the four consecutive input channels
// 4*c4 .. 4*c4+3 of output channel r (the source order [tap][cout][cig]: 128-byte runs per row), the bf16 values cross a
// shared-memory tile, and thread (ci, q) writes four consecutive output channels of input channel ci to the transposed copy
// [tap][cin][cog] (64-byte runs; a thread that walked the source order would write single elements).  Same arithmetic as sgd_update_kernel.
// With src.on the kernel also forms the conv gradients it consumes: the weight-gradient kernels leave fp32 partials per row
// split (and bias-gradient partials), and instead of a reduction launch per layer the update adds them here, in split
// order and with conv1's pad entries zeroed - wgrad_reduce_kernel's arithmetic - and stores the sums to g as that kernel does.
struct ConvSplitSrc {
    int on;
    int splits[5], bparts[5], cout[5];
    const float* ws[5]; long long stride[5];       // layer l: ws[l][z * stride[l] + index within the layer's filters]
    const float* bpart[5]; long long b_off4[5];    // bias partials [bparts][cout]; first 16-byte vector of the layer's biases
};
__global__ void __launch_bounds__(256) sgd_update_conv_kernel(float* __restrict__ w, float* __restrict__ v, float* __restrict__ g,
                                                              __nv_bfloat16* __restrict__ shadow, float d, float lr, float mu,
                                                              __nv_bfloat16* __restrict__ wt, const TransposeJobs jobs, float gscale,
                                                              int bias_blocks, long long tail_begin4, long long tail_end4,
                                                              float tail_d, const ConvSplitSrc src) {
    pdl_sync();
    __shared__ __nv_bfloat16 tile[32][36];       // [input channel][output channel], padded
    const int tile_block = (int)blockIdx.x - bias_blocks;
    if (tile_block < 0) {
        // blocks before the filter tiles (they have the longest sums): the plain update of the 16-byte vectors
        // [tail_begin4, tail_end4) (the biases, when the FC weights have been updated by their weight-gradient kernels),
        // sgd_update_kernel's arithmetic, one launch less.  Eight lanes per vector, for the conv layers' sums.
        const long long i = tail_begin4 + (long long)blockIdx.x * 32 + (threadIdx.x >> 3);
        const int k = threadIdx.x & 7;
        int lb = -1;
        if (src.on) {
            #pragma unroll
            for (int l = 0; l < 5; ++l)
                if (i >= src.b_off4[l] && i < src.b_off4[l] + src.cout[l] / 4) lb = l;
        }
        // a conv layer's bias gradient from its partials (the lanes of a warp may belong to different layers: all of them add)
        float4 gv = make_float4(0.f, 0.f, 0.f, 0.f);
        if (src.on) {
            const float* bp = lb >= 0 ? src.bpart[lb] + 4 * (i - src.b_off4[lb]) : src.bpart[0];
            gv = bias_sum8(bp, lb >= 0 ? src.cout[lb] : 0, lb >= 0 ? src.bparts[lb] : 0, k);
        }
        if (i < tail_end4 && k == 0) {
            float4 wv = ((float4*)w)[i], vv = ((float4*)v)[i];
            if (lb >= 0) ((float4*)g)[i] = gv;
            else gv = ((const float4*)g)[i];
            sgd_step(wv.x, vv.x, gscale * gv.x, tail_d, lr, mu);
            sgd_step(wv.y, vv.y, gscale * gv.y, tail_d, lr, mu);
            sgd_step(wv.z, vv.z, gscale * gv.z, tail_d, lr, mu);
            sgd_step(wv.w, vv.w, gscale * gv.w, tail_d, lr, mu);
            ((float4*)w)[i] = wv;
            ((float4*)v)[i] = vv;
            __nv_bfloat162 lo2 = __floats2bfloat162_rn(wv.x, wv.y), hi2 = __floats2bfloat162_rn(wv.z, wv.w);
            ((uint2*)shadow)[i] = make_uint2(*(uint32_t*)&lo2, *(uint32_t*)&hi2);
        }
        return;
    }
    int q = 0;
    while (q + 1 < jobs.n && tile_block >= jobs.tile0[q + 1]) ++q;
    const TransposeJob J = jobs.j[q];
    const int cog = J.cout / J.groups;
    const int ci_blocks = (J.cig + 31) / 32, co_blocks = J.cout / 32;     // cout is a multiple of 32 in every layer
    int t = tile_block - jobs.tile0[q];
    const int cib = t % ci_blocks; t /= ci_blocks;
    const int cob = t % co_blocks, tap = t / co_blocks;
    const int r = threadIdx.x >> 3, c4 = threadIdx.x & 7;
    const int co = cob * 32 + r, ci = cib * 32 + 4 * c4;
    if (ci < J.cig) {                            // cig is a multiple of 4
        const long long e = J.src_off + ((long long)tap * J.cout + co) * J.cig + ci;
        float4 wv = *(float4*)(w + e), vv = *(float4*)(v + e);
        float4 gv;
        if (src.on) {
            const long long t = e - J.src_off;
            gv = sum_splits<8>(src.ws[q] + t, src.stride[q], src.splits[q]);
            if (q == 0) {                        // conv1: entries of the 12 x 12 zero-padded filter outside 11 x 11 stay zero
                float* gp = &gv.x;
                #pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int ch = (int)((t + k) % 48), tp = (int)((t + k) / (48 * 96));
                    const int ky = (tp / 3) * 4 + (ch / 3) / 4, kx = (tp % 3) * 4 + (ch / 3) % 4;
                    if (ky > 10 || kx > 10) gp[k] = 0.f;
                }
            }
            *(float4*)(g + e) = gv;
        } else {
            gv = *(const float4*)(g + e);
        }
        sgd_step(wv.x, vv.x, gscale * gv.x, d, lr, mu);
        sgd_step(wv.y, vv.y, gscale * gv.y, d, lr, mu);
        sgd_step(wv.z, vv.z, gscale * gv.z, d, lr, mu);
        sgd_step(wv.w, vv.w, gscale * gv.w, d, lr, mu);
        *(float4*)(w + e) = wv;
        *(float4*)(v + e) = vv;
        const __nv_bfloat162 lo2 = __floats2bfloat162_rn(wv.x, wv.y), hi2 = __floats2bfloat162_rn(wv.z, wv.w);
        *(uint2*)(shadow + e) = make_uint2(*(const uint32_t*)&lo2, *(const uint32_t*)&hi2);
        tile[4 * c4][r] = lo2.x; tile[4 * c4 + 1][r] = lo2.y; tile[4 * c4 + 2][r] = hi2.x; tile[4 * c4 + 3][r] = hi2.y;
    }
    __syncthreads();
    const int ci2 = cib * 32 + r, cq = 4 * c4;   // now: thread (input channel r of the tile, four output channels from cq)
    if (ci2 < J.cig) {
        const int co0 = cob * 32 + cq, grp = co0 / cog, col = co0 - grp * cog;
        __nv_bfloat16* dst = wt + J.dst_off + ((long long)tap * J.cig * J.groups + grp * J.cig + ci2) * cog + col;
        const __nv_bfloat162 a = __halves2bfloat162(tile[r][cq], tile[r][cq + 1]), b = __halves2bfloat162(tile[r][cq + 2], tile[r][cq + 3]);
        *(uint2*)dst = make_uint2(*(const uint32_t*)&a, *(const uint32_t*)&b);
    }
}
// exchange-and-average with both replicas in one HBM: w_a = w_b = (w_a+w_b)/2, same for momentum; refresh both shadows.
__global__ void replica_average_kernel(float* __restrict__ wa, float* __restrict__ wb, float* __restrict__ va,
                                       float* __restrict__ vb, __nv_bfloat16* __restrict__ sa,
                                       __nv_bfloat16* __restrict__ sb, long long n4) {
    pdl_sync();
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += stride) {
        const float4 a = ((float4*)wa)[i], b = ((float4*)wb)[i];
        const float4 c = ((float4*)va)[i], d = ((float4*)vb)[i];
        const float4 w = make_float4(0.5f * (a.x + b.x), 0.5f * (a.y + b.y), 0.5f * (a.z + b.z), 0.5f * (a.w + b.w));
        const float4 v = make_float4(0.5f * (c.x + d.x), 0.5f * (c.y + d.y), 0.5f * (c.z + d.z), 0.5f * (c.w + d.w));
        ((float4*)wa)[i] = w; ((float4*)wb)[i] = w;
        ((float4*)va)[i] = v; ((float4*)vb)[i] = v;
        __nv_bfloat162 lo = __floats2bfloat162_rn(w.x, w.y), hi = __floats2bfloat162_rn(w.z, w.w);
        const uint2 s = make_uint2(*(uint32_t*)&lo, *(uint32_t*)&hi);
        ((uint2*)sa)[i] = s; ((uint2*)sb)[i] = s;
    }
}
// Momentum update of two replicas and their exchange-and-average in one pass: each replica's own (w, v, g) goes through
// sgd_step (the update kernels' arithmetic), then w and v of both are replaced by 0.5 * (a + b) (replica_average_kernel's
// arithmetic) and both bf16 copies are written: six 16-byte loads and six stores per four parameter indices, 44 bytes per
// index, against 22 + 22 + 36 for the three separate passes, with bit-identical results.
__device__ __forceinline__ float4 ld_stream(const float* p) {       // read once, do not keep in L1
    float4 r;
    asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w) : "l"(p));
    return r;
}
__global__ void __launch_bounds__(256) sgd_update_average_kernel(float* __restrict__ wa, float* __restrict__ va, const float* __restrict__ ga,
                                                                 float* __restrict__ wb, float* __restrict__ vb, const float* __restrict__ gb,
                                                                 __nv_bfloat16* __restrict__ sa, __nv_bfloat16* __restrict__ sb,
                                                                 long long n4, long long n_decay4, float lr, float mu, float wd) {
    pdl_sync();
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += stride) {
        float4 a = ((const float4*)wa)[i], c = ((const float4*)va)[i];
        float4 b = ((const float4*)wb)[i], e = ((const float4*)vb)[i];
        const float4 g0 = ld_stream(ga + 4 * i), g1 = ld_stream(gb + 4 * i);
        const float d = i < n_decay4 ? lr * wd : 0.f;
        sgd_step(a.x, c.x, g0.x, d, lr, mu); sgd_step(a.y, c.y, g0.y, d, lr, mu);
        sgd_step(a.z, c.z, g0.z, d, lr, mu); sgd_step(a.w, c.w, g0.w, d, lr, mu);
        sgd_step(b.x, e.x, g1.x, d, lr, mu); sgd_step(b.y, e.y, g1.y, d, lr, mu);
        sgd_step(b.z, e.z, g1.z, d, lr, mu); sgd_step(b.w, e.w, g1.w, d, lr, mu);
        const float4 w = make_float4(0.5f * (a.x + b.x), 0.5f * (a.y + b.y), 0.5f * (a.z + b.z), 0.5f * (a.w + b.w));
        const float4 v = make_float4(0.5f * (c.x + e.x), 0.5f * (c.y + e.y), 0.5f * (c.z + e.z), 0.5f * (c.w + e.w));
        ((float4*)wa)[i] = w; ((float4*)wb)[i] = w;
        ((float4*)va)[i] = v; ((float4*)vb)[i] = v;
        __nv_bfloat162 lo = __floats2bfloat162_rn(w.x, w.y), hi = __floats2bfloat162_rn(w.z, w.w);
        const uint2 s = make_uint2(*(uint32_t*)&lo, *(uint32_t*)&hi);
        ((uint2*)sa)[i] = s; ((uint2*)sb)[i] = s;
    }
}
// The same for two replicas that SHARE one copy of parameters and momentum (they are identical at the start of every
// iteration: identical initialisation, and every exchange makes them equal again, so one copy holds both): each replica's
// update starts from the shared (w, v) with its own gradient, the averages go back to the shared arrays.  Same arithmetic in
// the same order as above, hence the same bits; 16 bytes read and 10 written per index (26 instead of 44).
__global__ void __launch_bounds__(256) sgd_update_average_shared_kernel(float* __restrict__ w, float* __restrict__ v, const float* __restrict__ ga,
                                                                        const float* __restrict__ gb, __nv_bfloat16* __restrict__ shadow,
                                                                        long long n4, long long n_decay4, float lr, float mu, float wd) {
    pdl_sync();
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += stride) {
        float4 a = ((const float4*)w)[i], c = ((const float4*)v)[i];
        float4 b = a, e = c;
        const float4 g0 = ld_stream(ga + 4 * i), g1 = ld_stream(gb + 4 * i);
        const float d = i < n_decay4 ? lr * wd : 0.f;
        sgd_step(a.x, c.x, g0.x, d, lr, mu); sgd_step(a.y, c.y, g0.y, d, lr, mu);
        sgd_step(a.z, c.z, g0.z, d, lr, mu); sgd_step(a.w, c.w, g0.w, d, lr, mu);
        sgd_step(b.x, e.x, g1.x, d, lr, mu); sgd_step(b.y, e.y, g1.y, d, lr, mu);
        sgd_step(b.z, e.z, g1.z, d, lr, mu); sgd_step(b.w, e.w, g1.w, d, lr, mu);
        const float4 wn = make_float4(0.5f * (a.x + b.x), 0.5f * (a.y + b.y), 0.5f * (a.z + b.z), 0.5f * (a.w + b.w));
        const float4 vn = make_float4(0.5f * (c.x + e.x), 0.5f * (c.y + e.y), 0.5f * (c.z + e.z), 0.5f * (c.w + e.w));
        ((float4*)w)[i] = wn; ((float4*)v)[i] = vn;
        __nv_bfloat162 lo = __floats2bfloat162_rn(wn.x, wn.y), hi = __floats2bfloat162_rn(wn.z, wn.w);
        ((uint2*)shadow)[i] = make_uint2(*(uint32_t*)&lo, *(uint32_t*)&hi);
    }
}
// After an all-reduce(sum) of parameters and momentum over R replicas on R GPUs: w <- scale w, v <- scale v (scale = 1/R:
// the average) and the bf16 copy of w: 8 bytes read and 10 written per index.
__global__ void __launch_bounds__(256) scale_refresh_kernel(float* __restrict__ w, float* __restrict__ v,
                                                            __nv_bfloat16* __restrict__ shadow, long long n4, float scale) {
    pdl_sync();
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += stride) {
        float4 a = ((const float4*)w)[i], c = ((const float4*)v)[i];
        a.x *= scale; a.y *= scale; a.z *= scale; a.w *= scale;
        c.x *= scale; c.y *= scale; c.z *= scale; c.w *= scale;
        ((float4*)w)[i] = a; ((float4*)v)[i] = c;
        __nv_bfloat162 lo = __floats2bfloat162_rn(a.x, a.y), hi = __floats2bfloat162_rn(a.z, a.w);
        ((uint2*)shadow)[i] = make_uint2(*(uint32_t*)&lo, *(uint32_t*)&hi);
    }
}
// The paper's own form of the exchange ("Data parallelism" figure, steps 2 and 3): every replica has RECEIVED the other
// replicas' parameters and momenta into buffers of its own GPU (peer copies or an all-gather: the caller's) and now averages.
// slot[r] = the arrays of the replica of rank r in rank order, the local replica's own arrays at r = self (so every rank adds
// in the same order and all ranks end bit-identical); w, v = the local arrays, overwritten; also writes the bf16 copy.
struct RecvList { const float* w[8]; const float* v[8]; int count; };
__global__ void __launch_bounds__(256) average_received_kernel(float* __restrict__ w, float* __restrict__ v, __nv_bfloat16* __restrict__ shadow,
                                                               const RecvList rl, long long n4, float inv_count) {
    pdl_sync();
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += stride) {
        float4 a = ((const float4*)rl.w[0])[i], c = ((const float4*)rl.v[0])[i];
        #pragma unroll 1
        for (int r = 1; r < rl.count; ++r) {
            const float4 b = ((const float4*)rl.w[r])[i], d = ((const float4*)rl.v[r])[i];
            a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
            c.x += d.x; c.y += d.y; c.z += d.z; c.w += d.w;
        }
        a.x *= inv_count; a.y *= inv_count; a.z *= inv_count; a.w *= inv_count;
        c.x *= inv_count; c.y *= inv_count; c.z *= inv_count; c.w *= inv_count;
        ((float4*)w)[i] = a; ((float4*)v)[i] = c;
        __nv_bfloat162 lo = __floats2bfloat162_rn(a.x, a.y), hi = __floats2bfloat162_rn(a.z, a.w);
        ((uint2*)shadow)[i] = make_uint2(*(uint32_t*)&lo, *(uint32_t*)&hi);
    }
}
__global__ void shadow_kernel(const float* __restrict__ w, __nv_bfloat16* __restrict__ shadow, long long n4) {
    pdl_sync();
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += stride) {
        const float4 wv = ((const float4*)w)[i];
        __nv_bfloat162 lo = __floats2bfloat162_rn(wv.x, wv.y), hi = __floats2bfloat162_rn(wv.z, wv.w);
        ((uint2*)shadow)[i] = make_uint2(*(uint32_t*)&lo, *(uint32_t*)&hi);
    }
}

// Transposed bf16 copies of the conv filters from the bf16 copy of the weights, in the 32 x 32 tiles of
// sgd_update_conv_kernel (8-byte reads along the input channels, 8-byte writes along the output channels through a
// shared-memory tile); wt2 != nullptr: a second destination (the other replica's copy after an average, when both are equal).
__global__ void __launch_bounds__(256) conv_transpose_shadow_kernel(const __nv_bfloat16* __restrict__ shadow, __nv_bfloat16* __restrict__ wt,
                                                                    __nv_bfloat16* __restrict__ wt2, const TransposeJobs jobs) {
    pdl_sync();
    __shared__ __nv_bfloat16 tile[32][36];       // [input channel][output channel], padded
    int q = 0;
    while (q + 1 < jobs.n && (int)blockIdx.x >= jobs.tile0[q + 1]) ++q;
    const TransposeJob J = jobs.j[q];
    const int cog = J.cout / J.groups;
    const int ci_blocks = (J.cig + 31) / 32, co_blocks = J.cout / 32;
    int t = (int)blockIdx.x - jobs.tile0[q];
    const int cib = t % ci_blocks; t /= ci_blocks;
    const int cob = t % co_blocks, tap = t / co_blocks;
    const int r = threadIdx.x >> 3, c4 = threadIdx.x & 7;
    const int co = cob * 32 + r, ci = cib * 32 + 4 * c4;
    if (ci < J.cig) {                            // cig is a multiple of 4
        const uint2 u = *(const uint2*)(shadow + J.src_off + ((long long)tap * J.cout + co) * J.cig + ci);
        const __nv_bfloat162 lo2 = *(const __nv_bfloat162*)&u.x, hi2 = *(const __nv_bfloat162*)&u.y;
        tile[4 * c4][r] = lo2.x; tile[4 * c4 + 1][r] = lo2.y; tile[4 * c4 + 2][r] = hi2.x; tile[4 * c4 + 3][r] = hi2.y;
    }
    __syncthreads();
    const int ci2 = cib * 32 + r, cq = 4 * c4;   // now: thread (input channel r of the tile, four output channels from cq)
    if (ci2 < J.cig) {
        const int co0 = cob * 32 + cq, grp = co0 / cog, col = co0 - grp * cog;
        const long long d = J.dst_off + ((long long)tap * J.cig * J.groups + grp * J.cig + ci2) * cog + col;
        const __nv_bfloat162 a = __halves2bfloat162(tile[r][cq], tile[r][cq + 1]), b2 = __halves2bfloat162(tile[r][cq + 2], tile[r][cq + 3]);
        const uint2 o = make_uint2(*(const uint32_t*)&a, *(const uint32_t*)&b2);
        *(uint2*)(wt + d) = o;
        if (wt2) *(uint2*)(wt2 + d) = o;
    }
}

// ------------------------------------------- canonical <-> internal parameter order
struct ParamSeg { long long canon_off, int_off, count; int kind, a, b, c; };  // kind 0 copy, 1 conv [co][ci][k][k], 2 conv1 s2d, 3 fc6
struct ParamSegs { ParamSeg s[16]; };
__device__ __forceinline__ long long canon_to_internal(const ParamSeg& S, long long i) {
    if (S.kind == 0) return S.int_off + i;
    if (S.kind == 1) {          // a = cout, b = cig, c = k : canonical ((co*cig+ci)*k+ky)*k+kx -> (tap*cout+co)*cig+ci
        const int kk2 = S.c * S.c;
        const int tap = (int)(i % kk2);
        long long r = i / kk2;
        const int ci = (int)(r % S.b), co = (int)(r / S.b);
        return S.int_off + ((long long)tap * S.a + co) * S.b + ci;
    }
    if (S.kind == 2) {          // conv1: [96][3][11][11] -> [tap 3x3][96][48], channel ((ky%4)*4 + kx%4)*3 + c
        const int kx = (int)(i % 11), ky = (int)((i / 11) % 11), c = (int)((i / 121) % 3), co = (int)(i / 363);
        const int tap = (ky >> 2) * 3 + (kx >> 2), ch = ((ky & 3) * 4 + (kx & 3)) * 3 + c;
        return S.int_off + ((long long)tap * 96 + co) * 48 + ch;
    }
    // fc6: [4096][c*36 + hw] -> [4096][hw*256 + c]
    const int k = (int)(i % 9216), n = (int)(i / 9216);
    return S.int_off + (long long)n * 9216 + (k % 36) * 256 + k / 36;
}
__global__ void params_gather_kernel(const float* __restrict__ arena, float* __restrict__ canon, const ParamSegs segs,
                                     long long total) {
    pdl_sync();
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += stride) {
        int s = 0;
        while (s < 15 && i >= segs.s[s + 1].canon_off) ++s;
        canon[i] = arena[canon_to_internal(segs.s[s], i - segs.s[s].canon_off)];
    }
}
__global__ void params_scatter_kernel(float* __restrict__ arena, const float* __restrict__ canon, const ParamSegs segs,
                                      long long total) {
    pdl_sync();
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += stride) {
        int s = 0;
        while (s < 15 && i >= segs.s[s + 1].canon_off) ++s;
        arena[canon_to_internal(segs.s[s], i - segs.s[s].canon_off)] = canon[i];
    }
}

}  // namespace kn
