// Stand-alone quantizers: activation rows (Q_a of Eq. 2) and weight packing (W8 / W4 per output channel).
// Integer codes are compared bit for bit with the CPU definition, so every floating-point step here is an
// explicit IEEE binary32 operation (__fdiv_rn, rintf); nothing may be contracted or approximated.
#include "taq_common.cuh"
#include "taq_ptx.cuh"

namespace taq {

__device__ inline float warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// One warp per row.  Memory-bound: the row is read twice (absmax, then codes); the second read hits L1/L2.
__global__ void __launch_bounds__(256) quantize_rows_kernel(const float* __restrict__ x, long long rows, int cols, int qmax,
                                                            int8_t* __restrict__ codes, float* __restrict__ scales) {
    const int lane = threadIdx.x & 31;
    const long long warps_total = (long long)gridDim.x * (blockDim.x >> 5);
    for (long long r = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < rows; r += warps_total) {
        const float* xr = x + r * cols;
        float a = 0.f;
        if ((cols & 3) == 0) {
            const float4* x4 = reinterpret_cast<const float4*>(xr);
            for (int i = lane; i < cols / 4; i += 32) {
                float4 v = x4[i];
                a = fmaxf(a, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
            }
        } else {
            for (int i = lane; i < cols; i += 32) a = fmaxf(a, fabsf(xr[i]));
        }
        a = warp_max(a);
        const float s = quant_scale(a, (float)qmax);
        if (lane == 0) scales[r] = s;
        int8_t* cr = codes + r * cols;
        if ((cols & 3) == 0) {
            const float4* x4 = reinterpret_cast<const float4*>(xr);
            char4* c4 = reinterpret_cast<char4*>(cr);
            for (int i = lane; i < cols / 4; i += 32) {
                float4 v = x4[i];
                c4[i] = make_char4((signed char)quant_code(v.x, s, qmax), (signed char)quant_code(v.y, s, qmax),
                                   (signed char)quant_code(v.z, s, qmax), (signed char)quant_code(v.w, s, qmax));
            }
        } else {
            for (int i = lane; i < cols; i += 32) cr[i] = (int8_t)quant_code(xr[i], s, qmax);
        }
    }
}

cudaError_t launch_quantize_rows(const float* x, long long rows, int cols, int qmax, int8_t* codes, float* scales,
                                 cudaStream_t stream) {
    if (rows == 0) return cudaSuccess;
    long long blocks = (rows + 7) / 8;
    if (blocks > 148LL * 32) blocks = 148LL * 32;   // grid-stride beyond 32 resident waves
    quantize_rows_kernel<<<(unsigned)blocks, 256, 0, stream>>>(x, rows, cols, qmax, codes, scales);
    return cudaGetLastError();
}

// rint(x / s) clamped to +-127, bit-identical to quant_code (one IEEE division, then rintf) at a fraction of its cost.
// fma(x, r, 1.5 * 2^23) leaves rint(x r) in the low bits.  The rounded quotient fl(x / s) and the product with the
// correctly rounded reciprocal both lie between x r_lo and x r_hi (r two ulps down and up), so when both ends round to
// the same integer that integer is the code; only otherwise the division decides.
__device__ __noinline__ int code_127_by_division(float x, float s) { return (int)fminf(fmaxf(rintf(__fdiv_rn(x, s)), -127.f), 127.f); }
__device__ __forceinline__ int quant_code_127(float x, float s, float r_lo, float r_hi) {
    const uint32_t a = __float_as_uint(fmaf(x, r_lo, 12582912.0f)), c = __float_as_uint(fmaf(x, r_hi, 12582912.0f));
    if (a != c) return code_127_by_division(x, s);     // (fp16 data: about 4 values in 10000, e.g. exactly half of the row maximum)
    return (int)(a << 24) >> 24;                       // the low byte, sign-extended
}
// The same for eight fp16 values with one test for all of them: with a branch per value 8192 x 640 values took 9.5 us, now 4.9;
// 64 x 1280, a launch of one wave, 2.9 -> 2.4 (values in L2; from HBM 6.1 and 2.8).
__device__ __noinline__ uint2 codes8_by_division(uint4 v, float s) {
    const __half* h = reinterpret_cast<const __half*>(&v);
    uint32_t w[2] = {0, 0};
#pragma unroll
    for (int e = 0; e < 8; ++e) w[e >> 2] |= (uint32_t)((int)fminf(fmaxf(rintf(__fdiv_rn(__half2float(h[e]), s)), -127.f), 127.f) & 0xFF) << (8 * (e & 3));
    return make_uint2(w[0], w[1]);
}
__device__ __forceinline__ uint2 codes8(const uint4& v, float s, float r_lo, float r_hi) {
    const __half2* h = reinterpret_cast<const __half2*>(&v);
    uint32_t lo[8], bad = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float2 f = __half22float2(h[e]);
        lo[2 * e] = __float_as_uint(fmaf(f.x, r_lo, 12582912.0f));
        lo[2 * e + 1] = __float_as_uint(fmaf(f.y, r_lo, 12582912.0f));
        bad |= (lo[2 * e] ^ __float_as_uint(fmaf(f.x, r_hi, 12582912.0f))) | (lo[2 * e + 1] ^ __float_as_uint(fmaf(f.y, r_hi, 12582912.0f)));
    }
    if (bad) return codes8_by_division(v, s);
    auto low4 = [&](int i) { return __byte_perm(__byte_perm(lo[i], lo[i + 1], 0x0040), __byte_perm(lo[i + 2], lo[i + 3], 0x0040), 0x5410); };
    return make_uint2(low4(0), low4(4));
}

// Per-token quantizer of fp16 activations (the inputs of the integer-activation projections): one warp per row of
// `cols` fp16 values (a multiple of 8), which it keeps in registers between the absmax pass and the code pass when the
// row is short enough (KEEP x 256 columns), so that the row is read once; KEEP as small as the row allows.  Same results as quantize_rows_kernel.
template <int KEEP>
__global__ void __launch_bounds__(256) quantize_rows_f16_kernel(const __half* x, long long rows, int cols, int8_t* codes, float* scales) {
    // Starts early; its rows may come from the predecessor, and its codes go where the predecessor's predecessor may still read.
    // Only behind the wait may the successor (the integer GEMM) start: it reads its weights at once, which whatever ran before
    // this kernel may have written.
    ptx::pdl_wait();
    ptx::pdl_trigger();
    const int lane = threadIdx.x & 31;
    const long long warps_total = (long long)gridDim.x * (blockDim.x >> 5);
    const int chunks = cols / 8;                                 // 16-byte chunks of a row
    for (long long r = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < rows; r += warps_total) {
        const uint4* xr = reinterpret_cast<const uint4*>(x + r * cols);
        uint4 keep[KEEP];
        __half2 a2 = __float2half2_rn(0.f);                      // (maxima of fp16 magnitudes are exact)
        auto absmax8 = [&](const uint4& v) {
            const __half2* h = reinterpret_cast<const __half2*>(&v);
#pragma unroll
            for (int e = 0; e < 4; ++e) a2 = __hmax2(a2, __habs2(h[e]));
        };
#pragma unroll
        for (int j = 0; j < KEEP; ++j) {
            const int i = lane + 32 * j;
            keep[j] = make_uint4(0, 0, 0, 0);
            if (i < chunks) keep[j] = xr[i];
        }
#pragma unroll
        for (int j = 0; j < KEEP; ++j) absmax8(keep[j]);
        for (int i = lane + 32 * KEEP; i < chunks; i += 32) absmax8(xr[i]);
        const float a = warp_max(fmaxf(__low2float(a2), __high2float(a2)));
        const float s = quant_scale(a, 127.f);
        const float rs = __frcp_rn(s);
        const float r_lo = s > 0.f ? __uint_as_float(__float_as_uint(rs) - 2u) : 0.f, r_hi = s > 0.f ? __uint_as_float(__float_as_uint(rs) + 2u) : 0.f;
        if (lane == 0) scales[r] = s;
        uint2* cr = reinterpret_cast<uint2*>(codes + r * cols);
#pragma unroll
        for (int j = 0; j < KEEP; ++j) {
            const int i = lane + 32 * j;
            if (i < chunks) cr[i] = codes8(keep[j], s, r_lo, r_hi);
        }
        for (int i = lane + 32 * KEEP; i < chunks; i += 32) cr[i] = codes8(xr[i], s, r_lo, r_hi);
    }
}

cudaError_t launch_quantize_rows_f16(const __half* x, long long rows, int cols, int8_t* codes, float* scales, cudaStream_t stream) {
    if (rows == 0) return cudaSuccess;
    long long blocks = (rows + 7) / 8;
    if (blocks > 148LL * 32) blocks = 148LL * 32;
    auto* kern = cols <= 512 ? quantize_rows_f16_kernel<2> : cols <= 768 ? quantize_rows_f16_kernel<3> : cols <= 1280 ? quantize_rows_f16_kernel<5> : quantize_rows_f16_kernel<8>;
    return launch_pdl(kern, dim3((unsigned)blocks), dim3(256), 0, stream, x, rows, cols, codes, scales);
}

// ---- helpers of the token-sensitivity sweep (Eq. 1) -------------------------------------------------------------
__global__ void __launch_bounds__(256) mse_partial_kernel(const __half* __restrict__ a, const __half* __restrict__ b, long long n, double* __restrict__ partials) {
    double acc = 0.0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float dlt = __half2float(a[i]) - __half2float(b[i]);
        acc += (double)dlt * (double)dlt;
    }
    __shared__ double sh[256];
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {           // fixed tree: the same sum for the same inputs
        if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) partials[blockIdx.x] = sh[0];
}
__global__ void __launch_bounds__(256) mse_final_kernel(const double* __restrict__ partials, long long n, double* __restrict__ out) {
    __shared__ double sh[256];
    sh[threadIdx.x] = partials[threadIdx.x];
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = sh[0] / (double)n;
}
cudaError_t launch_mse_f16(const __half* a, const __half* b, long long n, double* partials, double* out, cudaStream_t stream) {
    mse_partial_kernel<<<256, 256, 0, stream>>>(a, b, n, partials);
    mse_final_kernel<<<1, 256, 0, stream>>>(partials, n, out);
    return cudaGetLastError();
}
__global__ void sensitivity_masks_kernel(uint8_t* masks, int batch, int n_ctx) {
    const long long total = (long long)(n_ctx + 1) * batch * n_ctx;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const int t = (int)(i % n_ctx), which = (int)(i / ((long long)batch * n_ctx));
        masks[i] = (which == n_ctx || t != which) ? 1 : 0;
    }
}
cudaError_t launch_sensitivity_masks(uint8_t* masks, int batch, int n_ctx, cudaStream_t stream) {
    sensitivity_masks_kernel<<<64, 256, 0, stream>>>(masks, batch, n_ctx);
    return cudaGetLastError();
}

// TPG threads per (output channel, group): eight for groups of up to 128 elements (the usual W4), a warp for those of up to 512, half a
// block for longer ones (a whole row of an 8-bit matrix).  A thread keeps up to sixteen elements in registers between the absmax and
// the codes: 16-byte loads, neighbouring threads on neighbouring ones, one word of codes per two threads, codes by the
// reciprocal where it decides, with one test for four of them.  What bounds it is the chain of one group (load, absmax, an IEEE division,
// codes, store) and the launch, not the 6.6 MB of a 1280 x 1280 matrix (1 us): with a warp per group and four groups in a
// row the chain had four divisions and twenty shuffles instead of one and three (launches in a graph: 320 x 320 4.2 -> 2.5 us, 1280 x 1280
// 5.5 -> 4.0, 2560 x 2560 19.2 -> 10.4; whole rows of 8-bit codes 5.5 -> 4.5).  The kernel starts under its predecessor's tail: without
// that the four matrices of a 1280-channel layer, call by call, took 3 us more.
template <int TPG>
__global__ void __launch_bounds__(256) pack_weights_kernel(const float* W, const float* bias, uint8_t* blob, int n_out, int k_in, int bits, int group) {
    constexpr int KEEP = 4, PER_BLOCK = 256 / TPG;                      // float4 per thread in registers; groups per block
    const WeightLayout L = weight_layout(n_out, k_in, bits, group);
    const int lane = threadIdx.x & 31, t = threadIdx.x % TPG, slot = threadIdx.x / TPG;
    const int qmax = bits == 8 ? 127 : 7;
    const long long items = (long long)n_out * L.n_groups;
    float* scales = reinterpret_cast<float*>(blob + L.off_scales);
    float* bias_out = reinterpret_cast<float*>(blob + L.off_bias);
    __shared__ float part[8];
    // (W may come from the previous kernel, and the one before it may still read the blob.)
    ptx::pdl_wait();
    ptx::pdl_trigger();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        PackedHeader h;
        h.magic = kWeightMagic; h.version = 1; h.n_out = n_out; h.k_in = k_in; h.bits = bits; h.group = group;
        h.n_groups = L.n_groups; h.has_bias = bias != nullptr;
        h.off_codes = L.off_codes; h.off_scales = L.off_scales; h.off_bias = L.off_bias; h.total_bytes = L.total;
        *reinterpret_cast<PackedHeader*>(blob) = h;
    }
    // (every thread of a block makes the same number of rounds: the longer groups meet at barriers, the others at shuffles)
    for (long long it0 = (long long)blockIdx.x * PER_BLOCK; it0 < items; it0 += (long long)gridDim.x * PER_BLOCK) {
        const bool real = it0 + slot < items;
        const long long it = real ? it0 + slot : items - 1;
        const int n = items < (1LL << 31) ? (int)((uint32_t)it / (uint32_t)L.n_groups) : (int)(it / L.n_groups), g = (int)(it - (long long)n * L.n_groups);
        const int lo = g * L.group_len, n4 = (min(k_in, lo + L.group_len) - lo) / 4;              // (group lengths and fan-ins are multiples of 8)
        const float4* w4 = reinterpret_cast<const float4*>(W + (size_t)n * k_in + lo);
        float4 keep[KEEP];
        float a = 0.f;
        auto absmax4 = [&](const float4& v) { a = fmaxf(a, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w)))); };
#pragma unroll
        for (int j = 0; j < KEEP; ++j) keep[j] = t + TPG * j < n4 ? ptx::load_global(w4 + t + TPG * j) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int j = 0; j < KEEP; ++j) absmax4(keep[j]);
        for (int i = t + TPG * KEEP; i < n4; i += TPG) absmax4(ptx::load_global(w4 + i));
        __syncwarp();
#pragma unroll
        for (int o = TPG < 32 ? TPG / 2 : 16; o > 0; o >>= 1) a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, o));
        if (TPG > 32) {
            __syncthreads();
            if (lane == 0) part[threadIdx.x >> 5] = a;
            __syncthreads();
#pragma unroll
            for (int k = 0; k < TPG / 32; ++k) a = fmaxf(a, part[slot * (TPG / 32) + k]);
        }
        const float s = quant_scale(a, (float)qmax);
        const float rs = s > 0.f ? __frcp_rn(s) : 0.f;
        const float r_lo = __uint_as_float(__float_as_uint(rs) - 2u), r_hi = __uint_as_float(__float_as_uint(rs) + 2u);
        if (real && t == 0) {
            scales[(size_t)n * L.n_groups + g] = s;
            if (g == 0) bias_out[n] = bias ? ptx::load_global(bias + n) : 0.f;
        }
        uint8_t* row = blob + L.off_codes + (size_t)n * L.row_bytes;
        auto encode = [&](const float4& v, int i, bool have) {           // elements 4 i .. 4 i + 3 of the group
            const float x[4] = {v.x, v.y, v.z, v.w};
            int c[4] = {0, 0, 0, 0};
            if (s > 0.f) {                                               // (see quant_code_127)
                uint32_t bad = 0;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const uint32_t u = __float_as_uint(fmaf(x[e], r_lo, 12582912.0f));
                    bad |= u ^ __float_as_uint(fmaf(x[e], r_hi, 12582912.0f));
                    c[e] = (int)(u << 24) >> 24;                         // the low byte, sign-extended
                }
                if (bad) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) c[e] = quant_code_127(x[e], s, r_lo, r_hi);
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) c[e] = min(max(c[e], -qmax), qmax);
            }
            if (bits == 8) {
                if (real && have) reinterpret_cast<char4*>(row + lo)[i] = make_char4((signed char)c[0], (signed char)c[1], (signed char)c[2], (signed char)c[3]);
            } else {                                                     // a word is eight elements: two neighbouring threads
                // (w4_nibble_pos: elements 0..3 in nibbles 0, 4, 1, 5, elements 4..7 in 2, 6, 3, 7)
                uint32_t word = (uint32_t)(c[0] + 8) | (uint32_t)(c[1] + 8) << 16 | (uint32_t)(c[2] + 8) << 4 | (uint32_t)(c[3] + 8) << 20;
                word <<= 8 * (lane & 1);
                __syncwarp();
                word |= __shfl_xor_sync(0xffffffffu, word, 1);
                if (real && have && (lane & 1) == 0) reinterpret_cast<uint32_t*>(row + lo / 2)[i >> 1] = word;
            }
        };
#pragma unroll
        for (int j = 0; j < KEEP; ++j)
            if (TPG < 32 || TPG * j < n4) encode(keep[j], t + TPG * j, t + TPG * j < n4);          // (several groups in a warp: all of its threads shuffle)
        if (TPG >= 32)
            for (int i0 = TPG * KEEP; i0 < n4; i0 += TPG) encode(i0 + t < n4 ? ptx::load_global(w4 + i0 + t) : make_float4(0.f, 0.f, 0.f, 0.f), i0 + t, i0 + t < n4);
    }
}

cudaError_t launch_pack_weights(const taq_weight_desc& d, const float* W, const float* bias, void* packed, cudaStream_t stream) {
    const WeightLayout L = weight_layout(d.n_out, d.k_in, d.bits, d.group);
    const long long items = (long long)d.n_out * L.n_groups, per_block = L.group_len > 512 ? 2 : L.group_len > 128 ? 8 : 32;
    long long blocks = (items + per_block - 1) / per_block;
    if (blocks > 148LL * 32) blocks = 148LL * 32;
    auto* kern = L.group_len > 512 ? pack_weights_kernel<128> : L.group_len > 128 ? pack_weights_kernel<32> : pack_weights_kernel<8>;
    return launch_pdl(kern, dim3((unsigned)blocks), dim3(256), 0, stream, W, bias, (uint8_t*)packed, d.n_out, d.k_in, d.bits, d.group);
}

__global__ void __launch_bounds__(256) unpack_weights_kernel(const uint8_t* __restrict__ blob, int8_t* __restrict__ codes_out,
                                                             float* __restrict__ scales_out, int n_out, int k_in, int bits, int group) {
    const WeightLayout L = weight_layout(n_out, k_in, bits, group);
    const long long total = (long long)n_out * k_in;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += stride) {
        const int n = (int)(i / k_in), k = (int)(i % k_in);
        codes_out[i] = (int8_t)load_code(blob + L.off_codes, L.row_bytes, bits, n, k);
    }
    const float* scales = reinterpret_cast<const float*>(blob + L.off_scales);
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < (long long)n_out * L.n_groups; i += stride) scales_out[i] = scales[i];
}

cudaError_t launch_unpack_weights(const taq_weight_desc& d, const void* packed, int8_t* codes, float* scales, cudaStream_t stream) {
    long long total = (long long)d.n_out * d.k_in;
    long long blocks = (total + 255) / 256;
    if (blocks > 148LL * 16) blocks = 148LL * 16;
    unpack_weights_kernel<<<(unsigned)blocks, 256, 0, stream>>>((const uint8_t*)packed, codes, scales, d.n_out, d.k_in, d.bits, d.group);
    return cudaGetLastError();
}

}  // namespace taq
