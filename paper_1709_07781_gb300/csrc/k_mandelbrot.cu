// Escape-time Mandelbrot image: the paper's compute-bound workload for
// kernel actors (Sec. 5.4), here a plain CUDA kernel and an actor stage.
//
// Pixel (x, y) is c = (re_min + x dre, im_min + y dim); from z = 0 the step
// z <- z^2 + c is applied while |z|^2 <= 4, at most max_iter times, and the
// pixel holds the number of steps. Every operation is one round-to-nearest
// single-precision operation in a fixed order (__fmul_rn / __fadd_rn /
// __fsub_rn cannot be contracted into fused multiply-adds), so each count is
// reproducible bit for bit on any IEEE machine that does the same operations.
//
// The work is ALU-bound: no memory traffic to speak of. What bounds it is the
// FP32 pipes, so a step is made of as few operations as give the same bits:
//   * A thread carries two neighbouring pixels, one in either half of 64-bit
//     registers, so the paired f32x2 operations of sm_100-class GPUs do both
//     with one instruction and nothing has to be packed or unpacked.
//   * 2 zr zi + ci is the product p = zr zi and one fused 2 p + ci. Doubling is
//     exact, so this rounds as the definition's two products and a sum do
//     (below 2^-126, where p loses bits that 2 zr zi keeps, both vanish against
//     |ci| >= 2^-90, and for ci = 0 every term is a zero of the same sign).
//   * The escape test runs once per eight steps, on the last of them: once
//     |z|^2 > 4 it stays so for |c|^2 <= 3.999 (|c| < 1.99976, so |z^2 + c| >
//     2.00024 and its square 4.0009, where a step's rounding moves it by less
//     than 0.0001), or becomes infinite or NaN, which does not compare as at most
//     4 either. Where eight steps fail it, the orbit at their start is kept, and
//     looked through step by step after the loop, once for all pixels of a warp:
//     the count is exact.
// A pixel with |c|^2 above 3.999 (it escapes at once but for the tip at -2), or
// with 0 < |im c| < 2^-90, takes the definition's operations, in pairs and eight
// steps at a time too, with the largest |z|^2 of the eight tested. 1920 x 1080,
// 1000 steps, a view of the tip (-1.945 to -1.938): 83 us with one pixel a
// thread, 128 us with a pixel after the other and a test on every step for what
// is above 3.6, 66 us now; the last 1e-5 before -2: 36 us and 32 us.
// 1920 x 1080, 100 steps: 63 us with one pixel a thread and a test on every step,
// 43 us now (six paired operations a step for two pixels: 30 us at one
// per two cycles).
#include "ka_internal.h"

namespace ka {
namespace {

constexpr int kMbBlock = 128;

// Pairs of single-precision values in one 64-bit register, and the paired
// round-to-nearest multiply and add of sm_100-class GPUs (one instruction for
// two IEEE operations, each rounded as __fmul_rn / __fadd_rn would).
__device__ __forceinline__ uint64_t pair(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpair(uint64_t v, float &a, float &b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t mul_rn2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t add_rn2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ uint64_t fma_rn2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// Sum and difference of two products: as fused operations on them with the
// factors 1 and -1. (A paired add or sub of paired products, both .rn, came out
// as one fused operation on the factors, which rounds once too few.)
__device__ __forceinline__ uint64_t sum2(uint64_t a, uint64_t b) { return fma_rn2(a, pair(1.0f, 1.0f), b); }
__device__ __forceinline__ uint64_t diff2(uint64_t a, uint64_t b) { return fma_rn2(b, pair(-1.0f, -1.0f), a); }


// Whether the short steps and a test every kMbRun steps give the definition's
// counts for c.
__device__ __forceinline__ bool short_exact(float cr, float ci) {
    const float a = fabsf(ci);
    return cr * cr + ci * ci <= 3.999f && (a == 0.0f || a >= 0x1p-90f);
}

// One step of two orbits: the short one, or by the definition's operations
// (2 zr by an addition, exact as the product with 2 is).
template <bool SHORT>
__device__ __forceinline__ void advance(uint64_t &zr, uint64_t &zi, uint64_t rr, uint64_t ii, uint64_t cr,
                                        uint64_t ci) {
    if (SHORT) {
        const uint64_t p = mul_rn2(zr, zi);
        zr = add_rn2(diff2(rr, ii), cr);
        zi = fma_rn2(pair(2.0f, 2.0f), p, ci);
    } else {
        const uint64_t p = mul_rn2(add_rn2(zr, zr), zi);
        zr = add_rn2(diff2(rr, ii), cr);
        zi = sum2(p, ci);
    }
}

// a with its half i replaced by that of b.
__device__ __forceinline__ uint64_t with_half(uint64_t a, uint64_t b, int i) {
    return i == 0 ? (a & 0xFFFFFFFF00000000ull) | (b & 0xFFFFFFFFull) : (a & 0xFFFFFFFFull) | (b & 0xFFFFFFFF00000000ull);
}

constexpr uint32_t kMbRun = 8;  // steps between two tests

// Steps of two orbits until each escapes, at most max_iter; `open`: the pixels
// that there are (bit i). SHORT: for short_exact c. Otherwise any c: with the
// definition's operations, and the test is on the largest |z|^2 of the run
// (the first above 4 is a number or infinite: one step from |z| <= 2).
template <bool SHORT>
__device__ __forceinline__ void escape_steps(uint64_t c0, uint64_t c1, uint32_t open, uint32_t max_iter,
                                             uint32_t (&n)[2]) {
    uint64_t zr = 0, zi = 0, cr = c0, ci = c1;  // the running orbits (a pixel that has escaped: 0, c too)
    uint64_t sr = 0, si = 0;                    // each pixel's orbit where it is finished from, step n
    uint32_t most[2] = {kMbRun, kMbRun};        // and the steps left to look at there
    uint32_t escaped = 3u & ~open, k = 0u;
    for (uint32_t runs = max_iter / kMbRun; runs != 0u; --runs) {
        const uint64_t zr_0 = zr, zi_0 = zi;
        float m[2] = {0.0f, 0.0f};
#pragma unroll
        for (uint32_t i = 0; i < kMbRun; ++i) {
            const uint64_t rr = mul_rn2(zr, zr), ii = mul_rn2(zi, zi);
            if (!SHORT || i == kMbRun - 1u) {
                float q[2];
                unpair(sum2(rr, ii), q[0], q[1]);
                m[0] = SHORT ? q[0] : fmaxf(m[0], q[0]);
                m[1] = SHORT ? q[1] : fmaxf(m[1], q[1]);
            }
            advance<SHORT>(zr, zi, rr, ii, cr, ci);
        }
        if (!(m[0] <= 4.0f) || !(m[1] <= 4.0f)) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                if (!(m[i] <= 4.0f)) {  // in this run: found at the end, by all threads at once
                    sr = with_half(sr, zr_0, i);
                    si = with_half(si, zi_0, i);
                    n[i] = k;
                    escaped |= 1u << i;
                    zr = with_half(zr, 0, i);
                    zi = with_half(zi, 0, i);
                    cr = with_half(cr, 0, i);
                    ci = with_half(ci, 0, i);
                }
            }
            if (escaped == 3u) break;
        }
        k += kMbRun;
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        if (!((escaped >> i) & 1u)) {  // the last steps, fewer than a run
            sr = with_half(sr, zr, i);
            si = with_half(si, zi, i);
            n[i] = k;
            most[i] = max_iter - k;
        }
    }
#pragma unroll 1
    for (uint32_t j = 0; j < kMbRun; ++j) {
        const uint64_t rr = mul_rn2(sr, sr), ii = mul_rn2(si, si);
        float m[2];
        unpair(sum2(rr, ii), m[0], m[1]);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            if (((open >> i) & 1u) && (m[i] > 4.0f || j == most[i])) {
                n[i] += j;
                open &= ~(1u << i);
            }
        }
        if (open == 0u) break;
        advance<SHORT>(sr, si, rr, ii, c0, c1);
    }
}

__global__ void __launch_bounds__(kMbBlock, 16) k_mandelbrot(uint32_t *out, uint32_t width, uint32_t pixels, float re_min,
                                                          float im_min, float dre, float dim, uint32_t max_iter) {
    const uint64_t p0 = (uint64_t(blockIdx.x) * kMbBlock + threadIdx.x) * 2u;
    if (p0 >= pixels) return;
    const bool two = p0 + 1u < pixels;
    const uint32_t y0 = uint32_t(p0) / width, x0 = uint32_t(p0) - y0 * width;
    const bool wrap = x0 + 1u == width;
    const uint32_t x1 = wrap ? 0u : x0 + 1u, y1 = wrap ? y0 + 1u : y0;
    const float ar = __fadd_rn(re_min, __fmul_rn(float(x0), dre)), ai = __fadd_rn(im_min, __fmul_rn(float(y0), dim));
    float br = __fadd_rn(re_min, __fmul_rn(float(x1), dre)), bi = __fadd_rn(im_min, __fmul_rn(float(y1), dim));
    if (!two) br = bi = 0.0f;
    uint32_t n[2] = {0u, 0u};
    if (short_exact(ar, ai) && short_exact(br, bi)) {
        escape_steps<true>(pair(ar, br), pair(ai, bi), two ? 3u : 1u, max_iter, n);
    } else {
        escape_steps<false>(pair(ar, br), pair(ai, bi), two ? 3u : 1u, max_iter, n);
    }
    if (two && (reinterpret_cast<uintptr_t>(out) & 7u) == 0u) {
        *reinterpret_cast<uint2 *>(out + p0) = make_uint2(n[0], n[1]);
    } else {
        out[p0] = n[0];
        if (two) out[p0 + 1u] = n[1];
    }
}

__global__ void k_set_word(uint32_t *w, uint32_t v) { *w = v; }

}  // namespace

ka_status launch_mandelbrot(uint32_t *out, uint32_t width, uint32_t height, float re_min, float im_min, float re_max,
                            float im_max, uint32_t max_iter, uint32_t *n_out, cudaStream_t stream) {
    const uint64_t pixels = uint64_t(width) * height;
    if (pixels > 0xFFFFFFFFull || (pixels && !out)) return KA_E_ARG;
    if (pixels) {
        // the same single-precision expressions as the definition
        const float dre = (re_max - re_min) / float(width);
        const float dim = (im_max - im_min) / float(height);
        // one pair of pixels a thread and no grid stride: pixels differ in
        // work, and the scheduler deals blocks to the SMs that are free
        const uint64_t blocks = (pixels + 2 * kMbBlock - 1) / (2 * kMbBlock);
        k_mandelbrot<<<unsigned(blocks), kMbBlock, 0, stream>>>(out, width, uint32_t(pixels), re_min, im_min, dre,
                                                                dim, max_iter);
        const ka_status s = cuda_status(cudaGetLastError());
        if (s != KA_OK) return s;
    }
    if (n_out) {
        k_set_word<<<1, 1, 0, stream>>>(n_out, uint32_t(pixels));
        return cuda_status(cudaGetLastError());
    }
    return KA_OK;
}

}  // namespace ka

using namespace ka;

extern "C" ka_status ka_mandelbrot(uint32_t *d_out, uint32_t width, uint32_t height, float re_min, float im_min,
                                   float re_max, float im_max, uint32_t max_iter, void *stream) {
    return launch_mandelbrot(d_out, width, height, re_min, im_min, re_max, im_max, max_iter, nullptr,
                             static_cast<cudaStream_t>(stream));
}
