// Host-side block quantiser of the lw library (pure CPU, no CUDA calls).
//
// Implements the generic rule q = round((x - mu)/s), x^ = s*q + mu with the scale chosen from the
// block's range [paper Eq. 1] for the "basic" formats q8_0 / q4_0 and the K-quant q4_K [Sec 2.2],
// plus plain f16 rounding.  Per-format constants follow the public ggml conventions.

#include <cmath>
#include <cstdint>
#include <cstring>
#include <memory>
#include <new>
#if defined(__x86_64__)
#include <immintrin.h>
#endif

#include "lw_internal.h"

namespace lw {

// fp32 -> binary16, round to nearest even, integer arithmetic on the bit patterns.
static inline uint16_t f32_to_f16_bits(float value) {
    uint32_t u;
    std::memcpy(&u, &value, sizeof u);
    const uint32_t sgn = (u >> 16) & 0x8000u;
    u &= 0x7FFFFFFFu;
    if (u >= 0x7F800000u) return (uint16_t)(sgn | (u > 0x7F800000u ? 0x7E00u : 0x7C00u));
    if (u >= 0x477FF000u) return (uint16_t)(sgn | 0x7C00u);        // >= 65520 rounds to infinity
    if (u < 0x33000001u) return (uint16_t)sgn;                      // <= 2^-25 rounds to zero
    const int e = (int)(u >> 23) - 127;                             // unbiased exponent
    uint32_t sig = (u & 0x007FFFFFu) | 0x00800000u;                 // 24-bit significand
    int drop = 13;                                                  // bits to discard for a normal half
    if (e < -14) drop += -14 - e;                                   // subnormal half: discard more
    const uint32_t kept = sig >> drop;
    const uint32_t rem = sig & ((1u << drop) - 1u);
    const uint32_t half_ulp = 1u << (drop - 1);
    uint32_t r = kept;
    if (rem > half_ulp || (rem == half_ulp && (kept & 1u))) ++r;
    uint32_t out;
    if (e < -14) out = r;                                           // may carry into the smallest normal
    else out = ((uint32_t)(e + 15) << 10) + (r - 0x400u);           // carry bumps the exponent
    return (uint16_t)(sgn | out);
}

static inline float f16_bits_to_f32(uint16_t h) {
    const uint32_t sgn = (uint32_t)(h & 0x8000u) << 16;
    const uint32_t ex = (h >> 10) & 0x1Fu;
    uint32_t man = h & 0x3FFu;
    uint32_t u;
    if (ex == 0) {
        if (man == 0) {
            u = sgn;
        } else {                                                    // subnormal: normalise
            int shift = 0;
            while (!(man & 0x400u)) { man <<= 1; ++shift; }
            u = sgn | ((uint32_t)(127 - 14 - shift) << 23) | ((man & 0x3FFu) << 13);
        }
    } else if (ex == 31) {
        u = sgn | 0x7F800000u | (man << 13);
    } else {
        u = sgn | ((ex + 112u) << 23) | (man << 13);
    }
    float f;
    std::memcpy(&f, &u, sizeof f);
    return f;
}

static inline bool is_inf_or_nan_half(uint16_t h) { return (h & 0x7C00u) == 0x7C00u; }

static inline void put_half(uint8_t* p, uint16_t h) {
    p[0] = (uint8_t)h;
    p[1] = (uint8_t)(h >> 8);
}

static int quantize_rows_f16(const float* src, int64_t n, uint8_t* dst) {
    for (int64_t i = 0; i < n; ++i) {
        const uint16_t h = f32_to_f16_bits(src[i]);
        if (is_inf_or_nan_half(h)) return LW_ERR_NONFINITE;
        put_half(dst + 2 * i, h);
    }
    return LW_OK;
}

static int quantize_rows_q8_0(const float* src, int64_t n, uint8_t* dst) {
    for (int64_t blk = 0; blk * 32 < n; ++blk, src += 32, dst += 34) {
        float peak = 0.f;
        for (int i = 0; i < 32; ++i) peak = std::fmax(peak, std::fabs(src[i]));
        const float step = peak / 127.f;
        const float inv = step != 0.f ? 1.f / step : 0.f;
        const uint16_t h = f32_to_f16_bits(step);
        if (is_inf_or_nan_half(h)) return LW_ERR_NONFINITE;
        put_half(dst, h);
        int8_t* q = reinterpret_cast<int8_t*>(dst + 2);
        for (int i = 0; i < 32; ++i) q[i] = (int8_t)std::lroundf(src[i] * inv);
    }
    return LW_OK;
}

static int quantize_rows_q4_0(const float* src, int64_t n, uint8_t* dst) {
    for (int64_t blk = 0; blk * 32 < n; ++blk, src += 32, dst += 18) {
        int arg = 0;
        for (int i = 1; i < 32; ++i)
            if (std::fabs(src[i]) > std::fabs(src[arg])) arg = i;   // first strict maximum of |x|
        const float step = (src[arg] + 0.f) / -8.f;                 // (a block of zeros, of either sign: 0 / -8)
        const float inv = step != 0.f ? 1.f / step : 0.f;
        const uint16_t h = f32_to_f16_bits(step);
        if (is_inf_or_nan_half(h)) return LW_ERR_NONFINITE;
        put_half(dst, h);
        for (int j = 0; j < 16; ++j) {
            int lo = (int)(src[j] * inv + 8.5f);
            int hi = (int)(src[j + 16] * inv + 8.5f);
            lo = lo > 15 ? 15 : lo;
            hi = hi > 15 ? 15 : hi;
            dst[2 + j] = (uint8_t)(lo | (hi << 4));
        }
    }
    return LW_OK;
}

// q4_1, q5_0, q5_1: BITS-bit codes; with OFFSET the grid runs from the block's minimum in steps of
// (max - min)/(2^BITS - 1), without it the signed extreme sits on code 0 as in q4_0.  Fifth bits go to
// a little-endian word after the fp16 fields, the low four bits to nibbles laid out as in q4_0.
template <int BITS, bool OFFSET>
static int quantize_rows_legacy(const float* src, int64_t n, uint8_t* dst) {
    constexpr int kTop = (1 << BITS) - 1;
    constexpr int kBytes = 2 + (OFFSET ? 2 : 0) + (BITS == 5 ? 4 : 0) + 16;
    for (int64_t blk = 0; blk * 32 < n; ++blk, src += 32, dst += kBytes) {
        int code[32];
        uint16_t hd, hm = 0;
        if (OFFSET) {
            float lo = src[0], hi = src[0];
            for (int i = 1; i < 32; ++i) {
                lo = src[i] < lo ? src[i] : lo;
                hi = src[i] > hi ? src[i] : hi;
            }
            const float step = (hi - lo) / (float)kTop;
            const float inv = step != 0.f ? 1.f / step : 0.f;
            hd = f32_to_f16_bits(step);
            hm = f32_to_f16_bits(lo);
            for (int i = 0; i < 32; ++i) {
                const int c = (int)((src[i] - lo) * inv + 0.5f);
                code[i] = c > kTop ? kTop : c;
            }
        } else {
            int arg = 0;
            for (int i = 1; i < 32; ++i)
                if (std::fabs(src[i]) > std::fabs(src[arg])) arg = i;   // first strict maximum of |x|
            constexpr float kHalf = (float)(1 << (BITS - 1));
            const float step = (src[arg] + 0.f) / -kHalf;               // (as in q4_0)
            const float inv = step != 0.f ? 1.f / step : 0.f;
            hd = f32_to_f16_bits(step);
            for (int i = 0; i < 32; ++i) {
                const int c = (int)(src[i] * inv + kHalf + 0.5f);
                code[i] = c > kTop ? kTop : c;
            }
        }
        if (is_inf_or_nan_half(hd) || is_inf_or_nan_half(hm)) return LW_ERR_NONFINITE;
        uint8_t* p = dst;
        put_half(p, hd);
        p += 2;
        if (OFFSET) {
            put_half(p, hm);
            p += 2;
        }
        if (BITS == 5) {
            uint32_t high = 0;
            for (int i = 0; i < 32; ++i) high |= (uint32_t)(code[i] >> 4) << i;
            for (int b = 0; b < 4; ++b) p[b] = (uint8_t)(high >> (8 * b));
            p += 4;
        }
        for (int j = 0; j < 16; ++j) p[j] = (uint8_t)((code[j] & 15) | ((code[j + 16] & 15) << 4));
    }
    return LW_OK;
}

static int quantize_rows_q4_K(const float* src, int64_t n, uint8_t* dst) {
    for (int64_t sb = 0; sb * 256 < n; ++sb, src += 256, dst += 144) {
        float step[8], offs[8];
        float step_max = 0.f, offs_max = 0.f;
        for (int s = 0; s < 8; ++s) {
            float lo = 0.f, hi = src[32 * s];
            for (int i = 0; i < 32; ++i) {
                lo = std::fmin(lo, src[32 * s + i]);
                hi = std::fmax(hi, src[32 * s + i]);
            }
            hi = std::fmax(hi, lo);
            step[s] = (hi - lo) / 15.f;
            offs[s] = -lo;
            if (step[s] > step_max) step_max = step[s];
            if (offs[s] > offs_max) offs_max = offs[s];       // keeps +0 when every offset is -0
        }
        const uint16_t hd = f32_to_f16_bits(step_max / 63.f);
        const uint16_t hm = f32_to_f16_bits(offs_max / 63.f);
        if (is_inf_or_nan_half(hd) || is_inf_or_nan_half(hm)) return LW_ERR_NONFINITE;
        const float d = f16_bits_to_f32(hd), dmin = f16_bits_to_f32(hm);
        put_half(dst, hd);
        put_half(dst + 2, hm);
        uint32_t sc[8], mn[8];
        for (int s = 0; s < 8; ++s) {
            const float a = d != 0.f ? std::roundf(step[s] / d) : 0.f;
            const float b = dmin != 0.f ? std::roundf(offs[s] / dmin) : 0.f;
            sc[s] = (uint32_t)std::fmin(a, 63.f);
            mn[s] = (uint32_t)std::fmin(b, 63.f);
        }
        uint8_t* packed = dst + 4;
        for (int j = 0; j < 4; ++j) {
            packed[j] = (uint8_t)(sc[j] | ((sc[j + 4] >> 4) << 6));
            packed[4 + j] = (uint8_t)(mn[j] | ((mn[j + 4] >> 4) << 6));
            packed[8 + j] = (uint8_t)((sc[j + 4] & 15u) | ((mn[j + 4] & 15u) << 4));
        }
        uint8_t* qs = dst + 16;
        for (int g = 0; g < 4; ++g) {
            const float dl0 = d * (float)sc[2 * g], ml0 = dmin * (float)mn[2 * g];
            const float dl1 = d * (float)sc[2 * g + 1], ml1 = dmin * (float)mn[2 * g + 1];
            for (int l = 0; l < 32; ++l) {
                float a = 0.f, b = 0.f;
                if (dl0 != 0.f) a = std::fmin(15.f, std::fmax(0.f, std::roundf((src[64 * g + l] + ml0) / dl0)));
                if (dl1 != 0.f) b = std::fmin(15.f, std::fmax(0.f, std::roundf((src[64 * g + 32 + l] + ml1) / dl1)));
                qs[32 * g + l] = (uint8_t)((uint32_t)a | ((uint32_t)b << 4));
            }
        }
    }
    return LW_OK;
}

// q2_K: the affine min/max rule on runs of 16 weights: three code steps per run, steps and offsets
// rounded to 4 bits against fp16 d = max step/15 and dmin = max offset/15.
static int quantize_rows_q2_K(const float* src, int64_t n, uint8_t* dst) {
    for (int64_t sb = 0; sb * 256 < n; ++sb, src += 256, dst += 84) {
        float step[16], offs[16];
        float step_max = 0.f, offs_max = 0.f;
        for (int t = 0; t < 16; ++t) {
            float lo = 0.f, hi = src[16 * t];
            for (int i = 0; i < 16; ++i) {
                lo = std::fmin(lo, src[16 * t + i]);
                hi = std::fmax(hi, src[16 * t + i]);
            }
            hi = std::fmax(hi, lo);
            step[t] = (hi - lo) / 3.f;
            offs[t] = -lo;
            if (step[t] > step_max) step_max = step[t];
            if (offs[t] > offs_max) offs_max = offs[t];       // keeps +0 when every offset is -0
        }
        const uint16_t hd = f32_to_f16_bits(step_max / 15.f);
        const uint16_t hm = f32_to_f16_bits(offs_max / 15.f);
        if (is_inf_or_nan_half(hd) || is_inf_or_nan_half(hm)) return LW_ERR_NONFINITE;
        const float d = f16_bits_to_f32(hd), dmin = f16_bits_to_f32(hm);
        std::memset(dst, 0, 84);
        put_half(dst + 80, hd);
        put_half(dst + 82, hm);
        for (int t = 0; t < 16; ++t) {                 // run t: weights 16t..16t+15, pair number t
            const float a = d != 0.f ? std::roundf(step[t] / d) : 0.f;
            const float b = dmin != 0.f ? std::roundf(offs[t] / dmin) : 0.f;
            const uint32_t sc = (uint32_t)std::fmin(a, 15.f), mn = (uint32_t)std::fmin(b, 15.f);
            dst[t] = (uint8_t)(sc | (mn << 4));
            const float dl = d * (float)sc, ml = dmin * (float)mn;
            const int half = t >> 3, quarter = (t >> 1) & 3, l0 = (t & 1) * 16;
            for (int i = 0; i < 16; ++i) {
                float c = 0.f;
                if (dl != 0.f) c = std::fmin(3.f, std::fmax(0.f, std::roundf((src[16 * t + i] + ml) / dl)));
                uint8_t& byte = dst[16 + 32 * half + l0 + i];
                byte = (uint8_t)(byte | ((uint32_t)c << (2 * quarter)));
            }
        }
    }
    return LW_OK;
}

// q5_K: the q4_K rule with 31 code steps per sub-block; the fifth bit of each code goes to qh.
static int quantize_rows_q5_K(const float* src, int64_t n, uint8_t* dst) {
    for (int64_t sb = 0; sb * 256 < n; ++sb, src += 256, dst += 176) {
        float step[8], offs[8];
        float step_max = 0.f, offs_max = 0.f;
        for (int s = 0; s < 8; ++s) {
            float lo = 0.f, hi = src[32 * s];
            for (int i = 0; i < 32; ++i) {
                lo = std::fmin(lo, src[32 * s + i]);
                hi = std::fmax(hi, src[32 * s + i]);
            }
            hi = std::fmax(hi, lo);
            step[s] = (hi - lo) / 31.f;
            offs[s] = -lo;
            if (step[s] > step_max) step_max = step[s];
            if (offs[s] > offs_max) offs_max = offs[s];       // keeps +0 when every offset is -0
        }
        const uint16_t hd = f32_to_f16_bits(step_max / 63.f);
        const uint16_t hm = f32_to_f16_bits(offs_max / 63.f);
        if (is_inf_or_nan_half(hd) || is_inf_or_nan_half(hm)) return LW_ERR_NONFINITE;
        const float d = f16_bits_to_f32(hd), dmin = f16_bits_to_f32(hm);
        std::memset(dst, 0, 176);
        put_half(dst, hd);
        put_half(dst + 2, hm);
        uint32_t sc[8], mn[8];
        for (int s = 0; s < 8; ++s) {
            const float a = d != 0.f ? std::roundf(step[s] / d) : 0.f;
            const float b = dmin != 0.f ? std::roundf(offs[s] / dmin) : 0.f;
            sc[s] = (uint32_t)std::fmin(a, 63.f);
            mn[s] = (uint32_t)std::fmin(b, 63.f);
        }
        uint8_t* packed = dst + 4;
        for (int j = 0; j < 4; ++j) {
            packed[j] = (uint8_t)(sc[j] | ((sc[j + 4] >> 4) << 6));
            packed[4 + j] = (uint8_t)(mn[j] | ((mn[j + 4] >> 4) << 6));
            packed[8 + j] = (uint8_t)((sc[j + 4] & 15u) | ((mn[j + 4] & 15u) << 4));
        }
        uint8_t* qh = dst + 16;
        uint8_t* qs = dst + 48;
        for (int g = 0; g < 4; ++g) {
            const float dl0 = d * (float)sc[2 * g], ml0 = dmin * (float)mn[2 * g];
            const float dl1 = d * (float)sc[2 * g + 1], ml1 = dmin * (float)mn[2 * g + 1];
            for (int l = 0; l < 32; ++l) {
                float a = 0.f, b = 0.f;
                if (dl0 != 0.f) a = std::fmin(31.f, std::fmax(0.f, std::roundf((src[64 * g + l] + ml0) / dl0)));
                if (dl1 != 0.f) b = std::fmin(31.f, std::fmax(0.f, std::roundf((src[64 * g + 32 + l] + ml1) / dl1)));
                const uint32_t ca = (uint32_t)a, cb = (uint32_t)b;
                qs[32 * g + l] = (uint8_t)((ca & 15u) | ((cb & 15u) << 4));
                qh[l] = (uint8_t)(qh[l] | ((ca >> 4) << (2 * g)) | ((cb >> 4) << (2 * g + 1)));
            }
        }
    }
    return LW_OK;
}

// q6_K: every run of 16 weights gets a symmetric grid that puts its signed extreme (the first of
// equal magnitudes) on code 0, i.e. -32 steps; the sixteen steps become int8 multiples of one fp16
// factor d = (largest |step|)/127, and the codes are rounded against the step the decoder will use.
static int quantize_rows_q6_K(const float* src, int64_t n, uint8_t* dst) {
    for (int64_t sb = 0; sb * 256 < n; ++sb, src += 256, dst += 210) {
        float step[16];
        float largest = 0.f;
        for (int t = 0; t < 16; ++t) {
            float mag = 0.f, extreme = 0.f;
            for (int i = 0; i < 16; ++i) {
                const float v = src[16 * t + i];
                if (std::fabs(v) > mag) {
                    mag = std::fabs(v);
                    extreme = v;
                }
            }
            step[t] = extreme / -32.f;
            if (std::fabs(step[t]) > largest) largest = std::fabs(step[t]);
        }
        const uint16_t hd = f32_to_f16_bits(largest / 127.f);
        if (is_inf_or_nan_half(hd)) return LW_ERR_NONFINITE;
        const float d = f16_bits_to_f32(hd);
        std::memset(dst, 0, 210);
        put_half(dst + 208, hd);
        uint8_t* ql = dst;
        uint8_t* qh = dst + 128;
        for (int t = 0; t < 16; ++t) {             // run t holds weights 16t..16t+15; its scale is number t
            long sc = 0;
            if (d != 0.f) sc = std::lround(step[t] / d);
            if (sc > 127) sc = 127;
            if (sc < -127) sc = -127;
            dst[192 + t] = (uint8_t)(int8_t)sc;
            const float e = d * (float)sc;
            const int half = t >> 3, quarter = (t >> 1) & 3, l0 = (t & 1) * 16;
            for (int i = 0; i < 16; ++i) {
                long code = 32;
                if (e != 0.f) code = std::lround(src[16 * t + i] / e) + 32;
                if (code < 0) code = 0;
                if (code > 63) code = 63;
                const int l = l0 + i;
                uint8_t& low = ql[64 * half + l + 32 * (quarter & 1)];
                if (quarter < 2) low = (uint8_t)(low | (code & 15));
                else low = (uint8_t)(low | ((code & 15) << 4));
                qh[32 * half + l] = (uint8_t)(qh[32 * half + l] | ((code >> 4) << (2 * quarter)));
            }
        }
    }
    return LW_OK;
}

// ------------------------------------------------------------------ AVX2 forms ---
//
// The same rules eight weights at a time, byte for byte: every operation is the IEEE operation of the scalar form in the
// same order (multiplications and additions are not contracted), roundf is built from truncation (exact for every input),
// ties for an extreme go to the first occurrence as above.  A block whose scale is subnormal (its reciprocal may
// overflow) goes to the scalar form.  q4_K, 4 Mi weights, one core: 53 ms scalar, of which two thirds were calls of
// roundf, fmin and fmax.
#if defined(__x86_64__)
#define LW_QUANTIZE_AVX2 1
#pragma GCC push_options
#pragma GCC target("avx2,f16c")

namespace v8 {

static inline __m256 abs8(__m256 x) { return _mm256_and_ps(x, _mm256_castsi256_ps(_mm256_set1_epi32(0x7FFFFFFF))); }

// roundf: half away from zero
static inline __m256 round8(__m256 x) {
    const __m256 t = _mm256_round_ps(x, _MM_FROUND_TO_ZERO | _MM_FROUND_NO_EXC);
    const __m256 up = _mm256_cmp_ps(abs8(_mm256_sub_ps(x, t)), _mm256_set1_ps(0.5f), _CMP_GE_OQ);
    const __m256 one = _mm256_or_ps(_mm256_set1_ps(1.f), _mm256_and_ps(x, _mm256_set1_ps(-0.f)));    // 1 with x's sign
    return _mm256_add_ps(t, _mm256_and_ps(up, one));
}

static inline float max_of(__m256 x) {
    __m128 m = _mm_max_ps(_mm256_castps256_ps128(x), _mm256_extractf128_ps(x, 1));
    m = _mm_max_ps(m, _mm_movehl_ps(m, m));
    return _mm_cvtss_f32(_mm_max_ss(m, _mm_shuffle_ps(m, m, 1)));
}
static inline float min_of(__m256 x) {
    __m128 m = _mm_min_ps(_mm256_castps256_ps128(x), _mm256_extractf128_ps(x, 1));
    m = _mm_min_ps(m, _mm_movehl_ps(m, m));
    return _mm_cvtss_f32(_mm_min_ss(m, _mm_shuffle_ps(m, m, 1)));
}

// Weights that are checked and quantised together while they are in the first-level cache (16 KB, a whole number of blocks
// of every format); the quantising loops request the next chunk's lines as they go, so that main memory is read meanwhile.
constexpr int64_t kChunk = 4096;
template <int WEIGHTS>
static inline void prefetch_next(const float* src) {
    for (int i = 0; i < WEIGHTS; i += 16) _mm_prefetch(reinterpret_cast<const char*>(src + kChunk + i), _MM_HINT_T0);
}

// Is every one of n floats (a multiple of 8) finite?
static bool all_finite(const float* src, int64_t n) {
    const __m256i expo = _mm256_set1_epi32(0x7F800000);
    __m256i bad = _mm256_setzero_si256();
    for (int64_t i = 0; i < n; i += 8) {
        const __m256i b = _mm256_and_si256(_mm256_castps_si256(_mm256_loadu_ps(src + i)), expo);
        bad = _mm256_or_si256(bad, _mm256_cmpeq_epi32(b, expo));
    }
    return _mm256_testz_si256(bad, bad);
}

// A scale of zero or of normal size has a reciprocal that the vector form may use.
static inline bool plain_scale(float s) { return s == 0.f || std::fabs(s) >= 1.17549435e-38f; }

// Four vectors of small integers (0..255 or -128..127) to 32 bytes in order.
static inline __m256i pack32(__m256i a, __m256i b, __m256i c, __m256i d) {
    const __m256i ab = _mm256_packs_epi32(a, b), cd = _mm256_packs_epi32(c, d);
    const __m256i p = _mm256_packs_epi16(ab, cd);          // dwords a0 b0 c0 d0 | a1 b1 c1 d1
    return _mm256_permutevar8x32_epi32(p, _mm256_setr_epi32(0, 4, 1, 5, 2, 6, 3, 7));
}

// 16 nibble bytes {code j | code j + 16 << 4} of 32 codes below 16
static inline __m128i nibbles16(__m256i codes) {
    return _mm_or_si128(_mm256_castsi256_si128(codes), _mm_slli_epi16(_mm256_extracti128_si256(codes, 1), 4));
}

// Index of the first of 32 values that equals v (there is one).
static inline int first_equal(const __m256 (&x)[4], float v) {
    const __m256 w = _mm256_set1_ps(v);
    uint32_t m = 0;
    for (int i = 0; i < 4; ++i) m |= (uint32_t)_mm256_movemask_ps(_mm256_cmp_ps(x[i], w, _CMP_EQ_OQ)) << (8 * i);
    return __builtin_ctz(m);
}

static int rows_f16(const float* src, int64_t n, uint8_t* dst) {
    const __m128i expo = _mm_set1_epi16(0x7C00);
    __m128i bad = _mm_setzero_si128();
    for (int64_t i = 0; i < n; i += 8) {
        const __m128i h = _mm256_cvtps_ph(_mm256_loadu_ps(src + i), _MM_FROUND_TO_NEAREST_INT | _MM_FROUND_NO_EXC);
        bad = _mm_or_si128(bad, _mm_cmpeq_epi16(_mm_and_si128(h, expo), expo));
        _mm_storeu_si128(reinterpret_cast<__m128i*>(dst + 2 * i), h);
    }
    return _mm_testz_si128(bad, bad) ? LW_OK : LW_ERR_NONFINITE;
}

static int rows_q8_0(const float* src, int64_t n, uint8_t* dst) {
    for (int64_t blk = 0; blk * 32 < n; ++blk, src += 32, dst += 34) {
        prefetch_next<32>(src);
        __m256 x[4], m = _mm256_setzero_ps();
        for (int i = 0; i < 4; ++i) x[i] = _mm256_loadu_ps(src + 8 * i), m = _mm256_max_ps(m, abs8(x[i]));
        const float step = max_of(m) / 127.f;
        if (!plain_scale(step)) {
            if (const int rc = quantize_rows_q8_0(src, 32, dst)) return rc;
            continue;
        }
        const float inv = step != 0.f ? 1.f / step : 0.f;
        const uint16_t h = f32_to_f16_bits(step);
        if (is_inf_or_nan_half(h)) return LW_ERR_NONFINITE;
        put_half(dst, h);
        __m256i q[4];
        for (int i = 0; i < 4; ++i) q[i] = _mm256_cvttps_epi32(round8(_mm256_mul_ps(x[i], _mm256_set1_ps(inv))));
        _mm256_storeu_si256(reinterpret_cast<__m256i*>(dst + 2), pack32(q[0], q[1], q[2], q[3]));
    }
    return LW_OK;
}

// q4_0, q4_1, q5_0, q5_1
template <int BITS, bool OFFSET>
static int rows_legacy(const float* src, int64_t n, uint8_t* dst) {
    constexpr int kTop = (1 << BITS) - 1;
    constexpr int kBytes = 2 + (OFFSET ? 2 : 0) + (BITS == 5 ? 4 : 0) + 16;
    for (int64_t blk = 0; blk * 32 < n; ++blk, src += 32, dst += kBytes) {
        prefetch_next<32>(src);
        __m256 x[4];
        for (int i = 0; i < 4; ++i) x[i] = _mm256_loadu_ps(src + 8 * i);
        float step, lo = 0.f;
        if (OFFSET) {
            __m256 a = x[0], b = x[0];
            for (int i = 1; i < 4; ++i) a = _mm256_min_ps(a, x[i]), b = _mm256_max_ps(b, x[i]);
            lo = src[first_equal(x, min_of(a))];           // (the sign of a zero minimum is that of the first zero)
            step = (src[first_equal(x, max_of(b))] - lo) / (float)kTop;
        } else {
            __m256 y[4], m = _mm256_setzero_ps();
            for (int i = 0; i < 4; ++i) y[i] = abs8(x[i]), m = _mm256_max_ps(m, y[i]);
            constexpr float kHalf = (float)(1 << (BITS - 1));
            step = (src[first_equal(y, max_of(m))] + 0.f) / -kHalf;
        }
        if (!plain_scale(step)) {
            const int rc = BITS == 4 && !OFFSET ? quantize_rows_q4_0(src, 32, dst) : quantize_rows_legacy<BITS, OFFSET>(src, 32, dst);
            if (rc) return rc;
            continue;
        }
        const float inv = step != 0.f ? 1.f / step : 0.f;
        const uint16_t hd = f32_to_f16_bits(step), hm = OFFSET ? f32_to_f16_bits(lo) : 0;
        if (is_inf_or_nan_half(hd) || is_inf_or_nan_half(hm)) return LW_ERR_NONFINITE;
        __m256i q[4];
        for (int i = 0; i < 4; ++i) {
            __m256 v;
            if (OFFSET) v = _mm256_add_ps(_mm256_mul_ps(_mm256_sub_ps(x[i], _mm256_set1_ps(lo)), _mm256_set1_ps(inv)), _mm256_set1_ps(0.5f));
            else if (BITS == 4) v = _mm256_add_ps(_mm256_mul_ps(x[i], _mm256_set1_ps(inv)), _mm256_set1_ps(8.5f));
            else v = _mm256_add_ps(_mm256_add_ps(_mm256_mul_ps(x[i], _mm256_set1_ps(inv)), _mm256_set1_ps(16.f)), _mm256_set1_ps(0.5f));
            q[i] = _mm256_min_epi32(_mm256_cvttps_epi32(v), _mm256_set1_epi32(kTop));
        }
        const __m256i c = pack32(q[0], q[1], q[2], q[3]);
        uint8_t* p = dst;
        put_half(p, hd);
        p += 2;
        if (OFFSET) {
            put_half(p, hm);
            p += 2;
        }
        if (BITS == 5) {
            const uint32_t high = (uint32_t)_mm256_movemask_epi8(_mm256_slli_epi16(c, 3));      // bit 4 of every code
            std::memcpy(p, &high, 4);
            p += 4;
        }
        _mm_storeu_si128(reinterpret_cast<__m128i*>(p), nibbles16(_mm256_and_si256(c, _mm256_set1_epi8(15))));
    }
    return LW_OK;
}

// Largest (smallest) of each of eight rows of eight.
template <class Op>
static inline __m256 fold8(const __m256 (&r)[8], Op op) {
    __m256 t[4];
    for (int i = 0; i < 4; ++i)       // lanes: {r 2i even pairs, r 2i+1 ..}
        t[i] = op(_mm256_unpacklo_ps(r[2 * i], r[2 * i + 1]), _mm256_unpackhi_ps(r[2 * i], r[2 * i + 1]));      // a0 b0 a1 b1 | ..
    __m256 u[2];
    for (int i = 0; i < 2; ++i)
        u[i] = op(_mm256_shuffle_ps(t[2 * i], t[2 * i + 1], 0x44), _mm256_shuffle_ps(t[2 * i], t[2 * i + 1], 0xEE));   // a b c d | a b c d
    const __m256 lo = _mm256_permute2f128_ps(u[0], u[1], 0x20), hi = _mm256_permute2f128_ps(u[0], u[1], 0x31);
    return op(lo, hi);
}
struct Max8 {
    __m256 operator()(__m256 a, __m256 b) const { return _mm256_max_ps(a, b); }
};
struct Min8 {
    __m256 operator()(__m256 a, __m256 b) const { return _mm256_min_ps(a, b); }
};

// round(v / d) clamped to 0 .. top, zero where d is zero
static inline __m256i scale_codes(__m256 v, float d, float top) {
    if (d == 0.f) return _mm256_setzero_si256();
    return _mm256_cvttps_epi32(_mm256_min_ps(round8(_mm256_div_ps(v, _mm256_set1_ps(d))), _mm256_set1_ps(top)));
}
// round((x + m) / d) clamped to 0 .. top
static inline __m256i affine_codes(__m256 x, __m256 m, __m256 d, __m256 top) {
    const __m256 r = round8(_mm256_div_ps(_mm256_add_ps(x, m), d));
    return _mm256_cvttps_epi32(_mm256_min_ps(_mm256_max_ps(r, _mm256_setzero_ps()), top));
}

// q4_K and q5_K
template <bool FIVE>
static int rows_k45(const float* src, int64_t n, uint8_t* dst) {
    constexpr int kBytes = FIVE ? 176 : 144;
    constexpr float kTop = FIVE ? 31.f : 15.f;
    for (int64_t sb = 0; sb * 256 < n; ++sb, src += 256, dst += kBytes) {
        prefetch_next<256>(src);
        __m256 mn8[8], mx8[8];
        for (int s = 0; s < 8; ++s) {
            const __m256 a = _mm256_loadu_ps(src + 32 * s), b = _mm256_loadu_ps(src + 32 * s + 8);
            const __m256 c = _mm256_loadu_ps(src + 32 * s + 16), d = _mm256_loadu_ps(src + 32 * s + 24);
            mn8[s] = _mm256_min_ps(_mm256_min_ps(a, b), _mm256_min_ps(c, d));
            mx8[s] = _mm256_max_ps(_mm256_max_ps(a, b), _mm256_max_ps(c, d));
        }
        const __m256 lo = _mm256_min_ps(fold8(mn8, Min8()), _mm256_setzero_ps());
        const __m256 hi = _mm256_max_ps(fold8(mx8, Max8()), lo);
        const __m256 step = _mm256_div_ps(_mm256_sub_ps(hi, lo), _mm256_set1_ps(kTop));
        const __m256 offs = _mm256_xor_ps(lo, _mm256_set1_ps(-0.f));
        const uint16_t hd = f32_to_f16_bits(std::fabs(max_of(step)) / 63.f), hm = f32_to_f16_bits(std::fabs(max_of(offs)) / 63.f);   // (a zero is +0)
        if (is_inf_or_nan_half(hd) || is_inf_or_nan_half(hm)) return LW_ERR_NONFINITE;
        const float d = f16_bits_to_f32(hd), dmin = f16_bits_to_f32(hm);
        put_half(dst, hd);
        put_half(dst + 2, hm);
        const __m256i sc8 = scale_codes(step, d, 63.f), mn_8 = scale_codes(offs, dmin, 63.f);
        alignas(32) uint32_t sc[8], mn[8];
        alignas(32) float dl[8], ml[8];
        _mm256_store_si256(reinterpret_cast<__m256i*>(sc), sc8);
        _mm256_store_si256(reinterpret_cast<__m256i*>(mn), mn_8);
        _mm256_store_ps(dl, _mm256_mul_ps(_mm256_set1_ps(d), _mm256_cvtepi32_ps(sc8)));
        _mm256_store_ps(ml, _mm256_mul_ps(_mm256_set1_ps(dmin), _mm256_cvtepi32_ps(mn_8)));
        uint8_t* packed = dst + 4;
        for (int j = 0; j < 4; ++j) {
            packed[j] = (uint8_t)(sc[j] | ((sc[j + 4] >> 4) << 6));
            packed[4 + j] = (uint8_t)(mn[j] | ((mn[j + 4] >> 4) << 6));
            packed[8 + j] = (uint8_t)((sc[j + 4] & 15u) | ((mn[j + 4] & 15u) << 4));
        }
        __m256i high = _mm256_setzero_si256();               // q5_K: fifth bits of the eight sub-blocks, bit s of byte l
        for (int g = 0; g < 4; ++g) {
            __m256i c[2];
            for (int h = 0; h < 2; ++h) {
                const int s = 2 * g + h;
                if (dl[s] == 0.f) {
                    c[h] = _mm256_setzero_si256();
                    continue;
                }
                const __m256 m = _mm256_set1_ps(ml[s]), dv = _mm256_set1_ps(dl[s]), top = _mm256_set1_ps(kTop);
                __m256i q[4];
                for (int i = 0; i < 4; ++i) q[i] = affine_codes(_mm256_loadu_ps(src + 32 * s + 8 * i), m, dv, top);
                c[h] = pack32(q[0], q[1], q[2], q[3]);
                if (FIVE) {
                    const __m256i bit = _mm256_and_si256(_mm256_srli_epi16(c[h], 4), _mm256_set1_epi8(1));
                    high = _mm256_or_si256(high, _mm256_and_si256(_mm256_sll_epi16(bit, _mm_cvtsi32_si128(s)), _mm256_set1_epi8((char)(1 << s))));
                    c[h] = _mm256_and_si256(c[h], _mm256_set1_epi8(15));
                }
            }
            _mm256_storeu_si256(reinterpret_cast<__m256i*>(dst + (FIVE ? 48 : 16) + 32 * g), _mm256_or_si256(c[0], _mm256_slli_epi16(c[1], 4)));
        }
        if (FIVE) _mm256_storeu_si256(reinterpret_cast<__m256i*>(dst + 16), high);
    }
    return LW_OK;
}

static int rows_q2_K(const float* src, int64_t n, uint8_t* dst) {
    for (int64_t sb = 0; sb * 256 < n; ++sb, src += 256, dst += 84) {
        prefetch_next<256>(src);
        __m256 lo[2], hi[2], step[2], offs[2];
        for (int h = 0; h < 2; ++h) {
            __m256 mn8[8], mx8[8];
            for (int t = 0; t < 8; ++t) {
                const __m256 a = _mm256_loadu_ps(src + 128 * h + 16 * t), b = _mm256_loadu_ps(src + 128 * h + 16 * t + 8);
                mn8[t] = _mm256_min_ps(a, b);
                mx8[t] = _mm256_max_ps(a, b);
            }
            lo[h] = _mm256_min_ps(fold8(mn8, Min8()), _mm256_setzero_ps());
            hi[h] = _mm256_max_ps(fold8(mx8, Max8()), lo[h]);
            step[h] = _mm256_div_ps(_mm256_sub_ps(hi[h], lo[h]), _mm256_set1_ps(3.f));
            offs[h] = _mm256_xor_ps(lo[h], _mm256_set1_ps(-0.f));
        }
        const uint16_t hd = f32_to_f16_bits(std::fabs(max_of(_mm256_max_ps(step[0], step[1]))) / 15.f);
        const uint16_t hm = f32_to_f16_bits(std::fabs(max_of(_mm256_max_ps(offs[0], offs[1]))) / 15.f);
        if (is_inf_or_nan_half(hd) || is_inf_or_nan_half(hm)) return LW_ERR_NONFINITE;
        const float d = f16_bits_to_f32(hd), dmin = f16_bits_to_f32(hm);
        put_half(dst + 80, hd);
        put_half(dst + 82, hm);
        alignas(32) uint32_t sc[16], mn[16];
        alignas(32) float dl[16], ml[16];
        for (int h = 0; h < 2; ++h) {
            const __m256i s = scale_codes(step[h], d, 15.f), m = scale_codes(offs[h], dmin, 15.f);
            _mm256_store_si256(reinterpret_cast<__m256i*>(sc + 8 * h), s);
            _mm256_store_si256(reinterpret_cast<__m256i*>(mn + 8 * h), m);
            _mm256_store_ps(dl + 8 * h, _mm256_mul_ps(_mm256_set1_ps(d), _mm256_cvtepi32_ps(s)));
            _mm256_store_ps(ml + 8 * h, _mm256_mul_ps(_mm256_set1_ps(dmin), _mm256_cvtepi32_ps(m)));
        }
        for (int t = 0; t < 16; ++t) dst[t] = (uint8_t)(sc[t] | (mn[t] << 4));
        for (int half = 0; half < 2; ++half) {
            __m256i bytes = _mm256_setzero_si256();
            for (int quarter = 0; quarter < 4; ++quarter) {      // runs 8 half + 2 quarter and + 1: weights 128 half + 32 quarter ..
                __m256i q[4];
                for (int i = 0; i < 4; ++i) {
                    const int t = 8 * half + 2 * quarter + (i >> 1);
                    q[i] = dl[t] != 0.f ? affine_codes(_mm256_loadu_ps(src + 128 * half + 32 * quarter + 8 * i), _mm256_set1_ps(ml[t]),
                                                       _mm256_set1_ps(dl[t]), _mm256_set1_ps(3.f))
                                        : _mm256_setzero_si256();
                }
                bytes = _mm256_or_si256(bytes, _mm256_sll_epi16(pack32(q[0], q[1], q[2], q[3]), _mm_cvtsi32_si128(2 * quarter)));
            }
            _mm256_storeu_si256(reinterpret_cast<__m256i*>(dst + 16 + 32 * half), bytes);
        }
    }
    return LW_OK;
}

static int rows_q6_K(const float* src, int64_t n, uint8_t* dst) {
    for (int64_t sb = 0; sb * 256 < n; ++sb, src += 256, dst += 210) {
        prefetch_next<256>(src);
        alignas(32) float step[16], e[16];
        float largest = 0.f;
        for (int t = 0; t < 16; ++t) {
            const __m256 a = _mm256_loadu_ps(src + 16 * t), b = _mm256_loadu_ps(src + 16 * t + 8), fa = abs8(a), fb = abs8(b);
            const float mag = max_of(_mm256_max_ps(fa, fb));
            const __m256 w = _mm256_set1_ps(mag);
            const int at = __builtin_ctz((unsigned)_mm256_movemask_ps(_mm256_cmp_ps(fa, w, _CMP_EQ_OQ)) |
                                         (unsigned)_mm256_movemask_ps(_mm256_cmp_ps(fb, w, _CMP_EQ_OQ)) << 8);
            const float extreme = mag != 0.f ? src[16 * t + at] : 0.f;      // the first of equal magnitudes
            step[t] = extreme / -32.f;
            if (std::fabs(step[t]) > largest) largest = std::fabs(step[t]);
        }
        const uint16_t hd = f32_to_f16_bits(largest / 127.f);
        if (is_inf_or_nan_half(hd)) return LW_ERR_NONFINITE;
        const float d = f16_bits_to_f32(hd);
        __m256i sc8[2];
        bool plain = d != 0.f;
        for (int h = 0; h < 2 && plain; ++h) {
            const __m256 r = round8(_mm256_div_ps(_mm256_load_ps(step + 8 * h), _mm256_set1_ps(d)));
            const __m256 c = _mm256_max_ps(_mm256_min_ps(r, _mm256_set1_ps(127.f)), _mm256_set1_ps(-127.f));
            sc8[h] = _mm256_cvttps_epi32(c);
            _mm256_store_ps(e + 8 * h, _mm256_mul_ps(_mm256_set1_ps(d), _mm256_cvtepi32_ps(sc8[h])));
        }
        if (!plain) {
            // (largest / 127 below half the smallest fp16: every step is tiny; the scalar form decides)
            if (const int rc = quantize_rows_q6_K(src, 256, dst)) return rc;
            continue;
        }
        put_half(dst + 208, hd);
        const __m256i s16 = _mm256_permute4x64_epi64(_mm256_packs_epi32(sc8[0], sc8[1]), 0xD8);
        _mm_storeu_si128(reinterpret_cast<__m128i*>(dst + 192),
                         _mm_packs_epi16(_mm256_castsi256_si128(s16), _mm256_extracti128_si256(s16, 1)));
        for (int half = 0; half < 2; ++half) {
            __m256i low[2] = {_mm256_setzero_si256(), _mm256_setzero_si256()}, high = _mm256_setzero_si256();
            for (int quarter = 0; quarter < 4; ++quarter) {
                __m256i q[4];
                for (int i = 0; i < 4; ++i) {
                    const int t = 8 * half + 2 * quarter + (i >> 1);
                    if (e[t] == 0.f) {
                        q[i] = _mm256_set1_epi32(32);
                        continue;
                    }
                    // |x / e| <= 33: e is the run's step to half a unit of its scale, or the scale is 127 of the largest
                    const __m256 r = round8(_mm256_div_ps(_mm256_loadu_ps(src + 128 * half + 32 * quarter + 8 * i), _mm256_set1_ps(e[t])));
                    const __m256 k = _mm256_min_ps(_mm256_max_ps(r, _mm256_set1_ps(-32.f)), _mm256_set1_ps(31.f));
                    q[i] = _mm256_add_epi32(_mm256_cvttps_epi32(k), _mm256_set1_epi32(32));
                }
                const __m256i c = pack32(q[0], q[1], q[2], q[3]);
                const __m256i nib = _mm256_and_si256(c, _mm256_set1_epi8(15));
                low[quarter & 1] = _mm256_or_si256(low[quarter & 1], quarter < 2 ? nib : _mm256_slli_epi16(nib, 4));
                const __m256i up = _mm256_and_si256(_mm256_srli_epi16(c, 4), _mm256_set1_epi8(3));
                high = _mm256_or_si256(high, _mm256_sll_epi16(up, _mm_cvtsi32_si128(2 * quarter)));
            }
            _mm256_storeu_si256(reinterpret_cast<__m256i*>(dst + 64 * half), low[0]);
            _mm256_storeu_si256(reinterpret_cast<__m256i*>(dst + 64 * half + 32), low[1]);
            _mm256_storeu_si256(reinterpret_cast<__m256i*>(dst + 128 + 32 * half), high);
        }
    }
    return LW_OK;
}

static int quantize_chunks(int fmt, const float* src, int64_t n, uint8_t* dst, bool check) {
    for (int64_t at = 0; at < n; at += kChunk) {
        const int64_t m = n - at < kChunk ? n - at : kChunk;
        const float* s = src + at;
        uint8_t* d = dst + lw_row_bytes(fmt, kChunk) * (size_t)(at / kChunk);
        if (check && !all_finite(s, m)) return LW_ERR_NONFINITE;
        int rc = LW_ERR_FORMAT;
        switch (fmt) {
            case LW_F16: rc = rows_f16(s, m, d); break;
            case LW_Q8_0: rc = rows_q8_0(s, m, d); break;
            case LW_Q4_0: rc = rows_legacy<4, false>(s, m, d); break;
            case LW_Q4_1: rc = rows_legacy<4, true>(s, m, d); break;
            case LW_Q5_0: rc = rows_legacy<5, false>(s, m, d); break;
            case LW_Q5_1: rc = rows_legacy<5, true>(s, m, d); break;
            case LW_Q4_K: rc = rows_k45<false>(s, m, d); break;
            case LW_Q5_K: rc = rows_k45<true>(s, m, d); break;
            case LW_Q2_K: rc = rows_q2_K(s, m, d); break;
            case LW_Q6_K: rc = rows_q6_K(s, m, d); break;
        }
        if (rc != LW_OK) return rc;
    }
    return LW_OK;
}

// A non-finite weight anywhere leaves dst as it is.  The blocks go to a buffer and are copied when all of them are made, so that
// main memory is read once (4 Mi weights: q4_K 3.6 -> 3.8 ms).  For f16, whose blocks are half as large as the weights, above
// kHeldMost, or without the buffer, all weights are looked over first (q4_K 3.6 -> 4.6 ms).
constexpr size_t kHeldMost = (size_t)32 << 20;
static int quantize(int fmt, const float* src, int64_t n, uint8_t* dst) {
    const size_t bytes = lw_row_bytes(fmt, n);
    const bool hold = fmt != LW_F16 && bytes <= kHeldMost;
    const std::unique_ptr<uint8_t[]> held(hold ? new (std::nothrow) uint8_t[bytes] : nullptr);
    if (!held) return all_finite(src, n) ? quantize_chunks(fmt, src, n, dst, false) : LW_ERR_NONFINITE;
    const int rc = quantize_chunks(fmt, src, n, held.get(), true);
    if (rc == LW_OK) std::memcpy(dst, held.get(), bytes);
    return rc;
}

static bool available() {
    static const bool yes = __builtin_cpu_supports("avx2") && __builtin_cpu_supports("f16c");
    return yes;
}

}  // namespace v8
#pragma GCC pop_options
#endif

int quantize_host(int fmt, const float* src, int64_t n, void* dst) {
    if (!src || !dst) return LW_ERR_NULL;
    if (lw_block_elems(fmt) == 0) return LW_ERR_FORMAT;
    if (lw_row_bytes(fmt, n) == 0) return LW_ERR_SHAPE;
    uint8_t* out = static_cast<uint8_t*>(dst);
#ifdef LW_QUANTIZE_AVX2
    if (v8::available()) return v8::quantize(fmt, src, n, out);
#endif
    for (int64_t i = 0; i < n; ++i)
        if (!std::isfinite(src[i])) return LW_ERR_NONFINITE;
    switch (fmt) {
        case LW_F16: return quantize_rows_f16(src, n, out);
        case LW_Q8_0: return quantize_rows_q8_0(src, n, out);
        case LW_Q4_0: return quantize_rows_q4_0(src, n, out);
        case LW_Q4_K: return quantize_rows_q4_K(src, n, out);
        case LW_Q6_K: return quantize_rows_q6_K(src, n, out);
        case LW_Q5_K: return quantize_rows_q5_K(src, n, out);
        case LW_Q2_K: return quantize_rows_q2_K(src, n, out);
        case LW_Q4_1: return quantize_rows_legacy<4, true>(src, n, out);
        case LW_Q5_0: return quantize_rows_legacy<5, false>(src, n, out);
        case LW_Q5_1: return quantize_rows_legacy<5, true>(src, n, out);
    }
    return LW_ERR_FORMAT;
}

}  // namespace lw
