// aq_dequant: the dequantised matrix of Eq. 1, w = scale * q + min, evaluated
// in binary32 (the product is exact, so the sum is the only rounding) and
// rounded once to the output type.
//
// Bound: HBM traffic, (bits+1)/8 bytes read + sizeof(out) bytes written per
// weight.  One warp per fragment (16 rows x 128 k): the warp reads its
// fragment with 16-byte loads and writes row segments of 64 / 128 bytes, with an
// evict-first hint.  A CTA takes 64 rows x 256 k.  CTAs go along the rows, so that
// what is being written at one time is a few whole rows, and the slabs are counted
// through, so that an odd number of them leaves no warp idle; float32 rows of up
// to 3200 go down the columns, whose CTAs read what lies together, unless there is
// only one CTA per SM (3406 x 576 at 4 bits 4.8 us down, 4.2 along the rows).  Times of the
// kernel, us, down the columns without the hint / along the rows / down with the
// hint: binary16, 16384 x 8192 at 3 bits 63.2 / 56.5 (5.94 TB/s) / 63.7, 16384 x
// 3072 24.1 / 18.5 / 19.7, 15811 x 352 at 2 bits 4.48 / 4.10 / 4.48 (with pairs of
// slabs 4.83); float32, 16384 x 8192 142 / 136 / 142, 16384 x 4096 72.7 / 66.4 /
// 69.2, 2603 x 3104 11.3 / 11.7 / 11.1, 4899 x 2080 at 4 bits 13.4 / 14.1 / 13.3,
// 2220 x 1088 at 2 bits 4.8 / 6.2 / 4.8.
#include "aq_internal.h"
#include "aq_layout.cuh"

namespace aq {

template <typename T> struct OutVec;   // 8 consecutive output elements
template <> struct OutVec<__half> {
    uint4 v;
    __device__ __forceinline__ void set(const float* w) {
        __half2 a = __floats2half2_rn(w[0], w[1]), b = __floats2half2_rn(w[2], w[3]);
        __half2 c = __floats2half2_rn(w[4], w[5]), d = __floats2half2_rn(w[6], w[7]);
        v = make_uint4(*reinterpret_cast<uint32_t*>(&a), *reinterpret_cast<uint32_t*>(&b),
                       *reinterpret_cast<uint32_t*>(&c), *reinterpret_cast<uint32_t*>(&d));
    }
};
template <> struct OutVec<__nv_bfloat16> {
    uint4 v;
    __device__ __forceinline__ void set(const float* w) {
        __nv_bfloat162 a = __floats2bfloat162_rn(w[0], w[1]), b = __floats2bfloat162_rn(w[2], w[3]);
        __nv_bfloat162 c = __floats2bfloat162_rn(w[4], w[5]), d = __floats2bfloat162_rn(w[6], w[7]);
        v = make_uint4(*reinterpret_cast<uint32_t*>(&a), *reinterpret_cast<uint32_t*>(&b),
                       *reinterpret_cast<uint32_t*>(&c), *reinterpret_cast<uint32_t*>(&d));
    }
};

// lane (g,t): 8 decoded values of block j, row half hi
template <int BITS>
__device__ __forceinline__ void decode_unit(const SlotWords<BITS>& sw, const uint8_t* fb, int g, int j, int hi,
                                            float* w) {
    const __half2 dm = *reinterpret_cast<const __half2*>(fb + ((g + 8 * hi) * 4 + j) * 4);
    const float d = __low2float(dm), m = __high2float(dm);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        // the two codes as floats without a conversion: 2^23 + q has q in its low mantissa bits, and
        // (2^23 + q) - 2^23 is exact, so the value is the same as (float)q
        const uint32_t p = code_pair<BITS>(sw, j, hi, i, 0u);
        const float q0 = __uint_as_float((p & 0xffffu) | 0x4B000000u) - 8388608.f;
        const float q1 = __uint_as_float(__byte_perm(p, 0x4B000000u, 0x7632)) - 8388608.f;
        w[2 * i] = fmaf(d, q0, m);
        w[2 * i + 1] = fmaf(d, q1, m);
    }
}

// n: slabs of 128 k that exist (along the rows), groups of four row tiles (down the columns)
template <int BITS, typename T, bool DOWN>
__global__ void __launch_bounds__(256) dequant_kernel(const uint8_t* __restrict__ frags, int64_t N, int64_t K, int NT,
                                                      unsigned n, T* __restrict__ out) {
    constexpr int FB = frag_bytes(BITS);
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int warp = threadIdx.x >> 5;
    const unsigned at = DOWN ? blockIdx.x : 2 * blockIdx.x + (warp & 1), rest = at % n;
    const int64_t R = (int64_t)(DOWN ? rest : at / n) * 4 + (warp >> 1);
    const int64_t S = DOWN ? 2 * (int64_t)(at / n) + (warp & 1) : rest;
    if (R >= NT || S * 128 >= K) return;
    const uint8_t* fb = frags + frag_index(S, R, NT) * FB;
    LaneCodes<BITS> lc;
    load_lane_codes<BITS>(lc, fb, lane);
    SlotWords<BITS> sw;
    sw.gather(lc);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
        for (int hi = 0; hi < 2; ++hi) {
            float w[8];
            decode_unit<BITS>(sw, fb, g, j, hi, w);
            const int64_t row = R * 16 + g + 8 * hi;
            const int64_t k0 = S * 128 + 32 * j + 8 * t;
            if (row < N && k0 < K) {
                if constexpr (sizeof(T) == 4) {
                    float4* o = reinterpret_cast<float4*>(out + row * K + k0);
                    __stcs(o, make_float4(w[0], w[1], w[2], w[3]));
                    __stcs(o + 1, make_float4(w[4], w[5], w[6], w[7]));
                } else {
                    OutVec<T> ov;
                    ov.set(w);
                    __stcs(reinterpret_cast<uint4*>(out + row * K + k0), ov.v);
                }
            }
        }
    }
}

static int64_t slabs_of(const aq_handle_s* h) { return (h->K + 127) / 128; }
static int64_t groups_of(const aq_handle_s* h) { return (h->NT + 3) / 4; }

template <int BITS, typename T, bool DOWN>
static void launch_as(const aq_handle_s* h, void* out, cudaStream_t s) {
    const int64_t slabs = slabs_of(h), groups = groups_of(h);
    const unsigned grid = (unsigned)(DOWN ? (slabs + 1) / 2 * groups : (slabs * groups + 1) / 2);
    dequant_kernel<BITS, T, DOWN><<<grid, 256, 0, s>>>(h->frags, h->N, h->K, h->NT, (unsigned)(DOWN ? groups : slabs), (T*)out);
}

template <int BITS>
static cudaError_t launch_bits(const aq_handle_s* h, void* out, aq_dtype_t dt, cudaStream_t s) {
    if (dt == AQ_F16) launch_as<BITS, __half, false>(h, out, s);
    else if (dt == AQ_BF16) launch_as<BITS, __nv_bfloat16, false>(h, out, s);
    else if (h->K > 3200 || slabs_of(h) * groups_of(h) <= 2 * sm_count()) launch_as<BITS, float, false>(h, out, s);
    else launch_as<BITS, float, true>(h, out, s);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_dequant(const aq_handle_s* h, void* out, aq_dtype_t dt, cudaStream_t s) {
    switch (h->bits) {
        case 2: return launch_bits<2>(h, out, dt, s);
        case 3: return launch_bits<3>(h, out, dt, s);
        default: return launch_bits<4>(h, out, dt, s);
    }
}

}  // namespace aq
