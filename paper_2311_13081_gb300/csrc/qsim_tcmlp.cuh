// qsim_tcmlp.cuh -- tensor-core MLP passes of the learner (tcgen05), forward and backward, for
// a CTA that holds whole 128-sample tiles: in -> H -> H -> out with in <= 96, H in {32, 64,
// 128}, out <= 4.
//
// Every product runs as tcgen05.mma (M 128, kind::f16) on fp16 hi / lo halves of both
// operands (qsim_tcgen05.cuh), three products per K step of 16.  In all passes but FWD:
//  * operands are scaled by powers of two before the split, so that they use the halves' range
//    whatever their size: weights by network and layer (the image's exponents), inputs by 256
//    gathered samples, the first hidden layer and both deltas by a bound formed of those;
//  * the two small products of a chain come first and its K steps are spread over up to four
//    accumulators (added up in FP32), so that the tensor core's truncation of partial sums at
//    full size happens two to four times a chain;
//  * weight gradients are added up over tiles in FP32 outside the tensor memory.
// Gradients are then as close to 64 bits as the FP32 engines' were or closer (relative error of
// a whole gradient, geometric mean over 128 - 512 samples a CTA, five observation layouts and
// 16 seeds, FP32 engines / here: actor 2.3e-7 / 2.1e-7 at hidden 32, 2.9e-7 / 2.5e-7 at 64,
// 4.2e-7 / 3.8e-7 at 128; critics at 128 2.3e-7 / 1.7e-7; without the scaling and with one or
// two accumulators 3.1e-7, 3.8e-7, 7.1e-7 and 5.9e-7, and a weight column of an input of 1e-4
// lost all but two to four digits).
// FWD, the target networks' pass at hidden 32 and 64, keeps operands as they are (magnitudes
// below 65,504) and one chain: those bits feed the critics' FP32 regression.
//
// One layout serves both directions.  An operand lies as [row][column] in 8 x 8 core matrices
// (8 rows x 16 bytes), column groups 128 B apart, row groups KC x 128 B apart.  Read K-major
// it is an operand whose K runs along the columns (forward products, and dZ2 in dZ2 W2);
// read MN-major it is one whose K runs along the rows: the samples for the weight
// gradients (dW1^T = X^T dZ1, dW2^T = H1^T dZ2: the gradient's input index falls on the
// tensor-memory lanes, so the gradient leaves in coalesced rows), the output units for
// dZ2 W2.  Nothing is transposed or staged twice.
//
// Bound: latency of the chain MMA -> tensor-memory read -> split -> shared memory -> MMA with
// one CTA per SM (a chain of MMAs from one thread completes one every ~65 cycles; the parts
// of a product, issued by as many warps, run side by side).  256 samples at hidden 128 through
// one critic, forward and backward, in the first, unscaled form: 54 us, the SIMT engine 202.
// Scaling and the parts together cost 4 % of the batched training cases.
#pragma once
#include "qsim_smlp.cuh"
#include "qsim_tcgen05.cuh"

namespace qsim {
namespace tce {

constexpr int KP = 96, KC1 = KP / 8;  // input columns of a tile, zero-padded
constexpr int TR = 128;               // rows of a tile
constexpr int TILE_HALVES = TR * KP;  // one half (hi or lo) of an input tile
constexpr int TILE_FLOATS = TILE_HALVES;  // a tile in scratch: hi then lo
constexpr int TMEM_COLS = 512;
constexpr int TILES_X = 2;  // input tiles that share an exponent (a pass of the replay gather)
constexpr int DRAIN_POLLS = 1 << 24;

enum Mode { FWD, FWDX, CRIT, DQ, ACT };

// Shared memory of a pass, bytes.  At hidden 128 the forward-only pass holds W1, W2 and one
// half (64 columns) of H1; the backward passes hold all of H1, and W2 takes W1's place
// tile by tile.
template <int H, int MODE = CRIT>
struct Lay {
    static constexpr bool FW = MODE == FWD || MODE == FWDX;
    static constexpr bool WIDE = H == 128, HALVES = WIDE && FW, SHARE = WIDE && !FW;
    static constexpr int KC2 = H / 8;
    static constexpr int HC = HALVES ? 64 : H;  // columns of H1 held at once
    static constexpr int DH = WIDE ? 64 : H;    // columns of dZ2 held at once
    static constexpr int X = 0;
    static constexpr int W1 = X + 4 * TR * KP;
    static constexpr int W2 = SHARE ? W1 : W1 + 4 * H * KP;
    static constexpr int H1 = W2 + 4 * H * H;
    static constexpr int D2 = H1 + 4 * TR * HC;
    static constexpr int B1 = D2 + (FW ? 0 : 4 * TR * DH);
    static constexpr int B2 = B1 + 4 * H;
    static constexpr int W3 = B2 + 4 * H;
    static constexpr int B3 = W3 + 16 * H;
    static constexpr int RED = B3 + 16;    // 8 warp maxima, 16 weight maxima, 16 output-bias sums
    static constexpr int BAR = RED + 160;  // two mbarriers
    static constexpr int PART = BAR + 16;  // [2][128][4] partial outputs, then [H][4] action columns of W1; or
    static constexpr int SUMS = PART;      // [4][6][H] column sums of the 4 row groups
    static constexpr int END = PART + (96 * H > 4096 + 16 * H ? 96 * H : 4096 + 16 * H);
};
constexpr int lay_bytes() {
    int m = Lay<128, CRIT>::END;
    if (Lay<128, FWD>::END > m) m = Lay<128, FWD>::END;
    if (Lay<64, CRIT>::END > m) m = Lay<64, CRIT>::END;
    return m;
}
constexpr int SMEM_BYTES = lay_bytes();

// The halves of a network's W1 (zero-padded to 96 columns) and W2 as the passes read them:
// W1 hi | lo | W2 hi | lo.  Kept in the run's scratch for a launch: made of the weights when
// the launch starts on the run, and rewritten by every Adam and Polyak step, so that a pass
// loads them with 16-byte copies instead of splitting the weights again (9 passes an update).
__host__ __device__ constexpr int img_floats(int H) { return H * KP + H * H; }

__host__ __device__ constexpr bool shape_ok(int Bc, int H, int DA, int DC) {
    return Bc > 0 && Bc % TR == 0 && (H == 32 || H == 64 || H == 128) && DA <= KP && DC <= KP &&
           DA % 2 == 0 && DC % 2 == 0;
}

__device__ __forceinline__ float exp2i(int e) { return __int_as_float((e + 127) << 23); }
__device__ __forceinline__ int ilog2(float x) { return (int)((__float_as_uint(x) >> 23) & 255u) - 127; }

// Powers of two that operands are multiplied by before they are split, so that the halves keep
// their 22 bits whatever the values' size.  Exponents stay within +-60 each.
__device__ __forceinline__ int scale_to(int top, float log2_bound) {  // bound x 2^e <= 2^top
    const float e = (float)top - ceilf(log2_bound + 0.01f);
    return e > -1e9f && e < 1e9f ? (int)fminf(fmaxf(e, -60.0f), 60.0f) : 0;  // (zero, infinite, NaN: as it is)
}
__device__ __forceinline__ int scale_max(int top, float m) {  // 2^(top - 1) <= m 2^e < 2^top
    return m > 0.0f ? scale_to(top, (float)(ilog2(m) + 1) - 0.02f) : 0;
}
struct Pow2 {  // x 2^e, e the sum of two or three exponents
    float a;
    __device__ __forceinline__ explicit Pow2(int e) : a(exp2i(min(max(e, -120), 120))) {}
    __device__ __forceinline__ float operator()(float x) const { return x * a; }
};
// Inputs fill the halves' range (each gather picks their exponent anew); weights leave room to grow
// until their exponents are picked again.
constexpr int X_TOP = 15, W_TOP = 13;
// Exponents of a network's image: W1 and W2.
struct NetScale {
    int e1, e2;
};
constexpr float kScaleTop = 32768.0f, kScaleLow = 8.0f;  // an image's largest half outside: made again

// shared-memory descriptor: no swizzle, leading / stride byte offsets
__device__ __forceinline__ uint64_t sd(uint32_t addr, int lbo, int sbo) {
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) |
           ((uint64_t)1 << 46);
}
// An operand of KC column groups at `a`: K along the columns (K-major), or along the rows
// (MN-major).
template <bool MN>
__device__ __forceinline__ uint64_t op(uint32_t a, int kc) { return MN ? sd(a, kc * 128, 128) : sd(a, 128, kc * 128); }
template <bool TA, bool TB>
__host__ __device__ constexpr uint32_t idesc(int n) {
    return (1u << 4) | ((TA ? 1u : 0u) << 15) | ((TB ? 1u : 0u) << 16) | ((uint32_t)(n >> 3) << 17) |
           ((uint32_t)(TR >> 4) << 24);
}

// One chain D (+)= A B over KS K steps of operands with KCA and KCB column groups: the small
// products first (see the file header), or in FWD order, the three of a K step in a row.  Everything but the base addresses is a constant, so
// that the issuing lane does little more than issue.
template <bool TA, bool TB, int KCA, int KCB, int KS, bool ROW = false>
__device__ __forceinline__ void chain(uint32_t d, uint32_t ah, uint32_t al, uint32_t bh, uint32_t bl, uint32_t id,
                                      uint32_t acc) {
    const uint64_t dah = op<TA>(ah, KCA), dal = op<TA>(al, KCA), dbh = op<TB>(bh, KCB), dbl = op<TB>(bl, KCB);
    constexpr uint64_t sa = (TA ? 2 * KCA * 128 : 256) / 16, sb = (TB ? 2 * KCB * 128 : 256) / 16;
    if constexpr (ROW) {
#pragma unroll
        for (int j = 0; j < KS; ++j) {
            tc::mma_ss(d, dah + j * sa, dbh + j * sb, id, j ? 1u : acc);
            tc::mma_ss(d, dah + j * sa, dbl + j * sb, id, 1);
            tc::mma_ss(d, dal + j * sa, dbh + j * sb, id, 1);
        }
    } else {
#pragma unroll
        for (int j = 0; j < KS; ++j) {
            tc::mma_ss(d, dah + j * sa, dbl + j * sb, id, j ? 1u : acc);
            tc::mma_ss(d, dal + j * sa, dbh + j * sb, id, 1);
        }
#pragma unroll
        for (int j = 0; j < KS; ++j) tc::mma_ss(d, dah + j * sa, dbh + j * sb, id, 1);
    }
}

// A product's K steps as one chain, or (two accumulators, dcols columns apart) as two halves
// that two warps issue side by side: a chain completes one MMA per ~65 cycles, two of them
// one per ~33.  Part w of PARTS = 2 (the first or second half of the K steps) or the whole.
template <bool TA, bool TB, int PARTS, int KCA, int KCB, int KS, bool ROW = false>
__device__ __forceinline__ void chain_part(int w, uint32_t d, int dcols, uint32_t ah, uint32_t al, uint32_t bh, uint32_t bl,
                                           uint32_t id, uint32_t acc) {
    constexpr uint32_t sa = (KS / PARTS) * (TA ? 2 * KCA * 128 : 256), sb = (KS / PARTS) * (TB ? 2 * KCB * 128 : 256);
    const uint32_t oa = (uint32_t)w * sa, ob = (uint32_t)w * sb;
    chain<TA, TB, KCA, KCB, KS / PARTS, ROW>(d + (uint32_t)(w * dcols), ah + oa, al + oa, bh + ob, bl + ob, id, acc);
}

// 16 columns of a product: the sum of its parts' accumulators, added in FP32.
template <int PARTS>
__device__ __forceinline__ void ld_acc(uint32_t t, int dcols, float* x) {
    uint32_t v[16], w[16];
    if constexpr (PARTS == 1) tc::ld16(t, v);
    else tc::ld16x2(t, v, t + (uint32_t)dcols, w);
#pragma unroll
    for (int e = 0; e < 16; ++e) x[e] = PARTS == 1 ? __uint_as_float(v[e]) : __uint_as_float(v[e]) + __uint_as_float(w[e]);
    if constexpr (PARTS == 3) {
        tc::ld16(t + (uint32_t)(2 * dcols), v);
#pragma unroll
        for (int e = 0; e < 16; ++e) x[e] += __uint_as_float(v[e]);
    }
    if constexpr (PARTS == 4) {
        tc::ld16x2(t + (uint32_t)(2 * dcols), v, t + (uint32_t)(3 * dcols), w);
#pragma unroll
        for (int e = 0; e < 16; ++e) x[e] += __uint_as_float(v[e]) + __uint_as_float(w[e]);
    }
}

// Column sums over a warp's 32 lanes of N columns held per lane: column lane / (32 / N).
template <int N>
__device__ __forceinline__ float colsum(const float* v) {
    const int lane = threadIdx.x & 31;
    float t[N];
#pragma unroll
    for (int i = 0; i < N; ++i) t[i] = v[i];
    int o = 16;
#pragma unroll
    for (int n = N; n > 1; n >>= 1) {
        const bool hi = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < n / 2; ++i) {
            const float send = hi ? t[i] : t[i + n / 2], keep = hi ? t[i + n / 2] : t[i];
            t[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
        o >>= 1;
    }
    float r = t[0];
    for (; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    return r;
}

// A network's image and the exact divisions by its shape (indices below 2^24).
struct Img {
    unsigned char* p = nullptr;
    int in = 0, H = 0;
    uint32_t mi = 0, mh = 0;
    float s1 = 1.0f, s2 = 1.0f;
    __device__ __forceinline__ Img() {}
    __device__ __forceinline__ Img(unsigned char* q, int in_, int H_, NetScale sc)
        : p(q), in(in_), H(H_), mi(0xffffffffu / (uint32_t)in_ + 1u), mh(0xffffffffu / (uint32_t)H_ + 1u),
          s1(exp2i(sc.e1)), s2(exp2i(sc.e2)) {}
    // Byte offset of parameter i (flat index) in the hi half, the distance to its lo half and
    // its scale; false for biases and the output layer.
    __device__ __forceinline__ bool at(int i, int& o, int& lo, float& s) const {
        if (i < H * in) {
            const int j = (int)__umulhi((uint32_t)i, mi);
            o = 2 * tc::cano16(j, i - j * in, KC1);
            lo = 2 * H * KP;
            s = s1;
            return true;
        }
        i -= H * in + H;
        if (i < 0 || i >= H * H) return false;
        const int j = (int)__umulhi((uint32_t)i, mh);
        o = 4 * H * KP + 2 * tc::cano16(j, i - j * H, H / 8);
        lo = 2 * H * H;
        s = s2;
        return true;
    }
    // Parameters i (and i + 1 when two; i even then, so both lie in one row).
    __device__ __forceinline__ void put(int i, float v, float w, bool two) const {
        int o, lo;
        float s;
        if (!at(i, o, lo, s)) return;
        uint32_t h, l;
        tc::split2(v * s, w * s, h, l);
        if (two) {
            *reinterpret_cast<uint32_t*>(p + o) = h;
            *reinterpret_cast<uint32_t*>(p + o + lo) = l;
        } else {
            *reinterpret_cast<uint16_t*>(p + o) = (uint16_t)h;
            *reinterpret_cast<uint16_t*>(p + o + lo) = (uint16_t)l;
        }
    }
    // One value per lane, consecutive lanes consecutive parameters (all lanes call; the ones
    // with i >= hi store nothing): pairs leave as 4 bytes.
    __device__ __forceinline__ void put_lanes(int i, int hi, float v) const {
        const int lane = threadIdx.x & 31;
        const float w = __shfl_down_sync(0xffffffffu, v, 1);
        if (i >= hi) return;
        const bool two = lane < 31 && i + 1 < hi;
        if ((i & 1) == 0) put(i, v, w, two);
        else if (lane == 0) put(i, v, 0.0f, false);
    }
};

// The whole image of a network (one CTA), 8 columns of a row per thread.
__device__ __noinline__ void img_make(unsigned char* img, const float* W, int in, int H, NetScale sc) {
    auto rows = [&](const float* src, int cols, int kc, unsigned char* hi, unsigned char* lo, float s) {
        for (int i = threadIdx.x; i < H * kc; i += LT) {
            const int j = i / kc, k0 = 8 * (i - j * kc);
            float v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = k0 + e < cols ? s * ldcg(src + (size_t)j * cols + k0 + e) : 0.0f;
            uint32_t h[4], l[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) tc::split2(v[2 * e], v[2 * e + 1], h[e], l[e]);
            const int o = 2 * tc::cano16(j, k0, kc);
            *reinterpret_cast<uint4*>(hi + o) = make_uint4(h[0], h[1], h[2], h[3]);
            *reinterpret_cast<uint4*>(lo + o) = make_uint4(l[0], l[1], l[2], l[3]);
        }
    };
    rows(W, in, KC1, img, img + 2 * H * KP, exp2i(sc.e1));
    rows(W + H * in + H, H, H / 8, img + 4 * H * KP, img + 4 * H * KP + 2 * H * H, exp2i(sc.e2));
}

__device__ __forceinline__ void copy16(uint32_t dst, const unsigned char* src, int bytes) {
    for (int i = 16 * threadIdx.x; i < bytes; i += 16 * LT)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(dst + (uint32_t)i), "l"(src + i) : "memory");
}

// Largest magnitude among N halves (16-byte aligned) that this thread reads.
template <int N>
__device__ __forceinline__ float max_half(const unsigned char* p) {
    constexpr int PER = N / 8 / LT, REST = N / 8 - PER * LT;
    __half2 m = __float2half2_rn(0.0f);
    auto take = [&](const uint4& v) {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) m = __hmax2(m, __habs2(*reinterpret_cast<const __half2*>(&w[e])));
    };
    const uint4* q = reinterpret_cast<const uint4*>(p) + threadIdx.x;
    uint4 v[PER + 1];
#pragma unroll
    for (int i = 0; i < PER; ++i) v[i] = __ldcg(q + i * LT);
    if (REST && threadIdx.x < REST) v[PER] = __ldcg(q + PER * LT);
#pragma unroll
    for (int i = 0; i < PER; ++i) take(v[i]);
    if (REST && threadIdx.x < REST) take(v[PER]);
    return fmaxf(__low2float(m), __high2float(m));
}

// The FP32 value of one unit's pre-activation as the SIMT engine forms it (products added in
// input order, then the bias).  A critic's regression takes the ReLU's sign from it where
// the tensor cores' value lies too close to zero to tell, so that the same units pass as in
// FP32: a unit on the other side of zero moves a gradient by a sample's share.  A heuristic
// band, not a bound: kBand x (largest weight) x (sum of the inputs' magnitudes), the sum of
// the largest errors of the two sums over 65,536 units of learner-like inputs and weights
// (FP32 in input order 1.1e-7 of that product, scaled halves 3.8e-8; root mean squares
// 1.3e-8 and 7e-9).  Some 3 units in 10^6 fall into it.  The second layer's adds the first's:
// over H units of root-mean-square weight max / sqrt(3), five times the root mean square
// comes to about 0.25 sqrt(H) max|W2| of the first layer's band.
constexpr float kBand = 1.5e-7f;
__device__ __noinline__ float exact_unit1(const float* W, int in, const float* xrow, const float* bias, int j) {
    float z = 0.0f;
    const float* w = W + (size_t)j * in;
#pragma unroll 1
    for (int k0 = 0; k0 < in; k0 += 8) {  // 16 loads in flight
        float x[8], v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int k = min(k0 + e, in - 1);
            x[e] = ldcg(xrow + k);
            v[e] = ldcg(w + k);
        }
#pragma unroll
        for (int e = 0; e < 8; ++e)
            if (k0 + e < in) z = fmaf(x[e], v[e], z);
    }
    return z + ldcg(bias + j);
}
// The same for a unit of the second layer, by a whole warp: its lanes form the row's first
// layer, then its units' products are added in order.
template <int H>
__device__ __noinline__ float exact_unit2(const float* W, int in, const float* xrow, int j) {
    const int lane = threadIdx.x & 31;
    const float* b1 = W + (size_t)H * in;
    const float* W2 = b1 + H;
    float z2 = 0.0f;
#pragma unroll 1
    for (int u = 0; u < H; u += 32) {  // this lane's unit u + lane of the first layer
        const float* w = W + (size_t)(u + lane) * in;
        const float w2 = ldcg(W2 + (size_t)j * H + u + lane);
        float z = 0.0f;
#pragma unroll 1
        for (int k0 = 0; k0 < in; k0 += 16) {
            float v[16];
            const float x = ldcg(xrow + min(k0 + (lane & 15), in - 1));
#pragma unroll
            for (int k = 0; k < 16; ++k) v[k] = ldcg(w + min(k0 + k, in - 1));
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const float xk = __shfl_sync(0xffffffffu, x, k);
                if (k0 + k < in) z = fmaf(xk, v[k], z);
            }
        }
        z = fmaxf(z + ldcg(b1 + u + lane), 0.0f);
        for (int k = 0; k < 32; ++k)
            z2 = fmaf(__shfl_sync(0xffffffffu, z, k), __shfl_sync(0xffffffffu, w2, k), z2);
    }
    return z2 + ldcg(W2 + H * H + j);
}

// 8 values of row r, columns c0 .. c0 + 7, as hi / lo halves
__device__ __forceinline__ void put8(unsigned char* hi, unsigned char* lo, int kc, int r, int c0, const float* v) {
    uint32_t h[4], l[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) tc::split2(v[2 * e], v[2 * e + 1], h[e], l[e]);
    const int at = 2 * tc::cano16(r, c0, kc);
    *reinterpret_cast<uint4*>(hi + at) = make_uint4(h[0], h[1], h[2], h[3]);
    *reinterpret_cast<uint4*>(lo + at) = make_uint4(l[0], l[1], l[2], l[3]);
}

struct Args {
    const float* W;  // W1[H][in] b1 W2[H][H] b2 W3[out][H] b3
    int in, out;
    const float* X;  // input tiles (hi / lo halves), Bc / 128 of them
    int Bc;
    float* Y;        // FWD: outputs [Bc][out]
    bool tanh_out;
    const float* y;  // CRIT: regression targets [Bc]
    float invB;
    float* G;        // CRIT, ACT: gradient in the layout of W
    const float* mu; // DQ: actions that take the input's last 4 columns [Bc][4]
    float* da;       // DQ: out, dLoss/d(actor pre-activation) [Bc][4]; ACT: in
    const unsigned char* img;  // halves of W1 and W2
    // (all but FWD:) their exponents and largest magnitudes; the exponents of the input tiles,
    // one for every TILES_X of them
    NetScale e;
    float w1m, w2m;
    const int* xe;
    int limit;    // polls of a wait before it gives up
    int* dead;    // shared flag: a wait of this CTA gave up (what the passes left is not to be used)
    const float* x32;  // CRIT: the FP32 inputs [Bc][in] and each row's sum of magnitudes [Bc]
    const float* xn;
};

// One network pass over the CTA's tiles.  FWD and FWDX: outputs only; FWD takes operands as they
// are and adds the three products of a K step in a row into one accumulator.  CRIT: squared-error gradient of a
// critic, returns this thread's part of the mean squared error.  DQ: -mean Q of a critic at
// actions mu, gradient with respect to the actor's pre-activations; returns this thread's
// part of -mean Q.  ACT: parameter gradient of the actor from da.
template <int H, int MODE>
__device__ __noinline__ float pass(const Args& a, float* sm, uint32_t tmem, int* status) {
    using L = Lay<H, MODE>;
    constexpr int KC2 = L::KC2, KCH = L::HC / 8, NC = H / 2, KCD = L::DH / 8;
    constexpr bool FW = L::FW, SC = MODE != FWD;  // outputs only; scaled operands
    constexpr bool ROW = MODE == FWD;
    constexpr bool WG = MODE == CRIT || MODE == ACT, BWD = !FW;
    // Accumulators (H columns each) that a product is spread over: the fewer of its K steps
    // add up in one, the less the tensor core truncates.  Layer 1 and 2 forward, dZ1,
    // weight gradients.
    constexpr int P1 = !SC ? 1 : (L::HALVES ? 2 : 3), P2 = !SC ? 1 : (H == 32 ? 2 : 4);
    constexpr int PB = H == 64 || (H == 128 && !WG) ? 4 : 2, PG = H == 128 ? 2 : 4;
    constexpr int NB = SC ? 4 : 1;  // arrivals a barrier phase
    constexpr int OUT = MODE == CRIT || MODE == DQ ? 1 : 4;  // forward only: 1 or 4 (a.out)
    unsigned char* sb = reinterpret_cast<unsigned char*>(sm);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int r = 32 * (warp & 3) + lane, half = warp >> 2, cb = half * NC;  // this thread's row and columns
    const int in = a.in, out = FW ? a.out : OUT;
    unsigned char *Xh = sb + L::X, *Xl = Xh + 2 * TILE_HALVES;
    unsigned char *W1h = sb + L::W1, *W1l = W1h + 2 * H * KP, *W2h = sb + L::W2, *W2l = W2h + 2 * H * H;
    unsigned char *H1h = sb + L::H1, *H1l = H1h + 2 * TR * L::HC, *D2h = sb + L::D2, *D2l = D2h + 2 * TR * L::DH;
    float* b1 = reinterpret_cast<float*>(sb + L::B1);
    float* b2 = reinterpret_cast<float*>(sb + L::B2);
    float* W3 = reinterpret_cast<float*>(sb + L::W3);
    float* b3 = reinterpret_cast<float*>(sb + L::B3);
    float* red = reinterpret_cast<float*>(sb + L::RED);
    float* part = reinterpret_cast<float*>(sb + L::PART);
    float* w1a = part + 1024;  // DQ: [H][4], W1's action columns
    float* sums = reinterpret_cast<float*>(sb + L::SUMS);
    const uint32_t bar0 = tc::smem_u32(sb + L::BAR), bar1 = bar0 + 8;
    const uint32_t uXh = tc::smem_u32(Xh), uXl = tc::smem_u32(Xl), uW1h = tc::smem_u32(W1h), uW1l = tc::smem_u32(W1l),
                   uW2h = tc::smem_u32(W2h), uW2l = tc::smem_u32(W2l), uH1h = tc::smem_u32(H1h),
                   uH1l = tc::smem_u32(H1l), uD2h = tc::smem_u32(D2h), uD2l = tc::smem_u32(D2l);
    // layer 1, layer 2 (in FWD beside it), dZ1, dW2 (beside dZ1 and dW1), dW1 (once dZ1 has been
    // read)
    constexpr int A2 = SC ? 0 : 1, AU = PB > PG ? PB : PG;
    const uint32_t tP = tmem, tQ = tP + A2 * H, tB = tmem, tU = tmem + AU * H, tV = tmem;
    static_assert((A2 + P2) * H <= TMEM_COLS && P1 * H <= TMEM_COLS && PB * H <= TMEM_COLS &&
                      (!WG || (AU + PG) * H <= TMEM_COLS), "tensor memory");
    const uint32_t lanes = (uint32_t)(32 * (warp & 3)) << 16;
    const float* gW1 = a.W;
    const float* gb1 = gW1 + H * in;
    const float* gW2 = gb1 + H;
    const float* gb2 = gW2 + H * H;
    const float* gW3 = gb2 + H;
    const float* gb3 = gW3 + out * H;
    uint32_t ph0 = 0, ph1 = 0;
    // A wait that gives up marks the pass and then, once, waits on with a limit of its own: the
    // MMAs in flight are over before the operands, accumulators and barriers are used again.
    bool stuck = false;
    auto wait = [&](uint32_t bar, uint32_t& ph) {
        if (!stuck && !tc::bar_wait(bar, ph, a.limit)) {
            *a.dead = 1;
            if (lane == 0 && status) atomicCAS(status, DEV_OK, DEV_TIMEOUT);
            stuck = !tc::bar_wait(bar, ph, DRAIN_POLLS);
        }
        ph ^= 1u;
        tc::fence_after();
    };
    auto sync = [&] {  // operands in shared memory and tensor-memory reads done, for the next MMAs
        tc::fence_async_smem();
        tc::fence_before();
        __syncthreads();
        tc::fence_after();
    };
    auto load_tile = [&](int t) {
        copy16(uXh, reinterpret_cast<const unsigned char*>(a.X + (size_t)t * TILE_FLOATS), 4 * TILE_HALVES);
    };
    // (the padded columns of W1 meet zero columns of X)
    auto load_w1 = [&] { copy16(uW1h, a.img, 4 * H * KP); };
    auto load_w2 = [&] { copy16(uW2h, a.img + 4 * H * KP, 4 * H * H); };
    if (tid == 0) {
        tc::bar_init(bar0, NB);
        tc::bar_init(bar1, NB);
    }
    // Lane 0 of warps w0 .. w0 + NB - 1 issue the parts of a product and arrive, each when its
    // MMAs are done; a warp without a part arrives at once.
    auto issue = [&](int w0, int parts, uint32_t bar, auto&& part) {
        const int w = warp - w0;
        if (lane != 0 || w < 0 || w >= NB) return;
        if (w < parts) {
            part(w);
            tc::commit(bar);
        } else {
            tc::bar_arrive(bar);
        }
    };
    load_tile(0);
    load_w1();
    if constexpr (!L::SHARE) load_w2();
    float w3m = 0.0f, b1m = 0.0f;
    for (int i = tid; i < H; i += LT) {
        const float b = ldcg(gb1 + i);
        b1[i] = b;
        b1m = fmaxf(b1m, fabsf(b));
        b2[i] = ldcg(gb2 + i);
    }
    for (int i = tid; i < out * H; i += LT) {
        const float w = ldcg(gW3 + i);
        W3[i] = w;
        w3m = fmaxf(w3m, fabsf(w));
    }
    if (tid < out) b3[tid] = ldcg(gb3 + tid);
    if constexpr (MODE == DQ)
        for (int i = tid; i < 4 * H; i += LT) w1a[i] = ldcg(gW1 + (size_t)(i >> 2) * in + in - 4 + (i & 3));
    if constexpr (SC) {
        for (int o = 16; o > 0; o >>= 1) {
            b1m = fmaxf(b1m, __shfl_xor_sync(0xffffffffu, b1m, o));
            w3m = fmaxf(w3m, __shfl_xor_sync(0xffffffffu, w3m, o));
        }
        if (lane == 0) {
            red[warp] = b1m;
            red[8 + warp] = w3m;
        }
        __syncthreads();
        for (int i = 0; i < LT / 32; ++i) {
            b1m = fmaxf(b1m, red[i]);
            w3m = fmaxf(w3m, red[8 + i]);
        }
        __syncthreads();
    }
    const float lw1 = SC ? log2f(a.w1m * (float)in) : 0.0f, lb1 = SC ? log2f(b1m) : 0.0f;
    const float lw3 = BWD ? log2f(w3m * (float)OUT) : 0.0f, lw2 = BWD ? log2f(a.w2m * (float)H) : 0.0f;
    float acc_loss = 0.0f;
    for (int t = 0; t < a.Bc / TR; ++t) {
        const bool first = t == 0;
        const size_t row = (size_t)t * TR + r;
        // exponents of the tile's inputs (largest below 2^X_TOP) and of its first hidden layer, from
        // the bound inputs x largest input x largest weight, or the largest bias
        const int ex = SC ? a.xe[t / TILES_X] : 0;
        const int eh = SC ? scale_to(15, fmaxf(lw1 + (float)(X_TOP - ex), lb1) + 1.0f) : 0;
        const Pow2 k1(SC ? -(ex + a.e.e1) : 0), k2(SC ? -(eh + a.e.e2) : 0);
        const float sh = SC ? exp2i(eh) : 1.0f;
        // (the tile's and W1's copies were issued before the loop or in the previous tile)
        asm volatile("cp.async.wait_all;" ::: "memory");
        if constexpr (MODE == DQ) {
            __syncthreads();  // the tile is complete before its action columns are replaced
            if (half == 0) {
                const float sx = exp2i(ex);
#pragma unroll
                for (int c = 0; c < 4; c += 2) {
                    uint32_t h, l;
                    tc::split2(sx * ldcg(a.mu + row * 4 + c), sx * ldcg(a.mu + row * 4 + c + 1), h, l);
                    const int at = 2 * tc::cano16(r, in - 4 + c, KC1);
                    *reinterpret_cast<uint32_t*>(Xh + at) = h;
                    *reinterpret_cast<uint32_t*>(Xl + at) = l;
                }
            }
        }
        sync();
        // ---- layer 1
        issue(0, P1, bar0, [&](int w) {
            chain_part<false, false, P1, KC1, KC1, KP / 16, ROW>(w, tP, H, uXh, uXl, uW1h, uW1l, idesc<false, false>(H), 0);
        });
        wait(bar0, ph0);
        if constexpr (L::SHARE) load_w2();
        if (!BWD && t + 1 < a.Bc / TR) load_tile(t + 1);  // layer 1 has read the tile
        uint32_t m1[(NC + 31) / 32], amb[(NC + 31) / 32];  // units that passed the ReLU; too close to tell
        float hn = 0.0f, tau1 = 0.0f;
        if constexpr (MODE == CRIT) tau1 = kBand * a.w1m * ldcg(a.xn + row);
#pragma unroll
        for (int i = 0; i < (NC + 31) / 32; ++i) m1[i] = amb[i] = 0u;
        auto epi1 = [&](int c_at) {  // H1's columns from c_at on are this half's
#pragma unroll
            for (int c0 = 0; c0 < NC; c0 += 16) {
                float v[16], x[16];
                ld_acc<P1>(tP + lanes + cb + c0, H, v);
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    const float z = (SC ? k1(v[e]) : v[e]) + b1[cb + c0 + e];
                    x[e] = fmaxf(z, 0.0f);
                    if (BWD && x[e] > 0.0f) m1[(c0 + e) >> 5] |= 1u << ((c0 + e) & 31);
                    if constexpr (MODE == CRIT) {
                        hn += x[e];
                        if (fabsf(z) < tau1) amb[(c0 + e) >> 5] |= 1u << ((c0 + e) & 31);
                    }
                    if (SC) x[e] *= sh;
                }
                put8(H1h, H1l, KCH, r, c_at + c0, x);
                put8(H1h, H1l, KCH, r, c_at + c0 + 8, x + 8);
            }
        };
        if constexpr (L::HALVES) {
            for (int hh = 0; hh < 2; ++hh) {
                if (half == hh) epi1(0);
                sync();
                const uint32_t wo = (uint32_t)hh * 1024u;  // W2's columns 64 hh ..
                if constexpr (SC) {
                    // (the first half beside layer 1, whose other half is still read; the second in
                    // its place)
                    issue(0, 2, bar0, [&](int w) {
                        chain_part<false, false, 2, KCH, KC2, 4>(w, tQ + (hh ? 0 : 2 * H), H, uH1h, uH1l, uW2h + wo, uW2l + wo,
                                                                 idesc<false, false>(H), 0);
                    });
                } else {
                    issue(0, 1, bar0, [&](int) {
                        chain<false, false, KCH, KC2, 4, ROW>(tQ, uH1h, uH1l, uW2h + wo, uW2l + wo, idesc<false, false>(H), hh);
                    });
                }
                wait(bar0, ph0);
            }
        } else {
            epi1(cb);
            if constexpr (MODE == CRIT) {
#pragma unroll
                for (int i = 0; i < (NC + 31) / 32; ++i)
                    for (uint32_t m = amb[i]; m; m &= m - 1) {
                        const int b = __ffs(m) - 1, c = cb + 32 * i + b;
                        const float z = fmaxf(exact_unit1(gW1, in, a.x32 + row * in, gb1, c), 0.0f);
                        m1[i] = z > 0.0f ? m1[i] | (1u << b) : m1[i] & ~(1u << b);
                        const int at = 2 * tc::cano16(r, c, KCH);
                        const __half x = __float2half_rn(sh * z);
                        *reinterpret_cast<__half*>(H1h + at) = x;
                        *reinterpret_cast<__half*>(H1l + at) = __float2half_rn(sh * z - __half2float(x));
                    }
                part[half * TR + r] = hn;
            }
            if constexpr (L::SHARE) asm volatile("cp.async.wait_all;" ::: "memory");
            sync();
            // ---- layer 2
            issue(0, P2, bar0, [&](int w) {
                chain_part<false, false, P2, KCH, KC2, H / 16, ROW>(w, tQ, H, uH1h, uH1l, uW2h, uW2l,
                                                                    idesc<false, false>(H), 0);
            });
            wait(bar0, ph0);
        }
        float tau2 = 0.0f;
        if constexpr (MODE == CRIT) {
            tau2 = kBand * a.w2m * (part[r] + part[TR + r]) + 0.25f * sqrtf((float)H) * a.w2m * tau1;
            __syncthreads();  // part is about to be reused
#pragma unroll
            for (int i = 0; i < (NC + 31) / 32; ++i) amb[i] = 0u;
        }
        float h2[NC], po[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int c0 = 0; c0 < NC; c0 += 16) {
            float v[16];
            ld_acc<P2>(tQ + lanes + cb + c0, H, v);
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                const int c = cb + c0 + e;
                const float z = (SC ? k2(v[e]) : v[e]) + b2[c];
                const float x = fmaxf(z, 0.0f);
                h2[c0 + e] = x;
                if (MODE == CRIT && fabsf(z) < tau2) amb[(c0 + e) >> 5] |= 1u << ((c0 + e) & 31);
#pragma unroll
                for (int o = 0; o < (FW ? 4 : OUT); ++o)
                    if (o < out) po[o] = fmaf(W3[o * H + c], x, po[o]);
            }
        }
        if constexpr (MODE == CRIT) {
#pragma unroll
            for (int i = 0; i < (NC + 31) / 32; ++i) {
                uint32_t who = __ballot_sync(0xffffffffu, amb[i] != 0u);  // (warp-uniform from here)
                while (who) {
                    const int src = __ffs(who) - 1;
                    who &= who - 1;
                    uint32_t m = __shfl_sync(0xffffffffu, amb[i], src);
                    const size_t rs = (size_t)t * TR + 32 * (warp & 3) + src;
                    while (m) {
                        const int b = __ffs(m) - 1;
                        m &= m - 1;
                        const float z = exact_unit2<H>(gW1, in, a.x32 + rs * in, cb + 32 * i + b);
#pragma unroll
                        for (int c = 32 * i; c < NC && c < 32 * i + 32; ++c)
                            if (lane == src && c == 32 * i + b) h2[c] = fmaxf(z, 0.0f);
                    }
                }
            }
        }
#pragma unroll
        for (int o = 0; o < 4; ++o) part[(half * TR + r) * 4 + o] = po[o];
        tc::fence_before();
        __syncthreads();
        tc::fence_after();
        float yv[4];
#pragma unroll
        for (int o = 0; o < 4; ++o) yv[o] = o < out ? part[r * 4 + o] + part[(TR + r) * 4 + o] + b3[o] : 0.0f;
        if constexpr (FW) {
            if (half == 0)
                for (int o = 0; o < out; ++o) a.Y[row * out + o] = a.tanh_out ? tanhf(yv[o]) : yv[o];
        } else {
            // ---- output deltas and their scale
            float dz3[OUT], big = 0.0f;
            if constexpr (MODE == CRIT) {
                const float e = yv[0] - ldcg(a.y + row);
                dz3[0] = 2.0f * e * a.invB;
                if (half == 0) acc_loss += e * e * a.invB;
            } else if constexpr (MODE == DQ) {
                dz3[0] = -a.invB;
                if (half == 0) acc_loss += -yv[0] * a.invB;
            } else {
#pragma unroll
                for (int o = 0; o < OUT; ++o) dz3[o] = ldcg(a.da + row * 4 + o);
            }
#pragma unroll
            for (int o = 0; o < OUT; ++o) big = fmaxf(big, fabsf(dz3[o]));
            for (int o = 16; o > 0; o >>= 1) big = fmaxf(big, __shfl_xor_sync(0xffffffffu, big, o));
            if (lane == 0) red[warp] = big;
            __syncthreads();
            for (int i = 0; i < LT / 32; ++i) big = fmaxf(big, red[i]);
            // exponents of dZ2 and dZ1, from the bounds |dZ2| <= outputs x largest delta x largest
            // weight, |dZ1| <= H x largest dZ2 x largest weight
            const float l2 = log2f(big) + lw3;
            const int se = scale_to(15, l2), sf = scale_to(15, l2 + lw2);
            const float sc = exp2i(se), inv = exp2i(-se), invf = exp2i(-sf);
            const Pow2 kb(sf - se - a.e.e2), ku(-(se + eh)), kv(-(sf + ex));
#pragma unroll
            for (int o = 0; o < OUT; ++o) dz3[o] *= sc;
            float d2[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                float v = 0.0f;
#pragma unroll
                for (int o = 0; o < OUT; ++o) v = fmaf(dz3[o], W3[o * H + cb + c], v);
                d2[c] = h2[c] > 0.0f ? v : 0.0f;
            }
            constexpr int CN = NC < 32 ? NC : 32;  // columns per column sum
            const int cl = lane / (32 / CN);
            float* mys = sums + (warp & 3) * 6 * H + cb;  // this row group's sums: gb1, gb2, gW3[o]
            // ---- dZ2 -> shared memory; dZ1 = dZ2 W2, dW2^T = H1^T dZ2
            if constexpr (H != 128) {
#pragma unroll
                for (int c = 0; c < NC; c += 8) put8(D2h, D2l, KCD, r, cb + c, d2 + c);
                sync();
                issue(0, PB, bar0, [&](int w) {
                    chain_part<false, true, PB, KCD, KC2, H / 16>(w, tB, H, uD2h, uD2l, uW2h, uW2l, idesc<false, true>(H), 0);
                });
                if (WG)
                    issue(4, PG, bar1, [&](int w) {
                        chain_part<true, true, PG, KCH, KCD, TR / 16>(w, tU, H, uH1h, uH1l, uD2h, uD2l, idesc<true, true>(H),
                                                                      0);
                    });
            } else {
                for (int hh = 0; hh < 2; ++hh) {
                    if (half == hh) {
#pragma unroll
                        for (int c = 0; c < NC; c += 8) put8(D2h, D2l, KCD, r, c, d2 + c);
                    }
                    sync();
                    issue(0, PB / 2, bar0, [&](int w) {
                        const uint32_t wo = (uint32_t)hh * 8u * KC2 * 128u;  // W2's rows 64 hh ..
                        chain_part<false, true, PB / 2, KCD, KC2, 4>(w, tB + hh * (PB / 2) * H, H, uD2h, uD2l, uW2h + wo,
                                                                     uW2l + wo, idesc<false, true>(H), 0);
                    });
                    if (WG)
                        issue(4, PG, bar1, [&](int w) {
                            chain_part<true, true, PG, KCH, KCD, TR / 16>(w, tU + 64 * hh, H, uH1h, uH1l, uD2h, uD2l,
                                                                          idesc<true, true>(64), 0);
                        });
                    if (hh == 0) {
                        wait(bar0, ph0);
                        if (WG) wait(bar1, ph1);
                    }
                }
            }
            if constexpr (WG) {  // while they run: the sums over the samples
#pragma unroll
                for (int c = 0; c < NC; c += CN) {
                    float x = colsum<CN>(d2 + c);
                    if (lane % (32 / CN) == 0) mys[H + c + cl] = x;
#pragma unroll
                    for (int o = 0; o < OUT; ++o) {
                        float p[CN];
#pragma unroll
                        for (int e = 0; e < CN; ++e) p[e] = dz3[o] * h2[c + e];
                        x = colsum<CN>(p);
                        if (lane % (32 / CN) == 0) mys[(2 + o) * H + c + cl] = x;
                    }
                }
                if (half == 0)
#pragma unroll
                    for (int o = 0; o < OUT; ++o) {
                        const float x = smlp::warp_sum(dz3[o]);
                        if (lane == 0) red[24 + 4 * warp + o] = x;
                    }
            }
            wait(bar0, ph0);
            if (L::SHARE && t + 1 < a.Bc / TR) load_w1();  // W2 has been read
            // ---- dZ1
            float d1[NC];
#pragma unroll
            for (int c0 = 0; c0 < NC; c0 += 16) {
                float v[16];
                ld_acc<PB>(tB + lanes + cb + c0, H, v);
#pragma unroll
                for (int e = 0; e < 16; ++e) d1[c0 + e] = (m1[(c0 + e) >> 5] >> ((c0 + e) & 31)) & 1u ? kb(v[e]) : 0.0f;
            }
            if constexpr (MODE == DQ) {
                // dLoss/d(action): the last 4 input columns
                float dx[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
                for (int c = 0; c < NC; ++c)
#pragma unroll
                    for (int q = 0; q < 4; ++q) dx[q] = fmaf(d1[c], w1a[(cb + c) * 4 + q], dx[q]);
#pragma unroll
                for (int q = 0; q < 4; ++q) part[(half * TR + r) * 4 + q] = dx[q];
                if (t + 1 < a.Bc / TR) load_tile(t + 1);
                __syncthreads();
                if (half == 0)
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float m = ldcg(a.mu + row * 4 + q);
                        a.da[row * 4 + q] = (part[r * 4 + q] + part[(TR + r) * 4 + q]) * invf * (1.0f - m * m);
                    }
            } else {
                wait(bar1, ph1);  // H1 has been read: dZ1 takes its place
#pragma unroll
                for (int c = 0; c < NC; c += 8) put8(H1h, H1l, KCH, r, cb + c, d1 + c);
                sync();
                issue(0, PG, bar0, [&](int w) {
                    chain_part<true, true, PG, KC1, KCH, TR / 16>(w, tV, H, uXh, uXl, uH1h, uH1l, idesc<true, true>(H), 0);
                });
#pragma unroll
                for (int c = 0; c < NC; c += CN) {
                    const float x = colsum<CN>(d1 + c);
                    if (lane % (32 / CN) == 0) mys[c + cl] = x;
                }
                // gradients: lane = input index, so each column is a coalesced row
                float* G = a.G;
                auto flush = [&](uint32_t acc, float* g, int ld, int rows, const Pow2& k) {
#pragma unroll
                    for (int c0 = 0; c0 < NC; c0 += 16) {
                        float v[16];
                        ld_acc<PG>(acc + lanes + cb + c0, H, v);
                        if (r < rows) {
                            float* p = g + (size_t)(cb + c0) * ld + r;
                            float old[16];
#pragma unroll
                            for (int e = 0; e < 16; ++e) old[e] = first ? 0.0f : p[(size_t)e * ld];
#pragma unroll
                            for (int e = 0; e < 16; ++e) p[(size_t)e * ld] = k(v[e]) + old[e];
                        }
                    }
                };
                flush(tU, G + H * in + H, H, H, ku);
                __syncthreads();  // the column sums are complete
                for (int j = tid; j < H; j += LT) {
                    auto total = [&](int q) {
                        float s = 0.0f;
#pragma unroll
                        for (int w = 0; w < 4; ++w) s += sums[(w * 6 + q) * H + j];
                        return s * (q == 0 ? invf : inv);
                    };
                    auto add = [&](float* p, float x) { *p = first ? x : *p + x; };
                    add(G + H * in + j, total(0));
                    add(G + H * in + H + H * H + j, total(1));
#pragma unroll
                    for (int o = 0; o < OUT; ++o) add(G + H * in + 2 * H + H * H + o * H + j, total(2 + o));
                }
                if (tid < OUT) {
                    float* p = G + H * in + 2 * H + H * H + OUT * H + tid;
                    const float x = (red[24 + tid] + red[28 + tid] + red[32 + tid] + red[36 + tid]) * inv;
                    *p = first ? x : *p + x;
                }
                wait(bar0, ph0);
                if (t + 1 < a.Bc / TR) load_tile(t + 1);
                flush(tV, G, in, in, kv);
            }
        }
        // the next tile reuses the tile buffers, the partial outputs and the tensor memory
        tc::fence_before();
        __syncthreads();
        tc::fence_after();
    }
    return acc_loss;
}

}  // namespace tce
}  // namespace qsim
