// Tensor-core path of the dense pattern-sparse layers (sm_103a, tcgen05).
//
// The contraction y[q, co] = sum over (ci, tap) x[q + shift(tap), ci] w[co, ci, tap] runs as an
// implicit GEMM on the 5th-generation tensor cores with the pruned taps as zeros: the pattern-
// sparse FFMA kernel (conv.cu) is bound by instruction issue at 0.44 of the FP32 peak, 28-30
// useful TFLOP/s at keep 0.3; with 0.133 of the weights kept a dense fp16 product of three terms
// costs 3 / 0.133 = 22 tensor FLOP per useful one, and the tensor cores have 25 times the FP32
// rate, 60 at keep 1.
//
// Precision.  Every fp32 operand is held as two fp16 values, v = (h + l 2^-11) 2^-k with one
// power of two k per layer (weights) or per stage (inputs: 16 channels of the staged positions).  The
// pair carries 22 to 23 bits of a scaled value down to 2^-14 and errs by 2^-36 below; an input stage's
// largest is kept in [2^11, 2^15), the layer's largest weight in [2^14, 2^15).  Sums that smaller inputs
// may have put off are found by a bound and taken again in fp32 (redo_unit).  A chain of MMAs first sums
// the cross terms h_x l_w + l_x h_w of the nine taps, then adds h_x h_w with the accumulator scaled
// by 2^-11 in the first of those MMAs (scale-input-d); the dropped l_x l_w is 2^-24.6 of a product
// (rms), and tiles of one column block (MT 1: small batches, where the FFMA kernel's split sums round
// less) sum it as well.  The tensor core's accumulator truncates, so a chain covers 16 channels
// only and the sums are then added in fp32 registers, rounded to nearest, by eight warps; what the
// truncation takes away on average is put back into the weights (tensor_bias).
// fp16 inputs are exact and need two products.
//
// Measured against pconv_tm (us, batch 32 or 64, keep 0.3; fp32): 256->256 56x56 517 -> 201,
// 512->512 14x14 183 -> 70, 64->64 224x224 with the pool 547 -> 326, 256->256 28x28 stride 2
// 200 -> 55; fp16 256->256 28x28 keep 1 808 -> 75.  What bounds it: the MMA rate and the last wave
// (56x56: 5.36 waves of CTA pairs run as 6; 73 % of the tensor pipe) on the 56x56 and 28x28 layers of
// 256 and 512 filters, the input staging (six warps: split into pairs, store) with 64 filters or
// stride 2, one partial wave on the smallest.
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <climits>
#include <cmath>
#include <cstdint>
#include <cstring>

#include "tensor.h"

namespace patconv {
namespace {

constexpr int kThreads = 512;
constexpr int kPromoteWarps = 8;        // warps 0-7: sums in registers, epilogue
constexpr int kProducerWarps = 6;       // warps 8-13: input staging
constexpr int kLoaderWarp = 14, kMmaWarp = 15;
constexpr int kProducers = kProducerWarps * 32;
constexpr int kMaxWSlots = 6, kMaxXStages = 3, kMaxRaw = 2;   // as tensor_plan deals shared memory out
// items a producer thread's copies run ahead, plus one, by the words of a channel in an item
constexpr int ring_of(int words) { return words == 1 ? 6 : (words == 2 ? 4 : 3); }
constexpr int kHdr = 8;                 // stage headers in flight
constexpr unsigned kHeadBytes = 1024 + 2 * 256 * 4;   // barriers, headers, two units' biases
constexpr uint32_t kTmemColumns = 512;
constexpr long long kDrainCycles = 2000000000LL;   // about one second
constexpr long long kSettleCycles = 20000;         // about 10 us
constexpr unsigned kErrData = 1u, kErrSpace = 2u, kErrDrain = 4u;

// division of 0 <= n < 2^31 by a constant d >= 2
struct FastDiv {
    uint32_t d, m, s;
};
FastDiv fast_div(uint32_t d) {
    FastDiv f;
    f.d = d;
    uint32_t l = 0;
    while ((1ull << l) < d) ++l;
    f.s = l - 1;
    f.m = (uint32_t)((1ull << (31 + l)) / d + 1);
    return f;
}
__device__ __forceinline__ uint32_t fdiv(uint32_t n, const FastDiv& f) { return __umulhi(n, f.m) >> f.s; }

struct TcParams {
    const void* x;
    void* y;
    const float* bias;
    const unsigned char* wimg;
    const uint32_t* perm;
    const uint64_t* desc;
    const uint32_t* kofs;
    const float4* vals;
    unsigned* status;
    long long wait_limit;
    int no_fill;
    int N, C, H, W, Cout, Ho, Wo, G, relu, pool;
    int wexp;                  // weights are scaled by 2^wexp
    float wbias;               // ... and by 1 + wbias (in their lo parts)
    float unheld;              // a slow block's factor to the smallest sum it may be part of
    int all_slow;              // weights that their pairs do not hold: every block
    int NC, KS, n_cb, cb_split;
    int ll;                    // fp32: the products of the lo parts too
    int Wp, Ip, mstep, P;       // position pitch of a row, of an image (flat); tile step; staged positions
    int tw, th, tiles_x, tiles_y;   // rectangles of tw x th outputs (tw 0: flat tiles)
    long long Q;
    int tiles, n_fchunks, n_units;
    int vec, ppr, n_entries, items;   // values a copy; copies of a staged row (vec > 1); table entries; items of a block
    FastDiv d_ip, d_wp, d_p, d_ppr;
    int box, rw, rs;           // input by boxes of rows of rw values; their stages
    float* ws;
    size_t ws_stride;
    int xs, hs, ls;            // input stages, slots of the hi and lo weights
    unsigned plane, x_stage, w_slot, pool_off, tab_off, ring_off, x_off, h_off, l_off;
    uint16_t masks[kMaxPatterns];
};

struct Unit {
    long long q0;              // flat tiles: first position of the tile in the padded output grid
    int n, oy0, ox0;           // rectangles: image and first output
    int fc, r0;                // filter chunk, its first filter
    int cb0, cb1, ks;
};

// Unit u of a CTA pair: two neighbouring position tiles, one per CTA, and the filters both share.
__device__ __forceinline__ Unit unit_of(const TcParams& p, int u, int rank) {
    Unit U;
    const int fc = u % p.n_fchunks;
    int t = u / p.n_fchunks;
    U.ks = t / p.tiles;
    t = 2 * (t - U.ks * p.tiles) + rank;
    U.q0 = (long long)t * p.mstep;
    if (p.tw) {
        const int ty = t / p.tiles_x;
        U.ox0 = (t - ty * p.tiles_x) * p.tw;
        U.n = ty / p.tiles_y;
        U.oy0 = (ty - U.n * p.tiles_y) * p.th;
    }
    U.r0 = fc * p.NC;
    U.fc = fc;
    U.cb0 = U.ks * p.cb_split;
    U.cb1 = min(p.n_cb, U.cb0 + p.cb_split);
    return U;
}

// Output of tile position i.  Rectangles have rows of Wp positions, the first tw of them outputs;
// flat tiles are 128 MT consecutive positions of all images' rows of Wo + 1 and columns of Ho + 1.
struct Point {
    int n, oy, ox;
    bool in;
};
__device__ __forceinline__ Point point_of(const TcParams& p, const Unit& U, int i) {
    Point o;
    if (p.tw) {
        const int r = (int)fdiv((uint32_t)i, p.d_wp), c = i - r * p.Wp;
        o.n = U.n;
        o.oy = U.oy0 + r;
        o.ox = U.ox0 + c;
        o.in = r < p.th && c < p.tw && o.n < p.N && o.oy < p.Ho && o.ox < p.Wo;
    } else {
        const long long q = U.q0 + i;
        const uint32_t n = fdiv((uint32_t)q, p.d_ip), r = (uint32_t)q - n * (uint32_t)p.Ip;
        o.n = (int)n;
        o.oy = (int)fdiv(r, p.d_wp);
        o.ox = (int)r - o.oy * p.Wp;
        o.in = q < p.Q && o.n < p.N && o.oy < p.Ho && o.ox < p.Wo;
    }
    return o;
}

__device__ __forceinline__ uint32_t smem_u32(const void* ptr) { return (uint32_t)__cvta_generic_to_shared(ptr); }
__device__ __forceinline__ void mbar_init(uint32_t a, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(a), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t a, uint32_t tx) {
    asm volatile("mbarrier.arrive.expect_tx.release.cta.shared::cta.b64 _, [%0], %1;" ::"r"(a), "r"(tx) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t a) {
    asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(a) : "memory");
}
// Arrival on the leader's barrier at the same offset, with the CTA's scope: what it announces is
// read by the tensor core only, after a proxy fence, or not at all (a block's header goes from the
// staging warps to the summing warps of its own CTA over a barrier of its own).  (A cluster-wide release waits
// for the thread's loads in flight: the 56x56 layer 241 against 203 us; cluster-wide acquires cost a
// wait some 200 clocks.)
__device__ __forceinline__ void mbar_arrive_leader(uint32_t a) {
    asm volatile(
        "{\n\t.reg .b32 R;\n\tmapa.shared::cluster.u32 R, %0, 0;\n\t"
        "mbarrier.arrive.shared::cluster.b64 _, [R];\n\t}" ::"r"(a) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t a, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred P;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, P;\n\t}"
        : "=r"(done) : "r"(a), "r"(parity) : "memory");
    return done != 0;
}
// Bounded wait; a wait that runs out records its code and raises the CTA's abort flag, which ends
// every other wait of the CTA too.
__device__ __forceinline__ bool wait_bar(uint32_t a, uint32_t parity, const TcParams& p, volatile int* abort_flag,
                                         unsigned code) {
    if (mbar_try(a, parity)) return true;
    const long long t0 = clock64();
    while (true) {
        if (mbar_try(a, parity)) return true;
        if (*abort_flag) return false;
        if (clock64() - t0 > p.wait_limit) {
            atomicOr(p.status, code);
            *abort_flag = 1;
            return false;
        }
    }
}
// the same by a whole warp, with one outcome for all its lanes
__device__ __forceinline__ bool wait_warp(uint32_t a, uint32_t parity, const TcParams& p, volatile int* abort_flag,
                                          unsigned code) {
    return __all_sync(0xFFFFFFFFu, wait_bar(a, parity, p, abort_flag, code));
}
__device__ __forceinline__ void box_load(uint32_t dst, const CUtensorMap* map, int x, int y, int c, int n, uint32_t mbar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(c), "r"(n), "r"(mbar) : "memory");
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(mbar) : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void commit(uint32_t mbar) {   // this CTA's barrier
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar) : "memory");
}
__device__ __forceinline__ void commit_pair(uint32_t mbar) {   // the barrier at this offset in both CTAs
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(mbar), "h"((uint16_t)3) : "memory");
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// One lane of a converged warp
__device__ __forceinline__ bool elect_one() {
    uint32_t r;
    asm volatile("{\n\t.reg .pred P;\n\telect.sync _|P, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, P;\n\t}" : "=r"(r)::"memory");
    return r != 0;
}
// Shared-memory matrix descriptor, K-major without swizzle: 8 rows x 16 bytes are 128 contiguous
// bytes, the next 8 rows follow at once (stride offset 128), the next 8 channels lie `lead` bytes
// further.  The low word holds the address and the lead, the high word is this constant.
constexpr uint32_t kDescHi = 8u | (1u << 14);
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr, uint32_t lead) { return (addr >> 4) | (lead << 12); }
// D = A B (ACC 0), D = A B + D (1), D = A B + D 2^-11 (2)
template <int ACC>
__device__ __forceinline__ void mma(uint32_t d, uint32_t a, uint32_t b, uint32_t idesc) {
    if constexpr (ACC == 2)
        asm volatile(
            "{\n\t.reg .pred P;\n\t.reg .b64 A, B;\n\tsetp.eq.b32 P, 0, 0;\n\tmov.b64 A, {%1, %4};\n\tmov.b64 B, {%2, %4};\n\t"
            "tcgen05.mma.cta_group::2.kind::f16 [%0], A, B, %3, {%5, %5, %5, %5, %5, %5, %5, %5}, P, 11;\n\t}"
            ::"r"(d), "r"(a), "r"(b), "r"(idesc), "n"(kDescHi), "r"(0) : "memory");
    else
        asm volatile(
            "{\n\t.reg .pred P;\n\t.reg .b64 A, B;\n\tsetp.eq.b32 P, %5, 1;\n\tmov.b64 A, {%1, %4};\n\tmov.b64 B, {%2, %4};\n\t"
            "tcgen05.mma.cta_group::2.kind::f16 [%0], A, B, %3, P;\n\t}"
            ::"r"(d), "r"(a), "r"(b), "r"(idesc), "n"(kDescHi), "n"(ACC) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t ta, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(ta) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
// all threads of a named barrier: true where any of them passes true
template <int ID, int NT>
__device__ __forceinline__ bool bar_or(bool v) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred P, Q;\n\tsetp.ne.u32 P, %1, 0;\n\t"
        "barrier.cta.red.or.pred Q, %2, %3, P;\n\tselp.u32 %0, 1, 0, Q;\n\t}"
        : "=r"(r) : "r"(v ? 1u : 0u), "n"(ID), "n"(NT) : "memory");
    return r != 0;
}

__device__ __forceinline__ float relu_of(float v, int relu) { return relu ? fmaxf(v, 0.0f) : v; }

template <typename T>
__device__ __forceinline__ T out_of(float v);
template <>
__device__ __forceinline__ float out_of<float>(float v) { return v; }
template <>
__device__ __forceinline__ __half out_of<__half>(float v) { return __float2half_rn(v); }

// ---------------------------------------------------------------------------- input staging

// two fp32 products, and two fused multiply-adds, in one instruction each
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    float2 r;
    asm("{\n\t.reg .b64 A, B, R;\n\tmov.b64 A, {%2, %3};\n\tmov.b64 B, {%4, %5};\n\tmul.rn.f32x2 R, A, B;\n\tmov.b64 {%0, %1}, R;\n\t}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    float2 r;
    asm("{\n\t.reg .b64 A, B, C, R;\n\tmov.b64 A, {%2, %3};\n\tmov.b64 B, {%4, %5};\n\tmov.b64 C, {%6, %7};\n\t"
        "fma.rn.f32x2 R, A, B, C;\n\tmov.b64 {%0, %1}, R;\n\t}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return r;
}
// One position and 8 channels: the fp16 pair of each value times s; *mx the largest |hi| so far.
__device__ __forceinline__ void split8(const float (&v)[8], float s, uint4* hi, uint4* lo, __half2* mx) {
    uint32_t h[4], l[4];
    const float2 s1 = make_float2(s, s), s2 = make_float2(s * 2048.0f, s * 2048.0f), m = make_float2(-2048.0f, -2048.0f);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float2 x = make_float2(v[2 * j], v[2 * j + 1]);
        const float2 p = mul2(x, s1);
        const __half2 hh = __floats2half2_rn(p.x, p.y);
        const float2 r = fma2(__half22float2(hh), m, mul2(x, s2));
        const __half2 ll = __floats2half2_rn(r.x, r.y);
        *mx = __hmax2_nan(*mx, __habs2(hh));
        h[j] = *reinterpret_cast<const uint32_t*>(&hh);
        l[j] = *reinterpret_cast<const uint32_t*>(&ll);
    }
    *hi = make_uint4(h[0], h[1], h[2], h[3]);
    *lo = make_uint4(l[0], l[1], l[2], l[3]);
}

// The staged window of a unit as a table, one word per position: the element offset of its input
// (of input (2 oy, 2 ox) at stride 2) from image n0's channel 0 in bits 2-31, kOut where it lies
// outside every image; at stride 2 bits 0 and 1 say whether the next column and row exist.
constexpr uint32_t kOut = 0xFFFFFFFFu;

template <int S>
__device__ __forceinline__ uint32_t window_entry(const TcParams& p, const Unit& U, int i, int n0) {
    int n, y, x;
    if (p.tw) {
        const int r = (int)fdiv((uint32_t)i, p.d_wp);
        n = U.n;
        y = U.oy0 + r - 1;
        x = U.ox0 + (i - r * p.Wp) - 1;
    } else {
        const long long q = U.q0 - p.Wp - 1 + i;
        if (q < 0) return kOut;
        n = (int)fdiv((uint32_t)q, p.d_ip);
        const uint32_t r = (uint32_t)q - (uint32_t)n * (uint32_t)p.Ip;
        y = (int)fdiv(r, p.d_wp);
        x = (int)r - y * p.Wp;
        if (y >= p.Ho || x >= p.Wo) return kOut;
    }
    if (n >= p.N || y < 0 || x < 0 || y * S >= p.H || x * S >= p.W) return kOut;
    const uint32_t off = ((uint32_t)(n - n0) * (uint32_t)p.C * p.H + y * S) * p.W + x * S;
    uint32_t flags = 0;
    if (S == 2) flags = (2 * x + 1 < p.W ? 1u : 0u) | (2 * y + 1 < p.H ? 2u : 0u);
    return off << 2 | flags;
}
// the first image a window touches
__device__ __forceinline__ int first_image(const TcParams& p, const Unit& U) {
    const long long n = p.tw ? (long long)U.n : max(U.q0 - p.Wp - 1, 0LL) / p.Ip;
    return (int)min((long long)(p.N - 1), n);
}

// Staging state of a producer thread that does not depend on the input type.
struct Stage {
    int e = 0, s = 0, ph = 0;   // blocks staged, their slot, its round
    int par = 0;
};

// The end of a block: the six warps' extremes (mx: maximum, or union of bits for fp16; mn minimum)
// in every producer thread.  false where one of the warps gave up waiting.
template <bool MAX>
__device__ __forceinline__ bool combine(uint32_t* mx, uint32_t* mn, bool ok, uint2* red, int* par, int warp, int lane) {
    *mx = MAX ? __reduce_max_sync(0xFFFFFFFFu, *mx) : __reduce_or_sync(0xFFFFFFFFu, *mx);
    *mn = __reduce_min_sync(0xFFFFFFFFu, *mn);
    if (lane == 0) red[*par * 8 + warp] = make_uint2(*mx, *mn);
    if (bar_or<1, kProducers>(!ok)) return false;
#pragma unroll
    for (int w = 0; w < kProducerWarps; ++w) {
        const uint2 r = red[*par * 8 + w];
        *mx = MAX ? max(*mx, r.x) : (*mx | r.x);
        *mn = min(*mn, r.y);
    }
    *par ^= 1;
    return true;
}
// A block's header: the factor of its sums, and whether it holds values that their pairs do not.
__device__ __forceinline__ void publish(const TcParams& p, Stage* sg, uint32_t xfull, float2* hdr, uint32_t hready, int kexp, bool slow,
                                        int tid, int lane) {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    if (lane == 0 && !p.no_fill) mbar_arrive_leader(xfull + 8 * sg->s);
    if (tid == 0) {   // (the slot's header of kHdr blocks ago was read before this block's stage was freed)
        hdr[sg->e & (kHdr - 1)] = make_float2(__uint_as_float((uint32_t)(127 - kexp - p.wexp) << 23), slow || p.all_slow ? 1.0f : 0.0f);
        mbar_arrive(hready + 8 * (sg->e & (kHdr - 1)));
    }
    ++sg->e;
    if (++sg->s == p.xs) { sg->s = 0; ++sg->ph; }
}

// The end of staging: the MMAs' last commits signal xempty in both CTAs of the pair, also for stages
// that nobody fills again, and a CTA must not exit before these arrivals have landed in its shared
// memory.  One thread waits for the last use of every stage (the uses before it were waited for when
// the stage was filled again).  Not inlined: inside the staging loops' code it cost them registers
// (64 bytes of spills more; 64 -> 64 at 224x224 with the pool 330 -> 337 us).
__device__ __noinline__ void stages_done(const TcParams& p, const Stage& sg, uint32_t xempty, volatile int* abort_flag, int tid) {
    if (tid != 0) return;
    for (int k = max(0, sg.e - p.xs); k < sg.e; ++k)
        if (!wait_bar(xempty + 8 * (k % p.xs), (uint32_t)(k / p.xs) & 1u, p, abort_flag, kErrSpace)) return;
}

// Item i of a block: plane and channel half k, position.
template <int S>
__device__ __forceinline__ bool item_of(const TcParams& p, int i, int items, int* k, int* pos) {
    *k = S == 1 ? (i >= p.P ? 1 : 0) : (int)fdiv((uint32_t)i, p.d_p);
    *pos = i - *k * p.P;
    return i < items;
}
// whether the item's input exists, and its element offset from the block's first channel plane
template <int S>
__device__ __forceinline__ bool input_of(const TcParams& p, uint32_t t, int k, uint32_t HW, uint32_t* off) {
    bool in = t != kOut;
    *off = (t >> 2) + ((k & 1) ? 8u * HW : 0u);
    if constexpr (S == 2) {
        const int pl = k >> 1;   // 2 (odd rows) + (odd columns)
        in = in && (!(pl & 1) || (t & 1u)) && (!(pl & 2) || (t & 2u));
        *off += (uint32_t)(pl >> 1) * p.W + (uint32_t)(pl & 1);
    }
    return in;
}

// asynchronous copy of n = 0 or BYTES bytes, zero-filled to BYTES
template <int BYTES>
__device__ __forceinline__ void copy_async(uint32_t dst, const char* src, uint32_t n) {
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %3, %2;" ::"r"(dst), "l"(src), "r"(n), "n"(BYTES) : "memory");
}

// The first position of a flat tile's window as row and column of the padded grid.
__device__ __forceinline__ void window_start(const TcParams& p, const Unit& U, int* row, int* col) {
    const long long q = U.q0 - p.Wp - 1 + 2 * p.Wp;   // never negative
    const uint32_t r = fdiv((uint32_t)q, p.d_wp);
    *row = (int)r - 2;
    *col = (int)((uint32_t)q - r * (uint32_t)p.Wp);
}
// Entry m of a unit's table of copies: VEC inputs of one row from a column that is a multiple of VEC.
// x: their element offset from image n0's channel 0 (kOut: zeros).  y: the first staged position they
// go to, plus VEC, in bits 0-15, and a bit a value from bit 28 on that says it is staged: VEC
// neighbouring positions at stride 1; at stride 2 the even and odd columns of VEC / 2 positions (of
// even rows; bit 27 says the odd row below exists).
template <int S, int VEC>
__device__ __forceinline__ uint2 copy_entry(const TcParams& p, const Unit& U, int m, int n0) {
    constexpr int NP = VEC / S;   // positions of a copy
    int row = 0, col = 0;
    if (!p.tw) {                  // flat: from the copy of the window's first position on
        window_start(p, U, &row, &col);
        m += col / NP;
    }
    const int r = (int)fdiv((uint32_t)m, p.d_ppr), j = m - r * p.ppr;
    int n, y, x, c0, p0;          // x, y in the output grid
    if (p.tw) {
        n = U.n;
        y = U.oy0 + r - 1;
        x = ((U.ox0 - 1) & ~(NP - 1)) + NP * j;
        c0 = x - (U.ox0 - 1);
        p0 = r * p.Wp + c0;
        if (S == 1 && r >= p.th + 2) {   // the last entry: the two positions after the last row
            y = -1;
            c0 = 0;
            p0 = r * p.Wp;
        }
    } else {
        row += r;
        x = c0 = NP * j;
        p0 = r * p.Wp + x - col;
        y = -1;
        n = 0;
        if (row >= 0) {
            n = (int)fdiv((uint32_t)row * (uint32_t)p.Wp, p.d_ip);
            y = row - n * (p.Ho + 1);
        }
    }
    uint2 e;
    e.x = kOut;
    e.y = 0;
#pragma unroll
    for (int a = 0; a < NP; ++a) {
        if (c0 + a >= 0 && c0 + a < p.Wp && p0 + a >= 0 && p0 + a < p.P) e.y |= (S == 1 ? 1u : 3u) << (28 + S * a);
    }
    if (e.y) e.y |= (uint32_t)(p0 + VEC);
    if (n < p.N && y >= 0 && y < p.Ho && x >= 0 && x * S < p.W) {
        e.x = ((uint32_t)(n - n0) * (uint32_t)p.C * p.H + (uint32_t)(y * S)) * p.W + (uint32_t)(x * S);
        if (S == 2 && 2 * y + 1 < p.H) e.y |= 1u << 27;
    }
    return e;
}

// Staging by six warps: a thread takes items of eight channels, copies the item's values
// asynchronously to its own column of a ring in shared memory (neighbouring lanes neighbouring
// addresses), and RING - 1 items later splits them and stores 16 bytes of hi and of lo a position.
// The copies run ahead over blocks and units.  What held this part was first the latency of its loads
// (two items ahead in registers: 0.85 clocks a value), then the number of copies, a warp's copy
// taking some 16 clocks whether of 4 or 8 bytes a lane: so where rows are a multiple of VEC inputs
// and x is aligned to them a copy brings VEC values (256 -> 256, 28x28 to 14x14, batch 64: 64 us with
// one, 51 with two).  fp16 inputs are exact: their 16 bits go to the stage as they are; the copy has no
// 2-byte form, so VEC is 2 or 4.
template <int S, typename T, int VEC>
__device__ __forceinline__ void produce_async(const TcParams& p, unsigned char* smem, uint32_t xfull, uint32_t xempty,
                                            volatile int* abort_flag, uint2* red, float2* hdr, uint32_t hready, int rank, int pair, int pairs) {
    constexpr bool F32 = sizeof(T) == 4;
    static_assert(F32 || VEC > 1, "fp16 values are copied in pairs at least");
    constexpr int HL = F32 ? 2 : 1;
    constexpr int V = VEC;                           // values of a channel in an item
    constexpr int WV = F32 ? V : V / 2;              // words they take
    constexpr int RING = ring_of(WV);
    constexpr int SLOT = (8 * WV + 1) * kProducers;  // words of a ring slot: the values, where they go
    const int tid = (int)threadIdx.x - kPromoteWarps * 32, lane = tid & 31, warp = tid >> 5;
    const uint32_t HW = (uint32_t)p.H * p.W, HWB = HW * (uint32_t)sizeof(T);
    uint32_t* table = reinterpret_cast<uint32_t*>(smem + p.tab_off);
    uint2* table2 = reinterpret_cast<uint2*>(table);
    const int steps = (p.items + kProducers - 1) / kProducers;
    float* ring = reinterpret_cast<float*>(smem + p.ring_off);
    // byte offset in the stage of an item's value a: positions side by side, at stride 2 the odd
    // columns in a plane of their own
    auto place = [&](int a) { return S == 1 ? 16u * a : 16u * (a >> 1) + (a & 1) * (2u * HL * p.plane); };
    // item i of a unit, from a table entry: whether its inputs exist, their offset, and where it goes
    // (byte offset in the stage plus 16 VEC; from bit 28 on: the values that are staged)
    auto decode = [&](int i, auto&& entry, uint32_t* off, uint32_t* dst) {
        *dst = 0;
        if (i >= p.items) return false;
        if constexpr (VEC > 1) {
            const int k = (int)fdiv((uint32_t)i, p.d_p);   // channel half, at stride 2 + 2 (odd rows)
            const uint2 e = entry(i - k * p.n_entries);
            const int odd_row = S == 2 ? k >> 1 : 0;
            *off = e.x + ((k & 1) ? 8u * HW : 0u) + (uint32_t)odd_row * p.W;
            if (e.y) *dst = (e.y & 0xF0000000u) | ((e.y & 0xFFFFu) * 16u + (uint32_t)(odd_row * 4 * HL + (k & 1)) * p.plane);
            return e.x != kOut && (!odd_row || (e.y & (1u << 27)));
        } else {
            const int k = (int)fdiv((uint32_t)i, p.d_p);
            const int pos = i - k * p.P;
            const uint32_t t = entry(pos).x;
            bool in = t != kOut;
            *off = (t >> 2) + ((k & 1) ? 8u * HW : 0u);
            const int odd_row = k >> 2, odd_col = (k >> 1) & 1;
            if constexpr (S == 2) {
                in = in && (!odd_col || (t & 1u)) && (!odd_row || (t & 2u));
                *off += (uint32_t)odd_row * p.W + (uint32_t)odd_col;
            }
            const int pl = S == 1 ? 0 : 2 * odd_row + odd_col;
            *dst = 0x10000000u | ((uint32_t)(pl * 2 * HL + (k & 1)) * p.plane + (uint32_t)(pos + 1) * 16u);
            return in;
        }
    };
    auto channel_of = [&](int i) { return (int)(fdiv((uint32_t)i, p.d_p) & 1u) * 8; };
    int kexp = 0;
    Stage sg;
    // the copies' cursor: unit, block, step, slot
    int iu = pair, icb = 0, icb1 = 0, ig = 0, islot = 0;
    const char* ix = nullptr;
    auto issue = [&]() {
        if (iu < p.n_units) {
            if (ig == 0 && icb == icb1) {   // a new unit: its window table
                const Unit U = unit_of(p, iu, rank);
                const int n0 = first_image(p, U);
                bar_or<1, kProducers>(false);
                for (int i = tid; i < p.n_entries; i += kProducers) {
                    if constexpr (VEC > 1) table2[i] = copy_entry<S, VEC>(p, U, i, n0);
                    else table[i] = window_entry<S>(p, U, i, n0);
                }
                bar_or<1, kProducers>(false);
                icb = U.cb0;
                icb1 = U.cb1;
                ix = reinterpret_cast<const char*>(p.x) + ((size_t)n0 * p.C + U.cb0 * 16) * HWB;
            }
            const int i = tid + ig * kProducers;
            uint32_t off, dst;
            const bool in = decode(i, [&](int m) {
                if constexpr (VEC > 1) return table2[m];
                else return make_uint2(table[m], 0u);
            }, &off, &dst);
            float* slot = ring + islot * SLOT;
            reinterpret_cast<uint32_t*>(slot)[8 * WV * kProducers + tid] = dst;
            if (dst != 0) {
                const int nch = in ? p.C - icb * 16 - channel_of(i) : 0;
                const char* src = in ? ix + (size_t)off * sizeof(T) : reinterpret_cast<const char*>(p.x);
                const uint32_t to = smem_u32(slot + WV * tid);
                if (nch >= 8 || nch <= 0) {
                    const uint32_t n = nch > 0 ? 4u * WV : 0u;
                    const size_t step = nch > 0 ? HWB : 0;
#pragma unroll
                    for (int j = 0; j < 8; ++j, src += step) copy_async<4 * WV>(to + j * (4 * WV * kProducers), src, n);
                } else {
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        copy_async<4 * WV>(to + j * (4 * WV * kProducers), src, j < nch ? 4u * WV : 0u);
                        if (j + 1 < nch) src += HWB;
                    }
                }
            }
            if (++ig == steps) {
                ig = 0;
                ix += (size_t)16 * HWB;
                if (++icb == icb1) iu += pairs;
            }
            if (++islot == RING) islot = 0;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int r = 0; r < RING - 1; ++r) issue();

    int slot = 0;
    for (int u = pair; u < p.n_units; u += pairs) {
        const Unit U = unit_of(p, u, rank);
        for (int cb = U.cb0; cb < U.cb1; ++cb) {
            const bool ok = sg.e < p.xs || wait_bar(xempty + 8 * sg.s, (sg.ph & 1) ^ 1, p, abort_flag, kErrSpace);
            unsigned char* st = smem + p.x_off + (size_t)sg.s * p.x_stage - 16 * VEC;
            uint32_t mn = 0xFFFFFFFFu, bad = 0;
            __half2 hmx = __half2half2(__ushort_as_half(0));
            float scale = __uint_as_float((uint32_t)(127 + kexp) << 23);
            auto split = [&](const float (&v)[WV][8], uint32_t dst) {
#pragma unroll
                for (int a = 0; a < V; ++a) {
                    if (!(dst & (0x10000000u << a))) continue;
                    unsigned char* d = st + (dst & 0x0FFFFFFFu) + place(a);
                    if constexpr (!F32) {   // a word holds two values of a channel
                        uint32_t w[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            w[j] = __byte_perm(__float_as_uint(v[a / 2 % WV][2 * j]), __float_as_uint(v[a / 2 % WV][2 * j + 1]), a & 1 ? 0x7632 : 0x5410);
                            bad |= ((w[j] & 0x7C007C00u) + 0x04000400u) & 0x80008000u;   // exponent 31: not finite
                        }
                        *reinterpret_cast<uint4*>(d) = make_uint4(w[0], w[1], w[2], w[3]);
                    } else {
                        // the smallest |v| as an ordered integer, a zero as the largest
#pragma unroll
                        for (int j = 0; j < 8; j += 2)
                            mn = min(min(mn, 2u * __float_as_uint(v[a][j]) - 1u), 2u * __float_as_uint(v[a][j + 1]) - 1u);
                        uint4 hi, lo;
                        split8(v[a], scale, &hi, &lo, &hmx);
                        *reinterpret_cast<uint4*>(d) = hi;
                        *reinterpret_cast<uint4*>(d + 2 * p.plane) = lo;
                    }
                }
            };
            for (int g = 0; g < steps; ++g) {
                asm volatile("cp.async.wait_group %0;" ::"n"(RING - 2) : "memory");
                float v[WV][8];
                const float* from = ring + slot * SLOT;
                const uint32_t dst = reinterpret_cast<const uint32_t*>(from)[8 * WV * kProducers + tid];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    if constexpr (WV == 4) {
                        const float4 t = *reinterpret_cast<const float4*>(from + 4 * (j * kProducers + tid));
                        v[0][j] = t.x;
                        v[1 % WV][j] = t.y;
                        v[2 % WV][j] = t.z;
                        v[3 % WV][j] = t.w;
                    } else if constexpr (WV == 2) {
                        const float2 t = *reinterpret_cast<const float2*>(from + 2 * (j * kProducers + tid));
                        v[0][j] = t.x;
                        v[WV - 1][j] = t.y;
                    } else {
                        v[0][j] = from[j * kProducers + tid];
                    }
                }
                issue();
                if (++slot == RING) slot = 0;
                if (ok) split(v, dst);
            }
            bool slow = false;
            if constexpr (!F32) {
                if (!combine<false>(&bad, &mn, ok, red, &sg.par, warp, lane)) return;
                slow = bad != 0;
            } else {
                // the larger half of the largest hi parts; NaN is the largest of all
                const uint32_t b = *reinterpret_cast<const uint32_t*>(&hmx);
                uint32_t mx = max(b & 0xFFFFu, b >> 16);
                if (!combine<true>(&mx, &mn, ok, red, &sg.par, warp, lane)) return;
                // hi parts up to 2^11 ... 2^15 use the pair's whole range; else the block is taken again
                // (from memory), its largest value scaled to [2^13, 2^14)
                if (mn != 0xFFFFFFFFu && (mx < 0x6800u || mx >= 0x7800u)) {
                    int u1 = u;
                    asm volatile("" : "+r"(u1));   // the unit again: held in registers for this rare path it cost
                                                   // spills (28x28 stride 2, batch 64: 55.7 -> 53.6 us)
                    const Unit U1 = unit_of(p, u1, rank);
                    const int n0 = first_image(p, U1);
                    auto again = [&](int i, float (&v)[V][8]) {
                        uint32_t off, dst;
                        const bool in = decode(i, [&](int m) {
                            if constexpr (VEC > 1) return copy_entry<S, VEC>(p, U1, m, n0);
                            else return make_uint2(window_entry<S>(p, U1, m, n0), 0u);
                        }, &off, &dst);
                        const int nch = in ? p.C - cb * 16 - channel_of(i) : 0;
                        const float* src = static_cast<const float*>(p.x) + ((size_t)n0 * p.C + cb * 16) * HW + off;
                        for (int j = 0; j < 8; ++j)
                            for (int a = 0; a < V; ++a) v[a][j] = j < nch ? __ldg(src + (size_t)j * HW + a) : 0.0f;
                        return dst;
                    };
                    mx = 0;
                    float v[V][8];
    #pragma unroll 1
                    for (int g = 0; g < steps; ++g) {
                        const uint32_t dst = again(tid + g * kProducers, v);
                        for (int a = 0; a < V; ++a)
                            if (dst & (0x10000000u << a))
                                for (int j = 0; j < 8; ++j) mx = max(mx, 2u * __float_as_uint(v[a][j]));
                    }
                    if (!combine<true>(&mx, &mn, ok, red, &sg.par, warp, lane)) return;
                    const int ex = (int)(mx >> 24) - 127;
                    slow = ex < -60 || ex > 120;   // also infinities and NaN
                    if (!slow) {
                        kexp = 13 - ex;
                        scale = __uint_as_float((uint32_t)(127 + kexp) << 23);
    #pragma unroll 1
                        for (int g = 0; g < steps; ++g) {
                            const uint32_t dst = again(tid + g * kProducers, v);
                            split(v, dst);
                        }
                    }
                }
                // under 2^-15 a scaled value's pair errs by more than 2^-21 of it (2^-36)
                slow = slow || (mn != 0xFFFFFFFFu && (int)((mn + 1u) >> 24) - 127 + kexp < -15);
            }
            publish(p, &sg, xfull, hdr, hready, kexp, slow, tid, lane);
        }
    }
    stages_done(p, sg, xempty, abort_flag, tid);
}

// Staging from boxes (stride 1, fp32, rectangles, rows of a multiple of 16 bytes): one tensor copy
// brings a block's window, 16 channels of th + 2 rows from the 16-byte boundary left of it, with zeros
// outside the image and beyond the last channel; the six warps only read, split and store, neighbouring
// lanes neighbouring positions.  With produce_async, a third of these warps' time went into issuing
// copies (some 1300 clocks for eight by each warp, all six at once after the block's barrier, the
// copies' data long there when it was wanted).  64 -> 64 at 224x224 with the pool, batch 32:
// 351 -> 326 us, 64 -> 128 at 112x112 153 -> 135; the next item's values are read before this one is
// split (334 against 328 in the benchmark's step; 375 with four items unrolled).
__device__ __forceinline__ void produce_box(const TcParams& p, const CUtensorMap* map, unsigned char* smem, uint32_t xfull, uint32_t xempty,
                                            uint32_t rfull, volatile int* abort_flag, uint2* red, float2* hdr, uint32_t hready, int rank, int pair, int pairs) {
    const int tid = (int)threadIdx.x - kPromoteWarps * 32, lane = tid & 31, warp = tid >> 5;
    const int cw = (p.th + 2) * p.rw;                // words of a channel's box
    const uint32_t bytes = 64u * (uint32_t)cw;       // of a box: a multiple of 256
    // the copies' cursor (thread 0): unit, block
    int iu = pair, icb = 0, icb1 = 0, issued = 0, x0 = 0, y0 = 0, n0 = 0;
    auto issue = [&]() {
        if (iu >= p.n_units) return;
        if (icb == icb1) {
            const Unit U = unit_of(p, iu, rank);
            icb = U.cb0;
            icb1 = U.cb1;
            x0 = (U.ox0 - 1) & ~3;                   // 16-byte boundary
            y0 = U.oy0 - 1;
            n0 = U.n;
        }
        const uint32_t s = (uint32_t)(issued % p.rs), bar = rfull + 8 * s;
        mbar_expect_tx(bar, bytes);
        box_load(smem_u32(smem) + p.ring_off + s * bytes, map, x0, y0, 16 * icb, n0, bar);
        ++issued;
        if (++icb == icb1) iu += pairs;
    };
    int done = 0, slot = 0, ph = 0;                  // blocks taken, their stage, its use
    // nothing in flight at the exit: after a timeout the boxes asked for land first
    auto drain = [&]() {
        if (tid != 0 || done == issued) return;
        const long long t0 = clock64();
        for (; done < issued; ++done)
            while (!mbar_try(rfull + 8 * (done % p.rs), (uint32_t)(done / p.rs) & 1u) && clock64() - t0 < kDrainCycles) {}
        if (clock64() - t0 >= kDrainCycles) atomicOr(p.status, kErrDrain);
    };
    if (tid == 0)
        for (int r = 0; r < p.rs; ++r) issue();
    int kexp = 0;
    Stage sg;
    for (int u = pair; u < p.n_units; u += pairs) {
        const Unit U = unit_of(p, u, rank);
        const int shift = (U.ox0 - 1) & 3, blocks = U.cb1 - U.cb0;
        for (int cb = 0; cb < blocks; ++cb) {
            bool ok = sg.e < p.xs || wait_bar(xempty + 8 * sg.s, (sg.ph & 1) ^ 1, p, abort_flag, kErrSpace);
            ok = ok && wait_bar(rfull + 8 * slot, (uint32_t)ph & 1u, p, abort_flag, kErrData);
            unsigned char* st = smem + p.x_off + (size_t)sg.s * p.x_stage;
            const float* raw = reinterpret_cast<const float*>(smem + p.ring_off + (uint32_t)slot * bytes) + shift;
            uint32_t mn = 0xFFFFFFFFu, mx = 0;
            __half2 hmx = __half2half2(__ushort_as_half(0));
            float scale = __uint_as_float((uint32_t)(127 + kexp) << 23);
            // item i: eight channels of a staged position (zeros: the two positions after the last row)
            auto take = [&](int i, float (&v)[8]) {
                const int k = i >= p.P ? 1 : 0, q = i - k * p.P, r = (int)fdiv((uint32_t)q, p.d_wp);
                const float* f = raw + 8 * k * cw + r * p.rw + (q - r * p.Wp);
                const bool in = r < p.th + 2;
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] = in ? f[j * cw] : 0.0f;
                return st + (uint32_t)k * p.plane + 16u * (uint32_t)q;
            };
            auto put = [&](const float (&v)[8], unsigned char* d) {
                // the smallest |v| as an ordered integer, a zero as the largest
#pragma unroll
                for (int j = 0; j < 8; j += 2)
                    mn = min(min(mn, 2u * __float_as_uint(v[j]) - 1u), 2u * __float_as_uint(v[j + 1]) - 1u);
                uint4 hi, lo;
                split8(v, scale, &hi, &lo, &hmx);
                *reinterpret_cast<uint4*>(d) = hi;
                *reinterpret_cast<uint4*>(d + 2 * p.plane) = lo;
            };
            if (ok) {
                float v[8];
                unsigned char* d = take(tid, v);
                for (int i = tid; i < 2 * p.P; i += kProducers) {
                    float w[8];
                    unsigned char* dn = d;
                    if (i + kProducers < 2 * p.P) dn = take(i + kProducers, w);
                    put(v, d);
                    d = dn;
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[j] = w[j];
                }
            }
            // the larger half of the largest hi parts; NaN is the largest of all
            const uint32_t b = *reinterpret_cast<const uint32_t*>(&hmx);
            mx = max(b & 0xFFFFu, b >> 16);
            if (!combine<true>(&mx, &mn, ok, red, &sg.par, warp, lane)) return drain();
            // as in produce_async: a block beyond the scale is taken again
            bool slow = false;
            if (mn != 0xFFFFFFFFu && (mx < 0x6800u || mx >= 0x7800u)) {
                mx = 0;
#pragma unroll 1
                for (int i = tid; i < 2 * p.P; i += kProducers) {
                    float v[8];
                    take(i, v);
                    for (int j = 0; j < 8; ++j) mx = max(mx, 2u * __float_as_uint(v[j]));
                }
                if (!combine<true>(&mx, &mn, ok, red, &sg.par, warp, lane)) return drain();
                const int ex = (int)(mx >> 24) - 127;
                slow = ex < -60 || ex > 120;   // also infinities and NaN
                if (!slow) {
                    kexp = 13 - ex;
                    scale = __uint_as_float((uint32_t)(127 + kexp) << 23);
#pragma unroll 1
                    for (int i = tid; i < 2 * p.P; i += kProducers) {
                        float v[8];
                        unsigned char* d = take(i, v);
                        put(v, d);
                    }
                    bar_or<1, kProducers>(false);   // all have read the box
                }
            }
            slow = slow || (mn != 0xFFFFFFFFu && (int)((mn + 1u) >> 24) - 127 + kexp < -15);
            ++done;
            if (++slot == p.rs) { slot = 0; ++ph; }
            if (tid == 0) issue();                  // into the stage just read
            publish(p, &sg, xfull, hdr, hready, kexp, slow, tid, lane);
        }
    }
    stages_done(p, sg, xempty, abort_flag, tid);
}

// fp16 rows of odd length, or inputs aligned to one value only: loads run two items ahead in registers.
template <int S>
__device__ __forceinline__ void produce_f16(const TcParams& p, unsigned char* smem, uint32_t xfull, uint32_t xempty,
                                            volatile int* abort_flag, uint2* red, float2* hdr, uint32_t hready, int rank, int pair, int pairs) {
    constexpr int UN = 2;
    constexpr int NPL = S == 1 ? 1 : 4;
    const int tid = (int)threadIdx.x - kPromoteWarps * 32, lane = tid & 31, warp = tid >> 5;
    const uint32_t HW = (uint32_t)p.H * p.W;
    uint32_t* table = reinterpret_cast<uint32_t*>(smem + p.tab_off);
    const int items = 2 * NPL * p.P, groups = (items + UN * kProducers - 1) / (UN * kProducers);
    Stage sg;
    for (int u = pair; u < p.n_units; u += pairs) {
        const Unit U = unit_of(p, u, rank);
        const int n0 = first_image(p, U);
        for (int i = tid; i < p.P; i += kProducers) table[i] = window_entry<S>(p, U, i, n0);
        bar_or<1, kProducers>(false);
        const unsigned short* xn = static_cast<const unsigned short*>(p.x) + (size_t)n0 * p.C * HW;
        auto load = [&](uint32_t (&v)[UN][8], int cb, int g) {
            const unsigned short* xc = xn + (size_t)cb * 16 * HW;   // uniform: a load adds the lane's offset
            const bool whole = cb * 16 + 16 <= p.C;
#pragma unroll
            for (int a = 0; a < UN; ++a) {
                int k, pos;
                uint32_t t = kOut, off;
                if (item_of<S>(p, tid + (g * UN + a) * kProducers, items, &k, &pos)) t = table[pos];
                const bool in = input_of<S>(p, t, k, HW, &off);
#pragma unroll
                for (int j = 0; j < 8; ++j) v[a][j] = 0;
                if (whole) {
                    if (in) {
#pragma unroll
                        for (int j = 0; j < 8; ++j) v[a][j] = __ldg(xc + (size_t)j * HW + off);
                    }
                } else {
                    const int nch = in ? p.C - cb * 16 - 8 * (k & 1) : 0;
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (j < nch) v[a][j] = __ldg(xc + (size_t)j * HW + off);
                }
            }
        };
        int cb = U.cb0, g = 0;
        uint32_t bad = 0;
        unsigned char* st = nullptr;
        bool ok = true, failed = false;
        // one group: the next one's loads, this one's stores, and the end of the block after its last
        auto step = [&](uint32_t (&cur)[UN][8], uint32_t (&nxt)[UN][8]) {
            const bool last = g == groups - 1;
            const int ncb = last ? cb + 1 : cb, ng = last ? 0 : g + 1;
            if (ncb < U.cb1) load(nxt, ncb, ng);
            if (g == 0) {
                ok = sg.e < p.xs || wait_bar(xempty + 8 * sg.s, (sg.ph & 1) ^ 1, p, abort_flag, kErrSpace);
                st = smem + p.x_off + (size_t)sg.s * p.x_stage;
                bad = 0;
            }
            if (ok) {
#pragma unroll
                for (int a = 0; a < UN; ++a) {
                    int k, pos;
                    if (!item_of<S>(p, tid + (g * UN + a) * kProducers, items, &k, &pos)) continue;
                    uint32_t w[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        w[j] = cur[a][2 * j] | cur[a][2 * j + 1] << 16;
                        bad |= ((w[j] & 0x7C007C00u) + 0x04000400u) & 0x80008000u;   // exponent 31: not finite
                    }
                    *reinterpret_cast<uint4*>(st + (uint32_t)k * p.plane + (uint32_t)pos * 16u) = make_uint4(w[0], w[1], w[2], w[3]);
                }
            }
            if (last) {
                uint32_t mn = 0;
                failed = !combine<false>(&bad, &mn, ok, red, &sg.par, warp, lane);
                if (failed) return;
                publish(p, &sg, xfull, hdr, hready, 0, bad != 0, tid, lane);
            }
            cb = ncb;
            g = ng;
        };
        uint32_t va[UN][8], vb[UN][8];
        load(va, cb, 0);
        while (true) {
            step(va, vb);
            if (failed) return;
            if (cb >= U.cb1) break;
            step(vb, va);
            if (failed) return;
            if (cb >= U.cb1) break;
        }
    }
    stages_done(p, sg, xempty, abort_flag, tid);
}

// ---------------------------------------------------------------------------- sums in fp32

// The pairs of a slow block's inputs err by up to 2^-36 2^-kexp each, and so a sum by up to the filter's
// sum of |w| times that.  2^21 times as much (p.unheld times the block's factor) and more is a sum to
// 2^-21 of itself.  Units with a smaller one, with an infinity or a NaN are noted in a bitmap, a bit per
// unit of the CTA in their order, the last bit for all from there on, and summed again by the eight
// summing warps after the CTA's last unit, when the pipeline's shared memory is theirs and nobody waits
// for them.  Summed at once in the epilogue, from global memory by a thread a position, such units took
// so long that one of 512 channels kept the other roles waiting for 27 ms, with a limit of one second.
constexpr unsigned kRedoOff = 896;   // in shared memory
constexpr int kRedoBits = 1024;

// Whether a thread's sums hold such a one: position tiles as in the epilogue.
template <int MT>
__device__ __forceinline__ bool unheld(const TcParams& p, const Unit& U, const float (&acc)[128], float lim, int half, int pos) {
    uint32_t top = 0;
    const uint32_t least = __float_as_uint(lim);
#pragma unroll
    for (int i = 0; i < (MT == 4 ? 2 : 1); ++i) {
        constexpr int NJ = MT == 4 ? 64 : 128;
        const int pl = pos + 128 * (MT == 4 ? 2 * half + i : (MT == 2 ? half : 0));
        const int r = (int)fdiv((uint32_t)pl, p.d_wp);
        const bool in = p.tw ? U.n < p.N && r < min(p.th, p.Ho - U.oy0) && pl - r * p.Wp < min(p.tw, p.Wo - U.ox0) : U.q0 + pl < p.Q;
        const int nf = in ? min(p.NC, p.Cout - U.r0) - (MT == 1 ? 128 * half : 0) : 0;
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            const uint32_t v = (__float_as_uint(acc[i * 64 + j]) & 0x7FFFFFFFu) - least;   // below: wraps
            top = max(top, j < nf ? v : 0u);
        }
    }
    return top >= 0x7F800000u - least;
}

// A unit's outputs from the packed layout in fp32, in the order of the FFMA kernel; only kept taps are
// read.  Rounds of eight tasks, a warp each: two groups of eight filters by 128 positions (or 32 pooled
// outputs), a lane four of the positions.  16 channels of the unit's window at a time are staged in fp32
// as the MMAs' operand is (a plane a channel, at stride 2 a parity and channel; zeros outside the
// image), so that a tap is one offset for all positions; a lane lists the kernels of one channel and
// group, a slot at a time, with their offsets, and all lanes apply the list.  us a call, keep 0.3, fp32:
//                              ordinary   one infinity   every unit   FFMA kernel
//   256 -> 256, 56x56, N 32      201          720          2710           517
//   512 -> 512, 14x14, N 32       70         1200          1250           187
//   64 -> 64, 224x224, N 32, pool 326         610          4860           553
// (from global memory 6600 and 34900, 21600 and 22000, 4000 and 99000).  The loads of shared memory and
// the two warps a scheduler bound it.
template <int S, typename T, int MT>
__device__ __forceinline__ void redo_unit(const TcParams& p, const Unit& U, unsigned char* smem, int tid, int warp, int lane) {
    constexpr int NG = 2, NPL = S == 1 ? 1 : 4;
    const bool pool = p.pool && p.KS == 1;
    const int PW = (int)(p.plane / 16);   // words of a plane: 16 channels' fit two of the pipeline's stages
    const uint32_t HW = (uint32_t)p.H * p.W;
    const int n0 = first_image(p, U), Hq = p.Ho >> 1, Wq = p.Wo >> 1, cols = max(p.tw >> 1, 1);
    uint32_t* table = reinterpret_cast<uint32_t*>(smem + p.tab_off);
    float* xs = reinterpret_cast<float*>(smem + p.x_off);
    float4* list = reinterpret_cast<float4*>(smem + p.ring_off) + 64 * warp;   // 32 kernels: weights, offsets
    bar_or<2, kPromoteWarps * 32>(false);
    for (int i = tid; i < p.P; i += kPromoteWarps * 32) table[i] = window_entry<S>(p, U, i, n0);
    const int tasks = (p.G + NG - 1) / NG * MT;
    for (int k0 = 0; k0 < tasks; k0 += kPromoteWarps) {
        const int g = (k0 + warp) / MT * NG, t = (k0 + warp) % MT;
        // slot `lane` of the groups: is its filter one of the unit's
        const uint32_t co = lane < NG * kF && g * kF + lane < p.G * kF ? p.perm[g * kF + lane] : kPadSlot;
        const uint32_t mine = __ballot_sync(0xFFFFFFFFu, co != kPadSlot && (int)co >= U.r0 && (int)co < U.r0 + p.NC);
        // this lane's four positions and their outputs
        Point o[4];
        const float* at[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            if (pool) {
                const int i = lane + 32 * t, r = i / cols, c = i - r * cols;
                o[b].n = U.n;
                o[b].oy = U.oy0 + 2 * r + (b >> 1);
                o[b].ox = U.ox0 + 2 * c + (b & 1);
                o[b].in = U.n < p.N && 2 * r < p.th && o[b].oy / 2 < Hq && o[b].ox / 2 < Wq;
                at[b] = xs + (o[b].in ? (2 * r + (b >> 1)) * p.Wp + 2 * c + (b & 1) : 0);
            } else {
                o[b] = point_of(p, U, 128 * t + 32 * b + lane);
                at[b] = xs + 128 * t + 32 * b + lane;
            }
        }
        float a[NG][kF][4];
#pragma unroll
        for (int i = 0; i < NG * kF * 4; ++i) a[i / (kF * 4)][i / 4 % kF][i % 4] = 0.0f;
        for (int cb = U.cb0; cb < U.cb1; ++cb) {
            bar_or<2, kPromoteWarps * 32>(false);   // the table is complete, the block before done with
            const T* xc = static_cast<const T*>(p.x) + ((size_t)n0 * p.C + cb * 16) * HW;
            const int nc = min(16, p.C - cb * 16);
            for (int i = tid; i < p.P; i += kPromoteWarps * 32) {
                const uint32_t e = table[i];
#pragma unroll
                for (int pl = 0; pl < NPL; ++pl) {
                    const bool in = e != kOut && (!(pl & 1) || (e & 1u)) && (!(pl & 2) || (e & 2u));
                    const T* v = xc + (in ? (e >> 2) + (uint32_t)(pl >> 1) * p.W + (uint32_t)(pl & 1) : 0u);
#pragma unroll
                    for (int c = 0; c < 16; ++c)
                        xs[(c * NPL + pl) * PW + i] = in && c < nc ? (float)__ldg(v + (size_t)c * HW) : 0.0f;
                }
            }
            bar_or<2, kPromoteWarps * 32>(false);
            if (mine == 0) continue;
            // lane 16 h + c: the kernels of channel c and group h, in the order of their slots
            const int h = lane >> 4, c = lane & 15;
            const size_t gc = (size_t)(g + h) * p.C + cb * 16 + c;
            uint64_t d = g + h < p.G && c < nc ? __ldg(p.desc + gc) : 0;
            int left = (int)(d & 15u);
            const float4* v = p.vals + (left ? __ldg(p.kofs + gc) : 0u);
            float4 w = left ? __ldg(v) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            d >>= 4;
#pragma unroll
            for (int f = 0; f < kF; ++f) {
                const bool has = left > 0 && (int)(d >> 3 & 7u) == f, use = has && (mine >> (kF * h + f) & 1u);
                const uint32_t bal = __ballot_sync(0xFFFFFFFFu, use);
                if (use) {
                    const int i = __popc(bal & ((1u << lane) - 1u));
                    uint32_t m = p.masks[d & 7u];
                    int off[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int k = __ffs((int)m) - 1, ty = k / 3, tx = k - 3 * ty;
                        m &= m - 1;
                        off[j] = c * NPL * PW + (S == 1 ? ty * p.Wp + tx
                                                        : ((ty != 1 ? 2 : 0) + (tx != 1 ? 1 : 0)) * PW + (ty == 0 ? 0 : p.Wp) + (tx == 0 ? 0 : 1));
                    }
                    list[2 * i] = w;
                    reinterpret_cast<int4*>(list)[2 * i + 1] = make_int4(off[0], off[1], off[2], off[3]);
                }
                if (has) {
                    d >>= 6;
                    ++v;
                    if (--left) w = __ldg(v);
                }
                __syncwarp();
                const int n1 = __popc(bal & 0xFFFFu), n2 = __popc(bal);
                auto apply = [&](int i, float (&s)[4]) {
                    const float4 u = list[2 * i];
                    const int4 q = reinterpret_cast<const int4*>(list)[2 * i + 1];
#pragma unroll
                    for (int b = 0; b < 4; ++b)
                        s[b] = fmaf(u.w, at[b][q.w], fmaf(u.z, at[b][q.z], fmaf(u.y, at[b][q.y], fmaf(u.x, at[b][q.x], s[b]))));
                };
                for (int i = 0; i < n1; ++i) apply(i, a[0][f]);
                for (int i = n1; i < n2; ++i) apply(i, a[1][f]);
                __syncwarp();
            }
        }
#pragma unroll
        for (int i = 0; i < NG * kF; ++i) {
            if (!(mine >> i & 1u)) continue;
            const float (&s)[4] = a[i / kF][i % kF];
            const int co_i = (int)__shfl_sync(0xFFFFFFFFu, co, i);
            const float bias = p.KS == 1 && p.bias ? p.bias[co_i] : 0.0f;
            if (pool) {
                const float m = fmaxf(fmaxf(s[0], s[1]), fmaxf(s[2], s[3]));
                if (o[0].in)
                    static_cast<T*>(p.y)[(((size_t)U.n * p.Cout + co_i) * Hq + o[0].oy / 2) * Wq + o[0].ox / 2] =
                        out_of<T>(relu_of(m + bias, p.relu));
                continue;
            }
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                if (!o[b].in) continue;
                const size_t to = (((size_t)o[b].n * p.Cout + co_i) * p.Ho + o[b].oy) * p.Wo + o[b].ox;
                if (p.KS > 1) p.ws[(size_t)U.ks * p.ws_stride + to] = s[b];
                else static_cast<T*>(p.y)[to] = out_of<T>(relu_of(s[b] + bias, p.relu));
            }
        }
    }
}

// The noted units (not inlined: the loops before it would spill).
template <int S, typename T, int MT>
__device__ __noinline__ void redo_units(const TcParams& p) {
    extern __shared__ __align__(128) unsigned char smem[];
    const uint32_t* redo = reinterpret_cast<const uint32_t*>(smem + kRedoOff);
    const int warp = __shfl_sync(0xFFFFFFFFu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int rank = blockIdx.x & 1, pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
    for (int i = 0; i < kRedoBits; ++i) {
        if (!(redo[i / 32] >> (i & 31) & 1u)) continue;
        for (long long u = pair + (long long)i * pairs; u < p.n_units; u += pairs) {
            redo_unit<S, T, MT>(p, unit_of(p, (int)u, rank), smem, threadIdx.x, warp, lane);
            if (i < kRedoBits - 1) break;
        }
    }
}

// ---------------------------------------------------------------------------- the kernel

template <int S, typename T, int MT>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1) pconv_tc(const __grid_constant__ TcParams p, const __grid_constant__ CUtensorMap tmap) {
    constexpr int HL = sizeof(T) == 4 ? 2 : 1;
    constexpr int TCOL = 256 / MT;                // accumulator columns of a 128-position tile
    constexpr bool LL = HL == 2 && MT == 1;
    extern __shared__ __align__(128) unsigned char smem[];
    const int warp = __shfl_sync(0xFFFFFFFFu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int rank = blockIdx.x & 1, pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
    const uint32_t bar0 = smem_u32(smem);
    const uint32_t xfull = bar0, xempty = xfull + 8 * kMaxXStages, hfull = xempty + 8 * kMaxXStages,
                   hempty = hfull + 8 * kMaxWSlots, lfull = hempty + 8 * kMaxWSlots, lempty = lfull + 8 * kMaxWSlots,
                   tfull = lempty + 8 * kMaxWSlots, tempty = tfull + 16, drain = tempty + 16, rfull = drain + 8, hready = rfull + 8 * kMaxRaw;
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(smem + 640);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + 644);
    float2* hdr = reinterpret_cast<float2*>(smem + 704);
    uint2* red = reinterpret_cast<uint2*>(smem + 768);
    uint32_t* redo = reinterpret_cast<uint32_t*>(smem + kRedoOff);

    if (threadIdx.x < kRedoBits / 32) redo[threadIdx.x] = 0;
    if (warp == kMmaWarp) {
        if (lane == 0) {
            // The leader (rank 0) issues the pair's MMAs: its `full` barriers take the arrivals of
            // both CTAs (of the weights: its own bytes and the peer's relay)
            for (int i = 0; i < p.xs; ++i) {
                mbar_init(xfull + 8 * i, 2 * kProducerWarps);
                mbar_init(xempty + 8 * i, 1);
            }
            for (int i = 0; i < p.hs; ++i) {
                mbar_init(hfull + 8 * i, rank == 0 ? 2 : 1);
                mbar_init(hempty + 8 * i, 1);
            }
            for (int i = 0; i < p.ls; ++i) {
                mbar_init(lfull + 8 * i, rank == 0 ? 2 : 1);
                mbar_init(lempty + 8 * i, 1);
            }
            for (int i = 0; i < 2; ++i) {
                mbar_init(tfull + 8 * i, 1);
                mbar_init(tempty + 8 * i, 2 * kPromoteWarps);
            }
            mbar_init(drain, 1);
            for (int i = 0; i < kMaxRaw; ++i) mbar_init(rfull + 8 * i, 1);
            for (int i = 0; i < kHdr; ++i) mbar_init(hready + 8 * i, 1);
            *abort_flag = 0;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(s_tmem)), "r"(kTmemColumns) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    cluster_sync();
    fence_after();
    const uint32_t tbase = __shfl_sync(0xFFFFFFFFu, *s_tmem, 0);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (warp < kPromoteWarps) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 176;");
        // ---- sums in fp32 registers, epilogue.  Warp w: tensor-memory lanes 32 (w % 4) ...,
        // columns 128 (w / 4) ...; a lane is one position of a tile, a column one filter.
        const int half = warp >> 2, pos = 32 * (warp & 3) + lane;
        const uint32_t tw = tbase + ((uint32_t)(32 * (warp & 3)) << 16) + 128u * half;
        float acc[128];
#pragma unroll
        for (int j = 0; j < 128; ++j) acc[j] = 0.0f;
        uint32_t e = 0, un = 0;
        bool ok = true;
        for (int u = pair; u < p.n_units; u += pairs) {
            const Unit U = unit_of(p, u, rank);
            // this unit's biases (read after the barrier below; the unit before it reads the others)
            float* s_bias = reinterpret_cast<float*>(smem + 1024) + 256 * (un & 1);
            ++un;
            s_bias[threadIdx.x] = p.bias && U.r0 + (int)threadIdx.x < p.Cout ? __ldg(p.bias + U.r0 + threadIdx.x) : 0.0f;
            float lim = -1.0f;
            // columns of this warp: 32-column groups that hold filters of the unit
            bool act[4];
#pragma unroll
            for (int jb = 0; jb < 4; ++jb) act[jb] = ((128 * half + 32 * jb) % TCOL) < p.NC;
            for (int cb = U.cb0; cb < U.cb1 && ok; ++cb, ++e) {
                const uint32_t b = e & 1u;
                const uint32_t hb = hready + 8 * (e & (kHdr - 1)), hp = (e / kHdr) & 1u;
                const bool h1 = mbar_try(hb, hp), t1 = mbar_try(tfull + 8 * b, (e >> 1) & 1u);
                ok = (h1 || wait_bar(hb, hp, p, abort_flag, kErrData)) &&
                     (t1 || wait_bar(tfull + 8 * b, (e >> 1) & 1u, p, abort_flag, kErrData));
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                fence_after();
                const float2 h = hdr[e & (kHdr - 1)];
                lim = fmaxf(lim, h.y != 0.0f ? h.x * p.unheld : -1.0f);
#pragma unroll
                for (int jb = 0; jb < 4; ++jb) {
                    if (act[jb]) {
                        uint32_t r[32];
                        tmem_ld32(tw + 256u * b + 32u * jb, r);
#pragma unroll
                        for (int j = 0; j < 32; ++j) acc[32 * jb + j] = fmaf(__uint_as_float(r[j]), h.x, acc[32 * jb + j]);
                    }
                }
                fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_leader(tempty + 8 * b);
            }
            if (bar_or<2, kPromoteWarps * 32>(!ok)) break;
            // before the pooled epilogue and after the other (all after: 64 -> 64 224x224 336 for 327 us; all
            // before: 256 -> 256 56x56 202.5 for 201.6, 90 -> 150 45x61 20.0 for 19.4)
            auto note_unheld = [&]() {
                if (lim >= 0.0f && unheld<MT>(p, U, acc, lim, half, pos)) {
                    const int bit = min((int)un - 1, kRedoBits - 1);
                    atomicOr(redo + bit / 32, 1u << (bit & 31));
                }
            };
            if (p.pool && p.KS == 1) {
                note_unheld();
                // 2x2 max-pool: a few filters of every position at a time through shared memory, each
                // row of outputs at an even pitch (a pooled output is two 8-byte loads), a warp a
                // filter, a lane up to MT pooled outputs whose offsets are the same for every filter.
                // MT 1: each half of the warps pools its own 128 filters.
                constexpr int TPH = MT == 4 ? 2 : 1;          // tiles of a warp
                constexpr int NF = MT == 4 ? 8 : 16;          // filters a step
                constexpr int NW = MT == 1 ? 4 : 8;           // warps sharing them
                const int pitch = (p.tw + 1) & ~1, plane = p.th * pitch;
                float* pb = reinterpret_cast<float*>(smem + p.pool_off) + (MT == 1 ? half * NF * plane : 0);
                const int Hq = p.Ho >> 1, Wq = p.Wo >> 1, HqWq = Hq * Wq;
                int wr[TPH];                                  // where this lane's positions go
#pragma unroll
                for (int i = 0; i < TPH; ++i) {
                    const int pl = pos + 128 * (MT == 4 ? 2 * half + i : (MT == 2 ? half : 0));
                    const int r = (int)fdiv((uint32_t)pl, p.d_wp), c = pl - r * p.Wp;
                    wr[i] = r < p.th && c < p.tw ? r * pitch + c : -1;
                }
                int rd[MT], yo[MT];                           // this lane's pooled outputs
                const int py0 = U.oy0 >> 1, px0 = U.ox0 >> 1, cols = p.tw >> 1;
#pragma unroll
                for (int i = 0; i < MT; ++i) {
                    const int o = lane + 32 * i, r = o / max(cols, 1), c = o - r * cols;
                    const bool in = U.n < p.N && 2 * r < p.th && cols > 0 && py0 + r < Hq && px0 + c < Wq;
                    rd[i] = in ? 2 * r * pitch + 2 * c : -1;
                    yo[i] = r * Wq + c;
                }
                T* y = static_cast<T*>(p.y) + ((size_t)U.n * p.Cout + U.r0) * HqWq + (size_t)py0 * Wq + px0;
                const int nf = min(p.NC, p.Cout - U.r0);
#pragma unroll
                for (int fb = 0; fb < 128 / TPH / NF; ++fb) {
                    const int f0 = (MT == 1 ? 128 * half : 0) + NF * fb;
                    bar_or<2, kPromoteWarps * 32>(false);
#pragma unroll
                    for (int i = 0; i < TPH; ++i) {
                        if (wr[i] >= 0) {
#pragma unroll
                            for (int k = 0; k < NF; ++k) pb[k * plane + wr[i]] = acc[i * 64 + NF * fb + k];
                        }
                    }
                    bar_or<2, kPromoteWarps * 32>(false);
#pragma unroll
                    for (int k = 0; k < NF / NW; ++k) {
                        const int f = warp % NW + NW * k;
                        if (f0 + f < nf) {
                            const float b = s_bias[f0 + f];
                            T* yf = y + (size_t)(f0 + f) * HqWq;
#pragma unroll
                            for (int i = 0; i < MT; ++i) {
                                if (rd[i] >= 0) {
                                    const float* q = pb + f * plane + rd[i];
                                    const float2 u = *reinterpret_cast<const float2*>(q);
                                    const float2 v = *reinterpret_cast<const float2*>(q + pitch);
                                    const float m = fmaxf(fmaxf(u.x, u.y), fmaxf(v.x, v.y));
                                    yf[yo[i]] = out_of<T>(relu_of(m + b, p.relu));
                                }
                            }
                        }
                    }
                }
            } else {
#pragma unroll
                for (int i = 0; i < (MT == 4 ? 2 : 1); ++i) {
                    constexpr int NJ = MT == 4 ? 64 : 128;
                    const int pl = pos + 128 * (MT == 4 ? 2 * half + i : (MT == 2 ? half : 0));
                    const int f0 = MT == 1 ? 128 * half : 0;
                    const Point o = point_of(p, U, pl);
                    // filters to store: one predicate a store, no branch (a branch every four filters
                    // kept their loads and stores from overlapping: fp16 28x28 72 -> 84 us)
                    const int nf = o.in ? min(p.NC, p.Cout - U.r0) - f0 : 0, HoWo = p.Ho * p.Wo;
                    const size_t o0 = (((size_t)o.n * p.Cout + U.r0 + f0) * p.Ho + o.oy) * p.Wo + o.ox;
                    if (p.KS > 1) {
                        float* w = p.ws + (size_t)U.ks * p.ws_stride + o0;
#pragma unroll
                        for (int j = 0; j < NJ; ++j) {
                            if (j < nf) *w = acc[i * 64 + j];
                            w += HoWo;
                        }
                    } else {
                        T* w = static_cast<T*>(p.y) + o0;
#pragma unroll
                        for (int j = 0; j < NJ; j += 4) {
                            const float4 b = *reinterpret_cast<const float4*>(s_bias + f0 + j);
                            const float bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                if (j + k < nf) *w = out_of<T>(relu_of(acc[i * 64 + j + k] + bv[k], p.relu));
                                w += HoWo;
                            }
                        }
                    }
                }
                note_unheld();
            }
#pragma unroll
            for (int j = 0; j < 128; ++j) acc[j] = 0.0f;
        }
        if (!bar_or<2, kPromoteWarps * 32>(!ok) && __any_sync(0xFFFFFFFFu, redo[lane] != 0)) redo_units<S, T, MT>(p);
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");
        if (warp < kPromoteWarps + kProducerWarps) {
            if (S == 1 && HL == 2 && MT > 1 && p.box) produce_box(p, &tmap, smem, xfull, xempty, rfull, abort_flag, red, hdr, hready, rank, pair, pairs);
            else if (p.vec == 4) produce_async<S, T, 4>(p, smem, xfull, xempty, abort_flag, red, hdr, hready, rank, pair, pairs);
            else if (p.vec == 2) produce_async<S, T, 2>(p, smem, xfull, xempty, abort_flag, red, hdr, hready, rank, pair, pairs);
            else if constexpr (HL == 2) produce_async<S, T, 1>(p, smem, xfull, xempty, abort_flag, red, hdr, hready, rank, pair, pairs);
            else produce_f16<S>(p, smem, xfull, xempty, abort_flag, red, hdr, hready, rank, pair, pairs);
            asm volatile("cp.async.wait_all;" ::: "memory");   // after a timeout: nothing in flight at the exit
        } else if (warp == kLoaderWarp) {
            // ---- weights: a slot holds this CTA's half of the unit's filters for a row of three
            // taps of a 16-channel block, [tap][8 channels][filter], the lo and hi parts in rings of
            // their own: a lo slot is free after its cross products, a hi slot after the last ones.
            // One copy a slot: copies of a quarter made the 56x56 layer a third slower.
            int hsl = 0, hph = 0, lsl = 0, lph = 0;
            bool ok = !p.no_fill;
            for (int u = pair; u < p.n_units && ok; u += pairs) {
                const Unit U = unit_of(p, u, rank);
                const unsigned char* src = p.wimg + ((size_t)(2 * U.fc + rank) * p.n_cb + U.cb0) * 6 * p.w_slot;
                for (int k = 3 * U.cb0; k < 3 * U.cb1; ++k) {
                    if (lph > 0) ok = wait_warp(lempty + 8 * lsl, (lph & 1) ^ 1, p, abort_flag, kErrSpace);
                    if (!ok) break;
                    if (elect_one()) {
                        mbar_expect_tx(lfull + 8 * lsl, p.w_slot);
                        bulk_load(bar0 + p.l_off + (uint32_t)lsl * p.w_slot, src + 3 * p.w_slot, p.w_slot, lfull + 8 * lsl);
                    }
                    __syncwarp();
                    if (++lsl == p.ls) { lsl = 0; ++lph; }
                    if (hph > 0) ok = wait_warp(hempty + 8 * hsl, (hph & 1) ^ 1, p, abort_flag, kErrSpace);
                    if (!ok) break;
                    if (elect_one()) {
                        mbar_expect_tx(hfull + 8 * hsl, p.w_slot);
                        bulk_load(bar0 + p.h_off + (uint32_t)hsl * p.w_slot, src, p.w_slot, hfull + 8 * hsl);
                    }
                    __syncwarp();
                    if (++hsl == p.hs) { hsl = 0; ++hph; }
                    src += k % 3 == 2 ? 4 * p.w_slot : p.w_slot;
                }
            }
            // nothing of this CTA in flight at its exit: the slots filled last have landed, and so have
            // the arrivals of the commits that free them (as in stages_done)
            const int nl = lph * p.ls + lsl, nh = hph * p.hs + hsl;
            for (int k = max(0, nl - p.ls); k < nl && ok; ++k)
                ok = wait_warp(lempty + 8 * (k % p.ls), (uint32_t)(k / p.ls) & 1u, p, abort_flag, kErrSpace);
            for (int k = max(0, nh - p.hs); k < nh && ok; ++k)
                ok = wait_warp(hempty + 8 * (k % p.hs), (uint32_t)(k / p.hs) & 1u, p, abort_flag, kErrSpace);
            const long long t0 = clock64();
            for (int k = max(0, nl - p.ls); k < nl; ++k)
                while (!mbar_try(lfull + 8 * (k % p.ls), (uint32_t)(k / p.ls) & 1u) && clock64() - t0 < kDrainCycles) {}
            for (int k = max(0, nh - p.hs); k < nh; ++k)
                while (!mbar_try(hfull + 8 * (k % p.hs), (uint32_t)(k / p.hs) & 1u) && clock64() - t0 < kDrainCycles) {}
            if (clock64() - t0 >= kDrainCycles) atomicOr(p.status, kErrDrain);
        } else if (warp == kMmaWarp && rank == 1) {
            // ---- the peer's relay: tells the leader of each weight slot that has landed here
            int hsl = 0, hph = 0, lsl = 0, lph = 0;
            bool ok = true;
            for (int u = pair; u < p.n_units && ok; u += pairs) {
                const Unit U = unit_of(p, u, rank);
                for (int k = 0; k < 3 * (U.cb1 - U.cb0); ++k) {
                    ok = wait_warp(lfull + 8 * lsl, (uint32_t)lph & 1u, p, abort_flag, kErrData);
                    if (!ok) break;
                    if (lane == 0) mbar_arrive_leader(lfull + 8 * lsl);
                    if (++lsl == p.ls) { lsl = 0; ++lph; }
                    ok = wait_warp(hfull + 8 * hsl, (uint32_t)hph & 1u, p, abort_flag, kErrData);
                    if (!ok) break;
                    if (lane == 0) mbar_arrive_leader(hfull + 8 * hsl);
                    if (++hsl == p.hs) { hsl = 0; ++hph; }
                }
            }
        } else if (warp == kMmaWarp) {
            // ---- the MMA issuer: the whole warp walks the stream (its operands then sit in uniform
            // registers; one lane in a divergent branch took 245 clocks an MMA), one lane issues
            uint32_t toff[9];
#pragma unroll
            for (int t = 0; t < 9; ++t) {
                const int ty = t / 3, tx = t % 3;
                if (S == 1) toff[t] = (uint32_t)(ty * p.Wp + tx);
                else
                    toff[t] = (uint32_t)((ty != 1 ? 2 : 0) + (tx != 1 ? 1 : 0)) * (HL * 2 * p.plane / 16) +
                              (uint32_t)((ty == 0 ? 0 : p.Wp) + (tx == 0 ? 0 : 1));
            }
            const uint32_t xlo = 2 * p.plane / 16;   // from a staged hi part to its lo part
            uint32_t e = 0;
            int s = 0, xph = 0, hsl = 0, hph = 0, lsl = 0, lph = 0;
            bool ok = true;
            for (int u = pair; u < p.n_units && ok; u += pairs) {
                const Unit U = unit_of(p, u, rank);
                const uint32_t idesc = (1u << 4) | ((uint32_t)(p.NC >> 3) << 17) | (16u << 24);
                const uint32_t wlead = (uint32_t)p.NC * 8u, wtap = 2 * wlead / 16;
                for (int cb = U.cb0; cb < U.cb1; ++cb, ++e) {
                    const uint32_t b = e & 1u;
                    if (e >= 2) ok = wait_warp(tempty + 8 * b, ((e >> 1) & 1u) ^ 1u, p, abort_flag, kErrSpace);
                    ok = ok && wait_warp(xfull + 8 * s, (uint32_t)xph & 1u, p, abort_flag, kErrData);
                    if (!ok) break;
                    fence_after();
                    const uint32_t xa = desc_lo(bar0 + p.x_off + (uint32_t)s * p.x_stage, p.plane);
                    const uint32_t d = tbase + 256u * b;
                    // l_x l_w (times 2^22) where asked for (small calls, 128-position tiles)
                    if (LL && p.ll) {
                        int l1 = lsl, lp1 = lph;
#pragma unroll
                        for (int r = 0; r < 3; ++r) {
                            ok = wait_warp(lfull + 8 * l1, (uint32_t)lp1 & 1u, p, abort_flag, kErrData);
                            if (!ok) break;
                            const uint32_t wl = desc_lo(bar0 + p.l_off + (uint32_t)l1 * p.w_slot, wlead);
                            if (elect_one()) {
#pragma unroll
                                for (int c = 0; c < 3; ++c) {
                                    const uint32_t xt = xa + toff[3 * r + c] + xlo;
#pragma unroll
                                    for (int i = 0; i < MT; ++i) {
                                        if (r + c == 0) mma<0>(d + TCOL * i, xt + 128u * i, wl + wtap * c, idesc);
                                        else mma<1>(d + TCOL * i, xt + 128u * i, wl + wtap * c, idesc);
                                    }
                                }
                            }
                            __syncwarp();
                            if (++l1 == p.ls) { l1 = 0; ++lp1; }
                        }
                        if (!ok) break;
                    }
                    // cross terms h_x l_w + l_x h_w (times 2^11)
                    int h1 = hsl, hp1 = hph;
#pragma unroll
                    for (int r = 0; r < 3; ++r) {
                        ok = wait_warp(lfull + 8 * lsl, (uint32_t)lph & 1u, p, abort_flag, kErrData) &&
                             wait_warp(hfull + 8 * h1, (uint32_t)hp1 & 1u, p, abort_flag, kErrData);
                        if (!ok) break;
                        const uint32_t wh = desc_lo(bar0 + p.h_off + (uint32_t)h1 * p.w_slot, wlead);
                        const uint32_t wl = desc_lo(bar0 + p.l_off + (uint32_t)lsl * p.w_slot, wlead);
                        if (elect_one()) {
#pragma unroll
                            for (int c = 0; c < 3; ++c) {
                                const uint32_t xt = xa + toff[3 * r + c];
#pragma unroll
                                for (int i = 0; i < MT; ++i) {
                                    if (r + c == 0) {
                                        if (LL && p.ll) mma<2>(d + TCOL * i, xt + 128u * i, wl + wtap * c, idesc);
                                        else mma<0>(d + TCOL * i, xt + 128u * i, wl + wtap * c, idesc);
                                    } else {
                                        mma<1>(d + TCOL * i, xt + 128u * i, wl + wtap * c, idesc);
                                    }
                                    if constexpr (HL == 2) mma<1>(d + TCOL * i, xt + 128u * i + xlo, wh + wtap * c, idesc);
                                }
                            }
                            commit_pair(lempty + 8 * lsl);
                        }
                        __syncwarp();
                        if (++lsl == p.ls) { lsl = 0; ++lph; }
                        if (++h1 == p.hs) { h1 = 0; ++hp1; }
                    }
                    if (!ok) break;
                    // h_x h_w, the cross terms scaled back by the first
#pragma unroll
                    for (int r = 0; r < 3; ++r) {
                        const uint32_t wh = desc_lo(bar0 + p.h_off + (uint32_t)hsl * p.w_slot, wlead);
                        if (elect_one()) {
#pragma unroll
                            for (int c = 0; c < 3; ++c) {
                                const uint32_t xt = xa + toff[3 * r + c];
#pragma unroll
                                for (int i = 0; i < MT; ++i) {
                                    if (r + c == 0) mma<2>(d + TCOL * i, xt + 128u * i, wh + wtap * c, idesc);
                                    else mma<1>(d + TCOL * i, xt + 128u * i, wh + wtap * c, idesc);
                                }
                            }
                            commit_pair(hempty + 8 * hsl);
                            if (r == 2) {
                                commit_pair(tfull + 8 * b);
                                commit_pair(xempty + 8 * s);
                            }
                        }
                        __syncwarp();
                        if (++hsl == p.hs) { hsl = 0; ++hph; }
                    }
                    if (++s == p.xs) { s = 0; ++xph; }
                }
            }
            if (!ok) {   // every MMA issued so far ends before the pair frees its tensor memory
                if (elect_one()) commit(drain);
                __syncwarp();
                const long long t0 = clock64();
                while (!mbar_try(drain, 0))
                    if (clock64() - t0 > kDrainCycles) { atomicOr(p.status, kErrDrain); break; }
                // arrivals of the commits before it may still be on their way to the peer: they get 10 us
                for (const long long t1 = clock64(); clock64() - t1 < kSettleCycles;) {}
            }
        }
    }
    __syncwarp();
    fence_before();
    __syncthreads();
    cluster_sync();   // the leader's MMAs read this CTA's shared memory and signal its barriers
    if (warp == kMmaWarp) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(kTmemColumns) : "memory");
    }
}

// ---------------------------------------------------------------------------- weights

// The fp16 pairs of every kept weight into the zeroed image [16-channel block][tap][hi, lo]
// [8 channels][filter][8]: one thread per (filter group, channel) of the packed layout.
__global__ void expand_weights(const uint32_t* perm, const uint64_t* desc, const uint32_t* kofs, const float4* vals,
                               const TcParams p, __half* out) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= (long long)p.G * p.C) return;
    const int g = (int)(i / p.C), c = (int)(i - (long long)g * p.C);
    uint64_t d = desc[i];
    const int cnt = (int)(d & 15u);
    d >>= 4;
    const float4* w4 = vals + kofs[i];
    const float s = __uint_as_float((uint32_t)(127 + p.wexp) << 23);
    for (int k = 0; k < cnt; ++k, d >>= 6) {
        const uint32_t co = perm[g * kF + ((d >> 3) & 7u)];
        const float4 w = w4[k];
        const float wv[4] = {w.x, w.y, w.z, w.w};
        uint32_t m = p.masks[d & 7u];
        for (int j = 0; j < 4; ++j) {
            const int t = __ffs((int)m) - 1;
            m &= m - 1;
            const float v = wv[j] * s;
            const __half h = __float2half_rn(v);
            const __half l = __float2half_rn(fmaf(v, p.wbias, v - __half2float(h)) * 2048.0f);
            const int hf = p.NC / 2, half = (int)co / hf;   // halves of chunks, numbered through
            const size_t tap = (((size_t)half * p.n_cb + c / 16) * 18 + t) * 2 + (c % 16) / 8;
            const size_t o = (tap * hf + co % hf) * 8 + c % 8;
            out[o] = h;
            out[o + (size_t)18 * hf * 8] = l;
        }
    }
}

void fill_layer(const pp_layer* L, TcParams* p) {
    const unsigned char* img = static_cast<const unsigned char*>(L->dev);
    p->perm = reinterpret_cast<const uint32_t*>(img + L->off_perm);
    p->desc = reinterpret_cast<const uint64_t*>(img + L->off_desc);
    p->kofs = reinterpret_cast<const uint32_t*>(img + L->off_kofs);
    p->vals = reinterpret_cast<const float4*>(img + L->off_vals);
    p->C = L->cin_g;
    p->Cout = L->cout;
    p->G = L->G;
    p->NC = tensor_nc(L);
    p->n_cb = (L->cin_g + 15) / 16;
    p->wexp = L->tc_exp;
    p->wbias = (float)tensor_bias(L);
    for (int i = 0; i < kMaxPatterns; ++i) p->masks[i] = L->masks[i];
}

using TcKernel = void (*)(const TcParams, const CUtensorMap);

template <int S, typename T, int MT>
TcKernel pick(size_t need) {
    static std::atomic<int> done[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    if (!done[dev].load(std::memory_order_acquire)) {
        int optin = 0;
        if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
            (size_t)optin < need ||
            cudaFuncSetAttribute(pconv_tc<S, T, MT>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin) != cudaSuccess)
            return nullptr;
        done[dev].store(1, std::memory_order_release);
    }
    return pconv_tc<S, T, MT>;
}
template <int S, typename T>
TcKernel pick(int mt, size_t need) {
    return mt == 1 ? pick<S, T, 1>(need) : (mt == 2 ? pick<S, T, 2>(need) : pick<S, T, 4>(need));
}

constexpr size_t kSmemMax = 227 * 1024;

size_t align_up(size_t n, size_t a) { return (n + a - 1) / a * a; }

}  // namespace

cudaError_t tensor_build_weights(const pp_layer* L, void* dst, cudaStream_t st) {
    TcParams p{};
    fill_layer(L, &p);
    cudaError_t e = cudaMemsetAsync(dst, 0, tensor_weight_bytes(L), st);
    if (e != cudaSuccess) return e;
    const long long n = (long long)L->G * L->cin_g;
    expand_weights<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(p.perm, p.desc, p.kofs, p.vals, p, static_cast<__half*>(dst));
    return cudaGetLastError();
}

bool tensor_plan(const pp_layer* L, int N, int H, int W, int pool, int es, size_t ws_bytes, int sms, TensorPlan* out,
                 int ll) {
    if (!L->tc_ok || sms < 2) return false;
    const int S = L->stride, Ho = (H - 1) / S + 1, Wo = (W - 1) / S + 1;
    const int HL = es == 4 ? 2 : 1;
    const size_t out_bytes = (size_t)N * L->cout * Ho * Wo * sizeof(float);
    TensorPlan pl;
    pl.NC = tensor_nc(L);
    pl.n_fchunks = tensor_chunks(L);
    pl.n_cb = (L->cin_g + 15) / 16;
    pl.w_slot = (unsigned)pl.NC * 48;
    pl.pool_off = kHeadBytes;
    const int mt_max = pl.NC <= 64 ? 4 : (pl.NC <= 128 ? 2 : 1);
    double best = 0;
    bool have = false;
    // Tiles of 128, 256 or 512 positions: flat (no pool), or rectangles of a k-th of the width and as
    // many rows as fit, evened out
    for (int i = 0; i < 3 * 10; ++i) {
        const int k = i % 10 < 7 ? i % 10 : (i % 10 == 9 ? 16 : 4 * (i % 10) - 20);   // 0 ... 6, 8, 12, 16
        TensorPlan c = pl;
        c.MT = 1 << (i / 10);
        if (c.MT > (ll ? 1 : mt_max)) break;
        if (pool && k == 0) continue;
        const int M = 128 * c.MT;
        long long tiles;
        if (k == 0) {
            c.Wp = Wo + 1;
            const long long ip = (long long)(Ho + 1) * c.Wp;
            if (ip * N >= (1LL << 30)) continue;
            c.Ip = (int)ip;
            c.Q = ip * N;
            c.mstep = M;
            tiles = (c.Q + M - 1) / M;
            c.P = S == 1 ? M + 2 * c.Wp + 2 : M + c.Wp + 1;
            if (c.P / c.Ip + 2LL > (1LL << 30) / ((long long)std::max(L->cin_g, L->cout) * H * W)) continue;
        } else {
            c.tw = (Wo + k - 1) / k;
            if (k > 1) c.tw = (c.tw + 1) / 2 * 2;
            // whole rows share the zero column between them; narrower ones stage both halo columns
            c.Wp = c.tw >= Wo || S == 2 ? c.tw + 1 : c.tw + 2;
            if (c.Wp < 2 || c.tw > M) continue;
            int th = std::min(Ho, (M - c.tw) / c.Wp + 1);
            if (pool) th = th / 2 * 2;
            if (th < 1) continue;
            c.tiles_y = (Ho + th - 1) / th;
            th = (Ho + c.tiles_y - 1) / c.tiles_y;
            if (pool) th = (th + 1) / 2 * 2;
            c.th = th;
            c.tiles_x = (Wo + c.tw - 1) / c.tw;
            tiles = (long long)N * c.tiles_x * c.tiles_y;
            c.P = S == 1 ? (th + 2) * c.Wp + 2 : (th + 1) * c.Wp + 1;
            c.Ip = 2;   // unused
            if ((long long)std::max(L->cin_g, L->cout) * H * W >= (1LL << 30)) continue;
        }
        if (tiles >= INT_MAX / 4) continue;
        c.tiles = (int)((tiles + 1) / 2);
        if (c.P >= 0xFFFF) continue;
        // the MMAs read 128 MT rows from every tap's offset on, staged or not
        const int rows = S == 1 ? M + 2 * c.Wp + 2 : M + c.Wp + 1;
        c.plane = (unsigned)align_up((size_t)std::max(rows, c.P) * 16, 128);
        c.x_stage = c.plane * 2 * HL * (S == 1 ? 1 : 4);
        // pooling: 32, 16 or 8 filters of a tile's outputs at an even row pitch
        const size_t pool_bytes = pool ? (size_t)32 / c.MT * c.th * ((c.tw + 1) & ~1) * 4 : 0;
        c.tab_off = (unsigned)(kHeadBytes + align_up(pool_bytes, 16));
        const long long units1 = (long long)c.tiles * c.n_fchunks, pairs = sms / 2;
        const double mma = 9.0 * (HL + 1 + ll) * c.MT * std::max(c.NC / 2.0, 32.0 + c.NC / 8.0) + 200.0;
        // a copy brings one, two or four values, where rows are a multiple of them (and x is aligned:
        // tensor_launch)
        for (int way = 1; way <= 8 && W % std::min(way, 4) == 0; way *= 2) {
            const int vec = std::min(way, 4);
            c.box = way == 8;
            // (not for tiles of 128: with this path in it their kernel ran 1 % slower on flat tiles,
            // 256 -> 256 at 56x56 201.6 against 199.9 us)
            if (c.box && (es != 4 || S != 1 || !c.tw || c.MT == 1)) continue;
            c.vec = vec;
            const int np = std::max(1, vec / S);   // positions of a copy
            c.ppr = c.tw ? (c.Wp + 2 * (np - 1)) / np : Wo / np + 1;
            // flat tiles: the copies from that of the first position to that of the last, P - 1 further
            c.n_entries = np == 1 && !c.tw ? c.P
                          : vec == 1       ? c.P
                          : c.tw           ? (S == 1 ? (c.th + 2) * c.ppr + 1 : (c.th + 1) * c.ppr)
                                           : (c.P - 1) / c.Wp * c.ppr + (c.P - 1) % c.Wp / np + 3;
            c.items = vec == 1 ? 2 * c.P * (S == 1 ? 1 : 4) : 2 * S * c.n_entries;
            c.ring_off = (unsigned)align_up(c.tab_off + std::max<size_t>(4 * (size_t)c.P, 8 * (size_t)c.n_entries), 128);
            const int words = es == 4 ? vec : std::max(1, vec / 2);
            c.x_off = c.ring_off + std::max(ring_of(1) * 9, ring_of(words) * (8 * words + 1)) * kProducers * 4;
            if (c.box) {   // two boxes (three: no change); the copies' ring, should x not be aligned, in their place
                c.rw = (3 + c.Wp + 3) & ~3;
                const size_t box = (size_t)64 * (c.th + 2) * c.rw;
                if (c.rw > 256 || c.th + 2 > 256) continue;
                c.rs = kMaxRaw;
                c.x_off = (unsigned)(c.ring_off + std::max(align_up(c.rs * box, 128), (size_t)ring_of(1) * 9 * kProducers * 4));
            }
            if (c.x_off >= kSmemMax) continue;
            const size_t left = kSmemMax - c.x_off;
            // three input stages with two blocks' weights, else two with at least a block's and a row
            c.xs = 0;
            for (int xs = kMaxXStages; xs >= 2 && !c.xs; --xs) {
                const int hs = xs == 3 ? 6 : 4, ls = 2;
                if ((size_t)xs * c.x_stage + (size_t)(hs + ls) * c.w_slot > left) continue;
                c.xs = xs;
                const int slots = (int)std::min<size_t>(10, (left - (size_t)xs * c.x_stage) / c.w_slot);
                c.ls = slots < 7 ? 2 : (slots < 10 ? 3 : 4);
                c.hs = slots - c.ls;   // 4 to kMaxWSlots
            }
            if (!c.xs || (ll && c.ls < 3)) continue;   // a block's three rows of lo weights stay
            c.ll = ll;
            c.h_off = c.x_off + c.xs * c.x_stage;
            c.l_off = c.h_off + c.hs * c.w_slot;
            c.smem = c.l_off + (size_t)c.ls * c.w_slot;
            // clocks of a 16-channel block: its MMAs, and what of its staging does not hide behind
            // them, by rounds of the staging threads; of a unit: its blocks or its stores.  Fitted to
            // 24 layers with every tile, copy and split each can take (849 points, 5 % rms weighted
            // towards the fast ones; the choice is 1.5 % from the best on average).
            static const double kRound[2][3] = {{840.0, 1280.0, 1920.0}, {840.0, 945.0, 1030.0}};   // fp32, fp16
            const int rounds = (c.items + kProducers - 1) / kProducers;
            // boxes: 400 clocks a round of eight channels (250 took layers that ran 1 % slower so)
            const double staging = c.box ? (2.0 * c.P + kProducers - 1) / kProducers * 400.0 : rounds * kRound[es == 2][vec == 1 ? 0 : vec / 2];
            const double stage = (mma + std::max(0.0, staging - 0.64 * mma)) * (c.hs + c.ls < 8 ? 1.09 : 1.0);
            for (int ks = 1; ks <= c.n_cb && (ks == 1 || units1 * ks <= 2 * pairs); ++ks) {
                const int cbs = (c.n_cb + ks - 1) / ks;
                if ((c.n_cb + cbs - 1) / cbs != ks) continue;
                if (ks > 1 && (size_t)ks * out_bytes > ws_bytes) break;
                const long long waves = (units1 * ks + pairs - 1) / pairs;
                const double stores = 128.0 * c.MT * c.NC * (ks > 1 ? 4 : es) / 10.0;
                double t = waves * (std::max(cbs * stage, stores) + 6000.0) * (1.0 + 0.5 / (c.tw ? c.tw : Wo)) + 6000.0;
                if (ks > 1) t += 4000.0 + (double)ks * out_bytes / 2000.0;
                if (!have || t < best) {
                    have = true;
                    best = t;
                    *out = c;
                    out->KS = ks;
                    out->cb_split = cbs;
                    out->units = units1 * ks;
                    out->ws_bytes = ks > 1 ? (size_t)ks * out_bytes : 0;
                    out->clocks = t;
                }
            }
        }
    }
    return have;
}

cudaError_t tensor_launch(const TensorCall& c, const TensorPlan& pl) {
    const pp_layer* L = c.L;
    TcParams p{};
    fill_layer(L, &p);
    p.x = c.x;
    p.y = c.y;
    p.bias = c.bias;
    p.wimg = static_cast<const unsigned char*>(L->tdev);
    p.status = c.status;
    p.wait_limit = c.wait_limit;
    p.no_fill = c.no_fill;
    p.N = c.N;
    p.H = c.H;
    p.W = c.W;
    p.Ho = c.Ho;
    p.Wo = c.Wo;
    p.relu = c.relu;
    // fp32: the inputs' errors (redo_unit) and, of at most 2^15 2^-kexp each, the inputs at weights that
    // err by 2^-36 2^-wexp; fp16: exact inputs of at most 2^16, and sums are rounded to 2^-12
    p.unheld = c.es == 4 ? std::ldexp(L->tc_l1, L->tc_exp - 15) + (float)L->tc_small : std::ldexp((float)L->tc_small, -8);
    p.all_slow = L->tc_small > 0;
    p.pool = c.pool;
    p.KS = pl.KS;
    p.cb_split = pl.cb_split;
    p.ll = pl.ll;
    p.Wp = pl.Wp;
    p.Ip = pl.Ip;
    p.mstep = pl.mstep;
    p.P = pl.P;
    p.vec = pl.vec;
    p.ppr = pl.ppr;
    p.n_entries = pl.n_entries;
    p.items = pl.items;
    p.tw = pl.tw;
    p.th = pl.th;
    p.tiles_x = pl.tiles_x;
    p.tiles_y = pl.tiles_y;
    p.Q = pl.Q;
    p.tiles = pl.tiles;
    p.n_fchunks = pl.n_fchunks;
    p.n_units = (int)pl.units;
    p.d_ip = fast_div((uint32_t)pl.Ip);
    p.d_wp = fast_div((uint32_t)pl.Wp);
    p.d_p = fast_div((uint32_t)(pl.vec > 1 ? pl.n_entries : pl.P));
    p.d_ppr = fast_div((uint32_t)std::max(2, pl.ppr));
    p.ws = static_cast<float*>(c.ws);
    p.ws_stride = (size_t)c.N * L->cout * c.Ho * c.Wo;
    p.xs = pl.xs;
    p.hs = pl.hs;
    p.ls = pl.ls;
    p.plane = pl.plane;
    p.x_stage = pl.x_stage;
    p.w_slot = pl.w_slot;
    p.pool_off = pl.pool_off;
    p.tab_off = pl.tab_off;
    p.ring_off = pl.ring_off;
    p.x_off = pl.x_off;
    p.h_off = pl.h_off;
    p.l_off = pl.l_off;
    p.rw = pl.rw;
    p.rs = pl.rs;
    CUtensorMap tmap;
    std::memset(&tmap, 0, sizeof(tmap));
    p.box = pl.box && reinterpret_cast<uintptr_t>(c.x) % 16 == 0 && encode_box(&tmap, c.x, c.N, p.C, c.H, c.W, pl.rw, pl.th + 2);
    if (pl.box ? !p.box : pl.vec > 1 && reinterpret_cast<uintptr_t>(c.x) % (pl.vec * (size_t)c.es) != 0) {   // single pixels after all
        p.vec = 1;
        p.n_entries = pl.P;
        p.items = 2 * pl.P * (L->stride == 1 ? 1 : 4);
        p.d_p = fast_div((uint32_t)p.P);
    }
    TcKernel k;
    if (L->stride == 1) k = c.es == 4 ? pick<1, float>(pl.MT, pl.smem) : pick<1, __half>(pl.MT, pl.smem);
    else k = c.es == 4 ? pick<2, float>(pl.MT, pl.smem) : pick<2, __half>(pl.MT, pl.smem);
    if (!k) return cudaErrorInvalidValue;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * (unsigned)std::min<long long>(pl.units, c.sms / 2));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = pl.smem;
    cfg.stream = c.st;
    cfg.attrs = attr;
    cfg.numAttrs = c.pdl ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k, p, tmap);
    const cudaError_t l = cudaGetLastError();
    return e != cudaSuccess ? e : l;
}

}  // namespace patconv
