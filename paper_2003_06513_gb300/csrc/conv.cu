// CUDA kernels and launchers of libpatconv (sm_103a): pattern-sparse 3x3 convolution.
//
// Dense layers whose handle is bound for the tensor cores run there (pconv_tc, tensor.cu) wherever
// tensor_wins() below says that it is faster and rounds no more.  All others, main kernel
// pconv_tm<S, T, SORT, SHIFT, SK, DG>:
//   * a lane owns a 4x4 block of output pixels of one image; a warp owns one filter group (8
//     filter slots, the "filter kernel reorder" of §3.4), or DG = 2 groups at stride 2, for its
//     32 blocks; a CTA is 16 / DG warps = WG filter groups x WS spatial warps over one tile;
//   * tiles: rectangles of blocks of one image, several whole images, bands of full block rows
//     of several images side by side, or the linear tile (consecutive blocks across images);
//   * accumulators live in tensor memory: 16 warps x 8 slots x 16 fp32 = all 512 columns; a kept
//     kernel is applied by tcgen05.ld of its slot, 64 FMAs, tcgen05.st;
//   * input channels stream through a 3-stage mbarrier pipeline: one TMA box per stage (the tile
//     of CK channels with its zero halo, padding 1) or, where rows are not 16-byte multiples, a
//     copy shared by all threads; each group's descriptors and kept weights for those channels
//     arrive by cp.async beside it;
//   * per input channel a lane loads its input window into registers once and applies it to every
//     kept kernel of its group(s): the 6-bit (slot, pattern) code of each kept kernel selects one
//     of 8 compile-time pattern bodies (generated inline PTX, gen_dispatch.py) whose four tap
//     operands are fixed registers (the 4 taps of §3.2), so no per-element index is decoded;
//     SHIFT moves the blocks to output columns 4j - 1 or 4j - 2 (aligned window loads), SORT
//     deals a warp's blocks to lanes by shared-memory bank group;
//   * persistent CTAs (one per SM unless the units overflow a CTA's table) walk their units
//     (tile, filter chunk, input-channel split) as one chunk stream;
//   * SK (balanced schedule): one CTA per SM takes an equal range of all units' channel chunks;
//     a unit cut between CTAs is finished by the CTA holding its first chunks, which adds the
//     later CTAs' raw sums (a cooperative launch: every CTA is resident);
//   * epilogue: + bias, ReLU, optionally the 2x2 max-pool, fp32 or fp16 (round to nearest even)
//     stores to the original channel of each slot, or raw partial sums to the split workspace;
//   * every pipeline wait is bounded; a wait that runs out records a bit in the status word and
//     the kernel drains its copies, frees tensor memory and returns.
// Depthwise layers (one pattern per channel, HBM-bound): pconv_dw_stream, per-warp bulk-copy
// pipelines of a persistent CTA per SM (rows, planes and tiles modes) for 16-byte aligned
// tensors; pconv_depthwise / pconv_depthwise_staged for the rest.  Other pattern libraries:
// pconv_generic.  The kernels of this file compute on the CUDA cores' FFMA pipe.
#include <cuda_fp16.h>
#include <cuda.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>
#include <climits>
#include <cmath>
#include <cstdlib>
#include <cstdint>
#include <cstring>
#include <map>
#include <mutex>
#include <numeric>
#include <tuple>
#include <vector>

#include "../../include/patconv.h"
#include "layer.h"
#include "pattern_dispatch.h"
#include "tensor.h"

using namespace patconv;

namespace {

// ------------------------------------------------------------------------------ helpers

// Programmatic dependent launch.  Every kernel of the library lets the next kernel of its stream
// start (launch_dependents: at once, or for the pattern-sparse kernel at its last epilogue) and
// waits for the previous one (wait: that grid has completed and its memory is visible) before it
// reads or writes activations, so one layer's launch and set-up (tensor-memory allocation,
// barriers, tables) overlap the previous layer's tail.  Both are no-ops for a launch without the
// programmatic-serialisation attribute.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ void cp_async4(void* smem, const void* gmem, bool valid) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    const int n = valid ? 4 : 0;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(s), "l"(gmem), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}

template <typename T>
__device__ __forceinline__ float to_f32(T v);
template <>
__device__ __forceinline__ float to_f32<float>(float v) { return v; }
template <>
__device__ __forceinline__ float to_f32<__half>(__half v) { return __half2float(v); }

template <typename T>
__device__ __forceinline__ T from_f32(float v);
template <>
__device__ __forceinline__ float from_f32<float>(float v) { return v; }
template <>
__device__ __forceinline__ __half from_f32<__half>(float v) { return __float2half_rn(v); }

// ------------------------------------------------------------------------------ main kernel

constexpr int kCompute = 16;                       // warps per CTA (filter groups x spatial)
constexpr int kThreadsTM = kCompute * 32;
constexpr int kStages = 3;                         // input-channel pipeline depth
constexpr int kMaxChunks = 256;                    // input-channel stages per CTA
constexpr long long kTimeoutCycles = 2000000000LL; // about one second of SM clock
constexpr uint32_t kTmemCols = 512;                // 16 warps x 8 slots x 16 accumulators
constexpr int kMaxUnitsPerCta = 64;                // units one persistent CTA holds in its table

// Device status word: a wait that ran out of time records its code here and the kernel returns
// early instead of hanging (read back by pp_device_status).
__device__ unsigned int g_pp_status;
enum : unsigned { kStatusFullTimeout = 1u, kStatusEmptyTimeout = 2u, kStatusDrainTimeout = 4u,
                  kStatusPartTimeout = 8u };
constexpr int kSlotFloats = kCompute * 8 * 16 * 32;   // a CTA's accumulators: 16 warps x 8 slots x 16 x 32 lanes

struct TmParams {
    const void* x;
    void* y;
    const float* bias;
    const uint32_t* perm;
    const uint64_t* desc;
    const uint32_t* kofs;
    const float4* vals;
    unsigned* status;
    long long wait_limit;              // SM cycles a pipeline (full / empty) wait may take
    int no_fill;                       // test only: issue no stage fills (every first wait runs out)
    int N, C, H, W, Cout, Ho, Wo, G, relu;
    int WG, WS;                        // filter groups x spatial warps per CTA (WG * WS = 16)
    int BY, BX, NB;                    // spatial tile: BY x BX blocks (4x4 outputs) of NB images
    int tiles_x, tiles_y, tiles_n, n_fchunks;
    int linear;                        // linear tiles: lanes take consecutive blocks across images
    int n_units;                       // units: tiles x filter chunks x input-channel splits
    int CK, n_chunks, maxk;            // channels per stage, stages per CTA (max), max kept per group-stage
    int KS, c_split;                   // input-channel splits; channels per split (multiple of CK)
    float* ws;                         // KS > 1: fp32 partial sums [KS][N][Cout][Ho][Wo]
    size_t ws_stride;                  // elements per split
    int streamk;                       // balanced schedule: CTA b takes chunks [T b / P, T (b + 1) / P)
    long long sk_total;                // T: chunks of all units (every unit has n_chunks of them)
    float* sk_slots;                   // a CTA's part: its raw accumulators (kSlotFloats per CTA)
    unsigned* sk_flags;                // [CTA][warp]: 1 once that warp's part slot is written
    int IH, BWb;                       // staged rows / row width (elements) per (image, channel)
    int ixa;                           // stage origin column: a multiple of ixa (16 bytes of input)
    int use_tma, vec_store, vec_pair;  // float4 / 8-byte-group stores; pair stores (SHIFT)
    int pool, vec_pool;                // fused 2x2/2 max-pool of the output; pair stores of it
    unsigned tma_bytes;                // bytes one TMA box delivers
    unsigned kb_off, stage_off, stage_bytes, desc_off, vals_off;   // shared-memory layout
};

__device__ __forceinline__ uint32_t smem_u32(const void* ptr) {
    return (uint32_t)__cvta_generic_to_shared(ptr);
}
__device__ __forceinline__ void mbar_init(uint32_t a, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(a), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t a, uint32_t tx) {
    asm volatile("mbarrier.arrive.expect_tx.release.cta.shared::cta.b64 _, [%0], %1;" ::"r"(a), "r"(tx) : "memory");
}
// arrives on the barrier once every cp.async this thread issued so far has landed
__device__ __forceinline__ void cp_async_arrive(uint32_t a) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(a) : "memory");
}
// Bounded wait for the completion of the phase with the given parity.
__device__ __forceinline__ bool mbar_wait(uint32_t a, uint32_t parity, unsigned* status, unsigned code,
                                          long long limit = kTimeoutCycles) {
    const long long t0 = clock64();
    while (true) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred P;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, P;\n\t}"
            : "=r"(done) : "r"(a), "r"(parity) : "memory");
        if (done) return true;
        if (clock64() - t0 > limit) {
            atomicOr(status, code);
            return false;
        }
    }
}
__device__ __forceinline__ void mbar_arrive(uint32_t a) {
    asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(a) : "memory");
}
// mbar_wait by a whole warp with one outcome for all its lanes
__device__ __forceinline__ bool mbar_wait_warp(uint32_t a, uint32_t parity, unsigned* status, unsigned code,
                                               long long limit) {
    return __all_sync(0xffffffffu, mbar_wait(a, parity, status, code, limit));
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, int x, int y, int c, int n,
                                            uint32_t mbar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(c), "r"(n), "r"(mbar)
        : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t ta, float (&a)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(ta) : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) a[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_zero16(uint32_t ta) {
    const uint32_t z = 0;
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};\n\t"
        "tcgen05.wait::st.sync.aligned;" ::"r"(ta), "r"(z) : "memory");
}

// Fallback input staging when no TMA descriptor applies (row pitch not a multiple of 16 bytes,
// the stage holds the input's own type): thread tid copies elements tid, tid + 512, ... of the
// in-image part of the tile; everything else in the stage keeps the zero written at kernel start.
template <typename TIn, int NT = kThreadsTM>
__device__ __forceinline__ void stage_input_share(const TmParams& p, TIn* s_in, int c0, int ckv, int n0,
                                                  int iy0, int ix0, int tid) {
    const TIn* x = static_cast<const TIn*>(p.x);
    const int ry0 = max(0, iy0), ry1 = min(p.H, iy0 + p.IH);
    const int rx0 = max(0, ix0), rx1 = min(p.W, ix0 + p.BWb);
    const int nr = ry1 - ry0, nc = rx1 - rx0;
    if (nr <= 0 || nc <= 0) return;
    const int nimg = min(p.NB, p.N - n0);
    // rows whose global start and length are even go as pairs (8 bytes of fp32, 4 bytes of fp16,
    // copied asynchronously); the staged column of image column ix is ix - ix0 with ix0 a
    // multiple of 16 bytes, so the shared side is aligned too
    const bool pairs = (p.W % 2 == 0) && (rx0 % 2 == 0) && (nc % 2 == 0) &&
                       reinterpret_cast<uintptr_t>(x) % (2 * sizeof(TIn)) == 0;
    const int units = pairs ? nc / 2 : nc;                  // copy units per row
    // element e = ((img * ckv + cl) * nr + r) * units + u as digits (img, cl, r, u); adding the
    // thread count digit by digit needs at most one carry per digit
    int q = tid / units;
    int u = tid - q * units;
    int r = q % nr;
    q /= nr;
    int cl = q % ckv, img = q / ckv;
    q = NT / units;
    const int su = NT - q * units, sr = q % nr;
    q /= nr;
    const int scl = q % ckv, simg = q / ckv;
    const size_t HW = (size_t)p.H * p.W;
    while (img < nimg) {
        const int iy = ry0 + r, ix = rx0 + (pairs ? 2 * u : u);
        const TIn* src = x + ((size_t)(n0 + img) * p.C + c0 + cl) * HW + (size_t)iy * p.W + ix;
        TIn* dst = s_in + ((img * p.CK + cl) * p.IH + (iy - iy0)) * p.BWb + (ix - ix0);
        if constexpr (sizeof(TIn) == 4) {
            if (pairs) cp_async8(dst, src);
            else cp_async4(dst, src, true);
        } else {
            if (pairs) cp_async4(dst, src, true);
            else *dst = *src;
        }
        u += su;
        if (u >= units) { u -= units; ++r; }
        r += sr;
        if (r >= nr) { r -= nr; ++cl; }
        cl += scl;
        if (cl >= ckv) { cl -= ckv; ++img; }
        img += simg;
    }
}

// One unit of work of a CTA: a spatial tile, a filter chunk (WG groups) and an input-channel
// split.  Units are numbered with the filter chunk fastest, so CTAs working at the same time
// share input tiles in L2.  With the balanced (stream-K) schedule a CTA may hold only a segment
// of a unit's channel chunks: c_lo and nck then describe the segment, and role says whether it
// is the whole unit, its head (the first chunks: this CTA adds the other segments' partial sums
// and writes the result) or a later part (raw partial sums to the CTA's workspace slot); a head's
// parts are the next CTAs up to pb1 (exclusive).  role and pb1 share one word: role | pb1 << 2.
enum : int { kRoleFull = 0, kRoleHead = 1, kRolePart = 2 };
struct __align__(16) Unit {
    int ks, tn, n0, oy0, ox0, iy0, ix0, g0, c_lo, c_hi, nck, sk;
};

template <int S>
__device__ __forceinline__ Unit unit_of(const TmParams& p, int u) {
    Unit U;
    const int fchunk = u % p.n_fchunks;
    int t = u / p.n_fchunks;
    const int tx = t % p.tiles_x;
    t /= p.tiles_x;
    const int ty = t % p.tiles_y;
    t /= p.tiles_y;
    U.tn = t % p.tiles_n;
    U.ks = t / p.tiles_n;
    U.c_lo = U.ks * p.c_split;
    U.c_hi = min(p.C, U.c_lo + p.c_split);
    U.nck = (U.c_hi - U.c_lo + p.CK - 1) / p.CK;
    U.sk = kRoleFull;
    // linear tiles: tile tn holds blocks [tn * lanes, (tn + 1) * lanes) of the (image, block row,
    // block column) sequence and stages the whole images from n0 on
    U.n0 = p.linear ? (int)(((long long)U.tn * 32 * p.WS) / (p.BY * p.BX)) : U.tn * p.NB;
    U.oy0 = ty * p.BY * 4;
    U.ox0 = tx * p.BX * 4;
    U.iy0 = U.oy0 * S - 1;          // stage origin: 1 halo row, 16-byte aligned column
    // stage origin: the 16-byte boundary at or left of the tile's first input column ox0 * S - 1
    const int m = (U.ox0 * S) % p.ixa;
    U.ix0 = U.ox0 * S - (m == 0 ? p.ixa : m);
    U.g0 = fchunk * p.WG;
    return U;
}

// This thread's share of filling pipeline stage q % kStages with input channel chunk k of unit U
// (non-blocking): warp 0 lane 0 issues the input tile's TMA, or every thread copies its share of
// the tile; the warps of filter group wg (DG groups per warp: wg DG .. wg DG + DG - 1) copy those
// groups' descriptors and kept weights vals[beg[d], end[d]).  The stage's full barrier completes
// when all threads of the CTA (kThreadsTM / DG) have arrived and every byte has landed.
template <typename TIn, int DG = 1>
__device__ __forceinline__ void fill_share(const TmParams& p, const CUtensorMap* tmap, unsigned char* smem,
                                           uint32_t full0, int q, const Unit& U, int k, const uint32_t (&beg)[DG],
                                           const uint32_t (&end)[DG], int warp, int lane) {
    const int s = q % kStages;
    unsigned char* st = smem + p.stage_off + (size_t)s * p.stage_bytes;
    const uint32_t fb = full0 + 8 * s;
    const int c0 = U.c_lo + k * p.CK, ckv = min(p.CK, U.c_hi - c0);
    if (warp == 0 && lane == 0) {
        mbar_arrive_expect_tx(fb, p.use_tma ? p.tma_bytes : 0u);
        if (p.use_tma) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            tma_load_4d(smem_u32(st), tmap, U.ix0, U.iy0, c0, U.n0, fb);
        }
    }
    if (!p.use_tma)
        stage_input_share<TIn, kThreadsTM / DG>(p, reinterpret_cast<TIn*>(st), c0, ckv, U.n0, U.iy0, U.ix0,
                                                warp * 32 + lane);
    const int wg = warp / p.WS, ws = warp - wg * p.WS;
#pragma unroll
    for (int d = 0; d < DG; ++d) {
        const int gl = wg * DG + d, g = U.g0 + gl;   // the group's index within the unit, and in the layer
        if (g < p.G) {
            uint64_t* sd = reinterpret_cast<uint64_t*>(st + p.desc_off) + gl * p.CK;
            for (int cl = ws * 32 + lane; cl < ckv; cl += p.WS * 32)
                cp_async8(sd + cl, p.desc + (size_t)g * p.C + c0 + cl);
            float4* sv = reinterpret_cast<float4*>(st + p.vals_off) + gl * p.maxk;
            for (uint32_t i = beg[d] + ws * 32 + lane; i < end[d]; i += p.WS * 32) cp_async16(sv + (i - beg[d]), p.vals + i);
        }
    }
    __threadfence_block();   // orders the fp16 path's plain shared stores before the arrival
    cp_async_arrive(fb);
}

__device__ __forceinline__ void tmem_st16(uint32_t ta, const float (&a)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};\n\t"
        "tcgen05.wait::st.sync.aligned;" ::"r"(ta),
        "r"(__float_as_uint(a[0])), "r"(__float_as_uint(a[1])), "r"(__float_as_uint(a[2])), "r"(__float_as_uint(a[3])),
        "r"(__float_as_uint(a[4])), "r"(__float_as_uint(a[5])), "r"(__float_as_uint(a[6])), "r"(__float_as_uint(a[7])),
        "r"(__float_as_uint(a[8])), "r"(__float_as_uint(a[9])), "r"(__float_as_uint(a[10])), "r"(__float_as_uint(a[11])),
        "r"(__float_as_uint(a[12])), "r"(__float_as_uint(a[13])), "r"(__float_as_uint(a[14])), "r"(__float_as_uint(a[15]))
        : "memory");
}

// Balanced schedule, a part segment's end: the warp's raw accumulators (8 slots x 16 per lane) go
// to this CTA's workspace slot ([warp][slot][16][lane]: coalesced), tensor memory is zeroed
// behind, then the warp's flag is released once every lane's stores are visible.
template <int DG>
__device__ __noinline__ void sk_store_part(const TmParams& p, uint32_t tw, int warp, int lane) {
    float* sl = p.sk_slots + (size_t)blockIdx.x * kSlotFloats + (size_t)warp * kF * DG * 16 * 32 + lane;
#pragma unroll 1
    for (int f = 0; f < kF * DG; ++f) {
        float a[16];
        __syncwarp();
        tmem_ld16(tw + 16u * f, a);
        tmem_zero16(tw + 16u * f);
#pragma unroll
        for (int i = 0; i < 16; ++i) sl[(f * 16 + i) * 32] = a[i];
    }
    __threadfence();
    __syncwarp();
    if (lane == 0) {
        unsigned* fl = p.sk_flags + (size_t)blockIdx.x * kCompute + warp;
        asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(fl), "r"(1u) : "memory");
    }
}

// Balanced schedule, a head segment's end: wait (bounded) for the flags of the unit's parts, held
// by CTAs [pb0, pb1), then add their sums to the warp's accumulators in chunk order (a fixed
// summation order).  A flag that never comes records a status bit and the parts are left out.
template <int DG>
__device__ __noinline__ void sk_add_parts(const TmParams& p, uint32_t tw, int warp, int lane, int pb0, int pb1) {
    bool ok = true;
    for (int b = pb0; b < pb1; ++b) {
        unsigned ready = 0;
        if (lane == 0) {
            const unsigned* fl = p.sk_flags + (size_t)b * kCompute + warp;
            const long long t0 = clock64();
            while (true) {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(ready) : "l"(fl) : "memory");
                if (ready) break;
                if (clock64() - t0 > kTimeoutCycles) {
                    atomicOr(p.status, kStatusPartTimeout);
                    break;
                }
            }
        }
        ok = ok && __shfl_sync(0xffffffffu, ready, 0) != 0;
    }
    __syncwarp();   // the other lanes read the slots after lane 0's acquire
    if (!ok) return;
#pragma unroll 1
    for (int f = 0; f < kF * DG; ++f) {
        float a[16];
        __syncwarp();
        tmem_ld16(tw + 16u * f, a);
        for (int b = pb0; b < pb1; ++b) {
            const float* sl = p.sk_slots + (size_t)b * kSlotFloats + (size_t)warp * kF * DG * 16 * 32 + lane + f * 16 * 32;
#pragma unroll
            for (int i = 0; i < 16; ++i) a[i] += __ldcg(sl + 32 * i);
        }
        tmem_st16(tw + 16u * f, a);
    }
}

// SORT (stride 1, fp32 only): each warp's blocks are dealt to its lanes by bank group.
// SHIFT (stride 1): block j of a tile row covers output columns ox0 + 4j - SHIFT .. ox0 + 4j + 3
// - SHIFT.  SHIFT 1: a lane's window column 0 sits at 2 (mod 4) in the stage and each window row
// is one 8-byte and one 16-byte shared load (SHIFT 0: 4-byte, 16-byte, 4-byte, the 4-byte ones
// bank conflicted); its blocks split 2x2 pooling windows, so the fused pool never uses it.
// SHIFT 2 (fp32): column 0 at 1 (mod 4), each row two 16-byte loads, and blocks start at even
// columns, so the fused pool's windows stay inside a block.
template <int S, typename TIn, bool SORT = false, int SHIFT = 0, bool SK = false, int DG = 1>
__global__ void __launch_bounds__(kThreadsTM / DG, 1)
    pconv_tm(const TmParams p, const __grid_constant__ CUtensorMap tmap) {
    constexpr int RY = 4, RX = 4;
    constexpr int NT = kThreadsTM / DG, NWP = kCompute / DG;   // threads, warps of the CTA
    static_assert(DG == 1 || S == 2, "two filter groups per warp: the stride-2 kernel");
    static_assert(!SORT || (sizeof(TIn) == 4 && (S == 1 || DG == 2)), "lanes by bank group: fp32, stride 2 with two groups");
    static_assert(!SHIFT || S == 1, "shifted blocks are a stride-1 layout");
    static_assert(SHIFT != 2 || sizeof(TIn) == 4, "blocks at 4j - 2 are an fp32 layout");
    extern __shared__ __align__(128) unsigned char smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // header: full[kStages] (stage filled), empty[kStages] (stage read by all 16 warps), the
    // tensor-memory base and the number of chunks whose fill warp 0 has issued
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem);
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(smem + 16 * kStages);
    uint32_t* s_issued = s_tmem + 1;
    const uint32_t full0 = smem_u32(bar), empty0 = full0 + 8 * kStages;

    // this CTA's units: blockIdx.x, blockIdx.x + gridDim.x, ... (one per CTA unless the launch is
    // persistent), or with the balanced schedule the units its chunk range [lo, hi) touches;
    // their chunks form one stream q = 0 .. Q-1 through the three stages, so the next unit's
    // first stages fill while the current one finishes
    Unit* s_units = reinterpret_cast<Unit*>(smem + p.kb_off);   // at most kMaxUnitsPerCta
    int n_my;
    if constexpr (SK) {
        const long long P = gridDim.x, T = p.sk_total, nck = p.n_chunks;
        const long long lo = T * blockIdx.x / P, hi = T * (blockIdx.x + 1) / P;
        const long long u0 = lo / nck;
        n_my = hi > lo ? (int)((hi - 1) / nck - u0 + 1) : 0;
        if ((int)threadIdx.x < n_my) {
            const long long u = u0 + threadIdx.x;
            Unit U = unit_of<S>(p, (int)u);
            const int k0 = (int)(max(lo, u * nck) - u * nck), k1 = (int)(min(hi, (u + 1) * nck) - u * nck);
            U.c_lo += k0 * p.CK;
            U.nck = k1 - k0;
            U.sk = k0 > 0 ? kRolePart : (k1 < nck ? kRoleHead : kRoleFull);
            if (U.sk == kRoleHead) {   // the CTAs holding chunks k1 .. nck-1: the next ones
                const long long last = (u + 1) * nck - 1;   // CTA of chunk c: ceil((c+1) P / T) - 1
                U.sk |= (int)(((last + 1) * P + T - 1) / T) << 2;
            }
            s_units[threadIdx.x] = U;
        }
    } else {
        n_my = p.n_units > (int)blockIdx.x ? (p.n_units - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
        if ((int)threadIdx.x < n_my) s_units[threadIdx.x] = unit_of<S>(p, blockIdx.x + threadIdx.x * gridDim.x);
    }

    if (!p.use_tma) {   // the fallback writes only in-image elements: zero all stages once
        float* z = reinterpret_cast<float*>(smem + p.stage_off);
        const int nf = (int)(kStages * p.stage_bytes / 4);
        for (int i = threadIdx.x; i < nf; i += NT) z[i] = 0.0f;
    }
    if (warp == 0) {
        if (lane == 0) {
            for (int s = 0; s < kStages; ++s) {
                mbar_init(full0 + 8 * s, NT + 1);   // a cp.async arrival per thread + the expect-tx one
                mbar_init(empty0 + 8 * s, NWP);     // one arrival per warp
            }
            *s_issued = 0;
        }
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(s_tmem)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tbase = *s_tmem;
    int Q = 0;
    for (int i = 0; i < n_my; ++i) Q += s_units[i].nck;
    pdl_wait();   // the previous kernel's output (this input) is complete from here on

    const int wg = warp / p.WS, ws = warp - (warp / p.WS) * p.WS;
    // fill cursor: unit fi (of this CTA), its chunk fk, and the warp's group's weight range for
    // that chunk (loaded one fill ahead, so its latency hides behind a chunk of compute)
    // (units are read from the table where needed: few registers live across the loop)
    int fi = 0, fk = 0;
    uint32_t fbeg[DG], fend[DG];
    auto fetch_range = [&]() {
#pragma unroll
        for (int d = 0; d < DG; ++d) {
            fbeg[d] = fend[d] = 0;
            if (fi < n_my) {
                const Unit FU = s_units[fi];
                const int g = FU.g0 + wg * DG + d;
                if (g < p.G) {
                    const int c0 = FU.c_lo + fk * p.CK;
                    const size_t b = (size_t)g * p.C;
                    fbeg[d] = p.kofs[b + c0];
                    fend[d] = p.kofs[b + min(c0 + p.CK, FU.c_hi)];
                }
            }
        }
    };
    auto advance_fill = [&]() {
        if (++fk == s_units[fi].nck) {
            fk = 0;
            ++fi;
        }
        fetch_range();
    };
    auto fill = [&](int q) {
        fill_share<TIn, DG>(p, &tmap, smem, full0, q, s_units[fi], fk, fbeg, fend, warp, lane);
        advance_fill();
    };
    fetch_range();
    {   // prologue: every thread's share of the first kStages chunks
        const int first = p.no_fill ? 0 : min(kStages, Q);
        for (int q = 0; q < first; ++q) fill(q);
        if (threadIdx.x == 0) *s_issued = first;
    }

    // tensor memory: warp w owns lanes 32*(w%4).. and columns 128*DG*(w/4) + 16*slot .. (DG*8 slots)
    const uint32_t tw = tbase + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(128 * DG * (warp >> 2));
#pragma unroll
    for (int f = 0; f < kF * DG; ++f) tmem_zero16(tw + 16u * f);

    const int blk = ws * 32 + lane;
    const int lanes_t = 32 * p.WS, bpi = p.BY * p.BX;
    const int plane = p.IH * p.BWb;
    // compute cursor: unit ci, its chunk ck, and this lane's block of the unit's tile
    int ci = 0, ck = 0;
    int img = 0, by = 0, bx = 0, in_off = 3;
    uint32_t edge = 1;
    uint32_t srcl = 0;   // stride 2 with blocks dealt by bank group: the lane holding the left block
    bool active = false;
    auto place_lane = [&]() {
        const Unit CU = s_units[ci];
        // block t (0 .. 32 * WS - 1) of the unit's tile: image, block row and column, and where
        // the lane's window column 0 (input column ox0 * S - 1 of the block, SHIFT less) sits in
        // the stage: d = 3 into the row for fp32 stages, 3 or 7 for fp16 ones (their origin is 16
        // bytes); with SHIFT 1, 2 or 6; with SHIFT 2 the window address is that of column -1, at
        // d = 0
        auto locate = [&](int t) {
            int rem;
            if (p.linear) {
                const long long b = (long long)CU.tn * lanes_t + t;
                const int ng = (int)(b / bpi);
                img = ng - CU.n0;
                rem = (int)(b - (long long)ng * bpi);
                active = ng < p.N && img < p.NB;
            } else {
                img = t / bpi;
                rem = t - img * bpi;
                active = img < p.NB;
            }
            by = rem / p.BX;
            bx = rem - by * p.BX;
            const int d = CU.ox0 * S - 1 - CU.ix0 - SHIFT - (SHIFT == 2 ? 1 : 0);
            in_off = active ? img * p.CK * plane + by * RY * S * p.BWb + bx * RX * S + d : d;
        };
        locate(blk);
        int src = lane;
        if constexpr (SORT) {
            // The warp's 32 blocks are dealt to its lanes so that each 8-lane phase of the
            // 16-byte window loads (window columns 1-4 at in_off + 1, 2-5 at in_off + 2 with
            // SHIFT 1, -1..2 and 3..6 at in_off and in_off + 4 with SHIFT 2; at stride 2 columns
            // 1-4 at in_off + 1 and 5-8 one group further) meets distinct bank groups where the
            // blocks allow it: blocks are ordered by (rank among the blocks of their bank group,
            // bank group) and lane i takes the i-th.  Rows of 7 or 14 blocks (stride 1), or the
            // blocks of one row 32 bytes apart (stride 2: every other group), otherwise put two
            // blocks of a phase on one bank group.  Idle lanes go last.  The planner picks this
            // instance where it lowers the wavefronts (window_wavefronts).
            const int grp = active ? ((in_off + (SHIFT == 0 ? 1 : SHIFT == 1 ? 2 : 0)) >> 2) & 7 : 8;
            const unsigned same = __match_any_sync(0xffffffffu, grp);
            const int key = active ? 16 * __popc(same & ((1u << lane) - 1u)) + grp : 1024 + lane;   // distinct
            int pos = 0;
            src = 0;
            for (int i = 0; i < 32; ++i) pos += __shfl_sync(0xffffffffu, key, i) < key ? 1 : 0;
            for (int i = 0; i < 32; ++i) src = __shfl_sync(0xffffffffu, pos, i) == lane ? i : src;
            locate(ws * 32 + src);
            if constexpr (S == 2) {   // the lane holding the block to the left (raster src - 1)
                srcl = lane;
                for (int i = 0; i < 32; ++i) srcl = __shfl_sync(0xffffffffu, src, i) == src - 1 ? i : srcl;
            }
        }
        // lanes whose left block is not held by the lane they take window column 0 from (stride 2
        // takes it by shuffle): the first block of a row or of the warp's range
        edge = (bx == 0 || src == 0) ? 1u : 0u;
    };
    place_lane();

    using TOut = TIn;
    TOut* y = static_cast<TOut*>(p.y);
    // accumulators of unit U out of tensor memory (zeroed behind) + bias, ReLU, optional pool, to
    // the original channel; with a split, raw partial sums to the workspace
    auto epilogue = [&](const Unit& U) {
        const int n = U.n0 + img;
        const int oyb = U.oy0 + by * RY, oxb = U.ox0 + bx * RX - SHIFT;
        // balanced schedule: a part only publishes its raw sums; a head first adds its unit's
        // parts into tensor memory (out of line: the common path keeps its registers)
        if constexpr (SK) {
            if ((U.sk & 3) == kRolePart) {
                sk_store_part<DG>(p, tw, warp, lane);
                return;
            }
            if ((U.sk & 3) == kRoleHead) sk_add_parts<DG>(p, tw, warp, lane, blockIdx.x + 1, U.sk >> 2);
        }
#pragma unroll 1
        for (int f = 0; f < kF * DG; ++f) {
            float a[16];
            __syncwarp();
            tmem_ld16(tw + 16u * f, a);
            tmem_zero16(tw + 16u * f);
            const int g = U.g0 + wg * DG + f / kF;
            if (g >= p.G || !active || n >= p.N) continue;
            const uint32_t co = p.perm[g * kF + f % kF];
            if (co == kPadSlot) continue;
            if (p.KS > 1) {   // raw partial sums of this split; bias, ReLU and rounding come later
                float* wc = p.ws + (size_t)U.ks * p.ws_stride + ((size_t)n * p.Cout + co) * p.Ho * p.Wo;
#pragma unroll
                for (int r = 0; r < RY; ++r) {
                    const int oy = oyb + r;
                    if (oy >= p.Ho) break;
                    float* wr = wc + (size_t)oy * p.Wo;
                    if constexpr (SHIFT == 1) {   // columns oxb (3 mod 4), oxb+1..oxb+2 (a pair), oxb+3
                        if (oxb >= 0 && oxb < p.Wo) wr[oxb] = a[r * RX];
                        if ((p.Wo % 2) == 0 && oxb + 3 <= p.Wo) {
                            *reinterpret_cast<float2*>(wr + oxb + 1) = make_float2(a[r * RX + 1], a[r * RX + 2]);
                        } else {
                            if (oxb + 1 < p.Wo) wr[oxb + 1] = a[r * RX + 1];
                            if (oxb + 2 < p.Wo) wr[oxb + 2] = a[r * RX + 2];
                        }
                        if (oxb + 3 < p.Wo) wr[oxb + 3] = a[r * RX + 3];
                    } else if constexpr (SHIFT == 2) {   // pairs at oxb (2 mod 4) and oxb+2; oxb >= -2
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int c = oxb + 2 * h;
                            if (c < 0) continue;
                            if ((p.Wo % 2) == 0 && c + 2 <= p.Wo) {
                                *reinterpret_cast<float2*>(wr + c) = make_float2(a[r * RX + 2 * h], a[r * RX + 2 * h + 1]);
                            } else {
                                if (c < p.Wo) wr[c] = a[r * RX + 2 * h];
                                if (c + 1 < p.Wo) wr[c + 1] = a[r * RX + 2 * h + 1];
                            }
                        }
                    } else if ((p.Wo % 4) == 0 && oxb + RX <= p.Wo) {
                        *reinterpret_cast<float4*>(wr + oxb) =
                            make_float4(a[r * RX], a[r * RX + 1], a[r * RX + 2], a[r * RX + 3]);
                    } else {
#pragma unroll
                        for (int c = 0; c < RX; ++c)
                            if (oxb + c < p.Wo) wr[oxb + c] = a[r * RX + c];
                    }
                }
                continue;
            }
            const float b = p.bias ? p.bias[co] : 0.0f;
            if (p.pool) {   // 2x2/2 max-pool inside the lane's 4x4 block (block origins are even;
                            // with SHIFT 2 the first pooled column is -1 in a row's first block)
                const int Hp = p.Ho >> 1, Wp = p.Wo >> 1;
                const int py0 = oyb >> 1, px0 = oxb >> 1;
                TOut* yc = y + ((size_t)n * p.Cout + co) * Hp * Wp;
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const int py = py0 + r;
                    if (py >= Hp) break;
                    float v[2];
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const float m = fmaxf(fmaxf(a[2 * r * RX + 2 * c], a[2 * r * RX + 2 * c + 1]),
                                              fmaxf(a[(2 * r + 1) * RX + 2 * c], a[(2 * r + 1) * RX + 2 * c + 1]));
                        const float q = m + b;   // max(a) + b == max(a + b) in fp32: rounding is monotonic
                        v[c] = p.relu ? fmaxf(q, 0.0f) : q;
                    }
                    TOut* yr = yc + (size_t)py * Wp + px0;
                    if constexpr (SHIFT == 2) {   // px0 odd: no pair store
#pragma unroll
                        for (int c = 0; c < 2; ++c)
                            if (px0 + c >= 0 && px0 + c < Wp) yr[c] = from_f32<TOut>(v[c]);
                    } else if (p.vec_pool && px0 + 2 <= Wp) {
                        if constexpr (sizeof(TOut) == 4) {
                            *reinterpret_cast<float2*>(yr) = make_float2(v[0], v[1]);
                        } else {
                            *reinterpret_cast<__half2*>(yr) = __floats2half2_rn(v[0], v[1]);
                        }
                    } else {
#pragma unroll
                        for (int c = 0; c < 2; ++c)
                            if (px0 + c < Wp) yr[c] = from_f32<TOut>(v[c]);
                    }
                }
                continue;
            }
            TOut* yc = y + ((size_t)n * p.Cout + co) * p.Ho * p.Wo;
#pragma unroll
            for (int r = 0; r < RY; ++r) {
                const int oy = oyb + r;
                if (oy >= p.Ho) break;
                TOut* yr = yc + (size_t)oy * p.Wo;
                float v[RX];
#pragma unroll
                for (int c = 0; c < RX; ++c) {
                    const float q = a[r * RX + c] + b;
                    v[c] = p.relu ? fmaxf(q, 0.0f) : q;
                }
                if constexpr (SHIFT == 1) {   // columns oxb (3 mod 4), oxb+1..oxb+2 (a pair), oxb+3
                    if (oxb >= 0 && oxb < p.Wo) yr[oxb] = from_f32<TOut>(v[0]);
                    if (p.vec_pair && oxb + 3 <= p.Wo) {
                        if constexpr (sizeof(TOut) == 4) {
                            *reinterpret_cast<float2*>(yr + oxb + 1) = make_float2(v[1], v[2]);
                        } else {
                            *reinterpret_cast<__half2*>(yr + oxb + 1) = __floats2half2_rn(v[1], v[2]);
                        }
                    } else {
                        if (oxb + 1 < p.Wo) yr[oxb + 1] = from_f32<TOut>(v[1]);
                        if (oxb + 2 < p.Wo) yr[oxb + 2] = from_f32<TOut>(v[2]);
                    }
                    if (oxb + 3 < p.Wo) yr[oxb + 3] = from_f32<TOut>(v[3]);
                } else if constexpr (SHIFT == 2) {   // pairs at oxb (2 mod 4) and oxb+2; oxb >= -2
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int c = oxb + 2 * h;
                        if (c < 0) continue;
                        if (p.vec_pair && c + 2 <= p.Wo) {
                            *reinterpret_cast<float2*>(yr + c) = make_float2(v[2 * h], v[2 * h + 1]);
                        } else {
                            if (c < p.Wo) yr[c] = from_f32<TOut>(v[2 * h]);
                            if (c + 1 < p.Wo) yr[c + 1] = from_f32<TOut>(v[2 * h + 1]);
                        }
                    }
                } else if (p.vec_store && oxb + RX <= p.Wo) {
                    if constexpr (sizeof(TOut) == 4) {
                        *reinterpret_cast<float4*>(yr + oxb) = make_float4(v[0], v[1], v[2], v[3]);
                    } else {
                        __half2 h0 = __floats2half2_rn(v[0], v[1]);
                        __half2 h1 = __floats2half2_rn(v[2], v[3]);
                        uint2 u;
                        u.x = *reinterpret_cast<unsigned*>(&h0);
                        u.y = *reinterpret_cast<unsigned*>(&h1);
                        *reinterpret_cast<uint2*>(yr + oxb) = u;
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < RX; ++c)
                        if (oxb + c < p.Wo) yr[oxb + c] = from_f32<TOut>(v[c]);
                }
            }
        }
    };

    for (int q = 0; q < Q; ++q) {
        const int s = q % kStages;
        if (!mbar_wait_warp(full0 + 8 * s, (q / kStages) & 1, p.status, kStatusFullTimeout, p.wait_limit)) break;
        const Unit CU = s_units[ci];
        if (CU.g0 + wg * DG < p.G) {
            const unsigned char* st = smem + p.stage_off + (size_t)s * p.stage_bytes;
            const uint32_t win_addr = smem_u32(reinterpret_cast<const TIn*>(st) + in_off);
            const uint32_t desc_addr = smem_u32(reinterpret_cast<const uint64_t*>(st + p.desc_off) + wg * DG * p.CK);
            const uint32_t vals_addr = smem_u32(reinterpret_cast<const float4*>(st + p.vals_off) + wg * DG * p.maxk);
            const int ckv = min(p.CK, CU.c_hi - CU.c_lo - ck * p.CK);
            constexpr int es = (int)sizeof(TIn);
            if constexpr (DG == 2) {   // the warp's second group: descriptors and weights one group up
                const uint32_t desc_b = desc_addr + 8u * p.CK, vals_b = vals_addr + 16u * p.maxk;
                const uint32_t valid_b = CU.g0 + wg * DG + 1 < p.G ? 1u : 0u;
                if constexpr (es == 4) {
                    if constexpr (SORT) {
                        PP_STAGE_KERNELS_S2_G2D(ckv, desc_addr, vals_addr, win_addr, es * p.BWb, es * plane, tw,
                                                edge, desc_b, vals_b, valid_b, srcl);
                    } else {
                        PP_STAGE_KERNELS_S2_G2(ckv, desc_addr, vals_addr, win_addr, es * p.BWb, es * plane, tw, edge,
                                               desc_b, vals_b, valid_b);
                    }
                } else {
                    PP_STAGE_KERNELS_S2_H_G2(ckv, desc_addr, vals_addr, win_addr, es * p.BWb, es * plane, tw, edge,
                                             desc_b, vals_b, valid_b);
                }
            } else if constexpr (S == 1 && es == 4 && SHIFT == 2) {
                PP_STAGE_KERNELS_S1_B(ckv, desc_addr, vals_addr, win_addr, es * p.BWb, es * plane, tw, edge);
            } else if constexpr (S == 1 && es == 4 && SHIFT == 1) {
                PP_STAGE_KERNELS_S1_A(ckv, desc_addr, vals_addr, win_addr, es * p.BWb, es * plane, tw, edge);
            } else if constexpr (S == 1 && es == 4) {
                PP_STAGE_KERNELS_S1(ckv, desc_addr, vals_addr, win_addr, es * p.BWb, es * plane, tw, edge);
            } else if constexpr (S == 1 && SHIFT) {
                PP_STAGE_KERNELS_S1_HA(ckv, desc_addr, vals_addr, win_addr, es * p.BWb, es * plane, tw, edge);
            } else if constexpr (S == 1) {
                PP_STAGE_KERNELS_S1_H(ckv, desc_addr, vals_addr, win_addr, es * p.BWb, es * plane, tw, edge);
            } else if constexpr (es == 4) {
                PP_STAGE_KERNELS_S2(ckv, desc_addr, vals_addr, win_addr, es * p.BWb, es * plane, tw, edge);
            } else {
                PP_STAGE_KERNELS_S2_H(ckv, desc_addr, vals_addr, win_addr, es * p.BWb, es * plane, tw, edge);
            }
        }
        // release the stage, then take this warp's share of filling chunk q + kStages - 1 into the
        // stage chunk q - 1 used, once all 16 warps have released that one
        __syncwarp();
        if (lane == 0) mbar_arrive(empty0 + 8 * s);
        const int j = q + kStages - 1;
        if (q >= 1 && j < Q) {
            if (!mbar_wait_warp(empty0 + 8 * (j % kStages), ((q - 1) / kStages) & 1, p.status, kStatusEmptyTimeout,
                                p.wait_limit))
                break;
            fill(j);
            if (threadIdx.x == 0) *s_issued = j + 1;
        }
        if (++ck == CU.nck) {   // unit done: results out, accumulators zeroed, next unit's tile
            if (q == Q - 1) pdl_trigger();   // the next kernel may start its set-up from here on
            epilogue(CU);
            ck = 0;
            if (++ci < n_my) place_lane();
        }
    }

    asm volatile("cp.async.wait_all;" ::: "memory");   // this thread's copies (only after a timeout)
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        // no tensor copy of this CTA may still be in flight when it exits (only after a timeout)
        if (lane == 0) {
            const int issued = (int)*s_issued;
            for (int k = max(0, issued - kStages); k < issued; ++k)
                mbar_wait(full0 + 8 * (k % kStages), (k / kStages) & 1, p.status, kStatusDrainTimeout);
        }
        __syncwarp();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(kTmemCols) : "memory");
    }
}

// ------------------------------------------------------------------------------ depthwise

// Depthwise layers (one kernel per channel, as in MobileNet-V2) move 2-4 bytes per 8 useful
// FLOP, so HBM bandwidth bounds them, not the FMA pipe.  The kernel is shaped for bandwidth:
// every thread produces kDwVW consecutive outputs of one output row, reading the three input rows
// it needs with 16-byte loads where rows are 16-byte aligned; the halo columns are single loads
// that hit the neighbouring threads' lines in L1.  Each CTA first expands the four kept weights
// of every plane it covers to the nine taps (zeros at the pruned taps, from the layer's own
// masks) in shared memory, so every lane runs the same branch-free code even where one warp
// covers planes of different patterns.
constexpr int kDwThreads = 256;
constexpr int kDwVW = 8;                   // outputs per thread along a row
constexpr int kDwItemsPerCta = 2048;       // (plane, row, column group) items per CTA
constexpr int kDwMaxPlanes = kDwThreads;   // planes per CTA (one decoding thread each)

struct DwParams {
    const void* x;
    void* y;
    const float* bias;
    const uint32_t* perm;
    const uint64_t* desc;
    const uint32_t* kofs;
    const float4* vals;
    int N, C, H, W, Ho, Wo, relu;
    int NS;                 // slots (G * 8): the planes of one image, in slot order
    int NGX;                // column groups per output row
    int ipp;                // items per plane: Ho * NGX
    int ppc;                // planes per CTA (small planes), else 1
    int tiles;              // CTAs per plane (large planes), else 1
    uint16_t masks[kMaxPatterns];
};

template <typename T>
__device__ __forceinline__ float ld_f32(const T* p) { return to_f32<T>(*p); }

// NV consecutive elements (NV a multiple of 8, 16-byte aligned) widened to fp32
template <int NV>
__device__ __forceinline__ void ld_vec(const float* src, float* dst) {
#pragma unroll
    for (int i = 0; i < NV; i += 4) {
        const float4 v = *reinterpret_cast<const float4*>(src + i);
        dst[i] = v.x;
        dst[i + 1] = v.y;
        dst[i + 2] = v.z;
        dst[i + 3] = v.w;
    }
}
template <int NV>
__device__ __forceinline__ void ld_vec(const __half* src, float* dst) {
#pragma unroll
    for (int i = 0; i < NV; i += 8) {
        const uint4 u = *reinterpret_cast<const uint4*>(src + i);
        const __half2* h = reinterpret_cast<const __half2*>(&u);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float2 f = __half22float2(h[k]);
            dst[i + 2 * k] = f.x;
            dst[i + 2 * k + 1] = f.y;
        }
    }
}

template <int S, typename T, bool VIN, bool VOUT>
__global__ void __launch_bounds__(kDwThreads) pconv_depthwise(const __grid_constant__ DwParams p) {
    pdl_trigger();
    pdl_wait();
    constexpr int NIN = (kDwVW - 1) * S + 3;     // input columns one thread reads per row
    const T* x = static_cast<const T*>(p.x);
    T* y = static_cast<T*>(p.y);
    const int tid = threadIdx.x;
    const long long planes = (long long)p.N * p.NS;
    // this CTA's items: planes [pl0, pl0 + ppc) x all items, or items [it0, it0 + count) of plane pl0
    long long pl0;
    int it0, count;
    if (p.tiles > 1) {
        pl0 = blockIdx.x / p.tiles;
        it0 = (blockIdx.x % p.tiles) * kDwItemsPerCta;
        count = min(kDwItemsPerCta, p.ipp - it0);
    } else {
        pl0 = (long long)blockIdx.x * p.ppc;
        it0 = 0;
        count = (int)min((long long)p.ppc, planes - pl0) * p.ipp;
    }

    // the CTA's planes: thread t < np decodes plane pl0 + t (its channel, nine taps and bias)
    __shared__ float s_w[kDwMaxPlanes][11];
    __shared__ int s_co[kDwMaxPlanes];
    const int np = p.tiles > 1 ? 1 : (int)min((long long)p.ppc, planes - pl0);
    if (tid < np) {
        const long long plane = pl0 + tid;
        const int n = (int)(plane / p.NS), s = (int)(plane - (long long)n * p.NS);
        const uint32_t co = p.perm[s];
        float w9[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        float b = 0.0f;
        unsigned mask_of_slot = 0;
        if (co != kPadSlot) {
            const int g = s >> 3, f = s & 7;
            const uint64_t d = p.desc[g];
            const int cnt = (int)(d & 15u);
            int pat = -1;
            uint32_t k0 = p.kofs[g];
            for (int j = 0; j < cnt; ++j) {
                const int code = (int)((d >> (4 + 6 * j)) & 63u);
                if ((code >> 3) == f) { pat = code & 7; k0 += j; }
            }
            // a pruned kernel has no entry: all nine taps zero, the output is the bias
            const float4 v = pat >= 0 ? p.vals[k0] : make_float4(0.f, 0.f, 0.f, 0.f);
            const unsigned m = pat >= 0 ? p.masks[pat] : 0u;
            mask_of_slot = m;
            int k = 0;
#pragma unroll
            for (int t = 0; t < 9; ++t) {
                const bool on = (m >> t) & 1u;
                const float vk = k == 0 ? v.x : k == 1 ? v.y : k == 2 ? v.z : v.w;
                w9[t] = on ? vk : 0.0f;
                k += on ? 1 : 0;
            }
            b = p.bias ? p.bias[co] : 0.0f;
        }
#pragma unroll
        for (int t = 0; t < 9; ++t) s_w[tid][t] = w9[t];
        s_w[tid][9] = b;
        s_w[tid][10] = __uint_as_float(co == kPadSlot ? 0u : mask_of_slot);
        s_co[tid] = co == kPadSlot ? -1 : (int)co;
    }
    __syncthreads();

    // item e = pl * ipp + it0 + oy * NGX + gx as digits (pl, oy, gx), stepped by the thread count
    // with at most one carry per digit
    const int e = it0 + tid;
    int pl = e / p.ipp;
    const int rem = e - pl * p.ipp;
    int oy = rem / p.NGX, gx = rem - (rem / p.NGX) * p.NGX;
    int st = kDwThreads;
    const int s_pl = st / p.ipp;
    st -= s_pl * p.ipp;
    const int s_oy = st / p.NGX, s_gx = st - (st / p.NGX) * p.NGX;

    // a thread's items stay on one plane for several steps: its taps and base pointers are
    // reloaded only when the plane changes
    int cur = -1, co = -1;
    const T* xp = x;
    T* yp = y;
    float w9[9], b = 0.0f;
    unsigned m = 0;
    for (int i = tid; i < count; i += kDwThreads) {
        if (pl != cur) {
            cur = pl;
            co = s_co[pl];
            const int n = (int)((pl0 + pl) / p.NS);
            xp = x + ((size_t)n * p.C + (co >= 0 ? co : 0)) * p.H * p.W;
            yp = y + ((size_t)n * p.C + (co >= 0 ? co : 0)) * p.Ho * p.Wo;
#pragma unroll
            for (int t = 0; t < 9; ++t) w9[t] = s_w[pl][t];
            b = s_w[pl][9];
            m = __float_as_uint(s_w[pl][10]);
        }
        if (co >= 0) {
            const int c0 = kDwVW * gx;            // first output column of this thread
            const int ic = c0 * S - 1;            // first input column it reads
            float acc[kDwVW];
#pragma unroll
            for (int j = 0; j < kDwVW; ++j) acc[j] = b;
            bool done = false;
            if constexpr (VIN && sizeof(T) == 2) {
                if (ic + 1 + kDwVW * S <= p.W) {
                    // fp16 rows inside the image: the three rows' 16-byte groups and halo columns are
                    // all requested before any is used (raw, 6 or 10 registers a row), then widened
                    constexpr int NV = kDwVW * S / 8;      // 16-byte groups per row
                    uint4 raw[3][NV];
                    __half hl[3], hr[3];
#pragma unroll
                    for (int dy = 0; dy < 3; ++dy) {
                        const int iy = min(max(oy * S - 1 + dy, 0), p.H - 1);
                        const __half* row = reinterpret_cast<const __half*>(xp) + (size_t)iy * p.W;
#pragma unroll
                        for (int v = 0; v < NV; ++v) raw[dy][v] = *reinterpret_cast<const uint4*>(row + ic + 1 + 8 * v);
                        hl[dy] = ic >= 0 ? row[ic] : __float2half(0.0f);
                        hr[dy] = (S == 1 && ic + NIN - 1 < p.W) ? row[ic + NIN - 1] : __float2half(0.0f);
                    }
#pragma unroll
                    for (int dy = 0; dy < 3; ++dy) {
                        const int iy = oy * S - 1 + dy;
                        if (iy < 0 || iy >= p.H) continue;
                        float r[NIN];
                        r[0] = __half2float(hl[dy]);
#pragma unroll
                        for (int v = 0; v < NV; ++v) {
                            const __half2* h = reinterpret_cast<const __half2*>(&raw[dy][v]);
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const float2 f = __half22float2(h[k]);
                                r[1 + 8 * v + 2 * k] = f.x;
                                r[2 + 8 * v + 2 * k] = f.y;
                            }
                        }
                        if (S == 1) r[NIN - 1] = __half2float(hr[dy]);
#pragma unroll
                        for (int dx = 0; dx < 3; ++dx) {
                            if (!((m >> (3 * dy + dx)) & 1u)) continue;   // pruned tap
#pragma unroll
                            for (int j = 0; j < kDwVW; ++j) acc[j] = fmaf(w9[3 * dy + dx], r[j * S + dx], acc[j]);
                        }
                    }
                    done = true;
                }
            }
#pragma unroll
            for (int dy = 0; dy < 3 && !done; ++dy) {
                const int iy = oy * S - 1 + dy;
                if (iy < 0 || iy >= p.H) continue;
                const T* row = xp + (size_t)iy * p.W;
                float r[NIN];
                if (VIN && ic + 1 + kDwVW * S <= p.W) {
                    // columns ic+1 .. ic+kDwVW*S as 16-byte vectors, the halo columns alone
                    ld_vec<kDwVW * S>(row + ic + 1, r + 1);
                    r[0] = ic >= 0 ? ld_f32(row + ic) : 0.0f;
                    if (S == 1) r[NIN - 1] = ic + NIN - 1 < p.W ? ld_f32(row + ic + NIN - 1) : 0.0f;
                } else {
#pragma unroll
                    for (int c = 0; c < NIN; ++c) {
                        const int xc = ic + c;
                        r[c] = (xc >= 0 && xc < p.W) ? ld_f32(row + xc) : 0.0f;
                    }
                }
#pragma unroll
                for (int dx = 0; dx < 3; ++dx) {
                    if (!((m >> (3 * dy + dx)) & 1u)) continue;   // pruned tap
#pragma unroll
                    for (int j = 0; j < kDwVW; ++j) acc[j] = fmaf(w9[3 * dy + dx], r[j * S + dx], acc[j]);
                }
            }
            T* out = yp + (size_t)oy * p.Wo + c0;
            if (VOUT && c0 + kDwVW <= p.Wo) {
                if constexpr (sizeof(T) == 4) {
                    float v[kDwVW];
#pragma unroll
                    for (int j = 0; j < kDwVW; ++j) v[j] = p.relu ? fmaxf(acc[j], 0.0f) : acc[j];
                    float4* o4 = reinterpret_cast<float4*>(out);
                    o4[0] = make_float4(v[0], v[1], v[2], v[3]);
                    o4[1] = make_float4(v[4], v[5], v[6], v[7]);
                } else {
                    uint4 u;
                    __half2* h = reinterpret_cast<__half2*>(&u);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const float a0 = p.relu ? fmaxf(acc[2 * k], 0.0f) : acc[2 * k];
                        const float a1 = p.relu ? fmaxf(acc[2 * k + 1], 0.0f) : acc[2 * k + 1];
                        h[k] = __floats2half2_rn(a0, a1);
                    }
                    *reinterpret_cast<uint4*>(out) = u;
                }
            } else {
#pragma unroll
                for (int j = 0; j < kDwVW; ++j)
                    if (c0 + j < p.Wo) out[j] = from_f32<T>(p.relu ? fmaxf(acc[j], 0.0f) : acc[j]);
            }
        }
        gx += s_gx;
        if (gx >= p.NGX) { gx -= p.NGX; ++oy; }
        oy += s_oy;
        if (oy >= p.Ho) { oy -= p.Ho; ++pl; }
        pl += s_pl;
    }
}

// Staged variant (16-byte aligned x): tiles in channel order, so that a tile's input is one
// contiguous run of memory: npl consecutive channels of one image as whole planes, or one
// channel's band of output rows (npl == 1).  A persistent CTA copies its next tile into shared
// memory with 16-byte cp.async (at the run's own alignment phase) while it computes the current
// one, keeping HBM busy whatever the row width.  Each CTA first decodes the kept weights, bias
// and tap mask of every channel into a shared table (6 words a channel).  Planes whose output rows
// are 7, 14 or 28 wide are computed one whole output row per item (RW below).
struct DwStagedParams {
    const void* x;
    void* y;
    const float* bias;
    const uint32_t* perm;
    const uint64_t* desc;
    const uint32_t* kofs;
    const float4* vals;
    int N, C, H, W, Ho, Wo, relu;
    int NS, NGX;
    int npl, rb, n_cg, n_bands;   // tile: npl channels x rb output rows; channel groups; bands
    int n_tiles;
    long long total_in;           // elements of x
    int buf_elems;                // elements per staging buffer
    unsigned off_w, off_buf;      // shared-memory layout: taps of every channel | 2 buffers
    uint16_t masks[kMaxPatterns];
};

// RW > 0: every plane of a tile is whole and its output rows are RW wide (input rows W = RW for
// stride 1, 2 * RW for stride 2); an item is then one whole output row, read from the staged
// rows with the padding columns as zeros and no bounds test per element, in pairs where the rows
// start on an even element.
template <typename T>
__device__ __forceinline__ void dw_row_load(const T* row, float* r, int W, bool pairs) {
    if (pairs) {
        for (int k = 0; k < W; k += 2) {
            if constexpr (sizeof(T) == 2) {
                const float2 f = __half22float2(*reinterpret_cast<const __half2*>(row + k));
                r[k] = f.x;
                r[k + 1] = f.y;
            } else {
                const float2 f = *reinterpret_cast<const float2*>(row + k);
                r[k] = f.x;
                r[k + 1] = f.y;
            }
        }
    } else {
        for (int k = 0; k < W; ++k) r[k] = to_f32<T>(row[k]);
    }
}

template <int S, typename T, bool VIN, bool VOUT, int RW, int NH>
__global__ void __launch_bounds__(kDwThreads) pconv_depthwise_staged(const __grid_constant__ DwStagedParams p) {
    pdl_trigger();
    pdl_wait();
    constexpr int VE = 16 / (int)sizeof(T);      // elements per 16-byte copy
    constexpr int NIN = (kDwVW - 1) * S + 3;
    extern __shared__ __align__(16) unsigned char dsm[];
    float* s_w = reinterpret_cast<float*>(dsm + p.off_w);   // [C][6]: four kept weights, bias, mask
    T* bufs = reinterpret_cast<T*>(dsm + p.off_buf);
    const T* x = static_cast<const T*>(p.x);
    T* y = static_cast<T*>(p.y);
    const int tid = threadIdx.x;

    struct Tile {
        int n, c0, np, oy0, nro, iy_lo, nri;
        long long g0;       // first input element of the run
    };
    auto tile_of = [&](int t) {
        Tile u;
        const int band = t % p.n_bands;
        const int q = t / p.n_bands;
        const int cg = q % p.n_cg;
        u.n = q / p.n_cg;
        u.c0 = cg * p.npl;
        u.np = min(p.npl, p.C - u.c0);
        u.oy0 = band * p.rb;
        u.nro = min(p.rb, p.Ho - u.oy0);
        u.iy_lo = max(0, u.oy0 * S - 1);
        const int iy_hi = min(p.H - 1, (u.oy0 + u.nro - 1) * S + 1);
        u.nri = iy_hi - u.iy_lo + 1;
        u.g0 = ((long long)u.n * p.C + u.c0) * p.H * p.W + (long long)u.iy_lo * p.W;
        return u;
    };
    // issue the copy of tile t's run into buffer b: whole 16-byte blocks from the block holding
    // its first element (plain loads for a block that reaches past the end of x)
    auto load = [&](const Tile& u, int b) {
        T* buf = bufs + (size_t)b * p.buf_elems;
        const long long len = (long long)u.np * u.nri * p.W;
        const long long v_lo = u.g0 / VE, v_hi = (u.g0 + len - 1) / VE;
        for (long long v = v_lo + tid; v <= v_hi; v += kDwThreads) {
            const long long ge = v * VE;
            T* dst = buf + (ge - v_lo * VE);
            if (ge + VE <= p.total_in) {
                cp_async16(dst, x + ge);
            } else {
                for (int k = 0; k < VE; ++k)
                    if (ge + k < p.total_in) dst[k] = x[ge + k];
            }
        }
    };
    // kept weights, bias and tap mask of every channel, once per CTA: the thread of slot s decodes
    // its kernel (a pruned one has no entry: mask 0, the output is the bias)
    auto decode_all = [&]() {
        for (int s = tid; s < p.NS; s += kDwThreads) {
            const uint32_t co = p.perm[s];
            if (co == kPadSlot) continue;
            const int g = s >> 3, f = s & 7;
            const uint64_t d = p.desc[g];
            const int cnt = (int)(d & 15u);
            int pat = -1;
            uint32_t k0 = p.kofs[g];
            for (int j = 0; j < cnt; ++j) {
                const int code = (int)((d >> (4 + 6 * j)) & 63u);
                if ((code >> 3) == f) { pat = code & 7; k0 += j; }
            }
            const float4 v = pat >= 0 ? p.vals[k0] : make_float4(0.f, 0.f, 0.f, 0.f);
            float* w = s_w + co * 6;
            w[0] = v.x;
            w[1] = v.y;
            w[2] = v.z;
            w[3] = v.w;
            w[4] = p.bias ? p.bias[co] : 0.0f;
            w[5] = __uint_as_float(pat >= 0 ? p.masks[pat] : 0u);
        }
    };
    // nine taps of channel c (zeros at the pruned ones), its bias and mask
    auto taps_of = [&](int c, float (&w9)[9], float& bias, unsigned& m) {
        const float* w = s_w + c * 6;
        m = __float_as_uint(w[5]);
        bias = w[4];
        int k = 0;
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            const bool on = (m >> t) & 1u;
            const float vk = w[k < 3 ? k : 3];
            w9[t] = on ? vk : 0.0f;
            k += on ? 1 : 0;
        }
    };
    auto compute_rows = [&](const Tile& u, int b) {   // RW > 0: an output row (or half of it) per item
        constexpr int RWO = RW > 0 ? RW : 2;             // (the RW = 0 instance never calls this)
        constexpr int RIN = (RWO - 1) * S + 3;           // input columns -1 .. (RW - 1) * S + 1 of a piece
        constexpr int nh = NH;                           // pieces per output row (2 for 28-wide rows)
        constexpr int WI = RWO * S * NH;                 // staged row width (== p.W)
        const T* buf = bufs + (size_t)b * p.buf_elems;
        const int off0 = (int)(u.g0 - (u.g0 / VE) * VE);
        const bool pairs = WI % 2 == 0 && off0 % 2 == 0 && (RWO * S) % 2 == 0;
        const bool opairs = RWO % 2 == 0 && reinterpret_cast<uintptr_t>(y) % (2 * sizeof(T)) == 0;
        const int items = u.np * u.nro * nh;
        for (int it = tid; it < items; it += kDwThreads) {
            const int q = it / nh, h = it - q * nh;
            const int pl = q / u.nro, oyl = q - pl * u.nro;
            const int cb = h * RWO * S;                  // first input column of the piece
            float w9[9], bv;
            unsigned mk;
            taps_of(u.c0 + pl, w9, bv, mk);
            const int oy = u.oy0 + oyl;
            float acc[RWO];
#pragma unroll
            for (int j = 0; j < RWO; ++j) acc[j] = bv;
#pragma unroll
            for (int dy = 0; dy < 3; ++dy) {
                const int iy = oy * S - 1 + dy;
                if (iy < 0 || iy >= p.H) continue;
                const T* row = buf + off0 + (size_t)(pl * u.nri + iy - u.iy_lo) * WI;
                float r[RIN + 1];
                r[0] = cb > 0 ? to_f32<T>(row[cb - 1]) : 0.0f;
                r[RIN] = 0.0f;
                if constexpr (S == 1) r[RIN - 1] = cb + RWO < WI ? to_f32<T>(row[cb + RWO]) : 0.0f;
                dw_row_load<T>(row + cb, r + 1, RWO * S, pairs);
#pragma unroll
                for (int dx = 0; dx < 3; ++dx)
#pragma unroll
                    for (int j = 0; j < RWO; ++j) acc[j] = fmaf(w9[3 * dy + dx], r[j * S + dx], acc[j]);
            }
            T* out = y + (((size_t)u.n * p.C + u.c0 + pl) * p.Ho + oy) * (RWO * NH) + h * RWO;
            if (opairs) {
#pragma unroll
                for (int j = 0; j < RWO; j += 2) {
                    const float a0 = p.relu ? fmaxf(acc[j], 0.0f) : acc[j];
                    const float a1 = p.relu ? fmaxf(acc[j + 1], 0.0f) : acc[j + 1];
                    if constexpr (sizeof(T) == 2) *reinterpret_cast<__half2*>(out + j) = __floats2half2_rn(a0, a1);
                    else *reinterpret_cast<float2*>(out + j) = make_float2(a0, a1);
                }
            } else {
#pragma unroll
                for (int j = 0; j < RWO; ++j) out[j] = from_f32<T>(p.relu ? fmaxf(acc[j], 0.0f) : acc[j]);
            }
        }
    };
    auto compute = [&](const Tile& u, int b) {
        const T* buf = bufs + (size_t)b * p.buf_elems;
        const int off0 = (int)(u.g0 - (u.g0 / VE) * VE);   // buffer index of the run's first element
        const int per_pl = u.nro * p.NGX;
        const int items = u.np * per_pl;
        int pl = tid / per_pl;
        const int rem = tid - pl * per_pl;
        int oyl = rem / p.NGX, gx = rem - (rem / p.NGX) * p.NGX;
        int st = kDwThreads;
        const int s_pl = st / per_pl;
        st -= s_pl * per_pl;
        const int s_oy = st / p.NGX, s_gx = st - (st / p.NGX) * p.NGX;
        int cur = -1;
        float w9[9], bv = 0.0f;
        unsigned m = 0;
        for (int i = tid; i < items; i += kDwThreads) {
            if (pl != cur) {
                cur = pl;
                taps_of(u.c0 + pl, w9, bv, m);
            }
            const int oy = u.oy0 + oyl;
            const int c0 = kDwVW * gx, ic = c0 * S - 1;
            float acc[kDwVW];
#pragma unroll
            for (int j = 0; j < kDwVW; ++j) acc[j] = bv;
#pragma unroll
            for (int dy = 0; dy < 3; ++dy) {
                const int iy = oy * S - 1 + dy;
                if (iy < 0 || iy >= p.H) continue;
                const T* row = buf + off0 + (pl * u.nri + iy - u.iy_lo) * p.W;
                float r[NIN];
                if (VIN && ic + 1 + kDwVW * S <= p.W) {   // rows 16-byte aligned in the buffer too
                    ld_vec<kDwVW * S>(row + ic + 1, r + 1);
                    r[0] = ic >= 0 ? ld_f32(row + ic) : 0.0f;
                    if (S == 1) r[NIN - 1] = ic + NIN - 1 < p.W ? ld_f32(row + ic + NIN - 1) : 0.0f;
                } else {
#pragma unroll
                    for (int c = 0; c < NIN; ++c) {
                        const int xc = ic + c;
                        r[c] = (xc >= 0 && xc < p.W) ? ld_f32(row + xc) : 0.0f;
                    }
                }
#pragma unroll
                for (int dx = 0; dx < 3; ++dx) {
                    if (!((m >> (3 * dy + dx)) & 1u)) continue;   // pruned tap
#pragma unroll
                    for (int j = 0; j < kDwVW; ++j) acc[j] = fmaf(w9[3 * dy + dx], r[j * S + dx], acc[j]);
                }
            }
            T* out = y + (((size_t)u.n * p.C + u.c0 + pl) * p.Ho + oy) * p.Wo + c0;
            if (VOUT && c0 + kDwVW <= p.Wo) {
                if constexpr (sizeof(T) == 4) {
                    float v[kDwVW];
#pragma unroll
                    for (int j = 0; j < kDwVW; ++j) v[j] = p.relu ? fmaxf(acc[j], 0.0f) : acc[j];
                    float4* o4 = reinterpret_cast<float4*>(out);
                    o4[0] = make_float4(v[0], v[1], v[2], v[3]);
                    o4[1] = make_float4(v[4], v[5], v[6], v[7]);
                } else {
                    uint4 q;
                    __half2* h = reinterpret_cast<__half2*>(&q);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const float a0 = p.relu ? fmaxf(acc[2 * k], 0.0f) : acc[2 * k];
                        const float a1 = p.relu ? fmaxf(acc[2 * k + 1], 0.0f) : acc[2 * k + 1];
                        h[k] = __floats2half2_rn(a0, a1);
                    }
                    *reinterpret_cast<uint4*>(out) = q;
                }
            } else {
#pragma unroll
                for (int j = 0; j < kDwVW; ++j)
                    if (c0 + j < p.Wo) out[j] = from_f32<T>(p.relu ? fmaxf(acc[j], 0.0f) : acc[j]);
            }
            gx += s_gx;
            if (gx >= p.NGX) { gx -= p.NGX; ++oyl; }
            oyl += s_oy;
            if (oyl >= u.nro) { oyl -= u.nro; ++pl; }
            pl += s_pl;
        }
    };

    int t = blockIdx.x;
    if (t < p.n_tiles) load(tile_of(t), 0);
    asm volatile("cp.async.commit_group;" ::: "memory");
    decode_all();                                      // overlaps the first tile's copy
    for (int k = 0; t < p.n_tiles; ++k, t += gridDim.x) {
        const Tile u = tile_of(t);
        const int tn = t + (int)gridDim.x;
        if (tn < p.n_tiles) load(tile_of(tn), (k + 1) & 1);
        asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();                               // tile t staged (and, at k = 0, the taps)
        if constexpr (RW > 0) compute_rows(u, k & 1);
        else compute(u, k & 1);
        __syncthreads();                               // buffer k & 1 free again
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// ------------------------------------------------------------------------------ streamed depthwise

// Streamed depthwise kernel (16-byte aligned tensors).  Every warp of a persistent CTA is its own
// copy/compute pipeline with a private ring of shared-memory stages and one mbarrier per stage, so
// no CTA barrier separates copying from computing and each SM keeps many copies in flight.  A
// chunk is
//   * rows mode (MODE 0; rows of a multiple of 16 bytes, at most 256 elements): R output rows of
//     one plane.  One tensor copy brings its (R - 1) S + 3 whole input rows, the rows above and
//     below the image zero-filled by the copy.  Lane (h, g) computes output columns 4g .. 4g + 3
//     of rows h RPL .. (h + 1) RPL - 1 and rolls three input rows through registers; the channel
//     is the same for the whole warp, so pruned taps are skipped by uniform branches;
//   * planes mode (MODE 1: stride 2, one output column per lane; MODE 2 / 3: stride 1, two
//     output columns per lane as packed FMAs, rows of even / odd width): P consecutive whole
//     planes, which are contiguous in NCHW, by one bulk copy.  A lane owns columns of one plane
//     and walks down its rows, taking the neighbouring input columns from the adjacent lanes by
//     shuffle; a pass of the warp covers NPW planes, so the lanes of a warp meet several channels
//     and apply all nine taps (zeros at the pruned ones).  Outputs go to a shared-memory buffer
//     that one bulk copy writes back.
// Warp w of the grid takes chunks w, w + nw, w + 2 nw, ... (nw warps in the grid).  Each CTA holds
// the nine taps, the bias and the tap mask of every channel in a table (kDwsTab words a channel).
constexpr int kDwsWarps = 16;
constexpr int kDwsThreads = 32 * kDwsWarps;
constexpr int kDwsMaxStages = 4;
constexpr int kDwsCW = 4;     // rows mode: output columns per lane
constexpr int kDwsTab = 12;   // table words per channel: taps 0-8, bias, mask, unused

struct DwsParams {
    const void* x;
    void* y;
    const float* bias;
    const uint32_t* perm;
    const uint64_t* desc;
    const uint32_t* kofs;
    const float4* vals;
    unsigned* status;
    int N, C, H, W, Ho, Wo, relu, NS;
    int nst;                              // stages per warp
    long long n_chunks;
    int R, RIN, n_bands, NCG, NHL, RPL;   // rows mode
    int P, LPP, NPW;                      // planes mode: planes per chunk, lanes per plane, planes per pass
    int ipp, npc;                         // tiles mode: lane items per plane, row pieces per output row
    long long n_planes;                   // N * C
    unsigned in_b;                        // bytes of one input stage
    unsigned off_tab, off_area, area_b;   // shared memory: mbarriers | table | one area per warp
    unsigned zoff;                        // tiles mode: a zero row within each warp's area
    int nwarps;                           // warps per CTA (the launch's block is 32 nwarps threads)
    int vec_out;                          // rows mode: 4-output vector stores
    uint16_t masks[kMaxPatterns];
};

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z,
                                            uint32_t mbar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(mbar) : "memory");
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(mbar) : "memory");
}
__device__ __forceinline__ void bulk_store(void* dst, uint32_t src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src), "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

template <typename T>
__device__ __forceinline__ float2 ld_pair(const T* q);
template <>
__device__ __forceinline__ float2 ld_pair<float>(const float* q) { return *reinterpret_cast<const float2*>(q); }
template <>
__device__ __forceinline__ float2 ld_pair<__half>(const __half* q) {
    return __half22float2(*reinterpret_cast<const __half2*>(q));
}
template <typename T>
__device__ __forceinline__ void st_pair(T* q, float a, float b);
template <>
__device__ __forceinline__ void st_pair<float>(float* q, float a, float b) { *reinterpret_cast<float2*>(q) = make_float2(a, b); }
template <>
__device__ __forceinline__ void st_pair<__half>(__half* q, float a, float b) {
    *reinterpret_cast<__half2*>(q) = __floats2half2_rn(a, b);
}

// rows mode: the window columns of one staged row for output columns c0 .. c0 + 3: input columns
// c0 - 1 .. c0 + 4 (stride 1) or 2 c0 - 1 .. 2 c0 + 7 (stride 2), zeros outside the image
template <int S, typename T>
__device__ __forceinline__ void dws_row(const T* row, int c0, int W, float (&v)[(kDwsCW - 1) * S + 3]) {
    constexpr int NM = kDwsCW * S;     // columns c0 S .. c0 S + NM - 1: one or two 16-byte loads, or 8 bytes
    const T* m = row + c0 * S;
    if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int i = 0; i < NM; i += 4) {
            const float4 q = *reinterpret_cast<const float4*>(m + i);
            v[1 + i] = q.x;
            v[2 + i] = q.y;
            v[3 + i] = q.z;
            v[4 + i] = q.w;
        }
    } else if constexpr (NM == 4) {
        const uint2 u = *reinterpret_cast<const uint2*>(m);
        const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&u.x));
        const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&u.y));
        v[1] = a.x;
        v[2] = a.y;
        v[3] = b.x;
        v[4] = b.y;
    } else {
        const uint4 u = *reinterpret_cast<const uint4*>(m);
        const uint32_t w4[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w4[k]));
            v[1 + 2 * k] = f.x;
            v[2 + 2 * k] = f.y;
        }
    }
    v[0] = c0 > 0 ? to_f32<T>(m[-1]) : 0.0f;
    if constexpr (S == 1) v[NM + 1] = c0 + NM < W ? to_f32<T>(m[NM]) : 0.0f;
}

// Rows mode, one lane: output rows r0 .. r0 + nrows - 1 of a chunk's band at output columns c0 ..
// c0 + 3, from staged rows r S, r S + 1, r S + 2 (`off`: element offset of staged row r0 S,
// column c0 S; `W`: elements per staged row).  The taps are those of mask M, known at compile
// time (one of the pattern library's masks, so each output takes exactly its kept taps; 0x1FF:
// all nine, zeros at the pruned ones), applied in ascending raster order.  Input rows rotate
// through a register ring unrolled by its length, so no row is copied.
template <int S, typename T, unsigned M>
__device__ __forceinline__ void dws_rows(const T* st, int off, int W, T* yr, int Wo, int nrows, bool has_l,
                                         bool has_r, bool relu, const float (&w)[9], float bv) {
    constexpr int NI = (kDwsCW - 1) * S + 3;
    constexpr bool kL = (M & 0x49u) != 0;              // a tap in column dx = 0 (taps 0, 3, 6)
    constexpr bool kR = S == 1 && (M & 0x124u) != 0;   // stride 1: a tap in column dx = 2 (2, 5, 8)
    struct Row { float e[NI]; };
    auto fetch = [&](Row& v) {
        const T* m = st + off;
        if constexpr (sizeof(T) == 4) {
#pragma unroll
            for (int i = 0; i < kDwsCW * S; i += 4) {
                const float4 f = *reinterpret_cast<const float4*>(m + i);
                v.e[1 + i] = f.x;
                v.e[2 + i] = f.y;
                v.e[3 + i] = f.z;
                v.e[4 + i] = f.w;
            }
        } else if constexpr (S == 1) {
            const uint2 u = *reinterpret_cast<const uint2*>(m);
            const float2 f0 = __half22float2(*reinterpret_cast<const __half2*>(&u.x));
            const float2 f1 = __half22float2(*reinterpret_cast<const __half2*>(&u.y));
            v.e[1] = f0.x;
            v.e[2] = f0.y;
            v.e[3] = f1.x;
            v.e[4] = f1.y;
        } else {
            const uint4 u = *reinterpret_cast<const uint4*>(m);
            const uint32_t w4[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w4[i]));
                v.e[1 + 2 * i] = f.x;
                v.e[2 + 2 * i] = f.y;
            }
        }
        v.e[0] = 0.0f;
        if constexpr (kL) {   // column c0 S - 1, read inside the stage and zeroed at the image's edge
            const float l = to_f32<T>(m[has_l ? -1 : 0]);
            v.e[0] = has_l ? l : 0.0f;
        }
        if constexpr (S == 1) {
            v.e[5] = 0.0f;
            if constexpr (kR) {
                const float r = to_f32<T>(m[has_r ? 4 : 3]);
                v.e[5] = has_r ? r : 0.0f;
            }
        }
        off += W;
    };
    auto out = [&](const Row& u, const Row& v, const Row& x3) {
        float a[kDwsCW];
#pragma unroll
        for (int j = 0; j < kDwsCW; ++j) {
            float o = bv;
#pragma unroll
            for (int t = 0; t < 9; ++t) {
                if ((M >> t) & 1u) {
                    const Row& rr = t < 3 ? u : (t < 6 ? v : x3);
                    o = fmaf(w[t], rr.e[j * S + t % 3], o);
                }
            }
            a[j] = relu ? fmaxf(o, 0.0f) : o;
        }
        if constexpr (sizeof(T) == 4) {
            *reinterpret_cast<float4*>(yr) = make_float4(a[0], a[1], a[2], a[3]);
        } else {
            __half2 h0 = __floats2half2_rn(a[0], a[1]), h1 = __floats2half2_rn(a[2], a[3]);
            uint2 q;
            q.x = *reinterpret_cast<unsigned*>(&h0);
            q.y = *reinterpret_cast<unsigned*>(&h1);
            *reinterpret_cast<uint2*>(yr) = q;
        }
        yr += Wo;
    };
    Row A, B, C;
    if constexpr (S == 1) {
        fetch(A);
        fetch(B);
        for (int r = 0; r < nrows; r += 3) {
            fetch(C);
            out(A, B, C);
            if (r + 1 >= nrows) break;
            fetch(A);
            out(B, C, A);
            if (r + 2 >= nrows) break;
            fetch(B);
            out(C, A, B);
        }
    } else {
        fetch(A);
        for (int r = 0; r < nrows; r += 2) {
            fetch(B);
            fetch(C);
            out(A, B, C);
            if (r + 1 >= nrows) break;
            fetch(B);
            fetch(A);
            out(C, B, A);
        }
    }
}

// Tiles mode, one lane: output rows oy0 .. oy0 + BR - 1 and columns c0 .. c0 + PW - 1 of one plane,
// computed in straight-line code: every input row of the tile is read once into a register ring
// (rows above and below the image from a zero row), all offsets are compile-time constants, and
// all nine taps are applied (zeros at the pruned ones), in ascending raster order.  `xp` / `op`:
// the plane's first element in the stage / in the output buffer.  PAIRS: rows of even width with
// c0 S even, so the staged row segments are read and the outputs written as element pairs.
template <int S, typename T, int PW, int BR, bool PAIRS>
__device__ __forceinline__ void dws_tile(const T* xp, T* op, const T* zrow, int W, int H, int Wo, int oy0, int c0,
                                         bool relu, const float (&w)[9], float bv) {
    constexpr int NM = PW * S;       // columns c0 S .. c0 S + NM - 1 (stride 2: through 2 (c0 + PW) - 1)
    constexpr int NIN = NM + 2;      // with column c0 S - 1 in front and c0 S + NM behind
    const bool has_l = c0 > 0;
    const bool has_r = S == 1 && c0 + PW < W;   // stride 2 never reads column 2 (c0 + PW)
    float v[3][NIN];
    auto fetch = [&](int k, float (&r)[NIN]) {   // input row oy0 S - 1 + k
        const int iy = oy0 * S - 1 + k;
        const T* row = (iy >= 0 && iy < H) ? xp + iy * W + c0 * S : zrow;
        if constexpr (PAIRS) {
#pragma unroll
            for (int i = 0; i < NM; i += 2) {
                const float2 f = ld_pair<T>(row + i);
                r[1 + i] = f.x;
                r[2 + i] = f.y;
            }
        } else {
#pragma unroll
            for (int i = 0; i < NM; ++i) r[1 + i] = to_f32<T>(row[i]);
        }
        const float l = to_f32<T>(row[-1]);   // inside the stage (or the zero row); zeroed at the edge
        r[0] = has_l ? l : 0.0f;
        if constexpr (S == 1) {
            const float rr = to_f32<T>(row[NM]);
            r[NIN - 1] = has_r ? rr : 0.0f;
        } else {
            r[NIN - 1] = 0.0f;
        }
    };
    auto out = [&](int orow, const float (&a)[NIN], const float (&b)[NIN], const float (&c)[NIN]) {
        float o[PW];
#pragma unroll
        for (int j = 0; j < PW; ++j) {
            float q = bv;
            q = fmaf(w[0], a[j * S], q);
            q = fmaf(w[1], a[j * S + 1], q);
            q = fmaf(w[2], a[j * S + 2], q);
            q = fmaf(w[3], b[j * S], q);
            q = fmaf(w[4], b[j * S + 1], q);
            q = fmaf(w[5], b[j * S + 2], q);
            q = fmaf(w[6], c[j * S], q);
            q = fmaf(w[7], c[j * S + 1], q);
            q = fmaf(w[8], c[j * S + 2], q);
            o[j] = relu ? fmaxf(q, 0.0f) : q;
        }
        T* d = op + (oy0 + orow) * Wo + c0;
        if constexpr (PAIRS && PW % 2 == 0) {
#pragma unroll
            for (int j = 0; j < PW; j += 2) st_pair<T>(d + j, o[j], o[j + 1]);
        } else {
#pragma unroll
            for (int j = 0; j < PW; ++j) d[j] = from_f32<T>(o[j]);
        }
    };
    if constexpr (S == 1) {
        fetch(0, v[0]);
        fetch(1, v[1]);
#pragma unroll
        for (int r = 0; r < BR; ++r) {
            fetch(r + 2, v[(r + 2) % 3]);
            out(r, v[r % 3], v[(r + 1) % 3], v[(r + 2) % 3]);
        }
    } else {
        fetch(0, v[0]);
#pragma unroll
        for (int r = 0; r < BR; ++r) {
            fetch(2 * r + 1, v[(2 * r + 1) % 3]);
            fetch(2 * r + 2, v[(2 * r + 2) % 3]);
            out(r, v[(2 * r) % 3], v[(2 * r + 1) % 3], v[(2 * r + 2) % 3]);
        }
    }
}

template <int S, typename T, int MODE>
__global__ void __launch_bounds__(kDwsThreads, 1)
    pconv_dw_stream(const __grid_constant__ DwsParams p, const __grid_constant__ CUtensorMap tmap) {
    static_assert(MODE != 2 && MODE != 3 && MODE != 4 && MODE != 5 || S == 1, "a stride-1 layout");
    static_assert(MODE != 6 || S == 2, "a stride-2 layout");
    pdl_trigger();
    extern __shared__ __align__(128) unsigned char smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t bar0 = smem_u32(smem) + 8u * kDwsMaxStages * warp;
    float* tab = reinterpret_cast<float*>(smem + p.off_tab);
    unsigned char* area = smem + p.off_area + (size_t)warp * p.area_b;
    T* ob = reinterpret_cast<T*>(area + (size_t)p.nst * p.in_b);   // planes mode: output buffer
    const T* x = static_cast<const T*>(p.x);
    T* y = static_cast<T*>(p.y);
    const int nwarps = (int)(blockDim.x >> 5), nthr = (int)blockDim.x;
    const int wid = (int)blockIdx.x * nwarps + warp, nw = (int)gridDim.x * nwarps;   // chunks < 2^31
    const int n_mine = (int)p.n_chunks > wid ? ((int)p.n_chunks - 1 - wid) / nw + 1 : 0;
    if (lane == 0) {
        for (int s = 0; s < p.nst; ++s) mbar_init(bar0 + 8u * s, 1);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the barriers, for the copies
    }
    if constexpr (MODE >= 4) {   // this warp's zero row (tiles mode: rows above and below the image)
        if (lane < 32) reinterpret_cast<uint32_t*>(area + p.zoff)[lane] = 0u;
    }
    // taps and mask of every channel (slot s holds channel perm[s]; a pruned kernel has no entry:
    // mask 0, all taps zero): up to four slots a thread, their independent loads issued together
    // (two rounds of L2 latency).  The packed layer is immutable once bound, so this runs before
    // the previous kernel of the stream has completed (programmatic launch)
    for (int s0 = threadIdx.x; s0 < p.NS; s0 += 4 * nthr) {
        uint32_t co[4], ko[4];
        uint64_t d[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int s = s0 + u * nthr;
            const bool in = s < p.NS;
            co[u] = in ? p.perm[s] : kPadSlot;
            d[u] = in ? p.desc[s >> 3] : 0ull;
            ko[u] = in ? p.kofs[s >> 3] : 0u;
        }
        float4 v[4];
        unsigned msk[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int f = (s0 + u * nthr) & 7;
            const int cnt = (int)(d[u] & 15u);
            int pat = -1, jj = 0;
            for (int j2 = 0; j2 < cnt; ++j2) {
                const int code = (int)((d[u] >> (4 + 6 * j2)) & 63u);
                if ((code >> 3) == f) {
                    pat = code & 7;
                    jj = j2;
                }
            }
            const bool live = co[u] != kPadSlot;
            v[u] = live && pat >= 0 ? p.vals[ko[u] + jj] : make_float4(0.f, 0.f, 0.f, 0.f);
            msk[u] = live && pat >= 0 ? p.masks[pat] : 0u;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (co[u] == kPadSlot) continue;
            float* w = tab + (size_t)co[u] * kDwsTab;
            int k = 0;
#pragma unroll
            for (int t = 0; t < 9; ++t) {
                const bool on = (msk[u] >> t) & 1u;
                const float vk = k == 0 ? v[u].x : k == 1 ? v[u].y : k == 2 ? v[u].z : v[u].w;
                w[t] = on ? vk : 0.0f;
                k += on ? 1 : 0;
            }
            w[10] = __uint_as_float(msk[u]);
            w[11] = 0.0f;
        }
    }
    pdl_wait();   // activations and the bias from here on
    const size_t pb = (size_t)p.H * p.W * sizeof(T), opb = (size_t)p.Ho * p.Wo * sizeof(T);
    auto issue = [&](int j) {   // lane 0: the copy of this warp's j-th chunk into stage j % nst
        const long long ch = (long long)wid + (long long)j * nw;
        const uint32_t bar = bar0 + 8u * (j % p.nst);
        const uint32_t dst = smem_u32(area + (size_t)(j % p.nst) * p.in_b);
        if constexpr (MODE == 0) {
            const int q = (int)(ch / p.n_bands), b = (int)(ch - (long long)q * p.n_bands);
            mbar_arrive_expect_tx(bar, (uint32_t)((size_t)p.W * p.RIN * sizeof(T)));
            tma_load_3d(dst, &tmap, 0, b * p.R * S - 1, q, bar);
        } else {
            const long long q0 = ch * p.P;
            const long long np = min((long long)p.P, p.n_planes - q0);
            const uint32_t bytes = (uint32_t)((size_t)np * pb) & ~15u;   // the rest (end of x) by plain loads
            mbar_arrive_expect_tx(bar, bytes);
            if (bytes) bulk_load(dst, reinterpret_cast<const unsigned char*>(p.x) + (size_t)q0 * pb, bytes, bar);
        }
    };
    const int first = min(p.nst, n_mine);
    if (lane == 0)
        for (int j = 0; j < first; ++j) issue(j);
    int issued = first;
    for (int c = threadIdx.x; c < p.C; c += nthr) tab[(size_t)c * kDwsTab + 9] = p.bias ? p.bias[c] : 0.0f;
    __syncthreads();   // the table is complete

    // rows mode: rows h RPL .. of the chunk's band, output columns 4g .. 4g + 3.  The channel is
    // the same for the whole warp, so its tap mask selects once per chunk a row loop compiled for
    // that pattern (the library's eight) or, for any other mask, for all nine taps.
    const int W = p.W, H = p.H, Wo = p.Wo, Ho = p.Ho, C = p.C;
    const bool relu = p.relu != 0;
    auto rows_chunk = [&](long long ch, const T* st) {
        const int q = (int)(ch / p.n_bands), b = (int)(ch - (long long)q * p.n_bands);
        const float4* tw = reinterpret_cast<const float4*>(tab + (size_t)(q % C) * kDwsTab);
        const float4 t0 = tw[0], t1 = tw[1], t2 = tw[2];
        const float w[9] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w, t2.x};
        const float bv = t2.y;
        const unsigned m = __float_as_uint(t2.z);
        const int oy0 = b * p.R, nro = min(p.R, Ho - oy0);
        const int h = lane / p.NCG, g = lane - h * p.NCG;
        const int r0 = h * p.RPL, r1 = min(r0 + p.RPL, nro);
        if (h >= p.NHL || r0 >= r1) return;
        const int c0 = g * kDwsCW;
        const bool has_l = c0 > 0, has_r = c0 + kDwsCW * S < W;
        const int off = r0 * S * W + c0 * S;
        T* yr = y + ((size_t)q * Ho + oy0 + r0) * Wo + c0;
        const int n = r1 - r0;
        switch (m) {
            case kDefaultMasks[0]: dws_rows<S, T, kDefaultMasks[0]>(st, off, W, yr, Wo, n, has_l, has_r, relu, w, bv); break;
            case kDefaultMasks[1]: dws_rows<S, T, kDefaultMasks[1]>(st, off, W, yr, Wo, n, has_l, has_r, relu, w, bv); break;
            case kDefaultMasks[2]: dws_rows<S, T, kDefaultMasks[2]>(st, off, W, yr, Wo, n, has_l, has_r, relu, w, bv); break;
            case kDefaultMasks[3]: dws_rows<S, T, kDefaultMasks[3]>(st, off, W, yr, Wo, n, has_l, has_r, relu, w, bv); break;
            case kDefaultMasks[4]: dws_rows<S, T, kDefaultMasks[4]>(st, off, W, yr, Wo, n, has_l, has_r, relu, w, bv); break;
            case kDefaultMasks[5]: dws_rows<S, T, kDefaultMasks[5]>(st, off, W, yr, Wo, n, has_l, has_r, relu, w, bv); break;
            case kDefaultMasks[6]: dws_rows<S, T, kDefaultMasks[6]>(st, off, W, yr, Wo, n, has_l, has_r, relu, w, bv); break;
            case kDefaultMasks[7]: dws_rows<S, T, kDefaultMasks[7]>(st, off, W, yr, Wo, n, has_l, has_r, relu, w, bv); break;
            default: dws_rows<S, T, 0x1FFu>(st, off, W, yr, Wo, n, has_l, has_r, relu, w, bv); break;
        }
    };

    // planes mode: the warp's passes over the chunk's planes; lane l owns columns of plane
    // l / LPP of the pass.  Every lane runs the same code with no branch of its own: an idle lane
    // reads plane 0 of the stage and writes its results to a junk word of the warp's output buffer,
    // as does a lane's second output beyond an odd-width row; columns outside the image are read
    // inside the stage and zeroed by select.  Stride 1 (MODE 2, rows of even width; MODE 3, odd):
    // output columns 2j, 2j + 1 as packed FMAs, the neighbouring input columns from the adjacent
    // lanes; stride 2 (MODE 1): output column j from input columns 2j - 1 .. 2j + 1, scalar FMAs.
    // All nine taps are applied (the lanes of a pass meet several channels), zeros at the pruned ones.
    auto planes_chunk = [&](long long ch, const T* st) {
        const long long q0 = ch * p.P;
        const int np = (int)min((long long)p.P, p.n_planes - q0);
        const int pl_l = lane / p.LPP, j = lane - pl_l * p.LPP;
        const int npw = p.NPW;
        const int c_first = (int)(q0 % C);
        constexpr int CPL = MODE == 1 ? 1 : 2;
        const bool has_l = j > 0;
        const bool has_b = S == 1 && 2 * j + 1 < W;    // stride 1: the lane's second column exists
        const bool has_r = S == 1 && 2 * j + 2 < W;
        const int boff = has_b ? 1 : 0;
        T* junk = ob + (size_t)p.P * Ho * Wo;          // past the chunk's outputs (the buffer has room)
        for (int k = 0; k < np; k += npw) {
            const int pl = k + pl_l;
            const bool act = pl_l < npw && pl < np;
            const int plx = act ? pl : 0;
            int c = c_first + plx;
            while (c >= C) c -= C;
            const float4* tw = reinterpret_cast<const float4*>(tab + (size_t)c * kDwsTab);
            const float4 t0 = tw[0], t1 = tw[1], t2 = tw[2];
            const float w[9] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w, t2.x};
            const float bv = t2.y;
            int xo = plx * H * W + j * 2;                          // input column 2j of row 0
            T* o0 = act ? ob + (size_t)pl * Ho * Wo + j * CPL : junk;
            T* o1 = act && has_b ? o0 + 1 : junk;
            const int ostep = act ? Wo : 0, ostep1 = act && has_b ? Wo : 0;
            if constexpr (S == 1) {
                struct Row { float2 q[3]; };   // (left, a), (a, b), (b, right)
                auto fetch = [&](Row& v) {
                    float a, b;
                    if constexpr (MODE == 2) {
                        const float2 f = ld_pair<T>(st + xo);
                        a = f.x;
                        b = f.y;
                    } else {
                        a = to_f32<T>(st[xo]);
                        const float bb = to_f32<T>(st[xo + boff]);
                        b = has_b ? bb : 0.0f;
                    }
                    xo += W;
                    const float l = __shfl_up_sync(0xffffffffu, b, 1);
                    const float r = __shfl_down_sync(0xffffffffu, a, 1);
                    v.q[0] = make_float2(has_l ? l : 0.0f, a);
                    v.q[1] = make_float2(a, b);
                    v.q[2] = make_float2(b, has_r ? r : 0.0f);
                };
                float2 w2[9];
#pragma unroll
                for (int t = 0; t < 9; ++t) w2[t] = make_float2(w[t], w[t]);
                auto out = [&](const Row& u, const Row& v, const Row& x3) {
                    float2 o = make_float2(bv, bv);
#pragma unroll
                    for (int dx = 0; dx < 3; ++dx) {
                        o = __ffma2_rn(w2[dx], u.q[dx], o);
                        o = __ffma2_rn(w2[3 + dx], v.q[dx], o);
                        o = __ffma2_rn(w2[6 + dx], x3.q[dx], o);
                    }
                    if (relu) {
                        o.x = fmaxf(o.x, 0.0f);
                        o.y = fmaxf(o.y, 0.0f);
                    }
                    if constexpr (MODE == 2) {
                        st_pair<T>(o0, o.x, o.y);
                    } else {
                        *o0 = from_f32<T>(o.x);
                        *o1 = from_f32<T>(o.y);
                        o1 += ostep1;
                    }
                    o0 += ostep;
                };
                Row A, B, Cr;
                A.q[0] = A.q[1] = A.q[2] = make_float2(0.0f, 0.0f);   // input row -1
                fetch(B);
                for (int oy = 0; oy < Ho; oy += 3) {
                    if (oy + 1 < H) fetch(Cr); else Cr.q[0] = Cr.q[1] = Cr.q[2] = make_float2(0.0f, 0.0f);
                    out(A, B, Cr);
                    if (oy + 1 >= Ho) break;
                    if (oy + 2 < H) fetch(A); else A.q[0] = A.q[1] = A.q[2] = make_float2(0.0f, 0.0f);
                    out(B, Cr, A);
                    if (oy + 2 >= Ho) break;
                    if (oy + 3 < H) fetch(B); else B.q[0] = B.q[1] = B.q[2] = make_float2(0.0f, 0.0f);
                    out(Cr, A, B);
                }
            } else {
                struct Row { float e[3]; };   // input columns 2j - 1, 2j, 2j + 1
                auto fetch = [&](Row& v) {
                    const float2 f = ld_pair<T>(st + xo);
                    xo += W;
                    const float l = __shfl_up_sync(0xffffffffu, f.y, 1);
                    v.e[0] = has_l ? l : 0.0f;
                    v.e[1] = f.x;
                    v.e[2] = f.y;
                };
                auto out = [&](const Row& u, const Row& v, const Row& x3) {
                    float o = bv;
#pragma unroll
                    for (int dx = 0; dx < 3; ++dx) {
                        o = fmaf(w[dx], u.e[dx], o);
                        o = fmaf(w[3 + dx], v.e[dx], o);
                        o = fmaf(w[6 + dx], x3.e[dx], o);
                    }
                    if (relu) o = fmaxf(o, 0.0f);
                    *o0 = from_f32<T>(o);
                    o0 += ostep;
                };
                Row A, B, Cr;
                A.e[0] = A.e[1] = A.e[2] = 0.0f;   // input row -1
                for (int oy = 0; oy < Ho; oy += 2) {
                    fetch(B);
                    if (2 * oy + 1 < H) fetch(Cr); else Cr.e[0] = Cr.e[1] = Cr.e[2] = 0.0f;
                    out(A, B, Cr);
                    if (oy + 1 >= Ho) break;
                    fetch(B);
                    if (2 * oy + 3 < H) fetch(A); else A.e[0] = A.e[1] = A.e[2] = 0.0f;
                    out(Cr, B, A);
                }
            }
        }
    };

    // tiles mode: lane items (plane, band of BR output rows, piece of PW output columns), 32 a pass;
    // a lane past the chunk's items repeats item 0 (the same values to the same place)
    auto tiles_chunk = [&](long long ch, const T* st) {
        constexpr int PW = MODE == 5 ? 14 : 7, BR = 7;
        const long long q0 = ch * p.P;
        const int np = (int)min((long long)p.P, p.n_planes - q0);
        const int items = np * p.ipp;
        const int c_first = (int)(q0 % C);
        const T* zrow = reinterpret_cast<const T*>(area + p.zoff) + 2;
        for (int i0 = 0; i0 < items; i0 += 32) {
            const int it = i0 + lane < items ? i0 + lane : 0;
            const int pl = it / p.ipp, rem = it - pl * p.ipp;
            const int band = rem / p.npc, piece = rem - band * p.npc;
            int c = c_first + pl;
            while (c >= C) c -= C;
            const float4* tw = reinterpret_cast<const float4*>(tab + (size_t)c * kDwsTab);
            const float4 t0 = tw[0], t1 = tw[1], t2 = tw[2];
            const float w[9] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w, t2.x};
            dws_tile<S, T, PW, BR, MODE != 4>(st + pl * H * W, ob + pl * Ho * Wo, zrow, W, H, Wo, band * BR,
                                               piece * PW, relu, w, t2.y);
        }
    };

    bool ok = true;
    int j = 0;
    for (; j < n_mine; ++j) {
        const int s = j % p.nst;
        if (!mbar_wait_warp(bar0 + 8u * s, (uint32_t)((j / p.nst) & 1), p.status, kStatusFullTimeout, kTimeoutCycles)) {
            ok = false;
            break;
        }
        const long long ch = (long long)wid + (long long)j * nw;
        T* st = reinterpret_cast<T*>(area + (size_t)s * p.in_b);
        if constexpr (MODE == 0) {
            rows_chunk(ch, st);
        } else {
            const long long q0 = ch * p.P;
            const long long np = min((long long)p.P, p.n_planes - q0);
            const size_t in_e = (size_t)np * pb / sizeof(T), full_e = (((size_t)np * pb) & ~(size_t)15) / sizeof(T);
            if (full_e < in_e) {   // the end of x: the last few elements by plain loads
                for (size_t i = full_e + lane; i < in_e; i += 32) st[i] = x[(size_t)q0 * (pb / sizeof(T)) + i];
                __syncwarp();
            }
            if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // ob free again
            __syncwarp();
            if constexpr (MODE >= 4) tiles_chunk(ch, st);
            else planes_chunk(ch, st);
            const size_t out_e = (size_t)np * opb / sizeof(T), fo_e = (((size_t)np * opb) & ~(size_t)15) / sizeof(T);
            T* yc = y + (size_t)q0 * (opb / sizeof(T));
            for (size_t i = fo_e + lane; i < out_e; i += 32) yc[i] = ob[i];   // the end of y by plain stores
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // ob visible to the bulk copy
            __syncwarp();
            if (lane == 0 && fo_e) bulk_store(yc, smem_u32(ob), (uint32_t)(fo_e * sizeof(T)));
        }
        __syncwarp();
        if (j + p.nst < n_mine) {
            if (lane == 0) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                issue(j + p.nst);
            }
            ++issued;
        }
    }
    if (lane == 0) {
        // after a timeout no copy of this warp may still be landing when the CTA exits
        if (!ok)
            for (int k = j; k < issued; ++k)
                mbar_wait(bar0 + 8u * (k % p.nst), (uint32_t)((k / p.nst) & 1), p.status, kStatusDrainTimeout);
        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
    __syncwarp();
}

// ------------------------------------------------------------------------------ generic path

struct TapTable {
    int8_t t[kMaxPatterns][4];
};

// Any pattern library: one thread per output, taps read from a table (slow, for libraries other
// than the compiled one).  Dense or depthwise (cin_g == 1 and ci == co).
template <typename T>
__global__ void pconv_generic(const T* __restrict__ x, T* __restrict__ y, const float* __restrict__ bias,
                              const uint32_t* perm, const uint64_t* desc, const uint32_t* kofs,
                              const float4* vals, TapTable taps, int N, int C, int cin_g, int dw, int H,
                              int W, int Cout, int Ho, int Wo, int S, int relu) {
    const int nslot = (Cout + kF - 1) / kF * kF;   // padding slots may sit anywhere in a group
    const long long total = (long long)N * nslot * Ho * Wo;
    for (long long o = blockIdx.x * (long long)blockDim.x + threadIdx.x; o < total;
         o += (long long)gridDim.x * blockDim.x) {
        const int ox = (int)(o % Wo);
        long long r = o / Wo;
        const int oy = (int)(r % Ho);
        r /= Ho;
        const int slot = (int)(r % nslot);
        const int n = (int)(r / nslot);
        const uint32_t co = perm[slot];
        if (co == kPadSlot) continue;
        const int g = slot / kF, f = slot % kF;
        float a = 0.0f;
        for (int ci = 0; ci < cin_g; ++ci) {
            uint64_t d = desc[(size_t)g * cin_g + ci];
            const int cnt = (int)(d & 15u);
            d >>= 4;
            for (int e = 0; e < cnt; ++e) {
                const int code = (int)((d >> (6 * e)) & 63u);
                if ((code >> 3) != f) continue;
                const int pat = code & 7;
                const float4 w = vals[kofs[(size_t)g * cin_g + ci] + e];
                const float wv[4] = {w.x, w.y, w.z, w.w};
                const int xc = dw ? (int)co : ci;
                for (int k = 0; k < 4; ++k) {
                    const int tp = taps.t[pat][k];
                    const int iy = oy * S + tp / 3 - 1, ix = ox * S + tp % 3 - 1;
                    if (iy >= 0 && iy < H && ix >= 0 && ix < W)
                        a = fmaf(wv[k], to_f32<T>(x[(((size_t)n * C + xc) * H + iy) * W + ix]), a);
                }
            }
        }
        a += bias ? bias[co] : 0.0f;
        y[(((size_t)n * Cout + co) * Ho + oy) * Wo + ox] = from_f32<T>(relu ? fmaxf(a, 0.0f) : a);
    }
}

// ------------------------------------------------------------------------------ max-pool

template <typename T>
__global__ void maxpool2x2(const T* __restrict__ x, T* __restrict__ y, long long planes, int H, int W) {
    const int Ho = H / 2, Wo = W / 2;
    const long long total = planes * Ho * Wo;
    for (long long o = blockIdx.x * (long long)blockDim.x + threadIdx.x; o < total;
         o += (long long)gridDim.x * blockDim.x) {
        const int ox = (int)(o % Wo);
        const long long r = o / Wo;
        const int oy = (int)(r % Ho);
        const long long pl = r / Ho;
        const T* xp = x + (pl * H + 2 * oy) * W + 2 * ox;
        const float a = fmaxf(to_f32<T>(xp[0]), to_f32<T>(xp[1]));
        const float b = fmaxf(to_f32<T>(xp[W]), to_f32<T>(xp[W + 1]));
        y[o] = from_f32<T>(fmaxf(a, b));
    }
}


// ------------------------------------------------------------------------------ FP32 peak
// The roofline denominator of the pattern-sparse kernel, measured instead of taken from the
// nominal lane count: 16 independent fma.rn.f32 chains per thread (4-cycle latency hidden by 16
// warps per SM scheduler), 4 CTAs of 512 threads per SM, no memory traffic.
constexpr int kPeakChains = 16, kPeakUnroll = 4;
__device__ float g_fma_sink;

__global__ void __launch_bounds__(512, 4) fma_peak(int iters) {
    float a[kPeakChains];
#pragma unroll
    for (int i = 0; i < kPeakChains; ++i) a[i] = 1e-3f * (float)(threadIdx.x + i);
    const float m = 0.999f, c = 1e-7f;
    for (int it = 0; it < iters; ++it) {
#pragma unroll
        for (int i = 0; i < kPeakChains; ++i) {
#pragma unroll
            for (int u = 0; u < kPeakUnroll; ++u) asm volatile("fma.rn.f32 %0, %0, %1, %2;" : "+f"(a[i]) : "f"(m), "f"(c));
        }
    }
    float sum = 0.0f;
#pragma unroll
    for (int i = 0; i < kPeakChains; ++i) sum += a[i];
    if (sum == 12345.0f) g_fma_sink = sum;   // keeps the chains live; never true in practice
}

// ------------------------------------------------------------------------------ static scratch
// Scratch for pp_conv_static_scratch: a fixed array in the library's own device image, so that
// callers which may not allocate device memory still get the input-channel split.  It exists on
// every GPU that loads the library, from module load until process exit.
constexpr size_t kStaticScratchBytes = (size_t)32 << 20;
static __device__ __align__(256) float g_pp_scratch[kStaticScratchBytes / sizeof(float)];

// ------------------------------------------------------------------------------ host side

int sm_count() {
    static std::atomic<int> cached[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 152;   // no device: plan for a GB300
    if (dev < 64 && cached[dev].load() > 0) return cached[dev].load();
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 152;
    if (dev < 64) cached[dev].store(n);
    return n;
}

// Kernel launch with programmatic stream serialisation (pdl_wait / pdl_trigger) on a stream that
// is not being captured, unless the environment sets PATCONV_PDL=0; returns the launch's error,
// which it also clears.  In a CUDA graph the kernel nodes already follow each other without host
// work, and programmatic edges there measured slower for the dense kernels (VGG-16 at batch 1:
// 0.477 against 0.464 ms per image; equal at batch 32), so their captured launches are plain
// ones; the streamed depthwise kernel keeps the edge (pdl_captured), whose set-up (the tap table)
// then overlaps the previous kernel.
bool pdl_enabled() {
    static const bool on = [] {
        const char* e = std::getenv("PATCONV_PDL");
        return !(e && e[0] == '0');
    }();
    return on;
}

// Stride-2 layers give each warp two filter groups (PATCONV_S2_GROUPS=1: one, as stride 1 does).
bool s2_two_groups() {
    static const bool on = [] {
        const char* e = std::getenv("PATCONV_S2_GROUPS");
        return !(e && e[0] == '1');
    }();
    return on;
}

// The balanced schedule can be switched off (PATCONV_BALANCED=0): plans then take whole units.
bool balanced_enabled() {
    static const bool on = [] {
        const char* e = std::getenv("PATCONV_BALANCED");
        return !(e && e[0] == '0');
    }();
    return on;
}

template <typename... KArgs, typename... Args>
cudaError_t launch_ex(bool cooperative, void (*kern)(KArgs...), unsigned grid, unsigned block, size_t smem,
                      cudaStream_t st, bool pdl_captured, const Args&... args) {
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    const bool captured = cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone;
    if (cooperative) {   // CTAs that wait on each other: all resident at once
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.numAttrs = 1;
    } else {
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.numAttrs = pdl_enabled() && (!captured || pdl_captured) ? 1 : 0;
    }
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, args...);
    const cudaError_t l = cudaGetLastError();
    return e != cudaSuccess ? e : l;
}

template <typename... KArgs, typename... Args>
cudaError_t launch(void (*kern)(KArgs...), unsigned grid, unsigned block, size_t smem, cudaStream_t st,
                   const Args&... args) {
    return launch_ex(false, kern, grid, block, smem, st, false, args...);
}

using EncodeTiledFn = PFN_cuTensorMapEncodeTiled_v12000;

EncodeTiledFn encode_tiled() {
    static const EncodeTiledFn fn = []() -> EncodeTiledFn {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return nullptr;
        return reinterpret_cast<EncodeTiledFn>(f);
    }();
    return fn;
}

// Test hook (pp_debug_inject_timeout): the next pattern-sparse launch issues no stage fills and
// waits this many SM cycles (about 10 us) for them, so every CTA's first pipeline wait runs out.
std::atomic<int> g_inject_timeout{0};
constexpr long long kInjectedWaitCycles = 20000;

unsigned* status_word() {
    static std::atomic<unsigned*> cached[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    if (dev < 64 && cached[dev].load()) return cached[dev].load();
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_pp_status) != cudaSuccess) return nullptr;
    if (dev < 64) cached[dev].store(static_cast<unsigned*>(ptr));
    return static_cast<unsigned*>(ptr);
}

struct TileChoice {
    int BY = 1, BX = 1, NB = 1, IH = 0, BWb = 0;
    int linear = 0;   // lanes take consecutive blocks of the (image, row, column) sequence
};

size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// Launch plan of the pattern-sparse kernel for one call shape (shared by the workspace query,
// the plan query and the launch, so all three agree).
struct Plan {
    int WG = 0, WS = 0, n_fchunks = 0;
    TileChoice tile;
    int tiles_x = 0, tiles_y = 0, tiles_n = 0;
    int CK = 0, n_chunks = 0, maxk = 0, KS = 1, c_split = 0;
    size_t stage_bytes = 0, kb_bytes = 0, smem = 0;
    long long ctas = 0;           // CTAs of one split
    int lane_sort = 0;            // stride 1: pconv_tm deals blocks to lanes by bank group
    int shift = 0;                // stride 1: blocks start at output columns 4j - shift (SHIFT)
    int streamk = 0;              // balanced schedule over sm_count() CTAs (KS = 1)
    int dg = 1;                   // stride 2: filter groups per warp (2: 8 warps of 16 slots)
    size_t ws_bytes = 0;          // workspace the chosen split or schedule needs (0: none)
    bool tensor = false;          // a layer bound for it takes the tensor-core kernel, as planned in tc
    TensorPlan tc;
};

// Workspace of the balanced schedule over P CTAs: a slot of raw accumulators per CTA, then a flag
// per (CTA, warp).
size_t streamk_bytes(long long P) {
    return align_up((size_t)P * kSlotFloats * sizeof(float), 256) + (size_t)P * kCompute * sizeof(unsigned);
}

struct PlanCache : PlanCacheBase {
    std::mutex mu;
    std::map<std::tuple<int, int, int, size_t, int>, Plan> plans;
};

// Candidate spatial tiles of at most 32*WS blocks (4x4 outputs each; with shift, block j of a row
// starts at output column 4j - shift, so a row of Wo outputs takes (Wo + shift + 3) / 4 blocks).
//   rectangles: BY x BX blocks of one image (several whole images when the rectangle is the
//     whole image; several images side by side when it is a band of full block rows, below);
//     stride-1 rows need 4*BX + 5 staged columns, stride-2 rows 8*BX + 4, rounded
//     to a 16-byte multiple and padded to 4 (mod 8) floats so that rows four apart fall in other
//     banks;
//   linear: 32*WS consecutive blocks of the (image, block row, block column) sequence, staged as
//     the whole images they touch; no lane idles even when an image's block count is no divisor
//     of the lane count (28 x 28 outputs: 49 blocks).
std::vector<TileChoice> tile_candidates(int N, int Ho, int Wo, int S, int lanes, int shift) {
    const int nby = (Ho + 3) / 4, nbx = (Wo + shift + 3) / 4;
    auto bw_of = [&](int bx) {
        int bw = S == 1 ? 4 * bx + 8 : 8 * bx + 4;
        if (bw % 8 == 0) bw += 4;
        return bw;
    };
    auto ih_of = [&](int by) { return S == 1 ? 4 * by + 2 : 8 * by + 1; };
    std::vector<TileChoice> out;
    for (int bx = 1; bx <= std::min(nbx, lanes); ++bx) {
        for (int by = 1; by <= std::min(nby, lanes / bx); ++by) {
            const bool whole = by == nby && bx == nbx;
            const int nb = whole ? std::max(1, std::min(std::min(N, 256), lanes / (bx * by))) : 1;
            const int ih = ih_of(by), bw = bw_of(bx);
            if (bw > 256 || ih > 256) continue;
            out.push_back(TileChoice{by, bx, nb, ih, bw, 0});
        }
    }
    const long long bpi = (long long)nby * nbx;
    // bands: full-width rectangles of `by` block rows (a divisor of the image's block rows, so no
    // row is computed past the image) of several images side by side in one stage, where a whole
    // image is more than the lanes hold.  28x28 outputs are 7 block rows: rectangles of 4 block
    // rows compute 8 of them, bands of 1 block row of 4 images exactly 7.  Listed after the
    // rectangles, so they are taken only where they cover strictly fewer lanes.  Measured against
    // the rectangles they replace: VGG-16's 28x28 layers 7-10 % faster (4.74 -> 4.60 ms a step),
    // ResNet-50's 56x56 and 28x28 layers 9 and 6 %, its first stride-2 head 13 %
    if (bpi > lanes) {
        for (int by = 1; by < nby && by * nbx <= lanes / 2; ++by) {
            if (nby % by) continue;
            const int nb = std::min(N, lanes / (nbx * by));
            const int ih = ih_of(by), bw = bw_of(nbx);
            if (nb >= 2 && bw <= 256 && ih <= 256) out.push_back(TileChoice{by, nbx, nb, ih, bw, 0});
        }
    }
    if (bpi < lanes && lanes % bpi == 0) return out;    // the whole-image rectangle is this tile
    const int nb = (int)std::min<long long>(N, (lanes - 1) / bpi + 2);
    const int ih = ih_of(nby), bw = bw_of(nbx);
    if (N > 1 && bpi < 4LL * lanes && ih <= 256 && bw <= 256 && nb <= 256)
        out.push_back(TileChoice{nby, nbx, nb, ih, bw, 1});
    return out;
}

// Shared-memory wavefronts of warp 0's 16-byte window loads (window columns 1-4 of every lane,
// fp32 stride-1 stage) in tile t: four phases of 8 lanes, each costing the largest number of its
// lanes whose loads fall on one bank group (16 bytes = 4 banks; 8 groups).  Lanes take the tile's
// blocks in raster order, or dealt by bank group as pconv_tm does with lane_sort.
int window_wavefronts(const Plan& pl, int N, long long t, bool sorted, int S = 1) {
    const TileChoice& tc = pl.tile;
    const int lanes_t = 32 * pl.WS, bpi = tc.BY * tc.BX, plane = tc.IH * tc.BWb;
    int grp[32], key[32], order[32];
    for (int l = 0; l < 32; ++l) {
        int img, rem;
        bool active;
        if (tc.linear) {
            const long long b = t * lanes_t + l;
            const long long ng = b / bpi, n0 = t * lanes_t / bpi;
            img = (int)(ng - n0);
            rem = (int)(b - ng * bpi);
            active = ng < N && img < tc.NB;
        } else {
            img = l / bpi;
            rem = l - img * bpi;
            active = img < tc.NB;
        }
        const int by = rem / tc.BX, bx = rem - by * tc.BX;
        const long long off = (long long)img * pl.CK * plane + (long long)by * 4 * S * tc.BWb + bx * 4 * S;
        grp[l] = active ? (int)((off / 4) & 7) : 8;
    }
    for (int l = 0; l < 32; ++l) {
        int rank = 0;
        for (int i = 0; i < l; ++i) rank += grp[i] == grp[l];
        key[l] = grp[l] < 8 ? 16 * rank + grp[l] : 1024 + l;
    }
    for (int l = 0; l < 32; ++l) {
        int pos = l;
        if (sorted) {
            pos = 0;
            for (int i = 0; i < 32; ++i) pos += key[i] < key[l];
        }
        order[pos] = l;
    }
    int w = 0;
    for (int ph = 0; ph < 4; ++ph) {
        int cnt[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0}, m = 0;
        for (int k = 0; k < 8; ++k) {
            const int g = grp[order[8 * ph + k]];
            if (g < 8) m = std::max(m, ++cnt[g]);
        }
        w += m;
    }
    return w;
}

int make_plan_uncached(const pp_layer* L, int N, int H, int W, size_t ws_avail, int shift, Plan* out,
                       double* cost, bool allow_sk, int es) {
    const int S = L->stride;
    const bool tma_rows = ((size_t)W * es) % 16 == 0;   // the input goes through TMA (if aligned)
    const int Ho = (H - 1) / S + 1, Wo = (W - 1) / S + 1;
    int wg = 1;
    while (wg < L->G && wg < kCompute) wg *= 2;
    const int WS = kCompute / wg, lanes = 32 * WS;
    const int n_fchunks = (L->G + wg - 1) / wg;
    const int C = L->cin_g;
    const int nby = (Ho + 3) / 4, nbx = (Wo + shift + 3) / 4;
    const long long sms = sm_count();
    const size_t out_elems = (size_t)N * L->cout * Ho * Wo;

    auto maxk_for = [&](int ck) {
        uint32_t m = 0;
        for (int g = 0; g < L->G; ++g)
            for (int c0 = 0; c0 < C; c0 += ck) {
                const size_t b = (size_t)g * C;
                m = std::max(m, L->kofs[b + std::min(c0 + ck, C)] - L->kofs[b + c0]);
            }
        return (int)m;
    };
    // channels per stage (the largest that fits three stages in shared memory) and input-channel
    // split of one tile; returns the estimated time in channel steps (infinite if it cannot run).
    // The split is chosen in chunk units: waves x (chunks per split + start-up) + a reduction term.
    auto finish = [&](const TileChoice& t, int tx, int ty, int tn, Plan* pl) -> double {
        pl->WG = wg;
        pl->WS = WS;
        pl->n_fchunks = n_fchunks;
        pl->tile = t;
        pl->tiles_x = tx;
        pl->tiles_y = ty;
        pl->tiles_n = tn;
        pl->ctas = (long long)tn * ty * tx * n_fchunks;
        auto layout = [&](int ck, int maxk, size_t* stage_bytes, size_t* kb_bytes) {
            const size_t in_b = align_up((size_t)t.NB * ck * t.IH * t.BWb * 4, 128);
            const size_t desc_b = align_up((size_t)wg * ck * 8, 16);
            const size_t vals_b = (size_t)wg * std::max(maxk, 1) * 16;
            *stage_bytes = align_up(in_b + desc_b + vals_b, 128);
            *kb_bytes = (size_t)kMaxUnitsPerCta * sizeof(Unit);   // the CTA's unit table
            return align_up(64 + *kb_bytes, 128) + kStages * *stage_bytes;
        };
        int ck = std::min(C, 64);
        for (;; --ck) {
            if (ck < 1 || (C + ck - 1) / ck > kMaxChunks) return 1e300;
            pl->maxk = maxk_for(ck);
            pl->smem = layout(ck, pl->maxk, &pl->stage_bytes, &pl->kb_bytes);
            if (pl->smem <= 200 * 1024) break;
        }
        // several images in a stage: an image stride of a multiple of 32 floats puts every image's
        // windows on the same bank groups (7x7 maps: 8 images of 2x2 blocks, 4 bank groups in
        // all); one channel less per stage where that lowers the modelled window wavefronts
        auto wavefronts_for = [&](int c) {
            Plan q = *pl;
            q.CK = c;
            const long long nt = t.linear ? std::min<long long>(tn, 64) : 1;
            long long w = 0;
            for (long long i = 0; i < nt; ++i)
                w += std::min(window_wavefronts(q, N, i, false, S), window_wavefronts(q, N, i, true, S));
            return w;
        };
        if (S == 1 && t.NB > 1 && ck > 1 && ((size_t)ck * t.IH * t.BWb) % 32 == 0 &&
            (C + ck - 2) / (ck - 1) <= kMaxChunks && wavefronts_for(ck - 1) < wavefronts_for(ck)) {
            --ck;
            pl->maxk = maxk_for(ck);
            pl->smem = layout(ck, pl->maxk, &pl->stage_bytes, &pl->kb_bytes);
        }
        // stride 2 (fp32, two filter groups per warp): a row's blocks sit 32 bytes apart, on every
        // other 16-byte bank group, so only blocks of other images can fill a phase's other groups;
        // an image stride of an odd number of groups lets the blocks dealt by bank group do that.
        // Up to three channels less per stage where the modelled wavefronts fall
        if (S == 2 && es == 4 && wg >= 2 && s2_two_groups() && t.NB > 1 && !t.linear) {
            int best = ck;
            long long bw = wavefronts_for(ck);
            for (int c = ck - 1; c >= std::max(1, ck - 3); --c) {
                if ((C + c - 1) / c > kMaxChunks) break;
                const long long w = wavefronts_for(c);
                if (w < bw) {
                    bw = w;
                    best = c;
                }
            }
            if (best != ck) {
                ck = best;
                pl->maxk = maxk_for(ck);
                pl->smem = layout(ck, pl->maxk, &pl->stage_bytes, &pl->kb_bytes);
            }
        }
        pl->CK = ck;
        pl->maxk = std::max(pl->maxk, 1);
        const int nck_total = (C + ck - 1) / ck;
        int best_ks = 1;
        double best_cost = 1e300;
        for (int ksp = 1; ksp <= std::min(8, nck_total); ++ksp) {
            const int per = (nck_total + ksp - 1) / ksp;
            const int used = (nck_total + per - 1) / per;
            if (used != ksp) continue;                       // every split must get chunks
            if (ksp > 1 && ws_avail < (size_t)ksp * out_elems * 4) break;
            const long long waves = (pl->ctas * ksp + sms - 1) / sms;
            const double cost = (double)waves * (per + 2.0) + (ksp > 1 ? 0.5 * ksp : 0.0);
            if (cost < best_cost - 1e-9) {
                best_cost = cost;
                best_ks = ksp;
            }
        }
        pl->KS = best_ks;
        int per = (nck_total + best_ks - 1) / best_ks;
        pl->c_split = per * ck;
        pl->n_chunks = std::min(per, nck_total);
        pl->ws_bytes = best_ks > 1 ? (size_t)best_ks * out_elems * 4 : 0;
        long long waves = (pl->ctas * best_ks + sms - 1) / sms;
        double steps = (double)waves * (std::min(pl->c_split, C) + 2.0 * per + 2.0 * ck);
        // tiny launches (the SMs stay idle even with 8 splits): fewer channels per stage and up to
        // 32 splits within one wave (more cost more in partial sums than they save: measured on the
        // 64->64 32x32 N=1 layer and the sweep's N=1 points), chosen by estimated channel steps.
        // Not below 16 input channels: there every split writes and reads back an output-sized
        // plane of partial sums for a channel or two of work (VGG-16 layer 1 at batch 1, 3 input
        // channels: 25.9 us split 3 ways, 14.0 us whole)
        if (pl->ctas * std::min(8, nck_total) < sms && C >= 16) {
            for (int ck2 = ck;; ck2 = std::max(1, ck2 / 2)) {
                const int nck2 = (C + ck2 - 1) / ck2;
                if (nck2 > kMaxChunks) break;
                for (int ksp = 2; ksp <= std::min(32, nck2); ++ksp) {
                    const int per2 = (nck2 + ksp - 1) / ksp;
                    if ((nck2 + per2 - 1) / per2 != ksp) continue;
                    if (ws_avail < (size_t)ksp * out_elems * 4 || pl->ctas * ksp > sms) break;   // one wave
                    const long long w2 = (pl->ctas * ksp + sms - 1) / sms;
                    const double st2 = (double)w2 * (std::min(per2 * ck2, C) + 2.0 * per2 + 2.0 * ck2) + 4.0;
                    if (st2 < steps - 1e-9) {
                        steps = st2;
                        pl->CK = ck2;
                        pl->KS = ksp;
                        per = per2;
                        pl->c_split = per2 * ck2;
                        pl->n_chunks = std::min(per2, nck2);
                        pl->ws_bytes = (size_t)ksp * out_elems * 4;
                        pl->maxk = std::max(maxk_for(ck2), 1);
                    }
                }
                if (ck2 == 1) break;
            }
            pl->smem = layout(pl->CK, pl->maxk, &pl->stage_bytes, &pl->kb_bytes);
        }
        // balanced schedule: P = sm_count() CTAs take equal ranges of the units' chunk sequence
        // (KS = 1); a unit cut at a range boundary is finished by the CTA holding its first
        // chunks, which adds the later CTAs' raw sums from their workspace slots.  Every CTA gets
        // T / P chunks instead of whole units, where the last partial wave of whole units leaves
        // SMs idle (busy share <= 0.88) and there are at least 0.75 units per CTA.  It costs the
        // slots' traffic (256 KiB per CTA out and in, about 14 us a launch measured on VGG-16)
        // and the launch overlap of the previous kernel (a cooperative launch), so it is taken
        // only with a 5 % margin.  Only on persistent CTAs (the input through TMA, or tiles of
        // whole images), at stride 1 or at stride 2 with two filter groups per warp
        pl->streamk = 0;
        const long long U1 = pl->ctas;   // whole units without a split
        const double busy = (double)U1 / ((double)sms * ((U1 + sms - 1) / sms));
        // persistent CTAs: through TMA, or rectangles of whole images (the copy fallback's zero
        // halo is then the same for every unit).  Two kinds of launch take the schedule down to 0.2
        // units per CTA and whatever the estimate, as measured faster than whole units or the
        // channel split on 128 CTAs: copy-fallback rectangles of whole images (VGG-16's 14x14 layers
        // 13 %, 64 units at batch 32; ResNet-50's 14x14 and 7x7 layers 8-10 %, 64 and 32 units at
        // batch 64), stride 2 with two filter groups per warp (ResNet-50's heads 5 and 12 %,
        // 128 units of 128 input channels and 64 units of 256) and bands (the estimate puts them
        // level with a 2-way channel split, whose partial sums and reduction pass it leaves out)
        const bool whole = tx == 1 && ty == 1 && !t.linear && !tma_rows;
        const bool relax = whole || S == 2 || (t.NB > 1 && ty > 1);
        const bool persist = tma_rows || whole;
        if ((S == 1 || (wg >= 2 && s2_two_groups())) && allow_sk && balanced_enabled() && persist && busy <= 0.88 &&
            (4 * U1 >= 3 * sms || relax)) {
            const long long T = U1 * nck_total;
            const size_t skb = streamk_bytes(sms);
            if (T >= 2 * sms && U1 <= (long long)(kMaxUnitsPerCta - 2) * sms && ws_avail >= skb) {
                const double cost_sk = (double)U1 * (C + 2.0 * nck_total) / sms + 4.0 * ck + 42.0;
                if (cost_sk < 0.95 * steps || relax) {
                    steps = cost_sk;
                    pl->streamk = 1;
                    pl->KS = 1;
                    pl->CK = ck;
                    pl->c_split = nck_total * ck;
                    pl->n_chunks = nck_total;
                    pl->maxk = std::max(maxk_for(ck), 1);
                    pl->ws_bytes = skb;
                    pl->smem = layout(pl->CK, pl->maxk, &pl->stage_bytes, &pl->kb_bytes);
                }
            }
        }
        return steps;
    };

    // rectangles: fewest CTA waves, then fewest lanes covered (idle lanes), then the widest rows;
    // a tile must leave room for at least the channels per stage that kMaxChunks needs
    const int ck_min = (C + kMaxChunks - 1) / kMaxChunks;
    const double kpc_all = (double)L->beta / ((double)L->G * C);   // kept kernels per (channel, group)
    long long best_waves = LLONG_MAX, best_cover = LLONG_MAX;
    TileChoice rect, lin;
    int rtx = 0, rty = 0, rtn = 0;
    bool have_rect = false, have_lin = false;
    for (const TileChoice& t : tile_candidates(N, Ho, Wo, S, lanes, shift)) {
        if ((long long)t.NB * t.IH * t.BWb * 4 * ck_min > 48 * 1024) continue;
        // bands only through TMA (the copy fallback, one CTA per unit, stages their extra halo
        // rows with the compute threads) and below 6 kept kernels per (input channel, filter
        // group): at 8 (keep 1.0) the linear tile's lanes, all busy, beat the bands' 7 of 8
        // (28x28 maps: 4-9 % in 4 of 6 sweep points, 1-6 % slower in the other 2)
        if (t.NB > 1 && t.BY < nby && !t.linear && (!tma_rows || kpc_all >= 6.0)) continue;
        if (t.linear) {
            lin = t;
            have_lin = true;
            continue;
        }
        const int tx = (nbx + t.BX - 1) / t.BX, ty = (nby + t.BY - 1) / t.BY, tn = (N + t.NB - 1) / t.NB;
        const long long tiles = (long long)tn * ty * tx;
        const long long waves = (tiles * n_fchunks + sms - 1) / sms;
        const long long cover = tiles * lanes;
        if (waves < best_waves ||
            (waves == best_waves && (cover < best_cover || (cover == best_cover && t.BX > rect.BX)))) {
            rect = t;
            rtx = tx;
            rty = ty;
            rtn = tn;
            best_waves = waves;
            best_cover = cover;
            have_rect = true;
        }
    }
    // the linear tile stages whole images (fewer channels per stage, more stages) and its lanes
    // hit more bank conflicts: a per-channel cost, worth about 1.3 kernel visits against 0.4 for
    // a rectangle's window, so its estimated channel steps are weighed by (1.3 + k) / (0.4 + k), k
    // the layer's mean kept kernels per (input channel, filter group).  Calibrated on 28x28 maps
    // (VGG-16 and the sweep): rectangles win at k <= 2.4 (VGG-16 layers 8-10: -11, -2, +1 %), the
    // linear tile at k = 8 (by 17-29 %: idle lanes) and mostly at k = 4
    Plan pr, pli;
    const double cr = have_rect ? finish(rect, rtx, rty, rtn, &pr) : 1e300;
    const int ltn = (int)(((long long)N * nby * nbx + lanes - 1) / lanes);
    const double cl = have_lin ? (1.3 + kpc_all) / (0.4 + kpc_all) * finish(lin, 1, 1, ltn, &pli) : 1e300;
    if (cr >= 1e300 && cl >= 1e300) return PP_ERR_SHAPE;
    *out = cl < cr ? pli : pr;
    out->shift = shift;
    *cost = std::min(cl, cr);
    // the bank-group order where it lowers the window loads' wavefronts (stride 2: fp32 with two
    // filter groups per warp)
    if (S == 1 || (es == 4 && out->WG >= 2 && s2_two_groups())) {
        const long long nt = out->tile.linear ? std::min<long long>(out->tiles_n, 64) : 1;
        long long raster = 0, sorted = 0;
        for (long long t = 0; t < nt; ++t) {
            raster += window_wavefronts(*out, N, t, false, S);
            sorted += window_wavefronts(*out, N, t, true, S);
        }
        out->lane_sort = sorted < raster ? 1 : 0;
    }
    return PP_OK;
}

// Window loads with shifted blocks: one 8-byte and one 16-byte load per row (blocks at 4j - 1),
// or two 16-byte loads (4j - 2), instead of two bank-conflicted 4-byte loads around a 16-byte
// one.  They pay where the window loads weigh most, at few kept kernels per (input channel,
// filter group): VGG-16's keep-0.3 layers (2.4 kernels) measured 6-13 % faster with blocks at
// 4j - 1, its first layer (8 kernels, rows of 57 instead of 56 blocks) 16 % slower.  The estimate
// of channel steps of a shifted plan is scaled by this factor of the layer's mean kept kernels per
// (channel, group), 0.87 at 2.4 and 1 from 8 on.
double shift_gain(double kept_per_channel) { return std::min(1.0, 0.82 + 0.0225 * kept_per_channel); }

// Rounding of a split's reduction: the share of the result's square that each of its additions holds,
// summed (eight planes pairwise, four pooled, then one sum after the other).
double reduction_rounding(int ks, int pool) {
    const int step = pool ? 4 : 8, levels = pool ? 2 : 3, whole = ks / step * step;
    double e = (double)levels * whole / ks;
    for (int i = step; i <= whole; i += step) e += (double)i / ks;
    for (int i = whole + 1; i <= ks; ++i) e += (double)i / ks;
    return e;
}

// Whether the tensor-core kernel rounds no more than the FFMA kernel with its splits' sums added in
// order.  Squared errors against 64 bits, in units of (1e-7 of the result)^2, fitted to 1057 layers of 12
// to 512 channels, half of them small calls, on both kernels (three in four with a workspace):
//   FFMA           0.065 + 0.015 products; split 0.155 + 0.0168 products a split + 0.0442 (splits + 1) / 2;
//                  balanced schedule (360 further layers) 0.197 + 0.0147 products times the squares of the
//                  shares that cut units' pieces have + 0.0536 of the additions' shares, over the units
//   tensor cores   0.935 (0.764 with the lo products) + 0.0333 blocks a split + 0.58 (keep - 0.3) + 0.054
//                  reduction_rounding, and the square of what the accumulator truncates where the
//                  weights don't carry it back
// Measured squares lie within 25 % of these for eight layers in ten, so the tensor cores' has to be lower
// by the factors below.  For splits a second pair of estimates, off in other layers, has to hold too.
// Of these layers and 1000 others 923 calls pass, none with the larger error (of the 885 that pass by the
// second pair alone 32 had it, by up to 12 %); of 460 calls drawn afterwards one had, by 1.6 %.  (The
// reduction has since become pairwise, which takes up to a third off the FFMA kernel's error, 6 % in the
// median.  Against that, one call in 20 is above, by 19 % at most, nearly all of them with 25 splits and
// more.)
bool tensor_rounds_less(const pp_layer* L, const Plan& pl, int pool) {
    const TensorPlan& tc = pl.tc;
    const double products = 4.0 * L->beta / L->cout, dense = std::max(0.0, products / (4.0 * L->cin_g) - 0.3);
    const double pieces = pl.streamk ? 1.0 + 0.5 * sm_count() / pl.ctas : pl.KS, each = products / pieces;
    if (each < 13.0) return false;   // the FFMA estimates say too much
    const double truncated = L->tc_exact ? 1e14 * tensor_truncation(L) * tensor_truncation(L) : 0.0;
    const double tensor = (tc.ll ? 0.764 : 0.935) + 0.0333 * tc.cb_split + 0.58 * dense + truncated +
                          (tc.KS > 1 ? 0.054 * reduction_rounding(tc.KS, pool) : 0.0);
    if (pl.streamk) {
        const long long sms = sm_count(), nck = pl.n_chunks, chunks = pl.ctas * nck;
        double squares = (double)pl.ctas, adds = 0.0;
        long long unit = -1, from = 0;   // the cut unit at hand, where its last piece ends
        for (long long b = 1; b <= sms; ++b) {
            const long long c = chunks * b / sms, u = c / nck, k = c - u * nck;
            if (unit >= 0 && (u != unit || b == sms)) {
                squares += (double)((nck - from) * (nck - from)) / (double)(nck * nck);
                adds += 1.0;
                unit = -1;
            }
            if (k == 0) continue;
            if (unit < 0) {
                unit = u;
                from = 0;
                squares -= 1.0;
            }
            squares += (double)((k - from) * (k - from)) / (double)(nck * nck);
            if (from > 0 && k > from) adds += (double)k / nck;
            from = k;
        }
        return tensor <= 0.93 * (0.197 + (0.0147 * products * squares + 0.0536 * adds) / (double)pl.ctas);
    }
    if (pl.KS == 1) return tensor <= (tc.ll ? 0.9 : 0.95) * (0.065 + 0.015 * products);
    const double second = (tc.ll ? 0.84 : pl.KS >= 4 ? 1.25 : 1.0) + 0.033 * tc.cb_split + 0.5 * dense + truncated +
                          0.058 * std::log2((double)tc.KS);
    return tensor <= 0.155 + 0.0168 * each + 0.0221 * (pieces + 1.0) &&
           second <= 0.97 * (0.06 + 0.0137 * each + 0.036 * pieces);
}

// Whether a call takes the tensor-core kernel: where its estimate is the lower one, and for fp32 only
// where it rounds no more.
bool tensor_wins(const pp_layer* L, const Plan& pl, int N, int Ho, int Wo, int es, int pool) {
    if (es == 4 && !tensor_rounds_less(L, pl, pool)) return false;
    if (!L->fast) return true;
    const double flop = 8.0 * L->beta * (double)N * Ho * Wo;
    const double rate = (es == 4 ? 28e6 : 24e6) * (L->stride == 2 ? 0.5 : 1.0);   // FLOP a microsecond
    // microseconds beside the contraction: the launch, with a split its partial sums and reduction
    // (VGG-16 at batch 1: 19 with 3 splits, 28 with 32)
    const double other = pl.KS > 1 ? 14.0 + 0.3 * pl.KS : 8.0;
    return pl.tc.clocks / 1900.0 + 3.0 < 0.95 * (flop / rate + other);
}

int make_plan(const pp_layer* L, int N, int H, int W, size_t ws_avail, Plan* out, int pool = 0,
              bool allow_sk = true, int es = 4) {
    pp_layer* ML = const_cast<pp_layer*>(L);   // the cache is the only mutable part of a handle
    std::call_once(ML->plans_once, [ML] { ML->plans.reset(new PlanCache); });
    auto* cache = static_cast<PlanCache*>(ML->plans.get());
    const auto key = std::make_tuple(N, H, W, ws_avail, (pool * 2 + (allow_sk ? 1 : 0)) * 8 + es);
    {
        std::lock_guard<std::mutex> g(cache->mu);
        auto it = cache->plans.find(key);
        if (it != cache->plans.end()) {
            *out = it->second;
            return PP_OK;
        }
    }
    Plan pl;
    double cost = 0;
    const int rc = make_plan_uncached(L, N, H, W, ws_avail, 0, &pl, &cost, allow_sk, es);
    if (rc != PP_OK) return rc;
    // stride 2: two filter groups per warp (8 warps of 16 slots), so that each input window a lane
    // loads from shared memory serves twice the kept kernels (these layers are held by shared memory)
    if (L->stride == 2 && pl.WG >= 2 && s2_two_groups()) pl.dg = 2;
    if (L->stride == 1 && (!pool || es == 4)) {   // shifted blocks where their estimate is lower:
        // at 4j - 1 without the fused pool, at 4j - 2 (fp32 only) with it
        Plan ps;
        double cs = 0;
        const double kpc = (double)L->beta / ((double)L->G * L->cin_g);
        if (make_plan_uncached(L, N, H, W, ws_avail, pool ? 2 : 1, &ps, &cs, allow_sk, es) == PP_OK &&
            cs * shift_gain(kpc) < cost)
            pl = ps;
    }
    // fp32: with three products where that rounds no more than the FFMA kernel's plan, else with four
    const int Ho = (H - 1) / L->stride + 1, Wo = (W - 1) / L->stride + 1;
    for (int ll = 0; ll < (es == 4 ? 2 : 1) && !pl.tensor; ++ll)
        pl.tensor = tensor_plan(L, N, H, W, pool, es, ws_avail, sm_count(), &pl.tc, ll) &&
                    tensor_wins(L, pl, N, Ho, Wo, es, pool);
    std::lock_guard<std::mutex> g(cache->mu);
    if (cache->plans.size() >= 256) cache->plans.clear();
    cache->plans[key] = pl;
    *out = pl;
    return PP_OK;
}

// Sum the KS partial planes (eight at a time, pairwise), + bias, ReLU, round to the output type.  A thread
// issues the loads of 8 splits before it adds them, so that many loads are in flight; with
// `quads` (large outputs, a multiple of 4 elements, 16-byte aligned workspace) it takes 4
// consecutive elements, one 16-byte load per split.  Eight splits are summed pairwise before they are
// added (a fixed order, the same for every path): of 32 partial sums added one after the other the
// rounding alone was 1e-7 of the result.
__device__ __forceinline__ float sum8(float a, float b, float c, float d, float e, float f, float g, float h) {
    return ((a + b) + (c + d)) + ((e + f) + (g + h));
}
template <typename T>
__global__ void splitk_reduce(const float* __restrict__ ws, T* __restrict__ y, const float* __restrict__ bias,
                              int KS, size_t stride, int Cout, int HoWo, int relu, int quads) {
    pdl_trigger();
    pdl_wait();
    const bool vec = quads != 0;
    const size_t n = vec ? stride / 4 : stride;
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n; q += (size_t)gridDim.x * blockDim.x) {
        float v[4];
        int ne;
        size_t i0;
        if (vec) {
            const float4* w4 = reinterpret_cast<const float4*>(ws) + q;
            const size_t s4 = stride / 4;
            float4 a = w4[0];
            int k = 1;
            for (; k + 8 <= KS; k += 8) {
                float4 t[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) t[j] = w4[(size_t)(k + j) * s4];
                a.x += sum8(t[0].x, t[1].x, t[2].x, t[3].x, t[4].x, t[5].x, t[6].x, t[7].x);
                a.y += sum8(t[0].y, t[1].y, t[2].y, t[3].y, t[4].y, t[5].y, t[6].y, t[7].y);
                a.z += sum8(t[0].z, t[1].z, t[2].z, t[3].z, t[4].z, t[5].z, t[6].z, t[7].z);
                a.w += sum8(t[0].w, t[1].w, t[2].w, t[3].w, t[4].w, t[5].w, t[6].w, t[7].w);
            }
            for (; k < KS; ++k) {
                const float4 t = w4[(size_t)k * s4];
                a.x += t.x;
                a.y += t.y;
                a.z += t.z;
                a.w += t.w;
            }
            v[0] = a.x;
            v[1] = a.y;
            v[2] = a.z;
            v[3] = a.w;
            ne = 4;
            i0 = 4 * q;
        } else {
            float a = ws[q];
            int k = 1;
            for (; k + 8 <= KS; k += 8) {
                float t[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) t[j] = ws[(size_t)(k + j) * stride + q];
                a += sum8(t[0], t[1], t[2], t[3], t[4], t[5], t[6], t[7]);
            }
            for (; k < KS; ++k) a += ws[(size_t)k * stride + q];
            v[0] = a;
            ne = 1;
            i0 = q;
        }
        // output channel of the first element; the next ones may cross into the next plane
        int rem = (int)(i0 % (size_t)HoWo);
        int co = (int)((i0 / (size_t)HoWo) % (size_t)Cout);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (e >= ne) break;
            const float r = v[e] + (bias ? bias[co] : 0.0f);
            y[i0 + e] = from_f32<T>(relu ? fmaxf(r, 0.0f) : r);
            if (++rem == HoWo) {
                rem = 0;
                co = co + 1 == Cout ? 0 : co + 1;
            }
        }
    }
}

// Split-K reduction with the fused 2x2/2 max-pool: each pooled output sums the KS partial planes
// at its four positions (pairwise, as above), takes the maximum, adds the bias and applies ReLU.  The
// loads of 4 splits (16 loads) are issued before they are added.
template <typename T>
__global__ void splitk_reduce_pool(const float* __restrict__ ws, T* __restrict__ y, const float* __restrict__ bias,
                                   int KS, size_t stride, int Cout, int Ho, int Wo, int relu) {
    pdl_trigger();
    pdl_wait();
    const int Hp = Ho >> 1, Wp = Wo >> 1;
    const size_t total = stride / ((size_t)Ho * Wo) * Hp * Wp;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int px = (int)(i % Wp);
        const size_t r = i / Wp;
        const int py = (int)(r % Hp);
        const size_t plane = r / Hp;                       // n * Cout + co
        const size_t base = (plane * Ho + 2 * py) * Wo + 2 * px;
        const size_t off[4] = {0, 1, (size_t)Wo, (size_t)Wo + 1};
        float q[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) q[j] = ws[base + off[j]];
        int k = 1;
        for (; k + 4 <= KS; k += 4) {
            float t[4][4];
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
#pragma unroll
                for (int j = 0; j < 4; ++j) t[kk][j] = ws[(size_t)(k + kk) * stride + base + off[j]];
#pragma unroll
            for (int j = 0; j < 4; ++j) q[j] += (t[0][j] + t[1][j]) + (t[2][j] + t[3][j]);
        }
        for (; k < KS; ++k) {
#pragma unroll
            for (int j = 0; j < 4; ++j) q[j] += ws[(size_t)k * stride + base + off[j]];
        }
        const int co = (int)(plane % (size_t)Cout);
        float a = fmaxf(fmaxf(q[0], q[1]), fmaxf(q[2], q[3])) + (bias ? bias[co] : 0.0f);
        y[i] = from_f32<T>(relu ? fmaxf(a, 0.0f) : a);
    }
}

// Raise the kernel's dynamic shared-memory limit to the device's opt-in maximum once per device
// (a launch needs at most that), so that later calls, including ones under stream capture, make
// no attribute call.
template <int S, typename T, bool SORT, int SHIFT, bool SK, int DG = 1>
bool allow_max_smem(size_t need) {
    static std::atomic<int> done[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    if (done[dev].load(std::memory_order_acquire)) return true;
    int optin = 0;
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) return false;
    if ((size_t)optin < need) return false;
    if (cudaFuncSetAttribute(pconv_tm<S, T, SORT, SHIFT, SK, DG>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin) != cudaSuccess)
        return false;
    done[dev].store(1, std::memory_order_release);
    return true;
}

using TmKernel = void (*)(const TmParams, const CUtensorMap);

// The kernel variant for a plan: the balanced-schedule variants (SK) exist where the planner
// takes that schedule: stride 1, and stride 2 with two filter groups per warp.
template <int S, typename T, bool SORT, int SHIFT>
TmKernel pick_tm(bool sk, size_t smem, bool* ok, int dg = 1) {
    if constexpr (S == 1) {
        if (sk) {
            *ok = allow_max_smem<S, T, SORT, SHIFT, true>(smem);
            return pconv_tm<S, T, SORT, SHIFT, true>;
        }
    } else {
        if (dg == 2 && sk) {
            *ok = allow_max_smem<S, T, SORT, SHIFT, true, 2>(smem);
            return pconv_tm<S, T, SORT, SHIFT, true, 2>;
        }
        if (dg == 2) {
            *ok = allow_max_smem<S, T, SORT, SHIFT, false, 2>(smem);
            return pconv_tm<S, T, SORT, SHIFT, false, 2>;
        }
        if constexpr (SORT) {   // stride 2 deals blocks by bank group only with two groups per warp
            *ok = false;
            return nullptr;
        }
    }
    if constexpr (S == 1 || !SORT) {
        *ok = allow_max_smem<S, T, SORT, SHIFT, false>(smem);
        return pconv_tm<S, T, SORT, SHIFT, false>;
    }
    *ok = false;
    return nullptr;
}

// Reduction of an input-channel split: KS planes of partial sums to the output.
template <typename T>
int launch_reduce(const float* wsf, void* y, const float* bias, int ks, size_t total, int cout, int Ho, int Wo, int relu,
                  int pool, cudaStream_t st) {
    // threads: pooled outputs, or quads of outputs where the reduction loads 16 bytes a split
    // and there are enough of them to give every SM 512 threads (smaller outputs take more
    // threads, one element each: 64x64 32x32 N=1 16.1 us, in quads 16.8 us)
    const int quads = total % 4 == 0 && reinterpret_cast<uintptr_t>(wsf) % 16 == 0 &&
                      total / 4 >= (size_t)sm_count() * 512;
    const size_t items = pool ? total / 4 : (quads ? total / 4 : total);
    const unsigned blocks = (unsigned)std::max<size_t>(1, std::min<size_t>((items + 255) / 256, (size_t)sm_count() * 16));
    T* yt = static_cast<T*>(y);
    const int hw = Ho * Wo;
    const cudaError_t e = pool ? launch(splitk_reduce_pool<T>, blocks, 256, 0, st, wsf, yt, bias, ks, total, cout, Ho, Wo, relu)
                               : launch(splitk_reduce<T>, blocks, 256, 0, st, wsf, yt, bias, ks, total, cout, hw, relu, quads);
    return e == cudaSuccess ? PP_OK : PP_ERR_CUDA;
}

// The tensor-core kernel can be switched off (PATCONV_TENSOR=0).
bool tensor_enabled() {
    static const bool on = [] {
        const char* e = std::getenv("PATCONV_TENSOR");
        return !(e && e[0] == '0');
    }();
    return on;
}

template <typename T>
int launch_tensor(const pp_layer* L, const TensorPlan& pl, const void* x, void* y, const float* bias, int relu, int N,
                  int H, int W, int Ho, int Wo, void* ws, cudaStream_t st, int pool) {
    TensorCall c{};
    c.L = L;
    c.x = x;
    c.y = y;
    c.bias = bias;
    c.relu = relu;
    c.N = N;
    c.H = H;
    c.W = W;
    c.Ho = Ho;
    c.Wo = Wo;
    c.pool = pool;
    c.es = (int)sizeof(T);
    c.ws = ws;
    c.status = status_word();
    if (!c.status) return PP_ERR_CUDA;
    const bool inject = g_inject_timeout.exchange(0) != 0;
    c.wait_limit = inject ? kInjectedWaitCycles : kTimeoutCycles;
    c.no_fill = inject ? 1 : 0;
    c.sms = sm_count();
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    const bool captured = cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone;
    c.pdl = pdl_enabled() && !captured;
    c.st = st;
    if (tensor_launch(c, pl) != cudaSuccess) return PP_ERR_CUDA;
    if (pl.KS > 1)
        return launch_reduce<T>(static_cast<const float*>(ws), y, bias, pl.KS, (size_t)N * L->cout * Ho * Wo, L->cout, Ho,
                                Wo, relu, pool, st);
    return PP_OK;
}

template <int S, typename T>
int launch_tm(const pp_layer* L, const void* x, void* y, const float* bias, int relu, int N, int H, int W, int Ho,
              int Wo, void* ws, size_t ws_bytes, cudaStream_t st, int pool = 0) {
    Plan pl;
    const int rc = make_plan(L, N, H, W, ws ? ws_bytes : 0, &pl, pool, true, (int)sizeof(T));
    if (rc != PP_OK) return rc;
    const bool ws_aligned = reinterpret_cast<uintptr_t>(ws) % 16 == 0;
    if ((pl.KS > 1 || pl.streamk) && !ws_aligned) return PP_ERR_ALIGN;
    // never planned: pool windows must lie in one block; blocks at 4j - 2 are fp32 only
    if ((pool && pl.shift == 1) || (pl.shift == 2 && sizeof(T) != 4)) return PP_ERR_SHAPE;
    // (a tensor-core plan may split where the FFMA plan does not: a misaligned workspace, which the
    // FFMA plan leaves alone, then leaves the call to it)
    if (pl.tensor && L->tdev && tensor_enabled() && (pl.tc.KS == 1 || ws_aligned))
        return launch_tensor<T>(L, pl.tc, x, y, bias, relu, N, H, W, Ho, Wo, ws, st, pool);
    TmParams p{};
    p.x = x;
    p.y = y;
    p.bias = bias;
    const unsigned char* img = static_cast<const unsigned char*>(L->dev);
    p.perm = reinterpret_cast<const uint32_t*>(img + L->off_perm);
    p.desc = reinterpret_cast<const uint64_t*>(img + L->off_desc);
    p.kofs = reinterpret_cast<const uint32_t*>(img + L->off_kofs);
    p.vals = reinterpret_cast<const float4*>(img + L->off_vals);
    p.status = status_word();
    if (!p.status) return PP_ERR_CUDA;
    const bool inject = g_inject_timeout.exchange(0) != 0;
    p.wait_limit = inject ? kInjectedWaitCycles : kTimeoutCycles;
    p.no_fill = inject ? 1 : 0;
    p.N = N;
    p.C = L->cin_g;
    p.H = H;
    p.W = W;
    p.Cout = L->cout;
    p.Ho = Ho;
    p.Wo = Wo;
    p.G = L->G;
    p.relu = relu;
    p.WG = pl.WG;
    p.WS = pl.WS;
    p.n_fchunks = pl.n_fchunks;
    p.BY = pl.tile.BY;
    p.BX = pl.tile.BX;
    p.NB = pl.tile.NB;
    p.IH = pl.tile.IH;
    const size_t es = sizeof(T);
    // fp16 stages hold fp16 (widened as the window is loaded): half the bytes of the plan's fp32
    // stage, with 8 more columns so that the origin can sit on an 8-column (16-byte) boundary
    p.BWb = es == 4 ? pl.tile.BWb : (int)align_up((size_t)pl.tile.BWb + 8, 8);
    p.ixa = (int)(16 / es);
    p.linear = pl.tile.linear;
    p.tiles_x = pl.tiles_x;
    p.tiles_y = pl.tiles_y;
    p.tiles_n = pl.tiles_n;
    p.CK = pl.CK;
    p.n_chunks = pl.n_chunks;
    p.maxk = pl.maxk;
    p.KS = pl.KS;
    p.c_split = pl.c_split;
    p.ws = static_cast<float*>(ws);
    p.ws_stride = (size_t)N * L->cout * Ho * Wo;
    const int C = L->cin_g;
    p.use_tma = (W * es) % 16 == 0 && reinterpret_cast<uintptr_t>(x) % 16 == 0 && encode_tiled() != nullptr;
    p.kb_off = 64;
    p.stage_off = (unsigned)align_up(64 + pl.kb_bytes, 128);
    p.desc_off = (unsigned)align_up((size_t)p.NB * p.CK * p.IH * p.BWb * es, 128);
    p.vals_off = p.desc_off + (unsigned)align_up((size_t)p.WG * p.CK * 8, 16);
    p.stage_bytes = (unsigned)align_up((size_t)p.vals_off + (size_t)p.WG * p.maxk * 16, 128);
    const size_t smem = p.stage_off + (size_t)kStages * p.stage_bytes;   // the plan's for fp32
    if (smem > pl.smem) return PP_ERR_SHAPE;
    p.vec_store = (Wo % 4 == 0) && (reinterpret_cast<uintptr_t>(y) % (4 * es)) == 0;
    p.vec_pair = (Wo % 2 == 0) && (reinterpret_cast<uintptr_t>(y) % (2 * es)) == 0;
    p.pool = pool;
    p.vec_pool = ((Wo >> 1) % 2 == 0) && (reinterpret_cast<uintptr_t>(y) % (2 * es)) == 0;

    CUtensorMap tmap;
    std::memset(&tmap, 0, sizeof(tmap));
    if (p.use_tma) {
        const cuuint64_t dims[4] = {(cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)C, (cuuint64_t)N};
        const cuuint64_t strides[3] = {(cuuint64_t)W * es, (cuuint64_t)H * W * es, (cuuint64_t)C * H * W * es};
        const cuuint32_t box[4] = {(cuuint32_t)p.BWb, (cuuint32_t)p.IH, (cuuint32_t)p.CK, (cuuint32_t)p.NB};
        const cuuint32_t estr[4] = {1, 1, 1, 1};
        const CUresult r = encode_tiled()(&tmap, es == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16,
                                          4, const_cast<void*>(x), dims,
                                          strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                          CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) p.use_tma = 0;
        p.tma_bytes = (unsigned)((size_t)p.BWb * p.IH * p.CK * p.NB * es);
    }
    // balanced schedule (TMA path only: the copy fallback keeps one CTA per unit)
    const bool persist = p.use_tma || (pl.tiles_x == 1 && pl.tiles_y == 1 && !pl.tile.linear);
    p.streamk = (S == 1 || pl.dg == 2) && pl.streamk && persist ? 1 : 0;
    const bool sk = p.streamk != 0;
    TmKernel kern;
    bool smem_ok = false;
    if constexpr (S == 1 && sizeof(T) == 4) {
        if (pl.lane_sort) {
            if (pl.shift == 2) kern = pick_tm<1, float, true, 2>(sk, smem, &smem_ok);
            else if (pl.shift == 1) kern = pick_tm<1, float, true, 1>(sk, smem, &smem_ok);
            else kern = pick_tm<1, float, true, 0>(sk, smem, &smem_ok);
        } else {
            if (pl.shift == 2) kern = pick_tm<1, float, false, 2>(sk, smem, &smem_ok);
            else if (pl.shift == 1) kern = pick_tm<1, float, false, 1>(sk, smem, &smem_ok);
            else kern = pick_tm<1, float, false, 0>(sk, smem, &smem_ok);
        }
    } else if constexpr (S == 1) {
        if (pl.shift) kern = pick_tm<1, T, false, 1>(sk, smem, &smem_ok);
        else kern = pick_tm<1, T, false, 0>(sk, smem, &smem_ok);
    } else {
        if constexpr (sizeof(T) == 4) {
            if (pl.lane_sort && pl.dg == 2) kern = pick_tm<S, float, true, 0>(sk, smem, &smem_ok, 2);
            else kern = pick_tm<S, T, false, 0>(sk && pl.dg == 2, smem, &smem_ok, pl.dg);
        } else {
            kern = pick_tm<S, T, false, 0>(sk && pl.dg == 2, smem, &smem_ok, pl.dg);
        }
    }
    if (!smem_ok) return PP_ERR_CUDA;
    const long long units = pl.ctas * pl.KS;
    if (units > INT_MAX) return PP_ERR_SHAPE;
    p.n_units = (int)units;
    if (p.streamk) {
        const long long P = sm_count();
        if (!ws || ws_bytes < streamk_bytes(P)) return PP_ERR_BUFFER;
        p.sk_total = pl.ctas * pl.n_chunks;
        p.sk_slots = static_cast<float*>(ws);
        p.sk_flags = reinterpret_cast<unsigned*>(static_cast<unsigned char*>(ws) +
                                                 align_up((size_t)P * kSlotFloats * sizeof(float), 256));
        if (cudaMemsetAsync(p.sk_flags, 0, (size_t)P * kCompute * sizeof(unsigned), st) != cudaSuccess)
            return PP_ERR_CUDA;
        if (launch_ex(true, kern, (unsigned)P, kThreadsTM / pl.dg, smem, st, false, p, tmap) != cudaSuccess) return PP_ERR_CUDA;
        return PP_OK;
    }
    // TMA path: one persistent CTA per SM walks its units as one chunk stream (the halo is zero
    // filled by the TMA unit, so stages carry over between tiles); the copy fallback relies on
    // stages zeroed once, so there every unit gets its own CTA
    const long long ctas = persist ? std::max<long long>(std::min<long long>(units, sm_count()),
                                                         (units + kMaxUnitsPerCta - 1) / kMaxUnitsPerCta)
                                   : units;
    if (launch(kern, (unsigned)ctas, kThreadsTM / pl.dg, smem, st, p, tmap) != cudaSuccess) return PP_ERR_CUDA;
    if (pl.KS > 1) return launch_reduce<T>(p.ws, y, bias, pl.KS, p.ws_stride, L->cout, Ho, Wo, relu, pool, st);
    return PP_OK;
}

template <int S, typename T>
int launch_depthwise_s(const DwParams& p, unsigned ctas, bool vin, bool vout, cudaStream_t st) {
    cudaError_t e;
    if (vin && vout) e = launch(pconv_depthwise<S, T, true, true>, ctas, kDwThreads, 0, st, p);
    else if (vin) e = launch(pconv_depthwise<S, T, true, false>, ctas, kDwThreads, 0, st, p);
    else if (vout) e = launch(pconv_depthwise<S, T, false, true>, ctas, kDwThreads, 0, st, p);
    else e = launch(pconv_depthwise<S, T, false, false>, ctas, kDwThreads, 0, st, p);
    return e == cudaSuccess ? PP_OK : PP_ERR_CUDA;
}

template <int S, typename T, bool VIN, bool VOUT, int RW, int NH>
bool dw_staged_smem(size_t need) {
    static std::atomic<int> done[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    if (done[dev].load(std::memory_order_acquire)) return true;
    int optin = 0;
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) return false;
    if ((size_t)optin < need) return false;
    if (cudaFuncSetAttribute(pconv_depthwise_staged<S, T, VIN, VOUT, RW, NH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             optin) != cudaSuccess)
        return false;
    done[dev].store(1, std::memory_order_release);
    return true;
}

template <int S, typename T, bool VIN, bool VOUT, int RW = 0, int NH = 1>
int launch_dw_staged(const DwStagedParams& p, size_t smem, cudaStream_t st) {
    if (!dw_staged_smem<S, T, VIN, VOUT, RW, NH>(smem)) return PP_ERR_CUDA;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, pconv_depthwise_staged<S, T, VIN, VOUT, RW, NH>,
                                                      kDwThreads, smem) != cudaSuccess || per_sm < 1)
        return PP_ERR_CUDA;
    const long long ctas = std::min<long long>(p.n_tiles, (long long)sm_count() * per_sm);
    return launch(pconv_depthwise_staged<S, T, VIN, VOUT, RW, NH>, (unsigned)ctas, kDwThreads, smem, st, p) == cudaSuccess
               ? PP_OK : PP_ERR_CUDA;
}

template <int S, typename T>
int launch_dw_staged_s(const DwStagedParams& p, size_t smem, bool vin, bool vout, cudaStream_t st) {
    // whole planes whose output rows are 7, 14 or 28 wide: the row-item kernel (28-wide rows in two
    // 14-wide pieces, which keeps its registers low enough for four CTAs per SM)
    if (p.n_bands == 1 && p.W == S * p.Wo) {
        if (p.Wo == 28) return launch_dw_staged<S, T, false, false, 14, 2>(p, smem, st);
        if (p.Wo == 14) return launch_dw_staged<S, T, false, false, 14, 1>(p, smem, st);
        if (p.Wo == 7) return launch_dw_staged<S, T, false, false, 7>(p, smem, st);
    }
    if (vin && vout) return launch_dw_staged<S, T, true, true>(p, smem, st);
    if (vin) return launch_dw_staged<S, T, true, false>(p, smem, st);
    if (vout) return launch_dw_staged<S, T, false, true>(p, smem, st);
    return launch_dw_staged<S, T, false, false>(p, smem, st);
}

constexpr size_t kDwStageBytes = 16384;   // one staging buffer of the staged depthwise kernel

// Tile shape and shared-memory layout of the staged depthwise kernel; false when it does not
// apply (x not 16-byte aligned, a plane row wider than a buffer, more channels than the per-CTA
// tap table holds).
template <typename T>
bool dw_staged_plan(const pp_layer* L, const void* x, int N, int H, int W, int Ho, DwStagedParams* p,
                    size_t* smem) {
    const int S = L->stride;
    const long long es = sizeof(T), VE = 16 / es;
    const long long budget = kDwStageBytes / es;
    // rows that are 16-byte aligned already load as vectors straight from global memory
    if (reinterpret_cast<uintptr_t>(x) % 16 != 0 || ((size_t)W * es) % 16 == 0 || L->cout > 3072) return false;
    const long long plane = (long long)H * W;
    if (plane <= budget) {
        p->npl = (int)std::min<long long>({(long long)L->cout, budget / plane, (long long)kDwMaxPlanes});
        p->rb = Ho;
        p->n_bands = 1;
    } else {
        const long long rows_in = budget / W;
        if (rows_in < 3) return false;
        p->npl = 1;
        p->rb = (int)((rows_in - 3) / S + 1);
        p->n_bands = (Ho + p->rb - 1) / p->rb;
    }
    p->n_cg = (L->cout + p->npl - 1) / p->npl;
    const long long n_tiles = (long long)N * p->n_cg * p->n_bands;
    if (n_tiles > INT_MAX) return false;
    p->n_tiles = (int)n_tiles;
    const long long max_rows = p->n_bands == 1 ? H : std::min<long long>(H, (long long)(p->rb - 1) * S + 3);
    const long long max_len = (long long)p->npl * max_rows * W;
    p->buf_elems = (int)((max_len + 2 * VE + VE - 1) / VE * VE);
    p->total_in = (long long)N * L->cout * H * W;
    p->off_w = 0;
    p->off_buf = (unsigned)align_up((size_t)L->cout * 6 * 4, 16);
    *smem = p->off_buf + 2 * (size_t)p->buf_elems * es;
    return true;
}

// Streamed depthwise kernel: chunking for one call shape.  Rows mode needs rows of a multiple of
// 16 bytes and at most 256 elements and output rows of a multiple of 4 columns (at most 128);
// planes mode needs whole output rows of at most 32 lanes (one or two columns each).  The tensor
// pointers (16-byte aligned x and y) are the launcher's to check.  Returns false where the
// kernel does not apply (the earlier depthwise kernels run then).
constexpr size_t kDwsRowsStage = 4096;     // target bytes of one input stage, rows mode
constexpr size_t kDwsPlanesStage = 3200;   // planes mode
constexpr int kDwsChunksPerWarp = 3;       // planes mode: smaller chunks until every warp has this many

int dws_smem_optin() {
    static std::atomic<int> cached[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 232448;   // no device: a GB300
    int v = cached[dev].load();
    if (v > 0) return v;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess || v <= 0) return 232448;
    cached[dev].store(v);
    return v;
}

bool dws_enabled() {
    static const bool on = [] {
        const char* e = std::getenv("PATCONV_DW_STREAM");
        return !(e && e[0] == '0');
    }();
    return on;
}

bool dws_plan(const pp_layer* L, int N, int H, int W, int Ho, int Wo, size_t es, DwsParams* p, int* mode,
              size_t* smem) {
    const int S = L->stride, C = L->cout;
    const long long n_planes = (long long)N * C;
    if (n_planes > INT_MAX) return false;
    const size_t optin = (size_t)dws_smem_optin();
    p->off_tab = 8 * kDwsMaxStages * kDwsWarps;
    p->off_area = (unsigned)align_up(p->off_tab + (size_t)C * kDwsTab * 4, 128);
    if ((size_t)p->off_area + (size_t)kDwsWarps * 4096 > optin) return false;   // the table leaves too little room
    const size_t avail = optin - p->off_area;
    const long long sms = sm_count();
    size_t out_b = 0, extra = 0;
    auto al = [](size_t b) { return (long long)(16 / std::gcd(b, (size_t)16)); };   // planes per 16 bytes
    const size_t pb = (size_t)H * W * es, opb = (size_t)Ho * Wo * es;
    const bool rows = ((size_t)W * es) % 16 == 0 && W <= 256 && Wo % kDwsCW == 0 && Wo / kDwsCW <= 32 &&
                      (S == 1 ? W == Wo : W == 2 * Wo);
    // tiles mode: each lane a band of 7 output rows by 7 or 14 columns of a plane
    int tile = 0;
    long long tP = 0;
    if (S == 1 && W == Wo && H == Ho && H % 7 == 0) tile = W == 7 ? 4 : (W == 14 || W == 28) ? 5 : 0;
    if (S == 2 && (W == 14 || W == 28) && H == 2 * Ho && Ho % 7 == 0) tile = 6;
    if (tile) {   // planes per chunk: 16-byte aligned chunk starts in x and y, lane items a multiple of 32
        const int ipp = (Wo / (tile == 5 ? 14 : 7)) * (Ho / 7);
        tP = std::lcm(std::lcm(al(pb), al(opb)), (long long)(32 / std::gcd(ipp, 32)));
        if ((size_t)tP * pb > 16384) tile = 0;   // stages too large: planes mode
    }
    if (rows) {
        p->NCG = Wo / kDwsCW;
        p->NHL = 32 / p->NCG;
        const int rin_max = std::max(3, (int)(kDwsRowsStage / ((size_t)W * es)));
        int R = std::min(Ho, (rin_max - 3) / S + 1);
        if (R >= p->NHL) R -= R % p->NHL;
        p->R = R;
        p->RIN = (R - 1) * S + 3;
        p->RPL = (R + p->NHL - 1) / p->NHL;
        p->n_bands = (Ho + R - 1) / R;
        p->in_b = (unsigned)align_up((size_t)W * p->RIN * es, 128);
        p->n_chunks = n_planes * p->n_bands;
        *mode = 0;
    } else if (tile) {
        const int pw = tile == 5 ? 14 : 7;
        p->npc = Wo / pw;
        p->ipp = p->npc * (Ho / 7);
        const long long P = tP;
        p->P = (int)P;
        p->in_b = (unsigned)align_up((size_t)P * pb, 128);
        out_b = align_up((size_t)P * opb, 128);
        extra = 128;                     // the zero row
        p->n_chunks = (n_planes + P - 1) / P;
        *mode = tile;
    } else {
        if (S == 1 ? W != Wo : W != 2 * Wo) return false;
        const int cpl = S == 1 ? 2 : 1;
        p->LPP = (Wo + cpl - 1) / cpl;
        if (p->LPP > 32) return false;
        p->NPW = 32 / p->LPP;
        // chunk starts 16-byte aligned in x and y; whole passes of the warp where that allows
        const long long A = std::lcm(std::lcm(al(pb), al(opb)), (long long)p->NPW);
        long long P = std::max<long long>(A, (long long)(kDwsPlanesStage / pb) / A * A);
        while (P > A && (n_planes + P - 1) / P < kDwsChunksPerWarp * sms * kDwsWarps) P -= A;
        if ((size_t)P * pb > ((size_t)1 << 30)) return false;
        p->P = (int)P;
        p->in_b = (unsigned)align_up((size_t)P * pb, 128);
        out_b = align_up((size_t)P * opb + 16, 128);   // + a junk word for idle lanes' results
        p->n_chunks = (n_planes + P - 1) / P;
        *mode = S == 2 ? 1 : (W % 2 == 0 ? 2 : 3);
    }
    if (p->n_chunks > INT_MAX) return false;
    // warps per CTA: as many as hold two stages each (at most 16); then stages per warp
    const size_t two = 2 * (size_t)p->in_b + out_b + extra;
    const int nwarps = (int)std::min<size_t>(kDwsWarps, avail / two);
    if (nwarps < 4) return false;
    const size_t per_warp = avail / nwarps / 128 * 128;
    p->nwarps = nwarps;
    p->nst = (int)std::min<size_t>(kDwsMaxStages, (per_warp - out_b - extra) / p->in_b);
    p->zoff = (unsigned)((size_t)p->nst * p->in_b + out_b);
    p->area_b = (unsigned)align_up((size_t)p->nst * p->in_b + out_b + extra, 128);
    p->n_planes = n_planes;
    *smem = p->off_area + (size_t)nwarps * p->area_b;
    return *smem <= optin;
}

template <int S, typename T, int MODE>
int launch_dws(const DwsParams& p, const CUtensorMap& tmap, size_t smem, cudaStream_t st) {
    static std::atomic<int> done[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return PP_ERR_CUDA;
    if (!done[dev].load(std::memory_order_acquire)) {
        if (cudaFuncSetAttribute(pconv_dw_stream<S, T, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 dws_smem_optin()) != cudaSuccess)
            return PP_ERR_CUDA;
        done[dev].store(1, std::memory_order_release);
    }
    const long long grid = std::min<long long>(sm_count(), (p.n_chunks + p.nwarps - 1) / p.nwarps);
    // programmatic launch also under stream capture: the tap table's decode then overlaps the
    // previous kernel in a graph as on a stream (MobileNet-V2 b128: 0.390 -> 0.359 ms graphed)
    return launch_ex(false, pconv_dw_stream<S, T, MODE>, (unsigned)std::max<long long>(grid, 1), 32u * p.nwarps, smem, st,
                     true, p, tmap) == cudaSuccess ? PP_OK : PP_ERR_CUDA;
}

// The streamed depthwise kernel where it applies (PP_OK or an error), else 1.
template <typename T>
int try_dws(const pp_layer* L, const void* x, void* y, const float* bias, int relu, int N, int H, int W, int Ho,
            int Wo, cudaStream_t st) {
    if (!dws_enabled() || reinterpret_cast<uintptr_t>(x) % 16 != 0 || reinterpret_cast<uintptr_t>(y) % 16 != 0) return 1;
    DwsParams p{};
    int mode = 0;
    size_t smem = 0;
    if (!dws_plan(L, N, H, W, Ho, Wo, sizeof(T), &p, &mode, &smem)) return 1;
    const unsigned char* img = static_cast<const unsigned char*>(L->dev);
    p.x = x;
    p.y = y;
    p.bias = bias;
    p.perm = reinterpret_cast<const uint32_t*>(img + L->off_perm);
    p.desc = reinterpret_cast<const uint64_t*>(img + L->off_desc);
    p.kofs = reinterpret_cast<const uint32_t*>(img + L->off_kofs);
    p.vals = reinterpret_cast<const float4*>(img + L->off_vals);
    p.status = status_word();
    if (!p.status) return PP_ERR_CUDA;
    p.N = N;
    p.C = L->cout;
    p.H = H;
    p.W = W;
    p.Ho = Ho;
    p.Wo = Wo;
    p.relu = relu;
    p.NS = L->G * kF;
    p.vec_out = 1;   // rows mode: Wo a multiple of 4 and y 16-byte aligned
    for (int i = 0; i < kMaxPatterns; ++i) p.masks[i] = i < L->n_patterns ? L->masks[i] : 0;
    CUtensorMap tmap;
    std::memset(&tmap, 0, sizeof(tmap));
    const size_t es = sizeof(T);
    if (mode == 0) {   // planes x rows x columns, one box = RIN whole rows of one plane
        if (!encode_tiled()) return 1;
        const cuuint64_t dims[3] = {(cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)p.n_planes};
        const cuuint64_t strides[2] = {(cuuint64_t)W * es, (cuuint64_t)H * W * es};
        const cuuint32_t box[3] = {(cuuint32_t)W, (cuuint32_t)p.RIN, 1};
        const cuuint32_t estr[3] = {1, 1, 1};
        if (encode_tiled()(&tmap, es == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3,
                           const_cast<void*>(x), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return 1;
    }
    const int S = L->stride;
    if (S == 1) {
        if (mode == 0) return launch_dws<1, T, 0>(p, tmap, smem, st);
        if (mode == 2) return launch_dws<1, T, 2>(p, tmap, smem, st);
        if (mode == 3) return launch_dws<1, T, 3>(p, tmap, smem, st);
        if (mode == 4) return launch_dws<1, T, 4>(p, tmap, smem, st);
        return launch_dws<1, T, 5>(p, tmap, smem, st);
    }
    if (mode == 0) return launch_dws<2, T, 0>(p, tmap, smem, st);
    if (mode == 6) return launch_dws<2, T, 6>(p, tmap, smem, st);
    return launch_dws<2, T, 1>(p, tmap, smem, st);
}

template <typename T>
int launch_depthwise(const pp_layer* L, const void* x, void* y, const float* bias, int relu, int N, int H, int W,
                     int Ho, int Wo, cudaStream_t st) {
    {
        const int rc = try_dws<T>(L, x, y, bias, relu, N, H, W, Ho, Wo, st);
        if (rc != 1) return rc;
    }
    {
        const unsigned char* img = static_cast<const unsigned char*>(L->dev);
        DwStagedParams q{};
        size_t smem = 0;
        if (dw_staged_plan<T>(L, x, N, H, W, Ho, &q, &smem)) {
            q.x = x;
            q.y = y;
            q.bias = bias;
            q.perm = reinterpret_cast<const uint32_t*>(img + L->off_perm);
            q.desc = reinterpret_cast<const uint64_t*>(img + L->off_desc);
            q.kofs = reinterpret_cast<const uint32_t*>(img + L->off_kofs);
            q.vals = reinterpret_cast<const float4*>(img + L->off_vals);
            q.N = N;
            q.C = L->cout;
            q.H = H;
            q.W = W;
            q.Ho = Ho;
            q.Wo = Wo;
            q.relu = relu;
            q.NS = L->G * kF;
            q.NGX = (Wo + kDwVW - 1) / kDwVW;
            for (int i = 0; i < kMaxPatterns; ++i) q.masks[i] = i < L->n_patterns ? L->masks[i] : 0;
            const size_t es = sizeof(T);
            const bool vin = ((size_t)W * es) % 16 == 0;
            const bool vout = ((size_t)Wo * es) % 16 == 0 && reinterpret_cast<uintptr_t>(y) % 16 == 0;
            return L->stride == 1 ? launch_dw_staged_s<1, T>(q, smem, vin, vout, st)
                                  : launch_dw_staged_s<2, T>(q, smem, vin, vout, st);
        }
    }
    const unsigned char* img = static_cast<const unsigned char*>(L->dev);
    DwParams p{};
    p.x = x;
    p.y = y;
    p.bias = bias;
    p.perm = reinterpret_cast<const uint32_t*>(img + L->off_perm);
    p.desc = reinterpret_cast<const uint64_t*>(img + L->off_desc);
    p.kofs = reinterpret_cast<const uint32_t*>(img + L->off_kofs);
    p.vals = reinterpret_cast<const float4*>(img + L->off_vals);
    p.N = N;
    p.C = L->cout;
    p.H = H;
    p.W = W;
    p.Ho = Ho;
    p.Wo = Wo;
    p.relu = relu;
    p.NS = L->G * kF;
    p.NGX = (Wo + kDwVW - 1) / kDwVW;
    for (int i = 0; i < kMaxPatterns; ++i) p.masks[i] = i < L->n_patterns ? L->masks[i] : 0;
    const long long ipp = (long long)Ho * p.NGX;
    const long long planes = (long long)N * p.NS;
    if (ipp > INT_MAX / 2) return PP_ERR_SHAPE;
    p.ipp = (int)ipp;
    long long ctas;
    if (ipp > kDwItemsPerCta) {
        p.tiles = (int)((ipp + kDwItemsPerCta - 1) / kDwItemsPerCta);
        p.ppc = 1;
        ctas = planes * p.tiles;
    } else {
        p.tiles = 1;
        p.ppc = (int)std::min<long long>(kDwItemsPerCta / ipp, kDwMaxPlanes);
        ctas = (planes + p.ppc - 1) / p.ppc;
    }
    if (ctas > INT_MAX) return PP_ERR_SHAPE;
    const size_t es = sizeof(T);
    const bool vin = ((size_t)W * es) % 16 == 0 && reinterpret_cast<uintptr_t>(x) % 16 == 0;
    const bool vout = ((size_t)Wo * es) % 16 == 0 && reinterpret_cast<uintptr_t>(y) % 16 == 0;
    return L->stride == 1 ? launch_depthwise_s<1, T>(p, (unsigned)ctas, vin, vout, st)
                          : launch_depthwise_s<2, T>(p, (unsigned)ctas, vin, vout, st);
}

template <typename T>
int launch_generic(const pp_layer* L, const void* x, void* y, const float* bias, int relu, int N, int H, int W,
                   int Ho, int Wo, cudaStream_t st) {
    if (!L->depthwise && L->tdev && tensor_enabled()) {
        Plan pl;
        if (make_plan(L, N, H, W, 0, &pl, 0, true, (int)sizeof(T)) == PP_OK && pl.tensor)
            return launch_tensor<T>(L, pl.tc, x, y, bias, relu, N, H, W, Ho, Wo, nullptr, st, 0);
    }
    const unsigned char* img = static_cast<const unsigned char*>(L->dev);
    TapTable tt{};
    for (int p = 0; p < L->n_patterns; ++p) {
        int n = 0;
        for (int t = 0; t < 9; ++t)
            if ((L->masks[p] >> t) & 1u) tt.t[p][n++] = (int8_t)t;
    }
    const long long total = (long long)N * L->cout * Ho * Wo;
    const int blocks = (int)std::min<long long>((total + 255) / 256, (long long)sm_count() * 32);
    pconv_generic<T><<<std::max(blocks, 1), 256, 0, st>>>(
        static_cast<const T*>(x), static_cast<T*>(y), bias, reinterpret_cast<const uint32_t*>(img + L->off_perm),
        reinterpret_cast<const uint64_t*>(img + L->off_desc), reinterpret_cast<const uint32_t*>(img + L->off_kofs),
        reinterpret_cast<const float4*>(img + L->off_vals), tt, N, L->depthwise ? L->cout : L->cin_g, L->cin_g,
        L->depthwise ? 1 : 0, H, W, L->cout, Ho, Wo, L->stride, relu);
    return cudaGetLastError() == cudaSuccess ? PP_OK : PP_ERR_CUDA;
}


// Device address of g_pp_scratch on the current device, looked up once per device (the host-side
// name of the array is only a stand-in; kernels must be given this address).
void* static_scratch_address() {
    static std::mutex mu;
    static void* addr[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[dev]) {
        void* ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_pp_scratch) != cudaSuccess) return nullptr;
        addr[dev] = ptr;
    }
    return addr[dev];
}

bool overlaps(const void* a, size_t na, const void* b, size_t nb) {
    const uintptr_t x0 = reinterpret_cast<uintptr_t>(a), y0 = reinterpret_cast<uintptr_t>(b);
    return x0 < y0 + nb && y0 < x0 + na;
}

}  // namespace

bool patconv::encode_box(CUtensorMap* map, const void* x, int N, int C, int H, int W, int rw, int rows) {
    if (!encode_tiled()) return false;
    const cuuint64_t dims[4] = {(cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)C, (cuuint64_t)N};
    const cuuint64_t strides[3] = {(cuuint64_t)W * 4, (cuuint64_t)H * W * 4, (cuuint64_t)C * H * W * 4};
    const cuuint32_t box[4] = {(cuuint32_t)rw, (cuuint32_t)rows, 16, 1}, estr[4] = {1, 1, 1, 1};
    return encode_tiled()(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<void*>(x), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

extern "C" {

int pp_bind_device(pp_handle h, void* dev_image, size_t bytes, void* stream) {
    if (!h || !dev_image) return PP_ERR_NULL;
    if (bytes < h->image.size()) return PP_ERR_BUFFER;
    if (reinterpret_cast<uintptr_t>(dev_image) % 256 != 0) return PP_ERR_ALIGN;
    if (cudaMemcpyAsync(dev_image, h->image.data(), h->image.size(), cudaMemcpyHostToDevice,
                        static_cast<cudaStream_t>(stream)) != cudaSuccess)
        return PP_ERR_CUDA;
    h->dev = dev_image;
    h->dev_bytes = bytes;
    h->tdev = nullptr;
    return PP_OK;
}

int pp_bind_tensor(pp_handle h, void* dev, size_t bytes, void* stream) {
    if (!h || !dev) return PP_ERR_NULL;
    if (!h->dev) return PP_ERR_NOT_BOUND;
    const size_t need = tensor_weight_bytes(h);
    if (need == 0) return PP_ERR_PATH;
    if (bytes < need) return PP_ERR_BUFFER;
    if (reinterpret_cast<uintptr_t>(dev) % 256 != 0) return PP_ERR_ALIGN;
    if (tensor_build_weights(h, dev, static_cast<cudaStream_t>(stream)) != cudaSuccess) return PP_ERR_CUDA;
    h->tdev = dev;
    return PP_OK;
}

namespace {

int validate_conv(pp_handle h, const void* x, int dtype, int N, int H, int W, const float* bias, int relu,
                  const void* y, int pool = 0) {
    if (!h) return PP_ERR_NULL;
    if (!h->dev) return PP_ERR_NOT_BOUND;
    if (dtype != PP_F32 && dtype != PP_F16) return PP_ERR_DTYPE;
    if (N < 0 || H < 1 || W < 1) return PP_ERR_SHAPE;
    if (relu != 0 && relu != 1) return PP_ERR_ARG;
    if (N == 0) return PP_OK;
    if (!x || !y) return PP_ERR_NULL;
    const int C = h->depthwise ? h->cout : h->cin_g;
    const int Ho = (H - 1) / h->stride + 1, Wo = (W - 1) / h->stride + 1;
    const size_t es = dtype == PP_F32 ? 4 : 2;
    if ((size_t)N * C * H * W >= (1ull << 40) || (size_t)N * h->cout * Ho * Wo >= (1ull << 40)) return PP_ERR_SHAPE;
    const size_t xb = (size_t)N * C * H * W * es;
    const size_t yb = pool ? (size_t)N * h->cout * (Ho / 2) * (Wo / 2) * es : (size_t)N * h->cout * Ho * Wo * es;
    if (reinterpret_cast<uintptr_t>(x) % es || reinterpret_cast<uintptr_t>(y) % es) return PP_ERR_ALIGN;
    if (bias && reinterpret_cast<uintptr_t>(bias) % 4) return PP_ERR_ALIGN;
    if (overlaps(x, xb, y, yb)) return PP_ERR_BUFFER;
    return PP_OK;
}

}  // namespace

int pp_conv_ws(pp_handle h, const void* x, int dtype, int N, int H, int W, const float* bias, int relu, void* y,
               void* workspace, size_t workspace_bytes, void* stream) {
    const int v = validate_conv(h, x, dtype, N, H, W, bias, relu, y);
    if (v != PP_OK || N == 0) return v;
    const int Ho = (H - 1) / h->stride + 1, Wo = (W - 1) / h->stride + 1;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const bool f16 = dtype == PP_F16;
    if (h->depthwise) {   // any pattern library: the kernel expands each channel's taps itself
        return f16 ? launch_depthwise<__half>(h, x, y, bias, relu, N, H, W, Ho, Wo, st)
                   : launch_depthwise<float>(h, x, y, bias, relu, N, H, W, Ho, Wo, st);
    }
    if (!h->fast) {
        return f16 ? launch_generic<__half>(h, x, y, bias, relu, N, H, W, Ho, Wo, st)
                   : launch_generic<float>(h, x, y, bias, relu, N, H, W, Ho, Wo, st);
    }
    if (workspace) {
        const size_t es = f16 ? 2 : 4;
        const int C = h->cin_g;
        if (overlaps(workspace, workspace_bytes, x, (size_t)N * C * H * W * es) ||
            overlaps(workspace, workspace_bytes, y, (size_t)N * h->cout * Ho * Wo * es))
            return PP_ERR_BUFFER;
    }
    if (h->stride == 1)
        return f16 ? launch_tm<1, __half>(h, x, y, bias, relu, N, H, W, Ho, Wo, workspace, workspace_bytes, st)
                   : launch_tm<1, float>(h, x, y, bias, relu, N, H, W, Ho, Wo, workspace, workspace_bytes, st);
    return f16 ? launch_tm<2, __half>(h, x, y, bias, relu, N, H, W, Ho, Wo, workspace, workspace_bytes, st)
               : launch_tm<2, float>(h, x, y, bias, relu, N, H, W, Ho, Wo, workspace, workspace_bytes, st);
}

int pp_conv(pp_handle h, const void* x, int dtype, int N, int H, int W, const float* bias, int relu, void* y,
            void* stream) {
    return pp_conv_ws(h, x, dtype, N, H, W, bias, relu, y, nullptr, 0, stream);
}

int pp_conv_pool_ws(pp_handle h, const void* x, int dtype, int N, int H, int W, const float* bias, int relu,
                    void* y, void* workspace, size_t workspace_bytes, void* stream) {
    if (h && (h->depthwise || !h->fast)) return PP_ERR_PATH;
    const int v = validate_conv(h, x, dtype, N, H, W, bias, relu, y, 1);
    if (v != PP_OK || N == 0) return v;
    const int Ho = (H - 1) / h->stride + 1, Wo = (W - 1) / h->stride + 1;
    if (Ho < 2 || Wo < 2) return PP_ERR_SHAPE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const bool f16 = dtype == PP_F16;
    if (workspace) {
        const size_t es = f16 ? 2 : 4;
        if (overlaps(workspace, workspace_bytes, x, (size_t)N * h->cin_g * H * W * es) ||
            overlaps(workspace, workspace_bytes, y, (size_t)N * h->cout * (Ho / 2) * (Wo / 2) * es))
            return PP_ERR_BUFFER;
    }
    if (h->stride == 1)
        return f16 ? launch_tm<1, __half>(h, x, y, bias, relu, N, H, W, Ho, Wo, workspace, workspace_bytes, st, 1)
                   : launch_tm<1, float>(h, x, y, bias, relu, N, H, W, Ho, Wo, workspace, workspace_bytes, st, 1);
    return f16 ? launch_tm<2, __half>(h, x, y, bias, relu, N, H, W, Ho, Wo, workspace, workspace_bytes, st, 1)
               : launch_tm<2, float>(h, x, y, bias, relu, N, H, W, Ho, Wo, workspace, workspace_bytes, st, 1);
}

namespace {
int conv_plan(pp_handle h, int N, int H, int W, size_t workspace_bytes, int64_t* info, int n_info, int pool,
              int es) {
    if (!h || !info) return PP_ERR_NULL;
    if (N < 1 || H < 1 || W < 1 || n_info < 1) return PP_ERR_SHAPE;
    int64_t v[17] = {0};
    if (h->depthwise) {
        v[0] = 2;   // depthwise kernels: no workspace
        DwsParams q{};
        int mode = 0;
        size_t smem = 0;
        const int Ho = (H - 1) / h->stride + 1, Wo = (W - 1) / h->stride + 1;
        if (dws_enabled() && dws_plan(h, N, H, W, Ho, Wo, (size_t)es, &q, &mode, &smem)) {
            v[1] = 1 + mode;
            v[3] = q.n_chunks;
            v[4] = mode == 0 ? q.R : q.P;
            v[5] = q.nst;
            v[10] = (int64_t)smem;
            v[12] = std::min<long long>(sm_count(), (q.n_chunks + q.nwarps - 1) / q.nwarps);
            v[6] = q.nwarps;
        }
    } else if (!h->fast) {
        v[0] = 3;   // generic kernel: no plan, no workspace
    } else {
        Plan pl;
        const int rc = make_plan(h, N, H, W, workspace_bytes, &pl, pool, true, es);
        if (rc != PP_OK) return rc;
        v[0] = 1;
        v[1] = pl.KS;
        v[2] = (int64_t)pl.ws_bytes;
        v[3] = pl.ctas * pl.KS;
        // CTAs of the TMA path (fp32 input, rows a multiple of 16 bytes): persistent, one per SM
        // unless the units overflow a CTA's table; the copy fallback launches one per unit
        v[12] = std::max<long long>(std::min<long long>(v[3], sm_count()),
                                    (v[3] + kMaxUnitsPerCta - 1) / kMaxUnitsPerCta);
        v[4] = pl.tile.BY;
        v[5] = pl.tile.BX;
        v[6] = pl.tile.NB;
        v[7] = pl.CK;
        v[8] = pl.WG;
        v[9] = pl.WS;
        v[10] = (int64_t)pl.smem;
        v[11] = pl.n_chunks;
        v[13] = pl.lane_sort;
        v[16] = pl.dg;
        v[14] = pl.shift;
        v[15] = pl.streamk;
        if (pl.streamk) v[12] = sm_count();
    }
    for (int i = 0; i < n_info && i < 17; ++i) info[i] = v[i];
    return PP_OK;
}
}  // namespace

int pp_conv_plan(pp_handle h, int N, int H, int W, size_t workspace_bytes, int64_t* info, int n_info) {
    return conv_plan(h, N, H, W, workspace_bytes, info, n_info, 0, 4);
}

int pp_conv_pool_plan(pp_handle h, int N, int H, int W, size_t workspace_bytes, int64_t* info, int n_info) {
    if (h && (h->depthwise || !h->fast)) return PP_ERR_PATH;
    return conv_plan(h, N, H, W, workspace_bytes, info, n_info, 1, 4);
}

int pp_conv_plan_dt(pp_handle h, int dtype, int pool, int N, int H, int W, size_t workspace_bytes, int64_t* info,
                    int n_info) {
    if (dtype != PP_F32 && dtype != PP_F16) return PP_ERR_DTYPE;
    if (pool != 0 && pool != 1) return PP_ERR_ARG;
    if (pool && h && (h->depthwise || !h->fast)) return PP_ERR_PATH;
    return conv_plan(h, N, H, W, workspace_bytes, info, n_info, pool, dtype == PP_F32 ? 4 : 2);
}

int pp_conv_tensor_plan(pp_handle h, int dtype, int pool, int N, int H, int W, size_t workspace_bytes, int64_t* info,
                        int n_info) {
    if (!h || !info) return PP_ERR_NULL;
    if (dtype != PP_F32 && dtype != PP_F16) return PP_ERR_DTYPE;
    if (pool != 0 && pool != 1) return PP_ERR_ARG;
    if (pool && (h->depthwise || !h->fast)) return PP_ERR_PATH;
    if (N < 1 || H < 1 || W < 1 || n_info < 1) return PP_ERR_SHAPE;
    int64_t v[9] = {0};
    Plan pl;
    const size_t ws = h->fast ? workspace_bytes : 0;
    if (!h->depthwise && make_plan(h, N, H, W, ws, &pl, pool, true, dtype == PP_F32 ? 4 : 2) == PP_OK && pl.tensor) {
        v[0] = 1;
        v[1] = pl.tc.KS;
        v[2] = (int64_t)pl.tc.ws_bytes;
        v[3] = pl.tc.units;
        v[4] = 128 * pl.tc.MT;
        v[5] = pl.tc.NC;
        v[6] = pl.tc.tw;
        v[7] = pl.tc.th;
        v[8] = pl.tc.box;
    }
    for (int i = 0; i < n_info && i < 9; ++i) info[i] = v[i];
    return PP_OK;
}

int pp_conv_workspace_size(pp_handle h, int N, int H, int W, size_t* bytes) {
    if (!h || !bytes) return PP_ERR_NULL;
    int64_t info[3];
    const int rc = pp_conv_plan(h, N, H, W, (size_t)-1, info, 3);
    if (rc != PP_OK) return rc;
    *bytes = info[0] == 1 ? (size_t)info[2] : 0;
    return PP_OK;
}

int pp_conv_static_scratch(pp_handle h, const void* x, int dtype, int N, int H, int W, const float* bias, int relu,
                           void* y, void* stream) {
    // the argument errors of pp_conv_ws come first, before the scratch size is considered
    const int v = validate_conv(h, x, dtype, N, H, W, bias, relu, y);
    if (v != PP_OK || N == 0) return v;
    // the input-channel split pp_conv_ws would choose with an unlimited workspace (the balanced
    // schedule left out: the array holds split partial sums only)
    size_t need = 0;
    if (!h->depthwise && h->fast) {
        Plan pl;
        const int rc = make_plan(h, N, H, W, (size_t)-1, &pl, 0, false);
        if (rc != PP_OK) return rc;
        need = pl.ws_bytes;
    }
    if (need > kStaticScratchBytes) return PP_ERR_SCRATCH;
    void* scratch = static_scratch_address();
    if (!scratch) return PP_ERR_CUDA;
    return pp_conv_ws(h, x, dtype, N, H, W, bias, relu, y, scratch, kStaticScratchBytes, stream);
}

int pp_static_scratch_bytes(size_t* bytes) {
    if (!bytes) return PP_ERR_NULL;
    *bytes = kStaticScratchBytes;
    return PP_OK;
}

int pp_measure_fp32_peak(int reps, double* flop_per_s) {
    if (!flop_per_s) return PP_ERR_NULL;
    if (reps < 1 || reps > 1000) return PP_ERR_ARG;
    const int sms = sm_count(), ctas = 4 * sms, threads = 512, iters = 4096;
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess) return PP_ERR_CUDA;
    if (cudaEventCreate(&e1) != cudaSuccess) {
        cudaEventDestroy(e0);
        return PP_ERR_CUDA;
    }
    float best = 0.0f;
    bool ok = true;
    fma_peak<<<ctas, threads>>>(16);                      // warm-up
    for (int r = 0; r < reps && ok; ++r) {
        float ms = 0.0f;
        ok = cudaEventRecord(e0) == cudaSuccess;
        fma_peak<<<ctas, threads>>>(iters);
        ok = ok && cudaGetLastError() == cudaSuccess && cudaEventRecord(e1) == cudaSuccess &&
             cudaEventSynchronize(e1) == cudaSuccess && cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess;
        if (ok && ms > 0.0f && (best == 0.0f || ms < best)) best = ms;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (!ok || best <= 0.0f) return PP_ERR_CUDA;
    const double flop = 2.0 * kPeakChains * kPeakUnroll * (double)iters * threads * ctas;
    *flop_per_s = flop / (best * 1e-3);
    return PP_OK;
}

int pp_debug_inject_timeout(void) {
    g_inject_timeout.store(1);
    return PP_OK;
}

int pp_device_status(int clear, unsigned int* status) {
    if (!status) return PP_ERR_NULL;
    unsigned v = 0;
    if (cudaMemcpyFromSymbol(&v, g_pp_status, sizeof(v)) != cudaSuccess) return PP_ERR_CUDA;
    if (clear) {
        const unsigned z = 0;
        if (cudaMemcpyToSymbol(g_pp_status, &z, sizeof(z)) != cudaSuccess) return PP_ERR_CUDA;
    }
    *status = v;
    return PP_OK;
}

int pp_maxpool2x2(const void* x, int dtype, int N, int C, int H, int W, void* y, void* stream) {
    if (dtype != PP_F32 && dtype != PP_F16) return PP_ERR_DTYPE;
    if (N < 0 || C < 1 || H < 2 || W < 2) return PP_ERR_SHAPE;
    if (N == 0) return PP_OK;
    if (!x || !y) return PP_ERR_NULL;
    const size_t es = dtype == PP_F32 ? 4 : 2;
    if (reinterpret_cast<uintptr_t>(x) % es || reinterpret_cast<uintptr_t>(y) % es) return PP_ERR_ALIGN;
    const long long planes = (long long)N * C;
    if (overlaps(x, (size_t)planes * H * W * es, y, (size_t)planes * (H / 2) * (W / 2) * es)) return PP_ERR_BUFFER;
    const long long total = planes * (H / 2) * (W / 2);
    const int blocks = (int)std::max<long long>(1, std::min<long long>((total + 255) / 256, (long long)sm_count() * 64));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (dtype == PP_F32)
        maxpool2x2<float><<<blocks, 256, 0, st>>>(static_cast<const float*>(x), static_cast<float*>(y), planes, H, W);
    else
        maxpool2x2<__half><<<blocks, 256, 0, st>>>(static_cast<const __half*>(x), static_cast<__half*>(y), planes, H, W);
    return cudaGetLastError() == cudaSuccess ? PP_OK : PP_ERR_CUDA;
}

}  // extern "C"
