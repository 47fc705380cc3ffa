// Tensor-core kernels of the surrogate network (sm_103a): BF16 operands
// staged in shared memory by bulk copies (cp.async.bulk on mbarriers),
// tcgen05.mma accumulating in FP32 in tensor memory, epilogues reading TMEM
// with tcgen05.ld.  Activations are planar (see zda_nn_internal.h): each
// 8-channel plane of a window is one contiguous run of rows, which is also
// the canonical no-swizzle operand layout (core matrix = 8 rows x 16 B).
//
// k_conv_tc  -- forward convolution and its input-gradient (transposed)
//               convolution.  A tile is mt x 128 consecutive padded
//               positions with all N output channels.  One window of the
//               input (the tile's positions plus a halo of Wp + 1 rows on
//               each side) serves all taps: tap t is the same window seen
//               from start row halo + off(t), i.e. a different descriptor
//               start address, so no im2col copy is ever made.
// k_wgrad_tc -- weight gradient of the first layer and the head: both operands
//               MN-major (channels contiguous), reduction over positions; M =
//               128 rows hold 128 / c_in taps' shifted copies of the input,
//               each copied pre-shifted.
// k_wgrad_win -- weight and bias gradient of the other layers, all taps of a
//               64-channel input from one window.
//
// Roles of k_conv_tc (608 threads): warp 0 lane 0 = producer, warps 1 and 10
// lane 0 = MMA issuers (M tile 0 / 1 of each tile, warp 1 also allocates
// TMEM), warps 2..9 and 11..18 = epilogue (warp w reads TMEM lanes 32 (w mod
// 4) .., four warps share the 16-channel chunks).  Every mbarrier wait is
// bounded; a timeout sets the error word and the CTA skips its stores, frees
// TMEM and exits.
#include <cuda_bf16.h>

#include <algorithm>

#include "zda_nn_internal.h"
#include "zda_nn_tc.cuh"

namespace zda {
namespace nn {

static __device__ __forceinline__ uint32_t pack_bf16(float a, float b)
{
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t *>(&h);
}

// Bounded wait that also gives up when another role has aborted.
static __device__ __forceinline__ bool wait_or_abort(uint32_t bar, uint32_t parity, int limit, volatile int *abort,
                                                     int *err, int code)
{
    for (int it = 0; it < limit; ++it) {
        if (mb_try(bar, parity)) return true;
        if ((it & 63) == 63 && *abort) return false;
    }
    *abort = 1;
    if (err) atomicCAS(err, 0, code);
    return false;
}

// Two sums at once (each rounded as a single one).
static __device__ __forceinline__ float2 add2(float2 a, float2 b)
{
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;"
        : "=l"(r)
        : "l"(*reinterpret_cast<unsigned long long *>(&a)), "l"(*reinterpret_cast<unsigned long long *>(&b)));
    return *reinterpret_cast<float2 *>(&r);
}

// Epilogue of one 16-channel chunk (channels cc .. cc + 15) of one position,
// f32: straight into the caller's [n][H][W][out_ld] tensor (interior positions only).
__device__ __forceinline__ void store_f32(const ConvParams &p, const float *v, int cc, int pos, int y, int x, bool inner,
                                          const float2 *bias)
{
    if (!inner || cc >= p.out_ld) return;
    const size_t pix = ((size_t)(pos / (p.Hp * p.Wp)) * (p.Hp - 2) + (y - 1)) * (p.Wp - 2) + (x - 1);
    float *o = static_cast<float *>(p.out0) + pix * p.out_ld + cc;
    const int nc = p.out_ld - cc < 16 ? p.out_ld - cc : 16;
    float w[16];
#pragma unroll
    for (int i = 0; i < 8; ++i) *reinterpret_cast<float2 *>(w + 2 * i) = add2(make_float2(v[2 * i], v[2 * i + 1]), bias[i]);
    if ((p.out_ld & 3) == 0) {
        float4 *o4 = reinterpret_cast<float4 *>(o);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (4 * i < nc) o4[i] = make_float4(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]);
    } else {
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (i < nc) o[i] = w[i];
    }
}

// The same, bf16 planes (border positions and those past P are zero).  ReLU
// after rounding is ReLU before it; m0, m1: the sign mask's rows of both planes.
__device__ __forceinline__ void store_bf16(const ConvParams &p, const float *v, int cc, int pos, bool inner,
                                           const float2 *bias, const uint4 &m0, const uint4 &m1)
{
    const int half = cc >= p.out_ld ? 1 : 0;
    const int c = cc - half * p.out_ld;           // channel within the output tensor
    uint32_t w[8];
    if (p.epi == EPI_RELU_BF16) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float2 s = add2(make_float2(v[2 * i], v[2 * i + 1]), bias[i]);
            const __nv_bfloat162 h = __hmax2(__floats2bfloat162_rn(s.x, s.y), __floats2bfloat162_rn(0.f, 0.f));
            w[i] = *reinterpret_cast<const uint32_t *>(&h);
        }
    } else {   // EPI_GRAD_BF16: keep where the activation was positive
        const uint32_t m[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
#pragma unroll
        for (int i = 0; i < 8; ++i) w[i] = pack_bf16(v[2 * i], v[2 * i + 1]) & __vcmpgts2(m[i], 0u);
    }
    if (!inner) {
#pragma unroll
        for (int i = 0; i < 8; ++i) w[i] = 0u;
    }
    uint16_t *ob = static_cast<uint16_t *>(half ? p.out1 : p.out0) + ((size_t)(c / 8) * p.rows + LEAD + pos) * 8;
    *reinterpret_cast<uint4 *>(ob) = make_uint4(w[0], w[1], w[2], w[3]);
    *reinterpret_cast<uint4 *>(ob + (size_t)p.rows * 8) = make_uint4(w[4], w[5], w[6], w[7]);
}

// Mask rows of a chunk (all ones where the gradient is not masked).
__device__ __forceinline__ void load_mask(const ConvParams &p, int cc, int pos, bool inner, uint4 &m0, uint4 &m1)
{
    m0 = m1 = make_uint4(0x00010001u, 0x00010001u, 0x00010001u, 0x00010001u);
    if (p.epi != EPI_GRAD_BF16 || !inner) return;
    const int half = cc >= p.out_ld ? 1 : 0, c = cc - half * p.out_ld;
    const uint16_t *mk = half ? p.mask1 : p.mask0;
    if (!mk) return;
    mk += ((size_t)(c / 8) * p.rows + LEAD + pos) * 8;
    m0 = __ldg(reinterpret_cast<const uint4 *>(mk));
    m1 = __ldg(reinterpret_cast<const uint4 *>(mk + (size_t)p.rows * 8));
}

// The MMAs of one tap for M tile m0 of the tile: NKS K-steps of 16 channels each.
template <int NKS>
__device__ __forceinline__ void issue_tap(uint32_t d0, uint32_t dn, int m0, uint64_t a0, uint32_t a_ks, uint64_t b0,
                                          uint32_t b_ks, uint32_t idesc, uint32_t acc0)
{
    const uint64_t am = a0 + (uint64_t)(m0 * 128);            // 128 rows x 16 B
    const uint32_t dm = d0 + m0 * dn;
    tc_mma(dm, am, b0, idesc, acc0);
#pragma unroll
    for (int ks = 1; ks < NKS; ++ks) tc_mma(dm, am + (uint64_t)(ks * a_ks), b0 + (uint64_t)(ks * b_ks), idesc, 1u);
}

// All MMAs of one unit (up to 32 input channels) of one tile with resident
// weights, fully unrolled over taps, M tiles and K steps.  abase: descriptor
// of the window at row `halo` (a tap adds its row offset: one 16-byte unit
// per row); bbase: descriptor of the unit's half of the first weight block
// of its group.
template <int TAPS, int NKS>
__device__ __forceinline__ void issue_unit(uint32_t d0, uint32_t dn, int m0, uint64_t abase, int Wp, uint64_t bbase,
                                           uint32_t wunits, uint32_t a_ks, uint32_t b_ks, uint32_t idesc, int uu)
{
#pragma unroll
    for (int tap = 0; tap < TAPS; ++tap) {
        const int off = TAPS == 9 ? (tap / 3 - 1) * Wp + (tap % 3 - 1) : 0;
        const uint64_t a0 = abase + (uint64_t)(int64_t)off;
        const uint64_t b0 = bbase + (uint64_t)(tap * wunits);
        issue_tap<NKS>(d0, dn, m0, a0, a_ks, b0, b_ks, idesc, (uu | tap) != 0);
    }
}

__device__ __forceinline__ void mb_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// Persistent, warp-specialised convolution.  Warp 0 (one lane) streams, per
// tile and input unit, the bulk-copied window into one of two to four stages; the
// weight blocks are either loaded once per CTA (resident: every layer whose
// weights fit beside the two windows) or streamed per tap through a ring
// (the concatenating layers); warp 1 (one lane) issues the MMAs
// into one of two TMEM accumulators (2 x mt x N columns); sixteen
// warps drain the other accumulator while the next tile's MMAs run.  With
// eight, whose instructions ran at a sixth of a warp's issue rate, a tile's
// epilogue took 1.6 us and bounded the layers of few MMAs and those that load a
// mask, which is now loaded before the wait (64 x 128 x 128 positions: first
// layer 51 -> 43 us, all 30 convolutions of a gradient 1472 -> 1254 us).
__global__ void __launch_bounds__(CONV_THREADS, 1)
    k_conv_tc(const ConvParams p)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const uint32_t raw = su32(smem), base = (raw + 1023u) & ~1023u;   // copy destinations: 1024-aligned
    // a unit = up to 4 planes (32 channels) of one input group; window stages hold one unit
    const int upl = p.cg / 8 < 4 ? p.cg / 8 : 4, uh = (p.cg / 8) / upl, nunits = p.ngroups * uh;
    const uint32_t win_bytes = (uint32_t)upl * p.plane;
    const uint32_t wslot = (uint32_t)p.N * p.cg * 2;              // one (group, tap) weight block
    const uint32_t uslot = (uint32_t)p.N * upl * 16;              // its share for one unit (streamed ring)
    const int ns = p.stages;
    const uint32_t sWin = base, sW = base + ns * win_bytes;
    const uint32_t sBar = sW + (p.resident ? p.ngroups * p.taps * wslot : p.slots * uslot);
    const uint32_t winFull = sBar, winEmpty = winFull + 8 * ns, accFull = winEmpty + 8 * ns, accEmpty = accFull + 16;
    const uint32_t wFull = accEmpty + 16, wEmpty = wFull + 8 * p.slots;
    const uint32_t sMisc = wEmpty + 8 * p.slots;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(smem + (sMisc - raw));
    volatile int *abort = reinterpret_cast<volatile int *>(smem + (sMisc + 4 - raw));

    const int tile_pos = p.mt * 128;
    const int ntiles = (p.P + tile_pos - 1) / tile_pos;
    const int my_tiles = blockIdx.x < ntiles ? (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    const uint32_t acc_cols = (uint32_t)(p.mt * p.N);

    if (threadIdx.x == 0) {
        for (int s = 0; s < ns; ++s) {
            mb_init(winFull + 8 * s, 1);
            mb_init(winEmpty + 8 * s, 2);          // one commit per MMA warp
        }
        for (int s = 0; s < 2; ++s) {
            mb_init(accFull + 8 * s, 2);
            mb_init(accEmpty + 8 * s, CONV_EPI_WARPS);
        }
        for (int s = 0; s < p.slots; ++s) {
            mb_init(wFull + 8 * s, 1);
            mb_init(wEmpty + 8 * s, 2);
        }
        *abort = 0;
        mb_fence_init();
    }
    if (warp == 1) tm_alloc(sMisc, p.ncols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tslot, 0);

    if (warp == 0) {
        if (elect_one()) {
            // ---------------- producer
            int u = 0, it = 0;
            bool ok = true;
            if (p.resident && my_tiles > 0) {
                mb_expect_tx(wFull, (uint32_t)(p.ngroups * p.taps) * wslot);
                for (int blk = 0; blk < p.ngroups * p.taps; ++blk)
                    bulk_load(sW + blk * wslot, p.wimg + (size_t)blk * p.N * p.cg, wslot, wFull);
            }
            for (int t = 0; t < my_tiles && ok; ++t) {
                const int p0 = ((int)blockIdx.x + t * (int)gridDim.x) * tile_pos;
                for (int uu = 0; uu < nunits && ok; ++uu, ++u) {
                    const int g = uu / uh, hf = uu % uh;
                    const int s = u % ns, k = u / ns;
                    if (k > 0 && !wait_or_abort(winEmpty + 8 * s, (k - 1) & 1, p.wait_limit, abort, p.err, 11)) {
                        ok = false;
                        break;
                    }
                    const uint16_t *src = g == 0 ? p.in0 : p.in1;
                    const uint32_t dst = sWin + s * win_bytes;
                    mb_expect_tx(winFull + 8 * s, (uint32_t)upl * p.R * 16);
                    for (int j = 0; j < upl; ++j)
                        bulk_load(dst + j * p.plane, src + ((size_t)(hf * upl + j) * p.rows + LEAD + p0 - p.halo) * 8,
                                  (uint32_t)p.R * 16, winFull + 8 * s);
                    for (int tap = 0; tap < p.taps && !p.resident; ++tap, ++it) {
                        const int sl = it % p.slots, kk = it / p.slots;
                        if (kk > 0 && !wait_or_abort(wEmpty + 8 * sl, (kk - 1) & 1, p.wait_limit, abort, p.err, 12)) {
                            ok = false;
                            break;
                        }
                        mb_expect_tx(wFull + 8 * sl, uslot);
                        bulk_load(sW + sl * uslot,
                                  p.wimg + (size_t)(g * p.taps + tap) * p.N * p.cg + (size_t)hf * p.N * upl * 8, uslot,
                                  wFull + 8 * sl);
                    }
                }
            }
        }
    } else if (warp == 1 || warp == 10) {
        if (elect_one()) {
            // ---------------- MMA issuers: warp 1 issues M tile 0, warp 10 M tile 1 (separate accumulators)
            const int m0 = warp == 1 ? 0 : 1;
            const uint32_t idesc = idesc_bf16(128, p.N, 0, 0);
            const uint32_t a_ks = (2 * (uint32_t)p.plane) >> 4, b_ks = ((uint32_t)p.N * 32) >> 4;
            const int taps = p.taps, Wp = p.Wp, halo = p.halo, nks = upl / 2, N = p.N;
            const uint32_t plane = (uint32_t)p.plane;
            const bool resident = p.resident != 0;
            int u = 0, it = 0;
            bool ok = true;
            if (resident && my_tiles > 0) ok = wait_or_abort(wFull, 0, p.wait_limit, abort, p.err, 17);
            for (int t = 0; t < my_tiles && ok; ++t) {
                const int b = t & 1, kb = t >> 1;
                if (kb > 0 && !wait_or_abort(accEmpty + 8 * b, (kb - 1) & 1, p.wait_limit, abort, p.err, 13)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t d0 = tmem + b * acc_cols;
                for (int uu = 0; uu < nunits && ok; ++uu, ++u) {
                    const int g = uu / uh, hf = uu % uh;
                    const int s = u % ns, k = u / ns;
                    if (!wait_or_abort(winFull + 8 * s, k & 1, p.wait_limit, abort, p.err, 14)) {
                        ok = false;
                        break;
                    }
                    const uint32_t win = sWin + s * win_bytes;
                    if (resident) {
                        tc_fence_after();
                        // descriptors advance by plain adds: the start-address field is the low
                        // 14 bits in 16-byte units and every address stays below 256 KB
                        const uint64_t abase = sdesc(win + (uint32_t)halo * 16, plane, 128);
                        const uint64_t bbase = sdesc(sW + (uint32_t)(g * taps) * wslot, 128, 256) +
                                               (uint64_t)(hf * nks * b_ks);
                        const uint32_t wunits = wslot >> 4;
                        const int kind = taps * 8 + nks;
                        if (kind == 9 * 8 + 2) issue_unit<9, 2>(d0, N, m0, abase, Wp, bbase, wunits, a_ks, b_ks, idesc, uu);
                        else if (kind == 9 * 8 + 1) issue_unit<9, 1>(d0, N, m0, abase, Wp, bbase, wunits, a_ks, b_ks, idesc, uu);
                        else if (kind == 1 * 8 + 2) issue_unit<1, 2>(d0, N, m0, abase, Wp, bbase, wunits, a_ks, b_ks, idesc, uu);
                        else issue_unit<1, 1>(d0, N, m0, abase, Wp, bbase, wunits, a_ks, b_ks, idesc, uu);
                    } else {
                        for (int tap = 0; tap < taps; ++tap, ++it) {
                            const int sl = it % p.slots, kk = it / p.slots;
                            if (!wait_or_abort(wFull + 8 * sl, kk & 1, p.wait_limit, abort, p.err, 15)) {
                                ok = false;
                                break;
                            }
                            tc_fence_after();
                            const int off = taps == 9 ? (tap / 3 - 1) * Wp + (tap % 3 - 1) : 0;
                            const uint64_t a0 = sdesc(win + (uint32_t)(halo + off) * 16, plane, 128);
                            const uint64_t b0 = sdesc(sW + sl * uslot, 128, 256);
                            const uint32_t acc0 = (uu | tap) != 0;
                            if (nks == 2) issue_tap<2>(d0, N, m0, a0, a_ks, b0, b_ks, idesc, acc0);
                            else issue_tap<1>(d0, N, m0, a0, a_ks, b0, b_ks, idesc, acc0);
                            tc_commit(wEmpty + 8 * sl);
                        }
                    }
                    if (ok) tc_commit(winEmpty + 8 * s);
                }
                if (ok) tc_commit(accFull + 8 * b);
            }
        }
    } else {
        // ---------------- epilogue: warp quarter q's TMEM lanes, 16-channel chunks h, h + 4, ... of both M tiles
        const int q = warp & 3, h = (warp < 10 ? warp - 2 : warp - 3) >> 2;
        const int HW = p.Hp * p.Wp, nchunk = p.N / 16;
        const int step = (int)((long)gridDim.x * tile_pos % HW), step128 = 128 % HW;
        const float inv_wp = 1.f / (float)p.Wp;
        float2 bias[8];                                // of chunk h (layers with biases have N <= 64)
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int c = h * 16 + i;
            reinterpret_cast<float *>(bias)[i] = (p.bias && c < p.nbias) ? __ldg(p.bias + c) : 0.f;
        }
        int rem0 = (int)(((long)blockIdx.x * tile_pos + q * 32 + lane) % HW);
        for (int t = 0; t < my_tiles; ++t) {
            const int b = t & 1, kb = t >> 1;
            const int p0 = ((int)blockIdx.x + t * (int)gridDim.x) * tile_pos;
            // both M tiles' positions: the row by a product (x + 1/2 is at least 1/2 off a multiple of Wp <= 178,
            // x < 1026 x 178, so rounding cannot reach the next row)
            int pos[2], y[2], x[2];
            bool inner[2];
            uint4 mk[2][2];
            int rem = rem0;
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                pos[m] = p0 + m * 128 + q * 32 + lane;
                y[m] = (int)(((float)rem + 0.5f) * inv_wp);
                x[m] = rem - y[m] * p.Wp;
                inner[m] = pos[m] < p.P && y[m] > 0 && y[m] < p.Hp - 1 && x[m] > 0 && x[m] < p.Wp - 1;
                if (h < nchunk) load_mask(p, h * 16, pos[m], inner[m], mk[m][0], mk[m][1]);
                rem += step128;
                rem -= rem >= HW ? HW : 0;
            }
            rem0 += step;
            rem0 -= rem0 >= HW ? HW : 0;
            bool ok = true;
            if (lane == 0) ok = wait_or_abort(accFull + 8 * b, kb & 1, p.wait_limit, abort, p.err, 16);
            ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
            if (!ok) break;
            tc_fence_after();
            const uint32_t trow = tmem + ((uint32_t)(q * 32) << 16) + b * acc_cols;
            for (int c16 = h; c16 < nchunk; c16 += 4) {
                float v[2][16];
                tm_ld16x2(trow + c16 * 16, trow + p.N + c16 * 16, v[0], v[1]);
                if (c16 + 4 >= nchunk) {               // the accumulator is free once the last values are out
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mb_arrive(accEmpty + 8 * b);
                }
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    if (p.epi == EPI_F32 || p.epi == EPI_GRAD_F32) {
                        store_f32(p, v[m], c16 * 16, pos[m], y[m], x[m], inner[m], bias);
                    } else {
                        if (c16 != h) load_mask(p, c16 * 16, pos[m], inner[m], mk[m][0], mk[m][1]);
                        store_bf16(p, v[m], c16 * 16, pos[m], inner[m], bias, mk[m][0], mk[m][1]);
                    }
                }
            }
            if (h >= nchunk) {                         // no chunk for this warp
                __syncwarp();
                if (lane == 0) mb_arrive(accEmpty + 8 * b);
            }
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tm_dealloc(tmem, p.ncols);
}

__global__ void __launch_bounds__(WG_THREADS, 1)
    k_wgrad_tc(const WgradParams p)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const uint32_t raw = su32(smem), base = (raw + 1023u) & ~1023u;
    const uint32_t planeb = (uint32_t)p.kt * 16;
    const uint32_t a_bytes = 16 * planeb, b_bytes = (uint32_t)(p.N / 8) * planeb;
    const uint32_t stage = a_bytes + b_bytes;
    const uint32_t sBar = base + WG_STAGES * stage;
    const uint32_t barF = sBar, barE = sBar + 8 * WG_STAGES, bar_done = barE + 8 * WG_STAGES;
    const uint32_t sTmem = bar_done + 8;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(smem + (sTmem - raw));
    const int g = blockIdx.x, split = blockIdx.y;
    const int tile0 = split * p.tiles_per_cta;
    const int tile1 = min(p.ntiles, tile0 + p.tiles_per_cta);
    const int ntile = max(0, tile1 - tile0);
    const uint32_t ncols = p.N < 32 ? 32 : p.N;

    if (threadIdx.x == 0) {
        for (int s = 0; s < WG_STAGES; ++s) {
            mb_init(barF + 8 * s, 1);
            mb_init(barE + 8 * s, 1);
        }
        mb_init(bar_done, 1);
        mb_fence_init();
    }
    if (warp == 2) tm_alloc(sTmem, ncols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tslot, 0);

    if (warp == 0 && elect_one()) {
        for (int i = 0; i < ntile; ++i) {
            const int s = i % WG_STAGES, u = i / WG_STAGES;
            if (u > 0 && !mb_wait(barE + 8 * s, (u - 1) & 1, p.wait_limit, p.err, 21)) break;
            const uint32_t sa = base + s * stage, sb = sa + a_bytes;
            const int y = (tile0 + i) * p.kt;
            mb_expect_tx(barF + 8 * s, stage);
            for (int j = 0; j < p.ntap_grp; ++j) {
                int t = g * p.ntap_grp + j;
                if (t >= p.taps) t = p.taps - 1;                 // padding copy: its rows are discarded
                const int off = p.taps == 9 ? (t / 3 - 1) * p.Wp + (t % 3 - 1) : 0;
                for (int c = 0; c < p.cin_planes; ++c)
                    bulk_load(sa + (j * p.cin_planes + c) * planeb, p.x + ((size_t)c * p.rows + LEAD + y + off) * 8, planeb,
                              barF + 8 * s);
            }
            for (int c = 0; c < p.N / 8; ++c)
                bulk_load(sb + c * planeb, p.dy + ((size_t)c * p.rows + LEAD + y) * 8, planeb, barF + 8 * s);
        }
    } else if (warp == 1 && elect_one()) {
        const uint32_t idesc = idesc_bf16(128, p.N, 1, 1);
        bool ok = true;
        for (int i = 0; i < ntile; ++i) {
            const int s = i % WG_STAGES, u = i / WG_STAGES;
            if (!mb_wait(barF + 8 * s, u & 1, p.wait_limit, p.err, 22)) {
                ok = false;
                break;
            }
            tc_fence_after();
            const uint32_t sa = base + s * stage, sb = sa + a_bytes;
            const uint64_t ad = sdesc(sa, 128, planeb), bd = sdesc(sb, 128, planeb);
            tc_mma(tmem, ad, bd, idesc, i != 0);
#pragma unroll 8
            for (int ks = 1; ks < p.kt / 16; ++ks)            // 16 rows x 16 B = 16 units per step
                tc_mma(tmem, ad + (uint64_t)(ks * 16), bd + (uint64_t)(ks * 16), idesc, 1u);
            tc_commit(barE + 8 * s);
        }
        if (ok && ntile > 0) tc_commit(bar_done);
    }
    __syncwarp();

    const bool done = ntile == 0 || mb_wait(bar_done, 0, p.wait_limit, p.err, 23);
    tc_fence_after();
    const int row = warp * 32 + lane;
    float *out = p.partial + (((size_t)split * p.ngroups + g) * 128 + row) * p.N;
    for (int c16 = 0; c16 < p.N / 16; ++c16) {
        float v[16];
        tm_ld16(tmem + ((uint32_t)(warp * 32) << 16) + c16 * 16, v);
        if (!done) continue;
        float4 *o = reinterpret_cast<float4 *>(out + c16 * 16);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            o[i] = ntile > 0 ? make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3])
                             : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 2) tm_dealloc(tmem, ncols);
}

// Weight gradient of the 64-channel 3x3 layers, every tap from one window.
//
// D[(tap, c_in)][c_out] = sum_p X[p + off(tap)][c_in] dY[p][c_out], both operands
// MN-major, reduction over positions.  A tap is the same window seen from
// another start row (a plain change of the descriptor's address: rows are 16
// bytes without swizzle), so a CTA streams X and dY through shared memory once
// for all nine taps.  The M = 128 rows of an MMA are two taps: the window is
// kept twice, the second copy one position ahead, and planes 8..15 are that
// copy's.  Three window rows times (dx = -1, 0 | 1, -) make six accumulators of
// 64 columns (384 of the 512 TMEM columns; a quarter of the MMAs' rows is not
// used).  k_wgrad_tc, which loads X once per pair of taps already shifted, reads
// 5 times the bytes and was bound by them: 2.27 ms of a 64 x 128 x 128 batch's
// gradient.
//
// The window is a ring of nine 64-position chunks; the tile at positions
// 64 t .. 64 t + 63 reads chunks t - 3 .. t + 3, so two are in flight.  A K step
// is 16 consecutive rows at any row: the first 16 rows of the ring are copied
// behind its end too, for the steps that straddle it.
// Roles (256 threads): warp 0 lane 0 producer, warps 1 and 2 lane 0 issue three
// accumulators each, warp 3 owns TMEM; all warps store (0..3 the first three
// accumulators, 4..7 the others).  Until then warps 4..7 of the first tensor's
// blocks add up the dY tiles in shared memory for the bias gradient, which
// took a kernel of its own and a second read of dY (24 us at 64 x 128 x 128
// positions).  Waits are bounded.
__global__ void __launch_bounds__(WW_THREADS, 1) k_wgrad_win(const WgradWinParams p)
{
    constexpr int RING = WW_SLOTS * WW_TILE, ROWS = RING + 16;
    constexpr uint32_t PLANE = ROWS * 16, DYB = 8 * WW_TILE * 16;
    extern __shared__ __align__(1024) uint8_t smem[];
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const uint32_t raw = su32(smem), base = (raw + 1023u) & ~1023u;
    const uint32_t sX = base, sDy = sX + 16 * PLANE, sBar = sDy + WW_DY * DYB;
    const uint32_t xF = sBar, xE = xF + 8 * WW_SLOTS, dF = xE + 8 * WW_SLOTS, dE = dF + 8 * WW_DY, bDone = dE + 8 * WW_DY;
    const uint32_t sMisc = bDone + 8;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(smem + (sMisc - raw));
    volatile int *abort = reinterpret_cast<volatile int *>(smem + (sMisc + 4 - raw));
    const int split = blockIdx.x, half = blockIdx.y;
    const int tile0 = split * p.tiles_per_cta, ntile = min(p.ntiles - tile0, p.tiles_per_cta);

    if (threadIdx.x == 0) {
        for (int s = 0; s < WW_SLOTS; ++s) {
            mb_init(xF + 8 * s, 1);
            mb_init(xE + 8 * s, 2);                // one commit per issuer
        }
        for (int s = 0; s < WW_DY; ++s) {
            mb_init(dF + 8 * s, 1);
            mb_init(dE + 8 * s, half ? 2 : 6);     // and one arrival per summing warp
        }
        mb_init(bDone, 2);
        *abort = 0;
        mb_fence_init();
    }
    if (warp == 3) tm_alloc(sMisc, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tslot, 0);

    if (warp == 0 && elect_one()) {
        const uint16_t *x = half ? p.x1 : p.x0;
        bool ok = true;
        for (int c = 0; c < ntile + 6 && ok; ++c) {          // chunk c: positions 64 (tile0 - 3 + c) ..
            const int s = c % WW_SLOTS;
            if (c >= WW_SLOTS && !wait_or_abort(xE + 8 * s, (c / WW_SLOTS - 1) & 1, p.wait_limit, abort, p.err, 31)) break;
            const long pos = (long)WW_TILE * (tile0 - 3 + c);
            mb_expect_tx(xF + 8 * s, 16 * WW_TILE * 16 + (s == 0 ? 16 * 256 : 0));
            for (int j = 0; j < 16; ++j) {
                const uint16_t *src = x + ((size_t)(j & 7) * p.rows + LEAD + pos + (j >> 3)) * 8;
                bulk_load(sX + j * PLANE + s * (WW_TILE * 16), src, WW_TILE * 16, xF + 8 * s);
                if (s == 0) bulk_load(sX + j * PLANE + RING * 16, src, 256, xF + 8 * s);
            }
            const int i = c - 6;                             // the tile that this chunk completes
            if (i < 0) continue;
            const int d = i % WW_DY;
            if (i >= WW_DY) ok = wait_or_abort(dE + 8 * d, (i / WW_DY - 1) & 1, p.wait_limit, abort, p.err, 32);
            if (!ok) break;
            mb_expect_tx(dF + 8 * d, DYB);
            for (int j = 0; j < 8; ++j)
                bulk_load(sDy + d * DYB + j * (WW_TILE * 16),
                          p.dy + ((size_t)j * p.rows + LEAD + (long)WW_TILE * (tile0 + i)) * 8, WW_TILE * 16, dF + 8 * d);
        }
    } else if ((warp == 1 || warp == 2) && elect_one()) {
        const uint32_t idesc = idesc_bf16(128, 64, 1, 1);
        const int g0 = (warp - 1) * 3;
        bool ok = true;
        for (int c = 0; c < 6 && ok; ++c) ok = wait_or_abort(xF + 8 * c, 0, p.wait_limit, abort, p.err, 33);
        for (int i = 0; i < ntile && ok; ++i) {
            const int c = i + 6, d = i % WW_DY;
            ok = wait_or_abort(xF + 8 * (c % WW_SLOTS), (c / WW_SLOTS) & 1, p.wait_limit, abort, p.err, 33) &&
                 wait_or_abort(dF + 8 * d, (i / WW_DY) & 1, p.wait_limit, abort, p.err, 34);
            if (!ok) break;
            tc_fence_after();
            const uint64_t bd = sdesc(sDy + d * DYB, 128, WW_TILE * 16);
#pragma unroll
            for (int g = 0; g < 3; ++g) {
                const int gg = g0 + g, off = (gg / 2 - 1) * p.Wp + ((gg & 1) ? 1 : -1);
                int r = (WW_TILE * (i + 3) + off) % RING;
#pragma unroll
                for (int ks = 0; ks < WW_TILE / 16; ++ks) {
                    tc_mma(tmem + gg * 64, sdesc(sX + r * 16, 128, PLANE), bd + (uint64_t)(ks * 16), idesc, (i | ks) != 0);
                    r += 16;
                    if (r >= RING) r -= RING;
                }
            }
            tc_commit(xE + 8 * (i % WW_SLOTS));              // chunk i has served its last tile
            tc_commit(dE + 8 * d);
        }
        if (ok) tc_commit(bDone);
    } else if (warp >= 4 && half == 0) {
        const int th = threadIdx.x - 128, plane = th >> 4, sub = th & 15;    // 16 threads to a plane of 8 channels
        float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        bool ok = true;
        for (int i = 0; i < ntile && ok; ++i) {
            const int d = i % WW_DY;
            ok = __all_sync(0xffffffffu, wait_or_abort(dF + 8 * d, (i / WW_DY) & 1, p.wait_limit, abort, p.err, 36));
            if (!ok) break;
            const uint4 *row = reinterpret_cast<const uint4 *>(smem + (sDy + d * DYB - raw)) + plane * WW_TILE + sub;
            uint4 v[WW_TILE / 16];
#pragma unroll
            for (int k = 0; k < WW_TILE / 16; ++k) v[k] = row[16 * k];
#pragma unroll
            for (int k = 0; k < WW_TILE / 16; ++k) {
                const uint32_t w[4] = {v[k].x, v[k].y, v[k].z, v[k].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    acc[2 * e] += __uint_as_float(w[e] << 16);
                    acc[2 * e + 1] += __uint_as_float(w[e] & 0xffff0000u);
                }
            }
            // The slot goes back to the bulk copies, which write through the async proxy: the values have to be in
            // registers (the sums hold them there) and this thread's reads ordered before that proxy's writes.
            asm volatile("" ::"f"(acc[0]), "f"(acc[1]), "f"(acc[2]), "f"(acc[3]), "f"(acc[4]), "f"(acc[5]), "f"(acc[6]), "f"(acc[7]));
            fence_async_shared();
            __syncwarp();
            if (lane == 0) mb_arrive(dE + 8 * d);
        }
        __syncwarp();
#pragma unroll
        for (int e = 0; e < 8; ++e)
            for (int o = 8; o > 0; o >>= 1) acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], o);
        if (sub == 0) {
            float4 *out = reinterpret_cast<float4 *>(p.bias + split * 64 + plane * 8);
            out[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
            out[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
        }
    }
    __syncwarp();
    const bool done = wait_or_abort(bDone, 0, p.wait_limit, abort, p.err, 35);
    tc_fence_after();
    // partial [..][group][c_out / 4][row][4]: a warp's 16-byte stores are one run
    const int row = (warp & 3) * 32 + lane, gb = (warp >> 2) * 3;
    for (int g = gb; g < gb + 3; ++g) {
        float4 *out = reinterpret_cast<float4 *>(p.partial + (((size_t)half * gridDim.x + split) * WW_GROUPS + g) * 128 * 64);
        for (int c16 = 0; c16 < 4; ++c16) {
            float v[16];
            tm_ld16(tmem + ((uint32_t)((warp & 3) * 32) << 16) + g * 64 + c16 * 16, v);
            if (!done) continue;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                out[(c16 * 4 + i) * 128 + row] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 3) tm_dealloc(tmem, 512);
}

size_t conv_smem_bytes(const ConvParams &p)
{
    const size_t upl = p.cg / 8 < 4 ? p.cg / 8 : 4;
    const size_t wbytes = p.resident ? (size_t)p.ngroups * p.taps * p.N * p.cg * 2 : (size_t)p.slots * p.N * upl * 16;
    return p.stages * upl * p.plane + wbytes + 16 * p.stages + 32 + 16 * p.slots + 8 + 1024;
}

size_t wgrad_smem_bytes(const WgradParams &p)
{
    return (size_t)WG_STAGES * (16 + p.N / 8) * p.kt * 16 + 16 * WG_STAGES + 16 + 1024;
}

// Resident CTAs x TMEM columns must stay within the SM's 512 columns, or a
// CTA's allocation would wait for another CTA to exit.
static size_t smem_for_tmem(size_t smem, uint32_t ncols)
{
    const size_t per_sm = 228 * 1024;
    const size_t max_ctas = 512 / ncols;
    const size_t need = per_sm / (max_ctas + 1) + 1;   // (max_ctas + 1) CTAs no longer fit
    return smem < need ? need : smem;
}

cudaError_t launch_conv(const ConvParams &p, cudaStream_t s)
{
    const size_t smem = smem_for_tmem(conv_smem_bytes(p), p.ncols);
    if (smem > 227 * 1024) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(k_conv_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0, per_sm = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_conv_tc, CONV_THREADS, smem)) != cudaSuccess)
        return e;
    per_sm = std::max(1, std::min(per_sm, (int)(512 / p.ncols)));
    if (p.mt != 2) return cudaErrorInvalidValue;     // the MMA issue loop is unrolled for two M tiles
    const int ntiles = (p.P + p.mt * 128 - 1) / (p.mt * 128);
    const int grid = std::max(1, std::min(ntiles, sms * per_sm));
    k_conv_tc<<<grid, CONV_THREADS, smem, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_wgrad_win(const WgradWinParams &p, int splits, cudaStream_t s)
{
    const size_t smem = (size_t)16 * (WW_SLOTS * WW_TILE + 16) * 16 + WW_DY * 8 * WW_TILE * 16 +
                        8 * (2 * WW_SLOTS + 2 * WW_DY + 1) + 8 + 1024;
    cudaError_t e = cudaFuncSetAttribute(k_wgrad_win, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_wgrad_win<<<dim3(splits, p.x1 ? 2 : 1), WW_THREADS, smem, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_wgrad(const WgradParams &p, int splits, cudaStream_t s)
{
    size_t smem = smem_for_tmem(wgrad_smem_bytes(p), p.N < 32 ? 32 : p.N);
    if (smem > 227 * 1024) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(k_wgrad_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_wgrad_tc<<<dim3(p.ngroups, splits), WG_THREADS, smem, s>>>(p);
    return cudaGetLastError();
}

}  // namespace nn
}  // namespace zda
