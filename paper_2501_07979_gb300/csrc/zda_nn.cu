// Zone surrogate network: host orchestration, C ABI (include/zda_nn.h) and
// the bandwidth-bound helper kernels (packing, pooling, upsampling, gradient
// combination, reductions, loss, Adam).  The convolutions and their
// gradients run in the tensor-core kernels of zda_nn_conv.cu.
//
// Activations live in zero-bordered NHWC arrays: level l (H_l = H >> l,
// W_l = W >> l) of n samples is a [n][H_l + 2][W_l + 2][C] array whose
// border positions hold zeros, so a 3x3 convolution with zero padding is a
// sum over nine constant position offsets (see k_conv_tc).
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "zda.h"
#include "zda_internal.h"
#include "zda_nn.h"
#include "zda_nn_internal.h"

using namespace zda::nn;

namespace {

zda_status nn_fail(zda_status s, const std::string &m)
{
    zda_internal_set_error(m.c_str());
    return s;
}

#define NN_CUDA(expr)                                                                         \
    do {                                                                                      \
        cudaError_t e_ = (expr);                                                              \
        if (e_ != cudaSuccess)                                                                \
            return nn_fail(ZDA_ERR_CUDA, std::string(#expr) + ": " + cudaGetErrorString(e_)); \
    } while (0)

constexpr int C = 64;      // network width
constexpr int NL = 15;     // parameterised layers
constexpr int LEV = 4;     // resolution levels

__device__ __forceinline__ uint16_t f2bf(float f)
{
    __nv_bfloat16 h = __float2bfloat16_rn(f);
    return *reinterpret_cast<uint16_t *>(&h);
}
__device__ __forceinline__ bool interior(int y, int x, int Hp, int Wp) { return y > 0 && y < Hp - 1 && x > 0 && x < Wp - 1; }

// ---------------------------------------------------------------- helper kernels
// Planar element offset of (channel plane c8, position pos) in a tensor of `rows` rows per plane.
__device__ __forceinline__ size_t pofs(long rows, int c8, long pos) { return ((size_t)c8 * rows + LEAD + pos) * 8; }

// The kernels below run one thread per position of a group of POS_PL planes
// (blockIdx.y), over the Pt positions of the 256-position tiles (borders and
// the tail past the last position are written as zeros).  They are bound by
// memory: a position is taken apart (two 32-bit divisions) once for its planes,
// whose loads are in flight together.  (One thread per position and plane with
// 64-bit divisions: 180 us for k_up and 60 for k_pack_input at 256 x 128 x 128
// positions, 164 for the k_skip_combine of a 64-sample gradient.)
constexpr int POS_PL = 4;

struct Lev {
    int n, H, W;        // samples, interior size of this level
    long rows;          // rows per plane
};

__device__ __forceinline__ bool decode(int n, int H, int W, int pos, int &s, int &y, int &x)
{
    const int Hp = H + 2, Wp = W + 2;
    s = pos / (Hp * Wp);
    const int rem = pos - s * (Hp * Wp);
    y = rem / Wp;
    x = rem - y * Wp;
    return s < n && interior(y, x, Hp, Wp);
}
__device__ __forceinline__ int this_pos() { return (int)(blockIdx.x * blockDim.x + threadIdx.x); }
__device__ __forceinline__ uint4 row_of(const uint16_t *t, long rows, int c8, long pos)
{
    return __ldg(reinterpret_cast<const uint4 *>(t + pofs(rows, c8, pos)));
}
__device__ __forceinline__ void set_row(uint16_t *t, long rows, int c8, long pos, const uint4 &v)
{
    *reinterpret_cast<uint4 *>(t + pofs(rows, c8, pos)) = v;
}
__device__ __forceinline__ void unpack(const uint4 &q, float *v)
{
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        v[2 * e] = __uint_as_float(w[e] << 16);
        v[2 * e + 1] = __uint_as_float(w[e] & 0xffff0000u);
    }
}
__device__ __forceinline__ uint4 packed(const float *v)
{
    uint32_t w[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) w[e] = (uint32_t)f2bf(v[2 * e]) | (uint32_t)f2bf(v[2 * e + 1]) << 16;
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// src [n][H][W][nc] f32 -> planar bf16, `planes` planes (channels >= nc zero)
__global__ void k_pack_rows(const float *src, int n, int H, int W, int nc, int planes, long rows, uint16_t *out)
{
    const int pos = this_pos();
    int s, y, x;
    const bool in = decode(n, H, W, pos, s, y, x);
    src += (((size_t)s * H + (y - 1)) * W + (x - 1)) * nc;
    for (int c8 = 0; c8 < planes; ++c8) {
        float v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = in && c8 * 8 + e < nc ? __ldg(src + c8 * 8 + e) : 0.f;
        set_row(out, rows, c8, pos, packed(v));
    }
}

// avgpool: coarse interior (i, j) = mean of fine interior (2i .. 2i+1, 2j .. 2j+1)
__global__ void k_pool(const uint16_t *in, Lev F, uint16_t *out, Lev Cc)
{
    const int pos = this_pos(), c0 = blockIdx.y * POS_PL;
    int s, y, x;
    const bool on = decode(Cc.n, Cc.H, Cc.W, pos, s, y, x);
    const long fp = ((long)s * (F.H + 2) + 2 * y - 1) * (F.W + 2) + 2 * x - 1;
    uint4 q[POS_PL][4];
#pragma unroll
    for (int c = 0; c < POS_PL; ++c)
#pragma unroll
        for (int a = 0; a < 4; ++a)
            q[c][a] = on ? row_of(in, F.rows, c0 + c, fp + (a >> 1) * (F.W + 2) + (a & 1)) : make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int c = 0; c < POS_PL; ++c) {
        float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            float v[8];
            unpack(q[c][a], v);
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[e] += v[e];
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] *= 0.25f;
        set_row(out, Cc.rows, c0 + c, pos, packed(acc));
    }
}

// nearest upsampling: fine interior (i, j) = coarse interior (i / 2, j / 2)
__global__ void k_up(const uint16_t *in, Lev Cc, uint16_t *out, Lev F)
{
    const int pos = this_pos(), c0 = blockIdx.y * POS_PL;
    int s, y, x;
    const bool on = decode(F.n, F.H, F.W, pos, s, y, x);
    const long cp = ((long)s * (Cc.H + 2) + (y - 1) / 2 + 1) * (Cc.W + 2) + (x - 1) / 2 + 1;
    uint4 q[POS_PL];
#pragma unroll
    for (int c = 0; c < POS_PL; ++c) q[c] = on ? row_of(in, Cc.rows, c0 + c, cp) : make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int c = 0; c < POS_PL; ++c) set_row(out, F.rows, c0 + c, pos, q[c]);
}

// transpose of nearest upsampling (sum over each 2x2 block) times the sign
// mask of the coarse activation: coarse output
__global__ void k_up_bwd_mask(const uint16_t *g, Lev F, const uint16_t *act, uint16_t *out, Lev Cc)
{
    const int pos = this_pos(), c0 = blockIdx.y * POS_PL;
    int s, y, x;
    const bool on = decode(Cc.n, Cc.H, Cc.W, pos, s, y, x);
    const long fp = ((long)s * (F.H + 2) + 2 * y - 1) * (F.W + 2) + 2 * x - 1;
    uint4 q[POS_PL][4], m[POS_PL];
#pragma unroll
    for (int c = 0; c < POS_PL; ++c) {
#pragma unroll
        for (int a = 0; a < 4; ++a)
            q[c][a] = on ? row_of(g, F.rows, c0 + c, fp + (a >> 1) * (F.W + 2) + (a & 1)) : make_uint4(0, 0, 0, 0);
        m[c] = on ? row_of(act, Cc.rows, c0 + c, pos) : make_uint4(0, 0, 0, 0);
    }
#pragma unroll
    for (int c = 0; c < POS_PL; ++c) {
        float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0}, mk[8];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            float v[8];
            unpack(q[c][a], v);
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[e] += v[e];
        }
        unpack(m[c], mk);
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] = mk[e] > 0.f ? acc[e] : 0.f;
        set_row(out, Cc.rows, c0 + c, pos, packed(acc));
    }
}

// skip gradient of level l, in place: mask(act > 0) * (g_skip + transpose of avgpool applied to g_coarse)
__global__ void k_skip_combine(uint16_t *gs, const uint16_t *gc, Lev Cc, const uint16_t *act, Lev F)
{
    const int pos = this_pos(), c0 = blockIdx.y * POS_PL;
    int s, y, x;
    const bool on = decode(F.n, F.H, F.W, pos, s, y, x);
    const long cp = ((long)s * (Cc.H + 2) + (y - 1) / 2 + 1) * (Cc.W + 2) + (x - 1) / 2 + 1;
    const uint4 none = make_uint4(0, 0, 0, 0);
    uint4 a[POS_PL], b[POS_PL], m[POS_PL];
#pragma unroll
    for (int c = 0; c < POS_PL; ++c) {
        a[c] = on ? *reinterpret_cast<const uint4 *>(gs + pofs(F.rows, c0 + c, pos)) : none;
        b[c] = on ? row_of(gc, Cc.rows, c0 + c, cp) : none;
        m[c] = on ? row_of(act, F.rows, c0 + c, pos) : none;
    }
#pragma unroll
    for (int c = 0; c < POS_PL; ++c) {
        float va[8], vb[8], vm[8];
        unpack(a[c], va);
        unpack(b[c], vb);
        unpack(m[c], vm);
#pragma unroll
        for (int e = 0; e < 8; ++e) va[e] = vm[e] > 0.f ? va[e] + 0.25f * vb[e] : 0.f;
        set_row(gs, F.rows, c0 + c, pos, packed(va));
    }
}

// Column sums of a planar bf16 tensor over positions < P (channels < nc):
// partial[block][c].  One plane (8 channels) per blockIdx.y; a thread sums
// whole 16-byte rows, four of them in flight, so the kernel is bound by
// reading g once.  (One 2-byte channel per thread took 1.39 ms of the 4.9 ms of
// a 64 x 128 x 128 batch's gradient.)
__global__ void __launch_bounds__(256) k_colsum(const uint16_t *g, long rows, long P, int nc, float *partial)
{
    __shared__ float red[8][8];
    const int c8 = blockIdx.y;
    const long step = (long)gridDim.x * 256;
    const uint4 *src = reinterpret_cast<const uint4 *>(g + pofs(rows, c8, 0));
    float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    auto add = [&](const uint4 &v) {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            acc[2 * e] += __uint_as_float(w[e] << 16);
            acc[2 * e + 1] += __uint_as_float(w[e] & 0xffff0000u);
        }
    };
    long p = (long)blockIdx.x * 256 + threadIdx.x;
    for (; p + 3 * step < P; p += 4 * step) {
        const uint4 a = __ldg(src + p), b = __ldg(src + p + step), c = __ldg(src + p + 2 * step), d = __ldg(src + p + 3 * step);
        add(a);
        add(b);
        add(c);
        add(d);
    }
    for (; p < P; p += step) add(__ldg(src + p));
#pragma unroll
    for (int e = 0; e < 8; ++e)
        for (int o = 16; o > 0; o >>= 1) acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], o);
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int e = 0; e < 8; ++e) red[threadIdx.x >> 5][e] = acc[e];
    __syncthreads();
    if (threadIdx.x < 8) {
        float t = 0.f;
        for (int w = 0; w < 8; ++w) t += red[w][threadIdx.x];
        const int c = c8 * 8 + threadIdx.x;
        if (c < nc) partial[(size_t)blockIdx.x * nc + c] = t;
    }
}

// Layer gradient from the wgrad partials and the bias partials [nblk][cout]:
// grads[w[co][t][ci]], grads[b[co]].  A block sums 64 neighbouring values of the
// partials (a whole 256-byte line of every split), four to a thread and
// LG_PARTS threads to a value, so a thread's ten or so 16-byte loads are all in
// flight; the last block sums the biases.  Bound by that one round of loads
// (30 MB of partials from L2).  One value per thread: 16 us a layer of a
// 64-sample gradient, 9 now; threads along c_in that each walked all splits
// alone: 20 us a layer of a one-sample gradient.
// win = 0: [splits][ngroups][128][N] of k_wgrad_tc; 1: [tensors][splits][6][16][128][4] of k_wgrad_win.
constexpr int LG_THREADS = 256, LG_VALUES = 64, LG_PARTS = LG_THREADS * 4 / LG_VALUES;
__global__ void __launch_bounds__(LG_THREADS) k_layer_grad(const float *wpart, int win, int splits, int ngroups, int ntap_grp,
                                                           int cin_pad, int N, const float *bpart, int nblk, int cout,
                                                           int cin, int taps, float *grad)
{
    __shared__ float red[LG_PARTS][LG_VALUES];
    const int first4 = threadIdx.x * 4 % LG_VALUES, part = threadIdx.x * 4 / LG_VALUES;
    const bool bias = blockIdx.x + 1 == gridDim.x;
    const int per = (win ? WW_GROUPS : ngroups) * 128 * N;   // values of a split
    // where value v of a split (all tensors in turn) comes from and goes to; runs of four share tap and c_in
    auto locate = [&](long v, size_t &from, int &co, int &t, int &ci) {
        if (win) {
            const int half = (int)(v / per), w = (int)(v % per), g = w / (128 * 64), row = w / 4 % 128;
            co = w / 512 % 16 * 4 + w % 4;
            t = (g & 1) && row >= 64 ? taps : g / 2 * 3 + ((g & 1) ? 2 : row / 64);   // taps: the unused second tap
            ci = half * 64 + row % 64;
            from = (size_t)half * splits * per + w;
        } else {
            const int row = (int)(v / N) % 128, g = (int)(v / (128 * N));
            co = (int)(v % N);
            t = g * ntap_grp + row / cin_pad;
            ci = row % cin_pad;
            from = (size_t)v;
        }
    };
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (bias) {
        float *f = reinterpret_cast<float *>(&s);
        for (int e = 0; e < 4; ++e)
            if (first4 + e < cout)
                for (int k = part; k < nblk; k += LG_PARTS) f[e] += __ldg(bpart + (size_t)k * cout + first4 + e);
    } else {
        size_t from;
        int co, t, ci;
        locate((long)blockIdx.x * LG_VALUES + first4, from, co, t, ci);
        const float4 *src = reinterpret_cast<const float4 *>(wpart + from);
        const int count = co < cout && t < taps && ci < cin ? splits : 0;
#pragma unroll 10
        for (int k = part; k < count; k += LG_PARTS) {
            const float4 v = __ldg(src + (size_t)k * (per / 4));
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
    }
    *reinterpret_cast<float4 *>(&red[part][first4]) = s;
    __syncthreads();
    if (threadIdx.x >= LG_VALUES) return;
    size_t from;
    int co = threadIdx.x, t = 0, ci = 0;
    if (!bias) locate((long)blockIdx.x * LG_VALUES + threadIdx.x, from, co, t, ci);
    if (co >= cout || t >= taps || ci >= cin) return;
    float sum = red[0][threadIdx.x];
#pragma unroll
    for (int q = 1; q < LG_PARTS; ++q) sum += red[q][threadIdx.x];
    grad[bias ? (long)cout * taps * cin + co : ((long)co * taps + t) * cin + ci] = sum;
}

struct PackLayer {
    long off;          // parameter offset of w
    int k, cin, cout;  // kernel size, true channels
    int cin_pad;       // input channels in the activation (16 for the input layer, else cin)
    int nf;            // forward GEMM N (cout padded to 32 for the head, else 64)
    long img_f, img_d; // element offsets of the forward / input-gradient images
};

// Operand image of one (group, tap) block, K-major, no swizzle: element
// (n, k) of an N x cg block at ks = k / 16: ks N 16 + (n / 8) 128 + ((k / 8) % 2) 64 + (n % 8) 8 + k % 8.
__device__ __forceinline__ long img_index(int n, int k, int N)
{
    return (long)(k / 16) * N * 16 + (n / 8) * 128 + ((k / 8) % 2) * 64 + (n % 8) * 8 + (k % 8);
}

__global__ void k_pack_weights(const float *params, PackLayer L, uint16_t *img)
{
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    const int taps = L.k * L.k;
    const int cg = L.cin_pad > 64 ? 64 : L.cin_pad;
    const long nf_tot = (long)taps * L.nf * L.cin_pad;           // forward image elements
    const long nd_tot = (long)taps * L.cin_pad * L.nf;           // input-gradient image elements
    if (i < nf_tot) {
        // forward: group g (64 channels), tap t, row n = c_out, column k = c_in within the group
        const int k = (int)(i % cg), n = (int)((i / cg) % L.nf), t = (int)((i / ((long)cg * L.nf)) % taps);
        const int g = (int)(i / ((long)cg * L.nf * taps));
        const int ci = g * cg + k;
        float v = 0.f;
        if (n < L.cout && ci < L.cin) v = params[L.off + (((long)n * taps + t) * L.cin) + ci];
        img[L.img_f + (long)(g * taps + t) * L.nf * cg + img_index(n, k, L.nf)] = f2bf(v);
    } else if (i < nf_tot + nd_tot) {
        // input gradient: tap t' (flipped), row n = c_in, column k = c_out
        const long j = i - nf_tot;
        const int k = (int)(j % L.nf), n = (int)((j / L.nf) % L.cin_pad), tp = (int)(j / ((long)L.nf * L.cin_pad));
        const int ty = tp / L.k, tx = tp % L.k;
        const int t = (L.k - 1 - ty) * L.k + (L.k - 1 - tx);
        float v = 0.f;
        if (k < L.cout && n < L.cin) v = params[L.off + (((long)k * taps + t) * L.cin) + n];
        img[L.img_d + (long)tp * L.cin_pad * L.nf + img_index(n, k, L.cin_pad)] = f2bf(v);
    }
}

__global__ void k_adam(float *p, const float *g, float *m, float *v, long n, float lr, float b1, float b2, float eps,
                       float c1, float c2)
{
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

__global__ void k_mse(const float *y, const float *t, long n, float *dy, float *partial)
{
    __shared__ float red[256];
    float acc = 0.f;
    const float sc = 2.f / (float)n;
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
        const float d = y[i] - t[i];
        dy[i] = sc * d;
        acc += d * d;
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[blockIdx.x] = red[0];
}

__global__ void __launch_bounds__(256) k_mse_final(const float *partial, int nblk, long n, float *loss)
{
    __shared__ double red[256];
    double s = 0.0;
    for (int b = threadIdx.x; b < nblk; b += 256) s += partial[b];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) *loss = (float)(red[0] / (double)n);
}

unsigned nblocks(long n, int t = 256) { return (unsigned)((n + t - 1) / t); }

// ---------------------------------------------------------------- layers
struct Layer {
    const char *name;
    int k, cin, cout, level;
    int cin_pad, nf;
    long off;          // parameter offset
    long img_f, img_d; // image offsets (elements)
};

}  // namespace

struct zda_nn {
    int device = 0;
    zda_nn_desc d{};
    int H[LEV], W[LEV];
    long rows[LEV];        // rows per plane of the level's planar tensors (batch capacity)
    Layer L[NL];
    long nparam = 0, img_elems = 0;
    double flops = 0;
    // workspace
    uint8_t *ws = nullptr;
    size_t ws_bytes = 0, need = 0;
    struct Off {
        size_t params, grads, m, v, img, x16, gy, wpart, bpart, mpart, err;
        size_t act[LEV][8];   // per level: enc_a, enc_b, in (pooled input), up, dec_a, dec_b, (level 3: bot_a, bot_b)
        size_t g[LEV][5];     // per level: gA, gB, gU, gS; levels 1 and 2: gI
    } o{};
    size_t wpart_floats = 0;
    int bpart_blocks = 240;      // at least WW_CTAS
    int adam_step = 0;
    long long launches = 0;
    int n_fwd = 0;
    bool bound = false;
    // Weight gradients run on a stream of their own beside the chain of input gradients (backward_chain).
    cudaStream_t side = nullptr;
    cudaEvent_t forked = nullptr, joined = nullptr;
    // optional CUDA-event timing of the convolution launches
    bool timing = false;
    std::vector<cudaEvent_t> ev;       // pairs (before, after)
    std::vector<double> ev_flops;      // useful FLOPs of each timed launch
    size_t ev_used = 0;
    ~zda_nn()
    {
        if (forked) cudaEventDestroy(forked);
        if (joined) cudaEventDestroy(joined);
        if (side) cudaStreamDestroy(side);
        for (cudaEvent_t e : ev) cudaEventDestroy(e);
    }
};

namespace {

enum { A_ENCA = 0, A_ENCB, A_IN, A_UP, A_DECA, A_DECB };
enum { G_A = 0, G_B, G_U, G_S, G_I };

template <class T> T *at(zda_nn *net, size_t off) { return reinterpret_cast<T *>(net->ws + off); }

long pos_count(const zda_nn *net, int lev, int n) { return (long)n * (net->H[lev] + 2) * (net->W[lev] + 2); }
long pos_tiles(const zda_nn *net, int lev, int n) { return (pos_count(net, lev, n) + 255) / 256 * 256; }
dim3 pos_grid(const zda_nn *net, int lev, int n) { return dim3(nblocks(pos_tiles(net, lev, n)), 8 / POS_PL); }
Lev lev(const zda_nn *net, int l, int n) { return Lev{n, net->H[l], net->W[l], net->rows[l]}; }

void build_layers(zda_nn *net)
{
    const int ic = net->d.in_ch, oc = net->d.out_ch;
    const char *names[NL] = {"enc0a", "enc0b", "enc1a", "enc1b", "enc2a", "enc2b", "bota", "botb",
                             "dec2a", "dec2b", "dec1a", "dec1b", "dec0a", "dec0b", "head"};
    const int lev[NL] = {0, 0, 1, 1, 2, 2, 3, 3, 2, 2, 1, 1, 0, 0, 0};
    long off = 0, img = 0;
    double fl = 0;
    for (int i = 0; i < NL; ++i) {
        Layer &l = net->L[i];
        l.name = names[i];
        l.level = lev[i];
        l.k = i == NL - 1 ? 1 : 3;
        l.cin = i == 0 ? ic : ((i == 8 || i == 10 || i == 12) ? 2 * C : C);
        l.cout = i == NL - 1 ? oc : C;
        l.cin_pad = i == 0 ? 16 : l.cin;
        l.nf = i == NL - 1 ? 32 : C;
        l.off = off;
        off += (long)l.cout * l.k * l.k * l.cin + l.cout;
        l.img_f = img;
        img += (long)l.k * l.k * l.nf * l.cin_pad;
        l.img_d = img;
        img += (long)l.k * l.k * l.nf * l.cin_pad;
        fl += 2.0 * net->H[l.level] * net->W[l.level] * l.k * l.k * l.cin * l.cout;
    }
    net->nparam = off;
    net->img_elems = img;
    net->flops = fl;
}

int round_up(int a, int b) { return (a + b - 1) / b * b; }

// Convolution (forward or input gradient) of one layer.
//   in0 / in1 : input tensors (in1 = second half of a concatenated input or null)
//   cg        : channels per input tensor;  N : GEMM output channels
zda_status conv(zda_nn *net, int lv, int n, int taps, const uint16_t *in0, const uint16_t *in1, int cg, int N,
                const uint16_t *wimg, const float *bias, int nbias, int epi, void *out0, void *out1, int out_ld,
                const uint16_t *mask0, const uint16_t *mask1, cudaStream_t s, double flops = 0.0)
{
    ConvParams p{};
    p.Hp = net->H[lv] + 2;
    p.Wp = net->W[lv] + 2;
    p.P = (int)pos_count(net, lv, n);
    p.taps = taps;
    p.halo = taps == 9 ? p.Wp + 1 : 0;
    p.mt = 2;
    p.R = p.mt * 128 + 2 * p.halo;
    p.plane = round_up(p.R, 8) * 16;
    p.rows = net->rows[lv];
    p.cg = cg;
    p.ngroups = in1 ? 2 : 1;
    p.N = N;
    // weights resident if they fit beside the two window stages, else a ring
    // of as many per-tap slots as fit (at most 8)
    const size_t budget = 220 * 1024;
    const size_t upl = std::min(cg / 8, 4);                    // window planes per unit (32 channels)
    const size_t win2 = 2 * upl * p.plane, wslot = (size_t)N * cg * 2, uslot = (size_t)N * upl * 16;
    p.resident = win2 + (size_t)p.ngroups * taps * wslot <= budget ? 1 : 0;
    // window stages: up to four where the resident weights leave room (3x3, 64 channels: 73 KB of weights, 33 KB a
    // stage at 128 x 128 pixels); two hide less of a window's latency (forward of 256 patches 2328 us, 2171 with four)
    p.stages = 2;
    if (p.resident) {
        const size_t left = budget - (size_t)p.ngroups * taps * wslot;
        p.stages = (int)std::max<size_t>(2, std::min<size_t>(4, left / (upl * p.plane)));
    }
    p.slots = p.resident ? 1 : (int)std::max<size_t>(2, std::min<size_t>(8, (budget - win2) / uslot));
    uint32_t nc = 32;
    while (nc < (uint32_t)(2 * p.mt * N)) nc <<= 1;   // two accumulators (double buffering)
    p.ncols = nc;
    p.in0 = in0;
    p.in1 = in1;
    p.wimg = wimg;
    p.bias = bias;
    p.nbias = nbias;
    p.epi = epi;
    p.out0 = out0;
    p.out1 = out1;
    p.out_ld = out_ld;
    p.mask0 = mask0;
    p.mask1 = mask1;
    p.err = at<int>(net, net->o.err);
    p.wait_limit = 1 << 22;
    const bool timed = net->timing && flops > 0.0;
    if (timed) {
        if (net->ev_used + 2 > net->ev.size()) {
            for (int k = 0; k < 64; ++k) {
                cudaEvent_t ev;
                NN_CUDA(cudaEventCreate(&ev));
                net->ev.push_back(ev);
            }
        }
        NN_CUDA(cudaEventRecord(net->ev[net->ev_used], s));
    }
    cudaError_t e = launch_conv(p, s);
    if (e != cudaSuccess) return nn_fail(ZDA_ERR_CUDA, std::string("conv launch: ") + cudaGetErrorString(e));
    if (timed) {
        NN_CUDA(cudaEventRecord(net->ev[net->ev_used + 1], s));
        net->ev_used += 2;
        net->ev_flops.push_back(flops);
    }
    net->launches++;
    return ZDA_OK;
}

// Weight + bias gradient of layer li: x0 (/x1) its input, g the gradient of its
// pre-activation output ([P][ldg] bf16).
zda_status layer_grad(zda_nn *net, int li, int n, const uint16_t *x0, const uint16_t *x1, const uint16_t *g, int ldg,
                      cudaStream_t s)
{
    const Layer &l = net->L[li];
    const long P = pos_count(net, l.level, n), rows = net->rows[l.level];
    const int Wp = net->W[l.level] + 2, taps = l.k * l.k;
    // all 3x3 layers but the first have 64 channels per tensor and take the one-window kernel
    static_assert(176 + 2 + 1 <= WW_MAX_HALO, "a window of the widest image fits its seven chunks");
    const bool win = taps == 9 && l.cin_pad % C == 0;
    int splits, ngroups = 0, ntap_grp = 0, nrow;
    cudaError_t e;
    if (win) {
        WgradWinParams p{};
        p.P = (int)P;
        p.Wp = Wp;
        p.ntiles = (int)((P + WW_TILE - 1) / WW_TILE);
        const int tensors = x1 ? 2 : 1, ctas = WW_CTAS / tensors;
        p.tiles_per_cta = std::max(WW_MIN_TILES, (p.ntiles + ctas - 1) / ctas);
        splits = (p.ntiles + p.tiles_per_cta - 1) / p.tiles_per_cta;
        nrow = tensors * WW_GROUPS * 128;
        if ((size_t)splits * nrow * C > net->wpart_floats)
            return nn_fail(ZDA_ERR_OOM, "weight-gradient partial buffer too small");
        p.rows = rows;
        p.x0 = x0;
        p.x1 = x1;
        p.dy = g;
        p.partial = at<float>(net, net->o.wpart);
        p.bias = at<float>(net, net->o.bpart);
        p.err = at<int>(net, net->o.err);
        p.wait_limit = 1 << 22;
        e = launch_wgrad_win(p, splits, s);
    } else {
        WgradParams p{};
        p.Hp = net->H[l.level] + 2;
        p.Wp = Wp;
        p.P = (int)P;
        p.taps = taps;
        p.cin_planes = l.cin_pad / 8;
        p.ntap_grp = ntap_grp = 16 / p.cin_planes;
        p.ngroups = ngroups = (p.taps + p.ntap_grp - 1) / p.ntap_grp;
        p.N = ldg;
        p.kt = WG_KT;
        p.ntiles = (p.P + p.kt - 1) / p.kt;
        splits = std::max(1, std::min(p.ntiles, (304 + p.ngroups - 1) / p.ngroups));
        p.tiles_per_cta = (p.ntiles + splits - 1) / splits;
        splits = (p.ntiles + p.tiles_per_cta - 1) / p.tiles_per_cta;
        nrow = ngroups * 128;
        if ((size_t)splits * nrow * p.N > net->wpart_floats)
            return nn_fail(ZDA_ERR_OOM, "weight-gradient partial buffer too small");
        p.rows = rows;
        p.x = x0;
        p.dy = g;
        p.partial = at<float>(net, net->o.wpart);
        p.err = at<int>(net, net->o.err);
        p.wait_limit = 1 << 22;
        e = launch_wgrad(p, splits, s);
    }
    if (e != cudaSuccess) return nn_fail(ZDA_ERR_CUDA, std::string("wgrad launch: ") + cudaGetErrorString(e));
    // bias partials: k_wgrad_win leaves one per block; else blocks of at least 1024 positions per plane, so that
    // small levels leave few of them
    int nblk = splits;
    if (!win) {
        nblk = (int)std::max<long>(1, std::min<long>(net->bpart_blocks, P / 1024));
        k_colsum<<<dim3(nblk, ldg / 8), 256, 0, s>>>(g, rows, P, l.cout, at<float>(net, net->o.bpart));
        net->launches++;
    }
    k_layer_grad<<<(unsigned)((long)nrow * ldg / LG_VALUES) + 1, LG_THREADS, 0, s>>>(
        at<float>(net, net->o.wpart), win ? 1 : 0, splits, ngroups, ntap_grp, l.cin_pad, ldg,
        at<float>(net, net->o.bpart), nblk, l.cout, l.cin, taps, at<float>(net, net->o.grads) + l.off);
    net->launches += 2;
    e = cudaGetLastError();
    if (e != cudaSuccess) return nn_fail(ZDA_ERR_CUDA, std::string("gradient reduction: ") + cudaGetErrorString(e));
    return ZDA_OK;
}

zda_status pack_all(zda_nn *net, cudaStream_t s)
{
    for (int i = 0; i < NL; ++i) {
        const Layer &l = net->L[i];
        PackLayer pl{l.off, l.k, l.cin, l.cout, l.cin_pad, l.nf, l.img_f, l.img_d};
        const long tot = 2L * l.k * l.k * l.nf * l.cin_pad;
        k_pack_weights<<<nblocks(tot), 256, 0, s>>>(at<float>(net, net->o.params), pl, at<uint16_t>(net, net->o.img));
        net->launches++;
    }
    NN_CUDA(cudaGetLastError());
    return ZDA_OK;
}

// useful forward FLOPs of layer i over n samples (true channel counts, H_l x W_l outputs)
double lf(const zda_nn *net, int i, int n)
{
    const Layer &l = net->L[i];
    return 2.0 * n * net->H[l.level] * net->W[l.level] * l.k * l.k * l.cin * l.cout;
}

const uint16_t *A(zda_nn *net, int lev, int k) { return at<uint16_t>(net, net->o.act[lev][k]); }
uint16_t *Aw(zda_nn *net, int lev, int k) { return at<uint16_t>(net, net->o.act[lev][k]); }
uint16_t *Gb(zda_nn *net, int lev, int k) { return at<uint16_t>(net, net->o.g[lev][k]); }
const uint16_t *Wf(zda_nn *net, int i) { return at<uint16_t>(net, net->o.img) + net->L[i].img_f; }
const uint16_t *Wd(zda_nn *net, int i) { return at<uint16_t>(net, net->o.img) + net->L[i].img_d; }
const float *Bias(zda_nn *net, int i) { return at<float>(net, net->o.params) + net->L[i].off + (long)net->L[i].cout * net->L[i].k * net->L[i].k * net->L[i].cin; }

}  // namespace

// ======================================================================== ABI
extern "C" {

zda_status zda_nn_create(int device, const zda_nn_desc *d, zda_nn **out)
{
    if (!d || !out) return nn_fail(ZDA_ERR_ARG, "null argument");
    *out = nullptr;
    if (d->batch < 1 || d->height < 8 || d->width < 8 || d->height % 8 || d->width % 8 || d->height > 1024 ||
        d->width > 176 || d->in_ch < 1 || d->in_ch > 16 || d->out_ch < 1 || d->out_ch > 32)
        return nn_fail(ZDA_ERR_ARG, "invalid network descriptor (H multiple of 8 in 8..1024, W multiple of 8 in "
                                    "8..176; 1..16 inputs; 1..32 outputs; batch >= 1)");
    const long P0 = (long)d->batch * (d->height + 2) * (d->width + 2);
    if (P0 * 64 > (1L << 31) - 1) return nn_fail(ZDA_ERR_ARG, "batch x image too large for 32-bit positions");
    zda_nn *net = new zda_nn();
    net->device = device;
    net->d = *d;
    for (int l = 0; l < LEV; ++l) {
        net->H[l] = d->height >> l;
        net->W[l] = d->width >> l;
        net->rows[l] = LEAD + pos_tiles(net, l, d->batch) + 256;   // zero lead rows, tiles, zero trail rows
    }
    build_layers(net);
    // workspace layout
    size_t o = 0;
    auto take = [&](size_t bytes) {
        const size_t r = o;
        o += (bytes + 255) / 256 * 256;
        return r;
    };
    const int B = d->batch;
    net->o.params = take(net->nparam * 4);
    net->o.grads = take(net->nparam * 4);
    net->o.m = take(net->nparam * 4);
    net->o.v = take(net->nparam * 4);
    net->o.img = take(net->img_elems * 2);
    net->o.x16 = take((size_t)net->rows[0] * 16 * 2);
    net->o.gy = take((size_t)net->rows[0] * 32 * 2);
    for (int l = 0; l < LEV; ++l) {
        const size_t t = (size_t)net->rows[l] * C * 2;
        for (int k = 0; k < 6; ++k) net->o.act[l][k] = take(t);
        for (int k = 0; k < (l == 1 || l == 2 ? 5 : 4); ++k) net->o.g[l][k] = take(t);
    }
    size_t wp = 0;
    for (int i = 0; i < NL; ++i) {
        const Layer &l = net->L[i];
        const int taps = l.k * l.k, ntg = 16 / (l.cin_pad / 8), ng = (taps + ntg - 1) / ntg;
        const size_t splits = (size_t)std::min<long>((pos_count(net, l.level, B) + 127) / 128, (304 + ng - 1) / ng) + 1;
        wp = std::max(wp, splits * ng * 128 * (size_t)(i == NL - 1 ? 32 : 64));
    }
    wp = std::max(wp, (size_t)WW_CTAS * WW_GROUPS * 128 * C);        // k_wgrad_win: one partial per block
    net->wpart_floats = wp;
    net->o.wpart = take(wp * 4);
    net->o.bpart = take((size_t)net->bpart_blocks * 64 * 4);
    net->o.mpart = take(1024 * 4);
    net->o.err = take(16);
    net->need = o;
    *out = net;
    return ZDA_OK;
}

void zda_nn_destroy(zda_nn *net) { delete net; }

zda_status zda_nn_param_count(const zda_nn *net, size_t *count)
{
    if (!net || !count) return nn_fail(ZDA_ERR_ARG, "null argument");
    *count = (size_t)net->nparam;
    return ZDA_OK;
}

zda_status zda_nn_forward_flops(const zda_nn *net, double *flops)
{
    if (!net || !flops) return nn_fail(ZDA_ERR_ARG, "null argument");
    *flops = net->flops;
    return ZDA_OK;
}

zda_status zda_nn_workspace_bytes(const zda_nn *net, size_t *bytes)
{
    if (!net || !bytes) return nn_fail(ZDA_ERR_ARG, "null argument");
    *bytes = net->need;
    return ZDA_OK;
}

zda_status zda_nn_bind_workspace(zda_nn *net, void *ws, size_t bytes)
{
    if (!net || !ws) return nn_fail(ZDA_ERR_ARG, "null argument");
    if (bytes < net->need) return nn_fail(ZDA_ERR_OOM, "workspace smaller than zda_nn_workspace_bytes");
    if (reinterpret_cast<uintptr_t>(ws) % 256) return nn_fail(ZDA_ERR_ARG, "workspace must be 256-byte aligned");
    NN_CUDA(cudaSetDevice(net->device));
    net->ws = static_cast<uint8_t *>(ws);
    net->ws_bytes = bytes;
    if (!net->side) NN_CUDA(cudaStreamCreateWithFlags(&net->side, cudaStreamNonBlocking));
    if (!net->forked) NN_CUDA(cudaEventCreateWithFlags(&net->forked, cudaEventDisableTiming));
    if (!net->joined) NN_CUDA(cudaEventCreateWithFlags(&net->joined, cudaEventDisableTiming));
    NN_CUDA(cudaMemset(ws, 0, net->need));
    net->bound = true;
    net->adam_step = 0;
    net->n_fwd = 0;
    return ZDA_OK;
}

static zda_status need_bound(zda_nn *net)
{
    if (!net) return nn_fail(ZDA_ERR_ARG, "null network");
    if (!net->bound) return nn_fail(ZDA_ERR_STATE, "no workspace bound");
    cudaError_t e = cudaSetDevice(net->device);
    if (e != cudaSuccess) return nn_fail(ZDA_ERR_CUDA, std::string("cudaSetDevice: ") + cudaGetErrorString(e));
    return ZDA_OK;
}

zda_status zda_nn_set_params(zda_nn *net, const float *params, int host, void *stream)
{
    zda_status st = need_bound(net);
    if (st != ZDA_OK) return st;
    if (!params) return nn_fail(ZDA_ERR_ARG, "null parameters");
    cudaStream_t s = (cudaStream_t)stream;
    const size_t b = net->nparam * 4;
    NN_CUDA(cudaMemcpyAsync(at<float>(net, net->o.params), params, b,
                            host ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice, s));
    NN_CUDA(cudaMemsetAsync(at<float>(net, net->o.m), 0, b, s));
    NN_CUDA(cudaMemsetAsync(at<float>(net, net->o.v), 0, b, s));
    net->adam_step = 0;
    st = pack_all(net, s);
    if (st != ZDA_OK) return st;
    if (host) NN_CUDA(cudaStreamSynchronize(s));
    return ZDA_OK;
}

static zda_status copy_out(zda_nn *net, size_t off, float *dst, int host, void *stream)
{
    zda_status st = need_bound(net);
    if (st != ZDA_OK) return st;
    if (!dst) return nn_fail(ZDA_ERR_ARG, "null output");
    cudaStream_t s = (cudaStream_t)stream;
    NN_CUDA(cudaMemcpyAsync(dst, at<float>(net, off), net->nparam * 4,
                            host ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice, s));
    if (host) NN_CUDA(cudaStreamSynchronize(s));
    return ZDA_OK;
}

zda_status zda_nn_get_params(zda_nn *net, float *params, int host, void *stream)
{
    return copy_out(net, net ? net->o.params : 0, params, host, stream);
}

zda_status zda_nn_get_grads(zda_nn *net, float *grads, int host, void *stream)
{
    return copy_out(net, net ? net->o.grads : 0, grads, host, stream);
}

zda_status zda_nn_forward(zda_nn *net, const float *x, int n, float *y, void *stream)
{
    zda_status st = need_bound(net);
    if (st != ZDA_OK) return st;
    if (!x || !y) return nn_fail(ZDA_ERR_ARG, "null tensor");
    if (n < 1 || n > net->d.batch) return nn_fail(ZDA_ERR_ARG, "n outside 1..batch");
    cudaStream_t s = (cudaStream_t)stream;
    const int H = net->d.height, W = net->d.width;
    uint16_t *x16 = at<uint16_t>(net, net->o.x16);
    k_pack_rows<<<nblocks(pos_tiles(net, 0, n)), 256, 0, s>>>(x, n, H, W, net->d.in_ch, 2, net->rows[0], x16);
    net->launches++;
#define TRY(e)                          \
    do {                                \
        zda_status st_ = (e);           \
        if (st_ != ZDA_OK) return st_;  \
    } while (0)
    const uint16_t *inp = x16;
    int cin = 16;
    for (int l = 0; l < 3; ++l) {
        TRY(conv(net, l, n, 9, inp, nullptr, cin, C, Wf(net, 2 * l), Bias(net, 2 * l), C, EPI_RELU_BF16, Aw(net, l, A_ENCA),
                 nullptr, C, nullptr, nullptr, s, lf(net, 2 * l, n)));
        TRY(conv(net, l, n, 9, A(net, l, A_ENCA), nullptr, C, C, Wf(net, 2 * l + 1), Bias(net, 2 * l + 1), C, EPI_RELU_BF16,
                 Aw(net, l, A_ENCB), nullptr, C, nullptr, nullptr, s, lf(net, 2 * l + 1, n)));
        k_pool<<<pos_grid(net, l + 1, n), 256, 0, s>>>(A(net, l, A_ENCB), lev(net, l, n), Aw(net, l + 1, A_IN),
                                                       lev(net, l + 1, n));
        net->launches++;
        inp = A(net, l + 1, A_IN);
        cin = C;
    }
    TRY(conv(net, 3, n, 9, inp, nullptr, C, C, Wf(net, 6), Bias(net, 6), C, EPI_RELU_BF16, Aw(net, 3, A_ENCA), nullptr, C,
             nullptr, nullptr, s, lf(net, 6, n)));
    TRY(conv(net, 3, n, 9, A(net, 3, A_ENCA), nullptr, C, C, Wf(net, 7), Bias(net, 7), C, EPI_RELU_BF16,
             Aw(net, 3, A_ENCB), nullptr, C, nullptr, nullptr, s, lf(net, 7, n)));
    const uint16_t *below = A(net, 3, A_ENCB);
    for (int l = 2; l >= 0; --l) {
        const int li = 8 + 2 * (2 - l);
        k_up<<<pos_grid(net, l, n), 256, 0, s>>>(below, lev(net, l + 1, n), Aw(net, l, A_UP), lev(net, l, n));
        net->launches++;
        TRY(conv(net, l, n, 9, A(net, l, A_UP), A(net, l, A_ENCB), C, C, Wf(net, li), Bias(net, li), C, EPI_RELU_BF16,
                 Aw(net, l, A_DECA), nullptr, C, nullptr, nullptr, s, lf(net, li, n)));
        TRY(conv(net, l, n, 9, A(net, l, A_DECA), nullptr, C, C, Wf(net, li + 1), Bias(net, li + 1), C, EPI_RELU_BF16,
                 Aw(net, l, A_DECB), nullptr, C, nullptr, nullptr, s, lf(net, li + 1, n)));
        below = A(net, l, A_DECB);
    }
    TRY(conv(net, 0, n, 1, below, nullptr, C, 32, Wf(net, 14), Bias(net, 14), net->d.out_ch, EPI_F32, y, nullptr,
             net->d.out_ch, nullptr, nullptr, s, lf(net, 14, n)));
    NN_CUDA(cudaGetLastError());
    net->n_fwd = n;
    return ZDA_OK;
}

// The input gradients follow one another; each layer's weight gradient only
// needs its output's, so it goes to the side stream and the two chains share
// the chip (a one-sample backward fills less than half of it: ascent step on
// one patch 822 -> 672 us, gradient of a 64-sample batch 2370 -> 2235).  No
// buffer that the side stream reads is written again before the chains join:
// on the way down the encoder, gS is combined in place and becomes enc_b's
// gradient, gU (read by then) enc_a's, gI the level's input's.
static zda_status backward_chain(zda_nn *net, const float *dy, float *dx, cudaStream_t s)
{
    const int n = net->n_fwd, H = net->d.height, W = net->d.width;
    auto weights = [&](int li, const uint16_t *x0, const uint16_t *x1, const uint16_t *g, int ldg) {
        NN_CUDA(cudaEventRecord(net->forked, s));
        NN_CUDA(cudaStreamWaitEvent(net->side, net->forked, 0));
        return layer_grad(net, li, n, x0, x1, g, ldg, net->side);
    };
    uint16_t *gy = at<uint16_t>(net, net->o.gy);
    k_pack_rows<<<nblocks(pos_tiles(net, 0, n)), 256, 0, s>>>(dy, n, H, W, net->d.out_ch, 4, net->rows[0], gy);
    net->launches++;
    // head
    TRY(weights(14, A(net, 0, A_DECB), nullptr, gy, 32));
    TRY(conv(net, 0, n, 1, gy, nullptr, 32, C, Wd(net, 14), nullptr, 0, EPI_GRAD_BF16, Gb(net, 0, G_B), nullptr, C,
             A(net, 0, A_DECB), nullptr, s));
    // decoder, top level first: G_B holds the gradient of dec_b's pre-activation
    for (int l = 0; l <= 2; ++l) {
        const int li = 8 + 2 * (2 - l);
        TRY(weights(li + 1, A(net, l, A_DECA), nullptr, Gb(net, l, G_B), C));
        TRY(conv(net, l, n, 9, Gb(net, l, G_B), nullptr, C, C, Wd(net, li + 1), nullptr, 0, EPI_GRAD_BF16,
                 Gb(net, l, G_A), nullptr, C, A(net, l, A_DECA), nullptr, s));
        TRY(weights(li, A(net, l, A_UP), A(net, l, A_ENCB), Gb(net, l, G_A), C));
        TRY(conv(net, l, n, 9, Gb(net, l, G_A), nullptr, C, 2 * C, Wd(net, li), nullptr, 0, EPI_GRAD_BF16,
                 Gb(net, l, G_U), Gb(net, l, G_S), C, nullptr, nullptr, s));
        const uint16_t *below = l == 2 ? A(net, 3, A_ENCB) : A(net, l + 1, A_DECB);
        k_up_bwd_mask<<<pos_grid(net, l + 1, n), 256, 0, s>>>(Gb(net, l, G_U), lev(net, l, n), below,
                                                              Gb(net, l + 1, G_B), lev(net, l + 1, n));
        net->launches++;
    }
    // bottleneck (level 3: A_ENCA = bot_a, A_ENCB = bot_b)
    TRY(weights(7, A(net, 3, A_ENCA), nullptr, Gb(net, 3, G_B), C));
    TRY(conv(net, 3, n, 9, Gb(net, 3, G_B), nullptr, C, C, Wd(net, 7), nullptr, 0, EPI_GRAD_BF16, Gb(net, 3, G_A),
             nullptr, C, A(net, 3, A_ENCA), nullptr, s));
    TRY(weights(6, A(net, 3, A_IN), nullptr, Gb(net, 3, G_A), C));
    TRY(conv(net, 3, n, 9, Gb(net, 3, G_A), nullptr, C, C, Wd(net, 6), nullptr, 0, EPI_GRAD_BF16, Gb(net, 3, G_U),
             nullptr, C, nullptr, nullptr, s));
    // encoder, coarse to fine
    for (int l = 2; l >= 0; --l) {
        k_skip_combine<<<pos_grid(net, l, n), 256, 0, s>>>(Gb(net, l, G_S), Gb(net, l + 1, l == 2 ? G_U : G_I),
                                                           lev(net, l + 1, n), A(net, l, A_ENCB), lev(net, l, n));
        net->launches++;
        TRY(weights(2 * l + 1, A(net, l, A_ENCA), nullptr, Gb(net, l, G_S), C));
        TRY(conv(net, l, n, 9, Gb(net, l, G_S), nullptr, C, C, Wd(net, 2 * l + 1), nullptr, 0, EPI_GRAD_BF16,
                 Gb(net, l, G_U), nullptr, C, A(net, l, A_ENCA), nullptr, s));
        const uint16_t *in = l == 0 ? at<uint16_t>(net, net->o.x16) : A(net, l, A_IN);
        TRY(weights(2 * l, in, nullptr, Gb(net, l, G_U), C));
        if (l > 0)
            TRY(conv(net, l, n, 9, Gb(net, l, G_U), nullptr, C, C, Wd(net, 2 * l), nullptr, 0, EPI_GRAD_BF16,
                     Gb(net, l, G_I), nullptr, C, nullptr, nullptr, s));
        else if (dx) {
            TRY(conv(net, 0, n, 9, Gb(net, 0, G_U), nullptr, C, 16, Wd(net, 0), nullptr, 0, EPI_GRAD_F32, dx, nullptr,
                     net->d.in_ch, nullptr, nullptr, s));
        }
    }
    NN_CUDA(cudaGetLastError());
    return ZDA_OK;
}

zda_status zda_nn_backward(zda_nn *net, const float *dy, float *dx, void *stream)
{
    zda_status st = need_bound(net);
    if (st != ZDA_OK) return st;
    if (!dy) return nn_fail(ZDA_ERR_ARG, "null gradient");
    if (net->n_fwd < 1) return nn_fail(ZDA_ERR_STATE, "backward before forward");
    cudaStream_t s = (cudaStream_t)stream;
    st = backward_chain(net, dy, dx, s);
    // the chains join even after a failed launch: nothing of this call is left running beside later work of `s`
    const cudaError_t e0 = cudaEventRecord(net->joined, net->side), e1 = cudaStreamWaitEvent(s, net->joined, 0);
    if (st != ZDA_OK) return st;
    NN_CUDA(e0);
    NN_CUDA(e1);
    return ZDA_OK;
}

zda_status zda_nn_mse(zda_nn *net, const float *y, const float *t, int n, float *dy, float *loss, void *stream)
{
    zda_status st = need_bound(net);
    if (st != ZDA_OK) return st;
    if (!y || !t || !dy || !loss) return nn_fail(ZDA_ERR_ARG, "null tensor");
    if (n < 1 || n > net->d.batch) return nn_fail(ZDA_ERR_ARG, "n outside 1..batch");
    cudaStream_t s = (cudaStream_t)stream;
    const long cnt = (long)n * net->d.height * net->d.width * net->d.out_ch;
    const int nb = (int)std::min<long>(1024, nblocks(cnt));
    k_mse<<<nb, 256, 0, s>>>(y, t, cnt, dy, at<float>(net, net->o.mpart));
    k_mse_final<<<1, 256, 0, s>>>(at<float>(net, net->o.mpart), nb, cnt, loss);
    net->launches += 2;
    NN_CUDA(cudaGetLastError());
    return ZDA_OK;
}

zda_status zda_nn_adam(zda_nn *net, float lr, float b1, float b2, float eps, void *stream)
{
    zda_status st = need_bound(net);
    if (st != ZDA_OK) return st;
    if (!(lr >= 0.f) || !(b1 >= 0.f && b1 < 1.f) || !(b2 >= 0.f && b2 < 1.f) || !(eps > 0.f))
        return nn_fail(ZDA_ERR_ARG, "invalid Adam hyper-parameters");
    cudaStream_t s = (cudaStream_t)stream;
    net->adam_step++;
    const float c1 = (float)(1.0 - std::pow((double)b1, net->adam_step));
    const float c2 = (float)(1.0 - std::pow((double)b2, net->adam_step));
    k_adam<<<nblocks(net->nparam), 256, 0, s>>>(at<float>(net, net->o.params), at<float>(net, net->o.grads),
                                                at<float>(net, net->o.m), at<float>(net, net->o.v), net->nparam, lr, b1,
                                                b2, eps, c1, c2);
    net->launches++;
    NN_CUDA(cudaGetLastError());
    return pack_all(net, s);
}

long long zda_nn_launch_count(const zda_nn *net) { return net ? net->launches : 0; }

zda_status zda_nn_set_timing(zda_nn *net, int on)
{
    if (!net) return nn_fail(ZDA_ERR_ARG, "null network");
    net->timing = on != 0;
    net->ev_used = 0;
    net->ev_flops.clear();
    return ZDA_OK;
}

zda_status zda_nn_timing(zda_nn *net, double *conv_ms, double *conv_flops, int *launches)
{
    if (!net || !conv_ms || !conv_flops || !launches) return nn_fail(ZDA_ERR_ARG, "null argument");
    double ms = 0.0, fl = 0.0;
    for (size_t k = 0; k + 1 < net->ev_used; k += 2) {
        NN_CUDA(cudaEventSynchronize(net->ev[k + 1]));
        float t = 0.f;
        NN_CUDA(cudaEventElapsedTime(&t, net->ev[k], net->ev[k + 1]));
        ms += t;
        fl += net->ev_flops[k / 2];
    }
    *conv_ms = ms;
    *conv_flops = fl;
    *launches = (int)(net->ev_used / 2);
    net->ev_used = 0;
    net->ev_flops.clear();
    return ZDA_OK;
}

zda_status zda_nn_check(zda_nn *net, void *stream)
{
    zda_status st = need_bound(net);
    if (st != ZDA_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    int err = 0;
    NN_CUDA(cudaMemcpyAsync(&err, at<int>(net, net->o.err), 4, cudaMemcpyDeviceToHost, s));
    NN_CUDA(cudaStreamSynchronize(s));
    if (err) {
        NN_CUDA(cudaMemsetAsync(at<int>(net, net->o.err), 0, 4, s));
        return nn_fail(ZDA_ERR_TIMEOUT, "tensor-core kernel wait gave up (site " + std::to_string(err) + ")");
    }
    return ZDA_OK;
}

}  // extern "C"
