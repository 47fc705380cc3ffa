// Two leap-frog steps per launch (sm_103a): the default on large annular zones
// (even n_z and z-PML, real-radius r-PML; the rule is at zone creation).
//
// Why: a step of the split kernels moves 144 B per cell (each half reads six
// components and writes three), one fused step 96 B, two fused steps 96 B for
// both.  Measured per step (no source, no DFT): 300 x 320 x 160 cells 388 us by
// the split step with its E half on TMA tiles, 323 here; 144 x 128 x 160 89 (by
// pairs) and 81.  With source, DFT history and its flush, per step of a forward
// and adjoint run: 412 -> 362, 102 -> 93; a lens of five such zones and the axis
// zone (a split step in a lens) 404 -> 293 ms per iteration.
//
// What bounds it now: instructions and their latency, not memory (on the 300 x
// 320 x 160 zone: DRAM at 33 % of its peak, shared memory at 38 %, 31 % of issue
// slots with 12 warps per SM; without loads and stores it would take 232 of 330
// us).  Tried and slower: one z-cell per thread at twice the warps (419 us: the
// extra shared-memory instructions), the planes of a thread carried in
// registers over the loop (361; with spills 1364).
//
// A thread block owns a tile of phi rows x z-cells and streams along r over a
// range of radii; each thread holds one z-pair of one row of the tile or of
// its halo, and keeps what it needs of the radii behind in registers.  Four
// planes follow each other down the radii; at radius r
//   A   H1(r)   from E0(r), E0(r+1), H0(r)      (first step, H half)
//       barrier
//   B   E1(r)   from E0(r), H1(r), H1(r-1)      (first step, E half)
//       H2(r-1) from H1(r-1), E1(r-1), E1(r)    (second step, H half), stored
//       barrier
//   C   E2(r-1) from E1(r-1), H2(r-1), H2(r-2)  (second step, E half), stored
// so one pass reads the state once, writes it once and advances it by two
// steps.  Each later plane needs one row and one z-cell less around the tile;
// the halo starts two rows and one z-pair wide and is worked out again by
// every tile (33 % more threads than cells at 16 rows x 16 pairs, none in phi
// where a tile holds the whole wedge).  A range recomputes the two radii
// before it and the one after it.
//
// Neighbouring rows and z-cells are read from shared memory: a ring of four
// slots, slot r = {E(r+1), H(r)}, filled two radii ahead by 16-byte cp.async
// copies, each thread its own pair.  Planes are updated in place (H0 -> H1 ->
// H2, E0 -> E1) once their last reader has passed a barrier.  All accesses to
// a thread's own pair and to the rows beside it are contiguous over the warp.
// The state is ping-ponged between the two field buffers and two sets of CPML
// auxiliaries (a halo reads what its owner must not have overwritten yet).
// Auxiliaries in the z slabs travel in the ring; those of the r slabs are
// loaded where they apply, and their first-step values wait in shared memory.
//
// Across the wedge's seam rows keep their own phase on both sides; a value is
// turned by e^{+-i m tau} where it is used, as in the split step.
#include "zda_two.h"

#include <algorithm>

namespace zda {

namespace {

typedef unsigned long long u64;
__device__ __forceinline__ u64 bits(float2 a) { return *reinterpret_cast<u64 *>(&a); }
__device__ __forceinline__ float2 pair(u64 a) { return *reinterpret_cast<float2 *>(&a); }
__device__ __forceinline__ float2 both(float s) { return make_float2(s, s); }
__device__ __forceinline__ float2 padd(float2 a, float2 b)
{
    u64 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(bits(a)), "l"(bits(b)));
    return pair(r);
}
__device__ __forceinline__ float2 pmul(float2 a, float2 b)
{
    u64 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(bits(a)), "l"(bits(b)));
    return pair(r);
}
__device__ __forceinline__ float2 pfma(float2 a, float2 b, float2 c)
{
    u64 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(bits(a)), "l"(bits(b)), "l"(bits(c)));
    return pair(r);
}
__device__ __forceinline__ float2 psub(float2 a, float2 b)
{
    u64 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(bits(a)), "l"(bits(b)));
    return pair(r);
}

struct C2 { float2 a[2]; };                       // the z-pair (k, k + 1)

__device__ __forceinline__ C2 get(const float2 *p)
{
    const float4 v = *reinterpret_cast<const float4 *>(p);
    return C2{{make_float2(v.x, v.y), make_float2(v.z, v.w)}};
}
__device__ __forceinline__ void put(float2 *p, const C2 &c)
{
    *reinterpret_cast<float4 *>(p) = make_float4(c.a[0].x, c.a[0].y, c.a[1].x, c.a[1].y);
}
__device__ __forceinline__ C2 turn(float2 ph, const C2 &c) { return C2{{c_mul(ph, c.a[0]), c_mul(ph, c.a[1])}}; }
__device__ __forceinline__ C2 none() { return C2{{make_float2(0.f, 0.f), make_float2(0.f, 0.f)}}; }

__device__ __forceinline__ float rcp_hw(float x)  // the hardware reciprocal, as in the split E update
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ void cp16(const void *dst_smem, const void *src, bool on)      // zeros where off
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst_smem)),
                 "l"(src), "r"(on ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

constexpr int SLOTS = 4;

struct Trio { C2 r, p, z; };                      // the three components of a field on a pair

// Shared memory of a block of at most NT threads.  A component plane holds one
// pair per thread at a fixed stride, so a thread's accesses are one register
// plus constants.  Byte offsets; `pad` float2 before and after the ring take
// the reads of halo threads past the tile's edges, whose results nobody uses.
struct TwoLayout {
    int pad, tab, zp, rp, bytes;                  // radius table, z-CPML ring [SLOTS][4][rows x nzq], r-CPML [2][4][NT]
};
__host__ __device__ __forceinline__ TwoLayout two_layout(int nt, int npair, int nrow, int nzq, int radii, int has_r)
{
    TwoLayout L;
    L.pad = 2 * npair + 2;
    L.tab = ((2 * L.pad + SLOTS * 6 * 2 * nt) * 8 + 15) & ~15;
    L.zp = L.tab + radii * 64;
    L.rp = L.zp + SLOTS * 4 * nrow * nzq * 16;
    L.bytes = L.rp + (has_r ? 2 * 4 * nt * 16 : 0);
    return L;
}

template <int NT>
__global__ void __launch_bounds__(NT, NT > 192 ? 1 : 2) k_two(const __grid_constant__ TwoParams q, const int n)
{
    constexpr int SLAB = 2 * NT, SLOT = 6 * SLAB;  // float2
    extern __shared__ __align__(16) char smem[];
    const StepParams &p = q.p;
    const int nr = p.nr, nphi = p.nphi, nz = p.nz, npair = q.npair, tid = threadIdx.x;
    const TwoLayout L = two_layout(NT, npair, q.nrow, q.nzq, q.i_range + 4, p.pr_in + p.pr_out > 0);
    const int S = 2 * npair, o = 2 * tid;

    // ---- this thread's pair
    const int tk = blockIdx.x % q.tiles_k, tj = blockIdx.x / q.tiles_k;
    const int np = nz / 2;
    const int p0 = (int)((long long)tk * np / q.tiles_k), p1 = (int)((long long)(tk + 1) * np / q.tiles_k);
    const int j0 = (int)((long long)tj * nphi / q.tiles_j), j1 = (int)((long long)(tj + 1) * nphi / q.tiles_j);
    const int ib = blockIdx.y * q.i_range, ie = min(nr, ib + q.i_range);
    if (ib >= nr) return;
    const bool on = tid < q.nrow * npair;
    const int row = tid / npair, pq = tid - row * npair;
    const int k = 2 * (p0 - 1 + pq);
    int jw = q.full ? row : j0 - 2 + row;          // the row in the wedge
    if (jw < 0) jw += nphi;
    while (jw >= nphi) jw -= nphi;                 // rows past a ragged last tile, idle threads
    const bool live = on && k >= 0 && k < nz;
    const bool own = on && pq >= 1 && pq <= p1 - p0 && (q.full || (row >= 2 && row < j1 - j0 + 2));
    const int up = (q.full && row == nphi - 1) ? -(nphi - 1) * S : S;      // the row above / below
    const int dn = (q.full && row == 0) ? (nphi - 1) * S : -S;
    const bool turn_up = jw == nphi - 1, turn_dn = jw == 0;
    const uint32_t si = (uint32_t)nphi * nz, g0 = (uint32_t)jw * nz + (live ? k : 0);
    float2 *const ring = reinterpret_cast<float2 *>(smem) + L.pad + o;     // this thread's place in slot 0

    // z-PML: position among the tile's slab pairs; ring of the auxiliaries (hr, hp, er, ep at stride zstr)
    auto in_z = [&](int kk) { return kk >= 0 && kk < nz && (kk < p.pz || kk >= nz - p.pz); };
    const bool zs = live && in_z(k);
    int zi = 0;
    if (zs) {
        for (int w = 0; w < pq; ++w) zi += in_z(2 * (p0 - 1 + w)) ? 1 : 0;
        zi += row * q.nzq;
    }
    const int zstr = 2 * q.nrow * q.nzq, kz = k < p.pz ? k : k - (nz - 2 * p.pz);
    float2 *const zring = reinterpret_cast<float2 *>(smem + L.zp) + 2 * zi;
    // r-PML: this thread's values by parity of the radius (hp, hz, ep, ez at stride SLAB)
    float2 *const rbuf = reinterpret_cast<float2 *>(smem + L.rp) + o;

    // per-radius factors, doubled for the packed instructions: {hA hB}{hC -}{eA eB}{eC -} per radius ib - 2 ..
    const float dt = p.dt;
    float4 *const tab = reinterpret_cast<float4 *>(smem + L.tab);
    for (int t = tid; t < ie - ib + 4; t += blockDim.x) {
        const int i = min(max(ib - 2 + t, 0), nr - 1);
        const float irn = p.t.inv_r_n[i], irh = p.t.inv_r_h[i];
        const float hA = irn * p.inv_dphi, hB = -irh * p.inv_dphi, eA = irh * p.inv_dphi, eB = -irn * p.inv_dphi;
        tab[4 * t] = make_float4(hA, hA, hB, hB);
        tab[4 * t + 1] = make_float4(0.5f * irh, 0.5f * irh, 0.f, 0.f);
        tab[4 * t + 2] = make_float4(eA, eA, eB, eB);
        tab[4 * t + 3] = make_float4(0.5f * irn, 0.5f * irn, 0.f, 0.f);
    }
    // dt / eps of the node and cell planes of the pair, 0 where E is not updated (outside the grid; E_r and
    // E_phi at k = 0); in the design layer it follows the density
    float cn[2], cc[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        cn[u] = live && k + u > 0 ? dt * rcp_hw(p.t.a_n[k + u]) : 0.f;
        cc[u] = live ? dt * rcp_hw(p.t.a_c[k + u]) : 0.f;
    }
    const bool design = live && (p.t.d_n[k] != 0.f || p.t.d_n[k + 1] != 0.f || p.t.d_c[k] != 0.f || p.t.d_c[k + 1] != 0.f);
    const int su = live && p.src_mode != SRC_NONE ? p.src_k - k : -1;      // the pair's source cell (0, 1)
    const bool src = su == 0 || su == 1;
    const bool special = zs || src || design;
    const size_t plane = (size_t)nr * nphi, ndes = p.des ? plane * p.des_nk : 0;
    const bool hist = own && ((p.des && k + 1 >= p.des_k0 && k < p.des_k0 + p.des_nk) || (p.mon && (p.mon_k == k || p.mon_k == k + 1)));

    const float2 c_dz = both(p.inv_dz), c_ndz = both(-p.inv_dz), c_dr = both(p.inv_dr);
    const float2 c_dt = both(dt), c_ndt = both(-dt);
    auto rslab = [&](int i) { return i < p.pr_in ? i >= 0 : (i >= nr - p.pr_out && i < nr); };
    auto rx_at = [&](int i) {                      // the pair in the r-slab arrays
        const int ir = i < p.pr_in ? i : i - (nr - p.pr_in - p.pr_out);
        return (uint32_t)(ir * nphi + jw) * nz + k;
    };
    auto zx_at = [&](int i) { return (uint32_t)(i * nphi + jw) * (2 * p.pz) + kz; };

    // ring slot r: E0(r + 1), H0(r) and the z-slab auxiliaries of radius r
    auto issue = [&](int r, float2 *g, float2 *zq) {
        if (on) {
            const bool eo = live && (unsigned)(r + 1) < (unsigned)nr, ho = live && (unsigned)r < (unsigned)nr;
            const uint32_t gh = (uint32_t)r * si + g0, ge = gh + si;       // not used where off
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                cp16(g + c * SLAB, q.iE[c] + (eo ? ge : 0u), eo);
                cp16(g + (3 + c) * SLAB, q.iH[c] + (ho ? gh : 0u), ho);
            }
            if (zs && ho) {
                const uint32_t z = zx_at(r);
#pragma unroll
                for (int c = 0; c < 4; ++c) cp16(zq + c * zstr, q.iP[c] + z, true);
            }
        }
        cp_commit();
    };

    // H of the pair at radius i.  e: E there, e_i: E_phi, E_z one radius out, E: this thread's place in the
    // plane of e, zq: its z auxiliaries.  Level 0 reads the r-slab auxiliaries from memory; level 1 stores.
    auto update_h = [&](int i, int level, bool store, const Trio &e, const C2 &ep_i, const C2 &ez_i, const float2 *E,
                        float2 *zq, Trio &h) {
        C2 ez_j = get(E + 2 * SLAB + up), er_j = get(E + up);
        const float2 ep_k = E[SLAB + 2], er_k = E[2];
        if (turn_up) {
            ez_j = turn(p.bloch, ez_j);
            er_j = turn(p.bloch, er_j);
        }
        const float4 t0 = tab[4 * (i - ib + 2)], t1 = tab[4 * (i - ib + 2) + 1];
        const float2 hA = make_float2(t0.x, t0.y), hB = make_float2(t0.z, t0.w), hC = make_float2(t1.x, t1.y);
        float2 tr[2], tp[2], tz[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const float2 dzp = psub(u ? ep_k : e.p.a[1], e.p.a[u]), dzr = psub(u ? er_k : e.r.a[1], e.r.a[u]);
            const float2 dr0 = psub(ez_i.a[u], e.z.a[u]), drz = pmul(dr0, c_dr), df = psub(ep_i.a[u], e.p.a[u]), sf = padd(ep_i.a[u], e.p.a[u]);
            tr[u] = pmul(dzp, c_ndz);                  // the curl; dt joins it in the last fma
            tp[u] = pfma(dr0, c_dr, pmul(dzr, c_ndz));
            tz[u] = pfma(df, c_dr, pmul(sf, hC));       // the small term is the one rounded
            if (zs && (unsigned)i < (unsigned)nr) {
                const float2 b = both(__ldg(p.t.bz_h + k + u)), c = both(__ldg(p.t.cz_h + k + u));
                const float2 v = pfma(zq[u], b, pmul(pmul(dzp, c_dz), c)), w = pfma(zq[zstr + u], b, pmul(pmul(dzr, c_dz), c));
                tr[u] = psub(tr[u], v);
                tp[u] = psub(tp[u], w);
                if (level == 0) {
                    zq[u] = v;
                    zq[zstr + u] = w;
                } else if (store) {
                    q.oP[PS_HR_Z][zx_at(i) + u] = v;
                    q.oP[PS_HP_Z][zx_at(i) + u] = w;
                }
            }
            if (rslab(i) && live) {
                const uint32_t rx = rx_at(i) + u;
                float2 *rq = rbuf + (i & 1) * 4 * SLAB + u;
                const float2 br = both(__ldg(p.t.br_h + i)), cr = both(__ldg(p.t.cr_h + i));
                const float2 a0 = level ? rq[0] : q.iP[PS_HP_R][rx], a1 = level ? rq[SLAB] : q.iP[PS_HZ_R][rx];
                const float2 v = pfma(a0, br, pmul(drz, cr)), w = pfma(a1, br, pmul(tz[u], cr));
                tp[u] = padd(tp[u], v);
                tz[u] = padd(tz[u], w);
                if (level == 0) {
                    rq[0] = v;
                    rq[SLAB] = w;
                } else if (store) {
                    q.oP[PS_HP_R][rx] = v;
                    q.oP[PS_HZ_R][rx] = w;
                }
            }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            tr[u] = pfma(psub(ez_j.a[u], e.z.a[u]), hA, tr[u]);
            tz[u] = pfma(psub(er_j.a[u], e.r.a[u]), hB, tz[u]);
            h.r.a[u] = pfma(tr[u], c_ndt, h.r.a[u]);
            h.p.a[u] = pfma(tp[u], c_dt, h.p.a[u]);
            h.z.a[u] = pfma(tz[u], c_ndt, h.z.a[u]);
        }
    };
    // E of the pair at radius i (0 <= i < n_r).  h: H there, hp_i, hz_i: one radius in, H: this thread's place
    // in the plane of h, zq: its z auxiliaries.
    auto update_e = [&](int i, int level, bool store, const Trio &h, const C2 &hp_i, const C2 &hz_i, const float2 *H,
                        float2 *zq, Trio &e) {
        C2 hz_j = get(H + 2 * SLAB + dn), hr_j = get(H + dn);
        const float2 hp_k = H[SLAB - 1], hr_k = H[-1];
        if (turn_dn) {
            hz_j = turn(p.bloch_inv, hz_j);
            hr_j = turn(p.bloch_inv, hr_j);
        }
        const float4 t0 = tab[4 * (i - ib + 2) + 2], t1 = tab[4 * (i - ib + 2) + 3];
        const float2 eA = make_float2(t0.x, t0.y), eB = make_float2(t0.z, t0.w), eC = make_float2(t1.x, t1.y);
        float2 tr[2], tp[2], tz[2], dzp[2], dzr[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            dzp[u] = psub(h.p.a[u], u ? h.p.a[0] : hp_k);
            dzr[u] = psub(h.r.a[u], u ? h.r.a[0] : hr_k);
            const float2 dr0 = psub(hz_i.a[u], h.z.a[u]), drz = pmul(dr0, c_dr);          // minus d H_z / dr
            const float2 df = psub(h.p.a[u], hp_i.a[u]), sf = padd(h.p.a[u], hp_i.a[u]);
            tp[u] = pfma(dr0, c_dr, pmul(dzr[u], c_dz));
            tz[u] = pfma(df, c_dr, pmul(sf, eC));
            if (rslab(i) && live) {
                const uint32_t rx = rx_at(i) + u;
                float2 *rq = rbuf + ((i & 1) * 4 + 2) * SLAB + u;
                const float2 br = both(__ldg(p.t.br_n + i));
                const float cr = __ldg(p.t.cr_n + i);
                const float2 a0 = level ? rq[0] : q.iP[PS_EP_R][rx], a1 = level ? rq[SLAB] : q.iP[PS_EZ_R][rx];
                const float2 v = pfma(a0, br, pmul(drz, both(-cr))), w = pfma(a1, br, pmul(tz[u], both(cr)));
                tp[u] = psub(tp[u], v);
                tz[u] = padd(tz[u], w);
                if (level == 0) {
                    rq[0] = v;
                    rq[SLAB] = w;
                } else if (store) {
                    q.oP[PS_EP_R][rx] = v;
                    q.oP[PS_EZ_R][rx] = w;
                }
            }
            tr[u] = pfma(dzp[u], c_ndz, pmul(psub(h.z.a[u], hz_j.a[u]), eA));
            tz[u] = pfma(psub(h.r.a[u], hr_j.a[u]), eB, tz[u]);
        }
        float cr_[2] = {cn[0], cn[1]}, cp_[2] = {cn[0], cn[1]}, cz_[2] = {cc[0], cc[1]};
        if (special) {
            if (zs) {
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const float2 b = both(__ldg(p.t.bz_n + k + u)), c = both(__ldg(p.t.cz_n + k + u));
                    const float2 v = pfma(zq[2 * zstr + u], b, pmul(pmul(dzp[u], c_dz), c));
                    const float2 w = pfma(zq[3 * zstr + u], b, pmul(pmul(dzr[u], c_dz), c));
                    tr[u] = psub(tr[u], v);
                    tp[u] = padd(tp[u], w);
                    if (level == 0) {
                        zq[2 * zstr + u] = v;
                        zq[3 * zstr + u] = w;
                    } else if (store) {
                        q.oP[PS_ER_Z][zx_at(i) + u] = v;
                        q.oP[PS_EP_Z][zx_at(i) + u] = w;
                    }
                }
            }
            if (design) {
                const uint32_t ij = (uint32_t)i * nphi + jw;
                const float rb0 = __ldg(p.rb_r + ij), rb1 = __ldg(p.rb_p + ij), rb2 = __ldg(p.rb_z + ij);
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const float an = __ldg(p.t.a_n + k + u), d = __ldg(p.t.d_n + k + u);
                    if (k + u > 0) {
                        cr_[u] = dt * rcp_hw(an + d * rb0);
                        cp_[u] = dt * rcp_hw(an + d * rb1);
                    }
                    cz_[u] = dt * rcp_hw(__ldg(p.t.a_c + k + u) + __ldg(p.t.d_c + k + u) * rb2);
                }
            }
            if (src) {
                const float2 pn = __ldg(p.t.ph_n + jw), ph = __ldg(p.t.ph_h + jw);
                float2 jr, jp;
                if (p.src_mode == SRC_PLANE_WAVE) {    // m = +1 part of an x-polarised sheet
                    const float a = __ldg(p.t.pulse + n + level) * p.src_scale;
                    jr = c_scale(pn, a);
                    jp = make_float2(-ph.y * a, ph.x * a);
                } else {
                    const float2 *sr = p.src_rad + (size_t)level * 2 * nr;
                    jr = c_mul(pn, sr[i]);
                    jp = c_mul(ph, sr[nr + i]);
                }
#pragma unroll
                for (int u = 0; u < 2; ++u)
                    if (u == su) {
                        tr[u] = psub(tr[u], jr);
                        tp[u] = psub(tp[u], jp);
                    }
            }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            e.r.a[u] = pfma(tr[u], both(cr_[u]), e.r.a[u]);
            if (i > 0) {
                e.p.a[u] = pfma(tp[u], both(cp_[u]), e.p.a[u]);
                e.z.a[u] = pfma(tz[u], both(cz_[u]), e.z.a[u]);
            }
        }
        if (hist && store) {                       // history slot of the time-blocked DFT
            float2 *hs = p.dft_hist + (size_t)((n + level) % DFT_BLOCK) * p.dft_ne;
            const size_t ij = (size_t)i * nphi + jw;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int dk = k + u - p.des_k0;
                if (p.des && dk >= 0 && dk < p.des_nk) {
                    float2 *d = hs + ij * p.des_nk + dk;
                    d[0] = e.r.a[u];
                    d[ndes] = e.p.a[u];
                    d[2 * ndes] = e.z.a[u];
                }
                if (p.mon && k + u == p.mon_k) {
                    hs[3 * ndes + ij] = e.r.a[u];
                    hs[3 * ndes + plane + ij] = e.p.a[u];
                }
            }
        }
    };

    // A thread's own planes wait in its own places of the ring: carried over the loop in registers they
    // spill, and what shared memory leaves of L1 does not hold the spills.
    auto trio = [&](const float2 *f) { return Trio{get(f), get(f + SLAB), get(f + 2 * SLAB)}; };
    auto keep = [&](float2 *f, const Trio &t) {
        put(f, t.r);
        put(f + SLAB, t.p);
        put(f + 2 * SLAB, t.z);
    };
    const int zslot = 4 * zstr;
    const int r0 = ib - 2;
    // slots of radii r - 2, r - 1, r, r + 1 (r + 2 takes the first one's place) and their z auxiliaries
    float2 *g2 = ring + 3 * SLOT, *g1 = ring, *g = ring + SLOT, *gn = ring + 2 * SLOT;
    float2 *z2 = zring + 3 * zslot, *z1 = zring, *z = zring + zslot, *zn = zring + 2 * zslot;
    issue(r0 - 1, g1, z1);
    issue(r0, g, z);
    issue(r0 + 1, gn, zn);
    cp_wait<1>();
    __syncthreads();

    for (int r = r0; r <= ie; ++r) {
        cp_wait<1>();                              // this thread's part of slot r
        // ---- A
        const Trio e0 = trio(g1);
        Trio h1 = trio(g + 3 * SLAB);
        update_h(r, 0, false, e0, get(g + SLAB), get(g + 2 * SLAB), g1, z, h1);
        keep(g + 3 * SLAB, h1);
        __syncthreads();
        // ---- B
        const Trio h1p = trio(g1 + 3 * SLAB);
        Trio e1 = e0;                              // outside the grid E stays 0 (conducting walls)
        if ((unsigned)r < (unsigned)nr) update_e(r, 0, own && r >= ib && r < ie, h1, h1p.p, h1p.z, g + 3 * SLAB, z, e1);
        keep(g1, e1);
        const bool mine = own && r - 1 >= ib;      // r - 1 < ie always
        Trio e2 = trio(g2), h2 = h1p;
        update_h(r - 1, 1, mine, e2, e1.p, e1.z, g2, z1, h2);
        const C2 h2p = get(g2 + 4 * SLAB), h2z = get(g2 + 5 * SLAB);       // H2 one radius in
        keep(g1 + 3 * SLAB, h2);
        const uint32_t w = (uint32_t)(r - 1) * si + g0;
        if (mine) {
            put(q.oH[0] + w, h2.r);
            put(q.oH[1] + w, h2.p);
            put(q.oH[2] + w, h2.z);
        }
        __syncthreads();
        // ---- C
        issue(r + 2, g2, z2);
        if (mine) {
            update_e(r - 1, 1, true, h2, h2p, h2z, g1 + 3 * SLAB, z1, e2);
            put(q.oE[0] + w, e2.r);
            put(q.oE[1] + w, e2.p);
            put(q.oE[2] + w, e2.z);
        }
        float2 *const t = g2, *const tz_ = z2;
        g2 = g1; g1 = g; g = gn; gn = t;
        z2 = z1; z1 = z; z = zn; zn = tz_;
    }
    cp_wait<0>();
}

}  // namespace

bool two_applies(const StepParams &p)
{
    return !p.bor && !p.rpml_metric && p.nz % 2 == 0 && p.pz % 2 == 0 && p.nz >= 4;
}

TwoPlan two_plan(const StepParams &p, int rows, int ranges, int sms, size_t smem_limit)
{
    TwoPlan best;
    if (!two_applies(p)) return best;
    const int full = p.nphi <= rows + 4 ? 1 : 0;
    const int tiles_j = full ? 1 : (p.nphi + rows - 1) / rows;
    const int nrow = full ? p.nphi : (p.nphi + tiles_j - 1) / tiles_j + 4;
    const int np = p.nz / 2;
    double best_cost = 1e30;
    for (int tiles_k = 1; tiles_k <= np; ++tiles_k) {
        const int npair = (np + tiles_k - 1) / tiles_k + 2;
        if (nrow * npair > TWO_THREADS || (tiles_k > 1 && npair < 6)) continue;
        const int nt = nrow * npair > 192 ? TWO_THREADS : 192;
        TwoPlan t;
        t.tiles_j = tiles_j; t.tiles_k = tiles_k; t.full = full; t.nrow = nrow; t.npair = npair;
        for (int a = 0; a < tiles_k; ++a) {
            const int p0 = (int)((long long)a * np / tiles_k);
            int nq = 0;
            for (int w = 0; w < npair; ++w) {
                const int k = 2 * (p0 - 1 + w);
                nq += k >= 0 && k < p.nz && (k < p.pz || k >= p.nz - p.pz) ? 1 : 0;
            }
            t.nzq = std::max(t.nzq, nq);
        }
        const int r_lo = ranges > 0 ? ranges : 1, r_hi = ranges > 0 ? ranges : std::max(1, p.nr / 8);
        for (int nrg = r_lo; nrg <= r_hi; ++nrg) {
            const int len = (p.nr + nrg - 1) / nrg;
            const TwoLayout L = two_layout(nt, npair, nrow, t.nzq, len + 4, p.pr_in + p.pr_out > 0);
            if ((size_t)L.bytes > smem_limit) continue;
            // blocks of an SM by shared memory and by registers (168 a thread)
            const int occ = std::max(1, std::min((int)((smem_limit + 1024) / (L.bytes + 1024)), 65536 / (168 * nt)));
            const long long blocks = (long long)tiles_j * tiles_k * ((p.nr + len - 1) / len);
            // blocks differ (slabs, design layer): more than one wave of them queues up with half a block to
            // spare, a single wave waits for its slowest (144 x 128 x 160 cells, us per step of a run at 1 to 6 ranges:
            // 187, 115, 93, 117, 107, 98)
            const double slots = (double)sms * occ, waves = blocks <= slots ? 1.2 : blocks / slots + 0.6;
            // a radius costs its serial chain and little for each thread more (over 120 zones 2.8 us at 288 threads,
            // 3.0 at 384), and longer the more of the z-pairs lie in the PML (3.0 us at a tenth, 3.8 at a quarter)
            const double per_radius = (950.0 + 1.22 * occ * t.threads()) * (1.0 + 1.8 * 2 * p.pz / p.nz);
            const double cost = waves * (len + 5.0) * per_radius;
            if (cost < best_cost) {
                best_cost = cost;
                best = t;
                best.cost = cost;
                best.ranges = (p.nr + len - 1) / len;
                best.smem = (size_t)L.bytes;
            }
        }
    }
    return best;
}

cudaError_t launch_two(const TwoPlan &pl, const TwoParams &q0, int n, cudaStream_t s)
{
    TwoParams q = q0;
    q.tiles_j = pl.tiles_j; q.tiles_k = pl.tiles_k;
    q.full = pl.full; q.nrow = pl.nrow; q.npair = pl.npair; q.nzq = pl.nzq;
    q.i_range = (q.p.nr + pl.ranges - 1) / pl.ranges;
    auto kern = pl.nrow * pl.npair > 192 ? k_two<TWO_THREADS> : k_two<192>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pl.smem);
    if (e != cudaSuccess) return e;
    kern<<<dim3(pl.tiles_j * pl.tiles_k, pl.ranges), pl.threads(), pl.smem, s>>>(q, n);
    return cudaGetLastError();
}

}  // namespace zda
