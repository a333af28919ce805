// lpm_advance.cuh - the particle step of the paper's main loop (Sec. 3.2, Eq. 1-2),
// fused over a whole segment of steps with the particle state in registers, in-kernel
// deposition, and the concentration snapshot (every n-th step) at the segment end.
// Instantiated per block size in lpm_advance_b*.cu.
#pragma once

#include <mutex>

#include "lpm_device.cuh"
#include "lpm_launch.h"

namespace lpm {

constexpr int KEY_NONE = -1;
constexpr int KEY_OUT = -2;

// Warp-aggregated 64-bit fixed-point accumulation: lanes holding the same key add their
// values once through the lowest lane of the group (key KEY_NONE: nothing; KEY_OUT: the
// out-of-grid counter). Every lane of the warp must call it.
__device__ __forceinline__ void warp_accumulate(int key, unsigned long long v,
                                                unsigned long long *grid,
                                                unsigned long long *out_ctr,
                                                unsigned long long *s_warp, long long n_cells,
                                                unsigned int *err)
{
    const int lane = threadIdx.x & 31;
    const unsigned peers = __match_any_sync(0xffffffffu, key);
    s_warp[lane] = v;
    __syncwarp();
    if (key != KEY_NONE && lane == __ffs(peers) - 1) {
        unsigned long long sum = 0;
        unsigned m = peers;
        while (m) {
            const int b = __ffs(m) - 1;
            sum += s_warp[b];
            m &= m - 1;
        }
        if (key == KEY_OUT) atomicAdd(out_ctr, sum);
        else if (key < n_cells) atomicAdd(grid + key, sum);
        else atomicOr(err, ERR_INDEX);
    }
    __syncwarp();
}

// The same over the grids of all scenarios (grid_all [n_scen][cells]): key = scenario *
// n_cells + cell, or -2 - scenario for that scenario's counter `out` (-1: nothing).
__device__ __forceinline__ void warp_accumulate_scen(long long key, unsigned long long v,
                                                     const StepParams &P,
                                                     unsigned long long *grid_all, int out,
                                                     unsigned long long *s_warp, long long n_cells)
{
    const int lane = threadIdx.x & 31;
    const unsigned peers = __match_any_sync(0xffffffffu, key);
    s_warp[lane] = v;
    __syncwarp();
    if (key != -1 && lane == __ffs(peers) - 1) {
        unsigned long long sum = 0;
        unsigned m = peers;
        while (m) {
            const int b = __ffs(m) - 1;
            sum += s_warp[b];
            m &= m - 1;
        }
        if (key >= 0) {
            if (key < n_cells * P.n_scen) atomicAdd(grid_all + key, sum);
            else atomicOr(P.err, ERR_INDEX);
        } else {
            atomicAdd(P.ctr_all + (long long)out * P.ctr_stride + (-2 - key), sum);
        }
    }
    __syncwarp();
}

// Adds v to counter `which` of scenario s (s < 0: nothing), one atomic per scenario present
// in the warp. Every lane of the warp must call it.
__device__ __forceinline__ void warp_count_scen(int s, unsigned long long v, int which,
                                                const StepParams &P, unsigned long long *s_warp)
{
    const int lane = threadIdx.x & 31;
    const unsigned peers = __match_any_sync(0xffffffffu, s);
    s_warp[lane] = v;
    __syncwarp();
    if (s >= 0 && lane == __ffs(peers) - 1) {
        unsigned long long sum = 0;
        unsigned m = peers;
        while (m) {
            const int b = __ffs(m) - 1;
            sum += s_warp[b];
            m &= m - 1;
        }
        if (sum) atomicAdd(P.ctr_all + (long long)which * P.ctr_stride + s, sum);
    }
    __syncwarp();
}

// The scenario's perturbation of (u, v) at (x, y, t_k) on level cell k with fraction c:
// its phases and amplitudes are one 32-byte row msc (see StepParams::mode_sc).
__device__ __forceinline__ void mode_wind(const StepParams &P, const float *msc, int k, float c,
                                          float x, float y, float tk, float &du, float &dv)
{
    float4 ph, am;
    ld_pair(reinterpret_cast<const float4 *>(msc), ph, am);
    const float pa[MAX_MODES] = {ph.x, ph.y, ph.z, ph.w};
    const float aa[MAX_MODES] = {am.x, am.y, am.z, am.w};
    float su = 0.0f, sv = 0.0f;
#pragma unroll
    for (int m = 0; m < MAX_MODES; ++m) {
        if (m < P.n_modes) {
            // phase in cycles, reduced exactly to [-1/2, 1/2]; the hardware sine on
            // [-pi, pi] errs by less than 5e-7 (a velocity error of that fraction of the
            // amplitude)
            const float r = fmaf(P.mode_fx[m], x, fmaf(P.mode_fy[m], y, fmaf(P.mode_om[m], tk, pa[m])));
            const float as = aa[m] * __sinf(6.28318548f * (r - rintf(r)));
            su = fmaf(as, P.mode_eu[m], su);
            sv = fmaf(as, P.mode_ev[m], sv);
        }
    }
    const float pz = fmaf(c, P.mode_prof[k + 1] - P.mode_prof[k], P.mode_prof[k]);
    du = pz * su;
    dv = pz * sv;
}

// Concentration-grid cell of a position, or KEY_OUT outside the grid.
__device__ __forceinline__ int grid_cell(const StepParams &P, float x, float y, float z)
{
    const int ix = grid_axis(x, P.gx0, P.ginv_dx);
    const int iy = grid_axis(y, P.gy0, P.ginv_dy);
    const int iz = grid_axis(z, P.gz0, P.ginv_dz);
    if (ix >= 0 && ix < P.cx && iy >= 0 && iy < P.cy && iz >= 0 && iz < P.cz)
        return (iz * P.cy + iy) * P.cx + ix;
    return KEY_OUT;
}

// Initial mass of a particle released at step sp (the scenario's table, Sec. 3.2).
__device__ __forceinline__ float m0_of(const StepParams &P, const ScenDev &sc, int sp)
{
    int ix = sc.m0_off + (sp - sc.rel_first);
    if (!LPM_IN_BOUNDS(P.err, ix >= 0 && ix < P.n_m0)) ix = 0;
    return __ldg(P.m0 + ix);
}

__device__ __forceinline__ float mass_at(const StepParams &P, const ScenDev &sc, int sp, int k_end)
{
    // decayed mass at the end of step k_end (age (k_end + 1 - s_p) dt), Sec. 2 / Sec. 3.2
    const float m0 = m0_of(P, sc, sp);
    const float age = (float)(k_end + 1 - sp) * P.dt;
    return m0 * expf(-P.lambda * age);
}

// Daughters of a decay chain deposited with their parent at step k (cell of the 2D grid).
static __device__ __noinline__ void deposit_species(const StepParams &P, const ScenDev &sc, int scen,
                                             int sp, int k, int kind, int cell2)
{
    const float m0 = m0_of(P, sc, sp);
    const float age = (float)(k + 1 - sp) * P.dt;
    const long long plane = (long long)P.cx * P.cy;
    for (int j = 1; j < P.n_species; ++j) {
        const unsigned long long v = to_fixed(m0 * chain_amount(P, j, age), sc.scale);
        atomicAdd(P.sp_dep_all + (((long long)(j - 1) * P.n_scen + scen) * 2 + kind) * plane + cell2, v);
    }
}

// The deposition words of a particle: one Philox block (stream 1) serves a pair of steps,
// words 0 and 1 for the even step, 2 and 3 for the odd one (dry, then wet test). A step
// runner may keep the odd step's words from the even step in a DepCache; it has to fill it
// (dep_begin) before a first step that is odd.
struct DepCache {
    uint32_t c, d;                   // words of the odd step of the current pair
};

__device__ __forceinline__ U4 dep_block(const StepParams &P, unsigned long long gid, int k)
{
    return philox4x32_10_rk((uint32_t)gid, (uint32_t)(gid >> 32), (uint32_t)(k >> 1), 1u, P.rk);
}

__device__ __forceinline__ void dep_begin(const StepParams &P, unsigned long long gid, int k,
                                          DepCache &dc)
{
    dc.c = dc.d = 0u;
    if ((P.t_dry | P.t_wet) && (k & 1)) {
        const U4 w = dep_block(P, gid, k);
        dc.c = w.c;
        dc.d = w.d;
    }
}

__device__ __forceinline__ void dep_words(const StepParams &P, unsigned long long gid, int k,
                                          DepCache *dc, uint32_t &w_dry, uint32_t &w_wet)
{
    const bool odd = (k & 1) != 0;
    if (dc) {
        w_dry = dc->c;
        w_wet = dc->d;
        if (!odd) {
            const U4 w = dep_block(P, gid, k);
            w_dry = w.a;
            w_wet = w.b;
            dc->c = w.c;
            dc->d = w.d;
        }
    } else {
        const U4 w = dep_block(P, gid, k);
        w_dry = odd ? w.c : w.a;
        w_wet = odd ? w.d : w.b;
    }
}

// The draws of the steps k and k + 1 of a particle, for DRAWS_GIVEN: the three normals, and in
// w the deposition tests' outcomes (bit 0 dry, bit 1 wet). dc holds the odd step's words where
// k is odd (dep_begin) and is left ready for k + 2. Free of branches, so that the two steps'
// chains overlap.
__device__ __forceinline__ void draw_pair(const StepParams &P, unsigned long long gid, int k,
                                          DepCache &dc, float4 &a, float4 &b)
{
    const U4 wa = philox4x32_10_rk((uint32_t)gid, (uint32_t)(gid >> 32), (uint32_t)k, 0u, P.rk);
    const U4 wb =
        philox4x32_10_rk((uint32_t)gid, (uint32_t)(gid >> 32), (uint32_t)(k + 1), 0u, P.rk);
    normals3(wa, a.x, a.y, a.z);
    normals3(wb, b.x, b.y, b.z);
    uint32_t fa = 0u, fb = 0u;
    if (P.t_dry | P.t_wet) {
        const bool odd = (k & 1) != 0;
        const U4 w = dep_block(P, gid, k + 1);   // of the even one of the two steps
        fa = ((odd ? dc.c : w.a) < P.t_dry ? 1u : 0u) | ((odd ? dc.d : w.b) < P.t_wet ? 2u : 0u);
        fb = ((odd ? w.a : w.c) < P.t_dry ? 1u : 0u) | ((odd ? w.b : w.d) < P.t_wet ? 2u : 0u);
        dc.c = w.c;
        dc.d = w.d;
    }
    a.w = __uint_as_float(fa);
    b.w = __uint_as_float(fb);
}

enum { DRAWS_LAST = 0, DRAWS_FIRST = 1, DRAWS_GIVEN = 2 };

// Per-step quantities shared by every particle of a tile.
struct StepTime {
    int k;
    int h0;                          // first slab of the time pair (not read by the plain step)
    float f;                         // fraction between the slabs
    const float4 *pair;              // time pair of the step
    float du, dv;                    // wind offset of the scenario + bias
};

// The wind offset of (hourly) row `wo` between slabs h0 and h1, plus the bias.
__device__ __forceinline__ float2 step_offset(const StepParams &P, const float2 *wo, int h0, int h1,
                                              float f)
{
    float2 d = make_float2(P.bias_u, P.bias_v);
    if (wo) {
        const float2 o0 = __ldg(wo + h0);
        const float2 o1 = __ldg(wo + h1);
        d.x += fmaf(f, o1.x - o0.x, o0.x);
        d.y += fmaf(f, o1.y - o0.y, o0.y);
    }
    return d;
}

template <bool ONCE = false>
__device__ __forceinline__ StepTime step_time(const StepParams &P, const float2 *wind_offset, int k)
{
    StepTime T;
    T.k = k;
    TimeSlab ts = time_slab(P, step_since<ONCE>(P, k));
    if (!LPM_IN_BOUNDS(P.err, ts.h0 >= 0 && ts.h0 < P.n_pair)) ts.h0 = 0;
    T.h0 = ts.h0;
    T.f = ts.f;
    T.pair = P.pair + (long long)ts.h0 * P.slab * 2;
    const float2 d = step_offset(P, wind_offset, ts.h0, ts.h1, ts.f);
    T.du = d.x;
    T.dv = d.y;
    return T;
}

// Step times of a launch are the same for every particle: each block computes those of its
// (at most STEP_TAB) steps once with step_time and keeps them in shared memory, 24 bytes a
// step; step_time_tab reads one back (measured: the per-particle step_time cost 3.5 % of the
// step). HOUR: h0 is read too (gridded K_h, Eq. 3 columns, scenarios' wind offsets).
struct StepTable {
    float4 a[STEP_TAB];              // pair address (64 bits), f, du
    float2 b[STEP_TAB];              // dv, h0
};

__device__ __forceinline__ void step_table_set(StepTable &tab, int i, const StepTime &T)
{
    const unsigned long long p = reinterpret_cast<unsigned long long>(T.pair);
    tab.a[i] = make_float4(__uint_as_float((unsigned int)p), __uint_as_float((unsigned int)(p >> 32)),
                           T.f, T.du);
    tab.b[i] = make_float2(T.dv, __int_as_float(T.h0));
}

template <bool HOUR>
__device__ __forceinline__ StepTime step_time_tab(uint32_t tab, int i, int k)
{
    const float4 a = ld_shared4(tab + 16 * i);
    const float2 b = ld_shared2(tab + 16 * STEP_TAB + 8 * i);
    StepTime T;
    T.k = k;
    T.f = a.z;
    T.pair = reinterpret_cast<const float4 *>((unsigned long long)__float_as_uint(a.x) |
                                              ((unsigned long long)__float_as_uint(a.y) << 32));
    T.du = a.w;
    T.dv = b.x;
    T.h0 = HOUR ? __float_as_int(b.y) : 0;
    return T;
}

// Weather at a point from the time-paired records: 8 spatial corners, each one 32-byte
// load of (slab h, slab h+1 - slab h), blended in time, then in x, y and z. With the
// boundary-layer columns (EXT and blp), K_z and its derivative come from Eq. 3 instead
// (4 more 32-byte loads of the time-paired (u*, 1/L, H_z) at the cell's corner columns,
// bilinear in x, y); with msc (MODES) the scenario's perturbation modes are added to
// (u, v). Only the EXT or MODES instantiations carry that code.
template <bool EXT, class LEV, bool MODES, bool FIELDS>
__device__ __forceinline__ Met sample_met_pair(const StepParams &P, const LEV &L, const StepTime &T,
                                               float x, float y, float z, const float *msc)
{
    const float4 *pair = T.pair;
    const float f = T.f;
    int i, j, k;
    float a, b, c;
    axis(x, P.x0, P.inv_dx, P.nx2, i, a);
    axis(y, P.y0, P.inv_dy, P.ny2, j, b);
    level(P, L, z, k, c);
    if (!LPM_IN_BOUNDS(P.err, i >= 0 && i <= P.nx - 2 && j >= 0 && j <= P.ny - 2 && k >= 0 &&
                                  k <= P.nz - 2))
        i = j = k = 0;
    // x first (the x + 1 record is the next line), then the two slots of rows and of levels
    const Corners q = cell_corners(P, i, j, k, b, c);
    const F2 ff = pack2(f, f), aa = pack2(a, a), bb = pack2(q.b, q.b);
    Rec4 yl[2];
#pragma unroll
    for (int l = 0; l < 2; ++l) {
        Rec4 xr[2];
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            const float4 *p = record_at<32>(pair, q.rec[2 * l + m]);
            xr[m] = lerp4(ld_blend(p, ff), ld_blend(p + 8, ff), aa);
        }
        yl[l] = lerp4s(xr[0], xr[1], bb, q.sy);
    }
    const float4 r = unpack4(lerp4s(yl[0], yl[1], pack2(q.c, q.c), q.sz));
    Met m;
    m.u = r.x;
    m.v = r.y;
    m.w = r.z;
    if (MODES && msc) {
        float du, dv;
        mode_wind(P, msc, k, c, x, y, step_start(P, T.k), du, dv);
        m.u += du;
        m.v += dv;
    }
    if (EXT && P.blpair) {
        const float4 *blp = P.blpair + (long long)T.h0 * P.nx * P.ny * 2;
        const F2 b2 = pack2(b, b);
        Rec4 xr[2];
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            const float4 *p = record_at<32>(blp, (unsigned int)((j + m) * P.nx + i));
            xr[m] = lerp4(ld_blend(p, ff), ld_blend(p + 2, ff), aa);
        }
        const float4 col = unpack4(lerp4(xr[0], xr[1], b2));
        kz_eq3(col.x, col.y, col.z, P.kz_min, z, m.kz, m.dkz);
    } else {
        m.kz = fmaxf(r.w, 0.0f);
        // the vertical derivative only where a drift term reads it (the drift-corrected
        // walk and the Langevin variant)
        m.dkz = 0.0f;
        if ((FIELDS && P.drift) || (EXT && P.langevin)) {
            const bool inside = z >= L.z_lo && z <= L.z_hi;
            const float d = unpack2(sub2(yl[1].zw, yl[0].zw)).y;
            m.dkz = inside ? (q.sz ? -d : d) * level_entry(P, L, k).y : 0.0f;
        }
    }
    if (FIELDS && P.khpair) {
        const float2 *khp = P.khpair + (long long)T.h0 * P.slab;
        float ey[2];
#pragma unroll
        for (int l = 0; l < 2; ++l) {
            float ex[2];
#pragma unroll
            for (int mm = 0; mm < 2; ++mm) {
                const float2 *p = record_at<8>(khp, q.rec[2 * l + mm]);
                const float2 v0 = __ldg(p), v1 = __ldg(p + 4);
                const float e0 = fmaf(f, v0.y, v0.x), e1 = fmaf(f, v1.y, v1.x);
                ex[mm] = fmaf(a, e1 - e0, e0);
            }
            ey[l] = lerps(ex[0], ex[1], q.b, q.sy);
        }
        m.kh = fmaxf(lerps(ey[0], ey[1], q.c, q.sz), 0.0f);
    } else {
        m.kh = 0.0f;
    }
    return m;
}

// One step of one active particle (Sec. 3.2 main loop: weather at the old position, K,
// wind then random walk by Eq. 1-2, reflection, lateral exit, dry then wet deposition).
// Updates (x, y, z) and returns the new status. (du, dv) is the wind offset of the
// particle's scenario plus the bias at t_k. With GRIDS, deposition and exit add their mass
// to the scenario's grids and counters; *fold receives dz/dz_pre (+-1, 0 when clamped).
// FIELDS: the run may have a gridded K_h or the drift correction (uniform run-time tests).
// DRAWS: where the draws come from. DRAWS_FIRST: they stand before the gathers, so that the two
// overlap where registers allow it (measured at 128 registers a thread: 2e4 particles over a day
// 4.55 -> 4.38 ms; at 64 it costs spills: 1e7 particles 40.8 -> 41.9 ms); DRAWS_LAST: after
// them; DRAWS_GIVEN: `given` holds them (draw_pair).
template <bool GRIDS, bool EXT = false, class LEV, bool MODES = EXT, bool FIELDS = true,
          int DRAWS = DRAWS_LAST>
__device__ __forceinline__ uint32_t particle_step(const StepParams &P, const LEV &LV,
                                                  const StepTime &T, const ScenDev &sc,
                                                  const ScenDev *scg, unsigned long long gid,
                                                  int sp, float sig_h_uniform, float du, float dv,
                                                  float &x, float &y, float &z, float *fold,
                                                  float *wv = nullptr, const float *msc = nullptr,
                                                  DepCache *dc = nullptr,
                                                  float4 given = make_float4(0.f, 0.f, 0.f, 0.f))
{
    const int k = T.k;
    float n0, n1, n2;
    auto draw = [&]() {
        if (DRAWS == DRAWS_GIVEN) {
            n0 = given.x;
            n1 = given.y;
            n2 = given.z;
            return;
        }
        const U4 w = philox4x32_10_rk((uint32_t)gid, (uint32_t)(gid >> 32), (uint32_t)k, 0u, P.rk);
        normals3(w, n0, n1, n2);
    };
    if (DRAWS != DRAWS_LAST) draw();
    // 1. weather at the old position and t_k (with the scenario's perturbation modes: msc);
    // 2. diffusivities
    const Met m = sample_met_pair<EXT, LEV, MODES, FIELDS>(P, LV, T, x, y, z, msc);
    const float sig_h = FIELDS && P.khpair ? sqrtf(P.k2 * m.kh * P.dt) : sig_h_uniform;
    const float sig_z = sqrtf(P.k2 * m.kz * P.dt);
    // 3. N(0,1) draws
    if (DRAWS == DRAWS_LAST) draw();
    // 4. Eq. (1)-(2): wind then turbulent displacement
    // (fused multiply-adds, written out: every instantiation rounds alike)
    const float xn = __fmaf_rn(n0, sig_h, __fmaf_rn(m.u + du, P.dt, x));
    const float yn = __fmaf_rn(n1, sig_h, __fmaf_rn(m.v + dv, P.dt, y));
    float zn;
    if (EXT && wv) {
        // vertical Langevin variant (well-mixed for Gaussian turbulence of variance
        // sigma_w^2 = K_z / T_L): w' relaxes over T_L, is kicked by sqrt(2 sigma^2 dt / T_L) n
        // and drifts by (1 + w'^2 / sigma^2) d(sigma^2)/dz dt / 2; z follows w + w'. At its
        // release step a particle starts with sigma_w n' (n' from stream 2).
        float s2 = P.k_scale * m.kz / P.t_lagr, ds2 = P.k_scale * m.dkz / P.t_lagr;
        if (s2 < 1e-6f) {
            s2 = 1e-6f;
            ds2 = 0.0f;
        }
        if (sp == k) {
            const U4 r = philox4x32_10((uint32_t)gid, (uint32_t)(gid >> 32), (uint32_t)k, 2u,
                                       P.seed_lo, P.seed_hi);
            *wv = sqrtf(s2) * sqrtf(-2.0f * logf(unit_uniform(r.a))) *
                  cospif(2.0f * unit_uniform(r.b));
        }
        float wp = *wv;
        wp = wp - wp / P.t_lagr * P.dt + 0.5f * (1.0f + wp * wp / s2) * ds2 * P.dt +
             sqrtf(2.0f * s2 * P.dt / P.t_lagr) * n2;
        *wv = wp;
        zn = z + (m.w + wp) * P.dt;
    } else {
        zn = __fmaf_rn(n2, sig_z, __fmaf_rn(m.w, P.dt, z));
        if (FIELDS && P.drift) zn = __fmaf_rn(P.k_scale * m.dkz, P.dt, zn);
    }
    // 5. reflection, at most 4 folds, then clamp: the first fold by selects (near the ground
    // most warps hold a lane that folds once), the rest of the loop only where that leaves a
    // height outside [zf_lo, zf_hi] (0 and z_top, or infinite where nothing reflects)
    const bool g0 = zn < P.zf_lo, t0 = zn > P.zf_hi;
    float fs = g0 || t0 ? -1.0f : 1.0f;
    zn = g0 ? -zn : t0 ? 2.0f * P.z_top - zn : zn;
    if (zn < P.zf_lo || zn > P.zf_hi) {
#pragma unroll 1
        for (int it = 1; it < 4; ++it) {
            if (P.reflect_ground && zn < 0.0f) { zn = -zn; fs = -fs; }
            else if (P.reflect_top && zn > P.z_top) { zn = 2.0f * P.z_top - zn; fs = -fs; }
            else break;
        }
        if (P.reflect_ground && zn < 0.0f) { zn = 0.0f; fs = 0.0f; }
        if (P.reflect_top && zn > P.z_top) { zn = P.z_top; fs = 0.0f; }
    }
    if (fold) *fold = fs;
    if (EXT && wv) *wv *= fs;            // a reflection reverses the turbulent velocity
    x = xn; y = yn; z = zn;
    // lateral boundary and non-finite positions: one test of the box [fx_lo, fx_hi] x
    // [fy_lo, fy_hi] x |z| <= 1e30 (the domain, cut at 1e30) clears a particle of both (a NaN
    // fails it)
    if (!((xn >= P.fx_lo) & (xn <= P.fx_hi) & (yn >= P.fy_lo) & (yn <= P.fy_hi) &
          (fabsf(zn) <= 1e30f))) {
        if (!isfinite(xn + yn + zn)) {
            atomicOr(P.err, ERR_NAN);
            return ST_EXITED;
        }
        if (P.lateral_exit && (xn < P.x_lo || xn > P.x_hi || yn < P.y_lo || yn > P.y_hi)) {
            if (GRIDS)
                atomicAdd(scg->ctr + C_EXITED * P.ctr_stride, to_fixed(mass_at(P, sc, sp, k), sc.scale));
            return ST_EXITED;
        }
    }
    // 6. dry deposition below the mixing height, then wet where it rains
    bool dry, wet;
    if (DRAWS == DRAWS_GIVEN) {
        dry = __float_as_uint(given.w) & 1u;
        wet = __float_as_uint(given.w) & 2u;
    } else {
        if (!(P.t_dry | P.t_wet)) return ST_ACTIVE;
        uint32_t w_dry, w_wet;
        dep_words(P, gid, k, dc, w_dry, w_wet);
        dry = w_dry < P.t_dry;
        wet = w_wet < P.t_wet;
    }
    if (!(dry | wet)) return ST_ACTIVE;
    int kind = -1;
    if (dry && zn < P.h_mix) kind = 0;
    if (kind < 0 && wet && P.rain) {
        int ir = (int)floorf((xn - P.x0) * P.inv_dx + 0.5f);
        int jr = (int)floorf((yn - P.y0) * P.inv_dy + 0.5f);
        ir = min(max(ir, 0), P.nx - 1);
        jr = min(max(jr, 0), P.ny - 1);
        int hr = (int)floorf(__fdiv_rn(step_since<!GRIDS>(P, k), P.met_dt));
        hr = min(max(hr, 0), P.n_t - 1);
        if (__ldg(P.rain + ((long long)hr * P.ny + jr) * P.nx + ir)) kind = 1;
    }
    if (kind < 0) return ST_ACTIVE;
    if (GRIDS) {
        const unsigned long long v = to_fixed(mass_at(P, sc, sp, k), sc.scale);
        const int ix = grid_axis(xn, P.gx0, P.ginv_dx);
        const int iy = grid_axis(yn, P.gy0, P.ginv_dy);
        if (ix >= 0 && ix < P.cx && iy >= 0 && iy < P.cy) {
            const long long cell = ((long long)kind * P.cy + iy) * P.cx + ix;
            atomicAdd(scg->dep + cell, v);
        } else {
            atomicAdd(scg->ctr + (C_DEP_OUT_DRY + kind) * P.ctr_stride, v);
        }
        atomicAdd(scg->ctr + (C_DEP_DRY + kind) * P.ctr_stride, v);
        if (EXT && P.n_species > 1 && ix >= 0 && ix < P.cx && iy >= 0 && iy < P.cy)
            deposit_species(P, sc, (int)(scg - P.scen), sp, k, kind, iy * P.cx + ix);
    }
    return kind == 0 ? ST_DEP_DRY : ST_DEP_WET;
}

// Occupancy variants: the register budget per thread is 128 (OCC 0), 80 (OCC 1) or 64
// (OCC 2), i.e. 16, 24 or 32 resident warps per SM. OCC_PAIR: 128, and warps in pairs, one of
// which draws for the other.
//
// With at most two warps of particles a scheduler a step is one chain of dependent instructions
// (1500 cycles for the 430 of the plain step). 40 % of them are the draws, which depend on the
// particle's id and the step alone: in an OCC_PAIR block half of the warps compute them up to
// PAIR_STEPS steps ahead for the other half, through two buffers in shared memory, with one
// barrier of the pair's 64 threads a buffer. 2160 particles x 2160 steps 1.74 -> 1.32 ms, 2e4 x
// 2880 3.36 -> 2.93, 38900 x 720 0.76 -> 0.68, 6 members x 240 0.36 -> 0.32; buffers of 4 or 16
// steps 5 and 1 % slower, a pair on one scheduler 9 %.
template <int BLOCK, int OCC>
struct MinBlocks {
    static constexpr int per_sm_threads = OCC == 0 || OCC == OCC_PAIR ? 512 : OCC == 1 ? 768 : 1024;
    static constexpr int value = per_sm_threads / BLOCK > 0 ? per_sm_threads / BLOCK : 1;
};

// Advance: each thread keeps a particle in registers and runs steps [k0, k1) over the
// launch's particles (Ranges): sorted ones of A, release-ordered tiles of B. The persistent
// grid takes tiles of a block's size from an atomic queue: neighbours in the sorted order
// share weather records, so they run on one SM and, held by the block's barrier, at nearly
// the same step (handing single warps out instead cost 10 %, without the barrier 14 %). A
// launch that fits the grid at once is spread evenly over its blocks. With MIXED the lanes of
// a warp may belong to different scenarios (the sorted particles of a batched context): each
// lane finds its scenario from its home slot and carries its own wind offset; the results are
// bit-identical to the per-scenario path. EXT adds, as uniform run-time options, the dosage
// samples (every P.dose_every steps) inside the time loop, K_z from Eq. 3 (P.blpair), the
// daughters of a decay chain (P.n_species > 1), the Langevin variant and the scenarios'
// perturbation modes (P.n_modes > 0); MODES carries the modes alone, FIELDS a gridded K_h and
// the drift correction. TABLE: the levels have a lookup table. The plain instantiations carry
// none of that code.
//
// Bound by issued instructions and the gathers (at 64 registers 32 warps an SM keep the
// schedulers 70 % busy and the L1 data pipe 58 %, DRAM idle; 549 -> 399 instructions a warp step,
// a mid-run launch of 1e7 particles 1.006 -> 0.782 ms), so the step is kept short of branches
// and constant loads. A lane's time loop starts at its own
// release step and ends with the particle: no status is tested inside it, and the lanes of a
// tile of late releases all work from the loop's first turn. (The dosage samples gather a
// warp's lanes at the same step, so with them the loop runs over common steps.)
template <int BLOCK, int OCC, bool MIXED, bool EXT, bool MODES, bool FIELDS, bool TABLE>
__global__ void __launch_bounds__(BLOCK, (MinBlocks<BLOCK, OCC>::value))
advance_kernel(const StepParams P, const Ranges R, unsigned int *queue, int k0, int k1, int do_bin)
{
    extern __shared__ float4 s_adv_dyn[];            // the level tables, sized by the launch
    __shared__ unsigned long long s_acc[BLOCK];
    __shared__ unsigned long long s_steps;
    __shared__ unsigned int s_tile;
    __shared__ StepTable s_tab;                      // the launch's step times
    constexpr bool PAIR = OCC == OCC_PAIR;
    // Units of a warp's 32 particles: those of A, then those of the B tiles. (A launch of the
    // pair that has another number of units for its shape has nothing to do.)
    constexpr unsigned int WARPS = BLOCK / (PAIR ? 64 : 32);
    __shared__ float4 s_draw[PAIR ? WARPS : 1][2][PAIR ? PAIR_STEPS : 1][32];
    __shared__ int s_stop[PAIR ? WARPS : 1][2];      // the pair's particles have all stopped
    const long long live = R.a_live ? (long long)*R.a_live : 0;
    const unsigned int units_a = (unsigned int)((live + 31) >> 5);
    const unsigned int n_units = units_a + ((unsigned int)R.n_b << R.unit_shift);
    if (n_units < R.unit_min || n_units > R.unit_max) return;
    // (the rule for the first is at Levels)
    using Lev = Levels<OCC != 2 || EXT || MODES, TABLE>;
    const Lev LV = load_levels<Lev>(P, reinterpret_cast<unsigned char *>(s_adv_dyn + P.nz),
                                    s_adv_dyn);
    unsigned long long *s_warp = s_acc + (threadIdx.x & ~31);
    const int lane = threadIdx.x & 31;
    // a pair's warps sit on different schedulers, and two pairs of a block on all four: warps
    // 0 1 and 6 7 move particles, 2 3 and 4 5 draw for them
    const unsigned int w = threadIdx.x >> 5;
    const unsigned int warp = PAIR ? (w & 1u) + 2u * (w >> 2) : w;
    const bool drawer = PAIR && (((w >> 1) ^ (w >> 2)) & 1u);
    const long long n_cells = (long long)P.cx * P.cy * P.cz;
    // the uniform horizontal diffusivity gives one displacement scale for the run
    const float sig_h_uniform = sqrtf(P.k2 * fmaxf(P.kh_uniform, 0.0f) * P.dt);
    const uint32_t tab = shared_addr(&s_tab);
    for (int i = threadIdx.x; i < k1 - k0; i += BLOCK)
        step_table_set(s_tab, i, step_time(P, MIXED ? nullptr : P.scen[0].wind_offset, k0 + i));
    if (threadIdx.x == 0) s_steps = 0ull;
    __syncthreads();

    // A block's tile is a run of neighbouring units: as many as it has warps, or, when all
    // units fit the grid at once, the same share for every block.
    const bool one_round = n_units <= WARPS * gridDim.x;
    const unsigned int tile_units =
        one_round ? max(1u, (n_units + gridDim.x - 1u) / gridDim.x) : WARPS;
    for (unsigned int tile = blockIdx.x; tile * tile_units < n_units;) {
        const unsigned int unit = tile * tile_units + warp;
        if (warp < tile_units && unit < n_units) {
            const bool in_a = unit < units_a;
            float4 *state;
            long long first;                         // slot of lane 0
            int count, tscen;
            if (in_a) {
                state = R.state_a;
                first = (long long)unit * 32;
                count = (int)min(32LL, live - first);
                tscen = 0;
            } else {
                const unsigned int u = unit - units_a;
                const Tile tl = R.b_tiles[R.b_first + (u >> R.unit_shift)];
                const int off = (int)(u & ((1u << R.unit_shift) - 1u)) * 32;
                state = R.state_b;
                first = tl.first + off;
                count = max(0, min(32, tl.count - off));
                tscen = tl.scen;
                // (a unit past the end of its tile holds nothing, wherever it would begin)
                if (!LPM_IN_BOUNDS(P.err, (count == 0 || (first >= 0 && first + count <= P.slot_cap)) &&
                                              tscen >= 0 && tscen < P.n_scen))
                    count = 0;
            }
            const ScenDev &scg = P.scen[tscen];

            // ---- load the particle ------------------------------------------------------
            const long long slot = first + lane;
            float *wsrc = in_a ? R.w_a : R.w_b;
            const bool lang = EXT && P.langevin && wsrc;
            const bool modes = MODES && P.n_modes > 0 && P.mode_sc;
            float x = 0.0f, y = 0.0f, z = 0.0f, wv = 0.0f;   // wv: Langevin w' (EXT)
            uint32_t st = ST_EXITED;
            int sp = 0, sj = tscen;                          // sj: scenario of the particle
            unsigned long long gid = 0ull;
            if (lane < count) {
                long long home = in_a ? (long long)__ldg(R.pidx + slot) : slot;
                if (!LPM_IN_BOUNDS(P.err, home >= 0 && home < P.slot_cap)) home = 0;
                if (MIXED && in_a) sj = scen_of(P, home);
                if (MIXED && !LPM_IN_BOUNDS(P.err, sj >= 0 && sj < P.n_scen)) sj = 0;
                const ScenDev &q = P.scen[sj];
                gid = (unsigned long long)(__ldg(&q.id0) + (home - __ldg(&q.first_slot)));
                const float4 s = state[slot];
                x = s.x; y = s.y; z = s.z;
                const uint32_t tag = __float_as_uint(s.w);
                st = tag >> TAG_SHIFT;
                sp = (int)(tag & TAG_STEP);
                wv = lang ? wsrc[slot] : 0.0f;
            }
            const ScenDev &sc = P.scen[sj];
            const float *msc = modes ? P.mode_sc + 8 * sj : nullptr;

            // ---- time loop --------------------------------------------------------------
            unsigned int steps = 0u;                        // active steps of this particle
            float2 o0 = make_float2(0.f, 0.f), o1 = o0;     // wind offsets at h0, h1 (MIXED)
            int cur_h = -1;
            int k = k0;
            if (st == ST_UNRELEASED && sp >= k0 && sp < k1) {
                x = __ldg(&sc.src_x); y = __ldg(&sc.src_y); z = __ldg(&sc.src_z);
                st = ST_ACTIVE;
                k = sp;
            }
            const int k_own = k;                            // this lane's first step
            DepCache dc{0u, 0u};                            // odd-step deposition words
            if (st == ST_ACTIVE) dep_begin(P, gid, k, dc);
            auto advance = [&](int k, float4 given = make_float4(0.f, 0.f, 0.f, 0.f)) {
                const StepTime T = step_time_tab<FIELDS || EXT || MIXED>(tab, k - k0, k);
                float du = T.du, dv = T.dv;
                if (MIXED && P.woff) {
                    if (T.h0 != cur_h) {
                        cur_h = T.h0;
                        const float2 *w = P.woff + (long long)sj * P.n_t;
                        o0 = __ldg(w + T.h0);
                        o1 = __ldg(w + min(T.h0 + 1, P.n_t - 1));
                    }
                    // the same expression as step_offset's, so sorting changes no bit
                    du = P.bias_u + fmaf(T.f, o1.x - o0.x, o0.x);
                    dv = P.bias_v + fmaf(T.f, o1.y - o0.y, o0.y);
                }
                return particle_step<true, EXT, Lev, MODES, FIELDS,
                                     PAIR ? DRAWS_GIVEN : OCC != 2 ? DRAWS_FIRST : DRAWS_LAST>(
                    P, LV, T, sc, &sc, gid, sp, sig_h_uniform, du, dv, x, y, z, nullptr,
                    lang ? &wv : nullptr, msc, &dc, given);
            };
            if constexpr (PAIR) {
                // Both warps of the pair loaded the same particles, so both come to the same
                // number of turns, and to the same barriers; a turn that finds s_stop set ends
                // both. The drawer reads s_stop[h] between barriers n and n + 1 (n = h mod 2),
                // its partner writes it next between n + 1 and n + 2; the buffers likewise.
                const int turns =
                    (__reduce_max_sync(0xffffffffu, st == ST_ACTIVE ? k1 - k_own : 0) +
                     PAIR_STEPS - 1) / PAIR_STEPS;
                float4(*buf)[PAIR_STEPS][32] = s_draw[warp];
                auto fill = [&](int turn) {
#pragma unroll 1
                    for (int j = 0; j < PAIR_STEPS; j += 2) {
                        float4 a, b;
                        draw_pair(P, gid, k_own + turn * PAIR_STEPS + j, dc, a, b);
                        buf[turn & 1][j][lane] = a;
                        buf[turn & 1][j + 1][lane] = b;
                    }
                };
                if (drawer && turns > 0) fill(0);
#pragma unroll 1
                for (int turn = 0; turn < turns; ++turn) {
                    if (!drawer) {
                        const bool stop = !__any_sync(0xffffffffu, st == ST_ACTIVE && k < k1);
                        if (lane == 0) s_stop[warp][turn & 1] = stop;
                    }
                    __syncwarp();
                    asm volatile("bar.sync %0, 64;" ::"r"((int)warp + 1) : "memory");
                    if (*(volatile int *)&s_stop[warp][turn & 1]) break;
                    if (drawer) {
                        if (turn + 1 < turns) fill(turn + 1);
                    } else {
#pragma unroll 1
                        for (int j = 0; j < PAIR_STEPS; ++j) {
                            if (st == ST_ACTIVE && k < k1) {
                                st = advance(k, buf[turn & 1][j][lane]);
                                ++k;
                            }
                        }
                    }
                }
                steps = (unsigned int)(k - k_own);
                if (drawer) {                               // its partner has the results
                    count = 0;
                    st = ST_EXITED;
                }
            } else if (!EXT || !P.dose_every) {
                if (st == ST_ACTIVE) {
#pragma unroll 1
                    do {
                        st = advance(k);
                        ++k;
                    } while (st == ST_ACTIVE && k < k1);
                    steps = (unsigned int)(k - k_own);
                }
            } else {
#pragma unroll 1
                for (k = k0; k < k1; ++k) {
                    // the samples are warp-collective: the warp stays together
                    if (!__any_sync(0xffffffffu, st == ST_ACTIVE)) break;
                    if (st == ST_ACTIVE && k >= k_own) {
                        st = advance(k);
                        ++steps;
                    }
                    // every dose_every-th step, the decayed masses at t_{k+1}
                    if ((k + 1) % P.dose_every == 0) {
                        const bool on = st == ST_ACTIVE && k >= k_own;
                        const int cell = on ? grid_cell(P, x, y, z) : KEY_NONE;
                        unsigned long long v = 0ull;
                        if (on) v = to_fixed(mass_at(P, sc, sp, k), __ldg(&sc.scale) * P.dose_mul);
                        if (MIXED) {
                            long long key = -1;
                            if (on) key = cell >= 0 ? (long long)sj * n_cells + cell : -2LL - sj;
                            warp_accumulate_scen(key, v, P, P.dose_all, C_DOSE_OUT, s_warp, n_cells);
                        } else {
                            warp_accumulate(cell, v, P.dose_all + (long long)tscen * n_cells,
                                            scg.ctr + C_DOSE_OUT * P.ctr_stride, s_warp, n_cells,
                                            P.err);
                        }
                    }
                }
            }

            // ---- store ------------------------------------------------------------------
            const bool on = lane < count && st == ST_ACTIVE;
            if (lane < count) {
                state[slot] = make_float4(x, y, z, __uint_as_float((st << TAG_SHIFT) |
                                                                            (uint32_t)sp));
                // only a moving particle has a turbulent velocity (0 once deposited or
                // exited, and before its release)
                if (lang) wsrc[slot] = on ? wv : 0.0f;
            }

            // ---- sort keys for the sort that follows (its inputs: A slots, then B lanes) ----
            if (R.keys && !drawer) {
                const unsigned int dead_key =
                    (unsigned int)sort_dead_key(P.nx, P.ny, P.nz, R.key_shift, 0);
                long long idx = -1;
                unsigned int key = KEY_NONE_U;
                if (in_a) {
                    if (lane < count) idx = slot;
                } else {
                    idx = live + (long long)(unit - units_a) * 32 + lane;
                }
                if (on) {
                    int ix, jy, kz;
                    float fa, fb, fc;
                    axis(x, P.x0, P.inv_dx, P.nx2, ix, fa);
                    axis(y, P.y0, P.inv_dy, P.ny2, jy, fb);
                    level(P, LV, z, kz, fc);
                    key = cell_key(P, ix, jy, kz) >> R.key_shift;
                } else if (lane < count) {
                    key = dead_key;
                }
                if (idx >= 0) R.keys[idx] = key;
                sort_count(R.counts, key);
            }

            // ---- end-of-segment concentration snapshot (every n-th step, Sec. 3.2) --------
            if (do_bin) {
                int cell = KEY_NONE;
                unsigned long long v = 0ull;
                if (on) {
                    v = to_fixed(mass_at(P, sc, sp, k1 - 1), __ldg(&sc.scale));
                    cell = grid_cell(P, x, y, z);
                }
                if (MIXED) {
                    long long key = -1;
                    if (on) key = cell >= 0 ? (long long)sj * n_cells + cell : -2LL - sj;
                    warp_accumulate_scen(key, v, P, P.conc_all, C_BIN_OUT, s_warp, n_cells);
                } else {
                    warp_accumulate(cell, v, scg.conc, scg.ctr + C_BIN_OUT * P.ctr_stride, s_warp,
                                    n_cells, P.err);
                }
                // daughters of a decay chain, species by species (the same cells)
                for (int d = 1; EXT && d < P.n_species; ++d) {
                    unsigned long long vd = 0ull;
                    if (on) {
                        const float m0 = m0_of(P, sc, sp);
                        vd = to_fixed(m0 * chain_amount(P, d, (float)(k1 - sp) * P.dt),
                                      __ldg(&sc.scale));
                    }
                    unsigned long long *base = P.sp_conc_all + (long long)(d - 1) * P.n_scen * n_cells;
                    if (MIXED) {
                        long long key = -1;
                        if (on) key = cell >= 0 ? (long long)sj * n_cells + cell : -2LL - sj;
                        warp_accumulate_scen(key, vd, P, base, C_SP_OUT + d - 1, s_warp, n_cells);
                    } else {
                        warp_accumulate(cell, vd, base + (long long)tscen * n_cells,
                                        scg.ctr + (C_SP_OUT + d - 1) * P.ctr_stride, s_warp,
                                        n_cells, P.err);
                    }
                }
            }

            // ---- active particle-steps --------------------------------------------------
            if (MIXED) {
                warp_count_scen(lane < count ? sj : -1, steps, C_ACTIVE_STEPS, P, s_warp);
            } else {
                const unsigned int sum = __reduce_add_sync(0xffffffffu, steps);
                if ((threadIdx.x & 31) == 0 && sum) atomicAdd(&s_steps, (unsigned long long)sum);
            }
        }
        if (one_round) break;
        __syncthreads();
        if (threadIdx.x == 0) s_tile = gridDim.x + atomicAdd(queue, 1u);
        __syncthreads();
        tile = s_tile;
    }
    if (!MIXED) {
        __syncthreads();
        if (threadIdx.x == 0 && s_steps)
            atomicAdd(P.scen[0].ctr + C_ACTIVE_STEPS * P.ctr_stride, s_steps);
    }
}

template <int BLOCK, int OCC, bool MIXED, bool EXT, bool MODES, bool FIELDS, bool TABLE>
void adv_prefer_l1()
{
    // the kernel needs a few KB of shared memory per block: ask for a small carve-out so the
    // rest of the SM's unified L1 serves the weather gathers (measured +0.7 to +1.7 %)
    cudaFuncSetAttribute(advance_kernel<BLOCK, OCC, MIXED, EXT, MODES, FIELDS, TABLE>,
                         cudaFuncAttributePreferredSharedMemoryCarveout,
                         OCC == OCC_PAIR ? 40 : 10);
    (void)cudaGetLastError();
}

template <int BLOCK, int OCC, bool MIXED, bool EXT, bool MODES, bool FIELDS, bool TABLE>
cudaError_t launch_adv(const AdvanceLaunch &L)
{
    static std::once_flag once;          // per instantiation; contexts may use several threads
    std::call_once(once, adv_prefer_l1<BLOCK, OCC, MIXED, EXT, MODES, FIELDS, TABLE>);
    const size_t smem = adv_dyn_smem(L.params->nz, L.params->n_lut);
    advance_kernel<BLOCK, OCC, MIXED, EXT, MODES, FIELDS, TABLE><<<L.grid, BLOCK, smem,
                                                                  L.stream>>>(
        *L.params, L.ranges, L.queue, L.k0, L.k1, L.do_bin);
    return cudaGetLastError();
}

template <int BLOCK, int OCC, bool MIXED, bool EXT, bool MODES, bool FIELDS, bool TABLE>
int occ_adv(size_t smem)
{
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &n, advance_kernel<BLOCK, OCC, MIXED, EXT, MODES, FIELDS, TABLE>, BLOCK, smem);
    return n;
}

// (occupancy variant, mixed scenarios, options: AdvanceLaunch::variant) -> instantiation, for
// one block size
#define LPM_ADV_CASE(FN, BLOCK, OCC, MIX, VAR, ...)                                    \
    case OCC * 100 + MIX * 10 + VAR:                                                   \
        return FN<BLOCK, OCC, (MIX != 0), adv_is_ext(VAR),                          \
                  (adv_is_ext(VAR) || VAR == ADV_MODES || VAR == ADV_MODES_FIELDS),        \
                  (adv_is_ext(VAR) || VAR == ADV_FIELDS || VAR == ADV_MODES_FIELDS),       \
                  (VAR == ADV_PLAIN || VAR == ADV_EXT || VAR == ADV_MODES)>(__VA_ARGS__);
#define LPM_ADV_CASES2(FN, BLOCK, VAR, ...)                                            \
    LPM_ADV_CASE(FN, BLOCK, 0, 0, VAR, __VA_ARGS__)                                    \
    LPM_ADV_CASE(FN, BLOCK, 0, 1, VAR, __VA_ARGS__)                                    \
    LPM_ADV_CASE(FN, BLOCK, 1, 0, VAR, __VA_ARGS__)                                    \
    LPM_ADV_CASE(FN, BLOCK, 1, 1, VAR, __VA_ARGS__)                                    \
    LPM_ADV_CASE(FN, BLOCK, 2, 0, VAR, __VA_ARGS__)                                    \
    LPM_ADV_CASE(FN, BLOCK, 2, 1, VAR, __VA_ARGS__)
#define LPM_ADV_CASES(FN, BLOCK, ...)                                                  \
    LPM_ADV_CASES2(FN, BLOCK, 0, __VA_ARGS__)                                          \
    LPM_ADV_CASES2(FN, BLOCK, 1, __VA_ARGS__)                                          \
    LPM_ADV_CASES2(FN, BLOCK, 2, __VA_ARGS__)                                          \
    LPM_ADV_CASES2(FN, BLOCK, 3, __VA_ARGS__)                                          \
    LPM_ADV_CASES2(FN, BLOCK, 4, __VA_ARGS__)                                          \
    LPM_ADV_CASES2(FN, BLOCK, 5, __VA_ARGS__)

#define LPM_ADVANCE_TU(BLOCK)                                                          \
    cudaError_t launch_advance_b##BLOCK(const AdvanceLaunch &L)                         \
    {                                                                                  \
        switch (L.occ * 100 + (L.mixed ? 10 : 0) + L.variant()) {                      \
            LPM_ADV_CASES(launch_adv, BLOCK, L)                                        \
        }                                                                              \
        return cudaErrorInvalidValue;                                                  \
    }                                                                                  \
    int occupancy_b##BLOCK(int occ, bool mixed, int variant, size_t smem)              \
    {                                                                                  \
        switch (occ * 100 + (mixed ? 10 : 0) + variant) {                              \
            LPM_ADV_CASES(occ_adv, BLOCK, smem)                                        \
        }                                                                              \
        return 0;                                                                      \
    }

#define LPM_ADVANCE_PAIR_TU(BLOCK)                                                     \
    cudaError_t launch_advance_pair(const AdvanceLaunch &L)                             \
    {                                                                                  \
        switch (L.mixed * 10 + L.variant()) {                                          \
            LPM_ADV_CASES_PAIR(launch_adv, BLOCK, L)                                   \
        }                                                                              \
        return cudaErrorInvalidValue;                                                  \
    }                                                                                  \
    int occupancy_pair(bool mixed, int variant, size_t smem)                           \
    {                                                                                  \
        switch (mixed * 10 + variant) {                                                \
            LPM_ADV_CASES_PAIR(occ_adv, BLOCK, smem)                                   \
        }                                                                              \
        return 0;                                                                      \
    }
#define LPM_ADV_CASE_PAIR(FN, BLOCK, MIX, VAR, ...)                                    \
    case MIX * 10 + VAR:                                                               \
        return FN<BLOCK, OCC_PAIR, (MIX != 0), false,                                  \
                  (VAR == ADV_MODES || VAR == ADV_MODES_FIELDS),                       \
                  (VAR == ADV_FIELDS || VAR == ADV_MODES_FIELDS),                      \
                  (VAR == ADV_PLAIN || VAR == ADV_MODES)>(__VA_ARGS__);
#define LPM_ADV_CASES_PAIR(FN, BLOCK, ...)                                             \
    LPM_ADV_CASE_PAIR(FN, BLOCK, 0, 0, __VA_ARGS__)                                    \
    LPM_ADV_CASE_PAIR(FN, BLOCK, 0, 2, __VA_ARGS__)                                    \
    LPM_ADV_CASE_PAIR(FN, BLOCK, 0, 3, __VA_ARGS__)                                    \
    LPM_ADV_CASE_PAIR(FN, BLOCK, 0, 4, __VA_ARGS__)                                    \
    LPM_ADV_CASE_PAIR(FN, BLOCK, 1, 0, __VA_ARGS__)                                    \
    LPM_ADV_CASE_PAIR(FN, BLOCK, 1, 2, __VA_ARGS__)                                    \
    LPM_ADV_CASE_PAIR(FN, BLOCK, 1, 3, __VA_ARGS__)                                    \
    LPM_ADV_CASE_PAIR(FN, BLOCK, 1, 4, __VA_ARGS__)

}  // namespace lpm
