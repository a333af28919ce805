// lpm_adjoint.cu - receptor concentrations and their reverse-mode gradient.
//
// Forward: every particle runs the horizon with the step of the main loop (particle_step)
// and the decayed mass is spread on the receptors with a Gaussian kernel (with the ground
// image) every `every` steps. Backward: a reverse sweep carrying mu = dL/dX through the
// transposed Jacobian of each step and accumulating the parameter partials; events
// (deposition, exit) are frozen; sums over particles are reduced in FP64. The backward
// needs the forward's states, kept in one of three forms:
//  - trajectory, sorted (sorting on): CK-step segments over the particles re-sorted
//    between segments (by weather cell; several scenarios: by scenario, then cell tile),
//    every state stored;
//  - trajectory in release order (sorting off): every state stored, one thread per
//    particle over the whole horizon;
//  - checkpoints every CK steps when the trajectory does not fit: each CK-step segment is
//    recomputed from its checkpoint (same keyed draws and FP32 arithmetic, so the same
//    path and events) before it is swept, in the sorted segments or in release order.
#include <mutex>

#include "lpm_advance.cuh"
#include "lpm_adjoint.h"

namespace lpm {

// Weather and its spatial gradient: val = (u, v, w, K_z, K_h), g[q][d] = d val[q] / d x_d.
// KHG: K_h may be a gridded field (else uniform, gradient 0, none of its code compiled).
template <bool KHG, class LEV>
__device__ __forceinline__ void sample_met_grad(const StepParams &P, const LEV &L,
                                                const StepTime &T, float sig_h_uniform, float x,
                                                float y, float z, float val[5], float g[5][3])
{
    int i, j, k;
    float a, b, c;
    axis(x, P.x0, P.inv_dx, P.nx2, i, a);
    axis(y, P.y0, P.inv_dy, P.ny2, j, b);
    level(P, L, z, k, c);
    const float fx = (x - P.x0) * P.inv_dx, fy = (y - P.y0) * P.inv_dy;
    const float gx = (fx >= 0.0f && fx <= (float)(P.nx - 1)) ? P.inv_dx : 0.0f;
    const float gy0 = (fy >= 0.0f && fy <= (float)(P.ny - 1)) ? P.inv_dy : 0.0f;
    const float gz0 = (z >= L.z_lo && z <= L.z_hi) ? level_entry(P, L, k).y : 0.0f;
    const Corners q = cell_corners(P, i, j, k, b, c);
    const F2 ff = pack2(T.f, T.f), aa = pack2(a, a), bb = pack2(q.b, q.b), cc = pack2(q.c, q.c);
    Rec4 yl[2], dx[2], dy[2];
#pragma unroll
    for (int l = 0; l < 2; ++l) {
        Rec4 xr[2], df[2];
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            const float4 *p = record_at<32>(T.pair, q.rec[2 * l + m]);
            const Rec4 v0 = ld_blend(p, ff), v1 = ld_blend(p + 8, ff);
            df[m] = sub4(v1, v0);
            xr[m] = lerp4(v0, v1, aa);
        }
        yl[l] = lerp4s(xr[0], xr[1], bb, q.sy);
        dx[l] = lerp4s(df[0], df[1], bb, q.sy);
        dy[l] = sub4(xr[1], xr[0]);
    }
    const float4 r = unpack4(lerp4s(yl[0], yl[1], cc, q.sz));
    // d/dx: x-differences blended in y and z; d/dy: y-differences blended in z; a swapped
    // axis negates its differences (exactly), and so does its sign here
    const float4 ddx = unpack4(lerp4s(dx[0], dx[1], cc, q.sz));
    const float4 ddy = unpack4(lerp4s(dy[0], dy[1], cc, q.sz));
    const float4 ddz = unpack4(sub4(yl[1], yl[0]));
    const float gy = q.sy ? -gy0 : gy0, gz = q.sz ? -gz0 : gz0;
    val[0] = r.x; val[1] = r.y; val[2] = r.z; val[3] = r.w;
    g[0][0] = ddx.x * gx; g[0][1] = ddy.x * gy; g[0][2] = ddz.x * gz;
    g[1][0] = ddx.y * gx; g[1][1] = ddy.y * gy; g[1][2] = ddz.y * gz;
    g[2][0] = ddx.z * gx; g[2][1] = ddy.z * gy; g[2][2] = ddz.z * gz;
    g[3][0] = ddx.w * gx; g[3][1] = ddy.w * gy; g[3][2] = ddz.w * gz;
    if (!(val[3] > 0.0f)) {
        val[3] = 0.0f;
        g[3][0] = g[3][1] = g[3][2] = 0.0f;
    }
    if (KHG && P.khpair) {
        const float2 *khp = P.khpair + (long long)T.h0 * P.slab;
        float ey[2], lx[2], dk[2];
#pragma unroll
        for (int l = 0; l < 2; ++l) {
            float ex[2], de[2];
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                const float2 *p = record_at<8>(khp, q.rec[2 * l + m]);
                const float2 v0 = __ldg(p), v1 = __ldg(p + 4);
                const float e0 = fmaf(T.f, v0.y, v0.x), e1 = fmaf(T.f, v1.y, v1.x);
                de[m] = e1 - e0;
                ex[m] = fmaf(a, de[m], e0);
            }
            ey[l] = lerps(ex[0], ex[1], q.b, q.sy);
            lx[l] = lerps(de[0], de[1], q.b, q.sy);
            dk[l] = ex[1] - ex[0];
        }
        val[4] = lerps(ey[0], ey[1], q.c, q.sz);
        g[4][0] = lerps(lx[0], lx[1], q.c, q.sz) * gx;
        g[4][1] = lerps(dk[0], dk[1], q.c, q.sz) * gy;
        g[4][2] = (ey[1] - ey[0]) * gz;
        if (!(val[4] > 0.0f)) {
            val[4] = 0.0f;
            g[4][0] = g[4][1] = g[4][2] = 0.0f;
        }
    } else {
        val[4] = fmaxf(P.kh_uniform, 0.0f);
        g[4][0] = g[4][1] = g[4][2] = 0.0f;
    }
    (void)sig_h_uniform;
}

// The time parts of step k as step_time computes them (without an offset), packed for a
// per-block table: the steps of a segment are the same for every particle.
template <bool ONCE>
__device__ __forceinline__ float4 step_time_parts(const StepParams &P, int k)
{
    const StepTime T = step_time<ONCE>(P, nullptr, k);
    const unsigned long long p = reinterpret_cast<unsigned long long>(T.pair);
    return make_float4(__uint_as_float((unsigned int)p), __uint_as_float((unsigned int)(p >> 32)),
                       T.f, __int_as_float(T.h0));
}

// step_time(P, wind_offset, k) from the packed time parts of step k.
__device__ __forceinline__ StepTime step_time_from(const StepParams &P, const float2 *wind_offset,
                                                   float4 a, int k)
{
    StepTime T;
    T.k = k;
    T.pair = reinterpret_cast<const float4 *>((unsigned long long)__float_as_uint(a.x) |
                                              ((unsigned long long)__float_as_uint(a.y) << 32));
    T.f = a.z;
    T.h0 = __float_as_int(a.w);
    const float2 d = step_offset(P, wind_offset, T.h0, min(T.h0 + 1, P.n_t - 1), T.f);
    T.du = d.x;
    T.dv = d.y;
    return T;
}

__device__ __forceinline__ long long release_step_of(const ScenDev &sc, long long slot)
{
    const long long p = sc.part_first + (slot - sc.first_slot);
    return sc.rel_first + (p * (long long)(sc.rel_last - sc.rel_first)) / sc.n_total;
}

__device__ __forceinline__ float4 pack_state(float x, float y, float z, uint32_t st, int sp)
{
    return make_float4(x, y, z, __uint_as_float((st << TAG_SHIFT) | ((uint32_t)sp & TAG_STEP)));
}

// Receptors a particle at (x, y) can be within the cut-off distance of: entries [lo, hi) of
// the bin lists (empty outside the bins).
__device__ __forceinline__ void receptors_near(const AdjParams &A, float x, float y, int &lo,
                                               int &hi)
{
    lo = hi = 0;
    const float fx = (x - A.rbx0) * A.rinv_bin, fy = (y - A.rby0) * A.rinv_bin;
    if (!(fx >= 0.0f && fy >= 0.0f && fx < (float)A.rnbx && fy < (float)A.rnby)) return;
    const int b = (int)fy * A.rnbx + (int)fx;
    lo = __ldg(A.rbin_off + b);
    hi = __ldg(A.rbin_off + b + 1);
}

// Adds mass m at (x, y, z) to the receptor sums C[r] (shared or global).
__device__ __forceinline__ void sample_receptors(const AdjParams &A, const float4 *s_rec, float x,
                                                 float y, float z, float m, double *C)
{
    int lo, hi;
    receptors_near(A, x, y, lo, hi);
    for (int t = lo; t < hi; ++t) {
        const int r = __ldg(A.rbin_idx + t);
        const float4 q = s_rec[r];
        const float dx = x - q.x, dy = y - q.y, dz = z - q.z, dzi = z + q.z;
        const float h2 = dx * dx + dy * dy;
        const float d1 = h2 + dz * dz, d2 = h2 + dzi * dzi;
        if (d1 > A.cut2 && d2 > A.cut2) continue;
        const float G = A.norm * (expf(-d1 * A.inv2s2) + expf(-d2 * A.inv2s2));
        atomicAdd(C + r, (double)(m * G));
    }
}

// ---------------------------------------------------------------------------------
// Forward: receptor concentrations, and checkpoints or the whole trajectory.
// ---------------------------------------------------------------------------------
// 7 blocks per SM (72 registers): measured 5 % faster than 8 (64 registers, 16 B spilled)
// on the batched inversion's forward
template <bool TRAJ>
__global__ void __launch_bounds__(ADJ_BLOCK, 7)
adj_forward_kernel(const StepParams P, const AdjParams A)
{
    extern __shared__ float4 s_dyn[];             // sized by the launch: adj_smem_forward
    float4 *s_rec = s_dyn;                        // [R]
    double *s_C = reinterpret_cast<double *>(s_rec + A.R);    // [R]
    unsigned char *s_lut = reinterpret_cast<unsigned char *>(s_C + A.R);   // [n_lut]
    __shared__ float4 s_ent[MAX_LEVELS];           // warps span many levels here
    const auto LV = load_levels<Levels<true, false>>(P, s_lut, s_ent);
    for (int r = threadIdx.x; r < A.R; r += ADJ_BLOCK) {
        s_rec[r] = A.rec[r];
        s_C[r] = 0.0;
    }
    __syncthreads();
    const Tile tile = A.tiles[blockIdx.x];
    const ScenDev sc = P.scen[tile.scen];
    const float sig_h_uniform = sqrtf(2.0f * P.k_scale * fmaxf(P.kh_uniform, 0.0f) * P.dt);
    if ((int)threadIdx.x < tile.count) {
        const long long slot = tile.first + threadIdx.x;
        const unsigned long long gid = (unsigned long long)(sc.id0 + (slot - sc.first_slot));
        const int sp = (int)release_step_of(sc, slot);
        const float m0 = __ldg(P.m0 + sc.m0_off + (sp - sc.rel_first));
        float x = sc.src_x, y = sc.src_y, z = sc.src_z;
        float4 *row = nullptr;
        int k0 = 0;
        if (TRAJ) {
            const longlong2 tt = A.traj_tile[blockIdx.x];
            row = A.traj + tt.x + threadIdx.x;
            k0 = (int)tt.y;
        } else {
            for (int c = 0; c < A.n_ck && c * CK <= sp; ++c)
                A.ckpt[(long long)c * A.n_slots + slot] = pack_state(x, y, z, ST_UNRELEASED, sp);
        }
        uint32_t st = ST_ACTIVE;
        int kn = sp;                              // one past the last step taken
        for (int k = sp; k < A.n_steps; ++k) {
            if (!TRAJ && k > sp && k % CK == 0)
                A.ckpt[(long long)(k / CK) * A.n_slots + slot] = pack_state(x, y, z, ST_ACTIVE, sp);
            const StepTime T = step_time<true>(P, sc.wind_offset, k);
            const float xb = x, yb = y, zb = z;
            float fs = 1.0f;
            st = particle_step<false>(P, LV, T, sc, nullptr, gid, sp, sig_h_uniform, T.du, T.dv,
                                      x, y, z, TRAJ ? &fs : nullptr);
            if (TRAJ && k >= k0 &&                // rows start at the tile's first release
                LPM_IN_BOUNDS(P.err, (row - A.traj) + (long long)(k - k0) * ADJ_BLOCK < A.traj_cap))
                __stcs(row + (long long)(k - k0) * ADJ_BLOCK, make_float4(xb, yb, zb, fs));
            kn = k + 1;
            if (st != ST_ACTIVE) {
                if (!TRAJ)
                    for (int c = k / CK + 1; c < A.n_ck; ++c)
                        A.ckpt[(long long)c * A.n_slots + slot] = pack_state(x, y, z, st, sp);
                break;
            }
            if ((k + 1) % A.every == 0) {
                const float m = m0 * expf(-P.lambda * (float)(k + 1 - sp) * P.dt) * A.inv_ns;
                sample_receptors(A, s_rec, x, y, z, m, s_C);
            }
        }
        if (TRAJ)
            A.fin[slot] = make_float4(x, y, z, __uint_as_float((uint32_t)kn |
                                                               (st != ST_ACTIVE ? 0x80000000u : 0u)));
    }
    __syncthreads();
    for (int r = threadIdx.x; r < A.R; r += ADJ_BLOCK)
        if (s_C[r] != 0.0) atomicAdd(A.C + (long long)tile.scen * A.R + r, s_C[r]);
}

// ---------------------------------------------------------------------------------
// Backward: reverse sweep.
// ---------------------------------------------------------------------------------
struct Adjoint {
    float mu0, mu1, mu2;                  // dL/dX of the state after the current step
    float gsk, gbu, gbv, gq;              // partials: s_K, b_u, b_v, emission of the release hour
};

// One step of the reverse sweep: the receptor term of the state Xa after step k (when k
// is a sample step and not the step that ended the run), then mu <- J_k^T mu with the
// Jacobian of step k at the state X before it (fold = the step's reflection sign). The
// receptor weights dL/dC / n_s come from s_w, or from wg (the particle's scenario's row of
// A.w) for a particle whose scenario is not its block's.
template <bool KHG, bool DRAWS_FIRST = false, class LEV>
__device__ __forceinline__ void reverse_step(const StepParams &P, const AdjParams &A,
                                             const LEV &LV, const StepTime &T,
                                             const float4 *s_rec, const float *s_w,
                                             unsigned long long gid, int sp, float m0, float mq,
                                             float sig_h_uniform, float sq2dt, float4 X,
                                             float fold, float4 Xa, bool sample, Adjoint &J,
                                             const double *wg = nullptr)
{
    const int k = T.k;
    if (sample) {
        const float decay = expf(-P.lambda * (float)(k + 1 - sp) * P.dt);
        const float m = m0 * decay;
        int lo, hi;
        receptors_near(A, Xa.x, Xa.y, lo, hi);
        for (int t = lo; t < hi; ++t) {
            const int r = __ldg(A.rbin_idx + t);
            const float4 q = s_rec[r];
            const float dx = Xa.x - q.x, dy = Xa.y - q.y, dz = Xa.z - q.z, dzi = Xa.z + q.z;
            const float h2 = dx * dx + dy * dy;
            const float d1 = h2 + dz * dz, d2 = h2 + dzi * dzi;
            if (d1 > A.cut2 && d2 > A.cut2) continue;
            const float e1 = A.norm * expf(-d1 * A.inv2s2);
            const float e2 = A.norm * expf(-d2 * A.inv2s2);
            const float wr = wg ? (float)(wg[r] * (double)A.inv_ns) : s_w[r];
            const float c1 = -wr * m * A.inv_s2;
            J.mu0 += c1 * (e1 + e2) * dx;
            J.mu1 += c1 * (e1 + e2) * dy;
            J.mu2 += c1 * (e1 * dz + e2 * dzi);
            J.gq += wr * mq * decay * (e1 + e2);
        }
    }
    float val[5], g[5][3], n0, n1, n2;
    auto draw = [&]() {
        const U4 w = philox4x32_10_rk((uint32_t)gid, (uint32_t)(gid >> 32), (uint32_t)k, 0u, P.rk);
        normals3(w, n0, n1, n2);
    };
    if (DRAWS_FIRST) draw();
    sample_met_grad<KHG>(P, LV, T, sig_h_uniform, X.x, X.y, X.z, val, g);
    if (!DRAWS_FIRST) draw();
    const float kz = P.k_scale * val[3];
    const float sig_z = sqrtf(2.0f * kz * P.dt);
    const float cz = val[3] > 0.0f ? sq2dt / (2.0f * sqrtf(val[3])) : 0.0f;
    // a uniform K_h has one scale for the run and no gradient
    float sig_h = sig_h_uniform, ch = 0.0f;
    if (KHG) {
        const float kh = P.k_scale * val[4];
        sig_h = sqrtf(2.0f * kh * P.dt);
        ch = val[4] > 0.0f ? sq2dt / (2.0f * sqrtf(val[4])) : 0.0f;
    }
    // parameter partials: s_K, b_u, b_v
    J.gsk += (J.mu0 * n0 * sig_h + J.mu1 * n1 * sig_h + J.mu2 * fold * n2 * sig_z) * A.inv2sk;
    J.gbu += J.mu0 * P.dt;
    J.gbv += J.mu1 * P.dt;
    // mu <- J^T mu
    const float mz = J.mu2 * fold;
    float nm[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const float jx = KHG ? P.dt * g[0][d] + n0 * ch * g[4][d] : P.dt * g[0][d];
        const float jy = KHG ? P.dt * g[1][d] + n1 * ch * g[4][d] : P.dt * g[1][d];
        const float jz = P.dt * g[2][d] + n2 * cz * g[3][d];
        nm[d] = J.mu0 * jx + J.mu1 * jy + mz * jz;
    }
    J.mu0 += nm[0];
    J.mu1 += nm[1];
    J.mu2 = mz + nm[2];
}

// Sums of a group's particles (FP64) and one atomic per parameter and group: the source
// partials are the sum of mu at release.
__device__ __forceinline__ void reduce_gradient(const AdjParams &A, const Tile &tile, Adjoint J,
                                                bool valid, int qidx, double *s_g, double *s_gq)
{
    if (!valid) J = Adjoint{0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    // warp sums in FP64, so the totals do not depend on which particles share a warp
    double d[6] = {J.mu0, J.mu1, J.mu2, J.gsk, J.gbu, J.gbv};
#pragma unroll
    for (int i = 0; i < 6; ++i)
        for (int o = 16; o > 0; o >>= 1) d[i] += __shfl_xor_sync(0xffffffffu, d[i], o);
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int i = 0; i < 6; ++i) atomicAdd(&s_g[i], d[i]);
    if (J.gq != 0.f) atomicAdd(&s_gq[qidx], (double)J.gq);
    __syncthreads();
    double *G = A.grad + (long long)tile.scen * A.ng;
    const int lane = threadIdx.x % ADJ_BLOCK;
    if (lane < 6 && s_g[lane] != 0.0)
        atomicAdd(G + (lane < 3 ? lane : A.nq + lane), s_g[lane]);
    for (int i = lane; i < A.nq; i += ADJ_BLOCK)
        if (s_gq[i] != 0.0) atomicAdd(G + 3 + i, s_gq[i]);
}

// Receptors and the group's scenario's dL/dC (scaled by 1 / samples) into shared memory.
__device__ __forceinline__ void load_receptors(const AdjParams &A, const Tile &tile, float4 *s_rec,
                                               float *s_w, double *s_g, double *s_gq)
{
    const int lane = threadIdx.x % ADJ_BLOCK;
    for (int r = lane; r < A.R; r += ADJ_BLOCK) {
        if (threadIdx.x < ADJ_BLOCK) s_rec[r] = A.rec[r];
        s_w[r] = (float)(A.w[(long long)tile.scen * A.R + r] * (double)A.inv_ns);
    }
    for (int i = lane; i < A.nq; i += ADJ_BLOCK) s_gq[i] = 0.0;
    if (lane < 6) s_g[lane] = 0.0;
    __syncthreads();
}

// Checkpoint form: each thread recomputes its particle's path one CK-step segment at a
// time from the checkpoint (same keyed draws and FP32 arithmetic, so the same path and
// events) into a local buffer, then sweeps the segment in reverse.
template <bool KHG>
__global__ void __launch_bounds__(ADJ_BLOCK)
adj_backward_kernel(const StepParams P, const AdjParams A)
{
    extern __shared__ float4 s_dyn[];             // sized by the launch: adj_smem_backward
    float4 *s_rec = s_dyn;                        // [R]
    double *s_g = reinterpret_cast<double *>(s_rec + A.R);    // [6]
    double *s_gq = s_g + 6;                       // [nq]
    float *s_w = reinterpret_cast<float *>(s_gq + A.nq);      // [R]
    unsigned char *s_lut = reinterpret_cast<unsigned char *>(s_w + A.R);   // [n_lut]
    __shared__ float4 s_ent[MAX_LEVELS];           // warps span many levels here
    const auto LV = load_levels<Levels<true, false>>(P, s_lut, s_ent);
    const Tile tile = A.tiles[blockIdx.x];
    load_receptors(A, tile, s_rec, s_w, s_g, s_gq);
    const ScenDev sc = P.scen[tile.scen];
    const float sig_h_uniform = sqrtf(2.0f * P.k_scale * fmaxf(P.kh_uniform, 0.0f) * P.dt);
    const float sq2dt = sqrtf(2.0f * P.k_scale * P.dt);
    Adjoint J{0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    // Loops run over warp-uniform step ranges with per-lane predicates, so the lanes of a
    // warp (consecutive particles of one release step) stay converged through the
    // recomputation and the reverse sweep.
    const bool valid = (int)threadIdx.x < tile.count;
    const long long slot = tile.first + (valid ? threadIdx.x : 0);
    const unsigned long long gid = (unsigned long long)(sc.id0 + (slot - sc.first_slot));
    const int sp = (int)release_step_of(sc, slot);
    const int tix = sc.m0_off + (sp - sc.rel_first);
    const float m0 = __ldg(P.m0 + tix);
    const float mq = __ldg(A.mq + tix);
    const int qidx = __ldg(A.qi + tix);
    float4 seg[CK + 1];
    signed char sfold[CK];
    for (int c = A.n_ck - 1; c >= 0; --c) {
        const int k_lo = c * CK, k_hi = min(A.n_steps, k_lo + CK);
        bool run = valid && sp < k_hi;
        float x = 0.f, y = 0.f, z = 0.f;
        if (run) {
            const float4 s0 = A.ckpt[(long long)c * A.n_slots + slot];
            const uint32_t st0 = __float_as_uint(s0.w) >> TAG_SHIFT;
            run = st0 == ST_ACTIVE || st0 == ST_UNRELEASED;        // else: event before k_lo
            x = s0.x; y = s0.y; z = s0.z;
            if (st0 == ST_UNRELEASED) { x = sc.src_x; y = sc.src_y; z = sc.src_z; }
        }
        if (!__any_sync(0xffffffffu, run)) continue;
        const int kstart = max(k_lo, sp);
        // recompute the segment: seg[k - k_lo] = state before step k
        bool alive = run;
        int klast = k_lo - 1;                // last step this lane took
        bool ev = false;
        for (int k = k_lo; k < k_hi; ++k) {
            if (alive && k >= kstart) {
                seg[k - k_lo] = make_float4(x, y, z, 0.f);
                const StepTime T = step_time<true>(P, sc.wind_offset, k);
                float fs;
                const uint32_t st = particle_step<false>(P, LV, T, sc, nullptr, gid, sp,
                                                         sig_h_uniform, T.du, T.dv, x, y, z,
                                                         &fs);
                sfold[k - k_lo] = (signed char)fs;
                klast = k;
                if (st != ST_ACTIVE) { alive = false; ev = true; }
            }
        }
        if (run) seg[klast + 1 - k_lo] = make_float4(x, y, z, 0.f);
        __syncwarp();
        // reverse sweep over the steps this lane took
        for (int k = k_hi - 1; k >= k_lo; --k) {
            if (!(run && k >= kstart && k <= klast)) continue;
            const int i = k - k_lo;
            const bool sample = (k + 1) % A.every == 0 && !(ev && k == klast);
            reverse_step<KHG>(P, A, LV, step_time<true>(P, sc.wind_offset, k), s_rec, s_w, gid, sp, m0,
                              mq, sig_h_uniform, sq2dt, seg[i], (float)sfold[i], seg[i + 1],
                              sample, J);
        }
        __syncwarp();
    }
    reduce_gradient(A, tile, J, valid, qidx, s_g, s_gq);
}

// Trajectory form: the forward kept every state, so the sweep reads them back (one
// coalesced 16-B row entry per step, prefetched one step ahead) instead of recomputing.
template <bool KHG>
__global__ void __launch_bounds__(ADJ_BLOCK)
adj_backward_traj_kernel(const StepParams P, const AdjParams A)
{
    extern __shared__ float4 s_dyn[];             // sized by the launch: adj_smem_backward
    float4 *s_rec = s_dyn;                        // [R]
    double *s_g = reinterpret_cast<double *>(s_rec + A.R);    // [6]
    double *s_gq = s_g + 6;                       // [nq]
    float *s_w = reinterpret_cast<float *>(s_gq + A.nq);      // [R]
    unsigned char *s_lut = reinterpret_cast<unsigned char *>(s_w + A.R);   // [n_lut]
    __shared__ float4 s_ent[MAX_LEVELS];           // warps span many levels here
    const auto LV = load_levels<Levels<true, false>>(P, s_lut, s_ent);
    const Tile tile = A.tiles[blockIdx.x];
    load_receptors(A, tile, s_rec, s_w, s_g, s_gq);
    const ScenDev sc = P.scen[tile.scen];
    const float sig_h_uniform = sqrtf(2.0f * P.k_scale * fmaxf(P.kh_uniform, 0.0f) * P.dt);
    const float sq2dt = sqrtf(2.0f * P.k_scale * P.dt);
    Adjoint J{0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    const bool valid = (int)threadIdx.x < tile.count;
    const long long slot = tile.first + (valid ? threadIdx.x : 0);
    const unsigned long long gid = (unsigned long long)(sc.id0 + (slot - sc.first_slot));
    const int sp = (int)release_step_of(sc, slot);
    const int tix = sc.m0_off + (sp - sc.rel_first);
    const float m0 = __ldg(P.m0 + tix);
    const float mq = __ldg(A.mq + tix);
    const int qidx = __ldg(A.qi + tix);
    const longlong2 tt = A.traj_tile[blockIdx.x];
    const float4 *row = A.traj + tt.x + threadIdx.x;
    const int k0 = (int)tt.y;
    float4 Xa = A.fin[slot];                      // state after the last step taken
    const uint32_t fw = __float_as_uint(Xa.w);
    const bool ev = (fw >> 31) != 0;
    // steps [kb, kn) of this lane (empty for padding lanes); rows exist from k0 on
    const int kn = valid ? (int)(fw & 0x7fffffffu) : 0;
    const int kb = valid ? max(sp, k0) : 0;
    // warp-uniform range with per-lane predicates, as in the checkpoint form
    const int k_top = __reduce_max_sync(0xffffffffu, kn) - 1;
    const int k_bot = __reduce_min_sync(0xffffffffu, kb < kn ? kb : 0x7fffffff);
    float4 Xn = make_float4(0.f, 0.f, 0.f, 0.f);
    const long long row0 = row - A.traj;
    if (k_top >= kb && k_top < kn &&
        LPM_IN_BOUNDS(P.err, row0 + (long long)(k_top - k0) * ADJ_BLOCK < A.traj_cap))
        Xn = __ldcs(row + (long long)(k_top - k0) * ADJ_BLOCK);
    for (int k = k_top; k >= k_bot; --k) {
        const bool act = k >= kb && k < kn;
        const float4 X = Xn;
        if (k - 1 >= kb && k - 1 < kn &&
            LPM_IN_BOUNDS(P.err, row0 + (long long)(k - 1 - k0) * ADJ_BLOCK < A.traj_cap))
            Xn = __ldcs(row + (long long)(k - 1 - k0) * ADJ_BLOCK);
        if (!act) continue;
        const bool sample = (k + 1) % A.every == 0 && !(ev && k == kn - 1);
        reverse_step<KHG>(P, A, LV, step_time<true>(P, sc.wind_offset, k), s_rec, s_w, gid, sp, m0, mq,
                          sig_h_uniform, sq2dt, X, X.w, Xa, sample, J);
        Xa = X;
    }
    reduce_gradient(A, tile, J, valid, qidx, s_g, s_gq);
}

// Dynamic shared memory of the kernels, sized by the receptors, the emission series and the
// level table
// (small arrays keep the shared-memory carve-out small and leave the rest of the SM's
// unified L1 to the weather gathers).
static size_t adj_smem_forward(const StepParams &P, const AdjParams &A, int groups = 1)
{
    return (size_t)A.R * (sizeof(float4) + groups * sizeof(double)) + (size_t)P.n_lut;
}

static size_t adj_smem_backward(const StepParams &P, const AdjParams &A, int groups = 1)
{
    return (size_t)A.R * (sizeof(float4) + groups * sizeof(float)) +
           (size_t)groups * (6 + A.nq) * sizeof(double) + (size_t)P.n_lut;
}

// ---------------------------------------------------------------------------------
// Sorted form: one launch per CK-step segment over the particles alive at its start in
// weather-cell order (with several scenarios: by scenario, then cell tile), then its
// releases; between segments the survivors are re-sorted (lpm_sort.cu). The states of a
// segment are stored row by row in that order; the backward sweeps the segments in
// reverse and hands dL/dX from one segment to the previous one through G.mu, indexed by
// home slot. A group of ADJ_BLOCK entries keeps the receptor sums and gradients of one
// scenario (its first entry's) in shared memory; entries of another scenario, at a scenario
// boundary of the sorted order, add theirs to the global sums directly.
// ---------------------------------------------------------------------------------

// Threads of the segment kernels' blocks, in groups of ADJ_BLOCK entries with receptor sums of
// their own. The forwards take two groups a block: neighbours in the sorted order then share
// the SM's L1 at nearly the same step (hits 86 -> 92 %) and one copy of the tables, of which
// more would cost blocks; 4 a SM (64 registers) with the trajectory, 3 (80) without, where
// the row stores do not hold it up (1e6 x 1080 and 2e5 x 720 with checkpoints, whole gradients:
// 15.8 and 5.3 ms; 4 and 4: 15.8 and 5.7; 3 and 3: 16.0 and 5.4; blocks of 512: 15.9 and 5.7).
// The reverse sweep at 5 blocks of 128 a SM (96 registers): blocks of 256 at 2 or 3 a SM 16.1 and
// 16.7 ms, of 384 16.4, of 640 16.6. Its one group a block is indexed as several would be: written
// for one alone it measured 15.28 -> 15.12 ms with one scenario (1e6 x 1080) and 33.35 -> 33.86
// with several (inversion of 16 x 1e5; start of the block, entries and sums changed one by one
// made no difference).
//
// FEW: segments of at most 4 groups an SM are bound by a step's latency: one group a block, 128
// registers a thread, the draws before the gathers so that the two overlap.
constexpr int SEG_BWD_BLOCK = 128;
constexpr int seg_fwd_block(bool few) { return few ? 128 : 256; }
constexpr int SEG_FEW = 4;

constexpr int seg_fwd_blocks(int mode, bool few)
{
    return few ? 4 : mode == SEG_STORE ? 4 : 3;
}

template <bool MULTI>
__device__ __forceinline__ bool seg_entry(const StepParams &P, const AdjSeg &G, int group,
                                          bool from_a, unsigned int live, long long &home,
                                          int &scen)
{
    const int lane = threadIdx.x % ADJ_BLOCK;
    if (from_a) {
        const long long e = (long long)group * ADJ_BLOCK + lane;
        if (e >= (long long)live) {
            scen = 0;
            home = P.scen[0].first_slot;
            return false;
        }
        home = G.ord[e];
        scen = MULTI ? scen_of(P, home) : 0;
        return true;
    }
    const Tile t = G.tiles[G.b_first + (group - G.tiles_a)];
    const bool ok = lane < t.count;
    scen = MULTI ? t.scen : 0;
    home = t.first + (ok ? lane : 0);
    return ok;
}

// The scenario of a group that has entries: that of its first one.
template <bool MULTI>
__device__ __forceinline__ int seg_group_scen(const StepParams &P, const AdjSeg &G, int group,
                                              bool from_a)
{
    if (!MULTI) return 0;
    if (from_a) return scen_of(P, G.ord[(long long)group * ADJ_BLOCK]);
    return G.tiles[G.b_first + (group - G.tiles_a)].scen;
}

// True when no group of the block starting at `group0` has entries: groups of A at or beyond
// the live count, groups beyond the segment's.
__device__ __forceinline__ bool seg_block_empty(const AdjSeg &G, int group0, int n, int n_groups,
                                                unsigned int live)
{
    for (int g = group0; g < min(group0 + n, n_groups); ++g)
        if (g >= G.tiles_a || (long long)g * ADJ_BLOCK < (long long)live) return false;
    return true;
}

// Receptor forward of a segment (MODE: SegMode). MULTI: entries of several scenarios (else
// all of scenario 0); FIELDS: a gridded K_h, or no level table. Instructions bound it as they do
// the advance kernel: the step times come from a table, the deposition words from one block for
// two steps, the samples by a countdown.
template <int MODE, bool MULTI, bool FIELDS, bool FEW>
__global__ void __launch_bounds__(seg_fwd_block(FEW), seg_fwd_blocks(MODE, FEW))
adj_forward_seg_kernel(const StepParams P, const AdjParams A, const AdjSeg G, int n_groups)
{
    constexpr bool SAMPLE = MODE != SEG_RECOMPUTE;          // receptor sums, sort inputs
    constexpr bool ROWS = MODE != SEG_CKPT;                 // every state into traj / fin
    constexpr int BLOCK = seg_fwd_block(FEW), GROUPS = BLOCK / ADJ_BLOCK;
    const int group0 = blockIdx.x * GROUPS;
    const unsigned int live = group0 < G.tiles_a ? *G.live : 0u;
    if (seg_block_empty(G, group0, GROUPS, n_groups, live)) return;
    extern __shared__ float4 s_dyn[];             // sized by the launch: adj_smem_forward
    float4 *s_rec = s_dyn;                        // [R]
    double *s_C = reinterpret_cast<double *>(s_rec + A.R);    // [GROUPS][R]
    unsigned char *s_lut = reinterpret_cast<unsigned char *>(s_C + GROUPS * A.R);   // [n_lut]
    __shared__ float4 s_ta[CK];                   // the segment's step times
    using Lev = Levels<MULTI, !FIELDS>;           // (the rule is at Levels)
    __shared__ float4 s_ent[Lev::SMEM ? MAX_LEVELS : 1];
    const Lev LV = load_levels<Lev>(P, s_lut, s_ent);
    for (int i = threadIdx.x; i < G.k_hi - G.k_lo; i += BLOCK)
        s_ta[i] = step_time_parts<true>(P, G.k_lo + i);
    if (SAMPLE) {
        for (int r = threadIdx.x; r < A.R; r += BLOCK) s_rec[r] = A.rec[r];
        for (int r = threadIdx.x; r < GROUPS * A.R; r += BLOCK) s_C[r] = 0.0;
    }
    __syncthreads();
    const int group = group0 + threadIdx.x / ADJ_BLOCK;
    const bool from_a = group < G.tiles_a;
    const bool used = group < n_groups && (!from_a || (long long)group * ADJ_BLOCK < (long long)live);
    double *C = s_C + (threadIdx.x / ADJ_BLOCK) * A.R;      // the group's sums
    const int bs = SAMPLE && used ? seg_group_scen<MULTI>(P, G, group, from_a) : 0;
    const float sig_h_uniform = sqrtf(P.k2 * fmaxf(P.kh_uniform, 0.0f) * P.dt);
    const uint32_t tab = shared_addr(s_ta);
    const long long e = (long long)group * ADJ_BLOCK + threadIdx.x % ADJ_BLOCK;
    long long home;
    int scen;
    if (used && seg_entry<MULTI>(P, G, group, from_a, live, home, scen)) {
        const ScenDev &sc = P.scen[scen];
        const unsigned long long gid =
            (unsigned long long)(__ldg(&sc.id0) + (home - __ldg(&sc.first_slot)));
        const int sp = (int)release_step_of(sc, home);
        const float m0 = __ldg(P.m0 + sc.m0_off + (sp - sc.rel_first));
        const float2 *wind = sc.wind_offset;
        float x = sc.src_x, y = sc.src_y, z = sc.src_z;
        if (from_a) {
            const float4 s0 = MODE == SEG_RECOMPUTE ? G.ck[e] : G.sorted[e];
            if (MODE == SEG_CKPT) G.ck[e] = s0;
            x = s0.x; y = s0.y; z = s0.z;
        }
        uint32_t st = ST_ACTIVE;
        int k = max(sp, G.k_lo);
        float4 *row = ROWS ? G.traj + (long long)(k - G.k_lo) * G.width + e : nullptr;
        int until = A.every - 1 - k % A.every;     // steps before the next sample step
        DepCache dc;
        dep_begin(P, gid, k, dc);
#pragma unroll 1
        do {
            const StepTime T = step_time_from(P, wind, ld_shared4(tab + 16 * (k - G.k_lo)), k);
            const float xb = x, yb = y, zb = z;
            float fs = 1.0f;
            st = particle_step<false, false, Lev, false, FIELDS, FEW>(
                P, LV, T, sc, nullptr, gid, sp, sig_h_uniform, T.du, T.dv, x, y, z,
                ROWS ? &fs : nullptr, nullptr, nullptr, &dc);
            if (ROWS) {
                __stcs(row, make_float4(xb, yb, zb, fs));
                row += G.width;
            }
            ++k;
            if (SAMPLE && --until < 0) {
                until = A.every - 1;
                if (st == ST_ACTIVE) {
                    const float m = m0 * expf(-P.lambda * (float)(k - sp) * P.dt) * A.inv_ns;
                    sample_receptors(A, s_rec, x, y, z, m,
                                     scen == bs ? C : A.C + (long long)scen * A.R);
                }
            }
        } while (st == ST_ACTIVE && k < G.k_hi);
        if (ROWS)
            G.fin[e] = make_float4(x, y, z, __uint_as_float((uint32_t)k |
                                                            (st != ST_ACTIVE ? 0x80000000u : 0u)));
        if (SAMPLE) {
            const float4 out = pack_state(x, y, z, st, sp);      // what the sort reads
            if (from_a) G.sorted[e] = out;
            else G.home[home] = out;
        }
    }
    if (SAMPLE) {
        __syncthreads();
        if (used)
            for (int r = threadIdx.x % ADJ_BLOCK; r < A.R; r += ADJ_BLOCK)
                if (C[r] != 0.0) atomicAdd(A.C + (long long)bs * A.R + r, C[r]);
    }
}

// Reverse sweep of a segment (KHG: gridded K_h, or no level table). Bound by the latency of
// its gathers at 19 warps an SM (96 registers hold the record differences; issue 56 % busy);
// a uniform K_h's scale is taken out of the loop, its vanishing derivative dropped (571 -> 480
// executed instructions a step with that, the tabled times and the shared round keys). The draws come
// before the gathers with several scenarios too, whose gathers miss the L1 more often
// (inversion of 16 x 1e5: 35.0 -> 34.2 ms); with one they measured no faster there.
template <bool KHG, bool MULTI, bool FEW>
__global__ void __launch_bounds__(SEG_BWD_BLOCK, FEW ? 4 : 5)
adj_backward_seg_kernel(const StepParams P, const AdjParams A, const AdjSeg G, int n_groups)
{
    constexpr int GROUPS = SEG_BWD_BLOCK / ADJ_BLOCK;
    const int group0 = blockIdx.x * GROUPS;
    const unsigned int live = group0 < G.tiles_a ? *G.live : 0u;
    if (seg_block_empty(G, group0, GROUPS, n_groups, live)) return;
    extern __shared__ float4 s_dyn[];             // sized by the launch: adj_smem_backward
    const int gi = threadIdx.x / ADJ_BLOCK;
    float4 *s_rec = s_dyn;                        // [R]
    double *s_g = reinterpret_cast<double *>(s_rec + A.R);    // [GROUPS][6]
    double *s_gq = s_g + 6 * GROUPS;              // [GROUPS][nq]
    float *s_w = reinterpret_cast<float *>(s_gq + GROUPS * A.nq);      // [GROUPS][R]
    unsigned char *s_lut = reinterpret_cast<unsigned char *>(s_w + GROUPS * A.R);   // [n_lut]
    s_g += 6 * gi;
    s_gq += A.nq * gi;
    s_w += A.R * gi;
    using Lev = Levels<MULTI, !KHG>;              // (the rule is at Levels)
    __shared__ float4 s_ent[Lev::SMEM ? MAX_LEVELS : 1];
    const Lev LV = load_levels<Lev>(P, s_lut, s_ent);
    // the segment's step times, once per block
    __shared__ float4 s_ta[CK];
    for (int i = threadIdx.x; i < G.k_hi - G.k_lo; i += SEG_BWD_BLOCK)
        s_ta[i] = step_time_parts<false>(P, G.k_lo + i);
    const int group = group0 + gi;
    const bool from_a = group < G.tiles_a;
    const bool used = group < n_groups && (!from_a || (long long)group * ADJ_BLOCK < (long long)live);
    Tile tb{0, 0, 0};
    if (used) tb.scen = seg_group_scen<MULTI>(P, G, group, from_a);
    load_receptors(A, tb, s_rec, s_w, s_g, s_gq);     // (ends with a barrier)
    const float sig_h_uniform = sqrtf(P.k2 * fmaxf(P.kh_uniform, 0.0f) * P.dt);
    const float sq2dt = sqrtf(2.0f * P.k_scale * P.dt);
    const uint32_t tab = shared_addr(s_ta);
    const long long e = (long long)group * ADJ_BLOCK + threadIdx.x % ADJ_BLOCK;
    long long home = P.scen[0].first_slot;
    int scen = 0;
    const bool valid = used && seg_entry<MULTI>(P, G, group, from_a, live, home, scen);
    const ScenDev &sc = P.scen[scen];
    const float2 *wind = sc.wind_offset;
    // receptor weights of another scenario than the group's come from global memory
    const double *wg = MULTI && scen != tb.scen ? A.w + (long long)scen * A.R : nullptr;
    const unsigned long long gid = (unsigned long long)(sc.id0 + (home - sc.first_slot));
    const int sp = (int)release_step_of(sc, home);
    const int tix = sc.m0_off + (sp - sc.rel_first);
    const float m0 = __ldg(P.m0 + tix);
    const float mq = __ldg(A.mq + tix);
    const int qidx = __ldg(A.qi + tix);
    float4 Xa = valid ? G.fin[e] : make_float4(0.f, 0.f, 0.f, 0.f);
    const uint32_t fw = __float_as_uint(Xa.w);
    const bool ev = (fw >> 31) != 0;
    const int kn = valid ? (int)(fw & 0x7fffffffu) : 0;
    const int kb = valid ? max(sp, G.k_lo) : 0;
    Adjoint J{0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    // a particle that ran through the segment carries dL/dX from the next one
    if (valid && !ev && kn == G.k_hi && G.k_hi < A.n_steps) {
        const float4 m = G.mu[home];
        J.mu0 = m.x; J.mu1 = m.y; J.mu2 = m.z;
    }
    // each lane sweeps its own steps, last first; a row is read one step ahead
    if (kb < kn) {
        int k = kn - 1;
        const float4 *row = G.traj + (long long)(k - G.k_lo) * G.width + e;
        float4 Xn = __ldcs(row);
        int since = (k + 1) % A.every;             // 0: step k is a sample step
        bool first = ev;                           // the step that ended the run has no sample
#pragma unroll 1
        do {
            const float4 X = Xn;
            row -= G.width;
            if (k > kb) Xn = __ldcs(row);
            const bool sample = since == 0 && !first;
            first = false;
            since = since == 0 ? A.every - 1 : since - 1;
            const StepTime T = step_time_from(P, wind, ld_shared4(tab + 16 * (k - G.k_lo)), k);
            reverse_step<KHG, FEW || MULTI>(P, A, LV, T, s_rec, s_w, gid, sp, m0, mq,
                                            sig_h_uniform, sq2dt, X, X.w, Xa, sample, J, wg);
            Xa = X;
        } while (--k >= kb);
    }
    // released earlier: hand mu to the previous segment; released here: mu is the
    // particle's share of the source partials
    if (sp < G.k_lo) {
        if (valid) G.mu[home] = make_float4(J.mu0, J.mu1, J.mu2, 0.f);
        J.mu0 = J.mu1 = J.mu2 = 0.f;
    }
    if (MULTI && valid && scen != tb.scen) {
        // another scenario than the group's: its partials straight into its gradient
        double *Gs = A.grad + (long long)scen * A.ng;
        atomicAdd(Gs + 0, (double)J.mu0);
        atomicAdd(Gs + 1, (double)J.mu1);
        atomicAdd(Gs + 2, (double)J.mu2);
        atomicAdd(Gs + 3 + A.nq + 0, (double)J.gsk);
        atomicAdd(Gs + 3 + A.nq + 1, (double)J.gbu);
        atomicAdd(Gs + 3 + A.nq + 2, (double)J.gbv);
        if (J.gq != 0.f) atomicAdd(Gs + 3 + qidx, (double)J.gq);
    }
    reduce_gradient(A, tb, J, valid && scen == tb.scen, qidx, s_g, s_gq);
}

// The kernels need a few KB of shared memory per block: ask for a small carve-out so the
// rest of the unified L1 serves the weather gathers (once per process). 10 % measured best
// (adjoint 1e6 particles: 25 % 1.20e10, 10 % 1.27e10, 5 % 1.08e10 particle-steps/s).
static void adj_set_carveout()
{
    const int pct = 10;
    cudaFuncSetAttribute(adj_forward_kernel<true>, cudaFuncAttributePreferredSharedMemoryCarveout, pct);
    cudaFuncSetAttribute(adj_forward_kernel<false>, cudaFuncAttributePreferredSharedMemoryCarveout, pct);
    cudaFuncSetAttribute(adj_backward_kernel<false>, cudaFuncAttributePreferredSharedMemoryCarveout, pct);
    cudaFuncSetAttribute(adj_backward_kernel<true>, cudaFuncAttributePreferredSharedMemoryCarveout, pct);
    cudaFuncSetAttribute(adj_backward_traj_kernel<true>, cudaFuncAttributePreferredSharedMemoryCarveout, pct);
    const void *seg[] = {
#define LPM_SEG_FWD_ALL(M) (const void *)adj_forward_seg_kernel<M, false, false, false>,   \
                           (const void *)adj_forward_seg_kernel<M, false, true, false>,     \
                           (const void *)adj_forward_seg_kernel<M, true, false, false>,     \
                           (const void *)adj_forward_seg_kernel<M, true, true, false>,      \
                           (const void *)adj_forward_seg_kernel<M, false, false, true>,     \
                           (const void *)adj_forward_seg_kernel<M, false, true, true>,      \
                           (const void *)adj_forward_seg_kernel<M, true, false, true>,      \
                           (const void *)adj_forward_seg_kernel<M, true, true, true>
        LPM_SEG_FWD_ALL(SEG_STORE), LPM_SEG_FWD_ALL(SEG_CKPT), LPM_SEG_FWD_ALL(SEG_RECOMPUTE),
#undef LPM_SEG_FWD_ALL
        (const void *)adj_backward_seg_kernel<false, false, false>,
        (const void *)adj_backward_seg_kernel<true, false, false>,
        (const void *)adj_backward_seg_kernel<false, true, false>,
        (const void *)adj_backward_seg_kernel<true, true, false>,
        (const void *)adj_backward_seg_kernel<false, false, true>,
        (const void *)adj_backward_seg_kernel<true, false, true>,
        (const void *)adj_backward_seg_kernel<false, true, true>,
        (const void *)adj_backward_seg_kernel<true, true, true>};
    for (const void *f : seg) cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, pct);
    (void)cudaGetLastError();
}

static void adj_prefer_l1()
{
    static std::once_flag once;              // contexts on several host threads may launch
    std::call_once(once, adj_set_carveout);
}

cudaError_t launch_adj_forward_seg(cudaStream_t s, const StepParams &P, const AdjParams &A,
                                   const AdjSeg &G, int n_groups, int mode, int n_sm)
{
    if (n_groups <= 0) return cudaSuccess;
    adj_prefer_l1();
    const bool few = n_groups <= SEG_FEW * n_sm;
    const int groups = seg_fwd_block(few) / ADJ_BLOCK;
    const int n = (n_groups + groups - 1) / groups;
    const size_t sm = adj_smem_forward(P, A, groups);
    const bool multi = P.n_scen > 1, fields = P.khpair || P.lut_last < 0;
#define LPM_SEG_FWD(M, U, F)                                                              \
    (few ? adj_forward_seg_kernel<M, U, F, true>                                          \
               <<<n, seg_fwd_block(true), sm, s>>>(P, A, G, n_groups)                     \
         : adj_forward_seg_kernel<M, U, F, false>                                         \
               <<<n, seg_fwd_block(false), sm, s>>>(P, A, G, n_groups))
#define LPM_SEG_FWD_MODE(M)                                                              \
    (multi ? (fields ? LPM_SEG_FWD(M, true, true) : LPM_SEG_FWD(M, true, false))          \
           : (fields ? LPM_SEG_FWD(M, false, true) : LPM_SEG_FWD(M, false, false)))
    switch (mode) {
    case SEG_STORE: LPM_SEG_FWD_MODE(SEG_STORE); break;
    case SEG_CKPT: LPM_SEG_FWD_MODE(SEG_CKPT); break;
    case SEG_RECOMPUTE: LPM_SEG_FWD_MODE(SEG_RECOMPUTE); break;
    default: return cudaErrorInvalidValue;
    }
#undef LPM_SEG_FWD_MODE
#undef LPM_SEG_FWD
    return cudaGetLastError();
}

cudaError_t launch_adj_backward_seg(cudaStream_t s, const StepParams &P, const AdjParams &A,
                                    const AdjSeg &G, int n_groups, int n_sm)
{
    if (n_groups <= 0) return cudaSuccess;
    adj_prefer_l1();
    const bool few = n_groups <= SEG_FEW * n_sm;
    constexpr int GROUPS = SEG_BWD_BLOCK / ADJ_BLOCK;
    const int n = (n_groups + GROUPS - 1) / GROUPS;
    const size_t sm = adj_smem_backward(P, A, GROUPS);
    const bool multi = P.n_scen > 1, fields = P.khpair || P.lut_last < 0;
#define LPM_SEG_BWD(K, U)                                                                 \
    (few ? adj_backward_seg_kernel<K, U, true><<<n, SEG_BWD_BLOCK, sm, s>>>(P, A, G, n_groups) \
         : adj_backward_seg_kernel<K, U, false><<<n, SEG_BWD_BLOCK, sm, s>>>(P, A, G, n_groups))
    if (fields && multi)
        LPM_SEG_BWD(true, true);
    else if (fields)
        LPM_SEG_BWD(true, false);
    else if (multi)
        LPM_SEG_BWD(false, true);
    else
        LPM_SEG_BWD(false, false);
#undef LPM_SEG_BWD
    return cudaGetLastError();
}

cudaError_t launch_adj_forward(cudaStream_t s, const StepParams &P, const AdjParams &A, int n_tiles)
{
    if (n_tiles <= 0) return cudaSuccess;
    adj_prefer_l1();
    if (A.traj)
        adj_forward_kernel<true><<<n_tiles, ADJ_BLOCK, adj_smem_forward(P, A), s>>>(P, A);
    else
        adj_forward_kernel<false><<<n_tiles, ADJ_BLOCK, adj_smem_forward(P, A), s>>>(P, A);
    return cudaGetLastError();
}

cudaError_t launch_adj_backward(cudaStream_t s, const StepParams &P, const AdjParams &A, int n_tiles)
{
    if (n_tiles <= 0) return cudaSuccess;
    adj_prefer_l1();
    // (the release-order sweep measured faster with the gridded-K_h branch kept at run time)
    const size_t sm = adj_smem_backward(P, A);
    if (A.traj)
        adj_backward_traj_kernel<true><<<n_tiles, ADJ_BLOCK, sm, s>>>(P, A);
    else if (P.khpair)
        adj_backward_kernel<true><<<n_tiles, ADJ_BLOCK, sm, s>>>(P, A);
    else
        adj_backward_kernel<false><<<n_tiles, ADJ_BLOCK, sm, s>>>(P, A);
    return cudaGetLastError();
}

}  // namespace lpm
