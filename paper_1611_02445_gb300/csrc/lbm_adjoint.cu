// lbm_adjoint.cu -- discrete adjoint of the fused step, with checkpoint and recompute.
//
// The paper has no adjoint. Forward map of one step: s_{t+1} = C(G s_t), where G is the
// gather with halfway bounce-back (a permutation of (direction, node) slots) and C the
// node-local collision. For a loss L(s_T):
//   lambda_T = dL/ds_T,
//   mu_t     = J_C(G s_t)^T lambda_{t+1}          (node-local),
//   lambda_t = G^T mu_t: lambda_k(x) = mu_k(x + c_k) if x + c_k is not solid, else
//              mu_inv(k)(x)   (the transpose of the bounce-back permutation),
// and dL/dF(x), dL/dtau accumulate (dC/dF)^T lambda and (dC/dtau)^T lambda.
// One adjoint kernel per step reads s_t with the forward gather and mu_{t+1} with the
// transposed gather (both pull-shaped) and writes mu_t. Gradients accumulate in FP64:
// per node for F_x, per CTA for tau (a CTA always walks the same groups, so the sums are
// deterministic for a device).
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "lbm_async.cuh"
#include "lbm_internal.cuh"
#include "lbm_store.cuh"

namespace lbm {

constexpr int ADJ_THREADS = GROUP_LANES;   // one thread per node of a work group
static_assert(GROUP_MAX_NODES == ADJ_THREADS && GROUP_MAX_NODES_F64 == ADJ_THREADS, "one thread per lane");
// Resident CTAs per SM: 38 values a node are in flight in registers (FP32: 3 x 256 threads at
// 80 registers keep 117 KB of gathers in flight per SM, FP64: 2 x 256 at 128 keep 156 KB).
template <int DT> constexpr int adj_ctas() { return DT == LBM_F64 ? 2 : 3; }

template <int DT> using Arith = typename Store<DT>::R;

// The work groups' tables as a kernel reads them.
struct NodeTables {
    const int4* groups;
    const uint32_t* fidx;
    const uint32_t* non_empty;
    int64_t n_groups;
    int Tx, plane_x;
    // x coordinate of the node n of the compact lists
    __device__ __forceinline__ int x_of(int64_t n) const {
        const uint32_t gi = fidx[n];
        return TILE * (int)(non_empty[gi >> 6] % (uint32_t)Tx) + (int)(gi & 3u);
    }
};

// Deterministic sum over a CTA in FP64, valid in thread 0.
__device__ __forceinline__ double block_sum(double v, double* sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < ADJ_THREADS / 32; w++) s += sh[w];
    __syncthreads();
    return s;
}

// rho and u_x = (j_x - F_x / 2) / rho of one stored node in FP64 (the loss and its seed).
template <int DT>
__device__ __forceinline__ void stored_ux(const typename Store<DT>::T* __restrict__ f, double Fx, double& r, double& ux) {
    double jx = 0.0;
    r = 0.0;
#pragma unroll
    for (int i = 0; i < Q; i++) {
        const double v = to_f64<DT>(f[i * GROUP_LANES], i);
        r += v;
        if (cx(i)) jx += cx(i) > 0 ? v : -v;
    }
    ux = (jx - 0.5 * Fx) / r;
}

// Outlet-flux loss, pass 1: per-CTA sums of u_x and node counts over the non-solid nodes of
// the plane x = plane_x, u = (sum c f* - F/2)/rho from the stored populations.
template <int DT>
__global__ void __launch_bounds__(ADJ_THREADS) k_loss_partials(const typename Store<DT>::T* __restrict__ f,
                                                               NodeTables nt, const Arith<DT>* __restrict__ gfield_c,
                                                               StepParams p, double* __restrict__ partials) {
    __shared__ double sh[ADJ_THREADS / 32];
    double su = 0.0, cnt = 0.0;
    for (int64_t g = blockIdx.x; g < nt.n_groups; g += gridDim.x) {
        const int4 h = nt.groups[g];
        const int t = threadIdx.x;
        if (t >= h.w || nt.x_of(h.z + t) != nt.plane_x) continue;
        double r, ux;
        stored_ux<DT>(f + (p.sg0 + g) * (Q * GROUP_LANES) + t, gfield_c ? (double)gfield_c[h.z + t] : p.g[0], r, ux);
        su += ux;
        cnt += 1.0;
    }
    su = block_sum(su, sh);
    cnt = block_sum(cnt, sh);
    if (threadIdx.x == 0) {
        partials[blockIdx.x * 2] = su;
        partials[blockIdx.x * 2 + 1] = cnt;
    }
}

// Fixed-order sum of partials with `width` components each: one CTA, every ADJ_THREADS-th
// partial per thread, then a tree. (A single thread per component took 118 us for the 6 441
// partials of a 128^3 pack, a chain of dependent loads and FP64 additions.)
__global__ void __launch_bounds__(ADJ_THREADS) k_sum_partials(const double* __restrict__ partials, int64_t nb, int width,
                                                              double* __restrict__ out) {
    __shared__ double sh[ADJ_THREADS / 32];
    for (int c = 0; c < width; c++) {
        double v = 0.0;
        for (int64_t b = threadIdx.x; b < nb; b += ADJ_THREADS) v += partials[b * width + c];
        v = block_sum(v, sh);
        if (threadIdx.x == 0) out[c] = v;
    }
}

// Density and momentum of the gathered populations: as in the collision, through sums and
// differences of opposite directions; FP64 as exact integers in 2^-58 fixed point when every
// population lies in [2^-6, 1) (no FP64 instruction), else in FP64. That bound keeps every sum
// below 19, where the fixed point holds 32: a density of any size is accepted here (LBM_F64_NATIVE
// steps it in FP64), and one of 3 or more has a rest population of 1 or more.
template <typename R> __device__ __forceinline__ void pull_moments(const R v[Q], R& sum, R j[3]) {
    const R s = ((v[0] + (v[1] + v[3])) + ((v[2] + v[4]) + (v[5] + v[6]))) +
                (((v[7] + v[9]) + (v[8] + v[10])) + ((v[11] + v[14]) + (v[12] + v[13]))) +
                ((v[15] + v[18]) + (v[16] + v[17]));
    const R d79 = v[7] - v[9], d810 = v[8] - v[10], d1114 = v[11] - v[14], d1213 = v[12] - v[13],
            d1518 = v[15] - v[18], d1617 = v[16] - v[17];
    sum = s;
    j[0] = (((v[1] - v[3]) + d79) - d810) + (d1114 + d1213);
    j[1] = (((v[2] - v[4]) + d79) + d810) + (d1518 + d1617);
    j[2] = (((v[5] - v[6]) + d1114) - d1213) + (d1518 - d1617);
}

// 1 / rho: FP32 as it is; FP64 near 1 from the pair reciprocal and one FP64 Newton step.
__device__ __forceinline__ float inverse(float rho, int64_t) { return 1.0f / rho; }
__device__ __forceinline__ double inverse(double rho, int64_t fix) {
    if (fix < (5ll << (FIX_SHIFT - 3)) || fix >= (7ll << (FIX_SHIFT - 2))) return 1.0 / rho;
    const double ir = df_to_double_pos(df_recip(df_from_fix(fix)));
    return __fma_rn(__fma_rn(-rho, ir, 1.0), ir, ir);
}

// Transposed collision Jacobian at one node, in moment form. v: gathered populations
// (f, or h = f - w for the shifted formats), lam: adjoint of the post-collision values.
// Replaces lam by mu (adjoint of the gathered values), returns dL/dF_x and sets tau1, tau2 with
// dL/dtau = (tau1 + tau2 / 2) omega^2. The weighted moments of lam come from the sums and
// differences of opposite directions: 210 operations in FP64, which bound the FP64 adjoint (2
// lanes per SM); written as 16 sums of 19 products each, whose terms with a zero coefficient
// the compiler has to keep, they were 500.
// XF: the force has no y or z component.
template <typename R, bool SHIFT, bool XF>
__device__ __forceinline__ R collide_adjoint(const R v[Q], R lam[Q], int type, const StepParams& p, R Fx, R Fy, R Fz,
                                             R& tau1, R& tau2) {
    const R w0 = R(wgt(0)), w1 = R(wgt(1)), w2 = R(wgt(7));
    R D, j[3];
    int64_t fix = 0;
    if constexpr (sizeof(R) == 8) {
        int64_t q[Q], fj[3];
        bool bad = false;
#pragma unroll
        for (int i = 0; i < Q; i++) q[i] = fix_from_double_fast(v[i], bad, 5u);
        fix_moments(q, fix, fj[0], fj[1], fj[2]);
        D = fix_to_double(fix);
        for (int a = 0; a < 3; a++) j[a] = fix_to_double(fj[a]);
        if (bad) {
            pull_moments(v, D, j);
            fix = 0;
        }
    } else {
        pull_moments(v, D, j);
    }
    const R rho = SHIFT ? R(1) + D : D;
    const R ir = inverse(rho, fix);
    const R ux = (j[0] + R(0.5) * Fx) * ir, uy = (XF ? j[1] : j[1] + R(0.5) * Fy) * ir,
            uz = (XF ? j[2] : j[2] + R(0.5) * Fz) * ir;
    // weighted moments of lam
    const R lx = lam[1] + lam[3], ly = lam[2] + lam[4], lz = lam[5] + lam[6];
    const R a1 = lam[7] + lam[9], a2 = lam[8] + lam[10], b1 = lam[11] + lam[14], b2 = lam[12] + lam[13],
            c1 = lam[15] + lam[18], c2 = lam[16] + lam[17];
    const R pxy = a1 + a2, pxz = b1 + b2, pyz = c1 + c2;
    const R d79 = lam[7] - lam[9], d810 = lam[8] - lam[10], d1114 = lam[11] - lam[14], d1213 = lam[12] - lam[13],
            d1518 = lam[15] - lam[18], d1617 = lam[16] - lam[17];
    const R M0 = w0 * lam[0] + (w1 * ((lx + ly) + lz) + w2 * ((pxy + pxz) + pyz));
    const R M1x = w1 * (lam[1] - lam[3]) + w2 * ((d79 - d810) + (d1114 + d1213));
    const R M1y = w1 * (lam[2] - lam[4]) + w2 * ((d79 + d810) + (d1518 + d1617));
    const R M1z = w1 * (lam[5] - lam[6]) + w2 * ((d1114 - d1213) + (d1518 - d1617));
    const R Mxx = w1 * lx + w2 * (pxy + pxz), Myy = w1 * ly + w2 * (pxy + pyz), Mzz = w1 * lz + w2 * (pxz + pyz);
    const R Mxy = w2 * (a1 - a2), Mxz = w2 * (b1 - b2), Myz = w2 * (c1 - c2);
    R rhobar = 0, ubx = 0, uby = 0, ubz = 0, Fbx = 0;
    R keep = 0;   // coefficient of lam_i kept in mu_i
    tau1 = tau2 = R(0);
    if (type == LBM_INLET) {
        const R ex = par<R>(p.u_in[0], p.u_in_f[0]), ey = par<R>(p.u_in[1], p.u_in_f[1]),
                ez = par<R>(p.u_in[2], p.u_in_f[2]);
        const R M2ex = Mxx * ex + Mxy * ey + Mxz * ez, M2ey = Mxy * ex + Myy * ey + Myz * ez,
                M2ez = Mxz * ex + Myz * ey + Mzz * ez;
        rhobar = M0 * (R(1) - R(1.5) * (ex * ex + ey * ey + ez * ez)) + R(3) * (M1x * ex + M1y * ey + M1z * ez) +
                 R(4.5) * (ex * M2ex + ey * M2ey + ez * M2ez);
#pragma unroll
        for (int i = 0; i < Q; i++) lam[i] = rhobar;
        return R(0);
    }
    const R M2ux = Mxx * ux + Mxy * uy + Mxz * uz, M2uy = Mxy * ux + Myy * uy + Myz * uz,
            M2uz = Mxz * ux + Myz * uy + Mzz * uz;
    // gradient of the second-order equilibrium in u: 3 M1 + 9 M2 u - 3 u M0
    const R M03 = R(3) * M0;
    const R gx = R(3) * M1x + (R(9) * M2ux - M03 * ux), gy = R(3) * M1y + (R(9) * M2uy - M03 * uy),
            gz = R(3) * M1z + (R(9) * M2uz - M03 * uz);
    if (type == LBM_OUTLET) {
        const R ro = par<R>(p.rho_out, p.rho_out_f);
        ubx = ro * gx;
        uby = ro * gy;
        ubz = ro * gz;
    } else {
        const R omega = par<R>(p.omega, p.omega_f), beta = par<R>(p.beta, p.beta_f);
        const R uu = ux * ux + uy * uy + uz * uz, uF = XF ? ux * Fx : ux * Fx + uy * Fy + uz * Fz;
        const R M1u = M1x * ux + M1y * uy + M1z * uz, M1F = XF ? M1x * Fx : M1x * Fx + M1y * Fy + M1z * Fz;
        const R uM2u = ux * M2ux + uy * M2uy + uz * M2uz;
        const R M2Fx = XF ? Mxx * Fx : Mxx * Fx + Mxy * Fy + Mxz * Fz, M2Fy = XF ? Mxy * Fx : Mxy * Fx + Myy * Fy + Myz * Fz,
                M2Fz = XF ? Mxz * Fx : Mxz * Fx + Myz * Fy + Mzz * Fz;
        const R uM2F = XF ? M2ux * Fx : M2ux * Fx + M2uy * Fy + M2uz * Fz;
        const R P = R(3) * M1u + (R(4.5) * uM2u - R(1.5) * uu * M0);   // sum w lam (e_i - 1)
        rhobar = omega * (M0 + P);
        const R orho = omega * rho, b9 = R(9) * beta, b3M0 = beta * M03;
        ubx = orho * gx + (b9 * M2Fx - b3M0 * Fx);
        uby = orho * gy + (XF ? b9 * M2Fy : b9 * M2Fy - b3M0 * Fy);
        ubz = orho * gz + (XF ? b9 * M2Fz : b9 * M2Fz - b3M0 * Fz);
        Fbx = beta * gx;
        // dL/dtau: sum lam (v - v^eq) / tau^2 + (1/(2 tau^2)) sum lam w Q
        R Lv = lam[0] * v[0];
#pragma unroll
        for (int i = 1; i < Q; i++) Lv += lam[i] * v[i];
        tau1 = Lv - (D * M0 + rho * P);
        tau2 = R(3) * M1F - M03 * uF + R(9) * uM2F;
        keep = R(1) - omega;
    }
    Fbx += R(0.5) * ubx * ir;
    rhobar -= (ubx * ux + uby * uy + ubz * uz) * ir;
    const R jbx = ubx * ir, jby = uby * ir, jbz = ubz * ir;
    const auto put = [&](int a, int b, R c) {
        lam[a] = keep * lam[a] + (rhobar + c);
        lam[b] = keep * lam[b] + (rhobar - c);
    };
    lam[0] = keep * lam[0] + rhobar;
    put(1, 3, jbx);
    put(2, 4, jby);
    put(5, 6, jbz);
    put(7, 9, jbx + jby);
    put(8, 10, jby - jbx);
    put(11, 14, jbx + jbz);
    put(12, 13, jbx - jbz);
    put(15, 18, jby + jbz);
    put(16, 17, jby - jbz);
    return Fbx;
}

// One reverse step: mu_out = J_C(G s_t)^T lambda_{t+1}, lambda_{t+1} = G^T mu_in. The first one
// (sT not NULL) takes the seed lambda_T = dL/df* = (c_x - u_x)/(rho |P|) on the plane, 0
// elsewhere, and starts the per-node gradient with the direct term dL/dF_x = -1/(2 rho |P|).
//
// Persistent CTAs walk the work groups, one thread per non-solid node; the next group's
// neighbour records, words, ranks and forces come in by cp.async while a group is computed,
// its header a group earlier. A node's 19 sources are formed as in the step (record + rank;
// the bounced ones are its own) and serve both gathers: the forward one of direction i and,
// with the same source, the transposed one of direction inv(i), lambda_inv(i)(x) =
// mu_inv(i)(x - c_i). The 38 loads go to registers and are all in flight before the
// arithmetic. I32: as in the step, all indices fit 31 bits.
//
// 128^3 pack, FP32 (0.84 M nodes): 71 us with one 128-thread CTA per 128 nodes that looked up the
// neighbour ranks, lanes and masks of each source (long-scoreboard stalls), 52 us with one CTA
// per work group and no prefetch, 40 us so (ncu, cold). 80^3 pack, FP64 (0.2 M nodes): 195 -> 94 us,
// FP64 pipe 80 % busy with about 220 operations a node.
template <int DT> struct AdjSmem {
    static constexpr int MAX_TILES = DT == LBM_F64 ? GROUP_MAX_TILES_F64 : GROUP_MAX_TILES_4B;
    int4 hdr[4];
    int4 rec[2][MAX_TILES * (NBR_STRIDE / 2)];
    uint4 rank[2][ADJ_THREADS];
    uint32_t word[2][ADJ_THREADS];
    Arith<DT> gf[2][ADJ_THREADS];
    double sum[ADJ_THREADS / 32];
};

template <int DT, bool XF, bool I32>
__global__ void __launch_bounds__(ADJ_THREADS, adj_ctas<DT>())
k_adjoint(const typename Store<DT>::T* st, const typename Store<DT>::T* sT, const Arith<DT>* mu_in,
          Arith<DT>* mu_out, NodeTables nt,   // not __restrict__: the launch before may still write them

          const int64_t* __restrict__ nrec, const uint32_t* __restrict__ fword, const uint4* __restrict__ frank,
          const Arith<DT>* __restrict__ gfield_c, StepParams p, const double* __restrict__ sums, double* gbar,
          double* tau_part) {
    using R = Arith<DT>;
    using IX = typename std::conditional<I32, int32_t, int64_t>::type;
    constexpr int CH = NBR_STRIDE / 2;   // 16-byte chunks of a tile's records
    __shared__ AdjSmem<DT> sm;
    const int64_t G = gridDim.x;
    const int t = threadIdx.x;
    const auto issue_header = [&](int64_t g, int it) {
        if (t == 0 && g < nt.n_groups) cp_async16(&sm.hdr[it & 3], nt.groups + g);
    };
    const auto issue_meta = [&](int64_t g, int it) {
        if (g >= nt.n_groups) return;
        const int4 h = sm.hdr[it & 3];
        const int slot = it & 1;
        const int4* src = reinterpret_cast<const int4*>(nrec + (int64_t)h.x * NBR_STRIDE);
        for (int k = t; k < h.y * CH; k += ADJ_THREADS) cp_async16(&sm.rec[slot][k], src + k);
        if (t < h.w) {
            cp_async4(&sm.word[slot][t], fword + h.z + t);
            cp_async16(&sm.rank[slot][t], frank + h.z + t);
            if (gfield_c) {
                if (sizeof(R) == 8) cp_async8(&sm.gf[slot][t], gfield_c + h.z + t);
                else cp_async4(&sm.gf[slot][t], gfield_c + h.z + t);
            }
        }
    };
    const int64_t g0 = G - 1 - blockIdx.x;   // as in k_step_run: the CTAs with one group more come last
    issue_header(g0, 0);
    issue_header(g0 + G, 1);
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    issue_meta(g0, 0);
    cp_async_commit();
    grid_wait();   // the tables are constant; from here on the launch before is complete
    grid_release();
    R tau1 = R(0), tau2 = R(0), err1 = R(0), err2 = R(0);
    int it = 0;
    for (int64_t g = g0; g < nt.n_groups; g += G, it++) {
        cp_async_wait<0>();
        __syncthreads();   // meta(g), header(g + G) visible; slot (it + 1) & 1 no longer read
        issue_meta(g + G, it + 1);
        issue_header(g + 2 * G, it + 2);
        cp_async_commit();
        const int4 h = sm.hdr[it & 3];
        if (t >= h.w) continue;
        const int64_t n = (int64_t)h.z + t;
        const int slot = it & 1;
        const uint32_t w = sm.word[slot][t];
        const uint4 rk = sm.rank[slot][t];
        const int type = (int)((w >> WORD_TYPE_SHIFT) & 3u);
        const int lt = (int)((w >> WORD_LT_SHIFT) & (uint32_t)WORD_LT_MASK), s = (int)((w >> WORD_SLOT_SHIFT) & 63u);
        const int x = s & 3, y = (s >> 2) & 3, z = s >> 4;
        const IX own = (IX)((p.sg0 + g) * (Q * GROUP_LANES)) + t;
        const char* r13 = reinterpret_cast<const char*>(sm.rec[slot]) + (lt * NBR_STRIDE + 13) * 8;
        const int oxm = ((x - 1) >> 2) * 8, oxp = ((x + 1) >> 2) * 8;
        const int oym = ((y - 1) >> 2) * 24, oyp = ((y + 1) >> 2) * 24;
        const int ozm = ((z - 1) >> 2) * 72, ozp = ((z + 1) >> 2) * 72;
        R v[Q], lam[Q];
#pragma unroll
        for (int i = 0; i < Q; i++) {
            IX src = own;   // the source's index in data block 0
            bool bounce = false;
            if (i > 0) {
                const int off = (cx(i) > 0 ? oxm : cx(i) < 0 ? oxp : 0) + (cy(i) > 0 ? oym : cy(i) < 0 ? oyp : 0) +
                                (cz(i) > 0 ? ozm : cz(i) < 0 ? ozp : 0);
                bounce = (w >> i) & 1u;
                const IX nsrc = *reinterpret_cast<const IX*>(r13 + off) + (IX)rank_of(rk, i);   // I32: the low word
                src = bounce ? own : nsrc;
            }
            v[i] = to_arith<DT>(st[src + (bounce ? inv(i) : i) * GROUP_LANES], i);
            if (!sT) lam[inv(i)] = mu_in[src + (bounce ? i : inv(i)) * GROUP_LANES];
        }
        const R Fx = gfield_c ? sm.gf[slot][t] : par<R>(p.g[0], p.g_f[0]);
        double gb = 0.0;
        if (!sT) {
            gb = __ldcg(gbar + n);
        } else {
            const bool plane = nt.x_of(n) == nt.plane_x;
            double r = 1.0, ux = 0.0;
            const double count = sums[1];
            if (plane) {
                stored_ux<DT>(sT + own, gfield_c ? (double)Fx : p.g[0], r, ux);
                gb = -0.5 / (r * count);
            }
#pragma unroll
            for (int i = 0; i < Q; i++) lam[i] = plane ? (R)((cx(i) - ux) / (r * count)) : R(0);
        }
        R a1, a2;
        const R Fb = collide_adjoint<R, Store<DT>::SHIFT, XF>(v, lam, type, p, Fx, par<R>(p.g[1], p.g_f[1]),
                                                              par<R>(p.g[2], p.g_f[2]), a1, a2);
#pragma unroll
        for (int i = 0; i < Q; i++) mu_out[own + i * GROUP_LANES] = lam[i];
        gbar[n] = gb + (double)Fb;
        // dL/dtau over the thread's nodes: FP64 as it is, FP32 as sum and error (TwoSum)
        if constexpr (sizeof(R) == 8) {
            tau1 += a1;
            tau2 += a2;
        } else {
            const dfl s1 = two_sum(tau1, a1), s2 = two_sum(tau2, a2);
            tau1 = s1.h;
            err1 += s1.l;
            tau2 = s2.h;
            err2 += s2.l;
        }
    }
    cp_async_wait<0>();
    const double total = block_sum(((double)tau1 + (double)err1) + 0.5 * ((double)tau2 + (double)err2), sm.sum);
    if (t == 0) tau_part[g0] = __ldcg(tau_part + g0) + total;   // times omega^2: applied to the sum
}

// Per-node gradient in group order -> dense array (zeroed by the caller).
__global__ void __launch_bounds__(ADJ_THREADS) k_gbar_dense(const double* __restrict__ gbar, NodeTables nt, int nx,
                                                            int ny, int Ty, int64_t n_nodes, double* __restrict__ dense) {
    for (int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; n < n_nodes; n += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t gi = nt.fidx[n];
        const int s = (int)(gi & 63u);
        const uint32_t tile = nt.non_empty[gi >> 6], row = tile / (uint32_t)nt.Tx;
        const int x = TILE * (int)(tile - row * (uint32_t)nt.Tx) + (s & 3);
        const int y = TILE * (int)(row % (uint32_t)Ty) + ((s >> 2) & 3);
        const int z = TILE * (int)(row / (uint32_t)Ty) + (s >> 4);
        dense[x + (int64_t)nx * (y + (int64_t)ny * z)] = gbar[n];
    }
}

namespace {

// One device allocation cut into 256-byte aligned parts.
struct Workspace {
    char* p = nullptr;
    size_t size = 0;
    size_t part(size_t bytes) {
        const size_t at = size;
        size += (std::max<size_t>(bytes, 1) + 255) / 256 * 256;
        return at;
    }
    cudaError_t alloc() { return dmalloc(reinterpret_cast<void**>(&p), size); }
    template <typename T> T* at(size_t off) const { return reinterpret_cast<T*>(p + off); }
    ~Workspace() {
        if (p) dfree(p);
    }
};

// Persistent grid of the reverse step, and the number of its dL/dtau partials.
template <int DT> int64_t adj_grid(const lbm_ctx* c) {
    return std::max<int64_t>(1, std::min<int64_t>(c->n_groups, 152 * adj_ctas<DT>()));
}

template <int DT, bool XF>
cudaError_t launch_reverse(lbm_ctx* c, const void* st, const void* sT, const Arith<DT>* mu_in, Arith<DT>* mu_out,
                           const NodeTables& nt, const double* sums, double* gbar, double* taup, bool chained) {
    using TT = typename Store<DT>::T;
    const Arith<DT>* gf = c->gfield ? static_cast<const Arith<DT>*>(c->gfield_c) : nullptr;
    const TT *a = static_cast<const TT*>(st), *b = static_cast<const TT*>(sT);
    const unsigned grid = (unsigned)adj_grid<DT>(c);
    return launch_chained(idx32(c) ? k_adjoint<DT, XF, true> : k_adjoint<DT, XF, false>, grid, (unsigned)ADJ_THREADS, 0,
                          c->stream, chained, a, b, mu_in, mu_out, nt, c->nrec, c->fword, c->frank, gf, c->p, sums, gbar,
                          taup);
}

template <int DT>
cudaError_t run_adjoint(lbm_ctx* c, int T, int K, int plane_x, double* loss, double* dL_dg, int dg_on_device,
                        double* dL_dtau, bool* started) {
    using TT = typename Store<DT>::T;
    using R = Arith<DT>;
    cudaError_t e;
    const size_t copy = ((size_t)c->n_sgroups * Q * GROUP_LANES * sizeof(TT) + 255) / 256 * 256;
    const bool grads = dL_dg || dL_dtau;
    const int n_ck = (T + K - 1) / K;        // segments; s_0, s_K, ... are their first states
    const int seg_len = std::min(K, T);
    const int nbl = (int)std::max<int64_t>(1, std::min<int64_t>(c->n_groups, 152 * 4));
    const size_t N = (size_t)c->nx * c->ny * c->nz;
    const bool host_dense = grads && dL_dg && !dg_on_device;
    // One allocation before any work, so that a failure leaves the state as it was: the
    // checkpoints after the first (s_0 stays in the context's own copy), one segment's
    // states, two adjoint buffers and the FP64 gradient accumulators. (Nine allocations took
    // about 0.1 ms each to make and release.)
    Workspace ws;
    const size_t lossp = ws.part(sizeof(double) * 2 * nbl), sums = ws.part(sizeof(double) * 2);
    size_t ck = 0, seg = 0, mu0 = 0, mu1 = 0, gbar = 0, taup = 0, dense = 0;
    if (grads) {
        ck = ws.part(copy * (n_ck - 1));
        seg = ws.part(copy * seg_len);
        mu0 = ws.part((size_t)c->n_sgroups * Q * GROUP_LANES * sizeof(R));
        mu1 = ws.part((size_t)c->n_sgroups * Q * GROUP_LANES * sizeof(R));
        gbar = ws.part(sizeof(double) * c->n_own_nonsolid);
        taup = ws.part(sizeof(double) * adj_grid<DT>(c));
        if (host_dense) dense = ws.part(N * sizeof(double));
    }
    if ((e = ws.alloc()) != cudaSuccess) return e;
    *started = true;
    // Forward. Without gradients the context's two copies alternate as in lbm_step. With them
    // every state goes where the reverse sweep reads it: the first state of a segment into its
    // checkpoint, the others of the last segment into the segment's slots (which the reverse
    // sweep then need not recompute), s_T into the context's other copy; the states between
    // alternate between that copy and a slot of the segment not yet in use.
    char* const ckp = ws.at<char>(ck);
    char* const sb = ws.at<char>(seg);
    const void* const s0 = c->f[c->cur];
    void* const other = c->f[1 - c->cur];
    const auto first_of = [&](int sgi) -> const void* { return sgi == 0 ? s0 : ckp + copy * (sgi - 1); };
    if (!grads) {
        for (int t = 0; t < T; t++) {
            if ((e = launch_step(c, c->f[c->cur], c->f[1 - c->cur], t > 0)) != cudaSuccess) return e;
            c->cur ^= 1;
        }
    } else {
        const int last = n_ck - 1, t_last = last * K;   // the last segment: states t_last ... T - 1
        const void* from = s0;
        for (int t = 0; t < T; t++) {
            void* to;
            if (t + 1 == T) to = other;
            else if ((t + 1) % K == 0) to = ckp + copy * ((t + 1) / K - 1);
            else if (t + 1 > t_last) to = sb + copy * (t + 1 - t_last);
            else to = from == other ? static_cast<void*>(sb) : other;
            if ((e = launch_step(c, from, to, t > 0)) != cudaSuccess) return e;
            from = to;
        }
        c->cur ^= 1;
    }
    // loss on s_T
    const TT* sT = static_cast<const TT*>(c->f[c->cur]);
    const NodeTables nt = {c->groups, c->fidx, c->non_empty, c->n_groups, c->Tx, plane_x};
    k_loss_partials<DT><<<nbl, ADJ_THREADS, 0, c->stream>>>(
        sT, nt, c->gfield ? static_cast<const R*>(c->gfield_c) : nullptr, c->p, ws.at<double>(lossp));
    k_sum_partials<<<1, ADJ_THREADS, 0, c->stream>>>(ws.at<double>(lossp), nbl, 2, ws.at<double>(sums));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    double h_sums[2] = {0.0, 0.0};
    if ((e = cudaMemcpyAsync(h_sums, ws.at<double>(sums), sizeof(h_sums), cudaMemcpyDeviceToHost, c->stream)) !=
        cudaSuccess)
        return e;
    if ((e = cudaStreamSynchronize(c->stream)) != cudaSuccess) return e;
    *loss = h_sums[1] > 0 ? h_sums[0] / h_sums[1] : 0.0;
    if (!grads || h_sums[1] == 0) {
        if (dL_dtau) *dL_dtau = 0.0;
        if (dL_dg && h_sums[1] == 0) {
            if (dg_on_device) e = cudaMemsetAsync(dL_dg, 0, N * sizeof(double), c->stream);
            else std::fill(dL_dg, dL_dg + N, 0.0);
        }
        return e;
    }
    // reverse sweep
    if ((e = cudaMemsetAsync(ws.at<double>(taup), 0, sizeof(double) * adj_grid<DT>(c), c->stream)) != cudaSuccess) return e;
    R* mu[2] = {ws.at<R>(mu0), ws.at<R>(mu1)};
    int mcur = 0;
    const bool xf = c->p.g[1] == 0.0 && c->p.g[2] == 0.0;
    const auto reverse = [&](const void* st, const void* seed) {
        mcur ^= 1;
        return xf ? launch_reverse<DT, true>(c, st, seed, mu[1 - mcur], mu[mcur], nt, ws.at<double>(sums),
                                             ws.at<double>(gbar), ws.at<double>(taup), !seed)
                  : launch_reverse<DT, false>(c, st, seed, mu[1 - mcur], mu[mcur], nt, ws.at<double>(sums),
                                              ws.at<double>(gbar), ws.at<double>(taup), !seed);
    };
    for (int sgi = n_ck - 1; sgi >= 0; sgi--) {
        const int t0 = sgi * K, t1 = std::min(T, t0 + K);
        const auto state = [&](int t) -> const void* { return t == t0 ? first_of(sgi) : sb + copy * (t - t0); };
        if (sgi != n_ck - 1)
            for (int t = t0 + 1; t < t1; t++)
                if ((e = launch_step(c, state(t - 1), sb + copy * (t - t0), true)) != cudaSuccess) return e;
        for (int t = t1 - 1; t >= t0; t--)
            if ((e = reverse(state(t), t == T - 1 ? sT : nullptr)) != cudaSuccess) return e;
    }
    double tau_sum = 0.0;
    if (dL_dtau) {
        k_sum_partials<<<1, ADJ_THREADS, 0, c->stream>>>(ws.at<double>(taup), adj_grid<DT>(c), 1, ws.at<double>(sums));
        if ((e = cudaMemcpyAsync(&tau_sum, ws.at<double>(sums), sizeof(double), cudaMemcpyDeviceToHost, c->stream)) !=
            cudaSuccess)
            return e;
    }
    if (dL_dg) {
        double* d = dg_on_device ? dL_dg : ws.at<double>(dense);
        if ((e = cudaMemsetAsync(d, 0, N * sizeof(double), c->stream)) != cudaSuccess) return e;
        const unsigned gs = (unsigned)std::max<int64_t>(
            1, std::min<int64_t>((c->n_own_nonsolid + ADJ_THREADS - 1) / ADJ_THREADS, 152 * 32));
        k_gbar_dense<<<gs, ADJ_THREADS, 0, c->stream>>>(ws.at<double>(gbar), nt, c->nx, c->ny, c->Ty, c->n_own_nonsolid, d);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if (!dg_on_device) {
            if ((e = cudaMemcpyAsync(dL_dg, d, N * sizeof(double), cudaMemcpyDeviceToHost, c->stream)) != cudaSuccess)
                return e;
        }
    }
    e = cudaStreamSynchronize(c->stream);
    if (dL_dtau) *dL_dtau = tau_sum * (c->p.omega * c->p.omega);
    return e;
}

}  // namespace

cudaError_t launch_adjoint(lbm_ctx* c, int T, int K, int plane_x, double* loss, double* dL_dg, int dg_on_device,
                           double* dL_dtau, bool* started) {
    *started = false;
    switch (c->dtype) {
        case LBM_F64: return run_adjoint<LBM_F64>(c, T, K, plane_x, loss, dL_dg, dg_on_device, dL_dtau, started);
        case LBM_F32: return run_adjoint<LBM_F32>(c, T, K, plane_x, loss, dL_dg, dg_on_device, dL_dtau, started);
        default: return run_adjoint<LBM_F16S>(c, T, K, plane_x, loss, dL_dg, dg_on_device, dL_dtau, started);
    }
}

}  // namespace lbm
