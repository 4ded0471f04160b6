// adjoint_kernels.cu -- reverse-mode derivative (adjoint) of one coupled time
// step of liblbp (sm_103a).
//
// The forward step n (lbm_kernels.cu, particle_kernels.cu) maps the
// post-collision populations fhat^{n-1} and the particle state (r^n, V^n) to
// fhat^n and (r^{n+1}, V^{n+1}):
//   f_a(x)   = fhat^{n-1}_a(x - e_a)                               (Eq. 20)
//   rho~, u  = sum_a f_a, sum_a e_a f_a                            (Eqs. 12-13)
//   F_H      = gamma U_inf e^N from u at the 8 cell corners        (Eq. 8; or Eq. 7 / Eq. 6)
//   F(x_p)  += -F_H W_p(q)                                          (Eq. 9)
//   V' = V + (F_H + F_R + F_ext)/M,  r' = r + V'                   (Eqs. 1-2)
//   fhat_a   = (1 - w) f_a + w f^eq_a(rho~, u) + 3 w_a F.e_a,  w = 1/tau   (Eqs. 15, 17-19)
// Given the adjoints lam = dL/dfhat^n (FP32 planes), dL/dV^{n+1}, dL/dr^{n+1},
// these kernels produce dL/dfhat^{n-1}, dL/dV^n, dL/dr^n and add this step's
// share of dL/domega, dL/dgamma_i, dL/dR_i, dL/dM_i and dL/dkT.
//
// k_adj_particles : eight lanes per particle, one per corner of its cell, a
//   vector's components one per lane (as k_particles, and for the same reason:
//   an FP64 warp instruction takes 64 cycles whatever its lanes).  From the
//   recorded state it gathers u(x_p), re-evaluates the particle's forward step
//   in FP64 and runs what the chain rule needs of it through the update and
//   the random force -- all before the launch dependency resolves, beside the
//   lattice kernel of the reverse step before; then it gathers
//   lam_F(x_p) = sum_a 3 w_a e_a lam_a(x_p) (the adjoint of the body-force term)
//   and runs the chain rule back through the spreading weights and the
//   Stokeslet fit, about 90 FP64 instructions for four particles.  What the fit
//   sends back to the fluid is lam_u(x_p), the adjoint of the node velocity at
//   each corner: it is appended, as (x, 3 FP64 values), to the 256-byte record
//   of the corner's row segment (the same records the forward step uses for
//   forces), and the segments of the next reverse step are marked for its
//   lattice kernel.  Before, a gather kernel and an FP64 kernel with all of a
//   particle's components in every lane took 4.3 + 13.6 us with 8 particles and
//   47 + 87 us with 16384, and the replay copied the particle state twice a step;
//   a reverse sweep of 200 steps at 64^3: 13.3 -> 6.6 ms with its replay (and the
//   recording, which copied the trajectory twice a step, 4.0 -> 2.0 ms), of 20
//   steps at 256^3: 28.5 -> 26.3 ms.
// k_adj_lattice : the fused adjoint of collision, moments and streaming, one
//   thread per node, one block per 128-node row segment:
//     lam_feq_a = w lam_a
//     lam_rho   = w sum_a w_a lam_a
//     lam_u     = w sum_a w_a lam_a (3 e_a + 9 (e_a.u) e_a - 3 u) + lam_u(particles)
//     lam_f_a   = (1 - w) lam_a + lam_rho + e_a.lam_u
//     dL/dw    += sum_a lam_a (f^eq_a - f_a)
//   and, streaming being a permutation, dL/dfhat^{n-1}_a(x - e_a) = lam_f_a(x).
//   The adjoint buffer holds dL/df (the streamed populations) rather than
//   dL/dfhat, so that every node stores its 15 results at its own address
//   (aligned, like the forward pass) and reads dL/dfhat^n_a(x) as the value at
//   x + e_a (a shifted read, which the forward pass shows costs nothing).  It
//   reads that, the populations fhat^{n-1} (pulled, as forward) and writes
//   the result: 180 bytes per node in FP32.  The record entries of a node are summed in an order fixed by
//   their values, so the result does not depend on which particle appended
//   first; entries that did not fit a record go to a dense FP64 buffer (FP64
//   atomics, order-dependent in that rare case).  dL/dw is summed per block in
//   FP32 and added in FP64 to the block's own accumulator slot (no atomics).
#include <cuda_runtime.h>

#include <cstring>

#include "lbp_internal.cuh"

namespace lbp {

struct AdjPArgs {
    const void *g;           // fhat^{n-1}, storage type St, 15 planes of P
    const float *lam;        // dL/dfhat^n, FP32, 15 planes of P
    long long P, N;
    const int *prep;         // box of each particle (batches)
    const double *r, *v;     // r^n, V^n, [3][cap]
    const double *prev_r;    // r of the next reverse step (to mark its segments), or null
    int cap, np;
    const double *fext, *inv_mass, *gamma, *radius, *sig;
    const unsigned char *pinned;
    double kT;
    unsigned long long seed;
    long long step;          // Philox counter of step n
    double sqrt3;
    int mode, exclude_inside;
    const double *gv, *gr;   // dL/dV^{n+1}, dL/dr^{n+1}: [np][3] or null
    double *lam_v, *lam_r;   // in: adjoint of V^{n+1}, r^{n+1}; out: of V^n, r^n ([3][cap])
    double *acc;             // [4][np]: dL/dgamma, dL/dR, dL/dM, dL/dkT (added)
    unsigned long long *rec; // records of this adjoint step
    double *fqd;             // [3][N] overflow accumulator (FP64)
    unsigned *marks;         // the next reverse step's marks, or null
    unsigned mark_epoch;
};

constexpr int APN = 16;              // particles per block
constexpr int AP_T = 8 * APN + 32;   // eight threads each, and the triggering warp

// the sum over the three components of a value held one component per lane
__device__ __forceinline__ double sum_over_components(double v) {
    return from_comp(v, 0) + from_comp(v, 1) + from_comp(v, 2);
}

template <typename St, int MAXR>
__global__ void __launch_bounds__(AP_T, 3) k_adj_particles(const AdjPArgs A, const RepTable<MAXR> rt) {
    if (threadIdx.x >= 8 * APN) {
        // lets this reverse step's lattice kernel launch as soon as the one before
        // is complete (see k_particles)
        grid_dependency_wait();
        grid_dependents_launch();
        return;
    }
    const typename St::T *G = static_cast<const typename St::T *>(A.g);
    const int p = threadIdx.x & 7, kc = comp_of(p);
    const int ip = blockIdx.x * APN + (threadIdx.x >> 3);
    const bool live = ip < A.np;
    const int i = live ? ip : A.np - 1, cap = A.cap;  // lanes past the last particle shadow it (no stores)
    const int ik = kc * cap + i;
    const double rk = __ldcg(A.r + ik), Vk = __ldcg(A.v + ik);
    double lV = __ldcg(A.lam_v + ik) + (A.gv ? A.gv[3 * (size_t)i + kc] : 0.0);
    double lr = __ldcg(A.lam_r + ik) + (A.gr ? A.gr[3 * (size_t)i + kc] : 0.0);
    const double fek = A.fext[ik];
    const double gam = A.gamma[i], R = A.radius[i], invM = A.inv_mass[i], sg = A.sig[i];
    const bool pin = A.pinned[i] != 0;
    const Rep &rp = rt.rep[MAXR == 1 ? 0 : A.prep[i]];
    const int nx = rp.nx, ny = rp.ny, nz = rp.nz;
    const double bk = floor(rk), qk = rk - bk;
    const int base = (int)bk;
    const int c0 = p & 1, c1 = (p >> 1) & 1, c2 = p >> 2;
    const int X = wrapi(from_comp(base, 0) + c0, nx), Y = wrapi(from_comp(base, 1) + c1, ny),
              Z = wrapi(from_comp(base, 2) + c2, nz);
    const int xs[3] = {wrapi(X + 1, nx), X, wrapi(X - 1, nx)};
    const int ys[3] = {wrapi(Y + 1, ny), Y, wrapi(Y - 1, ny)};
    const int zs[3] = {wrapi(Z + 1, nz), Z, wrapi(Z - 1, nz)};
    // u(x_p) of the streamed f (pull)
    double u[3];
    {
        float s[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int a = 1; a < Q; ++a) {
            const float g = St::gather(G + ((long long)a * A.P + rp.node_off +
                                            ((long long)zs[ez(a) + 1] * ny + ys[ey(a) + 1]) * nx + xs[ex(a) + 1]), a);
            if (ex(a)) s[0] += ex(a) > 0 ? g : -g;
            if (ey(a)) s[1] += ey(a) > 0 ? g : -g;
            if (ez(a)) s[2] += ez(a) > 0 ? g : -g;
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) u[k] = widen_f32(s[k]);
    }
    // the random force of this step (same Philox numbers as the forward step)
    unsigned long long ctr[4] = {(unsigned long long)A.step, (unsigned long long)i, 0ull, 0ull};
    philox4x64_10(ctr, A.seed, 0ull);
    const unsigned long long bits = kc == 0 ? ctr[0] : kc == 1 ? ctr[1] : ctr[2];
    const double xi =
        __dmul_rn(A.sqrt3, __fma_rn(__ull2double_rn(2ull * (bits >> 11) + 1ull), 0x1.0p-53, -1.0));
    const double FR = __dmul_rn(sg, xi);
    // this corner's trilinear weight W_p and dW_p/dq_k
    const double q0 = from_comp(qk, 0), q1 = from_comp(qk, 1), q2 = from_comp(qk, 2);
    const double t0 = c0 ? q0 : 1.0 - q0, t1 = c1 ? q1 : 1.0 - q1, t2 = c2 ? q2 : 1.0 - q2;
    const double t01 = t0 * t1, Wp = t01 * t2;
    const double dw[3] = {c0 ? t1 * t2 : -(t1 * t2), c1 ? t0 * t2 : -(t0 * t2), c2 ? t01 : -t01};
    // forward re-evaluation of F_H (component kc), with the fit's corner terms
    const double V[3] = {from_comp(Vk, 0), from_comp(Vk, 1), from_comp(Vk, 2)};
    double FH = 0.0, e[3] = {0.0, 0.0, 0.0}, ek = 0.0, U = 0.0, num = 0.0, inw = 0.0, iden = 0.0, urk = 0.0;
    double d[3] = {0.0, 0.0, 0.0}, ir = 0.0, ir3 = 0.0, x = 0.0, k1 = 0.0, k2 = 0.0, av[3] = {0.0, 0.0, 0.0};
    bool fit = false, use = false;
    const double cR = 0.75 * R;
    if (A.mode == LBP_STOKESLET) {
        d[0] = (double)c0 - q0;
        d[1] = (double)c1 - q1;
        d[2] = (double)c2 - q2;
        const double mk = (sum_components(u[0], u[1], u[2], p) - 8.0 * Vk) * 0.125;
        const double mm = sum_over_components(mk * mk);
        if (mm > 0.0) inw = rsqrt(mm);
        ek = mk * inw;
#pragma unroll
        for (int k = 0; k < 3; ++k) e[k] = from_comp(ek, k);
        const double rr = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
        ir = rr > 0.0 ? rsqrt(rr) : 0.0;
        const double dist = rr * ir;
        const bool moving = mm > 0.0;
        use = moving && !(dist < 1e-12 || (A.exclude_inside && dist < R));
        double pn = 0.0, pd = 0.0;
        if (use) {
            ir3 = ir * ir * ir;
            x = e[0] * d[0] + e[1] * d[1] + e[2] * d[2];
            k1 = 1.0 - cR * ir;
            k2 = cR * x * ir3;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                av[k] = k1 * e[k] - k2 * d[k];
                pn += (u[k] - V[k]) * av[k];
                pd += av[k] * av[k];
            }
        }
        const double nd = sum_pair(pn, pd, p);
        num = __shfl_sync(0xffffffffu, nd, 0, 8);
        const double den = __shfl_sync(0xffffffffu, nd, 1, 8);
        if (moving && den != 0.0) {
            iden = 1.0 / den;
            U = num * iden;
            fit = true;
        }
        FH = gam * U * ek;
    } else if (A.mode == LBP_POINTWISE) {
        urk = sum_components(Wp * u[0], Wp * u[1], Wp * u[2], p);
        FH = -gam * (Vk - urk);
    } else {
        FH = -gam * Vk;
    }
    // r' = r + V'  then  V' = V + (F_H + F_R + F_ext)/M, backwards
    double lFH = 0.0, gG = 0.0, gR = 0.0, gM = 0.0, gK = 0.0;
    if (!pin) {
        lV += lr;
        lFH = lV * invM;
    }
    {
        const double lFR_xi = sum_over_components(lFH * xi);
        const double lF_tot = sum_over_components(lV * (FH + FR + fek));
        if (!pin) {
            gM = -lF_tot * invM * invM;
            // F_R = sigma xi, sigma = sqrt(2 gamma kT)
            if (sg > 0.0) {
                const double isg = 1.0 / sg;
                gG += lFR_xi * (A.kT * isg);
                gK += lFR_xi * (gam * isg);
            }
        }
    }
    const double F[3] = {from_comp(FH, 0), from_comp(FH, 1), from_comp(FH, 2)};
    int next_seg = 0;  // the row segment of corner p of the next reverse step's cell
    if (A.marks && A.prev_r) {
        const int b = (int)floor(__ldcg(A.prev_r + ik));
        const int x1 = wrapi(from_comp(b, 0) + c0, nx), y1 = wrapi(from_comp(b, 1) + c1, ny),
                  z1 = wrapi(from_comp(b, 2) + c2, nz);
        next_seg = (int)(rp.seg_off + ((long long)z1 * ny + y1) * rp.nchunks + x1 / SEG);
    }

    // ---- the lattice kernel of the reverse step before is complete
    // (it read its marks from the array that the next step's go to)
    grid_dependency_wait();
    if (A.marks && A.prev_r && live) A.marks[next_seg] = A.mark_epoch;
    double lq = 0.0, lu[3] = {0.0, 0.0, 0.0};  // adjoints of q (component kc) and of u(x_p)
    if (A.mode != LBP_BROWNIAN) {
        // lam_F(x_p) (aligned): dL/dfhat_a(x_p) = dL/df^{n+1}_a(x_p + e_a), the buffer's layout
        float s[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int a = 1; a < Q; ++a) {
            const float l = (3.f * wgtf(a)) *
                            __ldcg(A.lam + ((long long)a * A.P + rp.node_off +
                                            ((long long)zs[1 - ez(a)] * ny + ys[1 - ey(a)]) * nx + xs[1 - ex(a)]));
            if (ex(a)) s[0] += ex(a) > 0 ? l : -l;
            if (ey(a)) s[1] += ey(a) > 0 ? l : -l;
            if (ez(a)) s[2] += ez(a) > 0 ? l : -l;
        }
        const double lF[3] = {widen_f32(s[0]), widen_f32(s[1]), widen_f32(s[2])};
        // F(x_p) += -F_H W_p(q)
        double fl = F[0] * lF[0] + F[1] * lF[1] + F[2] * lF[2];
        lFH -= sum_components(Wp * lF[0], Wp * lF[1], Wp * lF[2], p);
        const double lf[3] = {from_comp(lFH, 0), from_comp(lFH, 1), from_comp(lFH, 2)};
        if (A.mode == LBP_STOKESLET) {
            // the adjoint of the fit, with zero terms where there was none
            const double eF = e[0] * lf[0] + e[1] * lf[1] + e[2] * lf[2];
            const double lU = fit ? gam * eF : 0.0;
            if (fit) gG += U * eF;
            const double lnum = lU * iden, lden = -lnum * num * iden;
            double ple[3] = {0.0, 0.0, 0.0}, plc = 0.0, pq[3] = {fl * dw[0], fl * dw[1], fl * dw[2]};
            if (use && fit) {
                double la[3];
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    lu[k] = lnum * av[k];
                    la[k] = lnum * (u[k] - V[k]) + 2.0 * lden * av[k];
                }
                const double dla = d[0] * la[0] + d[1] * la[1] + d[2] * la[2];
                const double lk1 = e[0] * la[0] + e[1] * la[1] + e[2] * la[2];
                const double c3 = cR * ir3;
                const double cd = c3 * lk1 + 3.0 * dla * (k2 * (ir * ir)), ce = c3 * dla;  // of d_k and e_k below
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    ple[k] = k1 * la[k] - ce * d[k];
                    pq[k] += cd * d[k] - k2 * la[k] - ce * e[k];
                }
                plc = -lk1 * ir - dla * x * ir3;
            }
            const double le = gam * U * lFH + sum_components(ple[0], ple[1], ple[2], p);
            lq = -sum_components(pq[0], pq[1], pq[2], p);
            const double lc = sum_pair(plc, 0.0, p);  // in even lanes
            if (fit) gR += 0.75 * lc;
            // e = m/|m| with m the mean of the w_p
            const double ee = sum_over_components(ek * le);
            const double lm = fit ? (le - ek * ee) * (inw * 0.125) : 0.0;
#pragma unroll
            for (int k = 0; k < 3; ++k) lu[k] += from_comp(lm, k);
            // w_p = u_p - V
            lV -= sum_components(lu[0], lu[1], lu[2], p);
        } else {
            gG += -sum_over_components((Vk - urk) * lFH);
            const double ul = gam * (u[0] * lf[0] + u[1] * lf[1] + u[2] * lf[2]);
            fl -= ul;
            lq = -sum_components(fl * dw[0], fl * dw[1], fl * dw[2], p);
            lV -= gam * lFH;
#pragma unroll
            for (int k = 0; k < 3; ++k) lu[k] = gam * Wp * lf[k];
        }
    } else {
        gG += -sum_over_components(Vk * lFH);
        lV -= gam * lFH;
    }
    if (!live) return;  // past the shuffles
    if (p < 3) {
        A.lam_v[ik] = lV;
        A.lam_r[ik] = lr + lq;  // q = r - floor(r)
    }
    // gG and gK are in every lane, gR in the even ones
    if (p < 4) {
        double *acc = A.acc + (size_t)(p == 2 ? 1 : p == 1 ? 2 : p) * A.np + i;
        *acc = __ldcg(acc) + (p == 0 ? gG : p == 1 ? gM : p == 2 ? gR : gK);
    }
    // lam_u(x_p) of this corner to the record of its row segment
    if (A.mode != LBP_BROWNIAN && !(lu[0] == 0.0 && lu[1] == 0.0 && lu[2] == 0.0)) {
        const long long row = (long long)Z * ny + Y;
        unsigned long long *rec = A.rec + (size_t)(rp.seg_off + row * rp.nchunks + X / SEG) * REC_WORDS;
        const unsigned int slot = atomicAdd(reinterpret_cast<unsigned int *>(rec), 1u);
        if (slot < (unsigned)REC_SLOTS) {
            reinterpret_cast<int *>(rec + REC_X0)[slot] = X;
#pragma unroll
            for (int k = 0; k < 3; ++k)
                rec[REC_F0 + 3 * slot + k] = (unsigned long long)__double_as_longlong(lu[k]);
        } else {
            const long long node = rp.node_off + row * nx + X;
#pragma unroll
            for (int k = 0; k < 3; ++k) atomicAdd(A.fqd + k * A.N + node, lu[k]);
        }
    }
}

// Sum the record entries whose x is this node's in ascending order of their
// value bits (a fixed order whatever the order of the appends).
__device__ __forceinline__ void adj_record_sum(const unsigned long long *rec, unsigned mask,
                                               double &a0, double &a1, double &a2) {
    while (mask) {
        int best = -1;
        unsigned long long b0 = 0, b1 = 0, b2 = 0;
        for (unsigned m = mask; m; m &= m - 1) {
            const int sl = __ffs(m) - 1;
            const unsigned long long v0 = __ldcg(rec + REC_F0 + 3 * sl), v1 = __ldcg(rec + REC_F0 + 3 * sl + 1),
                                     v2 = __ldcg(rec + REC_F0 + 3 * sl + 2);
            if (best < 0 || v0 < b0 || (v0 == b0 && (v1 < b1 || (v1 == b1 && v2 < b2)))) {
                best = sl;
                b0 = v0;
                b1 = v1;
                b2 = v2;
            }
        }
        a0 += __longlong_as_double((long long)b0);
        a1 += __longlong_as_double((long long)b1);
        a2 += __longlong_as_double((long long)b2);
        mask &= ~(1u << best);
    }
}

// At least 6 blocks per SM: 80 registers (32 bytes spilled) instead of 96,
// measured 6.5% faster at 256^3 (more bytes in flight per SM).
template <typename St, int MAXR>
__global__ void __launch_bounds__(SEG, 6) k_adj_lattice(const typename St::T *__restrict__ G,
                                                     const float *lam, float *lam_out,
                                                     long long P, const RepTable<MAXR> rt,
                                                     const unsigned long long *rec_cur,
                                                     unsigned long long *rec_prev, double *fqd,
                                                     long long N, double *acc_omega, const Marks mk, bool flip) {
    __shared__ float s_red[SEG / 32];
    // the block's box (batches: one block per row segment of every box, in box
    // order); consecutive reverse steps run through them in opposite directions,
    // so that each first reads what the one before wrote last (in L2)
    const unsigned block = flip ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
    const int rb = find_block_rep(rt, block);
    const Rep &rp = rt.rep[rb];
    const int nx = rp.nx, ny = rp.ny, nz = rp.nz, nchunks = rp.nchunks;
    const float omega = rp.omega;
    const unsigned item = block - rt.item_off[rb];
    const unsigned row = divide(item, rp.dchunks);
    const int chunk = (int)(item - row * (unsigned)nchunks);
    const size_t seg = (size_t)rp.seg_off + (size_t)row * nchunks + chunk;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) rec_prev[seg * REC_WORDS] = 0ull;
    const int x0 = chunk * SEG + threadIdx.x;
    const bool act = x0 < nx;
    const int x = act ? x0 : nx - 1;
    // node index and the offsets of x - e (index e + 1), periodic
    const int z = (int)divide(row, rp.dny), y = (int)(row - (unsigned)z * ny);
    const int slab = nx * ny;
    const int d = (int)rp.node_off + (int)row * nx + x;
    const int ox[3] = {x == nx - 1 ? 1 - nx : 1, 0, x == 0 ? nx - 1 : -1};
    const int oy[3] = {y == ny - 1 ? (1 - ny) * nx : nx, 0, y == 0 ? (ny - 1) * nx : -nx};
    const int oz[3] = {z == nz - 1 ? (1 - nz) * slab : slab, 0, z == 0 ? (nz - 1) * slab : -slab};
    float g[Q], l[Q];
#pragma unroll
    for (int a = 0; a < Q; ++a) {
        const int o = ox[ex(a) + 1] + oy[ey(a) + 1] + oz[ez(a) + 1];   // x - e_a
        const int op = ox[1 - ex(a)] + oy[1 - ey(a)] + oz[1 - ez(a)];  // x + e_a
        g[a] = St::gather(G + (long long)a * P + d + o, a);
        // dL/dfhat^n_a(x) = dL/df^{n+1}_a(x + e_a): the buffer holds the latter
        l[a] = __ldcg(lam + (long long)a * P + d + op);
    }
    // the records come from this reverse step's particle kernel: only marked
    // segments wait for it (and block 0, so that this grid never ends before it)
    const bool marked = mk.epoch == 0 || __ldcg(mk.seg + seg) == mk.epoch;
    if (marked || blockIdx.x == 0) grid_dependency_wait();
    grid_dependents_launch();
    const unsigned long long rw = marked ? __ldcg(rec_cur + seg * REC_WORDS + lane) : 0ull;
    // particle contributions lam_u(x)
    float pu0 = 0.f, pu1 = 0.f, pu2 = 0.f;
    const int cnt = (int)(unsigned)(__shfl_sync(0xffffffffu, rw, 0) & 0xffffffffull);
    if (cnt > 0) {
        const int used = cnt < REC_SLOTS ? cnt : REC_SLOTS;
        unsigned mask = 0;
        for (int sl = 0; sl < used; ++sl) {
            const unsigned long long xw2 = __shfl_sync(0xffffffffu, rw, REC_X0 + (sl >> 1));
            if ((int)(unsigned)(xw2 >> (32 * (sl & 1))) == x) mask |= 1u << sl;
        }
        double a0 = 0.0, a1 = 0.0, a2 = 0.0;
        if (mask && act)
            adj_record_sum(rec_cur + seg * REC_WORDS, mask, a0, a1, a2);
        if (cnt > REC_SLOTS && act) {
            a0 += __ldcg(fqd + d);
            a1 += __ldcg(fqd + N + d);
            a2 += __ldcg(fqd + 2 * N + d);
            fqd[d] = 0.0;
            fqd[N + d] = 0.0;
            fqd[2 * N + d] = 0.0;
        }
        pu0 = (float)a0;
        pu1 = (float)a1;
        pu2 = (float)a2;
    }
    // forward moments and equilibrium (deviation form, as the forward kernel)
    float drho = 0.f;
#pragma unroll
    for (int a = 0; a < Q; ++a) drho += g[a];
    const float c78 = g[7] - g[8], c910 = g[9] - g[10], c1112 = g[11] - g[12], c1314 = g[13] - g[14];
    const float ux = (g[1] - g[2]) + c78 + c910 + c1112 - c1314;
    const float uy = (g[3] - g[4]) + c78 + c910 - c1112 + c1314;
    const float uz = (g[5] - g[6]) + c78 - c910 + c1112 + c1314;
    const float base = drho - 1.5f * (ux * ux + uy * uy + uz * uz);
    // dL/domega partial and the equilibrium-part adjoints, per opposite pair
    float dom = l[0] * ((2.f / 9.f) * base - g[0]);
    float swl = (2.f / 9.f) * l[0];  // sum_a w_a lam_a
    float lx = 0.f, ly = 0.f, lz = 0.f;  // sum_pairs W e (3 d + 9 eu s)
#define LBP_ADJ_PAIR(A, W, EX, EY, EZ)                                              \
    {                                                                               \
        const float eu = (EX) * ux + (EY) * uy + (EZ) * uz;                         \
        const float sym = (W) * (base + 4.5f * eu * eu);                            \
        const float anti = (3.f * (W)) * eu;                                        \
        dom += l[A] * (sym + anti - g[A]) + l[A + 1] * (sym - anti - g[A + 1]);     \
        const float s = l[A] + l[A + 1], dd = l[A] - l[A + 1];                      \
        swl += (W) * s;                                                             \
        const float c = (W) * (3.f * dd + 9.f * eu * s);                            \
        lx += (EX) * c;                                                             \
        ly += (EY) * c;                                                             \
        lz += (EZ) * c;                                                             \
    }
    LBP_ADJ_PAIR(1, 1.f / 9.f, 1.f, 0.f, 0.f)
    LBP_ADJ_PAIR(3, 1.f / 9.f, 0.f, 1.f, 0.f)
    LBP_ADJ_PAIR(5, 1.f / 9.f, 0.f, 0.f, 1.f)
    LBP_ADJ_PAIR(7, 1.f / 72.f, 1.f, 1.f, 1.f)
    LBP_ADJ_PAIR(9, 1.f / 72.f, 1.f, 1.f, -1.f)
    LBP_ADJ_PAIR(11, 1.f / 72.f, 1.f, -1.f, 1.f)
    LBP_ADJ_PAIR(13, 1.f / 72.f, -1.f, 1.f, 1.f)
#undef LBP_ADJ_PAIR
    const float lrho = omega * swl;
    const float lux = omega * lx - 3.f * ux * lrho + pu0;
    const float luy = omega * ly - 3.f * uy * lrho + pu1;
    const float luz = omega * lz - 3.f * uz * lrho + pu2;
    const float om1 = 1.f - omega;
    if (act) {
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            const float v = om1 * l[a] + lrho + (float)ex(a) * lux + (float)ey(a) * luy + (float)ez(a) * luz;
            lam_out[(long long)a * P + d] = v;  // dL/df^n_a(x), aligned
        }
    }
    // dL/domega: the block's 128 terms summed in FP32 (fixed tree), added in
    // FP64 to the block's own slot.  (A tree of FP64 shuffles kept the narrow
    // FP64 pipe of this GPU busy at every block's end.)
    float v = act ? dom : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) s_red[warp] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < SEG / 32; ++w) s += s_red[w];
        acc_omega[block] = __ldcg(acc_omega + block) + (double)s;
    }
}

template <typename F>
static cudaError_t by_storage_adj(int precision, F &&f) {
    switch (precision) {
        case LBP_BF16: return f(StoreBF16{});
        case LBP_F16: return f(StoreF16{});
        default: return f(StoreF32{});
    }
}

// The box table of an adjoint launch: every box with its blocks of one
// 128-node row segment each (item_off, for the lattice kernel) -- one entry
// for a single box.
template <int MAXR>
static RepTable<MAXR> adj_table(const Sim &s) {
    RepTable<MAXR> t;
    memset(&t, 0, sizeof(t));
    t.nrep = s.nrep;
    unsigned off = 0;
    for (int r = 0; r < s.nrep; ++r) {
        t.rep[r] = s.reps[r];
        t.item_off[r] = off;
        off += (unsigned)s.reps[r].ny * (unsigned)s.reps[r].nz * (unsigned)s.reps[r].nchunks;
    }
    t.item_off[s.nrep] = off;
    return t;
}

// Run f(RepTable<1 or MAX_BATCH>) for a single box or a batch.
template <typename F>
static cudaError_t by_batch_adj(const Sim &s, F &&f) {
    if (s.nrep == 1) return f(adj_table<1>(s));
    return f(adj_table<MAX_BATCH>(s));
}

cudaError_t launch_adj_particles(Sim &s, const AdjStep &a, cudaStream_t st, bool chained) {
    if (s.np == 0) return cudaSuccess;
    AdjPArgs A;
    A.g = a.g;
    A.lam = a.lam;
    A.P = s.P;
    A.N = s.N;
    A.prep = s.prep;
    A.r = a.state;
    A.v = a.state + 3 * (size_t)s.cap;
    A.prev_r = a.prev_state;
    A.cap = s.cap;
    A.np = s.np;
    A.fext = s.fext;
    A.inv_mass = s.inv_mass;
    A.gamma = s.gamma;
    A.radius = s.radius;
    A.sig = s.sig;
    A.pinned = s.pinned;
    A.kT = s.kT;
    A.seed = s.seed;
    A.step = a.step;
    A.sqrt3 = s.sqrt3;
    A.mode = s.mode;
    A.exclude_inside = s.exclude_inside;
    A.gv = a.gv;
    A.gr = a.gr;
    A.lam_v = a.lam_v;
    A.lam_r = a.lam_r;
    A.acc = a.acc;
    A.rec = s.rec[a.parity];
    A.fqd = reinterpret_cast<double *>(s.fq);
    A.marks = a.next && s.mode != LBP_BROWNIAN ? s.marks[a.next & 1] : nullptr;
    A.mark_epoch = a.next;
    const unsigned grid = (unsigned)((s.np + APN - 1) / APN);
    return by_batch_adj(s, [&](const auto &rt) {
        constexpr int MAXR = sizeof(rt.rep) / sizeof(Rep);
        return by_storage_adj(s.precision, [&](auto tag) {
            using St = decltype(tag);
            return launch_k(k_adj_particles<St, MAXR>, grid, AP_T, 0, st, chained, A, rt);
        });
    });
}

cudaError_t launch_adj_lattice(Sim &s, const AdjStep &a, cudaStream_t st, bool pdl) {
    const unsigned grid = (unsigned)adj_lattice_blocks(s);
    const Marks mk{s.marks[a.epoch & 1], a.epoch};
    return by_batch_adj(s, [&](const auto &rt) {
        constexpr int MAXR = sizeof(rt.rep) / sizeof(Rep);
        return by_storage_adj(s.precision, [&](auto tag) {
            using St = decltype(tag);
            const unsigned long long *rec = s.rec[a.parity];
            return launch_k(k_adj_lattice<St, MAXR>, grid, SEG, 0, st, pdl, static_cast<const typename St::T *>(a.g),
                            a.lam, a.lam_out, (long long)s.P, rt, rec, s.rec[a.parity ^ 1],
                            reinterpret_cast<double *>(s.fq), (long long)s.N, a.acc_omega, mk, a.parity != 0);
        });
    });
}

// Marks pay where the lattice kernel's blocks are more than are resident (six per SM).
bool adj_lattice_marks(const Sim &s) { return s.np > 0 && adj_lattice_blocks(s) > 6 * s.num_sms; }

int adj_lattice_blocks(const Sim &s) {
    int n = 0;
    for (int r = 0; r < s.nrep; ++r) n += s.reps[r].ny * s.reps[r].nz * s.reps[r].nchunks;
    return n;
}

int adj_lattice_first_block(const Sim &s, int replica) {
    int n = 0;
    for (int r = 0; r < replica; ++r) n += s.reps[r].ny * s.reps[r].nz * s.reps[r].nchunks;
    return n;
}

// dL/dfhat_a(y) of the first recorded state = dL/df_a(y + e_a) of its first
// step (the buffer's layout), to the FP64 [15][N] ABI layout, every box periodic on its own.
// A block serves SEG consecutive nodes, 15 values a thread in flight together, widened
// on their bits: the FP64 pipe and two 64-bit divisions a value took 1.75 ms at
// 256^3, the bytes take 0.45 ms; measured 0.44 ms.
template <int MAXR>
__global__ void __launch_bounds__(SEG) k_adj_out(const float *__restrict__ src, double *dst, const RepTable<MAXR> rt,
                                                 long long N, long long P) {
    const int rb = find_block_rep(rt, blockIdx.x);
    const Rep &rp = rt.rep[rb];
    const int nx = rp.nx, ny = rp.ny, nz = rp.nz;
    const unsigned node = (blockIdx.x - rt.item_off[rb]) * SEG + threadIdx.x;
    if (node >= (unsigned)nx * ny * nz) return;
    const unsigned row = divide(node, rp.dchunks);  // see node_table
    const int x = (int)(node - row * (unsigned)nx);
    const int z = (int)divide(row, rp.dny), y = (int)(row - (unsigned)z * ny);
    const int slab = nx * ny;
    const long long i = rp.node_off + node;
    // offsets of x + e (index e + 1), periodic
    const int ox[3] = {x == 0 ? nx - 1 : -1, 0, x == nx - 1 ? 1 - nx : 1};
    const int oy[3] = {y == 0 ? (ny - 1) * nx : -nx, 0, y == ny - 1 ? (1 - ny) * nx : nx};
    const int oz[3] = {z == 0 ? (nz - 1) * slab : -slab, 0, z == nz - 1 ? (1 - nz) * slab : slab};
    float v[Q];
#pragma unroll
    for (int a = 0; a < Q; ++a)
        v[a] = __ldg(src + (long long)a * P + i + ox[ex(a) + 1] + oy[ey(a) + 1] + oz[ez(a) + 1]);
#pragma unroll
    for (int a = 0; a < Q; ++a) dst[(long long)a * N + i] = widen_f32(v[a]);
}

cudaError_t launch_f32_to_f64(Sim &s, const float *src, double *dst, cudaStream_t st) {
    auto launch = [&](const auto &rt) {
        constexpr int MAXR = sizeof(rt.rep) / sizeof(Rep);
        k_adj_out<MAXR><<<rt.item_off[rt.nrep], SEG, 0, st>>>(src, dst, rt, s.N, s.P);
        return cudaGetLastError();
    };
    return s.nrep == 1 ? launch(node_table<1>(s)) : launch(node_table<MAX_BATCH>(s));
}

}  // namespace lbp
