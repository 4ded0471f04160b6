// particle_kernels.cu -- two-way coupling kernel of liblbp (sm_103a).
//
// k_particles, eight lanes per particle (one per corner of its cell) and four
// particles per warp, every step:
//   A. gathers u^N at the corners of the particle's cell from the stored
//      populations (a pull, i.e. the streamed f^n of Eq. 20): 14 independent
//      loads per lane;
//   B. fits the Stokeslet flow of Eq. 8, draws the Philox random force
//      (Eqs. 4-5) and advances V and r (Eqs. 1-2);
//   C. appends the shares of the reaction force -F_H (Eq. 9) at the corner
//      nodes to the force records of the row segments holding those nodes (the
//      stream-collide kernel applies them) and marks the segments of the next
//      step's corners.
//
// What bounds it: the FP64 pipe, and with many particles the gather.  A warp's
// FP64 instruction takes 64 cycles whatever its active lanes and whether or not
// it depends on the one before (measured: chains and independent FMAs alike;
// four warps of an SM proceed beside one another), a reciprocal square root
// seven of them, a division ten.  So a warp's time is 64 cycles times its FP64
// instructions, and they are kept few, and out of the way:
//   * vector operations run with one component per lane: lane p of a particle
//     holds component comp_of(p) of r, V, F, ... (lanes 0, 2, 1 store x, y, z),
//     so an update of three components is one instruction; the sum over the
//     corners leaves each component in its lanes (sum_components), and the two
//     sums of the normal equation share their additions (sum_pair);
//   * what depends on positions alone -- the cell, the corner geometry with its
//     reciprocal square root, the spreading fractions -- and the random force
//     are done before the launch dependency resolves, beside the previous
//     lattice pass (the step index comes from the previous particle kernel,
//     step_in), or with many particles (MANY), whose gather takes longer than the
//     end of that pass, while the gather is in flight; a warp of its own lets the
//     lattice pass of this step launch;
//   * comparisons and the widening of u^N are done on the bits;
//   * every warp works by itself (no shared memory, no block barrier), so that
//     with many particles the fits of some overlap the gathers of others.
// About 60 FP64 instructions for four particles remain between the end of the
// previous lattice pass and the update.  Before, after the gather one warp of a
// block did the scalar work of 8 particles (187 instructions, few particles) or
// one thread all of a particle's (530, many), with block barriers between the
// phases.  us per step, before -> after: 10.8 -> 7.8 (32^3, one particle),
// 14.4 -> 10.4 (64^3, 256), 49.6 -> 45.3 (128^3, 2000), 38.9 -> 35.2 (the same,
// BF16), 336.4 -> 327.8 (256^3, 16384), 212.4 -> 209.0 (the same, BF16).
// Four lanes per particle, with two corners each (85 instructions for eight
// particles), measured slower than eight lanes from 7000 particles (73.4 against
// 67.5 at 128^3) to 131072 (1186 against 1174 at 256^3): not kept.
//
// Exchange I/O (lbp_step_exchange with device buffers or page-locked host
// buffers, seen through their device views): the lanes read the external forces
// from the caller's [n][3] buffer and keep them, and write the new positions
// and velocities to the caller's buffers (a warp's are contiguous).  For host
// buffers the last block to finish then sets a completion flag in page-locked
// memory after a system-scope fence, and the host returns without waiting for
// the lattice pass.
//
// Precision split.  FP32: the gathered u^N (the lattice arithmetic is FP32).
// FP64: everything after the gather -- positions, velocities, the cell and
// fraction of r, the relative velocities w_p = u_p - V, e^N, the corner
// geometry, the basis a_p and the eight-point sums of the normal equation
// with its solve U_inf = (sum w.a)/(sum |a|^2), F_H, the random force and the
// Langevin update.
//
// Reaction forces are 64-bit fixed-point integers (scale 2^56).  -F_H is
// converted once and split over the eight corners by the trilinear fractions
// with integer arithmetic (the 1 - q share is the remainder), so the eight
// shares sum to -F_H exactly and the momentum the fluid receives is exactly
// what the particle lost.  Each share is appended to the record of its row
// segment (slot index from an integer atomic on the record's count).  The
// per-node force is the integer sum of the matching entries, so it is exact
// and independent of the order in which particles appended them (no
// floating-point atomics).  When a record is full the share goes to a dense
// per-node accumulator (integer atomics), which the stream-collide block of
// an overflowed segment adds to the record sum; the total is the same exact
// integer sum whichever shares found a slot.
#include <cuda_runtime.h>

#include "lbp_internal.cuh"

namespace lbp {

struct ParticleArgs {
    const void *g;   // deviation populations fhat^{n-1} (storage type of the handle)
    const int *prep; // replica (box) of each particle
    long long P;
    long long N;
    const double *r_in, *v_in;  // the state to advance, and where it goes (the same, but for a replay)
    double *r, *v;
    double *fh, *fr;            // null in a replay
    double *fext;  // written only when fext_in is given (lbp_step_exchange)
    const double *inv_mass, *gamma, *radius, *sig;
    const unsigned char *pinned;
    int cap, np;
    const long long *d_step;  // step index, bumped by the lattice pass
    // the step index as left by the previous particle kernel of the same call, if
    // chained, and for the next one: two slots by parity, because blocks of this
    // grid may start after others have finished
    const long long *step_in;
    long long *step_out;
    bool chained;
    unsigned long long seed;
    double sqrt3;
    int mode, exclude_inside;
    unsigned long long *rec; // force records of this step's parity
    unsigned long long *fq;  // [3][N] fixed-point overflow accumulator
    unsigned *marks;         // next step's marks (Marks), or null
    unsigned mark_epoch;
    float *ring;        // per-particle VACF ring (FP32), or null
    __half *ring16;     // ensemble VACF/MSD ring (fp16 hi/lo planes), or null
    int ring_ld, ring_dup;
    int ring_cap;
    long long *d_vacf;  // [0] first sampled step, [2] samples written
    int *err;
    double *inj;        // [3] momentum put in by F_R + F_ext (null: not tracked)
    // lbp_step_exchange with page-locked host buffers ([n][3] FP64, device views
    // of host memory; null: none): the external forces to use (and keep), and
    // the positions and velocities after the update; done_flag (host memory) is
    // set to the step index once every block has written them
    const double *fext_in;
    double *r_out, *v_out;
    unsigned *done_ticket;
    long long *done_flag;
};

// e^N = m/|m| of the mean relative velocity m (times 8), given by its component
// in each lane; false if m = 0
__device__ __forceinline__ bool direction(double mk, double (&e)[3]) {
    double m0 = from_comp(mk, 0), m1 = from_comp(mk, 1), m2 = from_comp(mk, 2);
    const long long any = __double_as_longlong(m0) | __double_as_longlong(m1) | __double_as_longlong(m2);
    double mm = __fma_rn(m2, m2, __fma_rn(m1, m1, __dmul_rn(m0, m0)));
    if (__double_as_longlong(mm) <= __double_as_longlong(1e-280)) {
        // tiny mean: rescale before the norm so that it does not underflow
        const double sc = 1.0 / fmax(fabs(m0), fmax(fabs(m1), fabs(m2)));
        m0 = __dmul_rn(m0, sc);
        m1 = __dmul_rn(m1, sc);
        m2 = __dmul_rn(m2, sc);
        mk = __dmul_rn(mk, sc);
        mm = __fma_rn(m2, m2, __fma_rn(m1, m1, __dmul_rn(m0, m0)));
    }
    const double ek = __dmul_rn(mk, rsqrt(mm));
#pragma unroll
    for (int k = 0; k < 3; ++k) e[k] = from_comp(ek, k);
    return (any & 0x7fffffffffffffffll) != 0;
}

constexpr int PN = 16;             // particles per block (32: 334.5 against 332.6 us a step at 256^3)
constexpr int PL_T = 8 * PN + 32;  // eight threads each, and the triggering warp

// the particle warps of a block (the triggering warp has left)
__device__ __forceinline__ void sync_particles() { asm volatile("bar.sync 1, %0;" ::"n"(8 * PN) : "memory"); }

// No spills at 96 registers, 20 warps per SM (at 64, 30 warps: 340.6 against
// 332.8 us a step at 256^3 with 16384 particles).
template <typename St, int MAXR, bool MANY>
__global__ void __launch_bounds__(PL_T, 4) k_particles(const ParticleArgs A, const RepTable<MAXR> rt) {
    if (threadIdx.x >= 8 * PN) {
        // lets the lattice pass of this step launch as soon as the one before it is
        // complete, whatever the others are still preparing; it waits for this
        // grid's completion before it reads anything this kernel writes
        grid_dependency_wait();
        grid_dependents_launch();
        return;
    }
    const typename St::T *G = static_cast<const typename St::T *>(A.g);
    const int p = threadIdx.x & 7, kc = comp_of(p);
    const int ip = blockIdx.x * PN + (threadIdx.x >> 3);
    const bool live = ip < A.np, owner = live && p < 3;  // the others shadow and store nothing
    const int i = live ? ip : A.np - 1, cap = A.cap;
    const int ik = kc * cap + i;

    // ---- state of the particle, written before the previous lattice pass
    const double rk = __ldcg(A.r_in + ik), Vk = __ldcg(A.v_in + ik);
    double fek;
    if (A.fext_in) {
        fek = A.fext_in[3 * (size_t)i + kc];
        if (owner) A.fext[ik] = fek;  // kept for the steps that follow
    } else {
        fek = __ldcg(A.fext + ik);
    }
    const double gam = A.gamma[i], Rd = A.radius[i], invM = A.inv_mass[i], sg = A.sig[i];
    const bool pin = A.pinned[i] != 0;
    const Rep &rp = rt.rep[MAXR == 1 ? 0 : A.prep[i]];
    const int nx = rp.nx, ny = rp.ny, nz = rp.nz;
    const int Lk = kc == 0 ? nx : kc == 1 ? ny : nz;

    // cell: base = floor(r), q = r - base (exact); this lane's corner
    const double bk = floor(rk), qk = rk - bk;
    const int base = (int)bk;
    const int c0 = p & 1, c1 = (p >> 1) & 1, c2 = p >> 2;
    const int X = wrapi(from_comp(base, 0) + c0, nx), Y = wrapi(from_comp(base, 1) + c1, ny),
              Z = wrapi(from_comp(base, 2) + c2, nz);
    // q as 31-bit fraction floor(q 2^31), for the spreading
    const unsigned frac = __double2uint_rz(qk * 2147483648.0);
    // the corner's fit geometry: with d = x_p - r_i (the corner minus the cell
    // fraction, exact) and r = |d|, the coefficients 1 - 3R/(4 r) and 1/r^3 of
    // Eq. 8; or the trilinear weight for Eq. 7.  A corner with r < 1e-12 (or r < R
    // with exclude_inside) is left out of the fit.
    double d0 = 0.0, d1 = 0.0, d2 = 0.0, k1 = 0.0, ir3 = 0.0, Wp = 0.0;
    bool use = false;
    auto geometry = [&] {
        if (A.mode == LBP_BROWNIAN) return;
        const double q0 = from_comp(qk, 0), q1 = from_comp(qk, 1), q2 = from_comp(qk, 2);
        if (A.mode == LBP_STOKESLET) {
            d0 = c0 ? __dsub_rn(1.0, q0) : -q0;
            d1 = c1 ? __dsub_rn(1.0, q1) : -q1;
            d2 = c2 ? __dsub_rn(1.0, q2) : -q2;
            const double rr = __fma_rn(d2, d2, __fma_rn(d1, d1, __dmul_rn(d0, d0)));
            use = !(rr < 1e-24 || (A.exclude_inside && rr < Rd * Rd));
            if (use) {
                const double ir = rsqrt(rr);
                k1 = __fma_rn(-(0.75 * Rd), ir, 1.0);
                ir3 = __dmul_rn(__dmul_rn(ir, ir), ir);
            }
        } else {
            Wp = (c0 ? q0 : 1.0 - q0) * (c1 ? q1 : 1.0 - q1) * (c2 ? q2 : 1.0 - q2);
        }
    };
    // Eqs. 4-5: F_R = sqrt(2 gamma kT) xi, xi = sqrt3 (2u - 1) with
    // u = ((x >> 11) + 1/2) 2^-53 from Philox(counter = (step, i, 0, 0), key = (seed, 0)).
    // 2u - 1 is formed as fma((double)(2k + 1), 2^-53, -1): the same correctly
    // rounded value as 2 ((double)k + 1/2) 2^-53 - 1, so F_R is bit-identical
    // to the oracle's.
    auto random_force = [&](long long step) {
        unsigned long long ctr[4] = {(unsigned long long)step, (unsigned long long)i, 0ull, 0ull};
        philox4x64_10(ctr, A.seed, 0ull);
        const unsigned long long x = kc == 0 ? ctr[0] : kc == 1 ? ctr[1] : ctr[2];
        const double tt = __fma_rn(__ull2double_rn(2ull * (x >> 11) + 1ull), 0x1.0p-53, -1.0);
        return __dmul_rn(sg, __dmul_rn(A.sqrt3, tt));
    };
    long long step = 0;
    double Rk = 0.0;
    if (A.chained) step = __ldcg(A.step_in);
    if (!MANY) {
        geometry();
        if (A.chained) Rk = random_force(step);
    }

    // ---- the previous lattice pass is complete: populations, step index, records
    grid_dependency_wait();
    float sx = 0.f, sy = 0.f, sz = 0.f;
    {
        // u at corner p, u = sum_a e_a g_a(x_p - e_a) (FP32)
        const int xs[3] = {wrapi(X + 1, nx), X, wrapi(X - 1, nx)};  // x - e for e = -1, 0, 1
        const int ys[3] = {wrapi(Y + 1, ny), Y, wrapi(Y - 1, ny)};
        const int zs[3] = {wrapi(Z + 1, nz), Z, wrapi(Z - 1, nz)};
        float g[Q];
#pragma unroll
        for (int a = 1; a < Q; ++a)
            g[a] = St::gather(G + ((long long)a * A.P + rp.node_off +
                                   ((long long)zs[ez(a) + 1] * ny + ys[ey(a) + 1]) * nx + xs[ex(a) + 1]), a);
        if (!A.chained) step = __ldcg(A.d_step);
        if (MANY) geometry();
        if (MANY || !A.chained) Rk = random_force(step);
#pragma unroll
        for (int a = 1; a < Q; ++a) {
            if (ex(a)) sx += ex(a) > 0 ? g[a] : -g[a];
            if (ey(a)) sy += ey(a) > 0 ? g[a] : -g[a];
            if (ez(a)) sz += ez(a) > 0 ? g[a] : -g[a];
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *A.step_out = step + 1;
        if (A.ring || A.ring16) {
            const long long m = step - A.d_vacf[0];
            if (m >= 0) A.d_vacf[2] = m + 1;
        }
    }

    // ---- friction force: component kc in every lane
    const double u0 = widen_f32(sx), u1 = widen_f32(sy), u2 = widen_f32(sz);
    double Fk = 0.0;
    if (A.mode == LBP_STOKESLET) {
        // Eq. 8: w_p = u_p - V, e^N = mean(w)/|mean(w)|, basis
        // a_p = (1 - 3R/(4 r_p)) e^N - 3R (e^N.d_p)/(4 r_p^3) d_p, and the normal
        // equation U_inf sum|a_p|^2 = sum w_p.a_p, solved for U_inf;
        // F_H = gamma U_inf e^N (Eq. 7 with u_inf = U_inf e^N + V)
        double e[3];
        const bool eok = direction(__fma_rn(-8.0, Vk, sum_components(u0, u1, u2, p)), e);
        const double w0 = __dsub_rn(u0, from_comp(Vk, 0)), w1 = __dsub_rn(u1, from_comp(Vk, 1)),
                     w2 = __dsub_rn(u2, from_comp(Vk, 2));
        double tn = 0.0, td = 0.0;
        if (eok && use) {
            const double x = __fma_rn(e[2], d2, __fma_rn(e[1], d1, __dmul_rn(e[0], d0)));
            const double k2 = __dmul_rn(__dmul_rn(0.75 * Rd, x), ir3);
            const double a0 = __fma_rn(k1, e[0], -__dmul_rn(k2, d0));
            const double a1 = __fma_rn(k1, e[1], -__dmul_rn(k2, d1));
            const double a2 = __fma_rn(k1, e[2], -__dmul_rn(k2, d2));
            tn = __fma_rn(w2, a2, __fma_rn(w1, a1, __dmul_rn(w0, a0)));
            td = __fma_rn(a2, a2, __fma_rn(a1, a1, __dmul_rn(a0, a0)));
        }
        const double nd = sum_pair(tn, td, p);
        const double num = __shfl_sync(0xffffffffu, nd, 0, 8), den = __shfl_sync(0xffffffffu, nd, 1, 8);
        if (eok) {
            const long long db = __double_as_longlong(den);
            const double U = db > 0 && db <= 0x7ff0000000000000ll ? num / den : 0.0;  // den > 0
            Fk = __dmul_rn(__dmul_rn(gam, U), kc == 0 ? e[0] : kc == 1 ? e[1] : e[2]);
        }
    } else if (A.mode == LBP_POINTWISE) {
        // Eq. 7 with u(r_i) = sum_p W_p u^N_p, corner after corner
        double ur = 0.0;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const double v0 = __shfl_sync(0xffffffffu, u0, c, 8), v1 = __shfl_sync(0xffffffffu, u1, c, 8),
                         v2 = __shfl_sync(0xffffffffu, u2, c, 8);
            ur = __fma_rn(__shfl_sync(0xffffffffu, Wp, c, 8), kc == 0 ? v0 : kc == 1 ? v1 : v2, ur);
        }
        Fk = __dmul_rn(-gam, __dsub_rn(Vk, ur));
    } else {
        // Eq. 6: friction against a fluid at rest; nothing is returned to the fluid
        Fk = __dmul_rn(-gam, Vk);
    }

    // ---- share of corner p of the fixed-point reaction force -F_H.
    // Per axis the far corner (c = 1) takes floor(v q) -- the signed high half
    // of (2 v) (q31 2^32) -- and the near corner the rest, so the eight shares
    // add up to v exactly.  |v| < 2^61 (|F_H| < 32), so 2 v stays within int64.
    if (A.mode != LBP_BROWNIAN) {
        const bool ok = below(Fk, FIX_LIMIT);
        const unsigned oks = __ballot_sync(0xffffffffu, ok) >> (threadIdx.x & 24) & 0xffu;
        const long long fix = ok ? __double2ll_rn(-Fk * FIX_SCALE) : 0ll;
        long long q31[3];
        unsigned long long sh[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) q31[k] = (long long)((unsigned long long)from_comp(frac, k) << 32);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            long long v = from_comp(fix, k), far = __mul64hi(2 * v, q31[0]);
            v = c0 ? far : v - far;
            far = __mul64hi(2 * v, q31[1]);
            v = c1 ? far : v - far;
            far = __mul64hi(2 * v, q31[2]);
            sh[k] = (unsigned long long)(c2 ? far : v - far);
        }
        if (oks != 0xffu) {
            if (live && p == 0) atomicOr(A.err, ERR_RANGE);
        } else if (live) {
            const long long row = (long long)Z * ny + Y;
            unsigned long long *rec = A.rec + (size_t)(rp.seg_off + row * rp.nchunks + X / SEG) * REC_WORDS;
            const unsigned int slot = atomicAdd(reinterpret_cast<unsigned int *>(rec), 1u);
            if (slot < (unsigned)REC_SLOTS) {
                reinterpret_cast<int *>(rec + REC_X0)[slot] = X;
#pragma unroll
                for (int k = 0; k < 3; ++k) rec[REC_F0 + 3 * slot + k] = sh[k];
            } else {
                const long long node = rp.node_off + row * nx + X;
#pragma unroll
                for (int k = 0; k < 3; ++k) atomicAdd(A.fq + k * A.N + node, sh[k]);
            }
        }
    }

    // ---- Eqs. 1-2, dt = 1: V += (F_H + F_R + F_ext)/M; r += V; periodic wrap
    double Vn = Vk, rn = rk;
    if (!pin) {
        Vn = __fma_rn(__dadd_rn(__dadd_rn(Fk, Rk), fek), invM, Vk);
        rn = __dadd_rn(rk, Vn);
        const double L = (double)Lk;
        const long long Lb = __double_as_longlong(L);
        if (negative(rn)) rn = __dadd_rn(rn, L);
        if (__double_as_longlong(rn) >= Lb) rn = __dsub_rn(rn, L);
        if (!below(Vn, __longlong_as_double(0x7ff0000000000000ll)) || negative(rn) ||
            __double_as_longlong(rn) >= Lb) {
            rn = 0.0;  // keep the next gather inside the box; reported as LBP_ENAN
            if (live) atomicOr(A.err, ERR_NAN);
        }
    }
    if (owner) {
        if (A.fh) {
            A.fh[ik] = Fk;
            A.fr[ik] = Rk;
        }
        A.v[ik] = Vn;
        A.r[ik] = rn;
        if (A.r_out) A.r_out[3 * (size_t)i + kc] = rn;
        if (A.v_out) A.v_out[3 * (size_t)i + kc] = Vn;
        if (A.done_flag) __threadfence_system();  // the host copies before the block's ticket
    }
    if (A.marks) {
        // mark the row segment of corner p of the next step's cell
        const int b = __double2int_rd(rn);
        const int x1 = wrapi(from_comp(b, 0) + c0, nx), y1 = wrapi(from_comp(b, 1) + c1, ny),
                  z1 = wrapi(from_comp(b, 2) + c2, nz);
        if (live) A.marks[rp.seg_off + ((long long)z1 * ny + y1) * rp.nchunks + x1 / SEG] = A.mark_epoch;
    }
    if (owner && (A.ring || A.ring16)) {
        const long long m = step - A.d_vacf[0];
        const long long j = (long long)kc * A.np + i;
        if (m >= 0 && A.ring) A.ring[(m % A.ring_cap) * 3 * (long long)A.np + j] = (float)Vn;
        if (m >= 0 && A.ring16) {
            // the sample as fp16 hi/lo of 4096 V (the tensor-core correlator's
            // operands), at its ring row and, for the first rows, once more
            // after the end of the ring
            const int row = (int)(m % A.ring_cap);
            const double a = Vn * (double)VACF_RING_SCALE;
            const __half hi = __double2half(a);
            const __half lo = __double2half(a - (double)__half2float(hi));
            __half *w = A.ring16 + (long long)row * 2 * A.ring_ld + j;
            w[0] = hi;
            w[A.ring_ld] = lo;
            if (row < A.ring_dup) {
                w += (long long)A.ring_cap * 2 * A.ring_ld;
                w[0] = hi;
                w[A.ring_ld] = lo;
            }
            if (!below(a, 65504.0)) atomicOr(A.err, ERR_RANGE);
        }
    }

    if (A.inj) {
        // conservation budget: the momentum F_R + F_ext put into the block's
        // unpinned particles, one FP64 atomic per component
        __shared__ double s_inj[3][PN];
        if (p < 3) s_inj[kc][threadIdx.x >> 3] = live && !pin ? Rk + fek : 0.0;
        sync_particles();
        if (threadIdx.x < 3) {
            double v = 0.0;
            for (int j = 0; j < PN; ++j) v += s_inj[threadIdx.x][j];
            atomicAdd(A.inj + threadIdx.x, v);
        }
    }

    // the last block to finish tells the host that every position and velocity
    // is in its buffers (the lattice pass may still run)
    if (A.done_flag) {
        sync_particles();
        if (threadIdx.x == 0) {
            const unsigned ticket = atomicAdd(A.done_ticket, 1u);
            if (ticket == gridDim.x - 1) {
                *A.done_ticket = 0u;
                __threadfence_system();
                *reinterpret_cast<volatile long long *>(A.done_flag) = step;
            }
        }
    }
}

// Few particles: the preparation before the launch dependency resolves (us a
// step: 10.4 against 11.4 with 256 particles at 64^3, 67.9 against 68.6 with 7000
// at 128^3).  From 48 per SM on: while the gather is in flight (98.1 against 97.4
// with 8000 at 160^3, 331.8 against 327.8 with 16384 at 256^3).
bool particles_few(const Sim &s) { return s.np < 48 * (s.num_sms > 0 ? s.num_sms : 1); }

template <bool MANY, int MAXR>
static cudaError_t launch_particles_m(const Sim &s, const ParticleArgs &A, const RepTable<MAXR> &t, cudaStream_t st) {
    const unsigned grid = (unsigned)((s.np + PN - 1) / PN);
    switch (s.precision) {
        case LBP_BF16: return launch_k(k_particles<StoreBF16, MAXR, MANY>, grid, PL_T, 0, st, A.chained, A, t);
        case LBP_F16: return launch_k(k_particles<StoreF16, MAXR, MANY>, grid, PL_T, 0, st, A.chained, A, t);
        default: return launch_k(k_particles<StoreF32, MAXR, MANY>, grid, PL_T, 0, st, A.chained, A, t);
    }
}

template <int MAXR>
static cudaError_t launch_particles_t(const Sim &s, const ParticleArgs &A, const RepTable<MAXR> &t, cudaStream_t st) {
    return particles_few(s) ? launch_particles_m<false>(s, A, t, st) : launch_particles_m<true>(s, A, t, st);
}

cudaError_t launch_particles(Sim &s, const void *src, int parity, cudaStream_t st, const ParticleIO *io,
                             bool chained, unsigned mark_epoch) {
    if (s.np == 0) return cudaSuccess;
    ParticleArgs A;
    A.g = src;
    A.prep = s.prep;
    A.P = s.P;
    A.N = s.N;
    const bool replay = io && io->state_out;
    A.r_in = replay ? io->state_in : s.r;
    A.v_in = replay ? io->state_in + 3 * (size_t)s.cap : s.v;
    A.r = replay ? io->state_out : s.r;
    A.v = replay ? io->state_out + 3 * (size_t)s.cap : s.v;
    A.fh = replay ? nullptr : s.fh;
    A.fr = replay ? nullptr : s.fr;
    A.fext = s.fext;
    A.inv_mass = s.inv_mass;
    A.gamma = s.gamma;
    A.radius = s.radius;
    A.sig = s.sig;
    A.pinned = s.pinned;
    A.cap = s.cap;
    A.np = s.np;
    A.d_step = s.d_step;
    A.step_in = s.d_step + 1 + parity;
    A.step_out = s.d_step + 1 + (parity ^ 1);
    A.chained = chained;
    A.seed = s.seed;
    A.sqrt3 = s.sqrt3;
    A.mode = s.mode;
    A.exclude_inside = s.exclude_inside;
    A.fq = s.fq;
    A.rec = s.rec[parity];
    // Eq. 6 spreads nothing: no segment of the next step waits
    A.marks = mark_epoch && s.mode != LBP_BROWNIAN ? s.marks[mark_epoch & 1] : nullptr;
    A.mark_epoch = mark_epoch;
    A.ring = s.vacf_lag >= 0 && s.vacf_pp ? s.ring : nullptr;
    A.ring16 = s.vacf_lag >= 0 && !s.vacf_pp ? static_cast<__half *>(s.ring16) : nullptr;
    A.ring_ld = s.ring_ld;
    A.ring_dup = vacf_ring_dup_rows();
    A.ring_cap = s.vacf_cap;
    A.d_vacf = s.d_vacf;
    A.err = s.d_err;
    A.inj = replay ? nullptr : s.inj;  // the recording has counted these steps
    A.fext_in = io ? io->fext_in : nullptr;
    A.r_out = io ? io->r_out : nullptr;
    A.v_out = io ? io->v_out : nullptr;
    A.done_ticket = io && io->signal ? s.d_xticket : nullptr;
    A.done_flag = io && io->signal ? s.h_xflag_dev : nullptr;
    if (s.nrep == 1) {
        RepTable<1> t;
        t.nrep = 1;
        t.item_off[0] = 0;
        t.item_off[1] = 0;
        t.rep[0] = s.reps[0];
        return launch_particles_t(s, A, t, st);
    } else {
        RepTable<MAX_BATCH> t;  // kernel parameter
        t.nrep = s.nrep;
        for (int r = 0; r <= s.nrep; ++r) t.item_off[r] = 0;
        for (int r = 0; r < s.nrep; ++r) t.rep[r] = s.reps[r];
        return launch_particles_t(s, A, t, st);
    }
}

// ---------------------------------------------------------------------------
// Layout helpers: ABI arrays are [n][3]; device state is [3][ld].
// ---------------------------------------------------------------------------
__global__ void k_aos_to_soa(const double *aos, double *soa, int n, int ld, int offset) {
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < 3 * n; t += gridDim.x * blockDim.x) {
        const int i = t / 3, k = t - 3 * i;
        soa[(long long)k * ld + offset + i] = aos[t];
    }
}

__global__ void k_soa_to_aos(const double *soa, double *aos, int n, int ld) {
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < 3 * n; t += gridDim.x * blockDim.x) {
        const int i = t / 3, k = t - 3 * i;
        aos[t] = soa[(long long)k * ld + i];
    }
}

cudaError_t launch_aos_to_soa(const double *aos, double *soa, int n, int ld, int offset,
                              cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_aos_to_soa<<<(3 * n + 255) / 256, 256, 0, st>>>(aos, soa, n, ld, offset);
    return cudaGetLastError();
}

cudaError_t launch_soa_to_aos(const double *soa, double *aos, int n, int ld, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_soa_to_aos<<<(3 * n + 255) / 256, 256, 0, st>>>(soa, aos, n, ld);
    return cudaGetLastError();
}

// Cell base index and cell fraction of the current positions, with the same
// expressions k_particles uses (for bit-exact checks of the indexing).
__global__ void k_cells(const double *r, int cap, int np, int *base, double *frac) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= np) return;
    for (int k = 0; k < 3; ++k) {
        const double rk = r[(long long)k * cap + i];
        const double b = floor(rk);
        base[3 * i + k] = (int)b;
        frac[3 * i + k] = rk - b;
    }
}

cudaError_t launch_cells(Sim &s, int *base, double *frac, cudaStream_t st) {
    if (s.np == 0) return cudaSuccess;
    k_cells<<<(s.np + 127) / 128, 128, 0, st>>>(s.r, s.cap, s.np, base, frac);
    return cudaGetLastError();
}

__global__ void k_philox(const unsigned long long *ctr, const unsigned long long *key,
                         unsigned long long *out, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        unsigned long long c[4] = {ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]};
        philox4x64_10(c, key[0], key[1]);
        for (int k = 0; k < 4; ++k) out[4 * i + k] = c[k];
    }
}

cudaError_t launch_philox(const unsigned long long *ctr, const unsigned long long *key,
                          unsigned long long *out, int64_t n, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    long long grid = (n + 255) / 256;
    if (grid > 4096) grid = 4096;
    k_philox<<<(unsigned)grid, 256, 0, st>>>(ctr, key, out, n);
    return cudaGetLastError();
}

}  // namespace lbp
