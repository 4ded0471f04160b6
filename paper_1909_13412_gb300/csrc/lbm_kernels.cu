// lbm_kernels.cu -- D3Q15 lattice kernels of liblbp (sm_103a).
//
// Storage: 15 planes (structure of arrays, x fastest), plane stride P >= N,
// holding the deviation g_a = fhat_a - w_a of the post-collision populations
// from the rest state, as FP32, BF16 or scaled FP16 (the Store* types of
// lbp_internal.cuh); every kernel is a template on the storage type.  With sum_a w_a = 1 and sum_a w_a e_a = 0 the moments
// of Eqs. 12-13 are rho~ - 1 = sum_a g_a and u = sum_a e_a g_a, and the
// collision of Eqs. 15, 17 and 19 becomes, exactly,
//     g'_a = g_a + (geq_a - g_a)/tau,
//     geq_a = w_a [(rho~ - 1) + 3 e_a.u + 9/2 (e_a.u)^2 - 3/2 u.u],
// so FP32 arithmetic acts on the small deviations instead of on O(0.1)
// populations.
#include <cuda_runtime.h>

#include <type_traits>

#include <cstring>

#include "lbp_internal.cuh"

namespace lbp {

// ---------------------------------------------------------------------------
// Fused pull-stream + moments + BGK collision (Eqs. 20, 12, 13, 15, 17, 19).
//
// One thread per node and one block per SEG-node segment of an x-row: a full
// grid, not a persistent loop, so the hardware block scheduler keeps the
// blocks in flight on a narrow window of consecutive rows (the 15 read and 15
// write streams stay local in DRAM) and balances the tail.  The 15 loads of a
// node are independent, so every thread keeps 60 bytes in flight.  Address
// arithmetic is 32-bit offsets from per-population plane pointers passed as
// kernel parameters, and the collision (collide_values) is written per
// opposite pair (a, a+1), e_{a+1} = -e_a, with 1/tau folded into per-class
// constants: eight operations a pair.  The FP32 kernel stays bound by DRAM
// bandwidth (measured on GB300 at 256^3: within 2% of a plain copy); the
// 2-byte kernels, which move half the bytes, are bound by instruction issue.
// ---------------------------------------------------------------------------
template <typename St>
__device__ __forceinline__ void collide_store(const float g[Q], const Planes<St> &pl, int d,
                                              float omega, float F0, float F1, float F2, bool &bad) {
    float o[Q];
    collide_st<St>(g, omega, F0, F1, F2, o);
    bad |= nonfinite_node(o);
#pragma unroll
    for (int a = 0; a < Q; ++a) St::cstore(pl.d[a] + d, a, o[a]);
}

// Index arithmetic shared by both variants: node d of (x, row) and the
// offsets of the pull sources x - e, y - e, z - e (index e + 1), periodic.
struct NodeIdx {
    int d;
    int ox[3], oy[3], oz[3];
};

// The block of the sweep that this thread block serves.  Where the two
// population buffers are not much larger than L2 (sweeps_back), consecutive passes
// run through the lattice in opposite directions, so that a pass first reads what
// the one before wrote last, and read with the first lines to be evicted those
// of the other buffer, whose contents are of no more use (BACK).  Elsewhere the
// direction changes little (FP32 at 256^3 the same) and early eviction loses the
// lines that neighbouring row segments share (328 -> 362 us at 256^3).
// us per step, FP32: 20.8 -> 16.8 (100^3, one particle), 24.8 -> 21.5 (100^3, 900),
// 31.4 -> 29.0 (112^3, 1000), 45.2 -> 43.6 (128^3, 2000); at 140^3 61.7 -> 65.0.
template <bool BACK>
__device__ __forceinline__ unsigned block_of(bool flip) {
    return BACK && flip ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
}

__device__ __forceinline__ NodeIdx node_index(int x, unsigned row, int nx, int ny, int nz, Divisor dny) {
    NodeIdx n;
    const int z = (int)divide(row, dny);
    const int y = (int)(row - (unsigned)z * ny);
    const int slab = nx * ny;
    n.d = (int)row * nx + x;
    n.ox[0] = x == nx - 1 ? 1 - nx : 1;
    n.ox[1] = 0;
    n.ox[2] = x == 0 ? nx - 1 : -1;
    n.oy[0] = y == ny - 1 ? (1 - ny) * nx : nx;
    n.oy[1] = 0;
    n.oy[2] = y == 0 ? (ny - 1) * nx : -nx;
    n.oz[0] = z == nz - 1 ? (1 - nz) * slab : slab;
    n.oz[1] = 0;
    n.oz[2] = z == 0 ? (nz - 1) * slab : -slab;
    return n;
}

// Each block serves R rows (consecutive in y) of one SEG-node x-segment of one
// replica box: a thread issues the 15 R loads of its R nodes before any
// arithmetic.  R = 2 for the 2-byte storage types, whose 15 loads per node
// alone keep too few bytes in flight; R = 1 for FP32.  The block finds its box
// in the replica table (a kernel parameter; one entry for a single box).
// Two rows per block are held to 64 registers (eight blocks of 128 threads per
// SM): the batched ensemble's short rows need the occupancy (0.793 ms per
// launch there, against 0.833 ms at the compiler's 72 registers).
// BACK: see block_of.
template <int BX, typename St, int R, int MAXR, bool BACK>
__global__ void __launch_bounds__(BX, R == 2 ? 8 : 1) k_stream_collide(Planes<St> pl, const RepTable<MAXR> rt,
                                                       long long *bump, int *err, bool flip) {
    const unsigned block = block_of<BACK>(flip);
    const int r = find_block_rep(rt, block);
    const Rep &rp = rt.rep[r];
    const int nx = rp.nx, ny = rp.ny, nz = rp.nz, nchunks = rp.nchunks;
    const unsigned nrows = (unsigned)ny * (unsigned)nz;
    const unsigned item = block - rt.item_off[r];
    const unsigned grp = divide(item, rp.dchunks);
    const int chunk = (int)(item - grp * (unsigned)nchunks);
    const int x = chunk * BX + threadIdx.x;
    grid_dependency_wait();  // chained: the pass before is complete
    grid_dependents_launch();
    if (blockIdx.x == 0 && threadIdx.x == 0) *bump += 1;
    if (x >= nx) return;
    const int base = (int)rp.node_off;
    NodeIdx n[R];
    float g[R][Q];
#pragma unroll
    for (int h = 0; h < R; ++h) {
        const unsigned row = grp * R + h < nrows ? grp * R + h : nrows - 1;
        n[h] = node_index(x, row, nx, ny, nz, rp.dny);
        n[h].d += base;
#pragma unroll
        for (int a = 0; a < Q; ++a)
            g[h][a] = St::template cload<BACK>(pl.s[a] + (n[h].d + n[h].ox[ex(a) + 1] + n[h].oy[ey(a) + 1] +
                                          n[h].oz[ez(a) + 1]), a);
    }
    bool bad = false;
#pragma unroll
    for (int h = 0; h < R; ++h)
        if (grp * R + h < nrows) collide_store<St>(g[h], pl, n[h].d, rp.omega, rp.gx, rp.gy, rp.gz, bad);
    if (bad) atomicOr(err, ERR_LATTICE);
}

// Sum, exactly in 64-bit fixed point, the record entries whose x is this
// lane's x; rw is this lane's word of the 256-byte record (see lbp_internal.cuh).
__device__ __forceinline__ void record_sum(unsigned long long rw, int cnt, int x, long long &a0,
                                           long long &a1, long long &a2) {
    const int used = cnt < REC_SLOTS ? cnt : REC_SLOTS;
    for (int sl = 0; sl < used; ++sl) {
        const unsigned long long xw2 = __shfl_sync(0xffffffffu, rw, REC_X0 + (sl >> 1));
        const int xs = (int)(unsigned)(xw2 >> (32 * (sl & 1)));
        const long long v0 = (long long)__shfl_sync(0xffffffffu, rw, REC_F0 + 3 * sl);
        const long long v1 = (long long)__shfl_sync(0xffffffffu, rw, REC_F0 + 3 * sl + 1);
        const long long v2 = (long long)__shfl_sync(0xffffffffu, rw, REC_F0 + 3 * sl + 2);
        if (xs == x) {
            a0 += v0;
            a1 += v1;
            a2 += v2;
        }
    }
}

// ---------------------------------------------------------------------------
// The same pass with the body force of Eqs. 18-19 (particles present).
// Every SEG-node segment of a row owns one force record (lbp_internal.cuh)
// filled by this step's particle kernel.  Every warp loads the 256-byte
// record of each of its rows -- one 8-byte word per lane -- together with its
// population loads (the address depends only on the block index, so no load
// waits on another), then each lane sums, exactly in 64-bit fixed point, the
// entries whose x is its own and adds 3 w_a F.e_a to its post-collision
// populations.  If a record overflowed (count > REC_SLOTS) the particle kernel
// put the shares that did not fit into the dense per-node accumulator: the
// lanes of that (rare) segment also read and clear their node's accumulator
// and add it to the record sum -- still an exact integer sum of all the node's
// shares.  The block clears the counts of its rows' records of the previous
// step, which the next step's particle kernel refills.
// ---------------------------------------------------------------------------
// Where a segment's mark is compared with the epoch: ahead of the population loads,
// which then wait for it, or after them.  Which is faster depends on what the
// compiler makes of the rest: us per step early / late, 256^3 with one particle (and
// 16777), FP32 rows 1, 2, 4: 347 / 334, 296 / 297 (330 / 333), 341 / 296 (383 / 338);
// FP16 rows 2: 206 / 216; BF16 rows 1, 2, 4: 241 / 243, 226 / 208 (268 / 265), 220 / 220,
// and at 255 x 256 x 256 BF16 rows 2 240 / 223.
template <typename St, int R>
constexpr bool LATE_MARK = std::is_same<St, StoreF32>::value ? R != 2 : std::is_same<St, StoreBF16>::value && R == 2;

template <int BX, typename St, int R, int MAXR, bool BACK>
__global__ void __launch_bounds__(BX, R == 2 ? 8 : 1) k_stream_collide_forced(
    Planes<St> pl, const RepTable<MAXR> rt, const unsigned long long *rec_cur, unsigned long long *rec_prev,
    unsigned long long *fq, long long Ntot, long long *bump, int *err, const Marks mk, bool flip) {
    static_assert(BX == SEG, "one block per force-record segment");
    const unsigned block = block_of<BACK>(flip);
    const int r = find_block_rep(rt, block);
    const Rep &rp = rt.rep[r];
    const int nx = rp.nx, ny = rp.ny, nz = rp.nz, nchunks = rp.nchunks;
    const unsigned nrows = (unsigned)ny * (unsigned)nz;
    const int lane = threadIdx.x & 31;
    const unsigned item = block - rt.item_off[r];
    const unsigned grp = divide(item, rp.dchunks);
    const int chunk = (int)(item - grp * (unsigned)nchunks);
    const size_t seg0 = (size_t)rp.seg_off;
    // the previous step's records (this step's particle kernel writes the others)
    if (threadIdx.x < R && grp * R + threadIdx.x < nrows)
        rec_prev[(seg0 + (size_t)(grp * R + threadIdx.x) * nchunks + chunk) * REC_WORDS] = 0ull;
    const int xw = chunk * BX + (threadIdx.x & ~31);
    if (xw >= nx) return;  // whole warp past the end of the row
    const int x0 = xw + lane;
    const bool act = x0 < nx;
    const int x = act ? x0 : nx - 1;
    const int base = (int)rp.node_off;
    NodeIdx n[R];
    float g[R][Q];
    unsigned long long rw[R];
    unsigned mark[R];
    bool bad = false, forced[R];
#pragma unroll
    for (int h = 0; h < R; ++h) {
        const unsigned row = grp * R + h < nrows ? grp * R + h : nrows - 1;
        n[h] = node_index(x, row, nx, ny, nz, rp.dny);
        n[h].d += base;
        if (LATE_MARK<St, R>) {
            mark[h] = 0;
            if (mk.epoch != 0) mark[h] = __ldcg(mk.seg + seg0 + (size_t)row * nchunks + chunk);
        } else {
            forced[h] = mk.epoch == 0 || __ldcg(mk.seg + seg0 + (size_t)row * nchunks + chunk) == mk.epoch;
        }
#pragma unroll
        for (int a = 0; a < Q; ++a)
            g[h][a] = St::template cload<BACK>(pl.s[a] + (n[h].d + n[h].ox[ex(a) + 1] + n[h].oy[ey(a) + 1] +
                                          n[h].oz[ez(a) + 1]), a);
    }
    // the loads above do not depend on this step's particle kernel; the records do
    // (the wait is a no-op unless launched as its programmatic dependent)
    bool wait = blockIdx.x == 0;
#pragma unroll
    for (int h = 0; h < R; ++h) {
        if (LATE_MARK<St, R>) forced[h] = mark[h] == mk.epoch;  // no marks: 0 == 0
        wait = wait || forced[h];
    }
    if (wait) grid_dependency_wait();
    grid_dependents_launch();
    if (blockIdx.x == 0 && threadIdx.x == 0) *bump += 1;
#pragma unroll
    for (int h = 0; h < R; ++h) {
        const unsigned row = grp * R + h < nrows ? grp * R + h : nrows - 1;
        rw[h] = 0ull;
        if (forced[h]) rw[h] = __ldcg(rec_cur + (seg0 + (size_t)row * nchunks + chunk) * REC_WORDS + lane);
    }
#pragma unroll
    for (int h = 0; h < R; ++h) {
        const int cnt = (int)(unsigned)(__shfl_sync(0xffffffffu, rw[h], 0) & 0xffffffffull);
        float F0 = rp.gx, F1 = rp.gy, F2 = rp.gz;  // uniform body force of the box
        if (cnt > 0 && grp * R + h < nrows) {
            long long a0 = 0, a1 = 0, a2 = 0;
            record_sum(rw[h], cnt, x, a0, a1, a2);
            if (cnt > REC_SLOTS && act) {
                const int d = n[h].d;
                a0 += (long long)__ldcg(fq + d);
                a1 += (long long)__ldcg(fq + Ntot + d);
                a2 += (long long)__ldcg(fq + 2 * Ntot + d);
                fq[d] = 0ull;
                fq[Ntot + d] = 0ull;
                fq[2 * Ntot + d] = 0ull;
            }
            const float inv = 1.3877787807814457e-17f;  // 2^-56
            F0 = __fmaf_rn(inv, fix_to_float(a0), F0);
            F1 = __fmaf_rn(inv, fix_to_float(a1), F1);
            F2 = __fmaf_rn(inv, fix_to_float(a2), F2);
        }
        if (act && grp * R + h < nrows) collide_store<St>(g[h], pl, n[h].d, rp.omega, F0, F1, F2, bad);
    }
    if (bad) atomicOr(err, ERR_LATTICE);
}

// ---------------------------------------------------------------------------
// Paired-node variant for the 2-byte storage types (every box with even nx).
// A thread owns two neighbouring nodes (x, x + 1), x even, and moves each
// plane's pair of 2-byte deviations with one 4-byte load and one 4-byte store;
// a 64-thread block covers one SEG-node segment of R rows.  The pull streaming
// in x is done in registers: for e_x = +1 the pair (x - 1, x) is the high
// half of the left lane's pair and the low half of the lane's own, for
// e_x = -1 the pair (x + 1, x + 2) is the high half of its own and the low
// half of the right lane's (warp shuffles); the lanes at a warp's or a row's
// end load the neighbouring pair themselves (periodic in x).  This halves the
// load and store instructions per node and leaves the conversions packed, so
// the kernel is no longer bound by instruction issue.  Per node the
// arithmetic is that of collide_st: results equal the one-node kernels'
// bit for bit.  Its steps are not chained, so its loads could be read-only ones;
// us per step at 254 x 256 x 256 with 16384 particles, through L2 / read-only: one row
// BF16 298 / 277, FP16 276 / 278, two rows 264 / 280, 295 / 270 (without particles
// within 3 % either way): the best of each storage is not slower through L2.
// ---------------------------------------------------------------------------
template <typename St>
__device__ __forceinline__ void unpack2(unsigned v, int a, float &lo, float &hi);
template <>
__device__ __forceinline__ void unpack2<StoreBF16>(unsigned v, int, float &lo, float &hi) {
    lo = __uint_as_float(v << 16);
    hi = __uint_as_float(v & 0xffff0000u);
}
// FP16: the collision-space values h (StoreF16::cload), not scaled
template <>
__device__ __forceinline__ void unpack2<StoreF16>(unsigned v, int, float &lo, float &hi) {
    lo = __half2float(__ushort_as_half((unsigned short)(v & 0xffffu)));
    hi = __half2float(__ushort_as_half((unsigned short)(v >> 16)));
}
template <typename St>
__device__ __forceinline__ unsigned pack2(float lo, float hi, int a);
template <>
__device__ __forceinline__ unsigned pack2<StoreBF16>(float lo, float hi, int) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const unsigned *>(&p);
}
template <>
__device__ __forceinline__ unsigned pack2<StoreF16>(float lo, float hi, int) {
    const __half2 p = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const unsigned *>(&p);
}

constexpr int PAIR_BX = SEG / 2;  // threads per block of the paired kernel

// True if either 2-byte value of a packed pair is a NaN or an infinity (its
// exponent field all ones: 0x7f80 for bfloat16, 0x7c00 for binary16).
template <typename St>
__device__ __forceinline__ bool packed_nonfinite(unsigned v);
template <>
__device__ __forceinline__ bool packed_nonfinite<StoreBF16>(unsigned v) {
    return (v & 0x7f80u) == 0x7f80u || (v & 0x7f800000u) == 0x7f800000u;
}
template <>
__device__ __forceinline__ bool packed_nonfinite<StoreF16>(unsigned v) {
    return (v & 0x7c00u) == 0x7c00u || (v & 0x7c000000u) == 0x7c000000u;
}

template <typename St, int R, int MAXR, bool FORCED>
__global__ void __launch_bounds__(PAIR_BX) k_stream_collide_pair(
    Planes<St> pl, const RepTable<MAXR> rt, const unsigned long long *rec_cur,
    unsigned long long *rec_prev, unsigned long long *fq, long long Ntot, long long *bump, int *err) {
    const int r = find_block_rep(rt, blockIdx.x);
    const Rep &rp = rt.rep[r];
    const int nx = rp.nx, ny = rp.ny, nz = rp.nz, nchunks = rp.nchunks;
    const unsigned nrows = (unsigned)ny * (unsigned)nz;
    const int lane = threadIdx.x & 31;
    const unsigned item = blockIdx.x - rt.item_off[r];
    const unsigned grp = divide(item, rp.dchunks);
    const int chunk = (int)(item - grp * (unsigned)nchunks);
    const size_t seg0 = (size_t)rp.seg_off;
    if (FORCED && threadIdx.x < R && grp * R + threadIdx.x < nrows)
        rec_prev[(seg0 + (size_t)(grp * R + threadIdx.x) * nchunks + chunk) * REC_WORDS] = 0ull;
    if (!FORCED && blockIdx.x == 0 && threadIdx.x == 0) *bump += 1;
    const int xw = chunk * SEG + 2 * (threadIdx.x & ~31);  // first node of the warp
    if (xw >= nx) return;
    const int x0 = xw + 2 * lane;
    const bool act = x0 < nx;
    const int x = act ? x0 : nx - 2;       // even; inactive lanes read a valid pair
    const int xl = x == 0 ? nx - 2 : x - 2;  // left and right pairs, periodic
    const int xr = x + 2 == nx ? 0 : x + 2;
    const bool own_left = lane == 0;               // no left lane in the warp
    const bool own_right = lane == 31 || x0 + 2 >= nx;  // no (active) right lane
    const int base = (int)rp.node_off;
    float g[R][2][Q];
    unsigned long long rw[R];
    int drow[R];
#pragma unroll
    for (int h = 0; h < R; ++h) {
        const unsigned row = grp * R + h < nrows ? grp * R + h : nrows - 1;
        const NodeIdx n = node_index(0, row, nx, ny, nz, rp.dny);
        drow[h] = base + n.d;
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            const int rb = drow[h] + n.oy[ey(a) + 1] + n.oz[ez(a) + 1];  // source row start
            const unsigned *src = reinterpret_cast<const unsigned *>(pl.s[a] + rb);
            const unsigned v = __ldcg(src + (x >> 1));
            unsigned w = v;
            if (ex(a) > 0) {
                // pull from x - 1: (x - 1, x) = (hi of left pair, lo of own)
                unsigned left = __shfl_up_sync(0xffffffffu, v, 1);
                if (own_left) left = __ldcg(src + (xl >> 1));
                w = __byte_perm(left, v, 0x5432);
            } else if (ex(a) < 0) {
                // pull from x + 1: (x + 1, x + 2) = (hi of own, lo of right pair)
                unsigned right = __shfl_down_sync(0xffffffffu, v, 1);
                if (own_right) right = __ldcg(src + (xr >> 1));
                w = __byte_perm(v, right, 0x5432);
            }
            unpack2<St>(w, a, g[h][0][a], g[h][1][a]);
        }
    }
    if (FORCED) {
        // the records come from this step's particle kernel (not read-only loads: those
        // may be moved ahead of the wait)
        grid_dependency_wait();
        if (blockIdx.x == 0 && threadIdx.x == 0) *bump += 1;
#pragma unroll
        for (int h = 0; h < R; ++h) {
            const unsigned row = grp * R + h < nrows ? grp * R + h : nrows - 1;
            rw[h] = __ldcg(rec_cur + (seg0 + (size_t)row * nchunks + chunk) * REC_WORDS + lane);
        }
    }
#pragma unroll
    for (int h = 0; h < R; ++h) {
        float F[2][3] = {{rp.gx, rp.gy, rp.gz}, {rp.gx, rp.gy, rp.gz}};
        if (FORCED) {
            const int cnt = (int)(unsigned)(__shfl_sync(0xffffffffu, rw[h], 0) & 0xffffffffull);
            if (cnt > 0 && grp * R + h < nrows) {
                long long s0[3] = {0, 0, 0}, s1[3] = {0, 0, 0};
                record_sum(rw[h], cnt, x, s0[0], s0[1], s0[2]);
                record_sum(rw[h], cnt, x + 1, s1[0], s1[1], s1[2]);
                if (cnt > REC_SLOTS && act) {
                    const int d = drow[h] + x;
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        s0[k] += (long long)__ldcg(fq + k * Ntot + d);
                        s1[k] += (long long)__ldcg(fq + k * Ntot + d + 1);
                        fq[k * Ntot + d] = 0ull;
                        fq[k * Ntot + d + 1] = 0ull;
                    }
                }
                const float inv = 1.3877787807814457e-17f;  // 2^-56
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    F[0][k] = __fmaf_rn(inv, fix_to_float(s0[k]), F[0][k]);
                    F[1][k] = __fmaf_rn(inv, fix_to_float(s1[k]), F[1][k]);
                }
            }
        }
        if (act && grp * R + h < nrows) {
            float o0[Q], o1[Q];
            collide_st<St>(g[h][0], rp.omega, F[0][0], F[0][1], F[0][2], o0);
            collide_st<St>(g[h][1], rp.omega, F[1][0], F[1][1], F[1][2], o1);
            if (nonfinite_node(o0) || nonfinite_node(o1)) atomicOr(err, ERR_LATTICE);
#pragma unroll
            for (int a = 0; a < Q; ++a)
                reinterpret_cast<unsigned *>(pl.d[a] + drow[h])[x >> 1] = pack2<St>(o0[a], o1[a], a);
        }
    }
}

// Read and clear the overflow accumulators of a node pair (through L2: the particle
// kernels' atomics add to them).  16-byte aligned: the four-node kernel needs rows of
// a multiple of four in every box, so planes, rows and pairs start at even nodes.  One
// by one, a lane made twelve 8-byte loads and stores: us per step with 8 particles per
// 1000 nodes, BF16, 100^3 72 -> 38, 160^3 390 -> 224, 256^3 1128 -> 726.  (In the two-node
// kernel pairs cost registers: 254 x 256 x 256, BF16, two rows 265 -> 281; not used there.)
__device__ __forceinline__ ulonglong2 take_shares(unsigned long long *fq) {
    ulonglong2 *at = reinterpret_cast<ulonglong2 *>(fq);
    const ulonglong2 v = __ldcg(at);
    *at = make_ulonglong2(0ull, 0ull);
    return v;
}

// Sum, exactly, the record entries whose x is one of x .. x + 3 (one pass
// over the slots for four nodes; the same integer sums as record_sum).
__device__ __forceinline__ void record_sum4(unsigned long long rw, int cnt, int x, long long s[4][3]) {
    const int used = cnt < REC_SLOTS ? cnt : REC_SLOTS;
    for (int sl = 0; sl < used; ++sl) {
        const unsigned long long xw2 = __shfl_sync(0xffffffffu, rw, REC_X0 + (sl >> 1));
        const int k = (int)(unsigned)(xw2 >> (32 * (sl & 1))) - x;
        const long long v0 = (long long)__shfl_sync(0xffffffffu, rw, REC_F0 + 3 * sl);
        const long long v1 = (long long)__shfl_sync(0xffffffffu, rw, REC_F0 + 3 * sl + 1);
        const long long v2 = (long long)__shfl_sync(0xffffffffu, rw, REC_F0 + 3 * sl + 2);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
            if (k == kk) {
                s[kk][0] += v0;
                s[kk][1] += v1;
                s[kk][2] += v2;
            }
    }
}

// ---------------------------------------------------------------------------
// Four-node variant for the 2-byte storage types (every box with nx a
// multiple of 4).  One warp per SEG-node row segment (and R rows): lane l owns
// the nodes x .. x + 3, x = segment start + 4 l, and moves each plane's four
// 2-byte deviations with one 8-byte load and one 8-byte store, so a warp
// touches the segment's 256 contiguous bytes per plane.  The pull in x is done
// in registers as in the paired kernel: for e_x = +1 the node left of x is the
// top element of the left lane's group, for e_x = -1 the node right of x + 3
// is the bottom element of the right lane's group (warp shuffles); the lanes
// at a warp's or a row's end load that one element themselves (periodic in
// x).  A thread keeps 15 R 8-byte loads in flight in 30 R registers, twice the
// bytes per register of the paired kernel, and collides the pairs (x, x + 1)
// and (x + 2, x + 3) in turn, packing the results over the pulled values.
// Per node the arithmetic is that of collide_st, and the force sums are
// the same exact integer sums: results equal the other kernels' bit for bit.
// ---------------------------------------------------------------------------
// Row segments (warps) per block.  With several rows a block of four: us per step at
// 256^3 with 16777 particles, BF16, blocks of two / four: two rows 308 / 299, four rows
// 551 / 456 (the same within 1 % with one particle); one row: see below.
constexpr int quad_warps(int R) { return R == 1 ? 2 : 4; }
// With one row the kernel is bound by latency and instruction issue: it is held
// to 72 registers for 28 warps per SM.  us a step at 256^3 with 16384 particles,
// BF16 / FP16: 24 warps (80 registers) 206.5 / 222.0, 28 in blocks of four
// 202.1 / 198.7, in blocks of two 200.9 / 197.6, 32 (64 registers) 213.5 / 211.2.
// Nothing between the population loads and the record load needs a loaded value
// (the shuffles of the pull come after), so that the two latencies overlap; a
// record loaded after the shuffles measured 224.8 / 212.6, and as a read-only load
// it may move ahead of the wait and miss its particle kernel's entries.
// Through L2, chained and with marks (see Marks) it is at 200.9 / 197.6 where the
// cached, unmarked kernel was at 213.0 / 215.3.  More rows keep more loads in
// flight and need the registers.

// The pass without particles in FP16 is better at 80 registers once the buffers are
// beyond L2 (BACK: see block_of); us per step, 72 / 80: 7.4 / 8.4 (64^3), 51.5 / 53.2
// (160^3), 96.3 / 88.6 (200^3), 159.7 / 151.2 (256^3), 354 / 322 (320^3), 699 / 643 (400^3).
template <typename St, int R, bool FORCED, bool BACK>
constexpr int QUAD_BLOCKS = R > 1 ? 1 : St::SCALED && !FORCED && !BACK ? 12 : 14;

template <typename St, int R, int MAXR, bool FORCED, bool BACK>
__global__ void __launch_bounds__(32 * quad_warps(R), QUAD_BLOCKS<St, R, FORCED, BACK>) k_stream_collide_quad(
    Planes<St> pl, const RepTable<MAXR> rt, const unsigned long long *rec_cur,
    unsigned long long *rec_prev, unsigned long long *fq, long long Ntot, long long *bump, int *err, const Marks mk, bool flip) {
    if (!FORCED && blockIdx.x == 0 && threadIdx.x == 0) *bump += 1;
    const unsigned item = block_of<BACK>(flip) * quad_warps(R) + (threadIdx.x >> 5);
    if (item >= rt.item_off[MAXR == 1 ? 1 : rt.nrep]) return;  // whole warp past the last segment
    const int r = find_block_rep(rt, item);
    const Rep &rp = rt.rep[r];
    const int nx = rp.nx, ny = rp.ny, nz = rp.nz, nchunks = rp.nchunks;
    const unsigned nrows = (unsigned)ny * (unsigned)nz;
    const int lane = threadIdx.x & 31;
    const unsigned it = item - rt.item_off[r];
    // the row segment by one multiplication (Divisor)
    const unsigned grp = divide(it, rp.dchunks);
    const int chunk = (int)(it - grp * (unsigned)nchunks);
    const size_t seg0 = (size_t)rp.seg_off;
    if (FORCED && lane < R && grp * R + lane < nrows)
        rec_prev[(seg0 + (size_t)(grp * R + lane) * nchunks + chunk) * REC_WORDS] = 0ull;
    const int x0 = chunk * SEG + 4 * lane;
    const bool act = x0 < nx;
    const int x = act ? x0 : nx - 4;         // inactive lanes read a valid group
    const int xl = x == 0 ? nx - 1 : x - 1;  // periodic neighbours of the group
    const int xr = x + 4 == nx ? 0 : x + 4;
    const bool own_left = lane == 0;                    // no left lane in the warp
    const bool own_right = lane == 31 || x0 + 4 >= nx;  // no (active) right lane
    const int base = (int)rp.node_off;
    uint2 p[R][Q];
    unsigned short edge[R][Q];  // the group's neighbour node, in the lanes that have no lane for it
    unsigned long long rw[R];
    int drow[R];
    bool forced[R];
#pragma unroll
    for (int h = 0; h < R; ++h) {
        const unsigned row = grp * R + h < nrows ? grp * R + h : nrows - 1;
        const NodeIdx n = node_index(0, row, nx, ny, nz, rp.dny);
        drow[h] = base + n.d;
        forced[h] = FORCED && (mk.epoch == 0 || __ldcg(mk.seg + seg0 + (size_t)row * nchunks + chunk) == mk.epoch);
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            const typename St::T *src = pl.s[a] + (drow[h] + n.oy[ey(a) + 1] + n.oz[ez(a) + 1]);
            const uint2 *at = reinterpret_cast<const uint2 *>(src + x);
            p[h][a] = BACK ? load_last(at) : __ldcg(at);
            edge[h][a] = 0;
            if (ex(a) > 0 && own_left) edge[h][a] = load_word(src + xl);
            if (ex(a) < 0 && own_right) edge[h][a] = load_word(src + xr);
        }
    }
    if (FORCED) {
        // the records come from this step's particle kernel (not read-only loads: those
        // may be moved ahead of the wait); nothing before needs the loaded populations
        bool wait = blockIdx.x == 0;
#pragma unroll
        for (int h = 0; h < R; ++h) wait = wait || forced[h];
        if (wait) grid_dependency_wait();
        grid_dependents_launch();
        if (blockIdx.x == 0 && threadIdx.x == 0) *bump += 1;
#pragma unroll
        for (int h = 0; h < R; ++h) {
            const unsigned row = grp * R + h < nrows ? grp * R + h : nrows - 1;
            rw[h] = 0ull;
            if (forced[h]) rw[h] = __ldcg(rec_cur + (seg0 + (size_t)row * nchunks + chunk) * REC_WORDS + lane);
        }
    }
    // the pull in x, in registers
#pragma unroll
    for (int h = 0; h < R; ++h)
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            const uint2 v = p[h][a];
            if (ex(a) > 0) {
                // from x - 1: (x - 1, x, x + 1, x + 2)
                unsigned left = __shfl_up_sync(0xffffffffu, v.y, 1);
                if (own_left) left = (unsigned)edge[h][a] << 16;
                p[h][a] = make_uint2(__byte_perm(left, v.x, 0x5432), __byte_perm(v.x, v.y, 0x5432));
            } else if (ex(a) < 0) {
                // from x + 1: (x + 1, x + 2, x + 3, x + 4)
                unsigned right = __shfl_down_sync(0xffffffffu, v.x, 1);
                if (own_right) right = edge[h][a];
                p[h][a] = make_uint2(__byte_perm(v.x, v.y, 0x5432), __byte_perm(v.y, right, 0x5432));
            }
        }
#pragma unroll
    for (int h = 0; h < R; ++h) {
        const bool row_ok = grp * R + h < nrows;
        float F[4][3];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            F[k][0] = rp.gx;
            F[k][1] = rp.gy;
            F[k][2] = rp.gz;
        }
        // no force anywhere in this warp's row segment (no record entry, no body
        // force): the collision with literal zero forces, whose force terms the
        // compiler folds away -- the same operations on the same values as with
        // F = 0 passed in, so the results are the same bits
        bool unforced = rp.gx == 0.f && rp.gy == 0.f && rp.gz == 0.f;
        if (FORCED) {
            const int cnt = (int)(unsigned)(__shfl_sync(0xffffffffu, rw[h], 0) & 0xffffffffull);
            unforced = unforced && cnt == 0;
            if (cnt > 0 && row_ok) {
                long long sum[4][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
                record_sum4(rw[h], cnt, x, sum);
                if (cnt > REC_SLOTS && act) {
                    const int d = drow[h] + x;
#pragma unroll
                    for (int c = 0; c < 3; ++c)
#pragma unroll
                        for (int k = 0; k < 4; k += 2) {
                            const ulonglong2 v = take_shares(fq + c * Ntot + d + k);
                            sum[k][c] += (long long)v.x;
                            sum[k + 1][c] += (long long)v.y;
                        }
                }
                const float inv = 1.3877787807814457e-17f;  // 2^-56
#pragma unroll
                for (int k = 0; k < 4; ++k)
#pragma unroll
                    for (int c = 0; c < 3; ++c) F[k][c] = __fmaf_rn(inv, fix_to_float(sum[k][c]), F[k][c]);
            }
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            float g0[Q], g1[Q], o0[Q], o1[Q];
#pragma unroll
            for (int a = 0; a < Q; ++a) unpack2<St>(j ? p[h][a].y : p[h][a].x, a, g0[a], g1[a]);
            if (unforced) {
                collide_st<St>(g0, rp.omega, 0.f, 0.f, 0.f, o0);
                collide_st<St>(g1, rp.omega, 0.f, 0.f, 0.f, o1);
            } else {
                collide_st<St>(g0, rp.omega, F[2 * j][0], F[2 * j][1], F[2 * j][2], o0);
                collide_st<St>(g1, rp.omega, F[2 * j + 1][0], F[2 * j + 1][1], F[2 * j + 1][2], o1);
            }
#pragma unroll
            for (int a = 0; a < Q; ++a) {
                const unsigned w = pack2<St>(o0[a], o1[a], a);
                if (j) p[h][a].y = w; else p[h][a].x = w;
            }
        }
        if (act && row_ok) {
            // the packed collided rest populations of the four nodes: a NaN or an
            // infinity (also one from the rounding to 2 bytes) has an all-ones exponent
            if (packed_nonfinite<St>(p[h][0].x) || packed_nonfinite<St>(p[h][0].y)) atomicOr(err, ERR_LATTICE);
#pragma unroll
            for (int a = 0; a < Q; ++a) *reinterpret_cast<uint2 *>(pl.d[a] + drow[h] + x) = p[h][a];
        }
    }
}

constexpr int SC_BX = SEG;

cudaError_t prepare_lbm_kernels() { return cudaSuccess; }

template <typename St>
static Planes<St> planes_of(const Sim &s, const void *src, void *dst) {
    Planes<St> pl;
    const typename St::T *a0 = static_cast<const typename St::T *>(src);
    typename St::T *b0 = static_cast<typename St::T *>(dst);
    for (int a = 0; a < Q; ++a) {
        pl.s[a] = a0 + (long long)a * s.P;
        pl.d[a] = b0 + (long long)a * s.P;
    }
    return pl;
}

// Run f(StoreX{}) for the handle's storage type.
template <typename F>
static cudaError_t by_storage(const Sim &s, F &&f) {
    switch (s.precision) {
        case LBP_BF16: return f(StoreBF16{});
        case LBP_F16: return f(StoreF16{});
        default: return f(StoreF32{});
    }
}

bool quad_kernel_ok(const Sim &s);

// The lattice kernel's shape before any lbp_autotune: the autotuner's pick on
// GB300 at 256^3 and for the 68-box ensemble -- one node per thread with two
// rows of SEG nodes per block for FP32 (0.302 ms against 0.315-0.322 with one
// row at 256^3; 0.769 against 0.957 ms for the ensemble), four nodes per
// thread with one row for the 2-byte types (0.172 ms against 0.245 ms for one
// node per thread with two rows) where every box's nx is a multiple of 4, else
// one node per thread with two rows.
void default_shape(const Sim &s, int &rows, int &variant) {
    if (s.precision != LBP_F32 && quad_kernel_ok(s)) {
        variant = 3;
        rows = 1;
    } else {
        variant = 0;
        rows = 2;
    }
}

bool sweeps_back(const Sim &s) {
    return 2ll * storage_bytes(s.precision) * Q * s.P <= 2ll * s.l2_bytes;
}

// Run f(std::bool_constant<BACK>{}).
template <typename F>
static cudaError_t by_sweep(const Sim &s, F &&f) {
    return sweeps_back(s) ? f(std::true_type{}) : f(std::false_type{});
}

template <typename F>
static cudaError_t by_rows(int R, F &&f) {
    switch (R) {
        case 2: return f(std::integral_constant<int, 2>{});
        case 4: return f(std::integral_constant<int, 4>{});
        default: return f(std::integral_constant<int, 1>{});
    }
}

// Replica table for a launch whose blocks cover R rows of SEG nodes.
template <int MAXR>
static RepTable<MAXR> rep_table(const Sim &s, int R) {
    RepTable<MAXR> t;
    memset(&t, 0, sizeof(t));
    t.nrep = s.nrep;
    unsigned off = 0;
    for (int r = 0; r < s.nrep; ++r) {
        t.rep[r] = s.reps[r];
        t.item_off[r] = off;
        const unsigned rows = (unsigned)s.reps[r].ny * (unsigned)s.reps[r].nz;
        off += (rows + R - 1) / R * (unsigned)s.reps[r].nchunks;
    }
    t.item_off[s.nrep] = off;
    return t;
}

// Run f(RepTable<1 or MAX_BATCH>) for a single box or a batch.
template <typename F>
static cudaError_t by_batch(const Sim &s, int R, F &&f) {
    if (s.nrep == 1) return f(rep_table<1>(s, R));
    return f(rep_table<MAX_BATCH>(s, R));
}

bool pair_kernel_ok(const Sim &s) {
    if (s.precision == LBP_F32) return false;
    for (int r = 0; r < s.nrep; ++r)
        if (s.reps[r].nx % 2) return false;
    return true;
}

bool quad_kernel_ok(const Sim &s) {
    if (s.precision == LBP_F32) return false;
    for (int r = 0; r < s.nrep; ++r)
        if (s.reps[r].nx % 4) return false;
    return true;
}

bool staged_kernel_ok(const Sim &s) {
    const int H = 16 / storage_bytes(s.precision);
    for (int r = 0; r < s.nrep; ++r)
        if (s.reps[r].nx % H || s.reps[r].nx > STAGED_NODES) return false;
    return true;
}

// The one-node and four-node kernels load their populations through L2 and let
// the next step's particle kernel start.
bool lattice_chains(const Sim &s) { return s.variant == 0 || s.variant == 3; }

// Marks let the segments without forces collide beside the particle kernel.
// That pays once the pass has more row segments than are resident at a time: below,
// all already wait with their loads done, and the particle kernel only loses issue
// slots to them (11.1 -> 11.3 us at 32^3).  With FP32 and one row a block it only pays
// while the buffers are about the size of L2 (with / without, one particle: 26.7 / 31.8
// at 112^3, 38.3 / 43.3 at 128^3, 69.1 / 65.5 at 144^3, 334 / 305 at 256^3), and with
// four rows in the four-node kernel while most groups of rows stay unmarked, a particle
// marking four rows (256^3 BF16: 202 / 217 with one particle, 493 / 456 with 16777).
bool lattice_marks(const Sim &s) {
    if (!lattice_chains(s) || s.np == 0) return false;
    if (s.precision == LBP_F32 && s.rows == 1 && !sweeps_back(s)) return false;
    long long items = 0;  // blocks of the one-node kernel, warps of the four-node one
    for (int r = 0; r < s.nrep; ++r)
        items += ((long long)s.reps[r].ny * s.reps[r].nz + s.rows - 1) / s.rows * s.reps[r].nchunks;
    if (s.variant == 3 && s.rows == 4 && 4ll * s.np > items) return false;
    return items > (s.variant == 0 ? 8ll : 28ll) * s.num_sms;
}

// Replica table of the staged kernel: items of whole rows (Rep::pad = rows per item).
template <int MAXR>
static RepTable<MAXR> rep_table_staged(const Sim &s) {
    RepTable<MAXR> t;
    memset(&t, 0, sizeof(t));
    t.nrep = s.nrep;
    unsigned off = 0;
    for (int r = 0; r < s.nrep; ++r) {
        t.rep[r] = s.reps[r];
        const int rows = staged_rows(s.reps[r].nx, s.reps[r].ny);
        t.rep[r].pad = rows;
        t.item_off[r] = off;
        off += (unsigned)s.reps[r].nz * (unsigned)((s.reps[r].ny + rows - 1) / rows);
    }
    t.item_off[s.nrep] = off;
    return t;
}

bool variant_ok(const Sim &s, int variant) {
    return variant == 0 || (variant == 1 && pair_kernel_ok(s)) || (variant == 2 && staged_kernel_ok(s)) ||
           (variant == 3 && quad_kernel_ok(s));
}

// variant 0: one node per thread; 1: two nodes per thread (2-byte storage,
// even nx); 2: bulk-copy staged persistent kernel (lbm_staged.cu); 3: four
// nodes per thread, one warp per row segment (2-byte storage, nx % 4 == 0).
// pdl: launched right after the step's particle kernel, as its programmatic
// dependent (forced passes only).
template <bool FORCED>
static cudaError_t launch_sc(Sim &s, const void *src, void *dst, const unsigned long long *rec_cur,
                             unsigned long long *rec_prev, long long *bump, int rows, int variant,
                             cudaStream_t st, bool pdl = false, unsigned epoch = 0, bool flip = false) {
    constexpr int BX = SC_BX;
    if (!variant_ok(s, variant)) variant = 0;
    if (variant == 2) {
        return by_storage(s, [&](auto tag) {
            using St = decltype(tag);
            if (s.nrep == 1)
                return launch_staged_t<St, 1, FORCED>(planes_of<St>(s, src, dst), rep_table_staged<1>(s), rec_cur,
                                                      rec_prev, s.fq, s.N, bump, s.d_err, s.wait_cycles, s.wait_probe,
                                                      s.num_sms, st, pdl);
            return launch_staged_t<St, MAX_BATCH, FORCED>(planes_of<St>(s, src, dst), rep_table_staged<MAX_BATCH>(s),
                                                          rec_cur, rec_prev, s.fq, s.N, bump, s.d_err,
                                                          s.wait_cycles, s.wait_probe, s.num_sms, st, pdl);
        });
    }
    const bool use_pair = variant == 1, use_quad = variant == 3;
    const Marks mk{s.marks[epoch & 1], epoch};
    return by_storage(s, [&](auto tag) {
        using St = decltype(tag);
        return by_sweep(s, [&](auto sc) {
        constexpr bool BACK = decltype(sc)::value;
        return by_rows(rows, [&](auto rc) {
            constexpr int R = decltype(rc)::value;
            return by_batch(s, R, [&](const auto &rt) {
                constexpr int MAXR = sizeof(rt.rep) / sizeof(Rep);
                const unsigned grid = rt.item_off[rt.nrep];
                if constexpr (!std::is_same<St, StoreF32>::value) {
                    if (use_pair)
                        return launch_k(k_stream_collide_pair<St, R, MAXR, FORCED>, grid, PAIR_BX, 0, st, pdl,
                                        planes_of<St>(s, src, dst), rt, rec_cur, rec_prev, s.fq, s.N, bump, s.d_err);
                    if (use_quad)
                        return launch_k(k_stream_collide_quad<St, R, MAXR, FORCED, BACK && R == 1>,
                                        (grid + quad_warps(R) - 1) / quad_warps(R), 32 * quad_warps(R), 0, st, pdl,
                                        planes_of<St>(s, src, dst), rt, rec_cur, rec_prev, s.fq, s.N, bump, s.d_err, mk, flip);
                }
                if constexpr (FORCED)
                    return launch_k(k_stream_collide_forced<BX, St, R, MAXR, BACK>, grid, BX, 0, st, pdl,
                                    planes_of<St>(s, src, dst), rt, rec_cur, rec_prev, s.fq, s.N, bump, s.d_err, mk,
                                    flip);
                else
                    return launch_k(k_stream_collide<BX, St, R, MAXR, BACK>, grid, BX, 0, st, pdl,
                                    planes_of<St>(s, src, dst), rt, bump, s.d_err, flip);
            });
        });
        });
    });
}

cudaError_t launch_stream_collide_cfg(Sim &s, const void *src, void *dst, long long *bump,
                                      int rows, int variant, cudaStream_t st) {
    return launch_sc<false>(s, src, dst, nullptr, nullptr, bump, rows, variant, st);
}

cudaError_t launch_stream_collide_forced_cfg(Sim &s, const void *src, void *dst,
                                             const unsigned long long *rec_cur,
                                             unsigned long long *rec_prev, long long *bump, int rows,
                                             int variant, cudaStream_t st) {
    return launch_sc<true>(s, src, dst, rec_cur, rec_prev, bump, rows, variant, st);
}

cudaError_t launch_stream_collide(Sim &s, const void *src, void *dst, int parity, cudaStream_t st, bool chained) {
    return launch_sc<false>(s, src, dst, nullptr, nullptr, s.d_step, s.rows, s.variant, st, chained && s.variant == 0, 0,
                            parity != 0);
}

cudaError_t launch_stream_collide_forced(Sim &s, const void *src, void *dst, int parity,
                                         cudaStream_t st, bool pdl, unsigned epoch) {
    return launch_sc<true>(s, src, dst, s.rec[parity], s.rec[parity ^ 1], s.d_step, s.rows, s.variant, st, pdl, epoch,
                           parity != 0);
}

// ---------------------------------------------------------------------------
// FP64 <-> deviation storage.  f is [15][N] FP64 (the ABI layout).
//
// blockIdx.y is the population; a thread serves CONV_PER nodes CONV_T apart, so
// that its loads are in flight together and the index needs no division.
// Reading: the widening is done on the bits (widen_f32), because the FP64 pipe
// (2 lanes per clock and SM) would otherwise take two operations a value, 0.8 ms
// at 256^3 against 0.45 ms for the bytes; only the addition of w_a stays on it.
// Measured at 256^3, BF16 storage: 1.04 -> 0.51 ms.
// ---------------------------------------------------------------------------
constexpr int CONV_T = 256, CONV_PER = 4;

static dim3 conv_grid(long long N) {
    return dim3((unsigned)((N + CONV_T * CONV_PER - 1) / (CONV_T * CONV_PER)), Q);
}

template <typename St>
__global__ void __launch_bounds__(CONV_T) k_from_f64(const double *__restrict__ f, typename St::T *__restrict__ g,
                                                     long long N, long long P) {
    const int a = blockIdx.y;
    const long long i0 = blockIdx.x * (long long)(CONV_T * CONV_PER) + threadIdx.x;
    double v[CONV_PER];
#pragma unroll
    for (int k = 0; k < CONV_PER; ++k)
        if (i0 + k * CONV_T < N) v[k] = f[(long long)a * N + i0 + k * CONV_T];
#pragma unroll
    for (int k = 0; k < CONV_PER; ++k)
        if (i0 + k * CONV_T < N) St::store(g + (long long)a * P + i0 + k * CONV_T, a, (float)(v[k] - wgt(a)));
}

template <typename St>
__global__ void __launch_bounds__(CONV_T) k_to_f64(const typename St::T *__restrict__ g, double *__restrict__ f,
                                                   long long N, long long P) {
    const int a = blockIdx.y;
    const long long i0 = blockIdx.x * (long long)(CONV_T * CONV_PER) + threadIdx.x;
    float v[CONV_PER];
#pragma unroll
    for (int k = 0; k < CONV_PER; ++k)
        if (i0 + k * CONV_T < N) v[k] = St::load(g + (long long)a * P + i0 + k * CONV_T, a);
#pragma unroll
    for (int k = 0; k < CONV_PER; ++k)
        if (i0 + k * CONV_T < N) f[(long long)a * N + i0 + k * CONV_T] = wgt(a) + widen_f32(v[k]);
}

// Eq. 17 at every node: g_a = f^eq_a(rho~, u) - w_a, computed in FP64 and
// stored in the handle's storage type.  rho: [N] or null (1); u: [3][N] or null (0).
template <typename St>
__global__ void k_set_equilibrium(const double *__restrict__ rho, const double *__restrict__ u,
                                  typename St::T *__restrict__ g, long long N, long long P) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N;
         i += (long long)gridDim.x * blockDim.x) {
        const double dr = rho ? rho[i] - 1.0 : 0.0;
        const double ux = u ? u[i] : 0.0, uy = u ? u[N + i] : 0.0, uz = u ? u[2 * N + i] : 0.0;
        const double uu = ux * ux + uy * uy + uz * uz;
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            const double eu = ex(a) * ux + ey(a) * uy + ez(a) * uz;
            St::store(g + (long long)a * P + i, a, (float)(wgt(a) * (dr + 3.0 * eu + 4.5 * eu * eu - 1.5 * uu)));
        }
    }
}

static unsigned grid_for(long long work, int threads, int num_sms) {
    long long g = (work + threads - 1) / threads;
    const long long cap = (long long)num_sms * 16;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (unsigned)g;
}

cudaError_t launch_fill_rest(Sim &s, void *dst, cudaStream_t st) {
    // all three storage types encode 0 as all-zero bits
    return cudaMemsetAsync(dst, 0, (size_t)storage_bytes(s.precision) * Q * s.P, st);
}

cudaError_t launch_from_f64(Sim &s, const double *f, void *dst, cudaStream_t st) {
    return by_storage(s, [&](auto tag) {
        using St = decltype(tag);
        k_from_f64<St><<<conv_grid(s.N), CONV_T, 0, st>>>(
            f, static_cast<typename St::T *>(dst), s.N, s.P);
        return cudaGetLastError();
    });
}

cudaError_t launch_set_equilibrium(Sim &s, const double *rho, const double *u, void *dst,
                                   cudaStream_t st) {
    return by_storage(s, [&](auto tag) {
        using St = decltype(tag);
        k_set_equilibrium<St><<<grid_for(s.N, 256, s.num_sms), 256, 0, st>>>(
            rho, u, static_cast<typename St::T *>(dst), s.N, s.P);
        return cudaGetLastError();
    });
}

cudaError_t launch_to_f64(Sim &s, const void *src, double *f, cudaStream_t st) {
    return by_storage(s, [&](auto tag) {
        using St = decltype(tag);
        k_to_f64<St><<<conv_grid(s.N), CONV_T, 0, st>>>(
            static_cast<const typename St::T *>(src), f, s.N, s.P);
        return cudaGetLastError();
    });
}

// ---------------------------------------------------------------------------
// Totals of the stored populations for the conservation budget: per block, in
// FP64, the sums over its nodes of sum_a g_a (mass minus the node count) and
// sum_a e_a g_a (momentum; sum_a w_a e_a = 0), so out[4 b + k], k = 0..3.
// Streaming permutes the populations, so these are also the totals of the
// streamed f; the collision conserves the mass and adds exactly the body
// force (Eqs. 15, 18-19).  A fixed grid and a fixed reduction order: the
// result is the same on every call for the same state.
// ---------------------------------------------------------------------------
constexpr int BUDGET_THREADS = 256;

template <typename St>
__global__ void __launch_bounds__(BUDGET_THREADS) k_budget(const typename St::T *__restrict__ g, long long N,
                                                           long long P, double *out) {
    __shared__ double sh[4][BUDGET_THREADS];
    double m = 0.0, p0 = 0.0, p1 = 0.0, p2 = 0.0;
    for (long long i = blockIdx.x * (long long)BUDGET_THREADS + threadIdx.x; i < N;
         i += (long long)gridDim.x * BUDGET_THREADS) {
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            const double v = (double)St::load(g + (long long)a * P + i, a);
            m += v;
            if (ex(a)) p0 += ex(a) > 0 ? v : -v;
            if (ey(a)) p1 += ey(a) > 0 ? v : -v;
            if (ez(a)) p2 += ez(a) > 0 ? v : -v;
        }
    }
    sh[0][threadIdx.x] = m;
    sh[1][threadIdx.x] = p0;
    sh[2][threadIdx.x] = p1;
    sh[3][threadIdx.x] = p2;
    __syncthreads();
    for (int w = BUDGET_THREADS / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w)
#pragma unroll
            for (int k = 0; k < 4; ++k) sh[k][threadIdx.x] += sh[k][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x < 4) out[4 * blockIdx.x + threadIdx.x] = sh[threadIdx.x][0];
}

int budget_blocks(const Sim &s) { return 2 * s.num_sms; }

cudaError_t launch_budget(Sim &s, const void *src, double *out, cudaStream_t st) {
    return by_storage(s, [&](auto tag) {
        using St = decltype(tag);
        k_budget<St><<<budget_blocks(s), BUDGET_THREADS, 0, st>>>(static_cast<const typename St::T *>(src), s.N,
                                                                 s.P, out);
        return cudaGetLastError();
    });
}

// ---------------------------------------------------------------------------
// Moments of the streamed populations (Eqs. 12-13) and p = rho~/3, in FP64.
//
// The FP64 sums of the 15 FP32 values of a node are 41 additions and 15
// conversions on an FP64 pipe of 2 lanes per clock and SM, which is what bounds
// them (2.27 ms at 256^3, where moving the bytes takes 0.21 ms).  The values
// of a node nearly always lie within 18 binades of the largest, and then every
// partial sum of the FP64 evaluation is exact (45 bits), so the same sums are
// formed in integers: with 2^E > max |g|, each value is split into a multiple
// of 2^(E - 20) and a multiple of 2^(E - 41) by two additions of a constant
// whose mantissa then holds the part as an integer.  A node with a value
// that does not split exactly (below 2^(E - 18), with bits under 2^(E - 41)),
// with a huge, an infinite or a NaN value takes the FP64 additions, as does a
// value range near the FP32 denormals.  A block serves SEG consecutive nodes,
// whatever the rows (with one block per row segment, rows of one node took 2.11 ms
// for 4 M nodes, now 0.07).  Measured with u read: 2.28 -> 0.25 ms at 256^3 (BF16 storage),
// 5.86 -> 0.92 ms for 68 boxes of 43 M nodes (FP32).
// ---------------------------------------------------------------------------
struct Moments {
    double drho, u[3];
};

// the integer v (|v| < 2^51) times 2^e, exact
__device__ __forceinline__ double scaled_int(long long v, int e) {
    // 1.5 2^52 + v by its bits; the subtraction leaves v, exactly
    const double d = __longlong_as_double(0x4338000000000000ll + v) - 6755399441055744.0;
    const int hi = __double2hiint(d);
    return __hiloint2double(v != 0 ? hi + (e << 20) : hi, __double2loint(d));
}

__device__ __forceinline__ Moments moments_fp64(const float g[Q]) {
    Moments m = {0.0, {0.0, 0.0, 0.0}};
#pragma unroll
    for (int a = 0; a < Q; ++a) {
        const double v = (double)g[a];
        m.drho += v;
        m.u[0] += ex(a) * v;
        m.u[1] += ey(a) * v;
        m.u[2] += ez(a) * v;
    }
    return m;
}

__device__ __forceinline__ Moments moments(const float g[Q]) {
    int top = 0;  // largest |g| by its bits: a NaN compares above everything finite
#pragma unroll
    for (int a = 0; a < Q; ++a) top = max(top, __float_as_int(g[a]) & 0x7fffffff);
    const int f = max(top >> 23, 32);  // exponent field: |g| < 2^E with E = f - 126
    if (f > 250) return moments_fp64(g);
    const int c1 = ((f + 4) << 23) | 0x400000, c2 = ((f - 17) << 23) | 0x400000;
    const float C1 = __int_as_float(c1), C2 = __int_as_float(c2);  // 1.5 2^(E + 3), 1.5 2^(E - 18)
    int hr = 0, hx = 0, hy = 0, hz = 0, lr = 0, lx = 0, ly = 0, lz = 0;
    bool exact = true;
#pragma unroll
    for (int a = 0; a < Q; ++a) {
        const float t = __fadd_rn(g[a], C1);
        const float r = __fsub_rn(g[a], __fsub_rn(t, C1));
        const float s = __fadd_rn(r, C2);
        exact = exact && __fsub_rn(s, C2) == r;
        const int h = __float_as_int(t) - c1, l = __float_as_int(s) - c2;
        hr += h;
        lr += l;
        if (ex(a)) { hx += ex(a) > 0 ? h : -h; lx += ex(a) > 0 ? l : -l; }
        if (ey(a)) { hy += ey(a) > 0 ? h : -h; ly += ey(a) > 0 ? l : -l; }
        if (ez(a)) { hz += ez(a) > 0 ? h : -h; lz += ez(a) > 0 ? l : -l; }
    }
    if (!exact) return moments_fp64(g);
    const int e = f - 126 - 41;
    Moments m;
    m.drho = scaled_int(((long long)hr << 21) + lr, e);
    m.u[0] = scaled_int(((long long)hx << 21) + lx, e);
    m.u[1] = scaled_int(((long long)hy << 21) + ly, e);
    m.u[2] = scaled_int(((long long)hz << 21) + lz, e);
    return m;
}

template <typename St, int MAXR>
__global__ void __launch_bounds__(SEG) k_fields(const typename St::T *__restrict__ src, double *rho, double *u,
                                                double *p, const RepTable<MAXR> rt, long long N, long long P) {
    const int r = find_block_rep(rt, blockIdx.x);
    const Rep &rp = rt.rep[r];
    const unsigned node = (blockIdx.x - rt.item_off[r]) * SEG + threadIdx.x;
    if (node >= (unsigned)rp.nx * rp.ny * rp.nz) return;
    const unsigned row = divide(node, rp.dchunks);  // see node_table
    const int x = (int)(node - row * (unsigned)rp.nx);
    const NodeIdx n = node_index(x, row, rp.nx, rp.ny, rp.nz, rp.dny);
    const long long i = rp.node_off + n.d;
    float g[Q];
#pragma unroll
    for (int a = 0; a < Q; ++a)
        g[a] = St::load(src + (long long)a * P + i + n.ox[ex(a) + 1] + n.oy[ey(a) + 1] + n.oz[ez(a) + 1], a);
    const Moments m = moments(g);
    if (rho) rho[i] = 1.0 + m.drho;
    if (u) {
        u[i] = m.u[0];
        u[N + i] = m.u[1];
        u[2 * N + i] = m.u[2];
    }
    if (p) p[i] = (1.0 + m.drho) / 3.0;
}

cudaError_t launch_fields(Sim &s, const void *src, double *rho, double *u, double *p,
                          cudaStream_t st) {
    return by_storage(s, [&](auto tag) {
        using St = decltype(tag);
        auto launch = [&](const auto &rt) {
            constexpr int MAXR = sizeof(rt.rep) / sizeof(Rep);
            k_fields<St, MAXR><<<rt.item_off[rt.nrep], SEG, 0, st>>>(static_cast<const typename St::T *>(src), rho, u,
                                                                     p, rt, s.N, s.P);
            return cudaGetLastError();
        };
        return s.nrep == 1 ? launch(node_table<1>(s)) : launch(node_table<MAX_BATCH>(s));
    });
}

}  // namespace lbp
