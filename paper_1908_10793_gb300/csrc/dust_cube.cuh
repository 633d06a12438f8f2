// Step and gas-predictor kernels of three-dimensional grids (mixed precision).
// One block per tile of zones (or per part of a tile, see tile_parts): the
// tile's gas box staged in shared memory, the deposit accumulated in a shared
// box.  A warp takes an equal range of the block's zones, whose grains are
// contiguous in the sorted store, and walks them 32 at a time:
//
// - Push: one grain per lane, whatever zone it lies in, relative to its key
//   zone in single precision (see dust_slab.cuh for the arithmetic).  Each
//   lane leaves a record (four impulse channels, the nine products of its x
//   and y weights, its z weights) in the warp's shared buffer.
// - Deposit: one stencil node per lane.  The 27 lanes walk the records in
//   store order (key, then id), each summing its node's weight times the
//   impulse into four registers; at the end of a zone's chunk (its grains by
//   rank, kSlabCap at a time) the sums are rounded once and added to the
//   shared box, and the host node receives the rest of the chunk's rounded
//   total.  The order of the sums, hence the integers, is fixed by the sort
//   and depends on neither the tile nor its parts.
//
// Bound: instruction issue (69% of the slots inside the loop on the 128^3 box,
// 16 warps per SM) beside 10 us of staging and flush per tile.  Why one node
// per lane: a lane's sums are four registers (three lanes per zone with nine
// nodes each held 36), all lanes are in the same zone at the same time, so
// uneven zones cost nothing, and the push runs on 32 lanes whatever the zones
// hold.  Step kernel, before (three owner lanes per zone) and with this one:
// 128^3 box 1434 -> 1183 us, 50M-grain cylindrical disk (two grains per zone)
// 6943 -> 5940 us, 33M-grain spherical disk 6214 -> 4597 us, 50x37x29 box 120 ->
// 70 us, one zone in two hundred grains deep (200k grains) 2761 -> 240 us.
// Three blocks per SM (80 registers) spill: 1635 us; 320 or 384 threads: 1430
// and 1580 us.
#pragma once

#include "dust_cube_math.cuh"

namespace dust {

// Records: 16 words (impulse 0-3, x-y products 4 + a + 3 b, z weights 13 + c)
// and the constants -1 and 1 at words 16 and 17, at a stride of 20 words: the 16-byte stores of
// eight neighbouring lanes then fall on different banks.
constexpr int kCubeThreads = 256;
constexpr int kCubeRec = 20;
constexpr int kCubeOne = 16;

// Chunk sums below this (and the host's share) take the 32-bit rounding; the
// host's rest, which differs from its share by rounding only, then needs that
// rounding to stay below 1.47e8.
constexpr float kCubeNarrow = 2e9f;

// With at most kSlabCap = 128 grains a lane's sum is rounded by at most
// 128 x 2^-24 of the sum of |weight x impulse|, 27 lanes and the total by twice
// that of the sum of |impulse| times the |weights|' sum, and the weights' sum
// differs from 1 by a few 2^-24: 1.7e-5 x 128 x 2^35 = 7.5e7 for grains with
// an impulse below 2^34 whose weights' sizes add up to less than 2 (they are
// positive but near the axis and the poles).  Larger ones belong to chunks whose
// sums are nearly always too large for 32 bits.  A NaN is not calm.
template <int GEOM>
__device__ __forceinline__ bool cube_calm(const float D[4], const float w[3][3])
{
    constexpr float top = 17179869184.f;
    bool ok = (fabsf(D[0]) < top) & (fabsf(D[1]) < top) & (fabsf(D[2]) < top) & (fabsf(D[3]) < top);
    if (GEOM == GEOM_CYL || GEOM == GEOM_SPH) {
        float s = fabsf(w[0][0]) + fabsf(w[0][1]) + fabsf(w[0][2]);
        if (GEOM == GEOM_SPH) s *= fabsf(w[1][0]) + fabsf(w[1][1]) + fabsf(w[1][2]);
        ok = ok & (s < 2.f);
    }
    return ok;
}

// Zone constants of one direction: centre (double and single), inverse width.
struct __align__(16) CubeZone {
    double c;
    float cf, iw;
};

// Byte offsets inside the block's shared memory.
struct CubeLayout {
    size_t dep, rec, off, zone, lim, nu, lo, hw, vl, vh, bar, total;
};

__host__ __device__ inline CubeLayout cube_layout(int bvol, int tvol, int T0, int T1, int T2)
{
    CubeLayout L;
    const size_t tsum = (size_t)T0 + T1 + T2;
    size_t o = (size_t)bvol * 4 * sizeof(float);   // gas box first: 128-byte aligned for the bulk copy
    L.dep = o;  o += (size_t)bvol * 4 * sizeof(long long);
    L.rec = o;  o += (size_t)(kCubeThreads / 32) * 32 * kCubeRec * sizeof(float);
    L.zone = o; o += tsum * sizeof(CubeZone);
    L.bar = o;  o += 16;
    L.lim = o;  o += tsum * sizeof(float2);
    L.off = o;  o += (size_t)(tvol + 1) * sizeof(int);
    L.nu = o;   o += (size_t)T0 * sizeof(float);
    L.lo = o;   o += (size_t)(T1 + 1) * sizeof(float);
    L.hw = o;   o += (size_t)T1 * sizeof(float);
    L.vl = o;   o += (size_t)(T0 + T1) * sizeof(float);
    L.vh = o;   o += (size_t)(T0 + T1) * sizeof(float);
    L.total = (o + 15) & ~(size_t)15;
    return L;
}

inline size_t cube_smem_bytes(const GridDev &g)
{
    const int bvol = (g.T[0] + 2) * (g.T[1] + 2) * (g.T[2] + 2);
    return cube_layout(bvol, g.tvol, g.T[0], g.T[1], g.T[2]).total;
}

// The shared deposit box.  In a block of at most 65535 grains each word takes
// at most one piece per grain, so a piece v with |v| < 2^31 is added exactly
// as two 32-bit counters that need no carry: the sum of the pieces modulo
// 2^32, and H, the sum of v >> 16 (signed, below 2^31 in size).  The pieces'
// low 16 bits add up to less than 2^32, so they are (sum - 65536 H) modulo
// 2^32, and the word is 65536 H plus them.  Both adds return nothing, so no
// lane waits for the shared-memory round trip.  Larger pieces go to the global
// deposit.  A denser block keeps the box as int64 words added as two 32-bit
// atomics with the carry.
struct CubeBox {
    unsigned long long *sdep;
    unsigned long long *dep;    // the global deposit
    int bvol, B0, B1;
    int o0, o1, o2;
    bool split;
};

__device__ __forceinline__ void cube_add_split(unsigned *blo, int bvol, int ch, int lin, int v)
{
    atomicAdd(&blo[ch * bvol + lin], (unsigned)v);
    atomicAdd(reinterpret_cast<int *>(blo) + 4 * bvol + ch * bvol + lin, v >> 16);
}

__device__ __forceinline__ long long cube_word(const unsigned *blo, int bvol, int ch, int lin)
{
    const int hi = (int)blo[(4 + ch) * bvol + lin];
    return (long long)hi * 65536 + (long long)(blo[ch * bvol + lin] - ((unsigned)hi << 16));
}

__device__ __forceinline__ void cube_add(const GridDev &g, const CubeBox &b, int ch, int lin, long long v)
{
    if (!b.split) shared_add_i64(&b.sdep[ch * b.bvol + lin], v);
    else if (v >= -2147483647LL && v <= 2147483647LL)
        cube_add_split(reinterpret_cast<unsigned *>(b.sdep), b.bvol, ch, lin, (int)v);
    else box_piece_to_global(g, b.dep, b.o0, b.o1, b.o2, b.B0, b.B1, lin, ch, v);
}

// Chunk sums too large for the 32-bit rounding, or a tile too dense for the
// split box: 64-bit roundings and sums.  lin: this lane's node; base: the
// host's.  Returns whether a sum was out of range.
template <int NCH>
__device__ __noinline__ bool cube_quantise_wide(const GridDev &g, const CubeBox &b, int lin, int base, float a0,
                                                float a1, float a2, float a3)
{
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const float acc[4] = {a0, a1, a2, a3};
    bool big = false;
#pragma unroll 1
    for (int ch = 0; ch < NCH; ++ch) {
        const float v = ch == 0 ? acc[0] : (ch == 1 ? acc[1] : (ch == 2 ? acc[2] : acc[3]));
        long long piece = 0;
        if (lane < 27) {
            big |= !(fabsf(v) < 4.5e15f);
            piece = rround(v);
        }
        long long sum = piece;  // lane 13 holds minus the chunk's total
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(FULL, sum, o);
        if (lane == 13) {
            if (sum != 0) cube_add(g, b, ch, base, -sum);
        } else if (lane < 27) {
            cube_add(g, b, ch, lin, piece);
        }
    }
    return big;
}

// The three weights of each direction of a grain at offsets u (dl: in zone
// widths) from its zone's centre; qf the coordinates.
template <int GEOM>
__device__ __forceinline__ void cube_weights(int tsc, bool vol, const float u[3], const float dl[3],
                                             const float qf[3], const float zcf[3], float znu, float zlo, float zhi,
                                             float zhw, const float zvl[2], const float zvh[2], float w[3][3])
{
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        if ((GEOM == GEOM_CYL || GEOM == GEOM_SPH) && d == 0) {
            if (vol) cube_w_vol<GEOM>(0, u[0], zcf[0], zvl[0], zvh[0], w[0]);
            else if (GEOM == GEOM_CYL) cube_w_cyl(tsc, dl[0], znu, w[0]);
            else cube_w_sphr<false>(tsc, dl[0], znu, w[0]);
        } else if (GEOM == GEOM_SPH && d == 1) {
            if (vol) cube_w_vol<GEOM>(1, u[1], zcf[1], zvl[1], zvh[1], w[1]);
            else cube_w_theta(tsc, qf[1], zlo, zhi, u[1], zhw, w[1]);
        } else {
            cube_w_cart(tsc, dl[d], w[d]);
        }
    }
}

// What a grain still needs after the push of its 32: the exact key prediction,
// or (a grain whose half-step zone is not its key zone, with stale keys) the
// whole step on its own, or the 64-bit rounding of its chunk (cube_calm).
enum { CUBE_KEY = 1, CUBE_STRAY = 2, CUBE_WILD = 4 };

// The block's constants as the out-of-line paths read them.
struct CubeRare {
    CubeBox box;
    const float *sgas;
    int o[3], B[3];
    int wk;                  // weighting: 0 CIC, 1 TSC, 2 volume
    int32_t nkeys;
    float h, dt;
};

// First half drift in double precision, boundaries, exact zone search and
// weights of a grain that is not in its key zone (see slab_exact_first_half).
// The drift and the boundaries are the general path's functions, whose sums have
// one product each that can be fused; of the volume weights' shell volumes, in
// double precision, the compiler chooses which.  Returns false if it left the
// grid.
template <int GEOM>
__device__ __forceinline__ bool cube_exact_first_half(const GridDev &g, const PhysDev &ph, double shift, int wk, float h,
                                                      SlabExact &e)
{
#pragma unroll
    for (int d = 0; d < 3; ++d) e.inc[d] = 0.f;
    drift<float, GEOM>(ph, e.q, e.q, e.p, h, false, e.inc);
    if (!apply_bc<float, GEOM>(g, ph, shift, e.q, e.p)) return false;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        e.qf[d] = (float)e.q[d];
        const int i = locate(g, d, e.q[d]);
        e.host[d] = i;
        const float off = (float)(e.q[d] - g.zc[d][i]);
        e.iw[d] = g.ziw_f[d][i];
        const float dd = fm(off, e.iw[d]);
        const int tsc = wk == 1;
        if (wk == 2 && (((GEOM == GEOM_CYL || GEOM == GEOM_SPH) && d == 0) || (GEOM == GEOM_SPH && d == 1)))
            w_volume<float, GEOM>(g, d, e.q[d], i, e.w[d]);
        else if (GEOM == GEOM_CYL && d == 0) cube_w_cyl(tsc, dd, g.znu_f[d][i], e.w[d]);
        else if (GEOM == GEOM_SPH && d == 0) cube_w_sphr<true>(tsc, dd, g.znu_f[d][i], e.w[d]);
        else if (GEOM == GEOM_SPH && d == 1)
            cube_w_theta(tsc, e.qf[d], g.zlo_f[d][i], g.zlo_f[d][i + 1], off, fd(0.5f, e.iw[d]), e.w[d]);
        else cube_w_cart(tsc, dd, e.w[d]);
    }
    return true;
}

// Out of line, so that the hot loop keeps its registers: the rest of the step
// of the lanes with todo != 0 (grain at sorted position gi, read from src).
// CUBE_KEY: the grain's end position and momentum are in the store.
// CUBE_STRAY: the whole step, from the store, in the order of the one-thread-
// per-grain kernel; the grain deposits by itself (the rule of deposit_fixed),
// in the box through the node lanes (its record: impulse, the products of its
// y and z weights, its x weights) or, with a stencil that leaves the box, into
// the global deposit.
struct CubeRareOut {
    int32_t nkey;   // key for the next sort
    int lin;        // a stray's host node in the box, -1: nothing left to deposit
};

template <int GEOM>
__device__ __noinline__ CubeRareOut cube_rare(const TiledArgs<float> &TA, const CubeRare &R, int todo, int gi, int src,
                                              int sp, float value, int32_t nkey, float4 *rec)
{
    CubeRareOut out{nkey, -1};
    if (todo == 0) return out;
    const StepArgs<float> &A = TA.s;
    const GridDev &g = A.g;
    const StoreDev<float> &O = TA.dst;
    double q[3];
    float pnew[3];
    bool alive = true;
    if (todo & CUBE_STRAY) {
        SlabExact ex;
#pragma unroll
        for (int d = 0; d < 3; ++d) { ex.q[d] = A.s.q[d][src]; ex.p[d] = A.s.p[d][src]; }
        alive = cube_exact_first_half<GEOM>(g, A.ph, shift_mid_of(A), R.wk, R.h, ex);
        // removed in its first half drift, in place: its other columns stay
        const bool stays = !alive && !TA.perm;
#pragma unroll
        for (int d = 0; d < 3; ++d) { q[d] = ex.q[d]; pnew[d] = ex.p[d]; }
        if (alive) {
            int lb[3];
            bool inbox = true;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                int l = ex.host[d] - R.o[d];
                if (g.bc[d] == DUST_BC_PERIODIC) {
                    if (l < 0) l += g.n[d];
                    else if (l >= R.B[d]) l -= g.n[d];
                }
                lb[d] = l;
                inbox &= (l >= 1) && (l <= R.B[d] - 2);
            }
            float G[4] = {0.f, 0.f, 0.f, 0.f};
            if (inbox) gather_box<3, 3>(R.sgas, lb, R.B[0], R.B[1], ex.w, G);
            else gather_global<3, 3>(g, A.gas, ex.host, ex.w, G);
            float tau, E, cg, h1;
            if (!A.s.param && ((A.sp.coef_const >> sp) & 1u)) {
                tau = A.sp.tau_eff_f[sp];
                E = A.sp.E_f[sp];
                cg = A.sp.cg_f[sp];
                h1 = A.sp.h1_f[sp];
            } else {
                tau = stopping_time<float, GEOM>(A.ph, A.sp.mode[sp], value, ex.qf, G[0]);
                const float x = R.dt / tau;
                E = expf(-x);
                cg = -expm1f(-x);
                h1 = (x == 0.f) ? R.dt : R.dt * cg / x;
            }
            const float vg[3] = {G[1], G[2], G[3]};
            float pp[3], D[4], inc2[3];
            cube_kick<GEOM>(A.ph, A.sp.mqf[sp], ex.qf, ex.p, vg, tau, R.dt, E, cg, h1, pp, D);
            cube_drift2<GEOM>(A.ph, R.h, ex.qf, pp, inc2);
            float moved = 0.f;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                q[d] += (double)inc2[d];
                moved = fmaxf(moved, fm(fabsf(fa(ex.inc[d], inc2[d])), ex.iw[d]));
                pnew[d] = pp[d];
            }
            alive = apply_bc<float, GEOM>(g, A.ph, shift_end_of(A), q, pnew);
            if (!(isfinite(pp[0]) && isfinite(pp[1]) && isfinite(pp[2]))) atomicOr(&A.status[ST_FLAGS], DUST_FLAG_NAN);
            atomicMax(&A.status[ST_MAXMOVE], __float_as_uint(moved));
            if (inbox) {
                out.lin = lb[0] + R.B[0] * (lb[1] + R.B[1] * lb[2]);
                rec[0] = make_float4(D[0], D[1], D[2], D[3]);
                rec[1] = make_float4(fm(ex.w[1][0], ex.w[2][0]), fm(ex.w[1][1], ex.w[2][0]), fm(ex.w[1][2], ex.w[2][0]),
                                     fm(ex.w[1][0], ex.w[2][1]));
                rec[2] = make_float4(fm(ex.w[1][1], ex.w[2][1]), fm(ex.w[1][2], ex.w[2][1]), fm(ex.w[1][0], ex.w[2][2]),
                                     fm(ex.w[1][1], ex.w[2][2]));
                rec[3] = make_float4(fm(ex.w[1][2], ex.w[2][2]), ex.w[0][0], ex.w[0][1], ex.w[0][2]);
            } else {
                deposit_fixed_rolled<3, 3>(g, R.box.dep, ex.host, ex.w, D, A.status);
            }
        }
        if (!alive) {
            q[0] = __longlong_as_double(0x7ff8000000000000LL);
            atomicAdd(reinterpret_cast<unsigned long long *>(&A.status[ST_REMOVED_LO]), 1ull);
            out.nkey = R.nkeys;
        }
        if (stays) {
            O.q[0][gi] = q[0];
        } else {
#pragma unroll
            for (int d = 0; d < 3; ++d) { O.q[d][gi] = q[d]; O.p[d][gi] = pnew[d]; }
        }
    } else {
#pragma unroll
        for (int d = 0; d < 3; ++d) { q[d] = O.q[d][gi]; pnew[d] = O.p[d][gi]; }
    }
    if (TA.emit_keys) {
        if (alive) out.nkey = predict_key<float, GEOM>(g, A.ph, q, pnew, R.h);
        TA.key_out[gi] = out.nkey;
    }
    return out;
}

// The same for the predictor: the impulse of a grain that is not in its key
// zone at x^n.  Returns whether a channel was out of range.
template <int GEOM>
__device__ __noinline__ bool cube_rare_predict(const TiledArgs<float> &TA, const CubeRare &R, int src, int sp, float value)
{
    const StepArgs<float> &A = TA.s;
    const GridDev &g = A.g;
    const double q[3] = {A.s.q[0][src], A.s.q[1][src], A.s.q[2][src]};
    const float pn[3] = {A.s.p[0][src], A.s.p[1][src], A.s.p[2][src]};
    int host[3], lb[3];
    float w[3][3], qf[3], iwd;
    bool inbox = true;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        zone_weights<float, GEOM>(g, d, R.wk, q[d], host[d], w[d], iwd);
        qf[d] = (float)q[d];
        int l = host[d] - R.o[d];
        if (g.bc[d] == DUST_BC_PERIODIC) {
            if (l < 0) l += g.n[d];
            else if (l >= R.B[d]) l -= g.n[d];
        }
        lb[d] = l;
        inbox &= (l >= 1) && (l <= R.B[d] - 2);
    }
    float G[4] = {0.f, 0.f, 0.f, 0.f};
    if (inbox) gather_box<3, 3>(R.sgas, lb, R.B[0], R.B[1], w, G);
    else gather_global<3, 3>(g, A.gas, host, w, G);
    const float tau = stopping_time<float, GEOM>(A.ph, A.sp.mode[sp], value, qf, G[0]);
    const float taup = fmaxf(tau, fabsf(R.dt));
    const float coef = 0.5f * R.dt * A.sp.mqf[sp] / taup;
    const float D[4] = {coef * (pn[0] - G[1]), coef * (pn[1] - G[2]), coef * (pn[2] - G[3]), 0.f};
    if (!inbox) {
        deposit_fixed_rolled<3, 3>(g, R.box.dep, host, w, D, A.status);
        return false;
    }
    return deposit_box_per_grain<3, 3>([&](int ch, int lin, long long v) { cube_add(g, R.box, ch, lin, v); }, lb,
                                       R.B[0], R.B[1], w, D);
}

// First zone of share k of nk of the zones [z0, z1): the first at which the
// work of the zones before it, 2 per grain and 3 per zone, reaches k / nk of
// the whole.  The whole warp searches, 32 zones at a time.
__device__ __forceinline__ int cube_share(const int *koff, int z0, int z1, int k, int nk)
{
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const float goal = (2.f * (float)(koff[z1] - koff[z0]) + 3.f * (float)(z1 - z0)) * ((float)k / (float)nk);
    int lo = z0, hi = z1;  // the work before lo is below the goal or lo == z0; before hi it reaches it
    while (hi > lo) {
        const int step = (hi - lo + 31) >> 5;
        const int z = min(lo + (lane + 1) * step, hi);
        const bool reached = z == hi || 2.f * (float)(koff[z] - koff[z0]) + 3.f * (float)(z - z0) >= goal;
        const int f = __ffs(__ballot_sync(FULL, reached)) - 1;  // the first probe that reaches it
        hi = min(lo + (f + 1) * step, hi);
        lo = lo + f * step;
        if (step == 1) break;
    }
    return hi;
}

// Grains removed before the last sort sit after every zone's segment: they
// keep the removed-grain key and are moved as they are (all blocks share them).
__device__ __forceinline__ void cube_move_removed(const TiledArgs<float> &TA)
{
    const GridDev &g = TA.s.g;
    const StoreDev<float> &S = TA.s.s;
    if (!TA.emit_keys && !TA.perm) return;
    const int D0 = TA.key_off[g.nkeys], D1 = (int)S.n;
    for (int gi = D0 + (int)(blockIdx.x * blockDim.x + threadIdx.x); gi < D1; gi += (int)(gridDim.x * blockDim.x)) {
        if (TA.emit_keys) TA.key_out[gi] = (int32_t)g.nkeys;
        if (TA.perm) {
            const StoreDev<float> &O = TA.dst;
            const int src = TA.perm[gi];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                O.q[d][gi] = S.q[d][src];
                O.p[d][gi] = S.p[d][src];
            }
            O.id[gi] = TA.perm_id[gi];
            if (S.species) O.species[gi] = S.species[src];
            if (S.param) O.param[gi] = S.param[src];
        }
    }
    if (TA.emit_keys && blockIdx.x == 0 && threadIdx.x == 0 && D1 > D0)
        atomicAdd(&TA.count_out[g.nkeys], (int32_t)(D1 - D0));
}

// Part `part` of `parts` of one tile.  TX > 0: the copy compiled for a
// TX x TY x TZ tile with TSC weights.  MODE as in slab_tile.  PRED: the gas
// predictor (Sec. 3.1) instead of the step: the drag impulse over half a step
// of the grains at x^n, deposited at x^n into TA.s.dep; nothing is moved.
// VAR: 0, or CUBE_FULL (the sort's gather is fused into the step and the keys
// of the next sort are predicted: every step of the default sort interval)
// with CUBE_SPECIES / CUBE_PARAM as the store has these columns; the tests for
// them then leave the hot code.
enum { CUBE_FULL = 1, CUBE_SPECIES = 2, CUBE_PARAM = 4 };

template <int GEOM, int MODE, int TX, int TY, int TZ, bool PRED, int VAR>
__device__ __forceinline__ void cube_tile(const TiledArgs<float> &TA, const int tile, const int part, const int parts,
                                          unsigned char *smem_raw)
{
    const StepArgs<float> &A = TA.s;
    const GridDev &g = A.g;
    constexpr bool FIX = TX > 0;
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int NCH = PRED ? 3 : 4;  // the predictor's impulse has no energy channel
    const int T0 = FIX ? TX : g.T[0], T1 = FIX ? TY : g.T[1], T2 = FIX ? TZ : g.T[2];
    const int tvol = FIX ? TX * TY * TZ : g.tvol;
    const int tsc = FIX ? 1 : TA.tsc;
    const bool vol = FIX ? false : TA.vol != 0;
    PhysDev ph = A.ph;
    if (MODE > 0) ph.pusher = DUST_PUSHER_EM;
    if (GEOM == GEOM_SB && MODE == 1) ph.fargo = 1;
    if (GEOM == GEOM_SB && MODE == 2) ph.fargo = 0;

    const StoreDev<float> &S = A.s;
    const StoreDev<float> &O = TA.dst;  // the same store without a permutation
    constexpr bool kFull = (VAR & CUBE_FULL) != 0;
    const bool perm = kFull || TA.perm != nullptr, emit = kFull || TA.emit_keys != 0;
    const bool has_species = kFull ? (VAR & CUBE_SPECIES) != 0 : S.species != nullptr;
    const bool has_param = kFull ? (VAR & CUBE_PARAM) != 0 : S.param != nullptr;
    // the block's zones (tile-local keys)
    const int zb0 = (int)(((int64_t)part * tvol) / parts), zb1 = (int)(((int64_t)(part + 1) * tvol) / parts);
    const int64_t kbase = (int64_t)tile * tvol;
    const int g0 = TA.key_off[kbase + zb0], g1 = TA.key_off[kbase + zb1];  // its grains (fewer than 2^31)

    int tc[3];
    tc[0] = tile % g.nt[0];
    tc[1] = (tile / g.nt[0]) % g.nt[1];
    tc[2] = tile / (g.nt[0] * g.nt[1]);
    const int B[3] = {T0 + 2, T1 + 2, T2 + 2};
    const int o[3] = {tc[0] * T0 - 1, tc[1] * T1 - 1, tc[2] * T2 - 1};
    const int bvol = B[0] * B[1] * B[2];
    const CubeLayout L = cube_layout(bvol, tvol, T0, T1, T2);
    float *sgas = reinterpret_cast<float *>(smem_raw);
    unsigned long long *sdep = reinterpret_cast<unsigned long long *>(smem_raw + L.dep);
    unsigned *blo = reinterpret_cast<unsigned *>(sdep);
    CubeZone *szone = reinterpret_cast<CubeZone *>(smem_raw + L.zone);
    int *skoff = reinterpret_cast<int *>(smem_raw + L.off);
    float2 *slim = reinterpret_cast<float2 *>(smem_raw + L.lim);
    float *sznu = reinterpret_cast<float *>(smem_raw + L.nu);
    float *szlo = reinterpret_cast<float *>(smem_raw + L.lo);
    float *szhw = reinterpret_cast<float *>(smem_raw + L.hw);
    float *szvl = reinterpret_cast<float *>(smem_raw + L.vl), *szvh = reinterpret_cast<float *>(smem_raw + L.vh);
    unsigned long long *sbar = reinterpret_cast<unsigned long long *>(smem_raw + L.bar);
    for (int k = threadIdx.x; k < 2 * bvol; k += blockDim.x)
        reinterpret_cast<uint4 *>(sdep)[k] = make_uint4(0u, 0u, 0u, 0u);
    // No grains: nothing to stage or deposit.  The test stands after the clear,
    // which covers the latency of the two offsets (before it: 128^3 box 1.9%
    // slower); a ring of 200k grains in 192x512x32 zones, most of whose tiles are
    // empty, takes 151 us a step with the test here and 200 us with one after
    // the staging.
    if (g1 <= g0) return;
    // the gas box by one bulk tensor copy, overlapping the tables below
    gas_box_begin<float>(TA.gas_tmap, sgas, o, bvol, sbar, TA.wait_extra_tx);
    const int tsum = T0 + T1 + T2;
    for (int t = threadIdx.x; t < tsum + T1 + 1; t += blockDim.x) {
        if (t < tsum) {
            const int d = t < T0 ? 0 : (t < T0 + T1 ? 1 : 2);
            const int l = t - (d == 0 ? 0 : (d == 1 ? T0 : T0 + T1));
            const int z = tc[d] * (d == 0 ? T0 : (d == 1 ? T1 : T2)) + l;
            const bool ok = z < g.n[d];
            CubeZone e;
            e.c = ok ? g.zc[d][z] : 0.0;
            e.cf = ok ? g.zc_f[d][z] : 0.f;
            e.iw = ok ? g.ziw_f[d][z] : 0.f;
            szone[t] = e;
            // how far below and above the zone's centre (in zone widths) a grain
            // may end and is certainly inside the grid (the offset's error is
            // ~1e-7): inside its zone, or, on a uniform direction, at most two
            // zones away and short of the grid's edge
            const bool uni = g.edge_kind[d] == EDGE_UNIFORM;
            slim[t] = make_float2(uni ? -fminf(1.999f, (float)z + 0.499f) : -0.499f,
                                  uni ? fminf(1.999f, (float)(g.n[d] - 1 - z) + 0.499f) : 0.499f);
            if (d == 0 && (GEOM == GEOM_CYL || GEOM == GEOM_SPH)) sznu[l] = ok ? g.znu_f[0][z] : 0.f;
            if (d == 1 && GEOM == GEOM_SPH) szhw[l] = ok ? 0.5f / e.iw : 0.f;
        } else if (GEOM == GEOM_SPH) {
            const int z = tc[1] * T1 + (t - tsum);
            szlo[t - tsum] = z <= g.n[1] ? g.zlo_f[1][z] : 0.f;
        }
    }
    if ((GEOM == GEOM_CYL || GEOM == GEOM_SPH) && vol) {
        for (int t = threadIdx.x; t < T0 + (GEOM == GEOM_SPH ? T1 : 0); t += blockDim.x) {
            const int d = t < T0 ? 0 : 1;
            const int z = d == 0 ? tc[0] * T0 + t : tc[1] * T1 + (t - T0);
            float vl = 0.f, vh = 0.f;
            if (z < g.n[d]) {
                const double c = g.zc[d][z];
                vl = (float)(1.0 / vol_shell<GEOM>(d, vol_node(g, d, z - 1), c));
                vh = (float)(1.0 / vol_shell<GEOM>(d, c, vol_node(g, d, z + 1)));
            }
            szvl[t] = vl;
            szvh[t] = vh;
        }
    }
    // store positions fit in 32 bits (fewer than 2^31 grains)
    for (int k = zb0 + threadIdx.x; k <= zb1; k += blockDim.x) skoff[k] = TA.key_off[kbase + k];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nwarps = blockDim.x >> 5;
    float *rec = reinterpret_cast<float *>(smem_raw + L.rec) + warp * (32 * kCubeRec);
    rec[lane * kCubeRec + kCubeOne] = -1.f;
    rec[lane * kCubeRec + kCubeOne + 1] = 1.f;
    __syncthreads();
    if (!gas_box_finish<float>(g, A.gas, TA.gas_tmap, sgas, o, B, sbar, A.status, TA.wait_ns)) return;

    CubeBox box;
    box.sdep = sdep;
    box.dep = A.dep;
    box.bvol = bvol;
    box.B0 = B[0]; box.B1 = B[1];
    box.o0 = o[0]; box.o1 = o[1]; box.o2 = o[2];
    box.split = g1 - g0 <= 65535;
    CubeRare R;
    R.box = box;
    R.sgas = sgas;
#pragma unroll
    for (int d = 0; d < 3; ++d) { R.o[d] = o[d]; R.B[d] = B[d]; }
    R.wk = vol ? 2 : (tsc & 1);
    R.nkeys = (int32_t)g.nkeys;
    R.h = (float)(0.5 * A.dt);
    R.dt = (float)A.dt;
    const bool split = box.split;

    // this lane's stencil node (lanes 0-26; x fastest), its place relative to
    // the host node and in a record.  Lane 13 (the host) sums minus the impulse
    // itself (weight -1): the host takes the rest of the rounded total.  Lane
    // 27 sums the host's share, which only bounds that rest.
    const int na = lane % 3, nb = (lane / 3) % 3, nc = lane / 9;
    const int nlin = (na - 1) + B[0] * ((nb - 1) + B[1] * (nc - 1));
    const float *rw = rec + (lane < 27 ? (lane == 13 ? kCubeOne : 4 + na + 3 * nb) : 4 + 4);
    const float *rz = rec + (lane < 27 ? (lane == 13 ? kCubeOne + 1 : 13 + nc) : 13 + 1);

    const float h = (float)(0.5 * A.dt), dt = (float)A.dt;
    int nremoved = 0;
    float moved = 0.f;
    bool big = false, bad = false;
    float2 acc01 = make_float2(0.f, 0.f), acc23 = make_float2(0.f, 0.f);
    bool wild = false;  // not all of these grains, or of an open chunk before them, are calm

    // each warp: a range of the block's zones with an equal share of the work
    // (a zone's roundings cost about as much as 1.5 grains), its grains 32 at
    // a time
    const int zw0 = warp == 0 ? zb0 : cube_share(skoff, zb0, zb1, warp, nwarps);
    const int zw1 = warp == nwarps - 1 ? zb1 : cube_share(skoff, zb0, zb1, warp + 1, nwarps);
    const int Gend = skoff[zw1];
    int zc = zw0;
    // this lane's grain of the next 32: its columns, loaded before the deposit
    // of the current ones, and its source position 32 grains further on
    double q[3] = {0.0, 0.0, 0.0};
    float pn[3] = {0.f, 0.f, 0.f}, par = 0.f;
    int sp = 0, src = 0, src_next = 0, pid = 0;
    auto load_grain = [&](int gi) {
        if (gi < Gend) {
            src = perm ? src_next : gi;
            if (perm) {
                if (gi + 32 < Gend) src_next = TA.perm[gi + 32];
                if (!PRED) pid = TA.perm_id[gi];
            }
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                q[d] = S.q[d][src];
                pn[d] = S.p[d][src];
            }
            sp = has_species ? S.species[src] : 0;
            par = has_param ? S.param[src] : 0.f;
        }
    };
    {
        const int gi = skoff[zw0] + lane;
        if (perm && gi < Gend) src_next = TA.perm[gi];
        load_grain(gi);
    }
    auto add = [&](float W, float4 De) {
        const float2 W2 = make_float2(W, W);
        acc01 = __ffma2_rn(W2, make_float2(De.x, De.y), acc01);
        acc23 = __ffma2_rn(W2, make_float2(De.z, De.w), acc23);
    };
    // A chunk's sums, rounded, into the box around its host node base.  Sums
    // below kCubeNarrow take the 32-bit rounding, which gives the same integers
    // as the 64-bit one at a fraction of its cost; the host's rest has to fit in
    // 32 bits as well for its modular sum to be exact.  Lane 27 holds the host's
    // share, which the rest differs from by the rounding of 27 lanes' partial
    // sums: bounded where the chunk is calm (below), not by the final sums, of
    // which nothing but that rounding is left where large impulses cancel.
    auto chunk_end = [&](int base, bool calm) {
        const int lin = base + nlin;
        const float top = fmaxf(fmaxf(fabsf(acc01.x), fabsf(acc01.y)), fabsf(acc23.x));
        const bool narrow = top < kCubeNarrow && (NCH < 4 || fabsf(acc23.y) < kCubeNarrow);
        if (__all_sync(FULL, narrow) && calm) {
            if (lane < 27) {
                int v[4] = {__float2int_rn(acc01.x), __float2int_rn(acc01.y), __float2int_rn(acc23.x),
                            NCH == 4 ? __float2int_rn(acc23.y) : 0};
#pragma unroll
                for (int ch = 0; ch < NCH; ++ch) {
                    // the other nodes minus the chunk's total (modulo 2^32)
                    const int r = __reduce_add_sync(0x07ffffffu, v[ch]);
                    if (lane == 13) v[ch] = -r;
                }
#pragma unroll
                for (int ch = 0; ch < NCH; ++ch) cube_add_split(blo, bvol, ch, lin, v[ch]);
            }
        } else {
            big |= cube_quantise_wide<NCH>(g, box, lin, base, acc01.x, acc01.y, acc23.x, acc23.y);
        }
        acc01 = make_float2(0.f, 0.f);
        acc23 = make_float2(0.f, 0.f);
    };
    for (int P0 = skoff[zw0]; P0 < Gend; P0 += 32) {
        const int m = min(32, Gend - P0);
        const int gi = P0 + lane;
        const bool valid = lane < m;
        const int gq = P0 + min(lane, m - 1);
        // the zone of each grain: zc plus the number of later zones of the
        // range that start at or before it (offsets are nondecreasing; 32
        // zones at a time, counted by a binary search over the lanes)
        int myz = zc;
        for (int zb = zc;; zb += 32) {
            const int v = zb + 1 + lane < zw1 ? skoff[zb + 1 + lane] : 0x7fffffff;
            int c = 0;
#pragma unroll
            for (int s = 16; s > 0; s >>= 1)
                if (__shfl_sync(FULL, v, c + s - 1) <= gq) c += s;
            const int last = __shfl_sync(FULL, v, 31);
            if (last <= gq) c = 32;
            myz += c;
            if (last > P0 + m - 1) break;
        }
        zc = __shfl_sync(FULL, myz, 31);
        // grains that end a chunk: their zone's last, or kSlabCap by rank
        const int rank = gq - skoff[myz];
        const bool at_end = ((rank + 1) & (kSlabCap - 1)) == 0 || gq + 1 == skoff[myz + 1];
        unsigned ends = __ballot_sync(FULL, valid && at_end);

        int lx, ly, lz;
        if (FIX) {
            lx = myz % (FIX ? TX : 2);
            ly = (myz / (FIX ? TX : 1)) % (FIX ? TY : 2);
            lz = myz / (FIX ? TX * TY : 1);
        } else {
            lx = myz % T0;
            ly = (myz / T0) % T1;
            lz = myz / (T0 * T1);
        }
        const int hl = (lx + 1) + B[0] * ((ly + 1) + B[1] * (lz + 1));  // the zone in the box
        int32_t nkey = (int32_t)g.nkeys;   // next sort key (removed: nkeys)
        int todo = 0;
        // the record: weights, and the impulse of a grain in its key zone (zero:
        // the grain deposits by itself, or is removed)
        float w[3][3] = {{0.f, 1.f, 0.f}, {0.f, 1.f, 0.f}, {0.f, 1.f, 0.f}};
        float D[4] = {0.f, 0.f, 0.f, 0.f};
        if (valid) {
            const CubeZone Z[3] = {szone[lx], szone[T0 + ly], szone[T0 + T1 + lz]};
            const double zcd[3] = {Z[0].c, Z[1].c, Z[2].c};
            const float zcf[3] = {Z[0].cf, Z[1].cf, Z[2].cf}, zif[3] = {Z[0].iw, Z[1].iw, Z[2].iw};
            float znu = 0.f, zlo = 0.f, zhi = 0.f, zhw = 0.f;
            float zvl[2] = {0.f, 0.f}, zvh[2] = {0.f, 0.f};
            if (GEOM == GEOM_CYL || GEOM == GEOM_SPH) {
                znu = sznu[lx];
                if (vol) {
                    zvl[0] = szvl[lx];
                    zvh[0] = szvh[lx];
                    if (GEOM == GEOM_SPH) {
                        zvl[1] = szvl[T0 + ly];
                        zvh[1] = szvh[T0 + ly];
                    }
                }
            }
            if (GEOM == GEOM_SPH) {
                zlo = szlo[ly];
                zhi = szlo[ly + 1];
                zhw = szhw[ly];
            }
            const float value = has_param ? par : A.sp.tau_f[sp];
            float u[3] = {0.f, 0.f, 0.f}, qf[3] = {0.f, 0.f, 0.f}, dl[3];
            bool live = !isnan(q[0]), ingroup = false;
            if constexpr (PRED) {
                if (live) {
                    ingroup = true;
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        u[d] = __double2float_rn(q[d] - zcd[d]);
                        qf[d] = fa(zcf[d], u[d]);
                        dl[d] = fm(u[d], zif[d]);
                        ingroup &= fabsf(dl[d]) <= 0.50001f;
                    }
                    if (ingroup) {
                        cube_weights<GEOM>(tsc, vol, u, dl, qf, zcf, znu, zlo, zhi, zhw, zvl, zvh, w);
                        const int lb[3] = {lx + 1, ly + 1, lz + 1};
                        float G[4] = {0.f, 0.f, 0.f, 0.f};
                        gather_box<3, 3>(sgas, lb, B[0], B[1], w, G);
                        const float tau = stopping_time<float, GEOM>(ph, A.sp.mode[sp], value, qf, G[0]);
                        const float taup = fmaxf(tau, fabsf(dt));
                        const float coef = 0.5f * dt * A.sp.mqf[sp] / taup;
                        D[0] = fm(coef, fs(pn[0], G[1]));
                        D[1] = fm(coef, fs(pn[1], G[2]));
                        D[2] = fm(coef, fs(pn[2], G[3]));
                    } else {
                        todo = CUBE_STRAY;
                    }
                }
            } else {
                float inc1[3] = {0.f, 0.f, 0.f};
                if (live) {
#pragma unroll
                    for (int d = 0; d < 3; ++d) u[d] = __double2float_rn(q[d] - zcd[d]);
                    cube_drift1<GEOM>(ph, h, zcf, pn, u, inc1);
                    ingroup = true;
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        qf[d] = fa(zcf[d], u[d]);
                        dl[d] = fm(u[d], zif[d]);
                        ingroup &= fabsf(dl[d]) <= 0.50001f;
                    }
                    if (!ingroup) todo = CUBE_STRAY;
                }
                float pnew[3] = {pn[0], pn[1], pn[2]};
                bool alive = true;
                // kick, second half drift, deposit impulse
                if (ingroup) {
                    cube_weights<GEOM>(tsc, vol, u, dl, qf, zcf, znu, zlo, zhi, zhw, zvl, zvh, w);
                    // 27-node gather (Eq. Delta_vp) from the staged gas box; the
                    // grains of one zone read the same nodes (broadcast loads)
                    float G[4] = {0.f, 0.f, 0.f, 0.f};
                    const int lb[3] = {lx + 1, ly + 1, lz + 1};
                    gather_box<3, 3>(sgas, lb, B[0], B[1], w, G);
                    float tau, E, cg, h1;
                    if (!has_param && ((A.sp.coef_const >> sp) & 1u)) {
                        // the species' propagators for this dt (host, once)
                        tau = A.sp.tau_eff_f[sp];
                        E = A.sp.E_f[sp];
                        cg = A.sp.cg_f[sp];
                        h1 = A.sp.h1_f[sp];
                    } else {
                        tau = stopping_time<float, GEOM>(ph, A.sp.mode[sp], value, qf, G[0]);
                        const float x = dt / tau;
                        E = expf(-x);
                        cg = -expm1f(-x);
                        h1 = (x == 0.f) ? dt : dt * cg / x;
                    }
                    const float vg[3] = {G[1], G[2], G[3]};
                    float pp[3], inc2[3];
                    cube_kick<GEOM>(ph, A.sp.mqf[sp], qf, pn, vg, tau, dt, E, cg, h1, pp, D);
                    // second half drift, then one double-precision update by
                    // the summed increment
                    cube_drift2<GEOM>(ph, h, qf, pp, inc2);
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        const float sum = fa(inc1[d], inc2[d]);
                        q[d] += (double)sum;
                        moved = fmaxf(moved, fm(fabsf(sum), zif[d]));
                        u[d] = fa(u[d], inc2[d]);  // the end offset
                        pnew[d] = pp[d];
                    }
                    // certainly inside the grid (slim above), or the exact
                    // boundary treatment
                    bool inner = true;
                    const float2 lim[3] = {slim[lx], slim[T0 + ly], slim[T0 + T1 + lz]};
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        const float t = fm(u[d], zif[d]);
                        inner = inner && t > lim[d].x && t < lim[d].y;
                    }
                    alive = inner || apply_bc<float, GEOM>(g, ph, shift_end_of(A), q, pnew);
                    bad |= !(isfinite(pp[0]) && isfinite(pp[1]) && isfinite(pp[2]));
                    if (!alive) {
                        q[0] = __longlong_as_double(0x7ff8000000000000LL);
                        ++nremoved;
                    }
                    if (emit && alive) {
                        // key for the next sort: the zone of the next step's
                        // half-step position (same dt), relative to this key
                        // zone in single precision; the exact prediction when
                        // the grain moves more than one zone or leaves the grid
                        bool fast = true, in = true;
                        int zn[3] = {tc[0] * T0 + lx, tc[1] * T1 + ly, tc[2] * T2 + lz};
                        cube_drift_key<GEOM>(ph, h, zcf, pnew, u);
#pragma unroll
                        for (int d = 0; d < 3; ++d) {
                            // zone offset floor(t + 1/2) for |t| < 3/2, by comparisons
                            const float t = fm(u[d], zif[d]);
                            zn[d] += (t >= 0.5f ? 1 : 0) - (t < -0.5f ? 1 : 0);
                            fast &= fabsf(t) < 1.5f;
                            in &= (unsigned)zn[d] < (unsigned)g.n[d];
                        }
                        if (!in) {
                            // through a periodic end of uniform zones: the zone one
                            // period on, where no edge is near enough (1e-3 zones,
                            // against an error of ~1e-6) for the exact prediction
                            // to differ
#pragma unroll
                            for (int d = 0; d < 3; ++d) {
                                fast &= fabsf(fabsf(fm(u[d], zif[d])) - 0.5f) > 1e-3f;
                                if ((unsigned)zn[d] < (unsigned)g.n[d]) continue;
                                fast &= g.bc[d] == DUST_BC_PERIODIC && g.edge_kind[d] == EDGE_UNIFORM &&
                                        !(GEOM == GEOM_SB && d == 0);
                                zn[d] += zn[d] < 0 ? g.n[d] : -g.n[d];
                            }
                        }
                        if (fast) {
                            // tile and place in it: shifts and masks for the
                            // compiled copy's power-of-two sides
                            int tt[3], ll[3];
#pragma unroll
                            for (int d = 0; d < 3; ++d) {
                                const int Td = d == 0 ? T0 : (d == 1 ? T1 : T2);
                                if (FIX) {
                                    tt[d] = (int)((unsigned)zn[d] / (unsigned)Td);
                                    ll[d] = (int)((unsigned)zn[d] % (unsigned)Td);
                                } else {
                                    int l = zn[d] - tc[d] * Td, t = tc[d];
                                    if (l < -1 || l > Td) { t = zn[d] / Td; l = zn[d] - t * Td; }
                                    else if (l < 0) { l += Td; --t; }
                                    else if (l >= Td) { l -= Td; ++t; }
                                    ll[d] = l;
                                    tt[d] = t;
                                }
                            }
                            nkey = (tt[0] + g.nt[0] * (tt[1] + g.nt[1] * tt[2])) * tvol +
                                   ll[0] + T0 * (ll[1] + T1 * ll[2]);
                        } else {
                            todo |= CUBE_KEY;
                        }
                    }
                }
                if (perm || live) {
                    O.q[0][gi] = q[0]; O.q[1][gi] = q[1]; O.q[2][gi] = q[2];
                    O.p[0][gi] = pnew[0]; O.p[1][gi] = pnew[1]; O.p[2][gi] = pnew[2];
                }
                if (perm) {
                    // the columns the step does not change
                    O.id[gi] = pid;
                    if (has_species) O.species[gi] = (uint8_t)sp;
                    if (has_param) O.param[gi] = par;
                }
                if (emit) TA.key_out[gi] = nkey;
            }
        }
        if (!cube_calm<GEOM>(D, w)) todo |= CUBE_WILD;
        if (__any_sync(FULL, todo != 0)) {
            const float value = has_param ? par : A.sp.tau_f[sp];
            wild = wild || __any_sync(FULL, (todo & CUBE_WILD) != 0);
            todo &= ~CUBE_WILD;
            if (!__any_sync(FULL, todo != 0)) {
            } else if constexpr (PRED) {
                if (todo) big |= cube_rare_predict<GEOM>(TA, R, src, sp, value);
            } else {
                const CubeRareOut r = cube_rare<GEOM>(TA, R, todo, gi, src, sp, value, nkey,
                                                      reinterpret_cast<float4 *>(rec + lane * kCubeRec));
                nkey = r.nkey;
                // strays: one at a time, a chunk of one grain (no partial sums)
                // whose weights are multiplied in the per-grain rule's order
                unsigned strays = __ballot_sync(FULL, r.lin >= 0);
                if (strays) {
                    __syncwarp();
                    const float2 s01 = acc01, s23 = acc23;
                    for (; strays; strays &= strays - 1u) {
                        const int k = __ffs(strays) - 1;
                        const float *e = rec + k * kCubeRec;
                        const int i = lane < 27 ? lane : 13;
                        const float W = lane == 13 ? -1.f : fm(e[13 + i % 3], e[4 + i / 3]);
                        acc01 = make_float2(fm(W, e[0]), fm(W, e[1]));
                        acc23 = make_float2(fm(W, e[2]), fm(W, e[3]));
                        chunk_end(__shfl_sync(FULL, r.lin, k), split);
                    }
                    acc01 = s01;
                    acc23 = s23;
                    __syncwarp();
                }
            }
        }
        {
            float4 *r4 = reinterpret_cast<float4 *>(rec + lane * kCubeRec);
            r4[0] = make_float4(D[0], D[1], D[2], D[3]);
            r4[1] = make_float4(w[0][0] * w[1][0], w[0][1] * w[1][0], w[0][2] * w[1][0], w[0][0] * w[1][1]);
            r4[2] = make_float4(w[0][1] * w[1][1], w[0][2] * w[1][1], w[0][0] * w[1][2], w[0][1] * w[1][2]);
            r4[3] = make_float4(w[0][2] * w[1][2], w[2][0], w[2][1], w[2][2]);
        }
        if (!PRED && emit) {
            // count runs of equal keys on consecutive lanes: one atomic per run
            const int prev = __shfl_up_sync(FULL, nkey, 1);
            const bool start = valid && (lane == 0 || prev != nkey);
            const unsigned starts = __ballot_sync(FULL, start);
            if (start) {
                const unsigned later = starts & ~((2u << lane) - 1u);
                const int end = later ? __ffs(later) - 1 : m;
                atomicAdd(&TA.count_out[nkey], end - lane);
            }
        }
        load_grain(gi + 32);
        __syncwarp();
        const bool quick = split && !wild;
        // ---- deposit: one node per lane, the records in order, a rounding
        // at the end of every chunk
        // groups of four records; stale records after the range's last grain
        // (which ends a chunk) only reach sums that are never used
#pragma unroll 1
        for (int k = 0; k < m; k += 4) {
            const unsigned e = (ends >> k) & 15u;
            float W[4];
            float4 De[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                W[j] = fm(rw[(k + j) * kCubeRec], rz[(k + j) * kCubeRec]);
                De[j] = *reinterpret_cast<const float4 *>(rec + (k + j) * kCubeRec);
            }
            if (e == 0u) {
#pragma unroll
                for (int j = 0; j < 4; ++j) add(W[j], De[j]);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    add(W[j], De[j]);
                    if (e & (1u << j)) chunk_end(__shfl_sync(FULL, hl, k + j), quick);
                }
            }
        }
        wild = wild && !(ends >> 31);  // only a chunk that these grains left open goes on
        __syncwarp();
    }
    if (big || bad) atomicOr(&A.status[ST_FLAGS], (big ? DUST_FLAG_OVERFLOW : 0) | (bad ? DUST_FLAG_NAN : 0));
    __syncthreads();

    // ---- flush the deposit box
    // a thread takes one channel of a node, channels fastest, so that the adds
    // of a warp fall on whole consecutive zones; four words are read before
    // their adds are issued (one at a time took 8.5 of a tile's 83 us)
    for (int t0 = threadIdx.x; t0 < 4 * bvol; t0 += 4 * blockDim.x) {
        long long v[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int t = t0 + r * (int)blockDim.x, c = t & 3, lin = t >> 2;
            v[r] = t >= 4 * bvol ? 0 : (split ? cube_word(blo, bvol, c, lin) : (long long)sdep[c * bvol + lin]);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            if (v[r] == 0) continue;
            const int t = t0 + r * (int)blockDim.x, lin = t >> 2;
            const int row = lin / B[0], bz = row / B[1];
            const int i = map_zone(o[0] + lin - row * B[0], g.n[0], g.bc[0]);
            const int j = map_zone(o[1] + row - bz * B[1], g.n[1], g.bc[1]);
            const int k = map_zone(o[2] + bz, g.n[2], g.bc[2]);
            // fewer than 2^31 zones
            atomicAdd(A.dep + 4 * (size_t)(unsigned)(i + g.n[0] * (j + g.n[1] * k)) + (t & 3), (unsigned long long)v[r]);
        }
    }
    const unsigned mv = __reduce_max_sync(FULL, __float_as_uint(moved));
    const unsigned nr = __reduce_add_sync(FULL, (unsigned)nremoved);
    if (lane == 0) {
        if (mv) atomicMax(&A.status[ST_MAXMOVE], mv);
        if (nr) atomicAdd(reinterpret_cast<unsigned long long *>(&A.status[ST_REMOVED_LO]), (unsigned long long)nr);
    }
}

template <int GEOM, int MODE, int TX, int TY, int TZ, bool PRED, int VAR>
__global__ void __launch_bounds__(kCubeThreads, 2)
cube_kernel(const __grid_constant__ TiledArgs<float> TA, const int parts)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    cube_tile<GEOM, MODE, TX, TY, TZ, PRED, VAR>(TA, blockIdx.x / parts, blockIdx.x % parts, parts, smem_raw);
    if (!PRED) cube_move_removed(TA);
}

using CubeKernel = void (*)(TiledArgs<float>, int);

// The copy for the 8^3 tile and the store's columns.
template <int GEOM, bool PRED>
CubeKernel cube_pick(const TiledArgs<float> &a)
{
    if constexpr (!PRED) {
        const bool sp = a.s.s.species != nullptr, par = a.s.s.param != nullptr;
        if (a.perm && a.emit_keys && !(sp && par))
            return sp ? cube_kernel<GEOM, 1, 8, 8, 8, false, CUBE_FULL | CUBE_SPECIES>
                      : (par ? cube_kernel<GEOM, 1, 8, 8, 8, false, CUBE_FULL | CUBE_PARAM>
                             : cube_kernel<GEOM, 1, 8, 8, 8, false, CUBE_FULL>);
    }
    return cube_kernel<GEOM, 1, 8, 8, 8, PRED, 0>;
}

template <int GEOM, int MODE, bool PRED>
cudaError_t launch_cube(const TiledArgs<float> &a, cudaStream_t s)
{
    const GridDev &g = a.s.g;
    const int64_t ntiles = (int64_t)g.nt[0] * g.nt[1] * g.nt[2];
    const size_t smem = cube_smem_bytes(g);
    CubeKernel kern = cube_kernel<GEOM, MODE, 0, 0, 0, PRED, 0>;
    if constexpr (MODE == 1)
        if (slab_shape_id(g, 0, a.tsc, MODE) == SHAPE_8C) kern = cube_pick<GEOM, PRED>(a);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int parts = tile_parts(ntiles, a.s.s.n, g.tvol, 13.0, 0.014, 0.022);
    kern<<<(unsigned)(ntiles * parts), kCubeThreads, smem, s>>>(a, parts);
    return cudaGetLastError();
}

}  // namespace dust
