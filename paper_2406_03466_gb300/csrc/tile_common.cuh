// Device helpers shared by the tile-pass kernels (register stages in
// hbm.cu, tensor-core blocks in tc.cu): asynchronous tile copies, the walk
// over (slot, tile) pairs, per-thread address vectors and the packed stage
// records of a pass descriptor.
#pragma once
#include <cuda_runtime.h>

#include <type_traits>

#include "engine.cuh"

namespace svk {
namespace {

// ------------------------------------------------------------ tile passes
//
// A block owns one contiguous range of (slot, tile) pairs.  Tiles arrive by
// cp.async in one of two buffers, so the next tile is in flight while the
// current one is computed.  Every register stage loads the thread's 2^R
// amplitudes from shared memory, applies the fused 2x2 group of each of its
// register bits (at most one per bit) and stores them back in place.  The
// pass descriptor is a __grid_constant__ parameter: its stage vectors are
// read with warp-uniform indices through the constant cache.  Each thread
// computes its per-stage address bases once per launch.

__device__ __forceinline__ void cp_async_amp(uint32_t sdst, const float2 *g) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(sdst), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_async_amp(uint32_t sdst, const double2 *g) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sdst), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }
// Waits for all but the most recently committed group.
__device__ __forceinline__ void cp_async_wait_prior() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// Offsets of this thread's amplitudes (tile-local index tid + k 2^(t-R))
// through the per-bit vector table v: returns the tid part and fills the
// parts of the R register bits.
template <int R>
__device__ __forceinline__ uint32_t bit_vectors(const uint32_t *v, int t, int tid,
                                                uint32_t (&k)[R]) {
    const int tb = t - R;
    uint32_t g = 0;
    for (int b = 0; b < tb; ++b)
        if ((tid >> b) & 1) g ^= v[b];
#pragma unroll
    for (int j = 0; j < R; ++j) k[j] = v[tb + j];
    return g;
}

// Block blk's contiguous share [t0, t_end) of `tiles` (slot, tile) pairs.
__device__ __forceinline__ void block_range(int64_t tiles, int nblk, int blk, int64_t &t0,
                                            int64_t &t_end) {
    const int64_t per = (tiles + nblk - 1) / nblk;
    t0 = per * blk;
    t_end = min(tiles, t0 + per);
}

// Position of one tile in the walk over (slot, tile): global offset of the
// tile's first amplitude within its state.
// fix: the fixed tile-number bits of the slot's reference (sparse passes).
struct TileCursor {
    int slot;
    uint32_t local, base, fix;
};
__device__ __forceinline__ uint32_t fixed_bits(const int64_t *refs, uint32_t fixed, int slot) {
    return fixed ? (uint32_t)refs[2 * (int64_t)slot] & fixed : 0u;
}

__device__ __forceinline__ TileCursor tile_cursor(const TilePass &P, int64_t tix,
                                                  const int64_t *refs = nullptr,
                                                  uint32_t fixed = 0) {
    TileCursor c;
    c.slot = (int)(tix >> P.n_tile_bits);
    c.local = (uint32_t)(tix & ((int64_t(1) << P.n_tile_bits) - 1));
    c.base = 0;
    for (int k = 0; k < P.n_tile_bits; ++k)
        if ((c.local >> k) & 1u) c.base ^= P.gpre[k] ^ (k ? P.gpre[k - 1] : 0u);
    c.fix = fixed_bits(refs, fixed, c.slot);
    c.base ^= c.fix;
    return c;
}

// Next tile: counting up flips tile-number bits 0..ctz(local + 1) (past the
// last slot: not used).
__device__ __forceinline__ TileCursor tile_next(const TilePass &P, TileCursor c,
                                                const int64_t *refs = nullptr,
                                                uint32_t fixed = 0, int n_slots = 0) {
    ++c.local;
    if ((c.local >> P.n_tile_bits) != 0u) {
        c.local = 0;
        ++c.slot;
        if (fixed && c.slot < n_slots) c.fix = fixed_bits(refs, fixed, c.slot);
        c.base = c.fix;
    } else {
        c.base ^= P.gpre[__ffs((int)c.local) - 1];
    }
    return c;
}

// Shared-memory record of one stage (32 bytes, read with warp-uniform
// addresses): word 0 holds one op byte per register bit, (u + 1) | real << 6
// | parametrised << 7 for pass-local op u (0: no op); word 1 + i holds
// ldq[i] | stq[i] << 16 (byte offsets, < 2^16 for every supported tile);
// word 5 holds the ops' fmode bytes; word 7 bits 16-19: M when the stage runs
// in split form (below), with ops on register bits 0..M-1.
template <bool kSplit>
__device__ __forceinline__ void build_stage_recs(const TilePass &P, uint4 *rec) {
    for (int s = threadIdx.x; s < P.n_stages; s += blockDim.x) {
        const TileStage &sg = P.st[s];
        uint32_t w[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        for (int i = 0; i < P.R && i < 4; ++i) {
            const int u = sg.op[i];
            if (u >= 0) {
                const uint32_t ob = (uint32_t)(u + 1) | (((P.real_mask >> u) & 1ull) ? 64u : 0u) |
                                    (((P.param_mask >> u) & 1ull) ? 128u : 0u);
                w[0] |= ob << (8 * i);
            }
            w[1 + i] = sg.ldq[i] | (sg.stq[i] << 16);
            if (u >= 0) w[5] |= (uint32_t)(P.fmode[u] & 3) << (8 * i);
        }
        int m = 0;
        bool all_real = true;
        for (; m < P.R && m < 4 && sg.op[m] >= 0; ++m)
            all_real = all_real && ((P.real_mask >> sg.op[m]) & 1ull);
        if (kSplit && m >= 2 && !all_real && (m == 4 || (w[0] >> (8 * m)) == 0u))
            w[7] = (uint32_t)m << 16;
        rec[2 * s] = make_uint4(w[0], w[1], w[2], w[3]);
        rec[2 * s + 1] = make_uint4(w[4], w[5], w[6], w[7]);
    }
}

template <int R>
__device__ __forceinline__ uint32_t read_stage_rec(const uint4 *rec, int s, uint32_t (&lq)[R],
                                                   uint32_t (&sq)[R]) {
    static_assert(R <= 4, "stage records hold four register bits");
    const uint4 a = rec[2 * s];
    uint32_t w[4] = {a.y, a.z, a.w, 0u};
    if constexpr (R > 3) w[3] = rec[2 * s + 1].x;
#pragma unroll
    for (int j = 0; j < R; ++j) {
        lq[j] = w[j] & 0xffffu;
        sq[j] = w[j] >> 16;
    }
    return a.x;
}

// Whether some stage has ops and does not run in split form.
__device__ __forceinline__ bool has_plain_stage(int n_stages, const uint4 *rec) {
    bool plain = false;
    for (int s = 0; s < n_stages; ++s) plain = plain || (rec[2 * s].x && !(rec[2 * s + 1].w >> 16));
    return plain;
}

// The four entries of matrix u (32-byte aligned records) as two 16-byte loads.
__device__ __forceinline__ void load_mat(const float2 *sm, int u, float2 &m0, float2 &m1,
                                         float2 &m2, float2 &m3) {
    const float4 *p = reinterpret_cast<const float4 *>(sm) + 2 * u;
    const float4 x = p[0], y = p[1];
    m0 = make_float2(x.x, x.y);
    m1 = make_float2(x.z, x.w);
    m2 = make_float2(y.x, y.y);
    m3 = make_float2(y.z, y.w);
}
__device__ __forceinline__ void load_mat(const double2 *sm, int u, double2 &m0, double2 &m1,
                                         double2 &m2, double2 &m3) {
    m0 = sm[4 * u];
    m1 = sm[4 * u + 1];
    m2 = sm[4 * u + 2];
    m3 = sm[4 * u + 3];
}

// A real rotation [[c, -s], [s, c]] with c > 0 (|angle| < pi/2) as three
// shears: x += alpha y; y += beta x; x += alpha y, with alpha = -s / (1 + c)
// = -tan(angle / 2) and beta = s (both in [-1, 1]): three fused
// multiply-adds per amplitude pair and component instead of four.
// alpha and beta are given per component: the same value twice for a complex
// amplitude, two circuits' values for a pair of real states (kPair).
template <typename C, int R, int I>
__device__ __forceinline__ void rot3_bit(C (&a)[1 << R], const C alpha, const C beta) {
    if constexpr (std::is_same<C, float2>::value) {
        const uint64_t pa = f2of(alpha), pb = f2of(beta);
#pragma unroll
        for (int r = 0; r < (1 << R); ++r) {
            if (r & (1 << I)) continue;
            uint64_t x = f2of(a[r]), y = f2of(a[r | (1 << I)]);
            x = f2fma(pa, y, x);
            y = f2fma(pb, x, y);
            x = f2fma(pa, y, x);
            a[r] = f2unpack(x);
            a[r | (1 << I)] = f2unpack(y);
        }
    } else {
#pragma unroll
        for (int r = 0; r < (1 << R); ++r) {
            if (r & (1 << I)) continue;
            C x = a[r], y = a[r | (1 << I)];
            x.x = fmaR(alpha.x, y.x, x.x);
            x.y = fmaR(alpha.y, y.y, x.y);
            y.x = fmaR(beta.x, x.x, y.x);
            y.y = fmaR(beta.y, x.y, y.y);
            x.x = fmaR(alpha.x, y.x, x.x);
            x.y = fmaR(alpha.y, y.y, x.y);
            a[r] = x;
            a[r | (1 << I)] = y;
        }
    }
}
template <typename C, typename Real> __device__ __forceinline__ C both(Real v) {
    C c;
    c.x = c.y = v;
    return c;
}

// Real 2x2 matrices of a pair of real states (component = state) on register
// bit I.
template <typename C, int R, int I>
__device__ __forceinline__ void u1p_bit(C (&a)[1 << R], const C m0, const C m1, const C m2,
                                        const C m3) {
#pragma unroll
    for (int r = 0; r < (1 << R); ++r) {
        if (r & (1 << I)) continue;
        const C x = a[r], y = a[r | (1 << I)];
        if constexpr (std::is_same<C, float2>::value) {
            a[r] = f2unpack(f2fma(f2of(m0), f2of(x), f2mul(f2of(m1), f2of(y))));
            a[r | (1 << I)] = f2unpack(f2fma(f2of(m2), f2of(x), f2mul(f2of(m3), f2of(y))));
        } else {
            a[r].x = fmaR(m0.x, x.x, m1.x * y.x);
            a[r].y = fmaR(m0.y, x.y, m1.y * y.y);
            a[r | (1 << I)].x = fmaR(m2.x, x.x, m3.x * y.x);
            a[r | (1 << I)].y = fmaR(m2.y, x.y, m3.y * y.y);
        }
    }
}

// What a pass's staged matrices are.  kAny: complex or real per group.
// kReal: every group real.  kPair: the amplitude's components are the real
// amplitudes of two circuits and entry k of a matrix is (first circuit's,
// second circuit's).  kNoSplit: kAny whose stages all keep matrices.
enum MatKind { kAny = 0, kReal = 1, kPair = 2, kNoSplit = 3 };

// The imaginary parts of a staged real matrix are unused: for a real
// rotation with c > 0 they carry the shear form (m0.y = alpha, m1.y = beta,
// m2.y = 1); otherwise m2.y = 0.  Called once per staged matrix.
template <typename C>
__device__ __forceinline__ void stage_shears(C *m) {
    using Real = decltype(m[0].x);
    const Real c = m[0].x, s = m[2].x;
    const bool rot = m[3].x == c && m[1].x == -s && c > (Real)0;
    m[0].y = rot ? -s / ((Real)1 + c) : (Real)0;
    m[1].y = rot ? s : (Real)0;
    m[2].y = rot ? (Real)1 : (Real)0;
    m[3].y = (Real)0;
}

// A pair of real states' rotations come as m0 = alpha, m1 = beta, m2 = m3 =
// 0 (k_group_mats), which no orthogonal matrix has.
template <typename C> __device__ __forceinline__ bool is_shear_pair(const C m2, const C m3) {
    return m2.x == 0 && m3.x == 0;
}

// Matrix (m0..m3) of an op on register bit I, by what the pass stages; real:
// the op's own flag (kAny).
template <typename C, int R, int I, int kMat>
__device__ __forceinline__ void op_bit(bool real, const C m0, const C m1, const C m2, const C m3,
                                       C (&a)[1 << R]) {
    if constexpr (kMat == kPair) {
        if (is_shear_pair(m2, m3)) rot3_bit<C, R, I>(a, m0, m1);
        else u1p_bit<C, R, I>(a, m0, m1, m2, m3);
    } else if (kMat == kReal || real) {
        if (m2.y != 0) rot3_bit<C, R, I>(a, both<C>(m0.y), both<C>(m1.y));
        else u1r_bit<C, decltype(m0.x), R, I>(a, m0.x, m1.x, m2.x, m3.x);
    } else {
        u1_bit<C, R, I>(a, m0, m1, m2, m3);
    }
}

// (alpha, beta) of op u's shear form.
template <typename C, int kMat>
__device__ __forceinline__ void load_shear(const C *sm, int u, C &alpha, C &beta) {
    if constexpr (kMat == kPair) {
        if constexpr (std::is_same<C, float2>::value) {
            const float4 v = reinterpret_cast<const float4 *>(sm)[2 * u];
            alpha = make_float2(v.x, v.y);
            beta = make_float2(v.z, v.w);
        } else {
            alpha = sm[4 * u];
            beta = sm[4 * u + 1];
        }
    } else {
        C m0, m1, m2, m3;
        load_mat(sm, u, m0, m1, m2, m3);
        alpha = both<C>(m0.y);
        beta = both<C>(m1.y);
    }
}

// The group ops of one stage (op bytes `ops`), register bits I..R-1 in order.
template <typename C, int R, int I, int kMat>
__device__ __forceinline__ void tile_ops_fwd(uint32_t ops, const C *sm, C (&a)[1 << R]) {
    if constexpr (I < R) {
        const uint32_t ob = (ops >> (8 * I)) & 0xffu;
        if (ob) {
            C m0, m1, m2, m3;
            load_mat(sm, (int)(ob & 63u) - 1, m0, m1, m2, m3);
            op_bit<C, R, I, kMat>((ob & 64u) != 0, m0, m1, m2, m3, a);
        }
        tile_ops_fwd<C, R, I + 1, kMat>(ops, sm, a);
    }
}

// The forward stage ops when register bits 0..M-1 carry real rotations in
// shear form and the others carry no op (stage flags): the arithmetic of
// tile_ops_fwd without its per-op branches, so the compiler can overlap one
// op's dependent FMA chains with the next op's.
template <typename C, int R, int I, int M, int kMat>
__device__ __forceinline__ void tile_ops_fwd_rot(uint32_t ops, const C *sm, C (&a)[1 << R]) {
    if constexpr (I < M) {
        C alpha, beta;
        load_shear<C, kMat>(sm, (int)((ops >> (8 * I)) & 63u) - 1, alpha, beta);
        rot3_bit<C, R, I>(a, alpha, beta);
        tile_ops_fwd_rot<C, R, I + 1, M, kMat>(ops, sm, a);
    }
}

// ------------------------------------------------------------ split form
//
// Every 2x2 unitary is diag(p0, p1) R diag(1, q) with a real rotation R of
// c, s >= 0 and unit phases p0, p1, q.  A stage with complex groups on M >= 2
// register bits multiplies its amplitudes once by the product of the groups'
// q (a table over the M register bits), applies the M rotations as shears,
// and multiplies once by the product of the p: per amplitude 4 + 1.5 M + 4
// instructions instead of 8 M for M complex 2x2 products.  With M = 1 the
// products cost less.

// The split form of a group's matrix u (FP64): out = (alpha, beta), p0, p1, q
// with the rotation's shears alpha = -s / (1 + c), beta = s.  The larger of
// c and s fixes q, so nothing is divided by a small number.
__device__ __forceinline__ void split_form(const double2 (&u)[4], double2 *out) {
    const double c = sqrt(u[0].x * u[0].x + u[0].y * u[0].y);
    const double s = sqrt(u[2].x * u[2].x + u[2].y * u[2].y);
    double2 p0 = make_double2(1.0, 0.0), p1 = p0, q;
    if (c > 1e-30) p0 = make_double2(u[0].x / c, u[0].y / c);
    if (s > 1e-30) p1 = make_double2(u[2].x / s, u[2].y / s);
    if (c >= s) q = cmul(u[3], cconj(p1));                          // u11 = p1 c q
    else q = cmul(make_double2(-u[1].x, -u[1].y), cconj(p0));       // u01 = -p0 s q
    const double l = sqrt(q.x * q.x + q.y * q.y);
    out[0] = make_double2(-s / (1.0 + c), s);
    out[1] = p0;
    out[2] = p1;
    out[3] = make_double2(q.x / l, q.y / l);
}

// a * p in two products and two fused multiply-adds.
template <typename C> __device__ __forceinline__ C phase_mul(const C a, const C p) {
    C r;
    r.x = fmaR(a.x, p.x, -(a.y * p.y));
    r.y = fmaR(a.x, p.y, a.y * p.x);
    return r;
}

// Table entries 2q and 2q + 1 (a table starts on 16 bytes).
__device__ __forceinline__ void load_phases(const float2 *tab, int q, float2 &p, float2 &n) {
    const float4 v = reinterpret_cast<const float4 *>(tab)[q];
    p = make_float2(v.x, v.y);
    n = make_float2(v.z, v.w);
}
__device__ __forceinline__ void load_phases(const double2 *tab, int q, double2 &p, double2 &n) {
    p = tab[2 * q];
    n = tab[2 * q + 1];
}

// a[r] *= tab[r mod 2^M]; kFirst: entry 0 is 1.
template <typename C, int R, int M, bool kFirst>
__device__ __forceinline__ void apply_phases(const C *tab, C (&a)[1 << R]) {
#pragma unroll
    for (int q = 0; q < (1 << M) / 2; ++q) {
        C p, n;
        load_phases(tab, q, p, n);
#pragma unroll
        for (int r = 0; r < (1 << R); r += 1 << M) {
            if (!kFirst || q) a[r + 2 * q] = phase_mul(a[r + 2 * q], p);
            a[r + 2 * q + 1] = phase_mul(a[r + 2 * q + 1], n);
        }
    }
}

// (alpha, beta) of a staged split form.
template <typename C>
__device__ __forceinline__ void split_shears(const C *sm, uint32_t ops, int i, C &alpha, C &beta) {
    const C v = sm[4 * ((int)((ops >> (8 * i)) & 63u) - 1)];
    alpha = both<C>(v.x);
    beta = both<C>(v.y);
}

template <typename C, int R, int I, int M>
__device__ __forceinline__ void split_rots(uint32_t ops, const C *sm, C (&a)[1 << R]) {
    if constexpr (I < M) {
        C alpha, beta;
        split_shears(sm, ops, I, alpha, beta);
        rot3_bit<C, R, I>(a, alpha, beta);
        split_rots<C, R, I + 1, M>(ops, sm, a);
    }
}

// A forward stage in split form with groups on register bits 0..M-1.
template <typename C, int R, int M>
__device__ __forceinline__ void split_fwd(uint32_t ops, const C *sm, const C *tab,
                                          C (&a)[1 << R]) {
    apply_phases<C, R, M, true>(tab, a);
    split_rots<C, R, 0, M>(ops, sm, a);
    apply_phases<C, R, M, false>(tab + (1 << R), a);
}

// Stage flags, the w word of a stage's second record, set for the staged
// matrices of the current slot.  Bits 0-3: M > 0 when register bits
// 0..M-1 carry ops with real matrices in shear form (rotations with c > 0)
// and the other bits none (the forward's branch-free path); bits 4-7: the
// same M when those ops are moreover parametrised with the single Ry sum
// (fmode 1; the reverse's); 0 otherwise.  Called by every thread once the
// slot's shear forms are in shared memory; visible after the next barrier.
// kPair: every op is real and its parameters all rotate about Y.
template <typename C, int kMat>
__device__ __forceinline__ void set_stage_flags(const TilePass &P, uint4 *rec, const C *sm) {
    for (int s = threadIdx.x; s < P.n_stages; s += blockDim.x) {
        const uint32_t ops = rec[2 * s].x, modes = rec[2 * s + 1].y;
        int m = 0;
        bool single = true, rot = !(rec[2 * s + 1].w >> 16);  // no shears in split form
        for (int i = 0; i < P.R; ++i) {
            const uint32_t ob = (ops >> (8 * i)) & 0xffu;
            if (!ob) break;
            const C *mt = sm + 4 * ((int)(ob & 63u) - 1);
            rot = rot && (ob & 64u) && (kMat == kPair ? is_shear_pair(mt[2], mt[3]) : mt[2].y != 0);
            if (rot) {
                single = single && (ob & 128u) && (kMat == kPair || ((modes >> (8 * i)) & 3u) == 1u);
                m = i + 1;
            }
        }
        // the bits above M must carry no op
        if (m > 0 && m < 4 && (ops >> (8 * m)) != 0u) m = 0;
        rec[2 * s + 1].w =
            (rec[2 * s + 1].w & 0xf0000u) | (uint32_t)m | (single ? (uint32_t)m << 4 : 0u);
    }
}

// Partial sum over the lanes of NV values x[0..NV-1] (NV = 8 or 16):
// afterwards x[m] (m < NV / 4) holds value 4 m + (lane & 3) summed over the
// four lanes that differ in lane bits 0-1 (a reduce-scatter of two levels;
// the kept half follows the lane bit).
template <typename Real, int NV>
__device__ __forceinline__ void warp_reduce_quad(Real (&x)[NV], int lane) {
    constexpr unsigned full = 0xffffffffu;
#pragma unroll
    for (int j = 0, M = NV; j < 2; ++j, M >>= 1) {
        const bool b = (lane >> j) & 1;
#pragma unroll
        for (int m = 0; m < M / 2; ++m) {
            const Real keep = b ? x[2 * m + 1] : x[2 * m], give = b ? x[2 * m] : x[2 * m + 1];
            x[m] = keep + __shfl_xor_sync(full, give, 1 << j);
        }
    }
}

// Sums of a split stage's group on register bit I at the point after its
// rotation, before its phases p (a phase per group only turns K_01, and the
// other groups' phases drop out), of psi = a and m = i lambda:
//   k[0] = k0 - k1 = sum p0 . m0 - p1 . m1,  k[1] = k2 = sum p0 . m1 + p1 . m0,
//   k[2] = k3 = sum Re(p0 conj l1) - Re(p1 conj l0)
// (x . y as real 2-vectors; with i lambda in place of lambda the first two
// are packed products).  k0 + k1 is of no account to a rotation's derivative.
template <typename C, typename Real, int R, int I>
__device__ __forceinline__ void split_sums(const C (&a)[1 << R], const C (&m)[1 << R], Real *k) {
    if constexpr (std::is_same<C, float2>::value) {
        uint64_t d0 = 0, d1 = 0, e0 = 0, e1 = 0;
        float t0 = 0.f, t1 = 0.f;
#pragma unroll
        for (int r = 0; r < (1 << R); ++r) {
            if (r & (1 << I)) continue;
            const C p0 = a[r], p1 = a[r | (1 << I)], m0 = m[r], m1 = m[r | (1 << I)];
            d0 = f2fma(f2of(p0), f2of(m0), d0);
            d1 = f2fma(f2of(p1), f2of(m1), d1);
            e0 = f2fma(f2of(p0), f2of(m1), e0);
            e1 = f2fma(f2of(p1), f2of(m0), e1);
            t0 = fmaR(p0.x, m1.y, fmaR(-p0.y, m1.x, t0));
            t1 = fmaR(p1.y, m0.x, fmaR(-p1.x, m0.y, t1));
        }
        const float2 D0 = f2unpack(d0), D1 = f2unpack(d1), E0 = f2unpack(e0), E1 = f2unpack(e1);
        k[0] = (D0.x + D0.y) - (D1.x + D1.y);
        k[1] = (E0.x + E0.y) + (E1.x + E1.y);
        k[2] = t0 + t1;
    } else {
        Real d = 0, e = 0, t = 0;
#pragma unroll
        for (int r = 0; r < (1 << R); ++r) {
            if (r & (1 << I)) continue;
            const C p0 = a[r], p1 = a[r | (1 << I)], m0 = m[r], m1 = m[r | (1 << I)];
            d = fmaR(p0.x, m0.x, fmaR(p0.y, m0.y, fmaR(-p1.x, m1.x, fmaR(-p1.y, m1.y, d))));
            e = fmaR(p0.x, m1.x, fmaR(p0.y, m1.y, fmaR(p1.x, m0.x, fmaR(p1.y, m0.y, e))));
            t = fmaR(p0.x, m1.y, fmaR(-p0.y, m1.x, fmaR(p1.y, m0.x, fmaR(-p1.x, m0.y, t))));
        }
        k[0] = d;
        k[1] = e;
        k[2] = t;
    }
}

// x[m] (m < 3) = value 4 m + (lane & 3) of the twelve, summed over the four
// lanes that differ in lane bits 0-1 (warp_reduce_quad of twelve values).
template <typename Real>
__device__ __forceinline__ void warp_reduce_quad12(Real (&x)[12], int lane) {
    constexpr unsigned full = 0xffffffffu;
#pragma unroll
    for (int j = 0, M = 12; j < 2; ++j, M >>= 1) {
        const bool b = (lane >> j) & 1;
#pragma unroll
        for (int m = 0; m < M / 2; ++m) {
            const Real keep = b ? x[2 * m + 1] : x[2 * m], give = b ? x[2 * m] : x[2 * m + 1];
            x[m] = keep + __shfl_xor_sync(full, give, 1 << j);
        }
    }
}

// Every op of pass P has a real matrix.
__host__ __device__ inline bool pass_all_real(const TilePass &P) {
    const uint64_t all = P.n_ops >= 64 ? ~0ull : ((1ull << P.n_ops) - 1ull);
    return (P.real_mask & all) == all;
}

}  // namespace
}  // namespace svk
