// Tile passes over states in device memory (states too large for one
// block's shared memory: 14..30 qubits).
//
// A circuit is cut into passes (planner: plan_passes).  In a pass every block
// loads tiles of 2^t amplitudes whose non-local index bits are fixed, runs
// the pass's register stages on the tile in shared memory (the same stage
// engine as the on-chip kernels, with tile-local qubit positions), and
// stores the tile back in place.  The lowest qubits are always local, so
// every load and store moves whole 128-byte segments.  Blocks are persistent:
// each walks (slot, tile) pairs with a grid stride.
//
// Kernels: per-slot fused group matrices, |ref> initialisation, forward
// pass, reverse (adjoint) pass with per-group reduced matrices accumulated
// per block and added to global FP64 sums, <H> and lambda = H psi over whole
// states, and the per-slot gradient assembly.
#include <cuda_runtime.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <type_traits>
#include <utility>
#include <vector>

#include "engine.cuh"
#include "hbm.h"
#include "tile_common.cuh"

namespace svk {
namespace {

// Real circuits in pairs: a circuit whose groups are all real, started from
// a basis state, keeps real amplitudes, so one array of complex amplitudes
// carries the states of two circuit slots, slot 2j in the real parts and slot
// 2j + 1 in the imaginary parts (an odd last slot is paired with itself).
// Every pass then moves and multiplies half as much per circuit; the matrices
// stay per circuit (packed FMAs take one per component).

// Group matrices of complex64 problems need more than FP32 (a matrix entry's
// rounding acts on a whole state) but not FP64 to the last bit, and GB300 does
// 2 FP64 multiply-adds a clock and SM: sines by argument reduction to a table
// of step pi / 64 and a short Taylor polynomial in the remainder (Tang's
// table-driven method, ACM TOMS 15(2), 1989), inverse roots by one Newton
// step from the FP32 ones.  Errors below 1e-10; with the library's
// FP64 functions the kernel took 15-20 us where this takes 4.
__device__ const double kSinTab[33] = {  // sin(j pi / 64)
    0.0, 0.049067674327418015, 0.0980171403295606, 0.14673047445536175,
    0.19509032201612828, 0.2429801799032639, 0.2902846772544624, 0.33688985339222005,
    0.3826834323650898, 0.4275550934302821, 0.47139673682599764, 0.5141027441932218,
    0.5555702330196022, 0.5956993044924334, 0.6343932841636455, 0.6715589548470184,
    0.7071067811865476, 0.7409511253549591, 0.773010453362737, 0.8032075314806449,
    0.8314696123025452, 0.8577286100002721, 0.881921264348355, 0.9039892931234433,
    0.9238795325112867, 0.9415440651830208, 0.9569403357322088, 0.970031253194544,
    0.9807852804032304, 0.989176509964781, 0.9951847266721969, 0.9987954562051724,
    1.0};

__device__ __forceinline__ void quick_sincos(double h, double *s, double *c) {
    if (!(fabs(h) < 1e6)) {
        sincos(h, s, c);
        return;
    }
    const double kf = rint(h * 20.371832715762604);
    const double r = fma(kf, -1.9135106236677394e-18, fma(kf, -0.04908738521234052, h));
    const int k = (int)kf & 127, j = k & 31;
    const double sj = __ldg(kSinTab + j), cj = __ldg(kSinTab + 32 - j);
    const double S = (k & 32) ? cj : sj, C = (k & 32) ? -sj : cj;
    const float rf = (float)r, z = rf * rf;
    const double sr = r + (double)(rf * z * (-1.f / 6.f + z * (1.f / 120.f)));  // sin r
    const double cr = (double)(z * (-0.5f + z * (1.f / 24.f)));                 // cos r - 1
    const double sn = S + fma(S, cr, C * sr), cs = C + fma(C, cr, -S * sr);
    *s = (k & 64) ? -sn : sn;
    *c = (k & 64) ? -cs : cs;
}

__device__ __forceinline__ double quick_rsqrt(double x) {
    const double y = (double)rsqrtf((float)x);
    return y * fma(-0.5 * x * y, y, 1.5);
}
// sqrt of x >= 0 (NaN below).
__device__ __forceinline__ double quick_sqrt(double x) {
    return x < 1e-30 && x >= 0.0 ? 0.0 : x * quick_rsqrt(x);
}

// Axis (M_RX, M_RY, M_RZ) and half-angle sine and cosine of one member, or
// M_X, M_H.
__device__ int quick_member(const Member &mb, const SlotInfo &si, double &s, double &c) {
    if (mb.kind <= M_RZ) {
        double t = mb.angle;
        if (mb.param >= 0)
            t = si.theta[mb.param] + (mb.param == si.shift_param ? si.shift : 0.0);
        quick_sincos(0.5 * t, &s, &c);
        return mb.kind;
    }
    if (mb.kind == M_ENC_RY_ASIN) {  // the half angles of member_matrix
        const double x = enc_input<float>(si.x[mb.param]);
        const double h = 0.5 * (1.0 + quick_sqrt((1.0 - x) * (1.0 + x))), rh = quick_rsqrt(h);
        c = h * rh;
        s = 0.5 * x * rh;
        return M_RY;
    }
    if (mb.kind == M_ENC_RZ_ACOS_SQ) {
        const double x = enc_input<float>(si.x[mb.param]), u = x * x;
        c = quick_sqrt(0.5 * (1.0 + u));
        s = quick_sqrt(0.5 * (1.0 - u));
        return M_RZ;
    }
    s = c = mb.kind == M_H ? 0.70710678118654752440 : 1.0;
    return mb.kind;
}

// Group g's matrix as i^k [[a, -conj(b)], [b, conj(a)]]: returns k, the number
// of its X and H members (-i X and -i H have determinant 1).  L lanes (consecutive, all with the same g) share a group: each forms every
// L-th member, so a group's loads and sines are in flight together; all
// multiply them.  Called by whole warps.
template <int L>
__device__ int quick_group(const Program &p, int g, const SlotInfo &si, double2 &a, double2 &b) {
    const Group grp = p.groups[g];
    const int lane = threadIdx.x & (L - 1);
    a = make_double2(1.0, 0.0);
    b = make_double2(0.0, 0.0);
    int last = grp.m_end - grp.m_begin;  // the longest group of the warp
    for (int off = 16; off; off >>= 1) last = max(last, __shfl_xor_sync(0xffffffffu, last, off));
    int turns = 0;
    for (int m0 = 0; m0 < last; m0 += L) {
        double ms = 0.0, mc = 1.0;
        int ax = M_RZ;  // past the end: the identity
        if (grp.m_begin + m0 + lane < grp.m_end)
            ax = quick_member(p.members[grp.m_begin + m0 + lane], si, ms, mc);
#pragma unroll
        for (int l = 0; l < L; ++l) {
            const int axis = L > 1 ? __shfl_sync(0xffffffffu, ax, l, L) : ax;
            const double s = L > 1 ? __shfl_sync(0xffffffffu, ms, l, L) : ms;
            const double c = L > 1 ? __shfl_sync(0xffffffffu, mc, l, L) : mc;
            double2 na, nb;
            if (axis == M_RX) {  // (c a - i s b, c b - i s a)
                na = make_double2(fma(s, b.y, c * a.x), fma(-s, b.x, c * a.y));
                nb = make_double2(fma(s, a.y, c * b.x), fma(-s, a.x, c * b.y));
            } else if (axis == M_RY) {  // (c a - s b, c b + s a)
                na = make_double2(fma(-s, b.x, c * a.x), fma(-s, b.y, c * a.y));
                nb = make_double2(fma(s, a.x, c * b.x), fma(s, a.y, c * b.y));
            } else if (axis == M_X) {  // -i (b, a)
                na = make_double2(b.y, -b.x);
                nb = make_double2(a.y, -a.x);
                ++turns;
            } else if (axis == M_H) {  // -i s (a + b, a - b)
                na = make_double2(s * (a.y + b.y), -s * (a.x + b.x));
                nb = make_double2(s * (a.y - b.y), -s * (a.x - b.x));
                ++turns;
            } else {  // ((c - i s) a, (c + i s) b)
                na = make_double2(fma(s, a.y, c * a.x), fma(-s, a.x, c * a.y));
                nb = make_double2(fma(-s, b.y, c * b.x), fma(s, b.x, c * b.y));
            }
            a = na;
            b = nb;
        }
    }
    return turns;
}

// i^k v.
__device__ __forceinline__ double2 turn(double2 v, int k) {
    if (k & 2) v = make_double2(-v.x, -v.y);
    return (k & 1) ? make_double2(-v.y, v.x) : v;
}

// split_form of i^k [[a, -conj(b)], [b, conj(a)]]: with a = c pa and b = s pb
// there p0 = i^k pa, p1 = i^k pb and q = conj(pa pb).
__device__ __forceinline__ void quick_split(double2 a, double2 b, int k, double2 *out) {
    const double c2 = fma(a.x, a.x, a.y * a.y), s2 = fma(b.x, b.x, b.y * b.y);
    double2 pa = make_double2(1.0, 0.0), pb = pa;
    double c = 0.0, s = 0.0;
    if (!(c2 < 1e-30)) {
        const double r = quick_rsqrt(c2);
        c = c2 * r;
        pa = make_double2(a.x * r, a.y * r);
    }
    if (!(s2 < 1e-30)) {
        const double r = quick_rsqrt(s2);
        s = s2 * r;
        pb = make_double2(b.x * r, b.y * r);
    }
    const double d = 1.0 + c, y = (double)(1.f / (float)d);  // 1 / d by one Newton step
    out[0] = make_double2(-s * (y * fma(-d, y, 2.0)), s);
    out[1] = turn(pa, k);
    out[2] = turn(pb, k);
    out[3] = cconj(cmul(pa, pb));
}

// (c, s) of a group of Y rotations and Ry encodings, exactly (complex128);
// false for any other member.
__device__ bool y_group(const Program &p, int g, const SlotInfo &si, double2 &cs) {
    const Group grp = p.groups[g];
    cs = make_double2(1.0, 0.0);
    for (int m = grp.m_begin; m < grp.m_end; ++m) {
        const int kind = p.members[m].kind;
        if (kind != M_RY && kind != M_ENC_RY_ASIN) return false;
        double2 r[4];
        member_matrix<double, double2>(p.members[m], si, r);
        const double c = r[0].x, s = r[2].x;
        cs = make_double2(fma(cs.x, c, -cs.y * s), fma(cs.x, s, cs.y * c));
    }
    return true;
}

// What the passes read of every state's groups (hbm.h: GroupBuf): the fused
// 2x2 matrices and, without pair, their split forms; with pair entry k is
// (first slot's, second slot's), and where both matrices are rotations their
// shears alpha, beta stand in entries 0 and 1 (zeros in 2 and 3).  Formed in
// FP64 and rounded once, so that a pass's error is its own.  A pair's real
// rotations are taken with c >= 0 (a state's sign is of no account to its
// energy and its gradient).
// kind: 0 complex, 1 pair, 2 one real slot per state (both components the
// slot's).  y_only: every group is Y rotations and encodings, whose shears are
// formed whatever their values are: the on-chip engine reads no other form,
// and a slot whose matrix is NaN (an encoded input outside [-1, 1]) must leave
// the other slot of its pair alone.  L lanes per group (complex64).
template <typename Real, int L>
__global__ void __launch_bounds__(32)
k_group_mats(Program p, SlotSource src, int kind, bool y_only, typename CT<Real>::T *out,
             double2 *split, int64_t *refs, ClearList clear) {
    using C = typename CT<Real>::T;
    constexpr bool kQuick = std::is_same<Real, float>::value;
    pdl_trigger();
    pdl_wait();
    const bool pair = kind == 1;
    const int G = p.n_groups, n_states = pair ? (src.n_slots + 1) / 2 : src.n_slots;
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t b = tid; b < 2 * n_states; b += step)
        refs[b] = resolve(src, pair ? min((int)b, src.n_slots - 1) : (int)b >> 1).ref;
    for (int k = 0; k < 3; ++k)
        for (int64_t x = tid; x < clear.n[k]; x += step) clear.p[k][x] = 0.0;
    const int64_t total = (int64_t)n_states * G;
    // whole warps: the quick groups shuffle
    for (int64_t x = tid; (x & ~31ll) < total * L; x += step) {
        const int64_t i = min(x / L, total - 1);
        const int b = (int)(i / G), g = (int)(i % G);
        double2 d[4], u, v;
        C m[4];
        if (kind == 0) {
            const SlotInfo si = resolve(src, b);
            if (kQuick) {
                const int k = quick_group<L>(p, g, si, u, v);
                d[0] = turn(u, k);
                d[1] = turn(make_double2(-v.x, v.y), k);
                d[2] = turn(v, k);
                d[3] = turn(cconj(u), k);
                quick_split(u, v, k, split + i * 4);
            } else {
                group_matrix<double, double2, Real>(p, g, si, d);
                split_form(d, split + i * 4);
            }
            for (int k = 0; k < 4; ++k) m[k] = cmk<C>(d[k].x, d[k].y);
        } else {
            double r[2][4];
            bool rot = true;
            for (int c = 0; c < (pair ? 2 : 1); ++c) {
                const SlotInfo si = resolve(src, pair ? min(2 * b + c, src.n_slots - 1) : b);
                if (!kQuick && y_group(p, g, si, u)) {
                    r[c][0] = r[c][3] = u.x;
                    r[c][1] = -u.y;
                    r[c][2] = u.y;
                } else if (kQuick && quick_group<L>(p, g, si, u, v) == 0) {
                    r[c][0] = r[c][3] = u.x;
                    r[c][1] = -v.x;
                    r[c][2] = v.x;
                } else {
                    group_matrix<double, double2, Real>(p, g, si, d);
                    for (int k = 0; k < 4; ++k) r[c][k] = d[k].x;
                }
                rot = y_only || (rot && r[c][0] == r[c][3] && r[c][1] == -r[c][2]);
            }
            if (!pair)
                for (int k = 0; k < 4; ++k) r[1][k] = r[0][k];
            for (int c = 0; c < 2 && rot; ++c) {
                const double sg = r[c][0] < 0.0 ? -1.0 : 1.0, s = sg * r[c][2];
                r[c][0] = -s / (1.0 + sg * r[c][0]);
                r[c][1] = s;
                r[c][2] = r[c][3] = 0.0;
            }
            for (int k = 0; k < 4; ++k) m[k] = cmk<C>(r[0][k], r[1][k]);
        }
        if (x == i * L)  // one lane of the group writes
            for (int k = 0; k < 4; ++k) out[i * 4 + k] = m[k];
    }
}

// Phase tables of the split stages, tabs[state][stage][0][r] = product of
// the groups' q and tabs[state][stage][1][r] = product of their p over the
// stage's register bits (every: of all stages).  Products in FP64: a table entry multiplies whole
// slices of a state, so its rounding does not average out.
template <typename Real>
__global__ void k_phase_tables(Program p, int n_states, const double2 *split, int every,
                               typename CT<Real>::T *tabs) {
    pdl_trigger();
    pdl_wait();
    const int NA = 1 << p.R;
    const int64_t total = (int64_t)n_states * p.n_stages * 2 * NA;
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < total;
         x += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(x & (NA - 1)), post = (int)(x >> p.R) & 1;
        const int64_t ss = x >> (p.R + 1);
        const Stage *sg = p.stages + ss % p.n_stages;
        const double2 *e = split + ss / p.n_stages * p.n_groups * 4;
        double2 f = make_double2(1.0, 0.0);
        bool real = true;
        for (int o = sg->op_begin; o < sg->op_end; ++o) {
            const Op op = p.ops[o];
            real = real && p.groups[op.group].real;
            const int b = (r >> op.a) & 1;
            if (post) f = cmul(f, e[op.group * 4 + 1 + b]);
            else if (b) f = cmul(f, e[op.group * 4 + 3]);
        }
        if (every || (!real && sg->op_end - sg->op_begin >= 2)) tabs[x] = cmk<typename CT<Real>::T>(f.x, f.y);
    }
}

// Sets amplitude |ref_b> of every (zeroed) slot state to 1.
template <typename C>
__global__ void k_set_ref(C *states, int n, SlotSource src) {
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < src.n_slots; b += gridDim.x * blockDim.x) {
        const SlotInfo si = resolve(src, b);
        C one;
        one.x = 1;
        one.y = 0;
        states[((int64_t)b << n) + si.ref] = one;
    }
}

// One forward stage: a branch-free path when register bits 0..M-1 carry
// real rotations in shear form or the stage runs in split form (M from the
// stage flags), tile_ops_fwd otherwise.
template <typename C, int R, int kMat>
__device__ __forceinline__ void stage_ops_fwd(uint32_t ops, uint32_t flags, const C *sm,
                                              const C *tab, C (&a)[1 << R]) {
    const uint32_t m = flags & 15u;
    if constexpr (R >= 4) {
        if (m == 4) return tile_ops_fwd_rot<C, R, 0, 4, kMat>(ops, sm, a);
    }
    if constexpr (R >= 3) {
        if (m == 3) return tile_ops_fwd_rot<C, R, 0, 3, kMat>(ops, sm, a);
    }
    if (m == 2) return tile_ops_fwd_rot<C, R, 0, 2, kMat>(ops, sm, a);
    if (m == 1) return tile_ops_fwd_rot<C, R, 0, 1, kMat>(ops, sm, a);
    if constexpr (kMat == kAny) {
        const uint32_t ms = (flags >> 16) & 15u;
        if constexpr (R >= 4) {
            if (ms == 4) return split_fwd<C, R, 4>(ops, sm, tab, a);
        }
        if constexpr (R >= 3) {
            if (ms == 3) return split_fwd<C, R, 3>(ops, sm, tab, a);
        }
        if (ms == 2) return split_fwd<C, R, 2>(ops, sm, tab, a);
    }
    tile_ops_fwd<C, R, 0, kMat>(ops, sm, a);
}

// Stages slot's matrices of the pass in shared memory (the reverse's
// transposed and conjugated): (alpha, beta) and p0 conj(p1) of a split
// stage's groups and its phase tables, shear forms for real rotations
// elsewhere, and the stage flags.  Called by every thread at a slot's first
// tile, once the previous tile's stages are past their last barrier; visible
// after the next barrier.
template <typename C, int R, int kMat, bool kRev>
__device__ __forceinline__ void stage_mats(const TilePass &P, uint4 *rec, const GroupMats &gm,
                                           int slot, C *sm, C *tab) {
    constexpr int NA = 1 << R;
    const int tid = threadIdx.x, T = blockDim.x;
    const C *mats = (const C *)gm.mats + (size_t)slot * gm.G * 4;
    __syncthreads();  // the stage records (first slot)
    for (int x = tid; x < P.n_stages * R * 4; x += T) {
        const int s = x / (R * 4), i = (x >> 2) % R, e = x & 3;
        const int u = (int)((rec[2 * s].x >> (8 * i)) & 63u) - 1;
        if (u < 0) continue;
        const int g = P.grp[u];
        C d;
        if (kMat == kAny && (rec[2 * s + 1].w >> 16)) {
            if (e > 1) continue;
            const double2 *f = gm.split + ((size_t)slot * gm.G + g) * 4;
            double2 v = f[0];
            if (e == 1) v = cmul(f[1], cconj(f[2]));
            else if (kRev) v = make_double2(-v.x, -v.y);  // the inverse rotation
            d = cmk<C>(v.x, v.y);
        } else if (kRev) {
            const C *m = mats + g * 4;
            if (kMat == kPair && is_shear_pair(m[2], m[3])) {
                d = m[e];
                d.x = -d.x;
                d.y = -d.y;
            } else {
                d = m[e == 1 ? 2 : (e == 2 ? 1 : e)];
                if (kMat != kPair) d.y = -d.y;
            }
        } else {
            d = mats[g * 4 + e];
        }
        sm[4 * u + e] = d;
    }
    if constexpr (kMat == kAny) {
        const C *tabs = (const C *)gm.tabs + ((size_t)slot * gm.n_stages + gm.stage0) * 2 * NA;
        for (int x = tid; x < P.n_stages * 2 * NA; x += T)
            if (rec[2 * (x / (2 * NA)) + 1].w >> 16) tab[x] = kRev ? cconj(tabs[x]) : tabs[x];
    }
    if constexpr (kMat == kAny)  // no shears, no flags
        if (!has_plain_stage(P.n_stages, rec)) return;
    __syncthreads();
    if constexpr (kMat != kPair) {
        for (int x = tid; x < P.n_stages * R; x += T) {
            const int s = x / R;
            const uint32_t ob = (rec[2 * s].x >> (8 * (x % R))) & 0xffu;
            if ((ob & 64u) && !(kMat == kAny && (rec[2 * s + 1].w >> 16)))
                stage_shears(sm + 4 * ((int)(ob & 63u) - 1));
        }
        __syncthreads();
    }
    set_stage_flags<C, kMat>(P, rec, sm);
}

template <typename Real, int R, int kMat, bool kDep = false>
__device__ __forceinline__ void tile_fwd_body(const TilePass &P, int n, int n_slots,
                                              const GroupMats &gm,
                                              const typename CT<Real>::T *src_states,
                                              typename CT<Real>::T *states, int64_t t0,
                                              int64_t t_end, unsigned char *smem,
                                              const Sparse &sp) {
    using C = typename CT<Real>::T;
    constexpr int NA = 1 << R;
    constexpr uint32_t kBufs = 2u;
    const int tid = threadIdx.x, T = blockDim.x, t = P.t, S = P.n_stages;
    const uint32_t tbytes = (uint32_t)sizeof(C) << t;
    uint2 *tb = reinterpret_cast<uint2 *>(smem + kBufs * tbytes);
    uint4 *rec = reinterpret_cast<uint4 *>(smem + kBufs * tbytes + (uint32_t)S * T * 8u);
    C *sm = reinterpret_cast<C *>(rec + 2 * S);
    C *tab = sm + 4 * P.n_ops;  // kAny: phase tables [stage][2][NA]
    build_stage_recs<kMat == kAny>(P, rec);
    for (int s = 0; s < S; ++s) {
        const TileStage &sg = P.st[s];
        uint32_t lb = 0, sb = 0;
        for (int k = 0; k < t - R; ++k)
            if ((tid >> k) & 1) {
                lb ^= sg.ldt[k];
                sb ^= sg.stt[k];
            }
        tb[s * T + tid] = make_uint2(lb, sb);
    }
    uint32_t gk[R], pk[R], nk[R];
    const uint32_t g0 = bit_vectors<R>(P.gl, t, tid, gk);
    const uint32_t p0 = bit_vectors<R>(P.ldperm, t, tid, pk);
    const uint32_t n0 = bit_vectors<R>(P.nat, t, tid, nk);
    const uint32_t sh = (uint32_t)__cvta_generic_to_shared(smem);
    if constexpr (kDep) pdl_wait();  // the pass's descriptor work needs no memory
    if (t0 >= t_end) return;
    auto fetch = [&](const TileCursor &c, int buf) {
        const C *src = src_states + ((int64_t)c.slot << n) + c.base;
        const uint32_t d = sh + (uint32_t)buf * tbytes;
        if (sp.zero | (uint32_t)sp.init) {  // known zeros are not read
            const int64_t *rf = sp.refs + 2 * (int64_t)c.slot;
            const uint32_t ra = (uint32_t)rf[0], rb = (uint32_t)rf[1];
#pragma unroll
            for (int k = 0; k < NA; ++k) {
                const uint32_t so = p0 ^ xsel<R>(k, pk), go = g0 ^ xsel<R>(k, gk);
                C v;
                v.x = v.y = 0;
                if (sp.init) {
                    if (kMat == kPair) v.y = (c.base ^ go) == rb ? 1 : 0;
                    v.x = (c.base ^ go) == ra ? 1 : 0;
                } else if (((go ^ ra) & sp.zero) == 0u) {
                    cp_async_amp(d + so, src + go);
                    continue;
                }
                *reinterpret_cast<C *>(smem + (uint32_t)buf * tbytes + so) = v;
            }
        } else {
#pragma unroll
            for (int k = 0; k < NA; ++k) cp_async_amp(d + (p0 ^ xsel<R>(k, pk)), src + (g0 ^ xsel<R>(k, gk)));
        }
        cp_async_commit();
    };
    TileCursor cur = tile_cursor(P, t0, sp.refs, sp.fixed);
    fetch(cur, 0);
    TileCursor nxt = tile_next(P, cur, sp.refs, sp.fixed, n_slots);
    int mslot = -1;
    for (int64_t tix = t0, i = 0; tix < t_end; ++tix, ++i) {
        const int buf = (int)(i & 1);
        if (cur.slot != mslot) {  // the previous tile's stages are past their last barrier
            stage_mats<C, R, kMat, false>(P, rec, gm, cur.slot, sm, tab);
            mslot = cur.slot;
        }
        cp_async_wait_all();
        __syncthreads();
        if (tix + 1 < t_end) fetch(nxt, buf ^ 1);
        unsigned char *tile = smem + (uint32_t)buf * tbytes;
        for (int s = 0; s < S; ++s) {
            const uint2 bb = tb[s * T + tid];
            uint32_t lq[R], sq[R];
            const uint32_t ops = read_stage_rec<R>(rec, s, lq, sq);
            C a[NA];
#pragma unroll
            for (int r = 0; r < NA; ++r) a[r] = *reinterpret_cast<const C *>(tile + (bb.x ^ xsel<R>(r, lq)));
            stage_ops_fwd<C, R, kMat>(ops, rec[2 * s + 1].w, sm, tab + s * 2 * NA, a);
            __syncthreads();
#pragma unroll
            for (int r = 0; r < NA; ++r) *reinterpret_cast<C *>(tile + (bb.y ^ xsel<R>(r, sq))) = a[r];
            __syncthreads();
        }
        C *dst = states + ((int64_t)cur.slot << n) + cur.base;
#pragma unroll
        for (int k = 0; k < NA; ++k)
            dst[g0 ^ xsel<R>(k, gk)] = *reinterpret_cast<const C *>(tile + (n0 ^ xsel<R>(k, nk)));
        cur = nxt;
        nxt = tile_next(P, nxt, sp.refs, sp.fixed, n_slots);
    }
}

// src: the states the pass reads; states: where it writes them (the same
// buffer, or another one when the pass's output is also kept as a stored
// forward state).
template <typename Real, int R, int kMat>
__global__ void __launch_bounds__(256, R >= 4 ? 2 : 3)
k_tile_fwd(const __grid_constant__ TilePass P, int n, int n_slots, GroupMats gm,
           const typename CT<Real>::T *src, typename CT<Real>::T *states, Sparse sp) {
    extern __shared__ __align__(16) unsigned char smem[];
    pdl_trigger();
    int64_t t0, t_end;
    block_range((int64_t)n_slots << P.n_tile_bits, gridDim.x, blockIdx.x, t0, t_end);
    tile_fwd_body<Real, R, kMat, true>(P, n, n_slots, gm, src, states, t0, t_end, smem, sp);
}

// The derivative of a rotation exp(-i theta P / 2) inside a fused group is
// Im tr(Q rho) for a Hermitian Q, with rho_ab = sum psi_a conj(lambda_b) over
// the amplitude pairs of the group's qubit.  Only the Hermitian matrix
// K = (rho - rho^dag) / 2i enters (Im tr(Q rho) = tr(Q K)), and i K gives
// the same derivatives as rho, also after conjugation by the group's
// members.  Four sums fix K:
//   k0 = Im rho_00, k1 = Im rho_11, k2 = Im rho_01 + Im rho_10,
//   k3 = Re rho_01 - Re rho_10,
// and i K = [[i k0, (k3 + i k2) / 2], [(-k3 + i k2) / 2, i k1]].
template <typename C, typename Real, int R, int I>
__device__ __forceinline__ void kmat_bit(const C (&a)[1 << R], const C (&l)[1 << R], Real *k) {
#pragma unroll
    for (int r = 0; r < (1 << R); ++r) {
        if (r & (1 << I)) continue;
        const C p0 = a[r], p1 = a[r | (1 << I)], l0 = l[r], l1 = l[r | (1 << I)];
        k[0] = fmaR(p0.y, l0.x, fmaR(-p0.x, l0.y, k[0]));
        k[1] = fmaR(p1.y, l1.x, fmaR(-p1.x, l1.y, k[1]));
        k[2] = fmaR(p0.y, l1.x, fmaR(-p0.x, l1.y, fmaR(p1.y, l0.x, fmaR(-p1.x, l0.y, k[2]))));
        k[3] = fmaR(p0.x, l1.x, fmaR(p0.y, l1.y, fmaR(-p1.x, l0.x, fmaR(-p1.y, l0.y, k[3]))));
    }
}

// The one sum a group needs when its only rotation is its last member
// (fmode md): 1: k3 (RY), 2: k2 (RX), 3: k0 - k1 (RZ), over the pairs of
// register bit I.
template <typename C, typename Real, int R, int I>
__device__ __forceinline__ Real single_sum(const C (&a)[1 << R], const C (&l)[1 << R],
                                           uint32_t md) {
    Real v = 0;
    if (md == 1) {
        if constexpr (std::is_same<C, float2>::value) {
            // k3 = sum x0 . y1 - x1 . y0 (as real 2-vectors): packed FMA
            // chains (two per product when there are four or more pairs, so
            // that the chains are half as long), their halves added at the end
            constexpr int NC = (1 << R) >= 8 ? 2 : 1;
            uint64_t pa[NC], pb[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) pa[c] = pb[c] = 0;
            int m = 0;
#pragma unroll
            for (int r = 0; r < (1 << R); ++r) {
                if (r & (1 << I)) continue;
                pa[m % NC] = f2fma(f2of(a[r]), f2of(l[r | (1 << I)]), pa[m % NC]);
                pb[m % NC] = f2fma(f2of(a[r | (1 << I)]), f2of(l[r]), pb[m % NC]);
                ++m;
            }
            float2 A = f2unpack(pa[0]), B = f2unpack(pb[0]);
            if constexpr (NC > 1) {
                const float2 A1 = f2unpack(pa[1]), B1 = f2unpack(pb[1]);
                A.x += A1.x;
                A.y += A1.y;
                B.x += B1.x;
                B.y += B1.y;
            }
            v = (A.x + A.y) - (B.x + B.y);
        } else {
#pragma unroll
            for (int r = 0; r < (1 << R); ++r) {
                if (r & (1 << I)) continue;
                const C x0 = a[r], x1 = a[r | (1 << I)], y0 = l[r], y1 = l[r | (1 << I)];
                v = fmaR(x0.x, y1.x, fmaR(x0.y, y1.y, fmaR(-x1.x, y0.x, fmaR(-x1.y, y0.y, v))));
            }
        }
    } else if (md == 2) {
#pragma unroll
        for (int r = 0; r < (1 << R); ++r) {
            if (r & (1 << I)) continue;
            const C x0 = a[r], x1 = a[r | (1 << I)], y0 = l[r], y1 = l[r | (1 << I)];
            v = fmaR(x0.y, y1.x, fmaR(-x0.x, y1.y, fmaR(x1.y, y0.x, fmaR(-x1.x, y0.y, v))));
        }
    } else {
#pragma unroll
        for (int r = 0; r < (1 << R); ++r) {
            if (r & (1 << I)) continue;
            const C x0 = a[r], x1 = a[r | (1 << I)], y0 = l[r], y1 = l[r | (1 << I)];
            v = fmaR(x0.y, y0.x, fmaR(-x0.x, y0.y, fmaR(-x1.y, y1.x, fmaR(x1.x, y1.y, v))));
        }
    }
    return v;
}

// k3 = sum x0 y1 - x1 y0 of each of a pair's two real states (component =
// state) over the pairs of register bit I; k0..k2 vanish for real states.
template <typename C, int R, int I>
__device__ __forceinline__ C pair_sum(const C (&a)[1 << R], const C (&l)[1 << R]) {
    if constexpr (std::is_same<C, float2>::value) {
        // chains split as in single_sum
        constexpr int NC = (1 << R) >= 8 ? 2 : 1;
        uint64_t pa[NC], pb[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) pa[c] = pb[c] = 0;
        int m = 0;
#pragma unroll
        for (int r = 0; r < (1 << R); ++r) {
            if (r & (1 << I)) continue;
            pa[m % NC] = f2fma(f2of(a[r]), f2of(l[r | (1 << I)]), pa[m % NC]);
            pb[m % NC] = f2fma(f2of(a[r | (1 << I)]), f2of(l[r]), pb[m % NC]);
            ++m;
        }
        float2 A = f2unpack(pa[0]), B = f2unpack(pb[0]);
        if constexpr (NC > 1) {
            const float2 A1 = f2unpack(pa[1]), B1 = f2unpack(pb[1]);
            A.x += A1.x;
            A.y += A1.y;
            B.x += B1.x;
            B.y += B1.y;
        }
        return make_float2(A.x - B.x, A.y - B.y);
    } else {
        C v;
        v.x = v.y = 0;
#pragma unroll
        for (int r = 0; r < (1 << R); ++r) {
            if (r & (1 << I)) continue;
            const C x0 = a[r], x1 = a[r | (1 << I)], y0 = l[r], y1 = l[r | (1 << I)];
            v.x = fmaR(x0.x, y1.x, fmaR(-x1.x, y0.x, v.x));
            v.y = fmaR(x0.y, y1.y, fmaR(-x1.y, y0.y, v.y));
        }
        return v;
    }
}

// Reverse of tile_ops_fwd, register bits I, I-1, ..., 0: per op, first its
// sums (at the point after the group) into k — k0..k3 at k[4 I ..], or with
// kSingle the one sum of its fmode at k[I] — then the inverse group (sm
// holds the adjoint matrices) on psi and lambda.
// kPair: the single Ry sum of each of the two states, at k[2 I] and k[2 I + 1].
template <typename C, typename Real, int R, int I, int NV, bool kSingle, int kMat>
__device__ __forceinline__ void tile_ops_rev(uint32_t ops, uint32_t modes, const C *sm,
                                             C (&a)[1 << R], C (&al)[1 << R], Real (&k)[NV]) {
    if constexpr (I >= 0) {
        const uint32_t ob = (ops >> (8 * I)) & 0xffu;
        if (ob) {
            if (ob & 128u) {
                if constexpr (kMat == kPair) {
                    const C v = pair_sum<C, R, I>(a, al);
                    k[2 * I] = v.x;
                    k[2 * I + 1] = v.y;
                } else if constexpr (kSingle) {
                    k[I] = single_sum<C, Real, R, I>(a, al, (modes >> (8 * I)) & 3u);
                } else {
                    kmat_bit<C, Real, R, I>(a, al, &k[4 * I]);
                }
            }
            C m0, m1, m2, m3;
            load_mat(sm, (int)(ob & 63u) - 1, m0, m1, m2, m3);
            op_bit<C, R, I, kMat>((ob & 64u) != 0, m0, m1, m2, m3, a);
            op_bit<C, R, I, kMat>((ob & 64u) != 0, m0, m1, m2, m3, al);
        }
        tile_ops_rev<C, Real, R, I - 1, NV, kSingle, kMat>(ops, modes, sm, a, al, k);
    }
}

// tile_ops_rev for register bits I..0 that all carry parametrised real
// rotations in shear form with the single Ry sum (stage flags, bits 4-7):
// the same arithmetic without its per-op branches, so the compiler can
// overlap one op's dependent FMA chains with the next op's.
template <typename C, typename Real, int R, int I, int NV, int kMat>
__device__ __forceinline__ void tile_ops_rev_rot(uint32_t ops, const C *sm, C (&a)[1 << R],
                                                 C (&al)[1 << R], Real (&k)[NV]) {
    if constexpr (I >= 0) {
        if constexpr (kMat == kPair) {
            const C v = pair_sum<C, R, I>(a, al);
            k[2 * I] = v.x;
            k[2 * I + 1] = v.y;
        } else {
            k[I] = single_sum<C, Real, R, I>(a, al, 1u);
        }
        C alpha, beta;
        load_shear<C, kMat>(sm, (int)((ops >> (8 * I)) & 63u) - 1, alpha, beta);
        rot3_bit<C, R, I>(a, alpha, beta);
        rot3_bit<C, R, I>(al, alpha, beta);
        tile_ops_rev_rot<C, Real, R, I - 1, NV, kMat>(ops, sm, a, al, k);
    }
}

// One reverse stage of single-sum ops: the branch-free path when register
// bits 0..M-1 carry parametrised real rotations (M from the stage flags),
// tile_ops_rev otherwise.
template <typename C, typename Real, int R, int NV, int kMat>
__device__ __forceinline__ void stage_ops_rev(uint32_t ops, uint32_t modes, uint32_t m,
                                              const C *sm, C (&a)[1 << R], C (&al)[1 << R],
                                              Real (&k)[NV]) {
    if constexpr (R >= 4) {
        if (m == 4) return tile_ops_rev_rot<C, Real, R, 3, NV, kMat>(ops, sm, a, al, k);
    }
    if constexpr (R >= 3) {
        if (m == 3) return tile_ops_rev_rot<C, Real, R, 2, NV, kMat>(ops, sm, a, al, k);
    }
    if (m == 2) return tile_ops_rev_rot<C, Real, R, 1, NV, kMat>(ops, sm, a, al, k);
    if (m == 1) return tile_ops_rev_rot<C, Real, R, 0, NV, kMat>(ops, sm, a, al, k);
    tile_ops_rev<C, Real, R, R - 1, NV, true, kMat>(ops, modes, sm, a, al, k);
}

template <typename C, typename Real, int R, int I>
__device__ __forceinline__ void split_unrots(uint32_t ops, const C *sm, C (&a)[1 << R],
                                             C (&m)[1 << R], Real *k) {
    if constexpr (I >= 0) {
        split_sums<C, Real, R, I>(a, m, k + 3 * I);
        C alpha, beta;
        split_shears(sm, ops, I, alpha, beta);
        rot3_bit<C, R, I>(a, alpha, beta);
        rot3_bit<C, R, I>(m, alpha, beta);
        split_unrots<C, Real, R, I - 1>(ops, sm, a, m, k);
    }
}

// A reverse stage in split form with groups on register bits 0..M-1 (tab:
// conjugated): the phases p off, per group its sums and its rotation off,
// the phases q off.  In between al holds i lambda (only names and signs).
// k: three sums per register bit.
template <typename C, typename Real, int R, int M>
__device__ __forceinline__ void split_rev(uint32_t ops, const C *sm, const C *tab,
                                          C (&a)[1 << R], C (&al)[1 << R], Real *k) {
    constexpr int NA = 1 << R, NM = 1 << M;
#pragma unroll
    for (int q = 0; q < NM / 2; ++q) {
        C p[2];
        load_phases(tab + NA, q, p[0], p[1]);
#pragma unroll
        for (int r = 0; r < NA; r += NM)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int j = r + 2 * q + h;
                a[j] = phase_mul(a[j], p[h]);
                const C l = phase_mul(al[j], p[h]);
                al[j].x = -l.y;
                al[j].y = l.x;
            }
    }
    split_unrots<C, Real, R, M - 1>(ops, sm, a, al, k);
#pragma unroll
    for (int q = 0; q < NM / 2; ++q) {
        C p[2];
        load_phases(tab, q, p[0], p[1]);
#pragma unroll
        for (int r = 0; r < NA; r += NM)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int j = r + 2 * q + h;
                C l;
                l.x = al[j].y;
                l.y = -al[j].x;
                const bool one = q == 0 && h == 0;  // that entry is 1
                if (!one) a[j] = phase_mul(a[j], p[h]);
                al[j] = one ? l : phase_mul(l, p[h]);
            }
    }
}

// Adds the block's sums of slot b (FP64 over warps and lane quads), as i K
// in reduced-matrix form, to rho_g[b][group][8] and clears them.  Called by
// every thread.
// kPair: b is a slot pair; lanes of lane bit 0 = c hold the sums of slot 2b + c
// (rho_g has a row for each, also past an odd last slot).
// A split stage (rec, sm: its staged records and forms): value 3 i + c of the
// stage, i its register bit, lies in the lanes = 3 i + c mod 4; its phases
// turn the sum k3 + i k2 by p0 conj(p1).
template <typename Real, bool kSingle, int kMat, int R>
__device__ void flush_acc(const TilePass &P, Real *acc, int wps, double *rho_g, int b, int G,
                          const uint4 *rec, const typename CT<Real>::T *sm) {
    __syncthreads();
    if constexpr (kMat == kAny && !kSingle) {
        // four threads a group, one per sum (whole warps: they exchange them)
        const int items = P.n_stages * R * 4;
        for (int x = threadIdx.x; (x & ~31) < items; x += blockDim.x) {
            const int y = min(x, items - 1), s = y / (4 * R), i = (y >> 2) % R, c = y & 3;
            const uint32_t ob = (rec[2 * s].x >> (8 * i)) & 0xffu;
            const bool on = x < items && (rec[2 * s + 1].w >> 16) && (ob & 128u);
            const int u = max(0, (int)(ob & 63u) - 1);
            double k = 0.0;
            if (on && c < 3)
                for (int w = 0; w < wps; ++w) {
                    Real *r = acc + (u * wps + w) * 32 + ((3 * i + c) & 3);
                    double ka = 0.0, kb = 0.0;
#pragma unroll
                    for (int q = 0; q < 32; q += 8) {
                        ka += (double)r[q];
                        kb += (double)r[q + 4];
                        r[q] = r[q + 4] = 0;
                    }
                    k += ka + kb;
                }
            const double k1 = __shfl_sync(0xffffffffu, k, 1, 4), k2 = __shfl_sync(0xffffffffu, k, 2, 4);
            if (!on || c > 2) continue;
            const double fx = sm[4 * u + 1].x, fy = sm[4 * u + 1].y;  // p0 conj(p1)
            // i K = [[i (k0 - k1) / 2, z], [-conj(z), -i (k0 - k1) / 2]]
            double *dst = rho_g + ((size_t)b * G + P.grp[u]) * 8;
            if (c == 0) {
                atomicAdd(dst + 1, 0.5 * k);
                atomicAdd(dst + 7, -0.5 * k);
            } else if (c == 1) {
                const double re = 0.5 * (fx * k2 - fy * k1);
                atomicAdd(dst + 2, re);
                atomicAdd(dst + 4, -re);
            } else {
                const double im = 0.5 * (fx * k1 + fy * k2);
                atomicAdd(dst + 3, im);
                atomicAdd(dst + 5, im);
            }
        }
        __syncthreads();
        if (!has_plain_stage(P.n_stages, rec)) return;
    }
    if constexpr (kMat == kPair) {
        for (int x = threadIdx.x; x < P.n_ops * 2; x += blockDim.x) {
            const int u = x >> 1, c = x & 1;
            if (!((P.param_mask >> u) & 1ull)) continue;
            double k = 0.0;
            for (int w = 0; w < wps; ++w) {
                Real *r = acc + (u * wps + w) * 32 + c;
                double ka = 0.0, kb = 0.0;
#pragma unroll
                for (int q = 0; q < 32; q += 4) {
                    ka += (double)r[q];
                    kb += (double)r[q + 2];
                    r[q] = r[q + 2] = 0;
                }
                k += ka + kb;
            }
            if (k == 0.0) continue;
            double *dst = rho_g + ((size_t)(2 * b + c) * G + P.grp[u]) * 8;
            atomicAdd(dst + 2, 0.5 * k);
            atomicAdd(dst + 4, -0.5 * k);
        }
        __syncthreads();
        return;
    }
    for (int x = threadIdx.x; x < P.n_ops * 4; x += blockDim.x) {
        const int u = x >> 2;
        if (!((P.param_mask >> u) & 1ull)) continue;
        // kSingle: one sum per op in all lanes, stored as the component of
        // its fmode; otherwise lane q holds component q & 3.
        const int c = kSingle ? (P.fmode[u] == 1 ? 3 : (P.fmode[u] == 2 ? 2 : 0)) : (x & 3);
        if (kSingle && (x & 3)) continue;
        double k = 0.0;
        for (int w = 0; w < wps; ++w)
            for (int q = kSingle ? 0 : c; q < 32; q += kSingle ? 1 : 4) {
                Real &r = acc[(u * wps + w) * 32 + q];
                k += (double)r;
                r = 0;
            }
        if (k == 0.0) continue;
        // i K = [[i k0, (k3 + i k2) / 2], [(-k3 + i k2) / 2, i k1]]
        double *dst = rho_g + ((size_t)b * G + P.grp[u]) * 8;
        if (c == 0) {
            atomicAdd(dst + 1, k);
        } else if (c == 1) {
            atomicAdd(dst + 7, k);
        } else if (c == 2) {
            atomicAdd(dst + 3, 0.5 * k);
            atomicAdd(dst + 5, 0.5 * k);
        } else {
            atomicAdd(dst + 2, 0.5 * k);
            atomicAdd(dst + 4, -0.5 * k);
        }
    }
    __syncthreads();
}

// One reverse pass: un-applies the pass on psi and lambda tiles and sums the
// reduced matrices of its parametrised groups (as i K) into
// rho_g[slot][group][8].  The sums run in the state's precision over one
// warp and at most 64 tiles, then in FP64.
template <typename Real, int R, bool kSingle, int kMat, int NB = 2, bool kDep = false>
__device__ __forceinline__ void tile_rev_body(const TilePass &P, int n, int n_slots,
                                              const GroupMats &gm,
                                              const typename CT<Real>::T *psi_src,
                                              typename CT<Real>::T *psi, typename CT<Real>::T *lam,
                                              double *rho_g, int64_t t0, int64_t t_end,
                                              unsigned char *smem, const int64_t *refs,
                                              uint32_t fixed, bool write_psi = true) {
    using C = typename CT<Real>::T;
    constexpr int NA = 1 << R;
    constexpr int kFlushTiles = 64;
    const int G = gm.G;
    const int tid = threadIdx.x, T = blockDim.x, t = P.t, S = P.n_stages;
    const int lane = tid & 31, wps = T >> 5;
    const uint32_t tbytes = (uint32_t)sizeof(C) << t;
    // NB tile buffers (2: the next tile's copy overlaps this one's stages;
    // 1: more blocks per SM, the copy after the tile is written back)
    uint2 *tb = reinterpret_cast<uint2 *>(smem + 2 * NB * tbytes);
    uint4 *rec = reinterpret_cast<uint4 *>(smem + 2 * NB * tbytes + (uint32_t)S * T * 8u);
    C *sm = reinterpret_cast<C *>(rec + 2 * S);
    constexpr bool kSplit = kMat == kAny && !kSingle;
    C *tab = sm + 4 * P.n_ops;  // kSplit: phase tables [stage][2][NA]
    Real *acc = reinterpret_cast<Real *>(tab + (kSplit ? S * 2 * NA : 0));
    build_stage_recs<kSplit>(P, rec);
    for (int s = 0; s < S; ++s) {
        const TileStage &sg = P.st[s];
        uint32_t lb = 0, sb = 0;
        for (int k = 0; k < t - R; ++k)
            if ((tid >> k) & 1) {
                lb ^= sg.ldt[k];
                sb ^= sg.stt[k];
            }
        tb[s * T + tid] = make_uint2(lb, sb);
    }
    for (int x = tid; x < P.n_ops * wps * 32; x += T) acc[x] = 0;
    Real *accw = acc + (tid >> 5) * 32 + lane;  // [op][warp][lane]: sum k_(lane & 3)
    uint32_t gk[R], pk[R], nk[R];
    const uint32_t g0 = bit_vectors<R>(P.gl, t, tid, gk);
    const uint32_t p0 = bit_vectors<R>(P.ldperm, t, tid, pk);
    const uint32_t n0 = bit_vectors<R>(P.nat, t, tid, nk);
    const uint32_t sh = (uint32_t)__cvta_generic_to_shared(smem);
    if constexpr (kDep) pdl_wait();
    if (t0 >= t_end) return;
    // psi tile of buffer j at [j tbytes], lambda tile at [(NB + j) tbytes]
    auto fetch = [&](const TileCursor &c, int buf) {
        const int64_t off = ((int64_t)c.slot << n) + c.base;
        const C *sp = psi_src + off, *sl = lam + off;
        const uint32_t dp = sh + (uint32_t)buf * tbytes, dl = dp + NB * tbytes;
#pragma unroll
        for (int k = 0; k < NA; ++k) {
            const uint32_t so = n0 ^ xsel<R>(k, nk), go = g0 ^ xsel<R>(k, gk);
            cp_async_amp(dp + so, sp + go);
            cp_async_amp(dl + so, sl + go);
        }
        cp_async_commit();
    };
    TileCursor cur = tile_cursor(P, t0, refs, fixed);
    fetch(cur, 0);
    TileCursor nxt = tile_next(P, cur, refs, fixed, n_slots);
    int mslot = -1, since = 0;
    for (int64_t tix = t0, i = 0; tix < t_end; ++tix, ++i) {
        const int buf = NB == 2 ? (int)(i & 1) : 0;
        if (cur.slot != mslot || since == kFlushTiles) {
            if (mslot >= 0) flush_acc<Real, kSingle, kMat, R>(P, acc, wps, rho_g, mslot, G, rec, sm);
            since = 0;
        }
        if (cur.slot != mslot) {  // adjoint matrices of this slot's groups
            stage_mats<C, R, kSplit || kMat != kAny ? kMat : kNoSplit, true>(P, rec, gm, cur.slot, sm,
                                                                            tab);
            mslot = cur.slot;
        }
        cp_async_wait_all();
        __syncthreads();
        if (NB == 2 && tix + 1 < t_end) fetch(nxt, buf ^ 1);
        unsigned char *tp = smem + (uint32_t)buf * tbytes, *tl = tp + NB * tbytes;
        for (int s = S - 1; s >= 0; --s) {
            const uint2 bb = tb[s * T + tid];
            uint32_t lq[R], sq[R];
            const uint32_t ops = read_stage_rec<R>(rec, s, lq, sq);
            const uint32_t modes = kSingle ? rec[2 * s + 1].y : 0u;
            C a[NA], al[NA];
#pragma unroll
            for (int r = 0; r < NA; ++r) {
                const uint32_t ad = bb.y ^ xsel<R>(r, sq);
                a[r] = *reinterpret_cast<const C *>(tp + ad);
                al[r] = *reinterpret_cast<const C *>(tl + ad);
            }
            // the stage's sums: over lane quads in registers, then per lane
            // into the warp's accumulators
            constexpr int NV = kMat == kPair ? (R <= 2 ? 4 : 8) : kSingle ? 4 : (4 * R <= 8 ? 8 : 16);
            Real kk[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) kk[v] = 0;
            bool split = false;
            if constexpr (kSingle && kMat != kAny && std::is_same<C, float2>::value) {
                stage_ops_rev<C, Real, R, NV, kMat>(ops, modes, (rec[2 * s + 1].w >> 4) & 15u, sm, a,
                                                     al, kk);
            } else {
                if constexpr (kSplit) {
                    const uint32_t ms = (rec[2 * s + 1].w >> 16) & 15u;
                    if (ms) {
                        Real k3[12];
#pragma unroll
                        for (int v = 0; v < 12; ++v) k3[v] = 0;
                        const C *ts = tab + s * 2 * NA;
                        if constexpr (R >= 4) {
                            if (ms == 4) split_rev<C, Real, R, 4>(ops, sm, ts, a, al, k3);
                        }
                        if constexpr (R >= 3) {
                            if (ms == 3) split_rev<C, Real, R, 3>(ops, sm, ts, a, al, k3);
                        }
                        if (ms == 2) split_rev<C, Real, R, 2>(ops, sm, ts, a, al, k3);
                        warp_reduce_quad12<Real>(k3, lane);
#pragma unroll
                        for (int m = 0; m < 3; ++m) {
                            const int i = (4 * m + (lane & 3)) / 3;
                            const uint32_t ob = (ops >> (8 * i)) & 0xffu;
                            if (ob & 128u) accw[((int)(ob & 63u) - 1) * wps * 32] += k3[m];
                        }
                    } else {
                        tile_ops_rev<C, Real, R, R - 1, NV, kSingle, kMat>(ops, modes, sm, a, al, kk);
                    }
                    split = ms != 0;
                } else {
                    tile_ops_rev<C, Real, R, R - 1, NV, kSingle, kMat>(ops, modes, sm, a, al, kk);
                }
            }
            if (!split) {
                warp_reduce_quad<Real, NV>(kk, lane);
                if constexpr (kMat == kPair) {  // lane: bit 2 m + (lane >> 1 & 1), state lane & 1
#pragma unroll
                    for (int m = 0; m < NV / 4; ++m) {
                        const int i = 2 * m + ((lane >> 1) & 1);
                        const uint32_t ob = i < R ? (ops >> (8 * i)) & 0xffu : 0u;
                        if (ob & 128u) accw[((int)(ob & 63u) - 1) * wps * 32] += kk[m];
                    }
                } else if constexpr (kSingle) {  // lane: the sum of register bit lane & 3
                    const int m = lane & 3;
                    const uint32_t ob = m < R ? (ops >> (8 * m)) & 0xffu : 0u;
                    if (ob & 128u) accw[((int)(ob & 63u) - 1) * wps * 32] += kk[0];
                } else {
#pragma unroll
                    for (int m = 0; m < R; ++m) {
                        const uint32_t ob = (ops >> (8 * m)) & 0xffu;
                        if (ob & 128u) accw[((int)(ob & 63u) - 1) * wps * 32] += kk[m];
                    }
                }
            }
            __syncthreads();
#pragma unroll
            for (int r = 0; r < NA; ++r) {
                const uint32_t ad = bb.x ^ xsel<R>(r, lq);
                *reinterpret_cast<C *>(tp + ad) = a[r];
                *reinterpret_cast<C *>(tl + ad) = al[r];
            }
            __syncthreads();
        }
        const int64_t off = ((int64_t)cur.slot << n) + cur.base;
        C *dp = psi + off, *dl = lam + off;
        if (write_psi) {
#pragma unroll
            for (int k = 0; k < NA; ++k) {
                const uint32_t so = p0 ^ xsel<R>(k, pk), go = g0 ^ xsel<R>(k, gk);
                dp[go] = *reinterpret_cast<const C *>(tp + so);
                dl[go] = *reinterpret_cast<const C *>(tl + so);
            }
        } else {  // the next reverse pass restarts psi from a stored state
#pragma unroll
            for (int k = 0; k < NA; ++k) {
                const uint32_t so = p0 ^ xsel<R>(k, pk), go = g0 ^ xsel<R>(k, gk);
                dl[go] = *reinterpret_cast<const C *>(tl + so);
            }
        }
        ++since;
        if (NB == 1 && tix + 1 < t_end) {
            __syncthreads();  // every thread has read its part of the tile
            fetch(nxt, 0);
        }
        cur = nxt;
        nxt = tile_next(P, nxt, refs, fixed, n_slots);
    }
    flush_acc<Real, kSingle, kMat, R>(P, acc, wps, rho_g, mslot, G, rec, sm);
}

// NB = 1: launched with 64 threads only (at least five blocks per SM).
template <typename Real, int R, bool kSingle, int kMat, int NB = 2>
__global__ void __launch_bounds__(NB == 1 ? 64 : 256, NB == 1 ? 5 : (R >= 4 ? 1 : 2))
k_tile_rev(const __grid_constant__ TilePass P, int n, int n_slots, GroupMats gm,
           const typename CT<Real>::T *psi_src,
           typename CT<Real>::T *psi, typename CT<Real>::T *lam, double *rho_g, Sparse sp,
           int write_psi) {
    extern __shared__ __align__(16) unsigned char smem[];
    pdl_trigger();
    int64_t t0, t_end;
    block_range((int64_t)n_slots << P.n_tile_bits, gridDim.x, blockIdx.x, t0, t_end);
    tile_rev_body<Real, R, kSingle, kMat, NB, true>(P, n, n_slots, gm, psi_src, psi, lam, rho_g,
                                               t0, t_end, smem, sp.refs, sp.fixed, write_psi != 0);
}

// Sum of v over the block (every thread gets it); red: one double per warp.
__device__ __forceinline__ double block_sum(double v, double *red) {
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];
    return s;
}

// ------------------------------------- several problems, one persistent launch
//
// The forward (or reverse) sweeps of several problems of any qubit count and
// depth (one tile shape) run as one launch of resident blocks.  Each pass of
// each problem is a task cut into chunks of tiles; the chunks of all tasks
// form one ticket sequence, level by level (pass 0 of every problem, then
// pass 1, ...).  A block takes the next ticket, waits until the task its
// chunk depends on (the same problem's previous pass) has completed all of
// its chunks, runs the chunk with the ordinary pass body and counts it done.
// Every ticket before a waited-on chunk was taken by a running block, so the
// wait always ends; it is bounded anyway (kSweepWaitNs of wall time), after
// which the block records SV_DEVERR_SWEEP_WAIT and stops.

constexpr unsigned long long kSweepWaitNs = 20ull * 1000 * 1000 * 1000;  // 20 s

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned int ld_acquire(const unsigned int *p) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

template <typename Real, int R, bool kRev>
__global__ void __launch_bounds__(256, (R >= 4 && kRev) ? 1 : 2)
k_tile_sweep(const SweepTask *tasks, int n_tasks, long long n_tickets,
             unsigned long long *ticket, unsigned int *done, int *err) {
    using C = typename CT<Real>::T;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ long long s_tk;
    __shared__ int s_task, s_fail;
    TilePass &P = *reinterpret_cast<TilePass *>(smem);
    unsigned char *rest = smem + ((sizeof(TilePass) + 255) & ~size_t(255));
    int hint = 0, cur = -1;
    for (;;) {
        if (threadIdx.x == 0) {
            const long long tk = (long long)atomicAdd(ticket, 1ull);
            int j = hint;
            if (tk < n_tickets)
                while (j + 1 < n_tasks && tasks[j + 1].chunk_begin <= tk) ++j;
            s_tk = tk;
            s_task = j;
            s_fail = 0;
            if (tk < n_tickets && tasks[j].dep >= 0) {
                const SweepTask &d = tasks[tasks[j].dep];
                const unsigned int need = (unsigned int)d.n_chunks;
                unsigned long long t_start = 0;
                while (ld_acquire(done + tasks[j].dep) < need) {
                    const unsigned long long now = global_ns();
                    if (!t_start) t_start = now;
                    if (now - t_start > kSweepWaitNs) {
                        s_fail = 1;
                        if (err) atomicCAS(err, 0, SV_DEVERR_SWEEP_WAIT);
                        break;
                    }
                    __nanosleep(256);
                }
            }
        }
        __syncthreads();
        const long long tk = s_tk;
        const int j = s_task;
        if (tk >= n_tickets || s_fail) break;
        hint = j;
        const SweepTask T = tasks[j];
        // every thread acquires the dependency's writes for its own loads
        if (T.dep >= 0) (void)ld_acquire(done + T.dep);
        if (j != cur) {  // this pass's descriptor into shared memory
            const uint32_t *src = reinterpret_cast<const uint32_t *>(T.P);
            uint32_t *dst = reinterpret_cast<uint32_t *>(smem);
            for (int i = threadIdx.x; i < (int)(sizeof(TilePass) / 4); i += blockDim.x) dst[i] = src[i];
            cur = j;
        }
        __syncthreads();
        const long long c = tk - T.chunk_begin;
        const int64_t t0 = c * (int64_t)T.chunk_tiles;
        const int64_t t1 = min(T.tiles, t0 + (int64_t)T.chunk_tiles);
        const GroupMats gm{T.mats, T.tabs, (const double2 *)T.split, T.G, T.n_stages, T.stage0, 0};
        if constexpr (kRev)
            tile_rev_body<Real, R, false, kAny>(P, T.n, T.n_slots, gm,
                                                 (const C *)T.psi, (C *)T.psi, (C *)T.lam, T.rho,
                                                 t0, t1, rest, T.refs, T.fixed);
        else
            tile_fwd_body<Real, R, kAny>(P, T.n, T.n_slots, gm,
                                         (const C *)T.psi, (C *)T.psi, t0, t1, rest,
                                         Sparse{T.refs, T.fixed, 0u, 0, 0});
        __syncthreads();  // every store of the chunk issued
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(done + j, 1u);
        }
    }
}

// ------------------------------------------------------ H over tile passes

// Tile walk of an H pass (the same counting as TileCursor).
__device__ __forceinline__ TileCursor h_cursor(const HPass &P, int64_t tix) {
    TileCursor c;
    c.slot = (int)(tix >> P.n_tile_bits);
    c.local = (uint32_t)(tix & ((int64_t(1) << P.n_tile_bits) - 1));
    c.base = 0;
    for (int k = 0; k < P.n_tile_bits; ++k)
        if ((c.local >> k) & 1u) c.base ^= P.gpre[k] ^ (k ? P.gpre[k - 1] : 0u);
    return c;
}

__device__ __forceinline__ TileCursor h_next(const HPass &P, TileCursor c) {
    ++c.local;
    if ((c.local >> P.n_tile_bits) != 0u) {
        c.local = 0;
        c.base = 0;
        ++c.slot;
    } else {
        c.base ^= P.gpre[__ffs((int)c.local) - 1];
    }
    return c;
}

// Per-tile record of one class of terms: its coefficient sum_t c_t i^phase_t
// times the term's sign on the tile's non-local bits and the class's sign
// on the group's flip bits, and its Z mask on the thread bits.
template <typename Real> struct HCoef {
    uint32_t zt, pad;
    Real re, im;
};

// One H pass: for the pass's X-mask groups g,
//   lambda_j (+)= sum_g D_g(j ^ x_g) psi_(j ^ x_g),
//   D_g(k) = sum_(t in g) c_t i^phase_t (-1)^|k & z_t|,
// and E[slot] += sum_j Re(conj(psi_j) lambda_j) over this pass's part of
// lambda.  psi tiles arrive by cp.async (double-buffered) in natural order;
// the thread's amplitudes are j = tid + k 2^(t-R).  A group whose classes
// put no Z on a register bit takes one value per thread (its signed class
// coefficients summed).  The others read D_g at the thread's 2^R amplitudes
// from a per-tile table: one row of 2^R values per distinct Z mask on the
// thread bits (the row's class coefficients times their register-bit signs,
// built once per tile by the whole block), each row added with the sign of
// its thread-bit mask.  Products in the state's precision, sums over the
// block's amplitudes in FP64.  kLam = false: energies only.  kPairE (with
// kRealH): each state holds the real states of slots 2 slot and 2 slot + 1,
// whose energies are summed apart (those below e_rows are written).
template <typename Real, int R, bool kLam, bool kRealH, bool kPairE>
__global__ void __launch_bounds__(256)
k_tile_h(const __grid_constant__ HPass P, int n, int n_slots, const typename CT<Real>::T *psi,
         typename CT<Real>::T *lam, double *E, int e_rows) {
    using C = typename CT<Real>::T;
    constexpr int NA = 1 << R;
    static_assert(R <= kHRegBitsMax, "H kernel register bits");
    extern __shared__ __align__(16) unsigned char smem[];
    // 256 threads whenever R >= 3 (tiles of 2^11 and 2^12 amplitudes)
    pdl_trigger();
    const int tid = threadIdx.x, T = R >= 3 ? 256 : (int)blockDim.x, t = P.t;
    const uint32_t tbytes = (uint32_t)sizeof(C) << t;
    // psi tiles at [0, 2 tbytes), the lambda tile being added to at [2 tbytes,
    // 3 tbytes), then this tile's row table (NA values per row, real parts,
    // then imaginary parts unless kRealH)
    constexpr int kRowVals = kRealH ? NA : 2 * NA;
    Real *etab = reinterpret_cast<Real *>(smem + 3 * tbytes);
    HGroup *grp = reinterpret_cast<HGroup *>(etab + P.n_rows * kRowVals);
    HCoef<Real> *coef = reinterpret_cast<HCoef<Real> *>(grp + P.n_groups);
    HTerm *trm = reinterpret_cast<HTerm *>(coef + P.n_classes);
    HClass *cls = reinterpret_cast<HClass *>(trm + P.n_terms);
    HRow *rows = reinterpret_cast<HRow *>(cls + P.n_classes);
    double *red = reinterpret_cast<double *>(rows + P.n_rows);
    for (int i = tid; i < P.n_terms; i += T) trm[i] = P.terms[i];
    for (int i = tid; i < P.n_groups; i += T) grp[i] = P.groups[i];
    for (int i = tid; i < P.n_classes; i += T) cls[i] = P.classes[i];
    for (int i = tid; i < P.n_rows; i += T) rows[i] = P.rows[i];
    __syncthreads();
    const bool add = kLam && !P.first;
    uint32_t gk[R];
    const uint32_t g0 = bit_vectors<R>(P.gl, t, tid, gk);
    const uint32_t sh = (uint32_t)__cvta_generic_to_shared(smem);
    const int64_t tiles = (int64_t)n_slots << P.n_tile_bits;
    const int64_t per = (tiles + gridDim.x - 1) / gridDim.x;
    const int64_t t0 = per * blockIdx.x, t_end = min(tiles, t0 + per);
    pdl_wait();  // the plan's arrays are older than the stream's work
    if (t0 >= t_end) return;
    auto fetch = [&](const TileCursor &c, int buf) {
        const C *src = psi + ((int64_t)c.slot << n) + c.base;
        const uint32_t d = sh + (uint32_t)buf * tbytes;
#pragma unroll
        for (int k = 0; k < NA; ++k)
            cp_async_amp(d + (uint32_t)(tid + k * T) * (uint32_t)sizeof(C), src + (g0 ^ xsel<R>(k, gk)));
        cp_async_commit();
    };
    TileCursor cur = h_cursor(P, t0);
    fetch(cur, 0);
    TileCursor nxt = h_next(P, cur);
    double e_acc = 0.0, e_acc2 = 0.0;
    int eslot = cur.slot;
    auto add_energy = [&]() {  // the slot's energy so far
        const double s = block_sum(e_acc, red);
        if constexpr (kPairE) {
            const double s2 = block_sum(e_acc2, red);
            if (tid == 0) atomicAdd(&E[2 * eslot], s);
            if (tid == 0 && 2 * eslot + 1 < e_rows) atomicAdd(&E[2 * eslot + 1], s2);
        } else {
            if (tid == 0) atomicAdd(&E[eslot], s);
        }
        e_acc = e_acc2 = 0.0;
    };
    for (int64_t tix = t0, i = 0; tix < t_end; ++tix, ++i) {
        const int buf = (int)(i & 1);
        if (cur.slot != eslot) {
            add_energy();
            eslot = cur.slot;
        }
        for (int c = tid; c < P.n_classes; c += T) {  // this tile's class records
            const HClass cl = cls[c];
            Real re = 0, im = 0;
            for (int ti = cl.t_begin; ti < cl.t_end; ++ti) {
                const HTerm tm = trm[ti];
                const Real v =
                    (__popc((cur.base ^ cl.xnl) & tm.z) & 1u) ? (Real)-tm.coeff : (Real)tm.coeff;
                if (tm.phase == 0) re += v;
                else if (tm.phase == 1) im += v;
                else if (tm.phase == 2) re -= v;
                else im -= v;
            }
            if (__popc(cl.xl & cl.zl) & 1u) {
                re = -re;
                im = -im;
            }
            HCoef<Real> h;
            h.zt = cl.zl & (uint32_t)(T - 1);
            h.pad = 0;
            h.re = re;
            h.im = im;
            coef[c] = h;
        }
        if (P.n_rows) {  // the row table: E[k] = sum_c coef_c (-1)^|k & kz_c|
            __syncthreads();
            for (int x = tid; x < P.n_rows * NA; x += T) {
                const HRow rw = rows[x / NA];
                const int k = x & (NA - 1);
                Real er = 0, ei = 0;
                for (int c = rw.c_begin; c < rw.c_end; ++c) {
                    const bool neg = __popc((uint32_t)k & (cls[c].zl >> (t - R))) & 1u;
                    er += neg ? -coef[c].re : coef[c].re;
                    if constexpr (!kRealH) ei += neg ? -coef[c].im : coef[c].im;
                }
                Real *e = etab + (x / NA) * kRowVals;
                e[k] = er;
                if constexpr (!kRealH) e[NA + k] = ei;
            }
        }
        cp_async_wait_all();
        __syncthreads();
        C *L = lam + ((int64_t)cur.slot << n) + cur.base;
        C *lt = reinterpret_cast<C *>(smem + 2 * tbytes);
        if (add) {  // this tile's lambda so far, in flight during the sums
            const uint32_t d = sh + 2 * tbytes;
#pragma unroll
            for (int k = 0; k < NA; ++k)
                cp_async_amp(d + (uint32_t)(tid + k * T) * (uint32_t)sizeof(C), L + (g0 ^ xsel<R>(k, gk)));
            cp_async_commit();
        }
        if (tix + 1 < t_end) fetch(nxt, buf ^ 1);
        else cp_async_commit();  // keeps "all but the newest group" meaning the lambda tile
        const C *tile = reinterpret_cast<const C *>(smem + (uint32_t)buf * tbytes);
        const C *Sg = psi + ((int64_t)cur.slot << n);
        // lambda_k = acc[k] (real part .x, imaginary part .y)
        C acc[NA];
#pragma unroll
        for (int k = 0; k < NA; ++k) acc[k].x = acc[k].y = 0;
        auto add_real = [&](int k, Real d, const C &pk) {
            acc[k].x = fmaR(d, pk.x, acc[k].x);
            acc[k].y = fmaR(d, pk.y, acc[k].y);
        };
        // byte offset in shared memory of partner j ^ x (j = tid + k T) is
        // gb ^ (k T sizeof(C)): thread and register bits are disjoint, and
        // the buffer offset is above every in-tile offset
        const uint32_t bufb = (uint32_t)buf * tbytes;
        for (int g = 0; g < P.n_groups; ++g) {
            const HGroup &gr = grp[g];
            const uint32_t xl = gr.xl, xfar = gr.xfar, kact = gr.kact;
            const uint32_t gb = ((uint32_t)(tid ^ (int)xl) * (uint32_t)sizeof(C)) ^ bufb;
            auto partner = [&](int k) -> C {
                return xfar ? Sg[(cur.base ^ g0 ^ xsel<R>(k, gk)) ^ xfar]
                            : *reinterpret_cast<const C *>(
                                  smem + (gb ^ ((uint32_t)(k * T) * (uint32_t)sizeof(C))));
            };
            if (kact == 0) {
                // no class has a Z on a register bit: one value per thread
                Real vr = 0, vi = 0;
                for (int c = gr.c_begin; c < gr.c_end; ++c) {
                    const HCoef<Real> h = coef[c];
                    const bool nt = __popc((uint32_t)tid & h.zt) & 1u;
                    vr += nt ? -h.re : h.re;
                    if constexpr (!kRealH) vi += nt ? -h.im : h.im;
                }
                if constexpr (kRealH && std::is_same<C, float2>::value) {
                    // one packed FP32-pair FMA per amplitude
                    const uint64_t d2 = f2pack(vr, vr);
#pragma unroll
                    for (int k = 0; k < NA; ++k) acc[k] = f2unpack(f2fma(d2, f2of(partner(k)), f2of(acc[k])));
                } else {
#pragma unroll
                    for (int k = 0; k < NA; ++k) {
                        const C pk = partner(k);
                        if constexpr (kRealH) {
                            add_real(k, vr, pk);
                        } else {
                            acc[k].x = fmaR(vr, pk.x, fmaR(-vi, pk.y, acc[k].x));
                            acc[k].y = fmaR(vr, pk.y, fmaR(vi, pk.x, acc[k].y));
                        }
                    }
                }
                continue;
            }
            // D(tid, k) = sum over the group's rows of (-1)^|tid & zt| E_row[k]
            Real vr[NA], vi[NA];
#pragma unroll
            for (int k = 0; k < NA; ++k) vr[k] = vi[k] = 0;
            for (int r = gr.r_begin; r < gr.r_end; ++r) {
                const Real sg = (__popc((uint32_t)tid & rows[r].zt) & 1u) ? (Real)-1 : (Real)1;
                const Real *e = etab + r * kRowVals;
#pragma unroll
                for (int k = 0; k < NA; ++k) {
                    vr[k] = fmaR(sg, e[k], vr[k]);
                    if constexpr (!kRealH) vi[k] = fmaR(sg, e[NA + k], vi[k]);
                }
            }
#pragma unroll
            for (int k = 0; k < NA; ++k) {
                const C pk = partner(k);
                if constexpr (kRealH) {
                    add_real(k, vr[k], pk);
                } else {
                    acc[k].x = fmaR(vr[k], pk.x, fmaR(-vi[k], pk.y, acc[k].x));
                    acc[k].y = fmaR(vr[k], pk.y, fmaR(vi[k], pk.x, acc[k].y));
                }
            }
        }
        if (add) cp_async_wait_prior();  // own copies of the lambda tile have landed
        Real part = 0, part2 = 0;
#pragma unroll
        for (int k = 0; k < NA; ++k) {
            const C pj = tile[tid + k * T];
            if constexpr (kPairE) {
                part = fmaR(pj.x, acc[k].x, part);
                part2 = fmaR(pj.y, acc[k].y, part2);
            } else {
                part = fmaR(pj.x, acc[k].x, fmaR(pj.y, acc[k].y, part));
            }
            if constexpr (kLam) {
                const uint32_t go = g0 ^ xsel<R>(k, gk);
                C out = acc[k];
                if (add) {  // each thread reads back only its own copies
                    const C old = lt[tid + k * T];
                    out.x += old.x;
                    out.y += old.y;
                }
                L[go] = out;
            }
        }
        e_acc += (double)part;
        if constexpr (kPairE) e_acc2 += (double)part2;
        __syncthreads();  // coef and this buffer are rewritten next
        cur = nxt;
        nxt = h_next(P, nxt);
    }
    add_energy();
}

// D_g(j) = sum_{t in g} c_t i^{phase_t} (-1)^{|j & z_t|} for one amplitude.
template <typename Real>
__device__ __forceinline__ void diag_of(const Observable &o, const TermGroup &tg, uint32_t j,
                                        Real &dre, Real &dim) {
    dre = 0;
    dim = 0;
    for (int t = tg.t_begin; t < tg.t_end; ++t) {
        const Term tm = o.terms[t];
        const Real c = (__popc(j & tm.z) & 1u) ? (Real)-tm.coeff : (Real)tm.coeff;
        if (tm.phase == 0) dre += c;
        else if (tm.phase == 1) dim += c;
        else if (tm.phase == 2) dre -= c;
        else dim -= c;
    }
}


// out[b] += sum_j sum_g Re(conj(psi_{j^x_g}) psi_j D_g(j)); grid.y = slot.
// Products in the state's precision over 8 amplitudes, sums in FP64.
template <typename Real>
__global__ void k_expect_big(Observable o, int n, const typename CT<Real>::T *states, double *out) {
    using C = typename CT<Real>::T;
    __shared__ double red[32];
    const int b = blockIdx.y;
    const C *S = states + ((int64_t)b << n);
    const int64_t dim = int64_t(1) << n;
    double acc = 0.0;
    for (int64_t j0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) * 8; j0 < dim;
         j0 += (int64_t)gridDim.x * blockDim.x * 8) {
        Real part = 0;
        for (int u = 0; u < 8 && j0 + u < dim; ++u) {
            const uint32_t j = (uint32_t)(j0 + u);
            const C pj = S[j];
            for (int g = 0; g < o.n_tgroups; ++g) {
                const TermGroup tg = o.tgroups[g];
                const C px = S[j ^ tg.x];
                Real dr, di;
                diag_of<Real>(o, tg, j, dr, di);
                const Real wr = fmaR(px.x, pj.x, px.y * pj.y);
                const Real wi = fmaR(px.x, pj.y, -px.y * pj.x);
                part = fmaR(wr, dr, fmaR(-wi, di, part));
            }
        }
        acc += (double)part;
    }
    const double s = block_sum(acc, red);
    if (threadIdx.x == 0) atomicAdd(&out[b], s);
}

// lambda = H psi over whole states; E[b] += sum_j Re(conj(psi_j) lambda_j).
template <typename Real>
__global__ void k_apply_h_big(Observable o, int n, const typename CT<Real>::T *psi,
                              typename CT<Real>::T *lam, double *E) {
    using C = typename CT<Real>::T;
    __shared__ double red[32];
    const int b = blockIdx.y;
    const C *S = psi + ((int64_t)b << n);
    C *Lm = lam + ((int64_t)b << n);
    const int64_t dim = int64_t(1) << n;
    double acc = 0.0;
    for (int64_t j0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) * 8; j0 < dim;
         j0 += (int64_t)gridDim.x * blockDim.x * 8) {
        Real part = 0;
        for (int u = 0; u < 8 && j0 + u < dim; ++u) {
            const uint32_t j = (uint32_t)(j0 + u);
            C l;
            l.x = 0;
            l.y = 0;
            for (int g = 0; g < o.n_tgroups; ++g) {
                const TermGroup tg = o.tgroups[g];
                const uint32_t jx = j ^ tg.x;
                const C px = S[jx];
                Real dr, di;
                diag_of<Real>(o, tg, jx, dr, di);
                l.x = fmaR(dr, px.x, fmaR(-di, px.y, l.x));
                l.y = fmaR(dr, px.y, fmaR(di, px.x, l.y));
            }
            Lm[j] = l;
            const C pj = S[j];
            part = fmaR(pj.x, l.x, fmaR(pj.y, l.y, part));
        }
        acc += (double)part;
    }
    const double s = block_sum(acc, red);
    if (threadIdx.x == 0) atomicAdd(&E[b], s);
}

// Data-driven circuit learning (Sec. 4.2, Eq. 3): with Q(b) = |psi_b|^2 and
// the target P, M = (P + Q)/2, adds JS = 1/2 sum_b (P log(P/M) + Q log(Q/M))
// to js[slot] and writes lambda_b = w_b psi_b with w_b = dJS/dQ(b) =
// 1/2 log(Q(b)/M(b)) (0 where Q(b) = 0), so that the reverse sweep with
// lambda gives dJS/dtheta.  Per amplitude the arithmetic is in the state's
// precision (FP32 for complex64, whose states carry FP32 rounding anyway;
// FP64 for complex128); the sums over amplitudes are FP64.  grid.y = slot.
template <typename Real>
__global__ void k_ddcl_lambda(int n, const typename CT<Real>::T *psi, const double *target,
                              typename CT<Real>::T *lam, double *js) {
    using C = typename CT<Real>::T;
    __shared__ double red[32];
    const int b = blockIdx.y;
    const C *S = psi + ((int64_t)b << n);
    C *Lm = lam + ((int64_t)b << n);
    const int64_t dim = int64_t(1) << n;
    double acc = 0.0;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < dim;
         j += (int64_t)gridDim.x * blockDim.x) {
        const C a = S[j];
        const Real q = fmaR(a.x, a.x, a.y * a.y), p = (Real)target[j];
        const Real m = (Real)0.5 * (p + q);
        Real w = 0, term = 0;
        if (p > (Real)0) term = p * log(p / m);
        if (q > (Real)0) {
            const Real l = log(q / m);
            term = fmaR(q, l, term);
            w = (Real)0.5 * l;
        }
        acc += (double)term;
        C out;
        out.x = w * a.x;
        out.y = w * a.y;
        Lm[j] = out;
    }
    const double s = block_sum(acc, red);
    if (threadIdx.x == 0) atomicAdd(&js[b], 0.5 * s);
}

// Per-slot gradients from the summed reduced matrices: one thread per
// (slot, group); slot_grads[b][param] += weight_b * dE_b/dtheta.
template <typename Real>
__global__ void k_group_grads(Program p, SlotSource src, const double *rho_g, CostSource cs,
                              const double *E, double *slot_grads) {
    pdl_trigger();
    pdl_wait();
    const int G = p.n_groups, P = p.n_params;
    const int64_t total = (int64_t)src.n_slots * G;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int b = (int)(i / G), g = (int)(i % G);
        if (!p.groups[g].has_param) continue;
        const SlotInfo si = resolve(src, b);
        const double wgt = cost_weight(cs, si.instance, E[b]);
        double r8[8];
        for (int v = 0; v < 8; ++v) r8[v] = wgt * rho_g[(size_t)i * 8 + v];
        group_gradients<Real>(p, g, r8, si, slot_grads + (size_t)b * P);
    }
}

// A kernel's dynamic shared-memory limit only ever grows (per device and
// kernel), so a launch sequence that ran once has every limit it needs.
// While a sequence is captured into a CUDA graph no attribute is changed: a
// launch that would need a larger limit fails instead.
thread_local bool t_capturing = false;
std::mutex g_smem_mu;
std::map<std::pair<int, const void *>, uint32_t> g_smem_limit;

template <typename K> cudaError_t allow_smem(K kernel, uint32_t bytes);

}  // namespace

cudaError_t allow_smem_attr(const void *kernel, uint32_t bytes) { return allow_smem(kernel, bytes); }

void forget_smem_limits() {
    std::lock_guard<std::mutex> lk(g_smem_mu);
    g_smem_limit.clear();
}

namespace {

template <typename K> cudaError_t allow_smem(K kernel, uint32_t bytes) {
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(g_smem_mu);
    uint32_t &have = g_smem_limit[{dev, (const void *)kernel}];
    if (bytes <= have) return cudaSuccess;
    if (t_capturing) return cudaErrorInvalidValue;
    const cudaError_t e =
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) have = bytes;
    return e;
}

// Resident blocks of kernel k on the whole GPU (*full), at most max_blocks.  The
// occupancy of a launch shape is a constant of the device: kept per thread,
// since a call of a small state is launch after launch.
template <typename K>
int fill_blocks(K kernel, int threads, uint32_t smem, int64_t max_blocks, int *full = nullptr) {
    struct Seen {
        const void *kernel;
        int dev, threads, blocks;
        uint32_t smem;
    };
    static thread_local std::vector<Seen> seen;
    int dev = 0;
    cudaGetDevice(&dev);
    int64_t b = 0;
    for (const Seen &s : seen)
        if (s.kernel == (const void *)kernel && s.dev == dev && s.threads == threads && s.smem == smem) {
            b = s.blocks;
            break;
        }
    if (!b) {
        int sms = 0, per = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, smem) != cudaSuccess ||
            per < 1)
            per = 1;
        b = (int64_t)sms * per;
        if (seen.size() >= 256) seen.clear();
        seen.push_back({(const void *)kernel, dev, threads, (int)b, smem});
    }
    if (full) *full = (int)b;
    if (b > max_blocks) b = max_blocks;
    return b < 1 ? 1 : (int)b;
}

// Whether a pass is launched as a dependent of the one before, which hides
// its launch and its descriptor work.  Such blocks start wherever blocks of
// the pass before end, packed onto few SMs when they do not fill the GPU: no
// harm to a handful of FP32 blocks, but complex128 passes share one SM's FP64
// unit then (12 qubits, 32 instances: 1200 against 800 us), and a half-filled
// grid idles the other half.  Full grids over more than 64 MiB lose as well:
// their tiles' L2 lines are on the other die (20-qubit states, 512 MiB a
// pass: 5833 against 5482 us).
bool pass_dep(int c128, int t, int64_t n_tiles, int blocks, int full) {
    return !c128 && ((n_tiles << t) * 8) <= (int64_t(64) << 20) && (blocks <= 64 || blocks >= full);
}

int grid_1d(int64_t work, int threads) {
    int64_t b = (work + threads - 1) / threads;
    if (b > 8192) b = 8192;
    return b < 1 ? 1 : (int)b;
}

}  // namespace

// ----------------------------------------------------------- launchers

#define HBM_DISPATCH_R(c128, R_, ...)                                      \
    do {                                                                    \
        if (c128) {                                                         \
            using Real = double;                                            \
            switch (R_) {                                                   \
            case 2: { constexpr int RR = 2; __VA_ARGS__; } break;                  \
            case 3: { constexpr int RR = 3; __VA_ARGS__; } break;                  \
            default: return cudaErrorInvalidValue;                          \
            }                                                               \
        } else {                                                            \
            using Real = float;                                             \
            switch (R_) {                                                   \
            case 2: { constexpr int RR = 2; __VA_ARGS__; } break;                  \
            case 3: { constexpr int RR = 3; __VA_ARGS__; } break;                  \
            case 4: { constexpr int RR = 4; __VA_ARGS__; } break;                  \
            default: return cudaErrorInvalidValue;                          \
            }                                                               \
        }                                                                   \
    } while (0)

cudaError_t launch_group_mats(int c128, const Program &p, const SlotSource &src, void *base,
                              cudaStream_t st, int kind, const ClearList &clear, bool every) {
    const int n_states = kind == 1 ? (src.n_slots + 1) / 2 : src.n_slots;
    const GroupBuf b = group_buf(c128, p, (size_t)n_states, kind != 0);
    double2 *split = (double2 *)((char *)base + b.split);
    int64_t *refs = (int64_t *)((char *)base + b.refs);
    void *tabs = (char *)base + b.tabs;
    // Not dependent launches (pass_dep).  One warp a block: the FP64 work of a few thousand groups spreads over
    // every SM (32 slots x 190 groups: 22 us in blocks of 128 threads).  Four
    // lanes a group while that fits the SMs' schedulers in one wave: the
    // latency of a group's loads and sines counts then, not their number.
    const int64_t groups = (int64_t)n_states * std::max(1, p.n_groups);
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const bool wide = !c128 && groups * 4 <= (int64_t)sms * 4 * 32;
    const int g = grid_1d(wide ? groups * 4 : groups, 32);
    const bool y_only = every && kind != 0;  // (the on-chip engine's real kinds)
    cudaError_t e =
        c128   ? launch_dep_if(false, k_group_mats<double, 1>, g, 32, 0, st, p, src, kind, y_only, (double2 *)base, split, refs, clear)
        : wide ? launch_dep_if(false, k_group_mats<float, 4>, g, 32, 0, st, p, src, kind, y_only, (float2 *)base, split, refs, clear)
               : launch_dep_if(false, k_group_mats<float, 1>, g, 32, 0, st, p, src, kind, y_only, (float2 *)base, split, refs, clear);
    if (e == cudaSuccess && kind == 0 && p.n_stages > 0) {
        const int gt = grid_1d(((int64_t)n_states * p.n_stages * 2) << p.R, 64);
        e = c128 ? launch_dep_if(false, k_phase_tables<double>, gt, 64, 0, st, p, n_states, split, (int)every, (double2 *)tabs)
                 : launch_dep_if(false, k_phase_tables<float>, gt, 64, 0, st, p, n_states, split, (int)every, (float2 *)tabs);
    }
    return e == cudaSuccess ? cudaGetLastError() : e;
}

cudaError_t launch_init_states(int c128, void *states, int n, const SlotSource &src,
                               cudaStream_t st) {
    const size_t bytes = ((size_t)src.n_slots << n) * (c128 ? 16 : 8);
    cudaError_t e = cudaMemsetAsync(states, 0, bytes, st);
    if (e != cudaSuccess) return e;
    const int g = grid_1d(src.n_slots, 128);
    if (c128) k_set_ref<double2><<<g, 128, 0, st>>>((double2 *)states, n, src);
    else k_set_ref<float2><<<g, 128, 0, st>>>((float2 *)states, n, src);
    return cudaGetLastError();
}

Sparse sparse_pass(TilePass *P, uint32_t support, const int64_t *refs, bool init) {
    Sparse sp{};
    sp.refs = refs;
    sp.init = init;
    uint32_t prev = 0, acc = 0;
    int nt = 0;
    const int n_tile_bits = P->n_tile_bits;
    for (int k = 0; k < n_tile_bits; ++k) {
        const uint32_t bit = P->gpre[k] ^ prev;
        prev = P->gpre[k];
        if (bit & support) {
            acc ^= bit;
            P->gpre[nt++] = acc;
        } else {
            sp.fixed |= bit;
        }
    }
    P->n_tile_bits = nt;
    for (int b = 0; b < P->t; ++b) sp.zero |= P->gl[b] & ~support;
    return sp;
}

uint32_t tile_table_bytes(int c128, const TilePass &P, bool rev, bool any) {
    const bool read = any || (!pass_all_real(P) && !(rev && P.all_single));
    return read ? (uint32_t)P.n_stages * ((c128 ? 32u : 16u) << P.R) : 0u;
}

uint32_t tile_fwd_smem(int c128, const TilePass &P, bool any) {
    const uint32_t csz = c128 ? 16u : 8u, T = 1u << (P.t - P.R);
    const uint32_t tab = tile_table_bytes(c128, P, false, any);
    return 2u * (csz << P.t) + (uint32_t)P.n_stages * (T * 8u + 32u) + (uint32_t)P.n_ops * 4u * csz + tab;
}

// Reverse passes with at least this many register stages run single-buffered.
constexpr int kOneBufStages = 6;

uint32_t tile_rev_smem(int c128, const TilePass &P, int bufs, bool any) {
    const uint32_t csz = c128 ? 16u : 8u, rsz = c128 ? 8u : 4u, T = 1u << (P.t - P.R);
    const uint32_t tab = tile_table_bytes(c128, P, true, any);
    return 2u * (uint32_t)bufs * (csz << P.t) + (uint32_t)P.n_stages * (T * 8u + 32u) + (uint32_t)P.n_ops * 4u * csz +
           tab + (uint32_t)P.n_ops * T * rsz;
}

cudaError_t launch_tile_fwd(int c128, const TilePass &P, int n, int n_slots,
                            const GroupMats &gm, void *states, int64_t max_blocks, cudaStream_t st,
                            const void *src, bool pair, const Sparse &sp) {
    const uint32_t smem = tile_fwd_smem(c128, P);
    const int threads = 1 << (P.t - P.R);
    if (!src) src = states;
    HBM_DISPATCH_R(c128, P.R, {
        using C = typename CT<Real>::T;
        auto k = pair ? k_tile_fwd<Real, RR, kPair>
                      : (pass_all_real(P) ? k_tile_fwd<Real, RR, kReal> : k_tile_fwd<Real, RR, kAny>);
        cudaError_t e = allow_smem(k, smem);
        if (e != cudaSuccess) return e;
        int full = 0;
        const int blocks = fill_blocks(k, threads, smem, max_blocks, &full);
        e = launch_dep_if(pass_dep(c128, P.t, (int64_t)n_slots << P.n_tile_bits, blocks, full), k, blocks, threads,
                          smem, st, P, n, n_slots, gm, (const C *)src, (C *)states, sp);
        if (e != cudaSuccess) return e;
    });
    return cudaGetLastError();
}

cudaError_t launch_tile_rev(int c128, const TilePass &P, int n, int n_slots,
                            const GroupMats &gm, void *psi, void *lam, double *rho_g, int64_t max_blocks,
                            cudaStream_t st, const void *psi_src, bool write_psi, bool pair,
                            const Sparse &sp) {
    // passes of many stages are arithmetic-bound: one tile buffer, more
    // blocks per SM (complex64 real single-sum passes, tiles of 2^10 at 16
    // amplitudes per thread: 64 threads)
    const bool one_buf = !c128 && P.R == 4 && P.t == 10 &&
                         (pair || (P.all_single && pass_all_real(P))) &&
                         P.n_stages >= kOneBufStages;
    const uint32_t smem = tile_rev_smem(c128, P, one_buf ? 1 : 2);
    const int threads = 1 << (P.t - P.R);
    HBM_DISPATCH_R(c128, P.R, {
        using C = typename CT<Real>::T;
        auto k = pair ? k_tile_rev<Real, RR, true, kPair>
                 : P.all_single ? (pass_all_real(P) ? k_tile_rev<Real, RR, true, kReal>
                                                    : k_tile_rev<Real, RR, true, kAny>)
                                : (pass_all_real(P) ? k_tile_rev<Real, RR, false, kReal>
                                                    : k_tile_rev<Real, RR, false, kAny>);
        if constexpr (std::is_same<Real, float>::value && RR == 4) {
            if (one_buf) k = pair ? k_tile_rev<Real, RR, true, kPair, 1> : k_tile_rev<Real, RR, true, kReal, 1>;
        }
        cudaError_t e = allow_smem(k, smem);
        if (e != cudaSuccess) return e;
        int full = 0;
        const int blocks = fill_blocks(k, threads, smem, max_blocks, &full);
        e = launch_dep_if(pass_dep(c128, P.t, (int64_t)n_slots << P.n_tile_bits, blocks, full), k, blocks, threads,
                       smem, st, P, n, n_slots, gm, (const C *)(psi_src ? psi_src : psi), (C *)psi, (C *)lam, rho_g, sp,
                       write_psi ? 1 : 0);
        if (e != cudaSuccess) return e;
    });
    return cudaGetLastError();
}

cudaError_t launch_tile_h(int c128, const HPass &P, int n, int n_slots, const void *psi, void *lam,
                          double *E, int64_t max_blocks, cudaStream_t st, int pair_rows) {
    const uint32_t smem = tile_h_smem(c128, P);
    // 2^R amplitudes per thread (R = h_reg_bits(t), the planner's bucketing)
    const int R = h_reg_bits(P.t);
    const int threads = 1 << (P.t - R);
    if (P.t < 7 || P.t > 12 || P.R != R) return cudaErrorInvalidValue;
    auto go = [&](auto k, auto *psi_t, auto *lam_t) -> cudaError_t {
        cudaError_t e = allow_smem(k, smem);
        if (e != cudaSuccess) return e;
        int full = 0;
        const int blocks = fill_blocks(k, threads, smem, max_blocks, &full);
        return launch_dep_if(pass_dep(c128, P.t, (int64_t)n_slots << P.n_tile_bits, blocks, full), k, blocks,
                             threads, smem, st, P, n, n_slots, psi_t, lam_t, E, pair_rows);
    };
    auto pick2 = [&](auto rr, auto re, auto pr) -> cudaError_t {
        constexpr int RR = decltype(rr)::value;
        constexpr bool RE = decltype(re)::value, PR = decltype(pr)::value;
        if (c128) {
            if (lam) return go(k_tile_h<double, RR, true, RE, PR>, (const double2 *)psi, (double2 *)lam);
            return go(k_tile_h<double, RR, false, RE, PR>, (const double2 *)psi, (double2 *)nullptr);
        }
        if (lam) return go(k_tile_h<float, RR, true, RE, PR>, (const float2 *)psi, (float2 *)lam);
        return go(k_tile_h<float, RR, false, RE, PR>, (const float2 *)psi, (float2 *)nullptr);
    };
    auto pick = [&](auto rr) -> cudaError_t {
        if (pair_rows > 0) {
            if (!P.real) return cudaErrorInvalidValue;
            return pick2(rr, std::true_type(), std::true_type());
        }
        if (P.real) return pick2(rr, std::true_type(), std::false_type());
        return pick2(rr, std::false_type(), std::false_type());
    };
    if (R == 4) return pick(std::integral_constant<int, 4>());
    if (R == 3) return pick(std::integral_constant<int, 3>());
    return pick(std::integral_constant<int, 2>());
}

void set_capturing(bool on) { t_capturing = on; }

uint32_t tile_sweep_smem(int c128, bool rev, const TilePass &P) {
    return (uint32_t)((sizeof(TilePass) + 255) & ~size_t(255)) +
           (rev ? tile_rev_smem(c128, P, 2, true) : tile_fwd_smem(c128, P, true));
}

int tile_sweep_blocks_per_sm(int c128, int R, bool rev, uint32_t smem, int threads) {
    int per = 0;
    HBM_DISPATCH_R(c128, R, {
        cudaError_t e;
        if (rev) {
            auto k = k_tile_sweep<Real, RR, true>;
            e = allow_smem(k, smem);
            if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, threads, smem);
        } else {
            auto k = k_tile_sweep<Real, RR, false>;
            e = allow_smem(k, smem);
            if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, threads, smem);
        }
        if (e != cudaSuccess) return 0;
    });
    return per;
}

cudaError_t launch_tile_sweep(int c128, int R, bool rev, const SweepTask *tasks, int n_tasks,
                              long long n_tickets, unsigned long long *ticket, unsigned int *done,
                              int *err, int blocks, int threads, uint32_t smem, cudaStream_t st) {
    HBM_DISPATCH_R(c128, R, {
        if (rev) {
            auto k = k_tile_sweep<Real, RR, true>;
            cudaError_t e = allow_smem(k, smem);
            if (e != cudaSuccess) return e;
            k<<<blocks, threads, smem, st>>>(tasks, n_tasks, n_tickets, ticket, done, err);
        } else {
            auto k = k_tile_sweep<Real, RR, false>;
            cudaError_t e = allow_smem(k, smem);
            if (e != cudaSuccess) return e;
            k<<<blocks, threads, smem, st>>>(tasks, n_tasks, n_tickets, ticket, done, err);
        }
    });
    return cudaGetLastError();
}

static dim3 whole_state_grid(int n, int rows);

// The JS divergence of one state's output distribution from the target and
// its derivative table D[j] = dJS/dP_theta(j) = 1/2 log(P_theta(j) / M(j)),
// M = (P + P_theta) / 2 (0 where P_theta(j) = 0); per-amplitude arithmetic
// in Real, the sum in FP64 (js zeroed by the launcher).
template <typename Real>
__global__ void k_ddcl_diag(int n, const typename CT<Real>::T *psi, const double *target,
                            double *D, double *js) {
    using C = typename CT<Real>::T;
    __shared__ double red[32];
    const int64_t dim = int64_t(1) << n;
    double acc = 0.0;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < dim;
         j += (int64_t)gridDim.x * blockDim.x) {
        const C a = psi[j];
        const Real q = fmaR(a.x, a.x, a.y * a.y), p = (Real)target[j];
        const Real m = (Real)0.5 * (p + q);
        Real w = 0, term = 0;
        if (p > (Real)0) term = p * log(p / m);
        if (q > (Real)0) {
            const Real l = log(q / m);
            term = fmaR(q, l, term);
            w = (Real)0.5 * l;
        }
        acc += (double)term;
        D[j] = (double)w;
    }
    const double s = block_sum(acc, red);
    if (threadIdx.x == 0) atomicAdd(js, 0.5 * s);
}

// out[r] = sum_j D[j] |psi_r(j)|^2 for n_rows states (grid.y = row; out
// zeroed by the launcher); products in Real, sums in FP64.
template <typename Real>
__global__ void k_diag_expect(int n, const typename CT<Real>::T *states, const double *D,
                              double *out) {
    using C = typename CT<Real>::T;
    __shared__ double red[32];
    const int r = blockIdx.y;
    const C *S = states + ((int64_t)r << n);
    const int64_t dim = int64_t(1) << n;
    double acc = 0.0;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < dim;
         j += (int64_t)gridDim.x * blockDim.x) {
        const C a = S[j];
        acc += (double)((Real)D[j] * fmaR(a.x, a.x, a.y * a.y));
    }
    const double s = block_sum(acc, red);
    if (threadIdx.x == 0) atomicAdd(&out[r], s);
}

// out[j] = in[j'] where j' moves bit b of j to bit who.q[b]: a table indexed
// by qubit values rewritten in a relabeled bit layout (who.q[b] = the qubit
// held by bit b).  Grid-stride, one entry per thread step.
struct QubitOfBit {
    int32_t q[30];
};
__global__ void k_relayout(int n, QubitOfBit who, const double *in, double *out) {
    const int64_t dim = int64_t(1) << n;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < dim;
         j += (int64_t)gridDim.x * blockDim.x) {
        int64_t src = 0;
        for (int b = 0; b < n; ++b) src |= ((j >> b) & 1) << who.q[b];
        out[j] = in[src];
    }
}

cudaError_t launch_relayout(int n, const int32_t *qubit_of_bit, const double *in, double *out,
                            cudaStream_t st) {
    if (n < 1 || n > 30) return cudaErrorInvalidValue;
    QubitOfBit w{};
    for (int b = 0; b < n; ++b) w.q[b] = qubit_of_bit[b];
    const int64_t dim = int64_t(1) << n;
    const int64_t blocks = std::min<int64_t>((dim + 255) / 256, 152 * 16);
    k_relayout<<<(unsigned)blocks, 256, 0, st>>>(n, w, in, out);
    return cudaGetLastError();
}

cudaError_t launch_ddcl_diag(int c128, int n, const void *psi, const double *target, double *D,
                             double *js, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(js, 0, sizeof(double), st);
    if (e != cudaSuccess) return e;
    const dim3 g = whole_state_grid(n, 1);
    if (c128) k_ddcl_diag<double><<<g, 256, 0, st>>>(n, (const double2 *)psi, target, D, js);
    else k_ddcl_diag<float><<<g, 256, 0, st>>>(n, (const float2 *)psi, target, D, js);
    return cudaGetLastError();
}

cudaError_t launch_diag_expect(int c128, int n, int n_rows, const void *states, const double *D,
                               double *out, cudaStream_t st) {
    if (n_rows <= 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(double) * n_rows, st);
    if (e != cudaSuccess) return e;
    const dim3 g = whole_state_grid(n, n_rows);
    if (c128) k_diag_expect<double><<<g, 256, 0, st>>>(n, (const double2 *)states, D, out);
    else k_diag_expect<float><<<g, 256, 0, st>>>(n, (const float2 *)states, D, out);
    return cudaGetLastError();
}

cudaError_t launch_ddcl_lambda(int c128, int n, int n_rows, const void *psi, const double *target,
                               void *lam, double *js, cudaStream_t st) {
    if (n_rows <= 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(js, 0, sizeof(double) * n_rows, st);
    if (e != cudaSuccess) return e;
    const dim3 g = whole_state_grid(n, n_rows);
    if (c128) k_ddcl_lambda<double><<<g, 256, 0, st>>>(n, (const double2 *)psi, target, (double2 *)lam, js);
    else k_ddcl_lambda<float><<<g, 256, 0, st>>>(n, (const float2 *)psi, target, (float2 *)lam, js);
    return cudaGetLastError();
}

static dim3 whole_state_grid(int n, int rows) {
    const int64_t per = ((int64_t(1) << n) + 2047) / 2048;  // 256 threads x 8 amplitudes
    int64_t x = per;
    const int64_t cap = rows >= 1024 ? 1 : (int64_t)2048 / rows;
    if (x > cap) x = cap < 1 ? 1 : cap;
    return dim3((unsigned)x, (unsigned)rows, 1);
}

cudaError_t launch_expect_big(int c128, const Observable &o, int n, int n_rows,
                              const void *states, double *out, cudaStream_t st) {
    if (n_rows <= 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(double) * n_rows, st);
    if (e != cudaSuccess) return e;
    const dim3 g = whole_state_grid(n, n_rows);
    if (c128) k_expect_big<double><<<g, 256, 0, st>>>(o, n, (const double2 *)states, out);
    else k_expect_big<float><<<g, 256, 0, st>>>(o, n, (const float2 *)states, out);
    return cudaGetLastError();
}

cudaError_t launch_apply_h_big(int c128, const Observable &o, int n, int n_rows, const void *psi,
                               void *lam, double *E, cudaStream_t st) {
    if (n_rows <= 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(E, 0, sizeof(double) * n_rows, st);
    if (e != cudaSuccess) return e;
    const dim3 g = whole_state_grid(n, n_rows);
    if (c128) k_apply_h_big<double><<<g, 256, 0, st>>>(o, n, (const double2 *)psi, (double2 *)lam, E);
    else k_apply_h_big<float><<<g, 256, 0, st>>>(o, n, (const float2 *)psi, (float2 *)lam, E);
    return cudaGetLastError();
}

cudaError_t launch_group_grads(int c128, const Program &p, const SlotSource &src,
                               const double *rho_g, const CostSource &cs, const double *E,
                               double *slot_grads, cudaStream_t st) {
    const int g = grid_1d((int64_t)src.n_slots * p.n_groups, 128);
    return c128 ? launch_dep(k_group_grads<double>, g, 128, 0, st, p, src, rho_g, cs, E, slot_grads)
                : launch_dep(k_group_grads<float>, g, 128, 0, st, p, src, rho_g, cs, E, slot_grads);
}

}  // namespace svk
