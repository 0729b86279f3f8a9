// On-chip adjoint gradients, one state per group of 2^(n-R) threads
// (whole warps), the state in shared memory between the register
// stages.  Three kinds of state:
//   complex  any circuit of fused groups; every stage in split form (phases,
//            real rotations, phases; tile_common.cuh);
//   pair     circuits of Y rotations with a real observable: two slots' real
//            states in the components of one array (slots 2j and 2j + 1);
//   real     the same circuits with one real state per array, for calls of few
//            slots, where an SM's rate per state counts, not the states per SM.
// A circuit of Y rotations is one of Ry and Ry-encoding groups and CNOTs: its
// states stay real, half the memory and multiply-adds of the complex form
// (complex128 runs at 2 FP64 multiply-adds a clock and SM: 11 qubits, 3
// layers, 12 references, adjoint: 510 us as complex states, one per SM, 190 as real ones).
#include <cuda_runtime.h>

#include <algorithm>

#include "engine.cuh"
#include "hbm.h"
#include "kernels.h"
#include "tile_common.cuh"

namespace svk {
namespace {

enum ChipKind { kChipComplex = 0, kChipPair = 1, kChipReal = 2 };

// ------------------------------------------------- amplitudes of any kind

__device__ __forceinline__ float fmaA(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fmaA(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float2 fmaA(float2 a, float2 b, float2 c) {
    return f2unpack(f2fma(f2of(a), f2of(b), f2of(c)));
}
__device__ __forceinline__ double2 fmaA(double2 a, double2 b, double2 c) {
    return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y));
}
template <typename A> __device__ __forceinline__ A zeroA() { return A{}; }
__device__ __forceinline__ float subA(float a, float b) { return a - b; }
__device__ __forceinline__ double subA(double a, double b) { return a - b; }
__device__ __forceinline__ float2 subA(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 subA(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }

template <typename Real, int kKind> struct Amp { using T = typename CT<Real>::T; };
template <typename Real> struct Amp<Real, kChipReal> { using T = Real; };

// Values per group sum: complex k0 - k1, k2, k3; real k3 per state.
template <int kKind> constexpr int kSums = kKind == kChipComplex ? 3 : (kKind == kChipPair ? 2 : 1);

// Real rotations (shears) of one kind of amplitude on register bits 0..M-1 (M
// at run time, bits without a group hold alpha = beta = 0).
template <typename A, int R, int I>
__device__ __forceinline__ void shear_bit(A (&a)[1 << R], const A al, const A be) {
#pragma unroll
    for (int r = 0; r < (1 << R); ++r) {
        if (r & (1 << I)) continue;
        A x = a[r], y = a[r | (1 << I)];
        x = fmaA(al, y, x);
        y = fmaA(be, x, y);
        x = fmaA(al, y, x);
        a[r] = x;
        a[r | (1 << I)] = y;
    }
}

// One stage's record (32 bytes): words 0-1 the groups of register bits 0..3
// (16 bits each), word 2 M | parametrised bits << 8, words 3-6 the bits'
// load | store << 16 address vectors (byte offsets < 2^16).
__device__ __forceinline__ void build_recs(const Program &p, int R, int asz, uint4 *rec) {
    for (int s = threadIdx.x; s < p.n_stages; s += blockDim.x) {
        const Stage *sg = p.stages + s;
        uint32_t w[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        for (int o = sg->op_begin; o < sg->op_end; ++o) {  // one op per bit, bits 0..M-1
            const Op op = p.ops[o];
            w[op.a >> 1] |= (uint32_t)op.group << (16 * (op.a & 1));
            w[2] += 1u;
            if (p.groups[op.group].has_param) w[2] |= 1u << (8 + op.a);
        }
        for (int i = 0; i < R; ++i)
            w[3 + i] = (sg->ldq[i] * asz) | ((sg->stq[i] * asz) << 16);
        rec[2 * s] = make_uint4(w[0], w[1], w[2], w[3]);
        rec[2 * s + 1] = make_uint4(w[4], w[5], w[6], w[7]);
    }
}

template <int R> struct StageRec {
    uint32_t g01, g23, info, lq[R], sq[R];
    __device__ __forceinline__ StageRec(const uint4 *rec, int s) {
        const uint4 a = rec[2 * s], b = rec[2 * s + 1];
        g01 = a.x;
        g23 = a.y;
        info = a.z;
        const uint32_t w[4] = {a.w, b.x, b.y, b.z};
#pragma unroll
        for (int i = 0; i < R; ++i) {
            lq[i] = w[i] & 0xffffu;
            sq[i] = w[i] >> 16;
        }
    }
    __device__ __forceinline__ int m() const { return (int)(info & 7u); }
    __device__ __forceinline__ int group(int i) const {
        return (int)(((i & 2) ? g23 : g01) >> (16 * (i & 1)) & 0xffffu);
    }
    __device__ __forceinline__ bool param(int i) const { return (info >> (8 + i)) & 1u; }
};

// This thread's load | store << 16 base of every stage.
__device__ __forceinline__ void build_bases(const Program &p, int tid, int Ts, int asz,
                                            uint32_t *tb) {
    for (int s = 0; s < p.n_stages; ++s) {
        const Stage *sg = p.stages + s;
        uint32_t lb = 0, sb = 0;
        for (int k = 0; k < sg->n_thr; ++k)
            if ((tid >> k) & 1) {
                lb ^= sg->ldt[k];
                sb ^= sg->stt[k];
            }
        tb[s * Ts + tid] = (lb * asz) | ((sb * asz) << 16);
    }
}

template <typename A, int R, int I>
__device__ __forceinline__ void real_rots(const StageRec<R> &st, int m, const A *coef,
                                          A (&a)[1 << R]) {
    if constexpr (I < R) {
        if (I < m) {
            const A *c = coef + 2 * st.group(I);
            shear_bit<A, R, I>(a, c[0], c[1]);
            real_rots<A, R, I + 1>(st, m, coef, a);
        }
    }
}

// k3 of register bit I and its inverse rotation on psi and lambda.
template <typename A, int R, int I>
__device__ __forceinline__ void real_unrots(const StageRec<R> &st, int m, const A *coef,
                                            A (&a)[1 << R], A (&l)[1 << R], A (&k)[R]) {
    if constexpr (I >= 0) {
        if (I < m) {
            A p = zeroA<A>(), q = zeroA<A>();
#pragma unroll
            for (int r = 0; r < (1 << R); ++r) {
                if (r & (1 << I)) continue;
                p = fmaA(a[r], l[r | (1 << I)], p);
                q = fmaA(a[r | (1 << I)], l[r], q);
            }
            k[I] = subA(p, q);
            const A *c = coef + 2 * st.group(I);
            const A al = subA(zeroA<A>(), c[0]), be = subA(zeroA<A>(), c[1]);
            shear_bit<A, R, I>(a, al, be);
            shear_bit<A, R, I>(l, al, be);
        }
        real_unrots<A, R, I - 1>(st, m, coef, a, l, k);
    }
}

// Forward stages of one state between the buffers X and Y (each stage reads
// one and writes the other: one barrier a stage); returns the final one.
template <typename Real, int R, int kKind>
__device__ __forceinline__ unsigned char *chip_forward(const Program &p, const uint4 *rec,
                                                       const uint32_t *tb, int Ts, int tid,
                                                       const typename Amp<Real, kKind>::T *coef,
                                                       const typename CT<Real>::T *tabs,
                                                       unsigned char *X, unsigned char *Y) {
    using A = typename Amp<Real, kKind>::T;
    constexpr int NA = 1 << R;
    for (int s = 0; s < p.n_stages; ++s) {
        const StageRec<R> st(rec, s);
        const uint32_t b = tb[s * Ts + tid], lb = b & 0xffffu, sb = b >> 16;
        const int m = st.m();
        A a[NA];
#pragma unroll
        for (int r = 0; r < NA; ++r) a[r] = *reinterpret_cast<const A *>(X + (lb ^ xsel<R>(r, st.lq)));
        if constexpr (kKind == kChipComplex) {
            const A *tab = tabs + s * 2 * NA;
            if (m) {
                apply_phases<A, R, R, true>(tab, a);
#pragma unroll
                for (int i = 0; i < R; ++i)
                    if (i < m) {
                        const A c = coef[2 * st.group(i)];
                        if (i == 0) rot3_bit<A, R, 0>(a, both<A>(c.x), both<A>(c.y));
                        if constexpr (R > 1)
                            if (i == 1) rot3_bit<A, R, 1>(a, both<A>(c.x), both<A>(c.y));
                        if constexpr (R > 2)
                            if (i == 2) rot3_bit<A, R, 2>(a, both<A>(c.x), both<A>(c.y));
                        if constexpr (R > 3)
                            if (i == 3) rot3_bit<A, R, 3>(a, both<A>(c.x), both<A>(c.y));
                    }
                apply_phases<A, R, R, false>(tab + NA, a);
            }
        } else {
            real_rots<A, R, 0>(st, m, coef, a);
        }
#pragma unroll
        for (int r = 0; r < NA; ++r) *reinterpret_cast<A *>(Y + (sb ^ xsel<R>(r, st.sq))) = a[r];
        __syncthreads();
        unsigned char *t = X;
        X = Y;
        Y = t;
    }
    return X;
}

// |ref> (pair: of both slots) in natural order.
template <typename Real, int R, int kKind>
__device__ __forceinline__ void chip_init(int n, int w, int tid, int64_t ra, int64_t rb,
                                          typename Amp<Real, kKind>::T *X) {
    using A = typename Amp<Real, kKind>::T;
#pragma unroll
    for (int k = 0; k < (1 << R); ++k) {
        const uint32_t j = (uint32_t)tid + ((uint32_t)k << (n - R));
        A v = zeroA<A>();
        if constexpr (kKind == kChipReal) {
            if ((int64_t)j == ra) v = 1;
        } else {
            if ((int64_t)j == ra) v.x = 1;
            if (kKind == kChipPair && (int64_t)j == rb) v.y = 1;
        }
        X[swizzle(j, w)] = v;
    }
}

// lambda = H psi from the diagonal tables and this thread's part of <H> (pair:
// of both slots), FP64 sums.
template <typename Real, int R, int kKind>
__device__ __forceinline__ void chip_h(const Observable &o, const typename CT<Real>::T *dtab,
                                       const typename Amp<Real, kKind>::T *psi,
                                       typename Amp<Real, kKind>::T *lam, int n, int tid, int w,
                                       double &ea, double &eb) {
    using A = typename Amp<Real, kKind>::T;
    constexpr int NA = 1 << R;
    const int sh = n - R;
    uint32_t v[R];
    const uint32_t s0 = natural_vectors<R>(tid, sh, w, v);
    A acc[NA];
#pragma unroll
    for (int k = 0; k < NA; ++k) acc[k] = zeroA<A>();
    for (int g = 0; g < o.n_tgroups; ++g) {
        const TermGroup tg = o.tgroups[g];
        const typename CT<Real>::T *D = dtab + ((size_t)g << n);
#pragma unroll
        for (int k = 0; k < NA; ++k) {
            const uint32_t jx = ((uint32_t)tid | ((uint32_t)k << sh)) ^ tg.x;
            const typename CT<Real>::T d = __ldg(D + jx);
            const A px = psi[s0 ^ xsel<R>(k, v) ^ tg.sx];
            if constexpr (kKind == kChipReal) {
                acc[k] = fmaA(d.x, px, acc[k]);
            } else if constexpr (kKind == kChipPair) {
                acc[k] = fmaA(both<A>(d.x), px, acc[k]);
            } else {
                acc[k].x = fmaR(d.x, px.x, fmaR(-d.y, px.y, acc[k].x));
                acc[k].y = fmaR(d.x, px.y, fmaR(d.y, px.x, acc[k].y));
            }
        }
    }
    ea = eb = 0.0;
#pragma unroll
    for (int k = 0; k < NA; ++k) {
        const uint32_t sj = s0 ^ xsel<R>(k, v);
        const A pj = psi[sj];
        lam[sj] = acc[k];
        if constexpr (kKind == kChipReal) {
            ea += (double)(pj * acc[k]);
        } else if constexpr (kKind == kChipPair) {
            ea += (double)(pj.x * acc[k].x);
            eb += (double)(pj.y * acc[k].y);
        } else {
            ea += (double)fmaR(pj.x, acc[k].x, pj.y * acc[k].y);
        }
    }
}

// Warp sums of a stage's values k (three, two or one per register bit) to
// rw[group][warp][kSums].
template <typename Real, int R, int kKind>
__device__ __forceinline__ void chip_store_sums(const StageRec<R> &st, const Real (&val)[12],
                                                int lane, int warp, int wps, Real *rw) {
    constexpr int NS = kSums<kKind>;
    constexpr int NV = NS == 3 ? 12 : (NS == 2 ? (R <= 2 ? 4 : 8) : 4);
    Real x[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) x[v] = val[v];
    if constexpr (NV == 12) warp_reduce_quad12<Real>(x, lane);
    else warp_reduce_quad<Real, NV>(x, lane);
#pragma unroll
    for (int q = 0; q < NV / 4; ++q) {
#pragma unroll
        for (int off = 4; off < 32; off <<= 1) x[q] += __shfl_xor_sync(0xffffffffu, x[q], off);
        const int v = 4 * q + lane, i = v / NS;
        if (lane < 4 && i < R && st.param(i)) rw[(st.group(i) * wps + warp) * NS + v % NS] = x[q];
    }
}

// a * conj(p).
template <typename C> __device__ __forceinline__ C phase_mulc(const C a, const C p) {
    C r;
    r.x = fmaR(a.x, p.x, a.y * p.y);
    r.y = fmaR(a.y, p.x, -(a.x * p.y));
    return r;
}

template <typename C, typename Real, int R, int I>
__device__ __forceinline__ void chip_split_unrots(const StageRec<R> &st, int m, const C *coef,
                                                  C (&a)[1 << R], C (&l)[1 << R], Real *k) {
    if constexpr (I >= 0) {
        if (I < m) {
            split_sums<C, Real, R, I>(a, l, k + 3 * I);
            const C c = coef[2 * st.group(I)];
            rot3_bit<C, R, I>(a, both<C>(-c.x), both<C>(-c.y));
            rot3_bit<C, R, I>(l, both<C>(-c.x), both<C>(-c.y));
        }
        chip_split_unrots<C, Real, R, I - 1>(st, m, coef, a, l, k);
    }
}

// A reverse stage of complex groups (hbm.cu's split_rev with M at run time and
// unconjugated tables): l holds i lambda between the two phase products.
template <typename C, typename Real, int R>
__device__ __forceinline__ void chip_split_rev(const StageRec<R> &st, int m, const C *coef,
                                               const C *tab, C (&a)[1 << R], C (&l)[1 << R],
                                               Real *k) {
    constexpr int NA = 1 << R;
#pragma unroll
    for (int q = 0; q < NA / 2; ++q) {
        C ph[2];
        load_phases(tab + NA, q, ph[0], ph[1]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = 2 * q + h;
            a[j] = phase_mulc(a[j], ph[h]);
            const C v = phase_mulc(l[j], ph[h]);
            l[j].x = -v.y;
            l[j].y = v.x;
        }
    }
    chip_split_unrots<C, Real, R, R - 1>(st, m, coef, a, l, k);
#pragma unroll
    for (int q = 0; q < NA / 2; ++q) {
        C ph[2];
        load_phases(tab, q, ph[0], ph[1]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = 2 * q + h;
            C v;
            v.x = l[j].y;
            v.y = -l[j].x;
            if (j) a[j] = phase_mulc(a[j], ph[h]);  // entry 0 is 1
            l[j] = j ? phase_mulc(v, ph[h]) : v;
        }
    }
}

struct ChipArgs {
    Program p;
    Observable o;
    SlotSource src;
    CostSource cs;
    GroupMats gm;
    const int64_t *refs;  // [states][2]
    const void *dtab;
    double *slot_grads, *slot_E;
    ChipShape sh;
};

// Adjoint: forward, lambda = H psi, reverse sweep, gradients of every slot
// times its cost weight.  Coefficients come from k_group_mats (FP64, rounded
// once), phase tables from k_phase_tables.
template <typename Real, int R, int kKind, int kThreads, int kBlocks>
__global__ void __launch_bounds__(kThreads, kBlocks) k_chip_adjoint(const __grid_constant__ ChipArgs c) {
    using A = typename Amp<Real, kKind>::T;
    using C = typename CT<Real>::T;
    constexpr int NA = 1 << R, NS = kSums<kKind>, kPer = kKind == kChipPair ? 2 : 1;
    extern __shared__ __align__(16) unsigned char smem[];
    pdl_trigger();
    const Program &p = c.p;
    const int n = p.n, w = p.swz_bits, Ts = 1 << (n - R), G = p.n_groups, P = p.n_params;
    const int ls = threadIdx.x >> (n - R), tid = threadIdx.x & (Ts - 1), wps = Ts >> 5;
    const int n_states = (c.src.n_slots + kPer - 1) / kPer;
    const int state = blockIdx.x * c.sh.S + ls;
    const bool live = state < n_states;
    const int b = live ? state : n_states - 1;
    uint4 *rec = reinterpret_cast<uint4 *>(smem + c.sh.off_rec);
    uint32_t *tb = reinterpret_cast<uint32_t *>(smem + c.sh.off_tb);
    unsigned char *mine = smem + c.sh.off_slot + (size_t)ls * c.sh.slot_bytes;
    unsigned char *X = mine, *Y = mine + (sizeof(A) << n);
    A *coef = reinterpret_cast<A *>(mine + c.sh.o_coef);
    C *tabs = reinterpret_cast<C *>(mine + c.sh.o_tabs);
    Real *rw = reinterpret_cast<Real *>(mine + c.sh.o_rw);
    double *grad = reinterpret_cast<double *>(mine + c.sh.o_grad);  // [kPer][P]
    double *red = reinterpret_cast<double *>(smem + c.sh.off_red);
    build_recs(p, R, (int)sizeof(A), rec);  // the plan is older than the stream's work
    if (ls == 0) build_bases(p, tid, Ts, (int)sizeof(A), tb);
    pdl_wait();
    for (int x = tid; x < 2 * G; x += Ts) {
        const int g = x >> 1;
        if constexpr (kKind == kChipComplex) {
            const double2 *f = c.gm.split + ((size_t)b * G + g) * 4;
            coef[x] = (x & 1) ? cmk<C>(1, 0) : cmk<C>(f[0].x, f[0].y);
            if (x & 1) {
                const double2 v = cmul(f[1], cconj(f[2]));  // p0 conj(p1)
                coef[x] = cmk<C>(v.x, v.y);
            }
        } else {
            const C v = ((const C *)c.gm.mats)[((size_t)b * G + g) * 4 + (x & 1)];
            if constexpr (kKind == kChipPair) coef[x] = v;
            else coef[x] = v.x;
        }
    }
    if constexpr (kKind == kChipComplex) {
        const C *t = (const C *)c.gm.tabs + (size_t)b * c.gm.n_stages * 2 * NA;
        for (int x = tid; x < p.n_stages * 2 * NA; x += Ts) tabs[x] = t[x];
    }
    for (int q = tid; q < kPer * P; q += Ts) grad[q] = 0.0;
    chip_init<Real, R, kKind>(n, w, tid, c.refs[2 * b], c.refs[2 * b + 1], reinterpret_cast<A *>(X));
    __syncthreads();
    unsigned char *psi = chip_forward<Real, R, kKind>(p, rec, tb, Ts, tid, coef, tabs, X, Y);
    unsigned char *lam = psi == X ? Y : X;
    double ea, eb;
    chip_h<Real, R, kKind>(c.o, (const C *)c.dtab, reinterpret_cast<const A *>(psi),
                           reinterpret_cast<A *>(lam), n, tid, w, ea, eb);
    ea = slot_sum(ea, Ts, red);
    if (kPer == 2) {
        __syncthreads();
        eb = slot_sum(eb, Ts, red);
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = tid >> 5;
    for (int s = p.n_stages - 1; s >= 0; --s) {
        const StageRec<R> st(rec, s);
        const uint32_t bb = tb[s * Ts + tid], lb = bb & 0xffffu, sb = bb >> 16;
        const int m = st.m();
        A a[NA], l[NA];
#pragma unroll
        for (int r = 0; r < NA; ++r) {
            const uint32_t ad = sb ^ xsel<R>(r, st.sq);
            a[r] = *reinterpret_cast<const A *>(psi + ad);
            l[r] = *reinterpret_cast<const A *>(lam + ad);
        }
        if (m) {
            Real val[12];
#pragma unroll
            for (int v = 0; v < 12; ++v) val[v] = 0;
            if constexpr (kKind == kChipComplex) {
                chip_split_rev<C, Real, R>(st, m, coef, tabs + s * 2 * NA, a, l, val);
            } else {
                A k[R];
#pragma unroll
                for (int i = 0; i < R; ++i) k[i] = zeroA<A>();
                real_unrots<A, R, R - 1>(st, m, coef, a, l, k);
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    if constexpr (kKind == kChipPair) {
                        val[2 * i] = k[i].x;
                        val[2 * i + 1] = k[i].y;
                    } else {
                        val[i] = k[i];
                    }
                }
            }
            if ((st.info >> 8) & 15u) chip_store_sums<Real, R, kKind>(st, val, lane, warp, wps, rw);
        }
        __syncthreads();
        if (s > 0) {  // nothing reads the states before the first stage
#pragma unroll
            for (int r = 0; r < NA; ++r) {
                const uint32_t ad = lb ^ xsel<R>(r, st.lq);
                *reinterpret_cast<A *>(psi + ad) = a[r];
                *reinterpret_cast<A *>(lam + ad) = l[r];
            }
            __syncthreads();
        }
    }
    // derivatives of every group's members
    for (int g = tid; g < G; g += Ts) {
        const Group grp = p.groups[g];
        if (!grp.has_param) continue;
        double k[NS];
        for (int v = 0; v < NS; ++v) {
            k[v] = 0.0;
            for (int q = 0; q < wps; ++q) k[v] += (double)rw[(g * wps + q) * NS + v];
        }
        if constexpr (kKind == kChipComplex) {
            const C f = coef[2 * g + 1];
            const double re = 0.5 * (f.x * k[2] - f.y * k[1]), im = 0.5 * (f.x * k[1] + f.y * k[2]);
            const double r8[8] = {0.0, 0.5 * k[0], re, im, -re, im, 0.0, -0.5 * k[0]};
            group_gradients<Real>(p, g, r8, resolve(c.src, b), grad);
        } else {
            // Y rotations commute: each parameter of the group has k3
            for (int m = grp.m_begin; m < grp.m_end; ++m) {
                const int q = p.members[m].kind == M_RY ? p.members[m].param : -1;
                if (q < 0) continue;
                for (int v = 0; v < NS; ++v) atomicAdd(&grad[v * P + q], k[v]);
            }
        }
    }
    __syncthreads();
    if (!live) return;
    for (int v = 0; v < kPer; ++v) {
        const int slot = kPer * state + v;
        if (slot >= c.src.n_slots) break;
        const double e = v ? eb : ea;
        const SlotInfo si = resolve(c.src, slot);
        const double wgt = cost_weight(c.cs, si.instance, e);
        for (int q = tid; q < P; q += Ts) c.slot_grads[(int64_t)slot * P + q] = wgt * grad[v * P + q];
        if (tid == 0) c.slot_E[slot] = e;
    }
}

}  // namespace

const char *chip_shape(int kind, int n, int R, int c128, int G, int P, int n_stages, int n_states,
                       int sms, ChipShape *out) {
    const uint32_t csz = c128 ? 16 : 8, rsz = csz / 2;
    const uint32_t asz = kind == kChipReal ? rsz : csz, per = kind == kChipPair ? 2 : 1;
    const uint32_t ns = kind == kChipComplex ? 3 : per;
    const int Ts = 1 << (n - R);
    if (n - R < 5 || n - R > 9) return "threads per state outside one warp .. 512";
    ChipShape s{};
    s.R = R;
    auto up = [](size_t x) { return (uint32_t)((x + 15) & ~size_t(15)); };
    s.o_coef = 2u * (asz << n);
    s.o_tabs = s.o_coef + up((size_t)G * 2 * asz);
    s.o_rw = s.o_tabs + (kind == kChipComplex ? (uint32_t)n_stages * (2 * csz << R) : 0u);
    s.o_grad = s.o_rw + up((size_t)G * (Ts / 32) * ns * rsz);
    s.slot_bytes = s.o_grad + up((size_t)P * per * 8);
    s.off_rec = 0;
    s.off_tb = s.off_rec + (uint32_t)n_stages * 32;
    s.off_red = s.off_tb + up((size_t)n_stages * Ts * 4);
    s.off_slot = s.off_red + 32 * 8;
    // blocks of at least 128 threads, while there is a block for every SM
    int S = std::max(1, 128 / Ts);
    while (S > 1 && (n_states + S - 1) / S < sms) S >>= 1;
    while (S > 1 && s.off_slot + (size_t)S * s.slot_bytes > 200u * 1024u) S >>= 1;
    s.S = S;
    s.blocks = (n_states + S - 1) / S;
    const size_t bytes = s.off_slot + (size_t)S * s.slot_bytes;
    if (bytes > 220u * 1024u) return "state too large for the on-chip engine";
    s.smem = (uint32_t)bytes;
    *out = s;
    return nullptr;
}

template <typename Real, int R, int kKind, int kThreads, int kBlocks>
static cudaError_t run_chip_adjoint(const ChipArgs &a, cudaStream_t st) {
    auto k = k_chip_adjoint<Real, R, kKind, kThreads, kBlocks>;
    cudaError_t e = allow_smem_attr((const void *)k, a.sh.smem);
    if (e != cudaSuccess) return e;
    // not as a dependent launch: its blocks would gather on the SMs where the
    // small blocks before it end (200 one-warp states: 840 against 290 us)
    return launch_dep_if(false, k, a.sh.blocks, a.sh.S << (a.p.n - R), a.sh.smem, st, a);
}

template <int kKind>
static cudaError_t chip_adjoint_kind(int c128, const ChipArgs &a, cudaStream_t st) {
    if (c128) {
        if (a.sh.R == 2) return run_chip_adjoint<double, 2, kKind, 512, 1>(a, st);
        if (a.sh.R == 3) return run_chip_adjoint<double, 3, kKind, 512, 1>(a, st);
        return cudaErrorInvalidValue;
    }
    if (a.sh.R == 2) return run_chip_adjoint<float, 2, kKind, 512, 1>(a, st);
    if (a.sh.R == 3) return run_chip_adjoint<float, 3, kKind, 512, 1>(a, st);
    if (a.sh.R == 4 && (a.sh.S << (a.p.n - 4)) > 256)
        return run_chip_adjoint<float, 4, kKind, 512, 1>(a, st);
    if (a.sh.R == 4) return run_chip_adjoint<float, 4, kKind, 256, 2>(a, st);
    return cudaErrorInvalidValue;
}

cudaError_t launch_chip_adjoint(int c128, int kind, const ChipShape &sh, const Program &p,
                                const Observable &o, const SlotSource &src, const CostSource &cs,
                                void *group_base, const void *dtab, double *slot_grads,
                                double *slot_E, cudaStream_t st) {
    const int mats = kind == kChipComplex ? 0 : kind;  // 1: pairs, 2: single real states
    const int n_states = kind == kChipPair ? (src.n_slots + 1) / 2 : src.n_slots;
    cudaError_t e = launch_group_mats(c128, p, src, group_base, st, mats, ClearList{}, true);
    if (e != cudaSuccess) return e;
    const GroupBuf gb = group_buf(c128, p, (size_t)n_states, mats != 0);
    ChipArgs a{};
    a.p = p;
    a.o = o;
    a.src = src;
    a.cs = cs;
    a.gm = group_mats_of(gb, group_base, 0);
    a.refs = (const int64_t *)((const char *)group_base + gb.refs);
    a.dtab = dtab;
    a.slot_grads = slot_grads;
    a.slot_E = slot_E;
    a.sh = sh;
    if (kind == kChipComplex) return chip_adjoint_kind<kChipComplex>(c128, a, st);
    if (kind == kChipPair) return chip_adjoint_kind<kChipPair>(c128, a, st);
    return chip_adjoint_kind<kChipReal>(c128, a, st);
}

}  // namespace svk
