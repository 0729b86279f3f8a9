// Launchers of the tile-pass kernels (hbm.cu): states in device memory.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

#include "kernels.h"
#include "svk_types.h"

namespace svk {

// pair (here and below): two real circuits per state (slots 2j and 2j + 1 in
// the components of state j); the launchers' slot counts are then pairs,
// except in a SlotSource and in pair_rows.
// What the passes read of every state's groups, in one buffer (offsets in
// bytes): mats [states][groups][4] complex of the state's precision; without
// pair also split [states][groups][4] double2, the groups' split forms, and
// tabs [states][stages][2][2^R] complex, the split stages' phase tables; refs
// [states][2], the states' reference indices (pair: of its two slots;
// otherwise the slot's twice).
struct GroupBuf {
    size_t split = 0, tabs = 0, refs = 0, bytes = 0;
    int G = 0, n_stages = 0;
};
inline GroupBuf group_buf(int c128, const Program &p, size_t n_states, bool pair) {
    const size_t csz = c128 ? 16 : 8;
    GroupBuf b;
    b.G = p.n_groups;
    b.n_stages = p.n_stages;
    size_t off = n_states * b.G * 4 * csz;
    b.split = off;
    if (!pair) off += n_states * b.G * 64;
    b.tabs = off;
    if (!pair) off += (n_states * b.n_stages * 2 * csz) << p.R;
    b.refs = off;
    b.bytes = off + n_states * 16;
    return b;
}
// The part of a pass whose first stage is stage0 of the plan.
struct GroupMats {
    const void *mats, *tabs;
    const double2 *split;
    int32_t G, n_stages, stage0, pad;
};
inline GroupMats group_mats_of(const GroupBuf &b, const void *base, int stage0) {
    const char *p = (const char *)base;
    return GroupMats{p, p + b.tabs, (const double2 *)(p + b.split), b.G, b.n_stages, stage0, 0};
}
// kind: 0 complex states, 1 pairs, 2 one real state per slot (coefficients as
// of a pair of the slot with itself).  every: phase tables of every stage (the
// on-chip engine), not only of the passes' split stages.
// Arrays of doubles set to zero on the way (sums that later kernels add to).
struct ClearList {
    double *p[3];
    int64_t n[3];
};
cudaError_t launch_group_mats(int c128, const Program &p, const SlotSource &src, void *base,
                              cudaStream_t st, int kind = 0,
                              const ClearList &clear = ClearList{}, bool every = false);
// Zeroes the slot states and sets amplitude |ref> of each to 1.
cudaError_t launch_init_states(int c128, void *states, int n, const SlotSource &src,
                               cudaStream_t st);
// Where a pass's states are known to be zero.  A state starts as |ref>, and a
// pass spreads it over the index bits local to it only, so before pass i
// every amplitude is zero whose bits outside the union of the earlier passes'
// local bits differ from ref's.  A sparse pass walks the tiles that can hold
// a nonzero amplitude (its TilePass counts the tile-number bits inside the
// union; `fixed` are the others, taken from ref), and reads only amplitudes
// whose local bits in `zero` equal ref's (the others are zero and need not be
// in memory).  init: the state before the pass is |ref> itself, not read.
// All zero: a dense pass.
struct Sparse {
    const int64_t *refs;  // [states][2]
    uint32_t fixed, zero;
    int32_t init, pad;
};
// The sparse form of pass P when the amplitudes' bits in `support` (an index
// mask) are the ones that may differ from ref; sets P's tile count.
Sparse sparse_pass(TilePass *P, uint32_t support, const int64_t *refs, bool init);
// Phase tables of the split stages in that shared memory (reverse passes of
// one sum a group have none): at most 4 KB, on top of kPassSmem.
uint32_t tile_table_bytes(int c128, const TilePass &P, bool rev, bool any = false);
// Largest shared memory of a pass without its phase tables; with them it is
// still within the 227 KB of a block.
constexpr uint32_t kPassSmem = 220u * 1024u;
// Shared memory of one block of the forward / reverse kernels of pass P.
// (any: of a kernel that takes complex and real passes alike).
uint32_t tile_fwd_smem(int c128, const TilePass &P, bool any = false);
uint32_t tile_rev_smem(int c128, const TilePass &P, int bufs = 2, bool any = false);
// Forward pass P over n_slots states of n qubits.
// src (null: states) holds the pass's input; the output goes to states.
cudaError_t launch_tile_fwd(int c128, const TilePass &P, int n, int n_slots,
                            const GroupMats &gm, void *states, int64_t max_blocks, cudaStream_t st,
                            const void *src = nullptr, bool pair = false,
                            const Sparse &sp = Sparse{});
// Reverse pass P on psi and lambda; adds the reduced matrices of its
// parametrised groups to rho_g[slot][G][8].  psi_src (null: psi) holds the
// psi the pass reads (a stored forward state); its output psi goes to psi
// unless write_psi is false (the next reverse pass restarts psi from a
// stored state, or this is the last one).  pair: rho_g has two rows per state.
cudaError_t launch_tile_rev(int c128, const TilePass &P, int n, int n_slots,
                            const GroupMats &gm, void *psi, void *lam, double *rho_g, int64_t max_blocks,
                            cudaStream_t st, const void *psi_src = nullptr,
                            bool write_psi = true, bool pair = false,
                            const Sparse &sp = Sparse{});
// Codes a kernel writes to the library's device error word when a bounded
// device-side wait gives up (reported as SV_ERR_TIMEOUT by sv_sync_status).
constexpr int SV_DEVERR_MMA_WAIT = 1;
constexpr int SV_DEVERR_SWEEP_WAIT = 2;
// Raises kernel's dynamic shared-memory limit to `bytes` (limits only grow;
// no attribute change while a graph capture runs: fails instead).
cudaError_t allow_smem_attr(const void *kernel, uint32_t bytes);
// Forgets the limits set so far (a device reset drops them).
void forget_smem_limits();
// Forward pass P with every register stage applied as one dense 16 x 16
// complex block on the tensor cores (tc.cu; complex64, R = 4, t = 11 or 12).
// err: the device error word (bounded waits), or null.
uint32_t tile_fwd_tc_smem(const TilePass &P);
bool tile_fwd_tc_supported(int c128, const TilePass &P);
cudaError_t launch_tile_fwd_tc(const TilePass &P, int n, int n_slots, const void *mats, int G,
                               void *states, int64_t max_blocks, cudaStream_t st, int *err,
                               const void *src = nullptr);
// One block that waits `limit` times on an mbarrier nothing arrives on and
// records SV_DEVERR_MMA_WAIT: the bounded-wait path, for tests.
cudaError_t launch_wait_expiry(int *err, uint32_t limit, cudaStream_t st);
// Persistent sweeps of several problems (forward, or reverse with rev):
// tasks (device) in ticket order; ticket (device, zero) and done[n_tasks]
// (device, zero) are the scheduler's counters; every task uses the same tile
// shape (threads = 2^(t - R)); smem: the largest tile_sweep_smem over the
// tasks; blocks: at most the resident blocks (tile_sweep_blocks_per_sm x SMs).
// Launchers skip kernel attribute calls while a graph capture runs.
void set_capturing(bool on);
uint32_t tile_sweep_smem(int c128, bool rev, const TilePass &P);
int tile_sweep_blocks_per_sm(int c128, int R, bool rev, uint32_t smem, int threads);
cudaError_t launch_tile_sweep(int c128, int R, bool rev, const SweepTask *tasks, int n_tasks,
                              long long n_tickets, unsigned long long *ticket, unsigned int *done,
                              int *err, int blocks, int threads, uint32_t smem, cudaStream_t st);
// One tile pass of lambda = H psi (lam may be null: energies only); adds this
// pass's part of <psi|H|psi> to E[slot] (zero E before the first pass).
// pair_rows > 0: pairs of real states whose E has pair_rows entries.
cudaError_t launch_tile_h(int c128, const HPass &P, int n, int n_slots, const void *psi, void *lam,
                          double *E, int64_t max_blocks, cudaStream_t st, int pair_rows = 0);
// Data-driven circuit learning: js[r] = JS(target | |psi_r|^2) (zeroed here
// first) and lam_r = dJS/d|psi_r|^2 * psi_r elementwise.
cudaError_t launch_ddcl_lambda(int c128, int n, int n_rows, const void *psi, const double *target,
                               void *lam, double *js, cudaStream_t st);
// js[0] = JS divergence of one state's output distribution from `target`;
// D[j] = dJS/dP_theta(j) (device [2^n] doubles).
cudaError_t launch_ddcl_diag(int c128, int n, const void *psi, const double *target, double *D,
                             double *js, cudaStream_t st);
// out[r] = sum_j D[j] |psi_r(j)|^2 for n_rows states of 2^n amplitudes.
cudaError_t launch_diag_expect(int c128, int n, int n_rows, const void *states, const double *D,
                               double *out, cudaStream_t st);
// out[j] = in[j with bit b moved to bit qubit_of_bit[b]]: a 2^n table indexed
// by qubit values, rewritten for states whose bit b holds qubit qubit_of_bit[b].
cudaError_t launch_relayout(int n, const int32_t *qubit_of_bit, const double *in, double *out,
                            cudaStream_t st);
// out[r] = <psi_r|H|psi_r> (zeroed here first).
cudaError_t launch_expect_big(int c128, const Observable &o, int n, int n_rows,
                              const void *states, double *out, cudaStream_t st);
// lam = H psi and E[r] = <psi_r|H|psi_r> (E zeroed here first).
cudaError_t launch_apply_h_big(int c128, const Observable &o, int n, int n_rows, const void *psi,
                               void *lam, double *E, cudaStream_t st);
// slot_grads[b][param] += weight_b * gradient from rho_g[b][group][8] (zero it first).
cudaError_t launch_group_grads(int c128, const Program &p, const SlotSource &src,
                               const double *rho_g, const CostSource &cs, const double *E,
                               double *slot_grads, cudaStream_t st);

// On-chip adjoint of chip.cu.  kind: 0 complex, 1 pairs of real states, 2
// single real states (circuits of Y rotations and CNOTs, real observable).
// The plan has R register bits, sorted stages of at most one group a bit.
struct ChipShape {
    int32_t R, S, blocks;  // S states per block
    uint32_t smem, off_rec, off_tb, off_slot, off_red, slot_bytes;
    uint32_t o_coef, o_tabs, o_rw, o_grad;
};
const char *chip_shape(int kind, int n, int R, int c128, int G, int P, int n_stages, int n_states,
                       int sms, ChipShape *out);
// group_base: group_buf(...) bytes; dtab: the observable's diagonal tables.
cudaError_t launch_chip_adjoint(int c128, int kind, const ChipShape &sh, const Program &p,
                                const Observable &o, const SlotSource &src, const CostSource &cs,
                                void *group_base, const void *dtab, double *slot_grads,
                                double *slot_E, cudaStream_t st);

}  // namespace svk
