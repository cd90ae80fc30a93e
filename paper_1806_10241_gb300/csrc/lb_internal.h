// Internal interface between the C ABI (lb_capi.cu) and the kernels
// (lb_kernels.cu).  Not part of the public ABI.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "../../include/lb.h"

namespace lbk {

enum Storage { ST_FP64 = 0, ST_FP32 = 1, ST_BF16 = 2, ST_FP16 = 3 };

constexpr int NQ = 19;        // 9 (f) + 5 (g) + 5 (h) planes
// FP16 storage holds the deviations times 2^10 (away from the subnormal
// range); kFp16InvScaleBits is 2^-10 as an FP16 bit pattern
constexpr double kFp16Scale = 1024.0;
constexpr unsigned short kFp16InvScaleBits = 0x1400;
constexpr int NSUM = 12;      // diagnostic partial sums per block
constexpr int MAX_DIAG_BLOCKS = 4096;

// Everything a kernel needs about one lattice, in double precision; the
// launchers convert to the compute type.
struct HostParams {
    int nr, nz, pitch;
    long long plane;          // elements per plane = nz * pitch
    int storage;
    double r0;
    double nu, alpha, omega3, omega_hi, g_beta, T0, body_fx, rho0;
    int planar, sign_literal, explicit_sources;
    // sides 0..3 as lb_side; entry 4 the outer segment of a split top
    int flow[5], swirl[5], heat[5];
    double uwx[5], uwy[5], omega[5], Tw[5];
    int top_split;            // columns >= top_split of the top follow entry 4 (0: one segment)
    double scale;             // storage scale of the deviations (16-bit)
    const float *ytab;        // device table: y[pitch] then 1/y[pitch] (FP64, rounded once)
};

struct Launch {
    int seg_rows;             // rows per z-segment
    int warps_per_block;
    int use_tma;              // FP32 / 16-bit rows: 0 plain loads, 1 TMA ring, 2 TMA ring read in place
};

// Elements per row of a plane: nr rounded up to 32 (4- and 8-byte storage)
// or 64 (2-byte storage) elements.
int pitch_for(int nr, int storage);
// The lattice part of h (shape, pitch, storage, storage scale) from a grid
// descriptor, after the checks lb_required_bytes and lb_create make.  On
// failure h is untouched and err (n bytes) holds a one-line message.
lb_status host_from_desc(const lb_grid_desc *d, HostParams *h, char *err, size_t n);
// The physical part of h from lb_params, after the checks lb_set_params
// makes (relaxation rates, boundary codes and their pairing, the axis only on
// the inner side of a cylinder, finite wall values); needs the lattice part
// (r0).  On failure h is untouched and err holds a one-line message.
lb_status host_set_params(const lb_params *p, HostParams *h, char *err, size_t n);

// lb_diag from the NSUM sums of the diagnostics (result[] of launch_diag),
// the device status word (LB_OK, else reported as the status) and the step.
void diag_from_sums(const HostParams &h, const double *res, int kstatus, int64_t step, lb_diag *out);

// One time step src -> dst; `step` seeds the stochastic rounding of 16-bit
// storage.
cudaError_t launch_step(const HostParams &p, const Launch &l, const void *src, void *dst,
                        unsigned long long step, const void *tmap, int *status, cudaStream_t s);
// Tensor map (CUtensorMap, 128 bytes) of a distribution buffer for the TMA
// row fetches of the FP32 / 16-bit step, box_cols columns per row: ring_cols
// for the row rings, 64 for the tiles.
int ring_cols(int storage);
cudaError_t make_tensor_map(const HostParams &p, void *buf, int box_cols, void *map_out);
// Whether the lattice's node update keeps its pinned order of operations (then
// it takes one launch per step).
bool step_is_pinned(const HostParams &h);
// T time steps on tiles in shared memory (FP32 / 16-bit storage), from the
// buffer of tmap (64-column boxes) to dst.
struct TileLaunch {
    int T, rows, warps;       // time steps, rows of a full tile, warps per block
    int strip;                // long strips marched through a ring of rows
    int parts;                // launches that the pass is cut into
};
// The pass for a lattice: of T steps, or (T = 0) of as many as pay.
TileLaunch tile_plan(const HostParams &p, int T);
// Passes of a call of n steps, up to T in each: as few as that takes, their
// number odd or even as n is, so that the current buffer alternates with the
// step count as it does with one launch per step.  Pass p takes
// n / m + (p < n % m) steps.
inline int64_t pass_count(int64_t n, int T)
{
    const int64_t m = (n + T - 1) / T;
    return m + ((n - m) & 1);
}
// pass: the number of the pass in the lattice's life, from 1 on; begun: the
// lattice's device word for it (k_tiles).
cudaError_t launch_tile(const HostParams &p, const TileLaunch &l, const void *tmap, void *dst, unsigned long long step,
                        int *status, unsigned *begun, unsigned pass, cudaStream_t s);
// Pre-collision fields of rows [row0, row1) into out[5][row1-row0][nr] (double);
// only_ux: plane 1 alone.
cudaError_t launch_fields(const HostParams &p, const void *src, double *out, int row0, int row1, bool only_ux,
                          cudaStream_t s);
// Bounded-wait self-test: a warp polls an mbarrier nothing arrives at,
// `polls` times, and sets *status to LB_ERR_TIMEOUT.
cudaError_t launch_wait_selftest(int *status, int polls, cudaStream_t s);
// Stream function of nrows rows from their axial velocity ux[nrows][nr]
// (pre-collision fields): psi[nrows][nr] on the cell faces y = r0 + j + 1
// (psi may be null) and rowmax[nrows] = max |Psi| per row.
cudaError_t launch_psi(const double *ux, double *psi, double *rowmax, int nrows, int nr, double r0, cudaStream_t s);
// Grid of a lattice's diagnostics: gx x gy blocks of 128 columns and seg rows.
struct DiagGrid {
    int gx, gy, seg;
};
DiagGrid diag_grid(const HostParams &p, int max_blocks);
// Diagnostics of the stored state src: block partial sums (partial), the
// pre-collision T next to the walls (strips, 4 (nr + nz) doubles of scratch) and
// the final values in result[NSUM]: 0 sum(rho - rho0), 1 sum((rho - rho0) y), 2
// sum T, 3 max |u|, 4..7 Nusselt number per side, 8 divergence flag, 9 / 10 the
// equivalent conductivity k_eq of the inner / outer wall of an annulus.
cudaError_t launch_diag(const HostParams &p, const void *src, double *partial, double *strips, double *result,
                        cudaStream_t s);
// Equilibria of host-format fields [5][rows][nr] (double) into rows [row0,row1) of dst.
cudaError_t launch_init_fields(const HostParams &p, const double *fields, void *dst, int row0,
                               int row1, cudaStream_t s);
// Absolute distributions [19][rows][nr] (double) <-> storage, rows [row0,row1).
cudaError_t launch_export(const HostParams &p, const void *src, double *out, int row0, int row1,
                          cudaStream_t s);
cudaError_t launch_import(const HostParams &p, const double *in, void *dst, int row0, int row1,
                          cudaStream_t s);

size_t storage_bytes(int storage);

// Batched step (FP32 / 16-bit storage): device descriptors built on the host
size_t batch_desc_bytes();
size_t batch_ctl_bytes();
int batch_items(const HostParams &h, int seg_rows);
// One lattice's descriptor: parameters, both buffers and their TMA tensor
// maps, the step count and current buffer when the batch was made, and the
// lattice's device status word (bounded-wait timeouts).
cudaError_t batch_fill_desc(const HostParams &h, void *buf0, void *buf1, unsigned long long step0, int parity0,
                            int seg_rows, const TileLaunch &l, int *status, void *out);
// The automatic pass of a batch, a lattice's tiles under it (none for a pinned
// one), and one pass of T
// <= l.T steps from batch step t on (total: the tiles of all lattices, prefix
// their prefix sums; flip: 0 when the state of step t lies in the buffers that
// were current when the batch was made).
TileLaunch tile_plan_batch(const HostParams *const *h, int n);
int batch_tile_count(const HostParams &h, const TileLaunch &l);
cudaError_t launch_batch_tiles(int storage, const TileLaunch &l, int T, const void *desc, const int *prefix, int n,
                               int total, unsigned long long t, int flip, cudaStream_t s);
int batch_grid(int storage, int wpb);
// Warps of the batched step (row_fetch 1 or 3, wpb warps per block) that can
// be resident on the device at once.
cudaError_t batch_resident_warps(int storage, int row_fetch, int wpb, int *out);
// Kernel attributes of the batched step; called before any stream capture.
cudaError_t batch_prepare(int storage);
// row_fetch: 1 plain loads (persistent grid of `blocks`), 3 TMA ring read in
// place (one warp per work item).  The launch takes batch step t0, plus the
// device counter in ctl when from_counter is set (launches inside a graph).
cudaError_t launch_batch(int storage, int row_fetch, const void *desc, const int *prefix, int n, int total,
                         void *ctl, int wpb, int blocks, unsigned long long t0, int from_counter,
                         cudaStream_t s);
// The same step of the batch's pinned lattices (step_is_pinned), which
// launch_batch and launch_batch_persist leave out.
cudaError_t launch_batch_pinned(int storage, const void *desc, const int *prefix, int n, int total, void *ctl, int wpb,
                                unsigned long long t0, int from_counter, cudaStream_t s);
// nsteps batch steps t0 .. t0 + nsteps - 1 in one cooperative launch (every
// work item resident; items wait only for their neighbours' progress in
// done[total], cleared here first).
cudaError_t launch_batch_persist(int storage, const void *desc, const int *prefix, int n, int total, int wpb,
                                 unsigned long long t0, int nsteps, int *done, cudaStream_t s);
// The device counter of a batch: set to value, or advanced by it (add != 0).
cudaError_t launch_batch_counter(void *ctl, unsigned long long value, int add, cudaStream_t s);
// Batched diagnostics: one descriptor per lattice (its partial-sum buffer and
// the grid of its own diagnostics; returns the number of blocks, -1 above
// MAX_DIAG_BLOCKS), block prefix sums over the lattices, and the two launches
// that write each lattice's sums and status word into
// out + m * slot_doubles after t batch steps.
size_t batch_diag_bytes();
int batch_fill_diag(const HostParams &h, double *partial, void *out);
cudaError_t launch_batch_diag(int storage, const void *desc, const void *bdiag, const int *bprefix, int n, int total,
                              unsigned long long t, double *out, int slot_doubles, cudaStream_t s);
// Message for lb_last_error(NULL) on this thread.
void set_global_error(const char *msg);
Launch default_launch(const HostParams &p);

}  // namespace lbk
