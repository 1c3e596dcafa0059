// One-level restricted additive Schwarz on the GPU: set-up tables, ILU(0)
// factorisation and the level-scheduled subdomain solves (Section 3.1).
#pragma once

#include "common.cuh"

namespace ras {

// One distinct overlapped-box shape: its wavefront (level) schedule is shared
// by every subdomain of that shape.
struct ShapeInfo {
    int bx, by, bz, ncell;
    int nlev, nchunk;
    int lvl_off;     // into lvl_tab: nlev + 1 level starts
    int cell_off;    // into cidx_tab: local indices in level order (multiple of 4 aligned)
    int chunk_off;   // into chunk_tab: nchunk + 1 level indices (blocks: 4-integer steps)
    int maxw;        // widest level
    // blocks of 2 x 2 cells of a plane (FP32 / BF16 factors; nlev, lvl_off, cell_off, maxw
    // then count blocks): blocks along x and y, their number, plane stride and guard in
    // shared memory
    int mx, my, nblk, mp, guard;
};

// One subdomain: overlapped box origin, its shape, owned box (relative to the
// overlapped origin) and the offset of its factor records.
struct SubInfo {
    int e0x, e0y, e0z, shape;
    int ox0, oy0, oz0, ox1, oy1, oz1;
    long long foff;
};

// one subdomain with its shape (one load for the sweeps)
struct BoxInfo {
    SubInfo sub;
    ShapeInfo shape;
};

struct Ras1 {
    int nx, ny, nz, N;
    int nsub = 0, nshape = 0;
    int prec = 64;          // 64, 32, 16
    int rec_bytes = 32;     // bytes of one factor record (4 values)
    int block = 128;        // threads per subdomain CTA
    int chunk_cells = 1024; // max cells per staged chunk (the schedule asked for)
    int launch = 128;       // threads per CTA of the sweeps
    int sched = 0;          // counts the changes of the schedule
    int ycap = 0, lcap = 0; // smem capacities of the sweeps (cells or blocks, levels + 1)
    int gcap = 0;           // zero guard band on each side of their vector
    int ycap_cells = 0, lcap_cells = 0, gcap_cells = 0;   // the same cell by cell
    int maxw = 0;           // widest level of cells over the box shapes
    int maxwb = 0;          // widest level of the sweeps (cells or blocks)
    int bxy = 1;            // largest box plane (cells)
    int fac_block = 32;     // threads per box of the factorisation (its pencils)
    std::vector<int> h_lvl; // host copy of the level starts (rescheduling)
    size_t smem_apply = 0, smem_factor = 0;
    size_t ring_bytes = 0;  // record ring of the sweeps in blocks
    long long nrec = 0;     // factor records (incl. padding)
    long long ncell_total = 0;  // sum of overlapped cells
    long long nown = 0;
    SubInfo *d_subs = nullptr;
    BoxInfo *d_boxes = nullptr;
    ShapeInfo *d_shapes = nullptr;
    int *d_lvl = nullptr, *d_chunk = nullptr;
    int *d_cidx = nullptr;  // level-ordered local index of each cell (block)
    void *d_fwd = nullptr, *d_bwd = nullptr;
    int *d_err = nullptr;   // the factors' and the sweeps' error word, then one for the handle's coarse level
    // AS (kind 0) and right-RAS (kind 2): each box's whole solution goes to zbuf
    // (at the box's record offset), then every cell sums the boxes covering it
    int kind = 1;
    double *zbuf = nullptr;
    int *d_clo[3] = {}, *d_chi[3] = {}; // per axis and coordinate: first / last part covering it
    int parts[3] = {1, 1, 1};
    std::vector<SubInfo> subs;
    std::vector<ShapeInfo> shapes;
    int kernel = 0;   // ras_set_apply_kernel's value (0 and 1 run the same sweeps)
};

int ras1_setup(Ras1 &R, int nx, int ny, int nz, int px, int py, int pz, int overlap, int prec,
               int kind = 1);
void ras1_free(Ras1 &R);
// numeric ILU(0) of every A_i = R_i^delta A (R_i^delta)^T; no synchronisation
int ras1_factor(Ras1 &R, const Stencil7 &A, cudaStream_t st);
// the status in the error word d_err[0]: a zero or non-finite pivot, a sweep's wait that ran out
int ras1_status(int word);
// z = M^{-1} r (accumulate = 0) or z += M^{-1} r (accumulate = 1), with
// M^{-1} = sum_i (R_i^0)^T A_i^{-1} R_i^delta (left-RAS, kind 1),
// sum_i (R_i^delta)^T A_i^{-1} R_i^delta (AS, kind 0) or
// sum_i (R_i^delta)^T A_i^{-1} R_i^0 (right-RAS, kind 2)
int ras1_apply(Ras1 &R, const double *r, double *z, int accumulate, cudaStream_t st);
// new chunk size / threads per box for the subdomain solves (0: default); synchronous
int ras1_set_schedule(Ras1 &R, int chunk_cells, int threads);
// the kernel choice 0 or 1 (RAS_EINVAL if not eligible); both run the same sweeps
int ras1_set_kernel(Ras1 &R, int kernel);

// parameters of one handle's apply kernel
struct ApplyParams {
    const SubInfo *subs;
    const ShapeInfo *shapes;
    const BoxInfo *boxes;
    const int *lvl, *chunk;
    const int *cidx;          // per shape, level order: local index of each cell (block)
    const unsigned char *fwd, *bwd;
    const double *r;
    double *z;
    int nx, ny, nz;
    int accumulate;
    int ycap, gcap, lcap, chunk_cells;
    const int4 *steps;   // sweeps in blocks: per shape and step (schedule_tables)
    int *err;            // a wait that ran out
    int polls;           // its poll limit (0: the default)
    int kind;        // 1 left-RAS; 0 AS, 2 right-RAS (box solutions to zbuf)
    double *zbuf;
};
// Left-RAS (kind 1) of several handles in one launch: a persistent kernel whose CTAs
// take boxes (handle, box) from a work queue, largest first (see k_ras_apply_batch)
struct BatchApply {
    const ApplyParams *inst;          // [handles] device copies of the handles' parameters
    const int *box_inst, *box_local;  // [CTAs] handle and box of every CTA
    const long long *off;             // [handles] offset of the handle's cells in r and z
    const unsigned char *active;      // [handles] 0: skip
    const double *r;
    double *z;
    int accumulate;                   // z += (instead of =) the correction
    int nitems;                       // boxes in the work queue (box_inst / box_local order)
    int *qcount;                      // device work counter, cleared before each launch
    int polls;                        // poll limit of the sweeps' waits (0: the default)
};
// the poll limit of the sweeps' waits for the next launch (barrier_polls)
int ras1_polls();
// makes the sweeps that take it ready to launch (before a capture)
int ras1_limit_ready(int prec);
void ras1_apply_params(const Ras1 &R, ApplyParams &P);
// parameters of one handle's ILU(0) factorisation kernel on operator A
struct FactorParams {
    const SubInfo *subs;
    const ShapeInfo *shapes;
    const int *lvl;
    Stencil7 A;
    void *fwd, *bwd;
    int nx, ny, nz;
    int *err;
};
void ras1_factor_params(const Ras1 &R, const Stencil7 &A, FactorParams &P);
// the ILU(0) factorisations of several handles in one launch: CTA b factors box
// d_box_local[b] of handle d_box_inst[b] (d_inst: device copies of the handles'
// parameters); no synchronisation (a zero pivot is left in the handle's error word)
int ras1_factor_batch(const FactorParams *d_inst, const int *d_box_inst, const int *d_box_local,
                      const unsigned char *d_active, int nbox, int prec, int block, size_t smem, cudaStream_t st);
// persistent launch of `grid` CTAs over the B.nitems boxes of the work queue
int ras1_apply_batch(const BatchApply &B, int grid, int prec, int block, size_t smem, cudaStream_t st);
// CTAs of the batched solve that are co-resident on the device (its persistent grid)
int ras1_batch_grid(int prec, int block, size_t smem, int nitems, int *grid);
double ras1_bytes(const Ras1 &R);

}  // namespace ras
