// runtime.h -- host-side helpers shared by the C-ABI translation units (not part of the ABI).
#pragma once

#include <cuda.h>
#include <stddef.h>
#include <stdint.h>

#include <vector>

#include "lbm.h"
#include "pbatch.cuh"

namespace lbm {

struct HostLattice {
    int Q = 0, R = 0;
    double theta = 0;
    int c[37][2] = {};
    double w[37] = {};
    int opp[37] = {};
};

bool host_lattice(int Q, HostLattice& H);
size_t storage_size(int storage);
int set_error(int code, const char* fmt, ...);
void clear_error();
const char* last_error();
// A fluid node with blocked links: its offset in the unpadded grid (y nx + x) and link masks (bit i:
// link i pulls from, or passes through, a solid node of the body, or of a static wall).
struct LinkNode {
    size_t node;
    uint64_t body, wall;
};
double drive_value(int drive, double u0, double omega, long n);
int fit_sincos(const double* fx, size_t stride, long n0, long n1, double omega, double coef[3]);

// Kernel of regularized D2Q37 with 16-bit storage, by the grid's sides: one node per thread on 32 x 4 tiles (2), or
// two neighbouring nodes per thread, direct (31) or staged (32).  A block of 31 covers 64 nodes of a row, where
// an odd number of 32-node columns, one, three or five, leaves more idle than two nodes per thread gain (us a step, 2 /
// 31: 32 x 9375 10.7 / 17.0, 96 x 3125 9.8 / 11.8, 160 x 1875 9.8 / 10.4; 224 x 1339 9.8 / 9.8, 64 x 4687 9.7 / 9.1,
// 1024 x 292 9.7 / 8.0), and a small grid has too few warps of two nodes: without boundary nodes 64^2 2.2 / 3.0,
// 256 x 512 4.7 / 6.0, 384^2 5.6 / 5.9, 448^2 7.0 / 6.4; with them, whose own latency hides the others', plates of
// 64^2 3.1 / 3.2, 181^2 3.8 / 4.5, 256^2 4.7 / 4.3.  The staged tiles, 128 wide and direct at the
// seam, pay on wide grids well past the L2, of more than 200 MB (31 / 32: 128 x 23437 87 / 102, 384 x 7812 81 / 85,
// 640 x 4687 78 / 76, 2048 x 1464 76 / 70).  In a batch, which keeps the chip full whatever one grid's size, they do
// unless the grid is narrow and tall (16 instances of 256 x 600 31 / 32: 74 / 89; 24 of 384^2 104 / 104, 16 of 512^2
// 116 / 111); and kernels with and without staging do not share an SM well (16 grids of 288 to 864 a side all 32:
// 137 us a step, those below 448 on 31: 147), so a square grid takes 32 whatever its size.
inline int pair_variant(int nx, int ny, bool boundary, size_t bytes, bool batch) {
    const int c = (nx + 31) / 32;
    if (batch && (nx >= 448 || ny < 2 * nx)) return 32;
    if (c % 2 == 1 && c < 7) return 2;
    if (batch) return 31;
    if ((size_t)nx * ny <= (size_t)(boundary ? 40000 : 160000)) return 2;
    return nx >= 640 && bytes > (size_t)200000000 ? 32 : 31;
}

// What another translation unit may read of a simulation: its layout, tile shape and the launch
// parameters of its step kernel (device pointers to its geometry arrays included).
struct SimView {
    int device, Q, storage, collision, nx, ny, pitch, bx, by, drive;
    int body_row0, body_row1;  // rows that hold nodes with body links
    int nlf;                   // force groups of the two-buffer bounce-back step (noalloc)
    int slots;                 // tiles with body links as lbm_step_noalloc counts them (0: not more than it accepts)
    double u0, omega;
    InstDev inst;
    void* buf[2];
    int cur;
    long steps_done;
    double2* history;
    size_t esize, n_fluid;
    int aa;  // in-place single buffer (buf[1] is null)
    int variant;
    int ntiles;
    const CUtensorMap* maps;  // staged variants: load boxes of buf[0], buf[1]
};
SimView sim_view(const lbm_sim* s);

// What a geometry's device lists hold: boundary nodes, those of them with body links, and body links (bounce-back
// walls only); of a checked geometry.
struct SolidLists {
    size_t nb, nbf, nfl;
};
SolidLists solid_lists(const HostLattice& H, int nx, int ny, const lbm_geometry& g);
int check_geometry(const HostLattice& H, int nx, int ny, const lbm_geometry& g);

// Whether the sums of the forces of a long call's steps are left to one launch every kForceSteps steps.  Up to 1024
// groups, so that a simulation holds at most 1 MB of partials; wide flat plates, whose steps are short, would gain
// beyond (40 rows of 4992 nodes, 1014 groups, 7.8 us a step FP32; of 5088, not deferred, 10.9).
inline bool defers_forces(bool may_defer, bool aa, int groups) { return may_defer && !aa && groups > 0 && groups <= 1024; }

// Device memory of a simulation, by offsets in one block: node classes, then the uploaded lists (boundary nodes,
// their links, body links), then what starts at zero (ticket, error word, group partials -- of two steps, which
// the in-place even step records, or of the steps summed at once -- and history).  Populations of up to 64 MB join
// it; larger ones are allocated by themselves.  (An allocation or its release costs about 30 us, 100 us and
// more above 256 MB; a grid of 256^2 took ten of them.)
struct SimLayout {
    size_t nodes, links, flinks, zero, history, pops;
    size_t pop, nbuf;              // bytes of a population buffer, and buffers
    bool together;
    size_t bytes() const { return pops + (together ? nbuf * pop : 0); }  // of the block
};
SimLayout sim_layout(const HostLattice& H, int nx, int ny, const lbm_geometry& g, const SolidLists& n, size_t history,
                     bool may_defer);

// lbm_create for a batch: the force history holds `history` steps at once, forces are not deferred, and
// admit(context, device bytes, force groups) is asked before anything is allocated (a code it returns is passed on).
struct CreatePlan {
    size_t history;
    int (*admit)(void* context, size_t bytes, int groups);
    void* context;
};
int sim_create(int lattice, int nx, int ny, double tau, double omega, const lbm_geometry* geom, const CreatePlan* plan,
               lbm_sim** out);

// Make the links by node that the tile kernels read (may allocate).
int sim_tile_links(lbm_sim* s);
// Store plain scaled deviations (no uniform-stream offset); only before the first step.
void sim_disable_stream_offset(lbm_sim* s);
// Record that `steps` steps were run on the simulation's buffers by another launcher.
void sim_advance(lbm_sim* s, long steps);
// The per-step constants (drive, 16-bit stream offsets) of the simulation's next `count` steps,
// exactly as lbm_step would set them.
void sim_step_constants(const lbm_sim* s, long count, StepConst* out);

}  // namespace lbm
