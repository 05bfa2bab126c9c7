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

// Whether the sums of the forces of a long call's steps are left to one launch every kForceSteps steps; with many
// groups (grids of a thousand nodes a side and more) the sum is no part of a step worth saving.
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
