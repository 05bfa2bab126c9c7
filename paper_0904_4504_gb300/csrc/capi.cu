// capi.cu -- host runtime and C ABI of liblbm.so (declarations and contracts in include/lbm.h).
//
// The runtime rasterizes the geometry, classifies nodes and blocked links once, owns the device
// buffers of a simulation, tabulates the drive in FP64, launches the fused step kernel once per
// time step on the simulation's stream, and reads back the FP64 force history.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "deferred.h"
#include "lbm.h"
#include "runtime.h"
#include "pbatch.cuh"

namespace lbm {

void* find_tma_launcher_q9(int storage, int coll, int variant);
void* find_q9v_launcher(int storage, int coll, int variant);
void tma_box_q9(int storage, int bx, int* bw, int* pad);

// D2Q37 launch tables, one translation unit per storage type (step_q37_inst.cuh).
#define LBM_Q37_DECLS(SFX)                                          \
    void* find_launcher_q37_##SFX(int coll);                        \
    PbKernel find_pbatch_q37_##SFX(int coll, int variant);          \
    void* find_launcher_q37_##SFX##_ds(int coll);                   \
    void* find_occ_launcher_q37_##SFX(int coll, int variant);       \
    void* find_tma_launcher_q37_##SFX(int coll, int variant);       \
    void tma_box_q37_##SFX(int bx, int* bw, int* pad);
LBM_Q37_DECLS(f64)
LBM_Q37_DECLS(f32)
LBM_Q37_DECLS(bf16)
LBM_Q37_DECLS(f16)
#undef LBM_Q37_DECLS

struct Q37Table {
    void* (*plain)(int coll);
    PbKernel (*pbatch)(int coll, int variant);
    void* (*plain_ds)(int coll);
    void* (*occ)(int coll, int variant);
    void* (*tma)(int coll, int variant);
    void (*box)(int bx, int* bw, int* pad);
};

static const Q37Table* q37_table(int storage) {
#define LBM_Q37_ROW(SFX)                                                                          \
    {find_launcher_q37_##SFX, find_pbatch_q37_##SFX, find_launcher_q37_##SFX##_ds, find_occ_launcher_q37_##SFX, \
     find_tma_launcher_q37_##SFX, tma_box_q37_##SFX}
    static const Q37Table rows[4] = {LBM_Q37_ROW(f64), LBM_Q37_ROW(f32), LBM_Q37_ROW(bf16), LBM_Q37_ROW(f16)};
#undef LBM_Q37_ROW
    return storage >= ST_F64 && storage <= ST_F16 ? &rows[storage] : nullptr;
}

static TmaStepLaunchFn find_tma_launcher(int Q, int storage, int coll, int variant) {
    void* f = nullptr;
    if (Q == 9) f = find_tma_launcher_q9(storage, coll, variant);
    else if (Q == 37 && q37_table(storage)) f = q37_table(storage)->tma(coll, variant);
    return reinterpret_cast<TmaStepLaunchFn>(f);
}

// Tile of a staged variant (see lbm_set_variant); false for other variants.
static bool variant_tile(int variant, int storage, int* bx, int* by) {
    switch (variant) {
        case 1:
        case 2:
        case 10: *bx = 32; *by = 4; return true;
        case 3: *bx = 32; *by = 8; return true;
        case 4: *bx = 32; *by = 16; return true;
        case 11: *bx = 64; *by = 2; return true;
        case 12: *bx = 64; *by = 4; return true;
        case 13: *bx = 64; *by = 2; return true;
        case 18: *bx = 64; *by = 4; return true;
        case 23: *bx = 64; *by = 2; return true;
        case 24: *bx = 64; *by = 4; return true;
        case 25: *bx = 128; *by = 2; return true;
        case 26:
        case 27: *bx = 64; *by = 3; return true;
        case 28: *bx = 128; *by = 3; return true;
        case 20: *bx = 64; *by = 4; return true;
        case 30: *bx = storage == ST_F32 ? 64 : 128; *by = 4; return true;
        case 31: *bx = 64; *by = 1; return true;
        case 32: *bx = 128; *by = 2; return true;
        case 21: *bx = 64; *by = 2; return true;
        case 22: *bx = 128; *by = 2; return true;
        default: return false;
    }
}

static void tma_box(int Q, int storage, int bx, int* bw, int* pad) {
    *bw = *pad = 0;
    if (Q == 9) tma_box_q9(storage, bx, bw, pad);
    else if (Q == 37 && q37_table(storage)) q37_table(storage)->box(bx, bw, pad);
}

// Tensor map of one population buffer: 3-D (x, y, direction), boxes of bw x by x 1.
static int encode_map(CUtensorMap* map, void* base, int storage, int nx, int ny, int Q, int pitch, int bw, int by) {
    static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    if (!encode) {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess || !fn)
            return set_error(LBM_ECUDA, "cuTensorMapEncodeTiled is not available");
        encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    }
    const size_t es = storage_size(storage);
    CUtensorMapDataType dt = storage == ST_F32   ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                             : storage == ST_F16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16
                             : storage == ST_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                                  : CU_TENSOR_MAP_DATA_TYPE_FLOAT64;
    const cuuint64_t dims[3] = {(cuuint64_t)nx, (cuuint64_t)ny, (cuuint64_t)Q};
    const cuuint64_t strides[2] = {(cuuint64_t)pitch * es, (cuuint64_t)pitch * es * ny};
    const cuuint32_t box[3] = {(cuuint32_t)bw, (cuuint32_t)by, 1};
    const cuuint32_t estr[3] = {1, 1, 1};
    const CUresult r = encode(map, dt, 3, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                              CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_error(LBM_ECUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
    return LBM_OK;
}

void* find_launcher_q9(int storage, int coll);
void* find_launcher_q9_ds(int storage, int coll);
PbKernel find_pbatch_q9(int storage, int coll, int variant);

static void* find_launcher(int Q, int storage, int coll) {
    if (Q == 9) return find_launcher_q9(storage, coll);
    if (Q == 37 && q37_table(storage)) return q37_table(storage)->plain(coll);
    return nullptr;
}

StepLaunchFn find_direct_launcher(int Q, int storage, int coll, int variant) {
    if (variant != 30) return find_occ_launcher(Q, storage, coll, variant);
    return Q == 9 ? reinterpret_cast<StepLaunchFn>(find_q9v_launcher(storage, coll, variant)) : nullptr;
}

StepLaunchFn find_occ_launcher(int Q, int storage, int coll, int variant) {
    if (Q != 37 || !(variant >= 1 && variant <= 4 || variant == 31) || !q37_table(storage)) return nullptr;
    return reinterpret_cast<StepLaunchFn>(q37_table(storage)->occ(coll, variant));
}

bool pdl_enabled() {
    static const bool on = [] {
        const char* e = std::getenv("LBM_PDL");
        return !(e && e[0] == '0');
    }();
    return on;
}

StepLaunchFn find_aa_launcher_q9(int storage, int coll, int phase);
StepLaunchFn find_aa_launcher_q37_wide(int storage, int coll, int phase);
StepLaunchFn find_aa_launcher_q37_half(int storage, int coll, int phase);

StepLaunchFn find_aa_launcher(int Q, int storage, int coll, int phase) {
    if (Q == 9) return find_aa_launcher_q9(storage, coll, phase);
    if (Q == 37) return storage <= ST_F32 ? find_aa_launcher_q37_wide(storage, coll, phase)
                                          : find_aa_launcher_q37_half(storage, coll, phase);
    return nullptr;
}

StepLaunchFn find_step_launcher(int Q, int storage, int coll, int wall) {
    if (wall == 0) return reinterpret_cast<StepLaunchFn>(find_launcher(Q, storage, coll));
    void* f = nullptr;
    if (Q == 9) f = find_launcher_q9_ds(storage, coll);
    else if (Q == 37 && q37_table(storage)) f = q37_table(storage)->plain_ds(coll);
    return reinterpret_cast<StepLaunchFn>(f);
}
PbKernel find_pbatch_kernel(int Q, int storage, int coll, int variant) {
    if (Q == 9) return find_pbatch_q9(storage, coll, variant);
    if (Q == 37 && q37_table(storage)) return q37_table(storage)->pbatch(coll, variant);
    return PbKernel{nullptr, dim3(), 0, 0, 0};
}

// ---------------------------------------------------------------------------------------------
// errors
// ---------------------------------------------------------------------------------------------

static thread_local std::string g_err;

int set_error(int code, const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    g_err = buf;
    return code;
}

void clear_error() { g_err.clear(); }

const char* last_error() { return g_err.c_str(); }

// ---------------------------------------------------------------------------------------------
// lattice tables on the host (same constants as the device, lattice.cuh)
// ---------------------------------------------------------------------------------------------

template <class L>
static void fill_lattice(HostLattice& H) {
    H.Q = L::Q;
    H.R = L::R;
    H.theta = L::theta();
    for (int i = 0; i < L::Q; ++i) {
        H.c[i][0] = cx_of<L>(i);
        H.c[i][1] = cy_of<L>(i);
        H.w[i] = w_of<L>(i);
        H.opp[i] = opp_of<L>(i);
    }
}

bool host_lattice(int Q, HostLattice& H) {
    if (Q == 9) { fill_lattice<D2Q9>(H); return true; }
    if (Q == 37) { fill_lattice<D2Q37>(H); return true; }
    return false;
}

size_t storage_size(int storage) {
    switch (storage) {
        case ST_F64: return 8;
        case ST_F32: return 4;
        case ST_BF16:
        case ST_F16: return 2;
        default: return 0;
    }
}

// ---------------------------------------------------------------------------------------------
// geometry: labels, node classes and blocked links
// ---------------------------------------------------------------------------------------------

static uint8_t max_label(const uint8_t* m, int n) {
    uint8_t v = 0;
    for (int x = 0; x < n; ++x) v = std::max(v, m[x]);
    return v;
}

int check_geometry(const HostLattice& H, int nx, int ny, const lbm_geometry& g) {
    switch (g.kind) {
        case LBM_GEOM_NONE:
            return LBM_OK;
        case LBM_GEOM_PLATE:
            if (ny < 2 * H.R + 1) return set_error(LBM_EINVAL, "plate needs ny >= %d", 2 * H.R + 1);
            return LBM_OK;
        case LBM_GEOM_BEAM:
            if (g.lx < 1 || g.ly < 1 || g.lx > nx - 2 * H.R || g.ly > ny - 2 * H.R)
                return set_error(LBM_EINVAL, "beam %dx%d does not fit a %dx%d box with a %d-node gap", g.lx, g.ly,
                                 nx, ny, H.R);
            return LBM_OK;
        case LBM_GEOM_MASK:
            if (!g.mask) return set_error(LBM_EINVAL, "LBM_GEOM_MASK needs a mask");
            for (int y = 0; y < ny; ++y) {
                if (max_label(g.mask + (size_t)y * nx, nx) <= LBM_WALL) continue;
                for (size_t k = (size_t)y * nx;; ++k)
                    if (g.mask[k] > LBM_WALL) return set_error(LBM_EINVAL, "mask label %d at %zu", g.mask[k], k);
            }
            return LBM_OK;
        default:
            return set_error(LBM_EINVAL, "unknown geometry kind %d", g.kind);
    }
}

// Labels of row y of a checked geometry; returns false (row not written) if the row is all fluid.
bool label_row(const HostLattice& H, int nx, int ny, const lbm_geometry& g, int y, uint8_t* row) {
    switch (g.kind) {
        case LBM_GEOM_PLATE:
            // (the static wall is written last: on the smallest boxes the two do not meet)
            if (y >= H.R && y < ny - H.R) return false;
            std::fill_n(row, nx, (uint8_t)(y >= ny - H.R ? LBM_WALL : LBM_BODY));
            return true;
        case LBM_GEOM_BEAM: {
            const int x0 = (nx - g.lx) / 2, y0 = (ny - g.ly) / 2;
            if (y < y0 || y >= y0 + g.ly) return false;
            std::fill_n(row, nx, (uint8_t)0);
            std::fill_n(row + x0, g.lx, (uint8_t)LBM_BODY);
            return true;
        }
        case LBM_GEOM_MASK: {
            const uint8_t* m = g.mask + (size_t)y * nx;
            if (!max_label(m, nx)) return false;
            std::copy_n(m, nx, row);
            return true;
        }
        default:
            return false;
    }
}

// Node classes and blocked links of a geometry.  Only rows within R of a row holding a solid node can
// have solid or boundary nodes; the others are bulk fluid and are not visited (a large domain around a
// small body is mostly such rows).
struct GeomScan {
    std::vector<int> rows;          // the visited rows, increasing
    std::vector<uint8_t> cls;       // [rows][nx] NodeClass
    std::vector<LinkNode> links;    // boundary nodes in increasing node order
    size_t n_fluid = 0;
};

static int gcd_int(int a, int b) {
    while (b) {
        const int t = a % b;
        a = b;
        b = t;
    }
    return a;
}

// For every fluid node, the links whose pull source, or a lattice node strictly between source and
// node, is solid; the first solid node met walking back from the node decides body or wall.
void scan_geometry(const HostLattice& H, int nx, int ny, const lbm_geometry& g, GeomScan& out) {
    const int R = H.R;
    auto wrap = [](int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); };  // nx, ny > R
    // labels of the rows holding a solid, the solids within R along x of their nodes, and whether a
    // row's labels are all the same
    struct Row {
        int y;
        bool uniform;
        int lo, hi;                 // columns [lo, hi) outside of which nothing is near a solid of this row
    };
    std::vector<Row> solid;
    std::vector<int> at(ny, -1);    // y -> index in solid
    std::vector<uint8_t> lab, near, row(nx);
    size_t n_solid = 0;
    for (int y = 0; y < ny; ++y) {
        if (!label_row(H, nx, ny, g, y, row.data())) continue;
        at[y] = (int)solid.size();
        const bool uniform = std::all_of(row.begin(), row.end(), [&](uint8_t l) { return l == row[0]; });
        lab.insert(lab.end(), row.begin(), row.end());
        near.resize(lab.size(), 0);
        uint8_t* O = near.data() + near.size() - nx;
        for (int x = 0; x < nx; ++x) {
            if (!row[x]) continue;
            ++n_solid;
            for (int d = -R; d <= R; ++d) O[wrap(x + d, nx)] = 1;
        }
        const int lo = (int)(std::find(O, O + nx, 1) - O);
        int hi = nx;
        while (hi > lo && !O[hi - 1]) --hi;
        solid.push_back(Row{y, uniform, lo, hi});
    }
    out.n_fluid = (size_t)nx * ny - n_solid;
    out.rows.clear();
    out.cls.clear();
    out.links.clear();
    // nodes of a link walking back from its node, nearest first: (x, y) steps
    struct Walk {
        int n, dx[3], dy[3];
    };
    std::vector<Walk> walk(H.Q);
    for (int i = 1; i < H.Q; ++i) {
        const int cx = H.c[i][0], cy = H.c[i][1], n = gcd_int(std::abs(cx), std::abs(cy));
        walk[i].n = n;
        for (int k = 1; k <= n; ++k) {
            walk[i].dx[k - 1] = -k * cx / n;
            walk[i].dy[k - 1] = -k * cy / n;
        }
    }
    std::vector<uint8_t> visit(ny, 0);
    for (const Row& r : solid)
        for (int d = -R; d <= R; ++d) visit[wrap(r.y + d, ny)] = 1;
    for (int y = 0; y < ny; ++y) {
        if (!visit[y]) continue;
        out.rows.push_back(y);
        const size_t base = out.cls.size();
        out.cls.resize(base + nx, NODE_BULK);
        uint8_t* cls = out.cls.data() + base;
        const uint8_t* L[7];        // label rows y - R .. y + R (null: all fluid)
        bool uniform = true;
        int lo = nx, hi = 0;
        std::fill(row.begin(), row.end(), 0);
        for (int d = -R; d <= R; ++d) {
            const int k = at[wrap(y + d, ny)];
            L[d + R] = k < 0 ? nullptr : lab.data() + (size_t)k * nx;
            if (k < 0) continue;
            uniform = uniform && solid[k].uniform;
            const uint8_t* I = near.data() + (size_t)k * nx;
            for (int x = solid[k].lo; x < solid[k].hi; ++x) row[x] |= I[x];
            lo = std::min(lo, solid[k].lo);
            hi = std::max(hi, solid[k].hi);
        }
        uint64_t b = 0, w = 0;
        for (int x = lo; x < hi; ++x) {
            if (L[R] && L[R][x]) {
                cls[x] = NODE_SOLID;
                continue;
            }
            if (!row[x]) continue;
            if (x == 0 || !uniform) {  // the nodes of a row among uniform rows all have the same links
                b = w = 0;
                for (int i = 1; i < H.Q; ++i)
                    for (int k = 0; k < walk[i].n; ++k) {
                        const uint8_t* l = L[walk[i].dy[k] + R];
                        const uint8_t v = l ? l[wrap(x + walk[i].dx[k], nx)] : 0;
                        if (v) {
                            (v == LBM_BODY ? b : w) |= 1ull << i;
                            break;
                        }
                    }
            }
            if (b | w) {
                cls[x] = NODE_BOUNDARY;
                out.links.push_back(LinkNode{(size_t)y * nx + x, b, w});
            }
        }
    }
}

// Geometry-only part of the momentum exchange (the rest populations w_i rho0 bounced on body
// links, count[i] of direction i), -sum over body links of c_i 2 w_i rho0, and the moving-wall part per unit wall velocity,
// -sum of c_i c_ix 2 w_i rho0 / theta.
void constant_force(const HostLattice& H, const std::vector<size_t>& count, double rho0, double& fx, double& fy,
                    double& mx, double& my) {
    fx = fy = mx = my = 0.0;
    for (int i = 1; i < H.Q; ++i) {
        const double n = (double)count[i] * 2.0 * H.w[i] * rho0;
        fx -= H.c[i][0] * n;
        fy -= H.c[i][1] * n;
        mx -= H.c[i][0] * H.c[i][0] * n / H.theta;
        my -= H.c[i][1] * H.c[i][0] * n / H.theta;
    }
}

// Tiles of bx x by nodes that hold body links.
static int body_tiles(int nx, int bx, int by, const std::vector<LinkNode>& links) {
    std::vector<uint8_t> row((nx + bx - 1) / bx, 0);  // of the current row of tiles (links are in node order)
    int n = 0, y = 0;
    size_t first = 0;                                  // first node of row y
    for (const LinkNode& ln : links) {
        if (!ln.body) continue;
        for (; ln.node - first >= (size_t)nx; first += nx)
            if (++y % by == 0) std::fill(row.begin(), row.end(), 0);
        uint8_t& seen = row[(unsigned)(ln.node - first) / (unsigned)bx];
        n += !seen;
        seen = 1;
    }
    return n;
}

double drive_value(int drive, double u0, double omega, long n) {
    const double t = (double)n + 0.5;
    return drive == LBM_DRIVE_WALL ? u0 * std::sin(omega * t) : u0 * omega * std::cos(omega * t);
}

// ---------------------------------------------------------------------------------------------
// fit (FP64 least squares on {sin, cos, 1})
// ---------------------------------------------------------------------------------------------

int fit_sincos(const double* fx, size_t stride, long n0, long n1, double omega, double coef[3]) {
    double M[3][4] = {{0}};
    for (long n = n0; n < n1; ++n) {
        const double t = (double)n + 0.5;
        const double b[3] = {std::sin(omega * t), std::cos(omega * t), 1.0};
        const double y = fx[(size_t)n * stride];
        for (int r = 0; r < 3; ++r) {
            for (int c = 0; c < 3; ++c) M[r][c] += b[r] * b[c];
            M[r][3] += b[r] * y;
        }
    }
    for (int c = 0; c < 3; ++c) {  // Gaussian elimination with partial pivoting
        int p = c;
        for (int r = c + 1; r < 3; ++r)
            if (std::fabs(M[r][c]) > std::fabs(M[p][c])) p = r;
        if (std::fabs(M[p][c]) < 1e-300) return set_error(LBM_ERANGE, "fit window too short");
        if (p != c)
            for (int k = 0; k < 4; ++k) std::swap(M[p][k], M[c][k]);
        for (int r = 0; r < 3; ++r) {
            if (r == c) continue;
            const double f = M[r][c] / M[c][c];
            for (int k = c; k < 4; ++k) M[r][k] -= f * M[c][k];
        }
    }
    for (int r = 0; r < 3; ++r) coef[r] = M[r][3] / M[r][r];
    return LBM_OK;
}

}  // namespace lbm

using namespace lbm;

// ---------------------------------------------------------------------------------------------
// the simulation object
// ---------------------------------------------------------------------------------------------

struct lbm_sim {
    int device = 0;
    int Q = 0, nx = 0, ny = 0, pitch = 0;
    double tau = 0, omega = 0;
    lbm_geometry geom{};
    HostLattice lat{};
    size_t esize = 0;
    std::vector<uint8_t> labels;       // LBM_GEOM_MASK: a copy; else kept by the first call that needs them (labels_of)
    std::vector<LinkNode> link_nodes;  // boundary nodes and their link masks
    size_t n_fluid = 0, n_boundary = 0;
    double fconst[2] = {0, 0}, fmov[2] = {0, 0};
    int nbf = 0;                       // boundary nodes with body links, first and last row of them
    int body_row0 = 0, body_row1 = -1;
    int link_groups = 0;               // force groups of the two-buffer step
    // device memory: one block for everything small (and the populations, where they are small too)
    unsigned char* d_block = nullptr;
    void* buf[2] = {nullptr, nullptr};
    bool own_buf = false;              // the populations have allocations of their own
    double2* d_history = nullptr;
    bool own_history = false;          // the history has outgrown the block
    ulonglong2* d_links = nullptr;     // [ny][pitch] links by node: tile kernels only (ensure_links)
    int* d_err = nullptr;
    size_t cap = 0;
    size_t device_bytes = 0;
    size_t h2d_bytes = 0, d2h_bytes = 0;  // host<->device traffic over the simulation's life
    // state
    long steps_done = 0;
    int cur = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int bx = 32, by = 4, ntx = 0, ntiles = 0;
    int slots = 0, slots_bx = 0, slots_by = 0;  // count_slots
    int plain_bx = 32, plain_by = 4;   // tile of the plain kernel (lbm_set_tile)
    int variant = 0;                   // 0 plain kernel, else a staged variant (lbm_set_variant)
    bool stream_off = false;           // 16-bit body frame: store h - H(U(n)), see InstDev
    double U_stream = 0.0;             // U(n) = sum_{k<n} g(k + 1/2) for n = steps_done
    StepLaunchFn launch = nullptr;     // plain step in use (variant 0, or an occupancy variant 1-2)
    StepLaunchFn launch_default = nullptr;
    TmaStepLaunchFn tma_launch = nullptr;
    bool aa = false;                   // in-place single buffer (LBM_LAYOUT_AA)
    StepLaunchFn aa_launch[2] = {nullptr, nullptr};  // even (pull-push) and odd (local) steps
    CUtensorMap maps[2];               // staged variants: load boxes of buffer k
    CUtensorMap store_maps[2];         // variants 13, 14: the tile's own box in buffer k
    InstDev dev{};

    // Steps run in longer calls leave the sum of their forces to one launch every kForceSteps steps; with many
    // groups (grids of a thousand nodes a side and more) the sum is no part of a step worth saving.
    int lost_forces = 0;               // steps that ran and whose forces could not be summed
    bool may_defer = true;             // (a batch runs its instances step by step)
    bool defers_forces() const { return lbm::defers_forces(may_defer, aa, dev.ngroups); }
};

namespace {

#define CUDA_TRY(expr)                                                                           \
    do {                                                                                         \
        cudaError_t e_ = (expr);                                                                 \
        if (e_ != cudaSuccess) {                                                                 \
            return set_error(e_ == cudaErrorMemoryAllocation ? LBM_ENOMEM : LBM_ECUDA, "%s: %s", \
                             #expr, cudaGetErrorString(e_));                                     \
        }                                                                                        \
    } while (0)

template <class T>
int dev_alloc(lbm_sim* s, T** p, size_t count) {
    *p = nullptr;
    if (count == 0) count = 1;
    CUDA_TRY(cudaMalloc((void**)p, count * sizeof(T)));
    s->device_bytes += count * sizeof(T);
    return LBM_OK;
}

void free_sim(lbm_sim* s) {
    if (!s) return;
    if (s->stream) cudaStreamSynchronize(s->stream);
    if (s->own_buf) {
        cudaFree(s->buf[0]);
        cudaFree(s->buf[1]);
    }
    if (s->own_history) cudaFree(s->d_history);
    cudaFree(s->d_links);
    cudaFree(s->d_block);
    if (s->own_stream && s->stream) cudaStreamDestroy(s->stream);
    delete s;
}

// The labels the simulation runs with: into a caller's buffer (which allocates nothing), and kept.
void fill_labels(const lbm_sim* s, unsigned char* out) {
    if (!s->labels.empty()) {
        std::copy(s->labels.begin(), s->labels.end(), out);
        return;
    }
    for (int y = 0; y < s->ny; ++y) {
        unsigned char* row = out + (size_t)y * s->nx;
        if (!label_row(s->lat, s->nx, s->ny, s->geom, y, row)) std::fill_n(row, s->nx, (unsigned char)0);
    }
}

const std::vector<uint8_t>& labels_of(lbm_sim* s) {
    if (s->labels.empty()) {
        std::vector<uint8_t> lab((size_t)s->nx * s->ny);
        fill_labels(s, lab.data());
        s->labels.swap(lab);
    }
    return s->labels;
}

// Links by node (InstDev::links), which the tile kernels read.
__global__ void scatter_links(const uint2* nodes, const ulonglong2* links, int n, int pitch, ulonglong2* out) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) out[(size_t)nodes[k].y * pitch + nodes[k].x] = links[k];
}

int ensure_links(lbm_sim* s) {
    if (s->d_links) return LBM_OK;
    const size_t plane = (size_t)s->ny * s->pitch;
    int rc = dev_alloc(s, &s->d_links, plane);
    if (rc) return rc;
    CUDA_TRY(cudaMemsetAsync(s->d_links, 0, plane * sizeof(ulonglong2), s->stream));
    if (s->dev.nb > 0) scatter_links<<<(s->dev.nb + 127) / 128, 128, 0, s->stream>>>(s->dev.bnodes, s->dev.blinks, s->dev.nb, s->pitch, s->d_links);
    CUDA_TRY(cudaGetLastError());
    CUDA_TRY(cudaStreamSynchronize(s->stream));
    s->dev.links = s->d_links;
    return LBM_OK;
}

// Tiles with body links, which lbm_step_noalloc accepts up to LBM_NOALLOC_MAX_SLOTS of: tiles of the
// simulation's shape, but of 32 x 4 nodes for the kernels of neighbouring nodes that lbm_create chooses by itself
// (30 with FP32, 31, 32), so that its choice decides nothing.  Counted only where the nodes with body links are
// more than that, here and not in the step.
void count_slots(lbm_sim* s) {
    const bool own = s->variant != 31 && s->variant != 32 && !(s->variant == 30 && s->geom.storage == LBM_STORE_F32);
    const int bx = own ? s->bx : 32, by = own ? s->by : 4;
    if (s->nbf <= LBM_NOALLOC_MAX_SLOTS || (bx == s->slots_bx && by == s->slots_by)) return;
    s->slots = body_tiles(s->nx, bx, by, s->link_nodes);
    s->slots_bx = bx;
    s->slots_by = by;
}

// Tiles of the current tile shape.
int setup_tiles(lbm_sim* s) {
    s->ntx = (s->nx + s->bx - 1) / s->bx;
    s->ntiles = s->ntx * ((s->ny + s->by - 1) / s->by);
    s->dev.ntx = s->ntx;
    s->dev.ntiles = s->ntiles;
    count_slots(s);
    return LBM_OK;
}

// The body's links (InstDev::flinks), sorted by direction, then node.
void fill_flinks(const lbm_sim* s, const std::vector<size_t>& count, unsigned char* host) {
    const size_t plane = (size_t)s->ny * s->pitch;
    double2* cw = reinterpret_cast<double2*>(host);
    std::vector<size_t> at(s->Q + 1, 0);
    for (int i = 0; i < s->Q; ++i) {
        cw[i] = make_double2(s->lat.c[i][0] * s->lat.w[i], s->lat.c[i][1] * s->lat.w[i]);
        at[i + 1] = at[i] + count[i];
    }
    uint2* list = reinterpret_cast<uint2*>(host + kFLinkTable);
    for (const LinkNode& ln : s->link_nodes) {
        const size_t idx = ln.node / (size_t)s->nx * s->pitch + ln.node % (size_t)s->nx;
        for (uint64_t m = ln.body; m; m &= m - 1) {
            const int i = __builtin_ctzll(m);
            list[at[i]++] = make_uint2((unsigned)(s->lat.opp[i] * plane + idx), (unsigned)(i | (s->lat.c[i][0] + 3) << 8));
        }
    }
}

// Make room for the force history of `need` steps.  Everything goes through the simulation's stream: its steps
// are ordered with that stream only, and a clear on the default stream could wait behind other work there and
// come after them.
int ensure_capacity(lbm_sim* s, size_t need) {
    if (need <= s->cap) return LBM_OK;
    size_t cap = std::max<size_t>(std::max<size_t>(need, 2 * s->cap), 1024);
    double2* hist = nullptr;
    CUDA_TRY(cudaMalloc((void**)&hist, cap * sizeof(double2)));
    // an in-place even step has already written the force of the step after it
    const size_t keep = s->d_history ? std::min(s->cap, (size_t)s->steps_done + (s->aa ? 1 : 0)) : 0;
    cudaError_t e = cudaMemsetAsync(hist + keep, 0, (cap - keep) * sizeof(double2), s->stream);
    if (e == cudaSuccess && keep > 0)
        e = cudaMemcpyAsync(hist, s->d_history, keep * sizeof(double2), cudaMemcpyDeviceToDevice, s->stream);
    // the old history may be freed, and the next steps may run on another stream
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
    if (e != cudaSuccess) {
        cudaFree(hist);
        return set_error(LBM_ECUDA, "force history of %zu steps: %s", need, cudaGetErrorString(e));
    }
    if (s->own_history) cudaFree(s->d_history);
    s->device_bytes += (cap - (s->own_history ? s->cap : 0)) * sizeof(double2);
    s->d_history = hist;
    s->own_history = true;
    s->cap = cap;
    return LBM_OK;
}

// Scaled equilibrium deviation H_i of the uniform stream U x (no rest term), and its moments.
void stream_offset(const lbm_sim* s, double U, float* H, float* HM) {
    const HostLattice& L = s->lat;
    const double b = U * U / L.theta;
    double M[6] = {0, 0, 0, 0, 0, 0};
    for (int i = 0; i < L.Q; ++i) {
        const double a = L.c[i][0] * U / L.theta;
        double poly = a + 0.5 * (a * a - b);
        if (s->geom.eq_order >= 4) poly += (a * a * a - 3 * a * b) / 6.0 + (a * a * a * a - 6 * a * a * b + 3 * b * b) / 24.0;
        const double Hi = s->geom.rho0 * poly / s->dev.s;
        H[i] = (float)Hi;
        const double w = L.w[i], cx = L.c[i][0], cy = L.c[i][1];
        M[0] += w * H[i];
        M[1] += w * cx * H[i];
        M[2] += w * cy * H[i];
        M[3] += w * cx * cx * H[i];
        M[4] += w * cx * cy * H[i];
        M[5] += w * cy * cy * H[i];
    }
    if (HM)
        for (int k = 0; k < 6; ++k) HM[k] = (float)M[k];
}

// The same constants for the kernels: H_i depends on c_ix only, so they get it per c_ix (index
// c_ix + 3), and the moments HM.
void stream_offset_cx(const lbm_sim* s, double U, float* H7, float* HM) {
    float H[37];
    stream_offset(s, U, H, HM);
    for (int k = 0; k < 7; ++k) H7[k] = 0.f;
    for (int i = 0; i < s->lat.Q; ++i) H7[s->lat.c[i][0] + 3] = H[i];
}

// Even and odd parts in c_x of the stored state's offsets, for m = |c_x| (see InstDev).
void stream_offset_eo(const float* H7, float* He, float* Ho) {
    for (int m = 0; m < 4; ++m) {
        He[m] = 0.5f * (H7[3 + m] + H7[3 - m]);
        Ho[m] = 0.5f * (H7[3 + m] - H7[3 - m]);
    }
}

// Switch to a kernel variant other than 0 (two-buffer layout, bounce-back walls).
int use_variant(lbm_sim* s, int variant) {
    if ((variant >= 1 && variant <= 4) || variant == 30 || variant == 31) {
        StepLaunchFn f = find_direct_launcher(s->Q, s->geom.storage, s->geom.collision, variant);
        if (!f) return set_error(LBM_EINVAL, "variant %d is not built for this lattice/storage/collision", variant);
        variant_tile(variant, s->geom.storage, &s->bx, &s->by);
        s->variant = variant;
        s->tma_launch = nullptr;
        s->launch = f;
        return setup_tiles(s);
    }
    int bx, by, bw, pad, rc;
    TmaStepLaunchFn fn = find_tma_launcher(s->Q, s->geom.storage, s->geom.collision, variant);
    if (!fn || !variant_tile(variant, s->geom.storage, &bx, &by))
        return set_error(LBM_EINVAL, "variant %d is not built for this lattice/storage/collision", variant);
    tma_box(s->Q, s->geom.storage, bx, &bw, &pad);
    // (32 leaves the boundary nodes to their own blocks; the others' tiles read their links)
    if (variant != 32 && (rc = ensure_links(s))) return rc;
    // everything that can fail comes before the first change: a staged kernel with the boxes of another would wait
    // for bytes that never come
    CUtensorMap maps[2], store_maps[2];
    for (int k = 0; k < 2; ++k) {
        if ((rc = encode_map(&maps[k], s->buf[k], s->geom.storage, s->nx, s->ny, s->Q, s->pitch, bw, by)))
            return rc;
        if ((rc = encode_map(&store_maps[k], s->buf[k], s->geom.storage, s->nx, s->ny, s->Q, s->pitch, bx, by)))
            return rc;
    }
    std::copy_n(maps, 2, s->maps);
    std::copy_n(store_maps, 2, s->store_maps);
    s->bx = bx;
    s->by = by;
    s->variant = variant;
    s->tma_launch = fn;
    return setup_tiles(s);
}

int check_sim(lbm_sim* s) {
    if (!s) return set_error(LBM_EINVAL, "null simulation");
    CUDA_TRY(cudaSetDevice(s->device));
    return LBM_OK;
}

}  // namespace

namespace lbm {

// Read-only view of a simulation for other translation units of the library.
SimView sim_view(const lbm_sim* s) {
    SimView v;
    v.device = s->device;
    v.Q = s->Q;
    v.storage = s->geom.storage;
    v.collision = s->geom.collision;
    v.nx = s->nx;
    v.ny = s->ny;
    v.pitch = s->pitch;
    v.bx = s->bx;
    v.by = s->by;
    v.nlf = s->link_groups;
    v.slots = s->slots;
    v.body_row0 = s->body_row0;
    v.body_row1 = s->body_row1;
    v.drive = s->geom.drive;
    v.u0 = s->geom.u0;
    v.omega = s->omega;
    v.inst = s->dev;
    v.buf[0] = s->buf[0];
    v.buf[1] = s->buf[1];
    v.cur = s->cur;
    v.steps_done = s->steps_done;
    v.history = s->d_history;
    v.esize = s->esize;
    v.n_fluid = s->n_fluid;
    v.aa = s->aa ? 1 : 0;
    v.variant = s->variant;
    v.ntiles = s->ntiles;
    v.maps = s->maps;
    return v;
}

SimLayout sim_layout(const HostLattice& H, int nx, int ny, const lbm_geometry& g, const SolidLists& n, size_t history,
                     bool may_defer) {
    const auto up256 = [](size_t v) { return (v + 255) / 256 * 256; };
    const size_t es = storage_size(g.storage), align = 128 / es, plane = (nx + align - 1) / align * align * ny;
    const bool aa = g.layout == LBM_LAYOUT_AA, by_links = g.wall_scheme == LBM_SCHEME_BOUNCEBACK;
    const int groups = aa || !by_links ? (int)((n.nbf + 31) / 32) : force_groups((int)n.nfl, force_group_len((int)n.nfl));
    SimLayout at;
    at.pop = up256(plane * H.Q * es);
    at.nbuf = aa ? 1 : 2;
    at.together = at.nbuf * at.pop <= (size_t)64 << 20;
    at.nodes = up256(plane);
    at.links = up256(at.nodes + n.nb * sizeof(uint2));
    at.flinks = up256(at.links + n.nb * sizeof(ulonglong2));
    at.zero = up256(at.flinks + (by_links ? kFLinkTable + n.nfl * sizeof(uint2) : 0));
    const size_t partials = (size_t)std::max(1, groups) * (aa ? 2 : defers_forces(may_defer, aa, groups) ? kForceSteps : 1);
    at.history = up256(at.zero + 256 + partials * sizeof(double2));
    at.pops = up256(at.history + history * sizeof(double2));
    return at;
}

// Counted, for masks; for a plate and a beam from their sides, as an upper bound: a direction's links around a
// rectangle are what each of its gcd(|c_x|, |c_y|) steps shifts out of it.
SolidLists solid_lists(const HostLattice& H, int nx, int ny, const lbm_geometry& g) {
    SolidLists n{0, 0, 0};
    const bool by_links = g.wall_scheme == LBM_SCHEME_BOUNCEBACK;
    if (g.kind == LBM_GEOM_PLATE) {
        n.nb = (size_t)nx * std::min(2 * H.R, ny - 2 * H.R);
        n.nbf = (size_t)nx * std::min(H.R, ny - 2 * H.R);
        for (int i = 1; by_links && i < H.Q; ++i) n.nfl += (size_t)nx * std::max(0, H.c[i][1]);
    } else if (g.kind == LBM_GEOM_BEAM) {
        const size_t lx = g.lx, ly = g.ly;
        n.nb = n.nbf = (lx + 2 * H.R) * (ly + 2 * H.R) - lx * ly;
        for (int i = 1; by_links && i < H.Q; ++i) {
            const int cx = std::abs(H.c[i][0]), cy = std::abs(H.c[i][1]), k = gcd_int(cx, cy);
            n.nfl += k * std::min(lx * ly, cx / k * ly + cy / k * lx - (size_t)(cx / k) * (cy / k));
        }
    } else if (g.kind == LBM_GEOM_MASK) {
        GeomScan scan;
        scan_geometry(H, nx, ny, g, scan);
        n.nb = scan.links.size();
        for (const LinkNode& ln : scan.links) {
            n.nbf += ln.body != 0;
            n.nfl += by_links ? __builtin_popcountll(ln.body) : 0;
        }
    }
    return n;
}

int sim_tile_links(lbm_sim* s) { return ensure_links(s); }

void sim_disable_stream_offset(lbm_sim* s) {
    if (s->steps_done == 0) s->stream_off = false;
    s->dev.stream_off = s->stream_off ? 1 : 0;
}

void sim_advance(lbm_sim* s, long steps) {
    if (s->stream_off)
        for (long k = 0; k < steps; ++k) s->U_stream += drive_value(s->geom.drive, s->geom.u0, s->omega, s->steps_done + k);
    s->steps_done += steps;
    s->cur ^= (int)(steps & 1);
}

void sim_step_constants(const lbm_sim* s, long count, StepConst* out) {
    double U = s->U_stream;
    for (long k = 0; k < count; ++k) {
        StepConst& c = out[k];
        std::memset(&c, 0, sizeof(c));
        c.dv = drive_value(s->geom.drive, s->geom.u0, s->omega, s->steps_done + k);
        if (s->stream_off) {
            float* H = c.H;  // HM[6], Hl[7], Hs[7], He[4], Ho[4]
            stream_offset_cx(s, U, H + 6, H);
            stream_offset_cx(s, U + c.dv, H + 13, nullptr);
            stream_offset_eo(H + 13, H + 20, H + 24);
            U += c.dv;
        }
    }
}

}  // namespace lbm

extern "C" {

const char* lbm_last_error(void) { return last_error(); }

int lbm_geometry_links(int lattice, int nx, int ny, const lbm_geometry* geom, unsigned char* cls,
                       unsigned long long* body, unsigned long long* wall, size_t count, size_t* n_fluid,
                       size_t* n_boundary) {
    clear_error();
    HostLattice H;
    if (!host_lattice(lattice, H)) return set_error(LBM_EINVAL, "unknown lattice %d", lattice);
    if (!geom) return set_error(LBM_EINVAL, "null geometry");
    if (nx < 2 * H.R + 1 || ny < 2 * H.R + 1)
        return set_error(LBM_EINVAL, "grid %dx%d below %d nodes per side", nx, ny, 2 * H.R + 1);
    if ((long long)nx * ny > (1ll << 31) / 2) return set_error(LBM_EINVAL, "grid %dx%d too large", nx, ny);
    const size_t N = (size_t)nx * ny;
    if ((cls || body || wall) && count < N) return set_error(LBM_EINVAL, "outputs hold %zu < %zu nodes", count, N);
    int rc = check_geometry(H, nx, ny, *geom);
    if (rc) return rc;
    GeomScan scan;
    scan_geometry(H, nx, ny, *geom, scan);
    if (cls) {
        std::fill(cls, cls + N, (unsigned char)NODE_BULK);
        for (size_t k = 0; k < scan.rows.size(); ++k)
            std::copy_n(scan.cls.data() + k * nx, nx, cls + (size_t)scan.rows[k] * nx);
    }
    if (body) std::fill(body, body + N, 0ull);
    if (wall) std::fill(wall, wall + N, 0ull);
    for (const LinkNode& ln : scan.links) {
        if (body) body[ln.node] = ln.body;
        if (wall) wall[ln.node] = ln.wall;
    }
    if (n_fluid) *n_fluid = scan.n_fluid;
    if (n_boundary) *n_boundary = scan.links.size();
    return LBM_OK;
}

int lbm_lattice_velocities(int lattice, int* c_xy, double* w, double* theta) {
    HostLattice H;
    if (!host_lattice(lattice, H)) return set_error(LBM_EINVAL, "unknown lattice %d", lattice);
    for (int i = 0; i < H.Q; ++i) {
        if (c_xy) { c_xy[2 * i] = H.c[i][0]; c_xy[2 * i + 1] = H.c[i][1]; }
        if (w) w[i] = H.w[i];
    }
    if (theta) *theta = H.theta;
    return H.Q;
}

int lbm_params_from_tau_omega(int lattice, double tau_omega, double delta_min, int p_min, double* tau,
                              double* omega, int* period) {
    HostLattice H;
    if (!host_lattice(lattice, H)) return set_error(LBM_EINVAL, "unknown lattice %d", lattice);
    if (!(tau_omega > 0.0) || !(delta_min > 0.0) || p_min < 1)
        return set_error(LBM_EINVAL, "need tau_omega > 0, delta_min > 0, p_min >= 1");
    const double pi = 3.14159265358979323846;
    const double need = std::ceil(2.0 * pi * delta_min / std::sqrt(2.0 * H.theta * tau_omega));
    if (!(need < 2e9)) return set_error(LBM_EINVAL, "tau_omega %g needs too many steps per period", tau_omega);
    const int P = std::max(p_min, (int)need);
    const double om = 2.0 * pi / P;
    if (tau) *tau = 0.5 + tau_omega / om;
    if (omega) *omega = om;
    if (period) *period = P;
    return LBM_OK;
}

int lbm_create(int lattice, int nx, int ny, double tau, double omega, const lbm_geometry* geom, lbm_sim** out) {
    return sim_create(lattice, nx, ny, tau, omega, geom, nullptr, out);
}

}  // extern "C"

int lbm::sim_create(int lattice, int nx, int ny, double tau, double omega, const lbm_geometry* geom,
                    const CreatePlan* plan, lbm_sim** out) {
    clear_error();
    if (!out) return set_error(LBM_EINVAL, "null output handle");
    *out = nullptr;
    if (!geom) return set_error(LBM_EINVAL, "null geometry");
    HostLattice H;
    if (!host_lattice(lattice, H)) return set_error(LBM_EINVAL, "lattice must be LBM_D2Q9 or LBM_D2Q37");
    if (nx < 2 * H.R + 1 || ny < 2 * H.R + 1)
        return set_error(LBM_EINVAL, "grid %dx%d below %d nodes per side", nx, ny, 2 * H.R + 1);
    if ((long long)nx * ny > (1ll << 31) / 2) return set_error(LBM_EINVAL, "grid %dx%d too large", nx, ny);
    if (!(tau > 0.5) || !std::isfinite(tau)) return set_error(LBM_EINVAL, "tau must be > 1/2 (got %g)", tau);
    if (!(omega > 0.0) || !std::isfinite(omega)) return set_error(LBM_EINVAL, "omega must be > 0 (got %g)", omega);
    lbm_geometry g = *geom;
    if (g.rho0 == 0.0) g.rho0 = 1.0;
    if (!(g.rho0 > 0.0)) return set_error(LBM_EINVAL, "rho0 must be > 0");
    if (!(g.u0 >= 0.0) || !(g.u0 < omega))
        return set_error(LBM_EINVAL, "need 0 <= u0 < omega (displacement below one node), got u0=%g omega=%g", g.u0,
                         omega);
    if (g.drive != LBM_DRIVE_WALL && g.drive != LBM_DRIVE_BODYFORCE) return set_error(LBM_EINVAL, "bad drive");
    if (g.eq_order != 2 && g.eq_order != 4) return set_error(LBM_EINVAL, "eq_order must be 2 or 4");
    if (lattice == LBM_D2Q9 && g.eq_order != 2) return set_error(LBM_EINVAL, "D2Q9 supports eq_order 2 only");
    if (g.collision != LBM_COLL_BGK && g.collision != LBM_COLL_REGULARIZED)
        return set_error(LBM_EINVAL, "bad collision");
    if (g.wall_scheme != LBM_SCHEME_BOUNCEBACK && g.wall_scheme != LBM_SCHEME_DIFFUSE)
        return set_error(LBM_EINVAL, "bad wall scheme %d", g.wall_scheme);
    if (g.layout != LBM_LAYOUT_AB && g.layout != LBM_LAYOUT_AA) return set_error(LBM_EINVAL, "bad layout %d", g.layout);
    if (g.layout == LBM_LAYOUT_AA && g.wall_scheme != LBM_SCHEME_BOUNCEBACK)
        return set_error(LBM_EINVAL, "the in-place (AA) layout is built for bounce-back walls only");
    const size_t es = storage_size(g.storage);
    if (!es) return set_error(LBM_EINVAL, "bad storage type %d", g.storage);
    if (es == 2 && !(g.u0 > 0.0))
        return set_error(LBM_EINVAL, "16-bit storage is scaled by u0 and needs u0 > 0");
    StepLaunchFn fn = find_step_launcher(lattice, g.storage, g.collision, g.wall_scheme);
    if (!fn) return set_error(LBM_EINVAL, "no kernel for this lattice/storage/collision/wall");
    StepLaunchFn aa0 = nullptr, aa1 = nullptr;
    if (g.layout == LBM_LAYOUT_AA) {
        aa0 = find_aa_launcher(lattice, g.storage, g.collision, 0);
        aa1 = find_aa_launcher(lattice, g.storage, g.collision, 1);
        if (!aa0 || !aa1) return set_error(LBM_EINVAL, "no in-place kernel for this lattice/storage/collision");
    }

    lbm_sim* s = new (std::nothrow) lbm_sim();
    if (!s) return set_error(LBM_ENOMEM, "host allocation");
    s->Q = lattice;
    s->nx = nx;
    s->ny = ny;
    s->tau = tau;
    s->omega = omega;
    s->lat = H;
    s->esize = es;
    s->launch = fn;
    s->launch_default = fn;
    s->aa = g.layout == LBM_LAYOUT_AA;
    s->aa_launch[0] = aa0;
    s->aa_launch[1] = aa1;
    int rc = cudaGetDevice(&s->device) == cudaSuccess ? LBM_OK : LBM_ECUDA;
    if (rc) { delete s; return set_error(rc, "no CUDA device"); }
    rc = check_geometry(H, nx, ny, g);
    if (rc) { delete s; return rc; }
    const int align = (int)(128 / es);
    s->pitch = (nx + align - 1) / align * align;
    const size_t plane = (size_t)ny * s->pitch;
    if ((size_t)H.Q * plane >= (1ull << 32)) {  // the kernels address populations with 32-bit offsets
        delete s;
        return set_error(LBM_EINVAL, "grid %dx%d: %d x %zu populations exceed 2^32", nx, ny, H.Q, plane);
    }
    GeomScan scan;
    scan_geometry(H, nx, ny, g, scan);
    if (g.kind == LBM_GEOM_MASK) s->labels.assign(g.mask, g.mask + (size_t)nx * ny);
    g.mask = nullptr;
    s->geom = g;
    s->n_fluid = scan.n_fluid;
    s->link_nodes.swap(scan.links);
    s->n_boundary = s->link_nodes.size();
    std::vector<size_t> link_count(H.Q, 0);
    for (const LinkNode& ln : s->link_nodes) {
        if (!ln.body) continue;
        s->body_row1 = (int)(ln.node / (size_t)nx);
        if (s->nbf++ == 0) s->body_row0 = s->body_row1;
        for (uint64_t m = ln.body; m; m &= m - 1) ++link_count[__builtin_ctzll(m)];
    }
    constant_force(H, link_count, g.rho0, s->fconst[0], s->fconst[1], s->fmov[0], s->fmov[1]);

    InstDev& d = s->dev;
    const bool by_links = g.wall_scheme == LBM_SCHEME_BOUNCEBACK;
    SolidLists lists{s->link_nodes.size(), (size_t)s->nbf, 0};
    for (size_t n : link_count) lists.nfl += by_links ? n : 0;
    // force groups: by links for the two-buffer bounce-back step, by nodes (32 a group) otherwise.  (Along one
    // direction and its opposite at most 2 min(fluid, solid) links, or 2 fluid where a link passes over other
    // nodes, are blocked: 18 links a node of the grid in D2Q37, 4 in D2Q9, below 2^31 with Q plane < 2^32.)
    d.nb = (int)lists.nb;
    d.nbf = s->nbf;
    d.nfl = (int)lists.nfl;
    d.glen = force_group_len(d.nfl);
    s->link_groups = by_links ? force_groups(d.nfl, d.glen) : (s->nbf + 31) / 32;
    d.ngroups = s->aa ? (s->nbf + 31) / 32 : s->link_groups;
    if (plan) s->may_defer = false;
    s->cap = std::max<size_t>(1024, plan ? plan->history : 0);
    const SimLayout at = sim_layout(H, nx, ny, g, lists, s->cap, s->may_defer);
    if (plan && (rc = plan->admit(plan->context, at.bytes() + (at.together ? 0 : at.nbuf * at.pop), d.ngroups))) {
        delete s;
        return rc;
    }

    if (cudaStreamCreateWithFlags(&s->stream, cudaStreamNonBlocking) != cudaSuccess) {
        delete s;
        return set_error(LBM_ECUDA, "stream creation failed");
    }
    s->own_stream = true;

#define TRY_OR_FREE(x)          \
    do {                        \
        int r_ = (x);           \
        if (r_) {               \
            free_sim(s);        \
            return r_;          \
        }                       \
    } while (0)

    TRY_OR_FREE(dev_alloc(s, &s->d_block, at.bytes()));
    for (size_t k = 0; k < at.nbuf; ++k) {
        if (at.together) s->buf[k] = s->d_block + at.pops + k * at.pop;
        else TRY_OR_FREE(dev_alloc(s, (unsigned char**)&s->buf[k], at.pop));
        s->own_buf = !at.together;
    }
    d.cls = s->d_block;
    d.bnodes = reinterpret_cast<const uint2*>(s->d_block + at.nodes);
    d.blinks = reinterpret_cast<const ulonglong2*>(s->d_block + at.links);
    d.flinks = s->d_block + at.flinks;
    d.ticket = reinterpret_cast<unsigned int*>(s->d_block + at.zero);
    d.err = s->d_err = reinterpret_cast<int*>(s->d_block + at.zero + 128);
    d.partials = reinterpret_cast<double2*>(s->d_block + at.zero + 256);
    s->d_history = reinterpret_cast<double2*>(s->d_block + at.history);

    // lists of boundary nodes, body nodes first, and of body links
    std::vector<unsigned char> host(at.zero - at.nodes, 0);
    uint2* nodes = reinterpret_cast<uint2*>(host.data());
    ulonglong2* links = reinterpret_cast<ulonglong2*>(host.data() + (at.links - at.nodes));
    size_t body_place = 0, wall_place = (size_t)s->nbf;
    for (const LinkNode& ln : s->link_nodes) {
        const size_t k = ln.body ? body_place++ : wall_place++;
        nodes[k] = make_uint2((unsigned)(ln.node % (size_t)nx), (unsigned)(ln.node / (size_t)nx));
        links[k] = make_ulonglong2(ln.body, ln.wall);
    }
    if (by_links) fill_flinks(s, link_count, host.data() + (at.flinks - at.nodes));

    // node classes: bulk, the padding solid, then the visited rows, run by run (many runs: all rows at once)
    cudaStream_t st = s->stream;
    bool up = cudaMemsetAsync(s->d_block, NODE_BULK, plane, st) == cudaSuccess &&
              (s->pitch == nx || cudaMemset2DAsync(s->d_block + nx, s->pitch, NODE_SOLID, s->pitch - nx, ny, st) == cudaSuccess);
    std::vector<std::pair<size_t, size_t>> runs;  // [first, last) of scan.rows
    for (size_t k = 0; k < scan.rows.size(); ++k) {
        if (k == 0 || scan.rows[k] != scan.rows[k - 1] + 1) runs.emplace_back(k, k);
        runs.back().second = k + 1;
    }
    if (runs.size() <= 8) {
        for (const auto& r : runs)
            up = up && cudaMemcpy2DAsync(s->d_block + (size_t)scan.rows[r.first] * s->pitch, s->pitch,
                                         scan.cls.data() + r.first * nx, nx, nx, r.second - r.first,
                                         cudaMemcpyHostToDevice, st) == cudaSuccess;
        s->h2d_bytes += scan.cls.size();
    } else {
        std::vector<uint8_t> all((size_t)nx * ny, NODE_BULK);
        for (size_t k = 0; k < scan.rows.size(); ++k)
            std::copy_n(scan.cls.data() + k * nx, nx, all.data() + (size_t)scan.rows[k] * nx);
        up = up && cudaMemcpy2DAsync(s->d_block, s->pitch, all.data(), nx, nx, ny, cudaMemcpyHostToDevice, st) == cudaSuccess &&
             cudaStreamSynchronize(st) == cudaSuccess;
        s->h2d_bytes += all.size();
    }
    if (!host.empty())
        up = up && cudaMemcpyAsync(s->d_block + at.nodes, host.data(), host.size(), cudaMemcpyHostToDevice, st) == cudaSuccess;
    s->h2d_bytes += host.size();
    // the geometry is on the device when the call returns (other streams may read it, and the host buffers
    // end here); the zeroes are in order with the simulation's own work
    up = up && cudaMemsetAsync(s->d_block + at.zero, 0, at.pops - at.zero, st) == cudaSuccess &&
         cudaStreamSynchronize(st) == cudaSuccess;
    for (size_t k = 0; up && k < at.nbuf; ++k) up = cudaMemsetAsync(s->buf[k], 0, at.pop, st) == cudaSuccess;
    if (!up) {
        free_sim(s);
        return set_error(LBM_ECUDA, "upload of geometry failed");
    }

    d.fconst = make_double2(s->fconst[0], s->fconst[1]);
    const bool mw = g.drive == LBM_DRIVE_WALL && g.wall_scheme == LBM_SCHEME_BOUNCEBACK;
    d.fmov = mw ? make_double2(s->fmov[0], s->fmov[1]) : make_double2(0.0, 0.0);
    d.plane = (long long)plane;
    d.nx = nx;
    d.ny = ny;
    d.pitch = s->pitch;
    d.eq_order = g.eq_order;
    d.moving = g.drive == LBM_DRIVE_WALL;
    d.wall_ds = g.wall_scheme == LBM_SCHEME_DIFFUSE;
    d.body_force = g.drive == LBM_DRIVE_BODYFORCE;
    d.rho0 = g.rho0;
    d.s = es == 2 ? g.u0 : 1.0;
    d.inv_s = 1.0 / d.s;
    d.omega_c = 1.0 / tau;
    d.reg_a = (1.0 - 1.0 / tau) / (2.0 * H.theta * H.theta);
    d.reg_a2 = 2.0 * d.reg_a;
    d.src_k = (1.0 - 0.5 / tau) / H.theta;
    d.src_t = d.src_k / d.omega_c;
    d.mw_k = 2.0 * g.rho0 / (H.theta * d.s);
    d.rho0_f = (float)d.rho0;
    d.s_f = (float)d.s;
    d.inv_s_f = (float)d.inv_s;
    d.omega_c_f = (float)d.omega_c;
    const bool q9 = lattice == LBM_D2Q9;
    const double diag = (1.0 - 1.0 / tau) / (q9 ? reg_diag<D2Q9, float>() : reg_diag<D2Q37, float>());
    const double cross = (1.0 - 1.0 / tau) / (q9 ? reg_cross<D2Q9, float>() : reg_cross<D2Q37, float>());
    d.reg_f[0] = (float)diag;
    d.reg_f[1] = (float)(diag - (double)d.reg_f[0]);
    d.reg_f[2] = (float)cross;
    d.reg_f[3] = (float)(cross - (double)d.reg_f[2]);
    d.src_k_f = (float)d.src_k;
    const double src_t = d.src_k / (double)d.omega_c_f;  // (the rounded 1/tau times it is the source)
    d.src_t_f[0] = (float)src_t;
    d.src_t_f[1] = (float)(src_t - (double)d.src_t_f[0]);
    s->stream_off = es == 2 && g.drive == LBM_DRIVE_BODYFORCE;
    d.stream_off = s->stream_off ? 1 : 0;
    // default kernel: the fastest measured single-instance form -- for D2Q37 the plain kernel with an occupancy
    // floor on the default 32 x 4 tile (variant 1 for FP32, 2 for plain BGK with 16-bit storage), for the
    // regularized collision of 16-bit storage two nodes per thread where that pays (pair_variant); for FP32 and 16-bit
    // D2Q9 several nodes per thread (30) but on small grids, where fewer nodes per thread mean more warps (us a
    // step, 30 / 0; FP32: 2048^2 44.5 / 58.5, 1024^2 9.1 / 11.8, 512^2 3.6 / 3.7, 430^2 3.5 / 2.8, 128^2 2.1 / 1.9;
    // FP16: 2048^2 28.9 / 53.7, 1024^2 7.4 / 13.3, 512^2 3.6 / 4.3, 430^2 3.5 / 3.6, 362^2 3.2 / 2.7, 128^2 2.9 / 2.2) and on rows of
    // half a tile or less (24 x 60000 FP32 29.1 / 22.7, FP16 47 / 26)
    if (!s->aa && g.wall_scheme == LBM_SCHEME_BOUNCEBACK) {
        int v = 0;
        if (lattice == LBM_D2Q9) v = es <= 4 && nx > 32 && (size_t)nx * ny > ((size_t)1 << (es == 4 ? 18 : 17)) ? 30 : 0;
        else if (es == 4) v = 1;
        else if (es == 2)
            v = g.collision != LBM_COLL_REGULARIZED ? 2 : pair_variant(nx, ny, d.nb > 0, 2 * plane * H.Q * es, false);
        if (v) TRY_OR_FREE(use_variant(s, v));
    }
    TRY_OR_FREE(setup_tiles(s));
    *out = s;
    return LBM_OK;
}

extern "C" {

int lbm_set_tile(lbm_sim* s, int block_x, int block_y) {
    int rc = check_sim(s);
    if (rc) return rc;
    if (block_x < 32 || block_x % 32 || block_y < 1 || block_x * block_y > 512)
        return set_error(LBM_EINVAL, "tile %dx%d: need block_x a multiple of 32 and block_x*block_y <= 512", block_x,
                         block_y);
    CUDA_TRY(cudaStreamSynchronize(s->stream));
    s->plain_bx = s->bx = block_x;
    s->plain_by = s->by = block_y;
    s->variant = 0;
    s->tma_launch = nullptr;
    s->launch = s->launch_default;
    return setup_tiles(s);
}

int lbm_set_variant(lbm_sim* s, int variant) {
    int rc = check_sim(s);
    if (rc) return rc;
    if (variant == 0) return lbm_set_tile(s, s->plain_bx, s->plain_by);
    if (s->aa) return set_error(LBM_EINVAL, "the in-place (AA) layout runs the plain kernel (variant 0) only");
    if (s->geom.wall_scheme != LBM_SCHEME_BOUNCEBACK)
        return set_error(LBM_EINVAL, "kernel variants are built for bounce-back walls only");
    CUDA_TRY(cudaStreamSynchronize(s->stream));
    return use_variant(s, variant);
}

int lbm_step(lbm_sim* s, long n) {
    int rc = check_sim(s);
    if (rc) return rc;
    if (n < 0) return set_error(LBM_EINVAL, "negative step count");
    if (n == 0) return LBM_OK;
    // an in-place even step also writes the force of the step after it
    rc = ensure_capacity(s, (size_t)(s->steps_done + n + (s->aa ? 1 : 0)));
    if (rc) return rc;
    const dim3 block(s->bx, s->by);
    if (s->aa) {
        for (long k = 0; k < n; ++k) {
            const int phase = (int)(s->steps_done & 1);
            s->dev.src = s->buf[0];
            s->dev.dst = s->buf[0];
            // the drive of the next step, then that of this one
            set_drive(s->dev, drive_value(s->geom.drive, s->geom.u0, s->omega, s->steps_done + 1));
            s->dev.dv2 = s->dev.dv;
            std::copy_n(s->dev.mw, 4, s->dev.mw2);
            std::copy_n(s->dev.mw_f, 4, s->dev.mw2_f);
            set_drive(s->dev, drive_value(s->geom.drive, s->geom.u0, s->omega, s->steps_done));
            s->dev.stream_off = s->stream_off ? 1 : 0;
            s->dev.flip = (int)(s->steps_done & 1);
            if (s->stream_off) {
                stream_offset_cx(s, s->U_stream, s->dev.Hl, s->dev.HM);
                stream_offset_cx(s, s->U_stream + s->dev.dv, s->dev.Hs, nullptr);
                stream_offset_eo(s->dev.Hs, s->dev.He, s->dev.Ho);
            }
            s->dev.force_out = s->d_history + s->steps_done;
            const cudaError_t e = s->aa_launch[phase](s->dev, block, s->stream);
            if (e != cudaSuccess) return set_error(LBM_ECUDA, "step launch: %s", cudaGetErrorString(e));
            ++s->steps_done;
            if (s->stream_off) s->U_stream += s->dev.dv;
        }
        return LBM_OK;
    }
    // a short call sums each step's force in the step; 8 steps are where one launch for all is worth it (us a step in
    // calls of 7 / 8 steps: 64^2 FP32 3.6 / 2.6, 256^2 5.5 / 3.8, D2Q9 256^2 4.6 / 2.3, where the step is longer than its
    // sum 512^2 FP16 7.6 / 7.9, the same from 32 steps on)
    const bool defer = s->defers_forces() && n >= 8;
    unsigned int* const ticket = s->dev.ticket;
    double2* const partials = s->dev.partials;
    ForceSteps F;
    F.scale = s->dev.wall_ds ? 1.0 : -2.0 * s->dev.s;
    const auto step = [&](long, int held) {
        s->dev.src = s->buf[s->cur];
        s->dev.dst = s->buf[s->cur ^ 1];
        set_drive(s->dev, drive_value(s->geom.drive, s->geom.u0, s->omega, s->steps_done));
        s->dev.stream_off = s->stream_off ? 1 : 0;
        s->dev.flip = (int)(s->steps_done & 1);
        if (s->stream_off) {
            stream_offset_cx(s, s->U_stream, s->dev.Hl, s->dev.HM);
            stream_offset_cx(s, s->U_stream + s->dev.dv, s->dev.Hs, nullptr);
            stream_offset_eo(s->dev.Hs, s->dev.He, s->dev.Ho);
        }
        s->dev.force_out = s->d_history + s->steps_done;
        if (defer) {
            s->dev.ticket = nullptr;
            s->dev.partials = partials + (size_t)held * s->dev.ngroups;
            F.dv[held] = s->dev.dv;
        }
        const cudaError_t e = s->tma_launch ? s->tma_launch(s->dev, s->maps[s->cur], s->store_maps[s->cur ^ 1], s->stream)
                                            : s->launch(s->dev, block, s->stream);
        s->dev.ticket = ticket;
        s->dev.partials = partials;
        if (e != cudaSuccess) return (int)e;
        s->cur ^= 1;
        ++s->steps_done;
        if (s->stream_off) s->U_stream += s->dev.dv;
        return 0;
    };
    const auto sum = [&](int held) {
        if (!defer) return 0;
        F.n = held;
        F.force_out = s->d_history + s->steps_done - held;
        return (int)launch_pdl(sum_forces, dim3((held + 3) / 4), dim3(128), 0, s->stream, s->dev, F);
    };
    int lost = 0;
    rc = run_deferred(n, kForceSteps, step, sum, &lost);
    s->lost_forces += lost;
    if (rc) return set_error(LBM_ECUDA, "step launch: %s", cudaGetErrorString((cudaError_t)rc));
    return LBM_OK;
}

int lbm_synchronize(lbm_sim* s) {
    int rc = check_sim(s);
    if (rc) return rc;
    CUDA_TRY(cudaStreamSynchronize(s->stream));
    int err = 0;
    CUDA_TRY(cudaMemcpy(&err, s->d_err, sizeof(int), cudaMemcpyDeviceToHost));
    if (err & 4) return set_error(LBM_ETIMEOUT, "a bounded wait for staged tile loads timed out");
    if (err & 1) return set_error(LBM_ENONFINITE, "force became non-finite: the run diverged");
    return LBM_OK;
}

int lbm_force_history(lbm_sim* s, double* out_xy, size_t cap_steps, size_t* n_steps) {
    int rc = lbm_synchronize(s);
    if (rc && rc != LBM_ENONFINITE) return rc;
    if (n_steps) *n_steps = (size_t)s->steps_done;
    const size_t n = std::min(cap_steps, (size_t)s->steps_done);
    if (n && !out_xy) return set_error(LBM_EINVAL, "null output buffer");
    if (s->lost_forces)
        return set_error(LBM_ECUDA, "the forces of %d steps of a call that failed were not summed", s->lost_forces);
    if (n) CUDA_TRY(cudaMemcpy(out_xy, s->d_history, n * sizeof(double2), cudaMemcpyDeviceToHost));
    s->d2h_bytes += n * sizeof(double2);
    return rc;
}

int lbm_fit(lbm_sim* s, double skip_periods, double* f_in, double* f_q, double* f_0) {
    int rc = check_sim(s);
    if (rc) return rc;
    const double pi = 3.14159265358979323846;
    const double period = 2.0 * pi / s->omega;
    if (!(skip_periods >= 0.0)) return set_error(LBM_EINVAL, "skip_periods must be >= 0");
    const long n0 = (long)std::ceil(skip_periods * period);
    if ((double)(s->steps_done - n0) < period) return set_error(LBM_ERANGE, "less than one period after the skip");
    std::vector<double> h(2 * (size_t)s->steps_done);
    size_t n = 0;
    rc = lbm_force_history(s, h.data(), (size_t)s->steps_done, &n);
    if (rc) return rc;
    double coef[3];
    rc = fit_sincos(h.data(), 2, n0, s->steps_done, s->omega, coef);
    if (rc) return rc;
    const double sgn = s->geom.drive == LBM_DRIVE_WALL ? 1.0 : -1.0;
    if (f_in) *f_in = sgn * coef[0];
    if (f_q) *f_q = sgn * coef[1];
    if (f_0) *f_0 = coef[2];
    return LBM_OK;
}

int lbm_gamma_bar(lbm_sim* s, double f_in, double perimeter, double* gamma_bar) {
    int rc = check_sim(s);
    if (rc) return rc;
    if (!gamma_bar || !(perimeter > 0.0) || !(s->geom.u0 > 0.0))
        return set_error(LBM_EINVAL, "need an output, perimeter > 0 and u0 > 0");
    *gamma_bar = -f_in / (s->geom.u0 * s->geom.rho0 * std::sqrt(s->lat.theta / 2.0) * perimeter);
    return LBM_OK;
}

void lbm_destroy(lbm_sim* s) {
    if (!s) return;
    cudaSetDevice(s->device);
    free_sim(s);
}

int lbm_set_stream(lbm_sim* s, void* stream) {
    int rc = check_sim(s);
    if (rc) return rc;
    CUDA_TRY(cudaStreamSynchronize(s->stream));
    if (s->own_stream) cudaStreamDestroy(s->stream);
    s->stream = (cudaStream_t)stream;
    s->own_stream = false;
    return LBM_OK;
}

static double to_double(const void* base, int storage, size_t k) {
    switch (storage) {
        case ST_F64: return static_cast<const double*>(base)[k];
        case ST_F32: return static_cast<const float*>(base)[k];
        case ST_BF16: return (double)__bfloat162float(static_cast<const __nv_bfloat16*>(base)[k]);
        default: return (double)__half2float(static_cast<const __half*>(base)[k]);
    }
}

static void from_double(void* base, int storage, size_t k, double v) {
    switch (storage) {
        case ST_F64: static_cast<double*>(base)[k] = v; break;
        case ST_F32: static_cast<float*>(base)[k] = (float)v; break;
        case ST_BF16: static_cast<__nv_bfloat16*>(base)[k] = __double2bfloat16(v); break;
        default: static_cast<__half*>(base)[k] = __double2half(v); break;
    }
}

int lbm_get_state(lbm_sim* s, double* out, size_t count) {
    int rc = lbm_synchronize(s);
    if (rc && rc != LBM_ENONFINITE) return rc;
    const size_t N = (size_t)s->nx * s->ny, plane = (size_t)s->ny * s->pitch;
    if (!out || count != N * s->Q) return set_error(LBM_ERANGE, "need %zu values", N * s->Q);
    if (s->aa && (s->steps_done & 1))
        return set_error(LBM_ERANGE, "the in-place layout holds the state after an even number of steps only");
    const std::vector<uint8_t>& lab = labels_of(s);
    std::vector<unsigned char> host(plane * s->Q * s->esize);
    CUDA_TRY(cudaMemcpy(host.data(), s->buf[s->cur], host.size(), cudaMemcpyDeviceToHost));
    float H[37] = {0};
    if (s->stream_off) stream_offset(s, s->U_stream, H, nullptr);
    for (int i = 0; i < s->Q; ++i) {
        const double scale = s->lat.w[i] * s->dev.s;
        for (int y = 0; y < s->ny; ++y)
            for (int x = 0; x < s->nx; ++x) {
                const size_t k = (size_t)y * s->nx + x;
                // in place, after an even step count direction i sits in plane opp(i)
                const int pi = s->aa ? s->lat.opp[i] : i;
                const double v = to_double(host.data(), s->geom.storage, (size_t)pi * plane + (size_t)y * s->pitch + x);
                // with the stream offset the kernel forms h = stored + H in FP32; do the same here
                const double h = s->stream_off ? (double)(float)(v + H[i]) : v;
                out[(size_t)i * N + k] = lab[k] ? 0.0 : scale * h;
            }
    }
    return rc;
}

int lbm_set_state(lbm_sim* s, const double* g, size_t count) {
    int rc = lbm_synchronize(s);
    if (rc) return rc;
    const size_t N = (size_t)s->nx * s->ny, plane = (size_t)s->ny * s->pitch;
    if (!g || count != N * s->Q) return set_error(LBM_ERANGE, "need %zu values", N * s->Q);
    if (s->aa && (s->steps_done & 1))
        return set_error(LBM_ERANGE, "the in-place layout takes a state after an even number of steps only");
    const std::vector<uint8_t>& lab = labels_of(s);
    std::vector<unsigned char> host(plane * s->Q * s->esize, 0);
    float H[37] = {0};
    if (s->stream_off) stream_offset(s, s->U_stream, H, nullptr);
    for (int i = 0; i < s->Q; ++i) {
        const double inv = 1.0 / (s->lat.w[i] * s->dev.s);
        for (int y = 0; y < s->ny; ++y)
            for (int x = 0; x < s->nx; ++x) {
                const size_t k = (size_t)y * s->nx + x;
                const double v = lab[k] ? 0.0 : g[(size_t)i * N + k] * inv - (double)H[i];
                const int pi = s->aa ? s->lat.opp[i] : i;
                from_double(host.data(), s->geom.storage, (size_t)pi * plane + (size_t)y * s->pitch + x, v);
            }
    }
    // on the stream of the steps: a copy on the default stream may still be on its way when the call returns
    CUDA_TRY(cudaMemcpyAsync(s->buf[s->cur], host.data(), host.size(), cudaMemcpyHostToDevice, s->stream));
    CUDA_TRY(cudaStreamSynchronize(s->stream));
    return LBM_OK;
}

int lbm_get_labels(lbm_sim* s, unsigned char* out, size_t count) {
    int rc = check_sim(s);
    if (rc) return rc;
    const size_t N = (size_t)s->nx * s->ny;
    if (!out || count != N) return set_error(LBM_ERANGE, "need %zu labels", N);
    fill_labels(s, out);
    return LBM_OK;
}

int lbm_tune(lbm_sim* s, int steps, lbm_tune_entry* out, int cap, int* n_out) {
    int rc = check_sim(s);
    if (rc) return rc;
    if (steps < 1 || !n_out || (cap > 0 && !out)) return set_error(LBM_EINVAL, "need steps >= 1 and an output");
    // candidates: plain kernel tiles, then every staged variant built for this storage type
    const int tiles[][2] = {{32, 4}, {32, 8}, {64, 2}, {64, 4}, {128, 1}, {32, 2}};
    const int variants[] = {1, 2, 3, 4, 10, 11, 12, 13, 18, 20, 23, 24, 25, 26, 27, 30, 31, 32};
    std::vector<lbm_tune_entry> cand;
    for (auto& t : tiles) cand.push_back(lbm_tune_entry{0, t[0], t[1], 0.0});
    for (int v : variants)
        if (!s->aa && s->geom.wall_scheme == LBM_SCHEME_BOUNCEBACK &&
            (find_tma_launcher(s->Q, s->geom.storage, s->geom.collision, v) ||
             find_occ_launcher(s->Q, s->geom.storage, s->geom.collision, v) ||
             (s->Q == 9 && find_q9v_launcher(s->geom.storage, s->geom.collision, v)))) {
            int bx = 0, by = 0;
            variant_tile(v, s->geom.storage, &bx, &by);
            cand.push_back(lbm_tune_entry{v, bx, by, 0.0});
        }
    // a clone with the same geometry (as a label mask), parameters and storage
    lbm_geometry g = s->geom;
    g.kind = LBM_GEOM_MASK;
    g.mask = labels_of(s).data();
    lbm_sim* c = nullptr;
    if ((rc = lbm_create(s->Q, s->nx, s->ny, s->tau, s->omega, &g, &c))) return rc;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    int k = 0;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) rc = set_error(LBM_ECUDA, "events");
    for (auto& e : cand) {
        if (rc) break;
        rc = e.variant ? lbm_set_variant(c, e.variant) : lbm_set_tile(c, e.block_x, e.block_y);
        if (rc) break;
        if ((rc = lbm_step(c, 2))) break;  // warm-up (first launch sets kernel attributes)
        cudaEventRecord(e0, c->stream);
        if ((rc = lbm_step(c, steps))) break;
        cudaEventRecord(e1, c->stream);
        if (cudaEventSynchronize(e1) != cudaSuccess) { rc = set_error(LBM_ECUDA, "event sync"); break; }
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        e.us_per_step = 1000.0 * ms / steps;
        if (k < cap) out[k] = e;
        ++k;
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    lbm_destroy(c);
    *n_out = k;
    return rc;
}

int lbm_autotune(lbm_sim* s, int steps, lbm_tune_entry* best) {
    lbm_tune_entry e[32];
    int n = 0;
    int rc = lbm_tune(s, steps, e, 32, &n);
    if (rc) return rc;
    if (n == 0) return set_error(LBM_EINVAL, "no candidate");
    int b = 0;
    for (int k = 1; k < n; ++k)
        if (e[k].us_per_step < e[b].us_per_step) b = k;
    rc = e[b].variant ? lbm_set_variant(s, e[b].variant) : lbm_set_tile(s, e[b].block_x, e[b].block_y);
    if (rc == LBM_OK && best) *best = e[b];
    return rc;
}

int lbm_info(lbm_sim* s, lbm_info_t* o) {
    int rc = check_sim(s);
    if (rc) return rc;
    if (!o) return set_error(LBM_EINVAL, "null output");
    o->lattice = s->Q;
    o->nx = s->nx;
    o->ny = s->ny;
    o->pitch = s->pitch;
    o->storage = s->geom.storage;
    o->collision = s->geom.collision;
    o->eq_order = s->geom.eq_order;
    o->drive = s->geom.drive;
    o->tau = s->tau;
    o->omega = s->omega;
    o->u0 = s->geom.u0;
    o->rho0 = s->geom.rho0;
    o->theta = s->lat.theta;
    o->steps_done = s->steps_done;
    o->n_fluid = s->n_fluid;
    o->n_boundary = s->n_boundary;
    o->bytes_per_step = 2 * (size_t)s->Q * s->esize * s->n_fluid;
    o->device_bytes = s->device_bytes;
    o->block_x = s->bx;
    o->block_y = s->by;
    o->h2d_bytes = s->h2d_bytes;
    o->d2h_bytes = s->d2h_bytes;
    o->variant = s->variant;
    o->layout = s->aa ? LBM_LAYOUT_AA : LBM_LAYOUT_AB;
    o->force_1e4 = s->geom.storage == LBM_STORE_BF16 ? 0 : 1;
    return LBM_OK;
}

}  // extern "C"
