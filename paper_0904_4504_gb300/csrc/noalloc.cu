// noalloc.cu -- a time step that allocates no device memory (lbm_step_noalloc in include/lbm.h).
//
// Who needs it: callers that must not call cudaMalloc at the time they step the solver, e.g. code
// that records its work into a CUDA graph (allocation during stream capture is not allowed), an
// application whose device memory is owned by another allocator (a framework's caching pool) and
// is already fully reserved, or a loop with a fixed memory budget where an allocation that can fail
// or stall is not acceptable.  lbm_step itself may allocate (it grows the force history), so these
// callers step the lattice through this entry point instead: the populations and the force live in
// buffers the caller owns, and the only other memory the step kernel needs -- its force partials --
// lives in one file-scope device array below, loaded with the library and held by every GPU that uses it
// until the process exits.
//
// The kernel is the simulation's own step kernel, where it reads the populations directly and the
// caller's buffers are aligned for it, else the plain one.  The last force group of a call is found by a ticket
// that starts at zero and that it leaves at zero; one that a call left otherwise (it never completed, or overlapped
// another) must not be met again.  So every call takes the next of two halves of tickets, and a half is cleared
// as a whole before its first ticket is taken again: a call is one launch, but one call in kHalf (a clear before each
// took 4 x 256 D2Q9 FP64 from 6.8 to 9.2 us, numbered counts in one 64-bit word cost small grids 3 to 6 %).  A call
// recorded into a graph keeps its ticket for good, so there it is one of its own, and its clear is recorded too.
#include <cuda_runtime.h>

#include <mutex>

#include "lbm.h"
#include "runtime.h"
#include "step_kernel.cuh"

namespace {

// Scratch: the group partials of the force (16 B each), then the non-finite flag, the ticket of recorded calls and
// the tickets of the others.  With bounce-back walls a step has at most kMaxForceGroups groups; with diffuse walls
// one per 32 nodes with body links, and a geometry is accepted with up to LBM_NOALLOC_MAX_SLOTS tiles holding such
// nodes, 512 in a tile at most.  Shared by every call in the process on a given device.
constexpr size_t kPartialBytes = (size_t)LBM_NOALLOC_MAX_SLOTS * 16 * sizeof(double2);
constexpr unsigned kHalf = 1024;
constexpr size_t kTickets = kPartialBytes + 256;       // flag at kPartialBytes, recorded calls' ticket 128 above it
constexpr size_t kScratchBytes = kTickets + 2 * kHalf * sizeof(unsigned);
static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

constexpr int kMaxDevices = 64;
std::mutex g_addr_mutex;
std::mutex g_call_mutex;           // a call's ticket, the clear before it and its launch
unsigned g_calls[kMaxDevices] = {};
void* g_addr[kMaxDevices] = {};  // null until a lookup on that device has succeeded

// Device address of the scratch array on `device` (looked up with that device current; the name
// g_noalloc_scratch in host code is only a host-side stand-in, never a device address).  Only a
// successful lookup is kept: a failed one (say, inside a stream capture) is retried by the next call.
cudaError_t scratch_address(int device, void** out) {
    std::lock_guard<std::mutex> lock(g_addr_mutex);
    if (!g_addr[device]) {
        void* p = nullptr;
        const cudaError_t rc = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (rc != cudaSuccess) {
            cudaGetLastError();  // the failure is reported through the return code, not left pending
            *out = nullptr;
            return rc;
        }
        g_addr[device] = p;
    }
    *out = g_addr[device];
    return cudaSuccess;
}

}  // namespace

using namespace lbm;

extern "C" int lbm_step_noalloc(const lbm_sim* sim, long n, const void* g_in, void* g_out, double* force_out,
                                void* stream) {
    clear_error();
    if (!sim) return set_error(LBM_EINVAL, "null simulation");
    if (!g_in || !g_out || !force_out) return set_error(LBM_EINVAL, "null device buffer");
    if (g_in == g_out) return set_error(LBM_EINVAL, "g_in and g_out must be different buffers");
    if (n < 0) return set_error(LBM_EINVAL, "negative step index");
    const SimView v = sim_view(sim);
    if (v.slots > LBM_NOALLOC_MAX_SLOTS)
        return set_error(LBM_ERANGE,
                         "lbm_step_noalloc: the geometry has %d tiles with body links, more than the %d its static "
                         "scratch holds; use lbm_step, or a larger tile (lbm_set_tile)",
                         v.slots, LBM_NOALLOC_MAX_SLOTS);
    if (v.device < 0 || v.device >= kMaxDevices) return set_error(LBM_EINVAL, "device %d out of range", v.device);
    int cur = -1;
    if (cudaGetDevice(&cur) != cudaSuccess) return set_error(LBM_ECUDA, "cudaGetDevice failed");
    if (cur != v.device && cudaSetDevice(v.device) != cudaSuccess)
        return set_error(LBM_ECUDA, "cudaSetDevice(%d) failed", v.device);
    void* base = nullptr;
    const cudaError_t arc = scratch_address(v.device, &base);
    if (arc != cudaSuccess || !base)
        return set_error(LBM_ECUDA, "cudaGetSymbolAddress of the step scratch: %s", cudaGetErrorString(arc));
    // the simulation's kernel if it reads the populations directly: 30 with 8-byte loads, 31 with 4-byte
    // ones (for 32, its staged form, 31)
    StepLaunchFn fn = nullptr;
    const size_t misalign = reinterpret_cast<size_t>(g_in) | reinterpret_cast<size_t>(g_out);
    const int variant = v.variant == 32 ? 31 : v.variant;
    const bool fits = variant == 30 ? misalign % 8 == 0 : variant == 31 ? misalign % 4 == 0 : true;
    if (variant != 0 && fits && !v.aa) fn = find_direct_launcher(v.Q, v.storage, v.collision, variant);
    if (!fn) fn = find_step_launcher(v.Q, v.storage, v.collision, v.inst.wall_ds);
    if (!fn) return set_error(LBM_EINVAL, "no kernel for this simulation");

    unsigned char* b = static_cast<unsigned char*>(base);
    InstDev P = v.inst;
    P.src = g_in;
    P.dst = g_out;
    P.partials = reinterpret_cast<double2*>(b);
    P.err = reinterpret_cast<int*>(b + kPartialBytes);
    P.force_out = reinterpret_cast<double2*>(force_out);
    P.ngroups = v.nlf;
    P.flip = (int)(n & 1);
    set_drive(P, drive_value(v.drive, v.u0, v.omega, n));
    P.stream_off = 0;  // caller buffers hold plain scaled deviations: no offsets
    for (int m = 0; m < 4; ++m) P.He[m] = P.Ho[m] = 0.f;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaSuccess;
    // (the legacy default stream cannot be captured; the question costs a tenth of a short call)
    if (st != nullptr && st != cudaStreamLegacy) e = cudaStreamIsCapturing(st, &capture);
    if (e == cudaSuccess) {
        std::lock_guard<std::mutex> lock(g_call_mutex);
        if (capture != cudaStreamCaptureStatusNone) {
            P.ticket = reinterpret_cast<unsigned int*>(b + kPartialBytes + 128);
            if (P.ngroups > 0) e = cudaMemsetAsync(P.ticket, 0, sizeof(unsigned), st);
        } else if (P.ngroups > 0) {
            const unsigned at = g_calls[v.device]++ % (2 * kHalf);
            P.ticket = reinterpret_cast<unsigned int*>(b + kTickets) + at;
            if (at % kHalf == 0) e = cudaMemsetAsync(P.ticket, 0, kHalf * sizeof(unsigned), st);
        }
        if (e == cudaSuccess) e = fn(P, dim3(v.bx, v.by), st);
    }
    if (e == cudaSuccess && P.ngroups == 0) e = cudaMemsetAsync(force_out, 0, 2 * sizeof(double), st);
    if (cur != v.device) cudaSetDevice(cur);
    if (e != cudaSuccess) return set_error(LBM_ECUDA, "lbm_step_noalloc: %s", cudaGetErrorString(e));
    return LBM_OK;
}
