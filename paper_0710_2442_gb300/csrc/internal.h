// internal.h -- host-side declarations shared by the translation units of
// libwilson_gb300 (not part of the C ABI).
#pragma once

#include <functional>
#include <mutex>
#include <stdexcept>
#include <string>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "../../include/wilson.h"
#include "common.cuh"
#include "reduce.cuh"

namespace wl {

struct Error : std::runtime_error {
    int code;
    Error(int c, const std::string& m) : std::runtime_error(m), code(c) {}
};

#define WL_CUDA(call)                                                                          \
    do {                                                                                       \
        cudaError_t e_ = (call);                                                               \
        if (e_ != cudaSuccess)                                                                 \
            throw ::wl::Error(e_ == cudaErrorMemoryAllocation ? 3 : 2,                         \
                              std::string(#call) + ": " + cudaGetErrorString(e_));             \
    } while (0)

#define WL_LAUNCH_CHECK() WL_CUDA(cudaGetLastError())

#define WL_REQUIRE(cond, msg)                                      \
    do {                                                           \
        if (!(cond)) throw ::wl::Error(1, std::string(msg));       \
    } while (0)

// Launch of a kernel that begins with pdl_wait() (common.cuh), with the
// programmatic-serialization attribute: its blocks may be scheduled while the
// previous kernel on the stream drains, which hides the launch gap and the
// last wave's tail.  Launches into a stream that is being captured stay plain:
// measured, the attribute made the captured CG iterations slower (the graph
// already removes the launch gaps).  WILSON_PDL=0 launches every one plainly.
bool pdl_enabled();
template <typename... KArgs, typename... Args>
void launch_dep_smem(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                     const Args&... args) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) {
        (void)cudaGetLastError();
        cs = cudaStreamCaptureStatusActive;
    }
    cfg.numAttrs = pdl_enabled() && cs == cudaStreamCaptureStatusNone ? 1 : 0;
    WL_CUDA(cudaLaunchKernelEx(&cfg, kernel, args...));
}
template <typename... KArgs, typename... Args>
void launch_dep(void (*kernel)(KArgs...), dim3 grid, dim3 block, cudaStream_t st, const Args&... args) {
    launch_dep_smem(kernel, grid, block, 0, st, args...);
}

// ---------------------------------------------------------------------------
// device memory owned by the library
// ---------------------------------------------------------------------------
// The memory pools, one per device and use: the stateless calls' workspace (keeps all it
// ever took, so that only the first call of a size grows it), the fixed-point inputs of F64
// handle hops, and the solves' workspace (these two keep at most a thirty-second of the device's
// memory while unused).  An allocation that finds no memory first gives back what all of them hold
// unused; so does wilson_release_workspace.
enum Pool { POOL_STATELESS, POOL_HOP, POOL_SOLVE, kPools };
cudaError_t pool_alloc(void** p, size_t n, Pool which, cudaStream_t st);
cudaError_t device_alloc(void** p, size_t n);  // cudaMalloc, with that
void trim_pools();                             // on the current device

// While one is alive, the DevBufs that this thread allocates come from a pool
// with stream-ordered allocation on st, and go back to it on st (workspace.cu): a solve's
// 25 to 30 buffers a problem then cost a microsecond each instead of a cudaMalloc
// and a cudaFree, which waits for the device.
struct WorkspaceScope {
    explicit WorkspaceScope(cudaStream_t st);
    ~WorkspaceScope();
    WorkspaceScope(const WorkspaceScope&) = delete;
    WorkspaceScope& operator=(const WorkspaceScope&) = delete;

  private:
    bool before_;
    cudaStream_t st_before_;
};
// p, or null where there is no such scope; st: the stream to give it back on.
void* workspace_alloc(size_t n, cudaStream_t* st);

struct DevBuf {
    void* p = nullptr;
    size_t bytes = 0;
    bool pooled = false;
    cudaStream_t st = nullptr;  // of a pooled buffer
    DevBuf() = default;
    explicit DevBuf(size_t n) { alloc(n); }
    ~DevBuf() { release(); }
    DevBuf(const DevBuf&) = delete;
    DevBuf& operator=(const DevBuf&) = delete;
    DevBuf(DevBuf&& o) noexcept { take(o); }
    DevBuf& operator=(DevBuf&& o) noexcept {
        if (this != &o) { release(); take(o); }
        return *this;
    }
    void alloc(size_t n) {
        release();
        if (n) {
            p = workspace_alloc(n, &st);
            pooled = p != nullptr;
            if (!pooled) WL_CUDA(device_alloc(&p, n));
        }
        bytes = n;
    }
    void ensure(size_t n) { if (n > bytes) alloc(n); }
    void release() {
        if (p && pooled) cudaFreeAsync(p, st);
        else if (p) cudaFree(p);
        p = nullptr;
        bytes = 0;
        pooled = false;
    }
    template <class T>
    T* as() const { return static_cast<T*>(p); }

  private:
    void take(DevBuf& o) {
        p = o.p;
        bytes = o.bytes;
        pooled = o.pooled;
        st = o.st;
        o.p = nullptr;
        o.bytes = 0;
        o.pooled = false;
    }
};

// ---------------------------------------------------------------------------
// autotuner (tune.cu)
// ---------------------------------------------------------------------------
struct LaunchConfig {
    int block = 128;
    int variant = 0;
};

// The launch configuration for `key`.  On the first request (and when tuning
// is enabled, WILSON_TUNE != 0, and the stream is not being captured) every
// candidate is timed by running `run` on the stream with CUDA events, and the
// fastest is cached (in memory, and in the file named by WILSON_TUNE_CACHE if
// set).  `run` must be idempotent: it is executed several times.
// margin: a later candidate replaces the best one so far only when it is
// faster by more than this fraction (so that near-ties resolve to the
// earlier candidate).
LaunchConfig tune_launch(const std::string& key, const std::vector<LaunchConfig>& candidates,
                         const LaunchConfig& fallback, cudaStream_t st,
                         const std::function<void(const LaunchConfig&)>& run, double margin = 0.01);
// The decision for `key` if one is cached (in memory or in the cache file)
// and among `candidates`, else `fallback`; never times anything and never
// synchronises.
LaunchConfig tune_lookup(const std::string& key, const std::vector<LaunchConfig>& candidates,
                         const LaunchConfig& fallback);
const std::vector<LaunchConfig>& hop_candidates();

// Geometry from dims and phases; stride rounded up to 64 sites.
Geom make_geom(const int dims[4], const double ph[4][2]);

inline int spinor_chunk_rows(Prec p) { return p == P_F64 ? 12 : p == P_F32 ? 6 : 3; }
long long spinor_field_bytes(Prec p, int stride);          // one parity, one rhs
long long gauge_bytes(Prec p, int recon, int stride);      // both parities, 4 directions
long long gauge_block_bytes(Prec p, int recon, int stride);

// A prepared spinor field: nrhs x (1 or 2 parities) SoA blocks.
struct SpinorField {
    Prec prec = P_F32;
    int subset = 0;      // 0 even, 1 odd, 2 full
    int nrhs = 1;
    Geom g{};
    DevBuf buf;
    long long pbytes = 0;   // bytes of one parity block of one rhs
    int nparity() const { return subset == 2 ? 2 : 1; }
    // pointer to parity block p (absolute parity 0/1) of rhs k
    void* block(int p, int k = 0) const {
        int slot = subset == 2 ? p : 0;
        return static_cast<char*>(buf.p) + (size_t)(k * nparity() + slot) * pbytes;
    }
    // bytes from one right-hand side's blocks to the next one's
    long long rstep() const { return (long long)nparity() * pbytes; }
    void alloc(Prec p, int sub, int nr, const Geom& geom);
    void alloc_fx(int sub, int nr, const Geom& geom, int fields);  // F64, or `fields` fixed-point fields a block
};

struct GaugeField {
    Prec prec = P_F32;
    int recon = 12;
    Geom g{};
    DevBuf buf;
    // F64 links of the fixed-point hops (dslash_fx.cuh), 18 reals for either
    // recon; links out of their range are read from buf, or where there is
    // none from canon (canonical links the caller keeps).  canon alone: the
    // kernel for small lattices, which converts the links itself.
    DevBuf fx;
    const double* canon = nullptr;
};

// Per-device scratch: reduction partials and counters.
struct Reduction {
    DevBuf partials;   // doubles
    DevBuf counters;   // unsigned ints, zeroed
    DevBuf results;    // doubles
    int capacity = 0;
    void init(int cap, int ncounters, cudaStream_t st);
    // Slots counter_slot .. counter_slot + nrhs - 1 (one per right-hand side).
    RedArgs args(int counter_slot, int op, double* result, CGScalars* sc) const {
        RedArgs r;
        r.partials = partials.as<double>() + (size_t)counter_slot * capacity;
        r.counter = counters.as<unsigned int>() + counter_slot;
        r.result = result;
        r.sc = sc;
        r.op = op;
        r.slot_cap = capacity;
        return r;
    }
};

// ---------------------------------------------------------------------------
// kernel launchers
// ---------------------------------------------------------------------------
struct HopLaunch {
    void* out;             // output parity block (parity out_parity), or parity-0 block if full
    const void* in;        // input block of parity 1 - out_parity, or parity-0 block if full
    const void* x;         // xpay block, parity out_parity (or parity-0 block if full); may be null
    long long out_pstep;   // full launches: byte offset of the parity-1 block from the parity-0 block
    long long in_pstep;
    long long x_pstep;
    int nrhs;              // right-hand sides in one launch (0 or 1: one)
    long long out_rstep;   // byte offset between consecutive right-hand sides
    long long in_rstep;
    long long x_rstep;
    int skip_stride;       // ints between the per-rhs skip flags
    const GaugeField* gauge;
    Prec sprec;
    int out_parity;        // single-parity launches
    int full;              // 1: both output parities in one launch
    int dagger;            // 1: projectors swapped (the hop of g5 D g5)
    int xpay;              // out = x + a * D in   (else out = a * D in)
    double a;
    const RedArgs* red;    // |out|^2 into a reducer, or null
    const int* skip;       // device flags (one per rhs): nonzero -> that rhs does nothing
    int block;             // threads per block (0 = autotuned)
    int variant;           // kernel register-budget variant when block > 0
    int grid_cap;          // max blocks of a reducing launch (0 = no cap)
    int tune_only;         // 1: tune the launch configuration if it is not known yet, launch nothing else
    // F64 on the fixed-point hops (fx_hops(*gauge)); fields of fx_spinor_bytes per parity
    const void* fx_in;     // the input as a fixed-point field, or null
    void* fx_tmp;          // else room to convert it (null: the kernel that takes doubles)
    long long fx_pstep;    // steps of either
    long long fx_rstep;
    int fx_out;            // out is a fixed-point field (plain hop, fx_site_kernel only)
    int canon;             // bits kCanonIn, kCanonX, kCanonOut: that field is canonical (one rhs)
};
constexpr int kCanonIn = 1, kCanonX = 2, kCanonOut = 4;
int launch_hop(const HopLaunch& L, cudaStream_t st);  // returns a reducing launch's blocks per rhs

// FP64 hops on the integer pipe (dslash_fx.cu).  They run wherever the links
// have a fixed-point form, unless WILSON_HOP_VARIANT pins the FP64 stencil and the
// links are there as doubles.
bool fx_hops(const GaugeField& gf);
int launch_hop_fx(const HopLaunch& L, cudaStream_t st);
long long fx_spinor_bytes(int stride);  // one parity, one rhs
// Whether the kernel on fixed-point fields is taken, given room for them: below
// kFxSiteMin output sites the conversion costs more than it saves (12^4: 14 against 12.3 + 4.2 us
// a hop; 16^3 x 32: 43 against 27.6 + 6.2 us).
constexpr long long kFxSiteMin = 20000;
bool fx_site_kernel(const Geom& g, int nrhs, int full);
int hop_grid_blocks(const Geom& g, int block, int grid_cap);

// canonical <-> SoA
// n_rhs right-hand sides from rhs on, canonical fields back to back
void pack_spinor(const SpinorField& f, int rhs, int n_rhs, const double* canon, cudaStream_t st);
void unpack_spinor(const SpinorField& f, int rhs, int n_rhs, double* canon, cudaStream_t st);
// bad: counts the links out of the fixed-point range, if they are packed in that form
void pack_gauge(GaugeField& gf, const double* canon, cudaStream_t st, unsigned long long* bad = nullptr);
// The same with gf.fx, synchronising: false if a twelfth of the links or more are out of range.  A site is
// done over for each of its eight, and from half of the sites on the FP64 stencil is the
// faster one (24^3 x 48 hop: 131 us, 991 us where every site is done over, FP64 stencil 552 us).
bool pack_gauge_fx(GaugeField& gf, const double* canon, cudaStream_t st);

int device_sm_count();

// NVTX range for profilers (nsys/ncu timelines); no cost without a tool.
struct NvtxRange {
    explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
};

// The stateless operators (api.cu).
void stateless_op(double* out, const double* gauge, const double* in, const Geom& g, int parity, double kappa, int op,
                  cudaStream_t st, void* scratch, size_t scratch_bytes);

// Set the calling thread's message returned by wilson_last_error().
void record_error(const std::string& msg);

// Argument checks shared by the entry points (api.cu), so that every entry
// point validates the same way.
Geom checked_geom(const wilson_lattice* L);      // extents, phases, volume; WILSON_ERR_ARG
void check_ptr(const void* p, const char* what);  // non-null and 16-byte aligned; WILSON_ERR_ARG
void check_device();                              // a CUDA device exists; WILSON_ERR_CUDA
bool is_device_ptr(const void* p);                // device or managed memory

// DevBuf objects that borrow memory the library does not own through them
// (a fixed array, a stream-ordered pool): the guard detaches them before
// their destructors run, so those never free it.
struct BorrowGuard {
    DevBuf* bufs[8];
    int n = 0;
    void borrow(DevBuf& b, void* p, size_t bytes) {
        b.p = p;
        b.bytes = bytes;
        bufs[n++] = &b;
    }
    ~BorrowGuard() {
        for (int i = 0; i < n; i++) {
            bufs[i]->p = nullptr;
            bufs[i]->bytes = 0;
        }
    }
};

}  // namespace wl

// The opaque handles of the C ABI (wilson.h).
struct wilson_gauge_s {
    wl::GaugeField f;
    mutable std::mutex m;
    mutable wl::SpinorField tmp;  // intermediate field of the Schur operator
};
struct wilson_spinor_s {
    wl::SpinorField f;
    wl::Geom g;
};
