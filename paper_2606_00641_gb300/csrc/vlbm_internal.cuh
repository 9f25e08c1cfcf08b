// vlbm_internal.cuh -- internal types of the GB300 VLBM library (not ABI).
//
// Population storage: one in-place buffer per context, structure of arrays.
// Slot (j, cell) of a domain lives at  base + j * stride + cell, where j runs
// over lattice-major (lattice k, direction i) pairs and stride is the cell
// count rounded up to a multiple of 64 elements, so that every slot plane
// starts on a 128-byte boundary for every storage type.
//
// AA in-place streaming (two kernels that alternate):
//   parity 0 ("even") step at cell x:  read slot (i, x), write the
//       post-collision value of direction i to slot (opp(i), x);
//   parity 1 ("odd") step at cell x:   read slot (opp(i), x - c_i), write
//       the post-collision value of direction i to slot (i, x + c_i).
// The set of slots a cell reads equals the set it writes, so one buffer
// suffices and no two threads touch the same slot.  The logical
// (pre-collision) population of the state is slot (i, x) at parity 0 and
// slot (opp(i), x - c_i) at parity 1.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <map>
#include <string>
#include <type_traits>
#include <vector>

#include "vlbm.h"

#include <nvtx3/nvToolsExt.h>

namespace vlbm {

constexpr int kMaxLat = 9;  // per-lattice tables of Domain: ideal 8, Powell 9 (resistive 4; the
                            // dissipative model's 12 gradient lattices share params.tau_g)
constexpr int kBlockX = 128;     // threads per CTA along x for the step kernels
constexpr int kReduceBlocks = 1216;  // 8 CTAs per SM on 152 SMs
constexpr int kReduceThreads = 256;

// Status bits written by kernels into the context's device flag word.
constexpr unsigned kFlagNonPhysical = 1u;  // NaN, rho <= 0 or p <= 0
constexpr unsigned kFlagUnstable = 2u;     // max(|u| + c_f) >= cs at init
constexpr unsigned kFlagTimeout = 4u;      // a bounded device wait gave up

// Direction i of the axis-aligned sets: 0 rest, 2a+1 = +e_a, 2a+2 = -e_a.
__host__ __device__ constexpr int opp_axis(int i) { return i == 0 ? 0 : ((i & 1) ? i + 1 : i - 1); }

// The per-cell arithmetic (ideal_cell.cuh) is host-and-device: the step
// kernels run it on the GPU, and the same source also compiles for the host,
// where a test checks it cell by cell without a GPU.  The two device-only
// operations it needs go through these helpers.
#define VLBM_HD __host__ __device__

// Unsigned 32-bit division by a launch constant (Granlund and Montgomery, 1994,
// "Division by invariant integers using multiplication", their Figure 4.1).
struct FastDiv {
    uint32_t d, m, sh1, sh2;
    VLBM_HD __forceinline__ uint32_t div(uint32_t n) const
    {
#ifdef __CUDA_ARCH__
        const uint32_t t = __umulhi(m, n);
#else
        const uint32_t t = (uint32_t)(((uint64_t)m * n) >> 32);
#endif
        return (t + ((n - t) >> sh1)) >> sh2;
    }
};
inline FastDiv fast_div(uint32_t d)
{
    uint32_t l = 0;
    while (l < 32 && (uint64_t(1) << l) < d) ++l;
    const uint32_t m = (uint32_t)(((uint64_t(1) << 32) * ((uint64_t(1) << l) - d)) / d + 1);
    return {d, m, l < 1 ? l : 1, l < 1 ? 0 : l - 1};
}

// How a step's threads lie on the grid.  Rows: a CTA takes kBlockX cells of one x-row,
// y and z from the block index.  Planes: a CTA takes kBlockX consecutive cells of an
// xy-plane whatever row they are in, z from the block index, x and y by a division.
// Rows leave threads without a cell where nx is no multiple of kBlockX (half of them at
// nx = 64 or 130); where it is one, both give the same CTAs and rows need no division.
struct StepGrid {
    dim3 grid;
    bool planes;
    FastDiv nx;
};
inline StepGrid step_grid(int nx, int ny, int nz)
{
    const uint64_t plane = (uint64_t)nx * (uint64_t)ny, last = 0xFFFFFFFFull - kBlockX;
    StepGrid g;
    g.nx = fast_div((uint32_t)nx);
    g.planes = nx % kBlockX != 0 && plane <= last && (plane + kBlockX - 1) / kBlockX <= 0x7FFFFFFFull;
    if (g.planes) g.grid = dim3((unsigned)((plane + kBlockX - 1) / kBlockX), (unsigned)nz, 1);
    else g.grid = dim3((unsigned)((nx + kBlockX - 1) / kBlockX), (unsigned)ny, (unsigned)nz);
    return g;
}
// Launch of a step kernel; chained: it may overlap the end of the launch before it
// (programmatic dependent launch).  Its CTAs are set up once all of the previous step's are
// past their stores (chain_next), and wait in chain_wait() for that whole step and its writes
// before they touch memory.  For steps of a few microseconds, where the gap between
// launches counts.  Let in earlier, at the previous step's start, the waiting CTAs took
// whatever room was left and piled up on some SMs: graphs of 32 steps of 1.4 .. 1.9 or 2.5 .. 5
// CTAs per SM were up to 23 per cent slower than plain ones (2-D 256^2 3.8 -> 4.5 us a step);
// let in at the end they are 1.04 to 1.24 times as fast as plain ones at every size from 32
// to 1216 CTAs, plain 2-D, Powell, 3-D and channel steps alike (256^2: 3.4 us).
template <class A>
void launch_step_kernel(bool chained, void (*kernel)(A), dim3 grid, unsigned threads, cudaStream_t stream, const A &a)
{
    cudaLaunchAttribute chain = {};
    chain.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    chain.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.stream = stream;
    cfg.attrs = &chain;
    cfg.numAttrs = chained;
    cudaLaunchKernelEx(&cfg, kernel, a);  // its error is the caller's next cudaGetLastError
}
// The first statement of such a kernel that every thread with work reaches, and its last.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
// Calls f with the two run-time choices as compile-time ones.
template <class F> void with_flags(bool first, bool second, F f)
{
    if (first) {
        if (second) f(std::true_type{}, std::true_type{});
        else f(std::true_type{}, std::false_type{});
    } else {
        if (second) f(std::false_type{}, std::true_type{});
        else f(std::false_type{}, std::false_type{});
    }
}
// This thread's cell; false where it has none.
template <bool PLANES>
__device__ __forceinline__ bool step_cell(int nx, int ny, const FastDiv &by_nx, int &x, int &y, int &z)
{
    if (PLANES) {
        const uint32_t p = blockIdx.x * kBlockX + threadIdx.x;
        const uint32_t r = by_nx.div(p);
        x = (int)(p - r * by_nx.d);
        y = (int)r;
        z = (int)blockIdx.y;
        return y < ny;
    }
    x = (int)(blockIdx.x * kBlockX + threadIdx.x);
    y = (int)blockIdx.y;
    z = (int)blockIdx.z;
    return x < nx;
}

// Raise status bits in the flag word (atomically on the device).
VLBM_HD __forceinline__ void raise_flag(unsigned *flags, unsigned bits)
{
#ifdef __CUDA_ARCH__
    atomicOr(flags, bits);
#else
    *flags |= bits;
#endif
}

// Load through the read-only data cache on the device.
template <class T> VLBM_HD __forceinline__ T ro_load(const T *p)
{
#ifdef __CUDA_ARCH__
    return __ldg(p);
#else
    return *p;
#endif
}

// Weights of the axis sets: D2Q5 (1/3, 1/6; cs^2 = 1/3), D3Q7 (1/4, 1/8;
// cs^2 = 1/4).  In both, w_moving / cs^2 = 1/2.
template <int D> struct AxisSet;
template <> struct AxisSet<2> {
    static constexpr int Q = 5;
    static constexpr double w0 = 1.0 / 3.0, w1 = 1.0 / 6.0, cs2 = 1.0 / 3.0;
};
template <> struct AxisSet<3> {
    static constexpr int Q = 7;
    static constexpr double w0 = 1.0 / 4.0, w1 = 1.0 / 8.0, cs2 = 1.0 / 4.0;
};

// Weights in the compute precision C that sum to one exactly.  D3Q7's 1/4 and
// 1/8 are exact in binary; for D2Q5, w0 = 1 - 4 w1 (exact: Sterbenz), and the
// relaxation products omega w0 = omega - 4 (omega w1) (also exact).  With
// rounded products instead, every cell would gain or lose the same fraction of
// Q_k per step -- a drift of about one or two ulps per step in the FP32 domain
// sums of the 2-D forms.
template <int D, class C> struct ExactWeights {
    static constexpr C w1 = C(AxisSet<D>::w1);
    static constexpr C w0 = D == 2 ? C(1) - C(4) * w1 : C(AxisSet<D>::w0);
};
template <int D, class C> VLBM_HD __forceinline__ void relax_weights(C om, C &ow0, C &ow1)
{
    ow1 = om * ExactWeights<D, C>::w1;
    ow0 = D == 2 ? om - C(4) * ow1 : om * ExactWeights<D, C>::w0;
}

// Relaxation constants of one lattice: 1 - omega, omega w_0, omega w_moving and
// omega w_moving / cs^2.
template <class C> struct Relax {
    C omc, ow0, ow1, hom;
};

// With the source terms w_0 S_k and w_moving S_k.
struct RelaxSource {
    float omc, ow0, ow1, hom, src0, src1;
};

// The same for N lattices, worked out once on the host and passed as kernel
// parameters, so that an FP64 collision reads them as constant operands.  Formed
// from omega in every thread instead they were five operations per lattice and
// cell, the same for all cells: 40 of the 240 FP64 instructions of a D2Q5 cell
// (the FP64 pipe binds that kernel).  FP32 kernels, which HBM binds, form them from
// omega; their parameters hold no table.
template <class C, int N> struct RelaxTable {};
template <int N> struct RelaxTable<double, N> {
    Relax<double> relax[N];
};

template <int D, class C> VLBM_HD __forceinline__ Relax<C> relax_of(C om)
{
    Relax<C> r;
    r.omc = C(1) - om;
    relax_weights<D, C>(om, r.ow0, r.ow1);
    r.hom = C(0.5) * om;
    return r;
}

template <int D> VLBM_HD __forceinline__ RelaxSource relax_source(float om, float src0, float src1)
{
    const Relax<float> r = relax_of<D, float>(om);
    return {r.omc, r.ow0, r.ow1, r.hom, src0, src1};
}

// The constants of lattice k from the table, or worked out from omega[k].
template <int D, int N> VLBM_HD __forceinline__ Relax<double> relax_at(const RelaxTable<double, N> &t, int k)
{
    return t.relax[k];
}
template <int D, class C> VLBM_HD __forceinline__ Relax<C> relax_at(const C *omega, int k)
{
    return relax_of<D, C>(omega[k]);
}

// Single operations rounded to nearest, never fused or reordered; on the host (built without
// contraction) the plain operators are that.
#ifdef __CUDA_ARCH__
#define VLBM_RN(device, host) device
#else
#define VLBM_RN(device, host) host
#endif
VLBM_HD __forceinline__ float add_rn(float a, float b) { return VLBM_RN(__fadd_rn(a, b), a + b); }
VLBM_HD __forceinline__ float sub_rn(float a, float b) { return VLBM_RN(__fsub_rn(a, b), a - b); }
VLBM_HD __forceinline__ float mul_rn(float a, float b) { return VLBM_RN(__fmul_rn(a, b), a * b); }
VLBM_HD __forceinline__ float fma_rn(float a, float b, float c) { return VLBM_RN(__fmaf_rn(a, b, c), fmaf(a, b, c)); }
VLBM_HD __forceinline__ float rcp_rn(float a) { return VLBM_RN(__frcp_rn(a), 1.f / a); }
#undef VLBM_RN

// Keep an FP64 value in registers: without it the compiler adds a cell's populations
// up a second time for the relaxation, to hold fewer registers over the fluxes -- 32 of
// 202 FP64 instructions a cell in 2-D, 44 of 271 in 3-D, on the pipe that binds those
// kernels.  FP32 values are left as they are.
template <class C> VLBM_HD __forceinline__ void keep_f64(C &v)
{
#ifdef __CUDA_ARCH__
    if constexpr (sizeof(C) == 8) asm("" : "+d"(v));
#endif
}

// An opaque copy of a value: the compiler cannot reuse expressions computed
// from the original across it, so addresses built from the copy are
// recomputed where they are used instead of being held in registers.
__device__ __forceinline__ int64_t opaque(int64_t v)
{
    asm volatile("" : "+l"(v));
    return v;
}

// Storage codecs: deviation forms store (f - w_i ref_k) / scale_k.
template <class S> struct Codec;
template <> struct Codec<double> {
    static constexpr bool kDev = false;
    __device__ static __forceinline__ double load(const double *p) { return *p; }
    __device__ static __forceinline__ void store(double *p, double v) { *p = v; }
};
template <> struct Codec<float> {
    static constexpr bool kDev = false;
    __device__ static __forceinline__ float load(const float *p) { return *p; }
    __device__ static __forceinline__ void store(float *p, float v) { *p = v; }
};
template <> struct Codec<__half> {
    static constexpr bool kDev = true;
    __device__ static __forceinline__ float load(const __half *p) { return __half2float(*p); }
    __device__ static __forceinline__ void store(__half *p, float v) { *p = __float2half_rn(v); }
};
template <> struct Codec<__nv_bfloat16> {
    static constexpr bool kDev = true;
    __device__ static __forceinline__ float load(const __nv_bfloat16 *p) { return __bfloat162float(*p); }
    __device__ static __forceinline__ void store(__nv_bfloat16 *p, float v) { *p = __float2bfloat16_rn(v); }
};

// Compute precision of a storage type: FP64 storage computes in FP64, the
// others in FP32 (as the step kernel does).  GB300 runs FP64 arithmetic far
// slower than FP32, so per-population FP64 work is kept out of the passes
// that read every population.
template <class S> struct ComputeOf {
    using T = float;
};
template <> struct ComputeOf<double> {
    using T = double;
};

// CTAs of a domain-sum pass: one cell a thread up to kReduceBlocks CTAs.  A CTA's last
// act, adding its threads' eight sums, costs 40 FP64 additions a warp on a pipe that
// takes 16 cycles each, so a small domain is not spread over CTAs without cells:
// 30,000 cells took 31 us with all kReduceBlocks CTAs, 8 with 118.
inline int reduce_blocks(int64_t ncell)
{
    const int64_t need = (ncell + kReduceThreads - 1) / kReduceThreads;
    return (int)(need < 1 ? 1 : need < kReduceBlocks ? need : kReduceBlocks);
}

// The CTA's sum of its threads' NV values into its row of eight partials: shuffles within
// the warps, then one thread per value over the warps.  The CTA that finishes last adds
// the partials of all, each value by one warp in a fixed order (lane l every 32nd CTA from
// l on, then a shuffle tree), so the sums do not depend on which CTA that is.  `ticket`
// counts finished CTAs and is left at zero.  (A second kernel for the partials, which
// added the values one after another, took 17 us.)
template <int NV>
__device__ __forceinline__ void domain_sums(const double (&acc)[NV], double *partials, unsigned *ticket,
                                            double *__restrict__ sums)
{
    __shared__ double red[kReduceThreads / 32][8];
    __shared__ int last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        double v = acc[k];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
        if (lane == 0) red[warp][k] = v;
    }
    __syncthreads();
    if (threadIdx.x < NV) {
        double v = 0.0;
        for (int w = 0; w < kReduceThreads / 32; ++w) v += red[w][threadIdx.x];
        partials[(int64_t)blockIdx.x * 8 + threadIdx.x] = v;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (warp < NV) {
        double v = 0.0;
        for (int b = lane; b < (int)gridDim.x; b += 32) v += __ldcg(partials + (int64_t)b * 8 + warp);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
        if (lane == 0) sums[warp] = v;
    }
    if (threadIdx.x == 0) *ticket = 0u;
}

// Per-domain description (host and device copies).
struct Domain {
    int nx, ny, nz;
    int64_t ncell;
    int64_t stride;        // elements between slot planes
    int64_t offset;        // element offset of the domain's block in the buffer
    double gamma;
    double tau[kMaxLat];
    double source[kMaxLat];
    double q_ref[kMaxLat];
    double q_scale[kMaxLat];
    double force[3];
    double b_wall[3];
    int walls_y;
    double tau_m;          // Powell model: relaxation time of D (steps)
};

// Slab decomposition: the slot planes of a slab's two faces that wrap in the
// odd step (k_slab.cu).  lo: first layer, directions with c_a = +1; hi: last
// layer, directions with c_a = -1 (a = z in 3-D, y in 2-D).
// A slot may keep one row of the face layer out of the exchange (-1: none):
// with walls, the rows next to a wall hold the halfway bounce-back of their own
// cell in some c_a != 0 slots, which never stream across a face.
constexpr int kMaxHaloSlots = 32;
struct HaloSlots {
    int n;                  // slots per face
    int lo[kMaxHaloSlots];
    int hi[kMaxHaloSlots];
    int lo_keep[kMaxHaloSlots];  // row y of the face layer that stays (3-D), or -1
    int hi_keep[kMaxHaloSlots];
};

}  // namespace vlbm

struct vlbm_ctx {
    vlbm_params params;                 // parameters of domain 0 (copied)
    int model = 0, dim = 3, q = 7, nlat = 8, nvar = 8;
    int storage = VLBM_F32;
    size_t elem = 4;                    // bytes per stored population
    int nslot = 56;                     // slots per cell (lattices x directions)
    std::vector<vlbm::Domain> dom;
    bool batched = false;

    void *pop = nullptr;                // population buffer
    size_t pop_bytes = 0;
    unsigned *d_flags = nullptr;        // device status word; [1]: ticket of the domain sums
    unsigned *h_flags = nullptr;        // pinned host mirror of the status block (256 bytes)
    double *d_partials = nullptr;       // reduction scratch [kReduceBlocks x 8]
    double *d_sums = nullptr;           // reduction result [8], 128 bytes after d_flags
    double *d_refscale = nullptr;       // q_ref[8] then q_scale[8] of domain 0 (deviation storage, FP64)
    double h_refscale[16] = {};         // host copy (the upload's source; kept alive with the context)
    double *d_q = nullptr;              // staging for host fields (lazily sized)
    size_t d_q_bytes = 0;
    double *h_stage = nullptr;          // pinned host staging
    size_t h_stage_bytes = 0;

    cudaStream_t stream = nullptr;
    bool own_stream = false;
    cudaStream_t copy_stream = nullptr;  // host-field staging copies (overlap the chunk kernels)
    int sms = 0;                         // streaming multiprocessors of the device
    int bulk_ctas = 0;                   // persistent grid of the bulk-load step (0: not sized yet)
    int double_slots = 0;                // CTAs (2-D: strips) of the two-step pass that the device holds
                                         // (0: not asked yet, -1: the pass is not taken)
    void *double_doms = nullptr, *double_tiles = nullptr;  // 2-D: its constants and strip table
    int double_ntiles = 0;
    void *pop2 = nullptr;                // the two-step pass's other buffer (scratch between its two launches)
    bool chain = false;                  // step launches of the current call may be chained (launch_step_kernel)
    bool pop2_tried = false;
    bool two_step = true;                // vlbm_set_two_step
    bool pop2_captured = false;          // a graph of the caller's may hold pop2
    cudaEvent_t ev_copy[2]{}, ev_kern[2]{};  // per staging buffer: last copy / last kernel done
    cudaEvent_t flag_event = nullptr;
    bool flag_pending = false;
    int64_t steps_since_check = 0;

    int64_t step = 0;                   // completed (enqueued) steps
    int64_t launches = 0;               // kernels launched by this context
    vlbm_status sticky = VLBM_OK;
    std::string err;

    std::map<int, cudaGraphExec_t> graphs;  // key: parity*1024 + length
    std::map<int, int64_t> graph_launches;  // kernels one replay of that graph launches

    // batched form
    std::vector<void *> tile_tables;    // per tile shape: device (domain, first cell) pairs
    std::vector<int> tile_counts;       // tiles per table
    std::vector<int> tile_grid;         // CTAs launched per table
    int tune_choice = 0;
    void *d_dom = nullptr;              // device copy of the domain table

    // learned flux closure applied in every step (not owned)
    struct vlbm_closure *closure = nullptr;
    const float *solid = nullptr;       // homogenised solids: [7][N] caller-owned fields, or null
    // static equilibrium boundaries, faces x-, x+, y-, y+, z-, z+
    int face_kind[6] = {0, 0, 0, 0, 0, 0};  // VLBM_BC_PERIODIC or VLBM_BC_EQUILIBRIUM
    unsigned face_mask[6] = {0, 0, 0, 0, 0, 0};  // bit k: Q_k Dirichlet (else Neumann)
    double face_vals[6][8] = {};             // Dirichlet values

    // slab of a decomposed domain (k_slab.cu): the face planes move between
    // slabs after every step; halo_pending: a step ran and its exchange has
    // not been unpacked yet
    bool slab = false;
    bool halo_pending = false;
    vlbm::HaloSlots halo{};
    void *halo_buf = nullptr;           // vlbm_slabs_step: this slab's packed lo then hi message

    // allocator
    std::vector<std::pair<void *, size_t>> owned;
};

namespace vlbm {

// A named range on the host timeline of profilers that read NVTX (header-only NVTX3: without
// an attached tool each push and pop is a test of one pointer).
struct NvtxRange {
    explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange &) = delete;
    NvtxRange &operator=(const NvtxRange &) = delete;
};

// host helpers (vlbm_api.cu)
vlbm_status fail(vlbm_ctx *c, vlbm_status s, const std::string &msg);
vlbm_status cuda_check(vlbm_ctx *c, cudaError_t e, const char *what);

// launchers (k_ideal.cu)
vlbm_status ideal_init(vlbm_ctx *c, int d, const double *Q_dev);
vlbm_status ideal_init_range(vlbm_ctx *c, int d, const double *Q, int64_t c0, int64_t n, int64_t qstride);
vlbm_status ideal_moments_range(vlbm_ctx *c, int d, double *out, int64_t c0, int64_t n, int64_t ostride);
vlbm_status ideal_step(vlbm_ctx *c, int parity);
bool ideal_double_ok(vlbm_ctx *c);
vlbm_status ideal_double(vlbm_ctx *c, const void *in, void *out);

// launchers (k_double2d.cu): the 2-D two-step pass, single and batched domains
bool double_2d_ok(vlbm_ctx *c);
vlbm_status double_2d_prepare(vlbm_ctx *c);
vlbm_status double_2d(vlbm_ctx *c, const void *in, void *out);
vlbm_status ideal_moments(vlbm_ctx *c, int d, double *Q_dev);
vlbm_status ideal_gather(vlbm_ctx *c, int d, const int64_t *cells_dev, int n, double *out_dev);
vlbm_status ideal_sums(vlbm_ctx *c, int d, double *sums_dev);

// launchers (k_resistive.cu)
vlbm_status resistive_init(vlbm_ctx *c, int d, const double *Q_dev);
vlbm_status resistive_init_range(vlbm_ctx *c, int d, const double *Q, int64_t c0, int64_t n, int64_t qstride);
vlbm_status resistive_moments_range(vlbm_ctx *c, int d, double *out, int64_t c0, int64_t n, int64_t ostride);
vlbm_status resistive_step(vlbm_ctx *c, int parity);
vlbm_status resistive_moments(vlbm_ctx *c, int d, double *Q_dev);
vlbm_status resistive_gather(vlbm_ctx *c, int d, const int64_t *cells_dev, int n, double *out_dev);
vlbm_status resistive_sums(vlbm_ctx *c, int d, double *sums_dev);

// launchers (k_diss.cu): dissipative model, 2-D, F32 / F64 storage
vlbm_status diss_step(vlbm_ctx *c, int parity);
vlbm_status diss_init_range(vlbm_ctx *c, const double *Q, int64_t c0, int64_t n, int64_t qstride);
vlbm_status diss_moments_range(vlbm_ctx *c, double *out, int64_t c0, int64_t n, int64_t ostride);
vlbm_status diss_gather(vlbm_ctx *c, const int64_t *cells_dev, int n, double *out_dev);

// launchers (k_batch.cu)
vlbm_status batch_prepare(vlbm_ctx *c);
vlbm_status batch_step(vlbm_ctx *c, int parity, int choice);
int batch_num_choices();

// learned closure (k_closure.cu / k_ideal.cu)
vlbm_status ideal_step_corrected(vlbm_ctx *c, int parity, const float *dphi);
// porosity of the signed distance (HLBM), elementwise
vlbm_status porosity_from_distance(const float *phi, int64_t n, double eps_h, float *d, cudaStream_t s);
bool any_open_face(const vlbm_ctx *c);
// failure-detection self-check: a bounded wait that must give up (k_ideal.cu)
vlbm_status wait_check(vlbm_ctx *c, uint32_t tries);
vlbm_status open_fill(vlbm_ctx *c, int parity);
// closure input features of a 3-D FP32 context straight from its populations:
// x[cell][k] = BF16((Q_k - mu_k) * inv_sigma_k), Q_k summed in FP32 as by ideal_moments
vlbm_status ideal_features(vlbm_ctx *c, const float *mu, const float *inv_sigma, __nv_bfloat16 *x);
vlbm_status closure_step(vlbm_ctx *c, int parity);
int closure_cells(const vlbm_closure *cl, int *nx, int *ny, int *nz);

// precision of staged host fields (k_convert.cu): nvar fields of n values each,
// field v at v * stride, enqueued on the context's stream
vlbm_status widen_fields(vlbm_ctx *c, const float *in, int nvar, int64_t n, int64_t stride, double *out);
vlbm_status narrow_fields(vlbm_ctx *c, const double *in, int nvar, int64_t n, int64_t stride, float *out);

// slab halo (k_slab.cu): the face slot list of the context's model, and one
// launch that packs (face planes -> lo, hi messages) or unpacks (the reverse)
HaloSlots halo_slots(const vlbm_ctx *c);
vlbm_status halo_copy(vlbm_ctx *c, void *lo, void *hi, bool pack);

}  // namespace vlbm
