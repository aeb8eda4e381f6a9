// fvv_internal.h -- device-side descriptors shared by the kernels and the
// host runtime of libfvv.  Not part of the public ABI (see include/fvv.h).
#pragma once

#include <cmath>
#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

namespace fvv {

constexpr int kMaxCams = 64;
constexpr int kSrcBits = 26;
constexpr unsigned long long kKeyEmpty = ~0ull;
constexpr uint16_t kDepthBg = 65535;   // depth code of a background pixel
constexpr int kSplatSeg = 256;       // source pixels per splat warp (8 per lane, stride 32)
constexpr int kSplatThreads = 256;
constexpr int kResolveThreads = 256;

constexpr int kFlagCrack = 1;
constexpr int kFlagFill = 2;
constexpr int kFlagLayered = 4;
constexpr int kFlagPixelWeights = 8;

// Per (view, camera) quantities, composed on the host in FP64 and rounded
// to FP32 once (Sec. VI geometry).  M maps (u z, v z, z, 1) of the camera to
// (X, Y, Z) of the view; N maps (x Z, y Z, Z, 1) of the view to the camera.
struct alignas(16) CamGeom {
    float M[12];
    float N[12];
    float w;          // blend weight, 0 = inactive
    float pad[3];     // the camera's centre in the view's frame, depth units (per-pixel weights)
};

// One camera's frame in one slot of the device-resident frame ring.
struct alignas(16) FrameRef {
    const uint16_t* depth;   // [H][dpitch] depth codes, 0 = none, kDepthBg = background
    const uint32_t* rgba;    // [H][rpitch] R | G << 8 | B << 16
    const uint16_t* bg;      // [H][dpitch] static background depth model, or NULL
    int32_t W, H;
    int32_t dpitch;          // elements; rows 128-B aligned
    int32_t rpitch;          // elements
};

// One view of a batched launch.
struct alignas(16) ViewDesc {
    int32_t Wv, Hv;
    int32_t n_cams;
    int32_t n_active;
    int32_t slot;
    int32_t flags;
    float tau_crack, tau_vis, z_min;
    uint32_t d_lo, d_hi;
    float eps;                       // tolerance of the division-free rounding: the largest map_eps of its cameras
    float vk[4];                     // the view's cx, cy, 1/fx, 1/fy (per-pixel weights)
    unsigned long long* keys;        // scratch z-buffer [Hv * Wv] (the FG layer when layered)
    unsigned long long* keys_bg;     // layered: the BG layer's z-buffer [Hv * Wv], else NULL
    unsigned long long* keys_bgf;    // layered: the BG layer after the crack filter (keys_bg without it)
    unsigned long long* keys_next;   // nullable [Hv * Wv]: set to the empty key by the resolve (the
                                     // next batch's z-buffer, so that it needs no clear; single layer)
    uint8_t* out_rgb;                // [Hv] rows of 3 * Wv bytes
    int64_t out_pitch;               // bytes
    float* out_depth;                // nullable [Hv * Wv]
    uint8_t* out_hole;               // nullable [Hv * Wv]
    float* out_top3;                 // nullable [Hv * Wv * 3]
    unsigned long long* out_keys;    // nullable [Hv * Wv], after the crack filter
    const CamGeom* geom;             // [n_cams]
    int32_t active[kMaxCams];        // cameras with w > 0, ascending
    int32_t chunk_begin[kMaxCams + 1];  // prefix of splat warp segments over `active`
};

// Tolerance of the division-free rounding (fvv_kernels.cu, round_quotient2)
// for quotients that matter below `dim` (the larger side of the target
// image): half a last place below 2^ceil(log2 dim), and 2^-20 for the error
// of the fraction and the one threshold off an exact half (at quotient 1/2).
// m: the Z row of the map, applied to (x z, y z, z, 1) with x < W, y < H and
// z up to zhi.  Infinite (every point by division) where images beyond 2^20
// pixels a side leave the fraction too coarse, or where Z might leave the
// range whose reciprocal is a normal number: above 2^100, or, unless z_min
// keeps it off, nonzero below 2^-120 (Z is a multiple of its terms' last
// places, so coefficients that are zero or at least 2^-70 rule that out).
inline float settle_eps(int dim, float m0, float m1, float m2, float m3, float W, float H,
                                            float zhi, float zmin)
{
    const float b0 = m0 < 0 ? -m0 : m0, b1 = m1 < 0 ? -m1 : m1, b2 = m2 < 0 ? -m2 : m2, b3 = m3 < 0 ? -m3 : m3;
    const float big = (b0 * W + b1 * H + b2) * zhi + b3;
    const float tiny = 8.4703295e-22f;                                   // 2^-70
    const bool low = zmin < 7.8886091e-31f &&                            // 2^-100
                     ((b0 != 0.0f && b0 < tiny) || (b1 != 0.0f && b1 < tiny) || (b2 != 0.0f && b2 < tiny) ||
                      (b3 != 0.0f && b3 < tiny));
    if (dim > (1 << 20) || !(big < 1.2676506e30f) || low) return HUGE_VALF;
    int k = 0;
    while ((1 << k) < dim) ++k;
    return 2.9802322e-08f * float(1u << k) + 9.5367432e-07f;             // 2^(k - 25) + 2^-20
}

// Depths of view pixels for which a back-projection's tolerance holds: 2^-20
// to 2^60 (pixels outside take the division).
constexpr uint32_t kZNormLoBits = 0x35800000u, kZNormHiBits = 0x5D800000u;
constexpr float kZNormHi = 1.152921504606847e18f;

// That tolerance for back-projections from a Wv x Hv view into a W x H camera,
// the only ones that round without dividing (the splat divides).
inline float map_eps(const CamGeom& G, int W, int H, int Wv, int Hv, float z_min)
{
    return settle_eps(W > H ? W : H, G.N[8], G.N[9], G.N[10], G.N[11], float(Wv), float(Hv), kZNormHi, z_min);
}

// Persistent serving kernel (fvv_kernels.cu): one cooperative launch that
// takes batches of views from a ring the host writes, and runs steps a-e of
// each (clear, splat, resolve, separated by grid barriers).  The ring lives
// in pinned, mapped host memory; the kernel reads it through its device
// alias.  Every wait of the kernel is bounded by %globaltimer.
struct PersistBatch {
    const ViewDesc* views;             // device: the batch's parameter block
    const FrameRef* frames;            // device: the frame ring's table
    unsigned long long* keys;          // the batch's z-buffers, cleared first
    unsigned long long n_keys;
    int32_t n_views, max_h, band, splat_bx;
    int32_t keep, pad[3];
};
constexpr int kPersistRing = 16;
struct PersistQueue {
    PersistBatch batch[kPersistRing];   // batch b at b % kPersistRing
    volatile uint32_t posted;           // batches written so far (set after the batch)
    volatile uint32_t stop;             // 1: return at the next wait for work
    volatile uint32_t done;             // batches completed (set after their outputs)
    volatile int32_t err;               // 0, or the code of the wait that ran out
};
// Device memory of the kernel's grid barrier; zeroed before every launch.
struct PersistSync {
    unsigned int count, gen;
    int cmd;                            // 0: run the batch, 1: return
    int err;
};
constexpr int kPersistErrBarrier = 11;  // a grid barrier ran out
// Launch the kernel on `stream` (cooperative, every CTA resident) to take
// batches first, first + 1, ...; it returns after idle_ns without work, on
// q->stop, or when a grid barrier waits longer than wait_ns.  max_w, n_cams
// size its shared memory; pixel_weights: the context's option.  *ctas: the grid
// size.
cudaError_t launch_serve_persistent(PersistQueue* q_dev, PersistSync* sync, uint32_t first, int max_w, int n_cams,
                                    bool pixel_weights, uint64_t idle_ns, uint64_t wait_ns, cudaStream_t stream,
                                    int* ctas);
// The grid of that kernel for views up to max_w wide (0: none fits).
int persist_grid(int max_w, int n_cams, bool pixel_weights);
// The band, whether the resolve keeps depths and the splat's CTAs per view that
// the kernel, launched for views up to kernel_max_w wide, uses for a batch
// (points: as launch_resolve takes them).
void persist_batch_shape(int n_views, int max_h, int max_w, int n_cams, size_t points, int kernel_max_w,
                         int max_chunks, int ctas, PersistBatch* batch);

// Programmatic dependent launch: a kernel launched with launch_behind may
// start its CTAs once every CTA of the kernel before it on the stream has
// called launch_dependents (or exited), and calls wait_primary, which returns
// when that kernel is complete, before it touches memory.  What overlaps is
// the launch itself: 1.5 us of the gap between two dependent kernels.
// Such a kernel lives while the kernels before it still write.  So it reads what
// a kernel may have written with plain loads: no __ldg and no __restrict__, which
// let the compiler take the read-only path, where data has to stay unwritten for
// the whole life of the kernel, or move a load above the wait.  (Tables that the
// host wrote, and frames and parameters that were complete before the kernel in
// front started, may take that path.)
#ifdef __CUDACC__
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_primary() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Both, at the head of a kernel that does nothing worth overlapping.
__device__ __forceinline__ void behind()
{
    launch_dependents();
    wait_primary();
}

template <class... P, class... A>
cudaError_t launch_behind(void (*kernel)(P...), dim3 grid, dim3 threads, size_t smem, cudaStream_t stream, A... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = threads;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}
#endif

// Launchers (fvv_kernels.cu).  All asynchronous on `stream`.
cudaError_t launch_clear_keys(unsigned long long* keys, size_t n, cudaStream_t stream);
// layered: FG/BG layers (each view's keys_bg set, frames' bg models used).
cudaError_t launch_warp_splat(const ViewDesc* views, int n_views, int max_chunks,
                              const FrameRef* frames, cudaStream_t stream, bool layered = false);
// Layered: the crack filter of the BG layer (keys_bg -> keys_bgf), one pass.
cudaError_t launch_crack_bg(const ViewDesc* views, int n_views, int max_h, int max_w, cudaStream_t stream);
// points: the source pixels of all views' active cameras.
cudaError_t launch_resolve(const ViewDesc* views, int n_views, int max_h, int max_w, int n_cams, size_t points,
                           bool top3, const FrameRef* frames, cudaStream_t stream, bool layered = false,
                           bool pixel_weights = false);
cudaError_t launch_pack_rgba(const uint8_t* rgb, size_t rgb_pitch, uint32_t* rgba,
                             int rpitch, int W, int H, cudaStream_t stream);
size_t resolve_smem_bytes(int max_w, int n_cams, bool layered = false);
// The current device's streaming-multiprocessor count (1 if it cannot be read).
int device_sms();

}  // namespace fvv

struct fvv_camera;
namespace fvv {
// fvv_api.cu: message returned by fvv_last_error() on this thread.
void set_last_error(const char* msg);
// fvv_api.cu: FP64 composition of one view (maps M, N and weights w per camera).
void compose_view_into(int n_cams, const fvv_camera* cams, const double look_at[3],
                       double depth_unit_m, int n_ref, const fvv_camera& view, CamGeom* g);
}  // namespace fvv
