// fvv_kernels.cu -- CUDA kernels (sm_103a) of the view-synthesis hot path.
//
// FVV Live, Sec. VI: each reference pixel with depth is a 3D point that is
// projected into the virtual camera; cracks from magnification are handled
// by backward warping plus filtering; the contributions of several reference
// cameras are mixed according to their distance to the virtual camera;
// disoccluded pixels are holes.
//
//   k_clear_keys   reset the per-view z-buffers to the empty key
//   k_warp_splat   (a) forward warp + (b) 64-bit atomicMin z-buffer splat
//   k_resolve      (c) crack filter + (d) backward fetch and blend +
//                  (e) row hole fill, fused: one CTA per band of output rows
//   k_pack_rgba    upload: RGB8 rows -> RGBA8 (one aligned 32-bit gather per texel)
//
// Layered form (Sec. VI, per-camera FG and BG layers): a pixel signalled BG
// (kDepthBg) is a point of the BG layer at its camera's static model depth,
// every other valid pixel a point of the FG layer; each layer has its own
// z-buffer, crack filter and visibility test, and the FG layer is stacked
// over the BG layer before the hole fill.  The kernels take it as a
// template parameter, so the single-layer form carries none of it.
//
// Every FP32 operation of the warp, the filter and the blend is an explicit
// round-to-nearest intrinsic (__fmul_rn / __fadd_rn / __fsub_rn / __fdiv_rn)
// in a fixed, FMA-free order -- each product and each sum rounded once, each
// quotient a correctly rounded division -- so the results are exactly the
// IEEE values of that sequence.  The resolve runs that sequence packed, two
// pixels an instruction, and where only a quotient's rounding to an integer
// matters it finds that without the division (round_quotient2).
#include <algorithm>
#include <climits>
#include <cstdlib>
#include <type_traits>

#include "fvv_internal.h"

namespace fvv {

namespace {

__host__ __device__ inline size_t align16(size_t x) { return (x + 15) & ~size_t(15); }

// One active camera of a view, staged in the resolve kernel's shared memory
// and read by every lane at the same place.  (A broadcast 16-byte load still
// returns 512 bytes and takes about three wavefronts; constant-bank operands
// were slower, as the packed operations take theirs from registers, and so
// were records with every coefficient stored twice.)
struct alignas(16) RCam {
    float n0, n4, n8, w;             // backward map N by columns; the per-view blend weight
    float n2, n6, n10;
    int32_t k;                       // camera index
    float n3, n7, n11, unused;
    const uint16_t* depth;           // the camera's frame in the view's slot
    const uint32_t* rgba;
    int32_t dpitch, rpitch;          // elements
    uint32_t maxu, maxv;             // W - 1, H - 1
};
static_assert(sizeof(RCam) == 80, "RCam layout");

// What only the layered form and the per-pixel weights need of an active camera.
struct alignas(16) RExt {
    float4 cen;                // the camera's centre in the view's frame (per-pixel weights)
    const uint16_t* bg;        // layered: the static BG depth model, or NULL
    const void* unused;
};

// What a pixel's winner needs, by camera index (lanes read different entries).
struct alignas(16) RWin {
    const uint32_t* rgba;
    uint32_t magic, shift;     // s / W == (s * magic) >> shift for every s < 2^26
    uint32_t W, rpitch;
    float w;
    int32_t pos;               // position in the active list
};
static_assert(sizeof(RWin) == 32, "RWin layout");

constexpr int kSplatOcc = 5;                  // resident CTAs per SM the registers are held to, splat
constexpr int kResolveOcc = 3;                // likewise, resolve
// Cameras whose projections and gathers are in flight together: more cost
// registers (32 1280x720 views of nine cameras: 1710, 1549, 1568 and 1702 us
// with one to four).  One where per-pixel weights are in the group, too, whose
// code is long (eight 1080p views of three cameras 638 us with one, 719 with
// two), but not with layers (eight 1280x720 views of five 495 and 485 us).
constexpr int kGroup = 2;
// The wide form: four cameras at a time, three with per-pixel weights, in up to
// 96 registers, which the persistent serving kernel leaves beside it.  For
// launches of at most two CTAs per SM, where a gather's latency is all that counts
// (248x158 from eight 1074x810 cameras 41.0 us for 42.9, 296x220 from ten 25.4 for
// 26.5; four with per-pixel weights spill, 30.9 us for 30.0).  With up to four
// CTAs per SM it loses (one 1280x720 view 84 us for 77).  Never with the top-3
// output: its lists of a pixel's largest weights overfill the general form's
// registers as it is (24 to 44 bytes spilled; four 1280x720 views of nine cameras
// with it 267 us, 291 with a pixel a lane).
constexpr int kWideGroup = 4, kWideCtas = 2, kWideRegs = 96;
constexpr int kPairs = 1;                     // pixel pairs per lane: a warp's block is 64 kPairs pixels
constexpr int kBlock = 64 * kPairs;
constexpr int kResolveMaxBand = 4;            // output rows per resolve CTA
// Shared memory of a multi-row band: three CTAs per SM, and without kept depths
// (dense sources, so many gathers) some L1 left beside them.  Three rows of nine
// 1280x720 cameras, 67 KB, took 1.47 times as long as two; two rows of a
// magnified 1440x739 view, 70 KB, 0.91 times as long as one.
constexpr size_t kResolveSmem = 64 * 1024, kResolveSmemKept = 75 * 1024;
constexpr double kBandStart = 0.25;
// Whether the resolve keeps every pixel's depth in shared memory for the hole
// fill, or takes the two depths of a hole's sides from the keys again.  Kept,
// it is a sixth of the shared memory, and what the resident CTAs leave of that
// is the L1 that the gathers live in (1 to 4 % of a 32-view 1280x720 launch, nine
// points a pixel, 2 % holes); taken again, it is a hundred instructions a hole,
// which a magnified view is full of (1298x697 from nine 246x154 cameras, 0.4
// points a pixel: 88 us taken again, 53 us kept).  The line: fewer source points
// than this a pixel.
constexpr double kKeepPoints = 2.0;

constexpr uint32_t kHoleBit = 1u << 24;   // of a staged colour: no camera contributed

struct SmemLayout {
    size_t keys, rgb, dep, mask, cams, rows, ext, win, total;
};

// A staged key row: Wv keys from index 2 on (16-byte aligned rows) between
// one EMPTY sentinel on each side, so the crack filter reads x - 1 and x + 1
// without bounds tests.
__host__ __device__ inline int key_pitch(int W) { return (W + 4) & ~1; }
__host__ __device__ inline int rgb_pitch(int W) { return (W + 3) & ~3; }    // staged colours: 16-byte aligned rows
__host__ __device__ inline int row_chunks(int W) { return (W + kBlock - 1) / kBlock * (kBlock / 32); }   // 32-pixel chunks, whole blocks

// keep: every pixel's depth, for the hole fill (see kKeepPoints).
__host__ __device__ inline SmemLayout resolve_layout(int W, int n_cams, int band, bool keep)
{
    SmemLayout L;
    size_t o = 0;
    L.keys = o;   o = align16(o + size_t(band + 2) * key_pitch(W) * sizeof(unsigned long long));
    L.rgb = o;    o = align16(o + size_t(band) * rgb_pitch(W) * 4);
    L.dep = o;    o = align16(o + (keep ? size_t(band) * W * 4 : 0));
    L.mask = o;   o = align16(o + size_t(band) * row_chunks(W) * 4);
    L.cams = o;   o = align16(o + size_t(n_cams) * sizeof(RCam));
    L.rows = o;   o = align16(o + size_t(band) * n_cams * sizeof(float4));
    L.ext = o;    o = align16(o + size_t(n_cams) * sizeof(RExt));
    L.win = o;    o = align16(o + size_t(n_cams) * sizeof(RWin));
    L.total = o;
    return L;
}

__device__ __forceinline__ float key_z(unsigned long long k)
{
    return __uint_as_float(static_cast<uint32_t>(k >> 32));
}

}  // namespace

// ---------------------------------------------------------------------------
// z-buffer reset
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_clear_keys(unsigned long long* __restrict__ keys, size_t n)
{
    const size_t stride = size_t(gridDim.x) * blockDim.x;
    const size_t i0 = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    const size_t npair = n >> 1;
    for (size_t j = i0; j < npair; j += stride)
        asm volatile("st.global.L2::cache_hint.v2.u64 [%0], {%1, %2}, %3;" ::"l"(keys + 2 * j),
                     "l"(kKeyEmpty), "l"(kKeyEmpty), "l"(pol)
                     : "memory");
    if ((n & 1) && i0 == 0)
        keys[n - 1] = kKeyEmpty;
}

// ---------------------------------------------------------------------------
// cache-policy helpers (PTX createpolicy / cache_hint forms, sm_80+)
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint64_t policy_evict_first()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}

__device__ __forceinline__ uint64_t policy_evict_last()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}

// fire-and-forget 64-bit atomic minimum, kept in L2
__device__ __forceinline__ void red_min_key(unsigned long long* ptr, unsigned long long v, uint64_t pol)
{
    asm volatile("red.global.min.L2::cache_hint.u64 [%0], %1, %2;" ::"l"(ptr), "l"(v), "l"(pol)
                 : "memory");
}

// streaming loads (read once)
__device__ __forceinline__ uint32_t ld_stream_u16(const uint16_t* ptr, uint64_t pol)
{
    unsigned short v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.u16 %0, [%1], %2;"
                 : "=h"(v) : "l"(ptr), "l"(pol));
    return v;
}

__device__ __forceinline__ uint4 ld_stream_v4(const void* ptr, uint64_t pol)
{
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(ptr), "l"(pol));
    return v;
}

// Loads of frame data.  kCoh = false: the read-only (non-coherent) paths,
// for kernels during whose life the frames do not change.  kCoh = true
// (the persistent serving kernel, which outlives frame uploads): weak loads,
// which a gpu-scope acquire fence makes observe the latest writes.
template <bool kCoh, class T>
__device__ __forceinline__ T ld_frame(const T* p)
{
    if constexpr (kCoh) return *p;
    else return __ldg(p);
}

template <bool kCoh>
__device__ __forceinline__ uint32_t ld_depth_stream(const uint16_t* ptr, uint64_t pol)
{
    if constexpr (kCoh) return *ptr;
    else return ld_stream_u16(ptr, pol);
}

// Exact integer -> float conversion on the FP32/ALU pipes: for 0 <= d < 2^23,
// 2^23 + d is exactly representable and its low mantissa bits are d.
__device__ __forceinline__ float u23_to_float(uint32_t d)
{
    return __fsub_rn(__uint_as_float(0x4B000000u | d), 8388608.0f);
}

// R3's target pixel of a projected point: u' = X / Z and v' = Y / Z by
// correctly rounded division, then floor(u' + 0.5) (ties up), and the bounds
// test 0 <= t <= max as one unsigned compare per axis.  The float -> int
// floor saturates, so +-inf and out-of-range values fail the test as in the
// FP32 form; Z > z_min >= 0 (validated on the host) and a finite X, Y rule
// out NaN.  This is the defining form: the splat runs it for every point, the
// resolve only for the few that the division-free form below does not settle.
__device__ __forceinline__ uint2 target_pixel_div(float X, float Y, float Z)
{
    return make_uint2(static_cast<uint32_t>(__float2int_rd(__fadd_rn(__fdiv_rn(X, Z), 0.5f))),
                      static_cast<uint32_t>(__float2int_rd(__fadd_rn(__fdiv_rn(Y, Z), 0.5f))));
}

// Two FP32 values in one 64-bit register pair, and the packed operations on
// them: each half is the IEEE round-to-nearest operation, so a packed
// instruction gives the bits of two scalar ones at one issue slot.
using f32x2 = unsigned long long;

// ptxas contracts a packed product and the sum that takes it into one fused
// operation, .rn or not and with contraction switched off (the scalar forms
// are left alone).  So a product is written as a * b + (-0), which is the
// rounded product to the bit, with a -0 that the compiler cannot see through:
// it is memory that a program could change.
__device__ float2 g_neg_zero = {-0.0f, -0.0f};

__device__ __forceinline__ f32x2 neg_zero2() { return *reinterpret_cast<const volatile f32x2*>(&g_neg_zero); }

__device__ __forceinline__ f32x2 pk(float lo, float hi)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 upk(f32x2 a)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// a * b rounded once; nz = neg_zero2()
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b, f32x2 nz) { return fma2(a, b, nz); }
__device__ __forceinline__ f32x2 fma2_down(f32x2 a, f32x2 b, f32x2 c)   // rounded towards -inf
{
    f32x2 r;
    asm("fma.rm.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// floor(RN(RN(X / Z) + 0.5)) of two quotients without dividing.  With an
// approximate reciprocal r of Z, m = floor(X r) is the integer part of X / Z
// or its neighbour, and f = X - m Z is exact: a multiple of the coarser of
// Z's and X's last places that is no longer than Z.  So phi = f r is the
// fraction to a few 2^-23, and the answer is m or m + 1 according to phi
// against 1/2.  The two roundings of the defining form move that threshold
// by at most half a last place of the quotient (2^(k - 25) for quotients
// below 2^k) -- where phi comes that close to 1/2 the point is unsettled and
// the caller takes the defining form.  The integers live in the low bits of
// floats offset by 1.5 * 2^23, so rounding to an integer is one addition; a
// quotient beyond +-2^22 gives bits outside every bounds test, and a NaN
// (an overflowed reciprocal) is unsettled.
// t: the offset float's bits minus kMagicBits are the answer.
// near: phi - 1/2, whose magnitude is to be compared with settle_eps().
constexpr uint32_t kMagicBits = 0x4B400000u;       // 1.5 * 2^23

__device__ __forceinline__ void round_quotient2(f32x2 X, f32x2 Z, f32x2 r, f32x2& t, f32x2& near)
{
    const f32x2 magic = pk(12582912.0f, 12582912.0f), minus_one = pk(-1.0f, -1.0f), minus_half = pk(-0.5f, -0.5f);
    const f32x2 m = fma2_down(X, r, magic);
    const f32x2 f = fma2(fma2(m, minus_one, magic), Z, X);
    t = fma2(f, r, m);
    near = fma2(f, r, minus_half);
}

__device__ __forceinline__ bool target_pixel(float X, float Y, float Z, uint32_t maxu, uint32_t maxv,
                                             uint32_t& ui, uint32_t& vi)
{
    const uint2 t = target_pixel_div(X, Y, Z);
    ui = t.x;
    vi = t.y;
    return ui <= maxu && vi <= maxv;
}

// ---------------------------------------------------------------------------
// (a) + (b): forward warp and z-buffer splat.
// One warp = one segment of kSplatSeg consecutive source pixels of one row
// of one active camera.  kVec = false: lane l takes pixels l, l + 32, ...
// (2-byte loads), so every warp-wide atomic touches 32 consecutive source
// pixels, whose targets are neighbours in the view (few L2 sectors per
// atomic).  kVec = true: lane l takes the 8 consecutive pixels 8l .. 8l+7
// with one 16-byte load.  Segments of a view are numbered camera-major over
// the active cameras: chunk_begin[a] .. chunk_begin[a+1).  Each CTA belongs
// to one view and stages its maps and frame table in shared memory.
// ---------------------------------------------------------------------------
// The work of one CTA (bx, by) of a grid of gdx x (views) CTAs; the kernel
// below is its one-launch form, the persistent serving kernel calls it for
// virtual CTAs in turn (kCoh: coherent frame loads, see ld_frame).
template <bool kLayered, bool kVec, bool kCoh, int NT>
__device__ __forceinline__ void splat_cta(const ViewDesc* __restrict__ views, const FrameRef* __restrict__ frames,
                                          int bx, int by, int gdx)
{
    // per active camera: (m0, m2, m3, m1), (m4, m6, m7, m5), (m8, m10, m11, m9)
    __shared__ __align__(16) float4 s_M[kMaxCams][3];
    __shared__ __align__(16) FrameRef s_F[kMaxCams];
    __shared__ int s_cb[kMaxCams + 1];
    __shared__ int s_act[kMaxCams];
    __shared__ uint2 s_div[kMaxCams];              // segment -> row: (magic, shift) of segments per row
    constexpr int kWarps = NT / 32;
    constexpr int kPer = kSplatSeg / 32;           // pixels per lane per segment
    static_assert(kPer == 8, "a 16-byte load holds 8 depth codes");
    if (kCoh) __syncthreads();                     // the previous virtual CTA's reads of the staging are done
    const ViewDesc* V = views + by;
    const int na = V->n_active;
    const int first = bx * kWarps;
    if (first >= V->chunk_begin[na])
        return;                                   // uniform over the CTA
    for (int i = threadIdx.x; i < na * 3; i += NT) {
        const int a = i / 3, r = i - a * 3;
        const float* m = V->geom[V->active[a]].M + 4 * r;
        s_M[a][r] = make_float4(m[0], m[2], m[3], m[1]);
    }
    for (int i = threadIdx.x; i < na; i += NT) {
        s_act[i] = V->active[i];
        const FrameRef F = frames[V->slot * V->n_cams + V->active[i]];
        s_F[i] = F;
        // local / spr for local < 2^26 as (local * magic) >> shift, with
        // shift = 26 + ceil(log2 spr) and magic = ceil(2^shift / spr): the
        // excess local * e / 2^shift stays below 1 / spr
        const uint32_t spr = uint32_t((F.W + kSplatSeg - 1) / kSplatSeg);
        const uint32_t lg = spr > 1 ? 32u - uint32_t(__clz(spr - 1)) : 0u;
        s_div[i] = make_uint2(uint32_t(((1ull << (26u + lg)) + spr - 1) / spr), 26u + lg);
    }
    for (int i = threadIdx.x; i <= na; i += NT)
        s_cb[i] = V->chunk_begin[i];
    __syncthreads();

    const int lane = threadIdx.x & 31;
    const int total = s_cb[na];
    const float zmin = V->z_min;
    const uint32_t dlo = V->d_lo, dspan = V->d_hi - V->d_lo;
    const uint32_t Wv = uint32_t(V->Wv);
    const uint32_t maxu = Wv - 1, maxv = uint32_t(V->Hv - 1);
    unsigned long long* __restrict__ keys = V->keys;
    unsigned long long* __restrict__ keys_bg = V->keys_bg;
    const uint64_t pol_stream = policy_evict_first();
    const uint64_t pol_keys = policy_evict_last();

    // persistent warps: segment seg, seg + stride, ... of this view; the
    // segments grow, so the camera search resumes where it stopped
    int a = 0;
    for (int seg = first + int(threadIdx.x >> 5); seg < total; seg += gdx * kWarps) {
        while (seg >= s_cb[a + 1])
            ++a;
        const int k = s_act[a];
        const FrameRef& F = s_F[a];
        const int spr = (F.W + kSplatSeg - 1) / kSplatSeg;
        const uint32_t local = uint32_t(seg - s_cb[a]);
        const uint2 dv = s_div[a];
        const int v = int((static_cast<unsigned long long>(local) * dv.x) >> dv.y);
        const int u0 = (int(local) - v * spr) * kSplatSeg;
        const uint16_t* row = F.depth + size_t(v) * F.dpitch;
        // the lane's first pixel and the step between its pixels
        const int ub = u0 + (kVec ? kPer * lane : lane);
        constexpr int kStep = kVec ? 1 : 32;

        uint32_t d[kPer];
        // 16-byte loads need 16-byte aligned rows; a vector lies wholly
        // inside or wholly past the row's pitch (pitch and ub multiples of 8)
        if (kVec && !kCoh && (F.dpitch & 7) == 0 && (reinterpret_cast<uintptr_t>(F.depth) & 15u) == 0) {
            uint4 q = make_uint4(0u, 0u, 0u, 0u);
            if (ub < F.dpitch)
                q = ld_stream_v4(row + ub, pol_stream);
            d[0] = q.x & 0xFFFFu; d[1] = q.x >> 16; d[2] = q.y & 0xFFFFu; d[3] = q.y >> 16;
            d[4] = q.z & 0xFFFFu; d[5] = q.z >> 16; d[6] = q.w & 0xFFFFu; d[7] = q.w >> 16;
#pragma unroll
            for (int j = 0; j < kPer; ++j)
                if (ub + j >= F.W) d[j] = 0u;
        } else {
#pragma unroll
            for (int j = 0; j < kPer; ++j) {
                const int u = ub + kStep * j;
                d[j] = u < F.W ? ld_depth_stream<kCoh>(row + u, pol_stream) : 0u;
            }
        }
        // layered: a BG-signalled pixel takes its depth from the model and
        // splats into the BG layer (bit j of bgm)
        uint32_t bgm = 0;
        if (kLayered) {
            const uint16_t* brow = F.bg ? F.bg + size_t(v) * F.dpitch : nullptr;
#pragma unroll
            for (int j = 0; j < kPer; ++j)
                if (d[j] == kDepthBg) {
                    d[j] = brow ? ld_depth_stream<kCoh>(brow + ub + kStep * j, pol_stream) : 0u;
                    bgm |= 1u << j;
                }
        }

        const float4 Mx = s_M[a][0], My = s_M[a][1], Mz = s_M[a][2];
        const float fv = u23_to_float(uint32_t(v));
        // per-row products m1 v, m5 v, m9 v (the order stays ((m0 u + m1 v) + m2))
        const float rx = __fmul_rn(Mx.w, fv), ry = __fmul_rn(My.w, fv), rz = __fmul_rn(Mz.w, fv);
        const unsigned long long khi = static_cast<unsigned long long>(k) << kSrcBits;
        const uint32_t src0 = uint32_t(v) * uint32_t(F.W) + uint32_t(ub);
        const float fu0 = u23_to_float(uint32_t(ub));

        // branch-free per point (only the atomic is predicated), so the eight
        // independent projections and divisions of a lane can interleave
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const uint32_t dd = d[j];
            const float fu = __fadd_rn(fu0, float(kStep * j));   // exact: small integers
            const float z = u23_to_float(dd);
            const float a0 = __fadd_rn(__fadd_rn(__fmul_rn(Mx.x, fu), rx), Mx.y);
            const float a1 = __fadd_rn(__fadd_rn(__fmul_rn(My.x, fu), ry), My.y);
            const float a2 = __fadd_rn(__fadd_rn(__fmul_rn(Mz.x, fu), rz), Mz.y);
            const float X = __fadd_rn(__fmul_rn(a0, z), Mx.z);
            const float Y = __fadd_rn(__fmul_rn(a1, z), My.z);
            const float Z = __fadd_rn(__fmul_rn(a2, z), Mz.z);
            uint32_t tu, tv;
            const bool hit = target_pixel(X, Y, Z, maxu, maxv, tu, tv);
            // dd in [dlo, dhi] (dlo >= 1, so a code of 0 wraps above the span)
            if (dd - dlo <= dspan && Z > zmin && hit) {
                const unsigned long long key =
                    (static_cast<unsigned long long>(__float_as_uint(Z)) << 32) | khi |
                    static_cast<unsigned long long>(src0 + uint32_t(kStep * j));
                unsigned long long* dst = (kLayered && ((bgm >> j) & 1u)) ? keys_bg : keys;
                red_min_key(dst + (tv * Wv + tu), key, pol_keys);
            }
        }
    }
}

template <bool kLayered, bool kVec>
__global__ void __launch_bounds__(kSplatThreads, kSplatOcc)
k_warp_splat(const ViewDesc* __restrict__ views, const FrameRef* __restrict__ frames)
{
    launch_dependents();
    splat_cta<kLayered, kVec, false, kSplatThreads>(views, frames, int(blockIdx.x), int(blockIdx.y), int(gridDim.x));
}

// ---------------------------------------------------------------------------
// (c) crack / outlier rule on the three staged key rows.  Pairs, in order:
// (left, right), (up, down), (up-left, down-right), (up-right, down-left).
// A pair is consistent when both keys are present and zmax <= (1+tau) zmin.
// An empty pixel takes min(a, b) of the first consistent pair; a present
// pixel takes it from the first consistent pair with z_p > (1+tau) zmax.
// ---------------------------------------------------------------------------
// The rule for a pixel whose neighbour at (dy, dx) is get(dy, dx).
template <class Get>
__device__ __forceinline__ unsigned long long crack_rule_at(Get get, unsigned long long kp, float f1)
{
    const int ady[4] = {0, -1, -1, -1}, adx[4] = {-1, 0, -1, 1};
    const int bdy[4] = {0, 1, 1, 1}, bdx[4] = {1, 0, 1, -1};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const unsigned long long a = get(ady[q], adx[q]);
        const unsigned long long b = get(bdy[q], bdx[q]);
        if (a == kKeyEmpty || b == kKeyEmpty)
            continue;
        const float za = key_z(a), zb = key_z(b);
        const float zlo = za < zb ? za : zb;
        const float zhi = za < zb ? zb : za;
        if (!(zhi <= __fmul_rn(f1, zlo)))
            continue;
        if (kp == kKeyEmpty || key_z(kp) > __fmul_rn(f1, zhi))
            return a < b ? a : b;
    }
    return kp;
}

// The rule at mid, all of whose neighbours are in memory (padded rows whose
// index -1 and Wv hold EMPTY, or a pixel off the image's border).  It works on
// the high words alone, which are the depths' bits: positive depths order like their bits, and EMPTY's high word is
// the largest and, as a float, a NaN, which fails every comparison it should.
// A present pixel no deeper than (1+tau) times its nearest present neighbour
// keeps its key without the pair walk: every consistent pair's far depth is at
// least that neighbour's, and the rounded product is monotone, so no pair can
// satisfy z_p > (1+tau) zmax.  Nothing changes without a present neighbour,
// either.  The pairs are judged without a branch, the last first, and only the
// chosen one's keys are loaded: empty pixels, which a magnified view is full
// of, diverged at each pair before (1298x697 from
// nine cameras 61 us then, 53 us now; 1907x1003 from five 158 and 139 us).
__device__ __forceinline__ unsigned long long crack_rule_ptr(const unsigned long long* mid, int pitch, float f1)
{
    const unsigned long long kp = *mid;
    const int off[4] = {1, pitch, pitch + 1, pitch - 1};             // the pairs are mid[-off], mid[off]
    auto hi = [&](int o) { return reinterpret_cast<const uint32_t*>(mid + o)[1]; };
    uint32_t lo4[4], hi4[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint32_t a = hi(-off[q]), b = hi(off[q]);
        lo4[q] = min(a, b);
        hi4[q] = max(a, b);
    }
    const uint32_t zb = min(min(lo4[0], lo4[1]), min(lo4[2], lo4[3]));
    const float z = key_z(kp);                                       // a NaN where empty
    if (zb == 0xFFFFFFFFu || z <= __fmul_rn(f1, __uint_as_float(zb)))
        return kp;
    int o = 0;
#pragma unroll
    for (int q = 3; q >= 0; --q) {
        const float zhi = __uint_as_float(hi4[q]);
        if (zhi <= __fmul_rn(f1, __uint_as_float(lo4[q])) && !(z <= __fmul_rn(f1, zhi))) o = off[q];
    }
    const unsigned long long a = mid[-o], b = mid[o];                // (o == 0: the key itself)
    return a < b ? a : b;
}

// Layered form: the BG layer's crack filter as its own pass, read straight
// from the z-buffer (L1/L2), so the resolve stages one key ring only.  A CTA
// takes 64 x 4 pixels, so that its rows are read from L2 one and a half times
// and not three (eight 1280x720 views: 64 us with
// 256 x 1 pixels and a branch at each pair, 35 us so).
constexpr int kBgW = 64, kBgH = 4;
__global__ void __launch_bounds__(kBgW * kBgH) k_crack_bg(const ViewDesc* __restrict__ views)
{
    const ViewDesc* V = views + blockIdx.z;
    const int Wv = V->Wv, Hv = V->Hv;
    const int x = blockIdx.x * kBgW + threadIdx.x, y = blockIdx.y * kBgH + threadIdx.y;
    behind();
    if (x >= Wv || y >= Hv)
        return;
    const unsigned long long* kb = V->keys_bg + size_t(y) * Wv + x;
    const float f1 = __fadd_rn(1.0f, V->tau_crack);
    unsigned long long k;
    if (x > 0 && x < Wv - 1 && y > 0 && y < Hv - 1) {
        k = crack_rule_ptr(kb, Wv, f1);
    } else {
        auto get = [&](int dy, int dx) {
            const int yy = y + dy, xx = x + dx;
            return (yy < 0 || yy >= Hv || xx < 0 || xx >= Wv) ? kKeyEmpty : kb[ptrdiff_t(dy) * Wv + dx];
        };
        k = crack_rule_at(get, *kb, f1);
    }
    V->keys_bgf[size_t(y) * Wv + x] = k;
}

__device__ __forceinline__ void cp_async8(void* smem_dst, const void* gsrc)
{
    const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(smem_dst));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(gsrc) : "memory");
}

__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc)
{
    const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(smem_dst));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gsrc) : "memory");
}

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ bool w_before(float wa, int ka, float wb, int kb)
{
    return wa > wb || (wa == wb && ka < kb);
}

// min(|a|, |b|, |c|), NaN if any is
__device__ __forceinline__ float min3_abs(float a, float b, float c)
{
    float r;
    asm("min.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// min(255, floor(acc / wsum + 0.5)), each operation rounded as written
__device__ __forceinline__ uint32_t blend_channel(float acc, float wsum)
{
    float v = floorf(__fadd_rn(__fdiv_rn(acc, wsum), 0.5f));
    v = v > 255.0f ? 255.0f : v;
    return uint32_t(v);
}

// That value for the three channels of two pixels, as R | G << 8 | B << 16.
// acc is a sum of at most 64 terms w c with c <= 255 and wsum the sum of the
// same w, so the quotient stays below 255.01 and the minimum never acts.
__device__ __forceinline__ uint2 blend_rgb2(f32x2 accr, f32x2 accg, f32x2 accb, f32x2 wsum)
{
    constexpr float eps = 7.6293945e-06f + 9.5367432e-07f;               // settle_eps of 256
    const float2 ws = upk(wsum);
    const f32x2 r = pk(rcp_approx(ws.x), rcp_approx(ws.y));
    f32x2 tr, tg, tb, nr, ng, nb;
    round_quotient2(accr, wsum, r, tr, nr);
    round_quotient2(accg, wsum, r, tg, ng);
    round_quotient2(accb, wsum, r, tb, nb);
    const float2 a = upk(tr), b = upk(tg), c = upk(tb), na = upk(nr), nbb = upk(ng), ncc = upk(nb);
    const float mn = min3_abs(min3_abs(na.x, nbb.x, ncc.x), min3_abs(na.y, nbb.y, ncc.y), 1.0f);
    if (mn > eps) {
        // the low byte of each offset float is the value
        auto rgb = [](float x, float y, float z) {
            return __byte_perm(__byte_perm(__float_as_uint(x), __float_as_uint(y), 0x3340), __float_as_uint(z), 0x3410) &
                   0xFFFFFFu;
        };
        return make_uint2(rgb(a.x, b.x, c.x), rgb(a.y, b.y, c.y));
    }
    const float2 R = upk(accr), G = upk(accg), B = upk(accb);
    return make_uint2(blend_channel(R.x, ws.x) | (blend_channel(G.x, ws.x) << 8) | (blend_channel(B.x, ws.x) << 16),
                      blend_channel(R.y, ws.y) | (blend_channel(G.y, ws.y) << 8) | (blend_channel(B.y, ws.y) << 16));
}

// A texel's depth code and colour where ok, zeros elsewhere, without a branch
// around the loads.
template <bool kCoh>
__device__ __forceinline__ void gather(bool ok, const uint16_t* d, const uint32_t* c, uint32_t& dk, uint32_t& ck)
{
    if constexpr (kCoh) {
        asm volatile("{\n"
                     ".reg .pred p;\n"
                     ".reg .u16 t;\n"
                     "setp.ne.u32 p, %4, 0;\n"
                     "mov.u16 t, 0;\n"
                     "mov.u32 %1, 0;\n"
                     "@p ld.global.u16 t, [%2];\n"
                     "@p ld.global.u32 %1, [%3];\n"
                     "cvt.u32.u16 %0, t;\n"
                     "}"
                     : "=&r"(dk), "=&r"(ck)
                     : "l"(d), "l"(c), "r"(uint32_t(ok)));
    } else {
        asm("{\n"
            ".reg .pred p;\n"
            ".reg .u16 t;\n"
            "setp.ne.u32 p, %4, 0;\n"
            "mov.u16 t, 0;\n"
            "mov.u32 %1, 0;\n"
            "@p ld.global.nc.u16 t, [%2];\n"
            "@p ld.global.nc.u32 %1, [%3];\n"
            "cvt.u32.u16 %0, t;\n"
            "}"
            : "=&r"(dk), "=&r"(ck)
            : "l"(d), "l"(c), "r"(uint32_t(ok)));
    }
}

// Per-pixel angular weight of a camera whose centre in the view's frame is
// (cx, cy, cz), at the surface point (px, py, pz) at distance lb from the
// view's centre: 1 / (chord + 0.001) with chord = sqrt(2 (1 - cos)) of the
// angle at the point between the rays to the camera and to the view.
__device__ __forceinline__ float pixel_weight(float cx, float cy, float cz, float px, float py, float pz, float lb)
{
    const float ax = __fsub_rn(cx, px), ay = __fsub_rn(cy, py), az = __fsub_rn(cz, pz);
    const float la = __fsqrt_rn(__fadd_rn(__fadd_rn(__fmul_rn(ax, ax), __fmul_rn(ay, ay)), __fmul_rn(az, az)));
    const float dot = __fadd_rn(__fadd_rn(__fmul_rn(ax, px), __fmul_rn(ay, py)), __fmul_rn(az, pz));
    const float q = __fdiv_rn(dot, __fmul_rn(la, lb));
    float t = __fadd_rn(1.0f, q);
    t = t > 0.0f ? t : 0.0f;
    const float chord = __fsqrt_rn(__fadd_rn(t, t));
    return __fdiv_rn(1.0f, __fadd_rn(chord, 0.001f));
}

// ---------------------------------------------------------------------------
// (c) + (d) + (e).  One CTA resolves a band of consecutive output rows of one
// view, launched view after view so that the resident CTAs share one view's
// frames in L2.  The band's key rows and their two neighbours are staged in
// shared memory.  A warp takes kBlock consecutive pixels of a row at a time,
// each lane 2 kPairs of them (x, x + 32, ...), so that every projection,
// rounding and sum runs packed over two pixels.  All lanes walk the view's
// active cameras together, kGroup at a time (their projections and gathers are
// issued before any is consumed): a camera's record is one broadcast load, and
// a pixel's own winner, whose contribution comes first, is masked when its turn
// comes.
// It is bound by instruction issue (three quarters of the slots, with 24 warps
// an SM that 80 registers and three CTAs' shared memory allow) and by what the
// shared memory leaves as L1 for the gathers.  32 views of 1280x720 from nine
// cameras take 899 us; 1169 us with a pixel a lane, sixteen divisions a pixel
// and a loop over each pixel's own list of other cameras, as it was.  Slower
// than this form: four pixels a lane (registers), larger CTAs or more of them
// (L1).
// kTop3: also track the three largest contributing weights (only when that
// output is requested).  kPixW: per-pixel angular weights (each contribution
// weighted by the angle at its surface point) instead of the view's
// per-camera weights.
// ---------------------------------------------------------------------------
template <bool kTop3, bool kLayered, bool kPixW, bool kCoh, int NT, bool kWide = false>
__device__ __forceinline__ void resolve_cta(const ViewDesc* __restrict__ views, const FrameRef* __restrict__ frames,
                                            int band, bool keep, int bx, int by, unsigned char* smem)
{
    if (kCoh) __syncthreads();                     // the previous virtual CTA is done with the shared memory
    const ViewDesc* V = views + by;
    const int Wv = V->Wv, Hv = V->Hv;
    const int y0 = bx * band;
    if (y0 >= Hv)
        return;                                    // uniform over the CTA
    const int rows = min(band, Hv - y0);
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31;
    const int wid = __shfl_sync(0xffffffffu, tid >> 5, 0);            // uniform to the compiler, too
    const int nc = V->n_cams, na = V->n_active;
    const SmemLayout L = resolve_layout(Wv, nc, band, keep);
    const int KP = key_pitch(Wv), RP = rgb_pitch(Wv);
    unsigned long long* s_keys = reinterpret_cast<unsigned long long*>(smem + L.keys);
    uint32_t* s_rgb = reinterpret_cast<uint32_t*>(smem + L.rgb);      // R | G << 8 | B << 16 | kHoleBit
    float* s_dep = reinterpret_cast<float*>(smem + L.dep);            // (keep)
    uint32_t* s_mask = reinterpret_cast<uint32_t*>(smem + L.mask);    // per 32-pixel chunk: the pixels that are no holes
    RCam* cams = reinterpret_cast<RCam*>(smem + L.cams);
    float4* s_row = reinterpret_cast<float4*>(smem + L.rows);         // [band][na]: N1 y, N5 y, N9 y
    RExt* s_ext = reinterpret_cast<RExt*>(smem + L.ext);
    RWin* s_win = reinterpret_cast<RWin*>(smem + L.win);

    if constexpr (!kCoh) wait_primary();           // the splat's keys
    // key rows y0 - 1 .. y0 + rows (empty outside the view), with sentinels;
    // 16 bytes a copy where the rows start on 16 bytes
    for (int i = 0; i < rows + 2; ++i) {
        unsigned long long* dst = s_keys + i * KP + 2;
        const int yy = y0 - 1 + i;
        if (tid == 0) dst[-1] = kKeyEmpty;
        if (tid == NT - 1) dst[Wv] = kKeyEmpty;
        if (yy >= 0 && yy < Hv) {
            const unsigned long long* src = V->keys + size_t(yy) * Wv;
            if (kCoh) {
                // written by other CTAs of the same kernel: L2 loads
                for (int x = tid; x < Wv; x += NT) dst[x] = __ldcg(src + x);
            } else if ((Wv & 1) == 0) {
                for (int x = 2 * tid; x < Wv; x += 2 * NT) cp_async16(dst + x, src + x);
            } else {
                for (int x = tid; x < Wv; x += NT) cp_async8(dst + x, src + x);
            }
        } else {
            for (int x = tid; x < Wv; x += NT) dst[x] = kKeyEmpty;
        }
    }
    cp_async_commit();

    // the active cameras' records, in active order
    for (int a = tid; a < na; a += NT) {
        const int k = V->active[a];
        const CamGeom& G = V->geom[k];
        const FrameRef& F = frames[V->slot * nc + k];
        RCam C;
        C.n0 = G.N[0]; C.n4 = G.N[4]; C.n8 = G.N[8]; C.w = G.w;
        C.n2 = G.N[2]; C.n6 = G.N[6]; C.n10 = G.N[10]; C.k = k;
        C.n3 = G.N[3]; C.n7 = G.N[7]; C.n11 = G.N[11]; C.unused = 0.0f;
        C.depth = F.depth;
        C.rgba = F.rgba;
        C.dpitch = F.dpitch;
        C.rpitch = F.rpitch;
        C.maxu = uint32_t(F.W - 1);
        C.maxv = uint32_t(F.H - 1);
        cams[a] = C;
        // s / W for s < 2^26: shift = 26 + ceil(log2 W), magic = ceil(2^shift / W);
        // then s * magic / 2^shift = s / W + e with 0 <= e < s / 2^shift < 1 / W,
        // which never carries past the next integer
        const uint32_t W = C.maxu + 1u, lg = W > 1u ? 32u - uint32_t(__clz(W - 1u)) : 0u;
        RWin Q;
        Q.rgba = C.rgba;
        Q.shift = 26u + lg;
        Q.magic = uint32_t(((1ull << Q.shift) + uint64_t(W) - 1) / uint64_t(W));
        Q.W = W;
        Q.rpitch = uint32_t(C.rpitch);
        Q.w = C.w;
        Q.pos = a;
        s_win[C.k] = Q;
        if (kLayered || kPixW) {
            RExt E;
            E.cen = make_float4(G.pad[0], G.pad[1], G.pad[2], 0.0f);
            E.bg = F.bg;
            E.unused = nullptr;
            s_ext[a] = E;
        }
    }
    // per-row products N1 y, N5 y, N9 y (the order stays ((N0 x + N1 y) + N2))
    for (int i = tid; i < rows * na; i += NT) {
        const int r = i / na;
        const float* N = V->geom[V->active[i - r * na]].N;
        const float fy = u23_to_float(uint32_t(y0 + r));
        s_row[i] = make_float4(__fmul_rn(N[1], fy), __fmul_rn(N[5], fy), __fmul_rn(N[9], fy), 0.0f);
    }
    if (!kLayered && !kCoh && V->keys_next) {
        // the next batch's z-buffer rows of this band, emptied while the key
        // rows are in flight (kept in L2 for that batch's splat); the buffer
        // starts on a 128-byte line, so even keys pair up
        const uint64_t pol = policy_evict_last();
        unsigned long long* kn = V->keys_next + size_t(y0) * Wv;
        const int n = rows * Wv, odd = int((size_t(y0) * Wv) & 1);
        if (tid == 0 && odd)
            asm volatile("st.global.L2::cache_hint.u64 [%0], %1, %2;" ::"l"(kn), "l"(kKeyEmpty), "l"(pol) : "memory");
        if (tid == 0 && ((n - odd) & 1))
            asm volatile("st.global.L2::cache_hint.u64 [%0], %1, %2;" ::"l"(kn + n - 1), "l"(kKeyEmpty), "l"(pol)
                         : "memory");
        for (int i = odd + 2 * tid; i < n - 1; i += 2 * NT)
            asm volatile("st.global.L2::cache_hint.v2.u64 [%0], {%1, %2}, %3;" ::"l"(kn + i), "l"(kKeyEmpty),
                         "l"(kKeyEmpty), "l"(pol)
                         : "memory");
    }

    const bool crack = (V->flags & kFlagCrack) != 0;
    const bool fill = (V->flags & kFlagFill) != 0;
    const float f1 = __fadd_rn(1.0f, V->tau_crack);
    const float tau_vis = V->tau_vis, zmin = V->z_min;
    const uint32_t dlo = V->d_lo, dspan = V->d_hi - V->d_lo;
    float* __restrict__ top3 = V->out_top3;
    // (the persistent kernel's views have no outputs but the colour, and no next z-buffer)
    float* __restrict__ odepth = kCoh ? nullptr : V->out_depth;
    unsigned long long* __restrict__ okeys = kCoh ? nullptr : V->out_keys;
    const f32x2 nz = neg_zero2();
    const float eps = V->eps;
    cp_async_wait<0>();
    __syncthreads();                          // key rows and records staged

    bool any_hole = false;
    const int nb = (Wv + kBlock - 1) / kBlock;                    // blocks per row
    const int nch = nb * (kBlock / 32);
    for (int r = 0, blk = wid;; blk += NW) {      // block blk of row r, row after row
        while (r < rows && blk >= nb) {
            blk -= nb;
            ++r;
        }
        if (r >= rows) break;
        const int xb = blk * kBlock + lane;
        const int y = y0 + r;
        const size_t rowbase = size_t(y) * Wv;
        const unsigned long long* up = s_keys + r * KP + 2;
        const float4* rowp = s_row + r * na;
        constexpr int P = 2 * kPairs;                                // pixel i of the lane: x = xb + 32 i
        bool bg_layer[P];
        int w[P];
        float Zs[P], zmn[P], ww[P];
        uint32_t cw[P];
        bool some = false, z_norm = true;
#pragma unroll
        for (int i = 0; i < P; ++i) {
            const int x = xb + 32 * i;
            const bool in = x < Wv;
            unsigned long long kk = kKeyEmpty;
            if (in) kk = crack ? crack_rule_ptr(up + KP + x, KP, f1) : up[KP + x];
            // layered: the FG layer is stacked over the BG layer, so the BG
            // layer is resolved only where the filtered FG layer is empty
            bg_layer[i] = false;
            if (kLayered && in && kk == kKeyEmpty) {
                kk = V->keys_bgf[rowbase + x];          // filtered by k_crack_bg (raw without the filter)
                bg_layer[i] = true;
            }
            if (okeys && in) okeys[rowbase + x] = kk;
            const bool present = kk != kKeyEmpty;
            some |= present;
            any_hole |= in && !present;
            const uint32_t m = __ballot_sync(0xffffffffu, present);
            if (lane == 0) s_mask[r * nch + ((xb + 32 * i) >> 5)] = m;
            w[i] = -1;
            ww[i] = 1.0f;
            cw[i] = 0u;
            Zs[i] = 1.0f;
            zmn[i] = __uint_as_float(0x7F800000u);       // a hole gathers nothing
            if (present) {
                Zs[i] = key_z(kk);
                zmn[i] = zmin;
                z_norm = z_norm && __float_as_uint(Zs[i]) - kZNormLoBits <= kZNormHiBits - kZNormLoBits;
                w[i] = int((kk >> kSrcBits) & 63u);
                const uint32_t s = uint32_t(kk & ((1u << kSrcBits) - 1u));
                const RWin& Q = s_win[w[i]];         // the winner is always active (only active cameras splat)
                const uint32_t sv = uint32_t((static_cast<unsigned long long>(s) * Q.magic) >> Q.shift);
                cw[i] = ld_frame<kCoh>(Q.rgba + sv * Q.rpitch + (s - sv * Q.W));
                ww[i] = Q.w;
            }
        }
        if (!__any_sync(0xffffffffu, some)) {                        // a block of holes
#pragma unroll
            for (int i = 0; i < P; ++i) {
                const int x = xb + 32 * i;
                if (x >= Wv) continue;
                s_rgb[r * RP + x] = kHoleBit;
                if (odepth) odepth[rowbase + x] = 0.0f;
                if (kTop3 && top3)
                    for (int q = 0; q < 3; ++q) top3[3 * (rowbase + x) + q] = 0.0f;
            }
            continue;
        }
        f32x2 x2[kPairs], Z2[kPairs];
#pragma unroll
        for (int p = 0; p < kPairs; ++p) {
            x2[p] = pk(u23_to_float(uint32_t(xb + 64 * p)), u23_to_float(uint32_t(xb + 64 * p + 32)));
            Z2[p] = pk(Zs[2 * p], Zs[2 * p + 1]);
        }
        // per-pixel weights: the surface points in the view's frame
        float px[P], py[P], lb[P];
        if (kPixW) {
            const float fy = u23_to_float(uint32_t(y));
#pragma unroll
            for (int i = 0; i < P; ++i) {
                px[i] = __fmul_rn(__fmul_rn(__fsub_rn(u23_to_float(uint32_t(xb + 32 * i)), V->vk[0]), V->vk[2]), Zs[i]);
                py[i] = __fmul_rn(__fmul_rn(__fsub_rn(fy, V->vk[1]), V->vk[3]), Zs[i]);
                lb[i] = __fsqrt_rn(__fadd_rn(__fadd_rn(__fmul_rn(px[i], px[i]), __fmul_rn(py[i], py[i])),
                                             __fmul_rn(Zs[i], Zs[i])));
                if (w[i] >= 0) {
                    const float4 c = s_ext[s_win[w[i]].pos].cen;
                    ww[i] = pixel_weight(c.x, c.y, c.z, px[i], py[i], Zs[i], lb[i]);
                }
            }
        }
        const f32x2 off = pk(-8388608.0f, -8388608.0f);
        auto channel = [&](uint32_t c0, uint32_t c1, int sel) {          // one colour byte of two texels, as floats
            return add2(pk(__uint_as_float(__byte_perm(c0, 0x4B000000u, 0x7440 + sel)),
                           __uint_as_float(__byte_perm(c1, 0x4B000000u, 0x7440 + sel))), off);
        };
        f32x2 accr[kPairs], accg[kPairs], accb[kPairs], wsum[kPairs];
        float t0[P], t1[P], t2[P];
        int k0[P], k1[P], k2[P];
        if (kTop3) {
#pragma unroll
            for (int i = 0; i < P; ++i) {
                t0[i] = ww[i];
                t1[i] = t2[i] = -1.0f;
                k0[i] = w[i];
                k1[i] = k2[i] = INT_MAX;
            }
        }
        auto seed = [&]() {
#pragma unroll
            for (int p = 0; p < kPairs; ++p) {
                wsum[p] = pk(ww[2 * p], ww[2 * p + 1]);
                accr[p] = mul2(wsum[p], channel(cw[2 * p], cw[2 * p + 1], 0), nz);
                accg[p] = mul2(wsum[p], channel(cw[2 * p], cw[2 * p + 1], 1), nz);
                accb[p] = mul2(wsum[p], channel(cw[2 * p], cw[2 * p + 1], 2), nz);
            }
        };
        auto project = [&](int a, int p, f32x2& X, f32x2& Y, f32x2& Zk) {
            const RCam& C = cams[a];
            const float4 rp = rowp[a];
            const f32x2 a0 = add2(add2(mul2(pk(C.n0, C.n0), x2[p], nz), pk(rp.x, rp.x)), pk(C.n2, C.n2));
            const f32x2 a1 = add2(add2(mul2(pk(C.n4, C.n4), x2[p], nz), pk(rp.y, rp.y)), pk(C.n6, C.n6));
            const f32x2 a2 = add2(add2(mul2(pk(C.n8, C.n8), x2[p], nz), pk(rp.z, rp.z)), pk(C.n10, C.n10));
            X = add2(mul2(a0, Z2[p], nz), pk(C.n3, C.n3));
            Y = add2(mul2(a1, Z2[p], nz), pk(C.n7, C.n7));
            Zk = add2(mul2(a2, Z2[p], nz), pk(C.n11, C.n11));
        };
        // cameras a0 .. a0 + N - 1 of the active list: project, settle the
        // targets, issue every gather, then accumulate in order.
        // Straight-line but for the rare redo loop, so the chains interleave.
        auto group = [&](auto size, int a0) {
            constexpr int N = decltype(size)::value;
            uint32_t tu[N][P], tv[N][P], dk[N][P], ck[N][P], di[N][P];
            f32x2 zk[N][kPairs];
            float nearest = z_norm ? 1.0f : 0.0f;
#pragma unroll
            for (int j = 0; j < N; ++j) {
#pragma unroll
                for (int p = 0; p < kPairs; ++p) {
                    f32x2 X, Y, u2, v2, nu2, nv2;
                    project(a0 + j, p, X, Y, zk[j][p]);
                    const float2 z = upk(zk[j][p]);
                    const f32x2 rz = pk(rcp_approx(z.x), rcp_approx(z.y));
                    round_quotient2(X, zk[j][p], rz, u2, nu2);
                    round_quotient2(Y, zk[j][p], rz, v2, nv2);
                    const float2 u = upk(u2), v = upk(v2), nu = upk(nu2), nv = upk(nv2);
                    tu[j][2 * p] = __float_as_uint(u.x) - kMagicBits;
                    tu[j][2 * p + 1] = __float_as_uint(u.y) - kMagicBits;
                    tv[j][2 * p] = __float_as_uint(v.x) - kMagicBits;
                    tv[j][2 * p + 1] = __float_as_uint(v.y) - kMagicBits;
                    nearest = min3_abs(min3_abs(nearest, nu.x, nv.x), nu.y, nv.y);
                }
            }
            if (!(nearest > eps)) {                  // one lane in 1000 (two cameras, four points, 1280 pixels)
#pragma unroll 1
                for (int a = 0; a < N; ++a) {
#pragma unroll 1
                    for (int p = 0; p < kPairs; ++p) {
                        // which points it was (the division is a hundred instructions)
                        f32x2 X, Y, Zk, u2, v2, nu2, nv2;
                        project(a0 + a, p, X, Y, Zk);
                        const float2 Xs = upk(X), Ys = upk(Y), Zq = upk(Zk);
                        const f32x2 rz = pk(rcp_approx(Zq.x), rcp_approx(Zq.y));
                        round_quotient2(X, Zk, rz, u2, nu2);
                        round_quotient2(Y, Zk, rz, v2, nv2);
                        const float2 nu = upk(nu2), nv = upk(nv2);
#pragma unroll 1
                        for (int h = 0; h < 2; ++h) {
                            const float n = h ? min3_abs(nu.y, nv.y, 1.0f) : min3_abs(nu.x, nv.x, 1.0f);
                            if (z_norm && n > eps) continue;
                            const uint2 t = target_pixel_div(h ? Xs.y : Xs.x, h ? Ys.y : Ys.x, h ? Zq.y : Zq.x);
#pragma unroll
                            for (int j = 0; j < N; ++j)
#pragma unroll
                                for (int i = 0; i < P; ++i)
                                    if (j == a && i == 2 * p + h) {
                                        tu[j][i] = t.x;
                                        tv[j][i] = t.y;
                                    }
                        }
                    }
                }
            }
#pragma unroll
            for (int j = 0; j < N; ++j) {
                const RCam& C = cams[a0 + j];
                const int4 dim = *reinterpret_cast<const int4*>(&C.dpitch);
#pragma unroll
                for (int i = 0; i < P; ++i) {
                    const float2 z = upk(zk[j][i >> 1]);
                    const bool ok = ((i & 1) ? z.y : z.x) > zmn[i] && C.k != w[i] && tu[j][i] <= uint32_t(dim.z) &&
                                    tv[j][i] <= uint32_t(dim.w);
                    di[j][i] = tv[j][i] * uint32_t(dim.x) + tu[j][i];
                    gather<kCoh>(ok, C.depth + di[j][i], C.rgba + tv[j][i] * uint32_t(dim.y) + tu[j][i], dk[j][i], ck[j][i]);
                }
            }
            // the BG layer's depth in camera k: its model where camera k
            // signals BG, none elsewhere (there camera k sees FG)
            if (kLayered) {
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    const uint16_t* bgk = s_ext[a0 + j].bg;
#pragma unroll
                    for (int i = 0; i < P; ++i)
                        if (bg_layer[i])
                            dk[j][i] = (dk[j][i] == kDepthBg && bgk) ? uint32_t(ld_frame<kCoh>(bgk + di[j][i])) : 0u;
                }
            }
            if (a0 == 0) seed();                     // the winners' colours, whose loads overlapped the group
#pragma unroll
            for (int j = 0; j < N; ++j) {
                const RCam& C = cams[a0 + j];
#pragma unroll
                for (int p = 0; p < kPairs; ++p) {
                    const float2 z = upk(zk[j][p]);
                    const float2 d = upk(add2(pk(__uint_as_float(0x4B000000u | dk[j][2 * p]),
                                                 __uint_as_float(0x4B000000u | dk[j][2 * p + 1])), off));
                    float wk[2];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int i = 2 * p + h;
                        // in [dlo, dhi] (0 -- no gather, no depth -- wraps above) and within tau_vis; a
                        // rejected camera adds +0 to each sum, which leaves it as it is
                        const float zh = h ? z.y : z.x;
                        const bool pass = dk[j][i] - dlo <= dspan &&
                                          fabsf(__fsub_rn(h ? d.y : d.x, zh)) <= __fmul_rn(tau_vis, zh);
                        if constexpr (kPixW) {
                            wk[h] = 0.0f;
                            if (pass) {
                                const float4 c = s_ext[a0 + j].cen;
                                wk[h] = pixel_weight(c.x, c.y, c.z, px[i], py[i], Zs[i], lb[i]);
                            }
                        } else {
                            wk[h] = pass ? C.w : 0.0f;
                        }
                        if (kTop3 && pass) {
                            const int k = C.k;
                            if (w_before(wk[h], k, t0[i], k0[i])) {
                                t2[i] = t1[i]; k2[i] = k1[i]; t1[i] = t0[i]; k1[i] = k0[i]; t0[i] = wk[h]; k0[i] = k;
                            } else if (w_before(wk[h], k, t1[i], k1[i])) {
                                t2[i] = t1[i]; k2[i] = k1[i]; t1[i] = wk[h]; k1[i] = k;
                            } else if (w_before(wk[h], k, t2[i], k2[i])) {
                                t2[i] = wk[h]; k2[i] = k;
                            }
                        }
                    }
                    const f32x2 w2 = pk(wk[0], wk[1]);
                    accr[p] = add2(accr[p], mul2(w2, channel(ck[j][2 * p], ck[j][2 * p + 1], 0), nz));
                    accg[p] = add2(accg[p], mul2(w2, channel(ck[j][2 * p], ck[j][2 * p + 1], 1), nz));
                    accb[p] = add2(accb[p], mul2(w2, channel(ck[j][2 * p], ck[j][2 * p + 1], 2), nz));
                    wsum[p] = add2(wsum[p], w2);
                }
            }
        };
        if (na > 1) {
            constexpr int kG = kWide ? kWideGroup - (kPixW ? 1 : 0) : kPixW && !kLayered ? 1 : kGroup;
            int a = 0;
            for (; na - a >= kG; a += kG) group(std::integral_constant<int, kG>{}, a);
            if constexpr (kG > 2)
                for (; na - a >= 2; a += 2) group(std::integral_constant<int, 2>{}, a);
            if (kG > 1 && a < na) group(std::integral_constant<int, 1>{}, a);
        }

#pragma unroll
        for (int p = 0; p < kPairs; ++p) {
            // the winner is the only camera: w c / w is within 2^-22 c of c, which it rounds to
            uint2 rgb2 = make_uint2(cw[2 * p] & 0xFFFFFFu, cw[2 * p + 1] & 0xFFFFFFu);
            float2 ws = make_float2(ww[2 * p], ww[2 * p + 1]);
            if (na > 1) {
                rgb2 = blend_rgb2(accr[p], accg[p], accb[p], wsum[p]);
                ws = upk(wsum[p]);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int i = 2 * p + h, x = xb + 32 * i;
                if (x >= Wv) continue;
                const bool present = w[i] >= 0;
                s_rgb[r * RP + x] = present ? (h ? rgb2.y : rgb2.x) : kHoleBit;
                if (keep) s_dep[r * Wv + x] = Zs[i];               // (read where present)
                if (odepth) odepth[rowbase + x] = present ? Zs[i] : 0.0f;
                if (kTop3 && top3) {
                    const float wh = h ? ws.y : ws.x;
                    top3[3 * (rowbase + x) + 0] = present ? __fdiv_rn(t0[i], wh) : 0.0f;
                    top3[3 * (rowbase + x) + 1] = present && t1[i] >= 0.0f ? __fdiv_rn(t1[i], wh) : 0.0f;
                    top3[3 * (rowbase + x) + 2] = present && t2[i] >= 0.0f ? __fdiv_rn(t2[i], wh) : 0.0f;
                }
            }
        }
    }

    // (e) hole fill: nearest non-hole left / right, the deeper one wins.  A
    // warp takes a 32-pixel chunk with holes: the nearest non-hole inside the
    // chunk is a bit search, beyond it a bit search over 32 chunks at a time
    // (a walk chunk by chunk took half of a view that is mostly holes).
    // Only holes are written and only non-holes are read.
    const bool band_has_hole = __syncthreads_or(any_hole) != 0;
    if (fill && band_has_hole) {
        for (int r = 0, c = wid;; c += NW) {
            while (r < rows && c >= nch) {
                c -= nch;
                ++r;
            }
            if (r >= rows) break;
            const int x = (c << 5) + lane;
            const uint32_t* mrow = s_mask + r * nch;
            const uint32_t m = mrow[c];
            const bool hole = x < Wv && !((m >> lane) & 1u);
            if (!__any_sync(0xffffffffu, hole)) continue;
            auto non_empty = [&](int g) {                                // chunks g .. g + 31 of the row, a bit each
                return __ballot_sync(0xffffffffu, g + lane < nch && mrow[g + lane] != 0u);
            };
            int gl = c & ~31, gr = gl;
            const uint32_t nz = non_empty(gl);
            uint32_t bl = nz & ((1u << (c & 31)) - 1u), br = nz & (0xFFFFFFFEu << (c & 31));
            while (!bl && gl > 0) bl = non_empty(gl -= 32);
            while (!br && gr + 32 < nch) br = non_empty(gr += 32);
            const int cl = gl + 31 - __clz(bl), cr = gr + __ffs(br) - 1; // (read where bl, br are not 0)
            const int left = bl ? (cl << 5) + 31 - __clz(mrow[cl]) : -1;
            const int right = br ? (cr << 5) + __ffs(mrow[cr]) - 1 : -1;
            const uint32_t below = (1u << lane) - 1u;
            const uint32_t ml = m & below, mr = m & ~below;              // (a hole's own bit is 0)
            const int l = ml ? (c << 5) + 31 - __clz(ml) : left;
            const int rt = mr ? (c << 5) + __ffs(mr) - 1 : right;
            if (hole && (l >= 0 || rt >= 0)) {
                uint32_t* c_rgb = s_rgb + r * RP;
                const size_t rowbase = size_t(y0 + r) * Wv;
                auto depth_at = [&](int xx) {
                    if (keep) return s_dep[r * Wv + xx];
                    const unsigned long long* up = s_keys + r * KP + 2;
                    unsigned long long kk = crack ? crack_rule_ptr(up + KP + xx, KP, f1) : up[KP + xx];
                    if (kLayered && kk == kKeyEmpty) kk = V->keys_bgf[rowbase + xx];
                    return key_z(kk);
                };
                const int src = l < 0 ? rt : (rt < 0 ? l : (depth_at(rt) > depth_at(l) ? rt : l));
                c_rgb[x] = c_rgb[src] | kHoleBit;
                if (odepth) odepth[rowbase + x] = depth_at(src);
            }
        }
        __syncthreads();
    }

    // RGB8 rows: four pixels -> three aligned 32-bit words where the row
    // allows it, single bytes for the rest
    for (int r = 0; r < rows; ++r) {
        const int y = y0 + r;
        const uint32_t* c_rgb = s_rgb + r * RP;
        uint8_t* orow = V->out_rgb + size_t(y) * size_t(V->out_pitch);
        int xdone = 0;
        if ((reinterpret_cast<uintptr_t>(orow) & 3u) == 0) {
            const int nq = Wv >> 2;
            uint32_t* o32 = reinterpret_cast<uint32_t*>(orow);
            for (int q = tid; q < nq; q += NT) {
                const uint4 p = reinterpret_cast<const uint4*>(c_rgb)[q];
                o32[3 * q + 0] = __byte_perm(p.x, p.y, 0x4210);
                o32[3 * q + 1] = __byte_perm(p.y, p.z, 0x5421);
                o32[3 * q + 2] = __byte_perm(p.z, p.w, 0x6542);
            }
            xdone = nq << 2;
        }
        for (int i = 3 * xdone + tid; i < 3 * Wv; i += NT) {
            const int x = i / 3;
            orow[i] = uint8_t(c_rgb[x] >> (8 * (i - 3 * x)));
        }
        const size_t rowbase = size_t(y) * Wv;
        if (!kCoh && V->out_hole)
            for (int x = tid; x < Wv; x += NT) V->out_hole[rowbase + x] = uint8_t((c_rgb[x] & kHoleBit) >> 24);
    }
}

template <bool kTop3, bool kLayered, bool kPixW>
__global__ void __launch_bounds__(kResolveThreads, kResolveOcc)
k_resolve(const ViewDesc* __restrict__ views, const FrameRef* __restrict__ frames, int band, int keep)
{
    extern __shared__ __align__(16) unsigned char smem[];
    resolve_cta<kTop3, kLayered, kPixW, false, kResolveThreads>(views, frames, band, keep != 0, int(blockIdx.x),
                                                                int(blockIdx.y), smem);
}

template <bool kLayered, bool kPixW>
__global__ void __maxnreg__(kWideRegs)
k_resolve_wide(const ViewDesc* __restrict__ views, const FrameRef* __restrict__ frames, int band, int keep)
{
    extern __shared__ __align__(16) unsigned char smem[];
    resolve_cta<false, kLayered, kPixW, false, kResolveThreads, true>(views, frames, band, keep != 0, int(blockIdx.x),
                                                                      int(blockIdx.y), smem);
}

// ---------------------------------------------------------------------------
// Persistent serving kernel.  One cooperative launch (every CTA resident)
// loops: CTA 0 waits for the next posted batch, then all CTAs run its clear,
// splat and resolve as virtual CTAs, with a grid barrier between the steps
// and a gpu-scope fence after each barrier (so weak loads see the other
// CTAs' writes and the frames uploaded before the batch was posted), and
// CTA 0 publishes the batch's completion.  It returns when no batch comes
// for idle_ns, on q->stop, or when a barrier runs out (sync->err, then
// q->err).
// ---------------------------------------------------------------------------
namespace {

__device__ __forceinline__ uint64_t gtimer()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Sense-counting grid barrier with a bounded wait (limit_ns); false once any
// CTA gave up.
__device__ bool persist_barrier(PersistSync* sync, unsigned int& gen, uint64_t limit_ns)
{
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned int g = gen;
        __threadfence();
        if (atomicAdd(&sync->count, 1u) == gridDim.x - 1) {
            atomicExch(&sync->count, 0u);
            __threadfence();
            atomicExch(&sync->gen, g + 1);
        } else {
            const uint64_t t0 = gtimer();
            while (*reinterpret_cast<volatile unsigned int*>(&sync->gen) == g) {
                if (*reinterpret_cast<volatile int*>(&sync->err) != 0) break;
                if (gtimer() - t0 > limit_ns) {
                    atomicCAS(&sync->err, 0, kPersistErrBarrier);
                    break;
                }
                __nanosleep(256);
            }
        }
        __threadfence();                      // acquire: later loads see the writes before the barrier
        gen = g + 1;
        s_ok = *reinterpret_cast<volatile int*>(&sync->err) == 0;
    }
    __syncthreads();
    return s_ok != 0;
}

}  // namespace

// What the persistent kernel leaves of an SM for kernels beside it, which would
// otherwise wait until it returns: registers for a resolve in its wide form (256
// threads of 96, two warps to each quarter of the SM; the depth filter takes 512
// of 32) and shared memory for the filter, which as it is static has at most 48 KB.
constexpr int kBesideRegs = kResolveThreads * kWideRegs;
constexpr size_t kSmShared = 228 * 1024, kCtaReserved = 1024;   // of an SM; what each CTA takes beside its own
constexpr size_t kBesideSmem = 48 * 1024 + kCtaReserved;

// Two CTAs an SM, three warps of each quarter.  What is left of the registers,
// 40,960, serves fewer threads without spills better than more with them: 16
// viewers of up to 1920x1080, saturated, on nine 1280x720 cameras, 12,950 views/s
// with 192 threads of 104 registers, 12,750 with 256 of 80, 11,500 with 160 of
// 120, 9,700 with one CTA of 384.  (224 of 88 serve 13,300, but put four warps on
// some quarters, beside which the wide form does not fit.  256 of 112 serve
// 15,300, but a filtered tick or a synthesis beside that waits until the kernel
// idles: with ticks filtered at 30 Hz and 478 views/s, p99 is 0.3 to 1.5 ms here
// and 19.4 there.)  The two kinds of weights are instances, as both in one kernel
// spill (12,650).
constexpr int kPersistThreads = 192;
template <bool kPixW>
__global__ void __maxnreg__(104)
k_serve_persistent(PersistQueue* q, PersistSync* sync, uint32_t first, uint64_t idle_ns, uint64_t wait_ns)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ PersistBatch s_b;
    __shared__ int s_cmd;
    unsigned int gen = 0;                     // the host zeroes *sync before the launch
    for (uint32_t b = first;; ++b) {
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            int cmd = 1;
            const uint64_t t0 = gtimer();
            for (;;) {
                if (q->stop) break;
                if (q->posted > b) {
                    cmd = 0;
                    break;
                }
                if (gtimer() - t0 > idle_ns) break;
                __nanosleep(1000);
            }
            sync->cmd = cmd;
        }
        if (!persist_barrier(sync, gen, wait_ns)) break;
        if (threadIdx.x == 0) {
            s_cmd = *reinterpret_cast<volatile int*>(&sync->cmd);
            if (!s_cmd) {
                // field by field through volatile reads: the host wrote it
                const volatile PersistBatch& src = q->batch[b % kPersistRing];
                s_b.views = src.views;
                s_b.frames = src.frames;
                s_b.keys = src.keys;
                s_b.n_keys = src.n_keys;
                s_b.n_views = src.n_views;
                s_b.max_h = src.max_h;
                s_b.band = src.band;
                s_b.splat_bx = src.splat_bx;
                s_b.keep = src.keep;
            }
        }
        __syncthreads();
        if (s_cmd) break;
        const PersistBatch B = s_b;
        // (a0) the batch's z-buffers
        const size_t stride = size_t(gridDim.x) * blockDim.x;
        for (size_t i = size_t(blockIdx.x) * blockDim.x + threadIdx.x; i < B.n_keys; i += stride)
            B.keys[i] = kKeyEmpty;
        if (!persist_barrier(sync, gen, wait_ns)) break;
        // (a) + (b)
        for (int v = int(blockIdx.x); v < B.splat_bx * B.n_views; v += int(gridDim.x))
            splat_cta<false, false, true, kPersistThreads>(B.views, B.frames, v % B.splat_bx, v / B.splat_bx, B.splat_bx);
        if (!persist_barrier(sync, gen, wait_ns)) break;
        // (c) + (d) + (e)
        const int nb = (B.max_h + B.band - 1) / B.band;
        for (int v = int(blockIdx.x); v < nb * B.n_views; v += int(gridDim.x))
            resolve_cta<false, false, kPixW, true, kPersistThreads>(B.views, B.frames, B.band, B.keep != 0, v % nb, v / nb, smem);
        if (!persist_barrier(sync, gen, wait_ns)) break;
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            __threadfence_system();           // the batch's outputs before its completion
            q->done = b + 1;
            __threadfence_system();
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        q->err = *reinterpret_cast<volatile int*>(&sync->err);
        __threadfence_system();
    }
}

// ---------------------------------------------------------------------------
// upload: RGB8 rows -> RGBA8 rows (R | G << 8 | B << 16)
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_pack_rgba(const uint8_t* __restrict__ rgb, size_t pitch,
                                                   uint32_t* __restrict__ rgba, int rpitch, int W)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= W)
        return;
    const uint8_t* p = rgb + size_t(y) * pitch + 3 * size_t(x);
    rgba[size_t(y) * rpitch + x] = uint32_t(p[0]) | (uint32_t(p[1]) << 8) | (uint32_t(p[2]) << 16);
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
int device_sms()
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) {
        cudaGetLastError();
        sms = 1;
    }
    return sms;
}

namespace {

// Splat depth loads: 16-byte vectors (8 pixels per lane) or 2-byte loads at
// a stride of 32 pixels.  FVV_SPLAT_VEC=0/1 picks one for measurements.
bool splat_vec()
{
    static const int v = [] {
        const char* e = std::getenv("FVV_SPLAT_VEC");
        return e ? (e[0] == '1' ? 1 : 0) : 0;
    }();
    return v != 0;
}

}  // namespace

// The widest view a context admits: 41 bytes of shared memory per pixel and
// the cameras' records.  (A single-row band of the resolve takes 32 bytes per
// pixel, so every admitted view fits.)
size_t resolve_smem_bytes(int max_w, int n_cams, bool layered)
{
    (void)layered;
    size_t o = align16(4 * (size_t(max_w) + 2) * 8) + 2 * align16(size_t(max_w) * 4) + align16(size_t(max_w));
    return o + size_t(n_cams) * 144 + kMaxCams * sizeof(int) + 64 * sizeof(int);
}

namespace {

// See kKeepPoints.
bool keep_depths(size_t points, int max_w, int max_h, int n_views)
{
    return double(points) < kKeepPoints * double(max_w) * double(max_h) * n_views;
}

// Output rows per resolve CTA, 1..kResolveMaxBand, within smem_cap bytes.  A
// warp takes kBlock pixels at a time, so a band's blocks should fill the eight
// warps evenly (one row of 1280 pixels is 20 blocks, three rounds of which the
// last is half empty; two rows are five full rounds); and the bands should
// spread evenly over the SMs, which matters for one small view (a few bands per
// SM) and not for a batch.  Estimated rows of work on the busiest SM, plus the
// start-up of each of its CTAs as kBandStart rows (717x491, eight views of 13
// cameras: 134 us with the two rows that 0.25 gives, 141 with the four of 0.35).
// resident: CTAs that an SM runs at once; fewer than that take as long, since a
// lone CTA waits for its gathers (949x490 from ten 1859x1434 cameras: 131 us
// with single rows, 208 with the four that the work alone would suggest).
int resolve_band(int w, int h, int n_views, int n_cams, bool keep, int threads, int sms, int resident, size_t smem_cap)
{
    int best = 1;
    double cost = 0.0;
    for (int b = 1; b <= kResolveMaxBand; ++b) {
        if (b > 1 && resolve_layout(w, n_cams, b, keep).total > smem_cap) break;
        const int NW = threads / 32;
        const int blocks = b * ((w + kBlock - 1) / kBlock), rounds = (blocks + NW - 1) / NW;
        const double per_row = double(rounds) * NW / blocks;          // 1 when the warps fill evenly
        const long long ctas = (long long)((h + b - 1) / b) * n_views;
        const double c = double(std::max<long long>((ctas + sms - 1) / sms, resident)) * (b * per_row + kBandStart);
        if (b == 1 || c < cost) {
            best = b;
            cost = c;
        }
    }
    return best;
}

}  // namespace

cudaError_t launch_clear_keys(unsigned long long* keys, size_t n, cudaStream_t stream)
{
    if (n == 0) return cudaSuccess;
    size_t blocks = ((n >> 1) + 255) / 256;
    const size_t cap = size_t(device_sms()) * 16;
    if (blocks < 1) blocks = 1;
    if (blocks > cap) blocks = cap;
    k_clear_keys<<<unsigned(blocks), 256, 0, stream>>>(keys, n);
    return cudaGetLastError();
}

cudaError_t launch_warp_splat(const ViewDesc* views, int n_views, int max_chunks,
                              const FrameRef* frames, cudaStream_t stream, bool layered)
{
    if (n_views <= 0 || max_chunks <= 0) return cudaSuccess;
    constexpr int kWarps = kSplatThreads / 32;      // one warp per segment at a time
    // persistent warps: about two resident waves over all views of the batch
    const int sms = device_sms();
    const int want = (2 * kSplatOcc * sms + n_views - 1) / n_views;
    const int need = (max_chunks + kWarps - 1) / kWarps;
    const int bx = need < want ? need : (want < 1 ? 1 : want);
    dim3 grid(static_cast<unsigned>(bx), static_cast<unsigned>(n_views));
    const bool vec = splat_vec();
    if (layered) {
        if (vec) k_warp_splat<true, true><<<grid, kSplatThreads, 0, stream>>>(views, frames);
        else k_warp_splat<true, false><<<grid, kSplatThreads, 0, stream>>>(views, frames);
    } else {
        if (vec) k_warp_splat<false, true><<<grid, kSplatThreads, 0, stream>>>(views, frames);
        else k_warp_splat<false, false><<<grid, kSplatThreads, 0, stream>>>(views, frames);
    }
    return cudaGetLastError();
}

cudaError_t launch_crack_bg(const ViewDesc* views, int n_views, int max_h, int max_w, cudaStream_t stream)
{
    if (n_views <= 0 || max_h <= 0 || max_w <= 0) return cudaSuccess;
    dim3 grid(static_cast<unsigned>((max_w + kBgW - 1) / kBgW), static_cast<unsigned>((max_h + kBgH - 1) / kBgH),
              static_cast<unsigned>(n_views));
    return launch_behind(k_crack_bg, grid, dim3(kBgW, kBgH), 0, stream, views);
}

cudaError_t launch_resolve(const ViewDesc* views, int n_views, int max_h, int max_w, int n_cams, size_t points,
                           bool top3, const FrameRef* frames, cudaStream_t stream, bool layered,
                           bool pixel_weights)
{
    if (n_views <= 0 || max_h <= 0) return cudaSuccess;
    // the layout grows with the width and the camera count, so the widest
    // view of the batch bounds every CTA's shared memory.  Launched view after
    // view: the CTAs resident at one time cover about one view, whose frames
    // stay in L2 for its gathers.
    const bool keep = keep_depths(points, max_w, max_h, n_views);
    const int band = resolve_band(max_w, max_h, n_views, n_cams, keep, kResolveThreads, device_sms(), kResolveOcc,
                                  keep ? kResolveSmemKept : kResolveSmem);
    const size_t smem = resolve_layout(max_w, n_cams, band, keep).total;
    auto go = [&](auto kernel) {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
        if (e != cudaSuccess) return e;
        dim3 grid(static_cast<unsigned>((max_h + band - 1) / band), static_cast<unsigned>(n_views));
        return launch_behind(kernel, grid, kResolveThreads, smem, stream, views, frames, band, keep ? 1 : 0);
    };
    const bool wide = !top3 && (long long)((max_h + band - 1) / band) * n_views <= (long long)kWideCtas * device_sms();
    if (wide) {
        if (pixel_weights) return layered ? go(k_resolve_wide<true, true>) : go(k_resolve_wide<false, true>);
        return layered ? go(k_resolve_wide<true, false>) : go(k_resolve_wide<false, false>);
    }
    if (pixel_weights) {
        if (layered) return top3 ? go(k_resolve<true, true, true>) : go(k_resolve<false, true, true>);
        return top3 ? go(k_resolve<true, false, true>) : go(k_resolve<false, false, true>);
    }
    if (layered) return top3 ? go(k_resolve<true, true, false>) : go(k_resolve<false, true, false>);
    return top3 ? go(k_resolve<true, false, false>) : go(k_resolve<false, false, false>);
}

// The persistent kernel's shared memory: two-row bands of the widest view where
// two CTAs of that leave kBesideSmem (with kept depths up to 1688 pixels, without
// up to 2024, nine cameras), else single rows.
namespace {
constexpr size_t kPersistStatic = 7424;                         // at least the kernel's static shared memory

size_t persist_smem(int max_w, int n_cams)
{
    constexpr size_t cap = (kSmShared - kBesideSmem) / 2 - kCtaReserved - kPersistStatic;
    for (const bool keep : {true, false}) {
        const size_t two = resolve_layout(max_w, n_cams, 2, keep).total;
        if (two <= cap) return two;
    }
    return resolve_layout(max_w, n_cams, 1, true).total;
}

auto persist_kernel(bool pixel_weights)
{
    return pixel_weights ? k_serve_persistent<true> : k_serve_persistent<false>;
}
}  // namespace

void persist_batch_shape(int n_views, int max_h, int max_w, int n_cams, size_t points, int kernel_max_w,
                         int max_chunks, int ctas, PersistBatch* batch)
{
    // bands within the shared memory that the running kernel was launched
    // with; the splat's segments spread over about one virtual CTA per real one
    const bool keep = keep_depths(points, max_w, max_h, n_views);
    batch->keep = keep ? 1 : 0;
    batch->band = resolve_band(max_w, max_h, n_views, n_cams, keep, kPersistThreads, ctas, 1, persist_smem(kernel_max_w, n_cams));
    constexpr int kWarps = kPersistThreads / 32;
    const int need = (max_chunks + kWarps - 1) / kWarps;
    const int want = (ctas + n_views - 1) / n_views;
    batch->splat_bx = std::max(1, std::min(need, want));
}

int persist_grid(int max_w, int n_cams, bool pixel_weights)
{
    const auto kernel = persist_kernel(pixel_weights);
    const size_t smem = persist_smem(max_w, n_cams);
    // An SM's split between L1 and shared memory changes only while it is idle,
    // so what kernels beside this one need has to be shared memory when it starts.
    cudaFuncAttributes fa{};
    int per_sm = 0;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) !=
            cudaSuccess ||
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kPersistThreads, smem) != cudaSuccess ||
        cudaFuncGetAttributes(&fa, kernel) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    auto leaves_room = [&](int n) {
        // registers belong to the quarters of an SM, and a CTA's warps to one each in turn
        const int warps = n * kPersistThreads / 32, quarter = (warps + 3) / 4 * 32 * fa.numRegs;
        return quarter + kBesideRegs / 4 <= 65536 / 4 &&
               size_t(n) * (smem + fa.sharedSizeBytes + kCtaReserved) + kBesideSmem <= kSmShared;
    };
    while (per_sm > 1 && !leaves_room(per_sm)) --per_sm;
    return per_sm * device_sms();
}

cudaError_t launch_serve_persistent(PersistQueue* q_dev, PersistSync* sync, uint32_t first, int max_w, int n_cams,
                                    bool pixel_weights, uint64_t idle_ns, uint64_t wait_ns, cudaStream_t stream,
                                    int* ctas)
{
    const size_t smem = persist_smem(max_w, n_cams);
    const int grid = persist_grid(max_w, n_cams, pixel_weights);
    if (grid < 1) return cudaErrorInvalidValue;
    *ctas = grid;
    void* args[] = {&q_dev, &sync, &first, &idle_ns, &wait_ns};
    return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(persist_kernel(pixel_weights)), dim3(unsigned(grid)),
                                       dim3(kPersistThreads), args, smem, stream);
}

cudaError_t launch_pack_rgba(const uint8_t* rgb, size_t rgb_pitch, uint32_t* rgba, int rpitch,
                             int W, int H, cudaStream_t stream)
{
    if (W <= 0 || H <= 0) return cudaSuccess;
    dim3 grid(static_cast<unsigned>((W + 255) / 256), static_cast<unsigned>(H));
    k_pack_rgba<<<grid, 256, 0, stream>>>(rgb, rgb_pitch, rgba, rpitch, W);
    return cudaGetLastError();
}

}  // namespace fvv
