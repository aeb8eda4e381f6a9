// fvv_jbf.cu -- joint bilateral depth pre-filter (Sec. VI: a colour-guided
// joint bilateral filter fills small gaps in the live depth, in particular
// along object boundaries).
//
// A pixel without depth (code 0) takes the weighted mean of the valid codes
// in its (2r+1) x (2r+1) window; every other pixel keeps its code.  The
// weight of neighbour q is s[dy][dx] * c[|dR|] * c[|dG|] * c[|dB|] with
// s = exp(-(dx^2 + dy^2) / (2 sigma_s^2)) and c[t] = exp(-t^2 / (2
// sigma_c^2)), both evaluated on the host in FP64 and rounded to FP32 once.
// Neighbours are visited in row-major window order and every FP32 operation
// is an explicit round-to-nearest intrinsic, so the result is exactly that
// of the stated operation sequence.  The code is floor(acc / wsum + 0.5)
// clamped to [d_lo, d_hi], written only when at least min_valid neighbours
// are valid codes; the background signal is neither a source nor filled.
// One pass, out of place.
//
// The filter reads 2 + 3 bytes and writes 2 bytes per pixel, but is bound by
// instruction issue in the windows of the pixels without depth (see k_jbf).
#include <cmath>
#include <cstring>
#include <type_traits>

#include "fvv_jbf.h"
#include "fvv_runtime.h"

namespace fvv {

namespace {

__device__ __forceinline__ float code_to_float(uint32_t d)   // exact for d < 2^23
{
    return __fsub_rn(__uint_as_float(0x4B000000u | d), 8388608.0f);
}

// A CTA filters a kTileW x kTileH tile of camera blockIdx.z.  Phase 1
// stages the tile and its halo (codes and colour bytes) in shared memory: 16
// bytes a lane when the rows are 16-byte aligned, else element by element,
// neighbouring lanes on neighbouring elements.  Phase 2 writes the tile's codes
// back out and lists the pixels without one; a tile without any is done.  Phase
// 2b turns each staged pixel into what a window visits: the code as FP32 (-1
// when it is no source) and the colour with its channels in ten-bit fields,
// one 8-byte load per neighbour.  Phase 3 deals the listed
// pixels out to the threads, so a tile's few holes are filtered by many threads
// at once instead of idling the rest of their warps; each filtered pixel walks
// its window in shared memory in the stated order (the radius is a template
// parameter, so the window unrolls) and overwrites its output.
//
// Latency sets the time: of the staging's loads, which a thread therefore has
// all in flight together, and of phase 3, 49 neighbours in order for each of
// some 46,000 pixels of a 1280x720 frame.  The three channel differences come
// from one subtraction of biased fields, each in [1, 511], and index a table of
// c[|d|] by the signed difference, so a neighbour costs about 17 instructions
// (with byte-wise absolute differences and separate loads of code, colour and
// spatial weight it cost over 40), and one that is no source adds zeros, so
// that no branch keeps the next ones' loads back.  Nine 1280x720 frames of
// radius 3 took 101 us before; 84 us with the cheaper neighbours, 76 us with
// wider tiles, which stage less halo per pixel, 65 us without the branch and
// 61 us with the staging's loads in flight.  Three CTAs per SM (40 registers)
// take 67 us.  Tiles are 128 x 16 pixels for 512 threads up to radius 3 (47 KB
// of shared memory, four CTAs per SM of 32 registers a thread, which spills 52 to
// 56 bytes); above that the arrays would pass the 48 KB of static
// shared memory, and a tile is 64 x 16 (nothing spilled).
constexpr int kTileH = 16;
constexpr int kDM = 8, kCM = 32;          // left margins of the staged rows: pixels, colour bytes
template <int R>
struct Tile {
    static constexpr int kW = R <= 3 ? 128 : 64, kThreads = 4 * kW;
};
static_assert(kJbfMaxRadius <= kDM && 3 * kJbfMaxRadius <= kCM, "halo wider than the margins");

template <int R>
__global__ void __launch_bounds__(Tile<R>::kThreads, 2048 / Tile<R>::kThreads) k_jbf(const __grid_constant__ JbfParams P)
{
    constexpr int kTileW = Tile<R>::kW, kThreads = Tile<R>::kThreads;
    constexpr int kDW = kDM + kTileW + kDM;        // staged code row, pixels
    constexpr int kCW = kCM + 3 * kTileW + kCM;    // staged colour row, bytes
    constexpr int side = 2 * R + 1;
    constexpr int hh = kTileH + 2 * R;
    __shared__ __align__(16) uint16_t s_d[hh][kDW];
    __shared__ __align__(16) uint8_t s_c[hh][kCW];
    // per staged pixel: the code as FP32 bits (-1 when it is no source) and
    // the colour R | G << 10 | B << 20, for the window walks of phase 3 (rows
    // padded so that neighbouring rows fall in other banks)
    __shared__ __align__(16) uint2 s_px[hh][kDW + 2];
    __shared__ uint16_t s_list[kTileW * kTileH];
    __shared__ float s_wc[512];                    // [256 + d]: c[|d|]
    __shared__ int s_n;
    const JbfCam& C = P.cam[blockIdx.z];
    const int x0 = blockIdx.x * kTileW, y0 = blockIdx.y * kTileH;
    const int W = P.width;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool vec = C.vec != 0;
    if (tid == 0) s_n = 0;
    // the colour weights in shared memory: the filtered pixels of a warp index
    // them at different places, which parameter (constant) memory would
    // serialise (the spatial weights' places are compile-time constants)
    for (int i = tid; i < 512; i += kThreads) s_wc[i] = i > 0 ? P.c[i < 256 ? 256 - i : i - 256] : 0.0f;
    // phase 1: outside the image a code of 0 (never a source) and colour 0.
    // With aligned rows a row with its margins is kD16 + kC16 16-byte pieces,
    // dealt out over the threads; without, a warp takes a row.
    constexpr int kD16 = kDW / 8, kC16 = kCW / 16;
    if (vec) {
        constexpr int kPieces = hh * (kD16 + kC16), kEach = (kPieces + kThreads - 1) / kThreads;
        uint4 v[kEach];
#pragma unroll
        for (int e = 0; e < kEach; ++e) {                          // all of a thread's loads in flight together
            const int i = tid + e * kThreads;
            const int hy = i / (kD16 + kC16), q = i - hy * (kD16 + kC16), gy = y0 - R + hy;
            const bool code = q < kD16;
            // the piece's first byte in the image row, and the row's length
            const int t = code ? q : q - kD16;
            const int b = code ? 2 * (x0 - kDM) + 16 * t : 3 * x0 - kCM + 16 * t, len = code ? 2 * W : 3 * W;
            v[e] = make_uint4(0u, 0u, 0u, 0u);
            if (i >= kPieces || gy < 0 || gy >= P.height || b < 0 || b >= len) continue;
            const uint8_t* row = code ? reinterpret_cast<const uint8_t*>(C.src + size_t(gy) * C.src_pitch)
                                      : C.rgb + size_t(gy) * C.rgb_pitch;
            if (b + 16 <= len) {
                v[e] = __ldg(reinterpret_cast<const uint4*>(row + b));
            } else {                                               // the ragged end
                uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                for (int c = 0; c < 16; ++c)
                    if (b + c < len) w[c >> 2] |= uint32_t(__ldg(row + b + c)) << (8 * (c & 3));
                v[e] = make_uint4(w[0], w[1], w[2], w[3]);
            }
        }
#pragma unroll
        for (int e = 0; e < kEach; ++e) {
            const int i = tid + e * kThreads;
            if (i >= kPieces) break;
            const int hy = i / (kD16 + kC16), q = i - hy * (kD16 + kC16);
            uint8_t* dst = q < kD16 ? reinterpret_cast<uint8_t*>(&s_d[hy][0]) + 16 * q : &s_c[hy][0] + 16 * (q - kD16);
            *reinterpret_cast<uint4*>(dst) = v[e];
        }
    } else {
        for (int hy = warp; hy < hh; hy += kThreads / 32) {
            const int gy = y0 - R + hy;
            const bool row_in = gy >= 0 && gy < P.height;
            const uint16_t* drow = C.src + size_t(row_in ? gy : 0) * C.src_pitch;
            const uint8_t* crow = C.rgb + size_t(row_in ? gy : 0) * C.rgb_pitch;
#pragma unroll
            for (int t0 = 0; t0 < kTileW + 2 * R; t0 += 32) {
                const int t = t0 + lane, x = x0 - R + t;
                if (t < kTileW + 2 * R)
                    s_d[hy][kDM - R + t] = (row_in && x >= 0 && x < W) ? __ldg(drow + x) : uint16_t(0);
            }
#pragma unroll
            for (int t0 = 0; t0 < 3 * (kTileW + 2 * R); t0 += 32) {
                const int t = t0 + lane, b = 3 * (x0 - R) + t;
                if (t < 3 * (kTileW + 2 * R))
                    s_c[hy][kCM - 3 * R + t] = (row_in && b >= 0 && b < 3 * W) ? __ldg(crow + b) : uint8_t(0);
            }
        }
    }
    __syncthreads();
    // phase 2: the tile's codes go out (pixels without one as 0 for now), 8
    // at a time or neighbouring lanes side by side, and those pixels are listed
    constexpr int kC8 = kTileW / 8;
    if (vec) {
        for (int i = tid; i < kTileH * kC8; i += kThreads) {
            const int ty = i / kC8, c8 = i - ty * kC8;
            const int y = y0 + ty, x = x0 + 8 * c8;
            if (y < P.height && x < W) {
                const uint4 v = *reinterpret_cast<const uint4*>(&s_d[ty + R][kDM + 8 * c8]);
                const uint32_t w[4] = {v.x, v.y, v.z, v.w};
                uint16_t* orow = C.dst + size_t(y) * C.dst_pitch;
                const int ne = min(8, W - x);
                if (ne == 8)
                    *reinterpret_cast<uint4*>(orow + x) = v;
                for (int e = 0; e < ne; ++e) {
                    const uint16_t d = uint16_t(w[e >> 1] >> (16 * (e & 1)));
                    if (ne != 8) orow[x + e] = d;
                    if (d == 0) s_list[atomicAdd(&s_n, 1)] = uint16_t(ty * kTileW + 8 * c8 + e);
                }
            }
        }
    } else {
        for (int i = tid; i < kTileH * kTileW; i += kThreads) {
            const int ty = i / kTileW, tx = i - ty * kTileW;
            const int y = y0 + ty, x = x0 + tx;
            if (y < P.height && x < W) {
                const uint16_t d = s_d[ty + R][kDM + tx];
                C.dst[size_t(y) * C.dst_pitch + x] = d;
                if (d == 0) s_list[atomicAdd(&s_n, 1)] = uint16_t(i);
            }
        }
    }
    __syncthreads();
    const int n_holes = s_n;
    if (n_holes == 0) return;                      // uniform over the CTA
    // phase 2b: four staged pixels a thread (the columns a window reaches,
    // rounded out to quads; the rounding's columns are never visited)
    constexpr int kLeft = (R + 3) / 4 * 4, kQuads = (kTileW + 2 * kLeft) / 4;
    for (int i = tid; i < hh * kQuads; i += kThreads) {
        const int hy = i / kQuads, q = i - hy * kQuads, col = kDM - kLeft + 4 * q;
        const uint2 dd = *reinterpret_cast<const uint2*>(&s_d[hy][col]);
        const uint32_t* c = reinterpret_cast<const uint32_t*>(&s_c[hy][kCM + 3 * (col - kDM)]);
        const uint32_t c0 = c[0], c1 = c[1], c2 = c[2];
        const uint32_t code[4] = {dd.x & 0xFFFFu, dd.x >> 16, dd.y & 0xFFFFu, dd.y >> 16};
        const uint32_t rgb[4] = {c0, __byte_perm(c0, c1, 0x0543), __byte_perm(c1, c2, 0x0432), c2 >> 8};
        uint32_t o[8];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const bool src = code[e] >= P.d_lo && code[e] <= P.d_hi && code[e] != kDepthBg;
            o[2 * e] = __float_as_uint(src ? code_to_float(code[e]) : -1.0f);
            o[2 * e + 1] = (rgb[e] & 0xFFu) | ((rgb[e] & 0xFF00u) << 2) | ((rgb[e] & 0xFF0000u) << 4);
        }
        uint4* dst = reinterpret_cast<uint4*>(&s_px[hy][col]);
        dst[0] = make_uint4(o[0], o[1], o[2], o[3]);
        dst[1] = make_uint4(o[4], o[5], o[6], o[7]);
    }
    __syncthreads();
    // phase 3: one listed pixel per thread at a time
    for (int j = tid; j < n_holes; j += kThreads) {
        const int i = s_list[j];
        const int ty = i / kTileW, tx = i - ty * kTileW;
        const int cy = ty + R, cx = kDM + tx;                      // centre in the staged tile
        const uint2* px = &s_px[cy][cx];
        const uint32_t c0 = px->y + (256u | (256u << 10) | (256u << 20));
        float acc = 0.0f, wsum = 0.0f;
        int n = 0;
#pragma unroll
        for (int dy = -R; dy <= R; ++dy) {
#pragma unroll
            for (int dx = -R; dx <= R; ++dx) {
                const uint2 q = px[dy * (kDW + 2) + dx];
                const float qf = __uint_as_float(q.x);
                const uint32_t df = c0 - q.y;                      // fields 256 + dR, 256 + dG, 256 + dB
                float w = __fmul_rn(__fmul_rn(__fmul_rn(P.s[(dy + R) * side + (dx + R)], s_wc[df & 1023u]),
                                              s_wc[(df >> 10) & 1023u]),
                                    s_wc[df >> 20]);
                w = qf < 0.0f ? 0.0f : w;                          // no source: a zero more in each sum
                acc = __fadd_rn(acc, __fmul_rn(w, qf));
                wsum = __fadd_rn(wsum, w);
                n += qf < 0.0f ? 0 : 1;
            }
        }
        uint32_t out = 0u;
        if (n >= P.min_valid && wsum > 0.0f) {
            float v = floorf(__fadd_rn(__fdiv_rn(acc, wsum), 0.5f));
            v = fminf(fmaxf(v, float(P.d_lo)), float(P.d_hi));
            out = uint32_t(v);
        }
        if (out != 0u)
            C.dst[size_t(y0 + ty) * C.dst_pitch + (x0 + tx)] = uint16_t(out);
    }
}

}  // namespace

bool jbf_options_ok(const fvv_options& o, std::string* why)
{
    if (o.jbf_radius < 0 || o.jbf_radius > kJbfMaxRadius) {
        *why = "jbf_radius must be in [0, 7]";
        return false;
    }
    if (o.jbf_radius == 0) return true;
    if (!(o.jbf_sigma_s > 0.0f) || !std::isfinite(o.jbf_sigma_s) || !(o.jbf_sigma_c > 0.0f) ||
        !std::isfinite(o.jbf_sigma_c)) {
        *why = "jbf_sigma_s and jbf_sigma_c must be finite and > 0";
        return false;
    }
    const int side = 2 * o.jbf_radius + 1;
    if (o.jbf_min_valid < 1 || o.jbf_min_valid >= side * side) {
        *why = "jbf_min_valid must be in [1, (2 jbf_radius + 1)^2 - 1]";
        return false;
    }
    return true;
}

void jbf_params(const fvv_options& o, int width, int height, JbfParams* P)
{
    std::memset(P, 0, sizeof *P);
    P->width = width;
    P->height = height;
    P->radius = o.jbf_radius;
    P->min_valid = o.jbf_min_valid;
    P->d_lo = o.d_lo;
    P->d_hi = o.d_hi;
    const int R = o.jbf_radius, side = 2 * R + 1;
    const double ss = double(o.jbf_sigma_s), sc = double(o.jbf_sigma_c);
    for (int dy = -R; dy <= R; ++dy)
        for (int dx = -R; dx <= R; ++dx)
            P->s[(dy + R) * side + (dx + R)] = float(std::exp(-double(dx * dx + dy * dy) / (2.0 * ss * ss)));
    for (int t = 0; t < 256; ++t) P->c[t] = float(std::exp(-double(t * t) / (2.0 * sc * sc)));
}

cudaError_t launch_jbf(const JbfParams& P_in, int n_cams, cudaStream_t stream)
{
    if (n_cams <= 0 || P_in.width <= 0 || P_in.height <= 0) return cudaSuccess;
    if (n_cams > kJbfMaxCams) return cudaErrorInvalidValue;
    // 16-byte accesses where every row of a camera starts 16-byte aligned
    // (a tile's first column sits whole 128-byte steps of codes and 192-byte
    // steps of colour on)
    JbfParams P = P_in;
    auto a16 = [](const void* p, int64_t pitch_bytes) {
        return (reinterpret_cast<uintptr_t>(p) & 15u) == 0 && pitch_bytes % 16 == 0;
    };
    for (int k = 0; k < n_cams; ++k) {
        JbfCam& c = P.cam[k];
        c.vec = a16(c.rgb, c.rgb_pitch) && a16(c.src, c.src_pitch * 2) && a16(c.dst, c.dst_pitch * 2) ? 1 : 0;
    }
    auto go = [&](auto radius) {
        constexpr int R = decltype(radius)::value;
        dim3 grid(unsigned((P.width + Tile<R>::kW - 1) / Tile<R>::kW), unsigned((P.height + kTileH - 1) / kTileH),
                  unsigned(n_cams));
        k_jbf<R><<<grid, Tile<R>::kThreads, 0, stream>>>(P);
    };
    switch (P.radius) {
    case 1: go(std::integral_constant<int, 1>{}); break;
    case 2: go(std::integral_constant<int, 2>{}); break;
    case 3: go(std::integral_constant<int, 3>{}); break;
    case 4: go(std::integral_constant<int, 4>{}); break;
    case 5: go(std::integral_constant<int, 5>{}); break;
    case 6: go(std::integral_constant<int, 6>{}); break;
    case 7: go(std::integral_constant<int, 7>{}); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace fvv

using fvv::fail;

extern "C" fvv_status fvv_depth_jbf(const uint8_t* rgb, size_t rgb_pitch, const uint16_t* depth, size_t depth_pitch,
                                    uint16_t* out, size_t out_pitch, int32_t width, int32_t height,
                                    const fvv_options* opt, void* stream)
{
    if (!rgb || !depth || !out || !opt) return fail(FVV_ERR_INVALID_ARG, "fvv_depth_jbf: NULL argument");
    if (width < 1 || height < 1) return fail(FVV_ERR_INVALID_ARG, "fvv_depth_jbf: width and height must be >= 1");
    std::string why;
    if (!fvv::jbf_options_ok(*opt, &why)) return fail(FVV_ERR_INVALID_ARG, "fvv_depth_jbf: " + why);
    if (opt->jbf_radius == 0) return fail(FVV_ERR_INVALID_ARG, "fvv_depth_jbf: jbf_radius is 0 (filter off)");
    if (opt->d_lo < 1 || opt->d_hi > 65534 || opt->d_lo > opt->d_hi)
        return fail(FVV_ERR_INVALID_ARG, "fvv_depth_jbf: need 1 <= d_lo <= d_hi <= 65534");
    if (rgb_pitch < size_t(width) * 3 || depth_pitch < size_t(width) * 2 || depth_pitch % 2 ||
        out_pitch < size_t(width) * 2 || out_pitch % 2 || (reinterpret_cast<uintptr_t>(depth) & 1) ||
        (reinterpret_cast<uintptr_t>(out) & 1))
        return fail(FVV_ERR_INVALID_ARG, "fvv_depth_jbf: bad pitch or alignment");
    const size_t ib = depth_pitch * size_t(height - 1) + size_t(width) * 2;
    const size_t ob = out_pitch * size_t(height - 1) + size_t(width) * 2;
    const uintptr_t i0 = reinterpret_cast<uintptr_t>(depth), o0 = reinterpret_cast<uintptr_t>(out);
    if (i0 < o0 + ob && o0 < i0 + ib)
        return fail(FVV_ERR_INVALID_ARG, "fvv_depth_jbf: out must not overlap depth (the filter is out of place)");
    for (const void* p : {static_cast<const void*>(rgb), static_cast<const void*>(depth),
                          static_cast<const void*>(out)})
        if (fvv::mem_kind(p) != fvv::MemKind::Device)
            return fail(FVV_ERR_INVALID_ARG, "fvv_depth_jbf: buffers must be device memory");
    fvv::JbfParams P;
    fvv::jbf_params(*opt, width, height, &P);
    P.cam[0].rgb = rgb;
    P.cam[0].rgb_pitch = int64_t(rgb_pitch);
    P.cam[0].src = depth;
    P.cam[0].src_pitch = int64_t(depth_pitch / 2);
    P.cam[0].dst = out;
    P.cam[0].dst_pitch = int64_t(out_pitch / 2);
    cudaError_t e = fvv::launch_jbf(P, 1, static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(FVV_ERR_CUDA, std::string("fvv_depth_jbf: ") + cudaGetErrorString(e));
    }
    return FVV_OK;
}
