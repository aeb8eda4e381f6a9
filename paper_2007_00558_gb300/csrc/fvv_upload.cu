// fvv_upload.cu -- batched frame upload: one tick of every camera of equal
// size lands in a frame-ring slot in one launch (RGB8 -> RGBA8 packing and
// the depth rows), after at most two bulk host-to-device copies.
#include "fvv_runtime.h"

namespace fvv {

namespace {

// Eq. (3) inverted for one pixel: its Y byte and the 4 MSBs from the U (top
// row of the 2x2 block) or V (bottom row) byte, bit i of the left pixel at bit
// 2i and of the right one at bit 2i + 1, gathered by two mask-and-shift steps.
__device__ __forceinline__ uint32_t code12(uint32_t ybyte, uint32_t uv, uint32_t right)
{
    uint32_t m = (uv >> right) & 0x55u;
    m = (m | (m >> 1)) & 0x33u;
    m = (m | (m >> 2)) & 0x0Fu;
    return (m << 8) | ((m & 1u) ? 255u - ybyte : ybyte);
}

// Every camera of one tick: RGB8 -> RGBA8 and depth rows into the slot.  A
// thread takes four texels of a row of camera blockIdx.z: with kVec three
// 4-byte loads of colour, one load of the four codes (8 bytes) or of their Y
// bytes (4) and chroma bytes (2), one 16-byte and one 8-byte store.  It is
// bound by HBM at 11 bytes per texel (10.5 with YUV420 depth); one texel a
// thread with byte loads, five loads and two stores a texel, took 42 us
// for nine 1280x720 cameras with YUV420 depth, this 16 us (87 MB: 5.4 TB/s).
// Without kVec, and at a row's ragged end, texel by texel.
constexpr int kQuadsX = 64, kRowsY = 4;
template <bool kVec>
__global__ void __launch_bounds__(kQuadsX * kRowsY) k_upload_all(const __grid_constant__ UploadAll u)
{
    const int x0 = 4 * (blockIdx.x * kQuadsX + threadIdx.x);
    const int y = blockIdx.y * kRowsY + threadIdx.y, k = blockIdx.z;
    if (x0 >= u.W || y >= u.H)
        return;
    const uint8_t* p = u.rgb + k * u.rgb_cam_stride + size_t(y) * u.rgb_pitch + 3 * size_t(x0);
    uint32_t* rgba = reinterpret_cast<uint32_t*>(u.slot + u.off_rgba[k]) + size_t(y) * u.rpitch + x0;
    uint16_t* dd = (u.ddst[k] ? u.ddst[k] : reinterpret_cast<uint16_t*>(u.slot + u.off_depth[k])) +
                   size_t(y) * u.dpitch + x0;
    const uint16_t* lut = u.lut[k];
    // depth: a row of codes, or of Y bytes and of the chroma plane of its row parity
    const uint8_t* blk = u.depth + k * u.depth_cam_stride;
    const size_t yb = size_t(u.W) * u.H, cb = size_t(u.W / 2) * (u.H / 2);
    const uint8_t* drow = u.yuv ? blk + size_t(y) * u.W + x0 : blk + size_t(y) * u.depth_pitch + 2 * size_t(x0);
    const uint8_t* crow = blk + yb + ((y & 1) ? cb : 0) + size_t(y >> 1) * (u.W / 2) + (x0 >> 1);
    if (kVec && x0 + 4 <= u.W) {
        const uint32_t* p4 = reinterpret_cast<const uint32_t*>(p);
        const uint32_t a = __ldg(p4), b = __ldg(p4 + 1), c = __ldg(p4 + 2);
        uint2 codes;
        if (u.yuv) {
            const uint32_t yy = __ldg(reinterpret_cast<const uint32_t*>(drow));
            const uint32_t cc = __ldg(reinterpret_cast<const uint16_t*>(crow));
            uint32_t d[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                d[i] = __ldg(lut + code12((yy >> (8 * i)) & 255u, (cc >> (8 * (i >> 1))) & 255u, i & 1));
            codes = make_uint2(d[0] | (d[1] << 16), d[2] | (d[3] << 16));
        } else {
            codes = __ldg(reinterpret_cast<const uint2*>(drow));
        }
        *reinterpret_cast<uint4*>(rgba) =
            make_uint4(a & 0xFFFFFFu, __byte_perm(a, b, 0x0543) & 0xFFFFFFu, __byte_perm(b, c, 0x0432) & 0xFFFFFFu, c >> 8);
        *reinterpret_cast<uint2*>(dd) = codes;
        return;
    }
    for (int i = 0; i < 4 && x0 + i < u.W; ++i) {
        rgba[i] = uint32_t(p[3 * i]) | (uint32_t(p[3 * i + 1]) << 8) | (uint32_t(p[3 * i + 2]) << 16);
        dd[i] = u.yuv ? __ldg(lut + code12(drow[i], crow[i >> 1], i & 1)) : reinterpret_cast<const uint16_t*>(drow)[i];
    }
}

}  // namespace

cudaError_t launch_upload_all(const UploadAll& u, cudaStream_t stream)
{
    if (u.W <= 0 || u.H <= 0 || u.n_cams <= 0) return cudaSuccess;
    // the wide form applies when every load it makes is aligned (the slot's
    // rows start on 128 bytes)
    auto mult = [](const void* p, size_t a, size_t b, size_t n) {
        return (reinterpret_cast<uintptr_t>(p) | a | b) % n == 0;
    };
    const bool vec = mult(u.rgb, u.rgb_cam_stride, u.rgb_pitch, 4) &&
                     (u.yuv ? mult(u.depth, u.depth_cam_stride, size_t(u.W), 4)
                            : mult(u.depth, u.depth_cam_stride, u.depth_pitch, 8));
    dim3 grid(unsigned((u.W + 4 * kQuadsX - 1) / (4 * kQuadsX)), unsigned((u.H + kRowsY - 1) / kRowsY),
              unsigned(u.n_cams));
    if (vec)
        k_upload_all<true><<<grid, dim3(kQuadsX, kRowsY), 0, stream>>>(u);
    else
        k_upload_all<false><<<grid, dim3(kQuadsX, kRowsY), 0, stream>>>(u);
    return cudaGetLastError();
}

}  // namespace fvv
