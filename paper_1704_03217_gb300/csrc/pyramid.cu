// pyramid.cu -- gradient pyramid of one image on the GPU.
//
// Steps (one kernel each, all integer, all HBM/L2-streaming):
//   level 0: gray conversion (PGM-G/GD, Sec. III-F) or RGB de-interleave
//   levels 1..L-1: 5x5 binomial [1 4 6 4 1]^2 / 256 with decimation by 2 and
//            replicated border (Sec. III-D, downsample factor s = 1/2)
//   per level and direction: colour space of Table 2 (Sec. III-E): RGB,
//            CIELab or YCrCb, integer definitions
//   per level and direction: Sobel gradients Gx, Gy (Eq. 1-2), S = 3 or 5,
//            replicated border, int16, pixel-interleaved; for the direction
//            descriptor (Sec. III-F) their signs.
#include <string.h>

#include "match_common.cuh"

namespace pgm {
namespace {

__device__ __forceinline__ int gray_q14(int r, int g, int b) {
    // BT.601 luma weights 0.299, 0.587, 0.114 in Q14 (sum 16384)
    return (4899 * r + 9617 * g + 1868 * b + 8192) >> 14;
}

// Level 0 and the downsampling take a batch of images (blockIdx.z); the grid
// covers the largest image and blocks outside an image's extent return.  The
// colour conversion, the gradients and the bit-planes depend only on the
// level images: one launch takes every level and direction of every image,
// its blocks numbered through (PyrBatch::cum), where a launch per level and
// direction left the chip to a few small blocks at a time (two frames of 1920 x
// 1080: 22 -> 7 launches, the build 296 -> 204 us).
__device__ __forceinline__ int pyr_item(const PyrBatch& B, int block) {
    int lo = 0, hi = B.n - 1;                 // the last item with cum <= block
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (B.cum[mid] <= block) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// ---------------------------------------------------------------- level 0
// mode 0: gray input copied; mode 1: RGB -> gray; mode 2: RGB -> 3 planes.
// A thread makes 4 consecutive pixels (one 32-bit store per output plane;
// level rows are 16-byte aligned).
__global__ void k_level0(const __grid_constant__ PyrBatch B) {
    const PyrItem& it = B.it[blockIdx.z];
    const int x = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= it.sw || y >= it.sh) return;
    const uint8_t* src = it.src + (size_t)y * it.pitch;
    uint8_t* out = it.dst;
    const size_t o = (size_t)y * it.drow + x;
    const int n = it.sw - x < 4 ? it.sw - x : 4;
    uint32_t p0 = 0, p1 = 0, p2 = 0;
    for (int k = 0; k < n; ++k) {
        if (it.mode == 0) {
            p0 |= (uint32_t)src[x + k] << (8 * k);
        } else {
            const int r = src[3 * (x + k)], g = src[3 * (x + k) + 1], b = src[3 * (x + k) + 2];
            if (it.mode == 1) {
                p0 |= (uint32_t)gray_q14(r, g, b) << (8 * k);
            } else {
                p0 |= (uint32_t)r << (8 * k);
                p1 |= (uint32_t)g << (8 * k);
                p2 |= (uint32_t)b << (8 * k);
            }
        }
    }
    if (n == 4) {
        *reinterpret_cast<uint32_t*>(out + o) = p0;
        if (it.mode == 2) {
            *reinterpret_cast<uint32_t*>(out + it.dplane + o) = p1;
            *reinterpret_cast<uint32_t*>(out + 2 * it.dplane + o) = p2;
        }
    } else {
        for (int k = 0; k < n; ++k) {
            out[o + k] = (uint8_t)(p0 >> (8 * k));
            if (it.mode == 2) {
                out[it.dplane + o + k] = (uint8_t)(p1 >> (8 * k));
                out[2 * it.dplane + o + k] = (uint8_t)(p2 >> (8 * k));
            }
        }
    }
}

// ------------------------------------------------------- binomial down
// Four consecutive output pixels per thread; blockIdx.z = image * C + channel.
// The separable sums are exact integers, so summing rows first equals the 2D
// sum of the definition.  Away from the left and right borders an input row's
// eleven bytes come from four aligned words (level rows are padded to 16
// bytes); a thread at a border reads them one by one, clamped.  Two frames of
// 1920 x 1080: 36 -> 28 us, the build 203 -> 198.
__global__ void k_down(const __grid_constant__ PyrBatch B, int C) {
    const PyrItem& it = B.it[blockIdx.z / C];
    const int ch = blockIdx.z % C;
    const int x = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= it.dw || y >= it.dh) return;
    const uint8_t* src = it.src + ch * it.splane;
    const int k[5] = {1, 4, 6, 4, 1};
    const bool inner = x > 0 && 2 * x + 8 < it.sw;      // columns 2 x - 2 .. 2 x + 8
    int acc[4] = {0, 0, 0, 0};
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        const uint8_t* r = src + (size_t)clampi(2 * y + j - 2, 0, it.sh - 1) * it.srow;
        int v[11];
        if (inner) {
            const uint32_t* q = reinterpret_cast<const uint32_t*>(r + 2 * x - 4);
            const uint32_t w[4] = {q[0], q[1], q[2], q[3]};
#pragma unroll
            for (int i = 0; i < 11; ++i) v[i] = (int)((w[(i + 2) / 4] >> (8 * ((i + 2) % 4))) & 255u);
        } else {
#pragma unroll
            for (int i = 0; i < 11; ++i) v[i] = r[clampi(2 * x + i - 2, 0, it.sw - 1)];
        }
#pragma unroll
        for (int o = 0; o < 4; ++o) {
            int s = 0;
#pragma unroll
            for (int i = 0; i < 5; ++i) s += k[i] * v[2 * o + i];
            acc[o] += k[j] * s;
        }
    }
    uint8_t* out = it.dst + ch * it.dplane + (size_t)y * it.drow + x;
    if (x + 4 <= it.dw) {
        *reinterpret_cast<uint32_t*>(out) = (uint32_t)((acc[0] + 128) >> 8) | (uint32_t)((acc[1] + 128) >> 8) << 8 |
                                            (uint32_t)((acc[2] + 128) >> 8) << 16 |
                                            (uint32_t)((acc[3] + 128) >> 8) << 24;
    } else {
        for (int o = 0; x + o < it.dw; ++o) out[o] = (uint8_t)((acc[o] + 128) >> 8);
    }
}

// ------------------------------------------------------- colour spaces
// Integer cube root of v <= 2^48: the floor of a float estimate, then one
// exact correction step each way.  The estimate 2^(log2(v) / 3) from the
// fast base-2 logarithm and exponential (each documented within 2 units in
// the last place here; log2(v) < 49) is within about 2e-6 of the root
// relatively, so for roots below 2^17 its integer part is off by at most
// one.  All 2^24 colours are checked against the oracle on the GPU.
__device__ __forceinline__ uint32_t icbrt48(unsigned long long v) {
    int c = v ? (int)exp2f(__log2f((float)v) * (1.0f / 3.0f)) : 0;
    const unsigned long long cc = (unsigned long long)(unsigned)c * (unsigned)c;
    if (c > 0 && cc * (unsigned)c > v) --c;
    const unsigned n = (unsigned)c + 1u;
    if ((unsigned long long)n * n * n <= v) ++c;
    return (uint32_t)c;
}

// CIELab companding function of t = T / (255 * 2^16), result scaled by 2^16.
__device__ __forceinline__ int lab_f(uint32_t T) {
    if (T > 148006u) {                                    // t > (6/29)^3: T 24389 > 216 255 2^16
        // t * 2^48 = floor(T 2^32 / 255) = T (2^32 - 1) / 255 + floor(T / 255); T < 2^24
        return (int)icbrt48((unsigned long long)T * 16843009ull + T / 255u);
    }
    // t * 841/108 + 4/29
    return (int)(((unsigned long long)T * (841 * 29) + 4ull * 65536 * 108 * 255) / (108u * 255 * 29));
}

__device__ __forceinline__ void to_lab(int r, int g, int b, int* o) {
    // D65 RGB -> XYZ / white, Q16 rows summing to 65536, linear RGB
    const int fx = lab_f(28439u * r + 24656u * g + 12441u * b);
    const int fy = lab_f(13937u * r + 46869u * g + 4730u * b);
    const int fz = lab_f(1164u * r + 7175u * g + 57197u * b);
    // 9039 <= f <= 65536: the numerator lies in [3263540, 1674444800]
    const int Ls = (int)((uint32_t)((116 * fy - 16 * 65536) * 255 + 3276800) / 6553600u);
    const int As = (500 * (fx - fy) + 128 * 65536 + 32768) >> 16;      // floor division
    const int Bs = (200 * (fy - fz) + 128 * 65536 + 32768) >> 16;
    o[0] = clampi(Ls, 0, 255);
    o[1] = clampi(As, 0, 255);
    o[2] = clampi(Bs, 0, 255);
}

__device__ __forceinline__ void to_ycrcb(int r, int g, int b, int* o) {
    int y = gray_q14(r, g, b);
    o[0] = y;
    o[1] = clampi(((r - y) * 11682 + (128 << 14) + 8192) >> 14, 0, 255);   // floor division
    o[2] = clampi(((b - y) * 9241 + (128 << 14) + 8192) >> 14, 0, 255);
}

// Four consecutive pixels per thread, one 32-bit access per plane (level rows
// are padded to 16 bytes; the pad is converted too and never read), and all
// but the cube roots in 32-bit integers: bound by integer issue, 66 -> 40 us for
// two frames of 1920 x 1080.
constexpr int CV_W = 128, CV_H = 8;           // pixels of a block
__global__ void __launch_bounds__(256) k_convert(const __grid_constant__ PyrBatch B) {
    const int k = pyr_item(B, blockIdx.x);
    const PyrItem& it = B.it[k];
    const int nbx = (it.sw + CV_W - 1) / CV_W, at = (int)blockIdx.x - B.cum[k];
    const int x = (at % nbx) * CV_W + 4 * (int)(threadIdx.x & 31), y = (at / nbx) * CV_H + (int)(threadIdx.x >> 5);
    if (x >= it.sw || y >= it.sh) return;
    const size_t o = (size_t)y * it.srow + x, plane = it.splane;
    const uint32_t r = *reinterpret_cast<const uint32_t*>(it.src + o);
    const uint32_t g = *reinterpret_cast<const uint32_t*>(it.src + plane + o);
    const uint32_t b = *reinterpret_cast<const uint32_t*>(it.src + 2 * plane + o);
    uint32_t c[3] = {0, 0, 0};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int R = (r >> (8 * i)) & 255, G = (g >> (8 * i)) & 255, Bl = (b >> (8 * i)) & 255;
        int v[3];
        if (it.mode == SP_LAB) to_lab(R, G, Bl, v); else to_ycrcb(R, G, Bl, v);
#pragma unroll
        for (int q = 0; q < 3; ++q) c[q] |= (uint32_t)v[q] << (8 * i);
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) *reinterpret_cast<uint32_t*>(it.dst + q * plane + o) = c[q];
}

// ----------------------------------------------------------------- Sobel
// Gx = sum_j s_j sum_i d_i I(x+i, y+j); Gy with the roles of the axes swapped.
// A CTA of 32 x 8 threads makes a 32 x 16 block of one image (two rows per
// thread).  The (32 + S - 1) x (16 + S - 1) input pixels of every channel
// (border replicated) go to shared memory, as aligned 32-bit words for blocks
// away from the left and right borders; the horizontal passes (d and s along
// x, both within int16) are kept per input row as one packed word, and the
// vertical passes finish Gx and Gy (separable and exact in integers).  The
// output words (px_words per pixel: 3 data words and a zero word for colour,
// one word for gray) leave as one 16-byte store per colour pixel.  A block at an
// image edge stages them in shared memory and also writes the replicated border of BORD pixels next to it (a
// border pixel repeats the descriptor of the nearest image pixel, which the
// block holds), so every patch with its centre in the image can be read
// without clamping.
// Bound by integer issue, then by the 64 bytes written per colour pixel (two
// directions): 151 -> 110 us for two frames of 1920 x 1080 (353 MB, 3.2 TB/s)
// with four outputs of a horizontal pass from three words (byte loads before),
// the split on packed halves and no staging inside the image.
constexpr int SB_TW = 32, SB_TH = 16, SB_TY = 8, SB_XO = 4;   // SB_XO: staged columns left of x0
__device__ __forceinline__ int sb_d(int S, int i) {
    return S == 5 ? (i == 0 ? -1 : i == 1 ? -2 : i == 2 ? 0 : i == 3 ? 2 : 1) : (i - 1);
}
__device__ __forceinline__ int sb_s(int S, int i) {
    return S == 5 ? (i == 0 ? 1 : i == 1 ? 4 : i == 2 ? 6 : i == 3 ? 4 : 1) : (i == 1 ? 2 : 1);
}
// two values split into signed bytes (match_common.cuh, split_bytes) on packed
// halves: t = a + 64 + 2^14 >= 0 per half holds a_l + 64 in its low 7 bits and
// a_h + 128 above
__device__ __forceinline__ uint32_t sb_split(int a0, int a1) {
    const uint32_t t = (uint32_t)(a0 + 16448) + ((uint32_t)(a1 + 16448) << 16);
    const uint32_t l = (t & 0x007f007fu) + 0x00c000c0u, h = (t >> 7) & 0x01ff01ffu;   // + 256, + 128
    return __byte_perm(l, h, 0x6420) ^ 0x80800000u;
}
template <int S, int C>
__global__ void __launch_bounds__(SB_TW * SB_TY) k_sobel(const __grid_constant__ PyrBatch B,
                                                         int dir_only) {
    constexpr int R = S / 2, IH = SB_TH + S - 1;
    constexpr int IWW = (SB_XO + SB_TW + R + 3) / 4;     // staged words per row (x0 - 4 .. )
    constexpr int IW = 4 * IWW, NT = SB_TW * SB_TY;
    constexpr int PXW = px_words(2 * C);                 // words per pixel in the output arrays
    constexpr int OW = SB_TW * PXW;                      // output words per tile row and array
    __shared__ __align__(16) uint8_t sI[C][IH][IW];      // column c holds x = x0 - SB_XO + c
    __shared__ __align__(16) uint32_t sH[C][IH][SB_TW];  // (sum d v) low 16, (sum s v) high 16
    __shared__ __align__(16) uint32_t sO[2][SB_TH][OW];  // descriptor words, split words
    const int item = pyr_item(B, blockIdx.x);
    const PyrItem& it = B.it[item];
    const int w = it.sw, h = it.sh, row = it.srow;
    const int nbx = (w + SB_TW - 1) / SB_TW, at = (int)blockIdx.x - B.cum[item];
    const int x0 = (at % nbx) * SB_TW, y0 = (at / nbx) * SB_TH;
    const size_t plane = it.splane;
    const uint8_t* in = it.src;
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * SB_TW + tx;
    if (x0 >= SB_XO && x0 + SB_TW + R <= w) {
        // interior in x: rows start 16-byte aligned and x0 - SB_XO is a
        // multiple of 4, so whole words are read; the words end inside the
        // padded row (x0 - 4 + IW <= row)
        for (int e = tid; e < C * IH * IWW; e += NT) {
            const int ch = e / (IH * IWW), rem = e - ch * (IH * IWW), r = rem / IWW, k = rem - r * IWW;
            const uint8_t* src = in + ch * plane + (size_t)clampi(y0 - R + r, 0, h - 1) * row;
            *reinterpret_cast<uint32_t*>(&sI[ch][r][4 * k]) =
                *reinterpret_cast<const uint32_t*>(src + x0 - SB_XO + 4 * k);
        }
    } else {
        for (int e = tid; e < C * IH * IW; e += NT) {
            const int ch = e / (IH * IW), rem = e - ch * (IH * IW), r = rem / IW, c = rem - r * IW;
            const uint8_t* src = in + ch * plane + (size_t)clampi(y0 - R + r, 0, h - 1) * row;
            sI[ch][r][c] = src[clampi(x0 - SB_XO + c, 0, w - 1)];
        }
    }
    __syncthreads();
    // four neighbouring outputs from three words
    for (int e = tid; e < C * IH * (SB_TW / 4); e += NT) {
        const int ch = e / (IH * (SB_TW / 4)), rem = e - ch * (IH * (SB_TW / 4));
        const int r = rem / (SB_TW / 4), q = rem - r * (SB_TW / 4);
        const uint32_t* wd = reinterpret_cast<const uint32_t*>(&sI[ch][r][4 * q]);   // x0 + 4 q - 4 ..
        int v[12];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const uint32_t u = wd[k];
#pragma unroll
            for (int i = 0; i < 4; ++i) v[4 * k + i] = (int)((u >> (8 * i)) & 255u);
        }
        uint32_t o[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            int sd = 0, ss = 0;
#pragma unroll
            for (int t = 0; t < S; ++t) {
                const int z = v[SB_XO - R + i + t];
                sd += sb_d(S, t) * z;
                ss += sb_s(S, t) * z;
            }
            o[i] = (uint32_t)(uint16_t)sd | ((uint32_t)ss << 16);
        }
        *reinterpret_cast<uint4*>(&sH[ch][r][4 * q]) = make_uint4(o[0], o[1], o[2], o[3]);
    }
    __syncthreads();
    int g[2][2 * C];
#pragma unroll
    for (int ch = 0; ch < C; ++ch) {
        int gx0 = 0, gy0 = 0, gx1 = 0, gy1 = 0;
#pragma unroll
        for (int j = 0; j <= S; ++j) {                  // rows 2 ty .. 2 ty + S
            const uint32_t v = sH[ch][2 * ty + j][tx];
            const int sd = (int)(int16_t)(v & 0xffffu), ss = (int)(v >> 16);
            if (j < S) { gx0 += sb_s(S, j) * sd; gy0 += sb_d(S, j) * ss; }
            if (j > 0) { gx1 += sb_s(S, j - 1) * sd; gy1 += sb_d(S, j - 1) * ss; }
        }
        int gx[2] = {gx0, gx1}, gy[2] = {gy0, gy1};
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            int a = gx[k], b2 = gy[k];
            if (dir_only == 1) {                  // direction only: G ./ |G|
                a = (a > 0) - (a < 0);
                b2 = (b2 > 0) - (b2 < 0);
            } else if (dir_only == 2) {           // 8-sector angle as an integer unit vector
                const int ax = abs(a), ay = abs(b2);
                int cx, cy;
                if (a == 0 && b2 == 0) { cx = 0; cy = 0; }
                else if (408 * ay <= 169 * ax) { cx = a > 0 ? 64 : -64; cy = 0; }
                else if (408 * ax <= 169 * ay) { cx = 0; cy = b2 > 0 ? 64 : -64; }
                else { cx = a > 0 ? 45 : -45; cy = b2 > 0 ? 45 : -45; }
                a = cx; b2 = cy;
            }
            g[k][ch] = a;
            g[k][C + ch] = b2;
        }
    }
    // dst and split point at pixel (0, 0) of padded arrays with rows of rw
    // words (a multiple of 4); pixel (x, y) starts at word y rw + x PXW
    const ptrdiff_t rw = (ptrdiff_t)(it.drow >> 1);
    uint32_t* const dst0 = reinterpret_cast<uint32_t*>(it.dst);
    uint32_t* const dst1 = it.split;
    // this block's output: its tile, widened by the border where it touches
    // an image edge
    const bool left = x0 == 0, right = x0 + SB_TW >= w, top = y0 == 0, bottom = y0 + SB_TH >= h;
    const bool edge = left || right || top || bottom;
    const int xa = left ? -BORD : x0, xb = right ? w + BORD : x0 + SB_TW;
    const int ya = top ? -BORD : y0, yb = bottom ? h + BORD : y0 + SB_TH;
    // pixel-interleaved int16 as 32-bit words (2C is even), and the same
    // words with every value a split into signed bytes a = 128 a_h + a_l
    // (a_l in [-64, 63]) for the dp2a cross products.  A block inside the image
    // stores its pixels at once (a warp's row is contiguous); one at an edge
    // stages them for the border.
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        uint32_t wv[PXW], sv[PXW];
#pragma unroll
        for (int q = 0; q < PXW; ++q) {
            const bool dw = q < C;
            wv[q] = dw ? (uint32_t)(uint16_t)g[k][2 * q] | ((uint32_t)(uint16_t)g[k][2 * q + 1] << 16) : 0u;
            sv[q] = dw ? sb_split(g[k][2 * q], g[k][2 * q + 1]) : 0u;
        }
        if (!edge) {
            const ptrdiff_t o = (ptrdiff_t)(y0 + 2 * ty + k) * rw + (ptrdiff_t)(x0 + tx) * PXW;
            if constexpr (PXW == 4) {
                *reinterpret_cast<uint4*>(dst0 + o) = make_uint4(wv[0], wv[1], wv[2], wv[3]);
                *reinterpret_cast<uint4*>(dst1 + o) = make_uint4(sv[0], sv[1], sv[2], sv[3]);
            } else {
                dst0[o] = wv[0];
                dst1[o] = sv[0];
            }
        } else {
#pragma unroll
            for (int q = 0; q < PXW; ++q) {
                sO[0][2 * ty + k][tx * PXW + q] = wv[q];
                sO[1][2 * ty + k][tx * PXW + q] = sv[q];
            }
        }
    }
    if (edge) {
        __syncthreads();
        // a border pixel takes the words of the nearest image pixel, which
        // lies in this tile; a warp walks one output row, a pixel per lane
        // (colour pixels as one 16-byte store)
        const int nx = xb - xa, nrow = yb - ya;
        for (int r = ty; r < 2 * nrow; r += SB_TY) {
            const int a = r >= nrow, y = ya + (a ? r - nrow : r);
            const int sy = clampi(y, 0, h - 1) - y0;
            uint32_t* const orow = (a ? dst1 : dst0) + (ptrdiff_t)y * rw;
            for (int i = tx; i < nx; i += SB_TW) {
                const int x = xa + i, sx = clampi(x, 0, w - 1) - x0;
                if constexpr (PXW == 4) {
                    *reinterpret_cast<uint4*>(orow + (ptrdiff_t)x * 4) =
                        *reinterpret_cast<const uint4*>(&sO[a][sy][sx * 4]);
                } else {
#pragma unroll
                    for (int q = 0; q < PXW; ++q) orow[(ptrdiff_t)x * PXW + q] = sO[a][sy][sx * PXW + q];
                }
            }
        }
    }
}

// ------------------------------------------------- direction bit-planes
// For the direction descriptor: word w of padded row yy of the nonzero and
// the sign bit-plane from the padded descriptor (bit b = x nch + c holds
// value c of padded pixel x; words past the row are zero).  One thread per
// word.
template <int NCH>
__global__ void k_bits(const __grid_constant__ PyrBatch B) {
    constexpr int PXE = 2 * px_words(NCH);       // int16 elements per padded pixel
    const int item = pyr_item(B, blockIdx.x);
    const PyrItem& it = B.it[item];
    const int nbx = (it.brow + 31) / 32, at = (int)blockIdx.x - B.cum[item];
    const int w = (at % nbx) * 32 + threadIdx.x, yy = (at / nbx) * 8 + threadIdx.y;
    const int pw = it.sw + 2 * BORD, ph = it.sh + 2 * BORD;
    if (w >= it.brow || yy >= ph) return;
    // padded pixel x of row yy: it.dst points at pixel (0, 0), rows drow int16
    const int16_t* row = reinterpret_cast<const int16_t*>(it.dst) + (ptrdiff_t)(yy - BORD) * it.drow -
                         (ptrdiff_t)BORD * PXE;
    uint32_t nz = 0, sg = 0;
    const int b0 = 32 * w, x0 = b0 / NCH, x1 = min((b0 + 31) / NCH, pw - 1);
    for (int x = x0; x <= x1; ++x) {           // whole pixels, one vector load each
        int v[NCH];
        if constexpr (NCH == 6) {
            const uint4 q = *reinterpret_cast<const uint4*>(row + (ptrdiff_t)x * PXE);
            v[0] = (int16_t)(q.x & 0xffff); v[1] = (int16_t)(q.x >> 16);
            v[2] = (int16_t)(q.y & 0xffff); v[3] = (int16_t)(q.y >> 16);
            v[4] = (int16_t)(q.z & 0xffff); v[5] = (int16_t)(q.z >> 16);
        } else {
            const uint32_t q = *reinterpret_cast<const uint32_t*>(row + (ptrdiff_t)x * PXE);
            v[0] = (int16_t)(q & 0xffff); v[1] = (int16_t)(q >> 16);
        }
#pragma unroll
        for (int c = 0; c < NCH; ++c) {
            const int k = x * NCH + c - b0;
            if (k < 0 || k >= 32) continue;
            nz |= (uint32_t)(v[c] != 0) << k;
            sg |= (uint32_t)(v[c] < 0) << k;
        }
    }
    it.bits[(size_t)yy * it.brow + w] = nz;
    it.bits[(size_t)(ph + yy) * it.brow + w] = sg;
}

}  // namespace

// One launch per step of the pyramid for a whole batch of images (all with
// the same parameters; sizes may differ).
pgm_status launch_pyramid_batch(const pgm_params* p, int n, const PyrPlan* plans,
                                const uint8_t* const* imgs, const int* cs, const size_t* pitches,
                                uint8_t* const* pyrs, cudaStream_t st) {
    static thread_local PyrBatch B;
    const PyrPlan& p0 = plans[0];
    const int L = p0.L, C = p0.C, nsch = p0.nsch;
    dim3 blk(32, 8);
    auto grid = [&](int w, int h, int z) { return dim3((w + 31) / 32, (h + 7) / 8, z); };
    const int dir_only = p->descriptor;      // 0 full, 1 signs, 2 sectors
    for (int base = 0; base < n; base += PYR_MAXB) {
        const int m = n - base < PYR_MAXB ? n - base : PYR_MAXB;
        KScope ks(PGM_K_PYRAMID, st, L);
        // level 0
        int mw = 0, mh = 0;
        memset(&B, 0, sizeof(B));
        B.n = m;
        for (int k = 0; k < m; ++k) {
            const PyrPlan& pp = plans[base + k];
            PyrItem& it = B.it[k];
            it.src = imgs[base + k]; it.pitch = pitches[base + k];
            it.sw = pp.W[0]; it.sh = pp.H[0];
            it.dst = pyrs[base + k] + pp.img_off[0]; it.drow = pp.img_row[0];
            it.dplane = pp.img_plane[0];
            it.mode = cs[base + k] == 1 ? 0 : (C == 1 ? 1 : 2);
            mw = pp.W[0] > mw ? pp.W[0] : mw; mh = pp.H[0] > mh ? pp.H[0] : mh;
        }
        k_level0<<<grid((mw + 3) / 4, mh, m), blk, 0, st>>>(B);
        for (int l = 1; l < L; ++l) {
            mw = mh = 0;
            for (int k = 0; k < m; ++k) {
                const PyrPlan& pp = plans[base + k];
                const uint8_t* pyr = pyrs[base + k];
                PyrItem& it = B.it[k];
                it.src = pyr + pp.img_off[l - 1]; it.sw = pp.W[l - 1]; it.sh = pp.H[l - 1];
                it.srow = pp.img_row[l - 1]; it.splane = pp.img_plane[l - 1];
                it.dst = pyrs[base + k] + pp.img_off[l]; it.dw = pp.W[l]; it.dh = pp.H[l];
                it.drow = pp.img_row[l]; it.dplane = pp.img_plane[l];
                mw = pp.W[l] > mw ? pp.W[l] : mw; mh = pp.H[l] > mh ? pp.H[l] : mh;
            }
            k_down<<<grid((mw + 3) / 4, mh, m * C), blk, 0, st>>>(B, C);
        }
        // every level and direction of every image, PYR_MAXB items a launch
        auto items = [&](int what) {              // 0 conversion, 1 gradients, 2 bit-planes
            int at = 0, launches = 0;
            auto flush = [&]() {
                B.n = at;
                const int blocks = B.cum[at];
                at = 0;
                if (blocks == 0) return;
                ++launches;
                if (what == 0) {
                    k_convert<<<blocks, 256, 0, st>>>(B);
                } else if (what == 2) {
                    if (C == 3) k_bits<6><<<blocks, dim3(32, 8), 0, st>>>(B);
                    else k_bits<2><<<blocks, dim3(32, 8), 0, st>>>(B);
                } else {
                    const dim3 sblk(SB_TW, SB_TY);
                    if (p->sobel == 5) {
                        if (C == 1) k_sobel<5, 1><<<blocks, sblk, 0, st>>>(B, dir_only);
                        else k_sobel<5, 3><<<blocks, sblk, 0, st>>>(B, dir_only);
                    } else {
                        if (C == 1) k_sobel<3, 1><<<blocks, sblk, 0, st>>>(B, dir_only);
                        else k_sobel<3, 3><<<blocks, sblk, 0, st>>>(B, dir_only);
                    }
                }
            };
            B.cum[0] = 0;
            for (int l = 0; l < L; ++l)           // the large levels first
                for (int s = 0; s < nsch; ++s) {
                    const int sp = p0.space[s][l];
                    if (what == 0 && sp != SP_LAB && sp != SP_YCRCB) continue;
                    for (int k = 0; k < m; ++k) {
                        const PyrPlan& pp = plans[base + k];
                        uint8_t* pyr = pyrs[base + k];
                        PyrItem& it = B.it[at];
                        it.sw = pp.W[l]; it.sh = pp.H[l];
                        it.srow = pp.img_row[l]; it.splane = pp.img_plane[l];
                        int blocks;
                        if (what == 0) {
                            it.src = pyr + pp.img_off[l];
                            it.dst = pyr + pp.cimg_off[s][l];
                            it.mode = sp;
                            blocks = ((it.sw + CV_W - 1) / CV_W) * ((it.sh + CV_H - 1) / CV_H);
                        } else {
                            it.src = pyr + pp.cimg_off[s][l];
                            it.dst = pyr + pp.desc_off[s][l]; it.drow = pp.desc_row[l];
                            it.split = reinterpret_cast<uint32_t*>(pyr + pp.split_off[s][l]);
                            blocks = ((it.sw + SB_TW - 1) / SB_TW) * ((it.sh + SB_TH - 1) / SB_TH);
                        }
                        if (what == 2) {
                            it.bits = reinterpret_cast<uint32_t*>(pyr + pp.bits_off[s][l]);
                            it.brow = pp.bit_row[l];
                            blocks = ((it.brow + 31) / 32) * ((it.sh + 2 * BORD + 7) / 8);
                        }
                        B.cum[at + 1] = B.cum[at] + blocks;
                        if (++at == PYR_MAXB) flush();
                    }
                }
            flush();
            return launches;
        };
        ks.n = L + items(0) + items(1) + (dir_only == 1 ? items(2) : 0);
        if (pgm_status r = launch_status("pyramid: launch"); r != PGM_OK) return r;
    }
    return PGM_OK;
}

}  // namespace pgm
