// Whole-plane kernels for 16-bit activations with two or more levels (k = 3, 5): base convolution, level 1 and its synthesis as
// one contraction on tcgen05 (see tensor_kernels.cuh for the algebra, the operand layout and the weights' three parts), levels
// >= 2 as fp32 FMA tiles on the low-pass band, both from the same planes in shared memory, by different warps of one block.
//
// A unit is 8 S images of one channel.  The roles of a block's 26 (22) warps, each a pipeline stage:
//   loaders (8, 4) the unit's planes, global memory -> operand layout (rows of an odd number of pixels are shifted in
//                  registers), the B operand when the channel changes
//   deep (12)      the level-2 coefficients from 4 x 4 pixels of the operand array, deeper levels from the low-pass band, their
//                  convolutions (4 x 4 register tiles), Proposition 2 down to one value R per 2 x 2 pixels
//   issuers (2)    ten MMAs of 128 x 48 x 16 per 32 rows x 8 columns x 8 images
//   epilogue (4)   accumulators + R / 2 + bias -> global memory
// With several operand arrays the next units are loaded and their levels >= 2 computed while this one's MMAs and epilogue run; where
// only one fits (56 x 56 and the like), the deep warps read the next unit from global memory instead.
//
// Measured forward against the block-per-plane kernels, bf16: 128 x 96 x 56 x 56, three levels, 188 -> 121 us; 128 x 192 x 28 x 28,
// two levels, 107 -> 63; 64 x 384 x 14 x 14, three levels, 58 -> 52; 64 x 96 x 30 x 30 46 -> 30, 64 x 96 x 57 x 55 143 -> 113.  What
// bounds it now is instruction issue (2.1 of 4 a cycle, most warps waiting for their own last instruction) beside shared memory,
// whose cycles the MMAs' A operand takes a third of.
#pragma once
#include "tensor_kernels.cuh"

namespace wt {
namespace pyramid {

using plane::FastDiv;
using plane::fdiv;
using plane::make_fastdiv;
using tensor::fence_after;
using tensor::fence_before;
using tensor::mbar_arrive;
using tensor::mma;
using tensor::mma_commit;
using tensor::NCOL;
using tensor::smem_desc;
using tensor::TABLE_BYTES;
using tensor::TAP_BYTES;
using tensor::TAPS;
using tensor::u64;

constexpr int EPI = 128, DEEP = 384, ISS = 2, OTHERS = EPI + DEEP + 32 * ISS;  // threads and (ISS) warps of the roles but the loaders
constexpr int MANY = 256, FEW = 128;  // loaders: through registers, or issuing asynchronous copies
constexpr int RING = 8, MAXL = 8, MAX_BUFS = 4, WS = plane::WT_STRIDE;
constexpr int BAR_DEEP = 3, BAR_LOAD = 4, BAR_EPI = 5;  // named barriers
constexpr int CHUNK = 144;                 // bytes from one chunk of eight images to the next: one image's chunks fall on different banks
constexpr int MIS = 560;                   // floats a channel: folded weights, M, scale, bias (see tensor::build_table)

struct PGeom {
    int B, C, H, W, HW, L, K;
    int S, period, rows, T, n, Pc;      // octets per unit, array rows from one octet to the next, rows allocated, M tiles, output chunks, chunks per row
    int upc, units;                     // units per channel, units
    int bufs, rbufs;                    // operand arrays, R sets
    int direct;                         // the deep warps read global memory: the one operand array holds the unit before theirs
    int nb, items;                      // planes whose levels >= 2 are computed together, conv tiles of one plane
    int a_bytes, r_floats, rslot, rpitch;
    int dslot;                          // floats of one plane's coefficients
    int Hl[MAXL + 1], Wl[MAXL + 1], tx[MAXL + 1], rowsl[MAXL + 1], pitch[MAXL + 1], offY[MAXL + 1], zpitch[MAXL + 1], offZ[MAXL + 1], first[MAXL + 2];
    int out_stride;                     // bytes of one plane of the output image
    int r_off, deep_off, wtab_off, parts_off, table_off, out_off, misc_off, smem;  // byte offsets
    int nblocks, vec;                   // vec: pixels a load (4, 2), 1: odd rows
    int no_copy;
    FastDiv d_period, d_n, d_items, d_nt[MAXL + 1], d_tx[MAXL + 1], d_hw[MAXL + 1], d_w[MAXL + 1];
    int *alarm;
    unsigned tag;
};

__device__ __forceinline__ void named_sync(int id, int count) {
    __syncwarp();
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}

// ------------------------------------------------------------------ loading
// Chunk j of a row holds columns 8j - 4 .. 8j + 3; what lies outside the plane is never written and stays zero.  A warp moves
// whole rows of the same one to eight images, a piece of four (two) pixels a lane, seven rows under way: few lines of global memory
// an instruction, and the chunks' distance keeps an image's pieces on different banks.  A lane's addresses are worked out once an
// octet: a warp alone issues an instruction every four to five cycles, so what counts here, as in the other roles, is how many
// instructions a unit takes.
template <typename T, int PIX, int WARPS>
__device__ __forceinline__ void load_rows(const PGeom &g, char *arr, const T *__restrict__ x, int c, int k, int warp, int lane) {
    using V = typename std::conditional<PIX == 4, uint2, unsigned>::type;
    constexpr int U = 7;
    const int pieces = g.W / PIX, lp = pieces > 16 ? 5 : pieces > 8 ? 4 : pieces > 4 ? 3 : 2;  // log2 of the lanes to a row
    const int sets = lp - 2, q = lane & ((1 << lp) - 1), col = PIX * q + 4;                      // log2 of the warps that share a row's images
    const int img = ((warp & ((1 << sets) - 1)) << (5 - lp)) + (lane >> lp), y0 = warp >> sets, dy = WARPS >> sets;
    const int rowb = g.Pc * CHUNK, sstep = dy * g.W * 2, dstep = dy * rowb;
    if (q >= pieces) return;
    for (int o = 0; o < g.S; ++o) {
        const int b = (k * g.S + o) * 8 + img;
        if (b >= g.B) continue;
        const char *src = reinterpret_cast<const char *>(x + ((size_t)b * g.C + c) * g.HW + y0 * g.W + PIX * q);
        char *dst = arr + (o * g.period + 4 + y0) * rowb + img * 16 + (col >> 3) * CHUNK + (col & 7) * 2;
        for (int left = g.H - y0; left > 0; left -= U * dy, src += U * sstep, dst += U * dstep) {
            V v[U];
#pragma unroll
            for (int i = 0; i < U; ++i)
                if (i * dy < left) v[i] = __ldg(reinterpret_cast<const V *>(src + i * sstep));
#pragma unroll
            for (int i = 0; i < U; ++i)
                if (i * dy < left) *reinterpret_cast<V *>(dst + i * dstep) = v[i];
        }
    }
}
// One tensor's rows into the operand layout, PIX pixels a copy; images that do not exist are zeros.  arr: the plane's first row.  A lane
// walks down the rows of one image (of two): few warps issue all copies of a unit, so the loop is as short as it can be.
template <int PIX, int WARPS, typename T, typename G>
__device__ __forceinline__ void copy_rows(const G &g, char *arr, int P, int shift, const T *__restrict__ x, int c, int k, int warp, int lane) {
    const int pieces = g.W / PIX, lp = pieces > 16 ? 5 : pieces > 8 ? 4 : pieces > 4 ? 3 : 2;  // log2 of the lanes to a row
    const int q = lane & ((1 << lp) - 1), per = WARPS * (32 >> lp), first = warp * (32 >> lp) + (lane >> lp);  // rows under way, this lane's
    const int col = PIX * q + shift, rowb = P * CHUNK, dy = per >= 8 ? per / 8 : 1, sstep = dy * g.W * 2, dstep = dy * rowb;
    if (q >= pieces) return;
    const unsigned to = plane::smem_addr(arr) + (col >> 3) * CHUNK + (col & 7) * 2;
    for (int o = 0; o < g.S; ++o)
        for (int img = first & 7; img < 8; img += per) {
            const int y0 = first >> 3, b = (k * g.S + o) * 8 + img;
            const int bytes = b < g.B ? 2 * PIX : 0;
            const char *src = reinterpret_cast<const char *>(b < g.B ? x + ((size_t)b * g.C + c) * g.HW + y0 * g.W + PIX * q : x);
            const int step = b < g.B ? sstep : 0;
            unsigned dst = to + (o * g.period + y0) * rowb + img * 16;
#pragma unroll 4
            for (int y = y0; y < g.H; y += dy, src += step, dst += dstep) {
                if (PIX == 8) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
                else asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(dst), "l"(src), "n"(2 * PIX), "r"(bytes) : "memory");
            }
        }
}

// Rows of an odd number of pixels start at any element: aligned 32-bit words, shifted by one pixel where need be.  P chunks a row, the
// first begins SHIFT columns to the left of the plane; arr: the plane's first row.  ZERO: images that do not exist are zeros.
template <typename T, int SHIFT, int WARPS, bool ZERO, typename G>
__device__ __forceinline__ void load_shifted(const G &g, char *arr, int P, const T *__restrict__ x, int c, int k, int warp, int lane) {
    constexpr int U = 2;
    const int img = lane & 7;
    const unsigned rowb = (unsigned)P * CHUNK;
    const long long total = (long long)g.B * g.C * g.HW;
    const unsigned *words = reinterpret_cast<const unsigned *>(x);
    const unsigned short *pix = reinterpret_cast<const unsigned short *>(x);
    for (int o = 0; o < g.S; ++o) {
        const int b = (k * g.S + o) * 8 + img;
        const bool there = b < g.B;
        if (!ZERO && !there) continue;
        const long long plane = there ? ((long long)b * g.C + c) * g.HW : 0;
        for (int y0 = warp; y0 < g.H; y0 += U * WARPS) {
            for (int j = lane >> 3; j < P; j += 4) {
                const int x0 = 8 * j - SHIFT;
                unsigned v[U][5];
#pragma unroll
                for (int i = 0; i < U; ++i) {
                    const int y = y0 + i * WARPS;
                    const long long e = plane + (long long)y * g.W + x0, w = e >> 1;  // (arithmetic shift: e may be negative)
#pragma unroll
                    for (int q = 0; q < 5; ++q) v[i][q] = 0u;
                    if (y < g.H && x0 < g.W && there) {
                        if (w >= 0 && 2 * (w + 5) <= total) {
#pragma unroll
                            for (int q = 0; q < 5; ++q) v[i][q] = __ldg(words + w + q);
                        } else {
#pragma unroll
                            for (int q = 0; q < 10; ++q)
                                if (2 * w + q >= 0 && 2 * w + q < total) v[i][q >> 1] |= (unsigned)__ldg(pix + 2 * w + q) << (16 * (q & 1));
                        }
                    }
                }
#pragma unroll
                for (int i = 0; i < U; ++i) {
                    const int y = y0 + i * WARPS;
                    if (y >= g.H || x0 >= g.W) continue;
                    const bool odd = (plane + (long long)y * g.W + x0) & 1;
                    unsigned h[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) h[q] = odd ? __funnelshift_r(v[i][q], v[i][q + 1], 16) : v[i][q];
                    if (x0 < 0 || x0 + 8 > g.W) {
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            if ((unsigned)(x0 + q) >= (unsigned)g.W) h[q >> 1] &= q & 1 ? 0x0000ffffu : 0xffff0000u;
                    }
                    *reinterpret_cast<uint4 *>(arr + (unsigned)(o * g.period + y) * rowb + j * CHUNK + img * 16) = make_uint4(h[0], h[1], h[2], h[3]);
                }
            }
        }
    }
}
// A unit's planes on their way to L2, a line a request: what is left of the loads' latency is L2's.
template <typename T, int WARPS, typename G>
__device__ __forceinline__ void prefetch_planes(const G &g, const T *__restrict__ x, int c, int k, int warp, int lane) {
    for (int slot = warp; slot < 8 * g.S; slot += WARPS) {
        const int b = k * 8 * g.S + slot;
        if (b >= g.B) break;
        const char *p = reinterpret_cast<const char *>(x + ((size_t)b * g.C + c) * g.HW), *end = p + g.HW * 2;
        for (p += 128 * lane; p < end; p += 128 * 32) asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
    }
}

// ------------------------------------------------------------------ levels >= 2
// Eq. 5 with its factor inside the second sums (a power of two: the results are haar_butterfly's, but no sum is larger than they are).
__device__ __forceinline__ Haar4 butterfly(float a, float b, float c, float d) {
    const float s0 = a + b, d0 = a - b, s1 = 0.5f * (c + d), d1 = 0.5f * (c - d);
    return {fmaf(0.5f, s0, s1), fmaf(0.5f, s0, -s1), fmaf(0.5f, d0, d1), fmaf(0.5f, d0, -d1)};
}
struct Tile {
    int src, wt, z, meta;  // window, folded weights, output (float indices); meta: bit 31 valid, window pitch, Z pitch << 10, rows to store << 20
};
__device__ __forceinline__ Tile find_tile(const PGeom &g, int it) {
    Tile d;
    d.src = d.wt = d.z = d.meta = 0;
    if (it >= g.items * g.nb) return d;
    const int slot = fdiv(it, g.d_items);
    int r = it - slot * g.items, l = 2;
    while (r >= g.first[l + 1]) ++l;
    r -= g.first[l];
    const int sub = fdiv(r, g.d_nt[l]);
    r -= sub * (int)g.d_nt[l].d;
    const int ty = fdiv(r, g.d_tx[l]), tx = r - ty * g.tx[l];
    d.src = slot * g.dslot + g.offY[l] + (sub * g.rowsl[l] + 4 * ty) * g.pitch[l] + 4 * tx;
    d.wt = ((l - 2) * 4 + sub) * WS;
    d.z = slot * g.dslot + g.offZ[l] + (sub * g.Hl[l] + 4 * ty) * g.zpitch[l] + 4 * tx;
    int rows = g.Hl[l] - 4 * ty;
    if (rows > 4) rows = 4;
    d.meta = (int)(0x80000000u | (unsigned)g.pitch[l] | ((unsigned)g.zpitch[l] << 10) | ((unsigned)rows << 20));
    return d;
}
// KT = 3: the zeros around 3 x 3 kernels in their 5 x 5 tables meet no coefficient (which may be an infinity).
template <int KT>
__device__ __forceinline__ void run_tile(float *dp, const float *wtab, const Tile &d) {
    float w[25], acc[4][4];
    plane::load_weights(wtab + d.wt, w);
    plane::conv_tile<4, false, KT>(dp + d.src, d.meta & 0x3ff, w, acc);
    const int zp = (d.meta >> 10) & 0x3ff, rows = (d.meta >> 20) & 0xf;
#pragma unroll
    for (int r = 0; r < 4; ++r)
        if (r < rows) *reinterpret_cast<float4 *>(dp + d.z + r * zp) = make_float4(acc[r][0], acc[r][1], acc[r][2], acc[r][3]);
}
// Level-2 coefficients: a task is eight columns of four rows, two blocks of 4 x 4 pixels, either a chunk of the operand array or (rows
// of whole 16-byte words) straight from global memory; rows past the plane's H are not read from global memory (the operand array has
// zeros there).  row: the first of the four.
template <bool DIRECT>
__device__ __forceinline__ void load_blocks(uint4 (&w)[4], const char *q, int row_bytes, int row, int H) {
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        if (DIRECT) w[h] = row + h < H ? __ldg(reinterpret_cast<const uint4 *>(q + h * row_bytes)) : make_uint4(0u, 0u, 0u, 0u);
        else w[h] = *reinterpret_cast<const uint4 *>(q + h * row_bytes);
    }
}
// `y`: where the first block's coefficients go, `sub` floats from subband to subband; in0, in1: blocks inside the grid; returns a
// quarter of the sum of their pixels.
template <typename T>
__device__ __forceinline__ float analyse_blocks(const uint4 (&w)[4], float *y, int sub, bool in0, bool in1) {
    float ll[2][4], sum = 0.f;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const unsigned av[4] = {w[2 * h].x, w[2 * h].y, w[2 * h].z, w[2 * h].w}, bv[4] = {w[2 * h + 1].x, w[2 * h + 1].y, w[2 * h + 1].z, w[2 * h + 1].w};
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const float2 t = tensor::unpack16(av[m], T()), u = tensor::unpack16(bv[m], T());
            ll[h][m] = fmaf(0.5f, t.x + t.y, 0.5f * (u.x + u.y));
        }
    }
    if (in0) {
        const Haar4 h = butterfly(ll[0][0], ll[0][1], ll[1][0], ll[1][1]);
        sum += h.ll;
        y[0] = h.ll;
        y[sub] = h.lh;
        y[2 * sub] = h.hl;
        y[3 * sub] = h.hh;
    }
    if (in1) {
        const Haar4 h = butterfly(ll[0][2], ll[0][3], ll[1][2], ll[1][3]);
        sum += h.ll;
        y[1] = h.ll;
        y[1 + sub] = h.lh;
        y[1 + 2 * sub] = h.hl;
        y[1 + 3 * sub] = h.hh;
    }
    return sum;
}
// A thread keeps its plane and columns and walks down the rows i0, i0 + di, ... of blocks; p: floats from row to row of coefficients.
template <typename T, bool DIRECT>
__device__ __forceinline__ void analyse(int H, int H2, int p, int sub, const char *q, int row_bytes, float *y, bool in0, bool in1, int i0, int di) {
#pragma unroll 1
    for (int i = i0; i < H2; i += di, q += 4 * di * row_bytes, y += di * p) {
        uint4 w[4];
        load_blocks<DIRECT>(w, q, row_bytes, 4 * i, H);
        analyse_blocks<T>(w, y, sub, in0, in1);
    }
}
// Level l >= 3 of nb planes from the low-pass band above it (reads past an odd grid meet the zeros around it).  in, out: the first
// plane's grids, without their borders.
__device__ __forceinline__ void analyse_deeper(const float *in, int pp, float *out, int p, int sub, int dslot, const FastDiv &d_hw, const FastDiv &d_w, int nb, int tid) {
    const int Wl = (int)d_w.d, n = (int)d_hw.d;
    for (int e = tid; e < n * nb; e += DEEP) {
        const int s = fdiv(e, d_hw), r = e - s * n, i = fdiv(r, d_w), j = r - i * Wl;
        const float *q = in + s * dslot + 2 * i * pp + 2 * j;
        const float2 a = *reinterpret_cast<const float2 *>(q), b = *reinterpret_cast<const float2 *>(q + pp);
        const Haar4 h = butterfly(a.x, a.y, b.x, b.y);
        float *y = out + s * dslot + i * p + j;
        y[0] = h.ll;
        y[sub] = h.lh;
        y[2 * sub] = h.hl;
        y[3 * sub] = h.hh;
    }
}
// R of nb planes (Proposition 2 from level 2 down to the level-1 band): 2 x 4 values from two neighbouring coefficients; a thread
// keeps its plane and columns and walks down the rows.
__device__ __forceinline__ void synthesise(const PGeom &g, const float *dp, float *R, int slot0, int nb, int s, int j2, int i0, int di) {
    const int H2 = g.Hl[2], zp = g.zpitch[2], zs = H2 * zp;
    if (s >= nb) return;
    const float *D = dp + s * g.dslot, *z = D + g.offZ[2] + i0 * zp + 2 * j2;
    float *o = R + (slot0 + s) * g.rslot + 2 * i0 * g.rpitch + 4 * j2;
#pragma unroll 1
    for (int i = i0; i < H2; i += di, z += di * zp, o += 2 * di * g.rpitch) {
        const float2 ll = *reinterpret_cast<const float2 *>(z), lh = *reinterpret_cast<const float2 *>(z + zs);
        const float2 hl = *reinterpret_cast<const float2 *>(z + 2 * zs), hh = *reinterpret_cast<const float2 *>(z + 3 * zs);
        float deep0 = 0.f, deep1 = 0.f, scale = 0.5f;
#pragma unroll 1
        for (int l = 3; l <= g.L; ++l) {
            scale *= 0.5f;
            const int sl = g.Hl[l] * g.zpitch[l], j = j2 >> (l - 3), by = (i >> (l - 3)) & 1;
            const float *q = D + g.offZ[l] + (i >> (l - 2)) * g.zpitch[l] + j;
            const float a = q[0], b = q[sl], c = q[2 * sl], d = q[3 * sl];
            deep0 += synth_term(a, b, c, d, by, l == 3 ? 0 : (2 * j2 >> (l - 3)) & 1, scale);
            deep1 += synth_term(a, b, c, d, by, l == 3 ? 1 : (2 * j2 >> (l - 3)) & 1, scale);
        }
        const float p0 = ll.x + lh.x, m0 = ll.x - lh.x, q0 = hl.x + hh.x, n0 = hl.x - hh.x;
        const float p1 = ll.y + lh.y, m1 = ll.y - lh.y, q1 = hl.y + hh.y, n1 = hl.y - hh.y;
        *reinterpret_cast<float4 *>(o) = make_float4(fmaf(0.5f, p0 + q0, deep0), fmaf(0.5f, p0 - q0, deep0), fmaf(0.5f, p1 + q1, deep1), fmaf(0.5f, p1 - q1, deep1));
        *reinterpret_cast<float4 *>(o + g.rpitch) = make_float4(fmaf(0.5f, m0 + n0, deep0), fmaf(0.5f, m0 - n0, deep0), fmaf(0.5f, m1 + n1, deep1), fmaf(0.5f, m1 - n1, deep1));
    }
}

// A group's rows x cols pixels from each pixel's own taps alone, read from global memory: see tensor::group_by_taps.
template <typename T>
__device__ __noinline__ void pixels_by_taps(const T *__restrict__ plane, int H, int W, int y, int x0, const float *M, T *d, int K, float bias, const float *more) {
    const int pad = (5 - K) / 2;
#pragma unroll 1
    for (int i = 0; i < 16; ++i) {
        const int a = i >> 3, oc = i & 7, b = oc & 1;
        if (y + a >= H || x0 + oc >= W) continue;
        float sum = 0.f;
#pragma unroll 1
        for (int rq = 0; rq < 100; ++rq) {
            const int r = rq / 10, q = rq - r * 10, u = r - a - 2, v = q - b - 2, ul = r >> 1, vl = q >> 1, yy = y - 4 + r, xx = x0 - 4 + 2 * (oc >> 1) + q;
            const bool base = u >= pad && u < 5 - pad && v >= pad && v < 5 - pad;
            if (!base && !(ul >= pad && ul < 5 - pad && vl >= pad && vl < 5 - pad)) continue;
            const float p = (unsigned)yy < (unsigned)H && (unsigned)xx < (unsigned)W ? (float)plane[yy * W + xx] : 0.f;
            sum = fmaf(p, M[(a * 2 + b) * 100 + rq], sum);
            if (sum != sum) break;  // (a NaN stays one)
        }
        d[a * W + oc] = (T)fmaf(0.5f, more[oc >> 1], sum + bias);
    }
}

// ------------------------------------------------------------------ the parameters' gradients
struct Parameters {
    const float *w0, *s0, *b0, *wl, *sl;
};
// Where they go, and the partial sums they come from: slot i of a channel is the i-th block's whose units meet the channel's (see
// EpiloguePtrs); level l of partl is l * C * np * 4 * K * K floats on.
struct Gradients {
    float *w0, *s0, *b0, *wl, *sl;
    const float *part0, *partl;
    int np, upc, units, nblocks;
    float ratio;  // blocks to a unit
    const void *x;  // the layer's input
};
// block_of_unit without a 64-bit division, whose subroutine costs the kernel's other roles registers (8 spilled: 128 x 192 x 28 x 28
// 137 -> 146 us): a guess in fp32, one off at most, and the exact ranges.
__device__ __forceinline__ int block_near(const Gradients &d, int v) {
    const unsigned n = d.nblocks, whole = (unsigned)d.units / n, rest = (unsigned)d.units % n;
    auto begin = [&](unsigned b) { return (int)(b * whole + b * rest / n); };
    int b = (int)((float)v * d.ratio);
    if (b >= d.nblocks) b = d.nblocks - 1;
    while (b + 1 < d.nblocks && begin(b + 1) <= v) ++b;
    while (b > 0 && begin(b) > v) --b;
    return b;
}
// One class (0: base convolution, 1 .. 4: level 1) of a channel's weight gradients by a warp whose sums are not all finite.  The
// contraction multiplies the zeros around the planes (to whole groups of 16 rows and chunks of 8 columns) too, so that an infinity or
// NaN has reached taps that do not meet it.  Taps that do meet one inside the plane keep their sum (any product with it is not finite);
// the others are added again, every product on its own, from global memory.  x, go: the channel's planes of the first image; sum: tap
// `lane` of 5 x 5 (lanes < 25).  The search for what a tap meets ends when every tap has met something: with NaNs everywhere at once.
template <typename T>
__device__ __noinline__ double taps_of_class(const PGeom &g, const T *__restrict__ x, const T *__restrict__ go, int cls, int lane, double sum) {
    const int s = cls ? 1 : 0, h = (g.H + s) >> s, w = (g.W + s) >> s;
    const float sy = (cls - 1) & 1 ? -1.f : 1.f, sx = (cls - 1) & 2 ? -1.f : 1.f;
    const size_t image = (size_t)g.C * g.HW;
    auto at = [&](const T *q, int i, int j) {  // a pixel, or the class's coefficient (Eq. 5)
        auto pixel = [&](int y, int xx) { return y < g.H && xx < g.W ? (float)q[y * g.W + xx] : 0.f; };
        return cls ? 0.5f * ((pixel(2 * i, 2 * j) + sx * pixel(2 * i, 2 * j + 1)) + sy * (pixel(2 * i + 1, 2 * j) + sx * pixel(2 * i + 1, 2 * j + 1))) : pixel(i, j);
    };
    unsigned todo = __ballot_sync(0xffffffffu, lane < 25 && !(fabs(sum) < 1e300));
#pragma unroll 1
    for (int b = 0; b < g.B && todo; ++b) {
        const T *px = x + b * image, *pg = go + b * image;
        unsigned met = 0;
#pragma unroll 4
        for (int e = lane; e < h * w; e += 32) {
            const int i = e / w, j = e - i * w;
            const bool in_x = !(fabsf(at(px, i, j)) <= 3.4028235e38f), in_g = !(fabsf(at(pg, i, j)) <= 3.4028235e38f);
            if (in_x || in_g)
#pragma unroll 1
                for (int t = 0; t < 25; ++t) {  // the partner: grad_out's coefficient t off x's, x's off grad_out's
                    const int dy = t / 5 - 2, dx = t % 5 - 2;
                    if ((in_x && (unsigned)(i - dy) < (unsigned)h && (unsigned)(j - dx) < (unsigned)w) ||
                        (in_g && (unsigned)(i + dy) < (unsigned)h && (unsigned)(j + dx) < (unsigned)w))
                        met |= 1u << t;
                }
        }
        todo &= ~__reduce_or_sync(0xffffffffu, met);
    }
#pragma unroll 1
    while (todo) {
        const int t = __ffs(todo) - 1, dy = t / 5 - 2, dx = t % 5 - 2, i0 = dy < 0 ? -dy : 0, j0 = dx < 0 ? -dx : 0, hh = h - (dy < 0 ? -dy : dy), ww = w - (dx < 0 ? -dx : dx);
        todo &= todo - 1;
        double total = 0.0;
#pragma unroll 1
        for (int b = 0; b < g.B; ++b) {
            const T *px = x + b * image, *pg = go + b * image;
            float acc = 0.f;
            if (hh > 0 && ww > 0)
#pragma unroll 4
                for (int e = lane; e < hh * ww; e += 32) {
                    const int i = i0 + e / ww, j = j0 + e % ww;
                    acc = fmaf(at(pg, i, j), at(px, i + dy, j + dx), acc);
                }
#pragma unroll
            for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            total += (double)acc;
        }
        if (lane == t) sum = total;
    }
    return sum;
}
// What unfold_epilogue_kernel does, class by class, a warp each and a lane a tap (at most 25 and the bias): fixed-order fp64 sums and
// Eq. 9.  The loaders do it when they have loaded their last unit: it hides behind that unit's other stages, where a launch of its own
// took 4 - 5 us.
// Classes of base convolution and level 1 whose sums are not finite are computed again, see taps_of_class.
template <typename T>
__device__ __noinline__ void unfold_classes(const PGeom &g, const Parameters &p, const Gradients &d, const T *__restrict__ go, int warp, int warps, int lane) {
    const int KK = g.K * g.K, classes = 1 + 4 * g.L;
    for (int e = blockIdx.x * warps + warp; e < g.C * classes; e += gridDim.x * warps) {
        const int c = e / classes, cls = e - c * classes, l = (cls - 1) >> 2, sub = (cls - 1) & 3;
        const int n = block_near(d, (c + 1) * d.upc - 1) - block_near(d, c * d.upc) + 1;
        const float *q, *w, *s;
        float *to, *ts;
        int stride = 4 * KK, taps = KK;
        if (cls == 0) {
            stride = KK + 1;
            q = d.part0 + (size_t)c * d.np * stride;
            w = p.w0 + (size_t)c * KK;
            s = p.s0 + c;
            to = d.w0 + (size_t)c * KK;
            ts = d.s0 + c;
            if (p.b0) taps = KK + 1;
        } else {
            const size_t f = ((size_t)l * g.C + c) * 4 + sub;
            q = d.partl + (size_t)l * g.C * d.np * stride + ((size_t)c * d.np * 4 + sub) * KK;
            w = p.wl + f * KK;
            s = p.sl + f;
            to = d.wl + f * KK;
            ts = d.sl + f;
        }
        double prod = 0.0, acc = 0.0;
        if (lane < taps)
            for (int i = 0; i < n; ++i) acc += (double)q[(size_t)i * stride + lane];
        if (cls < 5 && __any_sync(0xffffffffu, lane < KK && !(fabs(acc) < 1e300))) {
            const size_t first = (size_t)c * g.HW;
            const int pad = (5 - g.K) / 2, u = lane / 5 - pad, v = lane % 5 - pad;  // (lanes are taps of 5 x 5 there)
            const bool in = lane < 25 && u >= 0 && u < g.K && v >= 0 && v < g.K;
            const double mine = __shfl_sync(0xffffffffu, acc, in ? u * g.K + v : 0);
            const double again = taps_of_class<T>(g, static_cast<const T *>(d.x) + first, go + first, cls, lane, in ? mine : 0.0);
            const double back = __shfl_sync(0xffffffffu, again, lane < KK ? (lane / g.K + pad) * 5 + lane % g.K + pad : 0);
            if (lane < KK) acc = back;
        }
        if (lane < taps) {
            const float wv = lane < KK ? __ldg(w + lane) : __ldg(p.b0 + c), sv = __ldg(s);
            *(lane < KK ? to + lane : d.b0 + c) = (float)((double)sv * acc);
            prod = acc * (double)wv;
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) prod += __shfl_xor_sync(0xffffffffu, prod, o);
        if (lane == 0) *ts = (float)prod;
    }
}

// ------------------------------------------------------------------ the kernel
// FLIP = false: out = WTConv(x).  FLIP = true: the same on grad_out with rotated kernels and no bias: grad_x, and the parameters'
// gradients from the sums of the kernel before.
template <typename T, bool FLIP, int LOAD, int KT>
__global__ void __launch_bounds__(OTHERS + LOAD, 1)
pyramid_kernel(const __grid_constant__ PGeom g, const T *__restrict__ x, const __grid_constant__ Parameters prm, const __grid_constant__ Gradients grad,
               T *__restrict__ out, int *__restrict__ status) {
    const float *__restrict__ w0 = prm.w0, *__restrict__ s0 = prm.s0, *__restrict__ b0 = prm.b0, *__restrict__ wl = prm.wl, *__restrict__ sl = prm.sl;
    constexpr int THREADS = OTHERS + LOAD;
    extern __shared__ __align__(128) char sb[];
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    float *mis = reinterpret_cast<float *>(sb + g.misc_off);  // two channels' worth
    u64 *acc_full = reinterpret_cast<u64 *>(mis + 2 * MIS), *acc_empty = acc_full + RING, *full = acc_empty + RING, *freed = full + MAX_BUFS,
        *r_full = freed + MAX_BUFS, *r_free = r_full + MAX_BUFS, *mma_done = r_free + MAX_BUFS, *set_free = mma_done + MAX_BUFS, *fin = set_free + 2;
    volatile int *dead = reinterpret_cast<volatile int *>(fin + 1);
    unsigned *tmem_slot = reinterpret_cast<unsigned *>(fin + 1) + 1;
    const int u_begin = (int)((long long)blockIdx.x * g.units / gridDim.x), u_end = (int)((long long)(blockIdx.x + 1) * g.units / gridDim.x);
    const unsigned limit = g.no_copy ? plane::WAIT_LIMIT_TEST : tensor::WAIT_LIMIT;
    {   // everything starts as zeros: halos, gaps, missing images
        uint4 *v = reinterpret_cast<uint4 *>(sb);
        for (int i = tid; i < g.table_off / 16; i += THREADS) v[i] = make_uint4(0u, 0u, 0u, 0u);
        plane::fence_async_smem();
    }
    if (tid == 0) {
        *dead = 0;
        for (int i = 0; i < RING; ++i) {
            plane::mbar_init(acc_full + i, 2);  // the MMAs, and the issuer for what it has seen of the loaders
            plane::mbar_init(acc_empty + i, 4);
        }
        for (int i = 0; i < MAX_BUFS; ++i) {
            plane::mbar_init(full + i, LOAD);
            plane::mbar_init(freed + i, DEEP / 32);
            plane::mbar_init(mma_done + i, ISS);
            plane::mbar_init(r_full + i, DEEP / 32);
            plane::mbar_init(r_free + i, EPI / 32);
        }
        for (int i = 0; i < 2; ++i) plane::mbar_init(set_free + i, EPI / 32);
        plane::mbar_init(fin, ISS);
    }
    __syncwarp();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(plane::smem_addr(tmem_slot)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const unsigned tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    auto wait_for = [&](u64 *bar, unsigned parity) {  // bounded; a wait that runs out is recorded and ends all waiting: what follows is garbage, but ends, and no role leaves the others' barriers
        if (!*dead && !plane::mbar_wait(bar, parity, limit)) {
            *dead = 1;
            raise_timeout(status, g.alarm, g.tag);
        }
    };
    dependents_may_start();  // (what follows is another kernel that fills the SMs, or the program's)
    wait_for_predecessor();  // shared and tensor memory only up to here
    if (blockIdx.x == 0 && tid == 0) status[STATUS_LAUNCH] = (int)g.tag;
    const int jobs = g.T * g.n;
    const unsigned rowb = (unsigned)g.Pc * CHUNK;
    // units take the operand arrays in turn; `phase` is the parity of an array's barriers
    auto next = [&](int &buf, unsigned &phase, int n) {
        if (++buf == n) { buf = 0; phase ^= 1u; }
    };
    if (warp < EPI / 32) {
        // ---------------------------------------------------------------- epilogue: a ring slot always belongs to the same four warps
        const int m = warp * 32 + lane, img = m & 7;
        int c = u_begin / g.upc, k = u_begin - c * g.upc, par = 0, buf = 0;
        unsigned job = 0, phase = 0;
        for (int u = u_begin; u < u_end; ++u, next(buf, phase, g.rbufs)) {
            wait_for(r_full + buf, phase);
            plane::bulk_store_wait_read();  // the output image may be written again behind the barrier
            named_sync(BAR_EPI, EPI);
            const float *mc = mis + par * MIS, *R = reinterpret_cast<const float *>(sb + g.r_off) + buf * g.r_floats;
            float scale = 1.f, bias = 0.f;  // the loaders' (the deep warps may be ahead of them: known once the unit's first MMAs are done)
            for (int t = 0; t < g.T; ++t) {
                const int row2 = 2 * (16 * t + (m >> 3)), o = fdiv(row2, g.d_period), y = row2 - o * g.period, slot = o * 8 + img, b = k * 8 * g.S + slot;
                const bool mine = o < g.S && y < g.H && b < g.B, second = y + 1 < g.H;
                const size_t first = ((size_t)b * g.C + c) * g.HW;
                const float *more = R + slot * g.rslot + (y >> 1) * g.rpitch;
                // the output image keeps the plane's place inside its 16-byte word of global memory
                T *d = reinterpret_cast<T *>(sb + g.out_off + slot * g.out_stride) + ((int)first & 7) + y * g.W;
                for (int j = 0, left = g.W; j < g.n; ++j, left -= 8, ++job) {
                    const unsigned s = job % RING;
                    wait_for(acc_full + s, (job / RING) & 1u);
                    __syncwarp();
                    fence_after();
                    if (t == 0 && j == 0) {
                        scale = mc[544];
                        bias = mc[545];
                    }
                    float a[16], p1[16], p2[16];
                    const unsigned addr = tmem + s * NCOL + ((unsigned)warp << 21);
                    tensor::tmem_ld16(addr, a);
                    tensor::tmem_ld16(addr + 16, p1);
                    tensor::tmem_ld16(addr + 32, p2);
                    tensor::tmem_ld_wait();
                    tensor::tmem_arrived(a);
                    tensor::tmem_arrived(p1);
                    tensor::tmem_arrived(p2);
                    fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(acc_empty + s);
                    if (!mine) continue;
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        if (std::is_same<T, __half>::value) a[i] = fmaf(scale, fmaf(p2[i], 1.f / 4194304.f, fmaf(p1[i], 1.f / 2048.f, a[i])), bias);
                        else a[i] = (a[i] + (p1[i] + p2[i])) + bias;
                    }
                    const bool spread = !(fabsf(a[0]) <= 3.4e38f);  // an infinity or NaN in the window: it is in every column then
                    const float4 r4 = *reinterpret_cast<const float4 *>(more + 4 * j);
                    const float rv[4] = {r4.x, r4.y, r4.z, r4.w};
#pragma unroll
                    for (int i = 0; i < 16; ++i) a[i] = fmaf(0.5f, rv[(i & 7) >> 1], a[i]);
                    tensor::store8<T>(d + 8 * j, a, left, g.W);
                    if (second) tensor::store8<T>(d + g.W + 8 * j, a + 8, left, g.W);
                    if (spread) pixels_by_taps<T>(x + first, g.H, g.W, y, 8 * j, mc + 128, d + 8 * j, g.K, bias, more + 4 * j);
                }
            }
            plane::fence_async_smem();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(r_free + buf);
                if (k + 1 == g.upc) mbar_arrive(set_free + par);  // the channel's last unit
            }
            named_sync(BAR_EPI, EPI);
            // ---- whole 16-byte words by one bulk copy a plane, the pixels before and behind them one by one (sixteen lanes a plane)
            for (int slot = warp * 2 + (lane >> 4); slot < 8 * g.S; slot += EPI / 16) {
                const int b = k * 8 * g.S + slot, i = lane & 15;
                if (b >= g.B) break;
                const size_t first = ((size_t)b * g.C + c) * g.HW;
                const int at = (int)(first & 7), lo = (8 - at) & 7, hi = ((at + g.HW) & ~7) - at;  // whole words: [lo, hi) of [0, HW)
                const T *s = reinterpret_cast<const T *>(sb + g.out_off + slot * g.out_stride) + at;
                if (i == 0 && hi > lo) plane::bulk_s2g(out + first + lo, s + lo, (unsigned)(hi - lo) * 2);
                const int e = i < 8 ? i : hi + (i - 8);
                if (i < 8 ? e < lo : e < g.HW) out[first + e] = s[e];
            }
            if (++k == g.upc) { k = 0; ++c; par ^= 1; }
        }
        plane::bulk_store_wait_read();  // shared memory must outlive the stores' reads
    } else if (warp < (EPI + DEEP) / 32) {
        // ---------------------------------------------------------------- levels >= 2
        const int dt = tid - EPI;
        float *dp = reinterpret_cast<float *>(sb + g.deep_off), *wtab = reinterpret_cast<float *>(sb + g.wtab_off);
        const Tile own = find_tile(g, dt);
        const int sub2 = g.rowsl[2] * g.pitch[2];
        // analysis: images fastest where they are neighbours in shared memory, columns where the rows come from global memory
        const int cols = g.direct ? g.W / 8 : g.Pc, combos = g.nb * cols, a_s = g.direct ? dt / cols % g.nb : dt % g.nb,
                  a_j = g.direct ? dt % cols : dt / g.nb % g.Pc, a_i = dt < DEEP / combos * combos ? dt / combos : g.Hl[2];
        const int pairs = (g.Wl[2] + 1) / 2, sets = g.nb * pairs, s_j = dt % pairs, s_s = dt / pairs % g.nb, s_i = dt < DEEP / sets * sets ? dt / sets : g.Hl[2];
        int c = u_begin / g.upc, k = u_begin - c * g.upc, c_prev = -1, buf = 0;
        int rbuf = 0;
        unsigned phase = 0, rphase = 0;
        for (int u = u_begin; u < u_end; ++u, next(buf, phase, g.bufs), next(rbuf, rphase, g.rbufs)) {
            if (c != c_prev) {  // (every tile of the unit before has been computed: a barrier lies between)
                const int KK = g.K * g.K, pad = (5 - g.K) / 2;
                for (int e = dt; e < (g.L - 1) * 100; e += DEEP) {  // Eq. 8
                    const int cls = e / 25, t = e - cls * 25, tt = FLIP ? 24 - t : t, uu = tt / 5 - pad, vv = tt % 5 - pad;
                    const size_t f = ((size_t)(1 + (cls >> 2)) * g.C + c) * 4 + (cls & 3);
                    const bool in = uu >= 0 && uu < g.K && vv >= 0 && vv < g.K;
                    wtab[cls * WS + t] = in ? __ldg(wl + f * KK + uu * g.K + vv) * __ldg(sl + f) : 0.f;
                }
                c_prev = c;
            }
            if (!g.direct) wait_for(full + buf, phase);
            wait_for(r_free + rbuf, rphase ^ 1u);
            float *R = reinterpret_cast<float *>(sb + g.r_off) + rbuf * g.r_floats;
#pragma unroll 1
            for (int slot0 = 0; slot0 < 8 * g.S; slot0 += g.nb) {
                const int nb = 8 * g.S - slot0 < g.nb ? 8 * g.S - slot0 : g.nb, total = nb * g.items;
                float *y = dp + a_s * g.dslot + g.offY[2] + (a_i + 2) * g.pitch[2] + 2 * a_j + 2;
                if (g.direct) {
                    const int b = k * 8 * g.S + slot0 + a_s;
                    if (a_s < nb && b < g.B)
                        analyse<T, true>(g.H, g.Hl[2], g.pitch[2], sub2, reinterpret_cast<const char *>(x + ((size_t)b * g.C + c) * g.HW + 4 * a_i * g.W + 8 * a_j), 2 * g.W, y, true,
                                         2 * a_j + 1 < g.Wl[2], a_i, DEEP / combos);
                } else {
                    const int slot = slot0 + a_s;  // (chunks start four columns to the left)
                    if (a_s < nb)
                        analyse<T, false>(g.H, g.Hl[2], g.pitch[2], sub2, sb + buf * g.a_bytes + ((slot >> 3) * g.period + 4 + 4 * a_i) * (int)rowb + a_j * CHUNK + (slot & 7) * 16, (int)rowb,
                                          y - 1, a_j > 0 && 2 * a_j - 1 < g.Wl[2], 2 * a_j < g.Wl[2], a_i, DEEP / combos);
                    __syncwarp();
                    if (lane == 0 && slot0 + nb == 8 * g.S) mbar_arrive(freed + buf);
                }
                named_sync(BAR_DEEP, DEEP);
#pragma unroll 1
                for (int l = 3; l <= g.L; ++l) {
                    analyse_deeper(dp + g.offY[l - 1] + 2 * g.pitch[l - 1] + 2, g.pitch[l - 1], dp + g.offY[l] + 2 * g.pitch[l] + 2, g.pitch[l],
                                   g.rowsl[l] * g.pitch[l], g.dslot, g.d_hw[l], g.d_w[l], nb, dt);
                    named_sync(BAR_DEEP, DEEP);
                }
#pragma unroll 1
                for (int it = dt; it < total; it += DEEP) run_tile<KT>(dp, wtab, it == dt ? own : find_tile(g, it));  // (one copy of the tile code)
                named_sync(BAR_DEEP, DEEP);
                synthesise(g, dp, R, slot0, nb, s_s, s_j, s_i, DEEP / sets);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(r_full + rbuf);
            if (++k == g.upc) { k = 0; ++c; }
        }
    } else if (warp < (EPI + DEEP) / 32 + ISS) {
        // ---------------------------------------------------------------- issuers: a ring slot always belongs to the same one
        const int iw = warp - (EPI + DEEP) / 32;
        const unsigned elected = tensor::elect_one();
        const u64 bdesc = smem_desc(plane::smem_addr(sb + g.table_off), (NCOL / 8) * 128, 128);
        constexpr unsigned id = tensor::instr_desc<T>(NCOL, false);
        int buf = 0;
        unsigned job0 = 0, phase = 0;
        for (int u = u_begin; u < u_end; ++u, job0 += jobs, next(buf, phase, g.bufs)) {
            wait_for(full + buf, phase);
            fence_after();
            const u64 adesc = smem_desc(plane::smem_addr(sb + buf * g.a_bytes), CHUNK, 2 * rowb);
            for (int q = (int)((iw - job0) & (ISS - 1)); q < jobs; q += ISS) {
                const int t = fdiv(q, g.d_n), j = q - t * g.n;
                const unsigned jc = job0 + q, s = jc % RING;
                wait_for(acc_empty + s, ((jc / RING) & 1u) ^ 1u);
                __syncwarp();
                fence_after();
                const u64 ad = adesc + (u64)((unsigned)(32 * t) * rowb + (unsigned)j * CHUNK >> 4);
                if (elected) {
#pragma unroll
                    for (int r = 0; r < TAPS; ++r) mma(tmem + s * NCOL, ad + (u64)((unsigned)r * (rowb >> 4)), bdesc + (u64)(r * (TAP_BYTES >> 4)), id, r > 0);
                    mma_commit(acc_full + s);
                    mbar_arrive(acc_full + s);
                }
                __syncwarp();
            }
            if (elected) mma_commit(mma_done + buf);
            __syncwarp();
        }
        if (elected) mma_commit(fin);  // nothing may be in flight when tensor and shared memory are given back
        __syncwarp();
        plane::mbar_wait(fin, 0, limit);
    } else {
        // ---------------------------------------------------------------- loaders
        const int lt = tid - (THREADS - LOAD), lw = lt >> 5;
        // A wait for a barrier's phase says something only if the phase before it is known to be over (the parity is all it sees), so
        // every barrier's phases are waited for in turn: `freed` and `mma_done` of an array each time it is loaded, mma_done of the
        // unit before's array, whose last phase was waited for when that unit was loaded, at a change of channel; set_free when a
        // set of M, scale and bias is written again, which is every second channel.
        int c = u_begin / g.upc, k = u_begin - c * g.upc, channels = 0, buf = 0;
        unsigned phase = 0;
        for (int u = u_begin; u < u_end; ++u, next(buf, phase, g.bufs)) {
            char *arr = sb + buf * g.a_bytes;
            const bool change = u == u_begin || k == 0;
            float wreg = 0.f, breg = 0.f;
            if (change) {
                wreg = lt < 125 ? tensor::folded_weight(g, c, lt, FLIP, w0, s0, wl, sl) : 0.f;
                if (lt == 0 && !FLIP && b0) breg = __ldg(s0 + c) * __ldg(b0 + c);
            }
            if (!g.direct) wait_for(freed + buf, phase ^ 1u);
            wait_for(mma_done + buf, phase ^ 1u);
            if (g.no_copy) break;  // test mode: nothing is copied and nobody is told
            if (u + 1 + g.direct < u_end) {  // (the deep warps are a unit ahead where they read global memory)
                int cp = c, kp = k + 1 + g.direct;
                while (kp >= g.upc) { kp -= g.upc; ++cp; }
                prefetch_planes<T, LOAD / 32>(g, x, cp, kp, lw, lane);
            }
            if (LOAD == FEW && g.vec == 4) copy_rows<4, LOAD / 32>(g, arr + 4 * rowb, g.Pc, 4, x, c, k, lw, lane);
            else if (LOAD == FEW) copy_rows<2, LOAD / 32>(g, arr + 4 * rowb, g.Pc, 4, x, c, k, lw, lane);
            else if (g.vec == 4) load_rows<T, 4, LOAD / 32>(g, arr, x, c, k, lw, lane);
            else if (g.vec == 2) load_rows<T, 2, LOAD / 32>(g, arr, x, c, k, lw, lane);
            else load_shifted<T, 4, LOAD / 32, false>(g, arr + 4 * rowb, g.Pc, x, c, k, lw, lane);
            if (LOAD == FEW) asm volatile("cp.async.wait_all;" ::: "memory");
            if (change) {  // the MMAs that read the old B operand have completed
                const int set = channels & 1;
                if (u > u_begin) wait_for(mma_done + (buf ? buf : g.bufs) - 1, buf ? phase : phase ^ 1u);
                if (channels > 1) wait_for(set_free + set, ((channels >> 1) - 1) & 1u);  // the epilogue has left the channel before the last
                ++channels;
                float *mc = mis + set * MIS;
                if (lt < 125) mc[lt] = wreg;
                if (lt == 0) mc[545] = breg;
                tensor::build_table<T, LOAD, BAR_LOAD>(sb + g.table_off, sb + g.parts_off, mc, lt);
            }
            if (++k == g.upc) { k = 0; ++c; }
            plane::fence_async_smem();
            mbar_arrive(full + buf);
        }
        __syncwarp();
        if (FLIP) unfold_classes<T>(g, prm, grad, x, lw, LOAD / 32, lane);
    }
    fence_before();
    __syncthreads();
    __syncwarp();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// ------------------------------------------------------------------ host side
struct Request {
    int B, C, H, W, L, K;
    bool operator==(const Request &o) const { return B == o.B && C == o.C && H == o.H && W == o.W && L == o.L && K == o.K; }
};

inline bool copied(const PGeom &g) { return g.vec > 1 && g.S * g.HW >= 1500; }
// Microseconds of a plan, by which the candidates and then the kernels of a layer are compared: MMA jobs, tiles (dearer where nothing
// overlaps them or the loaders take the registers), passes, blocks of the analysis, octets and shifted rows of each round of units, a B operand
// a channel.  Fitted to two plans each of 295 shapes between 2 x 24 x 4 x 4 and 128 x 800 x 110 x 64 (5 % off).  (A second set of
// constants had chosen the plan; where the two differ, on one shape in five, this one's choice is 1.8 % faster among the layers it is taken for.)
inline double estimate(const PGeom &g) {
    const int rounds = (g.units + g.nblocks - 1) / g.nblocks, changes = (rounds + g.upc - 1) / g.upc, passes = (8 * g.S + g.nb - 1) / g.nb;
    const int blocks = (g.nb * (g.direct ? g.n : g.Pc) * ((g.H + 3) / 4) + DEEP - 1) / DEEP;  // a deep thread's, of the analysis of one pass
    const double tile = (g.K == 3 ? 0.0182 : 0.0259) + (g.bufs == 1 && !g.direct ? 0.0388 : 0) + (copied(g) ? 0 : 0.0112), shift = g.vec == 1 ? 0.00138 : g.vec == 2 ? 0.00049 : 0;
    return 6.19 + rounds * (0.301 * g.T * g.n + (0.61 + tile * g.items + shift * g.HW) * g.S + (0.194 * (g.L + 1) + 0.146 * blocks) * passes) + 0.65 * changes;
}
inline bool search(const Request &q, PGeom &best, double &best_cost) {
    using tensor::up;
    if ((q.K != 3 && q.K != 5) || q.L < 2 || q.L > MAXL || q.H < 4 || q.W < 4 || q.W > 64 || q.H > 128) return false;
    PGeom g = {};
    g.B = q.B; g.C = q.C; g.H = q.H; g.W = q.W; g.HW = q.H * q.W; g.L = q.L; g.K = q.K;
    g.vec = q.W % 4 == 0 ? 4 : q.W % 2 == 0 ? 2 : 1;
    g.n = (q.W + 7) / 8;
    g.Pc = g.n + 1;
    const int th = up(q.H, 2);
    g.period = th + 4;
    g.Hl[0] = q.H; g.Wl[0] = q.W;
    for (int l = 1; l <= MAXL; ++l) { g.Hl[l] = (g.Hl[l - 1] + 1) / 2; g.Wl[l] = (g.Wl[l - 1] + 1) / 2; }
    int off = 0;
    for (int l = 2; l <= q.L; ++l) {
        g.tx[l] = (g.Wl[l] + 3) / 4;
        g.rowsl[l] = up(g.Hl[l], 4) + 4;
        g.pitch[l] = 4 * g.tx[l] + 4;
        g.zpitch[l] = 4 * g.tx[l];
        g.offY[l] = off; off += 4 * g.rowsl[l] * g.pitch[l];
        g.offZ[l] = off; off += 4 * g.Hl[l] * g.zpitch[l];
        const int ty = (g.Hl[l] + 3) / 4;
        g.first[l] = g.items; g.items += 4 * ty * g.tx[l];
        g.d_nt[l] = make_fastdiv(ty * g.tx[l]);
        g.d_tx[l] = make_fastdiv(g.tx[l]);
        g.d_hw[l] = make_fastdiv(g.Hl[l] * g.Wl[l]);
        g.d_w[l] = make_fastdiv(g.Wl[l]);
    }
    g.first[q.L + 1] = g.items;
    g.d_items = make_fastdiv(g.items);
    g.dslot = up(off, 32) + 4;  // eight planes' coefficients fall on different banks
    g.rpitch = up(2 * g.Wl[2], 4);  // (two coefficients are four values)
    if (g.rpitch < 4 * g.n) g.rpitch = 4 * g.n;
    g.rslot = up(2 * g.Hl[2] * g.rpitch, 32) + 4;  // eight images' rows fall on different banks
    g.d_period = make_fastdiv(g.period);
    g.d_n = make_fastdiv(g.n);
    g.out_stride = up(g.HW * 2 + 14, 128) + 16;  // eight images' rows fall on different banks
    bool found = false;
    bool ahead = false;
    for (int bufs : {4, 3, 2, 0, 1})  // 0: one operand array, levels >= 2 a unit ahead, from global memory (128 x 96 x 56 x 56: 125 us, otherwise 141)
        for (int S = 1; S <= 16; ++S) {
            if ((S > 1 && 8 * (S - 1) >= q.B) || (bufs == 1 && ahead)) break;
            for (int nb = 8 * S < 32 ? 8 * S : 32; nb >= 1; --nb) {
                PGeom h = g;
                h.direct = bufs == 0;
                h.bufs = bufs ? bufs : 1; h.rbufs = bufs ? bufs : 2; h.S = S; h.nb = nb;
                if ((h.direct && q.W % 8 != 0) || nb * (h.direct ? q.W / 8 : h.Pc) > DEEP || nb * ((h.Wl[2] + 1) / 2) > DEEP) continue;
                h.rows = (S - 1) * h.period + th + 8;
                h.T = ((S - 1) * h.period + th + 31) / 32;
                h.a_bytes = h.rows * h.Pc * CHUNK;
                h.r_floats = 8 * S * h.rslot;
                int o = h.bufs * h.a_bytes;
                h.r_off = o; o += h.rbufs * h.r_floats * 4;
                h.deep_off = o; o += up(h.nb * h.dslot * 4, 16);
                h.wtab_off = o; o += (q.L - 1) * 4 * WS * 4;
                h.parts_off = o; o += 5760;
                o = up(o, 128);
                h.table_off = o; o += TABLE_BYTES;
                // the last tile's MMAs read up to 32 T + 8 rows; those behind the array feed no output, but lie inside the block's memory
                const int reach = (h.bufs - 1) * h.a_bytes + (32 * h.T + 8) * h.Pc * CHUNK;
                h.out_off = o; o += 8 * S * h.out_stride;
                h.misc_off = o; o += 2 * MIS * 4 + (2 * RING + 5 * MAX_BUFS + 3) * 8 + 16;
                h.smem = up(o > reach ? o : reach, 128);
                if (h.smem > plane::SMEM_LIMIT) continue;
                h.upc = (q.B + 8 * S - 1) / (8 * S);
                if ((long long)h.upc * q.C > 0x3fffffffLL) continue;
                h.units = h.upc * q.C;
                h.nblocks = plane::NUM_SMS < h.units ? plane::NUM_SMS : h.units;
                const double cost = estimate(h);
                ahead = ahead || h.direct;
                if (!found || cost < best_cost) {
                    best = h;
                    best_cost = cost;
                    found = true;
                }
                break;  // (fewer planes at a time only cost barriers)
            }
        }
    return found;
}

// A plan is searched once and kept (bounded); `find(geom, cost)` searches.
template <typename G, typename F>
bool kept_plan(const Request &q, G &out, double &cost, F find) {
    struct Entry {
        Request q;
        bool ok;
        double cost;
        G g;
    };
    static std::mutex mu;
    static std::vector<Entry> cache;
    {
        std::lock_guard<std::mutex> lock(mu);
        for (const Entry &e : cache)
            if (e.q == q) {
                if (e.ok) { out = e.g; cost = e.cost; }
                return e.ok;
            }
    }
    Entry e = {};
    e.q = q;
    e.ok = find(e.g, e.cost);
    {
        std::lock_guard<std::mutex> lock(mu);
        if (cache.size() >= 256) cache.clear();
        cache.push_back(e);
    }
    if (e.ok) { out = e.g; cost = e.cost; }
    return e.ok;
}
inline bool plan(const Request &q, PGeom &out, double &cost) {
    return kept_plan(q, out, cost, [&](PGeom &g, double &c) { return search(q, g, c); });
}

template <typename T, bool FLIP, int LOAD, int KT>
cudaError_t launch(const PGeom &g, const T *x, const Parameters &p, const Gradients &grad, T *out, char *ws, cudaStream_t st) {
    constexpr auto kern = pyramid_kernel<T, FLIP, LOAD, KT>;
    const cudaError_t e = plane::opt_in_smem<kern>();
    if (e != cudaSuccess) return e;
    return launch_overlapped(kern, (unsigned)g.nblocks, (unsigned)(OTHERS + LOAD), (size_t)g.smem, st, g, x, p, grad, out, reinterpret_cast<int *>(ws));
}
template <typename T, bool FLIP>
cudaError_t run(const Request &q, const T *x, const Parameters &p, const Gradients &grad, T *out, char *ws, cudaStream_t st, unsigned tag, bool no_copy) {
    PGeom g;
    double cost;
    if (!plan(q, g, cost)) return cudaErrorInvalidValue;
    g.tag = tag;
    g.alarm = call_alarm;
    g.no_copy = no_copy;
    // Four warps that issue asynchronous copies (80 registers a thread; 72 with eight) are slower than eight that load through registers where
    // units are small: forward, 128 x 96 x 56 x 56 (3136 pixels an image and octet) 126 -> 121 us, 128 x 192 x 28 x 28 (1568) 68.2 -> 62.9;
    // 64 x 192 x 28 x 28 with four levels (784) 48.0 -> 49.3, 16 x 64 x 14 x 14 8.9 -> 9.5.  Nothing was measured between 784 and 1568.
    const bool copies = copied(g);
    if (q.K == 3) return copies ? launch<T, FLIP, FEW, 3>(g, x, p, grad, out, ws, st) : launch<T, FLIP, MANY, 3>(g, x, p, grad, out, ws, st);
    return copies ? launch<T, FLIP, FEW, 5>(g, x, p, grad, out, ws, st) : launch<T, FLIP, MANY, 5>(g, x, p, grad, out, ws, st);
}

inline int describe(const Request &q, char *buf, size_t n) {
    PGeom g;
    double cost;
    if (!plan(q, g, cost)) return 0;
    const int o = snprintf(buf, n, "[pyramid S=%d T=%d n=%d buffers=%d%s deep=%d planes, units=%d, smem=%d, cost=%.1f us]", g.S, g.T, g.n, g.bufs, g.direct ? " direct" : "", g.nb, g.units, g.smem, cost);
    return o < 0 ? 0 : o;
}

#define WT_PYRAMID_INSTANTIATE(T, EXTERN)                                                                                                                  \
    EXTERN template cudaError_t run<T, false>(const Request &, const T *, const Parameters &, const Gradients &, T *, char *, cudaStream_t, unsigned, bool); \
    EXTERN template cudaError_t run<T, true>(const Request &, const T *, const Parameters &, const Gradients &, T *, char *, cudaStream_t, unsigned, bool);

}  // namespace pyramid
}  // namespace wt
