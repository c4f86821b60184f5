// Weight gradients of 16-bit layers with two or more levels on whole planes (k = 3, 5): base convolution and level 1 as one contraction
// on tcgen05 (see tensor_kernels.cuh for the algebra and the short chains), levels >= 2 as fp32 FMA tiles, both from the same planes of
// x and grad_out in shared memory, by different warps of one block.  pyramid_kernel<T, true> makes grad_x and, from
// the sums of this one, the parameters' gradients.
//
// A unit is 8 S images of one channel.  The roles of a block's 22 warps, each a pipeline stage:
//   drain (4)      the chains' accumulators into running sums; a channel's sums into its partial slot
//   deep (12)      coefficients of x and grad_out from 4 x 4 pixels, deeper levels from the low-pass bands; a thread keeps the 25 taps of
//                  one class (level, subband) in registers over all units of a channel
//   issuers (2)    one half of the window each: an MMA of 128 x 64 x 16 per 16 rows x 8 columns x 8 images
//   loaders (4)    asynchronous copies of both tensors' rows into the operand layout (rows of an odd number of pixels are shifted in
//                  registers)
// Measured with grad_x, bf16, against the block-per-plane kernels: 128 x 96 x 56 x 56, three levels, 376 -> 240 us; 128 x 192 x 28 x 28,
// two levels, 229 -> 132; 64 x 192 x 28 x 28, four levels, 145 -> 95.  What bounds it now, by time stamps of the roles: where one pair
// of arrays fills an SM (56 x 56) a unit's copies (5300 of 18600 cycles, 16 a copy instruction), its two analyses (4400 and 2900) and
// the first batch's tiles (2700) follow one another; with several pairs (28 x 28) the deep warps' passes do (two of 4500 cycles).
// Relative error of the weight gradients against fp64 (2-norm; base, all levels; in brackets the block-per-plane kernels): 128 x 96 x 56 x 56
// bf16 1.6e-7, 2.0e-7 (3.3e-7, 5.7e-7), f16 2.1e-7, 2.3e-7 (6.5e-7, 5.8e-7); 128 x 192 x 28 x 28 bf16 1.4e-7, 1.5e-7 (2.4e-7, 4.3e-7),
// f16 2.0e-7, 2.0e-7 (4.9e-7, 4.5e-7); over 20 smaller shapes 0.8 - 2.1e-7 (0.9 - 3.5e-7), no entry off by more than 3.6e-7 of the largest.
// Eight loader warps instead of four left 72 registers a thread: 254 -> 272 us.  One launch for this and grad_x's kernel, block by
// block, 250 -> 264: the second's set-up is no longer hidden.
#pragma once
#include "pyramid_kernels.cuh"

namespace wt {
namespace pyramid {

constexpr int WDRAIN = 128, WISS = 2, WLOAD = 128, WTHREADS = WDRAIN + DEEP + 32 * WISS + WLOAD;
constexpr int CHAINS = 3, CHAIN_MMAS = 8;  // accumulator sets, additions to one before it is drained
constexpr int BAR_DRAIN = 6;
constexpr int FLUSH = DEEP + 1;            // floats from tap to tap of the flush: a thread's taps fall on different banks

struct WGeom {
    int B, C, H, W, HW, L, K;
    int S, period;                      // octets per unit, array rows from one octet to the next
    int n, Px, Ws;                      // chunks per row of grad_out and of x (which begins four columns and rows before the plane); groups of 16 rows
    int upc, units, bufs;
    int nb;                             // planes whose levels >= 2 are computed together
    int x_bytes, g_bytes;               // operand arrays
    int dslot;                          // floats of one plane's coefficients
    int Hl[MAXL + 1], Wl[MAXL + 1], tx[MAXL + 1], rowsl[MAXL + 1], pitch[MAXL + 1], offY[MAXL + 1];  // x, zero borders of two
    int rowsd[MAXL + 1], pitchd[MAXL + 1], offD[MAXL + 1], tiles[MAXL + 1];                          // grad_out, no borders
    int tpc[MAXL + 1], cls0[MAXL + 1];  // threads to a class of a level, the level's first thread
    int th;                             // rows of a tile: four, or two where that leaves most threads idle
    int turns;                          // tiles a thread
    int taps;                           // taps flushed at a time
    int deep_off, scr_off, misc_off, zero_end, smem;
    int nblocks, np, no_copy;
    FastDiv d_tx[MAXL + 1], d_nt[MAXL + 1], d_hw[MAXL + 1], d_w[MAXL + 1];
    int *alarm;
    unsigned tag;
};

template <int TH>
__device__ __forceinline__ void gradient_tile(const float *D, int pd, const float *Y, int p, float (&acc)[25]) {
    float d[TH][4];
#pragma unroll
    for (int i = 0; i < TH; ++i) {
        const float4 v = *reinterpret_cast<const float4 *>(D + i * pd);
        d[i][0] = v.x; d[i][1] = v.y; d[i][2] = v.z; d[i][3] = v.w;
    }
    plane::wgrad_taps<TH, 5>(Y, p, d, acc);
}

template <typename T>
__global__ void __launch_bounds__(WTHREADS, 1)
pyramid_gradient_kernel(const __grid_constant__ WGeom g, const T *__restrict__ x, const T *__restrict__ go, float *__restrict__ part0,
                        float *__restrict__ partl /* level l at (l - 1) * C * np * 4 * KK */, int *__restrict__ status) {
    extern __shared__ __align__(128) char sb[];
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    float *mis = reinterpret_cast<float *>(sb + g.misc_off);  // 400 entries of dM, 16 bias sums
    u64 *full = reinterpret_cast<u64 *>(mis + 416), *freed = full + MAX_BUFS, *chained = freed + MAX_BUFS, *drained = chained + CHAINS, *fin = drained + CHAINS;
    volatile int *dead = reinterpret_cast<volatile int *>(fin + 1);
    unsigned *tmem_slot = reinterpret_cast<unsigned *>(fin + 1) + 1;
    const int u_begin = (int)((long long)blockIdx.x * g.units / gridDim.x), u_end = (int)((long long)(blockIdx.x + 1) * g.units / gridDim.x);
    const unsigned limit = g.no_copy ? plane::WAIT_LIMIT_TEST : tensor::WAIT_LIMIT;
    {   // everything starts as zeros: halos, gaps, rows behind the planes
        uint4 *v = reinterpret_cast<uint4 *>(sb);
        for (int i = tid; i < g.zero_end / 16; i += WTHREADS) v[i] = make_uint4(0u, 0u, 0u, 0u);
        plane::fence_async_smem();
    }
    if (tid == 0) {
        *dead = 0;
        for (int i = 0; i < MAX_BUFS; ++i) {
            plane::mbar_init(full + i, WLOAD);
            plane::mbar_init(freed + i, WISS + DEEP / 32);
        }
        for (int i = 0; i < CHAINS; ++i) {
            plane::mbar_init(chained + i, WISS);
            plane::mbar_init(drained + i, WDRAIN / 32);
        }
        plane::mbar_init(fin, WISS);
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
    dependents_may_start();
    wait_for_predecessor();  // shared and tensor memory only up to here
    if (blockIdx.x == 0 && tid == 0) status[STATUS_LAUNCH] = (int)g.tag;
    auto next = [&](int &i, unsigned &phase, int n) {
        if (++i == n) { i = 0; phase ^= 1u; }
    };
    const int KK = g.K * g.K, pad = (5 - g.K) / 2;
    const int total = g.Ws * g.n, chains = (total + CHAIN_MMAS - 1) / CHAIN_MMAS, len = (total + chains - 1) / chains;  // a half's MMAs of a unit
    int c = u_begin / g.upc, k = u_begin - c * g.upc;
    auto slot_of = [&](int ch) { return (int)blockIdx.x - block_of_unit((long long)ch * g.upc, g.nblocks, g.units); };
    if (warp < WDRAIN / 32) {
        // ---------------------------------------------------------------- drain
        const unsigned lanes = (unsigned)warp << 21, sums = tmem + CHAINS * tensor::WG_ACC + lanes;
        float *scr = reinterpret_cast<float *>(sb + g.scr_off);
        int set = 0;
        unsigned phase = 0;
        bool first = true;
        for (int u = u_begin; u < u_end; ++u) {
            for (int e = 0; e < total; e += len, next(set, phase, CHAINS)) {
                wait_for(chained + set, phase);
                __syncwarp();
                fence_after();
                tensor::drain_gradients(tmem + set * tensor::WG_ACC + lanes, sums, lane, first);
                first = false;
                fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(drained + set);
            }
            const int cu = c;
            if (++k == g.upc) { k = 0; ++c; }
            if (u + 1 < u_end && c == cu) continue;
            // ---- the channel's sums: entries of equal offset added in a fixed order (dM), then the taps
            tensor::spill_gradients(sums, scr, 4 * warp + (lane >> 3), lane);
            first = true;
            named_sync(BAR_DRAIN, WDRAIN);
            for (int e = tid; e < 400; e += WDRAIN) {
                const int ab = e / 100, rq = e - ab * 100, r = rq / 10, q = rq - r * 10;
                float sum = 0.f;
#pragma unroll
                for (int gp = 0; gp < 4; ++gp) sum += scr[(((2 * gp + (ab >> 1)) * 2 + (ab & 1)) * 16 + r + 2 * gp) * 10 + q];
                mis[e] = sum;
            }
            named_sync(BAR_DRAIN, WDRAIN);
            const size_t slot = (size_t)cu * g.np + slot_of(cu);
            for (int e = tid; e < 5 * KK; e += WDRAIN) {
                const int cls = e / KK, t = e - cls * KK, uu = t / g.K + pad, vv = t % g.K + pad;
                float sum = 0.f;
                if (cls == 0) {
#pragma unroll
                    for (int ab = 0; ab < 4; ++ab) sum += mis[ab * 100 + ((ab >> 1) + 2 + uu) * 10 + (ab & 1) + 2 + vv];
                    part0[slot * (KK + 1) + t] = sum;
                } else {
#pragma unroll
                    for (int ab = 0; ab < 4; ++ab)
#pragma unroll
                        for (int pq = 0; pq < 4; ++pq)
                            sum += 0.25f * tensor::haar_sign(cls - 1, ab >> 1, ab & 1) * tensor::haar_sign(cls - 1, pq >> 1, pq & 1) *
                                   mis[ab * 100 + (2 * uu + (pq >> 1)) * 10 + 2 * vv + (pq & 1)];
                    partl[(slot * 4 + cls - 1) * KK + t] = sum;
                }
            }
            // (the next channel's spill and dM wait behind this unit's barriers: all of a warp's reads lie before its next drain's end)
            named_sync(BAR_DRAIN, WDRAIN);
        }
    } else if (warp < (WDRAIN + DEEP) / 32) {
        // ---------------------------------------------------------------- levels >= 2
        const int dt = tid - WDRAIN;
        float *dp = reinterpret_cast<float *>(sb + g.deep_off);
        // analysis: images fastest, neighbours in shared memory; a chunk of x and one of grad_out at a time
        const int comb = g.nb * g.Px, di = DEEP / comb, a_s = dt % g.nb, a_j = dt / g.nb % g.Px, a_i = dt < di * comb ? dt / comb : g.Hl[2];
        const bool x0 = a_j > 0 && 2 * a_j - 1 < g.Wl[2], x1 = 2 * a_j < g.Wl[2], g0 = a_j < g.n, g1 = g0 && 2 * a_j + 1 < g.Wl[2];  // (chunks of x start four columns to the left)
        const int subx = g.rowsl[2] * g.pitch[2], subg = g.rowsd[2] * g.pitchd[2], rowx = g.Px * CHUNK, rowg = g.n * CHUNK;
        float *yx0 = dp + a_s * g.dslot + g.offY[2] + (a_i + 2) * g.pitch[2] + 2 * a_j + 1, *yg0 = dp + a_s * g.dslot + g.offD[2] + a_i * g.pitchd[2] + 2 * a_j;
        // the thread's class and its tiles: it, it + tpc, ... of all planes' tiles of the level
        int l = 2;
        while (l < g.L && dt >= g.cls0[l + 1]) ++l;
        const bool busy = dt < g.cls0[l] + 4 * g.tpc[l];
        const int tpc = g.tpc[l], sub = (dt - g.cls0[l]) / tpc, it0 = dt - g.cls0[l] - sub * tpc, per = g.tiles[l];
        float acc[25], gsum = 0.f;
#pragma unroll
        for (int i = 0; i < 25; ++i) acc[i] = 0.f;
        int buf = 0;
        unsigned phase = 0;
        for (int u = u_begin; u < u_end; ++u, next(buf, phase, g.bufs)) {
            wait_for(full + buf, phase);
            const char *xa = sb + buf * (g.x_bytes + g.g_bytes), *ga = xa + g.x_bytes;
#pragma unroll 1
            for (int slot0 = 0; slot0 < 8 * g.S; slot0 += g.nb) {
                const int nb = 8 * g.S - slot0 < g.nb ? 8 * g.S - slot0 : g.nb;
                if (a_s < nb) {
                    const int slot = slot0 + a_s, row0 = (slot >> 3) * g.period + 4 * a_i, at = a_j * CHUNK + (slot & 7) * 16;
                    const char *qx = xa + (row0 + 4) * rowx + at, *qg = ga + row0 * rowg + at;
                    float *yx = yx0, *yg = yg0;
#pragma unroll 1
                    for (int i = a_i; i < g.Hl[2]; i += di, qx += 4 * di * rowx, qg += 4 * di * rowg, yx += di * g.pitch[2], yg += di * g.pitchd[2]) {
                        uint4 wx[4], wg[4];
                        load_blocks<false>(wx, qx, rowx, 0, 0);
                        if (g0) load_blocks<false>(wg, qg, rowg, 0, 0);
                        analyse_blocks<T>(wx, yx, subx, x0, x1);
                        if (g0) gsum += analyse_blocks<T>(wg, yg, subg, true, g1);
                    }
                }
                __syncwarp();
                if (lane == 0 && slot0 + nb == 8 * g.S) mbar_arrive(freed + buf);
                named_sync(BAR_DEEP, DEEP);
#pragma unroll 1
                for (int m = 3; m <= g.L; ++m) {
                    analyse_deeper(dp + g.offY[m - 1] + 2 * g.pitch[m - 1] + 2, g.pitch[m - 1], dp + g.offY[m] + 2 * g.pitch[m] + 2, g.pitch[m],
                                   g.rowsl[m] * g.pitch[m], g.dslot, g.d_hw[m], g.d_w[m], nb, dt);
                    analyse_deeper(dp + g.offD[m - 1], g.pitchd[m - 1], dp + g.offD[m], g.pitchd[m], g.rowsd[m] * g.pitchd[m], g.dslot, g.d_hw[m], g.d_w[m], nb, dt);
                    named_sync(BAR_DEEP, DEEP);
                }
                const int there = g.B - (k * 8 * g.S + slot0), live = there < 0 ? 0 : there < nb ? there : nb;  // images that do not exist come last
                const int tiles = busy ? live * per : 0;
#pragma unroll 1
                for (int it = it0; it < tiles; it += tpc) {
                    const int s = fdiv(it, g.d_nt[l]), r = it - s * per, ty = fdiv(r, g.d_tx[l]), tx = r - ty * g.tx[l];
                    const float *D = dp + s * g.dslot + g.offD[l] + (sub * g.rowsd[l] + g.th * ty) * g.pitchd[l] + 4 * tx;
                    const float *Y = dp + s * g.dslot + g.offY[l] + (sub * g.rowsl[l] + g.th * ty) * g.pitch[l] + 4 * tx;
                    if (g.th == 4) gradient_tile<4>(D, g.pitchd[l], Y, g.pitch[l], acc);
                    else gradient_tile<2>(D, g.pitchd[l], Y, g.pitch[l], acc);
                }
                named_sync(BAR_DEEP, DEEP);
            }
            const int cu = c;
            if (++k == g.upc) { k = 0; ++c; }
            if (u + 1 < u_end && c == cu) continue;
            // ---- the channel's sums: every thread's taps, a few at a time, to shared memory (the coefficients' place); a class's threads in order
            const size_t slot = (size_t)cu * g.np + slot_of(cu);
#pragma unroll 1
            for (int t0 = 0; t0 < 25; t0 += g.taps) {
#pragma unroll
                for (int i = 0; i < 25; ++i)
                    if (i >= t0 && i < t0 + g.taps) dp[(i - t0) * FLUSH + dt] = acc[i];
                named_sync(BAR_DEEP, DEEP);
                const int nt = 25 - t0 < g.taps ? 25 - t0 : g.taps;
                for (int e = dt; e < (g.L - 1) * 4 * nt; e += DEEP) {
                    const int cls = e / nt, i = e - cls * nt, t = t0 + i, m = 2 + (cls >> 2), uu = t / 5 - pad, vv = t % 5 - pad;
                    if (uu < 0 || uu >= g.K || vv < 0 || vv >= g.K) continue;
                    const float *q = dp + i * FLUSH + g.cls0[m] + (cls & 3) * g.tpc[m];
                    float s[4] = {0.f, 0.f, 0.f, 0.f};
                    int j = 0;
                    for (; j + 4 <= g.tpc[m]; j += 4) {
#pragma unroll
                        for (int h = 0; h < 4; ++h) s[h] += q[j + h];
                    }
                    for (; j < g.tpc[m]; ++j) s[0] += q[j];
                    partl[(size_t)(m - 1) * g.C * g.np * 4 * KK + (slot * 4 + (cls & 3)) * KK + uu * g.K + vv] = (s[0] + s[1]) + (s[2] + s[3]);
                }
                named_sync(BAR_DEEP, DEEP);
            }
#pragma unroll
            for (int i = 0; i < 25; ++i) acc[i] = 0.f;
#pragma unroll
            for (int o = 16; o; o >>= 1) gsum += __shfl_xor_sync(0xffffffffu, gsum, o);
            if (lane == 0) mis[400 + (dt >> 5)] = gsum;
            gsum = 0.f;
            for (int i = dt; i < g.taps * FLUSH / 4 + 1; i += DEEP) reinterpret_cast<float4 *>(dp)[i] = make_float4(0.f, 0.f, 0.f, 0.f);  // the borders
            named_sync(BAR_DEEP, DEEP);
            if (dt == 0) {
                float sum = 0.f;
                for (int i = 0; i < DEEP / 32; ++i) sum += mis[400 + i];
                part0[slot * (KK + 1) + KK] = 4.f * sum;  // (quarters: level-2 coefficients)
            }
        }
    } else if (warp < (WDRAIN + DEEP) / 32 + WISS) {
        // ---------------------------------------------------------------- issuers: a half of the window each (MMAs into one accumulator stay in order)
        const int half = warp - (WDRAIN + DEEP) / 32;
        const unsigned elected = tensor::elect_one();
        constexpr unsigned id = tensor::instr_desc<T>(64, true);
        const unsigned rowx = (unsigned)g.Px * CHUNK, rowg = (unsigned)g.n * CHUNK;
        int buf = 0, set = 0;
        unsigned phase = 0, sphase = 0;
        for (int u = u_begin; u < u_end; ++u, next(buf, phase, g.bufs)) {
            wait_for(full + buf, phase);
            __syncwarp();
            fence_after();
            const unsigned xa = plane::smem_addr(sb + buf * (g.x_bytes + g.g_bytes));
            const u64 xd = smem_desc(xa + half * CHUNK, 8 * rowx, rowx), gd = smem_desc(xa + g.x_bytes, 8 * rowg, rowg);
            int w = 0, j = 0;
            for (int e = 0; e < total; e += len, next(set, sphase, CHAINS)) {
                wait_for(drained + set, sphase ^ 1u);
                __syncwarp();
                fence_after();
                for (int i = 0; i < len && e + i < total; ++i) {
                    if (elected)
                        mma(tmem + set * tensor::WG_ACC + half * 64, xd + (u64)((unsigned)(16 * w) * rowx + (unsigned)j * CHUNK >> 4),
                            gd + (u64)((unsigned)(16 * w) * rowg + (unsigned)j * CHUNK >> 4), id, i > 0);
                    if (++j == g.n) { j = 0; ++w; }
                }
                if (elected) mma_commit(chained + set);
                __syncwarp();
            }
            if (elected) mma_commit(freed + buf);
            __syncwarp();
        }
        if (elected) mma_commit(fin);  // nothing may be in flight when tensor and shared memory are given back
        __syncwarp();
        plane::mbar_wait(fin, 0, limit);
    } else {
        // ---------------------------------------------------------------- loaders
        const int lw = warp - (WTHREADS - WLOAD) / 32;
        int buf = 0;
        unsigned phase = 0;
        for (int u = u_begin; u < u_end; ++u, next(buf, phase, g.bufs)) {
            if (u + 1 < u_end) {
                const int kp = k + 1 == g.upc ? 0 : k + 1, cp = k + 1 == g.upc ? c + 1 : c;
                prefetch_planes<T, WLOAD / 32>(g, x, cp, kp, lw, lane);
                prefetch_planes<T, WLOAD / 32>(g, go, cp, kp, lw, lane);
            }
            wait_for(freed + buf, phase ^ 1u);
            if (g.no_copy) break;  // test mode: nothing is copied and nobody is told
            char *xa = sb + buf * (g.x_bytes + g.g_bytes) + 4 * g.Px * CHUNK, *ga = sb + buf * (g.x_bytes + g.g_bytes) + g.x_bytes;
            if (g.W % 8 == 0) {
                copy_rows<8, WLOAD / 32>(g, ga, g.n, 0, go, c, k, lw, lane);
                copy_rows<4, WLOAD / 32>(g, xa, g.Px, 4, x, c, k, lw, lane);
            } else if (g.W % 4 == 0) {
                copy_rows<4, WLOAD / 32>(g, ga, g.n, 0, go, c, k, lw, lane);
                copy_rows<4, WLOAD / 32>(g, xa, g.Px, 4, x, c, k, lw, lane);
            } else if (g.W % 2 == 0) {
                copy_rows<2, WLOAD / 32>(g, ga, g.n, 0, go, c, k, lw, lane);
                copy_rows<2, WLOAD / 32>(g, xa, g.Px, 4, x, c, k, lw, lane);
            } else {
                load_shifted<T, 0, WLOAD / 32, true>(g, ga, g.n, go, c, k, lw, lane);
                load_shifted<T, 4, WLOAD / 32, true>(g, xa, g.Px, x, c, k, lw, lane);
            }
            asm volatile("cp.async.wait_all;" ::: "memory");
            plane::fence_async_smem();
            mbar_arrive(full + buf);
            if (++k == g.upc) { k = 0; ++c; }
        }
    }
    fence_before();
    __syncthreads();
    __syncwarp();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// ------------------------------------------------------------------ host side
inline int trips(const WGeom &g) { return g.W % 2 ? g.S * ((g.H + 7) / 8) * ((g.n + 3) / 4 + (g.Px + 3) / 4) : 0; }  // a loader's, of shifted rows
// Microseconds of a backward call, fitted to the same plans as the forward's (4 % off; its choice is as fast as the other constants' was).
inline double estimate(const WGeom &g, double grad_x) {
    const int rounds = (g.units + g.nblocks - 1) / g.nblocks, changes = (rounds + g.upc - 1) / g.upc, passes = (8 * g.S + g.nb - 1) / g.nb;
    const int blocks = (g.nb * g.Px * ((g.H + 3) / 4) + DEEP - 1) / DEEP;
    return 3.37 + 1.224 * grad_x + rounds * (0.536 + 0.315 * trips(g) + (0.404 + 0.00065 * g.HW) * g.S + passes * (0.579 + 0.257 * (g.L - 2) + 0.224 * blocks + 0.1395 * g.turns * g.th)) + 1.54 * changes;
}
inline bool search_gradient(const Request &q, WGeom &best, double &best_cost) {
    using tensor::up;
    if ((q.K != 3 && q.K != 5) || q.L < 2 || q.L > MAXL || q.H < 4 || q.W < 4 || q.W > 64 || q.H > 128) return false;
    WGeom g = {};
    g.B = q.B; g.C = q.C; g.H = q.H; g.W = q.W; g.HW = q.H * q.W; g.L = q.L; g.K = q.K;
    g.n = (q.W + 7) / 8;
    g.Px = g.n + 1;
    const int th = up(q.H, 2);
    g.period = th + 4;
    g.Hl[0] = q.H; g.Wl[0] = q.W;
    for (int l = 1; l <= MAXL; ++l) { g.Hl[l] = (g.Hl[l - 1] + 1) / 2; g.Wl[l] = (g.Wl[l - 1] + 1) / 2; }
    int off = 0;
    for (int l = 2; l <= q.L; ++l) {
        const int ty = (g.Hl[l] + 3) / 4;
        g.tx[l] = (g.Wl[l] + 3) / 4;
        g.rowsl[l] = 4 * ty + 4;
        g.pitch[l] = 4 * g.tx[l] + 4;
        g.rowsd[l] = 4 * ty;
        g.pitchd[l] = 4 * g.tx[l];
        g.offY[l] = off; off += 4 * g.rowsl[l] * g.pitch[l];
        g.offD[l] = off; off += 4 * g.rowsd[l] * g.pitchd[l];
        g.d_tx[l] = make_fastdiv(g.tx[l]);
        g.d_hw[l] = make_fastdiv(g.Hl[l] * g.Wl[l]);
        g.d_w[l] = make_fastdiv(g.Wl[l]);
    }
    g.dslot = up(off, 32) + 4;  // eight planes' coefficients fall on different banks
    bool found = false;
    for (int bufs : {4, 3, 2, 1})
        for (int S = 1; S <= 16; ++S) {
            if (S > 1 && (8 * (S - 1) >= q.B || bufs == 1)) break;  // (one pair of arrays: nothing hides a unit's copies, so units stay small)
            for (int nb = 8 * S < 32 ? 8 * S : 32; nb >= 1; --nb) {
                WGeom h = g;
                h.bufs = bufs; h.S = S; h.nb = nb;
                if (8 * S % nb != 0 || nb * h.Px > DEEP) continue;
                h.Ws = ((S - 1) * h.period + up(q.H, 4) + 15) / 16;  // (the analysis reads blocks of four rows)
                h.x_bytes = (16 * h.Ws + 8) * h.Px * CHUNK;
                h.g_bytes = 16 * h.Ws * h.n * CHUNK;
                int o = h.bufs * (h.x_bytes + h.g_bytes);
                h.deep_off = o; o += up(h.nb * h.dslot * 4 < 5 * FLUSH * 4 + 16 ? 5 * FLUSH * 4 + 16 : h.nb * h.dslot * 4, 16);
                h.taps = (o - h.deep_off - 16) / (FLUSH * 4);
                if (h.taps > 25) h.taps = 25;
                h.zero_end = o;
                h.scr_off = o; o += tensor::SCR_BYTES;
                h.misc_off = o; o += 416 * 4 + (2 * MAX_BUFS + 2 * CHAINS + 1) * 8 + 16;
                h.smem = up(o, 128);
                if (h.smem > plane::SMEM_LIMIT) continue;
                // threads to a class: as few tiles a thread as fit
                int all = 0;
                for (int l = 2; l <= q.L; ++l) all += 4 * nb * ((g.Hl[l] + 1) / 2) * g.tx[l];
                h.th = all <= DEEP ? 2 : 4;
                for (int l = 2; l <= q.L; ++l) {
                    h.tiles[l] = (g.Hl[l] + h.th - 1) / h.th * g.tx[l];
                    h.d_nt[l] = make_fastdiv(h.tiles[l]);
                }
                int turns = 1, used;
                for (;; ++turns) {
                    used = 0;
                    for (int l = 2; l <= q.L; ++l) {
                        h.tpc[l] = (nb * h.tiles[l] + turns - 1) / turns;
                        h.cls0[l] = used;
                        used += 4 * h.tpc[l];
                    }
                    if (used <= DEEP || turns >= 4096) break;
                }
                if (used > DEEP) continue;
                h.turns = turns;
                h.upc = (q.B + 8 * S - 1) / (8 * S);
                if ((long long)h.upc * q.C > 0x3fffffffLL) continue;
                h.units = h.upc * q.C;
                h.nblocks = plane::NUM_SMS < h.units ? plane::NUM_SMS : h.units;
                const double cost = estimate(h, 0.0);
                if (!found || cost < best_cost) {
                    best = h;
                    best_cost = cost;
                    found = true;
                }
                break;  // (fewer planes at a time only cost barriers)
            }
        }
    if (!found) return false;
    best.np = 1;
    for (int ch = 0; ch < best.C; ++ch) {
        const int n = block_of_unit((ch + 1LL) * best.upc - 1, best.nblocks, best.units) - block_of_unit((long long)ch * best.upc, best.nblocks, best.units) + 1;
        if (n > best.np) best.np = n;
    }
    return true;
}
inline bool plan_gradient(const Request &q, WGeom &out, double &cost) {
    return kept_plan(q, out, cost, [&](WGeom &g, double &c) {
        PGeom flip;
        double grad_x;
        if (!plan(q, flip, grad_x) || !search_gradient(q, g, c)) return false;
        c = estimate(g, grad_x);
        return true;
    });
}
inline size_t backward_bytes(const Request &q) {
    WGeom g;
    double cost;
    if (!plan_gradient(q, g, cost)) return 0;
    const size_t KK = (size_t)q.K * q.K;
    return plane::STATUS_BYTES + sizeof(float) * (size_t)g.C * g.np * (KK + 1 + 4 * KK * q.L);
}

// The sums of the weight gradients, then grad_x and the gradients of the parameters.
template <typename T>
cudaError_t backward(const Request &q, const T *x, const T *go, const Parameters &p, const Gradients &out, T *gx, char *ws, cudaStream_t st, unsigned tag, bool no_copy) {
    WGeom g;
    double cost;
    if (!plan_gradient(q, g, cost)) return cudaErrorInvalidValue;
    g.tag = tag;
    g.alarm = call_alarm;
    g.no_copy = no_copy;
    const size_t KK = (size_t)q.K * q.K;
    float *part0 = reinterpret_cast<float *>(ws + plane::STATUS_BYTES), *partl = part0 + (size_t)g.C * g.np * (KK + 1);
    constexpr auto kern = pyramid_gradient_kernel<T>;
    cudaError_t e;
    if ((e = plane::opt_in_smem<kern>()) != cudaSuccess) return e;
    if ((e = launch_overlapped(kern, (unsigned)g.nblocks, (unsigned)WTHREADS, (size_t)g.smem, st, g, x, go, part0, partl, reinterpret_cast<int *>(ws))) != cudaSuccess)
        return e;
    Gradients to = out;
    to.part0 = part0;
    to.partl = partl;
    to.np = g.np;
    to.upc = g.upc;
    to.units = g.units;
    to.nblocks = g.nblocks;
    to.ratio = (float)g.nblocks / (float)g.units;
    to.x = x;
    return run<T, true>(q, go, p, to, gx, ws, st, tag, no_copy);
}

inline int describe_backward(const Request &q, char *buf, size_t n) {
    WGeom g;
    double cost;
    if (!plan_gradient(q, g, cost)) return 0;
    const int o = snprintf(buf, n, "[pyramid gradients S=%d n=%d buffers=%d deep=%d planes, units=%d, np=%d, smem=%d, cost=%.1f us]", g.S, g.n, g.bufs, g.nb,
                           g.units, g.np, g.smem, cost);
    if (o < 0) return 0;
    return (size_t)o < n ? o + describe(q, buf + o, n - o) : o;
}

#define WT_GRADIENT_INSTANTIATE(T, EXTERN)                                                                                                    \
    EXTERN template cudaError_t backward<T>(const Request &, const T *, const T *, const Parameters &, const Gradients &, T *, char *, cudaStream_t, unsigned, bool);

}  // namespace pyramid
}  // namespace wt
