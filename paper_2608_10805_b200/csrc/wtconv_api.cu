// C ABI of the WTConv library: validation, workspace planning and kernel dispatch.
// Declarations and the full contract are in include/wtconv.h.  The kernels themselves are compiled in the
// per-dtype instantiation units (inst_*.cu); this unit only declares those instantiations.
#include "../../include/wtconv.h"

#include "common.cuh"
#include "tiled_kernels.cuh"
#include "plane_kernels.cuh"
#include "panel_host.cuh"
#include "pyramid_gradient.cuh"
#include "team_kernels.cuh"
#include "window_kernels.cuh"
#include "tiled_host.cuh"
#include "reference_chain.cuh"

#include <atomic>
#include <chrono>
#include <cstring>
#include <mutex>

namespace wt {
namespace plane {
WT_PLANE_INSTANTIATE(float, extern)
WT_PLANE_INSTANTIATE(__half, extern)
WT_PLANE_INSTANTIATE(__nv_bfloat16, extern)
}  // namespace plane
namespace tensor {
WT_TENSOR_INSTANTIATE(__half, extern)
WT_TENSOR_INSTANTIATE(__nv_bfloat16, extern)
WT_WIDE_INSTANTIATE(__half, extern)
WT_WIDE_INSTANTIATE(__nv_bfloat16, extern)
}  // namespace tensor
namespace pyramid {
WT_PYRAMID_INSTANTIATE(__half, extern)
WT_PYRAMID_INSTANTIATE(__nv_bfloat16, extern)
WT_GRADIENT_INSTANTIATE(__half, extern)
WT_GRADIENT_INSTANTIATE(__nv_bfloat16, extern)
}  // namespace pyramid
namespace team {
WT_TEAM_INSTANTIATE(float, extern)
WT_TEAM_INSTANTIATE(__half, extern)
WT_TEAM_INSTANTIATE(__nv_bfloat16, extern)
}  // namespace team
namespace window {
WT_WINDOW_INSTANTIATE(float, extern)
WT_WINDOW_INSTANTIATE(__half, extern)
WT_WINDOW_INSTANTIATE(__nv_bfloat16, extern)
}  // namespace window
namespace host {
WT_TILED_INSTANTIATE(float, 3, extern)
WT_TILED_INSTANTIATE(float, 5, extern)
WT_TILED_INSTANTIATE(float, 7, extern)
WT_TILED_INSTANTIATE(__half, 3, extern)
WT_TILED_INSTANTIATE(__half, 5, extern)
WT_TILED_INSTANTIATE(__half, 7, extern)
WT_TILED_INSTANTIATE(__nv_bfloat16, 3, extern)
WT_TILED_INSTANTIATE(__nv_bfloat16, 5, extern)
WT_TILED_INSTANTIATE(__nv_bfloat16, 7, extern)
}  // namespace host
namespace refchain {
WT_REFCHAIN_INSTANTIATE(float, 3, extern)
WT_REFCHAIN_INSTANTIATE(float, 5, extern)
WT_REFCHAIN_INSTANTIATE(float, 7, extern)
WT_REFCHAIN_INSTANTIATE(__half, 3, extern)
WT_REFCHAIN_INSTANTIATE(__half, 5, extern)
WT_REFCHAIN_INSTANTIATE(__half, 7, extern)
WT_REFCHAIN_INSTANTIATE(__nv_bfloat16, 3, extern)
WT_REFCHAIN_INSTANTIATE(__nv_bfloat16, 5, extern)
WT_REFCHAIN_INSTANTIATE(__nv_bfloat16, 7, extern)
}  // namespace refchain
}  // namespace wt

namespace {

using namespace wt::host;

wtconv_status validate_desc(const wtconv_desc *d) {
    if (!d) return WTCONV_ERR_NULL;
    if (d->B < 1 || d->C < 1 || d->H < 1 || d->W < 1) return WTCONV_ERR_SHAPE;
    if ((int64_t)d->B * d->C > 0x7fffffffLL || (int64_t)d->H * d->W > 0x3fffffffLL) return WTCONV_ERR_SHAPE;
    if (d->k != 3 && d->k != 5 && d->k != 7) return WTCONV_ERR_KERNEL_SIZE;
    if (d->L < 0 || d->L > WTCONV_MAX_LEVELS) return WTCONV_ERR_LEVELS;
    if (d->dtype != WTCONV_F32 && d->dtype != WTCONV_F16 && d->dtype != WTCONV_BF16) return WTCONV_ERR_DTYPE;
    return WTCONV_OK;
}

bool overlaps(const void *a, size_t na, const void *b, size_t nb) {
    const char *pa = (const char *)a, *pb = (const char *)b;
    return pa < pb + nb && pb < pa + na;
}

wtconv_status check_device() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return WTCONV_ERR_CUDA;
    int major = 0;
    if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess) return WTCONV_ERR_CUDA;
    return major == 10 ? WTCONV_OK : WTCONV_ERR_ARCH;
}

// ------------------------------------------------------------------ status tags
// Every call that launches kernels with bounded waits carries a fresh non-zero tag (see the status words in
// common.cuh).  The sequence starts at a clock-derived value, so that tags left in a workspace by another process or
// an earlier load of the library are unlikely to repeat.
unsigned next_status_tag() {
    static std::atomic<unsigned> counter{
        (unsigned)std::chrono::steady_clock::now().time_since_epoch().count() * 2654435761u};
    unsigned t = counter.fetch_add(1u, std::memory_order_relaxed) + 1u;
    if (t == 0u) t = counter.fetch_add(1u, std::memory_order_relaxed) + 1u;
    return t;
}

// 1 if the last call on this workspace recorded a timeout, else 0, into the third status word.
__global__ void resolve_status_kernel(int *status) {
    const int timeout = status[wt::STATUS_TIMEOUT], launch = status[wt::STATUS_LAUNCH];
    status[wt::STATUS_RESOLVED] = (launch != 0 && timeout == launch) ? 1 : 0;
}

// ------------------------------------------------------------------ dispatch
// Which kernels serve a descriptor, and the scratch they need.  The answers come from the planners (searches of a few
// thousand candidates behind process-wide caches of large plan structures), and one call asks many times over, so every
// thread keeps the last few descriptors' answers in a small direct-mapped table (a lookup is some 20 ns; asking the
// planners afresh cost a call of the smallest layer 3 us).
struct Route {
    wtconv_desc key;
    bool set;
    // The FMA family (plane: any that keeps whole planes on chip; k3: 3 x 3 kernels in 5 x 5 tables of that family), and where the
    // tensor cores are taken in its place: wide = column panels, both directions.
    // pyramid = the block-per-plane kernels of several levels with base convolution and level 1 on the tensor cores.
    bool team, plane, window, k3, wide, tensor[2], pyramid[2];
    size_t family_bytes[2];  // workspace, forward / backward, of the family
    size_t bytes[2];         // and of what is taken
};
const Route &route(const wtconv_desc *d);

int team_force_g(const wtconv_desc *d) { return (int)((d->flags >> 16) & 63u); }  // "planes per work unit" override
bool use_ref_chain(const wtconv_desc *d) { return (d->flags & WTCONV_FLAG_REFERENCE_CHAIN) != 0; }
bool use_team_path(const wtconv_desc *d) { return route(d).team; }
bool use_plane_path(const wtconv_desc *d) { return route(d).plane; }
bool use_window_path(const wtconv_desc *d) { return route(d).window; }
bool use_wide_path(const wtconv_desc *d) { return route(d).wide; }
bool use_tensor_path(const wtconv_desc *d, int bwd) { return route(d).tensor[bwd]; }
bool use_pyramid_path(const wtconv_desc *d, int bwd) { return route(d).pyramid[bwd]; }
wt::pyramid::Request pyramid_request(const wtconv_desc *d) { return {d->B, d->C, d->H, d->W, d->L, d->k}; }
wt::tensor::Request tensor_request(const wtconv_desc *d, int bwd) { return {bwd, d->B, d->C, d->H, d->W, d->L, d->k}; }
// k = 3 through the k = 5 kernels.  A 3 x 3 depthwise kernel is a 5 x 5 kernel with a border of zeros, so wherever the
// kernels that keep planes on chip (k = 5 only) serve the shape, the parameters are copied into 5 x 5 tables at the
// head of the workspace, the k = 5 path runs on them, and the backward copies the inner 3 x 3 of the 5 x 5 weight
// gradients out (the border's gradients are dropped; the scale and bias gradients are unaffected, since the border
// weights are zero).  16 of 25 taps multiply zeros, and it is still 2-3 x faster than the per-level kernels.
bool use_k3_embedding(const wtconv_desc *d) { return route(d).k3; }
wtconv_desc as_k5(const wtconv_desc *d) {
    wtconv_desc d5 = *d;
    d5.k = 5;
    return d5;
}
// Workspace head of the embedding: w0 [C][25], wl [L][C][4][25], then the same two for the gradients; the k = 5
// path's own workspace follows.
struct EmbedLayout {
    size_t w0, wl, gw0, gwl, inner;  // byte offsets
    size_t nf0, nfl;                 // filters in w0 / wl
};
EmbedLayout embed_layout(const wtconv_desc *d) {
    EmbedLayout e;
    e.nf0 = (size_t)d->C;
    e.nfl = (size_t)d->L * d->C * 4;
    e.w0 = 0;
    e.wl = align_up(e.w0 + e.nf0 * 25 * sizeof(float));
    e.gw0 = align_up(e.wl + e.nfl * 25 * sizeof(float));
    e.gwl = align_up(e.gw0 + e.nf0 * 25 * sizeof(float));
    e.inner = align_up(e.gwl + e.nfl * 25 * sizeof(float));
    return e;
}
// filters [nf0] of a and [nfl] of b, 3 x 3 -> 5 x 5 with a zero border
__global__ void embed_k3_kernel(const float *__restrict__ a, const float *__restrict__ b, float *__restrict__ ae,
                                float *__restrict__ be, size_t nf0, size_t nfl) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (nf0 + nfl) * 25) return;
    const size_t f = i / 25;
    const int t = (int)(i - f * 25), u = t / 5, v = t - u * 5;
    const bool inner = u >= 1 && u <= 3 && v >= 1 && v <= 3;
    const int t3 = (u - 1) * 3 + (v - 1);
    if (f < nf0) ae[f * 25 + t] = inner ? a[f * 9 + t3] : 0.f;
    else be[(f - nf0) * 25 + t] = inner ? b[(f - nf0) * 9 + t3] : 0.f;
}
// the inner 3 x 3 of 5 x 5 gradients
__global__ void extract_k3_kernel(const float *__restrict__ ae, const float *__restrict__ be, float *__restrict__ a,
                                  float *__restrict__ b, size_t nf0, size_t nfl) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (nf0 + nfl) * 9) return;
    const size_t f = i / 9;
    const int t = (int)(i - f * 9), u = t / 3 + 1, v = t - (t / 3) * 3 + 1;
    if (f < nf0) a[f * 9 + t] = ae[f * 25 + u * 5 + v];
    else b[(f - nf0) * 9 + t] = be[(f - nf0) * 25 + u * 5 + v];
}

// `family` (backward): leave the tensor cores out.  `taps` (k = 5 only): 3 when the tables hold 3 x 3 kernels with a zero border; the block-per-plane kernels then
// leave the border out of their loops, the other kernel families multiply through it.
template <typename T, int K>
wtconv_status forward_tk(const wtconv_desc *d, const void *x, const float *w0, const float *s0, const float *b0,
                         const float *wl, const float *sl, void *out, char *ws, cudaStream_t st, int taps = 5) {
    if (use_ref_chain(d)) return wt::refchain::forward<T, K>(d, (const T *)x, w0, s0, b0, wl, sl, (T *)out, ws, st);
    if constexpr (K != 7 && sizeof(T) == 2) {
        if (taps == 5 && use_wide_path(d))
            return wt::tensor::wide_forward<T>(tensor_request(d, 0), (const T *)x, w0, s0, b0, wl, sl, (T *)out, ws, st, next_status_tag()) == cudaSuccess
                       ? WTCONV_OK
                       : WTCONV_ERR_CUDA;
        if (taps == 5 && use_pyramid_path(d, 0))
            return wt::pyramid::run<T, false>(pyramid_request(d), (const T *)x, {w0, s0, b0, wl, sl}, {}, (T *)out,
                                              ws + (use_k3_embedding(d) ? embed_layout(d).inner : 0), st, next_status_tag(),
                                              (d->flags & WTCONV_FLAG_TEST_NO_COPY) != 0) == cudaSuccess
                       ? WTCONV_OK
                       : WTCONV_ERR_CUDA;
        if (taps == 5 && use_tensor_path(d, 0))
            return wt::tensor::forward<T>(tensor_request(d, 0), (const T *)x, w0, s0, b0, wl, sl, (T *)out,
                                          ws + (use_k3_embedding(d) ? embed_layout(d).inner : 0), st, next_status_tag(),
                                          (d->flags & WTCONV_FLAG_TEST_NO_COPY) != 0, nullptr) == cudaSuccess
                       ? WTCONV_OK
                       : WTCONV_ERR_CUDA;
    }
    if constexpr (K == 3) {
        if (use_k3_embedding(d)) {
            const wtconv_desc d5 = as_k5(d);
            const EmbedLayout e = embed_layout(d);
            float *w0e = (float *)(ws + e.w0), *wle = (float *)(ws + e.wl);
            const size_t n = (e.nf0 + e.nfl) * 25;
            embed_k3_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(w0, wl, w0e, wle, e.nf0, e.nfl);
            if (launch_status() != WTCONV_OK) return WTCONV_ERR_CUDA;
            return forward_tk<T, 5>(&d5, x, w0e, s0, b0, wle, sl, out, ws + e.inner, st, 3);
        }
    }
    if constexpr (K == 5) {
        if (use_team_path(d))
            return wt::team::forward<T>(d->B, d->C, d->H, d->W, d->L, (const T *)x, w0, s0, b0, wl, sl, (T *)out, ws, st,
                                        next_status_tag(), (d->flags & WTCONV_FLAG_TEST_NO_COPY) != 0,
                                        team_force_g(d)) == cudaSuccess
                       ? WTCONV_OK
                       : WTCONV_ERR_CUDA;
    }
    if constexpr (K == 5) {
        if (use_window_path(d))
            return wt::window::forward<T>(d->B, d->C, d->H, d->W, d->L, (const T *)x, w0, s0, b0, wl, sl, (T *)out, ws, st,
                                          next_status_tag()) == cudaSuccess
                       ? WTCONV_OK
                       : WTCONV_ERR_CUDA;
    }
    if (use_plane_path(d)) {
        if constexpr (K != 3)
            return wt::plane::forward<T>(d->B, d->C, d->H, d->W, d->L, (const T *)x, w0, s0, b0, wl, sl, (T *)out, ws,
                                         st, next_status_tag(), d->flags >> 8,
                                         (d->flags & WTCONV_FLAG_TEST_NO_COPY) != 0, K == 7 ? 7 : taps) == cudaSuccess
                       ? WTCONV_OK
                       : WTCONV_ERR_CUDA;
    }
    return tiled_forward<T, K>(d, (const T *)x, w0, s0, b0, wl, sl, (T *)out, ws, st);
}

template <typename T, int K>
wtconv_status backward_tk(const wtconv_desc *d, const void *x, const void *g, const float *w0, const float *s0,
                          const float *b0, const float *wl, const float *sl, void *gx, float *gw0, float *gs0,
                          float *gb0, float *gwl, float *gsl, char *ws, cudaStream_t st, bool family, int taps = 5) {
    if (use_ref_chain(d))
        return wt::refchain::backward<T, K>(d, (const T *)x, (const T *)g, w0, s0, b0, wl, sl, (T *)gx, gw0, gs0, gb0, gwl, gsl,
                                            ws, st);
    if constexpr (K != 7 && sizeof(T) == 2) {
        if (!family && use_wide_path(d)) {
            wt::EpiloguePtrs ep = {};
            if (wt::tensor::wide_backward<T>(tensor_request(d, 1), (const T *)x, (const T *)g, w0, s0, wl, sl, b0 != nullptr, (T *)gx, ws, &ep, st,
                                             next_status_tag()) != cudaSuccess)
                return WTCONV_ERR_CUDA;
            return launch_epilogue(d, ep, w0, s0, b0, wl, sl, gw0, gs0, gb0, gwl, gsl, st);
        }
        if (!family && use_tensor_path(d, 1)) {
            wt::EpiloguePtrs ep = {};
            if (wt::tensor::backward<T>(tensor_request(d, 1), (const T *)x, (const T *)g, w0, s0, wl, sl, b0 != nullptr, (T *)gx,
                                        ws + (use_k3_embedding(d) ? embed_layout(d).inner : 0), &ep, st, next_status_tag(),
                                        (d->flags & WTCONV_FLAG_TEST_NO_COPY) != 0, nullptr) != cudaSuccess)
                return WTCONV_ERR_CUDA;
            return launch_epilogue(d, ep, w0, s0, b0, wl, sl, gw0, gs0, gb0, gwl, gsl, st);
        }
        if (!family && use_pyramid_path(d, 1))
            return wt::pyramid::backward<T>(pyramid_request(d), (const T *)x, (const T *)g, {w0, s0, b0, wl, sl}, {gw0, gs0, gb0, gwl, gsl}, (T *)gx,
                                            ws + (use_k3_embedding(d) ? embed_layout(d).inner : 0), st, next_status_tag(),
                                            (d->flags & WTCONV_FLAG_TEST_NO_COPY) != 0) == cudaSuccess
                       ? WTCONV_OK
                       : WTCONV_ERR_CUDA;
    }
    if constexpr (K == 3) {
        if (use_k3_embedding(d)) {
            const wtconv_desc d5 = as_k5(d);
            const EmbedLayout e = embed_layout(d);
            float *w0e = (float *)(ws + e.w0), *wle = (float *)(ws + e.wl), *gw0e = (float *)(ws + e.gw0), *gwle = (float *)(ws + e.gwl);
            const size_t n = (e.nf0 + e.nfl) * 25, n3 = (e.nf0 + e.nfl) * 9;
            embed_k3_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(w0, wl, w0e, wle, e.nf0, e.nfl);
            if (launch_status() != WTCONV_OK) return WTCONV_ERR_CUDA;
            const wtconv_status st5 = backward_tk<T, 5>(&d5, x, g, w0e, s0, b0, wle, sl, gx, gw0e, gs0, gb0, gwle, gsl, ws + e.inner, st, true, 3);
            if (st5 != WTCONV_OK) return st5;
            extract_k3_kernel<<<(unsigned)((n3 + 255) / 256), 256, 0, st>>>(gw0e, gwle, gw0, gwl, e.nf0, e.nfl);
            return launch_status();
        }
    }
    if constexpr (K == 5) {
        if (use_team_path(d)) {
            wt::EpiloguePtrs ep = {};
            if (wt::team::backward<T>(d->B, d->C, d->H, d->W, d->L, (const T *)x, (const T *)g, w0, s0, wl, sl, (T *)gx,
                                      ws, &ep, st, next_status_tag(), (d->flags & WTCONV_FLAG_TEST_NO_COPY) != 0,
                                      team_force_g(d)) != cudaSuccess)
                return WTCONV_ERR_CUDA;
            return launch_epilogue(d, ep, w0, s0, b0, wl, sl, gw0, gs0, gb0, gwl, gsl, st);
        }
    }
    if constexpr (K == 5) {
        if (use_window_path(d)) {
            wt::EpiloguePtrs ep = {};
            if (wt::window::backward<T>(d->B, d->C, d->H, d->W, d->L, (const T *)x, (const T *)g, w0, s0, wl, sl, (T *)gx, ws, &ep,
                                        st, next_status_tag()) != cudaSuccess)
                return WTCONV_ERR_CUDA;
            return launch_epilogue(d, ep, w0, s0, b0, wl, sl, gw0, gs0, gb0, gwl, gsl, st);
        }
    }
    if (use_plane_path(d)) {
        if constexpr (K != 3) {
            wt::EpiloguePtrs ep = {};
            if (wt::plane::backward<T>(d->B, d->C, d->H, d->W, d->L, (const T *)x, (const T *)g, w0, s0, wl, sl,
                                       (T *)gx, ws, &ep, st, next_status_tag(), d->flags >> 8,
                                       (d->flags & WTCONV_FLAG_TEST_NO_COPY) != 0, K == 7 ? 7 : taps) != cudaSuccess)
                return WTCONV_ERR_CUDA;
            return launch_epilogue(d, ep, w0, s0, b0, wl, sl, gw0, gs0, gb0, gwl, gsl, st);
        }
    }
    return tiled_backward<T, K>(d, (const T *)x, (const T *)g, w0, s0, b0, wl, sl, (T *)gx, gw0, gs0, gb0, gwl, gsl,
                                ws, st);
}

#define WT_DISPATCH(FN, ...)                                                                   \
    do {                                                                                       \
        switch (d->dtype * 8 + d->k) {                                                         \
            case WTCONV_F32 * 8 + 3: return FN<float, 3>(__VA_ARGS__);                         \
            case WTCONV_F32 * 8 + 5: return FN<float, 5>(__VA_ARGS__);                         \
            case WTCONV_F32 * 8 + 7: return FN<float, 7>(__VA_ARGS__);                         \
            case WTCONV_F16 * 8 + 3: return FN<__half, 3>(__VA_ARGS__);                        \
            case WTCONV_F16 * 8 + 5: return FN<__half, 5>(__VA_ARGS__);                        \
            case WTCONV_F16 * 8 + 7: return FN<__half, 7>(__VA_ARGS__);                        \
            case WTCONV_BF16 * 8 + 3: return FN<__nv_bfloat16, 3>(__VA_ARGS__);                \
            case WTCONV_BF16 * 8 + 5: return FN<__nv_bfloat16, 5>(__VA_ARGS__);                \
            case WTCONV_BF16 * 8 + 7: return FN<__nv_bfloat16, 7>(__VA_ARGS__);                \
        }                                                                                      \
        return WTCONV_ERR_DTYPE;                                                               \
    } while (0)

size_t fwd_ws_bytes(const wtconv_desc *d) { return route(d).bytes[0]; }
size_t bwd_ws_bytes(const wtconv_desc *d) { return route(d).bytes[1]; }
// wtconv_backward_static: the family serves where only its workspace fits the built-in array
bool static_takes_family(const wtconv_desc *d) {
    const Route &r = route(d);
    return r.bytes[1] > (size_t)WTCONV_STATIC_SCRATCH_BYTES && r.family_bytes[1] <= (size_t)WTCONV_STATIC_SCRATCH_BYTES;
}
// 7 x 7 layers whose per-level kernels need more than the built-in array: the block-per-plane kernels need partial sums only.
wtconv_desc static_desc(const wtconv_desc *d) {
    wtconv_desc on_planes = *d;
    on_planes.flags |= WTCONV_FLAG_NO_TEAM;
    const bool takes = d->k == 7 && bwd_ws_bytes(d) > (size_t)WTCONV_STATIC_SCRATCH_BYTES && bwd_ws_bytes(&on_planes) <= (size_t)WTCONV_STATIC_SCRATCH_BYTES;
    return takes ? on_planes : *d;
}

// What the kernels that keep a plane on one SM (or a team of them) take for a 16-bit layer with at most one level, in
// microseconds: fitted to 3000 shapes between 1 x 16 x 7 x 7 and 128 x 768 x 64 x 64 (13 % off; k = 3 in 5 x 5 tables 11 %).
// They pay for tiles of 4 x 4 pixels, for planes, for rows that are not 8-byte multiples, and a fixed part that is larger
// where teams work on the smallest planes.
double on_chip_us(const wtconv_desc *d, int bwd) {
    const double planes = (double)d->B * d->C * 1e-3, tiles = planes * ((d->W + 3) / 4 * 4) * ((d->H + 3) / 4 * 4) * 1e-3;
    const int hw = d->H * d->W;
    const double first = planes < 1 ? planes : 1, kpx = hw * 1e-3;
    const bool odd = d->W % 4 != 0, small = hw <= 100, least = hw <= 64;
    if (d->k == 5)
        return bwd ? 10.4 + (7.33 + 3.1 * odd) * tiles + 0.48 * planes + 8.5 * small + 3.0 * first + 0.4 * kpx
                   : 6.6 + (3.16 + 1.56 * odd) * tiles + (0.355 - 0.25 * least) * planes + 2.5 * small;
    return bwd ? 17.2 + (4.61 + 2.87 * odd) * tiles + 0.82 * planes + 8.9 * small + 2.2 * first + 0.3 * kpx
               : 9.8 + (2.2 + 1.56 * odd) * tiles + (0.43 - 0.26 * least) * planes + 3.1 * small;
}
// The tensor-core kernels win where the images of a channel fill their groups of eight and there are enough channels and images
// for the SMs.  They are taken where their own estimate (4 - 6 % off) is at least a tenth below: over those shapes they gained
// 14 % (forward, k = 5), 25 % (backward), 27 % and 35 % (k = 3, which also saves the table kernels), and lost in 1 of 40.
// (A time model is refitted by timing random shapes with and without WTCONV_FLAG_NO_WINDOW, which keeps a layer on its family.)
bool tensor_serves(const wtconv_desc *d, bool on_chip, int bwd) {
    if (d->dtype == WTCONV_F32 || !on_chip || d->L > 1 || (d->flags & ~WTCONV_FLAG_TEST_NO_COPY)) return false;
    if (d->W > 64 && d->W % 4 != 0) return false;  // panels whose rows are not 8-byte multiples: element shifts, often slower
    wt::tensor::KGeom g;
    return wt::tensor::plan(tensor_request(d, bwd), g) && g.cost * (1.1 / 1900) < on_chip_us(d, bwd);
}

// Planes beyond the on-chip kernels: tensor-core panels against the per-level (tiled) kernels, which need rows of whole 16-byte
// words to be fast, and the window kernels, which take the others.  Measured over 3500 shapes between 60 x 60 and 256 x 256:
// against the tiled kernels panels win nearly everywhere (forward 1.5 x, backward 1.7 x; the exceptions are small 3 x 3 layers
// of several levels, all launches).  Against the windows the backward wins everywhere (1.4 x) and the forward where the
// launches of the levels do not count and the panels are well filled: both directions follow the forward's estimate, because a
// workspace keeps its status words in one place.  The estimates (microseconds, fitted, 10 % off) count pixels (n, millions),
// 64 x 64 pixel tiles (t1) and the 32 x 32 coefficient tiles of levels 2, 3 and deeper (t2, t3, t4).
bool panels_win(const wtconv_desc *d, double cost) {
    const double n = (double)d->B * d->C * d->H * d->W * 1e-6, planes = (double)d->B * d->C * 1e-3;
    if (d->W % 8 == 0) return d->k == 5 || d->L <= 1 || n >= 4;
    auto tiles = [&](int px, int side) { return planes * ((d->W + px - 1) / px) * ((d->H + px - 1) / px) * side * side * 1e-3; };
    const int L = d->L;
    const double t1 = tiles(64, 64), t2 = L > 1 ? tiles(128, 32) : 0, t3 = L > 2 ? tiles(256, 32) : 0, t4 = (L > 3 ? tiles(512, 32) : 0) + (L > 4) * planes;
    const bool odd = d->W % 4 != 0, deep = L > 1, deeper = L > 2;
    const double c = cost / 1900;
    if (d->k == 5)
        return 1.03 * ((1.35 + 0.08 * odd) * c + 2.86 * n * deep + 6.56 * t2 + 5.97 * t3 + 10.0 * t4 + 10.3 * deep + 1.7 * L) <
               8.9 + (5.13 + 0.6 * odd + 0.7 * deep + 0.69 * deeper) * n + (0.13 + 0.96 * deep) * t1 + 4.4 * t3 + 1.5 * t4 + 0.58 * L + 15.9 * deeper;
    return 1.1 * ((1.34 + 0.09 * odd) * c + 2.94 * n * deep + 3.36 * t2 + 1.78 * t3 + 9.0 * t4 + 11.9 * deep + 1.3 * L) <
           10.2 + (4.68 + 0.93 * odd + 0.58 * deep + 0.86 * deeper) * n + 1.16 * deep * t1 + 5.7 * t3 + 1.65 * L + 13.2 * deeper;
}
bool wide_serves(const wtconv_desc *d, bool on_chip) {
    if (d->dtype == WTCONV_F32 || on_chip || d->k == 7 || d->flags) return false;
    wt::tensor::KGeom g;
    return wt::tensor::wide(tensor_request(d, 0)) && wt::tensor::plan(tensor_request(d, 1), g) && wt::tensor::plan(tensor_request(d, 0), g) &&
           panels_win(d, g.cost);
}

// What the block-per-plane kernels take for a 16-bit layer of several levels, in microseconds, from their plan: rounds of units, a thread's
// tiles of a round, rows fetched pixel by pixel; fitted to 320 shapes (6 % off).
double plane_deep_us(const wtconv_desc *d, int bwd) {
    wt::plane::Geom g;
    const int eb = (int)elem_bytes(d->dtype);
    const bool split = bwd && !wt::plane::plan_bwd_fused(d->B, d->C, d->H, d->W, d->L, eb, g);
    if ((!bwd || split) && !(bwd ? wt::plane::plan_wgrad : wt::plane::plan_forward)(d->B, d->C, d->H, d->W, d->L, eb, g, 0, 5)) return 0;
    const double planes = (double)d->B * d->C * 1e-3, tiles = planes * ((d->W + 3) / 4 * 4) * ((d->H + 3) / 4 * 4) * 1e-3, first = planes < 1 ? planes : 1;
    const int rounds = (g.units + g.nblocks - 1) / g.nblocks, all = g.NPL * (g.lvl_start[d->L + 1] + g.nbase), more = d->L - 2;
    const double work = (double)((all + g.nthreads - 1) / g.nthreads) * g.th * g.blocks_per_sm, px = (double)g.NPL * d->H * d->W / g.nthreads;
    const bool odd = d->W % 4 != 0, k3 = d->k == 3;
    if (bwd)
        return 7.2 + 3.4 * k3 + 0.97 * more + (-0.72 - 1.97 * k3 + 1.65 * odd + 1.32 * (odd && !k3) + 0.25 * (more > 0) + 7.76 * split + 5.4 * (g.th == 8)) * tiles +
               (0.56 + 0.61 * more) * planes + 6.6 * first + 3.6 * split + rounds * (3.66 + 0.0476 * work + 0.09 * more + (g.bulk ? 0 : 0.137) * px - 0.0363 * g.blocks_per_sm * px);
    return 3.7 + 2.27 * k3 + 0.66 * more + (2.39 - 0.91 * k3 + 0.99 * odd + 0.17 * (odd && !k3) + 0.35 * (more > 0)) * tiles + (0.53 + 0.26 * more) * planes + 2.0 * first +
           rounds * (1.33 + 0.0154 * work + (g.bulk ? 0 : 0.083) * px);
}
// Several levels: taken where their estimate is 7 - 13 % below that of the block-per-plane kernels, 20 % where a block has fewer than three
// octets of images (its first loads are not hidden then: 16 x 192 x 28 x 28 is 1.15 x as fast in a loop of calls, but a host step on chunks of
// it, whose inputs have just arrived, is 1.5 - 3.6 % slower).  3 x 3 kernels: the block-per-plane estimate is 7 % low forward and 12 % low
// backward with rows of an odd number of pixel pairs (64 x 150 x 14 x 14, two levels: forward 20.4 us against 27.0, backward 42.8 against 49.9).
// Measured on 315 random shapes of 4 - 128 images: taken forward 194, 1.27 x as fast (geometric mean), backward 150, 1.31 x; four and two of them
// lose more than 2 %, the worst 32 x 234 x 13 x 13 (three levels, forward 0.91 x).
bool pyramid_serves(const wtconv_desc *d, bool on_chip, int bwd) {
    if (d->dtype == WTCONV_F32 || !on_chip || d->L < 2 || (d->flags & ~WTCONV_FLAG_TEST_NO_COPY)) return false;
    wt::pyramid::PGeom g;
    wt::pyramid::WGeom w;
    double cost;
    const bool few = (d->B + 7) / 8 * (long long)d->C < 3 * 148;
    if (bwd) return wt::pyramid::plan_gradient(pyramid_request(d), w, cost) && (few ? 1.2 : d->W % 2 ? 1.13 : d->k == 3 && d->W % 4 ? 0.92 : 1.1) * cost < plane_deep_us(d, 1);
    return wt::pyramid::plan(pyramid_request(d), g, cost) && (few ? 1.2 : d->k == 3 ? 0.95 : d->W % 4 ? 1.1 : 1.07) * cost < plane_deep_us(d, 0);
}

// 7 x 7 kernels on whole planes: block per plane, or the per-level kernels.  The latter win where planes are few (a block per plane
// leaves SMs empty, and its chain of stages is longer) and without levels on large 16-bit planes, where they only stream.  Both directions
// follow one answer, because a workspace keeps its status words in one place: the block-per-plane kernels are taken where both
// estimates (microseconds, fitted to 444 shapes of up to 74 x 74 with up to three levels, 9 - 14 % off) are a fifth below (without levels, forward: three
// tenths).  Of 484 measured shapes that takes 285, 3.3 x as fast (geometric mean of both directions), none slower in either.
bool seven_on_planes(const wtconv_desc *d) {
    wt::plane::Geom g;
    if (!wt::plane::supported(d->H, d->W, 7, d->L, d->dtype) ||
        !wt::plane::plan_forward(d->B, d->C, d->H, d->W, d->L, (int)elem_bytes(d->dtype), g, 0, 7))
        return false;
    if (d->flags & WTCONV_FLAG_NO_TEAM) return true;
    const double planes = (double)d->B * d->C * 1e-3, px = planes * d->H * d->W * 1e-3, tiles = planes * ((d->W + 3) / 4 * 4) * ((d->H + 3) / 4 * 4) * 1e-3;
    const double unit = 0.1 * g.NPL * d->H * d->W / g.nthreads, late = !g.bulk && d->W % 4 ? unit : 0;  // a thread's pixels of a unit; fetched one by one
    const bool odd = d->W % 4 != 0, unaligned = d->W * elem_bytes(d->dtype) % 16 != 0;
    if (d->L == 0) {
        if (d->dtype != WTCONV_F32 && d->H * d->W > 1500) return false;
        const double level[2] = {3.79 + (7.17 + 1.98 * unaligned) * planes + (2.35 + 0.63 * unaligned) * px,
                                 9.81 + (31.2 + 7.75 * unaligned) * planes + (3.72 + 1.68 * unaligned) * px};
        return 1.4 * (4.63 + 4.2 * tiles + 0.28 * planes + 1.33 * late + 1.05 * unit) < level[0] &&
               1.25 * (13.1 + (9.98 + 0.4 * odd) * tiles + 1.17 * planes + 2.5 * late + 2.7 * unit) < level[1];
    }
    double grids = 0, coefficients = 0;  // 32 x 32 tiles and coefficients of a plane's levels
    const double base = (d->H + 31) / 32 * ((d->W + 31) / 32);
    for (int l = 1, h = (d->H + 1) / 2, w = (d->W + 1) / 2; l <= d->L; ++l, h = (h + 1) / 2, w = (w + 1) / 2) {
        grids += 4.0 * ((h + 31) / 32) * ((w + 31) / 32);
        coefficients += 4.0 * h * w;
    }
    const double all = planes * (coefficients + d->H * d->W) * 1e-3;
    const double level[2] = {5.63 + 2.5 * d->L + planes * (3.83 * base + 2.84 * grids) + 0.72 * all,
                             11.5 + 5.0 * d->L + planes * (15.5 * base + 11.7 * grids) + 0.61 * all};
    return 1.25 * (6.88 + 0.55 * d->L + (6.56 + 1.46 * odd) * tiles + (0.38 + 0.4 * d->L) * planes + 0.89 * late - 0.38 * unit) < level[0] &&
           1.25 * (17.6 + 2.39 * d->L + (14.66 + 2.4 * odd) * tiles + (0.71 + 1.33 * d->L) * planes + 1.22 * late + 0.1 * unit) < level[1];
}

Route find_route(const wtconv_desc *d) {
    Route r = {};
    r.key = *d;
    r.set = true;
    const int eb = (int)elem_bytes(d->dtype);
    if (use_ref_chain(d)) {
        const auto p = wt::refchain::make_plan(d);
        r.bytes[0] = r.family_bytes[0] = p.fwd_bytes;
        r.bytes[1] = r.family_bytes[1] = p.bwd_bytes;
        return r;
    }
    Route r5 = {};
    if (!(d->flags & WTCONV_FLAG_TILED_ONLY)) {
        // launch-plan overrides other than the planes per unit address the block-per-plane kernels
        if (!(d->flags & WTCONV_FLAG_NO_TEAM) && !((d->flags >> 8) & ~(63u << 8)))
            r.team = wt::team::supported(d->B, d->C, d->H, d->W, d->k, d->L, d->dtype, team_force_g(d));
        // (7 x 7 kernels: launch-plan overrides leave them on the per-level kernels, which have no plan to override)
        r.plane = r.team || (d->k == 7 ? !(d->flags >> 8) && seven_on_planes(d) : wt::plane::supported(d->H, d->W, d->k, d->L, d->dtype));
        // Large planes (k = 5): windows with levels 1-2 on chip, deeper levels on the whole-plane kernels over a carrier.
        // Measured on B200: with 16-byte aligned rows the per-level tiled kernels are as fast or faster (they stream whole
        // rows), with unaligned rows (225-wide 16-bit planes) they fall to element loads and the window kernels win.
        if (!r.plane && !(d->flags & WTCONV_FLAG_NO_WINDOW) && !(d->flags >> 8) &&
            (((size_t)d->W * eb) % 16 != 0 || (d->flags & WTCONV_FLAG_PREFER_WINDOW)))
            r.window = wt::window::supported(d->B, d->C, d->H, d->W, d->k, d->L, d->dtype);
        if (d->k == 3) {
            const wtconv_desc d5 = as_k5(d);
            r5 = route(&d5);
            r.k3 = r5.plane || r5.window;
        }
    }
    if (r.k3) {
        for (int bwd = 0; bwd < 2; ++bwd) r.family_bytes[bwd] = embed_layout(d).inner + r5.family_bytes[bwd];
    } else if (r.team) {
        r.family_bytes[0] = align_up(wt::plane::STATUS_BYTES);
        r.family_bytes[1] = align_up(wt::team::backward_workspace_bytes(d->B, d->C, d->H, d->W, d->L, eb, team_force_g(d)));
    } else if (r.plane) {
        r.family_bytes[0] = align_up(wt::plane::forward_workspace_bytes(d->B, d->C, d->H, d->W, d->L));
        r.family_bytes[1] = align_up(wt::plane::backward_workspace_bytes(d->B, d->C, d->H, d->W, d->L, eb, d->flags >> 8, d->k));
    } else if (r.window) {
        const auto p = wt::window::ws_plan(d->B, d->C, d->H, d->W, d->L, eb);
        r.family_bytes[0] = align_up(p.fwd_bytes);
        r.family_bytes[1] = align_up(p.bwd_bytes);
    } else {
        const auto p = make_tiled_plan(d);
        r.family_bytes[0] = p.fwd_bytes;
        r.family_bytes[1] = p.bwd_bytes;
    }
    const bool on_chip = d->k == 3 ? r5.plane : r.plane;
    r.wide = wide_serves(d, on_chip);
    for (int bwd = 0; bwd < 2; ++bwd) {
        r.bytes[bwd] = r.family_bytes[bwd];
        if (r.wide) {
            const auto p = wt::tensor::wide_plan(tensor_request(d, 1), bwd != 0);
            r.bytes[bwd] = bwd ? p.bwd_bytes : p.fwd_bytes;
        } else if ((r.tensor[bwd] = d->k != 7 && tensor_serves(d, on_chip, bwd))) {
            // (behind the embedding's tables, where the family keeps its status words too)
            const size_t own = align_up(bwd ? wt::tensor::backward_bytes(tensor_request(d, 1)) : wt::tensor::STATUS_BYTES);
            r.bytes[bwd] = (r.k3 ? embed_layout(d).inner : 0) + own;
        } else if ((r.pyramid[bwd] = d->k != 7 && pyramid_serves(d, on_chip && !(r.k3 ? r5.team : r.team), bwd))) {
            r.bytes[bwd] = (r.k3 ? embed_layout(d).inner : 0) + align_up(bwd ? wt::pyramid::backward_bytes(pyramid_request(d)) : wt::plane::STATUS_BYTES);
        }
    }
    return r;
}
const Route &route(const wtconv_desc *d) {
    thread_local Route table[64];
    unsigned h = 2166136261u;
    const unsigned v[8] = {(unsigned)d->B, (unsigned)d->C, (unsigned)d->H, (unsigned)d->W, (unsigned)d->k, (unsigned)d->L, (unsigned)d->dtype, d->flags};
    for (unsigned x : v) h = (h ^ x) * 16777619u;
    Route &r = table[(h ^ (h >> 15)) & 63u];
    if (!r.set || memcmp(&r.key, d, sizeof *d) != 0) {
        const Route found = find_route(d);  // (may look another descriptor up on the way)
        r = found;
    }
    return r;
}

struct ParamSizes {
    size_t w0, s0, wl, sl;
};
ParamSizes param_sizes(const wtconv_desc *d) {
    size_t KK = (size_t)d->k * d->k, C = d->C, L = d->L;
    return {C * KK * 4, C * 4, L * C * 4 * KK * 4, L * C * 4 * 4};
}

// ------------------------------------------------------------------ allocation-free backward
// Scratch for wtconv_backward_static: lives in the library image, so every GPU that loads the library holds
// these bytes until the process exits.  Its name is only a host-side handle; the device address is looked
// up once per device with cudaGetSymbolAddress (see static_scratch_for_current_device).
static __device__ __align__(256) unsigned char wt_static_scratch[WTCONV_STATIC_SCRATCH_BYTES];

constexpr int MAX_DEVICES = 64;
std::mutex g_scratch_mutex;
void *g_scratch_ptr[MAX_DEVICES] = {};

// Device address of wt_static_scratch on the current device; resolved on the first call per device.
wtconv_status static_scratch_for_current_device(void **out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return WTCONV_ERR_CUDA;
    if (dev < 0 || dev >= MAX_DEVICES) return WTCONV_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_scratch_mutex);
    if (!g_scratch_ptr[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, wt_static_scratch) != cudaSuccess || !p) return WTCONV_ERR_CUDA;
        g_scratch_ptr[dev] = p;
    }
    *out = g_scratch_ptr[dev];
    return WTCONV_OK;
}

// wtconv_step_host splits the batch into chunks so that uploads, kernels and downloads of different chunks overlap.
constexpr int STEP_MAX_CHUNKS = 8;
int pick_step_chunks(const wtconv_desc *d) {
    const size_t per_image = (size_t)d->C * d->H * d->W * elem_bytes(d->dtype);
    for (int n = STEP_MAX_CHUNKS; n >= 2; n /= 2)
        if (d->B % n == 0 && d->B / n >= 4 && ((size_t)(d->B / n) * per_image) % 16 == 0 &&
            (size_t)(d->B / n) * per_image >= ((size_t)4 << 20))
            return n;
    return 1;
}
// dst[i] = sum over chunks of src[c * stride + i], in chunk order (deterministic).
__global__ void sum_chunks_kernel(float *__restrict__ dst, const float *__restrict__ src, size_t n, int nch, size_t stride) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float a = src[i];
    for (int c = 1; c < nch; ++c) a += src[(size_t)c * stride + i];
    dst[i] = a;
}

// Internal copy stream of wtconv_step_host, one per device, created on first use and kept for the process.
std::mutex g_side_mutex;
cudaStream_t g_side_stream[MAX_DEVICES][2] = {};  // [0] downloads, [1] uploads
wtconv_status side_stream_for_current_device(cudaStream_t *out, int which = 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) return WTCONV_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_side_mutex);
    if (!g_side_stream[dev][which] &&
        cudaStreamCreateWithFlags(&g_side_stream[dev][which], cudaStreamNonBlocking) != cudaSuccess)
        return WTCONV_ERR_CUDA;
    *out = g_side_stream[dev][which];
    return WTCONV_OK;
}

// Events of wtconv_step_host, per device, created on first use and kept for the process (calls on one device
// must not overlap in time, so they can share them; creating and destroying twenty events per call costs more
// host time than a small layer's kernels take).
constexpr int STEP_EVENTS = 2 * STEP_MAX_CHUNKS + 4;
cudaEvent_t g_step_events[MAX_DEVICES][STEP_EVENTS] = {};
wtconv_status step_events_for_current_device(cudaEvent_t **out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) return WTCONV_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_side_mutex);
    for (int i = 0; i < STEP_EVENTS; ++i)
        if (!g_step_events[dev][i] &&
            cudaEventCreateWithFlags(&g_step_events[dev][i], cudaEventDisableTiming) != cudaSuccess)
            return WTCONV_ERR_CUDA;
    *out = g_step_events[dev];
    return WTCONV_OK;
}

// ------------------------------------------------------------------ what the queries tell of a family
const char *family_name(const wtconv_desc *d) {
    if (use_k3_embedding(d)) {  // the kernels that run: the k = 5 path's
        const wtconv_desc d5 = as_k5(d);
        return family_name(&d5);
    }
    return use_ref_chain(d) ? "reference-chain" : use_team_path(d) ? "team" : use_plane_path(d) && d->k != 7 ? "plane" : use_window_path(d) ? "window" : "tiled";
}
void describe_family(const wtconv_desc *d, char *buf, size_t n) {
    if (use_k3_embedding(d)) {
        const wtconv_desc d5 = as_k5(d);
        const int o = snprintf(buf, n, "3x3 kernels in 5x5 tables: ");
        if (o > 0 && (size_t)o < n) describe_family(&d5, buf + o, n - o);
        return;
    }
    if (use_ref_chain(d))
        snprintf(buf, n, "reference-chain (separate operators, intermediates in HBM)%s%s",
                 (d->flags & WTCONV_FLAG_ABLATE_FUSED_ANALYSIS) ? " +fused-analysis" : "",
                 (d->flags & WTCONV_FLAG_ABLATE_COLLAPSED_SYNTHESIS) ? " +collapsed-synthesis" : "");
    else if (use_team_path(d))
        wt::team::describe(d->B, d->C, d->H, d->W, d->L, (int)elem_bytes(d->dtype), buf, n, team_force_g(d));
    else if (use_window_path(d)) {
        wt::window::WGeom wf, wb;
        wt::window::make_plan(d->B, d->C, d->H, d->W, d->L, (int)elem_bytes(d->dtype), false, wf);
        wt::window::make_plan(d->B, d->C, d->H, d->W, d->L, (int)elem_bytes(d->dtype), true, wb);
        snprintf(buf, n, "window fwd[%dx%d px, %d thr x %d/SM, buffers=%d, %s] bwd[%dx%d px, %d thr x %d/SM, buffers=%d, np=%d]%s",
                 wf.WH, wf.WW, wf.g.nthreads, wf.g.blocks_per_sm, wf.nbuf, wf.aligned ? "aligned rows" : "unaligned rows", wb.WH, wb.WW,
                 wb.g.nthreads, wb.g.blocks_per_sm, wb.nbuf, wb.g.np, d->L > 2 ? " + whole-plane kernels on the level-2 carrier" : "");
    } else if (use_plane_path(d))
        wt::plane::describe(d->B, d->C, d->H, d->W, d->L, (int)elem_bytes(d->dtype), d->flags >> 8, buf, n, d->k);
    else
        snprintf(buf, n, "tiled fwd[%d launches] bwd[%d launches]%s", d->L + 1, d->L + 2,
                 d->k == 7 && !(d->flags & WTCONV_FLAG_TILED_ONLY) && !(d->flags >> 8) && wt::plane::supported(d->H, d->W, 7, d->L, d->dtype)
                     ? " (faster here than the block-per-plane kernels)" : "");
}
void family_launches(const wtconv_desc *d, int (&n)[2]) {
    if (use_k3_embedding(d)) {  // the k = 5 path's launches + the table kernel (+ the gradient copy in the backward)
        const wtconv_desc d5 = as_k5(d);
        family_launches(&d5, n);
        n[0] += 1;
        n[1] += 2;
        return;
    }
    if (use_ref_chain(d)) {
        const bool fa = d->flags & WTCONV_FLAG_ABLATE_FUSED_ANALYSIS, cs = d->flags & WTCONV_FLAG_ABLATE_COLLAPSED_SYNTHESIS;
        const int nf = (fa ? 1 : 0) + d->L * (fa ? 2 : 3) + (d->L > 1 && !fa ? d->L - 1 : 0) + 2 + (cs ? 1 : 2 * d->L + 1);
        n[0] = nf;
        n[1] = (4 * d->L + 3) + 7 + 9 * d->L;  // plain forward chain + gradient launches (approximate for L > 1 slices)
    } else if (use_window_path(d)) {
        // window kernel (+ carrier, scale fill and the whole-plane kernel when L > 2); backward: + second carrier, epilogue
        n[0] = d->L > 2 ? 4 : 1;
        n[1] = d->L > 2 ? 7 : 2;
    } else if (use_team_path(d)) {
        n[0] = 1;
        n[1] = 2;  // fused backward + epilogue (and nothing else on the stream)
    } else if (use_plane_path(d)) {
        n[0] = 1;
        wt::plane::Geom gq;
        // fused backward + epilogue, or weight-gradient + input-gradient + epilogue (and nothing else on the stream)
        n[1] = wt::plane::plan_bwd_fused(d->B, d->C, d->H, d->W, d->L, (int)elem_bytes(d->dtype), gq, d->flags >> 8, d->k) ? 2 : 3;
    } else {
        n[0] = d->L + 1;
        n[1] = d->L + 2;
    }
}

wtconv_status checked_backward(const wtconv_desc *d, const void *x, const void *grad_out, const float *w0, const float *s0,
                               const float *b0, const float *wl, const float *sl, void *grad_x, float *grad_w0, float *grad_s0,
                               float *grad_b0, float *grad_wl, float *grad_sl, void *workspace, size_t workspace_bytes, void *stream,
                               bool family) {
    wtconv_status st = validate_desc(d);
    if (st != WTCONV_OK) return st;
    if (!x || !grad_out || !w0 || !s0 || !grad_x || !grad_w0 || !grad_s0) return WTCONV_ERR_NULL;
    if (d->L > 0 && (!wl || !sl || !grad_wl || !grad_sl)) return WTCONV_ERR_NULL;
    if ((b0 == nullptr) != (grad_b0 == nullptr)) return WTCONV_ERR_NULL;
    if (((uintptr_t)x | (uintptr_t)grad_out | (uintptr_t)grad_x) & 15) return WTCONV_ERR_ALIGNMENT;
    const size_t need = family ? route(d).family_bytes[1] : bwd_ws_bytes(d);
    if (!workspace || workspace_bytes < need) return WTCONV_ERR_WORKSPACE;
    if ((uintptr_t)workspace & (ALIGN - 1)) return WTCONV_ERR_ALIGNMENT;
    const size_t nbytes = (size_t)d->B * d->C * d->H * d->W * elem_bytes(d->dtype);
    if (overlaps(x, nbytes, grad_x, nbytes) || overlaps(grad_out, nbytes, grad_x, nbytes)) return WTCONV_ERR_ALIAS;
    if ((st = check_device()) != WTCONV_OK) return st;
    char *ws = (char *)workspace;
    cudaStream_t cs = (cudaStream_t)stream;
    WT_DISPATCH(backward_tk, d, x, grad_out, w0, s0, b0, wl, sl, grad_x, grad_w0, grad_s0, grad_b0, grad_wl, grad_sl,
                ws, cs, family);
}

}  // namespace

extern "C" {

const char *wtconv_status_string(wtconv_status st) {
    switch (st) {
        case WTCONV_OK: return "ok";
        case WTCONV_ERR_NULL: return "a required pointer is NULL";
        case WTCONV_ERR_SHAPE: return "invalid shape";
        case WTCONV_ERR_KERNEL_SIZE: return "kernel size must be 3, 5 or 7";
        case WTCONV_ERR_LEVELS: return "level count out of range";
        case WTCONV_ERR_DTYPE: return "unknown dtype";
        case WTCONV_ERR_ALIGNMENT: return "pointer not sufficiently aligned";
        case WTCONV_ERR_WORKSPACE: return "workspace missing or too small";
        case WTCONV_ERR_ALIAS: return "an output overlaps an input";
        case WTCONV_ERR_ARCH: return "device is not compute capability 10.x";
        case WTCONV_ERR_CUDA: return "CUDA runtime error";
        case WTCONV_ERR_TIMEOUT: return "device-side wait timed out";
    }
    return "unknown status";
}

wtconv_status wtconv_level_shape(const wtconv_desc *d, int level, int32_t *Hl, int32_t *Wl) {
    if (!d || !Hl || !Wl) return WTCONV_ERR_NULL;
    if (d->H < 1 || d->W < 1) return WTCONV_ERR_SHAPE;
    if (level < 0 || level > WTCONV_MAX_LEVELS) return WTCONV_ERR_LEVELS;
    Shapes s = level_shapes(d);
    *Hl = s.Hs[level];
    *Wl = s.Ws[level];
    return WTCONV_OK;
}

wtconv_status wtconv_workspace_bytes(const wtconv_desc *d, size_t *fwd_bytes, size_t *bwd_bytes) {
    wtconv_status st = validate_desc(d);
    if (st != WTCONV_OK) return st;
    if (fwd_bytes) *fwd_bytes = fwd_ws_bytes(d);
    if (bwd_bytes) *bwd_bytes = bwd_ws_bytes(d);
    return WTCONV_OK;
}

const char *wtconv_plan_name(const wtconv_desc *d) {
    if (validate_desc(d) != WTCONV_OK) return nullptr;
    if (use_wide_path(d)) return "panel";
    const bool f = use_tensor_path(d, 0), b = use_tensor_path(d, 1);
    if (f && b) return "tensor";
    if (!f && !b) return family_name(d);
    const bool team = strcmp(family_name(d), "team") == 0;  // (or plane: the tensor cores take no other family's place in one direction)
    return f ? (team ? "tensor/team" : "tensor/plane") : (team ? "team/tensor" : "plane/tensor");
}

wtconv_status wtconv_plan_describe(const wtconv_desc *d, char *buf, size_t n) {
    wtconv_status st = validate_desc(d);
    if (st != WTCONV_OK) return st;
    if (!buf || n == 0) return WTCONV_ERR_NULL;
    buf[0] = 0;
    const bool pyr[2] = {use_pyramid_path(d, 0), use_pyramid_path(d, 1)};
    const bool on[2] = {use_wide_path(d) || use_tensor_path(d, 0) || pyr[0], use_wide_path(d) || use_tensor_path(d, 1) || pyr[1]};
    if (!on[0] && !on[1]) {
        describe_family(d, buf, n);
        return WTCONV_OK;
    }
    size_t o = (size_t)snprintf(buf, n, "%s", wtconv_plan_name(d));
    for (int bwd = 0; bwd < 2; ++bwd)
        if (on[bwd] && o + 1 < n) {
            buf[o++] = ' ';
            buf[o] = 0;
            o += (size_t)snprintf(buf + o, n - o, "%s", pyr[bwd] ? (bwd ? "bwd" : "fwd") : "");
            if (o < n) o += (size_t)(pyr[bwd] ? (bwd ? wt::pyramid::describe_backward : wt::pyramid::describe)(pyramid_request(d), buf + o, n - o) : wt::tensor::describe(tensor_request(d, bwd), buf + o, n - o));
        }
    if ((!on[0] || !on[1]) && o < n) {
        o += (size_t)snprintf(buf + o, n - o, "; the other direction: ");
        if (o < n) describe_family(d, buf + o, n - o);
    }
    return WTCONV_OK;
}

wtconv_status wtconv_launch_count(const wtconv_desc *d, int32_t *fwd, int32_t *bwd) {
    wtconv_status st = validate_desc(d);
    if (st != WTCONV_OK) return st;
    int n[2];
    family_launches(d, n);
    for (int dir = 0; dir < 2; ++dir) {
        if (use_wide_path(d) && d->L > 1)  // band kernel(s), levels 2 .. L, synthesis, panels (+ epilogue)
            n[dir] = d->L + (dir ? 4 : 2);
        else if (use_wide_path(d) || use_tensor_path(d, dir))
            n[dir] = dir ? 2 : 1;
        else if (use_pyramid_path(d, dir))
            n[dir] = dir ? 2 : 1;
    }
    if (fwd) *fwd = n[0];
    if (bwd) *bwd = n[1];
    return WTCONV_OK;
}

wtconv_status wtconv_forward(const wtconv_desc *d, const void *x, const float *w0, const float *s0, const float *b0,
                             const float *wl, const float *sl, void *out, void *workspace, size_t workspace_bytes,
                             void *stream) {
    wtconv_status st = validate_desc(d);
    if (st != WTCONV_OK) return st;
    if (!x || !w0 || !s0 || !out || (d->L > 0 && (!wl || !sl))) return WTCONV_ERR_NULL;
    if (((uintptr_t)x | (uintptr_t)out) & 15) return WTCONV_ERR_ALIGNMENT;
    const size_t need = fwd_ws_bytes(d);
    if (need > 0 && (!workspace || workspace_bytes < need)) return WTCONV_ERR_WORKSPACE;
    if (need > 0 && ((uintptr_t)workspace & (ALIGN - 1))) return WTCONV_ERR_ALIGNMENT;
    const size_t nbytes = (size_t)d->B * d->C * d->H * d->W * elem_bytes(d->dtype);
    if (overlaps(x, nbytes, out, nbytes)) return WTCONV_ERR_ALIAS;
    if ((st = check_device()) != WTCONV_OK) return st;
    char *ws = (char *)workspace;
    cudaStream_t cs = (cudaStream_t)stream;
    WT_DISPATCH(forward_tk, d, x, w0, s0, b0, wl, sl, out, ws, cs);
}

wtconv_status wtconv_backward(const wtconv_desc *d, const void *x, const void *grad_out, const float *w0,
                              const float *s0, const float *b0, const float *wl, const float *sl, void *grad_x,
                              float *grad_w0, float *grad_s0, float *grad_b0, float *grad_wl, float *grad_sl,
                              void *workspace, size_t workspace_bytes, void *stream) {
    return checked_backward(d, x, grad_out, w0, s0, b0, wl, sl, grad_x, grad_w0, grad_s0, grad_b0, grad_wl, grad_sl, workspace,
                            workspace_bytes, stream, false);
}

// Device staging layout of wtconv_step_host: x, g, out, gx (activation dtype), then the
// parameters, then the parameter gradients, then the kernels' own workspace.
wtconv_status wtconv_step_host_workspace_bytes(const wtconv_desc *d, size_t *bytes) {
    wtconv_status st = validate_desc(d);
    if (st != WTCONV_OK) return st;
    if (!bytes) return WTCONV_ERR_NULL;
    const size_t act = align_up((size_t)d->B * d->C * d->H * d->W * elem_bytes(d->dtype));
    ParamSizes ps = param_sizes(d);
    const size_t par = align_up(ps.w0) + 2 * align_up(ps.s0) + align_up(ps.wl) + align_up(ps.sl);
    size_t f = fwd_ws_bytes(d), b = bwd_ws_bytes(d);
    size_t scratch = f > b ? f : b;
    const int nch = pick_step_chunks(d);
    if (nch > 1) {  // the pipelined step runs the kernels on B / nch images: their scratch need not be smaller
        wtconv_desc dc = *d;
        dc.B = d->B / nch;
        f = fwd_ws_bytes(&dc);
        b = bwd_ws_bytes(&dc);
        if (f > scratch) scratch = f;
        if (b > scratch) scratch = b;
    }
    // parameters, their gradients, and one more gradient set per batch chunk of the pipelined step
    *bytes = 4 * act + (2 + STEP_MAX_CHUNKS) * par + align_up(scratch);
    return WTCONV_OK;
}

wtconv_status wtconv_step_host(const wtconv_desc *d, const void *h_x, const void *h_g, const float *h_w0,
                               const float *h_s0, const float *h_b0, const float *h_wl, const float *h_sl, void *h_out,
                               void *h_gx, float *h_gw0, float *h_gs0, float *h_gb0, float *h_gwl, float *h_gsl,
                               void *workspace, size_t workspace_bytes, void *stream) {
    wtconv_status st = validate_desc(d);
    if (st != WTCONV_OK) return st;
    if (!h_x || !h_g || !h_w0 || !h_s0 || !h_out || !h_gx || !h_gw0 || !h_gs0) return WTCONV_ERR_NULL;
    if (d->L > 0 && (!h_wl || !h_sl || !h_gwl || !h_gsl)) return WTCONV_ERR_NULL;
    if ((h_b0 == nullptr) != (h_gb0 == nullptr)) return WTCONV_ERR_NULL;
    size_t need = 0;
    wtconv_step_host_workspace_bytes(d, &need);
    if (!workspace || workspace_bytes < need) return WTCONV_ERR_WORKSPACE;
    if ((uintptr_t)workspace & (ALIGN - 1)) return WTCONV_ERR_ALIGNMENT;
    cudaStream_t cs = (cudaStream_t)stream;
    const size_t act_raw = (size_t)d->B * d->C * d->H * d->W * elem_bytes(d->dtype), act = align_up(act_raw);
    ParamSizes ps = param_sizes(d);
    char *p = (char *)workspace;
    char *dx_ = p, *dg = p + act, *dout = p + 2 * act, *dgx = p + 3 * act;
    p += 4 * act;
    auto take = [&](size_t n) { char *q = p; p += align_up(n); return q; };
    float *w0 = (float *)take(ps.w0), *s0 = (float *)take(ps.s0), *b0 = (float *)take(ps.s0);
    float *wl = (float *)take(ps.wl), *sl = (float *)take(ps.sl);
    float *gw0 = (float *)take(ps.w0), *gs0 = (float *)take(ps.s0), *gb0 = (float *)take(ps.s0);
    float *gwl = (float *)take(ps.wl), *gsl = (float *)take(ps.sl);
    const size_t rest = workspace_bytes - (size_t)(p - (char *)workspace);
    bool ok = true;
    auto h2d = [&](void *dst, const void *src, size_t n) {
        if (n) ok = ok && cudaMemcpyAsync(dst, src, n, cudaMemcpyHostToDevice, cs) == cudaSuccess;
    };
    auto d2h = [&](void *dst, const void *src, size_t n) {
        if (n) ok = ok && cudaMemcpyAsync(dst, src, n, cudaMemcpyDeviceToHost, cs) == cudaSuccess;
    };
    // The forward needs only x: its result travels back on an internal stream while grad_out is still on its
    // way up (the link is full duplex), and `stream` waits for that copy before it reaches the end of the step.
    cudaStream_t side = nullptr;
    if ((st = side_stream_for_current_device(&side)) != WTCONV_OK) return st;
    cudaEvent_t *pool = nullptr;
    if ((st = step_events_for_current_device(&pool)) != WTCONV_OK) return st;
    cudaEvent_t fwd_done = pool[STEP_EVENTS - 2], out_home = pool[STEP_EVENTS - 1];
    const float *b0p = h_b0 ? b0 : nullptr;
    const int nch = pick_step_chunks(d);
    if (nch > 1) {
        // Pipelined step: chunk c's upload and kernels run on `stream`, its results travel back on the internal
        // stream while chunk c+1 is uploaded.  Every chunk leaves its own parameter gradients; they are added
        // in chunk order at the end.
        const size_t par_bytes = (size_t)((char *)gsl + align_up(ps.sl) - (char *)gw0);  // one gradient set
        char *chunk_grads = p;
        p += (size_t)STEP_MAX_CHUNKS * par_bytes;
        const size_t rest_c = workspace_bytes - (size_t)(p - (char *)workspace);
        wtconv_desc dc = *d;
        dc.B = d->B / nch;
        const size_t cb = act_raw / nch;
        h2d(w0, h_w0, ps.w0);
        h2d(s0, h_s0, ps.s0);
        if (h_b0) h2d(b0, h_b0, ps.s0);
        h2d(wl, h_wl, ps.wl);
        h2d(sl, h_sl, ps.sl);
        // events: [0..nch) chunk computed, [nch] downloads done, [nch+1] stream position at entry,
        // [nch+2 .. 2 nch+2) chunk uploaded
        cudaEvent_t *ev = pool;
        cudaStream_t up = nullptr;
        if (ok && side_stream_for_current_device(&up, 1) != WTCONV_OK) ok = false;
        if (!ok) return WTCONV_ERR_CUDA;
        // uploads run on their own stream (behind whatever `stream` holds at entry), so that chunk c+1 arrives
        // while chunk c is being computed
        ok = ok && cudaEventRecord(ev[nch + 1], cs) == cudaSuccess && cudaStreamWaitEvent(up, ev[nch + 1], 0) == cudaSuccess;
        for (int c = 0; c < nch && ok; ++c) {
            const size_t o = (size_t)c * cb;
            ok = ok && cudaMemcpyAsync(dx_ + o, (const char *)h_x + o, cb, cudaMemcpyHostToDevice, up) == cudaSuccess;
            ok = ok && cudaMemcpyAsync(dg + o, (const char *)h_g + o, cb, cudaMemcpyHostToDevice, up) == cudaSuccess;
            ok = ok && cudaEventRecord(ev[nch + 2 + c], up) == cudaSuccess;
        }
        if (!ok) {  // nothing of this step may outlive the caller's stream position
            if (cudaEventRecord(ev[nch], up) == cudaSuccess) cudaStreamWaitEvent(cs, ev[nch], 0);
            return WTCONV_ERR_CUDA;
        }
        for (int c = 0; c < nch; ++c) {
            const size_t o = (size_t)c * cb;
            ok = ok && cudaStreamWaitEvent(cs, ev[nch + 2 + c], 0) == cudaSuccess;
            if (!ok) break;
            char *gq = chunk_grads + (size_t)c * par_bytes;  // same layout as the final gradient set
            float *cgw0 = (float *)gq, *cgs0 = (float *)(gq + ((char *)gs0 - (char *)gw0)),
                  *cgb0 = (float *)(gq + ((char *)gb0 - (char *)gw0)), *cgwl = (float *)(gq + ((char *)gwl - (char *)gw0)),
                  *cgsl = (float *)(gq + ((char *)gsl - (char *)gw0));
            st = wtconv_forward(&dc, dx_ + o, w0, s0, b0p, wl, sl, dout + o, p, rest_c, stream);
            if (st == WTCONV_OK)
                st = wtconv_backward(&dc, dx_ + o, dg + o, w0, s0, b0p, wl, sl, dgx + o, cgw0, cgs0, h_b0 ? cgb0 : nullptr,
                                     cgwl, cgsl, p, rest_c, stream);
            if (st != WTCONV_OK) break;
            ok = ok && cudaEventRecord(ev[c], cs) == cudaSuccess;
            ok = ok && cudaStreamWaitEvent(side, ev[c], 0) == cudaSuccess;
            if (ok) ok = cudaMemcpyAsync((char *)h_out + o, dout + o, cb, cudaMemcpyDeviceToHost, side) == cudaSuccess;
            if (ok) ok = cudaMemcpyAsync((char *)h_gx + o, dgx + o, cb, cudaMemcpyDeviceToHost, side) == cudaSuccess;
        }
        // join first, so that `stream` ends after both internal streams whatever happened above (every upload
        // event has either been waited for by `stream` or precedes the last one, which is waited for here)
        bool joined = cudaStreamWaitEvent(cs, ev[nch + 2 + nch - 1], 0) == cudaSuccess &&
                      cudaEventRecord(ev[nch], side) == cudaSuccess && cudaStreamWaitEvent(cs, ev[nch], 0) == cudaSuccess;
        if (st != WTCONV_OK) return st;
        if (!ok || !joined) return WTCONV_ERR_CUDA;
        const size_t nfl = par_bytes / sizeof(float);
        sum_chunks_kernel<<<(unsigned)((nfl + 255) / 256), 256, 0, cs>>>(gw0, (const float *)chunk_grads, nfl, nch, nfl);
        if (launch_status() != WTCONV_OK) return WTCONV_ERR_CUDA;
        d2h(h_gw0, gw0, ps.w0);
        d2h(h_gs0, gs0, ps.s0);
        if (h_b0) d2h(h_gb0, gb0, ps.s0);
        d2h(h_gwl, gwl, ps.wl);
        d2h(h_gsl, gsl, ps.sl);
        return ok ? WTCONV_OK : WTCONV_ERR_CUDA;
    }
    h2d(dx_, h_x, act_raw);
    h2d(w0, h_w0, ps.w0);
    h2d(s0, h_s0, ps.s0);
    if (h_b0) h2d(b0, h_b0, ps.s0);
    h2d(wl, h_wl, ps.wl);
    h2d(sl, h_sl, ps.sl);
    if (!ok) return WTCONV_ERR_CUDA;
    st = wtconv_forward(d, dx_, w0, s0, b0p, wl, sl, dout, p, rest, stream);
    if (st != WTCONV_OK) return st;
    ok = ok && cudaEventRecord(fwd_done, cs) == cudaSuccess;
    ok = ok && cudaStreamWaitEvent(side, fwd_done, 0) == cudaSuccess;
    if (ok) ok = cudaMemcpyAsync(h_out, dout, act_raw, cudaMemcpyDeviceToHost, side) == cudaSuccess;
    ok = ok && cudaEventRecord(out_home, side) == cudaSuccess;
    h2d(dg, h_g, act_raw);
    if (!ok) return WTCONV_ERR_CUDA;
    st = wtconv_backward(d, dx_, dg, w0, s0, b0p, wl, sl, dgx, gw0, gs0, h_b0 ? gb0 : nullptr, gwl, gsl, p, rest,
                         stream);
    if (st != WTCONV_OK) {
        cudaStreamWaitEvent(cs, out_home, 0);
        return st;
    }
    d2h(h_gx, dgx, act_raw);
    d2h(h_gw0, gw0, ps.w0);
    d2h(h_gs0, gs0, ps.s0);
    if (h_b0) d2h(h_gb0, gb0, ps.s0);
    d2h(h_gwl, gwl, ps.wl);
    d2h(h_gsl, gsl, ps.sl);
    ok = ok && cudaStreamWaitEvent(cs, out_home, 0) == cudaSuccess;  // join: the step ends when `out` is home too
    return ok ? WTCONV_OK : WTCONV_ERR_CUDA;
}

wtconv_status wtconv_set_alarm(int32_t *h_alarm) {
    wt::call_alarm = h_alarm;
    return WTCONV_OK;
}

wtconv_status wtconv_get_alarm(int32_t **h_alarm) {
    if (!h_alarm) return WTCONV_ERR_NULL;
    *h_alarm = wt::call_alarm;
    return WTCONV_OK;
}

wtconv_status wtconv_read_status(const wtconv_desc *d, void *workspace, int32_t *h_flag, void *stream) {
    wtconv_status st = validate_desc(d);
    if (st != WTCONV_OK) return st;
    if (!h_flag) return WTCONV_ERR_NULL;
    bool wide = use_wide_path(d);
    wtconv_desc in_scratch;
    if (!workspace) {  // the scratch array built into the library (wtconv_backward_static)
        void *scratch = nullptr;
        if ((st = check_device()) != WTCONV_OK) return st;
        if ((st = static_scratch_for_current_device(&scratch)) != WTCONV_OK) return st;
        workspace = scratch;
        in_scratch = static_desc(d);
        d = &in_scratch;
        wide = wide && !static_takes_family(d);
    }
    if ((uintptr_t)workspace & (ALIGN - 1)) return WTCONV_ERR_ALIGNMENT;
    if (!wide) {  // column panels: the status words open the workspace
        wtconv_desc d5;
        if (use_k3_embedding(d)) {  // the status words belong to the k = 5 path, behind the parameter tables
            workspace = (char *)workspace + embed_layout(d).inner;
            d5 = as_k5(d);
            d = &d5;
        }
        if (use_window_path(d) && d->L > 2)  // the carrier's whole-plane kernels keep the only status word of this path
            workspace = (char *)workspace + wt::window::ws_plan(d->B, d->C, d->H, d->W, d->L, (int)elem_bytes(d->dtype)).deep;
        else if (!use_plane_path(d)) {  // the tiled, window (L <= 2) and reference kernels wait for nothing and keep no status word
            *h_flag = 0;
            return WTCONV_OK;
        }
    }
    // the status words open every workspace the plane kernels use: compare the timeout tag with the tag of the
    // last launch on the device, then fetch the result
    int *words = (int *)workspace;
    resolve_status_kernel<<<1, 1, 0, (cudaStream_t)stream>>>(words);
    if (launch_status() != WTCONV_OK) return WTCONV_ERR_CUDA;
    return cudaMemcpyAsync(h_flag, words + wt::STATUS_RESOLVED, sizeof(int32_t), cudaMemcpyDeviceToHost,
                           (cudaStream_t)stream) == cudaSuccess
               ? WTCONV_OK
               : WTCONV_ERR_CUDA;
}

wtconv_status wtconv_backward_static(const wtconv_desc *d, const void *x, const void *grad_out, const float *w0,
                                     const float *s0, const float *b0, const float *wl, const float *sl, void *grad_x,
                                     float *grad_w0, float *grad_s0, float *grad_b0, float *grad_wl, float *grad_sl,
                                     void *stream) {
    wtconv_status st = validate_desc(d);
    if (st != WTCONV_OK) return st;
    const wtconv_desc in_scratch = static_desc(d);
    d = &in_scratch;
    const bool family = static_takes_family(d);
    if (!family && bwd_ws_bytes(d) > (size_t)WTCONV_STATIC_SCRATCH_BYTES) return WTCONV_ERR_WORKSPACE;  // shape needs more scratch than is built in
    if ((st = check_device()) != WTCONV_OK) return st;
    void *scratch = nullptr;
    if ((st = static_scratch_for_current_device(&scratch)) != WTCONV_OK) return st;
    // wtconv_backward never depends on what it finds in its workspace, so the contents a previous call left in
    // the shared array do not matter.
    return checked_backward(d, x, grad_out, w0, s0, b0, wl, sl, grad_x, grad_w0, grad_s0, grad_b0, grad_wl, grad_sl, scratch,
                            (size_t)WTCONV_STATIC_SCRATCH_BYTES, stream, family);
}

}  // extern "C"
