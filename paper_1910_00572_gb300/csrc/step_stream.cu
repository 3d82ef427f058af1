// Single-session launch of the streaming propagation (stream.cuh): the tiles of one grid,
// dealt to the persistent CTAs in turn.
#include <type_traits>

#include "per_device.h"
#include "stream.cuh"

namespace loc {
namespace {

using namespace stream;

__constant__ int g_stall = 0;              // see set_step_stall

template <typename T, bool AM, bool RAG>
__global__ void __launch_bounds__(stream::NT, 1) step_stream_kernel(const __grid_constant__ FastArgs a, int ntx,
                                                                    int ntiles) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const uint32_t sbase = su32(smem_raw);
    stream::Smem<T>& sm = *reinterpret_cast<stream::Smem<T>*>(smem_raw + (((sbase + 127u) & ~127u) - sbase));
    int reinit = 0;
    float in_scale = 0.0f;
    int tile = blockIdx.x;
    run_roles<T, AM, RAG, false>(
        sm, g_stall,
        [&](Item& it, Source& src) {
            if (tile >= ntiles) return;
            it.out = a.B_out;
            it.in = a.B_in;
            it.trav = a.trav;
            it.corr = a.corr;
            it.K = a.K;
            it.H = a.H;
            it.W = a.W;
            it.ty0 = (tile / ntx) * stream::TH;
            it.tx0 = (tile % ntx) * TW;
            it.g0 = a.g0;
            it.g1 = a.g1;
            it.g2 = a.g2;
#pragma unroll
            for (int d = 0; d < RING; ++d) it.gt[d] = a.gt[d];
            it.tile = tile;
            it.ntiles = ntiles;
            src.tmap = &a.tmap;
            src.sh = a.sh;
            tile += gridDim.x;
        },
        [&]() {
            // what earlier work on the stream wrote is read (and overwritten) from here on
            asm volatile("griddepcontrol.wait;" ::: "memory");
            // The next step's CTAs may take the SMs that this one's leave: their barriers, plans and
            // masks (all from the map and the launch's arguments) are then ready when the grid ends.
            // Not before the wait: a step that itself waits would let in the one after it, and so on,
            // until queues of small steps held the SMs that other streams' kernels need (a 64 x 64 x 16
            // step beside eight streams of queued 64 x 64 x 128 steps: 82 us, 23 like this; a 512 x 512 x
            // 64 step 232 against 75; steps of one stream alone the same to 1 %).
            asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
            reinit = a.sd->reinit;
            // restart: the input is M / (K n_free); read M and fold 1 / (K n_free) into the scale
            in_scale = (reinit ? a.inv_uniform : a.sd->inv_Z) * a.out_mult;
        },
        [&](Item& it, Source& src) {
            it.in_scale = in_scale;
            it.reinit = src.reinit = reinit;
        },
        [&](const Item& it, int slot) {
            retire_tile<AM>(sm, it, slot, a.partials, a.am_pv, a.am_pi, &a.sd->counter, [&](double Z, const ArgBest& b) {
                session_finish(a.sd, Z, a.log_out_mult);
                if constexpr (AM) {
                    // no result when the session restarts
                    const bool live = Z > 0.0 && isfinite(Z);
                    *a.am_idx = live ? b.i : -1;
                    if (live) *a.am_val = (float)((double)b.v / Z);
                }
            });
        });
    if (threadIdx.x == 0 && sm.fail) atomicOr(&a.sd->status, LOC_DEV_ERR_TIMEOUT);
}

template <typename T, bool AM, bool RAG = false>
cudaError_t launch(const FastArgs& a, cudaStream_t st) {
    static PerDevice sms;
    int dev = 0, n_sm = 0;
    cudaGetDevice(&dev);
    const size_t sb = sizeof(stream::Smem<T>) + 128;
    const cudaError_t e = sms.get(dev, &n_sm, [dev](int* n) {
        const cudaError_t p = prepare<T>(step_stream_kernel<T, AM, RAG>);
        return p != cudaSuccess ? p : cudaDeviceGetAttribute(n, cudaDevAttrMultiProcessorCount, dev);
    });
    if (e != cudaSuccess) return e;
    const int ntx = (a.W + TW - 1) / TW, ntiles = ntx * ((a.H + stream::TH - 1) / stream::TH);
    const int grid = ntiles < n_sm ? ntiles : n_sm;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(stream::NT);
    cfg.dynamicSmemBytes = sb;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, step_stream_kernel<T, AM, RAG>, a, ntx, ntiles);
}

}  // namespace

cudaError_t launch_step_stream(const void* args, int storage, bool argmax, cudaStream_t st) {
    const FastArgs& a = *static_cast<const FastArgs*>(args);
    switch (storage) {
        case LOC_F32: return argmax ? launch<float, true>(a, st) : launch<float, false>(a, st);
        case LOC_BF16: return argmax ? launch<__nv_bfloat16, true>(a, st) : launch<__nv_bfloat16, false>(a, st);
        case LOC_F16: return argmax ? launch<__half, true>(a, st) : launch<__half, false>(a, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_step_ragged(const StepArgs& g, int storage, cudaStream_t st) {
    FastArgs a;
    memset(&a.tmap, 0, sizeof(a.tmap));
    fill_args(a, g);
    switch (storage) {
        case LOC_F32: return launch<float, false, true>(a, st);
        case LOC_BF16: return launch<__nv_bfloat16, false, true>(a, st);
        case LOC_F16: return launch<__half, false, true>(a, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t set_step_stall(int tile) { return cudaMemcpyToSymbol(g_stall, &tile, sizeof(tile)); }

bool step_ragged_eligible(int K, int r_xy, int r_th) { return r_xy == R && r_th == RT && K >= 8 && K <= LOC_MAX_K; }

int stream_tile_rows() { return stream::TH; }

int stream_box_w(int storage) { return storage == LOC_F32 ? box_w<float>() : box_w<__half>(); }

}  // namespace loc
