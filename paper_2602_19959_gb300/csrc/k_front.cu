// Steps 1-2 of the path (§2) in the float32 form: per-track FC network and the per-event slice
// histogram, plus the first UNet convolution (1 -> 16 channels, k5) and its 2:1 max-pool, fused so
// that the histogram never leaves shared memory on its way into the UNet.
//
// A persistent grid walks the events, one event at a time per CTA (§3: each event is
// processed by one thread block); with fewer events than half the CTAs the chip holds, a cluster
// of 2, 4 or 8 CTAs shares each event by slices (s modulo the cluster's size: tracks crowd into
// neighbouring slices). Per event:
//   a. validate the event's offsets; bypass it (flag = 1, histogram of zeros) when they
//      are negative, decreasing or past the feature arrays, or the event holds more
//      than max_tracks tracks;
//   b. slice index per track, s = floor((z + 100) / 10) in float32 round-to-nearest;
//      a track is dropped when a feature is not finite or s is outside [0, 40);
//   c. stable counting sort of the valid tracks by slice (integer work only), with the
//      boundary tracks' second slices (§3) when the boundary width is non-zero;
//   d. hidden layers 1-5 of the FC net in chunks of 256 sorted tracks, as a register-tiled product
//      per warp (32 tracks x 32 outputs, 4 x 8 per lane; 8 tracks where a chunk has few), in place
//      in a shared-memory tile [feature][track];
//   e. output layer: softplus(W6[j] . h5 + b6[j]) of 48 tracks at a time, the tracks dealt out to
//      the warps whatever their slices, into shared memory; then the thread owning bins j and j + 1
//      of slice s adds the slice's values in sorted (= input) order, so the order depends only on
//      the event's own track list: results are bitwise reproducible and identical alone or in any
//      batch. No float atomics.
//   f. e1 = LeakyReLU(conv_k5(hist)), p1 = maxpool2(e1), stored in float32 rows; the CTAs of a
//      cluster first read each other's slices.
//
// What bounds it: with every SM busy, FMA issue in d and e (a chunk's hidden layers run at 80% of
// the FMA rate) and the stores of f (59 bytes per cycle and SM). One thread per track waited for
// the shared-memory port, a 16-byte weight read per four FMAs; output layer and sums in one loop
// left all but two warps idle in events whose tracks share a slice (500 cycles per track). 500
// events: 203 us, tiled hidden layers 145, separate sums 130 (sums of 16, 32, 48 and 64 tracks at
// a time 144, 134, 130, 125; 48 is what two CTAs per SM have room for with boundary tracks). 16
// events, one CTA each 66 us, tiled 46, eight CTAs each 37, separate sums 25 (4 CTAs each: the
// same within 1 us of 8).
#include <cooperative_groups.h>

#include "front_common.cuh"

namespace pvf {
namespace {

using namespace front;

namespace cg = cooperative_groups;

constexpr int kThreads = 256;
constexpr int kChunk = 256;               // tracks per FC chunk: 32 per warp
constexpr int kHPitch = kChunk + 4;       // floats per feature row of the chunk's tile [feature][track]
constexpr int kSub = 48;                  // tracks whose output values wait to be summed
constexpr int kGroup = 64;                // threads per slice of the output layer, two bins each
constexpr int kMaxSplit = 8;              // blocks that may share an event (portable cluster size)

struct FrontSmem {
    // byte offsets into dynamic shared memory
    static constexpr size_t fc = 0;                                   // kFcFloats floats
    static constexpr size_t enc1 = fc + sizeof(float) * kFcFloats;    // 6 c0 floats
    static constexpr size_t hist = (enc1 + sizeof(float) * kEnc1FloatsMax + 15) / 16 * 16;
    static constexpr size_t h5 = hist + sizeof(float) * kBins;        // 32 x kHPitch
    static constexpr size_t val = h5 + sizeof(float) * kFcHidden * kHPitch;  // kSub x 100
    static constexpr size_t cnt = val + sizeof(float) * kSub * kFcOut;       // 41 ints
    static constexpr size_t seg = cnt + sizeof(int) * 48;             // 41 ints
    static constexpr size_t run = seg + sizeof(int) * 48;             // 40 ints
    static constexpr size_t sorted = run + sizeof(int) * 48;          // uint16 [entries]
    __host__ __device__ static size_t slices(int entries) { return sorted + 2 * (size_t)((entries + 7) / 8 * 8); }
    __host__ __device__ static size_t total(int max_tracks, float edge) {
        return slices(front_entries(max_tracks, edge)) + (size_t)max_tracks + 16;
    }
};

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// One hidden layer for 8 TR tracks of the warp: lane (tg, og) computes outputs [8 og, 8 og + 8) of
// TR neighbouring tracks, in place in the tile (the warp's columns are its own). Eight weights and
// TR inputs from shared memory feed 8 TR FMAs (outputs in pairs), each output an fmaf chain over
// the inputs in order from its bias.
template <int TR, int NIN>
__device__ __forceinline__ void fc_layer(const float *__restrict__ w, const float *__restrict__ b, float *col, int og) {
    float2 acc[TR][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float2 bj = *reinterpret_cast<const float2 *>(b + 8 * og + 2 * j);
#pragma unroll
        for (int t = 0; t < TR; ++t) acc[t][j] = bj;
    }
#pragma unroll 4
    for (int i = 0; i < NIN; ++i) {
        const float4 w0 = *reinterpret_cast<const float4 *>(w + i * kFcHidden + 8 * og);
        const float4 w1 = *reinterpret_cast<const float4 *>(w + i * kFcHidden + 8 * og + 4);
        float x[TR];
        if constexpr (TR == 4) {
            const float4 v = *reinterpret_cast<const float4 *>(col + i * kHPitch);
            x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
        } else {
            x[0] = col[i * kHPitch];
        }
#pragma unroll
        for (int t = 0; t < TR; ++t) {
            const float2 xx = make_float2(x[t], x[t]);
            acc[t][0] = __ffma2_rn(make_float2(w0.x, w0.y), xx, acc[t][0]);
            acc[t][1] = __ffma2_rn(make_float2(w0.z, w0.w), xx, acc[t][1]);
            acc[t][2] = __ffma2_rn(make_float2(w1.x, w1.y), xx, acc[t][2]);
            acc[t][3] = __ffma2_rn(make_float2(w1.z, w1.w), xx, acc[t][3]);
        }
    }
    __syncwarp();                          // every lane has read its inputs
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
        for (int t = 0; t < TR; ++t) acc[t][j] = leaky2(acc[t][j]);
        float *d = col + (8 * og + 2 * j) * kHPitch;
        if constexpr (TR == 4) {
            *reinterpret_cast<float4 *>(d) = make_float4(acc[0][j].x, acc[1][j].x, acc[2][j].x, acc[3][j].x);
            *reinterpret_cast<float4 *>(d + kHPitch) = make_float4(acc[0][j].y, acc[1][j].y, acc[2][j].y, acc[3][j].y);
        } else {
            d[0] = acc[0][j].x;
            d[kHPitch] = acc[0][j].y;
        }
    }
    __syncwarp();
}

// Hidden layers 1-5 of a chunk's m tracks (entries ssorted[0..m)) into the tile: each warp takes
// 8 TR of them at a time. Lanes without a track carry zeros.
template <int TR, bool EDGE>
__device__ __forceinline__ void fc_hidden(const FrontArgs &a, const float *__restrict__ W, int64_t t0, int m,
                                          const uint16_t *ssorted, const uint8_t *sslice, float *tile, int tid) {
    static_assert(TR == 1 || TR == 4, "one or four tracks per lane");
    const int lane = tid & 31, tg = lane & 7, og = lane >> 3;
#pragma unroll 1
    for (int base = (tid >> 5) * 8 * TR; base < m; base += kThreads / 32 * 8 * TR) {
        if (lane < 8 * TR) {
            float x[kFcInPad] = {};
            if (base + lane < m) {
                const int en = ssorted[base + lane];
                track_features(a, t0 + entry_track<EDGE>(en), entry_slice<EDGE>(en, sslice), x);
            }
#pragma unroll
            for (int i = 0; i < kFcInPad; ++i) tile[i * kHPitch + base + lane] = x[i];
        }
        __syncwarp();
        float *col = tile + base + TR * tg;
        fc_layer<TR, kFcInPad>(W + fc_w_off(0), W + fc_b_off(0), col, og);
#pragma unroll 1
        for (int l = 1; l < 5; ++l)
            fc_layer<TR, kFcHidden>(W + fc_w_off(1) + (l - 1) * kFcWH, W + fc_b_off(1) + (l - 1) * kFcHidden, col, og);
    }
}

// ENC1 = false: steps a-e only (the histogram), nothing written to e1/p1.
// EDGE: boundary tracks fill a second slice (a.edge > 0).
// C0: UNet base width of the e1 / p1 tensors written here (16, or 32 in this float32 form).
// IV: e1 / p1 in the per-interval layout (kSlices windowed sequences per event).
template <bool ENC1, bool EDGE, int C0, bool IV = false>
__global__ void __launch_bounds__(kThreads, 2) k_front(FrontArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    float *sfc = reinterpret_cast<float *>(smem + FrontSmem::fc);
    float *senc = reinterpret_cast<float *>(smem + FrontSmem::enc1);
    float *shist = reinterpret_cast<float *>(smem + FrontSmem::hist);
    float *sh5 = reinterpret_cast<float *>(smem + FrontSmem::h5);
    float *sval = reinterpret_cast<float *>(smem + FrontSmem::val);
    int *scnt = reinterpret_cast<int *>(smem + FrontSmem::cnt);
    int *sseg = reinterpret_cast<int *>(smem + FrontSmem::seg);
    int *srun = reinterpret_cast<int *>(smem + FrontSmem::run);
    uint16_t *ssorted = reinterpret_cast<uint16_t *>(smem + FrontSmem::sorted);
    uint8_t *sslice = smem + FrontSmem::slices(EDGE ? 2 * a.max_tracks : a.max_tracks);

    const int tid = threadIdx.x;
    const cg::cluster_group cl = cg::this_cluster();
    const int nr = (int)cl.num_blocks(), rank = (int)cl.block_rank();   // blocks that share an event
    if constexpr (ENC1)
        for (int i = tid; i < 6 * C0; i += kThreads) senc[i] = a.enc1[i];
    if (!a.hist_in)
        for (int i = tid; i < kFcFloats / 4; i += kThreads)
            cp_async16(sfc + 4 * i, a.fc + 4 * i);     // arrive behind the first event's sort

    // the caller's inputs, and the buffers that earlier calls' kernels may still read, only after the
    // previous kernel of the stream has finished (no early trigger: see the launches of k_unet_f32.cu)
    grid_dep_wait();

    // persistent: the CTA walks the launch's events (weights loaded once above)
    for (int e = blockIdx.x / nr; e < a.n_events; e += gridDim.x / nr) {
        const int ge = a.ev_base + e;
        if (a.hist_in) {
            const float *src = a.hist_in + (size_t)ge * kBins;
            for (int i = tid; i < kBins; i += kThreads) shist[i] = src[i];
        } else {
            // ---- a-c. validate, slice per track, stable sort by slice
            for (int i = tid; i < kBins; i += kThreads) shist[i] = 0.0f;
            int64_t t0;
            int nvalid;
            validate_sort<kThreads, EDGE, true>(a, ge, tid, scnt, sseg, srun, ssorted, sslice, t0, nvalid, rank, nr);

            cp_async_wait_all();
            __syncthreads();

            // ---- d/e. hidden layers per track, then output layer + per-bin sequential sums
            const int grp = tid / kGroup, j = 2 * (tid % kGroup);    // bins j and j + 1 of the group's slices
            for (int c0 = 0; c0 < nvalid; c0 += kChunk) {
                const int m = min(kChunk, nvalid - c0);
                if (m > 64) fc_hidden<4, EDGE>(a, sfc, t0, m, ssorted + c0, sslice, sh5, tid);
                else fc_hidden<1, EDGE>(a, sfc, t0, m, ssorted + c0, sslice, sh5, tid);
                __syncthreads();
                float2 w[kFcHidden];
                float2 bj = make_float2(0.0f, 0.0f);
                if (j < kFcOut) {
#pragma unroll
                    for (int i = 0; i < kFcHidden; ++i)
                        w[i] = *reinterpret_cast<const float2 *>(sfc + fc_w_off(5) + i * kFcOut + j);
                    bj = *reinterpret_cast<const float2 *>(sfc + fc_b_off(5) + j);
                }
                for (int q0 = 0; q0 < m; q0 += kSub) {
                    // values of the next kSub tracks, four at a time, whatever their slices
                    const int mq = min(kSub, m - q0);
                    if (j < kFcOut) {
                        for (int r = 4 * grp; r < mq; r += 4 * (kThreads / kGroup)) {
                            float2 o[4] = {bj, bj, bj, bj};
#pragma unroll
                            for (int i = 0; i < kFcHidden; ++i) {
                                const float4 h = *reinterpret_cast<const float4 *>(sh5 + i * kHPitch + q0 + r);
                                o[0] = __ffma2_rn(w[i], make_float2(h.x, h.x), o[0]);
                                o[1] = __ffma2_rn(w[i], make_float2(h.y, h.y), o[1]);
                                o[2] = __ffma2_rn(w[i], make_float2(h.z, h.z), o[2]);
                                o[3] = __ffma2_rn(w[i], make_float2(h.w, h.w), o[3]);
                            }
#pragma unroll
                            for (int u = 0; u < 4; ++u)      // rows past mq hold a chunk's padding; nobody reads them
                                *reinterpret_cast<float2 *>(sval + (r + u) * kFcOut + j) =
                                    make_float2(softplus_f(o[u].x), softplus_f(o[u].y));
                        }
                    }
                    __syncthreads();
                    // their sums, per bin in sorted order
                    if (j < kFcOut) {
                        for (int s = rank + nr * grp; s < kSlices; s += nr * (kThreads / kGroup)) {
                            const int lo = max(sseg[s] - c0 - q0, 0), hi = min(sseg[s + 1] - c0 - q0, mq);
                            if (lo >= hi) continue;
                            float2 *bin = reinterpret_cast<float2 *>(shist + s * kSliceBins + j);
                            float2 acc = *bin;
#pragma unroll 4
                            for (int r = lo; r < hi; ++r) {
                                const float2 v = *reinterpret_cast<const float2 *>(sval + r * kFcOut + j);
                                acc.x = __fadd_rn(acc.x, v.x);
                                acc.y = __fadd_rn(acc.y, v.y);
                            }
                            *bin = acc;
                        }
                    }
                    __syncthreads();
                }
            }
            if (nr > 1) {                  // the other blocks' slices
                cl.sync();
                constexpr int R = kSliceBins / 4;
                for (int i = tid; i < kBins / 4; i += kThreads) {
                    const int r = (i / R) & (nr - 1);
                    if (r != rank)
                        reinterpret_cast<float4 *>(shist)[i] = reinterpret_cast<const float4 *>(cl.map_shared_rank(shist, r))[i];
                }
                cl.barrier_arrive();       // read: their owners may go on
            }
        }
        __syncthreads();

        const int gtid = tid + kThreads * rank, nt = kThreads * nr;
        if (a.hist_out) {
            float4 *dst = reinterpret_cast<float4 *>(a.hist_out + (size_t)ge * kBins);
            const float4 *src = reinterpret_cast<const float4 *>(shist);
            for (int i = gtid; i < kBins / 4; i += nt) dst[i] = src[i];
        }

        if constexpr (ENC1) {
            if (a.e1) enc1_pool_f32<C0, IV>(a, e, gtid, nt, shist, senc);   // null: the histogram alone was asked for
        }
        if (nr > 1 && !a.hist_in) cl.barrier_wait();
        __syncthreads();                   // shist and the sort arrays are reused next event
    }
}

// Persistent grid: as many CTAs as the shared memory lets reside (at most two per SM,
// the register limit at 256 threads), capped by the number of events. Where the events leave some
// of those CTAs idle, a cluster of 2, 4 or 8 shares each event.
template <bool ENC1, bool EDGE, int C0, bool IV = false>
cudaError_t launch_front_t(const FrontArgs &a, size_t smem, cudaStream_t s) {
    int sms = 0;
    cudaError_t err = current_device_sms(&sms);
    if (err == cudaSuccess) err = prepare_kernel((const void *)k_front<ENC1, EDGE, C0, IV>, smem, nullptr);
    if (err != cudaSuccess) return err;
    int per_sm = (int)((228 * 1024) / (smem + 1024));
    if (per_sm > 2) per_sm = 2;
    if (a.ctas_per_sm > 0 && a.ctas_per_sm < per_sm) per_sm = a.ctas_per_sm;
    if (per_sm < 1) per_sm = 1;
    int split = 1;
    while (split < kMaxSplit && 2 * split * (int64_t)a.n_events <= sms * per_sm) split *= 2;
    const int64_t most = split > 1 ? (int64_t)split * a.n_events : sms * per_sm;
    // dependent launch as in launch_pdl, but not for the histogram alone, whose weights are copied to
    // the static scratch by the call itself
    cudaLaunchAttribute attr[2];
    int n_attr = 0;
    if (ENC1) {
        attr[n_attr].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n_attr++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (split > 1) {
        attr[n_attr].id = cudaLaunchAttributeClusterDimension;
        attr[n_attr++].val.clusterDim = {(unsigned)split, 1, 1};
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(most < (int64_t)split * a.n_events ? most : (int64_t)split * a.n_events));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = n_attr;
    return cudaLaunchKernelEx(&cfg, k_front<ENC1, EDGE, C0, IV>, a);
}

}  // namespace

size_t front_smem_bytes(int max_tracks, float edge) { return FrontSmem::total(max_tracks, edge); }

cudaError_t launch_front_hist_only(const FrontArgs &a, size_t smem, cudaStream_t s) {
    if (a.n_events <= 0) return cudaSuccess;
    if (a.edge > 0.0f) return cudaErrorInvalidValue;   // the no-allocation path has no boundary tracks
    return launch_front_t<false, false, kC0>(a, smem, s);
}

cudaError_t launch_front(const FrontArgs &a, int precision, size_t smem, cudaStream_t s) {
    if (a.n_events <= 0) return cudaSuccess;
    // the tensor-core forms run k_front_tc
    if (precision != PVF_FP32) return cudaErrorInvalidValue;
    if (a.iv) {   // per-interval layout: width 16
        if (a.c0 != kC0) return cudaErrorInvalidValue;
        return a.edge > 0.0f ? launch_front_t<true, true, kC0, true>(a, smem, s)
                             : launch_front_t<true, false, kC0, true>(a, smem, s);
    }
    if (a.c0 == kC0Max)
        return a.edge > 0.0f ? launch_front_t<true, true, kC0Max>(a, smem, s)
                             : launch_front_t<true, false, kC0Max>(a, smem, s);
    if (a.c0 != kC0) return cudaErrorInvalidValue;
    return a.edge > 0.0f ? launch_front_t<true, true, kC0>(a, smem, s)
                         : launch_front_t<true, false, kC0>(a, smem, s);
}

}  // namespace pvf
