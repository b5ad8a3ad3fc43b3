// End of step 3 and step 4 of the path (§2): the final c0 -> 1 channel k5 convolution
// (float32 form; the tensor-core forms run it with dec1) and heuristic peak finding on its
// output.
//
// A persistent grid of 512-thread CTAs walks the events, one event at a time per CTA:
//   1. f[p] = b + sum_t sum_ci W[t][ci] d1[p + t - 2][ci]  (the logit; prob = sigmoid(f)),
//      kept in shared memory, optionally copied out;
//   2. local-maximum rule with a fixed threshold in place of the paper's learned ones:
//      bin i is a PV iff p[i] > 0.01, p[i] > p[j] for the 5 bins on its left and
//      p[i] >= p[j] for the 5 bins on its right (clipped at the ends). Because sigmoid
//      is strictly increasing these decisions are taken exactly on f (the threshold
//      becomes ln(0.01 / 0.99)), which avoids the float32 saturation of sigmoid
//      (which rounds to 1 for f > 16.6) turning distinct maxima into ties;
//   3. ordered compaction: each thread tests its 8 consecutive bins in registers against the
//      maxima of the five bins on either side (running maxima that a NaN passes through, so
//      that a comparison with it fails like the comparison with the bin itself); a
//      block-wide exclusive scan of the per-thread counts gives each PV its slot in a list in
//      shared memory, so PVs come in ascending z without atomics. The true count is always
//      reported;
//   4. z = centroid over bins [i - 3, i + 3] with weights p[j] = sigmoid(f[j]), one listed PV
//      per thread.
//
// What bounds it is instruction issue, and the block barriers between steps of unequal length
// (four CTAs per SM fill them): 8330 warp instructions per event with one PV per owning thread
// (a warp took as many rounds of seven exponentials and divisions as its busiest lane had PVs),
// pairwise comparisons and shuffled scans; 6100 as it stands. 2500 events of given logits: 30.9
// -> 20.2 us per call back to back (DRAM 15 -> 22%). The next event's logits load meanwhile.
// Float32 form, final conv included: 500 events 98 -> 72 us, 16 events 31 -> 20.
#include "pvf_internal.cuh"

namespace pvf {
namespace {

constexpr int kThreads = 512;
constexpr int kPerThread = 8;     // kThreads * kPerThread >= kBins
constexpr int kMaxPeaks = (kBins + kPeakHalfWin) / (kPeakHalfWin + 1);   // peaks lie at least 6 bins apart
// ln(0.01 / 0.99) rounded to float
constexpr float kThrLogit = -4.59511985013459f;
static_assert(kThreads * kPerThread >= kBins && kBins % kPerThread == 0 && kPeakHalfWin == 5 && kThreads / 32 <= 32,
              "bins per thread");

// A centroid weight, sigmoid(x). Below -80 the weight is held at that of -80 (1.8e-35): next to the
// peak's own weight (above 0.01) and added to a bin number of at least 0.5, nothing below 1e-30
// reaches the rounded z, and the exponential stays finite and the quotient normal (both would
// otherwise take the reciprocal's slow path, for every lane of the warp). x is not NaN.
__device__ __forceinline__ float sigmoid_f(float x) { return __frcp_rn(1.0f + expf(-fmaxf(x, -80.0f))); }

// The larger of two, NaN if either is.
__device__ __forceinline__ float max_nan(float a, float b) {
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

// Place of bin i (-8 .. kBins + 7) in shared memory. The 8 bins on either side hold -inf, which no
// finite logit fails against (the same as not comparing clipped neighbours) and whose weight
// vanishes in a centroid (the same as leaving it out). (16-byte reads 8 bins apart meet two-way
// bank conflicts; padding them away cost more in addresses than it saved.)
constexpr int kHalo = 8;
constexpr int kPadded = kBins + 2 * kHalo;
__device__ __forceinline__ constexpr int at(int i) { return i + kHalo; }

// The final conv of the float32 form stages d1 in chunks of bins, transposed to [channel][row].
template <int C0, bool IV> struct FinalTile {
    static constexpr int BINS = IV ? 1000 : 16384 / C0;      // bins per chunk (IV: ten sequences)
    static constexpr int SEQ_ROWS = kIvLen + 2 * kPad;
    static constexpr int ROWS = IV ? BINS / kSliceBins * SEQ_ROWS : BINS + 4;
    static constexpr int PITCH = (ROWS + 27) / 32 * 32 + 4;  // 4 modulo 32: 8 channels x 4 rows on 32 banks
    static constexpr size_t SMEM = sizeof(float) * C0 * PITCH;
    static_assert(!IV || kBins % BINS == 0, "whole sequences");
};

// CONV: the logit comes from the final conv over d1 (the float32 form, base width C0);
// otherwise it is read from a.logit_in.
// IV: d1 is in the per-interval layout; bin 100 s + j is position j + kIvPad of interval
// s's sequence.
template <bool CONV, int C0, bool IV = false>
__global__ void __launch_bounds__(kThreads, CONV ? 2 : 4) k_tail(TailArgs a) {
    __shared__ __align__(16) float sfb[CONV ? 1 : 2][kPadded];   // two events: the next one loads meanwhile
    __shared__ float sw[CONV ? 5 * C0 + 1 : 1];
    __shared__ uint16_t slist[kMaxPeaks + 1];
    __shared__ int swarp[kThreads / 32];
    extern __shared__ __align__(16) float sd[];     // CONV: the staged chunk

    const int tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5;
    if (tid < 2 * kHalo)
        for (float *f : {sfb[0], sfb[CONV ? 0 : 1]}) f[at(tid < kHalo ? tid - kHalo : kBins + tid - kHalo)] = __int_as_float(0xff800000);
    if constexpr (CONV) {
        for (int i = tid; i < 5 * C0 + 1; i += kThreads) sw[i] = a.final_w[i];
        __syncthreads();
    }
    // the logits (or d1) are the previous kernel's output (dependent launch)
    grid_dep_wait();
    grid_dep_launch();
    // persistent: the CTA walks the launch's events
    const int n_ev = launch_events(a.n_dyn, a.ev_base, a.n_events);
    // the logits of event e into buffer f (asynchronous copies)
    auto stage = [&](int e, float *f) {
        const float *src = a.logit_in + (size_t)(a.ev_base + e - a.logit_in_base) * kBins;
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(f + at(0));
        if ((reinterpret_cast<uintptr_t>(src) & 15) == 0) {
            for (int p = tid; p < kBins / 4; p += kThreads)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16 * p), "l"(src + 4 * p) : "memory");
        } else {
            for (int p = tid; p < kBins; p += kThreads)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + 4 * p), "l"(src + p) : "memory");
        }
    };
    if constexpr (!CONV)
        if ((int)blockIdx.x < n_ev) stage(blockIdx.x, sfb[0]);
    int buf = 0;
    for (int e = blockIdx.x; e < n_ev; e += gridDim.x) {
        const int ge = a.ev_base + e;
        float *sf = sfb[buf];
        if constexpr (!CONV) {
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncthreads();                   // staged; nobody reads the other buffer, slist or swarp any more
            buf ^= 1;
            if (e + (int)gridDim.x < n_ev) stage(e + gridDim.x, sfb[buf]);
        } else {
            using F = FinalTile<C0, IV>;
            const int64_t rows1 = padded_rows(IV ? kIvLen : kBins);
            // first storage row of the event's tensor (IV: of its first sequence)
            const float *d1 = reinterpret_cast<const float *>(a.d1) + (IV ? (size_t)e * kSlices : (size_t)e) * rows1 * C0;
            for (int b0 = 0; b0 < kBins; b0 += F::BINS) {
                const int row0 = IV ? b0 / kSliceBins * F::SEQ_ROWS : b0;
                const int rows = IV ? F::ROWS : min(F::ROWS, (int)rows1 - row0);
#pragma unroll 1
                for (int k8 = 0; k8 < C0; k8 += 8)
#pragma unroll 4
                    for (int i = tid; i < rows * 8; i += kThreads) {    // 8 channels x 4 rows per warp
                        const int k = k8 + (i & 7), r = i >> 3;
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                                         (uint32_t)__cvta_generic_to_shared(sd + k * F::PITCH + r)),
                                     "l"(d1 + (size_t)(row0 + r) * C0 + k)
                                     : "memory");
                    }
                asm volatile("cp.async.wait_all;" ::: "memory");
                __syncthreads();
                // two bins per thread where the chunk has them: the weights are read once for both
                constexpr int NB = (F::BINS + kThreads - 1) / kThreads;
                float acc[NB];
                const float *x[NB];
#pragma unroll
                for (int q = 0; q < NB; ++q) {
                    const int p = min(tid + q * kThreads, F::BINS - 1);
                    acc[q] = sw[5 * C0];
                    // storage row x + t = position x + t - 2
                    x[q] = sd + (IV ? p / kSliceBins * F::SEQ_ROWS + p % kSliceBins + kIvPad : p);
                }
#pragma unroll 1
                for (int t = 0; t < 5; ++t) {
#pragma unroll
                    for (int ci = 0; ci < C0; ++ci) {
                        const float w = sw[t * C0 + ci];
#pragma unroll
                        for (int q = 0; q < NB; ++q) acc[q] = fmaf(w, x[q][ci * F::PITCH + t], acc[q]);
                    }
                }
#pragma unroll
                for (int q = 0; q < NB; ++q) {
                    const int p = tid + q * kThreads;
                    if (p < F::BINS && b0 + p < kBins) sf[at(b0 + p)] = acc[q];
                }
                __syncthreads();               // sd is refilled; the last chunk's logits are in place
            }
        }
        if (a.logit_out) {
            float *dst = a.logit_out + (size_t)ge * kBins;
            for (int p = tid; p < kBins; p += kThreads) dst[p] = sf[at(p)];
        }
        if (a.pv_count) {
            const bool bypass = a.ev_flag && a.ev_flag[ge] != 0;
            // ---- candidate flags: thread tid owns bins [8 tid, 8 tid + 8) and loads them with their
            //      +-5 neighbours (bins 8 tid - 8 .. 8 tid + 15, 16-byte loads)
            const int i0 = tid * kPerThread;
            unsigned mask = 0;
            if (!bypass && i0 < kBins) {
                float w[kPerThread + 16];
#pragma unroll
                for (int k = 0; k < (kPerThread + 16) / 4; ++k) {
                    const float4 x = *reinterpret_cast<const float4 *>(sf + at(i0 - 8 + 4 * k));
                    w[4 * k] = x.x; w[4 * k + 1] = x.y; w[4 * k + 2] = x.z; w[4 * k + 3] = x.w;
                }
                // m[i] = the maximum of w[i .. i + 4], for i = 3 .. 16, from maxima of two and four
                float m[kPerThread + 11];
#pragma unroll
                for (int i = 3; i <= kPerThread + 10; ++i) m[i] = max_nan(w[i], w[i + 1]);
#pragma unroll
                for (int i = 3; i <= kPerThread + 8; ++i) m[i] = max_nan(max_nan(m[i], m[i + 2]), w[i + 4]);
#pragma unroll
                for (int b = 0; b < kPerThread; ++b) {
                    const float fi = w[b + 8];
                    if (fi > kThrLogit && fi > m[b + 3] && fi >= m[b + 9]) mask |= 1u << b;
                }
            }
            // ---- slots: at most two of a thread's 8 bins are peaks (they lie 6 bins apart), so two
            //      ballots rank them within the warp; the warps' counts are summed by every warp
            const int cnt = __popc(mask);
            const unsigned one = __ballot_sync(0xffffffffu, cnt >= 1), two = __ballot_sync(0xffffffffu, cnt >= 2);
            const unsigned below = (1u << lane) - 1u;
            if (lane == 0) swarp[warp] = __popc(one) + __popc(two);
            __syncthreads();
            const int v = lane < kThreads / 32 ? swarp[lane] : 0;
            const int total = __reduce_add_sync(0xffffffffu, v);
            int idx = __reduce_add_sync(0xffffffffu, lane < warp ? v : 0) + __popc(one & below) + __popc(two & below);
            while (mask) {
                const int k = __ffs(mask) - 1;
                mask &= mask - 1;
                slist[idx++] = (uint16_t)(i0 + k);
            }
            __syncthreads();
            float *zout = a.pv_z + (size_t)ge * a.max_pv;
            const int listed = min(total, a.max_pv);
            for (int s = tid; s < listed; s += kThreads) {
                const int i = slist[s];
                float num = 0.0f, den = 0.0f;
#pragma unroll
                for (int d = -kCentroidHalf; d <= kCentroidHalf; ++d) {
                    const float pj = sigmoid_f(sf[at(i + d)]);
                    num = fmaf(pj, (float)d, num);
                    den += pj;
                }
                // z = zc(i) + 0.1 * (sum p_j (j - i) / sum p_j), zc(i) = -100 + (i + 0.5) * 0.1
                zout[s] = fmaf((float)i + 0.5f + num / den, kBinW, kZLo);
            }
            if (tid == 0) {
                a.pv_count[ge] = bypass ? -1 : total;
                if (!bypass && total > a.max_pv) raise_status(a.status, PVF_WARN_TRUNCATED);
            }
        }
    }
}

// Persistent grid of resident CTAs (their launch bounds fix the registers: four per SM,
// two with the final conv), each
// walking events.
template <bool CONV, int C0, bool IV = false>
cudaError_t launch_tail_t(const TailArgs &a, cudaStream_t s) {
    int sms = 0;
    const size_t smem = CONV ? FinalTile<C0, IV>::SMEM : 0;
    cudaError_t err = current_device_sms(&sms);
    if (err == cudaSuccess && CONV) err = prepare_kernel((const void *)k_tail<CONV, C0, IV>, smem, nullptr);
    if (err != cudaSuccess) return err;
    int per_sm = CONV ? 2 : 4;
    if (a.ctas_per_sm > 0 && a.ctas_per_sm < per_sm) per_sm = a.ctas_per_sm;
    const dim3 grid(a.n_events < per_sm * sms ? a.n_events : per_sm * sms), block(kThreads);
    return launch_pdl(k_tail<CONV, C0, IV>, grid, block, smem, s, a);
}

}  // namespace

cudaError_t launch_tail(const TailArgs &a, int precision, cudaStream_t s) {
    if (a.n_events <= 0) return cudaSuccess;
    if (a.logit_in) return launch_tail_t<false, kC0>(a, s);
    // the final conv runs here in the FP32 form only (the tensor-core forms run it in
    // dec1's epilogue and pass logits)
    if (precision != PVF_FP32) return cudaErrorInvalidValue;
    if (a.iv) return a.c0 == kC0 ? launch_tail_t<true, kC0, true>(a, s) : cudaErrorInvalidValue;
    if (a.c0 == kC0Max) return launch_tail_t<true, kC0Max>(a, s);
    if (a.c0 == kC0) return launch_tail_t<true, kC0>(a, s);
    return cudaErrorInvalidValue;
}

}  // namespace pvf
