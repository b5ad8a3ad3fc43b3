// The last UNet layer of the tensor-core forms: dec1 ([u1 | e1] -> c0 channels, k5) with the
// final conv (c0 -> 1, float32) in its epilogue, for csrc/k_unet_tc.cu.
//
// With 16 output channels an MMA of one tap (M = 128 positions, N = 16) spends its time reading
// A: ten of them per 124 positions, and an epilogue that reads its weights from shared memory
// (four data cycles per 16-byte load, 75% of that path) once per position, took 77 us per 1000
// events where the tensors' traffic takes 40. Here a tile row is a block of four consecutive
// positions: u1 and e1 are stored by residue (position modulo 4, the "quad" layout), so the
// input position x = -2 .. 5 of every block is a plane of consecutive rows, and one MMA
// multiplies it into all the outputs j of the block that it reaches, stacked along N:
//     D[block][j][co] += X_x[block] * W_t,   t = x - j + 2 in 0 .. 4
// The weights lie with the taps in descending order, so every stack is a window of one image
// and no multiplication by a zero weight occurs. x runs upwards: an output adds its taps in
// ascending order, each over K in order, exactly as one tap at a time did, so results are bit
// for bit the same. An output's first product overwrites (its accumulator holds an earlier
// tile), which splits the first K step of x = -1, 0, 1 in two: 19 MMAs per 504 positions (16
// bits) instead of 41. A thread then holds four positions: the weights of the final conv are
// read once for all four, its partial sums come from the neighbouring lane (six values per
// four positions), and the logits leave as 16 bytes.
#pragma once

// Measured (1000 events): FP16 77.7 -> 56 us (73% of DRAM throughput: it is bound by its input,
// 256 KB per event), FP8 67 -> 37 us, wide FP16 (250 events) 45 -> 34, per-interval (500) 45 -> 35.
// Three epilogue warpgroups 56 and 41 us, four 66 and 55: no gain in 16 bits, a loss in FP8.

// (included inside k_unet_tc.cu's namespaces)

template <int PREC_, int C0_, int L_, int SEQ_ = 0> struct Dec1 {
    static constexpr int PREC = PREC_, COUT = C0_, L = L_, SEQ = SEQ_;
    static constexpr int LSEQ = SEQ ? SEQ - kPad : L;
    static constexpr int PW = is16(PREC) ? 8 : 16;
    static constexpr int PA = C0_ / PW, PIN = 2 * PA;        // K planes of u1, of both
    static constexpr int RQ = quad_rows(L);                  // rows of a residue plane
    static constexpr int BLOCKS = (L + 3) / 4;
    static constexpr int STRIDE = kTileM - 2;                // output blocks of a tile (one on each side is halo)
    static constexpr int TPE = (BLOCKS + STRIDE - 1) / STRIDE;
    static constexpr int ROWS = kTileM + 1, PLANE = ROWS * 16;
    static constexpr int A_STAGE = align_up(PIN * 4 * PLANE, 128);
    static constexpr int W_BYTES = 5 * PIN * COUT * 16;
    static constexpr int COLS = 4 * COUT, NB = 4, TMEM_COLS = NB * COLS;
    // narrow: two CTAs per SM, two epilogue warpgroups each; wide: one with four
        static constexpr int EWG = COUT == kC0 ? 2 : 4, CTAS = COUT == kC0 ? 2 : 1;
    static constexpr int THREADS = 64 + 128 * EWG;
    static constexpr int STAGES = is16(PREC) ? 3 : 4;
    static constexpr int NPAR = 2 * COUT + 5 * COUT + 1;     // bias, column scales, final conv
    static constexpr int OFF_W = 0;
    static constexpr int OFF_PAR = align_up(OFF_W + W_BYTES, 128);
    static constexpr int OFF_A = align_up(OFF_PAR + 4 * NPAR, 128);
    static constexpr int OFF_X = OFF_A + STAGES * A_STAGE;   // exchange: [EWG][2][4 warps][8] floats
    static constexpr int OFF_BAR = OFF_X + EWG * 2 * 4 * 8 * 4;
    static constexpr int W = 0, FULL = 1, EMPTY = FULL + STAGES, TF = EMPTY + STAGES, TE = TF + NB, XR = TE + NB,
                         DRAIN = XR + EWG, NBAR = DRAIN + 1;
    static constexpr int SMEM = OFF_BAR + 8 * NBAR + 16;
    static constexpr uint32_t FMT = PREC == PVF_BF16 ? 1u : 0u;
    static_assert(PIN % 2 == 0 && COUT % 16 == 0 && COLS <= 256 && TMEM_COLS <= 512, "operands");
    static_assert(CTAS * (SMEM + 1024) <= 228 * 1024 && CTAS * TMEM_COLS <= 512, "residency");
    static_assert(!SEQ || L == kSlices * SEQ - kPad, "per-interval geometry");
    static_assert(SEQ || L % 4 == 0, "whole blocks");
};

// Tile t: event, first block (the halo block before its first output).
template <class C> __device__ __forceinline__ void dec1_tile(int t, int &e, int &b0) {
    e = t / C::TPE;
    b0 = t % C::TPE * C::STRIDE - 1;
}

template <class C> __device__ bool dec1_producer(const TcArgs &a, unsigned char *smem, uint64_t *bar, volatile int *abort) {
    uint64_t *full = bar + C::FULL, *empty = bar + C::EMPTY;
    const int ntiles = a.n_events * C::TPE;
    int s = 0, n = 0;
    uint32_t ph = 1;
    bool ok = true;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++n) {
        if (!mbar_wait(&empty[s], ph, abort)) { ok = false; break; }
        int e, b0;
        dec1_tile<C>(t, e, b0);
        unsigned char *dst = smem + C::OFF_A + s * C::A_STAGE;
        // residues 0 and 1: rows hold blocks b0 .. b0 + 128 (x = 0, 1 and 4, 5 one row on), residues 2
        // and 3 blocks b0 - 1 .. b0 + 127 (x = -2, -1 and 2, 3); a block's storage row is block + 1.
        // Rows outside the event's are not copied: only discarded outputs would read them.
        const int lo01 = b0 + 1, lo23 = max(b0, 0), skip23 = lo23 - b0;
        const int n01 = min(C::ROWS, C::RQ - lo01), n23 = min(C::ROWS - skip23, C::RQ - lo23);
        mbar_arrive_expect_tx(&full[s], (uint32_t)(C::PIN * 2 * (n01 + n23) * 16));
        for (int k = 0; k < C::PIN; ++k) {
            const unsigned char *src = k < C::PA ? a.inA : a.inB;
            src += ((size_t)e * C::PA + (k < C::PA ? k : k - C::PA)) * (4 * C::RQ * 16);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int lo = r < 2 ? lo01 : lo23, skip = r < 2 ? 0 : skip23;
                bulk_g2s(dst + (k * 4 + r) * C::PLANE + skip * 16, src + ((size_t)r * C::RQ + lo) * 16,
                         (r < 2 ? n01 : n23) * 16, &full[s]);
            }
        }
        if (++s == C::STAGES) { s = 0; ph ^= 1; }
    }
    // copies still in flight land before the CTA can exit: wait (bounded) for the last ones
    const uint64_t t0 = globaltimer();
    for (int j = max(0, n - C::STAGES); j < n; ++j)
        while (!mbar_try_wait(&full[j % C::STAGES], (j / C::STAGES) & 1))
            if (globaltimer() - t0 > kWaitLimitNs) break;
    while (!mbar_try_wait(bar + C::W, 0))
        if (globaltimer() - t0 > 2 * kWaitLimitNs) break;
    return ok;
}

// The MMAs of one tile into accumulator d.
template <class C> __device__ __forceinline__ void dec1_mmas(uint32_t d, uint32_t as, uint32_t w_base) {
    const uint64_t a0 = smem_desc(as, 4 * C::PLANE, 128), b0 = smem_desc(w_base, 5 * C::COUT * 16, 128);
#pragma unroll
    for (int x = -2; x <= 5; ++x) {
        const int r = x & 3, row = x >= 4 || (x >= 2 && x < 4) ? 1 : 0;    // plane, first row (see the producer)
        const int jlo = x > 2 ? x - 2 : 0, jhi = x + 2 < 3 ? x + 2 : 3;
#pragma unroll
        for (int kb = 0; kb < C::PIN / 2; ++kb) {
            const uint64_t ad = desc_plus(a0, (2 * kb * 4 + r) * C::ROWS + row);
            // columns from output j on: the window starts at tap t = x - j + 2, row 4 - t of the image
            auto mma = [&](int j, int count, bool acc) {
                const uint64_t bd = desc_plus(b0, (2 * kb * 5 + 2 - x + j) * C::COUT);
                const uint32_t id = idesc_f32acc(kTileM, count * C::COUT, C::FMT);
                if constexpr (is16(C::PREC)) mma_f16(d + j * C::COUT, ad, bd, id, acc);
                else mma_fp8(d + j * C::COUT, ad, bd, id, acc);
            };
            if (kb == 0 && x <= 1) {        // output x + 2 starts here
                if (jhi > jlo) mma(jlo, jhi - jlo, true);
                mma(jhi, 1, false);
            } else {
                mma(jlo, jhi - jlo + 1, true);
            }
        }
    }
}

template <class C>
__device__ bool dec1_mma(const TcArgs &a, unsigned char *smem, uint64_t *bar, uint32_t tmem, volatile int *abort) {
    const int ntiles = a.n_events * C::TPE;
    int s = 0, b = 0;
    uint32_t ph_s = 0, ph_b = 1;
    bool ok = mbar_wait(bar + C::W, 0, abort);
    for (int t = blockIdx.x; ok && t < ntiles; t += gridDim.x) {
        if (!mbar_wait(&bar[C::TE + b], ph_b, abort) || !mbar_wait(&bar[C::FULL + s], ph_s, abort)) { ok = false; break; }
        tc_fence_after();
        dec1_mmas<C>(tmem + b * C::COLS, smem_u32(smem + C::OFF_A) + s * C::A_STAGE, smem_u32(smem + C::OFF_W));
        mma_commit(&bar[C::EMPTY + s]);
        mma_commit(&bar[C::TF + b]);
        if (++s == C::STAGES) { s = 0; ph_s ^= 1; }
        if (++b == C::NB) { b = 0; ph_b ^= 1; }
    }
    // every MMA issued above completes before TMEM is released
    mma_commit(bar + C::DRAIN);
    const uint64_t t0 = globaltimer();
    while (!mbar_try_wait(bar + C::DRAIN, 0)) if (globaltimer() - t0 > kWaitLimitNs) break;
    return ok;
}

template <class C, bool CAL>
__device__ bool dec1_epilogue(const TcArgs &a, unsigned char *smem, uint64_t *bar, uint32_t tmem, volatile int *abort,
                              int wg, int m) {
    const float *par = reinterpret_cast<const float *>(smem + C::OFF_PAR);
    const float *sbias = par, *scs = par + C::COUT, *sfin = par + 2 * C::COUT;
    const int lane = m & 31, w = m >> 5;
    const uint32_t lane_tmem = tmem + ((uint32_t)(w * 32) << 16);
    float *sx = reinterpret_cast<float *>(smem + C::OFF_X) + wg * 64;
    const int ntiles = a.n_events * C::TPE;
    int n = 0;                                      // this warpgroup's tiles: every EWG-th of the CTA's
    for (int i = wg, t = (int)blockIdx.x + wg * (int)gridDim.x; t < ntiles;
         i += C::EWG, t += C::EWG * (int)gridDim.x, ++n) {
        const int b = i % C::NB;
        int e, b0;
        dec1_tile<C>(t, e, b0);
        const int blk = b0 + m, p0 = 4 * blk;
        unsigned in = 0;                            // the block's positions inside the event (and a sequence)
        int sq[4], jq[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int p = p0 + j;
            sq[j] = 0;
            jq[j] = p;
            if constexpr (C::SEQ != 0) {
                sq[j] = (p + kPad) / C::SEQ;
                jq[j] = (p + kPad) % C::SEQ - kPad;
            }
            if (p >= 0 && p < C::L && jq[j] >= 0 && jq[j] < C::LSEQ) in |= 1u << j;
        }
        const bool whole = __all_sync(0xffffffffu, in == 15u);
        if (!mbar_wait(&bar[C::TF + b], (i / C::NB) & 1, abort)) return false;
        tc_fence_after();
        const uint32_t dcol = lane_tmem + b * C::COLS;
        // partial sums of the final conv per position: taps (0, 1), (2, 3) as pairs, and 4
        float2 g01[4], g23[4];
        float g4[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            g01[j] = g23[j] = make_float2(0.0f, 0.0f);
            g4[j] = 0.0f;
        }
#pragma unroll 1
        for (int c0 = 0; c0 < C::COUT; c0 += 8) {
            float v[4][8], bj[8], w4[8];
            tmem_ld8x4(dcol + c0, C::COUT, v);
            if (c0 + 8 >= C::COUT) {
                tc_fence_before();
                mbar_arrive(&bar[C::TE + b]);
            }
            lds8(sbias + c0, bj);
            if constexpr (is16(C::PREC)) {
#pragma unroll
                for (int j = 0; j < 4; ++j) bias_leaky(v[j], bj);
            } else {
                float sc[8];
                lds8(scs + c0, sc);
#pragma unroll
                for (int j = 0; j < 4; ++j) scale_bias_leaky(v[j], sc, bj);
            }
            if (!whole) {                           // zero padding outside the event or its sequence
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int c = 0; c < 8; ++c) v[j][c] = (in >> j) & 1u ? v[j][c] : 0.0f;
            }
            if constexpr (CAL) {
#pragma unroll
                for (int j = 0; j < 4; ++j) amax_fold(a.amax, a.amax_out, v[j], true);
            }
            // channels in order; taps (0, 1) and (2, 3) as packed FMAs (each lane an fmaf), from weights
            // stored per channel as (w0, w1, w2, w3), then tap 4
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const float4 wt = reinterpret_cast<const float4 *>(sfin)[c0 + c];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float2 vv = make_float2(v[j][c], v[j][c]);
                    g01[j] = __ffma2_rn(make_float2(wt.x, wt.y), vv, g01[j]);
                    g23[j] = __ffma2_rn(make_float2(wt.z, wt.w), vv, g23[j]);
                }
            }
            lds8(sfin + 4 * C::COUT + c0, w4);
#pragma unroll
            for (int c = 0; c < 8; ++c)
#pragma unroll
                for (int j = 0; j < 4; ++j) g4[j] = fmaf(w4[c], v[j][c], g4[j]);
        }
        // the six partial sums that the neighbouring blocks use: from the next lanes, and through
        // shared memory (two buffers) between the warps
        float up0 = __shfl_up_sync(0xffffffffu, g01[2].x, 1), up1 = __shfl_up_sync(0xffffffffu, g01[3].x, 1),
              up2 = __shfl_up_sync(0xffffffffu, g01[3].y, 1);
        float dn0 = __shfl_down_sync(0xffffffffu, g4[0], 1), dn1 = __shfl_down_sync(0xffffffffu, g23[0].y, 1),
              dn2 = __shfl_down_sync(0xffffffffu, g4[1], 1);
        float *x = sx + (n & 1) * 32;
        if (lane == 31) {
            x[w * 8] = g01[2].x; x[w * 8 + 1] = g01[3].x; x[w * 8 + 2] = g01[3].y;
        } else if (lane == 0) {
            x[w * 8 + 4] = g4[0]; x[w * 8 + 5] = g23[0].y; x[w * 8 + 6] = g4[1];
        }
        mbar_arrive(&bar[C::XR + wg]);
        if (!mbar_wait(&bar[C::XR + wg], n & 1, abort)) return false;
        if (lane == 0 && w > 0) {
            up0 = x[w * 8 - 8]; up1 = x[w * 8 - 7]; up2 = x[w * 8 - 6];
        } else if (lane == 31 && w < 3) {
            dn0 = x[w * 8 + 12]; dn1 = x[w * 8 + 13]; dn2 = x[w * 8 + 14];
        }
        if (m < 1 || m > C::STRIDE || in == 0) continue;
        // f(p) = b + sum_t g_t(p + t - 2), in tap order
        const float fb = sfin[5 * C::COUT];
        float f[4];
        f[0] = fb + up0; f[0] += up2; f[0] += g23[0].x; f[0] += g23[1].y; f[0] += g4[2];
        f[1] = fb + up1; f[1] += g01[0].y; f[1] += g23[1].x; f[1] += g23[2].y; f[1] += g4[3];
        f[2] = fb + g01[0].x; f[2] += g01[1].y; f[2] += g23[2].x; f[2] += g23[3].y; f[2] += dn0;
        f[3] = fb + g01[1].x; f[3] += g01[2].y; f[3] += g23[3].x; f[3] += dn1; f[3] += dn2;
        if constexpr (C::SEQ != 0) {
            // the logits of an interval's bins are its sequence's central positions
            // [kIvPad, kIvPad + kSliceBins)
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (((in >> j) & 1u) && jq[j] >= kIvPad && jq[j] < kIvPad + kSliceBins)
                    a.logits[(size_t)e * kBins + sq[j] * kSliceBins + jq[j] - kIvPad] = f[j];
        } else {
            float *out = a.logits + (size_t)e * C::L + p0;
            if ((reinterpret_cast<uintptr_t>(a.logits) & 15) == 0) {
                *reinterpret_cast<float4 *>(out) = make_float4(f[0], f[1], f[2], f[3]);
            } else {                                // a caller's buffer, aligned to 4 bytes only
#pragma unroll
                for (int j = 0; j < 4; ++j) out[j] = f[j];
            }
        }
    }
    return true;
}

template <class C, bool CAL> __global__ void __launch_bounds__(C::THREADS, C::CTAS) k_dec1_tc(TcArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + C::OFF_BAR);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bar + C::NBAR);
    volatile int *abort = reinterpret_cast<volatile int *>(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float *par = reinterpret_cast<float *>(smem + C::OFF_PAR);
    for (int k = threadIdx.x; k < C::NPAR; k += C::THREADS) {
        float v;
        if (k < C::COUT) v = a.bias[k];
        else if (k < 2 * C::COUT) v = a.cs ? a.cs[k - C::COUT] : 1.0f;
        else {   // the final conv: (w0, w1, w2, w3) per channel, then w4 per channel, then b
            const int f = k - 2 * C::COUT;
            v = f < 4 * C::COUT ? a.final_w[(f & 3) * C::COUT + (f >> 2)] : a.final_w[f];
        }
        par[k] = v;
    }
    if (threadIdx.x == 0) {
        for (int b = 0; b < C::NBAR; ++b)
            mbar_init(&bar[b], (b >= C::TE && b < C::TE + C::NB) || (b >= C::XR && b < C::XR + C::EWG) ? 128 : 1);
        *abort = 0;
        fence_mbar_init();
        // the weights are the handle's: they load before the previous kernel has finished
        mbar_arrive_expect_tx(bar + C::W, C::W_BYTES);
        bulk_g2s(smem + C::OFF_W, a.w, C::W_BYTES, bar + C::W);
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, C::TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    grid_dep_wait();
    grid_dep_launch();
    TcArgs r = a;
    r.n_events = launch_events(a.n_dyn, a.dyn_base, a.n_events);
    bool ok = true;
    if (warp == 0) {
        if (lane == 0) ok = dec1_producer<C>(r, smem, bar, abort);
    } else if (warp == 1) {
        if (lane == 0) ok = dec1_mma<C>(r, smem, bar, tmem, abort);
    } else {
        ok = dec1_epilogue<C, CAL>(r, smem, bar, tmem, abort, (warp - 2) >> 2, (warp & 3) * 32 + lane);
    }
    if (!ok) {
        *abort = 1;
        raise_status(a.status, PVF_ERR_TIMEOUT);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tmem, C::TMEM_COLS);
}

template <class C, bool CAL = false>
cudaError_t launch_dec1(const TcArgs &a, cudaStream_t s, const ProfHook *prof, int cap) {
    if constexpr (C::PREC == PVF_BF16 && !CAL)
        if (a.amax) return launch_dec1<C, true>(a, s, prof, cap);        // calibration runs in the BF16 form
    if (a.n_events <= 0) return cudaSuccess;
    // the shared-memory request is padded so that no more CTAs fit an SM than its tensor memory
    // serves (an allocation would otherwise wait for a neighbour)
    constexpr int kFit = 512 / C::TMEM_COLS;
    constexpr int pad = 228 * 1024 / kFit - 1024;
    constexpr int smem = C::SMEM > pad ? C::SMEM : pad;
    static_assert(smem <= 227 * 1024, "shared memory");
    int sms = 0;
    cudaError_t err = current_device_sms(&sms);
    if (err == cudaSuccess) err = prepare_kernel((const void *)k_dec1_tc<C, CAL>, (size_t)smem, nullptr);
    if (err != cudaSuccess) return err;
    const int per_sm = cap > 0 && cap < C::CTAS ? cap : C::CTAS;
    const int64_t tiles = (int64_t)a.n_events * C::TPE;
    const int grid = tiles < (int64_t)sms * per_sm ? (int)tiles : sms * per_sm;
    ProfScope ps(prof, "dec1_final", s);
    return launch_pdl(k_dec1_tc<C, CAL>, dim3(grid), dim3(C::THREADS), (size_t)smem, s, a);
}
