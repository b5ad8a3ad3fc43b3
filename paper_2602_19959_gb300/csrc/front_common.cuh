// Device code shared by the front kernels (k_front.cu: CUDA-core FC for the FP32 form and
// the static-scratch histogram; k_front_tc.cu: tcgen05 FC for the tensor-core forms):
// event validation, the stable slice sort, and enc1 + pool with its stores.
#pragma once

#include "pvf_internal.cuh"

namespace pvf {
namespace front {

__device__ __forceinline__ float softplus_f(float x) { return x > 20.0f ? x : log1pf(expf(x)); }

// Slice of a float32 z (round-to-nearest add and divide); -1 when outside [0, 40).
__device__ __forceinline__ int slice_of(float z) {
    float q = __fdiv_rn(__fadd_rn(z, 100.0f), 10.0f);
    if (!(q >= 0.0f && q < 40.0f)) return -1;
    return (int)floorf(q);
}

// Stores the 16 channels of plane-major storage row `row` of event e (two 16-bit planes, one e4m3
// plane).
template <class T>
__device__ __forceinline__ void store_row16(void *base, int64_t e, int64_t rows_e, int64_t row,
                                            const float v[kC0], float inv_scale) {
    if constexpr (sizeof(T) == 2) {
        unsigned char *cb = reinterpret_cast<unsigned char *>(base);
        *reinterpret_cast<uint4 *>(cb + planar_off(e, 0, 2, rows_e, row)) = pack8<T>(v);
        *reinterpret_cast<uint4 *>(cb + planar_off(e, 1, 2, rows_e, row)) = pack8<T>(v + 8);
    } else {
        uint4 pk;
        pack_e4m3<16>(v, inv_scale, reinterpret_cast<uint32_t *>(&pk));
        unsigned char *cb = reinterpret_cast<unsigned char *>(base);
        *reinterpret_cast<uint4 *>(cb + planar_off(e, 0, 1, rows_e, row)) = pk;
    }
}

// Channels [16 g, 16 g + 16) of position p of event e in a quad-layout tensor of C0 channels
// and `rows` rows per residue plane.
template <class T, int C0>
__device__ __forceinline__ void store_seg16_quad(void *base, int64_t e, int rows, int p, int g, const float v[16],
                                                 float inv_scale) {
    unsigned char *cb = reinterpret_cast<unsigned char *>(base);
    if constexpr (sizeof(T) == 2) {
        *reinterpret_cast<uint4 *>(cb + quad_off(e, 2 * g, C0 / 8, rows, p)) = pack8<T>(v);
        *reinterpret_cast<uint4 *>(cb + quad_off(e, 2 * g + 1, C0 / 8, rows, p)) = pack8<T>(v + 8);
    } else {
        uint4 pk;
        pack_e4m3<16>(v, inv_scale, reinterpret_cast<uint32_t *>(&pk));
        *reinterpret_cast<uint4 *>(cb + quad_off(e, g, C0 / 16, rows, p)) = pk;
    }
}
// All channels of position p set to zero.
template <class T, int C0> __device__ __forceinline__ void zero_quad(void *base, int64_t e, int rows, int p) {
    unsigned char *cb = reinterpret_cast<unsigned char *>(base);
    constexpr int P = C0 * (int)sizeof(T) / 16;
#pragma unroll
    for (int k = 0; k < P; ++k) *reinterpret_cast<uint4 *>(cb + quad_off(e, k, P, rows, p)) = make_uint4(0, 0, 0, 0);
}

// Channels [16 g, 16 g + 16) of storage row `row` of event e in a plane-major tensor of C0
// channels (16-bit: planes 2 g and 2 g + 1 of C0 / 8; e4m3: plane g of C0 / 16).
template <class T, int C0>
__device__ __forceinline__ void store_seg16_pm(void *base, int64_t e, int64_t rows_e, int64_t row, int g,
                                               const float v[16], float inv_scale) {
    unsigned char *cb = reinterpret_cast<unsigned char *>(base);
    if constexpr (sizeof(T) == 2) {
        *reinterpret_cast<uint4 *>(cb + planar_off(e, 2 * g, C0 / 8, rows_e, row)) = pack8<T>(v);
        *reinterpret_cast<uint4 *>(cb + planar_off(e, 2 * g + 1, C0 / 8, rows_e, row)) = pack8<T>(v + 8);
    } else {
        uint4 pk;
        pack_e4m3<16>(v, inv_scale, reinterpret_cast<uint32_t *>(&pk));
        *reinterpret_cast<uint4 *>(cb + planar_off(e, g, C0 / 16, rows_e, row)) = pk;
    }
}

template <class T>
__device__ __forceinline__ void zero_row16(void *base, int64_t e, int64_t rows_e, int64_t row) {
    float z[kC0];
#pragma unroll
    for (int i = 0; i < kC0; ++i) z[i] = 0.0f;
    store_row16<T>(base, e, rows_e, row, z, 1.0f);
}

// Sorted entries: bits 0-13 hold the track's index within the event, bits 14-15 the
// slice the entry fills relative to the track's own: 0 its own, 1 the slice below, 2 the
// slice above (the second slice of a boundary track, §3). sslice[t] holds the track's own
// slice in bits 0-5 and that tag in bits 6-7; 255 marks a dropped track.
// Without boundary tracks (EDGE = false) an entry is the track index and sslice[t] its
// slice: the kernels are then instantiated without any of this decoding.
constexpr int kEntTrack = 0x3FFF;
template <bool EDGE>
__device__ __forceinline__ int entry_track(int en) {
    return EDGE ? (en & kEntTrack) : en;
}
template <bool EDGE>
__device__ __forceinline__ int entry_slice(int en, const uint8_t *sslice) {
    if constexpr (!EDGE) {
        return sslice[en];
    } else {
        const int d = en >> 14;
        return (int)(sslice[en & kEntTrack] & 63u) - (d & 1) + (d >> 1);
    }
}

// Steps a-c for event ge: validation (bypass flag), slice per track, stable counting
// sort by slice. On return (after a block barrier) ssorted[0..nvalid) holds the event's
// entries grouped by slice, sseg[s]..sseg[s+1] bounding slice s: within a slice, first
// the slice's own valid tracks in input order, then the boundary tracks of the two
// neighbouring slices that also fill it (a.edge > 0), in input order. A valid track of
// slice s whose slice-relative z (float32) is below a.edge also fills s - 1 (s > 0); one
// at or above a.edge_hi = 10 - a.edge also fills s + 1 (s < 39).
// EDGE = false: no boundary tracks (a.edge is 0). scnt/srun must hold 48 ints each.
// SPLIT: an event shared by `nrank` blocks (a power of two), of which this one takes the slices
// s = rank modulo nrank: the other slices come out empty.
// Every thread of the block must call this.
template <int NT, bool EDGE, bool SPLIT = false>
__device__ __forceinline__ void validate_sort(const FrontArgs &a, int ge, int tid, int *scnt, int *sseg,
                                              int *srun, uint16_t *ssorted, uint8_t *sslice,
                                              int64_t &t0_out, int &nvalid_out, int rank = 0, int nrank = 1) {
    const auto own = [&](int s) { return !SPLIT || (s & (nrank - 1)) == rank; };
    const int src = a.ev_index ? a.ev_index[ge] : ge;      // gathered events: store index
    const int64_t t0 = a.offsets[src], t1 = a.offsets[src + 1];
    const bool bypass = t0 < 0 || t1 < t0 || t1 > a.n_tracks || (t1 - t0) > a.max_tracks;
    const int n = bypass ? 0 : (int)(t1 - t0);
    if (tid == 0) {
        a.ev_flag[ge] = bypass ? 1 : 0;
        if (bypass) raise_status(a.status, PVF_WARN_EVENTS_SKIPPED);
    }
    if (tid < 48) { scnt[tid] = 0; srun[tid] = 0; }
    __syncthreads();
    // slice per track (integer counts through shared atomics: exact)
    for (int t = tid; t < n; t += NT) {
        const int64_t gt = t0 + t;
        bool finite = true;
#pragma unroll
        for (int k = 0; k < kFeatures; ++k) finite &= isfinite(a.feat[k][gt]);
        const float z = a.feat[2][gt];
        const int s = finite ? slice_of(z) : -1;
        int tag = 0;
        if (s >= 0) {
            if (own(s)) atomicAdd(&scnt[s], 1);
            if constexpr (EDGE) {
                const float zr = __fsub_rn(z, -100.0f + 10.0f * (float)s);   // as feature 2
                if (s > 0 && zr < a.edge) tag = 1;
                else if (s < kSlices - 1 && zr >= a.edge_hi) tag = 2;
                const int s2 = s - (tag & 1) + (tag >> 1);
                if (tag && own(s2)) atomicAdd(&scnt[s2], 1);
            }
        }
        sslice[t] = s < 0 ? 255 : (uint8_t)(s | (tag << 6));
    }
    __syncthreads();
    // warp 0: the slices' bounds (a scan with two slices per lane; one thread adding them up took
    // 1400 cycles), then stable ranks by slice, walking the tracks in input order, once for their
    // own slices and once more for the second slices of boundary tracks
    if (tid < 32) {
        const unsigned lane = tid;
        static_assert(kSlices % 2 == 0 && kSlices <= 64, "two slices per lane");
        const int a0 = scnt[2 * lane < kSlices ? 2 * lane : kSlices], a1 = scnt[2 * lane < kSlices ? 2 * lane + 1 : kSlices];
        int incl = a0 + a1;          // scnt[kSlices] is 0
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if ((int)lane >= o) incl += y;
        }
        if (2 * lane < kSlices) {
            sseg[2 * lane] = incl - a0 - a1;
            sseg[2 * lane + 1] = incl - a1;
        }
        if (lane == 31) sseg[kSlices] = incl;
        __syncwarp();
#pragma unroll 1
        for (int pass = 0; pass < (EDGE ? 2 : 1); ++pass) {
            for (int base = 0; base < n; base += 32) {
                const int t = base + lane;
                int s = 255, en = t;
                if constexpr (!EDGE) {
                    if (t < n) s = sslice[t];
                } else if (t < n && sslice[t] != 255) {
                    const int own = sslice[t] & 63, tag = sslice[t] >> 6;
                    if (pass == 0) {
                        s = own;
                    } else if (tag) {
                        s = own - (tag & 1) + (tag >> 1);
                        en = t | (tag << 14);
                    }
                }
                if (!own(s)) s = 255;
                const unsigned peers = __match_any_sync(0xffffffffu, s);
                const unsigned lower = peers & ((1u << lane) - 1u);
                int before = 0;
                if (s != 255) before = srun[s];
                __syncwarp();
                if (s != 255) {
                    ssorted[sseg[s] + before + __popc(lower)] = (uint16_t)en;
                    if (lower == 0) srun[s] = before + __popc(peers);
                }
                __syncwarp();
            }
        }
    }
    __syncthreads();
    t0_out = t0;
    nvalid_out = sseg[kSlices];
}

// The nine features of track gt with feature 2 made slice-relative (exact offset).
__device__ __forceinline__ void track_features(const FrontArgs &a, int64_t gt, int s, float x[kFcInPad]) {
#pragma unroll
    for (int k = 0; k < kFeatures; ++k) x[k] = a.feat[k][gt];
    x[2] = __fsub_rn(x[2], -100.0f + 10.0f * (float)s);
#pragma unroll
    for (int k = kFeatures; k < kFcInPad; ++k) x[k] = 0.0f;
}

// Stores channels [8 h, 8 h + 8) of storage row `row` of event e: one of the two 16-bit planes, or
// half of the e4m3 plane's 16-byte row.
template <class T>
__device__ __forceinline__ void store_half8(void *base, int64_t e, int64_t rows_e, int64_t row, int h,
                                            const float v[8], float inv_scale) {
    if constexpr (sizeof(T) == 2) {
        *reinterpret_cast<uint4 *>(reinterpret_cast<unsigned char *>(base) + planar_off(e, h, 2, rows_e, row)) =
            pack8<T>(v);
    } else {
        uint2 pk;
        pack_e4m3<8>(v, inv_scale, reinterpret_cast<uint32_t *>(&pk));
        *reinterpret_cast<uint2 *>(reinterpret_cast<unsigned char *>(base) + planar_off(e, 0, 1, rows_e, row) + 8 * h) = pk;
    }
}

// Step f: e1 = LeakyReLU(conv_k5(hist) + b), p1 = maxpool2(e1), stored in the form's
// precision with the pad rows zeroed; calibration (AMAX) folds max |e1| into a.amax[0].
// Thread tid owns channels [8 h, 8 h + 8), h = tid & 1, of every position pair it takes,
// so its 40 weights and 8 biases stay in registers and the loop reads only the histogram
// from shared memory; the two threads of a pair write the two halves of each row.
// This is the per-interval layout of the tensor-core forms: e1 and p1 hold the event's kSlices
// sequences end to end, each the conv of the interval's kIvLen-bin window (its bins with
// kIvPad zero bins on each side), two zero rows before each sequence and two after the
// last (neighbouring sequences share the two between them).
template <class T, bool AMAX>
__device__ __forceinline__ void enc1_pool_t(const FrontArgs &a, int e, int tid, int nt, const float *shist,
                                            const float *senc) {
    constexpr int S1 = kIvLen + kPad, S2 = kIvLen / 2 + kPad;   // rows per sequence
    constexpr int RQ = quad_rows(kSlices * S1 - kPad);     // e1: the quad layout
    constexpr int64_t rows2 = (int64_t)kSlices * S2 + kPad;
    constexpr int NQ = kSlices * (kIvLen / 2);         // position pairs
    const float inv = a.e1_inv_scale;
    const int h = tid & 1;
    float w[5][8], bias[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
#pragma unroll
        for (int t = 0; t < 5; ++t) w[t][j] = senc[t * kC0 + 8 * h + j];
        bias[j] = senc[5 * kC0 + 8 * h + j];
    }
    float vmax = 0.0f;
#pragma unroll 2   // two position pairs in flight per thread: front 81.6 -> 79.5 us (FP16)
    for (int qi = tid >> 1; qi < NQ; qi += nt / 2) {
        // the pair's sequence and first position; e1 positions p1, p1 + 1, p1 row r2
        const int sq = qi / (kIvLen / 2), q = qi % (kIvLen / 2);
        const int p1 = sq * S1 + 2 * q;
        const int64_t r2 = (int64_t)sq * S2 + q + kPad;
        float hv[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const int b = 2 * q + k - 2 - kIvPad;    // bin of the interval at window position
            hv[k] = (b >= 0 && b < kSliceBins) ? shist[sq * kSliceBins + b] : 0.0f;
        }
        float v0[8], v1[8];
        // channel pairs (j, j + 1) as one packed two-lane FMA (each lane an fmaf, in the
        // same tap order): half the FMA instructions, identical results
#pragma unroll
        for (int j = 0; j < 8; j += 2) {
            float2 a0 = make_float2(bias[j], bias[j + 1]), a1 = a0;
#pragma unroll
            for (int t = 0; t < 5; ++t) {
                const float2 wt = make_float2(w[t][j], w[t][j + 1]);
                a0 = __ffma2_rn(wt, make_float2(hv[t], hv[t]), a0);
                a1 = __ffma2_rn(wt, make_float2(hv[t + 1], hv[t + 1]), a1);
            }
            a0 = leaky2(a0);
            a1 = leaky2(a1);
            v0[j] = a0.x; v0[j + 1] = a0.y;
            v1[j] = a1.x; v1[j + 1] = a1.y;
        }
        if constexpr (AMAX) {
#pragma unroll
            for (int j = 0; j < 8; ++j) vmax = fmaxf(vmax, fmaxf(fabsf(v0[j]), fabsf(v1[j])));
        }
        if constexpr (sizeof(T) == 2) {
            // the pooled row from the packed rows: the maximum of the rounded values is the
            // rounded maximum
            const uint4 r0 = pack8<T>(v0), r1v = pack8<T>(v1);
            unsigned char *d1 = reinterpret_cast<unsigned char *>(a.e1) + quad_off(e, h, 2, RQ, p1);
            *reinterpret_cast<uint4 *>(d1) = r0;
            *reinterpret_cast<uint4 *>(d1 + RQ * 16) = r1v;       // the next residue: p1 is even
            *reinterpret_cast<uint4 *>(reinterpret_cast<unsigned char *>(a.p1) + planar_off(e, h, 2, rows2, r2)) =
                make_uint4(max2<T>(r0.x, r1v.x), max2<T>(r0.y, r1v.y), max2<T>(r0.z, r1v.z), max2<T>(r0.w, r1v.w));
        } else {
            float vp[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) vp[j] = fmaxf(v0[j], v1[j]);
            unsigned char *d1 = reinterpret_cast<unsigned char *>(a.e1) + quad_off(e, 0, 1, RQ, p1) + 8 * h;
            uint2 pk;
            pack_e4m3<8>(v0, inv, reinterpret_cast<uint32_t *>(&pk));
            *reinterpret_cast<uint2 *>(d1) = pk;
            pack_e4m3<8>(v1, inv, reinterpret_cast<uint32_t *>(&pk));
            *reinterpret_cast<uint2 *>(d1 + RQ * 16) = pk;
            store_half8<T>(a.p1, e, rows2, r2, h, vp, inv);
        }
    }
    if constexpr (AMAX) {   // calibration: integer max on the float bits (order-independent)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
        if ((tid & 31) == 0) atomicMax(reinterpret_cast<int *>(a.amax), __float_as_int(vmax));
    }
    for (int idx = tid; idx < (kSlices + 1) * 2; idx += nt) {   // the two rows before each sequence and after the last
        const int sq = idx >> 1, k = idx & 1;
        zero_quad<T, kC0>(a.e1, e, RQ, sq * S1 + k - kPad);
        zero_row16<T>(a.p1, e, rows2, (int64_t)sq * S2 + k);
    }
}

// The same for whole events of the tensor-core forms, four positions per step: they share their
// eight histogram bins (shist is zero for two bins on either side), their addresses (one row of
// the four residue planes of e1, two rows of p1) and, in registers, the weights of the thread's 8
// channels. Same arithmetic per position as enc1_pool_t.
template <class T, bool AMAX>
__device__ __forceinline__ void enc1_pool_quads(const FrontArgs &a, int e, int tid, int nt, const float *shist,
                                                const float *senc) {
    static_assert(sizeof(T) <= 2 && kBins % 4 == 0, "plane-major forms");
    constexpr int RQ = quad_rows(kBins);
    constexpr int P = kC0 * (int)sizeof(T) / 16;                          // planes: 2, or 1 of e4m3
    const int64_t rows2 = padded_rows(kBins / 2);
    const float inv = a.e1_inv_scale;
    const int h = tid & 1;
    float2 w[5][4], bias[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
        for (int t = 0; t < 5; ++t) w[t][j] = make_float2(senc[t * kC0 + 8 * h + 2 * j], senc[t * kC0 + 8 * h + 2 * j + 1]);
        bias[j] = make_float2(senc[5 * kC0 + 8 * h + 2 * j], senc[5 * kC0 + 8 * h + 2 * j + 1]);
    }
    float vmax = 0.0f;
    constexpr int half = sizeof(T) == 2 ? 0 : 8;                          // e4m3: half a plane's row per thread
    unsigned char *e1 = reinterpret_cast<unsigned char *>(a.e1) + quad_off(e, P == 2 ? h : 0, P, RQ, 0) + half * h;
    unsigned char *p1 = reinterpret_cast<unsigned char *>(a.p1) + planar_off(e, P == 2 ? h : 0, P, rows2, kPad) + half * h;
#pragma unroll 1
    for (int q = tid >> 1; q < kBins / 4; q += nt / 2) {
        float hv[8];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float2 x = *reinterpret_cast<const float2 *>(shist + 4 * q - 2 + 2 * k);
            hv[2 * k] = x.x;
            hv[2 * k + 1] = x.y;
        }
        float v[4][8];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float2 acc = bias[j];
#pragma unroll
                for (int t = 0; t < 5; ++t) acc = __ffma2_rn(w[t][j], make_float2(hv[i + t], hv[i + t]), acc);
                acc = leaky2(acc);
                v[i][2 * j] = acc.x;
                v[i][2 * j + 1] = acc.y;
                if constexpr (AMAX) vmax = fmaxf(vmax, fmaxf(fabsf(acc.x), fabsf(acc.y)));
            }
        if constexpr (sizeof(T) == 2) {
            uint4 r[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                r[i] = pack8<T>(v[i]);
                *reinterpret_cast<uint4 *>(e1 + (size_t)(i * RQ + q) * 16) = r[i];
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)     // the maximum of the rounded values is the rounded maximum
                *reinterpret_cast<uint4 *>(p1 + (size_t)(2 * q + i) * 16) =
                    make_uint4(max2<T>(r[2 * i].x, r[2 * i + 1].x), max2<T>(r[2 * i].y, r[2 * i + 1].y),
                               max2<T>(r[2 * i].z, r[2 * i + 1].z), max2<T>(r[2 * i].w, r[2 * i + 1].w));
        } else {
            uint2 r[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                pack_e4m3<8>(v[i], inv, reinterpret_cast<uint32_t *>(&r[i]));
                *reinterpret_cast<uint2 *>(e1 + (size_t)(i * RQ + q) * 16) = r[i];
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
                *reinterpret_cast<uint2 *>(p1 + (size_t)(2 * q + i) * 16) =
                    make_uint2(max4_e4m3(r[2 * i].x, r[2 * i + 1].x), max4_e4m3(r[2 * i].y, r[2 * i + 1].y));
        }
    }
    if constexpr (AMAX) {   // calibration: integer max on the float bits (order-independent)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
        if ((tid & 31) == 0) atomicMax(reinterpret_cast<int *>(a.amax), __float_as_int(vmax));
    }
    if (tid < 4) {
        zero_quad<T, kC0>(a.e1, e, RQ, tid < 2 ? tid - kPad : kBins + tid - kPad);   // -2, -1 and L, L + 1
        zero_row16<T>(a.p1, e, rows2, tid < 2 ? tid : kBins / 2 + tid);
    }
}

// Step f of the wide network's tensor-core forms, the weights read from shared memory per position
// pair (same arithmetic, same order). senc holds W[t][co] (5 C0 floats) then b[co]; the C0 channels
// are produced 16 at a time, two to a packed FMA.
template <class T, bool AMAX, int C0>
__device__ __forceinline__ void enc1_pool_shared_t(const FrontArgs &a, int e, int tid, int nt, const float *shist,
                                                   const float *senc) {
    static_assert(C0 % 16 == 0 && sizeof(T) <= 2, "16-channel segments, plane-major forms");
    const int64_t rows2 = padded_rows(kBins / 2);
    const float inv = a.e1_inv_scale;
    float vmax = 0.0f;
    for (int q = tid; q < kBins / 2; q += nt) {
        float hv[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const int p = 2 * q + k - 2;
            hv[k] = (p >= 0 && p < kBins) ? shist[p] : 0.0f;
        }
#pragma unroll 1
        for (int g = 0; g < C0 / 16; ++g) {
            float v0[16], v1[16], vp[16];
#pragma unroll
            for (int j = 0; j < 16; j += 2) {
                const float *wj = senc + 16 * g + j;
                float2 a0 = *reinterpret_cast<const float2 *>(wj + 5 * C0), a1 = a0;
#pragma unroll
                for (int t = 0; t < 5; ++t) {
                    const float2 w = *reinterpret_cast<const float2 *>(wj + t * C0);
                    a0 = __ffma2_rn(w, make_float2(hv[t], hv[t]), a0);
                    a1 = __ffma2_rn(w, make_float2(hv[t + 1], hv[t + 1]), a1);
                }
                a0 = leaky2(a0);
                a1 = leaky2(a1);
                v0[j] = a0.x; v0[j + 1] = a0.y;
                v1[j] = a1.x; v1[j + 1] = a1.y;
                vp[j] = fmaxf(a0.x, a1.x);
                vp[j + 1] = fmaxf(a0.y, a1.y);
                if constexpr (AMAX)
                    vmax = fmaxf(fmaxf(vmax, fmaxf(fabsf(a0.x), fabsf(a1.x))), fmaxf(fabsf(a0.y), fabsf(a1.y)));
            }
            store_seg16_quad<T, C0>(a.e1, e, quad_rows(kBins), 2 * q, g, v0, inv);
            store_seg16_quad<T, C0>(a.e1, e, quad_rows(kBins), 2 * q + 1, g, v1, inv);
            store_seg16_pm<T, C0>(a.p1, e, rows2, q + kPad, g, vp, inv);
        }
    }
    if constexpr (AMAX) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
        if ((tid & 31) == 0) atomicMax(reinterpret_cast<int *>(a.amax), __float_as_int(vmax));
    }
    if (tid < 4) {
        const float z[16] = {};
        zero_quad<T, C0>(a.e1, e, quad_rows(kBins), tid < 2 ? tid - kPad : kBins + tid - kPad);
        for (int g = 0; g < C0 / 16; ++g)
            store_seg16_pm<T, C0>(a.p1, e, rows2, tid < 2 ? tid : kBins / 2 + tid, g, z, 1.0f);
    }
}

// Step f of the float32 form, channel-last rows, by `nt` threads (several blocks of an event where
// they share it). Thread tid owns channels [4 h, 4 h + 4), h = tid modulo C0 / 4, of every position
// pair it takes: its 20 weights and 4 biases stay in registers (read from shared memory per pair
// they bound the step), and the threads of a pair write whole rows. Same arithmetic per position
// as the other forms. IV: the per-interval layout, kSlices sequences per event (sequence
// e * kSlices + s = interval s), each the conv of the interval's kIvLen-bin window -- the
// interval's bins with kIvPad zero bins on each side -- with zero padding beyond the window, as
// each interval runs the UNet on its own.
template <int C0, bool IV>
__device__ __forceinline__ void enc1_pool_f32(const FrontArgs &a, int e, int tid, int nt, const float *shist,
                                              const float *senc) {
    constexpr int H = C0 / 4, L = IV ? kIvLen : kBins, Q = L / 2, NS = IV ? kSlices : 1;
    const int64_t rows1 = padded_rows(L), rows2 = padded_rows(Q);
    const int h = tid % H;
    float2 w[5][2], bias[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
#pragma unroll
        for (int t = 0; t < 5; ++t) w[t][j] = *reinterpret_cast<const float2 *>(senc + t * C0 + 4 * h + 2 * j);
        bias[j] = *reinterpret_cast<const float2 *>(senc + 5 * C0 + 4 * h + 2 * j);
    }
    float *e1 = reinterpret_cast<float *>(a.e1) + (int64_t)e * NS * rows1 * C0 + 4 * h;
    float *p1 = reinterpret_cast<float *>(a.p1) + (int64_t)e * NS * rows2 * C0 + 4 * h;
    for (int idx = tid / H; idx < NS * Q; idx += nt / H) {
        const int s = IV ? idx / Q : 0, q = IV ? idx % Q : idx;
        float hv[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const int b = 2 * q + k - 2 - (IV ? kIvPad : 0);      // bin of the event, or of the interval
            hv[k] = (b >= 0 && b < (IV ? kSliceBins : kBins)) ? shist[s * kSliceBins + b] : 0.0f;
        }
        float4 v[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            float2 acc[2] = {bias[0], bias[1]};
#pragma unroll
            for (int t = 0; t < 5; ++t)
#pragma unroll
                for (int j = 0; j < 2; ++j) acc[j] = __ffma2_rn(w[t][j], make_float2(hv[i + t], hv[i + t]), acc[j]);
            acc[0] = leaky2(acc[0]);
            acc[1] = leaky2(acc[1]);
            v[i] = make_float4(acc[0].x, acc[0].y, acc[1].x, acc[1].y);
            *reinterpret_cast<float4 *>(e1 + ((int64_t)s * rows1 + 2 * q + i + kPad) * C0) = v[i];
        }
        *reinterpret_cast<float4 *>(p1 + ((int64_t)s * rows2 + q + kPad) * C0) =
            make_float4(fmaxf(v[0].x, v[1].x), fmaxf(v[0].y, v[1].y), fmaxf(v[0].z, v[1].z), fmaxf(v[0].w, v[1].w));
    }
    // the pad rows of every sequence: 0, 1 and L + 2, L + 3
    const float4 z = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    for (int idx = tid / H; idx < NS * 4; idx += nt / H) {
        const int s = idx >> 2, k = idx & 3;
        *reinterpret_cast<float4 *>(e1 + ((int64_t)s * rows1 + (k < 2 ? k : L + k)) * C0) = z;
        *reinterpret_cast<float4 *>(p1 + ((int64_t)s * rows2 + (k < 2 ? k : Q + k)) * C0) = z;
    }
}

// The tensor-core forms' step f by `nt` threads (of one block, or of those that share the event): weights in registers at width 16 (IV: the per-interval layout),
// read from shared memory at width 32.
template <class T, int C0 = kC0, bool IV = false>
__device__ __forceinline__ void enc1_pool(const FrontArgs &a, int e, int tid, int nt, const float *shist,
                                          const float *senc) {
    if constexpr (C0 != kC0) {
        if (a.amax) enc1_pool_shared_t<T, true, C0>(a, e, tid, nt, shist, senc);
        else enc1_pool_shared_t<T, false, C0>(a, e, tid, nt, shist, senc);
    } else if constexpr (IV) {
        if (a.amax) enc1_pool_t<T, true>(a, e, tid, nt, shist, senc);
        else enc1_pool_t<T, false>(a, e, tid, nt, shist, senc);
    } else {
        if (a.amax) enc1_pool_quads<T, true>(a, e, tid, nt, shist, senc);
        else enc1_pool_quads<T, false>(a, e, tid, nt, shist, senc);
    }
}

}  // namespace front
}  // namespace pvf
