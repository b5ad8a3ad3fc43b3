// Step 3 of the path (§2, UNet-style 1D CNN) in plain float32 on CUDA cores: the
// "plain FP32 GPU form" that the tensor-core forms are measured against.
//
// Layers (positions L, channels):   enc2 16->32 @2000 (+pool)   enc3 32->64 @1000 (+pool)
//   enc4 64->128 @500   up3 128->64 @500->1000   dec3 [64+64]->64 @1000
//   up2 64->32 @1000->2000   dec2 [32+32]->32 @2000   up1 32->16 @2000->4000
//   dec1 [16+16]->16 @4000. Every conv is k5 with zero "same" padding, every conv and
// ConvT is followed by LeakyReLU(0.01); the skip concat is [upsampled, skip] and is
// read in place from the two tensors (never materialised); the 2:1 max-pool is taken in
// the producing conv's epilogue.
//
// Each CTA computes a tile of TP positions x all C_out channels of NS sequences (an event
// is one sequence; the per-interval layout's 40 short sequences go NS = 4 or 8 to a CTA,
// so that a CTA keeps 128 threads); each thread owns a PP x 8 register block (PP = 8, or 4 in
// small launches, consecutive positions x 8 channels; the ConvT 8 x 16). Inputs are staged through shared
// memory in chunks of KC channels, transposed to [channel][position] so a thread's PP + 4
// halo'd inputs are aligned float4 loads; the weights of the chunk sit next to them
// as [tap][channel][C_out]. The sum over (channel, tap) runs in a fixed order: results are
// deterministic.
//
// What bounds them is the FMA pipe (128 lanes per SM), if two other limits are kept off:
//   * issue slots: the FMAs are packed two-lane instructions (each lane an fmaf), on pairs
//     of neighbouring channels, which halves them;
//   * the shared-memory data path, where every 16-byte load costs a warp four cycles and
//     the 8-lane groups must hit distinct banks: a thread's 8 channels are 4 cg .. 4 cg + 3
//     and C_out / 2 + 4 cg .. + 3, so that neighbouring lanes read neighbouring 16 bytes.
//     (With 8 consecutive channels per thread the lanes lay 32 bytes apart: a two-way
//     conflict that held dec3 at 74% of the shared-memory path and 0.67 of the FMA peak.)
// The chunks are double buffered with cp.async (4-byte copies do the transposition), one
// block barrier per chunk.
// Measured (500 events, before -> after): dec3 780 -> 656 us (0.79 of the 80.5 TFLOP/s at
// 2.07 GHz), dec2 417 -> 339, enc4 408 -> 324, up3 281 -> 175, dec1 274 -> 190, enc3
// 218 -> 178, up2 158 -> 111, enc2 140 -> 101, up1 82 -> 82 (close to its memory traffic's
// share). 16 positions per thread (half the shared loads per FMA, half the warps): dec3
// 654, but dec1 217 and, with 16 events, 1.6x slower kernels; not taken.
#include "pvf_internal.cuh"

namespace pvf {
namespace {

__device__ __forceinline__ uint32_t s2u(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// 4 bytes global -> shared, asynchronous; zero-filled (nothing read) when !ok
__device__ __forceinline__ void cp4(float *dst, const float *src, bool ok) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(s2u(dst)), "l"(src), "r"(ok ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s2u(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Pitch (floats) of a staged channel row of n positions: a multiple of 4 (float4 loads) that
// is 4 modulo 32, so that 8 channels x 4 positions written by a warp's copies hit 32 banks.
constexpr int row_pitch(int n) { return (n + 27) / 32 * 32 + 4; }

// Channel of column j (0..7) of column group cg: two runs of four, half of COUT apart.
template <int COUT> __device__ __forceinline__ int col_of(int cg, int j) {
    return (j < 4 ? 0 : COUT / 2) + 4 * cg + (j & 3);
}

template <int CA, int CB, int COUT, int TP, int NS, bool POOL, int KC, int PP>
__global__ void __launch_bounds__((TP / PP) * (COUT / 8) * NS, 512 / ((TP / PP) * (COUT / 8) * NS))
k_conv5_f32(const float *__restrict__ inA, const float *__restrict__ inB,
            const float *__restrict__ W, const float *__restrict__ bias,
            float *__restrict__ out, float *__restrict__ outp, int L) {
    constexpr int CIN = CA + CB;
    constexpr int NCG = COUT / 8, NPG = TP / PP, NT = NCG * NPG * NS;
    constexpr int XR = TP + 4;              // halo'd rows of a sequence's tile
    constexpr int XP = row_pitch(NS * XR);
    static_assert(CA % KC == 0 && CB % KC == 0 && KC % 4 == 0, "channel chunks must not straddle");
    static_assert(COUT % 16 == 0 && TP % 8 == 0, "tiles");
    __shared__ __align__(16) float xs[2][KC][XP];
    __shared__ __align__(16) float ws[2][5][KC][COUT];

    const int tid = threadIdx.x;
    const int cg = tid % NCG, pg = tid / NCG % NPG, sq = tid / (NCG * NPG);
    const int64_t e0 = (int64_t)blockIdx.y * NS;      // first sequence of this CTA
    const int p0 = blockIdx.x * TP;
    const int64_t rowsE = padded_rows(L);

    auto stage_x = [&](int kc, int buf) {
        const bool fromA = kc < CA;
        const int C = fromA ? CA : CB;
        const float *src = (fromA ? inA : inB) + (fromA ? kc : kc - CA);
        // tile row r of sequence s <-> position p0 - 2 + r <-> storage row p0 + r
        for (int idx = tid; idx < NS * XR * KC; idx += NT) {
            const int k = idx % KC, rr = idx / KC;
            const int s = NS == 1 ? 0 : rr / XR, r = NS == 1 ? rr : rr % XR;
            const int64_t srow = (int64_t)p0 + r;
            const bool ok = srow < rowsE;
            cp4(&xs[buf][k][rr], src + ((e0 + s) * rowsE + (ok ? srow : 0)) * C + k, ok);
        }
    };
    auto stage_w = [&](int kc, int buf) {
        for (int idx = tid; idx < 5 * KC * COUT / 4; idx += NT) {
            const int t = idx / (KC * COUT / 4), rem = idx % (KC * COUT / 4);
            cp16(reinterpret_cast<float4 *>(&ws[buf][t][0][0]) + rem,
                 reinterpret_cast<const float4 *>(W + ((size_t)t * CIN + kc) * COUT) + rem);
        }
    };

    stage_w(0, 0);      // the handle's, like the biases; the inputs are the previous kernel's output
    float2 acc[PP][4];                        // [position][channel pair]
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float2 b = make_float2(bias[col_of<COUT>(cg, 2 * q)], bias[col_of<COUT>(cg, 2 * q + 1)]);
#pragma unroll
        for (int pi = 0; pi < PP; ++pi) acc[pi][q] = b;
    }

    grid_dep_wait();
    stage_x(0, 0);
    constexpr int NCH = CIN / KC;
#pragma unroll 1
    for (int c = 0; c < NCH; ++c) {
        const int buf = c & 1;
        cp_wait_all();
        __syncthreads();                     // chunk c staged; the other buffer is no longer read
        if (c + 1 < NCH) {
            stage_x((c + 1) * KC, buf ^ 1);
            stage_w((c + 1) * KC, buf ^ 1);
        }
#pragma unroll 4   // against 1: dec3 664 -> 652, dec2 350 -> 339, enc2 107 -> 100 us (500 events)
        for (int k = 0; k < KC; ++k) {
            float xv[PP + 4];
            const float4 *xr = reinterpret_cast<const float4 *>(&xs[buf][k][sq * XR + pg * PP]);
#pragma unroll
            for (int i = 0; i < PP / 4 + 1; ++i) {
                const float4 v = xr[i];
                xv[4 * i] = v.x; xv[4 * i + 1] = v.y; xv[4 * i + 2] = v.z; xv[4 * i + 3] = v.w;
            }
#pragma unroll
            for (int t = 0; t < 5; ++t) {
                const float4 wa = *reinterpret_cast<const float4 *>(&ws[buf][t][k][4 * cg]);
                const float4 wb = *reinterpret_cast<const float4 *>(&ws[buf][t][k][COUT / 2 + 4 * cg]);
                const float2 wv[4] = {make_float2(wa.x, wa.y), make_float2(wa.z, wa.w), make_float2(wb.x, wb.y),
                                      make_float2(wb.z, wb.w)};
#pragma unroll
                for (int pi = 0; pi < PP; ++pi) {
                    const float2 x2 = make_float2(xv[pi + t], xv[pi + t]);
#pragma unroll
                    for (int q = 0; q < 4; ++q) acc[pi][q] = __ffma2_rn(x2, wv[q], acc[pi][q]);
                }
            }
        }
    }

    const int64_t e = e0 + sq;
    float *ob = out + (size_t)e * rowsE * COUT;
#pragma unroll
    for (int pi = 0; pi < PP; ++pi) {
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[pi][q] = make_float2(leaky(acc[pi][q].x), leaky(acc[pi][q].y));
        const int p = p0 + pg * PP + pi;
        if (p < L) {
            float *d = ob + (size_t)(p + kPad) * COUT + 4 * cg;
            *reinterpret_cast<float4 *>(d) = make_float4(acc[pi][0].x, acc[pi][0].y, acc[pi][1].x, acc[pi][1].y);
            *reinterpret_cast<float4 *>(d + COUT / 2) =
                make_float4(acc[pi][2].x, acc[pi][2].y, acc[pi][3].x, acc[pi][3].y);
        }
    }
    if constexpr (POOL) {
        const int Lp = L / 2;
        float *pb = outp + (size_t)e * padded_rows(Lp) * COUT;
#pragma unroll
        for (int pi = 0; pi < PP; pi += 2) {
            const int p = p0 + pg * PP + pi;
            if (p + 1 < L) {
                float2 v[4];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    v[q] = make_float2(fmaxf(acc[pi][q].x, acc[pi + 1][q].x), fmaxf(acc[pi][q].y, acc[pi + 1][q].y));
                float *d = pb + (size_t)(p / 2 + kPad) * COUT + 4 * cg;
                *reinterpret_cast<float4 *>(d) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
                *reinterpret_cast<float4 *>(d + COUT / 2) = make_float4(v[2].x, v[2].y, v[3].x, v[3].y);
            }
        }
    }
    // pad rows of each sequence: written by its first and its last tile
    // (a single tile is both: it writes both sides)
    const bool first = blockIdx.x == 0, last = blockIdx.x == gridDim.x - 1;
#pragma unroll 1
    for (int side = 0; side < 2; ++side) {
        if (!(side == 0 ? first : last)) continue;
        const int base = side == 0 ? 0 : L + kPad;
        for (int i = tid; i < NS * 2 * COUT; i += NT) {
            const int64_t es = e0 + i / (2 * COUT);
            out[((size_t)es * rowsE + base) * COUT + i % (2 * COUT)] = 0.0f;
            if constexpr (POOL) {
                const int Lp = L / 2;
                const int pbase = side == 0 ? 0 : Lp + kPad;
                outp[((size_t)es * padded_rows(Lp) + pbase) * COUT + i % (2 * COUT)] = 0.0f;
            }
        }
    }
}

// ConvTranspose1d k2 s2 + LeakyReLU: out[2i + r][co] = lrelu(b[co] + sum_ci W[ci][r][co] in[i][ci]).
// A GEMM per event with M = input positions, N = 2 * C_out (column n = r * C_out + co). A
// thread owns 8 positions x 16 columns (four runs of four, N / 4 apart): per channel six
// 16-byte shared loads for 64 packed FMAs (8 x 8 blocks would need as many load cycles as
// FMA cycles).
template <int CIN, int COUT, int TP, int NS, int KC>
__global__ void __launch_bounds__((TP / 8) * (2 * COUT / 16) * NS, 256 / ((TP / 8) * (2 * COUT / 16) * NS))
k_convT_f32(const float *__restrict__ in, const float *__restrict__ W,
            const float *__restrict__ bias, float *__restrict__ out, int Lin) {
    constexpr int N = 2 * COUT;
    constexpr int NCG = N / 16, NPG = TP / 8, NT = NCG * NPG * NS;
    constexpr int XP = row_pitch(NS * TP);
    static_assert(CIN % KC == 0 && KC % 8 == 0 && N % 32 == 0, "channel chunks");
    __shared__ __align__(16) float xs[2][KC][XP];
    __shared__ __align__(16) float ws[2][KC][N];

    const int tid = threadIdx.x;
    const int cg = tid % NCG, pg = tid / NCG % NPG, sq = tid / (NCG * NPG);
    const int64_t e0 = (int64_t)blockIdx.y * NS;
    const int p0 = blockIdx.x * TP;
    const int64_t rowsIn = padded_rows(Lin);
    const int Lout = 2 * Lin;
    const int64_t rowsOut = padded_rows(Lout);

    auto stage_x = [&](int kc, int buf) {
        // 8 channels at a time: 32 contiguous bytes per position, distinct banks per warp
        for (int idx = tid; idx < NS * TP * KC; idx += NT) {
            const int k = idx % 8 + idx / (8 * NS * TP) * 8, rr = idx / 8 % (NS * TP);
            const int s = NS == 1 ? 0 : rr / TP, p = p0 + (NS == 1 ? rr : rr % TP);
            const bool ok = p < Lin;
            cp4(&xs[buf][k][rr], in + ((e0 + s) * rowsIn + (ok ? p + kPad : 0)) * CIN + kc + k, ok);
        }
    };
    auto stage_w = [&](int kc, int buf) {
        for (int idx = tid; idx < KC * N / 4; idx += NT)
            cp16(reinterpret_cast<float4 *>(&ws[buf][0][0]) + idx,
                 reinterpret_cast<const float4 *>(W + (size_t)kc * N) + idx);
    };

    stage_w(0, 0);      // the handle's, like the biases; the inputs are the previous kernel's output
    float2 acc[8][8];                        // [position][column pair]
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        const int co = (g * (N / 4) + 4 * cg) % COUT;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float2 b = make_float2(bias[co + 2 * h], bias[co + 2 * h + 1]);
#pragma unroll
            for (int pi = 0; pi < 8; ++pi) acc[pi][2 * g + h] = b;
        }
    }
    grid_dep_wait();
    stage_x(0, 0);
    constexpr int NCH = CIN / KC;
#pragma unroll 1
    for (int c = 0; c < NCH; ++c) {
        const int buf = c & 1;
        cp_wait_all();
        __syncthreads();
        if (c + 1 < NCH) {
            stage_x((c + 1) * KC, buf ^ 1);
            stage_w((c + 1) * KC, buf ^ 1);
        }
#pragma unroll 2
        for (int k = 0; k < KC; ++k) {
            const float4 *xr = reinterpret_cast<const float4 *>(&xs[buf][k][sq * TP + pg * 8]);
            const float4 xa = xr[0], xb = xr[1];
            const float xv[8] = {xa.x, xa.y, xa.z, xa.w, xb.x, xb.y, xb.z, xb.w};
            float2 wv[8];
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const float4 w4 = *reinterpret_cast<const float4 *>(&ws[buf][k][g * (N / 4) + 4 * cg]);
                wv[2 * g] = make_float2(w4.x, w4.y);
                wv[2 * g + 1] = make_float2(w4.z, w4.w);
            }
#pragma unroll
            for (int pi = 0; pi < 8; ++pi) {
                const float2 x2 = make_float2(xv[pi], xv[pi]);
#pragma unroll
                for (int q = 0; q < 8; ++q) acc[pi][q] = __ffma2_rn(x2, wv[q], acc[pi][q]);
            }
        }
    }
    float *ob = out + (size_t)(e0 + sq) * rowsOut * COUT;
#pragma unroll
    for (int pi = 0; pi < 8; ++pi) {
        const int i = p0 + pg * 8 + pi;
        if (i < Lin) {
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const int n = g * (N / 4) + 4 * cg;      // column n: output row 2 i + n / COUT
                const float2 a = acc[pi][2 * g], b = acc[pi][2 * g + 1];
                *reinterpret_cast<float4 *>(ob + (size_t)(2 * i + n / COUT + kPad) * COUT + n % COUT) =
                    make_float4(leaky(a.x), leaky(a.y), leaky(b.x), leaky(b.y));
            }
        }
    }
    const bool first = blockIdx.x == 0, last = blockIdx.x == gridDim.x - 1;
#pragma unroll 1
    for (int side = 0; side < 2; ++side) {   // a single tile is both first and last
        if (!(side == 0 ? first : last)) continue;
        const int base = side == 0 ? 0 : Lout + kPad;
        for (int i = tid; i < NS * 2 * COUT; i += NT)
            out[((size_t)(e0 + i / (2 * COUT)) * rowsOut + base) * COUT + i % (2 * COUT)] = 0.0f;
    }
}

// Dependent launches hide each other's launch and first weight tile. The kernels trigger nothing
// early: blocks of the next layer placed while this one still ran crowded the SMs that happened to
// be free (16 events: 184 us a call without dependent launches, 158 with them, 210 with a trigger
// behind the main loop, 234 at the start; 500 events 2333, 2312, 2312, 2366).

// n: sequences (a multiple of NS)
template <int CA, int CB, int COUT, int TP, int NS, bool POOL, int KC, int PP>
cudaError_t conv5_pp(const void *a, const void *b, const float *W, const float *bias, void *out,
                     void *outp, int L, dim3 grid, cudaStream_t s) {
    return launch_pdl(k_conv5_f32<CA, CB, COUT, TP, NS, POOL, KC, PP>, grid, dim3((TP / PP) * (COUT / 8) * NS), 0, s,
                      (const float *)a, (const float *)b, W, bias, (float *)out, (float *)outp, L);
}

template <int CA, int CB, int COUT, int TP, int NS, bool POOL, int KC>
cudaError_t conv5(const void *a, const void *b, const float *W, const float *bias, void *out,
                  void *outp, int L, int n, cudaStream_t s) {
    if constexpr (NS == 1) {
        // tiles of half the positions, half of them per thread, where each has an SM of its own: a
        // tile is bound by its SM's FMA pipe, which then has half the work (1 event 148 -> 117 us a
        // call, 9 events 156 -> 125; with up to 1.5 and 2 tiles per SM: 16 events 158 and 157
        // either way, 8 events of the wide network 271 and 274). Half the positions per thread in
        // tiles of the same size: no gain
        int sms = 0;
        const cudaError_t err = current_device_sms(&sms);
        if (err != cudaSuccess) return err;
        const dim3 half((L + TP / 2 - 1) / (TP / 2), n);
        if ((int64_t)half.x * half.y <= sms)
            return conv5_pp<CA, CB, COUT, TP / 2, NS, POOL, KC, 4>(a, b, W, bias, out, outp, L, half, s);
    }
    const dim3 grid((L + TP - 1) / TP, n / NS);
    return conv5_pp<CA, CB, COUT, TP, NS, POOL, KC, 8>(a, b, W, bias, out, outp, L, grid, s);
}

template <int CIN, int COUT, int TP, int NS, int KC>
cudaError_t convT(const void *in, const float *W, const float *bias, void *out, int Lin, int n,
                  cudaStream_t s) {
    dim3 grid((Lin + TP - 1) / TP, n / NS), block((TP / 8) * (2 * COUT / 16) * NS);
    return launch_pdl(k_convT_f32<CIN, COUT, TP, NS, KC>, grid, block, 0, s, (const float *)in, W, bias,
                      (float *)out, Lin);
}

// The layer sequence for base width C (levels C, 2C, 4C, 8C). Tiles halve as the channel
// counts double, so every CTA keeps 128 threads. Channels per chunk: 8 (double buffered,
// weights and inputs fit the 48 KB of static shared memory), 4 for the 256-channel output.
template <int C>
cudaError_t run_f32(const ConvF32Weights &w, const UnetBuffers &b, int n, cudaStream_t s,
                    const ProfHook *prof) {
    constexpr int R = kC0;                       // tile sizes are for base width R, halved at 2 R
    constexpr int K4 = C > kC0 ? 4 : 8;
    cudaError_t err;
#define PVF_TRY(name, x) do { ProfScope ps_(prof, name, s); err = (x); if (err != cudaSuccess) return err; } while (0)
    // each tensor is packed in its slot with its own per-event stride (L + 4) * C
    PVF_TRY("enc2", (conv5<C, 0, 2 * C, 256 * R / C, 1, true, 8>(b.s0, nullptr, w.w[0], w.b[0], b.e2, b.s1, 2000, n, s)));
    PVF_TRY("enc3", (conv5<2 * C, 0, 4 * C, 128 * R / C, 1, true, 8>(b.s1, nullptr, w.w[1], w.b[1], b.e3, b.s0, 1000, n, s)));
    PVF_TRY("enc4", (conv5<4 * C, 0, 8 * C, 64 * R / C, 1, false, K4>(b.s0, nullptr, w.w[2], w.b[2], b.deep, nullptr, 500, n, s)));
    PVF_TRY("up3", (convT<8 * C, 4 * C, 128 * R / C, 1, 16>(b.deep, w.uw[0], w.ub[0], b.up, 500, n, s)));
    PVF_TRY("dec3", (conv5<4 * C, 4 * C, 4 * C, 128 * R / C, 1, false, 8>(b.up, b.e3, w.w[3], w.b[3], b.deep, nullptr, 1000, n, s)));
    PVF_TRY("up2", (convT<4 * C, 2 * C, 256 * R / C, 1, 16>(b.deep, w.uw[1], w.ub[1], b.up, 1000, n, s)));
    PVF_TRY("dec2", (conv5<2 * C, 2 * C, 2 * C, 256 * R / C, 1, false, 8>(b.up, b.e2, w.w[4], w.b[4], b.deep, nullptr, 2000, n, s)));
    PVF_TRY("up1", (convT<2 * C, C, 512 * R / C, 1, 8>(b.deep, w.uw[2], w.ub[2], b.up, 2000, n, s)));
    PVF_TRY("dec1", (conv5<C, C, C, 512 * R / C, 1, false, 8>(b.up, b.e1, w.w[5], w.b[5], b.deep, nullptr, 4000, n, s)));
#undef PVF_TRY
    return cudaSuccess;
}

// The per-interval layout: kSlices sequences of kIvLen bins per event (104, 52, 26, 13
// positions per level), each layer one small tile per sequence, 4 or 8 sequences per CTA
// (kSlices is a multiple of both, so every group is full).
template <int C>
cudaError_t run_f32_iv(const ConvF32Weights &w, const UnetBuffers &b, int n, cudaStream_t s,
                       const ProfHook *prof) {
    constexpr int L1 = kIvLen, L2 = L1 / 2, L3 = L1 / 4, L4 = L1 / 8;
    static_assert(kSlices % 8 == 0, "full groups of sequences");
    const int ns = n * kSlices;                  // at most 64000 (the plan caps the chunk)
    cudaError_t err;
#define PVF_TRY(name, x) do { ProfScope ps_(prof, name, s); err = (x); if (err != cudaSuccess) return err; } while (0)
    PVF_TRY("enc2", (conv5<C, 0, 2 * C, 64, 4, true, 8>(b.s0, nullptr, w.w[0], w.b[0], b.e2, b.s1, L2, ns, s)));
    PVF_TRY("enc3", (conv5<2 * C, 0, 4 * C, 32, 4, true, 8>(b.s1, nullptr, w.w[1], w.b[1], b.e3, b.s0, L3, ns, s)));
    PVF_TRY("enc4", (conv5<4 * C, 0, 8 * C, 16, 4, false, 8>(b.s0, nullptr, w.w[2], w.b[2], b.deep, nullptr, L4, ns, s)));
    PVF_TRY("up3", (convT<8 * C, 4 * C, 16, 8, 16>(b.deep, w.uw[0], w.ub[0], b.up, L4, ns, s)));
    PVF_TRY("dec3", (conv5<4 * C, 4 * C, 4 * C, 32, 4, false, 8>(b.up, b.e3, w.w[3], w.b[3], b.deep, nullptr, L3, ns, s)));
    PVF_TRY("up2", (convT<4 * C, 2 * C, 32, 8, 16>(b.deep, w.uw[1], w.ub[1], b.up, L3, ns, s)));
    PVF_TRY("dec2", (conv5<2 * C, 2 * C, 2 * C, 64, 4, false, 8>(b.up, b.e2, w.w[4], w.b[4], b.deep, nullptr, L2, ns, s)));
    PVF_TRY("up1", (convT<2 * C, C, 64, 8, 8>(b.deep, w.uw[2], w.ub[2], b.up, L2, ns, s)));
    PVF_TRY("dec1", (conv5<C, C, C, 128, 4, false, 8>(b.up, b.e1, w.w[5], w.b[5], b.deep, nullptr, L1, ns, s)));
#undef PVF_TRY
    return cudaSuccess;
}

}  // namespace

cudaError_t launch_unet_f32(const ConvF32Weights &w, const UnetBuffers &b, int n, bool iv, cudaStream_t s,
                            const ProfHook *prof) {
    if (n <= 0) return cudaSuccess;
    if (iv) {
        if (w.c0 != kC0 || n * kSlices > 65535) return cudaErrorInvalidValue;
        return run_f32_iv<kC0>(w, b, n, s, prof);
    }
    if (w.c0 == kC0) return run_f32<kC0>(w, b, n, s, prof);
    if (w.c0 == kC0Max) return run_f32<kC0Max>(w, b, n, s, prof);
    return cudaErrorInvalidValue;
}

}  // namespace pvf
