// The encoder of the tensor-core UNet as one persistent kernel: enc2 (+ pool), enc3 (+ pool)
// and enc4 + up3 of whole events (base width 16), for csrc/k_unet_tc.cu, whose tile shapes,
// MMA sequences and epilogues it uses.
//
// Why one kernel. Run one after the other the three layers move 704 KB per event through
// memory (16-bit forms) and each was within 78% of the copy rate: p2 and p3 are written and
// read back only to cross a kernel boundary. Here they stay in shared memory, and 448 KB per
// event remain (p1 in; e2, e3 and u3, which the decoder reads, out).
//
// A CTA (one per SM: the four layers' weights take 137 KB in 16 bits) streams through its
// units, a unit being an event or, in small launches, half or a quarter of one. In an event
// 16 enc2 tiles of 128 positions feed 8 enc3 tiles feed 4 enc4 tiles, so the work is a
// steady 4 : 2 : 1 pattern that runs on from event to event without draining:
//   producer (warp 0)   p1 tiles (132 rows) into a ring of stages
//   MMA warps 1, 2, 3   one per layer (enc2; enc3; enc4 and its ConvT), so that a layer whose
//                       inputs are not there yet holds up no other
//   warpgroups 0, 1     enc2 accumulator -> e2 (memory) and p2 (shared memory, as the rows of
//                       enc3's operand tiles; the halo rows go to the neighbouring tile too),
//                       every other tile each
//   warpgroups 2, 3     enc3 accumulator -> e3 and p3, the same way
//   warpgroup 4         enc4 accumulator -> the ConvT's operand in tensor memory
//   warpgroup 5         ConvT accumulator -> u3
// A unit that does not
// start (end) at an event's edge recomputes one enc3 and one enc2 tile on that side for
// their last (first) rows and stores none of it.
#pragma once

// (included inside k_unet_tc.cu's namespaces)

template <class N> struct Enc {
    using C2 = typename N::Enc2;
    using C3 = typename N::Enc3;
    using C4 = typename N::Enc4Up3;
    static constexpr int T2N = C2::TPE, T3N = C3::TPE, T4N = C4::TPE;    // tiles per event
    static_assert(T2N == 2 * T3N && T3N == 2 * T4N && T4N % 4 == 0, "4 : 2 : 1 tiles");
    static_assert(C2::L == 2 * C3::L && C3::L == 2 * C4::L && !C2::SEQ, "whole events");
    static constexpr int ST = 3;                    // p1 stages
    static constexpr int NP2 = 3, NP3 = 3;          // p2 / p3 operand tiles
    static constexpr int RING = 8;                  // tile-done barriers of enc2 and enc3
    static constexpr int THREADS = 4 * 32 + 6 * 128;
    static constexpr int P2_BYTES = align_up(C3::PIN * C3::ROWS * 16, 128);
    static constexpr int P3_BYTES = align_up(C4::PIN * C4::ROWS * 16, 128);
    // tensor memory: two accumulators for enc2 and enc3, one for enc4, one for the ConvT, its operand
    static constexpr int COL2 = 0, COL3 = COL2 + 2 * C2::COUT, COL4 = COL3 + 2 * C3::COUT,
                         COL5 = COL4 + C4::COUT, COLA = COL5 + C4::N2, TMEM_COLS = 512;
    static_assert(COLA + C4::A2_COLS <= TMEM_COLS, "TMEM columns");
    // shared memory: weights, p1 stages, p2 and p3 tiles, barriers
    static constexpr int OFF_W2 = 0, OFF_W3 = align_up(OFF_W2 + C2::W_BYTES, 128),
                         OFF_W4 = align_up(OFF_W3 + C3::W_BYTES, 128),
                         OFF_W5 = align_up(OFF_W4 + C4::W_BYTES, 128),
                         OFF_A = align_up(OFF_W5 + C4::W2_BYTES, 128);
    // launch parameters (floats): biases of enc2, enc3, enc4, up3, then (e4m3) their column scales
    static constexpr int PB2 = 0, PB3 = PB2 + C2::COUT, PB4 = PB3 + C3::COUT, PB5 = PB4 + C4::COUT,
                         PS2 = PB5 + C4::CUP, PS3 = PS2 + C2::COUT, PS4 = PS3 + C3::COUT, PS5 = PS4 + C4::COUT,
                         NPAR = is16(C2::PREC) ? PS2 : PS5 + C4::N2;
    static constexpr int OFF_P2 = OFF_A + ST * C2::A_STAGE;
    static constexpr int OFF_P3 = OFF_P2 + NP2 * P2_BYTES;
    static constexpr int OFF_BAR = OFF_P3 + NP3 * P3_BYTES;
    // barriers: weights; p1 stages; accumulators full / free; p2 and p3 tiles free; tiles of
    // enc2 and enc3 whose pooled rows are in place (a ring: a layer can be at most NP2 (NP3)
    // operand tiles, i.e. less than RING of its tiles, ahead of the layer that waits)
    static constexpr int W2 = 0, W3 = 1, W4 = 2, FULL = 3, EMPTY = FULL + ST, T2F = EMPTY + ST, T2E = T2F + 2,
                         P2E = T2E + 2, T3F = P2E + NP2, T3E = T3F + 2, P3E = T3E + 2, T4F = P3E + NP3, T4E = T4F + 1,
                         A2F = T4E + 1, A2E = A2F + 1, T5F = A2E + 1, T5E = T5F + 1, D2 = T5E + 1, D3 = D2 + RING,
                         DRAIN = D3 + RING, NEVER = DRAIN + 3, NBAR = NEVER + 1;
    static_assert(2 * NP2 + 2 <= RING && 2 * NP3 + 2 <= RING, "tile-done ring");
    static constexpr int SMEM = OFF_BAR + 8 * NBAR + 16;
    static_assert(SMEM <= 227 * 1024, "shared memory");
};

struct EncArgs {
    TcArgs c2, c3, c4;      // enc2: inA = p1, out = e2; enc3: out = e3; enc4 + up3: out = u3
};

// Tiles of one unit: event e, enc4 tiles [k0, k1), and the enc3 and enc2 tiles these need.
struct EncUnit { int e, k0, k1, a3, b3, a2, b2; };
template <class E> __device__ __forceinline__ EncUnit enc_unit(int u, int lg) {
    EncUnit x;
    const int g = E::T4N >> lg;
    x.e = u >> lg;
    x.k0 = (u & ((1 << lg) - 1)) * g;
    x.k1 = x.k0 + g;
    x.a3 = x.k0 ? 2 * x.k0 - 1 : 0;
    x.b3 = x.k1 < E::T4N ? 2 * x.k1 + 1 : E::T3N;
    x.a2 = x.k0 ? 4 * x.k0 - 1 : 0;
    x.b2 = x.k1 < E::T4N ? 4 * x.k1 + 1 : E::T2N;
    return x;
}

// Units per event (log2: 1, 2 or 4 of them): the fewest rounds of work for the busiest of g CTAs, a half
// event costing 0.56 and a quarter 0.36 of a whole one (the recomputed tiles).
__device__ __forceinline__ int enc_split(int n, int g) {
    const int c1 = (n + g - 1) / g * 100, c2 = (2 * n + g - 1) / g * 56, c4 = (4 * n + g - 1) / g * 36;
    return c1 <= c2 && c1 <= c4 ? 0 : (c2 <= c4 ? 1 : 2);
}

template <class E>
__device__ bool enc_producer(const EncArgs &a, unsigned char *smem, uint64_t *bar, volatile int *abort) {
    using C = typename E::C2;
    uint64_t *full = bar + E::FULL, *empty = bar + E::EMPTY;
    const int n_ev = launch_events(a.c2.n_dyn, a.c2.dyn_base, a.c2.n_events);
    const int lg = enc_split(n_ev, gridDim.x), nu = n_ev << lg;
    int n = 0;
    bool ok = true;
    for (int u = blockIdx.x; ok && u < nu; u += gridDim.x) {
        const EncUnit x = enc_unit<E>(u, lg);
        for (int i = x.a2; i < x.b2; ++i, ++n) {
            const int s = n % E::ST;
            if (!mbar_wait(&empty[s], ((n / E::ST) & 1) ^ 1, abort)) { ok = false; break; }
            const int src0 = i * kTileM;          // tile row r <-> storage row src0 + r
            const int rows = min(C::ROWS, C::ROWS_E - src0);
            unsigned char *dst = smem + E::OFF_A + s * C::A_STAGE;
            if constexpr (C::PAIR) {   // the zero-weight 6th tap reads one row past the copied ones
                if (rows < C::ROWS) {
                    for (int k = 0; k < C::PIN; ++k)
                        *reinterpret_cast<uint4 *>(dst + k * C::ROWS * 16 + rows * 16) = make_uint4(0, 0, 0, 0);
                    fence_proxy_async_smem();
                }
            }
            mbar_arrive_expect_tx(&full[s], (uint32_t)(C::PIN * rows * 16));
            for (int k = 0; k < C::PIN; ++k)
                bulk_g2s(dst + k * C::ROWS * 16, a.c2.inA + planar_off(x.e, k, C::PIN, C::ROWS_E, src0), rows * 16,
                         &full[s]);
        }
    }
    // copies still in flight land before the CTA can exit: wait (bounded) for the last ones
    const uint64_t t0 = globaltimer();
    for (int j = max(0, n - E::ST); j < n; ++j)
        while (!mbar_try_wait(&full[j % E::ST], (j / E::ST) & 1))
            if (globaltimer() - t0 > kWaitLimitNs) break;
    for (int w = E::W2; w <= E::W4; ++w)
        while (!mbar_try_wait(bar + w, 0))
            if (globaltimer() - t0 > 2 * kWaitLimitNs) break;
    return ok;
}

// The MMA warps: all 32 threads run the loop, one issues. Ring positions are counted along
// and units are powers of two: this code runs once per tile between the MMAs, and with one
// warp for all layers and divisions in it, it and not the tensor core set the pace (3500
// cycles per enc2 tile, 2600 of them between the MMAs).
struct EncWarp {
    uint64_t *bar;
    volatile int *abort;
    uint32_t sb, tmem;                   // shared-memory base, tensor-memory base
    int nu, lg;                          // units, log2 of the units per event
    __device__ __forceinline__ bool wait(int b, uint32_t parity) const { return mbar_wait_warp(bar + b, parity, abort); }
};

template <class E> __device__ bool enc_mma2(const EncWarp &w) {
    using C = typename E::C2;
    int s = 0, b = 0;
    uint32_t ph_s = 0, ph_b = 0;
    if (!w.wait(E::W2, 0)) return false;
    for (int u = blockIdx.x; u < w.nu; u += gridDim.x) {
        const EncUnit x = enc_unit<E>(u, w.lg);
        for (int left = x.b2 - x.a2; left > 0; --left) {
            if (!w.wait(E::T2E + b, ph_b ^ 1) || !w.wait(E::FULL + s, ph_s)) return false;
            tc_fence_after();
            if (elect_one()) {
                issue_conv<C>(w.tmem + E::COL2 + b * C::COUT, w.sb + E::OFF_A + s * C::A_STAGE, w.sb + E::OFF_W2);
                mma_commit(w.bar + E::EMPTY + s);
                mma_commit(w.bar + E::T2F + b);
            }
            if (++s == E::ST) { s = 0; ph_s ^= 1; }
            if ((b ^= 1) == 0) ph_b ^= 1;
        }
    }
    return true;
}

// enc3 tile j needs enc2 tiles up to 2 j + 2, enc4 tile k enc3 tiles up to 2 k + 2, as far as
// the unit has them: of the tiles [a, b) of the layer below, the first `dep` counted from a
template <class E> __device__ bool enc_mma3(const EncWarp &w) {
    using C = typename E::C3;
    int p = 0, b = 0, r = 0;             // p2 tile, accumulator, tile-done ring
    uint32_t ph_b = 0, ph_r = 0;
    if (!w.wait(E::W3, 0)) return false;
    for (int u = blockIdx.x; u < w.nu; u += gridDim.x) {
        const EncUnit x = enc_unit<E>(u, w.lg);
        const int nin = x.b2 - x.a2;
        int seen = 0, dep = 2 * x.a3 + 3 - x.a2;
        for (int left = x.b3 - x.a3; left > 0; --left, dep += 2) {
            if (!w.wait(E::T3E + b, ph_b ^ 1)) return false;
            for (const int need = left > 1 ? min(dep, nin) : nin; seen < need; ++seen) {
                if (!w.wait(E::D2 + r, ph_r)) return false;
                if (++r == E::RING) { r = 0; ph_r ^= 1; }
            }
            tc_fence_after();
            if (elect_one()) {
                issue_conv<C>(w.tmem + E::COL3 + b * C::COUT, w.sb + E::OFF_P2 + p * E::P2_BYTES, w.sb + E::OFF_W3);
                mma_commit(w.bar + E::P2E + p);
                mma_commit(w.bar + E::T3F + b);
            }
            if (++p == E::NP2) p = 0;
            if ((b ^= 1) == 0) ph_b ^= 1;
        }
    }
    return true;
}

template <class E> __device__ bool enc_mma4(const EncWarp &w) {
    using C = typename E::C4;
    int n = 0, p = 0, r = 0;             // tiles, p3 tile, tile-done ring
    uint32_t ph_r = 0;
    if (!w.wait(E::W4, 0)) return false;
    for (int u = blockIdx.x; u < w.nu; u += gridDim.x) {
        const EncUnit x = enc_unit<E>(u, w.lg);
        const int nin = x.b3 - x.a3;
        int seen = 0, dep = 2 * x.k0 + 3 - x.a3;
        for (int left = x.k1 - x.k0; left > 0; --left, dep += 2, ++n) {
            for (const int need = left > 1 ? min(dep, nin) : nin; seen < need; ++seen) {
                if (!w.wait(E::D3 + r, ph_r)) return false;
                if (++r == E::RING) { r = 0; ph_r ^= 1; }
            }
            if (!w.wait(E::T4E, (n & 1) ^ 1)) return false;
            tc_fence_after();
            if (elect_one()) {
                issue_conv<C>(w.tmem + E::COL4, w.sb + E::OFF_P3 + p * E::P3_BYTES, w.sb + E::OFF_W4);
                mma_commit(w.bar + E::P3E + p);
                mma_commit(w.bar + E::T4F);
            }
            if (++p == E::NP3) p = 0;
            // its ConvT, once the epilogue has written the operand
            if (!w.wait(E::T5E, (n & 1) ^ 1) || !w.wait(E::A2F, n & 1)) return false;
            tc_fence_after();
            if (elect_one()) {
                issue_up_ts<C>(w.tmem + E::COL5, w.tmem + E::COLA, w.sb + E::OFF_W5);
                mma_commit(w.bar + E::A2E);
                mma_commit(w.bar + E::T5F);
            }
        }
    }
    return true;
}

// A pooled layer as the epilogue sees it: enc2 into enc3's operand tiles, or enc3 into enc4's.
// Both run the same code on these values (at run time): two warpgroups with a copy each, and
// the ConvT's roles, did not fit the instruction cache (28% of the stalls were for instructions:
// 152 -> 131 us per 1000 events). Shared-memory places are 32-bit addresses.
struct EncPool {
    unsigned char *out;                       // stored tensor, at this thread's row of an event's first tile
    size_t ev_bytes;                          // bytes per event of it
    uint32_t plane;                           // bytes per plane of it
    int bias, scale;                          // places in the parameter block
    float out_inv;
    int cols, len;                            // channels, positions per event
    uint32_t bufs, buf_bytes;                 // operand tiles of the next layer
    uint32_t full, free, tile_free, done;     // barriers (full, free: of this warpgroup's accumulator)
    uint32_t acc;                             // this lane's first column of its accumulator
    int up;                                   // log2 of its tiles per enc4 tile
};

// One tile row: bias, LeakyReLU, the stored row (st, at dst), and the 2:1 max-pool into row `row`
// of the operand tile buf of the next layer and row `nrow` of the neighbouring tile nbuf (0: none).
// Rows past the event (!valid) pool to zeros, and the event's first tile (lead >= 0) writes the
// zero rows before it. The even lane of a row pair writes the first 8 of each 16 channels (a
// plane in 16 bits, half a plane's row in e4m3), the odd lane the last 8. The accumulator is
// released (L.free) as soon as its last columns are in registers.
template <int PREC, bool CAL, int PLANE, class P>
__device__ __forceinline__ void enc_epi(const EncPool &L, const P &par, const TcArgs &a, unsigned char *dst, bool odd, bool valid, bool st,
                                        uint32_t buf, int row, uint32_t nbuf, int nrow, int lead) {
    const uint32_t half = !odd ? 0 : is16(PREC) ? PLANE : 8;
    const bool edge = nbuf || lead >= 0;
    uint32_t at = buf + half;
    nbuf += half + nrow * 16;
#pragma unroll 1
    for (int c0 = 0; c0 < L.cols; c0 += 16) {
        float v[16], bj[16];
        tmem_ld16(L.acc + c0, v);
        if (c0 + 16 >= L.cols) {
            tc_fence_before();
            mbar_arrive_at(L.free);
        }
        ldp(par, L.bias + c0, bj);
        if constexpr (is16(PREC)) {
            bias_leaky(v, bj);
        } else {
            float sc[16];
            ldp(par, L.scale + c0, sc);
            scale_bias_leaky(v, sc, bj);
        }
        // stored rows only: a recomputed tile of a split event has rows whose inputs nobody in this
        // unit wrote, and every row is stored by one unit
        if constexpr (CAL) amax_fold(a.amax, a.amax_out, v, st);
        uint4 w = make_uint4(0, 0, 0, 0);
        if constexpr (is16(PREC)) {
            using T = typename Elem<PREC>::T;
            uint32_t r[8], x[4];
#pragma unroll
            for (int q = 0; q < 8; ++q) r[q] = pack2<T>(v[2 * q], v[2 * q + 1]);
            if (st) {
                *reinterpret_cast<uint4 *>(dst) = make_uint4(r[0], r[1], r[2], r[3]);
                *reinterpret_cast<uint4 *>(dst + L.plane) = make_uint4(r[4], r[5], r[6], r[7]);
            }
            dst += 2 * L.plane;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t got = __shfl_xor_sync(0xffffffffu, odd ? r[q] : r[4 + q], 1);
                x[q] = max2<T>(odd ? r[4 + q] : r[q], got);
            }
            if (valid) w = make_uint4(x[0], x[1], x[2], x[3]);
        } else {
            uint32_t r[4];
            pack_e4m3<16>(v, L.out_inv, r);
            if (st) *reinterpret_cast<uint4 *>(dst) = make_uint4(r[0], r[1], r[2], r[3]);
            dst += L.plane;
            uint32_t x[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const uint32_t got = __shfl_xor_sync(0xffffffffu, odd ? r[q] : r[2 + q], 1);
                x[q] = max4_e4m3(odd ? r[2 + q] : r[q], got);
            }
            if (valid) w = make_uint4(x[0], x[1], 0, 0);
        }
        constexpr uint32_t STEP = (is16(PREC) ? 2 : 1) * PLANE;        // planes of 16 channels
        auto put = [&](uint32_t to, uint4 q) {
            if constexpr (is16(PREC)) sts16(to, q);
            else sts8(to, make_uint2(q.x, q.y));
        };
        if (buf) put(at + row * 16, w);
        if (edge) {          // a few rows of a tile
            if (nrow >= 0) put(nbuf, w);
            if (lead >= 0) put(at + lead * 16, make_uint4(0, 0, 0, 0));
        }
        at += STEP;
        nbuf += STEP;
    }
}

// The warpgroups of a pooled layer: each takes every other tile (those whose running number is
// odd or even, `half`) of its units into operand tiles [ja, jb) of the next layer; a unit's own
// tiles [s0, s1) are stored. This loop's scalar work is a sixth of the kernel's instructions, so
// nothing in it is recomputed per tile that a unit or the thread fixes.
template <class E, bool CAL>
__device__ bool enc_pool_role(const EncPool &L, const ParBlock<E::NPAR> &par, const TcArgs &a, int half, int m, int nu, int lg, volatile int *abort) {
    constexpr int PREC = E::C2::PREC;
    static_assert(E::NP2 == 3 && E::NP3 == 3 && E::RING == 8 && E::C3::ROWS == E::C4::ROWS, "operand tiles");
    const bool odd = (m & 1) != 0;
    int n0 = 0;                        // tiles before this unit
    int base = 0, touched = 0;         // operand tiles before this unit; those known to be free
    uint32_t tslot = 0, tph = 1, fph = 0;   // slot of tile `touched` and the parity to wait for; of the accumulator
    for (int u = blockIdx.x; u < nu; u += gridDim.x) {
        const EncUnit x = enc_unit<E>(u, lg);
        const bool two = L.up == 2;
        const int ta = two ? x.a2 : x.a3, tb = two ? x.b2 : x.b3;      // this layer's tiles
        const int ja = two ? x.a3 : x.k0, jb = two ? x.b3 : x.k1;      // the next layer's
        const int s0 = x.k0 << L.up, s1 = x.k1 << L.up;
        unsigned char *out = L.out + (size_t)x.e * L.ev_bytes;
        for (int i = ta + ((n0 ^ half) & 1); i < tb; i += 2) {
            const int jt = i >> 1, up = i & 1;
            const int last = base + min(jt + up, jb - 1) - ja;
            for (; touched <= last; ++touched) {                       // first use of a slot passes at once
                if (!mbar_wait_at(L.tile_free + 8 * tslot, tph, abort)) return false;
                if (++tslot == 3) { tslot = 0; tph ^= 1; }
            }
            if (!mbar_wait_at(L.full, fph, abort)) return false;
            fph ^= 1;
            tc_fence_after();
            const int p = i * kTileM + m;
            const bool valid = p < L.len, st = valid && i >= s0 && i < s1;
            // operand tiles jt and its neighbour (base + j - ja modulo 3), where this unit has them
            const int k = base + jt - ja, slot = k % 3;
            const uint32_t buf = jt >= ja && jt < jb ? L.bufs + slot * L.buf_bytes : 0;
            uint32_t nbuf = 0;
            int nrow = -1;
            // pooled position 64 i + m / 2; row r of operand tile jt holds position 128 jt - 2 + r
            const int row = 64 * up + (m >> 1) + kPad;
            if (up ? m >= kTileM - 4 && jt + 1 < jb : m < 4 && jt - 1 >= ja) {     // the neighbour's halo rows
                nbuf = L.bufs + (up ? (slot == 2 ? 0 : slot + 1) : (slot == 0 ? 2 : slot - 1)) * L.buf_bytes;
                nrow = up ? row - kTileM : row + kTileM;
            }
            enc_epi<PREC, CAL, E::C3::ROWS * 16>(L, par, a, out + (size_t)i * (kTileM * 16), odd, valid, st, buf, row, nbuf, nrow,
                                                 i == 0 && m < 4 ? m >> 1 : -1);
            fence_proxy_async_smem();     // the operand rows -> visible to the tensor core
            mbar_arrive_at(L.done + 8 * ((n0 + i - ta) & 7));
            if (st && (p == 0 || p == L.len - 1)) {          // the stored tensor's zero rows
                unsigned char *z = out + (size_t)i * (kTileM * 16) + (p == 0 ? -2 * 16 : 16);
                for (int c = 0; c < L.cols; c += is16(PREC) ? 8 : 16, z += L.plane) {
                    *reinterpret_cast<uint4 *>(z) = make_uint4(0, 0, 0, 0);
                    *reinterpret_cast<uint4 *>(z + 16) = make_uint4(0, 0, 0, 0);
                }
            }
        }
        n0 += tb - ta;
        base += jb - ja;
    }
    return true;
}

template <class E, bool CAL>
__global__ void __launch_bounds__(E::THREADS, 1) k_enc_tc(const __grid_constant__ EncArgs g, const __grid_constant__ ParBlock<E::NPAR> par) {
    using C2 = typename E::C2;
    using C3 = typename E::C3;
    using C4 = typename E::C4;
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + E::OFF_BAR);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bar + E::NBAR);
    volatile int *abort = reinterpret_cast<volatile int *>(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int b = 0; b < E::NBAR; ++b) {
            // epilogue-to-MMA barriers count a warpgroup's threads, the others one arrival
            const bool wg = b == E::T2E || b == E::T2E + 1 || b == E::T3E || b == E::T3E + 1 || b == E::T4E ||
                            b == E::A2F || b == E::T5E || (b >= E::D2 && b < E::DRAIN);
            mbar_init(&bar[b], wg ? 128 : 1);
        }
        *abort = 0;
        fence_mbar_init();
        // the weights are the handle's: they load before the previous kernel has finished
        mbar_arrive_expect_tx(bar + E::W2, C2::W_BYTES);
        bulk_g2s(smem + E::OFF_W2, g.c2.w, C2::W_BYTES, bar + E::W2);
        mbar_arrive_expect_tx(bar + E::W3, C3::W_BYTES);
        bulk_g2s(smem + E::OFF_W3, g.c3.w, C3::W_BYTES, bar + E::W3);
        mbar_arrive_expect_tx(bar + E::W4, C4::W_BYTES + C4::W2_BYTES);
        bulk_g2s(smem + E::OFF_W4, g.c4.w, C4::W_BYTES, bar + E::W4);
        bulk_g2s(smem + E::OFF_W5, g.c4.w2, C4::W2_BYTES, bar + E::W4);
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, E::TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    grid_dep_wait();      // p1 (and a device-side count) are the previous kernel's output
    grid_dep_launch();
    bool ok = true;
    if (warp == 0) {
        if (lane == 0) ok = enc_producer<E>(g, smem, bar, abort);
    } else {
        // (broadcast: a loaded event count is not known to be warp-uniform)
        const int n = __shfl_sync(0xffffffffu, launch_events(g.c2.n_dyn, g.c2.dyn_base, g.c2.n_events), 0);
        const int lg = enc_split(n, gridDim.x), nu = n << lg;
        if (warp < 4) {
            EncWarp w;
            w.bar = bar;
            w.abort = abort;
            w.sb = smem_u32(smem);
            w.tmem = __shfl_sync(0xffffffffu, tmem, 0);
            w.nu = nu;
            w.lg = lg;
            // a test of the bounded waits: the wait gives up after stall_test_us, before any MMA
            if (g.c2.stall_test_us && warp == 1)
                ok = mbar_wait_warp(&bar[E::NEVER], 0, abort, 1000ull * g.c2.stall_test_us);
            if (ok) {
                if (warp == 1) ok = enc_mma2<E>(w);
                else if (warp == 2) ok = enc_mma3<E>(w);
                else ok = enc_mma4<E>(w);
                // every MMA issued above completes before TMEM is released
                if (elect_one()) mma_commit(bar + E::DRAIN + warp - 1);
                const uint64_t t0 = globaltimer();
                while (!mbar_try_wait(bar + E::DRAIN + warp - 1, 0)) if (globaltimer() - t0 > kWaitLimitNs) break;
            }
        } else {
            const int q = warp & 3, m = q * 32 + lane, wg = (warp >> 2) - 1;
            const uint32_t lt = tmem + ((uint32_t)(q * 32) << 16);
            if (wg < 4) {
                const bool two = wg < 2;
                const TcArgs &a = two ? g.c2 : g.c3;
                const int half = wg & 1;
                EncPool L;
                L.plane = (two ? C2::ROWS_E : C3::ROWS_E) * 16;
                L.ev_bytes = (size_t)L.plane * (two ? C2::POUT : C3::POUT);
                L.out = a.out + (m + kPad) * 16;
                L.bias = two ? E::PB2 : E::PB3;
                L.scale = two ? E::PS2 : E::PS3;
                L.out_inv = a.out_inv;
                L.cols = two ? C2::COUT : C3::COUT;
                L.len = two ? C2::L : C3::L;
                L.bufs = smem_u32(smem + (two ? E::OFF_P2 : E::OFF_P3));
                L.buf_bytes = two ? E::P2_BYTES : E::P3_BYTES;
                L.full = smem_u32(bar + (two ? E::T2F : E::T3F) + half);
                L.free = smem_u32(bar + (two ? E::T2E : E::T3E) + half);
                L.tile_free = smem_u32(bar + (two ? E::P2E : E::P3E));
                L.done = smem_u32(bar + (two ? E::D2 : E::D3));
                L.acc = lt + (two ? E::COL2 : E::COL3) + half * L.cols;
                L.up = two ? 2 : 1;
                ok = enc_pool_role<E, CAL>(L, par, a, half, m, nu, lg, abort);
            } else {
                int n4 = 0;
                for (int u = blockIdx.x; ok && u < nu; u += gridDim.x) {
                    const EncUnit x = enc_unit<E>(u, lg);
                    for (int k = x.k0; k < x.k1; ++k, ++n4) {
                        const int p = k * kTileM + m;
                        const bool valid = p < C4::L;
                        if (wg == 4) {     // enc4 accumulator -> the ConvT's operand
                            if (!mbar_wait(&bar[E::T4F], n4 & 1, abort) ||
                                (n4 > 0 && !mbar_wait(&bar[E::A2E], (n4 - 1) & 1, abort))) { ok = false; break; }
                            tc_fence_after();
                            epi_conv<C4, C4::COUT, CAL, 16>(g.c4, smem, par, E::PB4, E::PS4, lt + E::COL4, 0, 0, x.e, p, m,
                                                   valid, nullptr, lt + E::COLA);
                            tmem_st_wait();
                            tc_fence_before();
                            mbar_arrive(&bar[E::A2F]);
                            mbar_arrive(&bar[E::T4E]);
                        } else {           // ConvT accumulator -> u3
                            if (!mbar_wait(&bar[E::T5F], n4 & 1, abort)) { ok = false; break; }
                            tc_fence_after();
                            epi_up<C4, C4::N2, CAL, 16>(g.c4, par, E::PB5, E::PS5, lt + E::COL5, 0, x.e, p, valid, true);
                            tc_fence_before();
                            mbar_arrive(&bar[E::T5E]);
                        }
                    }
                }
            }
        }
    }
    if (!ok) {
        *abort = 1;
        raise_status(g.c2.status, PVF_ERR_TIMEOUT);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tmem, E::TMEM_COLS);
}

template <class N, bool CAL = false>
cudaError_t launch_enc(const EncArgs &g, cudaStream_t s, const ProfHook *prof) {
    using E = Enc<N>;
    if constexpr (E::C2::PREC == PVF_BF16 && !CAL)
        if (g.c2.amax) return launch_enc<N, true>(g, s, prof);       // calibration runs in the BF16 form
    if (g.c2.n_events <= 0) return cudaSuccess;
    // one CTA per SM: all of its tensor memory, so the whole shared memory is requested too
    constexpr int smem = 227 * 1024;
    int sms = 0;
    cudaError_t err = current_device_sms(&sms);
    if (err == cudaSuccess) err = prepare_kernel((const void *)k_enc_tc<E, CAL>, (size_t)smem, nullptr);
    if (err != cudaSuccess) return err;
    const int grid = (int64_t)g.c2.n_events * E::T4N < sms ? g.c2.n_events * E::T4N : sms;
    ProfScope ps(prof, "enc_up3", s);
    ParBlock<E::NPAR> par;
    par.set(E::PB2, g.c2.bias, E::C2::COUT);
    par.set(E::PB3, g.c3.bias, E::C3::COUT);
    par.set(E::PB4, g.c4.bias, E::C4::COUT);
    par.set(E::PB5, g.c4.bias2, E::C4::CUP);
    if constexpr (!is16(E::C2::PREC)) {
        par.set(E::PS2, g.c2.cs, E::C2::COUT);
        par.set(E::PS3, g.c3.cs, E::C3::COUT);
        par.set(E::PS4, g.c4.cs, E::C4::COUT);
        par.set(E::PS5, g.c4.cs2, E::C4::N2);
    }
    return launch_pdl(k_enc_tc<E, CAL>, dim3(grid), dim3(E::THREADS), (size_t)smem, s, g, par);
}
