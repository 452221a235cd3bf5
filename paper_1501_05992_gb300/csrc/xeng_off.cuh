// X-engine, tcgen05 FP8 form over CTA pairs (K2e): the tiles off the 256-input
// diagonal blocks of arrays of more than 256 inputs (those blocks: xeng_diag.cuh).
//
// One work item is (channel, tile I of 128 inputs, block J of 256 inputs left of
// I's own block): two 128 x 128 tiles of the triangle.  CTA r of the pair takes
// tile r of J as its 128 accumulator rows, and both take I as the columns in [Re | Im]
// form: 128 columns of real parts, then 128 of imaginary ones.  The operands are the
// nibbles' codes u = v + 8 (0..15; the E4M3 bit pattern u has the value u * 2^-9),
//
//   D += R_J . [R_I | -M_I],   D += M_J . [M_I | R_I]
//
// where the two halves of the 256 columns are the two CTAs' shares of the MMA's B
// operand: CTA 0 converts I into (R, M), CTA 1 into (-M, R), each J tile into
// (R, M).  A pair of SMs so reads 8 KB of operands per M=256 N=256 K=32 MMA and SM
// where one SM alone (M=128) reads 12 KB, and converts each I tile into two planes
// instead of three.
//
// The accumulator times 2^18, P, is an integer below 2^24 and exact.  It differs from the
// product of the samples by terms in each input's sums of codes alone: with E =
// sum(ur + um) and D = sum(um - ur) over the T samples (those past the end have code 8),
// Re V_ij = P_re - 8 E_i - 8 E_j + 128 T and Im V_ij = -P_im - 8 D_i + 8 D_j.  The
// converters add the codes up on their way, so that every CTA has the sums of both of its
// tiles, and the epilogue takes the terms off.
//
// Roles per CTA: warps 0-7 epilogue (two per quarter of the accumulator's lanes),
// warps 8-23 converters (two teams of eight that take alternate 64-sample stages;
// in a team, half of the threads convert I and half J), warp 24 TMEM allocation and
// (leader CTA) the MMA issuer, warp 25 the TMA producer (one thread; a ring of
// six 16 KB stages).  Each CTA loads both of its tiles, I as well as its own half of J:
// the TMA unit takes between four and five cycles per 128-byte row, i.e. 0.3 us for a
// stage's two tiles, which hides behind the converters; a box holds a whole stage of a
// tile, so a stage is two instructions.  Nothing is prefetched into L2 (a prefetch
// takes the same time).  TMEM holds two accumulators.
//
// What bounds it: a stage takes 0.43 us, 0.24 us of it the tensor pipe; the converters'
// turn-around (waits, decoding, stores, proxy fence) is the rest, and without their
// decoding a stage takes 0.36 us.  Against one 128-input tile per CTA with its
// neighbour's (the form before), together with xeng_pair.cu's and xeng_tile.cu's
// share: 1024 inputs x 128 channels x 10000 samples 2.04 -> 1.73 ms, 512 x 384 x 5000
// 0.80 -> 0.70 ms, 384 x 384 x 5000 0.49 -> 0.45 ms, 500 samples added to 512 x 768 0.49
// -> 0.42 ms.
#pragma once

#include <cuda.h>

#include <type_traits>

#include "internal.cuh"
#include "tc_common.cuh"

namespace corr {
namespace off {
namespace {

constexpr int kTile = 128;
constexpr int kTc = 64;                       // samples per stage
constexpr int kPlaneBytes = kTc * kTile;      // one plane or one packed tile: 8 KB
constexpr int kPackedStages = 6, kPackedBytes = 2 * kPlaneBytes;      // I | J
constexpr int kPlaneStages = 3, kPlaneStageBytes = 4 * kPlaneBytes;   // R_J | M_J | B1 | B2
constexpr int kOffA1 = 0, kOffA2 = kPlaneBytes, kOffB1 = 2 * kPlaneBytes, kOffB2 = 3 * kPlaneBytes;
constexpr int kEpiWarps = 8, kConvWarps = 16, kTeams = 2, kTeamWarps = kConvWarps / kTeams;
// a team's packed slots are its own, so that the parity it waits on is unambiguous
static_assert(kPackedStages % kTeams == 0 && kPlaneStages >= kTeams, "slots per team");
constexpr int kFirstConvWarp = kEpiWarps, kMmaWarp = kFirstConvWarp + kConvWarps, kTmaWarp = kMmaWarp + 1;
constexpr int kThreads = (kTmaWarp + 1) * 32;
constexpr int kTmemCols = 512;

// shared-memory map (offsets from the 1024-aligned base, the same in both CTAs)
constexpr int kSmPlanes = 0;
constexpr int kSmPacked = kSmPlanes + kPlaneStages * kPlaneStageBytes;
constexpr int kSmSums = kSmPacked + kPackedStages * kPackedBytes;
constexpr int kSumsBuf = 2 * 2 * kTile;                            // ints: [tile J, I][r, m][slot]
constexpr int kSmBars = kSmSums + 2 * kSumsBuf * 4;
constexpr int kNumBars = 2 * kPackedStages + 2 * kPlaneStages + 4 + 4 + 2;
constexpr int kSmMisc = kSmBars + kNumBars * 8;
constexpr int kSmemBytes = kSmMisc + 128;
static_assert(kSmemBytes <= 227 * 1024, "shared memory");

struct ArrayParams {
    int32_t *acc;
    int n, n_tiles, per_chan, n_stages, item_begin;
};

struct Params {
    ArrayParams a[kTcMaxOffParts];
    int n_arrays, n_items;
    DeviceStatus *status;
    long long wait_limit;
    int inject_stall;
    uint32_t one, fifteen;                    // multipliers of imad()
    long long drain_limit;
    int add_after;                            // a launch before zeroes what this one adds to
};

struct Tmaps {
    CUtensorMap m[kTcMaxOffParts];
};

struct Item {
    int a, f, i_tile, j_tile;                 // array, channel, tile I, first tile of block J
};

// Items of a channel: tile I with the blocks left of its own, I / 2 of them.
__host__ __device__ __forceinline__ int items_per_channel(int n_tiles)
{
    const int h = n_tiles / 2;                // sum of I / 2 over I < n_tiles
    return n_tiles % 2 ? h * h : h * (h - 1);
}

__device__ __forceinline__ Item decode_item(const Params &p, int item)
{
    Item it;
    it.a = 0;
    while (it.a + 1 < p.n_arrays && item >= p.a[it.a + 1].item_begin) ++it.a;
    const ArrayParams &A = p.a[it.a];
    const int local = item - A.item_begin;
    it.f = local / A.per_chan;
    int k = local - it.f * A.per_chan;
    for (it.i_tile = 2; it.i_tile + 1 < A.n_tiles && k >= it.i_tile / 2; ++it.i_tile) k -= it.i_tile / 2;
    it.j_tile = 2 * k;
    return it;
}

template <bool kZeroInvalid>
__device__ __forceinline__ void decode_codes(uint32_t w, const Params &p, uint32_t &ur, uint32_t &um)
{
    const uint32_t x = w ^ 0x88888888u;           // (one XOR for both nibbles: one mask each then)
    um = x & 0x0F0F0F0Fu;
    ur = (x >> 4) & 0x0F0F0F0Fu;
    if (kZeroInvalid) {
        // a nibble code of 8 has u == 0 (bit 4 of u + 15 clear): 0 + 0i is u = 8, 8
        const uint32_t ok = imad(ur, p.one, 0x0F0F0F0Fu) & imad(um, p.one, 0x0F0F0F0Fu) & 0x10101010u;
        const uint32_t low = imad(ok >> 4, p.fifteen, 0u);
        ur = (ur & low) | (0x08080808u & ~low);
        um = (um & low) | (0x08080808u & ~low);
    }
}

// The items first_item, first_item + item_step, ... of a launch, by this pair of CTAs.
template <bool kFresh, bool kZeroInvalid>
__device__ __forceinline__ void off_body(const Tmaps &tmaps, const Params &p, uint8_t *smem, int first_item,
                                         int item_step)
{
    const uint32_t sbase = smem_u32(smem);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = int(cluster_rank());

    int *sums = reinterpret_cast<int *>(smem + kSmSums);
    const uint32_t bars = sbase + kSmBars;
    auto bar_packed_full = [&](int s) { return bars + 8u * s; };
    auto bar_packed_empty = [&](int s) { return bars + 8u * (kPackedStages + s); };
    constexpr int kP = 2 * kPackedStages;
    auto bar_plane_full = [&](int s) { return bars + 8u * (kP + s); };                // leader's is used
    auto bar_plane_empty = [&](int s) { return bars + 8u * (kP + kPlaneStages + s); };
    constexpr int kB = kP + 2 * kPlaneStages;
    auto bar_acc_full = [&](int b) { return bars + 8u * (kB + b); };
    auto bar_acc_empty = [&](int b) { return bars + 8u * (kB + 2 + b); };              // leader's is used
    auto bar_sums_full = [&](int b) { return bars + 8u * (kB + 4 + b); };
    auto bar_sums_empty = [&](int b) { return bars + 8u * (kB + 6 + b); };
    const uint32_t bar_drain = bars + 8u * (kB + 8), bar_never = bars + 8u * (kB + 9);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + kSmMisc);
    volatile int *abort = reinterpret_cast<volatile int *>(smem + kSmMisc + 8);
    volatile int *epi_ok = reinterpret_cast<volatile int *>(smem + kSmMisc + 16);

    if (threadIdx.x == 0) {
        for (int s = 0; s < kPackedStages; ++s) {
            mbar_init(bar_packed_full(s), 1);
            mbar_init(bar_packed_empty(s), kTeamWarps);
        }
        for (int s = 0; s < kPlaneStages; ++s) {
            mbar_init(bar_plane_full(s), 2 * kTeamWarps);
            mbar_init(bar_plane_empty(s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(bar_acc_full(b), 1);
            mbar_init(bar_acc_empty(b), 2 * kEpiWarps);
            mbar_init(bar_sums_full(b), kConvWarps);
            mbar_init(bar_sums_empty(b), kEpiWarps);
        }
        mbar_init(bar_drain, 1);
        mbar_init(bar_never, 1);
        *abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (int a = 0; a < p.n_arrays; ++a)
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmaps.m[a])) : "memory");
    }
    for (int e = threadIdx.x; e < 2 * kSumsBuf; e += blockDim.x) sums[e] = 0;
    __syncthreads();
    if (warp == kMmaWarp) {
        tmem_alloc<true>(smem_u32(tmem_slot), kTmemCols);
    }
    fence_before();
    __syncthreads();
    cluster_sync();            // both CTAs' barriers are initialised and their TMEM is allocated
    fence_after();
    const uint32_t tmem = *tmem_slot;
    let_next_launch_start();

    if (warp == kTmaWarp) {
        // ------------------------------------------------- TMA producer --
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0, issued = 0, issued_phase = 0;
            bool ok = true;
            for (int item = first_item; ok && item < p.n_items; item += item_step) {
                const Item it = decode_item(p, item);
                const int n_stages = p.a[it.a].n_stages;
                const CUtensorMap *tmap = &tmaps.m[it.a];
                const int xi = it.i_tile * kTile, xj = (it.j_tile + rank) * kTile;
                for (int s = 0; s < n_stages; ++s) {
                    if (!mbar_wait(bar_packed_empty(stage), phase ^ 1u, abort, p.status, 1, p.wait_limit)) {
                        ok = false;
                        break;
                    }
                    const uint32_t full = bar_packed_full(stage), dst = sbase + kSmPacked + stage * kPackedBytes;
                    mbar_expect_tx(full, kPackedBytes);
                    tma_load_3d(dst, tmap, full, xi, it.f, s * kTc);
                    tma_load_3d(dst + kPlaneBytes, tmap, full, xj, it.f, s * kTc);
                    issued |= 1u << stage;
                    issued_phase = (issued_phase & ~(1u << stage)) | (phase << stage);
                    if (++stage == kPackedStages) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
            }
            // every issued load must have landed before the CTA may exit
            for (int k = 0; k < kPackedStages; ++k) {
                if (!((issued >> k) & 1u)) continue;
                const long long t0 = clock64();
                while (!mbar_try(bar_packed_full(k), (issued_phase >> k) & 1u) && clock64() - t0 < p.drain_limit) {
                }
            }
        }
    } else if (warp == kMmaWarp) {
        // ------------------------------------- MMA issuer (leader CTA) --
        if (rank == 0) {
            const uint64_t desc = smem_desc(sbase + kSmPlanes, kPlaneBytes, 1024);
            const uint64_t dA1 = desc + (kOffA1 >> 4), dA2 = desc + (kOffA2 >> 4), dB1 = desc + (kOffB1 >> 4),
                           dB2 = desc + (kOffB2 >> 4);
            int stage = 0, local = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int item = first_item; ok && item < p.n_items; item += item_step, ++local) {
                const int n_stages = p.a[decode_item(p, item).a].n_stages;
                const int slot = local & 1;
                if (!mbar_wait(bar_acc_empty(slot), (uint32_t(local >> 1) & 1u) ^ 1u, abort, p.status, 2,
                               p.wait_limit))
                    break;
                fence_after();
                const uint32_t t = tmem + uint32_t(slot * 256);
                uint32_t accum = 0;
                for (int s = 0; s < n_stages; ++s) {
                    if (!mbar_wait(bar_plane_full(stage), phase, abort, p.status, 3, p.wait_limit)) {
                        ok = false;
                        break;
                    }
                    fence_after();
                    const uint64_t so = uint64_t((stage * kPlaneStageBytes) >> 4);
                    if (lane == 0) {
                        mma_f8_pair(t, dA1 + so, dB1 + so, accum);
                        mma_f8_pair(t, dA2 + so, dB2 + so, 1);
                        mma_f8_pair(t, dA1 + so + 256u, dB1 + so + 256u, 1);
                        mma_f8_pair(t, dA2 + so + 256u, dB2 + so + 256u, 1);
                        commit_both(bar_plane_empty(stage));
                    }
                    __syncwarp();
                    accum = 1;
                    if (++stage == kPlaneStages) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
                if (!ok) break;
                if (lane == 0) commit_both(bar_acc_full(slot));
                __syncwarp();
            }
            // drain all MMAs issued by this thread before TMEM is released
            if (lane == 0) commit_own(bar_drain);
            __syncwarp();
            const long long t0 = clock64();
            while (!mbar_try(bar_drain, 0) && clock64() - t0 < p.drain_limit) {
            }
        }
    } else if (warp >= kFirstConvWarp) {
        // ----------------------------------------------------- converters --
        // Thread u of a team owns chunk column c (16 inputs) of one tile (q < 16: I,
        // else J) and rows (q mod 16) + 16 k, k < 4, of each of the team's stages.
        const int ci = warp - kFirstConvWarp, team = ci / kTeamWarps;
        const int u = (ci % kTeamWarps) * 32 + lane, c = u & 7, q = u >> 3;
        const bool tile_i = q < 16;                       // the same for a warp (q >> 2)
        const int row0 = q & 15;
        const uint32_t src_off = uint32_t(kSmPacked + (tile_i ? 0 : kPlaneBytes) + row0 * 128 + c * 16);
        const uint32_t swz = uint32_t(row0 * 128 + ((c ^ (row0 & 7)) << 4));
        // J: R, M; I in CTA 0: R, M; I in CTA 1: -M, R
        const bool swap = tile_i && rank == 1;
        const uint32_t off_r = uint32_t(kSmPlanes) + swz + (tile_i ? (swap ? kOffB2 : kOffB1) : kOffA1);
        const uint32_t off_m = uint32_t(kSmPlanes) + swz + (tile_i ? (swap ? kOffB1 : kOffB2) : kOffA2);
        uint32_t g_end = 0, g = uint32_t(team);
        int pstage = team, cstage = team, local = 0;
        uint32_t pphase = 0, cphase = 1;
        bool ok = true;
        for (int item = first_item; ok && item < p.n_items; item += item_step, ++local) {
            g_end += uint32_t(p.a[decode_item(p, item).a].n_stages);
            // per-input code sums of this thread's 16 inputs: byte lanes (<= 16 rows of
            // codes <= 15 between widenings), then 16-bit lanes
            uint32_t b8[2][4], s16lo[2][4], s16hi[2][4];
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int k = 0; k < 4; ++k) b8[m][k] = s16lo[m][k] = s16hi[m][k] = 0;
            int since_widen = 0;
            for (; g < g_end; g += kTeams) {
                if (!mbar_wait(bar_packed_full(pstage), pphase, abort, p.status, 4, p.wait_limit) ||
                    !mbar_wait(bar_plane_empty(cstage), cphase, abort, p.status, 5, p.wait_limit)) {
                    ok = false;
                    break;
                }
                const uint8_t *src = smem + pstage * kPackedBytes + src_off;
                uint8_t *dr = smem + cstage * kPlaneStageBytes + off_r, *dm = smem + cstage * kPlaneStageBytes + off_m;
                auto convert = [&](auto negate) {         // the m plane holds -M
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const uint4 w = *reinterpret_cast<const uint4 *>(src + k * 16 * 128);
                        const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
                        uint32_t R[4], M[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            decode_codes<kZeroInvalid>(ww[e], p, R[e], M[e]);
                            b8[0][e] = imad(R[e], p.one, b8[0][e]);
                            b8[1][e] = imad(M[e], p.one, b8[1][e]);
                            if (decltype(negate)::value) M[e] |= 0x80808080u;
                        }
                        *reinterpret_cast<uint4 *>(dr + k * 16 * 128) = make_uint4(R[0], R[1], R[2], R[3]);
                        *reinterpret_cast<uint4 *>(dm + k * 16 * 128) = make_uint4(M[0], M[1], M[2], M[3]);
                    }
                };
                if (swap) convert(std::true_type{});
                else convert(std::false_type{});
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) {
                    remote_arrive(map_rank(bar_plane_full(cstage), 0));
                    mbar_arrive(bar_packed_empty(pstage));
                }
                pstage += kTeams;
                if (pstage >= kPackedStages) {
                    pstage -= kPackedStages;
                    pphase ^= 1u;
                }
                cstage += kTeams;
                if (cstage >= kPlaneStages) {
                    cstage -= kPlaneStages;
                    cphase ^= 1u;
                }
                if (++since_widen == 4) {
                    since_widen = 0;
#pragma unroll
                    for (int m = 0; m < 2; ++m)
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            s16lo[m][k] += b8[m][k] & 0x00FF00FFu;
                            s16hi[m][k] += (b8[m][k] >> 8) & 0x00FF00FFu;
                            b8[m][k] = 0;
                        }
                }
            }
            if (!ok) break;
            // reduce over the four lanes that share chunk column c (16-bit lanes stay
            // below 4 x 256 x 4 x 15 < 2^16), then hand the sums to the epilogue
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    s16lo[m][k] += b8[m][k] & 0x00FF00FFu;
                    s16hi[m][k] += (b8[m][k] >> 8) & 0x00FF00FFu;
                    s16lo[m][k] += __shfl_xor_sync(0xFFFFFFFFu, s16lo[m][k], 8);
                    s16lo[m][k] += __shfl_xor_sync(0xFFFFFFFFu, s16lo[m][k], 16);
                    s16hi[m][k] += __shfl_xor_sync(0xFFFFFFFFu, s16hi[m][k], 8);
                    s16hi[m][k] += __shfl_xor_sync(0xFFFFFFFFu, s16hi[m][k], 16);
                }
            const int buf = local & 1;
            if (!mbar_wait(bar_sums_empty(buf), ((local >> 1) & 1) ^ 1, abort, p.status, 6, p.wait_limit)) break;
            __syncwarp();
            if (lane < 8) {
                int *sb = sums + buf * kSumsBuf + (tile_i ? 2 * kTile : 0);
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    int *row_sums = sb + m * kTile;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int n0 = c * 16 + 4 * k;
                        atomicAdd(row_sums + sum_slot(n0 + 0), int(s16lo[m][k] & 0xFFFFu));
                        atomicAdd(row_sums + sum_slot(n0 + 1), int(s16hi[m][k] & 0xFFFFu));
                        atomicAdd(row_sums + sum_slot(n0 + 2), int(s16lo[m][k] >> 16));
                        atomicAdd(row_sums + sum_slot(n0 + 3), int(s16hi[m][k] >> 16));
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_sums_full(buf));
        }
    } else {
        // ------------------------------------------------------- epilogue --
        const int q = warp & 3, wp = warp >> 2;      // lane quarter; which of its two warps
        const int il = q * 32 + lane;                // this thread's input of its J tile
        int local = 0, votes = 0;
        bool ok = true;
        if (!kFresh && p.add_after) wait_for_launch_before();
        // the epilogue warps decide together whether to go on (two sets of votes in turn)
        auto agree = [&](bool mine) {
            volatile int *const v = epi_ok + kEpiWarps * (votes++ & 1);
            if (lane == 0) v[warp] = mine ? 1 : 0;
            named_sync(2, kEpiWarps * 32);
            bool all = true;
#pragma unroll
            for (int w = 0; w < kEpiWarps; ++w) all = all && v[w] != 0;
            return all;
        };
        if (p.inject_stall)      // test hook: a wait that nothing ever satisfies
            ok = agree(warp_wait(bar_never, 0, abort, p.status, 9, lane, p.wait_limit, 64));
        for (int item = first_item; ok && item < p.n_items; item += item_step, ++local) {
            const Item it = decode_item(p, item);
            const int n_in = p.a[it.a].n;
            uint8_t *const out_f =
                reinterpret_cast<uint8_t *>(p.a[it.a].acc) + (size_t)it.f * size_t(n_pairs(n_in)) * 8;
            const int slot = local & 1;
            const uint32_t ph = uint32_t(local >> 1) & 1u;
            ok = agree(mbar_wait(bar_acc_full(slot), ph, abort, p.status, 7, p.wait_limit) &&
                       mbar_wait(bar_sums_full(slot), ph, abort, p.status, 8, p.wait_limit));
            if (!ok) break;
            fence_after();
            // with E = sum(ur + um), D = sum(um - ur) of an input (a: this lane's, b: a
            // column's) and P the TMEM value times 2^18 (an exact integer below 2^24):
            //   Re V_ij = P_re - 8 E_b + (128 T - 8 E_a),  Im V_ij = -P_im - 8 D_b + 8 D_a
            // in fp32 on integers; adding 1.5 * 2^23 leaves V (|V| <= 128 T <= 2^22) as the
            // low bits of the encoding.  The column terms replace I's sums, as floats in
            // column order: -8 E_b, then -8 D_b.
            int *const sb = sums + slot * kSumsBuf;
            float *const col = reinterpret_cast<float *>(sb + 2 * kTile);
            const int Sr = sb[sum_slot(il)], Sm = sb[kTile + sum_slot(il)];
            const int Br = sb[2 * kTile + sum_slot(il)], Bm = sb[3 * kTile + sum_slot(il)];
            named_sync(2, kEpiWarps * 32);               // every sum has been read
            if (wp == 0) col[il] = float(-8 * (Br + Bm));
            else col[kTile + il] = float(-8 * (Bm - Br));
            named_sync(2, kEpiWarps * 32);
            const float row_re = float(128 * p.a[it.a].n_stages * kTc - 8 * (Sr + Sm)) + 12582912.0f;
            const float row_im = float(8 * (Sm - Sr)) + 12582912.0f;
            const uint32_t taddr = tmem + uint32_t(slot * 256) + (uint32_t(q * 32) << 16);
            const int i0 = it.i_tile * kTile, j = (it.j_tile + rank) * kTile + il;
#pragma unroll 1
            for (int c0 = 16 * wp; c0 < kTile && i0 + c0 < n_in; c0 += 32) {
                uint32_t xr[16], xi[16];
                tmem_ld16(taddr + c0, xr);
                tmem_ld16(taddr + kTile + c0, xi);
                tmem_wait_ld();
                int2 v[16];
#pragma unroll
                for (int k = 0; k < 16; k += 2) {
                    const float2 cr = *reinterpret_cast<const float2 *>(col + c0 + k),
                                 ci = *reinterpret_cast<const float2 *>(col + kTile + c0 + k);
                    const float2 re = __fadd2_rn(
                        __ffma2_rn(make_float2(__uint_as_float(xr[k]), __uint_as_float(xr[k + 1])),
                                   make_float2(262144.0f, 262144.0f), cr),
                        make_float2(row_re, row_re));
                    const float2 im = __fadd2_rn(
                        __ffma2_rn(make_float2(__uint_as_float(xi[k]), __uint_as_float(xi[k + 1])),
                                   make_float2(-262144.0f, -262144.0f), ci),
                        make_float2(row_im, row_im));
                    v[k] = make_int2(__float_as_int(re.x) - 0x4B400000, __float_as_int(im.x) - 0x4B400000);
                    v[k + 1] = make_int2(__float_as_int(re.y) - 0x4B400000, __float_as_int(im.y) - 0x4B400000);
                }
                put_rows16<kFresh>(out_f, i0 + c0, j, n_in, lane, i0 + c0 + 15 < n_in, v);
            }
            fence_before();
            __syncwarp();
            if (lane == 0) remote_arrive(map_rank(bar_acc_empty(slot), 0));
            // every warp has read this item's terms: clear them for the item that reuses
            // the buffer, then release it
            named_sync(2, kEpiWarps * 32);
            for (int e = threadIdx.x; e < kSumsBuf; e += kEpiWarps * 32) sb[e] = 0;
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_sums_empty(slot));
        }
    }

    __syncwarp();
    fence_before();
    cluster_sync();            // no CTA leaves or frees TMEM while its pair may still use either
    fence_after();
    if (warp == kMmaWarp) {
        tmem_dealloc<true>(tmem, kTmemCols);
    }
    wait_for_launch_before();
}

// The parameters of a launch over every channel of `count` arrays or parts of one.
inline cudaError_t make_params(const TcArray *arrays, const CUtensorMap *maps, int count, DeviceStatus *status,
                               const TcOptions &opt, Params &prm, Tmaps &tm)
{
    if (count < 1 || count > kTcMaxOffParts) return cudaErrorInvalidValue;
    long long items = 0;
    for (int k = 0; k < count; ++k) {
        const TcArray &A = arrays[k];
        tm.m[k] = maps[k];
        ArrayParams &P = prm.a[k];
        P.acc = A.acc;
        P.n = A.n;
        P.n_tiles = (A.n + kTile - 1) / kTile;
        if (P.n_tiles < 3) return cudaErrorInvalidValue;
        P.per_chan = items_per_channel(P.n_tiles);
        P.n_stages = (A.nt + kTc - 1) / kTc;
        P.item_begin = int(items);
        items += (long long)A.n_chan * P.per_chan;
    }
    if (items > 0x3FFFFFFF) return cudaErrorInvalidValue;
    prm.n_arrays = count;
    prm.n_items = int(items);
    prm.status = status;
    prm.wait_limit = opt.wait_limit > 0 ? opt.wait_limit : kDefaultWaitLimit;
    prm.drain_limit = kDefaultWaitLimit;
    prm.add_after = opt.add_after ? 1 : 0;
    prm.inject_stall = opt.inject_stall ? 1 : 0;
    prm.one = 1u;
    prm.fifteen = 15u;
    return cudaSuccess;
}

}  // namespace
}  // namespace off
}  // namespace corr
