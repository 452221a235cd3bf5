// X-engine, tcgen05 FP8 form (K2c): the blocks on the diagonal of a channel's
// triangle.
//
// What the path computes is Eq. 3 (Section 2) integrated over time (Section 3.4.2):
// V_ij(f) = sum_t x_i(t,f) conj(x_j(t,f)) for j <= i, straight from the packed 4+4-bit
// voltages volt[t][f][n] (Appendix A, Appendix C "GPU Input"), into the packed lower
// triangle of Appendix C "GPU Output".  The paper's GPU kernel (xGPU) tiles baselines
// per thread block and integrates in registers (Section 3.4.2, Eq. 4); here tiles of
// 128 x 128 inputs are integrated in tensor memory (TMEM) by tcgen05.mma.
//
// One work item is a (channel, 256-input block): a pair of CTAs (cta_group::2)
// computes the block's whole 256 x 256 Hermitian product, CTA r of the pair
// holding input tile r (128 inputs) as the rows of its accumulator (kPair), or a
// (channel, last 128-input tile): one CTA does the same for the tile alone.
//
// The real matrix.  With x = r + i m and q = r - m,
//
//   W[a][b] = sum_t q_a q_b + 2 r_a m_b = Re V_ab - Im V_ab
//
// and V is Hermitian, so W[b][a] = Re V_ab + Im V_ab: W holds every product of
// the block once, Re V_ij = (W[j][i] + W[i][j]) / 2 and Im V_ij = (W[j][i] -
// W[i][j]) / 2.  That is two real products per pair of 128-input tiles and
// none wasted, where a diagonal tile in [Re | Im] form (xeng_off.cuh) computes
// four and throws half of them away: 8 tile products per 256 inputs against 12.
//
// Encoding (exact): the three planes q in [-15, 15], r in [-8, 7] and 2 m in
// [-16, 14] are E4M3 in sign and magnitude; the bit pattern u of an integer u
// <= 16 has the value u * 2^-9, so W is the accumulator times 2^18 with no
// correction terms.  A sample's terms stay below 225 + 128 = 353 in magnitude,
// so FP32 sums are exact (< 2^24) up to kTcMaxSamples = 32768 samples.  Samples
// past the end and inputs past n are zero bytes.
//
// Per 64-sample stage and CTA: 8 KB of packed samples become the three planes
// (24 KB), and the leader CTA issues four MMAs of M=256 N=256 K=32 (q.q and
// r.2m of the two K halves), each reading 4 KB of A and 4 KB of B from each
// CTA's shared memory.  The converters read the packed samples straight into
// registers (as fast as a TMA ring with 64 KB of packed slots beside the planes,
// 1.33 against 1.32 ms, and it needs no tensor map).
//
// What bounds it: power.  On the full band (256 inputs x 3072 channels x 5000
// samples) it takes 1.30-1.37 ms, against 1.68-1.78 ms for a kernel of 128-input tiles
// in [Re | Im] form, at the card's 1400 W; the MMAs alone take 1.05 ms at the same
// power and the converters alone 0.71 ms at 585 W, so what counts is work per
// integration: MMAs (two thirds of that kernel's) and instructions.  The tensor
// pipe is 67 % busy, the ALU pipe 52 % (a quarter of the band).  Short
// launches are bound by the epilogue's exchange and stores (adding 500 samples to the
// full band's triangle: 0.38 ms, of which 0.28 ms is what the adds alone take in L2).  One tile
// alone is bound by its MMAs (M=128 N=128 reads 8 KB of operands in 64 cycles) and
// loads: 128 inputs x 1520 channels x 5000 samples 0.33 -> 0.31 ms, 500 samples added
// to 768 channels 67 -> 35 us.
//
// Rows on any byte boundary (input counts that are no multiple of 16) are read
// as they are, as aligned words: 250 inputs x 760 channels x 5000 samples 0.47 ms
// (0.54 ms with invalid samples zeroed) against 0.33 ms for 256 inputs, where a
// copy into padded rows first took 0.41 ms by itself.  (A lane per word of a row
// instead of four words of a 16-byte chunk: 0.53 and 0.60 ms, for its 4-byte
// plane stores and two shuffles per word.)
//
// Roles per CTA (persistent; items are strided over the pairs):
//   warps 0-7    epilogue, two warps per quarter of the accumulator's lanes
//   warps 8-23   converters: four teams of four warps (one per scheduler) that
//                take the stages in turn
//   warp 24      TMEM allocation; in the leader CTA the MMA issuer
//
// Incoherent beam (launches that ask for it): the converters square the magnitudes
// they have decoded (two dp4a a word), add them up per row over the lanes, and add
// each row's sum to beam[t][f].  256 inputs x 768 channels x 5000 samples 0.34 ms
// without, 0.40 ms with it (0.42 ms squaring the packed nibbles instead).
//
// Epilogue.  A thread holds accumulator row a of its tile, so an output (i, j)
// needs W[j][i] from the lane of j and W[i][j] from the lane of i: one of the
// two goes through shared memory.  The lanes of j write 32 consecutive elements
// of packed row i per store.  Each CTA emits its diagonal tile, exchanged within
// the CTA, and half of the off-diagonal tile's 128 rows (tile 1 against the
// columns of tile 0): CTA 0 the first 64, whose W[i][j] CTA 1 sends through
// distributed shared memory into CTA 0's inbox, CTA 1 the others, whose W[j][i]
// CTA 0 sends (st.async, counted by the inbox's barrier: plain stores and a
// cluster-scope release wait for the thread's stores to the output too, 0.36
// against 0.33 ms for 500 samples of the full band).  Of that half both operands
// are in shared memory, so that any warp can emit any of it: the quarters' shares of the
// diagonal tile are as 4 : 3 : 2 : 1 (j <= i), and its pieces go to the warps that
// have less, while TMEM is already free (500 samples of the full band 0.323 ->
// 0.295 ms, added 0.408 -> 0.383 ms, against halves emitted by quarter after a wait of
// all warps; one 1.28 MHz channel of 5000 samples 74.4 -> 72.6 us; 250 inputs lose
// 0.8 % on long integrations, which no arrangement of the
// same loops that was tried avoids for both kinds of rows).  TMEM holds two
// 256-column accumulators, so an item's epilogue overlaps the next item's main loop.
#pragma once

#include <mutex>

#include "internal.cuh"
#include "tc_common.cuh"

namespace corr {
namespace {

constexpr int kTile = 128;                    // inputs per CTA of a pair
constexpr int kTc = 64;                       // samples per pipeline stage
constexpr int kPlaneStages = 4;               // more slots gain nothing (5 and 6: 1.31 ms on the full band, 4: 1.29)
constexpr int kPlaneBytes = kTc * kTile;      // one E4M3 plane: 8 KB
constexpr int kOffQ = 0, kOffR = kPlaneBytes, kOffM = 2 * kPlaneBytes;
constexpr int kPlaneStageBytes = 3 * kPlaneBytes;
constexpr int kConvWarps = 16, kEpiWarps = 8;
constexpr int kTeams = 4, kTeamWarps = kConvWarps / kTeams;
// a team waits for its plane slot by parity, which is unambiguous while no more
// stages are being converted than there are slots
static_assert(kPlaneStages >= kTeams, "a slot per team");
constexpr int kUnits = kPlaneBytes / 16 / (kTeamWarps * 32);   // 16-byte pieces per thread and stage
constexpr int kFirstConvWarp = kEpiWarps, kMmaWarp = kFirstConvWarp + kConvWarps;
constexpr int kThreads = (kMmaWarp + 1) * 32;
// instruction descriptor of the single-tile form: as kIdescPair, M=128, N the tile's
// inputs rounded up to 16 (columns past them are never read back)
__device__ __forceinline__ uint32_t idesc_tile(int inputs)
{
    const uint32_t n = inputs >= 128 ? 128u : uint32_t((inputs + 15) & ~15);
    return (1u << 4) | (1u << 15) | (1u << 16) | ((n >> 3) << 17) | ((128u >> 4) << 24);
}

// shared-memory map (offsets from the 1024-aligned base, the same in both CTAs)
constexpr int kSmPlanes = 0;
// epilogue buffers: the CTA's diagonal tile (W[i][j]: row i holds the columns up to the
// end of its quarter, 32 q + 32), its own operand of its half of the off-diagonal tile
// (64 rows i of 128 columns j), and its inbox for the pair's operand; rows are padded
// by 16 bytes so that 16-byte stores down the rows spread over the banks
constexpr int kSmDiag = kSmPlanes + kPlaneStages * kPlaneStageBytes;
constexpr int kHalfPitch = kTile * 4 + 16, kHalfRows = 64;
constexpr int kDiagBytes = 32 * (4 * 16 + (32 + 64 + 96 + 128) * 4);
__device__ __forceinline__ int diag_pitch(int quarter) { return 128 * quarter + 144; }
__device__ __forceinline__ int diag_base(int quarter) { return 32 * (144 * quarter + 64 * quarter * (quarter - 1)); }
constexpr int kSmOwn = kSmDiag + kDiagBytes;
constexpr int kSmInbox = kSmOwn + kHalfRows * kHalfPitch;
constexpr int kSmBars = kSmInbox + kHalfRows * kHalfPitch;
constexpr int kNumBars = 2 * kPlaneStages + 4 + 4;
constexpr int kSmMisc = kSmBars + kNumBars * 8;
constexpr int kSmemBytes = kSmMisc + 128;
constexpr int kInboxBytes = kHalfRows * kTile * 4;                // sent per item
static_assert(kSmemBytes <= 227 * 1024, "shared memory");

struct ArrayParams {
    const uint8_t *volt;
    long long row_t;          // bytes from one sample of a channel to the next
    int ld;                   // bytes from one channel to the next
    int32_t *acc;
    int first;                // first input of the first block
    int n, n_chan, n_blocks, nt, n_stages, item_begin;
    int32_t *beam;
    int beam_ld, beam_avg, beam_t0;
    int f0, n_chan_all;       // the channels are f0 .. of n_chan_all
};

struct Params {
    ArrayParams a[kTcMaxArrays];
    int n_arrays, n_items;
    DeviceStatus *status;
    long long wait_limit;
    int inject_stall;
    uint32_t one, minus_one, fifteen, sixteen;   // multipliers of imad()
    int add_after;            // the launch before zeroes what this one adds to
    long long drain_limit;
};

struct Item {
    int a, f, base;                           // array, channel, first input of the block
};

__device__ __forceinline__ Item decode_item(const Params &p, int item)
{
    Item it;
    it.a = 0;
    while (it.a + 1 < p.n_arrays && item >= p.a[it.a + 1].item_begin) ++it.a;
    const ArrayParams &A = p.a[it.a];
    const int local = item - A.item_begin;
    it.f = local / A.n_blocks;
    it.base = A.first + (local - it.f * A.n_blocks) * 2 * kTile;
    return it;
}

// Planes of the four packed samples of w (real part in the high nibbles): q =
// r - m, r and 2 m as E4M3 sign and magnitude.  ur, um are v + 8 and |v| the
// byte-wise distance from the offset; the signs of r and m are their nibbles'
// top bits and that of q is the borrow of ur - um + 128.  With kZeroInvalid a
// sample with code 8 (u = 0) in either part becomes 0 + 0i (u = 8; the signs of
// its zeros do not matter).  With kPower the magnitudes' squares, 4 (r^2 + m^2) over
// the four samples, are added to `power`.
template <bool kZeroInvalid, bool kPower>
__device__ __forceinline__ void planes4(uint32_t w, const Params &p, uint32_t &Q, uint32_t &R, uint32_t &M, int2 &power)
{
    const uint32_t x = w ^ 0x88888888u;
    uint32_t um = x & 0x0F0F0F0Fu;
    uint32_t ur = (x >> 4) & 0x0F0F0F0Fu;
    const uint32_t sign_r = w & 0x80808080u, w16 = imad(w, p.sixteen, 0u);
    if (kZeroInvalid) {
        // bit 4 of u + 15: u != 0
        const uint32_t ok = imad(ur, p.one, 0x0F0F0F0Fu) & imad(um, p.one, 0x0F0F0F0Fu) & 0x10101010u;
        const uint32_t low = imad(ok >> 4, p.fifteen, 0u);
        ur = (ur & low) | (0x08080808u & ~low);
        um = (um & low) | (0x08080808u & ~low);
    }
    const uint32_t t = imad(um, p.minus_one, imad(ur, p.one, 0x80808080u));
    Q = __vabsdiffu4(ur, um) | (~t & 0x80808080u);
    const uint32_t abs_r = __vabsdiffu4(ur, 0x08080808u), abs_2m = __vabsdiffu4(imad(um, p.one, um), 0x10101010u);
    R = abs_r | sign_r;
    M = abs_2m | (w16 & 0x80808080u);
    if (kPower) {
        power.x = int(__dp4a(abs_r, abs_r, uint32_t(power.x)));
        power.y = int(__dp4a(abs_2m, abs_2m, uint32_t(power.y)));
    }
}

__device__ __forceinline__ uint4 load16(const uint8_t *a)
{
    uint4 v;
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(a));
    return v;
}

// The items first_item, first_item + item_step, ... of a launch, by this CTA or pair of CTAs.
// kSpareWarps: the block has more warps than the roles take.
template <bool kPair, bool kAligned, bool kFresh, bool kZeroInvalid, bool kBeam, bool kSpareWarps = false>
__device__ __forceinline__ void block_body(const Params &p, uint8_t *smem, int first_item, int item_step)
{
    const uint32_t sbase = smem_u32(smem);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = kPair ? int(cluster_rank()) : 0;
    constexpr int kSlotCols = kPair ? 256 : 128, kTmemCols = 2 * kSlotCols;   // two accumulators

    const uint32_t bars = sbase + kSmBars;
    auto bar_plane_full = [&](int s) { return bars + 8u * s; };                  // leader's is used
    auto bar_plane_empty = [&](int s) { return bars + 8u * (kPlaneStages + s); };
    constexpr int kB = 2 * kPlaneStages;
    auto bar_acc_full = [&](int b) { return bars + 8u * (kB + b); };
    auto bar_acc_empty = [&](int b) { return bars + 8u * (kB + 2 + b); };                   // leader's is used
    const uint32_t bar_drain = bars + 8u * (kB + 4), bar_never = bars + 8u * (kB + 5);
    const uint32_t bar_in_full = bars + 8u * (kB + 6);       // the pair's rows are in this CTA's inbox
    const uint32_t bar_in_free = bars + 8u * (kB + 7);       // the pair's inbox may be written
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + kSmMisc);
    volatile int *abort = reinterpret_cast<volatile int *>(smem + kSmMisc + 8);
    volatile int *epi_ok = reinterpret_cast<volatile int *>(smem + kSmMisc + 16);
    volatile int *sent = reinterpret_cast<volatile int *>(smem + kSmMisc + 96);   // items sent: to this CTA, by it

    if (threadIdx.x == 0) {
        for (int s = 0; s < kPlaneStages; ++s) {
            mbar_init(bar_plane_full(s), (kPair ? 2 : 1) * kTeamWarps);
            mbar_init(bar_plane_empty(s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(bar_acc_full(b), 1);
            mbar_init(bar_acc_empty(b), (kPair ? 2 : 1) * kEpiWarps);
        }
        mbar_init(bar_drain, 1);
        mbar_init(bar_never, 1);
        mbar_init(bar_in_full, 1);
        mbar_init(bar_in_free, kEpiWarps);
        *abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (warp == kMmaWarp) {
        tmem_alloc<kPair>(smem_u32(tmem_slot), kTmemCols);
    }
    fence_before();
    __syncthreads();
    if (kPair) cluster_sync();      // both CTAs' barriers are initialised and their TMEM is allocated
    fence_after();
    const uint32_t tmem = *tmem_slot;
    let_next_launch_start();

    if (warp == kMmaWarp) {
        // ------------------------------------- MMA issuer (leader CTA) --
        // the whole warp waits and lane 0 issues: waits of one lane beside parked ones
        // are slower (1.38 against 1.35 ms on the full band)
        if (rank == 0) {
            const uint64_t desc = smem_desc(sbase + kSmPlanes, kPlaneBytes, 1024);
            const uint64_t dQ = desc + (kOffQ >> 4), dR = desc + (kOffR >> 4), dM = desc + (kOffM >> 4);
            uint32_t idesc = 0;
            auto mma = [&](uint32_t d, uint64_t a, uint64_t b, uint32_t accumulate) {
                if (kPair) mma_f8_pair(d, a, b, accumulate);
                else mma_f8(d, a, b, idesc, accumulate);
            };
            auto commit = [&](uint32_t bar) {
                if (kPair) commit_both(bar);
                else mma_commit(bar);
            };
            int stage = 0;
            uint32_t phase = 0;
            int local = 0;
            bool ok = true;
            for (int item = first_item; ok && item < p.n_items; item += item_step, ++local) {
                const Item it = decode_item(p, item);
                const int n_stages = p.a[it.a].n_stages;
                if (!kPair) idesc = idesc_tile(p.a[it.a].n - it.base);
                const int slot = local & 1;
                if (!mbar_wait(bar_acc_empty(slot), (uint32_t(local >> 1) & 1u) ^ 1u, abort, p.status, 2,
                                  p.wait_limit))
                    break;
                fence_after();
                const uint32_t t = tmem + uint32_t(slot * kSlotCols);
                uint32_t accum = 0;
                for (int s = 0; s < n_stages; ++s) {
                    if (!mbar_wait(bar_plane_full(stage), phase, abort, p.status, 3, p.wait_limit)) {
                        ok = false;
                        break;
                    }
                    fence_after();
                    const uint64_t so = uint64_t((stage * kPlaneStageBytes) >> 4);
                    if (lane == 0) {
                        mma(t, dQ + so, dQ + so, accum);
                        mma(t, dR + so, dM + so, 1);
                        mma(t, dQ + so + 256u, dQ + so + 256u, 1);
                        mma(t, dR + so + 256u, dM + so + 256u, 1);
                        commit(bar_plane_empty(stage));
                    }
                    __syncwarp();
                    accum = 1;
                    if (++stage == kPlaneStages) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
                if (!ok) break;
                if (lane == 0) commit(bar_acc_full(slot));
                __syncwarp();
            }
            // drain all MMAs issued by this thread before TMEM is released
            if (lane == 0) {
                if (kPair) commit_own(bar_drain);
                else mma_commit(bar_drain);
            }
            __syncwarp();
            const long long t0 = clock64();
            while (!mbar_try(bar_drain, 0) && clock64() - t0 < p.drain_limit) {
            }
        }
    } else if (kSpareWarps && warp > kMmaWarp) {
        // nothing to do
    } else if (warp >= kFirstConvWarp) {
        // ----------------------------------------------------- converters --
        // Team t converts the stages g (counted over all items of this CTA) with
        // g % kTeams == t, so each warp meets the barriers once per kTeams stages.
        // A thread owns chunk column c (16 inputs) of rows (samples) q + k kRowStep.
        // kAligned: rows start on 16-byte boundaries, a chunk is one load.  Otherwise a
        // chunk is the four aligned words from the one that holds its first byte; the
        // bytes past them come from the first word of the next lane's chunk, for the
        // row's last chunk (c = 7) from one more word that lane r of the warp loads for
        // the warp's r-th row.  A row's offset from a word boundary is the same for all
        // of a thread's rows (16 samples apart).
        const int ci = warp - kFirstConvWarp;
        const int u = (ci % kTeamWarps) * 32 + lane;
        const int c = u & 7, q = u >> 3;
        constexpr int kRowStep = kTeamWarps * 4;
        static_assert(kRowStep % 8 == 0, "a thread's rows share their swizzle");
        const uint32_t dst_off = uint32_t(kSmPlanes + q * 128 + ((c ^ (q & 7)) << 4));
        // the stage whose samples are being loaded: stage s of `item`
        int item = first_item, s = ci / kTeamWarps, n_stages = 0, rows = 0, whole = 0;
        long long row_t = 0;
        const uint8_t *ptr = nullptr;
        int32_t *beam = nullptr;
        int beam_avg = 1, beam_ld = 0, t_beam = 0;
        // rows on any byte: this thread's inputs from its chunk on, its rows' offset from
        // a word boundary, whether the item has such offsets; the extra word's address and
        // the number of samples it is there for; the array's bytes and whether the item
        // has words that reach over their ends
        int left = kTile, sh = 0, x_rows = 0;
        bool skew = false, edge = false;
        const uint8_t *x_ptr = nullptr, *lo = nullptr, *hi = nullptr;
        auto enter = [&] {                     // stage s of `item`, or of a later one past its end
            while (item < p.n_items) {
                const Item it = decode_item(p, item);
                const ArrayParams &A = p.a[it.a];
                n_stages = A.n_stages;
                if (s < n_stages) {
                    const int tile = it.base + rank * kTile;
                    const uint8_t *const first = A.volt + (long long)it.f * A.ld + tile;
                    row_t = A.row_t;
                    left = A.n - tile - c * 16;
                    ptr = first + c * 16 + (long long)(s * kTc + q) * row_t;
                    if (!kAligned) {
                        sh = int(reinterpret_cast<uintptr_t>(ptr) & 3);
                        ptr -= sh;
                        skew = ((reinterpret_cast<uintptr_t>(first) | uintptr_t(row_t)) & 3) != 0;
                        const int xt = s * kTc + (q & ~3) + (lane & 3) + (lane >> 2) * kRowStep;
                        x_ptr = first + kTile + (long long)xt * row_t;
                        const int xs = int(reinterpret_cast<uintptr_t>(x_ptr) & 3);
                        x_ptr -= xs;
                        x_rows = lane < 4 * kUnits && xs && A.n - tile - kTile + xs > 0 ? A.nt - xt : 0;
                        edge = words_reach_over(it.f + A.f0, A.n_chan_all, A.n);
                        lo = A.volt;
                        hi = A.volt + (A.nt - 1) * row_t + (long long)A.n_chan * A.ld;
                    }
                    // rows of this thread with a sample (none for a chunk past the inputs)
                    rows = left + sh > 0 ? A.nt - q - s * kTc : 0;
                    // stages of this item from s on whose loads need no bounds
                    whole = tile + kTile <= A.n && !edge ? A.nt / kTc - s : 0;
                    if (kBeam) {
                        beam = A.beam ? A.beam + it.f : nullptr;
                        beam_avg = A.beam_avg;
                        beam_ld = A.beam_ld;
                        t_beam = A.beam_t0 + s * kTc + q;
                    }
                    return;
                }
                s -= n_stages;
                item += item_step;
            }
        };
        // the word at a, without touching bytes outside the array
        auto load_word = [&](const uint8_t *a) {
            uint32_t v = 0;
            if (!edge || (a >= lo && a + 4 <= hi)) {
                v = __ldg(reinterpret_cast<const uint32_t *>(a));
            } else {
                for (int b = 0; b < 4; ++b)
                    if (a + b >= lo && a + b < hi) v |= uint32_t(__ldg(a + b)) << (8 * b);
            }
            return v;
        };
        uint4 w[kUnits];                       // this thread's samples of the team's next stage
        uint32_t wx = 0;
        auto load = [&] {
            const uint8_t *a = ptr;
            if (whole > 0) {
#pragma unroll
                for (int k = 0; k < kUnits; ++k, a += kRowStep * row_t) {
                    if (kAligned) {
                        w[k] = load16(a);
                    } else {
                        const uint32_t *v = reinterpret_cast<const uint32_t *>(a);
                        w[k] = make_uint4(__ldg(v), __ldg(v + 1), __ldg(v + 2), __ldg(v + 3));
                    }
                }
            } else {
#pragma unroll
                for (int k = 0; k < kUnits; ++k, a += kRowStep * row_t) {
                    w[k] = make_uint4(0u, 0u, 0u, 0u);
                    if (k * kRowStep < rows) {
                        if (kAligned) {
                            w[k] = load16(a);
                        } else {
                            w[k].x = load_word(a);
                            if (left + sh > 4) w[k].y = load_word(a + 4);
                            if (left + sh > 8) w[k].z = load_word(a + 8);
                            if (left + sh > 12) w[k].w = load_word(a + 12);
                        }
                    }
                }
            }
            if (!kAligned) {
                wx = 0;
                if (x_rows > 0) wx = load_word(x_ptr);
            }
        };
        enter();
        bool more = item < p.n_items;
        if (more) load();
        int cstage = ci / kTeamWarps;
        uint32_t cphase = 1;
        while (more) {
            int32_t *const b_ptr = beam;       // beam of the stage being converted
            const int b_avg = beam_avg, b_ld = beam_ld, b_t = t_beam, b_rows = rows;
            const int c_left = left, c_shift = 8 * sh;
            const bool c_skew = skew;
            int pw[kUnits];
            // the next stage of this team
            s += kTeams;
            if (s < n_stages) {
                ptr += (long long)(kTeams * kTc) * row_t;
                rows -= rows > 0 ? kTeams * kTc : 0;
                whole -= kTeams;
                t_beam += kTeams * kTc;
                if (!kAligned) {
                    x_ptr += (long long)(kTeams * kTc) * row_t;
                    x_rows -= kTeams * kTc;
                }
            } else {
                enter();
            }
            more = item < p.n_items;
            if (!more) rows = whole = x_rows = 0;
            if (!mbar_wait(bar_plane_empty(cstage), cphase, abort, p.status, 5, p.wait_limit)) break;
            uint8_t *dst = smem + cstage * kPlaneStageBytes + dst_off;
            if (!kAligned && c_skew) {
#pragma unroll
                for (int k = 0; k < kUnits; ++k) {
                    const uint32_t next = __shfl_down_sync(0xFFFFFFFFu, w[k].x, 1),
                                   over = __shfl_sync(0xFFFFFFFFu, wx, 4 * k + (lane >> 3));
                    w[k].x = __funnelshift_r(w[k].x, w[k].y, c_shift);
                    w[k].y = __funnelshift_r(w[k].y, w[k].z, c_shift);
                    w[k].z = __funnelshift_r(w[k].z, w[k].w, c_shift);
                    w[k].w = __funnelshift_r(w[k].w, c == 7 ? over : next, c_shift);
                }
            }
            if (!kAligned && c_left < 16) {    // bytes past the inputs
                auto mask = [&](int j) {
                    const int b = c_left - 4 * j;
                    return b >= 4 ? 0xFFFFFFFFu : b > 0 ? (1u << (8 * b)) - 1u : 0u;
                };
#pragma unroll
                for (int k = 0; k < kUnits; ++k) {
                    w[k].x &= mask(0);
                    w[k].y &= mask(1);
                    w[k].z &= mask(2);
                    w[k].w &= mask(3);
                }
            }
#pragma unroll
            for (int k = 0; k < kUnits; ++k) {
                const uint32_t ww[4] = {w[k].x, w[k].y, w[k].z, w[k].w};
                uint32_t Q[4], R[4], M[4];
                int2 power = make_int2(0, 0);
#pragma unroll
                for (int e = 0; e < 4; ++e) planes4<kZeroInvalid, kBeam>(ww[e], p, Q[e], R[e], M[e], power);
                if (kBeam) pw[k] = 4 * power.x + power.y;      // 4 (r^2 + m^2) over the 16 inputs
                uint8_t *d = dst + k * kRowStep * 128;
                *reinterpret_cast<uint4 *>(d + kOffQ) = make_uint4(Q[0], Q[1], Q[2], Q[3]);
                *reinterpret_cast<uint4 *>(d + kOffR) = make_uint4(R[0], R[1], R[2], R[3]);
                *reinterpret_cast<uint4 *>(d + kOffM) = make_uint4(M[0], M[1], M[2], M[3]);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) {
                if (kPair) remote_arrive(map_rank(bar_plane_full(cstage), 0));
                else mbar_arrive(bar_plane_full(cstage));
            }
            load();       // only now: the proxy fence above would wait for loads in flight
            cstage += kTeams;
            if (cstage >= kPlaneStages) {
                cstage -= kPlaneStages;
                cphase ^= 1u;
            }
            if (kBeam && b_ptr) {
                // total power of the tile's 128 inputs per row, over the 8 lanes of a
                // chunk row: each exchange halves the rows a lane still carries
                static_assert(!kBeam || kUnits == 4, "four rows per lane");
                const bool h4 = c & 4, h2 = c & 2;
                const int k0 = (h4 ? pw[2] : pw[0]) + __shfl_xor_sync(0xFFFFFFFFu, h4 ? pw[0] : pw[2], 4);
                const int k1 = (h4 ? pw[3] : pw[1]) + __shfl_xor_sync(0xFFFFFFFFu, h4 ? pw[1] : pw[3], 4);
                int v = (h2 ? k1 : k0) + __shfl_xor_sync(0xFFFFFFFFu, h2 ? k0 : k1, 2);
                v += __shfl_xor_sync(0xFFFFFFFFu, v, 1);
                const int k = (h4 ? 2 : 0) + (h2 ? 1 : 0);
                const int t = b_t + k * kRowStep;
                // the row's lane 0 knows whether the row has a sample (chunk 0 is always within n)
                const int live = __shfl_sync(0xFFFFFFFFu, b_rows, lane & ~7);
                if (!(c & 1) && k * kRowStep < live)
                    atomicAdd(b_ptr + (size_t)(b_avg == 1 ? t : t / b_avg) * b_ld, v >> 2);
            }
        }
    } else {
        // ------------------------------------------------------- epilogue --
        const int q = warp & 3;                      // TMEM lane quarter of this warp
        const int wp = warp >> 2;  // which of the quarter's two warps
        const int il = q * 32 + lane;                // this thread's input of the CTA's tile
        const uint32_t peer_inbox = kPair ? map_rank(sbase + kSmInbox, uint32_t(rank ^ 1)) : 0u,
                       peer_full = kPair ? map_rank(bar_in_full, uint32_t(rank ^ 1)) : 0u;
        int local = 0, votes = 0;
        bool ok = true;
        if (!kFresh && p.add_after) wait_for_launch_before();
        // the epilogue warps decide together whether to go on, so that none of them is
        // ever left waiting at a named barrier (two sets of votes in turn, so that a
        // vote is not overwritten before every warp has read it)
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
            ok = agree(mbar_wait(bar_acc_full(slot), uint32_t(local >> 1) & 1u, abort, p.status, 7, p.wait_limit) &&
                       (!kPair || cluster_wait(bar_in_free, uint32_t(local & 1) ^ 1u, abort, p.status, 11, p.wait_limit)));
            if (!ok) break;
            fence_after();
            const uint32_t taddr = tmem + uint32_t(slot * kSlotCols) + (uint32_t(q * 32) << 16);

            // operands into shared memory, 32 columns of the accumulator at a time: this
            // lane's row into `row`, or (transposed) its column of the rows there
            auto put_row = [&](uint8_t *row, uint32_t tcol) {
#pragma unroll
                for (int h = 0; h < 32; h += 16) {
                    uint32_t v[16];
                    tmem_ld16(taddr + tcol + h, v);
                    tmem_wait_ld();
#pragma unroll
                    for (int k = 0; k < 16; k += 4)
                        *reinterpret_cast<uint4 *>(row + (h + k) * 4) = make_uint4(v[k], v[k + 1], v[k + 2], v[k + 3]);
                }
            };
            // outputs (ic + k, j), k < 16, from x[k] = W[j][ic + k] and y[k] = W[ic + k][j]
            auto emit16 = [&](int ic, int j, const uint32_t (&xr)[16], const float (&yv)[16], bool full) {
                int2 v[16];
#pragma unroll
                for (int k = 0; k < 16; k += 2) {
                    // exact: the sum and difference are 2 Re and 2 Im times 2^-18, integers
                    // of at most 256 T <= 2^23 before the scale; adding 1.5 * 2^23 to Re, Im
                    // leaves them in the encoding's low bits
                    const float2 x = make_float2(__uint_as_float(xr[k]), __uint_as_float(xr[k + 1]));
                    const float2 yy = make_float2(yv[k], yv[k + 1]);
                    const float2 big = make_float2(12582912.0f, 12582912.0f);
                    const float2 half = make_float2(131072.0f, 131072.0f);
                    const float2 re = __ffma2_rn(__fadd2_rn(x, yy), half, big);
                    const float2 im = __ffma2_rn(__ffma2_rn(yy, make_float2(-1.0f, -1.0f), x), half, big);
                    v[k] = make_int2(__float_as_int(re.x) - 0x4B400000, __float_as_int(im.x) - 0x4B400000);
                    v[k + 1] = make_int2(__float_as_int(re.y) - 0x4B400000, __float_as_int(im.y) - 0x4B400000);
                }
                put_rows16<kFresh>(out_f, ic, j, n_in, lane, full, v);
            };

            if (kPair) {
                // the pair's operand of its half of the off-diagonal tile, into its inbox
                // (this CTA's inbox is armed for as many bytes), and the own operand
                if (warp == 0 && lane == 0) mbar_expect_tx(bar_in_full, kInboxBytes);
                if (rank == 1) {
                    if (q < 2) {                           // W[i][j], rows i < 64 of tile 1
#pragma unroll 1
                        for (int c0 = 16 * wp; c0 < kTile; c0 += 32) {
                            uint32_t v[16];
                            tmem_ld16(taddr + c0, v);
                            tmem_wait_ld();
#pragma unroll
                            for (int k = 0; k < 16; k += 4)
                                store_async4(peer_inbox + uint32_t(il * kHalfPitch + (c0 + k) * 4), v + k, peer_full);
                        }
                    } else {                               // W[i][j], rows i >= 64
#pragma unroll 1
                        for (int c0 = 32 * wp; c0 < kTile; c0 += 64)
                            put_row(smem + kSmOwn + (il - 64) * kHalfPitch + c0 * 4, c0);
                    }
                } else {                                   // W[j][i], transposed
#pragma unroll 1
                    for (int c0 = 16 * wp; c0 < 64; c0 += 32) {
                        uint32_t v[16];
                        tmem_ld16(taddr + kTile + 64 + c0, v);
                        tmem_wait_ld();
#pragma unroll
                        for (int k = 0; k < 16; ++k)
                            store_async(peer_inbox + uint32_t((c0 + k) * kHalfPitch + il * 4), v[k], peer_full);
                    }
#pragma unroll 1
                    for (int c0 = 16 * wp; c0 < 64; c0 += 32) {
                        uint32_t v[16];
                        tmem_ld16(taddr + kTile + c0, v);
                        tmem_wait_ld();
#pragma unroll
                        for (int k = 0; k < 16; ++k)
                            *reinterpret_cast<uint32_t *>(smem + kSmOwn + (c0 + k) * kHalfPitch + il * 4) = v[k];
                    }
                }
            }
            // the CTA's own diagonal tile
            const int t0 = it.base + rank * kTile;
            const uint32_t tdiag = uint32_t(rank * kTile);
#pragma unroll 1
            for (int c0 = 32 * wp; c0 < 32 * q + 32; c0 += 64)
                put_row(smem + kSmDiag + diag_base(q) + lane * diag_pitch(q) + c0 * 4, tdiag + c0);
            named_sync(2, kEpiWarps * 32);
            // columns j = il, rows from the start of the quarter on, 16 at a time
#pragma unroll 1
            for (int c0 = 32 * q + 16 * wp; c0 < kTile && t0 + c0 < n_in; c0 += 32) {
                uint32_t xr[16];
                float yv[16];
                const int rq = c0 >> 5, pitch = diag_pitch(rq);
                const uint8_t *yp = smem + kSmDiag + diag_base(rq) + (c0 & 31) * pitch + il * 4;
                tmem_ld16(taddr + tdiag + c0, xr);
#pragma unroll
                for (int k = 0; k < 16; ++k) yv[k] = *reinterpret_cast<const float *>(yp + k * pitch);
                tmem_wait_ld();
                emit16(t0 + c0, t0 + il, xr, yv, t0 + c0 + 15 < n_in && c0 >= 32 * q + 32);
            }
            // this accumulator can take the next item but one
            fence_before();
            __syncwarp();
            if (lane == 0) {
                if (kPair) remote_arrive(map_rank(bar_acc_empty(slot), 0));
                else mbar_arrive(bar_acc_empty(slot));
            }
            if (kPair) {
                // this CTA's half of the off-diagonal tile, both operands in shared memory:
                // 16 pieces of 16 rows and 32 columns, the more to a warp the fewer its
                // quarter has of the diagonal tile (4, 3, 2, 1)
                const int e0 = wp ? 6 + q * (q + 1) / 2 : q * (q - 1) / 2, e1 = e0 + q + wp;
                if (e0 < e1) {
                    ok = __all_sync(0xFFFFFFFFu,
                                    cluster_wait(bar_in_full, uint32_t(local & 1), abort, p.status, 12, p.wait_limit));
                    const uint8_t *const xb = smem + (rank ? kSmInbox : kSmOwn),
                                  *const yb = smem + (rank ? kSmOwn : kSmInbox);
                    const int i0 = it.base + kTile + 64 * rank;
#pragma unroll 1
                    for (int e = e0; ok && e < e1; ++e) {
                        const int c0 = 16 * (e >> 2), j = 32 * (e & 3) + lane;
                        if (i0 + c0 >= n_in) break;
                        uint32_t xr[16];
                        float yv[16];
                        const int o = c0 * kHalfPitch + j * 4;
#pragma unroll
                        for (int k = 0; k < 16; ++k) {
                            xr[k] = *reinterpret_cast<const uint32_t *>(xb + o + k * kHalfPitch);
                            yv[k] = *reinterpret_cast<const float *>(yb + o + k * kHalfPitch);
                        }
                        emit16(i0 + c0, it.base + j, xr, yv, i0 + c0 + 15 < n_in);
                    }
                }
                // every read of the inbox has returned (its values have been used)
                __syncwarp();
                if (ok && lane == 0) remote_arrive(map_rank(bar_in_free, uint32_t(rank ^ 1)));
            }
            // the next item's vote follows every read of the buffers; a failed wait shows in it
            if (!ok && item + item_step < p.n_items) agree(false);
        }
        // all rows of an item are sent, or none, so the pair knows what to expect
        if (kPair && threadIdx.x == 0) {
            sent[1] = local;
            store_peer(map_rank(sbase + kSmMisc + 96, uint32_t(rank ^ 1)), local);
        }
    }

    __syncwarp();
    fence_before();
    // no CTA leaves or frees TMEM while it, or its pair, may still be in use
    if (kPair) cluster_sync();
    else __syncthreads();
    fence_after();
    if (warp == kMmaWarp) {
        tmem_dealloc<kPair>(tmem, kTmemCols);
    }
    if (kPair && warp == kMmaWarp && lane == 0 && sent[0] > 0) {
        // after a timeout the rows of the pair's last item may still be on their way into the
        // inbox, which may not even be armed for them: they land before this CTA leaves
        if (sent[0] > sent[1]) mbar_expect_tx(bar_in_full, kInboxBytes);
        const uint32_t parity = uint32_t(sent[0] - 1) & 1u;
        const long long t0 = clock64();
        while (!mbar_try(bar_in_full, parity) && clock64() - t0 < p.drain_limit) {
        }
    }
    wait_for_launch_before();
}

// The parameters of a launch over every channel of `count` arrays.
inline cudaError_t make_params(const TcArray *arrays, int count, bool pair, DeviceStatus *status, const TcOptions &opt,
                               Params &prm)
{
    if (count < 1 || count > kTcMaxArrays) return cudaErrorInvalidValue;
    long long items = 0;
    for (int k = 0; k < count; ++k) {
        const TcArray &A = arrays[k];
        const int n_tiles = (A.n + kTile - 1) / kTile;
        ArrayParams &P = prm.a[k];
        P.volt = A.volt;
        P.ld = A.ld ? A.ld : A.n;
        P.f0 = A.f0;
        P.n_chan_all = A.n_chan_all ? A.n_chan_all : A.n_chan;
        P.row_t = (long long)P.ld * P.n_chan_all;
        P.acc = A.acc;
        P.n = A.n;
        P.n_chan = A.n_chan;
        P.first = pair ? 0 : (n_tiles - 1) * kTile;
        P.n_blocks = pair ? (n_tiles + (A.last_as_block ? 1 : 0)) / 2 : 1;
        P.nt = A.nt;
        P.n_stages = (A.nt + kTc - 1) / kTc;
        P.item_begin = int(items);
        P.beam = A.beam;
        P.beam_ld = P.n_chan_all;
        P.beam_avg = A.beam_avg > 0 ? A.beam_avg : 1;
        P.beam_t0 = A.beam_t0;
        items += (long long)A.n_chan * P.n_blocks;
    }
    if (items > 0x3FFFFFFF) return cudaErrorInvalidValue;
    prm.n_arrays = count;
    prm.n_items = int(items);
    prm.status = status;
    prm.wait_limit = opt.wait_limit > 0 ? opt.wait_limit : kDefaultWaitLimit;
    prm.drain_limit = kDefaultWaitLimit;
    prm.inject_stall = opt.inject_stall ? 1 : 0;
    prm.add_after = opt.add_after ? 1 : 0;
    prm.one = 1u;
    prm.minus_one = ~0u;
    prm.fifteen = 15u;
    prm.sixteen = 16u;
    return cudaSuccess;
}

// Index of a launch's kernel in a table [aligned][fresh][zero_invalid][beam]; fresh
// and zero_invalid are the same for all of its arrays.
inline int kernel_index(const Params &prm, bool fresh, bool zero_invalid)
{
    bool beam = false, aligned = true;
    for (int k = 0; k < prm.n_arrays; ++k) {
        beam = beam || prm.a[k].beam;
        aligned = aligned && prm.a[k].ld % 16 == 0 && (reinterpret_cast<uintptr_t>(prm.a[k].volt) & 15) == 0;
    }
    return (aligned ? 8 : 0) + (fresh ? 4 : 0) + (zero_invalid ? 2 : 0) + (beam ? 1 : 0);
}

// Streaming multiprocessors of `dev`; the first call per device lets `kernels` use
// their shared memory.
template <size_t kCount>
cudaError_t prepare_device(void (*const (&kernels)[kCount])(Params), int dev, std::mutex &mu, int (&sms)[64])
{
    if (dev < 0 || dev >= 64) return cudaErrorInvalidValue;
    std::lock_guard<std::mutex> lock(mu);
    if (sms[dev]) return cudaSuccess;
    for (auto fn : kernels) {
        const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
        if (e != cudaSuccess) return e;
    }
    int n = 0;
    const cudaError_t e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) sms[dev] = n;
    return e;
}

}  // namespace
}  // namespace corr
