// X-engine, tcgen05 FP8 tensor-core path: device support and the split of an
// array's triangle over its kernels.
//
// Tiles are 128 inputs.  A channel's triangle of tiles is taken as
//   - the 256-input blocks on the diagonal (tiles 2 b, 2 b + 1): CTA pairs,
//     xeng_pair.cu;
//   - the last tile alone, where the number of tiles is odd (an array of up to 128
//     inputs is nothing else): single CTAs, xeng_tile.cu, or a block whose second tile is
//     empty (one_launch);
//   - the tiles off those blocks, from 257 inputs on: CTA pairs, xeng_off.cu; in few
//     rounds both kinds go in one launch, xeng_both.cu.
// Each is one persistent launch over every channel of up to kTcMaxArrays arrays; a call of
// one array may cut its last round into slices of samples, which take launches of their own.
// Whether invalid samples are zeroed (CORR_ZERO_INVALID) and whether the launch stores
// or adds are properties of the kernel, so arrays that differ in them go to different
// launches.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <mutex>
#include <utility>

#include "internal.cuh"
#include "tc_common.cuh"

namespace corr {
namespace {

constexpr int kTile = 128;
constexpr int kBoxSamples = 64;               // samples of a tensor-map box (a stage)
constexpr size_t kSmemNeeded = 227 * 1024;    // the largest kernel's shared memory, at most

PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
std::once_flag g_encode_once;

PFN_cuTensorMapEncodeTiled_v12000 encoder()
{
    std::call_once(g_encode_once, [] {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
        else
            cudaGetLastError();
    });
    return g_encode;
}

// Tensor map of an array: boxes of one tile's inputs, one channel and kBoxSamples
// samples.  The extent along the inputs is n: a box reaching past it (a ragged last
// tile) reads zero bytes, i.e. samples 0 + 0i.
cudaError_t encode_map(const TcArray &A, CUtensorMap *map)
{
    const cuuint64_t ld = cuuint64_t(A.ld ? A.ld : A.n);
    const cuuint64_t dims[3] = {cuuint64_t(A.n), cuuint64_t(A.n_chan), cuuint64_t(A.nt)};
    const cuuint64_t strides[2] = {ld, ld * cuuint64_t(A.n_chan_all ? A.n_chan_all : A.n_chan)};
    const cuuint32_t box[3] = {cuuint32_t(kTile), 1u, cuuint32_t(kBoxSamples)};
    const cuuint32_t estr[3] = {1u, 1u, 1u};
    const CUresult cr = encoder()(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<uint8_t *>(A.volt), dims, strides,
                                  box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return cr == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// The last round of an array of one block (or one tile) per channel.  Its channels go round
// the pairs of CTAs (the CTAs), and the last round may be nearly empty: 128 channels on 76 pairs take
// as long as 152, 768 as long as 836.  The channels left for it can be split into up to four
// slices of samples, which add into a zeroed triangle; the slices' items share that round.
// Returns the slices (1: as it is) and the channels before them.  In units of 64 samples
// per channel, 0.42 us: a slice has 16 at least (about what its stores take), and splitting
// costs the zeroing, the adds and a launch, more where it is a second launch (about 14 and
// 26).  256 inputs x 5000 samples: 4 channels 39.7 -> 21.3 us, 80 channels 72 -> 60 us,
// 768 channels 359 -> 345 us (with the beam 401 -> 390); 40 channels x 20000 samples 125 ->
// 94 us; 16 x 2200 24.9 -> 20.9 us.  128 inputs x 5000 samples: 40 channels 37.5 -> 20.9 us,
// 160 channels 68 -> 52 us, 768 channels 188 -> 171 us.
constexpr int kSplitCost = 26, kSplitCostAlone = 14;

int last_round_slices(int n_chan, int nt, int workers, int *before)
{
    const int stages = (nt + 63) / 64, rest = n_chan % workers;
    *before = n_chan - rest;
    int best = 1, best_cost = stages - (*before ? kSplitCost : kSplitCostAlone);
    for (int s = 2; s <= kTcMaxArrays && stages >= 16 * s && rest > 0; ++s) {
        const int cost = (rest * s + workers - 1) / workers * ((stages + s - 1) / s);
        if (cost < best_cost) {
            best = s;
            best_cost = cost;
        }
    }
    return best;
}

__global__ void __launch_bounds__(256) zero_kernel(int2 *__restrict__ out, size_t n)
{
    let_next_launch_start();
    for (size_t e = blockIdx.x * size_t(256) + threadIdx.x; e < n; e += gridDim.x * size_t(256))
        out[e] = make_int2(0, 0);
    wait_for_launch_before();
}

// Channels f0 .. f0 + n_chan - 1 and samples t0 .. t0 + nt - 1 of a whole array.
TcArray part_of(const TcArray &A, int f0, int n_chan, int t0, int nt)
{
    TcArray p = A;
    const long long ld = A.ld ? A.ld : A.n;
    p.f0 = f0;
    p.n_chan = n_chan;
    p.n_chan_all = A.n_chan;
    p.nt = nt;
    p.volt = A.volt + f0 * ld + t0 * (ld * A.n_chan);
    p.acc = A.acc + size_t(f0) * size_t(n_pairs(A.n)) * 2;
    p.beam_t0 = A.beam_t0 + t0;
    if (A.beam) p.beam = A.beam + f0;
    return p;
}

// Those channels in `slices` slices of samples, of whole stages but for the last.
void slices_of(const TcArray &A, int f0, int n_chan, int slices, TcArray *part)
{
    const int step = ((A.nt + 63) / 64 + slices - 1) / slices * 64;
    for (int k = 0; k < slices; ++k)
        part[k] = part_of(A, f0, n_chan, k * step, k + 1 < slices ? step : A.nt - k * step);
}

// The pair kernel's (pair) or the tile kernel's launches of these arrays.  alone: they are one
// array, whose channels are all that the call computes.
cudaError_t launch_blocks(bool pair, const TcArray *arrays, int count, bool alone, bool fresh, bool zero_invalid,
                          int dev, DeviceStatus *status, const TcOptions &opt, cudaStream_t s, int *launches)
{
    const auto launch = pair ? launch_xeng_pair : launch_xeng_tile;
    int sms = 0;
    cudaError_t e = alone ? cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) : cudaSuccess;
    if (e != cudaSuccess) return e;
    const TcArray &A = arrays[0];
    int before = 0;
    const int slices = alone && sms > 1 ? last_round_slices(A.n_chan, A.nt, pair ? sms / 2 : sms, &before) : 1;
    if (slices == 1) {
        e = launch(arrays, count, fresh, zero_invalid, dev, status, opt, *launches > 0, s);
        *launches += e == cudaSuccess;
        return e;
    }
    TcArray part[kTcMaxArrays];
    const int rest = A.n_chan - before;
    const size_t triangle = size_t(n_pairs(A.n));
    slices_of(A, before, rest, slices, part);
    if (fresh) {
        e = launch_overlapping(zero_kernel, sms, 256, 0, *launches > 0, s, reinterpret_cast<int2 *>(part[0].acc),
                               triangle * rest);
        if (e != cudaSuccess) return e;
        ++*launches;
    }
    if (before) {
        const TcArray head = part_of(A, 0, before, 0, A.nt);
        e = launch(&head, 1, fresh, zero_invalid, dev, status, opt, *launches > 0, s);
        if (e != cudaSuccess) return e;
        ++*launches;
    }
    TcOptions last = opt;
    last.add_after = fresh;
    e = launch(part, slices, false, zero_invalid, dev, status, last, *launches > 0, s);
    *launches += e == cudaSuccess;
    return e;
}

int tiles_of(const TcArray &A) { return (A.n + kTile - 1) / kTile; }

int rounds_of(long long items, int workers) { return int((items + workers - 1) / workers); }

// Whether the blocks and the tiles off them go in one launch, with the pairs of CTAs divided
// between the two kinds of items, and how: up to four rounds, where it takes no round more
// than all items together.  A CTA then has its next item's samples and MMAs behind the stores
// of the one before, where a second launch's CTA starts from nothing: 512 inputs x 38 channels
// x 100, 300 and 1000 samples 20.8 -> 18.5, 24.6 -> 19.7 and 32.8 -> 25.5 us, 1024 x 8 x 1000
// 32.7 -> 24.8, 640 x 32 x 300 30.8 -> 24.3, 512 x 60 x 1000 (four rounds) 47.3 -> 41.0.  With
// more rounds long integrations lose (512 x 152 x 6000, eight rounds, 333 -> 346 us): power
// bounds them, and one kind's pairs end before the other's.  The last of an odd number of
// tiles goes with the blocks, as one whose second tile is empty, where that takes no round
// more (384 x 20 x 100, a launch less, 14.2 -> 12.4 us).  Where it does, long integrations of
// more than one round keep their launches, since the last tiles' then fills the pairs that the
// last round leaves idle (384 x 52 x 5000 82 us, 104 with both kinds in one launch, 384 x 52 x
// 1000 32.9 and 34.9); short ones gain all the same (384 x 76 x 100 26.7 -> 20.6 us, 640 x 36 x
// 300 34.6 -> 27.8), except three rounds with a small last tile (272 x 98 x 300 28.8, 30.8).
// In a call with others (alone = false) the last tiles go with theirs.
constexpr int kBothRounds = 4, kBothShortStages = 11;

struct OneLaunch {
    bool fits = false, last_as_block = false;
    int rounds = 0, block_pairs = 0, off_pairs = 0;
};

OneLaunch one_launch(const TcArray &A, int sms, bool alone)
{
    OneLaunch l;
    const int tiles = tiles_of(A), half = tiles / 2, pairs = sms / 2;
    if (pairs < 2) return l;
    const long long blocks = (long long)A.n_chan * half,
                    offs = (long long)A.n_chan * (tiles % 2 ? half * half : half * (half - 1));
    const int rounds = l.rounds = rounds_of(blocks + offs, pairs);
    auto divide = [&](long long with_blocks) {
        l.block_pairs = rounds_of(with_blocks, rounds);
        l.off_pairs = rounds_of(offs, rounds);
        return l.block_pairs + l.off_pairs <= pairs;
    };
    if (rounds > kBothRounds) return l;
    l.last_as_block = alone && tiles % 2 && divide(blocks + A.n_chan);
    if (l.last_as_block) {
        l.fits = true;
    } else if (divide(blocks)) {
        const bool few = rounds == 2 || (rounds == 3 && A.n - 2 * kTile * half > kTile / 2);
        l.fits = tiles % 2 == 0 || rounds == 1 || (few && A.nt <= 64 * kBothShortStages);
    }
    return l;
}

// The last round of a call of one array of more than 256 inputs.  Its items, the blocks and the
// tiles off them, go round the pairs of CTAs together, and the last round may be nearly empty
// (512 inputs x 20 channels: 80 items on 76 pairs).  Then the tiles off the blocks of as many
// channels as that round needs, and the last tiles of an odd number of them (or these alone),
// can go in slices of samples, which add into zeroed elements.  Costs are in units of 64
// samples per item as for last_round_slices; slices cost about 20, and one per MB that is
// zeroed and added to: 512 inputs x 20 channels x 5000 samples 78.2 -> 57.6 us, 1024 x 5 x
// 9500 131 -> 92, 384 x 38 x 5000 74.0 -> 59.7, 640 x 24 x 5000 111 -> 96.  More last tiles than
// SMs stay whole (384 x 160 x 7000 286 us, 295 in slices), and so does what would save less than
// a sixteenth: in many rounds the last one is cheap, since power bounds the others (512 x 300 x
// 9000 927 us, 939 in slices).
struct LargePlan {
    int off_chans = 0;        // last channels whose tiles off the blocks go in slices
    int off_slices = 1, tile_slices = 1;
};
constexpr int kLargeSplitCost = 20;

LargePlan plan_large(const TcArray &A, int sms)
{
    LargePlan plan;
    const int tiles = tiles_of(A), half = tiles / 2, pairs = sms / 2, stages = (A.nt + 63) / 64;
    if (pairs < 1) return plan;
    const int per_off = tiles % 2 ? half * half : half * (half - 1);
    const long long items = (long long)A.n_chan * (half + per_off);
    const int lone = tiles % 2 && !one_launch(A, sms, true).last_as_block ? A.n_chan : 0;  // last tiles alone
    const int full = int(items / pairs), left = int(items % pairs);
    const int whole = rounds_of(items, pairs), idle = left ? sms - 2 * left : 0;
    // whole items; the last tiles take the SMs that the last round leaves idle first
    long long best = (long long)whole * stages;
    if (lone > idle) best += (long long)rounds_of(lone - idle, sms) * stages;
    best -= best / 16;
    const long long last_rows = A.n - 2 * kTile * half;
    const double mb_tiles = tiles % 2 ? double(A.n_chan) * double(n_pairs(last_rows)) * 8e-6 : 0.0,
                 mb_item = 2.0 * kTile * kTile * 8e-6;
    auto take = [&](long long cost, int chans, int so, int st) {
        const double mb = (st > 1 ? mb_tiles * (st + 1) : 0.0) + double(chans) * per_off * mb_item * (so + 1);
        cost += kLargeSplitCost + (long long)mb;
        if (cost >= best) return;
        best = cost;
        plan.off_chans = chans;
        plan.off_slices = so;
        plan.tile_slices = st;
    };
    const int last_tiles = tiles % 2 ? A.n_chan : 0, chans = (left + per_off - 1) / per_off;
    for (int st = 1; st <= (last_tiles && last_tiles <= sms ? kTcMaxArrays : 1) && stages >= 16 * st; ++st) {
        const int tile_stages = (stages + st - 1) / st;
        // slices of the last tiles alone
        if (st > 1 && last_tiles > idle)
            take((long long)whole * stages + (long long)rounds_of((long long)(last_tiles - idle) * st, sms) * tile_stages,
                 0, 1, st);
        // slices of the last round's items and of the last tiles in a round of their own
        if (!full || !chans || chans >= A.n_chan || (last_tiles && st == 1)) continue;
        for (int so = 2; so <= kTcMaxOffParts && stages >= 16 * so; ++so) {
            const int off_stages = (stages + so - 1) / so,
                      longest = last_tiles && tile_stages > off_stages ? tile_stages : off_stages;
            take((long long)full * stages +
                     (long long)rounds_of(2LL * chans * per_off * so + (long long)last_tiles * st, sms) * longest,
                 chans, so, st);
        }
    }
    return plan;
}

// Zeroes what the slices of a plan add to: for the last `chans` channels the elements left of
// each row's own 256-input block, and (tiles) every channel's last tile.  A warp per row.
__global__ void __launch_bounds__(256) zero_large_kernel(int2 *__restrict__ out, int n, int n_chan, int chans, int tiles)
{
    let_next_launch_start();
    const int base = (n - 1) / kTile * kTile, rows = n - 2 * kTile, lane = threadIdx.x & 31;
    const long long triangle = n_pairs(n), first = chans ? 2 * kTile : base;
    for (long long r = blockIdx.x * 8LL + (threadIdx.x >> 5); r < (long long)n_chan * rows; r += gridDim.x * 8LL) {
        const int f = int(r / rows), i = 2 * kTile + int(r - (long long)f * rows);
        if (i < first) continue;
        const int own = i / (2 * kTile) * (2 * kTile);
        const bool last = tiles && i >= base;
        const int end = last ? i + 1 : f >= n_chan - chans ? own : 0;
        int2 *const row = out + f * triangle + n_pairs(i);
        for (int j = (f >= n_chan - chans ? 0 : own) + lane; j < end; j += 32) row[j] = make_int2(0, 0);
    }
    wait_for_launch_before();
}

// Both kinds of items of A in one launch; sets A.last_as_block.
cudaError_t launch_one(TcArray &A, const OneLaunch &one, bool fresh, bool zero_invalid, int dev, DeviceStatus *status,
                       const TcOptions &opt, cudaStream_t s, int *launches)
{
    A.last_as_block = one.last_as_block;
    CUtensorMap map;
    cudaError_t e = encode_map(A, &map);
    if (e == cudaSuccess)
        e = launch_xeng_both(A, map, one.block_pairs, one.off_pairs, fresh, zero_invalid, dev, status, opt,
                             *launches > 0, s);
    *launches += e == cudaSuccess;
    return e;
}

// The launches of a call of one array of more than 256 inputs.
cudaError_t launch_large(TcArray A, bool fresh, bool zero_invalid, int dev, DeviceStatus *status, const TcOptions &opt,
                         cudaStream_t s, int *launches)
{
    int sms = 0;
    cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const LargePlan plan = plan_large(A, sms);
    const bool odd = tiles_of(A) % 2, off_cut = plan.off_slices > 1, tile_cut = plan.tile_slices > 1;
    const OneLaunch one = one_launch(A, sms, true);
    if (one.fits && !off_cut && !tile_cut) {
        e = launch_one(A, one, fresh, zero_invalid, dev, status, opt, s, launches);
        if (e != cudaSuccess || !odd || one.last_as_block) return e;
        e = launch_xeng_tile(&A, 1, fresh, zero_invalid, dev, status, opt, true, s);
        *launches += e == cudaSuccess;
        return e;
    }
    TcOptions add = opt;
    add.add_after = fresh;
    if (fresh && (off_cut || tile_cut)) {
        e = launch_overlapping(zero_large_kernel, sms, 256, 0, *launches > 0, s, reinterpret_cast<int2 *>(A.acc), A.n,
                               A.n_chan, plan.off_chans, int(tile_cut));
        if (e != cudaSuccess) return e;
        ++*launches;
    }
    e = launch_xeng_pair(&A, 1, fresh, zero_invalid, dev, status, opt, *launches > 0, s);
    if (e != cudaSuccess) return e;
    ++*launches;
    TcArray part[kTcMaxOffParts];
    CUtensorMap maps[kTcMaxOffParts];
    const int before = A.n_chan - plan.off_chans;
    for (int cut = 0; cut <= int(off_cut); ++cut) {
        const int count = cut ? plan.off_slices : 1;
        if (cut) slices_of(A, before, plan.off_chans, count, part);
        else part[0] = part_of(A, 0, before, 0, A.nt);
        for (int k = 0; k < count; ++k) {
            e = encode_map(part[k], &maps[k]);
            if (e != cudaSuccess) return e;
        }
        e = launch_xeng_off(part, maps, count, fresh && !cut, zero_invalid, dev, status, cut ? add : opt, true, s);
        if (e != cudaSuccess) return e;
        ++*launches;
    }
    if (odd) {
        if (tile_cut) slices_of(A, 0, A.n_chan, plan.tile_slices, part);
        else part[0] = A;
        e = launch_xeng_tile(part, tile_cut ? plan.tile_slices : 1, fresh && !tile_cut, zero_invalid, dev, status,
                             tile_cut ? add : opt, true, s);
        *launches += e == cudaSuccess;
    }
    return e;
}

constexpr int kBothIdleStages = 16;

// The launches of the arrays of one mode, longest integrations first (a CTA's
// last items are then its shortest).
// The launches of one call write disjoint parts of the output and may overlap: each lets
// the next one's CTAs take the SMs as its own leave them (in place of an empty last round
// per launch: 384 inputs x 384 channels x 5000 samples 0.51 -> 0.45 ms, 1024 x 128 x 10000
// 1.81 -> 1.73 ms), and ends only when the one before has.
cudaError_t launch_group(const TcArray *arrays, int count, bool fresh, bool zero_invalid, int dev,
                         DeviceStatus *status, const TcOptions &opt, cudaStream_t s, int *launches)
{
    TcArray sorted[kTcMaxArrays], part[kTcMaxArrays];
    int m = 0;
    for (int k = 0; k < count; ++k)
        if (arrays[k].nt > 0 && arrays[k].fresh == fresh && arrays[k].zero_invalid == zero_invalid)
            sorted[m++] = arrays[k];
    for (int x = 1; x < m; ++x)
        for (int y = x; y > 0 && sorted[y].nt > sorted[y - 1].nt; --y) std::swap(sorted[y], sorted[y - 1]);
    cudaError_t e = cudaSuccess;
    if (count == 1 && m == 1 && sorted[0].n > 2 * kTile)
        return launch_large(sorted[0], fresh, zero_invalid, dev, status, opt, s, launches);
    // One array of more than 256 inputs beside some of up to 128 has both kinds of items in one
    // launch, as one alone would, and the tiles take the SMs that it leaves: 512 and 128 inputs x
    // 27 channels, two blocks of 168 samples 59.6 -> 54.0 us, 512 and 128 x 35, five of 349, 182
    // -> 148, 512 x 23 x 312 and 128 x 26 x 433 24.6 -> 20.5.  Beside arrays of 129..256 inputs,
    // whose blocks fill the pairs that the first launch leaves, it loses (512 and 192 x 26, five
    // of 252, 133 -> 154); so do longer integrations of more than one round that leave over a
    // quarter of the pairs idle (512 x 21 x 4509, 128 x 41 x 331 and 96 x 86 x 1971 74 -> 80).
    int n = 0, apart = -1;
    for (int k = 0; k < m; ++k)
        if (sorted[k].n > kTile) apart = ++n == 1 && sorted[k].n > 2 * kTile ? k : -1;
    if (apart >= 0) {
        int sms = 0;
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        const OneLaunch one = one_launch(sorted[apart], sms, false);
        const bool full = one.rounds == 1 || 4 * (one.block_pairs + one.off_pairs) >= 3 * (sms / 2);
        if (one.fits && (full || sorted[apart].nt <= 64 * kBothIdleStages)) {
            e = launch_one(sorted[apart], one, fresh, zero_invalid, dev, status, opt, s, launches);
            if (e != cudaSuccess) return e;
        } else {
            apart = -1;
        }
    }
    n = 0;
    for (int k = 0; k < m; ++k)
        if (sorted[k].n > kTile && k != apart) part[n++] = sorted[k];
    // other launches of the call would fill the last round
    const bool alone = count == 1 && n == 1 && part[0].n <= 2 * kTile;
    if (n) e = launch_blocks(true, part, n, alone, fresh, zero_invalid, dev, status, opt, s, launches);
    if (e != cudaSuccess) return e;
    n = 0;
    CUtensorMap maps[kTcMaxArrays];
    for (int k = 0; k < m; ++k) {
        if (sorted[k].n <= 2 * kTile || k == apart) continue;
        e = encode_map(sorted[k], &maps[n]);
        if (e != cudaSuccess) return e;
        part[n++] = sorted[k];
    }
    if (n) e = launch_xeng_off(part, maps, n, fresh, zero_invalid, dev, status, opt, *launches > 0, s);
    if (e != cudaSuccess) return e;
    *launches += n > 0;
    n = 0;
    for (int k = 0; k < m; ++k)
        if (tiles_of(sorted[k]) % 2) part[n++] = sorted[k];
    if (n) e = launch_blocks(false, part, n, count == 1 && part[0].n <= kTile, fresh, zero_invalid, dev, status, opt, s,
                             launches);
    return e;
}

}  // namespace

bool tc_supported(int n_inputs, int device)
{
    if (n_inputs < 1 || device < 0 || device >= 64) return false;
    static int cached[64] = {0};                 // 0 unknown, 1 yes, -1 no
    if (cached[device] == 0) {
        cudaDeviceProp prop;
        bool ok = cudaGetDeviceProperties(&prop, device) == cudaSuccess && prop.major == 10 &&
                  prop.minor == 3 && prop.sharedMemPerBlockOptin >= kSmemNeeded &&
                  encoder() != nullptr;
        cudaGetLastError();
        cached[device] = ok ? 1 : -1;
    }
    return cached[device] == 1;
}

bool tc_any_rows(int n) { return n <= 2 * kTile; }

cudaError_t launch_xeng_tc_batch(const TcArray *arrays, int count, DeviceStatus *status,
                                 const TcOptions &opt, cudaStream_t s, int *launches)
{
    *launches = 0;
    if (count < 0 || count > kTcMaxArrays) return cudaErrorInvalidValue;
    if (!encoder()) return cudaErrorNotSupported;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    for (int k = 0; k < count; ++k) {
        const TcArray &A = arrays[k];
        if (A.nt <= 0) continue;
        const int ld = A.ld ? A.ld : A.n;
        if (A.nt > kTcMaxSamples || A.n < 1 || ld < A.n || A.n_chan < 1 || !A.acc) return cudaErrorInvalidValue;
        if (!tc_any_rows(A.n) && (ld % 16 != 0 || (reinterpret_cast<uintptr_t>(A.volt) & 15) != 0))
            return cudaErrorInvalidValue;
    }
    for (int mode = 0; mode < 4; ++mode) {
        e = launch_group(arrays, count, (mode & 1) != 0, (mode & 2) != 0, dev, status, opt, s, launches);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace corr
