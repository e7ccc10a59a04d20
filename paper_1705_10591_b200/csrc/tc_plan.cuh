// Tensor-core convolution, host side: tile and stage sizes, and the planner that picks operand roles, addressing
// mode, item size, filter residency and the split of the contraction for a shape.  Included by general_tf32.cu only.
#pragma once
#include <cstdlib>

#include "common.cuh"

namespace conv2d_b200 {
namespace {

constexpr int kCB = 16;                     // channels per staged block (two UMMA K steps of 8)
constexpr int kChunks = kCB / 4;            // 16-byte channel chunks per block
constexpr int kProducerWarps = 8;
constexpr int kProducers = kProducerWarps * 32;
static_assert(kProducers == 256, "the producer group arithmetic assumes 256 producer threads");
constexpr int kEpilogueWarps = 4;
// Warp roles by warp index.  An SM has four warp schedulers and warp w is served by scheduler w % 4.  The
// warp that issues the MMAs (warp 1) must never wait for an issue slot behind arithmetic-heavy
// warps -- measured: sharing its scheduler with two producer warps stretched each MMA issue from ~64 to
// 120-180 cycles -- so scheduler 1 hosts only that warp, one epilogue warp and two warps that only wait.
//   warp 0           filter copies (one thread)
//   warp 1           MMA issue (all lanes run the loop, an elected one issues), owner of the tensor-memory allocation
//   warps 4-7        epilogue, tensor-memory lane quarter = warp % 4
//   warps 2,3,8,10,11,12,14,15   activation producers (schedulers 0, 2, 3)
//   warps 9, 13      no work until the block's last item
//   warps 8-15       help to drain the block's last item once their own work is done (quarter = warp % 4)
constexpr int kThreads = 512;
__device__ __forceinline__ int producer_index(int warp)     // 0..7 for producer warps, -1 otherwise
{
    switch (warp) {
        case 2: return 0; case 3: return 1; case 8: return 2; case 10: return 3;
        case 11: return 4; case 12: return 5; case 14: return 6; case 15: return 7;
        default: return -1;
    }
}
constexpr int kMaxBStages = 16;
constexpr int kMaxAStages = 4;
constexpr int kUnitsPerThread = 3;          // (pixel, channel block) units a producer thread keeps in flight per pass
constexpr size_t kSmemLimit = 227 * 1024;
constexpr int kMaxTaps = 256;                // taps left as descriptor shifts (after folding)
constexpr size_t kBookBytes = 512 + kMaxTaps * 4;    // barriers, tensor-memory slot, flags, up to 64 bytes before a bank of stacked taps + the table of tap shifts
constexpr int kXposePitch = 36;             // floats per row of the epilogue's transposition tile (16-byte aligned, conflict-free)
constexpr size_t kXposeBytes = (size_t)kEpilogueWarps * 32 * kXposePitch * 4;
constexpr int kStackPitch = 68;             // ... of the tile of stacked taps: 16 maps x two 32-pixel blocks (conflict-free likewise)
static_assert(16 * kStackPitch <= 32 * kXposePitch, "it lies in the same place");
constexpr int kXchgBlockFloats = 32 * 32;   // exchange area of a two-block cluster: one 32-filter x 32-pixel block of partial sums
// bytes of that area for `slots` 32-pixel blocks per lane quarter: blocks, then one barrier per (quarter, slot)
constexpr size_t xchg_area_bytes(int slots) { return (size_t)kEpilogueWarps * slots * (kXchgBlockFloats * 4 + 8); }

struct Plan {
    int n_tile;       // filters per work item: 64 or 128 rows of the M operand
    int n_blocks;     // work-item columns over the filters
    int tile_px;      // pixels per work item: any multiple of 32 up to 512 (of 16 where items end with their image)
    int px_groups;    // MMAs per K step (each covers n_mma = tile_px / px_groups pixels)
    int nbuf;         // accumulator sets in tensor memory (2: write-back overlaps the next item)
    int npix;         // staged pixel rows per channel chunk
    int cblks;        // channel blocks (of the folded channels, see fold_r/fold_s)
    int fold_r, fold_s;  // taps folded into the channel dimension: 1 or R rows, 1 or S columns
    int patch_w, patch_tw, patch_rows, patch_cols;   // patch addressing (patch_w = 0: flat pixel run), see ItemGeom
    int crop, crop_items;   // flat addressing: 1 = items end with their image, crop_items of them each
    int wants_crop;         // 1: the rule would choose such items, but this plan was made without them
    int taps;
    int a_stages;
    int b_stages;
    int tps;          // taps per filter stage
    int cbg;          // channel blocks per activation stage
    int resident;     // 1: the whole filter block stays in shared memory for the life of the thread block
    int pair_taps;    // 1: at most 64 filters, horizontally adjacent taps stacked in one M = 128 operand (see make_plan)
    int pair_compact; // 1 (with pair_taps): a lone last tap of a filter row is a 64-row slice issued as M = 64 (resident bank only, put together from the plain one)
    size_t cb_bytes;  // bytes of one channel block of the re-ordered bank (all taps of one filter block)
    int s_slots;      // shift-table entries per filter row: S, or ceil(S / 2) with stacked taps
    int ovl;          // pixels by which consecutive flat items overlap (4 with stacked taps, else 0)
    int ksplit;       // 2: the channel blocks of a tile are shared by two work items that add into y
    int cluster;      // 1 (with ksplit = 2): the two items run as a two-block cluster and exchange partial sums on chip
    int xchg_slots;   // ... 32-pixel blocks each of them receives
    int tmem_cols;    // power of two >= 32
    int supertiles;   // work-item rows over the flat pixel sequence
    int grid;
    size_t smem_bytes;
    int virt;         // 1: virtual images (zero padding, strides)
    int virt_h, virt_w, off_h, off_w, shift0, ext, phases, phase_cols, mixed, quad2;     // see KernelArgs
    long long pairs;  // (tap, channel block) pairs of a filter block
    size_t bank_bytes;   // re-ordered filters of one filter block
    double staged_ratio; // staged pixels per output of a 448-pixel item
    double cost;      // (of the streamed plans: estimate the item size was chosen by, in cycles)
    double makespan;  // MMA work of the busiest block, in item pixels x taps x channel blocks (to compare patch widths)
    bool ok;
};

// Distance between the 4-channel chunks of a staged channel block, in 16-byte units: the pixel count plus one, so
// that it is odd.  A producer lane writes four adjacent pixels (64 bytes) per chunk; with lanes 64 bytes apart a
// 128-bit store instruction would hit only two of the eight 16-byte bank groups (4-way conflict, ~1 M conflict
// cycles per launch in the profiles).  With an odd chunk stride, lanes that would collide write different chunks
// at the same time (each lane rotates its chunk order), and the eight lanes of a store phase cover all banks.
inline int chunk_stride(int npix) { return npix + 1; }

// Shared memory of the re-ordering kernel that works in tiles (8 filters x one channel block x `taps`), and its limit.
constexpr size_t kRepackTileLimit = 48 * 1024;
inline size_t repack_tile_bytes(int taps) { return (size_t)8 * kCB * 4 * taps; }

// b_stages counts filter stages of `tps` taps each; an activation stage holds `cbg` channel blocks.
size_t smem_need(int a_stages, int npix, int n_tile, int b_stages, int tps, int cbg)
{
    return (size_t)a_stages * cbg * kCB * chunk_stride(npix) * 4 + (size_t)b_stages * tps * kCB * n_tile * 4 + kBookBytes;
}

// b16: the operands are 16-bit floats, bf16 or fp16 (16-byte unit = 8 channels, 32 channels per staged block, K = 16 per MMA); the
// byte layout of every stage is the same as for TF32 (16 channels of 4 bytes).
Plan plan_with_patch_width(const Shape& shape, bool b16, int want_patch_w, bool allow_compact = true, bool virt = false, bool narrow = false,
                           bool allow_crop = true)
{
    Plan p{};
    p.ok = false;
    Shape sh = shape;                                      // (virtual images: the extents of the virtual plane)
    const int st = sh.stride;
    if (st > 1 && !virt) return p;
    p.phases = p.phase_cols = 1;
    if (virt) {
        if (b16) return p;
        p.virt = 1;
        p.off_h = sh.pad_h;
        if (st == 1) {
            // zeros to the left of a row serve the row before as well; a multiple of four keeps quads of the image aligned
            p.off_w = sh.W % 4 == 0 ? (sh.pad_w + 3) / 4 * 4 : sh.pad_w;
            p.shift0 = p.off_w - sh.pad_w;
            p.virt_h = sh.H + sh.pad_h > sh.P ? sh.H + sh.pad_h : sh.P;
            p.virt_w = sh.W + p.off_w > sh.Q ? sh.W + p.off_w : sh.Q;
        } else {
            // Stride 2 with whole quads of columns: the zeros in front of a row are a multiple of four columns, so that four
            // adjacent pixels of the image are two virtual pixels of both phases of a row.  The taps then start `ext`
            // columns into their phases, and `shift0` virtual pixels further on.
            // Channel blocks: all phases of a 16-channel block after one another, each with its own taps -- or, with few
            // channels, the phases of every channel as staged channels with all ceil(R/st) x ceil(S/st) taps (zero filters
            // where a phase has none), where that takes fewer MMAs: 3 channels, 7 x 7, stride 2: 16 pairs instead of 49.
            // The taps of such staged channels lie by `ext`, which therefore follows from the padding whether the rows are whole quads or not:
            // filters packed for one width serve the others.
            const bool two = st == 2 && sh.S >= 2 && sh.R >= 2;
            const int shifted = two ? sh.pad_w % 2 : 0;
            const long long apart = (long long)((sh.C + kCB - 1) / kCB) * sh.R * sh.S;
            const long long together = ((long long)sh.C * st * st + kCB - 1) / kCB * ((sh.R + st - 1) / st) * ((sh.S + shifted + st - 1) / st);
            p.mixed = together < apart ? 1 : 0;
            p.quad2 = two && sh.W % 4 == 0 && env_int("CONV2D_B200_TF32_QUAD", 1) != 0 ? 1 : 0;
            p.off_w = p.quad2 ? (sh.pad_w + 3) / 4 * 4 : p.mixed ? sh.pad_w + shifted : sh.pad_w;
            p.ext = (p.off_w - sh.pad_w) % st;
            p.shift0 = (p.off_w - sh.pad_w) / st;
            p.virt_h = sh.P + (sh.R + st - 1) / st - 1;
            p.virt_w = sh.Q + p.shift0 + (sh.S + p.ext + st - 1) / st - 1;
            p.phase_cols = st < sh.S ? st : sh.S;
            p.phases = p.phase_cols * (st < sh.R ? st : sh.R);
        }
        // outputs that can be stored as quads or pairs start on such a column of the accumulators, too
        const int unit = (st == 1 && sh.W % 4 == 0) || p.quad2 || (sh.Q % 4 == 0 && (long long)sh.P * sh.Q % 4 == 0) ? 4 : (sh.Q % 2 == 0 && (long long)sh.P * sh.Q % 2 == 0 ? 2 : 1);
        const int cols = narrow && unit == 4 ? 2 : unit;
        p.virt_w = (p.virt_w + cols - 1) / cols * cols;
        if ((long long)p.virt_h * p.virt_w >= 1LL << 30) return p;
        sh.H = p.virt_h;
        sh.W = p.virt_w;
        sh.pad_h = sh.pad_w = 0;
        if ((long long)sh.R * sh.S + 1 + 2 * p.phases > kMaxTaps) return p;      // (tap shifts and the table of phases)
    }
    const long long total_pix = (long long)sh.N * sh.H * sh.W;
    if (total_pix >= (1LL << 31) - (1LL << 20)) return p;     // flat pixel indices stay within int32
    const int kp16 = (sh.K + 15) / 16 * 16;
    // Operand roles.  One tcgen05.mma takes the pipe 64 cycles for any N up to 128 and N / 2 beyond, and the warp that issues it ~90
    // at least, so an instruction should have N = 192 to 256.  For any
    // filter count that is possible with the pixels as the N operand: M = a block of 128 filters (zero
    // padded), N = 256 pixels, accumulator lanes = filters.  It also halves the filter bytes an item streams
    // per pixel compared with 128 pixels x 256 filters.
    // Up to 64 filters use M = 64 (one tcgen05.mma then covers 64 filters x 256 pixels; its accumulator
    // occupies lanes 0-15 of each 32-lane quarter -- established with a probe).
    p.n_tile = kp16 <= 64 ? 64 : 128;                      // filters per block = rows of the M operand
    p.n_blocks = (kp16 + p.n_tile - 1) / p.n_tile;
    const int cbc = b16 ? 2 * kCB : kCB;                 // channels per staged block
    // Few input channels (first layers, the bridge between the one-channel and the many-channel case) would
    // leave most of a staged channel block as zero padding.  Then taps are folded into the channel dimension:
    // "channel" (c, r, s) of pixel j is x[c] at pixel j + r*W + s, so the contraction runs over C*fold_r*fold_s
    // channels and only the remaining R/fold_r x S/fold_s taps are descriptor shifts.  The fold with the
    // fewest MMAs (remaining taps x channel blocks) wins; ties keep more taps as shifts (fewer loads).
    // Every folded tap multiplies the producers' loads, so by default only 1-3 channels are folded (measured:
    // 3 channels 7 x 7 on 224 x 224: 0.91 ms folded, 1.06 ms not; 1 channel 5 x 5: 0.32 vs 0.40 ms; but
    // 8 channels 3 x 3 on 112 x 112: 0.175 vs 0.093 ms).  CONV2D_B200_TF32_FOLD = 2 folds whenever C < 16.
    p.fold_r = p.fold_s = 1;
    const bool padded = sh.pad_h != 0 || sh.pad_w != 0;      // needs patch addressing: no folding
    const int fold_mode = padded || virt ? 0 : env_int("CONV2D_B200_TF32_FOLD", 1);
    if (sh.C < cbc && (fold_mode == 2 || (fold_mode == 1 && sh.C <= 3))) {
        long long best = (long long)sh.R * sh.S * ((sh.C + cbc - 1) / cbc);
        const int cand[3][2] = {{1, sh.S}, {sh.R, 1}, {sh.R, sh.S}};
        for (const auto& f : cand) {
            const long long ceff = (long long)sh.C * f[0] * f[1];
            if (ceff > 4096) continue;
            const long long mmas = (long long)(sh.R / f[0]) * (sh.S / f[1]) * ((ceff + cbc - 1) / cbc);
            if (mmas < best) { best = mmas; p.fold_r = f[0]; p.fold_s = f[1]; }
        }
    }
    const int c_eff = sh.C * p.fold_r * p.fold_s;
    const int r_eff = st > 1 ? (sh.R + st - 1) / st : sh.R / p.fold_r, s_eff = st > 1 ? (sh.S + p.ext + st - 1) / st : sh.S / p.fold_s;
    p.cblks = (c_eff + cbc - 1) / cbc;
    if (st > 1) {
        if (p.mixed) {
            p.phases = p.phase_cols = 1;
            p.cblks = (int)(((long long)sh.C * st * st + cbc - 1) / cbc);
        } else {
            // (with quad2 the two phases of a row are one block of 32 staged channels with the taps of both)
            if (p.quad2) { p.phases /= p.phase_cols; p.phase_cols = 1; }
            p.cblks *= p.phases;
            // (only the tiled re-ordering kernel groups the taps by phase; refused here and not where the filters are
            // re-ordered, so that a call that finds them packed takes the same path as the call that packed them)
            if (p.phases > 1 && repack_tile_bytes(sh.R * sh.S) > kRepackTileLimit) return p;
        }
    }
    const int stage_blocks = p.quad2 && !p.mixed ? 2 : 1;    // 16-channel blocks of a channel block
    // Stacked taps.  With at most 64 filters an M = 64 instruction runs the tensor pipe at half its rate.  Instead
    // half of the rows of an M = 128 operand hold the filters' tap (r, s) and the other half their tap (r, s + 1),
    // both multiplied with the pixels shifted for (r, s): the accumulator row of tap (r, s + 1), column j + 1, then
    // holds what that tap contributes to output j, and the epilogue adds the two rows of a map one column apart
    // (rows are ordered so that both lie in the lane quarter of one epilogue warp).  A row of
    // S taps takes ceil(S / 2) instructions instead of S (an odd last tap has zeros in the upper half).  In the
    // flat pixel run the last column of an item has no right neighbour, so consecutive items overlap by 4 pixels.
    // It pays when the MMAs dominate an item: the stacked operand doubles the filter bytes per instruction (a bank
    // that was resident in shared memory may have to be streamed).  Hence from 48 (tap, channel block) pairs on.  Stacked against
    // not, means of 420 random layers: fp32 with quads 0.91 at 48 to 59 pairs, 0.76 at 60 to 71, 0.85 from 96 on, single
    // pixels 0.86 to 1.06; below 48 fp32 0.97 to 0.99 (0.83 to 1.68) and 0.98 to 1.06.  (16-bit operands gain below 48, too: 0.90 to 0.93 from 24 on.)
    // CONV2D_B200_TF32_PAIR_TAPS = 0 / 2: never / whenever possible.
    const int pair_mode = env_int("CONV2D_B200_TF32_PAIR_TAPS", 1);
    p.pair_taps = (st == 1 && kp16 <= 64 && p.fold_r * p.fold_s == 1 && s_eff >= 2 && pair_mode != 0 &&
                   (pair_mode == 2 || (long long)r_eff * s_eff * p.cblks >= 48)) ? 1 : 0;
    // Compact stacking for banks that can stay in shared memory: pairs of taps as 128-row slices, the lone last tap of
    // an odd filter row as a 64-row slice that an M = 64 instruction adds onto the same accumulator lanes.  The bank
    // is then as large as the unstacked one, so a short contraction keeps its resident filters and still issues two
    // instructions per three taps instead of three at half rate (64 filters of 64 x 3 x 3 on 56 x 56 images).
    // 32 x 64 x 56 x 56, 64 of 3 x 3, padding 1: 29.8 -> 27.7 us (wholly stacked and streamed 28.7).  16-bit operands have half
    // as many MMAs and are bound by what shared memory moves: off (64 x 128 x 32 x 32, 64 of 3 x 3 in bf16: 22.8 us, 24.8 stacked).
    // The MMAs have to be what sets the pace: 36 pairs of tap and channel block (with fewer the write-back: 64 x 16 x 90 x 122, 19 of
    // 3 x 3 57.6 -> 67.7 us; 5 x 48 x 74 x 74, 48 of 3 x 3 12.5 -> 13.9), of which at most 38 fit (4 KB each): 3 x 3 on 49 to 64
    // channels, 6 x 6 on up to 16, 4 x 3 on 33 to 48 and the like, whose pixels are loaded as quads (else the producers: 7 x 64 x 95 x 95, 48 of 3 x 3, padding 1 26.5 -> 30.8).
    // CONV2D_B200_TF32_PAIR_COMPACT = 0 / 1: never / whenever possible.
    const int compact_mode = env_int("CONV2D_B200_TF32_PAIR_COMPACT", b16 ? 0 : 2);
    p.pair_compact = 0;
    const size_t compact_cb_bytes = (size_t)r_eff * ((s_eff / 2) * 128 + (s_eff & 1) * 64) * kCB * 4;
    if (allow_compact && !p.pair_taps && st == 1 && kp16 <= 64 && p.fold_r * p.fold_s == 1 && s_eff >= 2 && pair_mode != 0 &&
        !padded && (size_t)((c_eff + cbc - 1) / cbc) * compact_cb_bytes <= 152 * 1024 && compact_mode != 0 &&
        (compact_mode == 1 || ((long long)r_eff * s_eff * p.cblks >= 36 && (virt ? shape.W : sh.H * sh.W) % 4 == 0))) {
        p.pair_taps = 1;
        p.pair_compact = 1;
    }
    if (p.pair_taps) p.n_tile = 128;
    p.s_slots = p.pair_taps ? (s_eff + 1) / 2 : s_eff;
    p.taps = stage_blocks == 2 ? r_eff * sh.S : r_eff * p.s_slots;          // (with phases: of the phase that has most)
    if (p.taps > kMaxTaps) return p;
    const size_t extra = kXposeBytes;                     // epilogue transposition tile
    // Addressing mode.  In the flat pixel run the staged halo is (R-1) whole image rows; once that exceeds a
    // 256-pixel item the item is cut as a rectangle of the image instead (patch_w columns wide, of which the
    // first patch_tw produce outputs), whose halo is (R-1) patch rows.  The patch width with the least staged
    // pixels per output wins.
    p.patch_w = p.patch_tw = p.patch_rows = p.patch_cols = 0;
    const long long flat_halo = (long long)(r_eff - 1) * sh.W + (s_eff - 1) + p.shift0;
    const int patch_mode = virt ? 0 : padded ? 2 : env_int("CONV2D_B200_TF32_PATCH", 1);       // 0 never, 1 when the flat halo is large, 2 always
    if (p.fold_r * p.fold_s == 1 && patch_mode != 0) {
        double best_ratio = 0;
        const int forced_wp = want_patch_w ? want_patch_w : env_int("CONV2D_B200_TF32_PATCH_W", 0);
        for (int wp = 32; wp <= 128; wp *= 2) {
            const int tw = (wp - (s_eff - 1)) / 4 * 4;
            if (tw < 4 || (forced_wp && wp != forced_wp)) continue;
            const int th = 448 / wp > 0 ? 448 / wp : 1;                       // rows of a typical item
            const long long rows_p = (sh.P + th - 1) / th, cols_p = (sh.Q + tw - 1) / tw;
            const double ratio = (double)(rows_p * (th + r_eff - 1)) * wp * cols_p / ((double)sh.P * sh.Q);
            if (p.patch_w == 0 || ratio < best_ratio) { best_ratio = ratio; p.patch_w = wp; p.patch_tw = tw; }
        }
        // staged pixels per output of the flat run, for a 448-pixel item.  Patches also cost extra work items at
        // the ragged right edge and a narrower store run, so they must win clearly (measured: 3 x 3 on 224 x 224,
        // ratio 2.0 flat vs 1.3 in patches, is 10 % faster flat; 3 x 3 on 512 x 512, 3.3 vs 1.3, 20 % faster in patches;
        // 7 x 7 on 224 x 224, 4.2 vs 2.2, 20 % faster in patches).
        const double flat_ratio = (448.0 + flat_halo) / 448.0 * ((double)sh.H * sh.W) / ((double)sh.P * sh.Q);
        if (patch_mode == 1 && !(flat_ratio > 1.75 * best_ratio)) p.patch_w = p.patch_tw = 0;
        p.staged_ratio = best_ratio;
        if (p.patch_w) p.patch_cols = (sh.Q + p.patch_tw - 1) / p.patch_tw;
    }
    if (virt) p.staged_ratio = (448.0 + flat_halo) / 448.0 * ((double)sh.H * sh.W) / ((double)sh.P * sh.Q);
    if (padded && !p.patch_w) return p;
    if (p.pair_compact && p.patch_w && compact_mode != 1) return plan_with_patch_width(shape, b16, want_patch_w, false, virt, narrow, allow_crop);
    p.ovl = (p.pair_taps && !p.patch_w) ? 4 : 0;
    const long long halo = p.patch_w ? (long long)(r_eff - 1) * p.patch_w + (s_eff - 1) : flat_halo;
    // work items along the pixels for an item of px pixels (0: px is not possible in this mode)
    auto pixel_items = [&](int px) -> long long {
        if (!p.patch_w) return px > p.ovl ? (total_pix + (px - p.ovl) - 1) / (px - p.ovl) : 0;
        if (px % p.patch_w) return 0;
        const int th = px / p.patch_w;
        return (long long)sh.N * ((sh.P + th - 1) / th) * p.patch_cols;
    };
    const int chunk = kCB * p.n_tile * 4;
    const int sms = sm_count();

    p.cb_bytes = p.pair_compact ? compact_cb_bytes : (p.phases > 1 ? (size_t)sh.R * sh.S : (size_t)p.taps) * chunk;
    p.pairs = p.phases > 1 ? (long long)(p.cblks / p.phases) * sh.R * sh.S : (long long)p.taps * p.cblks;
    const size_t wbytes = (size_t)(p.cblks / p.phases) * p.cb_bytes;   // re-ordered filters of one filter block
    p.bank_bytes = wbytes;
    auto npix_of = [&](int tile_px) { return (int)(((long long)tile_px + halo + 7) / 8 * 8); };

    // Light problems (1x1-like: few taps x channel blocks) with a small filter bank keep it resident in
    // shared memory: nothing is streamed, items are small (finest balance over the SMs, two accumulator
    // sets), and the rest of shared memory becomes a deep activation ring whose stages carry several
    // channel blocks (these items are bound by memory latency: one producer pass should have 32-48 loads
    // per thread in flight).  Any other bank that fits next to a two-stage activation ring is kept resident too
    // (64 filters of 64 x 3 x 3: 39 us resident vs 43 us streamed).
    p.resident = 0;
    const int resident_mode = env_int("CONV2D_B200_TF32_RESIDENT", 2);      // 0 never, 1 light problems only, 2 whenever it fits
    if (resident_mode != 0 && p.n_blocks == 1 && wbytes <= 152 * 1024 &&
        (p.pairs <= 16 || resident_mode == 2)) {
        int res_px = 256;
        if (!p.patch_w) {
            // When all pixels fit in one round of items of at most 512 pixels, one item per block is the better
            // cut (64 x 32 x 32 pixels with 1 x 1 filters: 448 pixels per item 19.9 us, 256 per item 22.1 us).
            // (compact stacking issues one MMA per K step: at most 256 pixels per item)
            const long long one_round = ((total_pix + sms - 1) / sms + p.ovl + 31) / 32 * 32;
            if (one_round >= 64 && one_round <= (p.pair_compact ? 256 : 512)) res_px = (int)one_round;
        }
        {
            const int want = env_int("CONV2D_B200_TF32_TILE_PX", 0);
            if (want >= 64 && want <= (p.pair_compact ? 256 : 512) && want % 32 == 0 && pixel_items(want) > 0) res_px = want;
        }
        const int npix = npix_of(res_px);
        if (res_px <= 512 && npix <= 16000 && wbytes + extra + (size_t)2 * stage_blocks * kCB * chunk_stride(npix) * 4 + kBookBytes <= kSmemLimit) {
            p.resident = 1;
            p.tile_px = res_px;
            p.npix = npix;
            p.cbg = 1;
            p.a_stages = 2;
            p.b_stages = 1;
            p.tps = p.taps;
            auto need = [&](int a_stages, int cbg) { return wbytes + extra + (size_t)a_stages * cbg * stage_blocks * kCB * chunk_stride(npix) * 4 + kBookBytes; };
            while (p.cbg * 2 <= p.cblks && npix * p.cbg * stage_blocks * 2 <= kProducers * kUnitsPerThread &&
                   need(p.a_stages, p.cbg * 2) <= kSmemLimit) p.cbg *= 2;
            while (p.a_stages < kMaxAStages && need(p.a_stages + 1, p.cbg) <= kSmemLimit) ++p.a_stages;
            p.smem_bytes = need(p.a_stages, p.cbg);
        }
    }

    if (p.pair_compact && !p.resident) return plan_with_patch_width(shape, b16, want_patch_w, false, virt, narrow, allow_crop);    // compact stacking needs the resident bank
    if (!p.resident) {
        // Streamed filters.  Measured: all SMs together draw filter stages from L2 at no more than
        // ~5-6 TB/s, i.e. a 8 KB stage costs ~120 cycles on top of the MMAs that consume it unless it is
        // reused by more pixels.  Larger items amortise that; smaller ones leave room for a
        // second accumulator set (hidden write-back) and balance better.  Cost in cycles: rounds x one item's
        // MMA and stage time + exposed write-back.
        const size_t kLimit = kSmemLimit - extra;
        const double stage_cycles = chunk / 66.0;           // one (tap, channel block) of filters through L2
        const int forced_px = env_int("CONV2D_B200_TF32_TILE_PX", 0);
        const bool ksplit_allowed = env_int("CONV2D_B200_TF32_KSPLIT", 1) != 0;
        int best_px = 0;
        double best_cost = 0, flat_bound = 0;          // (flat_...: of the best items of the whole run)
        bool flat_adds = false;
        // Any multiple of 32 pixels per item: the item size follows from the pixel count and the 148 SMs
        // (64 x 32 x 32 pixels: 448 per item = 147 items in one round, where 512 would occupy 128 SMs).
        // One or two MMAs of equal width cover the item per K step; an MMA narrower than 128 pixels is
        // bound by its ~64-cycle issue cost.
        long long best_items = 0;
        // (CONV2D_B200_TF32_CROP = 0: never, 2: wherever they fit)
        const int crop_mode = p.patch_w || p.fold_r * p.fold_s != 1 || sh.C < kCB || forced_px ? 0 : env_int("CONV2D_B200_TF32_CROP", 1);
        auto consider = [&](int px, int groups, long long px_items, long long npix, int crop, int crop_items) {
            if (npix > 16000 || smem_need(2, (int)npix, p.n_tile, 2, 1, stage_blocks) > kLimit || px_items <= 0) return;
            const long long items = px_items * p.n_blocks;
            const long long rounds = (items + sms - 1) / sms;
            const int nbuf = 2 * px <= 512 ? 2 : 1;
            const double mma_step = groups * ((px / groups) / 2.0 > 64.0 ? (px / groups) / 2.0 : 64.0);
            const double tile_time = (double)p.pairs * (2 * mma_step + stage_cycles);
            const double writeback = (nbuf == 1 ? 1.0 : 0.15) * (px / 128.0) * (3000.0 * p.n_tile / 128.0);
            double cost = rounds * (tile_time + 0.5 * writeback);
            // With one accumulator set the MMAs of an item wait for the whole write-back of the item before it
            // (four warps, measured ~2000 cycles per 32-pixel block of 128 maps, ~1200 of 64); from the third round
            // of items on that outweighs the wider MMAs (64 x 64 x 56 x 56 -> 128 maps, 3 x 3: 480-pixel items
            // 69.1 us, 256-pixel items with two accumulator sets 64.6 us).
            if (nbuf == 1 && rounds >= 3)
                cost += (double)(rounds - 2) * 0.75 * (px / 32.0) * (p.n_tile >= 128 ? 2000.0 : 1200.0);
            // (items that leave half of the SMs idle are split in two along the channels further down)
            const bool split = items * 2 <= sms && p.cblks >= 2 && ksplit_allowed;
            if (split) cost = 0.5 * tile_time + writeback;
            // Items of an image against those of the whole run: also counted are the zero-fill and the adds of a contraction that is
            // split without a cluster (9000 cycles), and the producers (6 cycles per staged pixel and channel block) must
            // not become what sets the pace (128 x 256 x 11 x 139, 6 of 3 x 3: 441 items of 448 pixels 140 us, 640 of 256 175 us).
            const bool adds = split && (p.n_tile != 128 || p.pair_taps);
            const double turns = split ? 0.5 : (double)rounds, staging = turns * 6.0 * npix * p.cblks;
            const double bound = (turns * tile_time > staging ? turns * tile_time : staging) + (adds ? 9000.0 : 0.0);
            if (crop && adds && !flat_adds) cost += 9000.0;
            if (best_px != 0 && !(crop_mode >= 2 && crop != p.crop) &&
                (!(cost < (crop != p.crop ? 0.96 : 1.0) * best_cost) || (crop && crop_mode < 2 && staging > flat_bound))) return;
            if (crop && !allow_crop) { p.wants_crop = 1; return; }
            if (!crop) { flat_adds = adds; flat_bound = bound; }
            best_px = px;
            best_cost = cost;
            p.cost = cost;
            best_items = px_items;
            p.crop = crop;
            p.crop_items = crop_items;
            p.px_groups = groups;
            p.npix = (int)npix;
        };
        for (int px = 512; px >= 64; px -= 32) {
            if (forced_px && px != forced_px) continue;
            const int groups = (px + 255) / 256;
            if (px % (16 * groups) == 0) consider(px, groups, pixel_items(px), npix_of(px), 0, 0);
        }
        if (crop_mode != 0) {
            // The flat run also multiplies the windows of an image's last R - 1 rows, which wrap.  Items that are equal parts
            // of one image leave them out.  32 x 256 x 14 x 14, 256 of 3 x 3: 192 -> 176 pixels per item, 28.8 -> 26.9 us; 64 x 128 x
            // 32 x 32, 128 of 7 x 7: 147 items of 448 -> 128 of 416, 127 -> 115 us.  Of 150 random layers those whose estimate falls
            // by 4 % and more gain 3 % on average (up to 17 %, three lose 2.5 to 4 %), those with less between 0.87 and 1.3 without
            // a pattern; with few channels the producers set the pace, and more items stage more pixels (4 x 4 x 131 x 67, stride 2:
            // 14.9 -> 16.4 us).
            const long long plane = (long long)sh.H * sh.W, used = (long long)(sh.P - 1) * sh.W + sh.Q;
            for (int m = 1; m <= 64 && !p.wants_crop; ++m) {
                const long long cols = (used + m - 1) / m + p.ovl;
                const int groups = cols > 256 ? 2 : 1;
                const int n = (int)(((cols + groups - 1) / groups + 15) / 16 * 16);
                if (cols > 512) continue;
                if (cols < 64 && m > 1) break;
                consider(groups * n, groups, (long long)sh.N * m, npix_of(groups * n), 1, m);
            }
        }
        if (best_px == 0) return p;
        p.tile_px = best_px;
        p.supertiles = best_items > 0x7fffffffLL ? -1 : (int)best_items;
        // Filter stages: several taps per stage (up to 48 KB, trimmed below until three stages fit) so that the
        // warp that issues the MMAs pays its per-stage bookkeeping (barrier wait, commit: ~200 cycles, measured
        // by varying the stage size) once per 16-48 MMAs; the ring should hold
        // 64-128 KB in flight to cover the L2 latency.
        p.a_stages = 2;
        p.cbg = 1;
        p.tps = env_int("CONV2D_B200_TF32_STAGE_KB", 48) * 1024 / chunk;
        if (p.tps < 1) p.tps = 1;
        if (p.tps > p.taps) p.tps = p.taps;
        p.b_stages = 2;
        while (p.tps > 1 && smem_need(p.a_stages, p.npix, p.n_tile, 3, p.tps, p.cbg * stage_blocks) > kLimit) --p.tps;
        // equal stages: 6 taps as 3 + 3 instead of 5 + 1 (the short stage's MMAs would end long before the next
        // long stage has arrived)
        {
            const int per_block = (p.taps + p.tps - 1) / p.tps;
            p.tps = (p.taps + per_block - 1) / per_block;
        }
        // (phases have few MMAs per stage: stages of the image are worth more than filters far ahead)
        while (st > 1 && p.a_stages < kMaxAStages && smem_need(p.a_stages + 1, p.npix, p.n_tile, p.b_stages, p.tps, p.cbg * stage_blocks) <= kLimit) ++p.a_stages;
        while (p.b_stages < 4 && smem_need(p.a_stages, p.npix, p.n_tile, p.b_stages + 1, p.tps, p.cbg * stage_blocks) <= kLimit) ++p.b_stages;
        while (p.a_stages < kMaxAStages && p.taps <= 3 &&
               smem_need(p.a_stages + 1, p.npix, p.n_tile, p.b_stages, p.tps, p.cbg * stage_blocks) <= kLimit - 32 * 1024) ++p.a_stages;
        while (p.b_stages < kMaxBStages && smem_need(p.a_stages, p.npix, p.n_tile, p.b_stages + 1, p.tps, p.cbg * stage_blocks) <= kLimit &&
               (size_t)p.b_stages * p.tps * chunk < 128 * 1024) ++p.b_stages;
        p.smem_bytes = smem_need(p.a_stages, p.npix, p.n_tile, p.b_stages, p.tps, p.cbg * stage_blocks) + extra;
    }

    const int item_cols = p.tile_px;     // tensor-memory columns of one accumulator set
    if (!p.crop) {
        p.px_groups = (p.tile_px + 255) / 256;
        const int want = env_int("CONV2D_B200_TF32_PX_GROUPS", 0);
        if (want > 0 && want <= 2 && p.tile_px % (16 * want) == 0 && p.tile_px / want <= 256) p.px_groups = want;
    }
    if (p.pair_compact) p.px_groups = 1;
    p.nbuf = (2 * item_cols <= 512 && env_int("CONV2D_B200_TF32_NBUF", 2) != 1) ? 2 : 1;
    if (p.patch_w) p.patch_rows = (sh.P + p.tile_px / p.patch_w - 1) / (p.tile_px / p.patch_w);
    if (!p.crop) p.supertiles = pixel_items(p.tile_px) > 0x7fffffffLL ? -1 : (int)pixel_items(p.tile_px);
    if (p.supertiles <= 0) return p;
    // Too few tiles for the machine (e.g. 14 x 14 images): two work items per tile, each contracting half of
    // the channel-block groups and adding into a zeroed output.
    const int n_groups = (p.cblks + p.cbg - 1) / p.cbg;
    p.ksplit = ((long long)p.supertiles * p.n_blocks * 2 <= sms && n_groups >= 2 &&
                env_int("CONV2D_B200_TF32_KSPLIT", 1) != 0) ? 2 : 1;
    const long long items = (long long)p.supertiles * p.n_blocks * p.ksplit;
    if (items > 0x7fffffffLL) return p;
    p.grid = (int)(items < sms ? items : sms);
    // The split contraction as a two-block cluster: needs room for the exchange area behind the transposition tiles
    // (the filter ring gives up stages for it, down to two) and one item per block.
    p.cluster = 0;
    p.xchg_slots = 0;
    if (p.ksplit == 2 && !p.patch_w && !p.pair_taps && p.fold_r * p.fold_s == 1 && p.n_tile == 128 && !p.resident &&
        items <= sms && env_int("CONV2D_B200_TF32_KSPLIT_CLUSTER", 1) != 0) {
        const int slots = ((p.tile_px + 31) / 32 + 1) / 2;
        const size_t xb = xchg_area_bytes(slots);
        int bs = p.b_stages;
        while (bs > 2 && smem_need(p.a_stages, p.npix, p.n_tile, bs, p.tps, p.cbg * stage_blocks) + extra + xb > kSmemLimit) --bs;
        if (smem_need(p.a_stages, p.npix, p.n_tile, bs, p.tps, p.cbg * stage_blocks) + extra + xb <= kSmemLimit) {
            p.cluster = 1;
            p.xchg_slots = slots;
            p.b_stages = bs;
            p.smem_bytes = smem_need(p.a_stages, p.npix, p.n_tile, bs, p.tps, p.cbg * stage_blocks) + extra + xb;
        }
    }
    const int cols = (p.nbuf - 1) * item_cols + (item_cols + 31) / 32 * 32;      // (the write-back reads whole blocks of 32)
    p.tmem_cols = 32;
    while (p.tmem_cols < cols) p.tmem_cols <<= 1;
    p.makespan = (double)((items + sms - 1) / sms) * p.tile_px * p.pairs;
    p.ok = true;
    return p;
}

// Rough cycles of the busiest block: its MMAs with 400 for every filter stage (fitted when one lane alone ran the MMA loop), its
// producers (6 cycles per staged pixel and channel block, 5 where they load quads, a round trip to memory per block at
// least) and its write-back, which overlap for the most part; and the zero-fill and adds of a contraction split without a
// cluster (4.5 us).  Fitted to the times of 2070 random padded layers on virtual images and in patches (standard deviation
// 16 %; 19 % without the filter stages, which long halos make smaller and more).
double estimated_cycles(const Plan& p, bool quads)
{
    const int sms = sm_count();
    const double rounds = (double)(((long long)p.supertiles * p.n_blocks * p.ksplit + sms - 1) / sms);
    const double load = p.npix * (quads ? 5.0 : 6.0), blocks = rounds * p.cblks / p.ksplit;      // channel blocks in a row
    const double mma = p.makespan / p.ksplit + (p.resident ? 0.0 : blocks * ((p.taps + p.tps - 1) / p.tps) * 400.0);
    const double stage = blocks * (load > 1400.0 ? load : 1400.0);
    const double store = rounds * p.tile_px / 32.0 * (p.n_tile == 128 && !p.pair_taps ? 800.0 : 500.0);
    const double most = mma > stage ? (mma > store ? mma : store) : (stage > store ? stage : store);
    return 0.6 * most + 0.4 * (mma + stage + store) + (p.ksplit == 2 && !p.cluster ? 9000.0 : 0.0);
}

// Where patches are the better cut for zero padding.  Of 2070 random layers 112 were slower by 4 % and more on virtual images
// than in patches, 52 by more than 10 % (all layers together 14 % faster); with these rules it is 69 and 21, and none is slower
// by the rules:
bool patches_beat_virtual(const Plan& v, const Plan& patch, const Shape& sh)
{
    // a short contraction that only the virtual images split without a cluster: 5 x 80 x 65 x 33, 48 maps of 3 x 3 20.7 us
    // on virtual images, 15.4 in patches, 4 x 38 x 62 x 62, 115 of 7 x 3 26.8 and 16.8; 19 of 25 layers, none the other way (many
    // channels earn the split back: 9 x 256 x 116 x 10, 6 of 2 x 2 18.6 and 26.1)
    if (v.ksplit == 2 && !v.cluster && v.cblks <= 8 && patch.ksplit == 1 && patch.makespan < 16000.0) return true;
    // a clear difference of the estimates: 55 x 44 x 66 x 170, 7 maps of 5 x 5 259 and 188 us; 21 x 16 x 37 x 184, 4 of 7 x 7 67 and
    // 40; 2 x 272 x 51 x 247, 11 of 3 x 3 48 and 35
    const bool quads = sh.W % 4 == 0;
    const double ev = estimated_cycles(v, quads), ep = estimated_cycles(patch, quads && sh.pad_w % 4 == 0);
    return ev > 1.2 * ep && ev - ep > 6000.0;
}

// The patch width with the fewest staged pixels per output is the first choice.  A wider patch has a larger valid
// fraction (fewer MMA columns that only feed the next patch) and may need fewer rounds of items over the SMs: it is
// taken when the busiest block then has at least 5 % less MMA work (7 x 7 on 224 x 224, 64 -> 128 channels: 73 -> 61
// us with 64-column patches; 3 x 3 on 512 x 512: 101 -> 92 us; but 7 x 7 on 256 x 256: 196 us with 32 columns, 209 with 64,
// where both take two rounds of equal items).
Plan make_plan(const Shape& sh, bool b16 = false)
{
    // (the choice between virtual images, their widths and patches is made between plans without cropped items: with them the
    // estimates took virtual images for layers that patches do faster, 128 x 70 x 13 x 151, 32 of 4 x 4, padding 2: 93 -> 126 us);
    // planned once more only where the rule chooses them)
    auto cropped = [&](const Plan& p, bool narrow) {
        return p.ok && p.wants_crop ? plan_with_patch_width(sh, b16, 0, true, true, narrow) : p;
    };
    if (sh.stride > 1) {
        // Rows of a multiple of four columns allow 128-bit stores; where two columns less let the busiest block do a tenth
        // less (28 columns of output need 30: 145 items of 192 pixels instead of 133 of 224), pairs are the better cut.
        Plan p = plan_with_patch_width(sh, b16, 0, true, true, false, false);
        bool narrow = false;
        if (p.ok && sh.stride == 2 && env_int("CONV2D_B200_TF32_NARROW", 1) != 0) {
            const Plan q = plan_with_patch_width(sh, b16, 0, true, true, true, false);
            narrow = q.ok && q.makespan < 0.9 * p.makespan;
            if (narrow) p = q;
        }
        return cropped(p, narrow);
    }
    Plan best = plan_with_patch_width(sh, b16, 0);
    const int mode = env_int("CONV2D_B200_TF32_VIRT", 1);                 // 0 never, 1 by the rule, 2 always
    if (mode != 0 && (sh.pad_h != 0 || sh.pad_w != 0)) {
        // Padding: virtual images, unless their rows are so wide that patches stage far fewer pixels (and see above).
        const Plan v = plan_with_patch_width(sh, b16, 0, true, true, false, false);
        if (v.ok && (mode == 2 || !best.ok || !(v.staged_ratio > 1.75 * best.staged_ratio || patches_beat_virtual(v, best, sh)))) return cropped(v, false);
    }
    if (!best.ok || !best.patch_w || env_int("CONV2D_B200_TF32_PATCH_W", 0) != 0) return best;
    const int first = best.patch_w;
    for (int wp = 32; wp <= 128; wp *= 2) {
        if (wp == first) continue;
        const Plan q = plan_with_patch_width(sh, b16, wp);
        if (q.ok && q.patch_w == wp && q.makespan < 0.95 * best.makespan) best = q;
    }
    return best;
}

// How the re-ordered filters lie in the workspace: `rows` filters to a tap and filter block, `taps` to a channel block.  A call with
// packed filters may have another number and size of images and another padding than the one that packed them, so this (like the
// fold and the order of the taps) must follow from the filters' own sizes and the operand type.  Compact stacking
// depends on the image, too: it puts its pairs of taps together from the plain bank.
struct Bank { int rows, taps, stacked; };
Bank bank_layout(const Plan& p, const Shape& sh)
{
    if (p.pair_compact) return Bank{p.n_tile / 2, sh.R * sh.S, 0};
    return Bank{p.n_tile, p.taps, p.pair_taps};
}

size_t packed_floats(const Plan& p)
{
    return (size_t)p.n_blocks * (p.bank_bytes / 4);
}

}  // namespace
}  // namespace conv2d_b200
