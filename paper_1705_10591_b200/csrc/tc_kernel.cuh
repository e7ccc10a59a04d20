// Tensor-core convolution: the persistent kernel (filter copies, MMA issue, producers, epilogue) and its device
// helpers.  The design is described at the top of general_tf32.cu.  Included by general_tf32.cu only.
#pragma once
#include "tc_plan.cuh"
#include "ptx.cuh"
#include "tensor_map.cuh"
#include "fastdiv.cuh"

namespace conv2d_b200 {
namespace {


using namespace ptx;

// Tuning builds (-DCONV2D_B200_TC_DIAGNOSTICS) make the warp of block 0 that issues the MMAs count its cycles and leave
// them in status words 2-9 and 16.  The product build contains none of it: that warp's instruction stream is what
// bounds the heavy shapes, and a timer read with a memory clobber around every wait is not free.
#ifdef CONV2D_B200_TC_DIAGNOSTICS
constexpr bool kDiag = true;
#else
constexpr bool kDiag = false;
#endif
// Cycle counter read that the compiler may not move across memory operations or barriers (0 in product builds).
__device__ __forceinline__ long long clock_now()
{
    long long t = 0;
    if (kDiag) asm volatile("mov.u64 %0, %%clock64;" : "=l"(t) :: "memory");
    return t;
}
__device__ __forceinline__ unsigned long long wall_ns()
{
    unsigned long long t = 0;
    if (kDiag) asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

struct KernelArgs {
    const float* x;
    const float* wp;
    float* y;
    unsigned* status;
    int N, C, H, W, K, R, S, P, Q;
    int HW;
    int total_pix;
    FastDiv div_HW, div_W, div_npix, div_qn, div_patch_w;   // divisors of the pixel decoding (qn = npix / 4)
    int vec_shift;    // log2(vec)
    FastDiv div_ksplit, div_n_blocks, div_groups_lo, div_groups_hi, div_per_image, div_patch_cols;   // divisors of the item decoding
    int patch_item_rows;   // patch addressing: output rows of one item (tile_px / patch_w)
    int n_tile, n_blocks, tile_px, px_groups, nbuf, npix, cblks, taps, a_stages, b_stages, tps;
    int rot;          // quad producers rotate their chunk order per lane (see there)
    int cstride;      // 16-byte units between the 4-channel chunks of a staged channel block (npix + 1: odd)
    int patch_w, patch_tw, patch_rows, patch_cols;   // patch addressing (PATCH kernels): staged row pitch, valid output
                                                      // columns per patch row, patches per image down and across
    int pad_h, pad_w; // zero padding (patch addressing only): staged pixel (row, col) is image pixel (row - pad_h, col - pad_w)
    int row_pitch;    // pixels between vertically adjacent taps in the staged sequence: W, or patch_w
    int fp16;         // 16-bit operands only: 1 = IEEE half, 0 = bf16
    int fold_r, fold_s;  // taps folded into the channel dimension (1, 1: none); R, S below are what is left as shifts
    int helpers;      // 1: warps 8-15 share the write-back of a block's last item
    int pgroups;      // producer groups (1, 2 or 4): stage k is filled by group k % pgroups
    int quad2;        // 1: stride 2, producers load four adjacent pixels (two virtual pixels of both phases of a row) per word
    int quad;         // producers load four adjacent pixels per 128-bit (fp32) or 64-bit (16-bit operands) word (needs H*W % 4 == 0)
    int pair;         // 16-bit operands only: producers load two adjacent pixels per 32-bit word (needs H*W even)
    int cbg, groups;        // channel blocks per activation stage, number of such groups
    int resident;           // filters loaded once per thread block instead of streamed
    int vec;                // adjacent pixels a lane stores as one unit (1, 2 or 4)
    int pair_taps;          // stacked taps: accumulator lanes 64-127 hold the right-hand tap of each pair, one column to the right
    int s_slots, s_step;    // shift-table entries per filter row and the horizontal shift between them (2 with stacked taps)
    int pair_compact;       // stacked taps, resident bank: the odd last tap of a filter row is a 64-row slice of its own,
                            // issued as an M = 64 MMA onto the same accumulator lanes (no zero-padded upper half)
    int cb_bytes;           // resident filters: bytes of one channel block of the bank (all taps)
    int item_stride;        // flat addressing: pixels between the starts of consecutive items (tile_px minus the overlap)
    int crop;               // 1: items end with their image (div_per_image of them each), 0: they cut the whole sequence
    int ksplit;             // items per output tile (split of the contraction): 1 or 2
    int xchg_slots;         // cluster instances: 32-pixel blocks each block of a pair receives from its peer
    int xchg_bytes;         // ... and the bytes of the exchange area (rows + barriers) behind the transposition tiles
    unsigned max_polls;     // bound of every barrier wait
    int test_drop_stage;    // test hook: the filter copy with this ordinal is armed but never issued (-1: none)
    int early_x;            // 1: this call's filter re-ordering kernel directly precedes on the stream, so the image is
                            // final already and the producers need not wait for that kernel
    int early_next;         // 1: the next kernel on the stream may be placed while this one runs (see launch_pdl)
    // Virtual images (VIRT kernels): zero padding and strides, see staged_pixel_virtual.  H, W, HW are those of the image
    // in memory; div_HW and div_W divide by the virtual plane and row, total_pix counts virtual pixels.
    int st, off_h, off_w;   // stride; rows and columns of zeros before the image in the virtual one (before the stride)
    int shift0, ext;        // staged pixels between an output and its first tap; columns by which the taps start later in their phases
    int phases, phase_cols; // phases with taps of their own (1 where the taps are the same for all channels); columns of them
    int cblks_c;            // 16-channel blocks of one phase
    int mixed;              // 1: the phases of a channel are adjacent staged channels (few input channels), every tap for all
    int mix_c, mix_st2;     // ... channels of the image, stride * stride
    FastDiv div_phases;
    int items;              // work items = supertiles x n_blocks
    unsigned tmem_cols;
};

// Where the staged pixel sequence of a work item lives in the image.
//   flat  (PATCH = false): pixels of the whole batch numbered j = (n*H + h)*W + w; an item is the run
//          [j0, j0 + tile_px) plus its halo; vertically adjacent taps are W pixels apart.  The windows of an image's last
//          R - 1 rows wrap into the next image; where it pays the items leave them out (`crop`): they are equal
//          parts of one image.
//   patch (PATCH = true): an item is a rectangle of patch_rows... rows x patch_w columns of one image starting at
//          (row0, col0), stored row after row with pitch patch_w (the staged halo adds R-1 rows); vertically adjacent
//          taps are patch_w pixels apart.  Columns >= patch_tw of a patch row only feed outputs of the next patch and
//          are dropped.  This keeps the halo small on wide images, for which the flat run would not fit on chip.
struct ItemGeom {
    int j0;             // flat: first pixel
    int n, row0, col0;  // patch: image and top-left corner; flat: image from whose first pixel row0 counts
    int limit;          // flat: ... and the pixel at which the item's outputs end at the latest, counted from there, too
};
// Staged pixel jj -> (image n, offset inside one H*W plane); false when the pixel lies outside the batch / the image.
template <bool PATCH>
__device__ __forceinline__ bool staged_pixel(const KernelArgs& a, const ItemGeom& g, int jj, int& n, int& off)
{
    if (PATCH) {
        int pcol;
        const int prow = a.div_patch_w.divmod(jj, pcol);
        const int h = g.row0 + prow - a.pad_h, wc = g.col0 + pcol - a.pad_w;
        n = g.n;
        off = h * a.W + wc;
        return (unsigned)h < (unsigned)a.H && (unsigned)wc < (unsigned)a.W;
    }
    const int j = g.j0 + jj;
    n = a.div_HW.divmod(j, off);
    return j < a.total_pix;
}
// Accumulator column jj -> output (n, p, q); false when that output does not exist (window wraps over an edge).
template <bool PATCH>
__device__ __forceinline__ bool output_pixel(const KernelArgs& a, const ItemGeom& g, int jj, int& n, int& p, int& q)
{
    if (PATCH) {
        int pcol;
        const int prow = a.div_patch_w.divmod(jj, pcol);
        n = g.n;
        p = g.row0 + prow;
        q = g.col0 + pcol;
        return pcol < a.patch_tw && p < a.P && q < a.Q;
    }
    const int j = g.row0 + jj;
    if (j >= g.limit || jj >= a.item_stride) return false;           // (columns past the stride belong to the next item)
    int off;
    n = g.n + a.div_HW.divmod(j, off);
    p = a.div_W.divmod(off, q);
    return p < a.P && q < a.Q;
}

// Virtual images.  A padded convolution is computed on images that carry their zeros: rows of W + off_w columns, the
// first off_w of them zero (a multiple of four where the producers load quads), of which the zeros to the right of one
// row are those to the left of the next; in the same way the rows of zeros above an image are those below the one before.
// With a stride st the virtual pixel (h, w) of phase (a, b) is pixel (st*h + a - off_h, st*w + b - off_w) of the image:
// a stride-1 convolution whose taps (r, s) with r % st == a, s % st == b read phase (a, b) shifted by (r / st, s / st).
// Every staged channel block belongs to one phase and meets only that phase's taps: as many multiplications as the
// definition has (a rewritten image of st*st times as many channels has ceil(R/st)*ceil(S/st) taps on all of them).
struct Phase {
    int cblk, a, b;         // channel block of the image, phase
    int taps, cols;         // its taps, and how many of them lie in a row
    int col0;               // virtual columns before the first of them
    int base;               // taps of the phases before it
};
// (quad2: the phases are those of the rows, a.phase_cols = 1; each has the taps of both column phases, first those of
// column phase 0, and a channel block is two 16-channel blocks, one per column phase.)
// Phase number idx (once per block: the divisions would take a thread that runs alone some 1000 cycles per channel block,
// 32 x 128 x 56 x 56 with stride 2: 43.2 us with them on the way of the MMA thread, 41.7 without).
__device__ __forceinline__ uint2 describe_phase(const KernelArgs& a, int idx)
{
    const int pa = idx / a.phase_cols, pb = idx - pa * a.phase_cols;
    const int rows = (a.R - pa + a.st - 1) / a.st, end = a.S + a.ext;          // (taps in columns ext .. end - 1)
    const int col0 = pb < a.ext ? 1 : 0;
    const int cols = (end - pb + a.st - 1) / a.st - col0;
    const int rows_before = pa * (a.R / a.st) + min(pa, a.R % a.st);
    if (a.quad2 && a.phases > 1)
        return make_uint2((unsigned)(rows * a.S) | ((unsigned)a.S << 16), (unsigned)(rows_before * a.S) | ((unsigned)pa << 16));
    const int cols_before = pb * (end / a.st) + min(pb, end % a.st) - min(pb, a.ext);
    return make_uint2((unsigned)(rows * cols) | ((unsigned)cols << 16),
                      (unsigned)(rows_before * a.S + rows * cols_before) | ((unsigned)pa << 16) | ((unsigned)pb << 20) | ((unsigned)col0 << 24));
}
__device__ __forceinline__ Phase unpack_phase(uint2 v)
{
    Phase p;
    p.cblk = 0;
    p.taps = (int)(v.x & 0xffffu); p.cols = (int)(v.x >> 16);
    p.base = (int)(v.y & 0xffffu); p.a = (int)(v.y >> 16) & 15; p.b = (int)(v.y >> 20) & 15; p.col0 = (int)(v.y >> 24);
    return p;
}
// Channel block cb, from the block's table of phases.
__device__ __forceinline__ Phase phase_of(const KernelArgs& a, const uint2* phase_table, int cb)
{
    int idx;
    const int cblk = a.div_phases.divmod(cb, idx);
    Phase p = unpack_phase(phase_table[idx]);
    p.cblk = cblk;
    return p;
}
// Staged pixel -> image n and the image row and column of phase (0, 0), which may lie outside the image.
__device__ __forceinline__ bool staged_pixel_virtual(const KernelArgs& a, const ItemGeom& g, int jj, int& n, int& h, int& wc)
{
    const int j = g.j0 + jj;
    int rem;
    n = a.div_HW.divmod(j, rem);
    h = a.div_W.divmod(rem, wc);
    h = h * a.st - a.off_h;
    wc = wc * a.st - a.off_w;
    return j < a.total_pix;
}

// Producer helpers.  A stage holds `cbg` channel blocks of kCB channels for npix pixels, laid out
// [channel block][chunk][pixel] in 16-byte units.  A work unit is (channel block g, pixel jj), numbered
// i = g * npix + jj; thread t of the 256 producers owns units first + t, first + t + 256, ...  Consecutive
// lanes read consecutive pixels of one channel (coalesced) and write consecutive 16-byte units.
template <bool B16, bool FOLD, bool PATCH, bool VIRT, int CNT>
__device__ __forceinline__ void load_units(float (&v)[CNT][kCB], const KernelArgs& a, const uint2* phase_table, const ItemGeom& geom, int cb0, int first, int wtid, int nthr)
{
    const int units = a.npix * a.cbg;
#pragma unroll
    for (int u = 0; u < CNT; ++u) {
        const int i = first + u * nthr + wtid;
#pragma unroll
        for (int e = 0; e < kCB; ++e) v[u][e] = 0.f;
        if (i < units) {
            int jj;
            const int g = a.div_npix.divmod(i, jj);
            if (VIRT) {
                int n, h, wc;
                if (!staged_pixel_virtual(a, geom, jj, n, h, wc)) continue;
                const float* img = a.x + (size_t)n * a.C * a.HW;
                if (a.mixed) {
                    // staged channel (c, a, b): one pixel of every phase of a channel after the other
                    int vc = (cb0 + g) * kCB;
                    int c = vc / a.mix_st2, ph = vc - c * a.mix_st2;
                    int pa = ph / a.st, pb = ph - pa * a.st;
                    const float* src = img + (size_t)c * a.HW + h * a.W + wc;
#pragma unroll
                    for (int e = 0; e < kCB; ++e) {
                        if (c < a.mix_c && (unsigned)(h + pa) < (unsigned)a.H && (unsigned)(wc + pb) < (unsigned)a.W)
                            v[u][e] = __ldg(src + pa * a.W + pb);
                        if (++pb == a.st) { pb = 0; if (++pa == a.st) { pa = 0; ++c; src += a.HW; } }
                    }
                } else {
                    const Phase p = phase_of(a, phase_table, cb0 + g);
                    h += p.a;
                    wc += p.b;
                    const int c0 = p.cblk * kCB;
                    if ((unsigned)h < (unsigned)a.H && (unsigned)wc < (unsigned)a.W) {
                        const float* src = img + (size_t)c0 * a.HW + h * a.W + wc;
#pragma unroll
                        for (int e = 0; e < kCB; ++e)
                            if (c0 + e < a.C) v[u][e] = __ldg(src + (size_t)e * a.HW);
                    }
                }
                continue;
            }
            if (FOLD) {
                // Folded taps: staged channel vc = (c, r, s) of pixel j is x[c] at pixel j + r*W + s (zero beyond
                // the image: such windows belong to outputs that are dropped anyway).
                constexpr int kPer = B16 ? 2 * kCB : kCB;             // channels per 64-byte unit
                int n, off;
                if (staged_pixel<false>(a, geom, jj, n, off)) {
                    const int frs = a.fold_r * a.fold_s;
                    const int vc0 = (cb0 + g) * kPer;
                    int c = vc0 / frs, rem = vc0 - c * frs;
                    int r = rem / a.fold_s, sft = rem - r * a.fold_s;
                    const size_t base = (size_t)n * a.C * a.HW + off;
#pragma unroll
                    for (int e = 0; e < kPer; ++e) {
                        const int shift = r * a.W + sft;
                        const bool in = c < a.C && off + shift < a.HW;
                        if (B16) {
                            unsigned h = 0;
                            if (in) h = __ldg(reinterpret_cast<const unsigned short*>(a.x) + base + (size_t)c * a.HW + shift);
                            const unsigned prev = __float_as_uint(v[u][e >> 1]);
                            v[u][e >> 1] = __uint_as_float((e & 1) ? (prev | (h << 16)) : h);
                        } else {
                            if (in) v[u][e] = __ldg(a.x + base + (size_t)c * a.HW + shift);
                        }
                        if (++sft == a.fold_s) { sft = 0; if (++r == a.fold_r) { r = 0; ++c; } }
                    }
                }
            } else if (B16 && !FOLD && a.pair) {
                // Unit = 2 adjacent pixels x 16 channels: every load is one aligned 32-bit word holding the
                // two pixels of one channel (H*W even keeps pairs aligned and inside one image).
                const int half_n = a.npix >> 1;
                const int h = jj / half_n, pp = jj - h * half_n;
                const int c0 = (cb0 + g) * 2 * kCB + kCB * h;
                int n, off;
                if (staged_pixel<PATCH>(a, geom, 2 * pp, n, off) && c0 < a.C) {
                    const unsigned short* src = reinterpret_cast<const unsigned short*>(a.x) + ((size_t)n * a.C + c0) * a.HW + off;
#pragma unroll
                    for (int e = 0; e < kCB; ++e)
                        if (c0 + e < a.C) v[u][e] = __uint_as_float(__ldg(reinterpret_cast<const unsigned*>(src + (size_t)e * a.HW)));
                }
            } else if (B16) {
                // 32 16-bit channels of this pixel, packed two per 32-bit word (lower channel in the low half)
                const int c0 = (cb0 + g) * 2 * kCB;
                int n, off;
                if (staged_pixel<PATCH>(a, geom, jj, n, off) && c0 < a.C) {
                    const unsigned short* src = reinterpret_cast<const unsigned short*>(a.x) + ((size_t)n * a.C + c0) * a.HW + off;
#pragma unroll
                    for (int e = 0; e < kCB; ++e) {
                        unsigned lo = 0, hi = 0;
                        if (c0 + 2 * e < a.C) lo = __ldg(src + (size_t)(2 * e) * a.HW);
                        if (c0 + 2 * e + 1 < a.C) hi = __ldg(src + (size_t)(2 * e + 1) * a.HW);
                        v[u][e] = __uint_as_float(lo | (hi << 16));
                    }
                }
            } else {
                const int c0 = (cb0 + g) * kCB;
                int n, off;
                if (staged_pixel<PATCH>(a, geom, jj, n, off) && c0 < a.C) {
                    const float* src = a.x + ((size_t)n * a.C + c0) * a.HW + off;
#pragma unroll
                    for (int e = 0; e < kCB; ++e)
                        if (c0 + e < a.C) v[u][e] = __ldg(src + (size_t)e * a.HW);
                }
            }
        }
    }
}

template <bool B16, int CNT>
__device__ __forceinline__ void store_units(const float (&v)[CNT][kCB], float4* dst, const KernelArgs& a, int first, int wtid, int nthr)
{
    const int units = a.npix * a.cbg;
#pragma unroll
    for (int u = 0; u < CNT; ++u) {
        const int i = first + u * nthr + wtid;
        if (i < units) {
            int jj;
            const int g = a.div_npix.divmod(i, jj);
            if (B16 && a.pair) {
                const int half_n = a.npix >> 1;
                const int h = jj / half_n, pp = jj - h * half_n;
                float4* d = dst + ((size_t)g * kChunks + 2 * h) * a.cstride + 2 * pp;
#pragma unroll
                for (int m = 0; m < 2; ++m) {       // 8 channels per 16-byte unit; word k = channels 2k, 2k+1
                    unsigned lo[4], hi[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const unsigned w0 = __float_as_uint(v[u][8 * m + 2 * k]), w1 = __float_as_uint(v[u][8 * m + 2 * k + 1]);
                        lo[k] = __byte_perm(w0, w1, 0x5410);     // first pixel: low halves
                        hi[k] = __byte_perm(w0, w1, 0x7632);     // second pixel: high halves
                    }
                    d[m * a.cstride] = make_float4(__uint_as_float(lo[0]), __uint_as_float(lo[1]), __uint_as_float(lo[2]), __uint_as_float(lo[3]));
                    d[m * a.cstride + 1] = make_float4(__uint_as_float(hi[0]), __uint_as_float(hi[1]), __uint_as_float(hi[2]), __uint_as_float(hi[3]));
                }
                continue;
            }
            float4* d = dst + (size_t)g * kChunks * a.cstride + jj;
#pragma unroll
            for (int ch = 0; ch < kChunks; ++ch)
                d[ch * a.cstride] = B16 ? make_float4(v[u][4 * ch], v[u][4 * ch + 1], v[u][4 * ch + 2], v[u][4 * ch + 3])
                                      : make_float4(to_tf32_rna(v[u][4 * ch]), to_tf32_rna(v[u][4 * ch + 1]),
                                                    to_tf32_rna(v[u][4 * ch + 2]), to_tf32_rna(v[u][4 * ch + 3]));
        }
    }
}

// The four pixels of a quad from number `turn` on, cyclically.
__device__ __forceinline__ float4 turned(float4 v, int turn)
{
    if (turn & 1) v = make_float4(v.y, v.z, v.w, v.x);
    if (turn & 2) v = make_float4(v.z, v.w, v.x, v.y);
    return v;
}

// Work item -> (supertile, filter block, part of the contraction).  With ksplit = 2 two items share an
// output tile, each contracts half of the channel-block groups and both add their partial sums into y
// (zeroed beforehand); 0 + a + b does not depend on the order, so the result stays deterministic.
struct ItemInfo {
    int supertile, nb, g_begin, n_groups, rot;
    ItemGeom geom;
};
__device__ __forceinline__ ItemInfo decode_item(const KernelArgs& a, int item)
{
    ItemInfo it;
    // (multiply-high divisions: this runs at the head of every item on the MMA thread and on the producers)
    int part;
    const int rest = a.div_ksplit.divmod(item, part);
    it.supertile = a.div_n_blocks.divmod(rest, it.nb);
    it.g_begin = a.div_ksplit.div(part * a.groups);
    it.n_groups = a.div_ksplit.div((part + 1) * a.groups) - it.g_begin;
    // blocks stream the filter bank in rotated order (see kernel); n_groups is floor or ceil of groups / ksplit
    (it.n_groups == a.div_groups_lo.d ? a.div_groups_lo : a.div_groups_hi).divmod(rest, it.rot);
    it.geom.j0 = it.geom.row0 = it.supertile * a.item_stride;
    it.geom.n = it.geom.col0 = 0;
    it.geom.limit = a.total_pix;
    if (a.crop) {
        int part;
        it.geom.n = a.div_per_image.divmod(it.supertile, part);
        it.geom.row0 = part * a.item_stride;
        const int plane = (int)a.div_HW.d;
        it.geom.limit = plane;
        it.geom.j0 = it.geom.n * plane + it.geom.row0;
    }
    if (a.patch_w) {
        int rem, pc;
        it.geom.n = a.div_per_image.divmod(it.supertile, rem);
        const int pr = a.div_patch_cols.divmod(rem, pc);
        it.geom.row0 = pr * a.patch_item_rows;
        it.geom.col0 = pc * a.patch_tw;
    }
    return it;
}

// All MMAs of one tap of one channel block: K steps 0 and 1 for GROUPS pixel groups of n_mma pixels.  d: accumulator
// column of group 0; px_lo / flt_lo: low words of the pixel and filter descriptors of K step 0 (the K step and the group
// add constants to the start-address field); acc = 0 only for the very first tap of an item.  The whole warp executes it,
// the lane with `elected` != 0 issues.
template <bool B16, int GROUPS>
__device__ __forceinline__ void issue_tap(uint32_t d, uint32_t px_lo, uint32_t flt_lo, uint32_t px_kstep, uint32_t flt_kstep,
                                          uint32_t n_mma, uint32_t desc_hi, uint32_t idesc, uint32_t acc, uint32_t elected)
{
#define CONV2D_GROUP_MMA(KIND, D, PX)                                                                         \
    asm volatile(                                                                                             \
        "{\n\t.reg .pred p, q, e;\n\t.reg .b64 f, x;\n\t.reg .b32 t;\n\t"                                 \
        "setp.ne.b32 p, %7, 0;\n\tsetp.eq.b32 q, 0, 0;\n\tsetp.ne.b32 e, %8, 0;\n\t"                         \
        "mov.b64 f, {%2, %5};\n\tmov.b64 x, {%1, %5};\n\t"                                                  \
        "@e tcgen05.mma.cta_group::1.kind::" KIND " [%0], f, x, %6, p;\n\t"                                    \
        "add.u32 t, %2, %4;\n\tmov.b64 f, {t, %5};\n\tadd.u32 t, %1, %3;\n\tmov.b64 x, {t, %5};\n\t"         \
        "@e tcgen05.mma.cta_group::1.kind::" KIND " [%0], f, x, %6, q;\n\t}"                                   \
        ::"r"(D), "r"(PX), "r"(flt_lo), "r"(px_kstep), "r"(flt_kstep), "r"(desc_hi), "r"(idesc), "r"(acc),    \
          "r"(elected) : "memory")
#pragma unroll
    for (int g = 0; g < GROUPS; ++g) {
        if (B16) CONV2D_GROUP_MMA("f16", d + g * n_mma, px_lo + g * n_mma);
        else CONV2D_GROUP_MMA("tf32", d + g * n_mma, px_lo + g * n_mma);
    }
#undef CONV2D_GROUP_MMA
}

// The resident bank of compact stacking.  In the workspace the bank lies tap by tap, as for every layer of these filters (whether
// they are stacked depends on the image, too); its slices of two taps are put together here, one box of the tensor
// map (pair_map_of) each, a lane a slice.  147 KB of 64 filters of 64 x 3 x 3 arrive as early as a bank stored in slices
// (2 x 56 x 56: 8.9 us either way); issued by one lane through a map with 256-byte L2 promotion 0.6 us later, as 32 bulk copies of 256 bytes
// to a slice 10 us later.  Not inlined: in line
// it costs the producers 2 to 10 % (128 x 64 x 56 x 56: 72.3 -> 74 us), whose registers are at the limit.
__device__ __noinline__ void load_pairs(unsigned char* dst, const float* bank, const CUtensorMap* map, int rows, int S, uint64_t* full,
                                        volatile uint32_t* abort_flag, int lane)
{
    constexpr uint32_t kTap = 64 * 16 * kChunks;
    if (lane == 0) mbar_arrive_expect_tx(full, (uint32_t)(rows * S) * kTap);
    __syncwarp();
    const unsigned char* src = reinterpret_cast<const unsigned char*>(bank);
    const int slots = (S + 1) / 2;
    for (int i = lane; i < rows * slots; i += 32) {
        const int r = i / slots, s = 2 * (i - r * slots), t = r * S + s;
        if (s + 1 < S) tma_load_5d(dst + (size_t)t * kTap, map, 0, 0, 0, 0, t, smem_u32(full));
        else bulk_g2s(dst + (size_t)t * kTap, src + (size_t)t * kTap, kTap, full);
    }
    if (*abort_flag) { uint32_t dummy = 0; mbar_wait_bounded(full, 0u, &dummy, 1u << 16); }
}

// CLUSTER: the two work items of a split contraction (ksplit = 2) run as a two-block cluster, one item per block.
// Each block stores every other 32-pixel block of the tile: it sends its partial sums of the peer's blocks into the
// peer's shared memory (distributed shared memory, plain stores) and adds what the peer sent to its own
// accumulators before the ordinary write-back.  No zero-fill of y, no atomic adds, and a + b = b + a keeps the
// result independent of timing.
// VIRT: zero padding and strides on virtual images (staged_pixel_virtual); flat addressing, fp32 operands.
// M64: at most 64 filters without stacked taps (the write-back takes two blocks at a time; in instances of its own, since as
// run-time code it cost the 128-filter layers 1 %: more spills in roles that are at the register limit).
// PIX (virtual images): 0: the producers load quads of pixels; 1, 2: single pixels, with 2 before they wait for the stage.  Instances of their
// own: together in one, the quads' code made the single pixels slower (48 x 384 x 46 x 31, 18 of 3 x 3, padding 1: 88 us, 80 apart; 32 x 64 x
// 55 x 55, 64 of 3 x 3, padding 1: 30.6 and 30.1; 50 x 175 x 52 x 52, 352 of 3 x 3, stride 3: 172 and 165).
template <bool B16, bool FOLD, bool PATCH, bool STACK, bool CLUSTER = false, bool VIRT = false, bool M64 = false, int PIX = 0>
__global__ void __launch_bounds__(kThreads, 1)
general_tc_kernel(const KernelArgs a, const __grid_constant__ CUtensorMap pair_map)
{
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr bool kEarlyLoads = PIX == 2 || (PIX == 0 && (B16 || STACK || M64 || CLUSTER));      // producers load before they wait for the stage (see there)
    constexpr bool kTurn = STACK || M64;                  // quad producers: lanes start with different pixels (see there)
    const uint32_t a_block_bytes = (uint32_t)kCB * a.cstride * 4 * (VIRT && a.quad2 && !a.mixed ? 2 : 1);       // one channel block of a stage
    const uint32_t a_stage_bytes = a_block_bytes * (uint32_t)a.cbg;
    const uint32_t b_chunk_bytes = (uint32_t)kCB * a.n_tile * 4;        // one (channel block, tap)
    const uint32_t b_stage_bytes = b_chunk_bytes * (uint32_t)a.tps;
    unsigned char* a_smem = smem;
    unsigned char* b_smem = smem + (size_t)a.a_stages * a_stage_bytes;
    if (STACK) b_smem = smem + ((size_t)a.a_stages * a_stage_bytes + 127) / 128 * 128;       // (tensor-map copies write to multiples of 128 bytes; stages are multiples of 64)
    const int bank_blocks = VIRT ? a.cblks_c : a.cblks;                 // pieces of cb_bytes in a filter block's bank
    const size_t b_region_bytes = a.resident ? (size_t)bank_blocks * a.cb_bytes : (size_t)a.b_stages * b_stage_bytes;
    float* xpose = reinterpret_cast<float*>(b_smem + b_region_bytes);
    unsigned char* after_xpose = b_smem + b_region_bytes + kXposeBytes;
    float* xchg = reinterpret_cast<float*>(after_xpose);     // CLUSTER: [4 quarters][xchg_slots][8 column groups][32 lanes][4 floats] partial sums from the peer
    uint64_t* xbar = reinterpret_cast<uint64_t*>(after_xpose + (size_t)kEpilogueWarps * a.xchg_slots * kXchgBlockFloats * 4);   // [4][xchg_slots]
    uint64_t* bars = reinterpret_cast<uint64_t*>(after_xpose + (CLUSTER ? a.xchg_bytes : 0));
    uint64_t* a_full = bars;                               // [kMaxAStages]
    uint64_t* a_empty = a_full + kMaxAStages;              // [kMaxAStages]
    uint64_t* b_full = a_empty + kMaxAStages;              // [kMaxBStages]
    uint64_t* b_empty = b_full + kMaxBStages;              // [kMaxBStages]
    uint64_t* acc_full = b_empty + kMaxBStages;            // [2]
    uint64_t* acc_empty = acc_full + 2;                    // [2]
    uint64_t* tail_full = acc_empty + 2;                   // [1] the block's last item is complete (for warps 8-15)
    uint64_t* drain_bar = tail_full + 1;                   // [1] time-out path only: the MMAs issued so far have completed
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain_bar + 1);
    volatile uint32_t* abort_flag = tmem_slot + 1;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    volatile unsigned long long* t_entry = reinterpret_cast<volatile unsigned long long*>(tmem_slot + 2);
    uint32_t* tap_shift = tmem_slot + 4;                   // phases with taps of their own: [R * S] shift of every tap, in staged pixels
    // (behind the tap shifts; the planner keeps kMaxTaps entries for both)
    uint2* phase_table = reinterpret_cast<uint2*>(tap_shift + ((VIRT ? a.R * a.S : 0) + 1) / 2 * 2);
    if (VIRT)
        for (int i = tid; i < a.phases; i += kThreads) phase_table[i] = describe_phase(a, i);
    if (VIRT && a.phases > 1) {
        // one table per phase, behind one another in the order of the filter bank
        for (int t = tid; t < a.R * a.S; t += kThreads) {
            const int r = t / a.S, sx = t - r * a.S + a.ext, r2 = r / a.st, s2 = sx / a.st;
            if (a.quad2) {
                // taps of column phase 1 read the second 16-channel block of the channel block (the bank has those in even
                // columns of the filter first, in whichever phase `ext` puts them)
                const int pa = r - r2 * a.st, pb = sx - s2 * a.st, rows = (a.R - pa + 1) / 2;
                const int odd = (sx - a.ext) & 1, even_cols = (a.S + 1) / 2;
                const int base = (pa * (a.R / 2) + min(pa, a.R % 2)) * a.S + (odd ? rows * even_cols : 0);
                tap_shift[base + r2 * (odd ? a.S / 2 : even_cols) + ((sx - a.ext) >> 1)] =
                    (uint32_t)(r2 * a.row_pitch + s2) + (pb ? (uint32_t)(kChunks * a.cstride) : 0u);
                continue;
            }
            const Phase p = unpack_phase(describe_phase(a, (r - r2 * a.st) * a.phase_cols + sx - s2 * a.st));
            tap_shift[p.base + r2 * p.cols + s2 - p.col0] = (uint32_t)(r2 * a.row_pitch + s2);
        }
    }
    if (kDiag && tid == 0) *t_entry = wall_ns();

    if (tid == 0) {
        for (int i = 0; i < a.a_stages; ++i) { mbar_init(&a_full[i], kProducers / a.pgroups); mbar_init(&a_empty[i], 1); }
        for (int i = 0; i < a.b_stages; ++i) { mbar_init(&b_full[i], 1); mbar_init(&b_empty[i], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&acc_full[i], 1); mbar_init(&acc_empty[i], kEpilogueWarps); }
        mbar_init(tail_full, 1);
        mbar_init(drain_bar, 1);
        if (CLUSTER)
            for (int i = 0; i < kEpilogueWarps * a.xchg_slots; ++i) mbar_init(&xbar[i], 32);
        *abort_flag = 0;
        fence_mbar_init();
    }
    __syncthreads();
    if (CLUSTER) cluster_sync_all();        // the peer's barriers exist before anything can arrive on them
    if (warp == 1) { tmem_alloc(tmem_slot, a.tmem_cols); tmem_relinquish(); }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    // Everything above touched only this block's shared and tensor memory; it may overlap the tail of the
    // preceding kernel on the stream (the filter re-ordering of this call, or the previous call).  From here
    // on global memory is read and written: every role waits for the preceding kernel first, except that the
    // producers go ahead when that kernel is this call's own filter re-ordering.  That one lets this kernel start only after
    // everything before it on the stream has finished, it does not touch the image, and the
    // image is read only: the first activation stages are then in flight while the filters are still being written.
    if (a.early_next) grid_dep_launch();
    if (!(a.early_x && producer_index(warp) >= 0)) grid_dep_wait();

    // Work item -> (supertile, filter block); blocks rotate the order of the channel-block groups by the
    // item number, so that at any moment they stream different parts of the filter bank.
    const int acc_cols = a.tile_px;   // tensor-memory columns of one accumulator set

    if (warp == 0) {
        // ---------------- filters: global -> shared by bulk copy, up to `tps` taps of one channel block per stage
        if (STACK && a.pair_compact) load_pairs(b_smem, a.wp, &pair_map, bank_blocks * a.R, a.S, &b_full[0], abort_flag, lane);
        else if (lane == 0) {
            int s = 0, issued = 0;
            uint32_t ph = 0;
            bool alive = true;
            if (a.resident) {
                // the whole filter bank (a single filter block in this mode), once, one bulk copy per channel
                // block, all on one barrier
                const unsigned char* src = reinterpret_cast<const unsigned char*>(a.wp);
                const uint32_t piece = (uint32_t)a.cb_bytes;
                mbar_arrive_expect_tx(&b_full[0], piece * (uint32_t)bank_blocks);
                for (int cb = 0; cb < bank_blocks; ++cb)
                    bulk_g2s(b_smem + (size_t)cb * piece, src + (size_t)cb * piece, piece, &b_full[0]);
                alive = false;          // nothing to stream
                if (*abort_flag) { uint32_t dummy = 0; mbar_wait_bounded(&b_full[0], 0u, &dummy, 1u << 16); }
            }
            for (int item = blockIdx.x; item < a.items && alive; item += gridDim.x) {
                const ItemInfo ii = decode_item(a, item);
                const int nb = ii.nb;
                const unsigned char* src = reinterpret_cast<const unsigned char*>(a.wp)
                                         + (size_t)nb * bank_blocks * (VIRT ? (size_t)a.cb_bytes : (size_t)a.taps * b_chunk_bytes);
                for (int grp = 0; grp < ii.n_groups && alive; ++grp) {
                    int gr = grp + ii.rot;
                    if (gr >= ii.n_groups) gr -= ii.n_groups;
                    gr += ii.g_begin;
                    for (int g = 0; g < a.cbg && alive; ++g) {
                        const int cbr = gr * a.cbg + g;
                        if (cbr >= a.cblks) break;
                        int taps = a.taps;
                        size_t cb_at = (size_t)cbr * a.taps;            // taps of the bank before this channel block's
                        if (VIRT && a.phases > 1) {
                            const Phase p = phase_of(a, phase_table, cbr);
                            taps = p.taps;
                            cb_at = (size_t)p.cblk * (a.R * a.S) + p.base;
                        }
                        for (int t0 = 0; t0 < taps; t0 += a.tps) {
                            const int nt = min(a.tps, taps - t0);
                            if (!mbar_wait_bounded(&b_empty[s], ph ^ 1u, abort_flag, a.max_polls)) { alive = false; break; }
                            const uint32_t bytes = b_chunk_bytes * (uint32_t)nt;
                            mbar_arrive_expect_tx(&b_full[s], bytes);
                            if (issued != a.test_drop_stage)     // (test hook: a dropped copy makes the consumer's wait expire)
                                bulk_g2s(b_smem + (size_t)s * b_stage_bytes, src + (cb_at + t0) * b_chunk_bytes,
                                         bytes, &b_full[s]);
                            ++issued;
                            if (++s == a.b_stages) { s = 0; ph ^= 1u; }
                        }
                    }
                }
            }
            if (*abort_flag && !a.resident) {
                // let copies already in flight land before the block's shared memory is released
                const int pending = issued < a.b_stages ? issued : a.b_stages;
                for (int i = 0; i < pending; ++i) {
                    const int it = issued - 1 - i;
                    uint32_t dummy = 0;
                    mbar_wait_bounded(&b_full[it % a.b_stages], (uint32_t)(it / a.b_stages) & 1u, &dummy, 1u << 16);
                }
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issue.  All 32 lanes run the loop and one elected lane issues, which is faster than a loop that one
        // lane runs alone (presumably because warp-uniform operands need no moves).  In a loop of this shape with a
        // stage boundary every 6 to 10 MMAs, cycles per MMA of a lone lane / of the warp: N = 256 155 / 132, N = 224 (two
        // groups) 122 / 114, N = 176 139 / 99, N = 96 161 / 93 (the pipe's own: 128, 112, 88, 64).
        {
            const uint32_t elected = elect_one();
            const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem, 0);      // (warp-uniform for the compiler, too)
            const uint32_t n_mma = (uint32_t)(a.tile_px / a.px_groups);          // pixels per MMA
            const uint32_t idesc = B16 ? idesc_b16((uint32_t)a.n_tile, n_mma, a.fp16 != 0) : idesc_tf32((uint32_t)a.n_tile, n_mma);
            // (the start-address field of a descriptor holds bits 4-17 of the shared-memory address; the address of a
            // block that is not the first of its cluster has bits above those set, which must not leak into LBO)
            const uint32_t desc_hi = (128u >> 4) | (1u << 14);                  // SBO = 128 B, descriptor version 1
            const uint32_t a_lo_fixed = ((uint32_t)a.cstride & 0x3FFFu) << 16;  // LBO = chunk stride * 16 B
            const uint32_t b_lo_fixed = ((uint32_t)a.n_tile & 0x3FFFu) << 16;   // LBO = n_tile * 16 B
            const uint32_t a_kstep = 2u * (uint32_t)a.cstride;                  // 8 channels further, in 16-byte units
            const uint32_t b_kstep = 2u * (uint32_t)a.n_tile;
            bool alive = true;
            int as = 0, bs = 0, buf = 0;
            uint32_t a_phase = 0, b_phase = 0, acc_phase0 = 0, acc_phase1 = 0;
            // diagnostics of block 0 (status words 2..5): cycles this thread waited for activations and for a
            // free accumulator set, its total cycles, its item count
            long long wait_a = 0, wait_b = 0, wait_acc = 0, issue_cycles = 0;
            const long long t_begin = clock_now();
            if (kDiag && blockIdx.x == 0 && lane == 0) a.status[6] = (unsigned)(wall_ns() - *t_entry);   // ns from kernel entry to the start of the MMA loop
            int n_items = 0;
            if (a.resident) {
                if (!mbar_wait_bounded_warp(&b_full[0], 0u, abort_flag, a.max_polls)) alive = false;
                tc_fence_after_sync();
            }
            for (int item = blockIdx.x; item < a.items && alive; item += gridDim.x) {
                const ItemInfo ii = decode_item(a, item);
                // the accumulator set must have been drained by the epilogue of its previous item
                const uint32_t acc_phase = buf ? acc_phase1 : acc_phase0;
                long long tw = clock_now();
                if (!mbar_wait_bounded_warp(&acc_empty[buf], acc_phase ^ 1u, abort_flag, a.max_polls)) { alive = false; break; }
                tc_fence_after_sync();
                wait_acc += clock_now() - tw;
                const uint32_t d0 = tmem_u + (uint32_t)(buf * acc_cols);
                uint32_t accumulate = 0;
                for (int grp = 0; grp < ii.n_groups && alive; ++grp) {
                    tw = clock_now();
                    if (!mbar_wait_bounded_warp(&a_full[as], a_phase, abort_flag, a.max_polls)) { alive = false; break; }
                    tc_fence_after_sync();
                    wait_a += clock_now() - tw;
                    const long long t_issue0 = clock_now();
                    int gr = grp + ii.rot;
                    if (gr >= ii.n_groups) gr -= ii.n_groups;
                    gr += ii.g_begin;
                    uint32_t a_lo_block = a_lo_fixed | ((smem_u32(a_smem + (size_t)as * a_stage_bytes) >> 4) & 0x3FFFu);
                    for (int g = 0; g < a.cbg && alive; ++g, a_lo_block += a_block_bytes >> 4) {
                        if (gr * a.cbg + g >= a.cblks) break;
                        uint32_t row_shift = 0;                                  // r * row pitch, in pixels (= 16-byte units)
                        int sx = 0, sc = 0, taps = a.taps, tap0 = 0;
                        size_t bank_at = (size_t)(gr * a.cbg + g) * a.cb_bytes;   // (resident filters)
                        if (VIRT && a.phases > 1) {
                            const Phase p = phase_of(a, phase_table, gr * a.cbg + g);
                            taps = p.taps; tap0 = p.base;
                            bank_at = (size_t)p.cblk * a.cb_bytes + (size_t)p.base * b_chunk_bytes;
                        }
                        for (int t0 = 0; t0 < taps; t0 += a.tps) {
                            const int nt = min(a.tps, taps - t0);
                            uint32_t b_lo;
                            if (a.resident) {
                                b_lo = b_lo_fixed | ((smem_u32(b_smem + bank_at) >> 4) & 0x3FFFu);
                            } else {
                                const long long tb = clock_now();
                                if (!mbar_wait_bounded_warp(&b_full[bs], b_phase, abort_flag, a.max_polls)) { alive = false; break; }
                                wait_b += clock_now() - tb;
                                tc_fence_after_sync();
                                b_lo = b_lo_fixed | ((smem_u32(b_smem + (size_t)bs * b_stage_bytes) >> 4) & 0x3FFFu);
                            }
                            // (the taps of a phase lie in its table; all others step through the rows)
                            const bool table = VIRT && a.phases > 1;
                            const uint32_t* shift = tap_shift + tap0 + t0;
                            auto next_tap = [&](int t) {
                                uint32_t px_lo = a_lo_block + (VIRT ? (uint32_t)a.shift0 : 0u);
                                if (table) return px_lo + shift[t];
                                px_lo += row_shift + (uint32_t)sx;
                                sx += a.s_step;
                                if (++sc == a.s_slots) { sc = 0; sx = 0; row_shift += (uint32_t)a.row_pitch; }
                                return px_lo;
                            };
                            if (STACK && a.pair_compact) {
                                // pairs of taps as M = 128 slices, a lone last tap as an M = 64 slice of half the size
                                // (its chunk stride and K step are half as long too) onto the same accumulator lanes
                                const uint32_t idesc64 = B16 ? idesc_b16(64u, n_mma, a.fp16 != 0) : idesc_tf32(64u, n_mma);
                                // (first the pairs of all rows, then the lone taps: every change between the two shapes drains the
                                // pipe, 32 x 64 x 56 x 56, 64 of 3 x 3, padding 1: 28.0 -> 27.7 us)
                                const int pairs = a.S >> 1;
                                const uint32_t slice = b_chunk_bytes >> 4, px0 = a_lo_block + (VIRT ? (uint32_t)a.shift0 : 0u);
                                const uint32_t row_units = (uint32_t)pairs * slice + ((a.S & 1) ? slice >> 1 : 0u);
                                for (int r = 0; r < a.R; ++r)
                                    for (int u = 0; u < pairs; ++u) {
                                        issue_tap<B16, 1>(d0, px0 + (uint32_t)(r * a.row_pitch + 2 * u), b_lo + (uint32_t)r * row_units + (uint32_t)u * slice, a_kstep, b_kstep, n_mma, desc_hi, idesc, accumulate, elected);
                                        accumulate = 1;
                                    }
                                if (a.S & 1)
                                    for (int r = 0; r < a.R; ++r)
                                        issue_tap<B16, 1>(d0, px0 + (uint32_t)(r * a.row_pitch + 2 * pairs), b_lo + (uint32_t)r * row_units + (uint32_t)pairs * slice - (64u << 16), a_kstep, b_kstep >> 1, n_mma, desc_hi, idesc64, accumulate, elected);
                                accumulate = 1;
                            } else if (a.px_groups == 1) {
#pragma unroll 3
                                for (int t = 0; t < nt; ++t, b_lo += b_chunk_bytes >> 4) {
                                    issue_tap<B16, 1>(d0, next_tap(t), b_lo, a_kstep, b_kstep, n_mma, desc_hi, idesc, accumulate, elected);
                                    accumulate = 1;
                                }
                            } else {
                                for (int t = 0; t < nt; ++t, b_lo += b_chunk_bytes >> 4) {
                                    issue_tap<B16, 2>(d0, next_tap(t), b_lo, a_kstep, b_kstep, n_mma, desc_hi, idesc, accumulate, elected);
                                    accumulate = 1;
                                }
                            }
                            if (!a.resident) {
                                mma_commit(&b_empty[bs], elected);   // frees the filter stage when these MMAs have read it
                                if (++bs == a.b_stages) { bs = 0; b_phase ^= 1u; }
                            }
                        }
                    }
                    issue_cycles += clock_now() - t_issue0;
                    if (alive) mma_commit(&a_empty[as], elected);
                    if (++as == a.a_stages) { as = 0; a_phase ^= 1u; }
                }
                if (alive) mma_commit(&acc_full[buf], elected);
                if (alive && item + (int)gridDim.x >= a.items) mma_commit(tail_full, elected);
                if (buf) acc_phase1 ^= 1u; else acc_phase0 ^= 1u;
                if (++buf == a.nbuf) buf = 0;
                ++n_items;
            }
            if (!alive) {
                // A wait ran out: MMAs issued before that may still be reading shared memory and writing tensor
                // memory.  Let them finish (bounded) before the block frees its tensor memory and exits.
                mma_commit(drain_bar, elected);
                uint32_t dummy = 0;
                mbar_wait_bounded(drain_bar, 0u, &dummy, 1u << 16);
            }
            if (kDiag && blockIdx.x == 0 && lane == 0) {
                a.status[2] = (unsigned)wait_a;
                a.status[3] = (unsigned)wait_acc;
                a.status[4] = (unsigned)(clock_now() - t_begin);
                a.status[5] = (unsigned)n_items;
                a.status[9] = (unsigned)(issue_cycles - wait_b);
                a.status[16] = (unsigned)wait_b;
                a.status[7] = (unsigned)(wall_ns() - *t_entry);  // ns from kernel entry to the last MMA issued
            }
        }
    } else {
    if (producer_index(warp) >= 0) {
        // ---------------- producers: stage activations, running ahead across item boundaries
        // The producer warps form `pgroups` groups; stage k of the block's stage sequence is filled by group
        // k % pgroups, so that several stages' memory round trips are in flight at once (a stage of a light
        // problem has fewer 16-channel units than there are producer threads).
        const int nthr_shift = a.pgroups == 4 ? 6 : (a.pgroups == 2 ? 7 : 8);     // kProducers = 256 threads; no divisions here:
        const int nthr = 1 << nthr_shift;                                         // this is on the path to the first load
        const int gid = (producer_index(warp) * 32 + lane) >> nthr_shift;
        const int wtid = (producer_index(warp) * 32 + lane) - gid * nthr;
        bool alive = true;
        int kstage = 0;
        int next_as = 0;                 // ring slot and phase of stage `kstage`, advanced without divisions
        uint32_t next_phase = 0;
        const int units = a.npix * a.cbg;
        for (int item = blockIdx.x; item < a.items && alive; item += gridDim.x) {
            const ItemInfo ii = decode_item(a, item);
            // One stage = cbg consecutive channel blocks.  All loads of a pass (kUnitsPerThread units of
            // 16 channels per thread) are issued before its first store: a pass costs one memory round trip.
            for (int grp = 0; grp < ii.n_groups && alive; ++grp, ++kstage) {
                const int as = next_as;
                const uint32_t a_phase = next_phase;
                if (++next_as == a.a_stages) { next_as = 0; next_phase ^= 1u; }
                if ((kstage & (a.pgroups - 1)) != gid) continue;         // pgroups is 1, 2 or 4
                // The stage is waited for when the first loads are under way (kEarlyLoads): they need registers only, and a ring of two stages
                // has no time to spare for their latency (with the turned stores below 32 x 64 x 56 x 56, 64 of 3 x 3, padding 1: 27.7 -> 23.1 us;
                // 64 x 128 x 32 x 32, 128 of 3 x 3 in bf16 24.8 -> 23.4).  Of 128 fp32 filters in blocks of their own the wait comes first
                // (32 x 128 x 56 x 56, stride 2 30.5 us, 31.9 with the loads first; 28 x 45 x 100 x 100, 176 of 3 x 3 110 and 122).
                bool waited = !kEarlyLoads;
                if (waited && !mbar_wait_bounded(&a_empty[as], a_phase ^ 1u, abort_flag, a.max_polls)) { alive = false; break; }
                auto stage_free = [&]() {
                    if (!waited) {
                        waited = true;
                        if (!mbar_wait_bounded(&a_empty[as], a_phase ^ 1u, abort_flag, a.max_polls)) alive = false;
                    }
                    return alive;
                };
                float4* dst = reinterpret_cast<float4*>(a_smem + (size_t)as * a_stage_bytes);
                int gr = grp + ii.rot;
                if (gr >= ii.n_groups) gr -= ii.n_groups;
                gr += ii.g_begin;
                if (VIRT && !PIX && a.quad2) {
                    // Stride 2: four adjacent pixels of an image row are two virtual pixels of both phases of that row.
                    const int qn = a.npix >> 1;
                    for (int i = wtid; i < qn * a.cbg; i += nthr) {
                        int pq;
                        const int g = a.div_qn.divmod(i, pq), cb = gr * a.cbg + g;
                        float4 v[kCB];
#pragma unroll
                        for (int e = 0; e < kCB; ++e) v[e] = make_float4(0.f, 0.f, 0.f, 0.f);
                        int n, h, wc;
                        const bool in = staged_pixel_virtual(a, ii.geom, 2 * pq, n, h, wc) && (unsigned)wc < (unsigned)a.W && cb < a.cblks;
                        float4* d = dst + (size_t)g * (a_block_bytes >> 4) + 2 * pq;
                        // (phases as channels: two pixels, 32 bytes of a chunk, per lane; four lanes of eight start with the second, see the quads below)
                        const int second = kTurn ? (pq >> 2) & 1 : 0, turn = 2 * second;
                        if (a.mixed) {
                            // a chunk holds the four phases of a channel: two rows of the image
                            const int c0 = cb * kChunks;
                            if (in) {
                                const float* src = a.x + ((size_t)n * a.C + c0) * a.HW + h * a.W + wc;
#pragma unroll
                                for (int c = 0; c < kChunks; ++c) {
                                    if (c0 + c >= a.C) break;
                                    if ((unsigned)h < (unsigned)a.H) v[2 * c] = __ldg(reinterpret_cast<const float4*>(src + (size_t)c * a.HW));
                                    if ((unsigned)(h + 1) < (unsigned)a.H) v[2 * c + 1] = __ldg(reinterpret_cast<const float4*>(src + (size_t)c * a.HW + a.W));
                                }
                            }
                            if (!stage_free()) break;
#pragma unroll
                            for (int c = 0; c < kChunks; ++c) {
                                const float4 r0 = turned(v[2 * c], turn), r1 = turned(v[2 * c + 1], turn);
                                d[c * a.cstride + second] = make_float4(to_tf32_rna(r0.x), to_tf32_rna(r0.y), to_tf32_rna(r1.x), to_tf32_rna(r1.y));
                                d[c * a.cstride + (second ^ 1)] = make_float4(to_tf32_rna(r0.z), to_tf32_rna(r0.w), to_tf32_rna(r1.z), to_tf32_rna(r1.w));
                            }
                        } else {
                            const Phase p = phase_of(a, phase_table, cb);
                            const int c0 = p.cblk * kCB;
                            h += p.a;
                            if (in && (unsigned)h < (unsigned)a.H) {
                                const float* src = a.x + ((size_t)n * a.C + c0) * a.HW + h * a.W + wc;
#pragma unroll
                                for (int e = 0; e < kCB; ++e)
                                    if (c0 + e < a.C) v[e] = __ldg(reinterpret_cast<const float4*>(src + (size_t)e * a.HW));
                            }
                            if (!stage_free()) break;
#pragma unroll
                            for (int ch = 0; ch < kChunks; ++ch) {
                                float4* dc = d + ch * a.cstride;
                                const float4 v0 = v[4 * ch], v1 = v[4 * ch + 1], v2 = v[4 * ch + 2], v3 = v[4 * ch + 3];
                                dc[0] = make_float4(to_tf32_rna(v0.x), to_tf32_rna(v1.x), to_tf32_rna(v2.x), to_tf32_rna(v3.x));
                                dc[1] = make_float4(to_tf32_rna(v0.z), to_tf32_rna(v1.z), to_tf32_rna(v2.z), to_tf32_rna(v3.z));
                                dc += kChunks * a.cstride;                     // the block of the phase one column to the right
                                dc[0] = make_float4(to_tf32_rna(v0.y), to_tf32_rna(v1.y), to_tf32_rna(v2.y), to_tf32_rna(v3.y));
                                dc[1] = make_float4(to_tf32_rna(v0.w), to_tf32_rna(v1.w), to_tf32_rna(v2.w), to_tf32_rna(v3.w));
                            }
                        }
                    }
                } else if (!B16 && !FOLD && !PIX && (VIRT || a.quad)) {
                    // H*W a multiple of 4: a thread fetches 4 adjacent pixels of each of the 16 channels with
                    // 128-bit loads (a quarter of the load instructions, which otherwise crowd the SM's memory
                    // pipeline that the MMA instructions pass through as well) and writes four 16-channel units.
                    const int qn = a.npix >> 2;
                    for (int i = wtid; i < qn * a.cbg; i += nthr) {
                        int pq;
                        const int g = a.div_qn.divmod(i, pq);
                        const int c0 = (gr * a.cbg + g) * kCB;
                        // Register group ch of this lane holds chunk (ch + rot) & 3: lanes whose 64-byte pieces
                        // would fall on the same banks write different chunks in the same instruction.  Measured:
                        // a gain with 16-bit operands (below) only; with fp32 inputs the rotation is left out,
                        // as it splits every 512-byte load instruction over four channel planes (slower from DRAM).
                        const int rot = !kTurn && a.rot ? (pq >> 1) & 3 : 0;
                        // A lane's four pixels are 64 bytes of a chunk, so eight lanes that all stored their first would meet on two
                        // of the eight 16-byte bank groups.  Each lane takes its pixels in turn from (lane / 2) % 4 on: eight lanes
                        // then cover all groups.  That costs four selections per stored word, and pays where shared memory sets the pace
                        // (at most 64 filters: 32 x 64 x 56 x 56, 64 of 3 x 3, padding 1 25.0 -> 23.1 us; but 32 x 256 x 14 x 14, 256 of 3 x 3 24.9 -> 25.3).
                        const int turn = kTurn ? (pq >> 1) & 3 : 0;
                        float4 v[kCB];
#pragma unroll
                        for (int e = 0; e < kCB; ++e) v[e] = make_float4(0.f, 0.f, 0.f, 0.f);
                        int n, off;
                        bool in;
                        if (VIRT) {             // (stride 1: four columns of a row lie in the image together or not at all)
                            int h, wc;
                            in = staged_pixel_virtual(a, ii.geom, 4 * pq, n, h, wc) && (unsigned)h < (unsigned)a.H && (unsigned)wc < (unsigned)a.W;
                            off = h * a.W + wc;
                        } else {
                            in = staged_pixel<PATCH>(a, ii.geom, 4 * pq, n, off);
                        }
                        if (in && c0 < a.C) {
                            const float* src = a.x + ((size_t)n * a.C + c0) * a.HW + off;
#pragma unroll
                            for (int ch = 0; ch < kChunks; ++ch) {
                                const int cc = ((ch + rot) & 3) << 2;                 // first channel of this register group
                                const float* sc = src + (size_t)cc * a.HW;
                                const int left = a.C - c0 - cc;                       // channels that exist from there on
#pragma unroll
                                for (int j = 0; j < 4; ++j)
                                    if (j < left) v[4 * ch + j] = __ldg(reinterpret_cast<const float4*>(sc + (size_t)j * a.HW));
                            }
                        }
                        if (!stage_free()) break;
                        float4* d = dst + (size_t)g * kChunks * a.cstride + 4 * pq;
                        if (kTurn) {
#pragma unroll
                            for (int ch = 0; ch < kChunks; ++ch, d += a.cstride) {
                                float4 u[4];                       // pixel (i + turn) % 4
#pragma unroll
                                for (int j = 0; j < 4; ++j) {
                                    const float4 t = turned(v[4 * ch + j], turn);
                                    reinterpret_cast<float*>(&u[0])[j] = to_tf32_rna(t.x);
                                    reinterpret_cast<float*>(&u[1])[j] = to_tf32_rna(t.y);
                                    reinterpret_cast<float*>(&u[2])[j] = to_tf32_rna(t.z);
                                    reinterpret_cast<float*>(&u[3])[j] = to_tf32_rna(t.w);
                                }
#pragma unroll
                                for (int i = 0; i < 4; ++i) d[(i + turn) & 3] = u[i];
                            }
                        } else {
#pragma unroll
                            for (int ch = 0; ch < kChunks; ++ch) {
                                float4* dc = d + ((ch + rot) & 3) * a.cstride;
                                dc[0] = make_float4(to_tf32_rna(v[4 * ch].x), to_tf32_rna(v[4 * ch + 1].x), to_tf32_rna(v[4 * ch + 2].x), to_tf32_rna(v[4 * ch + 3].x));
                                dc[1] = make_float4(to_tf32_rna(v[4 * ch].y), to_tf32_rna(v[4 * ch + 1].y), to_tf32_rna(v[4 * ch + 2].y), to_tf32_rna(v[4 * ch + 3].y));
                                dc[2] = make_float4(to_tf32_rna(v[4 * ch].z), to_tf32_rna(v[4 * ch + 1].z), to_tf32_rna(v[4 * ch + 2].z), to_tf32_rna(v[4 * ch + 3].z));
                                dc[3] = make_float4(to_tf32_rna(v[4 * ch].w), to_tf32_rna(v[4 * ch + 1].w), to_tf32_rna(v[4 * ch + 2].w), to_tf32_rna(v[4 * ch + 3].w));
                            }
                        }
                    }
                } else if (B16 && !FOLD && a.quad) {
                    // 16-bit operands, same idea: 64-bit loads of 4 adjacent pixels for each of the 32 channels of a
                    // block, then the 4 x 32 block is turned around in registers into four 64-byte units.
                    const int qn = a.npix >> 2;
                    for (int i = wtid; i < qn * a.cbg; i += nthr) {
                        int pq;
                        const int g = a.div_qn.divmod(i, pq);
                        const int c0 = (gr * a.cbg + g) * 2 * kCB;
                        const int rot = a.rot ? (pq >> 1) & 3 : 0;    // chunk rotation of this lane, as above
                        uint2 v[2 * kCB];
#pragma unroll
                        for (int e = 0; e < 2 * kCB; ++e) v[e] = make_uint2(0u, 0u);
                        int n, off;
                        if (staged_pixel<PATCH>(a, ii.geom, 4 * pq, n, off) && c0 < a.C) {
                            const unsigned short* src = reinterpret_cast<const unsigned short*>(a.x) + ((size_t)n * a.C + c0) * a.HW + off;
#pragma unroll
                            for (int ch = 0; ch < kChunks; ++ch) {
                                const int cc = ((ch + rot) & 3) << 3;
                                const unsigned short* sc = src + (size_t)cc * a.HW;
                                const int left = a.C - c0 - cc;
#pragma unroll
                                for (int j = 0; j < 8; ++j, sc += a.HW)
                                    if (j < left) v[8 * ch + j] = __ldg(reinterpret_cast<const uint2*>(sc));
                            }
                        }
                        if (!stage_free()) break;
                        float4* d = dst + (size_t)g * kChunks * a.cstride + 4 * pq;
#pragma unroll
                        for (int ch = 0; ch < kChunks; ++ch) {        // 8 channels per 16-byte unit; word k = channels 2k, 2k+1
                            float4* dc = d + ((ch + rot) & 3) * a.cstride;
                            unsigned p0[4], p1[4], p2[4], p3[4];
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const uint2 lo = v[8 * ch + 2 * k], hi = v[8 * ch + 2 * k + 1];
                                p0[k] = __byte_perm(lo.x, hi.x, 0x5410); p1[k] = __byte_perm(lo.x, hi.x, 0x7632);
                                p2[k] = __byte_perm(lo.y, hi.y, 0x5410); p3[k] = __byte_perm(lo.y, hi.y, 0x7632);
                            }
                            dc[0] = make_float4(__uint_as_float(p0[0]), __uint_as_float(p0[1]), __uint_as_float(p0[2]), __uint_as_float(p0[3]));
                            dc[1] = make_float4(__uint_as_float(p1[0]), __uint_as_float(p1[1]), __uint_as_float(p1[2]), __uint_as_float(p1[3]));
                            dc[2] = make_float4(__uint_as_float(p2[0]), __uint_as_float(p2[1]), __uint_as_float(p2[2]), __uint_as_float(p2[3]));
                            dc[3] = make_float4(__uint_as_float(p3[0]), __uint_as_float(p3[1]), __uint_as_float(p3[2]), __uint_as_float(p3[3]));
                        }
                    }
                } else
                for (int first = 0; first < units; first += nthr * kUnitsPerThread) {
                    float v[kUnitsPerThread][kCB];
                    load_units<B16, FOLD, PATCH, VIRT>(v, a, phase_table, ii.geom, gr * a.cbg, first, wtid, nthr);
                    if (!stage_free()) break;
                    store_units<B16>(v, dst, a, first, wtid, nthr);
                }
                if (!stage_free()) break;                    // (a thread without a unit of this stage, too)
                fence_proxy_async_smem();
                mbar_arrive(&a_full[as]);
            }
        }
    }
    if (warp >= 4 && (warp < 4 + kEpilogueWarps || a.helpers)) {
        // ---------------- epilogue: drain finished accumulator sets (lane = pixel)
        // Warps 4-7 drain every item.  The write-back of a block's LAST item cannot hide behind any later
        // MMAs, so there the eight warps 8-15 (producers that have finished staging, and the two spare
        // warps) join in: each lane quarter is then drained by three warps that take every third 32-pixel
        // block.  Their transposition tiles reuse the activation ring, which is idle by then.
        const int quarter = warp & 3;                       // tensor-memory lanes this warp may read
        const bool helper = warp >= 4 + kEpilogueWarps;
        const int share = helper ? 1 + ((warp - 8) >> 2) : 0;
        const size_t plane = (size_t)a.P * a.Q;
        const int n_local = ((int)blockIdx.x < a.items) ? (a.items - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
        bool alive = true;
        for (int li = helper ? n_local - 1 : 0; li >= 0 && li < n_local; ++li) {
            const int item = (int)blockIdx.x + li * (int)gridDim.x;
            const int buf = a.nbuf == 2 ? (li & 1) : 0;                              // nbuf is 1 or 2
            const uint32_t acc_phase = (uint32_t)(a.nbuf == 2 ? li >> 1 : li) & 1u;
            const bool split = a.helpers && li == n_local - 1;
            const ItemInfo ii = decode_item(a, item);
            const int nb = ii.nb;
            const bool add = !CLUSTER && a.ksplit > 1;       // partial sums: add into the zeroed output
            // tcgen05.ld is warp-collective: take the decision for the whole warp
            // (warps 8-15 come late and only for the last item: they wait on a barrier of its own, whose
            // phase they cannot have missed)
            const long long t_wait0 = clock_now();
            alive = __all_sync(0xffffffffu, alive && mbar_wait_bounded(helper ? tail_full : &acc_full[buf],
                                                                       helper ? 0u : acc_phase, abort_flag, a.max_polls));
            if (!alive) break;
            tc_fence_after_sync();
            const long long t_busy0 = clock_now();
            if (kDiag && blockIdx.x == 0 && warp == 4 && lane == 0) a.status[10] += (unsigned)(t_busy0 - t_wait0);   // waited for accumulators
            const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(buf * acc_cols);
            // Lanes are filters, columns pixels: this thread holds adjacent pixels of ONE map.  A
            // warp-private shared-memory tile turns a 32-filter x 32-pixel block around so that each
            // store instruction again writes 32 adjacent pixels of one map.
            float* tile = helper ? reinterpret_cast<float*>(a_smem) + (size_t)(warp - 8) * 32 * kXposePitch
                                 : xpose + (size_t)(warp - 4) * 32 * kXposePitch;
            // Stacked taps: lanes 0-15 of the quarter hold 16 maps summed over the left-hand taps, lanes 16-31 the
            // same maps over the right-hand taps, one column to the right: those lanes write their row shifted
            // by one column (with the first column of the next block), and a map is the sum of two tile rows.
            constexpr bool stacked = STACK;         // (a template parameter: as a run-time flag it slowed the ordinary epilogue by 15 %)
            const int rpq = stacked ? 16 : a.n_tile / 4;    // maps per lane quarter: 32 (M = 128) or 16 (M = 64: lanes 0-15; stacked taps)
            const int blocks = (a.tile_px + 31) / 32;
            auto load_block = [&](uint32_t (&v0)[16], uint32_t (&v1)[16], uint32_t (&vx)[1], int b) {
                tmem_ld16(lane_base + (uint32_t)(b * 32), v0);
                tmem_ld16(lane_base + (uint32_t)(b * 32 + 16), v1);
                vx[0] = 0u;
                if (stacked && b + 1 < blocks) tmem_ld1(lane_base + (uint32_t)(b * 32 + 32), vx);
            };
            auto store_block = [&](const uint32_t (&v0)[16], const uint32_t (&v1)[16], const uint32_t (&vx)[1], int b) {
                __syncwarp();                                   // the previous block has been read out
                float4* row = reinterpret_cast<float4*>(tile + lane * kXposePitch);
                if (stacked) {
                    const bool up = lane >= 16;
                    auto sel = [&](uint32_t lo, uint32_t hi) { return __uint_as_float(up ? hi : lo); };
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        row[i] = make_float4(sel(v0[4 * i], v0[4 * i + 1]), sel(v0[4 * i + 1], v0[4 * i + 2]),
                                             sel(v0[4 * i + 2], v0[4 * i + 3]), sel(v0[4 * i + 3], i < 3 ? v0[(4 * i + 4) & 15] : v1[0]));
                        row[4 + i] = make_float4(sel(v1[4 * i], v1[4 * i + 1]), sel(v1[4 * i + 1], v1[4 * i + 2]),
                                                 sel(v1[4 * i + 2], v1[4 * i + 3]), sel(v1[4 * i + 3], i < 3 ? v1[(4 * i + 4) & 15] : vx[0]));
                    }
                } else if (lane < rpq) {                        // M = 64: only lanes 0-15 of a quarter hold rows
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        row[i] = make_float4(__uint_as_float(v0[4 * i]), __uint_as_float(v0[4 * i + 1]),
                                             __uint_as_float(v0[4 * i + 2]), __uint_as_float(v0[4 * i + 3]));
                        row[4 + i] = make_float4(__uint_as_float(v1[4 * i]), __uint_as_float(v1[4 * i + 1]),
                                                 __uint_as_float(v1[4 * i + 2]), __uint_as_float(v1[4 * i + 3]));
                    }
                }
                __syncwarp();
                // Each lane stores `vec` adjacent pixels of one map, so one instruction covers `vec` maps:
                // per-warp store throughput is bounded by instructions in flight, not bytes (measured
                // ~2.7 B/clk per warp with 4-byte lanes), hence the widest unit the alignment allows.
                const int vec = a.vec;                          // 1, 2 or 4 (W, Q, P*Q multiples of vec)
                const int lanes_per_row = 32 >> a.vec_shift;
                const int row_sub = lane >> (5 - a.vec_shift), pg = lane & (lanes_per_row - 1);
                int n, p, q;                                    // this lane's first pixel of the block
                const bool ok = output_pixel<PATCH>(a, ii.geom, b * 32 + pg * vec, n, p, q);
                float* o = a.y;
                if (ok) o = a.y + (((size_t)n * a.K + nb * a.n_tile + quarter * rpq + row_sub) * a.P + p) * a.Q + q;
                if (ok) {
                    const int kmax = min(rpq, a.K - nb * a.n_tile - quarter * rpq);   // maps of this quarter that exist
                    const float* src = tile + row_sub * kXposePitch + pg * vec;
                    if (vec == 4) {
#pragma unroll 4
                        for (int r = 0; r < 32; r += 4, o += 4 * plane, src += 4 * kXposePitch)
                            if (r + row_sub < kmax) {
                                float4 t = *reinterpret_cast<const float4*>(src);
                                if (stacked) {
                                    const float4 u = *reinterpret_cast<const float4*>(src + 16 * kXposePitch);
                                    t.x += u.x; t.y += u.y; t.z += u.z; t.w += u.w;
                                }
                                if (add) { atomicAdd(o, t.x); atomicAdd(o + 1, t.y); atomicAdd(o + 2, t.z); atomicAdd(o + 3, t.w); }
                                else *reinterpret_cast<float4*>(o) = t;
                            }
                    } else if (vec == 2) {
#pragma unroll 8
                        for (int r = 0; r < 32; r += 2, o += 2 * plane, src += 2 * kXposePitch)
                            if (r + row_sub < kmax) {
                                float2 t = *reinterpret_cast<const float2*>(src);
                                if (stacked) {
                                    const float2 u = *reinterpret_cast<const float2*>(src + 16 * kXposePitch);
                                    t.x += u.x; t.y += u.y;
                                }
                                if (add) { atomicAdd(o, t.x); atomicAdd(o + 1, t.y); }
                                else *reinterpret_cast<float2*>(o) = t;
                            }
                    } else {
#pragma unroll 8
                        for (int r = 0; r < 32; ++r, o += plane, src += kXposePitch)
                            if (r < kmax) {
                                const float t = stacked ? src[0] + src[16 * kXposePitch] : src[0];
                                if (add) atomicAdd(o, t); else *o = t;
                            }
                    }
                }
            };
            if (CLUSTER) {
                const uint32_t rank = cluster_ctarank(), peer = rank ^ 1u;
                // rows and barriers belong to a (lane quarter, block) pair; with the helper warps a quarter is
                // drained by three warps, block b going to warp (b / 2) mod 3 of the quarter on both sides
                float* my_rows = xchg + (size_t)quarter * a.xchg_slots * kXchgBlockFloats;
                uint64_t* my_bars = xbar + quarter * a.xchg_slots;
                const int nshare = a.helpers ? 3 : 1;
                uint32_t v0[16], v1[16], vx[1];
                vx[0] = 0u;
                // the blocks the peer stores: this block's partial sums go into the peer's shared memory as
                // [4-column group][lane][16 bytes], so that one store instruction of the warp writes 512 contiguous
                // bytes over the cluster network (a row per lane, i.e. 16-byte pieces 144 bytes apart, took 2150 cycles
                // per 32-pixel block, this layout 1290)
                const long long t_x0 = clock_now();
                long long t_xwait = 0;
                for (int b = (int)peer; b < blocks; b += 2) {
                    if ((b >> 1) % nshare != share) continue;
                    tmem_ld16(lane_base + (uint32_t)(b * 32), v0);
                    tmem_ld16(lane_base + (uint32_t)(b * 32 + 16), v1);
                    tmem_ld_wait();
                    const int slot = b >> 1;
                    const uint32_t dst = map_to_cta(smem_u32(my_rows + (size_t)slot * kXchgBlockFloats + lane * 4), peer);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        st_cluster_v4(dst + 512u * i, __uint_as_float(v0[4 * i]), __uint_as_float(v0[4 * i + 1]),
                                      __uint_as_float(v0[4 * i + 2]), __uint_as_float(v0[4 * i + 3]));
                        st_cluster_v4(dst + 2048u + 512u * i, __uint_as_float(v1[4 * i]), __uint_as_float(v1[4 * i + 1]),
                                      __uint_as_float(v1[4 * i + 2]), __uint_as_float(v1[4 * i + 3]));
                    }
                }
                // The arrivals come after the stores of all blocks (measured: the same time as arriving block by
                // block, ~1290 cycles per block either way: the remote stores themselves, ~150 cycles per 512-byte
                // instruction, are the cost; one arrival per warp behind a cluster-scope fence measured slower).
                for (int b = (int)peer; b < blocks; b += 2) {
                    if ((b >> 1) % nshare != share) continue;
                    mbar_arrive_remote(map_to_cta(smem_u32(&my_bars[b >> 1]), peer));
                }
                const long long t_x1 = clock_now();
                // this block's own blocks: accumulators + the peer's partial sums, then the ordinary write-back
                for (int b = (int)rank; b < blocks; b += 2) {
                    if ((b >> 1) % nshare != share) continue;
                    tmem_ld16(lane_base + (uint32_t)(b * 32), v0);
                    tmem_ld16(lane_base + (uint32_t)(b * 32 + 16), v1);
                    tmem_ld_wait();
                    const int slot = b >> 1;
                    const long long t_w0 = clock_now();
                    alive = __all_sync(0xffffffffu, mbar_wait_bounded_cluster(&my_bars[slot], 0u, abort_flag, a.max_polls));
                    t_xwait += clock_now() - t_w0;
                    if (!alive) break;
                    const float4* row = reinterpret_cast<const float4*>(my_rows + (size_t)slot * kXchgBlockFloats) + lane;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float4 t = row[32 * i], u = row[128 + 32 * i];
                        v0[4 * i] = __float_as_uint(__uint_as_float(v0[4 * i]) + t.x);
                        v0[4 * i + 1] = __float_as_uint(__uint_as_float(v0[4 * i + 1]) + t.y);
                        v0[4 * i + 2] = __float_as_uint(__uint_as_float(v0[4 * i + 2]) + t.z);
                        v0[4 * i + 3] = __float_as_uint(__uint_as_float(v0[4 * i + 3]) + t.w);
                        v1[4 * i] = __float_as_uint(__uint_as_float(v1[4 * i]) + u.x);
                        v1[4 * i + 1] = __float_as_uint(__uint_as_float(v1[4 * i + 1]) + u.y);
                        v1[4 * i + 2] = __float_as_uint(__uint_as_float(v1[4 * i + 2]) + u.z);
                        v1[4 * i + 3] = __float_as_uint(__uint_as_float(v1[4 * i + 3]) + u.w);
                    }
                    store_block(v0, v1, vx, b);
                }
                if (!alive) break;
                if (kDiag && blockIdx.x == 0 && warp == 4 && lane == 0) {     // cycles: sending, waiting for the peer, whole exchange
                    a.status[13] = (unsigned)(t_x1 - t_x0);
                    a.status[14] = (unsigned)t_xwait;
                    a.status[15] = (unsigned)(clock_now() - t_x0);
                }
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0 && !helper) mbar_arrive(&acc_empty[buf]);
                continue;
            }
            uint32_t va0[16], va1[16], vb0[16], vb1[16], vax[1], vbx[1];
            if (M64 && a.vec >= 2 && !add) {
                // At most 64 filters (a quarter holds 16 maps): two 32-pixel blocks share the tile and one pass over it,
                // each half of the warp stores one of them.  A block at a time the warps, not the MMAs or the memory,
                // set the pace of short contractions (900 cycles per block, most of them the latency of the steps).
                const int half = lane >> 4, lanes_per_row = 32 >> a.vec_shift;
                const int row_sub = (lane & 15) >> (5 - a.vec_shift), pg = lane & (lanes_per_row - 1);
                const int pairs = (blocks + 1) / 2, p_step = split ? 3 : 1;
                const int kmax = min(16, a.K - nb * a.n_tile - quarter * 16);      // maps of this quarter that exist
                auto load_pair = [&](int bp) {
                    tmem_ld16(lane_base + (uint32_t)(bp * 64), va0);
                    tmem_ld16(lane_base + (uint32_t)(bp * 64 + 16), va1);
                    if (2 * bp + 1 < blocks) {
                        tmem_ld16(lane_base + (uint32_t)(bp * 64 + 32), vb0);
                        tmem_ld16(lane_base + (uint32_t)(bp * 64 + 48), vb1);
                    }
                };
                int bp = split ? share : 0;
                if (bp < pairs) load_pair(bp);
                while (bp < pairs) {
                    tmem_ld_wait();
                    __syncwarp();                               // the previous pair has been read out
                    if (lane < 16) {
                        float4* ra = reinterpret_cast<float4*>(tile + lane * kXposePitch);
                        float4* rb = reinterpret_cast<float4*>(tile + (lane + 16) * kXposePitch);
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            ra[i] = make_float4(__uint_as_float(va0[4 * i]), __uint_as_float(va0[4 * i + 1]), __uint_as_float(va0[4 * i + 2]), __uint_as_float(va0[4 * i + 3]));
                            ra[4 + i] = make_float4(__uint_as_float(va1[4 * i]), __uint_as_float(va1[4 * i + 1]), __uint_as_float(va1[4 * i + 2]), __uint_as_float(va1[4 * i + 3]));
                        }
                        if (2 * bp + 1 < blocks) {
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                rb[i] = make_float4(__uint_as_float(vb0[4 * i]), __uint_as_float(vb0[4 * i + 1]), __uint_as_float(vb0[4 * i + 2]), __uint_as_float(vb0[4 * i + 3]));
                                rb[4 + i] = make_float4(__uint_as_float(vb1[4 * i]), __uint_as_float(vb1[4 * i + 1]), __uint_as_float(vb1[4 * i + 2]), __uint_as_float(vb1[4 * i + 3]));
                            }
                        }
                    }
                    __syncwarp();
                    const int b = 2 * bp + half;
                    bp += p_step;
                    if (bp < pairs) load_pair(bp);
                    int n, p, q;                                // this lane's first pixel of its block
                    if (b < blocks && output_pixel<PATCH>(a, ii.geom, b * 32 + pg * a.vec, n, p, q)) {
                        float* o = a.y + (((size_t)n * a.K + nb * a.n_tile + quarter * 16 + row_sub) * a.P + p) * a.Q + q;
                        const float* src = tile + (16 * half + row_sub) * kXposePitch + pg * a.vec;
                        if (a.vec == 4) {
#pragma unroll
                            for (int r = 0; r < 16; r += 2, o += 2 * plane, src += 2 * kXposePitch)
                                if (r + row_sub < kmax) *reinterpret_cast<float4*>(o) = *reinterpret_cast<const float4*>(src);
                        } else {
#pragma unroll
                            for (int r = 0; r < 16; ++r, o += plane, src += kXposePitch)
                                if (r < kmax) *reinterpret_cast<float2*>(o) = *reinterpret_cast<const float2*>(src);
                        }
                    }
                }
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0 && !helper) mbar_arrive(&acc_empty[buf]);
                continue;
            }
            if (STACK && (!VIRT || (a.vec >= 2 && !add))) {
                // Stacked taps, two blocks to a pass as well.  The two rows of a map are added in registers: lanes l and l + 16 hold
                // them, exchange a half of their columns (the right-hand taps' one column on) and each keep one half of the sums, so
                // the tile is written and read once per map (64 x 128 x 32 x 32, 64 of 3 x 3: 33.0 -> 31.0 us; single pixels, 27 x 208 x
                // 35 x 35: 35.0 -> 28.3.  On virtual images single pixels stay a block at a time: 48 x 384 x 46 x 31, 18 of 3 x 3 84 us, 98
                // with two, as their producers, which load single pixels, too, then wait longer).
                const int pairs = (blocks + 1) / 2, p_step = split ? 3 : 1;
                const int kmax = min(16, a.K - nb * 64 - quarter * 16);            // maps of this quarter that exist
                const bool up = lane >= 16;
                auto fill = [&](int h) {                // the block in va0, va1, vax -> half h of the tile
                    float4* row = reinterpret_cast<float4*>(tile + (lane & 15) * kStackPitch + (up ? 16 : 0) + 32 * h);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        float sum[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int i = 4 * q + e;
                            const uint32_t give = up ? (i < 15 ? va0[(i + 1) & 15] : va1[0]) : va1[i];
                            const uint32_t keep = up ? (i < 15 ? va1[(i + 1) & 15] : vax[0]) : va0[i];
                            sum[e] = __uint_as_float(keep) + __uint_as_float(__shfl_xor_sync(0xffffffffu, give, 16));
                        }
                        row[q] = make_float4(sum[0], sum[1], sum[2], sum[3]);
                    }
                };
                int bp = split ? share : 0;
                if (bp < pairs) load_block(va0, va1, vax, 2 * bp);
                while (bp < pairs) {
                    const int b0 = 2 * bp;
                    tmem_ld_wait();
                    __syncwarp();                               // the previous pair has been read out
                    fill(0);
                    if (b0 + 1 < blocks) {
                        load_block(va0, va1, vax, b0 + 1);
                        tmem_ld_wait();
                        fill(1);
                    }
                    __syncwarp();
                    bp += p_step;
                    if (bp < pairs) load_block(va0, va1, vax, 2 * bp);
                    int n, p, q;                                // this lane's first pixel
                    if (a.vec == 1 || add) {
                        // single pixels: 32 of one map to an instruction
                        for (int h = 0; h < 2; ++h)
                            if (b0 + h < blocks && output_pixel<PATCH>(a, ii.geom, (b0 + h) * 32 + lane, n, p, q)) {
                                float* o = a.y + (((size_t)n * a.K + nb * 64 + quarter * 16) * a.P + p) * a.Q + q;
                                const float* src = tile + 32 * h + lane;
#pragma unroll 8
                                for (int r = 0; r < kmax; ++r, o += plane, src += kStackPitch) { if (add) atomicAdd(o, *src); else *o = *src; }
                            }
                    } else {
                        // pairs or quads: each half of the warp stores one of the blocks
                        const int half = lane >> 4, lanes_per_row = 32 >> a.vec_shift;
                        const int row_sub = (lane & 15) >> (5 - a.vec_shift), pg = lane & (lanes_per_row - 1);
                        if (b0 + half < blocks && output_pixel<PATCH>(a, ii.geom, (b0 + half) * 32 + pg * a.vec, n, p, q)) {
                            float* o = a.y + (((size_t)n * a.K + nb * 64 + quarter * 16 + row_sub) * a.P + p) * a.Q + q;
                            const float* src = tile + row_sub * kStackPitch + 32 * half + pg * a.vec;
                            if (a.vec == 4) {
#pragma unroll
                                for (int r = 0; r < 16; r += 2, o += 2 * plane, src += 2 * kStackPitch)
                                    if (r + row_sub < kmax) *reinterpret_cast<float4*>(o) = *reinterpret_cast<const float4*>(src);
                            } else {
#pragma unroll
                                for (int r = 0; r < 16; ++r, o += plane, src += kStackPitch)
                                    if (r < kmax) *reinterpret_cast<float2*>(o) = *reinterpret_cast<const float2*>(src);
                            }
                        }
                    }
                }
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0 && !helper) mbar_arrive(&acc_empty[buf]);
                if (kDiag && blockIdx.x == 0 && warp == 4 && lane == 0) a.status[11] += (unsigned)(clock_now() - t_busy0);   // drained one item
                continue;
            }
            const int b_step = split ? 3 : 1;
            int b = split ? share : 0;
            if (b < blocks) load_block(va0, va1, vax, b);
            long long t_ld = 0;       // (diagnostics build: cycles spent waiting for tensor-memory loads)
            while (b < blocks) {
                long long t0 = clock_now();
                tmem_ld_wait();
                t_ld += clock_now() - t0;
                if (b + b_step < blocks) load_block(vb0, vb1, vbx, b + b_step);
                store_block(va0, va1, vax, b);
                if ((b += b_step) >= blocks) break;
                t0 = clock_now();
                tmem_ld_wait();
                t_ld += clock_now() - t0;
                if (b + b_step < blocks) load_block(va0, va1, vax, b + b_step);
                store_block(vb0, vb1, vbx, b);
                b += b_step;
            }
            if (kDiag && blockIdx.x == 0 && warp == 4 && lane == 0) a.status[12] += (unsigned)t_ld;
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0 && !helper) mbar_arrive(&acc_empty[buf]);
            if (kDiag && blockIdx.x == 0 && warp == 4 && lane == 0) a.status[11] += (unsigned)(clock_now() - t_busy0);   // drained one item
        }
    }
    }

    tc_fence_before_sync();
    __syncthreads();
    // (a block must not exit while its peer may still write into its shared memory or arrive on its barriers)
    if (CLUSTER) cluster_sync_all();
    if (warp == 1) tmem_dealloc(tmem, a.tmem_cols);
    if (tid == 0 && *abort_flag) atomicExch(a.status, 1u);
    if (kDiag && tid == 0 && blockIdx.x == 0) a.status[8] = (unsigned)(wall_ns() - *t_entry);   // ns from kernel entry to the block's end
}

}  // namespace
}  // namespace conv2d_b200
