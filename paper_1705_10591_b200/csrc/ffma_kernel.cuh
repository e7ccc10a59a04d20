// fp32 general-case kernel (Section 4, Algorithm 2) and its launchers, as templates.  Included by the translation units
// general_ffma_r*.cu, one per filter size, so that the instances compile in parallel; general_ffma.cu dispatches.
//
// Kept from the paper's design:
//   * a thread block covers some filters x some outputs over all C channels (Section 4.1);
//   * channels are staged CB at a time in shared memory: the image rows with their right/bottom halo as they lie in
//     memory, the filters transposed so that adjacent filters are adjacent words (Section 4.2, Fig. 6);
//   * a thread accumulates kThrK filters x TQ horizontally adjacent outputs (a segment) in registers, keeps one input
//     row segment of TQ+S-1 pixels in registers and reuses it for the S horizontal taps (Section 4.2);
//   * the next channel block is fetched while the current one is multiplied (Algorithm 2's prefetch), by asynchronous
//     copies into a second buffer, so no thread holds prefetched data in registers.
// Changed for B200: packed two-filter FMAs, 8 x TQ register tile, and the split of the work.  A block is `groups` filter
// groups x `segs` segments, where the segments are numbered through the rows of the whole batch: no block ends at the
// edge of a tile or of an image, and a block's rows with their halo are a run of image rows.  What is lost is the end of
// a row that fills no segment and the filters that fill no group of 8.
// Fixed tiles of 32 x 8 outputs (and five other shapes) x 64 filters were 53 % full on 25 x 33 maps of 112 filters, their
// filter reads had two-way bank conflicts (27 of 60 million wavefronts), and a 4-byte copy with three divisions for every
// element of a row of odd width took a quarter of the issue slots.  Us, before -> now:
//   32 x 96 x 27 x 35, 112 filters of 3 x 3: 282 -> 132 (38 of 74 TFLOP/s)   32 x 64 x 56 x 56, 64 of 3 x 3: 219 -> 159
//   16 x 128 x 32 x 32, 128 of 7 x 7: 764 -> 414        64 x 128 x 32 x 32, 128 of 3 x 3: 430 -> 384, of 1 x 1 72 -> 70
//   20 x 176 x 31 x 31, 32 of 7 x 7: 1077 -> 350        1 x 149 x 20 x 20, 80 of 3 x 3: 174 -> 71
// What bounds it now: issue slots (0.6 other instructions per packed FMA) and, on small problems, the SMs' work per round.
#pragma once
#include "common.cuh"
#include "fastdiv.cuh"

#include <cmath>

namespace conv2d_b200 {
namespace {

constexpr int kThrK = 8;              // filters per thread (F_T)
constexpr int kMaxGroups = 8;         // filter groups of a block
constexpr int kMaxThreads = 256;

// Asynchronous global -> shared copy of BYTES (4 or 16); only the first src_bytes are read, the rest is zero.
template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst_smem, const void* src, int src_bytes)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst_smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(d), "l"(src), "n"(BYTES), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

struct FfmaArgs {
    const float* x;
    const float* w;
    float* y;
    int N, C, H, W, K, P, Q;
    long long x_floats;               // N * C * H * W
    int groups, segs;                 // of a block
    int sps, strips;                  // segments of a row in a column strip (wide maps are cut into strips), strips
    int total_segs;                   // N * P * sps: segments of a strip
    int rows, pitch;                  // staged image rows (at most) and floats per row
    int vec_st;                       // widest store unit that the output rows allow (floats)
    FastDiv div_groups, div_sps, div_P, div_H;
};

// ALIGNED: W and the strips' first columns are multiples of four, so a staged row starts on 16 bytes wherever it lies.
// Otherwise a row is copied from the 16-byte boundary before it and starts 0 .. 3 floats into its place.
template <int R, int S, int CB, int TQ, bool ALIGNED>
__global__ void __launch_bounds__(kMaxThreads, 2)
general_ffma_kernel(const FfmaArgs a)
{
    constexpr int RS = R * S, kRaw = CB * RS;
    constexpr int VR = !ALIGNED ? 1 : (TQ % 4 == 0 ? 4 : (TQ % 2 == 0 ? 2 : 1));      // floats per read of a row segment (its alignment)
    constexpr int NV = (TQ + S - 1 + VR - 1) / VR;
    extern __shared__ __align__(16) float smem[];
    const int fpitch = a.groups * kThrK + 4;                          // filters of a tap, padded: transposed stores spread over banks
    const int img_floats = CB * a.rows * a.pitch, flt_floats = kRaw * fpitch;
    float* const img_smem = smem;                                     // [2][CB][rows][pitch]
    float* const flt_smem = smem + 2 * img_floats;                    // [2][CB][RS][fpitch]
    long long* const row_src = reinterpret_cast<long long*>(flt_smem + 2 * flt_floats);      // [rows]

    const int tid = threadIdx.x, nthr = blockDim.x;
    int tx;                                                           // filter group: adjacent threads, adjacent filter units
    const int ty = a.div_groups.divmod(tid, tx);
    const int strip = blockIdx.x % a.strips;
    const int seg0 = (blockIdx.x / a.strips) * a.segs;
    const int k0 = blockIdx.y * a.groups * kThrK;
    const int col0 = strip * a.sps * TQ;
    const int width = min(a.sps * TQ + S - 1, a.W - col0);            // columns of a staged row

    // segment -> (image, output row, column); the first staged image row is that of the block's first segment
    auto decode = [&](int seg, int& n, int& p, int& sq) {
        const int sr = a.div_sps.divmod(seg, sq);
        n = a.div_P.divmod(sr, p);
    };
    int n, p, sq;
    decode(seg0, n, p, sq);
    const int row0 = n * a.H + p;                                     // image rows numbered through the batch
    decode(min(seg0 + a.segs, a.total_segs) - 1, n, p, sq);
    const int rows_used = n * a.H + p - row0 + R;
    const bool live = ty < a.segs && seg0 + ty < a.total_segs;        // (threads past the block's end repeat its last segment)
    decode(min(seg0 + min(ty, a.segs - 1), a.total_segs - 1), n, p, sq);
    const int row_off = (n * a.H + p - row0) * a.pitch + sq * TQ;
    const unsigned plane = (unsigned)(a.H * a.W);
    // (unaligned rows: only the value modulo four of a row's place in x matters to its reader)
    const unsigned row_place = ((unsigned)n * (unsigned)a.C) * plane + (unsigned)p * (unsigned)a.W + (unsigned)col0;

    // Source of every staged row (channel 0), in floats from x: looked up by the copies.
    for (int row = tid; row < rows_used; row += nthr) {
        int h;
        const int in_n = a.div_H.divmod(row0 + row, h);
        row_src[row] = (long long)in_n * a.C * plane + (long long)h * a.W + col0;
    }
    __syncthreads();

    // The copies of a channel block.  Image rows with their halo: 16-byte pieces tid, tid + nthr, ... of all rows, the
    // position of the next piece by addition.  Filters: transposed on the way, a warp takes a filter's contiguous run
    // (so that an element costs little more than its copy); filter 8g + j of the block lies at 4g + j for j < 4 and at
    // 4 * groups + 4g + j - 4 otherwise, so that the 128-bit reads of adjacent groups are adjacent.  Only channels that
    // exist are copied and multiplied; filters that do not exist hold whatever was there and are not stored.
    const int pieces = (width + (ALIGNED ? 0 : 3) + 3) / 4;
    const int step_row = nthr / pieces, step_v = nthr - step_row * pieces;
    const int first_row = tid / pieces, first_v = tid - first_row * pieces;
    auto issue = [&](int c0, int buf) {
        const int channels = min(CB, a.C - c0);
        float* const img = img_smem + buf * img_floats;
        int row = first_row, v = first_v, cc = 0;
        while (row >= rows_used) { row -= rows_used; ++cc; }
#pragma unroll 1
        while (cc < channels) {
            long long src = row_src[row] + (long long)(c0 + cc) * plane;
            if (!ALIGNED) src &= ~3LL;
            src += 4 * v;
            const long long left = a.x_floats - src;                  // (the last piece of the tensor may be short)
            if (left > 0) cp_async<16>(img + (cc * a.rows + row) * a.pitch + 4 * v, a.x + src, left >= 4 ? 16 : (int)left * 4);
            v += step_v;
            row += step_row;
            if (v >= pieces) { v -= pieces; ++row; }
            while (row >= rows_used) { row -= rows_used; ++cc; }
        }
        float* const flt = flt_smem + buf * flt_floats;
        const int exist = channels * RS;                              // floats of a filter's run that exist
        constexpr int kLanes = kRaw >= 32 ? 32 : kRaw;                // threads per filter
        const int e0 = tid % kLanes;
#pragma unroll 1
        for (int kk = tid / kLanes; kk < a.groups * kThrK && k0 + kk < a.K; kk += nthr / kLanes) {
            const float* src = a.w + (k0 + kk) * a.C * RS + c0 * RS + e0;
            float* dst = flt + (kk & 4 ? a.groups * 4 : 0) + (kk >> 3) * 4 + (kk & 3) + e0 * fpitch;
#pragma unroll
            for (int e = 0; e < kRaw; e += kLanes, dst += kLanes * fpitch)
                if (e + e0 < exist) cp_async<4>(dst, src + e, 4);
        }
        cp_async_commit();
    };

    // Accumulators as (filter 2i, filter 2i+1) pairs: B200 reaches its fp32 FMA peak only with the two-wide
    // packed instruction (fma.rn.f32x2); the pixel is duplicated, the two filter taps are adjacent.
    float2 acc[kThrK / 2][TQ];
#pragma unroll
    for (int i = 0; i < kThrK / 2; ++i)
#pragma unroll
        for (int j = 0; j < TQ; ++j) acc[i][j] = make_float2(0.f, 0.f);

    issue(0, 0);
    for (int c0 = 0, it = 0; c0 < a.C; c0 += CB, ++it) {
        const int buf = it & 1;
        cp_async_wait_all();
        __syncthreads();                 // this block has landed; everyone is done with the previous one
        if (c0 + CB < a.C) issue(c0 + CB, buf ^ 1);      // the next block arrives under the multiplications below
        const int channels = min(CB, a.C - c0);
        const float* irow = img_smem + buf * img_floats + row_off;
        const float* ftap = flt_smem + buf * flt_floats + tx * 4;
        unsigned place = row_place + (unsigned)c0 * plane;
#pragma unroll(RS == 1 ? 4 : 1)
        for (int cc = 0; cc < channels; ++cc, irow += a.rows * a.pitch, place += plane) {
            const float* srow = irow;
#pragma unroll
            for (int r = 0; r < R; ++r, srow += a.pitch) {
                float2 px[VR * NV];                                   // (x, x)
                const float* at = ALIGNED ? srow : srow + ((place + r * a.W) & 3u);
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    if constexpr (VR == 4) {
                        const float4 t = reinterpret_cast<const float4*>(at)[v];
                        px[4 * v + 0] = make_float2(t.x, t.x); px[4 * v + 1] = make_float2(t.y, t.y);
                        px[4 * v + 2] = make_float2(t.z, t.z); px[4 * v + 3] = make_float2(t.w, t.w);
                    } else if constexpr (VR == 2) {
                        const float2 t = reinterpret_cast<const float2*>(at)[v];
                        px[2 * v + 0] = make_float2(t.x, t.x); px[2 * v + 1] = make_float2(t.y, t.y);
                    } else {
                        const float t = at[v];
                        px[v] = make_float2(t, t);
                    }
                }
#pragma unroll
                for (int s = 0; s < S; ++s, ftap += fpitch) {
                    const float4 lo = *reinterpret_cast<const float4*>(ftap);
                    const float4 hi = *reinterpret_cast<const float4*>(ftap + a.groups * 4);
                    const float2 flt[kThrK / 2] = {make_float2(lo.x, lo.y), make_float2(lo.z, lo.w),
                                                   make_float2(hi.x, hi.y), make_float2(hi.z, hi.w)};
#pragma unroll
                    for (int i = 0; i < kThrK / 2; ++i)
#pragma unroll
                        for (int j = 0; j < TQ; ++j) acc[i][j] = __ffma2_rn(px[s + j], flt[i], acc[i][j]);
                }
            }
        }
    }

    // ---- write the register tile ----
    const int q = col0 + sq * TQ;
    if (!live || q >= a.Q) return;
#pragma unroll
    for (int i = 0; i < kThrK; ++i) {
        const int k = k0 + tx * kThrK + i;
        if (k >= a.K) break;
        float* o = a.y + (((size_t)n * a.K + k) * a.P + p) * a.Q + q;
        float row[TQ];
#pragma unroll
        for (int j = 0; j < TQ; ++j) row[j] = (i & 1) ? acc[i / 2][j].y : acc[i / 2][j].x;
        if (VR == 4 && a.vec_st == 4 && q + TQ <= a.Q) {
#pragma unroll
            for (int v = 0; v < TQ / 4; ++v)
                *reinterpret_cast<float4*>(o + 4 * v) = make_float4(row[4 * v], row[4 * v + 1], row[4 * v + 2], row[4 * v + 3]);
        } else if (VR >= 2 && a.vec_st >= 2 && q + TQ <= a.Q) {
#pragma unroll
            for (int v = 0; v < TQ / 2; ++v)
                *reinterpret_cast<float2*>(o + 2 * v) = make_float2(row[2 * v], row[2 * v + 1]);
        } else {
#pragma unroll
            for (int j = 0; j < TQ; ++j)
                if (q + j < a.Q) o[j] = row[j];
        }
    }
}

// How a shape is split for segments of TQ outputs.
struct FfmaSplit {
    int groups = 0, kblocks = 0, segs = 0, sps = 0, strips = 0, threads = 0, rows = 0, pitch = 0;
    long long seg_blocks = 0;
    size_t smem = 0;
    bool x4 = false;
    double cost = 0;                  // estimated cycles; 0: no split
};

// Estimated cycles of a split for 1 x 1 filters.  Their contraction is short, so the latency of a block's stages and its
// stores count as much as its multiplications, and smaller blocks pay, down to a few threads that multiply among many that
// copy.  Fitted to 1300 random layers in all their splits: 5 % of them were slower by 4 % and more than in fixed tiles of
// 32 x 8 outputs x 64 filters with the estimate of the other filter sizes, 1.5 % with this one, all together 9 % faster
// (64 x 128 x 32 x 32, 128 filters 76 -> 70 us; 12 x 16 x 62 x 62, 384 filters 89 -> 49; 36 x 480 x 11 x 11, 7 filters 134 -> 61).
template <int CB, int TQ>
double pointwise_split_cost(const Shape& sh, const FfmaSplit& f, int resident, int sms)
{
    const double warps = f.threads / 32, stages = (sh.C + CB - 1) / CB, share = (double)f.seg_blocks * f.kblocks / sms;
    const int width = f.sps * TQ < sh.W ? f.sps * TQ : sh.W, threads = f.threads;
    const double pieces = stages * (double)(CB * f.rows * ((width + (f.x4 ? 0 : 3) + 3) / 4)) / threads;    // copies of a thread
    const double filters = stages * (double)(CB * f.groups * kThrK) / threads;
    const int unit = !f.x4 || TQ % 2 ? 1 : (TQ % 4 ? 2 : 4);                                               // floats of a read
    const int store = sh.Q % 4 == 0 && unit == 4 ? 4 : (sh.Q % 2 == 0 && unit >= 2 ? 2 : 1);
    const double issue = sh.C * (0.373 * kThrK * TQ + 1.34 + 0.233 * TQ / unit) + 237.0 * stages + 26.5 * pieces + 24.1 * filters
                       + 27.8 * kThrK * TQ / store + 69.7;                                                 // slots of a warp
    const double per_sm = ceil(share), conc = per_sm < resident ? per_sm : resident, beside = conc * warps / 4.0;
    const double alone = issue * (warps > 4 ? warps / 4.0 : 1.0) * 2.26 + 142.0 * stages + 19.1 * (pieces + filters) + 3650.0;
    double rounds = 1.0, count = per_sm;
    if (per_sm > resident) {
        rounds = share / conc + 6.75;
        count = (per_sm > share + 0.5 * conc ? per_sm : share + 0.5 * conc) + 2.7 * conc;
    }
    const double latency = rounds * alone, slots = count * warps / 4.0 * issue * (1.0 + 3.86 / beside);
    return latency > slots ? latency + 0.3 * slots : slots + 0.3 * latency;
}

template <int R, int S, int CB, int TQ>
FfmaSplit split_ffma(const Shape& sh)
{
    FfmaSplit best;
    const int sms = sm_count();
    const int row_segs = (sh.Q + TQ - 1) / TQ;
    // Column strips keep the staged rows short on wide maps (a block of 32 segments then covers several rows and the
    // R - 1 halo rows are shared): at most 8 segments a strip, 12 where one strip holds the whole row.
    FfmaSplit f;
    f.x4 = sh.W % 4 == 0;
    f.strips = row_segs <= 12 ? 1 : (row_segs + 7) / 8;
    f.sps = (row_segs + f.strips - 1) / f.strips;
    if (f.strips > 1) {
        while (f.x4 && f.sps * TQ % 4 != 0) ++f.sps;                 // 16-byte copies start at the strip's first column
        f.strips = (row_segs + f.sps - 1) / f.sps;
    }
    f.pitch = (f.sps * TQ + S - 1 + 3 + 3 + 3) / 4 * 4;              // room for whole 128-bit reads past the halo, or for the place in a 16-byte word
    const long long total = (long long)sh.N * sh.P * f.sps;
    if (total > 0x7fffffffLL - 4096 || (long long)sh.N * sh.H > 0x7fffffffLL - 65536) return best;
    const int kgroups = (sh.K + kThrK - 1) / kThrK;
    const int kb_min = (kgroups + kMaxGroups - 1) / kMaxGroups;
    const int kb_candidates[3] = {kb_min, kb_min * 2, kb_min * 4};
    for (int kb : kb_candidates) {
        if (kb > kgroups || (R == 1 && kb > 2 * kb_min)) continue;
        f.groups = (kgroups + kb - 1) / kb;
        f.kblocks = (kgroups + f.groups - 1) / f.groups;
        if (f.kblocks > 65535) continue;
        // (warp w of every block sits on scheduler w % 4: other counts leave two schedulers with half the work, 64 x 128 x
        // 32 x 32, 128 filters of 3 x 3: 381 us with 4 warps, 407 with 8, 441 with 6)
        // (1 x 1 filters, few of them: also a half and a quarter of the segments, the other threads only copy)
        for (int choice = 0; choice < (R == 1 && f.groups <= 2 ? 5 : 3); ++choice) {
            const int warps = choice < 3 ? 2 << choice : 4;
            f.threads = 32 * warps;
            f.segs = f.threads / f.groups >> (choice < 3 ? 0 : choice - 2);
            // rows that the segments of a block can touch, and the halo rows of every image among them (many small
            // images with large filters: fewer segments than threads, until their rows fit)
            for (;; f.segs /= 2) {
                const int out_rows = (f.segs + f.sps - 2) / f.sps + 1;
                const int crossings = (out_rows - 1 + sh.P - 1) / sh.P;
                const long long rows = out_rows + (long long)(R - 1) * (1 + crossings), all = (long long)sh.N * sh.H;
                f.rows = (int)(rows < all ? rows : all);
                f.smem = 2 * sizeof(float) * CB * ((size_t)f.rows * f.pitch + (size_t)R * S * (f.groups * kThrK + 4)) + 8 * (size_t)f.rows;
                if (f.smem <= 200 * 1024 || f.segs <= 1) break;
            }
            if (f.smem > 200 * 1024) continue;
            f.seg_blocks = (total + f.segs - 1) / f.segs * f.strips;
            const long long blocks = f.seg_blocks * f.kblocks;
            const int by_regs = 512 / f.threads, by_smem = (int)(220 * 1024 / (f.smem + 1024));
            const int res = by_regs < by_smem ? by_regs : by_smem;
            if constexpr (R == 1) {
                const double t = pointwise_split_cost<CB, TQ>(sh, f, res, sms);
                if (best.cost == 0 || t < best.cost) { best = f; best.cost = t; }
                continue;
            }
            // one warp's work on its scheduler, with its share of the copies of a channel block (an element of the image
            // rows or of the filters costs about 16 issue slots per 32 threads) and of the barrier at its end
            const double copies = CB * ((double)f.rows * f.pitch / 4 * 16.0 + (double)R * S * f.groups * kThrK * 8.0) / f.threads;
            const double row_cycles = f.x4 ? TQ + S + 4.0 : 2.0 * (TQ + S) + 6.0;
            const double warp = (double)((sh.C + CB - 1) / CB) * (CB * (R * S * (TQ * 8.0 * 1.1 + 4) + R * row_cycles + 6) + copies + 100.0);
            const long long per_sm = (blocks + sms - 1) / sms;
            const double conc = (double)(per_sm < res ? per_sm : res);
            const double per_sched = conc * warps / 4.0;             // warps beside one another on a scheduler
            const double eff = per_sched <= 1 ? 0.6 : (per_sched < 2 ? 0.6 + 0.25 * (per_sched - 1) : (per_sched < 3 ? 0.85 + 0.1 * (per_sched - 2) : 0.95));
            double t;
            if (per_sm <= res) t = (double)((per_sm * warps + 3) / 4) * warp / eff;
            else t = ((double)blocks / sms + 0.5 * conc) * warps / 4.0 * warp / eff;
            t += 3000;
            if (best.cost == 0 || t < best.cost) { best = f; best.cost = t; }
        }
    }
    return best;
}

template <int R, int S, int CB, int TQ, bool ALIGNED>
conv2d_status_t launch_split(const float* x, const float* w, float* y, const Shape& sh, const FfmaSplit& f, cudaStream_t stream)
{
    auto kern = general_ffma_kernel<R, S, CB, TQ, ALIGNED>;
    static SmemLimit smem_done;
    if (f.smem > 48 * 1024 && raise_smem_limit(reinterpret_cast<const void*>(kern), f.smem, smem_done) != cudaSuccess)
        return CONV2D_ERR_CUDA;
    FfmaArgs a{};
    a.x = x; a.w = w; a.y = y;
    a.N = sh.N; a.C = sh.C; a.H = sh.H; a.W = sh.W; a.K = sh.K; a.P = sh.P; a.Q = sh.Q;
    a.x_floats = (long long)sh.N * sh.C * sh.H * sh.W;
    a.groups = f.groups; a.segs = f.segs; a.sps = f.sps; a.strips = f.strips;
    a.total_segs = sh.N * sh.P * f.sps;
    a.rows = f.rows; a.pitch = f.pitch;
    a.vec_st = (sh.Q % 4 == 0 && reinterpret_cast<uintptr_t>(y) % 16 == 0) ? 4
             : (sh.Q % 2 == 0 && reinterpret_cast<uintptr_t>(y) % 8 == 0) ? 2 : 1;
    a.div_groups = FastDiv(f.groups); a.div_sps = FastDiv(f.sps); a.div_P = FastDiv(sh.P); a.div_H = FastDiv(sh.H);
    if (launch_ordinary(kern, dim3((unsigned)f.seg_blocks, (unsigned)f.kblocks), dim3(f.threads), f.smem, stream, a) != cudaSuccess) return CONV2D_ERR_CUDA;
    count_launch();
    return CONV2D_OK;
}

// Length of the segments by estimated time (all of them give the same bits: an output's additions run over (c, r, s) in
// the same order): 8 has the widest reads and stores, 7 leaves less of 14-, 27- or 33-column maps idle, 6 less of 12 or 30.
template <int R, int S, int CB>
conv2d_status_t launch_instance(const float* x, const float* w, float* y, const Shape& sh, cudaStream_t stream)
{
    const FfmaSplit f6 = split_ffma<R, S, CB, 6>(sh), f8 = split_ffma<R, S, CB, 8>(sh);
    const FfmaSplit f7 = split_ffma<R, S, CB, 7>(sh);
    int tq = 8;
    double cost = f8.cost;
    const double clearly = R == 1 ? 1.0 : 0.98;
    auto consider = [&](int len, const FfmaSplit& f) { if (f.cost > 0 && (cost == 0 || f.cost < clearly * cost)) { cost = f.cost; tq = len; } };
    consider(6, f6); consider(7, f7);
    const int forced = env_int("CONV2D_B200_FFMA_SEGMENT", 0);
    if (forced >= 6 && forced <= 8) tq = forced;
    const FfmaSplit& f = tq == 6 ? f6 : (tq == 7 ? f7 : f8);
    if (f.cost == 0 || f.seg_blocks > 0x7fffffffLL) return CONV2D_ERR_UNSUPPORTED;
    const bool x4 = f.x4 && reinterpret_cast<uintptr_t>(x) % 16 == 0;
#define CONV2D_FFMA_LAUNCH(TQ) \
    return x4 ? launch_split<R, S, CB, TQ, true>(x, w, y, sh, f, stream) : launch_split<R, S, CB, TQ, false>(x, w, y, sh, f, stream)
    switch (tq) {
    case 6: CONV2D_FFMA_LAUNCH(6);
    case 7: CONV2D_FFMA_LAUNCH(7);
    default: CONV2D_FFMA_LAUNCH(8);
    }
#undef CONV2D_FFMA_LAUNCH
}

}  // namespace
}  // namespace conv2d_b200
