// One input channel, rows of any alignment: the kernel for most shapes (see launch_single_channel for the others).
//
// What bounds it: the output is nearly all of the traffic, and it leaves an SM at the rate the chip can take only in
// aligned 128-bit pieces (four strided 32-bit stores per thread, as rows that start anywhere otherwise need, reach a
// quarter of it).  So a thread's unit is an aligned quad of the OUTPUT TENSOR, not of the output row: for a row of map k
// that starts m floats past a 16-byte boundary, the thread's four outputs start at column 4t - m, and only the two
// quads at the ends of a row are written piecewise.  m depends on the row and, where P*Q is not a multiple of four, on
// the map: maps are then processed in 2 or 4 classes (k mod 2, k mod 4) of equal m.
// The image rows of a band lie in shared memory as four planes, one per column residue modulo four: a lane reads
// column 4t - m + i from plane (i - m) mod 4 at a position that grows by one per lane, so a window may start at any
// column without bank conflicts and without vector loads that want alignment.
// Arithmetic: M maps of four outputs are accumulated together (packed FMAs: the lanes of a pair are two maps, or two
// adjacent outputs where a class has one map only); row r of the window is read once for all of them, each tap as one
// broadcast.  The additions of an output run over (r, s) in order.  Up to M = 8 few registers (about 80) leave 24 warps
// on an SM, which hide the staging of a block behind the arithmetic of others.
// Measured: 3 x 1083 x 1917, 16 maps of 3 x 3: 205 us a call with strided 32-bit stores, 84 us here (5.0 TB/s).  Two quads per
// thread and tap read (half the broadcasts, 16 warps) were slower everywhere: 2049 x 2049, 32 maps of 5 x 5 165 -> 214.
#include "common.cuh"
#include "fastdiv.cuh"
#include "ptx.cuh"

namespace conv2d_b200 {
namespace {

constexpr int kMaxThreads = 256;
constexpr int kMaxQuads = 256;               // widest block: 1024 output columns
constexpr double kLatency = 2500;            // cycles of a block's set-up and staging that only other blocks can hide
constexpr double kBlockCycles = 900;         // cycles of a scheduler per block whatever its size

struct FlatArgs {
    const float* x;
    const float* w;
    float* y;
    int H, W, K, R, P, Q;
    int class_shift;                         // maps are processed in 1 << class_shift classes
    int band_h, bands, cq, col_tiles;        // rows of a block, quads of a block per row
    int plane, npos;                         // floats between residue planes (8 mod 32), positions in use
    int cbs, splits, cbs_per_split;          // (class, map block) units in all, and how the blocks share them
    FastDiv div_cq;
};

__device__ __forceinline__ void cp_async4(float* dst_smem, const float* src, bool in)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst_smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(in ? 4 : 0) : "memory");
}

// Resident blocks per SM that the registers are kept down for.
template <int M>
struct Residency { static constexpr int kBlocks = M <= 2 ? 4 : (M <= 8 ? 3 : 2); };

// RT: filter rows, 0 = a.R.  M: maps accumulated together (1, or an even number).
// TURN: maps of every alignment together (one class).  All outputs of a thread start at column 4t; a map whose row starts m
// floats past a boundary is turned into aligned quads at the store, with the last m outputs of the lane to the left.
template <int RT, int S, int M, bool TURN>
__global__ void __launch_bounds__(kMaxThreads, Residency<M>::kBlocks)
single_channel_flat_kernel(const FlatArgs a)
{
    ptx::grid_dep_wait();
    constexpr int PB = M / 2;                             // pairs of maps
    constexpr int TF = M == 1 ? 2 : M;                    // floats per tap: (w, w), or one of every map
    extern __shared__ __align__(16) float smem[];
    const int R = RT ? RT : a.R;
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int split = blockIdx.x % a.splits;
    int rest = blockIdx.x / a.splits;
    const int ct = rest % a.col_tiles;
    rest /= a.col_tiles;
    const int band = rest % a.bands, n = rest / a.bands;
    const int row0 = band * a.band_h;
    const int th = min(a.band_h, a.P - row0);
    const int rows_in = th + R - 1;
    const int col_base = 4 * (ct * a.cq - 1);             // image column of staged column 0
    const int pitch = 4 * a.plane;                        // floats per staged row
    const int cb0 = split * a.cbs_per_split;
    const int ncb = min(a.cbs_per_split, a.cbs - cb0);
    const int cmask = (1 << a.class_shift) - 1;

    float* taps = smem;                                   // [ncb][R][S][TF]
    float* tile = smem + (size_t)a.cbs_per_split * R * S * TF;

    // ---- stage the band with its halo, column c of a row at plane c % 4, position c / 4
    const float* xin = a.x + ((size_t)n * a.H + row0) * a.W;
    for (int row = tid >> 5; row < rows_in; row += nthr >> 5) {
        const float* src = xin + (size_t)row * a.W;
        float* dst = tile + row * pitch + (tid & 3) * a.plane;
        for (int c = tid & 31; c < 4 * a.npos; c += 32) {
            const int col = col_base + c;
            const bool in = (unsigned)col < (unsigned)a.W;
            cp_async4(dst + (c >> 2), in ? src + col : a.x, in);
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    const int rs = R * S;
    for (int idx = tid; idx < ncb * rs * TF; idx += nthr) {
        const int e = M == 1 ? 0 : idx % TF;
        const int t = (idx / TF) % rs, cb = cb0 + idx / (TF * rs);
        const int k = (cb & cmask) + ((((cb >> a.class_shift) * M) + e) << a.class_shift);
        taps[idx] = k < a.K ? __ldg(a.w + (size_t)k * rs + t) : 0.f;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();

    // One map block after the other, every one over the whole band: the stores of a block then run on for band_h rows.
    const size_t map = (size_t)a.P * a.Q;
    const size_t map_step = map << a.class_shift;
    const int col0 = 4 * ct * a.cq;
    float* const band_out = a.y + (size_t)n * a.K * map + (size_t)row0 * a.Q;
    const unsigned band_m = (unsigned)n * (unsigned)a.K * (unsigned)map + (unsigned)row0 * (unsigned)a.Q;      // (only its value modulo 4 is used)
    const int units = th * a.cq, lane = tid & 31;
    const float* wt = taps;
#pragma unroll 1
    for (int cb = cb0; cb < cb0 + ncb; ++cb, wt += rs * TF) {
        const int k0 = (cb & cmask) + (((cb >> a.class_shift) * M) << a.class_shift);
        float* const map_out = band_out + (size_t)k0 * map;
        const unsigned map_m = band_m + (unsigned)k0 * (unsigned)map;
        const int live = (a.K - k0 + cmask) >> a.class_shift;                 // maps of this block that exist (or more)
        // (with TURN all lanes of a warp stay together: lanes past the end repeat the last unit and store nothing)
#pragma unroll 1
        for (int u0 = tid & ~31; u0 < units; u0 += nthr) {
            const bool exists = u0 + lane < units;
            const int u = exists ? u0 + lane : units - 1;
            int t;
            const int row = a.div_cq.divmod(u, t);
            const int row_off = row * a.Q;
            const int m = TURN ? 0 : (int)((map_m + (unsigned)row_off) & 3u);
            const int q0 = col0 + 4 * t - m;
            if (!TURN && (!exists || q0 >= a.Q)) continue;
            const float* base = tile + row * pitch + t;
            // window column i is staged column 4t + 4 - m + i
            const float* win_at[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) win_at[v] = base + ((v + 4 - m) & 3) * a.plane + ((v + 4 - m) >> 2);

            constexpr int NB = M == 1 ? 1 : PB;
            constexpr int NA = M == 1 ? 2 : 4;            // accumulators of a pair: two pairs of outputs, or four outputs
            float2 acc[NB][NA];
#pragma unroll
            for (int b = 0; b < NB; ++b)
#pragma unroll
                for (int j = 0; j < NA; ++j) acc[b][j] = make_float2(0.f, 0.f);
            const float* wr = wt;
#pragma unroll(RT ? RT : 1)
            for (int r = 0; r < R; ++r, wr += S * TF) {
                float v[S + 3];
#pragma unroll
                for (int i = 0; i < S + 3; ++i) v[i] = win_at[i & 3][r * pitch + (i >> 2)];
#pragma unroll
                for (int s = 0; s < S; ++s) {
                    if constexpr (M == 1) {
                        const float2 tap = *reinterpret_cast<const float2*>(wr + s * TF);
#pragma unroll
                        for (int j = 0; j < NA; ++j)
                            acc[0][j] = __ffma2_rn(make_float2(v[s + 2 * j], v[s + 2 * j + 1]), tap, acc[0][j]);
                    } else {
                        float2 tap[NB];
                        if constexpr (PB % 2 == 1) {
#pragma unroll
                            for (int b = 0; b < NB; ++b) tap[b] = *reinterpret_cast<const float2*>(wr + s * TF + 2 * b);
                        } else {
#pragma unroll
                            for (int b = 0; b < PB / 2; ++b) {
                                const float4 t4 = *reinterpret_cast<const float4*>(wr + s * TF + 4 * b);
                                tap[2 * b] = make_float2(t4.x, t4.y);
                                tap[2 * b + 1] = make_float2(t4.z, t4.w);
                            }
                        }
#pragma unroll
                        for (int b = 0; b < NB; ++b)
#pragma unroll
                            for (int j = 0; j < NA; ++j)
                                acc[b][j] = __ffma2_rn(make_float2(v[s + j], v[s + j]), tap[b], acc[b][j]);
                    }
                }
            }
            const bool whole = q0 >= 0 && q0 + 3 < a.Q;
#pragma unroll
            for (int e = 0; e < M; ++e) {
                if (e >= live) break;
                float* const out = map_out + e * map_step + (row_off + q0);
                float o[4];
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    o[j] = M == 1 ? ((j & 1) ? acc[0][(j / 2) % NA].y : acc[0][(j / 2) % NA].x)
                                  : ((e & 1) ? acc[e / 2][j % NA].y : acc[e / 2][j % NA].x);
                if constexpr (TURN) {
                    const int me = (int)((map_m + (unsigned)e * (unsigned)map + (unsigned)row_off) & 3u);
                    float l[3];                            // outputs 1, 2, 3 of the lane to the left
#pragma unroll
                    for (int j = 0; j < 3; ++j) l[j] = __shfl_up_sync(0xffffffffu, o[j + 1], 1);
                    if (!exists) continue;
                    const bool left = lane > 0 && t > 0;   // that lane holds the quad to the left
                    const bool right = lane < 31 && t + 1 < a.cq && u + 1 < units;      // the next lane takes this quad's end along
                    const float s1[6] = {me & 1 ? l[0] : l[1], me & 1 ? l[1] : l[2], me & 1 ? l[2] : o[0],
                                         me & 1 ? o[0] : o[1], me & 1 ? o[1] : o[2], me & 1 ? o[2] : o[3]};
                    const float4 v = make_float4(me & 2 ? s1[0] : s1[2], me & 2 ? s1[1] : s1[3], me & 2 ? s1[2] : s1[4], me & 2 ? s1[3] : s1[5]);
                    const int qa = q0 - me;                // first column of the aligned quad
                    float* const at = out - me;
                    if ((left || me == 0) && qa + 3 < a.Q) {
                        __stcs(reinterpret_cast<float4*>(at), v);
                    } else {
                        if (left && qa < a.Q) __stcs(at, v.x);                           // (me > 0 or the row's last quad)
                        if ((left || me <= 1) && qa + 1 >= 0 && qa + 1 < a.Q) __stcs(at + 1, v.y);
                        if ((left || me <= 2) && qa + 2 >= 0 && qa + 2 < a.Q) __stcs(at + 2, v.z);
                        if (qa + 3 >= 0 && qa + 3 < a.Q) __stcs(at + 3, v.w);
                        if (!left && me == 0 && qa < a.Q) __stcs(at, v.x);
                    }
                    if (!right) {                          // outputs 4 - me .. 3
#pragma unroll
                        for (int j = 1; j < 4; ++j)
                            if (j + me >= 4 && q0 + j < a.Q) __stcs(out + j, o[j]);
                    }
                } else if (whole) {
                    __stcs(reinterpret_cast<float4*>(out), make_float4(o[0], o[1], o[2], o[3]));
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if ((unsigned)(q0 + j) < (unsigned)a.Q) __stcs(out + j, o[j]);
                }
            }
        }
    }
}

// Cycles of a scheduler for one warp's (quad, map block).
inline double unit_cycles(int maps, int R, int S, bool turn)
{
    return (maps == 1 ? 4.0 : 4.0 * maps) * R * S + R * (S + 3) * 2.5 + 60 + (turn ? 75.0 * maps : 0.0);
}

template <int RT, int S, int M, bool TURN>
conv2d_status_t launch_flat(FlatArgs& a, const Shape& sh, cudaStream_t stream)
{
    constexpr int TF = M == 1 ? 2 : M;
    const int classes = 1 << a.class_shift;
    // (class, map block) units, the class fastest: whole rounds over the classes, then the classes that still have a map
    const int whole = sh.K / (classes * M), left = sh.K - whole * classes * M;
    a.cbs = whole * classes + (left < classes ? left : classes);
    const int sms = sm_count();
    const int nq = (sh.Q + (TURN || (a.class_shift == 0 && sh.Q % 4 == 0) ? 0 : 3) + 3) / 4;
    a.col_tiles = (nq + kMaxQuads - 1) / kMaxQuads;
    a.cq = (nq + a.col_tiles - 1) / a.col_tiles;
    a.div_cq = FastDiv(a.cq);
    a.npos = a.cq + 1 + (S + 2 + 3) / 4;
    a.plane = (a.npos + 23) / 32 * 32 + 8;
    // Rows of a block and the share of the maps it computes, by estimated cycles: the work of all blocks spread over the
    // SMs, the last block of an SM with nothing beside it, and the latency of staging (one trip to memory and the set-up).
    // (An SM serves its oldest block first, so blocks that start together end one after the other: few large blocks leave
    // the last one alone for a third of the run; 2048 x 2048, 32 filters of 5 x 5, 10 rows a block: FMA pipe 58 % busy.)
    double best = 0;
    size_t best_smem = 0;
    int best_threads = 0;
    for (int splits = 1; splits <= a.cbs; splits *= 2) {
        const int per = (a.cbs + splits - 1) / splits, used = (a.cbs + per - 1) / per;
        const size_t tap_bytes = (size_t)per * sh.R * S * TF * sizeof(float);
        if (tap_bytes > 64 * 1024) continue;
        for (int bh : {1, 2, 3, 4, 5, 6, 8, 12, 16}) {                       // (the search is on the path of every call)
            if (bh > sh.P) break;
            const size_t smem = tap_bytes + (size_t)(bh + sh.R - 1) * 4 * a.plane * sizeof(float);
            if (smem > (bh == 1 ? (size_t)200 : (size_t)72) * 1024) break;
            const long long blocks = (long long)sh.N * a.col_tiles * ((sh.P + bh - 1) / bh) * used;
            int threads = bh * a.cq >= kMaxThreads ? kMaxThreads : (bh * a.cq + 31) / 32 * 32;
            if (threads < 128 && blocks <= sms) threads = 128;         // (few blocks: the other threads share the staging)
            const int passes = (bh * a.cq + threads - 1) / threads;
            if (splits > 1 && best != 0 && blocks / used >= 2LL * sms) continue;      // (a share of the maps costs the whole staging)
            const int by_regs = Residency<M>::kBlocks * kMaxThreads / threads, by_smem = (int)(220 * 1024 / (smem + 1024));
            const double res = by_regs < by_smem ? by_regs : by_smem;
            // one block on a scheduler: what its warps issue, beside what it writes at an SM's share of the memory rate
            const double staging = (bh + sh.R - 1) * (4.0 * a.npos / 32.0) * 20.0 + (double)per * sh.R * S * TF / 32.0 * 20.0;
            const double issue = ((threads / 32) * (passes * per * unit_cycles(M, sh.R, S, TURN)) + staging) / 4 + kBlockCycles;
            const double write = (double)(sh.K < per * M ? sh.K : per * M) * bh * a.cq * 16.0 / 23.0;
            const double work = issue > write ? issue + 0.3 * write : write + 0.3 * issue;
            const double per_sm = (double)blocks / sms, each = (kLatency + work) / res;
            double t = per_sm * (each > work ? each : work) + 0.7 * work;
            // the time of one block with nothing beside it, whose few warps each sit on a scheduler of their own (without it
            // and the threads that only stage, 14 x 17 x 21, 23 maps of 5 x 3 ran on 42 warps: 12.3 us, now 5.0)
            const int units = (bh * a.cq + 31) / 32, deep = units < threads / 32 ? (units + 3) / 4 : (threads / 32 + 3) / 4;
            const double copies = (bh + sh.R - 1) * (4.0 * a.npos / 32.0) * 32.0 * 60.0 + (double)per * sh.R * S * TF * 250.0;
            const double alone = kLatency + deep * passes * per * unit_cycles(M, sh.R, S, TURN) * 1.3 + copies / threads;
            const double whole_blocks = (double)((blocks + sms - 1) / sms) * work;
            if (blocks <= 4LL * sms && t < whole_blocks) t = whole_blocks;
            if (t < alone) t = alone;
            if (best == 0 || t < best) {
                best = t; best_smem = smem; best_threads = threads;
                a.band_h = bh; a.splits = used; a.cbs_per_split = per;
            }
        }
    }
    if (best == 0) return CONV2D_ERR_UNSUPPORTED;                            // (more taps than shared memory holds)
    a.bands = (sh.P + a.band_h - 1) / a.band_h;
    const long long blocks = (long long)sh.N * a.col_tiles * a.bands * a.splits;
    if (blocks > 0x7fffffffLL) return CONV2D_ERR_UNSUPPORTED;
    auto kern = single_channel_flat_kernel<RT, S, M, TURN>;
    static SmemLimit smem_done;
    if (best_smem > 48 * 1024 && raise_smem_limit(reinterpret_cast<const void*>(kern), best_smem, smem_done) != cudaSuccess)
        return CONV2D_ERR_CUDA;
    if (launch_pdl(kern, dim3((unsigned)blocks), dim3(best_threads), best_smem, stream, a) != cudaSuccess) return CONV2D_ERR_CUDA;
    count_launch();
    return CONV2D_OK;
}

// Maps accumulated together: as many as a class fills.  More of them share the reads of a window row; empty ones cost
// as much as full ones.  16 maps leave two blocks on an SM: they pay from 9 taps on (2048 x 2048, 32 maps: 7 x 7 267 us
// with 8, 255 with 16; 4096 x 4096, 32 maps of 3 x 3 439 and 412; 2048 x 2048, 1 x 1 82 and 84 to 95).
// Classes or turned quads: where a class would have one or two maps only, each class reads the windows anew, which costs
// more than turning the quads of all maps at the store (14 x 375 x 1439, 4 maps of 5 x 5: 83 us in classes, 64 turned;
// 15 x 2463 x 567, 8 maps of 5 x 5 242 and 269; 7 x 1623 x 488, 6 maps of 3 x 3 36 and 49).
struct MapChoice { int maps; bool turn; double cost; };      // cost: cycles of a scheduler for one warp's quads of all maps
MapChoice choose_maps(const Shape& sh, int class_shift)
{
    auto cost = [&](int m, int classes, bool turn) {
        const int per_class = (sh.K + classes - 1) / classes, used = sh.K < classes ? sh.K : classes;
        return (double)used * ((per_class + m - 1) / m) * unit_cycles(m, sh.R, sh.S, turn);
    };
    MapChoice best{1, false, cost(1, 1 << class_shift, false)};
    for (int m : {2, 4, 6, 8, 12, 16}) {
        const double c = cost(m, 1 << class_shift, false);
        if ((m <= 8 || sh.R * sh.S >= 9) && c <= best.cost) best = MapChoice{m, false, c};
    }
    const int forced = env_int("CONV2D_B200_SC_TURN", -1);
    if (class_shift == 0 || forced == 0) return best;
    MapChoice turned{1, true, cost(1, 1, true)};
    for (int m : {2, 4, 8}) {
        const double c = cost(m, 1, true);
        if (c <= turned.cost) turned = MapChoice{m, true, c};
    }
    return forced > 0 || turned.cost < best.cost ? turned : best;
}

template <int RT, int S>
conv2d_status_t launch_maps(FlatArgs& a, const Shape& sh, cudaStream_t stream)
{
    const MapChoice c = choose_maps(sh, a.class_shift);
    if (c.turn) {
        a.class_shift = 0;
        switch (c.maps) {
        case 8: return launch_flat<RT, S, 8, true>(a, sh, stream);
        case 4: return launch_flat<RT, S, 4, true>(a, sh, stream);
        case 2: return launch_flat<RT, S, 2, true>(a, sh, stream);
        default: return launch_flat<RT, S, 1, true>(a, sh, stream);
        }
    }
    switch (c.maps) {
    case 16: return launch_flat<RT, S, 16, false>(a, sh, stream);
    case 12: return launch_flat<RT, S, 12, false>(a, sh, stream);
    case 8: return launch_flat<RT, S, 8, false>(a, sh, stream);
    case 6: return launch_flat<RT, S, 6, false>(a, sh, stream);
    case 4: return launch_flat<RT, S, 4, false>(a, sh, stream);
    case 2: return launch_flat<RT, S, 2, false>(a, sh, stream);
    default: return launch_flat<RT, S, 1, false>(a, sh, stream);
    }
}

int class_shift_of(const Shape& sh)
{
    const long long map = (long long)sh.P * sh.Q;
    return map % 4 == 0 ? 0 : (map % 2 == 0 ? 1 : 2);
}

}  // namespace

double single_channel_flat_cost(const Shape& sh) { return choose_maps(sh, class_shift_of(sh)).cost; }

conv2d_status_t launch_single_channel_flat(const float* x, const float* w, float* y, const Shape& sh, cudaStream_t stream)
{
    FlatArgs a{};
    a.x = x; a.w = w; a.y = y;
    a.H = sh.H; a.W = sh.W; a.K = sh.K; a.R = sh.R; a.P = sh.P; a.Q = sh.Q;
    a.class_shift = class_shift_of(sh);
    if (sh.R == sh.S) {
        switch (sh.R) {
        case 1: return launch_maps<1, 1>(a, sh, stream);
        case 3: return launch_maps<3, 3>(a, sh, stream);
        case 5: return launch_maps<5, 5>(a, sh, stream);
        case 7: return launch_maps<7, 7>(a, sh, stream);
        }
    }
    switch (sh.S) {
    case 1: return launch_maps<0, 1>(a, sh, stream);
    case 2: return launch_maps<0, 2>(a, sh, stream);
    case 3: return launch_maps<0, 3>(a, sh, stream);
    case 4: return launch_maps<0, 4>(a, sh, stream);
    case 5: return launch_maps<0, 5>(a, sh, stream);
    case 6: return launch_maps<0, 6>(a, sh, stream);
    case 7: return launch_maps<0, 7>(a, sh, stream);
    }
    return CONV2D_ERR_UNSUPPORTED;
}

}  // namespace conv2d_b200
