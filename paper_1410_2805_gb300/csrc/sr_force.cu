// Short-range pair force over the chaining mesh (Sec. 3.1, Eq. (force);
// Sec. 3.3: P3M with a chaining mesh on accelerators).
//
// For every particle i of a cell, the force from the particles of the 27
// cells around it (periodic):
//     a_i = G sum_j m_j r_ij f_SR(s),  f_SR(s) = (s+eps)^(-3/2) - P5(s),
// cut at s < r_cut^2 with a select instead of a branch (the paper folds the
// cutoff test into the force evaluation the same way, with fsel).
//
// GPU mapping.  A work item is up to 64 consecutive particles of one cell in
// clusters of 8, run by one warp.  The binning orders each cell's particles
// along a Hilbert curve of 4x4x4 sub-cells, so a cluster is compact: its
// bounds are about 0.5 cell widths a side, where a whole cell's are 0.9.
//   stage   The particles j of the neighbour cells are read in x-runs of
//           consecutive sorted particles ((2R+1)^2 rows, a second run when a
//           row wraps), 64 at a time; those within reach of the item's bounds
//           go to a per-warp shared tile (ballot + prefix count).
//   select  Per cluster, the tile's entries within reach of the cluster's own
//           bounds are compacted into a list (two entries a lane).
//   pairs   Four lanes hold the cluster's 8 particles, two each, and eight
//           lane groups share the list, two entries a step: four pairs per
//           lane and step, as two packed FP32 chains (fma.rn.f32x2), the two
//           entries in the two halves.
// What bounds it: issue slots and the FP32 pipe together.  On 128^3 Zel'dovich
// particles (0.84 ms) a scheduler issues in 70% of its cycles and the FP32 pipe
// is held in 54% (an f32x2 operation takes two of its cycles, three when its
// operands are three different registers); scalar arithmetic for the
// polynomial or the sums, which needs fewer pipe cycles and more slots, is
// 3-7% slower.  The pairs are half of the instructions, the selecting and
// staging most of the rest.
// Why clusters of 8: per particle of a Zel'dovich box, 970 candidates lie in
// the 27 cells, 655 within reach of a cell's bounds, 390 of an 8-cluster's and
// 285 of a 4-cluster's, 154 inside the cutoff (a bounding sphere instead of the
// bounds keeps 18% more).  4-clusters would pay in tests what they save in
// pairs; a last cluster of up to 4 on half the lanes costs more in the loop's
// variable strides than the 5% of pairs that it saves.  Items of 64 share one
// staging among 8 clusters (256^3 box: 6.9 ms a launch against 7.3 with items of
// 32, 8.6 with 16); smaller calls take smaller items to spread over the chip
// (auto_item_cap), the smallest share each item in a block (shared_items).
// Against one warp per cell-wide item whose lanes evaluate all that is within
// reach of the cell (scalar, 5 particles a lane): 256^3 launch 9.3 -> 6.9 ms,
// 128^3 1.19 -> 0.91 ms, 32^3 122 -> 57 us; with the constants as parameters,
// the packed selection, the longer tile and the unrolled last steps 256^3 6.5 ms,
// 128^3 0.84 ms.
//
// Periodic images without rounding error: an item whose cell lies within R of
// a high face (per axis) runs in the frame moved by -L: its own particles and
// the neighbours of unwrapped rows get -L (they lie in [L/2, L) for nc >= 4R:
// exact), those of rows that wrap high stay.  In smaller meshes neighbours of
// unwrapped rows may lie below L/2, so there such an item runs in a frame for
// each set of axes, with its own particles moved by -L on just these (exact both
// ways) and the rows that wrap high on just these as they are, in a form of the
// kernel of its own (with the frames in the one form, 250 thousand particles of
// differing masses took 206 us a call instead of 203, the step of the 256^3 box
// 38.2 ms instead of 37.9).  Elsewhere the neighbours of rows that wrap low get
// -L (exact, in [L/2, L)).  So r_ij = x_j' - x_i' carries only the rounding of
// one subtraction.
#include <cuda_runtime.h>
#include <stdint.h>

#include <cstring>

#include "hacc_internal.cuh"

namespace hacc {
namespace {

constexpr int kWarps = 4;
constexpr int kThreads = kWarps * 32;

// Two FP32 values in one 64-bit register pair; each operation rounds its
// halves as the scalar one does.
typedef unsigned long long f32x2;

// The pair-force constants, each in both halves: eps and P5's negated
// coefficients.  Doubled on the host, they reach the packed operations as
// operands from the parameter bank.  In registers of their own they made each
// step of the polynomial one of three different registers, which holds the FMA
// pipe three cycles instead of two, and took fourteen registers (128^3
// Zel'dovich launch 900 -> 879 us, 256^3 6.91 -> 6.76 ms).
struct PairConsts {
    f32x2 eps, c0, c1, c2, c3, c4, c5;
};

// The pair potential's, likewise: U's coefficients and phi0 negated, and -1.
struct PotConsts {
    f32x2 u0, u1, u2, u3, u4, u5, u6, phi0, minus;
};

struct KParams {
    const float4 *__restrict__ pos;
    const int4 *__restrict__ items;
    const int32_t *__restrict__ order;
    const int32_t *__restrict__ n_items;
    const int32_t *__restrict__ cell_start;
    int *work_counter;
    int nc;
    int R;            // neighbour cells per side of a cell's own (1: 27 cells, 2: 125 cells)
    int cull;         // 1: select per cluster; 0: by the item's bounds alone
    float L;
    float T, eps, G;
    int mode;
    float4 *out;
    const int32_t *__restrict__ perm;
    float4 *vel;
    float4 *pos_next;
    float h_kick, h_drift;
    float *phi_out;
    unsigned long long *within;
    unsigned long long *evaluated;
    const uint32_t *mass_flag;
    int nbox;
    float w, delta;   // cell/offset form: cell step (an FP32 value) and the remainder L - nc w of a wrap
    const int32_t *levels;
    KickTable kick;
    const BoxDev *boxes;
    const int32_t *ids;
    float4 *pos_pool;
    float4 *vel_pool;
    int *flags;
    PairConsts pair;
    PotConsts pot;
};

__device__ __forceinline__ float rsqrt_approx(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ f32x2 pack2(float a, float b) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
// A value that all lanes hold, known as such to the compiler: branches and
// loop bounds made of it stay warp-uniform (no reconvergence code).
__device__ __forceinline__ int uniform(int v) { return __shfl_sync(0xffffffffu, v, 0); }
// A value that all lanes hold, to be kept in a register of its own: it looks
// like any other result of a shuffle, where a constant would be loaded and
// doubled again in every round of the pair loop.
__device__ __forceinline__ float keep(float v) { return __shfl_xor_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ void unpack2(f32x2 v, float &a, float &b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

__device__ __forceinline__ float4 shift4(float4 v, float tx, float ty, float tz) {
    return make_float4(__fadd_rn(v.x, tx), __fadd_rn(v.y, ty), __fadd_rn(v.z, tz), v.w);
}

constexpr int kRound = 64;                // candidates staged per round
constexpr int kRing = 128;                // list entries held: two chunks
constexpr int kChunk = 64;                // list entries per call of the pair loop
constexpr int kMaxClusters = kItemMax / kCluster;
constexpr int kMaxRuns = 50;              // 2 (2R+1)^2 for R = 2

// The staged entries of a warp (the tile) and the list selected for a cluster,
// as arrays of x, y, z and, with M (masses differ), m.  The tile takes what five
// blocks of an SM leave: each flush of it ends every cluster's list with a
// part-filled step and a sum over the warp (256^3 launch 6.76 ms with 384
// entries, 6.57 with 512; six blocks with 384: 6.65).
template <bool M>
struct WarpBuf {
    static constexpr int kArrays = M ? 4 : 3;
    static constexpr int kTile = M ? 384 : 576;   // staged entries at most, whole rounds
    float tile[kArrays][kTile];
    float list[kArrays][kRing];
};
constexpr int kBufBytes = sizeof(WarpBuf<false>);
static_assert(sizeof(WarpBuf<true>) <= kBufBytes && WarpBuf<false>::kTile % kRound == 0 &&
                  WarpBuf<true>::kTile % kRound == 0, "one buffer for both forms");

// A warp's shared memory.  Runs: (first, end, bits, b1) of the sorted
// particles of each x-run, with (b2, d0) for the cell/offset form; bits 1/2/4:
// the staged j's x/y/z get -L; bits 3-5 and b1, for an item in several frames:
// the one that the run belongs to and the run's end, where end = first leaves it
// to another frame; in the cell/offset form bits 0-3 and 4-7 hold
// dy + 2 and dz + 2, bits 8-13 the wrap flags (1/2/4 low in x/y/z, 8/16/32
// high), and the x cell step of entry j is d0 + (j >= b1) + (j >= b2).
template <bool CI, bool POT>
struct WarpMem {
    char buf[kBufBytes];                  // a WarpBuf
    float4 own[kItemMax];                 // the item's particles in its frame
    float sum[3][kItemMax];               // and their sums
    float4 lo[kMaxClusters + 1], hi[kMaxClusters + 1];   // bounds of its clusters, and its own (last)
    int4 runs[kMaxRuns];
    int2 steps[CI ? kMaxRuns : 1];
    int tile_id[POT ? WarpBuf<true>::kTile : 1];         // sorted index of each entry (the j != i test of the potential)
    alignas(8) int id[POT ? kRing : 1];   // those of the list's
    int frames;                           // 0, or of an item in several frames: their axes, from bit 3 on those of the
                                          // present one, from bit 6 on its number
    template <bool M>
    __device__ __forceinline__ WarpBuf<M> &as() {
        return *reinterpret_cast<WarpBuf<M> *>(buf);
    }
};

// The item's neighbour cells as x-runs of consecutive sorted particles, one
// lane per run: row (dz, dy) of the (2R+1)^2 rows gives run `row` (cells
// cx-R..cx+R, or the part of them in [0, nc)) and, when rows wrap in x, run
// span^2 + row (the wrapped part).  fr: axes on which the item runs in the
// frame moved by -L; with `several`, for the rows that wrap high on just these.
// Returns the number of runs.
template <bool CI, bool POT>
__device__ __forceinline__ int build_runs(const KParams &P, WarpMem<CI, POT> &S, int cbase, int nc, int cx, int cy,
                                          int cz, int R, int fr, bool several, int lane) {
    const int span = 2 * R + 1, rows = span * span;
    const int lo = cx - R, hi = cx + R;
    const bool wraps = lo < 0 || hi >= nc;
    const int nrun = wraps ? 2 * rows : rows;
    for (int q = lane; q < nrun; q += 32) {
        const int r = q >= rows ? 1 : 0, rowi = q - r * rows;
        const int dz = rowi / span - R, dy = rowi % span - R;
        int rz = cz + dz, ry = cy + dy;
        int wb = 0;   // wrap flags: 1/2/4 low in x/y/z, 8/16/32 high
        if (rz < 0) { rz += nc; wb |= 4; }
        else if (rz >= nc) { rz -= nc; wb |= 32; }
        if (ry < 0) { ry += nc; wb |= 2; }
        else if (ry >= nc) { ry -= nc; wb |= 16; }
        const int32_t *row = P.cell_start + cbase + (rz * nc + ry) * nc;
        int ca = lo, cb = hi + 1;   // cells [ca, cb) of the row
        int d0 = -1;
        if (lo < 0) {           // [0, hi], then [nc + lo, nc) wrapped low
            ca = r ? nc + lo : 0;
            cb = r ? nc : hi + 1;
            if (r) wb |= 1;
            d0 = r ? -1 : 0;
        } else if (hi >= nc) {  // [lo, nc), then [0, hi - nc] wrapped high
            ca = r ? 0 : lo;
            cb = r ? hi - nc + 1 : nc;
            if (r) wb |= 8;
            d0 = r ? 1 : -1;
        }
        const int ja = row[ca], jb = row[cb];
        int bits, b1 = jb, end = jb;
        if (CI) {
            bits = (dy + 2) | ((dz + 2) << 4) | (wb << 8);
            // first entries of the run's second and third cell (R = 1)
            b1 = cb - ca > 1 ? row[ca + 1] : jb;
            const int b2 = cb - ca > 2 ? row[ca + 2] : jb;
            S.steps[q] = make_int2(b2, d0);
        } else {
            // -L on an axis: rows wrapped low, or every row not wrapped high in the moved frame
            bits = (wb & 7) | (several ? wb & 56 : fr & ~(wb >> 3));
            if (several && wb >> 3 != fr) end = ja;
        }
        S.runs[q] = make_int4(ja, end, bits, b1);
    }
    __syncwarp();
    return uniform(nrun);
}

// Frame r of an item that runs in one for each subset of `axes`: the r-th subset.
__device__ __forceinline__ int frame_of(int r, int axes) {
    int f = 0;
#pragma unroll
    for (int b = 1; b < 8; b <<= 1)
        if (axes & b) {
            f |= r & 1 ? b : 0;
            r >>= 1;
        }
    return f;
}

// From one frame of an item in several to frame r: its particles and bounds
// moved on the axes that differ, and the runs of the new frame.
template <bool CI, bool POT>
__device__ __forceinline__ void change_frame(WarpMem<CI, POT> &S, int axes, int from, int r, float L, int nrun,
                                             int lane) {
    const int to = frame_of(r, axes);
    const float tx = L * (float)((from & 1) - (to & 1)), ty = L * (float)((from >> 1 & 1) - (to >> 1 & 1)),
                tz = L * (float)((from >> 2) - (to >> 2));
    __syncwarp();
    for (int e = lane; e < kItemMax; e += 32) S.own[e] = shift4(S.own[e], tx, ty, tz);
    if (lane <= kMaxClusters) {
        S.lo[lane] = shift4(S.lo[lane], tx, ty, tz);
        S.hi[lane] = shift4(S.hi[lane], tx, ty, tz);
    }
    for (int q = lane; q < nrun; q += 32) {
        const int4 run = S.runs[q];
        S.runs[q].y = run.z >> 3 == to ? run.w : run.x;
    }
    if (lane == 0) S.frames = axes | to << 3 | r << 6;
    __syncwarp();
}

// Apply the force on sorted particle i (position x, y, z, mass m) as the
// launch's mode says: store it, kick, or kick and stream.
__device__ __forceinline__ void write_result(const KParams &P, int i, float gx, float gy, float gz, float x, float y,
                                             float z, float m, float h_kick, float h_drift, float L) {
    if (P.mode == kModeForce) {
        int o = P.perm ? P.perm[i] : i;
        P.out[o] = make_float4(gx, gy, gz, 0.0f);
    } else if (P.mode == kModeKickLevels) {
        const float hk = P.kick.h[P.levels[i]];
        if (hk != 0.0f) {
            float4 v = P.vel[i];
            v.x = __fmaf_rn(hk, gx, v.x);
            v.y = __fmaf_rn(hk, gy, v.y);
            v.z = __fmaf_rn(hk, gz, v.z);
            if (P.ids) P.vel_pool[P.ids[i]] = v;   // back to input order
            else P.vel[i] = v;                      // in place, sorted order
        }
    } else if (P.mode == kModeKick) {
        const int row = P.ids[i];
        float4 v = P.vel[i];
        v.x = __fmaf_rn(h_kick, gx, v.x);
        v.y = __fmaf_rn(h_kick, gy, v.y);
        v.z = __fmaf_rn(h_kick, gz, v.z);
        P.vel_pool[row] = v;
    } else {
        float4 v = P.vel[i];
        v.x = __fmaf_rn(h_kick, gx, v.x);
        v.y = __fmaf_rn(h_kick, gy, v.y);
        v.z = __fmaf_rn(h_kick, gz, v.z);
        float4 p;
        p.x = __fmaf_rn(h_drift, v.x, x);
        p.y = __fmaf_rn(h_drift, v.y, y);
        p.z = __fmaf_rn(h_drift, v.z, z);
        p.w = m;
        if (P.mode == kModeBatch) {
            // back to the box's pool row, wrapped into [0, L)
            bool ok = wrap1(p.x, L);
            ok &= wrap1(p.y, L);
            ok &= wrap1(p.z, L);
            if (!ok) atomicOr(P.flags, kFlagDomain);
            const int row = P.ids[i];
            P.vel_pool[row] = v;
            P.pos_pool[row] = p;
        } else {
            P.vel[i] = v;
            P.pos_next[i] = p;
        }
    }
}

// Squared distance of v from the box [lo, hi].  A j is dropped when it reaches
// a limit that carries a margin far above the rounding of the distance: it
// is outside the cutoff of every i of the box and would have added exactly
// nothing.  A NaN is dropped too.
__device__ __forceinline__ float box_dist2(float4 v, float4 lo, float4 hi) {
    const float ex = v.x - fminf(fmaxf(v.x, lo.x), hi.x);
    const float ey = v.y - fminf(fmaxf(v.y, lo.y), hi.y);
    const float ez = v.z - fminf(fmaxf(v.z, lo.z), hi.z);
    return __fmaf_rn(ex, ex, __fmaf_rn(ey, ey, ez * ez));
}

// A cluster's bounds in units of the reach 1/s, as centre c and negated half
// widths nh (s times them): the distance from them along an axis is
// s |v - c| + nh, cut to [0, 1] by the saturation of the FMA itself.  Axes past
// the reach saturate at 1, so a j is within reach when the squares sum to less
// than 1.  The roundings of c, of v - c and of the half widths and their product
// with s move a distance by a few ulp of the half width, more than the margin of
// the limit where a cluster is thousands of cutoffs wide (few particles in wide
// cells): the half widths are widened by 2^-21, eight such roundings.  Against
// clamping v to [lo, hi], half the instructions: no minimum and maximum, which
// run at half the rate, and the subtraction and the squares packed.
struct Reach {
    float cx, cy, cz, nhx, nhy, nhz, s;
};

__device__ __forceinline__ Reach reach_of(float4 lo, float4 hi, float s) {
    Reach b;
    b.s = s;
    b.cx = 0.5f * lo.x + 0.5f * hi.x;
    b.cy = 0.5f * lo.y + 0.5f * hi.y;
    b.cz = 0.5f * lo.z + 0.5f * hi.z;
    const float wide = -s * (1.0f + 0x1p-21f);
    b.nhx = wide * fmaxf(hi.x - b.cx, b.cx - lo.x);
    b.nhy = wide * fmaxf(hi.y - b.cy, b.cy - lo.y);
    b.nhz = wide * fmaxf(hi.z - b.cz, b.cz - lo.z);
    return b;
}

// The distances along an axis of two entries, in units of the reach.
__device__ __forceinline__ f32x2 axis_reach(f32x2 v, float c, float nh, float s) {
    float d0, d1;
    unpack2(add2(v, pack2(-c, -c)), d0, d1);
    return pack2(__saturatef(__fmaf_rn(fabsf(d0), s, nh)), __saturatef(__fmaf_rn(fabsf(d1), s, nh)));
}

// Compaction of the lanes with d2 < r2 in lane order, as predicated stores
// (no branch) of the coordinates (and mass with M) to the arrays of the tile or
// of the list, `at` + prefix count; returns the number of lanes that stored.
// Addresses are those of shared memory.
template <bool M>
__device__ __forceinline__ int put_tile(float d2, float r2, unsigned below, unsigned tile, int at, float4 v) {
    constexpr int kStep = 4 * WarpBuf<M>::kTile;   // bytes from one array to the next
    int n;
    if (M)
        asm volatile(
            "{\n.reg .pred p;\n.reg .b32 m, a;\n"
            "setp.lt.f32 p, %1, %2;\n"
            "vote.sync.ballot.b32 m, p, 0xffffffff;\n"
            "popc.b32 %0, m;\n"
            "and.b32 m, m, %3;\n"
            "popc.b32 a, m;\n"
            "add.s32 a, a, %5;\n"
            "mad.lo.u32 a, a, 4, %4;\n"
            "@p st.shared.f32 [a], %6;\n"
            "@p st.shared.f32 [a + %10], %7;\n"
            "@p st.shared.f32 [a + %11], %8;\n"
            "@p st.shared.f32 [a + %12], %9;\n}"
            : "=r"(n)
            : "f"(d2), "f"(r2), "r"(below), "r"(tile), "r"(at), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "n"(kStep),
              "n"(2 * kStep), "n"(3 * kStep)
            : "memory");
    else
        asm volatile(
            "{\n.reg .pred p;\n.reg .b32 m, a;\n"
            "setp.lt.f32 p, %1, %2;\n"
            "vote.sync.ballot.b32 m, p, 0xffffffff;\n"
            "popc.b32 %0, m;\n"
            "and.b32 m, m, %3;\n"
            "popc.b32 a, m;\n"
            "add.s32 a, a, %5;\n"
            "mad.lo.u32 a, a, 4, %4;\n"
            "@p st.shared.f32 [a], %6;\n"
            "@p st.shared.f32 [a + %9], %7;\n"
            "@p st.shared.f32 [a + %10], %8;\n}"
            : "=r"(n)
            : "f"(d2), "f"(r2), "r"(below), "r"(tile), "r"(at), "f"(v.x), "f"(v.y), "f"(v.z), "n"(kStep),
              "n"(2 * kStep)
            : "memory");
    return n;
}

template <bool M>
__device__ __forceinline__ int put3(float d2, float r2, unsigned below, unsigned ring, int at, float4 v) {
    static_assert(kRing == 128, "ring mask and array distances below");
    int n;
    if (M)
        asm volatile(
            "{\n.reg .pred p;\n.reg .b32 m, a;\n"
            "setp.lt.f32 p, %1, %2;\n"
            "vote.sync.ballot.b32 m, p, 0xffffffff;\n"
            "popc.b32 %0, m;\n"
            "and.b32 m, m, %3;\n"
            "popc.b32 a, m;\n"
            "add.s32 a, a, %5;\n"
            "and.b32 a, a, 127;\n"
            "mad.lo.u32 a, a, 4, %4;\n"
            "@p st.shared.f32 [a], %6;\n"
            "@p st.shared.f32 [a + 512], %7;\n"
            "@p st.shared.f32 [a + 1024], %8;\n"
            "@p st.shared.f32 [a + 1536], %9;\n}"
            : "=r"(n)
            : "f"(d2), "f"(r2), "r"(below), "r"(ring), "r"(at), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
            : "memory");
    else
        asm volatile(
            "{\n.reg .pred p;\n.reg .b32 m, a;\n"
            "setp.lt.f32 p, %1, %2;\n"
            "vote.sync.ballot.b32 m, p, 0xffffffff;\n"
            "popc.b32 %0, m;\n"
            "and.b32 m, m, %3;\n"
            "popc.b32 a, m;\n"
            "add.s32 a, a, %5;\n"
            "and.b32 a, a, 127;\n"
            "mad.lo.u32 a, a, 4, %4;\n"
            "@p st.shared.f32 [a], %6;\n"
            "@p st.shared.f32 [a + 512], %7;\n"
            "@p st.shared.f32 [a + 1024], %8;\n}"
            : "=r"(n)
            : "f"(d2), "f"(r2), "r"(below), "r"(ring), "r"(at), "f"(v.x), "f"(v.y), "f"(v.z)
            : "memory");
    return n;
}

__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

// This lane's two particles: their negated coordinates, doubled, and their
// sums over the list entries the lane's group took (one sum per half).
struct Pair {
    f32x2 nx[2], ny[2], nz[2];
    f32x2 ax[2], ay[2], az[2];
};

__device__ __forceinline__ f32x2 lds2(unsigned addr, int off) {
    f32x2 r;
    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(r) : "r"(addr + off));
    return r;
}

// One step: an entry pair per lane group (x, y, z[, m] of the two entries at
// `addr` and the following arrays of the list) against the lane's particles.
template <bool COUNT, bool EPS0, bool UM>
__device__ __forceinline__ void pair_step(const PairConsts &C, float T, unsigned addr, Pair &A, unsigned &cnt) {
    const f32x2 X = lds2(addr, 0), Y = lds2(addr, 4 * kRing), Z = lds2(addr, 8 * kRing);
    f32x2 M = 0ull;
    if (!UM) M = lds2(addr, 12 * kRing);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const f32x2 dx = add2(X, A.nx[k]), dy = add2(Y, A.ny[k]), dz = add2(Z, A.nz[k]);
        const f32x2 t2 = fma2(dx, dx, fma2(dy, dy, fma2(dz, dz, C.eps)));
        float t0, t1;
        unpack2(t2, t0, t1);
        const f32x2 r = pack2(rsqrt_approx(t0), rsqrt_approx(t1));
        f32x2 q = fma2(C.c5, t2, C.c4);   // -P5
        q = fma2(q, t2, C.c3);
        q = fma2(q, t2, C.c2);
        q = fma2(q, t2, C.c1);
        q = fma2(q, t2, C.c0);
        f32x2 f = fma2(mul2(r, r), r, q);   // t^(-3/2) - P5
        if (!UM) f = mul2(f, M);
        // the cutoff as a select on f (the paper's fsel)
        const bool in0 = EPS0 ? (t0 < T && t0 > 0.0f) : t0 < T, in1 = EPS0 ? (t1 < T && t1 > 0.0f) : t1 < T;
        float f0, f1;
        unpack2(f, f0, f1);
        f = pack2(in0 ? f0 : 0.0f, in1 ? f1 : 0.0f);
        if (COUNT) cnt += (t0 < T ? 1u : 0u) + (t1 < T ? 1u : 0u);
        A.ax[k] = fma2(f, dx, A.ax[k]);
        A.ay[k] = fma2(f, dy, A.ay[k]);
        A.az[k] = fma2(f, dz, A.az[k]);
    }
}

// The same for the pair potential: phi(s) = -t^(-1/2) - U(t) - phi0 inside
// the cutoff, U in t = s + eps; A.ax[k] = sum_j m_j phi over j != i, with the
// entries' sorted indices at `ids` and i that of the lane's first particle.
// Packed as the force is, for the same reasons (an entry at a time, the
// diagnostics of three boxes of 2 million particles took 4.89 ms, now 3.44).
__device__ __forceinline__ void potential_step(const PotConsts &C, f32x2 eps, float T, unsigned addr, unsigned ids,
                                               int i, Pair &A) {
    const f32x2 X = lds2(addr, 0), Y = lds2(addr, 4 * kRing), Z = lds2(addr, 8 * kRing), M = lds2(addr, 12 * kRing);
    const f32x2 j = lds2(ids, 0);
    const int j0 = (int)(uint32_t)j, j1 = (int)(j >> 32);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const f32x2 dx = add2(X, A.nx[k]), dy = add2(Y, A.ny[k]), dz = add2(Z, A.nz[k]);
        const f32x2 t2 = fma2(dx, dx, fma2(dy, dy, fma2(dz, dz, eps)));
        float t0, t1;
        unpack2(t2, t0, t1);
        const f32x2 r = pack2(rsqrt_approx(t0), rsqrt_approx(t1));
        f32x2 u = fma2(C.u6, t2, C.u5);   // -U
        u = fma2(u, t2, C.u4);
        u = fma2(u, t2, C.u3);
        u = fma2(u, t2, C.u2);
        u = fma2(u, t2, C.u1);
        u = fma2(u, t2, C.u0);
        u = mul2(add2(fma2(r, C.minus, u), C.phi0), M);
        float u0, u1;
        unpack2(u, u0, u1);
        A.ax[k] = add2(A.ax[k], pack2(t0 < T && j0 != i + k ? u0 : 0.0f, t1 < T && j1 != i + k ? u1 : 0.0f));
    }
}

// Run the item's clusters against the `fill` entries of the tile, and add
// to their sums, with the item moved by (tx, ty, tz) in the cell/offset form.
template <bool COUNT, bool POT, bool EPS0, bool UM, int F, bool CI>
__device__ __forceinline__ void flush_tile(const KParams &P, WarpMem<CI, POT> &S, int fill, int i0, int ni, float tx,
                                           float ty, float tz, float r2, int lane, unsigned &cnt, unsigned &evals) {
    constexpr int kTile = WarpBuf<!UM>::kTile;
    WarpBuf<!UM> &buf = S.template as<!UM>();
    // whole rounds of 64 entries: outside everything, massless
    const int full = uniform((fill + kRound - 1) & ~(kRound - 1));
#pragma unroll
    for (int h = 0; h < kRound; h += 32)
        if (fill + h + lane < full) {
#pragma unroll
            for (int a = 0; a < WarpBuf<!UM>::kArrays; ++a) buf.tile[a][fill + h + lane] = a < 3 ? 1e18f : 0.0f;
        }
    __syncwarp();
    const unsigned below = (1u << lane) - 1u;
    const int grp = lane >> 2, slot = lane & 3;
    const unsigned tile = smem_addr(buf.tile), ring = smem_addr(buf.list), mine = ring + 8 * grp;   // the list; this group's entry pairs
    const unsigned ids = smem_addr(S.id) + 8 * grp;   // POT: the list's sorted indices
    const float T = keep(P.T), s_reach = rsqrtf(r2);
#pragma unroll 1
    for (int c0 = 0; c0 < ni; c0 += kCluster) {
        float4 lo = S.lo[c0 / kCluster], hi = S.hi[c0 / kCluster];
        Pair A;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            float4 p = S.own[c0 + 2 * slot + k];
            if (CI) p = shift4(p, tx, ty, tz);
            A.nx[k] = pack2(-p.x, -p.x);
            A.ny[k] = pack2(-p.y, -p.y);
            A.nz[k] = pack2(-p.z, -p.z);
            A.ax[k] = A.ay[k] = A.az[k] = 0ull;
        }
        if (CI) {
            lo = shift4(lo, tx, ty, tz);
            hi = shift4(hi, tx, ty, tz);
        }
        const Reach B = reach_of(lo, hi, s_reach);
        int at = 0, todo = 0;   // ring position of the next entry; entries waiting
#pragma unroll 1
        for (int e0 = 0; e0 < full; e0 += kRound) {
            // entries e and e + 1 of the tile
            const int e = e0 + 2 * lane;
            const unsigned te = tile + 4 * e;
            const f32x2 X = lds2(te, 0), Y = lds2(te, 4 * kTile), Z = lds2(te, 8 * kTile);
            float4 v0 = make_float4(0.0f, 0.0f, 0.0f, 0.0f), v1 = v0;
            unpack2(X, v0.x, v1.x);
            unpack2(Y, v0.y, v1.y);
            unpack2(Z, v0.z, v1.z);
            if (!UM) unpack2(lds2(te, 12 * kTile), v0.w, v1.w);
            const f32x2 ex = axis_reach(X, B.cx, B.nhx, B.s), ey = axis_reach(Y, B.cy, B.nhy, B.s),
                        ez = axis_reach(Z, B.cz, B.nhz, B.s);
            float d0, d1;
            unpack2(fma2(ex, ex, fma2(ey, ey, mul2(ez, ez))), d0, d1);
            const int n0 = put3<!UM>(d0, 1.0f, below, ring, at, v0);
            const int n1 = put3<!UM>(d1, 1.0f, below, ring, at + n0, v1);
            if (POT) {
                const unsigned m0 = __ballot_sync(0xffffffffu, d0 < 1.0f), m1 = __ballot_sync(0xffffffffu, d1 < 1.0f);
                if (d0 < 1.0f) S.id[(at + __popc(m0 & below)) & (kRing - 1)] = S.tile_id[e];
                if (d1 < 1.0f) S.id[(at + n0 + __popc(m1 & below)) & (kRing - 1)] = S.tile_id[e + 1];
            }
            at += n0 + n1;
            todo = uniform(todo + n0 + n1);
            if (COUNT) evals += (unsigned)(n0 + n1) * (unsigned)min(kCluster, ni - c0);
            if (todo >= kChunk) {
                __syncwarp();
                const int base = (at - todo) & (kRing - 1);
                if constexpr (POT) {
#pragma unroll F
                    for (int t = 0; t < kChunk / 16; ++t)
                        potential_step(P.pot, P.pair.eps, T, mine + 4 * base + 64 * t, ids + 4 * base + 64 * t,
                                       i0 + c0 + 2 * slot, A);
                } else {
#pragma unroll F
                    for (int t = 0; t < kChunk / 16; ++t)
                        pair_step<COUNT, EPS0, UM>(P.pair, T, mine + 4 * base + 64 * t, A, cnt);
                }
                todo -= kChunk;
                __syncwarp();
            }
        }
        if (todo) {   // what is left, padded to whole steps
            const int base = (at - todo) & (kRing - 1), len = (todo + 15) & ~15;
            if (todo + lane < len) {
                const int q = base + todo + lane;
#pragma unroll
                for (int a = 0; a < WarpBuf<!UM>::kArrays; ++a) buf.list[a][q] = a < 3 ? 1e18f : 0.0f;
                if (POT) S.id[q] = -1;
            }
            __syncwarp();
            if constexpr (POT) {
#pragma unroll 1
                for (int q = 4 * base; q < 4 * (base + len); q += 64)
                    potential_step(P.pot, P.pair.eps, T, mine + q, ids + q, i0 + c0 + 2 * slot, A);
            } else {
                // 1 to 4 steps, without the loop's overhead
                unsigned q = mine + 4 * base;
                if (len > 32) {
                    pair_step<COUNT, EPS0, UM>(P.pair, T, q, A, cnt);
                    pair_step<COUNT, EPS0, UM>(P.pair, T, q + 64, A, cnt);
                    q += 128;
                }
                pair_step<COUNT, EPS0, UM>(P.pair, T, q, A, cnt);
                if (!(len & 16)) pair_step<COUNT, EPS0, UM>(P.pair, T, q + 64, A, cnt);
            }
            __syncwarp();
        }
        // sum over the eight groups: the halves of the warp first exchange one
        // particle each, then lanes of a half add up
        float s[6];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            float u, v;
            unpack2(A.ax[k], u, v);
            s[3 * k] = u + v;
            unpack2(A.ay[k], u, v);
            s[3 * k + 1] = u + v;
            unpack2(A.az[k], u, v);
            s[3 * k + 2] = u + v;
        }
        const bool up = lane & 16;
#pragma unroll
        for (int k = 0; k < (POT ? 1 : 3); ++k) {
            const float give = up ? s[k] : s[3 + k];
            float a = (up ? s[3 + k] : s[k]) + __shfl_xor_sync(0xffffffffu, give, 16);
            a += __shfl_xor_sync(0xffffffffu, a, 8);
            a += __shfl_xor_sync(0xffffffffu, a, 4);
            if ((lane & 12) == 0) S.sum[k][c0 + 2 * slot + (up ? 1 : 0)] += a;
        }
    }
    __syncwarp();
}

template <bool COUNT, bool POT, bool EPS0, bool UM, int F, bool CI, Sharing SH, bool FRAMES>
__device__ __forceinline__ void process_item(const KParams &P, int4 item, WarpMem<CI, POT> &S, int lane, int warp) {
    // geometry: the single box of the call, or this item's box of a batch
    int nc = P.nc;
    float L = P.L;
    int cbase = 0, parts = 1;
    if (P.boxes) {
        const BoxDev &bx = P.boxes[item.w];
        if (SH == kByParts && shared_items(bx.n)) parts = kWarps;
        nc = uniform(bx.nc);
        L = bx.L;
        cbase = uniform(bx.cell_base);
    }
    const int c = item.x - cbase, i0 = item.y, ni = item.z;
    const int cx = c % nc, cy = (c / nc) % nc, cz = c / (nc * nc);
    const int R = P.boxes ? 1 : P.R;
    // The rounds of a shared item go to its warps in turn, each run starting with
    // another warp: most runs are one full round and a part.  The warp of a batch
    // goes through the parts of a small box's item one after the other, so that
    // its sums are those of the box in a call of its own.  Of an item in several
    // frames a part takes its share of the frames, or, where they are fewer than
    // the parts, its share of the rounds of one (with all frames in every part, a
    // batch of 500 boxes of 3 cells a side and 1000 particles took 1234 us, now 957).
    int part = SH == kByBlock ? warp : 0;
    if (SH == kByBlock) parts = kWarps;
    // axes on which the item runs in the frame moved by -L, and those of its first frame
    const int axes = CI ? 0 : ((cx + R >= nc ? 1 : 0) | (cy + R >= nc ? 2 : 0) | (cz + R >= nc ? 4 : 0));
    const bool several = FRAMES && axes && nc < 4 * R;
    const int log_frames = several ? __popc(axes) : 0, first_frame = part & ((1 << log_frames) - 1);
    const int fr = several ? frame_of(first_frame, axes) : axes;
    int shares = max(1, parts >> log_frames), share = part >> log_frames;   // of the rounds of a frame; this part's
    {
        float4 lo = make_float4(1e30f, 1e30f, 1e30f, 0.0f), hi = make_float4(-1e30f, -1e30f, -1e30f, 0.0f);
#pragma unroll
        for (int h = 0; h < kItemMax; h += 32) {
            if (h >= ni) break;
            const bool on = h + lane < ni;
            float4 f = on ? P.pos[i0 + h + lane] : make_float4(-1e30f, -1e30f, -1e30f, 0.0f);
            f = shift4(f, fr & 1 ? -L : 0.0f, fr & 2 ? -L : 0.0f, fr & 4 ? -L : 0.0f);
            S.own[h + lane] = f;
#pragma unroll
            for (int k = 0; k < 3; ++k) S.sum[k][h + lane] = 0.0f;
            float4 a = on ? f : make_float4(1e30f, 1e30f, 1e30f, 0.0f);
            float4 b = on ? f : make_float4(-1e30f, -1e30f, -1e30f, 0.0f);
#pragma unroll
            for (int o = 1; o < kCluster; o <<= 1) {
                a.x = fminf(a.x, __shfl_xor_sync(0xffffffffu, a.x, o));
                b.x = fmaxf(b.x, __shfl_xor_sync(0xffffffffu, b.x, o));
                a.y = fminf(a.y, __shfl_xor_sync(0xffffffffu, a.y, o));
                b.y = fmaxf(b.y, __shfl_xor_sync(0xffffffffu, b.y, o));
                a.z = fminf(a.z, __shfl_xor_sync(0xffffffffu, a.z, o));
                b.z = fmaxf(b.z, __shfl_xor_sync(0xffffffffu, b.z, o));
            }
            if ((lane & (kCluster - 1)) == 0) {
                S.lo[(h + lane) / kCluster] = a;
                S.hi[(h + lane) / kCluster] = b;
            }
            lo = make_float4(fminf(lo.x, a.x), fminf(lo.y, a.y), fminf(lo.z, a.z), 0.0f);
            hi = make_float4(fmaxf(hi.x, b.x), fmaxf(hi.y, b.y), fmaxf(hi.z, b.z), 0.0f);
        }
#pragma unroll
        for (int o = kCluster; o < 32; o <<= 1) {
            lo.x = fminf(lo.x, __shfl_xor_sync(0xffffffffu, lo.x, o));
            hi.x = fmaxf(hi.x, __shfl_xor_sync(0xffffffffu, hi.x, o));
            lo.y = fminf(lo.y, __shfl_xor_sync(0xffffffffu, lo.y, o));
            hi.y = fmaxf(hi.y, __shfl_xor_sync(0xffffffffu, hi.y, o));
            lo.z = fminf(lo.z, __shfl_xor_sync(0xffffffffu, lo.z, o));
            hi.z = fmaxf(hi.z, __shfl_xor_sync(0xffffffffu, hi.z, o));
        }
        __syncwarp();
        // the item's bounds; with no cull, every cluster's as well
        if (lane == kMaxClusters || (!P.cull && lane < kMaxClusters)) {
            S.lo[lane] = lo;
            S.hi[lane] = hi;
        }
    }
    const float r2 = P.T * 1.001f + 1e-3f;
    if (FRAMES && lane == 0) S.frames = several ? axes | fr << 3 | first_frame << 6 : 0;
    const int nrun = build_runs<CI, POT>(P, S, cbase, nc, cx, cy, cz, R, fr, several, lane);
    // In the cell/offset form a wrapped neighbour lies the remainder L - nc w
    // beyond the whole cell steps: moving i by it instead keeps the j side
    // exact (the shifted i is exact too for any i within reach of the face),
    // so a change of the shift between runs ends a tile.
    const bool moves = CI && P.delta != 0.0f &&
                       !(cx >= R && cy >= R && cz >= R && cx + R < nc && cy + R < nc && cz + R < nc);
    float tx = 0.0f, ty = 0.0f, tz = 0.0f;
    unsigned cnt = 0, evals = 0;
    constexpr int kTile = WarpBuf<!UM>::kTile;
    const unsigned below = (1u << lane) - 1u, tile = smem_addr(S.buf);
    int fill = 0;
    // the stream of rounds: 64 particles of a run (past its end: its last one
    // again, never kept); the next round's loads are in flight while this one's
    // are tested
    int q = -1, j0 = 0, end = 0, bits = 0, b1 = 0;
    float sx = 0.0f, sy = 0.0f, sz = 0.0f;   // shift of the run's particles
    auto next = [&]() -> bool {
        j0 += SH == kWhole ? kRound : kRound * shares;
        while (j0 >= end) {
            if (++q >= nrun) return false;
            const int4 run = S.runs[q];
            j0 = uniform(run.x);
            if (SH != kWhole) j0 += kRound * ((share - q) & (shares - 1));
            end = uniform(run.y);
            bits = uniform(run.z);
            b1 = run.w;
            if (!CI) {
                sx = (bits & 1) ? -L : 0.0f;
                sy = (bits & 2) ? -L : 0.0f;
                sz = (bits & 4) ? -L : 0.0f;
            }
        }
        return true;
    };
    float4 n0, n1;
    auto load = [&]() {
        n0 = P.pos[min(j0 + lane, end - 1)];
        n1 = P.pos[min(j0 + 32 + lane, end - 1)];
    };
#pragma unroll 1
    for (;;) {
        bool more = next();
        if (more) load();
#pragma unroll 1
        while (more) {
            float4 v[2] = {n0, n1};
            if (!CI) {
                v[0] = shift4(v[0], sx, sy, sz);
                v[1] = shift4(v[1], sx, sy, sz);
            }
            const int j = j0 + lane, left = end - j0, run_bits = bits, step1 = b1;
            int2 st = make_int2(0, 0);
            if (CI) st = S.steps[q];
            // no flush after this round?  Then its successor's loads start now, else
            // after the flush (held across it, they would cost it eight registers)
            const bool calm = fill <= kTile - 2 * kRound;
            more = next();
            if (more && calm) load();
            if (CI) {
                sy = (float)((run_bits & 15) - 2) * P.w;
                sz = (float)(((run_bits >> 4) & 15) - 2) * P.w;
                if (moves) {
                    const int wb = run_bits >> 8;
                    const float ux = (wb & 1) ? P.delta : ((wb & 8) ? -P.delta : 0.0f);
                    const float uy = (wb & 2) ? P.delta : ((wb & 16) ? -P.delta : 0.0f);
                    const float uz = (wb & 4) ? P.delta : ((wb & 32) ? -P.delta : 0.0f);
                    if (ux != tx || uy != ty || uz != tz) {
                        if (fill)
                            flush_tile<COUNT, POT, EPS0, UM, F, CI>(P, S, fill, i0, ni, tx, ty, tz, r2, lane, cnt, evals);
                        fill = 0;
                        tx = ux;
                        ty = uy;
                        tz = uz;
                    }
                }
            }
            float4 lo = S.lo[kMaxClusters], hi = S.hi[kMaxClusters];
            if (CI) {
                lo = shift4(lo, tx, ty, tz);
                hi = shift4(hi, tx, ty, tz);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (h && left <= 32) break;
                if (CI) {
                    // whole cell steps of the FP32 width w move j into the frame of i's
                    // cell: exact for a j within reach of i's cell, so a close pair
                    // across a face gets its separation with one rounding at most
                    const int jj = j + 32 * h;
                    const float d = (float)(st.y + (jj >= step1) + (jj >= st.x));
                    v[h] = shift4(v[h], d * P.w, sy, sz);
                }
                const float d2 = box_dist2(v[h], lo, hi), lim = lane + 32 * h < left ? r2 : 0.0f;
                if (POT) {
                    const unsigned m = __ballot_sync(0xffffffffu, d2 < lim);
                    if (d2 < lim) S.tile_id[fill + __popc(m & below)] = j + 32 * h;
                }
                fill = uniform(fill + put_tile<!UM>(d2, lim, below, tile, fill, v[h]));
            }
            if (!calm) {
                if (fill > kTile - kRound) {
                    flush_tile<COUNT, POT, EPS0, UM, F, CI>(P, S, fill, i0, ni, tx, ty, tz, r2, lane, cnt, evals);
                    fill = 0;
                }
                if (more) load();
            }
        }
        if (fill) flush_tile<COUNT, POT, EPS0, UM, F, CI>(P, S, fill, i0, ni, tx, ty, tz, r2, lane, cnt, evals);
        if constexpr (FRAMES) {
            if (const int w = uniform(S.frames)) {   // on to the part's next frame, or the first of the next part
                const int all = w & 7, r = (w >> 6) + (SH == kWhole ? 1 : parts), n = 1 << __popc(all);
                const bool on = r < n, first = SH == kByParts && !on && part + 1 < parts;
                if (on || first) change_frame<CI, POT>(S, all, w >> 3 & 7, on ? r : (part + 1) & (n - 1), L, nrun, lane);
                if (on) {
                    fill = 0;
                    q = -1;
                    j0 = end = 0;
                    continue;
                }
            }
        }
        if (SH != kByParts || parts == 1) break;
        if constexpr (SH == kByParts) {
            // the parts' sums are added in order (items of a small box hold at most 32 particles)
            for (int k = 0; k < (POT ? 1 : 3); ++k) {
                const float a = S.sum[k][lane];
                S.sum[k][32 + lane] = part ? S.sum[k][32 + lane] + a : a;
                S.sum[k][lane] = 0.0f;
            }
            __syncwarp();
            if (++part == parts) break;
            share = part >> log_frames;
            fill = 0;
            q = -1;
            j0 = end = 0;
        }
    }

    // epilogue: a particle per lane, or per thread of the block that shares the item
    if (SH == kByBlock) __syncthreads();
#pragma unroll
    for (int h = 0; h < kItemMax; h += 32) {
        const int e = h + lane;
        if (e >= ni || (SH == kByBlock && h != 32 * warp)) continue;
        float sum[3];
#pragma unroll
        for (int k = 0; k < (POT ? 1 : 3); ++k) {
            if (SH == kByBlock) {
                const WarpMem<CI, POT> *w = &S - warp;
                sum[k] = ((w[0].sum[k][e] + w[1].sum[k][e]) + w[2].sum[k][e]) + w[3].sum[k][e];
            } else {
                sum[k] = S.sum[k][SH != kByParts || parts == 1 ? e : 32 + lane];
            }
        }
        const int i = i0 + e;
        const float4 p = P.pos[i];
        if (POT) {
            P.phi_out[i] = 0.5f * P.G * p.w * sum[0];
        } else {
            const float gm = UM ? P.G * p.w : P.G;   // UM: p.w is every mass of the box
            float h_kick = P.h_kick, h_drift = P.h_drift;
            if (P.boxes) {
                h_kick = P.boxes[item.w].h;
                h_drift = P.boxes[item.w].post;
            }
            write_result(P, i, gm * sum[0], gm * sum[1], gm * sum[2], p.x, p.y, p.z, p.w, h_kick, h_drift, L);
        }
    }
    if (COUNT) {
        // every particle met itself once (t = eps), which is no pair
        unsigned long long c64 = cnt;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) c64 += __shfl_down_sync(0xffffffffu, c64, o);
        if (lane == 0) atomicAdd(P.within, P.eps < P.T && warp == 0 ? c64 - (unsigned long long)ni : c64);
        if (lane == 0 && P.evaluated) atomicAdd(P.evaluated, (unsigned long long)evals);
    }
    __syncwarp();
}

// Takes items from the queue of `counter` until none is left; with `mixed` it
// leaves those of the boxes whose masses call for the other form.
template <bool COUNT, bool POT, bool EPS0, bool UM, int F, bool CI, Sharing SH, bool FRAMES>
__device__ __forceinline__ void work_loop(const KParams &P, WarpMem<CI, POT> &S, int lane, int *counter, bool mixed) {
    const int n_items = uniform(*P.n_items);
    const int warp = SH == kByBlock ? uniform(threadIdx.x >> 5) : 0;
    __shared__ int claimed;
    while (true) {
        int it = 0;
        if (SH == kByBlock) {
            __syncthreads();   // the sums of the item before are read
            if (threadIdx.x == 0) claimed = atomicAdd(counter, 1);
            __syncthreads();
            it = uniform(claimed);
        } else {
            if (lane == 0) it = atomicAdd(counter, 1);
            it = __shfl_sync(0xffffffffu, it, 0);
        }
        if (it >= n_items) break;
        int4 item = P.items[P.order ? P.order[it] : it];
        item.x = uniform(item.x);
        item.y = uniform(item.y);
        item.z = uniform(item.z);
        item.w = uniform(item.w);
        if (mixed && (P.mass_flag[item.w >> 5] >> (item.w & 31) & 1u) == (UM ? 1u : 0u)) continue;
        process_item<COUNT, POT, EPS0, UM, F, CI, SH, FRAMES>(P, item, S, lane, warp);
    }
}

// FRAMES: boxes of fewer than 4 R cells a side, whose items may run in several frames.
// MINB: blocks per SM the register allocation must allow; F: steps of the
// pair loop unrolled.  The autotuner picks.  SH: the warps of a block share each
// item (calls of few items, see shared_items).
template <bool COUNT, bool POT, bool EPS0, int MINB, int F, bool CI, Sharing SH, bool FRAMES>
__global__ void __launch_bounds__(kThreads, MINB) k_sr_force(KParams P) {
    extern __shared__ __align__(16) char smem[];
    WarpMem<CI, POT> *S = reinterpret_cast<WarpMem<CI, POT> *>(smem) + uniform(threadIdx.x >> 5);
    const int lane = __shfl_xor_sync(0xffffffffu, (threadIdx.x & 31) ^ 1, 1);   // as with uniform(): kept
    // equal masses in a box (its bit left 0 by the binning pass): applied once per i.
    // The boxes of a batch take the form that each takes alone, in two rounds of the
    // queue where both occur (both forms in one loop spilled registers).
    constexpr bool kBatches = !CI && SH != kByBlock;   // forms that batches take too
    unsigned some = ~0u, every = ~0u;
    if (!kBatches && !POT && P.mass_flag) {
        some = uniform(*P.mass_flag);
        every = some ? ~0u : 0u;
    } else if (!POT && P.mass_flag) {
        some = 0u;
        for (int k = lane; 32 * k < P.nbox; k += 32) {
            const unsigned v = P.mass_flag[k];
            some |= v;
            every &= P.nbox - 32 * k < 32 ? v | ~0u << (P.nbox - 32 * k) : v;
        }
        some = __reduce_or_sync(0xffffffffu, some);
        every = __reduce_and_sync(0xffffffffu, every);
    }
    const bool mixed = kBatches && some && ~every;
    if (!POT && ~every) work_loop<COUNT, POT, EPS0, !POT, F, CI, SH, FRAMES>(P, *S, lane, P.work_counter, mixed);
    if (some) work_loop<COUNT, POT, EPS0, false, F, CI, SH, FRAMES>(P, *S, lane, P.work_counter + mixed, mixed);
}

template <bool COUNT, bool POT, bool EPS0, int MINB, int F, bool CI, Sharing SH = kWhole, bool FRAMES = false>
cudaError_t launch_one(const KParams &P, int num_sms, cudaStream_t s) {
    auto *k = k_sr_force<COUNT, POT, EPS0, MINB, F, CI, SH, FRAMES>;
    const size_t bytes = kWarps * sizeof(WarpMem<CI, POT>);
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kThreads, bytes);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    k<<<num_sms * per_sm, kThreads, bytes, s>>>(P);
    note_launch();
    return cudaGetLastError();
}

f32x2 doubled(float v) {
    uint32_t u;
    std::memcpy(&u, &v, sizeof u);
    return ((f32x2)u << 32) | u;
}

// Variants 0..kForceVariants-1: (MINB, F) = (5, 4), (4, 4), (5, 2), (4, 2);
// all give bitwise the same forces.
template <bool COUNT, bool EPS0>
cudaError_t launch_variant(const KParams &P, int variant, int num_sms, cudaStream_t s) {
    switch (variant) {
        case 1: return launch_one<COUNT, false, EPS0, 4, 4, false>(P, num_sms, s);
        case 2: return launch_one<COUNT, false, EPS0, 5, 2, false>(P, num_sms, s);
        case 3: return launch_one<COUNT, false, EPS0, 4, 2, false>(P, num_sms, s);
        default: return launch_one<COUNT, false, EPS0, 5, 4, false>(P, num_sms, s);
    }
}

// Shared items and items in several frames: one variant each, bitwise the same forces.
template <Sharing SH, bool FRAMES>
cudaError_t launch_form(const KParams &P, bool eps0, bool count, int num_sms, cudaStream_t s) {
    if (count)
        return eps0 ? launch_one<true, false, true, 4, 1, false, SH, FRAMES>(P, num_sms, s)
                    : launch_one<true, false, false, 4, 1, false, SH, FRAMES>(P, num_sms, s);
    return eps0 ? launch_one<false, false, true, 5, 4, false, SH, FRAMES>(P, num_sms, s)
                : launch_one<false, false, false, 5, 4, false, SH, FRAMES>(P, num_sms, s);
}

}  // namespace

cudaError_t sr_force_launch(const Geometry &g, const ForceConsts &fc, const ForceLaunch &fl, int num_sms,
                            cudaStream_t s) {
    const bool pot = fl.mode == kModePotential;
    if (!fl.counter_clear) {
        const cudaError_t e = cudaMemsetAsync(fl.work_counter, 0, sizeof(int), s);
        if (e != cudaSuccess) return e;
    }
    KParams P;
    P.pos = fl.pos;
    P.items = fl.items;
    P.order = fl.order;
    P.n_items = fl.n_items;
    P.cell_start = fl.cell_start;
    P.work_counter = fl.work_counter;
    P.nc = g.nc;
    P.R = g.R;
    P.cull = fl.cull ? 1 : 0;
    P.L = g.Lf;
    P.T = fc.T;
    P.eps = fc.eps;
    P.G = fc.G;
    P.pair = PairConsts{doubled(fc.eps),   doubled(-fc.q[0]), doubled(-fc.q[1]), doubled(-fc.q[2]),
                        doubled(-fc.q[3]), doubled(-fc.q[4]), doubled(-fc.q[5])};
    P.pot = PotConsts{doubled(-fc.u[0]), doubled(-fc.u[1]), doubled(-fc.u[2]), doubled(-fc.u[3]), doubled(-fc.u[4]),
                      doubled(-fc.u[5]), doubled(-fc.u[6]), doubled(-fc.phi0),  doubled(-1.0f)};
    P.mode = fl.mode;
    P.out = fl.out;
    P.perm = fl.perm;
    P.vel = fl.vel;
    P.pos_next = fl.pos_next;
    P.h_kick = fl.h_kick;
    P.h_drift = fl.h_drift;
    P.phi_out = fl.phi_out;
    P.within = fl.within;
    P.evaluated = fl.evaluated;
    P.mass_flag = fl.mass_flag;
    P.nbox = fl.nbox;
    P.boxes = fl.boxes;
    P.ids = fl.ids;
    P.pos_pool = fl.pos_pool;
    P.vel_pool = fl.vel_pool;
    P.flags = fl.flags;
    P.w = fl.w;
    P.levels = fl.levels;
    P.kick = fl.kick;
    P.delta = fl.delta;
    const bool eps0 = !(fc.eps > 0.0f);
    const bool count = fl.within != nullptr;
    const int v = fl.variant;
    if (fl.cell_offset && pot)
        return eps0 ? launch_one<false, true, true, 4, 4, true>(P, num_sms, s)
                    : launch_one<false, true, false, 4, 4, true>(P, num_sms, s);
    if (fl.cell_offset)
        return eps0 ? launch_one<false, false, true, 4, 4, true>(P, num_sms, s)
                    : launch_one<false, false, false, 4, 4, true>(P, num_sms, s);
    const bool frames = fl.boxes ? fl.frames : g.nc < 4 * g.R;
    if (pot && frames)
        return eps0 ? launch_one<false, true, true, 4, 4, false, kWhole, true>(P, num_sms, s)
                    : launch_one<false, true, false, 4, 4, false, kWhole, true>(P, num_sms, s);
    if (pot)
        return eps0 ? launch_one<false, true, true, 4, 4, false>(P, num_sms, s)
                    : launch_one<false, true, false, 4, 4, false>(P, num_sms, s);
    if (fl.sharing == kByBlock)
        return frames ? launch_form<kByBlock, true>(P, eps0, count, num_sms, s)
                      : launch_form<kByBlock, false>(P, eps0, count, num_sms, s);
    if (fl.sharing == kByParts)
        return frames ? launch_form<kByParts, true>(P, eps0, count, num_sms, s)
                      : launch_form<kByParts, false>(P, eps0, count, num_sms, s);
    if (frames) return launch_form<kWhole, true>(P, eps0, count, num_sms, s);
    if (count)
        return eps0 ? launch_one<true, false, true, 4, 1, false>(P, num_sms, s)
                    : launch_one<true, false, false, 4, 1, false>(P, num_sms, s);
    return eps0 ? launch_variant<false, true>(P, v, num_sms, s) : launch_variant<false, false>(P, v, num_sms, s);
}

// ---- FP64 diagnostics ------------------------------------------------------
namespace {
__global__ void __launch_bounds__(256) k_diag(int64_t n, const float4 *__restrict__ pos,
                                               const float4 *__restrict__ vel, const float *__restrict__ phi,
                                               double *out) {
    double s[5] = {0, 0, 0, 0, 0};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        float4 v = vel[i];
        double m = pos[i].w;
        s[0] += m * v.x;
        s[1] += m * v.y;
        s[2] += m * v.z;
        s[3] += 0.5 * m * ((double)v.x * v.x + (double)v.y * v.y + (double)v.z * v.z);
        s[4] += phi ? (double)phi[i] : 0.0;
    }
    __shared__ double red[5][8];
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        double x = s[k];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
        if (lane == 0) red[k][w] = x;
    }
    __syncthreads();
    if (threadIdx.x < 5) {
        double x = 0;
        for (int q = 0; q < (int)(blockDim.x / 32); ++q) x += red[threadIdx.x][q];
        atomicAdd(out + threadIdx.x, x);
    }
}
// Per box of a batch: block (box q, part k) sums part k of the box's sorted
// range (a fixed split into kDiagParts) in a fixed order; k_diag_combine adds
// the parts of each box in order.  Nothing depends on the other boxes.
__global__ void __launch_bounds__(256) k_diag_batch(const BoxDev *__restrict__ boxes,
                                                     const int32_t *__restrict__ cell_start,
                                                     const float4 *__restrict__ pos, const float4 *__restrict__ vel,
                                                     const float *__restrict__ phi, double *__restrict__ partial) {
    const int q = blockIdx.x / kDiagParts, part = blockIdx.x % kDiagParts;
    const BoxDev bx = boxes[q];
    const int64_t a = cell_start[bx.cell_base];
    const int64_t len = (int64_t)cell_start[bx.cell_base + bx.nc * bx.nc * bx.nc] - a;
    const int64_t lo = a + len * part / kDiagParts, hi = a + len * (part + 1) / kDiagParts;
    double s[5] = {0, 0, 0, 0, 0};
    for (int64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) {
        const float4 v = vel[i];
        const double m = pos[i].w;
        s[0] += m * v.x;
        s[1] += m * v.y;
        s[2] += m * v.z;
        s[3] += 0.5 * m * ((double)v.x * v.x + (double)v.y * v.y + (double)v.z * v.z);
        s[4] += (double)phi[i];
    }
    __shared__ double red[5][8];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        double x = s[k];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
        if (lane == 0) red[k][w] = x;
    }
    __syncthreads();
    if (threadIdx.x < 5) {
        double x = 0;
        for (int r = 0; r < (int)(blockDim.x / 32); ++r) x += red[threadIdx.x][r];
        partial[((int64_t)q * kDiagParts + part) * 5 + threadIdx.x] = x;
    }
}

__global__ void __launch_bounds__(256) k_diag_combine(int nbox, const BoxDev *__restrict__ boxes,
                                                       const double *__restrict__ partial, double *__restrict__ out) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)nbox * 5) return;
    const int q = (int)(t / 5), k = (int)(t % 5);
    double x = 0;
    for (int part = 0; part < kDiagParts; ++part) x += partial[((int64_t)q * kDiagParts + part) * 5 + k];
    out[(int64_t)boxes[q].orig * 5 + k] = x;
}

__global__ void __launch_bounds__(256) k_mass_moment_ci(int64_t n, const int32_t *__restrict__ cell,
                                                         const float4 *__restrict__ off, int nc, double w,
                                                         double *out) {
    double s[3] = {0, 0, 0};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t c = cell[i];
        const float4 o = off[i];
        const double m = o.w;
        s[0] += m * fma((double)(c % nc) + 0.5, w, (double)o.x);
        s[1] += m * fma((double)((c / nc) % nc) + 0.5, w, (double)o.y);
        s[2] += m * fma((double)(c / (nc * nc)) + 0.5, w, (double)o.z);
    }
    __shared__ double red[3][8];
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        double x = s[k];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
        if (lane == 0) red[k][wp] = x;
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        double x = 0;
        for (int r = 0; r < (int)(blockDim.x / 32); ++r) x += red[threadIdx.x][r];
        atomicAdd(out + threadIdx.x, x);
    }
}
}  // namespace

cudaError_t diag_reduce_batch(int nbox, const BoxDev *boxes, const int32_t *cell_start, const float4 *pos,
                              const float4 *vel, const float *phi, double *partial, double *out, cudaStream_t s) {
    if (nbox <= 0) return cudaSuccess;
    k_diag_batch<<<(unsigned)nbox * kDiagParts, 256, 0, s>>>(boxes, cell_start, pos, vel, phi, partial);
    note_launch();
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_diag_combine<<<(unsigned)((nbox * 5 + 255) / 256), 256, 0, s>>>(nbox, boxes, partial, out);
    note_launch();
    return cudaGetLastError();
}

cudaError_t diag_mass_moment_ci(int64_t n, const int32_t *cell, const float4 *off, int nc, double w, double *out,
                                cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    int blocks = (int)((n + 255) / 256);
    if (blocks > 1024) blocks = 1024;
    k_mass_moment_ci<<<blocks, 256, 0, s>>>(n, cell, off, nc, w, out);
    note_launch();
    return cudaGetLastError();
}

cudaError_t diag_reduce(int64_t n, const float4 *pos, const float4 *vel, const float *phi, double *out,
                        cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(out, 0, 5 * sizeof(double), s);
    if (e != cudaSuccess || n <= 0) return e;
    int blocks = (int)((n + 255) / 256);
    if (blocks > 1024) blocks = 1024;
    k_diag<<<blocks, 256, 0, s>>>(n, pos, vel, phi, out);
    note_launch();
    return cudaGetLastError();
}

}  // namespace hacc
