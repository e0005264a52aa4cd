// pp_cells.cu -- the particle step of the mixed form on particles sorted by
// cell at the start of every step (Sec. III: the paper sorts the particle
// array by cell position in every step, between the current deposit and the
// field update, so that steps 1-3 run as one sweep that accumulates the
// current in small cache-resident buffers).
//
// One CTA per 8x8x8 tile of cells.  Because every particle of the tile's sorted
// range sits in the tile, the E/B window staged in shared memory is the tile
// plus the gather's reach only (12^3 nodes per component, copied by six TMA
// tensor copies that complete on an mbarrier whose wait is bounded in time),
// the current window the tile plus the deposit's reach (13^3 nodes), and the
// particles of one cell are consecutive in memory.  Per chunk of up to 4096
// particles of one species:
//
//  phase 1, one thread per particle (a warp on 32 consecutive particles, i.e.
//    one or two cells): gather (eq:pfields), push (Vay / Boris, optional
//    radiative cooling), move; the new cell, offset and momentum go straight
//    back to the particle arrays (coalesced); the old offset and the
//    displacement are staged for the deposit.  The chunk passes through the
//    tile two planes of cells at a time, whose window is expanded into pairs
//    of neighbours along x: the gather is 192 broadcast 8-byte loads and 258
//    packed FMAs for a PCS particle (384 4-byte loads and 504 scalar FMAs
//    node by node).  A particle whose support start changes on some axis (it
//    crosses a support boundary) is queued, with the axis and direction of
//    the change.
//  pieces: the chunk is cut into pieces of at most 8 consecutive particles
//    of one deposit group (the particles of one cell, and for even orders of
//    one octant of it, share their support start on every axis); the queue
//    (in chunk order) into crossing pieces of at most 8 consecutive entries
//    of one group that change their support start on the same single axis
//    in the same direction (so they share the union support: a cold beam's
//    particles of one cell that cross into the next one).
//  phase 2, the charge-conserving current (eq:cc1, eq:jj3, Esirkepov's
//    decomposition written as the 2nd-order current by a per-particle prefix
//    sum): one thread per (piece, component) sums the O (O+1)^2 site values
//    of its particles in registers and adds them to the tile's current
//    window with one shared atomic per site (about 48 x 3 per piece instead of
//    per particle); a crossing piece likewise over its union support (at most
//    (O+1)^3 sites per component); a particle that crosses on several axes
//    takes the general union form, with shared atomics per nonzero site.  A
//    warp's 32 items always share the component.
//
// The current window holds int32 fixed point (native shared integer atomics):
// each chunk takes its unit from its particles' motion so that no node can
// overflow, and after the chunk the nodes its cells reach are added into the
// FP32 mesh (one global atomic per nonzero node).  A piece's sum is FP32 in
// registers and is rounded to the unit once.
//
// Bound by issue and by the shared-memory pipe behind it: on the cold beam 67
// warp-instructions a particle at 50 % of the issue slots, 62 % of the shared
// pipe.  64^3 thermal PCS, 16.8 M particles, 1.92 ms a step (2.62 with scalar
// gathers and sums, the spline weights of each position apart and a CTA per
// tile); 268 M particle beam 28.95 ms against 34.2.
#include "pp_sorted.cuh"
#include "pp_tma.cuh"

namespace pp {

namespace {

constexpr int kT = 8;                            // tile edge (cells)
constexpr int kTCells = kT * kT * kT;
constexpr int kRLo = 2, kRHi = 3;                // node reach below / above a cell (gather and deposit, O <= 3)
constexpr int kW = kT + kRLo + kRHi;             // 13 window nodes per axis
constexpr int kWVol = kW * kW * kW;              // words per window component
#ifndef PP_CELLS_THREADS
#define PP_CELLS_THREADS 512
#endif
constexpr int kCT = PP_CELLS_THREADS;            // threads per tile CTA
constexpr int kCW = kCT / 32;
// The E/B window the gather reads: nodes -2 .. 9 of the tile on each axis
// (a PCS support reaches two nodes either side of a particle's cell), one box
// of kWG^3 nodes per component copied by one TMA tensor copy (rows of 48
// bytes, a multiple of 16 as the copy requires), the six components kFComp
// words apart (128-byte aligned), then a 128-byte slot for the mbarrier the
// copies complete on.  The current window keeps kW nodes per axis: a particle
// that moves to the next cell deposits one node further up.
constexpr int kWG = kT + kRLo + 2;                             // 12
constexpr int kFComp = (kWG * kWG * kWG + 31) / 32 * 32;       // 1728 words
constexpr uint32_t kFBoxBytes = sizeof(float) * kWG * kWG * kWG;  // 6912 bytes per component
constexpr size_t kFieldBytes = sizeof(float) * 6 * kFComp + 128;
// The gather reads the window as pairs: every node with its neighbour along x,
// 12 pairs a row (the last one's neighbour is 0), so that a row of a support is
// one or two aligned 8-byte shared loads from any start.  The lanes of a warp
// sit in one or two cells: the loads are broadcasts, one wavefront each as a
// 4-byte load's are.  Shared memory holds the pairs of two planes of cells (six
// of nodes); the particles of a chunk, sorted by cell, pass through them in
// turn.  A step along x, y and z is 2, 24 and 16 words modulo the 32 banks, so
// that the up to eight starts that one cell's particles have (one per octant)
// fall in distinct banks.
constexpr int kPZ = 2;                                         // cell planes of the pairs
constexpr int kPRow = kWG, kPPlane = kWG * kPRow + 8, kPComp = (kPZ + 4) * kPPlane;   // in pairs
static_assert(kPRow * 2 % 32 == 24 && kPPlane * 2 % 32 == 16, "pair strides");
constexpr size_t kPairBytes = 6 * kPComp * 8;
// A staging wait that has not completed after this long gives up (ST_TIMEOUT).
constexpr uint64_t kStageWaitNs = 1000000000ull;
#ifndef PP_CELLS_CHUNK
#define PP_CELLS_CHUNK 4096
#endif
constexpr int kCC = PP_CELLS_CHUNK;              // particles staged per chunk
constexpr int kCPer = kCC / kCT;                 // phase-1 particles per thread per chunk
// Pieces of at most 8 particles: more register sums to add than with 16 or 32,
// but the deposit items spread evenly over the threads (64^3 thermal PCS:
// 2.60 ms at 8 or 12, 2.64 at 16, 2.92 at 32).
#ifndef PP_CELLS_PIECE
#define PP_CELLS_PIECE 8
#endif
constexpr int kPiece = PP_CELLS_PIECE;           // most particles per deposit piece
// Staged arrays hold one pad word per 16 particles: the lanes of a deposit warp
// read particles about one piece (16) apart, which unpadded would fall in two
// banks.
constexpr int kCS = kCC + kCC / 16;              // words per staged array
__device__ __forceinline__ int sp(int q) { return q + (q >> 4); }
// Group word of a staged particle: its deposit group (bits 0-11), its
// crossing signature (bits 12-14: 0 no support start changes; 1 + 2a + up for
// a change on axis a alone, up when it moves up; 7 for changes on several
// axes) and kSkip (not deposited by a piece of non-crossing particles).
constexpr uint16_t kSkip = 0x8000;
constexpr int kSigShift = 12;
constexpr uint16_t kGrpMask = 0x0fff, kSigMask = 0x7000;
static_assert(kCC % kCT == 0 && kCT % 32 == 0, "chunk must split evenly over the CTA");
static_assert(kCPer * kCW <= 1024, "piece-count table");
// counts (queue, -, pieces), box (6), totals (3); then four tables of
// per-(round, warp) counts and the crossing pieces per bucket (4)
constexpr int kMisc = 20 + 4 * kCPer * kCW;
// A crossing piece is stored as its first queue entry (12 bits) and its
// length - 1 (3 bits).
static_assert(kCC <= 4096 && kPiece <= 8, "crossing-piece word");
// The lists of pieces are built when the chunk's gathers are done: they take
// the place of the pairs.
static_assert(sizeof(uint16_t) * (3 * kCC + 4) <= kPairBytes, "piece lists");
constexpr size_t kCellsSmem = kFieldBytes + kPairBytes + sizeof(float) * (3 * kWVol + 6 * kCS) + sizeof(uint16_t) * kCC +
                              sizeof(int) * kMisc;
// The current window: an int32 fixed-point window whose unit each chunk takes
// from its particles' motion, flushed into the FP32 mesh per chunk; or, with
// PP_CELLS_FIXED=0, an FP32 window of shared FP32 atomics flushed once per
// tile.  Shared FP32 atomics measured about four times the shared-memory
// wavefronts of int32 ones here (64^3 thermal PCS: 4.67 against 2.51 ms).
#ifndef PP_CELLS_FIXED
#define PP_CELLS_FIXED 1
#endif
#if PP_CELLS_FIXED
using JT = int;
#else
using JT = float;
#endif
constexpr float kFixedRange = 1073741824.0f;    // 2^30
__device__ __forceinline__ void jadd(JT *p, float v) {
#if PP_CELLS_FIXED
    atomicAdd(p, __float2int_rn(v));
#else
    atomicAdd(p, v);
#endif
}
static_assert(kCellsSmem <= 227 * 1024, "tile CTA must fit the opt-in shared memory");

__device__ __forceinline__ int wi(int i, int j, int k) { return i + kW * (j + kW * k); }

// Rows of the window's pairs, for the gather.
struct PairRow {
    const f2 *q;
    template <bool both>
    __device__ __forceinline__ ulonglong2 pairs(int j, int k) const {
        const f2 *r = q + k * kPPlane + j * kPRow;
        return make_ulonglong2(r[0], both ? r[2] : 0);
    }
};
struct PairWindow {
    const f2 *q;   // at the node two below the particle's cell
    PP_IF_CHECKED(int rx, ry, rz, O; int *status;)
    __device__ __forceinline__ PairRow operator()(int comp, int x, int y, int z) const {
        PP_IF_CHECKED(if (rx + x + 2 * (O >= 2) >= kPRow || ry + y + O >= kWG || rz + z + O >= kPZ + 4) {
            atomicOr(status, ST_BOUNDS);
            return PairRow{q};
        })
        return PairRow{q + comp * kPComp + z * kPPlane + y * kPRow + x};
    }
};

// Current accessor over the FP32 shared window (frame = the particle's cell).
struct CellsCurrentAcc {
    JT *J;
    int base;
    PP_IF_CHECKED(int wx = 0, wy = 0, wz = 0; int *st = nullptr; mutable int bad = 0;)
#ifdef PP_CHECKED
    __device__ __forceinline__ bool inside(int i, int j, int k) const {
        return wx + i >= 0 && wx + i < kW && wy + j >= 0 && wy + j < kW && wz + k >= 0 && wz + k < kW;
    }
    __device__ ~CellsCurrentAcc() {
        if (bad && st) atomicOr(st, ST_BOUNDS);
    }
#endif
    __device__ __forceinline__ void addJ(int comp, int i, int j, int k, float v) const {
        PP_IF_CHECKED(if (!inside(i, j, k)) { bad = 1; return; })
        jadd(J + comp * kWVol + base + wi(i, j, k), v);
    }
};

using CellsSpecies = SortedSpecies;

struct CellsArgs : SortedArgs {
    CUtensorMap tmap[6];         // E_x, E_y, E_z, B_x, B_y, B_z: boxes of kWG^3 nodes
};

// Deposit group of a particle: its cell in the tile, and for even orders the
// octant of the cell it sits in (the support start on integer nodes is
// floor(xi - (O-1)/2), which for even O depends on which half of the cell
// holds xi).
template <int O>
__device__ __forceinline__ int group_of(int rx, int ry, int rz, const float (&xi)[3]) {
    const int cell = rx + kT * (ry + kT * rz);
    if constexpr (O % 2 == 0) {
        const int oct = (xi[0] >= 0.5f ? 1 : 0) | (xi[1] >= 0.5f ? 2 : 0) | (xi[2] >= 0.5f ? 4 : 0);
        return (cell << 3) | oct;
    } else {
        return cell;
    }
}

// Window coordinates of the group's cell and of its support start.
template <int O>
__device__ __forceinline__ void group_frame(int grp, int (&cw)[3], int (&lo)[3]) {
    const int cell = (O % 2 == 0) ? (grp >> 3) : grp;
    const int r[3] = {cell & (kT - 1), (cell / kT) & (kT - 1), cell / (kT * kT)};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        cw[d] = r[d] + kRLo;
        if constexpr (O % 2 == 0) lo[d] = cw[d] - (O - 2) / 2 - 1 + ((grp >> d) & 1);
        else lo[d] = cw[d] - (O - 1) / 2;
    }
}

// Old and new fractional coordinates along the axes, from the offset x0 and the
// displacement d of a particle whose old support starts at the group's start
// (coordinate 0 of the support: the cell for odd orders, the middle of the cell
// or of the one below for even ones) and whose new one starts `step` nodes up.
template <int O>
__device__ __forceinline__ float group_origin(int grp, int axis) {
    return O % 2 == 0 ? (((grp >> axis) & 1) ? 0.5f : -0.5f) : 0.0f;
}

// Prefix of dS along the current's axis on the lower faces, suffix on the upper
// ones (they sum to zero), times the scale.
template <int O, int NA, int N>
__device__ __forceinline__ void face_prefix(const float (&DS)[N], float jscale, float (&C)[NA]) {
    float run = 0.0f;
#pragma unroll
    for (int m = 0; m < NA; ++m) {
        if (2 * m < O + 1) {
            run += DS[m];
            C[m] = run * jscale;
        }
    }
    run = 0.0f;
#pragma unroll
    for (int m = NA - 1; m >= 0; --m) {
        if (2 * m >= O + 1) {
            run -= DS[m + 1];
            C[m] = run * jscale;
        }
    }
}

// Component A of the current of the piece [s, e): the particles that cross no
// support boundary (flag clear) share the support start lo, so their
// O (O+1)^2 site values (those of deposit_esirkepov_inner, site by site) are
// summed in registers, two nodes of axis B to a packed pair, and added once.
template <int O, int A>
__device__ __forceinline__ void piece_current(JT *Jw, const float *s_o, const float *s_d, const uint16_t *s_grp,
                                              int s, int e, float jscale PP_IF_CHECKED(, int *st)) {
    constexpr int Bx = (A + 1) % 3, Cx = (A + 2) % 3, NP = (O + 2) / 2;
    const int grp = s_grp[s] & kGrpMask;
    int cw[3], lo[3];
    group_frame<O>(grp, cw, lo);
    f2 acc[O][NP][O + 1];
#pragma unroll
    for (int m = 0; m < O; ++m)
#pragma unroll
        for (int mb = 0; mb < NP; ++mb)
#pragma unroll
            for (int mc = 0; mc <= O; ++mc) acc[m][mb][mc] = 0;
#pragma unroll 1
    for (int q = s; q < e; ++q) {
        if (s_grp[q] & kSkip) continue;
        float S0[3][O + 1], DS[3][O + 1];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const float x0 = s_o[d * kCS + sp(q)];
            const float x1 = x0 + s_d[d * kCS + sp(q)], org = group_origin<O>(grp, d);
            float wn[O + 1];
            bspline2<O>(x0 - org, x1 - org, S0[d], wn);
#pragma unroll
            for (int m = 0; m <= O; ++m) DS[d][m] = wn[m] - S0[d][m];
        }
        float C[O];
        face_prefix<O, O>(DS[A], jscale, C);
        f2 sb[NP], db[NP];
#pragma unroll
        for (int mb = 0; mb < NP; ++mb) {
            sb[mb] = pack2(S0[Bx][2 * mb], 2 * mb < O ? S0[Bx][2 * mb + 1] : 0.0f);
            db[mb] = pack2(DS[Bx][2 * mb], 2 * mb < O ? DS[Bx][2 * mb + 1] : 0.0f);
        }
#pragma unroll
        for (int mc = 0; mc <= O; ++mc) {
            const f2 p = dup2(S0[Cx][mc] + 0.5f * DS[Cx][mc]);
            const f2 h = dup2(0.5f * S0[Cx][mc] + (1.0f / 3.0f) * DS[Cx][mc]);
#pragma unroll
            for (int mb = 0; mb < NP; ++mb) {
                const f2 Y = fma2(sb[mb], p, mul2(db[mb], h));
#pragma unroll
                for (int m = 0; m < O; ++m) acc[m][mb][mc] = fma2(dup2(C[m]), Y, acc[m][mb][mc]);
            }
        }
    }
#pragma unroll
    for (int m = 0; m < O; ++m)
#pragma unroll
        for (int mb = 0; mb <= O; ++mb)
#pragma unroll
            for (int mc = 0; mc <= O; ++mc) {
                int idx[3];
                idx[A] = lo[A] + m;
                idx[Bx] = lo[Bx] + mb;
                idx[Cx] = lo[Cx] + mc;
#ifdef PP_CHECKED
                if (idx[0] < 0 || idx[0] >= kW || idx[1] < 0 || idx[1] >= kW || idx[2] < 0 || idx[2] >= kW) {
                    atomicOr(st, ST_BOUNDS);
                    continue;
                }
#endif
                float v[2];
                unpack2(acc[m][mb / 2][mc], v[0], v[1]);
                jadd(Jw + A * kWVol + wi(idx[0], idx[1], idx[2]), v[mb % 2]);
            }
}

// Component A of the current of a particle whose support start moves on
// several axes: the general form on the union of its old and new supports
// (O + 2 nodes per axis).  Rare (a few particles per thousand even in a hot
// plasma), so kept out of line: the tile loop's code stays small enough for
// the instruction cache.
template <int O, int A>
__device__ __noinline__ void queued_current(JT *Jw, const float *s_o, const float *s_d, const uint16_t *s_grp,
                                               int q, float jscale PP_IF_CHECKED(, int *st)) {
    int cw[3], lo0[3];
    group_frame<O>(s_grp[q] & kGrpMask, cw, lo0);
    float xi0[3], xi1[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        xi0[d] = s_o[d * kCS + sp(q)];
        xi1[d] = xi0[d] + s_d[d * kCS + sp(q)];
    }
    CellsCurrentAcc acc{Jw, wi(cw[0], cw[1], cw[2])};
    PP_IF_CHECKED(acc.wx = cw[0]; acc.wy = cw[1]; acc.wz = cw[2]; acc.st = st;)
    float S0[3][O + 2], DS[3][O + 2];
    int lo[3];
    esirkepov_weights<O, float>(xi0, xi1, S0, DS, lo);
    esirkepov_component<O, float, A>(acc, S0, DS, lo, jscale);
}

// Component A of the current of a crossing piece: particles of one deposit
// group whose support start moves one node along axis XA alone, all in the
// same direction (up: to the next node), so that they share the union support
// (O + 2 nodes along XA, O + 1 along the others).  Their site values are those
// of the general union form (esirkepov_weights + esirkepov_component, site by
// site the same products; its sites that are zero for such a particle are
// left out here): NA faces along A (O + 1 when A is the crossing axis, else O,
// the last face being zero) times the union nodes across.  They are summed in
// registers over the piece and added once per site.  The work is written in
// axes rotated so that the crossing axis comes first (rotated axis r is axis
// (r + XA) mod 3, RA the rotated A), so that one body serves all three
// crossing axes.
template <int O, int RA>
__device__ __forceinline__ void cross_piece(JT *Jw, int A, int XA, const float *s_o, const float *s_d,
                                            const uint16_t *s_queue, int ks, int ke, int grp, bool up,
                                            float jscale PP_IF_CHECKED(, int *st)) {
    constexpr int RB = (RA + 1) % 3, RC = (RA + 2) % 3;
    constexpr int NA = (RA == 0) ? O + 1 : O;
    // pairs run along an axis that is not the crossing one: B, or C where B is
    constexpr bool kPairC = RB == 0;
    constexpr int RP = kPairC ? RC : RB, RS = kPairC ? RB : RC;   // axes of the pairs and of the single nodes
    constexpr int NP = (O + 2) / 2, NS = (RS == 0) ? O + 2 : O + 1;
    int cw[3], lo[3];
    group_frame<O>(grp, cw, lo);
    const int p[3] = {XA, XA == 2 ? 0 : XA + 1, XA == 0 ? 2 : XA - 1};   // physical axis of rotated axis r
    int lr[3], sr[3];   // support start and window stride per rotated axis
    float org[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        lr[r] = p[r] == 0 ? lo[0] : (p[r] == 1 ? lo[1] : lo[2]);
        sr[r] = p[r] == 0 ? 1 : (p[r] == 1 ? kW : kW * kW);
        org[r] = group_origin<O>(grp, p[r]);
    }
    lr[0] -= up ? 0 : 1;   // union start along the crossing axis: the lower of the old and new starts
    const float step = up ? 1.0f : -1.0f;
    f2 acc[NA][NP][NS];
#pragma unroll
    for (int m = 0; m < NA; ++m)
#pragma unroll
        for (int mp = 0; mp < NP; ++mp)
#pragma unroll
            for (int ms = 0; ms < NS; ++ms) acc[m][mp][ms] = 0;
#pragma unroll 1
    for (int e = ks; e < ke; ++e) {
        const int q = s_queue[e];
        float S0[3][O + 2], DS[3][O + 2];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const float x0 = s_o[p[r] * kCS + sp(q)];
            const float x1 = x0 + s_d[p[r] * kCS + sp(q)];
            float wo[O + 1], wn[O + 1];
            bspline2<O>(x0 - org[r], r == 0 ? x1 - org[r] - step : x1 - org[r], wo, wn);
            if (r == 0) {   // old weights from the union start (up) or one node above it
#pragma unroll
                for (int m = 0; m < O + 2; ++m) {
                    const float a0 = up ? (m <= O ? wo[m] : 0.0f) : (m >= 1 ? wo[m - 1] : 0.0f);
                    const float a1 = up ? (m >= 1 ? wn[m - 1] : 0.0f) : (m <= O ? wn[m] : 0.0f);
                    S0[r][m] = a0;
                    DS[r][m] = a1 - a0;
                }
            } else {
#pragma unroll
                for (int m = 0; m <= O; ++m) {
                    S0[r][m] = wo[m];
                    DS[r][m] = wn[m] - wo[m];
                }
                S0[r][O + 1] = 0.0f;
                DS[r][O + 1] = 0.0f;
            }
        }
        float C[NA];
        face_prefix<O, NA>(DS[RA], jscale, C);
        f2 sb[NP], db[NP];
#pragma unroll
        for (int mp = 0; mp < NP; ++mp) {
            sb[mp] = pack2(S0[RP][2 * mp], S0[RP][2 * mp + 1]);
            db[mp] = pack2(DS[RP][2 * mp], DS[RP][2 * mp + 1]);
        }
#pragma unroll
        for (int ms = 0; ms < NS; ++ms) {
            const f2 pc = dup2(S0[RS][ms] + 0.5f * DS[RS][ms]);
            const f2 hc = dup2(0.5f * S0[RS][ms] + (1.0f / 3.0f) * DS[RS][ms]);
#pragma unroll
            for (int mp = 0; mp < NP; ++mp) {
                const f2 Y = fma2(sb[mp], pc, mul2(db[mp], hc));
#pragma unroll
                for (int m = 0; m < NA; ++m) acc[m][mp][ms] = fma2(dup2(C[m]), Y, acc[m][mp][ms]);
            }
        }
    }
    JT *J = Jw + A * kWVol;
#pragma unroll
    for (int m = 0; m < NA; ++m)
#pragma unroll
        for (int mp = 0; mp <= O; ++mp)
#pragma unroll
            for (int ms = 0; ms < NS; ++ms) {
#ifdef PP_CHECKED
                if (lr[RA] + m < 0 || lr[RA] + m >= kW || lr[RP] + mp < 0 || lr[RP] + mp >= kW || lr[RS] + ms < 0 ||
                    lr[RS] + ms >= kW) {
                    atomicOr(st, ST_BOUNDS);
                    continue;
                }
#endif
                float v[2];
                unpack2(acc[m][mp / 2][ms], v[0], v[1]);
                jadd(J + (lr[RA] + m) * sr[RA] + (lr[RP] + mp) * sr[RP] + (lr[RS] + ms) * sr[RS], v[mp % 2]);
            }
}

// Component A of the current of the crossing piece [ks, ke) of the queue, of
// bucket xa: the crossing axis (cross_piece), or 3 for a single particle whose
// support start moves on several axes (the general union form).
template <int O>
__device__ __forceinline__ void xpiece_current(JT *Jw, int A, const float *s_o, const float *s_d,
                                               const uint16_t *s_grp, const uint16_t *s_queue, int ks, int ke, int xa,
                                               float jscale PP_IF_CHECKED(, int *st)) {
    if (xa == 3) {
        if (A == 0) queued_current<O, 0>(Jw, s_o, s_d, s_grp, s_queue[ks], jscale PP_IF_CHECKED(, st));
        else if (A == 1) queued_current<O, 1>(Jw, s_o, s_d, s_grp, s_queue[ks], jscale PP_IF_CHECKED(, st));
        else queued_current<O, 2>(Jw, s_o, s_d, s_grp, s_queue[ks], jscale PP_IF_CHECKED(, st));
        return;
    }
    const int g0 = s_grp[s_queue[ks]];
    const bool up = (((g0 & kSigMask) >> kSigShift) & 1) == 0;   // signature 1 + 2 xa + up
    const int grp = g0 & kGrpMask;
    const int ra = A >= xa ? A - xa : A - xa + 3;
    if (ra == 0) cross_piece<O, 0>(Jw, A, xa, s_o, s_d, s_queue, ks, ke, grp, up, jscale PP_IF_CHECKED(, st));
    else if (ra == 1) cross_piece<O, 1>(Jw, A, xa, s_o, s_d, s_queue, ks, ke, grp, up, jscale PP_IF_CHECKED(, st));
    else cross_piece<O, 2>(Jw, A, xa, s_o, s_d, s_queue, ks, ke, grp, up, jscale PP_IF_CHECKED(, st));
}

__device__ __forceinline__ unsigned lanemask_lt_() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Exclusive scan, in chunk order, of the per-(round, warp) counts
// c[0 .. kCPer kCW) by one warp; the total goes to *total.
__device__ __forceinline__ void scan_counts(int *c, int *total, int lane) {
    constexpr int kPerLane = (kCPer * kCW + 31) / 32;
    int v[kPerLane], sum = 0;
#pragma unroll
    for (int m = 0; m < kPerLane; ++m) {
        const int k = lane * kPerLane + m;
        v[m] = k < kCPer * kCW ? c[k] : 0;
        sum += v[m];
    }
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    int run = incl - sum;
#pragma unroll
    for (int m = 0; m < kPerLane; ++m) {
        const int k = lane * kPerLane + m;
        if (k < kCPer * kCW) c[k] = run;
        run += v[m];
    }
    if (lane == 31) *total = incl;
}

// BND: walls (reflection) and the open end (escape); a separate instantiation
// so that periodic runs carry none of their tests.
// One tile of one run: the whole particle step of the tile's particles of one
// species (item: tile times species, plus the species), its current added into
// the run's mesh.  Called by every thread of the CTA; smem is the CTA's dynamic
// shared memory.  The chunks of the species are independent, so a species to a
// CTA changes no sum but makes twice the blocks of a two-species plasma, of half
// the length: 128 CTAs instead of 64 at 32^3 cells (20 steps 6.52 -> 4.58 ms), a
// shorter last wave at 64^3 (2.25 -> 1.99 ms a step); where the blocks are many, a
// second staging of the window costs 0.4 % (268 M particle beam).
// Returns false when the CTA must stop: a staging wait ran out (here or in
// another CTA, ST_TIMEOUT).  phase: parity of the CTA's staging mbarrier, which
// the kernel initialised.  GMAPS: the tensor maps sit in global memory.
template <int O, int PUSH, bool BND, bool GMAPS>
__device__ __forceinline__ bool cells_tile(const CellsArgs &T, const int item, float *smem, uint32_t &phase) {
    float *F = smem;
    uint64_t *bar = (uint64_t *)((char *)smem + kFieldBytes - 128);
    f2 *Fp = (f2 *)((char *)smem + kFieldBytes);       // pairs of the gather, then the lists of pieces
    JT *Jw = (JT *)((char *)smem + kFieldBytes + kPairBytes);
    float *s_o = (float *)(Jw + 3 * kWVol);   // 3 x kCS: offsets at t (frame of the cell)
    float *s_d = s_o + 3 * kCS;           // 3 x kCS: displacement of the step
    uint16_t *s_grp = (uint16_t *)(s_d + 3 * kCS);   // group word (deposit group, crossing, kSkip)
    uint16_t *s_piece = (uint16_t *)Fp;               // piece starts (+ the end)
    uint16_t *s_queue = s_piece + kCC + 2;            // crossing particles, in chunk order
    uint16_t *s_xpiece = s_queue + kCC;               // crossing pieces by bucket: first entry | (length - 1) << 12
    int *misc = (int *)(s_grp + kCC);   // [0]: queue length; [2]: pieces;
                                               // [10..12]: fixed point: sum |dxi|
    int *cnt = misc + 16;                 // starts per (round, warp); four tables
    int *qcnt = cnt + kCPer * kCW;        // crossing particles per (round, warp)
    int *xtot = cnt + 4 * kCPer * kCW;    // crossing pieces per bucket
    const Geom &g = T.g;
    const int tile = item / T.ns, s = item - tile * T.ns;
    const CellsSpecies &S = T.sp[s];
    const int tx = tile % T.nt[0], ty = (tile / T.nt[0]) % T.nt[1], tz = tile / (T.nt[0] * T.nt[1]);
    const int ox = tx * kT, oy = ty * kT, oz = tz * kT;
    const int wx = ox - kRLo, wy = oy - kRLo, wz = oz - kRLo;
    const int64_t key0 = (int64_t)tile * kTCells * kSubKeys, key1 = key0 + kTCells * kSubKeys;
    // a tile that holds no particle (the mirror half of a box between walls) stages nothing
    if (S.cell_start[key1] == S.cell_start[key0]) return true;
    // ---- the E/B window by six TMA tensor copies (array coordinates of the
    // window's first node; the host checked that every tile's box lies inside
    // the padded arrays with an aligned x; rechecked here, uniformly, so that
    // no copy can start misaligned or outside)
    const int x0 = wx + g.G, y0 = wy + g.G, z0 = wz + g.G;
    if ((x0 & 3) || x0 < 0 || y0 < 0 || z0 < 0 || x0 + kWG > g.P[0] || y0 + kWG > g.P[1] || z0 + kWG > g.P[2]) {
        if (threadIdx.x == 0) atomicOr(T.status, ST_BOUNDS);
        return true;
    }
    if (threadIdx.x == 0) {
        // a CTA whose wait ran out stops the others at their next tile
        misc[3] = (*(volatile int *)T.status & ST_TIMEOUT) != 0;
        if (misc[3]) {
            mbar_arrive(bar);
        } else {
            fence_proxy_async_smem();   // the previous tile's reads of F come before the copies' writes
            mbar_arrive_expect(bar, 6 * kFBoxBytes);
#pragma unroll
            for (int c = 0; c < 6; ++c) {
                if (GMAPS) fence_tensormap_acquire(&T.tmap[c]);
                tma_load_3d(F + c * kFComp, &T.tmap[c], x0, y0, z0, bar);
            }
        }
    }
    for (int idx = threadIdx.x; idx < 3 * kWVol; idx += kCT) Jw[idx] = 0;
    // the window has arrived: waited for behind the first particles' loads, two
    // dependent trips to memory that otherwise start only then (beam 29.37 ->
    // 28.95 ms per step, 192^3 Weibel 18.95 -> 18.55)
    bool staged = false;

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    {
        int sb[kT / kPZ + 1];   // the slabs' first particles
#pragma unroll
        for (int m = 0; m <= kT / kPZ; ++m) sb[m] = S.cell_start[key0 + m * kPZ * kT * kT * kSubKeys];
        const int tb = sb[0], te = sb[kT / kPZ];
        for (int cb = tb; cb < te; cb += kCC) {
            const int cn = min(kCC, te - cb);
#if PP_CELLS_FIXED
            float sum[3] = {0.0f, 0.0f, 0.0f};
            int zlo = kT, zhi = -1;   // cell planes of the chunk's slabs
#endif
            // ---- phase 1: gather, push, move; write back; stage the deposit
            // the particle of the next round is fetched (through the pending
            // permutation) before the current one is computed, so that its
            // dependent global loads overlap the gather
            int32_t n_cw = 0;
            float n_o[3] = {0.0f, 0.0f, 0.0f}, n_u[3] = {0.0f, 0.0f, 0.0f};
            auto fetch = [&](int qf, int end) {
                if (qf >= end) return;
                const int64_t i = (int64_t)cb + qf;
                const int64_t src = S.perm ? (int64_t)S.perm[i] : i;
                n_cw = S.p.cell[src];
                n_o[0] = S.p.ox[src]; n_o[1] = S.p.oy[src]; n_o[2] = S.p.oz[src];
                n_u[0] = S.p.ux[src]; n_u[1] = S.p.uy[src]; n_u[2] = S.p.uz[src];
            };
#pragma unroll 1
            for (int slab = 0; slab < kT / kPZ; ++slab) {
                int s0 = sb[0], s1 = sb[1];   // sb[slab], sb[slab + 1] without a run-time index
#pragma unroll
                for (int m = 1; m < kT / kPZ; ++m)
                    if (slab == m) {
                        s0 = sb[m];
                        s1 = sb[m + 1];
                    }
                const int qa = max(cb, s0) - cb, qe = min(cb + cn, s1) - cb;
                if (qa >= qe) continue;
#if PP_CELLS_FIXED
                zlo = min(zlo, slab * kPZ);
                zhi = slab * kPZ + kPZ - 1;
#endif
                fetch(qa + threadIdx.x, qe);
                if (!staged) {
                    if (!cta_wait_bounded(bar, phase, kStageWaitNs, T.status)) return false;
                    phase ^= 1;
                    if (misc[3]) return false;
                    staged = true;
                }
                __syncthreads();   // the last slab's gathers, or the last chunk's pieces, are done
                for (int t = threadIdx.x; t < 6 * (kPZ + 4) * kWG; t += kCT) {   // window rows to pairs
                    const int c = t / ((kPZ + 4) * kWG), r = t - c * (kPZ + 4) * kWG;
                    const float4 *src = reinterpret_cast<const float4 *>(F + c * kFComp + (slab * kPZ * kWG + r) * kWG);
                    float4 *dst = reinterpret_cast<float4 *>(Fp + c * kPComp + (r / kWG) * kPPlane + (r % kWG) * kPRow);
                    const float4 a = src[0], b = src[1], d = src[2];
                    dst[0] = make_float4(a.x, a.y, a.y, a.z);
                    dst[1] = make_float4(a.z, a.w, a.w, b.x);
                    dst[2] = make_float4(b.x, b.y, b.y, b.z);
                    dst[3] = make_float4(b.z, b.w, b.w, d.x);
                    dst[4] = make_float4(d.x, d.y, d.y, d.z);
                    dst[5] = make_float4(d.z, d.w, d.w, 0.0f);
                }
                __syncthreads();
#pragma unroll 1
                for (int q = qa + threadIdx.x; q < qe; q += kCT) {
                    const int64_t idx = (int64_t)cb + q;
                    const int32_t cw0 = n_cw;
                    const float xi0[3] = {n_o[0], n_o[1], n_o[2]};
                    float u[3] = {n_u[0], n_u[1], n_u[2]};
                    fetch(q + kCT, qe);
                    int cc[3];
                    unpack_cell(cw0, cc[0], cc[1], cc[2]);
                    int rx = cc[0] - ox, ry = cc[1] - oy, rz = cc[2] - oz - slab * kPZ;
                    const bool here = (unsigned)rx < (unsigned)kT && (unsigned)ry < (unsigned)kT && (unsigned)rz < (unsigned)kPZ;
                    if (!here) rx = ry = rz = 0;
                    const float u0[3] = {u[0], u[1], u[2]};
                    const int grp = group_of<O>(rx, ry, rz + slab * kPZ, xi0);
                    if (S.qmdt != 0.0f) {   // uniform: no kick, no force
                        float E[3] = {0.0f, 0.0f, 0.0f}, B[3] = {0.0f, 0.0f, 0.0f};
                        gather_pairs<O>(PairWindow{Fp + rz * kPPlane + ry * kPRow + rx PP_IF_CHECKED(, rx, ry, rz, O, T.status)},
                                        xi0, E, B);
                        push_particle<PUSH, float>(S.qmdt, S.kdt, E, B, u);
                    }
                    const float gi = inv_sqrt(1.0f + u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
                    float dx[3], xi1[3];
                    bool ok = here;
                    int ncross = 0, xa = 0;
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        dx[d] = T.dtdx[d] * u[d] * gi;
                        xi1[d] = xi0[d] + dx[d];
                        ok = ok && (fabsf(dx[d]) < 1.0f);
                        if (floorf(xi0[d] - 0.5f * (O - 1)) != floorf(xi1[d] - 0.5f * (O - 1))) {
                            ++ncross;
                            xa = d;
                        }
                    }
                    if (!ok) {
                        // not in its sorted place (cannot happen after a sort), a cell or more in one
                        // step, or not finite: left unchanged, and the step flagged
                        atomicOr(T.status, !here ? ST_RANGE : (isfinite(u[0] + u[1] + u[2]) ? ST_CFL : ST_NAN));
                        s_grp[q] = (uint16_t)(grp | kSkip);
                        store_sorted(T, S, idx, cw0, xi0, u0);
                        continue;
                    }
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        s_o[d * kCS + sp(q)] = xi0[d];
                        s_d[d * kCS + sp(q)] = dx[d];
                    }
#if PP_CELLS_FIXED
                    sum[0] += fabsf(dx[0]); sum[1] += fabsf(dx[1]); sum[2] += fabsf(dx[2]);
#endif
                    // crossing signature: the axis and direction of a support start
                    // that moves on one axis alone, 7 when it moves on several
                    const float dxa = xa == 0 ? dx[0] : (xa == 1 ? dx[1] : dx[2]);
                    const int sig = ncross == 0 ? 0 : (ncross == 1 ? 1 + 2 * xa + (dxa > 0.0f ? 1 : 0) : 7);
                    s_grp[q] = (uint16_t)(grp | (sig << kSigShift) | (ncross ? kSkip : 0));
                    // the new state, written to the slot (the deposit reads the staged copy): the
                    // offset back into [0, 1), the cell wrapped
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        const float fl = floorf(xi1[d]);
                        xi1[d] -= fl;
                        int c = cc[d] + (int)fl;
                        if (xi1[d] >= 1.0f) {   // a small negative offset that rounds to 1
                            xi1[d] = 0.0f;
                            ++c;
                        }
                        c = c < 0 ? c + g.n[d] : c;
                        cc[d] = c >= g.n[d] ? c - g.n[d] : c;
                    }
                    int32_t cwd = pack_cell(cc[0], cc[1], cc[2]);
                    if constexpr (BND) {
                        reflect(cc[0], xi1[0], u[0], T.wall[0]);
                        reflect(cc[1], xi1[1], u[1], T.wall[1]);
                        reflect(cc[2], xi1[2], u[2], T.wall[2]);
                        cwd = pack_cell(cc[0], cc[1], cc[2]);
                        if (T.esc > 0.0 && (double)cc[0] + (double)xi1[0] < T.esc && u[0] < 0.0f) cwd |= kDeadBit;
                    }
                    store_sorted(T, S, idx, cwd, xi1, u);
                }
            }
#if PP_CELLS_FIXED
            // the previous chunk's values were last read before the barrier above
            if (threadIdx.x < 3) ((float *)misc)[10 + threadIdx.x] = 0.0f;
            __syncthreads();
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                float sd = sum[d];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) sd += __shfl_xor_sync(0xffffffffu, sd, o);
                if (lane == 0) atomicAdd((float *)misc + 10 + d, sd);
            }
#endif
            __syncthreads();
            // ---- pieces of non-crossing particles: starts at a group change and
            // every kPiece-th particle; crossing particles into the queue, in chunk
            // order (both by ballots and a scan of the per-(round, warp) counts)
            unsigned ball[kCPer], qball[kCPer];
#pragma unroll
            for (int r = 0; r < kCPer; ++r) {
                const int q = r * kCT + threadIdx.x;
                bool st = false, cr = false;
                if (q < cn) {
                    const int gq = s_grp[q];
                    st = q % kPiece == 0 || ((gq ^ s_grp[q - 1]) & kGrpMask) != 0;
                    cr = (gq & kSigMask) != 0;
                }
                ball[r] = __ballot_sync(0xffffffffu, st);
                qball[r] = __ballot_sync(0xffffffffu, cr);
                if (lane == 0) {
                    cnt[r * kCW + warp] = __popc(ball[r]);
                    qcnt[r * kCW + warp] = __popc(qball[r]);
                }
            }
            __syncthreads();
            if (warp == 0) scan_counts(cnt, misc + 2, lane);
            else if (warp == 1) scan_counts(qcnt, misc + 0, lane);
            __syncthreads();
#pragma unroll
            for (int r = 0; r < kCPer; ++r) {
                const int q = r * kCT + threadIdx.x;
                const unsigned below = lanemask_lt_();
                if (ball[r] & (1u << lane)) s_piece[cnt[r * kCW + warp] + __popc(ball[r] & below)] = (uint16_t)q;
                if (qball[r] & (1u << lane)) s_queue[qcnt[r * kCW + warp] + __popc(qball[r] & below)] = (uint16_t)q;
            }
            if (threadIdx.x == 0) s_piece[misc[2]] = (uint16_t)cn;
            __syncthreads();
            // ---- crossing pieces over the queue: starts at a change of group or
            // crossing, at a particle crossing on several axes and after one, and
            // every kPiece-th entry.  They are listed by bucket (the crossing axis,
            // or 3 for several axes), so that the 32 items of a warp take one form.
            const int nq = misc[0];
            auto xstart = [&](int k) {
                const int gk = s_grp[s_queue[k]];
                if (k % kPiece == 0 || (gk & kSigMask) == kSigMask) return true;
                const int gp = s_grp[s_queue[k - 1]];
                return (gp & kSigMask) == kSigMask || ((gk ^ gp) & (kGrpMask | kSigMask)) != 0;
            };
            int xflag = 0;   // per round: bit 2 start, bits 0-1 bucket
#pragma unroll
            for (int r = 0; r < kCPer; ++r) {
                const int k = r * kCT + threadIdx.x;
                int f = 0;
                if (k < nq && xstart(k)) f = 4 | ((((s_grp[s_queue[k]] & kSigMask) >> kSigShift) - 1) >> 1);
                xflag |= f << (3 * r);
#pragma unroll
                for (int bk = 0; bk < 4; ++bk) {
                    const unsigned m = __ballot_sync(0xffffffffu, f == (4 | bk));
                    if (lane == 0) cnt[bk * kCPer * kCW + r * kCW + warp] = __popc(m);
                }
            }
            __syncthreads();
            if (warp < 4) scan_counts(cnt + warp * kCPer * kCW, xtot + warp, lane);
            __syncthreads();
            const int xb1 = xtot[0], xb2 = xb1 + xtot[1], xb3 = xb2 + xtot[2];
#pragma unroll
            for (int r = 0; r < kCPer; ++r) {
                const int k = r * kCT + threadIdx.x;
                const int f = (xflag >> (3 * r)) & 7;
#pragma unroll
                for (int bk = 0; bk < 4; ++bk) {
                    const unsigned m = __ballot_sync(0xffffffffu, f == (4 | bk));
                    if (f == (4 | bk)) {
                        int e = k + 1;
                        while (e < nq && e % kPiece != 0 && !xstart(e)) ++e;
                        const int base = bk == 0 ? 0 : (bk == 1 ? xb1 : (bk == 2 ? xb2 : xb3));
                        s_xpiece[base + cnt[bk * kCPer * kCW + r * kCW + warp] + __popc(m & lanemask_lt_())] =
                            (uint16_t)(k | ((e - k - 1) << 12));
                    }
                }
            }
            __syncthreads();
            // ---- phase 2: current of the pieces, then of the crossing pieces; items in
            // blocks of 96 = 3 components x 32, so that a warp's items share the component
            const int np = misc[2];
            const int nblk = (np + 31) >> 5;
            // crossing pieces per bucket, their blocks of 32 (scalars: an array
            // indexed by the bucket would live in local memory)
            const int xn0 = xtot[0], xn1 = xtot[1], xn2 = xtot[2], xn3 = xtot[3];
            const int xk0 = (xn0 + 31) >> 5, xk1 = (xn1 + 31) >> 5, xk2 = (xn2 + 31) >> 5, xk3 = (xn3 + 31) >> 5;
            // current scale: -q w dx_a / dt, times the chunk's fixed-point unit; no
            // node can receive more than K_O |jscale_a| sum_p (|dxi_a| + 1e-6) from
            // the chunk (|C Y| <= K_O |dxi_a|, fixed_point_cy_bound), kept below 2^30
            // units; a piece or crossing piece converts its register sum once, so
            // a node collects at most one rounding half per piece, per crossing
            // piece and per particle crossing on several axes
            float jsc[3], unit[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
#if PP_CELLS_FIXED
                const float bound = fixed_point_cy_bound<O>() * fabsf(S.jscale[d]) *
                                    (((float *)misc)[10 + d] + 1e-6f * (float)cn) * 1.001f;
                unit[d] = bound > 0.0f ? kFixedRange / bound : 0.0f;
#else
                unit[d] = 1.0f;
#endif
                jsc[d] = S.jscale[d] * unit[d];
            }
            const int nitems = (nblk + xk0 + xk1 + xk2 + xk3) * 96;
#pragma unroll 1
            for (int it = threadIdx.x; it < nitems; it += kCT) {
                const int blk = it / 96, rr = it - blk * 96, comp = rr >> 5, j = rr & 31;
                // lane j of item block b takes piece (crossing piece) j * blocks + b:
                // consecutive pieces often share a cell, so lanes on consecutive
                // pieces would add to the same words
                if (blk < nblk) {
                    const int p = j * nblk + blk;
                    if (p >= np) continue;
                    const int ps = s_piece[p], pe = s_piece[p + 1];
                    if (comp == 0) piece_current<O, 0>(Jw, s_o, s_d, s_grp, ps, pe, jsc[0] PP_IF_CHECKED(, T.status));
                    else if (comp == 1) piece_current<O, 1>(Jw, s_o, s_d, s_grp, ps, pe, jsc[1] PP_IF_CHECKED(, T.status));
                    else piece_current<O, 2>(Jw, s_o, s_d, s_grp, ps, pe, jsc[2] PP_IF_CHECKED(, T.status));
                } else {   // crossing pieces: the block's bucket, then lane j's piece in it
                    int bk, lb = blk - nblk, nk, nn, base;
                    if (lb < xk0) {
                        bk = 0; nk = xk0; nn = xn0; base = 0;
                    } else if ((lb -= xk0) < xk1) {
                        bk = 1; nk = xk1; nn = xn1; base = xn0;
                    } else if ((lb -= xk1) < xk2) {
                        bk = 2; nk = xk2; nn = xn2; base = xn0 + xn1;
                    } else {
                        lb -= xk2;
                        bk = 3; nk = xk3; nn = xn3; base = xn0 + xn1 + xn2;
                    }
                    const int k = j * nk + lb;
                    if (k >= nn) continue;
                    const int v = s_xpiece[base + k];
                    const int ks = v & 0xfff, ke = ks + (v >> 12) + 1;
                    const float js = comp == 0 ? jsc[0] : (comp == 1 ? jsc[1] : jsc[2]);
                    xpiece_current<O>(Jw, comp, s_o, s_d, s_grp, s_queue, ks, ke, bk, js PP_IF_CHECKED(, T.status));
                }
            }
            __syncthreads();
#if PP_CELLS_FIXED
            // the window nodes the chunk's cells reach, into the FP32 mesh (and cleared):
            // 16 lanes to a row of kW nodes.  Over the exact box of the chunk's cells, by a
            // flat index, the divisions made this 7 % of the kernel's instructions; the
            // planes of its slabs, whole, also need no bounds kept per particle (268 M
            // particle beam 30.08 -> 29.34 ms per step, 192^3 Weibel 19.36 -> 18.91).
            {
                const int i = threadIdx.x & 15, rows = (zhi - zlo + kRLo + kRHi + 1) * kW;
#pragma unroll
                for (int comp = 0; comp < 3; ++comp)
                    for (int r = threadIdx.x >> 4; r < rows; r += kCT / 16) {
                        if (i >= kW) continue;
                        const int j = r % kW, k = zlo + r / kW;
                        JT *w = Jw + comp * kWVol + wi(i, j, k);
                        const int iv = *w;
                        if (iv == 0) continue;
                        *w = 0;
                        atomicAdd(T.J[comp] + g.at(wx + i, wy + j, wz + k), (float)iv / unit[comp]);
                    }
            }
            __syncthreads();
#endif
        }
    }
#if !PP_CELLS_FIXED
    // ---- the tile's current, once into the FP32 mesh
    for (int idx = threadIdx.x; idx < 3 * kWVol; idx += kCT) {
        const float v = Jw[idx];
        if (v == 0.0f) continue;
        const int comp = idx / kWVol, r = idx - comp * kWVol;
        const int i = r % kW, j = (r / kW) % kW, k = r / (kW * kW);
        atomicAdd(T.J[comp] + g.at(wx + i, wy + j, wz + k), v);
    }
#endif
    return true;
}

// Dynamic shared memory starts 128-byte aligned (the TMA destinations); the
// kernels check it and stop (ST_BOUNDS) otherwise.
__device__ __forceinline__ bool smem_aligned(const float *smem, int *status) {
    if ((smem_addr(smem) & 127) == 0) return true;
    if (threadIdx.x == 0) atomicOr(status, ST_BOUNDS);
    return false;
}

template <int O, int PUSH, bool BND>
__global__ void __launch_bounds__(kCT, 1) k_particles_cells(const __grid_constant__ CellsArgs T) {
    extern __shared__ __align__(128) float smem[];
    if (!smem_aligned(smem, T.status)) return;
    uint64_t *bar = (uint64_t *)((char *)smem + kFieldBytes - 128);
    if (threadIdx.x == 0) mbar_init(bar);
    __syncthreads();
    uint32_t phase = 0;
    cells_tile<O, PUSH, BND, false>(T, blockIdx.x, smem, phase);
}

// Batched form: the tiles and species of many runs as (run, item) work items, taken in
// order by persistent CTAs from a device counter (the items come sorted by
// run size, largest first, so that the last items are short).  Every run's
// arguments, tensor maps included, sit in device memory.
template <int O, int PUSH, bool BND>
__global__ void __launch_bounds__(kCT, 1) k_particles_cells_multi(const CellsArgs *args, const int2 *items,
                                                                 int nitems, int *next, int *status) {
    extern __shared__ __align__(128) float smem[];
    if (!smem_aligned(smem, status)) return;
    uint64_t *bar = (uint64_t *)((char *)smem + kFieldBytes - 128);
    int *item = (int *)(bar + 2);
    if (threadIdx.x == 0) mbar_init(bar);
    uint32_t phase = 0;
    for (;;) {
        if (threadIdx.x == 0) *item = atomicAdd(next, 1);
        __syncthreads();
        const int w = *item;
        __syncthreads();   // every thread has read it before thread 0 takes the next
        if (w >= nitems) return;
        const int2 it = items[w];
        if (!cells_tile<O, PUSH, BND, true>(args[it.x], it.y, smem, phase)) return;
        __syncthreads();
    }
}

}  // namespace

// Besides the tile shape: every tile's TMA box starts at an x that is a
// multiple of 4 nodes (G - kRLo is, and tile origins are multiples of 8) and
// ends inside the padded row (G >= kWG - kT - kRLo), with rows of a multiple
// of 16 bytes.
bool cells_supported(const Ctx &c) {
    if (c.fp64 || c.current_mode != PP_CURRENT_CONSERVING || c.g.G < kRLo || c.g.G < kRHi) return false;
    if ((c.g.G - kRLo) % 4 != 0 || c.g.G < kWG - kT - kRLo || c.g.P[0] % 4 != 0) return false;
    for (int a = 0; a < 3; ++a)
        if (c.g.n[a] % kT != 0 || c.tile[a] != kT) return false;
    return true;
}

// The argument block of one context, with the tensor maps of its E and B
// arrays; any = false when no species holds particles.
static cudaError_t cells_args(const Ctx &c, CellsArgs &T, bool &any) {
    any = false;
    sorted_args(c, T);
    const int box[3] = {kWG, kWG, kWG};
    for (int comp = 0; comp < 6; ++comp) {
        cudaError_t e = encode_box_map(&T.tmap[comp], comp < 3 ? T.E[comp] : T.B[comp - 3], c.g.P, box);
        if (e != cudaSuccess) return e;
    }
    any = T.ns > 0;
    return cudaSuccess;
}

template <class K>
static cudaError_t smem_attr(K kernel, unsigned long long &done) {
    return ensure_smem_attr(kernel, (int)kCellsSmem, done);
}

// All species in one launch; every species with particles must have been
// sorted since its particles last moved (Species::fresh).
cudaError_t launch_particles_cells(Ctx &c) {
    if (!cells_supported(c)) return cudaErrorInvalidConfiguration;
    if (!sorted_ready(c)) return cudaErrorInvalidValue;
    CellsArgs T;
    bool any = false;
    cudaError_t ea = cells_args(c, T, any);
    if (ea != cudaSuccess || !any) return ea;
    const unsigned blocks = (unsigned)((int64_t)c.ntile[0] * c.ntile[1] * c.ntile[2] * T.ns);
    const int o = c.d.shape_order, pu = c.d.pusher;
    const bool bnd = c.any_wall();
    static unsigned long long attr_done[2][2][4] = {};
#define PP_CB(O, PU, BD)                                                                                     \
    do {                                                                                                     \
        cudaError_t e_ = smem_attr(k_particles_cells<O, PU, BD>, attr_done[BD][PU][O]);                      \
        if (e_ != cudaSuccess) return e_;                                                                    \
        k_particles_cells<O, PU, BD><<<blocks, kCT, kCellsSmem, c.st>>>(T);                                  \
    } while (0)
#define PP_C(O, PU)                                                                                          \
    do {                                                                                                     \
        if (bnd) PP_CB(O, PU, true); else PP_CB(O, PU, false);                                               \
    } while (0)
    if (pu == PP_BORIS) {
        if (o == 1) PP_C(1, PP_BORIS); else if (o == 2) PP_C(2, PP_BORIS); else PP_C(3, PP_BORIS);
    } else {
        if (o == 1) PP_C(1, PP_VAY); else if (o == 2) PP_C(2, PP_VAY); else PP_C(3, PP_VAY);
    }
#undef PP_C
#undef PP_CB
    ++c.nlaunch;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    sorted_after(c);
    return cudaSuccess;
}

// Most work items of a context: its tiles times its species.
int64_t cells_items(const Ctx &c) { return (int64_t)c.ntile[0] * c.ntile[1] * c.ntile[2] * c.nspecies; }

size_t cells_args_bytes() { return sizeof(CellsArgs); }

int cells_batch_key(const Ctx &c) { return c.d.shape_order * 4 + c.d.pusher * 2 + (c.any_wall() ? 1 : 0); }

// The tiles and species of n contexts with one cells_batch_key in one persistent launch of
// nsm CTAs on st.  host_args / host_items: pinned host memory of at least
// n * cells_args_bytes() and (sum of cells_items) * 8 bytes, copied to the device
// scratch on st (the caller keeps them unchanged until the copy has run).
cudaError_t launch_particles_cells_batch(Ctx *const *ctxs, int n, cudaStream_t st, CellsBatchScratch &scr,
                                         void *host_args, void *host_items, int nsm) {
    if (n <= 0) return cudaSuccess;
    CellsArgs *A = (CellsArgs *)host_args;
    int2 *items = (int2 *)host_items;
    // runs with particles, largest first: their tiles become the first items
    int order[4096], m = 0;
    for (int k = 0; k < n && m < 4096; ++k) {
        Ctx &c = *ctxs[k];
        if (!cells_supported(c) || !sorted_ready(c)) return cudaErrorInvalidValue;
        bool any = false;
        cudaError_t ea = cells_args(c, A[m], any);
        if (ea != cudaSuccess) return ea;
        if (any) order[m++] = k;
    }
    int64_t ntot = 0;
    for (int a = 0; a < m; ++a) {   // insertion sort by tile count, descending
        for (int b = a; b > 0; --b) {
            const Ctx &x = *ctxs[order[b]], &y = *ctxs[order[b - 1]];
            const int64_t tx = (int64_t)x.ntile[0] * x.ntile[1] * x.ntile[2];
            const int64_t ty = (int64_t)y.ntile[0] * y.ntile[1] * y.ntile[2];
            if (tx <= ty) break;
            const int t = order[b]; order[b] = order[b - 1]; order[b - 1] = t;
            CellsArgs u = A[b]; A[b] = A[b - 1]; A[b - 1] = u;
        }
    }
    for (int a = 0; a < m; ++a) {
        const Ctx &c = *ctxs[order[a]];
        const int n_items = c.ntile[0] * c.ntile[1] * c.ntile[2] * A[a].ns;
        for (int t = 0; t < n_items; ++t) items[ntot++] = make_int2(a, t);
    }
    if (m == 0) return cudaSuccess;
    const size_t abytes = sizeof(CellsArgs) * (size_t)m, ibytes = sizeof(int2) * (size_t)ntot;
    if (abytes > scr.args_cap || ibytes > scr.items_cap) return cudaErrorMemoryAllocation;
    cudaError_t e = cudaMemcpyAsync(scr.args, A, abytes, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(scr.items, items, ibytes, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(scr.next, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    const Ctx &c0 = *ctxs[order[0]];
    const int o = c0.d.shape_order, pu = c0.d.pusher;
    const bool bnd = c0.any_wall();
    const unsigned grid = (unsigned)(nsm < ntot ? nsm : ntot);
    static unsigned long long attr_done[2][2][4] = {};
#define PP_MB(O, PU, BD)                                                                                     \
    do {                                                                                                     \
        cudaError_t e_ = smem_attr(k_particles_cells_multi<O, PU, BD>, attr_done[BD][PU][O]);                \
        if (e_ != cudaSuccess) return e_;                                                                    \
        k_particles_cells_multi<O, PU, BD><<<grid, kCT, kCellsSmem, st>>>(                                   \
            (const CellsArgs *)scr.args, (const int2 *)scr.items, (int)ntot, scr.next, c0.d_status);         \
    } while (0)
#define PP_M(O, PU)                                                                                          \
    do {                                                                                                     \
        if (bnd) PP_MB(O, PU, true); else PP_MB(O, PU, false);                                               \
    } while (0)
    if (pu == PP_BORIS) {
        if (o == 1) PP_M(1, PP_BORIS); else if (o == 2) PP_M(2, PP_BORIS); else PP_M(3, PP_BORIS);
    } else {
        if (o == 1) PP_M(1, PP_VAY); else if (o == 2) PP_M(2, PP_VAY); else PP_M(3, PP_VAY);
    }
#undef PP_M
#undef PP_MB
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    for (int a = 0; a < m; ++a) {
        Ctx &c = *ctxs[order[a]];
        ++c.nlaunch;
        sorted_after(c);
    }
    return cudaSuccess;
}

}  // namespace pp
