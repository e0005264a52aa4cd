// pp_rows.cu -- the particle step of the mixed form on meshes that 8^3 tiles
// do not divide, on particles sorted by cell at the start of every step
// (Sec. III: the paper sorts the particle array by cell position in every
// step, between the current deposit and the field update).
//
// The other kernel of such meshes takes one thread per particle on the global
// mesh, with an L2 reduction per site (144 of them for a PCS particle): 3.89 ms
// per step for 3.2 M particles on 60 x 45 x 37 cells, against 0.54 ms here (and
// 0.06 ms for the sort).  Few particles stay with it (rows_pay).
//
// One CTA of 16 warps per block of 8 x 8 x tz cells (tz = 4, 2 or 1: a slab of
// an 8^3 tile of the sort, whose particles are contiguous; the last tiles are
// partly empty).  The particles of a block are cut into batches of 32 and each
// warp takes a contiguous run of batches; after the E/B window is staged no
// barrier joins the warps again.  Per batch:
//
//  phase 1, one lane per particle: gather (eq:pfields), push (Vay / Boris,
//    optional radiative cooling), move; the new cell, offset and momentum go
//    straight back to the particle arrays (coalesced), the old offset and the
//    displacement stay in registers.
//  phase 2, the charge-conserving current (eq:cc1, eq:jj3, Esirkepov's
//    decomposition as the 2nd-order current by a per-particle prefix sum): the
//    weights of 16 particles go to shared memory, then each half-warp takes
//    one particle at a time, its 16 lanes the 4 x 4 nodes in y and z of the
//    particle's cell (nodes cell - 1 .. cell + 2), with the sites along x in
//    registers.  The sites of a cell are summed there over all its particles
//    in the warp; the window slides along the row of cells, and a node that
//    no later cell of the row can reach is added into the FP32 mesh.  A node's
//    current is summed in FP32 throughout, as the global-mesh kernel's is.
//
// Gather: the E/B window (12 x 12 x (tz + 4) nodes per component) is kept as
// quads, four consecutive nodes along x from every start, so that a particle's
// row of nodes is one aligned 16-byte shared load wherever its cell begins.
// The lanes of a warp sit in one or two cells, so the load is a broadcast: one
// wavefront, as for a 4-byte load, with four times the data.  The products run
// as packed pairs.
//
// Bound by issue: 82 warp-instructions a particle at 60 % of the issue slots
// (64^3 thermal PCS; 128 registers, of which PCS spills some 30 bytes a thread
// and TSC 116).  Emitting nodes four at a time through a shared ring, as
// vector reductions, was slower: more code than the instruction cache holds.
#include "pp_sorted.cuh"

namespace pp {

namespace {

constexpr int kT = kSortTile;                    // edge of the sort's tiles (cells)
constexpr int kRLo = 2;                          // nodes the window holds below the block
constexpr int kWG = kT + 4;                      // 12 window nodes along x and y
constexpr int kWZ = 8;                           // planes of the largest window (tz = 4)
// 16 warps at 128 registers (shared memory allows one CTA per SM); 12 warps at
// 168 registers execute 6 % fewer instructions and measured 6 % slower (64^3
// thermal PCS: 1.96 against 2.09 ms).
constexpr int kCT = 512;                         // threads per CTA
constexpr int kCW = kCT / 32;
static_assert(kCT % 32 == 0, "whole warps");

// Quads of a window row (a PCS support starts at node 8 at the latest, a CIC or
// TSC one at node 9) and of a plane.  A step along x, y and z is 4, 8 and 16
// words modulo the 32 banks: the up to eight starts that the particles of one
// cell have, one per octant, fall in distinct banks.
constexpr int kQRow = 10;
constexpr int kQPlane = kWG * kQRow + 4;
static_assert(kQRow * 4 % 32 == 8 && kQPlane * 4 % 32 == 16, "quad strides");

// Deposit record of a particle in shared memory, in 16-byte slots (M: mean of
// the old and new weight of a node, D: their difference over sqrt(12), C:
// prefix of the difference on the face above the node times the current scale):
//   0-3  y node k of the cell's four: (M, D, C, C)      4-7  z likewise
//   8, 9 x: (M0, D0, M1, D1), (M2, D2, M3, D3)          10, 11 x: (C0, C0, C1, C1), (C2, C2, 0, 0)
//   12, 13 x: node -1 and node 4 (M, D, C, C), the faces -1 and 3
//   14, 15 y and z: the node outside the four that a crossing particle reaches
// (slots 12-15 are zero for the others).  17 slots apart, so
// that the lanes of a store fall in distinct banks.
constexpr int kRec = 17 * 16;
constexpr int kSub = 16;                         // records of a warp, and one of zeros after them
constexpr int kRecWarp = (kSub + 1) * kRec;
// Current outside the 4 x 4 lanes, from particles that cross in y or z, per
// warp: rows of kRowX x-nodes.  Groups y up, y down, z up, z down: 3 components
// x 4 nodes of the other axis; then the four corners (y, z) x 3 components.
constexpr int kRowX = 13;
constexpr int kSideRows = 4 * 12 + 4 * 3;
constexpr int kSideWarp = kSideRows * kRowX * 4;
constexpr int kPlane = kWG * kWG;
constexpr size_t kRecBytes = (size_t)kCW * kRecWarp;
constexpr size_t kQuadBytes = (size_t)6 * kWZ * kQPlane * 16;
constexpr size_t kSideBytes = (size_t)kCW * kSideWarp;
constexpr size_t kRowsSmem = kRecBytes + kQuadBytes + kSideBytes;
static_assert(kRowsSmem <= 227 * 1024, "CTA must fit the opt-in shared memory");
static_assert(6 * kWZ * kPlane * 4 <= kRecBytes, "the raw window is staged where the records go");
static_assert(kRecBytes % 16 == 0 && kQuadBytes % 16 == 0 && kSideBytes % 16 == 0,
              "aligned regions");
// Fewest blocks of a launch before the blocks are made thinner: one per SM.
// Thinner blocks stage more window per particle, so they pay only where SMs
// would stand idle (32^3 x 8 per cell per species, 64 tiles: 0.110 ms per pass
// with tz = 2 against 0.127 with 1; 48 x 40 x 32, 120 tiles: 0.69 ms per four
// passes with tz = 4 against 0.75 with 2 and 0.79 with 1).
constexpr int kMinBlocks = 152;
struct RowsArgs : SortedArgs {
    int tz;                      // cells of a block along z
    int bounded;                 // walls on some axis, or an open end
};

// ---- deposit ----
// Node of the cell's four (0-3) where the support of the position x (cell
// units from the particle's old cell, |x - old offset| < 1) starts, and its
// fractional coordinate; -1 and 5 - O: the support reaches one node outside.
template <int O>
__device__ __forceinline__ int frame_support(float x, float &f) {
    const float y = O == 2 ? x - 0.5f : x;
    const float c = floorf(y);
    f = y - c;
    return (int)c + (O == 3 ? 0 : 1);
}

// Weights of one particle's move along one axis on the nodes of its cell
// (M, D, C as in the record) and on the node below (dn) or above (up) them
// that a crossing particle reaches: its new weight, 0 for the others.
struct AxisMove {
    float M[4], D[4], C[3], dn, up;
};
constexpr float kRsqrt12 = 0.28867513459481287f;

template <int O>
__device__ __forceinline__ void axis_move(float o, float d, float js, AxisMove &r) {
    float w0[O + 1], w[O + 1], f0, f1, S0[4], S1[4];
    // old weights: the support starts at node 0 (PCS), 0 or 1 (TSC), 1 (CIC)
    const int p0 = frame_support<O>(o, f0), p1 = frame_support<O>(o + d, f1);
    bspline2<O>(f0, f1, w0, w);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if constexpr (O == 3) S0[k] = w0[k];
        else if constexpr (O == 2) S0[k] = p0 ? (k ? w0[k - 1] : 0.0f) : (k < 3 ? w0[k] : 0.0f);
        else S0[k] = k == 1 ? w0[0] : (k == 2 ? w0[1] : 0.0f);
    }
    auto at = [&](int m) { return m >= 0 && m <= O ? w[m] : 0.0f; };   // m is a constant after unrolling
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        float v = p1 == 0 ? at(k) : (p1 == 1 ? at(k - 1) : 0.0f);
        if constexpr (O <= 2) v = p1 == 2 ? at(k - 2) : v;
        if constexpr (O >= 2) v = p1 == -1 ? at(k + 1) : v;
        S1[k] = v;
    }
    r.dn = O >= 2 && p1 == -1 ? w[0] : 0.0f;
    r.up = O >= 2 && p1 == 4 - O ? w[O] : 0.0f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float ds = S1[k] - S0[k];
        r.M[k] = S0[k] + 0.5f * ds;
        r.D[k] = ds * kRsqrt12;
        S1[k] = ds;
    }
    // prefix of the differences on the lower faces, suffix on the upper one
    // (they sum to zero)
    r.C[0] = (r.dn + S1[0]) * js;
    r.C[1] = (r.dn + S1[0] + S1[1]) * js;
    r.C[2] = -(r.up + S1[3]) * js;
}

template <bool B>
struct Out {
    static constexpr bool value = B;
};

// One node's current into the mesh (the sites that no particle reached are
// exact zeros).  p0, end: the padded array, for the checked build.
__device__ __forceinline__ void add_node(const RowsArgs &T, float *p, float v) {
    if (v == 0.0f) return;
    PP_IF_CHECKED(bool in = false; for (int c = 0; c < 3; ++c) in = in || (p >= T.J[c] && p < T.J[c] + T.g.padded_size());
                  if (!in) { atomicOr(T.status, ST_BOUNDS); return; })
    atomicAdd(p, v);
}

// Rows of the window's quads, for the gather.
struct QuadRow {
    const ulonglong2 *q;
    template <bool both>
    __device__ __forceinline__ ulonglong2 pairs(int j, int k) const {
        return q[k * kQPlane + j * kQRow];
    }
};
struct QuadWindow {
    const ulonglong2 *q;   // at the node two below the particle's cell
    PP_IF_CHECKED(int rx, ry, rz, O; int *status;)
    __device__ __forceinline__ QuadRow operator()(int comp, int x, int y, int z) const {
        PP_IF_CHECKED(if (rx + x >= kQRow || ry + y + O >= kWG || rz + z + O >= kWZ) {
            atomicOr(status, ST_BOUNDS);
            return QuadRow{q};
        })
        return QuadRow{q + comp * kWZ * kQPlane + z * kQPlane + y * kQRow + x};
    }
};

// One block: the whole particle step of its particles (all species), their
// current added into the mesh.  Called by every thread of the CTA; smem is the
// CTA's dynamic shared memory.
template <int O, int PUSH>
__global__ void __launch_bounds__(kCT, 1) k_particles_rows(const __grid_constant__ RowsArgs T) {
    extern __shared__ __align__(16) char smem[];
    const int item = blockIdx.x;   // the tile of the sort times the slabs per tile, plus the slab
    float *raw = (float *)smem;                                  // E/B window as loaded, before the records
    ulonglong2 *Q = (ulonglong2 *)(smem + kRecBytes);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    char *rec = smem + warp * kRecWarp;
    float *side = (float *)(smem + kRecBytes + kQuadBytes + warp * kSideWarp);
    const Geom &g = T.g;
    const int tz = T.tz, slabs = kT / tz;
    const int tile = item / slabs, slab = item - tile * slabs;
    const int ox = (tile % T.nt[0]) * kT, oy = ((tile / T.nt[0]) % T.nt[1]) * kT,
              oz = (tile / (T.nt[0] * T.nt[1])) * kT + slab * tz;
    const int64_t key0 = ((int64_t)tile * kSortTileCells + slab * tz * kT * kT) * kSubKeys;
    const int64_t key1 = key0 + tz * kT * kT * kSubKeys;
    {   // a block that holds no particle (the mirror half of a box between walls) stages nothing
        int held = 0;
        for (int s = 0; s < T.ns; ++s) held |= T.sp[s].cell_start[key1] - T.sp[s].cell_start[key0];
        if (!held) return;
    }
    // ---- the E/B window; nodes past the padding (beside the empty part of a
    // last tile) read as zero
    const int nz = tz + 4, rawc = nz * kPlane;   // words of a component
    const int x0 = ox - kRLo + g.G, y0 = oy - kRLo + g.G, z0 = oz - kRLo + g.G;
    for (int c = 0; c < 6; ++c) {
        const float *f = c == 0 ? T.E[0] : c == 1 ? T.E[1] : c == 2 ? T.E[2] : c == 3 ? T.B[0] : c == 4 ? T.B[1] : T.B[2];
        for (int t = threadIdx.x; t < rawc; t += kCT) {
            const int x = x0 + t % kWG, y = y0 + (t / kWG) % kWG, z = z0 + t / kPlane;
            const bool in = x < g.P[0] && y < g.P[1] && z < g.P[2];
            raw[c * rawc + t] = in ? f[((int64_t)z * g.P[1] + y) * g.P[0] + x] : 0.0f;
        }
    }
    for (int t = lane; t < kSideRows * kRowX; t += 32) side[t] = 0.0f;
    __syncthreads();
    // ---- rows of the window to quads
    for (int t = threadIdx.x; t < 6 * nz * kWG; t += kCT) {
        const int c = t / (nz * kWG), r = t - c * nz * kWG;   // component, row (z, y)
        float v[kWG + 4];
#pragma unroll
        for (int m = 0; m < kWG; m += 4) {
            const float4 q = *reinterpret_cast<const float4 *>(raw + c * rawc + r * kWG + m);
            v[m] = q.x; v[m + 1] = q.y; v[m + 2] = q.z; v[m + 3] = q.w;
        }
        v[kWG] = 0.0f;
        float4 *dst = reinterpret_cast<float4 *>(Q) + (c * kWZ + r / kWG) * kQPlane + (r % kWG) * kQRow;
#pragma unroll
        for (int m = 0; m < kQRow; ++m) dst[m] = make_float4(v[m], v[m + 1], v[m + 2], v[m + 3]);
    }
    __syncthreads();   // the raw window is read: its place now holds the records
    if (lane < 17) *reinterpret_cast<float4 *>(rec + kSub * kRec + lane * 16) = make_float4(0.0f, 0.0f, 0.0f, 0.0f);

    // ---- this warp's batches: a contiguous share of all species' batches of 32
    int nbatch = 0;
    for (int s = 0; s < T.ns; ++s) nbatch += (T.sp[s].cell_start[key1] - T.sp[s].cell_start[key0] + 31) >> 5;
    const int wb0 = (int)((int64_t)warp * nbatch / kCW), wb1 = (int)((int64_t)(warp + 1) * nbatch / kCW);
    const int half = lane >> 4, li = lane & 3, lj = (lane >> 2) & 3;
    int sbase = 0;   // batches of the species before
    for (int s = 0; s < T.ns; ++s) {
        const SortedSpecies &S = T.sp[s];
        const int tb = S.cell_start[key0], te = S.cell_start[key1];
        const int nb_s = (te - tb + 31) >> 5;
        const int b0 = max(wb0 - sbase, 0), b1 = min(wb1 - sbase, nb_s);
        sbase += nb_s;
        if (b0 >= b1) continue;
        const int pb = tb + 32 * b0, pe = min(tb + 32 * b1, te);   // this warp's particles

        // current of the cells' 4 x 4 lanes: sites along x of the cell `cur`
        // (block-local, x fastest; -1: none), as packed partial sums: faces
        // -1..3 of J_x, nodes -1..4 of J_y and J_z.  pxy, pz: this lane's mesh
        // node -1 of the window, the next to emit (J_x or J_y, and J_z).
        int cur = -1;
        unsigned dirty = 0;      // groups of `side` that hold current
        f2 a0[5], a1[6], a2[6];
        float *pxy = T.J[0], *pz = T.J[2];
#pragma unroll
        for (int m = 0; m < 5; ++m) a0[m] = 0;
#pragma unroll
        for (int m = 0; m < 6; ++m) a1[m] = a2[m] = 0;

        auto both = [&](f2 v) {   // the two half-warps' sums
            const float x = sum2(v);
            return x + __shfl_xor_sync(0xffffffffu, x, 16);
        };
        // Node m along x of the window into the mesh: J_x by half-warp 0, J_y by half-warp 1, then J_z
        auto emit = [&](int m, f2 v0, f2 v1, f2 v2) {
            const float s0 = both(v0), s1 = both(v1), s2 = both(v2);
            add_node(T, pxy + m, half ? s1 : s0);
            if (!half) add_node(T, pz + m, s2);
        };
        // Move the window to cell c of the same row.
        auto slide = [&](int c) {
#pragma unroll 1
            for (; cur < c; ++cur) {
                emit(0, a0[0], a1[0], a2[0]);
                ++pxy;
                ++pz;
#pragma unroll
                for (int m = 0; m < 4; ++m) a0[m] = a0[m + 1];
                a0[4] = 0;
#pragma unroll
                for (int m = 0; m < 5; ++m) {
                    a1[m] = a1[m + 1];
                    a2[m] = a2[m + 1];
                }
                a1[5] = a2[5] = 0;
            }
        };
        // Finish the row (the window's nodes and the rows beside it) and start
        // at cell c of another (-1: none).
        auto turn = [&](int c) {
            if (cur >= 0) {
#pragma unroll
                for (int m = 0; m < 6; ++m) {
                    emit(m, m < 5 ? a0[m] : 0, a1[m], a2[m]);
                    if (m < 5) a0[m] = 0;
                    a1[m] = a2[m] = 0;
                }
                const int base = (int)g.at(ox - kRLo, oy + ((cur >> 3) & 7) - 1, oz + (cur >> 6) - 1);
#pragma unroll 1
                for (; dirty & 15; dirty &= dirty - 1) {   // a row outside in y (groups 0, 1) or z (2, 3)
                    const int grp = __ffs(dirty) - 1;
                    const int py = g.P[0], pzs = g.P[0] * g.P[1];
                    const int in = grp < 2 ? pzs : py, out = grp < 2 ? py : pzs;   // strides of the two axes
                    // 13 nodes of two rows at a time by the half-warps; the outside node below is -1, above 4,
                    // and 3 for the component whose faces it carries
                    const int x = lane & 15;
                    float *p = side + (12 * grp + half) * kRowX + x;
                    const int m = base + x + half * in;
                    if (x < kRowX) {
#pragma unroll
                        for (int comp = 0; comp < 3; ++comp) {
                            const int o = m + out * ((grp & 1) ? -1 : (comp == 1 + (grp >> 1) ? 3 : 4));
#pragma unroll
                            for (int k = 0; k < 4; k += 2) {
                                add_node(T, T.J[comp] + o + k * in, p[(4 * comp + k) * kRowX]);
                                p[(4 * comp + k) * kRowX] = 0.0f;
                            }
                        }
                    }
                }
#pragma unroll 1
                for (; dirty; dirty &= dirty - 1) {   // a corner outside in both: a row per component
                    const int k = __ffs(dirty) - 5;
                    if (lane < kRowX) {
#pragma unroll
                        for (int comp = 0; comp < 3; ++comp) {
                            const int dy = (k & 2) ? -1 : (comp == 1 ? 3 : 4), dz = (k & 1) ? -1 : (comp == 2 ? 3 : 4);
                            float *p = side + (48 + 3 * k + comp) * kRowX + lane;
                            add_node(T, T.J[comp] + base + lane + (dz * g.P[1] + dy) * g.P[0], *p);
                            *p = 0.0f;
                        }
                    }
                }
                __syncwarp();
            }
            cur = c;
            const int at = (int)g.at(ox - kRLo + (c & 7), oy + ((c >> 3) & 7) - 1 + li, oz + (c >> 6) - 1 + lj);
            pxy = (half ? T.J[1] : T.J[0]) + at;
            pz = T.J[2] + at;
        };

        // the particle of the next batch is fetched before the current one is
        // computed, and its place in the pending permutation one batch before that
        int32_t n_cw = 0, n_src = 0;
        float n_o[3] = {0.0f, 0.0f, 0.0f}, n_u[3] = {0.0f, 0.0f, 0.0f};
        auto fetch = [&](int i) {
            if (i >= pe) return;
            const int src = S.perm ? n_src : i;
            if (S.perm && i + 32 < pe) n_src = S.perm[i + 32];
            n_cw = S.p.cell[src];
            n_o[0] = S.p.ox[src]; n_o[1] = S.p.oy[src]; n_o[2] = S.p.oz[src];
            n_u[0] = S.p.ux[src]; n_u[1] = S.p.uy[src]; n_u[2] = S.p.uz[src];
        };
        if (S.perm && pb + lane < pe) n_src = S.perm[pb + lane];
        fetch(pb + lane);
#pragma unroll 1
        for (int b = pb;; b += 32) {
            const bool fin = b >= pe;   // after the last batch: finish the row
            // ---- phase 1: gather, push, move, write back
            const bool valid = b + lane < pe;
            const int32_t cw0 = n_cw;
            float xi0[3] = {n_o[0], n_o[1], n_o[2]}, u[3] = {n_u[0], n_u[1], n_u[2]}, dx[3] = {0.0f, 0.0f, 0.0f};
            fetch(b + 32 + lane);
            int cx, cy, cz;
            unpack_cell(cw0, cx, cy, cz);
            int rx = cx - ox, ry = cy - oy, rz = cz - oz;
            const bool here = (unsigned)rx < (unsigned)kT && (unsigned)ry < (unsigned)kT && (unsigned)rz < (unsigned)tz;
            const bool act = valid && here;
            if (!act) rx = ry = rz = 0;
            int cross = 0;   // bit a: the particle reaches a node outside its cell's four along axis a; bit 3 + a: the lower
            if (valid) {
                const float u0[3] = {u[0], u[1], u[2]};
                if (S.qmdt != 0.0f) {   // uniform: no kick, no force
                    float E[3] = {0.0f, 0.0f, 0.0f}, B[3] = {0.0f, 0.0f, 0.0f};
                    gather_pairs<O>(QuadWindow{Q + rz * kQPlane + ry * kQRow + rx PP_IF_CHECKED(, rx, ry, rz, O, T.status)}, xi0, E, B);
                    push_particle<PUSH, float>(S.qmdt, S.kdt, E, B, u);
                }
                const float gi = inv_sqrt(1.0f + u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
                bool ok = here;
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    dx[d] = T.dtdx[d] * u[d] * gi;
                    ok = ok && (fabsf(dx[d]) < 1.0f);
                }
                if (!ok) {
                    // not in its sorted block (cannot happen after a sort), a cell or more in one
                    // step, or not finite: left unchanged, and the step flagged
                    atomicOr(T.status, !here ? ST_RANGE : (isfinite(u[0] + u[1] + u[2]) ? ST_CFL : ST_NAN));
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        u[d] = u0[d];
                        dx[d] = 0.0f;
                    }
                }
                float xi1[3];
                int cc[3] = {cx, cy, cz};
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    xi1[d] = xi0[d] + dx[d];
                    if constexpr (O >= 2) {
                        float f;
                        const int p1 = frame_support<O>(xi1[d], f);
                        if (p1 < 0 || p1 == 4 - O) cross |= (p1 < 0 ? 9 : 1) << d;
                    }
                    // re-bin: the offset back into [0, 1), the cell wrapped
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
                if (T.bounded && ok) {
                    reflect(cc[0], xi1[0], u[0], T.wall[0]);
                    reflect(cc[1], xi1[1], u[1], T.wall[1]);
                    reflect(cc[2], xi1[2], u[2], T.wall[2]);
                    cwd = pack_cell(cc[0], cc[1], cc[2]);
                    if (T.esc > 0.0 && (double)cc[0] + (double)xi1[0] < T.esc && u[0] < 0.0f) cwd |= kDeadBit;
                }
                if (!here) cwd = cw0;
                store_sorted(T, S, b + lane, cwd, xi1, u);
            }
            // ---- phase 2: the current, 16 particles at a time
            const int cell = act ? (rz << 6) | (ry << 3) | rx : -1;
            const unsigned actm = __ballot_sync(0xffffffffu, act);
            const unsigned crx = __ballot_sync(0xffffffffu, cross & 1), cry = __ballot_sync(0xffffffffu, cross & 2),
                           crz = __ballot_sync(0xffffffffu, cross & 4);
            unsigned lowy = 0, lowz = 0;
            if (cry | crz) {
                lowy = __ballot_sync(0xffffffffu, cross & 16);
                lowz = __ballot_sync(0xffffffffu, cross & 32);
            }
            AxisMove mx;   // x of this lane's particle
            axis_move<O>(xi0[0], dx[0], S.jscale[0], mx);
            // computed here, once for all 32 lanes, and not again in each half below
            asm volatile("" : "+f"(mx.M[0]), "+f"(mx.M[1]), "+f"(mx.M[2]), "+f"(mx.M[3]), "+f"(mx.D[0]), "+f"(mx.D[1]),
                         "+f"(mx.D[2]), "+f"(mx.D[3]), "+f"(mx.C[0]), "+f"(mx.C[1]), "+f"(mx.C[2]), "+f"(mx.dn), "+f"(mx.up));
#pragma unroll 1
            for (int sub = 0; sub < 32; sub += kSub) {
                if (!fin && !(actm >> sub)) break;
                if (!fin) {   // records: the x axis by the particle's own lane, y and z by the two half-warps
                    const int src = sub + (lane & 15);
                    const float yo = __shfl_sync(0xffffffffu, xi0[1], src), yd = __shfl_sync(0xffffffffu, dx[1], src);
                    const float zo = __shfl_sync(0xffffffffu, xi0[2], src), zd = __shfl_sync(0xffffffffu, dx[2], src);
                    AxisMove m;
                    const float jb = half ? S.jscale[2] : S.jscale[1];
                    axis_move<O>(half ? zo : yo, half ? zd : yd, jb, m);
                    float4 *r = reinterpret_cast<float4 *>(rec + (lane & 15) * kRec);
                    __syncwarp();   // the previous records are read
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const float c = k < 3 ? m.C[k] : 0.0f;
                        r[4 * half + k] = make_float4(m.M[k], m.D[k], c, c);
                    }
                    if constexpr (O >= 2) {
                        const float w = m.dn + m.up, c = (m.dn - m.up) * jb;   // one of the two, or neither
                        r[14 + half] = make_float4(0.5f * w, kRsqrt12 * w, c, c);
                    }
                    if ((lane & 16) == sub) {
                        r[8] = make_float4(mx.M[0], mx.D[0], mx.M[1], mx.D[1]);
                        r[9] = make_float4(mx.M[2], mx.D[2], mx.M[3], mx.D[3]);
                        r[10] = make_float4(mx.C[0], mx.C[0], mx.C[1], mx.C[1]);
                        r[11] = make_float4(mx.C[2], mx.C[2], 0.0f, 0.0f);
                        if constexpr (O >= 2) {
                            const float cd = mx.dn * S.jscale[0], cu = -mx.up * S.jscale[0];
                            r[12] = make_float4(0.5f * mx.dn, kRsqrt12 * mx.dn, cd, cd);
                            r[13] = make_float4(0.5f * mx.up, kRsqrt12 * mx.up, cu, cu);
                        }
                    }
                    __syncwarp();
                }
                const unsigned am = (actm >> sub) & 0xffffu, xm = (crx >> sub) & 0xffffu;
                // the particles in order: rows of cells, in them runs of one cell
                unsigned left = am;
#pragma unroll 1
                while (left || fin) {
                    int p = fin ? 0 : __ffs(left) - 1;
                    const int row = __shfl_sync(0xffffffffu, cell, sub + p) >> 3;
                    const unsigned inrow = __ballot_sync(0xffffffffu, (cell >> 3) == row) >> sub;
                    const int pend = p + __ffs(~((inrow & 0xffffu) >> p)) - 1;
                    const unsigned rowm = ((1u << pend) - 1u) & ~((1u << p) - 1u);
                    left &= ~((1u << pend) - 1u);
                    if (cur < 0 || (cur >> 3) != row) turn(__shfl_sync(0xffffffffu, cell, sub + p));
                    if (fin) break;
                    // ---- particles that cross in y or z: the row outside
                    if (O >= 2) {
                        const unsigned ly = lowy >> sub, lz = lowz >> sub;
                        unsigned ym = (cry >> sub) & rowm, zm = (crz >> sub) & rowm;
                        if (ym | zm) {
                            const unsigned yz = ym & zm;
                            dirty |= (ym & ~ly ? 1 : 0) | (ym & ly ? 2 : 0) | (zm & ~lz ? 4 : 0) | (zm & lz ? 8 : 0);
                            if (yz)
                                dirty |= (yz & ~ly & ~lz ? 16 : 0) | (yz & ~ly & lz ? 32 : 0) | (yz & ly & ~lz ? 64 : 0) |
                                         (yz & ly & lz ? 128 : 0);
                        }
                        // half-warp 0: a particle that crosses in y, half-warp 1: one in z (their rows differ).
                        // Lane 5 comp + en: a component at node en of the axis that stays inside (y, 4: the
                        // corner outside in both)
                        const int l15 = lane & 15, comp = l15 / 5, en = l15 - 5 * comp;
                        const bool corner = en == 4, own = (comp == 1) == (half == 0);
                        const char *rl = rec + (corner ? 240 : (half ? 0 : 64) + en * 16);   // node en
                        const char *rx_ = rec + (comp ? 128 : 160);
#pragma unroll 1
                        while (ym | zm) {
                            const int qy = __ffs(ym) - 1, qz = __ffs(zm) - 1;
                            ym &= ym - 1;
                            zm &= zm - 1;
                            const int q = max(half ? qz : qy, 0);
                            const unsigned xb = (qy >= 0 ? xm >> qy : 0u) | (qz >= 0 ? xm >> qz : 0u);
                            const int cq = __shfl_sync(0xffffffffu, cell, sub + q) & 7;
                            const int dy = (ly >> q) & 1, dz = (lz >> q) & 1;
                            const bool on = (half ? qz : qy) >= 0 && l15 < 15 &&
                                            (!corner || (half == 0 && ((crz >> (sub + q)) & 1)));
                            if (on) {
                                const float4 va = *reinterpret_cast<const float4 *>(rec + q * kRec + 224 + 16 * half);
                                const float4 vb = *reinterpret_cast<const float4 *>(rl + q * kRec);
                                const float4 s0 = *reinterpret_cast<const float4 *>(rx_ + q * kRec);
                                const float4 s1 = *reinterpret_cast<const float4 *>(rx_ + q * kRec + 16);
                                // J_x: (M M + D D) C_x; J_y takes C of y and M, D of z, J_z the reverse
                                const float cc = own ? va.z : vb.z;
                                const float al = comp == 0 ? fmaf(va.x, vb.x, va.y * vb.y) : cc * (own ? vb.x : va.x);
                                const float be = comp == 0 ? 0.0f : cc * (own ? vb.y : va.y);
                                const int r = corner ? 48 + (2 * dy + dz) * 3 + comp
                                                     : 24 * half + 12 * (half ? dz : dy) + comp * 4 + en;
                                float *d = side + r * kRowX + cq;
                                const float d1 = d[1] + fmaf(al, s0.x, be * s0.y), d2 = d[2] + fmaf(al, s0.z, be * s0.w);
                                const float d3 = d[3] + fmaf(al, s1.x, be * s1.y);
                                float d4 = d[4] + fmaf(al, s1.z, be * s1.w);
                                if (xb & 1) {   // one of the two crosses along x as well
                                    const float4 o0 = *reinterpret_cast<const float4 *>(rec + q * kRec + 192);
                                    const float4 o1 = *reinterpret_cast<const float4 *>(rec + q * kRec + 208);
                                    d[0] += comp ? fmaf(al, o0.x, be * o0.y) : al * o0.z;
                                    // face 3 of J_x is one below node 4
                                    if (comp) d[5] += fmaf(al, o1.x, be * o1.y);
                                    else d4 += al * o1.z;
                                }
                                d[1] = d1;
                                d[2] = d2;
                                d[3] = d3;
                                d[4] = d4;
                            }
                            __syncwarp();
                        }
                    }
#pragma unroll 1
                    while (p < pend) {
                    const int c = __shfl_sync(0xffffffffu, cell, sub + p);
                    const unsigned eq = (__ballot_sync(0xffffffffu, cell == c) >> sub) & 0xffffu;
                    const int e = p + __ffs(~(eq >> p)) - 1;
                    const unsigned runm = ((1u << e) - 1u) & ~((1u << p) - 1u);
                    if (c < cur) {   // out of order: cannot happen after a sort
                        if (lane == 0) atomicOr(T.status, ST_RANGE);
                        p = e;
                        continue;
                    }
                    slide(c);
                    // one particle per half-warp at the record pr; OUT: also the nodes outside along x
                    auto pair = [&](const char *pr, auto OUT) {
                        const ulonglong2 vy = *reinterpret_cast<const ulonglong2 *>(pr + li * 16);
                        const ulonglong2 vz = *reinterpret_cast<const ulonglong2 *>(pr + lj * 16 + 64);
                        const ulonglong2 x0 = *reinterpret_cast<const ulonglong2 *>(pr + 128);
                        const ulonglong2 x1 = *reinterpret_cast<const ulonglong2 *>(pr + 144);
                        const ulonglong2 c0 = *reinterpret_cast<const ulonglong2 *>(pr + 160);
                        const ulonglong2 c1 = *reinterpret_cast<const ulonglong2 *>(pr + 176);
                        const f2 yz = mul2(vy.x, vz.x);    // (My Mz, Dy Dz): their sum is the transverse weight
                        const f2 cy = mul2(vy.y, vz.x);    // Cy (Mz, Dz)
                        const f2 cz = mul2(vz.y, vy.x);    // Cz (My, Dy)
                        a0[1] = fma2(yz, c0.x, a0[1]);
                        a0[2] = fma2(yz, c0.y, a0[2]);
                        a0[3] = fma2(yz, c1.x, a0[3]);
                        a1[1] = fma2(cy, x0.x, a1[1]);
                        a1[2] = fma2(cy, x0.y, a1[2]);
                        a1[3] = fma2(cy, x1.x, a1[3]);
                        a1[4] = fma2(cy, x1.y, a1[4]);
                        a2[1] = fma2(cz, x0.x, a2[1]);
                        a2[2] = fma2(cz, x0.y, a2[2]);
                        a2[3] = fma2(cz, x1.x, a2[3]);
                        a2[4] = fma2(cz, x1.y, a2[4]);
                        if constexpr (decltype(OUT)::value) {
                            const ulonglong2 dn = *reinterpret_cast<const ulonglong2 *>(pr + 192);
                            const ulonglong2 up = *reinterpret_cast<const ulonglong2 *>(pr + 208);
                            a0[0] = fma2(yz, dn.y, a0[0]);
                            a1[0] = fma2(cy, dn.x, a1[0]);
                            a2[0] = fma2(cz, dn.x, a2[0]);
                            a0[4] = fma2(yz, up.y, a0[4]);
                            a1[5] = fma2(cy, up.x, a1[5]);
                            a2[5] = fma2(cz, up.x, a2[5]);
                        }
                    };
                    // both particles of a pair, then an odd run's last and zeros
                    const char *pr = rec + (p + half) * kRec;
                    const bool out = O >= 2 && (xm & runm);   // some of the run cross along x
                    int n = e - p;
                    if (!out) {
#pragma unroll 1
                        for (; n >= 4; n -= 4, pr += 4 * kRec) {
                            pair(pr, Out<false>());
                            pair(pr + 2 * kRec, Out<false>());
                        }
                    }
#pragma unroll 1
                    for (; n > 0; n -= 2, pr += 2 * kRec) {
                        if (n == 1 && half) pr = rec + kSub * kRec;
                        pair(pr, Out<(O >= 2)>());
                    }
                    p = e;
                    }
                }
                if (fin) break;
            }
            if (fin) break;
        }
    }
}

}  // namespace

// Mixed form, charge-conserving current, every size at least one 8-cell tile,
// and some size no multiple of 8.  On meshes that the tiles divide the tile
// kernel of pp_cells.cu serves, which the batched runs share: as fast at 64
// thermal PCS particles a cell (64^3: 1.93 ms, this one 1.96) though less exact
// where a net current is weak (its fixed-point sums leave up to 2e-5 of it in
// counter-streaming beams, this kernel 1e-6).  The two have not been compared at
// other loads.
bool rows_supported(const Ctx &c) {
    if (c.fp64 || c.current_mode != PP_CURRENT_CONSERVING || c.g.G < kWG - kT - kRLo) return false;
    bool divided = true;
    for (int a = 0; a < 3; ++a) {
        if (c.tile[a] != kT) return false;
        divided = divided && c.g.n[a] % kT == 0;
    }
    return !divided;
}

// Whether the row kernel and its sort take less time than the global-mesh kernel
// with a sort every 20 steps, the other route of the automatic deposit on such
// meshes.  The sort and the empty blocks cost by the mesh, the windows and rows
// by the tiles that hold particles, the global kernel by the particle: about
// 0.1, 0.3 and 0.9 ns (CIC, TSC, PCS), less where a launch is too small to fill
// the GPU.  So the line is a count of particles, n0 + a tiles of the fullest
// species + b tiles of all + c tiles of the mesh (in cells).  Particle phase and
// sort of two thermal species together, row and global kernel, ms a step:
//   163 x 161 x 157, 4 per cell: CIC 4.38, 1.59; TSC 5.55, 5.80; PCS 6.32, 14.5
//                    0.1 per cell, PCS: 3.29, 0.49; 1 per cell: 4.75, 3.53
//   60 x 45 x 37, 16 per cell: CIC 0.237, 0.166; TSC 0.318, 0.666; PCS 0.370, 1.76
//                 1 per cell, PCS: 0.190, 0.136; 2 per cell: 0.197, 0.198
//   20^3, 4 per cell: CIC 0.082, 0.022; TSC 0.090, 0.040; PCS 0.094, 0.078
// A hot plasma (u = 2) tips the balance at half the load of a thermal one; the
// line lies between the two.  Above `most` particles per cell the row kernel is
// taken all the same: the global kernel's error grows with the particles that
// add to a node one by one (J of counter-streaming electrons and ions against
// FP64, row and global: 32 per cell PCS 7e-7, 2.3e-6, TSC 6e-7, 1.3e-6, CIC
// 6e-7, 7e-7; 8 per cell PCS 7e-7, 9e-7).
bool rows_pay(const Ctx &c) {
    static constexpr double n0[4] = {0, 250e3, 80e3, 30e3}, a[4] = {0, 3.0, 0.9, 0.45}, b[4] = {0, 2.7, 0.65, 0.3},
                            m[4] = {0, 1.0, 0.3, 0.1}, most[4] = {0, 48, 8, 8};
    const int o = c.d.shape_order;
    double n = 0.0, fullest = 0.0, held = 0.0;
    for (int s = 0; s < c.nspecies; ++s) {
        const double h = (double)c.sp[s].tiles_held * kSortTileCells;
        n += (double)c.sp[s].n;
        held += h;
        fullest = h > fullest ? h : fullest;
    }
    const double mesh = (double)c.ntile[0] * c.ntile[1] * c.ntile[2] * kSortTileCells;
    const double filled = fullest < (double)c.g.cells() ? fullest : (double)c.g.cells();
    return n >= n0[o] + a[o] * fullest + b[o] * held + m[o] * mesh || n >= most[o] * filled;
}

// All species in one launch; every species with particles must have been
// sorted since its particles last moved (Species::fresh).
cudaError_t launch_particles_rows(Ctx &c) {
    if (!rows_supported(c)) return cudaErrorInvalidConfiguration;
    if (!sorted_ready(c)) return cudaErrorInvalidValue;
    RowsArgs T;
    sorted_args(c, T);
    if (T.ns == 0) return cudaSuccess;
    const int64_t tiles = (int64_t)c.ntile[0] * c.ntile[1] * c.ntile[2];
    T.tz = 4;   // the most the window's shared memory holds, unless that leaves SMs without a block
    while (T.tz > 1 && tiles * (kT / T.tz) < kMinBlocks) T.tz /= 2;
    T.bounded = c.any_wall() ? 1 : 0;
    const unsigned blocks = (unsigned)(tiles * (kT / T.tz));
    const int o = c.d.shape_order, pu = c.d.pusher;
    static unsigned long long attr_done[2][4] = {};
#define PP_C(O, PU)                                                                                          \
    do {                                                                                                     \
        cudaError_t e_ = ensure_smem_attr(k_particles_rows<O, PU>, (int)kRowsSmem, attr_done[PU][O]);        \
        if (e_ != cudaSuccess) return e_;                                                                    \
        k_particles_rows<O, PU><<<blocks, kCT, kRowsSmem, c.st>>>(T);                                        \
    } while (0)
    if (pu == PP_BORIS) {
        if (o == 1) PP_C(1, PP_BORIS); else if (o == 2) PP_C(2, PP_BORIS); else PP_C(3, PP_BORIS);
    } else {
        if (o == 1) PP_C(1, PP_VAY); else if (o == 2) PP_C(2, PP_VAY); else PP_C(3, PP_VAY);
    }
#undef PP_C
    ++c.nlaunch;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    sorted_after(c);
    return cudaSuccess;
}

}  // namespace pp
