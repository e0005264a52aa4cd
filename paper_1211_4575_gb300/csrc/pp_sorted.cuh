// pp_sorted.cuh -- what the two particle kernels of the mixed form share that
// run on particles sorted by cell at the start of every step (pp_cells.cu on
// meshes that 8^3 tiles divide, pp_rows.cu on the others): their arguments, the
// sort key that a moved particle is written back with, and the packed FP32
// pairs of the gather.
#pragma once

#include "pp_internal.cuh"
#include "pp_particle_common.cuh"

namespace pp {

constexpr int kSortTile = 8;                     // edge of the sort's tiles (cells)
constexpr int kSortTileCells = kSortTile * kSortTile * kSortTile;

struct SortedSpecies {
    MixedParticles p;            // read: slot i of the sorted order is p[perm[i]] (p[i] without perm)
    MixedParticles out;          // written: the new state of slot i, in the sorted order
    const int32_t *perm;         // pending sort permutation, or null
    int32_t *keys;               // written: the sort key of each slot's new state
    const int32_t *cell_start;   // per sort key, tile-major
    float qmdt;
    float kdt;                   // radiative cooling K / dt (0 = off)
    float jscale[3];             // -q w dx_a / dt
};

struct SortedArgs {
    Geom g;
    const float *E[3];
    const float *B[3];
    float *J[3];
    float dtdx[3];
    int nt[3];
    int ns;
    SortedSpecies sp[PP_MAX_SPECIES];
    int *status;
    int wall[3];                 // walls at 0 and wall[a] cells on axis a; 0 = periodic
    double esc;                  // open end: outgoing particles below x = esc cells leave; 0 = off
    int32_t dead_key;            // sort key of a particle that left: after every cell's keys
};

// Sort key of a particle in cell (x, y, z) with offsets o (the key of the cell
// sort: its 8^3 tile in tile order, its cell in the tile, the octant of the
// cell that holds it), or dead_key for a particle that left.
__device__ __forceinline__ int32_t sort_key(const SortedArgs &T, int32_t cw, const float (&o)[3]) {
    if (cw < 0) return T.dead_key;
    int x, y, z;
    unpack_cell(cw, x, y, z);
    const int tile = ((z / kSortTile) * T.nt[1] + y / kSortTile) * T.nt[0] + x / kSortTile;
    const int cell = ((z % kSortTile) * kSortTile + y % kSortTile) * kSortTile + x % kSortTile;
    const int oct = (o[0] >= 0.5f ? 1 : 0) | (o[1] >= 0.5f ? 2 : 0) | (o[2] >= 0.5f ? 4 : 0);
    return (tile * kSortTileCells + cell) * kSubKeys + oct;
}

__device__ __forceinline__ void store_sorted(const SortedArgs &T, const SortedSpecies &S, int64_t i, int32_t cw,
                                             const float (&o)[3], const float (&u)[3]) {
    S.out.cell[i] = cw;
    S.out.ox[i] = o[0]; S.out.oy[i] = o[1]; S.out.oz[i] = o[2];
    S.out.ux[i] = u[0]; S.out.uy[i] = u[1]; S.out.uz[i] = u[2];
    S.keys[i] = sort_key(T, cw, o);
}

// ---- packed FP32 pairs ----
// fma.rn.f32x2 issues at the rate of a scalar FMA of three distinct registers
// on this part (1.85 against 1.95 warp-instructions per clock and SM), with
// twice the work.
using f2 = unsigned long long;
__device__ __forceinline__ f2 pack2(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ f2 dup2(float a) { return pack2(a, a); }
__device__ __forceinline__ void unpack2(f2 v, float &a, float &b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ float sum2(f2 v) {
    float a, b;
    unpack2(v, a, b);
    return a + b;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// bspline of two fractional coordinates at once, packed.
template <int O>
__device__ __forceinline__ void bspline2(float fa, float fb, float (&a)[O + 1], float (&b)[O + 1]) {
    const f2 f = pack2(fa, fb), one = dup2(1.0f);
    const f2 g = fma2(f, dup2(-1.0f), one);
    if constexpr (O == 1) {
        unpack2(g, a[0], b[0]);
        unpack2(f, a[1], b[1]);
    } else if constexpr (O == 2) {
        const f2 h = fma2(one, f, dup2(-0.5f));
        unpack2(mul2(mul2(g, g), dup2(0.5f)), a[0], b[0]);
        unpack2(fma2(mul2(h, dup2(-1.0f)), h, dup2(0.75f)), a[1], b[1]);
        unpack2(mul2(mul2(f, f), dup2(0.5f)), a[2], b[2]);
    } else {
        // w1 = (3 f^3 - 6 f^2 + 4) / 6 = 2/3 - f^2 (1 - f/2), and w2 the same in g = 1 - f
        const f2 ff = mul2(f, f), gg = mul2(g, g), m = dup2(0.5f), c = dup2(2.0f / 3.0f), s = dup2(1.0f / 6.0f);
        unpack2(mul2(mul2(gg, s), g), a[0], b[0]);
        unpack2(fma2(ff, fma2(f, m, dup2(-1.0f)), c), a[1], b[1]);
        unpack2(fma2(gg, fma2(g, m, dup2(-1.0f)), c), a[2], b[2]);
        unpack2(mul2(mul2(ff, s), f), a[3], b[3]);
    }
}

// Weights and first node (relative to the node two below the particle's cell)
// of the offset o in [0, 1) on integer (half = false) or half-integer nodes.
// One of the two supports starts at a node fixed by the cell (fractional
// coordinate o), the other depends on the half of the cell that holds o
// (coordinate o - 1/2 or o + 1/2).
template <int O, bool half>
__device__ __forceinline__ int gather_support(float o, float (&w)[O + 1]) {
    constexpr bool fixed = (O % 2 == 1) != half;
    const bool up = o >= 0.5f;
    const float f = fixed ? o : (up ? o - 0.5f : o + 0.5f);
    bspline<O, float>(f, w);
    if constexpr (O == 3) return half ? (up ? 1 : 0) : 1;
    else if constexpr (O == 2) return half ? 1 : (up ? 2 : 1);
    else return half ? (up ? 2 : 1) : 2;
}

// E and B at the particle's offset o.  row(comp, x, y, z, k, j): the pairs of
// nodes (0, 1) and (2, 3) along x of row (j, k) of the support that starts at
// (x, y, z) relative to the node two below the particle's cell.  Per component
// sums over z of sums over y, the x pairs packed throughout, then over x.
template <int O, class RowOf>
__device__ __forceinline__ void gather_pairs(const RowOf &row, const float (&o)[3], float (&E)[3], float (&B)[3]) {
    float wx[2][O + 1], w[O + 1];
    f2 wy[2][O + 1], wz[2][O + 1];   // [0] integer, [1] half-integer nodes, each weight twice
    int x[2], y[2], z[2];
    x[0] = gather_support<O, false>(o[0], wx[0]);
    x[1] = gather_support<O, true>(o[0], wx[1]);
    y[0] = gather_support<O, false>(o[1], w);
#pragma unroll
    for (int m = 0; m <= O; ++m) wy[0][m] = dup2(w[m]);
    y[1] = gather_support<O, true>(o[1], w);
#pragma unroll
    for (int m = 0; m <= O; ++m) wy[1][m] = dup2(w[m]);
    z[0] = gather_support<O, false>(o[2], w);
#pragma unroll
    for (int m = 0; m <= O; ++m) wz[0][m] = dup2(w[m]);
    z[1] = gather_support<O, true>(o[2], w);
#pragma unroll
    for (int m = 0; m <= O; ++m) wz[1][m] = dup2(w[m]);
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        // E_a: half-integer along a; B_a: integer along a, half-integer across.
        const int hx = (c % 3 == 0) != (c >= 3), hy = (c % 3 == 1) != (c >= 3), hz = (c % 3 == 2) != (c >= 3);
        const auto at = row(c, x[hx], y[hy], z[hz]);
        f2 a = 0, b = 0;
#pragma unroll
        for (int k = 0; k <= O; ++k) {
            f2 s = 0, t = 0;
#pragma unroll
            for (int j = 0; j <= O; ++j) {
                const ulonglong2 v = at.template pairs<(O >= 2)>(j, k);
                s = j ? fma2(v.x, wy[hy][j], s) : mul2(v.x, wy[hy][j]);
                if (O >= 2) t = j ? fma2(v.y, wy[hy][j], t) : mul2(v.y, wy[hy][j]);
            }
            a = k ? fma2(s, wz[hz][k], a) : mul2(s, wz[hz][k]);
            if (O >= 2) b = k ? fma2(t, wz[hz][k], b) : mul2(t, wz[hz][k]);
        }
        a = mul2(a, pack2(wx[hx][0], wx[hx][1]));
        if constexpr (O == 3) a = fma2(b, pack2(wx[hx][2], wx[hx][3]), a);
        float r = sum2(a);
        if constexpr (O == 2) {
            float b0, b1;
            unpack2(b, b0, b1);
            r = fmaf(b0, wx[hx][2], r);
        }
        if (c < 3) E[c] = r;
        else B[c - 3] = r;
    }
}

// ---- host ----
// Every species with particles was sorted since its particles last moved.
inline bool sorted_ready(const Ctx &c) {
    for (int s = 0; s < c.nspecies; ++s)
        if (c.sp[s].n > 0 && !c.sp[s].fresh) return false;
    return true;
}

inline void sorted_args(const Ctx &c, SortedArgs &T) {
    T.g = c.g;
    const double h[3] = {c.d.dx, c.d.dy, c.d.dz};
    for (int d = 0; d < 3; ++d) {
        T.E[d] = (const float *)c.E[d];
        T.B[d] = (const float *)c.B[d];
        T.J[d] = (float *)c.J[d];
        T.dtdx[d] = (float)(c.drift_dt / h[d]);
        T.nt[d] = c.ntile[d];
        T.wall[d] = c.wall[d];
    }
    T.ns = 0;
    for (int s = 0; s < c.nspecies; ++s) {
        const Species &S = c.sp[s];
        if (S.n == 0) continue;
        SortedSpecies &t = T.sp[T.ns++];
        t.p = MixedParticles{S.cell, S.ox, S.oy, S.oz, S.fux, S.fuy, S.fuz};
        int32_t *c2 = (int32_t *)S.alt;
        float *f2 = (float *)(c2 + S.cap);
        t.out = MixedParticles{c2, f2, f2 + S.cap, f2 + 2 * S.cap, f2 + 3 * S.cap, f2 + 4 * S.cap, f2 + 5 * S.cap};
        t.perm = S.perm_pending ? S.perm : nullptr;
        t.keys = S.keys;
        t.cell_start = S.cell_start;
        t.qmdt = (float)(S.q * c.kick_dt / S.m);
        t.kdt = (float)(c.kick_dt != 0.0 ? S.rad / c.kick_dt : 0.0);
        for (int d = 0; d < 3; ++d) t.jscale[d] = (float)(-S.q * S.w * h[d] / c.drift_dt);
    }
    T.status = c.d_status;
    T.esc = c.escape_now;
    T.dead_key = (int32_t)c.nkeys;
}

// After the launch: every slot of the sorted order holds its particle's new
// state in the other buffer, with its next sort key.
inline void sorted_after(Ctx &c) {
    for (int s = 0; s < c.nspecies; ++s) {
        Species &S = c.sp[s];
        if (S.n == 0) continue;
        void *old = S.buf;
        S.buf = S.alt;
        S.alt = old;
        S.bind(false);
        S.perm_pending = false;
        S.keys_valid = true;
    }
}

}  // namespace pp
