// pp_mesh.cu -- mesh kernels of the step: periodic ghost fold of the deposited
// current, the high-order current solve (Sec. III eq:jj6 .. eq:penta), the
// implicit de-centred field update (eq:bnplus1, eq:enplus1, eq:EllipticB),
// the periodic ghost fill of E and B, and the FP64 mesh diagnostics.
//
// Mesh arrays are padded (Geom::at).  E and B keep their periodic ghost layers
// filled (the particle gather reads them), and so do the relaxation iterates:
// the implicit solver's stencils read those through linear offsets.
// Other stencils read interior values through periodic wrapping (Nb).
#include <atomic>

#include "pp_internal.cuh"

namespace pp {

__device__ __forceinline__ void unflatten(int64_t t, const Geom &g, int &i, int &j, int &k) {
    i = (int)(t % g.n[0]);
    int64_t r = t / g.n[0];
    j = (int)(r % g.n[1]);
    k = (int)(r / g.n[1]);
}

// ---------------------------------------------------------------------------
// Ghost fold: every interior node near a face collects the ghost images of
// itself (coordinates + m n inside the padding, all axes at once).  The ghosts
// are only read, each by one thread, and keep their values: nothing reads the
// ghosts of J (its stencils wrap), and the next pass clears the arrays.  One
// launch over the interior, in which a node without images costs its index
// alone; one pass per axis over all nodes, read and written, measured 0.36 ms
// on 256 x 128 x 128 nodes of FP32, this one about 0.03 ms.
// ---------------------------------------------------------------------------
template <typename R>
__global__ void __launch_bounds__(256) k_fold(Geom g, R *J0, R *J1, R *J2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y, k = blockIdx.z;
    if (i >= g.n[0] || j >= g.n[1]) return;
    const int c[3] = {i, j, k};
    int lo[3];   // lowest image coordinate per axis
    bool any = false;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        lo[a] = c[a];
        while (lo[a] - g.n[a] >= -g.G) lo[a] -= g.n[a];
        any = any || lo[a] != c[a] || c[a] + g.n[a] < g.n[a] + g.G;
    }
    if (!any) return;
    R s0 = R(0), s1 = R(0), s2 = R(0);
    for (int z = lo[2]; z < g.n[2] + g.G; z += g.n[2])
        for (int y = lo[1]; y < g.n[1] + g.G; y += g.n[1])
            for (int x = lo[0]; x < g.n[0] + g.G; x += g.n[0]) {
                const int64_t q = g.at(x, y, z);
                s0 += J0[q];
                s1 += J1[q];
                s2 += J2[q];
            }
    const int64_t q = g.at(i, j, k);
    J0[q] = s0;
    J1[q] = s1;
    J2[q] = s2;
}

template <typename R>
static cudaError_t fold_impl(Ctx &c) {
    const Geom &g = c.g;
    const dim3 b(32, 8), n((unsigned)((g.n[0] + 31) / 32), (unsigned)((g.n[1] + 7) / 8), (unsigned)g.n[2]);
    k_fold<R><<<n, b, 0, c.st>>>(g, (R *)c.J[0], (R *)c.J[1], (R *)c.J[2]);
    ++c.nlaunch;
    return cudaGetLastError();
}

cudaError_t launch_fold_J(Ctx &c) { return c.fp64 ? fold_impl<double>(c) : fold_impl<float>(c); }

cudaError_t launch_zero_J(Ctx &c) {
    // the components of J (and of J') follow one another in the mesh allocation
    return cudaMemsetAsync(c.J[0], 0, (size_t)c.g.padded_size() * c.rsz * 3, c.st);
}

// ---------------------------------------------------------------------------
// Reflecting walls (Sec. V "Boundary conditions").  On a walled axis a the
// mesh is the mirror-extended box of n0 = 2 n_a cells, the walls on the
// integer nodes 0 and n_a.  Along a, integer node i has the image
// (n0 - i) mod n0 and half node i+1/2 (index i) the image index n0 - 1 - i.
// Components staggered along a are odd across the wall and the others even:
// E_a and J_a, and every B_b with b != a.  Walls on several axes fold one axis
// after the other (the images of images are the corner images).
//
// avg = 0 (a deposit): the virtual images contribute the mirror of what the
// particles deposited, f(i) <- f(i) + P f(m(i)), and the image node receives
// P times that sum; a wall node, its own image, doubles.  avg = 1 (a load):
// f(i) <- (f(i) + P f(m(i))) / 2 on both nodes of the pair.  One thread per
// pair: i in [0, n_a] along a row (odd components stop at n_a - 1).
// ---------------------------------------------------------------------------
struct PaddedIndex {
    Geom g;
    __device__ __forceinline__ int64_t operator()(int i, int j, int k) const { return g.at(i, j, k); }
};
struct CompactIndex {
    int n0, n1;
    __device__ __forceinline__ int64_t operator()(int i, int j, int k) const {
        return i + (int64_t)n0 * (j + (int64_t)n1 * k);
    }
};

// Pairs along the wall normal `ax` (walls at 0 and nw cells), over the mesh
// extents ne of the other two axes: thread (i, p, r) holds the row position i
// along ax and the coordinates p, r along axes ax+1, ax+2 (mod 3).
template <typename R, class Ix>
__global__ void k_mirror(Ix ix, int ax, int nw, int nb, int nc, R *F0, R *F1, R *F2, int odd_mask, int avg) {
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int comp = blockIdx.y;
    if (t >= (int64_t)(nw + 1) * nb * nc) return;
    const int i = (int)(t % (nw + 1));
    const int64_t r = t / (nw + 1);
    const int pb = (int)(r % nb), pc = (int)(r / nb);
    const bool odd = (odd_mask >> comp) & 1;
    int m;
    if (odd) {
        if (i == nw) return;
        m = 2 * nw - 1 - i;
    } else {
        m = i == 0 ? 0 : 2 * nw - i;
    }
    int q[3], qm[3];
    q[ax] = i;
    qm[ax] = m;
    q[(ax + 1) % 3] = qm[(ax + 1) % 3] = pb;
    q[(ax + 2) % 3] = qm[(ax + 2) % 3] = pc;
    R *F = comp == 0 ? F0 : (comp == 1 ? F1 : F2);
    const int64_t a = ix(q[0], q[1], q[2]), b = ix(qm[0], qm[1], qm[2]);
    const R P = odd ? R(-1) : R(1);
    R v = F[a] + P * F[b];
    if (avg) v *= R(0.5);
    F[a] = v;
    if (b != a) F[b] = P * v;
}

// Components odd across a wall with normal ax: E_ax and J_ax (staggered along
// it); for B every component but B_ax.
static inline int odd_mask(bool bfield, int ax) { return bfield ? (7 & ~(1 << ax)) : (1 << ax); }

template <typename R, class Ix>
static cudaError_t mirror_axes(Ctx &c, Ix ix, R *F0, R *F1, R *F2, int ncomp, int bfield_or_rho, int avg) {
    for (int ax = 0; ax < 3; ++ax) {
        const int nw = c.wall[ax];
        if (!nw) continue;
        const int nb = c.g.n[(ax + 1) % 3], nc = c.g.n[(ax + 2) % 3];
        const int mask = bfield_or_rho < 0 ? 0 : odd_mask(bfield_or_rho == 1, ax);
        dim3 grid((unsigned)(((int64_t)(nw + 1) * nb * nc + 255) / 256), (unsigned)ncomp);
        k_mirror<R, Ix><<<grid, 256, 0, c.st>>>(ix, ax, nw, nb, nc, F0, F1, F2, mask, avg);
        ++c.nlaunch;
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <typename R>
static cudaError_t mirror_padded(Ctx &c, void *const F[3], int bfield, int avg) {
    return mirror_axes<R, PaddedIndex>(c, PaddedIndex{c.g}, (R *)F[0], (R *)F[1], (R *)F[2], 3, bfield, avg);
}

cudaError_t launch_mirror_J(Ctx &c) {
    if (!c.any_wall()) return cudaSuccess;
    return c.fp64 ? mirror_padded<double>(c, c.J, 0, 0) : mirror_padded<float>(c, c.J, 0, 0);
}

cudaError_t launch_mirror_fields(Ctx &c) {
    if (!c.any_wall()) return cudaSuccess;
    cudaError_t e = c.fp64 ? mirror_padded<double>(c, c.E, 0, 1) : mirror_padded<float>(c, c.E, 0, 1);
    if (e != cudaSuccess) return e;
    return c.fp64 ? mirror_padded<double>(c, c.B, 1, 1) : mirror_padded<float>(c, c.B, 1, 1);
}

cudaError_t launch_mirror_rho(Ctx &c, double *rho) {
    if (!c.any_wall()) return cudaSuccess;
    return mirror_axes<double, CompactIndex>(c, CompactIndex{c.g.n[0], c.g.n[1]}, rho, rho, rho, 1, -1, 0);
}

// ---------------------------------------------------------------------------
// Open lower end (Sec. V "Boundary conditions", outflow): each step the
// chosen components are multiplied by 1 - damping ((cells - d) / cells)^2 at
// distance d < cells from x = 0, d taken at the component's staggered
// position, on both sides of that mirror plane so that the extended mesh stays
// symmetric.  Columns: the first `cells` x-indices and the last `cells`.
// ---------------------------------------------------------------------------
template <typename R>
__global__ void k_damp(Geom g, R *F, int half, int cells, double damping) {
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int cols = 2 * cells;
    if (t >= (int64_t)cols * g.n[1] * g.n[2]) return;
    const int c = (int)(t % cols);
    const int64_t r = t / cols;
    const int j = (int)(r % g.n[1]), k = (int)(r / g.n[1]);
    const int N = g.n[0];
    const int i = c < cells ? c : N - 2 * cells + c;
    const double pos = i + (half ? 0.5 : 0.0);
    const double d = fmin(pos, N - pos);
    if (d >= cells) return;
    const double s = (cells - d) / cells;
    F[g.at(i, j, k)] *= (R)(1.0 - damping * s * s);
}

template <typename R>
static cudaError_t damp_impl(Ctx &c) {
    const int cells = c.open.cells;
    void **groups[2] = {c.E, c.B};
    const int half[2] = {1, 6};   // staggered in x: E_x; B_y, B_z
    const unsigned blocks = (unsigned)(((int64_t)2 * cells * c.g.n[1] * c.g.n[2] + 255) / 256);
    for (int f = 0; f < 2; ++f)
        for (int comp = 0; comp < 3; ++comp) {
            if (!((c.open.mask >> (3 * f + comp)) & 1)) continue;
            k_damp<R><<<blocks, 256, 0, c.st>>>(c.g, (R *)groups[f][comp], (half[f] >> comp) & 1, cells,
                                                c.open.damping);
            ++c.nlaunch;
            cudaError_t e = cudaGetLastError();
            if (e != cudaSuccess) return e;
        }
    return launch_ghost_fill(c, c.E, c.B);
}

cudaError_t launch_damp(Ctx &c) {
    if (!c.wall[0] || c.open.cells <= 0 || !c.open.mask) return cudaSuccess;
    return c.fp64 ? damp_impl<double>(c) : damp_impl<float>(c);
}

// ---------------------------------------------------------------------------
// Sliding window (Sec. V "Sliding window and injection of particles"): the
// content of the box moves one cell up in x.  In the physical half a node takes
// the value of the node one cell below (zero for the new bottom node); a node
// of the mirror half takes P times the new value of its image.  Written into
// scratch arrays, which then swap with E and B.
// ---------------------------------------------------------------------------
template <typename R>
__global__ void k_window_fields(Geom g, int nw, const R *I0, const R *I1, const R *I2, R *O0, R *O1, R *O2,
                                int odd_mask) {
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int comp = blockIdx.y;
    if (t >= g.cells()) return;
    const int i = (int)(t % g.n[0]);
    const int64_t r = t / g.n[0];
    const int j = (int)(r % g.n[1]), k = (int)(r / g.n[1]);
    const bool odd = (odd_mask >> comp) & 1;
    const R *in = comp == 0 ? I0 : (comp == 1 ? I1 : I2);
    R *out = comp == 0 ? O0 : (comp == 1 ? O1 : O2);
    const int top = odd ? nw - 1 : nw;   // last node of the physical half
    int src = i;
    R sign = R(1);
    if (i > top) {                        // mirror half: the image node
        src = odd ? 2 * nw - 1 - i : 2 * nw - i;
        sign = odd ? R(-1) : R(1);
    }
    out[g.at(i, j, k)] = src == 0 ? R(0) : sign * in[g.at(src - 1, j, k)];
}

template <typename R>
static cudaError_t window_fields_impl(Ctx &c) {
    dim3 grid((unsigned)((c.g.cells() + 255) / 256), 3);
    void **F[2] = {c.E, c.B};
    void **S[2] = {c.Xa, c.Xb};
    const int odd[2] = {1, 6};
    for (int f = 0; f < 2; ++f) {
        k_window_fields<R><<<grid, 256, 0, c.st>>>(c.g, c.wall[0], (const R *)F[f][0], (const R *)F[f][1],
                                                   (const R *)F[f][2], (R *)S[f][0], (R *)S[f][1], (R *)S[f][2],
                                                   odd[f]);
        ++c.nlaunch;
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        for (int a = 0; a < 3; ++a) {
            void *t = F[f][a];
            F[f][a] = S[f][a];
            S[f][a] = t;
        }
    }
    return launch_ghost_fill(c, c.E, c.B);
}

cudaError_t launch_window_fields(Ctx &c) {
    if (!c.wall[0]) return cudaSuccess;
    return c.fp64 ? window_fields_impl<double>(c) : window_fields_impl<float>(c);
}

// ---------------------------------------------------------------------------
// High-order current: along the axis of each component, J_out = P^{-1} J_in
// with P the symmetric cyclic line operator (c, b+c, a+b+c, b+c, c) that
// turns the 2nd-order difference into the high-order one; applied as the
// exact (or exponentially truncated) circulant inverse, taps precomputed in
// FP64 on the host.  out(i) = sum_m T[m] * in(i + off + m).
// ---------------------------------------------------------------------------
// Bound by load issue: 17 taps of FP32 values that L1 serves (a block spans 32
// nodes along x and 8 along its component's axis, so the 8 + 16 rows it reads
// stay there).  Taps arrive in the kernel's arguments, and only nodes within
// the reach of a face wrap.  The previous form (a 256-node row per block, taps
// loaded and converted from FP64, wrapped indices throughout) took 0.47 ms on
// 256 x 128 x 128 nodes, this one about 0.1 ms.
template <typename R>
struct Taps {
    R t[3][kMaxTaps];
    int L[3];      // taps
    int off[3];    // offset of the first
};

template <typename R>
__global__ void __launch_bounds__(256) k_current_solve(Geom g, const __grid_constant__ Taps<R> ts, const R *I0,
                                                       const R *I1, const R *I2, R *O0, R *O1, R *O2, int nb0, int nb1) {
    // blocks of component 0 and 1 (32 x 8 nodes in x and y, one z), then of
    // component 2 (x and z, one y)
    int b = blockIdx.x;
    const int comp = b < nb0 ? 0 : (b < nb0 + nb1 ? 1 : 2);
    b -= comp == 0 ? 0 : (comp == 1 ? nb0 : nb0 + nb1);
    const int bx = (g.n[0] + 31) / 32, ea = comp == 2 ? g.n[2] : g.n[1];
    const int by = (ea + 7) / 8;
    const int i = (b % bx) * 32 + (threadIdx.x & 31), v = ((b / bx) % by) * 8 + (threadIdx.x >> 5), w = b / (bx * by);
    if (i >= g.n[0] || v >= ea) return;
    const int j = comp == 2 ? w : v, k = comp == 2 ? v : w;
    const R *in = comp == 0 ? I0 : (comp == 1 ? I1 : I2);
    R *out = comp == 0 ? O0 : (comp == 1 ? O1 : O2);
    const int L = ts.L[comp], n = comp == 0 ? g.n[0] : ea;
    const int stride = comp == 0 ? 1 : (comp == 1 ? g.P[0] : g.P[0] * g.P[1]);
    const int x = comp == 0 ? i : v, x0 = x + ts.off[comp];
    const int q = (int)g.at(i, j, k);
    R acc = R(0);
    if (x0 >= 0 && x0 + L <= n) {
        const R *p = in + q + (x0 - x) * stride;
#pragma unroll 4
        for (int m = 0; m < L; ++m) acc += ts.t[comp][m] * p[m * stride];
    } else {
        const R *p = in + q - x * stride;
        int y = x0;
#pragma unroll 4
        for (int m = 0; m < L; ++m, ++y) acc += ts.t[comp][m] * p[(y < 0 ? y + n : (y >= n ? y - n : y)) * stride];
    }
    out[q] = acc;
}

template <typename R>
static cudaError_t current_solve_impl(Ctx &c) {
    const Geom &g = c.g;
    Taps<R> ts;
    for (int a = 0; a < 3; ++a) {
        const int n = c.ntaps[a];
        for (int m = 0; m < kMaxTaps; ++m) ts.t[a][m] = m < n ? (R)c.h_taps[a * kMaxTaps + m] : R(0);
        ts.L[a] = n;
        ts.off[a] = -(n / 2);
        if (c.full_circ[a])   // the whole period: rotate so that it starts n / 2 below the node
            for (int m = 0; m < n; ++m) ts.t[a][m] = (R)c.h_taps[a * kMaxTaps + (m + n - n / 2) % n];
    }
    const int64_t bx = (g.n[0] + 31) / 32;
    const int64_t xy = bx * ((g.n[1] + 7) / 8) * g.n[2], xz = bx * ((g.n[2] + 7) / 8) * g.n[1];
    k_current_solve<R><<<(unsigned)(2 * xy + xz), 256, 0, c.st>>>(
        g, ts, (const R *)c.J[0], (const R *)c.J[1], (const R *)c.J[2], (R *)c.Jt[0], (R *)c.Jt[1], (R *)c.Jt[2], (int)xy,
        (int)xy);
    ++c.nlaunch;
    return cudaGetLastError();
}

cudaError_t launch_current_solve(Ctx &c) {
    if (c.d.field_order == 2) return cudaSuccess;
    cudaError_t e = c.fp64 ? current_solve_impl<double>(c) : current_solve_impl<float>(c);
    if (e != cudaSuccess) return e;
    for (int a = 0; a < 3; ++a) {
        void *t = c.J[a];
        c.J[a] = c.Jt[a];
        c.Jt[a] = t;
    }
    return cudaSuccess;
}

// ---------------------------------------------------------------------------
// Field update.  Staggered first differences (Sec. III):
//   d^+ f (i+1/2) = sum_m k_m (f[i+m] - f[i+1-m]) / h
//   d^- f (i)     = sum_m k_m (f[i+m-1] - f[i-m]) / h
// and the Laplacian sum_a d^+_a d^-_a as the symmetric 11-point stencil lap[].
// ---------------------------------------------------------------------------
struct FieldCoef {
    double k[3];      // a, b, c
    double lap[6];    // offsets 0..5 of the 1D d^+ d^- stencil (times 1)
    double ih[3];     // 1/h per axis
    double ih2[3];    // 1/h^2 per axis
};

template <typename R>
struct Nb {
    const Geom &g;
    int c[3];
    __device__ __forceinline__ R at(const R *f, int axis, int s) const {
        int q[3] = {c[0], c[1], c[2]};
        q[axis] = wrap(c[axis] + s, g.n[axis]);
        return f[g.at(q[0], q[1], q[2])];
    }
    __device__ __forceinline__ R dplus(const R *f, int axis, const FieldCoef &k) const {
        R s = R(0);
#pragma unroll
        for (int m = 1; m <= 3; ++m) s += (R)k.k[m - 1] * (at(f, axis, m) - at(f, axis, 1 - m));
        return s * (R)k.ih[axis];
    }
    __device__ __forceinline__ R dminus(const R *f, int axis, const FieldCoef &k) const {
        R s = R(0);
#pragma unroll
        for (int m = 1; m <= 3; ++m) s += (R)k.k[m - 1] * (at(f, axis, m - 1) - at(f, axis, -m));
        return s * (R)k.ih[axis];
    }
    __device__ __forceinline__ R lap(const R *f, const FieldCoef &k) const {
        R center = f[g.at(c[0], c[1], c[2])];
        R s = R(0);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            R sa = (R)k.lap[0] * center;
#pragma unroll
            for (int o = 1; o <= 5; ++o) sa += (R)k.lap[o] * (at(f, a, o) + at(f, a, -o));
            s += sa * (R)k.ih2[a];
        }
        return s;
    }
};

template <typename R>
struct Vec3 {
    const R *p[3];
};

// Store v at interior cell (i, j, k) and at every periodic image of it inside
// the ghost layers, so that the array stays readable by linear offsets.  Every
// ghost cell is the image of exactly one interior cell.
template <typename R>
__device__ __forceinline__ void store_periodic(R *f, const Geom &g, int i, int j, int k, R v) {
    int x0 = i, y0 = j, z0 = k;
    while (x0 - g.n[0] >= -g.G) x0 -= g.n[0];
    while (y0 - g.n[1] >= -g.G) y0 -= g.n[1];
    while (z0 - g.n[2] >= -g.G) z0 -= g.n[2];
    for (int z = z0; z < g.n[2] + g.G; z += g.n[2])
        for (int y = y0; y < g.n[1] + g.G; y += g.n[1])
            for (int x = x0; x < g.n[0] + g.G; x += g.n[0]) f[g.at(x, y, z)] = v;
}

// rhs_a = B_a + alpha beta dt^2 (L B)_a - dt (curl^+ E)_a + alpha dt^2 (curl^+ J)_a
// (eq:EllipticB; the current term's sign follows from eq:bnplus1 + eq:enplus1)
template <typename R>
__global__ void k_rhs(Geom g, FieldCoef k, Vec3<R> E, Vec3<R> B, Vec3<R> J, R *O0, R *O1, R *O2, R ab_dt2,
                      R dt, R a_dt2) {
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= g.cells()) return;
    Nb<R> nb{g, {0, 0, 0}};
    unflatten(t, g, nb.c[0], nb.c[1], nb.c[2]);
    int64_t q = g.at(nb.c[0], nb.c[1], nb.c[2]);
    R *out[3] = {O0, O1, O2};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int b = (a + 1) % 3, c = (a + 2) % 3;
        R curlE = nb.dplus(E.p[c], b, k) - nb.dplus(E.p[b], c, k);
        R curlJ = nb.dplus(J.p[c], b, k) - nb.dplus(J.p[b], c, k);
        out[a][q] = B.p[a][q] + ab_dt2 * nb.lap(B.p[a], k) - dt * curlE + a_dt2 * curlJ;
    }
}

// ---- the implicit solver's kernels: W nodes along x per thread ----
// B and E arrive with valid ghost layers and every kernel that writes them here
// writes their images too, so stencils read through linear offsets and no pass
// copies ghosts.  With an even mesh size along x (rows of an even number of
// nodes, the interior starting at an even one) W = 2: every value along y and
// z is one aligned pair load, and a pair's row of x neighbours six or seven.
// Nothing is staged in shared memory and no barrier joins the threads: L1
// holds the rows that a block's 32 x 8 threads share.
template <typename R>
struct Coef {
    R k[3], lap[6], ih[3], ih2[3];
};
template <typename R, int W>
struct Nodes {
    R v[W];
};
template <int W, typename R>
__device__ __forceinline__ Nodes<R, W> ld(const R *p) {
    Nodes<R, W> r;
    if constexpr (W == 1) {
        r.v[0] = *p;
    } else if constexpr (sizeof(R) == 4) {
        const float2 t = *reinterpret_cast<const float2 *>(p);
        r.v[0] = t.x;
        r.v[1] = t.y;
    } else {
        const double2 t = *reinterpret_cast<const double2 *>(p);
        r.v[0] = t.x;
        r.v[1] = t.y;
    }
    return r;
}

// The row of x neighbours from node -N (N even for W = 2) to node N + W - 1 of
// the thread's nodes; the thread's own are given.
template <int N, typename R, int W>
struct Row {
    R v[2 * N + W];
    __device__ __forceinline__ Row(const R *p) {
#pragma unroll
        for (int m = 0; m < 2 * N + W; m += W) {
            const Nodes<R, W> t = ld<W>(p + m - N);
#pragma unroll
            for (int w = 0; w < W; ++w) v[m + w] = t.v[w];
        }
    }
    __device__ __forceinline__ R at(int o, int w) const { return v[N + o + w]; }
};
template <int W>
constexpr int even(int n) {
    return W == 2 ? (n + 1) / 2 * 2 : n;
}

// d^+ (plus) or d^- of f along `axis` at the thread's nodes.
template <typename R, int W>
__device__ __forceinline__ Nodes<R, W> diff(const R *f, int axis, int stride, bool plus, const Coef<R> &k) {
    Nodes<R, W> r;
#pragma unroll
    for (int w = 0; w < W; ++w) r.v[w] = R(0);
    if (axis == 0) {
        const Row<even<W>(3), R, W> x(f);
#pragma unroll
        for (int m = 1; m <= 3; ++m)
#pragma unroll
            for (int w = 0; w < W; ++w) r.v[w] += k.k[m - 1] * (plus ? x.at(m, w) - x.at(1 - m, w) : x.at(m - 1, w) - x.at(-m, w));
    } else {
#pragma unroll
        for (int m = 1; m <= 3; ++m) {
            const Nodes<R, W> u = ld<W>(f + (plus ? m : m - 1) * stride), d = ld<W>(f + (plus ? 1 - m : -m) * stride);
#pragma unroll
            for (int w = 0; w < W; ++w) r.v[w] += k.k[m - 1] * (u.v[w] - d.v[w]);
        }
    }
#pragma unroll
    for (int w = 0; w < W; ++w) r.v[w] *= k.ih[axis];
    return r;
}

// d^+ of J, whose ghosts are not valid: the thread's nodes wrap.  x: the
// nodes' coordinate along the axis, n its size.
template <typename R, int W>
__device__ __forceinline__ Nodes<R, W> diff_wrap(const R *f, int axis, int stride, int x, int n, const Coef<R> &k) {
    Nodes<R, W> r;
#pragma unroll
    for (int w = 0; w < W; ++w) {
        R s = R(0);
        const int c = axis == 0 ? x + w : x;
#pragma unroll
        for (int m = 1; m <= 3; ++m)
            s += k.k[m - 1] * (f[w + (wrap(c + m, n) - c) * stride] - f[w + (wrap(c + 1 - m, n) - c) * stride]);
        r.v[w] = s * k.ih[axis];
    }
    return r;
}

// L f at the thread's nodes: per axis the symmetric 11-point stencil.
// col: the 11 nodes along z.
template <typename R, int W>
__device__ __forceinline__ Nodes<R, W> laplace(const R *f, int sy, const Nodes<R, W> (&col)[11], const Coef<R> &k) {
    Nodes<R, W> r, s;
    const Row<even<W>(5), R, W> x(f);
#pragma unroll
    for (int w = 0; w < W; ++w) {
        s.v[w] = k.lap[0] * col[5].v[w];
#pragma unroll
        for (int o = 1; o <= 5; ++o) s.v[w] += k.lap[o] * (x.at(o, w) + x.at(-o, w));
        r.v[w] = s.v[w] * k.ih2[0];
        s.v[w] = k.lap[0] * col[5].v[w];
    }
#pragma unroll
    for (int o = 1; o <= 5; ++o) {
        const Nodes<R, W> u = ld<W>(f + o * sy), d = ld<W>(f - o * sy);
#pragma unroll
        for (int w = 0; w < W; ++w) s.v[w] += k.lap[o] * (u.v[w] + d.v[w]);
    }
#pragma unroll
    for (int w = 0; w < W; ++w) {
        r.v[w] += s.v[w] * k.ih2[1];
        s.v[w] = k.lap[0] * col[5].v[w];
#pragma unroll
        for (int o = 1; o <= 5; ++o) s.v[w] += k.lap[o] * (col[5 + o].v[w] + col[5 - o].v[w]);
        r.v[w] += s.v[w] * k.ih2[2];
    }
    return r;
}

// Store the thread's nodes (i, j, z) and their periodic images.
template <typename R, int W>
__device__ __forceinline__ void store_nodes(R *f, const Geom &g, int q, int i, int j, int z, const Nodes<R, W> &v) {
    const bool inner = i >= g.G && i + W <= g.n[0] - g.G && j >= g.G && j < g.n[1] - g.G && z >= g.G && z < g.n[2] - g.G;
    if (inner) {
        if constexpr (W == 1) f[q] = v.v[0];
        else if constexpr (sizeof(R) == 4) *reinterpret_cast<float2 *>(f + q) = make_float2(v.v[0], v.v[1]);
        else *reinterpret_cast<double2 *>(f + q) = make_double2(v.v[0], v.v[1]);
    } else {
#pragma unroll
        for (int w = 0; w < W; ++w) store_periodic(f, g, i + w, j, z, v.v[w]);
    }
}

template <typename R>
__device__ __forceinline__ const R *pick(const Vec3<R> &v, int a) {   // no run-time index into the arguments
    return a == 0 ? v.p[0] : (a == 1 ? v.p[1] : v.p[2]);
}

// rhs_a = B_a + alpha beta dt^2 (L B)_a - dt (curl^+ E)_a + alpha dt^2 (curl^+ J)_a
template <typename R, int W>
__global__ void __launch_bounds__(256) k_rhs_lin(Geom g, const __grid_constant__ Coef<R> k, Vec3<R> E, Vec3<R> B,
                                                 Vec3<R> J, R *O0, R *O1, R *O2, R ab_dt2, R dt, R a_dt2) {
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) * W, j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i >= g.n[0] || j >= g.n[1]) return;
    const int z = blockIdx.z % g.n[2], a = blockIdx.z / g.n[2];
    const int b = a == 2 ? 0 : a + 1, c = a == 0 ? 2 : a - 1;
    const int sy = g.P[0], sz = g.P[0] * g.P[1];
    const int q = (int)g.at(i, j, z);
    const R *f = pick(B, a) + q;
    Nodes<R, W> col[11];
#pragma unroll
    for (int m = 0; m < 11; ++m) col[m] = ld<W>(f + (m - 5) * sz);
    const Nodes<R, W> L = laplace<R, W>(f, sy, col, k);
    const int sb = b == 0 ? 1 : (b == 1 ? sy : sz), sc = c == 0 ? 1 : (c == 1 ? sy : sz);
    // curl_a = d_b F_c - d_c F_b
    const Nodes<R, W> e1 = diff<R, W>(pick(E, c) + q, b, sb, true, k), e2 = diff<R, W>(pick(E, b) + q, c, sc, true, k);
    Nodes<R, W> j1, j2;
    if (i >= 2 && i + W + 2 < g.n[0] && j >= 2 && j + 3 < g.n[1] && z >= 2 && z + 3 < g.n[2]) {
        j1 = diff<R, W>(pick(J, c) + q, b, sb, true, k);
        j2 = diff<R, W>(pick(J, b) + q, c, sc, true, k);
    } else {
        const int xb = b == 0 ? i : (b == 1 ? j : z), xc = c == 0 ? i : (c == 1 ? j : z);
        const int nb = b == 0 ? g.n[0] : (b == 1 ? g.n[1] : g.n[2]), nc = c == 0 ? g.n[0] : (c == 1 ? g.n[1] : g.n[2]);
        j1 = diff_wrap<R, W>(pick(J, c) + q, b, sb, xb, nb, k);
        j2 = diff_wrap<R, W>(pick(J, b) + q, c, sc, xc, nc, k);
    }
    R *out = a == 0 ? O0 : (a == 1 ? O1 : O2);
#pragma unroll
    for (int w = 0; w < W; ++w)
        out[q + w] = col[5].v[w] + ab_dt2 * L.v[w] - dt * (e1.v[w] - e2.v[w]) + a_dt2 * (j1.v[w] - j2.v[w]);
}

// One Chebyshev sweep (Saad's three-term form, see field_update_impl):
// r = rhs - X + kk L X, X_new = X + c1 (X - X_prev) + c2 r.  A thread marches
// through zper planes of one component with the 11 nodes along z in registers.
// FP32 on large meshes: bound by the latency of the neighbours' loads (L1 and
// L2), so a plane's streams are loaded one plane ahead; FP64: by the part's FP64
// rate (about 40 operations a node and component); small meshes: by launch and
// load latency, so the march is cut until every SM has threads.  Blocks of 32 x
// 16 nodes and six planes (256 x 128 x 128 nodes, the whole field update: 1.66 ms;
// 64 x 8 nodes 1.68; 16 planes 1.80; without the loads ahead 2.16).
template <typename R, int W>
__global__ void __launch_bounds__(256) k_cheb(Geom g, const __grid_constant__ Coef<R> k, Vec3<R> X, Vec3<R> Xp,
                                              Vec3<R> Rh, R *O0, R *O1, R *O2, R kk, R c1, R c2, int zper, int nzc) {
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) * W, j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i >= g.n[0] || j >= g.n[1]) return;
    const int a = blockIdx.z / nzc, z0 = (blockIdx.z - a * nzc) * zper, z1 = min(g.n[2], z0 + zper);
    const int sy = g.P[0], sz = g.P[0] * g.P[1];
    int q = (int)g.at(i, j, z0);
    const R *f = pick(X, a), *fp = pick(Xp, a), *rh = pick(Rh, a);
    R *out = a == 0 ? O0 : (a == 1 ? O1 : O2);
    Nodes<R, W> col[11];
#pragma unroll
    for (int m = 0; m < 11; ++m) col[m] = ld<W>(f + q + (m - 5) * sz);
    // the previous iterate and rhs one plane ahead, the column's top two
    Nodes<R, W> xpn = ld<W>(fp + q), rzn = ld<W>(rh + q), top = col[10];
    if (z0 + 1 < z1) top = ld<W>(f + q + 6 * sz);
    for (int z = z0;;) {
        const Nodes<R, W> xp = xpn, rz = rzn, next = top;
        if (z + 1 < z1) {
            xpn = ld<W>(fp + q + sz);
            rzn = ld<W>(rh + q + sz);
            if (z + 2 < z1) top = ld<W>(f + q + 7 * sz);
        }
        const Nodes<R, W> L = laplace<R, W>(f + q, sy, col, k);
        Nodes<R, W> nv;
#pragma unroll
        for (int w = 0; w < W; ++w) {
            const R x = col[5].v[w];
            const R r = rz.v[w] - x + kk * L.v[w];
            nv.v[w] = x + c1 * (x - xp.v[w]) + c2 * r;
        }
        store_nodes<R, W>(out, g, q, i, j, z, nv);
        if (++z >= z1) break;
        q += sz;
#pragma unroll
        for (int m = 0; m < 10; ++m) col[m] = col[m + 1];
        col[10] = next;
    }
}

// ---- every sweep in one launch, on small meshes ----
// The components do not mix, so one thread-block cluster takes a component from
// the first sweep to the last: its 16 CTAs hold 1/16 of the planes each, the
// iterate, the previous one and the right-hand side in shared memory, read the
// planes above and below from one another's shared memory and meet at the
// cluster's hardware barrier after each sweep.  Sweeps of their own cost 6.3 us
// (FP32) to 8.4 us (FP64) each however small the mesh; past a line they win all
// the same: they use all SMs, the clusters 48 (cluster_pays).
constexpr int kClusterCtas = 16, kClusterThreads = 512, kClusterSweeps = 64;

template <typename R>
struct Sweeps {
    R c1[kClusterSweeps], c2[kClusterSweeps];
    int n;
};

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// Address of this CTA's shared word p in the shared memory of CTA `rank`.
__device__ __forceinline__ uint32_t map_shared(const void *p, uint32_t rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return r;
}
template <int W, typename R>
__device__ __forceinline__ Nodes<R, W> ld_cluster(uint32_t a) {
    Nodes<R, W> r;
    if constexpr (sizeof(R) == 4 && W == 2)
        asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(r.v[0]), "=f"(r.v[1]) : "r"(a) : "memory");
    else if constexpr (sizeof(R) == 4)
        asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(r.v[0]) : "r"(a) : "memory");
    else if constexpr (W == 2)
        asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(r.v[0]), "=d"(r.v[1]) : "r"(a) : "memory");
    else
        asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(r.v[0]) : "r"(a) : "memory");
    return r;
}

// First plane of CTA r of the cluster.
__host__ __device__ __forceinline__ int first_plane(int r, int nz) { return r * nz / kClusterCtas; }

template <typename R, int W>
__global__ void __launch_bounds__(kClusterThreads, 1)
    k_cheb_cluster(Geom g, const __grid_constant__ Coef<R> k, const __grid_constant__ Sweeps<R> sw, R kk, Vec3<R> B, Vec3<R> Rh,
                   R *O0, R *O1, R *O2) {
    extern __shared__ __align__(16) char smem[];
    __shared__ uint32_t plane[2][24];   // per buffer the shared addresses of planes z0 - 5 .. z1 + 4, wherever they are
    const int a = blockIdx.x / kClusterCtas, rank = (int)cluster_rank();
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2], n2 = nx * ny;
    const int z0 = first_plane(rank, nz), np = first_plane(rank + 1, nz) - z0;
    const int pmax = (nz + kClusterCtas - 1) / kClusterCtas;
    R *buf[2] = {(R *)smem, (R *)smem + (size_t)pmax * n2};
    R *rh = (R *)smem + (size_t)2 * pmax * n2;
    const R *f = pick(B, a), *fr = pick(Rh, a);
    for (int t = threadIdx.x; t < np * n2; t += kClusterThreads) {
        const int q = (int)g.at(t % nx, (t / nx) % ny, z0 + t / n2);
        buf[0][t] = buf[1][t] = f[q];
        rh[t] = fr[q];
    }
    if ((int)threadIdx.x < 2 * (np + 10)) {
        const int b = threadIdx.x & 1, m = threadIdx.x >> 1, z = wrap(z0 - 5 + m, nz);
        int r = z * kClusterCtas / nz;
        while (first_plane(r + 1, nz) <= z) ++r;
        while (first_plane(r, nz) > z) --r;
        plane[b][m] = map_shared(buf[b] + (size_t)(z - first_plane(r, nz)) * n2, (uint32_t)r);
    }
    __syncthreads();
    cluster_barrier();
    const int cols = (nx / W) * ny;
    constexpr int N = even<W>(5);
    // neighbours of a column along x (as W-node groups) and y, wrapped, relative to it
    int ox[2 * N / W], oy[10], o = 0;
    auto column = [&](int c) {
        const int y = c / (nx / W), x = (c - y * (nx / W)) * W;
        o = y * nx + x;
#pragma unroll
        for (int m = 0; m < 2 * N / W; ++m) {
            const int d = m < N / W ? m * W - N : (m + 1) * W - N, v = x + d;
            ox[m] = d + (v < 0 ? nx : (v >= nx ? -nx : 0));
        }
#pragma unroll
        for (int m = 0; m < 10; ++m) {
            const int d = m < 5 ? m - 5 : m - 4, v = y + d;
            oy[m] = (d + (v < 0 ? ny : (v >= ny ? -ny : 0))) * nx;
        }
    };
    const bool single = cols <= kClusterThreads;   // a thread keeps its column
    if (single && (int)threadIdx.x < cols) column(threadIdx.x);
    for (int it = 0; it < sw.n; ++it) {
        const int cur = it & 1;
        const R c1 = sw.c1[it], c2 = sw.c2[it];
        for (int c = threadIdx.x; c < cols; c += kClusterThreads) {
            if (!single) column(c);
            Nodes<R, W> col[11];
#pragma unroll
            for (int m = 0; m < 11; ++m) col[m] = ld_cluster<W, R>(plane[cur][m] + o * (int)sizeof(R));
            for (int p = 0;;) {
                const R *u = (cur ? buf[1] : buf[0]) + p * n2 + o;
                R row[2 * N + W];
#pragma unroll
                for (int m = 0; m < 2 * N / W; ++m) {
                    const Nodes<R, W> t = ld<W>(u + ox[m]);
#pragma unroll
                    for (int w = 0; w < W; ++w) row[(m < N / W ? m * W : (m + 1) * W) + w] = t.v[w];
                }
#pragma unroll
                for (int w = 0; w < W; ++w) row[N + w] = col[5].v[w];
                R sx[W], sy[W], sz[W];
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    sx[w] = sy[w] = sz[w] = k.lap[0] * col[5].v[w];
#pragma unroll
                    for (int d = 1; d <= 5; ++d) {
                        sx[w] += k.lap[d] * (row[N + w + d] + row[N + w - d]);
                        sz[w] += k.lap[d] * (col[5 + d].v[w] + col[5 - d].v[w]);
                    }
                }
#pragma unroll
                for (int d = 1; d <= 5; ++d) {
                    const Nodes<R, W> hi = ld<W>(u + oy[4 + d]), lo = ld<W>(u + oy[5 - d]);
#pragma unroll
                    for (int w = 0; w < W; ++w) sy[w] += k.lap[d] * (hi.v[w] + lo.v[w]);
                }
                R *nw = (cur ? buf[0] : buf[1]) + p * n2 + o;   // the previous iterate, replaced node by node
                const R *rp = rh + p * n2 + o;
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    const R L = sx[w] * k.ih2[0] + sy[w] * k.ih2[1] + sz[w] * k.ih2[2];
                    const R xv = col[5].v[w];
                    const R r = rp[w] - xv + kk * L;
                    nw[w] = xv + c1 * (xv - nw[w]) + c2 * r;
                }
                if (++p >= np) break;
#pragma unroll
                for (int m = 0; m < 10; ++m) col[m] = col[m + 1];
                col[10] = ld_cluster<W, R>(plane[cur][p + 10] + o * (int)sizeof(R));
            }
        }
        cluster_barrier();   // every node written before any is read, every read done before the next sweep writes
    }
    const R *res = (sw.n & 1) ? buf[1] : buf[0];
    R *out = a == 0 ? O0 : (a == 1 ? O1 : O2);
    for (int t = threadIdx.x; t < np * cols; t += kClusterThreads) {
        const int x = (t % (nx / W)) * W, y = (t / (nx / W)) % ny, p = t / cols;
        Nodes<R, W> v;
#pragma unroll
        for (int w = 0; w < W; ++w) v.v[w] = res[p * n2 + y * nx + x + w];
        store_nodes<R, W>(out, g, (int)g.at(x, y, z0 + p), x, y, z0 + p, v);
    }
}

// Whether the cluster is faster than a launch per sweep: both estimated in us
// from measurements of the whole field update (dt = dx / 2; tolerance 1e-6 in
// FP32, 1e-12 in FP64).  What counts in the cluster is the heaviest CTA, with p
// planes: its warps' columns and, for each, the 11 nodes fetched before the
// march and the planes marched; with W = 1 a column holds half the work.  In
// FP64 a warp's rate shows from four warps on (below them its latency), and a
// second pass over the columns costs a full one.  Launches and cluster, us:
//   FP32 16^3 96, 33; 32^3 102, 58; 32 x 32 x 224 215, 156; 41^3 136, 115;
//   48^3 167, 122; 64 x 48 x 16 102, 105; 64 x 64 x 16 119, 126; 64 x 64 x 17
//   115, 165 (8192 nodes in one CTA, 4096 in the others); 52 x 54 x 17 103, 124;
//   61 x 61 x 17 134, 184; 63 x 47 x 33 137, 164.
//   FP64 16^3 203, 105; 8 x 8 x 64 211, 281; 9 x 9 x 64 202, 167; 12 x 12 x 48
//   204, 222; 16 x 20 x 17 203, 226; 17^3 202, 190; 20^3 212, 281;
//   24 x 24 x 16 212, 199; 28 x 24 x 16 211, 230.
// Of 148 meshes measured the estimates choose the slower form (by over 3 %) five
// times, by 4 to 20 %; limits of 70,000 and 6,000 nodes in all chose it 61 times.
template <typename R, int W>
static bool cluster_pays(const Geom &g) {
    const int p = (g.n[2] + kClusterCtas - 1) / kClusterCtas, cols = g.n[0] / W * g.n[1];
    int warps = (cols + 31) / 32;
    if (sizeof(R) == 4) {
        const double launches = 70.0 + 0.65e-3 * (double)g.cells();
        return 27.0 + warps * (W == 2 ? 1.0 : 0.62) * (1.1 + 0.45 * p) <= (launches > 100.0 ? launches : 100.0);
    }
    constexpr int kPass = kClusterThreads / 32;
    if (warps > kPass) warps = (warps + kPass - 1) / kPass * kPass;
    if (warps < 4) warps = 4;
    return 38.0 + p * warps * (W == 2 ? 17.3 : 7.7) <= 201.0;
}

template <typename R, int W>
static bool cluster_fits(const Geom &g, int sweeps, size_t &smem) {
    const int pmax = (g.n[2] + kClusterCtas - 1) / kClusterCtas;
    smem = (size_t)3 * pmax * g.n[0] * g.n[1] * sizeof(R);
    if (g.n[0] < 8 || g.n[1] < 8 || g.n[2] < kClusterCtas || pmax + 10 > 24 || sweeps > kClusterSweeps || smem > 224 * 1024 ||
        !cluster_pays<R, W>(g))
        return false;
    // once per device and kernel: whether a cluster can be resident (contexts may
    // step from several threads: a thread that sees `asked` also sees `ok`)
    static std::atomic<unsigned long long> asked{0}, ok{0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(asked.load(std::memory_order_acquire) & bit)) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = kClusterCtas;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(3 * kClusterCtas);
        cfg.blockDim = dim3(kClusterThreads);
        cfg.dynamicSmemBytes = 224 * 1024;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int n = 0;
        bool can = cudaFuncSetAttribute(k_cheb_cluster<R, W>, cudaFuncAttributeMaxDynamicSharedMemorySize, 224 * 1024) == cudaSuccess &&
                   cudaFuncSetAttribute(k_cheb_cluster<R, W>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                   cudaOccupancyMaxActiveClusters(&n, k_cheb_cluster<R, W>, &cfg) == cudaSuccess && n >= 1;
        if (!can) cudaGetLastError();
        if (can) ok.fetch_or(bit, std::memory_order_relaxed);
        asked.fetch_or(bit, std::memory_order_release);
    }
    return (ok.load(std::memory_order_relaxed) & bit) != 0;
}

// E_new = E + dt (curl^- (alpha B_new + beta B_old) - J), ghosts of E included.
// E is read at the thread's own nodes only, so it is updated in place.
template <typename R, int W>
__global__ void __launch_bounds__(256) k_e_update_lin(Geom g, const __grid_constant__ Coef<R> k, R *E0, R *E1, R *E2,
                                                      Vec3<R> Bn, Vec3<R> Bo, Vec3<R> J, R alpha, R beta, R dt) {
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) * W, j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i >= g.n[0] || j >= g.n[1]) return;
    const int z = blockIdx.z % g.n[2], a = blockIdx.z / g.n[2];
    const int b = a == 2 ? 0 : a + 1, c = a == 0 ? 2 : a - 1;
    const int sy = g.P[0], sz = g.P[0] * g.P[1];
    const int sb = b == 0 ? 1 : (b == 1 ? sy : sz), sc = c == 0 ? 1 : (c == 1 ? sy : sz);
    const int q = (int)g.at(i, j, z);
    const Nodes<R, W> n1 = diff<R, W>(pick(Bn, c) + q, b, sb, false, k), n2 = diff<R, W>(pick(Bn, b) + q, c, sc, false, k);
    const Nodes<R, W> o1 = diff<R, W>(pick(Bo, c) + q, b, sb, false, k), o2 = diff<R, W>(pick(Bo, b) + q, c, sc, false, k);
    const Nodes<R, W> cur = ld<W>(pick(J, a) + q);
    R *E = a == 0 ? E0 : (a == 1 ? E1 : E2);
    Nodes<R, W> e = ld<W>((const R *)E + q);
#pragma unroll
    for (int w = 0; w < W; ++w)
        e.v[w] += dt * (alpha * (n1.v[w] - n2.v[w]) + beta * (o1.v[w] - o2.v[w]) - cur.v[w]);
    store_nodes<R, W>(E, g, q, i, j, z, e);
}

// E_new = E + dt (curl^- (alpha B_new + beta B_old) - J)   (eq:enplus1, c^2 mu0 = 1)
template <typename R>
struct MixB {
    const R *Bn, *Bo;
    R al, be;
};

template <typename R>
__global__ void k_e_update(Geom g, FieldCoef k, R *E0, R *E1, R *E2, Vec3<R> Bn, Vec3<R> Bo, Vec3<R> J, R alpha,
                           R beta, R dt) {
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= g.cells()) return;
    Nb<R> nb{g, {0, 0, 0}};
    unflatten(t, g, nb.c[0], nb.c[1], nb.c[2]);
    int64_t q = g.at(nb.c[0], nb.c[1], nb.c[2]);
    R *E[3] = {E0, E1, E2};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int b = (a + 1) % 3, c = (a + 2) % 3;
        R cur = alpha * (nb.dminus(Bn.p[c], b, k) - nb.dminus(Bn.p[b], c, k)) +
                beta * (nb.dminus(Bo.p[c], b, k) - nb.dminus(Bo.p[b], c, k));
        E[a][q] = E[a][q] + dt * (cur - J.p[a][q]);
    }
}

// Periodic ghost fill of E (from its own interior) and B (from src, which may
// be a different array than B: the converged relaxation iterate).
template <typename R>
__global__ void k_ghost_fill(Geom g, R *E0, R *E1, R *E2, const R *S0, const R *S1, const R *S2, R *B0, R *B1, R *B2,
                             int e_ghost_only) {
    int64_t total = g.padded_size();
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= total) return;
    int i = (int)(t % g.P[0]);
    int64_t r = t / g.P[0];
    int j = (int)(r % g.P[1]);
    int k = (int)(r / g.P[1]);
    int ci = i - g.G, cj = j - g.G, ck = k - g.G;
    bool ghost = ci < 0 || cj < 0 || ck < 0 || ci >= g.n[0] || cj >= g.n[1] || ck >= g.n[2];
    int64_t src = g.at(wrap(ci, g.n[0]), wrap(cj, g.n[1]), wrap(ck, g.n[2]));
    if (ghost || !e_ghost_only) {
        E0[t] = E0[src]; E1[t] = E1[src]; E2[t] = E2[src];
    }
    B0[t] = S0[src]; B1[t] = S1[src]; B2[t] = S2[src];
}

template <typename R>
static Vec3<R> v3(void *const p[3]) {
    return Vec3<R>{{(const R *)p[0], (const R *)p[1], (const R *)p[2]}};
}

static FieldCoef field_coef(const Ctx &c) {
    FieldCoef k;
    double h[3] = {c.d.dx, c.d.dy, c.d.dz};
    for (int m = 0; m < 3; ++m) k.k[m] = c.fd[m];
    for (int m = 0; m < 6; ++m) k.lap[m] = c.lap[m];
    for (int a = 0; a < 3; ++a) {
        k.ih[a] = 1.0 / h[a];
        k.ih2[a] = 1.0 / (h[a] * h[a]);
    }
    return k;
}

template <typename R>
static Coef<R> coef_of(const FieldCoef &k) {
    Coef<R> r;
    for (int m = 0; m < 3; ++m) {
        r.k[m] = (R)k.k[m];
        r.ih[m] = (R)k.ih[m];
        r.ih2[m] = (R)k.ih2[m];
    }
    for (int m = 0; m < 6; ++m) r.lap[m] = (R)k.lap[m];
    return r;
}

// Planes a thread marches through: six, or as many as leave kMarchBlocks blocks
// (six per SM; 64^3 nodes: 0.216 ms with one plane, 0.232 with two, 0.277 with
// six; 128 x 64 x 64: 0.330 with two or three, 0.341 with one, 0.360 with six).
constexpr int kMarchBlocks = 912;

template <typename R, int W>
static cudaError_t field_update_impl(Ctx &c) {
    const Geom &g = c.g;
    const Coef<R> k = coef_of<R>(field_coef(c));
    // dt of this solve: the step, or the drift of a 4th-order substep
    double al = c.d.alpha, be = 1.0 - c.d.alpha, dt = c.drift_dt;
    double kk = al * al * dt * dt;
    const Ctx::Cheb &ch = c.cheb[c.cheb_sel];
    cudaError_t e;
    // blocks of 256 threads (64 for FP64, whose rate wants every SM busy), as wide
    // along x as the rows need, up to 16 threads
    const int nx = (g.n[0] + W - 1) / W, threads = sizeof(R) == 8 ? 64 : 256;
    int bx = 8;
    while (bx < 16 && bx < nx) bx *= 2;
    const dim3 blk((unsigned)bx, (unsigned)(threads / bx));
    dim3 grid((unsigned)((nx + bx - 1) / bx), (unsigned)((g.n[1] + blk.y - 1) / blk.y), (unsigned)(3 * g.n[2]));
    k_rhs_lin<R, W><<<grid, blk, 0, c.st>>>(g, k, v3<R>(c.E), v3<R>(c.B), v3<R>(c.J), (R *)c.R[0], (R *)c.R[1],
                                            (R *)c.R[2], (R)(al * be * dt * dt), (R)dt, (R)(al * dt * dt));
    ++c.nlaunch;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // Chebyshev semi-iteration on the spectrum [1, lmax] of the SPD operator,
    // starting from B^n (Saad, Iterative Methods, Alg. 12.1 in 3-term form).
    double theta = ch.theta, delta = ch.delta;
    int zper = 6;
    while (zper > 1 && (int64_t)grid.x * grid.y * 3 * ((g.n[2] + zper - 1) / zper) < kMarchBlocks) --zper;
    const int nzc = (g.n[2] + zper - 1) / zper;
    const dim3 pg(grid.x, grid.y, (unsigned)(3 * nzc));
    void **cur = c.B, **prev = c.B;
    void **bufs[2] = {c.Xa, c.Xb};
    int nb = 0;
    double rho_prev = delta > 0 ? delta / theta : 0.0;
    size_t smem = 0;
    const bool cluster = cluster_fits<R, W>(g, ch.iters, smem);
    Sweeps<R> sw;
    sw.n = ch.iters;
    for (int it = 0; it < ch.iters; ++it) {
        double c1, c2;
        if (it == 0) {
            c1 = 0.0;
            c2 = 1.0 / theta;
        } else {
            double sigma = theta / delta;
            double rho = 1.0 / (2.0 * sigma - rho_prev);
            c1 = rho * rho_prev;
            c2 = 2.0 * rho / delta;
            rho_prev = rho;
        }
        if (cluster) {
            sw.c1[it] = (R)c1;
            sw.c2[it] = (R)c2;
            continue;
        }
        // output: a scratch buffer that is neither cur nor (when prev is B) B
        void **out = (prev == c.B || prev == cur) ? bufs[nb] : prev;
        if (out == cur) out = bufs[1 - nb];
        k_cheb<R, W><<<pg, blk, 0, c.st>>>(g, k, v3<R>(cur), v3<R>(prev), v3<R>(c.R), (R *)out[0], (R *)out[1],
                                           (R *)out[2], (R)kk, (R)c1, (R)c2, zper, nzc);
        ++c.nlaunch;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        prev = cur;
        cur = out;
        nb = (out == bufs[0]) ? 1 : 0;
    }
    if (cluster) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = kClusterCtas;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(3 * kClusterCtas);
        cfg.blockDim = dim3(kClusterThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = c.st;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        cur = c.Xa;
        e = cudaLaunchKernelEx(&cfg, k_cheb_cluster<R, W>, g, k, sw, (R)kk, v3<R>(c.B), v3<R>(c.R), (R *)cur[0], (R *)cur[1],
                               (R *)cur[2]);
        ++c.nlaunch;
        if (e != cudaSuccess) return e;
    }
    c.last_iters = ch.iters;
    c.last_kk = kk;
    c.filtered_after_solve = false;
    // eq:enplus1 with B^{n+1} = cur, B^n = B
    k_e_update_lin<R, W><<<grid, blk, 0, c.st>>>(g, k, (R *)c.E[0], (R *)c.E[1], (R *)c.E[2], v3<R>(cur), v3<R>(c.B),
                                                 v3<R>(c.J), (R)al, (R)be, (R)dt);
    ++c.nlaunch;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // the last iterate, ghosts and all, becomes B; the old B joins the scratch
    for (int a = 0; a < 3 && cur != c.B; ++a) {
        void *t = c.B[a];
        c.B[a] = cur[a];
        cur[a] = t;
    }
    return cudaSuccess;
}

// Explicit FDTD variant (the cold-beam comparison of Sec. VIII): Yee's
// leap-frog with the same staggered differences, B in two half steps so that
// E and B stay at one time level:
//   B^{n+1/2} = B^n - dt/2 curl^+ E^n,  E^{n+1} = E^n + dt (curl^- B^{n+1/2} - J),
//   B^{n+1} = B^{n+1/2} - dt/2 curl^+ E^{n+1}.
// The half steps are k_rhs with alpha = 0, the full step k_e_update with
// alpha = 1.
template <typename R>
static cudaError_t field_update_explicit_impl(Ctx &c) {
    const Geom &g = c.g;
    FieldCoef k = field_coef(c);
    unsigned blocks = (unsigned)((g.cells() + 255) / 256);
    unsigned pblocks = (unsigned)((g.padded_size() + 255) / 256);
    const R half = (R)(0.5 * c.drift_dt);
    cudaError_t e;
    for (int pass = 0; pass < 2; ++pass) {
        // B half step into the scratch R, then B := R with its ghost layers
        k_rhs<R><<<blocks, 256, 0, c.st>>>(g, k, v3<R>(c.E), v3<R>(c.B), v3<R>(c.J), (R *)c.R[0], (R *)c.R[1],
                                           (R *)c.R[2], (R)0, half, (R)0);
        ++c.nlaunch;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        k_ghost_fill<R><<<pblocks, 256, 0, c.st>>>(g, (R *)c.E[0], (R *)c.E[1], (R *)c.E[2], (const R *)c.R[0],
                                                   (const R *)c.R[1], (const R *)c.R[2], (R *)c.B[0], (R *)c.B[1],
                                                   (R *)c.B[2], 1);
        ++c.nlaunch;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if (pass == 1) break;
        // E full step with B^{n+1/2}, then E's ghost layers (B copies onto itself)
        k_e_update<R><<<blocks, 256, 0, c.st>>>(g, k, (R *)c.E[0], (R *)c.E[1], (R *)c.E[2], v3<R>(c.B), v3<R>(c.B),
                                                v3<R>(c.J), (R)1, (R)0, (R)c.drift_dt);
        ++c.nlaunch;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        k_ghost_fill<R><<<pblocks, 256, 0, c.st>>>(g, (R *)c.E[0], (R *)c.E[1], (R *)c.E[2], (const R *)c.B[0],
                                                   (const R *)c.B[1], (const R *)c.B[2], (R *)c.B[0], (R *)c.B[1],
                                                   (R *)c.B[2], 1);
        ++c.nlaunch;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    c.last_iters = 0;   // no relaxation
    c.last_kk = 0.0;
    return cudaSuccess;
}

// ---------------------------------------------------------------------------
// Divergence filter (the paper's divergence cleaning of E for the direct
// current, and the periodic filter of E and B in long FP32 runs): each pass is
// one simultaneous smoothing step
//   E += tau grad^+ (div^- E - rho),   B += tau grad^- (div^+ B),
// tau = 1 / max(sum_a K_a^2), which removes the Nyquist-scale error in one
// pass and damps every other non-constant mode.
// ---------------------------------------------------------------------------
template <typename R>
__global__ void k_div_error(Geom g, FieldCoef k, Vec3<R> F, const double *rho, int plus, R *out) {
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= g.cells()) return;
    Nb<R> nb{g, {0, 0, 0}};
    unflatten(t, g, nb.c[0], nb.c[1], nb.c[2]);
    R d = plus ? nb.dplus(F.p[0], 0, k) + nb.dplus(F.p[1], 1, k) + nb.dplus(F.p[2], 2, k)
               : nb.dminus(F.p[0], 0, k) + nb.dminus(F.p[1], 1, k) + nb.dminus(F.p[2], 2, k);
    out[g.at(nb.c[0], nb.c[1], nb.c[2])] = rho ? d - (R)rho[t] : d;
}

template <typename R>
__global__ void k_grad_add(Geom g, FieldCoef k, const R *r, R *F0, R *F1, R *F2, R tau, int plus) {
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= g.cells()) return;
    Nb<R> nb{g, {0, 0, 0}};
    unflatten(t, g, nb.c[0], nb.c[1], nb.c[2]);
    int64_t q = g.at(nb.c[0], nb.c[1], nb.c[2]);
    R *F[3] = {F0, F1, F2};
#pragma unroll
    for (int a = 0; a < 3; ++a) F[a][q] += tau * (plus ? nb.dplus(r, a, k) : nb.dminus(r, a, k));
}

template <typename R>
static cudaError_t divergence_filter_impl(Ctx &c) {
    // rho at the particles' current positions; in the mixed form they are sorted
    // first, since the tile kernel adds a particle that left its sorted cell
    // site by site in FP64 (64^3 x 16, TSC, tiles sorted every 20 steps: a pass
    // of five filtered steps took 25.5 ms without the sort, 12.9 with it)
    cudaError_t e = cudaSuccess;
    for (int s = 0; s < c.nspecies && e == cudaSuccess; ++s)
        if (!c.fp64 && c.sp[s].n > 0 && !c.sp[s].fresh) e = launch_sort(c, s);
    if (e == cudaSuccess) e = launch_rho(c);
    if (e != cudaSuccess) return e;
    const Geom &g = c.g;
    FieldCoef k = field_coef(c);
    unsigned blocks = (unsigned)((g.cells() + 255) / 256);
    const R tau = (R)c.filter_tau;
    // scratch: the relaxation iterates (free after a solve); the solve's
    // right-hand side in R stays for the residual diagnostics
    R *eE = (R *)c.Xa[0], *eB = (R *)c.Xa[1];
    for (int p = 0; p < c.filter_passes; ++p) {
        k_div_error<R><<<blocks, 256, 0, c.st>>>(g, k, v3<R>(c.E), c.rho, 0, eE);
        k_grad_add<R><<<blocks, 256, 0, c.st>>>(g, k, eE, (R *)c.E[0], (R *)c.E[1], (R *)c.E[2], tau, 1);
        k_div_error<R><<<blocks, 256, 0, c.st>>>(g, k, v3<R>(c.B), nullptr, 1, eB);
        k_grad_add<R><<<blocks, 256, 0, c.st>>>(g, k, eB, (R *)c.B[0], (R *)c.B[1], (R *)c.B[2], tau, 0);
        c.nlaunch += 4;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    unsigned pblocks = (unsigned)((g.padded_size() + 255) / 256);
    k_ghost_fill<R><<<pblocks, 256, 0, c.st>>>(g, (R *)c.E[0], (R *)c.E[1], (R *)c.E[2], (const R *)c.B[0],
                                               (const R *)c.B[1], (const R *)c.B[2], (R *)c.B[0], (R *)c.B[1],
                                               (R *)c.B[2], 1);
    ++c.nlaunch;
    c.filtered_after_solve = true;   // B moved since the last solve: its residual no longer measures it
    return cudaGetLastError();
}

cudaError_t launch_divergence_filter(Ctx &c) {
    return c.fp64 ? divergence_filter_impl<double>(c) : divergence_filter_impl<float>(c);
}

cudaError_t launch_field_update(Ctx &c) {
    if (c.field_solver == PP_FIELD_EXPLICIT)
        return c.fp64 ? field_update_explicit_impl<double>(c) : field_update_explicit_impl<float>(c);
    if (c.g.n[0] % 2 == 0) return c.fp64 ? field_update_impl<double, 2>(c) : field_update_impl<float, 2>(c);
    return c.fp64 ? field_update_impl<double, 1>(c) : field_update_impl<float, 1>(c);
}

template <typename R>
static cudaError_t ghost_fill_impl(Ctx &c, void *const sE[3], void *const sB[3]) {
    (void)sE;
    unsigned pblocks = (unsigned)((c.g.padded_size() + 255) / 256);
    k_ghost_fill<R><<<pblocks, 256, 0, c.st>>>(c.g, (R *)c.E[0], (R *)c.E[1], (R *)c.E[2], (const R *)sB[0],
                                               (const R *)sB[1], (const R *)sB[2], (R *)c.B[0], (R *)c.B[1],
                                               (R *)c.B[2], 1);
    ++c.nlaunch;
    return cudaGetLastError();
}

cudaError_t launch_ghost_fill(Ctx &c, void *const sE[3], void *const sB[3]) {
    return c.fp64 ? ghost_fill_impl<double>(c, sE, sB) : ghost_fill_impl<float>(c, sE, sB);
}

// ---------------------------------------------------------------------------
// FP64 mesh diagnostics: sums (energies, charge) and maxima (|rho|, Gauss
// residual, its drift from G_0, div B, relaxation residual, |rhs|).
// ---------------------------------------------------------------------------
constexpr int kDiagSums = 4, kDiagMax = 6, kDiagN = kDiagSums + kDiagMax;

template <typename R>
__global__ void k_mesh_diag(Geom g, FieldCoef k, Vec3<R> E, Vec3<R> B, Vec3<R> Rh, const double *rho, double *G0,
                            int capture, double kk, double *partial) {
    double v[kDiagN];
    for (int m = 0; m < kDiagN; ++m) v[m] = 0.0;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < g.cells(); t += (int64_t)gridDim.x * blockDim.x) {
        Nb<R> nb{g, {0, 0, 0}};
        unflatten(t, g, nb.c[0], nb.c[1], nb.c[2]);
        int64_t q = g.at(nb.c[0], nb.c[1], nb.c[2]);
        double e0 = E.p[0][q], e1 = E.p[1][q], e2 = E.p[2][q];
        double b0 = B.p[0][q], b1 = B.p[1][q], b2 = B.p[2][q];
        v[0] += 0.5 * (e0 * e0 + e1 * e1 + e2 * e2);
        v[1] += 0.5 * (b0 * b0 + b1 * b1 + b2 * b2);
        v[2] += 0.5 * e0 * e0;
        double r = rho[t];
        v[3] += r;
        double divE = 0.0, divB = 0.0;
        for (int a = 0; a < 3; ++a) {
            divE += (double)nb.dminus(E.p[a], a, k);
            divB += (double)nb.dplus(B.p[a], a, k);
        }
        double G = divE - r;
        if (capture) G0[t] = G;
        v[4] = fmax(v[4], fabs(r));
        v[5] = fmax(v[5], fabs(G));
        v[6] = fmax(v[6], fabs(G - G0[t]));
        v[7] = fmax(v[7], fabs(divB));
        for (int a = 0; a < 3; ++a) {
            double res = (double)Rh.p[a][q] - ((double)B.p[a][q] - kk * (double)nb.lap(B.p[a], k));
            v[8] = fmax(v[8], fabs(res));
            v[9] = fmax(v[9], fabs((double)Rh.p[a][q]));
        }
    }
    __shared__ double sh[kDiagN][256];
    for (int m = 0; m < kDiagN; ++m) sh[m][threadIdx.x] = v[m];
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s)
            for (int m = 0; m < kDiagN; ++m) {
                double a = sh[m][threadIdx.x], b = sh[m][threadIdx.x + s];
                sh[m][threadIdx.x] = m < kDiagSums ? a + b : fmax(a, b);
            }
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int m = 0; m < kDiagN; ++m) partial[(int64_t)blockIdx.x * kDiagN + m] = sh[m][0];
}

__global__ void k_diag_final(const double *partial, int nblk, double *out) {
    int m = threadIdx.x;
    if (m >= kDiagN) return;
    double acc = 0.0;
    for (int b = 0; b < nblk; ++b) {
        double v = partial[(int64_t)b * kDiagN + m];
        acc = m < kDiagSums ? acc + v : fmax(acc, v);
    }
    out[m] = acc;
}

constexpr int kDiagBlocks = 512;

template <typename R>
static cudaError_t mesh_diag_impl(Ctx &c, double *host_out) {
    FieldCoef k = field_coef(c);
    int capture = c.have_G0 ? 0 : 1;
    double kk = c.last_kk;   // residual of the last solve
    int64_t want = (c.g.cells() + 255) / 256;
    int nblk = (int)(want < kDiagBlocks ? want : kDiagBlocks);
    k_mesh_diag<R><<<nblk, 256, 0, c.st>>>(c.g, k, v3<R>(c.E), v3<R>(c.B), v3<R>(c.R), c.rho, c.G0, capture, kk, c.d_red);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_diag_final<<<1, 32, 0, c.st>>>(c.d_red, nblk, c.d_out);
    c.nlaunch += 2;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    e = cudaMemcpyAsync(host_out, c.d_out, sizeof(double) * kDiagN, cudaMemcpyDeviceToHost, c.st);
    if (e != cudaSuccess) return e;
    c.have_G0 = true;
    return cudaSuccess;
}

cudaError_t launch_mesh_diag(Ctx &c, double *host_out) {
    return c.fp64 ? mesh_diag_impl<double>(c, host_out) : mesh_diag_impl<float>(c, host_out);
}

}  // namespace pp
