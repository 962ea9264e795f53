// Particle-side kernels of one time step:
//   k_links      indirect-addressing gather of fluid-particle links into the
//                fixed index array (Sec. 3), curved bounce-back of f and g on
//                each link (Sec. 2.3) and the momentum-exchange force and
//                torque (Sec. 2.4, Eq. force / Eq. torque) summed per
//                particle in exact fixed point; entry of each particle in
//                the pair-screening grid;
//   k_particles  pair screening through the cell grid, Newton-Euler update
//                with gravity, buoyancy and spring repulsion (Sec. 2.2,
//                Sec. 2.4) in FP64, and the raster of the new positions into
//                the next node bits (cleared over the old zones by k_links),
//                with the list of the nodes the particles left;
// plus the initialisation kernels (k_raster, k_geom_init), the
// direct-addressing comparison (k_direct_prep, k_links_direct), the near-tile
// bitmap of the opt-in split stream-collide (k_near_mask) and the batched
// forms of the step kernels.
#include <climits>
#include <type_traits>

#include "lbm_internal.cuh"

namespace lbm {

namespace {

constexpr int kBoxThreads = 128;
constexpr double kPi = 3.14159265358979323846;

__device__ __forceinline__ bool inside(const Dev &D, int i, int j)
{
    return i >= 0 && i < D.nx && j >= 0 && j < D.ny;
}

} // namespace

// The link kernel's window for zones of side N: the zone plus the two-node
// margin of the bounce-back stencil, wy = N + 4 rows of wx = N + 4 columns
// from (X0 - 2, Y0 - 2); wx is at most 64 (the fluid and owner masks of a row
// are 64-bit words).
__host__ __device__ inline int link_tile_wy(int N) { return N + 4; }
__host__ __device__ inline int link_tile_wx(int N) { return N + 4; }

// Shared memory of a CTA: its record, the fluid and owner row masks [wy] (u64
// each) and the list of links (at most one per slot).
struct alignas(16) LinkTeam {
    EllLink ell;   // an ellipse's FP64 frame
    int n;         // links found
    unsigned over; // a line with two links
};
constexpr int kLinkZoneMax = 60; // zone side: window rows of at most 64 columns
constexpr size_t link_smem(int N)
{
    const size_t b = sizeof(LinkTeam) + (size_t)2 * (N + 4) * sizeof(unsigned long long) +
                     (size_t)(12 * N - 12) * sizeof(int);
    return (b + 15) / 16 * 16;
}
// A kernel's dynamic shared memory is limited per function and process, not per
// handle, so the link kernels leave that limit alone (a handle that lowered it
// to its own zones would have later launches of one with larger zones refused):
// beside the kernels' static arrays (below 2 KB) every zone fits the default.
static_assert(link_smem(kLinkZoneMax) <= 46 * 1024, "the link kernels' shared memory exceeds the default limit");
size_t link_smem_bytes(int N) { return link_smem(N); }

bool link_zone_supported(int N) { return N <= kLinkZoneMax; }
static_assert(kLinkZoneMax + 4 <= 64, "the masks of a window row are 64-bit words");

// Counts (and overflow flag) of the screening grid of the next step, which
// the next step's link kernel fills: block p of the np blocks of a
// per-particle kernel clears its share.  The grid was last read by the
// previous step's update.
__device__ __forceinline__ void clear_cells_slice(const Dev &D, int parity, int p, int tid, int nthreads)
{
    int *grid = D.cells[parity ^ 1];
    const int nc = D.cell_gx * D.cell_gy + 1, per = (nc + D.np - 1) / D.np;
    const int c1 = min(nc, (p + 1) * per);
    for (int c = p * per + tid; c < c1; c += nthreads)
        if (in_bounds(D, c, (long long)nc * (1 + kCellCap))) grid[c] = 0;
}

// Entry of particle b at (xh, yh) in a screening grid (cleared beforehand);
// a full cell flags the grid, whose next screening then scans all pairs.
__device__ __forceinline__ void cell_insert(const Dev &D, int *grid, int b, float xh, float yh)
{
    const int ncell = D.cell_gx * D.cell_gy, c = cell_of(D, xh, yh);
    const long long size = (long long)(ncell + 1) + (long long)ncell * kCellCap;
    if (!in_bounds(D, c, ncell)) return;
    const int k = atomicAdd(grid + c, 1);
    if (k < kCellCap) {
        if (in_bounds(D, ncell + 1 + (long long)c * kCellCap + k, size)) grid[ncell + 1 + c * kCellCap + k] = b;
    } else grid[ncell] = 1;
}

// Zone of particle p one step back: its node bits, and for a crowded particle
// its owner nodes, cleared in the maps the raster fills next (they hold the
// positions of that time; every zone is cleared, so the words a zone shares
// with another's need no care).  One warp per call, lanes on zone rows.
__device__ __forceinline__ void clear_zone_bits(const Dev &D, int parity, int p, int lane)
{
    const GeomRec *G = D.geo[parity ^ 1] + p;
    const int X0 = G->X0, Y0 = G->Y0, N = G->N;
    const int w0 = max(X0, 0) >> 5, w1 = min(X0 + N - 1, D.nx - 1) >> 5;
    for (int r = lane; r < N; r += 32) {
        const int j = Y0 + r;
        if (j < 0 || j >= D.ny) continue;
        const BitsRow row = bits_row(D, j, parity ^ 1);
        for (int w = w0; w <= w1; ++w) bits_put(D, row, w, 0u);
    }
}
// (Whole block of nthreads threads.)
__device__ __forceinline__ void clear_zone_owner(const Dev &D, int *__restrict__ own_nxt, int parity, int p, int tid,
                                                 int nthreads)
{
    if (!D.crowd[parity ^ 1][p]) return;
    const GeomRec *G = D.geo[parity ^ 1] + p;
    const int X0 = G->X0, Y0 = G->Y0, N = G->N;
    for (int r = tid >> 5; r < N; r += nthreads / 32) {
        const int j = Y0 + r;
        if (j < 0 || j >= D.ny) continue;
        for (int c = tid & 31; c < N; c += 32) {
            const int i = X0 + c;
            if (i >= 0 && i < D.nx && in_bounds(D, (long long)j * D.nx + i, (long long)D.nx * D.ny))
                own_nxt[(long long)j * D.nx + i] = -1;
        }
    }
}

// Run of zone row r of particle p (empty: lo > hi) at a parity.
__device__ __forceinline__ int2 run_at(const Dev &D, int parity, int p, int r)
{
    const long long i = (long long)p * D.zone_max + r;
    return in_bounds(D, i, (long long)D.np * D.zone_max) ? D.runs[parity][i] : make_int2(1, 0);
}

// Row masks of the link kernel's window, 64 columns from XA: the fluid nodes
// of row j (none outside the domain), from the node bits; wide: more than 32
// columns matter.
__device__ __forceinline__ unsigned long long fluid_row(const Dev &D, int parity, int XA, int j, bool wide)
{
    if (j < 0 || j >= D.ny) return 0ull;
    const BitsRow row = bits_row(D, j, parity);
    const int w0 = XA >> 5, sh = XA & 31; // XA may be negative: words before the row are not fluid
    auto word = [&](int w) -> unsigned { return w >= 0 && w < D.bpitch ? ~bits_get(D, row, w) : 0u; };
    const unsigned a = word(w0), b = word(w0 + 1), c = wide ? word(w0 + 2) : 0u;
    unsigned long long m = ((unsigned long long)__funnelshift_r(b, c, sh) << 32) | __funnelshift_r(a, b, sh);
    const int in = D.nx - XA; // columns inside the domain
    if (in < 64) m &= in > 0 ? (1ull << in) - 1ull : 0ull;
    return m;
}

// 32 bits of m from bit s on (zeros outside its 64 bits).
__device__ __forceinline__ unsigned extract32(unsigned long long m, int s)
{
    if (s >= 0) return s < 64 ? (unsigned)(m >> s) : 0u;
    return s > -32 ? (unsigned)m << -s : 0u;
}

// Transpose of the warp's 32 x 32 bits: lane l holds row l before, column l
// after (bit r of it from row r).
__device__ __forceinline__ unsigned transpose32(unsigned x, int lane)
{
    unsigned keep = 0x0000ffffu; // the bits of a lane without bit s that stay
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        const unsigned y = __shfl_xor_sync(0xffffffffu, x, s);
        x = (lane & s) ? (x & ~keep) | ((y >> s) & keep) : (x & keep) | ((y << s) & ~keep);
        keep ^= keep << (s >> 1);
    }
    return x;
}

// One CTA of kTeam warps per particle.  Phases:
//  0. clear this CTA's share of the screening grid the next step's link
//     kernel fills, and the particle's zone one step back in the node bits
//     (and owner map) that the raster fills next;
//  1. row masks of the particle's window (zone plus the two-node margin of
//     the bounce-back stencil), a lane per row: fluid nodes from the node
//     bits, this particle's nodes from the row runs of its raster (a crowded
//     particle's from the owner map, since it may share nodes with another);
//     thread 0 publishes the particle's screening record (and the FP64 frame
//     of an ellipse); a warp prefetches into L2 the bit rows of the particle
//     `ahead` places later in launch order (one residency wave ahead).
//     (Prefetching the populations of that particle's window as well, by
//     tensor or row prefetches, or of this particle's links as they are
//     found, measured slower);
//  2. links.  Along any line of the zone (Sec. 3: the rows, the columns and
//     the two families of diagonals) the particle's nodes are one run, and
//     the only nodes that can be linked to it there are the two next to the
//     run's ends, one per direction: a warp per family (teams of one or two
//     warps take the families in turn) brings the row masks to a lane per
//     line (shears and 32 x 32 bit transposes), takes the run's ends, looks
//     the two nodes up in the fluid masks and appends the links to a list; a
//     line without a link empties its slot of the index array;
//  3. each link: its slot of the index array, wall fraction q, curved
//     bounce-back of f and g (Sec. 2.3) from the populations read at x_f,
//     x_f - e_k and x_f - 2 e_k, written into the solid node x_f + e_k
//     (direction kbar) of A in HBM, where the next pull stream picks it up
//     (one link per (solid node, kbar), and every read is of a fluid node, so
//     the writes never race the reads), and the momentum-exchange bracket of
//     Eq. force / Eq. torque, summed in exact fixed point per thread, per
//     warp and over the warps (so the forces are bit-reproducible, whatever
//     the list's order);
//  4. the particle enters the screening grid of this step's update.
template <typename T, int kTeam>
__device__ __forceinline__ void links_body(const Dev &D, T *A, const int *__restrict__ own,
                                           int *__restrict__ own_nxt, int parity, const int p, const int pa)
{
    extern __shared__ __align__(16) unsigned char sm[];
    using E = Elem<T>;
    constexpr unsigned F = 0xffffffffu;
    constexpr int kThreads = 32 * kTeam;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const GeomRec *Gp = D.geo[parity] + p;
    const int X0 = Gp->X0, Y0 = Gp->Y0, N = Gp->N;
    const int base = D.slot_base[p];
    const int crowded = D.crowd[parity][p];

    const int wy = link_tile_wy(N), wx = link_tile_wx(N);
    const int XA = X0 - 2, YA = Y0 - 2;
    LinkTeam &S = *reinterpret_cast<LinkTeam *>(sm);
    unsigned long long *Fm = reinterpret_cast<unsigned long long *>(sm + sizeof(LinkTeam)); // [wy]
    unsigned long long *Om = Fm + link_tile_wy(D.zone_max);                                  // [wy]
    int *list = reinterpret_cast<int *>(Om + link_tile_wy(D.zone_max)); // k | a << 4 | b << 10 | slot << 16

    // ---- 0., 1.
    clear_cells_slice(D, parity, p, tid, kThreads);
    if (p == 0 && tid == 0) D.status->nb = 0u; // the step's list of nodes left
    if (tid == 0) {
        S.n = 0;
        S.over = 0u;
    }
    if (warp == 0)
        for (int r = lane; r < wy; r += 32) Fm[r] = fluid_row(D, parity, XA, YA + r, wx > 32);
    if (!crowded) {
        if (warp == 1 % kTeam)
            for (int r = lane; r < wy; r += 32) {
                unsigned long long m = 0ull;
                if (r >= 2 && r < N + 2) {
                    const int2 run = run_at(D, parity, p, r - 2);
                    if (run.x <= run.y) m = ((2ull << (run.y - XA)) - 1ull) & (~0ull << (run.x - XA));
                }
                Om[r] = m;
            }
    } else {
        // four zone rows' loads of a warp in flight before the first ballot
        constexpr int kU = kTeam < 4 ? 4 : 8;
        for (int b0 = warp; b0 < N; b0 += kU * kTeam) {
            int lo[kU], hi[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int b = b0 + u * kTeam, j = Y0 + b, i = X0 + lane;
                if (b >= N) break;
                const int *row = own + (long long)j * D.nx;
                lo[u] = inside(D, i, j) ? row[i] : -1;
                hi[u] = N > 32 && inside(D, i + 32, j) ? row[i + 32] : -1;
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int b = b0 + u * kTeam;
                if (b >= N) break;
                const unsigned ol = __ballot_sync(F, lo[u] == p), oh = N > 32 ? __ballot_sync(F, hi[u] == p) : 0u;
                if (lane == 0) Om[b + 2] = (((unsigned long long)oh << 32) | ol) << 2;
            }
        }
    }
    if (warp == 2 % kTeam) clear_zone_bits(D, parity, p, lane);
    clear_zone_owner(D, own_nxt, parity, p, tid, kThreads);
    if (tid == kThreads - 1) {
        D.pos4[p] = make_float4(Gp->xh, Gp->yh, Gp->xl, Gp->yl);
        D.prc[p] = make_float2(Gp->r, Gp->C);
    }
    if (warp == kTeam - 1 && lane < 8 && Gp->r < 0.f) {
        const PartSoA &P = D.part[parity];
        ell_link_entry(S.ell, lane, ell_frame_cs(P.x[p], P.y[p], D.cs[parity][p], P.r[p], P.b[p]));
    }
    // L2 prefetch of the bit rows of particle pa, the one a residency wave
    // later in launch order (none: pa < 0)
    if (warp == 3 % kTeam && pa >= 0) {
        const GeomRec *Ga = D.geo[parity] + pa;
        const int xa = Ga->X0 - 2, ya = Ga->Y0 - 2;
        for (int r = lane; r < link_tile_wy(D.zone_max); r += 32) {
            const int j = ya + r;
            if (j >= 0 && j < D.ny && xa < D.nx)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(bits_src(D, bit_word(D, max(xa, 0), j, 0), 1)) : "memory");
        }
    }
    __syncthreads();

    // ---- 2. links: the rows, the columns, the diagonals of constant a - b,
    // those of constant a + b; lane l of a round takes line i
    constexpr int kFam = kTeam < 4 ? kTeam : 4; // families taken side by side
    for (int f = warp % kFam; f < 4; f += kFam) {
        const int M = 2 * N - 3, lines = f < 2 ? N : M;
        const int kf = f < 2 ? f + 1 : f + 3;                   // direction into the run's start: 1, 2, 5, 6
        const int sf = f == 0 ? 0 : f == 1 ? N : f == 2 ? 4 * N : 4 * N + M; // its slots; those of the end follow
        const int sb = sf + (f < 2 ? 2 * N : 2 * M);
        for (int i0 = 32 * (warp / kFam); i0 < lines; i0 += 32 * (kTeam / kFam)) {
            const int i = i0 + lane;
            // the particle's nodes on line i: bit t, the row b of the node
            // (its column a on a row)
            unsigned long long m = 0ull;
            if (f == 0) {
                if (i < N) m = Om[i + 2] >> 2;
            } else {
                for (int h = 0; h < N; h += 32) {
                    const int b = h + lane;
                    const unsigned long long R = b < N ? Om[b + 2] >> 2 : 0ull;
                    const unsigned x = extract32(R, f == 1 ? i0 : f == 2 ? i0 + b - (N - 2) : i0 + 1 - b);
                    m |= (unsigned long long)transpose32(x, lane) << h;
                }
            }
            // zone column a of line i at t (the row of f > 0)
            auto col = [&](int t) { return f == 0 ? t : f == 1 ? i : f == 2 ? t + i - (N - 2) : i + 1 - t; };
            auto fluid = [&](int t) -> bool {
                const int a = col(t), b = f == 0 ? i : t;
                return a >= 0 && a < N && b >= 0 && b < N && ((Fm[b + 2] >> (a + 2)) & 1ull);
            };
            bool lo = false, hi = false;
            int t0 = 0, t1 = 0;
            if (i < lines && m) {
                t0 = __ffsll((long long)m) - 2;  // before the run's start
                t1 = 64 - __clzll((long long)m); // after its end
                lo = fluid(t0);
                hi = fluid(t1);
                // two runs: a particle of higher index owns the nodes between
                // (none of them is fluid), or the owner map is a restored
                // image's; a link inside would be the line's second
                unsigned long long st = m & ~(m << 1), en = m & ~(m >> 1);
                st &= st - 1ull;
                en &= ~(1ull << (t1 - 1));
                while (st) {
                    if (fluid(__ffsll((long long)st) - 2) || fluid(__ffsll((long long)en))) S.over = 1u;
                    st &= st - 1ull;
                    en &= en - 1ull;
                }
            }
            const unsigned wl = __ballot_sync(F, lo), wh = __ballot_sync(F, hi);
            int at = 0;
            if (lane == 0) at = atomicAdd(&S.n, __popc(wl) + __popc(wh));
            at = __shfl_sync(F, at, 0);
            const unsigned below = (1u << lane) - 1u;
            if (i < lines) {
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const bool on = e ? hi : lo;
                    const int t = e ? t1 : t0, sl = (e ? sb : sf) + i, k = kf + 2 * e;
                    if (on) {
                        const int pos = at + (e ? __popc(wl) + __popc(wh & below) : __popc(wl & below));
                        list[pos] = k | (col(t) << 4) | ((f == 0 ? i : t) << 10) | (sl << 16);
                    } else if (in_bounds(D, (long long)base + sl, D.nslots)) {
                        D.slot_node[base + sl] = -1;
                        D.slot_q[base + sl] = 0.f;
                    }
                }
            }
        }
    }
    __syncthreads();
    const int nvalid = S.n;

    // ---- 3. bounce-back and momentum exchange, thread i on the links i,
    // i + kThreads, ...
    const GeomRec G = *Gp;
    const DiskDF dk = geom_df(G);
    const bool ell = G.r < 0.f; // an ellipse: q in FP64
    auto fluid = [&](int i, int j) -> bool { return (Fm[j - YA] >> (i - XA)) & 1ull; };
    long long vx = 0, vy = 0, vt = 0;
    // the constant part's directions, x + 65536 y (axis, diagonal), and its
    // torque moments; counts of the fallbacks, a field of 10 bits each (a
    // particle has at most 12 x 60 - 12 links)
    int axd = 0, dgd = 0, axt = 0, dgt = 0;
    unsigned falls = 0u;
    for (int li = tid; li < nvalid; li += kThreads) {
        const int inf = list[li], k = inf & 15, sl = inf >> 16;
        const int kx = ex(k), ky = ey(k), kb = opp(k);
        const int fi = X0 + ((inf >> 4) & 63), fj = Y0 + ((inf >> 10) & 63);
        const bool have1 = fluid(fi - kx, fj - ky);
        const bool have2 = fluid(fi - 2 * kx, fj - 2 * ky);
        // populations of fluid nodes: no team writes them during this kernel
        const long long n0 = (long long)fj * D.pitch + fi, dn = (long long)ky * D.pitch + kx;
        const long long n1 = have1 ? n0 - dn : n0, n2 = have2 ? n0 - 2 * dn : n0;
        auto tv = [&](long long e) -> float { return in_bounds(D, e, D.a_elems) ? E::ld(__ldg(A + e)) : 0.f; };
        const long long pk = k * D.ps, pb = kb * D.ps;
        const float fk0 = tv(pk + n0), fk1 = tv(pk + n1), fk2 = tv(pk + n2);
        const float fb0 = tv(pb + n0), fb1 = tv(pb + n1);
        const long long gk = pk + kQ9 * D.ps, gb = pb + kQ9 * D.ps;
        float gk0 = 0.f, gk1 = 0.f, gb0 = 0.f;
        if (k <= 4) {
            gk0 = tv(gk + n0);
            gk1 = tv(gk + n1);
            gb0 = tv(gb + n0);
        }
        float dxf, dyf;
        const float q = ell ? link_q_ellipse(fi, fj, k, S.ell, dxf, dyf) : link_q_df(fi, fj, k, dk, dxf, dyf);
        if (in_bounds(D, (long long)base + sl, D.nslots)) {
            D.slot_node[base + sl] = fj * D.nx + fi;
            D.slot_q[base + sl] = q;
        }
        // curved bounce-back in deviation form: every rule is an affine
        // combination of populations of equal weight, so it holds for
        // f~ = f - w unchanged
        const float rx = dxf + q * kx, ry = dyf + q * ky;
        const float uwx = G.ux - G.om * ry, uwy = G.uy + G.om * rx;
        const float wall = 6.f * w9(k) * -(kx * uwx + ky * uwy); // 2 w rho0 e_kbar.u_w / c_s^2
        int lvl;
        const float fnew = bouzidi32(q, fk0, fk1, fk2, fb0, fb1, have1, have2, wall, lvl);
        const long long ns = n0 + dn;
        if (in_bounds(D, pb + ns, D.a_elems)) A[pb + ns] = E::st(fnew);
        if (k <= 4 && in_bounds(D, gb + ns, D.a_elems))
            A[gb + ns] = E::st(thermal32(q, gk0, gk1, gb0, have1, G.wT));
        // momentum exchange: with f = w + f~ the bracket of Eq. force is
        // 2 w_k e_k + [f~_k^+ (e_k - u_w) - f~_kbar (e_kbar - u_w)]; the
        // constant part and its torque 2 w_k ((i - x_c) e_k,y - (j - y_c) e_k,x)
        // (q drops out) are kept as exact integer sums, assembled in FP64 by
        // the particle update
        const float bx = fk0 * (kx - uwx) - fnew * (-kx - uwx);
        const float by = fk0 * (ky - uwy) - fnew * (-ky - uwy);
        vx += fix_force(bx);
        vy += fix_force(by);
        vt += fix_torque(rx * by - ry * bx);
        const int tz = fi * ky - fj * kx, d = kx + 65536 * ky;
        falls += (lvl == 1 ? 1u : lvl == 2 ? 1u << 10 : 0u) + (k <= 4 && !have1 ? 1u << 20 : 0u);
        if (k <= 4) {
            axd += d;
            axt += tz;
        } else {
            dgd += d;
            dgt += tz;
        }
    }
    LinkSums R;
    R.fx = warp_sum64(vx);
    R.fy = warp_sum64(vy);
    R.tz = warp_sum64(vt);
    axd = __reduce_add_sync(F, axd);
    dgd = __reduce_add_sync(F, dgd);
    R.ax_t = __reduce_add_sync(F, axt);
    R.dg_t = __reduce_add_sync(F, dgt);
    falls = __reduce_add_sync(F, falls);
    R.ax_x = (short)(axd & 0xffff);
    R.ax_y = (axd - R.ax_x) >> 16;
    R.dg_x = (short)(dgd & 0xffff);
    R.dg_y = (dgd - R.dg_x) >> 16;
    R.pad[0] = R.pad[1] = R.pad[2] = R.pad[3] = 0;
    int c3[3] = {(int)(falls & 1023u), (int)((falls >> 10) & 1023u), (int)(falls >> 20)};
    // the particle's sums over the warps (exact integer sums, so the grouping
    // does not matter)
    __shared__ LinkSums s_ws[kTeam];
    __shared__ int s_wc[kTeam][3];
    if (lane == 0) {
        s_ws[warp] = R;
        s_wc[warp][0] = c3[0]; s_wc[warp][1] = c3[1]; s_wc[warp][2] = c3[2];
    }
    __syncthreads();
    if (tid == 0) {
#pragma unroll
        for (int w = 1; w < kTeam; ++w) {
            add_sums(R, s_ws[w]);
            c3[0] += s_wc[w][0]; c3[1] += s_wc[w][1]; c3[2] += s_wc[w][2];
        }
        D.lsum[p] = R;
        unsigned long long *C = D.status->cnt[parity];
        if (c3[0]) atomicAdd(&C[kCntBzLinear], (unsigned long long)c3[0]);
        if (c3[1]) atomicAdd(&C[kCntBzSimple], (unsigned long long)c3[1]);
        if (c3[2]) atomicAdd(&C[kCntThermHalf], (unsigned long long)c3[2]);
        if (nvalid) atomicAdd(&C[kCntLinks], (unsigned long long)nvalid);
        if (S.over) atomicOr(&D.status->err, kErrOverflow);
    }
    // ---- 4. the particle's position into the screening grid this step's
    // update reads (its counts cleared by the previous step's link kernel):
    // the atomic's round trip ends the CTA instead of lengthening the update
    if (tid == kThreads - 1) cell_insert(D, D.cells[parity], p, G.xh, G.yh);
}

// Spring repulsion magnitude of Sec. 2.4 for a gap (distance to the wall
// plane, or centre distance minus both radii): zero beyond the threshold s,
// else (C/eps) ((gap - s)/s)^2 along the gap vector.
__device__ __forceinline__ double repulsion(double gap, double s, double eps, double C)
{
    if (gap > s) return 0.0;
    const double t = (gap - s) / s;
    return C / eps * t * t;
}

// Total force = hydrodynamic (assembled from the link sums) + buoyant weight
// -(rho_p - rho_f) pi r^2 g y-hat + repulsion (walls, and every other disk
// with C_ab the mean of the two force scales C = pi r^2 (rho_p - rho_f) g).
// Each block takes kPB particles: warp w screens particle w against the
// particles listed in the 3 x 3 cells of the screening grid around its cell
// (filled with the step's starting positions by the link kernel; every
// pair in reach is among them), or, when a cell of that grid overflowed,
// against all particles in shared-memory tiles of kPartTile, and evaluates the
// pairs in reach from double-float centre differences, summed in 64-bit
// fixed point so that the result is the same whichever way the pairs were
// found and in whatever order; lane l of warp 0 then sums, integrates and
// stores particle l in FP64 (its constants 1/M, 1/I, W and C, and its
// geometry record, staged by the last warp while the others screen), and
// warp w rasters particle w.  Integration:
// U' = U + F/M, X' = X + (U + U')/2, Omega' = Omega + T/I,
// theta' = theta + (Omega + Omega')/2 with M = rho_p pi r^2 and I = M r^2 / 2
// (M = rho_p pi r b and I = M (r^2 + b^2) / 4 for an ellipse).
//
// Bound by the latency of the chain (screening, FP64 tail, raster) and by the
// SM's FP64 pipe (2 lanes a clock), so kPB is the smallest of 1, 2, 4, 8 that
// gives each SM one block: few particles spread over all SMs, many share a
// tail (one warp's FP64 instructions serve kPB particles).  No thread divides
// in FP64 for a constant, cos and sin of an orientation are kept with the
// state, an ellipse's supports are worked out at walls only, and the tail's
// inputs are copied asynchronously.  Update, us (CUDA events), before / after:
// 129 ellipses 37.1 / 19.7, 6 ellipses 22.9 / 14.7, 8 disks 13.0 / 12.5, 4800
// disks 19.2 / 15.8 (with kPB = 4 there 16.9, 16: 22, 32: 29).
constexpr int kPartTile = 512;
constexpr int kPartMax = 8;
constexpr int part_ctas(int pb) { return 32 / pb > 16 ? 16 : 32 / pb; } // 64 registers a thread (pb = 1: 128)

// Support distance of particle p along the unit vector (nx, ny): its radius
// for a disk.
__device__ __forceinline__ double support_of(const Dev &D, int parity, int p, double nx, double ny)
{
    const double r = D.part[parity].r[p], b = D.part[parity].b[p];
    if (!is_ellipse(r, b)) return r;
    return ell_support(ell_frame_cs(0.0, 0.0, D.cs[parity][p], r, b), nx, ny);
}

// Pair repulsion on particle a from particle b when either is an ellipse, in
// FP64: the gap along the line of centres is the centre distance minus both
// support distances along it.
__device__ __noinline__ void pair_force_ellipse(const Dev &D, int parity, int a, int b, long long &sx, long long &sy)
{
    const PartSoA &P = D.part[parity];
    const double dx = P.x[a] - P.x[b], dy = P.y[a] - P.y[b];
    const double dist = sqrt(dx * dx + dy * dy);
    const double gap = dist - support_of(D, parity, a, -dx / dist, -dy / dist) -
                       support_of(D, parity, b, dx / dist, dy / dist);
    if (gap > D.s_rep) return;
    auto scale = [&](int p) {
        const double r = P.r[p], pb = P.b[p];
        return kPi * r * (is_ellipse(r, pb) ? pb : r) * (P.rho[p] - D.rho_f) * D.g;
    };
    const double mag = repulsion(gap, D.s_rep, D.eps_w, 0.5 * (scale(a) + scale(b)));
    sx += fix_of(mag * dx / dist);
    sy += fix_of(mag * dy / dist);
}

// Pair repulsion on disk a from disk b (FP32 from double-float centres).
__device__ __noinline__ void pair_force(float4 pa, float2 ca, float4 pb, float2 cb, float s_rep,
                                        float inv_eps, long long &sx, long long &sy)
{
    float hx, ex_, hy, ey_;
    two_sum(pa.x, -pb.x, hx, ex_);
    two_sum(pa.y, -pb.y, hy, ey_);
    const float dx = hx + (ex_ + (pa.z - pb.z));
    const float dy = hy + (ey_ + (pa.w - pb.w));
    const float dist = sqrtf(dx * dx + dy * dy);
    const float gap = dist - ca.x - cb.x;
    if (gap > s_rep) return;
    const float t = (gap - s_rep) / s_rep;
    const float mag = 0.5f * (ca.y + cb.y) * inv_eps * t * t;
    sx += fix_of(mag * dx / dist);
    sy += fix_of(mag * dy / dist);
}

// Screening of particle a (position pa, (r, C) ca) against candidate b:
// circumscribed circles within reach (r < 0 marks an ellipse), then the
// pair force.  crowd: set when the two may share nodes after their moves,
// each less than one node along either axis: centres within 2 sqrt(2) of the
// sum of the radii, taken as 3 plus the FP32 rounding of the centres.
__device__ __forceinline__ void screen_pair(const Dev &D, int parity, int a, float4 pa, float2 ca, int b, float4 pb,
                                            float2 cb, float s_rep, float inv_eps, long long &sx, long long &sy,
                                            bool &crowd)
{
    const float dxf = pa.x - pb.x, dyf = pa.y - pb.y, rr = fabsf(ca.x) + fabsf(cb.x);
    const float lim = rr + s_rep + 1.f, touch = rr + 3.f + 2.4e-7f * (float)(D.nx + D.ny), d2 = dxf * dxf + dyf * dyf;
    if (b == a) return;
    crowd |= !(d2 > touch * touch);
    if (d2 > lim * lim) return;
    if (ca.x < 0.f || cb.x < 0.f) pair_force_ellipse(D, parity, a, b, sx, sy);
    else pair_force(pa, ca, pb, cb, s_rep, inv_eps, sx, sy);
}

// Zone of a disk at (x, y) with radius r: N x N nodes from
// (floor(x - r) - 1, floor(y - r) - 1); it holds every node of the disk and
// every fluid node linked to it.
struct Box {
    int X0, Y0, N;
};
__device__ __forceinline__ Box box_of(const GeomRec &G) { return Box{G.X0, G.Y0, G.N}; }

// Writes of a warp's raster: lane l holds the run [lo, hi] of zone row
// b0 + l (empty when lo > hi); the warp then stores row after row, lanes on
// consecutive nodes, so each row's atomicMax requests coalesce.
__device__ __forceinline__ void write_runs(const Dev &D, int *own, const Box &B, int b0, int lo, int hi, int p)
{
    const int lane = threadIdx.x & 31, nr = min(32, B.N - b0);
    for (int r = 0; r < nr; ++r) {
        const int l = __shfl_sync(0xffffffffu, lo, r), h = __shfl_sync(0xffffffffu, hi, r);
        const long long j0 = (long long)(B.Y0 + b0 + r) * D.nx;
        for (int i = l + lane; i <= h; i += 32)
            if (in_bounds(D, j0 + i, (long long)D.nx * D.ny)) atomicMax(own + j0 + i, p);
    }
}

// Run of row j of one ellipse.  Along a row the ellipse form is a convex
// quadratic in i, so the inside nodes form one run; when the run is not
// empty the node nearest the vertex of the parabola lies in it (checked with
// its two neighbours, against rounding of the vertex).  The run's ends are
// estimated from the quadratic's roots (FP32) and settled with the predicate
// at the ends only: FP32 outside the rounding band, the exact FP64 form
// inside it.
__device__ __noinline__ void ellipse_run(const Dev &D, const Box B, const GeomRec G, double x, double y, double2 cs,
                                         double r, double pb, int j, int &lo_out, int &hi_out)
{
    lo_out = 1;
    hi_out = 0;
    if (j < 0 || j >= D.ny) return;
    const int xmin = B.X0, xmax = B.X0 + B.N - 1;
    const EllDF F = ell_df(G.xh, G.xl, G.yh, G.yl, G.w0, G.w1, r, pb);
    auto inside = [&](int i) -> bool {
        const int side = ell_side_df(i, j, F);
        if (side) return side < 0;
        return in_ellipse(i, j, ell_frame_cs(x, y, cs, r, pb));
    };
    const float c = F.c, s = F.s;
    const float A2 = c * c * F.b2 + s * s * F.a2; // dx^2 coefficient
    const float Bc = c * s * (F.b2 - F.a2);       // half the dx dy coefficient
    const float Cc = s * s * F.b2 + c * c * F.a2; // dy^2 coefficient
    float dyh, dyl;
    df_offset(j, G.yh, G.yl, dyh, dyl);
    const float dy = dyh + dyl;
    const float B1 = Bc * dy, C0 = Cc * dy * dy - F.ab;
    const float mid = (G.xh - B1 / A2) + G.xl;
    const int im = (int)floorf(mid + 0.5f);
    const int in = inside(im) ? im : inside(im - 1) ? im - 1 : inside(im + 1) ? im + 1 : INT_MIN;
    if (in == INT_MIN) return; // then no node of the row is inside
    if (in < xmin || in > xmax) return; // (a centre beyond any lattice: see zone_lo)
    const float h = sqrtf(fmaxf(B1 * B1 - A2 * C0, 0.f)) / A2;
    int lo = max(min(in, (int)ceilf(mid - h)), xmin), hi = min(max(in, (int)floorf(mid + h)), xmax);
    while (lo > xmin && inside(lo - 1)) --lo;
    while (!inside(lo)) ++lo;
    while (hi < xmax && inside(hi + 1)) ++hi;
    while (!inside(hi)) --hi;
    lo_out = max(lo, 0);
    hi_out = min(hi, D.nx - 1);
}

// Run of row j of one disk: the node nearest the centre decides whether the
// row meets the disk; the ends come from an FP32 estimate settled with the
// exact predicate.
__device__ __forceinline__ void disk_run(const Dev &D, const Box &B, const GeomRec &G, double x, double y, double r,
                                         int j, int &lo_out, int &hi_out)
{
    lo_out = 1;
    hi_out = 0;
    if (j < 0 || j >= D.ny) return;
    const DiskDF dk = geom_df(G);
    const int ic = G.ic; // the node of each row nearest the centre
    const int xmin = B.X0, xmax = B.X0 + B.N - 1;
    if (ic < xmin || ic > xmax) return; // (a centre beyond any lattice: see zone_lo)
    if (!in_disk_df(ic, j, dk, x, y, r)) return; // then no node of the row is inside
    float dyh, dyl;
    df_offset(j, dk.yh, dk.yl, dyh, dyl);
    const float h = sqrtf(fmaxf(dk.r2h - dyh * dyh, 0.f));
    int lo = min(ic, (int)ceilf(dk.xh - h)), hi = max(ic, (int)floorf(dk.xh + h));
    lo = max(lo, xmin);
    hi = min(hi, xmax);
    while (lo > xmin && in_disk_df(lo - 1, j, dk, x, y, r)) --lo;
    while (!in_disk_df(lo, j, dk, x, y, r)) ++lo;
    while (hi < xmax && in_disk_df(hi + 1, j, dk, x, y, r)) ++hi;
    while (!in_disk_df(hi, j, dk, x, y, r)) --hi;
    lo_out = max(lo, 0);
    hi_out = min(hi, D.nx - 1);
}

// Nodes of run [lo, hi] of a row outside run [xlo, xhi] (one or two
// intervals; all of it when [xlo, xhi] is empty), in order.
template <typename F>
__device__ __forceinline__ void run_minus(int lo, int hi, int xlo, int xhi, F &&f)
{
    if (xlo > xhi) {
        for (int i = lo; i <= hi; ++i) f(i);
        return;
    }
    for (int i = lo; i <= min(hi, xlo - 1); ++i) f(i);
    for (int i = max(lo, xhi + 1); i <= hi; ++i) f(i);
}

// Raster of one particle by one warp, a lane per zone row: the row's run
// (lo, hi) of inside nodes, empty when lo > hi, kept by parity; its node bits
// (bits; at most three words a row, by atomic or); for a crowded particle
// its nodes in the owner map (own not null).  moved: its runs one step back
// are those of the other parity, from zone row Y0_old (a particle moves less
// than a node, so its old nodes lie in the rows of its new zone): the nodes
// it left are listed for the refilling.
__device__ __forceinline__ void raster_one(const Dev &D, int par, int *own, const GeomRec &G, double x, double y,
                                           double r, double2 cs, double pb, int p, bool bits, bool moved,
                                           int Y0_old)
{
    const int lane = threadIdx.x & 31;
    const Box B = box_of(G);
    int2 *runs = D.runs[par] + (long long)p * D.zone_max;
    for (int b0 = 0; b0 < B.N; b0 += 32) {
        const int j = B.Y0 + b0 + lane;
        int lo = 1, hi = 0;
        if (b0 + lane < B.N) {
            if (G.r < 0.f) ellipse_run(D, B, G, x, y, cs, r, pb, j, lo, hi);
            else disk_run(D, B, G, x, y, r, j, lo, hi);
            if (in_bounds(D, (long long)p * D.zone_max + b0 + lane, (long long)D.np * D.zone_max))
                runs[b0 + lane] = make_int2(lo, hi);
            if (bits && lo <= hi) {
                const BitsRow row = bits_row(D, j, par);
                for (int w = lo >> 5; w <= hi >> 5; ++w) {
                    const int c0 = max(lo - 32 * w, 0), c1 = min(hi - 32 * w, 31);
                    bits_or(D, row, w, (~0u << c0) & (~0u >> (31 - c1)));
                }
            }
            if (moved && j >= Y0_old && j < Y0_old + B.N && j >= 0 && j < D.ny) {
                const int2 o = run_at(D, par ^ 1, p, j - Y0_old);
                run_minus(o.x, o.y, lo, hi, [&](int i) {
                    const unsigned at = atomicAdd(&D.status->nb, 1u);
                    if (at < (unsigned)D.left_cap) D.left[at] = make_int2(j * D.nx + i, p);
                    else atomicOr(&D.status->err, kErrOverflow);
                });
            }
        }
        if (own) write_runs(D, own, B, b0, lo, hi, p);
    }
}

// Support distances of an ellipse along the wall normals x-hat and y-hat
// (kept out of line: the disk path does not carry its registers).
__device__ __noinline__ void wall_supports(double2 cs, double r, double b, double &hx, double &hy)
{
    const EllFrame E = ell_frame_cs(0.0, 0.0, cs, r, b);
    hx = ell_support(E, 1.0, 0.0);
    hy = ell_support(E, 0.0, 1.0);
}

// Asynchronous copy of kBytes (8 or 16, both addresses aligned to it) into
// shared memory.
template <int kBytes>
__device__ __forceinline__ void copy_async(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
                 "n"(kBytes)
                 : "memory");
}

// New state of a particle as the raster needs it.
struct RasterIn {
    GeomRec G;
    double x, y, r, b;
    double2 cs; // cos and sin of theta (an ellipse)
};

// Constants of the update of a particle (they depend only on its shape and
// density): 1/M, 1/I, the buoyant weight W = (rho_p - rho_f) A g and the
// repulsion force scale C = A (rho_p - rho_f) g, with the area A = pi r^2
// (pi r b for an ellipse), M = rho_p A and I = M r^2 / 2 (M (r^2 + b^2) / 4
// for an ellipse).  The update multiplies by 1/M and 1/I, which differs
// from dividing by M and I by at most one rounding of the increment.
__device__ __forceinline__ double4 part_consts(double r, double b, double rho, double rho_f, double g)
{
    const bool ell = is_ellipse(r, b);
    const double rb = ell ? b : r;
    const double M = rho * kPi * r * rb, I = ell ? 0.25 * M * (r * r + b * b) : 0.5 * M * r * r;
    return make_double4(1.0 / M, 1.0 / I, (rho - rho_f) * kPi * r * rb * g, kPi * r * rb * (rho - rho_f) * g);
}

// FP64 tail of the particle update for particle b: total force, Newton-Euler
// step, domain checks, new state and geometry record.  (psx, psy: the pair
// repulsion in fixed point; out: the new state for the raster; st, ls, Gc, pk: the
// particle's state fields x, y, ux, uy, theta, omega, r, rho, T, b, its link
// sums, its current geometry record and its constants, staged in shared
// memory during the screening.)
__device__ __forceinline__ void particle_tail(const Dev &D, int b, int parity, long long psx, long long psy, RasterIn &out,
                                              const double *st, const LinkSums &ls, const GeomRec &Gc,
                                              const double4 &pk)
{
    double x = st[0], y = st[1], ux = st[2], uy = st[3];
    double th = st[4], om = st[5];
    const double r = st[6], pb = st[9];
    // an ellipse: wall gaps to its support distances along the wall normals
    const bool ell = is_ellipse(r, pb);
    double Fx, Fy, Tz;
    if (D.direct) {
        const DirectSums &ds = D.dsum[b];
        LinkSums S;
        S.fx = fix_force(ds.f[0]);
        S.fy = fix_force(ds.f[1]);
        S.tz = fix_torque(ds.f[2]);
        S.ax_x = ds.c[0]; S.ax_y = ds.c[1]; S.ax_t = ds.c[2];
        S.dg_x = ds.c[3]; S.dg_y = ds.c[4]; S.dg_t = ds.c[5];
        assemble_force(S, x, y, Fx, Fy, Tz);
    } else {
        assemble_force(ls, x, y, Fx, Fy, Tz);
    }
    D.force[3 * b + 0] = Fx;
    D.force[3 * b + 1] = Fy;
    D.force[3 * b + 2] = Tz;
    const double Cb = pk.w;
    Fy -= pk.z;
    double hx = r, hy = r;
    // A wall gap takes the FP64 repulsion only where the FP32 centre of the
    // current geometry record puts it within the threshold plus a margin
    // (mar) far above that centre's rounding error (half an FP32 spacing,
    // 2.4e-4 at 4096): elsewhere the repulsion is zero either way, and GB300
    // runs FP64 at a small fraction of its FP32 rate.
    const float mar = 1e-3f + 2.4e-7f * (float)(D.nx + D.ny), near = D.s_repf + mar;
    const float rf0 = (float)r, nxf = (float)D.nx, nyf = (float)D.ny;
    // an ellipse reaches at most r along a wall normal: its support distances
    // are worked out where that may be within the threshold
    if (ell && (fminf(Gc.xh, nxf - 1.f - Gc.xh) + 0.5f - rf0 <= near || fminf(Gc.yh, nyf - 1.f - Gc.yh) + 0.5f - rf0 <= near))
        wall_supports(D.cs[parity][b], r, pb, hx, hy);
    const float hxf = (float)hx, hyf = (float)hy;
    if (!D.per_x) {
        if ((Gc.xh + 0.5f) - hxf <= near) Fx += repulsion((x + 0.5) - hx, D.s_rep, D.eps_w, Cb);
        if ((nxf - 0.5f - Gc.xh) - hxf <= near) Fx -= repulsion(((double)D.nx - 0.5 - x) - hx, D.s_rep, D.eps_w, Cb);
    }
    if (!D.per_y) {
        if ((Gc.yh + 0.5f) - hyf <= near) Fy += repulsion((y + 0.5) - hy, D.s_rep, D.eps_w, Cb);
        if ((nyf - 0.5f - Gc.yh) - hyf <= near) Fy -= repulsion(((double)D.ny - 0.5 - y) - hy, D.s_rep, D.eps_w, Cb);
    }
    if (psx) Fx += fix_value(psx);
    if (psy) Fy += fix_value(psy);
    if (!D.fixed) {
        const double ux1 = ux + Fx * pk.x, uy1 = uy + Fy * pk.x, om1 = om + Tz * pk.y;
        x += 0.5 * (ux + ux1);
        y += 0.5 * (uy + uy1);
        th += 0.5 * (om + om1);
        ux = ux1;
        uy = uy1;
        om = om1;
    }
    // a disk that would leave the cavity, move a node or more in one step
    // (beyond the reach of the near-tile bitmap), or whose state is no longer
    // finite raises the (sticky) domain error and stays where it was, so that
    // its zone stays inside the arrays every later kernel indexes
    // (decided in FP32 with the margin mar where that is certain, else in
    // FP64; a non-finite state fails both)
    const double xo = st[0], yo = st[1];
    const float xf = (float)x, yf = (float)y, rf = (float)r;
    const bool surely_in = xf - rf >= mar - 0.5f && xf + rf <= nxf - 0.5f - mar && yf - rf >= mar - 0.5f &&
                           yf + rf <= nyf - 0.5f - mar && fabsf(xf - Gc.xh) < 1.f - mar &&
                           fabsf(yf - Gc.yh) < 1.f - mar;
    if (!surely_in && !(x - r >= -0.5 && x + r <= (double)D.nx - 0.5 && y - r >= -0.5 && y + r <= (double)D.ny - 0.5 &&
                        fabs(x - xo) < 1.0 && fabs(y - yo) < 1.0)) {
        atomicOr(&D.status->err, kErrDomain);
        x = xo;
        y = yo;
    }
    // (both parities hold r, rho, T and b)
    const PartSoA &nxt = D.part[parity ^ 1];
    nxt.x[b] = x; nxt.y[b] = y; nxt.ux[b] = ux; nxt.uy[b] = uy; nxt.th[b] = th; nxt.om[b] = om;
    double2 cs = make_double2(1.0, 0.0);
    if (ell) {
        cos_sin_rn(th, cs.x, cs.y);
        D.cs[parity ^ 1][b] = cs;
    }
    const GeomRec Gn = move_geom(Gc, x, y, r, ell, cs, ux, uy, om);
    D.geo[parity ^ 1][b] = Gn;
    out.G = Gn;
    out.x = x; out.y = y; out.r = r; out.cs = cs; out.b = pb;
}

template <int kPB>
__device__ __forceinline__ void particles_body(const Dev &D, int parity, int *own_nxt, const int blk)
{
    constexpr int kPartPerBlock = kPB, kPartThreads = 32 * kPB;
    __shared__ float4 sp[kPartTile];
    __shared__ float2 sc[kPartTile];
    __shared__ long long sred[2][kPartPerBlock];
    __shared__ RasterIn sras[kPartPerBlock]; // the tail's results, handed to the raster warps
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int a = blk * kPartPerBlock + warp;
    if (blk == 0 && threadIdx.x < kNumCounters) D.status->cnt[parity ^ 1][threadIdx.x] = 0ull;
    const bool me = a < D.np;
    bool crowd = D.direct; // direct addressing reads the owner map of every particle
    // the last warp stages the tail's inputs (the block's particle states and
    // link sums) while every warp screens, so that the FP64 tail starts
    // without a global round trip
    __shared__ double s_cur[kPartPerBlock][kPartFields];
    __shared__ __align__(16) LinkSums s_ls[kPartPerBlock];
    __shared__ __align__(16) GeomRec s_geo[kPartPerBlock];
    __shared__ __align__(32) double4 s_pk[kPartPerBlock];
    if (warp == kPartPerBlock - 1) {
        // asynchronous copies: the warp goes on to its screening at once
        const int b0 = blk * kPartPerBlock, nb = min(kPartPerBlock, D.np - b0);
        for (int t = lane; t < nb * kPartFields; t += 32) {
            const int q = t / kPartFields, f = t - q * kPartFields;
            copy_async<8>(&s_cur[q][f], D.part[parity].x + (long long)f * D.np + b0 + q);
        }
        static_assert(sizeof(GeomRec) == 64 && sizeof(LinkSums) == 64, "records of four 16-byte words");
        for (int t = lane; t < nb * 4; t += 32) {
            copy_async<16>(reinterpret_cast<char *>(s_geo) + 16 * t, reinterpret_cast<const char *>(D.geo[parity] + b0) + 16 * t);
            if (!D.direct)
                copy_async<16>(reinterpret_cast<char *>(s_ls) + 16 * t, reinterpret_cast<const char *>(D.lsum + b0) + 16 * t);
        }
        for (int t = lane; t < nb * 2; t += 32)
            copy_async<16>(reinterpret_cast<char *>(s_pk) + 16 * t, reinterpret_cast<const char *>(D.pconst + b0) + 16 * t);
    }
    float4 pa = make_float4(0.f, 0.f, 0.f, 0.f);
    float2 ca = make_float2(1.f, 0.f);
    if (me) {
        pa = D.pos4[a];
        ca = D.prc[a];
    }
    const float s_rep = D.s_repf, inv_eps = D.inv_eps;
    long long sx = 0, sy = 0; // pair repulsion, fixed point
    const int *grid = D.cells[parity];
    const int gx = D.cell_gx, gy = D.cell_gy, ncell = gx * gy;
    if (!grid[ncell] && !D.all_pairs) {
        // candidates from the 3 x 3 cells around a's cell: lane l < 9 holds
        // cell l's count; candidate t goes to lane t mod 32
        int cnt = 0, cell = 0;
        if (me && lane < 9) {
            const int c0 = cell_of(D, pa.x, pa.y);
            const int cx = c0 % gx + lane % 3 - 1, cy = c0 / gx + lane / 3 - 1;
            if (cx >= 0 && cx < gx && cy >= 0 && cy < gy) {
                cell = cy * gx + cx;
                cnt = min(__ldg(grid + cell), kCellCap);
            }
        }
        int inc = cnt;
#pragma unroll
        for (int o = 1; o < 16; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        const int total = __shfl_sync(0xffffffffu, inc, 8), excl = inc - cnt;
        for (int t0 = 0; t0 < total; t0 += 32) {
            const int t = t0 + lane;
            int b = -1;
#pragma unroll
            for (int l = 0; l < 9; ++l) {
                const int e = __shfl_sync(0xffffffffu, excl, l), n = __shfl_sync(0xffffffffu, cnt, l);
                const int c = __shfl_sync(0xffffffffu, cell, l);
                if (t >= e && t < e + n) b = __ldg(grid + ncell + 1 + c * kCellCap + (t - e));
            }
            if (b >= 0) screen_pair(D, parity, a, pa, ca, b, D.pos4[b], D.prc[b], s_rep, inv_eps, sx, sy, crowd);
        }
    } else {
        // a cell overflowed: every pair, in shared-memory tiles
        for (int t0 = 0; t0 < D.np; t0 += kPartTile) {
            const int nb = min(kPartTile, D.np - t0);
            __syncthreads();
#pragma unroll 8
            for (int k = threadIdx.x; k < nb; k += kPartThreads) {
                sp[k] = D.pos4[t0 + k];
                sc[k] = D.prc[t0 + k];
            }
            __syncthreads();
            if (!me) continue;
            for (int u = lane; u < nb; u += 32)
                screen_pair(D, parity, a, pa, ca, t0 + u, sp[u], sc[u], s_rep, inv_eps, sx, sy, crowd);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        sx += __shfl_down_sync(0xffffffffu, sx, o);
        sy += __shfl_down_sync(0xffffffffu, sy, o);
    }
    if (lane == 0) {
        sred[0][warp] = sx;
        sred[1][warp] = sy;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    const int b = blk * kPartPerBlock + lane;
    if (warp == 0 && lane < kPartPerBlock && b < D.np)
        particle_tail(D, b, parity, sred[0][lane], sred[1][lane], sras[lane], s_cur[lane], s_ls[lane],
                      s_geo[lane], s_pk[lane]);
    // then the raster at the new positions: warp w rasters the block's
    // particle w (its own new state only, so no other block is waited for)
    __syncthreads();
    if (a < D.np) {
        const RasterIn &R = sras[warp];
        crowd = __any_sync(0xffffffffu, crowd);
        if (lane == 0) D.crowd[parity ^ 1][a] = crowd;
        raster_one(D, parity ^ 1, crowd ? own_nxt : nullptr, R.G, R.x, R.y, R.r, R.cs, R.b, a, true, true,
                   s_geo[warp].Y0);
    }
}


// Owner map: node (i,j) belongs to disk p iff (i - x)^2 + (j - y)^2 <= r^2
// (exact FP64; for an ellipse u^2 b^2 + v^2 a^2 <= a^2 b^2 in its frame);
// where particles overlap the highest index wins (atomicMax, so
// the result does not depend on the launch order).  One warp per particle,
// one lane per zone row: the predicate holds on one contiguous run of each
// row (it is monotone in |i - x|), so the run is found from an FP32 estimate
// of its ends and settled with the exact predicate at the ends only; the
// runs are then written row by row with coalesced atomicMax requests.

__device__ __forceinline__ void raster_body(const Dev &D, int *own, bool bits, int par, const int blk)
{
    const int p = blk * (kBoxThreads / 32) + (threadIdx.x >> 5);
    if (p >= D.np) return;
    const PartSoA &P = D.part[par];
    if (own && (threadIdx.x & 31) == 0) D.crowd[par][p] = 1;
    raster_one(D, par, own, D.geo[par][p], P.x[p], P.y[p], P.r[p], D.cs[par][p], P.b[p], p, bits, false, 0);
}

// Near-tile bitmap: every warp tile (one row, 32 kScNodes nodes) that meets a
// particle's zone at the current position widened by kNearMargin nodes.  One
// thread per particle and zone row; the bitmap is cleared beforehand.
__global__ void __launch_bounds__(128) k_near_mask(const Dev D, int span, int parity)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    const int Nm = D.zone_max + 2 * kNearMargin;
    const int p = g / Nm, r = g - p * Nm;
    if (p >= D.np) return;
    const GeomRec G = D.geo[parity][p];
    const int j = G.Y0 - kNearMargin + r;
    if (r >= G.N + 2 * kNearMargin || j < 0 || j >= D.ny) return;
    const int x0 = max(G.X0 - kNearMargin, 0), x1 = min(G.X0 + G.N - 1 + kNearMargin, D.pitch - 1);
    for (int t = x0 / span; t <= x1 / span; ++t) {
        const int b = j * D.near_tpr + t;
        atomicOr(D.near + (b >> 5), 1u << (b & 31));
    }
}

// ---- direct addressing (comparison with the index array)
// Per particle: clear its zone one step back in the next node bits and owner
// map, publish its centre for the pair screening, zero its sums.
__global__ void __launch_bounds__(kBoxThreads) k_direct_prep(const Dev D, int *__restrict__ own_nxt, int parity)
{
    const int p = blockIdx.x;
    clear_cells_slice(D, parity, p, threadIdx.x, kBoxThreads);
    if (p == 0 && threadIdx.x == 0) D.status->nb = 0u;
    if (threadIdx.x < 32) clear_zone_bits(D, parity, p, threadIdx.x);
    clear_zone_owner(D, own_nxt, parity, p, threadIdx.x, kBoxThreads);
    if (threadIdx.x == 0) {
        const GeomRec G = D.geo[parity][p];
        const DiskDF d0 = geom_df(G);
        D.pos4[p] = make_float4(d0.xh, d0.yh, d0.xl, d0.yl);
        D.prc[p] = make_float2(G.r, G.C);
        cell_insert(D, D.cells[parity], p, G.xh, G.yh);
    }
    if (threadIdx.x < 3) D.dsum[p].f[threadIdx.x] = 0.0;
    if (threadIdx.x < 6) D.dsum[p].c[threadIdx.x] = 0;
}

// One thread per lattice node (the straightforward mapping the paper starts
// from, Sec. 3): a fluid node tests its eight neighbours in the owner map
// and, for each one owned by a particle, applies the same wall fraction,
// bounce-back and momentum-exchange bracket as the index-array kernel, adding
// the bracket to the particle's sums with FP64 atomics.  Only nodes next to
// a disk do work, so most threads of a block idle.
template <typename T>
__global__ void __launch_bounds__(128)
    k_links_direct(const Dev D, T *A, const int *__restrict__ own, int parity)
{
    using E = Elem<T>;
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
    unsigned cnt[4] = {0u, 0u, 0u, 0u}; // links, linear, simple, thermal half-way
    if (i < D.nx && own[(long long)j * D.nx + i] == -1) {
        auto fluid = [&](int a, int b) {
            return a >= 0 && a < D.nx && b >= 0 && b < D.ny && own[(long long)b * D.nx + a] == -1;
        };
        auto tv = [&](int t, int a, int b) -> float {
            return E::ld(A[(long long)t * D.ps + (long long)b * D.pitch + a]);
        };
#pragma unroll 1
        for (int k = 1; k < kQ9; ++k) {
            const int kx = ex(k), ky = ey(k), si = i + kx, sj = j + ky;
            if (si < 0 || si >= D.nx || sj < 0 || sj >= D.ny) continue;
            const int p = own[(long long)sj * D.nx + si];
            if (p < 0) continue;
            const GeomRec G = D.geo[parity][p];
            const PartSoA &P = D.part[parity];
            float dxf, dyf;
            const float q = G.r < 0.f ? link_q_ellipse(i, j, k, ell_frame(P.x[p], P.y[p], P.th[p], P.r[p], P.b[p]),
                                                       dxf, dyf)
                                      : link_q_df(i, j, k, geom_df(G), dxf, dyf);
            const int kb = opp(k);
            const int i1 = i - kx, j1 = j - ky, i2 = i - 2 * kx, j2 = j - 2 * ky;
            const bool have1 = fluid(i1, j1), have2 = fluid(i2, j2);
            const int ii1 = have1 ? i1 : i, jj1 = have1 ? j1 : j;
            const int ii2 = have2 ? i2 : i, jj2 = have2 ? j2 : j;
            const float fk0 = tv(k, i, j), fk1 = tv(k, ii1, jj1), fk2 = tv(k, ii2, jj2);
            const float fb0 = tv(kb, i, j), fb1 = tv(kb, ii1, jj1);
            const float rx = dxf + q * kx, ry = dyf + q * ky;
            const float uwx = G.ux - G.om * ry, uwy = G.uy + G.om * rx;
            const float wall = 6.f * w9(k) * -(kx * uwx + ky * uwy);
            int lvl;
            const float fnew = bouzidi32(q, fk0, fk1, fk2, fb0, fb1, have1, have2, wall, lvl);
            const long long ns = (long long)sj * D.pitch + si;
            if (in_bounds(D, kb * D.ps + ns, D.a_elems)) A[kb * D.ps + ns] = E::st(fnew);
            if (k <= 4) {
                const float gnew = thermal32(q, tv(kQ9 + k, i, j), tv(kQ9 + k, ii1, jj1), tv(kQ9 + kb, i, j), have1,
                                             G.wT);
                if (in_bounds(D, (kQ9 + kb) * D.ps + ns, D.a_elems)) A[(kQ9 + kb) * D.ps + ns] = E::st(gnew);
                cnt[3] += !have1;
            }
            const float bx = fk0 * (kx - uwx) - fnew * (-kx - uwx);
            const float by = fk0 * (ky - uwy) - fnew * (-ky - uwy);
            DirectSums &ds = D.dsum[p];
            atomicAdd(&ds.f[0], (double)bx);
            atomicAdd(&ds.f[1], (double)by);
            atomicAdd(&ds.f[2], (double)(rx * by - ry * bx));
            const int tz = i * ky - j * kx, o = k <= 4 ? 0 : 3;
            if (kx) atomicAdd(&ds.c[o], kx);
            if (ky) atomicAdd(&ds.c[o + 1], ky);
            if (tz) atomicAdd(&ds.c[o + 2], tz);
            cnt[0] += 1u;
            cnt[1] += lvl == 1;
            cnt[2] += lvl == 2;
        }
    }
    // counters: one atomic per warp
    const unsigned F = 0xffffffffu;
    unsigned long long *C = D.status->cnt[parity];
    const unsigned c0 = __reduce_add_sync(F, cnt[0]), c1 = __reduce_add_sync(F, cnt[1]);
    const unsigned c2 = __reduce_add_sync(F, cnt[2]), c3 = __reduce_add_sync(F, cnt[3]);
    if ((threadIdx.x & 31) == 0) {
        if (c0) atomicAdd(&C[kCntLinks], (unsigned long long)c0);
        if (c1) atomicAdd(&C[kCntBzLinear], (unsigned long long)c1);
        if (c2) atomicAdd(&C[kCntBzSimple], (unsigned long long)c2);
        if (c3) atomicAdd(&C[kCntThermHalf], (unsigned long long)c3);
    }
}

// ---- single-instance kernels
// Warps per particle, one CTA each (link_team): eight while that is a single
// wave (three CTAs of 80 registers per SM), else four (eight CTAs of 64
// registers).  Link kernel, us, eight / four (CUDA events): 8 disks 9.9 / 11.9,
// 300 disks 12.1 / 14.2, 129 ellipses 21.3 / 23.0, 4800 disks 84.7 / 72.1.
// (12 CTAs per SM: 82.3.)  With many particles it is bound by its scattered
// accesses: the loads and stores of the links alone, from a kernel that does
// nothing else, take 61 us for 4800 disks in 4000^2 from HBM, in any layout of
// the planes.
// Sixteen for zones of more than 32 rows while there is a particle per SM or
// fewer: their lines and links then take one round instead of two.  Disks with
// zones of 34, 43 and 60 rows, eight / sixteen: 1 particle 12.0 / 10.7,
// 12.6 / 10.6, 14.6 / 12.5; 152 particles (one per SM) 12.1 / 10.8, 12.2 / 11.3,
// 14.8 / 13.5; 153 particles 12.3 / 14.6, 13.0 / 14.9, 15.2 / 18.1.
// One or two where many particles with small zones would wait for their turn:
// a CTA's chain of dependent loads is as long for a small zone, so what counts
// is how many particles an SM holds at once (32, 16 or 8).  Disks 0.3 or 4
// apart, one / two / four: zones of 5 rows, 27,556 of them 79 / 109 / 207;
// 9 rows, 24,649 106 / 117 / 223; 11 rows, 6,724 38 / 39 / 49; 13 rows, 44,521
// 222 / 243 / 336; 23 rows, 21,025 231 / 211 / 255; 31 rows, 8,464
// 160 / 139 / 154.  Below the lines of link_team four are as good or better:
// 11 rows, 3,136 particles (21 per SM) 34 / 34 / 31; 23 rows, 5,329 (35 per SM)
// 98 / 83 / 81; 43 rows, 5,184 208 / 159 / 152.
constexpr int link_ctas(int team) { return team <= 4 ? 32 / team : team == 8 ? 3 : 1; }
template <typename T, int kTeam>
__global__ void __launch_bounds__(32 * kTeam, link_ctas(kTeam))
    k_links(const Dev D, T *A, const int *__restrict__ own,
            int *__restrict__ own_nxt, int parity, int ahead)
{
    // CTAs in the link order (descending y, the rows stream-collide wrote
    // last first; after a sweep from the last row down, the reverse: so the
    // rows the next sweep begins with are gathered last)
    const int b = (int)blockIdx.x;
    const bool rev = D.sweep && parity;
    auto at = [&](int i) { return __ldg(D.lorder + (rev ? D.np - 1 - i : i)); };
    links_body<T, kTeam>(D, A, own, own_nxt, parity, at(b), b + ahead < D.np ? at(b + ahead) : -1);
}
template <int kPB>
__global__ void __launch_bounds__(32 * kPB, part_ctas(kPB)) k_particles(const Dev D, int parity, int *own_nxt)
{
    particles_body<kPB>(D, parity, own_nxt, (int)blockIdx.x);
}
__global__ void __launch_bounds__(kBoxThreads)
    k_raster(const Dev D, int *own, bool bits, int parity)
{
    raster_body(D, own, bits, parity, (int)blockIdx.x);
}
// The node bits before a step of `parity` from a state image's flag map, a
// thread per word.
__global__ void k_flags_in(const Dev D, const uint8_t *flags, int parity)
{
    const int w = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
    if (w >= D.bpitch) return;
    unsigned now = 0u, before = 0u;
    for (int b = 0; b < 32 && 32 * w + b < D.nx; ++b) {
        const uint8_t f = flags[(long long)j * D.pitch + 32 * w + b];
        now |= (f == kSolid ? 1u : 0u) << b;
        before |= (f == kNewborn ? 1u : 0u) << b;
    }
    bits_put(D, bits_row(D, j, parity), w, now);
    bits_put(D, bits_row(D, j, parity ^ 1), w, before);
}

// ---- batched kernels: one grid over all instances (InstArgs table, block
// offsets `start`).  The link kernel's look-ahead owner-row prefetch stays
// within the instance.
template <typename T, int kTeam>
__global__ void __launch_bounds__(32 * kTeam, link_ctas(kTeam))
    k_links_batch(const InstArgs *__restrict__ I, const int *__restrict__ start, int n, int parity, int ahead)
{
    __shared__ Dev sD;
    const int i = batch_find(start, n, (int)blockIdx.x);
    const InstArgs &a = I[i];
    copy_dev(sD, a.D);
    const int par = parity ^ a.poff;
    const int b = (int)blockIdx.x - __ldg(start + i);
    links_body<T, kTeam>(sD, static_cast<T *>(a.A[par]), a.own[par], a.own[par ^ 1], par, b,
                         b + ahead < sD.np ? b + ahead : -1);
}
template <int kPB>
__global__ void __launch_bounds__(32 * kPB, part_ctas(kPB))
    k_particles_batch(const InstArgs *__restrict__ I, const int *__restrict__ start, int n, int parity)
{
    __shared__ Dev sD;
    const int i = batch_find(start, n, (int)blockIdx.x);
    copy_dev(sD, I[i].D);
    const int par = parity ^ I[i].poff;
    particles_body<kPB>(sD, par, I[i].own[par ^ 1], (int)blockIdx.x - __ldg(start + i));
}
// Geometry records of both parities' states.
__global__ void k_geom_init(const Dev D)
{
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= D.np) return;
    for (int q = 0; q < 2; ++q) {
        const PartSoA &P = D.part[q];
        double2 cs;
        cos_sin_rn(P.th[a], cs.x, cs.y);
        D.cs[q][a] = cs;
        D.geo[q][a] = make_geom(P.x[a], P.y[a], P.r[a], P.b[a], P.th[a], P.ux[a], P.uy[a], P.om[a], P.T[a], P.rho[a],
                                D.rho_f, D.g);
    }
    const PartSoA &P = D.part[0];
    D.pconst[a] = part_consts(P.r[a], P.b[a], P.rho[a], D.rho_f, D.g);
}

// Link order: the particles by descending y in kOrderBands bands of rows,
// counting-sorted by one block (inside a band, in the order of the block's
// shared-memory atomics).  Stream-collide writes the rows in ascending y,
// so the rows it wrote last are still in L2 when the next link kernel
// gathers from them, and the CTAs of the particles there run first (at
// 4000^2 / 4800 disks: link kernel 78.6 against 84.0 us, step 0.3697
// against 0.3750 ms).  Only the order of the CTAs changes, not what any of
// them computes.
constexpr int kOrderBands = 1024;
__global__ void __launch_bounds__(kOrderBands) k_link_order(const Dev D, int parity)
{
    __shared__ int cnt[kOrderBands], at[kOrderBands];
    const int t = threadIdx.x;
    auto band = [&](int p) {
        const double y = D.part[parity].y[p];
        const int b = (int)((double)kOrderBands * (((double)D.ny - 1.0) - y) / (double)D.ny);
        return min(max(b, 0), kOrderBands - 1);
    };
    cnt[t] = 0;
    __syncthreads();
    for (int p = t; p < D.np; p += kOrderBands) atomicAdd(&cnt[band(p)], 1);
    __syncthreads();
    at[t] = cnt[t];
    __syncthreads();
    for (int o = 1; o < kOrderBands; o <<= 1) { // inclusive prefix sum
        const int v = t >= o ? at[t - o] : 0;
        __syncthreads();
        at[t] += v;
        __syncthreads();
    }
    at[t] -= cnt[t]; // first position of band t
    __syncthreads();
    for (int p = t; p < D.np; p += kOrderBands) {
        const int pos = atomicAdd(&at[band(p)], 1);
        if (in_bounds(D, pos, D.np)) D.lorder[pos] = p;
    }
}

__global__ void k_pack_particles(const Dev D, lbm_particle *out, int parity)
{
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= D.np) return;
    const PartSoA &C = D.part[parity];
    lbm_particle P;
    P.x = C.x[a]; P.y = C.y[a]; P.ux = C.ux[a]; P.uy = C.uy[a];
    P.theta = C.th[a]; P.omega = C.om[a]; P.r = C.r[a]; P.rho = C.rho[a];
    P.T = C.T[a]; P.b = C.b[a];
    out[a] = P;
}

namespace {

// f(storage tag, team tag) for a storage and a team size.
template <typename F>
auto link_dispatch(int storage, int team, F &&f)
{
    auto by_team = [&](auto t) {
        return team == 1   ? f(t, std::integral_constant<int, 1>{})
               : team == 2 ? f(t, std::integral_constant<int, 2>{})
               : team == 4 ? f(t, std::integral_constant<int, 4>{})
               : team == 8 ? f(t, std::integral_constant<int, 8>{})
                           : f(t, std::integral_constant<int, 16>{});
    };
    return storage == LBM_STORE_BF16   ? by_team(__nv_bfloat16{})
           : storage == LBM_STORE_FP16 ? by_team(__half{})
                                       : by_team(float{});
}

// Warps per particle for np particles with zones of at most N rows (see
// link_ctas).
int link_team(int np, int N, int sms)
{
    if (np <= sms && N > 32) return 16;
    if (np > 32 * sms && N <= 12) return 1;
    if (np > 56 * sms && N <= 40) return 2;
    return np <= link_ctas(8) * sms ? 8 : 4;
}
int sm_count()
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 0;
    return sms;
}

template <typename F>
cudaError_t part_dispatch(int pb, F &&f)
{
    switch (pb) {
    case 1: return f(std::integral_constant<int, 1>{});
    case 2: return f(std::integral_constant<int, 2>{});
    case 4: return f(std::integral_constant<int, 4>{});
    default: return f(std::integral_constant<int, 8>{});
    }
}
// Particles per block of the update (see particles_body).
int part_per_block(int np, int sms)
{
    int pb = 1;
    while (pb < kPartMax && np > pb * sms) pb *= 2;
    return pb;
}

// CTAs of a link kernel for zones of side N that the GPU holds at once (the
// distance of its prefetch).
template <typename K>
cudaError_t link_resident(K fn, int team, int N, int sms, int *ahead)
{
    int per_sm = 0;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, 32 * team, link_smem_bytes(N));
    if (e != cudaSuccess) return e;
    *ahead = max(1, sms * per_sm);
    return cudaSuccess;
}

} // namespace

cudaError_t prepare_links(Dev &D)
{
    D.link_ahead = 1;
    D.link_team = 4;
    D.part_pb = 8;
    if (D.np == 0) return cudaSuccess;
    const int sms = sm_count();
    if (!sms) return cudaErrorUnknown;
    D.link_team = link_team(D.np, D.zone_max, sms);
    D.part_pb = part_per_block(D.np, sms);
    return link_dispatch(D.storage, D.link_team, [&](auto t, auto team) {
        return link_resident(k_links<decltype(t), decltype(team)::value>, decltype(team)::value, D.zone_max, sms,
                                   &D.link_ahead);
    });
}

cudaError_t launch_links(const Dev &D, void *A, const int *own_cur, int *own_nxt, int parity,
                         cudaStream_t s)
{
    if (D.np == 0) return cudaSuccess;
    return link_dispatch(D.storage, D.link_team, [&](auto t, auto team) {
        using T = decltype(t);
        constexpr int W = decltype(team)::value;
        k_links<T, W><<<D.np, 32 * W, link_smem_bytes(D.zone_max), s>>>(D, static_cast<T *>(A), own_cur, own_nxt,
                                                                        parity, D.link_ahead);
        return cudaGetLastError();
    });
}

// ---- batched launches (one grid over all instances)
cudaError_t prepare_links_batch(int zone_max, int np, int storage, LinkPlan *plan)
{
    const int sms = sm_count();
    if (!sms) return cudaErrorUnknown;
    plan->team = link_team(np, zone_max, sms);
    plan->part_pb = part_per_block(np, sms);
    plan->smem = link_smem_bytes(zone_max);
    return link_dispatch(storage, plan->team, [&](auto t, auto team) {
        return link_resident(k_links_batch<decltype(t), decltype(team)::value>, decltype(team)::value, zone_max,
                                   sms, &plan->ahead);
    });
}

cudaError_t launch_links_batch(const InstArgs *I, const int *start, int n, int total, int storage, int parity,
                               const LinkPlan &plan, cudaStream_t s)
{
    if (total <= 0) return cudaSuccess;
    return link_dispatch(storage, plan.team, [&](auto t, auto team) {
        constexpr int W = decltype(team)::value;
        k_links_batch<decltype(t), W><<<total, 32 * W, plan.smem, s>>>(I, start, n, parity, plan.ahead);
        return cudaGetLastError();
    });
}

cudaError_t launch_particles_batch(const InstArgs *I, const int *start, int n, int total, int parity, int pb,
                                   cudaStream_t s)
{
    if (total <= 0) return cudaSuccess;
    return part_dispatch(pb, [&](auto t) {
        constexpr int kPB = decltype(t)::value;
        k_particles_batch<kPB><<<total, 32 * kPB, 0, s>>>(I, start, n, parity);
        return cudaGetLastError();
    });
}

// Blocks of each batched step kernel for one instance.
void batch_blocks(const Dev &D, dim3 sc_block, int part_pb, int out[kBatchPhases])
{
    out[kBLinks] = D.np;
    out[kBParticles] = (D.np + part_pb - 1) / part_pb;
    out[kBRefill] = (D.np + kBoxThreads - 1) / kBoxThreads;
    out[kBStream] = ((D.pitch / kScNodes + (int)sc_block.x - 1) / (int)sc_block.x) *
                    ((D.ny + (int)sc_block.y - 1) / (int)sc_block.y);
    out[kBBoundary] = kBoundaryBlocksPerInstance;
}

cudaError_t launch_near_mask(const Dev &D, int parity, cudaStream_t s)
{
    const size_t words = ((size_t)D.ny * D.near_tpr + 31) / 32;
    cudaError_t e = cudaMemsetAsync(D.near, 0, words * sizeof(unsigned), s);
    if (e != cudaSuccess || D.np == 0) return e;
    const int span = 32 * kScNodes;
    const long long threads = (long long)D.np * (D.zone_max + 2 * kNearMargin);
    k_near_mask<<<(unsigned)((threads + 127) / 128), 128, 0, s>>>(D, span, parity);
    return cudaGetLastError();
}

cudaError_t launch_links_direct(const Dev &D, void *A, const int *own_cur, int *own_nxt, int parity,
                                cudaStream_t s)
{
    if (D.np == 0) return cudaSuccess;
    k_direct_prep<<<D.np, kBoxThreads, 0, s>>>(D, own_nxt, parity);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    dim3 grid((D.nx + 127) / 128, D.ny);
    switch (D.storage) {
    case LBM_STORE_FP32: k_links_direct<float><<<grid, 128, 0, s>>>(D, static_cast<float *>(A), own_cur, parity); break;
    case LBM_STORE_BF16:
        k_links_direct<__nv_bfloat16><<<grid, 128, 0, s>>>(D, static_cast<__nv_bfloat16 *>(A), own_cur, parity);
        break;
    case LBM_STORE_FP16: k_links_direct<__half><<<grid, 128, 0, s>>>(D, static_cast<__half *>(A), own_cur, parity); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_particles(const Dev &D, int parity, int *own_nxt, cudaStream_t s)
{
    if (D.np == 0) return cudaSuccess;
    return part_dispatch(D.part_pb, [&](auto pb) {
        constexpr int kPB = decltype(pb)::value;
        k_particles<kPB><<<(D.np + kPB - 1) / kPB, 32 * kPB, 0, s>>>(D, parity, own_nxt);
        return cudaGetLastError();
    });
}

cudaError_t launch_raster(const Dev &D, int *own, bool bits, int parity, cudaStream_t s)
{
    if (D.np == 0) return cudaSuccess;
    const int per = kBoxThreads / 32;
    k_raster<<<(D.np + per - 1) / per, kBoxThreads, 0, s>>>(D, own, bits, parity);
    return cudaGetLastError();
}

cudaError_t launch_geom_init(const Dev &D, cudaStream_t s)
{
    if (D.np == 0) return cudaSuccess;
    k_geom_init<<<(D.np + 127) / 128, 128, 0, s>>>(D);
    return cudaGetLastError();
}

cudaError_t launch_link_order(const Dev &D, int parity, cudaStream_t s)
{
    if (D.np == 0) return cudaSuccess;
    k_link_order<<<1, kOrderBands, 0, s>>>(D, parity);
    return cudaGetLastError();
}

cudaError_t launch_cells_init(const Dev &D, cudaStream_t s)
{
    const size_t counts = ((size_t)D.cell_gx * D.cell_gy + 1) * sizeof(int);
    for (int b = 0; b < 2; ++b) {
        const cudaError_t e = cudaMemsetAsync(D.cells[b], 0, counts, s);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_flags_in(const Dev &D, const uint8_t *flags, int parity, cudaStream_t s)
{
    k_flags_in<<<dim3((D.bpitch + 31) / 32, D.ny), 32, 0, s>>>(D, flags, parity);
    return cudaGetLastError();
}

cudaError_t launch_pack_particles(const Dev &D, lbm_particle *out, int parity, cudaStream_t s)
{
    if (D.np == 0) return cudaSuccess;
    k_pack_particles<<<(D.np + 127) / 128, 128, 0, s>>>(D, out, parity);
    return cudaGetLastError();
}

} // namespace lbm
