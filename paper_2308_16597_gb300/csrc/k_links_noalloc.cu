// Allocation-free variant of the link kernel: gather the fixed index array
// of fluid-particle links, apply the curved bounce-back on every link and
// reduce the momentum-exchange force and torque per particle, with the index
// array held in a file-scope device array instead of a caller workspace.
//
// Who needs it: code that may not allocate device memory at the point where
// it computes particle forces, e.g. a host application whose device memory
// is owned by another allocator or pool it cannot extend, or a caller inside
// a section where cudaMalloc is not allowed.  Such a caller still owns and
// passes the distributions, the owner map, the particles and the force
// output; the only scratch (the index array) lives here.
//
// Zones of at most 60 nodes a side take the two kernels in the second half of
// this file, which keep the links on chip and hold the particles' records in
// that array; larger ones the three that follow.
//
// The array holds 2,097,152 slots (node + wall fraction, 8 bytes each) and
// the slot offsets of up to 32,768 particles: 16 MiB + 128 KiB held on every
// GPU that loads the library, for the life of the process.  All calls share
// it and it keeps the contents of the last call, so calls whose GPU work
// overlaps (on two streams, or from two threads) race on it.  Every call
// looks up the array's device address on the current device
// (cudaGetSymbolAddress); the first call on a device also loads the
// library's device code there, so make that first call before any stream
// capture.
#include <climits>
#include <cmath>

#include "lbm_internal.cuh"

namespace lbm {
namespace {

constexpr long long kStaticSlots = 1ll << 21;   // 2,097,152 slots
constexpr int kStaticParticles = 1 << 15;       // 32,768 particles
constexpr int kThreads = 256;

// [slot nodes: int32 x kStaticSlots][wall fractions: float x kStaticSlots]
// [slot offsets: int32 x (kStaticParticles + 1)][reject flag: uint32]
constexpr size_t kScratchBytes =
    (size_t)kStaticSlots * 8 + ((size_t)kStaticParticles + 1) * 4 + 256;

static __device__ __align__(256) unsigned char g_link_scratch[kScratchBytes];

struct Scratch {
    int *node;
    float *q;
    int *base;
    unsigned *reject; // set when a radius exceeds r_max for this call
};

__host__ __device__ inline Scratch carve(unsigned char *p)
{
    Scratch s;
    s.node = reinterpret_cast<int *>(p);
    s.q = reinterpret_cast<float *>(p + (size_t)kStaticSlots * 4);
    s.base = reinterpret_cast<int *>(p + (size_t)kStaticSlots * 8);
    s.reject = reinterpret_cast<unsigned *>(p + (size_t)kStaticSlots * 8 +
                                            ((size_t)kStaticParticles + 1) * 4);
    return s;
}

struct View {
    float *A;
    long long ps;
    int pitch, nx, ny, n;
    double r_max;
    const int *own;
    const lbm_particle *P;
    double *F;
};

// Force and torque of a particle from its links' exact sums (NaN for a particle one of
// whose lines holds two links); one copy of the code, so that both paths
// round alike.
__device__ __noinline__ void store_force(double *F, const LinkSums &S, double xc, double yc, bool broken)
{
    double f[3];
    assemble_force(S, xc, yc, f[0], f[1], f[2]);
    for (int i = 0; i < 3; ++i) F[i] = broken ? __longlong_as_double(0x7ff8000000000000ll) : f[i];
}

// Slot offsets: running sum of 12N - 12 over the particles (one thread).
// The reject flag is rewritten on every call: set when some radius exceeds
// the r_max the host checked the capacity against, or when a particle breaks
// the shape rule of lbm_init (semi-minor axis b negative, or, for an
// ellipse, b below 1 or above the semi-major axis r, or |theta| above 1.6e6),
// since the zone and the slot capacity are sized from r.
__global__ void k_static_bases(View v, unsigned char *scratch)
{
    Scratch s = carve(scratch);
    if (threadIdx.x == 0) {
        int acc = 0;
        unsigned bad = 0u;
        for (int a = 0; a < v.n; ++a) {
            s.base[a] = acc;
            const double r = v.P[a].r, b = v.P[a].b;
            const bool shape_ok = b >= 0.0 && (!is_ellipse(r, b) || (b >= 1.0 && b <= r &&
                                                                     fabs(v.P[a].theta) <= 1.6e6));
            if (!(r >= 1.0 && r <= v.r_max) || !shape_ok) bad = 1u;
            else acc += slot_capacity(r);
        }
        s.base[v.n] = acc;
        *s.reject = bad;
    }
}

__device__ __forceinline__ bool in_box(const View &v, int i, int j)
{
    return i >= 0 && i < v.nx && j >= 0 && j < v.ny;
}

// Phase 1: one CTA per particle fills its 12N - 12 slots (Sec. 3 mapping).
// A line holding two links is marked -2 (the particle's force becomes NaN).
__global__ void __launch_bounds__(kThreads) k_static_gather(View v, unsigned char *scratch)
{
    Scratch s = carve(scratch);
    if (*s.reject) return;
    const int p = blockIdx.x;
    const double xc = v.P[p].x, yc = v.P[p].y, r = v.P[p].r;
    const DiskDF dk = disk_df(xc, yc, r);
    const bool ell = is_ellipse(r, v.P[p].b);
    EllFrame E{};
    if (ell) E = ell_frame(xc, yc, v.P[p].theta, r, v.P[p].b);
    const int N = zone_size(r), cap = 12 * N - 12;
    const int X0 = zone_lo(xc, r), Y0 = zone_lo(yc, r);
    const int base = s.base[p];
    for (int t0 = threadIdx.x; t0 < cap; t0 += kThreads) {
        int k, line;
        slot_dir_line(t0, N, k, line);
        int found = 0, fi = 0, fj = 0;
        for (int t = 0; t < N; ++t) {
            int a, b;
            if (!zone_point(k, N, line, t, a, b)) continue;
            const int i = X0 + a, j = Y0 + b;
            if (!in_box(v, i, j) || v.own[(long long)j * v.nx + i] != -1) continue;
            const int si = i + ex(k), sj = j + ey(k);
            if (!in_box(v, si, sj) || v.own[(long long)sj * v.nx + si] != p) continue;
            if (++found == 1) {
                fi = i;
                fj = j;
            }
        }
        float dxf, dyf;
        s.node[base + t0] = found > 1 ? -2 : found ? fj * v.nx + fi : -1;
        s.q[base + t0] = !found ? 0.f : ell ? link_q_ellipse(fi, fj, k, E, dxf, dyf) : link_q_df(fi, fj, k, dk, dxf, dyf);
    }
}

// Phase 2: bounce-back and momentum exchange on the gathered slots, with the
// same device helpers, per-link arithmetic, exact fixed-point sums (here by
// one warp over the valid slots in slot order) and FP64 assembly as the
// workspace kernels, so the forces agree bit for bit.
// Shared memory: the compacted slot list and the per-link results,
// 24 bytes per slot of the largest zone.
__global__ void __launch_bounds__(kThreads) k_static_bbforce(View v, unsigned char *scratch, int capm)
{
    Scratch s = carve(scratch);
    const int p = blockIdx.x;
    if (*s.reject) {
        if (threadIdx.x < 3) v.F[3 * p + threadIdx.x] = __longlong_as_double(0x7ff8000000000000ll);
        return;
    }
    __shared__ int s_warp[kThreads / 32 + 1];
    extern __shared__ int list[]; // [capm] valid slots in slot order, then the per-link results
    float *lbx = reinterpret_cast<float *>(list + capm);
    float *lby = lbx + capm;
    float *ltq = lby + capm;
    int *lcode = reinterpret_cast<int *>(ltq + capm);
    int *ltz = lcode + capm;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const double xc = v.P[p].x, yc = v.P[p].y, r = v.P[p].r;
    const DiskDF dk = disk_df(xc, yc, r);
    const bool ell = is_ellipse(r, v.P[p].b);
    const float Ux = (float)v.P[p].ux, Uy = (float)v.P[p].uy, Om = (float)v.P[p].omega;
    const float wT = (float)(0.2 * v.P[p].T);
    const int N = zone_size(r), cap = 12 * N - 12;
    const int base = s.base[p];
    int broken = 0, nvalid = 0;
    float *A = v.A;
    const long long ps = v.ps;
    for (int s0 = 0; s0 < cap; s0 += kThreads) {
        const int sl = s0 + tid;
        const int node = sl < cap ? s.node[base + sl] : -1;
        broken |= node == -2;
        const bool valid = node >= 0;
        const unsigned m = __ballot_sync(0xffffffffu, valid);
        if (lane == 0) s_warp[warp] = __popc(m);
        __syncthreads();
        if (tid == 0) {
            int acc = 0;
            for (int w = 0; w < kThreads / 32; ++w) {
                const int c = s_warp[w];
                s_warp[w] = acc;
                acc += c;
            }
            s_warp[kThreads / 32] = acc;
        }
        __syncthreads();
        if (valid) list[nvalid + s_warp[warp] + __popc(m & ((1u << lane) - 1u))] = sl;
        nvalid += s_warp[kThreads / 32];
        __syncthreads();
    }
    for (int li = tid; li < nvalid; li += kThreads) {
        const int sl2 = list[li];
        const int nd = s.node[base + sl2];
        int k, line;
        slot_dir_line(sl2, N, k, line);
        const float q = s.q[base + sl2];
        const int fi = nd % v.nx, fj = nd / v.nx;
        const int kx = ex(k), ky = ey(k), kb = opp(k);
        const int i1 = fi - kx, j1 = fj - ky, i2 = fi - 2 * kx, j2 = fj - 2 * ky;
        const bool have1 = in_box(v, i1, j1) && v.own[(long long)j1 * v.nx + i1] == -1;
        const bool have2 = in_box(v, i2, j2) && v.own[(long long)j2 * v.nx + i2] == -1;
        const long long n0 = (long long)fj * v.pitch + fi;
        const long long n1 = have1 ? (long long)j1 * v.pitch + i1 : n0;
        const long long n2 = have2 ? (long long)j2 * v.pitch + i2 : n0;
        const float fk0 = A[k * ps + n0], fk1 = A[k * ps + n1], fk2 = A[k * ps + n2];
        const float fb0 = A[kb * ps + n0], fb1 = A[kb * ps + n1];
        float dxh, dxl, dyh, dyl;
        df_offset(fi, dk.xh, dk.xl, dxh, dxl);
        df_offset(fj, dk.yh, dk.yl, dyh, dyl);
        // an ellipse: the offset rounded from FP64, as the step's link kernel has it
        const float dxf = ell ? (float)((double)fi - xc) : dxh + dxl;
        const float dyf = ell ? (float)((double)fj - yc) : dyh + dyl;
        const float rx = dxf + q * kx, ry = dyf + q * ky;
        const float uwx = Ux - Om * ry, uwy = Uy + Om * rx;
        const float wall = 6.f * w9(k) * -(kx * uwx + ky * uwy);
        int lvl;
        const float fnew = bouzidi32(q, fk0, fk1, fk2, fb0, fb1, have1, have2, wall, lvl);
        const long long ns = (long long)(fj + ky) * v.pitch + (fi + kx);
        A[kb * ps + ns] = fnew;
        if (k <= 4)
            A[(kQ9 + kb) * ps + ns] = thermal32(q, A[(kQ9 + k) * ps + n0], A[(kQ9 + k) * ps + n1],
                                                A[(kQ9 + kb) * ps + n0], have1, wT);
        const float bx = fk0 * (kx - uwx) - fnew * (-kx - uwx);
        const float by = fk0 * (ky - uwy) - fnew * (-ky - uwy);
        lbx[li] = bx;
        lby[li] = by;
        ltq[li] = rx * by - ry * bx;
        lcode[li] = k | (lvl << 4) | ((k <= 4 && !have1) ? 64 : 0);
        ltz[li] = fi * ky - fj * kx;
    }
    broken = __syncthreads_or(broken);
    if (warp == 0) {
        LinkSums S;
        int c3[3];
        reduce_links(lbx, lby, ltq, lcode, ltz, nvalid, S, c3);
        if (lane == 0) {
            store_force(v.F + 3 * p, S, xc, yc, broken);
        }
    }
}

// ---------------------------------------------------------------------------
// Zones of at most 60 nodes a side (every radius lbm_init takes): two
// kernels instead of the three above, and no index array in memory.
//
// k_static_prep, one thread per particle: its record (the FP32 / int
// geometry of the step's link kernel and an ellipse's FP64 frame) into the
// static array, and per block of kPrepThreads whether one of its particles
// breaks the radius or shape rule.
//
// k_static_links, one CTA per particle: a bit mask per row of the window
// (zone and two-node margin) for fluid nodes and for nodes of this
// particle, links as intersections of a fluid mask with a shifted owner
// mask, spread evenly over the lanes; a link claims its line's bit, a line
// claimed twice is left out (and makes the force NaN); then one link per
// thread, all its loads issued at once, summed in the exact fixed point of
// the step's kernel (so the order of the links does not matter).
//
// Bound by latency: one wave of CTAs (8 of 128 threads per SM), each a chain
// of record, owner rows, populations.  1200 disks r = 10 in 2000^2: 28.7 us
// a call; the index-array path above, kept for the zones that a row mask of
// 64 bits does not hold, takes 746 us there (one thread adds up the slot
// offsets, and every slot walks N nodes with two dependent reads of the
// owner map).  k_static_links is launched while k_static_prep still runs.
// ---------------------------------------------------------------------------
constexpr int kPrepThreads = 128;
constexpr int kLinkThreads = 128;
constexpr int kMaskZone = 60; // window of at most 64 columns: a row's mask is one 64-bit word

struct StaticRec {
    GeomRec G;
    EllFrame E;
    double x, y;
};
static_assert(sizeof(StaticRec) % 16 == 0 && sizeof(StaticRec) * kStaticParticles +
              sizeof(int) * (kStaticParticles / kPrepThreads) <= (size_t)kStaticSlots * 8,
              "the records and block flags lie where the index array of the general path does");
__host__ __device__ inline StaticRec *records(unsigned char *p) { return reinterpret_cast<StaticRec *>(p); }
__host__ __device__ inline int *block_bad(unsigned char *p)
{
    return reinterpret_cast<int *>(p + sizeof(StaticRec) * kStaticParticles);
}

__global__ void __launch_bounds__(kPrepThreads) k_static_prep(View v, unsigned char *scratch)
{
    const int a = blockIdx.x * kPrepThreads + threadIdx.x;
    bool bad = false;
    if (a < v.n) {
        const lbm_particle P = v.P[a];
        const bool ell = is_ellipse(P.r, P.b);
        bad = !(P.r >= 1.0 && P.r <= v.r_max) ||
              !(P.b >= 0.0 && (!ell || (P.b >= 1.0 && P.b <= P.r && fabs(P.theta) <= 1.6e6)));
        StaticRec R;
        // the masses do not enter a link's record
        R.G = make_geom(P.x, P.y, P.r, 0.0, 0.0, P.ux, P.uy, P.omega, P.T, 0.0, 0.0, 0.0);
        R.E = EllFrame{};
        if (ell) {
            R.E = ell_frame(P.x, P.y, P.theta, P.r, P.b);
            R.G.r = -R.G.r;
        }
        R.x = P.x;
        R.y = P.y;
        if (!bad) records(scratch)[a] = R;
    }
    bad = __syncthreads_or(bad);
    if (threadIdx.x == 0) block_bad(scratch)[blockIdx.x] = bad;
}

__global__ void __launch_bounds__(kLinkThreads, 8) k_static_links(View v, unsigned char *scratch, int capm)
{
    constexpr unsigned F = 0xffffffffu;
    constexpr int kW = kLinkThreads / 32, kWin = kMaskZone + 4;
    extern __shared__ int list[]; // [capm] links: k | a << 4 | b << 12 at zone node (a, b)
    __shared__ unsigned long long Fm[kWin], Om[kWin];
    __shared__ unsigned occ[(12 * kMaskZone + 31) / 32], dup[(12 * kMaskZone + 31) / 32];
    __shared__ int s_n;
    __shared__ LinkSums s_ws[kW];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, p = blockIdx.x;
    // the records of k_static_prep (launched ahead of its end)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    bool bad = false;
    for (int t = tid; t < (v.n + kPrepThreads - 1) / kPrepThreads; t += kLinkThreads) bad |= block_bad(scratch)[t] != 0;
    const StaticRec &R = records(scratch)[p];
    for (int t = tid; t < (12 * kMaskZone + 31) / 32; t += kLinkThreads) occ[t] = dup[t] = 0u;
    if (tid == 0) s_n = 0;
    if (__syncthreads_or(bad)) {
        if (tid < 3) v.F[3 * p + tid] = __longlong_as_double(0x7ff8000000000000ll);
        return;
    }
    const GeomRec G = R.G;
    const int N = G.N, XA = G.X0 - 2, YA = G.Y0 - 2, wy = N + 4;
    // row masks: eight rows' loads of a warp in flight before the first ballot
    for (int r0 = 0; r0 < wy; r0 += 8 * kW) {
        int lo[8], hi[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const int r = r0 + warp + t * kW, j = YA + r, i = XA + lane;
            lo[t] = (r < wy && in_box(v, i, j)) ? __ldg(v.own + (long long)j * v.nx + i) : -2;
            hi[t] = (wy > 32 && r < wy && in_box(v, i + 32, j)) ? __ldg(v.own + (long long)j * v.nx + i + 32) : -2;
        }
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const int r = r0 + warp + t * kW;
            const unsigned fl = __ballot_sync(F, lo[t] == -1), ol = __ballot_sync(F, lo[t] == p);
            const unsigned fh = __ballot_sync(F, hi[t] == -1), oh = __ballot_sync(F, hi[t] == p);
            if (lane == 0 && r < wy) {
                Fm[r] = ((unsigned long long)fh << 32) | fl;
                Om[r] = ((unsigned long long)oh << 32) | ol;
            }
        }
    }
    __syncthreads();
    const unsigned long long Z = ((1ull << N) - 1ull) << 2;
    for (int e0 = warp * 32; e0 < 8 * N; e0 += kLinkThreads) {
        const int e = e0 + lane;
        unsigned long long m = 0ull;
        int k = 1, b = 0;
        if (e < 8 * N) {
            k = 1 + e / N;
            b = e - (k - 1) * N;
            const unsigned long long o = Om[b + 2 + ey(k)];
            m = Fm[b + 2] & (ex(k) > 0 ? o >> 1 : ex(k) < 0 ? o << 1 : o) & Z;
        }
        const int cnt = __popcll(m);
        int inc = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(F, inc, o);
            if (lane >= o) inc += t;
        }
        const int total = __shfl_sync(F, inc, 31), excl = inc - cnt;
        for (int j0 = 0; j0 < total; j0 += 32) {
            const int j = j0 + lane;
            int l = 0; // the lane whose item holds link j
#pragma unroll
            for (int step = 16; step > 0; step >>= 1) {
                const int ec = __shfl_sync(F, excl, l + step);
                if (ec <= j) l += step;
            }
            unsigned long long ml = __shfl_sync(F, m, l);
            const int kl = __shfl_sync(F, k, l), bl = __shfl_sync(F, b, l), el = __shfl_sync(F, excl, l);
            bool mine = false;
            int code = 0;
            if (j < total) {
                for (int t = j - el; t > 0; --t) ml &= ml - 1ull;
                const int a = __ffsll((long long)ml) - 3, sl = slot_of(kl, a, bl, N);
                if (sl >= 0) { // a corner line has no slot
                    const unsigned bit = 1u << (sl & 31);
                    mine = !(atomicOr(&occ[sl >> 5], bit) & bit);
                    if (!mine) atomicOr(&dup[sl >> 5], bit);
                    code = kl | (a << 4) | (bl << 12);
                }
            }
            const unsigned who = __ballot_sync(F, mine);
            int at = 0;
            if (lane == 0 && who) at = atomicAdd(&s_n, __popc(who));
            at = __shfl_sync(F, at, 0) + __popc(who & ((1u << lane) - 1u));
            if (mine) list[at] = code;
        }
    }
    __syncthreads();
    const int n = s_n;
    const DiskDF dk = geom_df(G);
    const bool ell = G.r < 0.f;
    float *A = v.A;
    const long long ps = v.ps;
    auto fluid = [&](int i, int j) -> bool { return (Fm[j - YA] >> (i - XA)) & 1ull; };
    LinkAcc acc;
    bool broken = false;
    for (int li = tid; li < n; li += kLinkThreads) {
        const int c = list[li], k = c & 15, a = (c >> 4) & 255, b = c >> 12;
        const int sl = slot_of(k, a, b, N);
        if ((dup[sl >> 5] >> (sl & 31)) & 1u) {
            broken = true;
            continue;
        }
        const int fi = G.X0 + a, fj = G.Y0 + b, kx = ex(k), ky = ey(k), kb = opp(k);
        const bool have1 = fluid(fi - kx, fj - ky), have2 = fluid(fi - 2 * kx, fj - 2 * ky);
        const long long n0 = (long long)fj * v.pitch + fi, dn = (long long)ky * v.pitch + kx;
        const long long n1 = have1 ? n0 - dn : n0, n2 = have2 ? n0 - 2 * dn : n0;
        // populations of fluid nodes: nothing writes them during the kernel
        const float fk0 = __ldg(A + k * ps + n0), fk1 = __ldg(A + k * ps + n1), fk2 = __ldg(A + k * ps + n2);
        const float fb0 = __ldg(A + kb * ps + n0), fb1 = __ldg(A + kb * ps + n1);
        float g0 = 0.f, g1 = 0.f, g2 = 0.f;
        if (k <= 4) {
            g0 = __ldg(A + (kQ9 + k) * ps + n0);
            g1 = __ldg(A + (kQ9 + k) * ps + n1);
            g2 = __ldg(A + (kQ9 + kb) * ps + n0);
        }
        float dxf, dyf;
        const float q = ell ? link_q_ellipse(fi, fj, k, R.E, dxf, dyf) : link_q_df(fi, fj, k, dk, dxf, dyf);
        const float rx = dxf + q * kx, ry = dyf + q * ky;
        const float uwx = G.ux - G.om * ry, uwy = G.uy + G.om * rx;
        const float wall = 6.f * w9(k) * -(kx * uwx + ky * uwy);
        int lvl;
        const float fnew = bouzidi32(q, fk0, fk1, fk2, fb0, fb1, have1, have2, wall, lvl);
        A[kb * ps + n0 + dn] = fnew;
        if (k <= 4) A[(kQ9 + kb) * ps + n0 + dn] = thermal32(q, g0, g1, g2, have1, G.wT);
        const float bx = fk0 * (kx - uwx) - fnew * (-kx - uwx);
        const float by = fk0 * (ky - uwy) - fnew * (-ky - uwy);
        acc.add(bx, by, rx * by - ry * bx, k, lvl, k <= 4 && !have1, fi * ky - fj * kx);
    }
    int c3[3];
    LinkSums S;
    acc.finish(S, c3);
    if (lane == 0) s_ws[warp] = S;
    broken = __syncthreads_or(broken);
    if (tid == 0) {
#pragma unroll
        for (int w = 1; w < kW; ++w) add_sums(S, s_ws[w]);
        store_force(v.F + 3 * p, S, R.x, R.y, broken);
    }
}

// Device address of the static array on the current device.  Looked up on
// every call rather than cached: the query is cheap once the device code is
// loaded, and a cached address would go stale when the context is reset
// (cudaDeviceReset), which places the array anew.  In host code the array's
// name is only a host-side stand-in, never a device address.
int scratch_address(unsigned char **out)
{
    void *ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_link_scratch) != cudaSuccess || !ptr) return LBM_ECUDA;
    *out = static_cast<unsigned char *>(ptr);
    return LBM_OK;
}

} // namespace
} // namespace lbm

extern "C" int lbm_link_forces_noalloc(float *d_dist, int64_t plane_stride, int32_t pitch,
                                       const int32_t *d_owner, int32_t nx, int32_t ny,
                                       const lbm_particle *d_particles, int32_t n, double r_max,
                                       double *d_forces, void *stream)
{
    using namespace lbm;
    if (n < 0 || nx < 1 || ny < 1 || pitch < nx || plane_stride < (int64_t)pitch * ny) return LBM_EINVAL;
    // the index array stores j * nx + i as int32
    if ((long long)nx * ny > INT_MAX) return LBM_EINVAL;
    if (n == 0) return LBM_OK;
    if (!d_dist || !d_owner || !d_particles || !d_forces || !(r_max >= 1.0) || r_max > 1e6)
        return LBM_EINVAL;
    if (n > kStaticParticles || (long long)n * slot_capacity(r_max) > kStaticSlots) return LBM_ENOSPC;
    // the force kernel holds the slot list and per-link results of the
    // largest zone in shared memory
    const int capm = slot_capacity(r_max);
    const size_t smem = (size_t)capm * 6 * sizeof(int);
    if (smem > (size_t)200 * 1024) return LBM_ENOSPC;
    unsigned char *scratch = nullptr;
    int rc = scratch_address(&scratch);
    if (rc) return rc;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    View v{d_dist, (long long)plane_stride, pitch, nx, ny, n, r_max, d_owner, d_particles, d_forces};
    if (zone_size(r_max) <= kMaskZone) {
        k_static_prep<<<(n + kPrepThreads - 1) / kPrepThreads, kPrepThreads, 0, s>>>(v, scratch);
        // launched while k_static_prep runs: the kernel waits for it itself
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at.val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(n);
        cfg.blockDim = dim3(kLinkThreads);
        cfg.dynamicSmemBytes = (size_t)capm * sizeof(int);
        cfg.stream = s;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        if (cudaLaunchKernelEx(&cfg, k_static_links, v, scratch, capm) != cudaSuccess) return LBM_ECUDA;
        return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_ECUDA;
    }
    k_static_bases<<<1, 32, 0, s>>>(v, scratch);
    k_static_gather<<<n, kThreads, 0, s>>>(v, scratch);
    if (smem > (size_t)48 * 1024 &&
        cudaFuncSetAttribute(k_static_bbforce, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
            cudaSuccess)
        return LBM_ECUDA;
    k_static_bbforce<<<n, kThreads, smem, s>>>(v, scratch, capm);
    if (cudaGetLastError() != cudaSuccess) return LBM_ECUDA;
    return LBM_OK;
}
