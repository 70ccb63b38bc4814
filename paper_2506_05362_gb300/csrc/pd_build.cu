// Set-up and rebuild kernels: node ordering, cell grid, bond CSR, contact
// candidate lists, and the small per-node reductions (damage, critical step,
// contact pairs for output).
#include "pd_build.cuh"
#include "pd_df.cuh"
#include "pd_grid.cuh"

namespace {

__device__ __forceinline__ double dadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double dsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double dmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double sq3(double a, double b, double c)
{
    return dadd(dadd(dmul(a, a), dmul(b, b)), dmul(c, c));
}

// ---- node ordering ---------------------------------------------------------
__device__ __forceinline__ uint64_t spread21(uint64_t v)
{
    v &= 0x1fffffull;
    v = (v | (v << 32)) & 0x1f00000000ffffull;
    v = (v | (v << 16)) & 0x1f0000ff0000ffull;
    v = (v | (v << 8)) & 0x100f00f00f00f00full;
    v = (v | (v << 4)) & 0x10c30c30c30c30c3ull;
    v = (v | (v << 2)) & 0x1249249249249249ull;
    return v;
}

__global__ void k_morton(const double *__restrict__ x, int64_t n, double lx, double ly, double lz,
                         double sx, double sy, double sz, uint64_t *key, uint32_t *val)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        uint64_t qx = (uint64_t)fmin(fmax(floor((x[3 * i] - lx) * sx), 0.0), 2097151.0);
        uint64_t qy = (uint64_t)fmin(fmax(floor((x[3 * i + 1] - ly) * sy), 0.0), 2097151.0);
        uint64_t qz = (uint64_t)fmin(fmax(floor((x[3 * i + 2] - lz) * sz), 0.0), 2097151.0);
        key[i] = spread21(qx) | (spread21(qy) << 1) | (spread21(qz) << 2);
        val[i] = (uint32_t)i;
    }
}

__global__ void k_grain_keys(const int32_t *__restrict__ grain, const uint32_t *__restrict__ order, int64_t n,
                             uint64_t *key)
{
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
        key[k] = (uint64_t)(uint32_t)grain[order[k]];
}

__global__ void k_gather_nodes(const uint32_t *__restrict__ perm, int64_t n, const double *__restrict__ x,
                               const double *__restrict__ vol, const int32_t *__restrict__ grain,
                               const double *__restrict__ v0, int32_t *perm_out, int32_t *inv, dbl4 *x4,
                               int32_t *grain_out, dbl4 *v, float4 *xh4, float4 *xl4, double cx, double cy,
                               double cz)
{
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = perm[k];
        perm_out[k] = (int32_t)i;
        inv[i] = (int32_t)k;
        dbl4 a;
        a.x = x[3 * i]; a.y = x[3 * i + 1]; a.z = x[3 * i + 2]; a.w = vol[i];
        x4[k] = a;
        grain_out[k] = grain[i];
        dbl4 vv;
        vv.x = v0 ? v0[3 * i] : 0.0; vv.y = v0 ? v0[3 * i + 1] : 0.0; vv.z = v0 ? v0[3 * i + 2] : 0.0; vv.w = 0.0;
        v[k] = vv;
        if (xh4) {
            // split of x relative to the bounding-box centre (xi is translation invariant)
            const double rx = a.x - cx, ry = a.y - cy, rz = a.z - cz;
            float4 h, l;
            h.x = __double2float_rn(rx); l.x = __double2float_rn(rx - (double)h.x);
            h.y = __double2float_rn(ry); l.y = __double2float_rn(ry - (double)h.y);
            h.z = __double2float_rn(rz); l.z = __double2float_rn(rz - (double)h.z);
            h.w = (float)a.w; l.w = 0.f;
            xh4[k] = h;
            xl4[k] = l;
        }
    }
}

// ---- grid --------------------------------------------------------------------
// Cell, FP32 position and bucket of every node; the bucket's counter gives the node's
// place in it.
__global__ void k_cell_keys(const dbl4 *__restrict__ x4, const dbl4 *__restrict__ u4, const float4 *__restrict__ hi,
                            const float4 *__restrict__ lo, int stride, int64_t n, double lx, double ly, double lz,
                            double inv, uint32_t mask, uint32_t *key, uint32_t *rank, uint32_t *count, uint64_t *cell,
                            float4 *pf)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const dbl4 a = x4[i];
        double px = a.x, py = a.y, pz = a.z;
        if (u4) {
            const dbl4 u = u4[i];
            px = dadd(px, u.x); py = dadd(py, u.y); pz = dadd(pz, u.z);
        } else if (hi) {
            const float4 h = hi[stride * i], l = lo[stride * i];
            px = dadd(px, df_to_double(df{h.x, l.x}));
            py = dadd(py, df_to_double(df{h.y, l.y}));
            pz = dadd(pz, df_to_double(df{h.z, l.z}));
        }
        const int cx = grid_coord(px, lx, inv), cy = grid_coord(py, ly, inv), cz = grid_coord(pz, lz, inv);
        cell[i] = grid_pack(cx, cy, cz);
        const float fx = (float)dsub(px, lx), fy = (float)dsub(py, ly), fz = (float)dsub(pz, lz);
        pf[i] = make_float4(fx, fy, fz, fmaxf(fabsf(fx), fmaxf(fabsf(fy), fabsf(fz))));
        const uint32_t b = grid_hash(cx, cy, cz, mask);
        key[i] = b;
        rank[i] = atomicAdd(count + b, 1u);
    }
}

// sum over the threads of lower index in the block, and the block's total
template <int THREADS>
__device__ __forceinline__ unsigned block_prefix(unsigned v, unsigned &total)
{
    __shared__ unsigned ws[THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[warp] = x;
    __syncthreads();
    unsigned before = 0;
    total = 0;
#pragma unroll
    for (int w = 0; w < THREADS / 32; ++w) {
        if (w < warp) before += ws[w];
        total += ws[w];
    }
    __syncthreads();
    return before + x - v;
}

// Entry ranges of the buckets: a block lays its 1024 buckets out one after another from
// where the cursor stands (which block comes first does not matter).
__global__ void __launch_bounds__(256) k_bucket_ranges(const uint32_t *__restrict__ count, uint32_t nbuckets,
                                                       unsigned *cursor, uint2 *range)
{
    __shared__ unsigned s_base;
    const uint32_t b = blockIdx.x * 1024 + threadIdx.x * 4;  // nbuckets is a multiple of 1024
    const uint4 c = *(const uint4 *)(count + b);
    unsigned total;
    unsigned s = block_prefix<256>(c.x + c.y + c.z + c.w, total);
    if (threadIdx.x == 0) s_base = atomicAdd(cursor, total);
    __syncthreads();
    s += s_base;
    range[b] = make_uint2(s, s + c.x);
    s += c.x;
    range[b + 1] = make_uint2(s, s + c.y);
    s += c.y;
    range[b + 2] = make_uint2(s, s + c.z);
    s += c.z;
    range[b + 3] = make_uint2(s, s + c.w);
}

__global__ void k_bucket_fill(const uint32_t *__restrict__ key, const uint32_t *__restrict__ rank,
                              const uint2 *__restrict__ range, const uint64_t *__restrict__ cell,
                              const float4 *__restrict__ pf, int64_t n, uint32_t *node, uint64_t *ecell, float4 *epf)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t e = range[key[i]].x + rank[i];
        node[e] = (uint32_t)i;
        ecell[e] = cell[i];
        epf[e] = pf[i];
    }
}

// ---- bonds -------------------------------------------------------------------
// What the filters say of a node alone, two bits a filter.  Inner sphere: both bits
// when the node is not strictly inside, so a bond is kept when its ends share a bit.
// Notch: the side of the plane (bit 0 above, bit 1 below) when the node is clearly off it:
// a bond whose ends share a bit does not cross the plane, whatever the rounding of the
// exact test (the margin is 10^6 times the error of the plane's FP64 value); a bond whose
// ends share none is tested by notch_drops.  Decided per bond, the spheres alone took
// four fifths of the bond search's time (FP64 on a few lanes of every warp).
__global__ void k_filter_sides(const dbl4 *__restrict__ x4, int64_t n, FilterSet f, uint16_t *sides)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const dbl4 x = x4[i];
        unsigned m = 0;
        for (int q = 0; q < f.nf; ++q) {
            const double *p = f.a[q];
            if (f.kind[q] == 1) {
                const double a = p[0] * x.x, b = p[1] * x.y, c = p[2] * x.z;
                const double v = ((a + b) + c) + p[3], tol = 1e-9 * (((fabs(a) + fabs(b)) + fabs(c)) + fabs(p[3]));
                if (v > tol) m |= 1u << (2 * q);
                if (v < -tol) m |= 2u << (2 * q);
            } else {
                const double d = sq3(dsub(x.x, p[0]), dsub(x.y, p[1]), dsub(x.z, p[2]));
                if (!(d < dmul(p[3], p[3]))) m |= 3u << (2 * q);
            }
        }
        sides[i] = (uint16_t)m;
    }
}

// Notch test of one bond with the endpoints in canonical order (smaller caller index first).
__device__ bool notch_drops(const double *x1, const double *x2, const double *p)
{
    double dx = dsub(x2[0], x1[0]), dy = dsub(x2[1], x1[1]), dz = dsub(x2[2], x1[2]);
    double num = dadd(dadd(dadd(dmul(p[0], x1[0]), dmul(p[1], x1[1])), dmul(p[2], x1[2])), p[3]);
    double den = dadd(dadd(dmul(p[0], dx), dmul(p[1], dy)), dmul(p[2], dz));
    if (den == 0.0) return false;
    double t = __ddiv_rn(-num, den);
    if (!(t > 0.0 && t < 1.0)) return false;
    double r0 = dadd(x1[0], dmul(t, dx)), r1 = dadd(x1[1], dmul(t, dy)), r2 = dadd(x1[2], dmul(t, dz));
    return r0 >= p[4] && r0 <= p[7] && r1 >= p[5] && r1 <= p[8] && r2 >= p[6] && r2 <= p[9];
}

// Whether a filter drops the bond between nodes i and j of sides si and sj.
__device__ __forceinline__ bool filters_drop(const FilterSet &f, unsigned si, unsigned sj, const dbl4 *x4,
                                             const int32_t *perm, int64_t i, int32_t j)
{
    const unsigned m = si & sj;
    unsigned open = ~(m | (m >> 1)) & 0x5555u & ((1u << (2 * f.nf)) - 1u);  // filters whose ends share no bit
    for (; open; open &= open - 1) {
        const int q = (__ffs(open) - 1) >> 1;
        if (f.kind[q] == 2) return true;
        const dbl4 a = x4[i], b = x4[j];
        const double pa[3] = {a.x, a.y, a.z}, pb[3] = {b.x, b.y, b.z};
        if (perm[i] < perm[j] ? notch_drops(pa, pb, f.a[q]) : notch_drops(pb, pa, f.a[q])) return true;
    }
    return false;
}

// The exact horizon test.  Out of line: inlined, its FP64 arithmetic is executed for
// every candidate with the result discarded (980 us instead of 270).
__device__ __noinline__ bool within64(const dbl4 *x4, int64_t i, int32_t j, double d2max)
{
    const dbl4 a = x4[i], b = x4[j];
    return sq3(dsub(b.x, a.x), dsub(b.y, a.y), dsub(b.z, a.z)) < d2max;
}

// The bond partners of node i, found by a warp: each of the 27 cells' entries is read by
// consecutive lanes (a cell one horizon wide holds some 27 lattice nodes).  FILL = false
// counts them; FILL = true writes them in the order they are found (k_order_rows sorts
// the rows).  A thread a node, walking all 700 entries by itself, took 2.4 ms for the
// 74,290 nodes of a hollow sphere (2,300 warps), this 0.27 (and 0.35 to fill).
template <bool FILL>
__global__ void __launch_bounds__(256) k_bonds(const dbl4 *__restrict__ x4, const int32_t *__restrict__ grain,
                                               const int32_t *__restrict__ perm, int64_t n, GridView g, double delta2,
                                               FilterSet f, const uint16_t *__restrict__ sides, int64_t *cnt,
                                               const int64_t *__restrict__ off, int32_t *found)
{
    const float deltaf = (float)sqrt(delta2);
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n; i += nwarps) {
        const float4 pi = g.pf[i];
        const int gi = grain[i];
        const unsigned si = f.nf ? sides[i] : 0u;
        const uint64_t pc = g.cell[i];
        const int cx = (int)((pc >> 42) & 0x1fffff) - 1048576, cy = (int)((pc >> 21) & 0x1fffff) - 1048576,
                  cz = (int)(pc & 0x1fffff) - 1048576;
        uint2 range = make_uint2(0u, 0u);  // lane c holds the entries of cell c
        uint64_t want = 0;
        if (lane < 27) {
            const int x = cx + lane % 3 - 1, y = cy + lane / 3 % 3 - 1, z = cz + lane / 9 - 1;
            range = __ldg(g.range + grid_hash(x, y, z, g.mask));
            want = grid_pack(x, y, z);
        }
        int64_t k = FILL ? off[i] : 0;
        for (int c = 0; c < 27; ++c) {
            const uint32_t e = __shfl_sync(0xffffffffu, range.y, c);
            const uint64_t w = __shfl_sync(0xffffffffu, want, c);
            for (uint32_t t0 = __shfl_sync(0xffffffffu, range.x, c); t0 < e; t0 += 32) {
                const uint32_t t = t0 + lane;
                bool ok = false;
                int32_t j = 0;
                if (t < e && __ldg(g.ecell + t) == w) {
                    // FP32 decides pairs clearly inside or outside the horizon; the exact
                    // FP64 predicate decides the band between
                    const float4 pj = __ldg(g.epf + t);
                    const float d2f = pf_dist2(pi, pj), sl = pf_slack(deltaf, pi, pj);
                    const float hi = deltaf + sl, lo = deltaf - sl;
                    j = (int32_t)__ldg(g.node + t);
                    ok = d2f < hi * hi && j != i && grain[j] == gi;
                    if (ok && !(d2f < lo * lo)) ok = within64(x4, i, j, delta2);
                    if (ok && f.nf) ok = !filters_drop(f, si, sides[j], x4, perm, i, j);
                }
                const unsigned m = __ballot_sync(0xffffffffu, ok);
                if (FILL && ok) found[k + __popc(m & lt)] = j;
                k += __popc(m);
            }
        }
        if (!FILL && lane == 0) cnt[i] = k;
    }
}

// Rows into ascending order, and the canonical (caller-order) slot of every bond, by
// counting: a warp takes a row, and an element's place is the number of elements below
// it, its canonical place the number whose caller index is below its own.  Rows of up to
// ORDER_ROW elements are staged in shared memory, longer ones read where they are.  Two
// radix sorts of all B bonds by 64-bit keys did this before, in 14 passes over 24 bytes
// a bond.
constexpr int ORDER_ROW = 512, ORDER_WARPS = 8;

// places of the elements q0 + 32 u + lane, u < U, of a row (row: staged, or null)
template <int U, typename E>
__device__ __forceinline__ void place(E element, const int2 *row, int q0, int len, int lane, int64_t k0, int64_t c0,
                                      int32_t *col, int32_t *kc_of)
{
    int2 e[U];
    int a[U], c[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int q = q0 + 32 * u + lane;
        e[u] = q < len ? element(q) : make_int2(-1, -1);
        a[u] = c[u] = 0;
    }
    auto count = [&](int2 r) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            a[u] += r.x < e[u].x;
            c[u] += r.y < e[u].y;
        }
    };
    if (row) {
#pragma unroll 4
        for (int q = 0; q < len; ++q) count(row[q]);
    } else {
        for (int q = 0; q < len; ++q) count(element(q));
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
        if (q0 + 32 * u + lane < len) {
            col[k0 + a[u]] = e[u].x;
            kc_of[k0 + a[u]] = (int32_t)(c0 + c[u]);
        }
}

__global__ void __launch_bounds__(32 * ORDER_WARPS) k_order_rows(const int32_t *__restrict__ found,
                                                                 const int64_t *__restrict__ rowptr,
                                                                 const int32_t *__restrict__ perm,
                                                                 const int64_t *__restrict__ crow, int64_t n,
                                                                 int32_t *col, int32_t *kc_of)
{
    __shared__ int2 s_row[ORDER_WARPS][ORDER_ROW];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int2 *row = s_row[warp];
    const int64_t nwarps = (int64_t)gridDim.x * ORDER_WARPS;
    for (int64_t i = (int64_t)blockIdx.x * ORDER_WARPS + warp; i < n; i += nwarps) {
        const int64_t k0 = rowptr[i];
        const int len = (int)(rowptr[i + 1] - k0);
        const int64_t c0 = crow[perm[i]];
        const bool staged = len <= ORDER_ROW;
        if (staged) {
            for (int q = lane; q < len; q += 32) {
                const int32_t j = found[k0 + q];
                row[q] = make_int2(j, perm[j]);
            }
            __syncwarp();
        }
        auto element = [&](int q) {
            if (staged) return row[q];
            const int32_t j = found[k0 + q];
            return make_int2(j, perm[j]);
        };
        int q0 = 0;
        for (; len - q0 > 64; q0 += 128) place<4>(element, staged ? row : nullptr, q0, len, lane, k0, c0, col, kc_of);
        if (len - q0 > 32) place<2>(element, staged ? row : nullptr, q0, len, lane, k0, c0, col, kc_of);
        else if (len > q0) place<1>(element, staged ? row : nullptr, q0, len, lane, k0, c0, col, kc_of);
        __syncwarp();
    }
}

// ---- contact candidates ---------------------------------------------------------
// Slot of j in the ascending row i, or -1.
__device__ __forceinline__ int64_t find_slot(const int64_t *rowptr, const int32_t *col, int64_t i, int32_t j)
{
    int64_t lo = rowptr[i], hi = rowptr[i + 1];
    while (lo < hi) {
        int64_t mid = (lo + hi) >> 1;
        if (col[mid] < j) lo = mid + 1; else hi = mid;
    }
    return (lo < rowptr[i + 1] && col[lo] == j) ? lo : -1;
}

// Visits the nodes closer to node i than the search distance (a superset of them: the
// step kernel applies the exact FP64 contact predicate).
template <typename F>
__device__ __forceinline__ void near_nodes(const GridView &g, int64_t i, float cutf, F f)
{
    const float4 pi = g.pf[i];
    const uint64_t pc = g.cell[i];
    const int cx = (int)((pc >> 42) & 0x1fffff) - 1048576, cy = (int)((pc >> 21) & 0x1fffff) - 1048576,
              cz = (int)(pc & 0x1fffff) - 1048576;
    for (int dz = -1; dz <= 1; ++dz)
        for (int dy = -1; dy <= 1; ++dy) {
            uint2 range[3];  // three cells' ranges in flight
#pragma unroll
            for (int dx = 0; dx < 3; ++dx)
                range[dx] = __ldg(g.range + grid_hash(cx + dx - 1, cy + dy, cz + dz, g.mask));
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) {
                const uint64_t want = grid_pack(cx + dx - 1, cy + dy, cz + dz);
                for (uint32_t t = range[dx].x; t < range[dx].y; ++t) {
                    const uint64_t ce = __ldg(g.ecell + t);
                    const float4 pj = __ldg(g.epf + t);
                    if (ce != want) continue;
                    const float lim = cutf + pf_slack(cutf, pi, pj);
                    if (!(pf_dist2(pi, pj) < lim * lim)) continue;
                    const int32_t j = (int32_t)__ldg(g.node + t);
                    if (j != i) f(j);
                }
            }
        }
}

// Contact candidates in one walk: a thread collects its node's candidates in ascending
// partner order (so that the step kernels add contact terms in an order that does not
// depend on the grid's), the block takes room for its rows from the cursor, and every
// row's range goes to rng.  A row of more than CAND_LOCAL candidates is walked again.
// (Counting, scanning and filling in separate passes walked the grid twice and took five
// launches.  With the counting sort above in place of a three-pass radix sort a rebuild on
// the 178,200-node plate is 4 launches and 78 us instead of 25 launches and 270 us, bound
// by the latency of the 27 cells' scattered entries.)  Lists that outgrow cap set PDE_CAPACITY; the cursor holds the room needed.
constexpr int CAND_LOCAL = 16;

__global__ void __launch_bounds__(128) k_cand(const int32_t *__restrict__ grain, const int64_t *__restrict__ rowptr,
                                              const int32_t *__restrict__ col, int64_t n, GridView g, float cutf,
                                              longlong2 *rng, int2 *cand, int64_t cap, unsigned long long *cursor,
                                              unsigned *err, double *disp, int *stale)
{
    __shared__ unsigned long long s_base;
    // a segment whose list went stale takes no further step (written by earlier kernels only)
    if (*(volatile const unsigned *)err & PDE_SKIN) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *disp = 0.0;
        *stale = 0;
    }
    for (int64_t i0 = (int64_t)blockIdx.x * 128; i0 < n; i0 += (int64_t)gridDim.x * 128) {
        const int64_t i = i0 + threadIdx.x;
        int32_t hit[CAND_LOCAL];
        unsigned k = 0;
        if (i < n)
            near_nodes(g, i, cutf, [&](int32_t j) {
                if (k < CAND_LOCAL) {
                    unsigned b = k;
                    for (; b > 0 && hit[b - 1] > j; --b) hit[b] = hit[b - 1];
                    hit[b] = j;
                }
                ++k;
            });
        unsigned total;
        const unsigned before = block_prefix<128>(k, total);
        if (threadIdx.x == 0) s_base = total ? atomicAdd(cursor, (unsigned long long)total) : 0ull;
        __syncthreads();
        const int64_t base = (int64_t)s_base;
        __syncthreads();
        const bool fits = base + total <= cap;  // uniform over the block
        if (!fits && threadIdx.x == 0) atomicOr(err, (unsigned)PDE_CAPACITY);
        if (i >= n) continue;
        const int64_t c0 = base + before;
        rng[i] = fits ? make_longlong2(c0, c0 + k) : make_longlong2(0, 0);
        if (!fits) continue;
        const int gi = grain[i];
        auto entry = [&](int32_t j) {
            return make_int2(j, grain[j] == gi ? (int)find_slot(rowptr, col, i, j) : -1);
        };
        int2 *row = cand + c0;
        if (k <= CAND_LOCAL) {
            for (unsigned q = 0; q < k; ++q) row[q] = entry(hit[q]);
        } else {
            unsigned m = 0;
            near_nodes(g, i, cutf, [&](int32_t j) {
                const int2 c = entry(j);
                unsigned b = m++;
                for (; b > 0 && row[b - 1].x > j; --b) row[b] = row[b - 1];
                row[b] = c;
            });
        }
    }
}

// Exact contact pairs from the candidate lists at the current state (for output).
template <bool FILL>
__global__ void k_pairs(const dbl4 *__restrict__ x4, const dbl4 *__restrict__ u4, const int32_t *__restrict__ perm,
                        const uint32_t *__restrict__ brk, const longlong2 *__restrict__ cp,
                        const int2 *__restrict__ cand, int64_t n, double R2, int64_t *cnt, const int64_t *__restrict__ off, int32_t *out)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const dbl4 a = x4[i], ua = u4[i];
        const double px = dadd(a.x, ua.x), py = dadd(a.y, ua.y), pz = dadd(a.z, ua.z);
        int64_t k = 0;
        const longlong2 rng = cp[i];
        for (int64_t q = rng.x; q < rng.y; ++q) {
            const int2 c = cand[q];
            if (c.y >= 0 && !((brk[c.y >> 5] >> (c.y & 31)) & 1u)) continue;
            const dbl4 bj = x4[c.x], uj = u4[c.x];
            const double r2 = sq3(dsub(dadd(bj.x, uj.x), px), dsub(dadd(bj.y, uj.y), py), dsub(dadd(bj.z, uj.z), pz));
            if (!(r2 < R2)) continue;
            if (FILL) {
                out[2 * (off[i] + k)] = perm[i];
                out[2 * (off[i] + k) + 1] = perm[c.x];
            }
            ++k;
        }
        if (!FILL) cnt[i] = k;
    }
}

// ---- reductions ------------------------------------------------------------------
__global__ void k_damage(const int64_t *__restrict__ rowptr, const uint32_t *__restrict__ brk,
                         const int32_t *__restrict__ perm, int64_t n, double *phi_caller)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k0 = rowptr[i], k1 = rowptr[i + 1];
        int64_t broken = 0;
        for (int64_t k = k0; k < k1; ++k) broken += (brk[k >> 5] >> (k & 31)) & 1u;
        const int64_t nb0 = k1 - k0;
        phi_caller[perm[i]] = nb0 ? 1.0 - (double)(nb0 - broken) / (double)nb0 : 0.0;
    }
}

__global__ void k_stable_dt(const dbl4 *__restrict__ x4, const int64_t *__restrict__ rowptr,
                            const int32_t *__restrict__ col, int64_t n, double c, double rho, double delta,
                            int conic, double *dt_out)
{
    __shared__ double s_min[256];
    double best = INFINITY;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k0 = rowptr[i], k1 = rowptr[i + 1];
        if (k1 == k0) continue;
        const dbl4 a = x4[i];
        double sum = 0.0;
        for (int64_t k = k0; k < k1; ++k) {
            const dbl4 b = x4[col[k]];
            const double L = sqrt(sq3(b.x - a.x, b.y - a.y, b.z - a.z));
            sum += b.w * (conic ? c * (delta - L) : c) / L;
        }
        best = fmin(best, sqrt(2.0 * rho / sum));
    }
    s_min[threadIdx.x] = best;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) s_min[threadIdx.x] = fmin(s_min[threadIdx.x], s_min[threadIdx.x + o]);
        __syncthreads();
    }
    if (threadIdx.x == 0) dt_out[blockIdx.x] = s_min[0];
}

// ---- canonical (caller-order) bond numbering ------------------------------------
__global__ void k_row_len_caller(const int64_t *__restrict__ rowptr, const int32_t *__restrict__ inv, int64_t n,
                                 int64_t *len)
{
    for (int64_t ic = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; ic < n; ic += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = inv[ic];
        len[ic] = rowptr[i + 1] - rowptr[i];
    }
}

__global__ void k_col_caller(const int32_t *__restrict__ col, const int32_t *__restrict__ perm,
                             const int32_t *__restrict__ kc_of, int64_t B, int32_t *out)
{
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < B; k += (int64_t)gridDim.x * blockDim.x)
        out[kc_of[k]] = perm[col[k]];
}

__global__ void k_bits_to_bytes(const uint32_t *__restrict__ brk, const int32_t *__restrict__ kc_of, int64_t B,
                                uint8_t *out)
{
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < B; k += (int64_t)gridDim.x * blockDim.x)
        out[kc_of[k]] = (uint8_t)((brk[k >> 5] >> (k & 31)) & 1u);
}

// The internal bitset from one byte per canonical slot.  A warp builds one word
// at a time: lane l takes internal slot 32 w + l (coalesced reads of the slot
// map), and the word is the ballot of the lanes' bits.
__global__ void k_bytes_to_bits(const uint8_t *__restrict__ in, const int32_t *__restrict__ kc_of, int64_t B,
                                uint32_t *brk)
{
    const int64_t nw = (B + 31) >> 5;
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < nw; w += nwarps) {
        const int64_t k = (w << 5) + lane;
        const bool bit = k < B && in[kc_of[k]] != 0;
        const uint32_t word = __ballot_sync(0xffffffffu, bit);
        if (lane == 0) brk[w] = word;
    }
}

// Canonical packed bits (bit c % 32 of word c / 32 for canonical slot c) from the
// internal bitset: the words are cleared first, then every broken internal slot
// ORs its canonical bit (breaks are sparse, so the atomics are few).
__global__ void k_bits_to_packed(const uint32_t *__restrict__ brk, const int32_t *__restrict__ kc_of, int64_t B,
                                 uint32_t *out)
{
    const int64_t nw = (B + 31) >> 5;
    for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < nw; w += (int64_t)gridDim.x * blockDim.x) {
        uint32_t word = brk[w];
        while (word) {
            const int b = __ffs(word) - 1;
            word &= word - 1;
            const int64_t k = (w << 5) + b;
            if (k < B) {
                const int32_t c = kc_of[k];
                atomicOr(out + (c >> 5), 1u << (c & 31));
            }
        }
    }
}

// the internal bitset from canonical packed bits, a word per warp as above
__global__ void k_packed_to_bits(const uint32_t *__restrict__ in, const int32_t *__restrict__ kc_of, int64_t B,
                                 uint32_t *brk)
{
    const int64_t nw = (B + 31) >> 5;
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < nw; w += nwarps) {
        const int64_t k = (w << 5) + lane;
        bool bit = false;
        if (k < B) {
            const int32_t c = kc_of[k];
            bit = (in[c >> 5] >> (c & 31)) & 1u;
        }
        const uint32_t word = __ballot_sync(0xffffffffu, bit);
        if (lane == 0) brk[w] = word;
    }
}

// ---- shared-memory tiles -----------------------------------------------------------
// Tile t = rows [t*T, (t+1)*T).  Keys (t << sh | node) for every bond target and
// for every row itself; sorted and de-duplicated they give the tile's node list.
__global__ void k_tile_keys(const int64_t *__restrict__ rowptr, const int32_t *__restrict__ col, int64_t n, int T,
                            int sh, uint64_t *keys)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t t = (uint64_t)(i / T) << sh;
        for (int64_t k = rowptr[i]; k < rowptr[i + 1]; ++k) keys[k] = t | (uint64_t)(uint32_t)col[k];
        keys[rowptr[n] + i] = t | (uint64_t)i;
    }
}

__global__ void k_unique_flags(const uint64_t *__restrict__ keys, int64_t m, int64_t *flag)
{
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < m; q += (int64_t)gridDim.x * blockDim.x)
        flag[q] = (q == 0 || keys[q] != keys[q - 1]) ? 1 : 0;
}

__global__ void k_unique_scatter(const uint64_t *__restrict__ keys, const int64_t *__restrict__ pos, int64_t m,
                                 int sh, int64_t ntiles, int32_t *ulist, int64_t *tile_ptr)
{
    const uint64_t mask = (1ull << sh) - 1ull;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < m; q += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t k = keys[q];
        if (q == 0 || k != keys[q - 1]) ulist[pos[q]] = (int32_t)(k & mask);
        if (q == 0 || (k >> sh) != (keys[q - 1] >> sh)) tile_ptr[k >> sh] = pos[q];
        if (q == m - 1) tile_ptr[ntiles] = pos[m];
    }
}

__device__ __forceinline__ int32_t lsearch(const int32_t *__restrict__ a, int32_t len, int32_t v)
{
    int32_t lo = 0, hi = len;
    while (lo < hi) {
        const int32_t mid = (lo + hi) >> 1;
        if (a[mid] < v) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// tile-local index of every bond target and of every row (tiles above cap get 0xffff)
__global__ void k_local_cols(const int64_t *__restrict__ rowptr, const int32_t *__restrict__ col, int64_t n, int T,
                             const int32_t *__restrict__ ulist, const int64_t *__restrict__ tile_ptr, int cap,
                             uint16_t *lcol, uint16_t *lrow)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t t = i / T;
        const int64_t base = tile_ptr[t];
        const int32_t len = (int32_t)(tile_ptr[t + 1] - base);
        const bool fits = len <= cap;
        lrow[i] = fits ? (uint16_t)lsearch(ulist + base, len, (int32_t)i) : 0xffffu;
        for (int64_t k = rowptr[i]; k < rowptr[i + 1]; ++k)
            lcol[k] = fits ? (uint16_t)lsearch(ulist + base, len, col[k]) : 0xffffu;
    }
}

// broken flag of every slot copied into bit 15 of its local index
__global__ void k_sync_lcol_flags(const uint32_t *__restrict__ brk, int64_t B, uint16_t *lcol)
{
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < B; k += (int64_t)gridDim.x * blockDim.x)
        lcol[k] = (uint16_t)((lcol[k] & 0x7fffu) | (((brk[k >> 5] >> (k & 31)) & 1u) << 15));
}

// neighbour index with the slot's broken flag in bit 31
__global__ void k_sync_colf_flags(const uint32_t *__restrict__ brk, const int32_t *__restrict__ col, int64_t B,
                                  int32_t *colf)
{
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < B; k += (int64_t)gridDim.x * blockDim.x)
        colf[k] = (int32_t)((uint32_t)col[k] | (((brk[k >> 5] >> (k & 31)) & 1u) << 31));
}

// Index arrays of the each-bond-once passes: split[i] = first slot of row i whose
// neighbour index exceeds i (rows are sorted ascending); for each such slot k
// (bond i -> j), mir[k] = the slot of i in row j, and mir of that slot = k.  A
// bond without its reverse (the lists are symmetric by construction) sets *bad.
__global__ void k_pair_index(const int64_t *__restrict__ rowptr, const int32_t *__restrict__ col, int64_t n,
                             int32_t *split, int32_t *mir, unsigned *bad)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k0 = rowptr[i], k1 = rowptr[i + 1];
        int64_t a = k0, b = k1;  // first slot with col > i
        while (a < b) {
            const int64_t m = (a + b) >> 1;
            if (col[m] > i) b = m; else a = m + 1;
        }
        split[i] = (int32_t)a;
        for (int64_t k = a; k < k1; ++k) {
            const int64_t j = col[k];
            int64_t lo = rowptr[j], hi = rowptr[j + 1];
            while (lo < hi) {
                const int64_t m = (lo + hi) >> 1;
                if (col[m] < i) lo = m + 1; else hi = m;
            }
            if (lo < rowptr[j + 1] && col[lo] == i) {
                mir[k] = (int32_t)lo;
                mir[lo] = (int32_t)k;
            } else {
                mir[k] = -1;
                atomicOr(bad, 1u);
            }
        }
    }
}

// ---- state conversion -----------------------------------------------------------
__global__ void k_to_caller(const dbl4 *__restrict__ in, const int32_t *__restrict__ perm, int64_t n, double *out)
{
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        const dbl4 a = in[k];
        const int64_t i = perm[k];
        out[3 * i] = a.x; out[3 * i + 1] = a.y; out[3 * i + 2] = a.z;
    }
}

// flag |= bit when any of a[0..m) is not finite (one atomic per warp that saw one)
__global__ void k_nonfinite(const double *__restrict__ a, int64_t m, unsigned bit, unsigned *flag)
{
    bool bad = false;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < m; k += (int64_t)gridDim.x * blockDim.x)
        bad |= !isfinite(a[k]);
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(flag, bit);
}

// flag |= bit when applying the caller-order doubles `staged` would change the
// current state: on the mixed path, when the split of a staged value (the one
// applying uses) differs from the live pair (hi, lo) at stride `stride`; else when
// it differs from the FP64 array d64.  The halves are compared as numbers (a zero
// of either sign counts as equal).  The live pairs lie on the FP64 grid, so a
// state read out and sent back unchanged splits into exactly the live pairs.
__global__ void k_state_differs(const double *__restrict__ staged, const int32_t *__restrict__ perm, int64_t n,
                                const float4 *__restrict__ hi, const float4 *__restrict__ lo, int stride,
                                const dbl4 *__restrict__ d64, unsigned bit, unsigned *flag)
{
    bool diff = false;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = perm[k];
        const double a = staged[3 * i], b = staged[3 * i + 1], c = staged[3 * i + 2];
        if (hi) {
            const float4 h = hi[stride * k], l = lo[stride * k];
            const df sa = df_from_double(a), sb = df_from_double(b), sc = df_from_double(c);
            diff |= (sa.hi != h.x) | (sa.lo != l.x) | (sb.hi != h.y) | (sb.lo != l.y) | (sc.hi != h.z) |
                    (sc.lo != l.z);
        } else {
            const dbl4 q = d64[k];
            diff |= (a != q.x) | (b != q.y) | (c != q.z);
        }
    }
    if (__any_sync(0xffffffffu, diff) && (threadIdx.x & 31) == 0) atomicOr(flag, bit);
}

__global__ void k_words_differ(const uint32_t *__restrict__ a, const uint32_t *__restrict__ b, int64_t nw,
                               uint32_t last_mask, unsigned bit, unsigned *flag)
{
    bool diff = false;
    for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < nw; w += (int64_t)gridDim.x * blockDim.x)
        diff |= ((a[w] ^ b[w]) & (w == nw - 1 ? last_mask : 0xffffffffu)) != 0u;
    if (__any_sync(0xffffffffu, diff) && (threadIdx.x & 31) == 0) atomicOr(flag, bit);
}

__global__ void k_from_caller(const double *__restrict__ in, const int32_t *__restrict__ perm, int64_t n, dbl4 *out)
{
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = perm[k];
        dbl4 a;
        a.x = in[3 * i]; a.y = in[3 * i + 1]; a.z = in[3 * i + 2]; a.w = 0.0;
        out[k] = a;
    }
}

__global__ void k_split(const dbl4 *__restrict__ u, int64_t n, float4 *hi, float4 *lo)
{
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        const dbl4 a = u[k];
        float4 h, l;
        h.x = __double2float_rn(a.x); l.x = __double2float_rn(a.x - (double)h.x);
        h.y = __double2float_rn(a.y); l.y = __double2float_rn(a.y - (double)h.y);
        h.z = __double2float_rn(a.z); l.z = __double2float_rn(a.z - (double)h.z);
        h.w = 0.f; l.w = 0.f;
        hi[k] = h;
        lo[k] = l;
    }
}

__global__ void k_vmax(const dbl4 *__restrict__ v, int64_t n, double *out)
{
    __shared__ double s_m[256];
    double m = 0.0;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        const dbl4 a = v[k];
        m = fmax(m, a.x * a.x + a.y * a.y + a.z * a.z);
    }
    s_m[threadIdx.x] = m;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) s_m[threadIdx.x] = fmax(s_m[threadIdx.x], s_m[threadIdx.x + o]);
        __syncthreads();
    }
    if (threadIdx.x == 0) out[blockIdx.x] = sqrt(s_m[0]);
}

}  // namespace

// ----------------------------------------------------------------------------------
static inline int grid_of(int64_t n, int threads = 256)
{
    int64_t b = (n + threads - 1) / threads;
    if (b > 8192) b = 8192;
    if (b < 1) b = 1;
    return (int)b;
}

void build_morton(const double *x_dev, int64_t n, const double lo[3], const double hi[3], uint64_t *key,
                  uint64_t *key_alt, uint32_t *val, uint32_t *val_alt, int grain_bits, const int32_t *grain_dev,
                  int64_t *tmp, uint32_t **order_out, cudaStream_t st)
{
    double s[3];
    for (int a = 0; a < 3; ++a) {
        double ext = hi[a] - lo[a];
        s[a] = ext > 0 ? 2097151.0 / ext : 0.0;
    }
    k_morton<<<grid_of(n), 256, 0, st>>>(x_dev, n, lo[0], lo[1], lo[2], s[0], s[1], s[2], key, val);
    uint64_t *k = key, *ka = key_alt;
    uint32_t *v = val, *va = val_alt;
    radix_sort_u64(&k, &ka, &v, &va, n, 63, tmp, st);
    if (grain_bits > 0) {
        k_grain_keys<<<grid_of(n), 256, 0, st>>>(grain_dev, v, n, k);
        radix_sort_u64(&k, &ka, &v, &va, n, grain_bits, tmp, st);
    }
    *order_out = v;
}

void gather_nodes(const uint32_t *order, int64_t n, const double *x, const double *vol, const int32_t *grain,
                  const double *v0, int32_t *perm, int32_t *inv, dbl4 *x4, int32_t *grain_out, dbl4 *v,
                  float4 *xh4, float4 *xl4, const double centre[3], cudaStream_t st)
{
    k_gather_nodes<<<grid_of(n), 256, 0, st>>>(order, n, x, vol, grain, v0, perm, inv, x4, grain_out, v, xh4, xl4,
                                               centre[0], centre[1], centre[2]);
}

void grid_build(GridView &g, const GridBuf &w, const dbl4 *x4, const dbl4 *u4, const float4 *hi, const float4 *lo,
                int stride, int64_t n, double cs, cudaStream_t st)
{
    g.inv = 1.0 / cs;
    g.mask = w.nbuckets - 1;
    cudaMemsetAsync(w.count, 0, sizeof(uint32_t) * (w.nbuckets + 4), st);
    k_cell_keys<<<grid_of(n), 256, 0, st>>>(x4, u4, hi, lo, stride, n, g.lo[0], g.lo[1], g.lo[2], g.inv, g.mask, w.key,
                                            w.rank, w.count, w.cell, w.pf);
    k_bucket_ranges<<<w.nbuckets / 1024, 256, 0, st>>>(w.count, w.nbuckets, w.bucket_cursor(), w.range);
    k_bucket_fill<<<grid_of(n), 256, 0, st>>>(w.key, w.rank, w.range, w.cell, w.pf, n, w.node, w.ecell, w.epf);
    g.range = w.range;
    g.node = w.node;
    g.ecell = w.ecell;
    g.epf = w.epf;
    g.cell = w.cell;
    g.pf = w.pf;
}

void bonds_count(const dbl4 *x4, const int32_t *grain, const int32_t *perm, int64_t n, const GridView &g,
                 double delta, const FilterSet &f, uint16_t *sides, int64_t *cnt, cudaStream_t st)
{
    if (f.nf) k_filter_sides<<<grid_of(n), 256, 0, st>>>(x4, n, f, sides);
    k_bonds<false><<<grid_of(32 * n), 256, 0, st>>>(x4, grain, perm, n, g, delta * delta, f, sides, cnt, nullptr, nullptr);
}

void bonds_fill(const dbl4 *x4, const int32_t *grain, const int32_t *perm, int64_t n, const GridView &g,
                double delta, const FilterSet &f, const uint16_t *sides, const int64_t *off, int32_t *found,
                cudaStream_t st)
{
    k_bonds<true><<<grid_of(32 * n), 256, 0, st>>>(x4, grain, perm, n, g, delta * delta, f, sides, nullptr, off, found);
}

void order_rows(const int32_t *found, const int64_t *rowptr, const int32_t *perm, const int64_t *crow, int64_t n,
                int32_t *col, int32_t *kc_of, cudaStream_t st)
{
    k_order_rows<<<grid_of(n, ORDER_WARPS), 32 * ORDER_WARPS, 0, st>>>(found, rowptr, perm, crow, n, col, kc_of);
}

void cand_build(const int32_t *grain, const int64_t *rowptr, const int32_t *col, int64_t n, const GridView &g,
                const GridBuf &w, double cut, longlong2 *rng, int2 *cand, int64_t cap, unsigned *err, double *disp,
                int *stale, cudaStream_t st)
{
    k_cand<<<grid_of(n, 128), 128, 0, st>>>(grain, rowptr, col, n, g, (float)cut, rng, cand, cap, w.cand_cursor(), err,
                                            disp, stale);
}

void pairs_count(const dbl4 *x4, const dbl4 *u4, const int32_t *perm, const uint32_t *brk, const longlong2 *cp,
                 const int2 *cand, int64_t n, double Rc, int64_t *cnt, cudaStream_t st)
{
    k_pairs<false><<<grid_of(n), 256, 0, st>>>(x4, u4, perm, brk, cp, cand, n, Rc * Rc, cnt, nullptr, nullptr);
}

void pairs_fill(const dbl4 *x4, const dbl4 *u4, const int32_t *perm, const uint32_t *brk, const longlong2 *cp,
                const int2 *cand, int64_t n, double Rc, const int64_t *off, int32_t *out, cudaStream_t st)
{
    k_pairs<true><<<grid_of(n), 256, 0, st>>>(x4, u4, perm, brk, cp, cand, n, Rc * Rc, nullptr, off, out);
}

void damage(const int64_t *rowptr, const uint32_t *brk, const int32_t *perm, int64_t n, double *phi,
            cudaStream_t st)
{
    k_damage<<<grid_of(n), 256, 0, st>>>(rowptr, brk, perm, n, phi);
}

int stable_dt_blocks(int64_t n) { return grid_of(n); }

void stable_dt(const dbl4 *x4, const int64_t *rowptr, const int32_t *col, int64_t n, double c, double rho,
               double delta, int conic, double *partial, cudaStream_t st)
{
    k_stable_dt<<<grid_of(n), 256, 0, st>>>(x4, rowptr, col, n, c, rho, delta, conic, partial);
}

void row_len_caller(const int64_t *rowptr, const int32_t *inv, int64_t n, int64_t *len, cudaStream_t st)
{
    k_row_len_caller<<<grid_of(n), 256, 0, st>>>(rowptr, inv, n, len);
}

void col_caller(const int32_t *col, const int32_t *perm, const int32_t *kc_of, int64_t B, int32_t *out,
                cudaStream_t st)
{
    k_col_caller<<<grid_of(B), 256, 0, st>>>(col, perm, kc_of, B, out);
}

void bits_to_bytes(const uint32_t *brk, const int32_t *kc_of, int64_t B, uint8_t *out, cudaStream_t st)
{
    k_bits_to_bytes<<<grid_of(B), 256, 0, st>>>(brk, kc_of, B, out);
}

void bytes_to_bits(const uint8_t *in, const int32_t *kc_of, int64_t B, uint32_t *brk, cudaStream_t st)
{
    k_bytes_to_bits<<<grid_of(B), 256, 0, st>>>(in, kc_of, B, brk);  // a warp per word
}

void bits_to_packed(const uint32_t *brk, const int32_t *kc_of, int64_t B, uint32_t *out, cudaStream_t st)
{
    const int64_t nw = (B + 31) / 32;
    cudaMemsetAsync(out, 0, sizeof(uint32_t) * (size_t)nw, st);
    k_bits_to_packed<<<grid_of(nw), 256, 0, st>>>(brk, kc_of, B, out);
}

void packed_to_bits(const uint32_t *in, const int32_t *kc_of, int64_t B, uint32_t *brk, cudaStream_t st)
{
    k_packed_to_bits<<<grid_of(B), 256, 0, st>>>(in, kc_of, B, brk);  // a warp per word
}

void to_caller(const dbl4 *in, const int32_t *perm, int64_t n, double *out, cudaStream_t st)
{
    k_to_caller<<<grid_of(n), 256, 0, st>>>(in, perm, n, out);
}

void check_finite(const double *a, int64_t m, unsigned bit, unsigned *flag, cudaStream_t st)
{
    k_nonfinite<<<grid_of(m), 256, 0, st>>>(a, m, bit, flag);
}

void state_differs(const double *staged, const int32_t *perm, int64_t n, const float4 *hi, const float4 *lo,
                   int stride, const dbl4 *d64, unsigned bit, unsigned *flag, cudaStream_t st)
{
    k_state_differs<<<grid_of(n), 256, 0, st>>>(staged, perm, n, hi, lo, stride, d64, bit, flag);
}

void words_differ(const uint32_t *a, const uint32_t *b, int64_t nw, uint32_t last_mask, unsigned bit, unsigned *flag,
                  cudaStream_t st)
{
    k_words_differ<<<grid_of(nw), 256, 0, st>>>(a, b, nw, last_mask, bit, flag);
}

void from_caller(const double *in, const int32_t *perm, int64_t n, dbl4 *out, cudaStream_t st)
{
    k_from_caller<<<grid_of(n), 256, 0, st>>>(in, perm, n, out);
}

void split_hilo(const dbl4 *u, int64_t n, float4 *hi, float4 *lo, cudaStream_t st)
{
    k_split<<<grid_of(n), 256, 0, st>>>(u, n, hi, lo);
}

int vmax_blocks(int64_t n)
{
    int b = grid_of(n);
    return b > 1024 ? 1024 : b;
}

void vmax(const dbl4 *v, int64_t n, double *partial, cudaStream_t st)
{
    k_vmax<<<vmax_blocks(n), 256, 0, st>>>(v, n, partial);
}

void build_tiles(const int64_t *rowptr, const int32_t *col, int64_t n, int64_t B, int T, int sh, int cap,
                 uint64_t *keys, uint64_t *keys_alt, int64_t *flag, int64_t *pos, int64_t *tmp, int32_t *ulist,
                 int64_t *tile_ptr, uint16_t *lcol, uint16_t *lrow, cudaStream_t st)
{
    const int64_t m = B + n;
    const int64_t ntiles = (n + T - 1) / T;
    int tbits = 1;
    while (((int64_t)1 << tbits) <= ntiles) ++tbits;
    k_tile_keys<<<grid_of(n, 128), 128, 0, st>>>(rowptr, col, n, T, sh, keys);
    uint64_t *k = keys, *ka = keys_alt;
    radix_sort_u64(&k, &ka, nullptr, nullptr, m, sh + tbits, tmp, st);
    k_unique_flags<<<grid_of(m), 256, 0, st>>>(k, m, flag);
    scan_exclusive_i64(flag, pos, m, tmp, st);
    k_unique_scatter<<<grid_of(m), 256, 0, st>>>(k, pos, m, sh, ntiles, ulist, tile_ptr);
    k_local_cols<<<grid_of(n, 128), 128, 0, st>>>(rowptr, col, n, T, ulist, tile_ptr, cap, lcol, lrow);
}

void sync_lcol_flags(const uint32_t *brk, int64_t B, uint16_t *lcol, cudaStream_t st)
{
    k_sync_lcol_flags<<<grid_of(B), 256, 0, st>>>(brk, B, lcol);
}

void pair_index(const int64_t *rowptr, const int32_t *col, int64_t n, int32_t *split, int32_t *mir, unsigned *bad,
                cudaStream_t st)
{
    k_pair_index<<<grid_of(n), 256, 0, st>>>(rowptr, col, n, split, mir, bad);
}

void sync_colf_flags(const uint32_t *brk, const int32_t *col, int64_t B, int32_t *colf, cudaStream_t st)
{
    if (B > 0) k_sync_colf_flags<<<grid_of(B), 256, 0, st>>>(brk, col, B, colf);
}
