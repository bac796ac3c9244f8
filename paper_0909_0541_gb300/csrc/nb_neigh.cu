// nb_neigh.cu -- fixed-radius neighbour search by the general treewalk
// (Sec. "General Treewalk", Fig. "general_treewalk": the descent of the force
// walk with another distance test and, in place of the particle-cell term,
// nothing; the paper names short-range interactions as its use).
//
// The neighbours of particle i are the j != i with |x_j - x_i|^2 <= h^2, the
// squared distance summed (x, y) then z in FP64 from the FP64 positions, each
// operation rounded on its own: the set is fixed by that definition, and the
// tree only prunes.  One warp walks one group breadth-first over the
// level-ordered records, as the force walk does.  A cell is skipped when its
// centre of mass lies farther from the group's box than h + s + (sqrt(3)/2) l
// (every member lies within (sqrt(3)/2) l of the cube's centre, which is s
// from the centre of mass), with a margin of 1e-5 of the root side and 1e-6 of
// the group's coordinates for the FP32 rounding of the records and boxes;
// every other cell is opened, and every particle reached is a candidate.  A
// cell of at most NG_RUN particles is not descended: its particles are one
// run of sorted slots, and testing them all costs less than walking to their
// leaves (runs of 4 and of 15: 2 and 4 % slower than 8 on that set).
//
// The particles reached are gathered in shared memory; those farther than h
// from the group's box are dropped, and the rest, the candidates, are tested
// 64 at a time, two per lane, against the members of the group (up to 64 of
// them, held in shared memory; a larger group is walked once per 64 members).
// The test runs in FP32 on group-relative coordinates and decides every pair
// whose distance
// is not within rounding of h (band below); the FP64 definition is evaluated
// only for pairs inside the band, so the result is the definition's.  On
// GB300 the FP64 pipe gives about 1/64 of the FP32 lanes: with the FP64 test
// on every pair, and the counts kept in global memory, a pass over 300,000
// uniform points with 48 neighbours each took 7.2 ms; it takes 0.30 ms (the
// fill pass 0.39 against 7.3), and took 0.35 (0.46) without the test against
// the box.
// The first pass counts, an exclusive scan gives the offsets, the second
// pass writes the caller indices, and each target's run is then sorted
// ascending: runs of up to 256 in registers by a bitonic network, longer
// ones in place by Batcher's odd-even merge sort.
#include <climits>

#include "nb_walk.cuh"

#define NG_T 256
#define NG_WARPS (NG_T / NB_WARP)
#define NG_SMEM 384   // positions of each frontier queue held in shared memory
#define NG_RUN 8      // cells of at most this many particles are taken whole
#define NG_MEM 64     // group members per work item
#define NG_CHUNK 64   // candidates tested at a time (two per lane)
// slots kept over from one frontier chunk plus those one chunk can add
#define NG_RAW (NG_CHUNK + NB_WARP * NG_RUN)

__device__ __forceinline__ double pair_d2(const double *a, const double *b)
{
    const double dx = __dsub_rn(b[0], a[0]), dy = __dsub_rn(b[1], a[1]), dz = __dsub_rn(b[2], a[2]);
    return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

struct NeighWarp {
    int32_t qa[NG_SMEM], qb[NG_SMEM];
    float4 mem[NG_MEM];       // the item's members, group-relative
    int32_t raw[NG_RAW];      // sorted slots the walk reached
    int32_t cand[2 * NG_CHUNK];   // those near the group's box: the candidates
};

// The band of FP32 squared distances that does not decide |d| <= h: at most
// lo2 is a neighbour, above hi2 is not.  With R = the members' extent about
// the group's centre plus h, a coordinate nb_rel(hi, lo, c) of a member, or
// of any candidate within about h of one, is off by at most 2^-23 1.01 R +
// 2^-47 X (X: the largest coordinate), so a distance is off by at most
// sqrt(3) (2 (2^-23 1.01 R + 2^-47 X) + 2^-24 R) < 5.3e-7 R + 2.5e-14 X; E
// allows about eight times that.  The squares add 3 roundings (2e-7 of the
// square, 1e-6 allowed).  Outside the range where FP32 squares are normal,
// and for non-finite boxes, every pair is left to FP64.
__device__ __forceinline__ void neigh_band(const float4 &lo, const float4 &hi, const float4 &c,
                                           double h, float *lo2, float *hi2)
{
    const float r = fmaxf(fmaxf(fmaxf(hi.x - c.x, c.x - lo.x), fmaxf(hi.y - c.y, c.y - lo.y)),
                          fmaxf(hi.z - c.z, c.z - lo.z));
    const float hf = (float)h;
    const float X = fmaxf(fmaxf(fabsf(c.x), fabsf(c.y)), fabsf(c.z)) + r + hf;
    const float E = 4e-6f * (r + hf) + 1e-12f * X;
    const float up = hf + E, dn = hf - E;
    float u = up * up * 1.000001f, d = dn > 0.0f ? dn * dn * 0.999999f : -1.0f;
    if (!(u >= 1e-30f && u <= 1e30f)) {   // (NaN included)
        u = INFINITY;
        d = -1.0f;
    }
    if (d < 1e-30f) d = -1.0f;
    *lo2 = d;
    *hi2 = u;
}

// One chunk of at most 64 candidates (slots cand[0 .. nc)) against the item's
// mt members.  cur0 / cur1: lane t's running value for members t and t + 32
// (their counts, or in the fill pass their write positions).
template <bool FILL>
__device__ __forceinline__ void neigh_chunk(const NeighWarp &W, const int32_t *cand, int32_t nc,
                                            int32_t f0, int32_t mt, const float4 &bc, float lo2,
                                            float hi2, double h2, const float4 *__restrict__ p_hi,
                                            const float4 *__restrict__ p_lo,
                                            const double *__restrict__ x64,
                                            const int32_t *__restrict__ perm,
                                            int32_t *__restrict__ idx, int64_t cap, int lane,
                                            unsigned lt, int32_t &cur0, int32_t &cur1,
                                            unsigned &bad)
{
    const unsigned FULL = 0xffffffffu;
    int32_t s[2], j[2] = {0, 0};
    float x[2], y[2], z[2];
    unsigned v[2];
#pragma unroll
    for (int q = 0; q < 2; q++) {
        const int32_t e = q * NB_WARP + lane;
        v[q] = __ballot_sync(FULL, e < nc);
        s[q] = cand[e < nc ? e : 0];
        const float4 h = p_hi[s[q]], l = p_lo[s[q]];
        x[q] = nb_rel(h.x, l.x, bc.x);
        y[q] = nb_rel(h.y, l.y, bc.y);
        z[q] = nb_rel(h.z, l.z, bc.z);
        if (FILL) j[q] = perm[s[q]];
    }
#pragma unroll 2
    for (int32_t t = 0; t < mt; t++) {
        const float4 m = W.mem[t];
        bool hit[2], in[2];
#pragma unroll
        for (int q = 0; q < 2; q++) {
            const float dx = x[q] - m.x, dy = y[q] - m.y, dz = z[q] - m.z;
            const float d2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
            hit[q] = !(d2 > hi2);
            in[q] = d2 <= lo2;
        }
        unsigned hm0 = __ballot_sync(FULL, hit[0]) & v[0];
        unsigned hm1 = __ballot_sync(FULL, hit[1]) & v[1];
        if (!(hm0 | hm1)) continue;
        if (__any_sync(FULL, (hit[0] && !in[0]) || (hit[1] && !in[1]))) {
            const int64_t ts = f0 + t;
            const double xi[3] = {x64[3 * ts], x64[3 * ts + 1], x64[3 * ts + 2]};
#pragma unroll
            for (int q = 0; q < 2; q++)
                if (hit[q] && !in[q]) {
                    const int64_t cs = s[q];
                    const double xc[3] = {x64[3 * cs], x64[3 * cs + 1], x64[3 * cs + 2]};
                    hit[q] = pair_d2(xi, xc) <= h2;
                }
            hm0 = __ballot_sync(FULL, hit[0]) & v[0];
            hm1 = __ballot_sync(FULL, hit[1]) & v[1];
        }
        if (FILL) {
            // a particle is not its own neighbour
            const unsigned w0 = hm0 & ~__ballot_sync(FULL, s[0] == f0 + t);
            const unsigned w1 = hm1 & ~__ballot_sync(FULL, s[1] == f0 + t);
            const int32_t base = __shfl_sync(FULL, t < NB_WARP ? cur0 : cur1, t & 31);
            const int32_t n0 = __popc(w0);
            if ((w0 >> lane) & 1u) {
                const int64_t pos = (int64_t)base + __popc(w0 & lt);
                if (pos >= 0 && pos < cap) idx[pos] = j[0];
                else bad |= NB_EF_BOUNDS;
            }
            if ((w1 >> lane) & 1u) {
                const int64_t pos = (int64_t)base + n0 + __popc(w1 & lt);
                if (pos >= 0 && pos < cap) idx[pos] = j[1];
                else bad |= NB_EF_BOUNDS;
            }
            if (lane == (t & 31)) {
                if (t < NB_WARP) cur0 += n0 + __popc(w1);
                else cur1 += n0 + __popc(w1);
            }
        } else if (lane == (t & 31)) {
            if (t < NB_WARP) cur0 += __popc(hm0) + __popc(hm1);
            else cur1 += __popc(hm0) + __popc(hm1);
        }
    }
}

// The slots raw[0 .. nr) (at most 64) that lie within reach of the group's
// box, appended to the candidates; returns their new number.
__device__ __forceinline__ int32_t neigh_near(NeighWarp &W, const int32_t *raw, int32_t nr,
                                              int32_t nc, const float4 &blo, const float4 &bhi,
                                              float reach, const float4 *__restrict__ p_hi,
                                              int lane, unsigned lt)
{
    const unsigned FULL = 0xffffffffu;
    int32_t s[2];
    bool keep[2];
#pragma unroll
    for (int q = 0; q < 2; q++) {
        const int32_t e = q * NB_WARP + lane;
        s[q] = raw[e < nr ? e : 0];
        keep[q] = e < nr && !far_enough(p_hi[s[q]], reach, 0.0f, blo, bhi, 1.0f);
    }
    const unsigned m0 = __ballot_sync(FULL, keep[0]), m1 = __ballot_sync(FULL, keep[1]);
    const int32_t n0 = __popc(m0);
    if (keep[0]) W.cand[nc + __popc(m0 & lt)] = s[0];
    if (keep[1]) W.cand[nc + n0 + __popc(m1 & lt)] = s[1];
    __syncwarp();
    return nc + n0 + __popc(m1);
}

// FILL false: count[perm[slot]] = neighbours; FILL true: write them at
// off[i] ...  One warp per work item: the force items that start at a
// multiple of 64 members give every group's runs of 64 members.
template <bool FILL>
__global__ void __launch_bounds__(NG_T, 4)
k_neigh(const nb_wrec *__restrict__ wrec, const int32_t *__restrict__ items,
        const int32_t *__restrict__ gfirst, const int32_t *__restrict__ gcount,
        const float4 *__restrict__ gbox, const int32_t *__restrict__ n_first,
        const int32_t *__restrict__ n_count, const int32_t *__restrict__ perm,
        const float4 *__restrict__ p_hi, const float4 *__restrict__ p_lo,
        const double *__restrict__ x64, long long *__restrict__ cnt, double h, double h2,
        const double *__restrict__ roots, int32_t *__restrict__ count,
        const int32_t *__restrict__ off, int32_t *__restrict__ idx, int64_t cap,
        int32_t *__restrict__ wq, int64_t wq_cap, int64_t n, int64_t max_items,
        const int32_t *__restrict__ sys_sorted, const int32_t *__restrict__ sys_root,
        unsigned *__restrict__ err)
{
    nb_grid_wait();
    const unsigned FULL = 0xffffffffu;
    __shared__ __align__(16) NeighWarp sw[NG_WARPS];
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int64_t gw = (int64_t)blockIdx.x * NG_WARPS + (threadIdx.x >> 5);
    NeighWarp &W = sw[threadIdx.x >> 5];
    int32_t *const qa = wq + gw * 2 * wq_cap;
    int32_t *const qb = qa + wq_cap;
    const int32_t G = (int32_t)cnt[CNT_GROUPS];
    const int32_t total = (int32_t)cnt[CNT_NODES];
    const int64_t nitems = cnt[CNT_ITEMS] < max_items ? cnt[CNT_ITEMS] : max_items;
    unsigned bad = 0;
    int32_t qmax = 0;
    for (;;) {
        long long it = 0;
        if (lane == 0) it = nb_atomic_add(&cnt[CNT_WALK_Q], 1LL);
        it = __shfl_sync(FULL, it, 0);
        if (it >= nitems) break;
        const int32_t g = items[2 * it], i0 = items[2 * it + 1] & ((1 << 27) - 1);
        if (i0 % NG_MEM) continue;   // the second half of a run of 64 members
        if (!nb_in(g >= 0 && g < G, cnt, err, SITE_GROUPS, g)) continue;
        const float4 blo = gbox[3 * (int64_t)g], bhi = gbox[3 * (int64_t)g + 1],
                     bc = gbox[3 * (int64_t)g + 2];
        const int32_t f = gfirst[g], ng = gcount[g];
        if (!nb_in(f >= 0 && ng >= 1 && (int64_t)f + ng <= n && i0 < ng, cnt, err, SITE_GROUPS, g))
            continue;
        const int32_t f0 = f + i0, mt = ng - i0 < NG_MEM ? ng - i0 : NG_MEM;
        const int32_t gsys = sys_sorted ? sys_sorted[f] : 0;
        float lo2, hi2;
        neigh_band(blo, bhi, bc, h, &lo2, &hi2);
        const float X = fmaxf(fmaxf(fmaxf(fabsf(blo.x), fabsf(bhi.x)),
                                    fmaxf(fabsf(blo.y), fabsf(bhi.y))),
                              fmaxf(fabsf(blo.z), fabsf(bhi.z)));
        const float reach = (float)(h + 1e-5 * roots[8 * (int64_t)gsys + 3]) +
                            1e-6f * (X + (float)h);
        __syncwarp();
        for (int32_t t = lane; t < mt; t += NB_WARP) {
            const float4 hh = p_hi[f0 + t], l = p_lo[f0 + t];
            W.mem[t] = make_float4(nb_rel(hh.x, l.x, bc.x), nb_rel(hh.y, l.y, bc.y),
                                   nb_rel(hh.z, l.z, bc.z), 0.0f);
        }
        int32_t cur0 = 0, cur1 = 0;
        const int32_t t0 = lane < mt ? perm[f0 + lane] : -1;
        const int32_t t1 = NB_WARP + lane < mt ? perm[f0 + NB_WARP + lane] : -1;
        if (FILL) {
            if (t0 >= 0) cur0 = off[t0];
            if (t1 >= 0) cur1 = off[t1];
        }
        int32_t *qin = qa, *qout = qb, *qin_s = W.qa, *qout_s = W.qb;
        if (lane == 0) qin_s[0] = sys_root ? sys_root[gsys] : 0;
        __syncwarp();
        int32_t na = 1, nr = 0, nc = 0;
        auto chunk = [&](int32_t from, int32_t m) {
            neigh_chunk<FILL>(W, W.cand + from, m, f0, mt, bc, lo2, hi2, h2, p_hi, p_lo, x64, perm,
                              idx, cap, lane, lt, cur0, cur1, bad);
            __syncwarp();
        };
        int depth_guard = 0;
        while (na > 0) {
            int32_t nb = 0;
            for (int32_t e0 = 0; e0 < na; e0 += NB_WARP) {
                const int32_t e = e0 + lane;
                int32_t b = 0;
                if (e < na) b = e < NG_SMEM ? qin_s[e] : qin[e];
                int32_t fc = 0, nch = 0, first = 0, take = 0;
                if (e < na && nb_in(b >= 0 && b < total, cnt, err, SITE_WALK_NODE, b)) {
                    const nb_wrec *w = wrec + b;
                    const int4 wb = w->b;
                    const float4 a = w->a;
                    const float2 wc = w->c;
                    const int32_t u = wb.x;
                    // (a leaf's record has l = s = 0: its particle is tested alone)
                    const float r = reach + wc.y + 0.8660254f * wc.x;
                    if (!far_enough(a, r, 0.0f, blo, bhi, 1.0f) &&
                        nb_in(u >= 0 && u < total, cnt, err, SITE_WALK_NODE, u)) {
                        first = n_first[u];
                        take = n_count[u];
                        if (!nb_in(first >= 0 && take >= 1 && (int64_t)first + take <= n, cnt, err,
                                   SITE_WALK_NODE, first)) {
                            take = 0;
                        } else if (take > NG_RUN) {
                            take = 0;
                            fc = wb.z;
                            if (nb_in(fc > b && (int64_t)fc + wb.w <= total, cnt, err,
                                      SITE_WALK_CHILD, b))
                                nch = wb.w;
                        }
                    }
                }
                // runs of slots into the buffer
                int32_t excl = 0;
#pragma unroll
                for (int q = 0; q < 4; q++)
                    excl += __popc(__ballot_sync(FULL, (take >> q) & 1) & lt) << q;
                const int32_t got = __reduce_add_sync(FULL, take);
#pragma unroll
                for (int k = 0; k < NG_RUN; k++)
                    if (k < take) W.raw[nr + excl + k] = first + k;
                nr += got;
                __syncwarp();
                while (nr >= NG_CHUNK) {
                    nr -= NG_CHUNK;
                    nc = neigh_near(W, W.raw + nr, NG_CHUNK, nc, blo, bhi, reach, p_hi, lane, lt);
                    if (nc >= NG_CHUNK) {
                        nc -= NG_CHUNK;
                        chunk(nc, NG_CHUNK);
                    }
                }
                __syncwarp();
                // children of opened cells to the next level's queue
                int32_t ex = 0;
                const int32_t tot = __reduce_add_sync(FULL, nch);
                if (tot == 0) continue;
                if (__any_sync(FULL, nch > 15)) {
                    int32_t incl = nch;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int32_t y = __shfl_up_sync(FULL, incl, o);
                        if (lane >= o) incl += y;
                    }
                    ex = incl - nch;
                } else {
#pragma unroll
                    for (int q = 0; q < 4; q++)
                        ex += __popc(__ballot_sync(FULL, (nch >> q) & 1) & lt) << q;
                }
                const int32_t start = nb + ex;
                for (int32_t k = 0; k < nch; k++) {
                    const int32_t pos = start + k;
                    if (pos < NG_SMEM) qout_s[pos] = fc + k;
                    else if (pos < wq_cap) qout[pos] = fc + k;
                }
                nb += tot;
            }
            if (nb > qmax) qmax = nb;
            if (nb > wq_cap) { bad |= NB_EF_QUEUE; break; }
            __syncwarp();
            int32_t *t = qin; qin = qout; qout = t;
            t = qin_s; qin_s = qout_s; qout_s = t;
            na = nb;
            if (++depth_guard > NB_DEPTHS + 1) { bad |= NB_EF_WALK; break; }
        }
        if (nr > 0) nc = neigh_near(W, W.raw, nr, nc, blo, bhi, reach, p_hi, lane, lt);
        if (nc > NG_CHUNK) {
            nc -= NG_CHUNK;
            chunk(nc, NG_CHUNK);
        }
        if (nc > 0) chunk(0, nc);
        // every particle found itself once (distance 0)
        if (FILL) {   // each run must end where the next one starts
            if (t0 >= 0 && cur0 != off[t0 + 1]) bad |= NB_EF_BOUNDS;
            if (t1 >= 0 && cur1 != off[t1 + 1]) bad |= NB_EF_BOUNDS;
        } else {
            if (t0 >= 0) count[t0] = cur0 - 1;
            if (t1 >= 0) count[t1] = cur1 - 1;
        }
    }
    bad = __reduce_or_sync(FULL, bad);
    qmax = __reduce_max_sync(FULL, qmax);
    if (lane == 0) {
        atomicMax(&cnt[CNT_QMAX], (long long)qmax);
        if (bad) atomicOr(err, bad);
    }
}

// offsets: off64[i] = off32[i] for i <= n
__global__ void k_neigh_offsets(const int32_t *__restrict__ off32, int64_t n,
                                int64_t *__restrict__ off64)
{
    nb_grid_wait();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i <= n;
         i += (int64_t)gridDim.x * blockDim.x)
        off64[i] = off32[i];
}

// 32 R values (value r 32 + lane in lane's register r) sorted ascending by
// a bitonic network: strides of 32 and more exchange registers of one lane,
// shorter ones go through shuffles
template <int R>
__device__ __forceinline__ void warp_sort(int32_t (&v)[R], int lane)
{
#pragma unroll
    for (int size = 2; size <= 32 * R; size <<= 1)
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            if (stride >= 32) {
#pragma unroll
                for (int r = 0; r < R; r++) {
                    const int q = r ^ (stride >> 5);
                    if (q > r) {
                        const int32_t lo = min(v[r], v[q]), hi = max(v[r], v[q]);
                        const bool up = ((r << 5) & size) == 0;
                        v[r] = up ? lo : hi;
                        v[q] = up ? hi : lo;
                    }
                }
            } else {
#pragma unroll
                for (int r = 0; r < R; r++) {
                    const int32_t o = __shfl_xor_sync(0xffffffffu, v[r], stride);
                    const bool up = (((r << 5) | lane) & size) == 0;
                    v[r] = ((lane & stride) == 0) == up ? min(v[r], o) : max(v[r], o);
                }
            }
        }
}

template <int R>
__device__ __forceinline__ void sort_run(int32_t *a, int32_t len, int lane)
{
    int32_t v[R];
#pragma unroll
    for (int r = 0; r < R; r++) {
        const int32_t e = r * 32 + lane;
        v[r] = e < len ? a[e] : INT_MAX;
    }
    warp_sort<R>(v, lane);
#pragma unroll
    for (int r = 0; r < R; r++) {
        const int32_t e = r * 32 + lane;
        if (e < len) a[e] = v[r];
    }
}

// every target's run sorted ascending in place, one warp per target: up to
// 256 entries in registers (the smallest of 1, 2, 4 or 8 per lane that holds
// the run), longer runs by Batcher's odd-even merge sort over the next power
// of two in memory, whose comparators all put the smaller value first, so
// slots past the run act as +infinity and are never touched.  Bound by the
// shuffles of the network (21 of them per register for 64 entries); with
// every run sorted in memory the pass over 300,000 runs of 48 took 0.54 ms
// (0.09 ms so).
__global__ void __launch_bounds__(256)
k_neigh_sort(const int32_t *__restrict__ off, int64_t n, int32_t *__restrict__ idx)
{
    nb_grid_wait();
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t i = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); i < n;
         i += warps) {
        int32_t *a = idx + off[i];
        const int32_t len = off[i + 1] - off[i];
        if (len <= 1) continue;
        if (len <= 32) { sort_run<1>(a, len, lane); continue; }
        if (len <= 64) { sort_run<2>(a, len, lane); continue; }
        if (len <= 128) { sort_run<4>(a, len, lane); continue; }
        if (len <= 256) { sort_run<8>(a, len, lane); continue; }
        int32_t P = 1;
        while (P < len) P <<= 1;
        for (int32_t p = 1; p < P; p <<= 1)
            for (int32_t k = p; k >= 1; k >>= 1) {
                // comparators (i + j, i + j + k) for j = k % p, k % p + 2k, ...
                // and i < k, inside one block of 2p
                const int32_t j0 = k % p;
                const int32_t pairs = ((P - k - j0 + 2 * k - 1) / (2 * k)) * k;
                for (int32_t e = lane; e < pairs; e += 32) {
                    const int32_t x = j0 + (e / k) * 2 * k + e % k;
                    const int32_t y = x + k;
                    if (y >= len || x / (2 * p) != y / (2 * p)) continue;
                    const int32_t u = a[x], v = a[y];
                    if (u > v) {
                        a[x] = v;
                        a[y] = u;
                    }
                }
                __syncwarp();
            }
    }
}

// the walk of both passes; returns the error bits (synchronised)
static int neigh_pass(nb_ctx *c, bool fill, double h, int32_t *idx, int64_t cap, unsigned *bits)
{
    CK_RET(cudaMemsetAsync(&c->cnt[CNT_WALK_Q], 0, sizeof(long long), c->stream));
    CK_RET(cudaMemsetAsync(&c->cnt[CNT_QMAX], 0, sizeof(long long), c->stream));
    const int blocks = c->walk_warps / NG_WARPS;
    const int32_t *ss = c->nsys > 1 ? c->sys_sorted : nullptr;
    const int32_t *sr = c->nsys > 1 ? c->sys_root : nullptr;
    if (fill)
        nb_launch(k_neigh<true>, blocks, NG_T, 0, nb_queue(c), c->wrec, c->items, c->gfirst,
                  c->gcount, c->gbox, c->n_first, c->n_count, c->perm, c->p_hi, c->p_lo, c->p_x64,
                  c->cnt, h, h * h, c->root, c->ccount, c->cstart, idx, cap, c->wq, c->wq_cap,
                  c->n, c->max_items, ss, sr, c->err);
    else
        nb_launch(k_neigh<false>, blocks, NG_T, 0, nb_queue(c), c->wrec, c->items, c->gfirst,
                  c->gcount, c->gbox, c->n_first, c->n_count, c->perm, c->p_hi, c->p_lo, c->p_x64,
                  c->cnt, h, h * h, c->root, c->ccount, nullptr, nullptr, 0, c->wq, c->wq_cap,
                  c->n, c->max_items, ss, sr, c->err);
    nb_launched(c, "k_neigh");
    return nb_read_err(c, bits);
}

int nb_neigh_run(nb_ctx *c, double h, int n_crit, int64_t *off, int32_t *idx, int64_t cap,
                 int64_t *total)
{
    const int64_t n = c->n;
    nb_launch_groups(c, 1.0f, n_crit, nullptr);
    for (int attempt = 0; attempt < 4; attempt++) {
        CK_RET(cudaMemsetAsync(c->ccount, 0, sizeof(int32_t) * (size_t)(n + 1), c->stream));
        unsigned bits = 0;
        int rc = neigh_pass(c, false, h, nullptr, 0, &bits);
        if (rc) return rc;
        if (bits & NB_EF_QUEUE) {   // a frontier outgrew the queues: grow them, walk again
            rc = nb_grow_queues(c);
            if (rc) return rc;
            continue;
        }
        if (bits) return nb_err_code(bits);
        // offsets in caller order (the count array is in caller order)
        nb_exclusive_scan(c, c->ccount, c->cstart, n + 1, nullptr, &c->cnt[CNT_LIST_TOT]);
        nb_launch(k_neigh_offsets, nb_grid(n + 1, 256, c->num_sms * 8), 256, 0, nb_queue(c),
                  c->cstart, n, off);
        nb_launched(c, "k_neigh_offsets");
        long long tot = 0;
        CK_RET(cudaMemcpyAsync(&tot, &c->cnt[CNT_LIST_TOT], sizeof(long long),
                               cudaMemcpyDeviceToHost, c->stream));
        CK_RET(cudaStreamSynchronize(c->stream));
        *total = tot;
        if (tot >= INT32_MAX) return NB_ERR_CAPACITY;
        if (!idx || cap < tot) return NB_OK;   // counts and offsets only
        rc = neigh_pass(c, true, h, idx, cap, &bits);
        if (rc) return rc;
        if (bits) return bits & NB_EF_BOUNDS ? NB_ERR_INTERNAL : nb_err_code(bits);
        nb_launch(k_neigh_sort, c->num_sms * 8, 256, 0, nb_queue(c), c->cstart, n, idx);
        nb_launched(c, "k_neigh_sort");
        CK_RET(cudaStreamSynchronize(c->stream));
        return cudaGetLastError() == cudaSuccess ? NB_OK : NB_ERR_CUDA;
    }
    return NB_ERR_CAPACITY;
}
