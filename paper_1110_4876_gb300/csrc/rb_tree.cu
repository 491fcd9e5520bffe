// rb_tree.cu -- the octree of Sect. 4.2 built from Morton-sorted particles,
// its cell moments and the records the walks read.
//
// Cells are the key prefixes (3 bits per depth) shared by two or more
// particles that split at the next depth (or sit at the depth cap of 21,
// where they are leaf groups).  Cells with a single occupied octant are
// skipped: they hold the same particles, centre of mass and quadrupole as
// that octant and a wider cell is never accepted where the narrower one is
// not, so the forces equal those of the paper's insertion tree.
//
// Between sorted particles i and i+1 ("split" i) the shared prefix depth is
// delta_i.  A cell of depth v is a maximal run of splits with delta >= v that
// contains a split with delta == v; its first such split is its
// representative.  Range minima of delta come straight from the keys
// (clz of the xor of the run's end keys), so each split finds its run with a
// galloping search.  Cells are laid out in depth-first pre-order together
// with one leaf entry per particle: entry order is (first particle, depth),
// and a per-particle bitmask of the depths of cells starting there gives
// every entry's position after one scan.
#include <algorithm>
#include <cfloat>

#include "rb_fp64.cuh"
#include "rb_internal.cuh"

namespace rb {
namespace {

template <bool kMultiBox>
__device__ __forceinline__ int lcp_level(const uint64_t* __restrict__ key,
                                         const int32_t* __restrict__ box, int a, int b) {
    if (kMultiBox && box[a] != box[b]) return -1;
    const uint64_t x = key[a] ^ key[b];
    if (x == 0ull) return kMaxDepth;
    return (__clzll((long long)x) - 1) / 3;
}

// One thread per split i in [0, n - 2]: find the run of cell depth
// v = delta_i; if i represents its cell, record the particle range and mark
// the cell's depth in mask[first].
template <bool kMultiBox>
__global__ void __launch_bounds__(256) k_nodes(const uint64_t* __restrict__ key,
                                               const int32_t* __restrict__ box, Ctl* ctl, int ncap,
                                               int32_t* __restrict__ node_a,
                                               int32_t* __restrict__ node_b,
                                               int8_t* __restrict__ node_v,
                                               uint32_t* __restrict__ mask) {
    const int n = sorted_n(ctl, ncap);
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) ctl->n_live_next = 0;   // committed by the gather
    if (i >= n - 1) return;
    const int v = lcp_level<kMultiBox>(key, box, i, i + 1);
    int8_t outv = -1;
    if (v >= 0) {
        // leftmost particle a with min(delta_a .. delta_i) >= v
        int good = i, step = 1, bad = -1;
        for (;;) {
            const int c = i - step;
            if (c < 0) { bad = -1; break; }
            if (lcp_level<kMultiBox>(key, box, c, i + 1) < v) { bad = c; break; }
            good = c;
            step <<= 1;
        }
        while (good - bad > 1) {
            const int mid = (good + bad) >> 1;
            if (lcp_level<kMultiBox>(key, box, mid, i + 1) >= v) good = mid; else bad = mid;
        }
        const int a = good;
        const bool rep = (a == i) || (lcp_level<kMultiBox>(key, box, a, i) > v);
        node_a[i] = a;
        outv = (int8_t)(v + 32);   // the split's cell; its representative is another split
        if (rep) {
            // rightmost particle b with min(delta_i .. delta_{b-1}) >= v
            int g2 = i + 1, st = 1, b2 = n;
            for (;;) {
                const int c = i + 1 + st;
                if (c >= n) { b2 = n; break; }
                if (lcp_level<kMultiBox>(key, box, i, c) < v) { b2 = c; break; }
                g2 = c;
                st <<= 1;
            }
            while (b2 - g2 > 1) {
                const int mid = (g2 + b2) >> 1;
                if (lcp_level<kMultiBox>(key, box, i, mid) >= v) g2 = mid; else b2 = mid;
            }
            node_b[i] = g2;
            outv = (int8_t)v;
            atomicOr(&mask[a], 1u << v);
        }
    }
    node_v[i] = outv;
}

// First entry starting at each particle: the exclusive scan of 1 + (cells
// starting there), start[n] and n_entries the total.  One launch: a block scans
// a tile of 2048 particles and finds the total of the earlier tiles by a
// decoupled look-back over one status word per tile (zero on entry; flag and
// count in one word, as in the radix passes, whose argument that every wait
// ends holds here too; bounded by half a second all the same).
constexpr int kScanTile = 2048;
constexpr uint32_t kScanAgg = 1u << 30, kScanPre = 2u << 30, kScanMask = (1u << 30) - 1u;

__global__ void __launch_bounds__(256) k_entry_scan(const uint32_t* __restrict__ mask, Ctl* ctl, int ncap,
                                                    int32_t* __restrict__ start, uint32_t* stat, bool hold) {
    __shared__ uint32_t ws[8], before_s;
    const int n = sorted_n(ctl, ncap);
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int base = b * kScanTile;
    if (base >= n) {
        if (b == 0 && tid == 0) {
            start[0] = 0;
            ctl->n_entries = 0;
        }
        return;
    }
    const int t0 = base + tid * 8;
    uint32_t v[8], s = 0;
#pragma unroll
    for (int r = 0; r < 8; r++) {
        v[r] = t0 + r < n ? 1u + __popc(mask[t0 + r]) : 0u;
        s += v[r];
    }
    uint32_t x = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += t;
    }
    if (lane == 31) ws[warp] = x;
    __syncthreads();
    uint32_t in = x - s, total = 0;   // counts before this thread within the tile
#pragma unroll
    for (int w = 0; w < 8; w++) {
        if (w < warp) in += ws[w];
        total += ws[w];
    }
    volatile uint32_t* st = stat;
    if (tid == 0 && (!hold || b > 0)) st[b] = (b == 0 ? kScanPre : kScanAgg) | total;
    if (warp == 0) {
        uint32_t excl = 0;
        unsigned long long since = 0;
        for (int j = b - 1; j >= 0;) {
            // the 32 nearest tiles not yet counted, down to the first prefix
            uint32_t w = kScanPre;
            if (j - lane >= 0) w = st[j - lane];
            const unsigned pre = __ballot_sync(0xffffffffu, w & kScanPre);
            const unsigned none = __ballot_sync(0xffffffffu, (w & (kScanPre | kScanAgg)) == 0u);
            const unsigned need = pre ? (2u << (__ffs(pre) - 1)) - 1u : 0xffffffffu;
            if (none & need) {
                unsigned long long now;
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
                if (since == 0) since = now;
                const bool give_up = (*(volatile int*)&ctl->err & kErrSortStall) || now - since > 500000000ull;
                if (__any_sync(0xffffffffu, give_up)) {
                    if (lane == 0) atomicOr(&ctl->err, kErrSortStall);
                    break;
                }
                continue;
            }
            excl += __reduce_add_sync(0xffffffffu, (need >> lane) & 1u ? w & kScanMask : 0u);
            if (pre) break;
            j -= 32;
        }
        if (lane == 0) {
            if (b > 0) st[b] = kScanPre | ((excl + total) & kScanMask);
            before_s = excl;
        }
    }
    __syncthreads();
    uint32_t run = before_s + in;
#pragma unroll
    for (int r = 0; r < 8; r++) {
        if (t0 + r < n) start[t0 + r] = (int32_t)run;
        run += v[r];
    }
    if (tid == 0 && base + kScanTile >= n) {
        start[n] = (int32_t)(before_s + total);
        ctl->n_entries = (int32_t)(before_s + total);
    }
}

// Entries in pre-order: cells (from their representative split) and leaves.
__global__ void __launch_bounds__(256) k_emit(const uint32_t* __restrict__ mask,
                                              const int32_t* __restrict__ start,
                                              const int32_t* __restrict__ node_a,
                                              const int32_t* __restrict__ node_b,
                                              const int8_t* __restrict__ node_v,
                                              const Ctl* __restrict__ ctl, int ncap,
                                              int32_t* __restrict__ e_first,
                                              int32_t* __restrict__ e_count,
                                              int32_t* __restrict__ e_skip,
                                              int8_t* __restrict__ e_level,
                                              int32_t* __restrict__ leaf_of,
                                              const uint64_t* __restrict__ key,
                                              int32_t* __restrict__ e_child,
                                              uint32_t* __restrict__ e_cmask,
                                              const int32_t* __restrict__ box,
                                              int32_t* __restrict__ box_root) {
    const int n = sorted_n(ctl, ncap);
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    // the root of a box starts at its first particle; the others stay -1
    // (empty boxes, and entry nbox, the box of particles that an open boundary
    // removed: those still hold slots of the gravity tree when the step's
    // collision search runs on it, and search nothing)
    if (i == 0 || box[i] != box[i - 1]) box_root[box[i]] = start[i];
    const uint32_t mk = mask[i];
    const int li = start[i] + __popc(mk);
    e_first[li] = i;
    e_count[li] = 1;
    e_skip[li] = li + 1;
    e_level[li] = 22;
    leaf_of[i] = li;
    if (i < n - 1) {
        const int vv = node_v[i];
        if (vv >= 0) {
            const int v = vv & 31;
            const int a = node_a[i];
            const int idx = start[a] + __popc(mask[a] & ((1u << v) - 1u));   // the split's cell
            if (vv < 32) {
                const int b = node_b[i];
                e_first[idx] = a;
                e_count[idx] = b - a + 1;
                e_skip[idx] = start[b + 1];
                e_level[idx] = (int8_t)v;
            }
            // child table (not for depth-21 groups, whose members share one key):
            // particles i and i + 1 part at depth v + 1, so the child of cell idx
            // that starts at particle i + 1 is its shallowest entry there; the
            // representative also enters the first child, entry idx + 1
            if (v < kMaxDepth) {
                const int sh = 3 * (kMaxDepth - 1 - v);
                const int o = (int)((key[i + 1] >> sh) & 7ull);
                e_child[8 * (size_t)idx + o] = start[i + 1];
                atomicOr(&e_cmask[idx], 1u << o);
                if (vv < 32) {
                    const int o0 = (int)((key[a] >> sh) & 7ull);
                    e_child[8 * (size_t)idx + o0] = idx + 1;
                    atomicOr(&e_cmask[idx], 1u << o0);
                }
            }
        }
    }
}

__device__ __forceinline__ uint32_t compact3(uint64_t x) {
    x &= 0x1249249249249249ull;
    x = (x ^ (x >> 2)) & 0x10c30c30c30c30c3ull;
    x = (x ^ (x >> 4)) & 0x100f00f00f00f00full;
    x = (x ^ (x >> 8)) & 0x1f0000ff0000ffull;
    x = (x ^ (x >> 16)) & 0x1f00000000ffffull;
    x = (x ^ (x >> 32)) & 0x1fffffull;
    return (uint32_t)x;
}

__device__ __forceinline__ void split_hilo(double v, float& hi, float& lo) {
    hi = __double2float_rn(v);
    lo = __double2float_rn(v - (double)hi);
}

// Integer cell index of depth v along each axis, from a member's key.
__device__ __forceinline__ void cell_index(uint64_t key, int v, double& ix, double& iy, double& iz) {
    const int sh = kMaxDepth - v;
    ix = (double)(compact3(key >> 2) >> sh);
    iy = (double)(compact3(key >> 1) >> sh);
    iz = (double)(compact3(key) >> sh);
}

struct GravRecArgs {
    const double *x, *y, *z, *m;
    const int32_t *box, *id;
    bool has_test;   // some particles are test particles (source mass 0)
    bool one;        // a single box
    const uint64_t* key;
    const BoxP* boxes;
    const int32_t *e_first, *e_skip, *e_child, *leaf_of;
    const uint32_t* e_cmask;
    const int8_t* e_level;
    const int32_t *e_count, *start;
    int piece0;      // first record behind the tree's entries
    double4_32a *d_a, *d_q0, *d_q1, *d_c;
    Rec4 ra, rb, rq0, rq1, rc_hi, rc_lo;
    const Ctl* ctl;
    int ncap;
    double crit_scale;  // 1 / theta^2
    bool leafq;         // leaves get FP32 multipole records (mass, Q = 0)
    bool q32;           // FP32 quadrupole records are read too (not by the FP64 walk)
    bool corners;       // cell corners are read (inside test, network inputs)
};

// Leaf record (FP64 and FP32) of particle p.
__device__ __forceinline__ void leaf_record(const GravRecArgs& A, int p) {
    const int e = A.leaf_of[p];
    const double x = A.x[p], y = A.y[p], z = A.z[p];
    const double m = A.has_test ? source_mass(A.boxes[A.box[p]], A.id[p], A.m[p]) : A.m[p];
    A.d_a[e] = make_double4_32a(x, y, z, -m);
    float hx, lx, hy, ly, hz, lz;
    split_hilo(x, hx, lx);
    split_hilo(y, hy, ly);
    split_hilo(z, hz, lz);
    A.ra[e] = make_float4(hx, hy, hz, lz);
    A.rb[e] = make_float4(lx, ly, -(float)m, __int_as_float(e + 1));
    if (A.leafq) {
        A.rq0[e] = make_float4((float)m, 0.f, 0.f, 0.f);
        A.rq1[e] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// A cell's moments come from its children (cells done before it, or particle
// leaves) in one pass: about the first child's position o, M = sum M_c,
// S = sum M_c d_c and Q_o = sum [Q_c + M_c (3 d_c d_c^T - |d_c|^2 I)],
// d_c = com_c - o; then the centre of mass is o + S / M and the parallel-axis
// theorem moves Q_o to it: Q = Q_o - M (3 s s^T - |s|^2 I), s = S / M (the
// traceless quadrupole about the centre of mass, reading R3).  Every |d_c| and
// |s| is below the cell's diagonal, so no term is much larger than the result.
// kF32Q: the quadrupole is only needed by the FP32 walk, so it is summed in
// FP32 on the hi/lo records (d_c good to ~1e-7 relative); mass and centre of
// mass stay FP64.  On GB300 FP64 instructions cost 64 times FP32 ones.
// Running sums of one cell's moments about its first child's position o.
struct MomSums {
    double M, sx, sy, sz;   // mass and sum of M_c d_c (FP64)
    double q[6];            // quadrupole about o (FP64 form)
    float qf[6];            // quadrupole about o (FP32 form)
};

__device__ __forceinline__ void mom_zero(MomSums& S) {
    S.M = S.sx = S.sy = S.sz = 0.0;
#pragma unroll
    for (int j = 0; j < 6; j++) {
        S.q[j] = 0.0;
        S.qf[j] = 0.f;
    }
}

// Adds child entry c (a particle leaf or a finished deeper cell).
template <bool kF32Q>
__device__ __forceinline__ void mom_add(const GravRecArgs& A, int c, double ox, double oy, double oz,
                                        float4 h0, float4 l0, MomSums& S) {
    const double4_32a a = A.d_a[c];
    const bool leaf = __double_as_longlong(a.w) < 0;   // leaf records hold -m (m >= 0)
    const double mc = leaf ? -a.w : A.d_q0[c].x;
    const double dx = a.x - ox, dy = a.y - oy, dz = a.z - oz;
    S.M += mc;
    S.sx = fma(mc, dx, S.sx);
    S.sy = fma(mc, dy, S.sy);
    S.sz = fma(mc, dz, S.sz);
    if (kF32Q) {
        const float4 h = A.ra[c], l = A.rb[c];
        const float fx = (h.x - h0.x) + (l.x - l0.x);
        const float fy = (h.y - h0.y) + (l.y - l0.y);
        const float fz = (h.z - h0.z) + (h.w - h0.w);
        float fm;
        if (leaf) {
            fm = -l.z;
        } else {
            const float4 c0 = A.rq0[c], c1 = A.rq1[c];
            fm = c0.x;
            S.qf[0] += c0.y; S.qf[1] += c0.z; S.qf[2] += c0.w;
            S.qf[3] += c1.x; S.qf[4] += c1.y; S.qf[5] += c1.z;
        }
        const float d2 = fmaf(fz, fz, fmaf(fy, fy, fx * fx));
        const float m3x = 3.f * fm * fx, m3y = 3.f * fm * fy;
        S.qf[0] += fmaf(m3x, fx, -fm * d2);
        S.qf[1] += fmaf(m3y, fy, -fm * d2);
        S.qf[2] += fmaf(3.f * fm * fz, fz, -fm * d2);
        S.qf[3] += m3x * fy;
        S.qf[4] += m3x * fz;
        S.qf[5] += m3y * fz;
    } else {
        if (!leaf) {
            const double4_32a c0 = A.d_q0[c], c1 = A.d_q1[c];
            S.q[0] += c0.y; S.q[1] += c0.z; S.q[2] += c0.w;
            S.q[3] += c1.x; S.q[4] += c1.y; S.q[5] += c1.z;
        }
        const double d2 = dx * dx + dy * dy + dz * dz;
        S.q[0] += mc * (3.0 * dx * dx - d2);
        S.q[1] += mc * (3.0 * dy * dy - d2);
        S.q[2] += mc * (3.0 * dz * dz - d2);
        S.q[3] += mc * (3.0 * dx * dy);
        S.q[4] += mc * (3.0 * dx * dz);
        S.q[5] += mc * (3.0 * dy * dz);
    }
}

// Levels shared by two Morton keys (3 bits a level below the unused top bit).
__device__ __forceinline__ int common_levels(uint64_t a, uint64_t b) {
    const uint64_t x = a ^ b;
    return x ? (__clzll((long long)x) - 1) / 3 : kMaxDepth;
}

// A depth-21 leaf group (members first..last share their key) stands in the
// insertion tree below a run of one-child cells that reaches depth 20 unless
// its parent cell, the deepest one holding another particle of the box, is
// at depth 20 itself.  Those one-child cells hold the group's members and
// are opened or accepted like any cell; of them the depth-20 one accepts
// first (narrowest, and the smallest for the inside rule), so the group's
// record carries that cell's width and corner.  Without such a cell the group
// is never accepted.
__device__ __forceinline__ bool group_has_chain(const GravRecArgs& A, int first, int last) {
    const int n = sorted_n(A.ctl, A.ncap);
    const uint64_t kf = A.key[first];
    const int b = A.box[first];
    int d = -1;   // depth of the group's parent cell
    if (first > 0 && A.box[first - 1] == b) d = max(d, common_levels(A.key[first - 1], kf));
    if (last + 1 < n && A.box[last + 1] == b) d = max(d, common_levels(kf, A.key[last + 1]));
    return d < kMaxDepth - 1;
}

// x 2^-v for x with exponent well inside the normal range (v <= 21).
__device__ __forceinline__ double scale_down(double x, int v) {
    return __longlong_as_double(__double_as_longlong(x) - ((long long)v << 52));
}

// Moves the quadrupole from the origin of the sums to the centre of mass at u
// (parallel-axis theorem).
template <bool kF32Q>
__device__ __forceinline__ void mom_shift(MomSums& S, double ux, double uy, double uz) {
    if (kF32Q) {
        const float fx = (float)ux, fy = (float)uy, fz = (float)uz, fm = (float)S.M;
        const float d2 = fmaf(fz, fz, fmaf(fy, fy, fx * fx));
        S.qf[0] -= fm * fmaf(3.f * fx, fx, -d2);
        S.qf[1] -= fm * fmaf(3.f * fy, fy, -d2);
        S.qf[2] -= fm * fmaf(3.f * fz, fz, -d2);
        S.qf[3] -= 3.f * fm * fx * fy;
        S.qf[4] -= 3.f * fm * fx * fz;
        S.qf[5] -= 3.f * fm * fy * fz;
    } else {
        const double d2 = ux * ux + uy * uy + uz * uz;
        S.q[0] -= S.M * (3.0 * ux * ux - d2);
        S.q[1] -= S.M * (3.0 * uy * uy - d2);
        S.q[2] -= S.M * (3.0 * uz * uz - d2);
        S.q[3] -= S.M * (3.0 * ux * uy);
        S.q[4] -= S.M * (3.0 * ux * uz);
        S.q[5] -= S.M * (3.0 * uy * uz);
    }
}

// The cell's centre of mass, its quadrupole moved there, and its records.
// first: its first slot; L: the side of its box's root cube.
template <bool kF32Q>
__device__ __forceinline__ void mom_finish(const GravRecArgs& A, int k, int depth, int end, int first, double L,
                                           double ox, double oy, double oz, MomSums& S) {
    // a leaf group's members are the entries k + 1 .. end - 1
    const bool group = depth == kMaxDepth;
    const bool chain = group && group_has_chain(A, first, first + (end - k - 2));
    const int v = chain ? kMaxDepth - 1 : depth;   // the depth whose cell the record describes
    const double w = scale_down(L, v);
    const double lo = -0.5 * L;
    double ix = 0.0, iy = 0.0, iz = 0.0;
    if (A.corners || !(S.M > 0.0)) cell_index(A.key[first], v, ix, iy, iz);
    double cx, cy, cz, ux, uy, uz;   // centre of mass and its offset from o
    if (S.M > 0.0) {
        const double iM = rcp64(S.M);
        ux = S.sx * iM; uy = S.sy * iM; uz = S.sz * iM;
        cx = ox + ux; cy = oy + uy; cz = oz + uz;
    } else {
        // no source mass (test particles only): the geometric centre
        cx = lo + (ix + 0.5) * w; cy = lo + (iy + 0.5) * w; cz = lo + (iz + 0.5) * w;
        ux = uy = uz = 0.0;
    }
    mom_shift<kF32Q>(S, ux, uy, uz);
    const bool never = group && !chain;   // a leaf group with no one-child cell above it
    const double ww = w * w;
    A.d_a[k] = make_double4_32a(cx, cy, cz, never ? __longlong_as_double(0x7ff0000000000000ll) : ww);
    if (kF32Q) {
        A.d_q0[k].x = S.M;   // the quadrupole is read from the FP32 records
    } else {
        A.d_q0[k] = make_double4_32a(S.M, S.q[0], S.q[1], S.q[2]);
        A.d_q1[k] = make_double4_32a(S.q[3], S.q[4], S.q[5], w);
    }
    double c0x = 0.0, c0y = 0.0, c0z = 0.0;
    if (A.corners) {
        // cell corner lo + i w, rounded as two separate operations
        c0x = __dadd_rn(lo, __dmul_rn(ix, w));
        c0y = __dadd_rn(lo, __dmul_rn(iy, w));
        c0z = __dadd_rn(lo, __dmul_rn(iz, w));
        A.d_c[k] = make_double4_32a(c0x, c0y, c0z, w);
    }
    float hx, lx, hy, ly, hz, lz;
    split_hilo(cx, hx, lx);
    split_hilo(cy, hy, ly);
    split_hilo(cz, hz, lz);
    const float crit = never ? __int_as_float(0x7f800000) : (float)(ww * A.crit_scale);
    A.ra[k] = make_float4(hx, hy, hz, lz);
    A.rb[k] = make_float4(lx, ly, crit, __int_as_float(end));
    if (A.q32) {
        if (kF32Q) {
            A.rq0[k] = make_float4((float)S.M, S.qf[0], S.qf[1], S.qf[2]);
            A.rq1[k] = make_float4(S.qf[3], S.qf[4], S.qf[5], 0.f);
        } else {
            A.rq0[k] = make_float4((float)S.M, (float)S.q[0], (float)S.q[1], (float)S.q[2]);
            A.rq1[k] = make_float4((float)S.q[3], (float)S.q[4], (float)S.q[5], 0.f);
        }
    }
    if (A.corners) {
        split_hilo(c0x, hx, lx);
        split_hilo(c0y, hy, ly);
        split_hilo(c0z, hz, lz);
        A.rc_hi[k] = make_float4(hx, hy, hz, (float)w);
        A.rc_lo[k] = make_float4(lx, ly, lz, 0.f);
    }
}

// Side of the root cube of the box that slot `first` lies in (one box: its
// side, loaded once per block).
__device__ __forceinline__ double root_side(const GravRecArgs& A, int first, double one) {
    return A.one ? one : A.boxes[A.box[first]].L;
}

// Sums of a warp's lanes, in a fixed butterfly order.
template <bool kF32Q>
__device__ __forceinline__ void mom_reduce(MomSums& S, int width) {
    for (int x = 1; x < width; x <<= 1) {
        S.M += __shfl_xor_sync(0xffffffffu, S.M, x);
        S.sx += __shfl_xor_sync(0xffffffffu, S.sx, x);
        S.sy += __shfl_xor_sync(0xffffffffu, S.sy, x);
        S.sz += __shfl_xor_sync(0xffffffffu, S.sz, x);
#pragma unroll
        for (int j = 0; j < 6; j++) {
            if (kF32Q) S.qf[j] += __shfl_xor_sync(0xffffffffu, S.qf[j], x);
            else S.q[j] += __shfl_xor_sync(0xffffffffu, S.q[j], x);
        }
    }
}

// One cell by eight lanes (lane o of 8 takes the child in octant o, which add
// their sums in a fixed butterfly order); groups without a cell (live false)
// join the shuffles.  Not for depth-21 groups, which have no child table.
template <bool kF32Q>
__device__ __forceinline__ void mom_cell_group(const GravRecArgs& A, bool live, int k, int depth, double one) {
    const int o = threadIdx.x & 7;
    MomSums S;
    mom_zero(S);
    double ox = 0.0, oy = 0.0, oz = 0.0, L = 0.0;
    int first = 0, end = 0;
    float4 h0 = make_float4(0.f, 0.f, 0.f, 0.f), l0 = h0;
    if (live) {
        const bool has = (A.e_cmask[k] >> o) & 1u;
        const int child = A.e_child[8 * (size_t)k + o];
        first = A.e_first[k];
        end = A.e_skip[k];
        const double4_32a a0 = A.d_a[k + 1];   // the first child is entry k + 1
        ox = a0.x; oy = a0.y; oz = a0.z;
        if (kF32Q) {
            h0 = A.ra[k + 1];
            l0 = A.rb[k + 1];
        }
        L = root_side(A, first, one);
        if (has) mom_add<kF32Q>(A, child, ox, oy, oz, h0, l0, S);
    }
    mom_reduce<kF32Q>(S, 8);
    if (live && o == 0) mom_finish<kF32Q>(A, k, depth, end, first, L, ox, oy, oz, S);
}

// One cell by one thread, from its children in pre-order.
template <bool kF32Q>
__device__ __forceinline__ void mom_cell(const GravRecArgs& A, int k, int depth, double one) {
    const int end = A.e_skip[k], first = A.e_first[k];
    const double4_32a a0 = A.d_a[k + 1];
    const double ox = a0.x, oy = a0.y, oz = a0.z, L = root_side(A, first, one);
    float4 h0 = make_float4(0.f, 0.f, 0.f, 0.f), l0 = h0;
    if (kF32Q) {
        h0 = A.ra[k + 1];
        l0 = A.rb[k + 1];
    }
    MomSums S;
    mom_zero(S);
    for (int c = k + 1; c < end; c = A.e_skip[c]) mom_add<kF32Q>(A, c, ox, oy, oz, h0, l0, S);
    mom_finish<kF32Q>(A, k, depth, end, first, L, ox, oy, oz, S);
}

// One cell of `count` particles by one thread, straight from their leaves.
template <bool kF32Q>
__device__ __forceinline__ void mom_cell_leaves(const GravRecArgs& A, int k, int count, double one) {
    const int end = A.e_skip[k], first = A.e_first[k], depth = A.e_level[k];
    const int c0 = A.leaf_of[first];
    const double4_32a a0 = A.d_a[c0];
    const double ox = a0.x, oy = a0.y, oz = a0.z, L = root_side(A, first, one);
    float4 h0 = make_float4(0.f, 0.f, 0.f, 0.f), l0 = h0;
    if (kF32Q) {
        h0 = A.ra[c0];
        l0 = A.rb[c0];
    }
    MomSums S;
    mom_zero(S);
#pragma unroll 2
    for (int j = 0; j < count; j++) mom_add<kF32Q>(A, A.leaf_of[first + j], ox, oy, oz, h0, l0, S);
    mom_finish<kF32Q>(A, k, depth, end, first, L, ox, oy, oz, S);
}

constexpr int kDepths = kMaxDepth + 1;
constexpr int kMomSlots = 1024;   // most slots of a block's range
constexpr int kDirect = 8;        // cells of at most this many particles are summed from their leaves
constexpr int kGroupCells = 16;   // depths with at most this many cells take eight lanes a cell
constexpr int kBuckets = kDirect - 1 + kDepths;   // cells of 2 .. kDirect particles, then by depth

// Moments of the cells whose particles lie within one range of `slots`
// consecutive slots (a block each), and the leaf records.  The cells of at most
// kDirect particles, three quarters of all, come straight from their leaves,
// all at once and sorted by their count, so that warps are full and alike; the
// larger ones from their children, depth by depth with block barriers.  Cells
// that go on past the range's end all hold its last slot, so there is at most
// one of each depth: span[range][depth] (-1: none), for k_moments_span.
// Bound by FP64 issue (an FP64 warp instruction holds the SM's FP64 pipe 16
// cycles whatever its active lanes; 52% of its cycles busy at 400k) at many
// particles, by the chain of depths at few.  Moments and leaf records of one
// build, all launches: 41 us at 2,400 particles, 51 at 30k, 72 at 100k and 271
// at 1M, against 92, 123, 146 and 350 us with one launch per depth (26
// launches; these are three).
template <bool kF32Q>
__global__ void __launch_bounds__(256, 4) k_moments_range(GravRecArgs A, int slots, int32_t* __restrict__ span) {
    __shared__ int cnt[kBuckets], off[kBuckets], over[kDepths];
    __shared__ uint16_t list[2 * kMomSlots];   // the range's cells by bucket, as entry - e0
    const int n = sorted_n(A.ctl, A.ncap);
    const int p0 = blockIdx.x * slots, tid = threadIdx.x;
    if (p0 >= n) {
        if (tid < kDepths) span[blockIdx.x * kDepths + tid] = -1;
        return;
    }
    const int p1 = min(n, p0 + slots);
    const int e0 = A.start[p0], e1 = A.start[p1];
    const double one = A.boxes[0].L;
    if (tid < kBuckets) cnt[tid] = 0;
    if (tid < kDepths) over[tid] = -1;
    for (int p = p0 + tid; p < p1; p += 256) leaf_record(A, p);
    __syncthreads();
    auto bucket = [&](int e, int& v) {   // -1: a leaf, or a cell that ends past the range
        v = A.e_level[e];
        if (v >= kDepths) return -1;     // 22 marks a particle leaf
        const int c = A.e_count[e];
        if (A.e_first[e] + c > p1) return -1;
        return c <= kDirect ? c - 2 : kDirect - 1 + v;
    };
    for (int e = e0 + tid; e < e1; e += 256) {
        int v;
        const int b = bucket(e, v);
        if (b >= 0) atomicAdd(&cnt[b], 1);
        else if (v < kDepths) over[v] = e;
    }
    __syncthreads();
    if (tid < kBuckets) {
        int o = 0;
        for (int b = 0; b < tid; b++) o += cnt[b];
        off[tid] = o;
    }
    if (tid < kDepths) span[blockIdx.x * kDepths + tid] = over[tid];
    __syncthreads();
    for (int e = e0 + tid; e < e1; e += 256) {
        int v;
        const int b = bucket(e, v);
        if (b >= 0) list[atomicAdd(&off[b], 1)] = (uint16_t)(e - e0);
    }
    __syncthreads();   // off[b] now ends bucket b
    const int direct = off[kDirect - 2];
    for (int t = tid; t < direct; t += 256) {
        const int e = e0 + list[t];
        mom_cell_leaves<kF32Q>(A, e, A.e_count[e], one);
    }
    __syncthreads();
    for (int v = kMaxDepth; v >= 0; v--) {
        const int c = cnt[kDirect - 1 + v], first = off[kDirect - 1 + v] - c;
        if (c == 0) continue;
        if (c <= kGroupCells && v < kMaxDepth) {
            // four cells a warp
            if ((tid >> 5) * 4 < c) {
                const bool live = (tid >> 3) < c;
                mom_cell_group<kF32Q>(A, live, live ? e0 + list[first + (tid >> 3)] : 0, v, one);
            }
        } else {
            for (int t = tid; t < c; t += 256) mom_cell<kF32Q>(A, e0 + list[first + t], v, one);
        }
        __syncthreads();
    }
}

// The cells that go on past their range.  Listed by range and depth they are
// in pre-order, so the ones inside such a cell follow it without a gap: those
// of its own range at larger depths, then all of the ranges it covers.  With
// own(c) the part of a cell held by its children that end within their range
// (finished by k_moments_range), a cell is the sum of own() over itself and the
// cells inside it: no chain through the depths.  Both parts are kept as cell
// records behind the tree's entries, piece(r, v) and, for v = kDepths, the sum
// over range r.
__device__ __forceinline__ int piece(const GravRecArgs& A, int r, int v) {
    return A.piece0 + r * (kDepths + 1) + v;
}

// Record of a piece: the sums about o as mass, centre of mass and quadrupole.
template <bool kF32Q>
__device__ __forceinline__ void put_piece(const GravRecArgs& A, int k, double ox, double oy, double oz, MomSums& S) {
    double ux = 0.0, uy = 0.0, uz = 0.0;
    if (S.M > 0.0) {
        const double iM = rcp64(S.M);
        ux = S.sx * iM; uy = S.sy * iM; uz = S.sz * iM;
    }
    const double cx = ox + ux, cy = oy + uy, cz = oz + uz;
    mom_shift<kF32Q>(S, ux, uy, uz);
    A.d_a[k] = make_double4_32a(cx, cy, cz, 0.0);
    float hx, lx, hy, ly, hz, lz;
    split_hilo(cx, hx, lx);
    split_hilo(cy, hy, ly);
    split_hilo(cz, hz, lz);
    A.ra[k] = make_float4(hx, hy, hz, lz);
    A.rb[k] = make_float4(lx, ly, 0.f, 0.f);
    if (kF32Q) {
        A.d_q0[k].x = S.M;
        A.rq0[k] = make_float4((float)S.M, S.qf[0], S.qf[1], S.qf[2]);
        A.rq1[k] = make_float4(S.qf[3], S.qf[4], S.qf[5], 0.f);
    } else {
        A.d_q0[k] = make_double4_32a(S.M, S.q[0], S.q[1], S.q[2]);
        A.d_q1[k] = make_double4_32a(S.q[3], S.q[4], S.q[5], 0.0);
    }
}

// own() of a range's cells (a warp per range, eight lanes per cell) and their
// sum.
template <bool kF32Q>
__global__ void __launch_bounds__(64) k_moments_own(GravRecArgs A, int slots, const int32_t* __restrict__ span, int nr) {
    const int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (r >= nr) return;
    const int mine = lane < kDepths ? span[r * kDepths + lane] : -1;
    const unsigned have = __ballot_sync(0xffffffffu, mine >= 0);
    unsigned left = have;
    while (left) {
        // the next four cells, one per group of lanes
        unsigned m = left;
        for (int g = 0; g < (lane >> 3) && m; g++) m &= m - 1;
        const int v = m ? __ffs(m) - 1 : 0;
        const bool live = m != 0;
        for (int g = 0; g < 4 && left; g++) left &= left - 1;
        const int k = __shfl_sync(0xffffffffu, mine, v);
        MomSums S;
        mom_zero(S);
        double ox = 0.0, oy = 0.0, oz = 0.0;
        if (live) {
            const int o = lane & 7;
            const int c0 = A.leaf_of[A.e_first[k]];   // sums about its first particle
            const double4_32a a0 = A.d_a[c0];
            ox = a0.x; oy = a0.y; oz = a0.z;
            float4 h0 = make_float4(0.f, 0.f, 0.f, 0.f), l0 = h0;
            if (kF32Q) {
                h0 = A.ra[c0];
                l0 = A.rb[c0];
            }
            if (v == kMaxDepth) {
                // a leaf group: its members, whatever ranges they lie in
                for (int c = k + 1 + o, end = A.e_skip[k]; c < end; c += 8)
                    mom_add<kF32Q>(A, c, ox, oy, oz, h0, l0, S);
            } else if ((A.e_cmask[k] >> o) & 1u) {
                const int c = A.e_child[8 * (size_t)k + o];
                const int first = A.e_first[c];
                if (first + A.e_count[c] <= (first / slots + 1) * slots)
                    mom_add<kF32Q>(A, c, ox, oy, oz, h0, l0, S);
            }
        }
        mom_reduce<kF32Q>(S, 8);
        if (live && (lane & 7) == 0) put_piece<kF32Q>(A, piece(A, r, v), ox, oy, oz, S);
    }
    __syncwarp();
    MomSums S;
    mom_zero(S);
    double ox = 0.0, oy = 0.0, oz = 0.0;
    if (have) {
        const int c0 = piece(A, r, __ffs(have) - 1);
        const double4_32a a0 = A.d_a[c0];
        ox = a0.x; oy = a0.y; oz = a0.z;
        if (mine >= 0) mom_add<kF32Q>(A, piece(A, r, lane), ox, oy, oz, A.ra[c0], A.rb[c0], S);
    }
    mom_reduce<kF32Q>(S, 32);
    if (lane == 0) put_piece<kF32Q>(A, piece(A, r, kDepths), ox, oy, oz, S);
}

// The cells themselves, a block per range: a warp per cell, or the whole block
// for a cell that covers many ranges.
constexpr int kLongCell = 128;

template <bool kF32Q>
__global__ void __launch_bounds__(256) k_moments_span(GravRecArgs A, int slots, const int32_t* __restrict__ span) {
    __shared__ MomSums part[8];
    const int r = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int mine = lane < kDepths ? span[r * kDepths + lane] : -1;
    const unsigned have = __ballot_sync(0xffffffffu, mine >= 0);
    if (!have) return;
    const double one = A.boxes[0].L;
    // this lane's share of the cell at depth v: pieces of its own range by the
    // lanes of warp w0, the sums of the ranges it covers by `width` lanes
    auto share = [&](int v, int r2, int at, int width, bool own, const double4_32a& a0, const float4& h0,
                     const float4& l0, MomSums& S) {
        mom_zero(S);
        if (own && mine >= 0 && lane >= v) mom_add<kF32Q>(A, piece(A, r, lane), a0.x, a0.y, a0.z, h0, l0, S);
        // a leaf group's piece is all of it
        for (int q = r + 1 + at; v < kMaxDepth && q < r2; q += width)
            mom_add<kF32Q>(A, piece(A, q, kDepths), a0.x, a0.y, a0.z, h0, l0, S);
        mom_reduce<kF32Q>(S, 32);
    };
    unsigned left = have, wide = 0;
    for (int j = 0; left; left &= left - 1, j++) {
        const int v = __ffs(left) - 1;
        const int k = __shfl_sync(0xffffffffu, mine, v);
        const int first = A.e_first[k];
        const int r2 = (first + A.e_count[k] - 1) / slots;
        if (r2 - r > kLongCell && v < kMaxDepth) {
            wide |= 1u << v;
            continue;
        }
        if ((j & 7) != warp) continue;
        const int end = A.e_skip[k], c0 = A.leaf_of[first];
        const double L = root_side(A, first, one);
        const double4_32a a0 = A.d_a[c0];
        MomSums S;
        share(v, r2, lane, 32, true, a0, A.ra[c0], A.rb[c0], S);
        if (lane == 0) mom_finish<kF32Q>(A, k, v, end, first, L, a0.x, a0.y, a0.z, S);
    }
    for (; wide; wide &= wide - 1) {
        const int v = __ffs(wide) - 1;
        const int k = __shfl_sync(0xffffffffu, mine, v);
        const int first = A.e_first[k];
        const int r2 = (first + A.e_count[k] - 1) / slots;
        const int c0 = A.leaf_of[first];
        const double4_32a a0 = A.d_a[c0];
        MomSums S;
        share(v, r2, threadIdx.x, 256, warp == 0, a0, A.ra[c0], A.rb[c0], S);
        __syncthreads();   // part is reused
        if (lane == 0) part[warp] = S;
        __syncthreads();
        if (warp == 0) {
            if (lane < 8) S = part[lane];
            else mom_zero(S);
            mom_reduce<kF32Q>(S, 8);
            if (lane == 0)
                mom_finish<kF32Q>(A, k, v, A.e_skip[k], first, root_side(A, first, one), a0.x, a0.y, a0.z, S);
        }
    }
}

struct CollRecArgs {
    const double *x, *y, *z, *r;
    const int32_t* box;
    const int32_t *e_first, *e_skip, *leaf_of, *e_count;
    const int8_t* e_level;
    Rec4 ra, rb;
    const Ctl* ctl;
    int ecap, ncap, nbox;
    float4* pbox = nullptr;   // box items (pairs lo, hi): slots, then runs of 32, then runs of 256
};

// Collision records on the gravity tree, at the positions after the second
// drift (Sect. 5.2, with a tighter pruning volume than Eq. 3's sphere): the
// tree's cells still hold the same particles, and a cell records the
// axis-aligned box of its particles' current positions (lower corner rounded
// down, upper corner rounded up to FP32), so the search stays exact without a
// second sort and build.  A cell's record also holds the largest particle
// slot below it (ra.w), so a search from slot i skips subtrees whose pairs
// with i are examined from the other particle.  A leaf's
// record holds its position (hi/lo), radius and slot; a removed particle's sits
// at +infinity and is never close.
// Boxes from particle ranges: a cell of the gravity tree holds the
// consecutive slots [first, first + count), so its box is the union of its
// particles' boxes, taken here from the fewest aligned runs that tile the
// range (single slots at its ends, runs of 32, 256 and 8192 slots).
// Minima and maxima are exact in any order, so the records equal those of a
// bottom-up merge over the children, in three launches instead of one per
// depth.  A box item is the pair (lo, hi): lo = lower corner and the largest
// live slot (int bits, -1 none), hi = upper corner; an item with no live
// particle is (+inf, -inf).
constexpr int kRunA = 32, kRunB = 256, kRunC = 8192;
constexpr int kRunsInB = kRunB / kRunA, kRunsInC = kRunC / kRunB;
static_assert(kRunsInC == 32, "a warp per run of 8192 slots");

struct BoxAcc {
    float lox, loy, loz, hix, hiy, hiz;
    int top;
};

__device__ __forceinline__ BoxAcc box_empty() {
    const float inf = __int_as_float(0x7f800000);
    return BoxAcc{inf, inf, inf, -inf, -inf, -inf, -1};
}

__device__ __forceinline__ void box_fold(BoxAcc& B, const BoxAcc& o) {
    B.lox = fminf(B.lox, o.lox); B.loy = fminf(B.loy, o.loy); B.loz = fminf(B.loz, o.loz);
    B.hix = fmaxf(B.hix, o.hix); B.hiy = fmaxf(B.hiy, o.hiy); B.hiz = fmaxf(B.hiz, o.hiz);
    B.top = max(B.top, o.top);
}

// Fold of the boxes of the lanes l with (l & ~(width - 1)) equal, width a
// power of two up to 32.
__device__ __forceinline__ void box_reduce(BoxAcc& B, int width) {
    for (int x = 1; x < width; x <<= 1) {
        BoxAcc o;
        o.lox = __shfl_xor_sync(0xffffffffu, B.lox, x);
        o.loy = __shfl_xor_sync(0xffffffffu, B.loy, x);
        o.loz = __shfl_xor_sync(0xffffffffu, B.loz, x);
        o.hix = __shfl_xor_sync(0xffffffffu, B.hix, x);
        o.hiy = __shfl_xor_sync(0xffffffffu, B.hiy, x);
        o.hiz = __shfl_xor_sync(0xffffffffu, B.hiz, x);
        o.top = __shfl_xor_sync(0xffffffffu, B.top, x);
        box_fold(B, o);
    }
}

__device__ __forceinline__ void item_put(float4* pbox, long long i, const BoxAcc& B) {
    pbox[2 * i] = make_float4(B.lox, B.loy, B.loz, __int_as_float(B.top));
    pbox[2 * i + 1] = make_float4(B.hix, B.hiy, B.hiz, 0.f);
}

__device__ __forceinline__ void item_fold(const float4* pbox, long long i, BoxAcc& B) {
    const float4 lo = pbox[2 * i], hi = pbox[2 * i + 1];
    B.lox = fminf(B.lox, lo.x); B.loy = fminf(B.loy, lo.y); B.loz = fminf(B.loz, lo.z);
    B.hix = fmaxf(B.hix, hi.x); B.hiy = fmaxf(B.hiy, hi.y); B.hiz = fmaxf(B.hiz, hi.z);
    B.top = max(B.top, __float_as_int(lo.w));
}

__device__ __forceinline__ void cell_put(const CollRecArgs& A, int k, const BoxAcc& B) {
    A.ra[k] = make_float4(B.lox, B.loy, B.loz, __int_as_float(B.top));
    A.rb[k] = make_float4(B.hix, B.hiy, B.hiz, __int_as_float(A.e_skip[k]));
}

// Collision records on the gravity tree, at the positions after the second
// drift (Sect. 5.2, with a tighter pruning volume than Eq. 3's sphere): the
// tree's cells still hold the same particles, and a cell records the
// axis-aligned box of its particles' current positions (lower corner rounded
// down, upper corner rounded up to FP32), so the search stays exact without a
// second sort and build.  A cell's record also holds the largest particle
// slot below it (ra.w), so a search from slot i skips subtrees whose pairs
// with i are examined from the other particle.  A leaf's
// record holds its position (hi/lo), radius and slot; a removed particle's sits
// at +infinity and is never close.  This launch also writes the box items of
// every slot and of the runs of 32 and 256 slots (kRunB threads per block).
__global__ void __launch_bounds__(kRunB) k_aabb_leaves(CollRecArgs A) {
    __shared__ BoxAcc wbox[kRunsInB];
    const int n = sorted_n(A.ctl, A.ncap);
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    BoxAcc B = box_empty();
    if (p < n) {
        const int e = A.leaf_of[p];
        if (A.box[p] >= A.nbox) {
            const float inf = __int_as_float(0x7f800000);
            A.ra[e] = make_float4(inf, inf, inf, __int_as_float(~p));
            A.rb[e] = make_float4(0.f, 0.f, 0.f, (float)A.r[p]);
        } else {
            float hx, lx, hy, ly, hz, lz;
            split_hilo(A.x[p], hx, lx);
            split_hilo(A.y[p], hy, ly);
            split_hilo(A.z[p], hz, lz);
            A.ra[e] = make_float4(hx, hy, hz, __int_as_float(~p));
            A.rb[e] = make_float4(lx, ly, lz, (float)A.r[p]);
            // hi = x rounded to nearest, lo the sign of x - hi: x lies in
            // [hi, next float up] or [next float down, hi]
            const float inf = __int_as_float(0x7f800000);
            B.lox = lx < 0.f ? nextafterf(hx, -inf) : hx;
            B.hix = lx > 0.f ? nextafterf(hx, inf) : hx;
            B.loy = ly < 0.f ? nextafterf(hy, -inf) : hy;
            B.hiy = ly > 0.f ? nextafterf(hy, inf) : hy;
            B.loz = lz < 0.f ? nextafterf(hz, -inf) : hz;
            B.hiz = lz > 0.f ? nextafterf(hz, inf) : hz;
            B.top = p;
        }
        item_put(A.pbox, p, B);
    }
    box_reduce(B, kRunA);
    const int w = threadIdx.x / kRunA;
    if (threadIdx.x % kRunA == 0) {
        if (p < n) item_put(A.pbox, (long long)A.ncap + p / kRunA, B);
        wbox[w] = B;
    }
    __syncthreads();
    if (w == 0) {
        BoxAcc C = (threadIdx.x < kRunsInB) ? wbox[threadIdx.x] : box_empty();
        box_reduce(C, kRunsInB);
        const int nruns = (A.ncap + kRunA - 1) / kRunA;
        if (threadIdx.x == 0 && blockIdx.x * kRunB < n)
            item_put(A.pbox, (long long)A.ncap + nruns + blockIdx.x, C);
    }
}

// The aligned pieces of [lo, hi) (units of the finer run) at a coarser run
// of `ratio` finer ones: the finer runs before the first coarse boundary,
// the coarse runs [c0, c1), the finer runs from c1 * ratio on.
struct Split {
    int head_end, c0, c1, tail_begin;
};
__device__ __forceinline__ Split split_runs(int lo, int hi, int ratio) {
    Split S;
    S.head_end = min(hi, (lo + ratio - 1) / ratio * ratio);
    S.tail_begin = max(S.head_end, hi / ratio * ratio);
    S.c0 = S.head_end / ratio;
    S.c1 = S.tail_begin / ratio;
    return S;
}

// Box items of the runs of 8192 slots, from their 32 runs of 256 (a warp per
// run).
__global__ void __launch_bounds__(256) k_aabb_runs(CollRecArgs A) {
    const int n = sorted_n(A.ctl, A.ncap);
    const long long nA = (A.ncap + kRunA - 1) / kRunA, nB = (A.ncap + kRunB - 1) / kRunB;
    const int lane = threadIdx.x & 31;
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    for (int c = w; (long long)c * kRunC < n; c += nw) {
        BoxAcc B = box_empty();
        const int q = c * kRunsInC + lane;   // its run of 256
        if ((long long)q * kRunB < n) item_fold(A.pbox, A.ncap + nA + q, B);
        box_reduce(B, 32);
        if (lane == 0) item_put(A.pbox, A.ncap + nA + nB + c, B);
    }
}

// Folds the items that tile slots [a, e), lane `lane` of 32 taking every
// 32nd one: slots and runs of 32 and 256 at both ends, runs of 8192 between.
// A cell of c slots needs at most 138 + c / 8192 items.
__device__ __forceinline__ void range_fold(const CollRecArgs& A, int a, int e, int lane, BoxAcc& B) {
    const long long nA = (A.ncap + kRunA - 1) / kRunA, nB = (A.ncap + kRunB - 1) / kRunB;
    const long long baseA = A.ncap, baseB = baseA + nA, baseC = baseB + nB;
    const Split s1 = split_runs(a, e, kRunA);                // slots | runs of 32
    const Split s2 = split_runs(s1.c0, s1.c1, kRunsInB);     // runs of 32 | runs of 256
    const Split s3 = split_runs(s2.c0, s2.c1, kRunsInC);     // runs of 256 | runs of 8192
    // seven pieces in turn, each (first item index, count); `off` carries
    // this lane's position from one piece into the next
    int off = lane;
    auto piece = [&](long long first, int count) {
#pragma unroll 1
        for (; off < count; off += 32) item_fold(A.pbox, first + off, B);
        off -= count;
    };
    piece(a, s1.head_end - a);
    piece(baseA + s1.c0, s2.head_end - s1.c0);
    piece(baseB + s2.c0, s3.head_end - s2.c0);
    piece(baseC + s3.c0, s3.c1 - s3.c0);
    piece(baseB + s3.tail_begin, s2.c1 - s3.tail_begin);
    piece(baseA + s2.tail_begin, s1.c1 - s2.tail_begin);
    piece(s1.tail_begin, e - s1.tail_begin);
}

// Every cell of the gravity build, in entry order (consecutive entries: the
// counts and first slots are read coalesced; particle leaves are skipped).
// A lane takes a cell of at most eight slots alone; larger cells are taken
// afterwards by the whole warp, one at a time.
__global__ void __launch_bounds__(256) k_aabb_cells(CollRecArgs A) {
    const int entries = min(A.ctl->n_entries, A.ecap);
    const int E = sorted_n(A.ctl, 1) ? entries : 0;
    const int lane = threadIdx.x & 31;
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    for (int e0 = 32 * w; e0 < E; e0 += 32 * nw) {
        const int k = e0 + lane;
        const bool cell = k < E && A.e_level[k] < 22;   // 22 marks a particle leaf
        int a = 0, c = 0;
        if (cell) {
            a = A.e_first[k];
            c = A.e_count[k];
        }
        if (cell && c <= 8) {
            BoxAcc B = box_empty();
#pragma unroll 4
            for (int j = 0; j < c; j++) item_fold(A.pbox, a + j, B);
            cell_put(A, k, B);
        }
        unsigned big = __ballot_sync(0xffffffffu, cell && c > 8);
        while (big) {
            const int src = __ffs(big) - 1;
            big &= big - 1;
            const int ab = __shfl_sync(0xffffffffu, a, src);
            const int cb = __shfl_sync(0xffffffffu, c, src);
            BoxAcc W = box_empty();
            range_fold(A, ab, ab + cb, lane, W);
            box_reduce(W, 32);
            if (lane == 0) cell_put(A, e0 + src, W);
        }
    }
}

}  // namespace

size_t entry_scan_words(int ncap) { return (size_t)ceil_div(ncap > 0 ? ncap : 1, kScanTile); }

// mask, e_cmask, box_root and scan_stat are cleared by the gather before.
void build_topology(const Tree& T, const PSet& P, Ctl* ctl, const BoxP* boxes, const SimC& C,
                    cudaStream_t s) {
    const int n = T.cap_n;
    if (n <= 0) return;
    const int nb = ceil_div(n, 256);
    if (C.nbox > 1)
        k_nodes<true><<<nb, 256, 0, s>>>(T.key, P.box, ctl, n, T.node_a, T.node_b, T.node_v, T.mask);
    else
        k_nodes<false><<<nb, 256, 0, s>>>(T.key, P.box, ctl, n, T.node_a, T.node_b, T.node_v,
                                          T.mask);
    k_entry_scan<<<ceil_div(n, kScanTile), 256, 0, s>>>(T.mask, ctl, n, T.start, T.scan_stat,
                                                        (C.hold_sort & kHoldScan) != 0);
    k_emit<<<nb, 256, 0, s>>>(T.mask, T.start, T.node_a, T.node_b, T.node_v, ctl, n, T.e_first,
                              T.e_count, T.e_skip, T.e_level, T.leaf_of, T.key, T.e_child, T.e_cmask, P.box,
                              T.box_root);
}

namespace {

// Hilbert index of (x, y) on a 2^lv grid (the classic quadrant rotation
// walk, most significant level first).
__device__ __forceinline__ uint32_t hilbert2(uint32_t x, uint32_t y, int lv) {
    const uint32_t n = 1u << lv;
    uint32_t d = 0;
    for (uint32_t s = n >> 1; s > 0; s >>= 1) {
        const uint32_t rx = (x & s) ? 1u : 0u, ry = (y & s) ? 1u : 0u;
        d += s * s * ((3u * rx) ^ ry);
        if (ry == 0) {
            if (rx == 1) {
                x = n - 1 - x;
                y = n - 1 - y;
            }
            const uint32_t t = x;
            x = y;
            y = t;
        }
    }
    return d;
}

// Hilbert index of (x, y, z) on a 2^lv grid: the axes are turned into the
// curve's "transposed" form (Skilling 2004, AIP Conf. Proc. 707: inverse
// undo of the excess work, then Gray decoding), whose bits interleaved
// from the top give the index.
__device__ __forceinline__ uint32_t hilbert3(uint32_t x, uint32_t y, uint32_t z, int lv) {
    uint32_t c[3] = {x, y, z};
    const uint32_t m = 1u << (lv - 1);
    for (uint32_t q = m; q > 1; q >>= 1) {
        const uint32_t p = q - 1;
#pragma unroll
        for (int a = 0; a < 3; a++) {
            if (c[a] & q) {
                c[0] ^= p;
            } else {
                const uint32_t t = (c[0] ^ c[a]) & p;
                c[0] ^= t;
                c[a] ^= t;
            }
        }
    }
    c[1] ^= c[0];
    c[2] ^= c[1];
    uint32_t t = 0;
    for (uint32_t q = m; q > 1; q >>= 1)
        if (c[2] & q) t ^= q - 1;
    uint32_t d = 0;
    for (int b = lv - 1; b >= 0; b--)
#pragma unroll
        for (int a = 0; a < 3; a++) d = (d << 1) | (((c[a] ^ t) >> b) & 1u);
    return d;
}

// Tile keys of the sorted slots: the box above a Hilbert key of the slot's
// integer coordinates (read back from its Morton key); value = the slot.
__global__ void __launch_bounds__(256) k_tile_keys(const uint64_t* __restrict__ key,
                                                   const int32_t* __restrict__ box,
                                                   const Ctl* __restrict__ ctl, int ncap, int mode,
                                                   uint64_t* __restrict__ tkey, uint32_t* __restrict__ tval) {
    const int n = sorted_n(ctl, ncap);
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint64_t k = key[i];
    const uint32_t ix = morton_compact3(k >> 2), iy = morton_compact3(k >> 1), iz = morton_compact3(k);
    const uint32_t h = mode == kTileHilbertXY ? hilbert2(ix >> 11, iy >> 11, 10)
                                              : hilbert3(ix >> 14, iy >> 14, iz >> 14, 7);
    tkey[i] = ((uint64_t)(uint32_t)box[i] << 21) | (uint64_t)h;
    tval[i] = (uint32_t)i;
}

}  // namespace

void build_tile_order(Tree& T, const PSet& P, Ctl* ctl, const SimC& C, int mode, int box_bits, cudaStream_t s) {
    if (mode == kTileMorton || T.cap_n <= 0) {
        T.order = nullptr;
        return;
    }
    k_tile_keys<<<ceil_div(T.cap_n, 256), 256, 0, s>>>(T.key, P.box, ctl, T.cap_n, mode, T.tkey, T.tval);
    const int which = radix_sort(T.tkey, T.tval, T.tkey_alt, T.tval_alt, T.cap_n, &ctl->n_live,
                                 21 + box_bits, nullptr, 0, T.thist, &ctl->err, s, 0, nullptr, nullptr,
                                 (C.hold_sort & kHoldTiles) != 0);
    T.order = which ? T.tval_alt : T.tval;
}

namespace {

// Slots of a block's range.  Few particles: short ranges, which end sooner
// (2,400: 54 us in ranges of 256 slots, 70 of 512 and 79 of 1024; 100k: 88, 92
// and 102).  More than fill the GPU that way (608 resident blocks): the longest
// that fill it once or a whole number of times, since long ranges fill the
// warps of a depth (1M: 340 us at 1024, 390 at 512).
int moment_slots(int n) {
    constexpr int kBlocks = 4 * 152;
    if (n <= kBlocks * 256) return 256;
    const int waves = ceil_div(n, kBlocks * kMomSlots);
    return ceil_div(ceil_div(n, (long long)kBlocks * waves), 8) * 8;
}

}  // namespace

size_t moment_span_words(int ncap) { return (size_t)ceil_div(ncap, moment_slots(ncap)) * kDepths; }
size_t moment_pieces(int ncap) { return (size_t)ceil_div(ncap, moment_slots(ncap)) * (kDepths + 1); }

void build_gravity_records(const Tree& T, const PSet& P, Ctl* ctl, const BoxP* boxes,
                           const SimC& C, bool fp64, cudaStream_t s, bool f32q) {
    const int n = T.cap_n;
    if (n <= 0) return;
    GravRecArgs A;
    A.x = P.x; A.y = P.y; A.z = P.z; A.m = P.m; A.box = P.box; A.id = P.id;
    A.has_test = C.has_test != 0;
    A.one = C.nbox == 1;
    A.key = T.key; A.boxes = boxes;
    A.e_first = T.e_first; A.e_skip = T.e_skip; A.e_child = T.e_child;
    A.e_cmask = T.e_cmask; A.leaf_of = T.leaf_of; A.e_level = T.e_level;
    A.e_count = T.e_count; A.start = T.start;
    A.d_a = T.d_a; A.d_q0 = T.d_q0; A.d_q1 = T.d_q1; A.d_c = T.d_c;
    A.ra = T.ra; A.rb = T.rb; A.rq0 = T.rq0; A.rq1 = T.rq1; A.rc_hi = T.rc_hi; A.rc_lo = T.rc_lo;
    A.ctl = ctl;
    A.ncap = n;
    A.crit_scale = C.crit_scale;
    A.q32 = !fp64;
    A.leafq = !fp64 && n <= kLeafQMax;
    A.corners = C.theta2 > (1.0 / 3.0) || C.learned;
    const bool q32 = f32q && !fp64;
    const int slots = moment_slots(n);
    const int nr = ceil_div(n, slots);
    A.piece0 = T.cap_e;
    if (q32) k_moments_range<true><<<nr, 256, 0, s>>>(A, slots, T.span);
    else k_moments_range<false><<<nr, 256, 0, s>>>(A, slots, T.span);
    if (nr == 1) return;
    const int nb = ceil_div(nr, 2);   // a warp per range
    if (q32) {
        k_moments_own<true><<<nb, 64, 0, s>>>(A, slots, T.span, nr);
        k_moments_span<true><<<nr, 256, 0, s>>>(A, slots, T.span);
    } else {
        k_moments_own<false><<<nb, 64, 0, s>>>(A, slots, T.span, nr);
        k_moments_span<false><<<nr, 256, 0, s>>>(A, slots, T.span);
    }
}

void build_collision_aabb(const Tree& T, const PSet& P, Ctl* ctl, const SimC& C, cudaStream_t s) {
    if (T.cap_n <= 0) return;
    CollRecArgs A;
    A.x = P.x; A.y = P.y; A.z = P.z; A.r = P.r;
    A.box = P.box;
    A.e_first = T.e_first; A.e_skip = T.e_skip; A.e_level = T.e_level; A.leaf_of = T.leaf_of;
    A.e_count = T.e_count;
    A.ra = T.ra; A.rb = T.rb; A.ctl = ctl; A.ecap = T.cap_e;
    A.ncap = T.cap_n; A.nbox = C.nbox;
    A.pbox = T.pbox;
    k_aabb_leaves<<<ceil_div(T.cap_n, kRunB), kRunB, 0, s>>>(A);
    k_aabb_runs<<<ceil_div(ceil_div(T.cap_n, kRunC), 8), 256, 0, s>>>(A);
    // a warp per 32 entries; the resident blocks (48 registers: 5 of 256 per SM)
    const int grid = std::min(ceil_div(T.cap_e, 256), 5 * 152);
    k_aabb_cells<<<grid, 256, 0, s>>>(A);
}

}  // namespace rb
