// rb_collide.cu -- tree collision search (Sect. 5.2) over the ghost images of
// Sect. 2.3.
//
// A warp takes up to 32 consecutive targets and searches the tree once for all
// of them.  The lanes hold a frontier of (ghost image, entry) items: each round
// they test up to 32 entries against the bounding box of the targets, push
// the children of cells that come within R_max of it and put the leaves that
// do into a list of candidates in shared memory; then every lane tests its
// own target against the candidates.  Cells are boxes of their particles'
// current positions (build_collision_aabb), so the pruning volume is a subset
// of Eq. 3's that still holds every overlap.
// Against a walk of each target's own (lane per target, the warp stepping
// through the union of 32 walks, about 260 dependent entries), a tile of the
// 1M sheet tests 370 entries and 73 candidates: 0.59 -> 0.28 ms (100k: 163 -> 60
// us, 2400: 125 -> 22 us).  Bound by instruction issue with many particles, by a
// tile's chain of rounds with few.
//
// The targets are consecutive slots, in Morton order whatever order the walk
// takes: a pair is recorded from its lower slot, so subtrees that lie before
// the run hold none and are pruned, which halves the candidates.  The order
// jumps between octants, and a target may have left the others since the tree
// was built (a wrap across a periodic face, a close encounter): a box around
// such a run would hold much of the tree, so it is cut at its widest gaps into
// compact parts.  Up to four of them are searched together, their items on one
// frontier and tagged with their part: in turn, a tile's 370 entries took 24
// rounds, half of whose lanes were idle (1M: 324 -> 283 us, 100k: 70 -> 60, 20k:
// 43 -> 37, 2400: 27 -> 22).
#include <algorithm>
#include <cfloat>

#include "rb_walk.cuh"

namespace rb {
namespace {

constexpr int kEntBits = 25;                 // entries < 2 (2^24 - 1) < 2^25
constexpr int kEntMask = (1 << kEntBits) - 1;
constexpr int kImgBatch = 32;                // images whose items share the frontier
constexpr int kImgShift = kEntBits, kSegShift = 30;
constexpr unsigned kImgMask = 31u;
constexpr int kSegs = 4;                     // parts of a tile searched together
constexpr int kStack = 448;
constexpr int kReserve = 160;                // depth-first room: 7 siblings on each of 22 levels

// Targets of a tile.  Tiles of 32 leave the GPU idle with few particles (2,400:
// 75 warps), and a tile's time is its own chain of rounds and candidates: fewer
// targets have fewer of both, at the price of more rounds in all.  Search of the
// sheet with 32, 8 and 4 targets a tile (parts searched in turn): 47, 29 and 27 us
// at 2,400 particles, 60, 39 and 35 at 10k, 51, 43 and 52 at 20k, 58, 50 and 61 at
// 30k, 63, 72 and 90 at 60k; of a periodic cube: 61, 33 and 31 us at 10k, 86, 45 and
// 54 at 30k, 63, 63 and 76 at 60k.
constexpr int kWidth4Max = 10000;
constexpr int kWidth8Max = 40000;

struct CollArgs {
    const double *x, *y, *z, *r;
    const int32_t *id, *box;
    Rec4 ra, rb;
    const int32_t *box_root, *e_skip, *e_child;
    const uint32_t* e_cmask;
    Ctl* ctl;
    uint64_t* pair_key;
    int pair_cap, ncap;
    int ngx, ngy, ngz;
    const ImgTab* img;      // [box][image] offsets at the time of this search
    int nimg;
    int32_t* tq;            // tile queues (emptied by the image-table launch)
    int nq;
    float rmaxf;            // largest radius, rounded up
    int width;              // targets of a tile (at most 32)
};

// A compact part of a tile's targets.
struct Segment {
    float lx, hx, ly, hy, lz, hz;   // bounding box
    float reach, size;              // widening; largest absolute values that enter its distances
    int min_slot;                   // lowest slot of its targets
    int count;                      // its targets
};

struct SearchSmem {
    Segment seg[kSegs];
    float4 ca[64], cb[64];        // candidates: image position hi and radius; lo and slot
    float4 ohi[kImgBatch];        // image offset (hi); w: sum of its absolute values
    float4 olo[kImgBatch];
    unsigned stack[kStack];       // (segment << 30) | (image of the batch << 25) | entry
    int cimg[64];                 // the candidates' images, (segment << 16) | image
    int hi[64], hj[64], hg[64];   // pairs found: slots, 2 * image + (1: clear of the threshold)
};

// Overlap test of Sect. 5.1 on the canonical orientation (a = lower id, b
// seen through image offset o), operation for operation as the oracle.
// kNeg: the offset is -o (b + (-o) and b - o round identically in IEEE
// arithmetic, so no negated copy of o is formed).
template <bool kNeg = false>
__device__ __forceinline__ bool overlap64(double xa, double ya, double za, double ra, double xb,
                                          double yb, double zb, double rb, double ox, double oy,
                                          double oz) {
    const double rx = __dsub_rn(kNeg ? __dsub_rn(xb, ox) : __dadd_rn(xb, ox), xa);
    const double ry = __dsub_rn(kNeg ? __dsub_rn(yb, oy) : __dadd_rn(yb, oy), ya);
    const double rz = __dsub_rn(kNeg ? __dsub_rn(zb, oz) : __dadd_rn(zb, oz), za);
    const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(rx, rx), __dmul_rn(ry, ry)), __dmul_rn(rz, rz));
    const double sr = __dadd_rn(ra, rb);
    return r2 < __dmul_rn(sr, sr);
}

__device__ __forceinline__ float redux_min(float v) {
    float r;
    asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float redux_max(float v) {
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}

struct Box3 {
    float lx, hx, ly, hy, lz, hz;
};

// Bounding box of the lanes with in; every lane gets it.
__device__ __forceinline__ Box3 warp_box(bool in, float x, float y, float z) {
    const float inf = __int_as_float(0x7f800000);
    Box3 B;
    B.lx = redux_min(in ? x : inf);
    B.hx = redux_max(in ? x : -inf);
    B.ly = redux_min(in ? y : inf);
    B.hy = redux_max(in ? y : -inf);
    B.lz = redux_min(in ? z : inf);
    B.hz = redux_max(in ? z : -inf);
    return B;
}

// Volume searched for a box widened by m on every side.
__device__ __forceinline__ float searched(const Box3& B, float m) {
    return (B.hx - B.lx + 2.f * m) * (B.hy - B.ly + 2.f * m) * (B.hz - B.lz + 2.f * m);
}

// This lane's target, tested against a list of candidates.
struct Target {
    int slot;
    float hx, lx, hy, ly, hz, lz, r;   // FP32 hi/lo position, radius
};

// Records the first `n` (<= 32) of the found pairs, a lane each.  Pairs whose
// FP32 distance lies within 1e-4 of the threshold get the exact FP64 test in
// the oracle's operation order on the canonical orientation (lower id a, image
// of b as seen from a): an FP64 instruction holds the SM's FP64 pipe 16 cycles
// per warp, so the others do without.
__device__ __forceinline__ void record_pairs(const CollArgs& A, const SearchSmem& S, int from, int n,
                                             const ImgTab* itab) {
    const int lane = threadIdx.x & 31;
    bool hit = false;
    uint64_t key = 0;
    if (lane < n) {
        const int i = S.hi[from + lane], j = S.hj[from + lane];
        const int g = S.hg[from + lane] >> 1;
        const int pid = A.id[i], jid = A.id[j];
        const bool low = pid < jid;
        hit = S.hg[from + lane] & 1;   // clear of the threshold
        if (!hit) {
            const double ox = itab[g].ox, oy = itab[g].oy, oz = itab[g].oz;
            // j the lower id: this particle is its image -g, whose offset is
            // exactly -o (the table is symmetric)
            hit = low ? overlap64(A.x[i], A.y[i], A.z[i], A.r[i], A.x[j], A.y[j], A.z[j], A.r[j], ox, oy, oz)
                      : overlap64<true>(A.x[j], A.y[j], A.z[j], A.r[j], A.x[i], A.y[i], A.z[i], A.r[i], ox, oy,
                                        oz);
        }
        const int ny = 2 * A.ngy + 1, nz = 2 * A.ngz + 1;
        int gx = g / (ny * nz) - A.ngx, gy = (g / nz) % ny - A.ngy, gz = g % nz - A.ngz;
        if (!low) {
            gx = -gx;
            gy = -gy;
            gz = -gz;
        }
        const uint64_t code = (uint64_t)((gx + 7) | ((gy + 7) << 4) | ((gz + 7) << 8));
        key = ((uint64_t)min(pid, jid) << 36) | ((uint64_t)max(pid, jid) << 12) | code;
    }
    const unsigned hits = __ballot_sync(kFull, hit);
    if (!hits) return;
    int base = 0;
    if (lane == 0) base = atomicAdd(&A.ctl->pair_count, __popc(hits));
    base = __shfl_sync(kFull, base, 0);
    if (hit) {
        const int at = base + __popc(hits & ((1u << lane) - 1u));
        if (at < A.pair_cap) A.pair_key[at] = key;
        else atomicOr(&A.ctl->err, kErrPairOverflow);
    }
}

// Every lane against the candidates [0, nc) of its segment, in FP32 on hi/lo
// positions (distance good to ~1e-7 relative).  Each unordered pair is found
// once, from its lower slot (the other particle reaches it through the
// opposite image).  Found pairs are queued and recorded 32 at a time: their
// ids and the pair counter are round trips to L2, which one by one, in the
// loop, took two fifths of the search at 1M.
__device__ __forceinline__ void test_candidates(const CollArgs& A, SearchSmem& S, int nc, int seg,
                                                const Target& T, const ImgTab* itab, int& nh) {
    const unsigned lt = (1u << (threadIdx.x & 31)) - 1u;
    for (int c = 0; c < nc; c++) {
        const float4 a = S.ca[c], b = S.cb[c];
        const float dx = (a.x - T.hx) + (b.x - T.lx);
        const float dy = (a.y - T.hy) + (b.y - T.ly);
        const float dz = (a.z - T.hz) + (b.z - T.lz);
        const float d2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
        const float sr = T.r + a.w;
        const float s2 = sr * sr;
        const int j = __float_as_int(b.w);
        const int ci = S.cimg[c];
        const bool near = seg == ci >> 16 && j > T.slot && d2 < s2 * 1.0001f;
        const unsigned m = __ballot_sync(kFull, near);
        if (!m) continue;
        if (near) {
            const int at = nh + __popc(m & lt);
            S.hi[at] = T.slot;
            S.hj[at] = j;
            S.hg[at] = ((ci & 0xffff) << 1) | (d2 < s2 * 0.9999f ? 1 : 0);
        }
        nh += __popc(m);
        if (nh >= 32) {
            nh -= 32;
            __syncwarp();
            record_pairs(A, S, nh, 32, itab);
            __syncwarp();
        }
    }
}

// The targets of nseg segments in one box against that box's tree: all images.
// seg: the lane's segment (-1: none).  A subtree whose particles all sit at
// slots up to a segment's lowest holds no pair that is recorded from there.
template <bool kCount>
__device__ __forceinline__ void search_segments(const CollArgs& A, SearchSmem& S, int nseg, int seg, const Target& T,
                                                int root, const ImgTab* itab, unsigned long long& visits,
                                                unsigned long long& tested) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    int nh = 0;   // pairs found and not yet recorded (warp-uniform, < 32)
    for (int g0 = 0; g0 < A.nimg; g0 += kImgBatch) {
        const int nb = min(kImgBatch, A.nimg - g0);
        __syncwarp();
        if (lane < nb) {
            const float4 h = itab[g0 + lane].hi;
            S.ohi[lane] = make_float4(h.x, h.y, h.z, fabsf(h.x) + fabsf(h.y) + fabsf(h.z));
            S.olo[lane] = itab[g0 + lane].lo;
            for (int q = 0; q < nseg; q++)
                S.stack[q * nb + lane] =
                    ((unsigned)q << kSegShift) | ((unsigned)lane << kImgShift) | (unsigned)root;
        }
        int fc = nb * nseg, nc = 0;   // items on the stack, candidates (warp-uniform)
        while (fc > 0) {
            // 32 items while their children fit above the depth-first reserve,
            // fewer near it: one item at a time adds at most 7 per level
            const int k = min(min(32, fc), max(1, (kStack - kReserve - fc) / 7));
            __syncwarp();
            const bool have = lane < k;
            const unsigned item = have ? S.stack[fc - k + lane] : 0u;
            const int e = (int)(item & kEntMask), img = (int)((item >> kImgShift) & kImgMask);
            const int sg = (int)(item >> kSegShift);
            fc -= k;
            __syncwarp();
            if (kCount) tested += (unsigned)k;
            bool open = false, cand = false;
            uint32_t cm = 0;
            int4 clo = make_int4(0, 0, 0, 0), chi = clo;
            float4 ra, rb, o;
            if (have) {
                const Segment& B = S.seg[sg];
                if (kCount) visits += (unsigned)B.count;
                ld_pair(A.ra, e, ra, rb);
                o = S.ohi[img];
                // float boxes and offsets: each subtraction below is good to
                // 2e-7 of the absolute values that enter it
                const float lim = B.reach + 4e-7f * (B.size + o.w);
                const bool leaf = __float_as_int(ra.w) < 0;
                const int top = leaf ? ~__float_as_int(ra.w) : __float_as_int(ra.w);
                // leaf: its position hi as a box of no extent (lo is below 6e-8 of it)
                const float ux = leaf ? ra.x : rb.x, uy = leaf ? ra.y : rb.y, uz = leaf ? ra.z : rb.z;
                const float ex = fmaxf(fmaxf(ra.x + (o.x - B.hx), (B.lx - o.x) - ux), 0.f);
                const float ey = fmaxf(fmaxf(ra.y + (o.y - B.hy), (B.ly - o.y) - uy), 0.f);
                const float ez = fmaxf(fmaxf(ra.z + (o.z - B.hz), (B.lz - o.z) - uz), 0.f);
                const float d2 = fmaf(ez, ez, fmaf(ey, ey, ex * ex));
                const bool close = top > B.min_slot && d2 < lim * lim;
                cand = close && leaf;
                open = close && !leaf;
                if (open) {
                    cm = __ldg(&A.e_cmask[e]);
                    asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                        : "=r"(clo.x), "=r"(clo.y), "=r"(clo.z), "=r"(clo.w), "=r"(chi.x), "=r"(chi.y),
                          "=r"(chi.z), "=r"(chi.w)
                        : "l"(A.e_child + 8 * (size_t)e));
                }
            }
            // candidates: position of the image, x + o as a hi/lo pair
            const unsigned mc = __ballot_sync(kFull, cand);
            auto put = [&](int at, int im, int q, const float4& pa, const float4& pb, int slot) {
                const float4 h = S.ohi[im], l = S.olo[im];
                float hx, lx, hy, ly, hz, lz;
                sub_hilo(pa.x, pb.x, -h.x, -l.x, hx, lx);
                sub_hilo(pa.y, pb.y, -h.y, -l.y, hy, ly);
                sub_hilo(pa.z, pb.z, -h.z, -l.z, hz, lz);
                S.ca[at] = make_float4(hx, hy, hz, pb.w);
                S.cb[at] = make_float4(lx, ly, lz, __int_as_float(slot));
                S.cimg[at] = (q << 16) | (g0 + im);
            };
            // room for 32 more
            auto make_room = [&]() {
                if (nc < 32) return;
                __syncwarp();
                test_candidates(A, S, nc, seg, T, itab, nh);
                __syncwarp();
                nc = 0;
            };
            make_room();
            if (cand) put(nc + __popc(mc & lt), img, sg, ra, rb, ~__float_as_int(ra.w));
            nc += __popc(mc);
            // an opened depth-21 group has no child table: its members are the
            // leaves up to its skip entry (any number: 32 at a time)
            for (unsigned m = __ballot_sync(kFull, open && cm == 0); m; m &= m - 1) {
                const unsigned gi = __shfl_sync(kFull, item, __ffs(m) - 1);
                const int ge = (int)(gi & kEntMask), end = A.e_skip[ge];
                const int gm = (int)((gi >> kImgShift) & kImgMask), gs = (int)(gi >> kSegShift);
                for (int c0 = ge + 1; c0 < end; c0 += 32) {
                    const int c = c0 + lane;
                    if (kCount) tested += (unsigned)min(32, end - c0);
                    make_room();
                    if (c < end) {
                        float4 pa, pb;
                        ld_pair(A.ra, c, pa, pb);
                        put(nc + lane, gm, gs, pa, pb, ~__float_as_int(pa.w));
                        if (kCount) visits += (unsigned)S.seg[gs].count;
                    }
                    nc += min(32, end - c0);
                }
            }
            // a lane's place among the pushed children, from ballots of the
            // bits of the counts (0 .. 8)
            const uint32_t nch = open ? (uint32_t)__popc(cm) : 0u;
            const unsigned b0 = __ballot_sync(kFull, nch & 1u), b1 = __ballot_sync(kFull, nch & 2u);
            const unsigned b2 = __ballot_sync(kFull, nch & 4u), b3 = __ballot_sync(kFull, nch & 8u);
            if (nch) {
                int pos = fc + __popc(b0 & lt) + 2 * __popc(b1 & lt) + 4 * __popc(b2 & lt) + 8 * __popc(b3 & lt);
                const unsigned gb = item & ~(unsigned)kEntMask;
                if (cm & 1u) S.stack[pos++] = gb | (unsigned)clo.x;
                if (cm & 2u) S.stack[pos++] = gb | (unsigned)clo.y;
                if (cm & 4u) S.stack[pos++] = gb | (unsigned)clo.z;
                if (cm & 8u) S.stack[pos++] = gb | (unsigned)clo.w;
                if (cm & 16u) S.stack[pos++] = gb | (unsigned)chi.x;
                if (cm & 32u) S.stack[pos++] = gb | (unsigned)chi.y;
                if (cm & 64u) S.stack[pos++] = gb | (unsigned)chi.z;
                if (cm & 128u) S.stack[pos++] = gb | (unsigned)chi.w;
            }
            fc += __popc(b0) + 2 * __popc(b1) + 4 * __popc(b2) + 8 * __popc(b3);
        }
        __syncwarp();
        test_candidates(A, S, nc, seg, T, itab, nh);
        __syncwarp();
    }
    record_pairs(A, S, 0, nh, itab);
    __syncwarp();
}

template <bool kCount>
__device__ __forceinline__ void collide(const CollArgs& A, SearchSmem& S, int wbase, int n,
                                        unsigned long long& visits, unsigned long long& iters) {
    const int lane = threadIdx.x & 31;
    const bool valid = lane < A.width && wbase + lane < n;
    const int i = valid ? wbase + lane : n - 1;
    const int box = A.box[i];
    const int root = A.box_root[box];   // -1: a removed particle, searches nothing
    Target T;
    T.slot = i;
    split_d(A.x[i], T.hx, T.lx);
    split_d(A.y[i], T.hy, T.ly);
    split_d(A.z[i], T.hz, T.lz);
    T.r = (float)A.r[i];
    unsigned todo = __ballot_sync(kFull, valid && root >= 0);
    while (todo) {
        // up to kSegs compact parts of the targets left, all in one box
        int nseg = 0, mine = -1;
        const int lead = __ffs(todo) - 1, b = __shfl_sync(kFull, box, lead), r = __shfl_sync(kFull, root, lead);
        const unsigned here = __ballot_sync(kFull, box == b);
        __syncwarp();   // the last search has read its segments
        for (; (todo & here) && nseg < kSegs; nseg++) {
            unsigned seg = here & todo;
            const int first = __ffs(seg) - 1;
            bool in = (seg >> lane) & 1u;
            const float reach = (redux_max(in ? T.r : 0.f) + A.rmaxf) * 1.0001f;
            Box3 B = warp_box(in, T.hx, T.hy, T.hz);
            // cut it at the widest gap along its widest side while that leaves
            // less to search; the other part stays in todo
            while (seg & (seg - 1)) {
                const float wx = B.hx - B.lx, wy = B.hy - B.ly, wz = B.hz - B.lz, w = fmaxf(wx, fmaxf(wy, wz));
                if (!(w > 4.f * reach)) break;
                const float c = w == wx ? T.hx : w == wy ? T.hy : T.hz;
                float next = __int_as_float(0x7f800000);   // the nearest target further along, if any
                for (unsigned m = seg; m; m &= m - 1) {
                    const float o = __shfl_sync(kFull, c, __ffs(m) - 1);
                    if (o > c) next = fminf(next, o);
                }
                const float gap = in && next < __int_as_float(0x7f800000) ? next - c : 0.f;
                const float widest = redux_max(gap);
                if (!(widest > 2.f * reach)) break;
                const float cut = redux_min(gap == widest ? c : __int_as_float(0x7f800000));
                const bool lo = in && c <= cut;
                const Box3 B1 = warp_box(lo, T.hx, T.hy, T.hz), B2 = warp_box(in && !lo, T.hx, T.hy, T.hz);
                if (!(searched(B1, reach) + searched(B2, reach) < 0.75f * searched(B, reach))) break;
                const unsigned part = __ballot_sync(kFull, lo);
                const bool up = (part >> first & 1u) == 0u;   // go on with the first target's part
                seg &= up ? ~part : part;
                in = (seg >> lane) & 1u;
                B = up ? B2 : B1;
            }
            todo &= ~seg;
            if (in) mine = nseg;
            const int min_slot = (int)__reduce_min_sync(kFull, in ? (unsigned)i : 0x7fffffffu);
            if (lane == 0) {
                const float size = fmaxf(fabsf(B.lx), fabsf(B.hx)) + fmaxf(fabsf(B.ly), fabsf(B.hy)) +
                                   fmaxf(fabsf(B.lz), fabsf(B.hz));
                S.seg[nseg] = Segment{B.lx, B.hx, B.ly, B.hy, B.lz, B.hz, reach, size, min_slot, __popc(seg)};
            }
        }
        __syncwarp();
        search_segments<kCount>(A, S, nseg, mine, T, r, A.img + (size_t)b * A.nimg, visits, iters);
    }
}

template <bool kCount>
__global__ void __launch_bounds__(kMaxWalkBlock, 4) k_collide(CollArgs A) {
    __shared__ SearchSmem sm[kMaxWalkBlock / 32];
    const int n = sorted_n(A.ctl, A.ncap);
    const int ntile = (n + A.width - 1) / A.width, q = sm_queue(A.nq);
    unsigned long long visits = 0, iters = 0;
    for (int t = next_tile(A.tq, A.nq, q, ntile); t >= 0; t = next_tile(A.tq, A.nq, q, ntile))
        collide<kCount>(A, sm[threadIdx.x >> 5], t * A.width, n, visits, iters);
    if (kCount) {   // visits: per lane
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) visits += __shfl_down_sync(kFull, visits, o);
        if ((threadIdx.x & 31) == 0) {
            atomicAdd(&A.ctl->n_visit, visits);
            atomicAdd(&A.ctl->n_siter, iters);
        }
    }
}

}  // namespace

void collision_search_prepare() {
    walk_prepare_kernel((const void*)k_collide<false>);
    walk_prepare_kernel((const void*)k_collide<true>);
}

void collision_search(const Tree& T, const PSet& P, Ctl* ctl, const BoxP* boxes, const SimC& C,
                      const Pairs& PR, int half_step_offset, cudaStream_t s, int block, double rmax, bool count) {
    if (T.cap_n <= 0) return;
    block = (block == 64 || block == 256) ? block : 128;
    CollArgs A;
    A.rmaxf = (float)rmax;
    if ((double)A.rmaxf < rmax) A.rmaxf = nextafterf(A.rmaxf, FLT_MAX);
    A.x = P.x; A.y = P.y; A.z = P.z; A.r = P.r; A.id = P.id; A.box = P.box;
    A.ra = T.ra; A.rb = T.rb; A.box_root = T.box_root; A.e_skip = T.e_skip;
    A.e_child = T.e_child; A.e_cmask = T.e_cmask;
    A.ctl = ctl;
    A.pair_key = PR.key; A.pair_cap = PR.cap; A.ncap = T.cap_n;
    A.ngx = C.ngx; A.ngy = C.ngy; A.ngz = C.ngz;
    A.img = T.img;
    A.tq = T.tq;
    A.nq = T.nq;
    A.nimg = build_image_table(boxes, ctl, C, half_step_offset, T.img, s, T.tq, T.nq);
    A.width = T.cap_n <= kWidth4Max ? 4 : T.cap_n <= kWidth8Max ? 8 : 32;
    const int grid = walk_grid(count ? (const void*)k_collide<true> : (const void*)k_collide<false>, block,
                               ceil_div(T.cap_n, A.width));
    if (count) k_collide<true><<<grid, block, 0, s>>>(A);
    else k_collide<false><<<grid, block, 0, s>>>(A);
}

}  // namespace rb
