// rb_twalk.cu -- Barnes-Hut gravity walk with one warp per target, or for two
// (Sect. 4.2, Eq. 1): the lanes take the target's cells, not its neighbours.
//
// The walks of rb_walk.cu give each lane a target and step the warp through
// the union of 32 walks, one tree entry after the other: about 700-1200
// dependent record loads per warp.  With few targets that chain is the time
// (2400 particles: 75 warps, 262 us; 39 us here).  Here a warp owns one target and keeps
// a stack of (ghost image, entry) items, which starts with the root of every
// image.  Each round the lanes pop up to 32 items, test each with the target's
// own opening test, evaluate the accepted cells and leaves, and push the
// children of the opened cells: 16 rounds of independent loads (2400
// particles) instead of the chain.  Each target tests exactly the entries its own walk visits, so
// accepted sets and counts are those of the other walks.
//
// FP64: the opening test is decided in FP32 on the hi/lo records wherever that
// is safe (a band of 1e-5 around the threshold, and anything that overflows or
// underflows FP32, is decided in FP64 in the oracle's operation order), and
// accepted entries are queued, cells and leaves apart, and evaluated 32 at a
// time: on GB300 an FP64 warp instruction holds the SM's FP64 pipe 16 cycles
// however many lanes are active, so that pipe's time goes only to accepted
// terms in full warps.  Every FP64 walk takes this form,
// one target per warp.  65,537 targets
// (theta = 0.5, 9 images; 464 cells and 55 exact terms each): 2.20 ms, against
// 5.34 ms for a warp stepping through the union of 32 targets' walks; its
// accepted terms alone are 1.2e9 FP64 lane operations, 1.9 ms at two lanes
// per SM and clock.
//
// FP32: a warp takes two neighbouring targets at once (k_twalk32x2) where there
// are enough of them to fill the GPU.  An item carries the targets that visit it
// in its two upper bits; its records are read once for both, whose terms are one
// packed FP32 operation each, and its children are pushed for the targets that
// opened it, so each target still tests exactly the entries of its own walk.
// Neighbours' walks have most entries in common (the rounds of a pair, 22 at
// 20,000 and 24 at 60,000 targets, are 1.06 times those of one).  One target per warp is bound by instruction issue (64%
// of the slots) and the L1 wavefronts of its gathers (70%); pairs by the latency
// of the gathers with 24 warps per SM.  30,011 targets of the sheet: 215 -> 160
// us, 50,000: 345 -> 250, 5,000: 69 -> 49.  Loading the children before the
// terms are formed is 5% of that, and leaves with multipole records of their own,
// which spare the selection, took it to 154, 242 and 47; 16 warps per SM (no spills) take 20% longer,
// 32 warps 8%.
#include <algorithm>
#include <type_traits>

#include "rb_fp64.cuh"
#include "rb_walk.cuh"

namespace rb {
namespace {

constexpr int kEntBits = 25;                        // entries < 2 (2^24 - 1) < 2^25
constexpr int kEntMask = (1 << kEntBits) - 1;
constexpr int kImgBatch = 32;                       // images whose items share the stack
constexpr int kStack = 512;
constexpr int kReserve = 160;                       // depth-first room: 7 siblings on each of 22 levels

constexpr int kUnit = 8;                            // targets a warp takes from a queue at once, at most

// FP32 targets from which a warp takes two at a time: 39 us both ways at 2,400
// in Morton order, 29 us for one against 37 for two at 1,000, 50 against 44 at
// 4,000.
constexpr int kPairMin = 3000;

struct TSmem32 {
    int stack[kStack];           // (image of the batch << kEntBits) | entry
    float4 txy[kImgBatch];       // negated target of each image: x, y hi; x, y lo
    float2 tz[kImgBatch];        // z hi, lo
    float2 sum[kUnit][3];        // results of the unit's targets: sums (hi, lo)
    int cnt[kUnit][4];           // accepted cells, exact terms, opening tests, slot
};
struct TSmem64 : TSmem32 {
    double t64[kImgBatch][3];    // the FP64 target point x - o
    int cells[64], leaves[64];   // accepted items not yet evaluated
    double sum64[kUnit][4];      // results of the unit's targets: sums, potential
};
template <bool k64>
using TSmem = std::conditional_t<k64, TSmem64, TSmem32>;

// Per-lane sums of one target; ends as the warp's total in every lane.
struct TSum {
    float sx, sy, sz, cx, cy, cz;   // FP32: Kahan sums of the flushed partial sums
    float fx, fy, fz;               // FP32: plain sums of the last <= 16 rounds
    double ax, ay, az, pot;         // FP64
    int ncell, nleaf, nmac;
};

// Per-lane totals over a warp's targets.
struct TTotal {
    unsigned ncell = 0, nmac = 0, nrecheck = 0, ncorr = 0, rounds = 0;
    unsigned long long nleaf = 0;
};

__device__ __forceinline__ void tsum_flush(TSum& L) {
    kadd(L.sx, L.cx, L.fx);
    kadd(L.sy, L.cy, L.fy);
    kadd(L.sz, L.cz, L.fz);
    L.fx = L.fy = L.fz = 0.f;
}

// The child entries of a cell's octants (slots of empty octants hold any value).
__device__ __forceinline__ void ld_children(const int32_t* e_child, int e, int4& lo, int4& hi) {
    asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(lo.x), "=r"(lo.y), "=r"(lo.z), "=r"(lo.w), "=r"(hi.x), "=r"(hi.y), "=r"(hi.z), "=r"(hi.w)
        : "l"(e_child + 8 * (size_t)e));
}

// One queued cell: monopole + quadrupole (reading R3),
// a = (M invs^3 + 2.5 (d.Qd) inv^7) d - inv^5 Q d.
template <bool kQuad, bool kSoft, bool kPot, typename Smem>
__device__ __forceinline__ void cell64(const GravArgs& A, const Smem& S, int item, TSum& L) {
    const int e = item & kEntMask;
    const double* t = S.t64[item >> kEntBits];
    const double4_32a a = ld_d4(&A.d_a[e]);
    const double4_32a q0 = ld_d4(&A.d_q0[e]);
    const double dx = a.x - t[0], dy = a.y - t[1], dz = a.z - t[2];
    const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
    const double inv = rsqrt64(r2);
    const double inv2 = inv * inv;
    if (kQuad && !kSoft) {
        // inv^5 ((M r^2 + 2.5 (d.Qd) inv^2) d - Q d): two operations fewer
        const double4_32a q1 = ld_d4(&A.d_q1[e]);
        const double qx = fma(q1.y, dz, fma(q1.x, dy, q0.y * dx));
        const double qy = fma(q1.z, dz, fma(q0.z, dy, q1.x * dx));
        const double qz = fma(q0.w, dz, fma(q1.z, dy, q1.y * dx));
        const double dqd = fma(dz, qz, fma(dy, qy, dx * qx));
        const double inv5 = inv2 * inv2 * inv;
        const double g = fma(2.5, dqd * inv2, q0.x * r2);
        L.ax = fma(inv5, fma(g, dx, -qx), L.ax);
        L.ay = fma(inv5, fma(g, dy, -qy), L.ay);
        L.az = fma(inv5, fma(g, dz, -qz), L.az);
        if (kPot) L.pot = fma(-q0.x, inv, fma(-0.5 * dqd, inv5, L.pot));
        return;
    }
    const double invs = kSoft ? rsqrt64(r2 + A.soft2) : inv;
    double fc = q0.x * (kSoft ? invs * invs * invs : inv2 * inv);
    if (kPot) L.pot = fma(-q0.x, invs, L.pot);
    if (kQuad) {
        const double4_32a q1 = ld_d4(&A.d_q1[e]);
        const double qx = fma(q1.y, dz, fma(q1.x, dy, q0.y * dx));
        const double qy = fma(q1.z, dz, fma(q0.z, dy, q1.x * dx));
        const double qz = fma(q0.w, dz, fma(q1.z, dy, q1.y * dx));
        const double dqd = fma(dz, qz, fma(dy, qy, dx * qx));
        const double inv5 = inv2 * inv2 * inv;
        const double s5 = dqd * inv5;
        fc = fma(2.5 * inv2, s5, fc);
        L.ax = fma(-inv5, qx, L.ax);
        L.ay = fma(-inv5, qy, L.ay);
        L.az = fma(-inv5, qz, L.az);
        if (kPot) L.pot = fma(-0.5, s5, L.pot);
    }
    L.ax = fma(fc, dx, L.ax);
    L.ay = fma(fc, dy, L.ay);
    L.az = fma(fc, dz, L.az);
}

// One queued leaf: exact term of Eq. 1 (the record holds -m).
template <bool kSoft, bool kPot, typename Smem>
__device__ __forceinline__ void leaf64(const GravArgs& A, const Smem& S, int item, TSum& L) {
    const double4_32a a = ld_d4(&A.d_a[item & kEntMask]);
    const double* t = S.t64[item >> kEntBits];
    const double dx = a.x - t[0], dy = a.y - t[1], dz = a.z - t[2];
    const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
    const double inv = rsqrt64(kSoft ? r2 + A.soft2 : r2);
    const double f = -a.w * (inv * inv * inv);
    L.ax = fma(f, dx, L.ax);
    L.ay = fma(f, dy, L.ay);
    L.az = fma(f, dz, L.az);
    if (kPot) L.pot = fma(a.w, inv, L.pot);
}

// Appends the lanes' items (those with want) to a queue of n items; a full
// warp of them is evaluated at once.  Returns the new length (< 32).
template <typename F>
__device__ __forceinline__ int queue64(int* q, int n, bool want, int item, unsigned lt, F&& eval) {
    const unsigned m = __ballot_sync(kFull, want);
    if (want) q[n + __popc(m & lt)] = item;
    n += __popc(m);
    if (n >= 32) {
        __syncwarp();
        n -= 32;
        eval(q[n + (threadIdx.x & 31)]);
        __syncwarp();
    }
    return n;
}

// Network inputs of an accepted band cell (the oracle's definition, in FP32
// from the walk records; r = p - com = -d) as a BF16 row of the warp's queue.
__device__ __forceinline__ void learn_row(const GravArgs& A, LearnQ& Q, int pos, int e, const float4& ra,
                                          const float4& rb, const float4& q0, const float4& q1, float dx,
                                          float dy, float dz, float inv) {
    const float4 ch = __ldg(&A.rc_hi[e]);
    const float4 cl = __ldg(&A.rc_lo[e]);
    const float w = ch.w, rw = 1.f / w;
    const float hx = -dx * inv, hy = -dy * inv, hz = -dz * inv;
    const float sc = rw * rw / q0.x;
    const float qxx = q0.y * sc, qyy = q0.z * sc, qzz = q0.w * sc;
    const float qxy = q1.x * sc, qxz = q1.y * sc, qyz = q1.z * sc;
    const float ux = qxx * hx + qxy * hy + qxz * hz;
    const float uy = qxy * hx + qyy * hy + qyz * hz;
    const float uz = qxz * hx + qyz * hy + qzz * hz;
    uint4 lo, hi;
    lo.x = mlp::pack2(hx, hy);
    lo.y = mlp::pack2(hz, w * inv);
    lo.z = mlp::pack2(__log2f((float)__ldg(&A.e_count[e])) * 0.30102999566f,
                      ((ra.x - ch.x) + (rb.x - cl.x)) * rw - 0.5f);
    lo.w = mlp::pack2(((ra.y - ch.y) + (rb.y - cl.y)) * rw - 0.5f,
                      ((ra.z - ch.z) + (ra.w - cl.z)) * rw - 0.5f);
    hi.x = mlp::pack2(hx * ux + hy * uy + hz * uz, sqrtf(ux * ux + uy * uy + uz * uz));
    hi.y = mlp::pack2(qxx * qxx + qyy * qyy + qzz * qzz + 2.f * (qxy * qxy + qxz * qxz + qyz * qyz),
                      qxx * (qyy * qzz - qyz * qyz) - qxy * (qxy * qzz - qyz * qxz) +
                          qxz * (qxy * qyz - qyy * qxz));
    hi.z = 0u;
    hi.w = 0u;
    reinterpret_cast<uint4*>(&Q.X[pos][0])[0] = lo;
    reinterpret_cast<uint4*>(&Q.X[pos][0])[1] = hi;
    Q.unit[pos] = q0.x * (inv * inv);
}

// Rows r0 .. r0 + 15 of the queue through the network; lane k < 16 adds the
// output of row r0 + k (all rows belong to the warp's target).
__device__ __forceinline__ void learn_rows(LearnQ& Q, const mlp::Packed& w, int r0, int lane, TSum& L) {
    __syncwarp();
    float out[4];
    mlp::forward_packed(w, &Q.X[r0][0], out);
    const int g = lane >> 2, q = lane & 3;
    if (q < 2) {
        Q.Y[g][2 * q] = out[0];
        Q.Y[g][2 * q + 1] = out[1];
        Q.Y[g + 8][2 * q] = out[2];
        Q.Y[g + 8][2 * q + 1] = out[3];
    }
    __syncwarp();
    if (lane < 16) {
        const float u = Q.unit[r0 + lane];
        L.fx = fmaf(u, Q.Y[lane][0], L.fx);
        L.fy = fmaf(u, Q.Y[lane][1], L.fy);
        L.fz = fmaf(u, Q.Y[lane][2], L.fz);
    }
    __syncwarp();
}

// Warp totals of hi/lo float pairs (two-sum: the low parts keep what the high
// parts lose), in a fixed butterfly order; every lane ends with the total.
__device__ __forceinline__ void reduce_hilo(float& hi, float& lo) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float h2 = __shfl_xor_sync(kFull, hi, o), l2 = __shfl_xor_sync(kFull, lo, o);
        const float s = hi + h2;
        const float b = s - hi;
        const float err = (hi - (s - b)) + (h2 - b);
        hi = s;
        lo = (lo + l2) + err;
    }
}

__device__ __forceinline__ double warp_sum64(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

template <bool kQuad, bool kInside, bool kSoft, bool kPot, bool k64, bool kLearn>
__device__ __forceinline__ void walk_target(const GravArgs& A, TSmem<k64>& S, LearnQ* LQ, const mlp::Packed* W,
                                            int i, TSum& L, TTotal& N) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    L.sx = L.sy = L.sz = L.cx = L.cy = L.cz = 0.f;
    L.fx = L.fy = L.fz = 0.f;
    L.ax = L.ay = L.az = L.pot = 0.0;
    L.ncell = L.nleaf = L.nmac = 0;
    const int box = A.box[i];
    const int root = A.box_root[box];
    if (root < 0) return;
    const int self = A.leaf_of[i];
    // the target as hi/lo floats: its own leaf's record holds them
    const float4 pa = A.ra[self], pb = A.rb[self];
    const ImgTab* itab = A.img + (size_t)box * A.nimg;
    const int centre = (A.ngx * (2 * A.ngy + 1) + A.ngy) * (2 * A.ngz + 1) + A.ngz;
    int rounds = 0;               // warp-uniform
    int nc = 0, nl = 0, qn = 0;   // queued cells, leaves (k64), network rows (kLearn)
    auto do_cell = [&](auto it) { cell64<kQuad, kSoft, kPot>(A, S, it, L); };
    auto do_leaf = [&](auto it) { leaf64<kSoft, kPot>(A, S, it, L); };
    for (int g0 = 0; g0 < A.nimg; g0 += kImgBatch) {
        const int nb = min(kImgBatch, A.nimg - g0);
        __syncwarp();
        if (lane < nb) {
            const ImgTab& T = itab[g0 + lane];
            const float4 oh = T.hi, ol = T.lo;
            float th, tl, uh, ul, vh, vl;
            sub_hilo(pa.x, pb.x, oh.x, ol.x, th, tl);
            sub_hilo(pa.y, pb.y, oh.y, ol.y, uh, ul);
            sub_hilo(pa.z, pa.w, oh.z, ol.z, vh, vl);
            S.txy[lane] = make_float4(-th, -uh, -tl, -ul);
            S.tz[lane] = make_float2(-vh, -vl);
            if constexpr (k64) {
                S.t64[lane][0] = __dsub_rn(A.x[i], T.ox);
                S.t64[lane][1] = __dsub_rn(A.y[i], T.oy);
                S.t64[lane][2] = __dsub_rn(A.z[i], T.oz);
            }
            S.stack[lane] = (lane << kEntBits) | root;
        }
        int fc = nb;   // items on the stack (warp-uniform)
        // the target's own leaf is no term of the central image
        const int self_item = ((centre - g0) << kEntBits) | self;   // matches no item of another batch
        const bool own = centre >= g0 && centre < g0 + nb;
        while (fc > 0) {
            // 32 items while their children fit above the depth-first reserve,
            // fewer near it: one item at a time adds at most 7 per level
            const int k = min(min(32, fc), max(1, (kStack - kReserve - fc) / 7));
            __syncwarp();
            const int item = lane < k ? S.stack[fc - k + lane] : -1;
            fc -= k;
            __syncwarp();
            bool open = false, acc = false, leaf = false, want = false;
            int e = 0;
            uint32_t cm = 0;
            float4 ra, rb, q0, q1;
            float dx = 0.f, dy = 0.f, dz = 0.f, r2 = 0.f, inv = 0.f;
            if (item >= 0) {
                e = item & kEntMask;
                const int g = item >> kEntBits;
                ld_pair(A.ra, e, ra, rb);
                if (!k64) ld_pair(A.rq0, e, q0, q1);   // of a leaf: its mass, Q = 0
                const float4 t = S.txy[g];
                const float2 tz = S.tz[g];
                rec_diff(ra, rb, make_float2(t.x, t.y), make_float2(t.z, t.w), tz, dx, dy, dz, r2);
                const float crit = rb.z;   // leaf: -m; cell: (w / theta)^2
                leaf = __float_as_int(crit) < 0;
                if (leaf) {
                    acc = !(own && item == self_item);
                    L.nleaf += acc;
                } else {
                    L.nmac++;
                    acc = crit < r2;
                    // also when r2 or crit leaves FP32's range (inf, NaN, tiny)
                    if (!(fabsf(crit - r2) > fmaf(1e-5f, r2, 1e-35f))) {
                        const ImgTab& T = itab[g0 + g];
                        acc = mac64(ld_d4(&A.d_a[e]), A.theta2, __dsub_rn(A.x[i], T.ox),
                                    __dsub_rn(A.y[i], T.oy), __dsub_rn(A.z[i], T.oz));
                        N.nrecheck++;
                    }
                    if (kInside && acc) {
                        const float4 ch = __ldg(&A.rc_hi[e]);
                        const float4 cl = __ldg(&A.rc_lo[e]);
                        const float ux = (-t.x - ch.x) + (-t.z - cl.x);
                        const float uy = (-t.y - ch.y) + (-t.w - cl.y);
                        const float uz = (-tz.x - ch.z) + (-tz.y - cl.z);
                        const float w = ch.w;
                        const float mx = fminf(fminf(ux, w - ux), fminf(fminf(uy, w - uy), fminf(uz, w - uz)));
                        if (!(fabsf(mx) > fmaf(1e-5f, w, 1e-35f))) {
                            const ImgTab& T = itab[g0 + g];
                            acc = !inside64(ld_d4(&A.d_c[e]), __dsub_rn(A.x[i], T.ox),
                                            __dsub_rn(A.y[i], T.oy), __dsub_rn(A.z[i], T.oz));
                            N.nrecheck++;
                        } else if (mx > 0.f) {
                            acc = false;
                        }
                    }
                    open = !acc;
                    L.ncell += acc;
                }
                if (!k64 && acc) {
                    // a leaf is the cell with Q = 0; its distance may be zero when softened
                    inv = rsqrt_nr(kSoft && leaf ? r2 + A.soft2f : r2);
                    const float inv2 = inv * inv;
                    const float invs = kSoft ? rsqrt_nr(r2 + A.soft2f) : inv;
                    float f = q0.x * (kSoft ? invs * invs * invs : inv2 * inv);
                    if (kQuad) {
                        const float qx = fmaf(q1.y, dz, fmaf(q1.x, dy, q0.y * dx));
                        const float qy = fmaf(q1.z, dz, fmaf(q0.z, dy, q1.x * dx));
                        const float qz = fmaf(q0.w, dz, fmaf(q1.z, dy, q1.y * dx));
                        const float dqd = fmaf(dz, qz, fmaf(dy, qy, dx * qx));
                        // none for a leaf: r^-5 and r^-7 overflow at distances where its term does not
                        const float inv5 = leaf ? 0.f : inv2 * inv2 * inv;
                        f = fmaf(2.5f, dqd * (inv5 * inv2), f);
                        L.fx = fmaf(-inv5, qx, L.fx);
                        L.fy = fmaf(-inv5, qy, L.fy);
                        L.fz = fmaf(-inv5, qz, L.fz);
                    }
                    L.fx = fmaf(f, dx, L.fx);
                    L.fy = fmaf(f, dy, L.fy);
                    L.fz = fmaf(f, dz, L.fz);
                    if (kLearn) want = !leaf && crit > A.band_scale * r2;
                }
            }
            // an opened cell's children (used after the terms below)
            int4 clo = make_int4(0, 0, 0, 0), chi = clo;
            if (open) {
                cm = __ldg(&A.e_cmask[e]);
                ld_children(A.e_child, e, clo, chi);
            }
            if constexpr (k64) {
                nc = queue64(S.cells, nc, acc && !leaf, item, lt, do_cell);
                nl = queue64(S.leaves, nl, acc && leaf, item, lt, do_leaf);
            }
            if (kLearn) {
                const unsigned m = __ballot_sync(kFull, want);
                if (m) {
                    if (want) {
                        learn_row(A, *LQ, qn + __popc(m & lt), e, ra, rb, q0, q1, dx, dy, dz, inv);
                        N.ncorr++;
                    }
                    qn += __popc(m);
                    while (qn >= 16) {
                        qn -= 16;
                        learn_rows(*LQ, *W, qn, lane, L);
                    }
                }
            }
            // children of the opened cells; a depth-21 group has no child
            // table: its members, the entries up to its skip entry, are
            // exact terms (any number of them: 32 at a time, not stacked)
            for (unsigned m = __ballot_sync(kFull, open && cm == 0); m; m &= m - 1) {
                const int src = __ffs(m) - 1;
                const int ge = __shfl_sync(kFull, e, src), gi = __shfl_sync(kFull, item, src);
                const int end = A.e_skip[ge], g = gi >> kEntBits;
                const float4 t = S.txy[g];
                const float2 tz = S.tz[g];
                for (int c0 = ge + 1; c0 < end; c0 += 32) {
                    const int c = c0 + lane, it = (g << kEntBits) | c;
                    const bool term = c < end && !(own && it == self_item);
                    L.nleaf += term;
                    if constexpr (k64) {
                        nl = queue64(S.leaves, nl, term, it, lt, do_leaf);
                    } else if (term) {
                        const float4 ga = __ldg(&A.ra[c]);
                        const float4 gb = __ldg(&A.rb[c]);
                        float ex, ey, ez, s2;
                        rec_diff(ga, gb, make_float2(t.x, t.y), make_float2(t.z, t.w), tz, ex, ey, ez, s2);
                        const float iv = rsqrt_nr(kSoft ? s2 + A.soft2f : s2);
                        const float f = -gb.z * (iv * iv * iv);
                        L.fx = fmaf(f, ex, L.fx);
                        L.fy = fmaf(f, ey, L.fy);
                        L.fz = fmaf(f, ez, L.fz);
                    }
                    if (!k64) tsum_flush(L);
                }
            }
            // a lane's place among the pushed children, from ballots of the
            // bits of the counts (0 .. 8)
            const uint32_t nch = open ? (uint32_t)__popc(cm) : 0u;
            const unsigned b0 = __ballot_sync(kFull, nch & 1u), b1 = __ballot_sync(kFull, nch & 2u);
            const unsigned b2 = __ballot_sync(kFull, nch & 4u), b3 = __ballot_sync(kFull, nch & 8u);
            if (nch) {
                int pos = fc + __popc(b0 & lt) + 2 * __popc(b1 & lt) + 4 * __popc(b2 & lt) + 8 * __popc(b3 & lt);
                const int gb = item & ~kEntMask;
                if (cm & 1u) S.stack[pos++] = gb | clo.x;
                if (cm & 2u) S.stack[pos++] = gb | clo.y;
                if (cm & 4u) S.stack[pos++] = gb | clo.z;
                if (cm & 8u) S.stack[pos++] = gb | clo.w;
                if (cm & 16u) S.stack[pos++] = gb | chi.x;
                if (cm & 32u) S.stack[pos++] = gb | chi.y;
                if (cm & 64u) S.stack[pos++] = gb | chi.z;
                if (cm & 128u) S.stack[pos++] = gb | chi.w;
            }
            fc += __popc(b0) + 2 * __popc(b1) + 4 * __popc(b2) + 8 * __popc(b3);
            if (!k64 && (++rounds & 15) == 0) tsum_flush(L);
        }
        if constexpr (k64) {
            // the queues refer to this batch's target points
            __syncwarp();
            if (lane < nc) do_cell(S.cells[lane]);
            if (lane < nl) do_leaf(S.leaves[lane]);
            nc = nl = 0;
        }
    }
    if (kLearn && qn > 0) {
        // the last partial tile: empty rows have zero inputs and no weight
        if (lane >= qn && lane < 16) {
            reinterpret_cast<uint4*>(&LQ->X[lane][0])[0] = make_uint4(0u, 0u, 0u, 0u);
            reinterpret_cast<uint4*>(&LQ->X[lane][0])[1] = make_uint4(0u, 0u, 0u, 0u);
            LQ->unit[lane] = 0.f;
        }
        learn_rows(*LQ, *W, 0, lane, L);
    }
    if (k64) {
        L.ax = warp_sum64(L.ax);
        L.ay = warp_sum64(L.ay);
        L.az = warp_sum64(L.az);
        if (kPot) L.pot = warp_sum64(L.pot);
    } else {
        tsum_flush(L);
        L.cx = -L.cx;
        L.cy = -L.cy;
        L.cz = -L.cz;
        reduce_hilo(L.sx, L.cx);
        reduce_hilo(L.sy, L.cy);
        reduce_hilo(L.sz, L.cz);
    }
    N.ncell += L.ncell;
    N.nleaf += L.nleaf;
    N.nmac += L.nmac;
    N.rounds += rounds;
    L.ncell = __reduce_add_sync(kFull, L.ncell);
    L.nleaf = __reduce_add_sync(kFull, L.nleaf);
    L.nmac = __reduce_add_sync(kFull, L.nmac);
}

__device__ __forceinline__ unsigned long long warp_total(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFull, v, o);
    return v;
}

// Units of `per` (<= kUnit) consecutive targets in tile order, from the
// per-SM queues; the warp walks them one after the other, then lane u writes
// the result of target u.
template <bool kQuad, bool kInside, bool kSoft, bool kPot, bool k64, bool kLearn>
__device__ __forceinline__ void target_units(const GravArgs& A, int per, TSmem<k64>& S, LearnQ* LQ,
                                             const mlp::Packed* W) {
    const int lane = threadIdx.x & 31;
    const int n = sorted_n(A.ctl, A.ncap);
    const int nunit = (n + per - 1) / per, q = sm_queue(A.nq);
    TTotal N;
    for (int u = next_tile(A.tq, A.nq, q, nunit); u >= 0; u = next_tile(A.tq, A.nq, q, nunit)) {
        const int j0 = u * per, cnt = min(per, n - j0);
        for (int j = 0; j < cnt; j++) {
            const int i = tile_slot(A.order, j0 + j);
            TSum L;
            walk_target<kQuad, kInside, kSoft, kPot, k64, kLearn>(A, S, LQ, W, i, L, N);
            if (lane == 0) {
                if constexpr (k64) {
                    S.sum64[j][0] = L.ax;
                    S.sum64[j][1] = L.ay;
                    S.sum64[j][2] = L.az;
                    if (kPot) S.sum64[j][3] = L.pot;
                } else {
                    S.sum[j][0] = make_float2(L.sx, L.cx);
                    S.sum[j][1] = make_float2(L.sy, L.cy);
                    S.sum[j][2] = make_float2(L.sz, L.cz);
                }
                S.cnt[j][0] = L.ncell;
                S.cnt[j][1] = L.nleaf;
                S.cnt[j][2] = L.nmac;
                S.cnt[j][3] = i;
            }
        }
        __syncwarp();
        if (lane < cnt) {
            const int i = S.cnt[lane][3];
            double a[3];
#pragma unroll
            for (int c = 0; c < 3; c++) {
                if constexpr (k64) a[c] = S.sum64[lane][c];
                else a[c] = (double)S.sum[lane][c].x + (double)S.sum[lane][c].y;
            }
            A.out.ax[i] = A.G * a[0];
            A.out.ay[i] = A.G * a[1];
            A.out.az[i] = A.G * a[2];
            if constexpr (kPot) A.out.phi[i] = A.G * S.sum64[lane][3];
            if (A.out.ncell) {
                A.out.ncell[i] = S.cnt[lane][0];
                A.out.nleaf[i] = S.cnt[lane][1];
                A.out.nmac[i] = S.cnt[lane][2];
            }
        }
        __syncwarp();
    }
    const unsigned long long c0 = warp_total(N.ncell), c1 = warp_total(N.nleaf), c2 = warp_total(N.nmac);
    const unsigned long long c3 = warp_total(N.nrecheck), c4 = kLearn ? warp_total(N.ncorr) : 0;
    if (lane == 0 && c1 + c2) {
        atomicAdd(&A.ctl->n_cell, c0);
        atomicAdd(&A.ctl->n_leaf, c1);
        atomicAdd(&A.ctl->n_mac, c2);
        if (!k64) {
            atomicAdd(&A.ctl->n_recheck, c3);
            atomicAdd(&A.ctl->n_iter, (unsigned long long)N.rounds);
        }
        if (kLearn) atomicAdd(&A.ctl->req_count, (int)c4);
    }
}

// ---- two targets per warp (FP32) ----

// An item's upper bits: image of the batch, then the targets that visit it.
constexpr int kImgBits = 5;
constexpr unsigned kItemMask = (1u << (kEntBits + kImgBits)) - 1u;   // entry and image
constexpr int kWhoShift = kEntBits + kImgBits;
static_assert(kImgBatch <= 1 << kImgBits && kWhoShift == 30, "two bits are left for the targets");

struct PSmem {
    unsigned stack[kStack];
    // negated targets of each image: x of both targets hi, then lo; y; z
    float4 tx[kImgBatch], ty[kImgBatch], tz[kImgBatch];
    float2 sum[kUnit][3];
    int cnt[kUnit][4];
};

// Per-lane sums of a pair of targets (x: the first, y: the second).
struct PSum {
    float2 fx, fy, fz;             // plain sums of the last <= 16 rounds
    float s[2][3], c[2][3];        // Kahan sums of the flushed partial sums
    int ncell[2], nleaf[2], nmac[2];
};

__device__ __forceinline__ void psum_flush(PSum& L) {
    kadd(L.s[0][0], L.c[0][0], L.fx.x);
    kadd(L.s[0][1], L.c[0][1], L.fy.x);
    kadd(L.s[0][2], L.c[0][2], L.fz.x);
    kadd(L.s[1][0], L.c[1][0], L.fx.y);
    kadd(L.s[1][1], L.c[1][1], L.fy.y);
    kadd(L.s[1][2], L.c[1][2], L.fz.y);
    L.fx = L.fy = L.fz = make_float2(0.f, 0.f);
}

__device__ __forceinline__ float2 two(float v) { return make_float2(v, v); }

// rsqrt_nr of both.
__device__ __forceinline__ float2 rsqrt2_nr(float2 x) {
    const float2 y = make_float2(rsqrtf(x.x), rsqrtf(x.y));
    return __fmul2_rn(y, __ffma2_rn(__fmul2_rn(__fmul2_rn(two(-0.5f), x), y), y, two(1.5f)));
}

// The records' differences to both targets, as rec_diff forms them.
__device__ __forceinline__ void rec_diff2(const float4& ra, const float4& rb, const float4& tx, const float4& ty,
                                          const float4& tz, float2& dx, float2& dy, float2& dz, float2& r2) {
    dx = __fadd2_rn(__fadd2_rn(two(ra.x), make_float2(tx.x, tx.y)), __fadd2_rn(two(rb.x), make_float2(tx.z, tx.w)));
    dy = __fadd2_rn(__fadd2_rn(two(ra.y), make_float2(ty.x, ty.y)), __fadd2_rn(two(rb.y), make_float2(ty.z, ty.w)));
    dz = __fadd2_rn(__fadd2_rn(two(ra.z), make_float2(tz.x, tz.y)), __fadd2_rn(two(ra.w), make_float2(tz.z, tz.w)));
    r2 = __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __fmul2_rn(dx, dx)));
}

// The walk of walk_target for the targets `who` (bit 0: i0, bit 1: i1) of one
// box, adding to L.
template <bool kQuad, bool kInside, bool kSoft>
__device__ __forceinline__ void walk_pair(const GravArgs& A, PSmem& S, int i0, int i1, unsigned who, int box, PSum& L,
                                          TTotal& N) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int root = A.box_root[box];
    if (root < 0) return;
    const int self0 = A.leaf_of[who & 1u ? i0 : i1], self1 = A.leaf_of[who & 2u ? i1 : i0];
    const ImgTab* itab = A.img + (size_t)box * A.nimg;
    const int centre = (A.ngx * (2 * A.ngy + 1) + A.ngy) * (2 * A.ngz + 1) + A.ngz;
    int rounds = 0;   // warp-uniform
    for (int g0 = 0; g0 < A.nimg; g0 += kImgBatch) {
        const int nb = min(kImgBatch, A.nimg - g0);
        __syncwarp();
        if (lane < nb) {
            const ImgTab& T = itab[g0 + lane];
            const float4 oh = T.hi, ol = T.lo;
            const float4 pa = A.ra[self0], pb = A.rb[self0], qa = A.ra[self1], qb = A.rb[self1];
            float h, l, h1, l1;
            sub_hilo(pa.x, pb.x, oh.x, ol.x, h, l);
            sub_hilo(qa.x, qb.x, oh.x, ol.x, h1, l1);
            S.tx[lane] = make_float4(-h, -h1, -l, -l1);
            sub_hilo(pa.y, pb.y, oh.y, ol.y, h, l);
            sub_hilo(qa.y, qb.y, oh.y, ol.y, h1, l1);
            S.ty[lane] = make_float4(-h, -h1, -l, -l1);
            sub_hilo(pa.z, pa.w, oh.z, ol.z, h, l);
            sub_hilo(qa.z, qa.w, oh.z, ol.z, h1, l1);
            S.tz[lane] = make_float4(-h, -h1, -l, -l1);
            S.stack[lane] = (who << kWhoShift) | ((unsigned)lane << kEntBits) | (unsigned)root;
        }
        int fc = nb;   // items on the stack (warp-uniform)
        // the targets' own leaves are no terms of the central image
        const bool own = centre >= g0 && centre < g0 + nb;
        const unsigned own0 = own ? ((unsigned)(centre - g0) << kEntBits) | (unsigned)self0 : ~0u;
        const unsigned own1 = own ? ((unsigned)(centre - g0) << kEntBits) | (unsigned)self1 : ~0u;
        while (fc > 0) {
            const int k = min(min(32, fc), max(1, (kStack - kReserve - fc) / 7));
            __syncwarp();
            const unsigned item = lane < k ? S.stack[fc - k + lane] : 0u;
            fc -= k;
            __syncwarp();
            unsigned opened = 0;   // targets that open the item's cell
            uint32_t cm = 0;
            int4 clo = make_int4(0, 0, 0, 0), chi = clo;
            int e = 0;
            if (item) {
                e = (int)(item & kEntMask);
                const int g = (int)((item & kItemMask) >> kEntBits);
                const bool on0 = item & (1u << kWhoShift), on1 = item & (2u << kWhoShift);
                float4 ra, rb;
                ld_pair(A.ra, e, ra, rb);
                const float4 tx = S.tx[g], ty = S.ty[g], tz = S.tz[g];
                float2 dx, dy, dz, r2;
                rec_diff2(ra, rb, tx, ty, tz, dx, dy, dz, r2);
                const float crit = rb.z;   // leaf: -m; cell: (w / theta)^2
                const bool leaf = __float_as_int(crit) < 0;
                bool a0, a1;
                if (leaf) {
                    a0 = on0 && (item & kItemMask) != own0;
                    a1 = on1 && (item & kItemMask) != own1;
                    L.nleaf[0] += a0;
                    L.nleaf[1] += a1;
                } else {
                    L.nmac[0] += on0;
                    L.nmac[1] += on1;
                    const ImgTab& T = itab[g0 + g];
                    // the FP64 test near the threshold, also when r2 or crit leaves FP32's range
                    auto accepted = [&](float d2, int i) {
                        if (fabsf(crit - d2) > fmaf(1e-5f, d2, 1e-35f)) return crit < d2;
                        N.nrecheck++;
                        return mac64(ld_d4(&A.d_a[e]), A.theta2, __dsub_rn(A.x[i], T.ox), __dsub_rn(A.y[i], T.oy),
                                     __dsub_rn(A.z[i], T.oz));
                    };
                    a0 = on0 && accepted(r2.x, i0);
                    a1 = on1 && accepted(r2.y, i1);
                    if (kInside && (a0 || a1)) {
                        const float4 ch = __ldg(&A.rc_hi[e]);
                        const float4 cl = __ldg(&A.rc_lo[e]);
                        auto outside = [&](float hx, float lx, float hy, float ly, float hz, float lz, int i) {
                            const float ux = (-hx - ch.x) + (-lx - cl.x);
                            const float uy = (-hy - ch.y) + (-ly - cl.y);
                            const float uz = (-hz - ch.z) + (-lz - cl.z);
                            const float w = ch.w;
                            const float mx =
                                fminf(fminf(ux, w - ux), fminf(fminf(uy, w - uy), fminf(uz, w - uz)));
                            if (fabsf(mx) > fmaf(1e-5f, w, 1e-35f)) return !(mx > 0.f);
                            N.nrecheck++;
                            return !inside64(ld_d4(&A.d_c[e]), __dsub_rn(A.x[i], T.ox), __dsub_rn(A.y[i], T.oy),
                                             __dsub_rn(A.z[i], T.oz));
                        };
                        a0 = a0 && outside(tx.x, tx.z, ty.x, ty.z, tz.x, tz.z, i0);
                        a1 = a1 && outside(tx.y, tx.w, ty.y, ty.w, tz.y, tz.w, i1);
                    }
                    L.ncell[0] += a0;
                    L.ncell[1] += a1;
                    opened = (on0 && !a0 ? 1u : 0u) | (on1 && !a1 ? 2u : 0u);
                    // the children on their way while the terms are formed
                    if (opened) {
                        cm = __ldg(&A.e_cmask[e]);
                        ld_children(A.e_child, e, clo, chi);
                    }
                }
                if (a0 || a1) {
                    // both targets' terms at once; a leaf is the cell with Q = 0, whose
                    // distance may be zero when softened
                    float4 q0, q1;
                    ld_pair(A.rq0, e, q0, q1);
                    const float2 rs = kSoft ? __fadd2_rn(r2, two(A.soft2f)) : r2;
                    const float2 inv = rsqrt2_nr(kSoft && leaf ? rs : r2);
                    const float2 inv2 = __fmul2_rn(inv, inv);
                    const float2 invs = kSoft ? rsqrt2_nr(rs) : inv;
                    float2 f = __fmul2_rn(two(q0.x), __fmul2_rn(kSoft ? __fmul2_rn(invs, invs) : inv2, invs));
                    if (kQuad) {
                        const float2 qx =
                            __ffma2_rn(two(q1.y), dz, __ffma2_rn(two(q1.x), dy, __fmul2_rn(two(q0.y), dx)));
                        const float2 qy =
                            __ffma2_rn(two(q1.z), dz, __ffma2_rn(two(q0.z), dy, __fmul2_rn(two(q1.x), dx)));
                        const float2 qz =
                            __ffma2_rn(two(q0.w), dz, __ffma2_rn(two(q1.z), dy, __fmul2_rn(two(q1.y), dx)));
                        const float2 dqd = __ffma2_rn(dz, qz, __ffma2_rn(dy, qy, __fmul2_rn(dx, qx)));
                        // none for a leaf, as above
                        const float2 inv5 = leaf ? two(0.f) : __fmul2_rn(__fmul2_rn(inv2, inv2), inv);
                        f = __ffma2_rn(two(2.5f), __fmul2_rn(dqd, __fmul2_rn(inv5, inv2)), f);
                        const float2 n5 = make_float2(a0 ? -inv5.x : 0.f, a1 ? -inv5.y : 0.f);
                        L.fx = __ffma2_rn(n5, qx, L.fx);
                        L.fy = __ffma2_rn(n5, qy, L.fy);
                        L.fz = __ffma2_rn(n5, qz, L.fz);
                    }
                    f = make_float2(a0 ? f.x : 0.f, a1 ? f.y : 0.f);
                    L.fx = __ffma2_rn(f, dx, L.fx);
                    L.fy = __ffma2_rn(f, dy, L.fy);
                    L.fz = __ffma2_rn(f, dz, L.fz);
                }
            }
            // members of an opened depth-21 group (no child table): exact terms, 32 at a time
            for (unsigned m = __ballot_sync(kFull, opened && cm == 0); m; m &= m - 1) {
                const int src = __ffs(m) - 1;
                const unsigned gi = __shfl_sync(kFull, item, src), go = __shfl_sync(kFull, opened, src);
                const int ge = (int)(gi & kEntMask), end = A.e_skip[ge];
                const unsigned gimg = gi & kItemMask & ~(unsigned)kEntMask;
                const float4 tx = S.tx[gimg >> kEntBits], ty = S.ty[gimg >> kEntBits], tz = S.tz[gimg >> kEntBits];
                for (int c0 = ge + 1; c0 < end; c0 += 32) {
                    const int c = c0 + lane;
                    const bool a0 = c < end && (go & 1u) && (gimg | (unsigned)c) != own0;
                    const bool a1 = c < end && (go & 2u) && (gimg | (unsigned)c) != own1;
                    L.nleaf[0] += a0;
                    L.nleaf[1] += a1;
                    if (a0 || a1) {
                        float4 pa, pb;
                        ld_pair(A.ra, c, pa, pb);
                        float2 dx, dy, dz, r2;
                        rec_diff2(pa, pb, tx, ty, tz, dx, dy, dz, r2);
                        const float2 iv = rsqrt2_nr(kSoft ? __fadd2_rn(r2, two(A.soft2f)) : r2);
                        float2 f = __fmul2_rn(two(-pb.z), __fmul2_rn(__fmul2_rn(iv, iv), iv));
                        f = make_float2(a0 ? f.x : 0.f, a1 ? f.y : 0.f);
                        L.fx = __ffma2_rn(f, dx, L.fx);
                        L.fy = __ffma2_rn(f, dy, L.fy);
                        L.fz = __ffma2_rn(f, dz, L.fz);
                    }
                    psum_flush(L);
                }
            }
            const uint32_t nch = opened ? (uint32_t)__popc(cm) : 0u;
            const unsigned b0 = __ballot_sync(kFull, nch & 1u), b1 = __ballot_sync(kFull, nch & 2u);
            const unsigned b2 = __ballot_sync(kFull, nch & 4u), b3 = __ballot_sync(kFull, nch & 8u);
            if (nch) {
                int pos = fc + __popc(b0 & lt) + 2 * __popc(b1 & lt) + 4 * __popc(b2 & lt) + 8 * __popc(b3 & lt);
                const unsigned gb = (opened << kWhoShift) | (item & kItemMask & ~(unsigned)kEntMask);
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
            if ((++rounds & 15) == 0) psum_flush(L);
        }
    }
    psum_flush(L);
    N.rounds += rounds;
}

// Units of `per` (even, <= kUnit) targets as in target_units, two at a time.
template <bool kQuad, bool kInside, bool kSoft>
__device__ __forceinline__ void pair_units(const GravArgs& A, int per, PSmem& S) {
    const int lane = threadIdx.x & 31;
    const int n = sorted_n(A.ctl, A.ncap);
    const int nunit = (n + per - 1) / per, q = sm_queue(A.nq);
    TTotal N;
    for (int u = next_tile(A.tq, A.nq, q, nunit); u >= 0; u = next_tile(A.tq, A.nq, q, nunit)) {
        const int j0 = u * per, cnt = min(per, n - j0);
        for (int j = 0; j < cnt; j += 2) {
            const bool both = j + 1 < cnt;
            const int i0 = tile_slot(A.order, j0 + j), i1 = both ? tile_slot(A.order, j0 + j + 1) : i0;
            const int box0 = A.box[i0], box1 = A.box[i1];
            PSum L;
            L.fx = L.fy = L.fz = make_float2(0.f, 0.f);
#pragma unroll
            for (int t = 0; t < 2; t++) {
#pragma unroll
                for (int c = 0; c < 3; c++) L.s[t][c] = L.c[t][c] = 0.f;
                L.ncell[t] = L.nleaf[t] = L.nmac[t] = 0;
            }
            // one walk for both, or one each when they lie in different boxes
            for (unsigned who = both && box0 == box1 ? 3u : 1u; who; who = who == 1u && both ? 2u : 0u)
                walk_pair<kQuad, kInside, kSoft>(A, S, i0, i1, who, who == 2u ? box1 : box0, L, N);
#pragma unroll
            for (int t = 0; t < 2; t++) {
                N.ncell += L.ncell[t];
                N.nleaf += L.nleaf[t];
                N.nmac += L.nmac[t];
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    L.c[t][c] = -L.c[t][c];
                    reduce_hilo(L.s[t][c], L.c[t][c]);
                }
                L.ncell[t] = __reduce_add_sync(kFull, L.ncell[t]);
                L.nleaf[t] = __reduce_add_sync(kFull, L.nleaf[t]);
                L.nmac[t] = __reduce_add_sync(kFull, L.nmac[t]);
                if (lane == 0 && j + t < cnt) {
#pragma unroll
                    for (int c = 0; c < 3; c++) S.sum[j + t][c] = make_float2(L.s[t][c], L.c[t][c]);
                    S.cnt[j + t][0] = L.ncell[t];
                    S.cnt[j + t][1] = L.nleaf[t];
                    S.cnt[j + t][2] = L.nmac[t];
                    S.cnt[j + t][3] = t ? i1 : i0;
                }
            }
        }
        __syncwarp();
        if (lane < cnt) {
            const int i = S.cnt[lane][3];
            double a[3];
#pragma unroll
            for (int c = 0; c < 3; c++) a[c] = (double)S.sum[lane][c].x + (double)S.sum[lane][c].y;
            A.out.ax[i] = A.G * a[0];
            A.out.ay[i] = A.G * a[1];
            A.out.az[i] = A.G * a[2];
            if (A.out.ncell) {
                A.out.ncell[i] = S.cnt[lane][0];
                A.out.nleaf[i] = S.cnt[lane][1];
                A.out.nmac[i] = S.cnt[lane][2];
            }
        }
        __syncwarp();
    }
    const unsigned long long c0 = warp_total(N.ncell), c1 = warp_total(N.nleaf), c2 = warp_total(N.nmac);
    const unsigned long long c3 = warp_total(N.nrecheck);
    if (lane == 0 && c1 + c2) {
        atomicAdd(&A.ctl->n_cell, c0);
        atomicAdd(&A.ctl->n_leaf, c1);
        atomicAdd(&A.ctl->n_mac, c2);
        atomicAdd(&A.ctl->n_recheck, c3);
        atomicAdd(&A.ctl->n_iter, (unsigned long long)N.rounds);
    }
}

template <bool kQuad, bool kInside, bool kSoft>
__global__ void __launch_bounds__(kMaxWalkBlock, 3) k_twalk32x2(GravArgs A, int per) {
    __shared__ PSmem s[kMaxWalkBlock / 32];
    pair_units<kQuad, kInside, kSoft>(A, per, s[threadIdx.x >> 5]);
}

template <bool kQuad, bool kInside, bool kSoft>
__global__ void __launch_bounds__(kMaxWalkBlock, 4) k_twalk32(GravArgs A, int per) {
    __shared__ TSmem<false> s[kMaxWalkBlock / 32];
    target_units<kQuad, kInside, kSoft, false, false, false>(A, per, s[threadIdx.x >> 5], nullptr, nullptr);
}

template <bool kQuad, bool kInside, bool kSoft, bool kPot>
__global__ void __launch_bounds__(kMaxWalkBlock, 2) k_twalk64(GravArgs A, int per) {
    __shared__ TSmem<true> s[kMaxWalkBlock / 32];
    target_units<kQuad, kInside, kSoft, kPot, true, false>(A, per, s[threadIdx.x >> 5], nullptr, nullptr);
}

// Learned walk: the network's weights and one row queue per warp in shared
// memory (static shared memory holds them for 128 threads).
template <bool kInside, bool kSoft>
__global__ void __launch_bounds__(128, 4) k_twalk32_learn(GravArgs A, int per) {
    __shared__ __align__(16) mlp::Packed w;
    __shared__ __align__(16) LearnQ lq[4];
    __shared__ TSmem<false> s[4];
    {
        const uint4* src = reinterpret_cast<const uint4*>(A.wpk);
        uint4* dst = reinterpret_cast<uint4*>(&w);
        for (int k = threadIdx.x; k < (int)(sizeof(mlp::Packed) / 16); k += blockDim.x) dst[k] = src[k];
    }
    __syncthreads();
    target_units<true, kInside, kSoft, false, false, true>(A, per, s[threadIdx.x >> 5], &lq[threadIdx.x >> 5], &w);
}

template <typename K>
void launch(K kernel, const GravArgs& A, int block, int cap_n, cudaStream_t s, bool pairs = false) {
    // several units per resident warp, so that the queues even out the
    // targets' different walks, and more targets per unit when there are many
    const void* fn = reinterpret_cast<const void*>(kernel);
    const long long fit = (long long)walk_grid(fn, block, 1ll << 40) * (block / 32);
    int per = (int)std::max<long long>(1, std::min<long long>(kUnit, cap_n / (8 * fit)));
    if (pairs) per = std::max(2, per & ~1);
    const int grid = walk_grid(fn, block, ceil_div(cap_n, per));
    kernel<<<grid, block, 0, s>>>(A, per);
}

}  // namespace

void target_walk_prepare() {
#define RB_P32(Q, I) \
    walk_prepare_kernel((const void*)k_twalk32<Q, I, true>); walk_prepare_kernel((const void*)k_twalk32<Q, I, false>); \
    walk_prepare_kernel((const void*)k_twalk32x2<Q, I, true>); walk_prepare_kernel((const void*)k_twalk32x2<Q, I, false>)
#define RB_P64(Q, I, S) \
    walk_prepare_kernel((const void*)k_twalk64<Q, I, S, true>); walk_prepare_kernel((const void*)k_twalk64<Q, I, S, false>)
    RB_P32(true, true); RB_P32(true, false); RB_P32(false, true); RB_P32(false, false);
    RB_P64(true, true, true); RB_P64(true, true, false); RB_P64(true, false, true); RB_P64(true, false, false);
    RB_P64(false, true, true); RB_P64(false, true, false); RB_P64(false, false, true); RB_P64(false, false, false);
#undef RB_P32
#undef RB_P64
    walk_prepare_kernel((const void*)k_twalk32_learn<true, true>);
    walk_prepare_kernel((const void*)k_twalk32_learn<true, false>);
    walk_prepare_kernel((const void*)k_twalk32_learn<false, true>);
    walk_prepare_kernel((const void*)k_twalk32_learn<false, false>);
}

void target_walk(const GravArgs& A, TargetWalk mode, bool quad, bool inside, bool soft, bool pot, int block,
                 int cap_n, cudaStream_t s) {
#define RB_L(...) launch(__VA_ARGS__, A, block, cap_n, s)
#define RB_SOFT(K, ...) do { if (soft) RB_L(K<__VA_ARGS__, true>); else RB_L(K<__VA_ARGS__, false>); } while (0)
#define RB_64(Q, I)                                                                                       \
    do {                                                                                                  \
        if (soft) { if (pot) RB_L(k_twalk64<Q, I, true, true>); else RB_L(k_twalk64<Q, I, true, false>); } \
        else { if (pot) RB_L(k_twalk64<Q, I, false, true>); else RB_L(k_twalk64<Q, I, false, false>); }    \
    } while (0)
#define RB_P(Q, I)                                                                       \
    do {                                                                                 \
        if (pairs) {                                                                     \
            if (soft) launch(k_twalk32x2<Q, I, true>, A, block, cap_n, s, true);         \
            else launch(k_twalk32x2<Q, I, false>, A, block, cap_n, s, true);             \
        } else {                                                                         \
            RB_SOFT(k_twalk32, Q, I);                                                    \
        }                                                                                \
    } while (0)
    if (mode == TargetWalk::kLearned) {
        block = 128;
        if (inside) RB_SOFT(k_twalk32_learn, true);
        else RB_SOFT(k_twalk32_learn, false);
    } else if (mode == TargetWalk::kFp64) {
        if (quad) { if (inside) RB_64(true, true); else RB_64(true, false); }
        else { if (inside) RB_64(false, true); else RB_64(false, false); }
    } else {
        block = kMaxWalkBlock;   // pairs at 30k: 162 us; in blocks of 128: 166
        const bool pairs = cap_n >= kPairMin;
        if (quad) { if (inside) RB_P(true, true); else RB_P(true, false); }
        else { if (inside) RB_P(false, true); else RB_P(false, false); }
    }
#undef RB_P
#undef RB_64
#undef RB_SOFT
#undef RB_L
}

}  // namespace rb
