// rb_sweep.cu -- plane-sweep collision detection along x (Sect. 5.3).
//
// The paper's sweep moves a plane through the 2N sorted x extents of the
// particle trajectories, keeps the list of trajectories the plane cuts, and
// tests each trajectory entering the list against every one already in it.
// On the GPU the same pair set comes from "sort and sweep":
//   1. every live particle gives an item: its trajectory's x extent
//      [x - |v_x| dt/2 - R - m, x + |v_x| dt/2 + R + m] (m = 1e-9 Lx), plus
//      copies shifted by +k Lx (k = 1..nghost_x) for ghost images across the
//      x boundary, emitted only when they can reach the box's own items;
//   2. items are radix-sorted by (box, quantised lower end);
//   3. one thread per sorted item P scans forward while the next item's lower
//      end is not beyond P's upper end: those are exactly the items whose
//      extents overlap P's and start after it, the trajectories already in the
//      paper's list when P enters it.  Each candidate (at least one original
//      particle, two different particles) is tested with the straight-line
//      criterion for every y/z image within reach, in FP32 clear of the
//      threshold, else in FP64 with the oracle's operation sequence on the
//      canonical orientation (lower id a, image of b).
// The quantisation is a monotone map of the FP64 extents, so the scan never
// stops before an overlapping item.
#include "rb_internal.cuh"

namespace rb {
namespace {

constexpr double kMarginRel = 1e-9;   // extents widened by 1e-9 Lx (reading S3)

struct SweepArgs {
    PSet P;
    Ctl* ctl;
    const BoxP* boxes;
    uint64_t* key;
    uint32_t* val;
    uint64_t* pair_key;
    int pair_cap, item_cap, ncap, nbox;
    int ngx, ngy, ngz, hs;
    double t0, half_dt, h;   // h = dt / 2: the trajectory's half length in time
};

__device__ __forceinline__ double ext_of(const SweepArgs& A, int i) {
    return __dadd_rn(__dmul_rn(fabs(A.P.vx[i]), A.h), A.P.r[i]);
}

// Largest half extent |v_x| dt/2 + R over the live particles, as the bits of
// a non-negative double (ordered like the values).
__global__ void __launch_bounds__(256) k_sweep_ext(SweepArgs A) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int n = min(A.ctl->n_live, A.ncap);
    unsigned long long b = 0ull;
    if (i < n && A.P.box[i] < A.nbox) b = (unsigned long long)__double_as_longlong(ext_of(A, i));
    for (int o = 16; o > 0; o >>= 1) b = max(b, __shfl_xor_sync(0xffffffffu, b, o));
    if ((threadIdx.x & 31) == 0 && b) atomicMax(&A.ctl->sweep_wbits, b);
}

// Quantised position of v in a box's sweep range [base, base + span):
// floor((v - base) * 2^32 / span), clamped; monotone in v.
__device__ __forceinline__ uint64_t quant(double v, double base, double scale) {
    const double q = floor(__dmul_rn(__dsub_rn(v, base), scale));
    if (!(q > 0.0)) return 0ull;
    if (q >= 4294967295.0) return 4294967295ull;
    return (uint64_t)q;
}

struct Range {
    double base, scale, top, lx, m;
};

__device__ __forceinline__ Range range_of(const SweepArgs& A, const BoxP& bp) {
    Range g;
    const double w = __longlong_as_double((long long)A.ctl->sweep_wbits);
    g.lx = bp.Lx;
    g.m = kMarginRel * bp.Lx;
    const double W = w + g.m;
    g.base = -0.5 * bp.Lx - W;
    g.top = 0.5 * bp.Lx + W;
    g.scale = 4294967296.0 / (bp.Lx + 2.0 * W);
    return g;
}

// Items: the particle and its copies shifted by +k Lx that can reach the box.
// Each warp reserves its items with one atomic (prefix sum of the lanes'
// counts).
__global__ void __launch_bounds__(256) k_sweep_items(SweepArgs A) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    const int n = min(A.ctl->n_live, A.ncap);
    int b = 0, cnt = 0;
    double lo0 = 0.0;
    Range g{};
    if (i < n) {
        b = A.P.box[i];
        if (b < A.nbox) {
            g = range_of(A, A.boxes[b]);
            lo0 = __dsub_rn(A.P.x[i], __dadd_rn(ext_of(A, i), g.m));
            cnt = 1;
            // copies k = 1..ngx whose lower end can still reach the box's items
            for (int k = 1; k <= A.ngx; k++) {
                if (__dadd_rn(lo0, __dmul_rn((double)k, g.lx)) > g.top) break;
                cnt++;
            }
        }
    }
    int incl = cnt;
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    int base = 0;
    if (lane == 31 && incl) base = atomicAdd(&A.ctl->sweep_items, incl);
    base = __shfl_sync(0xffffffffu, base, 31) + incl - cnt;
    for (int k = 0; k < cnt; k++) {
        const int pos = base + k;
        if (pos >= A.item_cap) break;   // cannot happen: item_cap = ncap (1 + nghost_x)
        // the lower end of copy k, as the scans recompute it
        const double e = __dadd_rn(ext_of(A, i), g.m);
        const double lo = __dsub_rn(__dadd_rn(A.P.x[i], __dmul_rn((double)k, g.lx)), e);
        A.key[pos] = ((uint64_t)b << 32) | quant(lo, g.base, g.scale);
        A.val[pos] = ((uint32_t)i << 3) | (uint32_t)k;
    }
}

// Particle data of the sorted items, gathered once so that the scans read
// neighbouring records instead of scattered particle slots: positions as hi/lo
// floats, velocities and radius as floats (the particle's own, unshifted).
struct __align__(16) SweepRec {
    float xh, yh, zh, r;
    float xl, yl, zl, vx;
    float vy, vz;
    uint32_t sc;     // (slot << 3) | copy
    float vsum;      // |vx| + |vy| + |vz|
};

__device__ __forceinline__ void split_hl(double v, float& hi, float& lo) {
    hi = __double2float_rn(v);
    lo = __double2float_rn(v - (double)hi);
}

__global__ void __launch_bounds__(256) k_sweep_gather(SweepArgs A, const uint32_t* __restrict__ val,
                                                      SweepRec* __restrict__ rec) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int nitem = min(sorted_counts(A.ctl).y, A.item_cap);
    if (k >= nitem) return;
    const uint32_t v = val[k];
    const int i = (int)(v >> 3);
    SweepRec q;
    split_hl(A.P.x[i], q.xh, q.xl);
    split_hl(A.P.y[i], q.yh, q.yl);
    split_hl(A.P.z[i], q.zh, q.zl);
    q.vx = (float)A.P.vx[i];
    q.vy = (float)A.P.vy[i];
    q.vz = (float)A.P.vz[i];
    q.r = (float)A.P.r[i];
    q.vsum = fabsf(q.vx) + fabsf(q.vy) + fabsf(q.vz);
    q.sc = v;
    rec[k] = q;
}

// Straight-line criterion (Sect. 5.3, readings S1/S2) for particle a and the
// image of b (offset o, y velocity offset dvy), in the oracle's operation
// sequence.
__device__ __forceinline__ bool line_hit(const PSet& P, int a, int b, double h, double ox, double oy, double oz,
                                         double dvy) {
    const double rx = __dsub_rn(__dadd_rn(P.x[b], ox), P.x[a]);
    const double ry = __dsub_rn(__dadd_rn(P.y[b], oy), P.y[a]);
    const double rz = __dsub_rn(__dadd_rn(P.z[b], oz), P.z[a]);
    const double ux = __dsub_rn(P.vx[b], P.vx[a]);
    const double uy = __dsub_rn(__dadd_rn(P.vy[b], dvy), P.vy[a]);
    const double uz = __dsub_rn(P.vz[b], P.vz[a]);
    const double uu = __dadd_rn(__dadd_rn(__dmul_rn(ux, ux), __dmul_rn(uy, uy)), __dmul_rn(uz, uz));
    const double ru = __dadd_rn(__dadd_rn(__dmul_rn(rx, ux), __dmul_rn(ry, uy)), __dmul_rn(rz, uz));
    double tau = 0.0;
    if (uu > 0.0) {
        tau = __ddiv_rn(-ru, uu);
        if (tau < -h) tau = -h;
        if (tau > h) tau = h;
    }
    const double dx = __dadd_rn(rx, __dmul_rn(ux, tau));
    const double dy = __dadd_rn(ry, __dmul_rn(uy, tau));
    const double dz = __dadd_rn(rz, __dmul_rn(uz, tau));
    const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
    const double s = __dadd_rn(P.r[a], P.r[b]);
    return d2 < __dmul_rn(s, s);
}

// Pairs found by a warp and not yet recorded.
struct SweepQueue {
    int si[64], sj[64];   // slots of the scanning item's particle and of the other one
    int img[64];          // image of the other as seen from the first: code, bit 12: clear of the threshold
};

// Records n (<= 32) queued pairs, a lane each, on the canonical orientation
// (lower id a, image of b); those not clear of the threshold take the exact
// criterion.
__device__ __forceinline__ void sweep_record(const SweepArgs& A, const SweepQueue& Q, int from, int n) {
    const int lane = threadIdx.x & 31;
    bool hit = false;
    uint64_t key = 0;
    if (lane < n) {
        const int i = Q.si[from + lane], j = Q.sj[from + lane], c = Q.img[from + lane];
        int gx = (c & 15) - 7, gy = ((c >> 4) & 15) - 7, gz = ((c >> 8) & 15) - 7;
        const int ii = A.P.id[i], ij = A.P.id[j];
        const bool flip = ij < ii;
        if (flip) {
            gx = -gx;
            gy = -gy;
            gz = -gz;
        }
        hit = (c >> 12) & 1;
        if (!hit) {
            const BoxP bp = A.boxes[A.P.box[i]];
            const double s = shear_offset(bp, time_of(A.ctl, A.t0, A.half_dt, A.hs));
            double ox, oy, oz;
            image_offset(bp, s, gx, gy, gz, ox, oy, oz);
            hit = line_hit(A.P, flip ? j : i, flip ? i : j, A.h, ox, oy, oz, __dmul_rn(-(double)gx, bp.shear_speed));
        }
        key = ((uint64_t)min(ii, ij) << 36) | ((uint64_t)max(ii, ij) << 12) |
              (uint64_t)((gx + 7) | ((gy + 7) << 4) | ((gz + 7) << 8));
    }
    const unsigned hits = __ballot_sync(0xffffffffu, hit);
    if (!hits) return;
    int base = 0;
    if (lane == 0) base = atomicAdd(&A.ctl->pair_count, __popc(hits));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (hit) {
        const int at = base + __popc(hits & ((1u << lane) - 1u));
        if (at < A.pair_cap) A.pair_key[at] = key;
        else atomicOr(&A.ctl->err, kErrPairOverflow);
    }
}

// One thread per sorted item scans the items that start before its own ends,
// the lanes of a warp in step.  A candidate's y images within reach are found
// by division instead of a loop over all, and the criterion is decided in FP32
// (positions as hi/lo differences) unless the distance lies within the error
// bound of the threshold; only those few take the FP64 criterion, when the
// queued pairs are recorded: an FP64 instruction holds the SM's FP64 pipe 16
// cycles per warp.  300,000 particles of a ring: 131 us, 712 with every
// candidate's y extent and criterion in FP64.
__global__ void __launch_bounds__(128) k_sweep_pairs(SweepArgs A, const SweepRec* __restrict__ rec) {
    __shared__ SweepQueue queue[4];
    SweepQueue& Q = queue[threadIdx.x >> 5];
    const int k = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int nitem = min(sorted_counts(A.ctl).y, A.item_cap);
    if (k - lane >= nitem) return;   // the whole warp
    bool scan = k < nitem;
    const SweepRec P = rec[scan ? k : nitem - 1];
    const int ci = (int)(P.sc & 7u);
    const int si = (int)(P.sc >> 3);
    const int b = (int)(A.key[scan ? k : nitem - 1] >> 32);
    const BoxP bp = A.boxes[b];
    uint64_t khi;
    {
        const Range g = range_of(A, bp);
        const double hi = __dadd_rn(__dadd_rn(A.P.x[si], __dmul_rn((double)ci, g.lx)), __dadd_rn(ext_of(A, si), g.m));
        khi = ((uint64_t)b << 32) | quant(hi, g.base, g.scale);
    }
    // more trajectories cut by the plane than the sweep is meant for (the
    // O(N N_SWEEPL) cost of Sect. 5.3 turning quadratic): report, do not scan
    const int lim = k + 1 + kMaxSweepScan;
    if (scan && lim < nitem && A.key[lim] <= khi) {
        atomicOr(&A.ctl->err, kErrSweepLong);
        scan = false;
    }
    const double s64 = shear_offset(bp, time_of(A.ctl, A.t0, A.half_dt, A.hs));
    const float h = (float)A.h, Ly = (float)bp.Ly, iLy = 1.f / Ly, Lz = (float)bp.Lz, iLz = 1.f / Lz;
    const float speed = (float)bp.shear_speed;
    // hi/lo positions and offsets are good to 2^-47 of their size
    const float far = 1e-13f * (fabsf(P.xh) + fabsf(P.yh) + fabsf(P.zh) +
                                (float)(A.ngx + 1) * (float)bp.Lx + (float)(A.ngy + 1) * Ly + (float)(A.ngz + 1) * Lz);
    int nq = 0;   // queued pairs (warp-uniform)
    for (int j = k + 1; ; j++) {
        scan = scan && j < nitem && A.key[j] <= khi;   // at the latest at lim (keys are sorted)
        if (((j - k) & 1023) == 0 && (*(volatile const int*)&A.ctl->err & kErrSweepLong)) scan = false;
        if (!__any_sync(0xffffffffu, scan)) break;
        SweepRec R;
        int gx = 0, sj = 0, gy = 1, gy1 = 0, gz0 = 0, gz1 = -1, gz = 0;
        float rx = 0.f, ry = 0.f, rz = 0.f, ux = 0.f, uy = 0.f, uz = 0.f, sr = 0.f, err = 0.f;
        if (scan) {
            R = rec[j];
            const int cj = (int)(R.sc & 7u);
            sj = (int)(R.sc >> 3);
            if ((ci == 0 || cj == 0) && sj != si) {
                // image of R's particle as seen from P's
                gx = cj - ci;
                float oxh = 0.f, oxl = 0.f, oyh = 0.f, oyl = 0.f;
                if (gx != 0) {
                    split_hl((double)gx * bp.Lx, oxh, oxl);
                    split_hl(-((double)gx * s64), oyh, oyl);
                }
                rx = ((R.xh - P.xh) + oxh) + ((R.xl - P.xl) + oxl);
                ry = ((R.yh - P.yh) + oyh) + ((R.yl - P.yl) + oyl);
                rz = (R.zh - P.zh) + (R.zl - P.zl);
                ux = R.vx - P.vx;
                uy = (R.vy - (float)gx * speed) - P.vy;
                uz = R.vz - P.vz;
                sr = P.r + R.r;
                // bound of the FP32 distance's error: differences rounded to
                // 2^-24, velocities and tau to a few times that
                const float vel = h * (P.vsum + R.vsum + fabsf((float)gx * speed));
                err = 1e-6f * (fabsf(rx) + fabsf(oxh) + fabsf(ry) + fabsf(oyh) + fabsf(rz) + vel + sr) + far;
                // |d| <= sr needs |r_y| <= sr + |u_y| h for an image, and the same in z
                const float ly = sr + fabsf(uy) * h + 2.f * err, lz = sr + fabsf(uz) * h + 2.f * err;
                gy = max(-A.ngy, (int)ceilf((-ly - ry) * iLy - 4e-6f));
                gy1 = min(A.ngy, (int)floorf((ly - ry) * iLy + 4e-6f));
                gz0 = max(-A.ngz, (int)ceilf((-lz - rz) * iLz - 4e-6f));
                gz1 = min(A.ngz, (int)floorf((lz - rz) * iLz + 4e-6f));
                gz = gz0;
                if (gz0 > gz1) gy = gy1 + 1;
            }
        }
        while (__any_sync(0xffffffffu, gy <= gy1)) {
            bool near = false, sure = false;
            int code = 0;
            if (gy <= gy1) {
                const float oy = (float)gy * Ly, oz = (float)gz * Lz;
                const float e = err + 1e-6f * (fabsf(oy) + fabsf(oz));
                const float y = ry + oy, z = rz + oz;
                const float uu = fmaf(uz, uz, fmaf(uy, uy, ux * ux));
                const float ru = fmaf(z, uz, fmaf(y, uy, rx * ux));
                const float tau = uu > 0.f ? fminf(fmaxf(-ru / uu, -h), h) : 0.f;
                const float dx = fmaf(ux, tau, rx), dy = fmaf(uy, tau, y), dz = fmaf(uz, tau, z);
                const float d2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
                const float out = sr + e, in = sr - e;
                near = !(d2 > out * out);
                sure = in > 0.f && d2 < in * in;
                code = (gx + 7) | ((gy + 7) << 4) | ((gz + 7) << 8) | (sure ? 1 << 12 : 0);
                if (++gz > gz1) {
                    gz = gz0;
                    gy++;
                }
            }
            const unsigned m = __ballot_sync(0xffffffffu, near);
            if (!m) continue;
            if (near) {
                const int at = nq + __popc(m & lt);
                Q.si[at] = si;
                Q.sj[at] = sj;
                Q.img[at] = code;
            }
            nq += __popc(m);
            if (nq >= 32) {
                nq -= 32;
                __syncwarp();
                sweep_record(A, Q, nq, 32);
                __syncwarp();
            }
        }
    }
    __syncwarp();
    sweep_record(A, Q, 0, nq);
}

__global__ void k_sweep_reset(Ctl* ctl) {
    ctl->sweep_items = 0;
    ctl->sweep_wbits = 0ull;
}

}  // namespace

void sweep_search(const PSet& P, Ctl* ctl, const BoxP* boxes, const SimC& C, Sweep& S,
                  const Pairs& PR, int half_step_offset, int ncap, cudaStream_t s) {
    if (ncap <= 0) return;
    SweepArgs A;
    A.P = P; A.ctl = ctl; A.boxes = boxes;
    A.key = S.key; A.val = S.val;
    A.pair_key = PR.key; A.pair_cap = PR.cap; A.item_cap = S.cap; A.ncap = ncap; A.nbox = C.nbox;
    A.ngx = C.ngx; A.ngy = C.ngy; A.ngz = C.ngz; A.hs = half_step_offset;
    A.t0 = C.t0; A.half_dt = C.half_dt; A.h = 0.5 * C.dt;
    k_sweep_reset<<<1, 1, 0, s>>>(ctl);
    k_sweep_ext<<<ceil_div(ncap, 256), 256, 0, s>>>(A);
    k_sweep_items<<<ceil_div(ncap, 256), 256, 0, s>>>(A);
    const int key_bits = 32 + S.box_bits;
    const int which = radix_sort(S.key, S.val, S.key_alt, S.val_alt, S.cap, &ctl->sweep_items, key_bits,
                                 nullptr, 0, S.hist, &ctl->err, s, 0, nullptr, nullptr, (C.hold_sort & kHoldSweep) != 0);
    if (which == 1) {
        A.key = S.key_alt;
        A.val = S.val_alt;
    }
    SweepRec* rec = static_cast<SweepRec*>(S.rec);
    k_sweep_gather<<<ceil_div(S.cap, 256), 256, 0, s>>>(A, A.val, rec);
    k_sweep_pairs<<<ceil_div(S.cap, 128), 128, 0, s>>>(A, rec);
}

}  // namespace rb
