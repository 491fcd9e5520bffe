// rb_step.cu -- the per-particle parts of a DKD step (Sect. 3): drift with
// boundaries (Sect. 2.3) fused with the Morton keys of the next tree build,
// the kick, the gather into Morton order, collision resolution (Sect. 5,
// Eq. 2) and the energy/momentum sums (Sect. 6.2).
//
// Drift, kick, boundary wrap and the pairs' separations use explicitly rounded
// FP64 operations (__dadd_rn, __dmul_rn, ...) so the compiler never fuses them:
// they give bit-identical results to any other IEEE FP64 implementation that
// evaluates the same expressions in the same order without fused multiply-adds.
// The impulse of a collision uses fused multiply-adds.
#include <algorithm>
#include <climits>
#include <cstddef>
#include <type_traits>

#include "rb_fp64.cuh"
#include "rb_internal.cuh"

namespace rb {
namespace {

__device__ __forceinline__ uint64_t spread3(uint32_t v) {
    uint64_t x = v & 0x1fffffu;
    x = (x | (x << 32)) & 0x1f00000000ffffull;
    x = (x | (x << 16)) & 0x1f0000ff0000ffull;
    x = (x | (x << 8)) & 0x100f00f00f00f00full;
    x = (x | (x << 4)) & 0x10c30c30c30c30c3ull;
    x = (x | (x << 2)) & 0x1249249249249249ull;
    return x;
}

// Integer coordinate floor(((x - lo) / L) * 2^21), clamped to [0, 2^21 - 1].
// k = (x - lo) * scale, with scale = (1/L, rounded) x 2^21 (a power-of-two
// scaling, so no further rounding), lies within 2^-30 of the oracle's
// fl((x - lo) / L) x 2^21; wherever k is at least 2^-23 from every grid line
// both have the same floor.  For k in [1, 2^21) the floor and that distance
// are read from k's bits with integer operations: on GB300 an FP64
// instruction holds the SM's FP64 pipe 16 cycles per warp, and this kernel's
// time is its FP64 instructions.  Other k and the few near a grid line (returns
// false) take the FP64 division.
__device__ __forceinline__ bool icoord_fast(double d, double scale, uint32_t& v) {
    const uint64_t b = (uint64_t)__double_as_longlong(__dmul_rn(d, scale));
    const int e = (int)(b >> 52) - 1023;   // unbiased exponent (sign set or NaN: e > 20)
    const int sh = 52 - min(max(e, 0), 20);   // fraction bits of k
    const uint64_t m = (b & 0xfffffffffffffull) | (1ull << 52);
    const uint64_t one = 1ull << sh, fr = m & (one - 1), tol = 1ull << (sh - 23);
    v = (uint32_t)(m >> sh);
    return e >= 0 && e <= 20 && fr >= tol && one - fr >= tol;
}

__device__ __forceinline__ uint32_t icoord_div(double d, double L) {
    double k = floor(__dmul_rn(__ddiv_rn(d, L), 2097152.0));
    if (!(k >= 0.0)) k = 0.0;
    if (k > 2097151.0) k = 2097151.0;
    return (uint32_t)k;
}

__device__ __forceinline__ uint64_t morton(uint32_t x, uint32_t y, uint32_t z) {
    return (spread3(x) << 2) | (spread3(y) << 1) | spread3(z);
}

__device__ __noinline__ uint64_t key_div(double dx, double dy, double dz, double L) {
    return morton(icoord_div(dx, L), icoord_div(dy, L), icoord_div(dz, L));
}

// Order-preserving integer image of a double: for a, b not NaN (and -0 not
// compared with +0), a < b exactly when dord(a) < dord(b), and for h > 0,
// dord(-h) = ~dord(h).  The boundary tests compare this way, without FP64
// instructions.  A NaN coordinate compares as beyond every bound; the
// non-finite check after the wrap reports it either way.
__device__ __forceinline__ int64_t dord(double v) {
    const int64_t b = __double_as_longlong(v);
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}

__device__ __forceinline__ bool finite_bits(double v) {
    return ((__double_as_longlong(v) >> 52) & 0x7ff) != 0x7ff;
}

__device__ __forceinline__ double time_at(const Ctl* ctl, int hs, double t0, double half_dt) {
    const double h = (double)(2 * ctl->step + hs);
    return __dadd_rn(t0, __dmul_rn(h, half_dt));
}

template <bool kSei>
__device__ __forceinline__ void drift_one(const SimC& C, double& x, double& y, double& z,
                                          double& vx, double& vy, double& vz) {
    if (!kSei) {
        x = __dadd_rn(x, __dmul_rn(vx, C.half_dt));
        y = __dadd_rn(y, __dmul_rn(vy, C.half_dt));
        z = __dadd_rn(z, __dmul_rn(vz, C.half_dt));
        return;
    }
    const double x0 = x, u0 = vx, v0 = vy, z0 = z, w0 = vz;
    x = __dadd_rn(__dadd_rn(__dmul_rn(C.axx, x0), __dmul_rn(C.axu, u0)), __dmul_rn(C.axv, v0));
    y = __dadd_rn(y, __dadd_rn(__dadd_rn(__dmul_rn(C.ayx, x0), __dmul_rn(C.ayu, u0)),
                               __dmul_rn(C.ayv, v0)));
    vx = __dadd_rn(__dadd_rn(__dmul_rn(C.aux, x0), __dmul_rn(C.auu, u0)), __dmul_rn(C.auv, v0));
    vy = __dadd_rn(__dadd_rn(__dmul_rn(C.avx, x0), __dmul_rn(C.avu, u0)), __dmul_rn(C.avv, v0));
    z = __dadd_rn(__dmul_rn(C.azz, z0), __dmul_rn(C.azw, w0));
    vz = __dadd_rn(__dmul_rn(C.awz, z0), __dmul_rn(C.aww, w0));
}

// Wraps in y (and z) repeat the oracle's one-box-length steps; a particle
// that would need more than this many is reported as a runaway.
constexpr int kMaxWraps = 1 << 12;

// Boundaries of a particle outside its box.
struct Wrapped {
    double x, y, z, vy;
    bool live, runaway;
};
__device__ __noinline__ Wrapped wrap_outside(const BoxP* box, bool z_periodic, const Ctl* ctl, int hs, double t0,
                                             double half_dt, double x, double y, double z, double vy) {
    const BoxP bp = *box;
    const int64_t ux = dord(bp.hx), uy = dord(bp.hy), uz = dord(bp.hz);   // ~u is -h
    Wrapped w{x, y, z, vy, true, false};
    const double vs = bp.shear_speed;
    const int64_t ox = dord(x);
    const bool up = ox >= ux, down = ox < ~ux;
    // the shear offset only for the few particles that cross in x
    const double s = (up || down) && vs != 0.0 ? fmod(__dmul_rn(vs, time_at(ctl, hs, t0, half_dt)), bp.Ly) : 0.0;
    if (up) {
        w.x = __dsub_rn(x, bp.Lx);
        w.y = __dadd_rn(y, s);
        w.vy = __dadd_rn(vy, vs);
    } else if (down) {
        w.x = __dadd_rn(x, bp.Lx);
        w.y = __dsub_rn(y, s);
        w.vy = __dsub_rn(vy, vs);
    }
    for (int k = 0; k < kMaxWraps && dord(w.y) >= uy; k++) w.y = __dsub_rn(w.y, bp.Ly);
    for (int k = 0; k < kMaxWraps && dord(w.y) < ~uy; k++) w.y = __dadd_rn(w.y, bp.Ly);
    const int64_t oy = dord(w.y);
    if (oy >= uy || oy < ~uy) w.runaway = true;
    if (z_periodic) {
        for (int k = 0; k < kMaxWraps && dord(w.z) >= uz; k++) w.z = __dsub_rn(w.z, bp.Lz);
        for (int k = 0; k < kMaxWraps && dord(w.z) < ~uz; k++) w.z = __dadd_rn(w.z, bp.Lz);
    }
    const int64_t oz = dord(w.z);
    const bool out = oz < ~uz || oz >= uz;
    if (z_periodic) w.runaway |= out;
    else w.live = !out;
    return w;
}

// Boundaries after a drift half; returns false if the particle left an open
// boundary.  *runaway is set when the wraps did not bring it back.  Most
// particles are inside and take no FP64 instruction here; with the wraps
// inlined, 7 were issued (predicated off) for every particle.
__device__ __forceinline__ bool wrap_one(const SimC& C, const BoxP& bp, const BoxP* box, const Ctl* ctl, int hs,
                                         double& x, double& y, double& z, double& vy, bool* runaway) {
    const int64_t ux = dord(bp.hx), uy = dord(bp.hy), uz = dord(bp.hz);   // ~u is -h
    const int64_t ox = dord(x), oy = dord(y), oz = dord(z);
    const bool in = ox >= ~ux && ox < ux && oy >= ~uy && oy < uy && oz >= ~uz && oz < uz;
    if (in || C.boundary == 0) return in;
    const Wrapped w = wrap_outside(box, C.z_periodic, ctl, hs, C.t0, C.half_dt, x, y, z, vy);
    x = w.x;
    y = w.y;
    z = w.z;
    vy = w.vy;
    if (w.runaway) *runaway = true;
    return w.live;
}

struct DriftArgs {
    PSet P;
    uint64_t* key;
    uint32_t* idx;
    int32_t* sbox;
    Ctl* ctl;
    const BoxP* boxes;
    const double *ax, *ay, *az;
    int ncap, ndrift, hs;
};

// Optional kick (v += a dt, kKick), one or two drift halves (kSei: Hill's
// equations) each followed by the boundaries, then, for the drifts that a sort
// follows (kKeys), the Morton key of the new position.  The time is the FP64
// pipe's: a SEI half with its key issues 36 FP64 instructions per warp (63 with
// the rare paths and the run-time options inlined).  1M particles of the sheet:
// 103 -> 79 us with keys, 93 -> 76 us for the kick and drift.
template <bool kKeys, bool kKick, bool kSei>
__global__ void __launch_bounds__(256) k_drift_keys(DriftArgs A, SimC C) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= A.ncap) return;
    if (kKeys) A.idx[i] = (uint32_t)i;
    bool live = A.P.box[i] < C.nbox;
    uint64_t key = kRemovedKey;
    if (live) {
        double x = A.P.x[i], y = A.P.y[i], z = A.P.z[i];
        double vx = A.P.vx[i], vy = A.P.vy[i], vz = A.P.vz[i];
        const BoxP bp = A.boxes[A.P.box[i]];
        if (kKick) {
            vx = __dadd_rn(vx, __dmul_rn(A.ax[i], C.dt));
            vy = __dadd_rn(vy, __dmul_rn(A.ay[i], C.dt));
            vz = __dadd_rn(vz, __dmul_rn(A.az[i], C.dt));
        }
        bool runaway = false;
        for (int d = 0; d < A.ndrift && live; d++) {
            drift_one<kSei>(C, x, y, z, vx, vy, vz);
            live = wrap_one(C, bp, &A.boxes[A.P.box[i]], A.ctl, A.hs + d, x, y, z, vy, &runaway);
        }
        if (runaway || !(finite_bits(x) && finite_bits(y) && finite_bits(z))) {
            atomicOr(&A.ctl->err, kErrNonFinite);
            live = false;
        }
        A.P.x[i] = x; A.P.y[i] = y; A.P.z[i] = z;
        A.P.vx[i] = vx; A.P.vy[i] = vy; A.P.vz[i] = vz;
        if (kKeys && live) {
            const double lo = -bp.hx;   // the root cube's side L is Lx
            const double dx = __dsub_rn(x, lo), dy = __dsub_rn(y, lo), dz = __dsub_rn(z, lo);
            uint32_t kx, ky, kz;
            const bool fx = icoord_fast(dx, bp.key_scale, kx), fy = icoord_fast(dy, bp.key_scale, ky);
            const bool fz = icoord_fast(dz, bp.key_scale, kz);
            key = fx && fy && fz ? morton(kx, ky, kz) : key_div(dx, dy, dz, bp.L);
        }
    }
    if (!live) A.P.box[i] = C.nbox;
    if (!kKeys) return;   // the particles keep their slots; removed ones stay flagged
    A.key[i] = key;
    A.sbox[i] = live ? A.P.box[i] : C.nbox;
    const unsigned b = __ballot_sync(0xffffffffu, live);
    if ((threadIdx.x & 31) == 0 && b) atomicAdd(&A.ctl->n_live_next, __popc(b));
}

// The gather into sorted order.  Also commits the live count, and clears what
// the topology kernels that follow fill in.
__global__ void __launch_bounds__(256) k_permute(PSet S, PSet D, const uint32_t* __restrict__ idx,
                                                 int32_t* __restrict__ slot_of_id, Ctl* ctl, int ncap,
                                                 Tree T, int nstat, int nbox) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int nlive = ctl->n_live_next;   // cleared by k_nodes
    if (i == 0) ctl->n_live = nlive;
    for (int k = i; k < nstat; k += gridDim.x * blockDim.x) T.scan_stat[k] = 0u;
    for (int k = i; k <= nbox; k += gridDim.x * blockDim.x) T.box_root[k] = -1;
    if (i >= ncap) return;
    T.mask[i] = 0u;
    reinterpret_cast<uint2*>(T.e_cmask)[i] = make_uint2(0u, 0u);   // two entries a slot
    const int j = (int)idx[i];
    D.x[i] = S.x[j]; D.y[i] = S.y[j]; D.z[i] = S.z[j];
    D.vx[i] = S.vx[j]; D.vy[i] = S.vy[j]; D.vz[i] = S.vz[j];
    D.m[i] = S.m[j]; D.r[i] = S.r[j];
    const int id = S.id[j];
    D.id[i] = id;
    D.box[i] = S.box[j];
    if (i < nlive) slot_of_id[id] = i;
}

struct ResolveArgs {
    PSet P;
    const uint64_t* key;          // sorted pairs (resolution order)
    const int32_t* slot_of_id;
    int32_t *head, *link;         // per particle: its pairs as the higher id, a list in any order
    int32_t* done;                // per pair: 1 once resolved
    int32_t* claim;               // pairs claimed by running warps
    Ctl* ctl;
    const ImgTab* img;            // [box][image] offsets at the detection time
    int nimg, ngx, ngy, ngz;
    bool advance;                 // this resolution ends a step
};

__device__ __forceinline__ int key_a(uint64_t k) { return (int)(k >> 36); }
__device__ __forceinline__ int key_b(uint64_t k) { return (int)((k >> 12) & 0xFFFFFFull); }

// Every pair joins the list of its higher particle id; head is -1 for every
// particle on entry.
__global__ void __launch_bounds__(256) k_pair_link(ResolveArgs A) {
    const int n = sorted_counts(A.ctl).x;
    if (blockIdx.x == 0 && threadIdx.x == 0) *A.claim = 0;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        A.link[k] = atomicExch(&A.head[key_b(A.key[k])], k);
        A.done[k] = 0;
    }
}

// The last pair before k in particle p's list (pairs in which p is the higher
// id), or -1.  A list holds as many pairs as the particle has contacts from
// below; they are resolved one after the other in any case.
__device__ __forceinline__ int last_before(const ResolveArgs& A, int p, int k) {
    int best = -1;
    for (int j = A.head[p]; j >= 0; j = A.link[j])
        if (j < k) best = max(best, j);
    return best;
}

// Everything about a pair that does not depend on velocities: the separation
// vector, the impulse factors of Eq. 2, and the previous pair in resolution
// order of either particle.
struct PairRec {
    double rx, ry, rz, dvy;   // separation (with the image offset), velocity offset of the image
    double ka, kb;            // impulse factors of u.r (of 1 + eps too, with a constant eps)
    double rabs;              // power law: |r|
    int32_t a, b;             // slots
    int32_t pa, pb;           // previous pair of either particle, or -1
};

// The queue is sorted by (a, b), a < b, so a particle's pairs as the higher id
// come before its pairs as the lower one: b's previous pair is one in its
// list, a's is the pair before this one if that has the same a, else the last
// one in a's list.
template <bool kPower>
__device__ __forceinline__ PairRec pair_rec(const ResolveArgs& A, const SimC& C, int k) {
    const uint64_t key = A.key[k];
    const int ia = key_a(key), ib = key_b(key), code = (int)(key & 0xFFFull);
    const int gx = (code & 15) - 7, gy = ((code >> 4) & 15) - 7, gz = ((code >> 8) & 15) - 7;
    const int g = ((gx + A.ngx) * (2 * A.ngy + 1) + (gy + A.ngy)) * (2 * A.ngz + 1) + (gz + A.ngz);
    PairRec R;
    R.a = A.slot_of_id[ia];
    R.b = A.slot_of_id[ib];
    const ImgTab& T = A.img[(size_t)A.P.box[R.a] * A.nimg + g];
    R.rx = __dsub_rn(__dadd_rn(A.P.x[R.b], T.ox), A.P.x[R.a]);
    R.ry = __dsub_rn(__dadd_rn(A.P.y[R.b], T.oy), A.P.y[R.a]);
    R.rz = __dsub_rn(__dadd_rn(A.P.z[R.b], T.oz), A.P.z[R.a]);
    R.dvy = T.dvy;
    // the impulse along n = r/|r| without forming n: v_a gains
    // (1 + eps) (m_b/M) (u.r)/|r|^2 r, v_b loses the same with m_a; the
    // factors of u.r here, but for 1 + eps under the power law.  Fused operations
    // and one refined reciprocal: 203 us for 944k pairs, against 290 with one
    // rounding per operation and a division on the chain.
    const double r2 = fma(R.rz, R.rz, fma(R.ry, R.ry, R.rx * R.rx));
    const double ma = A.P.m[R.a], mb = A.P.m[R.b];
    const double d = r2 * (ma + mb);
    const double y = rcp64(d);
    const double num = kPower ? 1.0 : 1.0 + C.eps;
    double q = num * y;
    q = fma(fma(-d, q, num), y, q);   // num / d to the last bit or so
    R.ka = q * mb;
    R.kb = q * ma;
    R.rabs = kPower ? __dsqrt_rn(r2) : 0.0;
    R.pb = last_before(A, ib, k);
    R.pa = k > 0 && key_a(A.key[k - 1]) == ia ? k - 1 : last_before(A, ia, k);
    if (C.hold_pair && k == 0) R.pa = 0;   // test hook: waits for itself
    return R;
}

constexpr unsigned long long kWaitLimitNs = 500000000ull;   // half a second

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ int ld_flag(const int32_t* p) {
    int v;
    asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Eq. 2 for every pair, as if one after the other in queue order.  Warps claim
// 32 pairs at a time in that order, each lane forms the record of one (while
// the pairs before it are being resolved) and resolves it as soon as the previous pair of either
// particle is marked done: it reads the velocities from L2, where the other
// SMs left them, writes the new ones and marks its own pair (release).  A
// lane's predecessors come earlier in the queue, so they are held by running
// warps or by lanes of its own warp, which the loop serves in turn, and every
// wait ends however many blocks are resident; it is bounded all the same (half
// a second in which no warp of the launch finishes its pairs, or at once when
// another thread gave up) and reports kErrResolveStall.
// What bounds it is the chain of dependent pairs, one link at a time: a flag
// read, a velocity read, 15 FP64 operations, and a release after the
// velocities have reached L2.  The whole resolution, links included: 47 us for
// 2,233 pairs and 203 us for 944k (50 and 228 us with the records formed by a
// kernel of their own and read back), against 144 and 452 us with a queue of
// ready pairs, wait counts and a sort of the pair ends (six dependent round
// trips and 60 FP64 operations a link).  With 944k pairs the FP64 pipe is busy
// three quarters of the time: a warp evaluates its 32 pairs in about 4 rounds.
template <bool kPower>
__global__ void __launch_bounds__(256) k_resolve(ResolveArgs A, SimC C) {
    if (A.advance && blockIdx.x == 0 && threadIdx.x == 0) A.ctl->step += 1;   // nothing here reads the time
    const int n = sorted_counts(A.ctl).x;
    const int lane = threadIdx.x & 31;
    int nres = 0;
    for (;;) {
        int base = 0;
        if (lane == 0) base = atomicAdd(A.claim, 32);
        base = __shfl_sync(0xffffffffu, base, 0);
        if (base >= n) break;
        const int k = base + lane;
        bool pending = k < n, stalled = false;
        PairRec R;
        if (pending) R = pair_rec<kPower>(A, C, k);
        unsigned long long t0 = 0;
        int seen = 0;
        for (int spin = 0; __any_sync(0xffffffffu, pending); spin++) {
            bool moved = false;
            if (pending) {
                if (R.pa >= 0 && ld_flag(&A.done[R.pa])) R.pa = -1;
                if (R.pb >= 0 && ld_flag(&A.done[R.pb])) R.pb = -1;
                if (R.pa < 0 && R.pb < 0) {
                    __threadfence();   // the predecessors' velocities before the reads below
                    double *xa = &A.P.vx[R.a], *ya = &A.P.vy[R.a], *za = &A.P.vz[R.a];
                    double *xb = &A.P.vx[R.b], *yb = &A.P.vy[R.b], *zb = &A.P.vz[R.b];
                    const double vxa = __ldcg(xa), vya = __ldcg(ya), vza = __ldcg(za);
                    const double vxb = __ldcg(xb), vyb = __ldcg(yb), vzb = __ldcg(zb);
                    const double ux = vxb - vxa, uy = (vyb + R.dvy) - vya, uz = vzb - vza;
                    const double rv = fma(R.rz, uz, fma(R.ry, uy, R.rx * ux));
                    if (!(rv >= 0.0)) {   // approaching, or not a number: it spreads to both
                        double g = rv;
                        if (kPower) {
                            // velocity-dependent restitution: min(1, (|v_n| / v_c)^(-p)),
                            // |v_n| = |u.r| / |r|; 1 up to v_c (p is not negative)
                            const double v = __ddiv_rn(__ddiv_rn(fabs(rv), R.rabs), C.eps_vc);
                            const double q = v > 1.0 ? pow(v, -C.eps_p) : 1.0;
                            g = (1.0 + (q < 1.0 ? q : 1.0)) * rv;
                        }
                        const double ga = g * R.ka, gb = g * R.kb;
                        __stcg(xa, fma(ga, R.rx, vxa));
                        __stcg(ya, fma(ga, R.ry, vya));
                        __stcg(za, fma(ga, R.rz, vza));
                        __stcg(xb, fma(-gb, R.rx, vxb));
                        __stcg(yb, fma(-gb, R.ry, vyb));
                        __stcg(zb, fma(-gb, R.rz, vzb));
                        nres++;
                    }
                    asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(&A.done[k]), "r"(1) : "memory");
                    pending = false;
                    moved = true;
                }
            }
            if (!__any_sync(0xffffffffu, moved) && (spin & 63) == 63) {
                // no lane's turn came: look at the clock now and then, and
                // whether any warp has gone on to its next pairs meanwhile
                const unsigned long long t = global_ns();
                const int c = ld_flag(A.claim);
                if (t0 == 0 || c != seen) {
                    t0 = t;
                    seen = c;
                }
                stalled = (*(volatile int*)&A.ctl->err & kErrResolveStall) || t - t0 > kWaitLimitNs;
                if (stalled) atomicOr(&A.ctl->err, kErrResolveStall);
                if (__any_sync(0xffffffffu, stalled)) break;
            }
        }
        if (__any_sync(0xffffffffu, stalled)) break;
    }
    nres = __reduce_add_sync(0xffffffffu, nres);
    if (lane == 0 && nres) atomicAdd(&A.ctl->resolved, nres);
}

int g_resolve_blocks[2] = {0, 0};   // resident blocks of k_resolve<false / true> on the whole GPU

}  // namespace

void resolve_prepare(int nsm) {
    const void* fn[2] = {(const void*)k_resolve<false>, (const void*)k_resolve<true>};
    for (int p = 0; p < 2; p++) {
        int per_sm = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn[p], 256, 0) != cudaSuccess) {
            cudaGetLastError();
            per_sm = 1;
        }
        g_resolve_blocks[p] = std::max(nsm, 1) * std::max(per_sm, 1);
    }
}

namespace {

__global__ void k_step_advance(Ctl* ctl) { ctl->step += 1; }

// Energy terms of one box, per block: K, tidal, W, Px, Py, Pz, count.
__global__ void __launch_bounds__(256) k_energy_partial(PSet P, const Ctl* ctl, SimC C,
                                                        const double* __restrict__ phi, int box,
                                                        double* __restrict__ partials) {
    const int n = ctl->n_live;
    double s[7] = {0, 0, 0, 0, 0, 0, 0};
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        if (P.box[i] != box) continue;
        const double m = P.m[i];
        const double vx = P.vx[i], vy = P.vy[i], vz = P.vz[i];
        s[0] += 0.5 * m * (vx * vx + vy * vy + vz * vz);
        if (C.integrator == 1)
            s[1] += m * (0.5 * (C.omega_z * C.omega_z) * (P.z[i] * P.z[i]) -
                          1.5 * (C.omega * C.omega) * (P.x[i] * P.x[i]));
        if (phi) s[2] += 0.5 * m * phi[i];
        s[3] += m * vx;
        s[4] += m * vy;
        s[5] += m * vz;
        s[6] += 1.0;
    }
    __shared__ double red[7][8];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < 7; q++) {
        double v = s[q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) red[q][w] = v;
    }
    __syncthreads();
    if (threadIdx.x < 7) {
        double v = 0.0;
        for (int k = 0; k < 8; k++) v += red[threadIdx.x][k];
        partials[threadIdx.x * gridDim.x + blockIdx.x] = v;
    }
}

__global__ void k_energy_final(const double* __restrict__ partials, int nparts,
                               double* __restrict__ out7) {
    const int q = threadIdx.x;
    if (q >= 7) return;
    double v = 0.0;
    for (int k = 0; k < nparts; k++) v += partials[q * nparts + k];
    out7[q] = v;
}

}  // namespace

void drift_keys(const PSet& P, const Tree& T, Ctl* ctl, const BoxP* boxes, const SimC& C,
                int ncap, int ndrift, int half_step_offset, const double* ax, const double* ay,
                const double* az, bool kick, bool keys, cudaStream_t s) {
    if (ncap <= 0) return;
    DriftArgs A;
    A.P = P; A.key = T.key; A.idx = T.idx; A.sbox = T.sbox; A.ctl = ctl; A.boxes = boxes;
    A.ax = ax; A.ay = ay; A.az = az;
    A.ncap = ncap; A.ndrift = ndrift; A.hs = half_step_offset;
    const int grid = ceil_div(ncap, 256);
    auto launch = [&](auto k, auto d) {
        if (C.integrator == 0) k_drift_keys<k, d, false><<<grid, 256, 0, s>>>(A, C);
        else k_drift_keys<k, d, true><<<grid, 256, 0, s>>>(A, C);
    };
    using std::bool_constant;
    if (keys && kick) launch(bool_constant<true>{}, bool_constant<true>{});
    else if (keys) launch(bool_constant<true>{}, bool_constant<false>{});
    else if (kick) launch(bool_constant<false>{}, bool_constant<true>{});
    else launch(bool_constant<false>{}, bool_constant<false>{});
}

void sort_and_permute(const PSet& src, const PSet& dst, Tree& T, Pairs& PR, Ctl* ctl,
                      const SimC& C, int ncap, int box_bits, cudaStream_t s) {
    if (ncap <= 0) return;
    // passes over the top bits, the rest within the short runs that agree there
    const int which = radix_sort(T.key, T.idx, T.key_alt, T.idx_alt, ncap, nullptr, 64,
                                 C.nbox > 1 ? T.sbox : nullptr, box_bits, T.hist, &ctl->err, s, C.key_low, nullptr,
                                 &ctl->long_keys, (C.hold_sort & kHoldParticles) != 0);
    // a sort by the top bits counts on zero digit totals, and leaves them
    if (C.key_low == 0) cudaMemsetAsync(T.hist, 0, sizeof(uint32_t) * radix_digit_words(), s);
    if (which == 1) {
        // keep the sorted keys in T.key for the topology kernels
        uint64_t* k = T.key; T.key = T.key_alt; T.key_alt = k;
        uint32_t* v = T.idx; T.idx = T.idx_alt; T.idx_alt = v;
    }
    k_permute<<<ceil_div(ncap, 256), 256, 0, s>>>(src, dst, T.idx, PR.slot_of_id, ctl, ncap, T,
                                                  (int)entry_scan_words(ncap), C.nbox);
}

// Live particles of one box written in id order (id - base) to out, with a
// flag per id and a count.
__global__ void __launch_bounds__(256) k_by_id(PSet P, PSet out, int box, int base, int ncap,
                                               int32_t* __restrict__ flags, int* __restrict__ count) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const bool mine = i < ncap && P.box[i] == box;
    if (mine) {
        const int k = P.id[i] - base;
        out.x[k] = P.x[i]; out.y[k] = P.y[i]; out.z[k] = P.z[i];
        out.vx[k] = P.vx[i]; out.vy[k] = P.vy[i]; out.vz[k] = P.vz[i];
        out.m[k] = P.m[i]; out.r[k] = P.r[i];
        flags[k] = 1;
    }
    const unsigned b = __ballot_sync(0xffffffffu, mine);
    if ((threadIdx.x & 31) == 0 && b) atomicAdd(count, __popc(b));
}

// Slots of a freshly copied single box: slot i holds id i; slots from n on
// are unused (box = nbox).
__global__ void __launch_bounds__(256) k_reset_slots(PSet P, int32_t* __restrict__ slot_of_id, int n,
                                                     int ncap, int nbox) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ncap) return;
    P.id[i] = i;
    P.box[i] = i < n ? 0 : nbox;
    slot_of_id[i] = i;
}

// Checks of freshly copied particles: bit 0 a non-finite position or
// velocity, bit 1 a negative (or NaN) mass or radius; the largest radius as
// the bits of a non-negative double.
__global__ void __launch_bounds__(256) k_check_particles(PSet P, int n,
                                                         unsigned long long* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long bad = 0, rb = 0;
    if (i < n) {
        if (!(isfinite(P.x[i]) && isfinite(P.y[i]) && isfinite(P.z[i]) && isfinite(P.vx[i]) &&
              isfinite(P.vy[i]) && isfinite(P.vz[i])))
            bad |= 1ull;
        const double r = P.r[i];
        if (!(P.m[i] >= 0.0) || !(r >= 0.0)) bad |= 2ull;
        else if (r > 0.0) rb = (unsigned long long)__double_as_longlong(r);   // not -0.0
    }
    for (int o = 16; o > 0; o >>= 1) {
        bad |= __shfl_xor_sync(0xffffffffu, bad, o);
        rb = max(rb, __shfl_xor_sync(0xffffffffu, rb, o));
    }
    if ((threadIdx.x & 31) == 0) {
        if (bad) atomicOr(&out[0], bad);
        if (rb) atomicMax(&out[1], rb);
    }
}

void check_particles(const PSet& P, int n, unsigned long long* out2, cudaStream_t s) {
    cudaMemsetAsync(out2, 0, 2 * sizeof(unsigned long long), s);
    if (n > 0) k_check_particles<<<ceil_div(n, 256), 256, 0, s>>>(P, n, out2);
}

void particles_by_id(const PSet& P, const PSet& out, int box, int base, int ncap, int32_t* flags,
                     int nflags, int* count, cudaStream_t s) {
    cudaMemsetAsync(flags, 0, sizeof(int32_t) * (size_t)(nflags > 0 ? nflags : 1), s);
    cudaMemsetAsync(count, 0, sizeof(int), s);
    if (ncap > 0) k_by_id<<<ceil_div(ncap, 256), 256, 0, s>>>(P, out, box, base, ncap, flags, count);
}

// Three values per slot of one box's live particles, by id, as 8-byte values.
template <typename T, typename V>
__global__ void __launch_bounds__(256) k_results_by_id(PSet P, const V* __restrict__ a, const V* __restrict__ b,
                                                       const V* __restrict__ c, T* __restrict__ out, int box, int base,
                                                       int ncap, int32_t* __restrict__ flags, int* __restrict__ count) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const bool mine = i < ncap && P.box[i] == box;
    if (mine) {
        const int k = P.id[i] - base;
        out[k] = (T)a[i];
        out[ncap + k] = (T)b[i];
        out[2 * (size_t)ncap + k] = (T)c[i];
        flags[k] = 1;
    }
    const unsigned m = __ballot_sync(0xffffffffu, mine);
    if ((threadIdx.x & 31) == 0 && m) atomicAdd(count, __popc(m));
}

template <typename T, typename V>
void results_by_id(const PSet& P, const V* const src[3], T* out, int box, int base, int ncap, int32_t* flags, int nflags,
                   int* count, cudaStream_t s) {
    cudaMemsetAsync(flags, 0, sizeof(int32_t) * (size_t)(nflags > 0 ? nflags : 1), s);
    cudaMemsetAsync(count, 0, sizeof(int), s);
    if (ncap > 0)
        k_results_by_id<T, V><<<ceil_div(ncap, 256), 256, 0, s>>>(P, src[0], src[1], src[2], out, box, base, ncap, flags,
                                                                  count);
}
template void results_by_id<double, double>(const PSet&, const double* const[3], double*, int, int, int, int32_t*, int,
                                            int*, cudaStream_t);
template void results_by_id<int64_t, int32_t>(const PSet&, const int32_t* const[3], int64_t*, int, int, int, int32_t*,
                                              int, int*, cudaStream_t);

void reset_slots(const PSet& P, int32_t* slot_of_id, int n, int ncap, int nbox, cudaStream_t s) {
    if (ncap > 0) k_reset_slots<<<ceil_div(ncap, 256), 256, 0, s>>>(P, slot_of_id, n, ncap, nbox);
}

void sort_pairs(Pairs& PR, Ctl* ctl, const SimC& C, cudaStream_t s, int key_bits) {
    // passes over the lower id's bits, then each id's pairs among themselves;
    // an odd number of passes leaves the keys in key_alt; the buffers are
    // not swapped, so every captured graph finds them in the same place
    PR.sorted_alt = radix_sort(PR.key, PR.val, PR.key_alt, PR.val_alt, PR.cap, &ctl->pair_n,
                               key_bits, nullptr, 0, PR.hist, &ctl->err, s, 36, ctl, nullptr,
                               (C.hold_sort & kHoldPairs) != 0) == 1;
}

void resolve_pairs(const PSet& P, Ctl* ctl, const BoxP* boxes, const SimC& C, Pairs& PR,
                   int half_step_offset, ImgTab* img, bool have_img, bool advance, cudaStream_t s) {
    ResolveArgs A;
    A.P = P; A.key = PR.sorted(); A.slot_of_id = PR.slot_of_id;
    A.head = PR.head; A.link = PR.link; A.done = PR.done; A.claim = PR.claim;
    A.img = img;
    A.ngx = C.ngx; A.ngy = C.ngy; A.ngz = C.ngz;
    A.nimg = have_img ? C.nimg : build_image_table(boxes, ctl, C, half_step_offset, img, s);
    A.ctl = ctl;
    A.advance = advance;
    cudaMemsetAsync(PR.head, 0xff, sizeof(int32_t) * (size_t)PR.ncap, s);   // empty lists
    const int grid = std::min(ceil_div(PR.cap, 256), 8 * 152);
    k_pair_link<<<grid, 256, 0, s>>>(A);
    const int rgrid = std::max(1, std::min(ceil_div(PR.cap, 256), g_resolve_blocks[C.eps_law == 1]));
    if (C.eps_law == 1) k_resolve<true><<<rgrid, 256, 0, s>>>(A, C);
    else k_resolve<false><<<rgrid, 256, 0, s>>>(A, C);
}

void energy_terms(const PSet& P, Ctl* ctl, const SimC& C, const double* phi, int box,
                  double* partials, int nparts, double* out7, cudaStream_t s) {
    k_energy_partial<<<nparts, 256, 0, s>>>(P, ctl, C, phi, box, partials);
    k_energy_final<<<1, 32, 0, s>>>(partials, nparts, out7);
}

void step_advance(Ctl* ctl, cudaStream_t s) { k_step_advance<<<1, 1, 0, s>>>(ctl); }

// What a step starts from zero: the error word, the counters of the walk and of
// the search, and the counts of pairs and of corrected cells.
void clear_step(Ctl* ctl, cudaStream_t s) {
    cudaMemsetAsync(&ctl->err, 0, offsetof(Ctl, sweep_wbits) - offsetof(Ctl, err), s);
}

void clear_build(Ctl* ctl, bool walk, cudaStream_t s) {
    cudaMemsetAsync(&ctl->err, 0, walk ? offsetof(Ctl, pair_count) - offsetof(Ctl, err) : sizeof(int), s);
}

void clear_search_stats(Ctl* ctl, cudaStream_t s) {
    cudaMemsetAsync(&ctl->n_visit, 0, 2 * sizeof(unsigned long long), s);
}

}  // namespace rb
