// rb_walk.cuh -- device pieces shared by the gravity walks (rb_walk.cu: the
// walks over 32 targets per warp; rb_twalk.cu: the walks with one or two
// targets per warp) and the collision search: kernel arguments, tile scheduling, the
// opening and inside tests, interaction terms and the learned walk's queue.
#pragma once
#include "rb_internal.cuh"
#include "rb_mlp.cuh"

namespace rb {

struct GravArgs {
    const double *x, *y, *z;
    const int32_t* box;
    Rec4 ra, rb, rq0, rq1, rc_hi, rc_lo;
    const double4_32a *d_a, *d_q0, *d_q1, *d_c;
    const int32_t *e_skip, *leaf_of, *box_root;
    const uint32_t* order;      // tile order of the targets (nullptr: Morton order of the slots)
    const int32_t* e_child;     // per cell entry: child entry of each octant (group walk)
    const uint32_t* e_cmask;    // per cell entry: octants holding a child (0: depth-21 group)
    const BoxP* boxes;
    Ctl* ctl;
    WalkOut out;
    int ncap;
    int ngx, ngy, ngz;
    int half_step_offset;
    double G, theta2, soft2, t0, half_dt;
    float soft2f;
    // recording of accepted cells in the band w/R > theta_lo (learned mode)
    uint64_t* req;
    int* req_count;
    int req_cap;
    float band_scale;   // (theta_lo / theta)^2: band iff (w/theta)^2 > band_scale R^2
    uint32_t thresh;    // keep a request when its hash < thresh (0xffffffff: all)
    uint32_t seed;
    // learned walk: cell particle counts (an input of the network) and weights
    const int32_t* e_count;
    const mlp::Packed* wpk;
    int ecap;   // entry capacity (every entry index below it is readable)
    const ImgTab* img;   // [box][image] offsets at the time of this walk
    int nimg;
    int32_t* tq;         // tile queues (emptied by the image-table launch)
    int nq;
};

// Resident blocks of a walk kernel (queried once per kernel and block size,
// outside any capture) and the persistent grid that runs `warps` warps of
// work on them: the same number of blocks on every SM, as many as the work
// fills and as fit.  With a grid of just the blocks that the work fills, the
// few SMs that get one block more end last: union walk of the sheet 425 -> 360
// us at 60k targets, 501 -> 380 at 100k, 585 -> 468 at 150k (the same from 200k
// on, where every SM is full either way), search 55 -> 47 us at 2400.  A block
// without work finds the queues empty and ends.
void walk_prepare_kernel(const void* fn);
int walk_grid(const void* fn, int block, long long warps);

// rb_twalk.cu: the walks with one or two targets per warp.  A holds the target
// order, records and image table; block is 64, 128 or 256 threads (FP64).
// FP32 walks take them up to a number of targets where the chain of entries that
// a warp of 32 targets steps through is longer than the work.  Walk times on the
// sheet (theta = 0.5, 9 images, targets in Hilbert order), two targets per warp
// against 32: 117 us against 319 at 20k targets, 154 against 325 at 30k, 242
// against 331 at 50k, 333 against 344 at 70k, 381 against 366 at 80k and 481
// against 378 at 100k.  In Morton order the 32 targets' walks have less in
// common: a whole gravity evaluation takes 579 us against 812 at 80k, 698 against
// 948 at 100k and 884 against 973 at 130k (sheet), 1772 against 2002 at 100k and
// 2491 against 2259 at 130k (Plummer sphere, theta = 0.5), 1344 against 1508 at
// 130k (periodic cube).  With the network, whose rows a warp's one target fills
// better than 32 lanes' band cells in turn: 573 us against 803 at 40k, 1516
// against 1818 at 100k, 3171 against 2968 at 200k (theta = 0.8).
constexpr int kTargetWalkMax = 75000;           // targets in a Hilbert order
constexpr int kTargetWalkMaxMorton = 125000;
constexpr int kTargetWalkMaxLearned = 130000;
static_assert(kTargetWalkMax <= kLeafQMax && kTargetWalkMaxMorton <= kLeafQMax && kTargetWalkMaxLearned <= kLeafQMax,
              "these walks read the leaves' multipole records");
enum class TargetWalk { kFp32, kFp64, kLearned };
void target_walk(const GravArgs& A, TargetWalk mode, bool quad, bool inside, bool soft, bool pot, int block,
                 int cap_n, cudaStream_t s);
void target_walk_prepare();
void collision_search_prepare();   // rb_collide.cu

namespace {

constexpr unsigned kFull = 0xffffffffu;

// The 32-byte pair of an entry in one 256-bit load.
__device__ __forceinline__ void ld_pair(const Rec4& r, int e, float4& a, float4& b) {
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
        : "l"(r.p + 2 * (size_t)e));
}

__device__ __forceinline__ double4_32a ld_d4(const double4_32a* p) { return *p; }

// Counter-based hash of a (target, cell, image) request for subsampling.
__device__ __forceinline__ uint32_t req_hash(uint32_t slot, uint32_t entry, uint32_t code,
                                             uint32_t seed) {
    uint32_t h = slot * 0x9E3779B1u ^ (entry + 0x7F4A7C15u) * 0x85EBCA77u ^ code * 0xC2B2AE3Du ^ seed;
    h ^= h >> 16;
    h *= 0x7FEB352Du;
    h ^= h >> 15;
    h *= 0x846CA68Bu;
    h ^= h >> 16;
    return h;
}

// Opening test in FP64, operation for operation as the oracle evaluates it.
__device__ __forceinline__ bool mac64(const double4_32a& a, double theta2, double tx, double ty,
                                      double tz) {
    const double dx = __dsub_rn(a.x, tx), dy = __dsub_rn(a.y, ty), dz = __dsub_rn(a.z, tz);
    const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
    return a.w < __dmul_rn(theta2, r2);
}

// 1/sqrt(x) from the hardware estimate plus one Newton step
// y' = y (3/2 - x y^2 / 2), which roughly halves its relative error.
__device__ __forceinline__ float rsqrt_nr(float x) {
    const float y = rsqrtf(x);
    return y * fmaf((-0.5f * x) * y, y, 1.5f);
}

// Compensated (Kahan) accumulation: in a sheet the net force is often a
// small remainder of much larger cancelling terms, and a plain FP32 running
// sum loses ~1e-5 of it.  The walk sums terms plainly over at most 16 warp
// iterations and adds those short partial sums into Kahan sums, whose
// running compensation c keeps the lost low-order bits.
__device__ __forceinline__ void kadd(float& s, float& c, float t) {
    const float y = t - c;
    const float u = s + y;
    c = (u - s) - y;
    s = u;
}

// Tile scheduling of the walks: queue q owns tiles [b_q, b_{q+1}) with
// b_q = floor(q T / nq) of the T tiles of 32 consecutive targets.
__device__ __forceinline__ int tile_begin(int q, int ntile, int nq) {
    return (int)(((long long)q * ntile) / nq);
}

__device__ __forceinline__ int sm_queue(int nq) {
    unsigned sm;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(sm));
    return (int)(sm % (unsigned)nq);
}

// Slot of the k-th target in tile order.
__device__ __forceinline__ int tile_slot(const uint32_t* order, int k) {
    return order ? (int)__ldg(&order[k]) : k;
}

// The warp's next tile, or -1 when every queue is empty: its own SM's queue
// first, then the following queues (32 probed per vote).  Warp-uniform.
__device__ __noinline__ int next_tile(int32_t* tq, int nq, int q, int ntile) {
    const int lane = threadIdx.x & 31;
    int t = -1;
    if (lane == 0) {
        const int b = tile_begin(q, ntile, nq);
        const int k = atomicAdd(&tq[q * kTileQStride], 1);
        if (k < tile_begin(q + 1, ntile, nq) - b) t = b + k;
    }
    t = __shfl_sync(kFull, t, 0);
    if (t >= 0) return t;
    for (int k0 = 1; k0 < nq; k0 += 32) {
        const int off = k0 + lane;
        int qq = q + off;
        if (qq >= nq) qq -= nq;
        int b = 0, len = 0;
        bool avail = false;
        if (off < nq) {
            b = tile_begin(qq, ntile, nq);
            len = tile_begin(qq + 1, ntile, nq) - b;
            avail = __ldcg(&tq[qq * kTileQStride]) < len;
        }
        for (unsigned m = __ballot_sync(kFull, avail); m; m &= m - 1) {
            const int src = __ffs(m) - 1;
            int got = -1;
            if (lane == src) {
                const int k = atomicAdd(&tq[qq * kTileQStride], 1);
                if (k < len) got = b + k;
            }
            got = __shfl_sync(kFull, got, src);
            if (got >= 0) return got;
        }
    }
    return -1;
}

// t = p - o for hi/lo float pairs: the rounding error of ph - oh is kept
// (Knuth's two-sum) and the low parts are subtracted, so t is good to about
// 2^-45 of |p| without any FP64 arithmetic.
__device__ __forceinline__ void sub_hilo(float ph, float pl, float oh, float ol, float& th, float& tl) {
    const float s = ph - oh;
    const float bb = s - ph;
    const float e = (ph - (s - bb)) + (-oh - bb);
    th = s;
    tl = e + (pl - ol);
}

__device__ __forceinline__ void split_d(double v, float& hi, float& lo) {
    hi = __double2float_rn(v);
    lo = __double2float_rn(v - (double)hi);
}

// Is the target point inside the closed cube of a cell (FP64, exact sequence)?
__device__ __forceinline__ bool inside64(const double4_32a& c, double tx, double ty, double tz) {
    return c.x <= tx && tx <= __dadd_rn(c.x, c.w) && c.y <= ty && ty <= __dadd_rn(c.y, c.w) &&
           c.z <= tz && tz <= __dadd_rn(c.z, c.w);
}

// Monopole + quadrupole term of an accepted cell (reading R3), the same
// arithmetic as the union walk's.  A particle leaf is the cell with Q = 0, but
// for its distance, which may be zero when softened, and for r^-5 and r^-7,
// which overflow at distances where its term does not.
template <bool kQuad, bool kSoft>
__device__ __forceinline__ void cell_term(float dx, float dy, float dz, float r2, const float4& q0,
                                          const float4& q1, bool leaf, float soft2f, float& fx, float& fy,
                                          float& fz) {
    const float inv = rsqrt_nr(kSoft && leaf ? r2 + soft2f : r2);
    const float inv2 = inv * inv;
    const float invs = kSoft ? rsqrt_nr(r2 + soft2f) : inv;
    float fc = q0.x * (kSoft ? invs * invs * invs : inv2 * inv);
    if (kQuad) {
        const float qx = fmaf(q1.y, dz, fmaf(q1.x, dy, q0.y * dx));
        const float qy = fmaf(q1.z, dz, fmaf(q0.z, dy, q1.x * dx));
        const float qz = fmaf(q0.w, dz, fmaf(q1.z, dy, q1.y * dx));
        const float dqd = fmaf(dz, qz, fmaf(dy, qy, dx * qx));
        const float inv5 = leaf ? 0.f : inv2 * inv2 * inv;
        fc = fmaf(2.5f, dqd * (inv5 * inv2), fc);
        fx = fmaf(-inv5, qx, fx);
        fy = fmaf(-inv5, qy, fy);
        fz = fmaf(-inv5, qz, fz);
    }
    fx = fmaf(fc, dx, fx);
    fy = fmaf(fc, dy, fy);
    fz = fmaf(fc, dz, fz);
}

// Record minus target for the negated target point (nxy: x, y hi; lxy: x, y
// lo; nz: z hi, lo).
__device__ __forceinline__ void rec_diff(const float4& ra, const float4& rb, float2 nxy, float2 lxy,
                                         float2 nz, float& dx, float& dy, float& dz, float& r2) {
    const float2 dxy = __fadd2_rn(__fadd2_rn(make_float2(ra.x, ra.y), nxy),
                                  __fadd2_rn(make_float2(rb.x, rb.y), lxy));
    dx = dxy.x;
    dy = dxy.y;
    const float2 zz = __fadd2_rn(make_float2(ra.z, ra.w), nz);
    dz = zz.x + zz.y;
    r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
}

// Per-warp queue of the learned walk: accepted band cells waiting for the
// network, which runs on 16 of them at a time (one m16 tile).
struct LearnQ {
    __nv_bfloat16 X[48][16];   // network inputs (columns 12..15 zero)
    float unit[48];            // M / R^2 (G is applied with the walk's sums)
    int own[48];               // lane whose sums receive the output
    float Y[16][4];            // outputs of the tile being applied
};

// Rows r0 .. r0 + 15 of the queue through the network; unit * output is
// added to the owning lanes' partial sums.  Warp-synchronous.
__device__ __forceinline__ void learn_flush(LearnQ& Q, const mlp::Packed& w, int r0, int lane,
                                            float& fx, float& fy, float& fz) {
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
#pragma unroll 4
    for (int k = 0; k < 16; k++)
        if (Q.own[r0 + k] == lane) {
            const float u = Q.unit[r0 + k];
            fx += u * Q.Y[k][0];
            fy += u * Q.Y[k][1];
            fz += u * Q.Y[k][2];
        }
    __syncwarp();
}

}  // namespace
}  // namespace rb
